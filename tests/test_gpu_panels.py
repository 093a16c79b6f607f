"""The panel kernels, which solve every system above the column slices' size,
on small systems (TB_SLICE=0): every panel width, so every form of the
Chebyshev step and of the FP32 CG product (one, two and four column pairs per
thread, S staged in shared memory or not), full and partly filled CTAs,
systems of s-only atoms.  Each test checks from the launch counters that the
slices took no part."""
import numpy as np
import pytest

from tbinputs import gauss_legendre_grid, si_system, water_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_1202_gb300 as pkg
    pkg.build()
    return pkg


def launches(P):
    return {k: P.tb_profile_read(k)[0] for k in P.tb.KERNELS}


@pytest.fixture
def ran(P, monkeypatch):
    """Counts the launches of a test per kernel class, on the panel kernels only."""
    monkeypatch.setenv("TB_SLICE", "0")
    before = launches(P)

    def delta():
        return {k: n - before[k] for k, n in launches(P).items()}

    yield delta
    assert delta()["slice"] == 0


# 64 atoms of silicon (identity diagonal blocks, 17 blocks a row: S staged) and
# 99 of water (s and sp atoms, rows too long to stage in the narrower panels, a
# last CTA with fewer rows in every form)
SYSTEMS = {"si64": lambda: si_system((2, 2, 2), sigma=0.05, seed=1),
           "water33": lambda: water_system(33, seed=6, excess_proton=False)}
STEPS = 12


@pytest.fixture(scope="module", params=list(SYSTEMS))
def case(request, P):
    s = SYSTEMS[request.param]()
    h = P.tb_create_system(s)
    lo, hi = (-20.0, 5.0) if s.eps.min() > -20 else (-40.0, 0.0)
    z, _ = gauss_legendre_grid(6, lo, hi, 1.0)
    cols = np.random.default_rng(3).permutation(s.n_orb)[:256].astype(np.int32)
    mp = pytest.MonkeyPatch()
    mp.setenv("TB_SLICE", "0")
    ref = P.tb_shifted_cocg(h, z, cols, opts=P.tb_default_opts(max_iter=STEPS, panel=64),
                            allow_unconverged=True)[0].cpu().numpy()
    mp.undo()
    return h, z, cols, ref


@pytest.mark.parametrize("method", [0, 1], ids=["chebyshev", "cg"])
@pytest.mark.parametrize("panel", [1, 2, 4, 8, 16, 32, 64, 128, 256])
def test_panel_widths(P, case, ran, panel, method):
    """A fixed number of outer steps of full solutions, mixed precision, for
    every panel width against the FP64 panels of 64 columns: the same
    recurrences with inner solves to 1e-13, so they agree to 1e-9 as the slices
    and the panels do."""
    h, z, cols, ref = case
    n = min(panel, len(cols))
    opts = P.tb_default_opts(precision=1, inner_method=method, max_iter=STEPS, panel=panel)
    x = P.tb_shifted_cocg(h, z, cols[:n], opts=opts, allow_unconverged=True)[0].cpu().numpy()
    assert np.abs(x - ref[:, :n]).max() <= 1e-9 * np.abs(ref).max()
    assert ran()["inner32_cheb" if method == 0 else "inner32_spmv"] > 0


@pytest.mark.parametrize("panel", [1, 8, 256])
def test_fp64_panel_widths(P, case, ran, panel):
    """The same in FP64: the scalars of the inner CG, one thread per column."""
    h, z, cols, ref = case
    n = min(panel, len(cols))
    opts = P.tb_default_opts(max_iter=STEPS, panel=panel)
    x = P.tb_shifted_cocg(h, z, cols[:n], opts=opts, allow_unconverged=True)[0].cpu().numpy()
    assert np.abs(x - ref[:, :n]).max() <= 1e-9 * np.abs(ref).max()
    assert ran()["inner_spmv"] > 0


@pytest.mark.parametrize("R,prec", [(1, 0), (2, 0), (7, 1), (64, 1), (256, 1)])
def test_lanczos_widths(P, R, prec):
    """The Lanczos process of R columns at once (one column per thread of its
    products, a pair from 256 columns of 640 atoms on) against the single-column
    call: the coefficients of 10 steps to 1e-8, as the existing batch checks."""
    s = si_system((4, 4, 5), sigma=0.05, seed=2)
    h = P.tb_create_system(s)
    cols = np.random.default_rng(R).permutation(s.n_orb)[:R].astype(np.int32)
    a, b, nrm = (np.asarray(v.cpu() if hasattr(v, "cpu") else v)
                 for v in P.tb_generalized_lanczos_batch(h, cols, 10, opts=P.tb_default_opts(precision=prec)))
    for c in sorted({0, R // 2, R - 1}):
        a0, b0, n0 = (np.asarray(v.cpu() if hasattr(v, "cpu") else v)
                      for v in P.tb_generalized_lanczos(h, int(cols[c]), 10))
        assert np.abs(a[c] - a0).max() <= 1e-8 * np.abs(a0).max()
        assert np.abs(b[c] - b0).max() <= 1e-8 * np.abs(b0).max()
        assert abs(nrm[c] - np.ravel(n0)[0]) <= 1e-10 * abs(np.ravel(n0)[0])


def test_ragged_and_padded_steps_of_a_large_box(P, ran):
    """400 water molecules (2400 orbitals, above the slices' size): one panel of
    256 columns takes the ragged four-pair step, four of 64 in flight and one of
    64 the padded two-pair one; the same populations after fixed steps to 1e-9."""
    s = water_system(400, seed=4, excess_proton=False)
    h = P.tb_create_system(s)
    z, w = gauss_legendre_grid(8, -60.0, -8.0, 1.0)
    cols = np.random.default_rng(5).permutation(s.n_orb)[:256].astype(np.int32)

    def q(n, panel):
        o = P.tb_default_opts(precision=1, max_iter=8, panel=panel)
        return P.tb_mulliken_orbital(h, z, w, cols[:n], 2.0, opts=o, allow_unconverged=True)[0].cpu().numpy()

    wide, narrow, one = q(256, 256), q(256, 64), q(64, 64)
    assert np.abs(wide - narrow).max() <= 1e-9 * np.abs(wide).max()
    assert np.abs(wide[:64] - one).max() <= 1e-9 * np.abs(wide).max()
    assert ran()["inner32_cheb"] > 0


def test_noalloc_request_of_the_whole_scratch(P):
    """The allocation-free call takes what fits ten vectors of one column, its two
    coefficient arrays, the norm and the reductions' sums in its fixed array
    (its capacity before the vectors were held in pairs): a request that fills it
    to the last 512 bytes.  Uncoupled atoms: the process ends at its first step."""
    import torch
    r256 = lambda b: (b + 255) // 256 * 256
    grid = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    cap = 16 << 20
    need = lambda n, k: (10 * r256(64 * n) + 256 + 256 + r256(grid * 32) + 64 * 32 + r256(65 * 4) + 256 + r256(8 * k) +
                         r256(8 * k + 8) + 256)
    n = next(n for n in range(cap // 640, 0, -4) if need(n, 32) <= cap)
    k = next(k for k in range(4000, 0, -1) if need(n, k) <= cap)
    assert cap - 512 < need(n, k) <= cap
    h = P.tb_create(np.ones(n), np.arange(n + 1), np.arange(n), np.ones(n), eps=np.linspace(-20.0, -5.0, n))
    a, b, nrm = (np.asarray(v) for v in P.tb_generalized_lanczos_noalloc(h, 7, k))
    assert len(a) == k and abs(a[0] - np.linspace(-20.0, -5.0, n)[7]) <= 1e-12 * 20 and nrm[0] == 1.0
    assert np.all(b == 0.0)


def test_four_columns_of_a_very_large_system(P, ran):
    """A ring of 100 000 s atoms, whose four columns make more pairs than threads are
    resident (two pairs per thread), against panels of eight (one): full solutions
    after fixed steps to 1e-9."""
    n = 100000
    i = np.arange(n)
    cols = np.sort(np.stack([(i - 1) % n, i, (i + 1) % n], axis=1), axis=1)
    S = np.where(cols == i[:, None], 1.0, 0.2)
    h = P.tb_create(np.ones(n), 3 * np.arange(n + 1), cols.ravel(), S.ravel(), eps=-13.0 + np.sin(i))
    z = np.array([-13.0 + 1j, -10.0 + 1j])
    pick = np.array([5, 31234, 60000, 99999, 7, 8, 9, 10], dtype=np.int32)

    def x(k, panel):
        o = P.tb_default_opts(precision=1, max_iter=6, panel=panel)
        return P.tb_shifted_cocg(h, z, pick[:k], opts=o, allow_unconverged=True)[0].cpu().numpy()[:, :4]

    a, b = x(4, 4), x(8, 8)
    assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
    assert ran()["inner32_cheb"] > 0
