"""Column slices (whole outer steps of a few columns per thread-block cluster,
the path of small systems) against the panel kernels and the dense oracle:
every slice width and cluster size, systems of one atom, of filling rows and
of s-only atoms, one column and ragged column counts, each kind of output."""
import numpy as np
import pytest

from tbinputs import gauss_legendre_grid, si_system, water_system
from oracle import dense

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_1202_gb300 as pkg
    pkg.build()
    return pkg


SYSTEMS = {"si64": lambda: si_system((2, 2, 2), sigma=0.05, seed=1),
           "si216": lambda: si_system((3, 3, 3), sigma=0.05, seed=2),
           "water8": lambda: water_system(8, seed=4, cutoff=3.0, excess_proton=False),
           "water33": lambda: water_system(33, seed=6)}


@pytest.fixture(scope="module", params=list(SYSTEMS))
def case(request, P):
    s = SYSTEMS[request.param]()
    return s, P.tb_create_system(s)


@pytest.fixture(scope="module", params=["si64", "water8"])
def small(request, P):
    s = SYSTEMS[request.param]()
    S = s.dense_S()
    H = dense.ased_hamiltonian(S, s.eps, s.K, s.orbital_atom())
    return s, H, S, P.tb_create_system(s)


def _grid(s, K=12, eta=1.0):
    lo, hi = (-20.0, 5.0) if s.eps.min() > -20 else (-40.0, 0.0)
    return gauss_legendre_grid(K, lo, hi, eta)


# (slice width, cluster size, S in registers): 0 = the library's choice; widths
# above the FP64 path's largest are clipped to it, and a shape that does not
# fit a system leaves it to the panel kernels
@pytest.mark.parametrize("nc,cl,reg", [(0, 0, -1), (1, 1, 0), (2, 3, 0), (4, 8, 0), (8, 2, 0), (2, 1, 1), (2, 4, 1),
                                       (4, 3, 1), (8, 8, 1)])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_fixed_steps_equal_the_panel_path(P, case, monkeypatch, prec, nc, cl, reg):
    """Twenty outer steps with forced seed switches: the same recurrences in
    another summation order, so the full solutions agree as the panel path
    agrees with the oracle's method after a fixed number of steps (1e-9; the
    inner solves of both stop at 1e-13)."""
    s, h = case
    z, w = _grid(s)
    cols = np.linspace(0, s.n_orb - 1, 13).astype(np.int32)
    opts = P.tb_default_opts(precision=prec, max_iter=20, force_switch_every=7, panel=16)
    monkeypatch.setenv("TB_SLICE", "0")
    ref, st0 = P.tb_shifted_cocg(h, z, cols, opts=opts, allow_unconverged=True)
    monkeypatch.setenv("TB_SLICE", "1")
    monkeypatch.setenv("TB_SLICE_NC", str(nc))
    monkeypatch.setenv("TB_SLICE_CL", str(cl))
    monkeypatch.setenv("TB_SLICE_REG", str(reg))
    x, st = P.tb_shifted_cocg(h, z, cols, opts=opts, allow_unconverged=True)
    ref, x = ref.cpu().numpy(), x.cpu().numpy()
    assert np.abs(x - ref).max() <= 1e-9 * np.abs(ref).max()
    assert st["outer_iterations"] == st0["outer_iterations"] and st["switches"] == st0["switches"]


@pytest.mark.parametrize("prec,nc,cl,reg", [(1, 2, 8, 1), (1, 4, 16, 0), (1, 2, 6, 0), (0, 1, 16, 0), (0, 2, 5, 0)])
def test_rows_with_more_copies_than_a_lane_keeps(P, monkeypatch, prec, nc, cl, reg):
    """A lane keeps the remote addresses of its row's first three copies; in
    larger clusters of a small system a row has up to cl - 1 of them.  Two
    bitwise equal runs (a copy stored late or to the wrong place shows there
    too) that agree with the panel path after fixed steps to 1e-9, as above."""
    s = SYSTEMS["si64"]()
    h = P.tb_create_system(s)
    z, w = _grid(s)
    cols = np.array([0, 101, 255], dtype=np.int32)
    opts = P.tb_default_opts(precision=prec, max_iter=12, panel=4)
    monkeypatch.setenv("TB_SLICE", "0")
    ref = P.tb_shifted_cocg(h, z, cols, opts=opts, allow_unconverged=True)[0].cpu().numpy()
    monkeypatch.setenv("TB_SLICE", "1")
    monkeypatch.setenv("TB_SLICE_NC", str(nc))
    monkeypatch.setenv("TB_SLICE_CL", str(cl))
    monkeypatch.setenv("TB_SLICE_REG", str(reg))
    x, y = (P.tb_shifted_cocg(h, z, cols, opts=opts, allow_unconverged=True)[0].cpu().numpy() for _ in range(2))
    assert np.array_equal(x, y)
    assert np.abs(x - ref).max() <= 1e-9 * np.abs(ref).max()


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("R,block", [(1, 0), (3, 32), (16, 64)])
def test_outputs_against_dense(P, small, monkeypatch, prec, R, block):
    """Converged solutions, Green's-function elements with their z-derivatives
    and populations against the dense definitions (broadening 1 eV, tol 1e-10:
    the forward error is at most |A^-1| tol ~ 1e-9 |x|); the sums of solutions
    and derivatives over one block of steps and over several."""
    monkeypatch.setenv("TB_SLICE_BLOCK", str(block))
    s, H, S, h = small
    z, w = _grid(s, K=6)
    cols = np.linspace(0, s.n_orb - 1, R).astype(np.int32)
    opts = P.tb_default_opts(precision=prec)
    G = dense.green_columns(H, S, z, cols)                    # [K][N][R]
    x, st = P.tb_shifted_cocg(h, z, cols, opts=opts)
    assert st["status"] == "TB_OK"
    assert np.abs(x.cpu().numpy() - np.transpose(G, (0, 2, 1))).max() <= 1e-8 * np.abs(G).max()
    rows = np.array([[int(c), 0] for c in cols]).ravel()
    g, dg, _ = P.tb_green_elements_dz(h, z, cols, 2 * np.arange(R + 1), rows, opts=opts)
    dG = dense.green_derivative_columns(H, S, z, cols)
    g, dg = g.cpu().numpy(), dg.cpu().numpy()
    for c in range(R):
        for m in range(2):
            assert np.abs(g[2 * c + m] - G[:, rows[2 * c + m], c]).max() <= 1e-8 * np.abs(G).max()
            assert np.abs(dg[2 * c + m] - dG[:, rows[2 * c + m], c]).max() <= 1e-6 * np.abs(dG).max()
    q, _ = P.tb_mulliken_orbital(h, z, w, cols, 2.0, opts=opts)
    assert np.abs(q.cpu().numpy() - dense.mulliken_orbital(H, S, z, w, 2.0)[cols]).max() <= 1e-8


def test_inner_solve_beyond_the_planned_rounds(P, small):
    """An inner tolerance below what the planned and the spare rounds of the
    refinement reach: the panel kernels take the call over (their FP64 CG
    finishes the inner solves) and the solutions meet the same bar."""
    s, H, S, h = small
    z, w = _grid(s, K=4)
    cols = [0, s.n_orb // 2]
    x, st = P.tb_shifted_cocg(h, z, cols, opts=P.tb_default_opts(precision=1, inner_tol=2e-16))
    assert st["status"] == "TB_OK" and st["inner_redos"] > 0
    G = dense.green_columns(H, S, z, cols)
    assert np.abs(x.cpu().numpy() - np.transpose(G, (0, 2, 1))).max() <= 1e-8 * np.abs(G).max()


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_one_atom(P, prec):
    """One sp atom: one group, the rest of its octet filling rows; G is
    diagonal, 1 / (z - level)."""
    eps = np.array([-13.5, -6.5, -6.5, -6.5])
    h = P.tb_create([4], [0, 1], [0], np.eye(4).ravel(), None, eps, 1.75)
    z = np.array([-13.0 + 0.5j, -6.0 + 0.5j])
    x, _ = P.tb_shifted_cocg(h, z, [0, 2], opts=P.tb_default_opts(precision=prec))
    want = np.zeros((2, 2, 4), dtype=complex)
    want[:, 0, 0], want[:, 1, 2] = 1 / (z + 13.5), 1 / (z + 6.5)
    assert np.abs(x.cpu().numpy() - want).max() <= 1e-10
