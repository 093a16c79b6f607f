"""Which kernels a call of a small system runs, from the launch counters: every
shape of the column slices that fits runs without the panel kernels beside it,
the ones that do not fit are known, and a solve that the slices cannot finish is
handed over to the panel kernels, also after some of its launches."""
import numpy as np
import pytest

from oracle import dense
from tbinputs import gauss_legendre_grid, si_system, water_system

pytestmark = pytest.mark.gpu

SYSTEMS = {"si64": lambda: si_system((2, 2, 2), sigma=0.05, seed=1),
           "si216": lambda: si_system((3, 3, 3), sigma=0.05, seed=2),
           "water8": lambda: water_system(8, seed=4, cutoff=3.0, excess_proton=False),
           "water33": lambda: water_system(33, seed=6)}
# (columns per slice, CTAs per cluster, S in registers); 0, 0, -1: the library's choice
SHAPES = [(0, 0, -1), (1, 1, 0), (2, 3, 0), (4, 8, 0), (8, 2, 0), (2, 1, 1), (2, 4, 1), (4, 3, 1), (8, 8, 1), (2, 8, 1),
          (4, 16, 0), (2, 6, 0), (1, 16, 0), (2, 5, 0)]
PANEL = ("inner_spmv", "inner32_spmv", "inner32_cheb", "refine_residual", "outer_spmm")


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_1202_gb300 as pkg
    pkg.build()
    return pkg


def launches(P, call):
    n0 = {k: P.tb_profile_read(k)[0] for k in P.tb.KERNELS}
    out = call()
    n = {k: P.tb_profile_read(k)[0] - n0[k] for k in P.tb.KERNELS}
    return n["slice"], sum(n[k] for k in PANEL), out


def _grid(s, K):
    lo, hi = (-20.0, 5.0) if s.eps.min() > -20 else (-40.0, 0.0)
    return gauss_legendre_grid(K, lo, hi, 1.0)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_shapes_that_run(P, monkeypatch, name, prec):
    s = SYSTEMS[name]()
    h = P.tb_create_system(s)
    z, _ = _grid(s, 12)
    cols = np.linspace(0, s.n_orb - 1, 13).astype(np.int32)
    for nc, cl, reg in SHAPES:
        monkeypatch.setenv("TB_SLICE_NC", str(nc))
        monkeypatch.setenv("TB_SLICE_CL", str(cl))
        monkeypatch.setenv("TB_SLICE_REG", str(reg))
        opts = P.tb_default_opts(precision=prec, max_iter=20, panel=16)
        n, panel, _ = launches(P, lambda: P.tb_shifted_cocg(h, z, cols, opts=opts, allow_unconverged=True))
        # S in registers (mixed): at most 18 steps a stream and one row per
        # thread, so not water's longer rows, nor 864 rows on one CTA
        fits = not (prec == 1 and reg == 1 and (name == "water33" or (name == "si216" and cl == 1)))
        assert (n > 0, panel > 0) == (fits, not fits), (nc, cl, reg)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("cells,slices", [((3, 4, 6), True), ((5, 4, 4), False)])
def test_largest_system_of_the_slices(P, prec, cells, slices):
    """2304 orbitals run on the slices, 2560 on the panel kernels."""
    s = si_system(cells, sigma=0.05, seed=1)
    h = P.tb_create_system(s)
    z, w = _grid(s, 8)
    opts = P.tb_default_opts(precision=prec, max_iter=2)
    n, panel, _ = launches(P, lambda: P.tb_mulliken_orbital(h, z, w, [1, 700], 2.0, opts=opts, allow_unconverged=True))
    assert (n > 0, panel > 0) == (slices, not slices)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_hand_over_in_a_later_launch(P, prec):
    """Inner tolerances at the edge of what the slices' inner solves reach: the
    first launches of a call pass, a later one does not, and the panel kernels
    solve the columns again from their start."""
    s = SYSTEMS["si64"]()
    h = P.tb_create_system(s)
    z, _ = _grid(s, 4)
    S = s.dense_S()
    H = dense.ased_hamiltonian(S, s.eps, s.K, s.orbital_atom())
    # just below the tolerance that every inner solve reaches, only the worst one
    # fails, at some step of some launch: bisected for one set of columns after
    # another until that is not the first launch
    for first in range(8):
        cols = np.arange(first, s.n_orb, 11, dtype=np.int32)
        lo, hi = 2e-16, 1e-14
        for _ in range(24):
            tol = (lo * hi) ** 0.5
            opts = P.tb_default_opts(precision=prec, inner_tol=tol)
            n, panel, (x, st) = launches(P, lambda: P.tb_shifted_cocg(h, z, cols, opts=opts))
            assert n > 0 and st["status"] == "TB_OK"
            if n > 1 and panel > 0:
                G = np.transpose(dense.green_columns(H, S, z, cols), (0, 2, 1))
                assert np.abs(x.cpu().numpy() - G).max() <= 1e-8 * np.abs(G).max()
                return
            lo, hi = (lo, tol) if panel == 0 else (tol, hi)
    pytest.fail("no hand-over after the first launch")
