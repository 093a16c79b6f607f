"""tb_solve_opts.state_bytes bounds the device memory of full solutions, and
the default panel widths of the column slices hold no more than a call's
outputs need: peaks of the memory pool that the library allocates from."""
import ctypes

import numpy as np
import pytest

from tbinputs import gauss_legendre_grid, si_system, water_system

pytestmark = pytest.mark.gpu

USED_HIGH = 8     # CU_MEMPOOL_ATTR_USED_MEM_HIGH
MB = 1 << 20


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_1202_gb300 as pkg
    pkg.build()
    return pkg


@pytest.fixture(scope="module")
def peak():
    """peak(call): most bytes of the device's default memory pool in use during the call."""
    import torch
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool = ctypes.c_int(), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0

    def run(call):
        torch.cuda.synchronize()
        v = ctypes.c_uint64(0)
        assert cu.cuMemPoolSetAttribute(pool, USED_HIGH, ctypes.byref(v)) == 0
        out = call()
        torch.cuda.synchronize()
        assert cu.cuMemPoolGetAttribute(pool, USED_HIGH, ctypes.byref(v)) == 0
        return v.value, out

    return run


def launches(P):
    return {k: P.tb_profile_read(k)[0] for k in P.tb.KERNELS}


_CACHE = {}


def system(P, *cells):
    if cells not in _CACHE:
        s = si_system(cells, sigma=0.05, seed=1)
        _CACHE[cells] = s, P.tb_create_system(s)
    return _CACHE[cells]


def vectors(npad, columns):
    """Bytes of the inner solve's vectors: 7 of 8 bytes per element, 5 of 4, a split one of 8, and 1 MB of scalars."""
    return 84 * npad * columns + MB


def test_many_columns_in_flight(P, peak):
    """864 columns and a budget for some of the shifts of 256 columns: x^k, p^k of
    the panels in flight within it, the panels' solutions once more (half of it)."""
    import torch
    s, h = system(P, 3, 3, 3)
    z, _ = gauss_legendre_grid(64, -20.0, 5.0, 1.0)
    out = torch.empty((64, s.n_orb, s.n_orb), dtype=torch.complex128, device="cuda")
    budget = 256 * MB
    opts = P.tb_default_opts(precision=1, max_iter=4, state_bytes=budget)
    used, _ = peak(lambda: P.tb_shifted_cocg(h, z, np.arange(s.n_orb), opts=opts, out=out, allow_unconverged=True))
    assert used <= 1.5 * budget + vectors(s.n_orb, 256)


def test_one_column(P, peak):
    """A budget of exactly the shifts of one column: no partner column's state,
    and still one chunk (every chunk would solve the column again)."""
    s, h = system(P, 6, 6, 6)
    z, _ = gauss_legendre_grid(64, -20.0, 5.0, 1.0)
    budget = 64 * 32 * s.n_orb
    opts = P.tb_default_opts(precision=1, max_iter=3, state_bytes=budget)
    used, (_, st) = peak(lambda: P.tb_shifted_cocg(h, z, [17], opts=opts, allow_unconverged=True))
    assert used <= budget + vectors(s.n_orb, 2)
    assert st["outer_iterations"] == 3


def test_blocks_of_steps_count(P, peak):
    """A budget below the slices' sums of steps: the panel kernels, within it."""
    s, h = system(P, 2, 2, 2)
    z, _ = gauss_legendre_grid(16, -20.0, 5.0, 1.0)
    budget = 5 * 32 * s.n_orb * 4
    opts = P.tb_default_opts(precision=1, max_iter=600, state_bytes=budget)
    used, _ = peak(lambda: P.tb_shifted_cocg(h, z, [3, 77, 130, 201], opts=opts, allow_unconverged=True))
    assert used <= budget + vectors(s.n_orb, 4)


def test_projected_state_of_wide_panels(P, peak):
    """300 rows per column and 256 shifts with derivatives, 5 GB in four panels of
    256 columns: four of 64, the values and derivatives twice (recurrences, output
    order)."""
    s, h = system(P, 3, 3, 3)
    R, M, K = s.n_orb, 300, 256
    z, _ = gauss_legendre_grid(K, -20.0, 5.0, 1.0)
    rows = np.concatenate([(np.arange(M) * 2 + c) % s.n_orb for c in range(R)]).astype(np.int32)
    ptr = np.arange(R + 1, dtype=np.int64) * M
    opts = P.tb_default_opts(precision=1, max_iter=4)
    used, _ = peak(lambda: P.tb_green_elements_dz(h, z, np.arange(R), ptr, rows, opts=opts, allow_unconverged=True))
    assert used <= 4 * 64 * K * M * (64 + 32) + vectors(s.n_orb, 256) + 32 * MB


@pytest.mark.parametrize("which", ["full", "rows"])
def test_wide_calls_stay_on_the_slices(P, which):
    """256 columns whose steps fill a block of 128 MB in fewer than one launch's
    steps (full solutions of 512 atoms; derivatives at 256 shifts)."""
    n0 = launches(P)["slice"]
    if which == "full":
        s, h = system(P, 4, 4, 4)
        z, _ = gauss_legendre_grid(16, -20.0, 5.0, 1.0)
        P.tb_shifted_cocg(h, z, np.arange(256), opts=P.tb_default_opts(precision=1, max_iter=4), allow_unconverged=True)
    else:
        s, h = system(P, 3, 3, 3)
        z, _ = gauss_legendre_grid(256, -20.0, 5.0, 1.0)
        ptr = np.arange(257, dtype=np.int64) * 8
        rows = np.tile(np.arange(8, dtype=np.int32), 256)
        P.tb_green_elements_dz(h, z, np.arange(256), ptr, rows, opts=P.tb_default_opts(precision=1, max_iter=4),
                               allow_unconverged=True)
    assert launches(P)["slice"] > n0


def test_small_systems_beside_a_large_one_stay_on_the_slices(P):
    """A batch of a system that the slices take and one that they do not."""
    s, _ = system(P, 2, 2, 2)
    hb = P.tb_create_batch([s, water_system(400, seed=4, excess_proton=False)])
    hb_cols = [3, int(hb.orb_off[1]) + 5]
    z, _ = gauss_legendre_grid(8, -40.0, 0.0, 1.0)
    n0 = launches(P)
    P.tb_shifted_cocg(hb, z, hb_cols, opts=P.tb_default_opts(precision=1, max_iter=4), allow_unconverged=True)
    n1 = launches(P)
    assert n1["slice"] > n0["slice"] and n1["inner32_cheb"] > n0["inner32_cheb"]
