"""The panel kernels against the dense and method oracles on small systems: the
checks of test_gpu_parity, test_gpu_adjoint, test_gpu_csc, test_gpu_batch and
test_gpu_slices once more with TB_SLICE=0, where by default the column slices
answer -- solutions, rows with derivatives, populations, vector-Jacobian
product, charge self-consistency, batches, step graphs, autotuner."""
import os
import subprocess
import sys

import numpy as np
import pytest

from test_gpu_adjoint import (si, test_band_energy_and_gradients, test_green_elements_dz_dense,  # noqa: F401
                              test_green_elements_dz_fixed_steps_match_method, test_mulliken_vjp)
from test_gpu_batch import (grid, systems, test_autotune_choice_is_used, test_batch_charges_equal_per_system,  # noqa: F401
                            test_batch_green_elements_and_stats, test_step_graphs_on_a_ragged_batch)
from test_gpu_csc import test_csc_loop_matches_oracle, w8, w8_loop  # noqa: F401
from test_gpu_parity import (P, c1, c1_mulliken, c1_ref, h1, prec, test_fixed_iterations_match_method_oracle,  # noqa: F401
                             test_full_mode_c1, test_graph_and_direct_launches_agree, test_green_elements,
                             test_max_shift_count, test_mulliken_orbital, test_non_identity_diagonal_blocks,
                             test_panel_split_with_ragged_tail, test_single_shift_single_column,
                             test_water_ragged_blocks)
from test_gpu_slices import small, test_outputs_against_dense  # noqa: F401

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(autouse=True)
def panel_kernels(P, monkeypatch):  # noqa: F811
    monkeypatch.setenv("TB_SLICE", "0")
    count = lambda: {k: P.tb_profile_read(k)[0] for k in ("slice", "outer_spmm")}
    before = count()
    yield
    after = count()
    assert after["slice"] == before["slice"] and after["outer_spmm"] > before["outer_spmm"]


def test_ragged_and_padded_forms_agree(P, tmp_path):  # noqa: F811
    """The ragged four-pair Chebyshev step and the ragged double-float products
    (exact orbital counts) against the padded ones: these only add exact zeros in
    the same order, so the populations are bit-identical, on one box and on a
    ragged batch.  Each form in a process of its own, where the counters say that
    its steps ran."""
    child = ("import sys, numpy as np, paper_1002_1202_gb300 as P\n"
             "from tests.test_gpu_batch import _batch_case\n"
             "systems, z, w = _batch_case()\n"
             "q = [P.tb_mulliken_charges(h, z, w, opts=P.tb_default_opts(precision=1))[0].cpu().numpy()\n"
             "     for h in (P.tb_create_batch(systems), P.tb_create_system(systems[2]))]\n"
             "assert P.tb_profile_read('slice')[0] == 0 and P.tb_profile_read('inner32_cheb')[0] > 0\n"
             "np.savez(sys.argv[1], *q)\n")
    q = []
    for rag in ("1", "0"):
        out = tmp_path / f"q{rag}.npz"
        env = dict(os.environ, TB_SLICE="0", TB_CHEB_CPT="4", TB_CHEB_RAG=rag, TB_DF_RAG=rag, PYTHONPATH=ROOT)
        subprocess.run([sys.executable, "-c", child, str(out)], env=env, cwd=ROOT, check=True, timeout=600)
        q.append(np.load(out))
    for k in q[0].files:
        assert np.array_equal(q[0][k], q[1][k])
    z, w = np.array([-13.0 + 1j]), np.array([1.0])     # this process runs the panel kernels too
    P.tb_mulliken_orbital(P.tb_create([4], [0, 1], [0], np.eye(4).ravel(), None, -np.arange(5.0, 9.0), 1.75), z, w, [0])
