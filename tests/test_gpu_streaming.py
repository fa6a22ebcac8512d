"""The streaming, tiled and cooperative kernels (bq_tune resident = 0), which states outside the resident
kernels' forms and sizes take: the schedule, tiling, solve and gradient tests of the other files on states
that start with the resident kernels switched off."""

import pytest

import test_gpu_batched
import test_gpu_grad
import test_gpu_parity
import test_gpu_rdiag
import test_gpu_secular
import test_gpu_tune
from parity import gpu_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    from paper_2203_05526_gb300 import build
    build.build()
    assert torch.cuda.is_available()


CASES = [
    (test_gpu_tune, "test_every_step_schedule_computes_the_same_step", dict(n=64)),
    (test_gpu_tune, "test_every_step_schedule_computes_the_same_step", dict(n=2000)),
    (test_gpu_tune, "test_solve_kernels_agree_and_tuned_solve_matches_streaming", {}),
    (test_gpu_tune, "test_tile_lengths_compute_the_same_step_and_gradients", {}),
    (test_gpu_tune, "test_lanes_per_point_split_the_same_sums", dict(n_modes=2)),
    (test_gpu_tune, "test_lanes_per_point_split_the_same_sums", dict(n_modes=3)),
    (test_gpu_batched, "test_solve_f64_ragged_batch_matches_oracle_per_system", {}),
    (test_gpu_batched, "test_solve_equals_streamed_stages", dict(dtype="f64", tol=1e-12)),
    (test_gpu_batched, "test_solve_equals_streamed_stages", dict(dtype="f32", tol=1e-6)),
    (test_gpu_batched, "test_solve_f32_every_envelope_kind_matches_stepping_and_oracle", dict(reverse=True)),
    (test_gpu_batched, "test_solve_f32_every_envelope_kind_matches_stepping_and_oracle", dict(reverse=False)),
    (test_gpu_batched, "test_solve_split_calls_and_time", {}),
    (test_gpu_parity, "test_graph_path_and_split_calls", {}),
    (test_gpu_parity, "test_two_mode_multi_tile_matches_oracle", {}),
    (test_gpu_parity, "test_three_modes_with_halo_beyond_shared_memory", {}),
    (test_gpu_parity, "test_three_modes_global_read_gradients_match_oracle_adjoint", {}),
    (test_gpu_parity, "test_separable_only_layout_matches_oracle", dict(n_modes=2, N=5)),
    (test_gpu_parity, "test_separable_only_layout_matches_oracle", dict(n_modes=3, N=4)),
    (test_gpu_secular, "test_two_modes_match_oracle", {}),
    (test_gpu_secular, "test_batch_schedules_and_persistent_solves", {}),
    (test_gpu_rdiag, "test_two_coupled_modes_diag_layout_matches_oracle", {}),
    (test_gpu_rdiag, "test_diag_layout_gradients_match_oracle_adjoint", dict(n_modes=2)),
    (test_gpu_grad, "test_grad_matches_oracle_adjoint", dict(n_modes=2, N=4, ck=24)),
    (test_gpu_grad, "test_grad_cooperative_segments_match_per_stage_launches_and_oracle", dict(ck=7)),
    (test_gpu_grad, "test_grad_recorded_segments_skip_recomputation", dict(record_segments=3)),
    (test_gpu_grad, "test_grad_cooperative_segments_with_more_items_than_ctas", {}),
]


@pytest.mark.parametrize("module,name,kw", CASES, ids=[f"{n}-{'-'.join(str(v) for v in k.values())}" for _, n, k in CASES])
def test_without_the_resident_kernels(monkeypatch, module, name, kw):
    made = []

    def state(*a, **k):
        st = gpu_state(*a, **k)
        st.set_tune(resident=0)
        assert st.get_tune()["resident"] == 0
        made.append(st)
        return st

    monkeypatch.setattr(module, "gpu_state", state)
    getattr(module, name)(**kw)
    assert made


def test_the_resident_kernels_match_the_streaming_ones():
    """What the file above runs and the default: two kernels' roundings over a few steps."""
    import numpy as np
    ps = test_gpu_tune._batch(n=64)
    a, b = gpu_state(ps, dtype="f32"), gpu_state(ps, dtype="f32")
    assert a.get_tune()["resident"] == 1
    b.set_tune(resident=0)
    a.step(ps[0].dt, 12)
    b.step(ps[0].dt, 12)
    ea, eb = a.evaluate(), b.evaluate()
    assert np.max(np.abs(ea - eb)) <= 1e-6 * max(1.0, np.max(np.abs(eb)))
