"""Autotuning of FP32 lists leaves flat_wide alone: FP32 chunks are never shared, so that timing its
two values would record noise as a choice."""
import pytest

from paper_2001_04890_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [0, 1])
def test_flat_wide_is_not_tuned_in_fp32(wide):
    L, M = 8, 48
    h, v = workloads.integrals(L, seed=1)
    ctx = binding.DMRG(h, v, L, 0, M, precision=binding.PREC_FP32)
    workloads.grow_middle_bond(ctx, L, L // 2, L // 2, M, 3, seed=1)
    for _ in range(8):
        ctx.set_tune(flat_wide=wide)
        assert ctx.autotune(reps=1)[1]["flat_wide"] == wide
    ctx.close()
