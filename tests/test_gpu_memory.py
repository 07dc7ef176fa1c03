"""Device memory that runs short: the prepared operands of H.psi are an option, their list entries
and images give way.

Failures are injected on the host (dmrg_debug_fail_alloc: the n-th device allocation from now
fails); the n that are not for prepared operands return DMRG_ENOMEM, as in test_gpu_failure.py.
"""
import numpy as np
import pytest

from paper_2001_04890_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

L, M = 8, 48
TOL = {binding.PREC_FP64: 1e-12, binding.PREC_FP32: 5e-6, binding.PREC_BF16X3: 1e-12}  # no side above 32: FP64


def _context(prec):
    h, v = workloads.integrals(L, seed=1)
    ctx = binding.DMRG(h, v, L, 0, M, precision=prec)
    workloads.grow_middle_bond(ctx, L, L // 2, L // 2, M, 3, seed=1)
    return ctx


@pytest.fixture(autouse=True)
def disarmed():
    yield
    binding.debug_fail_alloc(0)


def _launches(ctx, x):
    """Kernels of one H.psi: the prepared operands take one for psi more than the general kernels."""
    ctx.stats(reset=True)
    ctx.hpsi(x)
    return ctx.stats()["kernel_launches"]


@pytest.mark.parametrize("prec", [binding.PREC_FP64, binding.PREC_FP32, binding.PREC_BF16X3])
def test_every_allocation_of_the_plan_may_fail(prec):
    """H.psi is right without the memory of the prepared operands, and after DMRG_ENOMEM for other memory."""
    ctx = _context(prec)
    x = workloads.gaussian(ctx.psi_layout()[1], seed=3)
    ref, whole = ctx.hpsi(x), _launches(ctx, x)
    ctx.close()
    general, untouched = 0, 0
    for n in range(1, 200):
        c = _context(prec)
        binding.debug_fail_alloc(n)
        try:
            y = c.hpsi(x)
        except binding.DMRGError as err:
            assert err.code == binding.DMRG_ENOMEM
            y = None
        binding.debug_fail_alloc(0)
        assert np.max(np.abs(c.hpsi(x) - ref)) <= TOL[prec] * np.max(np.abs(ref)), n
        k = _launches(c, x)
        assert k <= whole
        if y is not None:
            assert np.max(np.abs(y - ref)) <= TOL[prec] * np.max(np.abs(ref)), n
            general += k < whole
            untouched = untouched + 1 if k == whole else 0
        c.close()
        if untouched >= 12:
            break  # past the last allocation
    assert general >= 6  # images, exponents, slabs, identities; psi spans and images, entries, stacks
