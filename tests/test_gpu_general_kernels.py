"""H.psi without prepared operands: the general kernels take the lists whose images find no memory
and those with an inner dimension above 120.

Against the operator oracle, relative to the largest element: 1e-12 (FP64) and 5e-6 (FP32
operators), the bounds that tests/test_gpu_oracle_large.py derives for the same sums.
"""
import numpy as np
import pytest

from oracle import baseline
from oracle import dmrg as od
from paper_2001_04890_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

TOL = {binding.PREC_FP64: 1e-12, binding.PREC_FP32: 5e-6}


def _grow(ctx, L, k, caps, most, seed):
    """Blocks of k and L-2-k sites, at most `most` electrons of a spin, at most caps states in a
    sector of the last step."""
    rng = np.random.default_rng(seed)

    def step(direction, cap):
        lay = ctx.enlarged_layout(direction)
        kept = [min(int(d), cap) if u <= most and n <= most else 0 for u, n, d in lay]
        O = np.concatenate([workloads.orthonormal_columns(int(d), m, rng).ravel() for (_, _, d), m in zip(lay, kept)])
        ctx.renormalize(direction, O, kept)

    ctx.set_position(0, 1)
    for s in range(k):
        step(+1, caps[0] if s == k - 1 else 10**6)
    ctx.set_position(L - 2, -1)
    for s in range(L - 1, k + 1, -1):
        step(-1, caps[1] if s == k + 2 else 10**6)
    ctx.set_position(k, 1)


_CACHE = {}


def _oracle(L, k, electrons, caps):
    key = (L, k, electrons, caps)
    if key not in _CACHE:
        _CACHE.clear()
        h, v = workloads.integrals(L, seed=3)
        b = baseline.OracleBuilder(h, v)
        _grow(b, L, k, caps, electrons // 2, seed=4)
        _CACHE[key] = od.HPsi(b.I, k, *b._blocks(), electrons // 2, electrons // 2)
    return _CACHE[key]


def _context(L, k, electrons, caps, prec):
    h, v = workloads.integrals(L, seed=3)
    ctx = binding.DMRG(h, v, electrons, 0, 10**6, precision=prec)
    _grow(ctx, L, k, caps, electrons // 2, seed=4)
    return ctx


def _launches(ctx, x):
    ctx.stats(reset=True)
    ctx.hpsi(x)
    return ctx.stats()["kernel_launches"]


def _without_images(ctx, x):
    """H.psi once with its first allocation failing: the context gives its images back."""
    before = _launches(ctx, x)
    binding.debug_fail_alloc(1)
    try:
        ctx.hpsi(x)
    finally:
        binding.debug_fail_alloc(0)
    assert _launches(ctx, x) < before  # no images of psi


CASES = [(10, 4, 10, c) for c in [(1, 33), (7, 9), (16, 16), (16, 17), (17, 16), (24, 8), (31, 33), (32, 32)]] + \
        [(12, 5, 12, c) for c in [(33, 64), (65, 63), (100, 100)]] + [(12, 6, 4, c) for c in [(119, 36), (120, 30)]]


@pytest.mark.parametrize("L,k,electrons,caps", CASES)
def test_general_kernels_at_tile_edges(L, k, electrons, caps):
    hp = _oracle(L, k, electrons, caps)
    x = workloads.gaussian(hp.dim, seed=5)
    ref = hp.apply(x)
    for prec, tol in TOL.items():
        ctx = _context(L, k, electrons, caps, prec)
        for wide, chunks in ((1, 8192.0), (0, 8192.0), (1, 1.0)):
            ctx.set_tune(target_chunks=chunks, min_chunk=2e5 if chunks > 1 else 0.0, flat_wide=wide)
            assert np.max(np.abs(ctx.hpsi(x) - ref)) <= tol * np.max(np.abs(ref))
            _without_images(ctx, x)
            assert np.max(np.abs(ctx.hpsi(x) - ref)) <= tol * np.max(np.abs(ref))
        ctx.close()


@pytest.mark.parametrize("caps", [(121, 36), (150, 20), (225, 36)])
def test_long_inner_dimensions(caps):
    """Lists that the prepared kernels do not take; no images are made for them."""
    hp = _oracle(12, 6, 4, caps)
    x = workloads.gaussian(hp.dim, seed=5)
    ref = hp.apply(x)
    for prec, tol in TOL.items():
        ctx = _context(12, 6, 4, caps, prec)
        assert max(int(d) for _, _, d in ctx.block_sectors(0)) == min(caps[0], 225)
        assert np.max(np.abs(ctx.hpsi(x) - ref)) <= tol * np.max(np.abs(ref))
        binding.debug_fail_alloc(1)
        try:
            with pytest.raises(binding.DMRGError) as err:  # nothing to give back
                ctx.hpsi(x)
        finally:
            binding.debug_fail_alloc(0)
        assert err.value.code == binding.DMRG_ENOMEM
        assert np.max(np.abs(ctx.hpsi(x) - ref)) <= tol * np.max(np.abs(ref))
        ctx.close()
