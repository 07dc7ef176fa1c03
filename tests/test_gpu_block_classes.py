"""H.psi at the sector sizes where its kernels change: tiles of 16 and 32 rows, 32 to 128
columns, odd remainders, stacks of tasks, and values that fixed point does not take.

The FP64 and FP32 products (Eq. dgemm) are compared with the operator oracle element by
element, relative to the largest element: 1e-12 (FP64) and 5e-6 (FP32 operators), the bounds
that tests/test_gpu_oracle_large.py derives for the same sums.
"""
import numpy as np
import pytest

from oracle import baseline
from oracle import dmrg as od
from paper_2001_04890_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def _grow(ctx, L, k, cap_left, cap_right, seed):
    """Blocks of k and L-2-k sites with at most cap states per sector of the last one."""
    rng = np.random.default_rng(seed)

    def step(direction, cap):
        lay = ctx.enlarged_layout(direction)
        kept = [min(int(d), cap) for _, _, d in lay]
        O = np.concatenate([workloads.orthonormal_columns(int(d), m, rng).ravel() for (_, _, d), m in zip(lay, kept)])
        ctx.renormalize(direction, O, kept)

    ctx.set_position(0, 1)
    for s in range(k):
        step(+1, cap_left if s == k - 1 else 10**6)
    ctx.set_position(L - 2, -1)
    for s in range(L - 1, k + 1, -1):
        step(-1, cap_right if s == k + 2 else 10**6)
    ctx.set_position(k, 1)


_CACHE = {}


def _oracle(L, caps):
    key = (L, caps)
    if key not in _CACHE:
        _CACHE.clear()
        h, v = workloads.integrals(L, seed=3)
        b = baseline.OracleBuilder(h, v)
        _grow(b, L, (L - 2) // 2, *caps, seed=4)
        lb, rb = b._blocks()
        _CACHE[key] = od.HPsi(b.I, (L - 2) // 2, lb, rb, L // 2, L // 2)
    return _CACHE[key]


def _context(L, caps, prec):
    h, v = workloads.integrals(L, seed=3)
    ctx = binding.DMRG(h, v, L, 0, 10**6, precision=prec)
    _grow(ctx, L, (L - 2) // 2, *caps, seed=4)
    return ctx


def _close(a, ref, tol):
    return np.max(np.abs(a - ref)) <= tol * np.max(np.abs(ref))


SMALL = [(10, c) for c in [(1, 1), (1, 33), (7, 9), (8, 8), (16, 16), (16, 17), (17, 16), (9, 25), (24, 8), (16, 20), (20, 15), (15, 28), (31, 33), (32, 32), (36, 5)]]
LARGE = [(12, c) for c in [(33, 64), (65, 63), (96, 97), (100, 100)]]


@pytest.mark.parametrize("L,caps", SMALL + LARGE)
def test_hpsi_at_tile_edges(L, caps):
    hp = _oracle(L, caps)
    x = workloads.gaussian(hp.dim, seed=5)
    ref = hp.apply(x)
    for prec, tol in ((binding.PREC_FP64, 1e-12), (binding.PREC_FP32, 5e-6)):
        ctx = _context(L, caps, prec)
        assert ctx.psi_layout()[1] == hp.dim
        assert _close(ctx.hpsi(x), ref, tol)
        for wide, chunks in ((0, 8192.0), (1, 1.0)):  # one group per chunk; one chunk per block
            ctx.set_tune(target_chunks=chunks, min_chunk=0.0, flat_wide=wide)
            assert _close(ctx.hpsi(x), ref, tol)
        ctx.close()


@pytest.mark.parametrize("scale", [2.0**300, 2.0**-300, 1.0])
def test_values_outside_fixed_point(scale):
    """Psi blocks of very large or small values, and of both, take the FP64 products."""
    L, caps = 10, (17, 16)
    hp = _oracle(L, caps)
    ctx = _context(L, caps, binding.PREC_FP64)
    x = workloads.gaussian(hp.dim, seed=6)
    if scale == 1.0:  # every other block tiny, against the linear combination of the two
        blocks, _ = ctx.psi_layout()
        mask = np.zeros(hp.dim, dtype=bool)
        for b in blocks[::2]:
            mask[b[6]:b[6] + b[4] * b[5]] = True
        y = np.where(mask, x * 2.0**-400, x)
        assert _close(ctx.hpsi(y), hp.apply(np.where(mask, 0.0, x)), 1e-12)
        assert _close(ctx.hpsi(np.where(mask, x, 0.0) * 2.0**-400), hp.apply(np.where(mask, x, 0.0)) * 2.0**-400, 1e-12)
    else:
        assert _close(ctx.hpsi(x * scale), hp.apply(x) * scale, 1e-12)
    ctx.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_propagate(bad):
    """A NaN or infinity in one psi block reaches the blocks that H couples to it and no other."""
    L, caps = 10, (9, 8)
    hp = _oracle(L, caps)
    ctx = _context(L, caps, binding.PREC_FP64)
    x = workloads.gaussian(hp.dim, seed=7)
    blocks, _ = ctx.psi_layout()
    b = blocks[len(blocks) // 2]
    e = np.zeros(hp.dim)
    e[b[6]:b[6] + b[4] * b[5]] = workloads.gaussian(b[4] * b[5], seed=8)
    clean = hp.apply(x)
    x[b[6] + 1] = bad
    y = ctx.hpsi(x)
    reached = hp.apply(e) != 0.0
    assert not np.isfinite(y[b[6]:b[6] + b[4] * b[5]]).any()
    assert np.max(np.abs(y[~reached] - clean[~reached]), initial=0.0) <= 1e-12 * np.max(np.abs(clean))
    ctx.close()
