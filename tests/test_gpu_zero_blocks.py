"""Operator and psi blocks of zeros beside values of any scale.

The FP64 products give every tile one exponent and make scale factors of them, and a tile of
zeros has none of its own.  Such blocks are ordinary: tasks follow symmetry and not values, and H
of a block's vacuum sector is one.  Powers of two only move exponents, so results must be the
same bits at every scale.
"""
import numpy as np
import pytest

from paper_2001_04890_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prepared", [True, False])
@pytest.mark.parametrize("m,n,p,q", [(3, 5, 4, 6), (20, 40, 33, 18), (40, 70, 50, 70)])
@pytest.mark.parametrize("zero", ["X", "Y", "Z"])
def test_a_zero_operand_adds_nothing(zero, m, n, p, q, prepared):
    """The task with the zero block leaves the other one's result as it is."""
    rng = np.random.default_rng(1)
    X, Y, Z = rng.standard_normal((2, m, n)), rng.standard_normal((n, p)), rng.standard_normal((2, p, q))
    f = np.array([1.0, -1.0])
    if zero == "Y":
        Y[:] = 0.0
    else:
        {"X": X, "Z": Z}[zero][0] = 0.0
    base = binding.selftest_chain(X[1:], Y, Z[1:], f[1:], prepared=prepared)
    assert np.isfinite(base).all() and (zero == "Y" or np.abs(base).max() > 1.0)
    for s in range(-150, 151):
        if zero == "Y":  # large and small operators
            D = binding.selftest_chain(np.ldexp(X, s), Y, np.ldexp(Z, s // 2), f, prepared=prepared)
            assert np.array_equal(D, np.zeros((m, q)))
        else:
            D = binding.selftest_chain(X, np.ldexp(Y, s), Z, f, prepared=prepared)
            assert np.array_equal(D, np.ldexp(base, s)), s


@pytest.mark.parametrize("prepared", [True, False])
@pytest.mark.parametrize("identity", ["X", "Z", "both"])
def test_identities_beside_zeros(identity, prepared):
    rng = np.random.default_rng(2)
    m, q = 13, 13
    Y = rng.standard_normal((m, q))
    X = None if identity != "Z" else np.zeros((1, m, m))
    Z = None if identity != "X" else np.zeros((1, q, q))
    for s in range(-150, 151):
        D = binding.selftest_chain(X, np.ldexp(Y, s), Z, [1.0], prepared=prepared)
        ref = np.ldexp(Y, s) if identity == "both" else np.zeros((m, q))
        assert np.max(np.abs(D - ref)) <= 2.0**-52 * np.max(np.abs(ref)), s  # Y to 58 bits of its largest


@pytest.mark.parametrize("first", [True, False])
def test_a_zero_tile_does_not_move_the_other_chunks(first):
    """The sum over an inner dimension of several tiles of 32: a tile of zeros that meets large
    values leaves the sum over small ones as exact as it is alone."""
    rng = np.random.default_rng(3)
    m, n, p, q = 18, 64, 20, 17
    X, Y, Z = rng.standard_normal((1, m, n)), rng.standard_normal((n, p)), rng.standard_normal((1, p, q))
    z, v = (slice(0, 32), slice(32, 64)) if first else (slice(32, 64), slice(0, 32))
    X[:, :, z] = 0.0
    Y[z] *= 2.0**200
    Y[v] *= 2.0**-200
    D = binding.selftest_chain(X, Y, Z, [1.0], prepared=False)
    ref = X[0][:, v] @ Y[v] @ Z[0]
    assert np.max(np.abs(D - ref)) <= 1e-14 * np.max(np.abs(ref))


def _context(prec):
    L, M = 8, 64
    h, v = workloads.integrals(L, seed=0)
    ctx = binding.DMRG(h, v, L, 0, M, precision=prec)
    workloads.grow_middle_bond(ctx, L, L // 2, L // 2, M, (L - 2) // 2, seed=0)
    for side in (0, 1):  # both blocks have a vacuum sector, whose H is zero
        assert (0, 0) in {(int(a), int(b)) for a, b, _ in ctx.block_sectors(side)}
    return ctx


@pytest.mark.parametrize("prec", [binding.PREC_FP64, binding.PREC_BF16X3])
def test_hpsi_at_every_scale(prec):
    """H (2^s x) = 2^s H x, bit for bit (blocks of at most 32 states run in FP64 in both modes)."""
    import torch
    ctx = _context(prec)
    _, dim = ctx.psi_layout()
    x = workloads.gaussian(dim, seed=1)
    y = ctx.hpsi(x)
    batch = binding.Batch([ctx])
    yb = batch.hpsi(x)
    sigma = torch.empty(dim, dtype=torch.float64, device="cuda")
    for s in range(-150, 151):
        xs = np.ldexp(x, s)
        assert np.array_equal(ctx.hpsi(xs), np.ldexp(y, s)), s
        assert np.array_equal(batch.hpsi(xs), np.ldexp(yb, s)), s
        ctx.hpsi_noalloc(torch.from_numpy(xs).cuda(), sigma)
        assert np.array_equal(sigma.cpu().numpy(), np.ldexp(y, s)), s
    batch.close()
    ctx.close()


def test_zero_psi_blocks_beside_large_operators():
    """A psi of one block: the others are zero, whatever the scale of the Hamiltonian."""
    L = 6
    h, v = workloads.integrals(L, seed=0)
    ref = None
    for s in range(0, 101, 2):
        ctx = binding.DMRG(np.ldexp(h, s), np.ldexp(v, s), L, 0, 40)
        workloads.grow_middle_bond(ctx, L, L // 2, L // 2, 40, 2, seed=0)
        blocks, dim = ctx.psi_layout()
        x = np.zeros(dim)
        b = blocks[len(blocks) // 2]
        x[b[6]:b[6] + b[4] * b[5]] = workloads.gaussian(int(b[4] * b[5]), seed=2)
        y = np.ldexp(ctx.hpsi(x), -s)
        ref = y if ref is None else ref
        assert np.max(np.abs(y - ref)) <= 1e-13 * np.max(np.abs(ref)), s
        ctx.close()
