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


def _failing(call):
    """The call with its first device allocation failing."""
    binding.debug_fail_alloc(1)
    try:
        return call()
    finally:
        binding.debug_fail_alloc(0)


@pytest.mark.parametrize("prec", [binding.PREC_FP64, binding.PREC_FP32, binding.PREC_BF16X3])
def test_images_are_given_back_when_a_call_needs_the_memory(prec):
    """The calls after H.psi allocate beside the images: one failure takes those, not the call."""
    ctx = _context(prec)
    x = workloads.gaussian(ctx.psi_layout()[1], seed=3)
    calls = {"hpsi": lambda c: c.hpsi(x), "set_psi": lambda c: (c.set_psi(x), c.get_psi())[1],
             "davidson": lambda c: (c.set_psi(x), c.davidson(1e-9, 400)[0])[1]}
    ref, whole = ctx.hpsi(x), _launches(ctx, x)
    energy = calls["davidson"](ctx)
    ctx.close()
    for name, call in calls.items():
        c = _context(prec)
        c.hpsi(x)
        if name == "davidson":
            c.set_psi(x)
        y = _failing(lambda: call(c))
        assert np.max(np.abs(y - {"hpsi": ref, "set_psi": x, "davidson": energy}[name])) <= TOL[prec] * np.max(np.abs(ref)), name
        assert np.max(np.abs(c.hpsi(x) - ref)) <= TOL[prec] * np.max(np.abs(ref))
        assert _launches(c, x) < whole  # the general kernels
        c.set_position(2, 1)
        c.set_position(3, 1)  # planned again, with images
        c.hpsi(x)
        assert _launches(c, x) == whole
        c.close()


def test_renormalization_gives_images_back():
    ctx = _context(binding.PREC_FP64)
    x = workloads.gaussian(ctx.psi_layout()[1], seed=3)
    rng = np.random.default_rng(5)
    kept = [min(int(d), 6) for _, _, d in ctx.enlarged_layout(1)]
    O = np.concatenate([workloads.orthonormal_columns(int(d), m, rng).ravel()
                        for (_, _, d), m in zip(ctx.enlarged_layout(1), kept)])
    out = []
    for fail in (False, True):
        c = _context(binding.PREC_FP64)
        c.hpsi(x)
        (_failing if fail else lambda f: f())(lambda: c.renormalize(1, O, kept))
        out.append(c.hpsi(workloads.gaussian(c.psi_layout()[1], seed=4)))
        c.close()
    ctx.close()
    assert np.array_equal(out[0], out[1])


def test_a_new_position_gives_the_old_images_back():
    """Any one allocation of the next position's plan may fail while the old position's images are there."""
    ctx = _context(binding.PREC_FP64)
    x = workloads.gaussian(ctx.psi_layout()[1], seed=3)
    lay = ctx.enlarged_layout(1)
    rng = np.random.default_rng(5)
    O = np.concatenate([workloads.orthonormal_columns(int(d), min(int(d), 6), rng).ravel() for _, _, d in lay])
    ctx.close()
    ref = None
    for n in [0] + list(range(1, 40)):
        c = _context(binding.PREC_FP64)
        c.hpsi(x)
        c.renormalize(1, O, [min(int(d), 6) for _, _, d in lay])
        z = workloads.gaussian(c.psi_layout()[1], seed=4)
        binding.debug_fail_alloc(n)
        y = c.hpsi(z)
        binding.debug_fail_alloc(0)
        ref = y if ref is None else ref
        assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref)), n
        c.close()


def test_a_batch_keeps_its_contexts_images():
    ctx = _context(binding.PREC_FP64)
    x = workloads.gaussian(ctx.psi_layout()[1], seed=3)
    batch = binding.Batch([ctx])
    y = batch.hpsi(x)
    whole = _launches(ctx, x)
    _failing(lambda: ctx.hpsi(x))
    assert _launches(ctx, x) < whole
    assert np.array_equal(batch.hpsi(x), y) and np.array_equal(batch.hpsi(x), y)
    batch.autotune(reps=1)
    assert np.max(np.abs(batch.hpsi(x) - y)) <= 1e-12 * np.max(np.abs(y))
    batch.close()
    ctx.close()


def test_a_captured_call_keeps_its_images():
    """A graph of dmrg_hpsi_noalloc outlives the call: its images are not given back under it."""
    import torch
    stream = torch.cuda.Stream()
    h, v = workloads.integrals(L, seed=1)
    ctx = binding.DMRG(h, v, L, 0, M, stream=stream.cuda_stream)
    workloads.grow_middle_bond(ctx, L, L // 2, L // 2, M, 3, seed=1)
    x = workloads.gaussian(ctx.psi_layout()[1], seed=3)
    ref = ctx.hpsi(x)
    with torch.cuda.stream(stream):
        psi = torch.from_numpy(x).cuda()
        sigma = torch.empty_like(psi)
        ctx.hpsi_noalloc(psi, sigma)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.hpsi_noalloc(psi, sigma)
    with pytest.raises(binding.DMRGError) as err:
        _failing(lambda: ctx.hpsi(x))
    assert err.value.code == binding.DMRG_ENOMEM
    sigma.zero_()
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(sigma.cpu().numpy(), ref)
    ctx.close()


def test_a_batch_takes_a_third_of_the_free_memory_for_images():
    """Not a third of what the members before left.  The rest of the device is filled for the second batch."""
    import torch
    h, v = workloads.integrals(16, seed=0)

    def members():
        out = []
        for n in range(4):
            c = binding.DMRG(h, v, 16, 0, 256, precision=binding.PREC_BF16X3)
            workloads.grow_middle_bond(c, 16, 8, 8, 256, 7, seed=n)
            c.set_tune(tc_min=1)  # their own lists need no images, the batch's (its own launch shape) do
            c.hpsi_flops()
            out.append(c)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        return out, torch.cuda.mem_get_info()[0]

    def images_of_a_batch(ctxs, free):
        batch = binding.Batch(ctxs)
        x = workloads.gaussian(batch.offsets[-1], seed=1)
        y = batch.hpsi(x)
        batch.close()  # what stays are the members' images
        return free - torch.cuda.mem_get_info()[0], y

    ctxs, free = members()
    images, ref = images_of_a_batch(ctxs, free)
    for c in ctxs:
        c.close()
    assert images > 2**27
    ctxs, free = members()
    left = int(2.5 * images)
    filler = torch.empty(free - left, dtype=torch.uint8, device="cuda")
    taken, y = images_of_a_batch(ctxs, torch.cuda.mem_get_info()[0])
    del filler
    torch.cuda.empty_cache()
    for c in ctxs:
        c.close()
    assert taken <= left / 3
    assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))
