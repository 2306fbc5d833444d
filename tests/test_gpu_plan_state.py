"""The plan's device state: explicit preparation (after which compute calls can be captured without a warm call) and
the reporting of a bounded device-side wait that ran out."""
import numpy as np
import pytest
import torch

from oracle import kvq_oracle as ko
from paper_2605_05699_b200 import binding as kb
from paper_2605_05699_b200 import workloads as wl
from tests import parity

pytestmark = pytest.mark.gpu

G = wl.GROUP
DT = {"f16": ko.F16, "bf16": ko.BF16}


@pytest.mark.parametrize("D,dtype,N", [(128, "f16", 6000), (256, "bf16", 3000), (96, "f16", 700)])
def test_prepared_plan_is_captured_without_a_warm_call(D, dtype, N):
    """A stream capture refuses allocations and blocking copies.  After kvq_plan_prepare the very first encode, append and
    decode of a plan are recorded into a CUDA graph as they are; the replay must give what the oracle gives."""
    tdt = wl.torch_dtype(dtype)
    plan = kb.Plan(D, G, 400 + D)
    sg = plan.signs()
    x = wl.make_vectors(N, D, dtype, "k_outlier", 401)
    lam = wl.make_lambda(2, D, 402)
    rpl = (N + 1) // 2
    xd, lamd = x.cuda(), lam.cuda()
    packed, scales = plan.empty_packed(N).zero_(), plan.empty_scales(N).zero_()
    out = torch.zeros(N, D, dtype=tdt, device="cuda")
    cache_p = torch.zeros(4, 3, D // 2, dtype=torch.uint8, device="cuda")
    cache_s = torch.zeros(4, 3, D // G, dtype=torch.float16, device="cuda")
    assert plan.describe()[1] == 0
    kb.kvq_plan_prepare(plan.handle, tdt)
    assert plan.describe()[1] > 0                      # the tables exist now
    kb.kvq_plan_prepare(plan.handle, tdt)              # idempotent
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        kb.kvq_encode(plan.handle, xd, lamd, packed, scales, rpl)
        kb.kvq_append(plan.handle, xd[:4], lamd, cache_p, cache_s, 1, 2)
        kb.kvq_decode(plan.handle, packed, scales, lamd, out, rpl)
    graph.replay()
    torch.cuda.synchronize()
    assert kb.kvq_plan_device_status(plan.handle) == 0
    ora = ko.encode(wl.raw_bits(x), DT[dtype], sg, lam.numpy(), G, rpl, want_v=True)
    pk, sb = packed.cpu().numpy(), wl.raw_bits(scales)
    parity.check_encode(pk, sb, ora, G, "captured encode", min_agree=0.9995 if N * D < 500000 else parity.CODE_AGREEMENT)
    ob, o64 = ko.decode(pk, sb, sg, lam.numpy(), G, DT[dtype], rpl, want_f64=True)
    parity.check_decode(wl.raw_bits(out), ob, o64, DT[dtype], "captured decode")
    assert bool((cache_p[:, 1] != 0).any()) and not bool(cache_p[:, [0, 2]].any())
    plan.close()


def inverse_transform(D):
    """The rotation that undoes the transform: the plan's forward table becomes the sign diagonal, entries of 1 among zeros."""
    n, k = np.arange(D), np.arange(1, D // 2)
    m = np.empty((D, D))
    m[0], m[D // 2] = D ** -0.5, (-1.0) ** n * D ** -0.5
    m[1:D // 2] = np.sqrt(2 / D) * np.cos(2 * np.pi * np.outer(k, n) / D)
    m[D // 2 + 1:] = -np.sqrt(2 / D) * np.sin(2 * np.pi * np.outer(k, n) / D)
    return torch.from_numpy(m.T.copy()).to(torch.float32)


@pytest.mark.parametrize("D", [64, 96, 128, 160, 256])
@pytest.mark.parametrize("dtype,group", [("f16", 32), ("bf16", 32), ("f16", 0)])
def test_a_recorded_encode_follows_the_plans_rotation(D, dtype, group):
    """The encode kernels scale their operands by the table's largest entry: it too has to be that of the tables as they are.  (A limit
    kept from the recording takes fp16 operands out of range where a rotation makes it more than four times as large.)"""
    N, rpl = 3000, 1100
    plan = kb.Plan(D, group or D, 70 + D)
    kb.kvq_plan_set_impl(plan.handle, kb.KVQ_IMPL_GEMM, kb.KVQ_IMPL_AUTO)
    sg = plan.signs()
    x, lam = wl.make_vectors(N, D, dtype, "k_outlier", 71), wl.make_lambda(3, D, 72)
    xd, lamd = x.cuda(), lam.cuda()
    packed, scales = plan.empty_packed(N), plan.empty_scales(N)
    kb.kvq_plan_prepare(plan.handle, wl.torch_dtype(dtype))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        kb.kvq_encode(plan.handle, xd, lamd, packed, scales, rpl)
    for R in (None, wl.make_rotation(D, 73), inverse_transform(D), None):
        plan.set_rotation(R)
        graph.replay()
        torch.cuda.synchronize()
        ora = ko.encode(wl.raw_bits(x), DT[dtype], sg, lam.numpy(), plan.group, rpl, want_v=True, rot=None if R is None else R.numpy().astype(np.float64))
        parity.check_encode(packed.cpu().numpy(), wl.raw_bits(scales), ora, plan.group, "replayed encode", min_agree=0.9995)
    assert kb.kvq_plan_device_status(plan.handle) == 0
    del graph
    plan.close()


@pytest.mark.parametrize("D", [64, 96, 128, 160, 256])
@pytest.mark.parametrize("S", [2500, 40])
def test_a_recorded_append_follows_the_plans_rotation(D, S):
    """A rotation rewrites the plan's tables and the append kernel's split operands in place: the power of two that a recorded append takes
    out again has to be the one that they carry, whatever the rotation.  (40 streams: the matrix-vector kernel.)"""
    T, rpl = 3, 32
    plan = kb.Plan(D, G, 60 + D)
    sg = plan.signs()
    x, lam = wl.make_vectors(S, D, "f16", "k_outlier", 61), wl.make_lambda(-(-S // rpl), D, 62)
    xd, lamd = x.cuda(), lam.cuda()
    packed = torch.zeros(S, T, D // 2, dtype=torch.uint8, device="cuda")
    scales = torch.zeros(S, T, D // G, dtype=torch.float16, device="cuda")
    kb.kvq_plan_prepare(plan.handle, torch.float16)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        kb.kvq_append(plan.handle, xd, lamd, packed, scales, 1, rpl)
    for R in (None, wl.make_rotation(D, 63), wl.make_rotation(D, 64, 0.02), inverse_transform(D), None):
        plan.set_rotation(R)
        packed.zero_(), scales.zero_()
        graph.replay()
        torch.cuda.synchronize()
        ora = ko.encode(wl.raw_bits(x), ko.F16, sg, lam.numpy(), G, rpl, want_v=True, rot=None if R is None else R.numpy().astype(np.float64))
        parity.check_encode(packed[:, 1].contiguous().cpu().numpy(), wl.raw_bits(scales[:, 1].contiguous()), ora, G, "replayed append", min_agree=0.9995 if S > 100 else 0.999)
        assert not bool(packed[:, [0, 2]].any()) and not bool(scales[:, [0, 2]].any())
    assert kb.kvq_plan_device_status(plan.handle) == 0
    del graph
    plan.close()


@pytest.mark.parametrize("D", [64, 256])
@pytest.mark.parametrize("factor", [64.0, 2.0 ** -12])
def test_appends_under_a_matrix_far_from_any_rotation(D, factor):
    """R is not checked.  One that takes the table's entries out of the range of the append kernel's operands is served as before."""
    S = 2500
    plan = kb.Plan(D, G, 80 + D)
    R = factor * wl.make_rotation(D, 81)
    x, lam = wl.make_vectors(S, D, "f16", "gaussian", 82), wl.make_lambda(1, D, 83) / factor
    packed = torch.zeros(S, 1, D // 2, dtype=torch.uint8, device="cuda")
    scales = torch.zeros(S, 1, D // G, dtype=torch.float16, device="cuda")
    for _ in range(2):   # set before the tables exist, and on them
        plan.set_rotation(R)
        kb.kvq_append(plan.handle, x.cuda(), lam.cuda(), packed, scales, 0)
        torch.cuda.synchronize()
        ora = ko.encode(wl.raw_bits(x), ko.F16, plan.signs(), lam.numpy(), G, want_v=True, rot=R.numpy().astype(np.float64))
        parity.check_encode(packed[:, 0].contiguous().cpu().numpy(), wl.raw_bits(scales[:, 0].contiguous()), ora, G, "append, scaled rotation", min_agree=0.9995)
        packed.zero_()
    plan.close()


def test_prepare_checks_its_arguments_first():
    L = kb.lib()
    p = kb.Plan(128, G, 1)
    assert L.kvq_plan_prepare(None, kb.KVQ_F16) == kb.KVQ_ERR_INVALID_ARG
    assert L.kvq_plan_prepare(p.handle, 5) == kb.KVQ_ERR_INVALID_ARG
    assert p.describe()[1] == 0
    p.close()


def test_a_bounded_wait_that_runs_out_is_reported_and_service_returns():
    """Every wait inside the kernels is bounded and ends in a status bit, never in a hang.  With the host-settable limit of
    the tensor-core encode kernel's first wait cut to one poll, a one-tile call gives up at a point where the waiting role
    has nothing in flight: the call returns, writes nothing, the status word carries the slot-time-out bit and reads as
    KVQ_ERR_TIMEOUT; after clearing it and restoring the limit the same call is correct."""
    D, N = 128, 100                                   # one tile
    plan = kb.Plan(D, G, 500)
    kb.kvq_plan_set_impl(plan.handle, kb.KVQ_IMPL_GEMM, kb.KVQ_IMPL_AUTO)
    sg = plan.signs()
    x = wl.make_vectors(N, D, "f16", "gaussian", 501)
    lam = wl.make_lambda(1, D, 502)
    xd, lamd = x.cuda(), lam.cuda()
    packed = torch.full((N, D // 2), 0xAB, dtype=torch.uint8, device="cuda")
    scales = torch.full((N, D // G), 1.25, dtype=torch.float16, device="cuda")
    kb.kvq_plan_set_wait_limit(plan.handle, 1)
    kb.kvq_encode(plan.handle, xd, lamd, packed, scales)
    torch.cuda.synchronize()                          # the launch ends by itself
    word = kb.kvq_plan_device_status(plan.handle)
    assert word & 7 == 4, "status word %d" % word     # bit 2: a wait for a pipeline slot ran out
    w = kb.ctypes.c_uint32()
    assert kb.lib().kvq_plan_device_status(plan.handle, kb.ctypes.byref(w)) == kb.KVQ_ERR_TIMEOUT
    assert bool((packed == 0xAB).all()) and bool((scales == 1.25).all())      # nothing was written
    kb.kvq_plan_clear_device_status(plan.handle)
    assert kb.kvq_plan_device_status(plan.handle) == 0
    kb.kvq_plan_set_wait_limit(plan.handle, 0)        # the default again
    kb.kvq_encode(plan.handle, xd, lamd, packed, scales)
    torch.cuda.synchronize()
    assert kb.kvq_plan_device_status(plan.handle) == 0
    ora = ko.encode(wl.raw_bits(x), ko.F16, sg, lam.numpy(), G, want_v=True)
    parity.check_encode(packed.cpu().numpy(), wl.raw_bits(scales), ora, G, "encode after a reported time-out", min_agree=0.9995)
    plan.close()


@pytest.mark.parametrize("D", [64, 128, 256])
def test_the_append_kernels_first_wait_is_reported_and_service_returns(D):
    """The same limit governs the append kernel's wait for its operands: they are then asked for when the wait begins, so that one poll is
    over before they can be there."""
    S = 100
    plan = kb.Plan(D, G, 510)
    kb.kvq_plan_set_impl(plan.handle, kb.KVQ_IMPL_GEMM, kb.KVQ_IMPL_AUTO)
    x, lam = wl.make_vectors(S, D, "f16", "gaussian", 511), wl.make_lambda(1, D, 512)
    xd, lamd = x.cuda(), lam.cuda()
    packed = torch.full((S, 2, D // 2), 0xAB, dtype=torch.uint8, device="cuda")
    scales = torch.full((S, 2, D // G), 1.25, dtype=torch.float16, device="cuda")
    kb.kvq_plan_set_wait_limit(plan.handle, 1)
    kb.kvq_append(plan.handle, xd, lamd, packed, scales, 1)
    torch.cuda.synchronize()
    word = kb.kvq_plan_device_status(plan.handle)
    assert word & 7 == 4, "status word %d" % word
    assert bool((packed == 0xAB).all()) and bool((scales == 1.25).all())
    kb.kvq_plan_clear_device_status(plan.handle)
    kb.kvq_plan_set_wait_limit(plan.handle, 0)
    kb.kvq_append(plan.handle, xd, lamd, packed, scales, 1)
    torch.cuda.synchronize()
    assert kb.kvq_plan_device_status(plan.handle) == 0
    ora = ko.encode(wl.raw_bits(x), ko.F16, plan.signs(), lam.numpy(), G, want_v=True)
    parity.check_encode(packed[:, 1].contiguous().cpu().numpy(), wl.raw_bits(scales[:, 1].contiguous()), ora, G, "append after a reported time-out", min_agree=0.9995)
    plan.close()


@pytest.mark.parametrize("D", [64, 96, 128])
@pytest.mark.parametrize("dtype", ["f16", "bf16"])
def test_the_block_flush_kernels_first_wait_is_reported_and_service_returns(D, dtype):
    """The same limit governs the one-launch block flush's wait for its first operand.  Five tiles per CTA: the loading role has tiles in flight and waits
    for a free stage, the quantizing and output roles wait for their first accumulators when the issuing role gives up; all of them leave, nothing is
    written, and the next call gives what the two-launch form gives."""
    S, rows, T = 5 * 148, 70, 75
    plan, two = kb.Plan(D, G, 520), kb.Plan(D, G, 520)
    kb.kvq_plan_set_impl(two.handle, kb.KVQ_IMPL_GEMM, kb.KVQ_IMPL_GEMM)
    dt = wl.torch_dtype(dtype)
    x, lam = wl.make_vectors(S * rows, D, dtype, "gaussian", 521).view(S, rows, D).cuda(), wl.make_lambda(1, D, 522).cuda()

    def caches():
        return [torch.full((S, T, D // 2), 0xAB, dtype=torch.uint8, device="cuda"), torch.full((S, T, D // G), 1.25, dtype=torch.float16, device="cuda"),
                torch.full((S, T, D), 3.0, dtype=dt, device="cuda")]

    got = caches()
    kb.kvq_plan_set_wait_limit(plan.handle, 1)
    n0 = kb.kvq_launch_count()
    kb.kvq_flush_block(plan.handle, x, lam, *got, 5)
    torch.cuda.synchronize()
    word = kb.kvq_plan_device_status(plan.handle)
    assert kb.kvq_launch_count() - n0 == 1 and word & 7 == 4, "status word %d" % word
    assert all(torch.equal(a, b) for a, b in zip(got, caches()))
    kb.kvq_plan_clear_device_status(plan.handle)
    for polls in (0xFFFFFFFF, 1 << 21, 0):   # longer than the default, long enough, the default again
        kb.kvq_plan_set_wait_limit(plan.handle, polls)
        for a in got:
            a[:, 5:].zero_()
        kb.kvq_flush_block(plan.handle, x, lam, *got, 5)
        torch.cuda.synchronize()
        assert bool(got[2][:, 5:].any(dim=-1).all()) and kb.kvq_plan_device_status(plan.handle) == 0
    packed, scales = two.empty_packed(S * rows), two.empty_scales(S * rows)
    kb.kvq_encode(two.handle, x.view(S * rows, D), lam, packed, scales)
    out = torch.empty(S * rows, D, dtype=dt, device="cuda")
    kb.kvq_decode(two.handle, packed, scales, lam, out)
    torch.cuda.synchronize()
    assert kb.kvq_plan_device_status(plan.handle) == 0
    for a, b, untouched in zip(got, (packed, scales, out), caches()):
        assert torch.equal(a[:, 5:].reshape(S * rows, -1).view(torch.uint8), b.view(torch.uint8)) and torch.equal(a[:, :5], untouched[:, :5])
    plan.close()
    two.close()


@pytest.mark.parametrize("D,dtype,group,nbits", [(64, "bf16", 32, 4), (96, "f16", 32, 4), (128, "f16", 32, 4), (128, "bf16", 128, 8),
                                                 (160, "bf16", 32, 4), (256, "bf16", 32, 4), (256, "f16", 256, 4), (256, "bf16", 32, 8)])
def test_a_call_queued_behind_another_sees_all_that_it_wrote(D, dtype, group, nbits):
    """A grid may come up while its predecessor runs out: chains encode -> decode -> encode of the decoded rows -> append -> decode,
    queued without a wait on one buffer set, on a side stream and as a replayed graph, against the same calls one by one."""
    N, S = 3 * 128 * 148 + 77, 37
    plan = kb.Plan(D, group, 5, bits=nbits)
    dt = wl.torch_dtype(dtype)
    kb.kvq_plan_prepare(plan.handle, dt)
    xs = [wl.make_vectors(N, D, dtype, "gaussian", 6 + i, device="cuda") for i in range(2)]
    new = wl.make_vectors(S, D, dtype, "gaussian", 9, device="cuda")
    lam = wl.make_lambda(3, D, 8).cuda()
    rpl, T = -(-N // 3), N // S

    def buffers():
        return [torch.zeros(N, D * nbits // 8, dtype=torch.uint8, device="cuda"),
                torch.zeros(N, D // group, dtype=torch.float16, device="cuda"), torch.zeros(N, D, dtype=dt, device="cuda")]

    def chain(b, wait):
        packed, scales, out = b
        for x in xs:
            for src in (x, out):
                kb.kvq_encode(plan.handle, src, lam, packed, scales, rpl)
                wait()
                kb.kvq_append(plan.handle, new, lam, packed[:S * T].view(S, T, -1), scales[:S * T].view(S, T, -1), T - 1, 13)
                wait()
                kb.kvq_decode(plan.handle, packed, scales, lam, out, rpl)
                wait()

    want = buffers()
    chain(want, torch.cuda.synchronize)
    side = torch.cuda.Stream()
    for _ in range(4):
        got = buffers()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            chain(got, lambda: None)
        torch.cuda.current_stream().wait_stream(side)
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want))
    got = buffers()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(got, lambda: None)
    for _ in range(3):
        for b in got:
            b.zero_()
        graph.replay()
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want))
    del graph
    assert kb.kvq_plan_device_status(plan.handle) == 0
    plan.close()


@pytest.mark.parametrize("D,dtype", [(64, "bf16"), (96, "f16"), (128, "f16"), (128, "bf16"), (160, "f16"), (256, "f16"), (256, "bf16")])
@pytest.mark.parametrize("small", [False, True])
def test_a_call_queued_behind_another_reads_the_lambda_and_the_rows_that_it_wrote(D, dtype, small):
    """What a grid reads right behind its wait is written by the grid ahead: a calibration's lambda (new vectors, other values, each
    turn; one turn with a channel so small that the decode takes its fp32 form), appended rows, their codes.  Small calls take
    the matrix-vector kernels.  Queued without a wait, on a side stream and as a replayed graph, against one by one."""
    N, S, T = (900, 300, 3) if small else (128 * 148 + 77, 1871, 10)
    plan = kb.Plan(D, G, 5)
    dt = wl.torch_dtype(dtype)
    kb.kvq_plan_prepare(plan.handle, dt)
    samples = [wl.make_vectors(2500, D, dtype, kind, 20 + i, device="cuda") for i, kind in enumerate(("lognormal", "gaussian", "k_outlier"))]
    samples.append(torch.zeros_like(samples[0]))
    samples[3][:, 0] = 60000.0                                     # |z_c| above 5000 on the cosine channels, 0 on the sine ones: lambda 1
    xs = [wl.make_vectors(N, D, dtype, "k_outlier", 30 + i, device="cuda") for i in range(len(samples))]

    def buffers():
        z = lambda *shape, dtype: torch.zeros(*shape, dtype=dtype, device="cuda")
        return [z(D, dtype=torch.float32), z(N, D // 2, dtype=torch.uint8), z(N, D // G, dtype=torch.float16), z(N, D, dtype=dt)]

    def chain(b, wait):
        lam, packed, scales, out = b
        pc, sc = packed[:S * T].view(S, T, -1), scales[:S * T].view(S, T, -1)
        for i, x in enumerate(xs):
            kb.kvq_calibrate_lambda(plan.handle, samples[i], lam)
            wait()
            kb.kvq_encode(plan.handle, x, lam, packed, scales)
            wait()
            kb.kvq_decode(plan.handle, packed, scales, lam, out)
            wait()
            for pos in range(T):                                   # the decoded rows go back in, one per stream and call
                kb.kvq_append(plan.handle, out[pos * S:(pos + 1) * S], lam, pc, sc, pos)
                wait()
                kb.kvq_decode(plan.handle, packed, scales, lam, out)
                wait()

    want = buffers()
    chain(want, torch.cuda.synchronize)
    same = lambda got: all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got, want))
    side = torch.cuda.Stream()
    for _ in range(4):
        got = buffers()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            chain(got, lambda: None)
        torch.cuda.current_stream().wait_stream(side)
        assert same(got)
    got = buffers()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(got, lambda: None)
    for _ in range(3):
        for b in got:
            b.zero_()
        graph.replay()
        assert same(got)
    del graph
    assert kb.kvq_plan_device_status(plan.handle) == 0
    plan.close()
