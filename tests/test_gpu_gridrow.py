"""The grid-row kernel where the choice by shape uses it: float32 weights, groups beyond 16 CTAs, each way the row statistics
cross a group, several streams at once, and stream capture."""
import math

import numpy as np
import pytest
import torch

import oracle
from helpers import TOL, assert_close_to_oracle, assert_guards_intact, bits_to_cuda_bf16, guarded_empty, small_fused_inputs, to_f64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def attnw():
    from paper_2407_13885_b200 import binding
    return binding


def scale_of(d):
    return float(np.float32(1.0 / math.sqrt(d)))


# one CTA (no exchange), 2 and 4 (every CTA reads all pairs), 5, 7, 8, 15 and 16 (owners of 32, 32, 16, 16 and 8 rows);
# a slab with one slot in use, a store box that is cut, row blocks of 4 rows, more row blocks than groups
SHAPES = [(1, 1, 4, 64), (3, 50, 60, 64), (1, 2, 256, 128), (1, 3, 260, 64), (1, 5, 512, 64), (2, 3, 1020, 128),
          (1, 2, 1284, 64), (1, 2, 1792, 128), (1, 9, 1924, 64), (1, 2, 3716, 64), (1, 1, 4096, 128)]


@pytest.mark.parametrize("B,H,N,d", SHAPES)
def test_float32_weights_match_oracle(attnw, B, H, N, d):
    q, k = small_fused_inputs(B, H, N, d, stream=N + d + 13)
    Q, K = bits_to_cuda_bf16(q), bits_to_cuda_bf16(k)
    ref = oracle.attnw(q, k, scale_of(d))
    for _ in range(2):  # the second launch finds the exchange area as the first one left it
        raw, P, g = guarded_empty((B, H, N, N), torch.float32)
        attnw.attnw_fused(Q, K, scale_of(d), P=P)
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        assert_guards_intact(raw, g)
        assert_close_to_oracle(P, ref, f"B{B} H{H} N{N} d{d}")


# groups of 17, 24, 33, 48, 64 and 101 CTAs (owners of 8, 8, 4, 4, 2 and 2 rows); the last row blocks and columns ragged
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("H,N,d", [(2, 4104, 64), (1, 6000, 128), (1, 8456, 64), (1, 12288, 128), (1, 16384, 64), (1, 25608, 64)])
def test_long_rows_match_oracle(attnw, dtype, H, N, d):
    q, k = small_fused_inputs(1, H, N, d, sigma=1.5, stream=N + 1)
    raw, P, g = guarded_empty((1, H, N, N), dtype)
    attnw.attnw_fused(bits_to_cuda_bf16(q), bits_to_cuda_bf16(k), scale_of(d), P=P)
    torch.cuda.synchronize()
    assert attnw.query_status() == 0
    assert_guards_intact(raw, g)
    rows = P.view(-1, N)
    assert float((torch.stack([r.double().sum() for r in rows.split(1)]) - 1.0).abs().max()) <= TOL[dtype]["rowsum"]
    ids = np.unique(np.concatenate([np.arange(0, H * N, 211 if N < 10000 else 997), [0, 127, 128, N - 1, H * N - 1]]))
    err = np.max(np.abs(to_f64(rows[torch.from_numpy(ids).cuda()]) - oracle.attnw_rows(q, k, scale_of(d), ids)))
    assert err <= TOL[dtype]["abs"]


# one CTA, an exchange where all read all, owners, and a group beyond 16 CTAs; a row whose largest logit is large itself
@pytest.mark.parametrize("N,d,sigma", [(256, 64, 4.0), (1000, 128, 4.0), (2048, 128, 4.0), (8192, 128, 4.0), (2048, 64, 60.0)])
def test_small_weights_keep_their_digits(attnw, N, d, sigma):
    # A weight's relative error: its logit and its row's sum in float32 (d products, each step within 2^-23 of the sum of the
    # products' sizes, twice), the exponential in f16 (2^-11) and the result in bf16 (2^-9), with a factor 2 on these.
    g = torch.Generator(device="cuda").manual_seed(N + d)
    Q, K = (torch.randn(1, 1, N, d, generator=g, device="cuda", dtype=torch.bfloat16).mul_(sigma) for _ in range(2))
    P = attnw.attnw_fused(Q, K, scale_of(d))
    torch.cuda.synchronize()
    assert attnw.query_status() == 0
    S = (Q[0, 0, :512].double() @ K[0, 0].double().T) * scale_of(d)
    ref = torch.softmax(S, -1)
    # within 2^-28 of its row's largest weight a weight is still a normal f16 number, whichever chunk it lies in
    m = ref >= ref.amax(-1, keepdim=True) * 2.0 ** -28
    size = (Q[0, 0, :512].double().abs() @ K[0, 0].double().abs().T) * scale_of(d)
    bound = 2.0 ** -8 + 2.0 ** -10 + 2 * size * d * 2.0 ** -23
    rel = (P[0, 0, :512].double() - ref).abs() / ref
    assert int(m.sum()) > 512
    assert bool((rel <= bound)[m].all()), float((rel / bound)[m].max())


def test_more_streams_than_exchange_areas(attnw):
    # twelve streams, two calls each in flight, on inputs of their own: no launch may read another's statistics
    d, N = 64, 1536
    cases = []
    for s in range(12):
        q, k = small_fused_inputs(1, 1, N, d, stream=700 + s)
        cases.append((bits_to_cuda_bf16(q), bits_to_cuda_bf16(k), oracle.attnw(q, k, scale_of(d))))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in cases]
    for _ in range(3):
        out = []
        for dtype in (torch.bfloat16, torch.float32):
            for (Q, K, _), s in zip(cases, streams):
                with torch.cuda.stream(s):
                    out.append(attnw.attnw_fused(Q, K, scale_of(d), out_dtype=dtype))
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        for n, P in enumerate(out):
            assert_close_to_oracle(P, cases[n % 12][2], f"stream {n % 12}")


LAST_TAG = 0x7fffffff


@pytest.mark.parametrize("entry", ["fused", "noalloc"])
def test_message_tags_start_over(attnw, entry):
    # before each call the tags run out, so that it starts over with those which the calls before have left in the exchange area:
    # the same groups on other inputs (4 CTAs, where all read all pairs, and 6, with owners), and groups of 16 in between
    d = 64
    call = attnw.attnw_fused if entry == "fused" else attnw.attnw_fused_noalloc
    for x, N in enumerate((1000, 1000, 1288, 1288, 4096, 1288, 1000)):
        q, k = small_fused_inputs(1, 2, N, d, sigma=2.0, stream=900 + x)
        Q, K = bits_to_cuda_bf16(q), bits_to_cuda_bf16(k)
        if x == 0:
            attnw.attnw_fused(Q, K, scale_of(d))  # the stream's exchange area
            with pytest.raises(attnw.AttnwError):
                attnw.selftest_exchange_tags(0)   # forward only
        attnw.selftest_exchange_tags(LAST_TAG)
        P = call(Q, K, scale_of(d))
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        assert_close_to_oracle(P, oracle.attnw(q, k, scale_of(d)), f"{entry} N{N}")


def test_captured_noalloc_calls_have_tags_of_their_own(attnw):
    # captured when the tags had run out; then replays and uncaptured calls, on other inputs each time, in turn
    d, N = 64, 1288
    calls = [small_fused_inputs(1, 2, N, d, sigma=2.0, stream=950 + x) for x in range(6)]
    Q, K = bits_to_cuda_bf16(calls[0][0]), bits_to_cuda_bf16(calls[0][1])
    P = torch.empty((1, 2, N, N), dtype=torch.bfloat16, device="cuda")
    attnw.attnw_fused(Q, K, scale_of(d))
    attnw.attnw_fused_noalloc(Q, K, scale_of(d), P=P)
    attnw.selftest_exchange_tags(LAST_TAG)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        attnw.attnw_fused_noalloc(Q, K, scale_of(d), P=P)
    for x, (q, k) in enumerate(calls):
        Q.copy_(bits_to_cuda_bf16(q))
        K.copy_(bits_to_cuda_bf16(k))
        P.fill_(float("nan"))
        graph.replay() if x % 2 == 0 else attnw.attnw_fused_noalloc(Q, K, scale_of(d), P=P)
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        assert_close_to_oracle(P, oracle.attnw(q, k, scale_of(d)), f"call {x}")


@pytest.mark.parametrize("entry,dtype", [("fused", torch.bfloat16), ("fused", torch.float32), ("noalloc", torch.bfloat16)])
@pytest.mark.parametrize("N", [256, 2048])
def test_captured_call_is_right_on_every_replay(attnw, entry, dtype, N):
    d = 64
    calls = [small_fused_inputs(1, 2, N, d, stream=800 + x) for x in range(3)]
    Q, K = bits_to_cuda_bf16(calls[0][0]), bits_to_cuda_bf16(calls[0][1])
    P = torch.empty((1, 2, N, N), dtype=dtype, device="cuda")

    def call():
        if entry == "fused":
            attnw.attnw_fused(Q, K, scale_of(d), P=P)
        else:
            attnw.attnw_fused_noalloc(Q, K, scale_of(d), P=P)

    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for q, k in calls:  # other inputs on each replay
        Q.copy_(bits_to_cuda_bf16(q))
        K.copy_(bits_to_cuda_bf16(k))
        P.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        assert_close_to_oracle(P, oracle.attnw(q, k, scale_of(d)), f"{entry} {dtype} N{N}")


# captured calls of many heads: one part on the resident kernel, the others beside it on the two-pass kernel
@pytest.mark.parametrize("H,N,d", [(12, 4096, 64), (8, 4040, 128)])
def test_captured_call_in_two_parts(attnw, H, N, d):
    X = torch.zeros(1, 64, 64, dtype=torch.bfloat16, device="cuda")
    W = torch.zeros(1, 64, 64, dtype=torch.bfloat16, device="cuda")
    calls = [small_fused_inputs(1, H, N, d, stream=820 + x) for x in range(2)]
    ids = np.unique(np.concatenate([np.arange(0, H * N, 617), [0, H * N - 1]]))
    Q, K = (bits_to_cuda_bf16(x) for x in calls[0])
    for behind_another in (False, True):  # the first node of its graph, and behind a launch that may overlap its own
        P = torch.empty((1, H, N, N), dtype=torch.bfloat16, device="cuda")
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            if behind_another:
                attnw.project_qk(X, W, W)
            launches = attnw.launch_count()
            attnw.attnw_fused(Q, K, scale_of(d), P=P)
            assert attnw.launch_count() == launches + 2
        for q, k in calls:
            Q.copy_(bits_to_cuda_bf16(q))
            K.copy_(bits_to_cuda_bf16(k))
            P.fill_(float("nan"))
            graph.replay()
            torch.cuda.synchronize()
            assert attnw.query_status() == 0
            assert not bool(torch.isnan(P).any())
            rows = P.view(-1, N)[torch.from_numpy(ids).cuda()]
            err = np.max(np.abs(to_f64(rows) - oracle.attnw_rows(q, k, scale_of(d), ids)))
            assert err <= TOL[torch.bfloat16]["abs"], err


def test_exchange_area_for_a_new_stream_while_another_is_captured():
    # in a process of its own, where no exchange area is free: a second stream needs one while a blocking stream is captured
    import os
    import subprocess
    import sys
    code = """if True:
        import torch
        from cuda.bindings import runtime as rt
        from paper_2407_13885_b200 import binding
        Q, K = (torch.randn(1, 2, 1000, 64, device="cuda").bfloat16() for _ in range(2))
        P = [torch.zeros(1, 2, 1000, 1000, dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        first, second = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        binding.attnw_fused(Q, K, 0.125, P=P[0], stream=first)
        torch.cuda.synchronize()
        _, blocking = rt.cudaStreamCreate()
        (err,) = rt.cudaStreamBeginCapture(blocking, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed)
        assert err == rt.cudaError_t.cudaSuccess
        binding.attnw_fused(Q, K, 0.125, P=P[1], stream=second)
        err, graph = rt.cudaStreamEndCapture(blocking)
        assert err == rt.cudaError_t.cudaSuccess, err
        torch.cuda.synchronize()
        assert binding.query_status() == 0 and torch.equal(P[0], P[1])
        binding.selftest_exchange_tags(100, stream=second)  # refused for a stream without an area
        """
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], cwd=root, check=True, timeout=300)


def test_two_captures_open_at_once(attnw):
    from cuda.bindings import runtime as rt
    H, N, d = 8, 4040, 64
    relaxed = rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed

    def ok(result):
        assert result[0] == rt.cudaError_t.cudaSuccess, result[0]
        return result[1] if len(result) > 1 else None

    calls = [tuple(bits_to_cuda_bf16(x) for x in small_fused_inputs(1, H, N, d, stream=840 + 2 * n)) for n in range(2)]
    want = [attnw.attnw_fused(Q, K, scale_of(d)) for Q, K in calls]
    P = [torch.full_like(w, float("nan")) for w in want]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in calls]
    for n, s in enumerate(streams):
        ok(rt.cudaStreamBeginCapture(s.cuda_stream, relaxed))
        attnw.attnw_fused(*calls[n], scale_of(d), P=P[n], stream=s)
    graphs = [ok(rt.cudaStreamEndCapture(s.cuda_stream)) for s in streams]
    for s, graph in zip(streams, graphs):
        run = ok(rt.cudaGraphInstantiate(graph, 0))
        ok(rt.cudaGraphLaunch(run, s.cuda_stream))
        torch.cuda.synchronize()
        ok(rt.cudaGraphExecDestroy(run))
        ok(rt.cudaGraphDestroy(graph))
    assert attnw.query_status() == 0
    for p, w in zip(P, want):
        assert float((p.float() - w.float()).abs().max()) <= TOL[torch.bfloat16]["abs"]


def test_chain_of_calls_sees_the_results_in_front(attnw):
    # each launch may begin before the kernel in front of it has ended: every call here reads what the call before has just
    # written, among ordinary kernels of torch, and the last result is that of the same chain with a wait after each call
    gen = torch.Generator(device="cuda").manual_seed(5)
    X = torch.randn(1, 200, 256, generator=gen, device="cuda", dtype=torch.bfloat16)
    W = [torch.randn(4, 64, 256, generator=gen, device="cuda", dtype=torch.bfloat16) / 16 for _ in range(2)]

    def chain(wait):
        x = X
        for _ in range(6):
            Q, K = attnw.project_qk(x, *W)
            wait()
            O = attnw.attn_fused(Q, K, Q, 0.125)
            wait()
            P = attnw.attnw_fused(O, K, 0.125, out_dtype=torch.float32)
            wait()
            R = attnw.softmax_rows(P.view(-1, 200), out_dtype=torch.float32)
            wait()
            P2 = attnw.attnw_fused(O, Q, 0.125)
            wait()
            x = (O + torch.matmul(R.view(1, 4, 200, 200).bfloat16() + P2, Q)).transpose(1, 2).reshape(1, 200, 256).contiguous()
            wait()
        return x

    want = chain(torch.cuda.synchronize)
    for _ in range(3):
        got = chain(lambda: None)
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        assert torch.equal(got, want)


# logits of sigma 16: weights far below the largest of their row
@pytest.mark.parametrize("N,d", [(256, 64), (1000, 128), (2048, 64), (8192, 128)])
def test_range_of_small_weights(attnw, N, d):
    g = torch.Generator(device="cuda").manual_seed(N + 3 * d)
    Q, K = (torch.randn(1, 1, N, d, generator=g, device="cuda", dtype=torch.bfloat16).mul_(4.0) for _ in range(2))
    S = (Q[0, 0, :256].double() @ K[0, 0].double().T) * scale_of(d)
    ref = torch.softmax(S, -1)
    top = ref.amax(-1, keepdim=True)
    size = (Q[0, 0, :256].double().abs() @ K[0, 0].double().abs().T) * scale_of(d)
    bound = 2.0 ** -8 + 2.0 ** -10 + 2 * size * d * 2.0 ** -23  # relative, as in test_small_weights_keep_their_digits
    assert bool((ref < top * 2.0 ** -60).any())

    def error(P):
        torch.cuda.synchronize()
        assert attnw.query_status() == 0
        return (P[0, 0, :256].double() - ref).abs()

    # half of the smallest 16-bit float, 2^-25, next to the largest, 2^15: absolute, with a factor 2
    assert bool((error(attnw.attnw_fused(Q, K, scale_of(d))) <= bound * ref + 2.0 ** -39 * top).all())
    # float32 to the end: float32 weights, and the two-pass kernel
    whole = ref >= top * 2.0 ** -100
    assert bool((error(attnw.attnw_fused(Q, K, scale_of(d), out_dtype=torch.float32)) <= bound * ref)[whole].all())
    attnw.set_fused_variant("two_pass")
    try:
        P = attnw.attnw_fused(Q, K, scale_of(d))
    finally:
        attnw.set_fused_variant("auto")
    assert bool((error(P) <= bound * ref)[whole].all())
