"""Stream order.  Calls that follow one another without a gap read what their predecessors wrote.  And the rule of the packed
buffer's stream order (include/tman.h): a kernel of the caller's own that signals early completion and then
writes a packed buffer is safe when another kernel, here one of the library's, stands between it and the decode call."""
import numpy as np
import pytest
import torch

from paper_2511_11248_b200 import binding as B, helpers as H, synth

pytestmark = pytest.mark.gpu

# signals first, writes 200 us later (bounded)
LATE_COPY = r"""
extern "C" __global__ void late_copy(const unsigned *src, unsigned *dst, int words)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int i = 0; i < 100000; ++i) {
        __nanosleep(500);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 200000ull) break;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
"""


@pytest.mark.parametrize("between", ["quantize", "quantize_i8", "prefill", "int8_prefill"])
def test_a_call_between_an_early_signalling_writer_and_a_decode(between):
    K, N, bits, G = 1024, 2048, 4, 128
    old, new = (synth.small_case(1, K, N, bits, G, seed=s) for s in (1, 2))
    dev = H.device_case(new)
    src, want = H.pack_case(new, dev), H.alloc_y(1, N)
    ws, wsg = H.alloc_workspace(B.OP_GEMV, 1, K, N, bits, G), H.alloc_workspace(B.OP_GEMM, 1, K, N, bits, G)
    B.tman_mpgemv(src, dev["x"], want, 1, K, N, bits, G, ws)
    dst = H.pack_case(old)
    codes = torch.ones((K, N), dtype=torch.uint8, device="cuda")
    ternary = H.alloc_packed(K, N, 2, G)
    B.tman_pack_weights(codes, torch.ones((K // G, N), dtype=torch.float16, device="cuda"), codes[:K // G], K, N, 2, G, ternary)
    a16, a8 = (torch.zeros((1, K), dtype=t, device="cuda") for t in (torch.int16, torch.int8))
    s, y, y2 = torch.ones(4, dtype=torch.float32, device="cuda"), H.alloc_y(1, N), H.alloc_y(1, N)
    late_copy = torch.cuda._compile_kernel(LATE_COPY, "late_copy")

    def other_kernel():
        if between == "quantize":
            B.tman_quantize_rows(dev["x"], 1, K, 32767, a16, s)
        elif between == "quantize_i8":
            B.tman_quantize_rows_i8(dev["x"], 1, K, a8, s)
        elif between == "prefill":
            B.tman_mpgemm(src, dev["x"], y2, 1, K, N, bits, G, wsg)
        else:
            B.tman_mpgemm_ternary_i8(ternary, a8, s, 1.0, y2, 1, K, N, G, wsg)

    other_kernel()
    B.tman_mpgemv(dst, dev["x"], y, 1, K, N, bits, G, ws)      # (the first decode after a packing runs in plain stream order)
    late_copy((8, 1, 1), (256, 1, 1), (src, dst, dst.numel() // 4))      # (allocations of a multiple of 256 bytes)
    other_kernel()
    B.tman_mpgemv(dst, dev["x"], y, 1, K, N, bits, G, ws)
    assert B.tman_read_status(ws) == 0 and B.tman_read_status(wsg) == 0
    assert torch.equal(dst, src)
    assert torch.equal(y, want)


@pytest.mark.parametrize("M,K,bits,G", [(1, 2048, 4, 128), (2, 2048, 4, 128), (1, 6144, 4, 128), (1, 6144, 2, 64), (1, 8192, 3, 32), (2, 6144, 4, 128),
                                        (2, 8192, 2, 32), (4, 4096, 3, 32), (4, 2048, 3, 64), (8, 1152, 2, 32)])
def test_chained_calls_read_what_the_call_before_wrote(M, K, bits, G):
    # two buffers in turn: a call's activations are the outputs of the call before it, written to the lines that the call two before it
    # read.  In one graph, and with the GPU waited for after every call: the same bits.
    steps = 24
    c = synth.small_case(M, K, K, bits, G, seed=K + M)
    w = c.scales.astype(np.float32).repeat(G, 0) * (c.codes.astype(np.float32) - c.zeros.astype(np.float32).repeat(G, 0))
    c.scales[:] = (c.scales / (np.sqrt(K) * w.std())).astype(np.float16)                 # outputs of the inputs' size
    packed, ws = H.pack_case(c), H.alloc_workspace(B.OP_GEMV, M, K, K, bits, G)
    x = H.device_case(c)["x"]

    def chain(bufs, outs, wait):
        bufs[0].copy_(x)
        for i in range(steps):
            B.tman_mpgemv(packed, bufs[i % 2], bufs[1 - i % 2], M, K, K, bits, G, ws)
            if wait:
                torch.cuda.synchronize()
            if i >= steps - 2:
                outs[i % 2].copy_(bufs[1 - i % 2])

    want, got = ([H.alloc_y(M, K) for _ in range(2)] for _ in range(2))
    bufs = [H.alloc_y(M, K) for _ in range(2)]
    chain(bufs, want, True)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(bufs, got, False)
    for _ in range(3):
        graph.replay()
    assert B.tman_read_status(ws) == 0
    assert all(bool(torch.isfinite(w).all()) and bool((w != 0).any()) for w in want)
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("M,K", [(1, 2560), (3, 2048), (8, 1536)])
def test_chained_integer_calls_read_what_the_call_before_wrote(M, K):
    # as above through the row quantization, one array of integers and one of row scales for all calls
    steps, G = 16, 128
    codes = torch.randint(0, 3, (K, K), dtype=torch.uint8, device="cuda", generator=torch.Generator("cuda").manual_seed(K))
    packed = H.alloc_packed(K, K, 2, G)
    B.tman_pack_weights(codes, torch.ones((K // G, K), dtype=torch.float16, device="cuda"), torch.ones((K // G, K), dtype=torch.uint8, device="cuda"), K, K, 2, G, packed)
    ws = H.guarded_bytes(B.tman_workspace_bytes(B.OP_TERNARY, M, K, K, 2, G), "workspace")
    B.tman_workspace_init(ws)
    x = H.device_case(synth.small_case(M, K, 8, 2, G, seed=K))["x"]
    a = torch.empty((M, K), dtype=torch.int16, device="cuda")
    s = torch.empty(8, dtype=torch.float32, device="cuda")

    def chain(bufs, wait):
        bufs[0].copy_(x)
        for i in range(steps):
            B.tman_quantize_rows(bufs[i % 2], M, K, 32767, a, s)
            if wait:
                torch.cuda.synchronize()
            B.tman_mpgemv_ternary(packed, a, s, 1.2 / K ** 0.5, bufs[1 - i % 2], None, M, K, K, G, ws)
            if wait:
                torch.cuda.synchronize()

    want, got = ([H.alloc_y(M, K) for _ in range(2)] for _ in range(2))
    chain(want, True)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        chain(got, False)
    for _ in range(3):
        graph.replay()
    assert B.tman_read_status(ws) == 0
    assert all(bool(torch.isfinite(w).all()) and bool((w != 0).any()) for w in want)
    assert all(torch.equal(a, b) for a, b in zip(got, want))
