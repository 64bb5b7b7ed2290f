"""The rule of the packed buffer's stream order (include/tman.h): a kernel of the caller's own that signals early completion and then
writes a packed buffer is safe when another kernel, here one of the library's, stands between it and the decode call."""
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
