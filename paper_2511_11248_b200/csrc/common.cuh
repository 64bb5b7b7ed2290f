// Shared declarations of the CUDA side: packed-buffer layout, workspace layout, argument checks.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>
#include <atomic>

#include "tman.h"

namespace tman {

// ---- packed buffer -----------------------------------------------------------------------
// 256-byte header, then bit-plane words, scales, zero-points (each section 256-byte padded).
struct PackedHeader {
    char     magic[8];      // "TMANB200"
    uint32_t version;       // kVersion
    uint32_t K, N, bits, group, lut_g;
    uint64_t planes_off, scales_off, zeros_off, total_bytes;
};
static_assert(sizeof(PackedHeader) == 64, "header fields occupy the first 64 bytes");

constexpr size_t   kHeaderBytes = 256;
constexpr uint32_t kVersion = 2;

// Bit of a plane word that holds the weight with k % 32 == r: weight 8*ph + j sits at bit 4*j + ph
// (an offline permutation, paper Sec. 4.1, that makes the prefill repacking come out in k order).
__host__ __device__ constexpr int plane_bit(int r) { return 4 * (r & 7) + (r >> 3); }

__host__ __device__ inline size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

struct Layout {
    size_t planes_off, scales_off, zeros_off, total;
    size_t planes_bytes, scales_bytes, zeros_bytes;
};

__host__ __device__ inline Layout make_layout(int K, int N, int bits, int group)
{
    Layout L;
    L.planes_bytes = (size_t)K * N * bits / 8;
    L.scales_bytes = (size_t)(K / group) * N * 2;
    L.zeros_bytes = (size_t)(K / group) * (N / 4) * 2;
    L.planes_off = kHeaderBytes;
    L.scales_off = L.planes_off + up256(L.planes_bytes);
    L.zeros_off = L.scales_off + up256(L.scales_bytes);
    L.total = L.zeros_off + up256(L.zeros_bytes);
    return L;
}

// device-side header check: every kernel that reads a packed buffer calls it first
__device__ inline bool header_matches(const void *packed, int K, int N, int bits, int group)
{
    const uint32_t *h = reinterpret_cast<const uint32_t *>(packed);
    // "TMAN" = 0x4E414D54, "B200" = 0x30303242 (little endian)
    bool ok = (h[0] == 0x4E414D54u) && (h[1] == 0x30303242u) && (h[2] == kVersion) &&
              (h[3] == (uint32_t)K) && (h[4] == (uint32_t)N) && (h[5] == (uint32_t)bits) &&
              (h[6] == (uint32_t)group) && (h[7] == 4u);
    return ok;
}

// ---- workspace ---------------------------------------------------------------------------
// [0, 256)      status word (u32) + padding
// [256, ...)     fp32 split-K partial sums; "no sum pending" sentinel between calls
constexpr size_t kWsStatusBytes = 256;

// ---- argument checks (host) --------------------------------------------------------------
inline tman_status check_format(int K, int N, int bits, int group)
{
    if (K <= 0 || N <= 0) return TMAN_ERR_SHAPE;
    if (bits < 1 || bits > 4) return TMAN_ERR_SHAPE;
    if (group != 32 && group != 64 && group != 128) return TMAN_ERR_SHAPE;
    if (K % 128 != 0 || N % 8 != 0) return TMAN_ERR_SHAPE;
    return TMAN_OK;
}

inline tman_status launch_status()
{
    return cudaGetLastError() == cudaSuccess ? TMAN_OK : TMAN_ERR_CUDA;
}

// Properties of the current device that launches are planned from.  They never change, so they are asked once per
// device (two attribute queries a call otherwise).
constexpr int kMaxDevices = 64;
struct DeviceInfo {
    std::atomic<int> sms;             // 0: not asked yet
    std::atomic<int> reserved_smem;   // shared memory the system keeps per CTA (valid once sms is set)
};
DeviceInfo *device_info(int *dev = nullptr);      // nullptr: the query failed

inline int sm_count()
{
    const DeviceInfo *d = device_info();
    return d ? d->sms.load(std::memory_order_acquire) : 0;
}

// Asks for the split of an SM's 256 KB between shared memory (132 KB) and L1 that the decode kernels which alternate in a layer of one or
// two rows have in common: an SM changes its split only when it is idle, so that kernels of different splits do not follow one another
// without a gap (a layer of alternating kernels 76 -> 86 us).  132 KB hold two CTAs of decode_digits_kernel and leave the lookups the L1
// that their loads in flight pass through (with 228 KB of shared memory 14336 x 4096, 4-bit, takes 12.3 us instead of 9.8).  A hint:
// failure changes nothing.
constexpr int kSharedPercent = 58;        // of 228 KB
template <typename Kernel> inline void prefer_common_split(Kernel kern)
{
    if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, kSharedPercent) != cudaSuccess) (void)cudaGetLastError();
}

// Launches `launch()` (cudaSuccess or an error) of a kernel that needs `bytes` of dynamic shared memory.  The kernel's
// limit is raised once per device, `raised[device]` remembers it; a launch that fails all the same (the context may have
// been reset in between) raises the limit again and tries once more.
template <typename Kernel, typename Launch>
inline tman_status launch_with_smem(Kernel kern, int bytes, int dev, std::atomic<bool> *raised, const Launch &launch)
{
    if (raised[dev].load(std::memory_order_relaxed)) {
        if (launch() == cudaSuccess) return TMAN_OK;
        (void)cudaGetLastError();
        raised[dev].store(false, std::memory_order_relaxed);
    }
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return TMAN_ERR_CUDA;
    if (launch() != cudaSuccess) return TMAN_ERR_CUDA;
    raised[dev].store(true, std::memory_order_relaxed);
    return TMAN_OK;
}

// ---- loads behind a wait (device) ----------------------------------------------------------
// What the kernels before this one in the stream wrote (activations, row scales), read after griddepcontrol.wait by a kernel that may
// have started while they ran: ordinary loads that stay behind the wait.  The read-only path (__ldg) is for data that nobody writes while
// the kernel is resident: a load by it may be moved above the wait, and it takes a line that an earlier call left in the SM's L1,
// which the launch of a kernel that starts early does not empty (calls that passed one buffer on to the next read what it held two calls
// before).
__device__ __forceinline__ uint4 ld_dependent(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float ld_dependent(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}

// ---- table building block (device) -------------------------------------------------------
// The 16 partial sums of four activations: out[p] = sum_{j<4} x_j * bit_j(p), accumulated in
// increasing j (paper Sec. 2.2: each bit pattern indexes a precomputed sum).
__device__ __forceinline__ void lut16(float x0, float x1, float x2, float x3, float (&out)[16])
{
    out[0] = 0.f;
    out[1] = x0;
    out[2] = x1;
    out[3] = x0 + x1;
    out[4] = x2;
    out[5] = x0 + x2;
    out[6] = x1 + x2;
    out[7] = out[3] + x2;
#pragma unroll
    for (int p = 0; p < 8; ++p) out[8 + p] = (p == 0) ? x3 : out[p] + x3;
}

// entry points implemented per file
tman_status launch_pack(const uint8_t *codes, const void *scales, const uint8_t *zeros, int K, int N,
                        int bits, int group, void *packed, cudaStream_t s);
// A packing on stream s is followed by one decode launch in plain stream order (no programmatic
// dependent launch): note_packed_write records the stream, packed_write_pending asks and clears.
void note_packed_write(cudaStream_t s);
bool packed_write_pending(cudaStream_t s, bool clear);
tman_status launch_dequant_ternary_int8(const void *packed, int K, int N, int group, int8_t *w8, uint32_t *status,
                                        cudaStream_t s);
tman_status launch_unpack(const void *packed, int K, int N, int bits, int group, uint8_t *codes,
                          void *scales, uint8_t *zeros, uint32_t *status, cudaStream_t s);
tman_status launch_debug_indices(const void *packed, int K, int N, int bits, int group, uint8_t *idx,
                                 uint32_t *status, cudaStream_t s);
tman_status launch_debug_luts(const void *x, int M, int K, float *lut, cudaStream_t s);
size_t      mpgemv_workspace_bytes(int M, int K, int N, int bits);
// The decode call's plan: passes over the weights, each with one kernel variant (see mpgemv.cu).
constexpr int kGemvMaxRows = 8;
constexpr int kGemvVariantCount = 4;
constexpr int kGemvSmemLimit = 227 * 1024;
constexpr int kGemvPlanSms = 148;
struct GemvPass { int variant, rows, variant_rows, words, nkappa, ctas_per_slice, smem_bytes; bool mma, digits; };
struct GemvPlan { int npass; GemvPass pass[kGemvMaxRows]; size_t ws_bytes; double cost_us; };
tman_status launch_quantize_rows(const void *x, int M, int K, int qmax, int16_t *a, float *s_a, cudaStream_t s);
tman_status launch_mpgemv_ternary(const void *packed, const int16_t *a, const float *s_a, float s_w, void *y,
                                  int32_t *acc_out, int M, int K, int N, int group, void *ws, size_t ws_bytes, cudaStream_t s);
size_t      mpgemv_ternary_workspace_bytes(int M, int K, int N);
tman_status launch_wait_timeout(void *ws, size_t ws_bytes, uint32_t limit, cudaStream_t s);
GemvPlan    plan_gemv(int M, int K, int N, int bits, int group, int sms, size_t ws_limit);
tman_status launch_workspace_init(void *ws, size_t ws_bytes, cudaStream_t s);
tman_status launch_mpgemv(const void *packed, const void *x, void *y, int M, int K, int N, int bits,
                          int group, void *ws, size_t ws_bytes, cudaStream_t s);
tman_status launch_mpgemv_grouped(int count, const void *const *packed, const void *x, void *const *y, int M, int K,
                                  const int *Ns, int bits, int group, void *ws, size_t ws_bytes, cudaStream_t s);
size_t      mpgemm_workspace_bytes(int M, int K, int N);
tman_status mpgemm_plan(int M, int K, int N, int bits, int *out8);
tman_status mpgemm_plan_for(int M, int K, int N, int bits, int sms, int resident, int *out8);
tman_status launch_quantize_rows_i8(const void *x, int M, int K, int8_t *a, float *s_a, cudaStream_t s);
tman_status launch_mpgemm_ternary_i8(const void *packed, const int8_t *a8, const float *row_scale, float w_scale, void *y,
                                     int M, int K, int N, int group, void *ws, cudaStream_t s);
tman_status mpgemm_read_stamps(const void *ws, int ctas, long long *out_host, cudaStream_t s);
tman_status launch_mpgemm_variant(int variant, const void *packed, const void *x, void *y, int M, int K, int N, int bits,
                                  int group, const void *wt_f16, void *ws, size_t ws_bytes, cudaStream_t s);
tman_status launch_mpgemm(const void *packed, const void *x, void *y, int M, int K, int N, int bits,
                          int group, void *ws, size_t ws_bytes, cudaStream_t s);
tman_status launch_microbench(int kind, int arg, void *results, size_t results_bytes, void *buffer, size_t buffer_bytes,
                              cudaStream_t s);
int         cluster_capacity(int threads, int smem_bytes, int cluster);

}  // namespace tman
