// Offline repack into the bit-plane layout, its inverse, and the test-only extractors.
// Pure integer work; every result has exactly one correct value.
#include "sm100_ptx.cuh"
#include "common.cuh"
#include <algorithm>
#include <mutex>
#include <vector>

namespace tman {

// The whole repack is one launch, bound by HBM: codes read once, packed words written once.
//   Plane blocks (the first `plane_blocks`): a tile of 32 strips (128 columns) x 8 words (256 k), one warp per word.
//     A lane owns one strip: it reads the four codes of a row as one 32-bit load (a warp reads 128 bytes of a row, 32
//     rows in flight per thread: five blocks an SM leave the registers for that, eight do not) and turns four rows' codes
//     at a time into bytes of the planes' words (bit transpose); a 4 x 4 byte transpose then gives the words of the four columns (paper Sec. 2.2: W = sum_i 2^i W_i).
//     The words go through shared memory so that eight adjacent words of a strip and plane leave as one 128-byte run:
//     written straight from the lanes they would be 16-byte pieces (half a sector) K/2 bytes apart.
//   Scale blocks (the rest): one thread per strip and four quantization blocks, 32 bytes of scales in one piece.
//   The first block also writes the header and zeroes the padding between sections, so that the whole buffer is a
//     function of the inputs.
// Byte loads, 16-byte pieces and four launches took 65.7 us for 4096 x 14336 4-bit codes (88 MB: 13.6 us at the copy
// rate).  With a shift and a mask per code bit and eight blocks an SM 20.6 us (2-bit 18.9); so 18.1 (17.5).
// VEC: codes and zeros are 4-byte aligned and scales 8-byte aligned (N % 8 == 0 keeps every row so); otherwise the same
// elements are read one by one.
constexpr int kPackThreads = 256, kPackStrips = 32, kPackWords = 8;

template <int BITS, bool VEC>
__global__ void __launch_bounds__(kPackThreads, 5) pack_kernel(const uint8_t *__restrict__ codes, const __half *__restrict__ scales,
                                                            const uint8_t *__restrict__ zeros, uint8_t *__restrict__ packed,
                                                            int K, int N, int group, int strip_tiles, int plane_blocks)
{
    __shared__ uint4 tile[BITS * kPackStrips * kPackWords];
    const Layout L = make_layout(K, N, BITS, group);
    const int words = K / 32, strips = N / 4;
    if ((int)blockIdx.x < plane_blocks) {
        const int st0 = ((int)blockIdx.x % strip_tiles) * kPackStrips, v0 = ((int)blockIdx.x / strip_tiles) * kPackWords;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int nb = st0 + lane, v = v0 + warp;
        if (nb < strips && v < words) {
            const uint8_t *src = codes + (size_t)(32 * v) * N + (size_t)4 * nb;
            uint32_t u[32];                                // byte c = code of column c, row r
#pragma unroll
            for (int r = 0; r < 32; ++r, src += N) {
                if constexpr (VEC) u[r] = __ldcs(reinterpret_cast<const uint32_t *>(src));
                else u[r] = (uint32_t)src[0] | ((uint32_t)src[1] << 8) | ((uint32_t)src[2] << 16) | ((uint32_t)src[3] << 24);
            }
            // Word bit 8 b + 4 h + ph is row 8 ph + 2 b + h: byte b of a plane is, per column, a 4 x 4 bit transpose of four
            // rows' codes, for h = 0 in the low nibbles and h = 1 in the high ones.
            uint32_t by[4][4];                             // [plane][b]: byte c = byte b of column c's word
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                uint32_t r[4];
#pragma unroll
                for (int ph = 0; ph < 4; ++ph) r[ph] = bsel(0x0F0F0F0Fu, u[8 * ph + 2 * b], u[8 * ph + 2 * b + 1] << 4);
                const uint32_t t0 = bsel(0x55555555u, r[0], r[1] << 1), t1 = bsel(0x55555555u, r[0] >> 1, r[1]);
                const uint32_t t2 = bsel(0x55555555u, r[2], r[3] << 1), t3 = bsel(0x55555555u, r[2] >> 1, r[3]);
                by[0][b] = bsel(0x33333333u, t0, t2 << 2);
                by[1][b] = bsel(0x33333333u, t1, t3 << 2);
                by[2][b] = bsel(0x33333333u, t0 >> 2, t2);
                by[3][b] = bsel(0x33333333u, t1 >> 2, t3);
            }
#pragma unroll
            for (int i = 0; i < BITS; ++i) {
                const uint32_t lo01 = __byte_perm(by[i][0], by[i][1], 0x5140), hi01 = __byte_perm(by[i][0], by[i][1], 0x7362);
                const uint32_t lo23 = __byte_perm(by[i][2], by[i][3], 0x5140), hi23 = __byte_perm(by[i][2], by[i][3], 0x7362);
                const uint4 w = make_uint4(__byte_perm(lo01, lo23, 0x5410), __byte_perm(lo01, lo23, 0x7632),
                                           __byte_perm(hi01, hi23, 0x5410), __byte_perm(hi01, hi23, 0x7632));
                // (word index XOR strip: the lanes of a store spread over all banks)
                tile[(i * kPackStrips + lane) * kPackWords + (warp ^ (lane & 7))] = w;
            }
        }
        __syncthreads();
        uint4 *planes = reinterpret_cast<uint4 *>(packed + L.planes_off);
#pragma unroll
        for (int e = threadIdx.x; e < BITS * kPackStrips * kPackWords; e += kPackThreads) {
            const int vv = e % kPackWords, st = (e / kPackWords) % kPackStrips, i = e / (kPackWords * kPackStrips);
            if (st0 + st < strips && v0 + vv < words)
                __stcs(planes + ((size_t)(st0 + st) * BITS + i) * words + v0 + vv,
                       tile[(i * kPackStrips + st) * kPackWords + (vv ^ (st & 7))]);
        }
    } else {
        const int nblk = K / group, quads = (nblk + 3) / 4;
        const long tid = (long)((int)blockIdx.x - plane_blocks) * kPackThreads + threadIdx.x;
        if (tid < (long)strips * quads) {
            const int nb = (int)(tid % strips), B0 = (int)(tid / strips) * 4;
            uint2 sc[4];
            uint16_t zz[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const size_t at = (size_t)min(B0 + q, nblk - 1) * N + (size_t)4 * nb;
                uint32_t z;
                if constexpr (VEC) {
                    sc[q] = __ldg(reinterpret_cast<const uint2 *>(scales + at));
                    z = __ldg(reinterpret_cast<const uint32_t *>(zeros + at));
                } else {
                    const uint16_t *h = reinterpret_cast<const uint16_t *>(scales) + at;
                    sc[q] = make_uint2((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16));
                    z = (uint32_t)zeros[at] | ((uint32_t)zeros[at + 1] << 8) | ((uint32_t)zeros[at + 2] << 16) | ((uint32_t)zeros[at + 3] << 24);
                }
                z &= 0x0F0F0F0Fu;                          // four zero-points -> nibbles
                zz[q] = (uint16_t)((z & 0xFu) | ((z >> 4) & 0xF0u) | ((z >> 8) & 0xF00u) | ((z >> 12) & 0xF000u));
            }
            uint2 *ps = reinterpret_cast<uint2 *>(packed + L.scales_off) + (size_t)nb * nblk;
            uint16_t *pz = reinterpret_cast<uint16_t *>(packed + L.zeros_off) + (size_t)nb * nblk;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (B0 + q < nblk) {
                    ps[B0 + q] = sc[q];
                    pz[B0 + q] = zz[q];
                }
        }
    }
    if (blockIdx.x == 0) {
        const int t = threadIdx.x;                         // header words and, byte by byte, the (< 256 each) padding bytes
        if (t < (int)(kHeaderBytes / 4)) {
            uint32_t h = 0u;
            if (t == 0) h = 0x4E414D54u;                   // "TMAN"
            else if (t == 1) h = 0x30303242u;              // "B200"
            else if (t == 2) h = kVersion;
            else if (t == 3) h = (uint32_t)K;
            else if (t == 4) h = (uint32_t)N;
            else if (t == 5) h = (uint32_t)BITS;
            else if (t == 6) h = (uint32_t)group;
            else if (t == 7) h = 4u;
            else if (t < 16) {
                const uint64_t off = t < 10 ? L.planes_off : t < 12 ? L.scales_off : t < 14 ? L.zeros_off : L.total;
                h = (uint32_t)(off >> (32 * (t & 1)));
            }
            reinterpret_cast<uint32_t *>(packed)[t] = h;
        }
        const size_t from[3] = {L.planes_off + L.planes_bytes, L.scales_off + L.scales_bytes, L.zeros_off + L.zeros_bytes};
        const size_t to[3] = {L.scales_off, L.zeros_off, L.total};
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (from[q] + t < to[q]) packed[from[q] + t] = 0;
    }
}

// Streams on which a packed buffer has been written since the last decode launch.  The decode kernel
// reads weights before it waits for its predecessor when launched with programmatic stream
// serialization, so launch_mpgemv asks here and falls back to plain stream order once after a pack.
static std::mutex g_pending_mutex;
static std::vector<cudaStream_t> g_pending_streams;
static std::atomic<size_t> g_pending_count;

void note_packed_write(cudaStream_t s)
{
    std::lock_guard<std::mutex> lock(g_pending_mutex);
    if (std::find(g_pending_streams.begin(), g_pending_streams.end(), s) == g_pending_streams.end())
        g_pending_streams.push_back(s);
    g_pending_count.store(g_pending_streams.size(), std::memory_order_release);
}

bool packed_write_pending(cudaStream_t s, bool clear)
{
    if (g_pending_count.load(std::memory_order_acquire) == 0) return false;      // no packing since the last decode call: no lock
    std::lock_guard<std::mutex> lock(g_pending_mutex);
    auto it = std::find(g_pending_streams.begin(), g_pending_streams.end(), s);
    if (it == g_pending_streams.end()) return false;
    if (clear) {
        g_pending_streams.erase(it);
        g_pending_count.store(g_pending_streams.size(), std::memory_order_release);
    }
    return true;
}

template <int BITS>
static void launch_pack_bits(bool vec, const uint8_t *codes, const void *scales, const uint8_t *zeros, int K, int N, int group,
                             void *packed, cudaStream_t s)
{
    const int strips = N / 4, strip_tiles = (strips + kPackStrips - 1) / kPackStrips;
    const long plane_blocks = (long)strip_tiles * ((K / 32 + kPackWords - 1) / kPackWords);
    const long scale_threads = (long)strips * ((K / group + 3) / 4);
    const unsigned grid = (unsigned)(plane_blocks + (scale_threads + kPackThreads - 1) / kPackThreads);
    auto kern = vec ? pack_kernel<BITS, true> : pack_kernel<BITS, false>;
    kern<<<grid, kPackThreads, 0, s>>>(codes, static_cast<const __half *>(scales), zeros, static_cast<uint8_t *>(packed), K, N,
                                       group, strip_tiles, (int)plane_blocks);
}

tman_status launch_pack(const uint8_t *codes, const void *scales, const uint8_t *zeros, int K, int N,
                        int bits, int group, void *packed, cudaStream_t s)
{
    const auto low = [](const void *q) { return reinterpret_cast<uintptr_t>(q); };
    const bool vec = ((low(codes) | low(zeros)) & 3) == 0 && (low(scales) & 7) == 0;
    if (bits == 1) launch_pack_bits<1>(vec, codes, scales, zeros, K, N, group, packed, s);
    else if (bits == 2) launch_pack_bits<2>(vec, codes, scales, zeros, K, N, group, packed, s);
    else if (bits == 3) launch_pack_bits<3>(vec, codes, scales, zeros, K, N, group, packed, s);
    else launch_pack_bits<4>(vec, codes, scales, zeros, K, N, group, packed, s);
    note_packed_write(s);
    return launch_status();
}

// ---- inverse -----------------------------------------------------------------------------
__global__ void unpack_kernel(const uint8_t *__restrict__ packed, uint8_t *__restrict__ codes,
                              __half *__restrict__ scales, uint8_t *__restrict__ zeros,
                              uint32_t *status, int K, int N, int bits, int group)
{
    if (!header_matches(packed, K, N, bits, group)) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicCAS(status, 0u, (uint32_t)TMAN_ERR_BAD_PACKED);
        return;
    }
    Layout L = make_layout(K, N, bits, group);
    const uint32_t *planes = reinterpret_cast<const uint32_t *>(packed + L.planes_off);
    long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long total = (long)(K / 32) * N;
    if (tid < total) {
        int n = (int)(tid % N), v = (int)(tid / N);
        int nb = n >> 2, c = n & 3;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        for (int i = 0; i < bits; ++i) w[i] = planes[(((size_t)nb * bits + i) * (K / 32) + v) * 4 + c];
        for (int r = 0; r < 32; ++r) {
            uint32_t q = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) q |= ((w[i] >> plane_bit(r)) & 1u) << i;
            codes[(size_t)(32 * v + r) * N + n] = (uint8_t)q;
        }
    }
    int nblk = K / group;
    if (tid < (long)nblk * N) {
        int n = (int)(tid % N), B = (int)(tid / N);
        int nb = n >> 2, c = n & 3;
        const __half *ps = reinterpret_cast<const __half *>(packed + L.scales_off);
        const uint16_t *pz = reinterpret_cast<const uint16_t *>(packed + L.zeros_off);
        scales[(size_t)B * N + n] = ps[((size_t)nb * nblk + B) * 4 + c];
        zeros[(size_t)B * N + n] = (uint8_t)((pz[(size_t)nb * nblk + B] >> (4 * c)) & 0xF);
    }
}

tman_status launch_unpack(const void *packed, int K, int N, int bits, int group, uint8_t *codes,
                          void *scales, uint8_t *zeros, uint32_t *status, cudaStream_t s)
{
    long total = (long)(K / 32) * N;   // >= (K/group)*N because group >= 32
    unpack_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(
        static_cast<const uint8_t *>(packed), codes, static_cast<__half *>(scales), zeros, status,
        K, N, bits, group);
    return launch_status();
}

// ---- test-only extractors ------------------------------------------------------------------
// idx[i][t][n] = the 4-bit table index of activations 4t .. 4t+3 (plane i, column n), gathered from
// the bits of plane word (i, t / 8, n) that hold those four weights.
__global__ void debug_indices_kernel(const uint8_t *__restrict__ packed, uint8_t *__restrict__ idx,
                                     uint32_t *status, int K, int N, int bits, int group)
{
    if (!header_matches(packed, K, N, bits, group)) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicCAS(status, 0u, (uint32_t)TMAN_ERR_BAD_PACKED);
        return;
    }
    Layout L = make_layout(K, N, bits, group);
    const uint32_t *planes = reinterpret_cast<const uint32_t *>(packed + L.planes_off);
    long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long total = (long)bits * (K / 32) * N;
    if (tid >= total) return;
    int n = (int)(tid % N);
    long r = tid / N;
    int v = (int)(r % (K / 32));
    int i = (int)(r / (K / 32));
    uint32_t w = planes[(((size_t)(n >> 2) * bits + i) * (K / 32) + v) * 4 + (n & 3)];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        uint32_t x = 0;
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) x |= ((w >> plane_bit(4 * e + jj)) & 1u) << jj;
        idx[((size_t)i * (K / 4) + 8 * v + e) * N + n] = (uint8_t)x;
    }
}

// ---- per-tensor ternary weights -> INT8 by two table lookups (paper Sec. 4.1 / Fig. 7, Sec. 6.2) -----------
// One thread takes the two plane words of 32 consecutive k of the four columns of a strip.  Level 1 (bit
// repacking): the planes are interleaved into 2-bit codes, eight to a register in k order, one code per
// nibble (the packed format's bit permutation makes a shift and a bit-select do it).  Level 2 (conversion
// table): a four-entry byte table {-1, 0, +1, 0} held in one register, looked up four codes at a time with
// a byte permute whose selector is the codes themselves.  Output: int8 [N][K], 32 bytes per thread and
// column, consecutive threads on consecutive k.
__global__ void dequant_ternary_int8_kernel(const uint8_t *__restrict__ packed, int8_t *__restrict__ w8,
                                            uint32_t *status, int K, int N, int group)
{
    if (!header_matches(packed, K, N, 2, group)) {
        if (threadIdx.x == 0 && blockIdx.x == 0) atomicCAS(status, 0u, (uint32_t)TMAN_ERR_BAD_PACKED);
        return;
    }
    const Layout L = make_layout(K, N, 2, group);
    const int words = K / 32;
    const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= (long)(N / 4) * words) return;
    const int nb = (int)(tid / words), v = (int)(tid % words);
    const uint4 *planes = reinterpret_cast<const uint4 *>(packed + L.planes_off);
    const uint4 w0 = __ldg(planes + ((size_t)nb * 2 + 0) * words + v);
    const uint4 w1 = __ldg(planes + ((size_t)nb * 2 + 1) * words + v);
    const uint32_t table = 0x000100FFu;              // byte c = value of code c: -1, 0, +1, (3 does not occur) 0
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint32_t p0 = c == 0 ? w0.x : c == 1 ? w0.y : c == 2 ? w0.z : w0.w;
        const uint32_t p1 = c == 0 ? w1.x : c == 1 ? w1.y : c == 2 ? w1.z : w1.w;
        // word bit 4j + ph belongs to weight 8ph + j: a0 holds, in its even bit pairs... interleave planes bit by bit
        const uint32_t a0 = (p0 & 0x55555555u) | ((p1 << 1) & 0xAAAAAAAAu);      // codes of the even word bits
        const uint32_t a1 = ((p0 >> 1) & 0x55555555u) | (p1 & 0xAAAAAAAAu);      // codes of the odd word bits
        uint32_t X[4];                               // X[ph]: nibble j = code of weight 8ph + j
        X[0] = a0 & 0x33333333u;
        X[2] = (a0 >> 2) & 0x33333333u;
        X[1] = a1 & 0x33333333u;
        X[3] = (a1 >> 2) & 0x33333333u;
        uint32_t out[8];
#pragma unroll
        for (int ph = 0; ph < 4; ++ph) {
            out[2 * ph] = __byte_perm(table, 0u, X[ph]);             // weights 8ph .. 8ph+3
            out[2 * ph + 1] = __byte_perm(table, 0u, X[ph] >> 16);   // weights 8ph+4 .. 8ph+7
        }
        uint4 *dst = reinterpret_cast<uint4 *>(w8 + ((size_t)(4 * nb + c) * K + (size_t)32 * v));
        dst[0] = make_uint4(out[0], out[1], out[2], out[3]);
        dst[1] = make_uint4(out[4], out[5], out[6], out[7]);
    }
}

tman_status launch_dequant_ternary_int8(const void *packed, int K, int N, int group, int8_t *w8, uint32_t *status,
                                        cudaStream_t s)
{
    const long total = (long)(N / 4) * (K / 32);
    dequant_ternary_int8_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(static_cast<const uint8_t *>(packed), w8,
                                                                             status, K, N, group);
    return launch_status();
}

tman_status launch_debug_indices(const void *packed, int K, int N, int bits, int group, uint8_t *idx,
                                 uint32_t *status, cudaStream_t s)
{
    long total = (long)bits * (K / 32) * N;
    debug_indices_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(
        static_cast<const uint8_t *>(packed), idx, status, K, N, bits, group);
    return launch_status();
}

__global__ void debug_luts_kernel(const __half *__restrict__ x, float *__restrict__ lut, int M, int K)
{
    long tid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    long total = (long)M * (K / 4);
    if (tid >= total) return;
    const __half *px = x + tid * 4;
    float t[16];
    lut16(__half2float(px[0]), __half2float(px[1]), __half2float(px[2]), __half2float(px[3]), t);
#pragma unroll
    for (int p = 0; p < 16; ++p) lut[tid * 16 + p] = t[p];
}

tman_status launch_debug_luts(const void *x, int M, int K, float *lut, cudaStream_t s)
{
    long total = (long)M * (K / 4);
    debug_luts_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(static_cast<const __half *>(x),
                                                                      lut, M, K);
    return launch_status();
}

}  // namespace tman
