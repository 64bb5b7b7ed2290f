// Decode of one and two rows on the warp-level integer tensor cores: codes as bytes against activations cut into 8-bit digits.
//
// Arithmetic.  A row's activations of a block of k become 32-bit integers (a power of two brings the largest to
// [2^29, 2^30)) and those four signed 8-bit digits, the columns of the MMA's B operand (mma.sync.m16n8k32, unsigned x signed bytes,
// 32-bit sums, exact).  The codes' bytes are plane words merged by rotations and bit-selects, two codes of three or four bits (four of two)
// a byte.  They are not taken apart completely: an operand holds a byte's lowest fields f0, f0 + 16 f1 and so on, and
// the activations carry the differences, x0 - x1 / 16 for f0 and x1 / 16 for f0 + 16 f1, so that the last operand needs no mask.
// Zero-point and scale are applied to a block's sum, s * (sum - z * sum of the activations), in fp32.
// Exactness: an activation of a field is an integer after the field's power of two has been taken out, rounded by at most 2^-26 (3 and 4
// bits) or 2^-24 (2 bits) of the largest of its block (blocks may have scales of any size); everything up to a block's sum is exact
// then, the rest fp32.
//
// Work split.  A CTA owns all of k for its columns, so that nothing is summed through global memory: its eight warps are teams that
// have the chunks of k among them and take the groups of 32 columns in turn; the warps' sums meet in shared memory once.  The CTA is
// small (half an SM's registers and shared memory), so that the next call's starts beside it: it reads its scales, fills its rings with
// weights and waits for this one there.
//
// What bounds it: issue slots and integer pipe, about 190 instructions (97 on the half-rate integer pipe, 76 of them the merging) per 32
// columns x 128 k, and at the ends 0.8 us from the predecessor's last store to this call's activations, 1.0 us until their digits are
// there, 0.4 us for the sums; HBM at the large end (4096 x 28672, 4-bit group 128 13.5 us, 4.6 TB/s; by lookup 15.9).  Measured and
// dropped: 16 warps of 64 registers, two CTAs an SM (spills: 19.3), 16 warps of 128 registers, one (14.9; 4096 x 4096 4.5 against
// 4.2), scales by ordinary loads a unit ahead (4096 x 6144 6.5 against 5.9), rings of 64-byte pieces of eight strips (as fast).
#pragma once
#include "decode_mma.cuh"

namespace tman {

constexpr int kDigitGroups = 40;               // groups of eight strips that a CTA takes at most
// Shared memory of a CTA: half of the common split (common.cuh) where it fits, else all of it.
constexpr int kDigitSmem = 130 * 1024, kDigitSmemHalf = 65 * 1024;

// A group of a CTA: up to eight neighbouring strips of one matrix.
struct DigitGroup {
    const uint8_t *planes;                     // of its first strip
    __half        *y;                          // of its first column
    int strips, Ng, n0, s0;                    // its first column; its first strip among the CTA's
};

struct DigitParams {
    const uint8_t *packed[kGemvMaxGroup];
    const uint8_t *planes[kGemvMaxGroup];
    const uint8_t *scales[kGemvMaxGroup];
    const uint8_t *zeros[kGemvMaxGroup];
    __half        *y[kGemvMaxGroup];           // first row of this launch
    int Ng[kGemvMaxGroup];                     // output columns of each matrix
    int strip0[kGemvMaxGroup + 1];             // first concatenated strip (four columns) of each matrix; the last one's end from entry `count` on
    int count;                                 // matrices in this launch
    const void    *x;                          // first row of this launch: fp16, or the integer path's 16-bit integers
    const float   *row_scale;                  // integer path: scale of each row, of the tensor, and the sums (may be null)
    float          w_scale;
    int32_t       *acc_out;
    uint32_t      *status;
    int M, K, nblk, bits, group;
    int chunks, pairs;                         // 128-deep chunks of k; units are two of them
    int strips_q, strips_r;                    // strips of a CTA: the quotient, one more in the first `strips_r` CTAs
    int tk_shift, pairs_q, pairs_r;            // warps of a team (a power of two), which have the pairs of chunks among them in the same way
    int scale_row, zero_row;                   // bytes of a strip's scales and zero-points in shared memory
    int tc;                                    // teams, which have the groups in turn
    int flush;                                 // turns of groups between two reductions over the warps
    uint32_t by_rows;                          // 2^31 / M, rounded up
};

// DEPTH: units of two chunks under way per warp.
constexpr int kDigitWarps = 8, kDigitWarpsShift = 3;
template <int BITS, int NB, int DEPTH> struct DigitCfg {
    static constexpr int STAGE = BITS * 512;                     // a warp's planes of a chunk
    static constexpr int ROW = 512;                              // digits of a row's chunk
    static constexpr int ROW_SCALES = NB * 16;                   // what undoes the scaling and the block's sum, for both digit pairs
    static constexpr int RING = kDigitWarps * DEPTH * 2 * STAGE;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) { asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async8(uint32_t dst, const void *src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src) { asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }
__device__ __forceinline__ uint4 lds128(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y) { asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory"); }
__device__ __forceinline__ void sts128(uint32_t a, uint4 v) { asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory"); }

// acc += A B (m16n8k32, A unsigned bytes, B signed bytes, 32-bit sums); FIRST: acc = A B
template <bool FIRST>
__device__ __forceinline__ void mma16832(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    if constexpr (FIRST)
        asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
            : "=r"(c[0]), "=r"(c[1]), "=r"(c[2]), "=r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
    else
        asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// One column's plane words as byte operands: step ks of four, part 0 and part 1 (the byte's fields below the part's own and that one).
// Word bit 4 j + ph belongs to weight 8 ph + j.  3 and 4 bits: step = ph, byte b holds the codes of j = 2 b and 2 b + 1, part 0 the first.
// 2 bits: step 2 p + h, byte b holds (ph, j) = (p, 2 b), (p + 2, 2 b), (p, 2 b + 1), (p + 2, 2 b + 1), two bits each; part i of step h
// the fields up to 2 h + i.
template <int BITS> struct CodeBytes {
    uint32_t a[2], b[2];
    __device__ __forceinline__ void prepare(const uint32_t (&w)[BITS])
    {
        const uint32_t r1 = rotl(w[1], 1);
        a[0] = bsel(0x55555555u, w[0], r1);
        a[1] = bsel(0xAAAAAAAAu, w[0], r1);
        if constexpr (BITS == 2) a[1] = rotr(a[1], 1);
        if constexpr (BITS == 3) b[0] = b[1] = rotl(w[BITS - 1], 2);
        if constexpr (BITS == 4) {
            const uint32_t r3 = rotl(w[BITS - 1], 1);
            b[0] = rotl(bsel(0x55555555u, w[BITS - 2], r3), 2);
            b[1] = rotl(bsel(0xAAAAAAAAu, w[BITS - 2], r3), 2);
        }
    }
    template <int KS> __device__ __forceinline__ void operands(uint32_t &part0, uint32_t &part1) const
    {
        if constexpr (BITS == 2) {
            const uint32_t x = a[KS >> 1];
            part0 = x & ((KS & 1) ? 0x3F3F3F3Fu : 0x03030303u);
            part1 = (KS & 1) ? x : x & 0x0F0F0F0Fu;
        } else {
            constexpr uint32_t M = KS == 0 ? 0x33333333u : KS == 1 ? 0x66666666u : KS == 2 ? 0xCCCCCCCCu : 0x99999999u;
            const uint32_t x = rotr(bsel(M, a[KS & 1], b[KS & 1]), KS);
            part0 = x & (BITS == 3 ? 0x07070707u : 0x0F0F0F0Fu);
            part1 = BITS == 3 ? x & 0x77777777u : x;
        }
    }
};

// How the eight columns of an n-tile are used; column = 2 x (lane & 3) + e, digit 0 the most significant.  NB = blocks of a chunk:
//   NB = 1: four digits of rows 2 t and 2 t + 1 (t = n-tile).   NB = 2: four digits of row t, block 0 and block 1; a word of the other
//   block meets zeros.   NB = 4: two digits (those of pair t & 1) of row t >> 1, blocks 0..3.
// NT = n-tiles.  INT: 2-bit codes, zero-point 1, 16-bit integer activations (times 64, 16, 4, 1 by their field, so that three digits hold
// them): the sums stay 32-bit integers to the end.  (Four tiles of it spill 76 bytes: seven rows 2048 x 2176 and back 16.8 us, by lookup 24.8.)
template <int BITS, int NB, int NT, int DEPTH, bool INT>
__global__ void __launch_bounds__(32 * kDigitWarps, 2) decode_digits_kernel(const __grid_constant__ DigitParams p)
{
    using C = DigitCfg<BITS, NB, DEPTH>;
    constexpr int WARPS = kDigitWarps, THREADS = 32 * WARPS;
    static_assert(!INT || (BITS == 2 && NB == 1), "the integer path: 2-bit codes, one block");
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    const int M = p.M;
    const int tc_shift = kDigitWarpsShift - p.tk_shift, team = warp >> p.tk_shift, wk = warp & ((1 << p.tk_shift) - 1);
    // shared memory: rings, groups, activations' digits, their scales and sums, zeros for the words of
    // other blocks, sums of the warps
    const uint32_t sm = (uint32_t)__cvta_generic_to_shared(smem);
    DigitGroup *const groups = reinterpret_cast<DigitGroup *>(smem + C::RING);
    const int slots = 2 * p.pairs;
    const uint32_t slot_bytes = (uint32_t)M * C::ROW, slot_scales = (uint32_t)M * C::ROW_SCALES;
    const uint32_t digits = sm + C::RING + kDigitGroups * sizeof(DigitGroup), scal = digits + slots * slot_bytes;
    const uint32_t zeros_at = scal + slots * slot_scales;
    const uint32_t scale_rows = zeros_at + (NB > 1 ? slot_bytes : 0u);
    const uint32_t zero_rows = scale_rows + (uint32_t)(p.strips_q + (p.strips_r ? 1 : 0)) * (uint32_t)p.scale_row;
    const uint32_t red = (zero_rows + (uint32_t)(p.strips_q + (p.strips_r ? 1 : 0)) * (uint32_t)p.zero_row + 15u) & ~15u;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- this CTA's strips in groups; this warp's chunks -----------------------------------------------------------------
    const int s_lo = p.strips_q * blockIdx.x + min((int)blockIdx.x, p.strips_r);
    const int s_hi = s_lo + p.strips_q + ((int)blockIdx.x < p.strips_r ? 1 : 0);
    const int pair0 = p.pairs_q * wk + min(wk, p.pairs_r), np = p.pairs_q + (wk < p.pairs_r ? 1 : 0), c0 = 2 * pair0;
    const bool odd = (p.chunks & 1) && pair0 + np == p.pairs;                    // the last pair has one chunk
    const uint32_t row_bytes = (uint32_t)p.K >> 1, strip_bytes = row_bytes * BITS;    // a plane of a strip: K / 32 words of four columns
    int ngroups = 0;
#pragma unroll
    for (int m = 0; m < kGemvMaxGroup; ++m) {
        const int lo = max(s_lo, p.strip0[m]), hi = min(s_hi, p.strip0[m + 1]);
        if (hi <= lo) continue;
        const int n = (hi - lo + 7) >> 3, at = tid - ngroups;
        if (at >= 0 && at < n) {
            const int s = lo + 8 * at, local = s - p.strip0[m];
            DigitGroup d;
            d.planes = p.planes[m] + (size_t)local * strip_bytes;
            d.y = p.y[m] + local * 4;
            d.strips = min(8, hi - s);
            d.Ng = p.Ng[m];
            d.n0 = local * 4;
            d.s0 = s - s_lo;
            groups[tid] = d;
        }
        ngroups += n;
    }
    const int lane_blk = NB == 1 ? 0 : NB == 2 ? tig >> 1 : tig;                 // the block whose scale this lane applies
    __syncthreads();

    // ---- scales and zero-points of all strips: a row each, its zero-points from a four-byte boundary on ------------
    if constexpr (!INT) {
        for (int s = s_lo + warp; s < s_hi; s += WARPS) {
            int m = 0;
#pragma unroll
            for (int t = 1; t < kGemvMaxGroup; ++t) m += s >= p.strip0[t] && t < p.count ? 1 : 0;
            const size_t at = (size_t)(s - p.strip0[m]) * (uint32_t)p.nblk;
            const uint8_t *sc = p.scales[m] + at * 8, *z = p.zeros[m] + (at >> 1) * 4;
            const uint32_t sc_row = scale_rows + (uint32_t)((s - s_lo) * p.scale_row), z_row = zero_rows + (uint32_t)((s - s_lo) * p.zero_row);
            for (int i = lane; i < p.nblk; i += 32) cp_async8(sc_row + i * 8, sc + (size_t)i * 8);
            for (int i = lane; i < (p.nblk + (int)(at & 1) + 1) >> 1; i += 32) cp_async4(z_row + i * 4, z + (size_t)i * 4);
        }
    }
    cp_async_commit();

    // ---- weight stream: units of eight strips x 256 k; a copy takes 128 bytes of four strips -------------------------
    const uint32_t ring = sm + (uint32_t)warp * (DEPTH * 2 * C::STAGE);
    int f_group = team, f_left = 0, f_strips = 0;
    uint32_t f_dst = ring + (uint32_t)((lane >> 3) * 128 + ((lane & 7) ^ ((lane >> 1) & 4)) * 16);      // (odd strips: halves swapped)
    const uint32_t f_end = f_dst + DEPTH * 2 * C::STAGE;
    const uint8_t *f_src = nullptr;
    auto fetch_group = [&]() {
        f_left = np;
        f_strips = 0;
        if (f_group < ngroups && np > 0) {
            const DigitGroup &d = groups[f_group];
            f_strips = d.strips - (lane >> 3);                                   // this lane's strip, and the fourth after it, if positive
            f_src = d.planes + (size_t)((lane >> 3) * strip_bytes + (uint32_t)(c0 * 64 + (lane & 7) * 16));
        }
        f_group += p.tc;
    };
    auto fetch = [&]() {
        if (f_strips > 0 && !(odd && f_left == 1 && (lane & 4))) {
#pragma unroll
            for (int i = 0; i < BITS; ++i) cp_async16(f_dst + i * 1024, f_src + (size_t)i * row_bytes);
            if (f_strips > 4) {
#pragma unroll
                for (int i = 0; i < BITS; ++i) cp_async16(f_dst + i * 1024 + 512, f_src + (size_t)(4 * BITS + i) * row_bytes);
            }
        }
        cp_async_commit();
        f_src += 128;
        f_dst += 2 * C::STAGE;
        if (f_dst == f_end) f_dst -= DEPTH * 2 * C::STAGE;
        if (--f_left == 0) fetch_group();
    };
    fetch_group();
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) fetch();

    bool bad = false;
    if (tid < 8 * p.count) {
        const int m = tid >> 3, q = tid & 7;
        const uint32_t want[8] = {0x4E414D54u, 0x30303242u, kVersion, (uint32_t)p.K, (uint32_t)p.Ng[m], (uint32_t)p.bits, (uint32_t)p.group, 4u};
        uint32_t v = want[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) v = q == i ? want[i] : v;
        bad = __ldg(reinterpret_cast<const uint32_t *>(p.packed[m]) + q) != v;
    }
    if constexpr (NB > 1)
        for (uint32_t i = tid * 16; i < slot_bytes; i += THREADS * 16) sts128(zeros_at + i, make_uint4(0u, 0u, 0u, 0u));

    // Everything below may depend on the previous kernel in the stream (activations).
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- activations to digits: half a warp a job, job = (chunk, row), eight activations a lane ------------------------
    const int half = lane >> 4, aw = (lane >> 2) & 3, aph = lane & 3;
    const int njobs = slots * M;                                                 // (a chunk beyond the last: zeros)
    auto load_job = [&](int j) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (j < njobs) {
            const int c = (int)__umulhi((uint32_t)j * 2u, p.by_rows), r = j - c * M;
            if (c < p.chunks) v = ld_dependent(reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(p.x) + (size_t)r * p.K + (size_t)c * 128 + aw * 32 + aph * 8));
        }
        return v;
    };
    auto run_job = [&](int j, const uint4 &raw) {
        const int c = (int)__umulhi((uint32_t)j * 2u, p.by_rows), r = j - c * M;
        const uint32_t slot = (uint32_t)c;
        const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
        int lo[4], hi[4];                                                        // the activations 2 i and 2 i + 1 as integers of their fields
        uint32_t back_hi = 0, back_lo = 0, sum_bits = 0;
        if constexpr (INT) {
            int sum = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                lo[i] = (int)(int16_t)(rw[i] & 0xFFFFu);
                hi[i] = (int)rw[i] >> 16;
                sum += lo[i] + hi[i];
                lo[i] <<= aph < 2 ? 6 : 4;
                hi[i] <<= aph < 2 ? 2 : 0;
            }
#pragma unroll
            for (int mask = 1; mask < 16; mask <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, mask);
            sum_bits = (uint32_t)sum;
        } else {
            uint32_t big = 0;
            float f[8], sum = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                big = __vmaxu2(big, rw[i] & 0x7FFF7FFFu);
                const float2 t = __half22float2(*reinterpret_cast<const __half2 *>(&rw[i]));
                f[2 * i] = t.x;
                f[2 * i + 1] = t.y;
            }
            big = max(big & 0xFFFFu, big >> 16);                                 // of the block: 16 / NB lanes
#pragma unroll
            for (int mask = 1; mask < 16 / NB; mask <<= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, mask));
            const uint32_t e = max(big >> 10, 1u);                               // biased exponent of the block's largest
            back_hi = (99u + e) << 23;                                           // 2^16 / factor
            back_lo = (83u + e) << 23;
            float fac = __uint_as_float((171u - e) << 23);                       // 2^(29 - exponent)
            if (__any_sync(0xffffffffu, e == 31u)) {
                // Infinities and NaN.  A block of one infinity takes it alone (finite values are nothing beside it) and is multiplied
                // back by infinity: an infinity, or NaN where its code is the zero-point.  More of them may cancel column by column,
                // which their sum does not show, so that such a block is NaN, as one with a NaN in it.
                int infs = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) infs += isinf(f[i]) ? 1 : 0;
#pragma unroll
                for (int mask = 1; mask < 16 / NB; mask <<= 1) infs += __shfl_xor_sync(0xffffffffu, infs, mask);
                if (e == 31u) {
                    fac = 1.f;
                    back_hi = big > 0x7C00u || infs > 1 ? 0x7FC00000u : 0x7F800000u;
                    back_lo = 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i) f[i] = isinf(f[i]) ? copysignf(268435456.f, f[i]) : 0.f;
                }
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) sum += f[i];
#pragma unroll
            for (int mask = 1; mask < 16 / NB; mask <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, mask);
            // in the upper digit pair's units, against zero-points held as z x 2^-24
            sum_bits = __float_as_uint(sum * fac * 256.f);
            const float flo = BITS > 2 || aph < 2 ? fac : fac * 0.25f;
            const float fhi = BITS > 2 || aph < 2 ? fac * 0.0625f : fac * 0.015625f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                lo[i] = __float2int_rn(f[2 * i] * flo);
                hi[i] = __float2int_rn(f[2 * i + 1] * fhi);
            }
        }
        uint32_t v0[4], v1[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            int d0, d1;
            if constexpr (BITS > 2) {
                d1 = hi[i];
                d0 = lo[i] - d1;
            } else {
                // fields 0, 2 are this lane's (aph < 2) or 1, 3; the neighbours in the byte belong to lane aph ^ 2
                const int other = __shfl_xor_sync(0xffffffffu, aph < 2 ? hi[i] : lo[i], 2);
                d0 = aph < 2 ? lo[i] - other : other - hi[i];
                d1 = aph < 2 ? other - hi[i] : hi[i];
            }
            v0[i] = ((uint32_t)d0 + 0x00808080u) ^ 0x00808080u;                  // signed digits
            v1[i] = ((uint32_t)d1 + 0x00808080u) ^ 0x00808080u;
        }
        auto transpose = [](const uint32_t (&v)[4], uint32_t (&o)[4]) {          // o[d]: digit d (0 the most significant) of the four
            const uint32_t t0 = __byte_perm(v[0], v[1], 0x5140), t1 = __byte_perm(v[2], v[3], 0x5140);
            const uint32_t t2 = __byte_perm(v[0], v[1], 0x7362), t3 = __byte_perm(v[2], v[3], 0x7362);
            o[3] = __byte_perm(t0, t1, 0x5410); o[2] = __byte_perm(t0, t1, 0x7632);
            o[1] = __byte_perm(t2, t3, 0x5410); o[0] = __byte_perm(t2, t3, 0x7632);
        };
        uint32_t o0[4], o1[4];
        transpose(v0, o0);
        transpose(v1, o1);
        if (j < njobs) {
            // step of this lane's bytes: ph, or (2 bits) 2 x (ph & 1) + (ph >> 1)
            const uint32_t ks = BITS > 2 ? (uint32_t)aph : (uint32_t)(2 * (aph & 1) + (aph >> 1));
            const uint32_t at = digits + slot * slot_bytes + (uint32_t)r * C::ROW + (ks >> 1) * 256u + (uint32_t)aw * 16u + (ks & 1u) * 8u;
#pragma unroll
            for (int d = 0; d < 4; ++d) sts64(at + d * 64, o0[d], o1[d]);
            if ((lane & (16 / NB - 1)) == 0) {
                const uint32_t b = (uint32_t)((lane & 15) / (16 / NB));
                sts128(scal + slot * slot_scales + (uint32_t)r * C::ROW_SCALES + b * 16u, make_uint4(back_hi, sum_bits, back_lo, 0u));
            }
        }
    };
    {
        uint4 cur = load_job(2 * warp + half);
        for (int j = 2 * warp; j < njobs; j += 2 * WARPS) {
            const uint4 nxt = load_job(j + 2 * WARPS + half);
            run_job(j + half, cur);
            cur = nxt;
        }
    }
    cp_async_wait<DEPTH>();                                                      // (the scales)
    __syncthreads();

    // ---- what this lane reads of them: the digits of its B columns, the scales of its accumulator columns -------------
    // (row of n-tile t, before M limits it; the digit; whether the lane's word lies in the column's block)
    const bool b_live = NB == 1 || (NB == 2 ? (tig >> 1) == (gid >> 2) : tig == (gid >> 1));
    auto b_offset = [&](int t) {
        const int row = NB == 1 ? 2 * t + (gid >> 2) : NB == 2 ? t : t >> 1;
        const int d = NB == 4 ? 2 * (t & 1) + (gid & 1) : gid & 3;
        return (uint32_t)(min(row, M - 1) * C::ROW + (d * 4 + tig) * 16);
    };
    auto acc_row = [&](int t) { return NB == 1 ? 2 * t + (tig >> 1) : NB == 2 ? t : t >> 1; };
    uint32_t b_at[NT], s_at[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
        b_at[t] = (b_live ? digits + (uint32_t)c0 * slot_bytes : zeros_at) + b_offset(t);
        const int pair = NB == 4 ? t & 1 : tig & 1;
        s_at[t] = scal + (uint32_t)c0 * slot_scales + (uint32_t)(min(acc_row(t), M - 1) * C::ROW_SCALES + lane_blk * 16 + pair * 8);
    }
    const uint32_t b_step = b_live ? slot_bytes : 0u;
    const bool low_pair = INT && (tig & 1) != 0;

    int turn = 0, first_turn = 0;
    uint32_t src = ring;
    const int turns = (ngroups + p.tc - 1) >> tc_shift;                               // the first team's
    const uint32_t src_lane[2] = {(uint32_t)(gid * 128 + (tig + 4 * (gid & 1)) * 16), (uint32_t)(gid * 128 + (tig + 4 * (1 - (gid & 1))) * 16)};
#pragma unroll 1
    for (int g = team;; g += p.tc, ++turn) {
        float out[NT][4];                                                        // (INT: 32-bit integers)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) out[t][c] = 0.f;
        const int n_units = g < ngroups ? np : 0;
        uint32_t sc_at = 0, z_at = 0;
        if (!INT && n_units > 0) {
            const DigitGroup &d = groups[g];
            const int s = d.s0 + min(gid, d.strips - 1);
            sc_at = scale_rows + (uint32_t)(s * p.scale_row + (c0 * NB + lane_blk) * 8);
            z_at = zero_rows + (uint32_t)(s * p.zero_row + ((((d.n0 >> 2) + min(gid, d.strips - 1)) & p.nblk & 1) + c0 * NB + lane_blk) * 2);
        }
        uint32_t b_slot = 0, s_slot = 0;                                         // of the unit's first chunk, from this warp's first
#pragma unroll 1
        for (int u = 0; u < n_units; ++u) {
            cp_async_wait<DEPTH - 1>();
            __syncwarp();
            uint4 w2[2][BITS];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < BITS; ++i) w2[h][i] = lds128(src + src_lane[h] + i * 1024);
            src += 2 * C::STAGE;
            if (src == ring + DEPTH * 2 * C::STAGE) src = ring;
            __syncwarp();                                                        // (all lanes have read the stage)
            fetch();
            auto chunk = [&](auto hc, const uint4 (&w)[BITS]) {
                constexpr int H = decltype(hc)::value;
                const uint32_t b_off = b_slot + H * b_step, s_off = s_slot + H * slot_scales;
                uint2 sc = make_uint2(0u, 0u);
                [[maybe_unused]] uint32_t z = 0;
                if constexpr (!INT) {
                    sc = lds64(sc_at + H * NB * 8);
                    z = lds16(z_at + H * NB * 2);
                }
                uint4 b[NT];
#pragma unroll
                for (int t = 0; t < NT; ++t) b[t] = lds128(b_at[t] + b_off);
                CodeBytes<BITS> cb[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint32_t ww[BITS];
#pragma unroll
                    for (int i = 0; i < BITS; ++i) ww[i] = comp(w[i], q);
                    cb[q].prepare(ww);
                }
                int acc[NT][2][4];
                auto step = [&](auto ksc, const uint4 (&b)[NT]) {
                    constexpr int KS = decltype(ksc)::value;
                    uint32_t p0[4], p1[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) cb[q].template operands<KS>(p0[q], p1[q]);
#pragma unroll
                    for (int t = 0; t < NT; ++t)
#pragma unroll
                        for (int s = 0; s < 2; ++s)
                            mma16832<KS == 0>(acc[t][s], p0[2 * s], p0[2 * s + 1], p1[2 * s], p1[2 * s + 1], (KS & 1) ? b[t].z : b[t].x,
                                              (KS & 1) ? b[t].w : b[t].y);
                };
                step(IntC<0>(), b);
                step(IntC<1>(), b);
#pragma unroll
                for (int t = 0; t < NT; ++t) b[t] = lds128(b_at[t] + b_off + 256u);
                step(IntC<2>(), b);
                step(IntC<3>(), b);
                if constexpr (INT) {
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        const int S = (int)lds32(s_at[t] + s_off + (low_pair ? 0u : 4u));      // (the low pair: no sum)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int v = acc[t][q >> 1][2 * (q & 1)] * 256 + acc[t][q >> 1][2 * (q & 1) + 1];
                            const int add = low_pair ? v >> 6 : v * 1024 - S;
                            out[t][q] = __int_as_float(__float_as_int(out[t][q]) + add);
                        }
                    }
                } else {
                    const uint32_t zp = __byte_perm(z, 0u, 0x4140);
                    const uint32_t ze = zp & 0x000F000Fu, zo = zp & 0x00F000F0u;    // as fp16 subnormals; columns 1 and 3 sixteen-fold
                    const float2 zef = __half22float2(*reinterpret_cast<const __half2 *>(&ze));
                    const float2 zof = __half22float2(*reinterpret_cast<const __half2 *>(&zo));
                    const float2 s01 = __half22float2(*reinterpret_cast<const __half2 *>(&sc.x));
                    const float2 s23 = __half22float2(*reinterpret_cast<const __half2 *>(&sc.y));
                    const float zf[4] = {-zef.x, -zof.x, -zef.y, -zof.y}, sf[4] = {s01.x, s01.y, s23.x, s23.y};
#pragma unroll
                    for (int t = 0; t < NT; ++t) {
                        const uint2 bs = lds64(s_at[t] + s_off);
                        const float back = __uint_as_float(bs.x), S = __uint_as_float(bs.y), S16 = S * 0.0625f;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int v = acc[t][q >> 1][2 * (q & 1)] * 256 + acc[t][q >> 1][2 * (q & 1) + 1];
                            const float u = fmaf(zf[q], (q & 1) ? S16 : S, (float)v);
                            out[t][q] = fmaf(sf[q] * back, u, out[t][q]);
                        }
                    }
                }
            };
            chunk(IntC<0>(), w2[0]);
            if (!(odd && u + 1 == np)) chunk(IntC<1>(), w2[1]);
            sc_at += 2 * NB * 8;
            z_at += 2 * NB * 2;
            b_slot += 2 * b_step;
            s_slot += 2 * slot_scales;
        }
        // ---- the lanes' sums of this group: digit pairs and blocks, then the warps' through shared memory -------------
        auto add = [](float a, float b) { return INT ? __int_as_float(__float_as_int(a) + __float_as_int(b)) : a + b; };
        const int at_turn = turn - first_turn;
        constexpr int ROWS = NB == 4 ? NT / 2 : NT;
#pragma unroll
        for (int t = 0; t < ROWS; ++t) {
            float v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = NB == 4 ? out[2 * t][q] + out[2 * t + (NB == 4 ? 1 : 0)][q] : out[t][q];
                v[q] = add(v[q], __shfl_xor_sync(0xffffffffu, v[q], 1));
                if constexpr (NB > 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], 2);
            }
            const int row = NB == 1 ? 2 * t + (tig >> 1) : t;
            if ((NB == 1 ? (tig & 1) == 0 : tig == 0) && row < M)
                sts128(red + (uint32_t)(((warp * p.flush + at_turn) * M + row) * 8 + gid) * 16u,
                       make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3])));
        }
        const bool last = turn + 1 >= turns;
        if (at_turn + 1 < p.flush && !last) continue;
        if (__syncthreads_or(bad)) {                                             // the same answer in every CTA: outputs stay untouched
            if (tid == 0 && blockIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_BAD_PACKED);
            cp_async_wait<0>();
            return;
        }
        const int items = (at_turn + 1) * p.tc * M * 8;
        for (int it = tid; it < items; it += THREADS) {
            const int strip = it & 7, gr = it >> 3, gs = (int)__umulhi((uint32_t)gr * 2u, p.by_rows), row = gr - gs * M, tm = gs & (p.tc - 1);
            const int tn = gs >> tc_shift, gq = first_turn * p.tc + gs;
            if (gq >= ngroups || strip >= groups[gq].strips) continue;
            const uint32_t at = red + (uint32_t)((((tm << p.tk_shift) * p.flush + tn) * M + row) * 8 + strip) * 16u, step_b = (uint32_t)(p.flush * M) * 128u;
            uint4 v = lds128(at);
            float r0 = __uint_as_float(v.x), r1 = __uint_as_float(v.y), r2 = __uint_as_float(v.z), r3 = __uint_as_float(v.w);
#pragma unroll 4
            for (int wq = 1; wq < 1 << p.tk_shift; ++wq) {
                v = lds128(at + wq * step_b);
                r0 = add(r0, __uint_as_float(v.x)); r1 = add(r1, __uint_as_float(v.y));
                r2 = add(r2, __uint_as_float(v.z)); r3 = add(r3, __uint_as_float(v.w));
            }
            const int Ng = groups[gq].Ng;
            if constexpr (INT) {
                const int4 ia = make_int4(__float_as_int(r0), __float_as_int(r1), __float_as_int(r2), __float_as_int(r3));
                if (p.acc_out) *reinterpret_cast<int4 *>(p.acc_out + (size_t)row * Ng + groups[gq].n0 + 4 * strip) = ia;
                const float f = ld_dependent(p.row_scale + row) * p.w_scale;
                r0 = (float)ia.x * f; r1 = (float)ia.y * f; r2 = (float)ia.z * f; r3 = (float)ia.w * f;
            }
            const __half2 h01 = __floats2half2_rn(r0, r1), h23 = __floats2half2_rn(r2, r3);
            *reinterpret_cast<uint2 *>(groups[gq].y + (size_t)row * Ng + 4 * strip) =
                make_uint2(*reinterpret_cast<const uint32_t *>(&h01), *reinterpret_cast<const uint32_t *>(&h23));
        }
        if (last) return;
        first_turn = turn + 1;
        __syncthreads();
    }
}

}  // namespace tman
