// Decode on the warp-level tensor cores: up to eight activation rows times bit-plane weights whose codes become matrix
// operands without a conversion.
//
// Work split.  A warp owns one 128-deep chunk of k for the whole call: its activations (the eight columns of the MMA's
// B operand) stay in 16 registers.  It walks over groups of 32 output columns: a lane's 16-byte load is one plane word
// (32 k) of the four columns of a strip, 8 strips x 4 words a warp.  TK warps with consecutive chunks form a team that
// walks the same groups; a CTA has TC teams (TK x TC <= 16).  CPW = 2: a warp owns two neighbouring chunks, so that K = 4096 needs
// no second CTA and no partial sums through memory; their activations are in shared memory.  After a group the team's sums are added through shared
// memory (one team barrier a group, two buffers); the K-slices of 128 x TK k that different CTAs own are combined through
// fp32 partial sums in the workspace whose "no sum pending" pattern says when they are there (see mpgemv.cu).
//
// Operands.  The plane words of a column are merged (two levels of rotate and bit-select) so that a mask yields two
// codes in the low bits of the two halves of a register: as fp16 these are code x 2^(d - 24), d the field's bit position
// (a half float below 2^-13 is its low eleven bits x 2^-24), exact matrix operands as they stand.  The 2^d is taken out
// of the activations the other operand holds, which are scaled by a power of two per row and chunk (CPW = 2: two chunks) so that
// their largest magnitude lies in [2^14, 2^15); sums are fp32 throughout.  d is at most 7: an activation down to 2^-21 of that largest
// one is exact, a smaller one is rounded to a multiple of 2^-24, an error below 2^-32 of the largest.  Zero-point and scale are applied to
// a block's sum:
// s * (sum - z * sum of the activations).
#pragma once
#include "sm100_ptx.cuh"
#include "common.cuh"

namespace tman {

constexpr int kGemvMaxGroup = 4;               // weight matrices of one grouped call

// "No sum pending": a NaN bit pattern that no floating-point operation returns.
constexpr uint32_t kGemvSentinel = 0x7FA5A5A5u;
constexpr uint32_t kGemvPollLimit = 1u << 21;  // polls of ~0.5 us each: about a second

struct MmaParams {
    const uint8_t  *packed[kGemvMaxGroup];
    const uint8_t  *planes[kGemvMaxGroup];
    const uint2    *scales[kGemvMaxGroup];   // four fp16 scales of a strip and block
    const uint16_t *zeros[kGemvMaxGroup];    // four zero-point nibbles of a strip and block
    __half         *y[kGemvMaxGroup];        // first row of this launch
    int Ng[kGemvMaxGroup];                   // output columns of each matrix
    int grp0[kGemvMaxGroup];                 // first 32-column group of each matrix
    int col0[kGemvMaxGroup];                 // first concatenated column of each matrix
    int count;                               // matrices in this launch
    const __half   *x;                       // first row of this launch
    float          *partials;
    uint32_t       *status;
    int M, K, N;                             // rows in this launch; N = total (concatenated) columns
    int bits, group, group_shift, nblk;
    int groups;                              // 32-column groups of all matrices
    int chunks;                              // 128-deep chunks of k
    int tk, tc, nkappa;                      // warps of a team (4, 8 or 16), teams of a CTA, K-slices
};

__device__ __forceinline__ uint32_t rotl(uint32_t v, int n) { return __funnelshift_l(v, v, n); }
__device__ __forceinline__ uint32_t rotr(uint32_t v, int n) { return __funnelshift_r(v, v, n); }
__device__ __forceinline__ uint32_t comp(const uint4 &v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }
template <int V> struct IntC { static constexpr int value = V; };

// acc += A B (m16n8k16, fp16 operands, fp32 sums); FIRST: acc = A B
template <bool FIRST>
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    if constexpr (FIRST)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
            : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The codes of one plane word (32 codes of a column) as MMA operands.  Word bit 4 j + ph belongs to weight 8 ph + j.
// Level 1: plane 0 and plane 1 rotated by one are merged by a bit-select, for even and for odd ph, into two-bit fields; with 3
// and 4 planes a second merge (rotated by two) makes fields of three or four bits.  In the resulting word X of ph the code of
// weight 8 ph + j sits at bits 4 j + ph and up (rotating instead of shifting keeps the last one whole).
// Level 2: a mask takes the codes of weights j and j + 4 as the two halves of a register, at bit ph (j even) or ph + 4 (j odd;
// j = 2, 3 after a rotation by eight): at most bit 10.
// R = 1: the whole word, ph = 0..3.  R = 2: ph = sub & 1 and 2 + (sub & 1).  R = 4: ph = sub.  (sub: from the lane; the masks
// that depend on it are LaneMasks, kept for the call.)
template <int R> struct LaneMasks {
    uint32_t lvl1, lvl2, m;                  // R = 2, 4: of this lane's first ph
    template <int BITS> __device__ __forceinline__ void set(int sub)
    {
        const int ph = R == 2 ? sub & 1 : sub;
        lvl1 = 0x55555555u << (ph & 1);
        lvl2 = rotl(0x33333333u, ph);
        m = (((1u << BITS) - 1u) * 0x00010001u) << ph;
    }
};
template <int BITS, int R> struct Prep { uint32_t a[R == 1 ? 2 : 1], b[BITS == 4 && R == 1 ? 2 : 1]; };
template <int BITS, int R>
__device__ __forceinline__ void prepare_word(const uint32_t (&w)[BITS], const LaneMasks<R> &lm, Prep<BITS, R> &t)
{
    const uint32_t r1 = rotl(w[1], 1);
    if constexpr (R == 1) {
        t.a[0] = bsel(0x55555555u, w[0], r1);
        t.a[1] = bsel(0xAAAAAAAAu, w[0], r1);
        if constexpr (BITS == 3) t.b[0] = rotl(w[2], 2);
        if constexpr (BITS == 4) {
            const uint32_t r3 = rotl(w[BITS - 1], 1);
            t.b[0] = rotl(bsel(0x55555555u, w[2], r3), 2);
            t.b[1] = rotl(bsel(0xAAAAAAAAu, w[2], r3), 2);
        }
    } else {
        t.a[0] = bsel(lm.lvl1, w[0], r1);
        if constexpr (BITS == 3) t.b[0] = rotl(w[2], 2);
        if constexpr (BITS == 4) t.b[0] = rotl(bsel(lm.lvl1, w[2], rotl(w[BITS - 1], 1)), 2);
    }
}
// Quarter Q: the four pairs (weights 8 ph + j and 8 ph + j + 4, j = 0..3) of ph = Q (R = 1), 2 Q + (sub & 1) (R = 2), sub (R = 4).
template <int BITS, int R, int Q>
__device__ __forceinline__ void quarter_pairs(const Prep<BITS, R> &t, const LaneMasks<R> &lm, uint32_t (&o)[4])
{
    uint32_t X, m;
    if constexpr (R == 1) {
        constexpr uint32_t L2 = Q == 0 ? 0x33333333u : Q == 1 ? 0x66666666u : Q == 2 ? 0xCCCCCCCCu : 0x99999999u;
        m = (((1u << BITS) - 1u) * 0x00010001u) << Q;
        X = t.a[Q & 1];
        if constexpr (BITS == 3) X = bsel(L2, X, t.b[0]);
        if constexpr (BITS == 4) X = bsel(L2, X, t.b[Q & 1]);
    } else {
        m = lm.m << (2 * Q);
        X = t.a[0];
        if constexpr (BITS > 2) X = bsel(Q == 0 ? lm.lvl2 : ~lm.lvl2, X, t.b[0]);
    }
    const uint32_t Y = rotr(X, 8);
    o[0] = X & m; o[1] = X & (m << 4); o[2] = Y & m; o[3] = Y & (m << 4);
}
// The factor 2^-d, d = ph + 4 (j & 1), that the activations carry against the fields' positions.
__device__ __forceinline__ float field_factor(int ph, int j) { return __uint_as_float((uint32_t)(127 - ph - 4 * (j & 1)) << 23); }

__device__ __forceinline__ float4 ld_volatile_f4(const float4 *p)
{
    float4 v;
    asm volatile("ld.volatile.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ bool has_sentinel(const float4 &v)
{
    return __float_as_uint(v.x) == kGemvSentinel || __float_as_uint(v.y) == kGemvSentinel ||
           __float_as_uint(v.z) == kGemvSentinel || __float_as_uint(v.w) == kGemvSentinel;
}
// Bounded wait of the split-K combine: polls up to four partial-sum quads (slices kp, kp + SP, ... below
// nkappa) until none of them holds the "no sum pending" pattern, at most `limit` times.  Returns
// whether they all arrived; the caller reports TMAN_ERR_TIMEOUT otherwise.
__device__ __forceinline__ bool wait_for_sums(const float4 *src, size_t stride4, int kp, int SP, int nkappa,
                                              uint32_t limit, float4 (&t)[4])
{
    bool ready = false;
    for (uint32_t tries = 0; !ready && tries < limit; ++tries) {
        ready = true;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (kp + q * SP < nkappa) t[q] = ld_volatile_f4(src + (size_t)(kp + q * SP) * stride4);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (kp + q * SP < nkappa) ready = ready && !has_sentinel(t[q]);
    }
    return ready;
}

constexpr int kMmaThreads = 512;
template <int BITS, int R, int NE, int CPW> struct MmaCfg {
    static constexpr int RED_WARP = 8 * 128;                                     // a warp's sums of a group: 8 columns of B x 32 columns
    static constexpr int RED_BYTES = 2 * 16 * RED_WARP;
    static constexpr int SCALE_BYTES = 16 * 8 * 4;                               // the power-of-two scale of every (column of B, warp)
    static constexpr int FRAG_CHUNK = 2048 + R * NE * 128;                       // a warp's activations of a chunk: B fragments, block sums
    static constexpr int PATCH_WARP = R > 1 ? BITS * 512 : 0;                    // R > 1: a group's plane words, redistributed among lanes
    static constexpr int SMEM = RED_BYTES + SCALE_BYTES + 16 * (PATCH_WARP + (CPW > 1 ? CPW * FRAG_CHUNK : 0));
    static constexpr int DEPTH = BITS == 2 ? 4 : 2;                              // groups whose loads are in flight per warp
};

// How the eight columns of B are used:
//   R = 1: column = block of the chunk x T + row, T = 8 / NB rows (NE = 2), NB = 128 / group blocks; a lane whose word lies in
//          another block than its column holds zeros.  NE = 1: only the even columns (T = 4 / NB rows), one value per accumulator pair.
//   R = 2, 4: column = row; the chunk's blocks of 64 / 32 k are multiplied one after the other, a lane's word in halves / quarters.
template <int BITS, int R, int NB, int NE, int CPW>
__global__ void __launch_bounds__(kMmaThreads, 1) decode_mma_kernel(const MmaParams p)
{
    using C = MmaCfg<BITS, R, NE, CPW>;
    constexpr int DEPTH = C::DEPTH;
    constexpr int T = (NE == 2 ? 8 : 4) / NB;                                    // rows the columns hold
    static_assert(R == 1 || (NB == 1 && NE == 2), "sub-word passes use all eight columns for rows");
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
    const int TK = p.tk, team = warp / TK, wk = warp - team * TK;                // this warp's team and place in it
    const int kappa = blockIdx.y, P = gridDim.x;
    const int words = p.K >> 5;
    constexpr int csh = CPW - 1;
    const int chunk = (kappa * TK + wk) * CPW;                                   // this warp's first chunk
    const bool active = chunk < p.chunks, both = CPW > 1 && chunk + 1 < p.chunks;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // ---- weight stream: groups g = first, first + stride, ... -------------------------------------------
    const int g_first = blockIdx.x + P * team, g_stride = P * p.tc;
    const uint32_t row_bytes = (uint32_t)words * 16u, strip_bytes = row_bytes * BITS;
    const uint32_t lane_off = (uint32_t)((active ? chunk : 0) * 4 + tig) * 16u;
    const int lane_blk = R == 1 ? (NE == 2 ? 2 * tig : tig) / T : tig & (R - 1); // block of the chunk whose scales this lane fetches
    const uint32_t blk_off = (uint32_t)((((active ? chunk : 0) << 7) >> p.group_shift) + lane_blk);
    uint4 wbuf[DEPTH][BITS];
    uint2 sbuf[DEPTH];
    uint32_t zbuf[DEPTH];
    auto matrix_of = [&](int g) {
        int mtx = 0;
#pragma unroll
        for (int t = 1; t < kGemvMaxGroup; ++t) mtx += (t < p.count && g >= p.grp0[t]) ? 1 : 0;
        return mtx;
    };
    auto load = [&](int g, int c, uint4 (&w)[BITS], uint2 &sc, uint32_t &z) {
        if (!(c ? both : active)) return;
        const int gc = min(g, p.groups - 1), mtx = matrix_of(gc);               // past the last group: the last again, never used
        const int nb = min((gc - p.grp0[mtx]) * 8 + gid, (p.Ng[mtx] >> 2) - 1);
        const uint8_t *q = p.planes[mtx] + (size_t)nb * strip_bytes + lane_off + 64 * c;
#pragma unroll
        for (int i = 0; i < BITS; ++i) w[i] = __ldcs(reinterpret_cast<const uint4 *>(q + (size_t)i * row_bytes));
        const size_t blk = (size_t)nb * p.nblk + blk_off + (uint32_t)(c << (7 - p.group_shift));
        sc = __ldg(p.scales[mtx] + blk);
        z = __ldg(p.zeros[mtx] + blk);
    };
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) load(g_first + (d >> csh) * g_stride, d & csh, wbuf[d], sbuf[d], zbuf[d]);

    bool hdr_ok = true;
#pragma unroll
    for (int g = 0; g < kGemvMaxGroup; ++g)
        if (g < p.count) {
            const uint4 h0 = __ldg(reinterpret_cast<const uint4 *>(p.packed[g])), h1 = __ldg(reinterpret_cast<const uint4 *>(p.packed[g]) + 1);
            hdr_ok = hdr_ok && h0.x == 0x4E414D54u && h0.y == 0x30303242u && h0.z == kVersion && h0.w == (uint32_t)p.K &&
                     h1.x == (uint32_t)p.Ng[g] && h1.y == (uint32_t)p.bits && h1.z == (uint32_t)p.group && h1.w == 4u;
        }

    // Everything below may depend on the previous kernel in the stream (activations, workspace).
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- this warp's activations: B fragments, block sums and scales ---------------------------------------
    // (of two chunks in shared memory, written and read by the same lane; of one in registers)
    uint4 xb1[4];
    float S1[R][NE];
    uint8_t *const frags = smem + C::RED_BYTES + C::SCALE_BYTES + 16 * C::PATCH_WARP + warp * (CPW * C::FRAG_CHUNK);
    float *const row_back = reinterpret_cast<float *>(smem + C::RED_BYTES);      // [B column][warp]: what undoes the scaling
    LaneMasks<R> lm;
    lm.template set<BITS>(R == 2 ? tig >> 1 : tig);
    {
        const int col = NE == 2 ? gid : gid >> 1;                                // B column of this lane
        const int b_row = col % T, b_blk = col / T;
        const bool live = b_row < p.M && (NE == 2 || !(gid & 1)) && (R > 1 || NB == 1 || (tig * NB) / 4 == b_blk);
        uint4 raw[CPW][4];
        float amax;
        __half2 mx = __floats2half2_rn(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < CPW; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int word = R == 1 ? tig : R == 2 ? 2 * (i >> 1) + (tig & 1) : i;
                const int ph = R == 1 ? i : R == 2 ? (tig >> 1) + 2 * (i & 1) : tig;
                raw[c][i] = make_uint4(0u, 0u, 0u, 0u);
                if (live && (c ? both : active))
                    raw[c][i] = ld_dependent(reinterpret_cast<const uint4 *>(p.x + (size_t)b_row * p.K + (size_t)(chunk + c) * 128 + word * 32 + ph * 8));
            }
#pragma unroll
        for (int c = 0; c < CPW; ++c)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t u = comp(raw[c][i], e);
                    mx = __hmax2(mx, __habs2(*reinterpret_cast<const __half2 *>(&u)));
                }
        amax = fmaxf(__low2float(mx), __high2float(mx));
#pragma unroll
        for (int mask = 1; mask < 4; mask <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, mask));
        const uint32_t be = min(__float_as_uint(amax) >> 23, 240u);              // amax = 1.f * 2^(be - 127)
        const float fac = __uint_as_float((be ? 268u - be : 127u) << 23);
        const float back = __uint_as_float((be ? be + 10u : 151u) << 23);         // 2^24 / fac
#pragma unroll
        for (int c = 0; c < CPW; ++c) {
            float sum[R];
#pragma unroll
            for (int b = 0; b < R; ++b) sum[b] = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t u = comp(raw[c][i], e);
                    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&u));
                    sum[R == 1 ? 0 : R == 2 ? i >> 1 : i] += f.x + f.y;
                }
#pragma unroll
            for (int mask = 1; mask < 4; mask <<= 1)
#pragma unroll
                for (int b = 0; b < R; ++b) sum[b] += __shfl_xor_sync(0xffffffffu, sum[b], mask);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                uint32_t xb[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t u0 = comp(raw[c][i], j >> 1), u1 = comp(raw[c][i], 2 + (j >> 1));
                    const __half2 h0 = *reinterpret_cast<const __half2 *>(&u0), h1 = *reinterpret_cast<const __half2 *>(&u1);
                    const float f = fac * field_factor(R == 1 ? i : R == 2 ? (tig >> 1) + 2 * (i & 1) : tig, j);
                    const __half2 h = __floats2half2_rn((j & 1 ? __high2float(h0) : __low2float(h0)) * f,
                                                        (j & 1 ? __high2float(h1) : __low2float(h1)) * f);
                    xb[j] = *reinterpret_cast<const uint32_t *>(&h);
                }
                if constexpr (CPW == 1) xb1[i] = make_uint4(xb[0], xb[1], xb[2], xb[3]);
                else *reinterpret_cast<uint4 *>(frags + c * C::FRAG_CHUNK + i * 512 + lane * 16) = make_uint4(xb[0], xb[1], xb[2], xb[3]);
            }
            // activation sums of the accumulator columns this lane holds, in the sums' units (against zero-points held as z x 2^-24)
#pragma unroll
            for (int b = 0; b < R; ++b)
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    const float v = __shfl_sync(0xffffffffu, sum[b] * fac, 4 * (2 * tig + e));   // a lane of that B column
                    if constexpr (CPW == 1) S1[b][e] = v;
                    else *reinterpret_cast<float *>(frags + c * C::FRAG_CHUNK + 2048 + (b * NE + e) * 128 + lane * 4) = v;
                }
        }
        if (tig == 0 && (NE == 2 || !(gid & 1))) row_back[col * 16 + warp] = back;
    }

    if (!hdr_ok) {                                   // the same answer in every CTA: outputs stay untouched
        if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_BAD_PACKED);
        return;
    }

    // ---- one group: 32 columns x this warp's 128 k ----------------------------------------------------------
    uint8_t *red = smem;
    uint8_t *patch = smem + C::RED_BYTES + C::SCALE_BYTES + warp * C::PATCH_WARP;
    auto group_sums = [&](const uint8_t *frag, const uint4 (&wr)[BITS], uint2 sc_l, uint32_t z_l, float4 (&out)[NE]) {
        float tot[2][2][NE];
#pragma unroll
        for (int gg = 0; gg < R; ++gg) {
            uint4 w[BITS];
            if constexpr (R == 1) {
#pragma unroll
                for (int i = 0; i < BITS; ++i) w[i] = wr[i];
            } else {
                const int from = R == 2 ? gid * 4 + 2 * gg + (tig & 1) : gid * 4 + gg;
#pragma unroll
                for (int i = 0; i < BITS; ++i) w[i] = *reinterpret_cast<const uint4 *>(patch + i * 512 + from * 16);
            }
            float acc[2][4];
            Prep<BITS, R> pw[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t ww[BITS];
#pragma unroll
                for (int i = 0; i < BITS; ++i) ww[i] = comp(w[i], c);
                prepare_word<BITS, R>(ww, lm, pw[c]);
            }
            auto quarter = [&](auto qc) {
                constexpr int Q = decltype(qc)::value;
                const uint4 bq = CPW == 1 ? xb1[(4 / R) * gg + Q] : *reinterpret_cast<const uint4 *>(frag + ((4 / R) * gg + Q) * 512 + lane * 16);
                const uint32_t b[4] = {bq.x, bq.y, bq.z, bq.w};
                uint32_t o[4][4];
#pragma unroll
                for (int c = 0; c < 4; ++c) quarter_pairs<BITS, R, Q>(pw[c], lm, o[c]);
#pragma unroll
                for (int s = 0; s < 2; ++s) mma16816<Q == 0>(acc[s], o[2 * s][0], o[2 * s + 1][0], o[2 * s][1], o[2 * s + 1][1], b[0], b[1]);
#pragma unroll
                for (int s = 0; s < 2; ++s) mma16816<false>(acc[s], o[2 * s][2], o[2 * s + 1][2], o[2 * s][3], o[2 * s + 1][3], b[2], b[3]);
            };
            quarter(IntC<0>());
            if constexpr (R <= 2) quarter(IntC<1>());
            if constexpr (R == 1) { quarter(IntC<2>()); quarter(IntC<3>()); }
            uint2 sc = sc_l;
            uint32_t z = z_l;
            if constexpr (R > 1) {
                sc.x = __shfl_sync(0xffffffffu, sc_l.x, gid * 4 + gg);
                sc.y = __shfl_sync(0xffffffffu, sc_l.y, gid * 4 + gg);
                z = __shfl_sync(0xffffffffu, z_l, gid * 4 + gg);
            }
            // zero-points as fp16 subnormals: nibbles of channels (0, 2) and, sixteen-fold, (1, 3)
            const uint32_t zp = __byte_perm(z, 0u, 0x4140);
            const uint32_t ze = zp & 0x000F000Fu, zo = zp & 0x00F000F0u;
            const float2 zef = __half22float2(*reinterpret_cast<const __half2 *>(&ze));
            const float2 zof = __half22float2(*reinterpret_cast<const __half2 *>(&zo));
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const uint32_t su = s ? sc.y : sc.x;
                const float2 sf = __half22float2(*reinterpret_cast<const __half2 *>(&su));
                const float z0 = s ? zef.y : zef.x, z1 = s ? zof.y : zof.x;
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    const float S = CPW == 1 ? S1[gg][e] : *reinterpret_cast<const float *>(frag + 2048 + (gg * NE + e) * 128 + lane * 4);
                    const float t0 = fmaf(-z0, S, acc[s][e]), t1 = fmaf(-z1, S * 0.0625f, acc[s][2 + e]);
                    tot[s][0][e] = gg == 0 ? sf.x * t0 : fmaf(sf.x, t0, tot[s][0][e]);
                    tot[s][1][e] = gg == 0 ? sf.y * t1 : fmaf(sf.y, t1, tot[s][1][e]);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) out[e] = make_float4(tot[0][0][e], tot[0][1][e], tot[1][0][e], tot[1][1][e]);
    };
    // shared-memory place of four columns (strip) of B column vc of a warp's sums; the XOR spreads a store over the banks
    auto red_at = [&](int buf, int w, int vc, int strip) { return red + ((buf * 16 + w) * 8 + vc) * 128 + ((strip ^ vc) & 7) * 16; };

    if (!active)                                     // a warp without a chunk: its sums are zero for the whole call
        for (int b = 0; b < 2; ++b)
            for (int q = lane; q < 64; q += 32)
                *reinterpret_cast<float4 *>(red + ((b * 16 + warp) * 8) * 128 + q * 16) = make_float4(0.f, 0.f, 0.f, 0.f);

    // the team's sums of its rows of a group: 32 columns, one per lane
    auto finish_group = [&](int g, int buf, int turn) {
        const int mtx = matrix_of(g);
        const int n = (g - p.grp0[mtx]) * 32 + lane;
        for (int m = (wk - turn) & (TK - 1); m < p.M; m += TK) {
            float v = 0.f;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int vc = b * T + m;
                const uint8_t *src = red_at(buf, team * TK, vc, lane >> 2) + (lane & 3) * 4;
                const float4 *back = reinterpret_cast<const float4 *>(row_back + vc * 16 + team * TK);
                for (int w = 0; w < TK; w += 4, src += 4 * C::RED_WARP, ++back) {
                    float t[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) t[q] = *reinterpret_cast<const float *>(src + q * C::RED_WARP);
                    const float4 f = *back;
                    v = fmaf(t[0], f.x, v); v = fmaf(t[1], f.y, v); v = fmaf(t[2], f.z, v); v = fmaf(t[3], f.w, v);
                }
            }
            if (n >= p.Ng[mtx]) continue;
            if (p.nkappa > 1) p.partials[((size_t)kappa * p.M + m) * p.N + p.col0[mtx] + n] = v;
            else p.y[mtx][(size_t)m * p.Ng[mtx] + n] = __float2half_rn(v);
        }
    };

    // own accumulator columns in shared memory (+ buffer x 16 warps)
    uint8_t *my_red[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) my_red[e] = red_at(0, warp, NE == 2 ? 2 * tig + e : tig, gid);
    int turn = 0, flip = 0;
    float4 out[NE];
#pragma unroll 1
    for (int g0 = g_first; g0 < p.groups; g0 += (DEPTH >> csh) * g_stride) {
#pragma unroll
        for (int d = 0; d < DEPTH; ++d) {
            const int g = g0 + (d >> csh) * g_stride, c = d & csh;
            if (g >= p.groups) break;                // uniform over the team
            if (c ? both : active) {
                if constexpr (R > 1) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < BITS; ++i) *reinterpret_cast<uint4 *>(patch + i * 512 + lane * 16) = wbuf[d][i];
                    __syncwarp();
                }
                float4 cur[NE];
                group_sums(frags + c * C::FRAG_CHUNK, wbuf[d], sbuf[d], zbuf[d], cur);
                load(g + (DEPTH >> csh) * g_stride, c, wbuf[d], sbuf[d], zbuf[d]);
#pragma unroll
                for (int e = 0; e < NE; ++e) {
                    if (CPW > 1 && c) { cur[e].x += out[e].x; cur[e].y += out[e].y; cur[e].z += out[e].z; cur[e].w += out[e].w; }
                    out[e] = cur[e];
                }
            }
            if (c != csh) continue;                  // the group's second chunk follows
            if (active) {
#pragma unroll
                for (int e = 0; e < NE; ++e)
                    if ((NE == 2 ? 2 * tig + e : tig) % T < p.M)
                        *reinterpret_cast<float4 *>(my_red[e] + flip * 16 * C::RED_WARP) = out[e];
            }
            asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(TK * 32) : "memory");
            finish_group(g, flip, turn);
            turn += p.M;
            flip ^= 1;
        }
    }

    // ---- combine K-slices: every CTA polls the partial sums of its share of the columns ----------
    if (p.nkappa > 1) {
        const int nthreads = blockDim.x;
        const int cta = blockIdx.y * gridDim.x + blockIdx.x, G = gridDim.x * gridDim.y;
        const int ng = p.N >> 2;
        const int g_lo = (int)(((long long)ng * cta) / G), g_hi = (int)(((long long)ng * (cta + 1)) / G);
        const int col_lo = g_lo * 4;
        const int ngrp = g_hi - g_lo;
        const int items = ngrp * p.M;                       // one item = four columns of one row
        const size_t stride4 = (size_t)p.M * p.N / 4;
        // SP adjacent lanes share an item and split the slices among them (slice kp goes to lane
        // kp % SP); their sums are added in a fixed order, so the result does not depend on timing
        int SP = 1;
        while (SP < 8 && 2 * SP <= p.nkappa && items * 2 * SP <= nthreads) SP *= 2;
        const int part = tid & (SP - 1);
        const float sv = __uint_as_float(kGemvSentinel);
        bool gave_up = false;
        for (int item0 = 0; item0 < items; item0 += nthreads / SP) {
            const int item = item0 + tid / SP;
            const bool alive = item < items;
            const int m = alive ? item / ngrp : 0, n = col_lo + 4 * (alive ? item % ngrp : 0);
            float4 *src = reinterpret_cast<float4 *>(p.partials + (size_t)m * p.N + n);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int kp = part; alive && kp < p.nkappa; kp += 4 * SP) {
                float4 t[4];
                if (!wait_for_sums(src, stride4, kp, SP, p.nkappa, kGemvPollLimit, t)) { gave_up = true; break; }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (kp + q * SP < p.nkappa) {
                        acc.x += t[q].x; acc.y += t[q].y; acc.z += t[q].z; acc.w += t[q].w;
                        src[(size_t)(kp + q * SP) * stride4] = make_float4(sv, sv, sv, sv);
                    }
            }
            for (int mask = 1; mask < SP; mask <<= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, mask);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, mask);
                acc.z += __shfl_xor_sync(0xffffffffu, acc.z, mask);
                acc.w += __shfl_xor_sync(0xffffffffu, acc.w, mask);
            }
            gave_up = __any_sync(0xffffffffu, gave_up);
            if (alive && part == 0 && !gave_up) {
                const __half2 h01 = __floats2half2_rn(acc.x, acc.y), h23 = __floats2half2_rn(acc.z, acc.w);
                uint2 o;
                o.x = *reinterpret_cast<const uint32_t *>(&h01);
                o.y = *reinterpret_cast<const uint32_t *>(&h23);
                const int g = [&] {
                    int t = 0;
#pragma unroll
                    for (int i = 1; i < kGemvMaxGroup; ++i) t += (i < p.count && n >= p.col0[i]) ? 1 : 0;
                    return t;
                }();
                *reinterpret_cast<uint2 *>(p.y[g] + (size_t)m * p.Ng[g] + (n - p.col0[g])) = o;
            }
        }
        if (gave_up) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_TIMEOUT);
    }
}

}  // namespace tman
