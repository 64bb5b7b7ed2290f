// Decode path: bit-serial table-lookup mpGEMV (paper Sec. 2.2 "Bit-serial table lookup", Fig. 2;
// Sec. 4.3 "Mapping of LUT-based Decoding").
//
// One and two activation rows (and three and four where that is faster, uses_mma below) by table lookup, described here, or, short
// reductions, on the integer tensor cores (decode_digits.cuh) where uses_digits says so; more rows on the tensor cores (decode_mma.cuh).
//
// Work split.  The reduction dimension is cut into K-slices of 16 or 32 plane words (16 for one
// activation row; 32, 16 for 2, 3-4 rows, whose table entries carry the rows as fp16 pairs).  One
// CTA owns one K-slice: it builds that slice's
// activation tables in shared memory once and reuses them for every output column it visits
// (the paper's "maximise reuse of cached lookup tables").  Inside a warp a lane owns ONE plane
// word, i.e. 32 consecutive activations = four 8-activation table groups, and one shared-memory
// bank column: tables are stored entry-major so that lane v always reads bank(s) of slot v,
// whatever its index.  Any mix of indices across the warp is therefore conflict-free, which is
// what allows 8-bit indices (two of the paper's 4-bit indices fused: one lookup covers eight
// weights of one bit-plane).
//
// Per lane and column: sum_i 2^i * sum_{4 groups} T[group][index byte]  (shift-accumulate).
// Lanes whose words share a quantization block are added first (one shuffle stage), then the
// zero-point times the block's activation sum is subtracted and the block scale applied, then the
// remaining lanes of the K-slice are reduced with a transposing shuffle reduction.  K-slices are
// combined through fp32 partial sums in the workspace.  The partial-sum area holds a sentinel bit
// pattern (a NaN no arithmetic produces) wherever no sum is pending; once its lookups are done,
// every CTA polls the sums of its share of the output columns until none of them is the sentinel,
// adds them in a fixed order, writes fp16 and puts the sentinel back.  The data are their own
// "ready" flag, so no fence and no counter sits between the last lookup and the output; the poll
// is bounded and reports TMAN_ERR_TIMEOUT.
//
// Streaming.  A warp works through units (a few strips of four columns).  Every strip's registers are
// refilled with the next unit's strip as soon as its lookups are done, so HBM reads overlap the lookups.  The first
// loads (header words, first unit) are issued before the kernel waits for the previous kernel in
// the stream (programmatic dependent launch); the host has checked that every read derived from
// (K, N, bits, group) is in bounds.  That is only sound while the previous kernel does not write the
// packed buffer: the host launches the call that follows a tman_pack_weights on the same stream
// in plain stream order instead (packed_write_pending below), and the header states the rule for
// kernels of the caller's own.
#include "decode_mma.cuh"
#include "decode_digits.cuh"

namespace tman {

constexpr int kGemvThreads = 512;
constexpr int kGemvWarps = kGemvThreads / 32;
constexpr int kGemvTableBytes = 128 * 1024;   // 4 groups x 256 entries x 32 slots x 4 B
constexpr int kGemvStageBytes = 16 * 80;      // activations of a half slice, behind its tables


// Up to kGemvMaxGroup weight matrices that share the activations (same K, bits, group) go through
// one launch: their output columns are concatenated, the tables are built once (paper Sec. 5:
// one table precomputation shared by the projections that read the same input).

struct GemvParams {
    const uint8_t  *packed[kGemvMaxGroup];
    const uint4    *planes[kGemvMaxGroup];   // one uint4 = one plane word of the four columns of a strip
    const uint2    *scales[kGemvMaxGroup];   // four fp16 scales of a strip and block
    const uint16_t *zeros[kGemvMaxGroup];    // four zero-point nibbles of a strip and block
    __half         *y[kGemvMaxGroup];        // first row of this launch
    int Ng[kGemvMaxGroup];                   // output columns of each matrix
    int unit0[kGemvMaxGroup];                // first warp-unit of each matrix
    int col0[kGemvMaxGroup];                 // first concatenated column of each matrix
    int count;                               // matrices in this launch
    const __half   *x;          // first row of this launch
    // integer path (per-tensor ternary weights, 16-bit integer activations): quantized activations,
    // their per-row scales, the tensor's weight scale, optional exact integer sums [M][N]
    const int16_t  *xi;
    const float    *row_scale;
    float           w_scale;
    int32_t        *acc_out;
    float          *partials;
    uint32_t       *status;
    int M;                      // rows in this launch (<= MT)
    int K, N, bits, group;      // N = total (concatenated) columns
    int nkappa;                 // K-slices
    int P;                      // CTAs per K-slice
    int units;                  // warp-units per K-slice
    int group_shift;            // log2(group)
    int nblk;                   // K / group
};

// Transposing reduction over the lanes selected by MASK, 2*MASK, ..., below END: every stage
// halves the number of values a lane keeps (or, once one is left, plainly adds).  `base` is the
// logical index of vals[0].
// INTS: the values are 32-bit integers kept in float registers (bit patterns) and are added as integers.
template <int N_, int MASK, int END, bool INTS = false>
struct LaneReduce {
    static __device__ __forceinline__ float add(float a, float b)
    {
        if constexpr (INTS) return __int_as_float(__float_as_int(a) + __float_as_int(b));
        else return a + b;
    }
    static __device__ __forceinline__ void run(float *vals, int v, int &base)
    {
        if constexpr (MASK < END) {
            if constexpr (N_ >= 2) {
                constexpr int H = N_ / 2;
                const bool up = (v & MASK) != 0;
#pragma unroll
                for (int j = 0; j < H; ++j) {
                    const float keep = up ? vals[j + H] : vals[j];
                    const float send = up ? vals[j] : vals[j + H];
                    vals[j] = add(keep, __shfl_xor_sync(0xffffffffu, send, MASK));
                }
                base += up ? H : 0;
                LaneReduce<H, MASK * 2, END, INTS>::run(vals, v, base);
            } else {
                vals[0] = add(vals[0], __shfl_xor_sync(0xffffffffu, vals[0], MASK));
                LaneReduce<1, MASK * 2, END, INTS>::run(vals, v, base);
            }
        }
    }
};

template <int MT> struct RowVec;
template <> struct RowVec<1> { using type = float; };
template <> struct RowVec<2> { using type = float2; };
template <> struct RowVec<4> { using type = float4; };

template <int MT>
__device__ __forceinline__ void load_rows(const uint8_t *p, float (&out)[MT])
{
    typename RowVec<MT>::type t = *reinterpret_cast<const typename RowVec<MT>::type *>(p);
    if constexpr (MT == 1) { out[0] = t; }
    else if constexpr (MT == 2) { out[0] = t.x; out[1] = t.y; }
    else { out[0] = t.x; out[1] = t.y; out[2] = t.z; out[3] = t.w; }
}

// byte offset of table entry (group c of the lane's word, index p, slot) inside the table area
__device__ __forceinline__ constexpr uint32_t table_imm(int c) { return (uint32_t)(c >> 1) * 65536u + (uint32_t)(c & 1) * 128u; }

// The tables start at the first byte of dynamic shared memory.  The kernel has no static shared
// memory, so that byte sits right after the per-CTA reserved region, at shared-window address
// kGemvSmemBase (the host checks cudaDevAttrReservedSharedMemoryPerBlock, the kernel checks its
// own base).  A lookup can then use the byte-permute result (index byte << 8 | slot offset) as
// the address register, with the table's offset folded into the instruction's immediate: no add
// per lookup.
constexpr uint32_t kGemvSmemBase = 1024;

template <int MT, uint32_t IMM>
__device__ __forceinline__ void lookup_rows(uint32_t off, float (&out)[MT])
{
    if constexpr (MT == 1) {
        asm volatile("ld.shared.f32 %0, [%1 + %2];" : "=f"(out[0]) : "r"(off), "n"(IMM));
    } else if constexpr (MT == 2) {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2 + %3];" : "=f"(out[0]), "=f"(out[1]) : "r"(off), "n"(IMM));
    } else {
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4 + %5];"
                     : "=f"(out[0]), "=f"(out[1]), "=f"(out[2]), "=f"(out[3]) : "r"(off), "n"(IMM));
    }
}

// The same lookup returning the raw 32-bit slots (two fp16 rows each).
template <int MT, uint32_t IMM>
__device__ __forceinline__ void lookup_slots(uint32_t off, uint32_t (&out)[MT])
{
    if constexpr (MT == 1) {
        asm volatile("ld.shared.b32 %0, [%1 + %2];" : "=r"(out[0]) : "r"(off), "n"(IMM));
    } else if constexpr (MT == 2) {
        asm volatile("ld.shared.v2.b32 {%0, %1}, [%2 + %3];" : "=r"(out[0]), "=r"(out[1]) : "r"(off), "n"(IMM));
    } else {
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4 + %5];"
                     : "=r"(out[0]), "=r"(out[1]), "=r"(out[2]), "=r"(out[3]) : "r"(off), "n"(IMM));
    }
}

// One unit's worth of a lane's inputs: its plane word of S strips, and the strips' scales and
// zero-points of the lane's quantization block.
template <int BITS, int S>
struct UnitRegs {
    uint4    w[S][BITS];
    uint2    sc[S];
    uint32_t z[S];
    int      g;        // matrix of the unit
    int      col;      // concatenated column of the lane's first strip
};

// BITS planes, MT rows per table entry, S strips per warp-unit and sub-warp, PRE = 1 when the
// lanes v and v^1 share a quantization block (group >= 64): they are added before scaling.
// HALF (MT = 1 only): K-slices of 16 plane words instead of 32, i.e. 64 KB of tables that cost
// half as much to build.  The two half-warps then work on different strips and read the same 64
// tables; entry rows hold all 64 slots (slot = word + 16 * index byte) and the second half-warp
// visits the index bytes of a word in the order 1,0,3,2, so that the 32 lanes still address 32
// different banks.
// GROUPED = 0: one matrix, the matrix index is a compile-time zero.
// HR (more than one activation row): a 32-bit table slot holds two rows as fp16 instead of one as fp32,
// so an entry of MT slots serves 2 * MT rows for the same shared-memory traffic.  Each row of the
// K-slice is first scaled by a power of two that brings its largest magnitude into [1, 2) (undone in
// fp32 at the end), so that entries use fp16's range whatever the activations' size; the bits * 4
// lookups of one plane word are accumulated in fp16 (low plane first), everything after that in fp32.
// INT (one row, HALF): per-tensor ternary weights (2-bit codes, zero-point 1, one scale) with 16-bit integer
// activations (paper Sec. 6.1: BitNet as W_INT2 A_INT16).  Tables hold exact integer sums (as fp32: a sum of
// eight 16-bit values is below 2^24), a word's lookups and the pair sum stay exact in fp32, and from there
// on the sums are 32-bit integers: the slice's lanes, the K-slices and the result are added as integers;
// only the final product with the row's and the tensor's scale is floating point (Sec. 4.3).
// One set of unit registers: every strip's registers are refilled with the next unit's strip as soon as its lookups are
// done (larger units, fewer per-unit fixed costs, same bytes in flight).
template <int BITS, int MT, int S, int PRE, int HALF, int GROUPED, int HR, int INT>
__global__ void __launch_bounds__(kGemvThreads, 1) mpgemv_kernel(const GemvParams p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    static_assert(!HALF || MT == 1, "half slices are for single-row tables");
    static_assert(!INT || (!HR && !GROUPED && BITS == 2), "the integer path is built for ternary weights, fp32-held integer tables");
    static_assert(!HR || !HALF, "fp16 row pairs use whole-warp or sub-warp slices");
    constexpr int R = HR ? 2 * MT : MT;    // activation rows of this launch
    constexpr int W = HALF ? 16 : 32 / MT; // plane words (lanes) per K-slice
    constexpr int SUBS = 32 / W;           // sub-warps, each on its own strips
    constexpr int V = 4 * S * R;          // values a lane produces per warp-unit
    constexpr int V1 = PRE ? V / 2 : V;   // values it still holds when scales are applied
    constexpr int NKEEP = (V >= W) ? V / W : 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kappa = blockIdx.y, j = blockIdx.x;
    const int words_total = p.K >> 5;
    const int word0 = kappa * W;
    const int nwords = min(W, words_total - word0);
    const int sub = lane / W, v = lane % W;
    const bool active = v < nwords;
    const int nblk = p.nblk;
    const int B = ((word0 + (active ? v : 0)) * 32) >> p.group_shift;

    // Let the next kernel in the stream start its own weight streaming while this one drains
    // (programmatic dependent launch); the header words are requested now and checked later.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool hdr_ok = true;
    {
        uint32_t hdr[kGemvMaxGroup][8];
#pragma unroll
        for (int g = 0; g < (GROUPED ? kGemvMaxGroup : 1); ++g)
            if (g < p.count) {
#pragma unroll
                for (int q = 0; q < 8; ++q) hdr[g][q] = __ldg(reinterpret_cast<const uint32_t *>(p.packed[g]) + q);
            }
#pragma unroll
        for (int g = 0; g < (GROUPED ? kGemvMaxGroup : 1); ++g)
            if (g < p.count)
                hdr_ok = hdr_ok && (hdr[g][0] == 0x4E414D54u) && (hdr[g][1] == 0x30303242u) && (hdr[g][2] == kVersion) &&
                         (hdr[g][3] == (uint32_t)p.K) && (hdr[g][4] == (uint32_t)p.Ng[g]) &&
                         (hdr[g][5] == (uint32_t)p.bits) && (hdr[g][6] == (uint32_t)p.group) && (hdr[g][7] == 4u);
    }

    // Loads are unconditional: a unit past the last one re-reads the last unit, a strip past the
    // last one re-reads the last strip, a lane past the end of a ragged last slice re-reads word 0
    // (its tables are all zero); none of those results is ever written.
    const uint32_t lane_word = (uint32_t)(word0 + (active ? v : 0));
    const uint32_t row_bytes = (uint32_t)words_total * 16u;      // one plane of one strip
    const uint32_t strip_bytes = row_bytes * BITS;
    struct UnitAddr { const uint8_t *pw; const uint2 *psc; const uint16_t *pz; int lu, nstrips; };
    auto unit_addr = [&](UnitRegs<BITS, S> &r, int wu) {
        const int u = min(wu, p.units - 1);
        int g = 0;
        if constexpr (GROUPED) {
#pragma unroll
            for (int t = 1; t < kGemvMaxGroup; ++t) g += (t < p.count && u >= p.unit0[t]) ? 1 : 0;
        }
        UnitAddr a;
        a.lu = GROUPED ? u - p.unit0[g] : u;
        a.nstrips = p.Ng[g] >> 2;
        a.pw = reinterpret_cast<const uint8_t *>(p.planes[g] + lane_word);
        a.psc = p.scales[g] + B;
        a.pz = p.zeros[g] + B;
        r.g = g;
        r.col = (GROUPED ? p.col0[g] : 0) + (a.lu * SUBS + sub) * S * 4;
        return a;
    };
    auto load_strip = [&](UnitRegs<BITS, S> &r, int s, const UnitAddr &a) {
        const uint32_t nb = (uint32_t)min((a.lu * SUBS + sub) * S + s, a.nstrips - 1);
        const uint8_t *q = a.pw + (size_t)nb * strip_bytes;
#pragma unroll
        for (int i = 0; i < BITS; ++i) {
            r.w[s][i] = __ldcs(reinterpret_cast<const uint4 *>(q));
            q += row_bytes;
        }
        if constexpr (INT) {
            r.sc[s] = make_uint2(0x3C003C00u, 0x3C003C00u);      // scale 1.0 four times (fp16), zero-point 1 four times
            r.z[s] = 0x1111u;
        } else {
            r.sc[s] = __ldg(a.psc + (size_t)nb * (uint32_t)nblk);
            r.z[s] = __ldg(a.pz + (size_t)nb * (uint32_t)nblk);
        }
    };
    auto load_unit = [&](UnitRegs<BITS, S> &r, int wu) {
        const UnitAddr a = unit_addr(r, wu);
#pragma unroll
        for (int s = 0; s < S; ++s) load_strip(r, s, a);
    };

    // Issue the first unit's weight loads before anything else: packed_bytes was checked on the
    // host, so these reads are in bounds whatever the header says, and no kernel that may still be
    // running writes the packed buffer (see the top of the file).  Their latency overlaps the table build.
    const int wu0 = j + p.P * warp, wstride = p.P * kGemvWarps;
    UnitRegs<BITS, S> regs;
    load_unit(regs, wu0);

    // The slice's activations, 64 bytes a word and row: one 16-byte piece a thread, passed on through shared memory (behind the tables,
    // or where they will be).  With every thread loading what its own table entries need instead: MLP of 4 x (4096 x 28672,
    // 14336 x 4096), 2-bit group 64, one row 79.7 us instead of 78.1, layer of 4608, 3-bit group 32, two rows 124.1 instead of 121.3.
    constexpr int PIECES = W * R * 4, STAGE_AT = HALF ? kGemvTableBytes / 2 : 0, STAGE_WORD = 80;     // (80: no bank conflicts)
    static_assert(!HALF || PIECES / 4 * STAGE_WORD == kGemvStageBytes, "room behind the tables");
    const int x_word = tid / 4 % W, x_row = tid / (4 * W);
    const bool x_live = tid < PIECES && x_word < nwords && x_row < p.M;
    const uint4 *const x_at = reinterpret_cast<const uint4 *>((INT ? reinterpret_cast<const uint16_t *>(p.xi) : reinterpret_cast<const uint16_t *>(p.x)) +
                                                              (size_t)x_row * p.K + (size_t)(word0 + x_word) * 32 + 8 * (tid & 3));

    // Everything below may depend on the previous kernel in the stream (activations, workspace).
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid < PIECES) {
        uint4 t = make_uint4(0u, 0u, 0u, 0u);
        if (x_live) t = ld_dependent(x_at);
        *reinterpret_cast<uint4 *>(smem + STAGE_AT + (tid >> 2) * STAGE_WORD + 16 * (tid & 3)) = t;
    }
    __syncthreads();

    if constexpr (HALF) {
        // thread (slot, chunk): slot = word + 16 * index byte of the table it fills, chunk = the
        // three high index bits of its 32 entries
        const int slot = tid & 63, chunk = tid >> 6;
        // index bit q of byte gc is word bit 8*gc + q, i.e. the weight 8*(q & 3) + 2*gc + (q >> 2)
        uint32_t pair[4];
#pragma unroll
        for (int ph = 0; ph < 4; ++ph)
            pair[ph] = *reinterpret_cast<const uint32_t *>(smem + STAGE_AT + (slot & 15) * STAGE_WORD + ph * 16 + (slot >> 4) * 4);
        float xv[8];
#pragma unroll
        for (int ph = 0; ph < 4; ++ph) {
            if constexpr (INT) {
                xv[ph] = (float)(int16_t)(pair[ph] & 0xFFFFu);
                xv[ph + 4] = (float)((int)pair[ph] >> 16);
            } else {
                const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&pair[ph]));
                xv[ph] = f.x;
                xv[ph + 4] = f.y;
            }
        }
        float lo[16];
        lut16(xv[0], xv[1], xv[2], xv[3], lo);
        float hi = 0.f;
        if (chunk & 1) hi += xv[5];
        if (chunk & 2) hi += xv[6];
        if (chunk & 4) hi += xv[7];
        uint8_t *dst = smem + (uint32_t)(chunk * 32) * 256u + (uint32_t)slot * 4u;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float base = q ? hi + xv[4] : hi;
#pragma unroll
            for (int e = 0; e < 16; ++e) *reinterpret_cast<float *>(dst + (q * 16 + e) * 256) = lo[e] + base;
        }
    } else if constexpr (HR) {
        // The activations of this thread's table slot: one plane word = 32 activations of rows 2*mb and 2*mb+1.
        const int vb = lane / MT, mb = lane % MT;
        uint4 xraw[2][4];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                xraw[r][c] = *reinterpret_cast<const uint4 *>(smem + STAGE_AT + ((2 * mb + r) * W + vb) * STAGE_WORD + 16 * c);
        __syncthreads();                                    // (the tables take its place)

        // largest magnitude of each row over the K-slice -> power-of-two scale (every warp computes the same)
        float inv[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            __half2 mx = __floats2half2_rn(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const __half2 *h = reinterpret_cast<const __half2 *>(&xraw[r][c]);
#pragma unroll
                for (int q = 0; q < 4; ++q) mx = __hmax2(mx, __habs2(h[q]));
            }
            float amax = fmaxf(__low2float(mx), __high2float(mx));
#pragma unroll
            for (int mask = MT; mask < 32; mask <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, mask));
            const uint32_t e = (__float_as_uint(amax) >> 23) & 0xFFu;      // amax = 1.f * 2^(e - 127)
            inv[r] = __uint_as_float((254u - e) << 23);
            if (warp == 0 && vb == 0)
                reinterpret_cast<float *>(smem + kGemvTableBytes)[2 * mb + r] = __uint_as_float(e << 23);
        }
        {
            // warp w fills, for index byte c = w % 4 of the word, the entries whose high index nibble is
            // 4 * (w / 4) .. 4 * (w / 4) + 3: the low-nibble sums of a byte are then computed once per warp
            const int c = warp & 3;
            float lo[2][16], xh[2][4];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                float xv[8];
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    // the c-th half2 of quarter qq: four-way select on the warp-uniform c
                    const uint4 q4 = xraw[r][qq];
                    const uint32_t u = c == 0 ? q4.x : c == 1 ? q4.y : c == 2 ? q4.z : q4.w;
                    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&u));
                    xv[qq] = f.x * inv[r];
                    xv[qq + 4] = f.y * inv[r];
                }
                lut16(xv[0], xv[1], xv[2], xv[3], lo[r]);
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) xh[r][qq] = xv[4 + qq];
            }
#pragma unroll
            for (int pq = 0; pq < 4; ++pq) {
                const int ph = 4 * (warp >> 2) + pq;
                float hi[2];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    hi[r] = 0.f;
                    if (ph & 1) hi[r] += xh[r][0];
                    if (ph & 2) hi[r] += xh[r][1];
                    if (ph & 4) hi[r] += xh[r][2];
                    if (ph & 8) hi[r] += xh[r][3];
                }
                uint8_t *dst = smem + table_imm(c) + (uint32_t)(ph * 16) * 256u + (uint32_t)lane * 4u;
#pragma unroll
                for (int pl = 0; pl < 16; ++pl)
                    *reinterpret_cast<__half2 *>(dst + pl * 256) = __floats2half2_rn(lo[0][pl] + hi[0], lo[1][pl] + hi[1]);
            }
        }
    } else {
        // The activations of this thread's table slot (one plane word = 32 activations of one row).
        const int vb = lane / MT, mb = lane % MT;
        uint4 xraw[4];                                      // 16-bit activations either way: fp16, or the integer path's quantized values
#pragma unroll
        for (int c = 0; c < 4; ++c) xraw[c] = *reinterpret_cast<const uint4 *>(smem + STAGE_AT + (mb * W + vb) * STAGE_WORD + 16 * c);
        __syncthreads();                                    // (the tables take its place)

        // ---- phase A: activation tables (paper Sec. 2.2; one table per 8 activations, 256 entries,
        // entry = 16-entry table of the low four + sum of the selected high four) -----------------
        {
            // warp w fills the entries whose high index nibble is w, for all four groups of the word
            const int ph = warp;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                // index bit q of byte c is word bit 8*c + q, i.e. the weight 8*(q & 3) + 2*c + (q >> 2):
                // the c-th pair of each quarter of the word
                float xv[8];
#pragma unroll
                for (int qq = 0; qq < 4; ++qq) {
                    if constexpr (INT) {
                        const short2 q2 = reinterpret_cast<const short2 *>(&xraw[qq])[c];
                        xv[qq] = (float)q2.x;
                        xv[qq + 4] = (float)q2.y;
                    } else {
                        const float2 f = __half22float2(reinterpret_cast<const __half2 *>(&xraw[qq])[c]);
                        xv[qq] = f.x;
                        xv[qq + 4] = f.y;
                    }
                }
                float lo[16];
                lut16(xv[0], xv[1], xv[2], xv[3], lo);
                float hi = 0.f;
                if (ph & 1) hi += xv[4];
                if (ph & 2) hi += xv[5];
                if (ph & 4) hi += xv[6];
                if (ph & 8) hi += xv[7];
                uint8_t *dst = smem + table_imm(c) + (uint32_t)(ph * 16) * 256u + (uint32_t)lane * 4u;
#pragma unroll
                for (int pl = 0; pl < 16; ++pl)
                    *reinterpret_cast<float *>(dst + pl * 256) = lo[pl] + hi;
            }
        }
    }
    __syncthreads();

    // header and layout check (uniform over the grid): a mismatch leaves every output untouched
    const bool base_ok = (uint32_t)__cvta_generic_to_shared(smem) == kGemvSmemBase;
    if (!hdr_ok || !base_ok) {
        if (tid == 0 && blockIdx.x == 0 && blockIdx.y == 0)
            atomicCAS(p.status, 0u, (uint32_t)(hdr_ok ? TMAN_ERR_LAYOUT : TMAN_ERR_BAD_PACKED));
        return;
    }

    // the activation sum of the lane's 32 activations (all-ones entries), for the zero-point term;
    // with PRE, of the two lanes that share the block
    const uint32_t sub_off = (uint32_t)(v * MT * 4);
    // HALF: slot offset inside a row = (v + 16 * byte) * 4; the byte visited at step jj is jj for
    // the first half-warp and jj ^ 1 for the second, so 64 * (jj & ~1) goes into the immediate and
    // the rest (0 or 64) into one of two registers
    const uint32_t off_even = (uint32_t)(v * 4 + 64 * sub), off_odd = (uint32_t)(v * 4 + 64 * (1 - sub));
    uint32_t sel_h[4];
#pragma unroll
    for (int jj = 0; jj < 4; ++jj) sel_h[jj] = 0x7604u | ((uint32_t)(jj ^ sub) << 4);
    float ssum[R];
    {
#pragma unroll
        for (int m = 0; m < R; ++m) ssum[m] = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if constexpr (HR) {
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const float2 f = __half22float2(
                        *reinterpret_cast<const __half2 *>(smem + table_imm(c) + 255u * 256u + sub_off + 4u * m));
                    ssum[2 * m] += f.x;
                    ssum[2 * m + 1] += f.y;
                }
            } else {
                float t[MT];
                if constexpr (HALF) load_rows<MT>(smem + 255u * 256u + (uint32_t)(v + 16 * c) * 4u, t);
                else load_rows<MT>(smem + table_imm(c) + 255u * 256u + sub_off, t);
#pragma unroll
                for (int m = 0; m < MT; ++m) ssum[m] += t[m];
            }
        }
        if constexpr (PRE) {
#pragma unroll
            for (int m = 0; m < R; ++m) ssum[m] += __shfl_xor_sync(0xffffffffu, ssum[m], 1);
        }
    }

    // ---- phase B: lookups, shift-accumulate, scale and zero-point (paper Sec. 4.3) --------------
    auto compute_unit = [&](UnitRegs<BITS, S> &r, int wu, int next_wu) {
        float vals[V];
        // what the end of the unit needs survives the refill of the strip registers
        uint2 sc_s[S];
        uint32_t z_s[S];
#pragma unroll
        for (int s = 0; s < S; ++s) { sc_s[s] = r.sc[s]; z_s[s] = r.z[s]; }
        const int g_u = r.g, col_u = r.col;
        const UnitAddr nxt = unit_addr(r, next_wu);
#pragma unroll
        for (int s = 0; s < S; ++s) {
#pragma unroll
            for (int c4 = 0; c4 < 4; ++c4) {
                float a[MT];
                __half2 a2[MT];
#pragma unroll
                for (int m = 0; m < MT; ++m) { a[m] = 0.f; a2[m] = __floats2half2_rn(0.f, 0.f); }
#pragma unroll
                for (int i = 0; i < BITS; ++i) {
                    const uint32_t w = (c4 == 0) ? r.w[s][i].x : (c4 == 1) ? r.w[s][i].y
                                     : (c4 == 2) ? r.w[s][i].z : r.w[s][i].w;
                    const __half2 pw = __floats2half2_rn((float)(1 << i), (float)(1 << i));
                    // byte 1 <- index byte c of the word, byte 0 <- the lane's slot offset
#define TMAN_LOOKUP(c)                                                                          \
    if constexpr (HR) {                                                                         \
        uint32_t t[MT];                                                                         \
        const uint32_t off = __byte_perm(w, sub_off, 0x7604u | ((uint32_t)(c) << 4));           \
        lookup_slots<MT, kGemvSmemBase + table_imm(c)>(off, t);                                 \
        _Pragma("unroll") for (int m = 0; m < MT; ++m)                                          \
            a2[m] = __hfma2(*reinterpret_cast<const __half2 *>(&t[m]), pw, a2[m]);              \
    } else {                                                                                    \
        float t[MT];                                                                            \
        if constexpr (HALF) {                                                                   \
            const uint32_t off = __byte_perm(w, ((c) & 1) ? off_odd : off_even, sel_h[c]);      \
            lookup_rows<MT, kGemvSmemBase + 64u * ((c) & ~1)>(off, t);                          \
        } else {                                                                                \
            const uint32_t off = __byte_perm(w, sub_off, 0x7604u | ((uint32_t)(c) << 4));       \
            lookup_rows<MT, kGemvSmemBase + table_imm(c)>(off, t);                              \
        }                                                                                       \
        _Pragma("unroll") for (int m = 0; m < MT; ++m) a[m] = fmaf(t[m], (float)(1 << i), a[m]); \
    }
                    TMAN_LOOKUP(0) TMAN_LOOKUP(1) TMAN_LOOKUP(2) TMAN_LOOKUP(3)
#undef TMAN_LOOKUP
                }
                if constexpr (HR) {
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        const float2 f = __half22float2(a2[m]);
                        vals[(s * 4 + c4) * R + 2 * m] = f.x;
                        vals[(s * 4 + c4) * R + 2 * m + 1] = f.y;
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < MT; ++m) vals[(s * 4 + c4) * MT + m] = a[m];
                }
            }
            load_strip(r, s, nxt);
        }

        // lanes v and v^1 hold the two words of one block: add them first, keeping half the columns
        int base = 0;
        LaneReduce<V, 1, PRE ? 2 : 1>::run(vals, v, base);
        const bool up = PRE && (v & 1);
        // scales and zero-points of the columns this lane still holds
        if constexpr (S >= 2 || !PRE) {
            constexpr int S1 = PRE ? S / 2 : S;
#pragma unroll
            for (int s = 0; s < S1; ++s) {
                const uint2 scq = up ? sc_s[s + (PRE ? S1 : 0)] : sc_s[s];
                const uint32_t zq = up ? z_s[s + (PRE ? S1 : 0)] : z_s[s];
                const __half2 s01 = *reinterpret_cast<const __half2 *>(&scq.x);
                const __half2 s23 = *reinterpret_cast<const __half2 *>(&scq.y);
                const float sc[4] = {__low2float(s01), __high2float(s01), __low2float(s23), __high2float(s23)};
#pragma unroll
                for (int c4 = 0; c4 < 4; ++c4) {
                    const float zf = (float)((zq >> (4 * c4)) & 0xFu);
#pragma unroll
                    for (int m = 0; m < R; ++m) {
                        float &val = vals[(s * 4 + c4) * R + m];
                        val = sc[c4] * fmaf(-zf, ssum[m], val);
                    }
                }
            }
        } else {
            // one strip, two of its four columns left
            const uint32_t scq = up ? sc_s[0].y : sc_s[0].x;
            const uint32_t zq = up ? (z_s[0] >> 8) : z_s[0];
            const __half2 s01 = *reinterpret_cast<const __half2 *>(&scq);
            const float sc[2] = {__low2float(s01), __high2float(s01)};
#pragma unroll
            for (int c2 = 0; c2 < 2; ++c2) {
                const float zf = (float)((zq >> (4 * c2)) & 0xFu);
#pragma unroll
                for (int m = 0; m < R; ++m) {
                    float &val = vals[c2 * R + m];
                    val = sc[c2] * fmaf(-zf, ssum[m], val);
                }
            }
        }
        // the other lanes of the K-slice (integer path: exact integers so far, added as integers from here on)
        if constexpr (INT) {
#pragma unroll
            for (int e = 0; e < V1; ++e) vals[e] = __int_as_float(__float2int_rn(vals[e]));
        }
        LaneReduce<V1, PRE ? 2 : 1, W, INT != 0>::run(vals, v, base);
        const bool writer = (V >= W) ? true : (v < V);
        if (writer && wu < p.units) {
            const int g = GROUPED ? g_u : 0;
            const int lim = GROUPED ? p.col0[g] + p.Ng[g] : p.N;   // end of this matrix's columns
#pragma unroll
            for (int e = 0; e < NKEEP; ++e) {
                const int idx = base + e, m = idx % R, n = col_u + idx / R;
                if (n < lim && m < p.M) {
                    float out = vals[e];
                    if constexpr (HR) out *= reinterpret_cast<const float *>(smem + kGemvTableBytes)[m];   // undo the row's scale
                    if (p.nkappa == 1) {
                        if constexpr (INT) {
                            const int acc = __float_as_int(out);
                            if (p.acc_out) p.acc_out[(size_t)m * p.N + n] = acc;
                            out = (float)acc * (ld_dependent(p.row_scale + m) * p.w_scale);
                        }
                        p.y[g][(size_t)m * p.Ng[g] + (n - (GROUPED ? p.col0[g] : 0))] = __float2half_rn(out);
                    } else {
                        p.partials[((size_t)kappa * R + m) * p.N + n] = out;     // integer path: the integer's bit pattern
                    }
                }
            }
        }
    };

    for (int wu = wu0; wu < p.units; wu += wstride) compute_unit(regs, wu, wu + wstride);

    // ---- combine K-slices: every CTA polls the partial sums of its share of the columns ----------
    if (p.nkappa > 1) {
        const int cta = blockIdx.y * gridDim.x + blockIdx.x, G = gridDim.x * gridDim.y;
        const int ng = p.N >> 2;
        const int g_lo = (int)(((long long)ng * cta) / G), g_hi = (int)(((long long)ng * (cta + 1)) / G);
        const int col_lo = g_lo * 4;
        const int ngrp = g_hi - g_lo;
        const int items = ngrp * p.M;                       // one item = four columns of one row
        const size_t stride4 = (size_t)R * p.N / 4;
        // SP adjacent lanes share an item and split the slices among them (slice kp goes to lane
        // kp % SP); their sums are added in a fixed order, so the result does not depend on timing
        int SP = 1;
        while (SP < 8 && 2 * SP <= p.nkappa && items * 2 * SP <= kGemvThreads) SP *= 2;
        const int part = tid & (SP - 1);
        const float sv = __uint_as_float(kGemvSentinel);
        using RED = LaneReduce<1, 1, 1, INT != 0>;          // its add(): floats, or integers kept in float registers
        bool gave_up = false;
        for (int item0 = 0; item0 < items; item0 += kGemvThreads / SP) {
            const int item = item0 + tid / SP;
            const bool alive = item < items;
            const int m = alive ? item / ngrp : 0, n = col_lo + 4 * (alive ? item % ngrp : 0);
            float4 *src = reinterpret_cast<float4 *>(p.partials + (size_t)m * p.N + n);
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);      // also the bit pattern of integer zero
            for (int kp = part; alive && kp < p.nkappa; kp += 4 * SP) {
                float4 t[4];
                if (!wait_for_sums(src, stride4, kp, SP, p.nkappa, kGemvPollLimit, t)) { gave_up = true; break; }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (kp + q * SP < p.nkappa) {
                        acc.x = RED::add(acc.x, t[q].x); acc.y = RED::add(acc.y, t[q].y);
                        acc.z = RED::add(acc.z, t[q].z); acc.w = RED::add(acc.w, t[q].w);
                        src[(size_t)(kp + q * SP) * stride4] = make_float4(sv, sv, sv, sv);
                    }
            }
            for (int mask = 1; mask < SP; mask <<= 1) {
                acc.x = RED::add(acc.x, __shfl_xor_sync(0xffffffffu, acc.x, mask));
                acc.y = RED::add(acc.y, __shfl_xor_sync(0xffffffffu, acc.y, mask));
                acc.z = RED::add(acc.z, __shfl_xor_sync(0xffffffffu, acc.z, mask));
                acc.w = RED::add(acc.w, __shfl_xor_sync(0xffffffffu, acc.w, mask));
            }
            gave_up = __any_sync(0xffffffffu, gave_up);
            if constexpr (INT) {
                if (alive && part == 0 && !gave_up) {
                    const int4 ia = make_int4(__float_as_int(acc.x), __float_as_int(acc.y), __float_as_int(acc.z), __float_as_int(acc.w));
                    if (p.acc_out) *reinterpret_cast<int4 *>(p.acc_out + (size_t)m * p.N + n) = ia;
                    const float sc = ld_dependent(p.row_scale + m) * p.w_scale;
                    acc = make_float4((float)ia.x * sc, (float)ia.y * sc, (float)ia.z * sc, (float)ia.w * sc);
                }
            }
            if (alive && part == 0 && !gave_up) {
                const __half2 h01 = __floats2half2_rn(acc.x, acc.y), h23 = __floats2half2_rn(acc.z, acc.w);
                uint2 o;
                o.x = *reinterpret_cast<const uint32_t *>(&h01);
                o.y = *reinterpret_cast<const uint32_t *>(&h23);
                int g = 0;
                if constexpr (GROUPED) {
#pragma unroll
                    for (int t = 1; t < kGemvMaxGroup; ++t) g += (t < p.count && n >= p.col0[t]) ? 1 : 0;
                }
                *reinterpret_cast<uint2 *>(p.y[g] + (size_t)m * p.Ng[g] + (n - p.col0[g])) = o;
            }
        }
        if (gave_up) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_TIMEOUT);
    }
}

template <int BITS, int MT, int S, int PRE, int HALF, int GROUPED, int HR, int INT = 0>
static tman_status launch_one(GemvParams p, int sms, cudaStream_t s)
{
    constexpr int W = HALF ? 16 : 32 / MT;
    constexpr int SUBS = 32 / W;
    // fp16 row pairs: the rows' scales follow the tables
    constexpr int kSmem = HALF ? kGemvTableBytes / 2 + kGemvStageBytes : kGemvTableBytes + (HR ? 64 : 0);
    const int words_total = p.K / 32;
    p.nkappa = (words_total + W - 1) / W;
    p.P = sms / p.nkappa;
    if (p.P < 1) p.P = 1;
    p.units = 0;
    for (int g = 0; g < p.count; ++g) {
        p.unit0[g] = p.units;
        p.units += (p.Ng[g] / 4 + S * SUBS - 1) / (S * SUBS);
    }
    for (int g = p.count; g < kGemvMaxGroup; ++g) p.unit0[g] = p.units;
    // Units of one strip: about half of a CTA's warps get one.  With all of them at work (fewer CTAs) and with one each (as many
    // CTAs as units) 4-bit 4096 x 1024 takes 3.84 and 3.64 us instead of 3.59, two rows 4.70 and 5.33 instead of 5.23.
    if (S == 1 && !INT && p.P * kGemvWarps > 2 * p.units) p.P = (2 * p.units + kGemvWarps - 1) / kGemvWarps;
    if (p.P > p.units) p.P = p.units;
    // every CTA must be resident while it polls for the others' partial sums
    if ((long long)p.nkappa * p.P > (long long)sms) return TMAN_ERR_UNSUPPORTED;
    int dev = 0;
    const DeviceInfo *info = device_info(&dev);
    if (!info) return TMAN_ERR_CUDA;
    if ((uint32_t)info->reserved_smem.load(std::memory_order_relaxed) != kGemvSmemBase) return TMAN_ERR_UNSUPPORTED;
    auto kern = mpgemv_kernel<BITS, MT, S, PRE, HALF, GROUPED, HR, INT>;
    static std::atomic<bool> raised[kMaxDevices];
    // the grid has at most one CTA per SM; the occupancy query says whether an SM can hold one at all
    // (asked once per device and variant)
    {
        static std::atomic<int> fits[kMaxDevices];          // 0 = not asked, 1 = fits, -1 = does not
        int f = fits[dev].load(std::memory_order_relaxed);
        if (f == 0) {
            int per_sm = 0;
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem) != cudaSuccess ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGemvThreads, kSmem) != cudaSuccess)
                return TMAN_ERR_CUDA;
            // they alternate with decode_digits_kernel in a layer (two rows of group 32 do not, and lose 4 % by it)
            if constexpr (INT || (MT == 1 && (PRE || !HR))) prefer_common_split(kern);
            f = per_sm >= 1 ? 1 : -1;
            fits[dev].store(f, std::memory_order_relaxed);
        }
        if (f < 0) return TMAN_ERR_UNSUPPORTED;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.P, (unsigned)p.nkappa);
    cfg.blockDim = dim3(kGemvThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    // The kernel reads weights before it waits for its predecessor, so the call that follows a weight
    // packing on this stream keeps plain stream order.
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = packed_write_pending(s, /*clear=*/true) ? 0 : 1;
    return launch_with_smem(kern, kSmem, dev, raised, [&] { return cudaLaunchKernelEx(&cfg, kern, p); });
}

template <int BITS, int MT, int PRE, int HR>
static tman_status launch_mt(GemvParams p, int sms, cudaStream_t s)
{
    // one row: fp32 tables over half-warp slices, large units; more rows: fp16 row pairs, smaller units
    // (measured: 2 strips per unit)
    constexpr int S = (HR && MT == 2) ? 2 : ((BITS == 2) ? 4 : 2);
    constexpr int HALF = HR ? 0 : 1;
    if (p.count > 1) return launch_one<BITS, MT, S, PRE, HALF, 1, HR>(p, sms, s);
    // One matrix of so few columns that a strip per sub-warp is enough: units of one strip, and fewer CTAs (launch_one).
    // In a graph, 4-bit 4096 x 1024: 3.86 -> 3.59 us (one row), 5.42 -> 5.23 (two), 2-bit 4096 x 512: 3.85 -> 3.12, 5.34 -> 4.16; near the
    // line (4096 x 2048) 4.19 -> 4.09 and 5.77 -> 5.74, above it the larger units are as fast or faster.
    constexpr int W = HALF ? 16 : 32 / MT;
    const int ctas = sms / ((p.K / 32 + W - 1) / W);
    if (p.N / 4 <= ctas * kGemvWarps * (32 / W)) return launch_one<BITS, MT, 1, PRE, HALF, 0, HR>(p, sms, s);
    return launch_one<BITS, MT, S, PRE, HALF, 0, HR>(p, sms, s);
}

// ---- the plan: which kernel variants serve a call (host arithmetic only) -------------------------
// A variant carries up to `rows` activation rows per pass over the weights in K-slices of `words` plane
// words; its table entries have `slots` 32-bit slots (one fp32 row, or two fp16 rows each; 0: no tables, the tensor-core
// kernel).  The time of a pass is modelled as fixed + per_mb x megabytes of bit planes; the constants were fitted to calls
// timed in a CUDA graph on a B200 (4-bit, group 128, 4096 x 4096 and 4096 x 28672; one row also 2-bit 4096 x 14336; the last
// two lines before the tensor-core kernel took two chunks of k per warp: 4096 x 28672 is modelled 20.5 and 23.1 us and takes 18.9
// and 20.6.  They only weigh one pass of more rows against several of fewer, which this does not change).
struct GemvVariant { int rows, words, slots, half_slices; double fixed_us, us_per_mb; };
static const GemvVariant kGemvVariants[kGemvVariantCount] = {
    {1, 16, 1, 1, 4.10, 0.190},
    {2, 32, 1, 0, 4.35, 0.216},
    {4, 16, 2, 0, 4.54, 0.272},
    {8, 8, 0, 0, 4.60, 0.316},
};

// Whether a pass of `rows` rows goes to the tensor-core kernel (decode_mma.cuh) instead of the table lookups.  From five
// rows always: an entry of eight fp16 rows costs four shared-memory wavefronts a lookup (4-bit 4096 x 28672, group 128:
// 42.0 us by lookup, 20.6 us here; 3-bit, group 64: 21.6; 2-bit: 19.3).  With three and four rows
// (two wavefronts) where the blocks are no shorter than two words: 4-bit, group 128
// 23.8 / 18.9, 3-bit, group 64 20.2 / 18.9 (4096 x 4096: 7.4 / 5.6), 2-bit, group 128 17.3 / 16.9 (6.8 / 5.5); but 4-bit, group 32
// 24.0 / 31.2.  2-bit, group 64 (few planes to look up, halves of a chunk to multiply) as far as a call is short: 4096 x 6144 8.4 / 7.0,
// 14336 x 4096 11.3 / 11.5, 4096 x 28672 17.3 / 18.2.  Where K fills the teams of warps badly the lookups would be faster here and
// there (three rows, 18944 x 3584: 2-bit, group 128 12.0 / 13.3, 3-bit, group 64 14.1 / 15.0; 2-bit, group 64, 11008 x 4096 9.6 / 10.5); such
// calls stay on the tensor cores, whose sums are fp32 throughout: the lookups' fp16 ones are three times further from the exact product.
// One and two rows are cheaper by lookup (4-bit, group 128, two rows: 17.2 / 18.4).
// (Lookup times from before activations came by ordinary loads; they take 0.5 to 1 us a call more now.  Over 450 drawn layers, MLPs and calls
// every class of three and four rows in groups of 64 and 128 is still faster here in the mean, by 0.5 to 3 us a call, two rows are not, by up
// to 1.7, nor groups of 32 above about 10 million weights.)
static bool uses_mma(int bits, int group, int rows, long long weights)
{
    return rows >= 5 || (rows >= 3 && group >= 64 && (bits >= 3 || group == 128 || weights <= 48000000ll));
}

static size_t variant_ws_bytes(const GemvVariant &v, int K, int N)
{
    // one fp32 partial sum per K-slice, row of the variant and column
    const size_t nkappa = (size_t)(K / 32 + v.words - 1) / (size_t)v.words;
    return kWsStatusBytes + nkappa * (size_t)v.rows * (size_t)N * sizeof(float);
}

// Limits a variant must meet on this device and call: its K-slices times at least one CTA each must be
// resident together (the CTAs poll one another's partial sums), its tables must fit the shared memory of
// an SM, and its partial sums must fit the caller's workspace.
static bool variant_feasible(const GemvVariant &v, int K, int N, int sms, size_t ws_limit)
{
    const int nkappa = (K / 32 + v.words - 1) / v.words;
    const int smem = (v.half_slices ? kGemvTableBytes / 2 : kGemvTableBytes) + 64;
    return nkappa <= sms && smem <= kGemvSmemLimit && variant_ws_bytes(v, K, N) <= ws_limit;
}

// How the tensor-core kernel cuts a pass: warps of a team (each one 128-deep chunk of k), teams per CTA, K-slices, CTAs per
// K-slice.  16 warps of a team give the fewest partial sums; 8 and 4 are for short K or few columns, where more CTAs get work.
struct MmaSplit { int tk, tc, nkappa, ctas, cpw; };
static MmaSplit split_mma(int M, int K, int N, int groups, int sms, size_t ws_limit)
{
    const int chunks = K / 128;
    MmaSplit best = {0, 0, 0, 0, 0};
    double best_us = 1e300;
    for (int way = 0; way < 4; ++way) {                     // 16 warps with two chunks each, then 16, 8, 4 with one
        const int cpw = way == 0 ? 2 : 1, tk = way == 0 ? 16 : 32 >> way;
        const int parts = (chunks + tk * cpw - 1) / (tk * cpw);
        if (parts > sms) continue;                          // every CTA must be resident while it polls
        if (parts > 1 && kWsStatusBytes + (size_t)parts * M * N * sizeof(float) > ws_limit) continue;
        int tc = 16 / tk, ctas = sms / parts;
        while (tc > 1 && (groups + tc - 1) / tc < ctas) tc >>= 1;
        if (ctas > (groups + tc - 1) / tc) ctas = (groups + tc - 1) / tc;
        const int steps = (groups + ctas * tc - 1) / (ctas * tc) * cpw;
        // a step costs half its time in latency however many warps take part, a tenth more with two chunks a warp (activations
        // from shared memory, a longer start); the partial sums are written, waited for and read back.  Two chunks against one,
        // in a graph, 4-bit group 128: 4096 x 4096 5.6 / 6.5 us (four rows), 6.5 / 6.9 (eight), 4096 x 28672 19.5 / 18.9 and 20.6 / 21.3;
        // 3-bit group 64, eight rows 21.6 / 24.3; 14336 x 4096, four rows 14.5 / 11.9.
        const double us = steps * 0.5 * (tk * tc / 16.0 + 1) * (cpw == 2 ? 1.1 : 1.0) + (cpw == 2 ? 0.25 : 0.0) + (parts > 1 ? 1.6 : 0.0) +
                          (double)parts * M * N * 8e-6 / 3.0 * (parts > 1);
        if (us < best_us) { best_us = us; best = {tk, tc, parts, ctas, cpw}; }
    }
    return best;
}

// ---- decode on the integer tensor cores (decode_digits.cuh) ----------------------------------------------------------
// How a launch is laid out: CTAs (two an SM: `two`), warps of a team, units of the warps' rings, turns between reductions (0: it does not
// fit); groups of a CTA, and units that the busiest warp takes (`steps`), which say how well the columns and K fill it.
struct DigitSplit { int ctas, tk_shift, depth, flush, smem, scale_row, zero_row, groups, steps; bool two; };
static DigitSplit split_digits(int rows, int K, int strips, int bits, int group, int nb, bool ints, int sms)
{
    DigitSplit d = {};
    const int pairs = (K / 128 + 1) / 2, nblk = K / group;
    const int slot = rows * (512 + nb * 16), turn = kDigitWarps * rows * 128;    // a chunk's activations; the warps' sums of a turn
    const int fixed = kDigitGroups * (int)sizeof(DigitGroup) + (nb > 1 ? rows * 512 : 0), ring = kDigitWarps * 2 * bits * 512;
    d.scale_row = ints ? 0 : (nblk * 8 + 127) / 128 * 128 + (nb == 4 ? 32 : 16);
    d.zero_row = ints ? 0 : (nblk * 2 + 4 + 127) / 128 * 128 + 4;
    // One CTA an SM, in half its shared memory so that the next call's can start beside it, or two of this call where there are five
    // groups each (4-bit 4096 x 28672: 14.8 us with one, 13.5 with two); else one with all of it.
    const bool two = strips >= 40 * sms;
    const int at_most = two ? 2 * sms : sms;
    d.ctas = strips < at_most ? strips : at_most;
    const int share = (strips + d.ctas - 1) / d.ctas, groups = (share + 7) / 8;
    d.two = two;
    d.groups = groups;
    const int rest = fixed + 2 * pairs * slot + share * (d.scale_row + d.zero_row) + 16;
    int room = kDigitSmemHalf;
    d.depth = rest + 2 * ring + turn <= room ? 2 : 1;
    if (rest + ring + turn > room) {
        room = kDigitSmem;
        d.depth = rest + 2 * ring + turn <= room ? 2 : 1;
    }
    // (on 148 SMs no call that comes here has one row of 4 bits in short groups with room for two units, or 2 bits in groups of 32 without)
    if (bits == 4 && nb > 1 && rows == 1) d.depth = 1;
    if (bits == 2 && nb == 4 && d.depth == 1) return d;
    const int base = rest + d.depth * ring;
    if (groups > kDigitGroups - kGemvMaxGroup || base + turn > room || (two && room > kDigitSmemHalf)) return d;
    d.tk_shift = kDigitWarpsShift;
    d.steps = 1 << 30;
    for (int shift = kDigitWarpsShift; shift >= 0; --shift) {
        const int tc = kDigitWarps >> shift, steps = (groups + tc - 1) / tc * ((pairs + (1 << shift) - 1) >> shift);
        if (steps < d.steps) { d.steps = steps; d.tk_shift = shift; }
    }
    const int tc = kDigitWarps >> d.tk_shift, turns = (groups + kGemvMaxGroup + tc - 1) / tc;
    d.flush = (room - base) / turn;
    if (d.flush > turns) d.flush = turns;
    d.smem = base + d.flush * turn;
    return d;
}

// Whether a pass of `rows` rows goes to the integer tensor cores instead of the table lookups (columns: of all matrices).  The difference
// of the two times is modelled from what a launch consists of, in us: preparing all activations in every CTA (by K), the units
// that the busiest warp takes (also where K does not fill the warps: 2176 takes as many as 4096) and the tiles of B that each is
// multiplied with, groups, and megabytes of planes, which cost the lookups more.  Constants: least squares over graphs of layers,
// MLPs and single calls with every call by either kernel, for 3600 draws of K = 1024..5120 and 256..40000 columns and for layers
// of nine common shapes, plus half a change of kernel between neighbours (0.4 us) and 0.2 us of margin.  On 400 further draws
// one row takes 0.979 of its time by lookup in the mean (a layer or MLP in 40 more than 2 % longer, at most 9 %).  Two rows go by it only
// beyond the lines within which they come here in any case, because the lookups' fp16 sums are three times further from the exact product
// (6.5e-4 of it against 2.1e-4): 0.905 in the mean, one layer or MLP in 30 more than 2 % longer (1920 x 9728 and back, 2-bit group 64 12 %).
// Examples, by lookup / by this rule, 4-bit group 128: layer of 4096 x (6144, 4096, 28672) and 14336 x 4096, one row 40.7 / 36.2 us,
// of 2048 x (3072, 2048, 16384) and 8192 x 2048 22.3 / 21.0, two rows 27.7 / 24.9.
// Lines outside the model: six and more units a warp in one CTA an SM (3584 x 22784 and back, 4-bit 22.6 / 28.3), few columns
// (4096 x 512 3.3 / 4.8), two rows in groups of 32 (four tiles).  Calls of one group a CTA and at most two units, 2 and 4 bits
// (4096 x 4096), gain more than the linear model says, 0.2 to 1.3 us.
struct DigitPrice { float base, k, unit, tile, group, mb, two; };
static const DigitPrice kDigitPrices[2][3] = {
    {{-1.44f, 0.23f, 0.28f, 0.14f, 0.33f, -0.09f, -0.46f}, {-1.52f, 0.39f, 0.34f, 0.03f, 0.52f, -0.12f, -0.44f},
     {-1.59f, 0.46f, 0.21f, 0.04f, 0.55f, -0.12f, -0.24f}},
    {{-2.23f, 0.36f, 0.11f, 0.22f, 0.48f, -0.12f, 0.70f}, {-1.67f, 0.31f, 0.03f, 0.18f, 0.30f, -0.02f, 0.18f},
     {-1.58f, 0.31f, -0.03f, 0.24f, 0.06f, -0.03f, 0.f}},
};
static bool uses_digits(int bits, int group, int rows, int K, long long columns, int sms)
{
    if (rows > 2 || K > 5120 || columns > 40960 || columns * rows < K / 2 || (group == 32 && rows == 2)) return false;
    const DigitSplit d = split_digits(rows, K, (int)(columns / 4), bits, group, 128 / group, false, sms);
    if (d.flush < 1) return false;
    const bool badly_filled = K > 2048 && columns >= 96ll * sms && columns < 160ll * sms;
    if (rows == 2 && columns <= (group == 128 ? 10 * K : K > 2048 ? 5120 : 8192) && !badly_filled) return true;
    if (d.steps >= 6 && !d.two) return false;
    const int tiles = group == 128 ? 1 : group == 64 ? rows : 2;
    if (rows == 1 && tiles == 1 && bits != 3 && d.groups == 1 && d.steps <= 2 && d.ctas == sms) return true;
    const DigitPrice &c = kDigitPrices[rows - 1][bits - 2];
    const float us = c.base + c.k * (float)K / 1024.f + (c.unit + c.tile * (float)(tiles - 1)) * (float)d.steps + c.group * (float)d.groups +
                     c.mb * (float)((double)K * (double)columns * bits / 8e6) + (d.two ? c.two : 0.f);
    return us < (tiles > 1 ? -0.3f : 0.f);
}

// The same for the integer path, whose product follows a row quantization (sums are exact either way): products 2560 x 6912 and back in
// turn, each with its quantization, two rows 13.8 by lookup / 13.6 us, six 28.9 / 23.1, eight (which the lookups take in two passes)
// 32.0 / 27.0.  One row as far as the busiest warp has three units at most: of 250 drawn pairs of products none loses more than 1 %, 0.912 of the
// time by lookup in the mean; with four units 10 % of them lose up to 7 % (3584 x 5504 and back 12.1 / 13.0).
static bool uses_digits_ternary(int rows, int K, int N, int group, int sms)
{
    if (K > 5120 || (long long)N * rows < K / 2) return false;
    const DigitSplit d = split_digits(rows, K, N / 4, 2, group, 1, true, sms);
    return d.flush > 0 && (rows >= 2 || d.steps <= 3);
}

GemvPlan plan_gemv(int M, int K, int N, int bits, int group, int sms, size_t ws_limit)
{
    // best[m]: least modelled time for m rows; a pass with variant v takes min(rows_v, m) of them
    const double plane_mb = (double)K * (double)N * bits / 8.0 / 1e6;
    double best[kGemvMaxRows + 1];
    int pick[kGemvMaxRows + 1];
    for (int m = 0; m <= kGemvMaxRows; ++m) { best[m] = 1e300; pick[m] = -1; }
    best[0] = 0.0;
    for (int m = 1; m <= M && m <= kGemvMaxRows; ++m) {
        best[m] = 1e300;
        pick[m] = -1;
        for (int vi = 0; vi < kGemvVariantCount; ++vi) {
            const GemvVariant &v = kGemvVariants[vi];
            if (!variant_feasible(v, K, N, sms, ws_limit)) continue;
            const int take = v.rows < m ? v.rows : m;
            if (take < v.rows && vi > 0 && kGemvVariants[vi - 1].rows >= take &&
                variant_feasible(kGemvVariants[vi - 1], K, N, sms, ws_limit))
                continue;                                   // a narrower variant carries these rows as well
            const double c = v.fixed_us + v.us_per_mb * plane_mb + best[m - take];
            if (c < best[m] - 1e-9) { best[m] = c; pick[m] = vi; }
        }
        if (pick[m] < 0) break;
    }
    GemvPlan g = {};
    if (M < 1 || M > kGemvMaxRows || pick[M] < 0) return g;      // npass == 0: no feasible plan
    g.cost_us = best[M];
    // widest passes first
    int left = M;
    while (left > 0) {
        const int vi = pick[left];
        const GemvVariant &v = kGemvVariants[vi];
        const int take = v.rows < left ? v.rows : left;
        GemvPass &ps = g.pass[g.npass++];
        ps.variant = vi;
        ps.rows = take;
        ps.variant_rows = v.rows;
        ps.words = v.words;
        ps.nkappa = (K / 32 + v.words - 1) / v.words;
        ps.ctas_per_slice = sms / ps.nkappa;
        ps.smem_bytes = v.half_slices ? kGemvTableBytes / 2 + kGemvStageBytes : kGemvTableBytes + 64;
        const size_t need = variant_ws_bytes(v, K, N);
        ps.digits = uses_digits(bits, group, take, K, N, sms);
        ps.mma = !ps.digits && uses_mma(bits, group, take, (long long)K * N);
        if (ps.digits) {
            const DigitSplit sp = split_digits(take, K, N / 4, bits, group, 128 / group, false, sms);
            ps.words = K / 32;
            ps.nkappa = 1;
            ps.ctas_per_slice = sp.ctas;
            ps.smem_bytes = sp.smem;
        }
        if (ps.mma) {
            const MmaSplit sp = split_mma(take, K, N, (N + 31) / 32, sms, need);
            ps.words = 4 * sp.tk * sp.cpw;
            ps.nkappa = sp.nkappa;
            ps.ctas_per_slice = sp.ctas;
            ps.smem_bytes = MmaCfg<4, 4, 2, 2>::SMEM;             // at most
        }
        if (need > g.ws_bytes) g.ws_bytes = need;
        left -= take;
    }
    return g;
}

template <int BITS, int R, int NB, int NE, int CPW>
static tman_status launch_mma_split(MmaParams p, const MmaSplit &sp, cudaStream_t s)
{
    p.chunks = p.K / 128;
    p.tk = sp.tk; p.tc = sp.tc; p.nkappa = sp.nkappa;
    constexpr int smem = MmaCfg<BITS, R, NE, CPW>::SMEM;
    auto kern = decode_mma_kernel<BITS, R, NB, NE, CPW>;
    static std::atomic<bool> raised[kMaxDevices];
    int dev = 0;
    if (!device_info(&dev)) return TMAN_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)sp.ctas, (unsigned)sp.nkappa);
    cfg.blockDim = dim3((unsigned)(32 * sp.tk * sp.tc));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = packed_write_pending(s, /*clear=*/true) ? 0 : 1;      // as in launch_one
    return launch_with_smem(kern, smem, dev, raised, [&] { return cudaLaunchKernelEx(&cfg, kern, p); });
}

template <int BITS, int R, int NB, int NE>
static tman_status launch_mma(const MmaParams &p, int sms, size_t ws_limit, cudaStream_t s)
{
    const MmaSplit sp = split_mma(p.M, p.K, p.N, p.groups, sms, ws_limit);
    if (!sp.ctas) return TMAN_ERR_UNSUPPORTED;
    return sp.cpw == 2 ? launch_mma_split<BITS, R, NB, NE, 2>(p, sp, s) : launch_mma_split<BITS, R, NB, NE, 1>(p, sp, s);
}

template <int BITS>
static tman_status launch_mma_rows(const GemvParams &g, int rows, int sms, size_t ws, cudaStream_t s)
{
    MmaParams p = {};
    p.count = g.count;
    for (int i = 0; i < kGemvMaxGroup; ++i) {
        p.packed[i] = g.packed[i];
        p.planes[i] = reinterpret_cast<const uint8_t *>(g.planes[i]);
        p.scales[i] = g.scales[i];
        p.zeros[i] = g.zeros[i];
        p.y[i] = g.y[i];
        p.Ng[i] = g.Ng[i];
        p.col0[i] = g.col0[i];
        p.grp0[i] = p.groups;
        if (i < g.count) p.groups += (g.Ng[i] + 31) / 32;
    }
    p.x = g.x;
    p.partials = g.partials; p.status = g.status;
    p.M = rows; p.K = g.K; p.N = g.N;
    p.bits = g.bits; p.group = g.group; p.group_shift = g.group_shift; p.nblk = g.nblk;
    // the columns of B hold the blocks of a chunk as long as there are enough of them for the rows
    if (p.group >= 64 && rows <= 4) return p.group == 128 ? launch_mma<BITS, 1, 1, 1>(p, sms, ws, s) : launch_mma<BITS, 1, 2, 2>(p, sms, ws, s);
    if (p.group == 128) return launch_mma<BITS, 1, 1, 2>(p, sms, ws, s);
    return p.group == 64 ? launch_mma<BITS, 2, 1, 2>(p, sms, ws, s) : launch_mma<BITS, 4, 1, 2>(p, sms, ws, s);
}

template <int BITS, int NB, int NT, int DEPTH, bool INT>
static tman_status launch_digits_split(DigitParams p, const DigitSplit &d, cudaStream_t s)
{
    p.chunks = p.K / 128;
    p.strips_q = p.strip0[kGemvMaxGroup] / d.ctas; p.strips_r = p.strip0[kGemvMaxGroup] % d.ctas;
    p.pairs = (p.chunks + 1) / 2;
    p.pairs_q = p.pairs >> d.tk_shift; p.pairs_r = p.pairs & ((1 << d.tk_shift) - 1);
    p.scale_row = d.scale_row; p.zero_row = d.zero_row;
    p.tk_shift = d.tk_shift; p.tc = kDigitWarps >> d.tk_shift; p.flush = d.flush;
    p.by_rows = (0x80000000u + (uint32_t)p.M - 1u) / (uint32_t)p.M;
    auto kern = decode_digits_kernel<BITS, NB, NT, DEPTH, INT>;
    static std::atomic<bool> raised[kMaxDevices];
    int dev = 0;
    if (!device_info(&dev)) return TMAN_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)d.ctas);
    cfg.blockDim = dim3(32 * kDigitWarps);
    cfg.dynamicSmemBytes = (size_t)d.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = packed_write_pending(s, /*clear=*/true) ? 0 : 1;      // as in launch_one
    if (!raised[dev].load(std::memory_order_relaxed)) prefer_common_split(kern);
    return launch_with_smem(kern, kDigitSmem, dev, raised, [&] { return cudaLaunchKernelEx(&cfg, kern, p); });
}

template <int BITS, int NB, int NT, bool INT>
static tman_status launch_digits(const DigitParams &p, int sms, cudaStream_t s)
{
    const DigitSplit d = split_digits(p.M, p.K, p.strip0[kGemvMaxGroup], BITS, p.group, NB, INT, sms);
    if (d.flush < 1) return TMAN_ERR_UNSUPPORTED;
    if constexpr (BITS == 4 && NB > 1 && NT == NB / 2) return launch_digits_split<BITS, NB, NT, 1, INT>(p, d, s);     // (split_digits)
    else if constexpr (BITS == 2 && NB == 4) return launch_digits_split<BITS, NB, NT, 2, INT>(p, d, s);
    else return d.depth == 2 ? launch_digits_split<BITS, NB, NT, 2, INT>(p, d, s) : launch_digits_split<BITS, NB, NT, 1, INT>(p, d, s);
}

template <int BITS>
static tman_status launch_digit_tiles(const DigitParams &p, int sms, cudaStream_t s)
{
    if (p.group == 128) return launch_digits<BITS, 1, 1, false>(p, sms, s);
    if (p.group == 64) return p.M == 1 ? launch_digits<BITS, 2, 1, false>(p, sms, s) : launch_digits<BITS, 2, 2, false>(p, sms, s);
    return launch_digits<BITS, 4, 2, false>(p, sms, s);
}

template <int BITS>
static tman_status launch_digit_rows(const GemvParams &g, int sms, cudaStream_t s)
{
    DigitParams p = {};
    p.count = g.count;
    for (int i = 0; i < kGemvMaxGroup; ++i) {
        p.packed[i] = g.packed[i];
        p.planes[i] = reinterpret_cast<const uint8_t *>(g.planes[i]);
        p.scales[i] = reinterpret_cast<const uint8_t *>(g.scales[i]);
        p.zeros[i] = reinterpret_cast<const uint8_t *>(g.zeros[i]);
        p.y[i] = g.y[i];
        p.Ng[i] = g.Ng[i];
        p.strip0[i + 1] = p.strip0[i] + (i < g.count ? g.Ng[i] / 4 : 0);
    }
    p.x = g.x;
    p.status = g.status;
    p.M = g.M; p.K = g.K; p.bits = g.bits; p.group = g.group; p.nblk = g.nblk;
    return launch_digit_tiles<BITS>(p, sms, s);
}

template <int BITS>
static tman_status launch_rows(GemvParams p, const GemvPass &ps, int sms, cudaStream_t s)
{
    p.M = ps.rows;
    if (ps.digits) return launch_digit_rows<BITS>(p, sms, s);
    const bool pre = p.group >= 64;
    if (ps.mma) return launch_mma_rows<BITS>(p, ps.rows, sms, variant_ws_bytes(kGemvVariants[ps.variant], p.K, p.N), s);
    if (ps.variant == 0) return pre ? launch_mt<BITS, 1, 1, 0>(p, sms, s) : launch_mt<BITS, 1, 0, 0>(p, sms, s);
    if (ps.variant == 1) return pre ? launch_mt<BITS, 1, 1, 1>(p, sms, s) : launch_mt<BITS, 1, 0, 1>(p, sms, s);
    return pre ? launch_mt<BITS, 2, 1, 1>(p, sms, s) : launch_mt<BITS, 2, 0, 1>(p, sms, s);
}

__global__ void ws_fill_kernel(uint32_t *ws, size_t words)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < words) ws[i] = (i < kWsStatusBytes / 4) ? 0u : kGemvSentinel;
}

// One CTA waits, with the combine's own bounded wait, for partial sums that nothing will ever write (the
// workspace holds "no sum pending" after tman_workspace_init), gives up after `limit` polls and reports
// it the way the decode kernel does.  For testing that a wait that runs out ends cleanly.
__global__ void wait_timeout_kernel(float *partials, uint32_t *status, uint32_t limit)
{
    float4 t[4];
    const bool ready = wait_for_sums(reinterpret_cast<const float4 *>(partials) + threadIdx.x, 0, 0, 1, 1, limit, t);
    const bool gave_up = __any_sync(0xffffffffu, !ready);
    if (gave_up && threadIdx.x == 0) atomicCAS(status, 0u, (uint32_t)TMAN_ERR_TIMEOUT);
}

tman_status launch_wait_timeout(void *ws, size_t ws_bytes, uint32_t limit, cudaStream_t s)
{
    if (ws_bytes < kWsStatusBytes + 32 * sizeof(float4)) return TMAN_ERR_BUFFER_TOO_SMALL;
    uint8_t *w8 = static_cast<uint8_t *>(ws);
    wait_timeout_kernel<<<1, 32, 0, s>>>(reinterpret_cast<float *>(w8 + kWsStatusBytes), reinterpret_cast<uint32_t *>(w8), limit);
    return launch_status();
}

// status word (and its padding) zero, everything after it "no sum pending"
tman_status launch_workspace_init(void *ws, size_t ws_bytes, cudaStream_t s)
{
    const size_t words = ws_bytes / 4;
    ws_fill_kernel<<<(unsigned)((words + 255) / 256), 256, 0, s>>>(static_cast<uint32_t *>(ws), words);
    return launch_status();
}

size_t mpgemv_workspace_bytes(int M, int K, int N, int bits)
{
    // what the preferred plan needs (on the reference device size: the choice of variants depends on the
    // SM count only through the limit on K-slices); a smaller workspace makes the call fall back to
    // variants with fewer rows per pass, down to what one row needs
    const GemvPlan g = plan_gemv(M, K, N, bits, 128, kGemvPlanSms, (size_t)-1);      // (the group has no part in the size)
    return g.npass ? g.ws_bytes : (size_t)-1;
}

tman_status launch_mpgemv_grouped(int count, const void *const *packed, const void *x, void *const *y, int M, int K,
                                  const int *Ns, int bits, int group, void *ws, size_t ws_bytes, cudaStream_t s)
{
    const int sms = sm_count();
    if (sms <= 0) return TMAN_ERR_CUDA;
    int ntot = 0;
    for (int g = 0; g < count; ++g) ntot += Ns[g];
    const GemvPlan plan = plan_gemv(M, K, ntot, bits, group, sms, ws_bytes);
    if (plan.npass == 0) return TMAN_ERR_UNSUPPORTED;
    uint8_t *w8 = static_cast<uint8_t *>(ws);
    GemvParams p;
    p.count = count;
    p.N = 0;
    for (int g = 0; g < kGemvMaxGroup; ++g) {
        const int gg = g < count ? g : 0;
        Layout L = make_layout(K, Ns[gg], bits, group);
        const uint8_t *pk = static_cast<const uint8_t *>(packed[gg]);
        p.packed[g] = pk;
        p.planes[g] = reinterpret_cast<const uint4 *>(pk + L.planes_off);
        p.scales[g] = reinterpret_cast<const uint2 *>(pk + L.scales_off);
        p.zeros[g] = reinterpret_cast<const uint16_t *>(pk + L.zeros_off);
        p.Ng[g] = g < count ? Ns[g] : 0;
        p.col0[g] = p.N;
        p.unit0[g] = 0;
        if (g < count) p.N += Ns[g];
    }
    p.status = reinterpret_cast<uint32_t *>(w8);
    p.partials = reinterpret_cast<float *>(w8 + kWsStatusBytes);
    p.xi = nullptr; p.row_scale = nullptr; p.w_scale = 0.f; p.acc_out = nullptr;
    p.K = K; p.bits = bits; p.group = group;
    p.M = 0; p.nkappa = 0; p.P = 0; p.units = 0;
    p.group_shift = (group == 32) ? 5 : (group == 64) ? 6 : 7;
    p.nblk = K / group;
    // a table entry carries up to four rows (two fp16 pairs), the tensor cores eight: normally one pass over the weights
    int m0 = 0;
    for (int ps = 0; ps < plan.npass; ++ps) {
        const int rows = plan.pass[ps].rows;
        p.x = static_cast<const __half *>(x) + (size_t)m0 * K;
        for (int g = 0; g < kGemvMaxGroup; ++g)
            p.y[g] = static_cast<__half *>(y[g < count ? g : 0]) + (size_t)m0 * p.Ng[g];
        tman_status st;
        if (bits == 2) st = launch_rows<2>(p, plan.pass[ps], sms, s);
        else if (bits == 3) st = launch_rows<3>(p, plan.pass[ps], sms, s);
        else st = launch_rows<4>(p, plan.pass[ps], sms, s);
        if (st != TMAN_OK) return st;
        m0 += rows;
    }
    return TMAN_OK;
}

// ---- integer path: per-tensor ternary weights, 16-bit integer activations ---------------------------
// Per-row symmetric quantization of the activations (paper Sec. 6.1, A_INT16; 8 bits for the matrix unit):
// s_a = max|x| / qmax and a = round(x / s_a), both in single precision with correctly rounded division and
// rounding to nearest even, so that the integers are the same on any IEEE machine.  One CTA per row.
//
// quantize_rows_regs_kernel: the row (K % 8 == 0, 16-byte aligned rows) is read once and kept in registers, VPT vectors of
// eight values a thread; one barrier; the quotient is the row's reciprocal times x, corrected to the correctly rounded
// quotient with two remainder steps (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", IBM J. Res. Dev. 34, 1990, division by a correctly rounded reciprocal: q' = q + (x - q s) y, the remainder
// exact by fused multiply-add; the first step brings q, off by at most 1.5 units in the last place, to a neighbour of the
// quotient, the second rounds it).  No intermediate leaves the normal range: 2^-24 <= |x| < 2^16 and 2^-40 < s < 2^10.
// Launched so that it may start while its predecessor drains; its successor may start when the predecessor has ended.
// Against two passes with a full division per value in one CTA of 512 threads a row: 2048 rows of 2560 and the INT8
// product with 6912 channels after them 61.3 -> 50.2 us; one row and its decode, mean of 2560 x 6912 and 6912 x 2560,
// 7.4 -> 5.7 us (6.0 with the successor let go before the wait, which suited two to four rows better: 7.7 against 8.0).
template <typename OUT>
__device__ __forceinline__ void store_eight(OUT *out, const int (&q)[8])
{
    if constexpr (sizeof(OUT) == 2)
        *reinterpret_cast<uint4 *>(out) =
            make_uint4(__byte_perm((uint32_t)q[0], (uint32_t)q[1], 0x5410), __byte_perm((uint32_t)q[2], (uint32_t)q[3], 0x5410),
                       __byte_perm((uint32_t)q[4], (uint32_t)q[5], 0x5410), __byte_perm((uint32_t)q[6], (uint32_t)q[7], 0x5410));
    else {
        const uint32_t a = __byte_perm((uint32_t)q[0], (uint32_t)q[1], 0x0040), b = __byte_perm((uint32_t)q[2], (uint32_t)q[3], 0x0040);
        const uint32_t c = __byte_perm((uint32_t)q[4], (uint32_t)q[5], 0x0040), d = __byte_perm((uint32_t)q[6], (uint32_t)q[7], 0x0040);
        *reinterpret_cast<uint2 *>(out) = make_uint2(__byte_perm(a, b, 0x5410), __byte_perm(c, d, 0x5410));
    }
}

template <typename OUT, int VPT>      // int16_t or int8_t
__global__ void __launch_bounds__(1024) quantize_rows_regs_kernel(const __half *x, int nvec, int qmax,
                                                                  OUT *__restrict__ a, float *__restrict__ s_a)
{
    __shared__ float red[32];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // (after the wait: a decode that follows reads its weights at once)
    const uint4 *row = reinterpret_cast<const uint4 *>(x) + (size_t)blockIdx.x * nvec;
    OUT *out = a + (size_t)blockIdx.x * nvec * 8;
    uint4 v[VPT];
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int at = threadIdx.x + i * blockDim.x;
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (at < nvec) v[i] = ld_dependent(row + at);
    }
    __half2 mx = __floats2half2_rn(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
        mx = __hmax2(mx, __hmax2(__hmax2(__habs2(h[0]), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3]))));
    }
    float amax = fmaxf(__low2float(mx), __high2float(mx));
    for (int mask = 16; mask > 0; mask >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, mask));
    const int warps = blockDim.x >> 5;
    if (warps > 1) {
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
        __syncthreads();
        amax = (int)(threadIdx.x & 31) < warps ? red[threadIdx.x & 31] : 0.f;
        for (int mask = 16; mask > 0; mask >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, mask));
    }
    const float scale = amax > 0.f ? __fdiv_rn(amax, (float)qmax) : 1.f;
    const float inv = __frcp_rn(scale);
    if (threadIdx.x == 0) s_a[blockIdx.x] = scale;
    auto quant = [&](float f) {
        float q = f * inv;
        q = fmaf(fmaf(-q, scale, f), inv, q);
        q = fmaf(fmaf(-q, scale, f), inv, q);
        return (int)max(-qmax, min(qmax, __float2int_rn(q)));
    };
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
        const int at = threadIdx.x + i * blockDim.x;
        if (at < nvec) {
            const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
            int q[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 f = __half22float2(h[e]);
                q[2 * e] = quant(f.x);
                q[2 * e + 1] = quant(f.y);
            }
            store_eight<OUT>(out + (size_t)at * 8, q);
        }
    }
}

// Any K and rows longer than the registers of a CTA hold: two passes over the row (the second from L1/L2), eight values at a time
// where the rows allow 16-byte accesses (VEC: K % 8 == 0), else one by one.  2048 rows of 32776: 76.7 us, one by one 177.6; one row
// of 65536: 9.9 and 21.6.
template <typename OUT, bool VEC>
__global__ void __launch_bounds__(1024) quantize_rows_kernel(const __half *__restrict__ x, int K, int qmax,
                                                             OUT *__restrict__ a, float *__restrict__ s_a)
{
    __shared__ float red[32];
    const __half *row = x + (size_t)blockIdx.x * K;
    OUT *out = a + (size_t)blockIdx.x * K;
    const int nvec = VEC ? K >> 3 : 0;
    const uint4 *row8 = reinterpret_cast<const uint4 *>(row);
    float amax = 0.f;
    for (int i = threadIdx.x; i < nvec; i += blockDim.x) {
        const uint4 q = __ldg(row8 + i);
        const __half2 *h = reinterpret_cast<const __half2 *>(&q);
        const __half2 m = __hmax2(__hmax2(__habs2(h[0]), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3])));
        amax = fmaxf(amax, fmaxf(__low2float(m), __high2float(m)));
    }
    for (int k = 8 * nvec + threadIdx.x; k < K; k += blockDim.x) amax = fmaxf(amax, fabsf(__half2float(row[k])));
    for (int mask = 16; mask > 0; mask >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, mask));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
        for (int mask = 16; mask > 0; mask >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, mask));
        if (threadIdx.x == 0) red[0] = v;
    }
    __syncthreads();
    amax = red[0];
    const float scale = amax > 0.f ? __fdiv_rn(amax, (float)qmax) : 1.f;
    if (threadIdx.x == 0) s_a[blockIdx.x] = scale;
    auto quant = [&](__half v) {
        const int r = __float2int_rn(__fdiv_rn(__half2float(v), scale));
        return (int)max(-qmax, min(qmax, r));
    };
    for (int i = threadIdx.x; i < nvec; i += blockDim.x) {
        const uint4 q = __ldg(row8 + i);
        const __half *h = reinterpret_cast<const __half *>(&q);
        int o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) o[e] = quant(h[e]);
        store_eight<OUT>(out + (size_t)i * 8, o);
    }
    for (int k = 8 * nvec + threadIdx.x; k < K; k += blockDim.x) out[k] = (OUT)quant(row[k]);
}

template <typename OUT>
static tman_status launch_quantize(const void *x, int M, int K, int qmax, OUT *a, float *s_a, cudaStream_t s)
{
    const __half *xh = static_cast<const __half *>(x);
    const int nvec = K / 8;
    // Few rows: the latency of one row counts, every vector its own thread.  Many rows: four vectors a thread, so that a
    // row's reduction is spread over fewer threads (2048 rows of 2560: 96 threads; the limit of 1024 threads holds 8 x 4
    // values each, longer rows are read twice).
    const bool few = M <= 2 * kGemvPlanSms && nvec <= 1024;
    const int vpt = few ? 1 : 4;
    if (K % 8 != 0 || nvec > 1024 * 4) {
        const int threads = K >= 8192 ? 1024 : (K >= 2048 ? 512 : 256);
        if (K % 8 == 0) quantize_rows_kernel<OUT, true><<<(unsigned)M, threads, 0, s>>>(xh, K, qmax, a, s_a);
        else quantize_rows_kernel<OUT, false><<<(unsigned)M, threads, 0, s>>>(xh, K, qmax, a, s_a);
        return launch_status();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)M);
    cfg.blockDim = dim3((unsigned)(((nvec + vpt - 1) / vpt + 31) / 32 * 32));
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto kern = few ? quantize_rows_regs_kernel<OUT, 1> : quantize_rows_regs_kernel<OUT, 4>;
    if constexpr (sizeof(OUT) == 2) {                                            // (a decode follows)
        static std::atomic<bool> preferred[2][kMaxDevices];
        int dev = 0;
        if (!device_info(&dev)) return TMAN_ERR_CUDA;
        if (!preferred[few][dev].load(std::memory_order_relaxed)) {
            prefer_common_split(kern);
            preferred[few][dev].store(true, std::memory_order_relaxed);
        }
    }
    return cudaLaunchKernelEx(&cfg, kern, xh, nvec, qmax, a, s_a) == cudaSuccess ? TMAN_OK : TMAN_ERR_CUDA;
}

tman_status launch_quantize_rows(const void *x, int M, int K, int qmax, int16_t *a, float *s_a, cudaStream_t s)
{
    return launch_quantize<int16_t>(x, M, K, qmax, a, s_a, s);
}

tman_status launch_quantize_rows_i8(const void *x, int M, int K, int8_t *a, float *s_a, cudaStream_t s)
{
    return launch_quantize<int8_t>(x, M, K, 127, a, s_a, s);
}

// Rows of 16-bit integer activations times ternary weights packed as 2-bit codes (zero-point 1; the
// packed buffer's scales and zero-points are not read).  y = fp16(s_a[m] * s_w * sum), acc_out (may be NULL)
// receives the exact integer sums.  Integer table entries are held exactly in fp32, one per row: passes of
// one row (K-slices of 16 plane words), two rows (16 words) or four rows (8 words) per table entry.
static void ternary_variant(int rows, int *mt, int *words)
{
    if (rows <= 1) { *mt = 1; *words = 16; }
    else if (rows == 2) { *mt = 2; *words = 16; }
    else { *mt = 4; *words = 8; }
}

size_t mpgemv_ternary_workspace_bytes(int M, int K, int N)
{
    int mt = 1, words = 16;
    ternary_variant(M < 4 ? M : 4, &mt, &words);
    const size_t nkappa = (size_t)(K / 32 + words - 1) / (size_t)words;
    return kWsStatusBytes + nkappa * (size_t)mt * (size_t)N * sizeof(float);
}

tman_status launch_mpgemv_ternary(const void *packed, const int16_t *a, const float *s_a, float s_w, void *y,
                                  int32_t *acc_out, int M, int K, int N, int group, void *ws, size_t, cudaStream_t s)
{
    const int sms = sm_count();
    if (sms <= 0) return TMAN_ERR_CUDA;
    uint8_t *w8 = static_cast<uint8_t *>(ws);
    GemvParams p = {};
    p.count = 1;
    Layout L = make_layout(K, N, 2, group);
    const uint8_t *pk = static_cast<const uint8_t *>(packed);
    for (int g = 0; g < kGemvMaxGroup; ++g) {
        p.packed[g] = pk;
        p.planes[g] = reinterpret_cast<const uint4 *>(pk + L.planes_off);
        p.scales[g] = reinterpret_cast<const uint2 *>(pk + L.scales_off);
        p.zeros[g] = reinterpret_cast<const uint16_t *>(pk + L.zeros_off);
        p.Ng[g] = g == 0 ? N : 0;
        p.col0[g] = g == 0 ? 0 : N;
    }
    p.N = N;
    p.x = nullptr;
    p.w_scale = s_w;
    p.status = reinterpret_cast<uint32_t *>(w8);
    p.partials = reinterpret_cast<float *>(w8 + kWsStatusBytes);
    p.K = K; p.bits = 2; p.group = group;
    p.group_shift = (group == 32) ? 5 : (group == 64) ? 6 : 7;
    p.nblk = K / group;
    const bool pre = group >= 64;
    if (uses_digits_ternary(M, K, N, group, sms)) {
        DigitParams d = {};
        d.count = 1;
        for (int i = 0; i < kGemvMaxGroup; ++i) {
            d.packed[i] = p.packed[0];
            d.planes[i] = reinterpret_cast<const uint8_t *>(p.planes[0]);
            d.y[i] = static_cast<__half *>(y);
            d.Ng[i] = N;
            d.strip0[i + 1] = N / 4;
        }
        d.x = a; d.row_scale = s_a; d.w_scale = s_w; d.acc_out = acc_out;
        d.status = p.status;
        d.M = M; d.K = K; d.bits = 2; d.group = group; d.nblk = p.nblk;
        return M <= 2 ? launch_digits<2, 1, 1, true>(d, sms, s) : M <= 4 ? launch_digits<2, 1, 2, true>(d, sms, s)
             : M <= 6 ? launch_digits<2, 1, 3, true>(d, sms, s) : launch_digits<2, 1, 4, true>(d, sms, s);
    }
    for (int m0 = 0; m0 < M; m0 += 4) {
        const int rows = (M - m0 < 4) ? (M - m0) : 4;
        int mt = 1, words = 16;
        ternary_variant(rows, &mt, &words);
        if ((K / 32 + words - 1) / words > sms) return TMAN_ERR_UNSUPPORTED;      // every K-slice needs a resident CTA
        p.M = rows;
        p.xi = a + (size_t)m0 * K;
        p.row_scale = s_a + m0;
        p.acc_out = acc_out ? acc_out + (size_t)m0 * N : nullptr;
        for (int g = 0; g < kGemvMaxGroup; ++g) p.y[g] = static_cast<__half *>(y) + (size_t)m0 * N;
        tman_status st;
        if (mt == 1) st = pre ? launch_one<2, 1, 4, 1, 1, 0, 0, 1>(p, sms, s) : launch_one<2, 1, 4, 0, 1, 0, 0, 1>(p, sms, s);
        else if (mt == 2) st = pre ? launch_one<2, 2, 2, 1, 0, 0, 0, 1>(p, sms, s) : launch_one<2, 2, 2, 0, 0, 0, 0, 1>(p, sms, s);
        else st = pre ? launch_one<2, 4, 1, 1, 0, 0, 0, 1>(p, sms, s) : launch_one<2, 4, 1, 0, 0, 0, 0, 1>(p, sms, s);
        if (st != TMAN_OK) return st;
    }
    return TMAN_OK;
}

tman_status launch_mpgemv(const void *packed, const void *x, void *y, int M, int K, int N, int bits,
                          int group, void *ws, size_t ws_bytes, cudaStream_t s)
{
    return launch_mpgemv_grouped(1, &packed, x, &y, M, K, &N, bits, group, ws, ws_bytes, s);
}

}  // namespace tman
