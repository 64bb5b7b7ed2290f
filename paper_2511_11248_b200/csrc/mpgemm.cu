// Prefill path: dequantization fused into a tcgen05 GEMM whose weight operand lives in tensor memory
// (paper Sec. 4.1 "Unified Layout through Fused LUT-based Dequantization", Fig. 7;
//  Sec. 4.2 "Pipelining to Hide Dequantization Overhead", Fig. 9).
//
// The product is computed transposed: channels are the rows of the tensor-core tile (128 per CTA), tokens its columns (up
// to 256).  A thread that rebuilds weights then owns one channel = one lane of tensor memory, writes its fp16 weights there
// in k order (tcgen05.st), and the MMA reads them as its A operand: weights never pass through shared memory, and a tile of
// few tokens costs few columns instead of a padded block of 128 rows.  The tokens' activations are the B operand, in shared
// memory as TMA leaves them.
// The output is cut into tiles of 128 channels (a CTA) or 256 (a pair of CTAs on two SMs, tcgen05.mma.cta_group::2: each CTA
// holds half of the tokens' rows and rebuilds its own 128 channels, so that an activation is fetched once per 256 channels).
// A tile's work is its K/128 units of 128 k.  The host chooses the tokens of a tile and deals the tiles to the workers (CTAs or
// pairs, at most one per SM or SM pair), whole as far as they go round; where whole tiles would leave SMs idle, the
// units of the last tiles are laid end to end and dealt in equal spans, and a tile whose units fall into several
// spans is summed through fp32 partial tiles in the workspace (see "split of the work").
// The integer path (per-tensor ternary weights, INT8 activations; paper Sec. 6.2) is the same kernel with kind::i8: codes become
// bytes by a table lookup, sums are exact 32-bit integers, the epilogue applies the token's and the tensor's scale.
// Four kinds of agents run concurrently, guarded by mbarriers (the paper's DMA / vector-core / matrix-core stages):
//   * warp 0, one lane : TMA loads of the activations (a ring of units, 128-byte swizzle) and, running ahead on a ring of its own, of the
//                        packed bit-plane words (runs of 128 bytes per strip and plane);
//   * warps 2..17      : four groups of four warps, each group every fourth unit of the walk: read the plane words of their channel,
//                        merge them into codes (level 1: bit-serial -> bit-parallel), turn codes into fp16 weights (level 2)
//                        and store them to tensor memory;
//   * warp 1, one lane : tcgen05.mma (fp16 x fp16 -> fp32 in tensor memory), one per 16 k; tcgen05.commit hands the
//                        activations' slot and the weights' columns back;
//   * warps 18..25     : epilogue (tcgen05.ld, round to fp16, exchange between neighbouring lanes, 4-byte stores).
// Barriers that both CTAs of a pair feed (weights ready, accumulator drained) live in its first CTA, which issues the MMAs;
// the commits arrive in both.  No TMA multicast: each CTA loads its own data.
// Every wait is bounded: when a bound is hit the kernel records TMAN_ERR_TIMEOUT, stops issuing
// work, and still reaches the common tear-down that frees tensor memory.
#include "common.cuh"

#include <mutex>

#include <cuda.h>

#include "sm100_ptx.cuh"

namespace tman {
namespace {

constexpr int BK = 64;                          // k of a 128-byte row of activations in shared memory
constexpr int UK = 128;                         // k of a unit: what a group of warps rebuilds at a time
constexpr int CH = 128;                         // channels a CTA rebuilds = lanes of tensor memory
constexpr int MAX_TOKENS = 256;                 // columns of an accumulator
constexpr int NUM_DEQ_WARPS = 16, DEQ_GROUPS = 4;
constexpr int NUM_EPI_WARPS = 8;                // two per quarter of the tensor-memory lanes (alternate 32-token chunks)
constexpr int GEMM_THREADS = 32 * (2 + NUM_DEQ_WARPS + NUM_EPI_WARPS);
constexpr int P_PLANE_BYTES = (CH / 4) * 128;   // one plane of a packed stage (two units): a 128-byte run per strip
constexpr int P_RING_BYTES = 64 * 1024;         // 8 stages for 2 bits, 4 for 3 and 4
constexpr int P_LOAD_BARS = 8, X_LOAD_BARS = 8; // "loaded" barriers of the packed stages and, integer path, of the activations', whatever the number of slots (see the dequantization)
constexpr int X_RING_BYTES = 128 * 1024;        // activation ring: stages of two units (8 of up to 32 rows, 4 of up to 64) or one (4 of up to 128)
constexpr int W_TILE_BYTES = CH * BK * 2;       // half a unit of fp16 weights in shared memory (LoadFull variant only)
constexpr int TMEM_COLS = 512;                  // accumulator from column 0, weight buffers of 64 columns behind it
constexpr int kMaxGemmCtas = 160;               // the workspace is sized for at most this many CTAs
constexpr int GEMM_SMEM = P_RING_BYTES + X_RING_BYTES + 512;

// Workspace: status word (kWsStatusBytes), one flag per epilogue warp of every CTA (spans), one per (epilogue warp of a
// CTA, sending piece) (even pieces), then one fp32 partial tile per CTA (a worker writes at most one per launch): per
// epilogue warp [token][channel], its 32 channels x half of the tokens.
constexpr int kMaxSplit = 32;                   // even pieces of a tile
constexpr size_t kGemmFlagsOff = kWsStatusBytes;
constexpr size_t kGemmPieceFlagsOff = kWsStatusBytes + 8192;
constexpr size_t kGemmPartialOff = kGemmPieceFlagsOff + (size_t)kMaxGemmCtas * NUM_EPI_WARPS * kMaxSplit * sizeof(uint32_t);
constexpr uint32_t kFlagEmpty = 0x7FA5A5A5u;    // what tman_workspace_init leaves behind
// Role time stamps (only in a library built with -DTMAN_ROLE_STAMPS; the workspace has room for them in
// every build so that its layout does not depend on the flag): per CTA and warp four 64-bit words --
// clocks spent in the role's first kind of wait, in its second kind, in the whole role, and a tag.
//   warp 0 (TMA producer): waits for a free slot or stage    warp 1 (MMA issuer): accumulator free / weights ready
//   warps 2..17 (dequantization): packed stage loaded / weight buffer free    warps 18..25 (epilogue): accumulators complete
constexpr int kStampWordsPerWarp = 4;
constexpr int kGemmWarps = 2 + NUM_DEQ_WARPS + NUM_EPI_WARPS;
constexpr size_t kStampBytesPerCta = (size_t)kGemmWarps * kStampWordsPerWarp * sizeof(long long);
#ifdef TMAN_ROLE_STAMPS
#define TMAN_STAMPED_WAIT(acc, call) ([&]() { const long long t_ = clock64(); const bool r_ = (call); (acc) += clock64() - t_; return r_; }())
#else
#define TMAN_STAMPED_WAIT(acc, call) (call)
#endif
constexpr size_t kPartialBytesPerCta = (size_t)MAX_TOKENS * CH * sizeof(float);

struct GemmParams {
    const uint8_t  *packed;
    const __half   *scales;
    const uint16_t *zeros;
    __half         *y;
    uint32_t       *status;
    uint32_t       *flags, *piece_flags;
    float          *partial;
    int M, K, N, bits, group;
    int nt;                    // tokens of a tile (a multiple of 16, of 32 in a pair)
    int wbufs, wcol;           // weight buffers in tensor memory and their first column
    int xu_sh, xst_sh;         // activation ring: log2 of the units of a stage and of the stages
    int tiles_m, tiles_n;
    int span_tiles;            // the last span_tiles tiles are dealt as equal spans of units (0: every tile whole)
    int split_s;               // even pieces of every tile (0: not split so)
    int col_fastest;           // tile number = row tile * tiles_n + column tile (else column tile * tiles_m + row tile)
    int acc_sh, acc_col;       // log2 of the accumulators in tensor memory (two: the epilogue of a tile overlaps the next one), their distance in columns
    const float *row_scale;    // integer path: scales of the tokens and of the tensor
    float w_scale;
    long long *stamps;         // role time stamps (written only by a build with TMAN_ROLE_STAMPS)
};

// Ablation variants of the kernel (paper Sec. 6.5 "Ablation Study"): what replaces the dequantization, or the
// pipelining.  Every variant computes the same numbers.
constexpr int kGemmProduct = 0;      // the product path, pipelined
constexpr int kGemmConvertDq = 1;    // codes converted to floating point one by one, then subtract and multiply
constexpr int kGemmLoadFull = 2;     // fp16 weights prepared in memory and loaded by TMA, no dequantization
constexpr int kGemmInt8 = 4;         // integer path: ternary weights as 8-bit integers, 8-bit activations, exact 32-bit sums (2-bit codes, whole tiles)
constexpr int kGemmSequential = 3;   // the product's dequantization; a unit is loaded when the one before it has been multiplied, and dequantized when it is loaded

template <int I> struct IntC { static constexpr int value = I; };

// ---- level 2: codes to fp16 weights ---------------------------------------------------------------
// w = fp16( s * (c - z) ), rounded once.  A code in the mantissa of an fp16 number between 1024 and 2048 is 1024 + c
// (1024 + 16 c four bits higher); one fused multiply-add takes the 1024 and the zero-point off exactly, one multiply applies
// the scale.  (A register table addressed by byte permutes, four lookups and a select per four 4-bit codes, gives the same
// weights with twice the operations on the half-rate integer pipe: 110 against 48 per 32 weights.)
struct BlockConsts {
    __half2 s2, sub;                             // scale; -(1024 + z) for the low code of a pair, -(64 + z) for the high one
    __device__ __forceinline__ void set(__half s, uint32_t z)
    {
        s2 = __half2half2(s);
        const uint32_t u = z * 0x00100001u + 0xD400E400u;        // the two constants with z in their mantissas
        sub = *reinterpret_cast<const __half2 *>(&u);
    }
};

// The same 32 weights without the conversion table: every code is extracted, converted to fp16 by an
// integer-to-float conversion, the zero-point subtracted and the scale multiplied (rounds like the table's
// entries do, so the result is the same bits).
template <int BITS>
__device__ __forceinline__ void dequant_word_convert(const uint32_t (&w)[BITS], __half s, uint32_t z, uint32_t (&out)[16])
{
    const __half2 s2 = __half2half2(s);
    const __half2 z2 = __half2half2(__ushort2half_rn((unsigned short)z));
#pragma unroll
    for (int ph = 0; ph < 4; ++ph)
#pragma unroll
        for (int jp = 0; jp < 4; ++jp) {
            // weights 8*ph + 2*jp and 8*ph + 2*jp + 1 sit at word bits 4*(2*jp) + ph and 4*(2*jp + 1) + ph
            uint32_t c0 = 0u, c1 = 0u;
#pragma unroll
            for (int i = 0; i < BITS; ++i) {
                c0 |= ((w[i] >> (8 * jp + ph)) & 1u) << i;
                c1 |= ((w[i] >> (8 * jp + 4 + ph)) & 1u) << i;
            }
            const __half2 c = __halves2half2(__ushort2half_rn((unsigned short)c0), __ushort2half_rn((unsigned short)c1));
            const __half2 e = __hmul2(s2, __hsub2(c, z2));
            out[4 * ph + jp] = *reinterpret_cast<const uint32_t *>(&e);
        }
}

// 32 weights of one channel (one plane word per bit) -> 16 half2 in k order.
template <int BITS>
__device__ __forceinline__ void dequant_word(const uint32_t (&w)[BITS], const BlockConsts &t, uint32_t (&out)[16])
{
    // level 1 (bit repacking): X[ph] nibble j = code of the weight at word bit 4j + ph, which the
    // packed format makes weight 8*ph + j: X[ph] holds weights 8ph .. 8ph+7 in order.  A 4 x 4
    // bit-block transpose of the plane words: first planes 0/1 and 2/3 are interleaved bit by bit,
    // then the two results two bits by two bits (each step is one shift and one bit-select).  Bits of a
    // nibble above the code are left over from its neighbours; the mask below drops them.
    uint32_t X[4];
    {
        const uint32_t a0 = bsel(0x55555555u, w[0], w[1] << 1), a1 = bsel(0x55555555u, w[0] >> 1, w[1]);
        if constexpr (BITS == 2) {
            X[0] = a0; X[1] = a1; X[2] = a0 >> 2; X[3] = a1 >> 2;
        } else if constexpr (BITS == 3) {
            X[0] = bsel(0x33333333u, a0, w[2] << 2);
            X[1] = bsel(0x33333333u, a1, w[2] << 1);
            X[2] = bsel(0x33333333u, a0 >> 2, w[2]);
            X[3] = bsel(0x33333333u, a1 >> 2, w[2] >> 1);
        } else {
            const uint32_t w3 = w[BITS - 1];
            const uint32_t b0 = bsel(0x55555555u, w[2], w3 << 1), b1 = bsel(0x55555555u, w[2] >> 1, w3);
            X[0] = bsel(0x33333333u, a0, b0 << 2);
            X[1] = bsel(0x33333333u, a1, b1 << 2);
            X[2] = bsel(0x33333333u, a0 >> 2, b0);
            X[3] = bsel(0x33333333u, a1 >> 2, b1);
        }
    }
    // level 2: byte b of X holds the codes of two adjacent weights; copied into both halves of a register, the low
    // half keeps the low nibble and the high half the high one
    constexpr uint32_t M1 = (1u << BITS) - 1u, MASK = M1 | (M1 << 20);
    const uint32_t magic = opaque_u32<0x64006400u>();
    const __half2 mul = __halves2half2(__ushort2half_rn(1), __float2half_rn(0.0625f));
#pragma unroll
    for (int ph = 0; ph < 4; ++ph)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const uint32_t c = and_or(__byte_perm(X[ph], 0u, 0x1111u * b), MASK, magic);
            const __half2 e = __hmul2(t.s2, __hfma2(*reinterpret_cast<const __half2 *>(&c), mul, t.sub));
            out[4 * ph + b] = *reinterpret_cast<const uint32_t *>(&e);
        }
}

// 32 ternary weights of one channel (2-bit codes, zero-point 1) -> 32 INT8 in k order (level 1 as above; level 2 looks four codes
// at a time up in a four-entry byte table with one byte permute).
__device__ __forceinline__ void dequant_word_int8(const uint32_t (&w)[2], uint32_t *out)
{
    const uint32_t table = 0x000100FFu;          // -1, 0, +1; (3 does not occur) 0
    const uint32_t a0 = bsel(0x55555555u, w[0], w[1] << 1), a1 = bsel(0x55555555u, w[0] >> 1, w[1]);
    const uint32_t X[4] = {a0 & 0x33333333u, a1 & 0x33333333u, (a0 >> 2) & 0x33333333u, (a1 >> 2) & 0x33333333u};
#pragma unroll
    for (int ph = 0; ph < 4; ++ph) {
        out[2 * ph] = __byte_perm(table, 0u, X[ph]);
        out[2 * ph + 1] = __byte_perm(table, 0u, X[ph] >> 16);
    }
}

// ---- split of the work ----------------------------------------------------------------------
// T tiles (row tile fastest), W workers.  The first `whole` tiles (a multiple of W) are dealt whole,
// round-robin.  The units of the remaining tiles (fewer than 2 W), laid end to end (a unit is as deep as the
// longest quantization block), are dealt in equal contiguous spans, so
// every worker is busy to the end whatever the shape.  A span is shorter than two tiles: at most
// the end of one tile, one whole tile and the start of the next.  A tile cut into several pieces
// ("split tile") is summed by the worker that owns its last unit: the others, which all have lower
// numbers, write their fp32 accumulators to the workspace and raise a flag.  A worker's walk: first
// the piece that it only contributes (so that it is ready long before it is needed), then its whole
// tiles, last the piece of the tile that it finishes.
// Even pieces (outputs with few tiles): as many workers as tiles x pieces, so that the spans are the pieces.  They finish
// together and share the summing: every piece sends the accumulators of the tokens that others sum, and adds up its own.
struct Segment { int tile, u0, u1; bool whole, finishes; };

struct Span {
    int full, Ur;              // tiles dealt whole round-robin; units of the remaining tiles (Ur x workers fits 31 bits, host)
    int next_whole;            // next round-robin tile of this worker
    int nu, W;
    Segment early, mid, late;  // the piece this worker only contributes; a whole tile of its span; the piece it finishes
    bool has_early, has_mid, has_late;
    __device__ Span(const GemmParams &p, int worker, int nworkers)
        : full(p.tiles_m * p.tiles_n - p.span_tiles), Ur(0), next_whole(worker), nu(p.K / UK), W(nworkers),
          has_early(false), has_mid(false), has_late(false)
    {
        if (p.span_tiles == 0) return;
        Ur = p.span_tiles * nu;
        const int lo = (int)((unsigned)(Ur * worker) / (unsigned)W);
        int hi = (int)((unsigned)(Ur * (worker + 1)) / (unsigned)W);
        for (int i = 0; i < 3 && hi > lo; ++i) {       // from the last tile of the span to the first
            const int tile = (int)((unsigned)(hi - 1) / (unsigned)nu), t0 = tile * nu;
            const int k0 = (lo > t0) ? lo - t0 : 0, k1 = hi - t0;
            Segment s;
            s.tile = full + tile;
            s.u0 = k0;
            s.u1 = k1;
            s.whole = (k0 == 0 && k1 == nu);
            s.finishes = (k1 == nu);
            if (s.whole) { mid = s; has_mid = true; }
            else if (s.finishes) { late = s; has_late = true; }
            else { early = s; has_early = true; }
            hi = t0 + k0;
        }
    }
    __device__ bool next(Segment &s)
    {
        if (has_early) { s = early; has_early = false; return true; }
        if (next_whole < full) {
            s.tile = next_whole;
            s.u0 = 0;
            s.u1 = nu;
            s.whole = s.finishes = true;
            next_whole += W;
            return true;
        }
        if (has_mid) { s = mid; has_mid = false; return true; }
        if (has_late) { s = late; has_late = false; return true; }
        return false;
    }
    // the worker that owns unit u of tile `tile` (one of the remaining tiles)
    __device__ int owner(int tile, int u) const
    {
        const int g = (tile - full) * nu + u;
        return (int)((unsigned)((g + 1) * W - 1) / (unsigned)Ur);
    }
};

template <int BITS, bool PAIR, int V>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
mpgemm_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
              const __grid_constant__ CUtensorMap tmap_wf, const GemmParams p)
{
    constexpr int NCTA = PAIR ? 2 : 1;
    constexpr bool INT8 = V == kGemmInt8;
    constexpr int W_COLS = INT8 ? UK / 4 : UK / 2, X_UNIT_ROW = INT8 ? UK : 2 * UK;   // a unit: columns of weights, bytes of a token
    constexpr int P_STAGE_BYTES = BITS * P_PLANE_BYTES, P_STAGES = BITS == 2 ? 8 : 4;
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t rank = PAIR ? cluster_ctarank() : 0u;   // in a pair, CTA 0 issues the MMAs and owns the shared barriers
    uint8_t *p_tiles = smem, *x_tiles = smem + P_RING_BYTES;
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + P_RING_BYTES + X_RING_BYTES);
    // packed stage loaded (TMA) / free (the four warps of the groups of its two units); activation stage loaded (TMA) / free (MMA commit); weights of a
    // buffer ready (the four warps of a group; in a pair both CTAs' in CTA 0) / free (MMA commit); accumulator full (commit) /
    // empty (epilogue warps; in a pair both CTAs' in CTA 0)
    const uint32_t ploaded0 = smem_u32(bars), pempty0 = smem_u32(bars + 8), xloaded0 = smem_u32(bars + 16), xempty0 = smem_u32(bars + 24),
                   full0 = smem_u32(bars + 32), empty0 = smem_u32(bars + 40), accf0 = smem_u32(bars + 48), acce0 = smem_u32(bars + 60);
    const uint32_t sums0 = smem_u32(bars + 52);            // partial sums of an epilogue warp loaded
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 50);
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // (the shuffle tells the compiler that it is uniform)

    // (down to the wait: beside the previous kernel of the stream, without a look at memory)
    if (threadIdx.x == 0) {
        for (int s = 0; s < 8; ++s) {
            mbar_init(ploaded0 + 8 * s, 1);
            mbar_init(pempty0 + 8 * s, 2 * (NUM_DEQ_WARPS / DEQ_GROUPS));
            mbar_init(xloaded0 + 8 * s, 1);
            mbar_init(xempty0 + 8 * s, 1);
            mbar_init(full0 + 8 * s, NCTA * (NUM_DEQ_WARPS / DEQ_GROUPS));
            mbar_init(empty0 + 8 * s, 1);
            mbar_init(sums0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf0 + 8 * b, 1);
            mbar_init(acce0 + 8 * b, NCTA * NUM_EPI_WARPS);
        }
        *tmem_slot = 0xFFFFFFFFu;
        fence_barrier_init();
    } else if (threadIdx.x == 32 * 2) {
        prefetch_tensormap(&tmap_x);
        prefetch_tensormap(V == kGemmLoadFull ? &tmap_wf : &tmap_w);
    }
    if constexpr (PAIR) cluster_sync_all();            // both CTAs' barriers are set up
    else __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // Tensor memory only now: the previous kernel may be one that signals early and allocates its own on this SM afterwards; it
    // would wait for this one's columns, and this one for its end.  (Warp 0 needs none and starts its loads meanwhile, which hides the
    // allocation: with all warps behind it every call took 0.8 us longer.)  The next kernel may start only then, for the same reason,
    // and because a decode reads its weights at once, which may have been written by the kernel this one has waited for.
    uint32_t tmem_base = 0xFFFFFFFFu;
    bool ok = true;
    if (warp != 0) {
        if (warp == 1) {
            if constexpr (PAIR) {
                tcgen05_alloc2(smem_u32(tmem_slot), TMEM_COLS);
                tcgen05_relinquish2();
            } else {
                tcgen05_alloc(smem_u32(tmem_slot), TMEM_COLS);
                tcgen05_relinquish();
            }
        }
        tcgen05_fence_before();
        asm volatile("bar.sync 1, %0;" ::"n"(GEMM_THREADS - 32) : "memory");
        tcgen05_fence_after();
        tmem_base = *reinterpret_cast<volatile uint32_t *>(tmem_slot);
        ok = tmem_base != 0xFFFFFFFFu;
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    const bool run = (smem_u32(smem) & 1023u) == 0u;       // the swizzled tiles need 1 KB alignment (same in every CTA)
    if (!run && threadIdx.x == 0 && blockIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_LAYOUT);
    long long wait_a = 0, wait_b = 0;                  // clocks in this thread's waits (time-stamp builds only)
#ifdef TMAN_ROLE_STAMPS
    const long long role_t0 = clock64();
#endif
    const int worker = (int)blockIdx.x / NCTA, nworkers = (int)gridDim.x / NCTA;
    const int wbufs = p.wbufs, rows_cta = p.nt / NCTA;
    Span span(p, worker, nworkers);
    Segment sg;
    // Tiles with consecutive numbers run at the same time; the host numbers them so that a round of
    // tiles touches the fewest bytes (row tiles of activations, column tiles of packed weights).
    auto tile_tm = [&](int tile) { return p.col_fastest ? tile / p.tiles_n : tile % p.tiles_m; };
    auto tile_ct = [&](int tile) { return p.col_fastest ? tile % p.tiles_n : tile / p.tiles_m; };
    auto tile_ch0 = [&](int tile) { return tile_ct(tile) * (NCTA * CH) + (int)rank * CH; };      // this CTA's first channel
    const uint32_t full_lead = PAIR ? mapa_u32(full0, 0) : full0, acce_lead = PAIR ? mapa_u32(acce0, 0) : acce0;
    const uint32_t acc_mask = (1u << p.acc_sh) - 1u;   // tile ti of the walk: accumulator ti & acc_mask, its barriers' turn ti >> acc_sh
    auto arrive_lead = [&](uint32_t bar) {
        if constexpr (PAIR) mbar_arrive_cluster(bar);
        else mbar_arrive(bar);
    };

    if (!run) {
        // nothing to do: every output stays untouched
    } else if (warp == 0) {
        // ---- stage 1: activations and packed words by TMA -----------------------------------------------
        // The warp walks as one (uniform registers: operands of the copies), an elected lane issues both streams: the packed
        // stage a unit needs, further packed stages as far as their ring has room, the activations.  What a load needs
        // is worked out once a segment: a division per load made this thread the slowest agent (0.6 us per 64 k).
        const bool lead = elect_one();
        const uint32_t x_stage_bytes = (uint32_t)(rows_cta * X_UNIT_ROW) << p.xu_sh;
        const uint32_t p_base = smem_u32(p_tiles), x_base = smem_u32(x_tiles), xst_mask = (1u << p.xst_sh) - 1u;
        const int xu = 1 << p.xu_sh;
        Span ps = span;
        Segment pg;
        int pu = 0, pend = 0, pstrip = 0, ahead = 0;       // ahead: packed stages issued beyond the one the activations have reached
        uint32_t pc = 0;                                   // packed stages issued
        bool pmore = V != kGemmLoadFull;
        auto packed_next = [&]() {
            pmore = ps.next(pg);
            if (pmore) { pu = pg.u0; pend = pg.u1; pstrip = tile_ch0(pg.tile) / 4; }
        };
        auto packed_issue = [&]() {
            const uint32_t bar = ploaded0 + 8 * (pc % P_LOAD_BARS), dst = p_base + pc % P_STAGES * P_STAGE_BYTES;
            if (lead) {
                mbar_expect_tx(bar, P_STAGE_BYTES);
#pragma unroll
                for (int i = 0; i < BITS; ++i) tma_load_3d(dst + i * P_PLANE_BYTES, &tmap_w, pu * (UK / 8), i, pstrip, bar);
            }
            ++pc;
            ++ahead;
            pu += 2;
            if (pu >= pend) packed_next();
        };
        auto packed_bar = [&]() { return pempty0 + 8 * (pc % P_STAGES); };
        auto packed_par = [&]() { return ((pc / P_STAGES) & 1u) ^ 1u; };
        if (pmore) packed_next();
        uint32_t xc = 0;                                   // activation stages issued
        while (ok && span.next(sg)) {
            const int row0 = tile_tm(sg.tile) * p.nt + (int)rank * rows_cta, ch0 = tile_ch0(sg.tile);
            for (int u = sg.u0; u < sg.u1; u += xu, ++xc) {
                if (V != kGemmLoadFull && ((u - sg.u0) & 1) == 0) {
                    if (ahead == 0) {
                        if (!TMAN_STAMPED_WAIT(wait_a, warp_all(mbar_wait(packed_bar(), packed_par())))) { ok = false; break; }
                        packed_issue();
                    }
                    --ahead;
                    while (pmore && warp_all(mbar_test(packed_bar(), packed_par()))) packed_issue();
                }
                const uint32_t st = xc & xst_mask, bar = xloaded0 + 8 * (INT8 ? xc % X_LOAD_BARS : st);
                if constexpr (V == kGemmSequential)
                    if (xc > 0 && !warp_all(mbar_wait(xempty0 + 8 * ((xc - 1) & xst_mask), ((xc - 1) >> p.xst_sh) & 1u))) { ok = false; break; }
                if (!TMAN_STAMPED_WAIT(wait_a, warp_all(mbar_wait(xempty0 + 8 * st, ((xc >> p.xst_sh) & 1u) ^ 1u)))) { ok = false; break; }
                if (lead) {
                    mbar_expect_tx(bar, x_stage_bytes + (V == kGemmLoadFull ? 2 * W_TILE_BYTES : 0));
                    tma_load_3d(x_base + st * x_stage_bytes, &tmap_x, 0, row0, INT8 ? u : 2 * u, bar);
                    if constexpr (V == kGemmLoadFull) {
                        tma_load_2d(p_base + st * (2 * W_TILE_BYTES), &tmap_wf, u * UK, ch0, bar);
                        tma_load_2d(p_base + st * (2 * W_TILE_BYTES) + W_TILE_BYTES, &tmap_wf, u * UK + BK, ch0, bar);
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ---- stage 3: tensor-core MMA (in a pair: issued by CTA 0 for both) ----------------------
        // (the warp walks as one, so that the operands of the MMAs sit in uniform registers; an elected lane issues)
        if (rank == 0) {
            const bool lead = elect_one();
            // (integer path: s32 sums of s8 x s8; else fp32 sums of fp16 x fp16)
            const uint32_t idesc = (INT8 ? (2u << 4) | (1u << 7) | (1u << 10) : 1u << 4) | ((uint32_t)(p.nt >> 3) << 17) | ((uint32_t)((NCTA * CH) >> 4) << 24);
            // descriptors in 16-byte units: only the low word (start address) changes
            const uint64_t bdesc0 = make_kmajor_sw128_desc(smem_u32(x_tiles)), adesc0 = make_kmajor_sw128_desc(smem_u32(p_tiles));
            const uint32_t half_units = (uint32_t)rows_cta * 8u, xst_mask = (1u << p.xst_sh) - 1u;
            const int xu_mask = (1 << p.xu_sh) - 1;
            uint32_t ti = 0, ph = 0u, s = 0, xst = 0;
            while (ok && span.next(sg)) {
                if (!TMAN_STAMPED_WAIT(wait_a, warp_all(mbar_wait(acce0 + 8 * (ti & acc_mask), ((ti >> p.acc_sh) & 1u) ^ 1u)))) { ok = false; break; }
                tcgen05_fence_after();
                const uint32_t acc_tmem = tmem_base + (uint32_t)p.acc_col * (ti & acc_mask), accf = accf0 + 8 * (ti & acc_mask);
                uint32_t acc = 0u;
                for (int u = sg.u0; u < sg.u1; ++u) {
                    if (!TMAN_STAMPED_WAIT(wait_b, warp_all(mbar_wait(full0 + 8 * s, ph)))) { ok = false; break; }
                    tcgen05_fence_after();
                    const int xi = (u - sg.u0) & xu_mask;                  // unit of the activation stage
                    const bool xlast = xi == xu_mask || u == sg.u1 - 1;
                    const uint64_t bdesc = bdesc0 + (INT8 ? 1u : 2u) * ((xst << p.xu_sh) + (uint32_t)xi) * half_units;
                    const uint64_t adesc = adesc0 + xst * (2 * W_TILE_BYTES / 16);
                    const uint32_t wt = tmem_base + (uint32_t)p.wcol + (uint32_t)W_COLS * s;
                    if (lead) {
#pragma unroll
                        for (int j = 0; j < (INT8 ? UK / 32 : UK / 16); ++j) {
                            const uint64_t bd = bdesc + 2 * (j & 3) + (j >> 2) * half_units;
                            if constexpr (INT8) {
                                if constexpr (PAIR) tcgen05_mma2_i8_ts(acc_tmem, wt + 8 * j, bd, idesc, acc);
                                else tcgen05_mma_i8_ts(acc_tmem, wt + 8 * j, bd, idesc, acc);
                            } else if constexpr (V == kGemmLoadFull) {
                                const uint64_t ad = adesc + 2 * (j & 3) + (j >> 2) * (W_TILE_BYTES / 16);
                                if constexpr (PAIR) tcgen05_mma2_f16(acc_tmem, ad, bd, idesc, acc);
                                else tcgen05_mma_f16(acc_tmem, ad, bd, idesc, acc);
                            } else {
                                if constexpr (PAIR) tcgen05_mma2_f16_ts(acc_tmem, wt + 8 * j, bd, idesc, acc);
                                else tcgen05_mma_f16_ts(acc_tmem, wt + 8 * j, bd, idesc, acc);
                            }
                            acc = 1u;
                        }
                        if constexpr (PAIR) {
                            tcgen05_commit2_both(empty0 + 8 * s);
                            if (xlast) tcgen05_commit2_both(xempty0 + 8 * xst);
                        } else {
                            tcgen05_commit(empty0 + 8 * s);
                            if (xlast) tcgen05_commit(xempty0 + 8 * xst);
                        }
                    }
                    acc = 1u;
                    if (xlast) xst = (xst + 1u) & xst_mask;
                    if (++s == (uint32_t)wbufs) { s = 0; ph ^= 1u; }
                }
                if (ok && lead) {
                    if constexpr (PAIR) tcgen05_commit2_both(accf);
                    else tcgen05_commit(accf);
                }
                ++ti;
            }
        }
    } else if (warp < 2 + NUM_DEQ_WARPS) {
        // ---- stage 2: dequantization of this CTA's channels --------------------------------------------
        // lane = channel (a warp may only touch its quarter of the tensor-memory lanes); group grp takes every fourth unit of
        // the walk, four plane words of a channel per thread.  The 128-byte swizzle of the packed boxes (16-byte piece XOR
        // strip) puts the eight strips a warp reads on different banks.
        const int quad = warp & 3, grp = (warp - 2) >> 2;
        const int strip = quad * 8 + (lane >> 2), c = lane & 3;
        const int nblk = p.K / p.group;
        uint32_t p_src[4];                                 // the lane's plane words in the half of a packed stage its strip's swizzle puts first
#pragma unroll
        for (int w = 0; w < 4; ++w) p_src[w] = (uint32_t)strip * 128u + (uint32_t)c * 4u + ((uint32_t)(w ^ (strip & 3)) * 16u);
        const uint32_t half_swap = ((uint32_t)strip >> 2) & 1u;
        const uint32_t w_tmem = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)p.wcol, xst_mask = (1u << p.xst_sh) - 1u;
        // Weight buffer of the group's next unit and its parity.  A wait names a turn of its barrier by the parity alone and would also
        // pass while the turn before it is incomplete; a group does not wait for the loads of the units between its own, and these
        // may arrive in any order.  What it knows from the unit before, four back: the weight buffer of that one was free, so the
        // unit `wbufs` before it has been multiplied and every load up to there is complete.  The packed stages' "loaded" barriers
        // take turns over eight stages, also where the ring has four slots: seven stages lie between two turns of a barrier, at least
        // seven units, or, with six or eight buffers (tiles of four or eight units and more), eleven or thirteen, so that the turn
        // before is among those loads.  (Four slots with a barrier each: the stages of one unit that end odd tiles leave turns
        // unseen.)  So do the activations' on the integer path.  On the fp16 path a barrier per slot is enough: this unit's weight
        // buffer is waited for first, so every load up to the unit six (four) back is complete, and the slot's turn before is no later.
        uint32_t s = (uint32_t)grp, ph = 0u;
        uint32_t pos = 0, xc0 = 0, pc0 = 0;                // units, activation stages and packed stages of the segments before
        // BPU: quantization blocks of a unit
        auto walk = [&](auto bpu_c) {
            constexpr int BPU = decltype(bpu_c)::value;
            while (ok && span.next(sg)) {
                const int n = tile_ch0(sg.tile) + quad * 32 + lane;
                // (LoadFull: the first group alone passes every unit's activations and weights on)
                constexpr int STEP = V == kGemmLoadFull ? 1 : DEQ_GROUPS;
                const int first = V == kGemmLoadFull ? (grp == 0 ? sg.u0 : sg.u1) : sg.u0 + ((int)((uint32_t)grp - pos) & (DEQ_GROUPS - 1));
                const int units = sg.u1 - sg.u0;
                pos += (uint32_t)units;
                // scales and zero-points of a unit's blocks, fetched one turn ahead (channels past the last: of the last)
                const int strip_n = min(n, p.N - 1) >> 2;
                const __half *psc = p.scales + ((size_t)strip_n * nblk + (size_t)first * BPU) * 4 + c;
                const uint16_t *pz = p.zeros + (size_t)strip_n * nblk + (size_t)first * BPU;
                __half sv[BPU];
                uint32_t zv[BPU];
                auto fetch = [&]() {
#pragma unroll
                    for (int w = 0; w < BPU; ++w) {
                        sv[w] = __ldg(psc + 4 * w);
                        zv[w] = __ldg(pz + w);
                    }
                    psc += 4 * BPU * STEP;
                    pz += BPU * STEP;
                };
                if (!INT8 && first < sg.u1) fetch();
                for (int u = first; u < sg.u1; u += STEP) {
                    const uint32_t i = (uint32_t)(u - sg.u0), xc = xc0 + (i >> p.xu_sh);
                    const uint32_t xbar = xloaded0 + 8 * (INT8 ? xc % X_LOAD_BARS : xc & xst_mask), xpar = (INT8 ? xc / X_LOAD_BARS : xc >> p.xst_sh) & 1u;
                    if constexpr (V != kGemmLoadFull) {
                        BlockConsts t[BPU];
                        __half s_cur[BPU];
                        uint32_t z_cur[BPU];
#pragma unroll
                        for (int w = 0; w < BPU; ++w) {
                            if constexpr (INT8) continue;
                            s_cur[w] = sv[w];
                            z_cur[w] = (zv[w] >> (4 * c)) & 0xFu;
                            t[w].set(sv[w], z_cur[w]);
                        }
                        if (!INT8 && u + STEP < sg.u1) fetch();
                        const uint32_t pc = pc0 + (i >> 1), ps = pc % P_STAGES;
                        if (!TMAN_STAMPED_WAIT(wait_a, mbar_wait(ploaded0 + 8 * (pc % P_LOAD_BARS), (pc / P_LOAD_BARS) & 1u))) { ok = false; break; }
                        uint32_t w4[4][BITS];
                        const uint32_t stage = ps * P_STAGE_BYTES + (((i & 1u) ^ half_swap) << 6);
#pragma unroll
                        for (int w = 0; w < 4; ++w)
#pragma unroll
                            for (int b = 0; b < BITS; ++b)
                                w4[w][b] = *reinterpret_cast<const uint32_t *>(smem + p_src[w] + stage + b * P_PLANE_BYTES);
                        if (!TMAN_STAMPED_WAIT(wait_b, mbar_wait(empty0 + 8 * s, ph ^ 1u))) { ok = false; break; }
                        tcgen05_fence_after();
                        __syncwarp();
                        if (lane == 0) {                                       // the packed words are in registers
                            mbar_arrive(pempty0 + 8 * ps);
                            if ((i & 1u) == 0u && u == sg.u1 - 1) mbar_arrive(pempty0 + 8 * ps);   // a last stage of one unit
                        }
                        if constexpr (V == kGemmSequential)
                            if (!mbar_wait(xbar, xpar)) { ok = false; break; }
                        const uint32_t dst = w_tmem + (uint32_t)W_COLS * s;
                        if constexpr (INT8) {
#pragma unroll
                            for (int w = 0; w < 4; w += 2) {
                                uint32_t out[16];
                                dequant_word_int8(w4[w], out);
                                dequant_word_int8(w4[w + 1], out + 8);
                                tcgen05_st_32x32b_x16(dst + (uint32_t)(8 * w), out);
                            }
                        } else
#pragma unroll
                        for (int w = 0; w < 4; ++w) {
                            constexpr int WPB = 4 / BPU;
                            uint32_t out[16];
                            if constexpr (V == kGemmConvertDq) dequant_word_convert<BITS>(w4[w], s_cur[w / WPB], z_cur[w / WPB], out);
                            else dequant_word<BITS>(w4[w], t[w / WPB], out);
                            tcgen05_st_32x32b_x16(dst + (uint32_t)(16 * w), out);
                        }
                        tcgen05_wait_st();
                    }
                    tcgen05_fence_before();
                    // the MMA of this unit also reads this CTA's activations
                    if (!TMAN_STAMPED_WAIT(wait_b, mbar_wait(xbar, xpar))) { ok = false; break; }
                    __syncwarp();
                    if (lane == 0) arrive_lead(full_lead + 8 * s);
                    s += STEP;
                    if (s >= (uint32_t)wbufs) { s -= (uint32_t)wbufs; ph ^= 1u; }
                }
                xc0 += (uint32_t)(units + (1 << p.xu_sh) - 1) >> p.xu_sh;
                pc0 += (uint32_t)(units + 1) >> 1;
            }
        };
        if (INT8 || p.group == 128) walk(IntC<1>());
        else if (p.group == 64) walk(IntC<2>());
        else walk(IntC<4>());
    } else {
        // ---- epilogue: this CTA's channels of a segment's accumulators ---------------------------------
        // A warp has 32 channels (one per lane) x half of the tile's tokens.  Whole tiles: round to fp16; neighbouring lanes
        // exchange every other token, so that a lane stores two adjacent channels of one token (4 bytes; a warp's store
        // covers 64 bytes of two tokens).  Split tiles: a segment writes the fp32 accumulators that others sum to this CTA's
        // partial tile and raises the warp's flag (of a span: all of them; of even pieces: all but its own share of the tokens,
        // with a flag for each of the others).  Whoever sums waits for the flags of the same warp in the other workers, fetches
        // their rows at once by bulk copies into the activation ring, which is idle by then (the finishing segment is the last
        // of its worker's walk), and adds them to its own accumulators in worker order.  (Fetched by ordinary loads, a
        // trip to L2 for every few of them, the sum made a call of 300 x 3584 x 4608 in two pieces take 25.8 us and one of 128 x 18944 x
        // 3584 in five 31.6; this way 20.2 and 26.3.)
        const int quad = warp & 3;
        const int ew = warp - 2 - NUM_DEQ_WARPS, half = p.nt >> 1, h0 = (ew >> 2) * half;
        const uint32_t acc0_tmem = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)h0;
        const bool odd = (lane & 1) != 0;
        auto partial_of = [&](int cta) { return p.partial + (size_t)cta * (kPartialBytesPerCta / 4) + (size_t)(ew * half * 32); };
        auto warp_flag = [&](int cta) { return p.flags + (size_t)cta * NUM_EPI_WARPS + ew; };
        auto piece_flag = [&](int cta, int sender) { return p.piece_flags + ((size_t)cta * NUM_EPI_WARPS + ew) * kMaxSplit + sender; };
        // (the loads before it stay inside the buffers whatever the header says; a header that does not match stops the stores)
        const bool hdr_ok = header_matches(p.packed, p.K, p.N, p.bits, p.group);
        if (!hdr_ok && lane == 0 && blockIdx.x == 0) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_BAD_PACKED);
        uint32_t ti = 0;
        while (ok && span.next(sg)) {
            const int m0 = tile_tm(sg.tile) * p.nt + h0, n = tile_ch0(sg.tile) + quad * 32 + lane, left = min(half, p.M - m0);   // tokens to do (may be <= 0)
            __half *y = p.y + (size_t)m0 * p.N + (n & ~1);
            const bool put = n < p.N && hdr_ok;
            // sums of tokens t, t + 1 of this lane's channel -> two channels of one of the tokens
            auto store2 = [&](int t, int end, uint32_t v0, uint32_t v1, float sc = 0.f) {
                const uint32_t keep = odd ? v1 : v0, got = __shfl_xor_sync(0xffffffffu, odd ? v0 : v1, 1);
                const uint32_t c0 = odd ? got : keep, c1 = odd ? keep : got;
                __half2 h;
                if constexpr (INT8) h = __floats2half2_rn((float)(int)c0 * sc, (float)(int)c1 * sc);
                else h = __floats2half2_rn(__uint_as_float(c0), __uint_as_float(c1));
                const int tt = t + (odd ? 1 : 0);
                if (tt < end && put) *reinterpret_cast<__half2 *>(y + (size_t)tt * p.N) = h;
            };
            const uint32_t acc_b = ti & acc_mask;
            if (!TMAN_STAMPED_WAIT(wait_a, mbar_wait(accf0 + 8 * acc_b, (ti >> p.acc_sh) & 1u))) { ok = false; break; }
            tcgen05_fence_after();
            const uint32_t acc_tmem = acc0_tmem + (uint32_t)p.acc_col * acc_b;
            if (sg.whole) {
#pragma unroll 1
                for (int t = 0; t < left; t += 16) {
                    uint32_t r[16];
                    tcgen05_ld_32x32b_x16(acc_tmem + (uint32_t)t, r);
                    float sc[8];
                    if constexpr (INT8) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) sc[e] = ld_dependent(p.row_scale + min(m0 + t + 2 * e + (odd ? 1 : 0), p.M - 1)) * p.w_scale;
                    }
                    tcgen05_wait_ld();
#pragma unroll
                    for (int e = 0; e < 8; ++e) store2(t + 2 * e, left, r[2 * e], r[2 * e + 1], INT8 ? sc[e] : 0.f);
                }
            } else if constexpr (!INT8) {
                const int S = p.split_s, me = S ? worker % S : 0;
                // this worker's share of the sum
                const int own0 = S ? min(half * me / S, left) : 0, own1 = S ? min(half * (me + 1) / S, left) : sg.finishes ? left : 0;
                const int first_w = S ? worker - me : sg.finishes ? span.owner(sg.tile, 0) : worker;
                const int senders = S ? S : worker - first_w;              // workers from first_w on, this one among even pieces
                const bool other = lane < senders && first_w + lane != worker;
                if (S || !sg.finishes) {
                    float *mine = partial_of((int)blockIdx.x) + lane;
#pragma unroll 1
                    for (int t = 0; t < left; t += 8) {
                        uint32_t r[8];
                        tcgen05_ld_32x32b_x8(acc_tmem + (uint32_t)t, r);
                        tcgen05_wait_ld();
#pragma unroll
                        for (int e = 0; e < 8; ++e)
                            if ((t + e < own0 || t + e >= own1) && t + e < left) __stcg(mine + (t + e) * 32, __uint_as_float(r[e]));
                    }
                    __threadfence();                       // every lane's stores, then the flags
                    __syncwarp();
                    uint32_t *to = S ? piece_flag((first_w + lane) * NCTA + (int)rank, me) : warp_flag((int)blockIdx.x);
                    if (S ? other : lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(to), "r"(1u) : "memory");
                }
                if (senders > 0) {
                    uint32_t *from = S ? piece_flag((int)blockIdx.x, lane) : warp_flag((first_w + lane) * NCTA + (int)rank);
                    uint64_t t0 = 0;
                    for (uint32_t spin = 0; other; ++spin) {
                        uint32_t fv;
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(fv) : "l"(from) : "memory");
                        if (fv == 1u) break;
                        if ((spin & 255u) == 255u) {
                            const uint64_t now = global_timer_ns();
                            if (t0 == 0) t0 = now;
                            else if (now - t0 > 1000000000ull) { ok = false; break; }
                        }
                    }
                    ok = warp_all(ok);
                    if (!ok) break;
                    if (other) *from = kFlagEmpty;         // back to "empty" for the next launch
                    asm volatile("fence.proxy.async;" ::: "memory");       // the others' stores, then the copies that read them
                    const int slots = S ? S - 1 : senders, step = 128 / slots;            // 16 KB a warp: so many tokens of every sender at a time
                    const float *src = partial_of((first_w + lane) * NCTA + (int)rank);
                    const uint32_t bar = sums0 + 8 * ew, slot_off = (uint32_t)ew * 16384u;
                    uint32_t par = 0;
#pragma unroll 1
                    for (int t0 = own0; t0 < own1; t0 += step) {
                        const int cnt = min(step, own1 - t0);
                        if (lane == 0) mbar_expect_tx(bar, (uint32_t)(slots * cnt) * 128u);
                        __syncwarp();
                        if (other)
                            bulk_load(smem_u32(x_tiles) + slot_off + (uint32_t)((lane - (S && lane > me ? 1 : 0)) * cnt) * 128u, src + t0 * 32, (uint32_t)cnt * 128u, bar);
                        ok = warp_all(mbar_wait(bar, par) || mbar_wait(bar, par));
                        if (!ok) break;
                        par ^= 1u;
#pragma unroll 1
                        for (int t = 0; t < cnt; t += 8) {
                            uint32_t r[8];
                            tcgen05_ld_32x32b_x8(acc_tmem + (uint32_t)(t0 + t), r);
                            tcgen05_wait_ld();
                            const float *rows = reinterpret_cast<const float *>(x_tiles + slot_off) + t * 32 + lane;
#pragma unroll 1
                            for (int o = 0; o < slots; ++o, rows += cnt * 32)
#pragma unroll
                                for (int e = 0; e < 8; ++e)
                                    if (t + e < cnt) r[e] = __float_as_uint(__uint_as_float(r[e]) + rows[e * 32]);
#pragma unroll
                            for (int e = 0; e < 8; e += 2) store2(t0 + t + e, t0 + cnt, r[e], r[e + 1]);
                        }
                        __syncwarp();
                    }
                }
            }
            // the accumulators are read: the next segment's MMAs may start
            tcgen05_fence_before();
            __syncwarp();
            if (lane == 0) arrive_lead(acce_lead + 8 * acc_b);
            ++ti;
        }
    }

    if (!ok) atomicCAS(p.status, 0u, (uint32_t)TMAN_ERR_TIMEOUT);
    tcgen05_fence_before();
#ifdef TMAN_ROLE_STAMPS
    if (lane == 0 && p.stamps != nullptr && run) {
        long long *st = p.stamps + ((size_t)blockIdx.x * kGemmWarps + warp) * kStampWordsPerWarp;
        st[0] = wait_a;
        st[1] = wait_b;
        st[2] = clock64() - role_t0;
        st[3] = 0x5354414D50ll;                        // "STAMP": this build writes time stamps
    }
#else
    (void)wait_a; (void)wait_b;
#endif
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();            // nobody touches the peer's memory after this
    if (warp == 1 && tmem_base != 0xFFFFFFFFu) {
        tcgen05_fence_after();
        if constexpr (PAIR) tcgen05_dealloc2(tmem_base, TMEM_COLS);
        else tcgen05_dealloc(tmem_base, TMEM_COLS);
    }
}

// ---- host side ---------------------------------------------------------------------------
// How a call's work is cut (host).  Pairs of CTAs beyond 16 tokens: a pair fetches an activation once per 256 channels and is
// as fast or faster at the sizes measured (4-bit, group 128: 40 x 4096 x 14336 18.1 us either way, 128 x 3584 x 18944 19.9
// against 21.8 with single CTAs, 128 x 18944 x 3584 26.4 / 28.6; 2-bit, 128 x 3584 x 4608 16.0 / 15.8); up to 16 tokens a single CTA
// needs half the columns.  The tokens go to as few tiles of at most 256 as hold them, or a few more where that deals out better;
// a unit takes 0.39 us up to 128 tokens (the dequantization bounds it) and follows the MMA above (0.72 at 256).  Where whole
// tiles leave workers idle the units are split: in equal spans over the last tiles, or, for few tiles, in even pieces; a
// split costs 4 to 6 us for the partial sums, written, announced and read back (40 x 4096 x 14336: 56 whole tiles 18.7 us, spans
// on 74 workers 21.5; 128 x 18944 x 3584 whole on 14 workers about 70, in five pieces 26.4).
struct GemmPlan { int pair, nt, tiles_m, tiles_n, span_tiles, workers, col_fastest, split_s; };

inline bool gemm_pair(int M) { return M > 16; }

// `resident`: how many workers (CTAs, or CTA pairs) of the chosen kernel the device can hold at the
// same time.  Workers wait for one another's partial tiles, so no more than that may be launched.
GemmPlan plan_gemm(int M, int K, int N, int bits, int sms, int resident)
{
    GemmPlan g = {};
    const bool pair = gemm_pair(M);
    g.pair = pair ? 1 : 0;
    const int ncta = pair ? 2 : 1, gran = pair ? 32 : 16;
    const long long all = (sms < kMaxGemmCtas ? sms : kMaxGemmCtas) / ncta > 0 ? (sms < kMaxGemmCtas ? sms : kMaxGemmCtas) / ncta : 1;
    long long workers = all < resident ? all : resident;
    if (workers < 1) workers = 1;
    const long long nu = K / UK;
    g.tiles_n = (N + CH * ncta - 1) / (CH * ncta);
    const bool may_split = nu * 2 * all * all < (1ll << 30);        // the spans' arithmetic is 32-bit
    // least time with tm tiles of tokens and w workers; fills in g
    auto cut = [&](int tm, long long w) {
        const int nt = ((M + tm - 1) / tm + gran - 1) / gran * gran, tiles_m = (M + nt - 1) / nt;
        const long long tiles = (long long)tiles_m * g.tiles_n;
        const double lo = 0.40 + 0.0002 * nt, hi = 0.0028 * nt, unit = lo > hi ? lo : hi, fix = 1.2 + 0.007 * nt, sums = 3.5 + 0.012 * nt;
        double best = (double)((tiles + w - 1) / w) * (nu * unit + fix);
        g.nt = nt; g.tiles_m = tiles_m; g.span_tiles = 0; g.split_s = 0;
        auto take = [&](double cost, long long span, int split) {
            if (cost < best - 1e-9) { best = cost; g.span_tiles = (int)span; g.split_s = split; }
        };
        if (!may_split) return best;
        // the remainder of the last round is cut into spans, together with one whole round when the remainder alone
        // would be cut into many pieces per tile
        const long long rest = tiles % w, span = (rest != 0 && rest < w / 2 && tiles > w) ? rest + w : rest;
        if (span != 0 && 2 * tiles > w)                // (fewer tiles: even pieces, at most one tile a worker)
            take((double)((tiles - span) / w) * (nu * unit + fix) + (double)((span * nu + w - 1) / w) * unit + fix + sums, span, 0);
        for (int S = 2; S <= kMaxSplit && tiles * S <= w && nu >= 2 * S; ++S)
            take((double)((nu + S - 1) / S) * unit + fix + sums + 0.8 * (S - 2), tiles, S);
        return best;
    };
    int tm_best = (M + MAX_TOKENS - 1) / MAX_TOKENS;
    double us = 1e300;
    for (int tm = tm_best, end = tm_best + 4; tm <= end; ++tm) {
        const double t = cut(tm, all);
        if (t < us - 1e-9 && (long long)g.tiles_m * g.tiles_n < (1ll << 31)) { us = t; tm_best = tm; }
    }
    cut(tm_best, workers);
    const long long tiles = (long long)g.tiles_m * g.tiles_n;
    if (g.split_s) workers = tiles * g.split_s;
    else if (tiles < workers) {                        // fewer tiles than workers: as many workers as units at most
        const long long units = g.span_tiles ? tiles * nu : tiles;
        if (workers > units) workers = units;
    }
    g.workers = (int)workers;
    // tile numbering: bytes a round of `workers` consecutive tiles touches, either way
    {
        const double a_tile = (double)g.nt * K * 2.0, b_tile = (double)CH * ncta * K * bits / 8.0;
        const long long rows_r = g.tiles_m < workers ? g.tiles_m : workers, cols_r = (workers + g.tiles_m - 1) / g.tiles_m;
        const long long cols_c = g.tiles_n < workers ? g.tiles_n : workers, rows_c = (workers + g.tiles_n - 1) / g.tiles_n;
        g.col_fastest = (rows_c * a_tile + cols_c * b_tile < rows_r * a_tile + cols_r * b_tile) ? 1 : 0;
    }
    return g;
}

// the bit-plane words as a 3-D array of 32-bit elements: (word and column inside a strip's plane row, plane, strip); one
// box = the eight words of two units for the strips of a CTA's channels, one plane
bool planes_map(EncodeTiledFn enc, CUtensorMap *map, const uint8_t *packed, int K, int N, int bits, int group)
{
    const cuuint64_t wt = (cuuint64_t)(K / 32);
    const cuuint64_t dims[3] = {wt * 4, (cuuint64_t)bits, (cuuint64_t)(N / 4)};
    const cuuint64_t strides[2] = {wt * 16, wt * 16 * (cuuint64_t)bits};
    const cuuint32_t box[3] = {(cuuint32_t)(2 * UK / 8), 1, (cuuint32_t)(CH / 4)};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<uint8_t *>(packed + make_layout(K, N, bits, group).planes_off), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BITS, bool PAIR, int V>
cudaLaunchConfig_t gemm_config(int ctas, cudaLaunchAttribute (&attr)[2], cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(GEMM_THREADS);
    cfg.dynamicSmemBytes = GEMM_SMEM;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = PAIR ? 2 : 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

template <int BITS, bool PAIR, int V>
tman_status launch_cfg(const CUtensorMap &tmap_x, const CUtensorMap &tmap_w, const CUtensorMap &tmap_wf, const GemmParams &p, int workers,
                       cudaStream_t s)
{
    auto kern = mpgemm_kernel<BITS, PAIR, V>;
    static std::atomic<bool> raised[kMaxDevices];
    int dev = 0;
    if (!device_info(&dev)) return TMAN_ERR_CUDA;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = gemm_config<BITS, PAIR, V>(workers * (PAIR ? 2 : 1), attr, s);
    return launch_with_smem(kern, GEMM_SMEM, dev, raised, [&] { return cudaLaunchKernelEx(&cfg, kern, tmap_x, tmap_w, tmap_wf, p); });
}

template <int BITS, int V>
tman_status launch_bits(const CUtensorMap &tmap_x, const CUtensorMap &tmap_w, const CUtensorMap &tmap_wf, const GemmParams &p, const GemmPlan &g,
                        cudaStream_t s)
{
    if (g.pair) return launch_cfg<BITS, true, V>(tmap_x, tmap_w, tmap_wf, p, g.workers, s);
    return launch_cfg<BITS, false, V>(tmap_x, tmap_w, tmap_wf, p, g.workers, s);
}

// Workers of one kernel variant that can be resident together on the current device (occupancy query,
// once per device and variant).
template <int BITS, bool PAIR>
int resident_cfg(int sms)
{
    auto kern = mpgemm_kernel<BITS, PAIR, kGemmProduct>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM) != cudaSuccess) return -1;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = gemm_config<BITS, PAIR, kGemmProduct>(sms / (PAIR ? 2 : 1) * (PAIR ? 2 : 1), attr, nullptr);
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) return -1;
    return n;
}

int resident_workers(int M, int bits, int sms)
{
    static std::mutex lock;
    static int cache[kMaxDevices][3][2];     // [device][bits - 2][pair], 0 = not asked yet
    int dev = 0;
    if (!device_info(&dev) || bits < 2 || bits > 4) return -1;
    const int pair = gemm_pair(M) ? 1 : 0;
    std::lock_guard<std::mutex> guard(lock);
    int &slot = cache[dev][bits - 2][pair];
    if (slot == 0) {
        int n = -1;
        if (bits == 2) n = pair ? resident_cfg<2, true>(sms) : resident_cfg<2, false>(sms);
        if (bits == 3) n = pair ? resident_cfg<3, true>(sms) : resident_cfg<3, false>(sms);
        if (bits == 4) n = pair ? resident_cfg<4, true>(sms) : resident_cfg<4, false>(sms);
        if (n < 1) return -1;                 // not cached: asked again next time
        slot = n;
    }
    return slot;
}

}  // namespace

tman_status mpgemm_plan_for(int M, int K, int N, int bits, int sms, int resident, int *out8)
{
    const GemmPlan g = plan_gemm(M, K, N, bits, sms, resident);
    out8[0] = g.pair; out8[1] = (g.nt + 127) / 128; out8[2] = g.tiles_m; out8[3] = g.tiles_n; out8[4] = g.span_tiles ? 0 : 1; out8[5] = g.workers;
    out8[6] = g.split_s ? 0 : g.span_tiles; out8[7] = g.split_s;
    return TMAN_OK;
}

tman_status mpgemm_plan(int M, int K, int N, int bits, int *out8)
{
    const int sms = sm_count();
    if (sms <= 0) return TMAN_ERR_CUDA;
    const int resident = resident_workers(M, bits, sms);
    if (resident < 1) return TMAN_ERR_CUDA;
    return mpgemm_plan_for(M, K, N, bits, sms, resident, out8);
}

size_t mpgemm_workspace_bytes(int M, int, int)
{
    (void)M;
    return kGemmPartialOff + (size_t)kMaxGemmCtas * (kPartialBytesPerCta + kStampBytesPerCta);
}

// Copies the role time stamps of the last prefill call out of the workspace (host buffer of
// ctas x 26 warps x 4 words).  Only a library built with TMAN_ROLE_STAMPS writes them.
tman_status mpgemm_read_stamps(const void *ws, int ctas, long long *out_host, cudaStream_t s)
{
#ifdef TMAN_ROLE_STAMPS
    if (ctas < 1 || ctas > kMaxGemmCtas) return TMAN_ERR_SHAPE;
    const uint8_t *src = static_cast<const uint8_t *>(ws) + kGemmPartialOff + (size_t)kMaxGemmCtas * kPartialBytesPerCta;
    if (cudaMemcpyAsync(out_host, src, (size_t)ctas * kStampBytesPerCta, cudaMemcpyDeviceToHost, s) != cudaSuccess) return TMAN_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return TMAN_ERR_CUDA;
    return TMAN_OK;
#else
    (void)ws; (void)ctas; (void)out_host; (void)s;
    return TMAN_ERR_UNSUPPORTED;
#endif
}

tman_status launch_mpgemm(const void *packed, const void *x, void *y, int M, int K, int N, int bits,
                          int group, void *ws, size_t ws_bytes, cudaStream_t s)
{
    return launch_mpgemm_variant(kGemmProduct, packed, x, y, M, K, N, bits, group, nullptr, ws, ws_bytes, s);
}

// variant: one of kGemmProduct .. kGemmSequential; wt_f16: for kGemmLoadFull the dequantized weights as fp16
// [N][K] (channel-major), otherwise unused.  The variants other than the product path exist for 4-bit only.
tman_status launch_mpgemm_variant(int variant, const void *packed, const void *x, void *y, int M, int K, int N, int bits,
                                  int group, const void *wt_f16, void *ws, size_t, cudaStream_t s)
{
    if (variant < kGemmProduct || variant > kGemmSequential) return TMAN_ERR_UNSUPPORTED;
    if (variant != kGemmProduct && bits != 4) return TMAN_ERR_UNSUPPORTED;
    if (variant == kGemmLoadFull && (!wt_f16 || (reinterpret_cast<uintptr_t>(wt_f16) & 15) != 0)) return TMAN_ERR_SHAPE;
    if (variant == kGemmLoadFull && (N % 32) != 0) return TMAN_ERR_UNSUPPORTED;     // whole 32-channel units only
    if ((reinterpret_cast<uintptr_t>(x) & 15) != 0 || (reinterpret_cast<uintptr_t>(y) & 15) != 0) return TMAN_ERR_SHAPE;
    EncodeTiledFn enc = encode_fn();
    if (!enc) return TMAN_ERR_CUDA;
    const int sms = sm_count();
    if (sms <= 0) return TMAN_ERR_CUDA;
    const int resident = resident_workers(M, bits, sms);
    if (resident < 1) return TMAN_ERR_CUDA;
    const GemmPlan g = plan_gemm(M, K, N, bits, sms, resident);
    const int rows_cta = g.nt / (g.pair ? 2 : 1);
    const cuuint32_t estr[3] = {1, 1, 1};

    const bool one_unit = variant == kGemmLoadFull || variant == kGemmSequential || rows_cta > 64;
    const int p_xu_sh = one_unit ? 0 : 1;
    // activations as [k-block][token][64 k]: boxes of one or two units x a CTA's token rows, 128-byte swizzle
    CUtensorMap tmap_x;
    {
        const cuuint64_t dims[3] = {(cuuint64_t)BK, (cuuint64_t)M, (cuuint64_t)(K / BK)};
        const cuuint64_t strides[2] = {(cuuint64_t)K * 2, (cuuint64_t)BK * 2};
        const cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)rows_cta, (cuuint32_t)(UK / BK << p_xu_sh)};
        if (enc(&tmap_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<void *>(x), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return TMAN_ERR_CUDA;
    }
    Layout L = make_layout(K, N, bits, group);
    const uint8_t *pk = static_cast<const uint8_t *>(packed);
    CUtensorMap tmap_w;
    if (!planes_map(enc, &tmap_w, pk, K, N, bits, group)) return TMAN_ERR_CUDA;

    uint8_t *w8 = static_cast<uint8_t *>(ws);
    GemmParams p;
    p.packed = pk;
    p.scales = reinterpret_cast<const __half *>(pk + L.scales_off);
    p.zeros = reinterpret_cast<const uint16_t *>(pk + L.zeros_off);
    p.y = static_cast<__half *>(y);
    p.status = reinterpret_cast<uint32_t *>(w8);
    p.flags = reinterpret_cast<uint32_t *>(w8 + kGemmFlagsOff);
    p.piece_flags = reinterpret_cast<uint32_t *>(w8 + kGemmPieceFlagsOff);
    p.partial = reinterpret_cast<float *>(w8 + kGemmPartialOff);
    p.M = M; p.K = K; p.N = N; p.bits = bits; p.group = group;
    p.nt = g.nt;
    // Tensor memory: behind an accumulator of up to 128 columns there is room for six weight buffers, behind 256 for four.
    // (LoadFull: two activation stages, with their weight tiles in the packed ring beside them.)
    const bool six = g.nt <= 128 && K >= 4 * UK && variant == kGemmProduct;
    p.wbufs = variant == kGemmLoadFull ? 2 : six ? 6 : 4;
    p.wcol = g.nt <= 128 ? 128 : 256;
    p.xu_sh = p_xu_sh;
    p.xst_sh = variant == kGemmLoadFull ? 1 : 3;
    while ((rows_cta * 256 << p.xu_sh << p.xst_sh) > X_RING_BYTES) --p.xst_sh;
    p.tiles_m = g.tiles_m;
    p.tiles_n = g.tiles_n;
    p.span_tiles = g.span_tiles;
    p.split_s = g.split_s;
    p.acc_sh = 0; p.acc_col = 0;
    p.row_scale = nullptr; p.w_scale = 0.f;
    p.col_fastest = g.col_fastest;
    p.stamps = reinterpret_cast<long long *>(w8 + kGemmPartialOff + (size_t)kMaxGemmCtas * kPartialBytesPerCta);
    // the fp16 weights [N][K]: boxes of half a unit x a CTA's channels, 128-byte swizzle; unused maps are copies of the activation map
    CUtensorMap tmap_wf = tmap_x;
    if (variant == kGemmLoadFull) {
        const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)N};
        const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
        const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)CH};
        if (enc(&tmap_wf, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(wt_f16), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return TMAN_ERR_CUDA;
    }
    if (bits == 2) return launch_bits<2, kGemmProduct>(tmap_x, tmap_w, tmap_wf, p, g, s);
    if (bits == 3) return launch_bits<3, kGemmProduct>(tmap_x, tmap_w, tmap_wf, p, g, s);
    if (variant == kGemmConvertDq) return launch_bits<4, kGemmConvertDq>(tmap_x, tmap_w, tmap_wf, p, g, s);
    if (variant == kGemmLoadFull) return launch_bits<4, kGemmLoadFull>(tmap_x, tmap_w, tmap_wf, p, g, s);
    if (variant == kGemmSequential) return launch_bits<4, kGemmSequential>(tmap_x, tmap_w, tmap_wf, p, g, s);
    return launch_bits<4, kGemmProduct>(tmap_x, tmap_w, tmap_wf, p, g, s);
}

// Integer path: ternary weights times 8-bit integer activations, y = fp16( row_scale[m] * w_scale * sum ).  Whole tiles only (the
// call has no workspace for partial sums).  Tiles of up to 192 tokens leave room for two accumulators, so that a tile's
// epilogue hides behind the next tile; 256 for one, whose epilogue does not.  A unit takes at least 0.2 us, whatever its
// tokens, in issuing its MMAs and commits (the multiplications themselves: 0.2 us at 192), which bounds most sizes.  Measured at
// 128 / 160 / 192 / 256 tokens a tile: 2048 x 2560 x 6912 41.0 / 36.2 / 35.4 / 39.5 us, 4096 x 6912 x 2560 74.3 / 62.1 / 50.9 / 65.3.
// (Weights through shared memory in tiles of 128 tokens x 256 channels of one CTA, one row of dequantization warps: 44.3 and 97.1.)
tman_status launch_mpgemm_ternary_i8(const void *packed, const int8_t *a8, const float *row_scale, float w_scale, void *y,
                                     int M, int K, int N, int group, void *ws, cudaStream_t s)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return TMAN_ERR_CUDA;
    const int sms = sm_count();
    if (sms <= 0) return TMAN_ERR_CUDA;
    GemmPlan g = {};
    g.pair = gemm_pair(M) ? 1 : 0;
    const int ncta = g.pair ? 2 : 1, gran = g.pair ? 32 : 16, workers = sms / ncta > 0 ? sms / ncta : 1;
    g.tiles_n = (N + CH * ncta - 1) / (CH * ncta);
    // least modelled time: rounds of tiles x (units of 128 k, and the epilogue where it does not hide behind them)
    double best = 1e300;
    for (int nt = gran; nt <= MAX_TOKENS; nt += gran) {
        const long long tiles = (long long)((M + nt - 1) / nt) * g.tiles_n, rounds = (tiles + workers - 1) / workers;
        const double unit_us = nt > 192 ? 0.00105 * nt : 0.2, tile_us = unit_us * (K / UK), epi_us = 0.4 + 0.008 * nt;
        const double us = nt > 192 ? rounds * (tile_us + epi_us) : rounds * (tile_us > epi_us ? tile_us : epi_us) + epi_us;
        if (us < best) { best = us; g.nt = nt; }
    }
    g.tiles_m = (M + g.nt - 1) / g.nt;
    const long long tiles = (long long)g.tiles_m * g.tiles_n;
    if (tiles >= (1ll << 31)) return TMAN_ERR_SHAPE;
    g.workers = (int)(tiles < workers ? tiles : workers);
    GemmParams p = {};
    p.M = M; p.K = K; p.N = N; p.bits = 2; p.group = group;
    p.nt = g.nt; p.tiles_m = g.tiles_m; p.tiles_n = g.tiles_n;
    p.packed = static_cast<const uint8_t *>(packed);
    p.y = static_cast<__half *>(y);
    p.status = static_cast<uint32_t *>(ws);
    p.row_scale = row_scale;
    p.w_scale = w_scale;
    const int rows_cta = g.nt / ncta;
    p.acc_sh = g.nt <= 192 ? 1 : 0;
    p.wcol = g.nt <= 128 ? 256 : g.nt <= 192 ? 384 : 256;
    p.wbufs = K >= 8 * UK && (g.nt <= 128 || g.nt > 192) ? 8 : 4;
    p.acc_col = g.nt <= 128 ? 128 : 192;
    p.xu_sh = 1;
    p.xst_sh = 3;
    while ((rows_cta * UK << p.xu_sh << p.xst_sh) > X_RING_BYTES) --p.xst_sh;
    const cuuint32_t estr[3] = {1, 1, 1};
    CUtensorMap tmap_x;
    {
        const cuuint64_t dims[3] = {(cuuint64_t)UK, (cuuint64_t)M, (cuuint64_t)(K / UK)};
        const cuuint64_t strides[2] = {(cuuint64_t)K, (cuuint64_t)UK};
        const cuuint32_t box[3] = {(cuuint32_t)UK, (cuuint32_t)rows_cta, (cuuint32_t)(1 << p.xu_sh)};
        if (enc(&tmap_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<int8_t *>(a8), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return TMAN_ERR_CUDA;
    }
    CUtensorMap tmap_w;
    if (!planes_map(enc, &tmap_w, p.packed, K, N, 2, group)) return TMAN_ERR_CUDA;
    return launch_bits<2, kGemmInt8>(tmap_x, tmap_w, tmap_x, p, g, s);
}

}  // namespace tman
