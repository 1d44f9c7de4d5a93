// Verification attention with fused visual mass: TMA + tcgen05 kernel (D = 128 or 64).
//
// One CTA owns one KV split of one (sequence, KV head) and the M = gamma * G
// query rows that read this head.  The GQA-grouped queries are the small side
// of the problem, so the products are taken transposed: per tile of 128 cache
// positions
//     S^T[pos, n] = K_tile[pos, :] . Q[n, :]          (MMA M = 128 positions, N = rows)
//     O^T[d, n]  += V_tile[:, d]^T . P^T[:, n]        (MMA M = 128 channels,  N = rows)
//     L[0..1, n] += [1; in_span]   . P^T[:, n]        (MMA M = 64: row 0 = l, row 1 = l_vis)
// so every TMEM lane of S^T is one cache position (all softmax threads do
// useful exponentials) and the padded dimension is N (granularity 16), not M.
// The softmax denominators l and the visual-span numerators l_vis come out of
// the tensor core as two extra accumulator rows fed by a constant 0/1 tile.
//
// The reference exponent m[n] of a row is the score of the first position of
// the split and stays fixed while scores stay within 2^60 of it; only when a
// score runs past that guard is the tile's maximum taken (a cross-lane
// reduction in this layout) and the accumulators rescaled.  fp32 and bf16
// share the exponent range, so nothing is lost in between.
//
// Warp roles (480 threads): warp 0 = TMA producer, warp 1 = issuer of the
// K.Q^T MMAs and TMEM owner, warp 14 = issuer of the P.V and sum MMAs (one
// thread each; two issuers because a single thread's issue rate, not the tensor
// pipe, bounded the loop), warps 2-13 = three softmax groups of four warps.
// The softmax stage has two organisations.  With a bf16 cache all three groups work on
// every tile, each on a third of the columns (a thread is one cache position, TMEM lane
// quarter = warp % 4).  Up to 80 rows tiles go through in pairs where the stream is long: one
// vote on the guard, one fence and one hand-over to the P.V issuer for 256 positions, while the
// products of the pair before and the K.Q^T of the next run beside.  (Handed over one by one, a
// tile costs about 2.1 k cycles of which the exponentials are 0.4 k; in pairs a long stream is
// bound by HBM at 80 rows too: 128K positions x 4, 331 us a layer against 347.  Where the
// line lies, and the other side of it: pick_config.)
// With an fp8 cache the groups take the tiles in turn (tile i belongs to
// group i % 3, a thread works through all N columns of its tile), so the latencies of one
// tile hide behind the exponentials of the two tiles the other groups are
// on; S^T has a TMEM buffer per tile in flight.  The reference exponents m[] are
// shared.  Tiles are handed to the P.V issuer strictly in order, through a
// counter of committed tiles: a group may move m (and rescale the accumulators)
// only while its tile is the oldest uncommitted one, and announces the move in an
// epoch counter; a group whose turn comes compares the epoch with the one it read
// m under and computes its tile once more if m has moved meanwhile.
// K and V tiles sit in separate shared-memory rings,
// each slot two 128-position x 64-channel boxes with the 128-byte swizzle; Q
// arrives by TMA in the same layout.  Every mbarrier wait is bounded; a wait
// that gives up raises LVSPEC_DEV_WAIT_EXPIRED.
//
// fp8 cache (kFp8): K and V are E4M3 codes with one scale per (sequence, KV head), half
// the bytes per position.  An MMA takes both operands in one kind, so the 8-bit tiles
// are multiplied as they are (kind::f8f6f4, K = 32 per instruction) and the bf16
// side is brought to them without losing its bits: a value is split into the E4M3
// number holding its leading four significant bits and the E4M3 number nearest to the
// rest (the next four), both exact for bf16 inputs in the normal range.  Q (scaled by a
// power of two so that its largest magnitude sits below 256) is split once per CTA into
// two operand tiles, and K.Q^T takes both in one accumulation (8 MMAs of K = 32 over the
// 2 x 128 channels); a probability is split by the softmax threads, head and rest sit
// in neighbouring columns of P^T, and V^T.P^T and the sum products run with N = 2 x
// rows: accumulator column 2n holds the head's part of row n, column 2n + 1 the rest's,
// added once in the epilogue.  Probabilities are kept within E4M3's range by the
// reference exponent: the largest score of the split's first tile gets probability 2^3,
// and a later score that would pass 2^8 moves the reference up.  The K scale folds into the
// softmax scale, the V scale into the epilogue.
//
// head_dim 64: one 64-channel box per K or V tile and four K.Q^T steps; the P.V product
// keeps its 128 rows, of which the upper 64 read what follows the box in shared memory
// and fill TMEM lanes nobody reads.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdio>
#include <cstdlib>
#include <type_traits>

#include "lvspec_internal.h"
#include "sm100_ptx.cuh"

#ifdef LVSPEC_TRACE
cudaError_t lvspec::trace_set_buffer_attention(unsigned long long *device_words)
{
    return cudaMemcpyToSymbol(g_lvspec_trace, &device_words, sizeof device_words);
}
#endif

namespace lvspec {
namespace {

using namespace ptx;

constexpr int kTilePos = 128;
constexpr int kSoftmaxGroups = 3;           // groups of 4 warps, each on its own share of the columns
constexpr int kSoftmaxWarp0 = 2;            // first softmax warp
constexpr int kSoftmaxWarps = 4 * kSoftmaxGroups;
constexpr int kSoftmaxThreads = 32 * kSoftmaxWarps;
constexpr int kPvWarp = kSoftmaxWarp0 + kSoftmaxWarps;   // issues the P.V and sum MMAs
constexpr int kThreads = 32 * (kPvWarp + 1);
constexpr int kMaxChunks = (LVSPEC_MAX_ROWS / 8 + kSoftmaxGroups - 1) / kSoftmaxGroups;   // per group that shares the columns
constexpr uint32_t kBoxBytes = 16384;       // 128 positions x 64 channels bf16, or x 128 channels E4M3
constexpr uint32_t kSlotBytes = 2 * kBoxBytes;   // a bf16 tile; an fp8 tile is one box
constexpr uint32_t kA2Bytes = 2048;         // one 64 x 16 (bf16) or 64 x 32 (E4M3) constant tile
constexpr float kGuard = 60.f;              // log2 units above m before a rescale
constexpr uint32_t kGuardBits = (127u + 60u) << 7;     // 2^kGuard as bf16 bits
constexpr float kGuard8 = 8.f;              // fp8 cache: probabilities stay below 2^8 (E4M3 ends at 448)
constexpr float kHead8 = 3.f;               // fp8 cache: the largest score of a row in the split's first tile has probability 2^3
constexpr float kMFloor = -1.0e30f;
constexpr int kQBarrier = 1 + kSoftmaxGroups;   // named barrier over all softmax threads
constexpr int kHand = 4;                   // barriers of each hand-over kind
constexpr int kMaxRowsFp8 = 80;             // fp8 cache: 6 accumulator columns per padded row in 512

struct TcConfig {
    int n_pad;   // MMA N: rows padded to a multiple of 16
    int ks, vs, pb;   // K slots, V slots, P buffers
    int sb;           // S^T buffers in TMEM (2 to 4)
    int step;         // tiles handed over at a time (all groups on every tile: 2 where the buffers allow)
    int pair_from;    // ... in a CTA of at least so many tiles; else one by one
    int tmem_cols;
    uint32_t split_magic, group_magic;   // for divisions by n_split and G
    int page_slots;   // paged cache: pool pages of this split's tiles, one entry per tile
    int slot_bytes;   // one K or V tile: 32 KB bf16, 16 KB fp8
};

// Byte offsets of the shared-memory regions (relative to a 1024-aligned base).
struct SmemMap {
    uint32_t k, v, q, p, a2, m, dl, tmx, bars, misc, pages, total;
};
inline SmemMap smem_map(const TcConfig &c)
{
    SmemMap s;
    uint32_t o = 0;
    s.k = o;    o += c.ks * c.slot_bytes;
    s.v = o;    o += c.vs * c.slot_bytes;
    s.q = o;    o += c.n_pad * 256;
    s.p = o;    o += c.pb * c.n_pad * 256;
    s.a2 = o;   o += 4 * kA2Bytes;
    s.m = o;    o += c.n_pad * 4;
    s.dl = o;   o += c.n_pad * 4;
    s.tmx = o;  o += 4 * c.n_pad * 4;
    s.bars = o; o += 8 * (2 * c.ks + 2 * c.vs + 4 * kHand + 4);
    s.misc = o; o += 16 + 4 * kSoftmaxWarps + 16;     // TMEM address, abort flag, epoch of m, committed tiles, per-warp maxima of |q|, arrival counted, exchange buffer in doubt
    s.pages = o; o += 4 * c.page_slots;
    s.total = o;
    return s;
}

struct TcParams {
    TcConfig cfg;
    SmemMap sm;     // worked out on the host: in the kernel it was thirty instructions of the cold start
    AttnParams a;
};

// x / d with m = ceil(2^32 / d) from the host (0 for d = 1): the product is off by one at most for
// x < 2^31.  A plain division is a hundred instructions on a cold instruction cache.
uint32_t magic_of(uint32_t d) { return d > 1 ? 0xFFFFFFFFu / d + 1u : 0u; }
__device__ __forceinline__ int div_by(int x, int d, uint32_t m)
{
    if (m == 0u) return x;
    const int q = (int)__umulhi((uint32_t)x, m);
    return q * d > x ? q - 1 : q;
}

// Position in a ring of n slots and the parity of the round: the per-tile loops count
// instead of dividing.
struct Ring {
    int idx, n;
    uint32_t parity;
    __device__ __forceinline__ Ring(int n_) : idx(0), n(n_), parity(0) {}
    __device__ __forceinline__ void next()
    {
        if (++idx == n) {
            idx = 0;
            parity ^= 1u;
        }
    }
};

__device__ __forceinline__ bool wait_unconditional(uint32_t bar, uint32_t parity)
{
    // used while tearing down: time-bounded, ignores the abort flag
    const uint64_t t0 = global_timer_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_timer_ns() - t0 > 1000000000ull) return false;
    return true;
}

// named barrier over the 128 threads of one softmax group (ids 1, 2, ...)
__device__ __forceinline__ void group_sync(int id)
{
    asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory");
}
__device__ __forceinline__ bool group_any(int id, bool pred)
{
    uint32_t out;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %2, 0;\n\t"
        "bar.red.or.pred p, %1, 128, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(out)
        : "r"(id), "r"((uint32_t)pred)
        : "memory");
    return out != 0;
}

// Accumulator values of the 8 rows of column chunk c8 in this warp's lanes: with an fp8
// cache every row has two columns (the products with the probabilities' leading bits and
// with the rest), added here.
template <bool kFp8>
__device__ __forceinline__ void load_acc8(uint32_t taddr, int c8, float (&v)[8])
{
    if (kFp8) {
        uint32_t a[8], b[8];
        tmem_ld_x8(taddr + c8 * 16, a);
        tmem_ld_x8(taddr + c8 * 16 + 8, b);
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = __uint_as_float(a[2 * k]) + __uint_as_float(a[2 * k + 1]);
            v[4 + k] = __uint_as_float(b[2 * k]) + __uint_as_float(b[2 * k + 1]);
        }
    } else {
        uint32_t a[8];
        tmem_ld_x8(taddr + c8 * 8, a);
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = __uint_as_float(a[k]);
    }
}

template <bool kFp8>
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    if (kFp8) mma_f8_ss(d, a, b, idesc, acc);
    else mma_f16_ss(d, a, b, idesc, acc);
}

// The columns (query rows g * G + hg) that see a cache position: a range [lo, lo + n).  The
// context before the draft slots (tail index t < 0) is visible to all; draft slot t to the
// queries of its own branch from t on (the plain chain is one branch); a slot at or beyond
// kv_len to none.
struct Seen {
    int lo;
    uint32_t n;
    __device__ __forceinline__ bool operator()(int col) const { return (uint32_t)(col - lo) < n; }
};
__device__ __forceinline__ Seen seen_by(int t, int G, int gamma, int branch_len)
{
    Seen s = {0, t < 0 ? 0xFFFFFFFFu : 0u};
    if (t >= 0 && t < gamma) {
        s.lo = t * G;
        s.n = (uint32_t)((t / branch_len + 1) * branch_len * G - s.lo);
    }
    return s;
}

// fp8 cache: exp2 of eight scaled scores of one position; returns the scores' maximum
// kMask: the tile reaches into the draft slots, a column may not see the position
// Each probability goes out as two E4M3 values in neighbouring bytes, its leading
// four significant bits and the rest (see the head of this file).
template <bool kMask>
__device__ __forceinline__ float exp_chunk(const uint32_t (&r)[8], const float *m8, float scale,
                                           Seen seen, int col0, uint4 &dst)
{
    const float4 ma = *reinterpret_cast<const float4 *>(m8);
    const float4 mb = *reinterpret_cast<const float4 *>(m8 + 4);
    const float mm[8] = {ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w};
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = fmaf(__uint_as_float(r[k]), scale, -mm[k]);
    if (kMask) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = seen(col0 + k) ? x[k] : -INFINITY;
    }
    float mx = fmaxf(fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3])),
                     fmaxf(fmaxf(x[4], x[5]), fmaxf(x[6], x[7])));
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float pr = ex2(x[k]);
        const float hd = e4m3_head(pr);
        w[k] = pack_e4m3x2(hd, pr - hd);
    }
    dst = make_uint4(w[0] | (w[1] << 16), w[2] | (w[3] << 16), w[4] | (w[5] << 16), w[6] | (w[7] << 16));
    return mx;
}

// One pass over this thread's position: exp2 of all n8 column chunks of S^T (four TMEM
// loads in flight per wait), the packed probabilities stored to this position's place in
// the P^T buffer; returns the largest scaled score.  kMask != 0: the tile reaches into the
// draft slots, so columns are masked by what their query may see; the common tile carries
// none of that.  The loop stays rolled: three groups run it at different places, and
// the instruction cache holds the short form better.
template <bool kMask>
__device__ __forceinline__ float softmax_pass(uint32_t s_addr, int n8, const float *m_s, float scale,
                                              Seen seen, uint8_t *prow, long long *tr,
                                              int tile)
{
    float gmax = -INFINITY;
#pragma unroll 1
    for (int cb = 0; cb < n8; cb += 4) {
        uint32_t r[4][8];
        LVSPEC_TILE_TS(tr, 3, tile, (cb >> 2) * 3);         // asks for four chunks of S^T
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (cb + u < n8) tmem_ld_x8(s_addr + (cb + u) * 8, r[u]);
        tmem_wait_ld();
        LVSPEC_TILE_TS(tr, 3, tile, (cb >> 2) * 3 + 1);     // has them
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (cb + u < n8) {
                uint4 pk;
                gmax = fmaxf(gmax, exp_chunk<kMask>(r[u], m_s + (cb + u) * 8, scale, seen, (cb + u) * 8, pk));
                *reinterpret_cast<uint4 *>(prow + (cb + u) * 2048) = pk;
            }
        LVSPEC_TILE_TS(tr, 3, tile, (cb >> 2) * 3 + 2);     // their probabilities stored
    }
    return gmax;
}

// The same for a group that works on a share of the columns, chunks [c_lo, c_hi), of every
// tile: exp2 of its chunks of S^T (up to
// four TMEM loads in flight per wait), packed probabilities into pk, returns the
// largest scaled score.  kMask: the tile reaches into the draft slots, so
// columns are masked by what their query may see; the common tile carries none of that.
template <bool kMask, int kC>
__device__ __forceinline__ float softmax_pass_share(uint32_t s_addr, int c_lo, int c_hi, const float *m_s,
                                              float scale, Seen seen, uint4 (&pk)[kC])
{
    float gmax = -INFINITY;
#pragma unroll
    for (int h = 0; h < (kC + 3) / 4; ++h) {
        const int cb = c_lo + 4 * h;
        if (cb < c_hi) {
            uint32_t r[4][8];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (4 * h + u < kC && cb + u < c_hi) tmem_ld_x8(s_addr + (cb + u) * 8, r[u]);
            tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (4 * h + u < kC && cb + u < c_hi)
                    gmax = fmaxf(gmax, exp_chunk<kMask>(r[u], m_s + (cb + u) * 8, scale, seen, (cb + u) * 8,
                                                              pk[4 * h + u]));
        }
    }
    return gmax;
}

// bf16 exponentials of eight columns of one position, two columns per instruction where the
// machine has a packed form; pmax takes the largest probabilities (bf16 pairs) for the guard.
// y = m - score * scale, so that the packed multiply-add needs no negated operand.
template <bool kMask>
__device__ __forceinline__ uint4 exp_chunk_bf16(const uint32_t *r, const float *m8, uint64_t neg_scale2,
                                                Seen seen, int col0, uint32_t &pmax)
{
    const ulonglong2 ma = *reinterpret_cast<const ulonglong2 *>(m8);
    const ulonglong2 mb = *reinterpret_cast<const ulonglong2 *>(m8 + 4);
    const uint64_t mm[4] = {ma.x, ma.y, mb.x, mb.y};
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float y0, y1;
        unpack_f32x2(fma_f32x2(pack_f32x2(r[2 * k], r[2 * k + 1]), neg_scale2, mm[k]), y0, y1);
        if (kMask) {
            y0 = seen(col0 + 2 * k) ? y0 : INFINITY;
            y1 = seen(col0 + 2 * k + 1) ? y1 : INFINITY;
        }
        w[k] = pack_bf16x2(ex2(-y0), ex2(-y1));
        pmax = max_bf16x2(pmax, w[k]);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// A group's share of the columns of one tile, n_c chunks from column col0 on: exponentials of
// this thread's position (up to four TMEM loads in flight per wait), stored as they come to
// its place in the P^T buffer.  The addresses are those of the share's first chunk.
template <bool kMask, int kC>
__device__ __forceinline__ void softmax_share_bf16(uint32_t s_addr, int n_c, const float *m_s, uint64_t neg_scale2,
                                                   Seen seen, int col0, uint8_t *prow, uint32_t &pmax)
{
    constexpr int kB = kC < 4 ? kC : 4;      // chunks in flight
#pragma unroll
    for (int h = 0; h < (kC + kB - 1) / kB; ++h) {
        if (kB * h < n_c) {
            uint32_t r[kB][8];
#pragma unroll
            for (int u = 0; u < kB; ++u)
                if (kB * h + u < kC && kB * h + u < n_c) tmem_ld_x8(s_addr + (kB * h + u) * 8, r[u]);
            tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < kB; ++u)
                if (kB * h + u < kC && kB * h + u < n_c)
                    *reinterpret_cast<uint4 *>(prow + (kB * h + u) * 2048) =
                        exp_chunk_bf16<kMask>(r[u], m_s + (kB * h + u) * 8, neg_scale2, seen, col0 + (kB * h + u) * 8, pmax);
        }
    }
}

// ---- merge of the splits inside the attention kernel ---------------------------------------
// Where all CTAs of a launch run at once and a head has at most 32 splits, no second kernel merges
// them: every split's CTA merges an equal share of its head's rows.  Between the end of its stream
// and its results a CTA then waits for its head's slowest CTA and one trip through L2, where a
// merge kernel waits for the whole grid to complete (1.7 us), for its own data, and keeps the next
// layer's launch waiting for a second completion (20 rows of 4K: 10.4 us a layer with the merge
// kernel, 8.9 so; 40 rows of 32K 26.4 -> 25.5, 80 rows 28.8 -> 28.0, fp8 cache 21.8 -> 20.6).
// The words themselves say that they have been written: a word of the exchange buffer nobody has
// written is kNoWord, which no partial is, and whoever has read a word makes it kNoWord again
// for the next launch.  So there is no fence and no flag between a partial and its reader, whose
// first request for the data is also its first look whether they are there (statistics first and
// rows once they are there, a request each: 0.3 us more; a flag behind a fence, 1.5 us more).
// Nobody waits without end, since the CTAs it waits for may not run (other grids share the GPU):
// after `merge_polls` requests a CTA gives its share up.  merge_word counts the CTAs of a head
// whose partials are written, and its upper half has a bit for every share given up; both move in one
// atomic operation, so either the one who gives up sees that all have arrived (and reads on) or the
// last to arrive sees the bit, and merges that share itself by the same arithmetic.
// A CTA that leaves because a wait has run out may leave words behind that nobody makes kNoWord again.
// It has raised LVSPEC_DEV_WAIT_EXPIRED, and while that stands (lvspec_device_status puts the buffer
// in order and takes it back) a word that has been written need not be this launch's: CTAs then
// read nothing before all of their head's have arrived, and give their shares up until then.
__device__ __forceinline__ bool all_there(const uint4 &x)
{
    return x.x != kNoWord && x.y != kNoWord && x.z != kNoWord && x.w != kNoWord;
}
// any value but the mark of a word nobody has written (a NaN's payload gives way)
__device__ __forceinline__ uint32_t passable(float x) { return min(__float_as_uint(x), kNoWord - 1u); }

// A row of a head and one warp's part of its merge: the splits first, first + step, ... of n.
struct MergePart {
    float *stat, *rows;      // statistics of split `lane`; this lane's four channels of the first split's row
    size_t stride;           // from one of the part's splits to the next
    int n, mine, first, step;
    size_t row;              // of the results
    __device__ __forceinline__ MergePart(const AttnParams &p, uint32_t group_magic, int b, int kvh, int r, int n_, int first_,
                                         int step_, int lane)
        : n(n_), first(first_), step(step_)
    {
        const size_t unit0 = ((size_t)b * p.Hkv + kvh) * p.n_split;
        stat = p.part_stat + ((unit0 + lane) * p.M + r) * 4;
        rows = p.part_o + ((unit0 + first) * p.M + r) * p.D + lane * 4;
        stride = (size_t)step * p.M * p.D;
        mine = step == 4 ? (n - first + 3) >> 2 : step == 2 ? (n - first + 1) >> 1 : n - first;
        const int g = div_by(r, p.G, group_magic), hg = r - g * p.G;
        row = ((size_t)b * p.gamma + g) * p.Hq + kvh * p.G + hg;
    }
};
struct MergedRow {
    float m, l, lv;      // reference exponent, softmax sum, its part in the visual span
    float4 o;            // this lane's four channels, over this warp's splits
};
// False when a word is still missing after `polls` requests.  kFlight: rows in flight per
// lane, no more than there are: this code runs once, on cold instruction caches (twelve instead of
// four cost 16 rows on 8 splits 0.9 us, eight instead of twelve cost 9 splits a warp 0.7 us).
template <int kFlight>
__device__ __forceinline__ bool merge_row(const AttnParams &p, const MergePart &t, int lane, uint32_t polls, MergedRow &res)
{
    const bool active = lane * 4 < p.D;
    uint4 st = make_uint4(0, 0, 0, 0), x[kFlight];
    // statistics and the first rows travel together
    if (lane < t.n) st = ld_relaxed_v4(t.stat);
    const float *src = t.rows;
    auto fetch = [&](int n) {
#pragma unroll
        for (int k = 0; k < kFlight; ++k) {
            x[k] = make_uint4(0, 0, 0, 0);
            if (active && k < n) x[k] = ld_relaxed_v4(src + k * t.stride);
        }
    };
    fetch(t.mine);
    uint32_t tries = 0;
    while (!__all_sync(0xffffffffu, all_there(st))) {
        if (tries++ >= polls) return false;
        if (!all_there(st)) st = ld_relaxed_v4(t.stat);
#pragma unroll
        for (int k = 0; k < kFlight; ++k)
            if (!all_there(x[k])) x[k] = ld_relaxed_v4(src + k * t.stride);
    }
    const float sm = __uint_as_float(st.x), sl = __uint_as_float(st.y), sv = __uint_as_float(st.z);
    const float m_mine = lane < t.n && sl > 0.f ? sm : -INFINITY;
    float m = m_mine;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float w = m_mine > -INFINITY ? exp2f(m_mine - m) : 0.f;
    float l = w * sl, lv = w * sv;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l += __shfl_xor_sync(0xffffffffu, l, o);
        lv += __shfl_xor_sync(0xffffffffu, lv, o);
    }
    res.m = m; res.l = l; res.lv = lv;
    res.o = make_float4(0.f, 0.f, 0.f, 0.f);
    int u = t.first;
#pragma unroll 1
    for (int left = t.mine; left > 0;) {
        for (;;) {
            bool ok = true;
#pragma unroll
            for (int k = 0; k < kFlight; ++k) ok = ok && all_there(x[k]);
            if (__all_sync(0xffffffffu, ok)) break;
            if (tries++ >= polls) return false;
#pragma unroll
            for (int k = 0; k < kFlight; ++k)
                if (!all_there(x[k])) x[k] = ld_relaxed_v4(src + k * t.stride);
        }
#pragma unroll
        for (int k = 0; k < kFlight; ++k, u += t.step) {
            // (a split of weight zero may hold anything, and a place beyond the last split holds zeros)
            const float wk = __shfl_sync(0xffffffffu, w, u & 31);
            if (k < left && wk != 0.f) {
                res.o.x = fmaf(wk, __uint_as_float(x[k].x), res.o.x);
                res.o.y = fmaf(wk, __uint_as_float(x[k].y), res.o.y);
                res.o.z = fmaf(wk, __uint_as_float(x[k].z), res.o.z);
                res.o.w = fmaf(wk, __uint_as_float(x[k].w), res.o.w);
            }
        }
        left -= kFlight;
        src += kFlight * t.stride;
        if (left > 0) fetch(left);
    }
    return true;
}
// A share's rows [r0, r0 + rows) and log2 of the warps per row.
struct Share {
    int r0, rows, shift;
    __device__ __forceinline__ Share(const AttnParams &p, uint32_t split_magic, int split, int n)
    {
        // (fewer splits than asked for, where a sequence has fewer tiles: the plain division)
        r0 = n == p.n_split ? div_by(split * p.M, n, split_magic) : split * p.M / n;
        rows = (n == p.n_split ? div_by(split * p.M + p.M, n, split_magic) : (split + 1) * p.M / n) - r0;
        shift = rows * 4 <= kSoftmaxWarps ? 2 : rows * 2 <= kSoftmaxWarps ? 1 : 0;
    }
};
// A row's results.
__device__ __forceinline__ void write_row(const AttnParams &p, const MergePart &t, int lane, const MergedRow &res)
{
    const float inv = 1.f / res.l;
    if (lane * 4 < p.D)
        *reinterpret_cast<uint2 *>(p.out + t.row * p.D + lane * 4) =
            make_uint2(pack_bf16x2(res.o.x * inv, res.o.y * inv), pack_bf16x2(res.o.z * inv, res.o.w * inv));
    if (lane == 0) {
        p.mass[t.row] = res.lv * inv;
        if (p.lse2) p.lse2[t.row] = res.m + log2f(res.l);
    }
}
// The words that this warp has read are nobody's again.
__device__ __forceinline__ void clear_part(const AttnParams &p, const MergePart &t, int lane)
{
    const uint4 none = make_uint4(kNoWord, kNoWord, kNoWord, kNoWord);
    float *dst = t.rows;
    if (lane * 4 < p.D)
#pragma unroll 4
        for (int k = 0; k < t.mine; ++k, dst += t.stride) st_relaxed_v4(dst, none);
    if (t.first == 0 && lane < t.n) st_relaxed_v4(t.stat, none);
}

// kFp8: E4M3 cache (tmap_q is not used: q is split into its two E4M3 tiles by the CTA).
// kTurns: the softmax groups take the tiles in turn (fp8 cache only); otherwise all groups
// work on every tile, each on a share of its columns, at most kC chunks of eight.
// Draft trees and page pools are run-time cases (a mask range per position, a look-up per
// tile): as template cases they gave nothing.
// kMerge: the launch may merge its splits itself.  With a bf16 cache a case of its own, because that code
// takes registers (128 a thread against 104 to 116): without it another kernel's CTAs find room beside this one's.
// With an fp8 cache it is 128 either way, and one instance decides by p.merge.
template <bool kFp8, bool kTurns, int kC, bool kMerge>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc_kernel(const TcParams P, const SeqInfo seq, const __grid_constant__ CUtensorMap tmap_k,
               const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_q)
{
    static_assert(kFp8 || !kTurns, "a bf16 cache does not go through in turns");
    static_assert(kMerge || !kFp8, "one instance per organisation of an fp8 cache");
    auto merges = [&] { return kFp8 ? P.a.merge != 0 : kMerge; };     // (asked anew: a register less)
    // bytes of one K or V tile: two 64-channel boxes at head_dim 128 (bf16), one box at
    // head_dim 64 and for an fp8 tile of 128 channels
    const uint32_t kSlot = (uint32_t)P.cfg.slot_bytes;
    const bool two_boxes = kSlot == kSlotBytes;
    const int D = P.a.D;
    const bool paged = P.a.page_size > 0;
    extern __shared__ uint8_t smem_raw[];
    const AttnParams &p = P.a;
    const TcConfig &cfg = P.cfg;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
#ifdef LVSPEC_TRACE
    unsigned long long *rec = nullptr;      // this CTA's record (one thread writes it)
    long long *tile_tr = nullptr;           // per-tile stamps of the one traced CTA (lane 0 of its warps)
    if (g_lvspec_trace && tid == 32) {
        const unsigned long long idx = atomicAdd(g_lvspec_trace, 1ull);
        if (idx < (unsigned long long)kTraceCtaRecords) {
            rec = g_lvspec_trace + 8 + idx * 8;
            rec[0] = 1;
            rec[1] = (unsigned long long)P.a.q;
            rec[2] = blockIdx.x + 1000 * blockIdx.y + 1000000 * blockIdx.z;
            rec[3] = lvspec_trace_now();
        }
    }
    if (g_lvspec_trace && blockIdx.x == 3 && blockIdx.y == 2 && blockIdx.z == 0 && lane == 0)
        tile_tr = reinterpret_cast<long long *>(g_lvspec_trace + 8 + 8 * kTraceCtaRecords);   // 4 roles x 32 tiles x 8 stamps
#else
    constexpr long long *tile_tr = nullptr;
#endif
    // the TMA unit fetches the descriptors while everything else is set up; a warp that
    // has nothing to do in the prologue asks for them, not the producer (whose first
    // load is what the whole CTA waits for)
    if (warp == kPvWarp) {
        if (lane == 0) prefetch_tensormap(&tmap_k);
        if (lane == 1 && !kFp8) prefetch_tensormap(&tmap_q);
        if (lane == 2) prefetch_tensormap(&tmap_v);
    }
    const int split = blockIdx.x, kvh = blockIdx.y, b = blockIdx.z;
    const int L = seq.kv_len[b], vs = seq.span_start[b], ve = seq.span_end[b];
    const int M = p.M, G = p.G, gamma = p.gamma, NP = cfg.n_pad;
    const int n8 = (M + 7) >> 3;

    // tiles [t_begin, t_begin + T) of this split: equal shares, sizes differ by at most one
    const int n_tiles = (L + kTilePos - 1) / kTilePos;
    const int t_base = div_by(n_tiles, p.n_split, P.cfg.split_magic), t_rem = n_tiles - t_base * p.n_split;
    const int t_begin = split * t_base + min(split, t_rem);
    const int T = t_base + (split < t_rem ? 1 : 0);

    // tiles per hand-over (no test of T where it is 1 anyway: with the widest shares the extra
    // register costs 1.5 % at 100 rows)
    const int step = kC == kMaxChunks || T >= cfg.pair_from ? cfg.step : 1;

    const size_t unit = ((size_t)b * p.Hkv + kvh) * p.n_split + split;
    float *part_o = p.part_o + unit * (size_t)M * P.a.D;
    float *part_stat = p.part_stat + unit * (size_t)M * 4;
    if (T <= 0) {   // a split with no tile: contributes nothing
        if (tid == 0) {
            grid_dependency_wait();
            grid_launch_dependents();
        }
        __syncthreads();
        for (int r = tid; !merges() && r < M; r += kThreads)
            *reinterpret_cast<float4 *>(part_stat + r * 4) = make_float4(kMFloor, 0.f, 0.f, 0.f);
        return;
    }

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t *gbase = smem_raw + (base - smem_u32(smem_raw));
    const SmemMap &sm = P.sm;
    float *m_s = reinterpret_cast<float *>(gbase + sm.m);
    float *dl_s = reinterpret_cast<float *>(gbase + sm.dl);
    float *tmx_s = reinterpret_cast<float *>(gbase + sm.tmx);
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(gbase + sm.misc);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(gbase + sm.misc + 4);
    // how often the reference exponents m[] have been set or moved; tiles handed to the P.V issuer
    volatile uint32_t *epoch_s = reinterpret_cast<volatile uint32_t *>(gbase + sm.misc + 8);
    volatile uint32_t *committed_s = reinterpret_cast<volatile uint32_t *>(gbase + sm.misc + 12);
    volatile uint32_t *arrived_s = reinterpret_cast<volatile uint32_t *>(gbase + sm.misc + 16 + 4 * kSoftmaxWarps);
    volatile uint32_t *doubt_s = arrived_s + 1;      // (the first softmax thread's)

    // barrier addresses
    const uint32_t bar0 = base + sm.bars;
    auto k_full = [&](int s) { return bar0 + 8 * s; };
    auto k_empty = [&](int s) { return bar0 + 8 * (cfg.ks + s); };
    auto v_full = [&](int s) { return bar0 + 8 * (2 * cfg.ks + s); };
    auto v_empty = [&](int s) { return bar0 + 8 * (2 * cfg.ks + cfg.vs + s); };
    const uint32_t bar1 = bar0 + 8 * (2 * cfg.ks + 2 * cfg.vs);
    // The hand-over barriers of tile i are those of index i % kRound, whatever the number of
    // S^T and P^T buffers: a parity wait tells a phase from its neighbours only, so whoever
    // waits for a phase must know the phase before it to be over, and the one after it not to
    // be.  Products end in order, and no product of a tile that is not yet handed over can end.
    // Whoever writes tile i has first waited for the product of tile i - pb, in turns as with
    // shared columns, and only then waits for that of tile i - 1 (ahead of a rescale, or of zeroing V
    // rows): with pb <= 4 the phase before that one, tile i - 5's, is over by then, while tile i - 4
    // being done a turn ago is nothing that could be relied on.  The wait for tile i - pb itself comes
    // after the one for tile i - 3 - pb (in turns, a turn ago) or i - 1 - pb (shared columns).  The K.Q^T of
    // tile i + 4 waits until tile i has been read (at most four S^T buffers).
    constexpr int kRound = kHand;
    static_assert(kHand == 4, "as many S^T and P^T buffers at most: see above");
    static_assert(kMergeRows <= kSoftmaxWarps, "a warp per row of a share");
    static_assert(kMergeSplits <= 32, "a bit of the word's upper half and a lane per split");
    auto s_full = [&](int i) { return bar1 + 8 * (i % kRound); };
    auto s_free = [&](int i) { return bar1 + 8 * (kHand + i % kRound); };
    auto p_full = [&](int i) { return bar1 + 8 * (2 * kHand + i % kRound); };
    auto p_free = [&](int i) { return bar1 + 8 * (3 * kHand + i % kRound); };
    auto hand_parity = [](int i) { return (uint32_t)(i / kRound) & 1u; };
    const uint32_t drain_bar = bar1 + 8 * (4 * kHand);
    const uint32_t done_bar = drain_bar + 8;
    const uint32_t q_full = drain_bar + 16;
    const uint32_t pv_done = drain_bar + 24;
    const int bh = b * p.Hkv + kvh;

    // the cache is read once per call: it should not push the split partials out of L2
    const uint64_t stream_policy = l2_evict_first_policy();
    // where tile i of this split sits in the [sequences or pages, heads, positions, 128]
    // maps: (position, sequence or page)
    volatile int32_t *page_s = reinterpret_cast<volatile int32_t *>(gbase + sm.pages);
    auto tile_at = [&](int i, int &pos0, int &map_row) {
        pos0 = (t_begin + i) * kTilePos;
        map_row = b;
        if (paged) {
            // a page holds a whole number of tiles; an entry outside the pool reads as zeros
            pos0 -= (pos0 / p.page_size) * p.page_size;
            map_row = page_s[i];
        }
    };
    auto load_k = [&](int i) {
        const int ks = i % cfg.ks;
        int pos0, map_row;
        tile_at(i, pos0, map_row);
        mbar_arrive_expect_tx(k_full(ks), kSlot);
        tma_load_4d_hint(base + sm.k + ks * kSlot, &tmap_k, k_full(ks), 0, pos0, kvh, map_row, stream_policy);
        if (two_boxes)
            tma_load_4d_hint(base + sm.k + ks * kSlot + kBoxBytes, &tmap_k, k_full(ks), 64, pos0, kvh, map_row,
                             stream_policy);
    };
    auto load_v = [&](int i) {
        const int vsl = i % cfg.vs;
        int pos0, map_row;
        tile_at(i, pos0, map_row);
        mbar_arrive_expect_tx(v_full(vsl), kSlot);
        tma_load_4d_hint(base + sm.v + vsl * kSlot, &tmap_v, v_full(vsl), 0, pos0, kvh, map_row, stream_policy);
        if (two_boxes)
            tma_load_4d_hint(base + sm.v + vsl * kSlot + kBoxBytes, &tmap_v, v_full(vsl), 64, pos0, kvh, map_row,
                             stream_policy);
    };

    // With one K slot (113 rows and more) a K tile can be loaded only when the one before has been
    // used: it is brought into L2 meanwhile, behind the loads that are needed sooner.  (120 rows of
    // 32K 39.4 -> 36.7 us a layer, 128 rows 38.9 -> 37.3; V tiles too: 41.2 and 40.1.)
    auto prefetch_k = [&](int i) {
        if constexpr (kC == kMaxChunks) {
            if (cfg.ks > 1 || i >= T) return;
            int pos0, map_row;
            tile_at(i, pos0, map_row);
            tma_prefetch_4d(&tmap_k, 0, pos0, kvh, map_row);
            if (two_boxes) tma_prefetch_4d(&tmap_k, 64, pos0, kvh, map_row);
        }
    };

    float scale_cta = p.scale_log2;     // softmax scale of this CTA (fp8 cache: with the K scale and q's shift)
    float v_scale = 1.f;

    // ------------------------------------------------------------------ prologue
    // The producer thread sets the barriers up and starts the first loads at
    // once; the other warps prepare shared memory and TMEM meanwhile.
    int first_k = 0, first_v = 0;   // loads issued before the CTA-wide barrier
    if (warp == 0) {
        {
            // one barrier per lane, all at once (an mbarrier.init costs about a hundred
            // cycles): barriers sit in the order k_full, k_empty, v_full, v_empty,
            // s_full[4], s_free[4], p_full[4], p_free[4], drain, done, q_full, pv_done
            const int n_kv = 2 * cfg.ks + 2 * cfg.vs;
            constexpr int n_sp = 4 * kHand;
            const int n_bars = n_kv + n_sp + 4;
            for (int i = lane; i < n_bars; i += 32) {
                const int j = i - n_kv;          // index among the barriers after the rings
                uint32_t count = 1;
                if (j >= kHand && j < 3 * kHand) count = kTurns ? 4 : kSoftmaxWarps;   // s_free, p_full: the warps that work on a tile
                else if (j == n_sp + 1) count = kSoftmaxWarps + 1;              // done
                mbar_init(bar0 + 8 * i, count);
            }
            if (lane == 0) {
                *abort_flag = 0;
                *epoch_s = 0;
                *committed_s = 0;
                *arrived_s = 0;
            }
            fence_proxy_async_smem();
        }
        __syncwarp();
        // The barriers are there: the other warps need not wait for the loads to be asked for (2.4 k cycles
        // from here to the last one), nor this one for them.
        asm volatile("bar.arrive 0, %0;" ::"n"(kThreads) : "memory");
        if (paged) {
            // the block table too may come from the kernel before this one: the warp reads
            // this split's entries (one per tile) after the wait, then lane 0 goes on
            grid_dependency_wait();
            const int32_t *row = p.block_table + (size_t)b * p.pages_per_seq;
            for (int i = lane; i < T; i += 32) page_s[i] = row[((t_begin + i) * kTilePos) / p.page_size];
            __syncwarp();
        }
        if (lane == 0) {
            // inputs may come from the kernel before this one in the stream
            grid_dependency_wait();
            // the first K tile comes from HBM and is needed first: it goes out before Q
            first_k = min(T, cfg.ks);
            first_v = min(T, cfg.vs);
            load_k(0);
            if (!kFp8) {
                mbar_arrive_expect_tx(q_full, (uint32_t)(M * D) * 2u);
                tma_load_4d(base + sm.q, &tmap_q, q_full, 0, kvh * G, 0, b);
                if (two_boxes) tma_load_4d(base + sm.q + NP * 128, &tmap_q, q_full, 64, kvh * G, 0, b);
            }
            for (int i = 0; i < first_v; ++i) {
                if (i > 0 && i < first_k) load_k(i);
                load_v(i);
            }
            for (int i = max(first_v, 1); i < first_k; ++i) load_k(i);    // a K ring deeper than the V ring
            prefetch_k(first_k);
        }
        __syncwarp();
    } else if (warp == 1) {
        tmem_alloc(base + sm.misc, (uint32_t)cfg.tmem_cols);
        tmem_relinquish();
    } else if (warp < kPvWarp) {
        const int idx = tid - 64;   // 0..kSoftmaxThreads-1
        // rows M..NP-1 of Q are padding: zero them (the TMA boxes cover rows < M only;
        // with an fp8 cache the split of q below writes every row)
        for (int i = idx; !kFp8 && i < (NP - M) * 16; i += kSoftmaxThreads) {
            const int r = M + (i >> 4), c = i & 15, h = c >> 3, cc = c & 7;
            *reinterpret_cast<uint4 *>(gbase + sm.q + h * (NP * 128) + r * 128 + cc * 16) =
                make_uint4(0, 0, 0, 0);
        }
        // columns beyond the last chunk (at most one chunk, 2 KB, per P buffer) stay zero
        if (n8 * 8 < NP)
            for (int i = idx; i < cfg.pb * 128; i += kSoftmaxThreads)
                *reinterpret_cast<uint4 *>(gbase + sm.p + (i >> 7) * (NP * 256) + n8 * 2048 + (i & 127) * 16) =
                    make_uint4(0, 0, 0, 0);
        for (int n = idx; n < NP; n += kSoftmaxThreads) {
            m_s[n] = kFp8 ? kMFloor : 0.f;
        }
        if (kFp8) {
            // (q may come from the kernel before this one)
            grid_dependency_wait();
            // ---- q as two E4M3 operand tiles (128-byte swizzle, one 128-byte row per query row)
            // chunk = 8 channels of one row (16 bytes of bf16 in, 8 + 8 bytes out)
            const int idx = tid - 32 * kSoftmaxWarp0;
            const int n_chunks = NP * 16;
            constexpr int kMine = (kMaxRowsFp8 * 16 + kSoftmaxThreads - 1) / kSoftmaxThreads;
            uint4 qv[kMine];
            float amax = 0.f;
#pragma unroll
            for (int u = 0; u < kMine; ++u) {
                const int ch = idx + u * kSoftmaxThreads;
                qv[u] = make_uint4(0, 0, 0, 0);
                if (ch < n_chunks) {
                    const int n = ch >> 4, c = ch & 15;
                    if (n < M) {
                        const int g = n / G, hg = n - g * G;
                        qv[u] = *reinterpret_cast<const uint4 *>(
                            p.q + (((size_t)b * gamma + g) * p.Hq + kvh * G + hg) * 128 + c * 8);
                    }
                    const uint32_t w[4] = {qv[u].x, qv[u].y, qv[u].z, qv[u].w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        amax = fmaxf(amax, fabsf(__uint_as_float(w[k] << 16)));
                        amax = fmaxf(amax, fabsf(__uint_as_float(w[k] & 0xFFFF0000u)));
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            volatile float *wmax = reinterpret_cast<volatile float *>(gbase + sm.misc + 16);
            if (lane == 0) wmax[warp - kSoftmaxWarp0] = amax;
            asm volatile("bar.sync %0, %1;" ::"r"(kQBarrier), "r"(kSoftmaxThreads) : "memory");
            amax = 0.f;
#pragma unroll
            for (int u = 0; u < kSoftmaxWarps; ++u) amax = fmaxf(amax, wmax[u]);
            // power of two that brings the largest magnitude into [128, 256) (NaN or Inf in q:
            // no shift; the result is then NaN as it would be with any cache)
            int shift = 0;
            if (amax > 0.f && amax < INFINITY) shift = 7 - ((int)((__float_as_uint(amax) >> 23) & 0xFF) - 127);
            shift = max(-100, min(100, shift));
            const float up = __uint_as_float((uint32_t)(127 + shift) << 23);
#pragma unroll
            for (int u = 0; u < kMine; ++u) {
                const int ch = idx + u * kSoftmaxThreads;
                if (ch < n_chunks) {
                    const int n = ch >> 4, c = ch & 15;
                    const uint32_t w[4] = {qv[u].x, qv[u].y, qv[u].z, qv[u].w};
                    uint32_t hd[4], rs[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float x0 = __uint_as_float(w[k] << 16) * up, x1 = __uint_as_float(w[k] & 0xFFFF0000u) * up;
                        const float h0 = e4m3_head(x0), h1 = e4m3_head(x1);
                        hd[k] = pack_e4m3x2(h0, h1);
                        rs[k] = pack_e4m3x2(x0 - h0, x1 - h1);
                    }
                    const uint32_t off = n * 128 + (((c >> 1) ^ (n & 7)) << 4) + ((c & 1) << 3);
                    *reinterpret_cast<uint2 *>(gbase + sm.q + off) = make_uint2(hd[0] | (hd[1] << 16), hd[2] | (hd[3] << 16));
                    *reinterpret_cast<uint2 *>(gbase + sm.q + NP * 128 + off) =
                        make_uint2(rs[0] | (rs[1] << 16), rs[2] | (rs[3] << 16));
                }
            }
            scale_cta = p.scale_log2 * p.k_scale[bh] * __uint_as_float((uint32_t)(127 - shift) << 23);
            v_scale = p.v_scale[bh];
        }
        fence_proxy_async_smem();
    }
    if (warp != 0) {
        // nobody polls a barrier while the grid before this one is still running
        grid_dependency_wait();
        tc_fence_before();
        asm volatile("bar.sync 0, %0;" ::"n"(kThreads) : "memory");
        tc_fence_after();
    }
#ifdef LVSPEC_TRACE
    if (rec) rec[4] = lvspec_trace_now();
#endif
    const uint32_t tmem_base = warp != 0 ? *tmem_slot : 0u;      // (the producer has no use for it)
    // accumulator columns: the S^T buffers, then O^T and the sums (fp8 cache: two columns per row)
    constexpr int kAccCols = kFp8 ? 2 : 1;
    const uint32_t tm_s0 = tmem_base, tm_o = tmem_base + cfg.sb * NP, tm_l = tm_o + kAccCols * NP;
    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            int nk = first_k, nv = first_v;   // loads issued so far
            // K and V slots free up at different times: poll both, never block on one
            uint64_t idle_since = 0;
            uint32_t spin = 0;
            while (nk < T || nv < T) {
                bool progress = false;
                if (nk < T && mbar_test_wait(k_empty(nk % cfg.ks), ((nk / cfg.ks) - 1) & 1)) {
                    load_k(nk);
                    ++nk;
                    prefetch_k(nk);
                    progress = true;
                }
                if (nv < T && mbar_test_wait(v_empty(nv % cfg.vs), ((nv / cfg.vs) - 1) & 1)) {
                    load_v(nv);
                    ++nv;
                    progress = true;
                }
                if (progress) {
                    idle_since = 0;
                } else {
                    if (*abort_flag) break;
                    if ((++spin & 255u) == 0) {
                        const uint64_t now = global_timer_ns();
                        if (idle_since == 0) idle_since = now;
                        else if (now - idle_since > 2000000000ull) {
                            *abort_flag = 1;
                            break;
                        }
                    }
                }
            }
            if (*abort_flag) {
                // wait (bounded) for the copies still in flight before the CTA leaves
                if (!kFp8) wait_unconditional(q_full, 0);
                for (int j = max(0, nk - cfg.ks); j < nk; ++j)
                    wait_unconditional(k_full(j % cfg.ks), (j / cfg.ks) & 1);
                for (int j = max(0, nv - cfg.vs); j < nv; ++j)
                    wait_unconditional(v_full(j % cfg.vs), (j / cfg.vs) & 1);
            }
        }
    } else if (warp == 1) {
        // -------------------------------------------------------------- MMA issuer
        // The whole warp runs the loop and one elected lane issues: the descriptors are
        // then the same in every lane and the compiler can keep them where the MMA
        // instruction takes its operands from, instead of moving them there per instruction.
        {
            const uint32_t idesc_qk = kFp8 ? make_idesc_e4m3(128, NP, 0, 0) : make_idesc_bf16(128, NP, 0, 0);
            // descriptors: everything but the start address is fixed, and the start
            // address field (address / 16) moves by compile-time steps
            const uint64_t kd0 = make_smem_desc(base + sm.k, 16, 1024, kSwizzle128B);
            uint64_t qd[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                qd[j] = make_smem_desc(base + sm.q + (j >> 2) * (NP * 128) + (j & 3) * 32, 16, 1024,
                                       kSwizzle128B);
            Ring k_ring(cfg.ks), s_ring(cfg.sb), hand(kRound), freed(kRound);
            auto issue_qk = [&](int i) -> bool {
                const int ks = k_ring.idx, sb = s_ring.idx;
                LVSPEC_TILE_TS(tile_tr, 1, i, 0);     // starts waiting for the K tile
                bool there = mbar_wait(k_full(ks), k_ring.parity, abort_flag);
                LVSPEC_TILE_TS(tile_tr, 1, i, 1);     // K tile there
                // the tile that used this S^T buffer last (tile i - sb) has been read
                if (i >= cfg.sb) {
                    there = mbar_wait(bar1 + 8 * (kHand + freed.idx), freed.parity, abort_flag) && there;
                    freed.next();
                }
                if (!__all_sync(0xffffffffu, there)) return false;
                LVSPEC_TILE_TS(tile_tr, 1, i, 2);     // S^T buffer free
                tc_fence_after();
                const uint64_t kd = kd0 + (uint64_t)(ks * (kSlot >> 4));
                const uint32_t d = tm_s0 + sb * NP;
                // bf16: 8 steps of 16 channels over the two 64-channel boxes (4 over the one box
                // of head_dim 64); fp8: 4 steps of 32 channels against q's leading bits, then the
                // same 4 against the rest
                if (elect_one()) {
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if (kFp8) mma_f8_ss(d, kd + (uint64_t)((j & 3) * 2), qd[j], idesc_qk, j > 0);
                        else if (j < 4 || two_boxes)
                            mma_f16_ss(d, kd + (uint64_t)((j >> 2) * (kBoxBytes >> 4) + (j & 3) * 2), qd[j],
                                       idesc_qk, j > 0);
                    }
                    mma_commit(bar1 + 8 * hand.idx);      // s_full of tile i
                    mma_commit(k_empty(ks));
                }
                __syncwarp();
                LVSPEC_TILE_TS(tile_tr, 1, i, 3);     // K.Q^T issued
                k_ring.next();
                s_ring.next();
                hand.next();
                return true;
            };
            // (fp8 cache: the CTA has split q itself, ahead of the barrier above)
            bool ok = kFp8 || __all_sync(0xffffffffu, mbar_wait(q_full, 0, abort_flag));
            for (int i = 0; ok && i < T; ++i) ok = issue_qk(i);
            // every MMA issued by the elected lane has finished before TMEM is released
            if (elect_one()) {
                mma_commit(drain_bar);
                wait_unconditional(drain_bar, 0);
            }
            __syncwarp();
        }
    } else if (warp == kPvWarp) {
        // ------------------------------------------------- P.V and sum MMA issuer
        // (whole warp in the loop, one elected lane issues: see the K.Q^T issuer)
        {
            // This warp is idle until the first P^T: it makes its constant tiles, 64 x 16 bf16 (K-major,
            // no swizzle: the 8 positions of chunk c at c * 1024, row r at (r / 8) * 128 +
            // (r % 8) * 16).  Row 0 = ones (sums l), row 1 = 1 inside the visual span (sums
            // l_vis), rows 2.. = 0.  Tile 0: block inside the span, 1: outside, 2: the 16-block
            // holding the span start, 3: the 16-block holding the span end.
            // (fp8 cache: the tiles are 64 x 32 E4M3, 16 positions per 16-byte chunk, and the
            // boundary tiles cover the 32-block holding the span's start / end)
#pragma unroll 1
            for (uint32_t i = lane * 16; i < 4 * kA2Bytes; i += 512)
                *reinterpret_cast<uint4 *>(gbase + sm.a2 + i) = make_uint4(0, 0, 0, 0);
            __syncwarp();
            if (lane < 16) {
                constexpr int kPer = kFp8 ? 16 : 8;             // positions per 16-byte chunk
                const int tile = lane >> 2, c = (lane >> 1) & 1, rr = lane & 1;
                const int p0 = ((tile == 2 ? vs : ve) & ~(2 * kPer - 1)) + c * kPer;
                // the chunk's positions [lo, hi) count
                const int lo = rr == 1 && tile >= 2 ? vs - p0 : 0;
                const int hi = rr == 0 || tile == 0 ? kPer : tile == 1 ? 0 : ve - p0;
                uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
                for (int k = 0; k < kPer; ++k) {
                    const bool one = k >= lo && k < hi;
                    if (kFp8) w[k >> 2] |= (one ? 0x38u : 0u) << (8 * (k & 3));       // E4M3 1.0
                    else w[k >> 1] |= (one ? 0x3F80u : 0u) << (16 * (k & 1));         // bf16 1.0
                }
                *reinterpret_cast<uint4 *>(gbase + sm.a2 + tile * kA2Bytes + c * 1024 + rr * 16) =
                    make_uint4(w[0], w[1], w[2], w[3]);
            }
            fence_proxy_async_smem();
            __syncwarp();
            const uint32_t idesc_pv = kFp8 ? make_idesc_e4m3(128, 2 * NP, 1, 1) : make_idesc_bf16(128, NP, 1, 1);
            const uint32_t idesc_sum = kFp8 ? make_idesc_e4m3(64, 2 * NP, 0, 1) : make_idesc_bf16(64, NP, 0, 1);
            // one MMA covers 16 positions of a bf16 tile, 32 of an fp8 tile
            constexpr int kSteps = kFp8 ? 4 : 8, kStepPos = kTilePos / kSteps;
            constexpr uint32_t kVStep = kStepPos * 128 >> 4, kPStep = kStepPos * 16 >> 4;   // descriptor units
            const uint64_t vd0 = make_smem_desc(base + sm.v, kBoxBytes, 1024, kSwizzle128B);
            const uint64_t pd0 = make_smem_desc(base + sm.p, 128, 2048, kSwizzleNone);
            const uint64_t a2d0 = make_smem_desc(base + sm.a2, 1024, 128, kSwizzleNone);
            Ring v_ring(cfg.vs), p_ring(cfg.pb), hand(kRound);
            for (int i = 0; i < T; ++i, v_ring.next(), p_ring.next(), hand.next()) {
                const int pb = p_ring.idx, vsl = v_ring.idx;
                LVSPEC_TILE_TS(tile_tr, 2, i, 0);     // starts waiting for P^T
                // p_full of tile i (two tiles handed over together: on the first one's barrier)
                bool there = true;
                if (kTurns || step == 1 || !(i & 1))
                    there = mbar_wait(bar1 + 8 * (2 * kHand + hand.idx), hand.parity, abort_flag);
                LVSPEC_TILE_TS(tile_tr, 2, i, 1);     // P^T there
                there = mbar_wait(v_full(vsl), v_ring.parity, abort_flag) && there;
                if (!__all_sync(0xffffffffu, there)) break;
                LVSPEC_TILE_TS(tile_tr, 2, i, 2);     // V tile there
                tc_fence_after();
                // V^T: channels contiguous (M-major), 64-channel halves kBoxBytes apart,
                // groups of 8 positions 1024 bytes apart.  (At head_dim 64 the product still
                // has 128 rows: its upper half reads whatever follows the box in shared memory
                // and lands in TMEM lanes nobody reads.)  P^T: rows contiguous in
                // 16-byte chunks (N-major), chunk stride 2048, groups of 8 positions 128
                // bytes apart.
                const uint64_t vd = vd0 + (uint64_t)(vsl * (kSlot >> 4));
                const uint64_t pd = pd0 + (uint64_t)(pb * ((NP * 256) >> 4));
                const int pos0 = (t_begin + i) * kTilePos;
                // constant tile per block of 16 (fp8: 32) positions: 0 inside the span, 1
                // outside, 2 / 3 the blocks holding the span's start / end
                int uniform = -1;
                if (pos0 >= vs && pos0 + kTilePos <= ve) uniform = 0;
                else if (pos0 + kTilePos <= vs || pos0 >= ve) uniform = 1;
                const uint32_t first_acc = i > 0 ? 1u : 0u;
                if (!elect_one()) {
                    // the other lanes wait at the end of the turn
                } else if (uniform >= 0) {
                    const uint64_t d2 = a2d0 + (uint64_t)(uniform * (kA2Bytes >> 4));
#pragma unroll
                    for (int j = 0; j < kSteps; ++j)
                        mma_ss<kFp8>(tm_l, d2, pd + (uint64_t)(j * kPStep), idesc_sum, j > 0 ? 1u : first_acc);
#pragma unroll
                    for (int j = 0; j < kSteps; ++j)
                        mma_ss<kFp8>(tm_o, vd + (uint64_t)(j * kVStep), pd + (uint64_t)(j * kPStep), idesc_pv,
                                     j > 0 ? 1u : first_acc);
                } else {
#pragma unroll
                    for (int j = 0; j < kSteps; ++j) {
                        const uint32_t acc = j > 0 ? 1u : first_acc;
                        const int pblk = pos0 + kStepPos * j;
                        int tile;
                        if (pblk >= vs && pblk + kStepPos <= ve) tile = 0;
                        else if (pblk + kStepPos <= vs || pblk >= ve) tile = 1;
                        else if ((vs & ~(kStepPos - 1)) == pblk) tile = 2;
                        else tile = 3;
                        mma_ss<kFp8>(tm_o, vd + (uint64_t)(j * kVStep), pd + (uint64_t)(j * kPStep), idesc_pv, acc);
                        mma_ss<kFp8>(tm_l, a2d0 + (uint64_t)(tile * (kA2Bytes >> 4)),
                                     pd + (uint64_t)(j * kPStep), idesc_sum, acc);
                    }
                }
                if (elect_one()) {
                    mma_commit(v_empty(vsl));
                    mma_commit(bar1 + 8 * (3 * kHand + hand.idx));     // p_free of tile i
                }
                __syncwarp();
                LVSPEC_TILE_TS(tile_tr, 2, i, 3);     // sums and P.V issued
            }
            // the elected lane's MMAs have finished: tell the softmax warps and the TMEM owner
            if (elect_one()) {
                mma_commit(pv_done);
                mma_commit(done_bar);
            }
            __syncwarp();
        }
    } else {
        // ------------------------------------------------------------ softmax warps
        // (read while nothing else is to be done: the first S^T is a tile's load and products away)
        if (kMerge && warp == kSoftmaxWarp0 && lane == 0)
            *doubt_s = *static_cast<volatile uint32_t *>(p.status) & LVSPEC_DEV_WAIT_EXPIRED;
        const int grp = (warp - kSoftmaxWarp0) >> 2;    // tiles grp, grp + 3, ... are this group's
        const int bar_id = 1 + grp;
        const int wq = warp & 3;                        // TMEM lane quarter of this warp
        const int row = wq * 32 + lane;                 // TMEM lane = position inside the tile
        const int gtid = ((warp - kSoftmaxWarp0) & 3) * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(wq * 32) << 16;
        const float scale = scale_cta;
        constexpr float kLimit = kFp8 ? kGuard8 : kGuard;    // a score this far above m moves m
        constexpr float kLift = kFp8 ? kHead8 : 0.f;         // where the reference position sits above m
        // this group's share of the columns (all tiles without turns; the epilogue always):
        // chunks of 8 columns [c_lo, c_hi), equal shares, at most kMaxChunks
        const int c_base = n8 / kSoftmaxGroups, c_rem = n8 - c_base * kSoftmaxGroups;
        const int c_lo = grp * c_base + min(grp, c_rem), c_hi = c_lo + c_base + (grp < c_rem ? 1 : 0);
        if constexpr (kTurns) {
            // bounded wait for a shared-memory counter to reach a value (the groups' turns)
            auto wait_counter = [&](volatile uint32_t *ctr, uint32_t at_least) {
                if (*ctr >= at_least) return;
                uint64_t t0 = 0;
                for (uint32_t spin = 1;; ++spin) {
                    if (*ctr >= at_least || *abort_flag) return;
                    if ((spin & 1023u) == 0) {
                        const uint64_t now = global_timer_ns();
                        if (t0 == 0) t0 = now;
                        else if (now - t0 > 2000000000ull) {
                            *abort_flag = 1;
                            return;
                        }
                    }
                }
            };
            // buffers of this group's tile advance by counting, not by dividing
            int sbi = grp % cfg.sb, pb = grp % cfg.pb;
            auto advance = [](int &idx, int n) {
                idx += kSoftmaxGroups;
                while (idx >= n) idx -= n;
            };
            // E4M3 has 17 binades, so the reference exponent of a row starts from the largest score
            // of the split's first tile, not from whatever score its first position happens to
            // have: all groups take a share of the columns (the last barrier keeps a group that is
            // late from meeting the hand-over barrier of tile 0 two phases on)
            {
                mbar_wait(s_full(0), 0, abort_flag);
                tc_fence_after();
                const int pos = t_begin * kTilePos + row;
                const Seen seen = seen_by(t_begin * kTilePos + kTilePos > L - gamma ? pos - L + gamma : -1, G, gamma, p.branch_len);
#pragma unroll 1
                for (int c8 = grp; c8 < n8; c8 += kSoftmaxGroups) {
                    uint32_t r[8];
                    tmem_ld_x8(tm_s0 + lane_addr + c8 * 8, r);
                    tmem_wait_ld();
                    float s2[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) s2[k] = warp_max_f32(seen(c8 * 8 + k) ? __uint_as_float(r[k]) * scale : -INFINITY);
                    if (lane == 0) {
                        float *dst = tmx_s + wq * NP + c8 * 8;
                        *reinterpret_cast<float4 *>(dst) = make_float4(s2[0], s2[1], s2[2], s2[3]);
                        *reinterpret_cast<float4 *>(dst + 4) = make_float4(s2[4], s2[5], s2[6], s2[7]);
                    }
                }
                asm volatile("bar.sync %0, %1;" ::"r"(kQBarrier), "r"(kSoftmaxThreads) : "memory");
                for (int n = tid - 32 * kSoftmaxWarp0; n < n8 * 8; n += kSoftmaxThreads)
                    m_s[n] = fmaxf(kMFloor, fmaxf(fmaxf(tmx_s[n], tmx_s[NP + n]),
                                                  fmaxf(tmx_s[2 * NP + n], tmx_s[3 * NP + n])) - kLift);
                asm volatile("bar.sync %0, %1;" ::"r"(kQBarrier), "r"(kSoftmaxThreads) : "memory");
            }
            for (int i = grp; i < T; i += kSoftmaxGroups) {
                const int pos0 = (t_begin + i) * kTilePos;
                const int pos = pos0 + row;
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 0);     // starts waiting for S^T
                mbar_wait(s_full(i), hand_parity(i), abort_flag);
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 1);     // S^T there
                tc_fence_after();
                const uint32_t s_addr = tm_s0 + sbi * NP + lane_addr;
                // The oldest uncommitted tile is the one whose group may move m.  Tile 0 is that
                // from the start; the others read m under an epoch and check it when their turn
                // comes.
                bool my_turn = i == 0;
                uint32_t e0 = 0;
                if (i > 0) {
                    e0 = *epoch_s;
                    __threadfence_block();
                }
                const bool tail = pos0 + kTilePos > L - gamma;
                const Seen seen = seen_by(tail ? pos - L + gamma : -1, G, gamma, p.branch_len);
                // P^T goes straight to shared memory: the P.V product that read this buffer last is done
                // (tile i - pb).  This wait stays ahead of those for tile i - 1 below: see kRound.
                if (i >= cfg.pb) mbar_wait(p_free(i - cfg.pb), hand_parity(i - cfg.pb), abort_flag);
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 2);     // P buffer free
                uint8_t *prow = gbase + sm.p + pb * (NP * 256) + row * 16;

                for (int attempt = 0; attempt < 3; ++attempt) {
                    const float gmax = !tail ? softmax_pass<false>(s_addr, n8, m_s, scale, seen, prow,
                                                             warp == kSoftmaxWarp0 ? tile_tr : nullptr, i)
                                     : softmax_pass<true>(s_addr, n8, m_s, scale, seen, prow, nullptr, i);
                    if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 3);     // exponentials done
                    if (!my_turn) {
                        wait_counter(committed_s, (uint32_t)i);
                        my_turn = true;
                        __threadfence_block();
                        const uint32_t e1 = *epoch_s;       // final: only this group can move m now
                        const bool stale = e1 != e0;
                        if (!group_any(bar_id, stale || gmax > kLimit)) break;
                        // m moved while some thread computed under the old one: once more
                        if (group_any(bar_id, stale)) continue;
                    } else if (!group_any(bar_id, gmax > kLimit)) {
                        break;
                    }

                    // ---- a score ran past the guard: move m up to the tile maximum ----
                    // (the masked form only where the tile reaches the draft slots)
                    auto tile_max = [&](auto masked) {
#pragma unroll 1
                        for (int c8 = 0; c8 < n8; ++c8) {
                            uint32_t r[8];
                            tmem_ld_x8(s_addr + c8 * 8, r);
                            tmem_wait_ld();
                            // eight reductions in flight, then their results stored
                            float s2[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                s2[k] = __uint_as_float(r[k]) * scale;
                                if constexpr (decltype(masked)::value) {
                                    if (!seen(c8 * 8 + k))
                                        s2[k] = -INFINITY;
                                }
                            }
#pragma unroll
                            for (int k = 0; k < 8; ++k) s2[k] = warp_max_f32(s2[k]);
                            if (lane == 0) {
                                float *dst = tmx_s + wq * NP + c8 * 8;
                                *reinterpret_cast<float4 *>(dst) = make_float4(s2[0], s2[1], s2[2], s2[3]);
                                *reinterpret_cast<float4 *>(dst + 4) = make_float4(s2[4], s2[5], s2[6], s2[7]);
                            }
                        }
                    };
                    if (tail) tile_max(std::true_type{});
                    else tile_max(std::false_type{});
                    group_sync(bar_id);
                    for (int n = gtid; n < n8 * 8; n += 128) {
                        const float mt = fmaxf(fmaxf(tmx_s[n], tmx_s[NP + n]),
                                               fmaxf(tmx_s[2 * NP + n], tmx_s[3 * NP + n])) - kLift;
                        const float mo = m_s[n];
                        const float mn = fmaxf(mo, mt);
                        dl_s[n] = mo - mn;              // <= 0
                        m_s[n] = mn;
                    }
                    group_sync(bar_id);
                    if (gtid == 0) {
                        __threadfence_block();
                        *epoch_s = *epoch_s + 1;
                    }
                    if (i > 0) {
                        // O^T and the sums were accumulated under the old m: rescale them once
                        // the P.V product of tile i - 1 has finished (that of tile i - pb has: see kRound)
                        mbar_wait(p_free(i - 1), hand_parity(i - 1), abort_flag);
                        tc_fence_after();
                        // (fp8 cache: accumulator columns 2n and 2n + 1 belong to row n)
                        for (int c = 0; c < n8 * kAccCols; ++c) {
                            uint32_t r[8];
                            tmem_ld_x8(tm_o + lane_addr + c * 8, r);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                r[k] = __float_as_uint(__uint_as_float(r[k]) * ex2(dl_s[(c * 8 + k) / kAccCols]));
                            tmem_st_x8(tm_o + lane_addr + c * 8, r);
                            if (wq == 0) {
                                tmem_ld_x8(tm_l + c * 8, r);
                                tmem_wait_ld();
#pragma unroll
                                for (int k = 0; k < 8; ++k)
                                    r[k] = __float_as_uint(__uint_as_float(r[k]) * ex2(dl_s[(c * 8 + k) / kAccCols]));
                                tmem_st_x8(tm_l + c * 8, r);
                            }
                        }
                        tmem_wait_st();
                        tc_fence_before();
                    }
                    group_sync(bar_id);
                }
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 4);     // this tile's turn came and m stood
                // m stands for this tile: the next tile's group may take its turn
                if (gtid == 0) {
                    __threadfence_block();
                    *committed_s = (uint32_t)i + 1;
                }
                if (pos0 + kTilePos > L) {
                    // slots at or beyond kv_len hold whatever the cache holds: zero their V
                    // rows so that 0 * junk cannot poison the accumulators.  Once the product of
                    // tile i - 1 is done, the V slot's barrier can only be in this tile's phase.
                    if (i > 0) mbar_wait(p_free(i - 1), hand_parity(i - 1), abort_flag);
                    const int vsl = i % cfg.vs;
                    mbar_wait(v_full(vsl), (i / cfg.vs) & 1, abort_flag);
                    if (pos >= L) {
                        uint8_t *vrow = gbase + sm.v + vsl * kSlot + row * 128;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            *reinterpret_cast<uint4 *>(vrow + c * 16) = make_uint4(0, 0, 0, 0);
                            if (two_boxes) *reinterpret_cast<uint4 *>(vrow + kBoxBytes + c * 16) = make_uint4(0, 0, 0, 0);
                        }
                    }
                }
                // one arrival per warp: S^T has been read (the K.Q^T of a later tile may overwrite
                // it) and P^T, with any zeroed V rows, is in shared memory
                tc_fence_before();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(s_free(i));
                    mbar_arrive(p_full(i));
                }
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 5);     // P^T handed over
                advance(sbi, cfg.sb);
                advance(pb, cfg.pb);
            }
        } else {
            // Tiles go through in twos where the buffers allow and the stream is long (256
            // positions): one vote on the guard, one fence and one hand-over for both.
            // Ring positions advance by counting, not by dividing.
            int sbi = 0, pb = 0;                 // S^T buffer and P buffer of tile i
            const uint64_t neg_scale2 = pack_f32x2(__float_as_uint(-scale), __float_as_uint(-scale));
            if (!kFp8) {
                // reference exponent of each row: its score at the split's first position
                mbar_wait(s_full(0), 0, abort_flag);
                tc_fence_after();
                if (wq == 0) {
                    for (int c8 = c_lo; c8 < c_hi; ++c8) {
                        uint32_t r[8];
                        tmem_ld_x8(tm_s0 + lane_addr + c8 * 8, r);
                        tmem_wait_ld();
                        if (lane == 0) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) m_s[c8 * 8 + k] = __uint_as_float(r[k]) * scale - kLift;
                        }
                    }
                }
                group_sync(bar_id);
            }
            for (int i = 0; i < T; i += step) {
                const int n_sub = min(step, T - i);
                int sb_u, pb_u;
                for (int attempt = 0; attempt < 3; ++attempt) {
                    // fp8 cache: E4M3 has 17 binades, so the reference exponent of a row starts
                    // from the largest score of the split's first tile (the path below), not
                    // from whatever score its first position happens to have
                    const bool first_max = kFp8 && i == 0 && attempt == 0;
                    float gmax = -INFINITY;
                    uint32_t pmax = 0u;
                    sb_u = sbi;
                    pb_u = pb;
#pragma unroll 1
                    for (int u = 0; u < n_sub; ++u) {
                        const int iu = i + u;
                        const int pos0 = (t_begin + iu) * kTilePos;
                        if (!kFp8 || attempt == 0 || iu == 1) {     // (a phase that is over is over at once)
                            if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, iu, 0);     // starts waiting for S^T
                            mbar_wait(s_full(iu), hand_parity(iu), abort_flag);
                            if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, iu, 1);     // S^T there
                            tc_fence_after();
                        }
                        const uint32_t s_addr = tm_s0 + sb_u * NP + lane_addr;
                        if (first_max) break;
                        const bool tail = pos0 + kTilePos > L - gamma;
                        Seen seen = {0, 0xFFFFFFFFu};
                        if (tail) seen = seen_by(pos0 + row - L + gamma, G, gamma, p.branch_len);
                        uint8_t *prow = gbase + sm.p + pb_u * (NP * 256) + row * 16;
                        // P^T goes straight to shared memory, once the P.V product that read this buffer is done
                        if (attempt == 0 && iu >= cfg.pb) mbar_wait(p_free(iu - cfg.pb), hand_parity(iu - cfg.pb), abort_flag);
                        if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, iu, 2);     // P buffer free
                        if constexpr (kFp8) {
                            uint4 pk[kC];   // this position's probabilities, 8 columns per entry
                            gmax = fmaxf(gmax,
                                !tail ? softmax_pass_share<false, kC>(s_addr, c_lo, c_hi, m_s, scale, seen, pk)
                                      : softmax_pass_share<true, kC>(s_addr, c_lo, c_hi, m_s, scale, seen, pk));
#pragma unroll
                            for (int j = 0; j < kC; ++j)
                                if (c_lo + j < c_hi) *reinterpret_cast<uint4 *>(prow + (c_lo + j) * 2048) = pk[j];
                        } else if (!tail) {
                            softmax_share_bf16<false, kC>(s_addr + c_lo * 8, c_hi - c_lo, m_s + c_lo * 8, neg_scale2, seen, c_lo * 8,
                                                          prow + c_lo * 2048, pmax);
                        } else {
                            softmax_share_bf16<true, kC>(s_addr + c_lo * 8, c_hi - c_lo, m_s + c_lo * 8, neg_scale2, seen, c_lo * 8,
                                                         prow + c_lo * 2048, pmax);
                        }
                        if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, iu, 3);     // probabilities stored
                        if (++sb_u == cfg.sb) sb_u = 0;
                        if (++pb_u == cfg.pb) pb_u = 0;
                    }
                    const bool beyond = kFp8 ? gmax > kLimit : (pmax & 0xFFFFu) > kGuardBits || (pmax >> 16) > kGuardBits;
                    if (!first_max && !group_any(bar_id, beyond)) break;

                    // ---- a score ran past the guard: move m up to these tiles' maximum (fp8: first
                    // to the first tile's) ----
                    for (int u = 0; u < (first_max ? 1 : n_sub); ++u) {
                        const int pos0 = (t_begin + i + u) * kTilePos;
                        const bool tail = pos0 + kTilePos > L - gamma;
                        const Seen seen = seen_by(tail ? pos0 + row - L + gamma : -1, G, gamma, p.branch_len);
                        const int sbu = sbi + u < cfg.sb ? sbi + u : sbi + u - cfg.sb;
                        const uint32_t s_addr = tm_s0 + sbu * NP + lane_addr;
                        for (int c8 = c_lo; c8 < c_hi; ++c8) {
                            uint32_t r[8];
                            tmem_ld_x8(s_addr + c8 * 8, r);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                float s2 = __uint_as_float(r[k]) * scale;
                                if (tail && !seen(c8 * 8 + k))
                                    s2 = -INFINITY;
                                s2 = warp_max_f32(s2);
                                if (lane == 0) {
                                    float *dst = tmx_s + wq * NP + c8 * 8 + k;
                                    *dst = u == 0 ? s2 : fmaxf(*dst, s2);
                                }
                            }
                        }
                    }
                    group_sync(bar_id);
                    for (int n = c_lo * 8 + gtid; n < c_hi * 8; n += 128) {
                        const float mt = fmaxf(fmaxf(tmx_s[n], tmx_s[NP + n]),
                                               fmaxf(tmx_s[2 * NP + n], tmx_s[3 * NP + n])) - kLift;
                        const float mo = m_s[n];
                        const float mn = fmaxf(mo, mt);
                        dl_s[n] = mo - mn;              // <= 0
                        m_s[n] = mn;
                    }
                    group_sync(bar_id);
                    if (i > 0) {
                        // O^T and the sums were accumulated under the old m: rescale this
                        // group's columns once PV(i-1) has finished
                        mbar_wait(p_free(i - 1), hand_parity(i - 1), abort_flag);
                        tc_fence_after();
                        // (fp8 cache: accumulator columns 2n and 2n + 1 belong to row n)
                        for (int c = c_lo * kAccCols; c < c_hi * kAccCols; ++c) {
                            uint32_t r[8];
                            tmem_ld_x8(tm_o + lane_addr + c * 8, r);
                            tmem_wait_ld();
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                r[k] = __float_as_uint(__uint_as_float(r[k]) * ex2(dl_s[(c * 8 + k) / kAccCols]));
                            tmem_st_x8(tm_o + lane_addr + c * 8, r);
                            if (wq == 0) {
                                tmem_ld_x8(tm_l + c * 8, r);
                                tmem_wait_ld();
#pragma unroll
                                for (int k = 0; k < 8; ++k)
                                    r[k] = __float_as_uint(__uint_as_float(r[k]) * ex2(dl_s[(c * 8 + k) / kAccCols]));
                                tmem_st_x8(tm_l + c * 8, r);
                            }
                        }
                        tmem_wait_st();
                        tc_fence_before();
                    }
                    group_sync(bar_id);
                }
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 4);     // the group agrees: no rescale
                if (grp == 0 && (t_begin + i + n_sub) * kTilePos > L) {
                    // slots at or beyond kv_len hold whatever the cache holds: zero their V
                    // rows so that 0 * junk cannot poison the accumulators (they sit in the last tile)
                    const int last = i + n_sub - 1, vz = last % cfg.vs, vr = last / cfg.vs;
                    // The slot's tile before is done with.  This group has waited for the products of
                    // all tiles up to last - pb before it wrote to their P^T buffers; only a V ring shorter
                    // than the P^T ring may hold a later one.  (A parity tells a phase from its neighbours
                    // only: the barrier of an older tile may be two phases on, and a wait there would
                    // not end.)
                    const int before = last - cfg.vs;
                    if (cfg.vs < cfg.pb && before >= 0) mbar_wait(p_free(before), hand_parity(before), abort_flag);
                    mbar_wait(v_full(vz), vr & 1, abort_flag);
                    if ((t_begin + last) * kTilePos + row >= L) {
                        uint8_t *vrow = gbase + sm.v + vz * kSlot + row * 128;
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            *reinterpret_cast<uint4 *>(vrow + c * 16) = make_uint4(0, 0, 0, 0);
                            if (two_boxes) *reinterpret_cast<uint4 *>(vrow + kBoxBytes + c * 16) = make_uint4(0, 0, 0, 0);
                        }
                    }
                }
                // one arrival per warp: S^T has been read (later K.Q^T may overwrite it) and P^T,
                // with any zeroed V rows, is in shared memory
                tc_fence_before();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    // (with one K slot the next K.Q^T goes first: the slot's load hangs on it)
                    if (cfg.ks > 1) mbar_arrive(p_full(i));
                    mbar_arrive(s_free(i));
                    if (n_sub == 2) mbar_arrive(s_free(i + 1));
                    if (cfg.ks == 1) mbar_arrive(p_full(i));
                }
                if (warp == kSoftmaxWarp0) LVSPEC_TILE_TS(tile_tr, 0, i, 5);     // P^T stored and handed over
                sbi = sb_u;
                pb = pb_u;
            }
        }

        // ---------------------------------------------------------------- epilogue
        // (every group takes its share of the columns)
        // (what the merge needs to know is worked out ahead of the wait for the last product)
        const int n_eff = min(p.n_split, n_tiles);        // splits with a tile of their own
        const Share share(p, P.cfg.split_magic, split, n_eff);
        const int shift = share.shift, rows = share.rows, each = (n_eff + (1 << shift) - 1) >> shift;   // each: splits of a warp
        const int w = warp - kSoftmaxWarp0, slot = w >> shift, part = w & ((1 << shift) - 1);
        const MergePart merge_part(p, P.cfg.group_magic, b, kvh, share.r0 + slot, n_eff, part, 1 << shift, lane);
        // the last P.V product has finished (and with it all before)
        mbar_wait(pv_done, 0, abort_flag);
        tc_fence_after();
        if (p.n_split == 1) {
            // a single split: nothing to merge, normalise and write the results here
            if (wq == 0) {
                for (int c8 = c_lo; c8 < c_hi; ++c8) {
                    float lsum[8];
                    load_acc8<kFp8>(tm_l, c8, lsum);      // lane 0: l, lane 1: l_vis
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int n = c8 * 8 + k;
                        const float lv = __shfl_sync(0xffffffffu, lsum[k], 1);
                        if (lane == 0 && n < M) {
                            const float inv = 1.f / lsum[k];
                            dl_s[n] = inv * v_scale;
                            const int g = n / G, hg = n - g * G;
                            p.mass[((size_t)b * gamma + g) * p.Hq + kvh * G + hg] = lv * inv;
                        }
                    }
                }
            }
            group_sync(bar_id);
            __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(p.out);
            for (int c8 = c_lo; c8 < c_hi; ++c8) {
                float o8[8];
                load_acc8<kFp8>(tm_o + lane_addr, c8, o8);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int n = c8 * 8 + k;
                    if (n < M && row < D) {
                        const int g = n / G, hg = n - g * G;
                        out[(((size_t)b * gamma + g) * p.Hq + kvh * G + hg) * D + row] =
                            __float2bfloat16_rn(o8[k] * dl_s[n]);
                    }
                }
            }
        } else {
            // This code runs once, on cold instruction caches, where every instruction
            // costs about ten cycles: short rolled loops, one chunk of 8 columns a turn;
            // only a last chunk that is not full takes the guarded path.
            // (TMEM lanes are channels: at head_dim 64 the upper half of the lanes holds nothing)
            float *po = part_o + (size_t)c_lo * 8 * D + row;
            const int m_store = row < D ? M : 0;
#pragma unroll 1
            for (int c8 = c_lo; c8 < c_hi; ++c8, po += 8 * D) {
                float o8[8];
                load_acc8<kFp8>(tm_o + lane_addr, c8, o8);
                if (kFp8) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) o8[k] *= v_scale;
                }
                auto put = [&](int k) {
                    if constexpr (kMerge) st_relaxed(po + k * D, passable(o8[k]));
                    else po[k * D] = o8[k];
                };
                if (c8 * 8 + 8 <= m_store) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) put(k);
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (c8 * 8 + k < m_store) put(k);
                }
            }
            if (wq == 0) {
#pragma unroll 1
                for (int c8 = c_lo; c8 < c_hi; ++c8) {
                    float lsum[8];
                    load_acc8<kFp8>(tm_l, c8, lsum);      // lane 0: l, lane 1: l_vis
                    // lane k takes column k of the chunk: l from lane 0, l_vis from lane 1
                    float lk = 0.f, lvk = 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float a = __shfl_sync(0xffffffffu, lsum[k], 0);
                        const float c = __shfl_sync(0xffffffffu, lsum[k], 1);
                        if (lane == k) { lk = a; lvk = c; }
                    }
                    if (lane < 8 && c8 * 8 + lane < M) {
                        const float mk = m_s[c8 * 8 + lane];
                        float *ps = part_stat + (c8 * 8 + lane) * 4;
                        if constexpr (kMerge) st_relaxed_v4(ps, make_uint4(passable(mk), passable(lk), passable(lvk), 0u));
                        else *reinterpret_cast<float4 *>(ps) = make_float4(mk, lk, lvk, 0.f);
                    }
                }
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(done_bar);

        if (merges()) {
            // ------------------------------------------------------------ merge
            float4 *sums = reinterpret_cast<float4 *>(gbase + sm.k);   // the rings are empty by now
            volatile uint32_t *verdict = epoch_s;
            unsigned long long *word = p.merge_word + bh;
            bool mine, doubt = w == 0 && lane == 0 && *doubt_s != 0u;
            uint64_t since = 0;
            for (;;) {
                MergedRow res;
                const bool got = slot >= rows ||
                    (each <= 4 ? merge_row<4>(p, merge_part, lane, p.merge_polls, res)
                     : each <= 8 ? merge_row<8>(p, merge_part, lane, p.merge_polls, res)
                                 : merge_row<12>(p, merge_part, lane, p.merge_polls, res));
                if (part > 0 && slot < rows) sums[w * 32 + lane] = res.o;
                uint32_t late;
                asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %2, 0;\n\tbar.red.or.pred p, %1, %3, q;\n\t"
                             "selp.u32 %0, 1, 0, p;\n\t}"
                             : "=r"(late) : "r"(kQBarrier), "r"((uint32_t)(!got || doubt)), "n"(kSoftmaxThreads) : "memory");
                mine = true;
                if (!late) {
                    if (part == 0 && slot < rows) {
                        for (int k = 1; k < (1 << shift); ++k) {
                            const float4 o = sums[(w + k) * 32 + lane];
                            res.o.x += o.x; res.o.y += o.y; res.o.z += o.z; res.o.w += o.w;
                        }
                        write_row(p, merge_part, lane, res);
                    }
                    break;
                }
                // Some split's CTA is late, or not even running (the GPU is shared with another grid): this
                // CTA leaves its share to the head's last one to arrive, unless that one has arrived.
                // Its own arrival comes first, so that a count of zero can only mean that all have and
                // the word is the next call's again.
                if (w == 0 && lane == 0) {
                    uint32_t keep = 1u;
                    if (*arrived_s) {
                        __threadfence_block();      // with the one ahead of arrived_s: this CTA's arrival is in the word
                        const unsigned long long bit = 1ull << (32 + split);
                        const uint32_t arrived = (uint32_t)atomicOr(word, bit);
                        if (arrived == 0) atomicAnd(word, ~bit);
                        keep = arrived == 0 || arrived >= (uint32_t)n_eff ? 1u : 0u;
                        if (!keep) atomicAdd(p.merge_word + kMergeCountWord, 1ull);
                        else doubt = false;            // every word there is from this launch now
                    }
                    if (keep && *abort_flag == 0) {
                        // (the data are there or on their way: a bound all the same)
                        const uint64_t now = global_timer_ns();
                        if (since == 0) since = now;
                        else if (now - since > 2000000000ull) *abort_flag = 1;
                    }
                    if (*abort_flag) {
                        atomicOr(p.status, LVSPEC_DEV_WAIT_EXPIRED);
                        keep = 0u;
                    }
                    *verdict = keep;
                }
                asm volatile("bar.sync %0, %1;" ::"r"(kQBarrier), "r"(kSoftmaxThreads) : "memory");
                mine = *verdict != 0;
                asm volatile("bar.sync %0, %1;" ::"r"(kQBarrier), "r"(kSoftmaxThreads) : "memory");
                if (!mine) break;
            }
            if (mine && slot < rows) clear_part(p, merge_part, lane);
        }
    }

    // ------------------------------------------------------------------ teardown
    // TMEM goes back once the MMAs have drained and every softmax warp is done
    if (warp == 1) {
        if (lane == 0) {
            bool all_done = false;
#ifdef LVSPEC_TRACE
            if (rec) rec[5] = lvspec_trace_now();
#endif
            for (int tries = 0; tries < 4 && !all_done; ++tries) all_done = wait_unconditional(done_bar, 0);
#ifdef LVSPEC_TRACE
            if (rec) rec[6] = lvspec_trace_now();
#endif
            if (*abort_flag || !all_done) atomicOr(p.status, LVSPEC_DEV_WAIT_EXPIRED);
            // this CTA is done but for freeing TMEM: a dependent launch may be scheduled
            // once every CTA has come this far (earlier, its CTAs would pile up on the
            // few SMs this grid leaves idle; with the merge to come, later still)
            if (!merges()) grid_launch_dependents();
        }
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)cfg.tmem_cols);
        if (merges()) {
            // this CTA's partials are written; the head's last one to say so sees to the shares that
            // others have given up, and leaves the word as the next call expects it
            const int n_eff = min(p.n_split, n_tiles);
            unsigned long long *word = p.merge_word + bh;
            unsigned long long before = 0;
            if (lane == 0) {
                __threadfence();
                before = atomicAdd(word, 1ull);
            }
            before = __shfl_sync(0xffffffffu, before, 0);
            if ((uint32_t)before == (uint32_t)n_eff - 1u) {
#pragma unroll 1
                for (uint32_t late = (uint32_t)(before >> 32); late != 0u; late &= late - 1u) {
                    const Share share(p, P.cfg.split_magic, __ffs(late) - 1, n_eff);
                    const int parts = 1 << share.shift;
                    constexpr uint32_t kPolls = 4096;      // (all partials are there; a bound all the same)
#pragma unroll 1
                    for (int r = share.r0; r < share.r0 + share.rows; ++r) {
                        // by the same arithmetic, part after part
                        MergedRow res;
                        bool ok = true;
#pragma unroll 1
                        for (int k = 0; k < parts && ok; ++k) {
                            MergedRow of_part;
                            ok = merge_row<4>(p, MergePart(p, P.cfg.group_magic, b, kvh, r, n_eff, k, parts, lane), lane, kPolls,
                                              of_part);
                            if (k > 0) {
                                of_part.o.x += res.o.x; of_part.o.y += res.o.y; of_part.o.z += res.o.z; of_part.o.w += res.o.w;
                            }
                            res = of_part;
                        }
                        const MergePart whole(p, P.cfg.group_magic, b, kvh, r, n_eff, 0, 1, lane);
                        if (ok) {
                            write_row(p, whole, lane, res);
                            clear_part(p, whole, lane);
                        } else if (lane == 0) {
                            atomicOr(p.status, LVSPEC_DEV_WAIT_EXPIRED);
                        }
                    }
                }
                if (lane == 0) atomicExch(word, 0ull);
            }
            if (lane == 0) {
                grid_launch_dependents();
                // The arrival comes before whatever the softmax warps do to the word once they see this.  All
                // are threads of one CTA: its scope is enough (a fence for the device holds the CTA's end up,
                // 0.3 us a layer of 4K or 16K).
                __threadfence_block();
                *arrived_s = 1;
            }
#ifdef LVSPEC_TRACE
            if (rec) rec[7] = lvspec_trace_now();
#endif
        }
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        fn = reinterpret_cast<EncodeTiledFn>(sym);
    }
    return fn;
}

// A cache as a 4-D tensor [sequences or pages][heads][positions][128 channels] with the
// caller's strides (in elements; the channels are contiguous).  bf16: boxes of 64 channels
// x 128 positions; E4M3: boxes of 128 channels x 128 positions.
bool make_kv_map(CUtensorMap *map, const void *ptr, bool fp8, int D, int positions, int heads, int outer,
                 int64_t s_pos, int64_t s_head, int64_t s_outer)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t esz = fp8 ? 1 : 2;
    const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)positions, (cuuint64_t)heads, (cuuint64_t)outer};
    const cuuint64_t strides[3] = {(cuuint64_t)s_pos * esz, (cuuint64_t)s_head * esz, (cuuint64_t)s_outer * esz};
    const cuuint32_t box[4] = {fp8 ? 128u : 64u, 128, 1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, fp8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
              const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// q [B][gamma][Hq][128] bf16 as a 4-D tensor; one box = 64 channels of the G heads of one
// KV head for all gamma queries: its rows land in shared memory in the order g * G + hg
bool make_q_map(CUtensorMap *map, const void *ptr, int B, int gamma, int Hq, int G, int D)
{
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t row = (cuuint64_t)D * 2;
    const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)Hq, (cuuint64_t)gamma, (cuuint64_t)B};
    const cuuint64_t strides[3] = {row, (cuuint64_t)Hq * row, (cuuint64_t)gamma * Hq * row};
    const cuuint32_t box[4] = {64, (cuuint32_t)G, (cuuint32_t)gamma, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(ptr), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr uint32_t kMaxSmem = 232448 - 1024;   // 227 KB less the alignment slack

TcConfig pick_config(int M, int page_slots, bool fp8, bool turns, int D)
{
    TcConfig c;
    c.n_pad = (M + 15) & ~15;
    c.page_slots = page_slots;
    const bool small_tiles = fp8 || D == 64;     // one 16 KB box per tile: twice the slots
    c.slot_bytes = small_tiles ? kBoxBytes : kSlotBytes;
    const int acc = fp8 ? 4 : 2;     // TMEM columns per padded row of O^T and the sums
    if (!turns) {
        // All groups on every tile: as many S^T and P^T buffers as fit, up to two pairs, before
        // more than two ring slots each.  128 KB of K/V in flight per CTA, 16 to 19 MB on the
        // device, are enough for HBM, and more of them at the start of a launch only put later tiles
        // ahead of the first one's (40 rows, 16 tiles per CTA: 26.9 us with 2 + 2 slots,
        // 27.9 with 3 + 2 or 2 + 3).  Half-size tiles: 3 + 4 slots and two P^T buffers rather than
        // 4 + 4 and one (120 rows of 32K at head_dim 64: 33.9 us a layer, 128 rows 43.5 with one
        // buffer).  At 128 rows a second P^T buffer before a second K slot: 37.3 us a layer of
        // 32K against 47.1.
        c.sb = 512 / c.n_pad - acc;
        if (c.sb > 4) c.sb = 4;
        const int tries[5][3] = {{2, 2, 4}, {2, 2, 3}, {2, 2, 2}, {1, 2, 2}, {2, 2, 1}};
        const int tries8[5][3] = {{4, 4, 4}, {4, 4, 3}, {4, 4, 2}, {3, 4, 2}, {3, 3, 1}};
        for (int t = 0; t < 5; ++t) {
            const int *tr = small_tiles ? tries8[t] : tries[t];
            c.ks = tr[0]; c.vs = tr[1]; c.pb = tr[2];
            if (smem_map(c).total <= kMaxSmem) break;
        }
    } else {
        // Tiles in turn (fp8 cache): as many S^T buffers as TMEM has columns for, up to one more than
        // there are softmax groups: the K.Q^T of a group's next tile is then done when the group
        // comes to it.  A fourth P^T buffer too: with three a group waited for the product of its tile
        // before, which is in the queue behind two others'.  Then also more slots of 16 KB.  us a layer, by
        // K + V slots / P^T buffers / S^T buffers:
        //   40 rows of 32K: 3 + 3 / 3 / 3 19.4, 3 + 3 / 3 / 4 19.2, 3 + 3 / 4 / 4 19.0, 4 + 4 / 4 / 4 18.5, 5 + 4 / 4 / 4 18.6
        //   56 rows of 64K: 23.9, 23.7, 23.0, 23.4, does not fit
        //   80 rows of 32K (two S^T buffers): 2 + 3 / 3 30.9, 2 + 3 / 4 31.0, 3 + 3 / 3 31.2, 3 + 3 / 4 31.5
        c.sb = 512 / c.n_pad - acc;
        if (c.sb > kHand) c.sb = kHand;
        const int tries[6][3] = {{4, 4, 4}, {3, 3, 4}, {2, 3, 3}, {3, 3, 2}, {3, 3, 1}, {2, 2, 1}};
        for (int t = c.n_pad > 64 ? 2 : c.n_pad > 48 ? 1 : 0; t < 6; ++t) {
            const int *tr = tries[t];
            c.ks = tr[0]; c.vs = tr[1]; c.pb = tr[2];
            if (smem_map(c).total <= kMaxSmem) break;
        }
    }
    // LVSPEC_TC_RING="K slots,V slots,P buffers,S buffers" overrides the choice (for
    // measurements; a combination that does not fit is refused by the launch)
    if (const char *e = std::getenv("LVSPEC_TC_RING")) {
        int ks, vs, pb, sb;
        if (std::sscanf(e, "%d,%d,%d,%d", &ks, &vs, &pb, &sb) == 4 && ks >= 1 && ks <= 8 && vs >= 1 && vs <= 8 &&
            pb >= 1 && sb >= 2 && pb <= kHand && sb <= kHand) {
            c.ks = ks; c.vs = vs; c.pb = pb; c.sb = sb;
        }
    }
    // Two tiles per hand-over need S^T and P^T buffers for the tiles after them too (with two
    // S^T buffers the K.Q^T of the next pair waits for this one: 112 padded rows, 128-frame
    // tree, 36.8 us a layer in pairs against 34.9 one by one), and a V ring that holds a pair.
    // In a short stream the first tile's product waits for the second tile to arrive, and
    // the last pair's products run when nothing else does: us a layer one by one / in pairs,
    // 20 rows: 8 tiles (batch 16) 18.6 / 19.2; 40 rows: 2 10.3 / 10.7, 12 22.7 / 23.0, 16 26.7 / 27.3; 56 rows:
    // 2 tiles 11.1 / 11.3, 7 or 8 19.4 / 19.7; 80 rows: 2 tiles 12.3 / 12.7, 7 or 8 20.2 / 20.0,
    // several hundred 347 / 331.  Half-size tiles (32 rows): 2 11.9 / 12.0, 4 14.1 / 13.7, 7 18.1 / 17.4.
    c.step = !turns && c.sb >= 4 && c.pb >= 2 && c.vs >= 2 ? 2 : 1;
    c.pair_from = small_tiles ? 3 : c.n_pad > 64 ? 5 : 17;
    int cols = 32;
    while (cols < (c.sb + acc) * c.n_pad) cols <<= 1;
    c.tmem_cols = cols;
    return c;
}

}  // namespace

bool attn_tc_supported(const AttnParams &p)
{
    if (p.fp8 && (p.M > kMaxRowsFp8 || p.page_size > 0 || p.branch_len != p.gamma)) return false;
    return (p.D == 128 || (p.D == 64 && !p.fp8)) && p.Lmax >= kTilePos && p.M <= LVSPEC_MAX_ROWS;
}

cudaError_t launch_attn_tc(const AttnParams &p, const SeqInfo &seq, cudaStream_t stream, int *launches)
{
    TcParams P;
    P.a = p;
    const bool paged = p.page_size > 0;
    // paged: one block-table entry per tile of the longest split, rounded up to 4
    const int tiles = (p.Lmax + kTilePos - 1) / kTilePos;
    const bool fp8 = p.fp8 != 0;
    // Tiles in turn with an fp8 cache (half the bytes per tile for the same work: 18.4 us a layer
    // at 40 rows of 32K against 23.5 with shared columns, 30.6 against 34.3 at 80).  A bf16
    // cache goes through with shared columns, in pairs of tiles where that pays, which beats
    // turns at every length (long streams of 80 rows: 321 us against 331).
    // LVSPEC_TC_TURNS=0/1 overrides the choice with an fp8 cache (for measurements).
    bool turns = fp8;
    if (const char *e = fp8 ? std::getenv("LVSPEC_TC_TURNS") : nullptr)
        if (e[0] == '0' || e[0] == '1') turns = e[0] == '1';
    P.cfg = pick_config(p.M, paged ? ((tiles + p.n_split - 1) / p.n_split + 4) & ~3 : 0, fp8, turns, p.D);
    P.cfg.split_magic = magic_of((uint32_t)p.n_split);
    P.cfg.group_magic = magic_of((uint32_t)p.G);
    if (smem_map(P.cfg).total > kMaxSmem || P.cfg.tmem_cols > 512) return cudaErrorInvalidConfiguration;
    P.sm = smem_map(P.cfg);
    CUtensorMap mk, mv, mq;
    const int map_len = paged ? p.page_size : p.Lmax;
    const int map_outer = paged ? p.n_pages : p.B;
    if (!make_kv_map(&mk, p.k, fp8, p.D, map_len, p.Hkv, map_outer, p.k_sp, p.k_sh, p.k_sb) ||
        !make_kv_map(&mv, p.v, fp8, p.D, map_len, p.Hkv, map_outer, p.v_sp, p.v_sh, p.v_sb))
        return cudaErrorInvalidValue;
    if (fp8) mq = mk;     // not used by the kernel
    else if (!make_q_map(&mq, p.q, p.B, p.gamma, p.Hq, p.G, p.D)) return cudaErrorInvalidValue;
    const size_t smem = smem_map(P.cfg).total + 1024;
    const bool tree = p.branch_len != p.gamma;
    if ((tree && paged) || (fp8 && (tree || paged))) return cudaErrorNotSupported;
    const int share = ((p.M + 7) / 8 + kSoftmaxGroups - 1) / kSoftmaxGroups;    // column chunks of a softmax group
    auto kernel = fp8 ? (turns ? attn_tc_kernel<true, true, 1, true> : attn_tc_kernel<true, false, 4, true>)
                  : p.merge ? (share <= 2 ? attn_tc_kernel<false, false, 2, true>
                               : share <= 4 ? attn_tc_kernel<false, false, 4, true> : attn_tc_kernel<false, false, kMaxChunks, true>)
                  : share <= 2 ? attn_tc_kernel<false, false, 2, false>
                  : share <= 4 ? attn_tc_kernel<false, false, 4, false> : attn_tc_kernel<false, false, kMaxChunks, false>;
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.n_split, p.Hkv, p.B);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.pdl ? 1 : 0;
    err = cudaLaunchKernelEx(&cfg, kernel, P, seq, mk, mv, mq);
    ++*launches;
    return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace lvspec
