// Tensor-core split-KV attention core over the latent cache for sm_103a
// (Eqs. 2-4 with the Sec. 3.3 score routing, in the absorbed form).
//
// One CTA = (one partition of the tile list, one group of N query rows).  Per
// 128-token tile, with tokens on the MMA's M dimension and query rows on N:
//     S^T [128 tok, N] = [k_rope | c] tile (K-major A) x q_abs^T (K-major B)
//     online softmax over tokens (TMEM lane = token, column = query row)
//     O^T [r, N]      += C^T (latent tile read as an MN-major A) x P^T
// S^T (two buffers) and O^T live in TMEM.  The cache streams through two
// rings of 64-column chunks: the QK ring (positional keys, then the latent
// chunks of each tile) feeds the score products, the PV ring (the latent
// chunks again, from L2) the value products, so that the softmax of tile t
// overlaps QK(t+1) and PV(t-1).  More than 80 query rows run as several
// independent CTAs per partition, each loading the cache boxes itself (the
// later ones hit in L2).  A sequence's last, partial tile issues only
// the value products of its 16-token steps that hold cached rows; the PV warp
// clears the rows past the end inside the last such step itself.
//
// Warp roles (512 threads): warps 0 and 3 = TMA producers (QK ring and query
// boxes; PV ring), warp 1 = QK MMA issuer and TMEM owner, warp 2 = PV MMA
// issuer, warps 4..15 = softmax / epilogue (three warps per TMEM lane quarter,
// each owning every third 16-column block of the query columns).  Every wait
// is bounded; a wait that runs out records a timeout in the status word and
// the CTA winds down without trapping.
#include <cudaTypedefs.h>
#include <math.h>
#include <stdlib.h>

#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace gbmla {
namespace {

constexpr int kTile = MLA_SPLIT_TILE;     // tokens per tile (MMA M)
constexpr int kHalf = 64;                 // tokens per TMA box (one page when paged)
constexpr int kChunkBytes = kTile * 128;  // 128 tokens x 64 bf16 columns, SW128 K-major
constexpr int kMaxSlots = 16;               // ring slots of both rings together
constexpr int kSoftmaxWarps = 12;
constexpr int kWhole = 1 << 30;             // flag bit beside a sequence index (batch < 2^30)
constexpr int kSoftmaxBase = 128;           // first softmax thread (after two producer and two MMA warps)
constexpr int kThreads = kSoftmaxBase + 32 * kSoftmaxWarps;

// P buffers: two, so that the softmax of tile t overlaps PV(t-1).  (With
// streamed queries an 80-row CTA has the room; with resident ones it then
// keeps only five ring slots.)
template <int N>
constexpr int kPBufs = 2;

// O^T buffers in TMEM: two where they fit beside the two S^T buffers (2N + 2 x 4N
// columns <= 512, i.e. N <= 48), so that a sequence's value products start in
// one while the previous sequence's partial drains from the other; else one.
template <int N>
constexpr int kOBufs = 10 * N <= 512 ? 2 : 1;
template <int N>
constexpr uint32_t kTmemCols = (2 * N + kOBufs<N> * 4 * N) <= 128 ? 128u
                               : (2 * N + kOBufs<N> * 4 * N) <= 256 ? 256u : 512u;


struct TcArgs {
    int batch, q_len, heads, rank, d_rope, rows, num_splits, max_kv;
    int paged, bt_stride, num_pages, qk_slots, pv_slots;
    float scale_log2;
    const int32_t *kv_len;
    const int32_t *block_table;
    float *o_part, *lse_part;
    // or NULL: a sequence whose tiles all lie in one partition writes its
    // (final) output and log-sum-exp here, at row b of [B, rows, ...], instead
    // of its partial slot (the combine then leaves that sequence alone)
    float *o_final, *lse_final;
    unsigned *status;
    uint64_t wait_ns;
};

struct __align__(8) Bars {
    uint64_t qk_full[kMaxSlots], qk_empty[kMaxSlots];  // QK ring: positional keys + latent chunks
    uint64_t pv_full[kMaxSlots], pv_empty[kMaxSlots];  // PV ring: latent chunks again
    uint64_t q_full, q_free;
    uint64_t s_full[2], s_free[2];
    uint64_t p_full[2], pv_done[2];  // per P buffer (t % NP): P(t) published / PV(t) completed
    uint64_t o_free, drain_qk, drain_pv;  // o_free: O^T buffer 0 drained
};

// With two O^T buffers, the barrier of the second.  (A kernel with one buffer
// keeps the plain layout: one more member there changed its register
// allocation enough to spill.)
struct BarsO2 : Bars {
    uint64_t o_free1;
};
template <int N>
using BarsT = std::conditional_t<kOBufs<N> == 2, BarsO2, Bars>;

template <class B>
__device__ __forceinline__ uint64_t *o_free_bar(B &b, int i)
{
    if constexpr (std::is_same_v<B, BarsO2>)
        return i ? &b.o_free1 : &b.o_free;
    else
        return &b.o_free;
}

template <int N>
struct Shared {
    float red[4][N];   // per TMEM-quadrant column partials
    alignas(16) float neg_m[N];  // minus the exponent base of each query column (0 while it has none)
    float m_used[N];   // exponent base of each query column (log2 domain; -inf: no key seen)
    float alpha[N];    // rescale factor of the current tile
    float lsum[N];     // softmax denominators at the epilogue (one O^T buffer)
    float inv_l[N];    // 1 / softmax denominator of the last closed sequence (two buffers)
    int lim[N];        // last visible position of each column (-1: padding column)
    int abort;         // any role gave up: producer / MMA stop issuing
    uint32_t tmem_base;
};

// The n tiles of a partition (from tile t_begin of the flattened list on),
// sequence by sequence; the same in every lane of a warp.  Tiles count from
// the partition's first.
struct Walk {
    const int32_t *kv;
    int q_len, max_kv, batch;
    int b, seq_start, nb, t, n;  // the current sequence, its first tile (negative: it began earlier) and tile count

    __device__ void init(const TcArgs &a, int64_t t_begin, int n_tiles)
    {
        kv = a.kv_len;
        batch = a.batch;
        q_len = a.q_len;
        max_kv = a.max_kv;
        t = 0;
        n = n_tiles;
        // the sequence holding tile t_begin, 32 sequences at a time (the whole warp)
        const int lane = threadIdx.x & 31;
        int64_t before = -t_begin;
        for (int b0 = 0;; b0 += 32) {
            const int64_t nt = b0 + lane < batch ? seq_tiles(kv[b0 + lane], q_len, max_kv) : 0;
            int64_t incl = nt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, before + incl > 0);
            if (hit || b0 + 32 >= batch) {
                const int src = hit ? __ffs(hit) - 1 : 31;
                b = b0 + src;
                nb = static_cast<int>(__shfl_sync(0xffffffffu, nt, src));
                seq_start = static_cast<int>(before + __shfl_sync(0xffffffffu, incl - nt, src));
                return;
            }
            before += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __device__ bool done() const { return t >= n; }
    __device__ int tile() const { return t - seq_start; }
    __device__ bool first() const { return t == 0 || t == seq_start; }
    __device__ bool last() const { return t + 1 == n || t + 1 == seq_start + nb; }
    __device__ bool last_of_partition() const { return t + 1 == n; }
    __device__ bool whole() const { return seq_start >= 0 && seq_start + nb <= n; }  // all its tiles are here
    __device__ void next()
    {
        ++t;
        if (t < n && t >= seq_start + nb) {
            seq_start += nb;
            for (++b; b < batch; ++b) {
                nb = static_cast<int>(seq_tiles(kv[b], q_len, max_kv));
                if (nb > 0) break;
            }
        }
    }
};

// Where the boxes of a tile live: a contiguous cache loads the tile as one
// 128-row box, a paged cache as one 64-row box per page.
struct TileLoc {
    int nh;            // boxes to load (0 if the first page is bad)
    uint32_t bytes;    // bytes the boxes deliver
    int32_t tok0, blk[2];
};

// The tiles of a partition in order, for a producer warp (the same in every
// lane).  Page ids are read 32 at a time, one per lane, so that no load from
// the block table stands between a free slot and its refill.
struct TileStream {
    Walk w;
    TileLoc at;
    int page_b, page_0, page_id;

    __device__ void init(const TcArgs &a, int64_t t_begin, int n_tiles)
    {
        w.init(a, t_begin, n_tiles);
        page_b = -1;
        page_0 = page_id = 0;
        locate(a);
    }
    __device__ void next(const TcArgs &a)
    {
        w.next();
        if (!w.done()) locate(a);
    }
    __device__ void locate(const TcArgs &a)
    {
        const int b = w.b, j = w.tile();
        if (!a.paged) {
            at.nh = 1;
            at.bytes = kChunkBytes;
            at.blk[0] = b;
            at.tok0 = j * kTile;
            return;
        }
        const int lane = threadIdx.x & 31;
        const int pages = (a.kv_len[b] + kHalf - 1) / kHalf;
        if (b != page_b || 2 * j + 1 >= page_0 + 32) {
            page_b = b;
            page_0 = 2 * j;
            page_id = page_0 + lane < pages ? a.block_table[static_cast<int64_t>(b) * a.bt_stride + page_0 + lane] : 0;
        }
        at.nh = pages - 2 * j > 1 ? 2 : 1;
        at.tok0 = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            at.blk[h] = __shfl_sync(0xffffffffu, page_id, 2 * j + h - page_0);
            if (h < at.nh && (at.blk[h] < 0 || at.blk[h] >= a.num_pages)) {
                if (lane == 0) record_status(a.status, kStatusBounds);
                at.nh = h;
            }
        }
        at.bytes = static_cast<uint32_t>(at.nh) * kHalf * 128;
    }
};

// A ring position: slot index and how many full passes over the ring came before.
struct RingPos {
    int slot, round;
    __device__ void advance(int cs)
    {
        if (++slot == cs) {
            slot = 0;
            ++round;
        }
    }
};

__device__ __forceinline__ void named_sync_softmax()
{
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kSoftmaxWarps) : "memory");
}

// The same barrier with a vote: does any softmax thread pass true?
__device__ __forceinline__ bool softmax_any(bool p)
{
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"(static_cast<uint32_t>(p)), "n"(32 * kSoftmaxWarps)
        : "memory");
    return r != 0;
}

// Two fp32 values in a 64-bit register, and the two-wide operations on them.
__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Sums of 16 columns over the 32 lanes of a warp: lane l gets, in v[0], the
// sum of column l % 16.
template <int CNT>
__device__ __forceinline__ void halve_step(float *v, int lane)
{
    const bool upper = (lane & CNT) != 0;
#pragma unroll
    for (int k = 0; k < CNT; ++k) {
        const float send = upper ? v[k] : v[k + CNT];
        const float keep = upper ? v[k + CNT] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, CNT);
    }
}

__device__ __forceinline__ float sum16(float (&v)[16], int lane)
{
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], 16);
    halve_step<8>(v, lane);
    halve_step<4>(v, lane);
    halve_step<2>(v, lane);
    halve_step<1>(v, lane);
    return v[0];
}

// Maxima of 16 columns over the 32 lanes: lane l < 16 gets column l's.
__device__ __forceinline__ float max16(const float (&v)[16], int lane)
{
    float mine = -INFINITY;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        float m;
        asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v[k]));
        mine = lane == k ? m : mine;
    }
    return mine;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    tc::ld_32x32b_x16(taddr, r);
    tc::wait_ld();
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16])
{
    uint32_t r[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(v[j]);
    tc::st_32x32b_x16(taddr, r);
    tc::wait_st();
}

// Where sequence b's output rows and log-sum-exps go: its partial slot b + k,
// or (whole: all its tiles in this partition, and a final buffer given) its
// final row b.
__device__ __forceinline__ float *out_rows(const TcArgs &a, int b, int part, bool whole)
{
    return whole && a.o_final ? a.o_final + static_cast<int64_t>(b) * a.rows * a.rank
                              : a.o_part + (static_cast<int64_t>(b) + part) * a.rows * a.rank;
}

__device__ __forceinline__ float *lse_rows(const TcArgs &a, int b, int part, bool whole)
{
    return whole && a.lse_final ? a.lse_final + static_cast<int64_t>(b) * a.rows
                                : a.lse_part + (static_cast<int64_t>(b) + part) * a.rows;
}

// Per-thread constants of a softmax warp.
struct SmCtx {
    int lane, tid, quarter, half, tok, n_own, group, part, nrc, n_items;
    uint32_t lane_base, tmem, o_col0;
    unsigned char *p_buf;  // NP buffers of NB x [128 tok x 32 B]
    uint64_t lim_ns;
    int64_t t_begin;
};

// The whole warp waits; once a wait has run out the warp waits no more, and the
// softmax warps leave together at their next vote (softmax_any).
__device__ __forceinline__ void sm_wait(const SmCtx &c, const TcArgs &a, int *abort, bool &failed, uint64_t *bar,
                                        uint32_t parity)
{
    if (failed || mbar_wait_warp(smem_u32(bar), parity, c.lim_ns)) return;
    failed = true;
    if (c.lane == 0) {
        record_status(a.status, kStatusTimeout);
        *abort = 1;
    }
}

// Scores of one 16-column block in the log2 domain, masked where needed.
template <int N>
__device__ __forceinline__ void sm_scores(const TcArgs &a, const Shared<N> &ss, uint32_t s_base, int cb, int pos,
                                          bool need_mask, float (&s)[16])
{
    tmem_ld16(s_base + cb * 16, s);
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        s[e] *= a.scale_log2;
        if (need_mask && pos > ss.lim[cb * 16 + e]) s[e] = -INFINITY;
    }
}

// Column maxima of the tile's scores over this warp's 32 tokens, into red[quarter].
template <int N, int KOWN>
__device__ __forceinline__ void sm_block_max(const SmCtx &c, const TcArgs &a, Shared<N> &ss, uint32_t s_base,
                                             int pos, bool need_mask)
{
#pragma unroll
    for (int ob = 0; ob < KOWN; ++ob) {
        if (ob < c.n_own) {
            const int cb = c.half + 3 * ob;
            float s[16];
            sm_scores<N>(a, ss, s_base, cb, pos, need_mask, s);
            const float mx = max16(s, c.lane);
            if (c.lane < 16) ss.red[c.quarter][cb * 16 + c.lane] = mx;
        }
    }
}

// Normalised partial output and log-sum-exp of sequence b, whose last tile
// in this partition was t_end_seg, in one step (one O^T buffer).
template <int N, int KOWN>
__device__ __forceinline__ bool sm_epilogue(const SmCtx &c, const TcArgs &a, Shared<N> &ss, Bars &bars,
                                            uint64_t (&l_part)[KOWN][8], int b, int t_end_seg, bool whole,
                                            bool &failed)
{
    sm_wait(c, a, &ss.abort, failed, &bars.pv_done[t_end_seg % kPBufs<N>], static_cast<uint32_t>((t_end_seg / kPBufs<N>) & 1));
    if (softmax_any(failed)) return false;
    tc::fence_after_sync();
#pragma unroll
    for (int ob = 0; ob < KOWN; ++ob) {
        if (ob < c.n_own) {
            const int cb = c.half + 3 * ob;
            float v[16];
#pragma unroll
            for (int e = 0; e < 8; ++e) unpack2(l_part[ob][e], v[2 * e], v[2 * e + 1]);
            const float ls = sum16(v, c.lane);
            if (c.lane < 16) ss.red[c.quarter][cb * 16 + c.lane] = ls;
        }
    }
    named_sync_softmax();
    const int cc = c.tid - kSoftmaxBase;
    if (cc < N) {
        const float l = ss.red[0][cc] + ss.red[1][cc] + ss.red[2][cc] + ss.red[3][cc];
        ss.lsum[cc] = l;
        ss.alpha[cc] = l > 0.f ? 1.f / l : 0.f;  // reused here as 1 / l
    }
    named_sync_softmax();
    const int valid_cols = a.rows - c.group * N;  // columns past it are padding
    float *out = out_rows(a, b, c.part, whole) + static_cast<int64_t>(c.group) * N * a.rank + c.tok;
    for (int m = 0; m < c.nrc; ++m) {
#pragma unroll
        for (int ob = 0; ob < KOWN; ++ob) {
            if (ob < c.n_own) {
                const int cb = c.half + 3 * ob;
                float o[16];
                tmem_ld16(c.tmem + c.lane_base + c.o_col0 + m * N + cb * 16, o);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int col = cb * 16 + e;
                    if (col < valid_cols) out[col * a.rank + m * 128] = o[e] * ss.alpha[col];
                }
            }
        }
    }
    if (cc < N) {
        const int row = c.group * N + cc;
        if (row < a.rows) {
            const float l = ss.lsum[cc];
            lse_rows(a, b, c.part, whole)[row] = l > 0.f ? (ss.m_used[cc] + log2f(l)) * 0.69314718055994531f : -INFINITY;
        }
    }
    tc::fence_before_sync();
    __syncwarp();
    if (c.lane == 0) tc::mbar_arrive(smem_u32(&bars.o_free));
    return true;
}

// Closing a sequence b of this partition (no wait on its value products):
// its softmax denominators (1 / l kept for the drain) and its log-sum-exp.
template <int N, int KOWN>
__device__ __forceinline__ void sm_close(const SmCtx &c, const TcArgs &a, Shared<N> &ss, uint64_t (&l_part)[KOWN][8],
                                         int b, bool whole)
{
#pragma unroll
    for (int ob = 0; ob < KOWN; ++ob) {
        if (ob < c.n_own) {
            const int cb = c.half + 3 * ob;
            float v[16];
#pragma unroll
            for (int e = 0; e < 8; ++e) unpack2(l_part[ob][e], v[2 * e], v[2 * e + 1]);
            const float ls = sum16(v, c.lane);
            if (c.lane < 16) ss.red[c.quarter][cb * 16 + c.lane] = ls;
        }
    }
    named_sync_softmax();
    const int cc = c.tid - kSoftmaxBase;
    if (cc < N) {
        const float l = ss.red[0][cc] + ss.red[1][cc] + ss.red[2][cc] + ss.red[3][cc];
        ss.inv_l[cc] = l > 0.f ? 1.f / l : 0.f;
        const int row = c.group * N + cc;
        if (row < a.rows)
            lse_rows(a, b, c.part, whole)[row] = l > 0.f ? (ss.m_used[cc] + log2f(l)) * 0.69314718055994531f : -INFINITY;
    }
    named_sync_softmax();  // inv_l is complete and red is free again
}

// The normalised partial output of sequence b (closed by sm_close), whose
// last tile here was t_end_seg, from O^T buffer obuf; then the buffer is free.
template <int N, int KOWN>
__device__ __forceinline__ bool sm_drain(const SmCtx &c, const TcArgs &a, Shared<N> &ss, BarsT<N> &bars, int b,
                                         int t_end_seg, int obuf, bool whole, bool &failed)
{
    sm_wait(c, a, &ss.abort, failed, &bars.pv_done[t_end_seg % kPBufs<N>], static_cast<uint32_t>((t_end_seg / kPBufs<N>) & 1));
    if (softmax_any(failed)) return false;
    tc::fence_after_sync();
    const int valid_cols = a.rows - c.group * N;  // columns past it are padding
    float *out = out_rows(a, b, c.part, whole) + static_cast<int64_t>(c.group) * N * a.rank + c.tok;
    const uint32_t o_col = c.o_col0 + static_cast<uint32_t>(obuf * 4 * N);
    for (int m = 0; m < c.nrc; ++m) {
#pragma unroll
        for (int ob = 0; ob < KOWN; ++ob) {
            if (ob < c.n_own) {
                const int cb = c.half + 3 * ob;
                float o[16];
                tmem_ld16(c.tmem + c.lane_base + o_col + m * N + cb * 16, o);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int col = cb * 16 + e;
                    if (col < valid_cols) out[col * a.rank + m * 128] = o[e] * ss.inv_l[col];
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncwarp();
    if (c.lane == 0) tc::mbar_arrive(smem_u32(o_free_bar(bars, obuf)));
    return true;
}

// Exponents s scale - m of one 16-column block (log2 domain, pairs of columns),
// masked where needed; returns their maximum.
template <int N>
__device__ __forceinline__ float sm_exponents(const TcArgs &a, const Shared<N> &ss, uint32_t s_base, int cb, int pos,
                                              bool need_mask, uint64_t (&x)[8])
{
    uint32_t r[16];
    tc::ld_32x32b_x16(s_base + cb * 16, r);
    const float4 *nm = reinterpret_cast<const float4 *>(ss.neg_m + cb * 16);
    const uint64_t scale = pack2(a.scale_log2, a.scale_log2);
    tc::wait_ld();
    float mx = -INFINITY;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 m = nm[q];
        x[2 * q] = fma2(pack2(__uint_as_float(r[4 * q]), __uint_as_float(r[4 * q + 1])), scale, pack2(m.x, m.y));
        x[2 * q + 1] = fma2(pack2(__uint_as_float(r[4 * q + 2]), __uint_as_float(r[4 * q + 3])), scale, pack2(m.z, m.w));
    }
    if (need_mask) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            float lo, hi;
            unpack2(x[e], lo, hi);
            if (pos > ss.lim[cb * 16 + 2 * e]) lo = -INFINITY;
            if (pos > ss.lim[cb * 16 + 2 * e + 1]) hi = -INFINITY;
            x[e] = pack2(lo, hi);
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        float lo, hi;
        unpack2(x[e], lo, hi);
        mx = fmaxf(mx, fmaxf(lo, hi));
    }
    return mx;
}

// Online softmax of the partition's tiles.  Per tile each thread reads its
// scores from TMEM once, as exponents over the column's base m; one barrier
// carries the vote on whether a base has to move (a score above it by more
// than 2^8, or a sequence's first tile), which is the only other reason to
// meet.  (Two passes over TMEM, exp2f of scalar arithmetic and five barriers a
// tile took 7500 cycles a tile at N = 80, twice the tensor pipe's share.)
template <int N>
__device__ __forceinline__ void softmax_role(const SmCtx &c, const TcArgs &a, Shared<N> &ss, BarsT<N> &bars)
{
    constexpr int NB = N / 16;
    constexpr int KOWN = (NB + 2) / 3;
    constexpr int NP = kPBufs<N>;
    uint64_t l_part[KOWN][8];  // running sums of the weights, pairs of columns, over this thread's tokens
    // the sequence open here, with kWhole set when all its tiles lie in this
    // partition (its rows then go to the final buffers, when given)
    int b_cur = -1;
    int u = -1;  // sequences begun here (the PV warp counts the same ones)
    int t_prev = -1;  // the previous tile (one O^T buffer: the drain runs at the next sequence's first tile)
    // a closed sequence whose drain waits for the next sequence's first P (two O^T buffers)
    int d_b = -1, d_t = -1;
    bool failed = false, stop = false;
    const int cc = c.tid - kSoftmaxBase;
    Walk w;
    w.init(a, c.t_begin, c.n_items);
    for (; !w.done(); w.next()) {
        const int t = w.t;
        const bool first = w.first(), last = w.last();
        const int b = w.b, j = w.tile();
        const int kv = a.kv_len[b];
        const int sb = static_cast<int>(t & 1);
        sm_wait(c, a, &ss.abort, failed, &bars.s_full[sb], static_cast<uint32_t>((t >> 1) & 1));
        tc::fence_after_sync();
        if (first) {
            if constexpr (kOBufs<N> == 1) {
                if (b_cur >= 0 && !sm_epilogue<N, KOWN>(c, a, ss, bars, l_part, b_cur & ~kWhole, t_prev,
                                                        (b_cur & kWhole) != 0, failed)) {
                    stop = true;
                    break;
                }
            }
            b_cur = b | (w.whole() ? kWhole : 0);
            ++u;
#pragma unroll
            for (int ob = 0; ob < KOWN; ++ob)
#pragma unroll
                for (int e = 0; e < 8; ++e) l_part[ob][e] = 0;
            if (cc < N) {
                const int row = c.group * N + cc;
                ss.lim[cc] = row < a.rows ? kv - a.q_len + row / a.heads : -1;
            }
        }
        t_prev = t;
        const int pos = j * kTile + c.tok;
        // the mask matters only where a token lies past the earliest query's last key
        const bool need_mask = j * kTile + kTile - 1 > kv - a.q_len;
        const uint32_t s_base = c.tmem + c.lane_base + sb * N;
        uint64_t x[KOWN][8];
        bool moved = false;
#pragma unroll 1
        for (bool move = first;; move = false, moved = true) {
            float mx = -INFINITY;
            if (!move) {
#pragma unroll
                for (int ob = 0; ob < KOWN; ++ob)
                    if (ob < c.n_own)
                        mx = fmaxf(mx, sm_exponents<N>(a, ss, s_base, c.half + 3 * ob, pos, need_mask, x[ob]));
            }
            if (moved || !softmax_any(move || mx > 8.f || failed)) break;
            // ---- bases: exact column maxima on a sequence's first tile, else
            // raised where a score passed by more than 2^8
            if (softmax_any(failed)) {
                stop = true;
                break;
            }
            sm_block_max<N, KOWN>(c, a, ss, s_base, pos, need_mask);
            named_sync_softmax();
            if (cc < N) {
                const float tmax = fmaxf(fmaxf(ss.red[0][cc], ss.red[1][cc]), fmaxf(ss.red[2][cc], ss.red[3][cc]));
                float m = first ? tmax : ss.m_used[cc], alpha = 1.f;
                if (!first && tmax != -INFINITY && (m == -INFINITY || tmax > m + 8.f)) {
                    alpha = m == -INFINITY ? 0.f : ex2(m - tmax);
                    m = tmax;
                }
                ss.m_used[cc] = m;
                ss.neg_m[cc] = m == -INFINITY ? 0.f : -m;
                ss.alpha[cc] = alpha;
            }
            named_sync_softmax();
            if (!first) {
                // O^T is rescaled once PV(t-1) has completed
                sm_wait(c, a, &ss.abort, failed, &bars.pv_done[(t - 1) % NP], static_cast<uint32_t>(((t - 1) / NP) & 1));
                tc::fence_after_sync();
#pragma unroll
                for (int ob = 0; ob < KOWN; ++ob) {
                    if (ob < c.n_own) {
                        const int cb = c.half + 3 * ob;
                        float al[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) al[e] = ss.alpha[cb * 16 + e];
#pragma unroll
                        for (int e = 0; e < 8; ++e) l_part[ob][e] = fma2(l_part[ob][e], pack2(al[2 * e], al[2 * e + 1]), 0);
#pragma unroll 1
                        for (int m = 0; m < c.nrc; ++m) {
                            const uint32_t ta = c.tmem + c.lane_base + c.o_col0 +
                                                static_cast<uint32_t>((u % kOBufs<N>) * 4 * N + m * N + cb * 16);
                            float o[16];
                            tmem_ld16(ta, o);
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] *= al[e];
                            tmem_st16(ta, o);
                        }
                    }
                }
            }
        }
        if (stop) break;
        tc::fence_before_sync();
        __syncwarp();
        if (c.lane == 0) tc::mbar_arrive(smem_u32(&bars.s_free[sb]));  // S(t) is in registers
        // ---- P(t) = 2^x in bf16 (MN-major, 16-column SW32 atoms) into buffer
        // t % NP, free again once PV(t - NP) has completed; running sums.
        // Each wait is on the next phase of its barrier.
        if (t >= NP)
            sm_wait(c, a, &ss.abort, failed, &bars.pv_done[t % NP], static_cast<uint32_t>(((t - NP) / NP) & 1));
#pragma unroll
        for (int ob = 0; ob < KOWN; ++ob) {
            if (ob < c.n_own) {
                const int cb = c.half + 3 * ob;
                uint32_t pk[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    float lo, hi;
                    unpack2(x[ob][e], lo, hi);
                    const __nv_bfloat162 pb = __floats2bfloat162_rn(ex2(lo), ex2(hi));
                    pk[e] = *reinterpret_cast<const uint32_t *>(&pb);
                    // the weights the MMA multiplies by
                    l_part[ob][e] = add2(l_part[ob][e], pack2(__uint_as_float(pk[e] << 16), __uint_as_float(pk[e] & 0xffff0000u)));
                }
                unsigned char *row = c.p_buf + (t % NP) * (N / 16) * (kTile * 32) + cb * (kTile * 32) + c.tok * 32;
                const int sw = (c.tok >> 2) & 1;
                *reinterpret_cast<uint4 *>(row + (sw * 16)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                *reinterpret_cast<uint4 *>(row + ((1 ^ sw) * 16)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
            }
        }
        tc::fence_proxy_async_smem();
        tc::fence_before_sync();
        __syncwarp();
        if (c.lane == 0) tc::mbar_arrive(smem_u32(&bars.p_full[t % NP]));
        if constexpr (kOBufs<N> == 2) {
            // Due now, in this order: the previous sequence's drain (deferred
            // until this first P was out, so that it overlaps this tile's value
            // products in the other O^T buffer); then, on a sequence's last
            // tile, its close -- and at the partition's end its drain.
#pragma unroll 1
            for (int k = 0; k < 2; ++k) {
                int db = -1, dt = 0, dbuf = 0;
                if (k == 0 && d_b >= 0) {
                    db = d_b;
                    dt = d_t;
                    dbuf = (u - 1) & 1;
                    d_b = -1;
                }
                if (k == 1 && last) {
                    named_sync_softmax();
                    sm_close<N, KOWN>(c, a, ss, l_part, b_cur & ~kWhole, (b_cur & kWhole) != 0);
                    if (!w.last_of_partition()) {
                        d_b = b_cur;
                        d_t = static_cast<int>(t);
                    } else {
                        db = b_cur;
                        dt = static_cast<int>(t);
                        dbuf = u & 1;
                    }
                    b_cur = -1;
                }
                if (db >= 0) {
                    named_sync_softmax();
                    if (!sm_drain<N, KOWN>(c, a, ss, bars, db & ~kWhole, dt, dbuf, (db & kWhole) != 0, failed)) {
                        stop = true;
                        break;
                    }
                }
            }
            if (stop) break;
        }
    }
    named_sync_softmax();
    if constexpr (kOBufs<N> == 1) {
        if (b_cur >= 0 && !stop)
            sm_epilogue<N, KOWN>(c, a, ss, bars, l_part, b_cur & ~kWhole, t_prev, (b_cur & kWhole) != 0, failed);
    }
}

// N: query rows per CTA (multiple of 16, <= 80).  SQ (streamed queries): no
// resident query buffer; each QK-ring slot holds a cache chunk and, behind it,
// the query chunk that multiplies it, loaded with it from L2.  The ring then
// gets the shared memory the resident queries held, so that more cache bytes
// are in flight per SM, at the price of re-reading the queries once per tile.
template <int N, bool SQ>
__global__ void __maxnreg__(128)
    attn_tc_kernel(const __grid_constant__ TcArgs a, const __grid_constant__ CUtensorMap map_c,
                   const __grid_constant__ CUtensorMap map_r, const __grid_constant__ CUtensorMap map_q)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ BarsT<N> bars;
    __shared__ Shared<N> ss;
    __shared__ int64_t red64[32];

    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                            ~static_cast<uintptr_t>(1023));
    const int ncc = a.rank / 64;    // latent chunks per tile
    const int nrc = a.rank / 128;   // r-chunks of O^T
    const int nqc = ncc + 1;        // chunks of a tile in the QK pass: positional keys, then latent
    const int CA = a.qk_slots;      // QK ring slots
    const int CB = a.pv_slots;      // PV ring slots (even)
    static_assert(!SQ || (N * 128) % 1024 == 0, "a streamed query chunk keeps the slots 1024-byte aligned");
    constexpr int kSlotA = SQ ? kChunkBytes + N * 128 : kChunkBytes;       // QK-ring slot
    unsigned char *q_buf = smem;                                          // nqc x [N x 128 B] (resident queries)
    unsigned char *ring_a = SQ ? smem : q_buf + ((nqc * N * 128 + 1023) & ~1023);  // CA x [kSlotA]
    unsigned char *ring_b = ring_a + CA * kSlotA;                         // CB x [128 x 128 B]
    unsigned char *p_buf = ring_b + CB * kChunkBytes;                     // NP x NB x [128 tok x 32 B]

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int group = blockIdx.x, part = blockIdx.y;
    const uint64_t lim_ns = a.wait_ns;

    if (tid == 0) {
        for (int i = 0; i < kMaxSlots; ++i) {
            mbar_init(&bars.qk_full[i], 1);
            mbar_init(&bars.qk_empty[i], 1);
            mbar_init(&bars.pv_full[i], 1);
            mbar_init(&bars.pv_empty[i], 1);
        }
        mbar_init(&bars.q_full, 1);
        mbar_init(&bars.q_free, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars.s_full[i], 1);
            mbar_init(&bars.s_free[i], kSoftmaxWarps);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars.p_full[i], kSoftmaxWarps);
            mbar_init(&bars.pv_done[i], 1);
        }
        mbar_init(&bars.o_free, kSoftmaxWarps);
        if constexpr (kOBufs<N> == 2) mbar_init(o_free_bar(bars, 1), kSoftmaxWarps);
        mbar_init(&bars.drain_qk, 1);
        mbar_init(&bars.drain_pv, 1);
        ss.abort = 0;
        tc::fence_barrier_init();
    }
    if (warp == 1) {
        tc::tmem_alloc(smem_u32(&ss.tmem_base), kTmemCols<N>);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // The queries come from the previous launch; the cache does not: every
    // kernel of this library that writes the cache (append, projection) lets
    // its dependents launch only once it has completed, so by the time this
    // kernel runs (launched by its predecessor's trigger, which follows the
    // predecessor's own wait) the cache is final.  So no thread waits here:
    // the TMA producers load cache tiles at once, the query lanes wait before
    // the first query load and the softmax warps before they write partials
    // (a predecessor may still read the partial buffers); the MMA warps touch
    // only shared and tensor memory.
    griddep_launch_dependents();

    if (part == 0 && group == 0) {
        for (int bb = tid; bb < a.batch; bb += kThreads) {
            const int kv = a.kv_len[bb];
            if (kv < a.q_len || kv > a.max_kv) record_status(a.status, kStatusBounds);
        }
    }
    const int64_t T = block_tile_sum(a.kv_len, a.batch, a.q_len, a.max_kv, red64);
    const int64_t t_begin = T ? part_begin(part, T, a.num_splits) : 0;
    const int64_t t_end = T ? part_begin(part + 1, T, a.num_splits) : 0;
    const int n_items = static_cast<int>(t_end - t_begin);
    const uint32_t tmem = ss.tmem_base;
    const uint32_t o_col0 = 2 * N;   // S^T buffers at columns [0, N) and [N, 2N); O^T buffer i at 2N + 4N i
    auto any_abort = [&]() {
        return __any_sync(0xffffffffu, *reinterpret_cast<volatile int *>(&ss.abort) != 0);
    };

    if (warp == 0 || warp == 3) {
        // ================================================================ TMA producers
        // Warp 0 refills the QK ring (nqc chunks per tile: positional keys,
        // then the latent chunks; with streamed queries each chunk's query box
        // behind it), warp 3 the PV ring (the ncc latent chunks again).  Each
        // runs its ring in order with the whole warp converged and one elected
        // lane issuing; what a load needs besides a free slot is known a tile
        // ahead.  (One such warp fills 117 GB/s per SM from L2 and saturates
        // HBM with 64 KB in flight.  A lane per slot, polling and computing
        // its coordinates by division when its slot came free, kept every slot
        // 2.5 us from release to refilled: 67 GB/s.)
        if (n_items > 0) {
            const bool is_qk = warp == 0;
            if (is_qk) {
                tc::prefetch_tensormap(&map_c);
                tc::prefetch_tensormap(&map_r);
                tc::prefetch_tensormap(&map_q);
            }
            // the QK pass keeps latent lines in L2 for the PV pass, which reads
            // them a last time; the positional keys are read once
            const uint64_t pol_keep = tc::policy_evict_last(), pol_drop = tc::policy_evict_first();
            bool ok = true;
            RingPos rp{0, 0};
            TileStream ts;
            ts.init(a, t_begin, n_items);
            if (is_qk) {
                const uint32_t ring = smem_u32(ring_a);
                auto cache_box = [&](int i) {  // chunk i of the tile into the slot at rp
                    const uint32_t full = smem_u32(&bars.qk_full[rp.slot]), dst = ring + rp.slot * kSlotA;
                    tc::mbar_arrive_expect_tx_elect(full, ts.at.bytes + (SQ ? N * 128 : 0));
                    const CUtensorMap *map = i == 0 ? &map_r : &map_c;
                    const int col = i == 0 ? 0 : 64 * (i - 1);
                    const uint64_t pol = i == 0 ? pol_drop : pol_keep;
                    if (ts.at.nh > 0) tc::tma_load_3d_hint_elect(dst, map, col, ts.at.tok0, ts.at.blk[0], full, pol);
                    if (ts.at.nh > 1)
                        tc::tma_load_3d_hint_elect(dst + kHalf * 128, map, col, ts.at.tok0, ts.at.blk[1], full, pol);
                };
                // the query columns chunk i multiplies: the positional part lies
                // behind the latent part in each query row
                auto query_box = [&](int i, int slot, int b) {
                    tc::tma_load_2d_hint_elect(ring + slot * kSlotA + kChunkBytes, &map_q, 64 * (i == 0 ? ncc : i - 1),
                                               b * a.rows + group * N, smem_u32(&bars.qk_full[slot]), pol_keep);
                };
                // The ring's first round: its cache boxes go out before the
                // previous launch (which writes the queries) has completed.
                const int64_t total = static_cast<int64_t>(n_items) * nqc;
                const int head = total < CA ? static_cast<int>(total) : CA;
                int i = 0;
                for (; rp.slot < head && rp.round == 0; rp.advance(CA)) {
                    cache_box(i);
                    if (++i == nqc) {
                        i = 0;
                        ts.next(a);
                    }
                }
                griddep_wait();
                if constexpr (SQ) {
                    Walk w;
                    w.init(a, t_begin, n_items);
                    for (int s = 0, k = 0; s < head; ++s) {
                        query_box(k, s, w.b);
                        if (++k == nqc) {
                            k = 0;
                            w.next();
                        }
                    }
                }
                while (!ts.w.done() && ok && !any_abort()) {
                    for (; i < nqc; ++i) {
                        ok = mbar_wait_warp(smem_u32(&bars.qk_empty[rp.slot]), (rp.round - 1) & 1, lim_ns);
                        if (!ok) break;
                        if (SQ && ts.at.nh > 0) {
                            const uint32_t dst = ring + rp.slot * kSlotA;
                            tc::tma_refill_q_elect(smem_u32(&bars.qk_full[rp.slot]), ts.at.bytes + N * 128,
                                                   i == 0 ? &map_r : &map_c, i == 0 ? 0 : 64 * (i - 1), ts.at.tok0, dst,
                                                   ts.at.blk[0], dst + kHalf * 128, ts.at.blk[1], ts.at.nh > 1,
                                                   i == 0 ? pol_drop : pol_keep, &map_q, 64 * (i == 0 ? ncc : i - 1),
                                                   ts.w.b * a.rows + group * N, dst + kChunkBytes, pol_keep);
                        } else {
                            cache_box(i);
                            if constexpr (SQ) query_box(i, rp.slot, ts.w.b);
                        }
                        rp.advance(CA);
                    }
                    i = 0;
                    ts.next(a);
                }
            } else {
                const uint32_t ring = smem_u32(ring_b);
                for (; !ts.w.done() && ok && !any_abort(); ts.next(a)) {
                    for (int m = 0; m < nrc; ++m, rp.advance(CB / 2)) {
                        const uint32_t full = smem_u32(&bars.pv_full[rp.slot]), dst = ring + rp.slot * 2 * kChunkBytes;
                        ok = rp.round == 0 || mbar_wait_warp(smem_u32(&bars.pv_empty[rp.slot]), (rp.round - 1) & 1, lim_ns);
                        if (!ok) break;
                        if (ts.at.nh > 0)
                            tc::tma_refill_pair_elect(full, 2 * ts.at.bytes, &map_c, 128 * m, ts.at.tok0, dst, kChunkBytes,
                                                      ts.at.blk[0], kHalf * 128, ts.at.blk[1], ts.at.nh > 1, pol_drop);
                        else
                            tc::mbar_arrive_expect_tx_elect(full, 0);
                    }
                }
            }
            if (!ok && lane == 0) {
                record_status(a.status, kStatusTimeout);
                ss.abort = 1;
            }
            __syncwarp();
        }
    } else if (warp == 1 || warp == 2) {
        // ================================================================ MMA issuers
        // Warp 1 issues the score products QK(t), warp 2 the value products
        // PV(t); each consumes its own ring in order.  The whole warp runs its
        // loop converged (every lane waits); one elected lane issues each MMA,
        // commit and arrive.
        const bool is_qk = warp == 1;
        uint64_t *drain = is_qk ? &bars.drain_qk : &bars.drain_pv;
        if (n_items > 0) {
            const uint32_t q_base = smem_u32(q_buf), p_base = smem_u32(p_buf);
            // descriptor templates (start address added per MMA)
            const uint64_t dq = tc::smem_desc(0, 16, 1024, tc::kSwizzle128B);
            const uint64_t dc = tc::smem_desc(0, kChunkBytes, 1024, tc::kSwizzle128B);
            const uint64_t dp = tc::smem_desc(0, 128 * 32, 256, tc::kSwizzle32B);
            auto with_addr = [](uint64_t tmpl, uint32_t saddr) {
                return tmpl | static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
            };
            Walk w;
            w.init(a, t_begin, n_items);
            RingPos rp{0, 0};
            bool ok = true;
            auto wait = [&](uint64_t *bar, uint32_t parity) {
                if (ok) ok = mbar_wait_warp(smem_u32(bar), parity, lim_ns);
                return ok;
            };
            if (is_qk) {
                const uint32_t id_qk = tc::idesc_bf16_f32(128, N, false, false);
                const uint32_t ring_base = smem_u32(ring_a);
                int seg = -1;
                for (int t = 0; t < n_items && ok; ++t, w.next()) {
                    if (any_abort()) break;
                    if (!SQ && w.first()) {
                        // resident queries: this warp's products of the last sequence
                        // have read the buffer (q_free); load the next one's
                        ++seg;
                        if (seg == 0) griddep_wait();
                        if (seg > 0 && !wait(&bars.q_free, (seg - 1) & 1)) break;
                        tc::mbar_arrive_expect_tx_elect(smem_u32(&bars.q_full), nqc * N * 128);
                        for (int i = 0; i < nqc; ++i)
                            tc::tma_load_2d_hint_elect(q_base + i * N * 128, &map_q, 64 * i, w.b * a.rows + group * N,
                                                       smem_u32(&bars.q_full), tc::policy_evict_first());
                        if (!wait(&bars.q_full, seg & 1)) break;
                    }
                    const int sb = t & 1;
                    if (t >= 2 && !wait(&bars.s_free[sb], ((t >> 1) - 1) & 1)) break;
                    const uint32_t d_s = tmem + sb * N;
                    for (int i = 0; i < nqc && ok; ++i) {
                        if (!wait(&bars.qk_full[rp.slot], rp.round & 1)) break;
                        tc::fence_after_sync();
                        const uint32_t cb = ring_base + rp.slot * kSlotA;
                        const uint32_t qb = SQ ? cb + kChunkBytes : q_base + (i == 0 ? ncc : i - 1) * N * 128;
                        // four steps of 16 columns (32 bytes); then the slot goes back
                        tc::mma4_bf16_commit_elect(d_s, with_addr(dq, cb), with_addr(dq, qb), id_qk, i != 0, 2, 2,
                                                   smem_u32(&bars.qk_empty[rp.slot]));
                        rp.advance(CA);
                    }
                    if (!ok) break;
                    tc::commit_elect(smem_u32(&bars.s_full[sb]));
                    if (!SQ && w.last()) tc::commit_elect(smem_u32(&bars.q_free));
                }
            } else {
                const uint32_t id_pv = tc::idesc_bf16_f32(128, N, true, true);
                const uint32_t ring_base = smem_u32(ring_b);
                int seg = -1;
                uint32_t o_cur = o_col0;
                for (int t = 0; t < n_items && ok; ++t, w.next()) {
                    if (any_abort()) break;
                    if (!wait(&bars.p_full[t % kPBufs<N>], (t / kPBufs<N>) & 1)) break;
                    bool first_pv = false;
                    if (w.first()) {
                        // buffer seg % kOBufs: wait until the sequence that used it last has drained
                        ++seg;
                        const int ob = seg % kOBufs<N>, use = seg / kOBufs<N>;
                        if (use >= 1 && !wait(o_free_bar(bars, ob), (use - 1) & 1)) break;
                        o_cur = o_col0 + static_cast<uint32_t>(ob * 4 * N);
                        first_pv = true;
                    }
                    // A sequence's last, partial tile of v rows: only the 16-token
                    // steps holding rows < v are issued, and in the last of them the
                    // rows v .. v16 - 1 of both chunks are cleared here first, so that
                    // stale or uninitialised bytes never meet a zero weight (0 x NaN
                    // is NaN).  Rows past v16 are never read.
                    const int v = a.kv_len[w.b] - w.tile() * kTile;
                    const bool tail = w.last() && v < kTile;
                    const int v16 = tail ? (v + 15) / 16 * 16 : kTile;
                    const uint32_t pb = p_base + (t % kPBufs<N>) * (N / 16) * (kTile * 32);
                    for (int m = 0; m < nrc && ok; ++m, rp.advance(CB / 2)) {
                        // ring entry: chunks 2m and 2m + 1, side by side
                        if (!wait(&bars.pv_full[rp.slot], rp.round & 1)) break;
                        tc::fence_after_sync();
                        unsigned char *entry = ring_b + rp.slot * 2 * kChunkBytes;
                        if (v16 > v) {
                            const int nz = (v16 - v) * 8;  // 16-byte pieces per chunk
                            for (int idx = lane; idx < 2 * nz; idx += 32) {
                                const int k = idx / nz, r = idx - k * nz;
                                uint4 *dst = reinterpret_cast<uint4 *>(entry + k * kChunkBytes + (v + r / 8) * 128) + r % 8;
                                *dst = make_uint4(0, 0, 0, 0);
                            }
                            tc::fence_proxy_async_smem();
                            __syncwarp();
                        }
                        const uint32_t cb = ring_base + rp.slot * 2 * kChunkBytes;
                        const uint32_t d_o = tmem + o_cur + m * N;
                        const uint32_t empty = smem_u32(&bars.pv_empty[rp.slot]);
                        if (v16 == kTile) {
                            tc::mma8_bf16_commit_elect(d_o, with_addr(dc, cb), with_addr(dp, pb), id_pv, first_pv ? 0u : 1u,
                                                       16 * 128 / 16, 16 * 32 / 16, empty);
                        } else {
                            for (int kk = 0; kk < v16 / 16; ++kk)
                                tc::mma_bf16_elect(d_o, with_addr(dc, cb + kk * 16 * 128),
                                                   with_addr(dp, pb + kk * 16 * 32), id_pv,
                                                   (first_pv && kk == 0) ? 0u : 1u);
                            tc::commit_elect(empty);
                        }
                    }
                    if (!ok) break;
                    tc::commit_elect(smem_u32(&bars.pv_done[t % kPBufs<N>]));
                }
            }
            if (!ok && lane == 0) {
                record_status(a.status, kStatusTimeout);
                ss.abort = 1;
            }
            // drain: every MMA this warp issued has completed before TMEM is freed
            tc::commit_elect(smem_u32(drain));
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(drain), 0, lim_ns)) && lane == 0)
                record_status(a.status, kStatusTimeout);
        }
    } else {
        // ================================================================ softmax / epilogue
        griddep_wait();  // before any partial is written (returns at once by the time S arrives)
        SmCtx c;
        c.lane = lane;
        c.tid = tid;
        c.quarter = warp & 3;                 // TMEM lane quarter this warp may access
        c.half = (warp - 4) >> 2;             // which column blocks it owns: half, half+3, ...
        c.tok = c.quarter * 32 + lane;        // token row of the tile
        c.n_own = c.half < N / 16 ? (N / 16 - c.half + 2) / 3 : 0;
        c.group = group;
        c.part = part;
        c.nrc = nrc;
        c.n_items = n_items;
        c.lane_base = static_cast<uint32_t>(c.quarter * 32) << 16;
        c.tmem = tmem;
        c.o_col0 = o_col0;
        c.p_buf = p_buf;
        c.lim_ns = lim_ns;
        c.t_begin = t_begin;
        softmax_role<N>(c, a, ss, bars);
    }

    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kTmemCols<N>);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

cudaError_t get_encoder()
{
    if (g_encode) return cudaSuccess;
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return e != cudaSuccess ? e : cudaErrorNotSupported;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return cudaSuccess;
}

// 3-d map over one cache: (columns, tokens per block, blocks), box 64 x box_rows x 1, SW128.
cudaError_t encode_cache_map(CUtensorMap *m, const void *base, int cols, int64_t tok_stride, int64_t blk_stride,
                             int tokens_per_block, int blocks, int box_rows)
{
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(tokens_per_block),
                          static_cast<cuuint64_t>(blocks)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(tok_stride) * 2, static_cast<cuuint64_t>(blk_stride) * 2};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_rows), 1};
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int N, bool SQ>
cudaError_t launch_cfg(const AttnArgs &a, int groups, cudaStream_t st)
{
    cudaError_t e = get_encoder();
    if (e != cudaSuccess) return e;
    const CacheView &c = a.cache;
    const bool paged = c.block_table != nullptr;
    const int tpb = paged ? c.page_size : c.capacity;
    const int blocks = paged ? c.num_pages : a.batch;
    CUtensorMap mc, mr, mq;
    const int box_rows = paged ? kHalf : kTile;
    if ((e = encode_cache_map(&mc, c.c_kv, a.rank, c.c_tok, c.c_blk, tpb, blocks, box_rows)) != cudaSuccess) return e;
    if ((e = encode_cache_map(&mr, c.k_rope, a.d_rope, c.r_tok, c.r_blk, tpb, blocks, box_rows)) != cudaSuccess) return e;
    {
        const int K = a.rank + a.d_rope;
        cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(a.batch) * a.q_len * a.num_heads};
        cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
        cuuint32_t box[2] = {64, N};
        cuuint32_t es[2] = {1, 1};
        CUresult r = g_encode(&mq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(a.q_abs), dims, strides,
                              box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    const int ncc = a.rank / 64;
    const int q_bytes = SQ ? 0 : (((ncc + 1) * N * 128) + 1023) & ~1023;
    const int slot_a = SQ ? kChunkBytes + N * 128 : kChunkBytes;  // QK-ring slot (with its query chunk)
    const int p_bytes = kPBufs<N> * (N / 16) * kTile * 32;
    const int fixed = 1024 /*alignment slack*/ + q_bytes;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const int static_bytes = static_cast<int>(sizeof(BarsT<N>) + sizeof(Shared<N>) + 32 * 8) + 128;
    const int avail = optin - static_bytes - fixed - p_bytes;
    // the PV ring (refilled from L2) gets six slots where four QK slots still
    // fit beside them (streamed queries), else four or two; the QK ring the
    // rest.  (Measured with 80 rows, whose second P buffer leaves four QK and
    // four PV slots: six PV slots beside three QK slots lose 16 %, two beside
    // five 46 %.)
    int pv_slots = SQ && avail >= 4 * slot_a + 6 * kChunkBytes ? 6 : avail >= 2 * slot_a + 4 * kChunkBytes ? 4 : 2;
    const int cap = tuning().tc_max_slots;  // testing aid: smaller rings
    if (cap >= 4 && pv_slots > cap - 2) pv_slots = 2;
    if (const int v = tuning().tc_pv_slots & ~1; v >= 2 && v <= kMaxSlots && avail >= 2 * slot_a + v * kChunkBytes &&
                                                  (cap < 4 || v <= cap - 2))
        pv_slots = v;  // testing aid
    int qk_slots = (avail - pv_slots * kChunkBytes) / slot_a;
    if (qk_slots > kMaxSlots) qk_slots = kMaxSlots;
    if (cap >= 4 && qk_slots > cap - pv_slots) qk_slots = cap - pv_slots;
    if (qk_slots < 2) return cudaErrorInvalidConfiguration;
    const size_t smem = static_cast<size_t>(fixed) + static_cast<size_t>(qk_slots) * slot_a +
                        static_cast<size_t>(pv_slots) * kChunkBytes + p_bytes;
    // (smem is whole KB, and so is the static part: its alignment is the dynamic part's)
    if ((e = allow_smem<attn_tc_kernel<N, SQ>>((optin - static_bytes) & ~1023)) != cudaSuccess) return e;
    TcArgs t;
    t.batch = a.batch;
    t.q_len = a.q_len;
    t.heads = a.num_heads;
    t.rank = a.rank;
    t.d_rope = a.d_rope;
    t.rows = a.q_len * a.num_heads;
    t.num_splits = a.num_splits;
    t.max_kv = a.max_kv;
    t.paged = paged;
    t.bt_stride = c.bt_stride;
    t.num_pages = c.num_pages;
    t.qk_slots = qk_slots;
    t.pv_slots = pv_slots;
    t.scale_log2 = a.sm_scale * 1.4426950408889634f;
    t.kv_len = a.kv_len;
    t.block_table = c.block_table;
    t.o_part = a.o_part;
    t.lse_part = a.lse_part;
    t.o_final = a.o_final;
    t.lse_final = a.lse_final;
    t.status = a.status;
    t.wait_ns = kWaitLimitNs;
    return launch_dependent(attn_tc_kernel<N, SQ>, dim3(groups, a.num_splits, 1), dim3(kThreads), smem, st, 1, t, mc,
                            mr, mq);
}

}  // namespace

TcShape attn_tc_shape(int rows)
{
    // Testing aid: the tuning knob tc_max_rows caps the query rows per CTA (16..80).
    int max_n = tuning().tc_max_rows > 0 ? tuning().tc_max_rows : 80;
    if (max_n < 16) max_n = 16;
    if (max_n > 80) max_n = 80;
    max_n -= max_n % 16;
    TcShape s;
    s.groups = (rows + max_n - 1) / max_n;
    s.n = (((rows + s.groups - 1) / s.groups + 15) / 16) * 16;
    return s;
}

cudaError_t launch_attn_tc(const AttnArgs &a, cudaStream_t st)
{
    const TcShape s = attn_tc_shape(a.q_len * a.num_heads);
    const bool sq = tuning().tc_query != 1;
    switch (s.n) {
    case 16: return sq ? launch_cfg<16, true>(a, s.groups, st) : launch_cfg<16, false>(a, s.groups, st);
    case 32: return sq ? launch_cfg<32, true>(a, s.groups, st) : launch_cfg<32, false>(a, s.groups, st);
    case 48: return sq ? launch_cfg<48, true>(a, s.groups, st) : launch_cfg<48, false>(a, s.groups, st);
    case 64: return sq ? launch_cfg<64, true>(a, s.groups, st) : launch_cfg<64, false>(a, s.groups, st);
    case 80: return sq ? launch_cfg<80, true>(a, s.groups, st) : launch_cfg<80, false>(a, s.groups, st);
    default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace gbmla

