// The projections of the decode step as grouped GEMMs (all bf16 weights,
// fp32 accumulation, bf16 results):
//   absorption (Sec. 1; Eq. 5 read right to left): q_lat[row] = q_nope[row] W_UK[g]   (W_UK: d_nope x r)
//   value up-projection (Eq. 5):                    o[row]     = W_UV[g] o_lat[row]    (W_UV: d_v x r)
//   output projection (Sec. 4.1):                   out[m]     = W_O concat_h o[m]     (W_O: D x H d_v)
// In every case C[phys(g, m), n] = sum_k A[phys(g, m), k] B_g(n, k) for the M
// rows of group g, with phys(g, m) = (m / hpg) * blk + g * hpg + m % hpg.
//
// All as one tcgen05 GEMM: up to 128 rows x BN columns per CTA, A and the
// weight tile loaded by TMA, the fp32 accumulator in TMEM.  A GEMM whose tiles
// would occupy few SMs (few rows, deep K: the output projection of a small
// batch) splits K over a cluster of up to four CTAs; each leaves its partial
// tile in shared memory, sends every other CTA its share of it, and sums its own
// share of the partials in a fixed order, so the result does not depend on timing.
//
// The same kernel, with PROJ set, projects the step's hidden states (the step
// before the cache append, Sec. 3.2 and Eq. 1): rows are the entries
// h[b, k, :], and the column tiles run over W^DKV (the latent), one tile for
// W^KR (the positional key) and W^Q (the queries).  Its epilogue writes the
// latent row and the positional key, rotated to the entry's position in fp32,
// straight into the (paged) cache, and splits each query head into its
// non-positional and positional parts.
#include <cudaTypedefs.h>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace gbmla {
namespace {

__device__ __forceinline__ int64_t phys_row(const GroupGemm &p, int g, int m)
{
    if (p.hpg == 1) return static_cast<int64_t>(m) * p.blk + g;
    return static_cast<int64_t>(m / p.hpg) * p.blk + g * p.hpg + m % p.hpg;
}

// Epilogue arguments of the projection (PROJ): column tiles [0, tiles_lat)
// hold the latent, tile tiles_lat the positional key, the rest the queries.
// The absorption GEMM (not PROJ) reuses it for the positional query: when
// rope_src is set, the CTAs of each row tile also write
// C[row, rank .. rank + d_rope) = R_p q_pe[row] for the rows of that tile,
// p = kv_len[b] - q_len + i for row (b, i, head) (rows in [B, q_len, heads] order).
struct ProjEpi {
    CacheView cache;
    const int32_t *start_pos;
    uint16_t *q_nope, *q_pe;
    int n_new, rank, d_rope, d_nope, heads, style;
    RopeTurns turns;
    int tiles_lat;
    uint32_t box_bytes[3];  // weight-tile bytes of the three column regions
    const uint16_t *rope_src;  // absorption: q_pe [B, q_len, heads, d_rope], or null
    const int32_t *kv_len;
    int q_len;
};

// eight fp32 bit patterns -> eight bf16 (round to nearest even)
__device__ __forceinline__ uint4 pack8_bf16(const uint32_t *v)
{
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
        w[e] = *reinterpret_cast<const uint32_t *>(&b);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// The bf16 results of a warp's 32 tile rows x BN columns, from TMEM to memory:
// 64 columns at a time go through a staging block (32 rows of 144 bytes: both
// sides free of bank conflicts), so that eight lanes store 128 contiguous bytes
// of a row.  store(col) returns, for a lane's eight columns from col, what
// stores them for the warp's row r (called by every lane).  Each lane storing its
// own row, 16 bytes a lane in 32 places, took 6800 cycles for the projection's 192
// columns; this 3400, of which the stores (32 bytes a clock an SM) 2500.
constexpr int kDrainRow = 144, kDrainWarp = 32 * kDrainRow, kDrainBytes = 4 * kDrainWarp;

__device__ __forceinline__ uint16_t *shfl_ptr(uint16_t *p, int lane)
{
    return reinterpret_cast<uint16_t *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(p), lane));
}

// 16 bytes to dst if ok: a predicated store, no branch
__device__ __forceinline__ void store16_if(bool ok, uint16_t *dst, const uint4 &v)
{
    asm volatile("{.reg .pred p; setp.ne.u32 p, %0, 0; @p st.global.v4.b32 [%1], {%2, %3, %4, %5};}" ::"r"(
                     static_cast<uint32_t>(ok)),
                 "l"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// the same with 8 bytes
__device__ __forceinline__ void store8_if(bool ok, uint16_t *dst, uint32_t x, uint32_t y)
{
    asm volatile("{.reg .pred p; setp.ne.u32 p, %0, 0; @p st.global.v2.b32 [%1], {%2, %3};}" ::"r"(static_cast<uint32_t>(ok)),
                 "l"(dst), "r"(x), "r"(y)
                 : "memory");
}

template <int BN, class Store>
__device__ __forceinline__ void drain_tile(uint32_t t_lane, unsigned char *stage, int lane, Store store)
{
#pragma unroll 1
    for (int j = 0; j < BN; j += 64) {
        uint32_t v[4][16];
#pragma unroll
        for (int u = 0; u < 4; ++u) tc::ld_32x32b_x16(t_lane + j + 16 * u, v[u]);
        tc::wait_ld();
        __syncwarp();  // the block before has been read
#pragma unroll
        for (int k = 0; k < 8; ++k)
            *reinterpret_cast<uint4 *>(stage + lane * kDrainRow + 16 * k) = pack8_bf16(&v[k >> 1][8 * (k & 1)]);
        __syncwarp();
        const auto row = store(j + 8 * (lane & 7));
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
            const int r = 4 * rr + (lane >> 3);
            row(r, *reinterpret_cast<const uint4 *>(stage + r * kDrainRow + 16 * (lane & 7)));
        }
    }
}

// The same by TMA stores: the tile's RT rows x 64 columns at a time, staged in
// the 128-byte swizzle as the box that store(j) sends (called by one thread).
// Plain stores leave an SM at 30 bytes a clock, TMA stores at 88 (192 KB from
// each of 152 SMs: 6700 and 2200 cycles).  Called by the four epilogue warps,
// also by one whose accumulator never came (good false): it keeps to the barriers.
// W_UV + W_O of 14 heads, 64 rows, 7.5 -> 6.9 us, of 32 heads and 640 rows 19.8 ->
// 18.6.  Not for the projection's queries: its latent tiles, whose rows lie where
// the cache has them, are as many stores and end last (13.54 and 13.49 us).
template <int BN, class Store>
__device__ __forceinline__ void drain_tile_tma(uint32_t t_lane, unsigned char *stage, int i, int RT, bool good, Store store)
{
#pragma unroll 1
    for (int j = 0; j < BN; j += 64) {
        unsigned char *row = stage + j * 256 + i * 128;
        if (good) {
            uint32_t v[4][16];
#pragma unroll
            for (int u = 0; u < 4; ++u) tc::ld_32x32b_x16(t_lane + j + 16 * u, v[u]);
            tc::wait_ld();
            if (i < RT) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    *reinterpret_cast<uint4 *>(row + ((k ^ (i & 7)) << 4)) = pack8_bf16(&v[k >> 1][8 * (k & 1)]);
            }
            tc::fence_proxy_async_smem();
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (threadIdx.x == 64 && good) store(j, smem_u32(stage + j * 256));
        __syncwarp();
    }
    if (threadIdx.x == 64) {
        tc::bulk_commit();
        tc::bulk_wait0();
    }
}

// R_pos of the DR projected positional-key values x (fp32; the angle reduced
// exactly as a fraction of a turn), rounded once to bf16 into `row`.
template <int DR>
__device__ __forceinline__ void rotate_store(const float (&x)[64], int64_t pos, int style, const RopeTurns &turns,
                                             uint16_t *row)
{
    constexpr int HALF = DR / 2;
    __align__(16) uint16_t y[DR];
    if (style == 0) {
#pragma unroll
        for (int k = 0; k < HALF; ++k) {
            float cs, sn;
            rope_cos_sin(pos, turns.f[k], &cs, &sn);
            y[k] = __bfloat16_as_ushort(__float2bfloat16_rn(x[k] * cs - x[k + HALF] * sn));
            y[k + HALF] = __bfloat16_as_ushort(__float2bfloat16_rn(x[k + HALF] * cs + x[k] * sn));
        }
    } else {
#pragma unroll
        for (int k = 0; k < HALF; ++k) {
            float cs, sn;
            rope_cos_sin(pos, turns.f[k], &cs, &sn);
            y[2 * k] = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * k] * cs - x[2 * k + 1] * sn));
            y[2 * k + 1] = __bfloat16_as_ushort(__float2bfloat16_rn(x[2 * k + 1] * cs + x[2 * k] * sn));
        }
    }
#pragma unroll
    for (int v = 0; v < DR / 8; ++v) reinterpret_cast<uint4 *>(row)[v] = reinterpret_cast<const uint4 *>(y)[v];
}

// Projection epilogue of a warp: `rows` tile rows from row m of this lane
// (the entry h[m / n_new, m % n_new]); every lane of the warp calls it.
template <int BN>
__device__ void proj_epilogue(const GroupGemm &p, const ProjEpi &e, uint32_t t_lane, unsigned char *stage, int lane, int m,
                              int rows)
{
    const int ty = blockIdx.y;
    if (ty > e.tiles_lat) {
        // ---- queries: column c of W^Q is element c % dq of head c / dq (eight
        // columns from a multiple of eight are of one part of one head: d_nope
        // and d_rope are multiples of eight)
        const int dq = e.d_nope + e.d_rope, nq = e.heads * dq;
        const int c0 = (ty - e.tiles_lat - 1) * BN, mw = m - lane;
        drain_tile<BN>(t_lane, stage, lane, [&](int col) {
            const int c = c0 + col, head = c / dq, el = c - head * dq;
            const int width = el < e.d_nope ? e.d_nope : e.d_rope;
            uint16_t *dst = el < e.d_nope ? e.q_nope + el : e.q_pe + (el - e.d_nope);
            dst += (static_cast<int64_t>(mw) * e.heads + head) * width;
            const int64_t step = static_cast<int64_t>(e.heads) * width;  // row to row
            const int rows_c = c < nq ? rows : 0;
            return [=](int r, const uint4 &v) { store16_if(r < rows_c, dst + r * step, v); };
        });
        return;
    }
    // ---- the entry's cache row: position start_pos[b] + k, through the block table when paged
    const CacheView &c = e.cache;
    bool ok = lane < rows;
    int64_t pos = 0, blk = 0, slot = 0;
    if (ok) {
        const int b = m / e.n_new, k = m % e.n_new;
        pos = static_cast<int64_t>(e.start_pos[b]) + k;
        ok = pos >= 0 && pos < c.capacity;
        if (ok && c.block_table) {
            const int32_t page = c.block_table[static_cast<int64_t>(b) * c.bt_stride + pos / c.page_size];
            ok = page >= 0 && page < c.num_pages;
            blk = page;
            slot = pos % c.page_size;
        } else {
            blk = b;
            slot = pos;
        }
        if (!ok) record_status(p.status, kStatusBounds);
    }
    if (ty < e.tiles_lat) {
        // ---- latent c = W^DKV h, rounded once
        uint16_t *crow = ok ? static_cast<uint16_t *>(const_cast<void *>(c.c_kv)) + blk * c.c_blk + slot * c.c_tok : nullptr;
        drain_tile<BN>(t_lane, stage, lane, [&](int col) {
            const int n = ty * BN + col;
            const bool in = n < e.rank;  // (the last tile may reach past the latent)
            return [=](int r, const uint4 &v) {
                uint16_t *row = shfl_ptr(crow, r);
                store16_if(row && in, row + n, v);
            };
        });
        return;
    }
    // ---- positional key R_pos W^KR h (d_rope = 32 or 64 columns of this tile)
    float x[64];
#pragma unroll
    for (int j = 0; j < 64; j += 16) {
        if (j < e.d_rope) {
            uint32_t v[16];
            tc::ld_32x32b_x16(t_lane + j, v);
            tc::wait_ld();
#pragma unroll
            for (int u = 0; u < 16; ++u) x[j + u] = __uint_as_float(v[u]);
        } else {
#pragma unroll
            for (int u = 0; u < 16; ++u) x[j + u] = 0.f;
        }
    }
    if (!ok) return;
    uint16_t *rrow = static_cast<uint16_t *>(const_cast<void *>(c.k_rope)) + blk * c.r_blk + slot * c.r_tok;
    if (e.d_rope == 64)
        rotate_store<64>(x, pos, e.style, e.turns, rrow);
    else
        rotate_store<32>(x, pos, e.style, e.turns, rrow);
}

// ---------------------------------------------------------------- tensor-core GEMM
// Both operands arrive by TMA.  The A rows of a group are one 4-d box
// (K, head in group, group, row block): a tile holds R = 128 / hpg row blocks
// of hpg rows, i.e. RT = R hpg <= 128 rows.  A bf16 A box lands directly in
// the 128B-swizzled K-major layout the MMA reads; an fp32 A (o_lat) lands as
// two 32-column boxes in a staging tile, which four warps convert to bf16.
constexpr int kStages = 16;  // most ring stages; fewer when K is short or shared memory runs out
// Rows of one column group of a split-K partial as received: 1 mod 8, so that
// lanes on different column groups of a row read different banks.
__host__ __device__ constexpr int recv_rows(int rt) { return (rt + 7) / 8 * 8 + 1; }
// warp 0 TMA, warp 1 MMA, warps 2..5 epilogue; of an fp32 A, warps 2..5 convert
// too, and in a launch of kConvThreads warps 6..9: two sets of four warps take
// turns with the ring's stages, so that one set's latency (wait, read, write,
// proxy fence: 850 cycles a chunk) hides behind the other's.  W_UV + W_O of 32
// heads: 32 rows 10.4 -> 9.9 us, 160 rows 13.2 -> 12.8.  Where K is split (two
// chunks a CTA: one row 7.9 -> 8.2) or two CTAs share an SM, one set remains.
constexpr int kGemmThreads = 192, kConvThreads = 320;
constexpr int kShortRows = 96;
constexpr int kM64Rows = 64;  // the tallest tile that MMAs of M = 64 take

// The tile row whose accumulator lane `lane` of TMEM quarter q holds: with M = 64
// the rows lie in the first 16 lanes of each quarter (the other lanes: none).
__device__ __forceinline__ int tile_row(bool m64, int q, int lane)
{
    return !m64 ? q * 32 + lane : lane < 16 ? q * 16 + lane : 128;
}

struct __align__(8) GemmBars {
    uint64_t full[kStages], raw_full[kStages], conv_done[kStages], empty[kStages], done, recv;
};

// A, the weight and C; of the projection, the weights of its three column regions.
template <bool PROJ>
struct GemmMaps {
    CUtensorMap a, b, c;
};
template <>
struct GemmMaps<true> {
    CUtensorMap a, b, b2, b3;
};

// BN: columns per CTA.  NMAJ: the weight is N-major.  AF32: A is fp32.
// PROJ: the projection (K-major weights b, b2, b3 by column region).
// SHORT: an fp32 A in tiles of at most kShortRows rows, whose stages hold just
// those (W_UV + W_O of 14 heads, one row 7.1 -> 6.6 us, 64 rows 8.0 -> 7.5);
// with taller tiles the fixed stage is 1 to 2 percent faster.
// SPLIT: K split over a cluster; a kernel holds one of the two ways out.
// (Two CTAs an SM stated, or the compiler takes 64 registers and spills in the
// split kernels: 24 heads, 64 rows 12.6 us instead of 11.7.  The projection is
// one CTA an SM and was slower with either bound: 160 rows 9.7 -> 10.2.)
// M64: tiles of at most 64 rows take MMAs of M = 64, which read half the A rows
// (8 rows of 24 heads, W_UV + W_O: 9.4 -> 8.6 us); a kernel of its own, because
// the choice at run time cost the tall tiles 2 to 5 percent.
template <int BN, bool NMAJ, bool AF32, bool PROJ, bool SHORT, bool SPLIT, bool M64>
__global__ void __launch_bounds__(AF32 ? kConvThreads : kGemmThreads, PROJ ? 0 : 2) gemm_tc_kernel(const __grid_constant__ GroupGemm p,
                                                               const __grid_constant__ GemmMaps<PROJ> maps,
                                                               const __grid_constant__ ProjEpi pe)
{
    static_assert(!PROJ || (!NMAJ && !AF32), "the projection reads bf16 h and K-major weights");
    constexpr uint32_t kTmem = BN <= 32 ? 32 : BN <= 64 ? 64 : BN <= 128 ? 128 : 256;  // accumulator columns
    constexpr int kBBytes = BN * 128;      // BN x 64 K (K-major) or 64 K x BN (N-major)
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ GemmBars bars;
    __shared__ uint32_t tmem_base;
    __shared__ int fail;
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                            ~static_cast<uintptr_t>(1023));
    const int nk = (p.K + 63) / 64;
    const int ks = SPLIT ? p.ksplit : 1;                // CTAs of the cluster sharing the K range
    const int kz = blockIdx.x % ks;                      // this CTA's share: chunks [c_begin, c_end)
    const int c_begin = kz * nk / ks, nkl = (kz + 1) * nk / ks - c_begin;
    const int NS = p.stages;                             // ring stages (<= kStages)
    // A stages sit a_stride apart: the tile's RT rows (rounded to 8).  The MMA
    // still reads 64 or 128 rows from its stage base: the rows past RT come from
    // the next stages or the B ring (inside the allocation), land in accumulator
    // rows >= RT and are never stored.
    // An fp32 A has no A stages of its own: each converter thread writes its
    // bf16 row over the first half of its raw fp32 row, which it has read
    // before, so a stage's bf16 tile is the first 16 KB of its raw stage.
    const int AS = AF32 ? 0 : p.a_stride;
    const int raw_box = SHORT ? p.a_stride : 128 * 128, raw_bytes = 2 * raw_box;  // fp32 A: two 32-column boxes
    unsigned char *sa = smem;                            // NS x A tile (bf16 A)
    unsigned char *sb = sa + NS * AS;                    // NS x B tile
    unsigned char *sr = sb + NS * kBBytes;               // NS x raw fp32 A, then its bf16 tile (AF32)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool epi = warp >= 2 && warp < 6;              // an epilogue warp
    const int R = p.rblk, RT = R * p.hpg;                // row blocks and rows per tile (<= 128)
    constexpr bool m64 = M64;
    const int mt = blockIdx.x / ks, n0 = blockIdx.y * BN, g = blockIdx.z;
    const int m0 = mt * RT;
    const uint32_t a_bytes = static_cast<uint32_t>(RT) * 128;  // per 64-column (bf16) or 32-column (fp32) box
    const uint64_t lim = kWaitLimitNs;

    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&bars.full[s], 1);
            mbar_init(&bars.raw_full[s], 1);
            mbar_init(&bars.conv_done[s], 4);
            mbar_init(&bars.empty[s], 1);
        }
        mbar_init(&bars.done, 1);
        mbar_init(&bars.recv, 1);
        fail = 0;
        tc::fence_barrier_init();
        if (SPLIT)  // the slabs of the other CTAs
            tc::mbar_arrive_expect_tx(smem_u32(&bars.recv), static_cast<uint32_t>((ks - 1) * (BN / ks) * recv_rows(RT) * 4));
    }
    if (warp == 1) {
        tc::tmem_alloc(smem_u32(&tmem_base), kTmem);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // a peer's shared memory is written only once its CTA has started: arrive
    // now, wait before the first such write
    if (SPLIT) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    // the activations come from the previous launch; with early_weights the
    // producer sends for the first weight tiles before it waits
    const bool early = !PROJ && p.early_weights && warp == 0;
    if (!early) griddep_wait();
    // the projection writes the cache: its dependents launch only once it has
    // completed (the attention kernel loads cache tiles before its own wait)
    if (!PROJ && !early) griddep_launch_dependents();
    const uint32_t tmem = tmem_base;
    auto bail = [&]() {
        record_status(p.status, kStatusTimeout);
        fail = 1;
    };
    bool ep_ok = false;  // split K: this epilogue thread saw its CTA's MMAs complete

    if (warp == 0) {
        // ---- A and weight tiles by TMA (converged warp, one elected lane
        // issues: with a lone lane and a division per chunk this loop took
        // 0.45 us a chunk and was the kernel's pace -- W_O of 640 rows 15 us
        // for 32 chunks, the projection of 640 rows 18.5)
        const CUtensorMap *mb = &maps.b;
        int brow = g * p.N + n0;
        uint32_t bbytes = kBBytes;
        if constexpr (PROJ) {
            const int ty = blockIdx.y, region = ty < pe.tiles_lat ? 0 : ty == pe.tiles_lat ? 1 : 2;
            mb = region == 0 ? &maps.b : region == 1 ? &maps.b2 : &maps.b3;
            brow = region == 0 ? n0 : region == 1 ? 0 : (ty - pe.tiles_lat - 1) * BN;
            bbytes = pe.box_bytes[region];
        }
        tc::prefetch_tensormap(mb);
        tc::prefetch_tensormap(&maps.a);
        auto load_b = [&](int c, int s) {
            const uint32_t fb = smem_u32(&bars.full[s]), dst = smem_u32(sb + s * kBBytes);
            tc::mbar_arrive_expect_tx_elect(fb, bbytes + (AF32 ? 0u : a_bytes));
            if (NMAJ) {
                // rows = K of group g, columns = N: one 64 x 64 box per 64 columns
#pragma unroll
                for (int j = 0; j < BN / 64; ++j)
                    tc::tma_load_2d_elect(dst + j * 64 * 128, &maps.b, n0 + 64 * j, g * p.K + 64 * c, fb);
            } else {
                tc::tma_load_2d_elect(dst, mb, 64 * c, brow, fb);
            }
        };
        auto load_a = [&](int c, int s) {
            if (AF32) {
                const uint32_t rb = smem_u32(&bars.raw_full[s]), rdst = smem_u32(sr + s * raw_bytes);
                tc::mbar_arrive_expect_tx_elect(rb, 2 * a_bytes);
                tc::tma_load_4d_elect(rdst, &maps.a, 64 * c, 0, g, mt * R, rb);
                tc::tma_load_4d_elect(rdst + raw_box, &maps.a, 64 * c + 32, 0, g, mt * R, rb);
            } else {
                tc::tma_load_4d_elect(smem_u32(sa + s * AS), &maps.a, 64 * c, 0, g, mt * R, smem_u32(&bars.full[s]));
            }
        };
        const int head = nkl < NS ? nkl : NS;  // the ring's first round
        for (int s = 0; s < head; ++s) {
            load_b(c_begin + s, s);
            if (!early) load_a(c_begin + s, s);
        }
        if (early) {
            griddep_wait();
            griddep_launch_dependents();
            for (int s = 0; s < head; ++s) load_a(c_begin + s, s);
        }
        for (int c = c_begin + head, s = 0, par = 0; c < c_begin + nkl; ++c) {
            if (!mbar_wait_warp(smem_u32(&bars.empty[s]), par, lim)) {
                if (lane == 0) bail();
                break;
            }
            load_b(c, s);
            load_a(c, s);
            if (++s == NS) {
                s = 0;
                par ^= 1;
            }
        }
    } else if (warp == 1) {
        // ---- MMA issuer (converged warp, one elected lane issues)
        const uint32_t idesc = tc::idesc_bf16_f32(m64 ? 64 : 128, BN, false, NMAJ);
        const uint64_t da = tc::smem_desc(0, 16, 1024, tc::kSwizzle128B);
        const uint64_t db = NMAJ ? tc::smem_desc(0, 64 * 128, 1024, tc::kSwizzle128B)
                                 : tc::smem_desc(0, 16, 1024, tc::kSwizzle128B);
        auto with_addr = [](uint64_t tmpl, uint32_t saddr) {
            return tmpl | static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
        };
        bool ok = true;
        for (int cc = 0, s = 0, par = 0; cc < nkl; ++cc) {
            ok = mbar_wait_warp(smem_u32(&bars.full[s]), par, lim) &&
                 (!AF32 || mbar_wait_warp(smem_u32(&bars.conv_done[s]), par, lim));
            if (!ok) break;
            tc::fence_after_sync();
            // four steps of 16 along K: 32 bytes of a K-major operand, 16 rows of an N-major one
            tc::mma4_bf16_commit_elect(tmem, with_addr(da, smem_u32(AF32 ? sr + s * raw_bytes : sa + s * AS)),
                                       with_addr(db, smem_u32(sb + s * kBBytes)), idesc, cc != 0, 2, NMAJ ? 16 * 128 / 16 : 2,
                                       smem_u32(&bars.empty[s]));
            if (++s == NS) {
                s = 0;
                par ^= 1;
            }
        }
        if (!ok && lane == 0) bail();
        tc::commit_elect(smem_u32(&bars.done));
    } else {
        if (AF32) {
            // ---- fp32 -> bf16: thread r converts tile row r (two 128-byte
            // swizzled fp32 rows), all of it read before the first write: in
            // turns, each write held back the next read, 900 cycles a chunk
            const int r = (tid - 64) & 127;
            // A stage belongs to one set, which so waits for each of its phases in
            // turn: a wait by parity must not miss one.
            const int set = warp < 6 ? 0 : 1, sets = static_cast<int>(blockDim.x - 64) / 128;
            for (int cc = 0, s = 0, par = 0; cc < nkl; ++cc) {
                const int cs = s, cp = par;
                if (++s == NS) {
                    s = 0;
                    par ^= 1;
                }
                if (sets == 2 && (cs & 1) != set) continue;
                if (!mbar_wait_warp(smem_u32(&bars.raw_full[cs]), cp, lim)) {
                    if (lane == 0) bail();
                    break;
                }
                if (!SHORT || r < RT) {
                    const uint4 *src0 = reinterpret_cast<const uint4 *>(sr + cs * raw_bytes + r * 128);
                    const uint4 *src1 = reinterpret_cast<const uint4 *>(sr + cs * raw_bytes + raw_box + r * 128);
                    uint4 *dst = reinterpret_cast<uint4 *>(sr + cs * raw_bytes + r * 128);  // over src0, in place
                    float4 x[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        x[j] = *reinterpret_cast<const float4 *>(&(j < 8 ? src0 : src1)[(j & 7) ^ (r & 7)]);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        // bf16 16-byte chunk j = fp32 chunks 2j, 2j + 1
                        const float4 a = x[2 * j], b = x[2 * j + 1];
                        const __nv_bfloat162 b0 = __floats2bfloat162_rn(a.x, a.y), b1 = __floats2bfloat162_rn(a.z, a.w);
                        const __nv_bfloat162 b2 = __floats2bfloat162_rn(b.x, b.y), b3 = __floats2bfloat162_rn(b.z, b.w);
                        dst[j ^ (r & 7)] =
                            make_uint4(*reinterpret_cast<const uint32_t *>(&b0), *reinterpret_cast<const uint32_t *>(&b1),
                                       *reinterpret_cast<const uint32_t *>(&b2), *reinterpret_cast<const uint32_t *>(&b3));
                    }
                }
                tc::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(smem_u32(&bars.conv_done[cs]));
            }
        }
        if (!PROJ && !AF32 && pe.rope_src) {
            // ---- the absorption's positional query, while the MMAs run.  The
            // tile's rows are whole (b, i) blocks of hpg heads (row m of group g
            // is head g hpg + m % hpg of token m / hpg), which share one
            // position: an item is one (token, pair) with one angle, applied to
            // the pair of every head of the group.  The items of this row tile
            // are spread over the CTAs that share it (column tiles, K shares).
            const int half = pe.d_rope / 2, hpg = p.hpg;
            const int slots = static_cast<int>(gridDim.y) * ks, slot = static_cast<int>(blockIdx.y) * ks + kz;
            const int tok0 = m0 / hpg, items = (min(RT, p.M - m0) / hpg) * half;
            // pair k: elements (k, k + half) in the half-split style, (2k, 2k + 1) interleaved
            const int s0 = pe.style == 0 ? 1 : 2, o1 = pe.style == 0 ? half : 1;
            for (int it = slot * 128 + (warp & 3) * 32 + lane; it < items; it += slots * 128) {
                const int k = it % half, bi = tok0 + it / half;  // bi = b q_len + i
                const int b = bi / pe.q_len, i = bi - b * pe.q_len;
                float cs, sn;
                rope_cos_sin(static_cast<int64_t>(__ldg(pe.kv_len + b)) - pe.q_len + i, pe.turns.f[k], &cs, &sn);
                const int64_t row0 = static_cast<int64_t>(bi) * p.blk + static_cast<int64_t>(g) * hpg;
                const int c0 = s0 * k, c1 = o1 + s0 * k;
                for (int h0 = 0; h0 < hpg; h0 += 4) {
                    uint16_t x0[4], x1[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (h0 + u < hpg) {
                            const uint16_t *src = pe.rope_src + (row0 + h0 + u) * pe.d_rope;
                            x0[u] = __ldg(src + c0);
                            x1[u] = __ldg(src + c1);
                        }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (h0 + u < hpg) {
                            const float a0 = __uint_as_float(static_cast<uint32_t>(x0[u]) << 16);
                            const float a1 = __uint_as_float(static_cast<uint32_t>(x1[u]) << 16);
                            uint16_t *dst = static_cast<uint16_t *>(p.C) + (row0 + h0 + u) * p.ldc + pe.rank;
                            dst[c0] = __bfloat16_as_ushort(__float2bfloat16_rn(a0 * cs - a1 * sn));
                            dst[c1] = __bfloat16_as_ushort(__float2bfloat16_rn(a1 * cs + a0 * sn));
                        }
                }
            }
        }
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31
        const bool ok = epi && mbar_wait_warp(smem_u32(&bars.done), 0, lim);
        if (epi && !ok && lane == 0) bail();
        const bool good = ok && !fail;
        const int q = warp & 3;
        const int i = tile_row(m64, q, lane);
        const int me = m0 + q * (m64 ? 16 : 32) + lane;
        const uint32_t t_lane = tmem + (static_cast<uint32_t>(q * 32) << 16);
        tc::fence_after_sync();
        if constexpr (SPLIT) {
            ep_ok = good;  // the partial leaves below
        } else if (!PROJ && p.tma_out) {
            if constexpr (!PROJ) {
                if (epi)
                    drain_tile_tma<BN>(t_lane, smem, i, RT, good, [&](int j, uint32_t src) {
                        if (n0 + j < p.N) tc::tma_store_4d(&maps.c, src, n0 + j, 0, g, mt * R);
                    });
            }
        } else if (good) {
            unsigned char *stage = smem + q * kDrainWarp;  // in the ring: its tiles have been read
            if (PROJ) {
                const int rows = m64 ? min(16, min(RT, p.M - m0) - q * 16) : min(RT, p.M - m0) - q * 32;
                proj_epilogue<BN>(p, pe, t_lane, stage, lane, me, rows);
            } else {
                // rows of C that are not whole 16 bytes: 8 bytes a store where they
                // are whole 8, else (and at the last columns) element by element
                const bool eight = p.ldc % 4 == 0;
                uint16_t *crow = i < RT && me < p.M ? static_cast<uint16_t *>(p.C) + phys_row(p, g, me) * p.ldc : nullptr;
                drain_tile<BN>(t_lane, stage, lane, [&](int col) {
                    const int n = n0 + col;
                    const bool full = eight && n + 8 <= p.N;
                    const int left = full ? 0 : p.N - n;  // columns to store one by one
                    return [=](int r, const uint4 &v) {
                        uint16_t *row = shfl_ptr(crow, r);
                        store8_if(row && full, row + n, v.x, v.y);
                        store8_if(row && full, row + n + 4, v.z, v.w);
                        if (row && left > 0) {
                            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                if (e < left) row[n + e] = static_cast<uint16_t>(w[e / 2] >> (16 * (e % 2)));
                        }
                    };
                });
            }
        }
    }
    if constexpr (SPLIT) {
        // (1) the CTA's partial into its ring (its own MMAs are done), a slab
        // [four columns][row] for every owner: CTA o owns columns [o cw, (o + 1)
        // cw); (2) one bulk copy a peer takes its slab there, behind the peer's
        // ring, and completes on the peer's barrier; (3) each owner sums its
        // slice in rank order (four columns per step) and stores the bf16
        // result.  Remote stores of the same 30 KB, 512 bytes a warp, and a
        // cluster barrier took 2700 cycles where the copies take 1900.
        const int cw = BN / ks, RP = recv_rows(RT);
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // every CTA has started
        if (ep_ok && !fail) {
            tc::fence_after_sync();
            const int q = warp & 3, i = tile_row(m64, q, lane);
            const uint32_t t_lane = tmem + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll 1
            for (int j = 0; j < BN; j += 32) {
                uint32_t v[2][16];
                tc::ld_32x32b_x16(t_lane + j, v[0]);
                tc::ld_32x32b_x16(t_lane + j + 16, v[1]);
                tc::wait_ld();
                if (i < RT) {  // (the slabs of the owners follow one another: column c at group c / 4)
                    uint4 *dst = reinterpret_cast<uint4 *>(smem) + j / 4 * RP + i;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const uint32_t *x = &v[e / 4][4 * (e % 4)];
                        dst[e * RP] = make_uint4(x[0], x[1], x[2], x[3]);
                    }
                }
                __syncwarp();
            }
            tc::fence_proxy_async_smem();
        }
        const uint32_t slab = static_cast<uint32_t>(cw * RP * 4);
        bool got = false;
        if (epi) {
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (warp == 2 && lane == 0 && ep_ok && !fail) {
                for (int d = 1; d < ks; ++d) {
                    const uint32_t o = static_cast<uint32_t>((kz + d) & (ks - 1));
                    tc::bulk_copy_cluster(tc::mapa(smem_u32(smem) + p.recv_off + kz * slab, o), smem_u32(smem) + o * slab, slab,
                                          tc::mapa(smem_u32(&bars.recv), o));
                }
            }
            got = mbar_wait_warp(smem_u32(&bars.recv), 0, lim);
            if (!got && lane == 0) bail();
        }
        __syncwarp();
        // a CTA leaves once every copy from its shared memory has landed
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        if (got && !fail) {
            const int q4 = cw / 4;  // 4, 8 or 16: the 128 threads keep their columns and step 128 / q4 rows
            const float4 *own = reinterpret_cast<const float4 *>(smem), *recv = reinterpret_cast<const float4 *>(smem + p.recv_off);
            const int ce = (tid - 64) % q4, n = n0 + kz * cw + 4 * ce;
#pragma unroll 2
            for (int i = (tid - 64) / q4; i < RT; i += 128 / q4) {
                const int me = m0 + i;
                float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int r = 0; r < 4; ++r) {  // ks is 2 or 4
                    if (r >= ks) break;
                    const float4 v = (r == kz ? own : recv)[(r * q4 + ce) * RP + i];
                    acc.x += v.x;
                    acc.y += v.y;
                    acc.z += v.z;
                    acc.w += v.w;
                }
                if (me >= p.M) continue;
                uint16_t *dst = static_cast<uint16_t *>(p.C) + phys_row(p, g, me) * p.ldc + n;
                const __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
                const uint32_t w[2] = {*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi)};
                if (n + 4 <= p.N && p.ldc % 4 == 0) {
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(w[0], w[1]);
                } else {
                    for (int e = 0; e < 4 && n + e < p.N; ++e) dst[e] = static_cast<uint16_t>(w[e / 2] >> (16 * (e % 2)));
                }
            }
        }
        __syncwarp();
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, kTmem);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode_gemm = nullptr;

cudaError_t get_encoder()
{
    if (g_encode_gemm) return cudaSuccess;
    cudaDriverEntryPointQueryResult q;
    void *fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return e != cudaSuccess ? e : cudaErrorNotSupported;
    g_encode_gemm = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return cudaSuccess;
}

int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

// A: (K, head in group, group, row block) with the row mapping's strides.
bool encode_a(const GroupGemm &p, int rblk, bool f32, CUtensorMap *ma)
{
    const int es = f32 ? 4 : 2;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(p.K), static_cast<cuuint64_t>(p.hpg), static_cast<cuuint64_t>(p.G),
                          static_cast<cuuint64_t>(p.M / p.hpg)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(p.lda) * es, static_cast<cuuint64_t>(p.hpg) * p.lda * es,
                             static_cast<cuuint64_t>(p.blk) * p.lda * es};
    cuuint32_t box[4] = {f32 ? 32u : 64u, static_cast<cuuint32_t>(p.hpg), 1u, static_cast<cuuint32_t>(rblk)};
    cuuint32_t es4[4] = {1, 1, 1, 1};
    return g_encode_gemm(ma, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4,
                         const_cast<void *>(p.A), dims, strides, box, es4, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The results: C (column, head in group, group, row block) in boxes of 64 columns
// x a tile's rows; only rows of whole 16 bytes.
bool encode_c(const GroupGemm &p, int rblk, CUtensorMap *mc)
{
    if (p.ldc % 8) return false;
    cuuint64_t dims[4] = {static_cast<cuuint64_t>(p.N), static_cast<cuuint64_t>(p.hpg), static_cast<cuuint64_t>(p.G),
                          static_cast<cuuint64_t>(p.M / p.hpg)};
    cuuint64_t strides[3] = {static_cast<cuuint64_t>(p.ldc) * 2, static_cast<cuuint64_t>(p.hpg) * p.ldc * 2,
                             static_cast<cuuint64_t>(p.blk) * p.ldc * 2};
    cuuint32_t box[4] = {64u, static_cast<cuuint32_t>(p.hpg), 1u, static_cast<cuuint32_t>(rblk)}, es4[4] = {1, 1, 1, 1};
    return g_encode_gemm(mc, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, p.C, dims, strides, box, es4,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A K-major weight [rows][K] in boxes of 64 K x box_rows rows.
bool encode_kmajor(const void *w, int64_t rows, int K, int box_rows, CUtensorMap *mb)
{
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(K), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(K) * 2};
    cuuint32_t box[2] = {64u, static_cast<cuuint32_t>(box_rows)}, es2[2] = {1, 1};
    return g_encode_gemm(mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(w), dims, strides, box, es2,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Row blocks per tile: the fewest tiles of at most 128 rows, evenly filled (160
// rows: 80 + 80, not 128 + 32; a short A box leaves the tile's other rows
// stale, and their results are dropped).
int rows_per_tile(const GroupGemm &p)
{
    const int blocks = p.M / p.hpg, most = 128 / p.hpg;
    const int tiles = (blocks + most - 1) / most;
    return (blocks + tiles - 1) / tiles;
}

// CTAs that share a tile's K range.  Split K over a cluster when the tiles are
// short (<= 64 rows: a small batch), K is deep (>= 8 chunks) and the tiles alone
// would leave most SMs idle: up to 4 ways, at least two chunks each, with a ring
// that lets two CTAs share an SM, so that the split grid runs in one wave (an
// fp32 A: one CTA per SM).  Tiles of more rows that would fill fewer than half
// the SMs (a mid-size batch against a wide weight): split K as well, one CTA per
// SM, at least eight chunks per share.  (Not for an fp32 A: there the reduction
// cost as much as the split saved.)
int split_of(bool f32, int rt, int64_t tiles, int nk, int sms)
{
    int ks = 1;
    if (rt <= 64 && nk >= 8)
        while (ks < 4 && tiles * ks * 2 <= (f32 ? sms : 2 * sms) && nk >= 4 * ks) ks *= 2;
    if (rt > 64 && !f32 && nk >= 16)
        while (ks < 4 && tiles * ks * 2 <= sms && nk >= 8 * ks) ks *= 2;
    return ks;
}

// What column tiles of bn cost (bf16 A), in KB through a CTA's shared memory:
// its chunks of both operands, four times its partial if K is split (staged,
// sent, received, summed) and 150 for the exchange's own latency, times the
// waves of CTAs.  W_UV + W_O of 32 heads, 2048 columns, with 128 against 64
// columns: 64 rows 12.6 and 11.2 us, 128 rows 13.9 and 12.6, 160 rows 13.3 and
// 13.7, 320 rows 17.3 and 14.9, 512 rows 20.9 and 17.9, 640 rows (two waves of
// 64) 21.7 and more.
int64_t tile_cost(const GroupGemm &p, int bn, int sms)
{
    const int rt = rows_per_tile(p) * p.hpg, nk = (p.K + 63) / 64;
    const int64_t tiles = static_cast<int64_t>((p.M + rt - 1) / rt) * ((p.N + bn - 1) / bn) * p.G;
    const int ks = split_of(false, rt, tiles, nk, sms);
    const int64_t slots = ks > 1 && rt <= 64 ? 2 * sms : sms;
    const int64_t in = static_cast<int64_t>((nk + ks - 1) / ks) * (rt + bn) * 128;
    const int64_t exchange = ks > 1 ? 4 * 4 * static_cast<int64_t>(rt) * bn + 150 * 1024 : 0;
    return (tiles * ks + slots - 1) / slots * (in + exchange);
}

// The ring for tiles of rt rows: as many stages as fit `budget` bytes, at most
// kStages and the K chunks.  A bf16 A stage holds just the tile's rows (rounded
// to 8), so that short tiles stream their weight with more chunks in flight.
// An MMA reads mma_rows (64 or 128) rows from its stage's base, and the last
// stage's rows past the tile may lie past the ring (an fp32 A's stages are its
// end): the allocation covers them, and they count against the budget.  (They
// once did not: 20 rows of 24 heads of 128 against W_O asked for 232704 bytes.)
struct Ring {
    int stages, a_stride;
    size_t bytes;
};

template <int BN, bool AF32>
Ring ring_for(int rt, int mma_rows, int chunks, size_t budget)
{
    Ring r;
    r.a_stride = AF32 && rt > kShortRows ? 128 * 128 : (rt + 7) / 8 * 8 * 128;
    const size_t a_bytes = AF32 ? 2 * r.a_stride : r.a_stride;  // fp32 A: raw stage, bf16 in place
    const size_t per_stage = a_bytes + BN * 128;
    int ns = static_cast<int>(budget / per_stage);
    if (ns > kStages) ns = kStages;
    if (ns > chunks) ns = chunks;
    if (ns < 1) ns = 1;
    auto bytes = [&](int n) {
        const size_t window = (AF32 ? static_cast<size_t>(n) * BN * 128 : 0) + (n - 1) * a_bytes + mma_rows * 128;
        return n * per_stage > window ? n * per_stage : window;
    };
    while (ns > 1 && bytes(ns) > budget) --ns;
    r.stages = ns;
    r.bytes = bytes(ns);
    return r;
}

// Shared memory of a CTA that has an SM for itself, behind the alignment of the
// ring; 640 rows of the projection (40 KB a chunk) 14.8 us with a ring of four
// chunks, 13.6 with the five that fit.
constexpr size_t kRingBytes = 224 * 1024;

using GemmKernel = void (*)(GroupGemm, GemmMaps<false>, ProjEpi);

template <auto Kernel, class K>
cudaError_t take_kernel(K *kernel)
{
    *kernel = Kernel;
    return allow_smem<Kernel>(1024 + kRingBytes);
}

// The kernel for tiles of rt rows.  split_of() splits neither the absorption
// (NMAJ: at most four K chunks) nor an fp32 A in tiles past 64 rows.
template <int BN, bool NMAJ, bool AF32>
cudaError_t gemm_kernel(int rt, bool split, GemmKernel *kernel)
{
    const bool m64 = rt <= kM64Rows;
    if (split) {
        if constexpr (!NMAJ) {
            if (m64) return take_kernel<gemm_tc_kernel<BN, false, AF32, false, AF32, true, true>>(kernel);
            if constexpr (!AF32) return take_kernel<gemm_tc_kernel<BN, false, false, false, false, true, false>>(kernel);
        }
        return cudaErrorInvalidConfiguration;
    }
    if (m64) return take_kernel<gemm_tc_kernel<BN, NMAJ, AF32, false, AF32, false, true>>(kernel);
    if constexpr (AF32)
        if (rt <= kShortRows) return take_kernel<gemm_tc_kernel<BN, NMAJ, AF32, false, true, false, false>>(kernel);
    return take_kernel<gemm_tc_kernel<BN, NMAJ, AF32, false, false, false, false>>(kernel);
}

template <int BN, bool NMAJ, bool AF32>
cudaError_t launch_tc(const GroupGemm &p, int sms, cudaStream_t st, const ProjEpi *rope = nullptr)
{
    cudaError_t e = get_encoder();
    if (e != cudaSuccess) return e;
    if (p.hpg < 1 || p.hpg > 128 || p.M % p.hpg) return cudaErrorInvalidValue;
    int rblk = rows_per_tile(p);
    const int ntiles = (p.N + BN - 1) / BN;
    const int nk = (p.K + 63) / 64;
    auto tiles_for = [&](int rb) { return static_cast<int64_t>((p.M / p.hpg + rb - 1) / rb) * ntiles * p.G; };
    // A grid too small to spread over the SMs and K too short to split (the
    // split below wants deep K): shorter row tiles instead, each CTA
    // re-reading its (small) weight tile from L2
    if (nk < 8)
        while (tiles_for(rblk) < 64 && rblk > 1 && rblk * p.hpg > 16) rblk = (rblk + 1) / 2;
    // fp32 A, more tiles than SMs (W_UV of a large batch): two CTAs share an SM,
    // in tiles as short as still leave one wave.  640 rows of 32 heads, 12.2 us
    // with 160 tiles of 128 rows and a ring of two chunks, 10.6 with 304 of 68
    // and four.
    const bool pairs = AF32 && tiles_for(rblk) > sms;
    if (pairs) {
        const int64_t n = 2 * sms / (static_cast<int64_t>(ntiles) * p.G), blocks = p.M / p.hpg;
        if (n * rblk >= blocks) rblk = static_cast<int>((blocks + n - 1) / n);
    }
    CUtensorMap ma, mb;
    if (!encode_a(p, rblk, AF32, &ma)) return cudaErrorInvalidValue;
    if (NMAJ) {  // [G K rows][N columns], 64 x 64 boxes
        cuuint64_t dims[2] = {static_cast<cuuint64_t>(p.N), static_cast<cuuint64_t>(p.G) * p.K};
        cuuint64_t strides[1] = {static_cast<cuuint64_t>(p.N) * 2};
        cuuint32_t box[2] = {64u, 64u}, es2[2] = {1, 1};
        CUresult r = g_encode_gemm(&mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(p.B), dims, strides,
                                   box, es2, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    } else if (!encode_kmajor(p.B, static_cast<int64_t>(p.G) * p.N, p.K, BN, &mb)) {  // [G N rows][K columns]
        return cudaErrorInvalidValue;
    }
    const int rt = rblk * p.hpg;
    const int mtiles = (p.M + rt - 1) / rt;
    const int64_t tiles = static_cast<int64_t>(mtiles) * ntiles * p.G;
    const int ks = split_of(AF32, rt, tiles, nk, sms);
    // Split K: the partial's staging lies in the ring, what the cluster sends
    // behind it (at most 66 KB each).  A short tile's ring leaves room for a
    // second CTA.
    const size_t part = ks > 1 ? static_cast<size_t>(BN) * recv_rows(rt) * 4 : 0;
    const size_t room = pairs || (ks > 1 && rt <= 64 && !AF32) ? 111 * 1024 : kRingBytes;
    size_t budget = room - part;
    const Ring ring = ring_for<BN, AF32>(rt, rt <= kM64Rows ? 64 : 128, (nk + ks - 1) / ks, budget);
    GroupGemm q = p;
    q.stages = ring.stages;
    q.a_stride = ring.a_stride;
    q.rblk = rblk;
    q.ksplit = ks;
    q.recv_off = static_cast<int>(ring.bytes > part ? ring.bytes : part);
    size_t smem = 1024 + (ks > 1 ? q.recv_off + part : ring.bytes);
    CUtensorMap mc = mb;
    q.tma_out = encode_c(p, rblk, &mc);
    const size_t stage = q.tma_out ? BN * 256 : kDrainBytes;  // the results' staging
    if (smem < 1024 + stage) smem = 1024 + stage;
    GemmKernel kernel;
    if ((e = gemm_kernel<BN, NMAJ, AF32>(rt, ks > 1, &kernel)) != cudaSuccess) return e;
    const int threads = AF32 && ks == 1 && !pairs ? kConvThreads : kGemmThreads;
    dim3 grid(mtiles * ks, ntiles, p.G);
    ProjEpi none{};
    return launch_dependent(kernel, grid, dim3(threads), smem, st, ks, q,
                            GemmMaps<false>{ma, mb, mc}, rope ? *rope : none);
}

// The projection: h [M = batch n_new, hidden] against W^DKV (rank rows), W^KR
// (d_rope rows, one column tile) and W^Q (H (d_nope + d_rope) rows, or none).
template <int BN>
cudaError_t launch_proj(const mla_dims &d, const CacheView &c, int batch, int n_new, const void *h,
                        const void *w_dkv, const void *w_kr, const void *w_q, const int32_t *start_pos, void *q_nope,
                        void *q_pe, unsigned *status, cudaStream_t st)
{
    cudaError_t e = get_encoder();
    if (e != cudaSuccess) return e;
    GroupGemm p{};
    p.M = batch * n_new;
    p.K = d.hidden;
    p.G = 1;
    p.hpg = 1;
    p.blk = 1;
    p.A = h;
    p.a_f32 = 0;
    p.lda = d.hidden;
    p.status = status;
    const int nq = w_q ? d.num_heads * (d.d_nope + d.d_rope) : 0;
    const int lat_rows = d.rank < BN ? d.rank : BN, rope_rows = d.d_rope < BN ? d.d_rope : BN, q_rows = nq < BN ? nq : BN;
    ProjEpi pe{};
    pe.cache = c;
    pe.start_pos = start_pos;
    pe.q_nope = static_cast<uint16_t *>(q_nope);
    pe.q_pe = static_cast<uint16_t *>(q_pe);
    pe.n_new = n_new;
    pe.rank = d.rank;
    pe.d_rope = d.d_rope;
    pe.d_nope = d.d_nope;
    pe.heads = d.num_heads;
    pe.style = d.rope_style;
    pe.turns = rope_turns(d.d_rope, d.rope_base);
    pe.tiles_lat = (d.rank + BN - 1) / BN;
    pe.box_bytes[0] = static_cast<uint32_t>(lat_rows) * 128;
    pe.box_bytes[1] = static_cast<uint32_t>(rope_rows) * 128;
    pe.box_bytes[2] = static_cast<uint32_t>(q_rows) * 128;
    const int rblk = rows_per_tile(p);
    CUtensorMap ma, m0, m1, m2;
    if (!encode_a(p, rblk, false, &ma) || !encode_kmajor(w_dkv, d.rank, d.hidden, lat_rows, &m0) ||
        !encode_kmajor(w_kr, d.d_rope, d.hidden, rope_rows, &m1))
        return cudaErrorInvalidValue;
    if (w_q) {
        if (!encode_kmajor(w_q, nq, d.hidden, q_rows, &m2)) return cudaErrorInvalidValue;
    } else {
        m2 = m0;  // never read: no query tiles
    }
    const int tiles = pe.tiles_lat + 1 + (nq + BN - 1) / BN;
    p.N = tiles * BN;
    const Ring ring = ring_for<BN, false>(rblk, 128, (p.K + 63) / 64, kRingBytes);
    size_t smem = 1024 + ring.bytes;
    p.stages = ring.stages;
    p.a_stride = ring.a_stride;
    p.rblk = rblk;
    p.ksplit = 1;
    if (smem < 1024 + kDrainBytes) smem = 1024 + kDrainBytes;  // the results' staging
    constexpr bool kShort = BN == 64;  // (few rows take 64 columns)
    void (*kernel)(GroupGemm, GemmMaps<true>, ProjEpi);
    e = kShort && rblk <= 64 ? take_kernel<gemm_tc_kernel<BN, false, false, true, false, false, kShort>>(&kernel)
                             : take_kernel<gemm_tc_kernel<BN, false, false, true, false, false, false>>(&kernel);
    if (e != cudaSuccess) return e;
    dim3 grid((p.M + rblk - 1) / rblk, tiles, 1);
    return launch_dependent(kernel, grid, dim3(kGemmThreads), smem, st, 1, p,
                            GemmMaps<true>{ma, m0, m1, m2}, pe);
}

}  // namespace

// The absorption GEMM with the positional-query rotation in its epilogue
// warps (N-major W_UK, bf16 q_nope).
cudaError_t launch_absorb_gemm(const GroupGemm &p, const mla_dims &d, const void *q_pe, const int32_t *kv_len,
                               int q_len, cudaStream_t st)
{
    if (p.M <= 0 || p.N <= 0 || p.G <= 0) return cudaSuccess;
    ProjEpi r{};
    r.rope_src = static_cast<const uint16_t *>(q_pe);
    r.kv_len = kv_len;
    r.q_len = q_len;
    r.heads = d.num_heads;
    r.rank = d.rank;
    r.d_rope = d.d_rope;
    r.style = d.rope_style;
    r.turns = rope_turns(d.d_rope, d.rope_base);
    const bool narrow = p.N <= 64 || p.M <= 32;
    const int sms = sm_count();
    return narrow ? launch_tc<64, true, false>(p, sms, st, &r) : launch_tc<128, true, false>(p, sms, st, &r);
}

cudaError_t launch_group_gemm(const GroupGemm &p, cudaStream_t st)
{
    if (p.M <= 0 || p.N <= 0 || p.G <= 0) return cudaSuccess;
    // column tile: 64 for narrow outputs and for few rows (more CTAs stream the
    // weight), else 128 -- or, of a bf16 A, what costs a CTA less
    const int sms = sm_count();
    const bool narrow = p.N <= 64 || p.M <= 32 || (!p.a_f32 && tile_cost(p, 64, sms) < tile_cost(p, 128, sms));
    if (p.a_f32) return narrow ? launch_tc<64, false, true>(p, sms, st) : launch_tc<128, false, true>(p, sms, st);
    return narrow ? launch_tc<64, false, false>(p, sms, st) : launch_tc<128, false, false>(p, sms, st);
}

cudaError_t launch_project(const mla_dims &d, const CacheView &c, int batch, int n_new, const void *h,
                           const void *w_dkv, const void *w_kr, const void *w_q, const int32_t *start_pos,
                           void *q_nope, void *q_pe, unsigned *status, cudaStream_t st)
{
    if (batch <= 0 || n_new <= 0) return cudaSuccess;
    // The kernel is bound by filling shared memory (both tiles per K chunk from
    // L2, about 130 GB/s per SM), one CTA per SM: so the column tile with the
    // least waves of CTAs times the bytes a chunk loads, 16 KB of h and 128
    // bytes per column; of equal ones the narrowest.  640 rows of the
    // Llama-3.2-1B shape (4672 columns): 64, 128, 192 and 256 columns take 3 x
    // 24, 2 x 32, 1 x 40 and 1 x 48 KB; 160 rows 1 x 24 with 64 columns.
    const int sms = sm_count();
    const int nq = w_q ? d.num_heads * (d.d_nope + d.d_rope) : 0;
    const int64_t mt = (static_cast<int64_t>(batch) * n_new + 127) / 128;
    int bn = 64;
    int64_t best = 0;
    for (int w : {64, 128, 192, 256}) {
        const int64_t ctas = mt * ((d.rank + w - 1) / w + 1 + (nq + w - 1) / w);
        const int64_t cost = (ctas + sms - 1) / sms * (128 + w);
        if (best == 0 || cost < best) {
            best = cost;
            bn = w;
        }
    }
    if (bn == 256)
        return launch_proj<256>(d, c, batch, n_new, h, w_dkv, w_kr, w_q, start_pos, q_nope, q_pe, status, st);
    if (bn == 192)
        return launch_proj<192>(d, c, batch, n_new, h, w_dkv, w_kr, w_q, start_pos, q_nope, q_pe, status, st);
    if (bn == 128)
        return launch_proj<128>(d, c, batch, n_new, h, w_dkv, w_kr, w_q, start_pos, q_nope, q_pe, status, st);
    return launch_proj<64>(d, c, batch, n_new, h, w_dkv, w_kr, w_q, start_pos, q_nope, q_pe, status, st);
}

}  // namespace gbmla
