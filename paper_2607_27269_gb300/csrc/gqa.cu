// mla_gqa_*: decode attention of the original GQA draft (Sec. 3.1, Eqs. 1-4),
// the model the converted MLA draft replaces, at the same shapes, so that the
// two caches can be compared byte for byte and second for second.  Each KV
// group g of sequence b keeps its own key cache K (stored rotated to its
// position) and value cache V; unit u = b * G + g is one such (sequence,
// group), with kv_len[b] tokens.
//
// The kernel is bound by the cache bytes: a unit has only q_len * H/G query
// rows (3 .. 56 in the draft shapes), so the tensor work is a few percent of
// the pipe, and what has to be hidden is the chain load -> scores -> softmax ->
// values.  One warp is one split-KV partition (the MLA path's partition, over
// the units' 128-token tiles): it keeps its own ring of TMA stages, issues its
// own loads and never waits on another warp, so that the SM's seven warps hide
// each other's chains and the ring keeps 224 KB per SM in flight or in use.
// Within a warp everything between the cache stage and the partial stays in
// registers (mma.m16n8k16, tokens on M, query rows on N in steps of 8):
//   S^T[16 tok, N]  = K (ldmatrix) x Q^T (fragments loaded and rotated once a unit)
//   P^T             = 2^(S^T scale - m) rounded to bf16, transposed 8 x 8 by movmatrix
//   O^T[D, N]      += V^T (ldmatrix.trans) x P^T
// A column's running maximum, sum and accumulators sit in the same lanes, so
// a rescale (a new maximum in a segment's first tile, later only a score that
// passes the base by 2^8) needs no exchange.
// More rows than a warp holds (32, or 24 of width 128) run as row groups (grid y)
// that each read the cache, as do fewer where the partitions leave warps idle.
//
// The first form of this kernel (one CTA per partition, tcgen05 with M = 128
// query rows of which 20 are real, one softmax warp) took 727 us on the
// 128-sequence paged batch (20 rows of 64) and 231 us on eight long sequences
// (3 rows of 128): the serial TMEM round trips per tile set the pace.
#include <cudaTypedefs.h>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace gbmla {
namespace {

constexpr int kTokTile = MLA_SPLIT_TILE;  // 128 tokens per tile of the partition
constexpr int kPage = 64;
constexpr int kStageBytes = 16384;        // K and V of one stage: 64 tokens of width 64, 32 of width 128
constexpr int kStages = 2;                // per warp
constexpr int kWarps = kGqaPartsPerSm;    // 7 warps x 2 stages x 16 KB of shared memory

struct GqaArgs {
    int batch, q_len, groups, hpg, rows, max_kv, num_splits;
    int paged, bt_stride, num_pages;
    float scale_log2;
    int style;
    const int32_t *kv_len;
    const int32_t *block_table;
    const uint16_t *q;  // [B, q_len, H, DK]
    float *o_part, *lse_part;
    unsigned *status;
    RopeTurns turns;
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ void ldsm4_trans(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

__device__ __forceinline__ uint32_t mov_trans(uint32_t x)
{
    uint32_t y;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h2);
}

// The warp's place in its partition: a segment is the partition's run of
// tokens [tok, tok_end) of unit u; stages cut it into TOK tokens each.  All
// members are the same in every lane.
struct Segments {
    int b, g, kv, tok, tok_end;
    int64_t left;  // tiles of the partition not yet in a segment

    // Tile t (of the flat list of all units' tiles) and n tiles from it on.
    __device__ void init(const GqaArgs &a, int64_t t, int64_t n, int lane)
    {
        left = n;
        int64_t before = 0;  // tiles of the sequences before the 32 looked at
        for (int b0 = 0;; b0 += 32) {
            const int bb = b0 + lane;
            const int64_t nb = bb < a.batch ? seq_tiles(a.kv_len[bb], a.q_len, a.max_kv) * a.groups : 0;
            int64_t incl = nb;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, before + incl > t);
            if (hit || b0 + 32 >= a.batch) {
                const int src = hit ? __ffs(hit) - 1 : 31;
                b = b0 + src;
                const int64_t at = t - before - __shfl_sync(0xffffffffu, incl - nb, src);  // tile within the sequence
                kv = a.kv_len[b];
                const int nt = static_cast<int>(seq_tiles(kv, a.q_len, a.max_kv));
                g = static_cast<int>(at / nt);
                open(static_cast<int>(at - static_cast<int64_t>(g) * nt), nt);
                return;
            }
            before += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    // The segment from tile j of the current unit, which has nt tiles.
    __device__ void open(int j, int nt)
    {
        const int n = static_cast<int>(min(static_cast<int64_t>(nt - j), left));
        left -= n;
        tok = j * kTokTile;
        tok_end = min((j + n) * kTokTile, kv);
    }
    __device__ bool more() const { return tok < tok_end; }
    // The next stage's tokens; at a segment's end the next unit's segment
    // (none is left when more() is false then).
    __device__ void next(const GqaArgs &a, int step)
    {
        tok += step;
        if (tok >= tok_end && left > 0) {
            if (++g == a.groups) {
                g = 0;
                do {  // (a length that cannot be served holds no tiles)
                    ++b;
                    kv = a.kv_len[b];
                } while (seq_tiles(kv, a.q_len, a.max_kv) == 0);
            }
            open(0, static_cast<int>(seq_tiles(kv, a.q_len, a.max_kv)));
        }
    }
};

// D: head width.  N: query rows of a row group, rounded up to 8.
template <int D, int N>
__global__ void __launch_bounds__(32 * kWarps, 1)
    gqa_attn_kernel(const __grid_constant__ GqaArgs a, const __grid_constant__ CUtensorMap map_k,
                    const __grid_constant__ CUtensorMap map_v)
{
    constexpr int KA = D / 64;                       // 64-column atoms of a row
    constexpr int TOK = kStageBytes / (4 * D);       // tokens per stage
    constexpr int NJ = N / 8;                        // 8-row column blocks
    constexpr int TB = D == 64 || N <= 16 ? 32 : 16; // tokens scored together (by registers)
    constexpr uint32_t kAtom = TOK * 128;            // TOK rows x 64 columns, 128-byte swizzle
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[kWarps][kStages];
    __shared__ int64_t red64[32];
    __shared__ uint64_t turns[64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int w = 0; w < kWarps; ++w)
            for (int s = 0; s < kStages; ++s) mbar_init(&bars[w][s], 1);
        tc::fence_barrier_init();
        tc::prefetch_tensormap(&map_k);
        tc::prefetch_tensormap(&map_v);
    }
    for (int k = tid; k < D / 2; k += 32 * kWarps) turns[k] = a.turns.f[k];
    // the cache is final when this kernel runs (a cache writer releases its
    // dependents only on completion); the queries and the partial buffers
    // belong to the previous launches: a warp waits before it reads queries
    griddep_launch_dependents();
    // a length that cannot be served holds no tiles, here and in the combine
    if (blockIdx.x == 0 && blockIdx.y == 0) {
        for (int b = tid; b < a.batch; b += 32 * kWarps) {
            const int kv = a.kv_len[b];
            if (kv < a.q_len || kv > a.max_kv) record_status(a.status, kStatusBounds);
        }
    }
    // (the block-wide sums also order the barriers' set-up before their use)
    const int64_t T = block_tile_sum(a.kv_len, a.batch, a.q_len, a.max_kv, red64) * a.groups;
    const int part = warp * gridDim.x + blockIdx.x;  // spread over the SMs first
    const bool mine = T > 0 && part < a.num_splits;
    const int64_t t_begin = mine ? part_begin(part, T, a.num_splits) : 0;
    const int64_t n_tiles = mine ? part_begin(part + 1, T, a.num_splits) - t_begin : 0;
    if (n_tiles == 0) {
        griddep_wait();
        return;
    }
    const int row0 = blockIdx.y * N;                 // first query row of this row group

    const uint32_t ring =
        ((smem_u32(smem_raw) + 1023u) & ~1023u) + static_cast<uint32_t>(warp) * (kStages * kStageBytes);
    const uint64_t policy = gridDim.y == 1 ? tc::policy_evict_first() : tc::policy_evict_last();
    Segments ld;  // where the next load goes
    ld.init(a, t_begin, n_tiles, lane);
    Segments sg = ld;
    // page ids of 32 consecutive pages of the load's unit, one per lane
    int page_u = -1, page_0 = 0, page_id = 0;
    unsigned bad = 0;  // stages whose page id is out of range: not loaded, not used

    // Load the stage at `ld` into slot s, and step on.
    auto load = [&](int s) {
        const int u = ld.b * a.groups + ld.g;
        int blk = u, tok0 = ld.tok;
        bool good = true;
        if (a.paged) {
            const int pg = ld.tok / kPage;
            if (u != page_u || pg >= page_0 + 32) {
                page_u = u;
                page_0 = pg;
                const int n = min(32, (ld.tok_end + kPage - 1) / kPage - pg);
                page_id = lane < n ? a.block_table[static_cast<int64_t>(u) * a.bt_stride + pg + lane] : 0;
            }
            blk = __shfl_sync(0xffffffffu, page_id, pg - page_0);
            tok0 = ld.tok % kPage;
            good = blk >= 0 && blk < a.num_pages;
            if (!good && lane == 0) record_status(a.status, kStatusBounds);
        }
        bad = good ? bad & ~(1u << s) : bad | (1u << s);
        const uint32_t bar = smem_u32(&bars[warp][s]);
        if (lane == 0) tc::mbar_arrive_expect_tx(bar, good ? kStageBytes : 0);
        __syncwarp();
        if (good && lane < 2 * KA)  // K atoms, then V atoms
            tc::tma_load_3d_hint(ring + s * kStageBytes + lane * kAtom, lane < KA ? &map_k : &map_v,
                                 64 * (lane % KA), tok0, blk, bar, policy);
        ld.next(a, TOK);
    };
    for (int s = 0; s < kStages; ++s)
        if (ld.more()) load(s);
    griddep_wait();

    uint32_t qf[D / 16][NJ][2];  // Q^T fragments: rows lane / 4 + 8 j, columns 16 k + 2 (lane % 4) (+ 8)
    float o[D / 16][NJ][4];      // O^T: d = 16 i + lane / 4 (+ 8), rows 8 j + 2 (lane % 4) (+ 1)
    float m[NJ][2], l[NJ][2];    // exponent base and sum of this lane's columns (the sum over its own tokens)
    int lim[NJ][2];              // last visible token of this lane's columns
    int slot = 0;
    uint32_t phase = 0;          // bit s: parity slot s waits for next
    bool ok = true;
    const int r4 = lane >> 2, c4 = (lane & 3) * 2;
    // ldmatrix row and 16-byte column of this lane
    const int k_row = (lane & 7) + ((lane >> 3) & 1) * 8, k_hi = lane >> 4;
    const int v_row = (lane & 7) + (lane >> 4) * 8, v_hi = (lane >> 3) & 1;

    while (sg.more()) {  // one segment (unit) per round
        const int u = sg.b * a.groups + sg.g, kv = sg.kv, tok_end = sg.tok_end, tok_base = sg.tok + kTokTile;
        // ---- the unit's rotated queries, straight into fragments: a rotation
        // pair (k, k + D/2) or (2k, 2k + 1) lies in one lane's columns
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            const int r = row0 + 8 * j + r4;
            const bool real = r < a.rows;
            const int i = r / a.hpg, hh = r - i * a.hpg;
            const int64_t pos = static_cast<int64_t>(kv) - a.q_len + i;
            const uint32_t *src = reinterpret_cast<const uint32_t *>(
                a.q + ((static_cast<int64_t>(sg.b) * a.q_len + (real ? i : 0)) * (a.groups * a.hpg) +
                       sg.g * a.hpg + (real ? hh : 0)) * D + c4);
            uint32_t w[D / 8];
#pragma unroll
            for (int k = 0; k < D / 8; ++k) w[k] = real ? src[4 * k] : 0u;
            if (a.style == 0) {
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
                    float x[2], y[2], cs, sn;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float p = e ? __uint_as_float(w[k] & 0xffff0000u) : __uint_as_float(w[k] << 16);
                        const float q = e ? __uint_as_float(w[k + D / 16] & 0xffff0000u)
                                          : __uint_as_float(w[k + D / 16] << 16);
                        rope_cos_sin(pos, turns[8 * k + c4 + e], &cs, &sn);
                        x[e] = p * cs - q * sn;
                        y[e] = q * cs + p * sn;
                    }
                    w[k] = pack_bf16(x[0], x[1]);
                    w[k + D / 16] = pack_bf16(y[0], y[1]);
                }
            } else {
#pragma unroll
                for (int k = 0; k < D / 8; ++k) {
                    float cs, sn;
                    rope_cos_sin(pos, turns[4 * k + c4 / 2], &cs, &sn);
                    const float p = __uint_as_float(w[k] << 16), q = __uint_as_float(w[k] & 0xffff0000u);
                    w[k] = pack_bf16(p * cs - q * sn, q * cs + p * sn);
                }
            }
#pragma unroll
            for (int k = 0; k < D / 8; ++k) qf[k / 2][j][k % 2] = w[k];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int rc = row0 + 8 * j + c4 + e;
                lim[j][e] = rc < a.rows ? kv - a.q_len + rc / a.hpg : kv - 1;  // (padding columns are never written)
                m[j][e] = -INFINITY;
                l[j][e] = 0.f;
            }
#pragma unroll
            for (int i2 = 0; i2 < D / 16; ++i2)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[i2][j][e] = 0.f;
        }

        for (int tok = sg.tok; tok < tok_end; tok += TOK) {
            const uint32_t kb = ring + slot * kStageBytes, vb = kb + KA * kAtom;
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[warp][slot]), (phase >> slot) & 1u, kWaitLimitNs))) {
                ok = false;
                break;
            }
            phase ^= 1u << slot;
            const int valid = min(kv - tok, TOK);  // cached rows of the stage
            if (valid < TOK) {
                // value rows past the unit's end may hold anything; their weights
                // are 0, and 0 x NaN is NaN: clear them
                for (int x = lane; x < (TOK - valid) * 8 * KA; x += 32) {
                    const int at = x / ((TOK - valid) * 8), y = x - at * (TOK - valid) * 8;
                    asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(vb + at * kAtom + (valid + y / 8) * 128 +
                                                                                  (y % 8) * 16),
                                 "r"(0)
                                 : "memory");
                }
                tc::fence_proxy_async_smem();  // before a later load overwrites them
                __syncwarp();
            }
            const bool need_mask = tok + TOK - 1 > kv - a.q_len;
            const float slack = tok < tok_base ? 0.f : 8.f;  // (log2 domain)
#pragma unroll 1
            for (int t0 = 0; t0 < ((bad >> slot) & 1u ? 0 : valid); t0 += TB) {
                // ---- scores of TB tokens (this lane's: t0 + 16 x + lane / 4 (+ 8)), log2 domain before the base
                float s[TB / 16][NJ][4];
#pragma unroll
                for (int x = 0; x < TB / 16; ++x)
#pragma unroll
                    for (int j = 0; j < NJ; ++j)
#pragma unroll
                        for (int e = 0; e < 4; ++e) s[x][j][e] = 0.f;
#pragma unroll
                for (int k = 0; k < D / 16; ++k) {
#pragma unroll
                    for (int x = 0; x < TB / 16; ++x) {
                        const int row = t0 + 16 * x + k_row;
                        uint32_t ka[4];
                        ldsm4(kb + (k / 4) * kAtom + row * 128 + ((((k % 4) * 2 + k_hi) ^ (lane & 7)) << 4), ka);
#pragma unroll
                        for (int j = 0; j < NJ; ++j) mma16816(s[x][j], ka, qf[k][j]);
                    }
                }
                if (need_mask) {
#pragma unroll
                    for (int x = 0; x < TB / 16; ++x)
#pragma unroll
                        for (int j = 0; j < NJ; ++j)
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (tok + t0 + 16 * x + r4 + (e >> 1) * 8 > lim[j][e & 1]) s[x][j][e] = -INFINITY;
                }
                // ---- exponent bases: the maximum so far in a segment's first
                // tile, later raised only when a score passes one by 2^8.  (A
                // weight of exactly 1 has no rounding error, and in a short
                // sequence the largest weight carries much of the sum: over the
                // maximum of the first 32 tokens alone the error against 64 bits
                // was 5 to 9 % larger at 50 to 600 tokens.)
                float mx[NJ][2];
                bool over = false;
#pragma unroll
                for (int j = 0; j < NJ; ++j)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float v = fmaxf(s[0][j][e], s[0][j][e + 2]);
#pragma unroll
                        for (int x = 1; x < TB / 16; ++x) v = fmaxf(v, fmaxf(s[x][j][e], s[x][j][e + 2]));
                        mx[j][e] = v * a.scale_log2;
                        over |= mx[j][e] > m[j][e] + slack;
                    }
                // (no branch per column: with one, partitions of many short
                // sequences held up the paged batch, 212 us against 202)
                if (__any_sync(0xffffffffu, over)) {
#pragma unroll
                    for (int j = 0; j < NJ; ++j)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            float v = mx[j][e];  // the column's maximum over the eight lanes that hold its tokens
#pragma unroll
                            for (int d = 4; d < 32; d <<= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, d));
                            const bool up = v > m[j][e] + slack;
                            const float alpha = up ? ex2(m[j][e] - v) : 1.f;  // (0 from a base of -inf)
                            m[j][e] = up ? v : m[j][e];
                            l[j][e] *= alpha;
#pragma unroll
                            for (int i = 0; i < D / 16; ++i) {
                                o[i][j][e] *= alpha;
                                o[i][j][e + 2] *= alpha;
                            }
                        }
                }
                // ---- weights, their sums, and P^T as fragments
                uint32_t pf[TB / 16][NJ][2];
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const float m0 = m[j][0] == -INFINITY ? 0.f : m[j][0], m1 = m[j][1] == -INFINITY ? 0.f : m[j][1];
#pragma unroll
                    for (int x = 0; x < TB / 16; ++x)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint32_t w = pack_bf16(ex2(fmaf(s[x][j][2 * h], a.scale_log2, -m0)),
                                                         ex2(fmaf(s[x][j][2 * h + 1], a.scale_log2, -m1)));
                            l[j][0] += __uint_as_float(w << 16);  // the weights the products use
                            l[j][1] += __uint_as_float(w & 0xffff0000u);
                            pf[x][j][h] = mov_trans(w);
                        }
                }
#pragma unroll
                for (int x = 0; x < TB / 16; ++x) {
                    const int row = t0 + 16 * x + v_row;
#pragma unroll
                    for (int i = 0; i < D / 16; ++i) {
                        uint32_t va[4];
                        ldsm4_trans(vb + (i / 4) * kAtom + row * 128 + ((((i % 4) * 2 + v_hi) ^ (lane & 7)) << 4), va);
#pragma unroll
                        for (int j = 0; j < NJ; ++j) mma16816(o[i][j], va, pf[x][j]);
                    }
                }
            }
            __syncwarp();  // every lane has read the slot
            if (ld.more()) load(slot);
            if (++slot == kStages) slot = 0;
        }
        if (!ok) break;

        // ---- the unit's partial: O / l and its log-sum-exp, slot u + part
        const int64_t at = (static_cast<int64_t>(u) + part) * a.rows;
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float sum = l[j][e];
#pragma unroll
                for (int d = 4; d < 32; d <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
                const int r = row0 + 8 * j + c4 + e;
                if (r < a.rows) {
                    const float inv = sum > 0.f ? 1.f / sum : 0.f;
                    float *out = a.o_part + (at + r) * D + r4;
#pragma unroll
                    for (int i = 0; i < D / 16; ++i) {
                        out[16 * i] = o[i][j][e] * inv;
                        out[16 * i + 8] = o[i][j][e + 2] * inv;
                    }
                    if (r4 == 0)
                        a.lse_part[at + r] = sum > 0.f ? (m[j][e] + log2f(sum)) * 0.69314718055994531f : -INFINITY;
                }
            }
        // on to the next unit's segment (every token of this one was used)
        sg.tok = tok_end;
        sg.next(a, 0);
    }
    if (!ok) {
        // a load did not arrive in time: record it, and give the warp's loads
        // in flight (bounded) time to land before its shared memory goes
        if (lane == 0) record_status(a.status, kStatusTimeout);
        for (int s = 0; s < kStages; ++s) mbar_wait(smem_u32(&bars[warp][s]), (phase >> s) & 1u, kWaitLimitNs);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode_gqa = nullptr;

cudaError_t encode_tile_map(CUtensorMap *m, const void *base, int cols, int64_t tok_stride, int64_t blk_stride,
                            int tokens_per_block, int blocks, int box_rows)
{
    if (!g_encode_gqa) {
        cudaDriverEntryPointQueryResult q;
        void *fn = nullptr;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return e != cudaSuccess ? e : cudaErrorNotSupported;
        g_encode_gqa = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(tokens_per_block),
                          static_cast<cuuint64_t>(blocks)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(tok_stride) * 2, static_cast<cuuint64_t>(blk_stride) * 2};
    cuuint32_t box[3] = {64, static_cast<cuuint32_t>(box_rows), 1}, es[3] = {1, 1, 1};
    CUresult r = g_encode_gqa(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, es,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int D, int N>
cudaError_t launch_dn(const GqaLaunch &g, int row_groups, cudaStream_t st)
{
    const CacheView &c = g.cache;
    const bool paged = c.block_table != nullptr;
    const int tpb = paged ? c.page_size : c.capacity;
    const int blocks = paged ? c.num_pages : g.batch * g.groups;
    constexpr int box_rows = kStageBytes / (4 * D);  // a stage's tokens (never across a page)
    static_assert(kPage % box_rows == 0, "a stage lies in one page");
    CUtensorMap mk, mv;
    cudaError_t e;
    if ((e = encode_tile_map(&mk, c.k_rope, D, c.r_tok, c.r_blk, tpb, blocks, box_rows)) != cudaSuccess) return e;
    if ((e = encode_tile_map(&mv, c.c_kv, D, c.c_tok, c.c_blk, tpb, blocks, box_rows)) != cudaSuccess) return e;
    GqaArgs a;
    a.batch = g.batch;
    a.q_len = g.q_len;
    a.groups = g.groups;
    a.hpg = g.hpg;
    a.rows = g.q_len * g.hpg;
    a.max_kv = g.max_kv;
    a.num_splits = g.num_splits;
    a.paged = paged;
    a.bt_stride = c.bt_stride;
    a.num_pages = c.num_pages;
    a.scale_log2 = g.sm_scale * 1.4426950408889634f;
    a.style = g.rope_style;
    a.kv_len = g.kv_len;
    a.block_table = c.block_table;
    a.q = static_cast<const uint16_t *>(g.q);
    a.o_part = g.o_part;
    a.lse_part = g.lse_part;
    a.status = g.status;
    a.turns = rope_turns(D, g.rope_base);
    constexpr size_t smem = 1024 + static_cast<size_t>(kWarps) * kStages * kStageBytes;
    if ((e = allow_smem<gqa_attn_kernel<D, N>>(smem)) != cudaSuccess) return e;
    // the partitions over the SMs' blocks first, then over each block's warps.
    // All row groups' blocks run at a time, one an SM: with a block more than there
    // are SMs (3 groups of 51 on 152) it waits for a whole block to end, 56 rows
    // in 3 groups 19.4 us instead of 13.4.
    const int per_group = g.sms > row_groups ? g.sms / row_groups : 1;
    int grid = g.num_splits < per_group ? g.num_splits : per_group;
    if (g.num_splits > grid * kWarps) grid = (g.num_splits + kWarps - 1) / kWarps;
    return launch_dependent(gqa_attn_kernel<D, N>, dim3(grid, row_groups, 1), dim3(32 * kWarps), smem, st, 1, a, mk,
                            mv);
}

template <int D>
cudaError_t launch_d(const GqaLaunch &g, int row_groups, int n, cudaStream_t st)
{
    switch (n) {
    case 8: return launch_dn<D, 8>(g, row_groups, st);
    case 16: return launch_dn<D, 16>(g, row_groups, st);
    case 24: return launch_dn<D, 24>(g, row_groups, st);
    case 32:
        if constexpr (D == 64) return launch_dn<D, 32>(g, row_groups, st);
        return cudaErrorInvalidConfiguration;
    default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace

int gqa_row_groups(int rows, int head_dim)
{
    // The accumulators (D x N fp32 over 32 lanes) and query fragments have to
    // fit a warp's registers: 32 rows of width 64 take 248, 24 of width 128
    // 255 without spills, 32 of width 128 spill 100 words.
    const int most = head_dim == 64 ? 32 : 24;
    return (rows + most - 1) / most;
}

cudaError_t launch_gqa_attn(const GqaLaunch &g, cudaStream_t st)
{
    if (g.batch <= 0) return cudaSuccess;
    const int rows = g.q_len * g.hpg;
    if (rows > 128) return cudaErrorInvalidConfiguration;
    // Rows a warp: as few as leave all row groups' partitions a warp of the SMs at
    // a time (they read the cache again, from L2).  Few partitions otherwise
    // leave the SMs to a handful of long chains: 28 rows of one sequence of 2000
    // tokens 13.8 us in one group, 8.0 in four of 8 rows; 56 rows of eight of 1000
    // 15.4 in two, 10.3 in seven; 32 rows in 512 partitions 17.7, 14.9 in two of 16.
    const int fewest = gqa_row_groups(rows, g.head_dim);
    int groups = fewest;
    const int forced = tuning().gqa_rows;  // testing aid: most rows a warp
    for (int most = forced > 0 ? forced : 8; most <= 24; most += 8) {
        const int more = (rows + most - 1) / most;
        if (more <= fewest) break;
        if (forced > 0 || g.num_splits <= g.sms / more * kWarps) {
            groups = more;
            break;
        }
    }
    const int n = ((rows + groups - 1) / groups + 7) / 8 * 8;
    if (g.head_dim == 64) return launch_d<64>(g, groups, n, st);
    if (g.head_dim == 128) return launch_d<128>(g, groups, n, st);
    return cudaErrorInvalidConfiguration;
}

}  // namespace gbmla
