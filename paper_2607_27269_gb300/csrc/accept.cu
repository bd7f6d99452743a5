// mla_acceptance_stats: acceptance statistics of a draft against its target at
// the same contexts (Sec. 3.3): the overlap alpha_sample = sum_y min(p_D, p_T)
// of the two softmax distributions (Eq. 9) and greedy agreement of their
// argmaxes (Eq. 10), one vocabulary row per context.
//
// A context's two rows go to one cluster of C CTAs (1 .. 8), which takes two
// passes over them: maxima, sums of exponentials and argmaxes (from HBM, the
// lines marked evict-last), then the overlap (from L2, as far as it holds the
// rows between their passes: 228 rows of 128256 bf16 are 117 MB, and 1.2 times
// the logits come from memory).  Exponentials are base 2 with log2(e) folded into
// one FMA, and pass 2 folds the normaliser into the exponent, p = 2^(x log2 e - c)
// with c = m log2 e + log2 Z, so that min(p_D, p_T) = 2^min(., .) costs one
// exponential per token, not two.
//
// Bound: HBM (both rows once), then issue slots (about 16 per token pair over
// both passes); between the two passes of a row stand reductions and a cluster
// barrier, some 2 us that only other CTAs' work can hide.  So three CTAs of
// 256 threads share an SM, and C is chosen by a model of what that costs.  640
// rows of 128256 bf16: 109.2 us with one CTA of 512 threads per row (304 at a
// time: a third wave of 32 rows, and the lines of 304 rows past the L2's 129
// MB), 78.7 us so; 40 rows of 151936 fp32: 35.4 us with the slices resident in
// shared memory (320 CTAs of 152 KB, three waves), 14.9 us so; 2 rows of 128256
// bf16: 8.9 -> 6.3 us.  The sums and orders are fixed: the bits do not depend on
// timing.
#include <math.h>

#include <atomic>

#include "common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace gbmla {
namespace {

constexpr float kLog2e = 1.4426950408889634f;

struct Stat {
    float m;   // maximum
    float s;   // sum of 2^((x - max(m, kLowest)) log2 e)
    int idx;   // where the maximum is (0x7fffffff: nowhere)
};

// 2^x (the hardware approximation; relative error ~2^-22, and 2^-inf = 0)
__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ---- packed forms for bf16 logits (fewer instructions per token): the
// vector maximum on raw bf16 pairs (exact), the exponent arguments and the
// sums of exponentials as two-wide fp32 FMAs and adds (each lane rounds as
// the scalar instruction does).
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b)
{
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ uint64_t pk(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void upk(uint64_t v, float &lo, float &hi)
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

// both logits of a bf16 pair as a packed fp32 pair (element 2k in the low half)
__device__ __forceinline__ uint64_t bf16x2_f32x2(uint32_t w) { return pk(bf16_lo(w), bf16_hi(w)); }

// Sum of 2^(t_e) over the four packed pairs t[0..3] (a tree of packed adds).
__device__ __forceinline__ float ex2_sum8(const uint64_t (&t)[4])
{
    uint64_t e[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float a, b;
        upk(t[q], a, b);
        e[q] = pk(ex2(a), ex2(b));
    }
    const uint64_t s = add2(add2(e[0], e[1]), add2(e[2], e[3]));
    float lo, hi;
    upk(s, lo, hi);
    return lo + hi;
}

// Sum over eight bf16 token pairs of min(p_D, p_T) = 2^min(x_D log2 e - c_D, x_T log2 e - c_T).
__device__ __forceinline__ float pmin_bf16(const uint4 &vd, const uint4 &vt, float cd, float ct)
{
    const uint64_t L = pk(kLog2e, kLog2e), CD = pk(-cd, -cd), CT = pk(-ct, -ct);
    const uint32_t wd[4] = {vd.x, vd.y, vd.z, vd.w}, wt[4] = {vt.x, vt.y, vt.z, vt.w};
    uint64_t t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float d0, d1, t0, t1;
        upk(fma2(bf16x2_f32x2(wd[q]), L, CD), d0, d1);
        upk(fma2(bf16x2_f32x2(wt[q]), L, CT), t0, t1);
        t[q] = pk(fminf(d0, t0), fminf(d1, t1));
    }
    return ex2_sum8(t);
}

template <typename T>
struct Vec;
template <>
struct Vec<float> {
    static constexpr int n = 4;
    __device__ static float one(const float *p) { return *p; }
};
template <>
struct Vec<uint16_t> {
    static constexpr int n = 8;
    __device__ static float one(const uint16_t *p) { return __uint_as_float(static_cast<uint32_t>(*p) << 16); }
};

// 16 bytes from global memory with an L2 eviction policy.
__device__ __forceinline__ uint4 ld_hint16(const void *p, uint64_t pol)
{
    uint4 w;
    asm volatile("ld.global.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                 : "l"(p), "l"(pol));
    return w;
}

// Reduction over the 32 lanes of a warp by shuffles; every lane gets the result.
template <typename Op>
__device__ __forceinline__ float warp_reduce(float v, Op op)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

constexpr int kRowThreads = 256;
constexpr int kRowCtas = 3;        // per SM
constexpr int kRowUnroll = 2;      // vectors per tensor and thread in a group
constexpr int kGroup = kRowThreads * kRowUnroll;  // vectors per tensor in a group
constexpr int kMaxCluster = 8;
// The lowest base of the exponents: logits below it (-inf, the type's lowest, -1e30
// and the like) are masks and weigh nothing.  A base b has x log2 e + c, c =
// -b log2 e rounded, off by up to |b| 2^-24 at x = b: 2^86 here, which vanishes when
// a real logit raises the base; 2^(1e22) = inf with a base of -1e30, and then NaN.
constexpr float kLowest = -2e9f;
constexpr float kRaise = 16.f;     // a base is raised once a logit passes it by this much

// Running statistics of one thread: the exact maximum and the first vector
// holding it, and sum of 2^((x - base) log2 e) over a base that follows the
// maximum loosely, so that after its first vectors a thread hardly ever
// rescales (fp32 has room for 2^23 times the largest term).
struct Run {
    float m, base, s;
    int at;  // first logit of the first vector whose maximum is m
};

__device__ __forceinline__ float vec_max(const uint4 &v, uint16_t)
{
    const uint32_t w = bmax2(bmax2(v.x, v.y), bmax2(v.z, v.w));
    return fmaxf(bf16_lo(w), bf16_hi(w));
}
__device__ __forceinline__ float vec_max(const uint4 &v, float)
{
    return fmaxf(fmaxf(__uint_as_float(v.x), __uint_as_float(v.y)), fmaxf(__uint_as_float(v.z), __uint_as_float(v.w)));
}

// Sum of 2^(x log2 e + c) over a vector's logits.
__device__ __forceinline__ float vec_exp_sum(const uint4 &v, float c, uint16_t)
{
    const uint64_t L = pk(kLog2e, kLog2e), C = pk(c, c);
    const uint64_t t[4] = {fma2(bf16x2_f32x2(v.x), L, C), fma2(bf16x2_f32x2(v.y), L, C),
                           fma2(bf16x2_f32x2(v.z), L, C), fma2(bf16x2_f32x2(v.w), L, C)};
    return ex2_sum8(t);
}
__device__ __forceinline__ float vec_exp_sum(const uint4 &v, float c, float)
{
    return (ex2(fmaf(__uint_as_float(v.x), kLog2e, c)) + ex2(fmaf(__uint_as_float(v.y), kLog2e, c))) +
           (ex2(fmaf(__uint_as_float(v.z), kLog2e, c)) + ex2(fmaf(__uint_as_float(v.w), kLog2e, c)));
}
__device__ __forceinline__ float vec_pmin(const uint4 &d, const uint4 &t, float cd, float ct, uint16_t)
{
    return pmin_bf16(d, t, cd, ct);
}
__device__ __forceinline__ float vec_pmin(const uint4 &d, const uint4 &t, float cd, float ct, float)
{
    auto p = [&](uint32_t x, uint32_t y) {
        return ex2(fminf(fmaf(__uint_as_float(x), kLog2e, -cd), fmaf(__uint_as_float(y), kLog2e, -ct)));
    };
    return (p(d.x, t.x) + p(d.y, t.y)) + (p(d.z, t.z) + p(d.w, t.w));
}

__device__ __forceinline__ void run_max(Run &r, float vm, int at)
{
    if (vm > r.m) {
        r.m = vm;
        r.at = at;
    }
}
__device__ __forceinline__ void run_base(Run &r)
{
    if (r.m > r.base + kRaise) {
        r.s *= ex2((r.base - r.m) * kLog2e);
        r.base = r.m;
    }
}

// A warp's (exact maximum, sum over base max(m, kLowest), first position) of its lanes' runs.
__device__ __forceinline__ Stat warp_runs(const Run &r)
{
    Stat o;
    o.m = warp_reduce(r.m, [](float a, float b) { return fmaxf(a, b); });
    o.s = warp_reduce(r.s * ex2((r.base - fmaxf(o.m, kLowest)) * kLog2e), [](float a, float b) { return a + b; });
    o.idx = __reduce_min_sync(0xffffffffu, r.m == o.m ? r.at : 0x7fffffff);
    return o;
}
// The same over n statistics in shared memory (n <= 64).
__device__ __forceinline__ Stat warp_stats(const Stat *p, int n)
{
    const int lane = threadIdx.x & 31;
    Run r{-INFINITY, kLowest, 0.f, 0x7fffffff};
    if (lane < n) {
        const Stat a = p[lane];
        r = Run{a.m, fmaxf(a.m, kLowest), a.s, a.idx};
    }
    if (lane + 32 < n) {
        const Stat b = p[lane + 32];
        const float mb = fmaxf(b.m, kLowest), base = fmaxf(r.base, mb);
        r.s = r.s * ex2((r.base - base) * kLog2e) + b.s * ex2((mb - base) * kLog2e);
        r.base = base;
        if (b.m > r.m || (b.m == r.m && b.idx < r.at)) {
            r.m = b.m;
            r.at = b.idx;
        }
    }
    return warp_runs(r);
}

__device__ __forceinline__ uint32_t map_rank(const void *p, int rank)
{
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(p)), "r"(rank));
    return remote;
}

// The two rows of a context go to one cluster of C CTAs (C = 1 .. 8), CTA
// `rank` taking every vector of its contiguous slice; clusters stride over the
// rows.  Pass 1 reads the slices from HBM (lines kept in L2), pass 2 reads
// them again.  One cluster barrier a row: each CTA pushes its statistics into
// every peer's shared memory before it, and the overlap shares of the row
// before (pushed to rank 0) are summed after it, in rank order.  A group's
// loads are issued one group ahead, across the passes and the rows too, so the
// reductions and the barrier wait with loads in flight.  The shared slots
// alternate between two sets: a peer reuses one only after a barrier that
// this CTA arrives at after reading it.
template <typename T>
__global__ void __launch_bounds__(kRowThreads, kRowCtas) accept_row_kernel(int rows, int vocab, int64_t stride,
                                                                const T *__restrict__ draft,
                                                                const T *__restrict__ target, float *alpha,
                                                                int32_t *argmax_d, int32_t *argmax_t,
                                                                int32_t *greedy, int C)
{
    static_assert(kMaxCluster * kRowThreads / 32 <= 64, "a warp merges the cluster's statistics two per lane");
    constexpr int VN = Vec<T>::n, kWarps = kRowThreads / 32, U = kRowUnroll;
    __shared__ Stat s_stat[2][2][kMaxCluster * kWarps];  // [row parity][draft, target][rank, warp]
    __shared__ float s_part[2][kMaxCluster * kWarps];    // rank 0's copy is read
    __shared__ Stat s_final[2];                 // warp 0 of rank 0: the row's statistics until its results are written
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x % C, n_cl = gridDim.x / C;
    const int nvec = vocab / VN;
    const int share = (nvec + C - 1) / C;
    const int v_lo = min(nvec, rank * share), v_hi = min(nvec, v_lo + share);
    const int mine = v_hi - v_lo;  // the slice's vectors
    // pairs of groups (two buffers take turns), or one group alone, which stays in
    // its buffer for pass 2 (1000 bf16 logits: 256 rows 5.3 -> 4.2 us)
    const bool one = mine > 0 && mine <= kGroup;
    const int pairs = one ? 0 : (mine + 2 * kGroup - 1) / (2 * kGroup);
    const int tail = rank == C - 1 ? nvec * VN + tid : vocab;  // the row's last, partial vector: a logit per thread
    const uint64_t keep = tc::policy_evict_last(), drop = tc::policy_evict_first();
    const uint32_t none = sizeof(T) == 2 ? 0xff80ff80u : 0xff800000u;  // -inf
    // Group `it` of this thread's vectors from its first vectors of the two
    // rows on; past the slice's end -inf, which changes no maximum or sum.
    struct Group {
        uint4 d[U], t[U];
    };
    auto load = [&](const uint4 *d, const uint4 *t, int it, uint64_t pol, Group &g) {
        const int first = it * kGroup;
        if (first + kGroup <= mine) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                g.d[u] = ld_hint16(d + first + u * kRowThreads, pol);
                g.t[u] = ld_hint16(t + first + u * kRowThreads, pol);
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                g.d[u] = g.t[u] = make_uint4(none, none, none, none);
                if (first + u * kRowThreads + tid < mine) {
                    g.d[u] = ld_hint16(d + first + u * kRowThreads, pol);
                    g.t[u] = ld_hint16(t + first + u * kRowThreads, pol);
                }
            }
        }
    };
    // warp 0 of rank 0: a row's results from its statistics and the ranks' shares
    auto finish = [&](int64_t row, int par) {
        // the first logit equal to the maximum, in the vector that holds it:
        // lanes 0.. look at the draft's, lanes 16.. at the target's
        const int which = lane >> 4;
        const Stat &f = s_final[which];
        const int y = f.idx + (lane & 15);
        const bool hit = f.idx != 0x7fffffff && (lane & 15) < VN && y < vocab &&
                         Vec<T>::one((which ? target : draft) + row * stride + y) == f.m;
        const unsigned hits = __ballot_sync(0xffffffffu, hit);
        float total = (lane < C * kWarps ? s_part[par][lane] : 0.f) + (lane + 32 < C * kWarps ? s_part[par][lane + 32] : 0.f);
        total = warp_reduce(total, [](float a, float b) { return a + b; });
        if (lane == 0) {
            const int id = (hits & 0xffffu) ? s_final[0].idx + __ffs(hits & 0xffffu) - 1 : s_final[0].idx;
            const int it = (hits >> 16) ? s_final[1].idx + __ffs(hits >> 16) - 1 : s_final[1].idx;
            if (alpha) alpha[row] = total;
            if (argmax_d) argmax_d[row] = id;
            if (argmax_t) argmax_t[row] = it;
            if (greedy) greedy[row] = id == it;
        }
        __syncwarp();
    };
    // a peer's shared memory is written only once all the cluster's CTAs have
    // started: arrive now, wait before the first push
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    griddep_wait();
    griddep_launch_dependents();
    int64_t row = blockIdx.x / C;
    const T *d = draft + row * stride, *t = target + row * stride;
    Group ga, gb;
    auto vec = [&](const T *x) { return reinterpret_cast<const uint4 *>(x) + v_lo + tid; };
    if (mine > 0) load(vec(d), vec(t), 0, keep, ga);
    int par = 0;
    for (;; par ^= 1) {
        // ---- pass 1: maxima, sums, argmaxes
        Run rd{-INFINITY, kLowest, 0.f, 0x7fffffff}, rt = rd;
        auto fold = [&](const Group &g, int it) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int at = v_lo + it * kGroup + u * kRowThreads + tid;
                run_max(rd, vec_max(g.d[u], T{}), at);
                run_max(rt, vec_max(g.t[u], T{}), at);
            }
            run_base(rd);
            run_base(rt);
            const float bd = -rd.base * kLog2e, bt = -rt.base * kLog2e;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                rd.s += vec_exp_sum(g.d[u], bd, T{});
                rt.s += vec_exp_sum(g.t[u], bt, T{});
            }
        };
        const uint4 *vd = vec(d), *vt = vec(t);
        if (one) fold(ga, 0);
#pragma unroll 1
        for (int k = 0; k < pairs; ++k) {
            load(vd, vt, 2 * k + 1, keep, gb);
            fold(ga, 2 * k);
            if (k + 1 < pairs)
                load(vd, vt, 2 * k + 2, keep, ga);
            else
                load(vd, vt, 0, drop, ga);
            fold(gb, 2 * k + 1);
        }
        if (rd.at != 0x7fffffff) rd.at *= VN;  // (a vector's first logit)
        if (rt.at != 0x7fffffff) rt.at *= VN;
        if (tail < vocab) {
            const float xd = Vec<T>::one(d + tail), xt = Vec<T>::one(t + tail);
            run_max(rd, xd, tail);
            run_max(rt, xt, tail);
            run_base(rd);
            run_base(rt);
            rd.s += ex2((xd - rd.base) * kLog2e);
            rt.s += ex2((xt - rt.base) * kLog2e);
        }
        const Stat sd = warp_runs(rd), st = warp_runs(rt);
        if (row < n_cl) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // (the first row only)
        if (lane < 2 * C) {  // lane r: draft to rank r; lane C + r: target to rank r
            const int which = lane / C;
            const Stat v = which ? st : sd;
            const uint32_t to = map_rank(&s_stat[par][which][rank * kWarps + warp], lane - which * C);
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to), "f"(v.m) : "memory");
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to + 4), "f"(v.s) : "memory");
            asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(to + 8), "r"(v.idx) : "memory");
        }
        __syncwarp();
        tc::cluster_sync();
        if (rank == 0 && warp == 0 && row >= n_cl) finish(row - n_cl, par ^ 1);
        // ---- the row's statistics over the ranks: p = 2^(x log2 e - c), c = base log2 e + log2 Z
        float cd, ct;
        {
            const Stat ad = warp_stats(s_stat[par][0], C * kWarps), at = warp_stats(s_stat[par][1], C * kWarps);
            if (rank == 0 && tid == 0) {
                s_final[0] = ad;
                s_final[1] = at;
            }
            cd = fmaxf(ad.m, kLowest) * kLog2e + log2f(ad.s);
            ct = fmaxf(at.m, kLowest) * kLog2e + log2f(at.s);
        }
        // ---- pass 2: sum of min(p_D, p_T), a last read of the lines
        const int64_t next = row + n_cl;
        const T *dn = draft + next * stride, *tn = target + next * stride;
        float acc = 0.f;
        auto overlap = [&](const Group &g) {
#pragma unroll
            for (int u = 0; u < U; ++u) acc += vec_pmin(g.d[u], g.t[u], cd, ct, T{});
        };
        if (one) {
            overlap(ga);
            if (next < rows) load(vec(dn), vec(tn), 0, keep, ga);
        }
#pragma unroll 1
        for (int k = 0; k < pairs; ++k) {
            load(vd, vt, 2 * k + 1, drop, gb);
            overlap(ga);
            if (k + 1 < pairs)
                load(vd, vt, 2 * k + 2, drop, ga);
            else if (next < rows)
                load(vec(dn), vec(tn), 0, keep, ga);
            overlap(gb);
        }
        if (tail < vocab)
            acc += ex2(fminf(fmaf(Vec<T>::one(d + tail), kLog2e, -cd), fmaf(Vec<T>::one(t + tail), kLog2e, -ct)));
        acc = warp_reduce(acc, [](float a, float b) { return a + b; });
        if (lane == 0)
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(map_rank(&s_part[par][rank * kWarps + warp], 0)), "f"(acc)
                         : "memory");
        __syncwarp();
        if (next >= rows) break;
        row = next;
        d = dn;
        t = tn;
    }
    tc::cluster_sync();
    if (rank == 0 && warp == 0) finish(row, par);
}

// Clusters of C CTAs of the row kernel that the device runs at a time (a
// property of the device; 0 if it cannot say), looked up once per device.
template <typename T>
int row_clusters(int C)
{
    constexpr int kMaxDevices = 64;
    static std::atomic<int> known[kMaxDevices][kMaxCluster + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
    int n = known[dev][C].load(std::memory_order_relaxed);
    if (n == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(kRowThreads);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, accept_row_kernel<T>, &cfg) != cudaSuccess) return 0;
        known[dev][C].store(n, std::memory_order_relaxed);
    }
    return n;
}

template <typename T>
cudaError_t launch_typed(int rows, int vocab, const void *draft, const void *target, int64_t stride, float *alpha,
                        int32_t *argmax_d, int32_t *argmax_t, int32_t *greedy, cudaStream_t st)
{
    // The cluster size with the least time by a model fitted to 950 measurements
    // (2 to 1200 rows of 1000 to 262144 logits, both types, from L2 and from
    // memory) of each of the eight sizes; its choice takes 1 % longer than the best
    // of them on average, 25 % at most.  A wave of rows costs its latency (more in
    // clusters, and with more CTAs an SM), the pairs of groups a CTA folds (mostly
    // whole ones: padding costs like logits), and what its rows, past the L2's
    // size, take to come from memory twice.  Of clusters of 3 and 5 a few less run
    // at a time than the device says (142 of 148, 82 of 87); those left over would
    // begin when the others have ended.  (A model of bytes alone took 7 CTAs a row
    // for 480 rows of 32000 bf16, 34 us against 20 with one, and two for 640 rows of
    // 128256 fp32, 164 us against 135 with six.)
    const bool f32 = sizeof(T) == 4;
    const double group = f32 ? 0.685 : 1.14, shared = f32 ? 0.016 : 0.282;  // a pair; a pair times the CTAs on the SM
    const int sms = row_clusters<T>(1) / kRowCtas > 0 ? row_clusters<T>(1) / kRowCtas : 1;
    double best = 0;
    int C = 0, n_cl = 0;
    const int forced = tuning().accept_cluster;  // testing aid: 1 .. 8 CTAs a cluster
    for (int c = 1; c <= kMaxCluster; ++c) {
        if (forced >= 1 && forced <= kMaxCluster && c != forced) continue;
        int n = row_clusters<T>(c);
        if (n <= 0) continue;
        if (c == 3 || c == 5) n -= n / 16;
        const int nvec = vocab / Vec<T>::n, share = (nvec + c - 1) / c;
        const double pairs = 0.91 * ((share + 2 * kGroup - 1) / (2 * kGroup)) + 0.09 * nvec / (2.0 * kGroup * c);
        auto wave = [&](int live) {
            const double load = static_cast<double>(live) * c / sms, mb = 2e-6 * live * vocab * sizeof(T);
            const double most = load > 2 ? 3 : load > 1 ? 2 : 1;  // CTAs on an SM
            return (c == 1 ? 0.234 : 0.925) + (load > 1 ? 0.368 + 0.868 * (load < 2 ? load - 1 : 1) : 0) +
                   pairs * (group > most * shared ? group : most * shared) + 0.108 * mb * (mb < 313 ? mb / 313 : 1);
        };
        const double us = rows / n * wave(n) + (rows % n ? wave(rows % n) : 0);
        if (C == 0 || us < best) {
            best = us;
            C = c;
            n_cl = rows < n ? rows : n;
        }
    }
    if (C == 0) return cudaErrorInvalidConfiguration;
    return launch_dependent(accept_row_kernel<T>, dim3(n_cl * C), dim3(kRowThreads), 0, st, C, rows, vocab, stride,
                            static_cast<const T *>(draft), static_cast<const T *>(target), alpha, argmax_d, argmax_t,
                            greedy, C);
}

}  // namespace

cudaError_t launch_acceptance(int rows, int vocab, int dtype, const void *draft, const void *target, int64_t stride,
                              float *alpha, int32_t *argmax_d, int32_t *argmax_t, int32_t *greedy, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    if (dtype == 0)
        return launch_typed<float>(rows, vocab, draft, target, stride, alpha, argmax_d, argmax_t, greedy, st);
    return launch_typed<uint16_t>(rows, vocab, draft, target, stride, alpha, argmax_d, argmax_t, greedy, st);
}

}  // namespace gbmla
