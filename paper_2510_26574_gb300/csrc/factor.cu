// rpchol_factor: pivoted partial Cholesky of the implicit Gaussian kernel
// matrix (Section 1.2; Appendix A, Algorithms 2 and 3), FP64 path.
//
// One round of Algorithm 2 is five stream-ordered launches; the current rank
// k and the accepted count m live on the device, so no round needs a host
// synchronisation:
//   k_propose  commit the previous round (k += m); greedy: argmax of rho from
//              per-tile (max, index); ARPC: prefix of per-tile sums of rho and
//              b inverse-CDF draws with Philox uniforms (stream 0).
//   k_gather   X(S',:) and F(S',:) of the proposals into contiguous panels.
//   k_blockH   H = K(S',S') - F(S',:) F(S',:)^T  (b x b).
//   k_reject   Algorithm 3 (sequential accept test with Philox z, stream 1,
//              rank-1 Schur updates), the accepted positions and L = chol(H(T,T)).
//   k_engine   kernel-column engine: for a 64-row tile, K(:,S) from the
//              norm expansion exp(-(|x_i|^2 + |x_s|^2 - 2 x_i.x_s)/eps), minus
//              F F(S,:)^T, times L^-T by forward substitution, written to
//              F(:, k:k+m); fused residual update rho -= rownorms(G)^2, clamp at
//              0, and the per-tile sum and (max, index) of rho for the next round.
#include <algorithm>
#include <climits>
#include <vector>

#include "common.cuh"
#include "factor.cuh"
#include "kexp.cuh"
#include "oz_digits.cuh"
#include "ozgemm.cuh"
#include "rej_root.cuh"
#include "trace.cuh"

namespace kevd {

constexpr int kPropChunks = 1024;   // chunks of the tile sums in a proposal step

static int tc_bn(int b) { return b <= 32 ? 32 : b <= 64 ? 64 : 128; }

// oz: the FP64 path with the engine on the tensor cores (ozmm.cu): the two
// N x b product arrays and the digit planes (OzWs) are carved after the rest;
// rounds_max bounds the padding of F's planes (16 columns per round).
static FactorWs carve_factor(void* base, int64_t N, int d, int r, int b, size_t* bytes, bool tc = false,
                             PanelWs* pw = nullptr, bool oz = false, OzWs* ow = nullptr, int rounds_max = 0,
                             bool pl = false) {
    Carver c(base);
    const int64_t nt = (N + kBM - 1) / kBM;
    FactorWs w{};
    w.st = c.take<FactorState>(1);
    w.xn = c.take<double>(N);
    w.tile_sum = c.take<double>(nt);
    w.tile_max = c.take<double>(nt);
    w.tile_idx = c.take<int64_t>(nt);
    w.pre = c.take<double>(kPropChunks + 32);
    w.prop = c.take<int64_t>(b);
    w.acc_pos = c.take<int32_t>(b);
    w.tpos = c.take<int32_t>(b);
    w.XSP = c.take<double>((size_t)d * b);
    w.FSP = c.take<double>((size_t)r * b);
    w.xnS = c.take<double>(b);
    w.H = c.take<double>((size_t)b * b);
    w.Lfull = c.take<double>((size_t)b * b);
    w.Lc = c.take<double>((size_t)b * b);
    if (tc) {
        const int BN = tc_bn(b);
        PanelWs p{};
        p.panel = c.take<uint16_t>((size_t)tc_chunks(d, r) * 2 * BN * kTcBK);
        p.Lf = c.take<float>((size_t)BN * BN);
        p.nS = c.take<float>(BN);
        p.pidx = c.take<int64_t>(BN);
        p.err = c.take<int>(4);
        if (pl) p.planes = c.take<uint16_t>(tc_plane_bytes(N, d, r, &p.nxh, &p.nH) / 2);
        if (pw) *pw = p;
    }
    if (oz && !tc) {
        OzWs o;
        w.ldD = (N + 1) / 2 * 2;
        o.ldX = (d + 15) / 16 * 16;
        const int64_t ldF = ((int64_t)r + 15 * (int64_t)std::max(rounds_max, 1) + 15) / 16 * 16;
        o.ldF = (int)std::min(ldF, (int64_t)std::max(rounds_max, 1) * ((b + 15) / 16 * 16));
        o.ldR = (b + 15) / 16 * 16;
        o.ldLi = (b + 1) / 2 * 2;
        // The size is that of every array by itself with rows as they are and r + 15 rounds
        // columns of F; the planes' rows are padded to 128, which two things make room for: F's
        // columns are also at most a padded block per round, and arrays that are never alive together
        // share memory (the pivot panels, read before R is written, lie in R's planes, L^-1, formed
        // after Dx is read, in Dx).  Small N, where they do not fit, take more.
        Carver exact(nullptr);
        exact.off = c.off;
        for (int u = 0; u < 2; ++u) exact.take<double>((size_t)w.ldD * b);
        for (const int64_t n : {(int64_t)N, (int64_t)b})
            for (const int64_t ld : {(int64_t)o.ldX, ldF, (int64_t)o.ldR}) exact.take<uint16_t>((size_t)kDigits * n * ld);
        for (const int64_t n : {(int64_t)N, (int64_t)N, (int64_t)b, (int64_t)b}) exact.take<int>(n);
        exact.take<double>((size_t)b * o.ldLi);
        exact.take<int>(4);
        const size_t px = oz_tile_elems(b, o.ldX / 16, kDigits), pf = oz_tile_elems(b, o.ldF / 16, kDigits);
        const size_t lp = oz_tile_elems(b, o.ldR / 16, kDigits);
        w.Dx = c.take<double>(std::max((size_t)w.ldD * b, lp / 4 + (size_t)b * o.ldLi));
        w.Df = c.take<double>((size_t)w.ldD * b);
        o.Lp = reinterpret_cast<uint16_t*>(w.Dx);
        o.Linv = reinterpret_cast<double*>(o.Lp + lp);
        o.Xp = c.take<uint16_t>(oz_tile_elems(N, o.ldX / 16, kDigits));
        o.xe = c.take<int>(N);
        o.Fp = c.take<uint16_t>(oz_tile_elems(N, o.ldF / 16, kDigits));
        o.Rp = c.take<uint16_t>(std::max(oz_tile_elems(N, o.ldR / 16, kDigits), px + pf));
        o.PXp = o.Rp;
        o.PFp = o.Rp + px;
        o.re = c.take<int>(N);
        o.pxe = c.take<int>(b);
        o.le = c.take<int>(b);
        o.flags = c.take<int>(4);
        c.off = std::max(c.off, exact.off);
        if (ow) *ow = o;
    }
    *bytes = c.off;
    return w;
}

// ---------------------------------------------------------------------------
// a1: squared norms, rho := diag K = 1, initial tile statistics.
// ---------------------------------------------------------------------------
template <typename TX>
__device__ __forceinline__ void prepare_body(const TX* __restrict__ X, int64_t N, int d, FactorWs w,
                                             double* __restrict__ rho, int64_t blk) {
    const int64_t i = blk * blockDim.x + threadIdx.x;
    if (blk == 0 && threadIdx.x == 0) {
        FactorState s = {};
        *w.st = s;
    }
    if (i < N) {
        const TX* x = X + i * d;
        double s = 0.0;
        for (int c = 0; c < d; ++c) s = fma((double)x[c], (double)x[c], s);
        w.xn[i] = s;
        rho[i] = 1.0;
        if (!isfinite(s)) w.st->bad = 1;   // benign race: every writer stores 1
        if ((i % kBM) == 0) {
            const int64_t t = i / kBM;
            const int64_t cnt = min((int64_t)kBM, N - i);
            w.tile_sum[t] = (double)cnt;
            w.tile_max[t] = 1.0;
            w.tile_idx[t] = i;
        }
    }
}

template <typename TX>
__global__ void k_prepare(const TX* __restrict__ X, int64_t N, int d, FactorWs w, double* __restrict__ rho) {
    prepare_body(X, N, d, w, rho, blockIdx.x);
}

// Warp-inclusive scan (Hillis-Steele over shuffles).
__device__ __forceinline__ double warp_incl_scan(double v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        double y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// All threads of the cluster; what they wrote to global memory before is visible after.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// a2: pivot proposal.
// ---------------------------------------------------------------------------

// Commits the previous round (one thread).
__device__ __forceinline__ void commit_round(FactorState* st) {
    if (st->m > 0) {
        st->sum_k += st->k;
        st->eng_rounds += 1;
    }
    st->k += st->m;
    st->kp += (st->m + 15) & ~15;
    st->sum_m_sq += (long long)st->m * st->m;
    st->m = 0;
}

// Greedy: the argmax of rho from the tile (max, index) pairs.  One block of 1024 threads.
__global__ void __launch_bounds__(1024) k_propose_greedy(FactorWs w, int64_t ntiles, int r, int rnd,
                                                         int64_t* __restrict__ proposals_out) {
    __shared__ double sh[32];
    __shared__ int64_t shi[32];
    __shared__ int s_go;
    FactorState* st = w.st;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    if (tid == 0) {
        commit_round(st);
        if (st->k >= r) st->done = 1;
        s_go = !st->done;
    }
    __syncthreads();
    if (!s_go) return;
    double v = -1.0;
    int64_t idx = LLONG_MAX;
    for (int64_t t = tid; t < ntiles; t += blockDim.x) argmax_merge(v, idx, w.tile_max[t], w.tile_idx[t]);
    warp_argmax(v, idx);
    if (lane == 0) {
        sh[wid] = v;
        shi[wid] = idx;
    }
    __syncthreads();
    if (wid == 0) {
        v = lane < nw ? sh[lane] : -1.0;
        idx = lane < nw ? shi[lane] : LLONG_MAX;
        warp_argmax(v, idx);
        if (lane == 0) {
            if (!(v > 0.0)) {
                st->done = 1;
            } else {
                w.prop[0] = idx;
                st->total = v;
                st->rounds += 1;
                if (proposals_out) proposals_out[rnd] = idx;
            }
        }
    }
}

// ARPC: b inverse-CDF draws from rho.  The tile sums are cut into 1,024 chunks, one thread
// each, whose offsets are found by a scan; a draw then looks for its chunk among the
// offsets (two loads per lane), its tile in the chunk and its row in the tile, 32 at a time.
// An FP64 operation takes a quarter of an SM's pipe for 17 cycles, so the chunks and the
// draws are spread over a cluster of 8 CTAs, with a warp per draw at b = 128: per round
// 16 / 11 us at N = 2,000,000 / 524,288 (one CTA, prefixes of all tiles written and
// searched: 96 / 59 us).
constexpr int kPropCluster = 8;
constexpr int kPropThreads = 512;

__device__ __forceinline__ void propose_body(FactorWs w, const double* __restrict__ rho, int64_t N, int64_t ntiles,
                                             int b, int r, uint64_t seed, int rnd, int64_t* __restrict__ proposals_out,
                                             double floor_sum, int cta) {
    constexpr unsigned kAll = 0xffffffffu;
    FactorState* st = w.st;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool go = !st->done && st->k + st->m < r;           // the same in every CTA
    const int64_t chunk = (ntiles + kPropChunks - 1) / kPropChunks;
    constexpr int kPer = kPropChunks / kPropCluster;
    double loc = 0.0, inc = 0.0;
    if (go && tid < kPer) {
        const int64_t t0 = min((int64_t)(cta * kPer + tid) * chunk, ntiles), t1 = min(t0 + chunk, ntiles);
#pragma unroll 8
        for (int64_t t = t0; t < t1; ++t) loc += w.tile_sum[t];
        inc = warp_incl_scan(loc);
        if (lane == 31) w.pre[kPropChunks + cta * (kPer / 32) + wid] = inc;
    }
    cluster_sync();                                           // every CTA has read the state
    if (cta == 0 && tid == 0) {
        commit_round(st);
        if (!go) st->done = 1;
    }
    if (!go) return;
    const double wv = __ldcg(w.pre + kPropChunks + lane);
    const double wi = warp_incl_scan(wv);
    const double S = __shfl_sync(kAll, wi, 31);
    if (tid < kPer) w.pre[cta * kPer + tid] = __shfl_sync(kAll, wi - wv, cta * (kPer / 32) + wid) + inc - loc;
    if (!(S > floor_sum)) {   // sum(rho) = 0, or at the caller's floor tol * N
        if (cta == 0 && tid == 0) st->done = 1;
        return;
    }
    if (cta == 0 && tid == 0) {
        st->total = S;
        st->rounds += 1;
    }
    cluster_sync();
    for (int j = cta + kPropCluster * wid; j < b; j += kPropCluster * (kPropThreads / 32)) {
        const double u = philox_uniform(seed, 0u, (uint32_t)rnd, (uint32_t)j);
        const double target = u * S;
        // the first chunk that ends above target
        int64_t t = -1;
        double acc = 0.0;
        unsigned hit = __ballot_sync(kAll, (lane < 31 ? __ldcg(w.pre + 32 * lane + 32) : S) > target);
        int i = kPropChunks - 1;
        if (hit) {
            i = 32 * (__ffs(hit) - 1);
            const int e = i + lane + 1;
            hit = __ballot_sync(kAll, (e < kPropChunks ? __ldcg(w.pre + e) : S) > target);
            i += __ffs(hit) - 1;
            acc = __ldcg(w.pre + i);
            // the first tile with mass in it that ends above target
            const int64_t t1 = min((i + 1) * chunk, ntiles);
            for (int64_t c0 = i * chunk; c0 < t1; c0 += 32) {
                const double v = c0 + lane < t1 ? w.tile_sum[c0 + lane] : 0.0;
                const double sv = warp_incl_scan(v);
                hit = __ballot_sync(kAll, v > 0.0 && acc + sv > target);
                if (hit) {
                    const int f = __ffs(hit) - 1;
                    const double before = __shfl_sync(kAll, sv, max(f - 1, 0));
                    if (f > 0) acc += before;
                    t = c0 + f;
                    break;
                }
                acc += __shfl_sync(kAll, sv, 31);
            }
        }
        if (t < 0) {   // u*S rounded to >= S, or a chunk's sum to below its end: the last tile with mass up to there
            t = min((i + 1) * chunk, ntiles) - 1;
            while (t > 0 && !(w.tile_sum[t] > 0.0)) --t;
            while (t < ntiles - 1 && !(w.tile_sum[t] > 0.0)) ++t;
            acc = -INFINITY;
        }
        const int64_t base = t * kBM;
        const int cnt = (int)min((int64_t)kBM, N - base);
        int64_t found = -1, last_pos = -1;
        for (int c0 = 0; c0 < cnt; c0 += 32) {
            const int rr = c0 + lane;
            const double v = rr < cnt ? rho[base + rr] : 0.0;
            const double sv = warp_incl_scan(v);
            const unsigned pos = __ballot_sync(kAll, rr < cnt && v > 0.0);
            if (pos) last_pos = base + c0 + 31 - __clz(pos);
            hit = __ballot_sync(kAll, rr < cnt && v > 0.0 && acc + sv > target);
            if (hit) {
                found = base + c0 + __ffs(hit) - 1;
                break;
            }
            acc += __shfl_sync(kAll, sv, 31);
        }
        if (found < 0) found = last_pos;   // rounding at the tile's upper edge
        if (found < 0) found = base;       // unreachable: the tile has mass
        if (lane == 0) {
            w.prop[j] = found;
            if (proposals_out) proposals_out[(int64_t)rnd * b + j] = found;
        }
    }
}

__global__ void __cluster_dims__(kPropCluster, 1, 1) __launch_bounds__(kPropThreads)
    k_propose(FactorWs w, const double* __restrict__ rho, int64_t N, int64_t ntiles, int b, int r, uint64_t seed,
              int rnd, int64_t* __restrict__ proposals_out, double floor_sum) {
    propose_body(w, rho, N, ntiles, b, r, seed, rnd, proposals_out, floor_sum, blockIdx.x);
}

// ---------------------------------------------------------------------------
// a3 (part 1): gather X(S',:) and F(S',:)[:, :k] into d x b and k x b panels.
// ---------------------------------------------------------------------------
template <typename TX, typename TF>
__device__ __forceinline__ void gather_body(FactorWs w, const TX* __restrict__ X, const TF* __restrict__ F,
                                            int64_t ldf, int d, int b, int blk) {
    const FactorState* st = w.st;
    if (st->done) return;
    const int k = st->k;
    const int lane = threadIdx.x & 31;
    const int c = blk * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (blk == 0 && threadIdx.x < b) w.xnS[threadIdx.x] = w.xn[w.prop[threadIdx.x]];
    if (c < d) {
        for (int j = lane; j < b; j += 32) w.XSP[(size_t)c * b + j] = (double)X[w.prop[j] * d + c];
    } else if (c - d < k) {
        const int cf = c - d;
        for (int j = lane; j < b; j += 32) w.FSP[(size_t)cf * b + j] = (double)F[w.prop[j] + (int64_t)cf * ldf];
    }
}

template <typename TX, typename TF>
__global__ void k_gather(FactorWs w, const TX* __restrict__ X, const TF* __restrict__ F, int64_t ldf, int d, int b) {
    gather_body(w, X, F, ldf, d, b, blockIdx.x);
}

// ---------------------------------------------------------------------------
// a3 (part 2): H = K(S',S') - F(S',:) F(S',:)^T.  Lower-triangle tiles of 4 x 4
// entries, a block each: a thread owns one entry and the terms c = g mod 8 of its sums (g the
// thread's group), in four accumulators by c mod 32, which a fixed tree adds.  Both
// halves of H come from one thread (the same value for (j, l) and (l, j)), so H is exactly
// symmetric.  Bound: the FP64 pipe (17 cycles per warp operation and SM) over b^2 / 2
// entries; 4 x 4 tiles leave 3 or 4 to each SM at b = 128.  Measured per round, b = 128, mean
// k of 900: 21 us (one warp per entry of both halves with strided loads and a shuffle
// tree per entry: 122 us; b = 64, mean k of 400: 12, was 28).
// ---------------------------------------------------------------------------
constexpr int kBlockHThreads = 128;   // 16 entries x 8 groups of terms

// Terms c = g, g + 8, g + 16, ... of P(:,j) . P(:,l), P n x b row-major; partial sums per
// c mod 32, added as a butterfly over 32 lanes adds them (16 first, then 8).
__device__ __forceinline__ double pair_terms(const double* __restrict__ P, int b, int n, int j, int l, int g) {
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int c0 = g;
#pragma unroll 2
    for (; c0 + 24 < n; c0 += 32) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double* row = P + (size_t)(c0 + 8 * i) * b;
            a[i] = fma(row[j], row[l], a[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (c0 + 8 * i < n) {
            const double* row = P + (size_t)(c0 + 8 * i) * b;
            a[i] = fma(row[j], row[l], a[i]);
        }
    return (a[0] + a[2]) + (a[1] + a[3]);
}

static int blockH_blocks(int b) { return ((b + 3) / 4) * ((b + 3) / 4 + 1) / 2; }

__device__ __forceinline__ void blockH_body(FactorWs w, int d, int b, double inv_eps, int blk) {
    __shared__ double part[2][8][16];
    const FactorState* st = w.st;
    const int nt = (b + 3) / 4;
    if (st->done || blk >= nt * (nt + 1) / 2) return;
    int J = (int)((sqrtf(8.f * blk + 1.f) - 1.f) * 0.5f);
    while (J * (J + 1) / 2 > blk) --J;
    while ((J + 1) * (J + 2) / 2 <= blk) ++J;
    const int p = threadIdx.x & 15, g = threadIdx.x >> 4;
    const int j = 4 * J + (p >> 2), l = 4 * (blk - J * (J + 1) / 2) + (p & 3);
    const int jc = min(j, b - 1), lc = min(l, b - 1);
    part[0][g][p] = pair_terms(w.XSP, b, d, jc, lc, g);
    part[1][g][p] = pair_terms(w.FSP, b, st->k, jc, lc, g);
    __syncthreads();
    if (threadIdx.x >= 16 || j >= b || l > j) return;
    double sum[2];
#pragma unroll
    for (int q = 0; q < 2; ++q)
        sum[q] = ((part[q][0][p] + part[q][4][p]) + (part[q][2][p] + part[q][6][p])) +
                 ((part[q][1][p] + part[q][5][p]) + (part[q][3][p] + part[q][7][p]));
    double kv;
    if (w.prop[j] == w.prop[l]) {
        kv = 1.0;   // k(x, x) = exp(0)
    } else {
        const double d2 = fmax(w.xnS[j] + w.xnS[l] - 2.0 * sum[0], 0.0);
        kv = exp(-d2 * inv_eps);
    }
    w.H[(size_t)j * b + l] = w.H[(size_t)l * b + j] = kv - sum[1];
}

__global__ void __launch_bounds__(kBlockHThreads) k_blockH(FactorWs w, int d, int b, double inv_eps) {
    blockH_body(w, d, b, inv_eps, blockIdx.x);
}

// ---------------------------------------------------------------------------
// a4: Algorithm 3 (ARPC) or the greedy acceptance (b = 1, accept iff H > 0).
//
// Algorithm 3 is a chain of b steps (accept H(i,i), scale a column by 1 / sqrt(H(i,i)),
// subtract its outer product), and one dependent FP64 operation takes 64 cycles and
// occupies a quarter of an SM's FP64 pipe for as long.  So the steps run in panels of 16
// columns on four warps, one matrix row per thread: every warp carries the panel's
// diagonal in its lanes and takes the decision itself (one barrier per accepted
// proposal, none per rejected one), the square root and the division share one
// reciprocal root (11 operations instead of ~20), and the columns right of the panel are
// updated 16 pivots at a time by all CTAs of a cluster, with H in global memory.  Every
// entry sees the same subtractions in the same order as with one step at a time.
// Measured per round at b = 128 / 64: 205 / 82 us (one CTA with two barriers and the whole
// square per step: 556 / 190 us).
// ---------------------------------------------------------------------------
constexpr int kRejW = 16;         // panel columns
constexpr int kRejThreads = 256;
constexpr int kRejCluster = 8;    // CTAs per problem

struct RejShared {
    double L[kRejW][128];         // panel columns: L(c0 + t, c0 + j)
    double zr[128];               // z_i rho0_i
    int tpos[128];
    int m;
};

// One cluster of kRejCluster CTAs per problem, `cta` the rank in it.  H is overwritten.
__device__ __forceinline__ void arpc_reject_body(FactorWs w, int b, int r, uint64_t seed, int rnd,
                                                 int64_t* __restrict__ pivots, RejShared& sh, int cta) {
    FactorState* st = w.st;
    if (st->done) return;                                        // the same in every CTA
    const int k = st->k;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (cta == 0) {
        for (int e = tid; e < b; e += blockDim.x)
            sh.zr[e] = philox_uniform(seed, 1u, (uint32_t)rnd, (uint32_t)e) * w.H[(size_t)e * b + e];
        __syncthreads();
    }
    int m = 0;
    for (int c0 = 0; c0 < b; c0 += kRejW) {
        const int nw = min(kRejW, b - c0);
        unsigned mask = 0;                                       // accepted columns of the panel
        if (cta == 0 && wid < 4) {
            const int l = c0 + tid;                              // this thread's row
            const bool row = tid < b - c0;
            double c[kRejW];
#pragma unroll
            for (int j = 0; j < kRejW; ++j)
                c[j] = row && j < nw && l >= c0 + j ? __ldcg(w.H + (size_t)l * b + c0 + j) : 0.0;
            double d = lane < nw ? __ldcg(w.H + (size_t)(c0 + lane) * (b + 1)) : 0.0;
            const double zr = lane < nw ? sh.zr[c0 + lane] : 0.0;
#pragma unroll
            for (int j = 0; j < kRejW; ++j) {
                if (j >= nw) break;
                const double h = __shfl_sync(0xffffffffu, d, j);
                if (!(h > 0.0 && __shfl_sync(0xffffffffu, zr, j) < h) || k + m >= r) continue;
                double s, y, v;
                if (h > 0x1p-900) {
                    rej_root(h, s, y);
                    v = rej_quot(c[j], s, y);
                } else {
                    s = sqrt(h);
                    v = c[j] / s;
                }
                sh.L[j][tid] = v;
                asm volatile("bar.sync 1, 128;" ::: "memory");
                const double lj = sh.L[j][lane & (kRejW - 1)];
                if (lane > j) d = fma(-lj, lj, d);
#pragma unroll
                for (int j2 = j + 1; j2 < kRejW; ++j2) c[j2] = fma(-v, sh.L[j][j2], c[j2]);
                if (row && l >= c0 + j) w.Lfull[(size_t)l * b + c0 + j] = v;
                if (tid == 0) sh.tpos[m] = c0 + j;
                mask |= 1u << j;
                ++m;
            }
            if (tid == 0) {
                sh.m = m;
                w.tpos[b - 1] = (int)mask;                       // (free until the end: positions are in sh.tpos)
            }
        }
        const int n0 = c0 + kRejW;
        cluster_sync();
        if (n0 >= b) break;
        // columns n0 .. of the rows below the panel, all CTAs: a warp takes a row
        mask = (unsigned)*(volatile int*)&w.tpos[b - 1];
        m = cta == 0 ? sh.m : 0;
        const int cnt = __popc(mask);
        for (int e = tid; e < cnt * (b - n0); e += blockDim.x) {   // the accepted columns into shared memory, packed
            const int a = e / (b - n0), l = e % (b - n0);
            unsigned t = mask;
            for (int q = 0; q < a; ++q) t &= t - 1;
            sh.L[a][l] = __ldcg(w.Lfull + (size_t)(n0 + l) * b + c0 + __ffs(t) - 1);
        }
        __syncthreads();
        for (int l = cta * (kRejThreads / 32) + wid; l < b - n0; l += kRejCluster * (kRejThreads / 32)) {
            double* Hr = w.H + (size_t)(n0 + l) * b + n0;
            double x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = lane + 32 * u <= l ? __ldcg(Hr + lane + 32 * u) : 0.0;
            for (int a = 0; a < cnt; ++a) {
                const double v = sh.L[a][l];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (32 * u <= l) x[u] = fma(-v, sh.L[a][(lane + 32 * u) & 127], x[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (lane + 32 * u <= l) Hr[lane + 32 * u] = x[u];
        }
        cluster_sync();
    }
    if (cta != 0) return;
    // (CTA 0's own columns of Lfull and its list of positions: ordered by the last barrier)
    m = sh.m;
    for (int e = tid; e < m * m; e += blockDim.x) {
        const int a = e / m, a2 = e % m;
        w.Lc[(size_t)a * b + a2] = a2 <= a ? w.Lfull[(size_t)sh.tpos[a] * b + sh.tpos[a2]] : 0.0;
    }
    for (int a = tid; a < m; a += blockDim.x) {
        w.acc_pos[a] = sh.tpos[a];
        pivots[k + a] = w.prop[sh.tpos[a]];
    }
    if (tid == 0) st->m = m;
}

// Greedy (b = 1): accept iff H > 0, L = sqrt(H).
__device__ __forceinline__ void greedy_reject_body(FactorWs w, int r, int64_t* __restrict__ pivots) {
    FactorState* st = w.st;
    if (st->done || threadIdx.x != 0) return;
    const int k = st->k;
    const double h = w.H[0];
    const int m = h > 0.0 && k < r ? 1 : 0;
    if (m) {
        w.Lc[0] = sqrt(h);
        w.acc_pos[0] = 0;
        pivots[k] = w.prop[0];
    } else {
        st->done = 1;                                            // greedy stops once H <= 0
    }
    st->m = m;
}

__global__ void __cluster_dims__(kRejCluster, 1, 1) __launch_bounds__(kRejThreads)
    k_reject(FactorWs w, int b, int r, uint64_t seed, int rnd, int64_t* __restrict__ pivots) {
    __shared__ RejShared sh;
    arpc_reject_body(w, b, r, seed, rnd, pivots, sh, blockIdx.x);
}

__global__ void k_reject_greedy(FactorWs w, int r, int64_t* __restrict__ pivots) { greedy_reject_body(w, r, pivots); }

// ---------------------------------------------------------------------------
// a5 + a6: the kernel-column engine (FP64).  Tile = 64 rows x BN = 8*TN columns.
// Warp w owns columns [w*TN, w*TN+TN); lane owns rows 2*lane, 2*lane+1.
// Warps whose columns are all >= m skip the products.
// ---------------------------------------------------------------------------
template <int TN>
__device__ __forceinline__ void engine_body(FactorWs w, const double* __restrict__ X, double* __restrict__ F,
                                            int64_t ldf, double* __restrict__ rho, int64_t N, int d, int b,
                                            double inv_eps, int64_t tile, double* smem) {
    constexpr int BN = 8 * TN;
    constexpr int APAD = kBM + 2;
    double* As = smem;                 // kBK x APAD
    double* Bs = As + kBK * APAD;      // kBK x BN
    double* Rs = smem;                 // kBM x (BN+1), reused after the products
    __shared__ double red[32];
    __shared__ int64_t redi[32];

    const FactorState* st = w.st;
    if (st->done) return;
    const int m = st->m;
    if (m == 0) return;
    const int k = st->k;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int64_t row0 = tile * kBM;
    const bool active = wid * TN < m;

    double acc[2][TN];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int c = 0; c < TN; ++c) acc[a][c] = 0.0;

    // ---- X(i,:) . X(s,:) over d ----
    for (int c0 = 0; c0 < d; c0 += kBK) {
#pragma unroll
        for (int p = 0; p < (kBM * kBK) / 256; ++p) {
            const int e = tid + 256 * p, i = e / kBK, kk = e % kBK;
            const int64_t row = row0 + i;
            As[kk * APAD + i] = (row < N && c0 + kk < d) ? X[row * d + c0 + kk] : 0.0;
        }
        for (int e = tid; e < kBK * BN; e += 256) {
            const int kk = e / BN, l = e % BN;
            Bs[kk * BN + l] = (l < m && c0 + kk < d) ? w.XSP[(size_t)(c0 + kk) * b + w.acc_pos[l]] : 0.0;
        }
        __syncthreads();
        if (active) {
#pragma unroll
            for (int kk = 0; kk < kBK; ++kk) {
                const double2 a = *reinterpret_cast<const double2*>(&As[kk * APAD + 2 * lane]);
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const double bv = Bs[kk * BN + wid * TN + c];
                    acc[0][c] = fma(a.x, bv, acc[0][c]);
                    acc[1][c] = fma(a.y, bv, acc[1][c]);
                }
            }
        }
        __syncthreads();
    }
    // ---- kernel values: exp(-(|x_i|^2 + |x_s|^2 - 2 x_i.x_s) / eps) ----
    if (active) {
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int64_t row = row0 + 2 * lane + a;
            const double xi = row < N ? w.xn[row] : 0.0;
#pragma unroll
            for (int c = 0; c < TN; ++c) {
                const int l = wid * TN + c;
                if (l < m) {
                    const int pos = w.acc_pos[l];
                    if (w.prop[pos] == row) {
                        acc[a][c] = 1.0;
                    } else {
                        const double d2 = fmax(xi + w.xnS[pos] - 2.0 * acc[a][c], 0.0);
                        acc[a][c] = exp(-d2 * inv_eps);
                    }
                }
            }
        }
    }
    // ---- minus F(i,:k) . F(s,:k) ----
    for (int c0 = 0; c0 < k; c0 += kBK) {
#pragma unroll
        for (int p = 0; p < (kBM * kBK) / 256; ++p) {
            const int e = tid + 256 * p, kk = e / kBM, i = e % kBM;
            const int64_t row = row0 + i;
            As[kk * APAD + i] = (row < N && c0 + kk < k) ? F[(int64_t)(c0 + kk) * ldf + row] : 0.0;
        }
        for (int e = tid; e < kBK * BN; e += 256) {
            const int kk = e / BN, l = e % BN;
            Bs[kk * BN + l] = (l < m && c0 + kk < k) ? w.FSP[(size_t)(c0 + kk) * b + w.acc_pos[l]] : 0.0;
        }
        __syncthreads();
        if (active) {
#pragma unroll
            for (int kk = 0; kk < kBK; ++kk) {
                const double2 a = *reinterpret_cast<const double2*>(&As[kk * APAD + 2 * lane]);
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const double bv = Bs[kk * BN + wid * TN + c];
                    acc[0][c] = fma(-a.x, bv, acc[0][c]);
                    acc[1][c] = fma(-a.y, bv, acc[1][c]);
                }
            }
        }
        __syncthreads();
    }
    // ---- R tile to shared memory ----
    if (active) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < TN; ++c) Rs[(2 * lane + a) * (BN + 1) + wid * TN + c] = acc[a][c];
    }
    __syncthreads();
    // ---- G = R L^-T by forward substitution, rho update ----
    double rnew = 0.0;
    double rmax = -1.0;
    int64_t ridx = LLONG_MAX;
    if (tid < kBM) {
        const int64_t row = row0 + tid;
        double* Ri = Rs + tid * (BN + 1);
        double nrm = 0.0;
        for (int j = 0; j < m; ++j) {
            const double* Lj = w.Lc + (size_t)j * b;
            double s = Ri[j];
            for (int l = 0; l < j; ++l) s = fma(-__ldg(Lj + l), Ri[l], s);
            const double g = s / __ldg(Lj + j);
            Ri[j] = g;
            nrm = fma(g, g, nrm);
        }
        if (row < N) {
            rnew = fmax(rho[row] - nrm, 0.0);
            rho[row] = rnew;
            rmax = rnew;
            ridx = row;
        }
    }
    __syncthreads();
    for (int e = tid; e < kBM * m; e += 256) {
        const int l = e / kBM, i = e % kBM;
        const int64_t row = row0 + i;
        if (row < N) F[(int64_t)(k + l) * ldf + row] = Rs[i * (BN + 1) + l];
    }
    // ---- per-tile sum and (max, lowest index) of rho ----
    double s = warp_sum(rnew);
    warp_argmax(rmax, ridx);
    if (lane == 0) {
        red[wid] = s;
        redi[wid] = ridx;
        red[16 + wid] = rmax;
    }
    __syncthreads();
    if (tid == 0) {
        double ts = 0.0, tm = -1.0;
        int64_t ti = LLONG_MAX;
        for (int q = 0; q < (kBM + 31) / 32; ++q) {
            ts += red[q];
            argmax_merge(tm, ti, red[16 + q], redi[q]);
        }
        w.tile_sum[tile] = ts;
        w.tile_max[tile] = tm;
        w.tile_idx[tile] = ti;
    }
    __syncthreads();   // shared buffers are reused by the next tile of a persistent caller
}

template <int TN>
__global__ void __launch_bounds__(256) k_engine(FactorWs w, const double* __restrict__ X, double* __restrict__ F,
                                                int64_t ldf, double* __restrict__ rho, int64_t N, int d, int b,
                                                double inv_eps) {
    extern __shared__ double smem_eng[];
    engine_body<TN>(w, X, F, ldf, rho, N, d, b, inv_eps, blockIdx.x, smem_eng);
}

// Digit planes of X (seven digits, one exponent per row from max |X(i, :)|),
// columns d .. ldX - 1 zero.  Block: 32 rows x 8 quarters of 16 columns; a thread cuts
// one row's quarter, so that a warp's store fills 32 rows' consecutive 32 bytes of a
// plane.
__global__ void __launch_bounds__(256) k_xplanes(const double* __restrict__ X, int64_t N, int d, OzWs o) {
    __shared__ unsigned long long red[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    const int nq = o.ldX / 16;
    const double* x = X + (i < N ? i : 0) * d;
    double v[16];
    unsigned long long mx = 0;
    for (int q = wid; q < nq; q += 8) {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            v[e] = i < N && 16 * q + e < d ? x[16 * q + e] : 0.0;
            mx = max(mx, (unsigned long long)__double_as_longlong(v[e]) & 0x7FFFFFFFFFFFFFFFull);
        }
    }
    red[wid][lane] = mx;
    __syncthreads();
    if (i >= N) return;
#pragma unroll
    for (int u = 0; u < 8; ++u) mx = max(mx, red[u][lane]);
    const int E = exp_of(__longlong_as_double((long long)mx));
    if (wid == 0) o.xe[i] = E;
    for (int q = wid; q < nq; q += 8) {
        long long t[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (nq > 8) v[e] = 16 * q + e < d ? x[16 * q + e] : 0.0;    // one quarter per warp is still in v
            t[e] = oz_T_f64<kDigits>(v[e], E);
        }
        oz_store_quarter<kDigits>(o.Xp, i, q, nq, t);
    }
}

// Pivot panels of the round as rows of the digit planes: row l < m of PXp is
// row S_l of Xp (exponent pxe_l), row l of PFp is row S_l of Fp over the padded
// rank kp; rows l >= m are zero.  One block per row l; a thread copies the 32 bytes of
// one quarter and plane (halves exchanged when the two rows' swizzles differ).
__global__ void __launch_bounds__(128) k_ozpanel(FactorWs w, OzWs o, int64_t N, int b) {
    const FactorState* st = w.st;
    if (st->done || st->m == 0) return;
    const int l = blockIdx.x;
    if (l >= b) return;
    const bool on = l < st->m;
    const int64_t row = on ? w.prop[w.acc_pos[l]] : 0;
    if (threadIdx.x == 0) o.pxe[l] = on ? o.xe[row] : -900;
    const int flip = ((int)(row >> 2) ^ (l >> 2)) & 1;
    auto gather = [&](const uint16_t* src, uint16_t* dst, int nq, int nused) {
        for (int u = threadIdx.x; u < nused * kDigits; u += blockDim.x) {
            const int q = u / kDigits, z = u % kDigits;
            const uint4* sp = reinterpret_cast<const uint4*>(src + oz_tile_at(row, q, z, nq, kDigits));
            uint4* dp = reinterpret_cast<uint4*>(dst + oz_tile_at(l, q, z, nq, kDigits));
            const uint4 zero = make_uint4(0, 0, 0, 0);
            dp[0] = on ? sp[flip] : zero;
            dp[1] = on ? sp[flip ^ 1] : zero;
        }
    };
    gather(o.Xp, o.PXp, o.ldX / 16, o.ldX / 16);
    gather(o.Fp, o.PFp, o.ldF / 16, st->kp / 16);
}

// L(T,T)^-1 of the round (lower triangular, m x m).  Each round's L is the Cholesky
// factor of Algorithm 3's accepted block, whose accept test keeps it well
// conditioned, so multiplying by the explicit inverse agrees with substitution to
// rounding (measured 2e-15 on KS data).  One warp per column c (forward substitution on
// L x = e_c): lane holds the right-hand sides of rows lane + 32 u; a step divides one of
// them (by a reciprocal and the residual's correction) and subtracts it from the rows
// below.  Four warps per CTA, so that each has a quarter of an SM's FP64 pipe to itself
// (one CTA for all columns: 489 us per round at b = 128, its chain of ~8,000 dependent
// operations; this one: 62 us, 4 more for the planes).
constexpr int kLinvWarps = 4;
__global__ void __launch_bounds__(32 * kLinvWarps) k_linv(FactorWs w, OzWs o, int b) {
    extern __shared__ double Ls[];                               // column l of L at Ls + l (m + 1), rows l .. m - 1 used
    const FactorState* st = w.st;
    if (st->done || st->m == 0) return;
    const int m = st->m, lane = threadIdx.x & 31;
    const int c = blockIdx.x * kLinvWarps + (threadIdx.x >> 5);
    const int cf = blockIdx.x * kLinvWarps;                      // no column of this CTA reads L's columns before cf
    if (cf >= m) return;
    const int ld = m + 1;
    double* inv = Ls + (size_t)m * ld;                            // 1 / L(l, l)
    for (int e = threadIdx.x; e < m * m; e += blockDim.x) {
        const int j = e / m, l = e % m;
        if (l >= cf && l <= j) Ls[(size_t)l * ld + j] = w.Lc[(size_t)j * b + l];
    }
    __syncthreads();
    for (int l = cf + threadIdx.x; l < m; l += blockDim.x) inv[l] = 1.0 / Ls[(size_t)l * ld + l];
    __syncthreads();
    if (c >= m) return;
    double x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = lane + 32 * u == c ? 1.0 : 0.0;
    for (int l = c; l < m; ++l) {
        const double* Ll = Ls + (size_t)l * ld;
        const double rhs = l < 32 ? x[0] : l < 64 ? x[1] : l < 96 ? x[2] : x[3];
        double v = rhs * inv[l];
        v = fma(fma(-v, Ll[l], rhs), inv[l], v);
        v = __shfl_sync(0xffffffffu, v, l & 31);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = lane + 32 * u;
            if (32 * u + 31 > l) {                               // rows below l in this group
                if (j == l) x[u] = v;
                else if (j > l && j < m) x[u] = fma(-Ll[j], v, x[u]);
            } else if (j == l) {
                x[u] = v;
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (lane + 32 * u < m) o.Linv[(size_t)(lane + 32 * u) * o.ldLi + c] = lane + 32 * u >= c ? x[u] : 0.0;
}

// Digit planes of the rows of L^-1 (columns past the diagonal and rows past m zero) and
// their exponents; one warp per row.
__global__ void __launch_bounds__(128) k_linv_planes(FactorWs w, OzWs o, int b) {
    const FactorState* st = w.st;
    if (st->done || st->m == 0) return;
    const int m = st->m, lane = threadIdx.x & 31, j = blockIdx.x * 4 + (threadIdx.x >> 5), nq = o.ldR / 16;
    if (j >= b) return;
    const double* row = o.Linv + (size_t)j * o.ldLi;
    unsigned long long mx = 0;
    for (int l = lane; l <= j && j < m; l += 32)
        mx = max(mx, (unsigned long long)__double_as_longlong(row[l]) & 0x7FFFFFFFFFFFFFFFull);
#pragma unroll
    for (int q = 16; q; q >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, q));
    const int E = exp_of(__longlong_as_double((long long)mx));
    if (lane == 0) o.le[j] = E;
    if (lane < nq) {
        long long t[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) t[e] = oz_T_f64<kDigits>(j < m && 16 * lane + e <= j ? row[16 * lane + e] : 0.0, E);
        oz_store_quarter<kDigits>(o.Lp, j, lane, nq, t);
    }
}

// R = K(:, T) - F(:, :k) F(T, :k)^T from the tensor-core products: the kernel
// values exp(-(|x_i|^2 + |x_s|^2 - 2 x_i.x_s) / eps) (1 at the pivot itself)
// minus Df, as digit planes with one exponent per row (the row maximum over
// the round's pivots).  Block: 32 rows x ldR / 16 warps, warp g taking the quarter of
// 16 pivots [16 g, 16 g + 16).  The squared distance (two operations) and the difference
// are FP64, 17 cycles per warp and SM each; the scaling by 1 / eps, the exponential
// (kexp_bits) and the digits run on the integer pipe.  R has to be a double here: on a common
// grid of 2^-62 a row far from every pivot loses its digits, and beyond exp(-43) all of them.
// Bound: the integer pipe (HBM: 30 bytes per value, 0.5 ms).  N = 1M, b = 128: 2.8 ms per
// round with nine FP64 operations per value, 1.5 ms now.
__global__ void __launch_bounds__(256) k_rprep(FactorWs w, OzWs o, int64_t N, KexpScale inv_eps,
                                               const unsigned long long* __restrict__ tblg) {
    const FactorState* st = w.st;
    if (st->done || st->m == 0) return;
    const int m = st->m, k = st->k;
    __shared__ unsigned long long red[8][32];
    __shared__ unsigned long long tbl[1024];
    __shared__ double s_xn[128];
    __shared__ int64_t s_row[128];
    for (int e = threadIdx.x; e < 1024; e += blockDim.x) tbl[e] = tblg[e];
    for (int l = threadIdx.x; l < m; l += blockDim.x) {
        const int pos = w.acc_pos[l];
        s_xn[l] = w.xnS[pos];
        s_row[l] = w.prop[pos];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5, nq = o.ldR / 16;
    const int l0 = 16 * g;
    for (int64_t row0 = (int64_t)blockIdx.x * 32; row0 < N; row0 += (int64_t)gridDim.x * 32) {
        const int64_t row = row0 + lane;
        const bool on = row < N;
        const double xi = on ? w.xn[row] : 0.0;
        long long R[16];                                       // bits of doubles, then their digits
        unsigned long long mx = 0;                             // max |R|
        // four values at a time, the next four in flight; rolled, R moving down
        double dx[4], df[4];
        auto load = [&](int u) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int64_t at = row + (int64_t)(l0 + 4 * u + e) * w.ldD;
                const bool in = on && l0 + 4 * u + e < m;
                dx[e] = in ? w.Dx[at] : 0.0;
                df[e] = in && k > 0 ? w.Df[at] : 0.0;
            }
        };
        load(0);
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
            double cx[4], cf[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                cx[e] = dx[e];
                cf[e] = df[e];
            }
            if (u < 3) load(u + 1);
#pragma unroll
            for (int e = 0; e < 12; ++e) R[e] = R[e + 4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int l = l0 + 4 * u + e;
                long long v = 0;
                if (on && l < m) {
                    const double kv = s_row[l] == row ? 1.0
                                                      : __longlong_as_double((long long)kexp_bits(
                                                            fma(-2.0, cx[e], xi + s_xn[l]), inv_eps, tbl));
                    v = __double_as_longlong(kv - cf[e]);
                    mx = max(mx, (unsigned long long)v & 0x7FFFFFFFFFFFFFFFull);
                }
                R[12 + e] = v;
            }
        }
        red[g][lane] = mx;
        __syncthreads();
        for (int q = 0; q < nq; ++q) mx = max(mx, red[q][lane]);
        __syncthreads();                                       // red is rewritten for the next rows
        if (!on) continue;
        const int E = exp_of(__longlong_as_double((long long)mx));
        if (g == 0) o.re[row] = E;
#pragma unroll
        for (int e = 0; e < 16; ++e) R[e] = oz_T_f64<kDigits>(__longlong_as_double(R[e]), E);
        oz_store_quarter<kDigits>(o.Rp, row, g, nq, R);
    }
}

// After G = R L^-T has been written to F(:, k:k+m): rho -= rownorms(G)^2 (clamped
// at 0) and the per-tile sum and (max, lowest index) of rho for the next round's
// sampler.  Block: one 64-row tile x 4 column groups.
__global__ void __launch_bounds__(256) k_rho_update(FactorWs w, const double* __restrict__ F, int64_t ldf,
                                                    double* __restrict__ rho, int64_t N) {
    const FactorState* st = w.st;
    if (st->done || st->m == 0) return;
    const int m = st->m, k = st->k;
    __shared__ double sn[4][64];
    __shared__ double red[2];
    __shared__ double redm[2];
    __shared__ int64_t redi[2];
    const int il = threadIdx.x & 63, g = threadIdx.x >> 6;
    const int64_t tile = blockIdx.x, row = tile * 64 + il;
    double nrm = 0.0;
    if (row < N) {
        for (int l = g; l < m; l += 4) {
            const double v = F[(int64_t)(k + l) * ldf + row];
            nrm = fma(v, v, nrm);
        }
    }
    sn[g][il] = nrm;
    __syncthreads();
    if (g == 0) {
        double rnew = 0.0, rmax = -1.0;
        int64_t ridx = LLONG_MAX;
        if (row < N) {
            const double tot = (sn[0][il] + sn[1][il]) + (sn[2][il] + sn[3][il]);
            rnew = fmax(rho[row] - tot, 0.0);
            rho[row] = rnew;
            rmax = rnew;
            ridx = row;
        }
        const double s2 = warp_sum(rnew);
        warp_argmax(rmax, ridx);
        if ((il & 31) == 0) {
            red[il >> 5] = s2;
            redm[il >> 5] = rmax;
            redi[il >> 5] = ridx;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && tile * 64 < N) {
        double tm = redm[0];
        int64_t ti = redi[0];
        argmax_merge(tm, ti, redm[1], redi[1]);
        w.tile_sum[tile] = red[0] + red[1];
        w.tile_max[tile] = tm;
        w.tile_idx[tile] = ti;
    }
}

// ---------------------------------------------------------------------------
// Commit the last round, sum(rho) in a fixed order, zero F(:, rank:r).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void finalize_body(FactorWs w, const double* __restrict__ rho, int64_t N) {
    __shared__ double sh[32];
    FactorState* st = w.st;
    const int64_t chunk = (N + blockDim.x - 1) / blockDim.x;
    const int64_t i0 = min((int64_t)threadIdx.x * chunk, N), i1 = min(i0 + chunk, N);
    double s = 0.0;
    for (int64_t i = i0; i < i1; ++i) s += rho[i];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) {
        if (st->m > 0) {
            st->sum_k += st->k;
            st->eng_rounds += 1;
        }
        st->k += st->m;
        st->kp += (st->m + 15) & ~15;
        st->sum_m_sq += (long long)st->m * st->m;
        st->m = 0;
        st->final_sum = s;
    }
}

__global__ void __launch_bounds__(1024) k_finalize(FactorWs w, const double* __restrict__ rho, int64_t N) {
    finalize_body(w, rho, N);
}

template <typename TF>
__global__ void k_zero_tail(const FactorState* st, TF* __restrict__ F, int64_t ldf, int64_t N, int r) {
    const int k = st->k;
    const int c = k + blockIdx.y;
    if (c >= r) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
        F[(int64_t)c * ldf + i] = TF(0);
}

template <int TN>
static size_t engine_smem() {
    constexpr int BN = 8 * TN;
    const size_t stage = (size_t)(kBK * (kBM + 2) + kBK * BN) * sizeof(double);
    const size_t rtile = (size_t)kBM * (BN + 1) * sizeof(double);
    return std::max(stage, rtile);
}

// ---------------------------------------------------------------------------
// Greedy rounds of an FP64 factor in one cooperative launch, for N <= 65,536.
//
// A greedy round is a step of r dependent ones, and in launches of its own (proposal,
// gather, H, acceptance, engine) it is mostly their latency: 48 us at N = 2,000, d = 64.
// Here a CTA owns a 64-row tile for all rounds, a thread a row (its residual in a register),
// a third warp takes H and its root meanwhile, and a round has one grid barrier, after which
// every CTA finds the argmax of the tiles' (max, index) pairs by itself.  What bounds it is
// the chain of d + k dependent FP64 operations of 64 cycles that a row's value is defined by:
// same operations in the same order as the kernels above, so the same bits: 15 us a round at
// N = 2,000, k up to 128.  The line at 1,024 tiles: up to there a pair of tile statistics per thread and
// 16 loads find the argmax, and all CTAs are resident (7 of 64 + 32 threads per SM); above,
// a round's work on the FP64 pipe outweighs the launches.  Whole factors below the line, this kernel /
// launches of their own (ms): N = 65,536, d = 64, r = 128 4.9 / 9.1, r = 512 44 / 66, d = 2,048,
// r = 32 16.3 / 20.5; N = 20,000, d = 64, r = 1,024 105 / 106.  Pairs alternate between two
// buffers, since a CTA may be one round ahead of another's reading.
// ---------------------------------------------------------------------------
constexpr int kGreedyTiles = 1024;
constexpr int kGreedyThreads = kBM + 32;
constexpr int kGreedyChunk = 512;         // columns of X(p,:) and F(p,:) in shared memory
constexpr int kGreedyPolls = 1 << 22;     // of the barrier, seconds in all

__global__ void __launch_bounds__(kGreedyThreads) k_greedy(FactorWs w, const double* __restrict__ X, double* F,
                                                           int64_t ldf, double* __restrict__ rho, int64_t N, int d,
                                                           int r, int rounds, double inv_eps,
                                                           int64_t* __restrict__ pivots,
                                                           int64_t* __restrict__ proposals_out) {
    __shared__ double sx[kGreedyChunk], sf[kGreedyChunk];
    __shared__ double sv[3];
    __shared__ int64_t si[3];
    __shared__ double s_h, s_root;
    __shared__ int s_ok;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int ntiles = gridDim.x;
    const int64_t row = (int64_t)blockIdx.x * kBM + tid;
    const bool owns = tid < kBM && row < N;
    const bool first = blockIdx.x == 0 && tid == 0;
    int* const arrived = w.tpos;              // zero at launch
    const double xi = owns ? w.xn[row] : 0.0;
    const double* const Xi = X + (owns ? row : 0) * d;
    const double* const Fi = F + (owns ? row : 0);
    double rv = owns ? rho[row] : 0.0, total = 0.0;
    int k = 0, ran = 0, done = 0;
    long long sum_k = 0;
    for (int rnd = 0; rnd < rounds; ++rnd) {
        if (k >= r) {
            done = 1;
            break;
        }
        // ---- argmax of rho ----
        const double* tmax = rnd & 1 ? w.pre : w.tile_max;
        const int64_t* tidx = rnd & 1 ? reinterpret_cast<const int64_t*>(w.tile_sum) : w.tile_idx;
        double v = -1.0;
        int64_t p = LLONG_MAX;
        for (int t = tid; t < ntiles; t += kGreedyThreads) argmax_merge(v, p, __ldcg(tmax + t), __ldcg(tidx + t));
        warp_argmax(v, p);
        if (lane == 0) {
            sv[wid] = v;
            si[wid] = p;
        }
        __syncthreads();
        v = sv[0];
        p = si[0];
        argmax_merge(v, p, sv[1], si[1]);
        argmax_merge(v, p, sv[2], si[2]);
        if (!(v > 0.0)) {
            done = 1;
            break;
        }
        total = v;
        ++ran;
        if (first && proposals_out) proposals_out[rnd] = p;
        // ---- X(p,:), F(p,:k) to shared memory, a chunk at a time; the row's chains; H in warp 2 ----
        auto stage_x = [&](int c0) {
            for (int c = tid; c < min(kGreedyChunk, d - c0); c += kGreedyThreads) sx[c] = X[p * d + c0 + c];
        };
        auto stage_f = [&](int c0) {
            for (int c = tid; c < min(kGreedyChunk, k - c0); c += kGreedyThreads)
                sf[c] = __ldcg(F + (int64_t)(c0 + c) * ldf + p);
        };
        const double xp = w.xn[p];
        stage_x(0);
        stage_f(0);
        __syncthreads();
        double acc = 0.0;                     // warp 2: terms c = lane mod 32 of F(p,:) . F(p,:)
        for (int c0 = 0; c0 < d; c0 += kGreedyChunk) {
            if (c0 > 0) {
                __syncthreads();
                stage_x(c0);
                __syncthreads();
            }
            const int n = min(kGreedyChunk, d - c0);
            if (owns) {
#pragma unroll 16
                for (int c = 0; c < n; ++c) acc = fma(Xi[c0 + c], sx[c], acc);
            }
        }
        if (owns) acc = p == row ? 1.0 : exp(-fmax(xi + xp - 2.0 * acc, 0.0) * inv_eps);
        for (int c0 = 0; c0 < k; c0 += kGreedyChunk) {
            if (c0 > 0) {
                __syncthreads();
                stage_f(c0);
                __syncthreads();
            }
            const int n = min(kGreedyChunk, k - c0);
            if (owns) {
#pragma unroll 16
                for (int c = 0; c < n; ++c) acc = fma(-Fi[(int64_t)(c0 + c) * ldf], sf[c], acc);
            } else if (wid == 2) {
                for (int c = lane; c < n; c += 32) acc = fma(sf[c], sf[c], acc);
            }
        }
        if (wid == 2) {
            const double h = 1.0 - warp_sum(acc);
            if (lane == 0) {
                s_h = h;
                s_root = sqrt(h);
            }
        }
        __syncthreads();
        if (!(s_h > 0.0)) {                   // greedy stops once H <= 0
            done = 1;
            break;
        }
        // ---- column k of F, the residual, the tile's (max, lowest index) ----
        double rmax = -1.0;
        int64_t ridx = LLONG_MAX;
        if (owns) {
            const double g = acc / s_root;
            F[(int64_t)k * ldf + row] = g;
            rv = fmax(rv - __dmul_rn(g, g), 0.0);
            rmax = rv;
            ridx = row;
        }
        if (first) pivots[k] = p;
        sum_k += k;
        ++k;
        if (rnd + 1 == rounds) break;
        if (wid < 2) {
            warp_argmax(rmax, ridx);
            if (lane == 0) {
                sv[wid] = rmax;
                si[wid] = ridx;
            }
        }
        __syncthreads();
        // ---- publish and wait for all tiles ----
        if (tid == 0) {
            argmax_merge(rmax, ridx, sv[1], si[1]);
            (rnd & 1 ? w.tile_max : w.pre)[blockIdx.x] = rmax;
            (rnd & 1 ? w.tile_idx : reinterpret_cast<int64_t*>(w.tile_sum))[blockIdx.x] = ridx;
            __threadfence();
            atomicAdd(arrived, 1);
            const int want = (rnd + 1) * ntiles;
            int got = 0;
            for (int i = 0; i < kGreedyPolls; ++i) {
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(got) : "l"(arrived) : "memory");
                if (got >= want) break;
            }
            s_ok = got >= want;
            if (got < want) w.st->timeout = 1;
        }
        __syncthreads();
        if (!s_ok) break;
    }
    if (owns) rho[row] = rv;
    if (first) {
        FactorState* st = w.st;
        st->k = k;
        st->kp = 16 * k;
        st->rounds = ran;
        st->done = done;
        st->total = total;
        st->sum_m_sq = k;
        st->sum_k = sum_k;
        st->eng_rounds = k;
    }
}

// CTAs of k_greedy for N rows, 0 where they cannot all be resident, N is past its line, or a
// round's chain of d steps could outlast the barrier's polls.
static int greedy_ctas(int64_t N, int d) {
    const int64_t ntiles = (N + kBM - 1) / kBM;
    if (ntiles > kGreedyTiles || d > (1 << 16)) return 0;
    int dev = 0, nsm = 0, per_sm = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_greedy, kGreedyThreads, 0) != cudaSuccess)
        return 0;
    return coop && ntiles <= (int64_t)nsm * per_sm ? (int)ntiles : 0;
}

static cudaError_t launch_greedy(int ctas, FactorWs w, const double* X, double* F, int64_t ldf, double* rho, int64_t N,
                                 int d, int r, int rounds, double inv_eps, int64_t* pivots, int64_t* proposals,
                                 cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(w.tpos, 0, sizeof(int32_t), s);
    if (e != cudaSuccess) return e;
    void* args[] = {&w, &X, &F, &ldf, &rho, &N, &d, &r, &rounds, &inv_eps, &pivots, &proposals};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_greedy), dim3(ctas), dim3(kGreedyThreads), args, 0,
                                       s);
}

template <int TN>
static cudaError_t prepare_engine() {
    return cudaFuncSetAttribute(k_engine<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)engine_smem<TN>());
}

template <int TN>
static void launch_engine(const FactorWs& w, const double* X, double* F, int64_t ldf, double* rho,
                          int64_t N, int d, int b, double inv_eps, int64_t ntiles, cudaStream_t s) {
    k_engine<TN><<<(unsigned)ntiles, 256, engine_smem<TN>(), s>>>(w, X, F, ldf, rho, N, d, b, inv_eps);
}

// Round launchers of the FP64 path, shared with the low-memory factor.
FactorWs carve_factor_fp64(void* base, int64_t N, int d, int r, int b, size_t* bytes) {
    return carve_factor(base, N, d, r, b, bytes);
}

void launch_prepare_fp64(const double* X, int64_t N, int d, const FactorWs& w, double* rho, cudaStream_t s) {
    k_prepare<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(X, N, d, w, rho);
}

void launch_propose(const FactorWs& w, const double* rho, int64_t N, int b, int r, int greedy, uint64_t seed, int rnd,
                    int64_t* proposals, double floor_sum, cudaStream_t s) {
    const int64_t ntiles = (N + kBM - 1) / kBM;
    if (greedy)
        k_propose_greedy<<<1, 1024, 0, s>>>(w, ntiles, r, rnd, proposals);
    else
        k_propose<<<kPropCluster, kPropThreads, 0, s>>>(w, rho, N, ntiles, b, r, seed, rnd, proposals, floor_sum);
}

void launch_blockH(const FactorWs& w, int d, int b, double inv_eps, cudaStream_t s) {
    k_blockH<<<blockH_blocks(b), kBlockHThreads, 0, s>>>(w, d, b, inv_eps);
}

cudaError_t launch_reject(const FactorWs& w, int b, int r, int greedy, uint64_t seed, int rnd, int64_t* pivots,
                          cudaStream_t s) {
    if (greedy) k_reject_greedy<<<1, 32, 0, s>>>(w, r, pivots);
    else k_reject<<<kRejCluster, kRejThreads, 0, s>>>(w, b, r, seed, rnd, pivots);
    return cudaGetLastError();
}

void launch_finalize(const FactorWs& w, const double* rho, int64_t N, cudaStream_t s) {
    k_finalize<<<1, 1024, 0, s>>>(w, rho, N);
}

cudaError_t launch_linv(const FactorWs& w, const OzWs& o, int b, cudaStream_t s) {
    // (the largest block's, so that calls with other blocks leave the limit as it is)
    constexpr int kMost = (128 * 128 + 2 * 128) * (int)sizeof(double);
    const cudaError_t e = cudaFuncSetAttribute(k_linv, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
    if (e != cudaSuccess) return e;
    k_linv<<<(b + kLinvWarps - 1) / kLinvWarps, 32 * kLinvWarps, ((size_t)b * b + 2 * b) * sizeof(double), s>>>(w, o, b);
    k_linv_planes<<<(b + 3) / 4, 128, 0, s>>>(w, o, b);
    return cudaGetLastError();
}

cudaError_t oz_cut_rowmajor(const double* X, int64_t N, int K, uint16_t* P, int* ex, cudaStream_t s) {
    OzWs o{};
    o.Xp = P;
    o.xe = ex;
    o.ldX = (K + 15) / 16 * 16;
    k_xplanes<<<(unsigned)((N + 31) / 32), 256, 0, s>>>(X, N, K, o);
    return cudaGetLastError();
}

}  // namespace kevd

using namespace kevd;

static int factor_rounds(const kevd_opts* o, int r, int b) {
    if (o->until_rank) return o->max_rounds > 0 ? o->max_rounds : 4 * ((r + b - 1) / b) + 16;
    return r / b;
}

static size_t factor_ws_bytes(int64_t N, int d, int r, int b, bool tc, bool oz, int rounds_max, bool pl) {
    size_t bytes = 0;
    carve_factor(nullptr, N, d, r, b, &bytes, tc, nullptr, oz, nullptr, rounds_max, pl);
    return bytes;
}

// The precision form's engine reads pre-split planes (as large as F) for blocks of b >= 32
// (a round rewrites the 16-column groups it shares with the last, which smaller blocks would
// do too often), while they stay within 48 GiB, so that a factor that only just fits the
// card keeps the engine that needs no copy, and where the caller gives a workspace.  The planes of
// X cost one pass over it, which the rounds have to win back: for d b <= 3 r^2, that is d <= 3 t^2 b
// with t = r / b rounds.  Whole factor at N = 200,000, planes against splitting in every round (ms):
// t = 1, b = 64, d = 128 0.51 / 0.54, d = 256 0.72 / 0.67; t = 1, b = 128, d = 256 0.79 / 0.89, d = 512
// 1.23 / 1.19; t = 2, b = 32, d = 256 0.84 / 0.89, d = 512 1.33 / 1.25; t = 4, b = 64, d = 2,048
// 5.16 / 6.05.
static bool pl_engine_for(const kevd_opts* o, int64_t N, int d, int r, int b, bool workspace) {
    int nxh, nH;
    return workspace && o->precision == KEVD_PREC_BF16X3 && b >= 32 && (int64_t)d * b <= 3 * (int64_t)r * r &&
           tc_plane_bytes(N, d, r, &nxh, &nH) <= ((size_t)48 << 30);
}

// The FP64 path runs its engine on the tensor cores (FP64-accurate digit planes,
// ozmm.cu) for ARPC with b >= 32 (each round's block of F's planes is padded to
// 16 columns) and N < 2^31, unless KEVD_ENGINE=fp64 asks for the FP64-pipe
// engine; the workspace then holds two N x b product arrays and the planes.
bool kevd::oz_engine_enabled() {
    const char* e = getenv("KEVD_ENGINE");
    return !(e && e[0] == 'f');
}

static bool oz_engine_for(const kevd_opts* o, int64_t N, int b, bool allow_oz) {
    return allow_oz && o->precision == KEVD_PREC_FP64 && o->mode == KEVD_ARPC && b >= 32 &&
           N < ((int64_t)1 << 31) && oz_engine_enabled();
}

size_t kevd_factor_ws_mode(int64_t N, int32_t d, int32_t r, const kevd_opts* o, bool allow_oz) {
    if (!o || N < 1 || d < 1 || r < 1) return 0;
    const int b = o->mode == KEVD_GREEDY ? 1 : o->block_b;
    if (b < 1 || b > 128) return 0;
    const bool tc = o->precision == KEVD_PREC_BF16X3;
    return factor_ws_bytes(N, d, r, b, tc, oz_engine_for(o, N, b, allow_oz), factor_rounds(o, r, b),
                           pl_engine_for(o, N, d, r, b, allow_oz));
}

size_t kevd_factor_ws(int64_t N, int32_t d, int32_t r, const kevd_opts* o) {
    return kevd_factor_ws_mode(N, d, r, o, true);
}

int rpchol_factor_impl(const void* X, int x_dtype, int64_t N, int32_t d, double eps, int32_t r,
                       const kevd_opts* opts, void* F, int f_dtype, int64_t ldf, int64_t* pivots, double* rho,
                       int64_t* proposals, kevd_factor_info* info, void* workspace, size_t ws_bytes, void* stream,
                       bool allow_oz) {
    if (!opts || !X || !F || !pivots || !rho || !info) return KEVD_EINVAL;
    if (N < 1 || d < 1 || r < 1 || r > N || ldf < N) return KEVD_EINVAL;
    if (!(eps > 0.0) || !isfinite(eps)) return KEVD_EINVAL;
    if (opts->mode != KEVD_GREEDY && opts->mode != KEVD_ARPC) return KEVD_EINVAL;
    const bool tc = opts->precision == KEVD_PREC_BF16X3;
    if (opts->precision == KEVD_PREC_FP64) {
        if (x_dtype != KEVD_F64 || f_dtype != KEVD_F64) return KEVD_EINVAL;
    } else if (tc) {
        if (x_dtype != KEVD_F32 || f_dtype != KEVD_F32) return KEVD_EINVAL;
    } else {
        return KEVD_EINVAL;
    }
    if (opts->reserved != 0 || opts->max_rounds < 0) return KEVD_EINVAL;
    if (!(opts->tol >= 0.0 && opts->tol < 1.0)) return KEVD_EINVAL;
    const int greedy = opts->mode == KEVD_GREEDY;
    const int b = greedy ? 1 : opts->block_b;
    if (b < 1 || b > 128) return KEVD_EINVAL;
    const int rounds = greedy && !opts->until_rank ? r : factor_rounds(opts, r, b);
    if (rounds < 1) return KEVD_EINVAL;
    size_t need = 0;
    PanelWs pw{};
    OzWs ow{};
    const bool oz = oz_engine_for(opts, N, b, allow_oz), pl = pl_engine_for(opts, N, d, r, b, allow_oz);
    FactorWs w = carve_factor(workspace, N, d, r, b, &need, tc, &pw, oz, &ow, factor_rounds(opts, r, b), pl);
    if (pl && ws_bytes < need)   // no room for the planes: the engine that splits its operands in every round, same bits
        w = carve_factor(workspace, N, d, r, b, &need, tc, &pw, oz, &ow, factor_rounds(opts, r, b), false);
    if (!workspace || ws_bytes < need || (reinterpret_cast<uintptr_t>(workspace) % kAlign)) return KEVD_EWORKSPACE;
    // the digit planes: X and F (A operands), the pivot panels (B), R and L^-1 of each round
    const unsigned long long* exp_tbl = nullptr;
    const OzOperand oX{ow.Xp, ow.ldX / 16, ow.xe, 0}, oPX{ow.PXp, ow.ldX / 16, ow.pxe, 0},
        oF{ow.Fp, ow.ldF / 16, nullptr, 1}, oPF{ow.PFp, ow.ldF / 16, nullptr, 1}, oR{ow.Rp, ow.ldR / 16, ow.re, 0},
        oL{ow.Lp, ow.ldR / 16, ow.le, 0};

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const double* Xd = static_cast<const double*>(X);
    double* Fd = static_cast<double*>(F);
    const float* Xf = static_cast<const float*>(X);
    float* Ff = static_cast<float*>(F);
    const int64_t ntiles = (N + kBM - 1) / kBM;
    const double inv_eps = 1.0 / eps;

    {
        TraceScope tr(kStOther, s);
        if (tc) {
            KEVD_CUDA_TRY(cudaMemsetAsync(pw.err, 0, sizeof(int), s));
            k_prepare<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(Xf, N, d, w, rho);
            if (pw.planes) launch_xsplit(Xf, N, d, pw, s);
        } else {
            k_prepare<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(Xd, N, d, w, rho);
            if (oz) {
                KEVD_CUDA_TRY(kexp_table(s, &exp_tbl));
                KEVD_CUDA_TRY(oz_cut_rowmajor(Xd, N, d, ow.Xp, ow.xe, s));
                KEVD_CUDA_TRY(cudaMemsetAsync(ow.flags, 0, sizeof(int), s));
            }
        }
    }
    KEVD_LAUNCH_CHECK();
    const int tn = b <= 8 ? 1 : b <= 16 ? 2 : b <= 32 ? 4 : b <= 64 ? 8 : 16;
    switch (tn) {
        case 1: KEVD_CUDA_TRY(prepare_engine<1>()); break;
        case 2: KEVD_CUDA_TRY(prepare_engine<2>()); break;
        case 4: KEVD_CUDA_TRY(prepare_engine<4>()); break;
        case 8: KEVD_CUDA_TRY(prepare_engine<8>()); break;
        default: KEVD_CUDA_TRY(prepare_engine<16>()); break;
    }

    const int gctas = greedy && !tc ? greedy_ctas(N, d) : 0;
    if (gctas > 0) {
        TraceScope tr(kStEngine, s);
        KEVD_CUDA_TRY(launch_greedy(gctas, w, Xd, Fd, ldf, rho, N, d, r, rounds, inv_eps, pivots, proposals, s));
    }
    for (int rnd = 0; rnd < rounds && gctas == 0; ++rnd) {
        {
            TraceScope tr(kStPropose, s);
            launch_propose(w, rho, N, b, r, greedy, opts->seed, rnd, proposals, opts->tol * N, s);
        }
        {
            TraceScope tr(kStGather, s);
            if (tc) k_gather<<<(unsigned)((d + r + 7) / 8), 256, 0, s>>>(w, Xf, (const float*)Ff, ldf, d, b);
            else k_gather<<<(unsigned)((d + r + 7) / 8), 256, 0, s>>>(w, Xd, (const double*)Fd, ldf, d, b);
        }
        {
            TraceScope tr(kStBlockH, s);
            launch_blockH(w, d, b, inv_eps, s);
        }
        {
            TraceScope tr(kStReject, s);
            KEVD_CUDA_TRY(launch_reject(w, b, r, greedy, opts->seed, rnd, pivots, s));
        }
        if (tc) {
            TraceScope tr(kStEngine, s);
            KEVD_CUDA_TRY(launch_engine_tc(w, pw, Xf, Ff, ldf, rho, N, d, b, inv_eps, r, s));
        } else {
            if (oz) {
                {
                    // X X(S,:)^T and F(:, :k) F(S, :k)^T on the tensor cores at FP64 accuracy
                    TraceScope tp(kStProducts, s);
                    k_ozpanel<<<b, 128, 0, s>>>(w, ow, N, b);
                    KEVD_CUDA_TRY(launch_ozmm(oX, oPX, N, b, ow.ldX, w.st, w.Dx, w.ldD, 0, nullptr, 0, ow.flags, s));
                    KEVD_CUDA_TRY(launch_ozmm(oF, oPF, N, b, -3, w.st, w.Df, w.ldD, 0, nullptr, 0, ow.flags, s));
                }
                TraceScope tr(kStEngine, s);
                // R = K(:, T) - F F(T,:)^T; G = R L^-T into F(:, k:k+m), on the tensor cores; rho
                k_rprep<<<(unsigned)std::min<int64_t>((N + 31) / 32, 152 * 8), 2 * ow.ldR, 0, s>>>(
                    w, ow, N, kexp_scale(inv_eps), exp_tbl);
                KEVD_CUDA_TRY(launch_linv(w, ow, b, s));
                KEVD_CUDA_TRY(launch_ozmm(oR, oL, N, b, -2, w.st, Fd, ldf, ldf, ow.Fp, ow.ldF / 16, ow.flags, s));
                k_rho_update<<<(unsigned)((N + 63) / 64), 256, 0, s>>>(w, Fd, ldf, rho, N);
            } else {
                TraceScope tr(kStEngine, s);
                switch (tn) {
                    case 1: launch_engine<1>(w, Xd, Fd, ldf, rho, N, d, b, inv_eps, ntiles, s); break;
                    case 2: launch_engine<2>(w, Xd, Fd, ldf, rho, N, d, b, inv_eps, ntiles, s); break;
                    case 4: launch_engine<4>(w, Xd, Fd, ldf, rho, N, d, b, inv_eps, ntiles, s); break;
                    case 8: launch_engine<8>(w, Xd, Fd, ldf, rho, N, d, b, inv_eps, ntiles, s); break;
                    default: launch_engine<16>(w, Xd, Fd, ldf, rho, N, d, b, inv_eps, ntiles, s); break;
                }
            }
        }
        KEVD_LAUNCH_CHECK();
        if (opts->until_rank && (rnd % 8) == 7) {
            FactorState hs;
            KEVD_CUDA_TRY(cudaMemcpyAsync(&hs, w.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
            KEVD_CUDA_TRY(cudaStreamSynchronize(s));
            if (hs.done || hs.k + hs.m >= r) break;
        }
    }
    {
        TraceScope tr(kStOther, s);
        k_finalize<<<1, 1024, 0, s>>>(w, rho, N);
        const dim3 zg((unsigned)std::min<int64_t>((N + 255) / 256, 64), r);
        if (tc) k_zero_tail<<<zg, 256, 0, s>>>(w.st, Ff, ldf, N, r);
        else k_zero_tail<<<zg, 256, 0, s>>>(w.st, Fd, ldf, N, r);
    }
    KEVD_LAUNCH_CHECK();
    FactorState hs;
    int herr = 0;
    KEVD_CUDA_TRY(cudaMemcpyAsync(&hs, w.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
    if (tc) KEVD_CUDA_TRY(cudaMemcpyAsync(&herr, pw.err, sizeof(int), cudaMemcpyDeviceToHost, s));
    if (oz) KEVD_CUDA_TRY(cudaMemcpyAsync(&herr, ow.flags, sizeof(int), cudaMemcpyDeviceToHost, s));
    KEVD_CUDA_TRY(cudaStreamSynchronize(s));
    trace_flush();
    if (herr || hs.timeout) return KEVD_ETIMEOUT;
    info->rank = hs.k;
    info->rounds = hs.rounds;
    info->trace_err = hs.final_sum;
    info->sum_m_sq = hs.sum_m_sq;
    info->sum_k = hs.sum_k;
    info->engine_rounds = hs.eng_rounds;
    if (hs.bad) return KEVD_EINVAL;
    return KEVD_OK;
}

extern "C" int rpchol_factor(const void* X, int x_dtype, int64_t N, int32_t d, double eps, int32_t r,
                             const kevd_opts* opts, void* F, int f_dtype, int64_t ldf, int64_t* pivots,
                             double* rho, int64_t* proposals, kevd_factor_info* info, void* workspace,
                             size_t ws_bytes, void* stream) {
    return rpchol_factor_impl(X, x_dtype, N, d, eps, r, opts, F, f_dtype, ldf, pivots, rho, proposals, info, workspace,
                              ws_bytes, stream, true);
}

// ===========================================================================
// Batched form: many independent problems (uneven N, d, eps, r, b) advance
// through Algorithm 2 in lockstep.  Every launch covers all problems (one grid
// dimension is the problem); the kernel-column engine is one persistent launch
// that walks a work list of (problem, 64-row tile) items.  The round loop is
// captured once into a CUDA graph (kevd_batch_create) and replayed
// (kevd_batch_run).  FP64 path, ARPC.
// ===========================================================================
namespace kevd {

struct BatchProb {
    const double* X;
    double* F;
    int64_t ldf;
    double* rho;
    int64_t* pivots;
    int64_t N;
    int d, r, b, rounds;
    double inv_eps;
    uint64_t seed;
    int64_t ntiles;
    FactorWs w;
};

__global__ void k_prepare_b(const BatchProb* __restrict__ P) {
    const BatchProb& p = P[blockIdx.y];
    if ((int64_t)blockIdx.x * blockDim.x >= p.N && blockIdx.x != 0) return;
    prepare_body(p.X, p.N, p.d, p.w, p.rho, blockIdx.x);
}

__global__ void __cluster_dims__(kPropCluster, 1, 1) __launch_bounds__(kPropThreads)
    k_propose_b(const BatchProb* __restrict__ P, int rnd) {   // a cluster per problem
    const BatchProb& p = P[blockIdx.y];
    if (rnd >= p.rounds) {   // this problem has run its t = r/b rounds
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            commit_round(p.w.st);
            p.w.st->done = 1;
        }
        return;
    }
    propose_body(p.w, p.rho, p.N, p.ntiles, p.b, p.r, p.seed, rnd, nullptr, 0.0, blockIdx.x);
}

__global__ void k_gather_b(const BatchProb* __restrict__ P) {
    const BatchProb& p = P[blockIdx.y];
    gather_body(p.w, p.X, (const double*)p.F, p.ldf, p.d, p.b, blockIdx.x);
}

__global__ void k_blockH_b(const BatchProb* __restrict__ P) {
    const BatchProb& p = P[blockIdx.z];
    blockH_body(p.w, p.d, p.b, p.inv_eps, blockIdx.x);   // blocks past the last tile return
}

__global__ void __cluster_dims__(kRejCluster, 1, 1) __launch_bounds__(kRejThreads)
    k_reject_b(const BatchProb* __restrict__ P, int rnd) {   // a cluster per problem
    __shared__ RejShared sh;
    const BatchProb& p = P[blockIdx.y];
    arpc_reject_body(p.w, p.b, p.r, p.seed, rnd, p.pivots, sh, blockIdx.x);
}

// Persistent engine over the work list; tile_off[q] = first item of problem q.
template <int TN>
__global__ void __launch_bounds__(256) k_engine_b(const BatchProb* __restrict__ P, const int64_t* __restrict__ tile_off,
                                                  int nprob) {
    extern __shared__ double smem_eb[];
    const int64_t total = tile_off[nprob];
    for (int64_t item = blockIdx.x; item < total; item += gridDim.x) {
        int lo = 0, hi = nprob - 1;   // last q with tile_off[q] <= item
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tile_off[mid] <= item) lo = mid; else hi = mid - 1;
        }
        const BatchProb& p = P[lo];
        engine_body<TN>(p.w, p.X, p.F, p.ldf, p.rho, p.N, p.d, p.b, p.inv_eps, item - tile_off[lo], smem_eb);
    }
}

__global__ void __launch_bounds__(1024) k_finalize_b(const BatchProb* __restrict__ P) {
    const BatchProb& p = P[blockIdx.x];
    finalize_body(p.w, p.rho, p.N);
}

__global__ void k_zero_tail_b(const BatchProb* __restrict__ P) {
    const BatchProb& p = P[blockIdx.y];
    const int k = p.w.st->k;
    const int64_t cols = p.r - k;
    const int64_t total = cols * p.N;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
        p.F[(int64_t)(k + e / p.N) * p.ldf + e % p.N] = 0.0;
}

}  // namespace kevd

struct kevd_batch {
    int nprob;
    int rounds;
    int dmax, rmax, bmax;
    int64_t nmax;
    kevd::BatchProb* dprobs;   // device, in the caller's workspace (all problems)
    // engine groups by column-tile class TN (1, 2, 4, 8, 16): problems of a
    // group share one persistent engine launch per round
    struct Group {
        int tn;
        int n;
        kevd::BatchProb* probs;   // device copy of the group's descriptors
        int64_t* tile_off;        // device
    };
    std::vector<Group> groups;
    std::vector<kevd::FactorState*> states;
    cudaGraphExec_t exec;
    bool graph;
};

namespace {

static int tn_class(int b) { return b <= 8 ? 1 : b <= 16 ? 2 : b <= 32 ? 4 : b <= 64 ? 8 : 16; }

// layout: all descriptors | per group (<= 5): descriptors + tile offsets | per-problem factor workspaces
static size_t batch_layout(const kevd_problem* probs, int nprob, size_t* per_off) {
    using namespace kevd;
    size_t off = align_up(sizeof(BatchProb) * nprob);
    off += 5 * (align_up(sizeof(BatchProb) * nprob) + align_up(sizeof(int64_t) * (nprob + 1)));
    for (int q = 0; q < nprob; ++q) {
        size_t bytes = 0;
        carve_factor(nullptr, probs[q].N, probs[q].d, probs[q].r, probs[q].b, &bytes);
        if (per_off) per_off[q] = off;
        off += align_up(bytes);
    }
    return off;
}

template <int TN>
static int engine_group(const kevd_batch::Group& g, cudaStream_t s) {
    using namespace kevd;
    int nsm = 0, per_sm = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return KEVD_ECUDA;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return KEVD_ECUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_engine_b<TN>, 256, engine_smem<TN>()) != cudaSuccess)
        return KEVD_ECUDA;
    const unsigned egrid = (unsigned)std::max(1, nsm * std::max(1, per_sm));
    k_engine_b<TN><<<egrid, 256, engine_smem<TN>(), s>>>(g.probs, g.tile_off, g.n);
    return KEVD_OK;
}

static int batch_enqueue_any(kevd_batch* h, cudaStream_t s) {
    using namespace kevd;
    const int np = h->nprob;
    k_prepare_b<<<dim3((unsigned)((h->nmax + 255) / 256), np), 256, 0, s>>>(h->dprobs);
    for (int rnd = 0; rnd < h->rounds; ++rnd) {
        k_propose_b<<<dim3(kPropCluster, np), kPropThreads, 0, s>>>(h->dprobs, rnd);
        k_gather_b<<<dim3((unsigned)((h->dmax + h->rmax + 7) / 8), np), 256, 0, s>>>(h->dprobs);
        k_blockH_b<<<dim3(blockH_blocks(h->bmax), 1, np), kBlockHThreads, 0, s>>>(h->dprobs);
        k_reject_b<<<dim3(kRejCluster, np), kRejThreads, 0, s>>>(h->dprobs, rnd);
        for (const auto& g : h->groups) {
            int st;
            switch (g.tn) {
                case 1: st = engine_group<1>(g, s); break;
                case 2: st = engine_group<2>(g, s); break;
                case 4: st = engine_group<4>(g, s); break;
                case 8: st = engine_group<8>(g, s); break;
                default: st = engine_group<16>(g, s); break;
            }
            if (st != KEVD_OK) return st;
        }
    }
    k_finalize_b<<<np, 1024, 0, s>>>(h->dprobs);
    k_zero_tail_b<<<dim3(64, np), 256, 0, s>>>(h->dprobs);
    return cudaGetLastError() == cudaSuccess ? KEVD_OK : KEVD_ECUDA;
}

template <int TN>
static cudaError_t batch_attrs() {
    using namespace kevd;
    return cudaFuncSetAttribute(k_engine_b<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)engine_smem<TN>());
}

}  // namespace

extern "C" size_t kevd_batch_workspace_bytes(const kevd_problem* probs, int nprob) {
    if (!probs || nprob < 1) return 0;
    for (int q = 0; q < nprob; ++q)
        if (probs[q].N < 1 || probs[q].d < 1 || probs[q].r < 1 || probs[q].b < 1 || probs[q].b > 128) return 0;
    return batch_layout(probs, nprob, nullptr);
}

extern "C" int kevd_batch_create(const kevd_problem* probs, int nprob, int use_graph, void* workspace,
                                 size_t ws_bytes, void* stream, kevd_batch** out) {
    using namespace kevd;
    if (!probs || nprob < 1 || !out) return KEVD_EINVAL;
    *out = nullptr;
    int bmax = 1, dmax = 1, rmax = 1, rounds = 0;
    int64_t nmax = 1;
    for (int q = 0; q < nprob; ++q) {
        const kevd_problem& p = probs[q];
        if (!p.X || !p.F || !p.pivots || !p.rho) return KEVD_EINVAL;
        if (p.N < 1 || p.d < 1 || p.r < 1 || p.r > p.N || p.ldf < p.N || p.b < 1 || p.b > 128 || p.r / p.b < 1)
            return KEVD_EINVAL;
        if (!(p.eps > 0.0) || !isfinite(p.eps)) return KEVD_EINVAL;
        bmax = std::max(bmax, p.b);
        dmax = std::max(dmax, p.d);
        rmax = std::max(rmax, p.r);
        nmax = std::max(nmax, p.N);
        rounds = std::max(rounds, p.r / p.b);
    }
    std::vector<size_t> offs(nprob);
    const size_t need = batch_layout(probs, nprob, offs.data());
    if (!workspace || ws_bytes < need || (reinterpret_cast<uintptr_t>(workspace) % kAlign)) return KEVD_EWORKSPACE;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    char* base = static_cast<char*>(workspace);
    kevd_batch* h = new kevd_batch();
    h->nprob = nprob;
    h->rounds = rounds;
    h->bmax = bmax;
    h->dmax = dmax;
    h->rmax = rmax;
    h->nmax = nmax;
    h->dprobs = reinterpret_cast<BatchProb*>(base);
    h->graph = use_graph != 0;
    h->exec = nullptr;
    std::vector<BatchProb> hp(nprob);
    for (int q = 0; q < nprob; ++q) {
        const kevd_problem& p = probs[q];
        BatchProb& b = hp[q];
        b.X = p.X;
        b.F = p.F;
        b.ldf = p.ldf;
        b.rho = p.rho;
        b.pivots = p.pivots;
        b.N = p.N;
        b.d = p.d;
        b.r = p.r;
        b.b = p.b;
        b.rounds = p.r / p.b;
        b.inv_eps = 1.0 / p.eps;
        b.seed = p.seed;
        b.ntiles = (p.N + kBM - 1) / kBM;
        size_t bytes = 0;
        b.w = carve_factor(base + offs[q], p.N, p.d, p.r, p.b, &bytes);
        h->states.push_back(b.w.st);
    }
    cudaError_t e = cudaSuccess;
    bool ok = cudaMemcpyAsync(h->dprobs, hp.data(), sizeof(BatchProb) * nprob, cudaMemcpyHostToDevice, s) == cudaSuccess;
    // engine groups
    std::vector<std::vector<BatchProb>> gp(5);
    std::vector<std::vector<int64_t>> gt(5, std::vector<int64_t>(1, 0));
    const int classes[5] = {1, 2, 4, 8, 16};
    for (int q = 0; q < nprob; ++q) {
        const int c = tn_class(hp[q].b);
        const int gi = c == 1 ? 0 : c == 2 ? 1 : c == 4 ? 2 : c == 8 ? 3 : 4;
        gp[gi].push_back(hp[q]);
        gt[gi].push_back(gt[gi].back() + hp[q].ntiles);
    }
    size_t goff = align_up(sizeof(BatchProb) * nprob);
    for (int gi = 0; gi < 5 && ok; ++gi) {
        kevd_batch::Group g;
        g.tn = classes[gi];
        g.n = (int)gp[gi].size();
        g.probs = reinterpret_cast<BatchProb*>(base + goff);
        g.tile_off = reinterpret_cast<int64_t*>(base + goff + align_up(sizeof(BatchProb) * nprob));
        goff += align_up(sizeof(BatchProb) * nprob) + align_up(sizeof(int64_t) * (nprob + 1));
        if (g.n == 0) continue;
        switch (g.tn) {
            case 1: e = batch_attrs<1>(); break;
            case 2: e = batch_attrs<2>(); break;
            case 4: e = batch_attrs<4>(); break;
            case 8: e = batch_attrs<8>(); break;
            default: e = batch_attrs<16>(); break;
        }
        ok = e == cudaSuccess &&
             cudaMemcpyAsync(g.probs, gp[gi].data(), sizeof(BatchProb) * g.n, cudaMemcpyHostToDevice, s) ==
                 cudaSuccess &&
             cudaMemcpyAsync(g.tile_off, gt[gi].data(), sizeof(int64_t) * (g.n + 1), cudaMemcpyHostToDevice, s) ==
                 cudaSuccess;
        h->groups.push_back(g);
    }
    if (!ok || cudaStreamSynchronize(s) != cudaSuccess) {
        delete h;
        return KEVD_ECUDA;
    }
    if (h->graph) {
        cudaStream_t cs = nullptr;
        cudaGraph_t g = nullptr;
        int st = KEVD_ECUDA;
        if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) == cudaSuccess &&
            cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
            st = batch_enqueue_any(h, cs);
            if (cudaStreamEndCapture(cs, &g) != cudaSuccess) st = KEVD_ECUDA;
        }
        if (st == KEVD_OK && cudaGraphInstantiate(&h->exec, g, 0) != cudaSuccess) st = KEVD_ECUDA;
        if (g) cudaGraphDestroy(g);
        if (cs) cudaStreamDestroy(cs);
        if (st != KEVD_OK) {
            delete h;
            return st;
        }
    }
    *out = h;
    return KEVD_OK;
}

extern "C" int kevd_batch_run(kevd_batch* h, void* stream, kevd_factor_info* infos) {
    using namespace kevd;
    if (!h) return KEVD_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (h->graph) {
        TraceScope tr(kStOther, s);   // the whole batched round loop
        KEVD_CUDA_TRY(cudaGraphLaunch(h->exec, s));
    } else {
        TraceScope tr(kStOther, s);
        const int st = batch_enqueue_any(h, s);
        if (st != KEVD_OK) return st;
    }
    std::vector<FactorState> hs(h->nprob);
    for (int q = 0; q < h->nprob; ++q)
        KEVD_CUDA_TRY(cudaMemcpyAsync(&hs[q], h->states[q], sizeof(FactorState), cudaMemcpyDeviceToHost, s));
    KEVD_CUDA_TRY(cudaStreamSynchronize(s));
    trace_flush();
    int status = KEVD_OK;
    for (int q = 0; q < h->nprob; ++q) {
        if (infos) {
            infos[q].rank = hs[q].k;
            infos[q].rounds = hs[q].rounds;
            infos[q].trace_err = hs[q].final_sum;
            infos[q].sum_m_sq = hs[q].sum_m_sq;
            infos[q].sum_k = hs[q].sum_k;
            infos[q].engine_rounds = hs[q].eng_rounds;
            infos[q].reserved = 0;
        }
        if (hs[q].bad) status = KEVD_EINVAL;
    }
    return status;
}

extern "C" void kevd_batch_destroy(kevd_batch* h) {
    if (!h) return;
    if (h->exec) cudaGraphExecDestroy(h->exec);
    delete h;
}
