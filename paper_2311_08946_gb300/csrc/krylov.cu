// a13: the global solve C u = r (Eq. 28) in FP64 by restarted GMRES(m)
// (Sec. 4) on a CSR sparse matrix-vector product, plain or right-
// preconditioned (Eq. 45) by the RAS operator of ras.cu.
//
// Layout: the Krylov basis V is (m+1) x n row-major (each basis vector
// contiguous); dot products are block partial sums reduced in a fixed order
// (deterministic).  Orthogonalisation is classical Gram-Schmidt applied
// twice (CGS2).  The m Arnoldi iterations of a restart cycle run in one
// cooperative kernel of clusters (k_arnoldi_fused) that keeps each CTA's part
// of the basis in shared memory; the Hessenberg matrix, Givens
// rotations and the residual estimate live on the device, and the host
// synchronises once per restart cycle to read the true residual.
#include <cstdlib>
#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "handles.cuh"

namespace pdd {

static constexpr int kRowsPerBlock = 32;    // 8 lanes per row, 256 threads
static constexpr int kDotBlock = 256;

struct GState {
    int stop, iters, k_used, err;
    double bnorm, res;
    double rr;                  // |b - C u|^2 of the cycle's end
};

// y = C x, or y = b - C x with b given; 8 lanes per row
__global__ void __launch_bounds__(256) k_spmv(int n, const int *rowptr, const int *col, const double *val,
                                              const double *x, double *y, const double *b) {
    const int row = blockIdx.x * kRowsPerBlock + (threadIdx.x >> 3), l = threadIdx.x & 7;
    double s = 0.0;
    if (row < n)
        for (int k = rowptr[row] + l; k < rowptr[row + 1]; k += 8) s += val[k] * x[col[k]];
    s += __shfl_xor_sync(0xffffffffu, s, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    if (row < n && l == 0) y[row] = b ? b[row] - s : s;
}

// partial[t * G + bx] = sum over the rows of block column bx of V[t] . w.  The grid is
// (row chunks G) x (groups of eight vectors); each thread takes rows of its chunk for the eight
// vectors of its group (independent loads).  The last block of a vector group to finish adds the
// group's partials in block order into hsum[t] (deterministic) and re-arms the group's counter.
static constexpr int kMaxDots = 257;
static constexpr int kDotThreads = 128, kDotVec = 8;
static constexpr int kDotGroups = (kMaxDots + kDotVec - 1) / kDotVec;
__global__ void __launch_bounds__(kDotThreads) k_dots(int n, int nv, const double *V, const double *w,
                                                      double *partial, double *hsum, unsigned *cnt,
                                                      const GState *gs) {
    if (gs && gs->stop) return;
    __shared__ double red[kDotThreads / 32][kDotVec];
    __shared__ bool last;
    const int G = gridDim.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t0 = blockIdx.y * kDotVec, nq = min(kDotVec, nv - t0);
    const int per = (n + G - 1) / G, a = blockIdx.x * per, b = min(n, a + per);
    double s[kDotVec];
#pragma unroll
    for (int q = 0; q < kDotVec; ++q) s[q] = 0.0;
    const double *v0 = V + (long)t0 * n;
    for (int r = a + threadIdx.x; r < b; r += kDotThreads) {
        const double wr = w[r];
#pragma unroll
        for (int q = 0; q < kDotVec; ++q)
            if (q < nq) s[q] += v0[(long)q * n + r] * wr;
    }
#pragma unroll
    for (int q = 0; q < kDotVec; ++q) {
        double v = s[q];
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[warp][q] = v;
    }
    __syncthreads();
    if (threadIdx.x < nq) {
        double v = 0.0;
        for (int q = 0; q < kDotThreads / 32; ++q) v += red[q][threadIdx.x];
        partial[(long)(t0 + threadIdx.x) * G + blockIdx.x] = v;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = (atomicAdd(cnt + blockIdx.y, 1u) == (unsigned)G - 1);
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int q = warp; q < nq; q += kDotThreads / 32) {
        const double *pp = partial + (long)(t0 + q) * G;
        double v = 0.0;
#pragma unroll 4
        for (int i = lane; i < G; i += 32) v += __ldcg(pp + i);
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) hsum[t0 + q] = v;
    }
    if (threadIdx.x == 0) cnt[blockIdx.y] = 0u;
}

// v = w / |w| with |w|^2 = hsum[0]; Hsub = |w|
__global__ void __launch_bounds__(kDotBlock) k_normalize(int n, const double *w, double *v, const double *hsum,
                                                         double *Hsub, const GState *gs) {
    if (gs && gs->stop) return;
    const double nrm = sqrt(hsum[0]);
    if (blockIdx.x == 0 && threadIdx.x == 0 && Hsub) *Hsub = nrm;
    const double inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) v[r] = w[r] * inv;
}

// y = H^-1 g (upper triangular k x k), column by column: one warp holds the right-hand side, 32 columns
// of H at a time staged in shared memory.  One thread walking rows of H in global memory took 45-100 us
// a cycle (13-25 us).
static constexpr int kUpperThreads = 256, kUpperCols = 32;
static constexpr int kUpperSlices = (kMaxDots - 1 + 31) / 32;
__global__ void __launch_bounds__(kUpperThreads) k_upper_solve(const double *H, int ldh, const double *g, double *y,
                                                               const GState *gs) {
    extern __shared__ double hs[];                        // [kUpperCols][k]
    const int k = gs->k_used, lane = threadIdx.x & 31;
    double s[kUpperSlices];
#pragma unroll
    for (int q = 0; q < kUpperSlices; ++q) s[q] = (lane + 32 * q < k) ? g[lane + 32 * q] : 0.0;
    for (int c0 = ((k - 1) / kUpperCols) * kUpperCols; k > 0 && c0 >= 0; c0 -= kUpperCols) {
        const int nc = min(kUpperCols, k - c0);
        __syncthreads();
        for (int e = threadIdx.x; e < nc * k; e += kUpperThreads) {
            const int c = e / k, r = e - c * k;
            if (r <= c0 + c) hs[e] = H[(long)(c0 + c) * ldh + r];
        }
        __syncthreads();
        if (threadIdx.x >= 32) continue;
        const double inv = lane < nc ? 1.0 / hs[lane * k + c0 + lane] : 0.0;      // of the tile's diagonal
        const int qc = c0 >> 5;                                                   // c0 is a multiple of 32
        for (int c = nc - 1; c >= 0; --c) {
            double sq = 0.0;
#pragma unroll
            for (int q = 0; q < kUpperSlices; ++q)
                if (q == qc) sq = s[q];
            const double v = __shfl_sync(0xffffffffu, sq * inv, c);
            if (lane == 0) y[c0 + c] = v;
#pragma unroll
            for (int q = 0; q < kUpperSlices; ++q) {
                const int r = lane + 32 * q;
                if (r < c0 + c) s[q] -= hs[c * k + r] * v;
            }
        }
    }
}

__global__ void k_xupdate(int n, const double *V, const double *y, const GState *gs, double *x) {
    const int k = gs->k_used;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        double s = x[r];
        for (int t = 0; t < k; ++t) s += V[(long)t * n + r] * y[t];
        x[r] = s;
    }
}

__global__ void k_cycle_start(GState *gs, const double *hsum, double *g, int m, double rtol, int max_iters,
                              int first) {
    if (threadIdx.x != 0) return;
    const double beta = sqrt(hsum[0]);
    if (first) gs->bnorm = beta;                      // x0 = 0, so r0 = b
    for (int i = 0; i <= m; ++i) g[i] = 0.0;
    g[0] = beta;
    gs->res = beta;
    gs->k_used = 0;
    gs->stop = (beta <= rtol * gs->bnorm || gs->iters >= max_iters || beta == 0.0) ? 1 : 0;
}

void spmv_csr(int n, const int *rowptr, const int *col, const double *val, const double *x, double *y,
              cudaStream_t st) {
    PDD_LAUNCH(k_spmv, cdiv(n, kRowsPerBlock), 256, 0, st, n, rowptr, col, val, x, y, (const double *)nullptr);
}

// ---------------------------------------------------------------------------
// One restart cycle's Arnoldi iterations in a single cooperative launch of clusters of CTAs.
// Each CTA owns `per` rows: it computes w = C v_j on them, keeps w and (as far as shared memory goes:
// 64 vectors of 400 rows) its part of the basis in shared memory, and takes part in two passes of
// classical Gram-Schmidt.  Dot products are added over a CTA's warps, then over the cluster through
// distributed shared memory, then over the clusters through global memory, always in the same order
// (deterministic).  |w| after the second pass comes from that pass: |w1|^2 - |h2|^2, w1 being almost
// orthogonal already (else it is summed again).  Every CTA keeps the rotations and decides on stopping
// by itself from the same sums, so an iteration has three grid-wide barriers.
// Why: four barriers, basis slices read from L2 by latency-bound loops, 152 partial sums per vector
// read by every CTA and a serial rotation on the critical path cost 22 us an iteration at n = 204 and
// 52 us at n = 32,768; what is left is the FP64 pipe (4 n j products an iteration) and the barriers: 13 and 35 us.
// With RAS (Eq. 44-45) z_j = M^-1 v_j comes first (two more barriers), one warp per subset.
// ---------------------------------------------------------------------------
static constexpr int kFusedThreads = 512, kFusedWarps = kFusedThreads / 32;
static constexpr int kClusterMax = 8, kClusterMany = 4;     // CTAs of a lone cluster, of each of several
static constexpr int kRowsPerCta = 64;                  // fewer clusters than the device holds below this
static constexpr size_t kFusedSmem = 222 * 1024;
static constexpr long long kBarrierLimit = 1LL << 22;   // polls (an L2 read each, ~0.2 us) before giving up

struct FusedArnoldi {
    int n, m;
    const int *rowptr, *col;
    const double *val;
    double *V, *part;            // part: 3 x kMaxDots x clusters partial sums
    double *w;                   // w in global memory when a CTA's rows do not fit in shared memory, else null
    double *H, *g;               // H column-major (ldh = m + 1)
    GState *gs;
    unsigned *bar;               // [0] arrivals, [1] generation
    double rtol;
    int max_iters;
    int per, ld, ks;             // rows of a CTA, their padded count, basis vectors kept in shared memory
    unsigned bar_extra;          // arrivals a barrier waits for beyond the clusters (0; 1 = never completes)
    long long bar_limit;         // polls before a barrier wait gives up
    // right preconditioner (Eq. 44-45); ras_P = 0: none
    int ras_P, ras_NP;
    const int *ras_wptr, *ras_widx, *ras_p1, *ras_l1, *ras_p2, *ras_l2;
    const float *ras_cinvT;
    float *ras_z;
    double *ras_Z;               // z_j = M^-1 v_j of the cycle, m x n (flexible GMRES)
};

// doubles of shared memory besides the basis: w, h, column, rotations, g, sums of the warps' row
// chunks and of the CTA (twice), the update's parts; the RAS right-hand sides share the latter two
__host__ __device__ constexpr size_t fused_fixed_doubles(int m, int ld) {
    return (size_t)ld + 5 * (size_t)(m + 2) + (size_t)kFusedWarps * 8 + (size_t)kFusedWarps * 8 + 2 * (size_t)(m + 2) +
           kFusedThreads + kFusedWarps * 64;
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// the double at p of this CTA's shared memory, in CTA `rank` of the cluster
__device__ __forceinline__ double remote_load(const double *p, unsigned rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    double v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r));
    return v;
}
__device__ __forceinline__ int remote_load(const int *p, unsigned rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    int v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(r) : "memory");
    return v;
}

// Grid-wide barrier, bounded.  The first cluster barrier orders the cluster's writes before thread 0
// of its first CTA, which alone arrives and polls (and gives up after bar_limit polls); the second one
// releases the cluster, all of whose CTAs read the outcome from the first, so they leave together (after
// one more cluster barrier: the first CTA's shared memory must outlive the others' reads).
// `meanwhile` runs between the arrival and the wait (one warp's scalar work).
template <typename Work>
__device__ __forceinline__ bool grid_barrier(const FusedArnoldi &F, unsigned nclusters, unsigned rank, int *s_bad,
                                             Work meanwhile) {
    cluster_arrive();
    meanwhile();
    cluster_wait();
    if (nclusters == 1 && F.bar_extra == 0) return true;
    if (rank == 0 && threadIdx.x == 0) {
        volatile unsigned *gen = F.bar + 1;
        const unsigned g0 = *gen;
        __threadfence();
        if (atomicAdd(F.bar, 1u) == nclusters - 1 + F.bar_extra) {
            atomicExch(F.bar, 0u);
            __threadfence();
            atomicAdd(F.bar + 1, 1u);
        } else {
            long long it = 0;
            while (*gen == g0) {
                if (++it > F.bar_limit) {
                    atomicExch(&F.gs->err, 1);
                    break;
                }
            }
        }
        __threadfence();
        *s_bad = *(volatile int *)&F.gs->err;
    }
    cluster_barrier();
    return remote_load(s_bad, 0) == 0;
}
__device__ __forceinline__ bool grid_barrier(const FusedArnoldi &F, unsigned nclusters, unsigned rank, int *s_bad) {
    return grid_barrier(F, nclusters, rank, s_bad, [] {});
}

__device__ __forceinline__ double warp_sum(double s) {
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// z_p = C_p^-1 (R_p v) of one subset by one warp: lane owns rows lane + 32 i (i < RR)
template <int RR>
__device__ __forceinline__ void ras_subset(const FusedArnoldi &F, int p, const double *vj, float *vs, int lane) {
    const int NP = F.ras_NP, wb = F.ras_wptr[p], np = F.ras_wptr[p + 1] - wb;
    for (int q = lane; q < NP; q += 32) vs[q] = q < np ? (float)__ldcg(vj + F.ras_widx[wb + q]) : 0.f;
    __syncwarp();
    const float *ci = F.ras_cinvT + (long)p * NP * NP + lane;
    float s[RR];
#pragma unroll
    for (int i = 0; i < RR; ++i) s[i] = 0.f;
    for (int q0 = 0; q0 < np; q0 += 16) {
        float c[16][RR];
#pragma unroll
        for (int u = 0; u < 16; ++u)
#pragma unroll
            for (int i = 0; i < RR; ++i)
                c[u][i] = (q0 + u < np && lane + 32 * i < NP) ? ci[(long)(q0 + u) * NP + 32 * i] : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const float v = vs[q0 + u < 128 ? q0 + u : 0];
#pragma unroll
            for (int i = 0; i < RR; ++i) s[i] = fmaf(c[u][i], v, s[i]);
        }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < RR; ++i)
        if (lane + 32 * i < NP) F.ras_z[(long)p * NP + lane + 32 * i] = s[i];
}

extern __shared__ __align__(16) double asm_[];            // the basis [ks][ld], w [ld], the small arrays

// loc[t] = sum over the CTA's rows of V_t . w for t <= j, loc[j + 1] = w . w when `norm` (j = -1 with
// norm: w . w alone in loc[0]).  Warps take units of eight vectors x a chunk of rows; in a warp, eight
// lanes name the vector and four row phases (the padded row count keeps them on different banks).
// SM: every vector is in shared memory (addressed as such; the general form loads through generic
// pointers).
template <bool SM>
__device__ __forceinline__ void local_dots_t(const FusedArnoldi &F, const double *ws, int rows, int r0, int j, bool norm,
                                             double *chunk, double *loc, int warp, int lane) {
    const int nv = j + 1 + (norm ? 1 : 0), ng = (nv + 7) >> 3;
    const int C = max(1, kFusedWarps / ng), rc = (rows + C - 1) / C, wo = F.ks * F.ld;
    for (int u = warp; u < ng * C; u += kFusedWarps) {
        const int g = u / C, c = u - g * C, t = 8 * g + (lane & 7);
        const int ra = c * rc + (lane >> 3), rb = min(rows, (c + 1) * rc);
        double s0 = 0.0, s1 = 0.0;
        if (SM) {
            const int vo = t > j ? wo : t * F.ld;
            if (t < nv) {
                int r = ra;
                for (; r + 4 < rb; r += 8) {
                    s0 += asm_[vo + r] * asm_[wo + r];
                    s1 += asm_[vo + r + 4] * asm_[wo + r + 4];
                }
                if (r < rb) s0 += asm_[vo + r] * asm_[wo + r];
            }
        } else {
            const double *v = t > j ? ws : (t < F.ks ? asm_ + (size_t)t * F.ld : F.V + (long)t * F.n + r0);
            if (t < nv) {
                int r = ra;
                for (; r + 4 < rb; r += 8) {
                    s0 += v[r] * ws[r];
                    s1 += v[r + 4] * ws[r + 4];
                }
                if (r < rb) s0 += v[r] * ws[r];
            }
        }
        s0 += s1;
        s0 += __shfl_xor_sync(0xffffffffu, s0, 8);
        s0 += __shfl_xor_sync(0xffffffffu, s0, 16);
        if (lane < 8) {
            if (C > 1) chunk[u * 8 + lane] = s0;
            else if (t < nv) loc[t] = s0;
        }
    }
    __syncthreads();
    if (C > 1) {
        for (int t = threadIdx.x; t < nv; t += kFusedThreads) {
            double a = 0.0, b = 0.0;                     // two chains over the chunks
            for (int c = 0; c < C; c += 2) {
                a += chunk[((t >> 3) * C + c) * 8 + (t & 7)];
                if (c + 1 < C) b += chunk[((t >> 3) * C + c + 1) * 8 + (t & 7)];
            }
            loc[t] = a + b;
        }
        __syncthreads();
    }
}
__device__ __forceinline__ void local_dots(const FusedArnoldi &F, const double *ws, int rows, int r0, int j, bool norm,
                                           double *chunk, double *loc, int warp, int lane) {
    if (j < F.ks && F.ks > 0) local_dots_t<true>(F, ws, rows, r0, j, norm, chunk, loc, warp, lane);
    else local_dots_t<false>(F, ws, rows, r0, j, norm, chunk, loc, warp, lane);
}

// the sum over the cluster's CTAs of loc[t]
__device__ __forceinline__ double cluster_sum(const double *loc, int t, unsigned csize) {
    double v[kClusterMax];
#pragma unroll
    for (unsigned q = 0; q < kClusterMax; ++q) v[q] = q < csize ? remote_load(loc + t, q) : 0.0;
    return ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
}

// out[t] = the sums of every CTA's loc[t], t < nv; `pp` this reduction's partial sums in global memory
__device__ __forceinline__ bool grid_sum(const FusedArnoldi &F, int nv, const double *loc, double *pp, double *out,
                                         unsigned ncl, unsigned cid, unsigned rank, unsigned csize, int *s_bad) {
    const int tid = threadIdx.x;
    cluster_barrier();                                   // every CTA of the cluster has its loc
    if (ncl == 1) {
        for (int t = tid; t < nv; t += kFusedThreads) out[t] = cluster_sum(loc, t, csize);
        __syncthreads();
        return F.bar_extra ? grid_barrier(F, ncl, rank, s_bad) : true;
    }
    for (int t = rank + tid * csize; t < nv; t += kFusedThreads * csize) pp[(long)t * ncl + cid] = cluster_sum(loc, t, csize);
    if (!grid_barrier(F, ncl, rank, s_bad)) return false;
    // eight lanes per sum
    for (int t0 = 0; t0 < nv; t0 += kFusedThreads / 8) {
        const int t = t0 + (tid >> 3);
        if (t0 + ((tid & ~31) >> 3) >= nv) break;        // none of the warp's four sums
        double s = 0.0;
        if (t < nv)
            for (unsigned c = tid & 7; c < ncl; c += 8) s += __ldcg(pp + (long)t * ncl + c);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if (t < nv && (tid & 7) == 0) out[t] = s;
    }
    __syncthreads();
    return true;
}

// w - sum_{t <= j} h_t V_t on the CTA's rows, each handed to put(row, value); the vectors of a row are
// spread over the warps when the rows are few.  `before` runs in the last warp first (scalar FP64 work
// in the other warps' shadow); a block barrier orders it before the put calls.
template <bool SM, typename Put, typename Work>
__device__ __forceinline__ void subtract_basis_t(const FusedArnoldi &F, const double *ws, int rows, int r0, int j,
                                                 const double *h, double *parts, Work before, Put put) {
    const int rw = max(1, (rows + 31) >> 5), np = max(1, kFusedWarps / rw), width = rw * 32;
    auto vec = [&](int t, int r) -> double {
        if (SM) return asm_[t * F.ld + r];
        return t < F.ks ? asm_[(size_t)t * F.ld + r] : F.V[(long)t * F.n + r0 + r];
    };
    if (threadIdx.x >= kFusedThreads - 32) before();
    if (np == 1) {
        __syncthreads();
        for (int r = threadIdx.x; r < rows; r += kFusedThreads) {
            double a0 = 0.0, a1 = 0.0;
            int t = 0;
            for (; t + 1 <= j; t += 2) {
                a0 += vec(t, r) * h[t];
                a1 += vec(t + 1, r) * h[t + 1];
            }
            if (t <= j) a0 += vec(t, r) * h[t];
            put(r, ws[r] - (a0 + a1));
        }
        __syncthreads();
        return;
    }
    const int part = threadIdx.x / width, r = threadIdx.x - part * width;
    if (part < np && r < rows) {
        double a0 = 0.0, a1 = 0.0;
        int t = part;
        for (; t + np <= j; t += 2 * np) {
            a0 += vec(t, r) * h[t];
            a1 += vec(t + np, r) * h[t + np];
        }
        if (t <= j) a0 += vec(t, r) * h[t];
        parts[part * width + r] = a0 + a1;
    }
    __syncthreads();
    if (threadIdx.x < rows) {
        double a = 0.0, b = 0.0;
        for (int p = 0; p < np; p += 2) {
            a += parts[p * width + threadIdx.x];
            if (p + 1 < np) b += parts[(p + 1) * width + threadIdx.x];
        }
        put((int)threadIdx.x, ws[threadIdx.x] - (a + b));
    }
    __syncthreads();
}
template <typename Put, typename Work>
__device__ __forceinline__ void subtract_basis(const FusedArnoldi &F, const double *ws, int rows, int r0, int j,
                                               const double *h, double *parts, Work before, Put put) {
    if (j < F.ks) subtract_basis_t<true>(F, ws, rows, r0, j, h, parts, before, put);
    else subtract_basis_t<false>(F, ws, rows, r0, j, h, parts, before, put);
}

__global__ void __launch_bounds__(kFusedThreads, 1) k_arnoldi_fused(FusedArnoldi F) {
    __shared__ int s_bad, s_stop;
    __shared__ double s_w2, s_inv;
    const int n = F.n, m = F.m, ldh = m + 1, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double *Vs = asm_;                                    // [ks][ld]
    double *ws_s = Vs + (size_t)F.ks * F.ld;              // [ld]
    double *h = ws_s + (F.w ? 0 : F.ld);                               // m + 2 each: this pass's sums, the column, rotations, g
    double *hcol = h + m + 2, *cs = hcol + m + 2, *sn = cs + m + 2, *gv = sn + m + 2;
    double *chunk = gv + m + 2;                           // [2 warps][8]
    double *loc0 = chunk + 2 * kFusedWarps * 8, *loc1 = loc0 + m + 2;
    double *parts = loc1 + m + 2;                         // [threads], then the RAS right-hand sides
    float *vs = reinterpret_cast<float *>(parts + kFusedThreads) + warp * 128;
    const unsigned rank = cluster_rank(), csize = cluster_size();
    const unsigned cid = blockIdx.x / csize, ncl = gridDim.x / csize;
    const int r0 = min(n, (int)blockIdx.x * F.per), rows = min(n, r0 + F.per) - r0;
    double *ws = F.w ? F.w + r0 : ws_s;
    const int iters0 = F.gs->iters;                       // written again only after the first grid-wide barrier
    const double bnorm = F.gs->bnorm;
    for (int i = tid; i <= m; i += kFusedThreads) gv[i] = F.g[i];
    for (int r = tid; r < rows; r += kFusedThreads)
        if (F.ks > 0) Vs[r] = F.V[r0 + r];
    if (tid == 0) s_stop = F.gs->stop;
    __syncthreads();
    bool done = s_stop != 0;
    for (int j = 0; j < m && !done; ++j) {
        const double *vj = F.V + (long)j * n;
        if (F.ras_P) {
            // z_j is kept: the cycle ends with u += Z y (the flexible form, exact for the products actually
            // taken, which the FP32 local solves make only nearly linear in v)
            const int nwarps = (int)gridDim.x * kFusedWarps, rr = (F.ras_NP + 31) >> 5;
            for (int p = (int)blockIdx.x + (int)gridDim.x * warp; p < F.ras_P; p += nwarps) {
                if (rr == 1) ras_subset<1>(F, p, vj, vs, lane);
                else if (rr == 2) ras_subset<2>(F, p, vj, vs, lane);
                else ras_subset<4>(F, p, vj, vs, lane);
            }
            if (!grid_barrier(F, ncl, rank, &s_bad)) break;
            double *zj = F.ras_Z + (long)j * n;
            for (int r = r0 + tid; r < r0 + rows; r += kFusedThreads) {
                const int q2 = F.ras_p2[r];
                const double a = (double)__ldcg(F.ras_z + (long)F.ras_p1[r] * F.ras_NP + F.ras_l1[r]);
                zj[r] = q2 >= 0 ? 0.5 * (a + (double)__ldcg(F.ras_z + (long)q2 * F.ras_NP + F.ras_l2[r])) : a;
            }
            if (!grid_barrier(F, ncl, rank, &s_bad)) break;
            vj = zj;
        }
        // w = C v_j: four lanes per row (each FP64 instruction of a warp takes the SM's unit 16 cycles, so
        // few shuffled additions and no empty rows), two rows of a lane group and 20 of their entries in
        // flight
        constexpr int U = 2, E = 5, RG = kFusedThreads / 4;
        for (int base = 0; base < rows; base += RG * U) {
            const int l = lane & 3;
            int ka[U], kb[U], c[U][E];
            double a[U][E], s[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int r = base + u * RG + (tid >> 2);
                ka[u] = kb[u] = 0;
                if (r < rows) {
                    ka[u] = F.rowptr[r0 + r] + l;
                    kb[u] = F.rowptr[r0 + r + 1];
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int k = ka[u] + 4 * e;
                    c[u][e] = k < kb[u] ? F.col[k] : -1;
                    a[u][e] = k < kb[u] ? F.val[k] : 0.0;
                }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (base + u * RG + 8 * warp >= rows) break;          // none of the warp's eight rows
                s[u] = 0.0;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (c[u][e] >= 0) s[u] += a[u][e] * __ldcg(vj + c[u][e]);
                for (int k0 = ka[u] + 4 * E; k0 < kb[u]; k0 += 32) {
                    int c2[8];
                    double a2[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int k = k0 + 4 * e;
                        c2[e] = k < kb[u] ? F.col[k] : -1;
                        a2[e] = k < kb[u] ? F.val[k] : 0.0;
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (c2[e] >= 0) s[u] += a2[e] * __ldcg(vj + c2[e]);
                }
                __syncwarp();
                s[u] += __shfl_xor_sync(0xffffffffu, s[u], 2);
                s[u] += __shfl_xor_sync(0xffffffffu, s[u], 1);
                const int r = base + u * RG + (tid >> 2);
                if (r < rows && l == 0) ws[r] = s[u];
            }
        }
        __syncthreads();
        // two passes of classical Gram-Schmidt against v_0 .. v_j, the second with |w|^2
        local_dots(F, ws, rows, r0, j, false, chunk, loc0, warp, lane);
        if (!grid_sum(F, j + 1, loc0, F.part, h, ncl, cid, rank, csize, &s_bad)) break;
        for (int t = tid; t <= j; t += kFusedThreads) hcol[t] = h[t];
        subtract_basis(F, ws, rows, r0, j, h, parts, [] {}, [&](int r, double v) { ws[r] = v; });
        local_dots(F, ws, rows, r0, j, true, chunk, loc1, warp, lane);
        if (!grid_sum(F, j + 2, loc1, F.part + (long)kMaxDots * ncl, h, ncl, cid, rank, csize, &s_bad)) break;
        // |w|^2 = |w1|^2 - |h2|^2 and its root's inverse, by the last warp while the others subtract; v_{j+1}
        double *vn = F.V + (long)(j + 1) * n + r0;
        subtract_basis(
            F, ws, rows, r0, j, h, parts,
            [&] {
                double h2 = 0.0;
                for (int t = lane; t <= j; t += 32) h2 += h[t] * h[t];
                h2 = warp_sum(h2);
                if (lane == 0) {
                    const double w2 = h[j + 1] - h2;
                    s_w2 = w2;
                    s_inv = w2 > 0.5 * h[j + 1] ? 1.0 / sqrt(w2) : -1.0;      // -1: the second pass took much away
                }
            },
            [&](int r, double v) {
                const double inv = s_inv;
                if (inv < 0.0) {
                    ws[r] = v;
                } else {
                    v *= inv;
                    vn[r] = v;
                    if (j + 1 < F.ks) Vs[(size_t)(j + 1) * F.ld + r] = v;
                }
            });
        for (int t = tid; t <= j; t += kFusedThreads) hcol[t] += h[t];
        if (s_inv < 0.0) {                                // sum |w|^2 itself
            local_dots(F, ws, rows, r0, -1, true, chunk, loc0, warp, lane);
            if (!grid_sum(F, 1, loc0, F.part + 2L * kMaxDots * ncl, h, ncl, cid, rank, csize, &s_bad)) break;
            if (tid == 0) {
                s_w2 = h[0];
                s_inv = h[0] > 0.0 ? 1.0 / sqrt(h[0]) : 0.0;
            }
            __syncthreads();
            for (int r = tid; r < rows; r += kFusedThreads) {
                const double v = ws[r] * s_inv;
                vn[r] = v;
                if (j + 1 < F.ks) Vs[(size_t)(j + 1) * F.ld + r] = v;
            }
        }
        __syncthreads();
        // Givens, in the shadow of the barrier that completes v_{j+1}: the previous rotations on column j, a
        // new one, g and the stop flag.  One lane walks the chain hi_{i+1} = c_i h_{i+1} - s_i hi_i (the
        // products c_i h_{i+1} made by the others), then the lanes form the rotated entries.
        auto givens = [&] {
            if (warp != kFusedWarps - 1) return;
            const double nrm = sqrt(s_w2);
            double hi = hcol[0];
            for (int i0 = 0; i0 < j; i0 += 32) {
                const int i = i0 + lane;
                const double hn = i < j ? hcol[i + 1] : 0.0, ci = i < j ? cs[i] : 0.0, si = i < j ? sn[i] : 0.0;
                const double p = ci * hn;
                double mine = 0.0;
                const int cnt = min(32, j - i0);
                for (int q = 0; q < cnt; ++q) {
                    if (lane == q) mine = hi;
                    hi = fma(-__shfl_sync(0xffffffffu, si, q), hi, __shfl_sync(0xffffffffu, p, q));
                }
                __syncwarp();
                if (i < j) hcol[i] = ci * mine + si * hn;
            }
            if (lane == 0) {
                const double top = fmax(fabs(hi), nrm);
                const double den = top > 1e-140 && top < 1e140 ? sqrt(hi * hi + nrm * nrm) : hypot(hi, nrm);
                const double rd = 1.0 / den;
                const double c = den > 0.0 ? hi * rd : 1.0, sv = den > 0.0 ? nrm * rd : 0.0;
                cs[j] = c;
                sn[j] = sv;
                hcol[j] = den;
                hcol[j + 1] = 0.0;
                gv[j + 1] = -sv * gv[j];
                gv[j] = c * gv[j];
                const double res = fabs(gv[j + 1]);
                const int iters = iters0 + j + 1;
                s_stop = res <= F.rtol * bnorm || iters >= F.max_iters || nrm == 0.0;
                if (blockIdx.x == 0) {
                    F.gs->iters = iters;
                    F.gs->k_used = j + 1;
                    F.gs->res = res;
                    if (s_stop) F.gs->stop = 1;
                }
            }
            __syncwarp();
        };
        if (!grid_barrier(F, ncl, rank, &s_bad, givens)) break;       // v_{j+1} is complete
        __syncthreads();
        done = s_stop != 0;
        if (blockIdx.x == 0) {
            double *Hc = F.H + (long)j * ldh;
            for (int i = tid; i <= j + 1; i += kFusedThreads) Hc[i] = hcol[i];
            for (int i = tid; i <= j + 1; i += kFusedThreads) F.g[i] = gv[i];
        }
    }
    cluster_barrier();                                    // no CTA ends while another reads its shared memory
}

// buffers of one GMRES(m) solve; gmres_csr allocates them, the allocation-free entry point carves
// them from its fixed array
struct GmresBufs {
    double *V, *w, *partial, *H, *g, *y, *fpart;
    unsigned *cnt, *bar;
    GState *gs;
};

// clusters of the fused Arnoldi kernel that fit on the current device at once (asked once per device:
// devices may differ)
static int device_clusters() {
    static constexpr int kDevs = 64;
    static int clusters_of[kDevs] = {0};
    static std::mutex mu;
    int dev = 0;
    PDD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kDevs) fail(PDD_EINVAL, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(mu);
    if (!clusters_of[dev]) {
        PDD_CUDA(cudaFuncSetAttribute(k_arnoldi_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmem));
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kClusterMany;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kClusterMany * 64);
        cfg.blockDim = dim3(kFusedThreads);
        cfg.dynamicSmemBytes = kFusedSmem;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int nc = 0;
        PDD_CUDA(cudaOccupancyMaxActiveClusters(&nc, k_arnoldi_fused, &cfg));
        if (nc < 1) fail(PDD_ECUDA, "the fused Arnoldi kernel does not fit on the device");
        clusters_of[dev] = nc;
    }
    return clusters_of[dev];
}

// the launch shape of one solve: clusters, CTAs of a cluster, rows of a CTA.  One cluster (no grid-wide
// barrier) up to 1,024 rows, where the FP64 work of 128 rows a CTA is below a barrier's 2 us; beyond
// that as many clusters as give each CTA 64 rows, or the device has: clusters of four, which fill its
// SMs (clusters of eight fit 15 times, on 120 of 152).
struct FusedShape {
    int clusters, csize, per, ld, ks;
    bool w_global;               // more rows a CTA than shared memory holds (above 3.9 million in all)
    size_t smem;
};
static FusedShape fused_shape(int n, int m) {
    FusedShape S{};
    S.clusters = n <= 1024 ? 1 : std::min(device_clusters(), cdiv(n, kClusterMany * kRowsPerCta));
    S.csize = S.clusters == 1 ? kClusterMax : kClusterMany;
    while (S.clusters == 1 && S.csize > 1 && (S.csize / 2) * 32 >= n) S.csize /= 2;
    if (S.clusters == 1) device_clusters();                     // (the shared-memory attribute)
    S.per = cdiv(n, S.clusters * S.csize);
    S.ld = (S.per + 13) / 16 * 16 + 2;                          // 2 mod 16 and >= per: the dots' bank rule
    size_t fixed = fused_fixed_doubles(m, S.ld) * sizeof(double);
    S.w_global = fixed > kFusedSmem;
    if (S.w_global) {
        fixed = fused_fixed_doubles(m, 0) * sizeof(double);
        S.ks = 0;
        S.smem = fixed;
        return S;
    }
    S.ks = (int)std::min<size_t>(m + 1, (kFusedSmem - fixed) / (S.ld * sizeof(double)));
    S.smem = fixed + (size_t)S.ks * S.ld * sizeof(double);
    return S;
}

static void launch_fused(const FusedShape &S, FusedArnoldi &F, cudaStream_t st) {
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = S.csize;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeCooperative;
    at[1].val.cooperative = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(S.clusters * S.csize);
    cfg.blockDim = dim3(kFusedThreads);
    cfg.dynamicSmemBytes = S.smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    PDD_CUDA(cudaLaunchKernelEx(&cfg, k_arnoldi_fused, F));
    count_launch();
}

// Failure injection on the host (tests): PDD_INJECT_BARRIER_TIMEOUT=1 makes every grid barrier
// of the fused Arnoldi kernel wait for one arrival more than the grid has, with a short poll
// limit; each block gives up after that limit, records the error and returns, and the solve
// reports PDD_ECUDA.  The device context stays usable.
static bool inject_barrier_timeout() {
    const char *v = std::getenv("PDD_INJECT_BARRIER_TIMEOUT");
    return v && v[0] == '1';
}

static SolveResult gmres_run(int n, const int *rowptr, const int *col, const double *val, const double *b, double *u,
                             const pdd_solve_opts &o, const GmresBufs &B, int m, int G, cudaStream_t st,
                             const RasPrecond *Mr = nullptr, double *Z = nullptr) {
    PDD_CUDA(cudaMemsetAsync(B.gs, 0, sizeof(GState), st));
    PDD_CUDA(cudaMemsetAsync(B.cnt, 0, sizeof(unsigned) * kDotGroups, st));
    PDD_CUDA(cudaMemsetAsync(B.bar, 0, sizeof(unsigned) * 2, st));
    PDD_CUDA(cudaMemsetAsync(u, 0, sizeof(double) * n, st));
    const int vb = std::min(cdiv(n, 256), 2048);
    const int max_iters = std::max(1, o.max_iters);
    const FusedShape S = fused_shape(n, m);
    const bool inject = inject_barrier_timeout();
    FusedArnoldi F{n, m, rowptr, col, val, B.V, B.fpart, S.w_global ? B.w : nullptr, B.H, B.g, B.gs, B.bar, o.rtol, max_iters, S.per, S.ld, S.ks,
                   inject ? 1u : 0u, inject ? (1LL << 14) : kBarrierLimit, 0, 0, nullptr, nullptr, nullptr,
                   nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
    if (Mr) {
        F.ras_P = Mr->P;
        F.ras_NP = Mr->NP;
        F.ras_wptr = Mr->wptr.p;
        F.ras_widx = Mr->widx.p;
        F.ras_p1 = Mr->p1.p;
        F.ras_l1 = Mr->l1.p;
        F.ras_p2 = Mr->p2.p;
        F.ras_l2 = Mr->l2.p;
        F.ras_cinvT = Mr->cinvT.p;
        F.ras_z = Mr->z.p;
        F.ras_Z = Z;
    }
    double *rr = &B.gs->rr;                                // device address: the residual's squared norm
    const size_t upper_smem = (size_t)kUpperCols * m * sizeof(double);
    allow_smem((const void *)k_upper_solve, upper_smem);
    SolveResult res;
    for (int cycle = 0;; ++cycle) {
        // the residual: b on the first cycle (u = 0), what the previous cycle ended with after that
        const double *r = cycle == 0 ? b : B.w;
        if (cycle == 0)
            PDD_LAUNCH(k_dots, dim3(G, 1), kDotThreads, 0, st, n, 1, r, r, B.partial, rr, B.cnt,
                       (const GState *)nullptr);
        PDD_LAUNCH(k_cycle_start, 1, 32, 0, st, B.gs, rr, B.g, m, o.rtol, max_iters, cycle == 0 ? 1 : 0);
        PDD_LAUNCH(k_normalize, vb, kDotBlock, 0, st, n, r, B.V, rr, (double *)nullptr, B.gs);
        launch_fused(S, F, st);
        PDD_LAUNCH(k_upper_solve, 1, kUpperThreads, upper_smem, st, B.H, m + 1, B.g, B.y, B.gs);
        // u += Z y (preconditioned: the z_j = M^-1 v_j of the cycle) or V y
        PDD_LAUNCH(k_xupdate, vb, 256, 0, st, n, Mr ? Z : B.V, B.y, B.gs, u);
        // true residual
        PDD_LAUNCH(k_spmv, cdiv(n, kRowsPerBlock), 256, 0, st, n, rowptr, col, val, u, B.w, b);
        PDD_LAUNCH(k_dots, dim3(G, 1), kDotThreads, 0, st, n, 1, B.w, B.w, B.partial, rr, B.cnt,
                   (const GState *)nullptr);
        GState hg{};
        PDD_CUDA(cudaMemcpyAsync(&hg, B.gs, sizeof(GState), cudaMemcpyDeviceToHost, st));
        PDD_CUDA(cudaStreamSynchronize(st));
        if (hg.err) fail(PDD_ECUDA, "GMRES grid barrier timed out");
        res.iters = hg.iters;
        if (hg.bnorm == 0.0) {                           // u = 0
            res.rel = 0.0;
            res.converged = 1;
            break;
        }
        // a NaN or an infinity in C or b, or a norm that overflows: no later cycle ends it
        if (!std::isfinite(hg.bnorm) || !std::isfinite(hg.rr)) {
            res.rel = std::nan("");
            break;
        }
        // (the test of the next cycle's start, rounding for rounding: a cycle that it skips would come again)
        const double beta = std::sqrt(hg.rr);
        res.rel = beta / hg.bnorm;
        if (beta <= o.rtol * hg.bnorm) {
            res.converged = 1;
            break;
        }
        if (hg.iters >= max_iters) break;
    }
    return res;
}

SolveResult gmres_csr(int n, const int *rowptr, const int *col, const double *val, const double *b, double *u,
                      const pdd_solve_opts &o, cudaStream_t st, const RasPrecond *Mr) {
    const int m = std::max(1, std::min(256, o.restart));
    const int G = std::max(1, std::min(1024, cdiv(n, 2 * kDotThreads)));
    DevBuf<double> V, w, partial, H, g, y, fpart;
    DevBuf<unsigned> cnt, bar;
    DevBuf<GState> gs;
    V.alloc((size_t)(m + 1) * n);
    w.alloc(n);
    partial.alloc(G);
    cnt.alloc(kDotGroups);
    H.alloc((size_t)(m + 1) * m);
    g.alloc(m + 1);
    y.alloc(m);
    gs.alloc(1);
    fpart.alloc((size_t)3 * kMaxDots * fused_shape(n, m).clusters);
    bar.alloc(2);
    const GmresBufs B{V.p, w.p, partial.p, H.p, g.p, y.p, fpart.p, cnt.p, bar.p, gs.p};
    DevBuf<double> Z;
    if (Mr) Z.alloc((size_t)m * n);
    return gmres_run(n, rowptr, col, val, b, u, o, B, m, G, st, Mr, Z.p);
}

// ---------------------------------------------------------------------------
// explicit transpose (counting sort by column, rows then sorted: deterministic)
// ---------------------------------------------------------------------------
__global__ void k_col_count(int64_t nnz, const int *col, int *cnt) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nnz; k += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&cnt[col[k]], 1);
}

__global__ void k_t_fill(int n, const int *rowptr, const int *col, const double *val, const int *ptr_t,
                         int *cursor, int *col_t, double *val_t) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = rowptr[i]; k < rowptr[i + 1]; ++k) {
        int c = col[k];
        int p = ptr_t[c] + atomicAdd(&cursor[c], 1);
        col_t[p] = i;
        val_t[p] = val[k];
    }
}

__global__ void k_t_sort(int n, const int *ptr_t, int *col_t, double *val_t) {
    int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    for (int k = ptr_t[r] + 1; k < ptr_t[r + 1]; ++k) {
        int c = col_t[k];
        double v = val_t[k];
        int q = k - 1;
        while (q >= ptr_t[r] && col_t[q] > c) {
            col_t[q + 1] = col_t[q];
            val_t[q + 1] = val_t[q];
            --q;
        }
        col_t[q + 1] = c;
        val_t[q + 1] = v;
    }
}

void csr_transpose(int n, int64_t nnz, const int *rowptr, const int *col, const double *val, DevBuf<int> &rowptr_t,
                   DevBuf<int> &col_t, DevBuf<double> &val_t, cudaStream_t st) {
    DevBuf<int> cnt, cursor;
    cnt.alloc(n + 1);
    cursor.alloc(n + 1);
    rowptr_t.alloc(n + 1);
    col_t.alloc(std::max<int64_t>(nnz, 1));
    val_t.alloc(std::max<int64_t>(nnz, 1));
    PDD_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int) * (n + 1), st));
    PDD_CUDA(cudaMemsetAsync(cursor.p, 0, sizeof(int) * (n + 1), st));
    PDD_LAUNCH(k_col_count, 1024, 256, 0, st, nnz, col, cnt.p);
    exclusive_scan_async(cnt.p, rowptr_t.p, n, st, nullptr);
    PDD_LAUNCH(k_t_fill, cdiv(n, 256), 256, 0, st, n, rowptr, col, val, rowptr_t.p, cursor.p, col_t.p, val_t.p);
    PDD_LAUNCH(k_t_sort, cdiv(n, 256), 256, 0, st, n, rowptr_t.p, col_t.p, val_t.p);
}

}  // namespace pdd

// ---------------------------------------------------------------------------
// Allocation-free variant of the CSR GMRES solve.
//
// Some callers cannot allocate device memory while they run: a host process
// whose device heap is owned by another allocator (a caching allocator that
// must not be bypassed or fragmented), a latency-critical loop that must not
// wait for an allocator, or a service that must not meet an out-of-memory
// failure half-way through a request.  For them
// pdd_solve_csr_noalloc runs the same GMRES kernels on a fixed workspace that
// lives in this file-scope device array, reserved when the library is loaded
// and held by every GPU that loads it until the process exits.
// ---------------------------------------------------------------------------
namespace pdd {

static constexpr size_t kNoAllocBytes = (size_t)64 << 20;          // 64 MiB per device
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

static constexpr int kMaxDevices = 64;
static void *g_noalloc_ptr[kMaxDevices] = {nullptr};
static std::mutex g_noalloc_mu;

// Device address of the scratch array on the current device (looked up once per device).
static void *noalloc_scratch(int dev) {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (dev < 0 || dev >= kMaxDevices) fail(PDD_EINVAL, "device ordinal out of range");
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) {
            set_error(cuda_msg(e, "cudaGetSymbolAddress(g_noalloc_scratch)"));
            throw Fail{PDD_ECUDA};
        }
        g_noalloc_ptr[dev] = p;
    }
    return g_noalloc_ptr[dev];
}

struct NoAllocLayout {
    size_t V, w, partial, cnt, H, g, y, gs, fpart, bar, total;
};

static NoAllocLayout noalloc_layout(int n, int m, int G, int clusters) {
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };
    NoAllocLayout L{};
    size_t off = 0;
    L.V = off; off += up(sizeof(double) * (size_t)(m + 1) * n);
    L.w = off; off += up(sizeof(double) * (size_t)n);
    L.partial = off; off += up(sizeof(double) * (size_t)G);
    L.cnt = off; off += up(sizeof(unsigned) * kDotGroups);
    L.H = off; off += up(sizeof(double) * (size_t)(m + 1) * m);
    L.g = off; off += up(sizeof(double) * (size_t)(m + 1));
    L.y = off; off += up(sizeof(double) * (size_t)m);
    L.gs = off; off += up(sizeof(GState));
    L.fpart = off; off += up(sizeof(double) * (size_t)3 * kMaxDots * clusters);
    L.bar = off; off += up(sizeof(unsigned) * 2);
    L.total = off;
    return L;
}

// The same iteration as gmres_csr, on buffers carved from `base`.
static SolveResult gmres_csr_fixed(int n, const int *rowptr, const int *col, const double *val,
                                   const double *b, double *u, const pdd_solve_opts &o, unsigned char *base,
                                   const NoAllocLayout &L, int m, int G, cudaStream_t st) {
    const GmresBufs B{(double *)(base + L.V), (double *)(base + L.w), (double *)(base + L.partial),
                      (double *)(base + L.H), (double *)(base + L.g), (double *)(base + L.y),
                      (double *)(base + L.fpart), (unsigned *)(base + L.cnt), (unsigned *)(base + L.bar),
                      (GState *)(base + L.gs)};
    return gmres_run(n, rowptr, col, val, b, u, o, B, m, G, st);
}

}  // namespace pdd

extern "C" pdd_status pdd_solve_csr_noalloc(int n, const int *rowptr, const int *col, const double *val,
                                            const double *b, double *u, const pdd_solve_opts *opts,
                                            pdd_solve_info *info, void *stream) {
    using namespace pdd;
    try {
        if (!opts) fail(PDD_EINVAL, "null solve options");
        if (opts->restart < 1 || opts->restart > 256 || opts->max_iters < 1 || !(opts->rtol > 0))
            fail(PDD_EINVAL, "restart in [1, 256], max_iters >= 1 and rtol > 0 required");
        if (opts->transpose) fail(PDD_EINVAL, "the allocation-free solve takes C itself (transpose = 0)");
        if (opts->precond != PDD_PRECOND_NONE) fail(PDD_EINVAL, "the allocation-free solve takes no preconditioner");
        if (n <= 0 || !rowptr || !col || !val || !b || !u) fail(PDD_EINVAL, "null array or n <= 0");
        const int m = opts->restart;
        const int G = std::max(1, std::min(1024, cdiv(n, 2 * kDotThreads)));
        const NoAllocLayout L = noalloc_layout(n, m, G, fused_shape(n, m).clusters);
        if (L.total > kNoAllocBytes)
            fail(PDD_EINVAL, "workspace of " + std::to_string(L.total) + " bytes exceeds the fixed " +
                                 std::to_string(kNoAllocBytes) + "-byte array: (restart + 2) * n * 8 bytes "
                                 "must stay below about 64 MiB");
        int dev = 0;
        PDD_CUDA(cudaGetDevice(&dev));
        unsigned char *base = (unsigned char *)noalloc_scratch(dev);
        SolveResult r = gmres_csr_fixed(n, rowptr, col, val, b, u, *opts, base, L, m, G, (cudaStream_t)stream);
        if (info) {
            info->iters = r.iters;
            info->rel_residual = r.rel;
            info->converged = r.converged;
        }
        if (!r.converged) fail(PDD_ENOCONV, "GMRES stopped at relative residual " + std::to_string(r.rel));
    } catch (const Fail &f) {
        return f.st;
    }
    return PDD_OK;
}
