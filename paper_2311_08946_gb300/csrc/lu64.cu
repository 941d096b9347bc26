// a7, FP64 form: blocked right-looking LU with partial pivoting of a batch of n x n FP64 matrices
// (row-major, in place), every step of a panel spread over the whole device.
//
// The FP64 pipe bounds it (2 FMAs a clock and SM): 2/3 n^3 operations cost 43 ms per SM at n = 1,024
// wherever they run, so what matters is that every SM takes part.  One CTA per disk left SMs idle
// whenever the disks were fewer than SMs or no multiple of them, and its panel steps had the other
// warps waiting.  Per panel of NB columns:
//   k_lu64_panel   one CTA per disk factors the panel in shared memory (two barriers a column: every
//                  warp finds the pivot from the warps' candidates, which the column's update has
//                  already collected for the next one), and lists which rows move;
//   k_lu64_rows    moves those rows in the columns outside the panel and solves U12 = L11^-1 A12, by
//                  column tiles;
//   k_lu64_update  A22 -= L21 U12 by tiles, 4 x 4 entries a thread.
// NB = 32, 16, 8 or 4, the widest whose panel fits in shared memory (n <= 863, 1,653, 3,045 and 5,259).
// 4 disks of n = 256: 2.63 -> 0.90 ms; 104 of n = 1,024: 113 -> 65 ms (57 at the FP64 peak); one of
// n = 3,072: 3,510 -> 38 ms.
#include <algorithm>

#include "handles.cuh"

namespace pdd {

static constexpr int kPanelThreads = 512;

template <int NB>
__host__ __device__ constexpr size_t lu64_panel_smem(int rows) {
    return (size_t)rows * (NB + 1) * sizeof(double) + (size_t)rows * sizeof(int);
}

// the largest (key, lowest row) of a warp's lanes, in every lane
__device__ __forceinline__ void pivot_reduce(unsigned long long &key, int &row, int width) {
    for (int o = width >> 1; o; o >>= 1) {
        const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
        const int r2 = __shfl_xor_sync(0xffffffffu, row, o);
        if (k2 > key || (k2 == key && r2 < row)) {
            key = k2;
            row = r2;
        }
    }
}

__device__ __forceinline__ unsigned long long abs_key(double v) {      // ordered like |v|
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffULL;
}

template <int NB>
__global__ void __launch_bounds__(kPanelThreads) k_lu64_panel(double *Aall, int n, long sA, int k0, int *permAll,
                                                              int *infoAll, int2 *movesAll, int *nmoves) {
    constexpr int LD = NB + 1, NW = kPanelThreads / 32;
    extern __shared__ __align__(16) double lsm[];
    __shared__ unsigned long long ck[2][NW];
    __shared__ int cr[2][NW], cnt;
    const int disk = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rows = n - k0, kb = min(NB, rows);
    double *A = Aall + disk * sA;
    int *perm = permAll + (long)disk * n;
    double *Pn = lsm;                                     // rows x LD
    int *src = reinterpret_cast<int *>(Pn + (size_t)rows * LD);        // which row each place holds
    for (int e = tid; e < rows * NB; e += kPanelThreads) {
        const int r = e / NB, c = e - r * NB;
        if (c < kb) Pn[r * LD + c] = A[(long)(k0 + r) * n + k0 + c];
    }
    for (int r = tid; r < rows; r += kPanelThreads) src[r] = r;
    if (tid == 0) cnt = 0;
    __syncthreads();
    unsigned long long key = 0;
    int at = 0x7fffffff, info = 0;
    for (int r = tid; r < rows; r += kPanelThreads) {
        const unsigned long long k = abs_key(Pn[r * LD]);
        if (k > key || at == 0x7fffffff) {
            key = k;
            at = r;
        }
    }
    for (int c = 0; c < kb; ++c) {
        const int b = c & 1;
        pivot_reduce(key, at, 32);
        if (lane == 0) {
            ck[b][warp] = key;
            cr[b][warp] = at;
        }
        __syncthreads();
        key = lane < NW ? ck[b][lane] : 0;
        at = lane < NW ? cr[b][lane] : 0x7fffffff;
        pivot_reduce(key, at, 32);
        const int p = at;                                 // c <= p < rows (some thread has a candidate)
        const double d = Pn[p * LD + c];
        __syncthreads();                                  // every thread has d before the rows change places
        if (warp == 0 && p != c) {
            if (lane < kb) {
                const double t = Pn[c * LD + lane];
                Pn[c * LD + lane] = Pn[p * LD + lane];
                Pn[p * LD + lane] = t;
            }
            if (lane == 0) {
                const int t = src[c];
                src[c] = src[p];
                src[p] = t;
            }
        }
        __syncthreads();
        if (d == 0.0 && info == 0) info = k0 + c + 1;
        const double inv = d != 0.0 ? 1.0 / d : 0.0;
        key = 0;
        at = 0x7fffffff;
        for (int r = c + 1 + tid; r < rows; r += kPanelThreads) {
            double *row = Pn + r * LD;
            const double l = row[c] * inv;
            row[c] = l;
            for (int cc = c + 1; cc < kb; ++cc) row[cc] -= l * Pn[c * LD + cc];
            if (c + 1 < kb) {
                const unsigned long long k = abs_key(row[c + 1]);
                if (k > key || at == 0x7fffffff) {
                    key = k;
                    at = r;
                }
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < rows * NB; e += kPanelThreads) {
        const int r = e / NB, c = e - r * NB;
        if (c < kb) A[(long)(k0 + r) * n + k0 + c] = Pn[r * LD + c];
    }
    // the rows that moved and their new entries of the permutation, staged in the panel's storage: every
    // old entry is read before one is written
    int2 *mv = movesAll + (long)disk * 2 * NB;
    int *staged = reinterpret_cast<int *>(lsm);
    __syncthreads();
    for (int r = tid; r < rows; r += kPanelThreads)
        if (src[r] != r) {
            mv[atomicAdd(&cnt, 1)] = make_int2(k0 + r, k0 + src[r]);      // at most 2 kb of them
            staged[r] = perm[k0 + src[r]];
        }
    __syncthreads();
    for (int r = tid; r < rows; r += kPanelThreads)
        if (src[r] != r) perm[k0 + r] = staged[r];
    if (tid == 0) {
        nmoves[disk] = cnt;
        if (info && infoAll[disk] == 0) infoAll[disk] = info;
    }
}

// columns outside the panel: rows moved, then (right of it) U12 = L11^-1 A12
static constexpr int kRowsCols = 64, kRowsThreads = 256;

template <int NB>
__global__ void __launch_bounds__(kRowsThreads, 2) k_lu64_rows(double *Aall, int n, long sA, int k0, const int2 *movesAll,
                                                            const int *nmoves) {
    __shared__ double T[2 * NB][kRowsCols];
    __shared__ double L[NB][NB + 1];
    const int disk = blockIdx.y, tid = threadIdx.x;
    const int kb = min(NB, n - k0);
    // column tiles left of the panel, then right of it
    const int left = (k0 + kRowsCols - 1) / kRowsCols;
    const bool right = (int)blockIdx.x >= left;
    const int c0 = right ? k0 + kb + ((int)blockIdx.x - left) * kRowsCols : (int)blockIdx.x * kRowsCols;
    const int cend = right ? n : k0, ncol = min(kRowsCols, cend - c0);
    if (ncol <= 0) return;
    double *A = Aall + disk * sA;
    const int2 *mv = movesAll + (long)disk * 2 * NB;
    const int nm = nmoves[disk];
    for (int e = tid; e < nm * kRowsCols; e += kRowsThreads) {
        const int i = e / kRowsCols, c = e - i * kRowsCols;
        if (c < ncol) T[i][c] = A[(long)mv[i].y * n + c0 + c];
    }
    __syncthreads();
    for (int e = tid; e < nm * kRowsCols; e += kRowsThreads) {
        const int i = e / kRowsCols, c = e - i * kRowsCols;
        if (c < ncol) A[(long)mv[i].x * n + c0 + c] = T[i][c];
    }
    if (!right) return;
    for (int e = tid; e < NB * NB; e += kRowsThreads) {
        const int r = e / NB, c = e - r * NB;
        L[r][c] = (r < kb && c < r) ? A[(long)(k0 + r) * n + k0 + c] : 0.0;
    }
    __syncthreads();
    if (tid < ncol) {
        double x[NB];
#pragma unroll
        for (int r = 0; r < NB; ++r) x[r] = r < kb ? A[(long)(k0 + r) * n + c0 + tid] : 0.0;
#pragma unroll
        for (int t = 0; t < NB - 1; ++t)
#pragma unroll
            for (int r = t + 1; r < NB; ++r) x[r] -= L[r][t] * x[t];
#pragma unroll
        for (int r = 0; r < NB; ++r)
            if (r < kb) A[(long)(k0 + r) * n + c0 + tid] = x[r];
    }
}

// A22 -= L21 U12 in TS x TS tiles, 4 x 4 entries a thread
template <int NB, int TS>
__global__ void __launch_bounds__((TS / 4) * (TS / 4)) k_lu64_update(double *Aall, int n, long sA, int k0) {
    constexpr int NT = (TS / 4) * (TS / 4);
    __shared__ double Ls[NB][TS + 1], Us[NB][TS];
    const int disk = blockIdx.z, tid = threadIdx.x;
    const int kb = min(NB, n - k0), b0 = k0 + kb;
    const int r0 = b0 + blockIdx.y * TS, c0 = b0 + blockIdx.x * TS;
    double *A = Aall + disk * sA;
    for (int e = tid; e < TS * NB; e += NT) {
        const int r = e / NB, t = e - r * NB;
        Ls[t][r] = (r0 + r < n && t < kb) ? A[(long)(r0 + r) * n + k0 + t] : 0.0;
    }
    for (int e = tid; e < NB * TS; e += NT) {
        const int t = e / TS, c = e - t * TS;
        Us[t][c] = (c0 + c < n && t < kb) ? A[(long)(k0 + t) * n + c0 + c] : 0.0;
    }
    const int ty = tid / (TS / 4), tx = tid % (TS / 4);
    // a thread's rows ty + (TS/4) a and columns tx + (TS/4) b: consecutive lanes, consecutive columns
    double acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = r0 + ty + (TS / 4) * a, c = c0 + tx + (TS / 4) * b;
            acc[a][b] = (r < n && c < n) ? A[(long)r * n + c] : 0.0;
        }
    __syncthreads();
#pragma unroll 4
    for (int t = 0; t < NB; ++t) {
        double l[4], u[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) l[a] = Ls[t][ty + (TS / 4) * a];
#pragma unroll
        for (int b = 0; b < 4; ++b) u[b] = Us[t][tx + (TS / 4) * b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] -= l[a] * u[b];
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int r = r0 + ty + (TS / 4) * a, c = c0 + tx + (TS / 4) * b;
            if (r < n && c < n) A[(long)r * n + c] = acc[a][b];
        }
}

__global__ void k_lu64_init(int n, int nd, int *perm, int *info) {
    const long i = blockIdx.x * 256L + threadIdx.x;
    if (i < (long)n * nd) perm[i] = (int)(i % n);
    if (i < nd) info[i] = 0;
}

static constexpr int kPanelSmem = 226 * 1024;        // 227 KB per CTA, less the static arrays

template <int NB>
static void lu64_run(double *A, int n, long sA, int *perm, int *info, int nd, int sms, cudaStream_t st) {
    DevBuf<int2> moves;
    DevBuf<int> nmoves;
    moves.alloc((size_t)nd * 2 * NB);
    nmoves.alloc(nd);
    PDD_CUDA(cudaFuncSetAttribute(k_lu64_panel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPanelSmem));
    for (int k0 = 0; k0 < n; k0 += NB) {
        const int kb = std::min(NB, n - k0), rem = n - k0 - kb;
        PDD_LAUNCH(k_lu64_panel<NB>, nd, kPanelThreads, lu64_panel_smem<NB>(n - k0), st, A, n, sA, k0, perm, info,
                   moves.p, nmoves.p);
        const int tiles = cdiv(k0, kRowsCols) + cdiv(rem, kRowsCols);
        if (tiles > 0)
            PDD_LAUNCH(k_lu64_rows<NB>, dim3(tiles, nd), kRowsThreads, 0, st, A, n, sA, k0, moves.p, nmoves.p);
        if (rem <= 0) continue;
        // tiles of 64, or of 32 while those would leave SMs without one (an update of a 64-tile with NB = 32
        // takes an SM 32 us)
        const int t64 = cdiv(rem, 64);
        if ((long)t64 * t64 * nd >= 2L * sms)
            PDD_LAUNCH((k_lu64_update<NB, 64>), dim3(t64, t64, nd), 256, 0, st, A, n, sA, k0);
        else
            PDD_LAUNCH((k_lu64_update<NB, 32>), dim3(cdiv(rem, 32), cdiv(rem, 32), nd), 64, 0, st, A, n, sA, k0);
    }
}

// false when the panel of n rows does not fit in shared memory or the batch exceeds a launch's grid (the
// caller's one-CTA form takes those)
bool lu_f64(double *A, int n, long strideA, int *perm, int *info, int nd, cudaStream_t st) {
    const size_t most = kPanelSmem;
    if (lu64_panel_smem<4>(n) > most || nd > 65535) return false;
    int dev = 0, sms = 0;
    PDD_CUDA(cudaGetDevice(&dev));
    PDD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PDD_LAUNCH(k_lu64_init, cdiv(std::max<long>((long)n * nd, nd), 256), 256, 0, st, n, nd, perm, info);
    if (lu64_panel_smem<32>(n) <= most) lu64_run<32>(A, n, strideA, perm, info, nd, sms, st);
    else if (lu64_panel_smem<16>(n) <= most) lu64_run<16>(A, n, strideA, perm, info, nd, sms, st);
    else if (lu64_panel_smem<8>(n) <= most) lu64_run<8>(A, n, strideA, perm, info, nd, sms, st);
    else lu64_run<4>(A, n, strideA, perm, info, nd, sms, st);
    return true;
}

}  // namespace pdd
