// a10-a12: Monte Carlo rows (Eq. 25-30 with the representation of Eq. 53,
// 56 and sigma = I), IMQ cardinals on perimeter arcs (Eq. 19-22).
//
//   a10 k_imq_inverse: K_lk = ((u_l - u_k)^2 + c^2)^-1/2 per perimeter stencil
//       (u the knots' local angles in radians), Cholesky factor and K^-1 in FP64
//       (one CTA per circle), and kappa_1(K).
//   a11 k_paths (short paths), k_paths_long, k_paths64 (FP64 form), with exit
//       points by k_exit32, k_exit64: Euler-Maruyama paths of dX = b dt + dW, dY = c Y dt,
//       dZ = f Y dt from the knot, stopped at the first step whose end point
//       leaves the open disk or the open domain (optionally both shrunk by the
//       Gobet-Menozzi shift).  A lane takes the next path id (of its row or of
//       the launch) as soon as its path exits.  Exit point: the
//       first crossing of the segment with the circle or dOmega (ties to
//       dOmega).  Normals: Philox4x32-10, key (seed, knot), counter (step,
//       path, 0, k) with k the subdomain's position in the row's list.  FP64
//       form: every quantity in FP64.  Mixed form: position, drift and normals
//       in FP32, weights Y, Z and all scores in FP64.  Per-path exit records
//       (side, angle or arclength, Y, Z) go to a device scratch buffer.
//   a12 k_mc_finalize: one CTA of 16 warps per slot; warp w owns batches w and
//       w + 16 (paths p = b mod 32) and its lanes own basis functions.  The
//       moments M_l = E[1_Gamma Y phi_l(u)], C_ij = -sum_l (K^-1)_lj M_l (IMQ)
//       or -M_j (Fourier cardinals), the slot's part of r_i = E[1_dOmega g Y +
//       Z]; standard errors by batch means over the 32 batches.
#include <algorithm>
#include <vector>

#include "exp64.cuh"
#include "handles.cuh"

namespace pdd {

static constexpr int kBatches = 32;
static constexpr int kMaxStencil = 96;
static constexpr double kFastKappa = 1e5;      // largest kappa_1(K) summed in FP32 (mixed form)
static constexpr double kDfKappa = 1e10;       // largest kappa_1(K) summed in double-float (mixed form)

// ---------------------------------------------------------------------------
// a10
// ---------------------------------------------------------------------------
// largest column sum of |A| (n x n in shared memory), by the block
__device__ double norm1_block(const double *A, int n, double *red) {
    double mx = 0.0;
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
        double s = 0.0;
        for (int l = 0; l < n; ++l) s += fabs(A[l * n + c]);
        mx = fmax(mx, s);
    }
    red[threadIdx.x] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int t = 0; t < blockDim.x; ++t) v = fmax(v, red[t]);
        red[0] = v;
    }
    __syncthreads();
    const double v = red[0];
    __syncthreads();
    return v;
}

__global__ void __launch_bounds__(128) k_imq_inverse(const int *circles, const int *knot_ptr,
                                                     const double *ku, const long *kinv_off,
                                                     double c2, double *kinv, double *kcond, int *bad) {
    extern __shared__ double sm[];                    // K (n x n), then L in place
    __shared__ double red[128];
    const int m = circles[blockIdx.x];
    const int a = knot_ptr[m], n = knot_ptr[m + 1] - a;
    double *K = sm;
    double *Z = sm + n * n;                           // n x n work for the inverse
    const int tid = threadIdx.x;
    for (int idx = tid; idx < n * n; idx += blockDim.x) {
        int l = idx / n, k = idx % n;
        double d = ku[a + l] - ku[a + k];
        K[idx] = 1.0 / sqrt(d * d + c2);
    }
    __syncthreads();
    const double nK = norm1_block(K, n, red);
    // right-looking Cholesky, lower triangle
    for (int j = 0; j < n; ++j) {
        if (tid == 0) {
            double v = K[j * n + j];
            if (!(v > 0.0)) atomicAdd(bad, 1);
            K[j * n + j] = sqrt(fmax(v, 1e-300));
        }
        __syncthreads();
        const double d = K[j * n + j];
        for (int i = j + 1 + tid; i < n; i += blockDim.x) K[i * n + j] /= d;
        __syncthreads();
        for (int idx = tid; idx < (n - j - 1) * (n - j - 1); idx += blockDim.x) {
            int i = j + 1 + idx / (n - j - 1), k = j + 1 + idx % (n - j - 1);
            if (k <= i) K[i * n + k] -= K[i * n + j] * K[k * n + j];
        }
        __syncthreads();
    }
    // K^-1 = L^-T L^-1: column c of the identity per thread
    for (int c = tid; c < n; c += blockDim.x) {
        for (int i = 0; i < n; ++i) {                 // L y = e_c
            double v = (i == c) ? 1.0 : 0.0;
            for (int k = 0; k < i; ++k) v -= K[i * n + k] * Z[k * n + c];
            Z[i * n + c] = v / K[i * n + i];
        }
        for (int i = n - 1; i >= 0; --i) {            // L^T x = y
            double v = Z[i * n + c];
            for (int k = i + 1; k < n; ++k) v -= K[k * n + i] * Z[k * n + c];
            Z[i * n + c] = v / K[i * n + i];
        }
    }
    __syncthreads();
    const double nZ = norm1_block(Z, n, red);
    if (tid == 0) kcond[m] = nK * nZ;                 // kappa_1(K)
    double *out = kinv + kinv_off[blockIdx.x];
    for (int idx = tid; idx < n * n; idx += blockDim.x) out[idx] = Z[idx];
}

// ---------------------------------------------------------------------------
// a11
// ---------------------------------------------------------------------------
struct PathArgs {
    // per slot: the row (knot) i; per global slot gs: its subdomain and the position of that
    // subdomain in Pi_i (Philox counter word 3; null: 0)
    const int *rows, *subs, *kword;
    const double *kx, *ky, *ccx, *ccy, *cr, *theta_s;
    int paths;                       // paths per row when npaths is null
    double h;
    uint64_t seed;
    int8_t *side;
    double *su, *Y, *Z;
    unsigned long long *steps;
    int *capped;
    const int *npaths;               // per-row path counts (adaptive), or null
    const long *rec_off;             // per-row record offsets, or null (slot * paths)
    float2 *ez;                      // mixed form: the unfolded FP32 increments (e, z) of each record
    double shift;                    // Gobet-Menozzi boundary shift c0 sqrt(h), or 0 (plain exit)
    const int *gslot;                // global slot of each launched slot, or null (slot)
    int max_steps;                   // step cap per path (0: 50 r^2 / h)
    int cvd, ncv;                    // control-variate monomial degree (0: none) and feature count
    double *cvq;                     // per-path features [rec][ncv]
};

// c0 = -zeta(1/2) / sqrt(2 pi): the Gobet-Menozzi shift in units of |sigma^T n| sqrt(h) (sigma = I)
static constexpr double kGmC0 = 0.5825971579390108;

__device__ __forceinline__ double circle_exit_t(double px, double py, double dx, double dy, double ox,
                                                double oy, double rad) {
    const double qx = px - ox, qy = py - oy;
    const double a = dx * dx + dy * dy;
    const double b = qx * dx + qy * dy;
    const double c = qx * qx + qy * qy - rad * rad;
    double disc = b * b - a * c;
    if (disc < 0.0) disc = 0.0;
    const double sq = sqrt(disc);
    return (b >= 0.0) ? -c / (b + sq) : (sq - b) / a;
}

// first crossing of the segment P -> P + D with the circle |z - o| = rad (P inside), in R
template <typename R>
__device__ __forceinline__ R circle_exit_tr(R px, R py, R dx, R dy, R ox, R oy, R rad) {
    const R qx = px - ox, qy = py - oy;
    const R a = dx * dx + dy * dy;
    const R b = qx * dx + qy * dy;
    const R c = qx * qx + qy * qy - rad * rad;
    R disc = b * b - a * c;
    if (disc < (R)0) disc = (R)0;
    const R sq = sqrt(disc);
    return (b >= (R)0) ? -c / (b + sq) : (sq - b) / a;
}

template <typename R>
struct Num;
template <>
struct Num<double> {
    __device__ static void normals(uint64_t s, uint32_t k, uint32_t q, uint32_t st, uint32_t p, double &a, double &b) {
        normals64(s, k, q, st, p, a, b);
    }
    __device__ static void drift(const Problem &P, double x, double y, double &bx, double &by) {
        pdd::drift(P, x, y, bx, by);
    }
    __device__ static double sq(double v) { return sqrt(v); }
};
template <>
struct Num<float> {
    __device__ static void normals(uint64_t s, uint32_t k, uint32_t q, uint32_t st, uint32_t p, float &a, float &b) {
        normals32(s, k, q, st, p, a, b);
    }
    __device__ static void drift(const Problem &P, float x, float y, float &bx, float &by) {
        if (P.b_kind == PDD_B_SINX_COSY) {
            bx = __sinf(reduce_2pi(x));
            by = __cosf(reduce_2pi(y));
        } else {
            bx = 0.f;
            by = 0.f;
        }
    }
    __device__ static float sq(float v) { return sqrtf(v); }
};

__device__ __forceinline__ float killing32(const Problem &P, float x, float y) {
    if (P.c_kind == PDD_C_QUADRATIC) return -(1.0f + x * x + y * y);
    if (P.c_kind == PDD_C_RBF) {
        float s = 0.f;
        const int nr = P.n_rbf;
        const float *cx = P.rbf32, *cy = P.rbf32 + nr, *cw = P.rbf32 + 2 * nr;
        for (int q = 0; q < nr; ++q) {
            const float dx = x - cx[q], dy = y - cy[q];
            s += cw[q] * __expf(-(dx * dx + dy * dy) * P.rbf_inv2s2);
        }
        return s < 0.f ? s : 0.f;
    }
    return 0.f;
}

// f of the manufactured solution from already evaluated b and c (FP32)
__device__ __forceinline__ float source32_given(const Problem &P, float x, float y, float bx, float by, float cv) {
    if (P.f_kind == PDD_F_RBF) {
        const int nq = P.n_frbf;
        const float *fx = P.frbf32, *fy = P.frbf32 + nq, *fw = P.frbf32 + 2 * nq;
        float s = 0.f;
        for (int q = 0; q < nq; ++q) {
            const float dx = x - fx[q], dy = y - fy[q];
            s += fw[q] * __expf(-(dx * dx + dy * dy) * P.frbf_inv2s2);
        }
        return s;
    }
    if (P.f_kind == PDD_F_ONE) return 1.0f;
    if (P.f_kind == PDD_F_MANUFACTURED) {
        float spx, cpx, spy, cpy;
        fast_sincospi(x, spx, cpx);
        fast_sincospi(y, spy, cpy);
        const float pi = 3.14159265358979f;
        const float u = spx * cpy, ux = pi * cpx * cpy, uy = -pi * spx * spy;
        return -(-pi * pi * u + bx * ux + by * uy + cv * u);
    }
    if (P.f_kind == PDD_F_EQ46) {
        float u, ux, uy, lap;
        u46_derivs(x, y, u, ux, uy, lap);
        return -(0.5f * lap + bx * ux + by * uy + cv * u);
    }
    return 0.f;
}

__device__ __forceinline__ float source32(const Problem &P, float x, float y) {
    float bx, by;
    Num<float>::drift(P, x, y, bx, by);
    return source32_given(P, x, y, bx, by, killing32(P, x, y));
}

// Control-variate features (CV): for the monomials psi = xr^a yr^b (1 <= a + b <= D <= 4) of
// xr = (x - cx) / r, yr = (y - cy) / r, the sums Q = sum_k Y_k sqrt(h) grad psi(X_k) . xi_k, which have
// mean zero whatever psi (xi_k is independent of X_k and Y_k): the regression control variate of
// Milstein and Tretyakov (features in the order d = a + b = 1..D, a = d..0).
static constexpr int kMaxCv = 14;

template <typename R>
__device__ __forceinline__ void cv_accumulate(R (&cq)[kMaxCv], int D, R xr, R yr, R s, R xi0, R xi1) {
    R px[5], py[5];
    px[0] = (R)1;
    py[0] = (R)1;
#pragma unroll
    for (int e = 1; e <= 4; ++e) {
        px[e] = px[e - 1] * xr;
        py[e] = py[e - 1] * yr;
    }
    int q = 0;
#pragma unroll
    for (int d = 1; d <= 4; ++d) {
        if (d > D) break;
#pragma unroll
        for (int a = d; a >= 0; --a) {
            const int b = d - a;
            R g = (R)0;
            if (a > 0) g += (R)a * px[a - 1] * py[b] * xi0;
            if (b > 0) g += (R)b * px[a] * py[b - 1] * xi1;
            cq[q] += s * g;
            ++q;
        }
    }
}

// packed FP32 pairs, each lane of the pair rounded like the scalar operation
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long r, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2p(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Gaussians in shared memory, two by two: (-x0, -x1, -y0, -y1) and (w0, w1), a missing second one with
// weight 0.  The sum of killing32 and source32_given, term by term and rounding by rounding; per pair two
// shared loads and five packed operations where the global form takes six loads and ten.
struct GaussTab {
    const float4 *xy;
    const float2 *w;
    int pairs;
    float ninv;              // -1 / (2 sigma^2)
};
__device__ __forceinline__ float gauss_sum(const GaussTab &G, float x, float y) {
    const unsigned long long x2 = pack2(x, x), y2 = pack2(y, y), n2 = pack2(G.ninv, G.ninv);
    float s = 0.f;
#pragma unroll 4
    for (int q = 0; q < G.pairs; ++q) {
        const float4 c = G.xy[q];
        const float2 w = G.w[q];
        const unsigned long long dx = add2(x2, pack2(c.x, c.y)), dy = add2(y2, pack2(c.z, c.w));
        float a0, a1;
        unpack2(mul2(fma2p(dx, dx, mul2(dy, dy)), n2), a0, a1);
        s = fmaf(w.x, __expf(a0), s);
        s = fmaf(w.y, __expf(a1), s);
    }
    return s;
}

// ---------------------------------------------------------------------------
// Mixed form: positions, drift and normals in FP32, weights in FP64.  Instruction issue bounds it
// (Philox, Box-Muller and the coefficients, some 150 instructions a step).
//   k_paths       one CTA per row, whose constants are the block's: starting a path takes a few
//                 instructions, for short paths (62 steps on the variable-coefficient cover).
//   k_paths_long  resident warps take the launch's records 256 at a time and hand them to the lanes
//                 that are free: no lanes idle while the last paths of a row finish, no part-filled last
//                 wave of CTAs; exit points by k_exit32, one thread per record.  Starting a path takes some
//                 eighty instructions (its row's constants), so it is for paths of kLongSteps steps and
//                 more on average.
// Control variate of degree 4, boundary shift (1,000 rows x 5,000 paths of 1,684 steps): 179 -> 141 ms in
// k_paths_long; drift, killing and source (2,276 rows x 10^4 paths): 16.5 ms in k_paths, 31 in
// k_paths_long; killing by 64 Gaussians (3,000 rows), read from shared memory two at a time: 68 -> 49 ms.
// ---------------------------------------------------------------------------
struct alignas(16) Slot32 {          // what a path reads when it starts
    float cx, cy, r2, rs, x0, y0, rad, ts;      // r2, rs: of the disk shrunk by the boundary shift
    long rbase;
    int i, max_steps;
    uint32_t kw;
    int pad[3];
};
struct Pool32 {
    const Slot32 *slots;
    int nslots;
    long total;                      // records of the launch
    unsigned *next;                  // chunks taken
    float4 *seg;                     // per record: the last step's segment (x, y, nx, ny)
    int nc, nf;                      // Gaussians of c and f kept in shared memory (0: none)
};
static constexpr int kP32Threads = 128, kP32Chunk = 256, kRowThreads = 256;
static constexpr double kLongSteps = 500.0;
static constexpr int kP32Staged = 1024;          // most Gaussians of c or f kept in shared memory (24 KB each)

__global__ void k_slots32(int n, PathArgs A, Slot32 *out) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= n) return;
    const int gsl = A.gslot ? A.gslot[slot] : slot;
    const int i = A.rows[slot], m = A.subs[gsl];
    const double rad = A.cr[m], rs = rad - A.shift;
    Slot32 s;
    s.cx = (float)A.ccx[m];
    s.cy = (float)A.ccy[m];
    s.r2 = (float)(rs * rs);
    s.rs = (float)rs;
    s.x0 = (float)A.kx[i];
    s.y0 = (float)A.ky[i];
    s.rad = (float)rad;
    s.ts = (float)A.theta_s[m];
    s.rbase = A.rec_off ? A.rec_off[slot] : (long)slot * A.paths;
    s.i = i;
    s.max_steps = A.max_steps > 0 ? A.max_steps : (int)fmin(2147483647.0, ceil(50.0 * rad * rad / A.h));
    s.kw = A.kword ? (uint32_t)A.kword[gsl] : 0u;
    s.pad[0] = s.pad[1] = s.pad[2] = 0;
    out[slot] = s;
}

// the slot of record g (the records of the slots are contiguous and in slot order)
template <typename SlotT>
__device__ __forceinline__ int slot_of(const PathArgs &A, const SlotT *slots, int nslots, long g) {
    if (!A.rec_off) return (int)((unsigned)g / (unsigned)A.paths);      // at most 2^31 records per launch
    int lo = 0, hi = nslots - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (slots[mid].rbase <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// a Gaussian family into shared memory (see GaussTab), by the block
__device__ __forceinline__ GaussTab stage_gauss(float4 *smem, const float *src, int n, float inv2s2) {
    GaussTab G;
    G.pairs = (n + 1) >> 1;
    G.ninv = -inv2s2;
    float2 *w = reinterpret_cast<float2 *>(smem + G.pairs);
    for (int q = threadIdx.x; q < G.pairs; q += blockDim.x) {
        const int a = 2 * q, b = 2 * q + 1 < n ? 2 * q + 1 : a;
        smem[q] = make_float4(-src[a], -src[b], -src[n + a], -src[n + b]);
        w[q] = make_float2(src[2 * n + a], 2 * q + 1 < n ? src[2 * n + b] : 0.f);
    }
    G.xy = smem;
    G.w = w;
    return G;
}
__host__ __device__ constexpr size_t gauss_smem(int n) { return (((size_t)(n + 1) / 2) * 24 + 15) / 16 * 16; }

// constants of a launch
struct Env32 {
    GaussTab gc, gf;
    float h, sh, d0, d1, d2, d3, dr2;
    bool sq_dom;
};
template <bool KILL, bool SRC>
__device__ __forceinline__ Env32 env32(const Problem &P, const PathArgs &A, const Pool32 &Q, unsigned char *smem) {
    Env32 E{};
    if (KILL && Q.nc) E.gc = stage_gauss(reinterpret_cast<float4 *>(smem), P.rbf32, Q.nc, P.rbf_inv2s2);
    if (SRC && Q.nf)
        E.gf = stage_gauss(reinterpret_cast<float4 *>(smem + (Q.nc ? gauss_smem(Q.nc) : 0)), P.frbf32, Q.nf,
                           P.frbf_inv2s2);
    const double sft = A.shift;
    E.sq_dom = P.dom_kind == 0;
    E.h = (float)A.h;
    E.sh = sqrtf((float)A.h);
    E.d0 = (float)(E.sq_dom ? P.dom[0] + sft : P.dom[0]);
    E.d1 = (float)(E.sq_dom ? P.dom[1] + sft : P.dom[1]);
    E.d2 = (float)(P.dom[2] - sft);
    E.d3 = (float)(P.dom[3] - sft);
    E.dr2 = (float)((P.dom[2] - sft) * (P.dom[2] - sft));
    return E;
}

// a path: position, weights Y = Yv (1 + e) and Z = Zv + Yv z (e, z: FP32 increments), step count
struct Path32 {
    float x, y, e, z;
    double Yv, Zv;
    int k;
};

// One Euler-Maruyama step of path S (of knot, on the circle (cx, cy) with squared radius r2): moves it, or
// returns true when its end point (nx, ny) is outside, the weights then being those after the step.
// `fold`: the iterations that fold the FP32 increments into the FP64 weights.
// CVD: control-variate degree, 0 (none), 4, or -1 (A.cvd at run time)
template <bool KILL, bool SRC, int CVD>
__device__ __forceinline__ bool step32(const Problem &P, const PathArgs &A, const Pool32 &Q, const Env32 &E, Path32 &S,
                                       int knot, uint32_t kw, int p, float cx, float cy, float r2, float crad,
                                       float rcrad, float *cq, bool fold, float &nx, float &ny) {
    float xi0, xi1;
    normals32(A.seed, (uint32_t)knot, kw, (uint32_t)S.k, (uint32_t)p, xi0, xi1);
    if constexpr (CVD != 0) {
        // Y_k sqrt(h) grad psi(X_k) . xi_k / r, with Y_k the weight before this step
        const float yk = (float)S.Yv * (1.0f + S.e);
        cv_accumulate<float>(*reinterpret_cast<float(*)[kMaxCv]>(cq), CVD > 0 ? CVD : A.cvd,
                             quotient(S.x - cx, crad, rcrad), quotient(S.y - cy, crad, rcrad),
                             quotient(yk * E.sh, crad, rcrad), xi0, xi1);
    }
    float bx, by;
    Num<float>::drift(P, S.x, S.y, bx, by);
    float cv = 0.f;
    if (KILL) {
        if (Q.nc) {
            const float s = gauss_sum(E.gc, S.x, S.y);
            cv = s < 0.f ? s : 0.f;
        } else {
            cv = killing32(P, S.x, S.y);
        }
    }
    // Z_{k+1} = Z_k + f_k h Y_k and Y_{k+1} = Y_k (1 + c_k h), with Y_k = Yv (1 + e)
    const float e = S.e;
    if (SRC) {
        const float fv = Q.nf ? gauss_sum(E.gf, S.x, S.y) : source32_given(P, S.x, S.y, bx, by, cv);
        S.z = fmaf(fv * E.h, 1.0f + e, S.z);
    }
    if (KILL) S.e = fmaf(cv * E.h, 1.0f + e, e);
    nx = S.x + bx * E.h + E.sh * xi0;
    ny = S.y + by * E.h + E.sh * xi1;
    ++S.k;
    const float ddx = nx - cx, ddy = ny - cy;
    bool out = !(ddx * ddx + ddy * ddy < r2);
    if (E.sq_dom) {
        out = out || !(nx > E.d0 && nx < E.d2 && ny > E.d1 && ny < E.d3);
    } else {
        const float ex0 = nx - E.d0, ey0 = ny - E.d1;
        out = out || !(ex0 * ex0 + ey0 * ey0 < E.dr2);
    }
    if (fold) {
        S.Zv = fma(S.Yv, (double)S.z, S.Zv);
        S.Yv = fma(S.Yv, (double)S.e, S.Yv);
        S.e = 0.f;
        S.z = 0.f;
    }
    if (!out) {
        S.x = nx;
        S.y = ny;
    }
    return out;
}

// the record of a path that left (k_exit32 finds the side and the exit point) or reached the step cap
template <bool CV>
__device__ __forceinline__ void record_exit(const PathArgs &A, const Pool32 &Q, long rec, const Path32 &S, float nx,
                                            float ny, const float *cq) {
    A.side[rec] = 3;
    Q.seg[rec] = make_float4(S.x, S.y, nx, ny);
    A.Y[rec] = S.Yv;
    A.Z[rec] = S.Zv;
    A.ez[rec] = make_float2(S.e, S.z);
    if constexpr (CV) {
#pragma unroll
        for (int q = 0; q < kMaxCv; ++q)
            if (q < A.ncv) A.cvq[rec * A.ncv + q] = (double)cq[q];
    }
}
template <bool CV>
__device__ __forceinline__ void record_capped(const PathArgs &A, long rec) {
    A.side[rec] = 2;
    A.su[rec] = 0.0;
    A.Y[rec] = 0.0;
    A.Z[rec] = 0.0;
    A.ez[rec] = make_float2(0.f, 0.f);
    if constexpr (CV)
        for (int q = 0; q < A.ncv; ++q) A.cvq[rec * A.ncv + q] = 0.0;
}

__device__ __forceinline__ void add_totals(const PathArgs &A, unsigned long long steps, int capped) {
    for (int o = 16; o; o >>= 1) {
        steps += __shfl_xor_sync(0xffffffffu, steps, o);
        capped += __shfl_xor_sync(0xffffffffu, capped, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (steps) atomicAdd(A.steps, steps);
        if (capped) atomicAdd(A.capped, capped);
    }
}

// one CTA per row; GAUSS: nc, nf Gaussians of c and f are kept in shared memory (a form of its own: the
// unused branches alone cost the variable-coefficient paths 4 of 16 ms; 4, 3 and 2 CTAs an SM take 49.0,
// 48.8 and 51.9 ms on the Gaussians' case)
template <bool KILL, bool SRC, bool CV, bool GAUSS>
__global__ void __launch_bounds__(kRowThreads, GAUSS ? 3 : 0) k_paths(Problem P, PathArgs A, int nc, int nf) {
    extern __shared__ __align__(16) unsigned char psm32[];
    GaussTab gc{}, gf{};
    if (GAUSS && KILL && nc) gc = stage_gauss(reinterpret_cast<float4 *>(psm32), P.rbf32, nc, P.rbf_inv2s2);
    if (GAUSS && SRC && nf)
        gf = stage_gauss(reinterpret_cast<float4 *>(psm32 + (nc ? gauss_smem(nc) : 0)), P.frbf32, nf, P.frbf_inv2s2);
    using R = float;
    __shared__ int next_path;
    const int slot = blockIdx.x;
    const int gsl = A.gslot ? A.gslot[slot] : slot;
    const int i = A.rows[slot], m = A.subs[gsl];
    const uint32_t kw = A.kword ? (uint32_t)A.kword[gsl] : 0u;
    const double rad = A.cr[m], ts = A.theta_s[m];
    // exit tests against the disk and the domain shrunk by the boundary shift (0: the true ones), in
    // the position type; computed once into shared memory so that the loop reads them instead of
    // recomputing FP64 expressions: circle centre, r^2, r, the square's (x0, y0, x1, y1) or the
    // disk domain's (cx, cy, R) and R^2, the starting point and the step constants
    __shared__ R kc[14];
    if (threadIdx.x == 0) {
        const double rs = rad - A.shift, sft = A.shift;
        const bool sqd = P.dom_kind == 0;
        kc[0] = (R)A.ccx[m];
        kc[1] = (R)A.ccy[m];
        kc[2] = (R)(rs * rs);
        kc[3] = (R)rs;
        kc[4] = (R)(sqd ? P.dom[0] + sft : P.dom[0]);
        kc[5] = (R)(sqd ? P.dom[1] + sft : P.dom[1]);
        kc[6] = (R)(P.dom[2] - sft);
        kc[7] = (R)(P.dom[3] - sft);
        kc[8] = (R)((P.dom[2] - sft) * (P.dom[2] - sft));
        kc[9] = (R)A.kx[i];
        kc[10] = (R)A.ky[i];
        kc[11] = (R)A.h;
        kc[12] = Num<R>::sq((R)A.h);
        kc[13] = (R)ts;
    }
    __syncthreads();
    const R rcx = kc[0], rcy = kc[1], r2 = kc[2];
    const int max_steps = A.max_steps > 0 ? A.max_steps : (int)fmin(2147483647.0, ceil(50.0 * rad * rad / A.h));
    const R h = kc[11], sh = kc[12];
    const float hf = (float)kc[11];
    const bool sq_dom = P.dom_kind == 0;
    const R d0 = kc[4], d1 = kc[5], d2 = kc[6], d3 = kc[7];
    const R dr2 = kc[8];
    const R x_start = kc[9], y_start = kc[10];
    const int npath = A.npaths ? A.npaths[slot] : A.paths;
    const long rbase = A.rec_off ? A.rec_off[slot] : (long)slot * A.paths;
    unsigned long long my_steps = 0;
    int my_capped = 0;
    if (threadIdx.x == 0) next_path = blockDim.x;
    __syncthreads();
    // One loop iteration is one Euler-Maruyama step of this lane's current path; a lane whose
    // path exits writes its record and starts its next path (the row's next free path id) in
    // the same iteration, so the lanes of a warp stay converged whatever the path lengths.
    int p = threadIdx.x;
    R x = x_start, y = y_start;
    R cq[kMaxCv];
#pragma unroll
    for (int q = 0; q < kMaxCv; ++q) cq[q] = (R)0;
    const R crad = (R)rad;
    double Yv = 1.0, Zv = 0.0;
    float e = 0.f, z = 0.f;    // mixed form: Y = Yv (1 + e), Z = Zv + Yv z (FP32 block increments)
    int k = 0;
    unsigned it = 0;           // loop iterations, equal in all active lanes
    while (p < npath) {
        const long rec = rbase + p;
        bool done = false;
        if (k >= max_steps) {
            A.side[rec] = 2;
            A.su[rec] = 0.0;
            A.Y[rec] = 0.0;
            A.Z[rec] = 0.0;
            A.ez[rec] = make_float2(0.f, 0.f);
            if constexpr (CV)
                for (int q = 0; q < A.ncv; ++q) A.cvq[rec * A.ncv + q] = 0.0;
            ++my_capped;
            done = true;
        } else {
            R xi0, xi1;
            Num<R>::normals(A.seed, (uint32_t)i, kw, (uint32_t)k, (uint32_t)p, xi0, xi1);
            if constexpr (CV) {
                // Y_k sqrt(h) grad psi(X_k) . xi_k / r, with Y_k the weight before this step
                const R yk = (float)Yv * (1.0f + e);
                cv_accumulate<R>(cq, A.cvd, (x - rcx) / crad, (y - rcy) / crad, yk * sh / crad, xi0, xi1);
            }
            R bx, by;
            Num<R>::drift(P, x, y, bx, by);
            double Yn = Yv, Zn = Zv;
            float en = e, zn = z;
            float cv = 0.f;
            if (KILL) {
                if (GAUSS && nc) {
                    const float s = gauss_sum(gc, x, y);
                    cv = s < 0.f ? s : 0.f;
                } else {
                    cv = killing32(P, x, y);
                }
            }
            // Z_{k+1} = Z_k + f_k h Y_k and Y_{k+1} = Y_k (1 + c_k h), with Y_k = Yv (1 + e)
            if (SRC) zn = fmaf((GAUSS && nf ? gauss_sum(gf, x, y) : source32_given(P, x, y, bx, by, cv)) * hf, 1.0f + e, z);
            if (KILL) en = fmaf(cv * hf, 1.0f + e, e);
            const R nx = x + bx * h + sh * xi0;
            const R ny = y + by * h + sh * xi1;
            ++k;
            const R ddx = nx - rcx, ddy = ny - rcy;
            const bool out_c = !(ddx * ddx + ddy * ddy < r2);
            bool in_d;
            if (P.dom_kind == 0) {
                in_d = nx > d0 && nx < d2 && ny > d1 && ny < d3;
            } else {
                const R ex0 = nx - d0, ey0 = ny - d1;
                in_d = ex0 * ex0 + ey0 * ey0 < dr2;
            }
            const bool out_d = !in_d;
            // fold the FP32 increments into the FP64 weights every 8 iterations of the loop (the
            // same iterations in every lane of the warp, so the FP64 work is not divergent); the
            // increments left at the exit go to the record and the finalize folds them
            if ((++it & 7) == 0) {
                Zn = fma(Yv, (double)zn, Zv);
                Yn = fma(Yv, (double)en, Yv);
                en = 0.f;
                zn = 0.f;
            }
            if (!out_c && !out_d) {
                x = nx;
                y = ny;
                Yv = Yn;
                Zv = Zn;
                e = en;
                z = zn;
            } else {
                // exit point on the segment, in FP32; with
                // the boundary shift the piece crossed first (on the shrunk boundaries) is scored at the
                // projection of the first point outside onto the true boundary
                const R dx = nx - x, dy = ny - y;
                R tc = (R)2, td = (R)2;
                int ed = -1;
                if (out_c) tc = circle_exit_tr<R>(x, y, dx, dy, rcx, rcy, kc[3]);
                if (out_d) {
                    if (sq_dom) {
                        R t;
                        if (nx <= d0) { t = (d0 - x) / dx; if (t < td) { td = t; ed = 3; } }
                        if (nx >= d2) { t = (d2 - x) / dx; if (t < td) { td = t; ed = 1; } }
                        if (ny <= d1) { t = (d1 - y) / dy; if (t < td) { td = t; ed = 0; } }
                        if (ny >= d3) { t = (d3 - y) / dy; if (t < td) { td = t; ed = 2; } }
                    } else {
                        td = circle_exit_tr<R>(x, y, dx, dy, d0, d1, d2);
                        ed = 0;
                    }
                }
                const bool proj = A.shift > 0.0;
                if (td <= tc) {
                    R ex = x + td * dx, ey = y + td * dy;
                    if (proj) {
                        ex = nx;
                        ey = ny;
                        if (sq_dom) {
                            const R x0 = (R)P.dom[0], y0 = (R)P.dom[1], x1 = (R)P.dom[2], y1 = (R)P.dom[3];
                            ex = ex < x0 ? x0 : (ex > x1 ? x1 : ex);
                            ey = ey < y0 ? y0 : (ey > y1 ? y1 : ey);
                            if (ed == 0) ey = y0;
                            else if (ed == 1) ex = x1;
                            else if (ed == 2) ey = y1;
                            else ex = x0;
                        }                                  // disk domain: the arclength is the angle's
                    }
                    A.side[rec] = 1;
                    A.su[rec] = boundary_s(P, (double)ex, (double)ey, ed);
                } else {
                    const R ex = proj ? nx : x + tc * dx, ey = proj ? ny : y + tc * dy;
                    R th = atan2(ey - rcy, ex - rcx);
                    const R two_pi = (R)PDD_TWO_PI;
                    if (th < (R)0) th += two_pi;
                    R u = th - kc[13];
                    if (u < (R)0) u += two_pi;
                    if (u >= two_pi) u -= two_pi;
                    A.side[rec] = 0;
                    A.su[rec] = (double)u;
                }
                A.Y[rec] = Yn;
                A.Z[rec] = Zn;
                A.ez[rec] = make_float2(en, zn);
                if constexpr (CV) {
#pragma unroll
                    for (int q = 0; q < kMaxCv; ++q)
                        if (q < A.ncv) A.cvq[rec * A.ncv + q] = (double)cq[q];
                }
                done = true;
            }
        }
        if (done) {
            my_steps += (unsigned long long)k;
            p = atomicAdd(&next_path, 1);
            x = x_start;
            y = y_start;
            Yv = 1.0;
            Zv = 0.0;
            e = 0.f;
            z = 0.f;
            k = 0;
            if constexpr (CV) {
#pragma unroll
                for (int q = 0; q < kMaxCv; ++q) cq[q] = (R)0;
            }
        }
    }
    // block totals
    __shared__ unsigned long long ss[8];
    __shared__ int sc[8];
    for (int o = 16; o; o >>= 1) {
        my_steps += __shfl_xor_sync(0xffffffffu, my_steps, o);
        my_capped += __shfl_xor_sync(0xffffffffu, my_capped, o);
    }
    if ((threadIdx.x & 31) == 0) {
        ss[threadIdx.x >> 5] = my_steps;
        sc[threadIdx.x >> 5] = my_capped;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        int c = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            t += ss[w];
            c += sc[w];
        }
        atomicAdd(A.steps, t);
        if (c) atomicAdd(A.capped, c);
    }
}

template <bool KILL, bool SRC, int CVD>
__global__ void __launch_bounds__(kP32Threads) k_paths_long(Problem P, PathArgs A, Pool32 Q) {
    constexpr unsigned kAll = 0xffffffffu;
    constexpr bool CV = CVD != 0;
    extern __shared__ __align__(16) unsigned char psm32[];
    const Env32 E = env32<KILL, SRC>(P, A, Q, psm32);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const unsigned nchunks = (unsigned)((Q.total + kP32Chunk - 1) / kP32Chunk);
    unsigned long long my_steps = 0;
    int my_capped = 0;
    // this warp's records still to start: [q_next, q_end), the first of them in slot q_slot
    long q_next = 0, q_end = 0;
    int q_slot = 0;
    bool drained = false, have = false;
    long rec = 0;
    int p = 0, knot = 0, max_steps = 0;
    uint32_t kw = 0;
    float cx = 0.f, cy = 0.f, r2 = 0.f, crad = 1.f, rcrad = 1.f;
    Path32 S{0.f, 0.f, 0.f, 0.f, 1.0, 0.0, 0};
    float cq[CV ? kMaxCv : 1];
    unsigned it = 0;           // loop iterations, equal in all lanes
    for (;;) {
        // free lanes take the next records, in lane order
        unsigned idle = __ballot_sync(kAll, !have);
        while (idle) {
            if (q_next >= q_end) {
                if (drained) break;
                unsigned c = 0;
                int sl = 0;
                if (lane == 0) {
                    c = atomicAdd(Q.next, 1u);
                    if (c < nchunks) sl = slot_of(A, Q.slots, Q.nslots, (long)c * kP32Chunk);
                }
                c = __shfl_sync(kAll, c, 0);
                q_slot = __shfl_sync(kAll, sl, 0);
                if (c >= nchunks) {
                    drained = true;
                    break;
                }
                q_next = (long)c * kP32Chunk;
                q_end = min(Q.total, q_next + kP32Chunk);
            }
            const long g = q_next + __popc(idle & below);
            if (!have && g < q_end) {
                int sl = q_slot;
                while (sl + 1 < Q.nslots && Q.slots[sl + 1].rbase <= g) ++sl;
                const Slot32 *L = Q.slots + sl;
                have = true;
                rec = g;
                p = (int)(g - L->rbase);
                S = Path32{L->x0, L->y0, 0.f, 0.f, 1.0, 0.0, 0};
                cx = L->cx;
                cy = L->cy;
                r2 = L->r2;
                knot = L->i;
                max_steps = L->max_steps;
                kw = L->kw;
                if constexpr (CV) {
                    crad = L->rad;
                    rcrad = 1.0f / crad;
#pragma unroll
                    for (int q = 0; q < kMaxCv; ++q) cq[q] = 0.f;
                }
            }
            q_next = min(q_end, q_next + __popc(idle));
            idle = __ballot_sync(kAll, !have);
        }
        if (idle == kAll) break;
        ++it;
        if (!have) continue;
        if (S.k >= max_steps) {
            record_capped<CV>(A, rec);
            ++my_capped;
            have = false;
        } else {
            float nx, ny;
            if (step32<KILL, SRC, CVD>(P, A, Q, E, S, knot, kw, p, cx, cy, r2, crad, rcrad, cq, (it & 7) == 0, nx, ny)) {
                record_exit<CV>(A, Q, rec, S, nx, ny, cq);
                have = false;
            }
        }
        if (!have) my_steps += (unsigned long long)S.k;
    }
    add_totals(A, my_steps, my_capped);
}

// The exit point of every record's last segment, in FP32: the first crossing with the circle or the
// domain's boundary (both shrunk by the boundary shift); with the shift the piece crossed first is
// scored at the projection of the first point outside onto the true boundary
__global__ void __launch_bounds__(256) k_exit32(Problem P, PathArgs A, Pool32 Q) {
    const long rec = blockIdx.x * 256L + threadIdx.x;
    if (rec >= Q.total || A.side[rec] != 3) return;
    const int slot = slot_of(A, Q.slots, Q.nslots, rec);
    const Slot32 *S = Q.slots + slot;
    const bool sq_dom = P.dom_kind == 0;
    const double sft = A.shift;
    const float d0 = (float)(sq_dom ? P.dom[0] + sft : P.dom[0]), d1 = (float)(sq_dom ? P.dom[1] + sft : P.dom[1]);
    const float d2 = (float)(P.dom[2] - sft), d3 = (float)(P.dom[3] - sft);
    const float dr2 = (float)((P.dom[2] - sft) * (P.dom[2] - sft));
    const float rcx = S->cx, rcy = S->cy, r2 = S->r2;
    const float4 s = Q.seg[rec];
    const float x = s.x, y = s.y, nx = s.z, ny = s.w;
    const float ddx = nx - rcx, ddy = ny - rcy;
    const bool out_c = !(ddx * ddx + ddy * ddy < r2);
    bool out_d;
    if (sq_dom) {
        out_d = !(nx > d0 && nx < d2 && ny > d1 && ny < d3);
    } else {
        const float ex0 = nx - d0, ey0 = ny - d1;
        out_d = !(ex0 * ex0 + ey0 * ey0 < dr2);
    }
    const float dx = nx - x, dy = ny - y;
    float tc = 2.f, td = 2.f;
    int ed = -1;
    if (out_c) tc = circle_exit_tr<float>(x, y, dx, dy, rcx, rcy, S->rs);
    if (out_d) {
        if (sq_dom) {
            float t;
            if (nx <= d0) { t = (d0 - x) / dx; if (t < td) { td = t; ed = 3; } }
            if (nx >= d2) { t = (d2 - x) / dx; if (t < td) { td = t; ed = 1; } }
            if (ny <= d1) { t = (d1 - y) / dy; if (t < td) { td = t; ed = 0; } }
            if (ny >= d3) { t = (d3 - y) / dy; if (t < td) { td = t; ed = 2; } }
        } else {
            td = circle_exit_tr<float>(x, y, dx, dy, d0, d1, d2);
            ed = 0;
        }
    }
    const bool proj = A.shift > 0.0;
    if (td <= tc) {
        float ex = x + td * dx, ey = y + td * dy;
        if (proj) {
            ex = nx;
            ey = ny;
            if (sq_dom) {
                const float x0 = (float)P.dom[0], y0 = (float)P.dom[1], x1 = (float)P.dom[2], y1 = (float)P.dom[3];
                ex = ex < x0 ? x0 : (ex > x1 ? x1 : ex);
                ey = ey < y0 ? y0 : (ey > y1 ? y1 : ey);
                if (ed == 0) ey = y0;
                else if (ed == 1) ex = x1;
                else if (ed == 2) ey = y1;
                else ex = x0;
            }                                             // disk domain: the arclength is the angle's
        }
        A.side[rec] = 1;
        A.su[rec] = boundary_s(P, (double)ex, (double)ey, ed);
    } else {
        const float ex = proj ? nx : x + tc * dx, ey = proj ? ny : y + tc * dy;
        float th = atan2f(ey - rcy, ex - rcx);
        const float two_pi = (float)PDD_TWO_PI;
        if (th < 0.f) th += two_pi;
        float u = th - S->ts;
        if (u < 0.f) u += two_pi;
        if (u >= two_pi) u -= two_pi;
        A.side[rec] = 0;
        A.su[rec] = (double)u;
    }
}

// ---------------------------------------------------------------------------
// FP64 form.  The FP64 pipe bounds it (1/64 of the FP32 rate: a warp instruction occupies an SM's
// unit for 16 cycles whatever the number of its lanes in use), so the design keeps the lanes full
// and takes FP64 instructions out of the step, with every value rounded as the plain expressions are:
//   * persistent warps; a lane whose path exits takes the launch's next path, of whatever row (rows
//     of unequal path lengths or fewer rows than SMs leave nothing idle);
//   * when the queue is empty, a warp with few paths left hands their states over and ends; the next
//     launch packs them into full warps (four launches, the last runs to completion);
//   * without drift, and with killing and source zero or by Gaussians, the second launch is k_walk64,
//     which finishes what the first hands over: the longest path's steps, one after the other, are the end
//     of the launch, so eight lanes take a path, form the normals of eight steps at once (they depend on
//     the step's number alone) and share a step's Gaussians;
//   * the exit point of a path (roots, divisions, an arctangent) is left to k_exit64, one thread per
//     record, instead of being computed by one lane while 31 wait;
//   * the uniforms are put together from their bits, the comparisons with the domain's box are integer
//     comparisons, the circle is tested in FP32 first.
// 4 x 4 lattice (116 rows x 1,000 paths): 9.4 -> 3.2 ms (6.1 without k_walk64), with 64 Gaussians of c
// and 16 of f 159 -> 61 ms (110); 140 circles with variable coefficients, 10^4
// paths a row: 325 -> 189 ms.
// ---------------------------------------------------------------------------
struct alignas(16) Slot64 {          // what a path reads when it starts
    double cx, cy, r, r2, x0, y0;    // r2: of the disk shrunk by the boundary shift
    long rbase;
    int i, max_steps;
    uint32_t kw;
};
struct alignas(16) PathState {
    double x, y, Y, Z;
    int slot, p, k, pad;
};
struct alignas(16) Seg64 {
    double x, y, nx, ny;
};
struct PathPool {
    const Slot64 *slots;
    int nslots;
    unsigned long long total;        // paths of the launch (first pass)
    unsigned long long *next;        // queue position
    const PathState *in;             // states handed over by the previous pass (null: first pass)
    const unsigned *n_in;
    PathState *out;                  // and by this one
    unsigned *n_out;
    int keep;                        // fewer live paths than this in a warp are handed over (0: none are)
    const double *cq_in;             // control-variate features of the states, [state][ncv]
    double *cq_out;
    Seg64 *seg;                      // per record: the last step's segment
};

static constexpr int kP64Threads = 64;
static constexpr int kP64WarpsPerSm = 8;
static constexpr int kP64Staged = 1024;        // most Gaussians kept in shared memory (24 KB)

__global__ void k_slots64(int n, PathArgs A, Slot64 *out) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= n) return;
    const int gsl = A.gslot ? A.gslot[slot] : slot;
    const int i = A.rows[slot], m = A.subs[gsl];
    const double rad = A.cr[m], rs = rad - A.shift;
    Slot64 s;
    s.cx = A.ccx[m];
    s.cy = A.ccy[m];
    s.r = rad;
    s.r2 = rs * rs;
    s.x0 = A.kx[i];
    s.y0 = A.ky[i];
    s.rbase = A.rec_off ? A.rec_off[slot] : (long)slot * A.paths;
    s.i = i;
    s.max_steps = A.max_steps > 0 ? A.max_steps : (int)fmin(2147483647.0, ceil(50.0 * rad * rad / A.h));
    s.kw = A.kword ? (uint32_t)A.kword[gsl] : 0u;
    out[slot] = s;
}

// an order-preserving integer of a double (-0 below +0; no NaN)
__device__ __forceinline__ long long order_key(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

// the leading 24 bits of a double as FP32, for |v| in [2^-126, 2^128); beside that range an arbitrary value,
// infinity and NaN among them.  In the circle's pre-test a displacement below it can only send the step to the
// FP64 comparison (its square may come out too large, never too small), one above it is tested for.
__device__ __forceinline__ float trunc32(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    return __uint_as_float(((__funnelshift_l(lo, hi, 3) ^ 0x40000000u) & 0x7fffffffu) | (hi & 0x80000000u));
}

template <bool KILL, bool SRC, bool CV>
__global__ void __launch_bounds__(kP64Threads) k_paths64(Problem P, PathArgs A, PathPool Q) {
    constexpr unsigned kAll = 0xffffffffu;
    // killing by Gaussians: exp_neg's table, then x, y, w (in global memory when they are many)
    extern __shared__ __align__(16) double psm64[];
    const double2 *etab = reinterpret_cast<const double2 *>(psm64);
    const int nr = KILL && P.c_kind == PDD_C_RBF ? P.n_rbf : 0;
    const bool staged = nr <= kP64Staged;
    const double *rx = staged ? psm64 + 2 * kExpTab : P.rbf_x, *ry = staged ? rx + nr : P.rbf_y;
    const double *rw = staged ? ry + nr : P.rbf_w;
    const double inv2s = nr ? 1.0 / (2.0 * P.rbf_sigma * P.rbf_sigma) : 0.0;
    if (nr) {
        double2 *et = reinterpret_cast<double2 *>(psm64);
        double *rt = psm64 + 2 * kExpTab;
        for (int q = threadIdx.x; q < kExpTab; q += kP64Threads) et[q] = kExp2Tab[q];
        for (int q = threadIdx.x; staged && q < nr; q += kP64Threads) {
            rt[q] = P.rbf_x[q];
            rt[nr + q] = P.rbf_y[q];
            rt[2 * nr + q] = P.rbf_w[q];
        }
        __syncthreads();
    }
    const bool sq_dom = P.dom_kind == 0, has_b = P.b_kind != PDD_B_ZERO;
    const double sft = A.shift;
    const double d0 = sq_dom ? P.dom[0] + sft : P.dom[0], d1 = sq_dom ? P.dom[1] + sft : P.dom[1];
    const double d2 = P.dom[2] - sft, d3 = P.dom[3] - sft;
    const double dr2 = (P.dom[2] - sft) * (P.dom[2] - sft);
    const long long q0 = order_key(d0 + 0.0), q1 = order_key(d1 + 0.0), q2 = order_key(d2), q3 = order_key(d3);
    const double h = A.h, sh = sqrt(A.h);
    const unsigned long long total = Q.in ? (unsigned long long)*Q.n_in : Q.total;
    unsigned long long my_steps = 0;
    int my_capped = 0;
    bool have = false, drained = false;
    double x = 0.0, y = 0.0, Yv = 1.0, Zv = 0.0, cx = 0.0, cy = 0.0, r2 = 0.0, crad = 1.0;
    float r2f = 0.f;
    long rec = 0;
    int slot = 0, p = 0, k = 0, knot = 0, max_steps = 0;
    uint32_t kw = 0;
    double cq[CV ? kMaxCv : 1];
    for (;;) {
        if (!have && !drained) {
            const unsigned long long g = atomicAdd(Q.next, 1ULL);
            drained = g >= total;
            if (!drained) {
                have = true;
                if (Q.in) {
                    const PathState s = Q.in[g];
                    slot = s.slot;
                    p = s.p;
                    k = s.k;
                    x = s.x;
                    y = s.y;
                    Yv = s.Y;
                    Zv = s.Z;
                } else {
                    slot = slot_of(A, Q.slots, Q.nslots, (long)g);
                    p = (int)(g - (unsigned long long)Q.slots[slot].rbase);
                    k = 0;
                    x = Q.slots[slot].x0;
                    y = Q.slots[slot].y0;
                    Yv = 1.0;
                    Zv = 0.0;
                }
                const Slot64 *S = Q.slots + slot;
                cx = S->cx;
                cy = S->cy;
                if (CV) crad = S->r;
                r2 = S->r2;
                r2f = (float)r2 * 0.9999f;
                rec = S->rbase + p;
                knot = S->i;
                max_steps = S->max_steps;
                kw = S->kw;
                if constexpr (CV) {
#pragma unroll
                    for (int q = 0; q < kMaxCv; ++q) cq[q] = (Q.in && q < A.ncv) ? Q.cq_in[g * A.ncv + q] : 0.0;
                }
            }
        }
        const unsigned live = __ballot_sync(kAll, have);
        if (__popc(live) < Q.keep || !live) {             // (below `keep` only once the queue is empty)
            if (have) {
                const unsigned o = atomicAdd(Q.n_out, 1u);
                Q.out[o] = PathState{x, y, Yv, Zv, slot, p, k, 0};
                if constexpr (CV) {
#pragma unroll
                    for (int q = 0; q < kMaxCv; ++q)
                        if (q < A.ncv) Q.cq_out[(size_t)o * A.ncv + q] = cq[q];
                }
            }
            break;
        }
        if (!have) continue;
        if (k >= max_steps) {
            A.side[rec] = 2;
            A.su[rec] = 0.0;
            A.Y[rec] = 0.0;
            A.Z[rec] = 0.0;
            if constexpr (CV)
                for (int q = 0; q < A.ncv; ++q) A.cvq[rec * A.ncv + q] = 0.0;
            ++my_capped;
            my_steps += (unsigned long long)k;
            have = false;
            continue;
        }
        double xi0, xi1;
        normals64(A.seed, (uint32_t)knot, kw, (uint32_t)k, (uint32_t)p, xi0, xi1);
        if constexpr (CV) {
            // Y_k sqrt(h) grad psi(X_k) . xi_k / r, with Y_k the weight before this step
            cv_accumulate<double>(cq, A.cvd, (x - cx) / crad, (y - cy) / crad, Yv * sh / crad, xi0, xi1);
        }
        double bx = 0.0, by = 0.0;
        if (has_b) drift(P, x, y, bx, by);
        double Yn = Yv, Zn = Zv, cv = 0.0;
        if (KILL) {
            if (nr) {
                double s = 0.0;
#pragma unroll 4
                for (int q = 0; q < nr; ++q) {
                    const double dx = x - rx[q], dy = y - ry[q];
                    s += rw[q] * exp_neg(-(dx * dx + dy * dy) * inv2s, etab);
                }
                cv = s < 0.0 ? s : 0.0;
            } else {
                cv = killing(P, x, y);
            }
            Yn = Yv * (1.0 + cv * A.h);
        }
        if (SRC) Zn = Zv + source_given(P, x, y, bx, by, cv) * Yv * A.h;
        const double nx = has_b ? x + bx * h + sh * xi0 : x + sh * xi0;
        const double ny = has_b ? y + by * h + sh * xi1 : y + sh * xi1;
        ++k;
        const double ddx = nx - cx, ddy = ny - cy;
        const float fx = trunc32(ddx), fy = trunc32(ddy);
        // surely inside below 0.9999 r^2 (the FP32 sum is off by 2^-21), for |ddx| and |ddy| below 2^49
        const unsigned top = max((unsigned)__double2hiint(ddx) & 0x7fffffffu, (unsigned)__double2hiint(ddy) & 0x7fffffffu);
        bool out = !(fx * fx + fy * fy < r2f && top < 0x43000000u);
        if (out) out = !(ddx * ddx + ddy * ddy < r2);
        if (sq_dom) {
            const long long kx = order_key(nx), ky = order_key(ny);
            out = out || !(kx > q0 && kx < q2 && ky > q1 && ky < q3);
        } else {
            const double ex0 = nx - d0, ey0 = ny - d1;
            out = out || !(ex0 * ex0 + ey0 * ey0 < dr2);
        }
        if (!out) {
            x = nx;
            y = ny;
            Yv = Yn;
            Zv = Zn;
            continue;
        }
        A.side[rec] = 3;                                  // k_exit64 finds the side and the exit point
        Q.seg[rec] = Seg64{x, y, nx, ny};
        A.Y[rec] = Yn;
        A.Z[rec] = Zn;
        if constexpr (CV) {
#pragma unroll
            for (int q = 0; q < kMaxCv; ++q)
                if (q < A.ncv) A.cvq[rec * A.ncv + q] = cq[q];
        }
        my_steps += (unsigned long long)k;
        have = false;
    }
    for (int o = 16; o; o >>= 1) {
        my_steps += __shfl_xor_sync(kAll, my_steps, o);
        my_capped += __shfl_xor_sync(kAll, my_capped, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (my_steps) atomicAdd(A.steps, my_steps);
        if (my_capped) atomicAdd(A.capped, my_capped);
    }
}

// The paths of Q.in to their ends, b = 0, c and f zero or by Gaussians: eight lanes per path.  They form
// the normals of the next eight steps one each; a step then runs in all of them alike, but for the
// exponentials of its Gaussians, of which each lane takes every eighth (added up in their order).
static constexpr int kWalkLanes = 8;
__device__ __forceinline__ double from_lane(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }

// sum_q w_q e(q), e evaluated by lane q mod 8 of the group that starts at lane `lead`
template <typename Eval>
__device__ __forceinline__ double walk_sum(int n, const double *w, int lead, int gl, Eval eval) {
    constexpr int B = 4;
    double s = 0.0;
    for (int q0 = 0; q0 < n; q0 += B * kWalkLanes) {
        double e[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int q = q0 + b * kWalkLanes + gl;
            e[b] = q < n ? eval(q) : 0.0;
        }
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
            for (int i = 0; i < kWalkLanes; ++i) {
                const int q = q0 + b * kWalkLanes + i;
                const double v = from_lane(e[b], lead + i);
                if (q < n) s += w[q] * v;
            }
    }
    return s;
}

template <bool KILL, bool SRC>
__global__ void __launch_bounds__(kP64Threads) k_walk64(Problem P, PathArgs A, PathPool Q) {
    extern __shared__ __align__(16) double psm64[];       // killing: exp_neg's table, then x, y, w as in k_paths64
    const double2 *etab = reinterpret_cast<const double2 *>(psm64);
    const int nr = KILL ? P.n_rbf : 0, nf = SRC ? P.n_frbf : 0;
    const bool staged = nr <= kP64Staged;
    const double *rx = staged ? psm64 + 2 * kExpTab : P.rbf_x, *ry = staged ? rx + nr : P.rbf_y;
    const double *rw = staged ? ry + nr : P.rbf_w;
    const double inv2s = KILL ? 1.0 / (2.0 * P.rbf_sigma * P.rbf_sigma) : 0.0;
    const double finv = SRC ? 1.0 / (2.0 * P.frbf_sigma * P.frbf_sigma) : 0.0;
    if (KILL) {
        double2 *et = reinterpret_cast<double2 *>(psm64);
        double *rt = psm64 + 2 * kExpTab;
        for (int q = threadIdx.x; q < kExpTab; q += kP64Threads) et[q] = kExp2Tab[q];
        for (int q = threadIdx.x; staged && q < nr; q += kP64Threads) {
            rt[q] = P.rbf_x[q];
            rt[nr + q] = P.rbf_y[q];
            rt[2 * nr + q] = P.rbf_w[q];
        }
        __syncthreads();
    }
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, gl = lane & (kWalkLanes - 1), lead = lane - gl;
    const bool sq_dom = P.dom_kind == 0;
    const double sft = A.shift;
    const double d0 = sq_dom ? P.dom[0] + sft : P.dom[0], d1 = sq_dom ? P.dom[1] + sft : P.dom[1];
    const double d2 = P.dom[2] - sft, d3 = P.dom[3] - sft;
    const double dr2 = (P.dom[2] - sft) * (P.dom[2] - sft);
    const long long q0 = order_key(d0 + 0.0), q1 = order_key(d1 + 0.0), q2 = order_key(d2), q3 = order_key(d3);
    const double sh = sqrt(A.h);
    const unsigned total = *Q.n_in;
    unsigned long long my_steps = 0;
    int my_capped = 0;
    bool have = false, drained = false;
    double x = 0.0, y = 0.0, cx = 0.0, cy = 0.0, r2 = 0.0, Yv = 1.0, Zv = 0.0;
    float r2f = 0.f;
    long rec = 0;
    int p = 0, k = 0, knot = 0, max_steps = 0;
    uint32_t kw = 0;
    for (;;) {
        unsigned g = 0;
        if (!have && !drained && gl == 0) g = (unsigned)min(atomicAdd(Q.next, 1ULL), (unsigned long long)total);
        g = __shfl_sync(kAll, g, lead);
        if (!have && !drained) {
            drained = g >= total;
            if (!drained) {
                const PathState s = Q.in[g];
                const Slot64 *S = Q.slots + s.slot;
                have = true;
                p = s.p;
                k = s.k;
                x = s.x;
                y = s.y;
                Yv = s.Y;
                Zv = s.Z;
                cx = S->cx;
                cy = S->cy;
                r2 = S->r2;
                r2f = (float)r2 * 0.9999f;
                rec = S->rbase + p;
                knot = S->i;
                max_steps = S->max_steps;
                kw = S->kw;
            }
        }
        if (!__ballot_sync(kAll, have)) break;
        double z0 = 0.0, z1 = 0.0;
        if (have) normals64(A.seed, (uint32_t)knot, kw, (uint32_t)(k + gl), (uint32_t)p, z0, z1);
        for (int j = 0; j < kWalkLanes; ++j) {
            const double xi0 = from_lane(z0, lead + j), xi1 = from_lane(z1, lead + j);
            double cv = 0.0, fv = 0.0;
            if (KILL || SRC) {
                if (!__ballot_sync(kAll, have)) break;
                if (KILL) {
                    const double sum = walk_sum(nr, rw, lead, gl, [&](int q) {
                        const double dx = x - rx[q], dy = y - ry[q];
                        return exp_neg(-(dx * dx + dy * dy) * inv2s, etab);
                    });
                    cv = sum < 0.0 ? sum : 0.0;
                }
                if (SRC)
                    fv = walk_sum(nf, P.frbf_w, lead, gl, [&](int q) {
                        const double dx = x - P.frbf_x[q], dy = y - P.frbf_y[q];
                        return exp(-(dx * dx + dy * dy) * finv);
                    });
            }
            if (!have) continue;
            if (k >= max_steps) {
                if (gl == 0) {
                    A.side[rec] = 2;
                    A.su[rec] = 0.0;
                    A.Y[rec] = 0.0;
                    A.Z[rec] = 0.0;
                    ++my_capped;
                    my_steps += (unsigned long long)k;
                }
                have = false;
                continue;
            }
            if (SRC) Zv = Zv + fv * Yv * A.h;
            if (KILL) Yv = Yv * (1.0 + cv * A.h);
            const double nx = x + sh * xi0, ny = y + sh * xi1;
            ++k;
            const double ddx = nx - cx, ddy = ny - cy;
            const float fx = trunc32(ddx), fy = trunc32(ddy);
            const unsigned top =
                max((unsigned)__double2hiint(ddx) & 0x7fffffffu, (unsigned)__double2hiint(ddy) & 0x7fffffffu);
            bool out = !(fx * fx + fy * fy < r2f && top < 0x43000000u);
            if (out) out = !(ddx * ddx + ddy * ddy < r2);
            if (sq_dom) {
                const long long kx = order_key(nx), ky = order_key(ny);
                out = out || !(kx > q0 && kx < q2 && ky > q1 && ky < q3);
            } else {
                const double ex0 = nx - d0, ey0 = ny - d1;
                out = out || !(ex0 * ex0 + ey0 * ey0 < dr2);
            }
            if (!out) {
                x = nx;
                y = ny;
                continue;
            }
            if (gl == 0) {
                A.side[rec] = 3;
                Q.seg[rec] = Seg64{x, y, nx, ny};
                A.Y[rec] = Yv;
                A.Z[rec] = Zv;
                my_steps += (unsigned long long)k;
            }
            have = false;
        }
    }
    for (int o = 16; o; o >>= 1) {
        my_steps += __shfl_xor_sync(kAll, my_steps, o);
        my_capped += __shfl_xor_sync(kAll, my_capped, o);
    }
    if (lane == 0) {
        if (my_steps) atomicAdd(A.steps, my_steps);
        if (my_capped) atomicAdd(A.capped, my_capped);
    }
}

// the exit point of every record's last segment, as in k_paths (in FP64)
__global__ void __launch_bounds__(256) k_exit64(Problem P, PathArgs A, PathPool Q) {
    const unsigned long long rec = blockIdx.x * 256ULL + threadIdx.x;
    if (rec >= Q.total || A.side[rec] != 3) return;
    const int slot = slot_of(A, Q.slots, Q.nslots, (long)rec);
    const int m = A.subs[A.gslot ? A.gslot[slot] : slot];
    const bool sq_dom = P.dom_kind == 0;
    const double sft = A.shift;
    const double d0 = sq_dom ? P.dom[0] + sft : P.dom[0], d1 = sq_dom ? P.dom[1] + sft : P.dom[1];
    const double d2 = P.dom[2] - sft, d3 = P.dom[3] - sft;
    const double dr2 = (P.dom[2] - sft) * (P.dom[2] - sft);
    const double rcx = Q.slots[slot].cx, rcy = Q.slots[slot].cy, r2 = Q.slots[slot].r2, rs = A.cr[m] - sft;
    const Seg64 s = Q.seg[rec];
    const double x = s.x, y = s.y, nx = s.nx, ny = s.ny;
    const double ddx = nx - rcx, ddy = ny - rcy;
    const bool out_c = !(ddx * ddx + ddy * ddy < r2);
    bool out_d;
    if (sq_dom) {
        out_d = !(nx > d0 && nx < d2 && ny > d1 && ny < d3);
    } else {
        const double ex0 = nx - d0, ey0 = ny - d1;
        out_d = !(ex0 * ex0 + ey0 * ey0 < dr2);
    }
    const double dx = nx - x, dy = ny - y;
    double tc = 2.0, td = 2.0;
    int ed = -1;
    if (out_c) tc = circle_exit_t(x, y, dx, dy, rcx, rcy, rs);
    if (out_d) {
        if (sq_dom) {
            double t;
            if (nx <= d0) { t = (d0 - x) / dx; if (t < td) { td = t; ed = 3; } }
            if (nx >= d2) { t = (d2 - x) / dx; if (t < td) { td = t; ed = 1; } }
            if (ny <= d1) { t = (d1 - y) / dy; if (t < td) { td = t; ed = 0; } }
            if (ny >= d3) { t = (d3 - y) / dy; if (t < td) { td = t; ed = 2; } }
        } else {
            td = circle_exit_t(x, y, dx, dy, d0, d1, d2);
            ed = 0;
        }
    }
    const bool proj = A.shift > 0.0;
    if (td <= tc) {
        double ex = x + td * dx, ey = y + td * dy;
        if (proj) {
            ex = nx;
            ey = ny;
            if (sq_dom) {
                const double x0 = P.dom[0], y0 = P.dom[1], x1 = P.dom[2], y1 = P.dom[3];
                ex = ex < x0 ? x0 : (ex > x1 ? x1 : ex);
                ey = ey < y0 ? y0 : (ey > y1 ? y1 : ey);
                if (ed == 0) ey = y0;
                else if (ed == 1) ex = x1;
                else if (ed == 2) ey = y1;
                else ex = x0;
            }                                             // disk domain: the arclength is the angle's
        }
        A.side[rec] = 1;
        A.su[rec] = boundary_s(P, ex, ey, ed);
    } else {
        const double ex = proj ? nx : x + tc * dx, ey = proj ? ny : y + tc * dy;
        double th = atan2(ey - rcy, ex - rcx);
        if (th < 0.0) th += PDD_TWO_PI;
        double u = th - A.theta_s[m];
        if (u < 0.0) u += PDD_TWO_PI;
        if (u >= PDD_TWO_PI) u -= PDD_TWO_PI;
        A.side[rec] = 0;
        A.su[rec] = u;
    }
}

// ---------------------------------------------------------------------------
// a12
// ---------------------------------------------------------------------------
// Dirichlet data in FP32 (mixed form's boundary scores)
__device__ __forceinline__ float gdata32(const Problem &P, float x, float y, float s) {
    switch (P.g_kind) {
        case PDD_G_EXP_SIN: return expf(x) * sinf(y);
        case PDD_G_SIN_COS: return sinpif(x) * cospif(y);
        case PDD_G_BOUNDARY_FOURIER: {
            const int kc = (P.n_gcoef + 1) / 2, ks = P.n_gcoef - kc;
            const float w = s * (float)(2.0 / P.perimeter);
            float acc = 0.f;
            for (int k = 0; k < kc; ++k) acc += (float)P.g_coef[k] * cospif(k * w);
            for (int k = 1; k <= ks; ++k) acc += (float)P.g_coef[kc + k - 1] * sinpif(k * w);
            return acc;
        }
        case PDD_G_ONE: return 1.f;
        case PDD_G_EQ46: {
            float u, ux, uy, lap;
            u46_derivs(x, y, u, ux, uy, lap);
            return u;
        }
        default: return 0.f;
    }
}

// Fourier cardinal of a knot (Eq. 18) at angular distance t, closed form; out of line (Monte Carlo
// rows of floating circles only) for the same reason as boundary_score
__device__ __noinline__ double fourier_cardinal_at(double t, int n) {
    const double x = remainder(t, PDD_TWO_PI);
    return (x == 0.0) ? 1.0 : sin(0.5 * n * x) * cos(0.5 * x) / (sin(0.5 * x) * n);
}

// g at the boundary point of arclength s (FP32 data in the mixed form); kept out of line so that
// the data families do not add to the register pressure of the finalize loop (taken only for
// paths that exit through dOmega)
__device__ __noinline__ double boundary_score(const Problem &P, double s, int mixed) {
    double ex, ey;
    boundary_point(P, s, ex, ey);
    return mixed ? (double)gdata32(P, (float)ex, (float)ey, (float)s) : gdata(P, ex, ey, s);
}

struct FinalArgs {
    // per slot: the row i; per global slot gs: its subdomain and its entry p of sub_rows, whose
    // stencil block starts at rowptr[i] + sub_off[p] and whose part of r_i goes to bs[p]
    const int *rows, *subs, *spos, *sub_off, *knot_ptr, *rowptr;
    const uint8_t *floating;
    const double *ku;
    const long *kinv_off;     // per circle (-1 when not IMQ)
    const double *kinv;
    const double *kcond;      // per circle: kappa_1(K) (0 when not IMQ)
    double c2;
    int paths, mc_floating, mixed;
    const int *npaths;               // per-row path counts, or null (paths)
    const long *rec_off;             // per-row record offsets, or null (slot * paths)
    const int *gslot;                // index of the row in the system's Monte Carlo arrays, or null (slot)
    const int8_t *side;
    const double *su, *Y, *Z;
    const float2 *ez;                // mixed form: unfolded increments, Y (1 + e) and Z + Y z
    const int *mom_ptr;
    double *moments, *bmean, *val, *se, *bs, *se_bs;
    int sums;                        // PDD_SUMS_* of the mixed form (AUTO: by kappa_1(K))
    // regression control variate (null: none): per launched slot, beta [ns_max + 1][ncv] (the basis
    // moments' rows, then r's) and the per-batch feature sums [32][ncv]
    const double *cv_beta, *cv_sq;
    int ncv, cv_stride;              // features, beta rows per slot (the launch's largest stencil + 1)
};

// 1 / sqrt(q) for q = qh + ql in double-float: one Newton step from rsqrtf, whose residual
// t = 1 - q r0^2 is formed without rounding error in its leading part (r0^2 and q r0^2 by FMA
// splits; 1 - h is exact because h is within 2^-22 of 1); relative error below 1e-13
__device__ __forceinline__ float2 df_rsqrt(float qh, float ql) {
    const float r0 = rsqrtf(qh);
    const float a = __fmul_rn(r0, r0);
    const float ae = fmaf(r0, r0, -a);
    const float h = __fmul_rn(qh, a);
    float he = fmaf(qh, a, -h);
    he = fmaf(qh, ae, he);
    he = fmaf(ql, a, he);
    const float t = __fsub_rn(__fsub_rn(1.0f, h), he);
    return make_float2(r0, __fmul_rn(__fmul_rn(0.5f, r0), t));
}

// Per-row finalize.  NQ = register slices of 32 stencil knots (the launch's largest stencil).
// Basis sums of the mixed form (sum mode, per stencil):
//   0: FP32 phi and FP32 sums of 16 paths (kappa_1(K) <= kFastKappa);
//   1: double-float phi and sums (kappa_1(K) <= kDfKappa);
//   2: FP64 (the FP64 form, Fourier cardinals, and larger kappa).
// C = -K^-T M amplifies the rounding of the moments by up to kappa(K): FP32 sums of FP32 phi
// were measured off by ~5e-11 kappa in C (0.03 at kappa 5.6e8); double-float phi is within
// 1e-13 relative (an emulation over 2e4 random angles), FP64 within 2^-52.
template <int NQ>
__global__ void __launch_bounds__(512) k_mc_finalize(Problem P, FinalArgs F) {
    extern __shared__ double fsm[];                   // [32 batches][ns] moments, then per-batch C
    __shared__ double bsum[kBatches];
    __shared__ int bcnt[kBatches];
    const int slot = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gs = F.gslot ? F.gslot[slot] : slot;
    const int i = F.rows[slot], m = F.subs[gs], pe = F.spos[gs];
    const int a = F.knot_ptr[m], ns = F.knot_ptr[m + 1] - a;
    const bool imq = !F.floating[m];
    double *Mb = fsm;                                 // kBatches x ns
    double *Cb = fsm + kBatches * ns;                 // kBatches x ns
    const int npath = F.npaths ? F.npaths[slot] : F.paths;
    const long base = F.rec_off ? F.rec_off[slot] : (long)slot * F.paths;
    // this lane's stencil angles (IMQ) or knot angles (Fourier cardinals), also as hi + lo FP32
    double uk[NQ];
    float ukf[NQ], ukl[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int l = lane + 32 * q;
        uk[q] = (l < ns) ? (imq ? F.ku[a + l] : PDD_TWO_PI * l / ns) : 0.0;
        ukf[q] = (float)uk[q];
        ukl[q] = (float)(uk[q] - (double)ukf[q]);
    }
    const float c2f = (float)F.c2, c2l = (float)(F.c2 - (double)c2f);
    // a forced mode applies to either path form (FP64 records carry no FP32 increments); the
    // automatic choice keeps FP64 sums for FP64 paths
    int mode = 2;
    if (imq) {
        if (F.sums != PDD_SUMS_AUTO) mode = F.sums - 1;
        else if (F.mixed) mode = F.kcond[m] <= kFastKappa ? 0 : (F.kcond[m] <= kDfKappa ? 1 : 2);
    }
    const int nq = (ns + 31) >> 5;                     // slices holding stencil knots (block-uniform)
    for (int bt = warp; bt < kBatches; bt += 16) {         // 16 warps, two batches each (p mod 32)
        double acc[NQ];
        float accf[NQ], accl[NQ];                          // FP32 or double-float sums of 16 paths
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            acc[q] = 0.0;
            accf[q] = 0.f;
            accl[q] = 0.f;
        }
        int pend = 0;                                      // mode 0: paths in the FP32 sums since the last fold
        double bs = 0.0;
        int cnt = 0;
        // chunks of 32 paths of this batch: lane l loads path bt + 32 (t0 + l)
        for (int t0 = 0; bt + kBatches * t0 < npath; t0 += 32) {
            const int pl = bt + kBatches * (t0 + lane);
            int sd = 2;
            double yv = 0.0, zv = 0.0, su = 0.0;
            double yraw = 0.0;
            float ey = 0.f;                                // mixed form: the unfolded increment of Y
            if (pl < npath) {
                sd = F.side[base + pl];
                yraw = F.Y[base + pl];
                zv = F.Z[base + pl];
                su = F.su[base + pl];
                if (F.mixed) {
                    const float2 q = F.ez[base + pl];
                    zv = fma(yraw, (double)q.y, zv);
                    ey = q.x;
                }
            }
            // Y (1 + e) in FP64 where it is used in FP64: always, except for the double-float basis
            // sums, which need it only for a boundary score
            yv = yraw;
            if (F.mixed && ey != 0.f && (mode != 1 || sd == 1)) yv = fma(yraw, (double)ey, yraw);
            if (sd != 2) {                                 // this lane's own contribution to r_i
                ++cnt;
                if (sd == 1) {
                    bs += boundary_score(P, su, F.mixed) * yv + zv;
                } else {
                    bs += zv;
                }
            }
            // the chunk's interface exits, in path order, into every lane's basis sums
            if (mode == 0) {
                // each lane converts its own record once; FP32 values are shuffled
                const float yf = (float)yv, suf = (float)su;
                for (int src = 0; src < 32; ++src) {
                    const int s_sd = __shfl_sync(0xffffffffu, sd, src);
                    const float s_yf = __shfl_sync(0xffffffffu, yf, src);
                    const float s_suf = __shfl_sync(0xffffffffu, suf, src);
                    if (s_sd != 0) continue;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        if (q >= nq) break;                // slices past the stencil hold no knot
                        const float df = s_suf - ukf[q];
                        accf[q] = fmaf(s_yf, rsqrtf(df * df + c2f), accf[q]);
                    }
                    if (++pend == 16) {
#pragma unroll
                        for (int q = 0; q < NQ; ++q) {
                            acc[q] += (double)accf[q];
                            accf[q] = 0.f;
                        }
                        pend = 0;
                    }
                }
            } else if (mode == 1) {
                // double-float: the record's Y and angle split once per lane by integer operations
                // (no FP64 instruction), Y (1 + e) formed in double-float, then shuffled
                float2 y2 = split_df_bits(yraw);
                if (ey != 0.f) {
                    const float p = __fmul_rn(y2.x, ey);
                    float pe = fmaf(y2.x, ey, -p);
                    pe = fmaf(y2.y, ey, pe);
                    y2 = df_add(y2, make_float2(p, pe));
                }
                const float2 s2 = split_df_bits(su);
                const float yh = y2.x, yl = y2.y, sh = s2.x, sl = s2.y;
                for (int src = 0; src < 32; ++src) {
                    const int s_sd = __shfl_sync(0xffffffffu, sd, src);
                    const float s_yh = __shfl_sync(0xffffffffu, yh, src);
                    const float s_yl = __shfl_sync(0xffffffffu, yl, src);
                    const float s_sh = __shfl_sync(0xffffffffu, sh, src);
                    const float s_sl = __shfl_sync(0xffffffffu, sl, src);
                    if (s_sd != 0) continue;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        if (q >= nq) break;
                        // d = u - u_l, then q = d^2 + c^2, both in double-float
                        float dh, dl;
                        two_sum(s_sh, -ukf[q], dh, dl);
                        dl = __fadd_rn(dl, __fsub_rn(s_sl, ukl[q]));
                        const float p = __fmul_rn(dh, dh);
                        float pe2 = fmaf(dh, dh, -p);
                        pe2 = fmaf(__fmul_rn(2.0f, dh), dl, pe2);
                        float qh, ql;
                        two_sum(p, c2f, qh, ql);
                        ql = __fadd_rn(ql, __fadd_rn(pe2, c2l));
                        const float2 phi = df_rsqrt(qh, ql);
                        // (accf, accl) += Y phi
                        const float mh = __fmul_rn(s_yh, phi.x);
                        float me = fmaf(s_yh, phi.x, -mh);
                        me = fmaf(s_yh, phi.y, me);
                        me = fmaf(s_yl, phi.x, me);
                        float sh2, se2;
                        two_sum(accf[q], mh, sh2, se2);
                        accf[q] = sh2;
                        accl[q] = __fadd_rn(accl[q], __fadd_rn(se2, me));
                    }
                    // (no periodic fold: a double-float sum of a batch's paths stays within ~1e-13)
                }
            } else {
                for (int src = 0; src < 32; ++src) {
                    const int s_sd = __shfl_sync(0xffffffffu, sd, src);
                    const double s_y = __shfl_sync(0xffffffffu, yv, src);
                    const double s_su = __shfl_sync(0xffffffffu, su, src);
                    if (s_sd != 0) continue;
#pragma unroll
                    for (int q = 0; q < NQ; ++q) {
                        const int l = lane + 32 * q;
                        if (l >= ns) continue;
                        double phi;
                        if (imq) {
                            const double d = s_su - uk[q];
                            phi = F.mixed ? rsqrt(d * d + F.c2) : 1.0 / sqrt(d * d + F.c2);
                        } else {
                            phi = fourier_cardinal_at(s_su - uk[q], ns);
                        }
                        acc[q] += s_y * phi;
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int l = lane + 32 * q;
            if (l < ns) Mb[bt * ns + l] = acc[q] + (double)accf[q] + (double)accl[q];
        }
        for (int o = 16; o; o >>= 1) {
            bs += __shfl_xor_sync(0xffffffffu, bs, o);
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        }
        if (lane == 0) {
            bsum[bt] = bs;
            bcnt[bt] = cnt;
        }
    }
    __syncthreads();
    // regression control variate: every batch sum of a payoff loses beta^T (the batch's feature sums)
    if (F.cv_beta) {
        const double *beta = F.cv_beta + (long)slot * F.cv_stride * F.ncv;
        const double *sq = F.cv_sq + (long)slot * kBatches * F.ncv;
        for (int e = threadIdx.x; e < kBatches * (ns + 1); e += blockDim.x) {
            const int bt = e / (ns + 1), l = e - bt * (ns + 1);
            const double *bl = beta + (long)(l < ns ? l : F.cv_stride - 1) * F.ncv;
            double c = 0.0;
            for (int q = 0; q < F.ncv; ++q) c += bl[q] * sq[bt * F.ncv + q];
            if (l < ns) Mb[bt * ns + l] -= c;
            else bsum[bt] -= c;
        }
        __syncthreads();
    }
    // per-batch C estimates (batch means)
    const double *Ki = imq ? F.kinv + F.kinv_off[m] : nullptr;
    for (int bt = warp; bt < kBatches; bt += 16)
        for (int j = lane; j < ns; j += 32) {
            double v = 0.0;
            const int nb = bcnt[bt];
            if (imq) {
                for (int l = 0; l < ns; ++l) v -= Ki[l * ns + j] * Mb[bt * ns + l];
            } else {
                v = -Mb[bt * ns + j];
            }
            Cb[bt * ns + j] = nb ? v / nb : 0.0;
        }
    __syncthreads();
    // (the batch loops below stay partly rolled: fully unrolled they spilled)
    if (warp == 0) {
        int ntot = 0;
#pragma unroll 4
        for (int w = 0; w < kBatches; ++w) ntot += bcnt[w];
        const double inv = ntot ? 1.0 / ntot : 0.0;
        const int off = F.sub_off[pe];
        const long rp = F.rowptr[i];
        for (int j = lane; j < ns; j += 32) {
            double mean = 0.0, msum = 0.0;
#pragma unroll 4
            for (int w = 0; w < kBatches; ++w) {
                mean += bcnt[w] * Cb[w * ns + j];
                msum += Mb[w * ns + j];
            }
            mean *= inv;
            double var = 0.0;
#pragma unroll 4
            for (int w = 0; w < kBatches; ++w) {
                double f = bcnt[w] * inv, d = Cb[w * ns + j] - mean;
                var += f * f * d * d;
            }
            var *= (double)kBatches / (kBatches - 1);
            F.val[rp + off + j] = mean;
            F.se[rp + off + j] = sqrt(var);
            F.moments[F.mom_ptr[gs] + j] = msum * inv;
        }
        if (lane == 0) {
            double tot = 0.0;
            for (int w = 0; w < kBatches; ++w) tot += bsum[w];
            const double bm = tot * inv;
            double var = 0.0;
            for (int w = 0; w < kBatches; ++w) {
                if (!bcnt[w]) continue;
                double f = bcnt[w] * inv, d = bsum[w] / bcnt[w] - bm;
                var += f * f * d * d;
            }
            var *= (double)kBatches / (kBatches - 1);
            F.bs[pe] = bm;
            F.bmean[gs] = bm;
            F.se_bs[pe] = sqrt(var);
        }
    }
}

// (row, subdomain) entries integrated by Monte Carlo: flag + compaction over sub_rows
__global__ void k_mc_flag(int nsub, const int *sub_m, const uint8_t *floating, int mc_floating, int *flag) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nsub) return;
    flag[p] = (!floating[sub_m[p]] || mc_floating) ? 1 : 0;
}

__global__ void k_mc_compact(int nsub, const int *flag, const int *pos, const int *sub_rows, const int *sub_m,
                             const int *sub_k, const int *knot_ptr, int *rows, int *subs, int *spos, int *kword,
                             int *ns) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= nsub || !flag[p]) return;
    int s = pos[p], m = sub_m[p];
    rows[s] = sub_rows[p];
    subs[s] = m;
    spos[s] = p;
    kword[s] = sub_k[p];
    ns[s] = knot_ptr[m + 1] - knot_ptr[m];
}

void build_imq_inverses(const pdd_cover &cov, double c2, DevBuf<double> &kinv, DevBuf<long> &koff_m,
                        DevBuf<double> &kcond, cudaStream_t st) {
    if (cov.max_stencil > kMaxStencil) fail(PDD_EINVAL, "stencil larger than the Monte Carlo kernels support");
    std::vector<int> per;
    std::vector<long> off(cov.M, -1);
    long tot = 0;
    for (int m = 0; m < cov.M; ++m) {
        int n = cov.h_knot_ptr[m + 1] - cov.h_knot_ptr[m];
        if (!cov.h_floating[m] && n > 0) {
            per.push_back(m);
            off[m] = tot;
            tot += (long)n * n;
        }
    }
    DevBuf<long> koff_c;
    DevBuf<int> circ, bad;
    kinv.alloc(std::max<long>(tot, 1));
    koff_m.alloc(cov.M);
    kcond.alloc(std::max(cov.M, 1));
    PDD_CUDA(cudaMemsetAsync(kcond.p, 0, sizeof(double) * std::max(cov.M, 1), st));
    bad.alloc(1);
    PDD_CUDA(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
    PDD_CUDA(cudaMemcpyAsync(koff_m.p, off.data(), cov.M * sizeof(long), cudaMemcpyHostToDevice, st));
    if (!per.empty()) {
        std::vector<long> offc(per.size());
        for (size_t q = 0; q < per.size(); ++q) offc[q] = off[per[q]];
        circ.alloc(per.size());
        koff_c.alloc(per.size());
        PDD_CUDA(cudaMemcpyAsync(circ.p, per.data(), per.size() * sizeof(int), cudaMemcpyHostToDevice, st));
        PDD_CUDA(cudaMemcpyAsync(koff_c.p, offc.data(), per.size() * sizeof(long), cudaMemcpyHostToDevice, st));
        const size_t smem = (size_t)2 * cov.max_stencil * cov.max_stencil * sizeof(double);
        allow_smem((const void *)k_imq_inverse, smem);
        PDD_LAUNCH(k_imq_inverse, (int)per.size(), 128, smem, st, circ.p, cov.knot_ptr.p, cov.ku.p, koff_c.p, c2,
                   kinv.p, kcond.p, bad.p);
    }
    int hb = 0;
    PDD_CUDA(cudaMemcpyAsync(&hb, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    PDD_CUDA(cudaStreamSynchronize(st));
    if (hb) fail(PDD_EINVAL, "IMQ matrix not positive definite (coincident stencil angles)");
}

// ---------------------------------------------------------------------------
// Regression control variate (Milstein and Tretyakov): per slot, beta = Cov(Q)^-1 Cov(Q, P) for the
// payoffs P = (1_Gamma Y phi_l(u), l < ns; the boundary payoff of r), covariances normalised by the
// path count, and the per-batch sums of the features Q.  Any beta leaves the estimators unbiased
// (E[Q] = 0); this one is the sample's least-squares choice.  FP64 throughout (the basis values
// too, in both forms: beta only needs to be near the optimum).  One CTA per slot; paths go
// through shared memory 256 at a time, their basis values (a root and a division each, computed by all
// threads) 32 at a time; then warps 0-3 add up Q Q' while warps 4-7 add up the payoffs' products, each sum
// in the order of the paths.  Bound by the FP64 pipe and, with the sums in that order, the chains of
// additions.  1,000 rows x 5,000 paths, 44 payoffs, 14 features: 14.3 -> 11.6 ms (the payoffs' threads
// used to form the basis values themselves, two warps of eight).
// ---------------------------------------------------------------------------
static constexpr int kCvThreads = 256;

__global__ void __launch_bounds__(kCvThreads) k_cv_regress(Problem P, FinalArgs F, const double *cvq,
                                                           double *beta_out, double *sq_out) {
    const int M = F.ncv;
    extern __shared__ double cvs[];
    double *Qs = cvs;                                 // [256][M] this chunk's features
    double *Ys = Qs + kCvThreads * M;                 // [256] Y at the exit (0: not an interface exit)
    double *Us = Ys + kCvThreads;                     // [256] exit angle
    double *QQ = Us + kCvThreads;                     // [M][M]
    double *QP = QQ + M * M;                          // [ns + 1][M]
    double *Pm = QP + (F.cv_stride) * M;              // [ns + 1] payoff sums
    double *Qm = Pm + F.cv_stride;                    // [M] feature sums
    double *SQ = Qm + M;                              // [32][M] per-batch feature sums
    double *L = SQ + kBatches * M;                    // [M][M] Cholesky factor
    double *Ws = L + M * M;                           // [32][ns] Y phi_l of 32 paths
    __shared__ int s_cnt;
    const int slot = blockIdx.x, tid = threadIdx.x;
    const int gs = F.gslot ? F.gslot[slot] : slot;
    const int m = F.subs[gs];
    const int a = F.knot_ptr[m], ns = F.knot_ptr[m + 1] - a;
    const bool imq = !F.floating[m];
    const int npath = F.npaths ? F.npaths[slot] : F.paths;
    const long base = F.rec_off ? F.rec_off[slot] : (long)slot * F.paths;
    for (int e = tid; e < M * M + F.cv_stride * M + F.cv_stride + M + kBatches * M; e += kCvThreads) QQ[e] = 0.0;
    __syncthreads();
    // per-thread sums: the thread's paths are p = tid (mod 256), all in batch tid mod 32
    double my_sq[kMaxCv], my_bq[kMaxCv], my_b = 0.0;
#pragma unroll
    for (int q = 0; q < kMaxCv; ++q) {
        my_sq[q] = 0.0;
        my_bq[q] = 0.0;
    }
    int my_cnt = 0;
    // QQ entry (i, j) per thread (M (M + 1) / 2 <= 105 < 256); QP rows per thread l = tid (mod ns + 1)
    int qi = -1, qj = -1;
    {
        int e = tid;
        for (int i = 0; i < M && qi < 0; ++i) {
            if (e < M - i) {
                qi = i;
                qj = i + e;
            } else {
                e -= M - i;
            }
        }
    }
    static_assert(kMaxStencil <= kCvThreads / 2 && kMaxCv * (kMaxCv + 1) <= kCvThreads, "warps 0-3, 4-7");
    const int lp = tid - kCvThreads / 2;              // this thread's payoff
    double acc_qq = 0.0;
    for (int c0 = 0; c0 < npath; c0 += kCvThreads) {
        const int p = c0 + tid;
        double yv = 0.0, ut = 0.0;
        if (p < npath) {
            const long rec = base + p;
            const int sd = F.side[rec];
            double y = F.Y[rec], z = F.Z[rec];
            if (F.mixed) {
                const float2 q = F.ez[rec];
                z = fma(y, (double)q.y, z);
                y = fma(y, (double)q.x, y);
            }
            for (int q = 0; q < M; ++q) Qs[tid * M + q] = (sd != 2) ? cvq[rec * M + q] : 0.0;
            if (sd != 2) {
                ++my_cnt;
                const double bp = (sd == 1) ? boundary_score(P, F.su[rec], F.mixed) * y + z : z;
                my_b += bp;
                for (int q = 0; q < M; ++q) {
                    const double qv = cvq[rec * M + q];
                    my_sq[q] += qv;
                    my_bq[q] += bp * qv;
                }
                if (sd == 0) {
                    yv = y;
                    ut = F.su[rec];
                }
            }
        } else {
            for (int q = 0; q < M; ++q) Qs[tid * M + q] = 0.0;
        }
        Ys[tid] = yv;
        Us[tid] = ut;
        __syncthreads();
        // basis payoffs: thread l < ns accumulates sum_p Y phi_l(u_p) Q_p and sum_p Y phi_l(u_p)
        double acc[kMaxCv], ps = 0.0;
#pragma unroll
        for (int q = 0; q < kMaxCv; ++q) acc[q] = 0.0;
        for (int s0 = 0; s0 < min(kCvThreads, npath - c0); s0 += 32) {
            for (int e = tid; e < 32 * ns; e += kCvThreads) {
                const int t = s0 + e / ns, l = e % ns;
                if (Ys[t] == 0.0) continue;
                const double d = Us[t] - (imq ? F.ku[a + l] : PDD_TWO_PI * l / ns);
                Ws[e] = Ys[t] * (imq ? 1.0 / sqrt(d * d + F.c2) : fourier_cardinal_at(d, ns));
            }
            __syncthreads();
            if (qi >= 0)
                for (int t = s0; t < s0 + 32; ++t) acc_qq += Qs[t * M + qi] * Qs[t * M + qj];
            if (lp >= 0 && lp < ns)
                for (int t = 0; t < 32; ++t) {
                    if (Ys[s0 + t] == 0.0) continue;
                    const double w = Ws[t * ns + lp];
                    ps += w;
#pragma unroll
                    for (int q = 0; q < kMaxCv; ++q)
                        if (q < M) acc[q] += w * Qs[(s0 + t) * M + q];
                }
            __syncthreads();
        }
        if (lp >= 0 && lp < ns) {
            Pm[lp] += ps;
            for (int q = 0; q < M; ++q) QP[lp * M + q] += acc[q];
        }
    }
    if (qi >= 0) {
        QQ[qi * M + qj] = acc_qq;
        QQ[qj * M + qi] = acc_qq;
    }
    // the features' sums per batch (lane = batch; the 8 warps added in order), then over batches;
    // the boundary payoff's sums by warp shuffles and the 8 warps in order (deterministic)
    __shared__ double wb[8][kMaxCv + 1];
    __shared__ int wc[8];
    for (int q = 0; q < M; ++q) Qs[tid * M + q] = my_sq[q];
#pragma unroll
    for (int q = 0; q <= kMaxCv; ++q) {
        double v = q < kMaxCv ? my_bq[q] : my_b;
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((tid & 31) == 0) wb[tid >> 5][q] = v;
    }
    for (int o = 16; o; o >>= 1) my_cnt += __shfl_xor_sync(0xffffffffu, my_cnt, o);
    if ((tid & 31) == 0) wc[tid >> 5] = my_cnt;
    __syncthreads();
    for (int e = tid; e < kBatches * M; e += kCvThreads) {
        const int bt = e / M, q = e - bt * M;
        double v = 0.0;
        for (int w = 0; w < kCvThreads / 32; ++w) v += Qs[(w * 32 + bt) * M + q];
        SQ[e] = v;
    }
    if (tid <= M) {
        double v = 0.0;
        for (int w = 0; w < kCvThreads / 32; ++w) v += wb[w][tid < M ? tid : kMaxCv];
        if (tid < M) QP[(F.cv_stride - 1) * M + tid] = v;
        else Pm[F.cv_stride - 1] = v;
    }
    if (tid == 0) {
        int c = 0;
        for (int w = 0; w < kCvThreads / 32; ++w) c += wc[w];
        s_cnt = c;
    }
    __syncthreads();
    if (tid < M) {
        double v = 0.0;
        for (int bt = 0; bt < kBatches; ++bt) v += SQ[bt * M + tid];
        Qm[tid] = v;
    }
    __syncthreads();
    // Cov(Q) = QQ / n - qm qm^T, Cholesky in place (thread 0; M <= 14)
    const double inv_n = s_cnt ? 1.0 / s_cnt : 0.0;
    if (tid == 0) {
        for (int i = 0; i < M; ++i)
            for (int j = 0; j < M; ++j) L[i * M + j] = QQ[i * M + j] * inv_n - Qm[i] * inv_n * Qm[j] * inv_n;
        for (int j = 0; j < M; ++j) {
            double dg = L[j * M + j];
            for (int k = 0; k < j; ++k) dg -= L[j * M + k] * L[j * M + k];
            dg = dg > 0.0 ? sqrt(dg) : 0.0;
            L[j * M + j] = dg;
            for (int i = j + 1; i < M; ++i) {
                double v = L[i * M + j];
                for (int k = 0; k < j; ++k) v -= L[i * M + k] * L[j * M + k];
                L[i * M + j] = dg > 0.0 ? v / dg : 0.0;
            }
        }
    }
    __syncthreads();
    // beta for each payoff row: rows l < ns (basis moments) and row cv_stride - 1 (r); zero when the
    // covariance is singular (no paths, or a feature that never moved)
    double *bo = beta_out + (long)slot * F.cv_stride * M;
    for (int l = tid; l < F.cv_stride; l += kCvThreads) {
        if (l >= ns && l != F.cv_stride - 1) {
            for (int q = 0; q < M; ++q) bo[l * M + q] = 0.0;
            continue;
        }
        double y[kMaxCv];
        bool ok = s_cnt > 1;
        for (int i = 0; i < M; ++i) {
            double v = QP[l * M + i] * inv_n - Qm[i] * inv_n * Pm[l] * inv_n;
            for (int k = 0; k < i; ++k) v -= L[i * M + k] * y[k];
            ok = ok && L[i * M + i] > 0.0;
            y[i] = ok ? v / L[i * M + i] : 0.0;
        }
        for (int i = M - 1; i >= 0; --i) {
            double v = y[i];
            for (int k = i + 1; k < M; ++k) v -= L[k * M + i] * y[k];
            y[i] = ok ? v / L[i * M + i] : 0.0;
        }
        for (int q = 0; q < M; ++q) bo[l * M + q] = y[q];
    }
    for (int e = tid; e < kBatches * M; e += kCvThreads) sq_out[(long)slot * kBatches * M + e] = SQ[e];
}

// adaptive path count of each row from its pilot standard errors
__global__ void k_need(int nmc, const int *rows, const int *subs, const int *spos, const int *sub_off,
                       const int *knot_ptr, const int *rowptr, const double *se, const double *se_bs, int P0,
                       int Pmax, double target, int *need) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= nmc) return;
    const int i = rows[slot], m = subs[slot], pe = spos[slot];
    const int a = knot_ptr[m], ns = knot_ptr[m + 1] - a, off = sub_off[pe];
    double mx = se_bs[pe];
    for (int j = 0; j < ns; ++j) mx = fmax(mx, se[rowptr[i] + off + j]);
    // rows at or below the target keep the pilot; the others rerun with ceil(P0 (se/target)^2)
    // paths rounded up to a multiple of 32, capped at Pmax
    if (!(mx > target)) {
        need[slot] = P0;
        return;
    }
    const double r = mx / target;
    const double want = fmin(ceil(P0 * r * r), (double)Pmax);
    int w = (int)want;
    w = ((w + 31) / 32) * 32;
    need[slot] = w > Pmax ? Pmax : w;
}

// buffers of the mixed form, kept over the waves of one assembly
struct Paths32Bufs {
    DevBuf<Slot32> slots;
    DevBuf<float4> seg;
    DevBuf<unsigned> next;
};

template <int CVD>
static const void *paths_long_kernel(bool kill, bool src) {
    return kill ? (src ? (const void *)k_paths_long<true, true, CVD> : (const void *)k_paths_long<true, false, CVD>)
                : (src ? (const void *)k_paths_long<false, true, CVD> : (const void *)k_paths_long<false, false, CVD>);
}
template <bool CV>
static void launch_paths(const Problem &P, const PathArgs &A, int nrows, int nc, int nf, size_t sm, cudaStream_t st) {
    const bool kill = P.c_kind != PDD_C_ZERO, src = P.f_kind != PDD_F_ZERO;
    auto kern = kill ? (src ? k_paths<true, true, CV, false> : k_paths<true, false, CV, false>)
                     : (src ? k_paths<false, true, CV, false> : k_paths<false, false, CV, false>);
    if (nc || nf)
        kern = kill ? (src ? k_paths<true, true, CV, true> : k_paths<true, false, CV, true>) : k_paths<false, true, CV, true>;
    PDD_LAUNCH(kern, nrows, kRowThreads, sm, st, P, A, nc, nf);
}

// nrows slots with `total` paths in all, their records contiguous in slot order
static void run_paths32(const Problem &P, const PathArgs &A, int nrows, long total, bool long_paths, Paths32Bufs &B,
                        cudaStream_t st) {
    const int nc = P.c_kind == PDD_C_RBF && P.n_rbf <= kP32Staged ? P.n_rbf : 0;
    const int nf = P.f_kind == PDD_F_RBF && P.n_frbf <= kP32Staged ? P.n_frbf : 0;
    const size_t sm = (nc ? gauss_smem(nc) : 0) + (nf ? gauss_smem(nf) : 0);
    if (!long_paths) {
        if (A.cvd > 0) launch_paths<true>(P, A, nrows, nc, nf, sm, st);
        else launch_paths<false>(P, A, nrows, nc, nf, sm, st);
        return;
    }
    int dev = 0, sms = 0, per_sm = 0;
    PDD_CUDA(cudaGetDevice(&dev));
    PDD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (B.slots.n < (size_t)nrows) B.slots.alloc(nrows);
    if (B.seg.n < (size_t)total) B.seg.alloc(total);
    if (!B.next.n) B.next.alloc(1);
    PDD_CUDA(cudaMemsetAsync(B.next.p, 0, sizeof(unsigned), st));
    PDD_LAUNCH(k_slots32, cdiv(nrows, 128), 128, 0, st, nrows, A, B.slots.p);
    Pool32 Q{B.slots.p, nrows, total, B.next.p, B.seg.p, nc, nf};
    const bool kill = P.c_kind != PDD_C_ZERO, src = P.f_kind != PDD_F_ZERO;
    const void *kern = A.cvd == 0 ? paths_long_kernel<0>(kill, src)
                                  : (A.cvd == 4 ? paths_long_kernel<4>(kill, src) : paths_long_kernel<-1>(kill, src));
    PDD_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kP32Threads, sm));
    const int grid = (int)std::max<long>(1, std::min<long>((long)sms * std::max(per_sm, 1), cdiv(total, kP32Threads)));
    Problem Pv = P;
    PathArgs Av = A;
    void *args[] = {&Pv, &Av, &Q};
    PDD_CUDA(cudaLaunchKernel(kern, dim3(grid), dim3(kP32Threads), args, sm, st));
    count_launch();
    PDD_LAUNCH(k_exit32, cdiv(total, 256), 256, 0, st, P, A, Q);
}

// buffers of the FP64 form's passes, kept over the waves of one assembly
struct Paths64Bufs {
    DevBuf<Slot64> slots;
    DevBuf<PathState> state[2];
    DevBuf<double> cq[2];
    DevBuf<Seg64> seg;
    DevBuf<unsigned long long> next;     // one queue per pass
    DevBuf<unsigned> count;
};
static constexpr int kP64Passes = 4;

template <bool CV>
static void launch_pass64(const Problem &P, const PathArgs &A, const PathPool &Q, int grid, size_t sm,
                          cudaStream_t st) {
    const bool kill = P.c_kind != PDD_C_ZERO, src = P.f_kind != PDD_F_ZERO;
    auto kern = kill ? (src ? k_paths64<true, true, CV> : k_paths64<true, false, CV>)
                     : (src ? k_paths64<false, true, CV> : k_paths64<false, false, CV>);
    PDD_LAUNCH(kern, grid, kP64Threads, sm, st, P, A, Q);
}

// nrows slots with `total` paths in all, their records contiguous in slot order
static void run_paths64(const Problem &P, const PathArgs &A, int nrows, long total, Paths64Bufs &B, cudaStream_t st) {
    int dev = 0, sms = 0;
    PDD_CUDA(cudaGetDevice(&dev));
    PDD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int ctas = std::max(1, std::min(cdiv(total, kP64Threads), sms * kP64WarpsPerSm * 32 / kP64Threads));
    const size_t lanes = (size_t)ctas * kP64Threads;
    if (B.slots.n < (size_t)nrows) B.slots.alloc(nrows);
    if (B.seg.n < (size_t)total) B.seg.alloc(total);
    if (B.state[0].n < lanes)
        for (auto &s : B.state) s.alloc(lanes);
    if (A.ncv && B.cq[0].n < lanes * A.ncv)
        for (auto &c : B.cq) c.alloc(lanes * A.ncv);
    if (!B.next.n) {
        B.next.alloc(kP64Passes);
        B.count.alloc(kP64Passes);
    }
    PDD_CUDA(cudaMemsetAsync(B.next.p, 0, kP64Passes * sizeof(unsigned long long), st));
    PDD_CUDA(cudaMemsetAsync(B.count.p, 0, kP64Passes * sizeof(unsigned), st));
    PDD_LAUNCH(k_slots64, cdiv(nrows, 128), 128, 0, st, nrows, A, B.slots.p);
    size_t sm = 0;
    if (P.c_kind == PDD_C_RBF)
        sm = (2 * (size_t)kExpTab + (P.n_rbf <= kP64Staged ? 3 * (size_t)P.n_rbf : 0)) * sizeof(double);
    PathPool Q{B.slots.p, nrows, (unsigned long long)total, nullptr, nullptr, nullptr, nullptr, nullptr, 0, nullptr,
               nullptr, B.seg.p};
    int grid = ctas;
    const bool kill = P.c_kind == PDD_C_RBF, src = P.f_kind == PDD_F_RBF;
    const bool walk = P.b_kind == PDD_B_ZERO && (P.c_kind == PDD_C_ZERO || kill) && (P.f_kind == PDD_F_ZERO || src) &&
                      A.cvd == 0;
    for (int pass = 0; pass < kP64Passes; ++pass) {
        const bool last = pass == kP64Passes - 1;
        Q.next = B.next.p + pass;
        Q.in = pass ? B.state[(pass - 1) & 1].p : nullptr;
        Q.n_in = pass ? B.count.p + pass - 1 : nullptr;
        Q.cq_in = B.cq[(pass + 1) & 1].p;
        Q.out = B.state[pass & 1].p;
        Q.cq_out = B.cq[pass & 1].p;
        Q.n_out = B.count.p + pass;
        Q.keep = last ? 0 : 16;
        if (walk && pass == 1) {
            const int most = cdiv(15L * ctas * (kP64Threads / 32), kP64Threads / kWalkLanes);     // its paths, at most
            auto kern = kill ? (src ? k_walk64<true, true> : k_walk64<true, false>)
                             : (src ? k_walk64<false, true> : k_walk64<false, false>);
            PDD_LAUNCH(kern, std::min(most, 8 * sms), kP64Threads, sm, st, P, A, Q);
            break;
        }
        if (A.cvd > 0) launch_pass64<true>(P, A, Q, grid, sm, st);
        else launch_pass64<false>(P, A, Q, grid, sm, st);
        grid = std::max(1, (grid + 1) / 2);               // every warp hands over at most half its lanes
    }
    PDD_LAUNCH(k_exit64, cdiv(total, 256), 256, 0, st, P, A, Q);
}

McStats assemble_mc(const pdd_cover &cov, const Problem &P, const pdd_assembly_opts &o, pdd_system &sys,
                    cudaStream_t st) {
    McStats ms;
    const int mcf = o.floating_method == PDD_FLOATING_MONTE_CARLO ? 1 : 0;
    const int nsub = cov.h_sub_ptr.empty() ? 0 : cov.h_sub_ptr.back();
    DevBuf<int> flag, pos;
    flag.alloc(nsub + 1);
    pos.alloc(nsub + 1);
    if (nsub > 0) PDD_LAUNCH(k_mc_flag, cdiv(nsub, 256), 256, 0, st, nsub, cov.sub_m.p, cov.floating.p, mcf, flag.p);
    const int nmc = nsub > 0 ? (int)exclusive_scan(flag.p, pos.p, nsub, st) : 0;
    sys.n_mc = nmc;
    ms.rows = nmc;
    if (nmc == 0) return ms;
    sys.mc_rows.alloc(nmc);
    sys.mc_subs.alloc(nmc);
    sys.mc_spos.alloc(nmc);
    sys.mc_kword.alloc(nmc);
    DevBuf<int> ns;
    ns.alloc(nmc + 1);
    sys.mom_ptr.alloc(nmc + 1);
    PDD_LAUNCH(k_mc_compact, cdiv(nsub, 256), 256, 0, st, nsub, flag.p, pos.p, cov.sub_rows.p, cov.sub_m.p,
               cov.sub_k.p, cov.knot_ptr.p, sys.mc_rows.p, sys.mc_subs.p, sys.mc_spos.p, sys.mc_kword.p, ns.p);
    const int nmom = (int)exclusive_scan(ns.p, sys.mom_ptr.p, nmc, st);
    sys.moments.alloc(std::max(nmom, 1));
    sys.bmean.alloc(nmc);

    // a10: IMQ inverses for every perimeter circle with a stencil
    DevBuf<double> kinv, kcond;
    DevBuf<long> koff_m;
    build_imq_inverses(cov, o.imq_c2, kinv, koff_m, kcond, st);

    // a11: paths into the record scratch, in waves that bound the scratch size
    const long P_ = o.paths;
    const int mixed = path_mixed(o) ? 1 : 0;
    const int cvd = o.cv_degree, ncv = cvd * (cvd + 3) / 2;          // control-variate features per path
    const int cv_stride = cov.max_stencil + 1;
    const size_t rec_bytes =
        1 + 3 * sizeof(double) + (mixed ? sizeof(float2) + sizeof(float4) : sizeof(Seg64)) +
        (size_t)ncv * sizeof(double);
    const size_t per_row = (size_t)P_ * rec_bytes;
    const int wave = (int)std::max<size_t>(1, std::min<size_t>(nmc, ((size_t)8 << 30) / per_row));
    DevBuf<int8_t> side;
    DevBuf<double> su, Y, Z;
    side.alloc((size_t)wave * P_);
    su.alloc((size_t)wave * P_);
    Y.alloc((size_t)wave * P_);
    Z.alloc((size_t)wave * P_);
    DevBuf<float2> ez;
    if (mixed) ez.alloc((size_t)wave * P_);
    DevBuf<double> cvq, cvbeta, cvsq;
    if (ncv) cvq.alloc((size_t)wave * P_ * ncv);
    const size_t cv_smem = ((size_t)kCvThreads * ncv + 2 * kCvThreads + 2 * ncv * ncv + (size_t)cv_stride * ncv +
                            cv_stride + ncv + (size_t)kBatches * ncv + 32 * cv_stride) * sizeof(double);
    if (ncv) allow_smem((const void *)k_cv_regress, cv_smem);
    DevBuf<unsigned long long> steps;
    DevBuf<int> capped;
    steps.alloc(1);
    capped.alloc(1);
    PDD_CUDA(cudaMemsetAsync(steps.p, 0, sizeof(unsigned long long), st));
    PDD_CUDA(cudaMemsetAsync(capped.p, 0, sizeof(int), st));
    cudaEvent_t e0, e1, e2;
    PDD_CUDA(cudaEventCreate(&e0));
    PDD_CUDA(cudaEventCreate(&e1));
    PDD_CUDA(cudaEventCreate(&e2));
    float tp = 0, tf = 0;
    const size_t fsm = (size_t)2 * kBatches * cov.max_stencil * sizeof(double);
    const int nq_launch = std::max(1, (cov.max_stencil + 31) / 32);
    allow_smem((const void *)k_mc_finalize<1>, fsm);
    allow_smem((const void *)k_mc_finalize<2>, fsm);
    allow_smem((const void *)k_mc_finalize<3>, fsm);
    // per-slot arrays (subs, spos, kword, momp, bmean) are indexed like the global slot gs: offset to
    // the wave's first slot when gsl is null, or the whole arrays with gsl
    Paths64Bufs p64;
    Paths32Bufs p32;
    // the steps of a path from a circle's centre (r^2 / 4h), on average over the slots
    double mean_steps = 0.0;
    for (int m = 0; m < cov.M; ++m)
        if (!cov.h_floating[m] || mcf)
            mean_steps += (cov.h_sub_ptr[m + 1] - cov.h_sub_ptr[m]) * (cov.h_r[m] * cov.h_r[m] / (4.0 * o.h)) / nmc;
    const bool long_paths = mean_steps >= kLongSteps;
    auto run_wave = [&](const int *rows, int nr, long nrec, const int *np, const long *roff, const int *gsl,
                        const int *momp, double *bmean, size_t w0) {
        const int *subs = sys.mc_subs.p + w0, *spos = sys.mc_spos.p + w0, *kword = sys.mc_kword.p + w0;
        PathArgs A{rows, subs, kword, cov.kx.p, cov.ky.p, cov.cx.p, cov.cy.p, cov.r.p,
                   cov.theta_s.p, o.paths, o.h, o.seed, side.p, su.p, Y.p, Z.p, steps.p, capped.p, np, roff, ez.p,
                   o.boundary_shift ? kGmC0 * sqrt(o.h) : 0.0, gsl, o.max_steps, cvd, ncv, cvq.p};
        PDD_CUDA(cudaEventRecord(e0, st));
        if (mixed) run_paths32(P, A, nr, nrec, long_paths, p32, st);
        else run_paths64(P, A, nr, nrec, p64, st);
        PDD_CUDA(cudaEventRecord(e1, st));
        FinalArgs F{rows, subs, spos, cov.sub_off.p, cov.knot_ptr.p, cov.rowptr.p, cov.floating.p,
                    cov.ku.p, koff_m.p, kinv.p, kcond.p, o.imq_c2, o.paths, mcf, mixed, np, roff, gsl, side.p, su.p,
                    Y.p, Z.p,
                    ez.p, momp, sys.moments.p, bmean, sys.val.p, sys.se.p, sys.bs.p, sys.se_bs.p, o.moment_sums,
                    nullptr, nullptr, ncv, cv_stride};
        if (ncv) {
            if (cvbeta.n < (size_t)nr * cv_stride * ncv) cvbeta.alloc((size_t)nr * cv_stride * ncv);
            if (cvsq.n < (size_t)nr * kBatches * ncv) cvsq.alloc((size_t)nr * kBatches * ncv);
            PDD_LAUNCH(k_cv_regress, nr, kCvThreads, cv_smem, st, P, F, cvq.p, cvbeta.p, cvsq.p);
            F.cv_beta = cvbeta.p;
            F.cv_sq = cvsq.p;
        }
        if (nq_launch == 1) PDD_LAUNCH(k_mc_finalize<1>, nr, 512, fsm, st, P, F);
        else if (nq_launch == 2) PDD_LAUNCH(k_mc_finalize<2>, nr, 512, fsm, st, P, F);
        else PDD_LAUNCH(k_mc_finalize<3>, nr, 512, fsm, st, P, F);
        PDD_CUDA(cudaEventRecord(e2, st));
        PDD_CUDA(cudaEventSynchronize(e2));
        float ta = 0, tb = 0;
        cudaEventElapsedTime(&ta, e0, e1);
        cudaEventElapsedTime(&tb, e1, e2);
        tp += ta;
        tf += tb;
    };
    for (int w0 = 0; w0 < nmc; w0 += wave) {
        const int nr = std::min(wave, nmc - w0);
        run_wave(sys.mc_rows.p + w0, nr, (long)nr * P_, nullptr, nullptr, nullptr, sys.mom_ptr.p + w0, sys.bmean.p + w0, w0);
    }
    ms.paths_total = (int64_t)nmc * P_;
    sys.mc_np.alloc(nmc);
    std::vector<int> need(nmc, (int)P_);
    // adaptive path counts: rows whose largest standard error exceeds the target rerun with
    // P0 (se/target)^2 paths (capped at paths_max); path ids continue the pilot's streams
    if (o.paths_max > o.paths && o.se_target > 0.0) {
        DevBuf<int> dneed;
        dneed.alloc(nmc);
        PDD_LAUNCH(k_need, cdiv(nmc, 256), 256, 0, st, nmc, sys.mc_rows.p, sys.mc_subs.p, sys.mc_spos.p,
                   cov.sub_off.p, cov.knot_ptr.p, cov.rowptr.p, sys.se.p, sys.se_bs.p, o.paths, o.paths_max,
                   o.se_target, dneed.p);
        PDD_CUDA(cudaMemcpyAsync(need.data(), dneed.p, nmc * sizeof(int), cudaMemcpyDeviceToHost, st));
        PDD_CUDA(cudaStreamSynchronize(st));
        std::vector<int> ext_slot, ext_row_host;
        std::vector<int> hrows(nmc);
        PDD_CUDA(cudaMemcpyAsync(hrows.data(), sys.mc_rows.p, nmc * sizeof(int), cudaMemcpyDeviceToHost, st));
        PDD_CUDA(cudaStreamSynchronize(st));
        for (int k = 0; k < nmc; ++k)
            if (need[k] > P_) ext_slot.push_back(k);
        size_t q = 0;
        const size_t budget = (size_t)8 << 30;
        while (q < ext_slot.size()) {
            std::vector<int> rows, np, gsl;
            std::vector<long> roff;
            size_t used = 0;
            long off = 0;
            while (q < ext_slot.size() && (rows.empty() || used + (size_t)need[ext_slot[q]] * rec_bytes <= budget)) {
                const int k = ext_slot[q++];
                rows.push_back(hrows[k]);
                np.push_back(need[k]);
                gsl.push_back(k);
                roff.push_back(off);
                off += need[k];
                used += (size_t)need[k] * rec_bytes;
                ms.paths_total += need[k];
                ++ms.extended_rows;
            }
            DevBuf<int> drows, dnp, dgsl;
            DevBuf<long> droff;
            drows.alloc(rows.size());
            dnp.alloc(rows.size());
            dgsl.alloc(rows.size());
            droff.alloc(rows.size());
            PDD_CUDA(cudaMemcpyAsync(drows.p, rows.data(), rows.size() * sizeof(int), cudaMemcpyHostToDevice, st));
            PDD_CUDA(cudaMemcpyAsync(dnp.p, np.data(), np.size() * sizeof(int), cudaMemcpyHostToDevice, st));
            PDD_CUDA(cudaMemcpyAsync(dgsl.p, gsl.data(), gsl.size() * sizeof(int), cudaMemcpyHostToDevice, st));
            PDD_CUDA(cudaMemcpyAsync(droff.p, roff.data(), roff.size() * sizeof(long), cudaMemcpyHostToDevice, st));
            if ((size_t)off > side.n) {
                side.alloc(off);
                su.alloc(off);
                Y.alloc(off);
                Z.alloc(off);
                if (mixed) ez.alloc(off);
                if (ncv) cvq.alloc((size_t)off * ncv);
            }
            run_wave(drows.p, (int)rows.size(), off, dnp.p, droff.p, dgsl.p, sys.mom_ptr.p, sys.bmean.p, 0);
        }
    }
    PDD_CUDA(cudaMemcpyAsync(sys.mc_np.p, need.data(), nmc * sizeof(int), cudaMemcpyHostToDevice, st));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaEventDestroy(e2);
    unsigned long long hs = 0;
    int hc = 0;
    PDD_CUDA(cudaMemcpyAsync(&hs, steps.p, sizeof(hs), cudaMemcpyDeviceToHost, st));
    PDD_CUDA(cudaMemcpyAsync(&hc, capped.p, sizeof(hc), cudaMemcpyDeviceToHost, st));
    PDD_CUDA(cudaStreamSynchronize(st));
    ms.steps = (int64_t)hs;
    ms.capped = hc;
    ms.ms_paths = tp;
    ms.ms_finalize = tf;
    return ms;
}

}  // namespace pdd

// ---------------------------------------------------------------------------
// a14 (perimeter rows): replay each row's paths with the same Philox streams
// (common random numbers).  The paths X do not depend on c, f or g; only the
// weights do.  With S_q = sum_k 1{c<0} psi_q(X_k) h / (1 + c(X_k) h),
// dY_tau/dw_q = Y_tau S_q and dZ/dw_q = sum_k f(X_k) h Y_k S_q(k).  The row adds
// lambda_i E[(1_dOmega g + 1_Gamma u_hat) dY_q + dZ_q] to dJ/dw_q and
// lambda_i E[1_dOmega psi^g_k(s) Y_tau] to dJ/da_k.
// ---------------------------------------------------------------------------
namespace pdd {

struct GradArgs {
    const double *u, *lambda;
    const int *knot_ptr;
    const uint8_t *floating;
    const double *ku;
    const long *kinv_off;
    const double *kinv;
    double c2;
    int n_par, splits;        // a row's paths are cut into `splits` parts, one CTA each
    double *partial;          // [slot][part][n_rbf + n_frbf + n_gcoef]
};

// Four lanes carry one path: they hold its state in common and each owns every fourth basis
// function (of c, f and g) and its running sums in shared memory, [index / 4][thread].  The cost is
// the FP64 pipe (one Gaussian per basis function and step, exp_neg, evaluated once: psi is kept in
// shared memory for the update that needs c first), so nothing else is repeated by the four lanes:
// lane s of a path draws the normals of step k + s for all four, the payoff's basis sum and the
// boundary series are split over them.  A warp owns a fixed range of path ids and its eight
// paths take the next id of that range in lane order (deterministic); a path that ends waits for
// the next group of four steps, so the normals of all eight are drawn together.
// 116 rows x 1,000 paths, 64 + 16 + 32 parameters: 1240 -> 86 ms.
static constexpr int kGradThreads = 128, kGradLanes = 4;
static constexpr int kGradMaxParams = 438;       // 3 nw + nf + ng: at most 164 KB of shared memory

__host__ __device__ constexpr size_t grad_smem_doubles(int nw, int nf, int ng) {
    return kMaxStencil + 2 * kExpTab + 3 * (size_t)(nw + nf) +
           (size_t)kGradThreads * (4 * ((nw + 3) / 4) + (nf + 3) / 4 + (ng + 3) / 4);
}

template <typename R, bool SRC>
__global__ void __launch_bounds__(kGradThreads) k_paths_grad(Problem P, PathArgs A, GradArgs G) {
    extern __shared__ __align__(16) double gsm[];
    constexpr int T = kGradThreads;
    constexpr unsigned kAll = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, sub = lane & 3, lead = lane & 28;
    const unsigned gmask = 0xfu << lead;
    const int nw = P.n_rbf, ng = (P.g_kind == PDD_G_BOUNDARY_FOURIER) ? P.n_gcoef : 0;
    const int nf = (P.f_kind == PDD_F_RBF) ? P.n_frbf : 0;
    const int nw4 = (nw + 3) / 4, nf4 = (nf + 3) / 4, ng4 = (ng + 3) / 4;
    double2 *etab = reinterpret_cast<double2 *>(gsm);     // exp_neg's table
    double *rx = gsm + 2 * kExpTab, *ry = rx + nw, *rw = ry + nw;
    double *fx = rw + nw, *fy = fx + nf, *fw = fy + nf;
    double *alpha = fw + nf;                              // kMaxStencil
    double *S = alpha + kMaxStencil + tid;                // [nw4][T] each: S_q, dZ_q, psi_q, the sums over paths
    double *dZ = S + (size_t)nw4 * T;
    double *psi = dZ + (size_t)nw4 * T;
    double *Gw = psi + (size_t)nw4 * T;
    double *Gf = Gw + (size_t)nw4 * T;                    // [nf4][T]: sum over paths of dZ_tau / dv_q
    double *Gg = Gf + (size_t)nf4 * T;                    // [ng4][T]
    const int slot = blockIdx.x / G.splits, part = blockIdx.x - slot * G.splits;
    const int gsl = A.gslot ? A.gslot[slot] : slot;
    const int i = A.rows[slot], m = A.subs[gsl];
    const uint32_t kw = A.kword ? (uint32_t)A.kword[gsl] : 0u;
    const int a = G.knot_ptr[m], ns = G.knot_ptr[m + 1] - a;
    const bool imq = !G.floating[m];
    // u_hat(u) = sum_l alpha_l phi_l(u) (IMQ) or sum_j u_j H_j(theta) (Fourier cardinals)
    for (int l = tid; l < ns; l += T) {
        double v = 0.0;
        if (imq) {
            const double *Ki = G.kinv + G.kinv_off[m];
            for (int j = 0; j < ns; ++j) v += Ki[l * ns + j] * G.u[a + j];
        } else {
            v = G.u[a + l];
        }
        alpha[l] = v;
    }
    for (int q = tid; q < kExpTab; q += T) etab[q] = kExp2Tab[q];
    for (int q = tid; q < nw; q += T) {
        rx[q] = P.rbf_x[q];
        ry[q] = P.rbf_y[q];
        rw[q] = P.rbf_w[q];
    }
    for (int q = tid; q < nf; q += T) {
        fx[q] = P.frbf_x[q];
        fy[q] = P.frbf_y[q];
        fw[q] = P.frbf_w[q];
    }
    for (int q = 0; q < nw4; ++q) Gw[q * T] = 0.0;
    for (int q = 0; q < nf4; ++q) Gf[q * T] = 0.0;
    for (int q = 0; q < ng4; ++q) Gg[q * T] = 0.0;
    __syncthreads();
    const double inv2f = nf ? 1.0 / (2.0 * P.frbf_sigma * P.frbf_sigma) : 0.0;
    const double cx = A.ccx[m], cy = A.ccy[m], rad = A.cr[m];
    // the same exit rule as k_paths: disk and domain shrunk by the boundary shift (0: plain)
    const double rs = rad - A.shift;
    const R rcx = (R)cx, rcy = (R)cy, r2 = (R)(rs * rs);
    Problem Ps = P;
    if (P.dom_kind == 0) {
        Ps.dom[0] += A.shift;
        Ps.dom[1] += A.shift;
        Ps.dom[2] -= A.shift;
        Ps.dom[3] -= A.shift;
    } else {
        Ps.dom[2] -= A.shift;
    }
    const int max_steps = A.max_steps > 0 ? A.max_steps : (int)fmin(2147483647.0, ceil(50.0 * rad * rad / A.h));
    const R h = (R)A.h, sh = Num<R>::sq((R)A.h);
    const double inv2s = nw ? 1.0 / (2.0 * P.rbf_sigma * P.rbf_sigma) : 0.0;
    const int npath = A.npaths ? A.npaths[slot] : A.paths;
    // this warp's path ids [next, last)
    const int per_w = (npath + G.splits * (T / 32) - 1) / (G.splits * (T / 32));
    int next = min(npath, (part * (T / 32) + (tid >> 5)) * per_w);
    const int last = min(npath, next + per_w);
    const R x_start = (R)A.kx[i], y_start = (R)A.ky[i];
    R x = x_start, y = y_start, n0 = (R)0, n1 = (R)0;
    double Yv = 1.0;
    int p = 0, k = 0;
    bool active = false;
    for (unsigned it = 0;; ++it) {
        if ((it & 3) == 0) {
            const unsigned want = __ballot_sync(kAll, !active && sub == 0);
            if (!active) {
                p = next + __popc(want & ((1u << lead) - 1u));
                if (p < last) {
                    active = true;
                    x = x_start;
                    y = y_start;
                    Yv = 1.0;
                    k = 0;
                    for (int q = 0; q < nw4; ++q) {
                        S[q * T] = 0.0;
                        dZ[q * T] = 0.0;
                    }
                }
            }
            next = min(last, next + __popc(want));
            if (!__any_sync(kAll, active)) break;
            if (active) Num<R>::normals(A.seed, (uint32_t)i, kw, (uint32_t)(k + sub), (uint32_t)p, n0, n1);
        }
        const int src = lead + (int)(it & 3);
        const R xi0 = __shfl_sync(kAll, n0, src), xi1 = __shfl_sync(kAll, n1, src);
        if (active && k >= max_steps) active = false;     // a capped path adds nothing to the c and g sums
        const double xd = (double)x, yd = (double)y;
        // c and f at X_k: each lane its own basis functions, the two sums over the four lanes
        double cv = 0.0, fv = 0.0;
        if (P.c_kind == PDD_C_RBF) {
            double s = 0.0;
#pragma unroll 2
            for (int q = sub, j = 0; q < nw; q += kGradLanes, ++j) {
                const double ddx = xd - rx[q], ddy = yd - ry[q];
                const double e = exp_neg(-(ddx * ddx + ddy * ddy) * inv2s, etab);
                psi[j * T] = e;
                s += rw[q] * e;
            }
            s += __shfl_xor_sync(kAll, s, 1);
            s += __shfl_xor_sync(kAll, s, 2);
            cv = s < 0.0 ? s : 0.0;
        } else {
            cv = (sizeof(R) == 8) ? killing(P, xd, yd) : (double)killing32(P, (float)x, (float)y);
        }
        const double yh = active ? Yv * A.h : 0.0;
        if (nf) {
            // f's weights: dZ_{k+1} / dv_q = dZ_k / dv_q + psi^f_q(X_k) Y_k h
            double s = 0.0;
            for (int q = sub, j = 0; q < nf; q += kGradLanes, ++j) {
                const double ddx = xd - fx[q], ddy = yd - fy[q];
                const double e = exp_neg(-(ddx * ddx + ddy * ddy) * inv2f, etab);
                Gf[j * T] += e * yh;
                s += fw[q] * e;
            }
            s += __shfl_xor_sync(kAll, s, 1);
            s += __shfl_xor_sync(kAll, s, 2);
            fv = s;
        }
        if (SRC && sizeof(R) == 4) fv = (double)source32(P, (float)x, (float)y);
        else if (SRC && !nf) fv = source(P, xd, yd);
        if (!active) continue;
        const double fac = cv < 0.0 ? A.h / (1.0 + cv * A.h) : 0.0;
        const double fhy = fv * yh;
#pragma unroll 4
        for (int j = 0; j < nw4; ++j) {
            const double s = S[j * T];
            if (SRC) dZ[j * T] += fhy * s;
            S[j * T] = s + psi[j * T] * fac;
        }
        Yv = Yv * (1.0 + cv * A.h);
        R bx, by;
        Num<R>::drift(P, x, y, bx, by);
        const R nx = x + bx * h + sh * xi0;
        const R ny = y + by * h + sh * xi1;
        ++k;
        const R ex0 = nx - rcx, ey0 = ny - rcy;
        const bool out_c = !(ex0 * ex0 + ey0 * ey0 < r2);
        const bool out_d = !inside_domain(Ps, (double)nx, (double)ny);
        if (!out_c && !out_d) {
            x = nx;
            y = ny;
            continue;
        }
        active = false;
        const double dx = (double)nx - xd, dy = (double)ny - yd;
        double tc = 2.0, td = 2.0;
        int ed = -1;
        if (out_c) tc = circle_exit_t(xd, yd, dx, dy, cx, cy, rs);
        if (out_d) {
            if (Ps.dom_kind == 0) {
                double t;
                if ((double)nx <= Ps.dom[0]) { t = (Ps.dom[0] - xd) / dx; if (t < td) { td = t; ed = 3; } }
                if ((double)nx >= Ps.dom[2]) { t = (Ps.dom[2] - xd) / dx; if (t < td) { td = t; ed = 1; } }
                if ((double)ny <= Ps.dom[1]) { t = (Ps.dom[1] - yd) / dy; if (t < td) { td = t; ed = 0; } }
                if ((double)ny >= Ps.dom[3]) { t = (Ps.dom[3] - yd) / dy; if (t < td) { td = t; ed = 2; } }
            } else {
                td = circle_exit_t(xd, yd, dx, dy, Ps.dom[0], Ps.dom[1], Ps.dom[2]);
                ed = 0;
            }
        }
        const bool proj = A.shift > 0.0;
        double payoff = 0.0;
        if (td <= tc) {
            double ex = xd + td * dx, ey = yd + td * dy;
            if (proj) {                          // projection onto the true boundary
                ex = (double)nx;
                ey = (double)ny;
                if (P.dom_kind == 0) {
                    ex = ex < P.dom[0] ? P.dom[0] : (ex > P.dom[2] ? P.dom[2] : ex);
                    ey = ey < P.dom[1] ? P.dom[1] : (ey > P.dom[3] ? P.dom[3] : ey);
                    if (ed == 0) ey = P.dom[1];
                    else if (ed == 1) ex = P.dom[2];
                    else if (ed == 2) ey = P.dom[3];
                    else ex = P.dom[0];
                }
            }
            const double su = boundary_s(P, ex, ey, ed);
            if (ng) {
                // the boundary series and its coefficients' derivatives share their basis values
                const int kc = (P.n_gcoef + 1) / 2;
                const double wv = PDD_TWO_PI * su / P.perimeter;
                for (int kk = sub, j = 0; kk < ng; kk += kGradLanes, ++j) {
                    const double basis = (kk < kc) ? cos(kk * wv) : sin((kk - kc + 1) * wv);
                    Gg[j * T] += Yv * basis;
                    payoff += P.g_coef[kk] * basis;
                }
                payoff += __shfl_xor_sync(gmask, payoff, 1);
                payoff += __shfl_xor_sync(gmask, payoff, 2);
            } else {
                boundary_point(P, su, ex, ey);
                payoff = gdata(P, ex, ey, su);
            }
        } else {
            const double ex = proj ? (double)nx : xd + tc * dx, ey = proj ? (double)ny : yd + tc * dy;
            double th = atan2(ey - cy, ex - cx);
            if (th < 0.0) th += PDD_TWO_PI;
            double su = th - A.theta_s[m];
            if (su < 0.0) su += PDD_TWO_PI;
            if (su >= PDD_TWO_PI) su -= PDD_TWO_PI;
            for (int l = sub; l < ns; l += kGradLanes) {
                double ph;
                if (imq) {
                    const double d = su - G.ku[a + l];
                    ph = 1.0 / sqrt(d * d + G.c2);
                } else {
                    double xx = remainder(su - PDD_TWO_PI * l / ns, PDD_TWO_PI);
                    ph = (xx == 0.0) ? 1.0 : sin(0.5 * ns * xx) * cos(0.5 * xx) / (sin(0.5 * xx) * ns);
                }
                payoff += alpha[l] * ph;
            }
            payoff += __shfl_xor_sync(gmask, payoff, 1);
            payoff += __shfl_xor_sync(gmask, payoff, 2);
        }
        for (int j = 0; j < nw4; ++j) Gw[j * T] += payoff * Yv * S[j * T] + dZ[j * T];
    }
    __syncthreads();
    // partial layout [c weights][f weights][g coefficients]; index q sits with the lanes of sub q mod 4
    const double scale = G.lambda[i] / npath;
    for (int q = tid; q < nw + nf + ng; q += T) {
        const double *src = (q < nw) ? Gw - tid : (q < nw + nf ? Gf - tid : Gg - tid);
        const int l = q < nw ? q : (q < nw + nf ? q - nw : q - nw - nf);
        src += (size_t)(l >> 2) * T + (l & 3);
        double s = 0.0;
        for (int t = 0; t < T; t += kGradLanes) s += src[t];
        G.partial[(long)blockIdx.x * G.n_par + q] = scale * s;
    }
}

void grad_mc(const pdd_cover &cov, const Problem &P, const pdd_assembly_opts &o, const pdd_system &sys,
             const double *u, const double *lambda, DevBuf<double> &partial, int &n_part, cudaStream_t st) {
    n_part = 0;
    const int nmc = sys.n_mc;
    const int nw = (P.c_kind == PDD_C_RBF) ? P.n_rbf : 0;
    const int ng = (P.g_kind == PDD_G_BOUNDARY_FOURIER) ? P.n_gcoef : 0;
    const int nf = (P.f_kind == PDD_F_RBF) ? P.n_frbf : 0;
    if (nmc == 0 || nw + nf + ng == 0) return;
    DevBuf<double> kinv, kcond;
    DevBuf<long> koff_m;
    build_imq_inverses(cov, o.imq_c2, kinv, koff_m, kcond, st);
    const int n_par = nw + nf + ng;
    // parts of a row: enough CTAs to even out rows of unequal path lengths over the SMs, each warp
    // keeping at least 64 paths of a full row (eight per group of four lanes) so that the lanes idle
    // while a warp's last paths finish stay few
    int dev = 0, sms = 0;
    PDD_CUDA(cudaGetDevice(&dev));
    PDD_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int splits = std::max(1, std::min({cdiv(8L * sms, nmc), cdiv(o.paths, 64 * (kGradThreads / 32)), 64}));
    partial.alloc((size_t)nmc * splits * n_par);
    DevBuf<unsigned long long> steps;
    DevBuf<int> capped;
    steps.alloc(1);
    capped.alloc(1);
    PathArgs A{sys.mc_rows.p, sys.mc_subs.p, sys.mc_kword.p, cov.kx.p, cov.ky.p, cov.cx.p, cov.cy.p, cov.r.p,
               cov.theta_s.p, o.paths, o.h, o.seed, nullptr, nullptr, nullptr, nullptr, steps.p, capped.p,
               sys.mc_np.p, nullptr, nullptr, o.boundary_shift ? kGmC0 * sqrt(o.h) : 0.0, nullptr, o.max_steps, 0, 0,
               nullptr};
    GradArgs G{u, lambda, cov.knot_ptr.p, cov.floating.p, cov.ku.p, koff_m.p, kinv.p, o.imq_c2, n_par, splits, partial.p};
    const size_t smem = grad_smem_doubles(nw, nf, ng) * sizeof(double);
    if (3 * nw + ng + nf > kGradMaxParams) fail(PDD_EINVAL, "too many gradient parameters for the replay kernel");
    const bool src = P.f_kind != PDD_F_ZERO;
#define PDD_GRAD_LAUNCH(R, SRCV)                                                                          \
    do {                                                                                                  \
        allow_smem((const void *)k_paths_grad<R, SRCV>, smem);                                            \
        PDD_LAUNCH((k_paths_grad<R, SRCV>), nmc * splits, kGradThreads, smem, st, P, A, G);                                   \
    } while (0)
    if (path_mixed(o)) {
        if (src) PDD_GRAD_LAUNCH(float, true); else PDD_GRAD_LAUNCH(float, false);
    } else {
        if (src) PDD_GRAD_LAUNCH(double, true); else PDD_GRAD_LAUNCH(double, false);
    }
#undef PDD_GRAD_LAUNCH
    n_part = nmc * splits;
}

}  // namespace pdd

namespace pdd {
__global__ void k_split_df(const double *v, float2 *out, long n) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t < n) out[t] = split_df_bits(v[t]);
}
}  // namespace pdd

// C ABI: the double-float split of the finalize's sum mode 1 (see include/pdd.h)
extern "C" pdd_status pdd_split_df(const double *v_dev, float *hilo_dev, long long n, void *stream) {
    using namespace pdd;
    try {
        if (n < 0 || (n > 0 && (!v_dev || !hilo_dev))) fail(PDD_EINVAL, "negative count or null buffer");
        if (((uintptr_t)hilo_dev & 7) != 0) fail(PDD_EINVAL, "output not 8-byte aligned");
        if (n == 0) return PDD_OK;
        cudaStream_t st = (cudaStream_t)stream;
        PDD_LAUNCH(k_split_df, (unsigned)cdiv((long)n, 256), 256, 0, st, v_dev, reinterpret_cast<float2 *>(hilo_dev),
                   (long)n);
        PDD_CUDA(cudaStreamSynchronize(st));
    } catch (const Fail &f) {
        return f.st;
    }
    return PDD_OK;
}
