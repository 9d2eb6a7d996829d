// Cholesky factor R = L L^H, L^-1 and R^-1 of the sample covariances in
// FP64, every job of a launch spread over many CTAs.
//
// What bounds it: GB300's FP64 pipe takes about two lanes per clock and SM,
// so the ~96 M lane instructions of p = 288 cost 25 ms on one SM whatever the
// code around them does (the one-CTA form measured 37.6 ms; p = 128: 4.6 ms,
// p = 64: 0.92 ms; a dirty + MVDR call takes 1.45 instead of 38.7 ms at p =
// 288, 256x256, 0.67 instead of 5.04 ms at p = 128, 0.26 instead of 1.22 ms at
// p = 64 with this form and the thresholds over all SMs).  Here the elimination
// of [R | I] runs in panels of kNb columns over all SMs:
//
//   k_fac_panel  one step of the chain: every CTA factors the kNb x kNb
//                diagonal block for itself (sqrt, reciprocal: the serial part;
//                cheaper than a second launch to share it) and eliminates it
//                from kItems vectors of its own - rows of L below the block
//                and columns of L^-1 left of it, p in all.
//   k_fac_trail  the panel's update of everything below it: the lower
//                triangle of R and the rows of the growing L^-1.
//   k_fac_out    FP32 copies, and R^-1 = L^-H L^-1 for the jobs that use it.
//
// Every element is computed by the same operations in the same order as in
// the one-CTA form that the fused server kernel and the smallest jobs keep
// (factor_job): the panels only group the subtractions, which each element
// takes in ascending column order either way.  Both give the same bits
// (tests/test_gpu_factor.py).
#include "cta_ops.cuh"

namespace img {
namespace {

// 16 columns: wide enough that the two launches of a panel (about 4 us of
// launch and ramp) stay below its chain, narrow enough that the redundant
// diagonal factor is a tenth of the work when many small jobs share the GPU.
constexpr int kNb = 16;
constexpr int kItems = 4;                           // vectors of a panel CTA
constexpr int kPanelWork = (kNb + kItems) * kNb;    // threads on elements, then one warp for divisions
constexpr int kPanelThreads = kPanelWork + 32;
constexpr int kTrailR = 16, kTrailC = 8;            // tile of a trailing CTA
constexpr int kInvT = 8;                            // tile edge of R^-1

// R^-1 is the wide solver's (cached vectors R^-1 a and the gradient's base);
// the other paths work from L^-1.
__device__ __forceinline__ bool needs_inverse(const JobDev &J) {
    return J.precision != IMG_PREC_FP32 && J.p > kMaxTcP && J.cost == IMG_COST_PWLS;
}

__global__ void k_fac_init(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.x];
    const int p = J.p;
    if (blockIdx.y == 0 && threadIdx.x == 0) {
        J.flags[3] = 0;                              // no bad pivot yet
        *J.vmax = 0ull;                              // (k_finalize)
    }
    for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < p * p; e += gridDim.y * blockDim.x) {
        const int col = e / p, row = e - col * p;
        const double2 r = J.R64[e];
        J.L64[e] = row >= col ? r : make_double2(0.0, 0.0);
        J.Li64[e] = make_double2(row == col ? 1.0 : 0.0, 0.0);
    }
}

__device__ __forceinline__ void bar_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// Thread (r, k): row r < kNb of the diagonal block, or vector r - kNb of this
// CTA, and column k.  Step j makes column j: (A) the pivot's root and
// reciprocal, (B) the scaled column, (C) its update of the columns k > j.  The
// columns of L^-1, which divide by the pivot, run one step behind; their
// divisions are one warp's, a component per lane, beside the next pivot's
// root.  The factored diagonal block itself is not stored: nothing reads it
// after its panel, and other CTAs of the launch may still have to read the
// unfactored one.
//
// Bound by the FP64 pipe's latency (root 590, reciprocal 550 cycles, 67 per
// dependent operation) and by its 19 cycles per warp instruction whatever
// lanes are live: with 8 vectors and each vector's own threads dividing, a
// panel took 49 us (34 in this form; a dirty + MVDR call of p = 288, 256x256
// went from 1.71 to 1.44 ms, of p = 64, 128x128 from 315 to 260 us).
__global__ void __launch_bounds__(kPanelThreads) k_fac_panel(JobDev *const *jobs, int j0) {
    const JobDev &J = *jobs[blockIdx.x];
    const int p = J.p;
    if (j0 >= p || (int)blockIdx.y * kItems >= p) return;
    const int nb = min(kNb, p - j0), below = p - j0 - nb;
    __shared__ double2 l[kNb][kNb];                          // finished columns of the block: l[row][col]
    __shared__ double2 xr[kNb + kItems];                     // column j of the rows
    __shared__ double sd[2][kItems][2], xc[2][kItems][2];    // entry j of the L^-1 columns before / after its
                                                             // division, by parity of j
    __shared__ double s_dj[kNb], s_inv;
    // step of the first bad pivot (a step number, not a flag: the dividing warp
    // may read it a step late and must not leave before the others do)
    __shared__ int s_bad;
    enum { kB1 = 1, kB2 = 2, kDiv = 3 };                     // named barriers
    if (threadIdx.x == 0) s_bad = J.flags[3] != 0 ? -1 : kNb + 1;
    if (threadIdx.x < 2 * kItems) sd[0][threadIdx.x >> 1][threadIdx.x & 1] = sd[1][threadIdx.x >> 1][threadIdx.x & 1] = 0.0;
    __syncthreads();
    if (s_bad < 0) return;                                   // a pivot of an earlier panel was bad
    if (threadIdx.x >= kPanelWork) {
        const int lane = threadIdx.x - kPanelWork, it = (lane >> 1) % kItems, c = lane & 1;
        for (int j = 0; j <= nb; ++j) {
            bar_sync(kDiv, kPanelThreads);                   // entry j - 1 is complete
            if (j > 0) {
                const double q = sd[(j - 1) & 1][it][c] / s_dj[j - 1];
                if (lane < 2 * kItems) xc[(j - 1) & 1][it][c] = q;
            }
            bar_sync(kB1, kPanelThreads);
            if (s_bad <= j) break;
        }
        return;
    }
    const int k = threadIdx.x % kNb, r = threadIdx.x / kNb, v = r - kNb;
    const int item = blockIdx.y * kItems + v;                // of p vectors: rows below, then columns of L^-1
    const bool diag = r < kNb;
    const bool isrow = !diag && item < below;
    const bool iscol = !diag && !isrow && item < p;
    double2 *src = nullptr;                                  // this thread's element
    if (k < nb) {
        if (diag && r < nb && r >= k) src = J.L64 + (size_t)(j0 + k) * p + j0 + r;
        else if (isrow) src = J.L64 + (size_t)(j0 + k) * p + j0 + nb + item;
        else if (iscol) src = J.Li64 + (size_t)(item - below) * p + j0 + k;
    }
    double2 a = src ? *src : make_double2(0.0, 0.0);
    if (iscol && k == 0) {
        sd[0][v][0] = a.x;
        sd[0][v][1] = a.y;
    }
    bar_arrive(kDiv, kPanelThreads);
    bool bad = false;
    for (int j = 0; j <= nb; ++j) {
        if (j < nb && diag && r == j && k == j) {
            const double d = a.x;
            if (!(d > 0.0 && isfinite(d))) s_bad = j;
            const double dj = sqrt(d);
            s_dj[j] = dj;
            s_inv = 1.0 / dj;
        }
        bar_sync(kB1, kPanelThreads);
        bad = s_bad <= j;
        if (bad) break;
        if (j < nb && k == j && ((diag && r > j) || isrow)) {
            const double inv = s_inv;
            a = make_double2(a.x * inv, a.y * inv);
            xr[r] = a;
            if (diag) l[r][j] = a;
        }
        bar_sync(kB2, kPanelWork);
        if (j < nb && k > j && ((diag && r >= k) || isrow)) {
            const double2 prod = zmulc(xr[r], xr[k]);
            a = make_double2(a.x - prod.x, a.y - prod.y);
        }
        if (j > 0 && iscol && k < nb) {
            const double2 x = make_double2(xc[(j - 1) & 1][v][0], xc[(j - 1) & 1][v][1]);
            if (k == j - 1) a = x;
            if (k >= j) {
                const double2 t = zmul(l[k][j - 1], x);
                a = make_double2(a.x - t.x, a.y - t.y);
            }
            if (k == j) {
                sd[j & 1][v][0] = a.x;
                sd[j & 1][v][1] = a.y;
            }
        }
        if (j < nb) bar_arrive(kDiv, kPanelThreads);
    }
    if (bad) {
        if (blockIdx.y == 0 && threadIdx.x == 0) J.flags[3] = 1;
        return;
    }
    if (src && !diag) *src = a;
}

// The panel's update of one tile: rows i below the panel, "columns" v of the
// augmented matrix (v < j0 + nb: column v of L^-1; else column v of the lower
// triangle of R).  FP64-pipe bound; 16 x 8 tiles keep one tile per SM near
// the end of a large factor, where tiles are few.
__global__ void __launch_bounds__(kTrailR * kTrailC) k_fac_trail(JobDev *const *jobs, int j0) {
    const JobDev &J = *jobs[blockIdx.x];
    const int p = J.p, i1 = j0 + kNb;                        // first row below (a full panel: rows follow)
    const int i0 = i1 + blockIdx.y * kTrailR, v0 = blockIdx.z * kTrailC;
    if (i0 >= p || v0 >= p || v0 > i0 + kTrailR - 1 || J.flags[3] != 0) return;
    __shared__ double2 A[kNb][kTrailR + 1], B[kNb][kTrailC + 1];
    const double2 *__restrict__ L = J.L64;
    const double2 *__restrict__ X = J.Li64;
    for (int e = threadIdx.x; e < kNb * kTrailR; e += blockDim.x) {
        const int kk = e / kTrailR, i = i0 + e % kTrailR;
        A[kk][e % kTrailR] = i < p ? L[(size_t)(j0 + kk) * p + i] : make_double2(0.0, 0.0);
    }
    for (int e = threadIdx.x; e < kNb * kTrailC; e += blockDim.x) {
        // L^-1 columns are contiguous along kk, rows of L along v
        const int kk = e % kNb, c = e / kNb, v = v0 + c;
        double2 b = make_double2(0.0, 0.0);
        if (v < i1) b = X[(size_t)v * p + j0 + kk];
        else if (v < p) b = L[(size_t)(j0 + kk) * p + v];
        B[kk][c] = b;
    }
    __syncthreads();
    const int ti = threadIdx.x % kTrailR, tc = threadIdx.x / kTrailR;
    const int i = i0 + ti, v = v0 + tc;
    if (i >= p || v > i) return;
    if (v < i1) {
        double2 *dst = J.Li64 + (size_t)v * p + i;
        double2 s = *dst;
#pragma unroll
        for (int kk = 0; kk < kNb; ++kk) {
            const double2 t = zmul(A[kk][ti], B[kk][tc]);
            s.x -= t.x;
            s.y -= t.y;
        }
        *dst = s;
    } else {
        double2 *dst = J.L64 + (size_t)v * p + i;
        double2 s = *dst;
#pragma unroll
        for (int kk = 0; kk < kNb; ++kk) {
            const double2 t = zmulc(A[kk][ti], B[kk][tc]);
            s.x -= t.x;
            s.y -= t.y;
        }
        *dst = s;
    }
}

// FP32 copies of R, L^-1 and L^-H, and R^-1(a, b) = sum_k conj(X(k, a)) X(k, b)
// over k >= max(a, b) in ascending order (the terms a tile starts with below
// that are exact zeros), 8 x 8 entries per CTA: the longest sum (p terms of
// 6 FP64 instructions) is then about a third of the launch.
__global__ void __launch_bounds__(kInvT * kInvT) k_fac_out(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.x];
    const int p = J.p, a0 = blockIdx.y * kInvT, b0 = blockIdx.z * kInvT;
    const bool bad = J.flags[3] != 0;
    if (a0 == 0 && b0 == 0 && threadIdx.x == 0) J.flags[0] = bad ? IMG_ENOTPD : 0;
    if (bad || a0 >= p || b0 >= p) return;
    const double2 *__restrict__ X = J.Li64;
    const int ta = threadIdx.x % kInvT, tb = threadIdx.x / kInvT;
    const int a = a0 + ta, b = b0 + tb;
    const bool live = a < p && b < p;
    const size_t e = (size_t)b * p + a;
    if (live) {
        const double2 x = X[e], xt = X[(size_t)a * p + b], r = J.R64[e];     // xt = L^-1(b, a)
        J.Li32[e] = make_float2((float)x.x, (float)x.y);
        J.LiH32[e] = make_float2((float)xt.x, (float)-xt.y);
        J.R32[e] = make_float2((float)r.x, (float)r.y);
    }
    if (!needs_inverse(J)) return;
    constexpr int kK = 32;
    __shared__ double2 XA[kInvT][kK + 1], XB[kInvT][kK + 1];
    double2 s = make_double2(0.0, 0.0);
    for (int k0 = max(a0, b0); k0 < p; k0 += kK) {
        __syncthreads();
        for (int q = threadIdx.x; q < kInvT * kK; q += blockDim.x) {
            const int kk = q % kK, c = q / kK, k = k0 + kk;
            const double2 z = make_double2(0.0, 0.0);
            XA[c][kk] = (k < p && a0 + c < p) ? X[(size_t)(a0 + c) * p + k] : z;
            XB[c][kk] = (k < p && b0 + c < p) ? X[(size_t)(b0 + c) * p + k] : z;
        }
        __syncthreads();
        const int n = min(kK, p - k0);
#pragma unroll 8
        for (int kk = 0; kk < n; ++kk) {
            const double2 t = zmulc(XB[tb][kk], XA[ta][kk]);
            s.x += t.x;
            s.y += t.y;
        }
    }
    if (live) J.Ri32[e] = make_float2((float)s.x, (float)s.y);
}

}  // namespace

// Factor n jobs of at most max_p antennas: two launches per kNb columns, or,
// while the launches cost more than one SM's FP64 pipe, one CTA per job in one
// launch.  A call of set_covariance + dirty image (64 pixels to 256, FP32),
// panels / one CTA: p = 2: 67 / 61 us, 4: 73 / 66, 6: 79 / 76, 8: 88 / 87, 10: 92
// / 98, 12: 97 / 106, 16: 106 / 136.
constexpr int kOneCtaP = 8;
cudaError_t launch_factor(JobDev *const *jobs, int n, int max_p, cudaStream_t st) {
    if (max_p <= kOneCtaP) return launch_factor_one(jobs, n, st);
    k_fac_init<<<dim3(n, (max_p * max_p + 1023) / 1024), 256, 0, st>>>(jobs);
    const int cols = (max_p + kTrailC - 1) / kTrailC;
    for (int j0 = 0; j0 < max_p; j0 += kNb) {
        k_fac_panel<<<dim3(n, (max_p + kItems - 1) / kItems), kPanelThreads, 0, st>>>(jobs, j0);
        const int below = max_p - j0 - kNb;
        if (below > 0) k_fac_trail<<<dim3(n, (below + kTrailR - 1) / kTrailR, cols), kTrailR * kTrailC, 0, st>>>(jobs, j0);
    }
    const int ti = (max_p + kInvT - 1) / kInvT;
    k_fac_out<<<dim3(n, ti, ti), kInvT * kInvT, 0, st>>>(jobs);
    return cudaGetLastError();
}

}  // namespace img
