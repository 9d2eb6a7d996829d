// Kernels of the bounded least-squares imager (SIMT FP32 operator path).
//
//   k_tables    separable steering tables (FP64 phase reduction + sincospi)
//   factor_job  Cholesky R = L L^H, L^-1 and R^-1 in FP64 by one CTA (the
//               fused server kernel, p <= 8; all other paths: factor.cu)
//   k_bounds    dirty image a^H R a and a^H R^-1 a over all pixels (many CTAs
//               per job), the adjoint operator with U = R_hat and R_hat^-1
//   k_finalize  MVDR bound, D, thresholds (Sec. III-D, Appendix A)
//   k_solve     persistent active-set + LSQR driver, one CTA per job
//               (Table I, Sec. V-A, Sec. V-B)
#include "cta_ops.cuh"
#include "tc_ops.cuh"
#include "tc_wide.cuh"
#include "cluster_fit.cuh"

#include <mutex>
#include <unordered_map>
#include "../../include/img.h"

namespace img {

// ---------------------------------------------------------------- tables
// El[il*p+k] = p^{-1/2} exp(-j 2 pi x_k l_il / lam), Em[im*p+k] = exp(-j 2 pi y_k m_im / lam).
// The phase argument t is reduced to r = t - rint(t) in FP64 before sincospi,
// so phases of hundreds of turns keep full accuracy.
// Tables of one job by the threads [t0, t0 + nt) of the grid dimension used.
__device__ void tables_job(const JobDev &J, int t0, int nt) {
    const int p = J.p;
    const int total = p * (J.n_l + J.n_m);
    const double sc = rsqrt((double)p);
    for (int e = t0; e < total; e += nt) {
        const bool isl = e < p * J.n_l;
        const int e2 = isl ? e : e - p * J.n_l;
        const int g = e2 / p, k = e2 - g * p;
        const double coord = isl ? J.ant[3 * k + 0] : J.ant[3 * k + 1];
        const double dir = isl ? J.lg[g] : J.mg[g];
        const double t = coord * dir / J.lam;
        const double r = t - rint(t);
        double s, c;
        sincospi(2.0 * r, &s, &c);
        if (isl) J.El[e2] = make_float2((float)(c * sc), (float)(-s * sc));
        else J.Em[e2] = make_float2((float)c, (float)(-s));
    }
}

__global__ void k_tables(JobDev *const *jobs) {
    tables_job(*jobs[blockIdx.y], blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// ---------------------------------------------------------------- factor
// Right-looking Cholesky in FP64, then L^-1 by forward substitution (one
// column per thread) and R^-1 = L^-H L^-1.  Status 0 ok, IMG_ENOTPD else.
__device__ void factor_job(const JobDev &J) {
    const int p = J.p;
    double2 *L = J.L64;
    __shared__ int bad;
    if (threadIdx.x == 0) {
        bad = 0;
    }
    for (int e = threadIdx.x; e < p * p; e += blockDim.x) L[e] = J.R64[e];
    __syncthreads();
    for (int j = 0; j < p; ++j) {
        // every thread reads the pivot itself; bad is written only by thread 0
        const double d = L[(size_t)j * p + j].x;
        const bool ok = d > 0.0 && isfinite(d);
        if (!ok) {
            if (threadIdx.x == 0) bad = 1;
            break;
        }
        const double dj = sqrt(d);
        const double inv = 1.0 / dj;
        __syncthreads();
        if (threadIdx.x == 0) L[(size_t)j * p + j] = make_double2(dj, 0.0);
        for (int i = j + 1 + threadIdx.x; i < p; i += blockDim.x) {
            double2 v = L[(size_t)j * p + i];
            L[(size_t)j * p + i] = make_double2(v.x * inv, v.y * inv);
        }
        __syncthreads();
        // trailing update of the lower triangle: L[i,k] -= L[i,j] conj(L[k,j]), j < k <= i
        const int m = p - j - 1;
        for (int t = threadIdx.x; t < m * m; t += blockDim.x) {
            const int k = j + 1 + t / m, i = j + 1 + t % m;
            if (i < k) continue;
            const double2 prod = zmulc(L[(size_t)j * p + i], L[(size_t)j * p + k]);
            const double2 v = L[(size_t)k * p + i];
            L[(size_t)k * p + i] = make_double2(v.x - prod.x, v.y - prod.y);
        }
        __syncthreads();
    }
    __syncthreads();
    if (bad) {
        if (threadIdx.x == 0) J.flags[0] = IMG_ENOTPD;
        return;
    }
    // zero the strict upper triangle
    for (int e = threadIdx.x; e < p * p; e += blockDim.x) {
        const int col = e / p, row = e - col * p;
        if (row < col) L[e] = make_double2(0.0, 0.0);
    }
    __syncthreads();
    // X = L^-1, column c by one thread
    double2 *X = J.Li64;
    for (int c = threadIdx.x; c < p; c += blockDim.x) {
        for (int i = 0; i < c; ++i) X[(size_t)c * p + i] = make_double2(0.0, 0.0);
        for (int i = c; i < p; ++i) {
            double2 s = make_double2(i == c ? 1.0 : 0.0, 0.0);
            for (int k = c; k < i; ++k) {
                const double2 t = zmul(L[(size_t)k * p + i], X[(size_t)c * p + k]);
                s.x -= t.x;
                s.y -= t.y;
            }
            const double lii = L[(size_t)i * p + i].x;
            X[(size_t)c * p + i] = make_double2(s.x / lii, s.y / lii);
        }
    }
    __syncthreads();
    // R^-1[a,b] = sum_k conj(X[k,a]) X[k,b], k >= max(a,b); FP32 copies
    for (int e = threadIdx.x; e < p * p; e += blockDim.x) {
        const int b = e / p, a = e - b * p;
        double2 s = make_double2(0.0, 0.0);
        for (int k = max(a, b); k < p; ++k) {
            const double2 t = zmulc(X[(size_t)b * p + k], X[(size_t)a * p + k]);
            s.x += t.x;
            s.y += t.y;
        }
        J.Ri32[e] = make_float2((float)s.x, (float)s.y);
        J.Li32[e] = make_float2((float)X[e].x, (float)X[e].y);
        const double2 xt = X[(size_t)a * p + b];               // L^-1(b, a)
        J.LiH32[e] = make_float2((float)xt.x, (float)-xt.y);
        J.R32[e] = make_float2((float)J.R64[e].x, (float)J.R64[e].y);
    }
    if (threadIdx.x == 0) J.flags[0] = 0;
}

// The smallest jobs' factor (launch_factor).
__global__ void k_factor_one(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.x];
    if (threadIdx.x == 0) *J.vmax = 0ull;            // (k_finalize)
    factor_job(J);
}
cudaError_t launch_factor_one(JobDev *const *jobs, int n, cudaStream_t st) {
    k_factor_one<<<n, kThreads, 0, st>>>(jobs);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- bounds
// dirty_i = Re(a_i^H R a_i) and h_i = a_i^H R^-1 a_i = ||L^-1 a_i||^2 for
// all pixels (eq. mfdimg and the MVDR denominator, the latter in whitened
// form: a sum of squares keeps its rounding error relative to h_i, where the
// quadratic form's error is relative to |a|^T |R^-1| |a|, far larger than h_i
// at a bright source), blockIdx.y = job.
__global__ void k_bounds(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.y];
    if (J.flags[0] != 0) return;
    extern __shared__ float4 smem4[];
    float2 *A = reinterpret_cast<float2 *>(smem4);
    float *red = reinterpret_cast<float *>(A + J.p * kTile);
    const int ntiles = (J.Q + kTile - 1) / kTile;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int pix0 = t * kTile;
        const int np = min(kTile, J.Q - pix0);
        fill_steer_adj(J, pix0, np, A);
        __syncthreads();
        adj_chunk(J.R32, J.p, A, red);
        if (threadIdx.x < np) J.dirty[pix0 + threadIdx.x] = red[threadIdx.x];
        __syncthreads();
        adj_chunk<true>(J.Li32, J.p, A, red);
        if (threadIdx.x < np) J.h[pix0 + threadIdx.x] = red[threadIdx.x];
        __syncthreads();
    }
}

// Tensor-core form of k_bounds: pass 1 with B = R_hat (dirty image), pass 2
// with B from V = L^-1 and the sum-of-squares epilogue (MVDR denominators
// ||L^-1 a_i||^2), over 128-pixel tiles.
template <int MODE>
__global__ void __launch_bounds__(kThreads, 1) k_bounds_tc(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.y];
    if (J.flags[0] != 0) return;
    constexpr bool BF = MODE == 2;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[2];
    __shared__ uint32_t slot;
    __shared__ double dbuf[kThreads / 32];
    __shared__ float red[2 * kTcM];
    TcWork T{};
    tc_carve(T, dyn, J.p);
    tc_setup(T, bars, &slot, J.p);
    const float sX = tc_steer_scale(J.p);
    const uint32_t idesc = idesc_f16(2 * T.Kp, BF ? 1 : 0);
    const int ntiles = tc_num_tiles(J.n_l, J.n_m);
    const int mine = ntiles > (int)blockIdx.x ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    for (int pass = 0; pass < 2; ++pass) {
        const float sB = tc_build_B<BF>(pass == 0 ? J.R32 : J.LiH32, J.p, T, dbuf);
        const float inv = pass == 0 ? 1.f / (sX * sX * sB) : 1.f / ((sX * sB) * (sX * sB));
        float *dst = pass == 0 ? J.dirty : J.h;
        tc_run_tiles(
            T, mine, idesc,
            [&](int t, int b) { tc_gen_X_steer<BF>(J, T, b, blockIdx.x + t * gridDim.x, sX); },
            [&](int t, int b) {
                if (pass == 0) tc_epilogue<BF>(T, b, red);
                else tc_epilogue<BF, true>(T, b, red);
                if (threadIdx.x < kTcM) {
                    const int i = tc_tile_pixel(blockIdx.x + t * gridDim.x, threadIdx.x, J.n_l, J.n_m);
                    if (i >= 0) dst[i] = red[threadIdx.x] * inv;
                }
                __syncthreads();
            });
    }
    post_late(J, T.timeouts);
    tc_teardown(T, J.p);
}

// max |entry| of R_hat (blockIdx.y = 0) and L^-H (1) per job, 8 blocks
// each, into J.opmax[8 w + block].
constexpr int kBoundsMaxBlocks = 8;
__global__ void k_emb_max_bounds(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.x];
    if (J.flags[0] != 0) return;
    const int w = blockIdx.y;
    const float mx = emb_absmax(w ? J.LiH32 : J.R32, J.p, blockIdx.z, gridDim.z);
    if (threadIdx.x == 0) J.opmax[w * gridDim.z + blockIdx.z] = mx;
}

// Chunked B images of R_hat (blockIdx.y = 0) and L^-H (1) per job; one
// CTA per (64-column chunk, block of kEmbRows rows): blockIdx.z = chunk *
// (512 / kEmbRows) + row block.
template <int MODE>
__global__ void k_emb_bounds(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.x];
    constexpr int kRB = 2 * kWideMaxP / kEmbRows;
    const int kc = blockIdx.z / kRB, rb = blockIdx.z - kc * kRB;
    if (J.flags[0] != 0 || kc >= wide_nk(J.p) || rb * kEmbRows >= 2 * wide_kp(J.p)) return;
    const int w = blockIdx.y;
    emb_B_chunk<MODE == 2>(w ? J.LiH32 : J.R32, J.p, J.Bimg + (size_t)w * wide_B_bytes(J.p),
                           warp_max_of(J.opmax + w * kBoundsMaxBlocks, kBoundsMaxBlocks), J.Bscale + w, kc, rb);
}

// Wide tensor-core bounds for 64 < p <= 256: dirty image (B = R_hat) and
// a^H R^-1 a = ||L^-1 a||^2 (B from V = L^-1, sum of squares) in one
// warp-specialised pass over the tiles.
template <int MODE>
__global__ void __launch_bounds__(kWideThreads, 1) k_bounds_wide(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.y];
    if (J.flags[0] != 0) return;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[kWideBars];
    __shared__ uint32_t slot;
    const int ntiles = tc_num_tiles(J.n_l, J.n_m);
    const int mine = ntiles > (int)blockIdx.x ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    float *dirty = J.dirty, *h = J.h;
    const int to = wide_adjoint<MODE == 2>(J, dyn, bars, &slot, J.Bimg, J.Bimg + wide_B_bytes(J.p), J.Bscale, 2,
                                           blockIdx.x, gridDim.x, mine, 2,
                                           [&](int s, int i, float v) { (s == 0 ? dirty : h)[i] = v; });
    post_late(J, to);
}

// max |entry| of one operator U, one value per CTA into the job's opmax, and
// its B image for k_psi_adj_wide (grid: chunks x row blocks).  Plain values
// per CTA need no cleared word before and no atomics.
template <class TC>
__global__ void k_emb_max_one(const JobDev *Jp, const TC *U) {
    const float mx = emb_absmax(U, Jp->p, blockIdx.x, gridDim.x);
    if (threadIdx.x == 0) Jp->opmax[blockIdx.x] = mx;
}
template <int MODE, class TC>
__global__ void k_emb_one(const JobDev *Jp, const TC *U, int nmax) {
    emb_B_chunk<MODE == 2>(U, Jp->p, Jp->Bimg, warp_max_of(Jp->opmax, nmax), Jp->Bscale, blockIdx.x, blockIdx.y);
}

// Wide tensor-core Psi^H vect(U) over all pixels of one job.
template <int MODE>
__global__ void __launch_bounds__(kWideThreads, 1) k_psi_adj_wide(const JobDev *Jp, double *out) {
    const JobDev &J = *Jp;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[kWideBars];
    __shared__ uint32_t slot;
    const int ntiles = tc_num_tiles(J.n_l, J.n_m);
    const int mine = ntiles > (int)blockIdx.x ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int to = wide_adjoint<MODE == 2>(J, dyn, bars, &slot, J.Bimg, J.Bimg, J.Bscale, 1, blockIdx.x, gridDim.x,
                                           mine, 0, [&](int, int i, float v) { out[i] = v; });
    post_late(J, to);
}

// ---------------------------------------------------------------- wide forward
// Blocks of G formed by k_fwd_wide, in fwd_pairs order, and the index of
// block (m, nb) in that order (-1: not formed).
struct FwdMap {
    int np;
    int m[16], nb[16];
    int idx[6][3];      // 2 Kp <= 768 features: 6 row blocks of 128, 3 column blocks of 256
};

// Pixel weights of a forward as FP32, w = x (FP64) or as they are (x null),
// and their maximum, one value per CTA.
__global__ void k_fwd_weights(const double *x, float *w, int Q, float *wmax) {
    float mx = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x) {
        float v;
        if (x) w[i] = v = (float)x[i];
        else v = w[i];
        mx = fmaxf(mx, fabsf(v));
    }
    mx = cta_max_t0(mx);
    if (threadIdx.x == 0) wmax[blockIdx.x] = mx;
}

template <int MODE>
__global__ void __launch_bounds__(kFwdThreads, 1) k_fwd_wide(const JobDev *Jp, const float *w, const float *wmax, int nmax,
                                                            FwdMap map, float *part) {
    const JobDev &J = *Jp;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[kFwdBars];
    __shared__ uint32_t slot;
    const int pr = blockIdx.y, S = gridDim.x;
    const int to = wide_forward<MODE == 2>(J, dyn, bars, &slot, w, wmax, nmax, map.m[pr], map.nb[pr], blockIdx.x, S,
                                           part + ((size_t)pr * S + blockIdx.x) * (kTcM * 256));
    post_late(J, to);
}

// K (p x p, column-major, interleaved; FP64 or FP32) from the S partials of the
// formed blocks.  With U(a, b) the sum of entry (a, b) of G, on or above the
// diagonal: K_kl = U(k,l) + U(Kp+k,Kp+l) + j (U(l,Kp+k) - U(k,Kp+l)) for k <=
// l, scaled back by 1 / (sX^2 sW); K_lk = conj(K_kl).  Every sum in a fixed
// order: group g of 4 takes s = g, g + 4, ..., then the groups in order.
//
// One CTA per 4 x 4 tile of (k, l): 4 entry kinds x 16 entries x 4 groups of
// threads.  Bound by the FP64 pipe (a conversion and an addition per
// partial), so only the entries that K takes are summed - about half of what
// the blocks hold - and small tiles keep every SM at it for small arrays.
constexpr int kAsmT = 4;
template <class Out>
__global__ void __launch_bounds__(256) k_fwd_assemble(int p, const float *part, int S, FwdMap map, const float *wmax,
                                                      int nmax, Out *K) {
    __shared__ double red[4][4][kAsmT * kAsmT];              // [group][kind][entry]
    __shared__ double s_inv;
    const int k0 = blockIdx.x * kAsmT, l0 = blockIdx.y * kAsmT;
    if (k0 > l0) return;
    const int Kp = wide_kp(p);
    constexpr size_t kBlk = (size_t)kTcM * 256;
    const int e = threadIdx.x & 15, kind = (threadIdx.x >> 4) & 3, g = threadIdx.x >> 6;
    const int hi = e >> 2, lo = e & 3;                       // lo runs along the stored rows
    // kinds: U(k, l), U(Kp+k, Kp+l), U(k, Kp+l) with k = k0 + hi, l = l0 + lo;
    // U(l, Kp+k) with l = l0 + hi, k = k0 + lo
    int a = (kind == 3 ? l0 : k0) + hi, b = (kind == 3 ? k0 : l0) + lo;
    const int ka = kind == 3 ? b : a, la = kind == 3 ? a : b;
    a += kind == 1 ? Kp : 0;
    b += kind >= 1 ? Kp : 0;
    double acc = 0.0;
    if (ka <= la && la < p) {
        const int m = a >> 7, nb = b >> 8;
        const float *q = part + (size_t)map.idx[m][nb] * S * kBlk + (size_t)(a - 128 * m) * 256 + (b - 256 * nb);
#pragma unroll 8
        for (int s = g; s < S; s += 4) acc += q[(size_t)s * kBlk];
    }
    red[g][kind][kind == 3 ? lo * kAsmT + hi : e] = acc;     // entry (k, l) at 4 (k - k0) + l - l0
    if (threadIdx.x < 32) {
        const float sX = steer_scale(p);
        const double inv = 1.0 / ((double)sX * sX * emb_scale_of(warp_max_of(wmax, nmax)));
        if (threadIdx.x == 0) s_inv = inv;
    }
    __syncthreads();
    const int k = k0 + (threadIdx.x >> 2), l = l0 + (threadIdx.x & 3);
    if (threadIdx.x >= kAsmT * kAsmT || k > l || l >= p) return;
    auto U = [&](int q) { return ((red[0][q][e] + red[1][q][e]) + red[2][q][e]) + red[3][q][e]; };
    const double re = (U(0) + U(1)) * s_inv;
    const double im = k == l ? 0.0 : (U(3) - U(2)) * s_inv;
    // component stores: a caller's FP64 matrix may be 8-byte aligned only
    Out *u = K + 2 * ((size_t)l * p + k), *v = K + 2 * ((size_t)k * p + l);
    u[0] = v[0] = (Out)re;
    u[1] = (Out)im;
    v[1] = (Out)-im;
}

// ---------------------------------------------------------------- full-image LSQR
// Unconstrained LS / WLS image with every pixel free: LSQR (Sec. V-A) on
// M = Psi (CLS) or W Psi D^-1 (PWLS, W = conj(L^-1) kron L^-1), b = vect(R_hat)
// or W vect(R_hat) = vect(I).  The bidiagonalisation runs as a stream of
// kernels, 12 per iteration for PWLS: the operators above, complex p x p
// products for the whitening, and the vector updates with their norms' partial
// sums (32 CTAs, a fixed order).  The FP64 scalars of the recurrences are in
// two sets, each written by CTA 0 of the one kernel (k_ls_scale_u, k_ls_xw)
// whose other CTAs read only the other set and the partial sums, so that every
// CTA forms the factors it needs itself.

// Sums of squares in the order of one CTA of 1024 threads: virtual thread t
// takes entries t, t + 1024, ..., its warp's butterfly gives one of 32 partial
// sums, which are added in warp order (ls_sum32).  The virtual warps are 32
// CTAs of one warp each: on one SM the FP64 additions alone took 15 us for
// 32,768 entries.
constexpr int kLsWarps = 32;
template <class F>
__device__ __forceinline__ void ls_sumsq_warp(int n, double *red, F value) {
    double acc = 0.0;
    int i = blockIdx.x * 32 + threadIdx.x;
    constexpr int st = 32 * kLsWarps, U = 8;
    for (; i + (U - 1) * st < n; i += U * st) {
        float x[U];
#pragma unroll
        for (int q = 0; q < U; ++q) x[q] = value(i + q * st);
#pragma unroll
        for (int q = 0; q < U; ++q) acc = fma((double)x[q], (double)x[q], acc);
    }
    for (; i < n; i += st) {
        const float x = value(i);
        acc = fma((double)x, (double)x, acc);
    }
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x == 0) red[blockIdx.x] = acc;
}
// Sum of the partial sums in order; one warp, every lane.
__device__ __forceinline__ double ls_sum32(const double *red) {
    const double r = red[threadIdx.x & 31];
    double s = 0.0;
#pragma unroll 8
    for (int w = 0; w < kLsWarps; ++w) s += __shfl_sync(0xffffffffu, r, w);
    return s;
}
__global__ void k_sumsq(const float *x, int n, double *red) {
    ls_sumsq_warp(n, red, [&](int i) { return x[i]; });
}
__global__ void k_sum32(const double *red, double *out) {
    const double s = ls_sum32(red);
    if (threadIdx.x == 0) *out = s;
}

// u = b: vect(R_hat) (CLS) or vect(I) (PWLS, W vect(R_hat) = vect(L^-1 R L^-H)).
__global__ void k_ls_init_u(const float2 *R32, int p, int pwls, float2 *u) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < p * p; e += gridDim.x * blockDim.x) {
        const int j = e / p, i = e - j * p;
        u[e] = pwls ? make_float2(i == j ? 1.f : 0.f, 0.f) : R32[e];
    }
}
// u = Mv - alpha u (n floats) and the partial sums of ||u||^2.
__global__ void k_ls_u(float *u, const float *Mv, int n, double *sc) {
    const float a = (float)sc[kLsAlpha];
    ls_sumsq_warp(n, sc + kLsRedU, [&](int i) {
        const float t = __fmaf_rn(-a, u[i], Mv[i]);
        u[i] = t;
        return t;
    });
}
// beta = ||u||, u /= beta (n complex), and max |u| per CTA into umax; CTA 0
// also leaves the scalars that go with u: beta and 1 / beta, and (not first)
// ||B||^2 and the plane rotation's part that needs no alpha.
__global__ void k_ls_scale_u(float2 *u, int n, double *sc, int first, float *umax) {
    __shared__ float s_us;
    const int lane = threadIdx.x & 31;
    const bool w0 = threadIdx.x < 32;
    double beta = 0.0, us = 0.0;
    if (w0) {
        beta = sqrt(ls_sum32(sc + kLsRedU));
        us = beta > 0.0 ? 1.0 / beta : 0.0;
        if (lane == 0) s_us = (float)us;
    }
    __syncthreads();
    const float f = s_us;
    float mx = 0.f;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        const float2 t = make_float2(u[e].x * f, u[e].y * f);
        u[e] = t;
        mx = fmaxf(mx, fmaxf(fabsf(t.x), fabsf(t.y)));
    }
    mx = cta_max_t0(mx);
    if (threadIdx.x == 0) umax[blockIdx.x] = mx;
    if (blockIdx.x != 0 || !w0) return;
    double anorm2 = sc[kLsAnorm2], rho = 0.0, c = 0.0, sn = 0.0;
    if (!first) {
        const double alpha = sc[kLsAlpha], rhobar = sc[kLsRhobar];
        anorm2 += alpha * alpha + beta * beta;
        rho = hypot(rhobar, beta);
        const double q = (lane == 0 ? rhobar : beta) / rho;
        c = __shfl_sync(0xffffffffu, q, 0);
        sn = __shfl_sync(0xffffffffu, q, 1);
    }
    if (lane != 0) return;
    sc[kLsBeta] = beta;
    sc[kLsUs] = us;
    if (first) {
        sc[kLsBnorm] = beta;
        return;
    }
    const double phibar = sc[kLsPhibar];
    sc[kLsAnorm2U] = anorm2;
    sc[kLsRho] = rho;
    sc[kLsC] = c;
    sc[kLsSn] = sn;
    sc[kLsPhi] = c * phibar;
    sc[kLsPhibarU] = sn * phibar;
}
// v = scale o y - beta v (first: v = scale o y) and the partial sums of ||v||^2.
__global__ void k_ls_v(float *v, const double *y, const float *scale, int Q, double *sc, int first) {
    const float b = first ? 0.f : (float)sc[kLsBeta];
    ls_sumsq_warp(Q, sc + kLsRedV, [&](int i) {
        const float t = __fmaf_rn(scale[i], (float)y[i], first ? 0.f : -__fmul_rn(b, v[i]));
        v[i] = t;
        return t;
    });
}
// alpha = ||v||, v /= alpha; first: w = v, x = 0; else x += t1 w, w = v + t2 w;
// the next forward's pixel weights wx = scale o v and their maximum per CTA;
// CTA 0 leaves the scalars that go with v.
__global__ void k_ls_xw(float *x, float *w, float *v, int Q, double *sc, int first, const float *scale, float *wx,
                        float *wmax) {
    __shared__ float s_c[3];                        // t1, t2, 1 / alpha
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x & 31;
        const double alpha = sqrt(ls_sum32(sc + kLsRedV));
        const double rho = first ? 1.0 : sc[kLsRho], c = sc[kLsC], sn = sc[kLsSn], phi = sc[kLsPhi];
        const double theta = sn * alpha;
        const double q = (lane == 0 ? phi : lane == 1 ? -theta : 1.0) / (lane == 2 ? alpha : rho);
        if (lane < 2) s_c[lane] = first ? 0.f : (float)q;
        if (lane == 2) s_c[2] = alpha > 0.0 ? (float)q : 1.f;
        if (blockIdx.x == 0 && lane == 0) {
            const double beta = sc[kLsBeta];
            sc[kLsAlpha] = alpha;
            if (first) {
                sc[kLsPhibar] = beta;
                sc[kLsRhobar] = alpha;
                sc[kLsAnorm2] = 0.0;
                sc[kLsRnorm] = beta;
                sc[kLsArnorm] = alpha * beta;
            } else {
                const double phibar = sc[kLsPhibarU];
                sc[kLsPhibar] = phibar;
                sc[kLsRhobar] = -c * alpha;
                sc[kLsAnorm2] = sc[kLsAnorm2U];
                sc[kLsRnorm] = phibar;
                sc[kLsArnorm] = phibar * alpha * fabs(c);
            }
        }
    }
    __syncthreads();
    const float t1 = s_c[0], t2 = s_c[1], ia = s_c[2];
    float mx = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x) {
        const float vi = __fmul_rn(v[i], ia);
        v[i] = vi;
        if (first) {
            w[i] = vi;
            x[i] = 0.f;
        } else {
            const float wi = w[i];
            x[i] = __fmaf_rn(t1, wi, x[i]);
            w[i] = __fmaf_rn(t2, wi, vi);
        }
        const float wv = scale[i] * vi;
        wx[i] = wv;
        mx = fmaxf(mx, fabsf(wv));
    }
    mx = cta_max_t0(mx);
    if (threadIdx.x == 0) wmax[blockIdx.x] = mx;
}
__global__ void k_ls_sigma(const float *x, const float *scale, double *sigma, int Q) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x)
        sigma[i] = (double)scale[i] * (double)x[i];
}
__global__ void k_d2c(const double2 *src, float2 *dst, int n) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
        dst[e] = make_float2((float)src[e].x, (float)src[e].y);
}

// C = op(A) op(B), p x p complex FP32 column-major; op 0: as is, 1: conjugate
// transpose.  16 x 16 output tiles, one output per thread, the next 32 terms'
// loads in flight behind the current ones: at p = 128 the product is latency,
// 64 tiles on 64 SMs (32 x 32 tiles, 16 CTAs: 13.6 us; 2 x 2 outputs on 64
// threads: 21 us).  cmax (may be null): max |C| per CTA.
__global__ void __launch_bounds__(256) k_cgemm(int p, const float2 *A, int opA, const float2 *B, int opB, float2 *C,
                                               float *cmax) {
    constexpr int kT = 16, kK = 32;
    __shared__ float2 As[kT][kK + 1], Bs[kK][kT + 1];
    const int i0 = blockIdx.x * kT, j0 = blockIdx.y * kT;
    float2 ra[2], rb[2];
    // this thread's entries q of a chunk, consecutive threads along the
    // memory's fast index: As[r][c] = op(A)[i0 + r, k0 + c], Bs[r][c] = op(B)[k0 + r, j0 + c]
    auto place = [&](int q, int &ar, int &ac, int &br, int &bc) {
        const int e = threadIdx.x + 256 * q;
        ar = opA ? e / kK : e % kT;
        ac = opA ? e % kK : e / kT;
        br = opB ? e / kT : e % kK;
        bc = opB ? e % kT : e / kK;
    };
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            int ar, ac, br, bc;
            place(q, ar, ac, br, bc);
            const int i = i0 + ar, k = k0 + ac, kk = k0 + br, j = j0 + bc;
            ra[q] = rb[q] = make_float2(0.f, 0.f);
            if (i < p && k < p) ra[q] = opA ? A[(size_t)i * p + k] : A[(size_t)k * p + i];
            if (kk < p && j < p) rb[q] = opB ? B[(size_t)kk * p + j] : B[(size_t)j * p + kk];
            if (opA) ra[q].y = -ra[q].y;
            if (opB) rb[q].y = -rb[q].y;
        }
    };
    const int ti = threadIdx.x & 15, tj = threadIdx.x >> 4;
    float2 acc = make_float2(0.f, 0.f);
    load(0);
    for (int k0 = 0; k0 < p; k0 += kK) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            int ar, ac, br, bc;
            place(q, ar, ac, br, bc);
            As[ar][ac] = ra[q];
            Bs[br][bc] = rb[q];
        }
        __syncthreads();
        if (k0 + kK < p) load(k0 + kK);
#pragma unroll
        for (int kk = 0; kk < kK; ++kk) cfma(acc, As[ti][kk], Bs[kk][tj]);
        __syncthreads();
    }
    const int i = i0 + ti, j = j0 + tj;
    const bool in = i < p && j < p;
    if (in) C[(size_t)j * p + i] = acc;
    if (!cmax) return;
    const float mx = cta_max_t0(in ? fmaxf(fabsf(acc.x), fabsf(acc.y)) : 0.f);
    if (threadIdx.x == 0) cmax[blockIdx.y * gridDim.x + blockIdx.x] = mx;
}

// ---------------------------------------------------------------- failure detection
// Self-test of the bounded waits every tensor-core kernel uses: one CTA
// allocates tensor memory, waits on an mbarrier that receives an arrival only
// when `arrive` is set - all its threads, or thread `thread` alone -, gives up
// after `polls` polls, frees the tensor memory on its normal exit path and
// reports through *status (IMG_OK or IMG_ETIMEOUT) or as an operator kernel of
// a job.  No fault, trap or endless loop is involved.
__global__ void k_wait_selftest(unsigned polls, int arrive, int thread, int *status, const JobDev *job) {
    __shared__ uint64_t bar;
    __shared__ uint32_t slot;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    if (threadIdx.x < 32) tmem_alloc(&slot, 32);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (arrive && threadIdx.x == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar)) : "memory");
    int timeouts = 0;
    if ((thread < 0 || (int)threadIdx.x == thread) && !mbar_wait(&bar, 0u, polls)) timeouts++;
    tc_fence_before();
    const bool late = cta_timed_out(timeouts);
    if (threadIdx.x < 32) tmem_dealloc(slot, 32);
    if (status && threadIdx.x == 0) *status = late ? IMG_ETIMEOUT : IMG_OK;
    if (job) post_late(*job, timeouts);
}

cudaError_t launch_wait_selftest(unsigned polls, int arrive, int thread, int *status, const JobDev *job,
                                 cudaStream_t st) {
    k_wait_selftest<<<1, kThreads, 0, st>>>(polls, arrive, thread, status, job);
    return cudaGetLastError();
}

// Bounds, preconditioner and thresholds:
//   C = N/(N-p) or 1; mvdr = C/h; D = h^2/C; std_MF = dirty/sqrt(N);
//   std_MVDR = mvdr/sqrt(N-p-1); gamma = chosen image, optionally inflated;
//   PWLS: x = D sigma (scale 1/D, upper D gamma); eps = kappa std with a floor.
struct FinalizeConsts {
    double C, sqN, dof, sqdof;
    bool pwls;
    __device__ explicit FinalizeConsts(const JobDev &J)
        : C(J.bias_c ? (double)J.N / (double)(J.N - J.p) : 1.0), sqN(sqrt((double)J.N)),
          dof((double)(J.N - J.p - 1)), sqdof(sqrt(dof)), pwls(J.cost == IMG_COST_PWLS) {}
};

// Pixel i; returns its value of the cost's dirty image (for the eps floor).
__device__ __forceinline__ double finalize_pixel(const JobDev &J, const FinalizeConsts &k, int i) {
    const double h = J.h[i];
    const double d = J.dirty[i];
    const double mv = k.C / h;
    const double mvsd = k.dof > 0 ? mv / k.sqdof : INFINITY;
    const double base = J.bound == IMG_BOUND_MF ? d : mv;
    const double sd = J.bound == IMG_BOUND_MF ? d / k.sqN : mvsd;
    double g = base;
    if (J.inflate == IMG_INFLATE_RATIO) g = (1.0 + J.alpha) * base;
    else if (J.inflate == IMG_INFLATE_STD) g = base + J.alpha * sd;
    const double D = h * h / k.C;
    double mb = mv;
    if (J.inflate == IMG_INFLATE_RATIO) mb = (1.0 + J.alpha) * mv;
    else if (J.inflate == IMG_INFLATE_STD) mb = mv + J.alpha * mvsd;
    J.mvb[i] = mb;
    J.gamma[i] = g;
    J.upper[i] = k.pwls ? D * g : g;
    J.scale[i] = k.pwls ? (float)(1.0 / D) : 1.0f;
    const double sdc = k.pwls ? mvsd : d / k.sqN;
    J.eps[i] = (float)(J.kappa * sdc);
    return k.pwls ? mv : d;
}

// Largest v > 0 over the CTA (0 when there is none; NaN is never larger).
__device__ __forceinline__ double block_max_pos(double mx, double *sbuf) {
    for (int o = 16; o; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) sbuf[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) mx = fmax(mx, sbuf[w]);
    return mx;
}

// All pixels by one CTA (the fused server kernel).
__device__ void finalize_job(const JobDev &J) {
    __shared__ double sbuf[kThreads / 32];
    const FinalizeConsts k(J);
    double mx = 0.0;
    for (int i = threadIdx.x; i < J.Q; i += blockDim.x) mx = fmax(mx, finalize_pixel(J, k, i));
    mx = block_max_pos(mx, sbuf);
    const float fl = (float)(J.eps_floor * mx);
    for (int i = threadIdx.x; i < J.Q; i += blockDim.x) J.eps[i] = fmaxf(J.eps[i], fl);
    if (threadIdx.x == 0) J.flags[1] = 1;
    __syncthreads();
}

// The same over the GPU (blockIdx.x = job): four FP64 divisions per pixel are
// bound by the FP64 pipe, 865 us for 256x256 pixels on one SM.  The maximum
// of the non-negative values goes through an integer atomicMax on their bits
// (zeroed with the factor), and the floor is a second launch.
__global__ void k_finalize(JobDev *const *jobs, int *batch_status) {
    const JobDev &J = *jobs[blockIdx.x];
    __shared__ double sbuf[kThreads / 32];
    if (batch_status && blockIdx.y == 0 && threadIdx.x == 0) batch_status[blockIdx.x] = J.flags[0];
    if (J.flags[0] != 0) return;
    const FinalizeConsts k(J);
    double mx = 0.0;
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < J.Q; i += gridDim.y * blockDim.x)
        mx = fmax(mx, finalize_pixel(J, k, i));
    mx = block_max_pos(mx, sbuf);
    if (threadIdx.x == 0 && mx > 0.0) atomicMax(J.vmax, (unsigned long long)__double_as_longlong(mx));
}
// The smallest jobs: both in one launch.
__global__ void k_finalize_one(JobDev *const *jobs, int *batch_status) {
    const JobDev &J = *jobs[blockIdx.x];
    if (batch_status && threadIdx.x == 0) batch_status[blockIdx.x] = J.flags[0];
    if (J.flags[0] == 0) finalize_job(J);
}
__global__ void k_eps_floor(JobDev *const *jobs) {
    const JobDev &J = *jobs[blockIdx.x];
    if (J.flags[0] != 0) return;
    const float fl = (float)(J.eps_floor * __longlong_as_double((long long)*J.vmax));
    for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < J.Q; i += gridDim.y * blockDim.x)
        J.eps[i] = fmaxf(J.eps[i], fl);
    if (blockIdx.y == 0 && threadIdx.x == 0) J.flags[1] = 1;
}

// ---------------------------------------------------------------- solver
struct SolveShared {
    double dbuf[kThreads / 32];
    double vbuf[kThreads / 32];
    int ibuf[kThreads / 32];
    int cbuf[kThreads / 32];
    float wsm[kTile];
    float red[kTile + 16 * kTile];
    float ls[8];          // LSQR: coefficients that warp 0 hands to the CTA
    float fm[kThreads / 32];
    uint64_t ldbar[2];    // tile loads into the two X buffers, and their parities
    uint32_t ldph;
    int lsi;
};
// At namespace scope, so that the solver's out-of-line functions address it
// (and the operand tiles, through dyn_smem) as shared memory.
__shared__ SolveShared g_solve;

// Clock cycles of a solve's phases (one thread's view; reported as doubles).
struct SolveCycles {
    long long gradient = 0, lsqr = 0, fwd = 0, adj = 0, aux[6] = {};
};

// c = T a_i for the support cache (T = L^-1 for PWLS, identity for LS), and
// its largest component magnitude (for the tensor-core operand scaling).
__device__ void cache_vector(const JobDev &J, int i, int slot, double *sbuf) {
    const int p = J.p;
    const int im = i / J.n_l, il = i - im * J.n_l;
    float2 *c = J.cvec + (size_t)slot * p;
    const bool pwls = J.cost == IMG_COST_PWLS;
    float mx = 0.f;
    for (int k = threadIdx.x; k < p; k += blockDim.x) {
        float2 s = make_float2(0.f, 0.f);
        if (!pwls) {
            s = steer(J, il, im, k);
        } else {
            for (int l = 0; l <= k; ++l) cfma(s, J.Li32[(size_t)l * p + k], steer(J, il, im, l));
        }
        c[k] = s;
        mx = fmaxf(mx, fmaxf(fabsf(s.x), fabsf(s.y)));
    }
    mx = block_max_f(mx, sbuf);
    if (threadIdx.x == 0) J.cmax[slot] = mx;
    __syncthreads();
}

// Power-of-two scale for the cached vectors of a list (max |entry| <= 1),
// lifted by kLift (the tiles' split parts stay normal FP16 numbers).
__device__ float list_scale(const JobDev &J, const int *pos, int n, double *sbuf) {
    float mx = 0.f;
    for (int j = threadIdx.x; j < n; j += blockDim.x) mx = fmaxf(mx, J.cmax[pos ? pos[j] : j]);
    mx = block_max_f(mx, sbuf);
    return (mx > 0.f ? exp2f(-ceilf(log2f(mx))) : 1.f) * kLift;
}

// K = base + sum_j wt[j] c_j c_j^H over a list of cached vectors, on tensor
// cores when MODE != 0 and Kp = 64, else on CUDA cores.
template <int MODE>
__device__ void forward_cache(const JobDev &J, TcWork &T, const int *pos, const float *wt, int n,
                              const float2 *base, bool base_identity, float2 *K, float2 *A,
                              float *wsm, double *dbuf) {
    if constexpr (MODE != 0) {
        if (T.Kp == 64) {
            constexpr bool BF = MODE == 2;
            const float sX = list_scale(J, pos, n, dbuf);
            tc_forward<BF>(T, J.p, n, wt, sX,
                           [&](int t, int np) { tc_gen_X_cache<BF>(J, T, 0, pos, t * kTcM, np, sX); },
                           base, base_identity, K, dbuf);
            return;
        }
    }
    forward_list(J, pos, wt, n, false, base, base_identity, K, A, wsm);
}

// Adjoint over a list of cached vectors: t_j = Re(c_j^H U c_j), handed to
// epi(j, t_j) on threads < tile size.  MODE 0: CUDA cores (FP32); 1/2:
// tensor cores with split FP16 / BF16 operands.
template <int MODE, class Epi>
__device__ void adjoint_list(const JobDev &J, const float2 *U, const int *pos, int n, float2 *A,
                             TcWork &T, float *red, double *dbuf, Epi epi) {
    if constexpr (MODE == 0) {
        for (int j0 = 0; j0 < n; j0 += kTile) {
            const int np = min(kTile, n - j0);
            fill_cache_adj(J, pos, j0, np, A);
            __syncthreads();
            adj_chunk(U, J.p, A, red);
            if (threadIdx.x < np) epi(j0 + threadIdx.x, red[threadIdx.x]);
            __syncthreads();
        }
    } else {
        constexpr bool BF = MODE == 2;
        const float sB = tc_build_B<BF>(U, J.p, T, dbuf);
        const float sXl = list_scale(J, pos, n, dbuf);
        const uint32_t idesc = idesc_f16(2 * T.Kp, BF ? 1 : 0);
        tc_run_tiles(
            T, (n + kTcM - 1) / kTcM, idesc,
            [&](int t, int b) {
                const int j0 = t * kTcM;
                tc_gen_X_cache<BF>(J, T, b, pos, j0, min(kTcM, n - j0), sXl);
            },
            [&](int t, int b) {
                const int j0 = t * kTcM;
                const int np = min(kTcM, n - j0);
                tc_epilogue<BF>(T, b, red);
                const float inv = 1.f / (sXl * sXl * sB);
                if (threadIdx.x < np) epi(j0 + threadIdx.x, red[threadIdx.x] * inv);
                __syncthreads();
            });
    }
}

// Full-image adjoint with generated steering vectors: epi(i, Re(a_i^H U a_i))
// for every pixel of tiles t0, t0 + dt, ..., on one thread per pixel.  SQ: epi(i, ||V a_i||^2) with V
// = U on CUDA cores (U column-major) and V = U^H on tensor cores (the B
// operand's convention), i.e. U = L^-1 resp. L^-H for the whitened MVDR
// denominator.
template <int MODE, bool SQ = false, class Epi, class Pre>
__device__ void adjoint_full(const JobDev &J, const float2 *U, float2 *A, TcWork &T, float *red,
                             double *dbuf, int t0, int dt, Epi epi, Pre pre) {
    const int Q = J.Q;
    if constexpr (MODE == 0) {
        const int ntiles = (Q + kTile - 1) / kTile;
        for (int t = t0; t < ntiles; t += dt) {
            const int pix0 = t * kTile;
            const int np = min(kTile, Q - pix0);
            fill_steer_adj(J, pix0, np, A);
            __syncthreads();
            adj_chunk<SQ>(U, J.p, A, red);
            if (threadIdx.x < np) {
                pre(pix0 + threadIdx.x);
                epi(pix0 + threadIdx.x, red[threadIdx.x]);
            }
            __syncthreads();
        }
    } else {
        constexpr bool BF = MODE == 2;
        const float sB = tc_build_B<BF>(U, J.p, T, dbuf);
        const float sX = tc_steer_scale(J.p);
        const float inv = SQ ? 1.f / ((sX * sB) * (sX * sB)) : 1.f / (sX * sX * sB);
        const uint32_t idesc = idesc_f16(2 * T.Kp, BF ? 1 : 0);
        const int ntiles = tc_num_tiles(J.n_l, J.n_m);
        tc_run_tiles(
            T, t0 < ntiles ? (ntiles - 1 - t0) / dt + 1 : 0, idesc,
            [&](int k, int b) { tc_gen_X_steer<BF>(J, T, b, t0 + k * dt, sX); },
            [&](int k, int b) {
                tc_epilogue<BF, SQ>(T, b, red);
                if (threadIdx.x < kTcM) {
                    const int i = tc_tile_pixel(t0 + k * dt, threadIdx.x, J.n_l, J.n_m);
                    if (i >= 0) epi(i, red[threadIdx.x] * inv);
                }
                __syncthreads();
            },
            [&](int k) {
                if (threadIdx.x < kTcM) {
                    const int i = tc_tile_pixel(t0 + k * dt, threadIdx.x, J.n_l, J.n_m);
                    if (i >= 0) pre(i);
                }
            });
    }
}

template <int MODE, bool SQ = false, class Epi>
__device__ void adjoint_full(const JobDev &J, const float2 *U, float2 *A, TcWork &T, float *red,
                             double *dbuf, Epi epi) {
    adjoint_full<MODE, SQ>(J, U, A, T, red, dbuf, 0, 1, epi, [](int) {});
}

// LSQR (Paige-Saunders) on the free set: min || b - M_F x ||, with
// M_F x = vect(sum_j s_j x_j c_j c_j^H) and (M_F^H u)_j = s_j Re(c_j^H U c_j).
// b is in J.W0 on entry.  The bidiagonalisation follows eq. initbeta ..
// eq. lanczos; rotations and stopping tests as in the FP64 oracle, scalars in
// FP64.  The u-space vector is kept unnormalised: W0 holds t with u = t * us
// (us = 1/beta), which saves a normalisation pass per iteration.  Returns the
// iteration count; the solution is in J.xs[0..f).
//
// The FP64 scalars are computed by warp 0 alone, independent divisions and
// roots in neighbouring lanes, and handed to the CTA as the FP32 coefficients
// it uses: the FP64 pipe takes a warp instruction per 16 cycles and SM, so the
// same scalars in all 8 warps cost 25,000 of the 50,000 cycles of an
// iteration at p = 48 (f <= 256).
template <int MODE>
__device__ int lsqr_cta(const JobDev &J, int f, float2 *A, TcWork &T, SolveShared &S, SolveCycles &cyc) {
    const int p = J.p, pp = p * p;
    const int *__restrict__ fpos = J.fpos;
    float2 *__restrict__ t = J.W0;
    float *v = J.v, *w = J.w, *xs = J.xs, *sF = J.sF, *wt = J.xs + J.cap;
    {
        const int *__restrict__ supp = J.supp;
        const float *__restrict__ scale = J.scale;
        for (int j = threadIdx.x; j < f; j += blockDim.x) sF[j] = scale[supp[fpos[j]]];
    }
    float acc = 0.f;     // per-thread partial (<= 16 terms), reduced in FP64
    for (int e = threadIdx.x; e < pp; e += blockDim.x) acc = fmaf(t[e].x, t[e].x, fmaf(t[e].y, t[e].y, acc));
    const bool w0 = threadIdx.x < 32;
    const int lane = threadIdx.x & 31;
    // scalars of the recurrence, valid in warp 0
    double alpha = 0.0, beta = 0.0, bnorm = 0.0, us = 0.0, phibar = 0.0, rhobar = 0.0, anorm2 = 0.0;
    {
        const double ss = block_sum_w0((double)acc, S.dbuf);
        if (w0) {
            beta = bnorm = phibar = sqrt(ss);
            us = 1.0 / beta;
            S.ls[0] = (float)us;
            S.lsi = beta == 0.0;
        }
    }
    for (int j = threadIdx.x; j < f; j += blockDim.x) xs[j] = 0.f;
    __syncthreads();
    if (S.lsi) {
        for (int j = threadIdx.x; j < f; j += blockDim.x) J.xs[j] = 0.f;
        __syncthreads();
        return 0;
    }
    auto adjoint = [&](auto epi) {
        adjoint_list<MODE>(J, t, fpos, f, A, T, S.red, S.dbuf, epi);
    };
    {
        const float fus = S.ls[0];
        adjoint([&](int j, float y) { v[j] = sF[j] * (y * fus); });
    }
    acc = 0.f;
    for (int j = threadIdx.x; j < f; j += blockDim.x) acc = fmaf(v[j], v[j], acc);
    {
        const double ss = block_sum_w0((double)acc, S.dbuf);
        if (w0) {
            alpha = rhobar = sqrt(ss);
            S.ls[5] = (float)(1.0 / alpha);
            S.ls[0] = (float)(alpha * us);
            S.lsi = alpha == 0.0;
        }
    }
    __syncthreads();
    int it = 0;
    if (S.lsi) {
        for (int j = threadIdx.x; j < f; j += blockDim.x) J.xs[j] = 0.f;
        __syncthreads();
        return 0;
    }
    {
        const float ia = S.ls[5];
        for (int j = threadIdx.x; j < f; j += blockDim.x) {
            v[j] *= ia;
            w[j] = v[j];
        }
    }
    __syncthreads();
    const int maxit = J.lsqr_maxit > 0 ? J.lsqr_maxit : 4 * f + 20;
    const double atol = J.lsqr_atol, btol = J.lsqr_btol;
    for (it = 1; it <= maxit; ++it) {
        // t <- M v - alpha u  (u = t * us), beta = ||t||
        for (int j = threadIdx.x; j < f; j += blockDim.x) wt[j] = sF[j] * v[j];
        __syncthreads();
        long long tc0 = clock64();
        const float fa = S.ls[0];
        acc = 0.f;
        forward_cache<MODE>(J, T, fpos, wt, f, nullptr, false, J.W1, A, S.wsm, S.dbuf);
        const float2 *__restrict__ W1 = J.W1;
        for (int e = threadIdx.x; e < pp; e += blockDim.x) {
            const float2 mv = W1[e];
            const float2 to = t[e];
            const float2 tn = make_float2(mv.x - fa * to.x, mv.y - fa * to.y);
            t[e] = tn;
            acc = fmaf(tn.x, tn.x, fmaf(tn.y, tn.y, acc));
        }
        cyc.fwd += clock64() - tc0;
        double ss = block_sum_w0((double)acc, S.dbuf);
        if (w0) {
            beta = sqrt(ss);
            us = beta > 0.0 ? 1.0 / beta : 0.0;
            anorm2 += alpha * alpha + beta * beta;
            S.ls[1] = (float)beta;
            S.ls[2] = (float)us;
        }
        __syncthreads();
        // v <- M^H u - beta v
        const float fb = S.ls[1], fus = S.ls[2];
        tc0 = clock64();
        adjoint([&](int j, float y) { v[j] = sF[j] * (y * fus) - fb * v[j]; });
        cyc.adj += clock64() - tc0;
        acc = 0.f;
        for (int j = threadIdx.x; j < f; j += blockDim.x) acc = fmaf(v[j], v[j], acc);
        ss = block_sum_w0((double)acc, S.dbuf);
        double absc = 0.0;
        if (w0) {
            // plane rotation; lanes 0..2: c, s, 1/alpha, then lanes 0, 1: the coefficients
            alpha = sqrt(ss);
            const double rho = hypot(rhobar, beta);
            const double q = (lane == 0 ? rhobar : lane == 1 ? beta : 1.0) / (lane == 2 ? alpha : rho);
            const double c = __shfl_sync(0xffffffffu, q, 0), sn = __shfl_sync(0xffffffffu, q, 1);
            const double ialpha = __shfl_sync(0xffffffffu, q, 2);
            const double theta = sn * alpha;
            rhobar = -c * alpha;
            const double phi = c * phibar;
            phibar = sn * phibar;
            absc = fabs(c);
            const double t = (lane == 0 ? phi : -theta) / rho;
            if (lane < 2) S.ls[3 + lane] = (float)t;
            if (lane == 0) S.ls[5] = alpha > 0.0 ? (float)ialpha : 1.f;
        }
        __syncthreads();
        const float t1 = S.ls[3], t2 = S.ls[4], ia = S.ls[5];
        acc = 0.f;
        for (int j = threadIdx.x; j < f; j += blockDim.x) {
            const float vj = v[j] * ia;                 // v <- v / alpha
            v[j] = vj;
            const float xj = xs[j] + t1 * w[j];
            xs[j] = xj;
            w[j] = vj + t2 * w[j];
            acc = fmaf(xj, xj, acc);
        }
        ss = block_sum_w0((double)acc, S.dbuf);
        if (w0) {
            const double q = sqrt(lane == 0 ? ss : anorm2);
            const double xnorm = __shfl_sync(0xffffffffu, q, 0), anorm = __shfl_sync(0xffffffffu, q, 1);
            const double rnorm = phibar;
            const double arnorm = phibar * alpha * absc;
            S.lsi = rnorm <= btol * bnorm + atol * anorm * xnorm || arnorm <= atol * anorm * rnorm;
            S.ls[0] = (float)(alpha * us);
        }
        __syncthreads();
        if (S.lsi) break;
    }
    __syncthreads();
    return min(it, maxit);
}

// ---------------------------------------------------------------- resident LSQR
// LSQR on the free set on tensor cores, f <= 256 (Kp = 32) or 512 (Kp = 64),
// with everything that an iteration touches on the SM: the free-set tiles in
// shared memory (tile t in buffer t & 1; tiles beyond the second are kept
// split in global memory and brought in by bulk copies, two tiles' worth
// fewer than there are per product, because the products walk the tiles in
// opposite directions), the p x p vector t in registers (thread tid: entries
// tid + 256 k), v, w, x, s_F of free pixels tid and tid + 256 in registers.
// Above that lsqr_cta regenerates the tiles from the cached vectors for every
// product (99,000 cycles per iteration at p = 48, f = 256 .. 349).  Same arithmetic and the same order of
// every sum as lsqr_cta's; the fused multiply-adds are written out, so that
// the rounding does not depend on what the compiler contracts where.
//
// Bound by latency: a chain of small phases in one CTA, so what counts is
// the barriers and the exposed scalars (a dependent FP64 instruction takes 67
// cycles, a division 550, hypot 1,050).  The weighted rows of the forward are
// staged 64 at a time into the B region, which is free until the B image of
// t is rebuilt; the norm of t and its largest entry share a reduction, so
// that warp 0 forms beta and the rotation while the others build B and the
// MMAs run; the stopping tests run behind the next iteration's staging.
//
// Forward: Kp = 64 as the Gram matrix of the tiles on tensor cores, Kp = 32
// in FP32 from the free vectors themselves (shared memory), thread-owned
// entries of t directly: at p <= 32 the Gram matrix's read-out costs more
// than the sums, and the products keep lsqr_cta's FP32 bits.
constexpr int kResF = 2 * kTcM;         // most free pixels, Kp = 32
constexpr int kResMaxF = 4 * kTcM;      // and Kp = 64
constexpr int kResRows = 64;            // weighted rows staged at a time

// Bytes behind the operand tiles: Kp = 64: the Gram read-out's overhang over
// the B region; Kp = 32: the free vectors.  Then the weights (kResMaxF floats).
__host__ __device__ inline size_t res_extra_bytes(int p) {
    return ((p + 31) / 32 * 32 == 32 ? (size_t)kResF * p * sizeof(float2) : 1024) + kResMaxF * sizeof(float);
}

// Named barriers of the resident LSQR (0 is __syncthreads).
__device__ __forceinline__ void bar_sync(int id, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// The split B image of t, which lies (p x p, column-major) at the start of the
// B region itself: each of warps 1 .. 7 takes its chunks of t to registers
// before any of them writes.  As tc_build_B, scaled by sc.
template <bool BF16>
__device__ __forceinline__ void res_build_B(const TcWork &T, int p, float sc) {
    constexpr int kNt = kThreads - 32, kMax = 3;             // 64 x 8 chunks over 224 threads
    const int Kp = T.Kp, nc8 = Kp / 8, items = Kp * nc8;
    const float2 *t = reinterpret_cast<const float2 *>(T.Bhi());
    const int tid = threadIdx.x - 32;
    const bool vec = (p & 1) == 0;
    float2 v[kMax][8];
#pragma unroll
    for (int q = 0; q < kMax; ++q) {
        const int it = tid + q * kNt, n = it / nc8, k0 = (it - n * nc8) * 8;
        const float2 *src = t + n * p + k0;
        if (vec && n < p && k0 + 8 <= p) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 x = reinterpret_cast<const float4 *>(src)[e];
                v[q][2 * e] = make_float2(x.x, x.y);
                v[q][2 * e + 1] = make_float2(x.z, x.w);
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[q][e] = n < p && k0 + e < p ? src[e] : make_float2(0.f, 0.f);
        }
    }
    bar_sync(2, kNt);
#pragma unroll
    for (int q = 0; q < kMax; ++q) {
        const int it = tid + q * kNt, n = it / nc8, c8 = it - n * nc8;
        if (it >= items) break;
        tc_put_B<BF16>(T, n, c8, v[q], sc);
    }
    fence_async_smem();
    bar_sync(2, kNt);
}

// Rows r0 .. r0 + nst - 1 of the free set, whose tile is in buffer xb, times
// sW w[row] (zero from row f on) as an MN-major operand of kResRows rows per feature block at dst
// (hi, then lo), re-split.
template <bool BF16>
__device__ __forceinline__ void res_stage_rows(const TcWork &T, unsigned char *dst, int xb, int r0, int nst, int f,
                                               const float *w, float sW) {
    const int nch = 2 * T.Kp / 8;
    const size_t half_bytes = (size_t)(2 * T.Kp / 64) * kResRows * 128;
    const int rt = r0 % kTcM;
#pragma unroll 2
    for (int it = threadIdx.x; it < nst * nch; it += kThreads) {
        const int rr = it / nch, c = it - rr * nch;
        const uint32_t src = sw128_off(rt + rr, c, kTcM);
        const uint32_t off = sw128_off(rr, c, kResRows);
        const float wr = r0 + rr < f ? sW * w[r0 + rr] : 0.f;
        const uint4 h4 = *reinterpret_cast<const uint4 *>(T.Xhi(xb) + src);
        const uint4 l4 = *reinterpret_cast<const uint4 *>(T.Xlo(xb) + src);
        const uint32_t hw[4] = {h4.x, h4.y, h4.z, h4.w}, lw[4] = {l4.x, l4.y, l4.z, l4.w};
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 h = unpack2<BF16>(hw[q]), l = unpack2<BF16>(lw[q]);
            split2<BF16>(__fmul_rn(wr, h.x + l.x), __fmul_rn(wr, h.y + l.y), hi[q], lo[q]);
        }
        *reinterpret_cast<uint4 *>(dst + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4 *>(dst + half_bytes + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
}

//
// Out of line: inlined into k_solve the two spilled 2.5 KB per thread.
// NP: free pixels per thread (1: f <= 256, at most two tiles).
template <int MODE, int NP>
__device__ __noinline__ int lsqr_resident(const JobDev &J, int f, TcWork &Tio, SolveCycles &cio) {
    constexpr bool BF = MODE == 2;
    TcWork T = Tio;
    T.base = dyn_smem();
    SolveCycles cyc;
    const int p = J.p, pp = p * p, Kp = T.Kp, N = 2 * Kp;
    const bool gram = Kp == 64;
    SolveShared &S = g_solve;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool w0 = warp == 0;
    const int ntiles = (f + kTcM - 1) / kTcM;
    const bool stream = NP > 1 && ntiles > 2;     // tiles beyond two come and go through the image
    const int *__restrict__ fpos = J.fpos;
    unsigned char *extra = T.Blo() + (T.Blo() - T.Bhi());
    float2 *C = reinterpret_cast<float2 *>(extra);                              // Kp = 32: free vectors
    float *wt = reinterpret_cast<float *>(extra + res_extra_bytes(p)) - kResMaxF;
    const float sX = list_scale(J, fpos, f, S.dbuf);
    const uint32_t tile_bytes = 2 * T.x_bytes();
    for (int t = 0; t < ntiles; ++t) {
        if (t >= 2) __syncthreads();              // the buffer's last tile is in the image
        tc_gen_X_cache<BF>(J, T, t & 1, fpos, t * kTcM, min(kTcM, f - t * kTcM), sX);
        if (stream) {
            __syncthreads();
            const uint4 *src = reinterpret_cast<const uint4 *>(T.Xhi(t & 1));
            uint4 *dst = reinterpret_cast<uint4 *>(J.ximg + (size_t)t * tile_bytes);
            for (uint32_t e = threadIdx.x; e < tile_bytes / 16; e += kThreads) dst[e] = src[e];
        }
    }
    if (stream) asm volatile("fence.proxy.async;" ::: "memory");
    uint32_t ldph = S.ldph;                       // parities of the tile loads
    // tile t from the image into its buffer (thread 32, after a barrier that
    // ended every use of the buffer); no more copies once one was late
    auto load_tile = [&](int t) {
        if (T.timeouts) return;
        uint64_t *bar = &S.ldbar[t & 1];
        mbar_expect_tx(bar, tile_bytes);
        tma_bulk_g2s(T.Xhi(t & 1), J.ximg + (size_t)t * tile_bytes, tile_bytes, bar);
    };
    auto wait_tile = [&](int b) {
        const uint32_t par = (ldph >> b) & 1u;
        if (mbar_wait(&S.ldbar[b], par, T.timeouts ? 1u : kSpinLimit)) return;
        // a late copy may still write the buffer: once more before going on
        if (T.timeouts++ == 0) mbar_wait(&S.ldbar[b], par);
    };
    if (!gram)
        for (int e = threadIdx.x; e < f * p; e += kThreads) {
            const int r = e / p;
            C[e] = J.cvec[(size_t)fpos[r] * p + e - r * p];
        }
    // free pixels tid + 256 m
    float sF[NP], v[NP] = {}, w[NP] = {}, x[NP] = {};
    bool mine[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        const int j = threadIdx.x + m * kThreads;
        mine[m] = j < f;
        sF[m] = mine[m] ? J.scale[J.supp[fpos[j]]] : 0.f;
    }
    float2 tr[16];
    const int da = kThreads % p, dn = kThreads / p;
    const int a_first = threadIdx.x % p, n_first = threadIdx.x / p;
    float acc = 0.f, mx = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int e = threadIdx.x + k * kThreads;
        tr[k] = e < pp ? J.W0[e] : make_float2(0.f, 0.f);
        acc = fmaf(tr[k].x, tr[k].x, fmaf(tr[k].y, tr[k].y, acc));
        mx = fmaxf(mx, fmaxf(fabsf(tr[k].x), fabsf(tr[k].y)));
    }
    // CTA sum (FP64, for cta_sum in warp 0) and maximum (for cta_max), up to
    // and including their barrier
    auto reduce = [&](float sum, float m) {
        double d = (double)sum;
        for (int o = 16; o; o >>= 1) {
            d += __shfl_xor_sync(0xffffffffu, d, o);
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        }
        if (lane == 0) {
            S.dbuf[warp] = d;
            S.fm[warp] = m;
        }
        __syncthreads();
    };
    auto cta_sum = [&]() {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kThreads / 32; ++q) t += S.dbuf[q];
        return t;
    };
    auto cta_max = [&]() {
        float m = S.fm[0];
#pragma unroll
        for (int q = 1; q < kThreads / 32; ++q) m = fmaxf(m, S.fm[q]);
        return m;
    };
    auto pow2_of = [](float m) { return m > 0.f ? exp2f(-ceilf(log2f(m))) : 1.f; };
    // scalars of the recurrence, valid in warp 0
    double alpha = 0.0, beta = 0.0, bnorm = 0.0, us = 0.0, phibar = 0.0, rhobar = 0.0, anorm2 = 0.0;
    double rho = 0.0, cs = 0.0, sn = 0.0, phi = 0.0;
    // y[m] = Re(c_j^H t c_j) (scaled back), j = tid + 256 m.  Warps 1 .. 7 build
    // the B image of t and issue the MMAs while warp 0 runs scalars().  Tiles in
    // descending order: the forward, ascending, then finds tiles 0 and 1 in the
    // buffers, and this finds the last two.
    const uint32_t idesc = idesc_f16(N, BF ? 1 : 0);
    auto adjoint = [&](float *y, auto scalars) {
        const long long c0 = clock64();
        const float sB = pow2_of(cta_max()) * kLift;
        float2 *ts = reinterpret_cast<float2 *>(T.Bhi());
#pragma unroll
        for (int k = 0; k < 16; ++k)
            if (threadIdx.x + k * kThreads < pp) ts[threadIdx.x + k * kThreads] = tr[k];
        if (w0) {
            bar_arrive(1, kThreads);
            scalars();
        } else {
            bar_sync(1, kThreads);
            res_build_B<BF>(T, p, sB);
            if (threadIdx.x == 32)
                for (int t = ntiles - 1; t >= max(0, ntiles - 2); --t) tc_issue(T, t & 1, idesc);
            __syncwarp();
        }
        const long long c1 = clock64();
        for (int t = ntiles - 1; t >= 0; --t) {
            T.wait(t & 1);
            tc_fence_after();
            S.red[t * 2 * kTcM + (warp >> 2) * kTcM + 32 * (warp & 3) + lane] = tc_row_dot<BF>(T, t & 1);
            if (NP > 1 && t >= 2) {
                // buffer and accumulator to tile t - 2
                tc_fence_before();
                __syncthreads();
                if (threadIdx.x == 32) {
                    load_tile(t - 2);
                    wait_tile(t & 1);
                    tc_issue(T, t & 1, idesc);
                }
                __syncwarp();
                ldph ^= 1u << (t & 1);
            }
        }
        tc_fence_before();
        __syncthreads();
        cyc.aux[3] += c1 - c0;
        cyc.aux[5] += clock64() - c1;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
            const int j = threadIdx.x + m * kThreads;
            const float *r = S.red + (j >> 7) * 2 * kTcM + (j & (kTcM - 1));
            y[m] = mine[m] ? (r[0] + r[kTcM]) * (1.f / (sX * sX * sB)) : 0.f;
        }
    };
    // write the solution and hand back the barriers' phases and the counters
    auto leave = [&](int its) {
#pragma unroll
        for (int m = 0; m < NP; ++m)
            if (mine[m]) J.xs[threadIdx.x + m * kThreads] = x[m];
        Tio.phase = T.phase;
        Tio.timeouts = T.timeouts;
        if (threadIdx.x == 0) S.ldph = ldph;
        cio.fwd += cyc.fwd;
        cio.adj += cyc.adj;
        for (int q = 0; q < 6; ++q) cio.aux[q] += cyc.aux[q];
        __syncthreads();
        return its;
    };
    auto norm_v = [&]() {
        float n = 0.f;
#pragma unroll
        for (int m = 0; m < NP; ++m) n = fmaf(v[m], v[m], n);
        return n;
    };
    reduce(acc, mx);
    float y[NP];
    adjoint(y, [&]() {
        beta = bnorm = phibar = sqrt(cta_sum());
        us = 1.0 / beta;
        S.ls[2] = (float)us;
        S.lsi = beta == 0.0;
    });
    if (S.lsi) return leave(0);
#pragma unroll
    for (int m = 0; m < NP; ++m)
        if (mine[m]) v[m] = sF[m] * (y[m] * S.ls[2]);
    reduce(norm_v(), 0.f);
    if (w0) {
        alpha = rhobar = sqrt(cta_sum());
        S.ls[5] = (float)(1.0 / alpha);
        S.ls[0] = (float)(alpha * us);
        S.lsi = alpha == 0.0;
    }
    __syncthreads();
    if (S.lsi) return leave(0);
    mx = 0.f;
#pragma unroll
    for (int m = 0; m < NP; ++m) {
        v[m] *= S.ls[5];
        w[m] = v[m];
        const float wj = sF[m] * v[m];
        if (mine[m]) wt[threadIdx.x + m * kThreads] = wj;
        mx = fmaxf(mx, fabsf(wj));
    }
    reduce(0.f, mx);
    const int maxit = J.lsqr_maxit > 0 ? J.lsqr_maxit : 4 * f + 20;
    const double atol = J.lsqr_atol, btol = J.lsqr_btol;
    const uint32_t fdesc = idesc_f16_mn(N, BF ? 1 : 0);
    int it = 0;
    for (it = 1; it <= maxit; ++it) {
        // t <- M v - alpha u  (u = t us), beta = ||t||; the stopping tests of
        // the iteration before arrive with the first barrier
        const long long c0 = clock64();
        bool stop = false;
        float fa = 0.f, inv = 0.f;
        const float *G = nullptr;
        if (gram) {
            const float sW = pow2_of(cta_max());
            const int ngrp = (f + kResRows - 1) / kResRows;
            for (int g = 0; g < ngrp; ++g) {
                const int b = g & 1, r0 = g * kResRows, ks = (min(kResRows, f - r0) + 15) / 16;
                const int xb = (r0 / kTcM) & 1;
                unsigned char *st = T.Bhi() + b * (2 * 2 * kResRows * 128);
                if (g >= 2) {
                    T.wait(b);
                    tc_fence_after();
                }
                // groups up to g - 2 are done: an odd one ended its tile
                if (stream && (g & 1) && g >= 3 && (g + 1) / 2 < ntiles && threadIdx.x == 32) load_tile((g + 1) / 2);
                if (NP > 1 && g >= 4 && !(g & 1)) {
                    wait_tile(xb);
                    ldph ^= 1u << xb;
                }
                res_stage_rows<BF>(T, st, xb, r0, 16 * ks, f, wt, sW);
                fence_async_smem();
                __syncthreads();
                if (g == 0) {
                    fa = S.ls[0];
                    stop = it > 1 && S.lsi;
                    if (stop) break;
                }
                if (threadIdx.x == 0) {
                    tc_fence_after();
                    const uint32_t ah = smem_u32(st), al = ah + 2 * kResRows * 128;
                    const uint32_t bo = (uint32_t)((r0 % kTcM) / 8) * 1024;
                    const uint32_t bh = smem_u32(T.Xhi(xb)) + bo, bl = smem_u32(T.Xlo(xb)) + bo;
                    const uint32_t d = T.tmem + (uint32_t)(2 * N);
                    constexpr uint32_t alb = kResRows * 128, blb = kTcM * 128;
                    for (int s = 0; s < ks; ++s) {
                        const uint32_t o = s * 2048;
                        mma_f16(d, sw128_desc_mn(ah + o, alb, 1024), sw128_desc_mn(bh + o, blb, 1024), fdesc,
                                (g > 0 || s > 0) ? 1u : 0u);
                        mma_f16(d, sw128_desc_mn(ah + o, alb, 1024), sw128_desc_mn(bl + o, blb, 1024), fdesc, 1u);
                        mma_f16(d, sw128_desc_mn(al + o, alb, 1024), sw128_desc_mn(bh + o, blb, 1024), fdesc, 1u);
                    }
                    mma_commit(&T.bar[b]);
                }
            }
            if (stop) break;
            for (int g = max(0, ngrp - 2); g < ngrp; ++g) T.wait(g & 1);
            tc_fence_after();
            inv = 1.f / (sX * sX * sW);
            const long long c1 = clock64();
            G = tc_read_fwd(T, reinterpret_cast<float *>(T.Bhi()));
            cyc.aux[0] += c1 - c0;
            cyc.aux[1] += clock64() - c1;
        } else {
            __syncthreads();
            fa = S.ls[0];
            if (it > 1 && S.lsi) break;
        }
        const long long c2 = clock64();
        acc = 0.f;
        mx = 0.f;
        {
            int a = a_first, n = n_first;
#pragma unroll
            for (int k0 = 0; k0 < 16; k0 += 4) {
                if (k0 * kThreads >= pp) break;
                // four entries at a time, their reads in flight together
                float2 kv[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const bool in = threadIdx.x + (k0 + q) * kThreads < pp;
                    kv[q] = make_float2(0.f, 0.f);
                    if (gram) {
                        if (in) kv[q] = tc_k_entry(G, Kp, a, n);
                    } else if (in) {
                        const float2 *ca = C + a, *cn = C + n;
#pragma unroll 4
                        for (int r = 0; r < f; ++r) {
                            const float wq = wt[r];
                            const float2 u = ca[r * p], z = cn[r * p];
                            cfma(kv[q], make_float2(wq * u.x, wq * u.y), make_float2(z.x, -z.y));
                        }
                    }
                    a += da;
                    n += dn;
                    if (a >= p) {
                        a -= p;
                        ++n;
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float2 &t = tr[k0 + q];
                    // (f > 256: alpha u is not rounded on its own, as in
                    // lsqr_cta, which took those sizes before)
                    if (gram && stream)
                        t = make_float2(__fmaf_rn(-fa, t.x, kv[q].x * inv), __fmaf_rn(-fa, t.y, kv[q].y * inv));
                    else if (gram)
                        t = make_float2(__fmaf_rn(kv[q].x, inv, -__fmul_rn(fa, t.x)),
                                        __fmaf_rn(kv[q].y, inv, -__fmul_rn(fa, t.y)));
                    else
                        t = make_float2(__fmaf_rn(-fa, t.x, 0.f + kv[q].x), __fmaf_rn(-fa, t.y, 0.f + kv[q].y));
                    acc = fmaf(t.x, t.x, fmaf(t.y, t.y, acc));
                    mx = fmaxf(mx, fmaxf(fabsf(t.x), fabsf(t.y)));
                }
            }
        }
        reduce(acc, mx);
        const long long c3 = clock64();
        cyc.aux[2] += c3 - c2;
        cyc.fwd += c3 - c0;
        // v <- M^H u - beta v
        adjoint(y, [&]() {
            beta = sqrt(cta_sum());
            us = beta > 0.0 ? 1.0 / beta : 0.0;
            S.ls[1] = (float)beta;
            S.ls[2] = (float)us;
            anorm2 += alpha * alpha + beta * beta;
            // the rotation's part that does not need alpha; lanes 0, 1: c, s
            rho = hypot(rhobar, beta);
            const double q = (lane == 0 ? rhobar : beta) / rho;
            cs = __shfl_sync(0xffffffffu, q, 0);
            sn = __shfl_sync(0xffffffffu, q, 1);
            phi = cs * phibar;
            phibar = sn * phibar;
        });
#pragma unroll
        for (int m = 0; m < NP; ++m)
            if (mine[m]) v[m] = __fmaf_rn(sF[m], __fmul_rn(y[m], S.ls[2]), -__fmul_rn(S.ls[1], v[m]));
        cyc.adj += clock64() - c3;
        reduce(norm_v(), 0.f);
        if (w0) {
            // lanes 0..2: the coefficients of x and w, 1/alpha
            alpha = sqrt(cta_sum());
            const double theta = sn * alpha;
            rhobar = -cs * alpha;
            const double q = (lane == 0 ? phi : lane == 1 ? -theta : 1.0) / (lane == 2 ? alpha : rho);
            if (lane < 2) S.ls[3 + lane] = (float)q;
            if (lane == 2) S.ls[5] = alpha > 0.0 ? (float)q : 1.f;
        }
        __syncthreads();
        acc = 0.f;
        mx = 0.f;
#pragma unroll
        for (int m = 0; m < NP; ++m) {
            if (!mine[m]) continue;
            const float t1 = S.ls[3], t2 = S.ls[4], ia = S.ls[5];
            const float vj = __fmul_rn(v[m], ia);       // v <- v / alpha
            v[m] = vj;
            const float xj = __fmaf_rn(t1, w[m], x[m]);
            x[m] = xj;
            w[m] = __fmaf_rn(t2, w[m], vj);
            acc = fmaf(xj, xj, acc);
            const float wj = sF[m] * vj;
            wt[threadIdx.x + m * kThreads] = wj;
            mx = fmaxf(mx, fabsf(wj));
        }
        reduce(acc, mx);
        if (w0) {
            const double ss = cta_sum();
            const double q = sqrt(lane == 0 ? ss : anorm2);
            const double xnorm = __shfl_sync(0xffffffffu, q, 0), anorm = __shfl_sync(0xffffffffu, q, 1);
            const double rnorm = phibar;
            const double arnorm = phibar * alpha * fabs(cs);
            S.lsi = rnorm <= btol * bnorm + atol * anorm * xnorm || arnorm <= atol * anorm * rnorm;
            S.ls[0] = (float)(alpha * us);
        }
    }
    // a stop is seen by the iteration after the one that caused it
    return leave(it <= maxit ? it - 1 : maxit);
}

__device__ __forceinline__ double flops_fwd(int p, int n) { return 4.0 * p * (double)p * n; }
__device__ __forceinline__ double flops_adj(int p, int n) { return 8.0 * p * (double)p * n; }

// Remove support slot sl (pixel i) by moving the last entry into it.
__device__ void supp_remove(const JobDev &J, int i, int &ns) {
    const int p = J.p;
    const int sl = J.slot[i];
    const int last = ns - 1;
    if (sl != last) {
        const int moved = J.supp[last];
        for (int k = threadIdx.x; k < p; k += blockDim.x)
            J.cvec[(size_t)sl * p + k] = J.cvec[(size_t)last * p + k];
        if (threadIdx.x == 0) {
            J.supp[sl] = moved;
            J.slot[moved] = sl;
            J.cmax[sl] = J.cmax[last];
        }
    }
    if (threadIdx.x == 0) J.slot[i] = -1;
    ns = last;
    __syncthreads();
}

// Gradient and multiplier test over tiles t0, t0 + dt, ...: lambda_L = g,
// lambda_U = -g (eq. etaL, eq. etaU), FP32; the smallest lambda below its
// threshold and its pixel, this thread's share.
template <int MODE>
__device__ void gradient_tiles(const JobDev &J, const float2 *Ug, float2 *A, TcWork &T, SolveShared &S, int t0, int dt,
                               float &bestf, int &bidx) {
    const float *__restrict__ scale = J.scale;
    const float *__restrict__ eps = J.eps;
    const unsigned char *set = J.set;             // through L2: the first CTA of a cluster writes it
    float *__restrict__ grad = J.grad;
    // this thread's pixel of the tile: its scale, threshold and set
    // are loaded before the tile's MMA is awaited
    float pscale = 0.f, peps = 0.f;
    unsigned char pset = 0;
    adjoint_full<MODE>(
        J, Ug, A, T, S.red, S.dbuf, t0, dt,
        [&](int i, float val) {
            const float g = -pscale * val;
            grad[i] = g;
            if (pset != IMG_SET_F) {
                const float lam = pset == IMG_SET_U ? -g : g;
                if (lam < -peps && (lam < bestf || (lam == bestf && i < bidx))) {
                    bestf = lam;
                    bidx = i;
                }
            }
        },
        [&](int i) {
            pscale = scale[i];
            peps = eps[i];
            pset = __ldcg(set + i);
        });
}

// A job's cluster: its first CTA runs the solve, the others wait at the
// cluster barrier for its gradients and take their share of the tiles (in one
// CTA they are a quarter to a half of a solve).  J.cmd: [0] the matrix of the
// next gradient (1: W1, 2: W0; 0: done), [1] waits that ran out, [2 + 2 r], [3
// + 2 r] rank r's smallest lambda (bits) and pixel.
enum : int { kCmdDone = 0, kCmdW1 = 1, kCmdW0 = 2 };
__device__ __forceinline__ int cluster_ctas() {
    int n;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
    return n;
}
__device__ __forceinline__ int cluster_rank() {
    int r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Persistent active-set driver (Table I), one CTA or one cluster per job.
// MODE selects the adjoint's arithmetic (0 CUDA cores FP32, 1 tensor cores
// FP16x3, 2 BF16x3).
template <int MODE, bool PREP>
__global__ void __launch_bounds__(kThreads, 1)
k_solve(JobDev *const *jobs, DevInfo *batch_info, double *const *sigma_out) {
    const int nctas = cluster_ctas(), rank = cluster_rank(), job = blockIdx.x / nctas;
    const JobDev &J = *jobs[job];
    // one 1024-aligned region serves the CUDA-core chunk or the tensor tiles
    unsigned char *dyn = dyn_smem();
    float2 *A = reinterpret_cast<float2 *>(dyn);
    SolveShared &S = g_solve;
    __shared__ uint64_t tc_bar[2];
    __shared__ uint32_t tc_slot;
    DevInfo info{};
    SolveCycles cyc;
    info.status = IMG_OK;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(info.t_begin_ns));
    const int p = J.p, Q = J.Q;
    const bool pwls = J.cost == IMG_COST_PWLS;
    // tensor memory is allocated once per CTA (the permit is relinquished)
    TcWork T{};
    if constexpr (MODE != 0) {
        tc_carve(T, dyn, p);
        if (threadIdx.x == 0) {
            mbar_init(&S.ldbar[0], 1);
            mbar_init(&S.ldbar[1], 1);
            S.ldph = 0;
        }
        tc_setup(T, tc_bar, &tc_slot, p);
    }
    if constexpr (PREP) {
        // the whole job in this CTA: steering tables, factor, dirty image and
        // MVDR denominators (the adjoint of k_bounds), bounds and thresholds
        tables_job(J, threadIdx.x, blockDim.x);
        __syncthreads();
        factor_job(J);
        __syncthreads();
        if (J.flags[0] == 0) {
            adjoint_full<MODE>(J, J.R32, A, T, S.red, S.dbuf, [&](int i, float v) { J.dirty[i] = v; });
            adjoint_full<MODE, true>(J, MODE == 0 ? J.Li32 : J.LiH32, A, T, S.red, S.dbuf,
                                     [&](int i, float v) { J.h[i] = v; });
            finalize_job(J);
        }
        __syncthreads();
    }
    if (J.flags[0] != 0 || J.flags[1] != 1) {
        info.status = J.flags[0] != 0 ? J.flags[0] : IMG_EINVAL;
        if (threadIdx.x == 0 && rank == 0) {
            *J.info = info;
            if (batch_info) batch_info[job] = info;
        }
        if constexpr (MODE != 0) tc_teardown(T, p);
        return;
    }
    if (rank != 0) {
        for (;;) {
            cluster_barrier();
            const int cmd = *(volatile int *)J.cmd;
            if (cmd == kCmdDone) break;
            float bestf = INFINITY;
            int bidx = 0x7fffffff;
            gradient_tiles<MODE>(J, cmd == kCmdW1 ? J.W1 : J.W0, A, T, S, rank, nctas, bestf, bidx);
            double best = bestf;
            block_argmin(best, bidx, S.vbuf, S.ibuf);
            if (threadIdx.x == 0) {
                J.cmd[2 + 2 * rank] = __float_as_int((float)best);
                J.cmd[3 + 2 * rank] = bidx;
            }
            if (T.timeouts) J.cmd[1] = 1;       // from any thread
            cluster_barrier();
        }
        if constexpr (MODE != 0) tc_teardown(T, p);
        return;
    }
    if (threadIdx.x == 0) J.cmd[1] = 0;
    for (int i = threadIdx.x; i < Q; i += blockDim.x) {
        J.x[i] = 0.0;
        J.set[i] = IMG_SET_L;
        J.slot[i] = -1;
        J.grad[i] = 0.f;
    }
    __syncthreads();
    const long long t_start = clock64();
    int nev = 0;          // decisions so far
    auto log_event = [&](int kind, int pixel, float val) {
        if (threadIdx.x == 0 && nev < J.ev_cap) {
            J.ev[nev] = (kind << 24) | pixel;
            J.evv[nev] = val;
        }
        ++nev;
    };
    int ns = 0;           // support size |F u U|
    bool flag = true;     // Freegradient-isnotzero
    int imin = -1;
    double lam_min = 0.0;
    const int max_outer = J.max_outer > 0 ? J.max_outer : 10 * Q + 100;
    int outer = 0;
    bool converged = false;
    float *wt = J.xs + J.cap;
    while (outer < max_outer) {
        ++outer;
        if (flag) {
            const int f = block_compact(ns, [&](int pos) { return J.set[J.supp[pos]] == IMG_SET_F; },
                                        J.fpos, S.cbuf);
            bool feasible = true;
            if (f > 0) {
                // b = B0 - sum_{U} s_i x_i c_i c_i^H   (eq. bsubproblemLS / MVDR)
                const int nu = block_compact(ns, [&](int pos) { return J.set[J.supp[pos]] == IMG_SET_U; },
                                             J.fpos + f, S.cbuf);
                for (int j = threadIdx.x; j < nu; j += blockDim.x) {
                    const int i = J.supp[J.fpos[f + j]];
                    wt[j] = -J.scale[i] * (float)J.x[i];
                }
                __syncthreads();
                forward_cache<MODE>(J, T, J.fpos + f, wt, nu, pwls ? nullptr : J.R32, pwls, J.W0, A, S.wsm,
                                    S.dbuf);
                info.op_flops += flops_fwd(p, nu);
                const long long t0 = clock64();
                int its;
                if (MODE != 0 && f <= (T.Kp == 64 ? kResMaxF : kResF)) {
                    TcWork Tl = T;            // by reference only here: T stays in registers
                    SolveCycles cl;
                    its = f <= kResF ? lsqr_resident<MODE, 1>(J, f, Tl, cl) : lsqr_resident<MODE, 2>(J, f, Tl, cl);
                    T.phase = Tl.phase;
                    T.timeouts = Tl.timeouts;
                    cyc.fwd += cl.fwd;
                    cyc.adj += cl.adj;
                    for (int q = 0; q < 6; ++q) cyc.aux[q] += cl.aux[q];
                } else its = lsqr_cta<MODE>(J, f, A, T, S, cyc);
                cyc.lsqr += clock64() - t0;
                info.lsqr_iters += its;
                info.op_flops += (its + 1) * (flops_fwd(p, f) + flops_adj(p, f));
                // feasibility with the relative tolerance tau, non-strict
                int bad = MODE != 0 && T.timeouts ? 1 : 0;
                const double tau = J.feas_tol;
                for (int j = threadIdx.x; j < f; j += blockDim.x) {
                    const double z = J.xs[j];
                    const double u = J.upper[J.supp[J.fpos[j]]];
                    if (!(z >= -tau * u && z <= (1.0 + tau) * u)) bad = 1;
                }
                feasible = __syncthreads_or(bad) == 0;
                if (MODE != 0 && !feasible && cta_timed_out(T.timeouts)) break;
            }
            if (feasible) {
                for (int j = threadIdx.x; j < f; j += blockDim.x) {
                    const int i = J.supp[J.fpos[j]];
                    J.x[i] = fmin(fmax((double)J.xs[j], 0.0), J.upper[i]);
                }
                flag = false;
                __syncthreads();
                // gradient: E = B0 - sum_S s_i x_i c_i c_i^H, U_g = T^H E T
                for (int j = threadIdx.x; j < ns; j += blockDim.x) {
                    const int i = J.supp[j];
                    wt[j] = -J.scale[i] * (float)J.x[i];
                }
                __syncthreads();
                forward_cache<MODE>(J, T, nullptr, wt, ns, pwls ? nullptr : J.R32, pwls, J.W1, A, S.wsm,
                                    S.dbuf);
                info.op_flops += flops_fwd(p, ns);
                const float2 *Ug = J.W1;
                if (pwls) {
                    cgemm_pp(p, J.W1, false, J.Li32, J.W2);
                    cgemm_pp(p, J.Li32, true, J.W2, J.W0);
                    Ug = J.W0;
                }
                const long long tg = clock64();
                int bidx = 0x7fffffff;
                float bestf = INFINITY;
                if (nctas > 1) {
                    if (threadIdx.x == 0) J.cmd[0] = Ug == J.W1 ? kCmdW1 : kCmdW0;
                    cluster_barrier();
                }
                gradient_tiles<MODE>(J, Ug, A, T, S, 0, nctas, bestf, bidx);
                double best = bestf;
                info.op_flops += flops_adj(p, Q);
                block_argmin(best, bidx, S.vbuf, S.ibuf);
                if (nctas > 1) {
                    cluster_barrier();
                    if (__ldcg(J.cmd + 1)) T.timeouts++;
                    for (int r = 1; r < nctas; ++r) {
                        const float b = __int_as_float(__ldcg(J.cmd + 2 + 2 * r));
                        const int i = __ldcg(J.cmd + 3 + 2 * r);
                        if (b < (float)best || (b == (float)best && i < bidx)) {
                            best = b;
                            bidx = i;
                        }
                    }
                }
                cyc.gradient += clock64() - tg;
                lam_min = best;
                if (bidx == 0x7fffffff) {
                    converged = true;
                    break;
                }
                imin = bidx;
            } else {
                // step towards z: mu_i per eq. mumax, smallest index on ties
                double best = INFINITY;
                int bidx = 0x7fffffff;
                for (int j = threadIdx.x; j < f; j += blockDim.x) {
                    const int i = J.supp[J.fpos[j]];
                    const double xi = J.x[i];
                    const double pd = (double)J.xs[j] - xi;
                    double mu = INFINITY;
                    if (pd > 0.0) mu = (J.upper[i] - xi) / pd;
                    else if (pd < 0.0) mu = -xi / pd;
                    if (mu < best || (mu == best && i < bidx)) { best = mu; bidx = i; }
                }
                block_argmin(best, bidx, S.vbuf, S.ibuf);
                const double mu = best;
                const int ic = bidx;
                // the blocking pixel moves to U when its direction is positive
                int dirup = 0;
                for (int j = threadIdx.x; j < f; j += blockDim.x)
                    if (J.supp[J.fpos[j]] == ic) dirup = ((double)J.xs[j] - J.x[ic] > 0.0) ? 1 : 0;
                const bool up = __syncthreads_or(dirup) != 0;
                for (int j = threadIdx.x; j < f; j += blockDim.x) {
                    const int i = J.supp[J.fpos[j]];
                    const double xi = J.x[i];
                    J.x[i] = xi + mu * ((double)J.xs[j] - xi);
                }
                __syncthreads();
                if (threadIdx.x == 0) {
                    J.set[ic] = up ? IMG_SET_U : IMG_SET_L;
                    J.x[ic] = up ? J.upper[ic] : 0.0;
                }
                log_event(up ? 2 : 1, ic, (float)mu);
                __syncthreads();
                if (!up) supp_remove(J, ic, ns);
                flag = true;
            }
        } else {
            // delete a constraint: pixel imin joins F at its current value
            const int i = imin;
            if (J.slot[i] < 0) {
                if (ns >= J.cap) {
                    info.status = IMG_ENOMEM;
                    break;
                }
                cache_vector(J, i, ns, S.dbuf);
                if (threadIdx.x == 0) {
                    J.supp[ns] = i;
                    J.slot[i] = ns;
                }
                ++ns;
            }
            if (threadIdx.x == 0) J.set[i] = IMG_SET_F;
            log_event(0, i, (float)lam_min);
            __syncthreads();
            flag = true;
        }
    }
    if (nctas > 1) {
        if (threadIdx.x == 0) J.cmd[0] = kCmdDone;
        cluster_barrier();
    }
    if constexpr (MODE != 0) {
        if (cta_timed_out(T.timeouts)) info.status = IMG_ETIMEOUT;
        tc_teardown(T, p);
    }
    if (!converged && info.status == IMG_OK) info.status = IMG_ENOTCONV;
    double *out = sigma_out ? sigma_out[job] : nullptr;
    int nf = 0, nu = 0;
    for (int i = threadIdx.x; i < Q; i += blockDim.x) {
        const double s = (double)J.scale[i] * J.x[i];
        J.sigma[i] = s;
        if (out) out[i] = s;
        nf += J.set[i] == IMG_SET_F;
        nu += J.set[i] == IMG_SET_U;
    }
    const double tf = block_sum((double)nf, S.dbuf);
    const double tu = block_sum((double)nu, S.dbuf);
    if (threadIdx.x == 0) {
        info.outer = outer;
        info.n_free = (int)tf;
        info.n_upper = (int)tu;
        info.converged = converged ? 1 : 0;
        info.lambda_min = lam_min;
        info.cyc_total = (double)(clock64() - t_start);
        info.cyc_gradient = (double)cyc.gradient;
        info.cyc_lsqr = (double)cyc.lsqr;
        info.cyc_lsqr_fwd = (double)cyc.fwd;
        info.cyc_lsqr_adj = (double)cyc.adj;
        for (int q = 0; q < 6; ++q) info.cyc_aux[q] = (double)cyc.aux[q];
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(info.t_end_ns));
        *J.ev_count = nev;
        *J.info = info;
        if (batch_info) batch_info[job] = info;
    }
}

// ---------------------------------------------------------------- operators
// K = sum_i x_i a_i a_i^H over all pixels, split over CTAs into partial
// matrices part[b] (p x p each), then summed in order by k_psi_reduce.
__global__ void k_psi_partial(const JobDev *Jp, const float *wx, float2 *part, int per_cta) {
    extern __shared__ float4 smem4[];
    float2 *C = reinterpret_cast<float2 *>(smem4);
    __shared__ float wsm[kTile];
    const JobDev &J = *Jp;
    const int i0 = blockIdx.x * per_cta;
    const int n = max(0, min(per_cta, J.Q - i0));
    const int p = J.p;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float2 *K = part + (size_t)blockIdx.x * p * p;
    for (int mt = 0; mt < p; mt += kTile) {
        for (int nt = 0; nt < p; nt += kTile) {
            const int r0 = mt + ty * 4, c0 = nt + tx * 4;
            float2 acc[4][4];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);
            for (int j0 = 0; j0 < n; j0 += kTile) {
                const int np = min(kTile, n - j0);
                for (int e = threadIdx.x; e < kTile * p; e += kThreads) {
                    const int j = e / p, k = e - j * p;
                    float2 c = make_float2(0.f, 0.f);
                    if (j < np) {
                        const int i = i0 + j0 + j;
                        const int im = i / J.n_l, il = i - im * J.n_l;
                        c = steer(J, il, im, k);
                    }
                    C[e] = c;
                }
                if (threadIdx.x < kTile) wsm[threadIdx.x] = threadIdx.x < np ? wx[i0 + j0 + threadIdx.x] : 0.f;
                __syncthreads();
                if (r0 < p && c0 < p) {
                    for (int j = 0; j < np; ++j) {
                        const float wj = wsm[j];
                        const float2 *cj = C + j * p;
                        float2 ck[4], cl[4];
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            const float2 t = (r0 + r < p) ? cj[r0 + r] : make_float2(0.f, 0.f);
                            ck[r] = make_float2(wj * t.x, wj * t.y);
                        }
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float2 t = (c0 + c < p) ? cj[c0 + c] : make_float2(0.f, 0.f);
                            cl[c] = make_float2(t.x, -t.y);
                        }
#pragma unroll
                        for (int r = 0; r < 4; ++r)
#pragma unroll
                            for (int c = 0; c < 4; ++c) cfma(acc[r][c], ck[r], cl[c]);
                    }
                }
                __syncthreads();
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int k = r0 + r, l = c0 + c;
                    if (k < p && l < p) K[(size_t)l * p + k] = acc[r][c];
                }
        }
    }
}

__global__ void k_psi_reduce(const float2 *part, int nparts, int pp, double2 *Kout) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < pp; e += gridDim.x * blockDim.x) {
        double sx = 0.0, sy = 0.0;
        for (int b = 0; b < nparts; ++b) {
            const float2 v = part[(size_t)b * pp + e];
            sx += v.x;
            sy += v.y;
        }
        Kout[e] = make_double2(sx, sy);
    }
}

__global__ void k_psi_adj(const JobDev *J, const float2 *U, double *out) {
    // out_i = Re(a_i^H U a_i) over all pixels (Psi^H vect(U))
    extern __shared__ float4 smem4[];
    float2 *A = reinterpret_cast<float2 *>(smem4);
    float *red = reinterpret_cast<float *>(A + J->p * kTile);
    const int ntiles = (J->Q + kTile - 1) / kTile;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int pix0 = t * kTile;
        const int np = min(kTile, J->Q - pix0);
        fill_steer_adj(*J, pix0, np, A);
        __syncthreads();
        adj_chunk(U, J->p, A, red);
        if (threadIdx.x < np) out[pix0 + threadIdx.x] = red[threadIdx.x];
        __syncthreads();
    }
}

__global__ void k_to_double(const float *src, double *dst, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

__global__ void k_z2c(const double2 *src, float2 *dst, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[i] = make_float2((float)src[i].x, (float)src[i].y);
}

__global__ void k_c2z(const float2 *src, double2 *dst, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[i] = make_double2(src[i].x, src[i].y);
}

__global__ void k_d2f(const double *src, float *dst, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = (float)src[i];
}

// ---------------------------------------------------------------- launchers
size_t solve_smem_bytes(int p, int mode) {
    size_t b = (size_t)p * kTile * sizeof(float2);
    const size_t tc = tc_smem_bytes(p) + res_extra_bytes(p);
    if (mode != 0) b = b > tc ? b : tc;
    return b + 1024;
}
size_t bounds_smem_bytes(int p) {
    return (size_t)p * kTile * sizeof(float2) + (kTile + 16 * kTile) * sizeof(float);
}

// Raise a kernel's dynamic shared-memory limit (and prefer the maximum
// shared-memory carve-out) only when a launch needs more than any before:
// changing a function's attributes while instances of it run can hold the
// launch back, which serialised independent launches on separate streams.
static std::mutex g_attr_mu;
static std::unordered_map<const void *, size_t> g_attr;

static cudaError_t ensure_smem(const void *func, size_t bytes) {
    std::lock_guard<std::mutex> lock(g_attr_mu);
    auto it = g_attr.find(func);
    if (it != g_attr.end() && it->second >= bytes) return cudaSuccess;
    const size_t want = bytes < 48 * 1024 ? 48 * 1024 : bytes;
    cudaError_t e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(func, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    g_attr[func] = want;
    return cudaSuccess;
}

static int g_num_sms = 0;
static int num_sms() {
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    return g_num_sms;
}

cudaError_t launch_tables(JobDev *const *jobs, int n, cudaStream_t st) {
    k_tables<<<dim3(16, n), kThreads, 0, st>>>(jobs);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_bounds_tc_t(JobDev *const *jobs, int n, int max_tiles, int max_p, cudaStream_t st) {
    const size_t sm = tc_smem_bytes(max_p) + 1024;
    cudaError_t e = ensure_smem((const void *)k_bounds_tc<MODE>, sm);
    if (e != cudaSuccess) return e;
    int per_job = (num_sms() + n - 1) / n;
    per_job = max(1, min(per_job, max_tiles));
    k_bounds_tc<MODE><<<dim3(per_job, n), kThreads, sm, st>>>(jobs);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_bounds_wide_t(JobDev *const *jobs, int n, int max_tiles, int max_p, cudaStream_t st) {
    k_emb_max_bounds<<<dim3(n, 2, kBoundsMaxBlocks), kThreads, 0, st>>>(jobs);
    k_emb_bounds<MODE><<<dim3(n, 2, wide_nk(max_p) * (2 * kWideMaxP / kEmbRows)), kThreads, 0, st>>>(jobs);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t sm = wide_smem_bytes(max_p);
    e = ensure_smem((const void *)k_bounds_wide<MODE>, sm);
    if (e != cudaSuccess) return e;
    int per_job = (num_sms() + n - 1) / n;
    per_job = max(1, min(per_job, max_tiles));
    k_bounds_wide<MODE><<<dim3(per_job, n), kWideThreads, sm, st>>>(jobs);
    return cudaGetLastError();
}

cudaError_t launch_bounds(JobDev *const *jobs, int n, int max_tiles, int max_p, int mode, cudaStream_t st) {
    if (mode != 0 && max_p > kMaxTcP) {
        if (mode == 1) return launch_bounds_wide_t<1>(jobs, n, max_tiles, max_p, st);
        return launch_bounds_wide_t<2>(jobs, n, max_tiles, max_p, st);
    }
    if (mode == 1) return launch_bounds_tc_t<1>(jobs, n, (max_tiles + 1) / 2, max_p, st);
    if (mode == 2) return launch_bounds_tc_t<2>(jobs, n, (max_tiles + 1) / 2, max_p, st);
    const size_t sm = bounds_smem_bytes(max_p);
    cudaError_t e = ensure_smem((const void *)k_bounds, sm);
    if (e != cudaSuccess) return e;
    int per_job = (2 * num_sms() + n - 1) / n;
    per_job = max(1, min(per_job, max_tiles));
    k_bounds<<<dim3(per_job, n), kThreads, sm, st>>>(jobs);
    return cudaGetLastError();
}

// Up to 512 pixels one CTA per job in one launch (set_covariance + dirty image
// at p = 16, two launches / one: 256 pixels: 105 / 103 us, 400: 106 / 103, 576: 106
// / 107, 1024: 108 / 115; p = 4, 64 pixels: 73 / 67).
constexpr int kFinalizeOne = 2;              // thread blocks of pixels
cudaError_t launch_finalize(JobDev *const *jobs, int n, int max_tiles, cudaStream_t st, int *batch_status) {
    // one pixel per thread while the CTAs of all jobs stay within a few waves
    const int need = (max_tiles * kTile + kThreads - 1) / kThreads;
    if (need <= kFinalizeOne) {
        k_finalize_one<<<n, kThreads, 0, st>>>(jobs, batch_status);
        return cudaGetLastError();
    }
    const dim3 grid(n, min(need, max(1, 8 * num_sms() / n)));
    k_finalize<<<grid, kThreads, 0, st>>>(jobs, batch_status);
    k_eps_floor<<<grid, kThreads, 0, st>>>(jobs);
    return cudaGetLastError();
}

template <int MODE, bool PREP>
static cudaError_t launch_solve_t(JobDev *const *jobs, int n, size_t sm, int ctas, DevInfo *batch_info,
                                  double *const *sigma_out, cudaStream_t st) {
    cudaError_t e = ensure_smem((const void *)k_solve<MODE, PREP>, sm);
    if (e != cudaSuccess) return e;
    if (ctas > 1)
        ctas = cluster_that_fits(ctas, [&](int c) {
            return active_clusters((const void *)k_solve<MODE, PREP>, c, kThreads, sm);
        });
    if (ctas > 1) {
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim = {(unsigned)ctas, 1, 1};
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(n * ctas);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = sm;
        cfg.stream = st;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k_solve<MODE, PREP>, jobs, batch_info, sigma_out);
    }
    k_solve<MODE, PREP><<<n, kThreads, sm, st>>>(jobs, batch_info, sigma_out);
    return cudaGetLastError();
}

cudaError_t launch_solve(JobDev *const *jobs, int n, int max_p, int mode, int ctas, DevInfo *batch_info,
                         double *const *sigma_out, cudaStream_t st) {
    const size_t sm = solve_smem_bytes(max_p, mode);
    if (mode == 1) return launch_solve_t<1, false>(jobs, n, sm, ctas, batch_info, sigma_out, st);
    if (mode == 2) return launch_solve_t<2, false>(jobs, n, sm, ctas, batch_info, sigma_out, st);
    return launch_solve_t<0, false>(jobs, n, sm, ctas, batch_info, sigma_out, st);
}

cudaError_t launch_job(JobDev *const *jobs, int n, int max_p, int mode, DevInfo *batch_info,
                       double *const *sigma_out, cudaStream_t st) {
    size_t sm = solve_smem_bytes(max_p, mode);
    if (mode == 0) {
        const size_t b = bounds_smem_bytes(max_p);
        sm = sm > b ? sm : b;
    }
    if (mode == 1) return launch_solve_t<1, true>(jobs, n, sm, 1, batch_info, sigma_out, st);
    if (mode == 2) return launch_solve_t<2, true>(jobs, n, sm, 1, batch_info, sigma_out, st);
    return launch_solve_t<0, true>(jobs, n, sm, 1, batch_info, sigma_out, st);
}

// Psi x over all pixels on CUDA cores: nparts CTAs write partial p x p sums into `part`
// (nparts * p * p float2 of scratch), reduced in a fixed order in FP64.
cudaError_t launch_psi(const JobDev *job_dev, const float *wx, float2 *part, int nparts, int Q,
                       int p, double2 *Kout, cudaStream_t st) {
    const size_t sm = (size_t)p * kTile * sizeof(float2);
    cudaError_t e = ensure_smem((const void *)k_psi_partial, sm);
    if (e != cudaSuccess) return e;
    int per = (Q + nparts - 1) / nparts;
    per = ((per + kTile - 1) / kTile) * kTile;
    const int used = (Q + per - 1) / per;
    k_psi_partial<<<used, kThreads, sm, st>>>(job_dev, wx, part, per);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_psi_reduce<<<(p * p + 255) / 256, 256, 0, st>>>(part, used, p * p, Kout);
    return cudaGetLastError();
}

// Partial blocks, one per CTA, at most one CTA per SM.
size_t psi_wide_part_floats(int sms) { return (size_t)sms * kTcM * 256; }

cudaError_t launch_psi_wide(const JobDev *job_dev, const FwdIn &in, float *part, int Q, int p, int n_l, int n_m, int mode,
                            double *K64, float *K32, cudaStream_t st) {
    if (p < 1 || p > kMaxWideFwdP || (mode != 1 && mode != 2)) return cudaErrorInvalidValue;
    if (fwd_pairs(p, nullptr, nullptr) > 16) return cudaErrorInvalidValue;
    FwdMap map{};
    map.np = fwd_pairs(p, map.m, map.nb);
    for (int a = 0; a < 6; ++a)
        for (int b = 0; b < 3; ++b) map.idx[a][b] = -1;
    for (int q = 0; q < map.np; ++q) map.idx[map.m[q]][map.nb[q]] = q;
    const int sms = num_sms();
    const int nblk = fwd_nblocks(n_l, n_m);
    const int S = max(1, min(nblk, sms / map.np));
    int nmax = in.nmax;
    if (nmax == 0) {
        nmax = max(1, min(min(sms, kOpMax), (Q + 4 * kThreads - 1) / (4 * kThreads)));
        k_fwd_weights<<<nmax, kThreads, 0, st>>>(in.x, in.w, Q, in.wmax);
    }
    const size_t sm = fwd_smem_bytes();
    cudaError_t e = (mode == 1) ? ensure_smem((const void *)k_fwd_wide<1>, sm) : ensure_smem((const void *)k_fwd_wide<2>, sm);
    if (e != cudaSuccess) return e;
    if (mode == 1)
        k_fwd_wide<1><<<dim3(S, map.np), kFwdThreads, sm, st>>>(job_dev, in.w, in.wmax, nmax, map, part);
    else
        k_fwd_wide<2><<<dim3(S, map.np), kFwdThreads, sm, st>>>(job_dev, in.w, in.wmax, nmax, map, part);
    const int nt = (p + kAsmT - 1) / kAsmT;
    if (K64) k_fwd_assemble<double><<<dim3(nt, nt), 256, 0, st>>>(p, part, S, map, in.wmax, nmax, K64);
    else k_fwd_assemble<float><<<dim3(nt, nt), 256, 0, st>>>(p, part, S, map, in.wmax, nmax, K32);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- full-image LSQR launchers
static inline int ls_grid(int n) { return max(1, min(4 * num_sms(), (n + kThreads - 1) / kThreads)); }
// Grid of the kernels that leave per-CTA maxima.
static inline int ls_max_grid(int n) { return max(1, min(kOpMax, (n + kThreads - 1) / kThreads)); }

// M v from the pixel weights wx that the vector step left.
cudaError_t ls_forward(const JobDev *jd, const JobDev &hj, LsBufs &b, int mode, float *fwd_part, float2 *part,
                       int nparts, cudaStream_t st) {
    const int Q = hj.Q, p = hj.p, pp = p * p;
    cudaError_t e;
    if (mode != 0) {
        const FwdIn in{nullptr, b.wx, b.wmax, ls_max_grid(Q)};
        e = launch_psi_wide(jd, in, fwd_part, Q, p, hj.n_l, hj.n_m, mode, nullptr, reinterpret_cast<float *>(b.Mv), st);
    } else {
        e = launch_psi(jd, b.wx, part, nparts, Q, p, b.Kd, st);
        if (e == cudaSuccess) k_d2c<<<ls_grid(pp), kThreads, 0, st>>>(b.Kd, b.Mv, pp);
    }
    if (e != cudaSuccess) return e;
    if (hj.cost == IMG_COST_PWLS) {
        // W vect(K) = vect(L^-1 K L^-H)
        const dim3 g((p + 15) / 16, (p + 15) / 16);
        k_cgemm<<<g, 256, 0, st>>>(p, b.Mv, 0, hj.Li32, 1, b.T1, nullptr);
        k_cgemm<<<g, 256, 0, st>>>(p, hj.Li32, 0, b.T1, 0, b.Mv, nullptr);
    }
    return cudaGetLastError();
}

// b.y = M^H u.  numax: per-CTA maxima of |u| in the job's opmax (CLS; 0 when
// they are not there).
cudaError_t ls_adjoint(const JobDev *jd, const JobDev &hj, LsBufs &b, int mode, int numax, cudaStream_t st) {
    const int Q = hj.Q, p = hj.p;
    const float2 *U = b.u;
    if (hj.cost == IMG_COST_PWLS) {
        // W^H vect(u) = vect(L^-H u L^-1)
        const dim3 g((p + 15) / 16, (p + 15) / 16);
        const bool fits = (int)(g.x * g.y) <= kOpMax;
        k_cgemm<<<g, 256, 0, st>>>(p, b.u, 0, hj.Li32, 0, b.T1, nullptr);
        k_cgemm<<<g, 256, 0, st>>>(p, hj.Li32, 1, b.T1, 0, b.Uw, fits ? hj.opmax : nullptr);
        U = b.Uw;
        numax = fits ? (int)(g.x * g.y) : 0;
    }
    cudaError_t e = mode != 0 ? launch_psi_adj_wide(jd, U, false, numax, b.y, Q, p, mode, st)
                              : launch_psi_adj(jd, U, b.y, Q, p, st);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// beta, u / beta (n complex); then v, alpha and the vector updates once b.y
// holds M^H u.
static void ls_u_step(const JobDev &hj, LsBufs &b, int n, int first, cudaStream_t st) {
    k_ls_scale_u<<<ls_max_grid(n), kThreads, 0, st>>>(b.u, n, b.sc, first, hj.opmax);
}
static void ls_v_step(const JobDev &hj, LsBufs &b, int first, cudaStream_t st) {
    const int Q = hj.Q;
    k_ls_v<<<kLsWarps, 32, 0, st>>>(b.v, b.y, hj.scale, Q, b.sc, first);
    k_ls_xw<<<ls_max_grid(Q), kThreads, 0, st>>>(b.x, b.w, b.v, Q, b.sc, first, hj.scale, b.wx, b.wmax);
}

cudaError_t ls_begin(const JobDev *jd, const JobDev &hj, LsBufs &b, int mode, cudaStream_t st) {
    const int p = hj.p, pp = p * p;
    k_ls_init_u<<<ls_grid(pp), kThreads, 0, st>>>(hj.R32, p, hj.cost == IMG_COST_PWLS, b.u);
    k_sumsq<<<kLsWarps, 32, 0, st>>>(reinterpret_cast<const float *>(b.u), 2 * pp, b.sc + kLsRedU);
    ls_u_step(hj, b, pp, 1, st);
    cudaError_t e = ls_adjoint(jd, hj, b, mode, ls_max_grid(pp), st);
    if (e != cudaSuccess) return e;
    ls_v_step(hj, b, 1, st);
    return cudaGetLastError();
}

cudaError_t ls_iterate(const JobDev *jd, const JobDev &hj, LsBufs &b, int mode, float *fwd_part, float2 *part,
                       int nparts, cudaStream_t st) {
    const int pp = hj.p * hj.p;
    // u <- M v - alpha u, beta = ||u||, u <- u / beta
    cudaError_t e = ls_forward(jd, hj, b, mode, fwd_part, part, nparts, st);
    if (e != cudaSuccess) return e;
    k_ls_u<<<kLsWarps, 32, 0, st>>>(reinterpret_cast<float *>(b.u), reinterpret_cast<const float *>(b.Mv), 2 * pp, b.sc);
    ls_u_step(hj, b, pp, 0, st);
    // v <- M^H u - beta v, alpha = ||v||, rotation, x and w updates
    e = ls_adjoint(jd, hj, b, mode, ls_max_grid(pp), st);
    if (e != cudaSuccess) return e;
    ls_v_step(hj, b, 0, st);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- K-snapshot full-image LSQR
// y = first ? yk : y + yk (the snapshot sum of M^H u, snapshot order fixed).
__global__ void k_ls_accum(double *y, const double *yk, int Q, int first) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x)
        y[i] = first ? yk[i] : y[i] + yk[i];
}

// Pixel scale of the K-snapshot solver variable: 1/D with
// D = (sum_k h_k)^2 / (K C) for PWLS (eq. D), 1 for CLS.
__global__ void k_snap_scale(SnapPtrs sp, int K, int Q, int pwls, double C, float *scale) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x) {
        double hs = 0.0;
        for (int k = 0; k < K; ++k) hs += (double)sp.h[k][i];
        scale[i] = pwls ? (float)(1.0 / ((hs * hs) / ((double)K * C))) : 1.0f;
    }
}

cudaError_t launch_snap_scale(const SnapPtrs &sp, int K, int Q, int pwls, double C, float *scale, cudaStream_t st) {
    k_snap_scale<<<ls_grid(Q), kThreads, 0, st>>>(sp, K, Q, pwls, C, scale);
    return cudaGetLastError();
}

// Buffers of snapshot k: its block of u and M v, the shared scratch, and the
// per-snapshot adjoint output yk.
static LsBufs snap_bufs(const LsSnap &s, const LsBufs &b, int k) {
    LsBufs bk = b;
    const size_t pp = (size_t)s.hj[0].p * s.hj[0].p;
    bk.u = b.u + (size_t)k * pp;
    bk.Mv = b.Mv + (size_t)k * pp;
    bk.y = s.yk;
    return bk;
}

// y = sum_k M_k^H u_k.
static cudaError_t snap_adjoint(const LsSnap &s, LsBufs &b, cudaStream_t st) {
    const int Q = s.hj[0].Q;
    for (int k = 0; k < s.K; ++k) {
        LsBufs bk = snap_bufs(s, b, k);
        // the maxima of the K blocks of u together are no block's own
        cudaError_t e = ls_adjoint(s.jd[k], s.hj[k], bk, s.mode[k], 0, st);
        if (e != cudaSuccess) return e;
        k_ls_accum<<<ls_grid(Q), kThreads, 0, st>>>(b.y, s.yk, Q, k == 0);
    }
    return cudaGetLastError();
}

// M_k v into block k of b.Mv for every snapshot.
static cudaError_t snap_forward(const LsSnap &s, LsBufs &b, cudaStream_t st) {
    for (int k = 0; k < s.K; ++k) {
        LsBufs bk = snap_bufs(s, b, k);
        cudaError_t e = ls_forward(s.jd[k], s.hj[k], bk, s.mode[k], s.fwd_part[k], s.part[k], s.nparts[k], st);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

cudaError_t ls_snap_begin(const LsSnap &s, LsBufs &b, cudaStream_t st) {
    const int p = s.hj[0].p, pp = p * p, n = s.K * pp;
    const int pwls = s.hj[0].cost == IMG_COST_PWLS;
    for (int k = 0; k < s.K; ++k)
        k_ls_init_u<<<ls_grid(pp), kThreads, 0, st>>>(s.hj[k].R32, p, pwls, b.u + (size_t)k * pp);
    k_sumsq<<<kLsWarps, 32, 0, st>>>(reinterpret_cast<const float *>(b.u), 2 * n, b.sc + kLsRedU);
    ls_u_step(s.hj[0], b, n, 1, st);
    cudaError_t e = snap_adjoint(s, b, st);
    if (e != cudaSuccess) return e;
    ls_v_step(s.hj[0], b, 1, st);
    return cudaGetLastError();
}

cudaError_t ls_snap_iterate(const LsSnap &s, LsBufs &b, cudaStream_t st) {
    const int pp = s.hj[0].p * s.hj[0].p, n = s.K * pp;
    cudaError_t e = snap_forward(s, b, st);
    if (e != cudaSuccess) return e;
    k_ls_u<<<kLsWarps, 32, 0, st>>>(reinterpret_cast<float *>(b.u), reinterpret_cast<const float *>(b.Mv), 2 * n, b.sc);
    ls_u_step(s.hj[0], b, n, 0, st);
    e = snap_adjoint(s, b, st);
    if (e != cudaSuccess) return e;
    ls_v_step(s.hj[0], b, 0, st);
    return cudaGetLastError();
}

cudaError_t ls_finish(const JobDev &hj, LsBufs &b, double *sigma, cudaStream_t st) {
    k_ls_sigma<<<ls_grid(hj.Q), kThreads, 0, st>>>(b.x, hj.scale, sigma, hj.Q);
    return cudaGetLastError();
}

cudaError_t ls_xnorm2(const JobDev &hj, LsBufs &b, double *out, cudaStream_t st) {
    k_sumsq<<<kLsWarps, 32, 0, st>>>(b.x, hj.Q, b.sc + kLsRedV);
    k_sum32<<<1, 32, 0, st>>>(b.sc + kLsRedV, out);
    return cudaGetLastError();
}

template <int MODE>
static cudaError_t launch_psi_adj_wide_t(const JobDev *job_dev, const void *U, bool u64, int nmax, double *out, int Q,
                                         int p, cudaStream_t st) {
    const dim3 eg(wide_nk(p), 2 * wide_kp(p) / kEmbRows);
    const bool have = nmax > 0;
    if (!have) nmax = min(16, (p * p + kThreads - 1) / kThreads);
    if (u64) {
        if (!have) k_emb_max_one<double2><<<nmax, kThreads, 0, st>>>(job_dev, static_cast<const double2 *>(U));
        k_emb_one<MODE, double2><<<eg, kThreads, 0, st>>>(job_dev, static_cast<const double2 *>(U), nmax);
    } else {
        if (!have) k_emb_max_one<float2><<<nmax, kThreads, 0, st>>>(job_dev, static_cast<const float2 *>(U));
        k_emb_one<MODE, float2><<<eg, kThreads, 0, st>>>(job_dev, static_cast<const float2 *>(U), nmax);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t sm = wide_smem_bytes(p);
    e = ensure_smem((const void *)k_psi_adj_wide<MODE>, sm);
    if (e != cudaSuccess) return e;
    const int ntiles = (Q + kTcM - 1) / kTcM + 64;   // >= 2-D tiles of any grid
    k_psi_adj_wide<MODE><<<min(ntiles, num_sms()), kWideThreads, sm, st>>>(job_dev, out);
    return cudaGetLastError();
}

cudaError_t launch_psi_adj_wide(const JobDev *job_dev, const void *U, bool u64, int nmax, double *out, int Q, int p,
                                int mode, cudaStream_t st) {
    if (p < 1 || p > kMaxWideP || (mode != 1 && mode != 2)) return cudaErrorInvalidValue;
    if (mode == 1) return launch_psi_adj_wide_t<1>(job_dev, U, u64, nmax, out, Q, p, st);
    return launch_psi_adj_wide_t<2>(job_dev, U, u64, nmax, out, Q, p, st);
}

// On CUDA cores (tensor cores: launch_psi_adj_wide).
cudaError_t launch_psi_adj(const JobDev *job_dev, const float2 *U, double *out, int Q, int p, cudaStream_t st) {
    const size_t sm = bounds_smem_bytes(p);
    cudaError_t e = ensure_smem((const void *)k_psi_adj, sm);
    if (e != cudaSuccess) return e;
    const int ntiles = (Q + kTile - 1) / kTile;
    k_psi_adj<<<min(ntiles, 2 * num_sms()), kThreads, sm, st>>>(job_dev, U, out);
    return cudaGetLastError();
}

cudaError_t launch_z2c(const double2 *src, float2 *dst, int n, cudaStream_t st) {
    k_z2c<<<min(1024, (n + 255) / 256 + 1), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_c2z(const float2 *src, double2 *dst, int n, cudaStream_t st) {
    k_c2z<<<min(1024, (n + 255) / 256 + 1), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_d2f(const double *src, float *dst, int n, cudaStream_t st) {
    k_d2f<<<min(1024, (n + 255) / 256 + 1), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

// Dirty images over K snapshots from each snapshot's MF image d_k and MVDR
// denominator h_k = a_{i,k}^H R_k^-1 a_{i,k} (Sec. III-C, Sec. III-D,
// eq. ASSC0): MF (1/K) sum d_k, MVDR C K / sum h_k, ASSC C / max h_k.
// FP64, snapshot order fixed.
__global__ void k_snapshot_image(SnapPtrs sp, int K, int Q, int kind, double C, double *out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Q; i += gridDim.x * blockDim.x) {
        double acc = 0.0;
        if (kind == IMG_SNAP_MF) {
            for (int k = 0; k < K; ++k) acc += (double)sp.d[k][i];
            out[i] = acc / (double)K;
        } else if (kind == IMG_SNAP_MVDR) {
            for (int k = 0; k < K; ++k) acc += (double)sp.h[k][i];
            out[i] = (C * (double)K) / acc;
        } else {
            for (int k = 0; k < K; ++k) acc = fmax(acc, (double)sp.h[k][i]);
            out[i] = C / acc;
        }
    }
}

cudaError_t launch_snapshot_image(const SnapPtrs &sp, int K, int Q, int kind, double C, double *out,
                                  cudaStream_t st) {
    k_snapshot_image<<<min(1024, (Q + 255) / 256), 256, 0, st>>>(sp, K, Q, kind, C, out);
    return cudaGetLastError();
}

cudaError_t launch_to_double(const float *src, double *dst, int n, cudaStream_t st) {
    k_to_double<<<min(1024, (n + 255) / 256 + 1), 256, 0, st>>>(src, dst, n);
    return cudaGetLastError();
}

}  // namespace img
