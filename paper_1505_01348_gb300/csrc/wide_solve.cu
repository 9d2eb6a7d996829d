// Wide active-set solver (Table I with LSQR subproblems, Sec. IV and V) for
// 64 < p <= 384 on tensor cores, as one CUDA graph per job.
//
// The Table I loop is a graph WHILE node whose body is one pass (or two:
// freeing the pixel chosen by the last gradient, then the next subproblem).
// The subproblem's LSQR is a SWITCH node: nothing (no free pixel), an
// initialisation and a WHILE node of iterations, or one kernel whose thread-block
// cluster iterates until the stopping tests hold; the feasible / infeasible
// branch is an IF/ELSE node.  Kernels set the conditions from device memory, so
// a whole solve runs without a host round trip.  Every kernel has a fixed grid
// and reads the sizes of the moment (|F|, |U|, support) from the control block.
//
// Operators (tc_items.cuh): the adjoint over the free set or over every pixel
// runs in (tile, unit) work items from a B image of U; the forward over a
// list forms Gram blocks from a list image.  Both split products FP16x3 or
// BF16x3 with FP32 accumulation.  Scalars of LSQR, feasibility, the step and
// the multiplier tests are FP64 or FP32 exactly as in the one-CTA solver.
//
// PWLS gradient: with d_i = R^-1 a_i cached per support pixel, the whitened
// residual is U_g = R^-1 - sum_S s_i x_i d_i d_i^H (= L^-H (I - sum s x c c^H)
// L^-1 with c_i = L^-1 a_i), so no p^3 sandwich runs per gradient.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "cta_ops.cuh"
#include "tc_items.cuh"
#include "cluster_fit.cuh"

namespace img {

constexpr int kWsThreads = 256;
// CTAs that the list operators' work is split for: the gradient's forward
// runs on that many, and the K groups of the free-list adjoint and the
// capacity of the forward's partial blocks - parts of the sums' order - follow
// from it whatever number of CTAs runs them.
constexpr int kListGrid = 32;
constexpr int kWsSums = 2048;           // per-CTA partial sums of the reductions
// 64-pixel stages per forward task (at least).  Fewer, longer tasks write
// fewer partial blocks for the reduction to read back (16 solves of 256x256,
// p = 288 in flight: 4 -> 0.539, 8 -> 0.551, 16 -> 0.561 images/s), but the
// split also fixes the order of the forward's partial sums, and with 4 the
// complete 256x256, p = 288 solve takes the FP64 oracle's decisions one for
// one at the same LSQR tolerance (with 16 a tie at decision 2013 of 2797
// falls the other way).
constexpr int kFwdPerTask = 4;

// Scalars of the LSQR recurrence: in the control block, or in CTA 0's shared
// memory when a cluster runs the whole subproblem.
struct VxState {
    double alpha, beta, us, bnorm, rhobar, phibar, anorm2, rho, c, sn, phi, xnorm2;
    float fus, fb, ia, t1, t2;
};

// Device control block of one wide solve.
struct WsCtl {
    int f, nu, ns;              // |F|, |U|, |F u U| of the current subproblem
    int pending;                // pixel the last gradient chose to free, or -1
    int outer;                  // Table I passes so far
    int stop;                   // the loop ends after this pass
    int converged, status, feasible, nev, timeouts;
    int it, maxit, lsqr_total;  // LSQR iterations of this subproblem / cap / sum
    int nsplit;                 // forward split of the current list
    int adj_rows;               // unit x K-group partial rows of the free-list adjoint
    float sXF, sXS;             // power-of-two scales of the F and support list images
    float sW;                   // weight scale used by the last forward
    float sB;                   // scale of the current B image
    unsigned mx_t, mx_w;        // max |entry| bits of the matrix being imaged / the weights
    unsigned long long key;     // argmin key of the multiplier test
    VxState vx;
    double fa;
    double lam_min, op_flops;
    unsigned long long t_begin;
    unsigned cond[4];           // last value of each loop / branch condition (host-driven mode)
    int cache_slot, cache_pixel; // support slot whose vectors k_ws_cache computes (-1: none)
    int nsums;                  // CTA shares of ||t||^2 left in sums by k_ws_fred
    int adj_sq;                 // full-image adjoint as sums of squares (MVDR denominators)
    unsigned long long launches;  // kernels executed in this solve
    double sums[kWsSums];
};

enum { kCondOuter = 0, kCondLsqrForm = 1, kCondLsqr = 2, kCondFeas = 3 };
// Values of kCondLsqrForm: a pass without free pixels, LSQR as kernels, as one
// cluster kernel.
enum : unsigned { kLsqrNone = 0, kLsqrKernels = 1, kLsqrCluster = 2 };

// Set a graph condition (h != 0 inside the solve graph) and mirror it in the
// control block for the host-driven mode.
__device__ __forceinline__ void ws_cond(WsCtl *ctl, int which, cudaGraphConditionalHandle h, unsigned v) {
    ctl->cond[which] = v;
    if (h) cudaGraphSetConditional(h, v);
}

// Device buffers of the wide solver (device pointers, passed by value).
struct WsBufs {
    WsCtl *ctl;
    float2 *dvec;               // cap x p: d_i = R^-1 a_i (PWLS); cvec for LS
    float *dmax;                // cap
    int *iota;                  // cap: 0, 1, 2, ...
    float *wl;                  // cap: weights of the current forward list
    float *padj;                // max(Q, cap) x (nu nk): unit (x K group) partial dots, row-contiguous
    float *pfwd;                // forward partial blocks (tasks x 128 x 256)
    unsigned char *ximgF, *ximgS, *ximgW, *bimg;   // list images: F, U or support, weighted; B image
    int npairs, pm[kItemsFwdMaxPairs], pnb[kItemsFwdMaxPairs];
    int max_tasks;              // capacity of pfwd in blocks
    int list_grid;              // CTAs that the free-list adjoint's K groups are chosen for
    int cluster_f;              // most free pixels of the cluster form of LSQR
    int fwd_per;                // 64-pixel stages per forward task (at least)
    int nrows_adj;              // rows of padj (max(Q, cap))
    int ld_adj;                 // partial dots per row of padj (nu nk)
};

enum { kListF = 0, kListU = 1, kListS = 2 };
enum { kRedB = 0, kRedT = 1, kRedG = 2 };

__device__ __forceinline__ float pow2_scale(float mx) { return mx > 0.f ? exp2f(-ceilf(log2f(mx))) : 1.f; }
__device__ __forceinline__ unsigned long long key_of(float lam, int i) {
    unsigned b = __float_as_uint(lam);
    b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);      // order-preserving
    return ((unsigned long long)b << 32) | (unsigned)i;
}
__device__ __forceinline__ float lam_of(unsigned long long key) {
    unsigned b = (unsigned)(key >> 32);
    b = (b & 0x80000000u) ? (b & 0x7fffffffu) : ~b;
    return __uint_as_float(b);
}
__device__ __forceinline__ double ws_flops_fwd(int p, int n) { return 4.0 * p * (double)p * n; }
__device__ __forceinline__ double ws_flops_adj(int p, int n) { return 8.0 * p * (double)p * n; }

// Count this kernel in the solve's launch total (block 0, thread 0).
__device__ __forceinline__ void ws_count(WsCtl *ctl) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&ctl->launches, 1ull);
}

__device__ void ws_log(const JobDev &J, WsCtl *ctl, int kind, int pixel, float val) {
    if (ctl->nev < J.ev_cap) {
        J.ev[ctl->nev] = (kind << 24) | pixel;
        J.evv[ctl->nev] = val;
    }
    ctl->nev++;
}

// ---------------------------------------------------------------- start / end
__global__ void k_ws_start(const JobDev *Jp, WsBufs B, cudaGraphConditionalHandle h_outer) {
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    for (int i = threadIdx.x; i < J.Q; i += blockDim.x) {
        J.x[i] = 0.0;
        J.set[i] = IMG_SET_L;
        J.slot[i] = -1;
        J.grad[i] = 0.f;
    }
    for (int j = threadIdx.x; j < J.cap; j += blockDim.x) B.iota[j] = j;
    if (threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        ctl->t_begin = t;
        ctl->launches = 1;
        ctl->f = ctl->nu = ctl->ns = 0;
        ctl->pending = -1;
        ctl->outer = 0;
        ctl->converged = 0;
        ctl->status = IMG_OK;
        ctl->feasible = 0;
        ctl->nev = 0;
        ctl->timeouts = 0;
        ctl->it = ctl->maxit = ctl->lsqr_total = 0;
        ctl->nsplit = 1;
        ctl->mx_t = ctl->mx_w = 0;
        ctl->lam_min = 0.0;
        ctl->op_flops = 0.0;
        ctl->stop = 0;
        if (J.flags[0] != 0 || J.flags[1] != 1) {
            ctl->status = J.flags[0] != 0 ? J.flags[0] : IMG_EINVAL;
            ctl->stop = 1;
        }
        ws_cond(ctl, kCondOuter, h_outer, ctl->stop ? 0u : 1u);
    }
}

__global__ void k_ws_end(const JobDev *Jp, WsBufs B, cudaGraphConditionalHandle h_outer) {
    ws_count(B.ctl);
    WsCtl *ctl = B.ctl;
    if (threadIdx.x == 0) ws_cond(ctl, kCondOuter, h_outer, ctl->stop ? 0u : 1u);
}

__global__ void k_ws_finish(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    __shared__ double sbuf[kWsThreads / 32];
    int nf = 0, nu = 0;
    for (int i = threadIdx.x; i < J.Q; i += blockDim.x) {
        J.sigma[i] = (double)J.scale[i] * J.x[i];
        nf += J.set[i] == IMG_SET_F;
        nu += J.set[i] == IMG_SET_U;
    }
    const double tf = block_sum((double)nf, sbuf);
    const double tu = block_sum((double)nu, sbuf);
    if (threadIdx.x == 0) {
        DevInfo info{};
        int st = ctl->status;
        if (st == IMG_OK && ctl->timeouts) st = IMG_ETIMEOUT;
        if (st == IMG_OK && !ctl->converged) st = IMG_ENOTCONV;
        info.status = st;
        info.outer = ctl->outer;
        info.lsqr_iters = ctl->lsqr_total;
        info.n_free = (int)tf;
        info.n_upper = (int)tu;
        info.converged = ctl->converged;
        info.lambda_min = ctl->lam_min;
        info.op_flops = ctl->op_flops;
        info.t_begin_ns = ctl->t_begin;
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        info.t_end_ns = t;
        info.cyc_total = (double)(t - ctl->t_begin);
        info.cyc_aux[0] = (double)ctl->launches;      // kernels this solve executed
        *J.ev_count = ctl->nev;
        *J.info = info;
    }
}

// ---------------------------------------------------------------- support cache
// c_i = T a_i (T = L^-1 for PWLS, I for LS) into cvec row `slot`, and for
// PWLS d_i = R^-1 a_i into dvec; their largest component magnitudes by
// atomicMax on the float bits (cmax / dmax of the slot start at zero).
// CTA b computes rows k = 32 b + lane; warp w sums the terms l = w, w + 8, ...
constexpr int kCacheRows = 32;
__global__ void __launch_bounds__(kWsThreads) k_ws_cache(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    const WsCtl *ctl = B.ctl;
    const int slot = ctl->cache_slot;
    if (ctl->stop || slot < 0) return;
    const int i = ctl->cache_pixel;
    const int p = J.p;
    const int im = i / J.n_l, il = i - im * J.n_l;
    const bool pwls = J.cost == IMG_COST_PWLS;
    __shared__ float2 sa[kItemsMaxP];
    __shared__ float2 part[2][8][kCacheRows];
    for (int k = threadIdx.x; k < p; k += blockDim.x) sa[k] = steer(J, il, im, k);
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int k = blockIdx.x * kCacheRows + lane;
    float2 sc = make_float2(0.f, 0.f), sd = make_float2(0.f, 0.f);
    if (k < p) {
        if (!pwls) {
            if (w == 0) sc = sa[k];
        } else {
            const float2 *__restrict__ Li = J.Li32 + k;
            const float2 *__restrict__ Ri = J.Ri32 + k;
#pragma unroll 4
            for (int l = w; l <= k; l += 8) cfma(sc, Li[(size_t)l * p], sa[l]);
#pragma unroll 4
            for (int l = w; l < p; l += 8) cfma(sd, Ri[(size_t)l * p], sa[l]);
        }
    }
    part[0][w][lane] = sc;
    part[1][w][lane] = sd;
    __syncthreads();
    if (w == 0) {
        float2 c = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
        for (int q = 0; q < 8; ++q) {
            c.x += part[0][q][lane].x;
            c.y += part[0][q][lane].y;
            d.x += part[1][q][lane].x;
            d.y += part[1][q][lane].y;
        }
        float mc = 0.f, md = 0.f;
        if (k < p) {
            J.cvec[(size_t)slot * p + k] = c;
            mc = fmaxf(fabsf(c.x), fabsf(c.y));
            if (pwls) {
                B.dvec[(size_t)slot * p + k] = d;
                md = fmaxf(fabsf(d.x), fabsf(d.y));
            }
        }
        for (int o = 16; o; o >>= 1) {
            mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, o));
            md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
        }
        if (lane == 0) {
            atomicMax(reinterpret_cast<unsigned *>(J.cmax + slot), __float_as_uint(mc));
            if (pwls) atomicMax(reinterpret_cast<unsigned *>(B.dmax + slot), __float_as_uint(md));
        }
    }
}

// Remove support slot of pixel i (swap with the last entry).
__device__ void ws_remove(const JobDev &J, const WsBufs &B, int i, int &ns) {
    const int p = J.p;
    const int sl = J.slot[i];
    const int last = ns - 1;
    const bool pwls = J.cost == IMG_COST_PWLS;
    if (sl != last) {
        const int moved = J.supp[last];
        for (int k = threadIdx.x; k < p; k += blockDim.x) {
            J.cvec[(size_t)sl * p + k] = J.cvec[(size_t)last * p + k];
            if (pwls) B.dvec[(size_t)sl * p + k] = B.dvec[(size_t)last * p + k];
        }
        if (threadIdx.x == 0) {
            J.supp[sl] = moved;
            J.slot[moved] = sl;
            J.cmax[sl] = J.cmax[last];
            if (pwls) B.dmax[sl] = B.dmax[last];
        }
    }
    if (threadIdx.x == 0) J.slot[i] = -1;
    ns = last;
    __syncthreads();
}

// Largest value of a per-slot maximum array over a position list (CTA).
__device__ float ws_list_max(const float *mx, const int *pos, int n) {
    __shared__ float sred[kWsThreads / 32];
    float m = 0.f;
    for (int j = threadIdx.x; j < n; j += blockDim.x) m = fmaxf(m, mx[pos ? pos[j] : j]);
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = m;
    __syncthreads();
    m = 0.f;
    for (int w = 0; w < kWsThreads / 32; ++w) m = fmaxf(m, sred[w]);
    __syncthreads();
    return m;
}

// K groups of the free-list adjoint: the largest divisor of nk that keeps
// the work items within the grid.
__device__ int ws_nkg(int items, int nk, int grid) {
    int best = 1;
    for (int d = 1; d <= nk; ++d)
        if (nk % d == 0 && items * d <= grid) best = d;
    return best;
}

__device__ int ws_nsplit(int n, int npairs, int max_tasks, int per) {
    const int stages = (n + kFwdPix - 1) / kFwdPix;
    int ns = (stages + per - 1) / per;             // about `per` stages per task
    const int cap = max(1, max_tasks / max(npairs, 1));
    ns = min(ns, cap);
    return max(ns, 1);
}

// ---------------------------------------------------------------- pass
// Table I, first part of a loop iteration: free the pending pixel (a pass of
// its own): give it a support slot when it has none (its vectors are then
// computed by k_ws_cache), move it to F and log it.
__global__ void k_ws_free(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (threadIdx.x != 0) return;
    ctl->cache_slot = -1;
    if (ctl->stop) return;
    const int max_outer = J.max_outer > 0 ? J.max_outer : 10 * J.Q + 100;
    const int i = ctl->pending;
    if (i < 0) return;
    if (ctl->outer >= max_outer) {
        ctl->stop = 1;
        return;
    }
    int ns = ctl->ns;
    if (J.slot[i] < 0) {
        if (ns >= J.cap) {
            ctl->status = IMG_ENOMEM;
            ctl->stop = 1;
            return;
        }
        J.supp[ns] = i;
        J.slot[i] = ns;
        J.cmax[ns] = 0.f;
        if (J.cost == IMG_COST_PWLS) B.dmax[ns] = 0.f;
        ctl->cache_slot = ns;
        ctl->cache_pixel = i;
        ctl->ns = ns + 1;
    }
    ctl->outer++;
    J.set[i] = IMG_SET_F;
    ws_log(J, ctl, 0, i, (float)ctl->lam_min);
    ctl->pending = -1;
}

// Then set up the subproblem of the next pass: compact F and U, the U
// weights -s_i x_i (eq. bsubproblemLS / MVDR), the F scales, the list scales
// and the LSQR iteration cap; h_form := the form of LSQR (none when F is empty).
__global__ void k_ws_pass(const JobDev *Jp, WsBufs B, cudaGraphConditionalHandle h_form) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    __shared__ int cbuf[kWsThreads / 32];
    __shared__ int s_skip;
    const int max_outer = J.max_outer > 0 ? J.max_outer : 10 * J.Q + 100;
    const int ns = ctl->ns;
    if (threadIdx.x == 0) {
        if (!ctl->stop && ctl->outer >= max_outer) ctl->stop = 1;
        s_skip = ctl->stop;
    }
    __syncthreads();
    if (s_skip) {
        if (threadIdx.x == 0) {
            ctl->f = 0;
            ws_cond(ctl, kCondLsqrForm, h_form, kLsqrNone);
        }
        return;
    }
    const int f = block_compact(ns, [&](int pos) { return J.set[J.supp[pos]] == IMG_SET_F; }, J.fpos, cbuf);
    const int nu = block_compact(ns, [&](int pos) { return J.set[J.supp[pos]] == IMG_SET_U; }, J.fpos + f, cbuf);
    float wm = 0.f;
    for (int j = threadIdx.x; j < nu; j += blockDim.x) {
        const int i = J.supp[J.fpos[f + j]];
        const float wv = -J.scale[i] * (float)J.x[i];
        B.wl[j] = wv;
        wm = fmaxf(wm, fabsf(wv));
    }
    for (int j = threadIdx.x; j < f; j += blockDim.x) J.sF[j] = J.scale[J.supp[J.fpos[j]]];
    const float mF = ws_list_max(J.cmax, J.fpos, f);
    const float mU = ws_list_max(J.cmax, J.fpos + f, nu);
    for (int o = 16; o; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
    __shared__ float swm[kWsThreads / 32];
    if ((threadIdx.x & 31) == 0) swm[threadIdx.x >> 5] = wm;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < kWsThreads / 32; ++w) wm = fmaxf(wm, swm[w]);
        ctl->outer++;
        ctl->f = f;
        ctl->nu = nu;
        ctl->sXF = pow2_scale(mF) * kLift;
        ctl->sXS = pow2_scale(mU) * kLift;
        ctl->mx_w = __float_as_uint(wm);
        ctl->nsplit = ws_nsplit(nu, B.npairs, B.max_tasks, B.fwd_per);
        ctl->maxit = J.lsqr_maxit > 0 ? J.lsqr_maxit : 4 * f + 20;
        ctl->it = 0;
        ctl->op_flops += ws_flops_fwd(J.p, nu);
        ws_cond(ctl, kCondLsqrForm, h_form, f == 0 ? kLsqrNone : f <= B.cluster_f ? kLsqrCluster : kLsqrKernels);
    }
}

// ---------------------------------------------------------------- images
// List image of the F list (cvec, scale sXF), of the U list (cvec, scale
// sXS) or of the support (dvec / cvec, scale sXS); every row of the tiles
// and the padding chunks are written.  U and S share one image buffer.
// weighted: the image of the rows times their weights wl (the second
// operand of a forward) into ximgW, scaled by sX sW with sW the power of two
// of max |wl| (stored for the reduction).
// CTA `rank` of `ctas` does its share.
template <bool BF16, int NC>
__device__ void ws_listimg(const JobDev &J, const WsBufs &B, const UnitGeom &g, int which, int weighted, int rank,
                           int ctas) {
    WsCtl *ctl = B.ctl;
    const bool S = which == kListS, Ul = which == kListU;
    const int n = S ? ctl->ns : (Ul ? ctl->nu : ctl->f);
    const int *pos = S ? B.iota : (Ul ? J.fpos + ctl->f : J.fpos);
    const float2 *vec = (S && J.cost == IMG_COST_PWLS) ? B.dvec : J.cvec;
    float sX = (S || Ul) ? ctl->sXS : ctl->sXF;
    unsigned char *img = weighted ? B.ximgW : ((S || Ul) ? B.ximgS : B.ximgF);
    if (weighted) {
        const float sW = pow2_scale(__uint_as_float(ctl->mx_w));
        if (rank == 0 && threadIdx.x == 0) ctl->sW = sW;
        sX *= sW;
    }
    const float *wgt = weighted ? B.wl : nullptr;
    list_image<BF16, NC>(vec, pos, wgt, n, J.p, g, sX, img, rank * blockDim.x + threadIdx.x, ctas * blockDim.x);
}
template <bool BF16>
__global__ void k_ws_listimg(const JobDev *Jp, WsBufs B, int which, int weighted) {
    ws_count(B.ctl);
    if (B.ctl->stop) return;
    ws_listimg<BF16, kImgChunksGrid>(*Jp, B, unit_geom(Jp->p), which, weighted, blockIdx.x, gridDim.x);
}

// B unit image of the matrix U (W0 for LSQR, W1 for the gradient) with the
// power-of-two scale of ctl->mx_t.
template <bool BF16, int NC>
__device__ void ws_emb(const JobDev &J, const WsBufs &B, const UnitGeom &g, const float2 *U, int rank, int ctas) {
    WsCtl *ctl = B.ctl;
    const float sc = pow2_scale(__uint_as_float(ctl->mx_t)) * kLift;
    if (rank == 0 && threadIdx.x == 0) ctl->sB = sc;
    unit_image<BF16, NC>(U, J.p, g, sc, B.bimg, rank * blockDim.x + threadIdx.x, ctas * blockDim.x);
}
template <bool BF16>
__global__ void k_ws_emb(const JobDev *Jp, WsBufs B, int grad, const float2 *Um) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    if (B.ctl->stop) return;
    ws_emb<BF16, kImgChunksGrid>(J, B, unit_geom(J.p), Um ? Um : (grad ? J.W1 : J.W0), blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------- operators
// Forward over the current list: F (weights wl = s_j v_j, cvec), U (weights
// -s_i x_i, cvec) or the support S (weights -s_i x_i, dvec / cvec): Gram
// blocks from the list's image and its weighted image.  The list's split over
// tasks (nsplit) fixes the order of the sums; how many of a block's 64-column
// chunks one task takes does not.  SLICE (the cluster's 8 CTAs): blocks are cut
// into slices while there are fewer blocks than CTAs.  As a kernel, whose CTAs
// share the GPU with other solves, whole blocks: each slice copies both A
// chunks again (16 images of 256x256, p = 288, first 1600 passes 5.05 instead of
// 4.97 s with slices, 4 images 2.42 instead of 2.37 s, one image the same).
// dyn, bars, tmem: as items_forward.
template <bool BF16, bool SLICE>
__device__ int ws_forward(const WsBufs &B, const UnitGeom &g, int which, int rank, int ctas, unsigned char *dyn,
                          uint64_t *bars, uint32_t tmem) {
    const WsCtl *ctl = B.ctl;
    const int n = which == kListF ? ctl->f : (which == kListU ? ctl->nu : ctl->ns);
    const unsigned char *XA = which == kListF ? B.ximgF : B.ximgS;
    if (n <= 0) return 0;
    const int nsplit = ctl->nsplit;
    const int blocks = B.npairs * nsplit;
    const int slices = !SLICE || blocks >= 2 * ctas ? 1 : (2 * blocks >= ctas ? 2 : 4), nq = 4 / slices;
    int to = 0;
    for (int task = rank; task < blocks * slices; task += ctas) {
        const int blk = task / slices, q0 = (task - blk * slices) * nq;
        const int pr = blk / nsplit, s = blk - pr * nsplit;
        if (64 * q0 >= items_fwd_n(g, B.pnb[pr])) continue;
        to += items_forward<BF16>(g, dyn, bars, tmem, XA, B.ximgW, n, B.pm[pr], B.pnb[pr], q0, nq, s, nsplit,
                                  B.pfwd + (size_t)blk * kTcM * 256);
        __syncthreads();
    }
    return to;
}

// A broken pipeline ends the solve: every later kernel sees stop.
__device__ __forceinline__ void ws_timeouts(WsCtl *ctl, int to) {
    if (to && threadIdx.x == 0) {
        atomicAdd(&ctl->timeouts, to);
        ctl->stop = 1;
    }
}

template <bool BF16>
__global__ void __launch_bounds__(kItemsFwdThreads, 1) k_ws_fwd(const JobDev *Jp, WsBufs B, int which) {
    ws_count(B.ctl);
    if (B.ctl->stop) return;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[6];
    __shared__ uint32_t tslot;
    // one tensor-memory allocation for all of this CTA's tasks
    if (threadIdx.x < 32) tmem_alloc(&tslot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    const int to = ws_forward<BF16, false>(B, unit_geom(Jp->p), which, blockIdx.x, gridDim.x, dyn, bars, tmem);
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(tmem, 256);
    ws_timeouts(B.ctl, to);
}

// Sum the forward partial blocks in a fixed order into K and form
//   kRedB: W0 = base + K             (subproblem data, base R_hat or I)
//   kRedT: W0 = K - fa W0            (LSQR: t <- M v - alpha u, u = t us)
//   kRedG: W1 = base + K             (gradient residual, base R_hat or R_hat^-1)
// with K = sum w_j v_j v_j^H (weights carry the sign); max |entry| into
// mx_t; for kRedB / kRedT the norm beta = ||W0|| (FP64, fixed order).
// Re K(a,b) = G(a,b) + G(Kp+a,Kp+b), Im K(a,b) = G(b,Kp+a) - G(a,Kp+b) with G
// read in its upper triangle.  One CTA per 32 x 32 tile of (a, b): the four
// source tiles are read row by row (coalesced) into shared memory, those
// stored below the diagonal transposed on the way.
constexpr int kRedTile = 32;

// address of the stored Gram entry (r, c), r <= c, in the first partial of
// its block (blocks are column-major: entry (r, c) of block (m, nb) at
// (c - 256 nb) 128 + r - 128 m); partial q follows at q 128 256
__device__ __forceinline__ const float *fred_at(const WsBufs &B, const int *pidx, int nsplit, int r, int c) {
    const int m = r >> 7, nb = c >> 8;
    return B.pfwd + (size_t)pidx[m * 4 + nb] * nsplit * kTcM * 256 + (size_t)(c - 256 * nb) * kTcM + (r - 128 * m);
}

__device__ void ws_fred(const JobDev &J, const WsBufs &B, const UnitGeom &g, int mode, int rank, int ctas) {
    WsCtl *ctl = B.ctl;
    const int p = J.p;
    const int Kp = g.Kp;
    const bool pwls = J.cost == IMG_COST_PWLS;
    const int n = mode == kRedT ? ctl->f : (mode == kRedB ? ctl->nu : ctl->ns);
    const int nsplit = ctl->nsplit;
    const float sX = mode == kRedT ? ctl->sXF : ctl->sXS;
    const float inv = n > 0 ? 1.f / (sX * sX * ctl->sW) : 0.f;
    const float fa = (float)ctl->fa;
    float2 *dst = mode == kRedG ? J.W1 : J.W0;
    if (rank == 0 && threadIdx.x == 0) ctl->mx_w = 0u;     // the weights are consumed
    __shared__ int pidx[6 * 4];
    __shared__ double sbuf[kWsThreads / 32];
    __shared__ float T[4][kRedTile][kRedTile + 1];   // G(a,b), G(Kp+a,Kp+b), G(a,Kp+b), G(b,Kp+a), as [a][b]
    if (threadIdx.x < 24) pidx[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x < B.npairs) pidx[B.pm[threadIdx.x] * 4 + B.pnb[threadIdx.x]] = threadIdx.x;
    __syncthreads();
    const int nt = (p + kRedTile - 1) / kRedTile;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;      // 32 x 8
    float mx = 0.f;
    for (int tile = rank; tile < nt * nt; tile += ctas) {
        float ss = 0.f;
        const int a0 = (tile % nt) * kRedTile, b0 = (tile / nt) * kRedTile;
        // what the sums are added to, loaded with the partials (after the
        // sums, each of the four rows' load waited for the store before it)
        float2 old[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int a = a0 + tx, b = b0 + ty + 8 * q, e = b * p + a;
            old[q] = make_float2(0.f, 0.f);
            if (a >= p || b >= p) continue;
            if (mode == kRedT) old[q] = dst[e];
            else if (!pwls) old[q] = J.R32[e];
            else if (mode == kRedG) old[q] = J.Ri32[e];
            else if (a == b) old[q] = make_float2(1.f, 0.f);
        }
        if (n > 0) {
            // the stored blocks are column-major: lanes run along the stored
            // row index (coalesced), i along the column.  Each thread gathers
            // the addresses of all its entries first, then sums the partials
            // with every load of a partial in flight at once.
            const float *src[4][6];
            float acc[4][6];
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                const int i = ty + 8 * ii;
                const int a = a0 + tx, b = b0 + i;           // element (a, b) = tile [tx][i]
                const int bt = b0 + tx, at = a0 + i;         // element (at, bt) = tile [i][tx]
                const bool up = (a0 < b0 || (a0 == b0 && a <= b)) && a < p && b < p;
                const bool lo = (a0 > b0 || (a0 == b0 && bt <= at)) && at < p && bt < p;
                src[ii][0] = up ? fred_at(B, pidx, nsplit, a, b) : nullptr;              // G(a, b)
                src[ii][1] = up ? fred_at(B, pidx, nsplit, Kp + a, Kp + b) : nullptr;    // G(Kp+a, Kp+b)
                src[ii][2] = lo ? fred_at(B, pidx, nsplit, bt, at) : nullptr;            // G(at, bt)
                src[ii][3] = lo ? fred_at(B, pidx, nsplit, Kp + bt, Kp + at) : nullptr;
                src[ii][4] = (a < p && b < p) ? fred_at(B, pidx, nsplit, a, Kp + b) : nullptr;     // G(a, Kp+b)
                src[ii][5] = (at < p && bt < p) ? fred_at(B, pidx, nsplit, bt, Kp + at) : nullptr; // G(b, Kp+a)
#pragma unroll
                for (int e = 0; e < 6; ++e) acc[ii][e] = 0.f;
            }
            for (int q = 0; q < nsplit; ++q) {
                const size_t off = (size_t)q * kTcM * 256;
                float v[4][6];
#pragma unroll
                for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                    for (int e = 0; e < 6; ++e) v[ii][e] = src[ii][e] ? __ldcg(src[ii][e] + off) : 0.f;
#pragma unroll
                for (int ii = 0; ii < 4; ++ii)
#pragma unroll
                    for (int e = 0; e < 6; ++e) acc[ii][e] += v[ii][e];
            }
#pragma unroll
            for (int ii = 0; ii < 4; ++ii) {
                const int i = ty + 8 * ii;
                if (src[ii][0]) {
                    T[0][tx][i] = acc[ii][0];
                    T[1][tx][i] = acc[ii][1];
                }
                if (src[ii][2]) {
                    T[0][i][tx] = acc[ii][2];
                    T[1][i][tx] = acc[ii][3];
                }
                if (src[ii][4]) T[2][tx][i] = acc[ii][4];
                if (src[ii][5]) T[3][i][tx] = acc[ii][5];
            }
        }
        __syncthreads();
        // outputs K(a, b) at dst[b p + a]: lanes along a (coalesced)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = ty + 8 * q, a = a0 + tx, b = b0 + j;
            if (a < p && b < p) {
                float2 k = make_float2(0.f, 0.f);
                if (n > 0) k = make_float2((T[0][tx][j] + T[1][tx][j]) * inv, (T[3][tx][j] - T[2][tx][j]) * inv);
                const float2 o = old[q];
                const float2 out = mode == kRedT ? make_float2(__fmaf_rn(-fa, o.x, k.x), __fmaf_rn(-fa, o.y, k.y))
                                                 : make_float2(o.x + k.x, o.y + k.y);
                dst[b * p + a] = out;
                mx = fmaxf(mx, fmaxf(fabsf(out.x), fabsf(out.y)));
                ss = fmaf(out.x, out.x, fmaf(out.y, out.y, ss));
            }
        }
        // this tile's share of ||W0||^2 (FP64); the vector step adds the
        // shares in tile order
        const double cs = mode == kRedG ? 0.0 : block_sum_w0((double)ss, sbuf);
        if (mode != kRedG && threadIdx.x == 0) ctl->sums[tile] = cs;
        __syncthreads();
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&ctl->mx_t, __float_as_uint(mx));
    if (mode != kRedG && rank == 0 && threadIdx.x == 0) ctl->nsums = nt * nt;
}
// Two CTAs per SM (128 registers, 248 bytes spilled): with the 166 it would
// take, few images are faster (256x256, p = 288: first 200 passes of one 84
// instead of 87 ms, first 1600 of four 2.33 instead of 2.37 s), but a CTA keeps
// the other images' off its SM, and 16 in flight take 5.42 s instead of 4.97.
__global__ void __launch_bounds__(kWsThreads, 2) k_ws_fred(const JobDev *Jp, WsBufs B, int mode) {
    ws_count(B.ctl);
    if (B.ctl->stop) return;
    ws_fred(*Jp, B, unit_geom(Jp->p), mode, blockIdx.x, gridDim.x);
}

// Adjoint over every pixel (gradient, bounds): unit partial dots into
// padj[row * ld_adj + u].
template <bool BF16>
__global__ void __launch_bounds__(kWideThreads, 1) k_ws_adj(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (ctl->stop) return;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[kWideBars];
    __shared__ uint32_t tslot;
    if (threadIdx.x < 32) tmem_alloc(&tslot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    float *out = B.padj;
    const int ld = B.ld_adj;
    const int to = items_adjoint<BF16, false>(
        J, unit_geom(J.p), dyn, bars, tmem, B.bimg, nullptr, nullptr, nullptr, J.Q, tc_num_tiles(J.n_l, J.n_m), 1,
        blockIdx.x, gridDim.x, ctl->adj_sq, [&](int u, int t, int r, float v) {
            const int i = tc_tile_pixel(t, r, J.n_l, J.n_m);
            if (i >= 0) out[(size_t)i * ld + u] = v;
        }, [](int) {});
    if (threadIdx.x < 32) tmem_dealloc(tmem, 512);
    ws_timeouts(ctl, to);
}

// Adjoint over the free list: (unit, K group) partial dots into padj.  The
// number of K groups - part of the order of the sums - is that of a grid of
// `list_grid` CTAs.  idle(warp): as items_adjoint.
template <bool BF16, class Idle>
__device__ int ws_adj_list(const JobDev &J, const WsBufs &B, const UnitGeom &g, int rank, int ctas,
                           unsigned char *dyn, uint64_t *bars, uint32_t tmem, Idle idle) {
    WsCtl *ctl = B.ctl;
    const int n = ctl->f;
    const int ntiles = (n + kTcM - 1) / kTcM;
    const int nkg = ws_nkg(ntiles * g.nu, g.nk, B.list_grid);
    if (rank == 0 && threadIdx.x == 0) ctl->adj_rows = g.nu * nkg;
    float *out = B.padj;
    const int ld = B.ld_adj;
    return items_adjoint<BF16, true>(J, g, dyn, bars, tmem, B.bimg, B.ximgF, J.cvec, J.fpos, n, ntiles, nkg, rank,
                                     ctas, false, [&](int u, int t, int r, float v) {
                                         const int j = t * kTcM + r;
                                         if (j < n) out[(size_t)j * ld + u] = v;
                                     }, idle);
}

// ---------------------------------------------------------------- LSQR
// One subproblem's LSQR (Sec. V-A): the phases of a Golub-Kahan iteration are
//
//   weighted list image | forward blocks | reduction t = M v - alpha u |
//   B image of t | free-list adjoint | vectors (one CTA)
//
// each a few microseconds of work for a list of some hundred pixels.  Two
// forms of the same phases, chosen by the length of the list (ws_cluster_f):
//
// * short lists, small operands: one kernel, a cluster of kLsqrCtas CTAs that
//   walks the phases, separated by cluster barriers, until the stopping tests hold.
//   As kernels of the solve's graph most of an iteration's ~45 us at p = 100
//   is launch, ramp and drain between the phases.  Eight CTAs are one portable
//   cluster: the hardware places them together, so no phase waits for another
//   solve's CTAs, and 16 solves in flight leave SMs for their gradients.
// * long lists, large operands: a graph WHILE node of one kernel per phase,
//   whose grids spread the images and the reduction over every SM.
//
// Shares and splits follow the list alone (not the CTA count), so every sum
// has the same order in both.
//
// The vector step's FP64 scalars hide where they can (a dependent FP64
// instruction takes 67 cycles, a division 550, hypot 1,050): ||t|| and the
// rotation's part that needs no alpha run in an idle warp of the adjoint
// phase, in the cluster the stopping tests during the next weighted image.
constexpr int kLsqrCtas = 8;
constexpr int kVxReg = 4;               // rows per thread held in registers (f <= 1024)

// beta = ||t|| from the reduction's shares (added as a CTA of 256 threads
// would: 32 shares at a time, butterfly, then in order), u's scale, and the
// rotation up to alpha.  One warp.
__device__ void vx_beta(const WsCtl *ctl, VxState &S, bool init) {
    const int lane = threadIdx.x & 31, n = ctl->nsums;
    double t = 0.0;
    for (int w = 0; w * 32 < n; ++w) {
        double d = w * 32 + lane < n ? ctl->sums[w * 32 + lane] : 0.0;
        for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        t += d;
    }
    const double beta = sqrt(t);
    const double us = beta > 0.0 ? 1.0 / beta : 0.0;
    if (lane == 0) {
        S.beta = beta;
        S.us = us;
        S.fus = (float)us;
        S.fb = (float)beta;
    }
    if (init) {
        if (lane == 0) {
            S.bnorm = S.phibar = beta;
            S.anorm2 = 0.0;
        }
    } else {
        const double alpha = S.alpha, phibar = S.phibar, rhobar = S.rhobar;
        double anorm2 = S.anorm2;
        anorm2 += alpha * alpha + beta * beta;
        const double rho = hypot(rhobar, beta);
        const double q = (lane == 0 ? rhobar : beta) / rho;
        const double c = __shfl_sync(0xffffffffu, q, 0), sn = __shfl_sync(0xffffffffu, q, 1);
        __syncwarp();
        if (lane == 0) {
            S.anorm2 = anorm2;
            S.rho = rho;
            S.c = c;
            S.sn = sn;
            S.phi = c * phibar;
            S.phibar = sn * phibar;
        }
    }
}

// The f-vectors (one CTA): v <- s_F (M^H u) - beta v (init: v <- s_F M^H u),
// M^H u = us times the adjoint's partial dots; alpha = ||v||; v <- v / alpha;
// init: w = v, x = 0, else x += t1 w, w = v + t2 w; the weights s_F v of the
// next forward and their maximum; ||x||^2.
__device__ void vx_step(const JobDev &J, const WsBufs &B, VxState &S, double *sb, float *swm, bool init) {
    WsCtl *ctl = B.ctl;
    const bool w0 = threadIdx.x < 32;
    const int lane = threadIdx.x & 31;
    const int f = ctl->f, ld = B.ld_adj, rows = ctl->adj_rows;
    const int r4 = rows >> 2;
    float *vv = J.v, *ww = J.w, *xx = J.xs;
    const float *sF = J.sF;
    float vr[kVxReg], wr[kVxReg], xr[kVxReg], fr[kVxReg];
#pragma unroll
    for (int q = 0; q < kVxReg; ++q) {
        const int j = threadIdx.x + q * kThreads;
        const bool ok = j < f, old = ok && !init;
        fr[q] = ok ? sF[j] : 0.f;
        vr[q] = old ? vv[j] : 0.f;
        wr[q] = old ? ww[j] : 0.f;
        xr[q] = old ? xx[j] : 0.f;
    }
    const float sc = 1.f / (ctl->sXF * ctl->sB);
    const float fus = S.fus, fb = S.fb;
    float ss = 0.f;
    // two rows per thread per step: every load of both rows is in flight
    // before the sums (rows <= nu nk <= 36 partial dots, 9 float4)
    float4 s4[2][9];
    auto load = [&](int j0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + h * kThreads;
            const bool ok = j < f;
            const float4 *pr = reinterpret_cast<const float4 *>(B.padj + (size_t)(ok ? j : 0) * ld);
#pragma unroll
            for (int q = 0; q < 9; ++q) s4[h][q] = (ok && q < r4) ? __ldcg(pr + q) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    // one row: its new v (before normalisation) from the loaded partial dots
    auto row = [&](int h, int j, float sf, float vo) {
        float y = 0.f;
#pragma unroll
        for (int q = 0; q < 9; ++q) y += (s4[h][q].x + s4[h][q].y) + (s4[h][q].z + s4[h][q].w);
        for (int u = 4 * r4; u < rows; ++u) y += __ldcg(B.padj + (size_t)j * ld + u);
        y *= sc;
        const float yf = __fmul_rn(y, fus);
        const float vn = init ? __fmul_rn(sf, yf) : __fmaf_rn(sf, yf, -__fmul_rn(fb, vo));
        ss = fmaf(vn, vn, ss);
        return vn;
    };
#pragma unroll
    for (int q = 0; q < kVxReg; q += 2) {
        const int j0 = threadIdx.x + q * kThreads;
        if (j0 < f) load(j0);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (j0 + h * kThreads < f) vr[q + h] = row(h, j0 + h * kThreads, fr[q + h], vr[q + h]);
    }
    for (int j0 = threadIdx.x + kVxReg * kThreads; j0 < f; j0 += 2 * kThreads) {
        load(j0);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = j0 + h * kThreads;
            if (j < f) vv[j] = row(h, j, sF[j], init ? 0.f : vv[j]);
        }
    }
    {
        const double t = block_sum_w0((double)ss, sb);
        if (w0) {
            // lanes 0..2: the coefficients of x and w, 1/alpha
            const double alpha = sqrt(t);
            const double rho = init ? 1.0 : S.rho, c = S.c, sn = S.sn, phi = S.phi;
            const double theta = sn * alpha;
            const double q = (lane == 0 ? phi : lane == 1 ? -theta : 1.0) / (lane == 2 ? alpha : rho);
            if (lane == 0) {
                S.alpha = alpha;
                S.rhobar = init ? alpha : -c * alpha;
                S.t1 = init ? 0.f : (float)q;
            }
            if (lane == 1) S.t2 = init ? 0.f : (float)q;
            if (lane == 2) S.ia = alpha > 0.0 ? (float)q : 1.f;
        }
        __syncthreads();
    }
    const float ia = S.ia, ft1 = S.t1, ft2 = S.t2;
    float xs2 = 0.f, wm = 0.f;
    auto update = [&](int j, float vn, float wo, float xo, float sf) {
        const float vj = __fmul_rn(vn, ia);
        vv[j] = vj;
        if (init) {
            ww[j] = vj;
            xx[j] = 0.f;
        } else {
            const float xj = __fmaf_rn(ft1, wo, xo);
            xx[j] = xj;
            ww[j] = __fmaf_rn(ft2, wo, vj);
            xs2 = fmaf(xj, xj, xs2);
        }
        const float wv = sf * vj;
        B.wl[j] = wv;
        wm = fmaxf(wm, fabsf(wv));
    };
#pragma unroll
    for (int q = 0; q < kVxReg; ++q) {
        const int j = threadIdx.x + q * kThreads;
        if (j < f) update(j, vr[q], wr[q], xr[q], fr[q]);
    }
#pragma unroll 4
    for (int j = threadIdx.x + kVxReg * kThreads; j < f; j += kThreads)
        update(j, vv[j], init ? 0.f : ww[j], init ? 0.f : xx[j], sF[j]);
    for (int o = 16; o; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
    if (lane == 0) swm[threadIdx.x >> 5] = wm;
    const double xnorm2 = block_sum_w0((double)xs2, sb);     // its barrier publishes swm too
    if (threadIdx.x == 0) {
        for (int w = 0; w < kThreads / 32; ++w) wm = fmaxf(wm, swm[w]);
        ctl->mx_w = __float_as_uint(wm);
        ctl->mx_t = 0u;                       // the image of t is consumed
        S.xnorm2 = xnorm2;
        // the next forward: t <- M v - alpha u with u = t us, so fa = alpha us
        ctl->fa = S.alpha * S.us;
        if (init) ctl->nsplit = ws_nsplit(f, B.npairs, B.max_tasks, B.fwd_per);
    }
}

// Paige-Saunders stopping tests after `it` iterations (0: after the
// initialisation); one warp, the same answer in every lane.
__device__ bool vx_more(const JobDev &J, const WsCtl *ctl, const VxState &S, int it) {
    const int lane = threadIdx.x & 31;
    if (it == 0) return S.alpha > 0.0 && S.beta > 0.0 && ctl->maxit >= 1;
    const double q = sqrt(lane == 0 ? S.xnorm2 : S.anorm2);
    const double xnorm = __shfl_sync(0xffffffffu, q, 0), anorm = __shfl_sync(0xffffffffu, q, 1);
    const double rnorm = S.phibar;
    const double arnorm = S.phibar * S.alpha * fabs(S.c);
    bool more = it < ctl->maxit;
    if (rnorm <= J.lsqr_btol * S.bnorm + J.lsqr_atol * anorm * xnorm) more = false;
    if (arnorm <= J.lsqr_atol * anorm * rnorm) more = false;
    return more;
}

// All CTAs' writes before, generic or by bulk copies' operands, visible after.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    asm volatile("fence.proxy.async;" ::: "memory");
}

// The phases as kernels: the adjoint with the scalars in an idle warp of CTA
// 0, and the vector step with the stopping tests.
template <bool BF16>
__global__ void __launch_bounds__(kThreads, 1) k_ws_adj_list(const JobDev *Jp, WsBufs B, int init) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (ctl->stop) return;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[kWideBars];
    __shared__ uint32_t tslot;
    if (threadIdx.x < 32) tmem_alloc(&tslot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    const int to = ws_adj_list<BF16>(J, B, unit_geom(J.p), blockIdx.x, gridDim.x, dyn, bars, tmem, [&](int warp) {
        if (blockIdx.x == 0 && warp == 7) vx_beta(ctl, ctl->vx, init);
    });
    if (threadIdx.x < 32) tmem_dealloc(tmem, 512);
    ws_timeouts(ctl, to);
}

__global__ void __launch_bounds__(kThreads) k_ws_vx(const JobDev *Jp, WsBufs B, int init,
                                                    cudaGraphConditionalHandle h_lsqr) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    __shared__ double sb[kThreads / 32];
    __shared__ float swm[kThreads / 32];
    __shared__ VxState S;
    if (ctl->stop) {
        if (threadIdx.x == 0) ws_cond(ctl, kCondLsqr, h_lsqr, 0u);
        return;
    }
    if (threadIdx.x == 0) S = ctl->vx;
    __syncthreads();
    vx_step(J, B, S, sb, swm, init);
    __syncwarp();
    if (threadIdx.x >= 32) return;
    const int it = init ? 0 : ctl->it + 1;
    const bool more = vx_more(J, ctl, S, it);
    if (threadIdx.x == 0) {
        ctl->it = it;
        ctl->vx = S;
        ws_cond(ctl, kCondLsqr, h_lsqr, more ? 1u : 0u);
    }
}

template <bool BF16>
__global__ void __cluster_dims__(kLsqrCtas, 1, 1) __launch_bounds__(kThreads, 1)
k_ws_lsqr(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (ctl->stop) return;
    unsigned char *dyn = dyn_smem();
    __shared__ uint64_t bars[kWideBars];
    __shared__ uint32_t tslot;
    __shared__ double sb[kThreads / 32];
    __shared__ float swm[kThreads / 32];
    __shared__ VxState S;
    const int rank = blockIdx.x;
    const UnitGeom g = unit_geom(J.p);
    if (threadIdx.x < 32) tmem_alloc(&tslot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tslot;
    // data b = base - sum_U s x c c^H, then M^H b
    ws_listimg<BF16, kImgChunksCluster>(J, B, g, kListF, 0, rank, kLsqrCtas);
    ws_listimg<BF16, kImgChunksCluster>(J, B, g, kListU, 0, rank, kLsqrCtas);
    ws_listimg<BF16, kImgChunksCluster>(J, B, g, kListU, 1, rank, kLsqrCtas);
    cluster_sync();
    for (int it = 0;; ++it) {
        const bool init = it == 0;
        if (!init) {
            // the tests of the iteration before run beside the weighted image
            if (rank == 0 && threadIdx.x < 32) {
                const bool more = vx_more(J, ctl, S, it - 1) && !*(volatile int *)&ctl->stop;
                if (threadIdx.x == 0) ctl->cond[kCondLsqr] = more;
            }
            ws_listimg<BF16, kImgChunksCluster>(J, B, g, kListF, 1, rank, kLsqrCtas);
            cluster_sync();
            if (!*(volatile unsigned *)&ctl->cond[kCondLsqr]) {
                if (rank == 0 && threadIdx.x == 0) ctl->it = it - 1;
                break;
            }
        }
        ws_timeouts(ctl, ws_forward<BF16, true>(B, g, init ? kListU : kListF, rank, kLsqrCtas, dyn, bars, tmem));
        cluster_sync();
        ws_fred(J, B, g, init ? kRedB : kRedT, rank, kLsqrCtas);
        cluster_sync();
        ws_emb<BF16, kImgChunksCluster>(J, B, g, J.W0, rank, kLsqrCtas);
        cluster_sync();
        ws_timeouts(ctl, ws_adj_list<BF16>(J, B, g, rank, kLsqrCtas, dyn, bars, tmem, [&](int warp) {
                        if (rank == 0 && warp == 7) vx_beta(ctl, S, init);
                    }));
        cluster_sync();
        if (rank == 0) vx_step(J, B, S, sb, swm, init);
        cluster_sync();
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------- feasibility
// After the subproblem: count its LSQR iterations, test 0 <= z <= u with the
// relative tolerance (non-strict, Table I); h_feas := feasible.
__global__ void k_ws_feas(const JobDev *Jp, WsBufs B, cudaGraphConditionalHandle h_feas) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    __shared__ int s_stop;
    if (threadIdx.x == 0) s_stop = ctl->stop;
    __syncthreads();
    if (s_stop) {
        if (threadIdx.x == 0) ws_cond(ctl, kCondFeas, h_feas, 0u);
        return;
    }
    const int f = ctl->f;
    int bad = 0;
    const double tau = J.feas_tol;
    for (int j = threadIdx.x; j < f; j += blockDim.x) {
        const double z = J.xs[j];
        const double u = J.upper[J.supp[J.fpos[j]]];
        if (!(z >= -tau * u && z <= (1.0 + tau) * u)) bad = 1;
    }
    const bool feasible = __syncthreads_or(bad) == 0;
    if (threadIdx.x == 0) {
        if (f > 0) {
            const int its = min(ctl->it, ctl->maxit);
            ctl->lsqr_total += its;
            ctl->op_flops += (its + 1) * (ws_flops_fwd(J.p, f) + ws_flops_adj(J.p, f));
        }
        ctl->feasible = feasible ? 1 : 0;
        ws_cond(ctl, kCondFeas, h_feas, feasible ? 1u : 0u);
    }
}

// Feasible: x_F = clip(z, 0, u); the support weights -s_i x_i for the
// gradient's residual, their maximum, the support list scale; reset the
// argmin key.
__global__ void k_ws_accept(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (ctl->stop) return;
    const int f = ctl->f, ns = ctl->ns;
    for (int j = threadIdx.x; j < f; j += blockDim.x) {
        const int i = J.supp[J.fpos[j]];
        J.x[i] = fmin(fmax((double)J.xs[j], 0.0), J.upper[i]);
    }
    __syncthreads();
    float wm = 0.f;
    for (int j = threadIdx.x; j < ns; j += blockDim.x) {
        const int i = J.supp[j];
        const float wv = -J.scale[i] * (float)J.x[i];
        B.wl[j] = wv;
        wm = fmaxf(wm, fabsf(wv));
    }
    const float mS = ws_list_max(J.cost == IMG_COST_PWLS ? B.dmax : J.cmax, nullptr, ns);
    __shared__ float swm[kWsThreads / 32];
    for (int o = 16; o; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
    if ((threadIdx.x & 31) == 0) swm[threadIdx.x >> 5] = wm;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 0; w < kWsThreads / 32; ++w) wm = fmaxf(wm, swm[w]);
        ctl->mx_w = __float_as_uint(wm);
        ctl->sXS = pow2_scale(mS) * kLift;
        ctl->nsplit = ws_nsplit(ns, B.npairs, B.max_tasks, B.fwd_per);
        ctl->key = ~0ull;
        ctl->op_flops += ws_flops_fwd(J.p, ns) + ws_flops_adj(J.p, J.Q);
    }
}

// Gradient g_i = -s_i Re(a_i^H U_g a_i) (eq. gls / eq. gmvdr) from the unit
// partial dots; lambda_L = g, lambda_U = -g (eq. etaL, eq. etaU); candidates
// lambda_i < -eps_i off F; smallest lambda, ties to the smallest pixel.
__global__ void k_ws_grad(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (ctl->stop) return;
    const UnitGeom g = unit_geom(J.p);
    const float sc = 1.f / (steer_scale(J.p) * kLift * ctl->sB);
    const int ld = B.ld_adj;
    unsigned long long best = ~0ull;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < J.Q; i += gridDim.x * blockDim.x) {
        float y = 0.f;
        for (int u = 0; u < g.nu; ++u) y += B.padj[(size_t)i * ld + u];
        const float gv = -J.scale[i] * (y * sc);
        J.grad[i] = gv;
        const unsigned char st = J.set[i];
        if (st != IMG_SET_F) {
            const float lam = st == IMG_SET_U ? -gv : gv;
            if (lam < -J.eps[i]) {
                const unsigned long long k = key_of(lam, i);
                best = k < best ? k : best;
            }
        }
    }
    for (int o = 16; o; o >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        best = ob < best ? ob : best;
    }
    if ((threadIdx.x & 31) == 0 && best != ~0ull) atomicMin(&ctl->key, best);
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->mx_t = 0u;
}

__global__ void k_ws_decide(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    WsCtl *ctl = B.ctl;
    if (threadIdx.x != 0 || ctl->stop) return;
    const unsigned long long k = ctl->key;
    if (k == ~0ull) {
        ctl->converged = 1;
        ctl->stop = 1;
        ctl->lam_min = INFINITY;
    } else {
        ctl->pending = (int)(k & 0xffffffffu);
        ctl->lam_min = (double)lam_of(k);
    }
}

// Infeasible: step towards z (eq. mumax), smallest pixel index on ties; the
// blocking pixel goes to U when its direction is positive, to L otherwise,
// exactly at its bound, and leaves the support when it goes to L.
__global__ void k_ws_step(const JobDev *Jp, WsBufs B) {
    ws_count(B.ctl);
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    __shared__ double sv[kWsThreads / 32];
    __shared__ int si[kWsThreads / 32];
    __shared__ int s_stop;
    if (threadIdx.x == 0) s_stop = ctl->stop;
    __syncthreads();
    if (s_stop) return;
    const int f = ctl->f;
    int ns = ctl->ns;
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
    block_argmin(best, bidx, sv, si);
    const double mu = best;
    const int ic = bidx;
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
        ws_log(J, ctl, up ? 2 : 1, ic, (float)mu);
    }
    __syncthreads();
    if (!up) ws_remove(J, B, ic, ns);
    if (threadIdx.x == 0) ctl->ns = ns;
}


// ---------------------------------------------------------------- bounds
// Dirty image and MVDR denominators (Sec. III-C, III-D) on the work-item
// adjoint: out_i = Re(a_i^H U a_i) for U = R_hat and U = R_hat^-1 over every
// pixel, from the unit image of U.  k_ws_bnd_max readies the control block
// (no solve runs on the context meanwhile) and reduces max |U|;
// k_ws_bnd_out sums each pixel's unit partial dots.
__global__ void k_ws_bnd_max(const JobDev *Jp, WsBufs B, const float2 *U, int first, int sq) {
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->adj_sq = sq;
    if (first && blockIdx.x == 0 && threadIdx.x == 0) {
        // bounds (first = 1): a failed factor leaves them alone; the
        // stand-alone adjoint (first = 2) does not depend on the factor
        ctl->stop = first == 1 && J.flags[0] != 0 ? 1 : 0;
        ctl->timeouts = 0;
    }
    const int pp = J.p * J.p;
    float mx = 0.f;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < pp; e += gridDim.x * blockDim.x)
        mx = fmaxf(mx, fmaxf(fabsf(U[e].x), fabsf(U[e].y)));
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&ctl->mx_t, __float_as_uint(mx));
}

__global__ void k_ws_bnd_out(const JobDev *Jp, WsBufs B, float *out) {
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0) post_late(J, ctl->timeouts);
    if (ctl->stop) return;
    const UnitGeom g = unit_geom(J.p);
    const float s1 = steer_scale(J.p) * kLift * ctl->sB;
    const float sc = ctl->adj_sq ? 1.f / (s1 * s1) : 1.f / s1;
    const int ld = B.ld_adj;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < J.Q; i += gridDim.x * blockDim.x) {
        float y = 0.f;
        for (int u = 0; u < g.nu; ++u) y += B.padj[(size_t)i * ld + u];
        out[i] = y * sc;
    }
}

__global__ void k_ws_adj_out(const JobDev *Jp, WsBufs B, double *out) {
    const JobDev &J = *Jp;
    WsCtl *ctl = B.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0) post_late(J, ctl->timeouts);
    if (ctl->stop) return;
    const UnitGeom g = unit_geom(J.p);
    const float sc = 1.f / (steer_scale(J.p) * kLift * ctl->sB);
    const int ld = B.ld_adj;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < J.Q; i += gridDim.x * blockDim.x) {
        float y = 0.f;
        for (int u = 0; u < g.nu; ++u) y += B.padj[(size_t)i * ld + u];
        out[i] = (double)(y * sc);
    }
}

__global__ void k_ws_bnd_reset(WsBufs B) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        B.ctl->mx_t = 0u;
        B.ctl->adj_sq = 0;                    // the solve's adjoints are dots
    }
}

// ================================================================ host side
namespace {

template <class K>
cudaError_t set_smem(K kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

struct Cap {
    cudaStream_t st;
    cudaGraph_t g;
    cudaError_t err = cudaSuccess;
    // begin a capture into g after dependency dep (null: none)
    void begin(cudaGraph_t graph, cudaGraphNode_t dep) {
        g = graph;
        if (err == cudaSuccess)
            err = cudaStreamBeginCaptureToGraph(st, g, dep ? &dep : nullptr, nullptr, dep ? 1 : 0,
                                                cudaStreamCaptureModeRelaxed);
    }
    // end the capture; returns the last captured node
    cudaGraphNode_t end() {
        cudaGraphNode_t leaf = nullptr;
        if (err == cudaSuccess) {
            cudaStreamCaptureStatus cs;
            const cudaGraphNode_t *deps = nullptr;
            size_t nd = 0;
            err = cudaStreamGetCaptureInfo(st, &cs, nullptr, nullptr, &deps, nullptr, &nd);
            if (err == cudaSuccess && nd == 1) leaf = deps[0];
        }
        cudaGraph_t out = nullptr;
        const cudaError_t e = cudaStreamEndCapture(st, &out);
        if (err == cudaSuccess) err = e;
        if (err == cudaSuccess && !leaf) err = cudaErrorStreamCaptureInvalidated;
        return leaf;
    }
    void check() {
        if (err == cudaSuccess) err = cudaGetLastError();
    }
};

cudaGraphNode_t add_cond(Cap &c, cudaGraph_t g, cudaGraphConditionalHandle h, cudaGraphConditionalNodeType type,
                         int size, cudaGraphNode_t dep, cudaGraph_t *bodies) {
    if (c.err != cudaSuccess) return nullptr;
    cudaGraphNodeParams prm = {};
    prm.type = cudaGraphNodeTypeConditional;
    prm.conditional.handle = h;
    prm.conditional.type = type;
    prm.conditional.size = (unsigned)size;
    cudaGraphNode_t node = nullptr;
    c.err = cudaGraphAddNode(&node, g, dep ? &dep : nullptr, nullptr, dep ? 1 : 0, &prm);
    if (c.err == cudaSuccess)
        for (int i = 0; i < size; ++i) bodies[i] = prm.conditional.phGraph_out[i];
    return node;
}

}  // namespace

struct WsHost {
    int device = 0;
    int bf16 = 0;
    int direct = 0;             // host-driven loop instead of the graph
    int sms = 1;
    unsigned *h_cond = nullptr; // pinned mirror of the conditions
    const JobDev *dj = nullptr;
    int p = 0, cap = 0, Q = 0;
    int g_red = 1;              // CTAs of the forward reduction (one tile each)
    UnitGeom g{};
    void *mem = nullptr;
    WsBufs B{};
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

size_t ws_bytes(const JobDev &hj, int sms, WsBufs *B, char *base) {
    const UnitGeom g = unit_geom(hj.p);
    const int cap = hj.cap, p = hj.p;
    size_t off = 0;
    auto take = [&](size_t n) {
        off = (off + 1023) & ~size_t(1023);
        char *r = base ? base + off : nullptr;
        off += n;
        return r;
    };
    WsBufs b{};
    b.npairs = items_fwd_pairs(g, b.pm, b.pnb);
    b.max_tasks = std::max(b.npairs, 2 * std::min(sms, kListGrid));
    b.list_grid = std::min(sms, kListGrid);
    b.fwd_per = kFwdPerTask;
    b.nrows_adj = std::max(hj.Q, cap);
    b.ld_adj = (g.nu * g.nk + 3) / 4 * 4;    // a multiple of 4: rows read as float4
    b.ctl = reinterpret_cast<WsCtl *>(take(sizeof(WsCtl)));
    b.dvec = hj.cost == IMG_COST_PWLS ? reinterpret_cast<float2 *>(take((size_t)cap * p * sizeof(float2))) : nullptr;
    b.dmax = reinterpret_cast<float *>(take((size_t)cap * sizeof(float)));
    b.iota = reinterpret_cast<int *>(take((size_t)cap * sizeof(int)));
    b.wl = reinterpret_cast<float *>(take((size_t)cap * sizeof(float)));
    b.padj = reinterpret_cast<float *>(take((size_t)b.ld_adj * b.nrows_adj * sizeof(float)));
    b.pfwd = reinterpret_cast<float *>(take((size_t)b.max_tasks * kTcM * 256 * sizeof(float)));
    b.ximgF = reinterpret_cast<unsigned char *>(take(list_image_bytes(g, cap)));
    b.ximgS = reinterpret_cast<unsigned char *>(take(list_image_bytes(g, cap)));
    b.ximgW = reinterpret_cast<unsigned char *>(take(list_image_bytes(g, cap)));
    b.bimg = reinterpret_cast<unsigned char *>(take(unit_image_bytes(g)));
    if (B) *B = b;
    return off + 1024;
}

// Most free pixels of LSQR as one cluster kernel (see there): 512 while the B
// image has one unit (p <= 128), none above that or where the GPU has no room
// for the cluster (a partition with fewer SMs).  us per iteration over passes
// that free one pixel each (20 iterations per pass), cluster / kernels, one
// image of p = 100, 72x72 pixels: f = 50 .. 100: 38 / 48, 250 .. 300: 50 / 57,
// 400 .. 500: 54 / 56, 500 .. 700: 65 / 54, 1000 .. 1500: 87 / 65 (8 SMs walk
// lists that fill 32 and more); p = 72: 48 / 53 and 56 / 50 to both sides of
// 500, p = 128: 54 / 57 and 66 / 55.  With 16 images in flight the 8 SMs of a
// cluster stay ahead for longer (p = 100, f = 500 .. 750: 72 / 78, 750 .. 1000: 84
// / 88), with 4 the lines cross at 600.  p = 130 at 64x64, f <= 150: 54 / 41, p =
// 288: 104 / 48 (the reduction and the B image need more than 8 SMs).
constexpr int kClusterF = 512;
template <bool BF>
static int ws_cluster_f(const UnitGeom &g) {
    const size_t sm = items_smem_bytes();
    if (g.nu != 1 || set_smem(k_ws_lsqr<BF>, sm) != cudaSuccess) return 0;
    return active_clusters((const void *)k_ws_lsqr<BF>, kLsqrCtas, kThreads, sm) > 0 ? kClusterF : 0;
}

// The launches of LSQR's initialisation and of one iteration as kernels.
template <bool BF>
static void ws_lsqr_begin(WsHost *w, cudaStream_t s, cudaGraphConditionalHandle h_lsqr) {
    const WsBufs &B = w->B;
    const JobDev *dj = w->dj;
    const size_t fsm = items_fwd_smem_bytes(), asm_ = items_smem_bytes();
    k_ws_listimg<BF><<<w->sms, kWsThreads, 0, s>>>(dj, B, kListF, 0);
    k_ws_listimg<BF><<<w->sms, kWsThreads, 0, s>>>(dj, B, kListU, 0);
    k_ws_listimg<BF><<<w->sms, kWsThreads, 0, s>>>(dj, B, kListU, 1);
    k_ws_fwd<BF><<<B.list_grid, kItemsFwdThreads, fsm, s>>>(dj, B, kListU);
    k_ws_fred<<<w->g_red, kWsThreads, 0, s>>>(dj, B, kRedB);
    k_ws_emb<BF><<<w->sms, kWsThreads, 0, s>>>(dj, B, 0, nullptr);
    k_ws_adj_list<BF><<<B.list_grid, kThreads, asm_, s>>>(dj, B, 1);
    k_ws_vx<<<1, kThreads, 0, s>>>(dj, B, 1, h_lsqr);
}
template <bool BF>
static void ws_lsqr_iterate(WsHost *w, cudaStream_t s, cudaGraphConditionalHandle h_lsqr) {
    const WsBufs &B = w->B;
    const JobDev *dj = w->dj;
    const size_t fsm = items_fwd_smem_bytes(), asm_ = items_smem_bytes();
    k_ws_listimg<BF><<<w->sms, kWsThreads, 0, s>>>(dj, B, kListF, 1);
    k_ws_fwd<BF><<<B.list_grid, kItemsFwdThreads, fsm, s>>>(dj, B, kListF);
    k_ws_fred<<<w->g_red, kWsThreads, 0, s>>>(dj, B, kRedT);
    k_ws_emb<BF><<<w->sms, kWsThreads, 0, s>>>(dj, B, 0, nullptr);
    k_ws_adj_list<BF><<<B.list_grid, kThreads, asm_, s>>>(dj, B, 0);
    k_ws_vx<<<1, kThreads, 0, s>>>(dj, B, 0, h_lsqr);
}

template <bool BF>
static cudaError_t ws_capture(WsHost *w, const JobDev *dj, const JobDev &hj, int sms) {
    const WsBufs &B = w->B;
    Cap c{};
    cudaStreamCreateWithFlags(&c.st, cudaStreamNonBlocking);
    cudaGraph_t G = nullptr;
    c.err = cudaGraphCreate(&G, 0);
    cudaGraphConditionalHandle h_outer = 0, h_form = 0, h_lsqr = 0, h_feas = 0;
    if (c.err == cudaSuccess) c.err = cudaGraphConditionalHandleCreate(&h_outer, G, 1, cudaGraphCondAssignDefault);
    if (c.err == cudaSuccess) c.err = cudaGraphConditionalHandleCreate(&h_form, G, 0, 0);
    if (c.err == cudaSuccess) c.err = cudaGraphConditionalHandleCreate(&h_lsqr, G, 0, 0);
    if (c.err == cudaSuccess) c.err = cudaGraphConditionalHandleCreate(&h_feas, G, 0, 0);
    const size_t fsm = items_fwd_smem_bytes(), asm_ = items_smem_bytes();
    if (c.err == cudaSuccess) c.err = set_smem(k_ws_fwd<BF>, fsm);
    if (c.err == cudaSuccess) c.err = set_smem(k_ws_adj_list<BF>, asm_);
    if (c.err == cudaSuccess) c.err = set_smem(k_ws_adj<BF>, asm_);
    const int g_grad = std::min((hj.Q + kWsThreads - 1) / kWsThreads, 4 * sms);
    const int g_img = sms;
    const int g_cache = (hj.p + kCacheRows - 1) / kCacheRows;
    const int g_fwd = std::min(sms, kListGrid);
    cudaStream_t s = c.st;
    // top level: start, the Table I loop, finish
    c.begin(G, nullptr);
    k_ws_start<<<1, kWsThreads, 0, s>>>(dj, B, h_outer);
    c.check();
    cudaGraphNode_t n0 = c.end();
    cudaGraph_t ob[1] = {};
    cudaGraphNode_t nw = add_cond(c, G, h_outer, cudaGraphCondTypeWhile, 1, n0, ob);
    c.begin(G, nw);
    k_ws_finish<<<1, kWsThreads, 0, s>>>(dj, B);
    c.check();
    c.end();
    // one loop iteration: free the pending pixel, subproblem, branch
    c.begin(ob[0], nullptr);
    k_ws_free<<<1, 32, 0, s>>>(dj, B);
    k_ws_cache<<<g_cache, kWsThreads, 0, s>>>(dj, B);
    k_ws_pass<<<1, kWsThreads, 0, s>>>(dj, B, h_form);
    c.check();
    cudaGraphNode_t n1 = c.end();
    // LSQR on F (Sec. V-A), in the form that k_ws_pass chose: a switch over
    // kLsqr* (its body 0 is empty), or an IF where there are only kernels
    cudaGraph_t lb[3] = {};
    cudaGraphNode_t nif;
    if (w->B.cluster_f > 0) {
        nif = add_cond(c, ob[0], h_form, cudaGraphCondTypeSwitch, 3, n1, lb);
        c.begin(lb[kLsqrCluster], nullptr);
        k_ws_lsqr<BF><<<kLsqrCtas, kThreads, asm_, s>>>(dj, B);
        c.check();
        c.end();
    } else {
        nif = add_cond(c, ob[0], h_form, cudaGraphCondTypeIf, 1, n1, lb + kLsqrKernels);
    }
    c.begin(lb[kLsqrKernels], nullptr);
    ws_lsqr_begin<BF>(w, s, h_lsqr);
    c.check();
    cudaGraphNode_t n2 = c.end();
    cudaGraph_t wb[1] = {};
    add_cond(c, lb[kLsqrKernels], h_lsqr, cudaGraphCondTypeWhile, 1, n2, wb);
    c.begin(wb[0], nullptr);
    ws_lsqr_iterate<BF>(w, s, h_lsqr);
    c.check();
    c.end();
    // feasibility, then the gradient (feasible) or the step (infeasible)
    c.begin(ob[0], nif);
    k_ws_feas<<<1, kWsThreads, 0, s>>>(dj, B, h_feas);
    c.check();
    cudaGraphNode_t n3 = c.end();
    cudaGraph_t fb[2] = {};
    cudaGraphNode_t nfe = add_cond(c, ob[0], h_feas, cudaGraphCondTypeIf, 2, n3, fb);
    c.begin(fb[0], nullptr);
    k_ws_accept<<<1, kWsThreads, 0, s>>>(dj, B);
    k_ws_listimg<BF><<<g_img, kWsThreads, 0, s>>>(dj, B, kListS, 0);
    k_ws_listimg<BF><<<g_img, kWsThreads, 0, s>>>(dj, B, kListS, 1);
    k_ws_fwd<BF><<<g_fwd, kItemsFwdThreads, fsm, s>>>(dj, B, kListS);
    k_ws_fred<<<w->g_red, kWsThreads, 0, s>>>(dj, B, kRedG);
    k_ws_emb<BF><<<g_img, kWsThreads, 0, s>>>(dj, B, 1, nullptr);
    k_ws_adj<BF><<<sms, kWideThreads, asm_, s>>>(dj, B);
    k_ws_grad<<<g_grad, kWsThreads, 0, s>>>(dj, B);
    k_ws_decide<<<1, 32, 0, s>>>(dj, B);
    c.check();
    c.end();
    c.begin(fb[1], nullptr);
    k_ws_step<<<1, kWsThreads, 0, s>>>(dj, B);
    c.check();
    c.end();
    c.begin(ob[0], nfe);
    k_ws_end<<<1, 32, 0, s>>>(dj, B, h_outer);
    c.check();
    c.end();
    if (c.err == cudaSuccess) c.err = cudaGraphInstantiate(&w->exec, G, 0);
    w->graph = G;
    cudaStreamDestroy(c.st);
    return c.err;
}

// The solve with the loop and branches taken on the host: the same kernels in
// the same order as the graph, with a stream synchronisation wherever the
// graph tests a condition.  For tools that cannot look inside graphs with
// conditional nodes (kernel profilers); the results are the same.
template <bool BF>
static cudaError_t ws_direct(WsHost *w, cudaStream_t s) {
    const WsBufs &B = w->B;
    const JobDev *dj = w->dj;
    const int sms = w->sms;
    const size_t fsm = items_fwd_smem_bytes(), asm_ = items_smem_bytes();
    const int g_grad = std::min((w->Q + kWsThreads - 1) / kWsThreads, 4 * sms);
    const int g_img = sms;
    const int g_cache = (w->p + kCacheRows - 1) / kCacheRows;
    const int g_fwd = std::min(sms, kListGrid);
    cudaError_t e = cudaSuccess;
    auto cond = [&](int which) -> unsigned {
        if (e == cudaSuccess) e = cudaMemcpyAsync(w->h_cond, &B.ctl->cond[0], 4 * sizeof(unsigned),
                                                  cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        return e == cudaSuccess ? w->h_cond[which] : 0u;
    };
    k_ws_start<<<1, kWsThreads, 0, s>>>(dj, B, 0);
    while (cond(kCondOuter)) {
        k_ws_free<<<1, 32, 0, s>>>(dj, B);
        k_ws_cache<<<g_cache, kWsThreads, 0, s>>>(dj, B);
        k_ws_pass<<<1, kWsThreads, 0, s>>>(dj, B, 0);
        const unsigned form = cond(kCondLsqrForm);
        if (form == kLsqrCluster) {
            k_ws_lsqr<BF><<<kLsqrCtas, kThreads, asm_, s>>>(dj, B);
        } else if (form == kLsqrKernels) {
            ws_lsqr_begin<BF>(w, s, 0);
            while (cond(kCondLsqr)) ws_lsqr_iterate<BF>(w, s, 0);
        }
        k_ws_feas<<<1, kWsThreads, 0, s>>>(dj, B, 0);
        if (cond(kCondFeas)) {
            k_ws_accept<<<1, kWsThreads, 0, s>>>(dj, B);
            k_ws_listimg<BF><<<g_img, kWsThreads, 0, s>>>(dj, B, kListS, 0);
            k_ws_listimg<BF><<<g_img, kWsThreads, 0, s>>>(dj, B, kListS, 1);
            k_ws_fwd<BF><<<g_fwd, kItemsFwdThreads, fsm, s>>>(dj, B, kListS);
            k_ws_fred<<<w->g_red, kWsThreads, 0, s>>>(dj, B, kRedG);
            k_ws_emb<BF><<<g_img, kWsThreads, 0, s>>>(dj, B, 1, nullptr);
            k_ws_adj<BF><<<sms, kWideThreads, asm_, s>>>(dj, B);
            k_ws_grad<<<g_grad, kWsThreads, 0, s>>>(dj, B);
            k_ws_decide<<<1, 32, 0, s>>>(dj, B);
        } else {
            k_ws_step<<<1, kWsThreads, 0, s>>>(dj, B);
        }
        k_ws_end<<<1, 32, 0, s>>>(dj, B, 0);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) break;
    }
    k_ws_finish<<<1, kWsThreads, 0, s>>>(dj, B);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

// Every kernel of the solve with the largest shared-memory carveout, so the
// SMs need no reconfiguration between the tensor-core kernels (near 200 KB
// of shared memory each) and the small ones in between.
template <bool BF>
static cudaError_t ws_carveout() {
    const int c = cudaSharedmemCarveoutMaxShared;
    const void *ks[] = {(const void *)k_ws_start, (const void *)k_ws_end, (const void *)k_ws_finish,
                        (const void *)k_ws_free, (const void *)k_ws_cache,
                        (const void *)k_ws_pass, (const void *)k_ws_listimg<BF>, (const void *)k_ws_emb<BF>,
                        (const void *)k_ws_fwd<BF>, (const void *)k_ws_fred, (const void *)k_ws_lsqr<BF>, (const void *)k_ws_adj_list<BF>, (const void *)k_ws_vx,
                        (const void *)k_ws_adj<BF>, (const void *)k_ws_feas,
                        (const void *)k_ws_accept, (const void *)k_ws_grad, (const void *)k_ws_decide,
                        (const void *)k_ws_step};
    for (const void *k : ks) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, c);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t ws_create(const JobDev &hj, const JobDev *dj, int mode, WsHost **out) {
    *out = nullptr;
    if (hj.p > kItemsMaxP || (mode != 1 && mode != 2)) return cudaErrorInvalidValue;
    WsHost *w = new WsHost();
    cudaGetDevice(&w->device);
    int sms = 1;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, w->device);
    w->bf16 = mode == 2;
    w->g = unit_geom(hj.p);
    w->sms = sms;
    w->dj = dj;
    w->p = hj.p;
    w->cap = hj.cap;
    w->Q = hj.Q;
    {
        const int ntr = (hj.p + kRedTile - 1) / kRedTile;
        w->g_red = std::min(ntr * ntr, kWsSums);
    }
    {
        const char *env = getenv("IMG_SOLVE_GRAPH");
        w->direct = env && env[0] == '0';
    }
    const size_t bytes = ws_bytes(hj, sms, nullptr, nullptr);
    cudaError_t e = cudaMalloc(&w->mem, bytes);
    if (e != cudaSuccess) {
        delete w;
        return e;
    }
    char *base = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(w->mem) + 1023) & ~uintptr_t(1023));
    ws_bytes(hj, sms, &w->B, base);
    w->B.cluster_f = w->bf16 ? ws_cluster_f<true>(w->g) : ws_cluster_f<false>(w->g);
    e = w->bf16 ? ws_carveout<true>() : ws_carveout<false>();
    if (e == cudaSuccess) e = set_smem(k_ws_adj<true>, items_smem_bytes());
    if (e == cudaSuccess) e = set_smem(k_ws_adj<false>, items_smem_bytes());
    if (e != cudaSuccess) {
        ws_destroy(w);
        return e;
    }
    if (w->direct) {
        e = cudaMallocHost(&w->h_cond, 4 * sizeof(unsigned));
        if (e == cudaSuccess) {
            // the attributes the graph build would set
            e = set_smem(k_ws_fwd<true>, items_fwd_smem_bytes());
            if (e == cudaSuccess) e = set_smem(k_ws_fwd<false>, items_fwd_smem_bytes());
            if (e == cudaSuccess) e = set_smem(k_ws_adj_list<true>, items_smem_bytes());
            if (e == cudaSuccess) e = set_smem(k_ws_adj<true>, items_smem_bytes());
            if (e == cudaSuccess) e = set_smem(k_ws_adj_list<false>, items_smem_bytes());
            if (e == cudaSuccess) e = set_smem(k_ws_adj<false>, items_smem_bytes());
        }
    } else {
        e = w->bf16 ? ws_capture<true>(w, dj, hj, sms) : ws_capture<false>(w, dj, hj, sms);
    }
    if (e != cudaSuccess) {
        ws_destroy(w);
        return e;
    }
    *out = w;
    return cudaSuccess;
}

cudaError_t ws_bounds(WsHost *w, const JobDev &hj, cudaStream_t st) {
    const WsBufs &B = w->B;
    const JobDev *dj = w->dj;
    const int sms = w->sms;
    const size_t asm_ = items_smem_bytes();
    const int gq = std::min((hj.Q + kWsThreads - 1) / kWsThreads, 4 * sms);
    for (int k = 0; k < 2; ++k) {
        // dirty image from R_hat; MVDR denominators ||L^-1 a||^2 from the B
        // image of L^-H (V = L^-1) with the sum-of-squares epilogue
        const float2 *U = k == 0 ? hj.R32 : hj.LiH32;
        k_ws_bnd_reset<<<1, 32, 0, st>>>(B);
        k_ws_bnd_max<<<sms, kWsThreads, 0, st>>>(dj, B, U, k == 0, k);
        if (w->bf16) {
            k_ws_emb<true><<<sms, kWsThreads, 0, st>>>(dj, B, 0, U);
            k_ws_adj<true><<<sms, kWideThreads, asm_, st>>>(dj, B);
        } else {
            k_ws_emb<false><<<sms, kWsThreads, 0, st>>>(dj, B, 0, U);
            k_ws_adj<false><<<sms, kWideThreads, asm_, st>>>(dj, B);
        }
        k_ws_bnd_out<<<gq, kWsThreads, 0, st>>>(dj, B, k == 0 ? hj.dirty : hj.h);
    }
    k_ws_bnd_reset<<<1, 32, 0, st>>>(B);
    return cudaGetLastError();
}

cudaError_t ws_psi_adj(WsHost *w, const JobDev &hj, const float2 *U, double *out, cudaStream_t st) {
    const WsBufs &B = w->B;
    const JobDev *dj = w->dj;
    const int sms = w->sms;
    const size_t asm_ = items_smem_bytes();
    const int gq = std::min((hj.Q + kWsThreads - 1) / kWsThreads, 4 * sms);
    k_ws_bnd_reset<<<1, 32, 0, st>>>(B);
    k_ws_bnd_max<<<sms, kWsThreads, 0, st>>>(dj, B, U, 2, 0);
    if (w->bf16) {
        k_ws_emb<true><<<sms, kWsThreads, 0, st>>>(dj, B, 0, U);
        k_ws_adj<true><<<sms, kWideThreads, asm_, st>>>(dj, B);
    } else {
        k_ws_emb<false><<<sms, kWsThreads, 0, st>>>(dj, B, 0, U);
        k_ws_adj<false><<<sms, kWideThreads, asm_, st>>>(dj, B);
    }
    k_ws_adj_out<<<gq, kWsThreads, 0, st>>>(dj, B, out);
    k_ws_bnd_reset<<<1, 32, 0, st>>>(B);
    return cudaGetLastError();
}

cudaError_t ws_launch(WsHost *w, cudaStream_t st) {
    if (w->direct) return w->bf16 ? ws_direct<true>(w, st) : ws_direct<false>(w, st);
    return cudaGraphLaunch(w->exec, st);
}

size_t ws_size(const JobDev &hj) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return ws_bytes(hj, sms, nullptr, nullptr);
}

void ws_destroy(WsHost *w) {
    if (!w) return;
    if (w->exec) cudaGraphExecDestroy(w->exec);
    if (w->graph) cudaGraphDestroy(w->graph);
    if (w->mem) cudaFree(w->mem);
    if (w->h_cond) cudaFreeHost(w->h_cond);
    delete w;
}

}  // namespace img
