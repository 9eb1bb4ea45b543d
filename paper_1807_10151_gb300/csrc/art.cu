// ART for the Bayesian criterion of Eq. (2.3) and its superiorization SupART
// (Sec. 3.4: the row-action method of Herman, Hurwitz and Lent).
//
// The method sweeps the consistent system r R (x - mu_X) + u = r (b - R mu_X),
// one auxiliary value u_i per ray, whose minimum-norm solution minimises
// r^2 ||R x - b||^2 + ||x - mu_X||^2.  From x = mu_X, u = 0, ray i updates
//     c = lambda (r (b_i - <R_i, x>) - u_i) / (1 + r^2 ||R_i||^2),
//     x <- x + r c R_i,   u_i <- u_i + c,
// and a cycle visits every ray once.  A cycle here takes the views in order
// and, within a view, the rays in S residue classes u = c (mod S), S the
// smallest spacing at which two rays of one view touch no common pixel.  The
// rays of one class run in parallel, one block each: their supports are
// disjoint, so this equals any sequential order of the class; a grid barrier
// (bounded) separates consecutive classes.  A ray's entries are the
// projectors' (the same exact-split delta and trapezoid), evaluated once for
// the ray sum <R_i, x> (a Kahan-compensated FP32 sum per thread, the
// threads' pairs added in double-float arithmetic) and again for the update
// (FP32 FMA).  One block per ray: its threads take a few rows each.
#include <algorithm>

#include "internal.cuh"

namespace supcg {

constexpr int kArtThreads = 64;      // k_art_init
constexpr int kArtLanes = 8;         // its lanes per ray
constexpr int kArtRayThreads = 256;  // k_art: one block per ray of a class

// The per-ray constants of a ray's entries (the projectors' exact split).
struct ArtRay {
    float tau_hi, qh, hi_o, lo_o, hi_i, lo_i, c_in, dI;
    int lo, hi, n_inner, nc;
    bool cb, axis;
};

__device__ __forceinline__ ArtRay art_ray_setup(const Prob &P, const ViewP &vp, int u)
{
    ArtRay R;
    R.cb = (vp.flags & kViewClassB) != 0;
    R.axis = (vp.flags & kViewAxis) != 0;
    R.nc = (vp.flags & kViewFwd3) ? 3 : 2;
    const int n_outer = R.cb ? P.nx : P.ny;
    R.n_inner = R.cb ? P.ny : P.nx;
    R.tau_hi = bin_pos(u, P.uc_hi);                                      // exact
    const float base = __fmaf_rn(vp.a_tau, bin_pos(u, P.uc), vp.g0);    // ray centre at outer index 0
    fwd_row_range(vp, base, R.n_inner, n_outer, &R.lo, &R.hi);
    R.hi_o = R.cb ? vp.cu_hi : vp.su_hi;   // outer coordinate
    R.lo_o = R.cb ? vp.cu_lo : vp.su_lo;
    R.hi_i = R.cb ? vp.su_hi : vp.cu_hi;   // inner coordinate
    R.lo_i = R.cb ? vp.su_lo : vp.cu_lo;
    R.c_in = R.cb ? P.cy : P.cx;
    R.dI = R.cb ? -1.0f : 1.0f;
    R.qh = __fsub_rn(base, vp.hwq);
    return R;
}

// Row o of the ray: the pixel offsets and unit weights of its (up to three)
// candidates; weight 0 for candidates off the image or outside the footprint.
__device__ __forceinline__ void art_row(const Prob &P, const ViewP &vp, const ArtRay &R, int o, int *pix, float *w)
{
    const float of = __int2float_rn(o);
    const float Oc = R.cb ? __fsub_rn(of, P.cx) : __fsub_rn(P.cy, of);
    const float rbig = __fmaf_rn(-R.hi_o, Oc, R.tau_hi);                 // exact
    const float rsmall = __fmaf_rn(R.lo_o, Oc, P.uc_lo);
    const float qc = ceil_magic(__fmaf_rn(of, vp.b_o, R.qh));            // first candidate
    const int q0 = magic_int(qc);
    float I = R.cb ? __fsub_rn(R.c_in, magic_float(qc)) : __fsub_rn(magic_float(qc), R.c_in);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (k) I = __fadd_rn(I, R.dI);                                     // exact
        const float big = __fmaf_rn(-R.hi_i, I, rbig);                   // exact
        const float ad = fabsf(__fsub_rn(big, __fmaf_rn(R.lo_i, I, rsmall)));
        const int q = q0 + k;
        const bool in = k < R.nc && q >= 0 && q < R.n_inner;
        w[k] = in ? weight_unit(ad, vp.E, vp.Sn, vp.ESn, R.axis) : 0.0f;
        pix[k] = in ? (R.cb ? q * P.nxp + o : o * P.nxp + q) : 0;
    }
}

// 1 / (1 + r^2 ||R_i||^2) for every ray (FP64), u = 0, and x = mu_X on the image
// (the starting point of the method).  Eight lanes per ray (no pixel is read, so the
// rows' order does not matter), its exact squares summed in double-float arithmetic:
// with a warp per ray and FP64 squares the narrow FP64 pipe held this at
// 2.35 ms for the 522000 rays of 512^2 / 720 views, 0.60 ms now.  A call without
// cycles, us, with a warp per ray (FP64), 1 lane, 4, 8 and 16: 64^2 / 40 views 84, 92, 78, 72,
// 73; 512^2 / 90 393, 219, 157, 144, 153; 512^2 / 720 2565, 655, 625, 653, 691; 1500 x 64 / 40
// 202, 383, 148, 122, 102 (one lane's rays are a serial chain of up to 1500 rows).
__global__ void __launch_bounds__(kArtThreads) k_art_init(const Prob *__restrict__ probs, double r)
{
    const Prob &P = probs[0];
    const long long rays = (long long)P.V * P.U;
    const int lane = threadIdx.x % kArtLanes;
    constexpr int PER = kArtThreads / kArtLanes;   // rays per block and turn
    for (long long b = (long long)blockIdx.x * PER; b < rays; b += (long long)gridDim.x * PER) {
        const long long i = b + threadIdx.x / kArtLanes;
        const bool have = i < rays;
        const int v = have ? (int)(i / P.U) : 0, u = have ? (int)(i - (long long)v * P.U) : 0;
        const ViewP vp = P.views[v];
        const ArtRay R = art_ray_setup(P, vp, u);
        df s = df_make(0.0f);
        for (int o = R.lo + lane; o <= R.hi; o += kArtLanes) {
            int pix[3];
            float w[3];
            art_row(P, vp, R, o, pix, w);
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if (w[k] != 0.0f) df_acc_prod(s, w[k], w[k]);
        }
#pragma unroll
        for (int o = kArtLanes / 2; o > 0; o >>= 1)
            s = df_add(s, df{__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.l, o)});
        if (have && lane == 0) {
            const double pl = (double)vp.P;
            P.art_rn[i] = 1.0 / (1.0 + r * r * pl * pl * df_to_double(s));
            P.art_u[i] = 0.0;
        }
    }
    const float mu = (float)P.sc->muX;
    const size_t n = (size_t)P.ny * P.nxp;
    for (size_t e = (size_t)blockIdx.x * kArtThreads + threadIdx.x; e < n; e += (size_t)gridDim.x * kArtThreads) {
        const int j = (int)(e % P.nxp);
        P.x[e] = (j < P.nx) ? mu : 0.0f;   // the padding stays 0
    }
}

// The step of one ray: c from its sum s (in units of the plateau length pl), u <- u + c; returns r c pl.
// A call, not inlined: an FP64 instruction holds the SM's pipe for tens of cycles per warp that issues it, and
// inlined under a test for one thread it may be issued, predicated off, by all.
__device__ __noinline__ float art_coef(df s, float pl, float b, double ui, double rn, double r, double lam, double *u)
{
    const double cc = lam * (r * ((double)b - (double)pl * df_to_double(s)) - ui) * rn;
    *u = ui + cc;
    return (float)(r * cc * (double)pl);
}

// `cycles` full ART cycles on P.x (one cooperative launch; every block takes part in every
// class barrier).  Block b takes the rays u = c + S (b + k nblocks) of class c.  The classes
// are a serial chain (1440 per cycle at 512^2 / 720 views), so what counts is the time from
// one barrier to the next: the first ROWS rows per thread of the block's next ray, their
// weights and its scalars are evaluated between the arrival at a barrier and the wait, so
// that after it only the pixels are read, summed and updated.  The pixels are read through
// L1 (the barrier's fence empties it of what other blocks have written since): a row's two or
// three candidates are neighbours, and past L1 each of them fetched its own sector from L2.
// A class takes 4.4 us, 6.6 before (the weights after the barrier, the threads' sums added in
// FP64, 128 threads per ray); of it about 2.5 us are the barrier and the SMs with three
// of the 363 blocks are the last to arrive.  Rows beyond the first
// ROWS * kArtRayThreads, and further rays of a block, are evaluated where they are used.
template <int ROWS>
__global__ void __launch_bounds__(kArtRayThreads) k_art(const Prob *__restrict__ probs, int cycles, double r,
                                                        double lam, int S)
{
    constexpr int N = 3 * ROWS, GROUP = ROWS * kArtRayThreads;
    __shared__ int flag;
    __shared__ __align__(16) double red[40];
    __shared__ float sh_rc;
    const Prob &P = probs[0];
    Scal *sc = P.sc;
    const int t = threadIdx.x;
    float *x = P.x;
    GridCount bar(P.bar + 4, gridDim.x + P.bar_extra);

    // the pixels and weights of rows o0, o0 + kArtRayThreads, ... of a ray
    auto rows_of = [&](const ViewP &vp, const ArtRay &R, int o0, int *pix, float *w) {
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
            const int o = o0 + q * kArtRayThreads;
            if (o <= R.hi) {
                art_row(P, vp, R, o, pix + 3 * q, w + 3 * q);
            } else {
                w[3 * q] = w[3 * q + 1] = w[3 * q + 2] = 0.0f;
                pix[3 * q] = pix[3 * q + 1] = pix[3 * q + 2] = 0;
            }
        }
    };
    // the ray under way: its first group's pixels and weights, thread 0's scalars
    int gpix[N];
    float gw[N], bi = 0.0f, pl = 0.0f;
    double ui = 0.0, rni = 0.0;
    bool more = false;   // rows beyond the first group
    auto prepare = [&](int v, int u) {
        const ViewP vp = P.views[v];
        const ArtRay R = art_ray_setup(P, vp, u);
        rows_of(vp, R, R.lo + t, gpix, gw);
        more = R.hi - R.lo >= GROUP;
        pl = vp.P;
        if (t == 0) {
            bi = P.bpad[(size_t)v * P.Up + u];
            ui = P.art_u[(size_t)v * P.U + u];   // (written only by this block, at the ray's last visit)
            rni = P.art_rn[(size_t)v * P.U + u];
        }
    };
    float ks, kc;   // Kahan pair of the thread's terms of <R_i, x>
    auto load_and_sum = [&](const int *pix, const float *w, float *xv) {
#pragma unroll
        for (int k = 0; k < N; ++k) xv[k] = (w[k] != 0.0f) ? x[pix[k]] : 0.0f;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const float y = __fmaf_rn(w[k], xv[k], -kc);
            const float tt = __fadd_rn(ks, y);
            kc = __fsub_rn(__fsub_rn(tt, ks), y);
            ks = tt;
        }
    };
    auto visit = [&](int v, int u) {
        float gx[N];   // (the class's other rays touch none of these pixels: still current at the update)
        ks = kc = 0.0f;
        load_and_sum(gpix, gw, gx);
        if (more) {
            const ViewP vp = P.views[v];
            const ArtRay R = art_ray_setup(P, vp, u);
            for (int o0 = R.lo + t + GROUP; o0 <= R.hi; o0 += GROUP) {
                int pix[N];
                float w[N], xv[N];
                rows_of(vp, R, o0, pix, w);
                load_and_sum(pix, w, xv);
            }
        }
        const df s = block_sum_pair<kArtRayThreads>(df{ks, -kc}, red);   // in thread 0
        if (t == 0) sh_rc = art_coef(s, pl, bi, ui, rni, r, lam, P.art_u + (size_t)v * P.U + u);
        __syncthreads();
        const float rcf = sh_rc;
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (gw[k] != 0.0f) x[gpix[k]] = __fmaf_rn(rcf, gw[k], gx[k]);
        if (more) {
            const ViewP vp = P.views[v];
            const ArtRay R = art_ray_setup(P, vp, u);
            for (int o0 = R.lo + t + GROUP; o0 <= R.hi; o0 += GROUP) {
                int pix[N];
                float w[N], xv[N];
                rows_of(vp, R, o0, pix, w);
#pragma unroll
                for (int k = 0; k < N; ++k) xv[k] = (w[k] != 0.0f) ? x[pix[k]] : 0.0f;
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (w[k] != 0.0f) x[pix[k]] = __fmaf_rn(rcf, w[k], xv[k]);
            }
        }
    };
    const int u0 = S * blockIdx.x;   // the block's first ray of a class: c + u0
    if (u0 < P.U) prepare(0, u0);
    for (int cyc = 0; cyc < cycles; ++cyc) {
        for (int v = 0; v < P.V; ++v) {
            for (int c = 0; c < S; ++c) {
                if (c + u0 < P.U) {
                    visit(v, c + u0);
                    for (int u = c + u0 + S * gridDim.x; u < P.U; u += S * gridDim.x) {   // block-uniform
                        prepare(v, u);
                        __syncthreads();   // sh_rc and red are reused
                        visit(v, u);
                    }
                }
                bar.arrive();
                const int nc = c + 1 < S ? c + 1 : 0, nv = nc ? v : (v + 1 < P.V ? v + 1 : 0);
                if (nc + u0 < P.U) prepare(nv, nc + u0);
                if (!bar.wait<true>(P.wait_limit, &sc->status, &flag)) return;   // bounded: SUPCG_ERR_TIMEOUT
            }
        }
    }
}

// Rows per thread.  One or two where they hold the longest ray in one group; beyond 512 rows or columns 4 where most
// rays are long (both sides above 512 and 1536 together), else 2 and further groups: four rows take 124 registers,
// so the device holds 304 blocks instead of 456, and a block's further rays of a class are prepared one after the
// other.  Two classes (a view), us, with 2 and 4 rows: 513^2 10.8 and 12.4, 700^2 14.4 and 15.6, 768^2 16.7 and
// 16.6, 850^2 19.2 and 17.4, 900^2 20.8 and 22.0, 1024^2 25.8 and 22.1, 2048^2 114 and 96; 1100 x 300 14.4 and 18.0,
// 1500 x 64 15.1 and 19.2, 2048 x 400 25.2 and 29.8, 1400 x 800 31.4 and 29.0, 2048 x 700 39.6 and 36.4.
template <typename F>
static int with_art_rows(int nx, int ny, F &&f)
{
    const int side = std::max(nx, ny);
    if (side <= kArtRayThreads) return f(k_art<1>);
    if (side <= 2 * kArtRayThreads || std::min(nx, ny) <= 512 || nx + ny <= 1536) return f(k_art<2>);
    return f(k_art<4>);
}

int art_max_blocks(int nx, int ny, int *out)
{
    return with_art_rows(nx, ny, [&](auto *kernel) { return resident_blocks((const void *)kernel, kArtRayThreads, 0, out); });
}

int launch_art_init(const Prob *d_prob, double r, long long rays, cudaStream_t st)
{
    const int blocks = (int)std::min<long long>(8192, (rays * kArtLanes + kArtThreads - 1) / kArtThreads);
    k_art_init<<<blocks, kArtThreads, 0, st>>>(d_prob, r);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

int launch_art(const Prob *d_prob, int nx, int ny, int cycles, double r, double lam, int S, int blocks, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kArtRayThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return with_art_rows(nx, ny, [&](auto *kernel) -> int {
        SUPCG_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, d_prob, cycles, r, lam, S));
        return SUPCG_OK;
    });
}

} // namespace supcg
