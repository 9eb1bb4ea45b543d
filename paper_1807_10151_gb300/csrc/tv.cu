// Total variation, its nonascending vector and S_TV (Sec. 3.1, Algorithm 1).
//
//   TV(y) = sum_{i<ny-1, j<nx-1} sqrt((y_ij - y_i+1,j)^2 + (y_ij - y_i,j+1)^2)
//   tbar_p = -dTV/dy_p where the partial exists (every TV term containing y_p
//            has a nonzero root, i.e. not both of its differences are 0), else 0
//   t = tbar / ||tbar||  (0 when tbar = 0)
//
// S_TV runs as one cooperative launch per call: each problem owns a fixed set
// of co-resident blocks that meet at bounded device barriers, so the
// data-dependent backtracking loop (repeat ... until TV(y~) <= TV(y)) runs
// on the device without returning to the host.  Every block sums the
// per-block FP64 partials in the same order, so all blocks take the same
// accept / reject decision.  Two kernels: k_stv_tile keeps the image in shared
// memory through the K steps (images that fit, up to about 1100^2), k_stv walks
// it in memory (larger images, and the learned direction's step).
#include "internal.cuh"

namespace supcg {

constexpr int kTvThreads = 256;

// The seven values of y (pitch ld) that tbar at pixel (i, j) depends on: the pixel,
// its lower and right neighbours, the upper row's pixel and its right neighbour,
// the left pixel and its lower neighbour (0 where the term they belong to does not
// exist).  Loading them apart from the arithmetic lets a thread issue the loads of
// several pixels before it waits for any.
struct Nb7 {
    float c, d, r, u, ur, l, ld;
};
__device__ __forceinline__ Nb7 nb7_load(const float *__restrict__ y, int ld, int ny, int nx, int i, int j)
{
    Nb7 v = {};
    const size_t p = (size_t)i * ld + j;
    v.c = y[p];
    if (i + 1 < ny && j + 1 < nx) {
        v.d = y[p + ld];
        v.r = y[p + 1];
    }
    if (i >= 1 && j + 1 < nx) {
        v.u = y[p - ld];
        v.ur = y[p - ld + 1];
    }
    if (j >= 1 && i + 1 < ny) {
        v.l = y[p - 1];
        v.ld = y[p + ld - 1];
    }
    return v;
}

// The root of a TV term with differences a (down) and b (right).  Where the two differences are near the
// rounding of the image a step's direction hangs on the last bit of this root, so it is pinned: one product
// rounded, the other inside the FMA, which of the two as the kernels have always had it (root in a pixel's
// own term and in the term of the pixel above it, root_b in that of the pixel left of it).
__device__ __forceinline__ float root(float a, float b) { return sqrtf(__fmaf_rn(a, a, __fmul_rn(b, b))); }
__device__ __forceinline__ float root_b(float a, float b) { return sqrtf(__fmaf_rn(b, b, __fmul_rn(a, a))); }

// tbar at pixel (i, j) from its seven values; *Tb receives the root of the TV term
// whose base is (i, j) (0 if that term does not exist).
__device__ __forceinline__ float tbar_from(const Nb7 &v, int ny, int nx, int i, int j, float *Tb)
{
    float g = 0.0f;
    bool undef = false;
    float tb = 0.0f;
    const float yc = v.c;
    if (i + 1 < ny && j + 1 < nx) {
        const float a = yc - v.d, b = yc - v.r;
        if (a == 0.0f && b == 0.0f) undef = true;
        else {
            const float T = root(a, b);
            tb = T;
            g += (a + b) / T;
        }
    }
    if (i >= 1 && j + 1 < nx) {
        const float yu = v.u;
        const float a = yu - yc, b = yu - v.ur;
        if (a == 0.0f && b == 0.0f) undef = true;
        else g -= a / root(a, b);
    }
    if (j >= 1 && i + 1 < ny) {
        const float yl = v.l;
        const float a = yl - v.ld, b = yl - yc;
        if (a == 0.0f && b == 0.0f) undef = true;
        else g -= b / root_b(a, b);
    }
    *Tb = tb;
    return undef ? 0.0f : -g;
}

// tbar at pixel (i, j) of y (pitch ld); *Tb as for tbar_from.
__device__ __forceinline__ float tbar_at(const float *__restrict__ y, int ld, int ny, int nx, int i, int j,
                                         float *Tb)
{
    return tbar_from(nb7_load(y, ld, ny, nx, i, j), ny, nx, i, j, Tb);
}

// A thread's pixels e0, e0 + stride, ... of an ny x nx image as (i, j), stepped
// without a division per pixel; S_TV's passes take them kStvGroup at a time, all
// of a group's loads issued before its arithmetic.
constexpr int kStvGroup = 2;
struct PixWalk {
    int i, j, si, sj, nx;
    __device__ PixWalk(int e0, int stride, int nx_) : nx(nx_)
    {
        i = e0 / nx;
        j = e0 - i * nx;
        si = stride / nx;
        sj = stride - si * nx;
    }
    __device__ __forceinline__ void next()
    {
        j += sj;
        i += si;
        if (j >= nx) {
            j -= nx;
            ++i;
        }
    }
};

// The FP32 image value of y + c t, as x_step stores it: from the pair (y, lo) where has_lo.  (k_stv's trials once
// took the high part's FMA alone, an ulp off the image that an accepted trial leaves and that k_stv_tile's trials
// take; the pair costs 5 % of K = 40 at 1400^2 and 8 % at 2048^2, 1764 -> 1862 and 2910 -> 3160 us.)
__device__ __forceinline__ float step_value(float y, float lo, bool has_lo, float c, float t)
{
    return has_lo ? df_add(df{y, lo}, df_prod(c, t)).h : __fmaf_rn(c, t, y);
}

// y <- y + c t at element p of the iterate: in double-float arithmetic on the pair
// (x, xlo) when the low part exists (the exact product c t added to it), else one
// FP32 FMA.  Returns the new FP32 image value x = RN(x + xlo).
__device__ __forceinline__ float x_step(float *__restrict__ x, float *__restrict__ xlo, size_t p, float c, float t,
                                        float *lo_out = nullptr)
{
    if (!xlo) {
        const float v = __fmaf_rn(c, t, x[p]);
        x[p] = v;
        if (lo_out) *lo_out = 0.0f;
        return v;
    }
    const df v = df_add(df{x[p], xlo[p]}, df_prod(c, t));
    x[p] = v.h;
    xlo[p] = v.l;
    if (lo_out) *lo_out = v.l;
    return v.h;
}

// Standalone TV and tbar of P.x (one image per problem): writes P.tbar and
// sc->tv_k = TV, sc->snorm2 = ||tbar||^2.
__global__ void __launch_bounds__(kTvThreads) k_tv_tbar(const Prob *__restrict__ probs, const int *__restrict__ prefix,
                                                        int count)
{
    __shared__ __align__(16) double red[40];
    __shared__ int flag;
    int local;
    const int pi = find_problem(prefix, count, blockIdx.x, &local);
    const Prob &P = probs[pi];
    const int nblk = prefix[pi + 1] - prefix[pi];
    const long long n = (long long)P.ny * P.nx;
    df s_tv = df_make(0.0f), s_nn = df_make(0.0f);   // double-float sums, FP64 per thread
    for (long long e = (long long)local * kTvThreads + threadIdx.x; e < n; e += (long long)nblk * kTvThreads) {
        const int i = (int)(e / P.nx), j = (int)(e - (long long)i * P.nx);
        float Tb;
        const float tb = tbar_at(P.x, P.nxp, P.ny, P.nx, i, j, &Tb);
        P.tbar[(size_t)i * P.nxp + j] = tb;
        df_acc(s_tv, Tb);
        df_acc_prod(s_nn, tb, tb);
    }
    double btv, bnn;
    block_sum_df2<kTvThreads>(s_tv, s_nn, red, &btv, &bnn);
    if (threadIdx.x == 0) {
        P.partial[local] = btv;
        P.partial[nblk + local] = bnn;
    }
    if (last_block(&P.counter[3], nblk, &flag)) {
        double tv, nn;
        block_sum_array2<kTvThreads>(P.partial, P.partial + nblk, nblk, red, &tv, &nn);
        if (threadIdx.x == 0) {
            P.sc->tv_k = tv;
            P.sc->snorm2 = nn;
            P.counter[3] = 0;
        }
    }
}

int launch_tv_tbar(const Launch &L)
{
    k_tv_tbar<<<L.blocks, kTvThreads, 0, L.st>>>(L.probs, L.prefix, L.count);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

// Sum of the block partials of one phase, identical in every block (per-thread values
// in FP64 or as double-float pairs).
__device__ __forceinline__ double phase_sum_of(const Prob &P, int nb, int slot, int local, double bs, double *red,
                                               int *flag, bool *ok);
__device__ __forceinline__ double phase_sum(const Prob &P, int nb, int slot, int local, df v, double *red,
                                            int *flag, bool *ok)
{
    return phase_sum_of(P, nb, slot, local, block_sum_df<kTvThreads>(v, red), red, flag, ok);
}
__device__ __forceinline__ double phase_sum(const Prob &P, int nb, int slot, int local, double v, double *red,
                                            int *flag, bool *ok)
{
    return phase_sum_of(P, nb, slot, local, block_sum<kTvThreads>(v, red), red, flag, ok);
}
__device__ __forceinline__ double phase_sum_of(const Prob &P, int nb, int slot, int local, double bs, double *red,
                                               int *flag, bool *ok)
{
    if (threadIdx.x == 0) P.partial[(size_t)slot * nb + local] = bs;
    *ok = coop_barrier(P.bar, nb + P.bar_extra, &P.sc->status, flag, P.wait_limit);
    if (!*ok) return 0.0;
    return block_sum_array<kTvThreads>(P.partial + (size_t)slot * nb, nb, red);
}

// S_TV(x, l, a, gamma, K), Algorithm 1, in place on P.x (one cooperative launch).
// trials_out (nullable): [count][K] trials of every nonascending step.  dir (nullable):
// the learned proposals, [count][ny][nx] (every problem of the launch has the same size).
// Also writes the displacement d = x_{k+1/2} - x_k in the forward projector's layouts
// (P.d, P.dT and, with mirror pairs, P.dm, P.dmT), which a while-body projects to move
// the residual.
__global__ void __launch_bounds__(kTvThreads, 3) k_stv(const Prob *__restrict__ probs, const int *__restrict__ prefix,
                                                    int count, int K_arg, double a_arg, double gamma_arg,
                                                    long long max_trials, int *trials_out, int want_snorm,
                                                    const float *__restrict__ dir_all)
{
    const float *dir = dir_all;
    __shared__ __align__(16) double red[40];
    __shared__ int flag;
    __shared__ double sh_inv;   // grid-uniform FP64 scalars: computed by thread 0, read by all
    __shared__ float sh_c;
    __shared__ float sh_t[32][33];   // tile transposes of d
    bool d_done = false;             // the last step wrote d
    int local;
    const int pi = find_problem(prefix, count, blockIdx.x, &local);
    const Prob &P = probs[pi];
    Scal *sc = P.sc;
    if (sc->done) return;
    // a parameter sweep gives every problem its own K, a, gamma
    const int K = P.stv_own ? P.stv_K : K_arg;
    const double a = P.stv_own ? P.stv_a : a_arg, gamma = P.stv_own ? P.stv_gamma : gamma_arg;
    const int nb = prefix[pi + 1] - prefix[pi];
    const int nx = P.nx, ny = P.ny, ld = P.nxp;
    const int n = ny * nx;   // < 2^31 (each side <= 16384)
    const int stride = nb * kTvThreads;
    const int e0 = local * kTvThreads + threadIdx.x;
    float *x = P.x;
    float *xl = P.xlo;   // low part of the iterate (null: FP32 updates)
    // a batched learned solve passes the proposals of all problems back to back ([count][ny][nx])
    if (dir) dir += (size_t)pi * ny * nx;
    float *tb = P.tbar;
    long long ell = sc->ell;
    // a^ell, carried from trial to trial and from call to call (Scal::apow); thread 0's, kept
    // in shared memory so that it takes no registers through the passes
    __shared__ double sh_apow;
    __shared__ int sh_apow_ok;
    if (threadIdx.x == 0) {
        sh_apow_ok = sc->apow_ok && sc->apow_ell == ell && sc->apow_a == a;
        sh_apow = sh_apow_ok ? sc->apow : 0.0;
    }
    long long total_trials = 0;
    double tv_first = 0.0, tv_last = 0.0;
    int slot = 0;   // partial buffers alternate between two slots (pairs of slots for 2-value phases)
    bool ok = true;
    // x_k is saved before the steps unless one plain step (K = 1) gives d as c tbar itself
    const bool saved = want_snorm || dir || K != 1;
    // d on the 32 x 32 tiles this block owns, in the row layout and transposed (and mirrored
    // with mirror pairs).  step: the last step y <- y + c tbar is taken here, pixel by pixel
    // (no block reads another's pixels after it, so no grid barrier follows); zero: no step
    // moved x.  Otherwise d = x - x_k from the copy saved before the steps, which a grid
    // barrier separates from here.
    auto write_d = [&](bool step, bool zero, float c) {
        const int tiles_j = (nx + 31) / 32, tiles = ((ny + 31) / 32) * tiles_j;
        const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 256 threads: 32 x 8
        for (int tile = local; tile < tiles; tile += nb) {
            const int ti = tile / tiles_j, tj = tile - ti * tiles_j;
            for (int r = ty; r < 32; r += 8) {
                const int i = ti * 32 + r, j = tj * 32 + tx;
                float dv = 0.0f;
                if (i < ny && j < nx) {
                    const size_t p = (size_t)i * ld + j;
                    float v, vl;
                    if (step) {
                        const float t = tb[p];
                        v = x_step(x, xl, p, c, t, &vl);
                        if (!saved) dv = __fmul_rn(c, t);
                    } else {
                        v = x[p];
                        vl = xl ? xl[p] : 0.0f;
                    }
                    if (saved && !zero) dv = __fadd_rn(__fsub_rn(v, P.z[p]), __fsub_rn(vl, P.g[p]));
                    P.d[p] = dv;
                    if (P.dm) P.dm[(size_t)i * ld + (nx - 1 - j)] = dv;
                }
                sh_t[r][tx] = dv;
            }
            __syncthreads();
            for (int r = ty; r < 32; r += 8) {
                const int j = tj * 32 + r, i = ti * 32 + tx;
                if (j < nx && i < ny) {
                    P.dT[(size_t)j * P.nyp + i] = sh_t[tx][r];
                    if (P.dmT) P.dmT[(size_t)(nx - 1 - j) * P.nyp + i] = sh_t[tx][r];
                }
            }
            __syncthreads();
        }
    };

    // the iterate before the steps, high part in z and low part in g (both are recomputed
    // after S_TV in a while-body), for ||s_k||^2 of the log and for d
    if (saved)
        for (int e = e0; e < n; e += stride) {
            const int i = e / nx, j = e - i * nx;
            const size_t p = (size_t)i * ld + j;
            P.z[p] = x[p];
            P.g[p] = xl ? xl[p] : 0.0f;
        }

    // Learned direction (dir != null, pitch nx): accepted only when nonascending for TV,
    // i.e. when the one-sided directional derivative D_TV(x; dir) is negative; then one
    // step of length 2^-j gamma sum_{i<K} a^(l+i) (j = rejected trials so far; halving,
    // since a long step shrinks too slowly by factors of a near 1) replaces the K steps of
    // Algorithm 1, and l advances by K + j, so ||s_k|| <= K gamma a^(l_k) as in Theorem 1.
    // Otherwise the K plain steps run.
    bool plain = true;
    if (dir) {
        double s_nn = 0.0, s_dd = 0.0, s_tv = 0.0;
        for (int e = e0; e < n; e += stride) {
            const int i = e / nx, j = e - i * nx;
            const size_t p = (size_t)i * ld + j;
            const size_t q = (size_t)i * nx + j;
            const float tp = dir[q];
            s_nn += (double)tp * (double)tp;
            if (i + 1 < ny && j + 1 < nx) {
                const float a1 = x[p] - x[p + ld], b1 = x[p] - x[p + 1];
                const float ta = tp - dir[q + nx], tb = tp - dir[q + 1];
                if (a1 == 0.0f && b1 == 0.0f) {
                    s_dd += (double)sqrtf(ta * ta + tb * tb);
                } else {
                    const double T = (double)sqrtf(a1 * a1 + b1 * b1);
                    s_tv += T;
                    s_dd += ((double)a1 * ta + (double)b1 * tb) / T;
                }
            }
        }
        {
            const double v1 = block_sum<kTvThreads>(s_nn, red);
            const double v2 = block_sum<kTvThreads>(s_dd, red);
            const double v3 = block_sum<kTvThreads>(s_tv, red);
            if (threadIdx.x == 0) {
                P.partial[(size_t)8 * nb + local] = v1;
                P.partial[(size_t)9 * nb + local] = v2;
                P.partial[(size_t)10 * nb + local] = v3;
            }
            ok = coop_barrier(P.bar, nb + P.bar_extra, &sc->status, &flag, P.wait_limit);
            if (ok) {
                s_nn = block_sum_array<kTvThreads>(P.partial + (size_t)8 * nb, nb, red);
                s_dd = block_sum_array<kTvThreads>(P.partial + (size_t)9 * nb, nb, red);
                s_tv = block_sum_array<kTvThreads>(P.partial + (size_t)10 * nb, nb, red);
            }
        }
        if (ok && s_dd < 0.0 && s_nn > 0.0) {
            plain = false;
            // the step scalars are the same in every thread: thread 0 evaluates the FP64
            // functions and the block reads the result (the FP64 pipe is narrow)
            if (threadIdx.x == 0) sh_inv = rsqrt_fp64(s_nn);
            long long j = 0;
            float c = 0.0f;
            double tv_t = 0.0;
            for (;;) {
                if (j >= max_trials) {
                    if (local == 0 && threadIdx.x == 0) atomicExch(&sc->status, (int)SUPCG_ERR_BACKTRACK);
                    ok = false;
                    break;
                }
                if (threadIdx.x == 0) {
                    const double geo = (a == 1.0) ? (double)K : (1.0 - pow(a, (double)K)) / (1.0 - a);
                    sh_c = (float)(ldexp(gamma * pow(a, (double)ell) * geo, -(int)min(j, 2000ll)) * sh_inv);
                }
                __syncthreads();
                c = sh_c;
                ++j;
                double sacc = 0.0;
                for (int e = e0; e < n; e += stride) {
                    const int i = e / nx, jj = e - i * nx;
                    if (i + 1 < ny && jj + 1 < nx) {
                        const size_t p = (size_t)i * ld + jj, q = (size_t)i * nx + jj;
                        const float yc = __fmaf_rn(c, dir[q], x[p]);
                        const float yd = __fmaf_rn(c, dir[q + nx], x[p + ld]);
                        const float yr = __fmaf_rn(c, dir[q + 1], x[p + 1]);
                        const float a1 = yc - yd, b1 = yc - yr;
                        sacc += (double)sqrtf(a1 * a1 + b1 * b1);
                    }
                }
                tv_t = phase_sum(P, nb, slot, local, sacc, red, &flag, &ok);
                slot ^= 1;
                if (!ok) break;
                if (tv_t <= s_tv) break;
            }
            if (ok) {
                for (int e = e0; e < n; e += stride) {
                    const int i = e / nx, jj = e - i * nx;
                    (void)x_step(x, xl, (size_t)i * ld + jj, c, dir[(size_t)i * nx + jj]);
                }
                ok = coop_barrier(P.bar, nb + P.bar_extra, &sc->status, &flag, P.wait_limit);
                ell += (long long)K + (j - 1);
                if (threadIdx.x == 0) sh_apow_ok = 0;
                total_trials = j;
                tv_first = s_tv;
                tv_last = tv_t;
                if (local == 0 && threadIdx.x == 0) sc->n_learned += 1;
            }
        } else if (local == 0 && threadIdx.x == 0) {
            sc->n_fallback += 1;
        }
    }

    for (int step = 0; plain && step < K && ok; ++step) {
        // t in the nonascending set at y (Sec. 3.1)
        df d_tv = df_make(0.0f), d_nn = df_make(0.0f);   // double-float sums, FP64 per thread
        for (PixWalk w(e0, stride, nx); w.i < ny;) {
            int gi[kStvGroup], gj[kStvGroup];
            Nb7 v[kStvGroup];
#pragma unroll
            for (int q = 0; q < kStvGroup; ++q) {
                gi[q] = w.i;
                gj[q] = w.j;
                if (w.i < ny) v[q] = nb7_load(x, ld, ny, nx, w.i, w.j);
                w.next();
            }
#pragma unroll
            for (int q = 0; q < kStvGroup; ++q) {
                if (gi[q] < ny) {
                    float Tb;
                    const float t = tbar_from(v[q], ny, nx, gi[q], gj[q], &Tb);
                    tb[(size_t)gi[q] * ld + gj[q]] = t;
                    df_acc(d_tv, Tb);
                    df_acc_prod(d_nn, t, t);
                }
            }
        }
        double s_tv, s_nn;
        // two sums through one barrier: slots 2*slot and 2*slot+1
        {
            double b1, b2;
            block_sum_df2<kTvThreads>(d_tv, d_nn, red, &b1, &b2);
            if (threadIdx.x == 0) {
                P.partial[(size_t)(4 + 2 * slot) * nb + local] = b1;
                P.partial[(size_t)(5 + 2 * slot) * nb + local] = b2;
            }
            ok = coop_barrier(P.bar, nb + P.bar_extra, &sc->status, &flag, P.wait_limit);
            if (!ok) break;
            block_sum_array2<kTvThreads>(P.partial + (size_t)(4 + 2 * slot) * nb, P.partial + (size_t)(5 + 2 * slot) * nb,
                                         nb, red, &s_tv, &s_nn);
            slot ^= 1;
        }
        const double tv_y = s_tv;
        if (step == 0) tv_first = tv_y;
        // the step scalars are the same in every thread: thread 0 evaluates the FP64
        // functions and the block reads the result (the FP64 pipe is narrow)
        if (threadIdx.x == 0) sh_inv = (s_nn > 0.0) ? rsqrt_fp64(s_nn) : 0.0;
        long long trials = 0;
        float c = 0.0f;
        double tv_t = 0.0;
        for (;;) {
            if (trials >= max_trials) {
                if (local == 0 && threadIdx.x == 0) atomicExch(&sc->status, (int)SUPCG_ERR_BACKTRACK);
                ok = false;
                break;
            }
            if (threadIdx.x == 0) {
                const double ap = sh_apow_ok ? sh_apow : pow(a, (double)ell);
                sh_c = (float)(gamma * ap * sh_inv);   // gamma a^l / ||tbar||
                sh_apow = ap * a;                      // a^(l + 1), for the next trial
                sh_apow_ok = 1;
            }
            __syncthreads();
            c = sh_c;                                                                     // y~ = y + c tbar
            ++ell;
            ++trials;
            df s = df_make(0.0f);
            for (PixWalk w(e0, stride, nx); w.i < ny;) {
                float yv[kStvGroup][3], lv[kStvGroup][3], tv[kStvGroup][3];
                bool in[kStvGroup];
#pragma unroll
                for (int q = 0; q < kStvGroup; ++q) {
                    in[q] = w.i + 1 < ny && w.j + 1 < nx;
                    if (in[q]) {
                        const size_t p = (size_t)w.i * ld + w.j;
                        yv[q][0] = x[p];
                        yv[q][1] = x[p + ld];
                        yv[q][2] = x[p + 1];
                        tv[q][0] = tb[p];
                        tv[q][1] = tb[p + ld];
                        tv[q][2] = tb[p + 1];
                        if (xl) {
                            lv[q][0] = xl[p];
                            lv[q][1] = xl[p + ld];
                            lv[q][2] = xl[p + 1];
                        }
                    }
                    w.next();
                }
#pragma unroll
                for (int q = 0; q < kStvGroup; ++q) {
                    if (in[q]) {   // the root of the TV term of y~ = y + c tbar based at the pixel
                        float y3[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) y3[k] = step_value(yv[q][k], xl ? lv[q][k] : 0.0f, xl != nullptr, c, tv[q][k]);
                        df_acc(s, root(y3[0] - y3[1], y3[0] - y3[2]));
                    }
                }
            }
            tv_t = phase_sum(P, nb, slot, local, s, red, &flag, &ok);
            slot ^= 1;
            if (!ok) break;
            if (tv_t <= tv_y) break;   // until TV(y~) <= TV(y)
        }
        total_trials += trials;
        if (!ok) break;
        if (trials_out && local == 0 && threadIdx.x == 0) trials_out[(size_t)pi * K + step] = (int)trials;
        if (step == K - 1 && !want_snorm) {   // the last step, with d
            write_d(true, false, c);
            d_done = true;
        } else {
            for (PixWalk w(e0, stride, nx); w.i < ny;) {   // y <- y~
                size_t gp[kStvGroup];
                float tv[kStvGroup];
#pragma unroll
                for (int q = 0; q < kStvGroup; ++q) {
                    gp[q] = (w.i < ny) ? (size_t)w.i * ld + w.j : ~(size_t)0;
                    if (w.i < ny) tv[q] = tb[gp[q]];
                    w.next();
                }
#pragma unroll
                for (int q = 0; q < kStvGroup; ++q)
                    if (gp[q] != ~(size_t)0) (void)x_step(x, xl, gp[q], c, tv[q]);
            }
            ok = coop_barrier(P.bar, nb + P.bar_extra, &sc->status, &flag, P.wait_limit);
        }
        tv_last = tv_t;
    }
    double sn = 0.0;
    if (ok && want_snorm) {
        double s = 0.0;
        for (int e = e0; e < n; e += stride) {
            const int i = e / nx, j = e - i * nx;
            const size_t p = (size_t)i * ld + j;
            const double dlt = ((double)x[p] - (double)P.z[p]) + ((xl ? (double)xl[p] : 0.0) - (double)P.g[p]);
            s += dlt * dlt;
        }
        sn = phase_sum(P, nb, slot, local, s, red, &flag, &ok);
    }
    if (local == 0 && threadIdx.x == 0) {
        sc->ell = ell;
        sc->apow = sh_apow;
        sc->apow_a = a;
        sc->apow_ell = ell;
        sc->apow_ok = sh_apow_ok;
        sc->trials = total_trials;
        sc->tv_k = tv_first;
        sc->tv_half = (K > 0) ? tv_last : tv_first;
        sc->snorm2 = sn;
    }
    // d, unless the last step wrote it (after the last barrier every block sees the final x);
    // no step ran when the plain loop had none (K = 0), and then no barrier either
    if (ok && !d_done) write_d(false, plain && K == 0, 0.0f);
}

// ------------------------------------------------------------ S_TV on resident tiles
// S_TV with every problem's image held on the chip, a tile of TI x 32 pixels per block:
// one grid barrier per trial.  In memory (k_stv) a step took three barriers with a pass
// over the image each, 20 us at 512^2, of which the arithmetic is about one; what counts
// is the number of barriers and of L2 round trips between them.  Here a trial forms
// y~ = y + c tbar itself (the pair (x, xlo), as the accepted step does) and, before the
// barrier that sums TV(y~), also tbar(y~) and its norm: if y~ is accepted, the next step
// starts at once.
//   A block holds y on its tile and one ring around it, and tbar of y there (its own
// pixels' and one ring pixel's per thread, in registers), so it has y~ on both and
// TV(y~), tbar(y~) on the tile.  tbar(y~) of the ring comes from the neighbours: each
// block publishes its outermost rows and columns before the barrier and reads the ring
// after it, together with the partial sums.  A ring pixel of y~ is computed by two
// blocks, from the same values in the same order, bit for bit alike.  The published
// values alternate between two buffers (z and g, free until the next gradient), since a
// block may still be reading one trial's while another writes the next one's.  x is
// written only at the end.
//   A TV term's roots and quotients are computed once, at its base pixel, and meet the
// pixels below and to the right of it in shared memory.  A pixel's values (y~, its
// term, tbar) are those of k_stv bit for bit: which kernel a problem takes depends on
// the other problems of its launch.  The two add up the same terms in another order.
// Measured, K = 40 at 512^2 (one call): 853 -> 338 us, 8.4 us per step; a grid barrier is
// about 1.4 us of it, the FP64 sum over the blocks' partials 1 us, and the rest some eight block
// barriers with the short passes between them.
constexpr int kStvThreads = 512, kStvWarps = kStvThreads / 32;

template <int TI>
struct StvTile {
    static constexpr int H = TI + 2, W = 34, LD = 35;       // the tile and its ring; odd pitch
    static constexpr int PX = TI / kStvWarps;               // pixels per thread
    static constexpr int RING = 2 * W + 2 * TI;             // pixels of the ring
    static_assert(RING <= kStvThreads - 64, "one ring pixel per thread, the first two warps left out");
    float hi[2][H * LD], lo[2][H * LD];                     // y and y~ (high and low parts), in turn
    float qa[H * LD], qb[H * LD];                           // a / T and b / T of the TV term based at the pixel
};
constexpr float kUndef = 4.0f;   // qa, qb of a term whose differences are both 0 (|a / T| <= 1 otherwise)

// Pixel k of the ring around the tile, in the coordinates of the held region.
template <int TI>
__device__ __forceinline__ void stv_ring(int k, int &i, int &j)
{
    using S = StvTile<TI>;
    if (k < S::W) { i = 0; j = k; return; }
    k -= S::W;
    if (k < S::W) { i = TI + 1; j = k; return; }
    k -= S::W;
    i = 1 + (k >> 1);
    j = (k & 1) ? S::W - 1 : 0;
}

// The step scalars of one thread.  An FP64 instruction holds the SM's FP64 pipe for about 38 cycles per warp
// that issues it; inlined, these were turned into predicated code that every warp issued (350 FP64
// instructions per step and block, the pipe 85 % busy: a quarter longer for 40 steps at 512^2).
struct StvScalars {
    double apow, gap;   // a^l (Scal::apow), gamma a^l
    float gh, gl;       // gamma a^l as two FP32 parts
};
__device__ __noinline__ void stv_set_pow(StvScalars *s, double apow, double gamma)
{
    s->apow = apow;
    s->gap = gamma * apow;
    s->gh = (float)s->gap;
    s->gl = (float)(s->gap - (double)s->gh);
}
// gamma a^l / sqrt(nn) rounded to FP32 (0 for nn = 0): on the FP32 pipe, within 2^-44 before the last rounding;
// in FP64, as k_stv has it, outside FP32's range and where an error of that size could turn the last rounding
// (one step in 2^17).
__device__ __noinline__ float stv_step(const StvScalars *s, double nn)
{
    if (!(nn > 0.0)) return 0.0f;
    const float nh = (float)nn, gh = s->gh;
    if (nh > 1e-30f && nh < 1e30f && gh > 1e-25f && gh < 1e25f) {
        const float nl = (float)(nn - (double)nh);
        const float y = rsqrtf(nh);
        const df m = df_mul(df{nh, nl}, df_prod(y, y));
        const float e = __fsub_rn(__fsub_rn(1.0f, m.h), m.l);                          // 1 - nn y^2
        const float yl = __fmul_rn(y, __fmaf_rn(__fmul_rn(0.375f, e), e, 0.5f * e));   // 1 / sqrt(nn) = y + yl
        const df p = df_prod(gh, y);
        const float tail = __fadd_rn(p.l, __fmaf_rn(gh, yl, __fmul_rn(s->gl, y)));
        const float c = __fadd_rn(p.h, tail);
        // What c leaves of the sum, exactly: were it 2^-17 of itself more, would c be the same?  (Half a unit of c
        // is 2^-25 c or more, and 2^-17 of it four times the error.)
        const float rest = __fadd_rn(__fsub_rn(p.h, c), tail);
        if (p.h > 1e-20f && p.h < 1e30f && __fadd_rn(c, __fmul_rn(rest, 1.0f + 0x1p-17f)) == c) return c;
    }
    return (float)(s->gap * rsqrt_fp64(nn));
}
__device__ __noinline__ void stv_first_pow(StvScalars *s, const Scal *sc, double a, double gamma)
{
    const bool carried = sc->apow_ok && sc->apow_ell == sc->ell && sc->apow_a == a;
    stv_set_pow(s, carried ? sc->apow : pow(a, (double)sc->ell), gamma);
}
__device__ __noinline__ void stv_next_pow(StvScalars *s, double a, double gamma) { stv_set_pow(s, s->apow * a, gamma); }
// u <= v for sums of roots (>= 0, or NaN: false), on the integer pipe.
__device__ __forceinline__ bool sum_le(double u, double v)
{
    const unsigned long long a = (unsigned long long)__double_as_longlong(u), b = (unsigned long long)__double_as_longlong(v);
    return a <= b && a <= 0x7FF0000000000000ull;
}

template <int TI>
__global__ void __launch_bounds__(kStvThreads, 2) k_stv_tile(const Prob *__restrict__ probs, const int *__restrict__ prefix,
                                                             int count, int K_arg, double a_arg, double gamma_arg,
                                                             long long max_trials, int *trials_out, int want_snorm)
{
    using S = StvTile<TI>;
    constexpr int LD = S::LD, PX = S::PX;
    extern __shared__ __align__(16) unsigned char stv_raw[];
    S &sm = *reinterpret_cast<S *>(stv_raw);
    __shared__ __align__(16) double red[40];
    __shared__ double sh_tot[2];
    __shared__ float sh_c;
    __shared__ int flag;
    int local;
    const int pi = find_problem(prefix, count, blockIdx.x, &local);
    const Prob &P = probs[pi];
    Scal *sc = P.sc;
    if (sc->done) return;
    const int K = P.stv_own ? P.stv_K : K_arg;
    const double a = P.stv_own ? P.stv_a : a_arg, gamma = P.stv_own ? P.stv_gamma : gamma_arg;
    const int nb = prefix[pi + 1] - prefix[pi];
    const int nx = P.nx, ny = P.ny, ld = P.nxp;
    const int tiles_j = (nx + 31) / 32;
    const int ti = local / tiles_j, i0 = ti * TI, j0 = (local - ti * tiles_j) * 32;
    const int t = threadIdx.x, tx = t & 31, ty = t >> 5, lane = tx;
    const bool has_lo = P.xlo != nullptr;
    // the step scalars live in the first thread of the last warp, whose FP64 work runs beside the other warps'
    const bool scalars = t == kStvThreads - 32;
    GridCount bar(P.bar + 2, nb + P.bar_extra);
    long long ell = sc->ell;
    __shared__ StvScalars sh_sc;
    if (scalars) stv_first_pow(&sh_sc, sc, a, gamma);
    // y on the tile and its ring (0 off the image: no formula below uses it)
    int cur = 0;
    for (int e = t; e < S::H * S::W; e += kStvThreads) {
        const int ri = e / S::W, rj = e - ri * S::W, i = i0 + ri - 1, j = j0 + rj - 1;
        const bool in = i >= 0 && i < ny && j >= 0 && j < nx;
        const size_t p = in ? (size_t)i * ld + j : 0;
        sm.hi[0][ri * LD + rj] = in ? P.x[p] : 0.0f;
        sm.lo[0][ri * LD + rj] = (in && has_lo) ? P.xlo[p] : 0.0f;
    }
    // this thread's ring pixel
    int rk = 0;
    size_t rp = 0;
    bool ring = false;
    if (t >= 64 && t - 64 < S::RING) {
        int ri, rj;
        stv_ring<TI>(t - 64, ri, rj);
        const int i = i0 + ri - 1, j = j0 + rj - 1;
        rk = ri * LD + rj;
        ring = i >= 0 && i < ny && j >= 0 && j < nx;
        if (ring) rp = (size_t)i * ld + j;
    }
    __syncthreads();
    // The tile's part of TV and (want_t) of ||tbar||^2 of buffer y, tbar into tn and its outermost rows and
    // columns published; the block's sums into its partial of `slot`.
    float tn[PX];
    auto tile_sums = [&](const float *y, bool want_t, int slot) {
        df d_tv = df_make(0.0f), d_nn = df_make(0.0f);
        float qs[PX];   // (a + b) / T of the own terms
        // a term's root, and its quotients into qa, qb
        auto term = [&](int q, bool exists, float *sum_q) {
            float T = 0.0f, va = 0.0f, vb = 0.0f, vs = 0.0f;
            if (exists) {
                const float yc = y[q], a1 = yc - y[q + LD], b1 = yc - y[q + 1];
                if (a1 == 0.0f && b1 == 0.0f) {
                    va = vb = vs = kUndef;
                } else {
                    const float Tl = root_b(a1, b1);
                    T = root(a1, b1);
                    va = __fdiv_rn(a1, T);
                    vb = __fdiv_rn(b1, Tl);
                    vs = __fdiv_rn(__fadd_rn(a1, b1), T);
                }
            }
            sm.qa[q] = va;
            sm.qb[q] = vb;
            *sum_q = vs;
            return T;
        };
        if (want_t) {
#pragma unroll
            for (int q = 0; q < PX; ++q) {
                const int r = ty + kStvWarps * q, i = i0 + r, j = j0 + tx;
                df_acc(d_tv, term((r + 1) * LD + tx + 1, i + 1 < ny && j + 1 < nx, &qs[q]));
            }
            if (t < 32 + TI) {   // the terms based above the tile and left of it
                const int ri = t < 32 ? 0 : t - 31, rj = t < 32 ? t + 1 : 0, i = i0 + ri - 1, j = j0 + rj - 1;
                float s;
                (void)term(ri * LD + rj, i >= 0 && j >= 0 && i + 1 < ny && j + 1 < nx, &s);
            }
            __syncthreads();
            float *pub = slot ? P.g : P.z;
#pragma unroll
            for (int q = 0; q < PX; ++q) {
                const int r = ty + kStvWarps * q, i = i0 + r, j = j0 + tx;
                const float up = sm.qa[r * LD + tx + 1], le = sm.qb[(r + 1) * LD + tx];
                const bool undef = qs[q] == kUndef || up == kUndef || le == kUndef;
                const float g = __fsub_rn(__fsub_rn(qs[q], up), le);
                tn[q] = (undef || i >= ny || j >= nx) ? 0.0f : -g;
                df_acc_prod(d_nn, tn[q], tn[q]);
                if (i < ny && j < nx && (r == 0 || r == TI - 1 || tx == 0 || tx == 31)) pub[(size_t)i * ld + j] = tn[q];
            }
        } else {
#pragma unroll
            for (int q = 0; q < PX; ++q) {
                const int r = ty + kStvWarps * q, e = (r + 1) * LD + tx + 1;
                if (i0 + r + 1 < ny && j0 + tx + 1 < nx) {
                    const float a1 = y[e] - y[e + LD], b1 = y[e] - y[e + 1];
                    df_acc(d_tv, root(a1, b1));
                }
            }
        }
        double b1, b2;
        block_sum_df2<kStvThreads>(d_tv, d_nn, red, &b1, &b2);
        if (t == 0) reinterpret_cast<double2 *>(P.partial)[(size_t)slot * nb + local] = make_double2(b1, b2);
    };
    // the sums of all blocks, in the same order in each: TV by warp 0, ||tbar||^2 by warp 1 (an FP64 add holds
    // a quarter of the SM's narrow FP64 pipe for many cycles, so the two chains run on different quarters)
    auto totals = [&](int slot) {
        const double *pp = P.partial + (size_t)slot * 2 * nb + ty;
        double v = 0.0;
        for (int b = lane; b < nb; b += 32 * 8) {
            double u[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) u[k] = b + 32 * k < nb ? __ldcg(pp + 2 * (b + 32 * k)) : 0.0;
            v += ((u[0] + u[1]) + (u[2] + u[3])) + ((u[4] + u[5]) + (u[6] + u[7]));
        }
        v = warp_sum(v);
        if (lane == 0) sh_tot[ty] = v;
    };
    // the barrier after tile_sums, then the totals; tbar of the ring pixel meanwhile
    float rt = 0.0f, rn = 0.0f;   // tbar of this thread's ring pixel: of y, of y~
    auto meet = [&](int slot, bool want_t) {
        bar.arrive();
        if (!bar.wait<false>(P.wait_limit, &sc->status, &flag)) return false;
        if (ty < 2) totals(slot);
        else if (want_t && ring) rn = __ldcg((slot ? P.g : P.z) + rp);
        __syncthreads();
        return true;
    };
    int slot = 0;
    bool ok = true, timed_out = false;
    long long total_trials = 0;
    float c = 0.0f, tc[PX];       // tc: tbar of y on the tile
    tile_sums(sm.hi[0], true, slot);
    if (!meet(slot, true)) return;
    const double tv_first = sh_tot[0];
    double tv_y = tv_first, tv_half = 0.0;   // TV of y; of the last accepted y~
    for (int step = 0; step < K && ok; ++step) {
        // y is the last accepted image (buffer cur), its tbar in tn and rn, TV and ||tbar||^2 in sh_tot
        const float *yh = sm.hi[cur], *yl = sm.lo[cur];
        float *zh = sm.hi[cur ^ 1], *zl = sm.lo[cur ^ 1];
#pragma unroll
        for (int q = 0; q < PX; ++q) tc[q] = tn[q];
        rt = rn;
        const double nn = sh_tot[1];
        const bool last = step == K - 1;
        long long trials = 0;
        for (;;) {
            if (trials >= max_trials) {
                if (local == 0 && t == 0) atomicExch(&sc->status, (int)SUPCG_ERR_BACKTRACK);
                ok = false;
                break;
            }
            if (scalars) sh_c = stv_step(&sh_sc, nn);   // gamma a^l / ||tbar||
            __syncthreads();
            c = sh_c;   // y~ = y + c tbar
            ++ell;
            ++trials;
            if (scalars) stv_next_pow(&sh_sc, a, gamma);   // for the next trial: a^(l + 1)
            auto move = [&](int q, float tq) {
                if (has_lo) {
                    const df v = df_add(df{yh[q], yl[q]}, df_prod(c, tq));
                    zh[q] = v.h;
                    zl[q] = v.l;
                } else {
                    zh[q] = __fmaf_rn(c, tq, yh[q]);
                }
            };
#pragma unroll
            for (int q = 0; q < PX; ++q) move((ty + kStvWarps * q + 1) * LD + tx + 1, tc[q]);
            if (ring) move(rk, rt);
            __syncthreads();
            slot ^= 1;
            tile_sums(zh, !last, slot);
            if (!meet(slot, !last)) {
                ok = false;
                timed_out = true;
                break;
            }
            if (sum_le(sh_tot[0], tv_y)) break;   // until TV(y~) <= TV(y); else y and its tbar stay
        }
        total_trials += trials;
        if (!ok) break;
        if (trials_out && local == 0 && t == 0) trials_out[(size_t)pi * K + step] = (int)trials;
        cur ^= 1;
        tv_y = tv_half = sh_tot[0];
    }
    const float *yh = sm.hi[cur], *yl = sm.lo[cur];
    __syncthreads();
    // ||s_k||^2 for the log, from the image before the steps (still in x)
    double sn = 0.0;
    if (ok && want_snorm) {
        double s = 0.0;
#pragma unroll
        for (int q = 0; q < PX; ++q) {
            const int r = ty + kStvWarps * q, i = i0 + r, j = j0 + tx;
            if (i < ny && j < nx) {
                const size_t p = (size_t)i * ld + j;
                const int e = (r + 1) * LD + tx + 1;
                const double dlt = ((double)yh[e] - (double)P.x[p]) + (has_lo ? (double)yl[e] - (double)P.xlo[p] : 0.0);
                s += dlt * dlt;
            }
        }
        s = block_sum<kStvThreads>(s, red);
        slot ^= 1;
        if (t == 0) reinterpret_cast<double2 *>(P.partial)[(size_t)slot * nb + local] = make_double2(s, 0.0);
        timed_out = !meet(slot, false);
        ok = !timed_out;
        sn = sh_tot[0];
    }
    if (local == 0 && scalars) {
        sc->ell = ell;
        sc->apow = sh_sc.apow;
        sc->apow_a = a;
        sc->apow_ell = ell;
        sc->apow_ok = 1;
        sc->trials = total_trials;
        sc->tv_k = tv_first;
        sc->tv_half = tv_half;
        sc->snorm2 = sn;
    }
    if (timed_out) return;
    // x and, after K steps, the displacement d in the projector's layouts; with one plain step d is c tbar
    // itself (the low part of x would not show in it), else the difference from the image before the steps
    const bool plain1 = K == 1 && !want_snorm;
    float *tr = sm.qa;   // the transpose of d, TI x 33
    float dv[PX];
#pragma unroll
    for (int q = 0; q < PX; ++q) {
        const int r = ty + kStvWarps * q, i = i0 + r, j = j0 + tx;
        dv[q] = 0.0f;
        if (i < ny && j < nx) {
            const size_t p = (size_t)i * ld + j;
            const int e = (r + 1) * LD + tx + 1;
            if (plain1) dv[q] = __fmul_rn(c, tc[q]);
            else dv[q] = __fadd_rn(__fsub_rn(yh[e], P.x[p]), has_lo ? __fsub_rn(yl[e], P.xlo[p]) : 0.0f);
            P.x[p] = yh[e];
            if (has_lo) P.xlo[p] = yl[e];
            if (ok) {
                P.d[p] = dv[q];
                if (P.dm) P.dm[(size_t)i * ld + (nx - 1 - j)] = dv[q];
            }
        }
    }
    if (!ok) return;
#pragma unroll
    for (int q = 0; q < PX; ++q) tr[(ty + kStvWarps * q) * 33 + tx] = dv[q];
    __syncthreads();
    for (int e = t; e < 32 * TI; e += kStvThreads) {   // consecutive threads on consecutive rows of the image
        const int cc = e / TI, r = e - cc * TI;
        const int i = i0 + r, j = j0 + cc;
        if (i < ny && j < nx) {
            P.dT[(size_t)j * P.nyp + i] = tr[r * 33 + cc];
            if (P.dmT) P.dmT[(size_t)(nx - 1 - j) * P.nyp + i] = tr[r * 33 + cc];
        }
    }
}

int stv_tiles(int nx, int ny, int ti) { return ((ny + ti - 1) / ti) * ((nx + 31) / 32); }

template <int TI>
static int stv_tile_blocks_t(int *out)
{
    int rc = func_attrs_once((const void *)k_stv_tile<TI>, (int)sizeof(StvTile<TI>), (int)cudaSharedmemCarveoutMaxShared);
    if (rc) return rc;
    return resident_blocks((const void *)k_stv_tile<TI>, kStvThreads, sizeof(StvTile<TI>), out);
}
int stv_tile_max_blocks(int ti, int *out)
{
    return ti == 32 ? stv_tile_blocks_t<32>(out) : (ti == 64 ? stv_tile_blocks_t<64>(out) : stv_tile_blocks_t<128>(out));
}

template <int TI>
static int launch_stv_tile_t(const Launch &L, int K, double a, double gamma, long long max_trials, int *trials_out,
                             int want_snorm)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.blocks);
    cfg.blockDim = dim3(kStvThreads);
    cfg.dynamicSmemBytes = sizeof(StvTile<TI>);
    cfg.stream = L.st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SUPCG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_stv_tile<TI>, L.probs, L.prefix, L.count, K, a, gamma, max_trials, trials_out,
                                      want_snorm));
    return SUPCG_OK;
}
int launch_stv_tile(const Launch &L, int ti, int K, double a, double gamma, long long max_trials, int *trials_out,
                    int want_snorm)
{
    if (ti == 32) return launch_stv_tile_t<32>(L, K, a, gamma, max_trials, trials_out, want_snorm);
    if (ti == 64) return launch_stv_tile_t<64>(L, K, a, gamma, max_trials, trials_out, want_snorm);
    return launch_stv_tile_t<128>(L, K, a, gamma, max_trials, trials_out, want_snorm);
}

int stv_max_blocks(int *out) { return resident_blocks((const void *)k_stv, kTvThreads, 0, out); }

int launch_stv(const Launch &L, int K, double a, double gamma, long long max_trials, int *trials_out,
               int want_snorm, const float *dir)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.blocks);
    cfg.blockDim = dim3(kTvThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = L.st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SUPCG_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_stv, L.probs, L.prefix, L.count, K, a, gamma, max_trials,
                                      trials_out, want_snorm, dir));
    return SUPCG_OK;
}

} // namespace supcg
