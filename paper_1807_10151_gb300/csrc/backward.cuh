// What the two backprojector kernels share: the thread layout, and the end of a block (its part's sums,
// the tile's last part adding them, the outputs and the sums over the image).
#pragma once

#include "internal.cuh"

namespace supcg {

constexpr int kBwdSplit = 2;                                             // thread groups splitting the views
constexpr int kBwdGroup = 128;                                           // threads per group
constexpr int kBwdThreads = kBwdSplit * kBwdGroup;
constexpr int kBwdRowStep = kBwdGroup / kBwdTileJ;                       // 4

// part, comp [s * PX + e]: this thread group's Kahan pair of pixel e for sinogram s (value part - comp, |comp| <=
// ulp(part) / 2); at(e, &i, &j): the pixel, false where it is not stored.  The groups' and the parts' sums are
// added in double-float arithmetic, in a fixed order.
template <bool DUAL, int PX, class At>
__device__ __forceinline__ void bwd_finish(const Prob &P, int ntiles, int pi, int mode, const Io &io, int parts, int vpart,
                                           int tile, int grp, int tg, bool bad, const float *part, const float *comp,
                                           float2 *comb, double *red, int *bad_sh, int *last_sh, At at)
{
    constexpr int NS = DUAL ? 2 : 1;
    const int t = threadIdx.x;
    if (bad) atomicExch(bad_sh, 1);
    __syncthreads();
    if (grp == 1)
#pragma unroll
        for (int e = 0; e < NS * PX; ++e) comb[e * kBwdGroup + tg] = make_float2(part[e], -comp[e]);
    __syncthreads();
    // this part's sums; the tile's last part to finish adds them in part order
    const size_t img = (size_t)P.ny * P.nxp;
    if (grp == 0)
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int e = 0; e < PX; ++e) {
                int i, j;
                if (at(e, &i, &j)) {
                    const float2 o2 = comb[(s * PX + e) * kBwdGroup + tg];
                    const df v = df_add(df{part[s * PX + e], -comp[s * PX + e]}, df{o2.x, o2.y});
                    P.bsplit[(size_t)(s * parts + vpart) * img + (size_t)i * P.nxp + j] = make_float2(v.h, v.l);
                }
            }
    if (t == 0 && *bad_sh && P.sc) atomicExch(&P.sc->status, (int)SUPCG_ERR_UNSUPPORTED);
    if (!last_block(&P.tilecnt[tile], parts, last_sh)) return;
    // output s: 0 the gradient (g from r), 1 h from q
    // Bayesian criterion (Eq. (2.3)): g = r^2 R^T r + (x - mu_X), h = r^2 R^T q + p, and
    // ||x - mu_X||^2 for f.  With a reference image, the selective error of Eq. (4.1) of
    // x = x_{k+1/2} over the centred ellipse S (this pass reads x anyway).
    const bool solve = DUAL || mode != BWD_PLAIN;
    const bool bayes = solve && P.r2 > 0.0;
    const bool want_se = (DUAL || mode == BWD_G) && P.se_ref != nullptr && !P.sc->init;
    const double muX = bayes ? P.sc->muX : 0.0;
    double sx = 0.0, sse = 0.0;
    if (grp == 0)
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int e = 0; e < PX; ++e) {
                int i, j;
                if (at(e, &i, &j)) {
                    const size_t o = (size_t)i * P.nxp + j;
                    float2 pv[kBwdMaxParts];   // the other blocks' sums: read past L1
#pragma unroll
                    for (int h = 0; h < kBwdMaxParts; ++h)
                        if (h < parts) pv[h] = __ldcg(P.bsplit + (size_t)(s * parts + h) * img + o);
                    df vs = {0.0f, 0.0f};
#pragma unroll
                    for (int h = 0; h < kBwdMaxParts; ++h)
                        if (h < parts) vs = df_add(vs, df{pv[h].x, pv[h].y});
                    float *out = s ? P.h : P.g;
                    if (bayes) {
                        double v = (double)vs.h + (double)vs.l;
                        if (s == 0) {
                            const double dx = (double)P.x[o] - muX;
                            v = P.r2 * v + dx;
                            sx += dx * dx;
                        } else {
                            v = P.r2 * v + (double)P.p[o];
                        }
                        const float vh = (float)v;
                        out[o] = vh;
                        if (solve && s == 0) P.glo[o] = (float)(v - (double)vh);
                    } else {
                        const float vh = __fadd_rn(vs.h, vs.l);   // the pair rounded to FP32
                        if (solve || !io.out) {
                            out[o] = vh;
                        } else {   // the caller's image
                            void *user = io.out + (size_t)pi * io.out_step;
                            const size_t oc = (size_t)i * P.nx + j;
                            if (io.storage == SUPCG_BF16) reinterpret_cast<__nv_bfloat16 *>(user)[oc] = __float2bfloat16_rn(vh);
                            else reinterpret_cast<float *>(user)[oc] = vh;
                        }
                        if (solve && s == 0) P.glo[o] = __fsub_rn(vs.l, __fsub_rn(vh, vs.h));   // its error, exactly
                    }
                    if (want_se && s == 0) {   // pixel centre inside the ellipse (FP64, as the definition)
                        const double ex = ((double)j - 0.5 * (P.nx - 1)) / P.se_ax;
                        const double ey = ((double)i - 0.5 * (P.ny - 1)) / P.se_ay;
                        if (ex * ex + ey * ey <= 1.0) {
                            const double dr = (double)P.x[o] - (double)P.se_ref[(size_t)i * P.nx + j];
                            sse += dr * dr;
                        }
                    }
                }
            }
    if (t == 0) P.tilecnt[tile] = 0;   // ready for the next launch
    if (!bayes && !want_se) return;
    // the tiles' sums, added in tile order by the last tile to finish: f = r^2 ||R x - b||^2 +
    // ||x - mu_X||^2, and SE = sqrt(sum over S)
    const double bs = block_sum<kBwdThreads>(sx, red);
    const double be = block_sum<kBwdThreads>(sse, red);
    if (t == 0) {
        P.partial[tile] = bs;
        P.partial[ntiles + tile] = be;
    }
    if (last_block(&P.counter[4], ntiles, last_sh)) {
        double tot, tse;
        block_sum_array2<kBwdThreads>(P.partial, P.partial + ntiles, ntiles, red, &tot, &tse);
        if (t == 0) {
            Scal *sc = P.sc;
            if (bayes) {
                sc->f = P.r2 * sc->f_ls + tot;
                if (sc->init) sc->f0 = sc->f;
            }
            if (want_se) P.se_log[sc->k] = sqrt(tse);   // body sc->k + 1 (k counts finished bodies)
            P.counter[4] = 0;
        }
    }
}

} // namespace supcg
