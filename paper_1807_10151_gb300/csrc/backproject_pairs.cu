// R^T y for geometries whose views come in mirror pairs (theta, pi - theta): pixel (X, Y) meets a bin of
// view v at the same distance as pixel (-X, Y) meets that bin of the mirror view w, so one weight serves
// both.  A tile is TI x 32 pixels and the same pixels mirrored left to right; each thread owns rows of a
// column and of its mirror column, and an item of the view list is a pair (v, w).  For each of the item's
// two bin ranges (those that the tile's left and right side meet under v) the window in shared memory holds
// the values of v and w side by side, for both sinograms where there are two, so that a candidate's weight,
// evaluated once, takes all it multiplies with one vector load: own side += weight x v, other side +=
// weight x w.
//
// Two sinograms over 512^2 / 720 views: 219 -> 161 us and 170 M -> 99 M warp instructions against the general
// kernel (backprojector.cu), which evaluates every weight twice; one sinogram 166 -> 119 us, eight images of
// 243^2 / 360 views 168 -> 126.  What is left is latency: 49 % of the issue slots are used, the l1tex data
// path is 60 % busy, no pipe is above 33 %, and two blocks per SM (128 registers) are all that fit.
#include "backward.cuh"

namespace supcg {

extern __shared__ __align__(128) float proj_dyn[];

constexpr int kPairChunk = 16;   // items per staged chunk (32 views)

template <bool DUAL>
struct PairAcc;                  // one pixel's running sum: of sinogram (r, q), or of the only one
template <> struct PairAcc<true> { typedef uint64_t T; };
template <> struct PairAcc<false> { typedef float T; };

// own += w y.v, oth += w y.w for the window element at index i: (v of r, v of q, w of r, w of q) or (v, w)
template <bool DUAL>
__device__ __forceinline__ void pair_add(float w, int i, typename PairAcc<DUAL>::T &own, typename PairAcc<DUAL>::T &oth)
{
    if constexpr (DUAL) {
        const float4 y = reinterpret_cast<const float4 *>(proj_dyn)[i];
        const uint64_t w2 = pk2(w, w);
        own = fma2_rn(w2, pk2(y.x, y.y), own);
        oth = fma2_rn(w2, pk2(y.z, y.w), oth);
    } else {
        const float2 y = reinterpret_cast<const float2 *>(proj_dyn)[i];
        own = __fmaf_rn(w, y.x, own);
        oth = __fmaf_rn(w, y.y, oth);
    }
}

// One item, both sides of each row in the two halves of an f32x2: the candidates and weights of the general
// kernel's bwd_view_x2 (the same FP32 steps), for windows that hold every candidate.  X2 = (X, -X), Y: the
// rows; win: each side's first window element minus its first bin.
template <bool DUAL, int NC, int PXR>
__device__ __forceinline__ void pair_x2(const ViewP &vp, uint64_t X2, const float *Y, float uc_hi, float uc_lo,
                                        const int *win, typename PairAcc<DUAL>::T *acc)
{
    const float E = vp.E, Sn = vp.Sn, ESn = vp.ESn;
    const uint64_t su2 = pk2(vp.su_hi, vp.su_hi), hwu2 = pk2(vp.hwu, vp.hwu), mag2 = pk2(kCeilMagic, kCeilMagic);
    const float b0 = __fmaf_rn(-vp.su_hi, Y[0], -uc_hi);
    const uint64_t pbb = fma2_rn(pk2(-vp.cu_hi, -vp.cu_hi), X2, pk2(b0, b0));
    // small = uc_lo + cu_lo X + su_lo Y in the view class's order (delta_small)
    const uint64_t c2 = pk2(vp.cu_lo, vp.cu_lo);
    uint64_t sm2[PXR];
    if (vp.flags & kViewClassB) {
        const uint64_t in2 = fma2_rn(c2, X2, pk2(uc_lo, uc_lo)), s2 = pk2(vp.su_lo, vp.su_lo);
#pragma unroll
        for (int e = 0; e < PXR; ++e) sm2[e] = fma2_rn(s2, pk2(Y[e], Y[e]), in2);
    } else {
#pragma unroll
        for (int e = 0; e < PXR; ++e) {
            const float in = __fmaf_rn(vp.su_lo, Y[e], uc_lo);
            sm2[e] = fma2_rn(c2, X2, pk2(in, in));
        }
    }
#pragma unroll
    for (int e = 0; e < PXR; ++e) {
        const uint64_t pb = fma2_rn(pk2((float)(kBwdRowStep * e), (float)(kBwdRowStep * e)), su2, pbb);   // exact
        const uint64_t uc = add2_rp(sub2_rn(sub2_rn(sm2[e], pb), hwu2), mag2);
        float ul, ur;
        upk2(uc, ul, ur);
        const int il = win[0] + magic_int(ul), ir = win[1] + magic_int(ur);
        const uint64_t big0 = add2_rn(sub2_rn(uc, mag2), pb);              // exact, as are big0 + 1, + 2
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const uint64_t bk = k ? add2_rn(big0, pk2((float)k, (float)k)) : big0;
            float dl, dr;
            upk2(sub2_rn(bk, sm2[e]), dl, dr);
            pair_add<DUAL>(weight_unit(fabsf(dl), E, Sn, ESn, false), il + k, acc[e], acc[PXR + e]);
            pair_add<DUAL>(weight_unit(fabsf(dr), E, Sn, ESn, false), ir + k, acc[PXR + e], acc[e]);
        }
    }
}

// The same pixel by pixel, with a check of the window (axis-aligned views, and windows that may miss a
// candidate); vp in shared memory, so that its registers are not kept for this rare path.
template <bool DUAL, bool AXIS, int NC, int PXR>
__device__ __noinline__ int pair_checked(const ViewP *vp, float X, float Y0, float uc_hi, float uc_lo, const int *lo,
                                         int win0, int bw, typename PairAcc<DUAL>::T *acc)
{
    int bad = 0;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const float Xs = s ? -X : X;
        const float pb0 = __fmaf_rn(-vp->cu_hi, Xs, __fmaf_rn(-vp->su_hi, Y0, -uc_hi));
#pragma unroll
        for (int e = 0; e < PXR; ++e) {
            const float sm = delta_small(*vp, Xs, __fsub_rn(Y0, (float)(kBwdRowStep * e)), uc_lo);
            const float pb = __fmaf_rn((float)(kBwdRowStep * e), vp->su_hi, pb0);
            int u0 = magic_int(ceil_magic(__fsub_rn(__fsub_rn(sm, pb), vp->hwu))) - lo[s];
            if (u0 < 0 || u0 > bw - NC) {   // outside the staged window: never for a valid window
                bad = 1;
                u0 = min(max(u0, 0), bw - NC);
            }
            const float big0 = __fadd_rn(__int2float_rn(u0 + lo[s]), pb);
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const float ad = fabsf(__fsub_rn(__fadd_rn(big0, (float)k), sm));
                pair_add<DUAL>(weight_unit(ad, vp->E, vp->Sn, vp->ESn, AXIS), win0 + s * bw + u0 + k, acc[s * PXR + e],
                               acc[(1 - s) * PXR + e]);
            }
        }
    }
    return bad;
}

// Modes as k_backward.  FIXED_PARTS as there; TI: tile rows.
template <bool DUAL, int FIXED_PARTS, int TI>
__global__ void __launch_bounds__(kBwdThreads, DUAL ? 2 : 3) k_backward_pairs(const Prob *__restrict__ probs,
                                                                const int *__restrict__ prefix, int count, int mode,
                                                                Io io)
{
    constexpr int NS = DUAL ? 2 : 1, PXR = TI / kBwdRowStep, PX = 2 * PXR;
    typedef typename PairAcc<DUAL>::T Acc;
    // proj_dyn: [2][kPairChunk][side][bw] window elements of 2 NS floats
    __shared__ ViewP vsh[2][kPairChunk];
    __shared__ int2 item_sh[2][kPairChunk];
    __shared__ int lo_sh[2][kPairChunk][2];
    __shared__ int kind_sh[2][kPairChunk];   // two candidates (0) / three (1), + 2 where a window check is needed; axis 4
    __shared__ float2 comb[kBwdGroup * NS * PX];
    __shared__ __align__(16) double red[40];
    __shared__ int bad_sh, last_sh;

    int local;
    const int pi = find_problem(prefix, count, blockIdx.x, &local);
    const Prob &P = probs[pi];
    if ((DUAL || mode != BWD_PLAIN) && P.sc->done) return;

    const int bw = P.bwp;
    const int nh = (P.nx + 1) / 2;           // columns of the left side; an odd image's middle one is its own mirror
    const int tiles_j = (nh + kBwdTileJ - 1) / kBwdTileJ;
    const int parts = FIXED_PARTS ? FIXED_PARTS : P.bparts;
    const int ntiles = (prefix[pi + 1] - prefix[pi]) / parts;
    const int vpart = local / ntiles, tile = local - vpart * ntiles;   // part-major, as k_backward
    const int ti = tile / tiles_j, tj = tile - ti * tiles_j;
    const int i0 = ti * TI, j0 = tj * kBwdTileJ;
    const int t = threadIdx.x;
    const int grp = t / kBwdGroup, tg = t - grp * kBwdGroup;   // group grp takes items grp (mod kBwdSplit)
    const int j = j0 + tg % kBwdTileJ, ly = tg / kBwdTileJ;
    const float X = __fsub_rn(__int2float_rn(j), P.cx);        // the mirror column's is -X, exactly
    const uint64_t X2 = pk2(X, -X);
    float Y[PXR];
#pragma unroll
    for (int e = 0; e < PXR; ++e) Y[e] = __fsub_rn(P.cy, __int2float_rn(i0 + ly + kBwdRowStep * e));
    const float uc_hi = P.uc_hi, uc_lo = P.uc_lo;
    // per pixel (left side first): FP32 sum of four views, folded into a Kahan pair, as k_backward
    Acc acc[PX];
    uint64_t part2[NS * PX / 2], comp2[NS * PX / 2];
#pragma unroll
    for (int e = 0; e < PX; ++e) acc[e] = 0;   // (the bits of zeros, also as a pair)
#pragma unroll
    for (int h = 0; h < NS * PX / 2; ++h) part2[h] = comp2[h] = pk2(0.0f, 0.0f);

    const float *sino = P.r;
    const void *user = io.in + (size_t)pi * io.in_step;
    const int Up = P.Up;
    // tile corners in pixel-centre coordinates, of the left side
    const float Xa = __fsub_rn(__int2float_rn(j0), P.cx), Xb = __fsub_rn(__int2float_rn(j0 + kBwdTileJ - 1), P.cx);
    const float Ya = __fsub_rn(P.cy, __int2float_rn(i0)), Yb = __fsub_rn(P.cy, __int2float_rn(i0 + TI - 1));
    if (t == 0) bad_sh = 0;

    const int ni = P.nbi;
    const int nchunks = (ni + kPairChunk - 1) / kPairChunk;
    auto stage = [&](int c) {   // chunk c into buffer c & 1
        const int buf = c & 1;
        if (t < 2 * kPairChunk) {   // one warp: an item's sides in neighbouring lanes
            const int it = t >> 1, side = t & 1, gi = c * kPairChunk + it;
            int lo = 0, kind = 0;
            bool inside = true;
            int2 vw = make_int2(-1, -1);
            if (gi < ni) {
                vw = P.bitems[gi];
                const ViewP vp = P.views[vw.x];
                if (side == 0) vsh[buf][it] = vp;
                const float Xl = side ? -Xa : Xa, Xr = side ? -Xb : Xb;
                const float m = fminf(fminf(det_coord(vp, Xl, Ya), det_coord(vp, Xl, Yb)),
                                      fminf(det_coord(vp, Xr, Ya), det_coord(vp, Xr, Yb)));
                lo = (__float2int_rd(__fadd_rn(m, P.uc)) - 3) & ~3;
                const int nc = (vp.flags & kViewBwd3) ? 3 : 2;
#pragma unroll
                for (int k = 0; k < 4; ++k) {   // the corners' first candidates bound every pixel's, as k_backward
                    const float Xc = (k & 1) ? Xr : Xl, Yc = (k & 2) ? Yb : Ya;
                    const float pbc = __fmaf_rn(-vp.cu_hi, Xc, __fmaf_rn(-vp.su_hi, Yc, -P.uc_hi));
                    const float smc = delta_small(vp, Xc, Yc, P.uc_lo);
                    const int q = magic_int(ceil_magic(__fsub_rn(__fsub_rn(smc, pbc), vp.hwu))) - lo;
                    inside = inside && q >= 1 && q <= bw - nc - 1;
                }
                kind = (vp.flags & kViewAxis) ? 4 : (nc == 3 ? 1 : 0);
            }
            lo_sh[buf][it][side] = lo;
            const bool both = __shfl_xor_sync(0xffffffffu, (int)inside, 1) && inside;
            if (side == 0) {
                item_sh[buf][it] = vw;
                kind_sh[buf][it] = kind + ((both || kind == 4) ? 0 : 2);
            }
        }
        __syncthreads();
        const int V2 = bw >> 1;
        float *wb = proj_dyn + buf * kPairChunk * 2 * bw * 2 * NS;
        for (int e = t; e < kPairChunk * 2 * V2; e += kBwdThreads) {
            const int is = e / V2, k2 = e - is * V2;   // (item, side), two bins
            const int2 vw = item_sh[buf][is >> 1];
            const int ub = lo_sh[buf][is >> 1][is & 1] + 2 * k2;
            float y[2 * NS][2];   // v of r, v of q, w of r, w of q; or v, w
#pragma unroll
            for (int a = 0; a < 2 * NS; ++a) y[a][0] = y[a][1] = 0.0f;
            if (vw.x >= 0 && ub >= 0 && ub + 1 < Up) {
                const float pl = vsh[buf][is >> 1].P;   // the weights are in units of the view's plateau length
#pragma unroll
                for (int a = 0; a < 2 * NS; ++a) {
                    const int v = a < NS ? vw.x : vw.y;
                    if (v < 0) continue;   // an unpaired view: its partner's values are zeros
                    if (!DUAL && mode == BWD_PLAIN) {   // the caller's sinogram, rows of U bins
                        const size_t o = (size_t)v * P.U + ub;
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            if (ub + k < P.U) y[a][k] = load_user(user, o + k, io.storage);
                    } else {
                        const float *sn = (DUAL && (a & 1)) ? P.q : sino;
                        const float2 f = __ldg(reinterpret_cast<const float2 *>(sn + (size_t)v * Up + ub));
                        y[a][0] = f.x; y[a][1] = f.y;
                    }
                    y[a][0] = __fmul_rn(y[a][0], pl);
                    y[a][1] = __fmul_rn(y[a][1], pl);
                }
            }
            float *dst = wb + (is * bw + 2 * k2) * 2 * NS;
            if constexpr (DUAL) {
                reinterpret_cast<float4 *>(dst)[0] = make_float4(y[0][0], y[1][0], y[2 * NS - 2][0], y[2 * NS - 1][0]);
                reinterpret_cast<float4 *>(dst)[1] = make_float4(y[0][1], y[1][1], y[2 * NS - 2][1], y[2 * NS - 1][1]);
            } else {
                reinterpret_cast<float4 *>(dst)[0] = make_float4(y[0][0], y[1][0], y[0][1], y[1][1]);
            }
        }
    };

    const int per_part = (nchunks + parts - 1) / parts;
    const int c_begin = min(nchunks, vpart * per_part), c_end = min(nchunks, c_begin + per_part);
    if (c_begin < c_end) stage(c_begin);
    __syncthreads();
    int bad = 0;
    for (int c = c_begin; c < c_end; ++c) {
        const int buf = c & 1;
        if (c + 1 < c_end) stage(c + 1);   // other buffer; its previous readers finished at the last barrier
        const int nv = min(kPairChunk, ni - c * kPairChunk);
        // two items (four views) of this thread group, then one Kahan-compensated fold
        for (int g0 = grp; g0 < nv; g0 += 2 * kBwdSplit) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int it = g0 + q * kBwdSplit;
                if (it >= nv) continue;
                const int kind = kind_sh[buf][it];
                const int base = (buf * kPairChunk + it) * 2 * bw;   // the left window's first element
                if (kind < 2) {
                    const ViewP vp = vsh[buf][it];
                    const int win[2] = {base - lo_sh[buf][it][0], base + bw - lo_sh[buf][it][1]};
                    if (kind == 0) pair_x2<DUAL, 2, PXR>(vp, X2, Y, uc_hi, uc_lo, win, acc);
                    else pair_x2<DUAL, 3, PXR>(vp, X2, Y, uc_hi, uc_lo, win, acc);
                } else {
                    Acc a[PX];   // (addressable copies only here)
#pragma unroll
                    for (int e = 0; e < PX; ++e) a[e] = acc[e];
                    const ViewP *vp = &vsh[buf][it];
                    const int *lo = lo_sh[buf][it];
                    if (kind == 4) bad |= pair_checked<DUAL, true, 2, PXR>(vp, X, Y[0], uc_hi, uc_lo, lo, base, bw, a);
                    else if (kind == 3) bad |= pair_checked<DUAL, false, 3, PXR>(vp, X, Y[0], uc_hi, uc_lo, lo, base, bw, a);
                    else bad |= pair_checked<DUAL, false, 2, PXR>(vp, X, Y[0], uc_hi, uc_lo, lo, base, bw, a);
#pragma unroll
                    for (int e = 0; e < PX; ++e) acc[e] = a[e];
                }
            }
#pragma unroll
            for (int h = 0; h < NS * PX / 2; ++h) {   // the fold, two values per instruction
                uint64_t a;
                if constexpr (DUAL) { a = acc[h]; acc[h] = 0; }
                else { a = pk2(acc[2 * h], acc[2 * h + 1]); acc[2 * h] = acc[2 * h + 1] = 0; }
                const uint64_t y = sub2_rn(a, comp2[h]);
                const uint64_t tt = add2_rn(part2[h], y);
                comp2[h] = sub2_rn(sub2_rn(tt, part2[h]), y);
                part2[h] = tt;
            }
        }
        __syncthreads();
    }
    float part[NS * PX], comp[NS * PX];
#pragma unroll
    for (int h = 0; h < NS * PX / 2; ++h) {   // DUAL: (r, q) of pixel h, else pixels 2h and 2h + 1
        const int a = DUAL ? h : 2 * h, b = DUAL ? PX + h : 2 * h + 1;
        upk2(part2[h], part[a], part[b]);
        upk2(comp2[h], comp[a], comp[b]);
    }
    bwd_finish<DUAL, PX>(P, ntiles, pi, mode, io, parts, vpart, tile, grp, tg, bad != 0, part, comp, comb, red, &bad_sh, &last_sh,
                         [&](int e, int *i, int *jj) {
                             const int s = e / PXR;
                             *i = i0 + ly + kBwdRowStep * (e - s * PXR);
                             *jj = s ? P.nx - 1 - j : j;
                             return *i < P.ny && j < nh && (s == 0 || *jj != j);
                         });
}

int backward_pairs_blocks(int nx, int ny, int parts, int ti)
{
    return parts * ((ny + ti - 1) / ti) * (((nx + 1) / 2 + kBwdTileJ - 1) / kBwdTileJ);
}

template <bool DUAL, int FP, int TI>
static int launch_pairs(const Launch &L, int mode, int bwp, const Io &io)
{
    constexpr int per_bin = 2 * kPairChunk * 2 * 2 * (DUAL ? 2 : 1) * 4;
    int rc = func_attrs_once((const void *)k_backward_pairs<DUAL, FP, TI>, per_bin * kPairWindowMax);
    if (rc) return rc;
    k_backward_pairs<DUAL, FP, TI><<<L.blocks, kBwdThreads, per_bin * bwp, L.st>>>(L.probs, L.prefix, L.count, mode, io);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

template <bool DUAL>
static int launch_pairs_any(const Launch &L, int mode, int bwp, const Io &io)
{
    if (L.bparts != kBwdViewParts) return launch_pairs<DUAL, 0, kPairTileI>(L, mode, bwp, io);
    if (L.bwdp_ti == 4) return launch_pairs<DUAL, kBwdViewParts, 4>(L, mode, bwp, io);
    if (L.bwdp_ti == 8) return launch_pairs<DUAL, kBwdViewParts, 8>(L, mode, bwp, io);
    return launch_pairs<DUAL, kBwdViewParts, kPairTileI>(L, mode, bwp, io);
}

int launch_backward_pairs(const Launch &L, bool dual, int mode, int bwp, const Io &io)
{
    return dual ? launch_pairs_any<true>(L, mode, bwp, io) : launch_pairs_any<false>(L, mode, bwp, io);
}

} // namespace supcg
