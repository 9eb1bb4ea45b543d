// The exact transpose R^T y of the forward projection (Eq. (2.2): normal
// equations R^T R x = R^T b), for any set of views; sets of mirror pairs take
// backproject_pairs.cu.
//
// Backward (pixel-driven, gather over bins, no atomics).  A tile of 32 x 32
// pixels (16 or 8 rows in small grids) is shared by P.bparts blocks (the geometry's view parts, 1 .. 8),
// each taking a contiguous part of the view chunks; for chunks of 32 views the bins that the tile projects
// onto are staged in shared memory with 16-byte vector loads; every pixel
// gathers the two (three) bins nearest to its projected centre with the same
// weight evaluated on the same FP32 operands as the forward kernel.  The last
// block of a tile to finish adds the parts' double-float sums in part order.
#include "backward.cuh"

namespace supcg {

// The kernel's dynamic shared memory (the staged sinogram windows), indexed by
// 32-bit float offsets so that operand loads are plain shared-memory loads.
extern __shared__ __align__(128) float proj_dyn[];

// ============================================================ backward
// Tiles of TI x 32 pixels, TI / 4 per thread, over one sinogram or, DUAL, two (the
// solver's R^T r and R^T q in one pass: each pixel's weights evaluated once and
// applied to both; twice the sums per thread, so two blocks per SM instead of
// three).  Either way, and for every TI, a pixel sums its views in the same order (same
// groups, folds and parts), so each output has the same bits.  TI = 32 spreads a view's
// constants and staging over the most pixels; images whose 32-row tiles would leave SMs
// without a block take 16 or 8 rows (bwd_tile_rows).
template <bool DUAL, int TILE>
struct BwdShape {
    static constexpr int NS = DUAL ? 2 : 1;                        // sinograms
    static constexpr int TI = TILE;                                // tile rows
    static constexpr int PX = TI * kBwdTileJ / kBwdGroup;          // pixels per thread
};

// Per pixel and view: the bins within hwu (half-width + margin) of the pixel's
// projected centre, two of them (three when the bins are finer than pixels),
// with a check of the staged window.  t[s * PX + e]: sinogram s, pixel e; the
// window of sinogram s starts qoff floats after that of sinogram 0.
template <bool AXIS, int NC, int PX, int NS>
__device__ __forceinline__ void bwd_view(const ViewP &vp, float pb0, const float *sm, int w_row, int lo,
                                         int bwin, int qoff, float *t, int *bad)
{
    const float E = vp.E, Sn = vp.Sn, ESn = vp.ESn;
#pragma unroll
    for (int e = 0; e < PX; ++e) {
        // delta = (u + pb) - small; pb = -uc_hi - cu_hi X - su_hi Y is exact, and so is
        // stepping it by su_hi per pixel row
        const float pb = __fmaf_rn((float)(kBwdRowStep * e), vp.su_hi, pb0);
        const float uc = ceil_magic(__fsub_rn(__fsub_rn(sm[e], pb), vp.hwu));
        int u0 = magic_int(uc);
        const int idx = u0 - lo;
        if (idx < 0 || idx > bwin - NC) {   // outside the staged window: never for a valid window
            *bad = 1;
            u0 = min(max(idx, 0), bwin - NC) + lo;
        }
        const float big0 = __fadd_rn(__int2float_rn(u0), pb);   // exact, as are big0 + 1 and big0 + 2
        const int wv = w_row + (u0 - lo);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const float ad = fabsf(__fsub_rn(__fadd_rn(big0, (float)k), sm[e]));
            const float w = weight_unit(ad, E, Sn, ESn, AXIS);
#pragma unroll
            for (int s = 0; s < NS; ++s)   // the window holds P * y
                t[s * PX + e] = __fmaf_rn(w, proj_dyn[wv + s * qoff + k], t[s * PX + e]);
        }
    }
}

// The same for the thread's pixels in pairs (2h, 2h + 1), every FP32 step as one
// f32x2 instruction; only for windows that hold every candidate (no checks).
// sm2[h] = (small of pixel 2h, of pixel 2h + 1); t2[s * PX / 2 + h] the pairs'
// running sums for sinogram s.
template <bool AXIS, int NC, int PX, int NS>
__device__ __forceinline__ void bwd_view_x2(const ViewP &vp, float pb0, const uint64_t *sm2, int w_row, int lo,
                                            int qoff, uint64_t *t2)
{
    const float E = vp.E, Sn = vp.Sn, ESn = vp.ESn;
    const uint64_t su2 = pk2(vp.su_hi, vp.su_hi), hwu2 = pk2(vp.hwu, vp.hwu), pbb = pk2(pb0, pb0);
    const uint64_t mag2 = pk2(kCeilMagic, kCeilMagic);
#pragma unroll
    for (int h = 0; h < PX / 2; ++h) {
        const uint64_t st = pk2((float)(kBwdRowStep * 2 * h), (float)(kBwdRowStep * (2 * h + 1)));
        const uint64_t pb = fma2_rn(st, su2, pbb);                          // exact
        const uint64_t uc = add2_rp(sub2_rn(sub2_rn(sm2[h], pb), hwu2), mag2);
        float uca, ucb;
        upk2(uc, uca, ucb);
        const int wa = w_row + (magic_int(uca) - lo), wb = w_row + (magic_int(ucb) - lo);
        const uint64_t big0 = add2_rn(sub2_rn(uc, mag2), pb);              // exact, as are big0 + 1, + 2
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const uint64_t bk = k ? add2_rn(big0, pk2((float)k, (float)k)) : big0;
            float da, db;
            upk2(sub2_rn(bk, sm2[h]), da, db);
            const uint64_t w = pk2(weight_unit(fabsf(da), E, Sn, ESn, AXIS), weight_unit(fabsf(db), E, Sn, ESn, AXIS));
#pragma unroll
            for (int s = 0; s < NS; ++s)   // the window holds P * y
                t2[s * PX / 2 + h] =
                    fma2_rn(w, pk2(proj_dyn[wa + s * qoff + k], proj_dyn[wb + s * qoff + k]), t2[s * PX / 2 + h]);
        }
    }
}

// R^T y over one sinogram (mode BWD_G: y = r into g, BWD_PLAIN: the caller's sinogram
// into the caller's image, or into g where io has none), or, DUAL, over two in one pass:
// g from r and h from q (h = A p for the beta of the next step of Algorithm 2,
// deferred to this pass: alpha takes p^T A p from the forward projector's ||q||^2).
// FIXED_PARTS: the view parts per tile when every problem of the launch has that
// (default) number, so the part arithmetic is compile-time; 0: each problem's own.
template <bool DUAL, int FIXED_PARTS, int TILE>
__global__ void __launch_bounds__(kBwdThreads, DUAL ? 2 : 3) k_backward(const Prob *__restrict__ probs,
                                                          const int *__restrict__ prefix, int count, int mode,
                                                          Io io)
{
    constexpr int NS = BwdShape<DUAL, TILE>::NS, TI = BwdShape<DUAL, TILE>::TI, PX = BwdShape<DUAL, TILE>::PX;
    // proj_dyn: [2][NS][kBwdViewChunk][bwin] sinogram windows
    __shared__ ViewP vsh[2][kBwdViewChunk];
    __shared__ int ulo_sh[2][kBwdViewChunk];
    __shared__ int kind_sh[2][kBwdViewChunk];   // variant: three bins (1) / two bins (2), + 3 if a window check is needed; axis 3
    __shared__ float2 comb[kBwdGroup * NS * PX];   // second group's sums, combined by the first
    __shared__ __align__(16) double red[40];
    __shared__ int bad_sh, last_sh;

    int local;
    const int pi = find_problem(prefix, count, blockIdx.x, &local);
    const Prob &P = probs[pi];
    if ((DUAL || mode != BWD_PLAIN) && P.sc->done) return;

    const int bwin = P.bwin;
    const int qoff = kBwdViewChunk * bwin;   // second sinogram's windows after the first's
    const int tiles_j = (P.nx + kBwdTileJ - 1) / kBwdTileJ;
    // part-major: every tile's first part, then its second, ...; the last part has the
    // fewest view chunks, so the grid's final (partial) wave holds the shortest blocks
    const int parts = FIXED_PARTS ? FIXED_PARTS : P.bparts;
    const int ntiles_p = (prefix[pi + 1] - prefix[pi]) / parts;
    const int vpart = local / ntiles_p, tile = local - vpart * ntiles_p;   // this block's part of the views
    const int ti = tile / tiles_j, tj = tile - ti * tiles_j;
    const int i0 = ti * TI, j0 = tj * kBwdTileJ;
    const int t = threadIdx.x;
    const int grp = t / kBwdGroup, tg = t - grp * kBwdGroup;   // group grp takes views vv = grp (mod kBwdSplit)
    const int lx = tg % kBwdTileJ, ly = tg / kBwdTileJ;
    const int j = j0 + lx;
    const float X = __fsub_rn(__int2float_rn(j), P.cx);
    float Y[PX];
#pragma unroll
    for (int e = 0; e < PX; ++e) Y[e] = __fsub_rn(P.cy, __int2float_rn(i0 + ly + kBwdRowStep * e));
    // per pixel: FP32 sum of up to four views (t2), folded into a Kahan-compensated pair (part, comp)
    // that runs over all views, FP64 only for the final value (the FP64 pipe is narrow).  The views are
    // issue-bound, so all three are kept as pixel pairs and the fold takes half the instructions; it
    // also ends the repacking that spilled 28 to 112 bytes (171.9 -> 168.3 us for eight 243^2 / 360)
    uint64_t part2[NS * PX / 2], comp2[NS * PX / 2], t2[NS * PX / 2];
#pragma unroll
    for (int h = 0; h < NS * PX / 2; ++h) t2[h] = part2[h] = comp2[h] = pk2(0.0f, 0.0f);
    uint64_t Y2[PX / 2];
#pragma unroll
    for (int h = 0; h < PX / 2; ++h) Y2[h] = pk2(Y[2 * h], Y[2 * h + 1]);
    const uint64_t X2 = pk2(X, X);

    const void *user = io.in + (size_t)pi * io.in_step;
    const int Up = P.Up;
    // tile corners in pixel-centre coordinates
    const float Xa = __fsub_rn(__int2float_rn(j0), P.cx), Xb = __fsub_rn(__int2float_rn(j0 + kBwdTileJ - 1), P.cx);
    const float Ya = __fsub_rn(P.cy, __int2float_rn(i0)), Yb = __fsub_rn(P.cy, __int2float_rn(i0 + TI - 1));
    if (t == 0) bad_sh = 0;

    const int nchunks = (P.V + kBwdViewChunk - 1) / kBwdViewChunk;
    // stage chunk c into buffer c&1
    auto stage = [&](int c) {
        const int buf = c & 1;
        const int v0 = c * kBwdViewChunk;
        if (t < kBwdViewChunk) {
            const int v = v0 + t;
            int lo = 0;
            int kind = 0;
            if (v < P.V) {
                const ViewP vp = P.views[v];
                vsh[buf][t] = vp;
                float m = fminf(fminf(det_coord(vp, Xa, Ya), det_coord(vp, Xa, Yb)),
                                fminf(det_coord(vp, Xb, Ya), det_coord(vp, Xb, Yb)));
                lo = (__float2int_rd(__fadd_rn(m, P.uc)) - 3) & ~3;
                // a pixel's first candidate is (up to rounding) linear in X and Y, so its values at
                // the tile's corners, with one bin of slack, bound it for every pixel of the tile;
                // they are computed exactly as each pixel's own
                const int nc = (vp.flags & kViewBwd3) ? 3 : 2;
                bool inside = true;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float Xc = (k & 1) ? Xb : Xa, Yc = (k & 2) ? Yb : Ya;
                    const float pbc = __fmaf_rn(-vp.cu_hi, Xc, __fmaf_rn(-vp.su_hi, Yc, -P.uc_hi));
                    const float smc = delta_small(vp, Xc, Yc, P.uc_lo);
                    const int q = magic_int(ceil_magic(__fsub_rn(__fsub_rn(smc, pbc), vp.hwu))) - lo;
                    inside = inside && q >= 1 && q <= bwin - nc - 1;
                }
                // axis-aligned views (two in a uniform set) always take the checked scalar path
                kind = ((vp.flags & kViewAxis) ? 3 : (nc == 3 ? 1 : 2) + (inside ? 0 : 3));
            }
            ulo_sh[buf][t] = lo;
            kind_sh[buf][t] = kind;
        }
        __syncthreads();
        const int V4 = bwin >> 2;
        float *wb = proj_dyn + buf * NS * qoff;
        for (int e = t; e < NS * kBwdViewChunk * V4; e += kBwdThreads) {
            const int s = (NS == 2 && e >= kBwdViewChunk * V4) ? 1 : 0;
            const int es = e - s * kBwdViewChunk * V4;
            const int vv = es / V4, k4 = es - vv * V4;
            const int v = v0 + vv;
            float4 val = make_float4(0.f, 0.f, 0.f, 0.f);
            const int ub = ulo_sh[buf][vv] + 4 * k4;
            if (v < P.V && ub >= 0 && ub + 3 < Up) {
                if (!DUAL && mode == BWD_PLAIN) {   // the caller's sinogram, rows of U bins
                    const size_t o = (size_t)v * P.U + ub;
                    val.x = load_user(user, o, io.storage);   // (ub < U: U > Up - 4, and ub is a multiple of 4)
                    if (ub + 1 < P.U) val.y = load_user(user, o + 1, io.storage);
                    if (ub + 2 < P.U) val.z = load_user(user, o + 2, io.storage);
                    if (ub + 3 < P.U) val.w = load_user(user, o + 3, io.storage);
                } else {
                    val = __ldg(reinterpret_cast<const float4 *>((s ? P.q : P.r) + (size_t)v * Up + ub));
                }
                const float pl = vsh[buf][vv].P;   // the weights are in units of the view's plateau length
                val.x = __fmul_rn(val.x, pl);
                val.y = __fmul_rn(val.y, pl);
                val.z = __fmul_rn(val.z, pl);
                val.w = __fmul_rn(val.w, pl);
            }
            *reinterpret_cast<float4 *>(wb + s * qoff + vv * bwin + 4 * k4) = val;
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
        const int nv = min(kBwdViewChunk, P.V - c * kBwdViewChunk);
        const int wb = buf * NS * qoff;
        // groups of four of this thread group's views, then one Kahan-compensated fold
        for (int g0 = grp; g0 < nv; g0 += 4 * kBwdSplit) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int vv = g0 + q * kBwdSplit;
                if (vv < nv) {
                    const ViewP vp = vsh[buf][vv];
                    const int wr = wb + vv * bwin;
                    const int lo = ulo_sh[buf][vv];
                    const float pb0 = __fmaf_rn(-vp.cu_hi, X, __fmaf_rn(-vp.su_hi, Y[0], -P.uc_hi));
                    // small = uc_lo + cu_lo X + su_lo Y in the view class's order (delta_small), in pairs
                    uint64_t sm2[PX / 2];
                    if (vp.flags & kViewClassB) {
                        const float in = __fmaf_rn(vp.cu_lo, X, P.uc_lo);
                        const uint64_t s2 = pk2(vp.su_lo, vp.su_lo), in2 = pk2(in, in);
#pragma unroll
                        for (int h = 0; h < PX / 2; ++h) sm2[h] = fma2_rn(s2, Y2[h], in2);
                    } else {
                        const uint64_t s2 = pk2(vp.su_lo, vp.su_lo), c2 = pk2(vp.cu_lo, vp.cu_lo),
                                       u2 = pk2(P.uc_lo, P.uc_lo);
#pragma unroll
                        for (int h = 0; h < PX / 2; ++h) sm2[h] = fma2_rn(c2, X2, fma2_rn(s2, Y2[h], u2));
                    }
                    const int kind = kind_sh[buf][vv];
                    if (kind < 3) {
                        if (kind == 1) bwd_view_x2<false, 3, PX, NS>(vp, pb0, sm2, wr, lo, qoff, t2);
                        else bwd_view_x2<false, 2, PX, NS>(vp, pb0, sm2, wr, lo, qoff, t2);
                    } else {   // a window check is needed: the scalar path
                        float sm[PX], t4[NS * PX];
#pragma unroll
                        for (int h = 0; h < PX / 2; ++h) upk2(sm2[h], sm[2 * h], sm[2 * h + 1]);
#pragma unroll
                        for (int h = 0; h < NS * PX / 2; ++h) upk2(t2[h], t4[2 * h], t4[2 * h + 1]);
                        if (kind == 3) bwd_view<true, 2, PX, NS>(vp, pb0, sm, wr, lo, bwin, qoff, t4, &bad);
                        else if (kind == 4) bwd_view<false, 3, PX, NS>(vp, pb0, sm, wr, lo, bwin, qoff, t4, &bad);
                        else bwd_view<false, 2, PX, NS>(vp, pb0, sm, wr, lo, bwin, qoff, t4, &bad);
#pragma unroll
                        for (int h = 0; h < NS * PX / 2; ++h) t2[h] = pk2(t4[2 * h], t4[2 * h + 1]);
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < NS * PX / 2; ++h) {   // the fold, two pixels per instruction
                const uint64_t y = sub2_rn(t2[h], comp2[h]);
                const uint64_t tt = add2_rn(part2[h], y);
                comp2[h] = sub2_rn(sub2_rn(tt, part2[h]), y);
                part2[h] = tt;
                t2[h] = pk2(0.0f, 0.0f);
            }
        }
        __syncthreads();
    }
    float part[NS * PX], comp[NS * PX];
#pragma unroll
    for (int h = 0; h < NS * PX / 2; ++h) {
        upk2(part2[h], part[2 * h], part[2 * h + 1]);
        upk2(comp2[h], comp[2 * h], comp[2 * h + 1]);
    }
    bwd_finish<DUAL, PX>(P, (prefix[pi + 1] - prefix[pi]) / parts, pi, mode, io, parts, vpart, tile, grp, tg, bad != 0, part,
                         comp, comb, red, &bad_sh, &last_sh, [&](int e, int *i, int *jj) {
                             *i = i0 + ly + kBwdRowStep * e;
                             *jj = j;
                             return *i < P.ny && j < P.nx;
                         });
}

// Blocks per problem: `parts` per pixel tile of `ti` rows.
int backward_blocks(int nx, int ny, int parts, int ti)
{
    return parts * ((ny + ti - 1) / ti) * ((nx + kBwdTileJ - 1) / kBwdTileJ);
}

// Rows of a launch's tiles, from its number of blocks with 32 rows: the lowest with which the grid still is
// no more than two blocks per SM, which all run at once (two of the solver's dual pass fit).  A block's time
// is a serial chain of view groups whose length hardly falls below its rows' share while the SM has nothing
// else to issue.  One R^T y with 32 rows and as chosen, us: 64^2 / 90 views 16.4 and 9.6 (8 rows),
// 128^2 / 180 20.6 and 14.4 (8), 160^2 / 200 20.6 and 16.4 (16), 192^2 / 240 20.6 and 18.5 (16); from
// 224^2 / 300 on (28.7) the 32-row grid has more than one block per SM and stays.  The solver's dual pass at 64^2:
// 25.6 and 14.6.  Over mirror pairs, tiles of half the rows (on both sides of the image) by the same rule:
// 9.6 us at 64^2 (4 rows; 12.3 with 8), the dual pass 14.3 (16.1).
int bwd_tile_rows(long long blocks32, int nsm)
{
    return 4 * blocks32 <= 2 * nsm ? 8 : (2 * blocks32 <= 2 * nsm ? 16 : kBwdTileI);
}

template <bool DUAL, int FP, int TILE>
static int launch_bwd(const Launch &L, int mode, int bwin, const Io &io)
{
    const int smem = 2 * (DUAL ? 2 : 1) * kBwdViewChunk * bwin * 4;
    int rc = func_attrs_once((const void *)k_backward<DUAL, FP, TILE>, 2 * (DUAL ? 2 : 1) * kBwdViewChunk * 256 * 4);
    if (rc) return rc;
    k_backward<DUAL, FP, TILE><<<L.blocks, kBwdThreads, smem, L.st>>>(L.probs, L.prefix, L.count, mode, io);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

template <bool DUAL>
static int launch_bwd_any(const Launch &L, int mode, int bwin, const Io &io)
{
    if (L.bparts != kBwdViewParts) return launch_bwd<DUAL, 0, kBwdTileI>(L, mode, bwin, io);
    if (L.bwd_ti == 8) return launch_bwd<DUAL, kBwdViewParts, 8>(L, mode, bwin, io);
    if (L.bwd_ti == 16) return launch_bwd<DUAL, kBwdViewParts, 16>(L, mode, bwin, io);
    return launch_bwd<DUAL, kBwdViewParts, kBwdTileI>(L, mode, bwin, io);
}

int launch_backward(const Launch &L, int mode, int bwin, const Io &io) { return launch_bwd_any<false>(L, mode, bwin, io); }
int launch_backward2(const Launch &L, int bwin) { return launch_bwd_any<true>(L, BWD_G, bwin, Io()); }

} // namespace supcg
