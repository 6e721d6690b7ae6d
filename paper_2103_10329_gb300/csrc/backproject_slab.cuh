// A^T on separable geometries by a thread per voxel column and z slab, over
// sinograms stored [view][v][u]: in shared memory (k_backproject_slab) or, for
// 16-bit storage and detector rows in its range of steps, in registers
// (k_backproject_reg).  These serve what the plane kernel (backproject.cuh) does
// not: bp_route in project.cuh has the lines and the figures.
//
// 16-bit storage takes them throughout, so far.  The plane kernel is faster there,
// too (865 against 1001 ms per step at 512^3 / 1440 views with BF16 storage), and
// more exact, but rounds differently: the filter has no response to a constant,
// so a step amplifies A^T's rounding about fifty times, and in the next step that
// moves entries of the 16-bit residual across rounding boundaries -- iterates
// then differ by up to 2.5e-4 after two steps, the size of 16-bit storage's own
// error.
#pragma once

#include "common.cuh"

namespace mgct {

// Separable geometry, weighted sinogram.
// Each thread owns one (x, y) voxel column and a slab of Z voxels along z,
// accumulated in shared memory.  Per view and per detector column u' whose
// rays meet the voxel column (|e_b| < 1), the z crossing of the ray through
// pixel (u', v') is f_z(v') = E0' + v' E1 (E0' uncentred), so the voxels the
// ray touches are floor(f_z) and floor(f_z) + 1 with weights (1 - t, t),
// t = f_z - floor(f_z): the exact transpose of the projector's bilinear tap
// in z.  Each pixel of the slab's v range is visited once and splatted into
// the thread's own shared-memory column (no two threads share a column, so
// no atomics, and the order of additions is fixed).  Lanes are adjacent x
// columns, so the pixel reads of a warp fall on one detector row.
constexpr int BS_TX = 32, BS_TY = 4, BS_THREADS = BS_TX * BS_TY;
constexpr float BS_MAGIC = 12582912.0f;  // 1.5 * 2^23
constexpr int BS_MAGIC_BITS = 0x4B400000;
template <int NCH>
struct SlabCfg {
    // 16 voxels per slab keep the shared slab at 10 KB so that 16 blocks (64
    // warps) fit per SM; guard rows: two below, three above (row pairs reach r + 2)
    static constexpr int Z = 16 / NCH, ROWS = Z + 5;
};

__device__ __forceinline__ float2 load_f2(const float2 *p) { return __ldg(p); }
template <typename ST>
__device__ __forceinline__ float2 load_f2(const ST *) { return make_float2(0.0f, 0.0f); }

// DFA = true: 32-bit rays, from the double-float column table; the z crossing is
// anchored, in double-float, at the detector row nearest the slab's centre, as a
// whole number of voxels and a rest, and a row's fraction formed from these with
// the step's low part (vf E1 less whole voxels in one rounding): a weight is
// accurate to ~1e-7 at any N, as in the plane kernel.  (From one float above the
// slab: 1e-6; the float32 table's uncentred heights near z = 1000: 6e-5.)
template <int NCH, typename ST, bool DFA = false>
__global__ void __launch_bounds__(BS_THREADS)
    k_backproject_slab(BPArgs a, const float4 *__restrict__ cols, const ST *__restrict__ sino,
                       float *__restrict__ out, int accumulate) {
    constexpr int Z = SlabCfg<NCH>::Z, ROWS = SlabCfg<NCH>::ROWS;
    __shared__ float acc[NCH][ROWS][BS_THREADS];
    const int tid = threadIdx.x;
    const int jx = blockIdx.x * BS_TX + (tid % BS_TX), jy = blockIdx.y * BS_TY + tid / BS_TX;
    // blockIdx.z = split * (z-slabs) + slab; split s takes views [i0, i1)
    // and writes partial volume s of `out`
    const int splits = a.splits;
    const int zblocks = gridDim.z / splits;
    const int split = blockIdx.z / zblocks;
    const int z0 = (blockIdx.z - split * zblocks) * Z;
    const int per = (a.nviews + splits - 1) / splits;
    const int i0 = split * per, i1 = min(a.nviews, i0 + per);
#pragma unroll
    for (int q = 0; q < NCH; ++q)
        for (int r = 0; r < ROWS; ++r) acc[q][r][tid] = 0.0f;
    if (jx < a.n && jy < a.n) {
        const float ic = 0.5f * (float)(a.n - 1);
        const float cu = 0.5f * (float)(a.nu - 1), cv = 0.5f * (float)(a.nv - 1);
        const float cx = (float)jx - ic, cy = (float)jy - ic;
        const float zlo = (float)z0 - 1.0f, zhi = (float)(z0 + Z);  // crossings that touch the slab
        const size_t view_elems = (size_t)a.nu * a.nv;
        for (int i = i0; i < i1; ++i) {
            const int k = a.view0 + i * a.stride;
            const float *G = reinterpret_cast<const float *>(a.views + k);
            // projected u range of the voxel column (the cube bound; z-free without tilt)
            const float X = (float)jx - __ldg(G + 0), Y = (float)jy - __ldg(G + 1);
            const float Q0 = __ldg(G + 12), Q1 = __ldg(G + 13), Q6 = __ldg(G + 18), Q7 = __ldg(G + 19);
            const float q2 = fmaf(Q7, Y, Q6 * X);
            const float u0 = fmaf(Q1, Y, Q0 * X) * __frcp_rn(q2);
            const float hu = (fabsf(Q0 - u0 * Q6) + fabsf(Q1 - u0 * Q7)) * __frcp_rn(q2 - __ldg(G + 21));
            const int ulo = max(0, (int)ceilf(u0 - hu + cu - 1e-3f));
            const int uhi = min(a.nu - 1, (int)floorf(u0 + hu + cu + 1e-3f));
            const ST *__restrict__ sv = sino + (size_t)i * view_elems;
            const float4 *__restrict__ ct = cols + (size_t)k * a.nu * (DFA ? 4 : 2);
            for (int ju = ulo; ju <= uhi; ++ju) {
                const float4 t0 = __ldg(ct + (DFA ? ju : 2 * ju));
                const float4 t1 = __ldg(ct + (DFA ? a.nu + ju : 2 * ju + 1));
                const bool ay = t0.x != 0.0f;
                const float ca = ay ? cy : cx, cb = ay ? cx : cy;
                // E0, E1: crossing height at row offset vf = 0 and its slope per
                // row; zb: the height E0 is counted from (uncentred z)
                float hb, E0, E1, vf;
                float E0i = 0.0f, E0f = 0.0f, El = 0.0f;  // DFA: E0 = E0i + E0f, E1's low part
                int vlo, vhi, zb;
                if constexpr (!DFA) {
                    hb = 1.0f - fabsf(fmaf(ca, t0.y, t0.z) - cb);
                    if (hb <= 0.0f) continue;
                    E0 = fmaf(ca, t1.x, t0.w) + ic;  // uncentred z crossing at v' = 0
                    E1 = fmaf(ca, t1.z, t1.y);
                    const float rE = __frcp_rn(E1);
                    const float ta = fmaf(zlo - E0, rE, cv), tb = fmaf(zhi - E0, rE, cv);
                    vlo = max(0, (int)ceilf(fminf(ta, tb) - 1e-3f));
                    vhi = min(a.nv - 1, (int)floorf(fmaxf(ta, tb) + 1e-3f));
                    vf = (float)vlo - cv;
                    zb = z0;
                } else {
                    const float4 t2 = __ldg(ct + 2 * a.nu + ju), t3 = __ldg(ct + 3 * a.nu + ju);
                    const DF eb = df_add(df_mul_f(DF{t0.y, t0.z}, ca), DF{t0.w, t1.x});
                    hb = 1.0f - fabsf(__fadd_rn(__fsub_rn(eb.hi, cb), eb.lo));
                    if (hb <= 0.0f) continue;
                    const DF Eb = df_add(DF{t1.y, t1.z}, df_mul_f(DF{t1.w, t2.x}, ca));  // centred, v' = 0
                    const DF E1d = df_add(DF{t2.y, t2.z}, df_mul_f(DF{t2.w, t3.x}, ca));
                    E1 = E1d.hi;
                    const float zc = (float)z0 - ic + 0.5f * (float)(Z - 1);  // slab centre, centred (exact)
                    const float va = rintf((zc - Eb.hi) / E1);                // anchor row, centred v'
                    if (!(fabsf(va) < 1.0e7f)) continue;
                    const DF c = df_add(df_add(Eb, df_mul_f(E1d, va)), DF{-zc, 0.0f});
                    E0 = (c.hi + c.lo) + 0.5f * (float)(Z - 1);  // height above z0 at the anchor row
                    E0i = floorf(E0);
                    E0f = (c.hi - (E0i - 0.5f * (float)(Z - 1))) + c.lo;
                    El = E1d.lo;
                    const float rE = __frcp_rn(E1);
                    const float ta = fmaf(-1.0f - E0, rE, va + cv), tb = fmaf((float)Z - E0, rE, va + cv);
                    vlo = max(0, (int)ceilf(fminf(ta, tb) - 1e-3f));
                    vhi = min(a.nv - 1, (int)floorf(fmaxf(ta, tb) + 1e-3f));
                    vf = ((float)vlo - cv) - va;  // rows from the anchor (exact)
                    zb = 0;
                }
                // the fraction of a row's height fz above voxel floor(fz)
                auto frac = [&](float v, float fz, float fl) {
                    return DFA ? fmaf(v, E1, E0i - fl) + fmaf(v, El, E0f) : fz - fl;
                };
                const ST *__restrict__ px = sv + (size_t)vlo * a.nu + ju;
                int jv = vlo;
                if constexpr (NCH == 1) {
                  if (E1 > 0.0f && E1 < 0.999f) {
                    // two rows at a time: their crossings floor(fz) are equal or
                    // one apart (0 < E1 < 1), so the pair touches three slab
                    // rows r, r + 1, r + 2 -- three read-modify-writes, not four
                    // floor(fz) from one addition rounded toward minus infinity
                    // (fz + 1.5 * 2^23 holds it in its low mantissa bits); a
                    // row index outside the slab wraps, as unsigned, to the top
                    // guard rows
                    const int rbase = BS_MAGIC_BITS + zb - 2;
                    for (; jv + 1 <= vhi; jv += 2, vf += 2.0f, px += 2 * (size_t)a.nu) {
                        const float fz0 = fmaf(vf, E1, E0), fz1 = fmaf(vf + 1.0f, E1, E0);
                        const float m0 = __fadd_rd(fz0, BS_MAGIC), m1 = __fadd_rd(fz1, BS_MAGIC);
                        const float t0 = frac(vf, fz0, m0 - BS_MAGIC), t1 = frac(vf + 1.0f, fz1, m1 - BS_MAGIC);
                        const int r = (int)min((unsigned)(__float_as_int(m0) - rbase), (unsigned)(ROWS - 3));
                        const bool same = __float_as_int(m1) == __float_as_int(m0);
                        const float y0 = hb * to_f32(__ldg(px)), y1 = hb * to_f32(__ldg(px + a.nu));
                        const float a0 = y0 * t0, b0 = y1 * t1;
                        const float lo1 = y1 - b0;
                        acc[0][r][tid] += (y0 - a0) + (same ? lo1 : 0.0f);
                        acc[0][r + 1][tid] += a0 + (same ? b0 : lo1);
                        if (!same) acc[0][r + 2][tid] += b0;
                    }
                  }
                }
                for (; jv <= vhi; ++jv, vf += 1.0f, px += a.nu) {
                    const float fz = fmaf(vf, E1, E0);
                    const float fl = floorf(fz);
                    const float t = frac(vf, fz, fl);
                    // row of voxel floor(fz) in the guarded slab: in [0, Z + 2]
                    const int r = min(max((int)fl - zb + 2, 0), ROWS - 2);
                    if constexpr (NCH == 1) {
                        const float yw = hb * to_f32(__ldg(px));
                        const float w1 = yw * t;
                        acc[0][r][tid] += yw - w1;
                        acc[0][r + 1][tid] += w1;
                    } else {
                        const float2 y2 = load_f2(px);
                        const float ya = hb * y2.x, yb = hb * y2.y;
                        acc[0][r][tid] += ya - ya * t;
                        acc[0][r + 1][tid] += ya * t;
                        acc[NCH - 1][r][tid] += yb - yb * t;
                        acc[NCH - 1][r + 1][tid] += yb * t;
                    }
                }
            }
        }
        const size_t nvox = (size_t)a.n * a.n * a.n;
        float *o = out + (size_t)split * NCH * nvox;
        for (int zz = 0; zz < Z; ++zz) {
            const int z = z0 + zz;
            if (z >= a.n) break;
            const size_t idx = ((size_t)z * a.n + jy) * a.n + jx;
#pragma unroll
            for (int q = 0; q < NCH; ++q) {
                float v = acc[q][zz + 2][tid];
                if (accumulate) v += o[idx + q * nvox];
                o[idx + q * nvox] = v;
            }
        }
    }
}

// Register form of the solver's A^T (separable geometry, weighted rows, one
// channel) for grids whose detector rows are finer than the voxels along z:
// 1/3 < E1 < 1 for every view, column and plane (LevelInfo::e1_lo / e1_hi).
// As in the slab kernel a thread owns one (x, y) voxel column and ZS voxels
// z0 .. z0 + ZS - 1 of it, but the slab lives in registers.  Measured from
// z0 - 1, a detector column's row crossings rise by E1 < 1 per row, so the
// unit interval j of heights, [j, j + 1), j = 0 .. ZS, holds floor(1/E1) or
// ceil(1/E1) rows (K = ceil(1/E1) slots, the later ones predicated).  With
// S_j the interval's sum of y and T_j its sum of y t (t = the row's height
// above j), the tent weights give voxel z0 - 1 + j the share hb (S_j - T_j)
// and voxel z0 + j the share hb T_j -- the slab kernel's two taps per row,
// summed per interval, every accumulator index fixed at compile time.
// A block is BR_TX x BR_TY voxel columns; a warp BR_WX x (32 / BR_WX) of them
// (on views whose rays run along a warp's long side, its lanes' detector
// columns and rows spread apart: warps of 32 x 1 columns 31.2 ms per launch at
// 256^3 / 720 views, 8 x 4 29.5).  16 voxels, the later slots' rows loaded
// before their test, 40 registers (12 blocks per SM).
constexpr int BR_TX = 32, BR_TY = 4, BR_THREADS = BR_TX * BR_TY;
constexpr int BR_WX = 8, BR_WY = 32 / BR_WX;
constexpr int BR_Z = 16;                               // voxels per thread along z
constexpr float BR_E1_LO = 1.0f / 3.0f + 1e-3f;        // eligible grids: BR_E1_LO < E1 < BR_E1_HI
constexpr float BR_E1_HI = 1.0f - 1e-3f;
constexpr float BR_K2 = 0.5f + 1e-3f;                  // E1 above this: at most two rows per interval

// One detector column's rows into acc: off is the element offset of the
// first row (row v, height w in [0, E1) above z0 - 1) in the view's
// sinogram.  EDGE: rows outside [0, nv) read as zero (not loaded).
template <int ZS, int K, bool EDGE, typename ST>
__device__ __forceinline__ void br_column(float (&acc)[ZS], const ST *__restrict__ sv, int off, int nu, float w,
                                          float E1, float hb, int v, int nv) {
#pragma unroll
    for (int j = 0; j <= ZS; ++j) {
        float y = 0.0f;
        if (!EDGE || (unsigned)v < (unsigned)nv) y = to_f32(__ldg(sv + off));
        float S = y, T = y * w;
        float wn = w + E1;  // height of the next row above j
        int adv = 1;
#pragma unroll
        for (int s = 1; s < K; ++s) {
            if (!EDGE) {
                // the row after the interval's last lies within the rows the
                // launch checked, so the load need not wait for the test
                const float yl = to_f32(__ldg(sv + off + s * nu));
                const bool in = wn < 1.0f;
                const float ys = in ? yl : 0.0f;
                S += ys;
                T = fmaf(ys, wn, T);
                if (in) {
                    wn += E1;
                    adv = s + 1;
                }
            } else if (wn < 1.0f) {
                float ys = 0.0f;
                if (!EDGE || (unsigned)(v + s) < (unsigned)nv) ys = to_f32(__ldg(sv + off + s * nu));
                S += ys;
                T = fmaf(ys, wn, T);
                wn += E1;
                adv = s + 1;
            }
        }
        if (j >= 1) acc[j - 1] = fmaf(hb, S - T, acc[j - 1]);
        if (j < ZS) acc[j] = fmaf(hb, T, acc[j]);
        w = wn - 1.0f;  // the first row of interval j + 1
        off += adv * nu;
        if (EDGE) v += adv;
    }
}

// Detector column ju of the view whose sinogram is sv into acc, weighted hb:
// E0 is the uncentred z crossing of its rays at v' = 0 and E1 its step per
// row, at the voxel column's plane; the slab's intervals start at zlo.
template <int ZS, typename ST>
__device__ __forceinline__ void br_add_column(float (&acc)[ZS], const ST *__restrict__ sv, int ju, int nu, int nv,
                                              float E0, float E1, float hb, float zlo, float cv) {
    // the launch checks the grid's range of E1; this keeps every read in
    // bounds whatever the table holds
    if (!(E1 > 0.3f && E1 < 1.0f)) return;
    const float rE = __frcp_rn(E1);
    // first row at or above z0 - 1 (one correction for the rounded quotient)
    float vf = ceilf(fmaf(zlo - E0, rE, cv));
    if (!(fabsf(vf) < 1.0e7f)) return;
    float w = fmaf(vf - cv, E1, E0) - zlo;
    if (w < 0.0f) {
        vf += 1.0f;
        w += E1;
    } else if (w >= E1) {
        vf -= 1.0f;
        w -= E1;
    }
    const int vs = (int)vf;
    // rows read: those of heights [0, ZS + 1), at most (ZS + 1) / E1 + 1 (the
    // truncation below loses one), one more for the drift of the stepped
    // heights, two after the last that the unconditional slots may read, and
    // one spare
    constexpr int nrb_max = (int)((float)(ZS + 1) / BR_E1_LO) + 6;
    const int nrb = min(nrb_max, (int)((float)(ZS + 1) * rE) + 6);
    if (vs >= nv || vs + nrb <= 0) return;
    const int off = vs * nu + ju;
    if (vs >= 0 && vs + nrb <= nv) {
        if (E1 > BR_K2) br_column<ZS, 2, false>(acc, sv, off, nu, w, E1, hb, vs, nv);
        else br_column<ZS, 3, false>(acc, sv, off, nu, w, E1, hb, vs, nv);
    } else {
        if (E1 > BR_K2) br_column<ZS, 2, true>(acc, sv, off, nu, w, E1, hb, vs, nv);
        else br_column<ZS, 3, true>(acc, sv, off, nu, w, E1, hb, vs, nv);
    }
}

template <typename ST, int ZS>
__global__ void __launch_bounds__(BR_THREADS, 12)
    k_backproject_reg(BPArgs a, const float4 *__restrict__ cols, const ST *__restrict__ sino,
                      float *__restrict__ out, int accumulate) {
    const int tid = threadIdx.x;
    const int w = tid >> 5, l = tid & 31;
    const int jx = blockIdx.x * BR_TX + (w % (BR_TX / BR_WX)) * BR_WX + l % BR_WX;
    const int jy = blockIdx.y * BR_TY + (w / (BR_TX / BR_WX)) * BR_WY + l / BR_WX;
    // blockIdx.z = split * (z-slabs) + slab, as in k_backproject_slab
    const int zblocks = gridDim.z / a.splits;
    const int split = blockIdx.z / zblocks;
    const int z0 = (blockIdx.z - split * zblocks) * ZS;
    const int per = (a.nviews + a.splits - 1) / a.splits;
    const int i0 = split * per, i1 = min(a.nviews, i0 + per);
    if (jx >= a.n || jy >= a.n) return;
    float acc[ZS];
#pragma unroll
    for (int q = 0; q < ZS; ++q) acc[q] = 0.0f;
    const float ic = 0.5f * (float)(a.n - 1);
    const float cu = 0.5f * (float)(a.nu - 1), cv = 0.5f * (float)(a.nv - 1);
    const float cx = (float)jx - ic, cy = (float)jy - ic;
    const float zlo = (float)z0 - 1.0f;  // interval 0 starts here
    const size_t view_elems = (size_t)a.nu * a.nv;
    for (int i = i0; i < i1; ++i) {
        const int k = a.view0 + i * a.stride;
        const float *G = reinterpret_cast<const float *>(a.views + k);
        const float X = (float)jx - __ldg(G + 0), Y = (float)jy - __ldg(G + 1);
        const float Q0 = __ldg(G + 12), Q1 = __ldg(G + 13), Q6 = __ldg(G + 18), Q7 = __ldg(G + 19);
        const float q0 = fmaf(Q1, Y, Q0 * X), q2 = fmaf(Q7, Y, Q6 * X);
        // a column of x-major rays weights this voxel column iff its rays
        // cross the plane x = jx strictly between y = jy - 1 and jy + 1,
        // i.e. iff its u lies between the projections of those two
        // points; likewise (jx -+ 1, jy) for y-major rays.  Both intervals
        // hold the voxel column's own projection, so their union is the
        // interval from the least to the greatest of the four.
        const float ua = (q0 - Q1) * __frcp_rn(q2 - Q7), ub = (q0 + Q1) * __frcp_rn(q2 + Q7);
        const float uc = (q0 - Q0) * __frcp_rn(q2 - Q6), ud = (q0 + Q0) * __frcp_rn(q2 + Q6);
        const float umin = fminf(fminf(ua, ub), fminf(uc, ud)), umax = fmaxf(fmaxf(ua, ub), fmaxf(uc, ud));
        const int ulo = max(0, (int)ceilf(umin + cu - 1e-3f));
        const int uhi = min(a.nu - 1, (int)floorf(umax + cu + 1e-3f));
        const ST *__restrict__ sv = sino + (size_t)i * view_elems;
        const float4 *__restrict__ ct = cols + (size_t)k * a.nu * 2;
        for (int ju = ulo; ju <= uhi; ++ju) {
            const float4 t0 = __ldg(ct + 2 * ju);
            const float4 t1 = __ldg(ct + 2 * ju + 1);
            const bool ay = t0.x != 0.0f;
            const float ca = ay ? cy : cx, cb = ay ? cx : cy;
            const float hb = 1.0f - fabsf(fmaf(ca, t0.y, t0.z) - cb);
            if (hb <= 0.0f) continue;
            br_add_column<ZS>(acc, sv, ju, a.nu, a.nv, fmaf(ca, t1.x, t0.w) + ic, fmaf(ca, t1.z, t1.y), hb, zlo, cv);
        }
    }
    const size_t nvox = (size_t)a.n * a.n * a.n;
    float *o = out + (size_t)split * nvox;
#pragma unroll
    for (int zz = 0; zz < ZS; ++zz) {
        const int z = z0 + zz;
        if (z < a.n) {
            const size_t idx = ((size_t)z * a.n + jy) * a.n + jx;
            float v = acc[zz];
            if (accumulate) v += o[idx];
            o[idx] = v;
        }
    }
}

// Column table (see LevelInfo::d_cols): one thread per (view, column); the
// axis choice is the projector's own ray_dir() at v' = 0.
__global__ void k_column_table(const ViewGeom *__restrict__ views, int K, int nu, float4 *__restrict__ cols) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= K * nu) return;
    const int k = t / nu, ju = t % nu;
    const ViewGeom &G = views[k];
    const float up = (float)ju - 0.5f * (float)(nu - 1);
    const RayDir d = ray_dir(G, up, 0.0f);
    const float wa = d.ax ? d.wy : d.wx, wb = d.ax ? d.wx : d.wy;
    const float rinv = __frcp_rn(wa);
    const float *N = d.ax ? G.NY : G.NX;
    cols[2 * (size_t)t] = make_float4(d.ax ? 1.0f : 0.0f, wb * rinv, fmaf(up, N[1], N[0]) * rinv,
                                      fmaf(up, N[4], N[3]) * rinv);
    cols[2 * (size_t)t + 1] = make_float4(G.Wc[2] * rinv, N[5] * rinv, G.Ev[2] * rinv, 0.0f);
}

// Number of view ranges for a slab launch of `blocks` blocks: enough for
// about four waves of resident blocks in all, as grid 0 has (coarse grids and
// OS-EMTR subsets otherwise fill a fraction of the SMs, and a launch of one
// or two waves loses its tail), at most 16 and what `cap` floats of partial
// volumes hold.
template <typename KF>
int slab_splits(KF kernel, int blocks, int nviews, size_t vol_floats, size_t cap) {
    int dev = 0, sms = 0, occ = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, BS_THREADS, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    int sp = (4 * sms * occ + blocks - 1) / blocks;
    if (sp > 16) sp = 16;
    if (sp > nviews) sp = nviews;
    if ((size_t)sp * vol_floats > cap) sp = (int)(cap / vol_floats);
    return sp < 1 ? 1 : sp;
}

// The register kernel's launch (see k_backproject_reg), with the slab
// kernel's view splits.
template <typename ST>
int launch_backproject_reg(const LevelInfo &L, BPArgs a, const ST *sino, float *out, int accumulate, cudaStream_t s,
                           float *split_buf, size_t cap) {
    dim3 grid((L.n + BR_TX - 1) / BR_TX, (L.n + BR_TY - 1) / BR_TY, (L.n + BR_Z - 1) / BR_Z);
    const size_t vol_floats = (size_t)L.n * L.n * L.n;
    if (split_buf && a.nviews > 1)
        a.splits = slab_splits(k_backproject_reg<ST, BR_Z>, (int)(grid.x * grid.y * grid.z), a.nviews, vol_floats,
                               cap);
    if (a.splits == 1) {
        MGCT_KERNEL(KK_BACKPROJECT, s,
                    k_backproject_reg<ST, BR_Z><<<grid, BR_THREADS, 0, s>>>(a, L.d_cols, sino, out, accumulate));
    } else {
        grid.z *= a.splits;
        MGCT_KERNEL(KK_BACKPROJECT, s,
                    k_backproject_reg<ST, BR_Z><<<grid, BR_THREADS, 0, s>>>(a, L.d_cols, sino, split_buf, 0));
        const int sb = (int)((vol_floats + 255) / 256 < 4096 ? (vol_floats + 255) / 256 : 4096);
        MGCT_KERNEL(KK_BACKPROJECT, s, k_sum_splits<<<sb, 256, 0, s>>>(vol_floats, a.splits, split_buf, out, accumulate));
    }
    return MGCT_OK;
}

// A^T of a weighted sinogram stored [view][v][u].
template <int NCH, typename ST>
int launch_backproject_slab(const LevelInfo &L, BPArgs a, const ST *sino, float *out, int accumulate, cudaStream_t s,
                            float *split_buf, size_t cap) {
    if constexpr (sizeof(ST) == 2) {
        if (L.e1_lo > BR_E1_LO && L.e1_hi < BR_E1_HI && (size_t)L.nu * (L.nv + 64) < ((size_t)1 << 31))
            return launch_backproject_reg<ST>(L, a, sino, out, accumulate, s, split_buf, cap);
    }
    constexpr int Z = SlabCfg<NCH>::Z;
    constexpr bool DFA = sizeof(ST) != 2;
    const float4 *cols = DFA ? L.d_cols_df : L.d_cols;
    dim3 grid((L.n + BS_TX - 1) / BS_TX, (L.n + BS_TY - 1) / BS_TY, (L.n + Z - 1) / Z);
    const size_t vol_floats = (size_t)NCH * L.n * L.n * L.n;
    const int blocks = (int)(grid.x * grid.y * grid.z);
    if (split_buf && a.nviews > 1) {
        if constexpr (DFA) {
            // a share costs one view's work: a partial volume written and read
            int sms = 0, occ = 0;
            MGCT_TRY(sm_count(&sms));
            MGCT_TRY(check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                                    &occ, k_backproject_slab<NCH, ST, DFA>, BS_THREADS, 0), "occupancy"));
            a.splits = view_splits(sms, occ > 0 ? occ : 1, blocks, a.nviews,
                                   (int)(cap / vol_floats < 64 ? cap / vol_floats : 64), 1.0);
        } else {
            a.splits = slab_splits(k_backproject_slab<NCH, ST, DFA>, blocks, a.nviews, vol_floats, cap);
        }
    }
    grid.z *= a.splits;
    float *dst = a.splits > 1 ? split_buf : out;
    MGCT_KERNEL(KK_BACKPROJECT, s, k_backproject_slab<NCH, ST, DFA><<<grid, BS_THREADS, 0, s>>>(
                                       a, cols, sino, dst, a.splits > 1 ? 0 : accumulate));
    if (a.splits > 1) {
        const int sb = (int)((vol_floats + 255) / 256 < 4096 ? (vol_floats + 255) / 256 : 4096);
        if constexpr (DFA) {
            MGCT_KERNEL(KK_BACKPROJECT, s, k_sum_parts<<<sb, 256, 0, s>>>(vol_floats, a.splits, split_buf, out, accumulate));
        } else {
            MGCT_KERNEL(KK_BACKPROJECT, s, k_sum_splits<<<sb, 256, 0, s>>>(vol_floats, a.splits, split_buf, out, accumulate));
        }
    }
    return MGCT_OK;
}

}  // namespace mgct
