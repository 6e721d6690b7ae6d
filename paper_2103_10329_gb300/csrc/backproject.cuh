// Voxel-driven back-projector A^T with the exact transpose of the projector's
// weights (the back-projection B of Sec. 2.1 is the adjoint of P).
//
// For voxel j and view k, a detector pixel contributes iff its ray crosses
// the voxel-centre plane of j along the ray's major axis a within one voxel of
// j in both in-plane axes; the weight is the projector's
//   dl * hat(f_b - j_b) * hat(f_z - j_z),   hat(t) = max(0, 1 - |t|).
// Such a ray passes through the cube [j-1, j+1]^3 (index units), so the
// candidates are the pixels inside the cube's projected bounding box.  With
// q = Q (j - S) the voxel centre projects to (u0, v0) = (q0, q1) / q2, and for
// a cube offset delta in [-1, 1]^3,
//   |u(delta) - u0| <= |Q_0 - u0 Q_2|_1 / (q2 - |Q_2|_1),
// likewise for v, which bounds the box without projecting the eight corners.
// Each candidate takes its ray direction and major axis from the projector's
// own routine (bit-identical axis choice), and its crossing from the centred
// numerator form (no cancellation of source-distance terms), in float32: the
// per-weight rounding (~1e-6 voxel at n = 64) averages out over the ~9 K
// contributions a voxel receives.  One thread per voxel, looping over the
// views; the per-view tables of a view chunk sit in shared memory.  No
// atomics.
#pragma once

#include "common.cuh"
#include "project.cuh"

namespace mgct {

constexpr int BP_BX = 32, BP_BY = 4, BP_BZ = 2;
constexpr int BP_CHUNK = 64;  // views staged in shared memory at a time

struct BPArgs {
    const ViewGeom *views;
    int n, nu, nv;
    float h;
    int view0, stride, nviews;
    int splits;  // tile kernels: shares of the views, each into its own partial volume (1: none)
    int cls;     // tile kernels: the ray class (1: y-major), or -1 for both in one launch
};

template <int NCH, typename ST>
struct SinoLoad;
template <typename ST>
struct SinoLoad<1, ST> {
    static __device__ __forceinline__ void add(const ST *__restrict__ p, size_t idx, float w, float (&acc)[1]) {
        acc[0] = fmaf(w, to_f32(__ldg(p + idx)), acc[0]);
    }
};
template <>
struct SinoLoad<2, float2> {
    static __device__ __forceinline__ void add(const float2 *__restrict__ p, size_t idx, float w, float (&acc)[2]) {
        float2 y = __ldg(p + idx);
        acc[0] = fmaf(w, y.x, acc[0]);
        acc[1] = fmaf(w, y.y, acc[1]);
    }
};

// Adds A^T (one view) at voxel (jx, jy, jz) into acc -- any geometry.
// WEIGHTED: the sinogram already carries each ray's dl (see the projector's
// weighted epilogues), so the weight is hat * hat; otherwise dl is computed
// per pixel.  Sinograms are [view][v][u].  Each candidate ray is set up as
// the projector sets it up: direction, slopes and centred crossing in
// double-float from the view table's double-float fields (G must hold them),
// and the crossing's offset from the voxel, p + c_a r - c, formed in
// double-float before it is rounded -- in float32 alone the numerators'
// cancellation leaves ~1e-6 voxel, 1e-5 of a weight near a hat's edge.
template <int NCH, typename ST, bool WEIGHTED>
__device__ __forceinline__ void bp_view(const ViewGeom &G, const BPArgs &a, int jx, int jy, int jz,
                                        const ST *__restrict__ sino_view, float (&acc)[NCH]) {
    const float X = (float)jx - G.S[0], Y = (float)jy - G.S[1], Z = (float)jz - G.S[2];
    const float q0 = fmaf(G.Q[2], Z, fmaf(G.Q[1], Y, G.Q[0] * X));
    const float q1 = fmaf(G.Q[5], Z, fmaf(G.Q[4], Y, G.Q[3] * X));
    const float q2 = fmaf(G.Q[8], Z, fmaf(G.Q[7], Y, G.Q[6] * X));
    const float inv = 1.0f / q2;
    const float u0 = q0 * inv, v0 = q1 * inv;
    const float den = 1.0f / (q2 - G.m2);
    const float hu = (fabsf(G.Q[0] - u0 * G.Q[6]) + fabsf(G.Q[1] - u0 * G.Q[7]) + fabsf(G.Q[2] - u0 * G.Q[8])) * den;
    const float hv = (fabsf(G.Q[3] - v0 * G.Q[6]) + fabsf(G.Q[4] - v0 * G.Q[7]) + fabsf(G.Q[5] - v0 * G.Q[8])) * den;
    const float cu = 0.5f * (float)(a.nu - 1), cv = 0.5f * (float)(a.nv - 1);
    // small absolute margin covers float32 rounding of the bound itself
    int ulo = max(0, (int)ceilf(u0 - hu + cu - 1e-3f));
    int uhi = min(a.nu - 1, (int)floorf(u0 + hu + cu + 1e-3f));
    int vlo = max(0, (int)ceilf(v0 - hv + cv - 1e-3f));
    int vhi = min(a.nv - 1, (int)floorf(v0 + hv + cv + 1e-3f));
    // voxel centre relative to the volume centre (exact half-integers)
    const float ic = 0.5f * (float)(a.n - 1);
    const float cx = (float)jx - ic, cy = (float)jy - ic, cz = (float)jz - ic;
    for (int jv = vlo; jv <= vhi; ++jv) {
        const float vp = (float)jv - cv;
        for (int ju = ulo; ju <= uhi; ++ju) {
            const float up = (float)ju - cu;
            const RayDir d = ray_dir(G, up, vp);
            const int ia = d.ax, ib = 1 - d.ax;
            const DF wa = df_affine(G.Wc[ia], G.Wc_lo[ia], G.Eu[ia], G.Eu_lo[ia], G.Ev[ia], G.Ev_lo[ia], up, vp);
            const DF wb = df_affine(G.Wc[ib], G.Wc_lo[ib], G.Eu[ib], G.Eu_lo[ib], G.Ev[ib], G.Ev_lo[ib], up, vp);
            const DF wz = df_affine(G.Wc[2], G.Wc_lo[2], G.Eu[2], G.Eu_lo[2], G.Ev[2], G.Ev_lo[2], up, vp);
            const float *N = d.ax ? G.NY : G.NX;
            const float *Nl = d.ax ? G.NY_lo : G.NX_lo;
            const DF nb = df_affine(N[0], Nl[0], N[1], Nl[1], N[2], Nl[2], up, vp);
            const DF nz = df_affine(N[3], Nl[3], N[4], Nl[4], N[5], Nl[5], up, vp);
            const DF rb = df_div(wb, wa), rz = df_div(wz, wa);
            // centred crossing of this ray with the voxel's plane, minus the voxel
            const float ca = d.ax ? cy : cx, cb = d.ax ? cx : cy;
            const DF xb = df_add(df_div(nb, wa), df_mul_f(rb, ca));
            const DF xz = df_add(df_div(nz, wa), df_mul_f(rz, ca));
            const float eb = __fadd_rn(__fsub_rn(xb.hi, cb), xb.lo);
            const float ez = __fadd_rn(__fsub_rn(xz.hi, cz), xz.lo);
            const float hb = 1.0f - fabsf(eb);
            const float hz = 1.0f - fabsf(ez);
            if (hb > 0.0f && hz > 0.0f) {
                float w = hb * hz;
                if (!WEIGHTED) w *= sqrtf(fmaf(rz.hi, rz.hi, fmaf(rb.hi, rb.hi, 1.0f))) * a.h;
                SinoLoad<NCH, ST>::add(sino_view, (size_t)jv * a.nu + ju, w, acc);
            }
        }
    }
}

// Separable geometries (no detector tilt: e_u horizontal, e_v vertical).
// Then w_x, w_y and the major axis depend on u' only, the in-plane crossing
// error e_b depends on u' only, and the z error is linear in v':
//   e_z(v') = E0 + v' E1,  E0 = (n0_z + u' nu_z + c_a Wc_z)/w_a - c_z,
//                          E1 = (nv_z + c_a Ev_z)/w_a,
// so each detector column is set up once for the thread's ZB voxels of one
// z-column, and each voxel walks exactly the pixels where |e_z| < 1.
// The column's quantities come from the double-float column table, and
// both cancellations are done in double-float: e_b = pb + c_a rb - c_b, and
// the z error is anchored at the detector row v_a nearest the thread's
// voxels (E0 + v_a E1 - c_z, small), so that in float32 only small terms
// remain -- the sample weights stay accurate to ~1e-7 at any N.
template <int NCH, typename ST, bool WEIGHTED, int ZB>
__device__ __forceinline__ void bp_view_sep(const ViewGeom &G, const float4 *__restrict__ cols, const BPArgs &a,
                                            int jx, int jy, int jz0, const ST *__restrict__ sino_view,
                                            float (&acc)[ZB][NCH]) {
    const float X = (float)jx - G.S[0], Y = (float)jy - G.S[1];
    // with no tilt the u coordinate and depth of a point ignore its z
    const float q0 = fmaf(G.Q[1], Y, G.Q[0] * X);
    const float q2 = fmaf(G.Q[7], Y, G.Q[6] * X);
    const float u0 = q0 / q2;
    const float hu = (fabsf(G.Q[0] - u0 * G.Q[6]) + fabsf(G.Q[1] - u0 * G.Q[7])) / (q2 - G.m2);
    const float cu = 0.5f * (float)(a.nu - 1), cv = 0.5f * (float)(a.nv - 1);
    const int ulo = max(0, (int)ceilf(u0 - hu + cu - 1e-3f));
    const int uhi = min(a.nu - 1, (int)floorf(u0 + hu + cu + 1e-3f));
    const float ic = 0.5f * (float)(a.n - 1);
    const float cx = (float)jx - ic, cy = (float)jy - ic;
    const float zm = (float)jz0 - ic + 0.5f * (float)(ZB - 1);  // centre of the thread's voxels (exact)
    for (int ju = ulo; ju <= uhi; ++ju) {
        const float4 t0 = __ldg(cols + ju), t1 = __ldg(cols + a.nu + ju);
        const float4 t2 = __ldg(cols + 2 * a.nu + ju), t3 = __ldg(cols + 3 * a.nu + ju);
        const bool ay = t0.x != 0.0f;
        const float ca = ay ? cy : cx, cb = ay ? cx : cy;
        const DF eb = df_add(df_mul_f(DF{t0.y, t0.z}, ca), DF{t0.w, t1.x});
        const float hb = 1.0f - fabsf(__fadd_rn(__fsub_rn(eb.hi, cb), eb.lo));
        if (hb <= 0.0f) continue;
        const DF Eb = df_add(DF{t1.y, t1.z}, df_mul_f(DF{t1.w, t2.x}, ca));  // centred height at v' = 0
        const DF E1d = df_add(DF{t2.y, t2.z}, df_mul_f(DF{t2.w, t3.x}, ca));
        const float E1 = E1d.hi;
        const float va = rintf((zm - Eb.hi) / E1);  // anchor row (centred units)
        if (!(fabsf(va) < 1.0e7f)) continue;
        const DF c = df_add(df_add(Eb, df_mul_f(E1d, va)), DF{-zm, 0.0f});
        const float cf = c.hi + c.lo;  // z error at the anchor row for the centre voxel
        const float rE1 = 1.0f / E1;
#pragma unroll
        for (int zz = 0; zz < ZB; ++zz) {
            const float E0 = cf - ((float)zz - 0.5f * (float)(ZB - 1));
            const float s1 = (-1.0f - E0) * rE1, s2 = (1.0f - E0) * rE1;
            const int vlo = max(0, (int)ceilf(fminf(s1, s2) + va + cv - 1e-3f));
            const int vhi = min(a.nv - 1, (int)floorf(fmaxf(s1, s2) + va + cv + 1e-3f));
            for (int jv = vlo; jv <= vhi; ++jv) {
                const float vp = (float)jv - cv;
                const float hz = 1.0f - fabsf(fmaf(vp - va, E1, E0));
                if (hz > 0.0f) {
                    float w = hb * hz;
                    if (!WEIGHTED) {
                        const float rz = fmaf(vp, t2.w, t1.w);  // (Wc_z + u' Eu_z + v' Ev_z) / w_a
                        w *= sqrtf(fmaf(rz, rz, fmaf(t0.y, t0.y, 1.0f))) * a.h;
                    }
                    SinoLoad<NCH, ST>::add(sino_view, (size_t)jv * a.nu + ju, w, acc[zz]);
                }
            }
        }
    }
}

// NF: floats of each table staged (VG_HI: the float32 part; 64: all of it)
template <typename ST, int NF = VG_HI>
__device__ __forceinline__ void stage_views(ViewGeom *Gs, const BPArgs &a, int c0, int cn, int tid, int nthreads) {
    for (int t = tid; t < cn * NF; t += nthreads) {
        const int vi = t / NF, e = t % NF;
        reinterpret_cast<float *>(&Gs[vi])[e] =
            __ldg(reinterpret_cast<const float *>(a.views + a.view0 + (c0 + vi) * a.stride) + e);
    }
}

template <int NCH, typename ST, bool WEIGHTED>
__global__ void __launch_bounds__(BP_BX *BP_BY *BP_BZ)
    k_backproject(BPArgs a, const ST *__restrict__ sino, float *__restrict__ out, int accumulate) {
    __shared__ ViewGeom Gs[BP_CHUNK];
    const int jx = blockIdx.x * BP_BX + threadIdx.x;
    const int jy = blockIdx.y * BP_BY + threadIdx.y;
    const int jz = blockIdx.z * BP_BZ + threadIdx.z;
    const bool active = jx < a.n && jy < a.n && jz < a.n;
    const int tid = threadIdx.x + BP_BX * (threadIdx.y + BP_BY * threadIdx.z);
    float acc[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) acc[c] = 0.0f;
    const size_t view_elems = (size_t)a.nu * a.nv;
    for (int c0 = 0; c0 < a.nviews; c0 += BP_CHUNK) {
        const int cn = min(BP_CHUNK, a.nviews - c0);
        __syncthreads();
        stage_views<ST, sizeof(ViewGeom) / 4>(Gs, a, c0, cn, tid, BP_BX * BP_BY * BP_BZ);
        __syncthreads();
        if (active) {
            for (int vi = 0; vi < cn; ++vi)
                bp_view<NCH, ST, WEIGHTED>(Gs[vi], a, jx, jy, jz, sino + (size_t)(c0 + vi) * view_elems, acc);
        }
    }
    if (!active) return;
    const size_t idx = ((size_t)jz * a.n + jy) * a.n + jx;
    const size_t nvox = (size_t)a.n * a.n * a.n;
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        float v = acc[c];
        if (accumulate) v += out[idx + c * nvox];
        out[idx + c * nvox] = v;
    }
}

constexpr int BPS_ZB = 4;  // voxels per thread along z (separable kernel)

template <int NCH, typename ST, bool WEIGHTED>
__global__ void __launch_bounds__(BP_BX *BP_BY *BP_BZ)
    k_backproject_sep(BPArgs a, const float4 *__restrict__ cols, const ST *__restrict__ sino, float *__restrict__ out,
                      int accumulate) {
    __shared__ ViewGeom Gs[BP_CHUNK];
    const int jx = blockIdx.x * BP_BX + threadIdx.x;
    const int jy = blockIdx.y * BP_BY + threadIdx.y;
    const int jz0 = (blockIdx.z * BP_BZ + threadIdx.z) * BPS_ZB;
    const bool active = jx < a.n && jy < a.n && jz0 < a.n;
    const int tid = threadIdx.x + BP_BX * (threadIdx.y + BP_BY * threadIdx.z);
    float acc[BPS_ZB][NCH];
#pragma unroll
    for (int z = 0; z < BPS_ZB; ++z)
#pragma unroll
        for (int c = 0; c < NCH; ++c) acc[z][c] = 0.0f;
    const size_t view_elems = (size_t)a.nu * a.nv;
    for (int c0 = 0; c0 < a.nviews; c0 += BP_CHUNK) {
        const int cn = min(BP_CHUNK, a.nviews - c0);
        __syncthreads();
        stage_views<ST>(Gs, a, c0, cn, tid, BP_BX * BP_BY * BP_BZ);
        __syncthreads();
        if (active) {
            for (int vi = 0; vi < cn; ++vi)
                bp_view_sep<NCH, ST, WEIGHTED, BPS_ZB>(Gs[vi], cols + (size_t)(a.view0 + (c0 + vi) * a.stride) * a.nu * 4,
                                                       a, jx, jy, jz0,
                                                       sino + (size_t)(c0 + vi) * view_elems, acc);
        }
    }
    if (!active) return;
    const size_t nvox = (size_t)a.n * a.n * a.n;
#pragma unroll
    for (int z = 0; z < BPS_ZB; ++z) {
        if (jz0 + z >= a.n) break;
        const size_t idx = ((size_t)(jz0 + z) * a.n + jy) * a.n + jx;
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            float v = acc[z][c];
            if (accumulate) v += out[idx + c * nvox];
            out[idx + c * nvox] = v;
        }
    }
}

// Separable geometries, weighted sinogram stored [view][u][v] (rows
// contiguous) with SINO_PAD zero rows before and after every column: the
// solver's A^T and, after k_weight_rays, the public one.
//
// A warp owns W voxel columns of one voxel-centre plane -- consecutive along
// the plane's in-plane axis b -- over ZT heights, its lanes the heights (lane
// l: z0 + l, z0 + 32 + l, ...).  The rays of one detector column cross the
// plane at one in-plane position b, so the column's z profile there,
//   g(z) = sum over rows of y hat(f_z(row) - z),
// is computed once, by all lanes together, and added with the weights
// (1 - t_b, t_b) to the two voxel columns jb and jb + 1 it falls between: no
// lane waits for another's columns, and the rows a warp reads are one
// contiguous run.  Columns of y-major rays take the planes y = const, those
// of x-major rays the planes x = const, in blocks of their own (two partial
// volumes added afterwards, or two launches where there is no room for them).
//
// Detector columns are taken 32 at a time, across views, a lane per column:
// the lane sets up everything that depends on (view, plane, column) alone, in
// double-float, and the warp sorts the 32 by jb (counting sort) into a table
// that the profile loop reads by broadcast.  The two voxel columns of the
// current jb stay in registers; the tile's others in shared memory.
//
// The row heights are anchored at the detector row nearest the tile's middle
// height and formed with one rounding each (ri E - z exactly fused), so a
// weight is accurate to ~1e-7 at any N.  Lane z's rows start at
// ri = ceil((z - 1 - E0) / E): that row's weight is its height above z - 1,
// the following ones' 1 - |height - z|, as long as the height stays below
// z + 1 (rows beyond are not loaded).
//
// Bound by issue slots and L1 wavefronts alike (profile at 256^3 / 144 views:
// 69 % issue-active, 73 % L1; 34 instructions and 9 wavefronts per column,
// plane and 32 heights, of which the profile's 3 or 4 row loads are 6
// wavefronts).  A thread per voxel column, as before, computed every profile
// twice, at 68 instructions, with lanes waiting for each other's columns.
constexpr int BT_WARPS = 8;   // planes per block
constexpr float BT_MAGIC = 12582912.0f;  // 1.5 * 2^23: ceil(x) in the low mantissa bits of x + BT_MAGIC rounded up
constexpr int BT_MAGIC_BITS = 0x4B400000;

// One detector column at one plane.  The rows of a height zl above the tile's
// middle start at ceil(fma(zl, rE, -d1 rE)), counted from the anchor row.
struct __align__(16) ColEntry {
    float E, Elo;     // E + Elo: height step per row
    float d1, rE;     // 1 + height of the anchor row; 1 / E
    long long base;   // element of the anchor row in the sinogram, less BT_MAGIC_BITS
    float tb;         // fraction along b
    float rlo;        // the first readable row, -SINO_PAD, from the anchor, plus BT_MAGIC
};

// NP: pairs of values a lane holds, two heights of one channel or the two
// channels of one height; W: voxel columns per warp.  Measured, public call at
// 256^3 / 720 views: W = 8 with two pairs and 24 resident warps, or one pair
// and 32, 22.0 ms; one pair and 24 warps 23.9; 16 columns with two pairs 25.6
// (its accumulators leave half the L1), with one 23.4; the slab kernel that
// this one replaced 52.0, the solver's register kernel 29.5 (22.0 here).
template <int NCH, int NP>
struct PlaneTile {
    static constexpr int ZT = NCH == 2 ? 32 * NP : 64 * NP, ZP = ZT + 1;
    static constexpr int W = 8;
    static constexpr int MIN_BLOCKS = NP == 2 ? 3 : 4;  // 80 and 64 registers
    static constexpr size_t acc_floats = (size_t)BT_WARPS * W * NCH * ZP;
    static constexpr size_t smem = sizeof(ColEntry) * 32 * BT_WARPS + sizeof(float) * acc_floats;
};

// packed float pairs (one instruction each)
__device__ __forceinline__ float2 add_up_f2(float2 a, float2 b) {  // rounded toward plus infinity
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "add.rp.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 mul_f2(float2 a, float2 b) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mul.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return d;
}
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

// A load where `w` is positive, 0 elsewhere (nothing read).
__device__ __forceinline__ float ld_if(const float *p, float w) {
    float v;
    asm("{\n\t.reg .pred q;\n\tsetp.gt.f32 q, %2, 0f00000000;\n\tmov.f32 %0, 0f00000000;\n\t"
        "@q ld.global.nc.f32 %0, [%1];\n\t}"
        : "=f"(v)
        : "l"(p), "f"(w));
    return v;
}
// Row s of a lane's pair, with (w) or without a weight that has to be positive.
__device__ __forceinline__ float2 bt_row(const float *pa, const float *pb, int s) {
    return make_float2(__ldg(pa + s), __ldg(pb + s));
}
__device__ __forceinline__ float2 bt_row(const float2 *pa, const float2 *, int s) { return __ldg(pa + s); }
__device__ __forceinline__ float2 bt_row(const float *pa, const float *pb, int s, float2 w) {
    return make_float2(ld_if(pa + s, w.x), ld_if(pb + s, w.y));
}
__device__ __forceinline__ float2 bt_row(const float2 *pa, const float2 *, int s, float2 w) {
    float2 v;
    asm("{\n\t.reg .pred q;\n\tsetp.gt.f32 q, %3, 0f00000000;\n\tmov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\t"
        "@q ld.global.nc.v2.f32 {%0, %1}, [%2];\n\t}"
        : "=f"(v.x), "=f"(v.y)
        : "l"(pa + s), "f"(w.x));
    return v;
}

// Profile at one height of any column, rows off the detector reading as zero;
// v: the height's first row, col: the column's row 0.
template <typename ST>
__device__ __forceinline__ float2 bt_profile_any(const ST *__restrict__ col, int v, int nv, float g, float E) {
    float2 a = make_float2(0.0f, 0.0f);
    for (int s = 0; v < nv; ++s, ++v) {
        const float h = fmaf((float)s, E, g) - 1.0f;
        if (!(h < 1.0f)) break;
        if (v < 0) continue;
        a = fma_f2(both(1.0f - fabsf(h)), bt_row(col, col, v), a);
    }
    return a;
}

// First row m of a pair of heights zl, as a number at BT_MAGIC, and 1 + (its
// height - zl).
__device__ __forceinline__ float2 bt_start(const ColEntry &t, float2 zl, float2 &m) {
    m = add_up_f2(fma_f2(zl, both(t.rE), both(-t.d1 * t.rE)), both(BT_MAGIC));
    const float2 ri = add_f2(m, both(-BT_MAGIC));
    return add_f2(fma_f2(ri, both(t.E), make_float2(-zl.x, -zl.y)), fma_f2(ri, both(t.Elo), both(t.d1)));
}

// Profile of table entry t at the pair zl of heights from ROWS rows: 3 or 4
// where 2/3 < E < 1 or 1/2 < E < 1, 5 for any E > 0.4.  Rows off the detector
// are the sinogram's zero rows: a start is clamped to those before and after
// the column, without a change of the weights.
template <int ROWS, int NCH, typename ST>
__device__ __forceinline__ float2 bt_profile(const ColEntry &t, const ST *__restrict__ anchor, float rspan, float2 zl) {
    // a second channel takes the first one's weights
    auto pair = [](float2 w) { return NCH == 2 ? make_float2(w.x, w.x) : w; };
    float2 m;
    const float2 g = bt_start(t, zl, m);
    const float rhi = t.rlo + rspan;
    const ST *pa = anchor + __float_as_int(fminf(fmaxf(m.x, t.rlo), rhi));
    const ST *pb = anchor + __float_as_int(fminf(fmaxf(m.y, t.rlo), rhi));
    if (ROWS < 5) {
        // the first two rows lie below z + 1 whatever g (g < E < 1); from the
        // third on the height is above z (2 E > 1)
        const float2 h1 = add_f2(g, both(t.E - 1.0f));
        const float2 w1 = make_float2(1.0f - fabsf(h1.x), 1.0f - fabsf(h1.y));
        const float2 w2 = fma_f2(g, both(-1.0f), both(fmaf(-2.0f, t.E, 2.0f)));
        const float2 y0 = bt_row(pa, pb, 0), y1 = bt_row(pa, pb, 1), y2 = bt_row(pa, pb, 2, w2);
        float2 p = mul_f2(pair(g), y0);
        if (ROWS == 4) {
            const float2 w3 = fma_f2(g, both(-1.0f), both(fmaf(-3.0f, t.E, 2.0f)));
            p = fma_f2(pair(w3), bt_row(pa, pb, 3, w3), p);
        }
        p = fma_f2(pair(w1), y1, p);
        return fma_f2(pair(w2), y2, p);
    }
    float2 h = add_f2(g, both(-1.0f)), p = both(0.0f);
#pragma unroll
    for (int s = 0; s < ROWS; ++s) {
        const float2 w = make_float2(1.0f - fabsf(h.x), 1.0f - fabsf(h.y));
        // beyond the second row often no lane has any (E >= 1)
        if (s < 2 || __any_sync(0xffffffffu, fmaxf(w.x, w.y) > 0.0f)) p = fma_f2(pair(w), bt_row(pa, pb, s, w), p);
        h = add_f2(h, both(t.E));
    }
    return p;
}

// The same for any E, row by row; nv: the detector's rows.
template <int NCH, typename ST>
__device__ __forceinline__ float2 bt_profile_loop(const ColEntry &t, const ST *__restrict__ anchor, int nv, float2 zl) {
    float2 m;
    const float2 g = bt_start(t, zl, m);
    const int row0 = __float_as_int(t.rlo) + SINO_PAD;  // the detector's row 0, as the rows' bits
    const ST *col = anchor + row0;
    float2 p = bt_profile_any(col, __float_as_int(m.x) - row0, nv, g.x, t.E);
    if (NCH == 1) p.y = bt_profile_any(col, __float_as_int(m.y) - row0, nv, g.y, t.E).x;
    return p;
}

template <int NCH, int NP, typename ST>
__global__ void __launch_bounds__(32 * BT_WARPS, PlaneTile<NCH, NP>::MIN_BLOCKS)
    k_backproject_plane(BPArgs a, const float4 *__restrict__ cols, const int2 *__restrict__ ranges,
                        const ST *__restrict__ sino, float *__restrict__ out, int accumulate) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using T = PlaneTile<NCH, NP>;
    constexpr int ZT = T::ZT, ZP = T::ZP, W = T::W;
    constexpr unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    ColEntry *tab = reinterpret_cast<ColEntry *>(smem_raw) + 32 * warp;
    float *acc = reinterpret_cast<float *>(smem_raw + sizeof(ColEntry) * 32 * BT_WARPS);  // [warp][W][NCH][ZP]
    // blockIdx.z = part * (z tiles) + tile; part = class * splits + split where
    // both classes run in one launch; split s takes views [i0, i1), and part q
    // writes partial volume q of `out`
    const int parts = a.splits * (a.cls < 0 ? 2 : 1);
    const int ztiles = gridDim.z / parts;
    const int part = blockIdx.z / ztiles;
    const int z0 = (blockIdx.z - part * ztiles) * ZT;
    const int cls = a.cls < 0 ? part / a.splits : a.cls;
    const int split = part - (a.cls < 0 ? cls * a.splits : 0);
    const int per = (a.nviews + a.splits - 1) / a.splits;
    const int i0 = split * per, i1 = min(a.nviews, i0 + per);
    // this warp's plane (of axis y for class 1, x for class 0), the tile's first
    // voxel along b and its width
    const int p0 = blockIdx.y * BT_WARPS, pl = p0 + warp, b0 = blockIdx.x * W;
    const int wb = min(W, a.n - b0);
    const float ic = 0.5f * (float)(a.n - 1);
    const float cu = 0.5f * (float)(a.nu - 1), cv = 0.5f * (float)(a.nv - 1);
    const float ca = (float)pl - ic, cb0 = (float)b0 - ic;
    const float zc = (float)(z0 + ZT / 2) - ic;  // the tile's middle height, centred (exact)
    float2 zl[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const float z = (float)(lane - ZT / 2 + i * (ZT / NP));
        zl[i] = make_float2(z, NCH == 2 ? z : z + 32.0f);
    }
    const float rspan = (float)(a.nv + SINO_PAD);  // from the first to the last readable start
    for (int t = tid; t < (int)T::acc_floats; t += 32 * BT_WARPS) acc[t] = 0.0f;
    __syncthreads();
    float *const accw = acc + warp * W * NCH * ZP + lane;

    for (int ib = i0; ib < i1 && pl < a.n; ib += 32) {
        // lane = view: the detector columns of this class whose rays cross the
        // plane strictly between voxels b0 - 1 and b0 + wb, i.e. between the
        // projections of those two points (with a margin far above their
        // rounding; the exact test is the column's own)
        int vlo = 0, cnt = 0;
        if (ib + lane < i1) {
            const int k = a.view0 + (ib + lane) * a.stride;
            const float *G = reinterpret_cast<const float *>(a.views + k);
            const float Sx = __ldg(G + 0), Sy = __ldg(G + 1);
            const float Q0 = __ldg(G + 12), Q1 = __ldg(G + 13), Q6 = __ldg(G + 18), Q7 = __ldg(G + 19);
            const float Xa = (float)(cls ? b0 - 1 : pl) - Sx, Ya = (float)(cls ? pl : b0 - 1) - Sy;
            const float db = (float)(wb + 1);
            const float qa0 = fmaf(Q1, Ya, Q0 * Xa), qa2 = fmaf(Q7, Ya, Q6 * Xa);
            const float qb0 = fmaf(cls ? Q0 : Q1, db, qa0), qb2 = fmaf(cls ? Q6 : Q7, db, qa2);
            const float ua = qa0 / qa2 + cu, ub = qb0 / qb2 + cu;
            const int2 r = __ldg(ranges + 2 * k + cls);
            vlo = max(r.x, (int)ceilf(fminf(ua, ub) - 1e-2f));
            cnt = max(0, min(r.y, (int)floorf(fmaxf(ua, ub) + 1e-2f)) - vlo + 1);
        }
        // inclusive prefix sums: the views' columns as one list of `total`
        int pre = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, pre, o);
            if (lane >= o) pre += v;
        }
        const int total = __shfl_sync(FULL, pre, 31);
        for (int first = 0; __any_sync(FULL, first < total); first += 32) {
            // lane = column `first + lane` of the list: its view is the number
            // of views that end at or before it
            const int idx = first + lane;
            int v = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(FULL, pre, v + o - 1) <= idx) v += o;
            const int ju = __shfl_sync(FULL, vlo, v & 31) + idx - __shfl_sync(FULL, pre - cnt, v & 31);
            const int i = ib + v;
            int jb = -2;  // not in the tile
            int rows = 0, on = 0;  // rows of a height (0: any number), pairs of heights with rows on the detector
            ColEntry te;
            if (idx < total) {
                const float4 *c = cols + (size_t)(a.view0 + i * a.stride) * 4 * a.nu + ju;
                const float4 t0 = __ldg(c), t1 = __ldg(c + a.nu), t2 = __ldg(c + 2 * a.nu), t3 = __ldg(c + 3 * a.nu);
                const DF rb{t0.y, t0.z}, pb{t0.w, t1.x}, ez0{t1.y, t1.z}, ezc{t1.w, t2.x}, e10{t2.y, t2.z},
                    e1c{t2.w, t3.x};
                float tb;
                split_coord(df_add(df_add(df_mul_f(rb, ca), pb), DF{-cb0, 0.0f}), jb, tb);
                const DF E0 = df_add(ez0, df_mul_f(ezc, ca));  // centred height at v' = 0
                const DF E1 = df_add(e10, df_mul_f(e1c, ca));
                const float E = E1.hi, rE = __frcp_rn(E);
                const float jf = rintf(fmaf(zc - E0.hi, rE, cv));  // anchor row: nearest the middle height
                const DF ha = df_add(df_add(E0, df_mul_f(E1, jf - cv)), DF{-zc, 0.0f});
                const float d1 = __fadd_rn(ha.hi, 1.0f) + ha.lo;
                const float c0 = -d1 * rE;
                // the row a height starts at: the very expression the lanes
                // evaluate, monotone in z
                auto row = [&](float z) { return __fadd_ru(__fmaf_rn(z, rE, c0), BT_MAGIC) - BT_MAGIC; };
                const float r0 = -jf, rend = (float)a.nv - jf;  // the detector's rows, from the anchor
                constexpr int ZS = ZT / NP;  // heights of a pair of the lanes
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const float rf = row((float)(-ZT / 2 + q * ZS)), rl = row((float)(-ZT / 2 + (q + 1) * ZS - 1));
                    if (fabsf(rf) < 1.0e6f && fabsf(rl) < 1.0e6f && rf < rend && rl + 2.0f * rE + 2.0f > r0) on |= 1 << q;
                }
                if (!((t0.x != 0.0f) == (cls != 0) && jb >= -1 && jb < wb && !(jb < 0 && tb == 0.0f) && E > 0.0f &&
                      fabsf(jf) < 1.0e6f && on))
                    jb = -2;
                rows = E > 0.501f && E < 1.0f ? (E > 0.667f ? 3 : 4) : (E > 0.401f ? 5 : 0);
                te.E = E;
                te.Elo = E1.lo;
                te.d1 = d1;
                te.rE = rE;
                te.base = (long long)(SINO_PAD + ((size_t)i * a.nu + ju) * (a.nv + SINO_PAD)) +
                          (long long)((int)jf - BT_MAGIC_BITS);
                te.tb = tb;
                te.rlo = BT_MAGIC + (r0 - (float)SINO_PAD);
            }
            auto sweep = [&](auto ltag) {
                constexpr bool LOOP = decltype(ltag)::value;
                const int key = (rows == 0) == LOOP ? jb : -2;
                if (!__any_sync(FULL, key >= -1)) return;
                // counting sort by jb
                int run = 0, at = 0;
#pragma unroll
                for (int j = -1; j < W; ++j) {
                    const unsigned g = __ballot_sync(FULL, key == j);
                    if (key == j) at = run + __popc(g & ((1u << lane) - 1u));
                    run += __popc(g);
                }
                if (key >= -1) tab[at] = te;
                __syncwarp();
                // bit masks over the table: entries of 3 rows, of 4, and of pair q
                const unsigned bit = key >= -1 ? 1u << at : 0u;
                unsigned m3 = __reduce_or_sync(FULL, rows == 3 ? bit : 0u), m4 = __reduce_or_sync(FULL, rows == 4 ? bit : 0u);
                unsigned mq[NP];
#pragma unroll
                for (int q = 0; q < NP; ++q) mq[q] = __reduce_or_sync(FULL, (on >> q) & 1 ? bit : 0u);
                float2 lo[NP], hi[NP];  // voxel columns j and j + 1
#pragma unroll
                for (int q = 0; q < NP; ++q) lo[q] = hi[q] = both(0.0f);
                const ColEntry *t = tab;
                float *dst = accw - NCH * ZP;
#pragma unroll 1
                for (int j = -1; j < W; ++j) {
                    const int ng = __popc(__ballot_sync(FULL, key == j));
#pragma unroll 1
                    for (int e = 0; e < ng; ++e, ++t) {
                        const ColEntry c = *t;
                        const ST *anchor = sino + c.base;
                        float2 p[NP];
#pragma unroll
                        for (int q = 0; q < NP; ++q) p[q] = both(0.0f);
                        auto each = [&](auto f) {
#pragma unroll
                            for (int q = 0; q < NP; ++q)
                                if (NP == 1 || (mq[q] & 1u)) p[q] = f(zl[q]);
                        };
                        if (LOOP) each([&](float2 z) { return bt_profile_loop<NCH>(c, anchor, a.nv, z); });
                        else if (m3 & 1u) each([&](float2 z) { return bt_profile<3, NCH>(c, anchor, rspan, z); });
                        else if (m4 & 1u) each([&](float2 z) { return bt_profile<4, NCH>(c, anchor, rspan, z); });
                        else each([&](float2 z) { return bt_profile<5, NCH>(c, anchor, rspan, z); });
                        m3 >>= 1;
                        m4 >>= 1;
#pragma unroll
                        for (int q = 0; q < NP; ++q) mq[q] >>= 1;
                        const float wl = 1.0f - c.tb;
#pragma unroll
                        for (int q = 0; q < NP; ++q) {
                            lo[q] = fma_f2(both(wl), p[q], lo[q]);
                            if (c.tb > 0.0f) hi[q] = fma_f2(both(c.tb), p[q], hi[q]);
                        }
                    }
                    if (j >= 0) {
#pragma unroll
                        for (int q = 0; q < NP; ++q) {
                            float *d = dst + q * (ZT / NP);
                            d[0] += lo[q].x;
                            d[NCH == 2 ? ZP : 32] += lo[q].y;
                        }
                    }
                    dst += NCH * ZP;
#pragma unroll
                    for (int q = 0; q < NP; ++q) {
                        lo[q] = hi[q];
                        hi[q] = both(0.0f);
                    }
                }
                __syncwarp();
            };
            sweep(std::false_type());
            sweep(std::true_type());
        }
    }
    // the block's BT_WARPS planes x W columns, the volume's rows in runs of W
    // (class 1) or BT_WARPS (class 0) voxels
    __syncthreads();
    const size_t nvox = (size_t)a.n * a.n * a.n;
    float *o = out + (size_t)part * NCH * nvox;
    for (int t = tid; t < BT_WARPS * W * ZT; t += 32 * BT_WARPS) {
        const int c = t % (BT_WARPS * W), zz = t / (BT_WARPS * W), z = z0 + zz;
        const int w = cls ? c / W : c % BT_WARPS, j = cls ? c % W : c / BT_WARPS;
        const int x = cls ? b0 + j : p0 + w, y = cls ? p0 + w : b0 + j;
        if (x < a.n && y < a.n && z < a.n) {
            const size_t idx = ((size_t)z * a.n + y) * a.n + x;
#pragma unroll
            for (int q = 0; q < NCH; ++q) {
                float v = acc[((w * W + j) * NCH + q) * ZP + zz];
                if (accumulate) v += o[idx + q * nvox];
                o[idx + q * nvox] = v;
            }
        }
    }
}

// Tilted detectors (turned about their normal by up to TILT_MAX), weighted
// sinogram stored [view][u][v].  As in the plane kernel a warp owns W voxel
// columns of one voxel-centre plane over 32 heights, its lanes the heights, and
// takes the detector columns 32 at a time, a lane per column for their set-up.
// With tilt a column's rays cross the plane at positions b that drift with the
// row, so each lane finds its own voxel columns and adds to them in shared
// memory (no other lane has its height).
//
// At fixed plane and column both coordinates of the crossing are quotients of
// affine functions of the row with the same denominator w_a.  With r rows from
// the anchor row (nearest the tile's middle height), k = Ev_a / w_a and
// s = r / (1 + k r) = r + d,
//   z = z_A + s sz,   b = b_A + s sb,
// where z_A, b_A and both slopes come from the view table in double-float and
// d = -k r^2 / (1 + k r) is a small correction: the height above a lane's z and
// the distance from a voxel column keep their digits (r sz - z and r sb - j in
// one rounding, z and j whole numbers), both errors are below 2.5e-7 voxel (5e-8
// and 3e-8 rms; b as one float from the tile's edge: 1.4e-6 and 3.5e-7).  A
// lane's first row is the ceiling of the inverse, r = s / (1 - k s), at height
// z - 1.
//
// A height's tent holds at most 4 rows where sz > 1/2, and these fall into at
// most 3 neighbouring voxel columns where 3 sb < 1: a lane adds 3 sums per
// column.  5 rows with a test of each ray's major axis serve sz > 0.4 and
// columns that hold rays of both classes; other steps and strong drifts go
// row by row, each ray set up in double-float as the projector sets it up.
//
// The per-voxel gather (k_backproject), which does that for every candidate
// pixel of a voxel, took 128 ms at 128^3 / 192^2 / 360 views (about 6000
// instructions a voxel, view and warp); this kernel 5.7 ms, bound by issue.
template <int NCH>
struct TiltTile {
    static constexpr int W = NCH == 2 ? 8 : 16, ZT = 32, ZP = ZT + 1;
    static constexpr int ROWS = W + 4;  // voxel columns b0 - 2 .. b0 + W + 1 (the outer ones are dropped)
};

struct __align__(16) TiltEntry {
    float sz, szlo;   // height step per row at the anchor
    float d1, rz;     // 1 + height of the anchor row above the tile's middle; 1 / sz
    float k;          // Ev_a / w_a
    float sb, sblo;   // sb + sblo: step along b per row at the anchor
    float bA;         // anchor row's b from the voxel column jA of the tile
    int jA, jv;       // that column, the nearest; anchor row
    long long base;   // element of the column's row 0
    int i, ju;        // view of the batch and column
};

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float2 tl_row(const float *p, float w) { return make_float2(ld_if(p, w), 0.0f); }
__device__ __forceinline__ float2 tl_row(const float2 *p, float w) { return bt_row(p, p, 0, both(w)); }

// Which classes the rays of a detector column may have (bit 0: x-major, bit 1:
// y-major): y-major where (w_y - w_x) (w_y + w_x) > 0, both factors affine in
// the row; both classes where a factor changes sign over the detector or
// comes within rounding of 0, otherwise the projector's own choice.
__device__ __forceinline__ int column_classes(const ViewGeom &G, float up, float cv) {
    const RayDir d0 = ray_dir(G, up, -cv), d1 = ray_dir(G, up, cv);
    const float eps = 1e-5f * (fabsf(d0.wx) + fabsf(d0.wy) + fabsf(d1.wx) + fabsf(d1.wy));
    const float a0 = d0.wy - d0.wx, a1 = d1.wy - d1.wx, b0 = d0.wy + d0.wx, b1 = d1.wy + d1.wx;
    const bool same = (fminf(a0, a1) > eps || fmaxf(a0, a1) < -eps) && (fminf(b0, b1) > eps || fmaxf(b0, b1) < -eps);
    return same ? 1 << d0.ax : 3;
}

// A ray's crossing of the plane at c_a of its axis ax, centred, and 1 / w_a, in
// double-float from the projector's own quantities.
__device__ __forceinline__ void ray_crossing(const ViewGeom &G, int ax, float up, float vp, float ca, DF &xb, DF &xz,
                                             DF &rwa) {
    const int ib = 1 - ax;
    const DF wa = df_affine(G.Wc[ax], G.Wc_lo[ax], G.Eu[ax], G.Eu_lo[ax], G.Ev[ax], G.Ev_lo[ax], up, vp);
    const DF wb = df_affine(G.Wc[ib], G.Wc_lo[ib], G.Eu[ib], G.Eu_lo[ib], G.Ev[ib], G.Ev_lo[ib], up, vp);
    const DF wz = df_affine(G.Wc[2], G.Wc_lo[2], G.Eu[2], G.Eu_lo[2], G.Ev[2], G.Ev_lo[2], up, vp);
    const float *N = ax ? G.NY : G.NX, *Nl = ax ? G.NY_lo : G.NX_lo;
    const DF nb = df_affine(N[0], Nl[0], N[1], Nl[1], N[2], Nl[2], up, vp);
    const DF nz = df_affine(N[3], Nl[3], N[4], Nl[4], N[5], Nl[5], up, vp);
    rwa = df_div(DF{1.0f, 0.0f}, wa);
    xb = df_mul(df_add(nb, df_mul_f(wb, ca)), rwa);
    xz = df_mul(df_add(nz, df_mul_f(wz, ca)), rwa);
}

template <int NCH, typename ST>
__global__ void __launch_bounds__(32 * BT_WARPS, 3)
    k_backproject_tilt(BPArgs a, const int2 *__restrict__ ranges, const ST *__restrict__ sino, float *__restrict__ out,
                       int accumulate) {
    using T = TiltTile<NCH>;
    constexpr int W = T::W, ZT = T::ZT, ZP = T::ZP;
    __shared__ TiltEntry tabs[BT_WARPS][32];
    __shared__ float acc[BT_WARPS][NCH][T::ROWS][ZP];
    constexpr unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // parts, classes, planes and tiles as in k_backproject_plane
    const int parts = a.splits * (a.cls < 0 ? 2 : 1);
    const int ztiles = gridDim.z / parts;
    const int part = blockIdx.z / ztiles;
    const int z0 = (blockIdx.z - part * ztiles) * ZT;
    const int cls = a.cls < 0 ? part / a.splits : a.cls;
    const int split = part - (a.cls < 0 ? cls * a.splits : 0);
    // a split takes every splits-th view, so that each has its share of both
    // classes whatever order the views come in: 48^3 / 60 views around a circle
    // 185 -> 129 us, 64^3 / 90 views 304 -> 264 us against ranges of views
    const int p0 = blockIdx.y * BT_WARPS, pl = p0 + warp, b0 = blockIdx.x * W;
    const float ic = 0.5f * (float)(a.n - 1);
    const float cu = 0.5f * (float)(a.nu - 1), cv = 0.5f * (float)(a.nv - 1);
    const float ca = (float)pl - ic, cb0 = (float)b0 - ic;
    const float zc = (float)(z0 + ZT / 2) - ic;  // the tile's middle height, centred (exact)
    const float zl = (float)(lane - ZT / 2);
    const int pitch = a.nv + SINO_PAD;
    TiltEntry *tab = tabs[warp];
    float(*accw)[T::ROWS][ZP] = acc[warp];
#pragma unroll
    for (int q = 0; q < NCH; ++q)
        for (int r = 0; r < T::ROWS; ++r) accw[q][r][lane] = 0.0f;

    for (int ib = split; ib < a.nviews && pl < a.n; ib += 32 * a.splits) {
        // lane = view: the columns of the tile's piece of the plane, a voxel
        // wider all round: between the projections of its corners
        int vlo = 0, cnt = 0;
        const int iv = ib + lane * a.splits;
        if (iv < a.nviews) {
            const int k = a.view0 + iv * a.stride;
            const ViewGeom &G = a.views[k];
            float lo = 1e30f, hi = -1e30f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float b = (float)(c & 1 ? min(b0 + W, a.n) : b0 - 1);
                const float Z = (float)(c & 2 ? min(z0 + ZT, a.n) : z0 - 1) - G.S[2];
                const float X = (cls ? b : (float)pl) - G.S[0], Y = (cls ? (float)pl : b) - G.S[1];
                const float q0 = fmaf(G.Q[2], Z, fmaf(G.Q[1], Y, G.Q[0] * X));
                const float q2 = fmaf(G.Q[8], Z, fmaf(G.Q[7], Y, G.Q[6] * X));
                const float u = q0 / q2 + cu;
                lo = fminf(lo, u);
                hi = fmaxf(hi, u);
            }
            const int2 r = __ldg(ranges + 2 * k + cls);
            vlo = max(r.x, (int)ceilf(lo - 1e-2f));
            cnt = max(0, min(r.y, (int)floorf(hi + 1e-2f)) - vlo + 1);
        }
        int pre = cnt;  // the views' columns as one list
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULL, pre, o);
            if (lane >= o) pre += v;
        }
        const int total = __shfl_sync(FULL, pre, 31);
        for (int first = 0; __any_sync(FULL, first < total); first += 32) {
            const int idx = first + lane;
            int v = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(FULL, pre, v + o - 1) <= idx) v += o;
            const int ju = __shfl_sync(FULL, vlo, v & 31) + idx - __shfl_sync(FULL, pre - cnt, v & 31);
            bool ok = idx < total;
            int form = 2;  // 0: 4 rows of one class, 1: 5 rows and a class test, 2: row by row
            TiltEntry t;
            if (ok) {
                const int i = ib + v * a.splits;
                t.i = i;
                t.ju = ju;
                t.base = (long long)SINO_PAD + ((long long)i * a.nu + ju) * pitch;
                const ViewGeom &G = a.views[a.view0 + i * a.stride];
                const float up = (float)ju - cu;
                const float *N = cls ? G.NY : G.NX, *Nl = cls ? G.NY_lo : G.NX_lo;
                const int classes = column_classes(G, up, cv);
                ok = (classes >> cls) & 1;
                // height (e0 + v' e1) / (w0 + v' w1): the anchor row, any row near it will do
                const float w0 = fmaf(up, G.Eu[cls], G.Wc[cls]), w1 = G.Ev[cls];
                const float e0 = fmaf(up, N[4], N[3]) + ca * fmaf(up, G.Eu[2], G.Wc[2]), e1 = fmaf(ca, G.Ev[2], N[5]);
                const float jf = rintf((zc * w0 - e0) / (e1 - zc * w1) + cv);
                DF xb, xz, rwa2;
                ray_crossing(G, cls, up, jf - cv, ca, xb, xz, rwa2);
                const DF va{G.Ev[cls], G.Ev_lo[cls]};
                const DF dz = df_add(df_add(DF{N[5], Nl[5]}, df_mul_f(DF{G.Ev[2], G.Ev_lo[2]}, ca)),
                                     df_mul(DF{-xz.hi, -xz.lo}, va));
                const DF sz = df_mul(dz, rwa2);
                const float rwa = rwa2.hi;
                const DF da = df_add(xz, DF{-zc, 0.0f}), ba = df_add(xb, DF{-cb0, 0.0f});
                t.sz = sz.hi;
                t.szlo = sz.lo;
                t.rz = 1.0f / sz.hi;
                t.d1 = __fadd_rn(da.hi, 1.0f) + da.lo;
                t.k = va.hi * rwa;
                const DF db = df_add(df_add(DF{N[2], Nl[2]}, df_mul_f(DF{G.Ev[1 - cls], G.Ev_lo[1 - cls]}, ca)),
                                     df_mul(DF{-xb.hi, -xb.lo}, va));
                const DF sb = df_mul(db, rwa2);
                t.sb = sb.hi;
                t.sblo = sb.lo;
                const float jA = rintf(ba.hi);
                t.bA = __fsub_rn(ba.hi, jA) + ba.lo;
                t.jA = (int)jA;
                t.jv = (int)jf;
                // over the tile's rows the steps differ from the anchor's by at
                // most (1 + kr)^2
                const float kr = fabsf(t.k) * (fabsf(t.d1) + (float)ZT) * t.rz;
                const float smin = t.sz / ((1.0f + kr) * (1.0f + kr)), bmax = fabsf(t.sb) / ((1.0f - kr) * (1.0f - kr));
                if (fabsf(jf) < 1.0e6f && kr < 0.25f) {
                    if (smin > 0.501f && bmax < 0.3f && classes != 3) form = 0;
                    else if (smin > 0.401f && bmax < 0.22f) form = 1;
                }
                if (ok && form < 2) {
                    // columns whose rows at the tile's heights all lie off the detector
                    const float s0 = ((float)(-ZT / 2) - t.d1) * t.rz, s1 = ((float)(ZT / 2) + 1.0f - t.d1) * t.rz;
                    const float ra = s0 / (1.0f - t.k * s0) + jf, rb = s1 / (1.0f - t.k * s1) + jf;
                    ok = ra < (float)a.nv + 1.0f && rb > -2.0f;
                }
            }
            // the table, ordered by form
            const unsigned below = (1u << lane) - 1u;
            int end[3], run = 0;
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                const unsigned m = __ballot_sync(FULL, ok && form == f);
                if (ok && form == f) tab[run + __popc(m & below)] = t;
                run += __popc(m);
                end[f] = run;
            }
            __syncwarp();
            auto rows = [&](const TiltEntry &c, auto ntag) {
                constexpr int R = decltype(ntag)::value;
                const float s1 = (zl - c.d1) * c.rz, ks = c.k * s1;
                const float r0 = __fadd_ru(fmaf(ks * s1, rcp_approx(1.0f - ks), s1), BT_MAGIC) - BT_MAGIC;
                const int row = (int)r0 + c.jv;
                const ST *p = sino + c.base + row;
                const float bA = fmaf(r0, c.sblo, c.bA);  // the low part of the following rows is below 5e-8
                float w[R], b[R];
                float2 y[R];
                // R = 5: the projector's axis choice, ray by ray (ray_dir's own operations)
                float cx = 0.0f, cy = 0.0f, vx = 0.0f, vy = 0.0f;
                if (R == 5) {
                    const ViewGeom &G = a.views[a.view0 + c.i * a.stride];
                    const float up = (float)c.ju - cu;
                    cx = __fmaf_rn(up, G.Eu[0], G.Wc[0]);
                    cy = __fmaf_rn(up, G.Eu[1], G.Wc[1]);
                    vx = G.Ev[0];
                    vy = G.Ev[1];
                }
#pragma unroll
                for (int s = 0; s < R; ++s) {
                    const float r = r0 + (float)s, kr = c.k * r;
                    const float d = -(kr * r) * rcp_approx(1.0f + kr);
                    const float g = fmaf(r, c.sz, -zl) + fmaf(d, c.sz, fmaf(r, c.szlo, c.d1));
                    b[s] = fmaf(d, c.sb, bA);
                    bool in = (unsigned)(row + s) < (unsigned)a.nv;
                    if (R == 5) {
                        const float vp = (float)(row + s) - cv;
                        in = in && (fabsf(__fmaf_rn(vp, vy, cy)) > fabsf(__fmaf_rn(vp, vx, cx))) == (cls != 0);
                    }
                    w[s] = in ? 1.0f - fabsf(g - 1.0f) : -1.0f;
                    y[s] = tl_row(p + s, w[s]);
                }
                // b[s] + (r0 + s) sb: the crossing from voxel column jA
                const float bl = floorf(fminf(fmaf(r0, c.sb, b[0]), fmaf(r0 + (float)(R - 1), c.sb, b[R - 1])));
                float2 p0 = both(0.0f), p1 = both(0.0f), p2 = both(0.0f);  // voxel columns bl, bl + 1, bl + 2
#pragma unroll
                for (int s = 0; s < R; ++s) {
                    const float q = fmaf(r0 + (float)s, c.sb, -1.0f - bl) + b[s], qm = 1.0f - fabsf(q);  // q in [-1, 1)
                    const float2 wy = make_float2(w[s] * y[s].x, NCH == 2 ? w[s] * y[s].y : 0.0f);
                    p1 = fma_f2(both(qm), wy, p1);
                    if (q < 0.0f) p0 = fma_f2(both(-q), wy, p0);
                    if (q > 0.0f) p2 = fma_f2(both(q), wy, p2);
                }
                const int j = (int)bl + c.jA;
                if ((unsigned)(j + 2) < (unsigned)(W + 2)) {
                    float *d = &accw[0][j + 2][lane];
                    d[0] += p0.x;
                    d[ZP] += p1.x;
                    d[2 * ZP] += p2.x;
                    if (NCH == 2) {
                        d = &accw[NCH - 1][j + 2][lane];
                        d[0] += p0.y;
                        d[ZP] += p1.y;
                        d[2 * ZP] += p2.y;
                    }
                }
            };
            for (int e = 0; e < end[0]; ++e) rows(tab[e], std::integral_constant<int, 4>());
            for (int e = end[0]; e < end[1]; ++e) rows(tab[e], std::integral_constant<int, 5>());
            for (int e = end[1]; e < end[2]; ++e) {
                const TiltEntry &c = tab[e];
                const ViewGeom &G = a.views[a.view0 + c.i * a.stride];
                const float up = (float)c.ju - cu, cz = (float)(z0 + lane) - ic;
                const float *N = cls ? G.NY : G.NX;
                const float w0 = fmaf(up, G.Eu[cls], G.Wc[cls]), w1 = G.Ev[cls];
                const float e0 = fmaf(up, N[4], N[3]) + ca * fmaf(up, G.Eu[2], G.Wc[2]), e1 = fmaf(ca, G.Ev[2], N[5]);
                // rows at heights z - 1 and z + 1, with a row to spare
                const float va = ((cz - 1.0f) * w0 - e0) / (e1 - (cz - 1.0f) * w1) + cv;
                const float vb = ((cz + 1.0f) * w0 - e0) / (e1 - (cz + 1.0f) * w1) + cv;
                const int rlo = (int)fmaxf(0.0f, floorf(fminf(va, vb)) - 1.0f);
                const int rhi = (int)fminf((float)(a.nv - 1), ceilf(fmaxf(va, vb)) + 1.0f);
                for (int row = rlo; row <= rhi; ++row) {
                    const float vp = (float)row - cv;
                    if (ray_dir(G, up, vp).ax != cls) continue;
                    DF xb, xz, rwa;
                    ray_crossing(G, cls, up, vp, ca, xb, xz, rwa);
                    const float hz = 1.0f - fabsf(__fadd_rn(__fsub_rn(xz.hi, cz), xz.lo));
                    if (!(hz > 0.0f)) continue;
                    int j;
                    float tb;
                    split_coord(df_add(xb, DF{-cb0, 0.0f}), j, tb);
                    if ((unsigned)(j + 2) >= (unsigned)(W + 2)) continue;
                    const float2 y = tl_row(sino + c.base + row, 1.0f);
                    const float wl = hz * (1.0f - tb), wh = hz * tb;
                    float *d = &accw[0][j + 2][lane];
                    d[0] = fmaf(wl, y.x, d[0]);
                    if (wh > 0.0f) d[ZP] = fmaf(wh, y.x, d[ZP]);
                    if (NCH == 2) {
                        d = &accw[NCH - 1][j + 2][lane];
                        d[0] = fmaf(wl, y.y, d[0]);
                        if (wh > 0.0f) d[ZP] = fmaf(wh, y.y, d[ZP]);
                    }
                }
            }
            __syncwarp();
        }
    }
    __syncthreads();
    const size_t nvox = (size_t)a.n * a.n * a.n;
    float *o = out + (size_t)part * NCH * nvox;
    for (int t = tid; t < BT_WARPS * W * ZT; t += 32 * BT_WARPS) {
        const int c = t % (BT_WARPS * W), zz = t / (BT_WARPS * W), z = z0 + zz;
        const int w = cls ? c / W : c % BT_WARPS, j = cls ? c % W : c / BT_WARPS;
        const int x = cls ? b0 + j : p0 + w, y = cls ? p0 + w : b0 + j;
        if (x < a.n && y < a.n && z < a.n) {
            const size_t idx = ((size_t)z * a.n + y) * a.n + x;
#pragma unroll
            for (int q = 0; q < NCH; ++q) {
                float v = acc[w][q][j + 2][zz];
                if (accumulate) v += o[idx + q * nvox];
                o[idx + q * nvox] = v;
            }
        }
    }
}

// k_class_ranges on tilted geometries: columns that may hold rays of a class.
__global__ void k_class_ranges_tilt(const ViewGeom *__restrict__ views, int K, int nu, int nv, int2 *__restrict__ ranges) {
    const int k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= K) return;
    int lo[2] = {nu, nu}, hi[2] = {-1, -1};
    for (int u = lane; u < nu; u += 32) {
        const int m = column_classes(views[k], (float)u - 0.5f * (float)(nu - 1), 0.5f * (float)(nv - 1));
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if ((m >> c) & 1) {
                lo[c] = min(lo[c], u);
                hi[c] = max(hi[c], u);
            }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        lo[c] = __reduce_min_sync(0xffffffffu, lo[c]);
        hi[c] = __reduce_max_sync(0xffffffffu, hi[c]);
        if (lane == 0) ranges[2 * k + c] = make_int2(lo[c], hi[c]);
    }
}

// Double-float column table (see LevelInfo::d_cols_df), one thread per (view,
// column): the axis choice is the projector's own ray_dir() at v' = 0; the
// quotients by w_a are taken in double-float from the view table's
// double-float fields.
__global__ void k_column_table_df(const ViewGeom *__restrict__ views, int K, int nu, float4 *__restrict__ cols) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= K * nu) return;
    const int k = t / nu, ju = t % nu;
    const ViewGeom &G = views[k];
    const float up = (float)ju - 0.5f * (float)(nu - 1);
    const RayDir d = ray_dir(G, up, 0.0f);
    const int ia = d.ax, ib = 1 - d.ax;
    const DF wa = df_affine(G.Wc[ia], G.Wc_lo[ia], G.Eu[ia], G.Eu_lo[ia], G.Ev[ia], G.Ev_lo[ia], up, 0.0f);
    const DF wb = df_affine(G.Wc[ib], G.Wc_lo[ib], G.Eu[ib], G.Eu_lo[ib], G.Ev[ib], G.Ev_lo[ib], up, 0.0f);
    const DF rinv = df_div(DF{1.0f, 0.0f}, wa);
    const float *N = d.ax ? G.NY : G.NX;
    const float *Nl = d.ax ? G.NY_lo : G.NX_lo;
    const DF rb = df_mul(wb, rinv);
    const DF pb = df_mul(df_affine(N[0], Nl[0], N[1], Nl[1], N[2], Nl[2], up, 0.0f), rinv);
    const DF ez0 = df_mul(df_affine(N[3], Nl[3], N[4], Nl[4], N[5], Nl[5], up, 0.0f), rinv);
    const DF ezc = df_mul(df_affine(G.Wc[2], G.Wc_lo[2], G.Eu[2], G.Eu_lo[2], G.Ev[2], G.Ev_lo[2], up, 0.0f), rinv);
    const DF e10 = df_mul(DF{N[5], Nl[5]}, rinv);
    const DF e1c = df_mul(DF{G.Ev[2], G.Ev_lo[2]}, rinv);
    float4 *o = cols + (size_t)k * 4 * nu + ju;
    o[0] = make_float4(d.ax ? 1.0f : 0.0f, rb.hi, rb.lo, pb.hi);
    o[(size_t)nu] = make_float4(pb.lo, ez0.hi, ez0.lo, ezc.hi);
    o[2 * (size_t)nu] = make_float4(ezc.lo, e10.hi, e10.lo, e1c.hi);
    o[3 * (size_t)nu] = make_float4(e1c.lo, 0.0f, 0.0f, 0.0f);
}

// First and last detector column of each ray class per view (LevelInfo::
// d_ranges; an empty class has first > last), a warp per view.
__global__ void k_class_ranges(const float4 *__restrict__ cols, int K, int nu, int2 *__restrict__ ranges) {
    const int k = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= K) return;
    int lo[2] = {nu, nu}, hi[2] = {-1, -1};
    for (int u = lane; u < nu; u += 32) {
        const int c = __ldg(cols + (size_t)k * 4 * nu + u).x != 0.0f;
        lo[c] = min(lo[c], u);
        hi[c] = max(hi[c], u);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        lo[c] = __reduce_min_sync(0xffffffffu, lo[c]);
        hi[c] = __reduce_max_sync(0xffffffffu, hi[c]);
        if (lane == 0) ranges[2 * k + c] = make_int2(lo[c], hi[c]);
    }
}

// out = (accumulate ? out : 0) + sum over s of part[s], in order of s.
__global__ void k_sum_splits(size_t len, int splits, const float *__restrict__ part, float *__restrict__ out,
                             int accumulate) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x) {
        float v = accumulate ? out[i] : 0.0f;
        for (int q = 0; q < splits; ++q) v += __ldg(part + (size_t)q * len + i);
        out[i] = v;
    }
}

// out = (accumulate ? out : 0) + the sum of `parts` partial volumes, as a
// balanced tree over their (zero-extended) 32: the partial sums of a float32
// chain of up to 32 would cost more digits than the back-projection itself.
template <int P>
__device__ __forceinline__ float tree_sum(const float *__restrict__ part, size_t len, int first, int parts) {
    if (first >= parts) return 0.0f;
    if constexpr (P == 1) return __ldg(part + (size_t)first * len);
    else return tree_sum<P / 2>(part, len, first, parts) + tree_sum<P / 2>(part, len, first + P / 2, parts);
}
__global__ void k_sum_parts(size_t len, int parts, const float *__restrict__ part, float *__restrict__ out,
                            int accumulate) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (size_t)gridDim.x * blockDim.x) {
        const float v = tree_sum<32>(part + i, len, 0, parts);
        out[i] = accumulate ? out[i] + v : v;
    }
}

// Number of view shares for a launch of `blocks` blocks on `sms` multiprocessors
// that hold `occ` blocks each, at most 16 and `most`: the one with the least
// estimated time, in units of a view's work on a full chip.  The multiprocessor
// with the most blocks, m of them, takes m / occ waves, of which a last one of r
// blocks takes 0.4 + 0.45 r / occ; every share writes and reads its partial
// volumes, `share` views' work: 1.5 in the plane kernel at a row step of 0.6 voxel
// (public call at 128^3 by 1, 2, 3 shares: 16 views 110, 100, 111 us, 90 views 493,
// 397, 381; at 200^3, 4 views by 1, 2, 4: 125, 168, 256 us), 0.5 in the tilt kernel,
// 1 in the slab kernel (one volume a share).
inline int view_splits(int sms, int occ, int blocks, int nviews, int most, double share) {
    int best = 1;
    double cost = 1e300;
    for (int sp = 1; sp <= 16 && sp <= nviews && (sp == 1 || sp <= most); ++sp) {
        const long long m = ((long long)blocks * sp + sms - 1) / sms;
        const double waves = (double)(m / occ) + (m % occ ? 0.4 + 0.45 * (double)(m % occ) / occ : 0.0);
        const double c = nviews * waves * occ * sms / ((double)blocks * sp) + share * sp;
        if (c < cost) {
            cost = c;
            best = sp;
        }
    }
    return best;
}

}  // namespace mgct

#include "backproject_slab.cuh"

namespace mgct {

// Launches a tile kernel (k_backproject_plane, k_backproject_tilt): both ray
// classes and the shares of the views in one launch, each into its own partial volume
// of split_buf (cap floats), or one class after the other without one.
template <int NCH, typename F, typename KF>
int launch_tiles(const LevelInfo &L, BPArgs a, dim3 grid, KF kernel, size_t smem, float *out, int accumulate,
                 cudaStream_t s, float *split_buf, size_t cap, double share, F run) {
    const size_t vol_floats = (size_t)NCH * L.n * L.n * L.n;
    const int room = split_buf ? (int)(cap / vol_floats < 64 ? cap / vol_floats : 64) : 0;
    if (room < 2) {
        for (a.cls = 1; a.cls >= 0; --a.cls) MGCT_KERNEL(KK_BACKPROJECT, s, run(a, grid, out, accumulate || a.cls == 0));
        return MGCT_OK;
    }
    int sms = 0, occ = 0;
    MGCT_TRY(sm_count(&sms));
    MGCT_TRY(check_cuda(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 32 * BT_WARPS, smem), "occupancy"));
    a.splits = view_splits(sms, occ > 0 ? occ : 1, 2 * (int)(grid.x * grid.y * grid.z), a.nviews, room / 2, share);
    const int parts = 2 * a.splits;
    grid.z *= parts;
    MGCT_KERNEL(KK_BACKPROJECT, s, run(a, grid, split_buf, 0));
    const int sb = (int)((vol_floats + 255) / 256 < 4096 ? (vol_floats + 255) / 256 : 4096);
    MGCT_KERNEL(KK_BACKPROJECT, s, k_sum_parts<<<sb, 256, 0, s>>>(vol_floats, parts, split_buf, out, accumulate));
    return MGCT_OK;
}

template <int NCH, int NP, typename ST>
int launch_backproject_plane(const LevelInfo &L, const BPArgs &a, const ST *sino, float *out, int accumulate,
                             cudaStream_t s, float *split_buf, size_t cap, double step) {
    using T = PlaneTile<NCH, NP>;
    // finer rows: more work a view
    const double share = 1.5 * std::exp2(-8.0 * std::max(0.0, 0.6 - step));
    constexpr size_t smem = T::smem;
    static_assert(smem <= 48 * 1024, "within the default shared-memory limit");
    const dim3 grid((L.n + T::W - 1) / T::W, (L.n + BT_WARPS - 1) / BT_WARPS, (L.n + T::ZT - 1) / T::ZT);
    return launch_tiles<NCH>(L, a, grid, k_backproject_plane<NCH, NP, ST>, smem, out, accumulate, s, split_buf, cap, share,
                             [&](const BPArgs &b, dim3 g, float *dst, int acc) {
                                 k_backproject_plane<NCH, NP, ST>
                                     <<<g, 32 * BT_WARPS, smem, s>>>(b, L.d_cols_df, L.d_ranges, sino, dst, acc);
                             });
}

template <int NCH, typename ST>
int launch_backproject_tilt(const LevelInfo &L, const BPArgs &a, const ST *sino, float *out, int accumulate,
                            cudaStream_t s, float *split_buf, size_t cap) {
    using T = TiltTile<NCH>;
    const dim3 grid((L.n + T::W - 1) / T::W, (L.n + BT_WARPS - 1) / BT_WARPS, (L.n + T::ZT - 1) / T::ZT);
    return launch_tiles<NCH>(L, a, grid, k_backproject_tilt<NCH, ST>, 0, out, accumulate, s, split_buf, cap, 0.5,
                             [&](const BPArgs &b, dim3 g, float *dst, int acc) {
                                 k_backproject_tilt<NCH, ST><<<g, 32 * BT_WARPS, 0, s>>>(b, L.d_ranges, sino, dst, acc);
                             });
}

// A^T of a weighted sinogram stored [view][u][v] on a separable geometry.
// Two pairs a lane halve the per-column work of a height, one wastes less of
// the last tile: one where the tiles of the larger kind hold over a quarter
// more heights.
template <int NCH, typename ST>
int launch_backproject_cols(const LevelInfo &L, const BPArgs &a, const ST *sino, float *out, int accumulate,
                            cudaStream_t s, float *split_buf, size_t cap, double step) {
    constexpr int Z1 = PlaneTile<NCH, 1>::ZT, Z2 = PlaneTile<NCH, 2>::ZT;
    const int t1 = (L.n + Z1 - 1) / Z1 * Z1, t2 = (L.n + Z2 - 1) / Z2 * Z2;
    if (4 * t2 <= 5 * t1) return launch_backproject_plane<NCH, 2, ST>(L, a, sino, out, accumulate, s, split_buf, cap, step);
    return launch_backproject_plane<NCH, 1, ST>(L, a, sino, out, accumulate, s, split_buf, cap, step);
}

inline BPArgs bp_args(const LevelInfo &L, int view0, int nviews, int stride) {
    BPArgs a;
    a.views = L.d_views;
    a.n = L.n;
    a.nu = L.nu;
    a.nv = L.nv;
    a.h = (float)L.h;
    a.view0 = view0;
    a.stride = stride;
    a.nviews = nviews;
    a.splits = 1;
    a.cls = -1;
    return a;
}

// NCH = 2 writes channel c to out + c * n^3.  WEIGHTED: the sinogram carries
// each ray's dl already (internal solver path) and is stored for `route`
// (weighted_strides).  split_buf (cap floats, or NULL): scratch for partial
// volumes.
template <int NCH, typename ST, bool WEIGHTED = false>
int launch_backproject(const mgct_geom *g, int level, int view0, int nviews, int stride, const ST *sino,
                       float *out, int accumulate, cudaStream_t s, BpRoute route = BpRoute::GATHER,
                       float *split_buf = nullptr, size_t cap = 0) {
    const LevelInfo &L = g->lev[level];
    const BPArgs a = bp_args(L, view0, nviews, stride);
    if constexpr (WEIGHTED) {
        if (route == BpRoute::SLAB) return launch_backproject_slab<NCH, ST>(L, a, sino, out, accumulate, s, split_buf, cap);
    }
    if constexpr (WEIGHTED && sizeof(ST) != 2) {
        if (route == BpRoute::PLANE)
            return launch_backproject_cols<NCH, ST>(L, a, sino, out, accumulate, s, split_buf, cap, g->row_step);
        if (route == BpRoute::TILT) return launch_backproject_tilt<NCH, ST>(L, a, sino, out, accumulate, s, split_buf, cap);
    }
    if constexpr (!WEIGHTED) {
        if (g->separable) {
            const int zper = BP_BZ * BPS_ZB;
            dim3 grid((L.n + BP_BX - 1) / BP_BX, (L.n + BP_BY - 1) / BP_BY, (L.n + zper - 1) / zper);
            MGCT_KERNEL(KK_BACKPROJECT, s,
                        k_backproject_sep<NCH, ST, WEIGHTED><<<grid, dim3(BP_BX, BP_BY, BP_BZ), 0, s>>>(a, L.d_cols_df, sino, out, accumulate));
            return MGCT_OK;
        }
    }
    dim3 grid((L.n + BP_BX - 1) / BP_BX, (L.n + BP_BY - 1) / BP_BY, (L.n + BP_BZ - 1) / BP_BZ);
    MGCT_KERNEL(KK_BACKPROJECT, s,
                k_backproject<NCH, ST, WEIGHTED><<<grid, dim3(BP_BX, BP_BY, BP_BZ), 0, s>>>(a, sino, out, accumulate));
    return MGCT_OK;
}

// The public A^T on tilt-free geometries.  Each ray's path length per plane,
// dl = h sqrt(1 + rb^2 + rz^2) (the projector's weight; rb per column, rz
// linear in v', both from the double-float column table), is applied to the
// caller's sinogram in one pass over it, which also turns it to [view][u][v]
// with its zero rows (32 x 32 tiles through shared memory), into the handle's
// quad scratch; the
// plane kernel then takes it like the solver's residual.
template <typename ST>
__global__ void __launch_bounds__(256)
    k_weight_rays(BPArgs a, const float4 *__restrict__ cols, const ST *__restrict__ sino, float *__restrict__ w) {
    __shared__ float tile[32][33];
    const int u0 = blockIdx.x * 32, v0 = blockIdx.y * 32, i = blockIdx.z;
    const int k = a.view0 + i * a.stride;
    const float4 *c = cols + (size_t)k * 4 * a.nu;
    const size_t base = (size_t)i * a.nv * a.nu;
    const int pitch = a.nv + SINO_PAD;
    const int ju = u0 + threadIdx.x;
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && threadIdx.y == 0 && threadIdx.x < SINO_PAD) w[threadIdx.x] = 0.0f;
    if (ju < a.nu) {
        // rb, (Wc_z + u' Eu_z) / w_a, Ev_z / w_a
        const float rb = __ldg(c + ju).y, ezc = __ldg(c + a.nu + ju).w, e1c = __ldg(c + 2 * a.nu + ju).w;
        for (int r = threadIdx.y; r < 32; r += 8) {
            tile[r][threadIdx.x] = 0.0f;  // the zero rows
            if (v0 + r >= a.nv) continue;
            const float rz = fmaf((float)(v0 + r) - 0.5f * (float)(a.nv - 1), e1c, ezc);
            const float dl = sqrtf(fmaf(rz, rz, fmaf(rb, rb, 1.0f))) * a.h;
            tile[r][threadIdx.x] = dl * to_f32(__ldg(sino + base + (size_t)(v0 + r) * a.nu + ju));
        }
    }
    __syncthreads();
    const int jv = v0 + threadIdx.x;
    if (jv < pitch)
        for (int r = threadIdx.y; r < 32 && u0 + r < a.nu; r += 8)
            w[SINO_PAD + ((size_t)i * a.nu + u0 + r) * pitch + jv] = tile[threadIdx.x][r];
}

// The same for the slab kernel, to [view][v][u].
template <typename ST>
__global__ void k_weight_rows(BPArgs a, const float4 *__restrict__ cols, const ST *__restrict__ sino,
                              float *__restrict__ w) {
    const int ju = blockIdx.x * blockDim.x + threadIdx.x;
    if (ju >= a.nu) return;
    const int jv = blockIdx.y, i = blockIdx.z;
    const float4 *c = cols + (size_t)(a.view0 + i * a.stride) * 4 * a.nu + ju;
    const float rb = __ldg(c).y, ezc = __ldg(c + a.nu).w, e1c = __ldg(c + 2 * a.nu).w;
    const float rz = fmaf((float)jv - 0.5f * (float)(a.nv - 1), e1c, ezc);
    const float dl = sqrtf(fmaf(rz, rz, fmaf(rb, rb, 1.0f))) * a.h;
    const size_t idx = ((size_t)i * a.nv + jv) * a.nu + ju;
    w[idx] = dl * to_f32(__ldg(sino + idx));
}

// The same on tilted geometries, each ray's slopes in double-float from the
// view table.
template <typename ST>
__global__ void __launch_bounds__(256)
    k_weight_rays_tilt(BPArgs a, const ST *__restrict__ sino, float *__restrict__ w) {
    __shared__ float tile[32][33];
    const int u0 = blockIdx.x * 32, v0 = blockIdx.y * 32, i = blockIdx.z;
    const ViewGeom &G = a.views[a.view0 + i * a.stride];
    const size_t base = (size_t)i * a.nv * a.nu;
    const int pitch = a.nv + SINO_PAD;
    const int ju = u0 + threadIdx.x;
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && threadIdx.y == 0 && threadIdx.x < SINO_PAD) w[threadIdx.x] = 0.0f;
    for (int r = threadIdx.y; r < 32; r += 8) {
        float v = 0.0f;  // the zero rows
        if (ju < a.nu && v0 + r < a.nv) {
            const float up = (float)ju - 0.5f * (float)(a.nu - 1), vp = (float)(v0 + r) - 0.5f * (float)(a.nv - 1);
            const int ia = ray_dir(G, up, vp).ax, ib = 1 - ia;
            const DF wa = df_affine(G.Wc[ia], G.Wc_lo[ia], G.Eu[ia], G.Eu_lo[ia], G.Ev[ia], G.Ev_lo[ia], up, vp);
            const DF wb = df_affine(G.Wc[ib], G.Wc_lo[ib], G.Eu[ib], G.Eu_lo[ib], G.Ev[ib], G.Ev_lo[ib], up, vp);
            const DF wz = df_affine(G.Wc[2], G.Wc_lo[2], G.Eu[2], G.Eu_lo[2], G.Ev[2], G.Ev_lo[2], up, vp);
            const float rb = df_div(wb, wa).hi, rz = df_div(wz, wa).hi;
            v = sqrtf(fmaf(rz, rz, fmaf(rb, rb, 1.0f))) * a.h * to_f32(__ldg(sino + base + (size_t)(v0 + r) * a.nu + ju));
        }
        tile[r][threadIdx.x] = v;
    }
    __syncthreads();
    const int jv = v0 + threadIdx.x;
    if (jv < pitch)
        for (int r = threadIdx.y; r < 32 && u0 + r < a.nu; r += 8)
            w[SINO_PAD + ((size_t)i * a.nu + u0 + r) * pitch + jv] = tile[threadIdx.x][r];
}

// Runs the public A^T by weighted rays and the kernel of bp_route, in chunks of
// views that fit the quad scratch, and sets *ran; leaves *ran = 0 (nothing
// launched) where it does not apply: the gather's route, no views, or a scratch
// smaller than one view.
template <typename ST>
int launch_backproject_public(const mgct_geom *g, int level, int view0, int nviews, int stride, const ST *sino,
                              float *out, int accumulate, cudaStream_t s, int *ran) {
    *ran = 0;
    const LevelInfo &L = g->lev[level];
    const size_t view_elems = (size_t)L.nu * L.nv;
    const size_t cap = 2 * quad_elems(g->lev[0].n) * 4;  // floats in the quad scratch
    if (nviews < 1) return MGCT_OK;
    const BpRoute route = bp_route(g, L, sizeof(float), nviews, true);
    const bool slab = route == BpRoute::SLAB;
    const size_t padded = slab ? view_elems : (size_t)L.nu * (L.nv + SINO_PAD);  // a view of weighted rays
    if (route == BpRoute::GATHER || !L.d_ranges || cap < padded + SINO_PAD || L.nv > 65535) return MGCT_OK;
    size_t chunk = (cap - SINO_PAD) / padded;
    if (chunk > (size_t)nviews) chunk = nviews;
    if (chunk > 65535) chunk = 65535;
    float *w = static_cast<float *>(g->d_scratch_quads);
    for (int c0 = 0; c0 < nviews; c0 += (int)chunk) {
        const int cn = nviews - c0 < (int)chunk ? nviews - c0 : (int)chunk;
        const BPArgs a = bp_args(L, view0 + c0 * stride, cn, stride);
        const dim3 wgrid((L.nu + 31) / 32, (L.nv + SINO_PAD + 31) / 32, cn);
        // what the weighted rays leave of the scratch holds partial volumes
        const size_t used = ((size_t)cn * padded + SINO_PAD + 63) & ~(size_t)63;
        float *free_buf = w + used;
        const size_t free_cap = cap > used ? cap - used : 0;
        const ST *sc = sino + (size_t)c0 * view_elems;
        const int acc = accumulate || c0 ? 1 : 0;
        if (slab) {
            MGCT_KERNEL(KK_BACKPROJECT, s, k_weight_rows<ST><<<dim3((L.nu + 127) / 128, L.nv, cn), 128, 0, s>>>(
                                               a, L.d_cols_df, sc, w));
            MGCT_TRY((launch_backproject_slab<1, float>(L, a, w, out, acc, s, free_buf, free_cap)));
        } else if (route == BpRoute::PLANE) {
            MGCT_KERNEL(KK_BACKPROJECT, s, k_weight_rays<ST><<<wgrid, dim3(32, 8), 0, s>>>(a, L.d_cols_df, sc, w));
            MGCT_TRY((launch_backproject_cols<1, float>(L, a, w, out, acc, s, free_buf, free_cap, g->row_step)));
        } else {
            MGCT_KERNEL(KK_BACKPROJECT, s, k_weight_rays_tilt<ST><<<wgrid, dim3(32, 8), 0, s>>>(a, sc, w));
            MGCT_TRY((launch_backproject_tilt<1, float>(L, a, w, out, acc, s, free_buf, free_cap)));
        }
    }
    *ran = 1;
    return MGCT_OK;
}

}  // namespace mgct
