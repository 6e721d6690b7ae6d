// The network's output layer at inference: a 3x3x3 convolution of 64 channels
// to one (channels-last bf16 in, float32 out).
//
// As an implicit GEMM over taps its N is 1: on tcgen05 (k_conv_ws, N padded to
// 16) every one of the 108 MMAs of a 128-voxel row block fetches a 4 KB
// operand from shared memory for almost no arithmetic, 2.88 ms at 256^3.  Here
// the 27 taps are the N instead: per voxel q the 27 products
//   T[tap][q] = sum_ci in[q][ci] w[tap][ci]
// are one GEMM row of K = 64, N = 27 (padded to 32) -- 16 register MMAs per 16
// voxels, the weights held in registers -- and an output voxel is the sum of
// 27 shifted entries, out[p] = bias + sum_tap T[tap][p + tap].  N = 32 is too
// small for tcgen05's operand fetch to pay, and the products never leave the
// SM: a block owns 32 x 8 columns and walks zb planes along z; each haloed
// input plane is read once into shared memory, its products written there tap
// by tap, and every thread adds the 9 + 9 + 9 of them that belong to its
// column's outputs at z - 1, z and z + 1, which roll in registers.  An
// output's additions run in the order of the taps whatever the tiling.
// Measured 0.72 ms at 256^3 (half of it the input's 2.1 GB with its halo at the
// copy rate), the network 6.98 -> 4.81 ms; at 32^3 and less no difference.
//
// Training keeps k_conv_ws for this layer: its output enters the loss gradient,
// which is rounded to bf16.
#pragma once

#include "conv3d.cuh"

namespace mgct {

constexpr int OL_TX = 32, OL_TY = 8, OL_C = 64;
constexpr int OL_ZMAX = 32, OL_ZMIN = 4;  // planes a block walks
constexpr int OL_HX = OL_TX + 2, OL_HY = OL_TY + 2, OL_HV = OL_HX * OL_HY;  // haloed plane, 340 voxels
constexpr int OL_MT = (OL_HV + 15) / 16;                                    // its 16-voxel row blocks
constexpr int OL_PITCH = OL_C + 8;   // bf16 per staged voxel: 16-byte rows fall on distinct banks
constexpr int OL_TP = 356;           // T's voxel pitch: the fragments' 4 columns x 8 rows fall on distinct banks
static_assert(OL_TP >= OL_MT * 16, "T holds every row of the blocks");
constexpr size_t OL_SMEM = (size_t)OL_MT * 16 * OL_PITCH * 2 + (size_t)27 * OL_TP * 4;

__global__ void __launch_bounds__(256, 2) k_conv_out(const __nv_bfloat16 *__restrict__ in,
                                                     const __nv_bfloat16 *__restrict__ w, int wrows,
                                                     const float *__restrict__ bias, float *__restrict__ out, int D,
                                                     int H, int W, int zb) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __nv_bfloat16 *sin = reinterpret_cast<__nv_bfloat16 *>(smem_raw);  // [OL_MT * 16][OL_PITCH]
    float *T = reinterpret_cast<float *>(smem_raw + (size_t)OL_MT * 16 * OL_PITCH * 2);  // [27][OL_TP]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x0 = blockIdx.x * OL_TX, y0 = blockIdx.y * OL_TY;
    const int chunks = (D + zb - 1) / zb;
    const int b = blockIdx.z / chunks, z0 = (blockIdx.z - b * chunks) * zb, z1 = min(D, z0 + zb);
    const size_t plane0 = (size_t)b * D * H * W;
    // B fragments of the MMAs: w[tap = n][ci = k], tap rows beyond 26 zero
    uint32_t bw[4][4][2];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int kt = 0; kt < 4; ++kt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int tap = nt * 8 + lane / 4, ci = kt * 16 + h * 8 + 2 * (lane % 4);
                bw[nt][kt][h] =
                    tap < 27 ? __ldg(reinterpret_cast<const uint32_t *>(w + ((size_t)tap * wrows) * OL_C + ci)) : 0u;
            }
    // rows of the last block beyond the plane stay zero
    for (int e = tid; e < (OL_MT * 16 - OL_HV) * OL_PITCH; e += 256) sin[OL_HV * OL_PITCH + e] = __float2bfloat16(0.0f);
    auto load = [&](int z) {
        for (int e = tid; e < OL_HV * (OL_C / 8); e += 256) {
            const int v = e / (OL_C / 8), c = e % (OL_C / 8);
            const int x = x0 - 1 + v % OL_HX, y = y0 - 1 + v / OL_HX;
            const bool ok = (unsigned)z < (unsigned)D && (unsigned)y < (unsigned)H && (unsigned)x < (unsigned)W;
            const __nv_bfloat16 *src = ok ? in + (plane0 + ((size_t)z * H + y) * W + x) * OL_C + c * 8 : in;
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sin + v * OL_PITCH + c * 8);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int tx = lane, ty = warp;
    const int x = x0 + tx, y = y0 + ty;
    const float bv = bias ? __ldg(bias) : 0.0f;
    float cur = 0.0f, prev = 0.0f;  // outputs z and z - 1 so far
    load(z0 - 1);
    for (int z = z0 - 1; z <= z1; ++z) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // plane z staged; T free
        for (int mt = warp; mt < OL_MT; mt += 8) {
            float d[4][4];
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) d[nt][q] = 0.0f;
#pragma unroll
            for (int kt = 0; kt < 4; ++kt) {
                uint32_t a[4];
                const uint32_t src = (uint32_t)__cvta_generic_to_shared(sin + (mt * 16 + lane % 16) * OL_PITCH + kt * 16 + (lane / 16) * 8);
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                             : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                             : "r"(src)
                             : "memory");
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
                    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                                 : "+f"(d[nt][0]), "+f"(d[nt][1]), "+f"(d[nt][2]), "+f"(d[nt][3])
                                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(bw[nt][kt][0]), "r"(bw[nt][kt][1]));
            }
            const int row = mt * 16 + lane / 4;
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int tap = nt * 8 + 2 * (lane % 4) + (q & 1);
                    if (nt < 3 || tap < 27) T[tap * OL_TP + row + (q & 2 ? 8 : 0)] = d[nt][q];
                }
        }
        __syncthreads();  // T complete; the input plane is free
        if (z < z1) load(z + 1);
        // this plane's shares of outputs z - 1, z and z + 1
        float s[3];
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            s[g] = 0.0f;
#pragma unroll
            for (int e = 0; e < 9; ++e) s[g] += T[(g * 9 + e) * OL_TP + (ty + e / 3) * OL_HX + tx + e % 3];
        }
        if (z - 1 >= z0 && x < W && y < H) out[plane0 + ((size_t)(z - 1) * H + y) * W + x] = (prev + s[2]) + bv;
        prev = cur + s[1];
        cur = s[0];
    }
}

// Planes a block walks: two of zb + 2 are halo, so as many as leave two blocks
// for each multiprocessor.
inline int conv_out_planes(int sms, int B, int D, int H, int W) {
    const long long tiles = (long long)B * ((H + OL_TY - 1) / OL_TY) * ((W + OL_TX - 1) / OL_TX);
    int zb = OL_ZMAX;
    while (zb > OL_ZMIN && tiles * ((D + zb - 1) / zb) < 2LL * sms) zb /= 2;
    return zb;
}

inline bool conv_out_fits(int sms, int B, int D, int H, int W) {  // the grid's y and z limits
    const int zb = conv_out_planes(sms, B, D, H, W);
    return (H + OL_TY - 1) / OL_TY <= 65535 && (long long)B * ((D + zb - 1) / zb) <= 65535;
}

// y = conv(in) of the output layer; w [27][wrows][64], row 0 of each tap.
inline int launch_conv_out(int sms, const __nv_bfloat16 *in, const __nv_bfloat16 *w, int wrows, const float *bias,
                           float *out, int B, int D, int H, int W, cudaStream_t s) {
    MGCT_TRY(check_cuda(cudaFuncSetAttribute(k_conv_out, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OL_SMEM),
                        "output layer shared memory"));
    const int zb = conv_out_planes(sms, B, D, H, W);
    const dim3 grid((W + OL_TX - 1) / OL_TX, (H + OL_TY - 1) / OL_TY, (unsigned)(B * ((D + zb - 1) / zb)));
    MGCT_KERNEL(KK_CONV, s, k_conv_out<<<grid, 256, OL_SMEM, s>>>(in, w, wrows, bias, out, D, H, W, zb));
    return MGCT_OK;
}

}  // namespace mgct
