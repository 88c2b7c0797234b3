// Exact transpose of the interpolated projector with warps of detector rows
// (the lanes, cells and z-fastest order of forward_cols.cu).
//
// Accumulators are quads: element (y, x, s), s fastest, holds what the cell
// (x, x+1) x (y, y+1) of plane s gives its four corners.  A lane sums its
// samples in registers while they stay in one cell, for the planes s and s + 1,
// and adds both quads with one vector reduction each when it leaves the cell:
// two 16-byte reductions per cell, neighbouring lanes to neighbouring
// addresses, instead of eight scalar ones per sample.  A second pass adds each
// voxel's four cells and writes the volume.
//
// Measured (ms; before: eight scalar reductions per sample into two layouts):
// 64^3 x 100 (128^2) 1.28 -> 0.29, 192^3 x 180 9.39 -> 2.46, 256^3 x 180 20.7 ->
// 5.65, 512^3 x 60 54.2 -> 18.9, 1024^3 x 3 (1024^2) 70.0 -> 39.5.  The scatter is
// bound by the reductions in L2.
#include <algorithm>

#include "forward_cols.cuh"
#include "ray.cuh"

namespace tigre {
namespace {

constexpr int kAdjRows = 8;   // detector rows per warp (x 4 columns)
constexpr int kAdjWarps = 4;  // warps per block

__device__ __forceinline__ void add_quad(float4* p, float2 a, float2 b)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a.x), "f"(a.y),
                 "f"(b.x), "f"(b.y)
                 : "memory");
}

template <typename TP>
__global__ void __launch_bounds__(32 * kAdjWarps) adj_cols_kernel(
    const TP* __restrict__ proj, float4* __restrict__ acc, const FwdAngle* __restrict__ params,
    FwdConst c, int a_first, uint32_t SX, uint32_t SY)
{
    const unsigned full = 0xffffffffu;
    constexpr int G = 32 / kAdjRows;
    const int p = ((int)blockIdx.x * kAdjWarps + (int)threadIdx.y) * G + (int)threadIdx.x / kAdjRows;
    const int q = (int)blockIdx.z * kAdjRows + (int)threadIdx.x % kAdjRows;
    const int a = blockIdx.y;
    const FwdAngle* P = params + a_first + a;
    const int layout = P->layout;
    Ray R;
    R.K = 0;
    R.ok = true;
    float yv = 0.0f;
    if (p < c.nu && q < c.nv) {
        yv = to_f32<TP>(proj[((int64_t)a * c.nv + q) * c.nu + p]);
        if (yv != 0.0f) setup_ray(P, c, p, q, R);
    }
    const bool active = R.ok && R.K > 0;
    const int K = active ? R.K : 0;
    const int kmax = __reduce_max_sync(full, K);
    if (kmax == 0) return;
    // the lanes at one depth: each starts a whole number of steps late
    const float dep0 = active ? R.x0[1] : 0.0f, ddep = active ? R.d[1] : 0.0f;
    const bool neg = __all_sync(full, !active || ddep < 0.0f);
    const bool same = neg || __all_sync(full, !active || ddep > 0.0f);
    const float sgn = neg ? -1.0f : 1.0f;
    float Y0 = active ? sgn * dep0 : 3.0e38f, D = active ? fabsf(ddep) : 1.0e-30f;
    for (int o = 16; o > 0; o >>= 1) {
        Y0 = fminf(Y0, __shfl_xor_sync(full, Y0, o));
        D = fmaxf(D, __shfl_xor_sync(full, D, o));
    }
    int shift = active && same ? (int)fminf((sgn * dep0 - Y0) / D, 1.0e8f) : 0;
    int J = __reduce_max_sync(full, shift + K);
    if (J > 2 * kmax + 64) {  // rays across far-apart corners: start together
        shift = 0;
        J = kmax;
    }
    const float hy = active ? R.h * yv : 0.0f;
    const float xx = !active ? 1.0f : layout ? R.x0[1] : R.x0[0], dx = layout ? R.d[1] : R.d[0];
    const float xy = !active ? 1.0f : layout ? R.x0[0] : R.x0[1], dy = layout ? R.d[0] : R.d[1];
    const float xs = active ? R.x0[2] : 1.0f, ds = R.d[2];
    const uint32_t bias = 0x4B000000u * (SY + SX + 1u);
    uint32_t cur = ~0u;
    const float2 zero = make_float2(0.0f, 0.0f);
    float2 lo0 = zero, lo1 = zero, hi0 = zero, hi1 = zero;  // (v00, vx), (vy, vxy) of planes s, s + 1
    for (int j = 0; j < J; ++j) {
        const int k = j - shift;
        if ((unsigned)k >= (unsigned)K) continue;
        const float kf = (float)k;
        uint32_t bx, by, bs;
        float ax, ay, as;
        split_bits(fmaf(kf, dx, xx), bx, ax);
        split_bits(fmaf(kf, dy, xy), by, ay);
        split_bits(fmaf(kf, ds, xs), bs, as);
        const uint32_t e = by * SY + bx * SX + bs - bias;
        if (e != cur) {
            if (cur != ~0u) {
                add_quad(acc + cur, lo0, lo1);
                add_quad(acc + cur + 1, hi0, hi1);
            }
            lo0 = lo1 = hi0 = hi1 = zero;
            cur = e;
        }
        const float s0 = hy * (1.0f - as), s1 = hy * as;
        const float2 wx = make_float2(1.0f - ax, ax);
        const float2 m0 = __fmul2_rn(wx, make_float2(1.0f - ay, 1.0f - ay));
        const float2 m1 = __fmul2_rn(wx, make_float2(ay, ay));
        lo0 = __ffma2_rn(m0, make_float2(s0, s0), lo0);
        lo1 = __ffma2_rn(m1, make_float2(s0, s0), lo1);
        hi0 = __ffma2_rn(m0, make_float2(s1, s1), hi0);
        hi1 = __ffma2_rn(m1, make_float2(s1, s1), hi1);
    }
    if (cur != ~0u) {
        add_quad(acc + cur, lo0, lo1);
        add_quad(acc + cur + 1, hi0, hi1);
    }
}

// vol[z][y][x] = what the four cells around it gave its corner of plane z.
// A block takes 32 planes x 32 x and marches `rows` y rows: a lane is a plane,
// a thread four neighbouring x, whose sums from the row of cells below stay in
// registers; each row is transposed in shared memory and written along x.
template <typename TV>
__global__ void __launch_bounds__(256) adj_cols_finish_kernel(const float4* __restrict__ acc,
                                                              TV* __restrict__ vol, int nx, int ny,
                                                              int nz, int rows)
{
    __shared__ float tile[32][33];  // [z][x]
    const int PX = nx + 2 * kPad, PS = nz + 2 * kPad;
    const int z0 = blockIdx.x * 32, x0 = blockIdx.y * 32, y0 = blockIdx.z * rows;
    const int y1 = min(y0 + rows, ny);
    const int s = z0 + (int)threadIdx.x + kPad, xt = x0 + 4 * (int)threadIdx.y;
    float below[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int y = y0 - 1; y < y1; ++y) {
        float4 e[5];  // cells (xt - 1 .. xt + 3, y): (v00, vx, vy, vxy)
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const int cx = xt - 1 + i + kPad;
            e[i] = s < PS && cx < PX ? acc[((int64_t)(y + kPad) * PX + cx) * PS + s]
                                     : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        if (y >= y0) {
            __syncthreads();  // the previous row is written
#pragma unroll
            for (int i = 0; i < 4; ++i)
                tile[threadIdx.x][4 * threadIdx.y + i] = below[i] + (e[i + 1].x + e[i].y);
            __syncthreads();
            const int x = x0 + (int)threadIdx.x;
            for (int k = threadIdx.y; k < 32 && z0 + k < nz; k += 8)
                if (x < nx)
                    vol[((int64_t)(z0 + k) * ny + y) * nx + x] = from_f32<TV>(tile[k][threadIdx.x]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) below[i] = e[i + 1].z + e[i].w;
    }
}

}  // namespace

template <typename TP, typename TV>
tigre_status launch_adjoint_columns(tigre_geometry* g, const TP* proj, float4* acc, TV* vol,
                                    int64_t a0, int64_t na, cudaStream_t st)
{
    const FwdConst c = make_fwd_const(g);
    const uint32_t SX = (uint32_t)(c.nz + 2 * kPad), SY = SX * (uint32_t)(c.nx + 2 * kPad);
    constexpr int kCols = 32 / kAdjRows * kAdjWarps;
    for (int64_t s = 0; s < na; s += 65535) {
        const int64_t cnt = std::min<int64_t>(65535, na - s);
        dim3 grid((unsigned)((c.nu + kCols - 1) / kCols), (unsigned)cnt,
                  (unsigned)((c.nv + kAdjRows - 1) / kAdjRows));
        adj_cols_kernel<TP><<<grid, dim3(32, kAdjWarps), 0, st>>>(
            proj + s * (int64_t)c.nu * c.nv, acc, (const FwdAngle*)g->fwd_params.ptr, c,
            (int)(a0 + s), SX, SY);
        TIGRE_LAUNCHED("adj_cols_kernel");
    }
    const int rows = std::max(16, (c.ny + 65534) / 65535);
    dim3 grid((unsigned)((c.nz + 31) / 32), (unsigned)((c.nx + 31) / 32),
              (unsigned)((c.ny + rows - 1) / rows));
    adj_cols_finish_kernel<TV><<<grid, dim3(32, 8), 0, st>>>(acc, vol, c.nx, c.ny, c.nz, rows);
    TIGRE_LAUNCHED("adj_cols_finish_kernel");
    return TIGRE_OK;
}

#define TIGRE_ADJ(TP, TV)                                                                        \
    template tigre_status launch_adjoint_columns<TP, TV>(tigre_geometry*, const TP*, float4*,    \
                                                         TV*, int64_t, int64_t, cudaStream_t);
#define TIGRE_ADJ_ALL(TP)          \
    TIGRE_ADJ(TP, float)           \
    TIGRE_ADJ(TP, __nv_bfloat16)   \
    TIGRE_ADJ(TP, __half)
TIGRE_ADJ_ALL(float)
TIGRE_ADJ_ALL(__nv_bfloat16)
TIGRE_ADJ_ALL(__half)

}  // namespace tigre
