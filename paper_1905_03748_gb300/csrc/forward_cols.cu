// Interpolated forward projector of whole volumes, warps of detector columns
// (the same sums as every other forward kernel, bit for bit).
//
// The rays of one detector column at one angle lie in one vertical plane, so
// they cross the same (x, y) cells and differ in z.  A lane is a detector row
// and the quads are stored with z fastest: the lanes of a column read
// neighbouring quads (16 bytes x the row spacing, about 1.15 planes), the
// second quad of a sample (plane s + 1) is the next element, and one layout
// serves every angle (half the workspace and half the build of the two layouts
// the row-warp kernel needs).
//
//  * Reuse.  Steps are half a voxel, so a sample's cell is often the previous
//    sample's.  The quads stay in registers and a lane loads only when its
//    element changes; the lanes of a column change cells nearly together.
//  * Two rays per lane (two columns), so that positions, splits and sums are
//    packed FP32 pairs (FFMA2 / FADD2): 26 warp instructions per 32 samples
//    instead of 38, the same roundings.
//  * Lock step.  A ray's samples are shifted by whole steps so that all lanes
//    are at the same depth; between the last ray's entry and the first ray's
//    exit no lane tests anything, before and after it each tests its range.
//  * Blocks of four neighbouring angles at one tile of columns share lines in
//    L1; 128 threads at 9 blocks per SM (56 registers; what the march does not
//    need is kept in shared memory).
//
// Measured (before: 16 pixels x 2 angles per warp, two layouts): 512^3 x 360
// 112.0 -> 90.5 ms, 256^3 x 90 (384^2) 7.1 -> 5.9, 1024^3 x 90 287 -> 209,
// 64^3 x 20 (128^2) 0.098 -> 0.079.  Bound (512^3 x
// 36 of 360 angles, ncu): L1 data pipe 78 %, FMA pipe 59 %, issue 50 %.  Not
// better: 48 registers at 10 blocks (spills: 116 ms at 512^3 x 360), 256
// threads at 4 blocks (97.1), 512 and 1024 threads (101, 108), warps of 32
// rows (111: the planes in use no longer fit L2), L1 prefetches 4 or 8 samples
// ahead (117), shifts that align the rays' middles (no change).
#include <algorithm>

#include "forward_cols.cuh"
#include "quad.cuh"
#include "ray.cuh"

namespace tigre {
namespace {

constexpr int kColWarps = 4;   // warps per block, angles per group
constexpr int kColBlocks = 9;  // blocks per SM (56 registers)

// Element (y, x, s) of the column quads, s fastest: the bilinear coefficients
// of the cell (x, x+1) x (y, y+1) of plane s of the zero-bordered volume.  A
// block makes 32 planes x 32 x of four y rows from five rows read along x, all
// its loads in flight at once (a march over eight rows, two barriers each,
// waited for memory nine times: 64^3 13.4 -> 3.6 us, 192^3 38.6 -> 24.9, 1024^3
// 4.5 -> 3.24 ms).  Bound by the 16-byte writes (5.4 TB/s at 1024^3).
constexpr int kQuadRows = 4;
template <typename T>
__global__ void __launch_bounds__(256) quad_columns_kernel(const T* __restrict__ vol,
                                                           float4* __restrict__ out, int nx, int ny,
                                                           int nz)
{
    __shared__ float tile[kQuadRows + 1][32][33];  // [y][z][x]
    const int PX = nx + 2 * kPad, PY = ny + 2 * kPad, PS = nz + 2 * kPad;
    const int s0 = blockIdx.x * 32, x0 = blockIdx.y * 32;
    const int lane = threadIdx.x, w = threadIdx.y;
    auto tap = [&](int yp, int i, int j) -> float {  // padded row, plane s0 + i, column x0 + j
        const int z = s0 + i - kPad, y = yp - kPad, x = x0 + j - kPad;
        const bool in = (unsigned)z < (unsigned)nz && (unsigned)y < (unsigned)ny &&
                        (unsigned)x < (unsigned)nx;
        return in ? to_f32<T>(vol[((int64_t)z * ny + y) * nx + x]) : 0.0f;
    };
    for (int64_t y0 = (int64_t)blockIdx.z * kQuadRows; y0 < PY; y0 += (int64_t)gridDim.z * kQuadRows) {
        __syncthreads();
#pragma unroll
        for (int u = 0; u < (kQuadRows + 1) * 4; ++u)
            tile[u / 4][(u % 4) * 8 + w][lane] = tap((int)y0 + u / 4, (u % 4) * 8 + w, lane);
        if (w < kQuadRows + 1) tile[w][lane][32] = tap((int)y0 + w, lane, 32);
        __syncthreads();
        const int s = s0 + lane;
        if (s < PS)
            for (int r = 0; r < kQuadRows && y0 + r < PY; ++r)
                for (int j = w; j < 32 && x0 + j < PX; j += 8)
                    out[((y0 + r) * PX + x0 + j) * PS + s] =
                        bilinear_coefficients(tile[r][lane][j], tile[r][lane][j + 1],
                                              tile[r + 1][lane][j], tile[r + 1][lane][j + 1]);
    }
}

// Both quads of a sample (planes s and s+1, adjacent in memory) when the
// element differs from the one the registers hold.
__device__ __forceinline__ void load_cell(const float4* __restrict__ q, uint32_t e, uint32_t& cur,
                                          float4& lo, float4& hi)
{
    // 16 e as a shift of both halves: an add on the integer pipe, where a wide
    // multiply-add would load the busier FMA pipe (with the march unrolled by
    // four, 512^3 x 360 92.8 -> 90.5 ms, 192^3 x 20 (320^2) 0.758 -> 0.717).
    const uint64_t byte = ((uint64_t)(e >> 28) << 32) | (e << 4);
    const float4* p = (const float4*)((const char*)q + byte);
    asm("{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %8, %9;\n\t"
        "@p ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%10];\n\t"
        "@p ld.global.nc.v4.f32 {%4, %5, %6, %7}, [%10+16];\n\t}"
        : "+f"(lo.x), "+f"(lo.y), "+f"(lo.z), "+f"(lo.w), "+f"(hi.x), "+f"(hi.y), "+f"(hi.z),
          "+f"(hi.w)
        : "r"(e), "r"(cur), "l"(p));
    cur = e;
}

struct ColGeom {
    uint32_t SX, SY;  // quads between x and y neighbours
    uint32_t bias;    // of an element index built from split_bits parts
    int ag;  // angles per block: 1 (at four tiles of columns) or kColWarps (at one)
    int na;     // angles of the launch (a batch has its table, or one angle a block)
    int tiles;  // row tiles of one member
    int64_t vol_stride, proj_stride;  // between a batch's members
};

template <typename TP, bool BATCH, int ROWS>
__global__ void __launch_bounds__(32 * kColWarps, kColBlocks) fwd_cols_kernel(
    const float4* __restrict__ quads, TP* __restrict__ proj, const FwdAngle* __restrict__ params,
    FwdConst c, int a_first, const int* __restrict__ order, ColGeom w)
{
    const unsigned full = 0xffffffffu;
    // what the march does not need stays out of its registers
    __shared__ int cold_K[2][32 * kColWarps], cold_shift[2][32 * kColWarps];
    __shared__ float cold_h[2][32 * kColWarps];
    const int tid = threadIdx.y * 32 + threadIdx.x;
    constexpr int G = 32 / ROWS;  // columns per warp and ray slot
    const int warp = threadIdx.y;
    float x0[3][2], d[3][2];
    float2 acc = make_float2(0.0f, 0.0f);
    int jb = 0, je = 1 << 30, J = 0;
    {
        const int member = BATCH ? (int)blockIdx.z / w.tiles : 0;
        if (BATCH) quads += member * w.vol_stride;
        const int tile = (int)blockIdx.z - member * w.tiles;
        const int pw = 2 * G * (w.ag == 1 ? (int)blockIdx.x * kColWarps + warp : (int)blockIdx.x);
        const int p0 = pw + (int)threadIdx.x / ROWS;
        const int q = tile * ROWS + (int)threadIdx.x % ROWS;
        const int g = (int)blockIdx.y * w.ag + (w.ag == 1 ? 0 : warp);
        const int a = order ? order[g] : g;
        if (a < 0 || (!BATCH && a >= w.na) || pw >= c.nu) return;  // the whole warp
        const FwdAngle* P = params + a_first + a;
        const int layout = P->layout;
        bool active[2];
        float dep0[2], ddep[2];
        int K[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const bool inside = q < c.nv && p0 + G * r < c.nu;
            Ray T;
            T.K = 0;
            T.ok = true;
            T.h = 0.0f;
            if (inside) setup_ray(P, c, p0 + G * r, q, T);
            active[r] = inside && T.ok && T.K > 0;
            cold_h[r][tid] = T.ok ? T.h : __int_as_float(0x7fc00000);
            K[r] = active[r] ? T.K : 0;
            // a ray without samples rests in a corner cell of the border
            x0[0][r] = !active[r] ? 1.0f : layout ? T.x0[1] : T.x0[0];
            x0[1][r] = !active[r] ? 1.0f : layout ? T.x0[0] : T.x0[1];
            x0[2][r] = !active[r] ? 1.0f : T.x0[2];
            d[0][r] = !active[r] ? 0.0f : layout ? T.d[1] : T.d[0];
            d[1][r] = !active[r] ? 0.0f : layout ? T.d[0] : T.d[1];
            d[2][r] = !active[r] ? 0.0f : T.d[2];
            dep0[r] = active[r] ? T.x0[1] : 0.0f;
            ddep[r] = active[r] ? T.d[1] : 0.0f;
        }
        const bool pos = __all_sync(full, (!active[0] || ddep[0] > 0.0f) && (!active[1] || ddep[1] > 0.0f));
        const bool neg = __all_sync(full, (!active[0] || ddep[0] < 0.0f) && (!active[1] || ddep[1] < 0.0f));
        float Y0 = 3.0e38f, D = 1.0e-30f;
        const float sgn = neg ? -1.0f : 1.0f;
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (active[r]) {
                Y0 = fminf(Y0, sgn * dep0[r]);
                D = fmaxf(D, fabsf(ddep[r]));
            }
        for (int o = 16; o > 0; o >>= 1) {
            Y0 = fminf(Y0, __shfl_xor_sync(full, Y0, o));
            D = fmaxf(D, __shfl_xor_sync(full, D, o));
        }
        int kmax = __reduce_max_sync(full, max(K[0], K[1]));
        int shift[2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            shift[r] = active[r] && (pos || neg) ? (int)fminf((sgn * dep0[r] - Y0) / D, 1.0e8f) : 0;
            J = max(J, shift[r] + K[r]);
        }
        J = __reduce_max_sync(full, J);
        // Warps whose rays cross far-apart corners in a step or two would
        // march the gap between them: those start together instead.
        const bool align = J <= 2 * kmax + 64;
        if (!align) J = kmax;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (!align) shift[r] = 0;
            if (active[r]) {
                jb = max(jb, shift[r]);
                je = min(je, shift[r] + K[r]);
            }
            cold_K[r][tid] = K[r];
            cold_shift[r][tid] = shift[r];
        }
        jb = __reduce_max_sync(full, jb);
        je = __reduce_min_sync(full, je);
        if (je < jb || J == 0) jb = je = J;  // (J = 0: no ray of the warp has samples)
    }
    const float2 x0x = make_float2(x0[0][0], x0[0][1]), dx = make_float2(d[0][0], d[0][1]);
    const float2 x0y = make_float2(x0[1][0], x0[1][1]), dy = make_float2(d[1][0], d[1][1]);
    const float2 x0s = make_float2(x0[2][0], x0[2][1]), ds = make_float2(d[2][0], d[2][1]);
    const float2 half = make_float2(8388607.5f, 8388607.5f), two23 = make_float2(8388608.0f, 8388608.0f);
    auto edge = [&](int j) {
        float s[2] = {0.0f, 0.0f};
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = j - cold_shift[r][tid];
            if ((unsigned)k < (unsigned)cold_K[r][tid]) {
                const float kf = (float)k;
                uint32_t bx, by, bs;
                float ax, ay, as;
                split_bits(fmaf(kf, d[0][r], x0[0][r]), bx, ax);
                split_bits(fmaf(kf, d[1][r], x0[1][r]), by, ay);
                split_bits(fmaf(kf, d[2][r], x0[2][r]), bs, as);
                const float4* p = quads + (by * w.SY + bx * w.SX + bs - w.bias);
                const float c0 = bilinear_value(load_quad(p), ax, ay);
                const float c1 = bilinear_value(load_quad(p + 1), ax, ay);
                s[r] = fmaf(as, c1 - c0, c0);
            }
        }
        acc = __fadd2_rn(acc, make_float2(s[0], s[1]));  // + 0 where not taken
    };
    for (int j = 0; j < jb; ++j) edge(j);
    {
        float2 kf = make_float2((float)(jb - cold_shift[0][tid]), (float)(jb - cold_shift[1][tid]));
        uint32_t cur0 = ~0u, cur1 = ~0u;
        float4 lo0 = make_float4(0, 0, 0, 0), hi0 = lo0, lo1 = lo0, hi1 = lo0;
#pragma unroll 4
        for (int j = jb; j < je; ++j) {
            const float2 px = __ffma2_rn(kf, dx, x0x), py = __ffma2_rn(kf, dy, x0y),
                         ps = __ffma2_rn(kf, ds, x0s);
            kf = __fadd2_rn(kf, make_float2(1.0f, 1.0f));
            const float2 mx = __fadd2_rn(px, half), my = __fadd2_rn(py, half), ms = __fadd2_rn(ps, half);
            const uint32_t e0 = __float_as_uint(my.x) * w.SY + __float_as_uint(mx.x) * w.SX +
                                __float_as_uint(ms.x) - w.bias;
            const uint32_t e1 = __float_as_uint(my.y) * w.SY + __float_as_uint(mx.y) * w.SX +
                                __float_as_uint(ms.y) - w.bias;
            load_cell(quads, e0, cur0, lo0, hi0);
            load_cell(quads, e1, cur1, lo1, hi1);
            const float2 ax = sub2(px, sub2(mx, two23)), ay = sub2(py, sub2(my, two23)),
                         as = sub2(ps, sub2(ms, two23));
            const float2 c0 = make_float2(bilinear_value(lo0, ax.x, ay.x), bilinear_value(lo1, ax.y, ay.y));
            const float2 c1 = make_float2(bilinear_value(hi0, ax.x, ay.x), bilinear_value(hi1, ax.y, ay.y));
            acc = __fadd2_rn(acc, __ffma2_rn(as, sub2(c1, c0), c0));
        }
    }
    for (int j = je; j < J; ++j) edge(j);
    {
        const int member = BATCH ? (int)blockIdx.z / w.tiles : 0;
        if (BATCH) proj += member * w.proj_stride;
        const int tile = (int)blockIdx.z - member * w.tiles;
        const int p0 = 2 * G * (w.ag == 1 ? (int)blockIdx.x * kColWarps + warp : (int)blockIdx.x) +
                       (int)threadIdx.x / ROWS;
        const int q = tile * ROWS + (int)threadIdx.x % ROWS;
        const int g = (int)blockIdx.y * w.ag + (w.ag == 1 ? 0 : warp);
        const int a = order ? order[g] : g;
#pragma unroll
        for (int r = 0; r < 2; ++r)
            if (q < c.nv && p0 + G * r < c.nu)
                proj[((int64_t)a * c.nv + q) * c.nu + p0 + G * r] =
                    from_f32<TP>((r ? acc.y : acc.x) * cold_h[r][tid]);
    }
}

}  // namespace

template <typename T>
tigre_status build_quad_columns(const tigre_geometry_desc& d, const T* vol, float4* out,
                                cudaStream_t st)
{
    const int nx = (int)d.n_voxel[0], ny = (int)d.n_voxel[1], nz = (int)d.n_voxel[2];
    const int PX = nx + 2 * kPad, PY = ny + 2 * kPad, PS = nz + 2 * kPad;
    dim3 grid((unsigned)((PS + 31) / 32), (unsigned)((PX + 31) / 32),
              (unsigned)std::min((PY + kQuadRows - 1) / kQuadRows, 65535));
    quad_columns_kernel<T><<<grid, dim3(32, 8), 0, st>>>(vol, out, nx, ny, nz);
    TIGRE_LAUNCHED("quad_columns_kernel");
    return TIGRE_OK;
}

template <typename TP>
tigre_status launch_forward_columns(tigre_geometry* g, const float4* quads, TP* proj, int a_first,
                                    int64_t na, const ColGroups& groups, int batch,
                                    int64_t vol_stride, int64_t proj_stride, cudaStream_t st)
{
    const FwdConst c = make_fwd_const(g);
    // Warps of 8 detector rows x 8 columns, or 16 x 4 on planes of quads larger
    // than 6.5 MB, where fewer strips of planes then live in L2 at a time, if the
    // detector is tall (16-row / 8-row ms, 60 angles of 256 rows: 640^2 13.8 /
    // 14.1, 1024^2 39.4 / 40.4; of 1024 rows: 1024^2 160 / 180) or one such warp
    // holds all its rows (640^2 x 16, 180 angles: 3.15 / 3.44).  Between the two
    // the taller tile costs more than it saves (180 angles: 1024^2 of 24 rows 18.6
    // / 14.1, 64 rows 33.9 / 31.2, 192 rows 80.8 / 79.0), and on small planes always
    // (512^3 x 360: 94.5 / 93.3, 128^3 x 90: 0.519 / 0.495).
    const bool large = (int64_t)c.nx * c.ny >= 640 * 640;
    const int rows = large && (c.nv >= 224 || c.nv <= 16) ? 16 : 8;
    const int ag = groups.four ? kColWarps : 1;
    const int cols = 2 * (32 / rows) * (kColWarps / ag), tiles = (c.nv + rows - 1) / rows;
    dim3 grid((unsigned)((c.nu + cols - 1) / cols), (unsigned)groups.count, (unsigned)(tiles * batch));
    ColGeom w;
    w.SX = (uint32_t)(c.nz + 2 * kPad);
    w.SY = w.SX * (uint32_t)(c.nx + 2 * kPad);
    w.bias = 0x4B000000u * (w.SY + w.SX + 1u);
    w.ag = ag;
    w.na = (int)na;
    w.tiles = tiles;
    w.vol_stride = vol_stride;
    w.proj_stride = proj_stride;
    auto kern = batch > 1 ? (rows == 16 ? fwd_cols_kernel<TP, true, 16> : fwd_cols_kernel<TP, true, 8>)
                          : (rows == 16 ? fwd_cols_kernel<TP, false, 16> : fwd_cols_kernel<TP, false, 8>);
    kern<<<grid, dim3(32, kColWarps), 0, st>>>(quads, proj, (const FwdAngle*)g->fwd_params.ptr, c,
                                               a_first, groups.table, w);
    TIGRE_LAUNCHED("fwd_cols_kernel");
    return TIGRE_OK;
}

#define TIGRE_COLS(T)                                                                           \
    template tigre_status build_quad_columns<T>(const tigre_geometry_desc&, const T*, float4*,  \
                                                cudaStream_t);                                  \
    template tigre_status launch_forward_columns<T>(tigre_geometry*, const float4*, T*, int,    \
                                                    int64_t, const ColGroups&, int, int64_t,    \
                                                    int64_t, cudaStream_t);
TIGRE_COLS(float)
TIGRE_COLS(__nv_bfloat16)
TIGRE_COLS(__half)

}  // namespace tigre
