// FDK reconstruction of a circular scan (the paper's analytic reconstruction,
// used for comparison and as an initialiser; Sec. 1 and Sec. 3.2).
//
//   1. each projection pixel is weighted by DSD / sqrt(DSD^2 + u^2 + v^2);
//   2. each detector row is convolved (linear convolution, zero outside the
//      detector) with the Ram-Lak ramp kernel of the detector pitch scaled to
//      the isocentre, tau = du DSO / DSD:  h[0] = 1/(4 tau^2),
//      h[odd k] = -1/(pi k tau)^2, h[even k] = 0, times tau for the sum;
//   3. the filtered projections are backprojected voxel by voxel with the FDK
//      distance weight (DSO/(DSO-s))^2, each angle times half its angular
//      weight (half the angle between its neighbours on the circle).
//
// Step 1, 2 and the angular factor run in one kernel (a block takes 8, 4 or 1
// detector rows into shared memory); step 3 is the voxel-driven backprojector.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace tigre {
namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr int kFdkMaxRowBytes = 160 * 1024;  // the longest detector row

// One block per (row q, angle a): out[a][q][p] = wa * sum_k w(k) y[k] h(p-k).
// The kernel is even and vanishes at even non-zero offsets, so each output
// sums h0 y[p] and h[j] (y[p-j] + y[p+j]) over odd j.
template <typename TP>
__global__ void __launch_bounds__(256) fdk_filter_kernel(const TP* __restrict__ proj,
                                                         float* __restrict__ out,
                                                         const float* __restrict__ h_odd,
                                                         const float* __restrict__ ang_w, int nu,
                                                         int nv, float h0, float u0, float du,
                                                         float v0, float dv, float dsd2)
{
    extern __shared__ float row[];
    const int q = blockIdx.x, a = blockIdx.y;
    const TP* src = proj + ((int64_t)a * nv + q) * nu;
    const float v = fmaf((float)q, dv, v0);
    for (int p = threadIdx.x; p < nu; p += blockDim.x) {
        const float u = fmaf((float)p, du, u0);
        row[p] = to_f32<TP>(src[p]) * sqrtf(dsd2) * rsqrtf(dsd2 + u * u + v * v);
    }
    __syncthreads();
    const float wa = ang_w[a];
    float* dst = out + ((int64_t)a * nv + q) * nu;
    for (int p = threadIdx.x; p < nu; p += blockDim.x) {
        float acc = h0 * row[p];
        // odd offsets j = 1, 3, 5, ...; h_odd[i] holds h at j = 2 i + 1
        for (int j = 1, i = 0; j < nu; j += 2, ++i) {
            const float l = p - j >= 0 ? row[p - j] : 0.0f;
            const float r = p + j < nu ? row[p + j] : 0.0f;
            acc = fmaf(h_odd[i], l + r, acc);
        }
        dst[p] = wa * acc;
    }
}

// The same filter for R rows of one angle per block, as two dense convolutions:
// an even output sums odd inputs only and an odd output even ones, so the rows
// are split by parity.  With G[d] = h at offset 2d + 1 (G[-d - 1] = G[d]), the
// outputs are
//   out[2m + 1] = h0 y[2m + 1] + sum_n G[m - n] y[2n],
//   out[2m]     = h0 y[2m]     + sum_n G[m - n - 1] y[2n + 1].
// A thread makes four neighbouring outputs of one parity for all R rows: per
// four inputs it reads two float4 of G and one of each row (the same for the
// whole warp) for 16 R multiply-adds, so it is bound by FMA where one output
// per thread was bound by two shared-memory loads per multiply-add.
// 509 x 397 x 361 (FP16 in): 6.11 -> 0.95 ms.
constexpr int kFdkThreads = 128;

template <typename TP, int R>
__global__ void __launch_bounds__(kFdkThreads) fdk_filter_rows_kernel(
    const TP* __restrict__ proj, float* __restrict__ out, const float* __restrict__ h_odd,
    const float* __restrict__ ang_w, int nu, int nv, float h0, float u0, float du, float v0,
    float dv, float dsd2)
{
    extern __shared__ float4 shared4[];
    // half rows of H values (a multiple of 4, zero beyond the detector):
    // rows[parity][r][H], then G[-H .. H + 4)
    const int H = ((nu + 1) / 2 + 3) & ~3;
    float* rows = (float*)shared4;
    float* G = rows + 2 * R * H + H;  // (G[0] here)
    const int q0 = blockIdx.x * R, a = blockIdx.y;
    for (int i = threadIdx.x; i < R * 2 * H; i += kFdkThreads) {
        const int r = i / (2 * H), p = i - r * 2 * H, q = q0 + r;
        float y = 0.0f;
        if (q < nv && p < nu) {
            const float v = fmaf((float)q, dv, v0), u = fmaf((float)p, du, u0);
            y = to_f32<TP>(proj[((int64_t)a * nv + q) * nu + p]) * sqrtf(dsd2) *
                rsqrtf(dsd2 + u * u + v * v);
        }
        rows[((p & 1) * R + r) * H + (p >> 1)] = y;
    }
    const int nh = nu / 2;  // odd offsets 1, 3, ... below nu
    for (int d = (int)threadIdx.x - H; d < H + 4; d += kFdkThreads) {
        const int i = d >= 0 ? d : -d - 1;
        G[d] = i < nh ? h_odd[i] : 0.0f;
    }
    __syncthreads();
    const float wa = ang_w[a];
    const int quads = H / 4;
    for (int t = threadIdx.x; t < 2 * quads; t += kFdkThreads) {
        const int par = t >= quads, m = 4 * (t - par * quads);  // outputs 2 (m + i) + par
        const float* in = rows + (1 - par) * R * H;             // inputs of the other parity
        const float* own = rows + par * R * H;
        float acc[R][4];
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[r][i] = 0.0f;
        for (int n = 0; n < H; n += 4) {
            // the centre tap enters between its neighbours, which nearly cancel
            // it on smooth rows: the far taps then add to small sums
            if (n == m)
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[r][i] = fmaf(h0, own[r * H + m + i], acc[r][i]);
            const float4 lo = *(const float4*)(G + m - n - 4), hi = *(const float4*)(G + m - n);
            const float g[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 y = *(const float4*)(in + r * H + n);
                // g[4 + i - j] = G[(m + i) - (n + j)], one earlier for even outputs
                const float yj[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        acc[r][i] = fmaf(par ? g[4 + i - j] : g[3 + i - j], yj[j], acc[r][i]);
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (q0 + r < nv) {
                float* dst = out + ((int64_t)a * nv + q0 + r) * nu;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (2 * (m + i) + par < nu) dst[2 * (m + i) + par] = wa * acc[r][i];
            }
    }
}

}  // namespace

// Angular weight of each angle: half the angle between its two neighbours
// on the circle (2 pi / N for N uniform angles); the FDK factor 1/2 is
// included here.
static std::vector<float> fdk_angle_factors(const std::vector<double>& angles)
{
    const size_t n = angles.size();
    std::vector<float> out(n);
    if (n == 1) {
        out[0] = (float)kPi;  // (2 pi) / 2
        return out;
    }
    const double two_pi = 2.0 * kPi;
    std::vector<std::pair<double, size_t>> s(n);
    for (size_t i = 0; i < n; ++i) s[i] = {std::fmod(std::fmod(angles[i], two_pi) + two_pi, two_pi), i};
    std::sort(s.begin(), s.end());
    for (size_t k = 0; k < n; ++k) {
        const double prev = s[(k + n - 1) % n].first, next = s[(k + 1) % n].first;
        const double gp = std::fmod(s[k].first - prev + two_pi, two_pi);
        const double gn = std::fmod(next - s[k].first + two_pi, two_pi);
        out[s[k].second] = (float)(0.25 * (gp + gn));  // 1/2 (gap mean) x 1/2 (FDK)
    }
    return out;
}

tigre_status fdk_impl(tigre_geometry* g, const void* proj, tigre_dtype pt, void* vol,
                      tigre_dtype vt, cudaStream_t st)
{
    TIGRE_TRY(check_geometry(g));
    if (!proj || !vol) return fail(TIGRE_ERR_INVALID_ARG, "null proj or vol pointer");
    if (!dtype_ok(pt) || !dtype_ok(vt)) return fail(TIGRE_ERR_INVALID_ARG, "bad dtype");
    const tigre_geometry_desc& d = g->desc;
    const int nu = (int)d.n_det[0], nv = (int)d.n_det[1];
    const int64_t na = (int64_t)g->angles.size();
    if ((size_t)nu * sizeof(float) > (size_t)kFdkMaxRowBytes)
        return fail(TIGRE_ERR_UNSUPPORTED, "detector rows longer than 40960 pixels");
    if (nv > 2147483647 || na > 65535) return fail(TIGRE_ERR_UNSUPPORTED, "too many rows or angles");
    // Ram-Lak taps at odd offsets and the angular factors (FP64 on the host).
    const double tau = d.d_det[0] * d.DSO / d.DSD;
    std::vector<float> host((size_t)(nu / 2 + 1) + (size_t)na, 0.0f);
    for (int j = 1, i = 0; j < nu; j += 2, ++i)
        host[(size_t)i] = (float)(-1.0 / (kPi * kPi * (double)j * (double)j * tau));
    const std::vector<float> aw = fdk_angle_factors(g->angles);
    std::copy(aw.begin(), aw.end(), host.begin() + (nu / 2 + 1));
    float* dtab = nullptr;
    float* filt = nullptr;
    TIGRE_CUDA(dev_alloc((void**)&dtab, sizeof(float) * host.size(), st));
    cudaError_t e = dev_alloc((void**)&filt, sizeof(float) * (size_t)(na * nv) * (size_t)nu, st);
    if (e != cudaSuccess) {
        dev_free(dtab, st);
        return cuda_fail(e, "device allocation (fdk filtered projections)");
    }
    tigre_status status = TIGRE_OK;
    e = cudaMemcpyAsync(dtab, host.data(), sizeof(float) * host.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // host table leaves scope after this call
    if (e != cudaSuccess) status = cuda_fail(e, "fdk table upload");
    if (status == TIGRE_OK) {
        const float u0 = (float)(-0.5 * (double)(nu - 1) * d.d_det[0] + d.off_det[0]);
        const float v0 = (float)(-0.5 * (double)(nv - 1) * d.d_det[1] + d.off_det[1]);
        const float h0 = (float)(0.25 / tau);
        const size_t smem = sizeof(float) * (size_t)nu;
        status = dispatch_dtype(pt, [&](auto tag) -> tigre_status {
            using TP = decltype(tag);
            // Blocks of 8 rows up to 2048 columns (73 KB: three per SM), of 4
            // up to 8192 (164 KB: one per SM); longer rows one by one.  360
            // angles, whole call, ms with 8 / 4 / 2 / 1 rows a block and the
            // row-by-row kernel: 512 columns x 64 rows 0.77 / 0.77 / 0.78 / 0.82 /
            // 2.05, 2048 x 64 3.16 / 3.23 / 3.52 / 3.92 / 17.2, 2048 x 9 1.20 / 1.02 /
            // 0.97 / 0.95 / 3.25; 4096 x 9 - / 2.96 / 2.52 / 2.38 / 10.3, 8192 x 9 - /
            // 13.2 / 11.9 / 9.0 / 38.4, 8192 x 1 - / 5.0 / 4.2 / 1.6 / 6.2.  An instance's
            // shared-memory limit is the process's: a call beyond the default
            // 48 KB sets it to what the instance's longest rows need, never to
            // its own rows' bytes, which another thread's launch may exceed
            // (below 48 KB the setting would cost 1 to 2 us of a 43 us call).
            auto rows = [&](auto kern, int R, int nu_max) -> tigre_status {
                const auto bytes = [R](int n) {
                    const int H = ((n + 1) / 2 + 3) & ~3;
                    return (int)sizeof(float) * (2 * R * H + 2 * H + 4);
                };
                if (bytes(nu) > 48 * 1024)
                    TIGRE_CUDA(cudaFuncSetAttribute(
                        kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes(nu_max)));
                kern<<<dim3((unsigned)((nv + R - 1) / R), (unsigned)na), kFdkThreads, bytes(nu), st>>>(
                    (const TP*)proj, filt, dtab, dtab + (nu / 2 + 1), nu, nv, h0, u0,
                    (float)d.d_det[0], v0, (float)d.d_det[1], (float)(d.DSD * d.DSD));
                TIGRE_LAUNCHED("fdk_filter_rows_kernel");
                return TIGRE_OK;
            };
            if (nu <= 2048) return rows(fdk_filter_rows_kernel<TP, 8>, 8, 2048);
            if (nu <= 8192) return rows(fdk_filter_rows_kernel<TP, 4>, 4, 8192);
            if (smem > 48 * 1024)
                TIGRE_CUDA(cudaFuncSetAttribute(fdk_filter_kernel<TP>,
                                                cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                kFdkMaxRowBytes));
            fdk_filter_kernel<TP><<<dim3((unsigned)nv, (unsigned)na), 256, smem, st>>>(
                (const TP*)proj, filt, dtab, dtab + (nu / 2 + 1), nu, nv, h0, u0,
                (float)d.d_det[0], v0, (float)d.d_det[1], (float)(d.DSD * d.DSD));
            TIGRE_LAUNCHED("fdk_filter_kernel");
            return TIGRE_OK;
        });
    }
    if (status == TIGRE_OK)
        status = backward_impl(g, filt, TIGRE_F32, vol, vt, 0, na, TIGRE_BP_FDK, 0, st);
    dev_free(filt, st);
    dev_free(dtab, st);
    return status;
}

}  // namespace tigre

extern "C" tigre_status tigre_fdk(tigre_geometry_t geo, const void* proj, tigre_dtype proj_dtype,
                                  void* vol, tigre_dtype vol_dtype, void* cuda_stream)
{
    return tigre::fdk_impl(geo, proj, proj_dtype, vol, vol_dtype, (cudaStream_t)cuda_stream);
}
