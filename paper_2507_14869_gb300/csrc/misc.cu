// Read-back kernels: posterior mean, label planes, label validation, and the
// image-quality metrics of Section 6 (PSNR, SSIM) in FP64.
#include "pcad_internal.h"

namespace pcad {

namespace {

__global__ void mean_kernel(const float *acc, float n, float *mean, long count)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count)
        mean[i] = acc[i] / n;
}

__global__ void labels_to_float_kernel(const uint8_t *x, int pitch, int H, int W, float *out)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (c < W && r < H)
        out[(size_t)r * W + c] = (float)x[(size_t)r * pitch + c];
}

__global__ void check_labels_kernel(const uint8_t *x, int pitch, int H, int W, int L, int *bad)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (c < W && r < H && (int)x[(size_t)r * pitch + c] >= L)
        atomicAdd(bad, 1);
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// scratch[0] += sum of squared luminance errors; int max label at scratch[7]
__global__ void psnr_kernel(const float *est, const uint8_t *clean, long n, double inv,
                            double *scratch)
{
    double se = 0.0;
    int mx = 0;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long)gridDim.x * blockDim.x) {
        const double d = (double)est[i] * inv - (double)clean[i] * inv;
        se += d * d;
        mx = max(mx, (int)clean[i]);
    }
    se = warp_sum(se);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&scratch[0], se);
        atomicMax(reinterpret_cast<int *>(&scratch[7]), mx);
    }
}

// Mean SSIM over the 11 x 11 Gaussian window (sigma 1.5) in FP64, the window
// as its row and column factors.  GB300 issues 2 FP64 operations per SM and
// clock, so the operation count is the time: one pass per row over the 4
// blurred fields x, y, x^2 + y^2 and xy (SSIM uses the two variances only
// through their sum), 11 taps along the row and 11 down the column, 88 fused
// operations per position against 605 products and sums for the 121 taps of
// the window taken at every position.  Measured: 8192^2 170 ms before, 15.3 ms
// now (the FP64 rate alone bounds it near 12 ms); 512^2 0.69 ms and 0.10 ms.
//
// A block of 128 threads walks down `rows` + 10 rows of 128 window columns: it
// stages the row's fields, each thread blurs its 11 columns and, from the 11th
// row on, takes the column sums of the position that ends there from its own
// ring of the last 10 rows in shared memory.
constexpr int kSsThreads = 128;
constexpr int kSsTap = 11;
constexpr int kSsSpan = kSsThreads + kSsTap - 1;

struct SsimWeights {
    double w[kSsTap];   // sum 1
};

__global__ void __launch_bounds__(kSsThreads)
    ssim_window_kernel(const float *est, const uint8_t *clean, int H, int W, int rows,
                       const SsimWeights k, double inv, double *scratch)
{
    __shared__ double b[4][kSsSpan];
    __shared__ double ring[kSsTap - 1][4][kSsThreads];
    const int tid = (int)threadIdx.x;
    const int c0 = (int)blockIdx.x * kSsThreads, r0 = (int)blockIdx.y * rows;
    const int rend = min(r0 + rows + kSsTap - 1, H);
    const bool own = c0 + tid < W - (kSsTap - 1);
    double sum = 0.0;
    int slot = 0;   // the ring's oldest row
    for (int r = r0; r < rend; ++r) {
        __syncthreads();   // the last row's fields are read
        for (int i = tid; i < kSsSpan; i += kSsThreads) {
            const int c = c0 + i;
            double x = 0.0, y = 0.0;
            if (c < W) {
                x = (double)clean[(size_t)r * W + c] * inv;
                y = (double)est[(size_t)r * W + c] * inv;
            }
            b[0][i] = x;
            b[1][i] = y;
            b[2][i] = x * x + y * y;
            b[3][i] = x * y;
        }
        __syncthreads();
        double h[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < kSsTap; ++a)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                h[q] += k.w[a] * b[q][tid + a];
        double m[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            m[q] = k.w[kSsTap - 1] * h[q];
        if (r - r0 >= kSsTap - 1) {
            int at = slot;
#pragma unroll
            for (int a = 0; a < kSsTap - 1; ++a) {
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    m[q] += k.w[a] * ring[at][q][tid];
                at = at + 1 == kSsTap - 1 ? 0 : at + 1;
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            ring[slot][q][tid] = h[q];
        slot = slot + 1 == kSsTap - 1 ? 0 : slot + 1;
        if (r - r0 < kSsTap - 1 || !own)
            continue;
        const double c1 = 1e-4, c2 = 9e-4;
        const double mm = m[0] * m[1], m2 = m[0] * m[0] + m[1] * m[1];
        sum += ((2.0 * mm + c1) * (2.0 * (m[3] - mm) + c2)) / ((m2 + c1) * (m[2] - m2 + c2));
    }
    sum = warp_sum(sum);
    if ((tid & 31) == 0)
        atomicAdd(&scratch[1], sum);
}

// Single-window (printed) form for images smaller than the window: two-pass
// unbiased sample statistics.
__global__ void ssim_global_kernel(const float *est, const uint8_t *clean, long n, double inv,
                                   double *scratch)
{
    if (blockIdx.x != 0 || threadIdx.x != 0)
        return;
    double sx = 0, sy = 0;
    for (long i = 0; i < n; ++i) {
        sx += (double)clean[i] * inv;
        sy += (double)est[i] * inv;
    }
    const double mx = sx / (double)n, my = sy / (double)n;
    double vx = 0, vy = 0, cxy = 0;
    for (long i = 0; i < n; ++i) {
        const double dx = (double)clean[i] * inv - mx;
        const double dy = (double)est[i] * inv - my;
        vx += dx * dx;
        vy += dy * dy;
        cxy += dx * dy;
    }
    vx /= (double)(n - 1);
    vy /= (double)(n - 1);
    cxy /= (double)(n - 1);
    const double c1 = 1e-4, c2 = 9e-4;
    scratch[1] = ((2 * mx * my + c1) * (2 * cxy + c2)) / ((mx * mx + my * my + c1) * (vx + vy + c2));
}

__global__ void metrics_finish_kernel(const double *scratch, long n, long npos, double inv,
                                      double *out)
{
    if (blockIdx.x != 0 || threadIdx.x != 0)
        return;
    const double mse = scratch[0] / (double)n;
    const int mxl = *reinterpret_cast<const int *>(&scratch[7]);
    const double peak = (double)mxl * inv;
    out[0] = mse == 0.0 ? (double)INFINITY : 20.0 * log10(peak / sqrt(mse));
    out[1] = npos > 0 ? scratch[1] / (double)npos : scratch[1];
}

}  // namespace

cudaError_t launch_mean(const float *acc, float n, float *mean, long count, cudaStream_t s)
{
    const int bs = 256;
    const long nb = (count + bs - 1) / bs;
    if (nb > 0)
        mean_kernel<<<(unsigned)nb, bs, 0, s>>>(acc, n, mean, count);
    return cudaGetLastError();
}

cudaError_t launch_labels_to_float(const uint8_t *x, int pitch, int H, int W, float *out,
                                   cudaStream_t s)
{
    dim3 grid((W + 255) / 256, H);
    labels_to_float_kernel<<<grid, 256, 0, s>>>(x, pitch, H, W, out);
    return cudaGetLastError();
}

// From this size on rows with gaps are packed on the device before they are read:
// host memory that no one has touched yet (what an allocator hands out from 128 KB
// on) takes a linear copy faster, 300^2 133 us against 381, 1000^2 235 against 1083,
// 8191 x 8189 2.8 ms against 46; in memory touched before, where the copy itself
// counts, packing costs 5 us (1000^2 29 against 24).
constexpr size_t kPackBytes = 128 << 10;

cudaError_t read_labels(uint8_t *host, int host_pitch, const uint8_t *x, int pitch, int H, int W,
                        void *packed, cudaStream_t s)
{
    if (host_pitch != W || (pitch != W && (size_t)H * W < kPackBytes))
        return cudaMemcpy2DAsync(host, host_pitch, x, pitch, W, H, cudaMemcpyDeviceToHost, s);
    if (pitch != W) {
        const cudaError_t e =
            cudaMemcpy2DAsync(packed, W, x, pitch, W, H, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess)
            return e;
        x = static_cast<const uint8_t *>(packed);
    }
    return cudaMemcpyAsync(host, x, (size_t)H * W, cudaMemcpyDeviceToHost, s);
}

cudaError_t launch_check_labels(const uint8_t *x, int pitch, int H, int W, int L, int *bad,
                                cudaStream_t s)
{
    dim3 grid((W + 255) / 256, H);
    check_labels_kernel<<<grid, 256, 0, s>>>(x, pitch, H, W, L, bad);
    return cudaGetLastError();
}

cudaError_t launch_metrics(const float *est, const uint8_t *clean, int H, int W, int L,
                           double *scratch, double *out, cudaStream_t s)
{
    cudaError_t e;
    e = cudaMemsetAsync(scratch, 0, 8 * sizeof(double), s);
    if (e != cudaSuccess)
        return e;
    const long n = (long)H * W;
    const double inv = 1.0 / (double)(L - 1);
    psnr_kernel<<<256, 256, 0, s>>>(est, clean, n, inv, scratch);
    long npos = 0;
    if (H >= 11 && W >= 11) {
        SsimWeights k;
        double tot = 0.0;
        for (int a = 0; a < kSsTap; ++a) {
            const double d = (double)a - 5.0;
            k.w[a] = exp(-(d * d) / (2.0 * 1.5 * 1.5));
            tot += k.w[a];
        }
        for (int a = 0; a < kSsTap; ++a)
            k.w[a] /= tot;
        // rows per block: every block repeats 10 rows of row blurs, so as many
        // rows as still leave a block per SM (one resident block saturates the
        // FP64 pipe), 128 at most
        int dev = 0, sms = 1;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
            return e;
        const int nc = (W - 10 + kSsThreads - 1) / kSsThreads, nr = H - 10;
        const long per = ((long)nr * nc + sms - 1) / sms;
        const int rows = (int)(per > 128 ? 128 : per);
        ssim_window_kernel<<<dim3(nc, (nr + rows - 1) / rows), kSsThreads, 0, s>>>(
            est, clean, H, W, rows, k, inv, scratch);
        npos = (long)(H - 10) * (W - 10);
    } else {
        ssim_global_kernel<<<1, 32, 0, s>>>(est, clean, n, inv, scratch);
    }
    metrics_finish_kernel<<<1, 32, 0, s>>>(scratch, n, npos, inv, out);
    return cudaGetLastError();
}

}  // namespace pcad
