// Welch power spectral density of observer pressure series (Section 3.3: the
// PSD of the pressure fluctuations by Welch's method with three Hann windows
// and 50% overlap).  Readings, shared with the declaration in fr.h: segment
// length L = 2 floor(nt / (nseg + 1)), step L / 2, periodic Hann window, each
// segment's mean removed, one-sided density averaged over the segments.
//
// Two kernels, all FP64: the table of cos/sin(2 pi m / L) and the windowed,
// mean-free segments y_n folded about L / 2 (one block per observer and segment,
// fixed-order reduction); and a direct DFT of the folded segments, one warp per
// pair of frequencies.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "fr.h"
#include "fr_pool.h"

int fr_set_error_from_fwh(int code, const char* msg);

namespace {

// Blocks x < nseg: segment x of observer y, folded: with y_n = w_n (x_n - mean),
// w_n = (1 - cos(2 pi n / L)) / 2 and H = L / 2, ws[o][s][0][n] = y_n + y_{L-n},
// ws[o][s][1][n] = y_n - y_{L-n} for 0 < n < H; y_n and 0 at n = 0 and H.
// Blocks x = nseg, together: the table cs[m] = (cos, sin)(2 pi m / L).
__global__ void k_psd_segments(const double* __restrict__ p, int ld, int L, double2* __restrict__ cs,
                               double* __restrict__ ws) {
    const int s = blockIdx.x, o = blockIdx.y, nseg = int(gridDim.x) - 1, H = L / 2;
    if (s == nseg) {
        for (int64_t m = int64_t(o) * blockDim.x + threadIdx.x; m < L; m += int64_t(gridDim.y) * blockDim.x) {
            double sn, c;
            sincospi(2.0 * double(m) / double(L), &sn, &c);
            cs[m] = make_double2(c, sn);
        }
        return;
    }
    const double* x = p + size_t(o) * ld + size_t(s) * H;
    __shared__ double red[256];
    double acc = 0.0;
    for (int n = threadIdx.x; n < L; n += blockDim.x) acc += x[n];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if (threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
        __syncthreads();
    }
    const double mean = red[0] / double(L);
    double* even = ws + (size_t(o) * nseg + s) * 2 * (H + 1);
    double* odd = even + H + 1;
    for (int n = threadIdx.x; n <= H; n += blockDim.x) {
        double sn, c;
        sincospi(2.0 * double(n) / double(L), &sn, &c);
        const double w = 0.5 - 0.5 * c, a = w * (x[n] - mean);
        const bool mid = n > 0 && n < H;
        const double b = mid ? w * (x[L - n] - mean) : 0.0;   // w_{L-n} = w_n
        even[n] = a + b;
        odd[n] = mid ? a - b : 0.0;
    }
}

// psd[o][k] = scale_k * mean over segments of |sum_n y_n e^{-2 pi i k n / L}|^2.
// A warp forms frequencies k and H - k (H = L / 2) from the same products: with
// theta = 2 pi k n / L the angle of H - k is pi n - theta, so its cosine and sine
// are (-1)^n cos and -(-1)^n sin theta, and the sums over even and odd n give both
// frequencies.  With the fold about H that is a quarter of the direct sum's FP64
// operations.  Lane l takes n = l (mod 32), so its n keep their parity, and walks
// the twiddle index k n mod L without a division.  Bound by latency at one
// observer (a chain of H / 32 steps; L = 974: 264 us with one thread per frequency, 30 us
// here) and by the FP64 pipe at many (36 observers, L = 324: 28 us).
constexpr int PSD_WARPS = 8, PSD_SEG = 4;
__global__ void __launch_bounds__(32 * PSD_WARPS) k_psd_dft(const double* __restrict__ ws, int nseg, int L,
                                                            const double2* __restrict__ cs, double inv_norm,
                                                            double* __restrict__ psd, int cap) {
    const int o = blockIdx.y, lane = threadIdx.x & 31, H = L / 2;
    const int k = blockIdx.x * PSD_WARPS + (threadIdx.x >> 5);
    if (2 * k > H) return;
    const int step = int((32ll * k) % L), idx0 = int((static_cast<long long>(k) * lane) % L);
    double pa = 0.0, pb = 0.0;   // powers at k and H - k, summed over the segments
    for (int s0 = 0; s0 < nseg; s0 += PSD_SEG) {
        const int ns = min(PSD_SEG, nseg - s0);
        const double* y = ws + (size_t(o) * nseg + s0) * 2 * (H + 1);
        double re[PSD_SEG], im[PSD_SEG];
#pragma unroll
        for (int s = 0; s < PSD_SEG; ++s) re[s] = im[s] = 0.0;
        int idx = idx0;
        for (int n = lane; n <= H; n += 32) {
            const double2 t = cs[idx];
#pragma unroll
            for (int s = 0; s < PSD_SEG; ++s)
                if (s < ns) {
                    re[s] += y[s * 2 * (H + 1) + n] * t.x;
                    im[s] -= y[(s * 2 + 1) * (H + 1) + n] * t.y;
                }
            idx += step;
            if (idx >= L) idx -= L;
        }
#pragma unroll
        for (int s = 0; s < PSD_SEG; ++s) {
#pragma unroll
            for (int d = 16; d > 1; d >>= 1) {
                re[s] += __shfl_xor_sync(0xffffffffu, re[s], d);
                im[s] += __shfl_xor_sync(0xffffffffu, im[s], d);
            }
            const double ro = __shfl_xor_sync(0xffffffffu, re[s], 1), io = __shfl_xor_sync(0xffffffffu, im[s], 1);
            // lane 0: (re, im) over even n, (ro, io) over odd n
            const double ra = re[s] + ro, ia = im[s] + io, rb = re[s] - ro, ib = io - im[s];
            if (s < ns) {
                pa += ra * ra + ia * ia;
                pb += rb * rb + ib * ib;
            }
        }
    }
    if (lane != 0) return;
    const double c = (k == 0 ? 1.0 : 2.0) * inv_norm / double(nseg);
    psd[size_t(o) * cap + k] = c * pa;
    if (2 * k != H) psd[size_t(o) * cap + H - k] = c * pb;
}

}  // namespace

extern "C" int fwh_psd(const double* p, int nobs, int nt, int ld, double dt, int nseg, double* psd, int cap,
                       int* nfreq_out, void* stream) {
    if (!p || !psd || !nfreq_out) return fr_set_error_from_fwh(FR_EINVAL, "null argument");
    if (nobs < 1 || nseg < 1 || ld < nt || !(dt > 0.0))
        return fr_set_error_from_fwh(FR_EINVAL, "bad sizes (nobs >= 1, nseg >= 1, ld >= nt, dt > 0 required)");
    const int L = 2 * (nt / (nseg + 1));
    if (L < 2) return fr_set_error_from_fwh(FR_EINVAL, "record too short for the segments");
    const int nf = L / 2 + 1;
    if (cap < nf) return fr_set_error_from_fwh(FR_EINVAL, "output capacity below L/2 + 1 frequencies");
    if (nobs > 65535) return fr_set_error_from_fwh(FR_EINVAL, "too many observers for one launch");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // sum of the squared window, on the host in double
    double w2 = 0.0;
    for (int n = 0; n < L; ++n) {
        const double w = 0.5 - 0.5 * std::cos(2.0 * M_PI * double(n) / double(L));
        w2 += w * w;
    }
    const double inv_norm = dt / w2;   // 1 / (f_s sum w^2)
    // one allocation: the table, then the folded segments
    const size_t bytes = sizeof(double2) * size_t(L) + sizeof(double) * size_t(nobs) * nseg * (L + 2);
    void* buf = nullptr;
    const bool pooled = fr_pool_alloc(&buf, bytes, s);
    if (!pooled && cudaMalloc(&buf, bytes) != cudaSuccess)
        return fr_set_error_from_fwh(FR_ENOMEM, "cannot allocate PSD scratch");
    double2* cs = static_cast<double2*>(buf);
    double* ws = reinterpret_cast<double*>(cs + L);
    k_psd_segments<<<dim3(nseg + 1, nobs), 256, 0, s>>>(p, ld, L, cs, ws);
    k_psd_dft<<<dim3((L / 4 + PSD_WARPS) / PSD_WARPS, nobs), 32 * PSD_WARPS, 0, s>>>(ws, nseg, L, cs, inv_norm, psd, cap);
    cudaError_t err = cudaGetLastError();
    if (err == cudaSuccess) err = cudaStreamSynchronize(s);
    if (pooled) fr_pool_free(buf, s);
    else cudaFree(buf);
    if (err != cudaSuccess) return fr_set_error_from_fwh(FR_ECUDA, cudaGetErrorString(err));
    *nfreq_out = nf;
    return FR_OK;
}
