// CKKS encoding and decoding on the device (Table 1 "encode" / "decode"):
// the canonical embedding evaluates the plaintext polynomial m at the
// primitive 2N-th roots zeta^(5^k) (slot k < N/2) and their conjugates.
// With zeta = exp(i pi / N) and omega = zeta^2,
//     m(zeta^(2j+1)) = sum_i (m_i zeta^i) omega^(i j),
// so all N evaluations are one length-N DFT of the twisted coefficients:
//   encode: E[j(k)] = scale z_k, E[j'(k)] = conj(scale z_k) (j = (5^k - 1)/2,
//           j' = (2N - 5^k - 1)/2), then m_i = round(Re(zeta^-i IDFT(E)_i));
//   decode: z_k = DFT(m_i zeta^i)[j(k)] / scale.
// This is the only floating-point stage of the library (float64); the
// result is rounded to integers before any modular arithmetic.
//
// The DFT is an iterative radix-2 transform of log2 N stages in two launches,
// 512 points per CTA in shared memory: the first reads its points in
// bit-reversed order straight from the slots (or coefficients) and runs the 8
// stages inside runs of 256, the second the rest over columns 256 apart, and
// writes the rounded coefficients (or slots).  One launch per stage was bound
// by launches: 17 of them, 85 us at N = 2^16 (one encode and one decode with
// their copies and transforms, 24 primes: 386 us so, 197 us with two launches
// and k_lift_wrap).  The stages are the same operations on the same twiddles,
// so the results are the same bit for bit.
#include <math.h>

#include <vector>

#include "launch.cuh"
#include "modarith.cuh"

namespace catfhe {

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

constexpr uint32_t kFftLow = 8;     // stages of the first launch
constexpr uint32_t kFftPts = 512;   // points per CTA, two per thread

// One butterfly with twiddle w.
__device__ __forceinline__ void fft_bfly(double2 &x0, double2 &x1, double2 w) {
    const double2 a = x0, b = cmul(w, x1);
    x0 = make_double2(a.x + b.x, a.y + b.y);
    x1 = make_double2(a.x - b.x, a.y - b.y);
}

// Stages 0 .. 7 of bit-reversed points.  ENC: point j of the input is the slot
// named by slot[j] (its conjugate where the top bit is set) times scale; else
// coefficient j times twist[j].
template <bool ENC>
__global__ void __launch_bounds__(kFftPts / 2)
k_fft_low(const double2 *__restrict__ z, double scale, const uint32_t *__restrict__ slot,
          const int64_t *__restrict__ m, const double2 *__restrict__ twist,
          const double2 *__restrict__ tw, double2 *__restrict__ out, uint32_t log_n) {
    grid_dep_wait();
    __shared__ double2 x[kFftPts];
    const uint32_t t = threadIdx.x, i0 = blockIdx.x * kFftPts;
#pragma unroll
    for (uint32_t u = 0; u < 2; u++) {
        const uint32_t i = t + u * (kFftPts / 2), j = __brev(i0 + i) >> (32 - log_n);
        if (ENC) {
            const uint32_t k = slot[j];
            const double2 s = z[k & 0x7fffffffu];
            const double2 v = make_double2(scale * s.x, scale * s.y);
            x[i] = make_double2(v.x, k >> 31 ? -v.y : v.y);
        } else {
            const double v = double(m[j]);
            x[i] = make_double2(v * twist[j].x, v * twist[j].y);
        }
    }
#pragma unroll
    for (uint32_t h = 0; h < kFftLow; h++) {
        __syncthreads();
        const uint32_t half = 1u << h, pos = t & (half - 1), a = ((t >> h) << (h + 1)) + pos;
        fft_bfly(x[a], x[a + half], tw[pos << (log_n - 1 - h)]);
    }
    __syncthreads();
#pragma unroll
    for (uint32_t u = 0; u < 2; u++) out[i0 + t + u * (kFftPts / 2)] = x[t + u * (kFftPts / 2)];
}

// Stages 8 .. log_n - 1: a CTA holds 512 >> (log_n - 8) adjacent columns.
// ENC: m_i = Re(x_i conj(zeta^i)) / N, rounded half away from zero; else point
// j goes to its slot, times scale (the conjugates are dropped).
template <bool ENC>
__global__ void __launch_bounds__(kFftPts / 2)
k_fft_high(const double2 *__restrict__ in, const double2 *__restrict__ tw,
           const double2 *__restrict__ twist, double scale, int64_t *__restrict__ m,
           const uint32_t *__restrict__ slot, double2 *__restrict__ z, uint32_t log_n) {
    grid_dep_wait();
    __shared__ double2 x[kFftPts];
    const uint32_t t = threadIdx.x, lb = log_n - kFftLow, lc = 9 - lb;  // log rows, log columns
    const uint32_t c0 = blockIdx.x << lc, cm = (1u << lc) - 1;
    // x[r << lc | c] is point (r << 8) + c0 + c
#pragma unroll
    for (uint32_t u = 0; u < 2; u++) {
        const uint32_t i = t + u * (kFftPts / 2);
        x[i] = in[((i >> lc) << kFftLow) + c0 + (i & cm)];
    }
    for (uint32_t h = 0; h < lb; h++) {
        __syncthreads();
        const uint32_t c = t & cm, r = t >> lc;  // column, butterfly of the column
        const uint32_t half = 1u << h, pr = r & (half - 1);
        const uint32_t a = ((((r >> h) << (h + 1)) + pr) << lc) | c;
        fft_bfly(x[a], x[a + (half << lc)],
                 tw[((pr << kFftLow) + c0 + c) << (lb - 1 - h)]);
    }
    __syncthreads();
#pragma unroll
    for (uint32_t u = 0; u < 2; u++) {
        const uint32_t i = t + u * (kFftPts / 2), j = ((i >> lc) << kFftLow) + c0 + (i & cm);
        if (ENC) {
            const double v = (x[i].x * twist[j].x + x[i].y * twist[j].y) * scale;
            m[j] = (int64_t)round(v);
        } else {
            const uint32_t k = slot[j];
            if (!(k >> 31)) z[k] = make_double2(x[i].x * scale, x[i].y * scale);
        }
    }
}

}  // namespace

// Tables: d_enc = [twist zeta^i (N)][omega^k (N/2)][omega^-k (N/2)],
// d_slot[j] = the slot k whose point j(k) is, or k | 2^31 where j is j'(k).
// Threads may make their first calls on one context at the same time.
int enc_tables(Context &c) {
    std::lock_guard<std::mutex> lock(c.mu);
    if (c.d_enc) return CATFHE_OK;
    const size_t n = c.n, half = n / 2;
    std::vector<double2> h(2 * n);
    const double pi = 3.14159265358979323846;
    for (size_t i = 0; i < n; i++) h[i] = make_double2(cos(pi * double(i) / double(n)), sin(pi * double(i) / double(n)));
    for (size_t k = 0; k < half; k++) {
        const double a = 2 * pi * double(k) / double(n);
        h[n + k] = make_double2(cos(a), sin(a));
        h[n + half + k] = make_double2(cos(a), -sin(a));
    }
    std::vector<uint32_t> idx(n);
    uint64_t e = 1;
    for (size_t k = 0; k < half; k++) {
        idx[(e - 1) / 2] = uint32_t(k);
        idx[(2 * n - e - 1) / 2] = uint32_t(k) | 0x80000000u;
        e = e * 5 % (2 * n);
    }
    double2 *d = nullptr;
    uint32_t *di = nullptr;
    if (cudaMalloc(&d, h.size() * sizeof(double2)) != cudaSuccess) return CATFHE_ENOMEM;
    if (cudaMalloc(&di, idx.size() * 4) != cudaSuccess) {
        cudaFree(d);
        return CATFHE_ENOMEM;
    }
    if (copy_in(d, h.data(), h.size() * sizeof(double2)) != cudaSuccess ||
        copy_in(di, idx.data(), idx.size() * 4) != cudaSuccess) {
        cudaFree(d);
        cudaFree(di);
        return CATFHE_ECUDA;
    }
    c.d_enc = d;
    c.d_slot = di;
    return CATFHE_OK;
}

int launch_encode_ckks(const Context &c, const double2 *slots, double scale, double2 *buf,
                       int64_t *m, cudaStream_t s) {
    const size_t n = c.n;
    const uint32_t lg = uint32_t(c.log_n), ctas = uint32_t(n / kFftPts);
    const double2 *twist = c.d_enc, *tw = c.d_enc + n + n / 2;
    launch_pdl(k_fft_low<true>, dim3(ctas), dim3(kFftPts / 2), 0, s, slots, scale, c.d_slot, m,
               twist, tw, buf, lg);
    launch_pdl(k_fft_high<true>, dim3(ctas), dim3(kFftPts / 2), 0, s, buf, tw, twist,
               1.0 / double(n), m, c.d_slot, buf, lg);
    note_launches(2);
    return cudaGetLastError() == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

int launch_decode_ckks(const Context &c, const int64_t *m, double inv_scale, double2 *buf,
                       double2 *slots, cudaStream_t s) {
    const size_t n = c.n;
    const uint32_t lg = uint32_t(c.log_n), ctas = uint32_t(n / kFftPts);
    const double2 *twist = c.d_enc, *tw = c.d_enc + n;
    launch_pdl(k_fft_low<false>, dim3(ctas), dim3(kFftPts / 2), 0, s, buf, 0.0, c.d_slot, m, twist,
               tw, buf, lg);
    launch_pdl(k_fft_high<false>, dim3(ctas), dim3(kFftPts / 2), 0, s, buf, tw, twist, inv_scale,
               (int64_t *)nullptr, c.d_slot, slots, lg);
    note_launches(2);
    return cudaGetLastError() == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

}  // namespace catfhe
