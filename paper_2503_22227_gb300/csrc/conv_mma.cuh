// Pieces of the tensor-core base conversion shared by its kernels (conv_mma.cu
// states the method; mmaplan.cpp the constants).
#pragma once

#include <cuda_fp16.h>

#include <type_traits>

#include "bulk.cuh"
#include "modarith.cuh"
#include "tcgen05.cuh"

namespace catfhe {

constexpr uint32_t kMmaTile = 256;      // coefficients per tile, threads per CTA
constexpr uint32_t kMmaPassBlocks = 8;  // column blocks per pass: 128 TMEM columns
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kFrac = 27;          // fraction bits of sum y_i / m_i

// Whether the value with residues r_i pre_i is above (M-1)/2, from its exact
// mixed-radix digits; `plan` in the Montgomery layout (global memory).  Rare.
static __device__ __noinline__ bool above_half(const uint64_t *plan, const uint64_t *s, size_t n) {
    const uint32_t k = uint32_t(plan[0] & 0xffff), T = uint32_t((plan[0] >> 16) & 0xffff);
    const uint64_t *off = plan + 1, *smod = off + k + T, *C = smod + 2 * k + 2 * T, *h = C + k * k;
    uint64_t a[kConvMaxK];
    bool gt = false;
    for (uint32_t j = 0; j < k; j++) {
        const uint64_t mj = smod[2 * j];
        U128 acc{0, 0};
        mac(acc, s[off[j] * n], C[j * k + j]);
        for (uint32_t i = 0; i < j; i++) mac(acc, a[i], C[i * k + j]);
        a[j] = csub(redc(acc, mj, smod[2 * j + 1]), mj);
        if (a[j] != h[j]) gt = a[j] > h[j];
    }
    return gt;
}

// Bytes b and b + 1 of a word (b = 0 or 2) as two fp16 values less 128:
// 0x6400 | byte is 1024 + byte.
template <int B>
__device__ __forceinline__ uint32_t two_bytes(uint32_t w) {
    uint32_t h, r;
    asm("prmt.b32 %0, %1, 0x64646464, %2;" : "=r"(h) : "r"(w), "n"(B ? 0x4342 : 0x4140));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0xE480E480u));  // -1152 each
    return r;
}

__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
    uint64_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}

// One target's residue from its D column sums (floats 3 * 2^22 + S_d).
template <int D>
__device__ __forceinline__ uint64_t from_sums(const uint32_t *b, const ulonglong2 k0,
                                              const float4 f) {
    const float big = 12582912.f;
    const float q = fmaf(__uint_as_float(b[D - 1]) - big, f.x,
                         fmaf(__uint_as_float(b[D - 2]), f.y, fmaf(__uint_as_float(b[D - 3]), f.z, f.w)));
    const uint32_t e = __float_as_uint(q + big);
    uint64_t r = mad_wide(b[1], 1u << 10, k0.x + b[0]);
    r = mad_wide(b[2], 1u << 20, r);
    r = mad_wide(b[3], 1u << 30, r);
    r = mad_wide(e, uint32_t(k0.y), r);
    uint32_t hi = uint32_t(r >> 32) + (b[4] << 8) + e * uint32_t(k0.y >> 32);
    if (D == 6) hi += b[D - 1] << 18;
    return uint64_t(uint32_t(r)) | uint64_t(hi) << 32;
}

// What a kernel knows of its plan from the header words.
struct MmaShape {
    uint32_t K, nblk, N, six;
    uint64_t counts;
    MmaLayout lay;
    __device__ __forceinline__ MmaShape(uint64_t head, uint64_t counts_)
        : K(uint32_t(head) & 0xff), nblk(uint32_t(head >> 8) & 0xff), N(kMmaBlock * nblk),
          six(uint32_t(head >> 32)), counts(counts_), lay(mma_layout(K, nblk)) {}
    __device__ __forceinline__ uint32_t targets(uint32_t b) const {
        return uint32_t(counts >> (4 * b)) & 0xf;
    }
};

// y's bytes as a row of the A operand.
__device__ __forceinline__ uint4 digit_row(uint64_t y) {
    const uint32_t lo = uint32_t(y), hi = uint32_t(y >> 32);
    return make_uint4(two_bytes<0>(lo), two_bytes<2>(lo), two_bytes<0>(hi), two_bytes<2>(hi));
}

// y / m in units of 2^-kFrac, short by less than 3; sc as in the source record.
__device__ __forceinline__ uint32_t digit_frac(uint64_t y, uint64_t sc) {
    return __umulhi(uint32_t(y >> uint32_t(sc >> 32)), uint32_t(sc));
}

// The core of v and the constant row: v, and 3072 (times 4096 in the matrix:
// the sums' float offset).
__device__ __forceinline__ uint4 quotient_row(uint32_t v) {
    return make_uint4(uint32_t(__half_as_ushort(__uint2half_rn(v))) | 0x6A000000u, 0, 0, 0);
}

// Whether sum y_i / m_i + 1/2, known as fr, is too close to a whole number.
__device__ __forceinline__ bool undecided(uint32_t fr, uint32_t K) {
    return (fr & ((1u << kFrac) - 1)) >= (1u << kFrac) - 3 * K;
}
// v once it is known whether the value is above (M-1)/2.
__device__ __forceinline__ uint32_t decided(uint32_t fr, bool above) {
    return ((fr - (1u << (kFrac - 1))) >> kFrac) + (above ? 1 : 0);
}

// This thread's rows of A from its sources S ([K][256]); returns the sum of
// y_i / m_i + 1/2.  In fours: all loads, then four independent chains, then
// the stores (which the compiler cannot tell from the loads).
__device__ __forceinline__ uint32_t write_digits(const uint64_t *recs, const uint64_t *S, uint4 *A,
                                                 uint32_t K, uint32_t tid) {
    uint32_t fr = 1u << (kFrac - 1);
    auto digits = [&](uint32_t i, auto count) {
        constexpr int C = decltype(count)::value;
        uint64_t y[C];
        ulonglong2 mw[C], sc[C];
#pragma unroll
        for (int j = 0; j < C; j++) {
            const uint64_t *o = recs + (i + j) * kMmaSrcWords;
            mw[j] = *reinterpret_cast<const ulonglong2 *>(o);
            sc[j] = *reinterpret_cast<const ulonglong2 *>(o + 2);
            y[j] = S[(i + j) * kMmaTile + tid];
        }
#pragma unroll
        for (int j = 0; j < C; j++) {
            y[j] = shoup_lazy(y[j], mw[j].y, sc[j].x, mw[j].x);  // [0, 2m)
            fr += digit_frac(y[j], sc[j].y);
        }
#pragma unroll
        for (int j = 0; j < C; j++) A[(i + j) * kMmaTile + tid] = digit_row(y[j]);
    };
    uint32_t i = 0;
    for (; i + 4 <= K; i += 4) digits(i, std::integral_constant<int, 4>{});
#pragma unroll 1
    for (; i < K; i++) digits(i, std::integral_constant<int, 1>{});
    return fr;
}

// The products of both sets of 128 rows with nb column blocks from b0 on;
// issued by one thread, one arrival on bar when they have completed.
__device__ __forceinline__ void issue_products(uint32_t tmem, const uint4 *A, const uint64_t *B,
                                               const MmaShape &p, uint32_t b0, uint32_t nb,
                                               uint64_t *bar) {
    for (uint32_t h = 0; h < 2; h++)
        for (uint32_t kc = 0; kc < p.lay.cores; kc += 2)
            mma_f16(tmem + 128 * h, mma_desc(A + kc * kMmaTile + 128 * h, kMmaTile * 16, 128),
                    mma_desc(B + (size_t(kc) * p.N + kMmaBlock * b0) * 2, p.N * 16, 128),
                    mma_idesc(kMmaBlock * nb), kc != 0);
    mma_commit(bar);
}

// Calls out(b, sums) for nb column blocks; one block's results are formed
// while the next one is read.
template <class F>
__device__ __forceinline__ void each_block(uint32_t tmem, uint32_t tid, uint32_t nb, F out) {
    const uint32_t rows = tmem + ((tid & 96u) << 16) + (tid >> 7) * 128;
    uint32_t va[16], vb[16];
    tmem_load16(rows, va);
    for (uint32_t b = 0; b < nb; b += 2) {
        tmem_wait16(va);
        if (b + 1 < nb) tmem_load16(rows + (b + 1) * kMmaBlock, vb);
        out(b, va);
        if (b + 1 < nb) {
            tmem_wait16(vb);
            if (b + 2 < nb) tmem_load16(rows + (b + 2) * kMmaBlock, va);
            out(b + 1, vb);
        }
    }
}

// Calls f(slot record, residue in (0.4 p, 1.6 p)) for the targets of a block.
template <int D, bool CHECK, class F>
__device__ __forceinline__ void block_targets(const uint32_t (&v)[16], const uint64_t *tgt,
                                              uint32_t cnt, F f) {
#pragma unroll
    for (int j = 0; j < int(kMmaBlock) / D; j++) {
        if (CHECK && uint32_t(j) >= cnt) break;  // the same for every thread
        const uint64_t *o = tgt + j * kMmaTgtWords;
        const ulonglong2 k0 = *reinterpret_cast<const ulonglong2 *>(o);
        const float4 w = *reinterpret_cast<const float4 *>(o + 2);
        f(o, 0 - k0.y, from_sums<D>(&v[j * D], k0, w));
    }
}
template <class F>
__device__ __forceinline__ void block_results(const uint32_t (&v)[16], const uint64_t *sm,
                                              const MmaShape &p, uint32_t b, F f) {
    const uint64_t *tgt = sm + p.lay.tgt + size_t(b) * kMmaSlots * kMmaTgtWords;
    const uint32_t cnt = p.targets(b);
    if ((p.six >> b) & 1)
        cnt == 2 ? block_targets<6, false>(v, tgt, cnt, f) : block_targets<6, true>(v, tgt, cnt, f);
    else
        cnt == 3 ? block_targets<5, false>(v, tgt, cnt, f) : block_targets<5, true>(v, tgt, cnt, f);
}

}  // namespace catfhe
