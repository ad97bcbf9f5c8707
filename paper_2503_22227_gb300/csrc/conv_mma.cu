// Exact, centred RNS base conversion with the sums over the sources on the
// tensor cores (the constants and the identity are stated in mmaplan.cpp).
//
// A CTA takes tiles of 256 coefficients, one per thread (two sets of 128 rows
// that share the plan's matrix).  A thread forms its
// coefficient's y_i (one Shoup product per source) and v, and writes the
// bytes of every y_i, less 128, as one 16-byte row of fp16 into the A
// operand; one elected thread issues the products with the plan's matrix
// (tcgen05, 2 x 128 x 128 accumulators in TMEM); then every thread reads its row
// back and turns the five or six sums of each target into a residue with four
// widening multiply-adds, three of them by constants.
//
// Why: the sums over the sources are the one dense contraction of the path.
// On the integer pipe a target costs three widening multiply-adds per source
// and a 64-bit Montgomery reduction (120 pipe cycles per warp at 8 sources),
// here 18 and no more per source.  Measured for half a batch of 8 at
// N = 2^16, l = 24 (ncu): ModUp (8 sources, 20 targets, three digits) 103 ->
// 59 us, the fused ModDown and rescale (5 sources, 23 targets) 57 -> 37 us;
// the step 1232 -> 1106 us.  What bounds it now is latency: 16 warps per SM
// issue on half of the cycles, in turns of digits, products and sums.  More
// CTAs per SM make it faster by itself (4 of 128 threads: 55 us) but leave no
// registers and shared memory to the other half's kernels, which run beside
// it (step 1196 us), so it takes 80 registers and two CTAs of 256 threads.
//
// v = floor(sum y_i / m_i + 1/2) comes from 27-bit fixed-point terms, each
// short by less than 3 units (y_i < 2 m_i: 15 terms stay below 2^32); when the
// sum is so close to a boundary that this matters (once in 5 * 10^6
// coefficients), the thread compares the exact mixed-radix digits with those
// of (M-1)/2.
//
// The next tile's sources come in by bulk copies while the products and the
// results of this one run.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "bulk.cuh"
#include "launch.cuh"
#include "modarith.cuh"
#include "tcgen05.cuh"

namespace catfhe {

namespace {

constexpr uint32_t kMmaTile = 256;      // coefficients per tile, threads per CTA
constexpr uint32_t kMmaPassBlocks = 8;  // column blocks per pass: 128 TMEM columns
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kFrac = 27;          // fraction bits of sum y_i / m_i

// Whether the value with residues r_i pre_i is above (M-1)/2, from its exact
// mixed-radix digits; `plan` in the Montgomery layout (global memory).  Rare.
__device__ __noinline__ bool above_half(const uint64_t *plan, const uint64_t *s, size_t n) {
    const uint32_t k = uint32_t(plan[0] & 0xffff), T = uint32_t((plan[0] >> 16) & 0xffff);
    const uint64_t *off = plan + 1, *smod = off + k + T, *C = smod + 2 * k + 2 * T, *h = C + k * k;
    uint64_t a[kMmaMaxK];
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

// The targets of one column block.  CHECK: fewer than a full block's.
template <bool LAZY, int D, bool CHECK>
__device__ __forceinline__ void block_out(const uint32_t (&v)[16], const uint64_t *tgt, uint32_t cnt,
                                          uint64_t *d) {
#pragma unroll
    for (int j = 0; j < int(kMmaBlock) / D; j++) {
        if (CHECK && uint32_t(j) >= cnt) break;  // the same for every thread
        const uint64_t *o = tgt + j * kMmaTgtWords;
        const ulonglong2 k0 = *reinterpret_cast<const ulonglong2 *>(o);
        const float4 f = *reinterpret_cast<const float4 *>(o + 2);
        uint64_t r = from_sums<D>(&v[j * D], k0, f);
        if (!LAZY) r = csub(r, 0 - k0.y);
        d[o[4]] = r;
    }
}

// LAZY: outputs in [0, 2p) instead of [0, p).
template <bool LAZY>
__global__ void __launch_bounds__(kMmaTile, 3)
k_conv_mma(const MmaList plans, const uint64_t *__restrict__ src, size_t src_item, size_t src_plan,
           uint64_t *__restrict__ dst, size_t dst_item, size_t dst_plan, uint32_t log_n,
           uint32_t tiles, int *status) {
    extern __shared__ __align__(128) uint64_t sm[];
    __shared__ __align__(8) uint64_t bars[3];  // plan image, products, sources
    __shared__ uint32_t tmem_slot;
    const uint32_t tid = threadIdx.x, z = blockIdx.z;
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_init(&bars[2], 1);
        mbar_init_fence();
    }
    if (tid < 32) tmem_alloc(&tmem_slot, kTmemCols);
    tcgen05_before_sync();
    __syncthreads();
    tcgen05_after_sync();
    const uint64_t head = plans.head[z], counts = plans.counts[z];
    const uint32_t K = uint32_t(head) & 0xff, nblk = uint32_t(head >> 8) & 0xff;
    const MmaLayout lay = mma_layout(K, nblk);
    const uint32_t cores = lay.cores, N = kMmaBlock * nblk;
    const uint32_t six = uint32_t(head >> 32);
    if (tid == 0) {
        mbar_expect_tx(&bars[0], lay.words * 8);
        bulk_load(sm, plans.img[z], lay.words * 8, &bars[0]);
    }
    grid_dep_wait();  // everything above reads only the plan
    // every wait is bounded; the CTA decides together whether to go on, so no
    // thread is left waiting at a barrier
    bool run = __syncthreads_and(mbar_wait(&bars[0], 0)), ok = run;
    const uint32_t tmem = tmem_slot;
    const uint64_t *Bm = sm + lay.b;
    uint4 *A = reinterpret_cast<uint4 *>(sm + lay.words);  // [core][256 rows]
    if ((K & 1) == 0) A[(K + 1) * kMmaTile + tid] = make_uint4(0, 0, 0, 0);  // padding core
    uint64_t *S = sm + lay.words + cores * kMmaTile * 2;  // [K][256] sources
    const size_t n = size_t(1) << log_n;
    const uint32_t lg_tpi = log_n - 8;  // tiles per item
    auto tile_src = [&](uint32_t tile) {
        return src + (tile >> lg_tpi) * src_item + z * src_plan +
               size_t(tile & ((1u << lg_tpi) - 1)) * kMmaTile;
    };
    auto fetch = [&](uint32_t tile) {  // by thread 0
        mbar_expect_tx(&bars[2], K * kMmaTile * 8);
        const uint64_t *s = tile_src(tile);
        for (uint32_t i = 0; i < K; i++)
            bulk_load(S + i * kMmaTile, s + sm[lay.src + i * kMmaSrcWords + 4], kMmaTile * 8,
                      &bars[2]);
    };
    if (run && tid == 0) fetch(blockIdx.x);  // the grid has no more CTAs than tiles
    uint32_t phase = 0, sphase = 0;
    for (uint32_t tile = blockIdx.x; tile < tiles && run; tile += gridDim.x) {
        ok = ok && mbar_wait(&bars[2], sphase);
        sphase ^= 1;
        if (ok) {
            uint32_t fr = 1u << (kFrac - 1);
            // sources in fours: all loads, then four independent chains, then
            // the stores (which the compiler cannot tell from the loads)
            auto digits = [&](uint32_t i, auto count) {
                constexpr int C = decltype(count)::value;
                uint64_t y[C];
                ulonglong2 mw[C], sc[C];
#pragma unroll
                for (int j = 0; j < C; j++) {
                    const uint64_t *o = sm + lay.src + (i + j) * kMmaSrcWords;
                    mw[j] = *reinterpret_cast<const ulonglong2 *>(o);
                    sc[j] = *reinterpret_cast<const ulonglong2 *>(o + 2);
                    y[j] = S[(i + j) * kMmaTile + tid];
                }
#pragma unroll
                for (int j = 0; j < C; j++) {
                    y[j] = shoup_lazy(y[j], mw[j].y, sc[j].x, mw[j].x);  // [0, 2m)
                    fr += __umulhi(uint32_t(y[j] >> uint32_t(sc[j].y >> 32)), uint32_t(sc[j].y));
                }
#pragma unroll
                for (int j = 0; j < C; j++) {
                    const uint32_t lo = uint32_t(y[j]), hi = uint32_t(y[j] >> 32);
                    A[(i + j) * kMmaTile + tid] = make_uint4(two_bytes<0>(lo), two_bytes<2>(lo),
                                                             two_bytes<0>(hi), two_bytes<2>(hi));
                }
            };
            uint32_t i = 0;
            for (; i + 4 <= K; i += 4) digits(i, std::integral_constant<int, 4>{});
#pragma unroll 1
            for (; i < K; i++) digits(i, std::integral_constant<int, 1>{});
            uint32_t v = fr >> kFrac;
            if ((fr & ((1u << kFrac) - 1)) >= (1u << kFrac) - 3 * K)
                v = ((fr - (1u << (kFrac - 1))) >> kFrac) + (above_half(plans.p[z], tile_src(tile) + tid, n) ? 1 : 0);
            // v, and 3072 (times 4096 in the matrix: the sums' float offset)
            A[K * kMmaTile + tid] =
                make_uint4(uint32_t(__half_as_ushort(__uint2half_rn(v))) | 0x6A000000u, 0, 0, 0);
            fence_proxy_async();
        }
        for (uint32_t b0 = 0; b0 < nblk; b0 += kMmaPassBlocks) {
            tcgen05_before_sync();
            run = __syncthreads_and(ok);
            if (!run) break;
            const uint32_t nb = nblk - b0 < kMmaPassBlocks ? nblk - b0 : kMmaPassBlocks;
            if (tid == 0) {
                tcgen05_after_sync();
                if (b0 == 0 && tile + gridDim.x < tiles) {
                    fence_proxy_async();
                    fetch(tile + gridDim.x);
                }
                for (uint32_t h = 0; h < 2; h++)
                    for (uint32_t kc = 0; kc < cores; kc += 2)
                        mma_f16(tmem + 128 * h,
                                mma_desc(A + kc * kMmaTile + 128 * h, kMmaTile * 16, 128),
                                mma_desc(Bm + (size_t(kc) * N + kMmaBlock * b0) * 2, N * 16, 128),
                                mma_idesc(kMmaBlock * nb), kc != 0);
                mma_commit(&bars[1]);
            }
            ok = mbar_wait(&bars[1], phase);
            phase ^= 1;
            tcgen05_after_sync();
            const uint32_t item = tile >> lg_tpi;
            uint64_t *d = dst + item * dst_item + z * dst_plan +
                          size_t(tile & ((1u << lg_tpi) - 1)) * kMmaTile + tid;
            __syncwarp();
            const uint32_t rows = tmem + ((tid & 96u) << 16) + (tid >> 7) * 128;
            auto out = [&](uint32_t b, const uint32_t (&v)[16]) {
                const uint64_t *tgt = sm + lay.tgt + size_t(b) * kMmaSlots * kMmaTgtWords;
                const uint32_t cnt = uint32_t(counts >> (4 * b)) & 0xf;
                if ((six >> b) & 1)
                    cnt == 2 ? block_out<LAZY, 6, false>(v, tgt, cnt, d)
                             : block_out<LAZY, 6, true>(v, tgt, cnt, d);
                else
                    cnt == 3 ? block_out<LAZY, 5, false>(v, tgt, cnt, d)
                             : block_out<LAZY, 5, true>(v, tgt, cnt, d);
            };
            // one block's results are formed while the next one is read
            uint32_t va[16], vb[16];
            tmem_load16(rows, va);
            for (uint32_t b = 0; b < nb; b += 2) {
                tmem_wait16(va);
                if (b + 1 < nb) tmem_load16(rows + (b + 1) * kMmaBlock, vb);
                out(b0 + b, va);
                if (b + 1 < nb) {
                    tmem_wait16(vb);
                    if (b + 2 < nb) tmem_load16(rows + (b + 2) * kMmaBlock, va);
                    out(b0 + b + 1, vb);
                }
            }
        }
    }
    if (!__syncthreads_and(ok) && tid == 0) {
        atomicOr(status, kStatusConvWait);
        // a bounded time for copies and products in flight
        mbar_wait(&bars[2], sphase);
        mbar_wait(&bars[1], phase ^ 1);
    }
    __syncthreads();
    if (tid < 32) tmem_free(tmem, kTmemCols);
}

}  // namespace

int launch_conv_mma(const Context &c, const MmaList &plans, const uint64_t *src, size_t src_item,
                    size_t src_plan, uint64_t *dst, size_t dst_item, size_t dst_plan,
                    uint32_t items, cudaStream_t s) {
    uint32_t smem = 0;
    bool lazy = true;
    for (uint32_t i = 0; i < plans.n; i++) {
        const uint32_t K = uint32_t(plans.head[i]) & 0xff;
        const MmaLayout lay = mma_layout(K, uint32_t(plans.head[i] >> 8) & 0xff);
        smem = std::max(smem, lay.words * 8 + lay.cores * kMmaTile * 16 + K * kMmaTile * 8);
        lazy = lazy && ((plans.head[i] >> 24) & 1);
    }
    const auto kernel = lazy ? k_conv_mma<true> : k_conv_mma<false>;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) !=
        cudaSuccess)
        return CATFHE_ECUDA;
    // every CTA loads its plan once and takes as many tiles as fill the chip
    // once: up to 2 CTAs per SM (their TMEM columns are the SM's 512; the
    // occupancy API answers 1 for a kernel that allocates TMEM)
    const uint32_t tiles = uint32_t(items * (c.n / kMmaTile));
    const uint32_t per_sm = std::min<uint32_t>(2, 227 * 1024 / (smem + 2048));
    const uint32_t slots = uint32_t(c.sms) * std::max<uint32_t>(1, per_sm);
    const uint32_t per_plan = std::max<uint32_t>(1, slots / plans.n);
    const uint32_t each = (tiles + per_plan - 1) / per_plan;
    const dim3 grid((tiles + each - 1) / each, 1, plans.n);
    launch_pdl(kernel, grid, dim3(kMmaTile), smem, s, plans, src, src_item, src_plan, dst,
               dst_item, dst_plan, uint32_t(c.log_n), tiles, c.d_status);
    note_launches(1);
    return cudaGetLastError() == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

}  // namespace catfhe
