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
#include <algorithm>

#include "conv_mma.cuh"
#include "launch.cuh"

namespace catfhe {

namespace {

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
    const MmaShape p(plans.head[z], plans.counts[z]);
    const uint32_t K = p.K;
    if (tid == 0) {
        mbar_expect_tx(&bars[0], p.lay.words * 8);
        bulk_load(sm, plans.img[z], p.lay.words * 8, &bars[0]);
    }
    grid_dep_wait();  // everything above reads only the plan
    // every wait is bounded; the CTA decides together whether to go on, so no
    // thread is left waiting at a barrier
    bool run = __syncthreads_and(mbar_wait(&bars[0], 0)), ok = run;
    const uint32_t tmem = tmem_slot;
    uint4 *A = reinterpret_cast<uint4 *>(sm + p.lay.words);  // [core][256 rows]
    if ((K & 1) == 0) A[(K + 1) * kMmaTile + tid] = make_uint4(0, 0, 0, 0);  // padding core
    uint64_t *S = sm + p.lay.words + p.lay.cores * kMmaTile * 2;  // [K][256] sources
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
            bulk_load(S + i * kMmaTile, s + sm[p.lay.src + i * kMmaSrcWords + 4], kMmaTile * 8,
                      &bars[2]);
    };
    if (run && tid == 0) fetch(blockIdx.x);  // the grid has no more CTAs than tiles
    uint32_t phase = 0, sphase = 0;
    for (uint32_t tile = blockIdx.x; tile < tiles && run; tile += gridDim.x) {
        ok = ok && mbar_wait(&bars[2], sphase);
        sphase ^= 1;
        if (ok) {
            const uint32_t fr = write_digits(sm + p.lay.src, S, A, K, tid);
            uint32_t v = fr >> kFrac;
            if (undecided(fr, K)) v = decided(fr, above_half(plans.p[z], tile_src(tile) + tid, n));
            A[K * kMmaTile + tid] = quotient_row(v);
            fence_proxy_async();
        }
        for (uint32_t b0 = 0; b0 < p.nblk; b0 += kMmaPassBlocks) {
            tcgen05_before_sync();
            run = __syncthreads_and(ok);
            if (!run) break;
            const uint32_t nb = p.nblk - b0 < kMmaPassBlocks ? p.nblk - b0 : kMmaPassBlocks;
            if (tid == 0) {
                tcgen05_after_sync();
                if (b0 == 0 && tile + gridDim.x < tiles) {
                    fence_proxy_async();
                    fetch(tile + gridDim.x);
                }
                issue_products(tmem, A, sm + p.lay.b, p, b0, nb, &bars[1]);
            }
            ok = mbar_wait(&bars[1], phase);
            phase ^= 1;
            tcgen05_after_sync();
            uint64_t *d = dst + (tile >> lg_tpi) * dst_item + z * dst_plan +
                          size_t(tile & ((1u << lg_tpi) - 1)) * kMmaTile + tid;
            __syncwarp();
            each_block(tmem, tid, nb, [&](uint32_t b, const uint32_t (&v)[16]) {
                block_results(v, sm, p, b0 + b, [&](const uint64_t *o, uint64_t q, uint64_t r) {
                    d[o[4]] = LAZY ? r : csub(r, q);
                });
            });
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

// BFV scale-and-round (internal.h, launch_bfv_round_mma): two conversions per
// coefficient without the values between them leaving the SM.  Plan a lifts
// [t x]_Q to B, times Q^-1 (B/b_j)^-1; its result L_j and x_b give the digits
// of z = round(t x / Q) for plan b directly: y_j = t Q^-1 (B/b_j)^-1 x_b - L_j
// mod b_j.  Both use the same A rows and accumulators in turn.  Half a batch of
// 16 at N = 2^14 with 8 + 8 primes: 112 us on the integer pipe
// (k_bfv_scale_round, full 64-bit products), 45 us so; 122 registers, since two
// CTAs are all that TMEM holds.
__global__ void __launch_bounds__(kMmaTile, 2)
k_bfv_round_mma(const MmaList plans, const uint64_t *__restrict__ src, size_t src_item,
                uint64_t *__restrict__ dst, size_t dst_item, uint32_t log_n, uint32_t tiles,
                int *status) {
    extern __shared__ __align__(128) uint64_t sm[];
    __shared__ __align__(8) uint64_t bars[3];  // plan images, products, sources
    __shared__ uint32_t tmem_slot;
    const uint32_t tid = threadIdx.x;
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
    const MmaShape pa(plans.head[0], plans.counts[0]), pb(plans.head[1], plans.counts[1]);
    uint64_t *sb = sm + pa.lay.words;  // plan b's image
    if (tid == 0) {
        mbar_expect_tx(&bars[0], (pa.lay.words + pb.lay.words) * 8);
        bulk_load(sm, plans.img[0], pa.lay.words * 8, &bars[0]);
        bulk_load(sb, plans.img[1], pb.lay.words * 8, &bars[0]);
    }
    grid_dep_wait();
    bool run = __syncthreads_and(mbar_wait(&bars[0], 0)), ok = run;
    const uint32_t tmem = tmem_slot, Ka = pa.K, Kb = pb.K;
    const uint32_t cores = pa.lay.cores > pb.lay.cores ? pa.lay.cores : pb.lay.cores;
    uint4 *A = reinterpret_cast<uint4 *>(sb + pb.lay.words);
    // every row finite: a plan's padding core has weights 0, and may hold the
    // other plan's digits
    for (uint32_t k = 0; k < cores; k++) A[k * kMmaTile + tid] = make_uint4(0, 0, 0, 0);
    uint64_t *S = sb + pb.lay.words + cores * kMmaTile * 2;  // [Ka] q limbs, then [Kb] b limbs
    uint64_t *Sb = S + Ka * kMmaTile;
    const size_t n = size_t(1) << log_n;
    const uint32_t lg_tpi = log_n - 8;
    auto tile_src = [&](uint32_t tile) {
        return src + (tile >> lg_tpi) * src_item + size_t(tile & ((1u << lg_tpi) - 1)) * kMmaTile;
    };
    auto fetch = [&](uint32_t tile) {  // by thread 0
        mbar_expect_tx(&bars[2], (Ka + Kb) * kMmaTile * 8);
        const uint64_t *s = tile_src(tile);
        for (uint32_t i = 0; i < Ka; i++)
            bulk_load(S + i * kMmaTile, s + sm[pa.lay.src + i * kMmaSrcWords + 4], kMmaTile * 8,
                      &bars[2]);
        for (uint32_t j = 0; j < Kb; j++)
            bulk_load(Sb + j * kMmaTile, s + sb[pb.lay.src + j * kMmaSrcWords + 4], kMmaTile * 8,
                      &bars[2]);
    };
    if (run && tid == 0) fetch(blockIdx.x);
    uint32_t phase = 0, sphase = 0;
    for (uint32_t tile = blockIdx.x; tile < tiles && run; tile += gridDim.x) {
        ok = ok && mbar_wait(&bars[2], sphase);
        sphase ^= 1;
        if (ok) {
            const uint32_t fr = write_digits(sm + pa.lay.src, S, A, Ka, tid);
            uint32_t v = fr >> kFrac;
            if (undecided(fr, Ka)) v = decided(fr, above_half(plans.p[0], tile_src(tile) + tid, n));
            A[Ka * kMmaTile + tid] = quotient_row(v);
            fence_proxy_async();
        }
        tcgen05_before_sync();
        run = __syncthreads_and(ok);
        if (!run) break;
        if (tid == 0) {
            tcgen05_after_sync();
            issue_products(tmem, A, sm + pa.lay.b, pa, 0, pa.nblk, &bars[1]);
        }
        ok = mbar_wait(&bars[1], phase);
        phase ^= 1;
        tcgen05_after_sync();
        __syncwarp();
        uint32_t fr = 1u << (kFrac - 1);
        each_block(tmem, tid, pa.nblk, [&](uint32_t b, const uint32_t (&v)[16]) {
            block_results(v, sm, pa, b, [&](const uint64_t *o, uint64_t q, uint64_t r) {
                const uint32_t j = uint32_t(o[4]);
                const uint64_t *rec = sb + pb.lay.src + j * kMmaSrcWords;
                const ulonglong2 mw = *reinterpret_cast<const ulonglong2 *>(rec);
                const ulonglong2 sc = *reinterpret_cast<const ulonglong2 *>(rec + 2);
                const uint64_t xb = Sb[j * kMmaTile + tid];
                // [0, 2q) + 2q - (0.4 q, 1.6 q) < 4q, then below 2q
                const uint64_t y = csub(shoup_lazy(xb, mw.y, sc.x, q) + 2 * q - r, 2 * q);
                fr += digit_frac(y, sc.y);
                A[j * kMmaTile + tid] = digit_row(y);
                Sb[j * kMmaTile + tid] = y;  // for the exact comparison
            });
        });
        uint32_t v = fr >> kFrac;
        if (undecided(fr, Kb)) v = decided(fr, above_half(plans.p[1], Sb + tid, kMmaTile));
        A[Kb * kMmaTile + tid] = quotient_row(v);
        fence_proxy_async();
        tcgen05_before_sync();
        run = __syncthreads_and(ok);
        if (!run) break;
        if (tid == 0) {
            tcgen05_after_sync();
            if (tile + gridDim.x < tiles) {
                fence_proxy_async();
                fetch(tile + gridDim.x);
            }
            issue_products(tmem, A, sb + pb.lay.b, pb, 0, pb.nblk, &bars[1]);
        }
        ok = mbar_wait(&bars[1], phase);
        phase ^= 1;
        tcgen05_after_sync();
        uint64_t *d = dst + (tile >> lg_tpi) * dst_item +
                      size_t(tile & ((1u << lg_tpi) - 1)) * kMmaTile + tid;
        __syncwarp();
        each_block(tmem, tid, pb.nblk, [&](uint32_t b, const uint32_t (&v2)[16]) {
            block_results(v2, sb, pb, b, [&](const uint64_t *o, uint64_t q, uint64_t r) {
                d[o[4]] = csub(r, q);
            });
        });
    }
    if (!__syncthreads_and(ok) && tid == 0) {
        atomicOr(status, kStatusConvWait);
        mbar_wait(&bars[2], sphase);
        mbar_wait(&bars[1], phase ^ 1);
    }
    __syncthreads();
    if (tid < 32) tmem_free(tmem, kTmemCols);
}

// CTAs of a launch over `tiles` tiles: as many as fill the chip once, each
// loading its plans once, with the tiles spread evenly over them.  Up to 2 per
// SM (their TMEM columns are the SM's 512; the occupancy API answers 1 for a
// kernel that allocates TMEM), less where shared memory is short.
uint32_t mma_grid(const Context &c, uint32_t tiles, uint32_t smem, uint32_t plans) {
    const uint32_t per_sm = std::max<uint32_t>(1, std::min<uint32_t>(2, 227 * 1024 / (smem + 2048)));
    const uint32_t per_plan = std::max<uint32_t>(1, uint32_t(c.sms) * per_sm / plans);
    const uint32_t each = (tiles + per_plan - 1) / per_plan;
    return (tiles + each - 1) / each;
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
    if (!allow_smem(reinterpret_cast<const void *>(kernel), smem)) return CATFHE_ECUDA;
    const uint32_t tiles = uint32_t(items * (c.n / kMmaTile));
    const dim3 grid(mma_grid(c, tiles, smem, plans.n), 1, plans.n);
    launch_pdl_split(kSharedPercent, kernel, grid, dim3(kMmaTile), smem, s, plans, src, src_item, src_plan, dst,
               dst_item, dst_plan, uint32_t(c.log_n), tiles, c.d_status);
    note_mma_launch();
    return cudaGetLastError() == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

// Whether both conversions' images fit one pass of the accumulators and one
// CTA's shared memory; its size.
static uint32_t bfv_round_smem(const MmaRef &a, const MmaRef &b) {
    const uint32_t Ka = uint32_t(a.head) & 0xff, Kb = uint32_t(b.head) & 0xff;
    const uint32_t na = uint32_t(a.head >> 8) & 0xff, nb = uint32_t(b.head >> 8) & 0xff;
    const MmaLayout la = mma_layout(Ka, na), lb = mma_layout(Kb, nb);
    if (na > kMmaPassBlocks || nb > kMmaPassBlocks) return 0;
    const uint32_t bytes = (la.words + lb.words) * 8 +
                           std::max(la.cores, lb.cores) * kMmaTile * 16 + (Ka + Kb) * kMmaTile * 8;
    return bytes <= 220 * 1024 ? bytes : 0;
}

bool bfv_round_mma_fits(const MmaRef &a, const MmaRef &b) {
    return a.p && b.p && bfv_round_smem(a, b) != 0;
}

int launch_bfv_round_mma(const Context &c, const MmaRef &a, const uint64_t *a_exact,
                         const MmaRef &b, const uint64_t *b_exact, const uint64_t *src,
                         size_t src_item, uint64_t *dst, size_t dst_item, uint32_t items,
                         cudaStream_t s) {
    MmaList l{};
    l.n = 2;
    l.img[0] = a.p, l.head[0] = a.head, l.counts[0] = a.counts, l.p[0] = a_exact;
    l.img[1] = b.p, l.head[1] = b.head, l.counts[1] = b.counts, l.p[1] = b_exact;
    const uint32_t smem = bfv_round_smem(a, b);
    if (!allow_smem(reinterpret_cast<const void *>(k_bfv_round_mma), smem)) return CATFHE_ECUDA;
    const uint32_t tiles = uint32_t(items * (c.n / kMmaTile));
    launch_pdl_split(kSharedPercent, k_bfv_round_mma, dim3(mma_grid(c, tiles, smem, 1)), dim3(kMmaTile), smem, s, l, src,
               src_item, dst, dst_item, uint32_t(c.log_n), tiles, c.d_status);
    note_mma_launch();
    return cudaGetLastError() == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

}  // namespace catfhe
