// Element-wise kernels of the hot path: the fused tensor product (paper
// Sec. 3.1.4: the four products and the middle sum of a CKKS multiply in one
// kernel), the key-switching inner product, the ModDown combine, the
// automorphism X -> X^g, and ChaCha20 sampling for keys and encryption.
//
// All are HBM-bound streams over limb-major data: a thread takes one or two
// 16-byte pairs of coefficients (sampling and the automorphism one coefficient),
// consecutive threads consecutive words, grids sized by the data (a whole batch
// of ciphertexts per launch).
#include <cmath>
#include "bulk.cuh"
#include "launch.cuh"
#include "modarith.cuh"

namespace catfhe {

static inline int ok() {
    note_launches(1);
    return cudaGetLastError() == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

static inline dim3 coeff_grid(size_t n, uint32_t y, uint32_t z = 1) {
    return dim3(unsigned((n + 255) / 256), y, z);
}

// ------------------------------------------------------------------ tensor

__device__ __forceinline__ ulonglong2 ld2(const uint64_t *p) {
    return *reinterpret_cast<const ulonglong2 *>(p);
}
__device__ __forceinline__ void st2(uint64_t *p, uint64_t a, uint64_t b) {
    *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(a, b);
}

// Two adjacent coefficients per thread (16-byte loads and stores).
__global__ void __launch_bounds__(256)
k_tensor(const TensorArgs A, const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const size_t n = size_t(1) << log_n;
    const size_t x = 2 * (size_t(blockIdx.x) * blockDim.x + threadIdx.x);
    const uint32_t i = blockIdx.y, item = blockIdx.z;
    if (x >= n) return;
    const DevMod m = mods[A.prime[i]];
    const uint64_t *a = A.gathered ? A.ga[item] : A.a + item * A.in_item;
    const uint64_t *b = A.gathered ? A.gb[item] : A.b + item * A.in_item;
    const size_t l0 = size_t(i) * n + x, l1 = (size_t(A.limbs) + i) * n + x;
    const ulonglong2 a0 = ld2(a + l0), a1 = ld2(a + l1), b0 = ld2(b + l0), b1 = ld2(b + l1);
    const size_t o = item * A.out_item + size_t(i) * n + x;
    const Tensor u = tensor_mod(a0.x, a1.x, b0.x, b1.x, m);
    const Tensor v = tensor_mod(a0.y, a1.y, b0.y, b1.y, m);
    st2(A.d0 + o, u.d0, v.d0);
    st2(A.d1 + o, u.d1, v.d1);
    st2(A.d2 + o, u.d2, v.d2);
}

int launch_tensor(const Context &c, const TensorArgs &a, uint32_t count, cudaStream_t s) {
    launch_pdl_split(kSharedPercent, k_tensor, coeff_grid(c.n / 2, a.limbs, count), dim3(256), 0, s, a, c.d_mods, c.log_n);
    return ok();
}

// ------------------------------------------------------------------ key-switch inner product

// y_p[i] = sum_j c_j[i] * key_j[p][i] (+ P * add_p[i] on ciphertext primes).

// The first limb of an item's own digits and of its addends.
template <bool GATHER>
__device__ __forceinline__ const uint64_t *ip_own(const IpArgs &A, uint32_t item, size_t n) {
    return GATHER ? A.ga[item] + size_t(A.level) * n : A.own + item * A.own_item;
}
template <bool GATHER>
__device__ __forceinline__ const uint64_t *ip_add0(const IpArgs &A, uint32_t item) {
    return GATHER ? A.ga[item] : A.add0 + item * A.add_item;
}

// The first limb of an item's second factor (products).
template <bool GATHER>
__device__ __forceinline__ const uint64_t *ip_b(const IpArgs &A, uint32_t item) {
    return GATHER ? A.gb[item] : A.b + item * A.add_item;
}

// Many digits (beta > 8): digit by digit, loads interleaved with products,
// so registers stay bounded.  The batch item is the fastest-varying block
// index, so the CTAs of all ciphertexts that read one block of the
// evaluation key are dispatched back to back: the key crosses HBM once per
// batch and is served from L2 after.
template <bool GATHER>
__global__ void __launch_bounds__(256)
k_ip_stream(const IpArgs A, const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const size_t n = size_t(1) << log_n;
    const uint32_t item = blockIdx.x, i = blockIdx.z;
    const size_t x = 2 * (size_t(blockIdx.y) * blockDim.x + threadIdx.x);
    if (x >= n) return;
    const DevMod m = mods[A.prime[i]];
    const uint32_t KL = A.L + A.K;
    const bool own_here = A.own != nullptr && i < A.level;
    const uint32_t own_digit = own_here ? i / A.alpha : 0xffffffffu;
    const uint64_t *ext = A.ext + item * A.ext_item;
    U128 a0{0, 0}, a1{0, 0}, b0{0, 0}, b1{0, 0};
    if (i < A.level && A.pfac[i] != 0) {
        if (A.add0) {
            const ulonglong2 d = ld2(ip_add0<GATHER>(A, item) + size_t(i) * n + x);
            mac(a0, d.x, A.pfac[i]);
            mac(a1, d.y, A.pfac[i]);
        }
        if (A.add1) {
            const ulonglong2 d = ld2(A.add1 + item * A.add_item + size_t(i) * n + x);
            mac(b0, d.x, A.pfac[i]);
            mac(b1, d.y, A.pfac[i]);
        }
    }
    for (uint32_t j = 0; j < A.beta; j++) {
        const ulonglong2 c = (j == own_digit) ? ld2(ip_own<GATHER>(A, item, n) + size_t(i) * n + x)
                                              : ld2(ext + (size_t(j) * A.M + i) * n + x);
        const ulonglong2 kb = ld2(A.key + ((size_t(j) * 2 + 0) * KL + A.key_limb[i]) * n + x);
        const ulonglong2 ka = ld2(A.key + ((size_t(j) * 2 + 1) * KL + A.key_limb[i]) * n + x);
        mac(a0, c.x, kb.x);
        mac(a1, c.y, kb.y);
        mac(b0, c.x, ka.x);
        mac(b1, c.y, ka.y);
    }
    uint64_t *y = A.y + item * A.y_item;
    st2(y + size_t(i) * n + x, csub(redc(a0, m.q, m.qinv), m.q), csub(redc(a1, m.q, m.qinv), m.q));
    st2(y + (size_t(A.M) + i) * n + x, csub(redc(b0, m.q, m.qinv), m.q),
        csub(redc(b1, m.q, m.qinv), m.q));
}

// Inner product with bulk-copy staging: a CTA owns one extended limb i and
// a tile of kIpTile coefficients for every ciphertext of the batch.  Thread
// 0 loads the tile of the 2 BETA key rows once (bulk copies into shared
// memory) and streams each ciphertext's digit (and fold) tiles through two
// shared buffers, the next ciphertext's copies in flight while the threads
// compute on the current one; all threads then read shared memory only.
// Used for BETA <= 8; every address is 16-byte aligned (the bulk-copy rule),
// which the host checks.  Tiles of 512
// coefficients (256 threads) up to 4 digits; 256 coefficients (128 threads)
// for 5 to 8 digits, so that the 2 BETA key tiles and the two buffers
// (72 KB at BETA = 8) leave room for 3 CTAs per SM.
// FORM, bits: the ciphertexts of the launch are gathered; the addends and the
// own digits are the tensor product of two ciphertexts, formed here from
// them (a0 and b0 in the two slots after the digits, a1 in the own digit's);
// there is a second addend (without it and products a buffer has one tile
// less: 16 rotations of 8 ciphertexts at N = 2^16 8043 -> 7924 us).
constexpr int kIpGathered = 1, kIpProduct = 2, kIpTwoAdds = 4;
template <int BETA, int FORM>
struct IpSlots {  // tiles of one ciphertext in a buffer
    static constexpr int value = BETA + (FORM & (kIpProduct | kIpTwoAdds) ? 2 : 1);
};

template <int BETA, int R>
struct IpTile {
    static constexpr uint32_t value = BETA * R <= 4 ? 512 : 256;
};

// blockIdx.z: a group of consecutive ciphertexts of the launch (the host
// splits them when one group per tile would leave the last wave of CTAs
// mostly empty); each group's CTA loads its key tiles once.
// R: keys of the launch.  Hoisted rotations multiply the same digits by one
// key each; with two keys the digits and the first polynomials of 8
// ciphertexts at N = 2^16, l = 24 (453 MB) are read once for both, 1550 ->
// 1098 MB a pair.  Tiles of 256
// coefficients from 3 digits on, so that the key tiles and the two buffers
// (40 KB at 3 digits) leave room for 4 CTAs per SM in the 164 KB split that
// these launches ask for (tiles of 512 are slower, 8080 instead of 8023 us).
// The batch of 16 rotations of 8: 8128 -> 8023 us (the transforms that run
// beside it bound it); 16 rotations of one: 1349 -> 1267 us; 4 at N = 2^12:
// 57.0 -> 52.7 us; 2 or 3 rotations at N >= 2^14 stay one to each stream.
template <int BETA, int FORM, int R>
__global__ void __launch_bounds__(IpTile<BETA, R>::value / 2)
k_ip_bulk(const IpArgs A, const DevMod *__restrict__ mods, uint32_t log_n, uint32_t count) {
    constexpr bool GATHER = (FORM & kIpGathered) != 0, PROD = (FORM & kIpProduct) != 0;
    constexpr int SLOTS = IpSlots<BETA, FORM>::value;
    grid_dep_wait();
    const uint32_t per = (count + gridDim.z - 1) / gridDim.z;
    const uint32_t first = blockIdx.z * per;
    if (first >= count) return;  // an empty group (the whole CTA, before any barrier)
    const uint32_t nloc = count - first < per ? count - first : per;
    constexpr uint32_t kIpTile = IpTile<BETA, R>::value;
    extern __shared__ __align__(128) uint64_t sm[];
    __shared__ __align__(8) uint64_t bars[3];  // buffer 0, buffer 1, keys
    const size_t n = size_t(1) << log_n;
    const uint32_t i = blockIdx.y, tid = threadIdx.x;
    const size_t x0 = size_t(blockIdx.x) * kIpTile;
    const uint32_t beta = A.beta, KL = A.L + A.K;
    const DevMod m = mods[A.prime[i]];
    const bool fold = i < A.level && A.pfac[i] != 0;
    const bool f0 = fold && A.add0, prod = PROD && i < A.level;
    const bool f1 = (FORM & kIpTwoAdds) != 0 && fold;
    const uint32_t own_digit = (A.own != nullptr && i < A.level) ? i / A.alpha : 0xffffffffu;
    constexpr uint32_t TB = kIpTile * 8;  // bytes per tile
    uint64_t *skey = sm;                                   // [R][2 BETA][tile]
    uint64_t *sbuf[2] = {sm + 2 * R * BETA * kIpTile, sm + (2 * R * BETA + SLOTS) * kIpTile};
    const uint32_t item_bytes = (beta + (f0 ? 1 : 0) + (prod || f1 ? 1 : 0)) * TB;

    auto issue_item = [&](uint32_t k, uint32_t b) {  // the group's k-th ciphertext
        const uint32_t item = first + k;
        uint64_t *dst = sbuf[b];
        mbar_expect_tx(&bars[b], item_bytes);
        const uint64_t *ext = A.ext + item * A.ext_item;
        for (uint32_t j = 0; j < beta; j++) {
            const uint64_t *src = (j == own_digit) ? ip_own<GATHER>(A, item, n) + size_t(i) * n
                                                   : ext + (size_t(j) * A.M + i) * n;
            bulk_load(dst + j * kIpTile, src + x0, TB, &bars[b]);
        }
        if (f0) bulk_load(dst + BETA * kIpTile, ip_add0<GATHER>(A, item) + size_t(i) * n + x0, TB, &bars[b]);
        if (f1) bulk_load(dst + (BETA + 1) * kIpTile, A.add1 + item * A.add_item + size_t(i) * n + x0, TB, &bars[b]);
        if (prod) bulk_load(dst + (BETA + 1) * kIpTile, ip_b<GATHER>(A, item) + size_t(i) * n + x0, TB, &bars[b]);
    };

    const uint32_t u = 2 * tid;  // this thread's two coefficients in the tile
    // products: b1's words by plain loads, an item ahead (a third extra tile in
    // each buffer would take 8 digits from 3 CTAs per SM to 2)
    auto load_b1 = [&](uint32_t k) {
        return ld2(ip_b<GATHER>(A, first + k) + (size_t(A.level) + i) * n + x0 + u);
    };
    ulonglong2 b1 = make_ulonglong2(0, 0);
    if (prod) b1 = load_b1(0);
    if (tid == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_init(&bars[2], 1);
        mbar_init_fence();
    }
    __syncthreads();
    if (tid == 0) {
        mbar_expect_tx(&bars[2], 2 * R * beta * TB);
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint64_t *key = r ? A.key2 : A.key;
            uint64_t *dst = skey + r * 2 * BETA * kIpTile;
            for (uint32_t j = 0; j < beta; j++) {
                bulk_load(dst + (2 * j) * kIpTile, key + ((size_t(j) * 2 + 0) * KL + A.key_limb[i]) * n + x0, TB, &bars[2]);
                bulk_load(dst + (2 * j + 1) * kIpTile, key + ((size_t(j) * 2 + 1) * KL + A.key_limb[i]) * n + x0, TB, &bars[2]);
            }
        }
        issue_item(0, 0);
        if (nloc > 1) issue_item(1, 1);
    }
    // every wait is bounded, and the CTA decides together whether to go on
    // (__syncthreads_and), so no thread is left waiting at a barrier
    bool ok = __syncthreads_and(mbar_wait(&bars[2], 0));
    for (uint32_t k = 0; k < nloc && ok; k++) {
        const uint32_t item = first + k, b = k & 1;
        ok = __syncthreads_and(mbar_wait(&bars[b], (k >> 1) & 1));
        if (!ok) break;
        const uint64_t *buf = sbuf[b];
        ulonglong2 d0 = make_ulonglong2(0, 0), d1 = d0, d2 = d0;
        if (prod) {  // the tensor product of this tile; the own digit's slot holds a1
            const ulonglong2 p0 = ld2(buf + BETA * kIpTile + u), q0 = ld2(buf + (BETA + 1) * kIpTile + u);
            const ulonglong2 p1 = ld2(buf + own_digit * kIpTile + u);
            const Tensor t = tensor_mod(p0.x, p1.x, q0.x, b1.x, m);
            const Tensor w = tensor_mod(p0.y, p1.y, q0.y, b1.y, m);
            d0 = make_ulonglong2(t.d0, w.d0);
            d1 = make_ulonglong2(t.d1, w.d1);
            d2 = make_ulonglong2(t.d2, w.d2);
            if (k + 1 < nloc) b1 = load_b1(k + 1);
        } else {
            if (f0) d0 = ld2(buf + BETA * kIpTile + u);
            if (f1) d1 = ld2(buf + (BETA + 1) * kIpTile + u);
        }
#pragma unroll
        for (int r = 0; r < R; r++) {
            const uint64_t *key = skey + r * 2 * BETA * kIpTile;
            U128 a0{0, 0}, a1{0, 0}, b0{0, 0}, b1s{0, 0};
            if (f0) {
                mac(a0, d0.x, A.pfac[i]);
                mac(a1, d0.y, A.pfac[i]);
            }
            if (prod || f1) {
                mac(b0, d1.x, A.pfac[i]);
                mac(b1s, d1.y, A.pfac[i]);
            }
#pragma unroll
            for (int j = 0; j < BETA; j++) {
                if (uint32_t(j) < beta) {
                    const ulonglong2 c = prod && uint32_t(j) == own_digit ? d2 : ld2(buf + j * kIpTile + u);
                    const ulonglong2 kb = ld2(key + (2 * j) * kIpTile + u);
                    const ulonglong2 ka = ld2(key + (2 * j + 1) * kIpTile + u);
                    mac(a0, c.x, kb.x);
                    mac(a1, c.y, kb.y);
                    mac(b0, c.x, ka.x);
                    mac(b1s, c.y, ka.y);
                }
            }
            uint64_t *y = (r ? A.y2 : A.y) + item * A.y_item + x0 + u;
            st2(y + size_t(i) * n, csub(redc(a0, m.q, m.qinv), m.q), csub(redc(a1, m.q, m.qinv), m.q));
            st2(y + (size_t(A.M) + i) * n, csub(redc(b0, m.q, m.qinv), m.q),
                csub(redc(b1s, m.q, m.qinv), m.q));
        }
        __syncthreads();  // everyone is done with buffer b
        if (tid == 0 && k + 2 < nloc) {
            fence_proxy_async();
            issue_item(k + 2, b);
        }
    }
    if (!ok && tid == 0) {
        atomicOr(A.status, kStatusIpWait);
        // give this CTA's copies still in flight a bounded time to land
        mbar_wait(&bars[0], 0);
        mbar_wait(&bars[1], 0);
    }
}

// Watchdog self-test: a barrier that expects 16 bytes of bulk-copy data that
// no copy ever brings; the bounded wait must give up after limit_ns and the
// kernel must report it in the status word and return.
__global__ void k_wait_selftest(int *status, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_expect_tx(&bar, 16);
    const bool ok = __syncthreads_and(mbar_wait(&bar, 0, limit_ns));
    if (!ok && threadIdx.x == 0) atomicOr(status, kStatusSelfTestWait);
}

int launch_wait_selftest(const Context &c, uint64_t limit_ns, cudaStream_t s) {
    k_wait_selftest<<<1, 64, 0, s>>>(c.d_status, limit_ns);
    return ok();
}

static bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// Ciphertext groups of a bulk inner-product launch: 1 to 4, whichever fills
// the waves of CTAs best (resident CTAs per SM from the occupancy API), with
// the groups' uneven sizes counted, and only if that beats one group by 10%
// (each more group reloads its key tiles).  At N = 2^14 with 8 digits, 64
// tiles x 9 limbs at 3 CTAs per SM is 1.26 waves in one group, 2.53 in two.
template <typename K>
static unsigned ip_groups(K kernel, unsigned threads, size_t smem, size_t ctas, uint32_t count) {
    if (count < 2) return 1;
    const int slots_i = resident_slots(reinterpret_cast<const void *>(kernel), int(threads), smem);
    if (slots_i <= 0) return 1;
    const double slots = double(slots_i);
    auto score = [&](uint32_t g) {
        const double waves = double(ctas) * g / slots;
        const uint32_t per = (count + g - 1) / g;
        return waves / std::ceil(waves) * (double(count) / g / per);
    };
    unsigned best = 1;
    const double one = score(1);
    double top = one;
    for (uint32_t g = 2; g <= 4 && g <= count; g++)
        if (score(g) > top + 1e-9) {
            top = score(g);
            best = g;
        }
    return top >= 1.1 * one ? best : 1;
}

template <int BETA, int FORM, int R>
static int ip_run_bulk(const Context &c, const IpArgs &a, uint32_t count, cudaStream_t s) {
    constexpr uint32_t tile = IpTile<BETA, R>::value;
    // two buffers of the ciphertexts' tiles, one when each CTA has a single
    // ciphertext (then more CTAs are resident, 5 instead of 3 per SM at 3 digits:
    // one product at N = 2^16, l = 24 201.8 -> 199.4 us, the 256-operation mix
    // 9.70 -> 9.55 ms)
    const auto kernel = k_ip_bulk<BETA, FORM, R>;
    const void *const k = reinterpret_cast<const void *>(kernel);
    constexpr int slots = IpSlots<BETA, FORM>::value;
    constexpr size_t one = size_t(2 * R * BETA + slots) * tile * 8, two = one + size_t(slots) * tile * 8;
    const unsigned groups =
        count > 1 ? ip_groups(kernel, tile / 2, two, c.n / tile * a.M, count) : 1;
    const size_t smem = groups >= count ? one : two;
    if (!allow_smem(k, two)) return CATFHE_ECUDA;
    launch_pdl_split(R > 1 ? kSharedPercent : 0, kernel, dim3(unsigned(c.n / tile), a.M, groups),
                     dim3(tile / 2), smem, s, a, c.d_mods, uint32_t(c.log_n), count);
    return ok();
}

template <int FORM, int R>
static int ip_run(const Context &c, const IpArgs &a, uint32_t count, cudaStream_t s) {
    switch (a.beta) {
        case 1:
            if constexpr (R > 1) return CATFHE_EINVAL;  // one digit: not paired
            else return ip_run_bulk<1, FORM, R>(c, a, count, s);
        case 2: return ip_run_bulk<2, FORM, R>(c, a, count, s);
        case 3: return ip_run_bulk<3, FORM, R>(c, a, count, s);
        case 4: return ip_run_bulk<4, FORM, R>(c, a, count, s);
        case 5: return ip_run_bulk<5, FORM, R>(c, a, count, s);
        case 6: return ip_run_bulk<6, FORM, R>(c, a, count, s);
        case 7: return ip_run_bulk<7, FORM, R>(c, a, count, s);
        case 8: return ip_run_bulk<8, FORM, R>(c, a, count, s);
        default:
            if constexpr (R > 1 || (FORM & kIpProduct) != 0) return CATFHE_EINVAL;
            else {
                launch_pdl(k_ip_stream<FORM == kIpGathered>, dim3(count, unsigned((c.n / 2 + 255) / 256), a.M),
                           dim3(256), 0, s, a, c.d_mods, uint32_t(c.log_n));
                return ok();
            }
    }
}

int launch_ip(const Context &c, const IpArgs &a, uint32_t count, cudaStream_t s) {
    // bulk copies: every buffer is a workspace, a key or a ciphertext, refused
    // at the entry points unless 16-byte aligned
    bool aligned = a.status != nullptr && aligned16(a.ext) && aligned16(a.key) && aligned16(a.y) &&
                   aligned16(a.own) && aligned16(a.add0) && aligned16(a.add1) && aligned16(a.key2) &&
                   aligned16(a.y2) && aligned16(a.b) &&
                   ((a.ext_item | a.own_item | a.add_item | a.y_item) & 1) == 0;
    for (uint32_t k = 0; a.gathered && k < count; k++)
        aligned = aligned && aligned16(a.ga[k]) && (!a.product || aligned16(a.gb[k]));
    if (!aligned) return CATFHE_EINVAL;
    if (a.product) {
        // two ciphertexts and nothing else, at most kIpBulkBeta digits
        if (a.add1 || a.key2 || !a.own || !a.add0) return CATFHE_EINVAL;
        return a.gathered ? ip_run<kIpProduct | kIpGathered, 1>(c, a, count, s)
                          : ip_run<kIpProduct, 1>(c, a, count, s);
    }
    if (a.add1)
        return a.gathered || a.key2 ? CATFHE_EINVAL : ip_run<kIpTwoAdds, 1>(c, a, count, s);
    if (a.key2) return a.gathered ? CATFHE_EINVAL : ip_run<0, 2>(c, a, count, s);
    return a.gathered ? ip_run<kIpGathered, 1>(c, a, count, s) : ip_run<0, 1>(c, a, count, s);
}

// ------------------------------------------------------------------ ModDown combine

// out_p[i] = (y_p[i] - lift_p[i]) * D^-1 (+ add_p[i]), coefficient form (the
// lift in [0, 4q), or formed here from the one special limb); with
// a Galois element g the coefficient at x goes to x g mod 2N, negated past N
// (one scattered store per word instead of permuted copies of the inputs).
__global__ void __launch_bounds__(256)
k_combine(const CombineArgs A, const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const size_t n = size_t(1) << log_n;
    const size_t x = 2 * (size_t(blockIdx.x) * blockDim.x + threadIdx.x);
    const uint32_t i = blockIdx.y % A.lo, p = blockIdx.y / A.lo, item = blockIdx.z;
    if (x >= n) return;
    const DevMod m = mods[A.prime[i]];
    const uint64_t q = m.q;
    const uint64_t *yp = A.y + item * A.y_item + p * A.y_poly + x;
    const ulonglong2 y = ld2(yp + size_t(i) * n);
    ulonglong2 l;
    if (A.lift) {
        l = ld2(A.lift + item * A.lift_item + p * A.lift_poly + size_t(i) * n + x);
    } else {
        const ulonglong2 v = ld2(yp + A.y_last);
        const LiftEntry e = A.lifts[i];
        l = make_ulonglong2(lift_word(v.x, e, m), lift_word(v.y, e, m));
    }
    uint64_t r0 = shoup(y.x + 4 * q - l.x, A.dinv[i], A.dinv_s[i], q);
    uint64_t r1 = shoup(y.y + 4 * q - l.y, A.dinv[i], A.dinv_s[i], q);
    if (A.add && p < A.add_polys) {
        const ulonglong2 d = ld2(A.add + item * A.add_item + p * A.add_poly + size_t(i) * n + x);
        r0 = add_mod(r0, d.x, q);
        r1 = add_mod(r1, d.y, q);
    }
    uint64_t *o = A.out + item * A.out_item + p * A.out_poly + size_t(i) * n;
    if (!A.galois) {
        st2(o + x, r0, r1);
        return;
    }
    const uint32_t k0 = (uint32_t(x) * A.galois) & uint32_t(2 * n - 1);
    const uint32_t k1 = (k0 + A.galois) & uint32_t(2 * n - 1);
    o[k0 & (n - 1)] = k0 >= n && r0 ? q - r0 : r0;
    o[k1 & (n - 1)] = k1 >= n && r1 ? q - r1 : r1;
}

int launch_combine(const Context &c, const CombineArgs &a, uint32_t count, cudaStream_t s) {
    launch_pdl(k_combine, coeff_grid(c.n / 2, 2 * a.lo, count), dim3(256), 0, s, a, c.d_mods,
               uint32_t(c.log_n));
    return ok();
}

// ------------------------------------------------------------------ automorphism

// NTT form: slot k = bitrev(i) holds a(psi^(2i+1)); sigma_g(a) there is
// a(psi^((2i+1) g)), a pure permutation of the slots.
__global__ void __launch_bounds__(256)
k_automorph_ntt(const uint64_t *__restrict__ in, uint64_t *__restrict__ out, uint64_t g,
                uint32_t log_n) {
    grid_dep_wait();
    const size_t n = size_t(1) << log_n;
    const size_t k = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const uint64_t mask2n = 2 * n - 1;
    const uint32_t i = __brev(uint32_t(k)) >> (32 - log_n);
    const uint64_t e = ((2 * uint64_t(i) + 1) * g) & mask2n;
    const uint32_t src = __brev(uint32_t((e - 1) >> 1)) >> (32 - log_n);
    const size_t limb = blockIdx.y;
    out[limb * n + k] = in[limb * n + src];
}

int launch_automorph_ntt(const Context &c, const uint64_t *in, uint64_t *out, uint32_t limbs_total,
                         uint64_t g, cudaStream_t s) {
    launch_pdl(k_automorph_ntt, coeff_grid(c.n, limbs_total), dim3(256), 0, s, in, out,
               uint64_t(g % (2 * c.n)), uint32_t(c.log_n));
    return ok();
}

// ------------------------------------------------------------------ plaintext product

__global__ void __launch_bounds__(256)
k_mul_plain(const uint64_t *__restrict__ a, const uint64_t *__restrict__ pt, uint64_t *out,
            uint32_t level, const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const size_t n = size_t(1) << log_n;
    const size_t x = 2 * (size_t(blockIdx.x) * blockDim.x + threadIdx.x);
    if (x >= n) return;
    const uint32_t limb = blockIdx.y, i = limb % level;
    const DevMod m = mods[i];
    const ulonglong2 v = ld2(a + size_t(limb) * n + x), w = ld2(pt + size_t(i) * n + x);
    st2(out + size_t(limb) * n + x, mul_mod(v.x, w.x, m), mul_mod(v.y, w.y, m));
}

int launch_mul_plain(const Context &c, const uint64_t *a, const uint64_t *pt, uint64_t *out,
                     uint32_t level, uint32_t n_limbs, cudaStream_t s) {
    if (n_limbs == 0) return CATFHE_OK;
    launch_pdl(k_mul_plain, coeff_grid(c.n / 2, n_limbs), dim3(256), 0, s, a, pt, out, level,
               c.d_mods, uint32_t(c.log_n));
    return ok();
}

// ------------------------------------------------------------------ simple maps

// Streams over the limbs of a map: they do a few instructions per word, so
// what counts is bytes in flight.  A thread takes two pairs of words, 512
// apart (16-byte loads, all issued before the first use).  One 8-byte word per
// thread reached half of the copy rate (a product by a constant at N = 2^16,
// 20 primes: 13.5 us of which 6.3 are its bytes) and was a quarter of the query
// server's device time: eight queries 79.0 -> 73.3 ms.
constexpr uint32_t kMapWords = 1024;  // per CTA of 256 threads

static inline dim3 map_grid(size_t n, uint32_t limbs) { return dim3(unsigned(n / kMapWords), limbs); }

template <class F>
__device__ __forceinline__ void map_words(const uint64_t *a, const uint64_t *b, uint64_t *out, F f) {
    const uint32_t x = blockIdx.x * kMapWords + 2 * threadIdx.x;
    const ulonglong2 a0 = ld2(a + x), a1 = ld2(a + x + kMapWords / 2);
    ulonglong2 b0 = make_ulonglong2(0, 0), b1 = b0;
    if (b) {
        b0 = ld2(b + x);
        b1 = ld2(b + x + kMapWords / 2);
    }
    st2(out + x, f(a0.x, b0.x), f(a0.y, b0.y));
    st2(out + x + kMapWords / 2, f(a1.x, b1.x), f(a1.y, b1.y));
}

// a and b in the map's source layout, out too.
template <bool SUB>
__global__ void __launch_bounds__(256)
k_add_sub(const uint64_t *a, const uint64_t *b, uint64_t *out, const LimbMap map,
          const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const uint32_t limb = blockIdx.y, g = limb / map.period, r = limb % map.period;
    const size_t o = (size_t(g) * map.src_stride + map.src_off[r]) << log_n;
    const uint64_t q = mods[map.prime[r]].q;
    map_words(a + o, b + o, out + o,
              [q](uint64_t u, uint64_t v) { return SUB ? sub_mod(u, v, q) : add_mod(u, v, q); });
}

int launch_add(const Context &c, const uint64_t *a, const uint64_t *b, uint64_t *out,
               const LimbMap &map, uint32_t n_limbs, cudaStream_t s) {
    launch_pdl(k_add_sub<false>, map_grid(c.n, n_limbs), dim3(256), 0, s, a, b, out, map, c.d_mods,
               uint32_t(c.log_n));
    return ok();
}

int launch_sub(const Context &c, const uint64_t *a, const uint64_t *b, uint64_t *out,
               const LimbMap &map, uint32_t n_limbs, cudaStream_t s) {
    launch_pdl(k_add_sub<true>, map_grid(c.n, n_limbs), dim3(256), 0, s, a, b, out, map, c.d_mods,
               uint32_t(c.log_n));
    return ok();
}

// out = a * k_r (a constant per map entry, Shoup pair), or a + k_r on the
// entries with add set (adding a constant polynomial in NTT form).
struct ConstArgs {
    uint64_t k[kMapMax], k_s[kMapMax];
    uint8_t add[kMapMax];
};

__global__ void __launch_bounds__(256)
k_const_op(const uint64_t *a, uint64_t *out, const LimbMap map, const ConstArgs C,
           const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const uint32_t limb = blockIdx.y, g = limb / map.period, r = limb % map.period;
    const size_t o = (size_t(g) * map.src_stride + map.src_off[r]) << log_n;
    const uint64_t q = mods[map.prime[r]].q, k = C.k[r], ks = C.k_s[r];
    if (C.add[r])
        map_words(a + o, nullptr, out + o, [=](uint64_t u, uint64_t) { return add_mod(u, k, q); });
    else
        map_words(a + o, nullptr, out + o, [=](uint64_t u, uint64_t) { return shoup(u, k, ks, q); });
}

int launch_const_op(const Context &c, const uint64_t *a, uint64_t *out, const LimbMap &map,
                    uint32_t n_limbs, const uint64_t *k, const uint64_t *k_s, const uint8_t *add,
                    cudaStream_t s) {
    ConstArgs C{};
    for (uint32_t r = 0; r < map.period; r++) {
        C.k[r] = k[r];
        C.k_s[r] = k_s[r];
        C.add[r] = add[r];
    }
    launch_pdl(k_const_op, map_grid(c.n, n_limbs), dim3(256), 0, s, a, out, map, C, c.d_mods,
               uint32_t(c.log_n));
    return ok();
}

__global__ void __launch_bounds__(256)
k_copy(const uint64_t *__restrict__ src, uint64_t *__restrict__ dst, const LimbMap map,
       uint32_t log_n) {
    grid_dep_wait();
    const uint32_t limb = blockIdx.y, g = limb / map.period, r = limb % map.period;
    map_words(src + ((size_t(g) * map.src_stride + map.src_off[r]) << log_n), nullptr,
              dst + ((size_t(g) * map.dst_stride + map.dst_off[r]) << log_n),
              [](uint64_t u, uint64_t) { return u; });
}

int launch_copy_limbs(const Context &c, const uint64_t *src, uint64_t *dst, const LimbMap &map,
                      uint32_t n_limbs, cudaStream_t s) {
    launch_pdl(k_copy, map_grid(c.n, n_limbs), dim3(256), 0, s, src, dst, map, uint32_t(c.log_n));
    return ok();
}

__global__ void __launch_bounds__(256)
k_pointwise(const uint64_t *__restrict__ a, const uint64_t *__restrict__ b, uint64_t *out,
            const LimbMap map, const DevMod *__restrict__ mods, uint32_t log_n) {
    const size_t n = size_t(1) << log_n;
    const size_t x = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const uint32_t limb = blockIdx.y, g = limb / map.period, r = limb % map.period;
    const size_t ia = (size_t(g) * map.src_stride + map.src_off[r]) * n + x;
    const size_t io = (size_t(g) * map.dst_stride + map.dst_off[r]) * n + x;
    out[io] = mul_mod(a[ia], b[io], mods[map.prime[r]]);
}

// out[dst] = a[src] * b[dst] over the map
int launch_pointwise(const Context &c, const uint64_t *a, const uint64_t *b, uint64_t *out,
                     const LimbMap &map, uint32_t n_limbs, cudaStream_t s) {
    k_pointwise<<<coeff_grid(c.n, n_limbs), 256, 0, s>>>(a, b, out, map, c.d_mods, c.log_n);
    return ok();
}

// out[i] = c0[i] + c1[i] * sk[i] (or c0 - c1 sk), limbs 0..limbs-1 mod q_i.
__global__ void __launch_bounds__(256)
k_mul_add(const uint64_t *c0, const uint64_t *c1, const uint64_t *__restrict__ sk, uint64_t *out,
          int negate, const DevMod *__restrict__ mods, uint32_t log_n) {
    grid_dep_wait();
    const size_t n = size_t(1) << log_n;
    const size_t x = 2 * (size_t(blockIdx.x) * blockDim.x + threadIdx.x);
    if (x >= n) return;
    const uint32_t i = blockIdx.y;
    const DevMod m = mods[i];
    const size_t o = size_t(i) * n + x;
    const ulonglong2 u = ld2(c1 + o), k = ld2(sk + o);
    const ulonglong2 b = c0 ? ld2(c0 + o) : make_ulonglong2(0, 0);
    const uint64_t p0 = mul_mod(u.x, k.x, m), p1 = mul_mod(u.y, k.y, m);
    if (negate)
        st2(out + o, sub_mod(b.x, p0, m.q), sub_mod(b.y, p1, m.q));
    else
        st2(out + o, add_mod(b.x, p0, m.q), add_mod(b.y, p1, m.q));
}

int launch_mul_add(const Context &c, const uint64_t *c0, const uint64_t *c1, const uint64_t *sk,
                   uint64_t *out, uint32_t limbs, int negate_product, cudaStream_t s) {
    launch_pdl(k_mul_add, coeff_grid(c.n / 2, limbs), dim3(256), 0, s, c0, c1, sk, out,
               negate_product, c.d_mods, uint32_t(c.log_n));
    return ok();
}

// b[i] = -a[i] sk[i] + e[i] + pfac_i sp[i] (NTT form, limbs of Q_L u P).
__global__ void __launch_bounds__(256)
k_ksk_row(const uint64_t *__restrict__ a, const uint64_t *__restrict__ sk,
          const uint64_t *__restrict__ e, const uint64_t *__restrict__ sp, uint64_t *b,
          const uint64_t *__restrict__ pfac, const uint64_t *__restrict__ pfac_s,
          const DevMod *__restrict__ mods, uint32_t log_n) {
    const size_t n = size_t(1) << log_n;
    const size_t x = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const uint32_t i = blockIdx.y;
    const DevMod m = mods[i];
    const size_t o = size_t(i) * n + x;
    uint64_t v = sub_mod(e[o], mul_mod(a[o], sk[o], m), m.q);
    if (pfac[i]) v = add_mod(v, shoup(sp[o], pfac[i], pfac_s[i], m.q), m.q);
    b[o] = v;
}

__global__ void __launch_bounds__(256)
k_scale_limbs(uint64_t *x, uint32_t limbs, const uint64_t *__restrict__ w,
              const uint64_t *__restrict__ w_s, const DevMod *__restrict__ mods, uint32_t log_n) {
    const size_t n = size_t(1) << log_n;
    const size_t j = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const uint32_t i = blockIdx.y % limbs;
    uint64_t *p = x + size_t(blockIdx.y) * n + j;
    *p = shoup(*p, w[i], w_s[i], mods[i].q);
}

int launch_scale_limbs(const Context &c, uint64_t *x, uint32_t limbs, uint32_t groups,
                       const uint64_t *w, const uint64_t *w_s, cudaStream_t s) {
    k_scale_limbs<<<coeff_grid(c.n, limbs * groups), 256, 0, s>>>(x, limbs, w, w_s, c.d_mods,
                                                                c.log_n);
    return ok();
}

int launch_ksk_row(const Context &c, const uint64_t *a, const uint64_t *sk, const uint64_t *e,
                   const uint64_t *sp, uint64_t *b, uint32_t limbs, const uint64_t *pfac,
                   const uint64_t *pfac_s, cudaStream_t s) {
    k_ksk_row<<<coeff_grid(c.n, limbs), 256, 0, s>>>(a, sk, e, sp, b, pfac, pfac_s, c.d_mods,
                                                     c.log_n);
    return ok();
}

// ------------------------------------------------------------------ sampling

__device__ __forceinline__ uint32_t rotl(uint32_t x, int r) { return (x << r) | (x >> (32 - r)); }

#define QR(a, b, c, d)                     \
    a += b; d ^= a; d = rotl(d, 16);       \
    c += d; b ^= c; b = rotl(b, 12);       \
    a += b; d ^= a; d = rotl(d, 8);        \
    c += d; b ^= c; b = rotl(b, 7);

// One ChaCha20 block (RFC 8439 Sec. 2.3): 16 output words.
__device__ __forceinline__ void chacha_block(const SampleArgs &A, uint32_t counter, uint32_t out[16]) {
    uint32_t s[16];
    s[0] = 0x61707865u; s[1] = 0x3320646eu; s[2] = 0x79622d32u; s[3] = 0x6b206574u;
#pragma unroll
    for (int i = 0; i < 8; i++) s[4 + i] = A.key[i];
    s[12] = counter; s[13] = A.tag; s[14] = A.i0; s[15] = A.i1;
    uint32_t x[16];
#pragma unroll
    for (int i = 0; i < 16; i++) x[i] = s[i];
#pragma unroll 1
    for (int r = 0; r < 10; r++) {
        QR(x[0], x[4], x[8], x[12]);
        QR(x[1], x[5], x[9], x[13]);
        QR(x[2], x[6], x[10], x[14]);
        QR(x[3], x[7], x[11], x[15]);
        QR(x[0], x[5], x[10], x[15]);
        QR(x[1], x[6], x[11], x[12]);
        QR(x[2], x[7], x[8], x[13]);
        QR(x[3], x[4], x[9], x[14]);
    }
#pragma unroll
    for (int i = 0; i < 16; i++) out[i] = x[i] + s[i];
}
#undef QR

// word w of the keystream = little-endian bytes 8w..8w+7: block w/8,
// 32-bit words 2(w%8) (low) and 2(w%8)+1 (high).
__global__ void __launch_bounds__(256)
k_sample(const SampleArgs A, uint64_t *out, const LimbMap map, const DevMod *__restrict__ mods,
         const uint64_t *__restrict__ mult, const uint64_t *__restrict__ mult_s, uint32_t n_limbs,
         uint32_t log_n) {
    const size_t n = size_t(1) << log_n;
    const size_t blk = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    uint32_t o[16];
    if (A.kind == kUniform) {
        // block b covers coefficients k = 4b .. 4b+3 (k = limb * N + j)
        if (blk * 4 >= size_t(n_limbs) * n) return;
        chacha_block(A, uint32_t(blk), o);
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const size_t k = blk * 4 + u;
            const uint32_t r = uint32_t(k / n);
            const size_t j = k % n;
            const uint64_t hi = uint64_t(o[4 * u]) | (uint64_t(o[4 * u + 1]) << 32);
            const uint64_t lo = uint64_t(o[4 * u + 2]) | (uint64_t(o[4 * u + 3]) << 32);
            const DevMod m = mods[map.prime[r % map.period]];
            const uint32_t g = r / map.period, rr = r % map.period;
            out[(size_t(g) * map.dst_stride + map.dst_off[rr]) * n + j] = reduce128(U128{lo, hi}, m);
        }
        return;
    }
    // block b covers coefficients j = 8b .. 8b+7 of the small polynomial
    if (blk * 8 >= n) return;
    chacha_block(A, uint32_t(blk), o);
    int64_t v[8];
#pragma unroll
    for (int u = 0; u < 8; u++) {
        const uint64_t w = uint64_t(o[2 * u]) | (uint64_t(o[2 * u + 1]) << 32);
        if (A.kind == kTernary) {
            v[u] = int64_t(w % 3) - 1;
        } else {
            const uint64_t low = w & ((uint64_t(1) << 40) - 1);
            int64_t mag = 0;
#pragma unroll
            for (int t = 0; t < 19; t++) mag += (low >= A.cdt[t]) ? 1 : 0;
            v[u] = (w >> 63) ? -mag : mag;
        }
    }
    for (uint32_t l = 0; l < n_limbs; l++) {
        const uint32_t g = l / map.period, rr = l % map.period;
        const DevMod m = mods[map.prime[rr]];
        uint64_t *dst = out + (size_t(g) * map.dst_stride + map.dst_off[rr]) * n + blk * 8;
#pragma unroll
        for (int u = 0; u < 8; u++) {
            uint64_t r = v[u] < 0 ? m.q - uint64_t(-v[u]) : uint64_t(v[u]);
            if (mult) r = shoup(r, mult[rr], mult_s[rr], m.q);
            dst[u] = r;
        }
    }
}

int launch_sample(const Context &c, const SampleArgs &a, uint64_t *out, const LimbMap &map,
                  uint32_t n_limbs, const uint64_t *mult, const uint64_t *mult_s,
                  cudaStream_t s) {
    size_t blocks = a.kind == kUniform ? (size_t(n_limbs) * c.n + 3) / 4 : (c.n + 7) / 8;
    k_sample<<<unsigned((blocks + 255) / 256), 256, 0, s>>>(a, out, map, c.d_mods, mult, mult_s,
                                                            n_limbs, c.log_n);
    return ok();
}

// int64 coefficients -> residues (times mult), optionally added to out.
__global__ void __launch_bounds__(256)
k_small_to_rns(const int64_t *__restrict__ in, uint64_t *out, const LimbMap map,
               const DevMod *__restrict__ mods, const uint64_t *__restrict__ mult,
               const uint64_t *__restrict__ mult_s, int accumulate, uint32_t log_n) {
    const size_t n = size_t(1) << log_n;
    const size_t x = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const uint32_t limb = blockIdx.y, g = limb / map.period, r = limb % map.period;
    const DevMod m = mods[map.prime[r]];
    const int64_t v = in[x];
    uint64_t res = v < 0 ? m.q - reduce64(uint64_t(-(v + 1)) + 1, m) : reduce64(uint64_t(v), m);
    res = csub(res, m.q);
    if (mult) res = shoup(res, mult[r], mult_s[r], m.q);
    uint64_t *o = out + (size_t(g) * map.dst_stride + map.dst_off[r]) * n + x;
    *o = accumulate ? add_mod(*o, res, m.q) : res;
}

int launch_small_to_rns(const Context &c, const int64_t *in, uint64_t *out, const LimbMap &map,
                        uint32_t n_limbs, const uint64_t *mult, const uint64_t *mult_s,
                        int accumulate, cudaStream_t s) {
    k_small_to_rns<<<coeff_grid(c.n, n_limbs), 256, 0, s>>>(in, out, map, c.d_mods, mult, mult_s,
                                                           accumulate, c.log_n);
    return ok();
}

}  // namespace catfhe
