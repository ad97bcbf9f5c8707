// Plans of the tensor-core base conversion (conv_mma.cu): the constants of
// one exact, centred conversion from K source to T target moduli in the form
// that kernel reads, one image copied to shared memory as it is.
//
// With y_i = r_i pre_i (M/m_i)^-1 mod m_i (in [0, 2 m_i)) and v = round(sum y_i / m_i), the
// centred value is x_c = sum y_i M/m_i - v M, so for a target p (weights
// W_i = post M/m_i mod p and V = -post M mod p)
//     x_c post = sum_i sum_e y_i[e] (2^(8e) W_i mod p) + v V   (mod p),
// y_i[e] the bytes of y_i: a product of a row of small integers and a matrix.
// Every weight is taken centred mod p and written in D balanced base-1024
// digits, one column each; the kernel multiplies byte - 128 (exact in fp16,
// as the digits are) and accumulates in fp32.  A column's sums stay below
// 2^22 in magnitude, checked here against its actual weights, so they are
// exact integers (relied on: products of fp16 whole numbers are exact and the
// tensor core adds whole numbers below 2^24 exactly, in any order); a constant row adds 3 * 2^22, which puts the sum's bits in
// the float's low mantissa.  S_d the sums of a target's columns, the result is
//     r = sum_d S_d 2^(10 d) + C0 - (e - 1) p,  C0 = 128 sum of all weights,
// e the rounded quotient, from the top three columns in fp32: r is in
// (0.4 p, 1.6 p).
#include <math.h>
#include <string.h>

#include <algorithm>

#include "internal.h"

namespace catfhe {

typedef unsigned __int128 u128;

// Integer of magnitude at most 2048 or a small power of two -> fp16 bits.
static uint16_t half_bits(int v) {
    if (v == 0) return 0;
    const uint16_t sign = v < 0 ? 0x8000 : 0;
    uint32_t m = uint32_t(v < 0 ? -v : v);
    int e = 31 - __builtin_clz(m);
    m = e <= 10 ? m << (10 - e) : m >> (e - 10);
    return uint16_t(sign | uint32_t(e + 15) << 10 | (m & 0x3ff));
}

static int bit_length(uint64_t x) { return 64 - __builtin_clzll(x); }

// Balanced base-1024 digits of the centred representative of w mod p.
static bool balanced_digits(uint64_t w, uint64_t p, int D, int out[6]) {
    int64_t v = w > p / 2 ? -int64_t(p - w) : int64_t(w);
    for (int d = 0; d < D; d++) {
        if (d == D - 1) {
            if (v < -512 || v > 512) return false;
            out[d] = int(v);
        } else {
            const int64_t lowbits = v & 1023;
            out[d] = int(lowbits >= 512 ? lowbits - 1024 : lowbits);
            v = (v - out[d]) >> 10;
        }
    }
    return true;
}

std::vector<uint64_t> build_mma_plan(const PlanSpec &s, uint64_t n, uint64_t target_unit) {
    const uint32_t K = uint32_t(s.src_mod.size()), T = uint32_t(s.dst_mod.size());
    if (K < 1 || K > kMmaMaxK || T < 1 || !plan_fits_mont(s)) return {};
    for (uint64_t m : s.src_mod)
        if (m >> 60 || !(m >> 32)) return {};
    for (uint64_t p : s.dst_mod)
        if (p >> 60 || !(p >> 40)) return {};
    // targets in blocks of columns: 5 digits for p below 2^50, else 6
    struct Block {
        int D;
        std::vector<uint32_t> t;
    };
    std::vector<Block> blocks;
    for (int D = 5; D <= 6; D++) {
        size_t first = blocks.size();
        for (uint32_t t = 0; t < T; t++) {
            if ((s.dst_mod[t] < (uint64_t(1) << 50) ? 5 : 6) != D) continue;
            if (blocks.size() == first || blocks.back().t.size() == size_t(int(kMmaBlock) / D))
                blocks.push_back(Block{D, {}});
            blocks.back().t.push_back(t);
        }
    }
    const uint32_t nblk = uint32_t(blocks.size()), N = kMmaBlock * nblk;
    if (nblk > kMmaMaxBlocks) return {};
    const MmaLayout lay = mma_layout(K, nblk);
    std::vector<uint64_t> img(lay.words, 0);
    uint64_t dmask = 0;
    for (uint32_t b = 0; b < nblk; b++) {
        dmask |= uint64_t(blocks[b].D == 6) << b;
        img[1] |= uint64_t(blocks[b].t.size()) << (4 * b);
    }
    img[0] = uint64_t(K) | uint64_t(nblk) << 8 | uint64_t(lay.cores) << 16 |
             uint64_t(s.lazy ? 1 : 0) << 24 | dmask << 32;
    const auto &m = s.src_mod;
    for (uint32_t i = 0; i < K; i++) {
        uint64_t Mi = 1 % m[i];  // M / m_i mod m_i
        for (uint32_t l = 0; l < K; l++)
            if (l != i) Mi = h_mulmod(Mi, m[l] % m[i], m[i]);
        const uint64_t pre = s.pre.empty() ? 1 : s.pre[i] % m[i];
        const uint64_t w = h_mulmod(pre, h_invmod(Mi, m[i]), m[i]);
        const int sh = bit_length(m[i]) - 31;
        uint64_t *o = img.data() + lay.src + size_t(i) * kMmaSrcWords;
        o[0] = m[i];
        o[1] = w;
        o[2] = h_shoup(w, m[i]);
        // y / m_i in units of 2^-27: (y >> sh) c / 2^32
        o[3] = uint64_t(((u128)1 << (sh + 59)) / m[i]) | uint64_t(sh) << 32;
        o[4] = s.src_off[i] * n;
    }
    uint16_t *B = reinterpret_cast<uint16_t *>(img.data() + lay.b);
    auto put = [&](uint32_t core, uint32_t col, uint32_t e, int v) {
        B[(size_t(core) * N + col) * 8 + e] = half_bits(v);
    };
    for (uint32_t b = 0; b < nblk; b++) {
        const int D = blocks[b].D;
        for (uint32_t j = 0; j < blocks[b].t.size(); j++) {
            const uint32_t t = blocks[b].t[j], col = kMmaBlock * b + j * uint32_t(D);
            const uint64_t p = s.dst_mod[t];
            const uint64_t post = s.post.empty() ? 1 : s.post[t] % p;
            int64_t bound[6] = {};
            int dig[6];
            uint64_t c0 = 0;  // 128 times the sum of the weights, mod p
            for (uint32_t i = 0; i < K; i++) {
                uint64_t W = post;
                for (uint32_t l = 0; l < K; l++)
                    if (l != i) W = h_mulmod(W, m[l] % p, p);
                const int bytes = (bit_length(2 * m[i]) + 7) / 8;
                for (int e = 0; e < bytes; e++) {
                    if (!balanced_digits(W, p, D, dig)) return {};
                    for (int d = 0; d < D; d++) {
                        put(i, col + uint32_t(d), uint32_t(e), dig[d]);
                        bound[d] += 128 * int64_t(dig[d] < 0 ? -dig[d] : dig[d]);
                    }
                    c0 = (c0 + h_mulmod(W, 128, p)) % p;
                    W = h_mulmod(W, 256, p);
                }
            }
            uint64_t V = post;
            for (uint32_t l = 0; l < K; l++) V = h_mulmod(V, m[l] % p, p);
            V = (p - V) % p;
            if (!balanced_digits(V, p, D, dig)) return {};
            for (int d = 0; d < D; d++) {
                put(K, col + uint32_t(d), 0, dig[d]);
                put(K, col + uint32_t(d), 1, 4096);  // times 3072: 3 * 2^22
                bound[d] += 2 * int64_t(K) * (dig[d] < 0 ? -dig[d] : dig[d]);
                if (bound[d] >= (int64_t(1) << 22)) return {};
            }
            uint64_t radix = 0;
            for (int d = 0; d < D; d++) radix += uint64_t(1) << (10 * d);
            const uint64_t magic = 0x4B400000ull;  // bits of the float 3 * 2^22
            uint64_t *o = img.data() + lay.tgt + (size_t(b) * kMmaSlots + j) * kMmaTgtWords;
            o[0] = c0 + p + magic * p - magic * radix;  // mod 2^64
            o[1] = 0 - p;
            const double big = 12582912.0, pd = double(p);
            const double ct = ldexp(1.0, 10 * (D - 1)) / pd, cm = ldexp(1.0, 10 * (D - 2)) / pd,
                         cl = ldexp(1.0, 10 * (D - 3)) / pd;
            const float f[4] = {float(ct), float(cm), float(cl),
                                float(double(c0) / pd - big * (double(float(cm)) + double(float(cl))))};
            memcpy(o + 2, f, 16);
            o[4] = s.dst_off[t] * target_unit;
        }
    }
    return img;
}

// Whether the tensor-core form takes less time than the split-weight one, by
// a model in cycles per warp of 32 coefficients: the integer kernel's multiply
// pipe (12 a product, 24 a Montgomery reduction, 70% busy; mixed
// source counts run one coefficient per thread, about a third slower) against
// the other's issue slots (half busy) and its start (matrix, TMEM) of about
// 2000.  A launch below two warps per scheduler (four per SM) takes as long as two.
// Measured on GB300, us (integer / tensor): 8 sources, 20 targets, 3 x 4 x
// 2^16 coefficients 103 / 59; 5 sources, 23 targets, 2^19 57 / 37; a whole
// product at N = 2^12, 24 primes (8 and 5 sources) 43.0 / 38.9; at 3 primes (3
// and 5 sources) 29.1 / 31.6, and at N = 2^16 57.2 / 59.9.
// The layouts without split weights are slower than both: with 9 special
// primes (9 sources, 10 when fused) a product of one ciphertext at N = 2^12 takes 35.8 /
// 32.3 us at 8 limbs and 52.3 / 39.2 at 24, at 2^15 64.5 / 58.8 and 149 / 129 (at 2
// and 5 limbs of 2^12 the host's time decides, 33-34 either way).
// beside: the other half of the operation runs at the same time.  To up to four
// targets little of the integer kernel's time is multiplications, and the
// tensor-core kernel's shared memory and TMEM keep the other half's CTAs out:
// products at 8 limbs with 4 special primes (8 sources, 4 targets) 229 / 239 us
// for 11 ciphertexts at N = 2^15, 260 / 270 for 6 at 2^16, a rotation of 4 169 /
// 177, so they need six times the gain (4 limbs, 8 special primes, 16
// ciphertexts at 2^16, 679 / 663, have it; alone, 3 ciphertexts of 8 limbs at
// 2^16 are 168 / 165).
bool mma_is_faster(const ConvPlans &cp, size_t coeffs, int sms, bool beside) {
    if (!cp.l.split) return true;
    double gain = 0, most = 0;
    for (uint32_t i = 0; i < cp.m.n; i++) {
        const double K = double(cp.m.head[i] & 0xff), T = double(mma_targets(cp.m.counts[i]));
        const double pair = (6 * K * (K + 1) + 24 * K + T * (12 * K + 24)) / 0.7;
        gain += (cp.l.kmin == cp.l.kmax ? 1.0 : 1.3) * pair - (40 * K + 30 * T + 150) / 0.48;
        most = std::max(most, T);
    }
    const double warps = std::max(2.0, double(coeffs) * cp.m.n / 32 / (4.0 * sms));
    return gain / cp.m.n * warps > (beside && most <= 4 ? 12000 : 2000);
}

}  // namespace catfhe
