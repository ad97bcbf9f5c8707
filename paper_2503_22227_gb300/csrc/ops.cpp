// Scheme operations: key generation, encryption, decryption, and the hot
// path (tensor -> ModUp -> inner product -> ModDown [-> rescale]), as
// sequences of batched kernel launches on one stream.
//
// Every step follows the definitions the CPU oracle computes (hybrid key
// switching with exact centred lifts; ModDown round(x / P), or
// (x - t [x t^-1]_P) / P for BGV; CKKS rescale round(c / q_{l-1}); BFV
// multiplication by exact round(t x / Q) over an auxiliary basis).
#include <string.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "internal.h"
#include "lanes.h"

namespace catfhe {


#define TRY(x)                      \
    do {                            \
        int rc_ = (x);              \
        if (rc_ != CATFHE_OK) return rc_; \
    } while (0)

// ----------------------------------------------------------------- workspace

struct Bump {
    char *base;
    size_t off = 0;
    template <class T>
    T *take(size_t count) {
        off = (off + 255) & ~size_t(255);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += count * sizeof(T);
        return p;
    }
};

static bool overlap(const void *a, size_t a_bytes, const void *b, size_t b_bytes) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + b_bytes && y < x + a_bytes;
}

static int get_ws(Context &c, void *ws, size_t ws_bytes, size_t need, char **out) {
    if (ws) {
        // kernels access the workspace in 8- and 16-byte words (and bulk
        // copies need 16-byte alignment): refuse a pointer that is not
        if (reinterpret_cast<uintptr_t>(ws) & 15) return CATFHE_EINVAL;
        if (ws_bytes < need) return CATFHE_EWORKSPACE;
        *out = static_cast<char *>(ws);
        return CATFHE_OK;
    }
    if (c.scratch.bytes < need) {
        cudaFree(c.scratch.ptr);
        c.scratch.ptr = nullptr;
        c.scratch.bytes = 0;
        if (cudaMalloc(&c.scratch.ptr, need) != cudaSuccess) return CATFHE_ENOMEM;
        c.scratch.bytes = need;
    }
    *out = static_cast<char *>(c.scratch.ptr);
    return CATFHE_OK;
}

// One launch's plans, all in one form: Montgomery when every plan fits it
// (with split weights when every plan fits those too), else exact; and the
// tensor-core form beside it when every plan has one and some plan has more
// than one source.  launch_conv chooses between the two.
static int make_list(Context &c, const std::vector<std::pair<std::string, PlanSpec>> &specs,
                     ConvPlans &cp) {
    bool all = true, all_split = true;
    for (const auto &s : specs) {
        all = all && plan_fits_mont(s.second);
        all_split = all_split && plan_fits_split(s.second);
    }
    PlanList &pl = cp.l;
    MmaList &ml = cp.m;
    pl.n = ml.n = uint32_t(specs.size());
    pl.mont = all ? 1 : 0;
    for (const auto &s : specs) cp.mma = cp.mma || s.second.src_mod.size() > 1;
    cp.mma = cp.mma && specs.size() <= kMmaPlans;
    for (size_t i = 0; i < specs.size() && cp.mma; i++) {
        const MmaRef r = get_mma_plan(c, specs[i].first, specs[i].second, c.n);
        ml.img[i] = r.p;
        ml.head[i] = r.head;
        ml.counts[i] = r.counts;
        cp.mma = r.p != nullptr;
        if (cp.mma) ml.p[i] = get_plan(c, specs[i].first, specs[i].second).p;
        if (cp.mma && !ml.p[i]) return CATFHE_ENOMEM;
    }
    pl.split = all && all_split ? 1 : 0;
    for (size_t i = 0; i < specs.size(); i++) {
        PlanSpec sp = specs[i].second;
        sp.exact = !all;
        sp.split = pl.split != 0;
        const PlanRef r = get_plan(c, specs[i].first, sp);
        if (!r.p) return CATFHE_ENOMEM;
        if (r.mont != (pl.mont != 0) || r.split != (pl.split != 0)) return CATFHE_EINVAL;
        pl.p[i] = r.p;
        pl.kmax = std::max<uint32_t>(pl.kmax, uint32_t(sp.src_mod.size()));
        pl.kmin = i == 0 ? uint32_t(sp.src_mod.size())
                         : std::min<uint32_t>(pl.kmin, uint32_t(sp.src_mod.size()));
        pl.words = std::max(pl.words, r.words);
    }
    return CATFHE_OK;
}

// The entries of a ModDown or rescale by the one prime at index `from`, for
// both polynomials' targets q_0 .. q_{lo-1}; `inv` is the map of the inverse
// transform of its limbs, which for BGV brings the factor t^-1 (the lift took a
// Shoup product per word and target for it: 16 products at N = 2^14 315.7 -> 309.2
// us).
static std::vector<LiftEntry> division_lifts(const Context &c, int from, int lo, LimbMap &inv) {
    const uint64_t m = c.mod(from);
    const bool bgv = c.scheme == CATFHE_BGV;
    inv.mods_off = bgv ? uint32_t(c.hmods.size()) : 0;
    std::vector<LiftEntry> t;
    for (int p = 0; p < 2; p++)
        for (int i = 0; i < lo; i++)
            t.push_back(lift_entry(m, c.mod(i), bgv ? c.t : 1));
    return t;
}

static LimbMap map_identity(uint32_t limbs, uint32_t first_prime = 0) {
    LimbMap m{};
    m.period = limbs;
    m.src_stride = m.dst_stride = limbs;
    for (uint32_t i = 0; i < limbs; i++) {
        m.src_off[i] = m.dst_off[i] = uint16_t(i);
        m.prime[i] = uint8_t(first_prime + i);
    }
    return m;
}

static uint64_t prod_mod(const Context &c, int from, int to, uint64_t m) {
    uint64_t r = 1 % m;
    for (int i = from; i < to; i++) r = h_mulmod(r, c.mod(i) % m, m);
    return r;
}

// The inverse of an odd g modulo a power of two (Newton iteration).
static uint64_t inv_mod_pow2(uint64_t g, uint64_t two_n) {
    uint64_t x = g;
    for (int i = 0; i < 6; i++) x *= 2 - g * x;
    return x & (two_n - 1);
}

// P = prod p_k mod m
static uint64_t pmod(const Context &c, uint64_t m) { return prod_mod(c, c.L, c.L + c.K, m); }

// ----------------------------------------------------------------- key switching pieces

// Global prime index of extended position i at level l (Q_l then P).
static int ext_prime(const Context &c, int level, int i) { return i < level ? i : c.L + (i - level); }

// Whether the lifted digits' forward NTT may leave its words unreduced: the
// inner product is their only reader and reduces its sums once (Montgomery,
// valid below 2^64 q); with words below 68q from an unreduced transform, its
// beta products and the folded P d term stay below (68 beta + 1) q^2.  Used
// when that bound holds for every prime below 2^57 of Q_l u P (larger
// primes are reduced anyway).
static bool ext_lazy(const Context &c, int level) {
    const int beta = (level + c.alpha - 1) / c.alpha;
    for (int i = 0; i < level + c.K; i++) {
        const uint64_t q = c.mod(ext_prime(c, level, i));
        if (q < (uint64_t(1) << 57) &&
            (unsigned __int128)(kWideWordsQ * uint64_t(beta) + 1) * q >=
                ((unsigned __int128)1 << 64))
            return false;
    }
    return true;
}

// Everything of a key switching at one level (fused: with the rescale) that does
// not depend on the call: limb maps, conversion plans, launch arguments with
// their constants.  Built on first use and kept by the context; a call copies
// the arguments and fills in its pointers.  (Computing them anew, inverses
// included, took 10 to 20 us of host time per call, as long as the device
// needs at the smallest sizes.)
struct KsConsts {
    // ModUp and the NTT of the lifted limbs (all positions for BFV)
    ConvPlans up;
    const LiftEntry *up_lifts = nullptr;  // digits of one prime: lifted by the transform
    LimbMap ext{};
    bool lazy = false;
    IpArgs ip{};
    // ModDown by P (fused: P q_{l-1})
    LimbMap special{};  // the division basis' limbs of y
    ConvPlans down;
    const LiftEntry *down_lifts = nullptr;  // division by one prime
    LimbMap lift{};                         // NTT schemes: the lift's transform
    NttEpilogue epi{};
    CombineArgs comb{};                     // BFV
};

static int build_modup(Context &c, int level, KsConsts &k) {
    const int M = level + c.K, beta = (level + c.alpha - 1) / c.alpha;
    const bool own_too = c.scheme == CATFHE_BFV, one = c.alpha == 1;
    LimbMap &m = k.ext;
    std::vector<std::pair<std::string, PlanSpec>> specs;
    std::vector<LiftEntry> lifts;
    uint32_t e = 0;
    for (int j = 0; j < beta; j++) {
        const int lo = j * c.alpha, hi = std::min((j + 1) * c.alpha, level);
        PlanSpec sp;
        sp.lazy = true;  // the lifted limbs go straight into an NTT
        for (int i = lo; i < hi; i++) {
            sp.src_mod.push_back(c.mod(i));
            sp.src_off.push_back(uint32_t(i));
        }
        for (int i = 0; i < M; i++) {
            if (!own_too && i >= lo && i < hi) continue;
            if (e >= uint32_t(kMapMax)) return CATFHE_EINVAL;
            const int p = ext_prime(c, level, i);
            m.dst_off[e] = uint16_t(j * M + i);
            m.src_off[e] = one ? uint16_t(j) : m.dst_off[e];
            m.prime[e] = uint8_t(p);
            e++;
            sp.dst_mod.push_back(c.mod(p));
            sp.dst_off.push_back(uint32_t(i));
            if (one) lifts.push_back(lift_entry(c.mod(j), c.mod(p), 1));
        }
        specs.emplace_back("modup/" + std::to_string(level) + "/" + std::to_string(j), sp);
    }
    m.period = e;
    m.src_stride = m.dst_stride = uint32_t(beta * M);
    k.lazy = ext_lazy(c, level);
    if (!one) return make_list(c, specs, k.up);
    k.up_lifts = upload_lifts(c, lifts);
    return k.up_lifts ? CATFHE_OK : CATFHE_ENOMEM;
}

static void build_ip(const Context &c, int level, IpArgs &a) {
    const int M = level + c.K, beta = (level + c.alpha - 1) / c.alpha;
    a.ext_item = size_t(beta) * M * c.n;
    a.y_item = size_t(2) * M * c.n;
    a.M = M;
    a.level = level;
    a.beta = beta;
    a.L = c.L;
    a.K = c.K;
    a.alpha = c.alpha;
    a.status = c.d_status;
    for (int i = 0; i < M; i++) {
        const int gp = ext_prime(c, level, i);
        a.prime[i] = uint8_t(gp);
        a.key_limb[i] = uint16_t(gp);
        if (i < level) {
            const uint64_t q = c.mod(i), r = (uint64_t)(((unsigned __int128)1 << 64) % q);
            a.pfac[i] = h_mulmod(pmod(c, q), r, q);  // P in Montgomery form
        }
    }
}

static int build_moddown(Context &c, int level, bool fused, KsConsts &k) {
    const int M = level + c.K, lo = fused ? level - 1 : level;
    const size_t n = c.n;
    const bool ntt_form = c.scheme != CATFHE_BFV;
    // division basis positions in y: P, then q_{l-1} when fused
    std::vector<int> dpos;
    for (int i = 0; i < c.K; i++) dpos.push_back(level + i);
    if (fused) dpos.push_back(level - 1);
    const int Kd = int(dpos.size());
    LimbMap &m = k.special;
    m.period = uint32_t(2 * Kd);
    m.src_stride = m.dst_stride = uint32_t(2 * M);
    for (int p = 0; p < 2; p++)
        for (int d = 0; d < Kd; d++) {
            m.src_off[p * Kd + d] = m.dst_off[p * Kd + d] = uint16_t(p * M + dpos[d]);
            m.prime[p * Kd + d] = uint8_t(ext_prime(c, level, dpos[d]));
        }
    if (Kd == 1) {  // lifted by the next kernel as it loads
        k.down_lifts = upload_lifts(c, division_lifts(c, ext_prime(c, level, dpos[0]), lo, m));
        if (!k.down_lifts) return CATFHE_ENOMEM;
    } else {
        PlanSpec sp;
        sp.lazy = ntt_form;  // NTT schemes transform the lift before the combine
        for (int d = 0; d < Kd; d++) {
            sp.src_mod.push_back(c.mod(ext_prime(c, level, dpos[d])));
            sp.src_off.push_back(uint32_t(dpos[d]));
        }
        for (int i = 0; i < lo; i++) {
            sp.dst_mod.push_back(c.mod(i));
            sp.dst_off.push_back(uint32_t(i));
        }
        if (c.scheme == CATFHE_BGV) {
            for (int d = 0; d < Kd; d++)
                sp.pre.push_back(h_invmod(c.t % sp.src_mod[d], sp.src_mod[d]));
            for (int i = 0; i < lo; i++) sp.post.push_back(c.t % c.mod(i));
        }
        TRY(make_list(c, {{"moddown/" + std::to_string(level) + (fused ? "/f" : ""), sp}}, k.down));
    }
    // D^-1 mod q_i, D = P (fused: P q_{l-1})
    LimbMap &l = k.lift;
    NttEpilogue &e = k.epi;
    CombineArgs &a = k.comb;
    l.period = l.dst_stride = uint32_t(2 * lo);
    l.src_stride = Kd == 1 ? uint32_t(2 * M) : uint32_t(2 * lo);
    e.status = c.d_status;
    e.y_stride = uint32_t(2 * M);
    e.out_stride = uint32_t(2 * lo);
    a.lifts = k.down_lifts;
    a.y_last = size_t(dpos[0]) * n;
    a.y_item = size_t(2) * M * n;
    a.y_poly = size_t(M) * n;
    a.lift_item = a.out_item = size_t(2) * lo * n;
    a.lift_poly = a.add_poly = a.out_poly = size_t(lo) * n;
    a.lo = uint32_t(lo);
    for (int i = 0; i < lo; i++) {
        const uint64_t q = c.mod(i);
        uint64_t D = pmod(c, q);
        if (fused) D = h_mulmod(D, c.mod(level - 1) % q, q);
        const uint64_t dinv = h_invmod(D, q), dinv_s = h_shoup(dinv, q);
        a.prime[i] = uint8_t(i);
        a.dinv[i] = dinv;
        a.dinv_s[i] = dinv_s;
        for (int p = 0; p < 2; p++) {
            const int r = p * lo + i;
            l.dst_off[r] = uint16_t(r);
            l.src_off[r] = Kd == 1 ? uint16_t(p * M + dpos[0]) : uint16_t(r);
            l.prime[r] = uint8_t(i);
            e.y_off[r] = uint16_t(p * M + i);
            e.out_off[r] = uint16_t(r);
            e.dinv[r] = dinv;
            e.dinv_s[r] = dinv_s;
        }
    }
    return CATFHE_OK;
}

// The entry `key` of a context's map of constants, built by make(entry) on
// first use; the context's lock covers the look-up and the building.
template <class T, class F>
static int kept(Context &c, std::map<int, std::shared_ptr<T>> &map, int key, const T **out, F make) {
    std::lock_guard<std::mutex> lock(c.mu);
    auto it = map.find(key);
    if (it == map.end()) {
        auto t = std::make_shared<T>();
        TRY(make(*t));
        it = map.emplace(key, t).first;
    }
    *out = it->second.get();
    return CATFHE_OK;
}

static int ks_consts(Context &c, int level, bool fused, const KsConsts **out) {
    return kept(c, c.ks, 2 * level + (fused ? 1 : 0), out, [&](KsConsts &k) -> int {
        TRY(build_modup(c, level, k));
        build_ip(c, level, k.ip);
        return build_moddown(c, level, fused, k);
    });
}

// ModUp of d2 (coefficient form, [level][N] per ciphertext, d2_item words
// apart) into ext ([count][beta][M][N]) and the NTT of the lifted limbs.
// Digits of one prime are lifted by the transform's first pass as it loads;
// wider ones are converted first.
static int modup_ntt(Context &c, const KsConsts &k, const uint64_t *d2c, size_t d2_item,
                     uint64_t *ext, uint32_t count, cudaStream_t s, bool beside) {
    const size_t n = c.n;
    if (k.up_lifts) {
        LimbMap m = k.ext;
        m.src_stride = uint32_t(d2_item / n);
        return launch_ntt_lift(c, d2c, ext, m, m.period * count, k.up_lifts, k.lazy, s);
    }
    TRY(launch_conv(c, k.up, d2c, d2_item, 0, ext, k.ip.ext_item, size_t(k.ip.M) * n, count, s,
                    beside));
    return k.lazy ? launch_ntt_fwd_lazy(c, ext, ext, k.ext, k.ext.period * count, s)
                  : launch_ntt_fwd(c, ext, ext, k.ext, k.ext.period * count, s);
}

// own, add0, add1: one limb group of `level` limbs per ciphertext, in_item
// words apart (null: none).
static IpArgs ip_args(const KsConsts &k, const uint64_t *ext, const uint64_t *own,
                      const uint64_t *key, const uint64_t *add0, const uint64_t *add1,
                      size_t in_item, uint64_t *y) {
    IpArgs a = k.ip;
    a.ext = ext;
    a.own = own;
    a.key = key;
    a.add0 = add0;
    a.add1 = add1;
    a.y = y;
    a.own_item = a.add_item = in_item;
    return a;
}

// gth (rotations): ciphertext i's add0 and own are the two polynomials of
// gth->a[i].  key2: a second key, its result in y2.
static int inner_product(Context &c, const KsConsts &k, const uint64_t *ext, const uint64_t *own,
                         const uint64_t *key, const uint64_t *add0, const uint64_t *add1,
                         size_t in_item, uint64_t *y, uint32_t count, cudaStream_t s,
                         const Gather *gth = nullptr, const uint64_t *key2 = nullptr,
                         uint64_t *y2 = nullptr) {
    IpArgs a = ip_args(k, ext, own, key, add0, add1, in_item, y);
    a.key2 = key2;
    a.y2 = y2;
    if (gth && gth->n) {
        a.gathered = 1;
        for (uint32_t i = 0; i < gth->n; i++) a.ga[i] = gth->a[i];
    }
    return launch_ip(c, a, count, s);
}

// ModDown of y ([count][2][M][N]; NTT form for CKKS/BGV, coefficient form
// for BFV) into out ([count][2][lo][N]).
// add (BFV): [.][lo][N] added to the first add_polys polynomials, add_item
// words per ciphertext.  g: sigma_g applied to the result (0: none).
static int moddown(Context &c, const KsConsts &k, uint64_t *y, uint64_t *lift, uint64_t *out,
                   uint32_t count, cudaStream_t s, bool beside, uint64_t g = 0, const Gather *gth = nullptr,
                   const uint64_t *add = nullptr, uint32_t add_polys = 0, size_t add_item = 0) {
    const bool ntt_form = c.scheme != CATFHE_BFV;
    if (gth && gth->n && (!ntt_form || add || gth->n != count)) return CATFHE_EINVAL;
    if (ntt_form) TRY(launch_ntt_inv(c, y, y, k.special, k.special.period * count, s));
    if (!k.down_lifts)
        TRY(launch_conv(c, k.down, y, size_t(k.ip.M) * c.n, 0, lift, k.comb.lift_poly, 0, 2 * count,
                        s, beside));
    if (ntt_form) {
        // NTT of the lift whose last pass writes (y - lift) D^-1 straight to out
        NttEpilogue e = k.epi;
        e.y = y;
        e.out = out;
        e.galois = uint32_t(g);
        e.galois_inv = g ? uint32_t(inv_mod_pow2(g, 2 * c.n)) : 0;
        if (gth && gth->n) {
            e.gathered = 1;
            for (uint32_t i = 0; i < gth->n; i++) e.gout[i] = gth->out[i];
        }
        const uint32_t limbs = k.lift.period * count;
        return k.down_lifts
                   ? launch_ntt_lift_combine(c, y, lift, k.lift, limbs, k.down_lifts, e, s)
                   : launch_ntt_fwd_combine(c, lift, k.lift, limbs, e, s);
    }
    CombineArgs a = k.comb;
    a.y = y;
    a.lift = k.down_lifts ? nullptr : lift;
    a.add = add;
    a.add_polys = add_polys;
    a.add_item = add_item;
    a.galois = uint32_t(g);
    a.out = out;
    return launch_combine(c, a, count, s);
}

// ----------------------------------------------------------------- op layouts

struct KsBufs {
    uint64_t *d0, *d1, *d2, *d2c, *ext, *y, *lift;
    // BFV
    uint64_t *xin, *tens, *dq, *add;
};

static void ks_layout(const Context &c, Bump &b, KsBufs &k, uint32_t count, int level,
                      bool fused) {
    const size_t n = c.n;
    const int M = level + c.K, beta = (level + c.alpha - 1) / c.alpha;
    const int lo = fused ? level - 1 : level;
    k.d0 = b.take<uint64_t>(size_t(count) * level * n);
    k.d1 = b.take<uint64_t>(size_t(count) * level * n);
    k.d2 = b.take<uint64_t>(size_t(count) * level * n);
    k.d2c = b.take<uint64_t>(size_t(count) * level * n);
    k.ext = b.take<uint64_t>(size_t(count) * beta * M * n);
    k.y = b.take<uint64_t>(size_t(count) * 2 * M * n);
    k.lift = b.take<uint64_t>(size_t(count) * 2 * lo * n);
    k.xin = k.tens = k.dq = k.add = nullptr;
    if (c.scheme == CATFHE_BFV) {
        const int kb = level + c.nb;
        k.xin = b.take<uint64_t>(size_t(count) * 4 * kb * n);
        k.tens = b.take<uint64_t>(size_t(count) * 3 * kb * n);
        k.dq = b.take<uint64_t>(size_t(count) * 3 * level * n);
        k.add = b.take<uint64_t>(size_t(count) * 2 * level * n);
    }
}

static size_t ks_bytes(const Context &c, uint32_t count, int level, bool fused) {
    Bump b{nullptr};
    KsBufs k{};
    ks_layout(c, b, k, count, level, fused);
    return (b.off + 255) & ~size_t(255);
}

// Key-switching operations on at least kSplitMin ciphertexts of N >= 2^14
// run as two halves on two streams forked from the caller's stream: one
// half's memory-bound kernels overlap the other's integer-bound ones
// (measured on the batch of 8 at N = 2^16, l = 24: 1596 -> 1526 us).  Their
// workspace holds both halves.
constexpr uint32_t kSplitMin = 4;
static bool split_ok(const Context &c, uint32_t count) { return count >= kSplitMin && c.log_n >= 14; }

static size_t ks_ws(const Context &c, uint32_t count, int level, bool fused) {
    const size_t whole = ks_bytes(c, count, level, fused);
    if (!split_ok(c, count)) return whole;
    const uint32_t c0 = (count + 1) / 2;
    return std::max(whole, ks_bytes(c, c0, level, fused) + ks_bytes(c, count - c0, level, fused));
}

size_t ws_bytes(const Context &c, int op, uint32_t level, uint32_t count) {
    Bump b{nullptr};
    const size_t n = c.n;
    switch (op) {
        case CATFHE_OP_MUL_RELIN:
        case CATFHE_OP_ROTATE:
            b.off = ks_ws(c, count, int(level), false);
            break;
        case CATFHE_OP_MUL_RELIN_RESCALE:
            b.off = ks_ws(c, count, int(level), true);
            break;
        case CATFHE_OP_ROTATE_HOISTED: {
            // two per-rotation buffer sets (rotations alternate over two
            // streams), then the shared lifted digits
            b.off = 2 * ks_bytes(c, count, int(level), false);
            const int M = int(level) + c.K, beta = (int(level) + c.alpha - 1) / c.alpha;
            b.take<uint64_t>(size_t(count) * beta * M * n);
            break;
        }
        case CATFHE_OP_RESCALE:
            b.take<uint64_t>(size_t(count) * 2 * n);
            b.take<uint64_t>(size_t(count) * 2 * (level ? level - 1 : 0) * n);
            break;
        case CATFHE_OP_DECRYPT:
            b.take<uint64_t>(size_t(level) * n);
            b.take<uint64_t>(size_t(level) * n);
            b.take<int64_t>(n);
            break;
        case CATFHE_OP_EXPORT:
            b.take<uint64_t>(size_t(count) * 2 * level * n);
            break;
        case CATFHE_OP_ENCODE:
            b.take<double2>(n / 2);
            b.take<double2>(2 * n);
            b.take<int64_t>(n);
            break;
        case CATFHE_OP_DECODE:
            b.take<uint64_t>(size_t(2) * level * n);
            b.take<int64_t>(n);
            b.take<double2>(2 * n);
            b.take<double2>(n / 2);
            break;
        default:
            return 0;
    }
    return b.off + 256;
}

// ----------------------------------------------------------------- hot path

static int key_for(const Keys &k, uint64_t id, const uint64_t **key) {
    auto it = k.ksk.find(id);
    if (it == k.ksk.end()) return CATFHE_ENOKEY;
    *key = it->second;
    return CATFHE_OK;
}

// The map of the a1 polynomials of ciphertexts [2][lvl][N]: limb lvl + i of
// each group into limb i of a buffer of lvl limbs per group.
static LimbMap map_second(int lvl) {
    LimbMap m{};
    m.period = uint32_t(lvl);
    m.src_stride = uint32_t(2 * lvl);
    m.dst_stride = uint32_t(lvl);
    for (int i = 0; i < lvl; i++) {
        m.src_off[i] = uint16_t(lvl + i);
        m.dst_off[i] = uint16_t(i);
        m.prime[i] = uint8_t(i);
    }
    return m;
}

// Whether a multiplication of `count` ciphertexts has no tensor kernel: the
// inverse transform and the inner product then form the products, which saves a
// launch and 5 passes over them but forms a1 b1 twice, and one CTA of the
// inner product forms those of its ciphertexts one after another.
// beside: other operations or another half run at the same time.
//
// The launch is what counts while the key switching is short, however the words
// are spread over ciphertexts: up to kProductWork words of lifted digits and
// sums ((digits + 2) (l + K) N per ciphertext).  us with the tensor kernel ->
// without: N = 2^12, 3 limbs, 1 digit 36.1 -> 33.0, 8 of them 36.5 -> 34.3, 8
// limbs x 2 36.9 -> 33.3; halves at 2^14, 3 limbs x 4 61.7 -> 57.6, BGV 2 limbs x
// 8 55.4 -> 49.9.  At the line both routes are level (2^12, 12 limbs x 4 41.1 ->
// 41.1; 2^14, 3 limbs x 3 44.6 -> 44.3); past it the products weigh more, 2^12,
// 2 limbs x 16 41.3 -> 44.0, 2^14, 2 limbs x 16 92.6 -> 96.7, 9 limbs x 5 97.3 ->
// 105.2, 2^15, 2 limbs x 4 67.7 -> 71.9, 2^16, 2 limbs x 8 167.0 -> 175.1.
// Up to kProductFew ciphertexts with nothing beside them keep the route to
// kProductWords words, where the kernels wait for their loads more than for
// multiplications: 2^14, 16 limbs x 2 75.3 -> 73.7, 24 limbs 74.0 -> 72.5, BGV 8
// limbs x 3 84.7 -> 83.5, 2^15, 16 limbs 79.4 -> 77.9, 2^16, 4 limbs 60.4 -> 58.8,
// 8 limbs 81.9 -> 79.2, with 8 special primes 7 limbs 91.2 -> 89.2 (and 2^14, 9
// limbs x 2 55.1 -> 56.0; one ciphertext at 2^16, 24 limbs is level, 198.0).  Below
// kProductLimbs limbs few of the inner product's CTAs have a product to form and
// the others wait for them: 2^16, 3 limbs 54.9 -> 56.0, 2^15, 2 limbs x 2 48.8 ->
// 50.2, so these stay with the tensor kernel.
// A batch on lanes: 8 operations 271.3 with it, 273.8 without, 16 463 and 472.
constexpr size_t kProductWork = size_t(1) << 20, kProductWords = size_t(1) << 19;
constexpr uint32_t kProductFew = 3, kProductLimbs = 4;
static bool forms_products(const Context &c, const IpArgs &ip, uint32_t level, uint32_t count,
                           bool beside) {
    if (ip.beta > kIpBulkBeta) return false;
    if (size_t(count) * (ip.beta + 2) * ip.M * c.n <= kProductWork) return true;
    return !beside && count <= kProductFew && level >= kProductLimbs &&
           size_t(count) * level * c.n <= kProductWords;
}

// CKKS / BGV: tensor in NTT form, INTT d2, ModUp, NTT, inner product with
// P*(d0, d1) folded in, ModDown (fused: by P q_{l-1}).
static int mul_relin_ntt(Context &c, const Keys &keys, const uint64_t *a, const uint64_t *b,
                         uint64_t *out, uint32_t count, int level, bool fused, KsBufs &k,
                         cudaStream_t s, const Gather *gth, bool other_half) {
    const uint64_t *rlk;
    TRY(key_for(keys, 0, &rlk));
    const KsConsts *ks;
    TRY(ks_consts(c, level, fused, &ks));
    const size_t n = c.n, half = size_t(level) * n, item = 2 * half;
    const bool gathered = gth && gth->n;
    if (forms_products(c, ks->ip, uint32_t(level), count, other_half || LaneScope::active())) {
        // no tensor kernel: the inverse transform forms a1 b1 as it loads, and
        // the inner product the three products of its own tile
        LimbMap m = map_second(level);
        NttFactor f{};
        f.b = b;
        if (gathered) {
            m.gathered = 1;
            for (uint32_t i = 0; i < gth->n; i++) {
                m.gsrc[i] = gth->a[i];
                f.gb[i] = gth->b[i];
            }
        }
        TRY(launch_ntt_inv(c, a, k.d2c, m, uint32_t(level) * count, s, &f));
        TRY(modup_ntt(c, *ks, k.d2c, half, k.ext, count, s, other_half));
        IpArgs ip = ip_args(*ks, k.ext, a + half, rlk, a, nullptr, item, k.y);
        ip.product = 1;
        ip.b = b;
        if (gathered) {
            ip.gathered = 1;
            for (uint32_t i = 0; i < gth->n; i++) {
                ip.ga[i] = gth->a[i];
                ip.gb[i] = gth->b[i];
            }
        }
        TRY(launch_ip(c, ip, count, s));
        return moddown(c, *ks, k.y, k.lift, out, count, s, other_half, 0, gth);
    }
    TensorArgs t{};
    t.a = a;
    t.b = b;
    if (gathered) {
        t.gathered = 1;
        for (uint32_t i = 0; i < gth->n; i++) {
            t.ga[i] = gth->a[i];
            t.gb[i] = gth->b[i];
        }
    }
    t.d0 = k.d0;
    t.d1 = k.d1;
    t.d2 = k.d2;
    t.in_item = item;
    t.out_item = half;
    t.limbs = uint32_t(level);
    for (int i = 0; i < level; i++) t.prime[i] = uint8_t(i);
    TRY(launch_tensor(c, t, count, s));
    LimbMap m = map_identity(uint32_t(level));
    TRY(launch_ntt_inv(c, k.d2, k.d2c, m, uint32_t(level) * count, s));
    TRY(modup_ntt(c, *ks, k.d2c, half, k.ext, count, s, other_half));
    TRY(inner_product(c, *ks, k.ext, k.d2, rlk, k.d0, k.d1, half, k.y, count, s));
    return moddown(c, *ks, k.y, k.lift, out, count, s, other_half, 0, gth);
}

// A BFV multiplication's constants at one level, kept like KsConsts.
struct BfvConsts {
    ConvPlans lift;       // Q_l -> B
    LimbMap in{};         // an input's q limbs into xin
    LimbMap mb{}, mq{};   // the b limbs of Q u B; all of them
    PlanRef pa, pb, pe;   // scale-and-round: both plans, and the exact one of z
    MmaRef ma, mz;        // its tensor-core form
    bool mma = false;
};

static int build_bfv(Context &c, int level, BfvConsts &k) {
    const int kb = level + c.nb;
    LimbMap &mb = k.mb, &mq = k.mq;
    mb.period = uint32_t(c.nb);
    mq.period = uint32_t(kb);
    mb.src_stride = mb.dst_stride = mq.src_stride = mq.dst_stride = uint32_t(kb);
    for (int i = 0; i < kb; i++) {
        mq.src_off[i] = mq.dst_off[i] = uint16_t(i);
        mq.prime[i] = uint8_t(i < level ? i : c.pb(i - level));
        if (i < level) continue;
        mb.src_off[i - level] = mb.dst_off[i - level] = uint16_t(i);
        mb.prime[i - level] = mq.prime[i];
    }
    k.in = map_identity(uint32_t(level));
    k.in.dst_stride = uint32_t(kb);
    const std::string l = std::to_string(level);
    PlanSpec A, B, sp;
    std::vector<uint64_t> tq;
    sp.lazy = true;  // NTT'd before the tensor
    for (int i = 0; i < level; i++) {
        sp.src_mod.push_back(c.mod(i));
        sp.src_off.push_back(uint32_t(i));
        A.src_mod.push_back(c.mod(i));
        A.src_off.push_back(uint32_t(i));
        A.pre.push_back(c.t % c.mod(i));
        B.dst_mod.push_back(c.mod(i));
        B.dst_off.push_back(uint32_t(i));
    }
    PlanSpec Am = A, Bm = B, Be = B;
    for (int j = 0; j < c.nb; j++) {
        const uint64_t bj = c.mod(c.pb(j));
        const uint64_t qinv = h_invmod(prod_mod(c, 0, level, bj), bj);
        const uint64_t tqi = h_mulmod(c.t % bj, qinv, bj);
        sp.dst_mod.push_back(bj);
        sp.dst_off.push_back(uint32_t(level + j));
        A.dst_mod.push_back(bj);
        A.dst_off.push_back(uint32_t(level + j));
        A.post.push_back(qinv);
        tq.push_back(tqi);
        tq.push_back(h_shoup(tqi, bj));
        B.src_mod.push_back(bj);
        B.src_off.push_back(0);
        // the tensor-core form: A's results times (B/b_j)^-1 meet the digits of
        // B's conversion, whose sources are x_b times t Q^-1
        uint64_t rest = 1;  // B / b_j mod b_j
        for (int i = 0; i < c.nb; i++)
            if (i != j) rest = h_mulmod(rest, c.mod(c.pb(i)) % bj, bj);
        Am.dst_mod.push_back(bj);
        Am.dst_off.push_back(uint32_t(j));
        Am.post.push_back(h_mulmod(qinv, h_invmod(rest, bj), bj));
        Bm.src_mod.push_back(bj);
        Bm.src_off.push_back(uint32_t(level + j));
        Bm.pre.push_back(tqi);
        Be.src_mod.push_back(bj);
        Be.src_off.push_back(uint32_t(j));
        Be.pre.push_back(rest);
    }
    TRY(make_list(c, {{"bfv_lift/" + l, sp}}, k.lift));
    // the fused kernels need both conversions in the Montgomery layout
    if (!plan_fits_mont(A) || !plan_fits_mont(B)) return CATFHE_EINVAL;
    k.pa = get_plan_extra(c, "bfv_sr_a/" + l, A, tq);
    k.pb = get_plan(c, "bfv_sr_b/" + l, B);
    k.pe = get_plan(c, "bfv_sr_e/" + l, Be);
    if (!k.pa.p || !k.pb.p || !k.pe.p) return CATFHE_ENOMEM;
    k.ma = get_mma_plan(c, "bfv_sr_a/" + l, Am, 1);
    k.mz = get_mma_plan(c, "bfv_sr_b/" + l, Bm, c.n);
    k.mma = bfv_round_mma_fits(k.ma, k.mz);
    return CATFHE_OK;
}

// BFV: lift to Q u B, NTT, tensor, INTT, exact round(t x / Q) back to Q,
// then relinearise d2 in coefficient form.
static int mul_relin_bfv(Context &c, const Keys &keys, const uint64_t *a, const uint64_t *b,
                         uint64_t *out, uint32_t count, int level, KsBufs &k, cudaStream_t s,
                         bool other_half) {
    const uint64_t *rlk;
    TRY(key_for(keys, 0, &rlk));
    const KsConsts *ks;
    const BfvConsts *bc;
    TRY(ks_consts(c, level, false, &ks));
    TRY(kept(c, c.bfv, level, &bc, [&](BfvConsts &b) { return build_bfv(c, level, b); }));
    const size_t n = c.n;
    const int kb = level + c.nb;
    // 1. the 4 input polys over Q_l u B in NTT form: the q limbs transformed
    // straight from the inputs, the b limbs from their centred lift
    uint64_t *xb = k.xin + size_t(count) * 2 * kb * n;  // b's half of xin
    for (int h = 0; h < 2; h++) {  // items: (ct, poly) of a, then of b
        const uint64_t *src = h ? b : a;
        uint64_t *dst = h ? xb : k.xin;
        TRY(launch_conv(c, bc->lift, src, size_t(level) * n, 0, dst, size_t(kb) * n, 0, 2 * count, s,
                        other_half));
        TRY(launch_ntt_fwd(c, src, dst, bc->in, uint32_t(level) * 2 * count, s));
    }
    TRY(launch_ntt_fwd(c, k.xin, k.xin, bc->mb, uint32_t(c.nb) * 4 * count, s));
    // 2. tensor over Q u B
    {
        TensorArgs t{};
        t.a = k.xin;
        t.b = xb;
        t.in_item = size_t(2) * kb * n;
        t.d0 = k.tens;
        t.d1 = k.tens + size_t(kb) * n;
        t.d2 = k.tens + size_t(2) * kb * n;
        t.out_item = size_t(3) * kb * n;
        t.limbs = uint32_t(kb);
        for (int i = 0; i < kb; i++) t.prime[i] = bc->mq.prime[i];
        TRY(launch_tensor(c, t, count, s));
    }
    TRY(launch_ntt_inv(c, k.tens, k.tens, bc->mq, uint32_t(kb) * 3 * count, s));
    // 3. exact round(t x / Q) back to Q_l
    if (bc->mma)
        TRY(launch_bfv_round_mma(c, bc->ma, bc->pa.p, bc->mz, bc->pe.p, k.tens, size_t(kb) * n, k.dq,
                                 size_t(level) * n, 3 * count, s));
    else
        TRY(launch_bfv_scale_round(c, bc->pa.p, bc->pa.words, bc->pb.p, bc->pb.words, k.tens,
                                   size_t(kb) * n, k.dq, size_t(level) * n, 3 * count, s));
    // 4. relinearise d2' (coefficient form) and add (d0', d1')
    const uint64_t *d2 = k.dq + size_t(2) * level * n;
    TRY(modup_ntt(c, *ks, d2, size_t(3) * level * n, k.ext, count, s, other_half));
    TRY(inner_product(c, *ks, k.ext, nullptr, rlk, nullptr, nullptr, 0, k.y, count, s));
    {
        const int M = level + c.K;
        LimbMap my = map_identity(uint32_t(M));
        for (int i = 0; i < M; i++) my.prime[i] = uint8_t(ext_prime(c, level, i));
        TRY(launch_ntt_inv(c, k.y, k.y, my, uint32_t(2 * M) * count, s));
    }
    // (d0', d1') are the first two of each ciphertext's three polynomials
    return moddown(c, *ks, k.y, k.lift, out, count, s, other_half, 0, nullptr, k.dq, 2,
                   size_t(3) * level * n);
}

// Two streams (and fork / join events) per device for split operations;
// the mutex is held while a split operation is enqueued.
struct SplitPool {
    bool ready = false;
    cudaStream_t st[2];
    cudaEvent_t fork, join[2];
};
static std::mutex g_split_mu;
static SplitPool g_split[64];

static int split_pool(SplitPool **out) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return CATFHE_ECUDA;
    SplitPool &p = g_split[dev];
    if (!p.ready) {
        for (int i = 0; i < 2; i++) {
            if (cudaStreamCreateWithFlags(&p.st[i], cudaStreamNonBlocking) != cudaSuccess ||
                cudaEventCreateWithFlags(&p.join[i], cudaEventDisableTiming) != cudaSuccess)
                return CATFHE_ECUDA;
        }
        if (cudaEventCreateWithFlags(&p.fork, cudaEventDisableTiming) != cudaSuccess)
            return CATFHE_ECUDA;
        p.ready = true;
    }
    *out = &p;
    return CATFHE_OK;
}

// Runs f(first, cnt, ws_base, stream) for the two halves of `count` items on
// the split streams, ordered after everything enqueued on s so far and before
// everything enqueued on s afterwards.
template <class F>
static int run_halves(const Context &c, uint32_t count, int level, bool fused, char *base,
                      cudaStream_t s, F f) {
    std::lock_guard<std::mutex> lock(g_split_mu);
    SplitPool *sp;
    TRY(split_pool(&sp));
    const uint32_t c0 = (count + 1) / 2;
    const uint32_t first[2] = {0, c0}, cnt[2] = {c0, count - c0};
    char *wb[2] = {base, base + ks_bytes(c, c0, level, fused)};
    if (cudaEventRecord(sp->fork, s) != cudaSuccess) return CATFHE_ECUDA;
    for (int h = 0; h < 2; h++) {
        if (cudaStreamWaitEvent(sp->st[h], sp->fork, 0) != cudaSuccess) return CATFHE_ECUDA;
        TRY(f(first[h], cnt[h], wb[h], sp->st[h]));
        if (cudaEventRecord(sp->join[h], sp->st[h]) != cudaSuccess) return CATFHE_ECUDA;
        if (cudaStreamWaitEvent(s, sp->join[h], 0) != cudaSuccess) return CATFHE_ECUDA;
    }
    return CATFHE_OK;
}

int op_mul_relin(Context &c, const Keys &keys, const uint64_t *a, const uint64_t *b,
                 uint64_t *out, uint32_t level, uint32_t count, bool fused, void *ws,
                 size_t ws_bytes_in, cudaStream_t s, const Gather *gth, bool split) {
    if (gth && gth->n && (c.scheme == CATFHE_BFV || gth->n != count || count > kGatherMax))
        return CATFHE_EINVAL;
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (fused && (c.scheme != CATFHE_CKKS)) return CATFHE_ESCHEME;
    if (fused && level < 2) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    const size_t need = ws_bytes(c, fused ? CATFHE_OP_MUL_RELIN_RESCALE : CATFHE_OP_MUL_RELIN,
                                 level, count);
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, need, &base));
    const int lvl = int(level);
    // Fused results are a limb shorter than the inputs: written over an input,
    // the second half's lie in the first half's inputs, which that one may still
    // read, so the halves run as one.
    const size_t in_bytes = size_t(count) * 2 * lvl * c.n * 8;
    const size_t out_bytes = size_t(count) * 2 * (lvl - 1) * c.n * 8;
    const bool over = fused && (overlap(a, in_bytes, out, out_bytes) ||
                                overlap(b, in_bytes, out, out_bytes));
    const bool halves = split && !over && !(gth && gth->n) && split_ok(c, count);
    auto run = [&](uint32_t first, uint32_t cnt, char *wbase, cudaStream_t st) -> int {
        Bump bump{wbase};
        KsBufs k{};
        ks_layout(c, bump, k, cnt, lvl, fused);
        const size_t n = c.n, lo = size_t(fused ? lvl - 1 : lvl);
        const uint64_t *ah = a + size_t(first) * 2 * lvl * n, *bh = b + size_t(first) * 2 * lvl * n;
        uint64_t *oh = out + size_t(first) * 2 * lo * n;
        if (c.scheme == CATFHE_BFV) return mul_relin_bfv(c, keys, ah, bh, oh, cnt, lvl, k, st, halves);
        return mul_relin_ntt(c, keys, ah, bh, oh, cnt, lvl, fused, k, st, gth, halves);
    };
    if (halves) return run_halves(c, count, lvl, fused, base, s, run);
    return run(0, count, base, s);
}

// HRotate of count ciphertexts at lvl with the Galois key gk, workspace k.
// sigma_g commutes with every step of the key switching: it permutes slots
// (and signs of coefficients), the centred lifts are odd functions and no
// division has ties.  So sigma_g(a0) + KS_gk(sigma_g(a1)) =
// sigma_g(a0 + KS_gk'(a1)) with gk' = sigma_g^-1(gk), the stored form of the
// key, bit for bit; only the kernel that writes the result permutes.
static int rotate_run(Context &c, const uint64_t *gk, const uint64_t *a, uint64_t g, uint64_t *out,
                      int lvl, uint32_t count, KsBufs &k, cudaStream_t s, const Gather *gth,
                      bool other_half) {
    const size_t n = c.n, item = size_t(2) * lvl * n, half = size_t(lvl) * n;
    const KsConsts *ks;
    TRY(ks_consts(c, lvl, false, &ks));
    if (c.scheme != CATFHE_BFV) {
        LimbMap m = map_second(lvl);
        if (gth && gth->n) {
            m.gathered = 1;
            for (uint32_t i = 0; i < gth->n; i++) m.gsrc[i] = gth->a[i];
        }
        TRY(launch_ntt_inv(c, a, k.d2c, m, uint32_t(lvl) * count, s));
        TRY(modup_ntt(c, *ks, k.d2c, half, k.ext, count, s, other_half));
        TRY(inner_product(c, *ks, k.ext, a + half, gk, a, nullptr, item, k.y, count, s, gth));
        return moddown(c, *ks, k.y, k.lift, out, count, s, other_half, g, gth);
    }
    // BFV (coefficient form): a1 is key switched, a0 added by the combine.  It
    // scatters its results, so a0 is copied first when out overlaps a.
    const uint64_t *add = a;
    const size_t bytes = size_t(count) * item * 8;
    if (overlap(a, bytes, out, bytes)) {
        TRY(launch_copy_limbs(c, a, k.add, map_identity(uint32_t(2 * lvl)),
                              uint32_t(2 * lvl) * count, s));
        add = k.add;
    }
    TRY(modup_ntt(c, *ks, a + half, item, k.ext, count, s, other_half));
    TRY(inner_product(c, *ks, k.ext, nullptr, gk, nullptr, nullptr, 0, k.y, count, s));
    {
        const int M = lvl + c.K;
        LimbMap my = map_identity(uint32_t(M));
        for (int i = 0; i < M; i++) my.prime[i] = uint8_t(ext_prime(c, lvl, i));
        TRY(launch_ntt_inv(c, k.y, k.y, my, uint32_t(2 * M) * count, s));
    }
    return moddown(c, *ks, k.y, k.lift, out, count, s, other_half, g, nullptr, add, 1, item);
}

int op_rotate(Context &c, const Keys &keys, const uint64_t *a, uint64_t g, uint64_t *out,
              uint32_t level, uint32_t count, void *ws, size_t ws_bytes_in, cudaStream_t s,
              const Gather *gth, bool split) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (gth && gth->n && (c.scheme == CATFHE_BFV || gth->n != count || count > kGatherMax))
        return CATFHE_EINVAL;
    g %= 2 * c.n;
    if (!(g & 1)) return CATFHE_EINVAL;
    const uint64_t *gk;
    TRY(key_for(keys, g, &gk));
    if (count == 0) return CATFHE_OK;
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_ROTATE, level, count), &base));
    const size_t n = c.n;
    const int lvl = int(level);
    const bool halves = split && !(gth && gth->n) && split_ok(c, count);
    auto run = [&](uint32_t first, uint32_t cnt, char *wbase, cudaStream_t st) -> int {
        Bump bump{wbase};
        KsBufs k{};
        ks_layout(c, bump, k, cnt, lvl, false);
        const uint64_t *ah = a + size_t(first) * 2 * lvl * n;
        uint64_t *oh = out + size_t(first) * 2 * lvl * n;
        return rotate_run(c, gk, ah, g, oh, lvl, cnt, k, st, gth, halves);
    };
    if (halves) return run_halves(c, count, lvl, false, base, s, run);
    return run(0, count, base, s);
}


// Hoisted rotations: one INTT + ModUp + NTT of a1, then per Galois element the
// inner product with its (permuted) key and ModDown, which permutes the result.
int op_rotate_hoisted(Context &c, const Keys &keys, const uint64_t *a, const uint64_t *gs,
                      uint32_t n_rot, uint64_t *out, uint32_t level, uint32_t count, void *ws,
                      size_t ws_bytes_in, cudaStream_t s) {
    if (c.scheme == CATFHE_BFV) return CATFHE_ESCHEME;
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (n_rot > 0 && !gs) return CATFHE_EINVAL;
    std::vector<const uint64_t *> gk(n_rot);
    std::vector<uint64_t> gv(n_rot);
    for (uint32_t r = 0; r < n_rot; r++) {
        gv[r] = gs[r] % (2 * c.n);
        if (!(gv[r] & 1)) return CATFHE_EINVAL;
        TRY(key_for(keys, gv[r], &gk[r]));
    }
    if (count == 0 || n_rot == 0) return CATFHE_OK;
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_ROTATE_HOISTED, level, count), &base));
    Bump bump{base};
    KsBufs ks[2];
    ks_layout(c, bump, ks[0], count, int(level), false);
    bump.off = ks_bytes(c, count, int(level), false);
    ks_layout(c, bump, ks[1], count, int(level), false);
    bump.off = 2 * ks_bytes(c, count, int(level), false);
    KsBufs &k = ks[0];
    const size_t n = c.n;
    const int lvl = int(level), M = lvl + c.K, beta = (lvl + c.alpha - 1) / c.alpha;
    uint64_t *ext0 = bump.take<uint64_t>(size_t(count) * beta * M * n);
    // a1 (NTT form) -> coefficient form -> lifted digits in NTT form, once
    const size_t item = size_t(2) * lvl * n, half = size_t(lvl) * n;
    TRY(launch_ntt_inv(c, a, k.d2c, map_second(lvl), uint32_t(lvl) * count, s));
    const KsConsts *kc;
    TRY(ks_consts(c, lvl, false, &kc));
    TRY(modup_ntt(c, *kc, k.d2c, half, ext0, count, s, false));
    auto down = [&](uint32_t r, KsBufs &kb, uint64_t *y, cudaStream_t st) {
        return moddown(c, *kc, y, kb.lift, out + size_t(r) * count * item, count, st, false,
                       gv[r]);
    };
    auto one = [&](uint32_t r, KsBufs &kb, cudaStream_t st) -> int {
        TRY(inner_product(c, *kc, ext0, a + half, gk[r], a, nullptr, item, kb.y, count, st));
        return down(r, kb, kb.y, st);
    };
    // two rotations by one inner product, which reads the digits once; the
    // second result stands in the set's own digit buffer, which holds it from
    // two digits on and is otherwise unused (the workspace is as before)
    auto two = [&](uint32_t r, KsBufs &kb, cudaStream_t st) -> int {
        TRY(inner_product(c, *kc, ext0, a + half, gk[r], a, nullptr, item, kb.y, count, st, nullptr,
                          gk[r + 1], kb.ext));
        TRY(down(r, kb, kb.y, st));
        return down(r + 1, kb, kb.ext, st);
    };
    const bool pair = beta >= 2 && uint32_t(beta) <= kIpBulkBeta;
    if (n_rot < 2 || c.log_n < 14) {
        uint32_t r = 0;
        for (; pair && r + 1 < n_rot; r += 2) TRY(two(r, k, s));
        for (; r < n_rot; r++) TRY(one(r, k, s));
        return CATFHE_OK;
    }
    // rotations alternate over the two split streams, each with its own
    // buffer set (in order on its stream), after the shared ModUp on s; pairs
    // only while both streams have one, so that the rest still overlaps
    std::lock_guard<std::mutex> lock(g_split_mu);
    SplitPool *sp;
    TRY(split_pool(&sp));
    if (cudaEventRecord(sp->fork, s) != cudaSuccess) return CATFHE_ECUDA;
    for (int h = 0; h < 2; h++)
        if (cudaStreamWaitEvent(sp->st[h], sp->fork, 0) != cudaSuccess) return CATFHE_ECUDA;
    uint32_t r = 0;
    for (; pair && r + 4 <= n_rot; r += 4)
        for (int h = 0; h < 2; h++) TRY(two(r + 2 * h, ks[h], sp->st[h]));
    for (; r < n_rot; r++) TRY(one(r, ks[r & 1], sp->st[r & 1]));
    for (int h = 0; h < 2; h++) {
        if (cudaEventRecord(sp->join[h], sp->st[h]) != cudaSuccess) return CATFHE_ECUDA;
        if (cudaStreamWaitEvent(s, sp->join[h], 0) != cudaSuccess) return CATFHE_ECUDA;
    }
    return CATFHE_OK;
}

// A rescale's constants at one level, kept like KsConsts.
struct RescaleConsts {
    LimbMap last{}, lift{};
    NttEpilogue epi{};
    const LiftEntry *lifts = nullptr;
};

static int build_rescale(Context &c, int lvl, RescaleConsts &k) {
    const int lo = lvl - 1;
    LimbMap &m = k.last, &l = k.lift;
    NttEpilogue &e = k.epi;
    m.period = m.dst_stride = l.src_stride = 2;
    m.src_stride = e.y_stride = uint32_t(2 * lvl);
    l.period = l.dst_stride = e.out_stride = uint32_t(2 * lo);
    e.status = c.d_status;
    for (int p = 0; p < 2; p++) {
        m.src_off[p] = uint16_t(p * lvl + lvl - 1);
        m.dst_off[p] = uint16_t(p);
        m.prime[p] = uint8_t(lvl - 1);
        for (int i = 0; i < lo; i++) {
            const int r = p * lo + i;
            l.src_off[r] = uint16_t(p);
            l.dst_off[r] = uint16_t(r);
            l.prime[r] = uint8_t(i);
            e.y_off[r] = uint16_t(p * lvl + i);
            e.out_off[r] = uint16_t(r);
            e.dinv[r] = p ? e.dinv[i] : h_invmod(c.mod(lvl - 1) % c.mod(i), c.mod(i));
            e.dinv_s[r] = h_shoup(e.dinv[r], c.mod(i));
        }
    }
    k.lifts = upload_lifts(c, division_lifts(c, lvl - 1, lo, m));
    return k.lifts ? CATFHE_OK : CATFHE_ENOMEM;
}

// CKKS rescale / BGV modulus switch: divide by q_{l-1}.
int op_rescale(Context &c, const uint64_t *a, uint64_t *out, uint32_t level, uint32_t count,
               void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (c.scheme == CATFHE_BFV) return CATFHE_ESCHEME;
    if (level < 2 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_RESCALE, level, count), &base));
    Bump bump{base};
    const size_t n = c.n;
    const int lvl = int(level), lo = lvl - 1;
    uint64_t *last = bump.take<uint64_t>(size_t(count) * 2 * n);
    uint64_t *lift = bump.take<uint64_t>(size_t(count) * 2 * lo * n);
    const RescaleConsts *k;
    TRY(kept(c, c.rescale, lvl, &k, [&](RescaleConsts &r) { return build_rescale(c, lvl, r); }));
    // INTT of the last limb of both polys: [count][2][level] -> [count][2][1]
    TRY(launch_ntt_inv(c, a, last, k->last, 2 * count, s));
    // NTT of the lift (lifted as it loads), its last pass writing
    // (a - lift) q_{l-1}^-1 to out
    NttEpilogue e = k->epi;
    e.y = a;
    e.out = out;
    return launch_ntt_lift_combine(c, last, lift, k->lift, uint32_t(2 * lo) * count, k->lifts, e, s);
}

int op_add(Context &c, const uint64_t *a, const uint64_t *b, uint64_t *out, uint32_t level,
           uint32_t count, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    LimbMap m{};
    m.period = 2 * level;
    m.src_stride = m.dst_stride = 2 * level;
    for (uint32_t i = 0; i < 2 * level; i++) {
        m.src_off[i] = m.dst_off[i] = uint16_t(i);
        m.prime[i] = uint8_t(i % level);
    }
    return launch_add(c, a, b, out, m, 2 * level * count, s);
}

static LimbMap map_ct(uint32_t level) {
    LimbMap m{};
    m.period = 2 * level;
    m.src_stride = m.dst_stride = 2 * level;
    for (uint32_t i = 0; i < 2 * level; i++) {
        m.src_off[i] = m.dst_off[i] = uint16_t(i);
        m.prime[i] = uint8_t(i % level);
    }
    return m;
}

int op_sub(Context &c, const uint64_t *a, const uint64_t *b, uint64_t *out, uint32_t level,
           uint32_t count, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    return launch_sub(c, a, b, out, map_ct(level), 2 * level * count, s);
}

static uint64_t reduce_signed(int64_t v, uint64_t q) {
    const uint64_t mag = v < 0 ? uint64_t(0) - uint64_t(v) : uint64_t(v);
    const uint64_t r = mag % q;
    return (v < 0 && r) ? q - r : r;
}

// Both polynomials times the integer k (any scheme; no rescale).
int op_mul_int(Context &c, const uint64_t *a, int64_t k, uint64_t *out, uint32_t level,
               uint32_t count, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    const LimbMap m = map_ct(level);
    std::vector<uint64_t> kv(2 * level), ks(2 * level);
    std::vector<uint8_t> add(2 * level, 0);
    for (uint32_t i = 0; i < 2 * level; i++) {
        const uint64_t q = c.mod(int(i % level));
        kv[i] = reduce_signed(k, q);
        ks[i] = h_shoup(kv[i], q);
    }
    return launch_const_op(c, a, out, m, 2 * level * count, kv.data(), ks.data(), add.data(), s);
}

// Adds the plaintext constant k to every slot: c0 += k (the constant
// polynomial k, which is k at every evaluation point in NTT form) for CKKS
// and BGV; for BFV (coefficient form) c0 += Delta k at coefficient 0 is not
// an element-wise map, so BFV is not supported here.
int op_add_const(Context &c, const uint64_t *a, int64_t k, uint64_t *out, uint32_t level,
                 uint32_t count, cudaStream_t s) {
    if (c.scheme == CATFHE_BFV) return CATFHE_ESCHEME;
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    const LimbMap m = map_ct(level);
    std::vector<uint64_t> kv(2 * level, 1), ks(2 * level);
    std::vector<uint8_t> add(2 * level, 0);
    for (uint32_t i = 0; i < 2 * level; i++) {
        const uint64_t q = c.mod(int(i % level));
        if (i < level) {
            kv[i] = reduce_signed(k, q);
            add[i] = 1;
        }
        ks[i] = h_shoup(kv[i], q);
    }
    return launch_const_op(c, a, out, m, 2 * level * count, kv.data(), ks.data(), add.data(), s);
}

// Plaintext upload: the signed coefficients are staged in the last limb of
// pt, converted to residues for the other limbs, then in place for the last
// (each thread reads its own coefficient before writing it), then NTT.
int op_plain_import(Context &c, const int64_t *coeffs, uint32_t level, uint64_t *pt,
                    cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    const size_t n = c.n;
    int64_t *stage = reinterpret_cast<int64_t *>(pt + size_t(level - 1) * n);
    if (cudaMemcpyAsync(stage, coeffs, n * 8, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return CATFHE_ECUDA;
    if (level > 1) {
        LimbMap m = map_identity(level - 1);
        TRY(launch_small_to_rns(c, stage, pt, m, level - 1, nullptr, nullptr, 0, s));
    }
    LimbMap ml{};
    ml.period = 1;
    ml.src_stride = ml.dst_stride = 1;
    ml.src_off[0] = ml.dst_off[0] = uint16_t(level - 1);
    ml.prime[0] = uint8_t(level - 1);
    TRY(launch_small_to_rns(c, stage, pt, ml, 1, nullptr, nullptr, 0, s));
    LimbMap m = map_identity(level);
    TRY(launch_ntt_fwd(c, pt, pt, m, level, s));
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

// CKKS / BGV rest in NTT form: one limb-wise product.  BFV rests in
// coefficient form: the negacyclic product is NTT, limb-wise product, INTT,
// all in out (each transform is safe in place).
int op_mul_plain(Context &c, const uint64_t *a, const uint64_t *pt, uint64_t *out, uint32_t level,
                 uint32_t count, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    if (c.scheme != CATFHE_BFV) return launch_mul_plain(c, a, pt, out, level, 2 * level * count, s);
    const LimbMap m = map_identity(level);
    TRY(launch_ntt_fwd(c, a, out, m, 2 * level * count, s));
    TRY(launch_mul_plain(c, out, pt, out, level, 2 * level * count, s));
    return launch_ntt_inv(c, out, out, m, 2 * level * count, s);
}

// Keeps the first new_level limbs of each polynomial (dropping primes keeps
// the message and, in CKKS, the scale).
int op_drop_level(Context &c, const uint64_t *a, uint32_t level, uint32_t new_level,
                  uint64_t *out, uint32_t count, cudaStream_t s) {
    if (level < 1 || int(level) > c.L || new_level < 1 || new_level > level) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    LimbMap m{};
    m.period = 2 * new_level;
    m.src_stride = 2 * level;
    m.dst_stride = 2 * new_level;
    for (uint32_t p = 0; p < 2; p++)
        for (uint32_t i = 0; i < new_level; i++) {
            m.src_off[p * new_level + i] = uint16_t(p * level + i);
            m.dst_off[p * new_level + i] = uint16_t(p * new_level + i);
            m.prime[p * new_level + i] = uint8_t(i);
        }
    return launch_copy_limbs(c, a, out, m, 2 * new_level * count, s);
}

int op_ntt(Context &c, uint64_t *limbs, uint32_t level, uint32_t count, int inverse,
           cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    LimbMap m = map_identity(level);
    return inverse ? launch_ntt_inv(c, limbs, limbs, m, level * count, s)
                   : launch_ntt_fwd(c, limbs, limbs, m, level * count, s);
}

// ----------------------------------------------------------------- keys

static SampleArgs sample_args(const Context &c, const uint8_t seed[32], uint32_t tag, uint32_t i0,
                              uint32_t i1, uint32_t kind) {
    SampleArgs a{};
    for (int i = 0; i < 8; i++)
        a.key[i] = uint32_t(seed[4 * i]) | (uint32_t(seed[4 * i + 1]) << 8) |
                   (uint32_t(seed[4 * i + 2]) << 16) | (uint32_t(seed[4 * i + 3]) << 24);
    a.tag = tag;
    a.i0 = i0;
    a.i1 = i1;
    a.kind = kind;
    memcpy(a.cdt, c.cdt, sizeof(a.cdt));
    return a;
}

enum { TAG_SK = 1, TAG_PK_A = 2, TAG_PK_E = 3, TAG_KSK_A = 4, TAG_KSK_E = 5, TAG_ENC_V = 6,
       TAG_ENC_E0 = 7, TAG_ENC_E1 = 8, TAG_CT_UNIFORM = 9 };

// Device array of t mod prime (Shoup pairs) for BGV error scaling.
struct DevConst {
    uint64_t *v = nullptr, *s = nullptr;
    ~DevConst() {
        cudaFree(v);
        cudaFree(s);
    }
    int set(const std::vector<uint64_t> &vals, const std::vector<uint64_t> &mods) {
        std::vector<uint64_t> sh(vals.size());
        for (size_t i = 0; i < vals.size(); i++) sh[i] = h_shoup(vals[i], mods[i]);
        if (cudaMalloc(&v, vals.size() * 8) != cudaSuccess) return CATFHE_ENOMEM;
        if (cudaMalloc(&s, vals.size() * 8) != cudaSuccess) return CATFHE_ENOMEM;
        // the kernels that read them may run on a stream of the caller's
        if (copy_in(v, vals.data(), vals.size() * 8) != cudaSuccess ||
            copy_in(s, sh.data(), vals.size() * 8) != cudaSuccess)
            return CATFHE_ECUDA;
        return CATFHE_OK;
    }
};

static int gen_ksk(Context &c, Keys &k, uint64_t id, const uint64_t *sp, cudaStream_t s) {
    const size_t n = c.n;
    const int E = c.L + c.K;
    uint64_t *key = nullptr, *e = nullptr, *rows = nullptr;
    if (cudaMalloc(&key, size_t(c.beta) * 2 * E * n * 8) != cudaSuccess) return CATFHE_ENOMEM;
    // a Galois key's rows are built aside, then permuted into place
    if (cudaMalloc(&e, size_t(E) * n * 8) != cudaSuccess ||
        (id && cudaMalloc(&rows, size_t(2) * E * n * 8) != cudaSuccess)) {
        cudaFree(e);
        cudaFree(key);
        return CATFHE_ENOMEM;
    }
    LimbMap m = map_identity(uint32_t(E));
    DevConst te, pf;
    std::vector<uint64_t> mods(E), tv(E);
    for (int i = 0; i < E; i++) {
        mods[i] = c.mod(i);
        tv[i] = c.scheme == CATFHE_BGV ? c.t % mods[i] : 1;
    }
    int rc = te.set(tv, mods);
    for (int j = 0; j < c.beta && rc == CATFHE_OK; j++) {
        uint64_t *kj = key + size_t(j) * 2 * E * n;
        uint64_t *bj = id ? rows : kj, *aj = bj + size_t(E) * n;
        rc = launch_sample(c, sample_args(c, k.seed, TAG_KSK_A, uint32_t(j), uint32_t(id), kUniform), aj,
                           m, uint32_t(E), nullptr, nullptr, s);
        if (!rc) rc = launch_ntt_fwd(c, aj, aj, m, uint32_t(E), s);
        if (!rc)
            rc = launch_sample(c, sample_args(c, k.seed, TAG_KSK_E, uint32_t(j), uint32_t(id), kGaussian),
                               e, m, uint32_t(E), c.scheme == CATFHE_BGV ? te.v : nullptr,
                               c.scheme == CATFHE_BGV ? te.s : nullptr, s);
        if (!rc) rc = launch_ntt_fwd(c, e, e, m, uint32_t(E), s);
        std::vector<uint64_t> pv(E, 0);
        for (int i = j * c.alpha; i < std::min((j + 1) * c.alpha, c.L); i++) pv[i] = pmod(c, c.mod(i));
        DevConst pfc;
        if (!rc) rc = pfc.set(pv, mods);
        if (!rc) rc = launch_ksk_row(c, aj, k.s_ntt, e, sp, bj, uint32_t(E), pfc.v, pfc.s, s);
        if (!rc && id)  // sigma_g^-1 (see Keys::ksk)
            rc = launch_automorph_ntt(c, rows, kj, uint32_t(2 * E), inv_mod_pow2(id, 2 * n), s);
        if (!rc) rc = cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
    }
    // Montgomery form: every limb times 2^64 mod its prime
    if (!rc) {
        std::vector<uint64_t> rv(E);
        for (int i = 0; i < E; i++) rv[i] = (uint64_t)(((unsigned __int128)1 << 64) % mods[i]);
        DevConst rm;
        rc = rm.set(rv, mods);
        if (!rc) rc = launch_scale_limbs(c, key, uint32_t(E), uint32_t(c.beta * 2), rm.v, rm.s, s);
        if (!rc) rc = cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
    }
    cudaFree(e);
    cudaFree(rows);
    if (rc) {
        cudaFree(key);
        return rc;
    }
    auto it = k.ksk.find(id);
    if (it != k.ksk.end()) cudaFree(it->second);
    k.ksk[id] = key;
    return CATFHE_OK;
}

int op_keygen(Context &c, const uint8_t seed[32], Keys **out) {
    Keys *k = new Keys();
    memcpy(k->seed, seed, 32);
    const size_t n = c.n;
    const int E = c.L + c.K;
    cudaStream_t s = 0;
    uint64_t *a = nullptr, *e = nullptr, *sp = nullptr;
    int rc = CATFHE_OK;
    if (cudaMalloc(&k->s_ntt, size_t(E) * n * 8) != cudaSuccess ||
        cudaMalloc(&k->pk, size_t(2) * c.L * n * 8) != cudaSuccess ||
        cudaMalloc(&e, size_t(E) * n * 8) != cudaSuccess ||
        cudaMalloc(&sp, size_t(E) * n * 8) != cudaSuccess)
        rc = CATFHE_ENOMEM;
    LimbMap mE = map_identity(uint32_t(E)), mL = map_identity(uint32_t(c.L));
    if (!rc) rc = launch_sample(c, sample_args(c, seed, TAG_SK, 0, 0, kTernary), k->s_ntt, mE,
                                uint32_t(E), nullptr, nullptr, s);
    if (!rc) rc = launch_ntt_fwd(c, k->s_ntt, k->s_ntt, mE, uint32_t(E), s);
    // public key over Q_L
    a = k->pk + size_t(c.L) * n;
    if (!rc) rc = launch_sample(c, sample_args(c, seed, TAG_PK_A, 0, 0, kUniform), a, mL,
                                uint32_t(c.L), nullptr, nullptr, s);
    if (!rc) rc = launch_ntt_fwd(c, a, a, mL, uint32_t(c.L), s);
    DevConst te, zero;
    std::vector<uint64_t> mods(c.L), tv(c.L), zv(c.L, 0);
    for (int i = 0; i < c.L; i++) {
        mods[i] = c.mod(i);
        tv[i] = c.scheme == CATFHE_BGV ? c.t % mods[i] : 1;
    }
    if (!rc) rc = te.set(tv, mods);
    if (!rc) rc = zero.set(zv, mods);
    if (!rc) rc = launch_sample(c, sample_args(c, seed, TAG_PK_E, 0, 0, kGaussian), e, mL,
                                uint32_t(c.L), c.scheme == CATFHE_BGV ? te.v : nullptr,
                                c.scheme == CATFHE_BGV ? te.s : nullptr, s);
    if (!rc) rc = launch_ntt_fwd(c, e, e, mL, uint32_t(c.L), s);
    if (!rc) rc = launch_ksk_row(c, a, k->s_ntt, e, nullptr, k->pk, uint32_t(c.L), zero.v, zero.s, s);
    // relinearisation key: s' = s^2
    if (!rc) rc = launch_pointwise(c, k->s_ntt, k->s_ntt, sp, mE, uint32_t(E), s);
    if (!rc) rc = cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
    if (!rc) rc = gen_ksk(c, *k, 0, sp, s);
    cudaFree(e);
    cudaFree(sp);
    if (rc) {
        cudaFree(k->s_ntt);
        cudaFree(k->pk);
        for (auto &kv : k->ksk) cudaFree(kv.second);
        delete k;
        return rc;
    }
    *out = k;
    return CATFHE_OK;
}

int op_gen_galois(Context &c, Keys &k, uint64_t g) {
    g %= 2 * c.n;
    if (!(g & 1)) return CATFHE_EINVAL;
    if (k.ksk.count(g)) return CATFHE_OK;
    const int E = c.L + c.K;
    uint64_t *sp = nullptr;
    if (cudaMalloc(&sp, size_t(E) * c.n * 8) != cudaSuccess) return CATFHE_ENOMEM;
    int rc = launch_automorph_ntt(c, k.s_ntt, sp, uint32_t(E), g, 0);
    if (!rc) rc = gen_ksk(c, k, g, sp, 0);
    cudaFree(sp);
    return rc;
}

void keys_free(Keys *k) {
    if (!k) return;
    cudaFree(k->s_ntt);
    cudaFree(k->pk);
    for (auto &kv : k->ksk) cudaFree(kv.second);
    delete k;
}

// Coefficient-form copies of the keys to host memory.
int op_keys_export(Context &c, const Keys &k, uint64_t id, int64_t *s_out, uint64_t *pk_out,
                   uint64_t *ksk_out) {
    const size_t n = c.n;
    const int E = c.L + c.K;
    size_t need = size_t(c.beta) * 2 * E * n;
    uint64_t *tmp = nullptr;
    if (cudaMalloc(&tmp, need * 8) != cudaSuccess) return CATFHE_ENOMEM;
    int rc = CATFHE_OK;
    LimbMap mE = map_identity(uint32_t(E));
    if (s_out) {
        rc = launch_ntt_inv(c, k.s_ntt, tmp, mE, 1, 0);  // limb q_0 only
        std::vector<uint64_t> h(n);
        if (!rc && cudaMemcpy(h.data(), tmp, n * 8, cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = CATFHE_ECUDA;
        const uint64_t q0 = c.mod(0);
        for (size_t j = 0; j < n && !rc; j++) s_out[j] = h[j] > q0 / 2 ? int64_t(h[j]) - int64_t(q0) : int64_t(h[j]);
    }
    if (!rc && pk_out) {
        LimbMap mL = map_identity(uint32_t(c.L));
        rc = launch_ntt_inv(c, k.pk, tmp, mL, uint32_t(2 * c.L), 0);
        if (!rc && cudaMemcpy(pk_out, tmp, size_t(2) * c.L * n * 8, cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = CATFHE_ECUDA;
    }
    if (!rc && ksk_out) {
        auto it = k.ksk.find(id);
        if (it == k.ksk.end()) rc = CATFHE_ENOKEY;
        // a Galois key is stored permuted: sigma_g gives its definition back
        if (!rc && id) rc = launch_automorph_ntt(c, it->second, tmp, uint32_t(c.beta * 2 * E), id, 0);
        if (!rc)
            rc = launch_ntt_inv(c, id ? tmp : it->second, tmp, mE, uint32_t(c.beta * 2 * E), 0);
        // undo the Montgomery form: times 2^-64 mod each prime
        std::vector<uint64_t> rv(E), mods(E);
        for (int i = 0; i < E && !rc; i++) {
            mods[i] = c.mod(i);
            rv[i] = h_invmod((uint64_t)(((unsigned __int128)1 << 64) % mods[i]), mods[i]);
        }
        DevConst ri;
        if (!rc) rc = ri.set(rv, mods);
        if (!rc) rc = launch_scale_limbs(c, tmp, uint32_t(E), uint32_t(c.beta * 2), ri.v, ri.s, 0);
        if (!rc && cudaMemcpy(ksk_out, tmp, need * 8, cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = CATFHE_ECUDA;
    }
    cudaFree(tmp);
    return rc;
}

// ----------------------------------------------------------------- encryption

int op_encrypt(Context &c, const Keys &k, const int64_t *msg, const uint8_t seed[32],
               uint64_t *ct, cudaStream_t s) {
    const size_t n = c.n;
    const int L = c.L;
    int64_t *dmsg = nullptr;
    uint64_t *v = nullptr, *tmp = nullptr;
    int rc = CATFHE_OK;
    if (cudaMalloc(&dmsg, n * 8) != cudaSuccess || cudaMalloc(&v, size_t(L) * n * 8) != cudaSuccess ||
        cudaMalloc(&tmp, size_t(2) * L * n * 8) != cudaSuccess)
        rc = CATFHE_ENOMEM;
    if (!rc && cudaMemcpyAsync(dmsg, msg, n * 8, cudaMemcpyHostToDevice, s) != cudaSuccess) rc = CATFHE_ECUDA;
    LimbMap mL = map_identity(uint32_t(L));
    std::vector<uint64_t> mods(L), tv(L), dv(L);
    uint64_t qmodt = 1;
    if (c.t)
        for (int i = 0; i < L; i++) qmodt = h_mulmod(qmodt, c.mod(i) % c.t, c.t);
    for (int i = 0; i < L; i++) {
        mods[i] = c.mod(i);
        tv[i] = c.scheme == CATFHE_BGV ? c.t % mods[i] : 1;
        // BFV Delta = floor(Q/t) = (Q - (Q mod t)) / t, mod q_i
        dv[i] = c.scheme == CATFHE_BFV
                    ? h_mulmod((mods[i] - qmodt % mods[i]) % mods[i], h_invmod(c.t % mods[i], mods[i]), mods[i])
                    : 1;
    }
    DevConst te, dl;
    if (!rc) rc = te.set(tv, mods);
    if (!rc) rc = dl.set(dv, mods);
    const bool bgv = c.scheme == CATFHE_BGV;
    uint64_t *t0 = tmp, *t1 = tmp + size_t(L) * n;
    if (!rc) rc = launch_sample(c, sample_args(c, seed, TAG_ENC_V, 0, 0, kTernary), v, mL, uint32_t(L),
                                nullptr, nullptr, s);
    if (!rc) rc = launch_ntt_fwd(c, v, v, mL, uint32_t(L), s);
    if (!rc) rc = launch_sample(c, sample_args(c, seed, TAG_ENC_E0, 0, 0, kGaussian), t0, mL,
                                uint32_t(L), bgv ? te.v : nullptr, bgv ? te.s : nullptr, s);
    if (!rc) rc = launch_sample(c, sample_args(c, seed, TAG_ENC_E1, 0, 0, kGaussian), t1, mL,
                                uint32_t(L), bgv ? te.v : nullptr, bgv ? te.s : nullptr, s);
    if (!rc) rc = launch_small_to_rns(c, dmsg, t0, mL, uint32_t(L),
                                      c.scheme == CATFHE_BFV ? dl.v : nullptr,
                                      c.scheme == CATFHE_BFV ? dl.s : nullptr, 1, s);
    uint64_t *c0 = ct, *c1 = ct + size_t(L) * n;
    if (c.scheme != CATFHE_BFV) {
        if (!rc) rc = launch_ntt_fwd(c, tmp, tmp, mL, uint32_t(2 * L), s);
        if (!rc) rc = launch_mul_add(c, t0, v, k.pk, c0, uint32_t(L), 0, s);
        if (!rc) rc = launch_mul_add(c, t1, v, k.pk + size_t(L) * n, c1, uint32_t(L), 0, s);
    } else {
        // v pk in NTT form, back to coefficients, plus (e0 + Delta m, e1)
        if (!rc) rc = launch_mul_add(c, nullptr, v, k.pk, c0, uint32_t(L), 0, s);
        if (!rc) rc = launch_mul_add(c, nullptr, v, k.pk + size_t(L) * n, c1, uint32_t(L), 0, s);
        if (!rc) rc = launch_ntt_inv(c, ct, ct, mL, uint32_t(2 * L), s);
        LimbMap m2{};
        m2.period = uint32_t(2 * L);
        m2.src_stride = m2.dst_stride = uint32_t(2 * L);
        for (int i = 0; i < 2 * L; i++) {
            m2.src_off[i] = m2.dst_off[i] = uint16_t(i);
            m2.prime[i] = uint8_t(i % L);
        }
        if (!rc) rc = launch_add(c, ct, tmp, ct, m2, uint32_t(2 * L), s);
    }
    if (!rc) rc = cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
    cudaFree(dmsg);
    cudaFree(v);
    cudaFree(tmp);
    return rc;
}

int op_ct_uniform(Context &c, const uint8_t seed[32], uint32_t index, uint32_t level, uint64_t *ct,
                  cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    LimbMap m = map_identity(level);
    for (uint32_t poly = 0; poly < 2; poly++)
        TRY(launch_sample(c, sample_args(c, seed, TAG_CT_UNIFORM, poly, index, kUniform),
                          ct + size_t(poly) * level * c.n, m, level, nullptr, nullptr, s));
    if (c.scheme != CATFHE_BFV) TRY(launch_ntt_fwd(c, ct, ct, m, 2 * level, s));
    return CATFHE_OK;
}

int op_import(Context &c, const uint64_t *host, uint32_t level, uint32_t count, int form,
              bool sync, uint64_t *ct, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    const size_t bytes = size_t(count) * 2 * level * c.n * 8;
    if (cudaMemcpyAsync(ct, host, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) return CATFHE_ECUDA;
    if (form == CATFHE_FORM_COEFF && c.scheme != CATFHE_BFV) {
        LimbMap m = map_identity(level);
        TRY(launch_ntt_fwd(c, ct, ct, m, 2 * level * count, s));
    }
    if (!sync) return CATFHE_OK;
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

int op_export(Context &c, const uint64_t *ct, uint32_t level, uint32_t count, int form,
              bool sync, uint64_t *host, void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    const size_t bytes = size_t(count) * 2 * level * c.n * 8;
    const uint64_t *src = ct;
    if (form == CATFHE_FORM_COEFF && c.scheme != CATFHE_BFV) {
        char *base;
        TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_EXPORT, level, count), &base));
        Bump b{base};
        uint64_t *tmp = b.take<uint64_t>(size_t(count) * 2 * level * c.n);
        LimbMap m = map_identity(level);
        TRY(launch_ntt_inv(c, ct, tmp, m, 2 * level * count, s));
        src = tmp;
    }
    if (cudaMemcpyAsync(host, src, bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess) return CATFHE_ECUDA;
    if (!sync) return CATFHE_OK;
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

// Packed transfers: the packed words are staged in the workspace (at least
// 2 count packed_words(level) words), copied and unpacked in stream order.
int op_import_packed(Context &c, const uint64_t *host, uint32_t level, uint32_t count, bool sync,
                     uint64_t *ct, void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    const size_t bytes = size_t(2) * count * packed_words(c, level) * 8;
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, bytes, &base));
    if (cudaMemcpyAsync(base, host, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
        return CATFHE_ECUDA;
    TRY(launch_unpack(c, reinterpret_cast<const uint64_t *>(base), ct, level, 2 * count, s));
    if (!sync) return CATFHE_OK;
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

int op_export_packed(Context &c, const uint64_t *ct, uint32_t level, uint32_t count, bool sync,
                     uint64_t *host, void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (count == 0) return CATFHE_OK;
    const size_t bytes = size_t(2) * count * packed_words(c, level) * 8;
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, bytes, &base));
    uint64_t *stage = reinterpret_cast<uint64_t *>(base);
    TRY(launch_pack(c, ct, stage, level, 2 * count, s));
    if (cudaMemcpyAsync(host, stage, bytes, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return CATFHE_ECUDA;
    if (!sync) return CATFHE_OK;
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

// [c0 + c1 s]_{Q_l} per coefficient (CKKS: centred, two's complement; BFV:
// round(t x / Q) mod t; BGV: x mod t) into res (device int64[N]), using
// 2 level N words of scratch at base.
static int decrypt_device(Context &c, const Keys &k, const uint64_t *ct, uint32_t level,
                          int64_t *res, char *base, cudaStream_t s) {
    Bump b{base};
    const size_t n = c.n;
    uint64_t *x = b.take<uint64_t>(size_t(level) * n);
    uint64_t *tmp = b.take<uint64_t>(size_t(level) * n);
    LimbMap m = map_identity(level);
    if (c.scheme != CATFHE_BFV) {
        TRY(launch_mul_add(c, ct, ct + size_t(level) * n, k.s_ntt, x, level, 0, s));
        TRY(launch_ntt_inv(c, x, x, m, level, s));
    } else {
        TRY(launch_ntt_fwd(c, ct + size_t(level) * n, tmp, m, level, s));
        TRY(launch_mul_add(c, nullptr, tmp, k.s_ntt, tmp, level, 0, s));
        TRY(launch_ntt_inv(c, tmp, tmp, m, level, s));
        TRY(launch_add(c, ct, tmp, x, m, level, s));
    }
    PlanSpec sp;
    for (uint32_t i = 0; i < level; i++) {
        sp.src_mod.push_back(c.mod(int(i)));
        sp.src_off.push_back(i);
    }
    sp.dst_off.push_back(0);
    std::string key = "decrypt/" + std::to_string(level);
    if (c.scheme == CATFHE_CKKS) {
        sp.dst_mod.push_back(0);
        if (plan_fits_mont(sp)) {
            std::lock_guard<std::mutex> lock(c.mu);
            const PlanRef exact = get_plan(c, key, sp);
            if (!exact.p) return CATFHE_ENOMEM;
            const std::string wkey = key + "/wrap";
            if (!c.plans.count(wkey) && !upload_words(c, wkey, wrap_consts(sp.src_mod)))
                return CATFHE_ENOMEM;
            return launch_lift_wrap(c, c.plans[wkey], exact.p, level, x,
                                    reinterpret_cast<uint64_t *>(res), s);
        }
    } else {
        sp.dst_mod.push_back(c.t);
        if (c.scheme == CATFHE_BFV) {
            // round(t x / Q) mod t = -[t x]_Q Q^-1 mod t
            for (uint32_t i = 0; i < level; i++) sp.pre.push_back(c.t % c.mod(int(i)));
            const uint64_t qt = prod_mod(c, 0, int(level), c.t);
            sp.post.push_back((c.t - h_invmod(qt, c.t)) % c.t);
        }
    }
    ConvPlans pl{};
    {
        std::lock_guard<std::mutex> lock(c.mu);
        TRY(make_list(c, {{key, sp}}, pl));
    }
    return launch_conv(c, pl, x, 0, 0, reinterpret_cast<uint64_t *>(res), 0, 0, 1, s);
}

int op_decrypt(Context &c, const Keys &k, const uint64_t *ct, uint32_t level, uint64_t factor,
               int64_t *msg, void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (c.scheme == CATFHE_BGV && (factor % c.t == 0 || h_invmod(factor % c.t, c.t) == 0))
        return CATFHE_EINVAL;
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_DECRYPT, level, 1), &base));
    const size_t n = c.n;
    int64_t *res = reinterpret_cast<int64_t *>(base + size_t(2) * level * n * 8);
    TRY(decrypt_device(c, k, ct, level, res, base, s));
    if (cudaMemcpyAsync(msg, res, n * 8, cudaMemcpyDeviceToHost, s) != cudaSuccess) return CATFHE_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return CATFHE_ECUDA;
    if (c.scheme == CATFHE_BGV) {
        const uint64_t finv = h_invmod(factor % c.t, c.t);
        for (size_t j = 0; j < n; j++) msg[j] = int64_t(h_mulmod(uint64_t(msg[j]), finv, c.t));
    }
    return CATFHE_OK;
}

// CKKS encode on the device: host slots (N/2 complex) -> plaintext in NTT form.
int op_encode_ckks(Context &c, const double *slots, double scale, uint32_t level, uint64_t *pt,
                   void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (c.scheme != CATFHE_CKKS) return CATFHE_ESCHEME;
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (!(scale > 0)) return CATFHE_EINVAL;
    TRY(enc_tables(c));
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_ENCODE, level, 1), &base));
    Bump b{base};
    const size_t n = c.n;
    double2 *dz = b.take<double2>(n / 2);
    double2 *buf = b.take<double2>(n);
    int64_t *m = b.take<int64_t>(n);
    if (cudaMemcpyAsync(dz, slots, n / 2 * sizeof(double2), cudaMemcpyHostToDevice, s) != cudaSuccess)
        return CATFHE_ECUDA;
    TRY(launch_encode_ckks(c, dz, scale, buf, m, s));
    // every limb's transform reduces the signed coefficients as it loads them
    LimbMap mp = map_identity(level);
    for (uint32_t i = 0; i < level; i++) mp.src_off[i] = 0;
    {
        std::lock_guard<std::mutex> lock(c.mu);
        LiftEntry e{};
        e.flags = kLiftSigned;
        if (!c.signed_lifts) c.signed_lifts = upload_lifts(c, std::vector<LiftEntry>(size_t(c.L), e));
        if (!c.signed_lifts) return CATFHE_ENOMEM;
    }
    TRY(launch_ntt_lift(c, reinterpret_cast<const uint64_t *>(m), pt, mp, level, c.signed_lifts,
                        false, s));
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

// CKKS decrypt + decode: ciphertext -> host slots (N/2 complex) / scale.
int op_decode_ckks(Context &c, const Keys &k, const uint64_t *ct, uint32_t level, double scale,
                   double *slots, void *ws, size_t ws_bytes_in, cudaStream_t s) {
    if (c.scheme != CATFHE_CKKS) return CATFHE_ESCHEME;
    if (level < 1 || int(level) > c.L) return CATFHE_ELEVEL;
    if (!(scale > 0)) return CATFHE_EINVAL;
    TRY(enc_tables(c));
    char *base;
    TRY(get_ws(c, ws, ws_bytes_in, ws_bytes(c, CATFHE_OP_DECODE, level, 1), &base));
    Bump b{base};
    const size_t n = c.n;
    char *dec = reinterpret_cast<char *>(b.take<uint64_t>(size_t(2) * level * n));
    int64_t *m = b.take<int64_t>(n);
    double2 *buf = b.take<double2>(n);
    double2 *dz = b.take<double2>(n / 2);
    TRY(decrypt_device(c, k, ct, level, m, dec, s));
    TRY(launch_decode_ckks(c, m, 1.0 / scale, buf, dz, s));
    if (cudaMemcpyAsync(slots, dz, n / 2 * sizeof(double2), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return CATFHE_ECUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? CATFHE_OK : CATFHE_ECUDA;
}

}  // namespace catfhe
