// The library's host code (ops.cpp, context.cpp, mmaplan.cpp, hostmath.cpp) on
// a fake CUDA runtime: what its uploads do when the device
// behaves as the runtime's documentation allows, not as it usually does.
//
// A copy from pageable memory only stages its bytes; they arrive when its
// stream, the legacy one, is waited for.  Work on another stream in between
// finds the buffer's old contents.  A failed allocation stays the thread's last
// error until somebody reads it, and every launch reads it.
//
//   host_uploads("encrypt", scheme)  the number of constants that kernels of an
//                                    encryption were given before they arrived
//   host_uploads("nomem", scheme)    the last error after a conversion's plans
//                                    were made without memory for its
//                                    tensor-core image
//   host_uploads("over", scheme)     the most streams that a fused product of
//                                    four runs on when it is written over an
//                                    input (-1 unless it runs on two elsewhere)
#include <stdlib.h>
#include <string.h>

#include <set>

#include "internal.h"

namespace {
struct Staged {
    void *dst;
    std::vector<char> bytes;
};
std::vector<Staged> staged;
int late = 0;
bool no_memory = false;
cudaError_t last = cudaSuccess;
std::set<cudaStream_t> used;

void arrive() {
    for (auto &c : staged) memcpy(c.dst, c.bytes.data(), c.bytes.size());
    staged.clear();
}

// A kernel reads constants at p.
void read_by_kernel(const uint64_t *p) {
    for (auto &c : staged)
        if (p && c.dst == p) late++;
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
    if (no_memory) return last = cudaErrorMemoryAllocation;
    *p = calloc(1, n);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {  // waits for everything
    if (p) arrive();
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { return memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind kind) {
    if (kind == cudaMemcpyHostToDevice) {
        const char *b = static_cast<const char *>(src);
        staged.push_back({dst, std::vector<char>(b, b + n)});
    } else {
        arrive();
        memcpy(dst, src, n);
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind, cudaStream_t) {
    return memcpy(dst, src, n), cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (s == nullptr || s == cudaStreamLegacy) arrive();
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    static uintptr_t next = 32;
    *s = reinterpret_cast<cudaStream_t>(next += 16);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
}

namespace catfhe {
int ctx_init(Context &c, const catfhe_params &p);
int op_encrypt(Context &c, const Keys &k, const int64_t *msg, const uint8_t seed[32], uint64_t *ct,
               cudaStream_t s);
int op_mul_relin(Context &c, const Keys &keys, const uint64_t *a, const uint64_t *b,
                 uint64_t *out, uint32_t level, uint32_t count, bool fused, void *ws,
                 size_t ws_bytes_in, cudaStream_t s, const Gather *gth, bool split);
size_t ws_bytes(const Context &c, int op, uint32_t level, uint32_t count);

int launch_tensor(const Context &, const TensorArgs &, uint32_t, cudaStream_t s) {
    used.insert(s);
    return 0;
}
int launch_ip(const Context &, const IpArgs &, uint32_t, cudaStream_t s) {
    used.insert(s);
    return 0;
}
int launch_conv(const Context &, const ConvPlans &, const uint64_t *, size_t, size_t, uint64_t *,
                size_t, size_t, uint32_t, cudaStream_t, bool) {
    return 0;
}
int launch_ntt_lift(const Context &, const uint64_t *, uint64_t *, const LimbMap &, uint32_t,
                    const LiftEntry *, bool, cudaStream_t) {
    return 0;
}
int launch_ntt_fwd_lazy(const Context &, const uint64_t *, uint64_t *, const LimbMap &, uint32_t,
                        cudaStream_t) {
    return 0;
}
int launch_ntt_fwd_combine(const Context &, uint64_t *, const LimbMap &, uint32_t,
                           const NttEpilogue &, cudaStream_t) {
    return 0;
}
int launch_ntt_lift_combine(const Context &, const uint64_t *, uint64_t *, const LimbMap &,
                            uint32_t, const LiftEntry *, const NttEpilogue &, cudaStream_t) {
    return 0;
}
int launch_ntt_fwd(const Context &, const uint64_t *, uint64_t *, const LimbMap &, uint32_t,
                   cudaStream_t) {
    return 0;
}
int launch_ntt_inv(const Context &, const uint64_t *, uint64_t *, const LimbMap &, uint32_t,
                   cudaStream_t, const NttFactor *) {
    return 0;
}
int launch_add(const Context &, const uint64_t *, const uint64_t *, uint64_t *, const LimbMap &,
               uint32_t, cudaStream_t) {
    return 0;
}
int launch_mul_add(const Context &, const uint64_t *, const uint64_t *, const uint64_t *,
                   uint64_t *, uint32_t, int, cudaStream_t) {
    return 0;
}
int launch_sample(const Context &, const SampleArgs &, uint64_t *, const LimbMap &, uint32_t,
                  const uint64_t *mult, const uint64_t *mult_s, cudaStream_t) {
    read_by_kernel(mult);
    read_by_kernel(mult_s);
    return 0;
}
int launch_small_to_rns(const Context &, const int64_t *, uint64_t *, const LimbMap &, uint32_t,
                        const uint64_t *mult, const uint64_t *mult_s, int, cudaStream_t) {
    read_by_kernel(mult);
    read_by_kernel(mult_s);
    return 0;
}
}  // namespace catfhe

using namespace catfhe;

extern "C" int host_uploads(const char *what, int scheme) {
    catfhe_params p{};
    p.scheme = scheme;
    p.log_n = p.log_n_max = strcmp(what, "over") ? 12 : 14;
    p.L = 3;
    p.K = 1;
    p.dnum = 1;
    for (int i = 0; i < 3; i++) p.q_bits[i] = 50;
    p.p_bits[0] = 60;
    p.t = 65537;
    Context c;
    if (ctx_init(c, p)) return -1;
    if (!strcmp(what, "encrypt")) {
        Keys k{};
        std::vector<int64_t> msg(c.n);
        std::vector<uint64_t> ct(2 * size_t(p.L) * c.n);
        const uint8_t seed[32] = {};
        const cudaStream_t own = reinterpret_cast<cudaStream_t>(16);  // a non-blocking stream
        if (op_encrypt(c, k, msg.data(), seed, ct.data(), own)) return -1;
        return late;
    }
    if (!strcmp(what, "over")) {
        // (the buffers' addresses are all that is looked at)
        static uint64_t key;
        Keys k{};
        k.ksk[0] = &key;
        uint64_t *at = reinterpret_cast<uint64_t *>(uintptr_t(1) << 40);
        const size_t words = 4 * 2 * 3 * c.n;
        const size_t need = ws_bytes(c, CATFHE_OP_MUL_RELIN, 3, 4);  // the larger
        auto streams = [&](uint64_t *out, bool fused) -> int {
            used.clear();
            if (op_mul_relin(c, k, at, at + words, out, 3, 4, fused, at + 4 * words, need, nullptr,
                             nullptr, true))
                return -1;
            return int(used.size());
        };
        // in its own buffer, and in place with the shape of the input: halves
        if (streams(at + 2 * words, true) != 2 || streams(at, false) != 2) return -1;
        const int a = streams(at, true), b = streams(at + words, true);
        const int shifted = streams(at + words / 2, true);
        return a > b ? (a > shifted ? a : shifted) : (b > shifted ? b : shifted);
    }
    PlanSpec s;
    for (uint32_t i = 0; i < 3; i++) {
        s.src_mod.push_back(c.mod(int(i)));
        s.src_off.push_back(i);
    }
    s.dst_mod.push_back(c.mod(3));
    s.dst_off.push_back(0);
    no_memory = true;
    const MmaRef image = get_mma_plan(c, "x", s, c.n);
    no_memory = false;
    if (image.p || !get_plan(c, "x", s).p) return -1;  // the integer form's plan
    return int(cudaGetLastError());
}
