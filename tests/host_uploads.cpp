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
#include <stdlib.h>
#include <string.h>

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
    p.log_n = p.log_n_max = 12;
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
