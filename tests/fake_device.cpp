// The CUDA runtime calls and kernel launchers of the host side (lbm_api.cu, lbm_adjoint.cu), on host memory:
// what lets tests drive the C ABI without a GPU.  Allocations can be made to fail; freed blocks are remembered,
// so that a launch that still names one is counted (fake_faults) instead of reading it.  The kernels do no
// physics: a buffer's first eight bytes hold the number of the state it belongs to, which a step counts up
// and every kernel checks.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "../include/lbm.h"
#include "../paper_2604_13407_gb300/csrc/lbm_internal.h"

using namespace lbm;

namespace {

std::map<const char *, size_t> g_live;
long g_mallocs_left = -1;      // allocations that still succeed; -1: all
size_t g_bytes_left = (size_t)-1;
long g_faults = 0, g_launches = 0, g_attributes = 0, g_mallocs = 0, g_small_asked = 0;
unsigned long long g_context = 1;
int g_small_ctas = 0;
std::string g_what, g_last;

void fault(const std::string &what)
{
    ++g_faults;
    if (g_what.empty()) g_what = what;
}
bool live(const void *p)
{
    auto it = g_live.upper_bound(static_cast<const char *>(p));
    if (it == g_live.begin()) return false;
    --it;
    return static_cast<const char *>(p) < it->first + it->second;
}
void need(const void *p, const char *what)
{
    if (p && !live(p)) fault(std::string(what) + " is not allocated");
}
int64_t &tag(const void *p) { return *static_cast<int64_t *>(const_cast<void *>(p)); }

// Every array a kernel may read is allocated, and the derived ones are there with what they derive from.
void check(const KParams &k, bool f32)
{
    ++g_launches;
    need(k.src, "src"), need(k.dst, "dst"), need(k.psi, "psi"), need(k.psi_out, "psi_out");
    need(k.solid, "solid"), need(k.wall_u, "wall_u"), need(k.q, "q"), need(k.fext, "fext"), need(k.fext_f, "fext_f");
    need(k.wall_rho, "wall_rho"), need(k.wall_psi, "wall_psi"), need(k.wall_psi_f, "wall_psi_f"), need(k.link, "link"), need(k.links, "links");
    if ((k.solid || k.wall_u || k.q) != (k.links != nullptr)) fault("links without walls, or walls without links");
    if (f32) {
        if ((k.wall_u || k.q) != (k.link != nullptr)) fault("link records without link walls, or the reverse");
        if ((k.fext != nullptr) != (k.fext_f != nullptr)) fault("fext without fext_f, or the reverse");
        if ((k.wall_psi != nullptr) != (k.wall_psi_f != nullptr)) fault("wall_psi without wall_psi_f, or the reverse");
    }
    if ((k.wall_rho != nullptr) != (k.wall_psi != nullptr)) fault("wall_rho without wall_psi, or the reverse");
}
void advance(const KParams &k) { tag(k.dst) = tag(k.src) + 1; }

template <int P>
struct Fake {
    static constexpr bool F32 = P != P_F64;
    static cudaError_t psi_pass(const KParams &k, cudaStream_t)
    {
        check(k, F32);
        tag(k.psi) = tag(k.src);
        return cudaSuccess;
    }
    static cudaError_t collide_pass(const KParams &k, cudaStream_t)
    {
        check(k, F32);
        if (tag(k.psi) != tag(k.src)) fault("collide: psi of another state");
        advance(k);
        g_last = "two_pass";
        return cudaSuccess;
    }
    static cudaError_t one(const KParams &k, const char *name)
    {
        check(k, F32);
        if (k.psi_out) tag(k.psi_out) = tag(k.src);
        advance(k);
        g_last = name;
        return cudaSuccess;
    }
    static cudaError_t fused_pass(const KParams &k, cudaStream_t) { return one(k, "staged"); }
    static cudaError_t tile_pass(const KParams &k, cudaStream_t) { return one(k, k.packed ? "tile packed" : "tile"); }
    static int small_ctas(const KParams &k) { return ++g_small_asked, k.q || k.wall_u ? 0 : g_small_ctas; }
    static cudaError_t small_steps(const KParams &k, int, int64_t n, int64_t, cudaStream_t)
    {
        check(k, F32);
        tag(n & 1 ? k.dst : k.src) = tag(k.src) + n;
        g_last = "small";
        return cudaSuccess;
    }
    static cudaError_t link_bits(const KParams &k, uint16_t *out, cudaStream_t)
    {
        need(k.solid, "solid"), need(out, "wall bits");
        return cudaSuccess;
    }
    static cudaError_t init(const KParams &k, const double *, const double *, const double *, cudaStream_t)
    {
        tag(k.dst) = 0;
        return cudaSuccess;
    }
    static cudaError_t moments(const KParams &k, double *, double *, double *, cudaStream_t)
    {
        check(k, F32);
        return cudaSuccess;
    }
    static int64_t diag_rows(const KParams &k) { return (int64_t)((k.nx + 31) / 32) * ((k.ny + 7) / 8); }
    static cudaError_t diag(const KParams &k, double *part, double *out, cudaStream_t)
    {
        check(k, F32);
        need(part, "part"), need(part + diag_rows(k) * 11 - 1, "end of part");
        std::memset(out, 0, 11 * sizeof(double));
        return cudaSuccess;
    }
    static cudaError_t get_state(const KParams &, double *, cudaStream_t) { return cudaSuccess; }
    static cudaError_t set_state(const KParams &k, const double *, cudaStream_t)
    {
        tag(k.dst) = 0;
        return cudaSuccess;
    }
    // Transposed step at A_t: reads what the one at A_{t+1} left.
    static cudaError_t adj_step(const KParams &k, const AdjArgs &a, cudaStream_t)
    {
        check(k, F32);
        const void *in[] = {a.g_in, a.dS_in, a.dpsi_in, a.rho_in, F32 ? nullptr : a.psi_in};
        const int64_t t = a.tail ? -1 : tag(k.src);
        for (const void *p : in) {
            need(p, "adjoint plane read");
            if (p && tag(p) != t + 1) fault("the transposed step reads planes of another state");
        }
        if (a.tail) {
            need(a.c_out, "c");
            for (const void *p : in)
                if (p == a.c_out) fault("c written over a plane that is read");
            tag(a.c_out) = t;
            return cudaSuccess;
        }
        if (tag(k.psi) != t) fault("the transposed step reads psi of another state");
        void *out[] = {a.g_out, a.dS_out, a.dpsi_out, a.rho_out, F32 ? nullptr : a.psi_out};
        for (void *p : out) {
            need(p, "adjoint plane written");
            if (p) tag(p) = t;
        }
        return cudaSuccess;
    }
    static cudaError_t adj_lambda(const KParams &, const void *g, const void *c, double *out, cudaStream_t)
    {
        need(out, "lambda0");
        if (tag(g) != 0 || tag(c) != -1) fault("lambda0 from other planes than the last ones");
        return cudaSuccess;
    }
    static cudaError_t objective(const KParams &k, int, double, double *acc, cudaStream_t)
    {
        *acc = (double)tag(k.src);
        return cudaSuccess;
    }
    static int64_t adj_blocks(const KParams &k) { return diag_rows(k); }
    static cudaError_t adj_reduce(const KParams &, const double *, double *out, cudaStream_t)
    {
        std::memset(out, 0, kAdjSlots * sizeof(double));
        return cudaSuccess;
    }
    static Launchers table()
    {
        Launchers L{};
        L.psi_pass = psi_pass, L.collide_pass = collide_pass, L.tile_pass = tile_pass;
        if (F32) L.fused_pass = fused_pass;
        L.small_ctas = small_ctas, L.small_steps = small_steps, L.link_bits = link_bits, L.init = init, L.moments = moments;
        L.diag_rows = diag_rows, L.diag = diag, L.get_state = get_state, L.set_state = set_state;
        L.adj_step = adj_step, L.adj_lambda = adj_lambda, L.objective = objective, L.adj_blocks = adj_blocks, L.adj_reduce = adj_reduce;
        L.fused_tile_x = 240, L.fused_align = P == P_F64 ? 2 : P == P_F32 ? 4 : 8, L.fused_geometry = F32;
        return L;
    }
};

}  // namespace

namespace lbm {
Launchers launchers_f64() { return Fake<P_F64>::table(); }
Launchers launchers_f32() { return Fake<P_F32>::table(); }
Launchers launchers_f16() { return Fake<P_F16>::table(); }
Launchers launchers_bf16() { return Fake<P_BF16>::table(); }
bool cluster_fits(const void *kernel, int device, int ctas, int threads, int smem_bytes);
}  // namespace lbm

extern "C" {
LBM_API void fake_limit(long mallocs, size_t bytes) { g_mallocs_left = mallocs, g_bytes_left = bytes; }
LBM_API void fake_reset(int small_ctas)
{
    g_mallocs_left = -1, g_bytes_left = (size_t)-1, g_small_ctas = small_ctas;
    g_faults = g_launches = g_attributes = g_mallocs = g_small_asked = 0;
    g_what.clear(), g_last.clear();
}
LBM_API long fake_faults() { return g_faults; }
LBM_API const char *fake_what() { return g_what.c_str(); }
LBM_API const char *fake_last_step() { return g_last.c_str(); }
LBM_API long fake_launches() { return g_launches; }
LBM_API long fake_small_asked() { return g_small_asked; }
LBM_API long fake_mallocs() { return g_mallocs; }
LBM_API long fake_attributes() { return g_attributes; }
LBM_API void fake_device_reset() { ++g_context; }
LBM_API size_t fake_bytes()
{
    size_t n = 0;
    for (const auto &b : g_live) n += b.second;
    return n;
}
LBM_API int fake_cluster_fits(int ctas) { return cluster_fits(reinterpret_cast<const void *>(&fake_cluster_fits), 0, ctas, 128, 1024); }
LBM_API lbm_status lbm_step_noalloc_f32(const lbm_params *, const float *, float *, int64_t, void *) { return LBM_ENOTSUP; }

cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = nullptr;
    if (g_mallocs_left == 0 || n > g_bytes_left) return cudaErrorMemoryAllocation;
    if (g_mallocs_left > 0) --g_mallocs_left;
    if (g_bytes_left != (size_t)-1) g_bytes_left -= n;
    *p = std::calloc(n + 64, 1);
    if (!*p) return cudaErrorMemoryAllocation;
    g_live[static_cast<char *>(*p)] = n + 64;
    ++g_mallocs;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    auto it = g_live.find(static_cast<char *>(p));
    if (it == g_live.end()) fault("freed twice");
    else {
        if (g_bytes_left != (size_t)-1) g_bytes_left += it->second - 64;
        if (it->second > (64u << 20)) std::free(p);  // (smaller blocks stay, so that no later one takes their address)
        g_live.erase(it);
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    if (kind != cudaMemcpyHostToDevice) need(s, "copied from");
    if (kind != cudaMemcpyDeviceToHost) need(d, "copied to");
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t)
{
    std::memset(d, v, n < 4096 ? n : 4096);  // (blocks are zeroed when they are allocated; the largest are never touched)
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = reinterpret_cast<cudaStream_t>(0x10), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = reinterpret_cast<cudaEvent_t>(0x20), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return ++g_attributes, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) { return *n = 1, cudaSuccess; }

// The driver calls that name the current context.
static int fake_cuCtxGetCurrent(void **c) { return *c = reinterpret_cast<void *>(0x30), 0; }
static int fake_cuCtxGetId(void *, unsigned long long *id) { return *id = g_context, 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **p, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *r)
{
    *p = std::strcmp(name, "cuCtxGetId") == 0 ? reinterpret_cast<void *>(&fake_cuCtxGetId) : reinterpret_cast<void *>(&fake_cuCtxGetCurrent);
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

// Registration and launch of the one kernel in lbm_api.cu (k_narrow: doubles to floats).
void **__cudaRegisterFatBinary(void *) { return reinterpret_cast<void **>(0x40); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *) { return *k = nullptr, cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **args, size_t, cudaStream_t)
{
    const double *in = *static_cast<const double **>(args[0]);
    float *out = *static_cast<float **>(args[1]);
    const int64_t n = *static_cast<int64_t *>(args[2]);
    need(in, "k_narrow in"), need(out, "k_narrow out");
    for (int64_t i = 0; i < n; ++i) out[i] = (float)in[i];
    return cudaSuccess;
}
}
