// msp_noalloc.cu -- msp_direct_noalloc: the all-pairs attraction of Eq. 8 for
// callers that must not allocate device memory.
//
// Some callers cannot let a library call cudaMalloc: a simulation loop that
// must never block on the allocator (cudaMalloc/cudaFree can synchronise the
// whole device and take unbounded time), or a host framework that owns every
// device allocation through its own pool and forbids libraries to allocate
// behind its back.  This entry point needs no context (msp_create allocates)
// and no workspace: its scratch is a fixed, file-scope device array that is
// part of the loaded library image.  Every GPU that loads the library holds
// that array (MSP_NOALLOC_MAX_N * 24 bytes) until the process exits.
#include <mutex>

#include "msp_direct.cuh"

namespace msp {
void set_last_error(const char* msg);
}

namespace {

constexpr size_t kNaPtsBytes = (size_t)MSP_NOALLOC_MAX_N * sizeof(float4);
constexpr size_t kNaListBytes = (size_t)MSP_NOALLOC_MAX_N * sizeof(int32_t);
constexpr size_t kNaBytes = (size_t)MSP_NOALLOC_MAX_N * 24;
static_assert(kNaPtsBytes + kNaListBytes +
                      msp::DirScratch::words(MSP_NOALLOC_MAX_N) * sizeof(int32_t) <= kNaBytes,
              "the scratch holds the packed copy, the target lists, their counts and the boxes");

// The scratch: the packed neurons (float4), the target lists (int32), their
// counts and the source tiles' boxes of up to MSP_NOALLOC_MAX_N neurons.  Shared
// by every call; everything in it is rewritten before it is read, so nothing left
// by an earlier call is ever used.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

// Device address of g_noalloc_scratch, looked up once per device and CUDA
// context.  The cache is keyed on the context's unique id (cuCtxGetId, reached
// through the runtime's driver entry points so that the library does not link
// libcuda): after a cudaDeviceReset the device's next context holds the array
// at a new address, and the next call looks it up again.
constexpr int kNaMaxDevices = 64;
std::mutex g_na_mu;
void* g_na_ptr[kNaMaxDevices] = {};
unsigned long long g_na_ctx[kNaMaxDevices] = {};

typedef int (*CtxGetCurrentFn)(void**);
typedef int (*CtxGetIdFn)(void*, unsigned long long*);

// id of the calling thread's current context, 0 if none or not available
unsigned long long current_context_id() {
    static CtxGetCurrentFn get_current = nullptr;
    static CtxGetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<CtxGetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<CtxGetIdFn>(f);
    });
    if (!get_current || !get_id) return 0;
    void* ctx = nullptr;
    unsigned long long id = 0;
    if (get_current(&ctx) != 0 || !ctx || get_id(ctx, &id) != 0) return 0;
    return id;
}

msp_status scratch_address(int dev, void** out) {
    if (dev < 0 || dev >= kNaMaxDevices) return MSP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lock(g_na_mu);
    const unsigned long long ctx = current_context_id();
    if (!g_na_ptr[dev] || ctx == 0 || ctx != g_na_ctx[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return MSP_ERR_CUDA;
        g_na_ptr[dev] = p;
        g_na_ctx[dev] = current_context_id();   // the lookup made the context current
    }
    *out = g_na_ptr[dev];
    return MSP_OK;
}

// 1 when p is device (or managed) memory of device `dev`
bool on_device(const void* p, int dev) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();   // a failed query leaves a (non-sticky) error: clear it
        return false;
    }
    return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == dev;
}

// the packed copy of the caller's arrays, for calls whose u lies over one of them
__global__ void k_dir_pack(int64_t n, msp::DirRaw src, float4* __restrict__ pts) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) pts[i] = src.get(i);
}

}  // namespace

extern "C" msp_status msp_direct_noalloc(int64_t n, const float* x, const float* y, const float* z,
                                         const uint8_t* type, const uint8_t* vac_axon,
                                         const uint8_t* vac_dend_e, const uint8_t* vac_dend_i,
                                         double sigma, float* u, void* stream) {
    if (n < 0 || n > MSP_NOALLOC_MAX_N) {
        msp::set_last_error("msp_direct_noalloc: n exceeds MSP_NOALLOC_MAX_N (its fixed scratch)");
        return MSP_ERR_INVALID_ARG;
    }
    if (!(sigma > 0.0)) {
        msp::set_last_error("msp_direct_noalloc: sigma must be positive");
        return MSP_ERR_INVALID_ARG;
    }
    if (n == 0) return MSP_OK;
    if (!x || !y || !z || !type || !vac_axon || !vac_dend_e || !vac_dend_i || !u) {
        msp::set_last_error("msp_direct_noalloc: null pointer");
        return MSP_ERR_INVALID_ARG;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        msp::set_last_error(cudaGetErrorString(e));
        return MSP_ERR_CUDA;
    }
    void* base = nullptr;
    msp_status st = scratch_address(dev, &base);
    if (st != MSP_OK) {
        msp::set_last_error("msp_direct_noalloc: cannot resolve the scratch array on this device");
        return st;
    }
    const void* ptrs[8] = {x, y, z, type, vac_axon, vac_dend_e, vac_dend_i, u};
    for (const void* p : ptrs)
        if (!on_device(p, dev)) {
            msp::set_last_error("msp_direct_noalloc: every array must be device memory of the "
                                "current device");
            return MSP_ERR_INVALID_ARG;
        }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const float k2 = (float)(1.4426950408889634 / (sigma * sigma));
    const msp::DirRaw src{x, y, z, type, vac_axon, vac_dend_e, vac_dend_i};
    unsigned char* sc = static_cast<unsigned char*>(base);
    float4* P = reinterpret_cast<float4*>(sc);
    int32_t* list = reinterpret_cast<int32_t*>(sc + kNaPtsBytes);
    const msp::DirScratch t(reinterpret_cast<int32_t*>(sc + kNaPtsBytes + kNaListBytes), n);
    // u may lie over an input: every input is packed first then, since the
    // kernels read them while they write u
    using msp::meets;
    const bool over = meets(u, n * 4, x, n * 4) || meets(u, n * 4, y, n * 4) ||
                      meets(u, n * 4, z, n * 4) || meets(u, n * 4, type, n) ||
                      meets(u, n * 4, vac_axon, n) || meets(u, n * 4, vac_dend_e, n) ||
                      meets(u, n * 4, vac_dend_i, n);
    const unsigned small = (unsigned)((n + 31) / 32), threads = msp::kDirSmallWarps * 32;
    int launches = n <= msp::kDirSmallN ? 1 : 3;
    if (over) {
        ++launches;
        k_dir_pack<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, src, P);
        const msp::DirPacked packed{P};
        if (n <= msp::kDirSmallN)
            msp::k_dir_small<false><<<small, threads, 0, s>>>(n, packed, k2, nullptr, 0, nullptr, u);
        else
            msp::dir_launch_tiles<false>(n, packed, nullptr, P, list, t, k2, nullptr, 0, nullptr, u, s);
    } else if (n <= msp::kDirSmallN) {
        msp::k_dir_small<false><<<small, threads, 0, s>>>(n, src, k2, nullptr, 0, nullptr, u);
    } else {
        msp::dir_launch_tiles<false>(n, src, P, P, list, t, k2, nullptr, 0, nullptr, u, s);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        msp::set_last_error(cudaGetErrorString(e));
        return MSP_ERR_CUDA;
    }
    msp::g_kernel_launches.fetch_add(launches, std::memory_order_relaxed);
    msp::set_last_error("");
    return MSP_OK;
}
