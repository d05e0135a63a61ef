// Kernels that every family of sample kernels uses, in an image of their own (a
// context of one family then does not load the level kernels' code): the reduction of
// the per-slot sums, the normals of one step, the static scratch.
#include <atomic>
#include <mutex>

#include "dk_device.cuh"
#include "dk_kernels.h"

namespace dk {

// Fixed-order reduction over slots: one block per entry.
__global__ void __launch_bounds__(256) reduce_kernel(const double* part, int n_slots, double* out) {
    const int e = blockIdx.x;
    const bool is_max = (e == 1);
    const double* row = part + (size_t)e * n_slots;
    double v = 0.0;
    for (int s = threadIdx.x; s < n_slots; s += 256) v = is_max ? fmax(v, row[s]) : v + row[s];
    __shared__ double sh[256];
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            const double o = sh[threadIdx.x + w];
            sh[threadIdx.x] = is_max ? fmax(sh[threadIdx.x], o) : sh[threadIdx.x] + o;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) out[e] = sh[0];
}

// out[e] += in[e] (entry 1, the max mass error: max): merges the sums of two
// disjoint sample ranges of one level.
__global__ void add_sums_kernel(double* out, const double* in, int stride) {
    for (int e = threadIdx.x; e < stride; e += blockDim.x) out[e] = e == 1 ? fmax(out[e], in[e]) : out[e] + in[e];
}

// Normals of one fine step, written out (the level kernel keeps them in
// registers); same device functions as the level kernel.
__global__ void noise_kernel(int n, uint32_t m, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1,
                             float* z, uint32_t* raw) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n * n / 2) return;
    const uint4 x = philox10(make_uint4(static_cast<uint32_t>(p), m, c2, c3), k0, k1);
    if (raw) reinterpret_cast<uint4*>(raw)[p] = x;
    if (z) {
        float a1, a2, b1, b2;
        box_muller(x.x, x.y, a1, a2);
        box_muller(x.z, x.w, b1, b2);
        reinterpret_cast<float4*>(z)[p] = make_float4(a1, a2, b1, b2);
    }
}

cudaError_t launch_noise(int n, uint32_t m, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1, float* z,
                         uint32_t* raw, cudaStream_t st) {
    const int pairs = n * n / 2;
    noise_kernel<<<(pairs + 255) / 256, 256, 0, st>>>(n, m, c2, c3, k0, k1, z, raw);
    return cudaGetLastError();
}

// -------------------------------------------- statically allocated scratch
// Scratch for the per-slot partial sums of mlmc_dk_run_level_static, whose
// callers cannot allocate device memory.  Every GPU that loads the library
// holds this array until the process exits; all calls share it.
static __device__ __align__(256) double g_static_partials[kStaticScratchDoubles];

namespace {
constexpr int kMaxDevices = 64;
double* g_static_ptr[kMaxDevices] = {};
std::atomic<int> g_static_ready[kMaxDevices];
std::mutex g_static_mutex;
}  // namespace

cudaError_t static_scratch(double** out, size_t* capacity) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if (!g_static_ready[dev].load(std::memory_order_acquire)) {
        // Set-up, once per device, with that device current: in host code the
        // array's name is only a host-side stand-in, so the kernels get the
        // device address from the runtime.
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ready[dev].load(std::memory_order_relaxed)) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_static_partials);
            if (e != cudaSuccess) return e;
            g_static_ptr[dev] = static_cast<double*>(p);
            g_static_ready[dev].store(1, std::memory_order_release);
        }
    }
    *out = g_static_ptr[dev];
    *capacity = kStaticScratchDoubles;
    return cudaSuccess;
}

cudaError_t load_common() {
    cudaFuncAttributes attr;
    return cudaFuncGetAttributes(&attr, reduce_kernel);
}

cudaError_t launch_reduce(const double* partials, int n_slots, int slot_stride, double* out, cudaStream_t st) {
    reduce_kernel<<<slot_stride, 256, 0, st>>>(partials, n_slots, out);
    return cudaGetLastError();
}

cudaError_t launch_add_sums(double* out, const double* in, int slot_stride, cudaStream_t st) {
    add_sums_kernel<<<1, 256, 0, st>>>(out, in, slot_stride);
    return cudaGetLastError();
}

}  // namespace dk
