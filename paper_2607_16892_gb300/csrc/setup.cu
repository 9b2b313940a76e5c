// One launch that readies a call: a small block of host parameters, carried in the kernel's own arguments,
// and up to two arrays filled with a constant.  A copy through staging memory and a memset each cost a
// launch of their own and a switch between the copy and the compute engines (about 4 us a call together),
// and the staging buffer has to be waited for before the next call may fill it.
#include <cstring>
#include <initializer_list>

#include "kvdro_internal.cuh"

namespace kvdro {
namespace {

constexpr int kThreads = 256;

template <int BYTES>
struct Payload {
    uint2 w[BYTES / 8];
};

template <int BYTES>
__global__ void __launch_bounds__(kThreads) k_setup(const __grid_constant__ Payload<BYTES> p, uint2* dst, int words,
                                                    Fill f0, Fill f1) {
    const int64_t i0 = (int64_t)blockIdx.x * kThreads + threadIdx.x, step = (int64_t)gridDim.x * kThreads;
    for (int64_t i = i0; i < words; i += step) dst[i] = p.w[i];
    for (const Fill& f : {f0, f1}) {  // 16 bytes a thread; the arrays start on 16-byte boundaries
        const uint4 v = make_uint4(f.value, f.value, f.value, f.value);
        for (int64_t i = i0; i < f.words / 4; i += step) reinterpret_cast<uint4*>(f.p)[i] = v;
        for (int64_t i = f.words / 4 * 4 + i0; i < f.words; i += step) f.p[i] = f.value;
    }
}

template <int BYTES>
cudaError_t launch(const void* payload, size_t bytes, void* dst, const Fill& f0, const Fill& f1, unsigned blocks,
                   cudaStream_t s) {
    Payload<BYTES> p;
    if (bytes) std::memcpy(&p, payload, bytes);
    k_setup<BYTES><<<blocks, kThreads, 0, s>>>(p, static_cast<uint2*>(dst), (int)((bytes + 7) / 8), f0, f1);
    return cudaGetLastError();
}

}  // namespace

cudaError_t setup_prepare() {
    cudaFuncAttributes at;
    for (const void* kernel : {(const void*)k_setup<2048>, (const void*)k_setup<4032>, (const void*)k_setup<16384>})
        if (const cudaError_t e = cudaFuncGetAttributes(&at, kernel)) return e;
    return cudaSuccess;
}

bool setup_fits(size_t bytes) { return bytes <= 16384; }

cudaError_t launch_setup(const void* payload, size_t bytes, void* dst, const Fill& f0, const Fill& f1, cudaStream_t s) {
    const int64_t work = (f0.words + f1.words) / 4 + 1;
    const int64_t most = 1216;  // eight blocks on each of 152 SMs
    const unsigned blocks = (unsigned)(work / kThreads + 1 < most ? work / kThreads + 1 : most);
    if (bytes <= 2048) return launch<2048>(payload, bytes, dst, f0, f1, blocks, s);
    if (bytes <= 4032) return launch<4032>(payload, bytes, dst, f0, f1, blocks, s);
    return launch<16384>(payload, bytes, dst, f0, f1, blocks, s);
}

}  // namespace kvdro
