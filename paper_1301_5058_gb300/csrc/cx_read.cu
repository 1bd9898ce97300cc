// cx_read.cu -- field reads into pinned host memory: one kernel takes a field
// from its pair order (cx_internal.h) to packed rows in natural order, in the
// caller's type, and writes them to the host array itself.
//
// A read through copies takes an in-place reordering of the field, the copy and
// the reordering back: three dependent operations, 25 us for a field of any
// small size.  The kernel is bound by the host link (large fields) or by its
// launch and the synchronisation (small ones): 256^2 in FP32 20.1 -> 14.1 us,
// 2048^2 122 -> 99, 16384^2 6.27 -> 5.57 ms (193 GB/s), 1024^2 in FP64 67 -> 56.
// The diagnostics' last kernel writes its record to the host in the same way
// (256^2 28 -> 23 us).  Pageable arrays still go through the copies.
#include <cuda.h>

#include <mutex>

#include "cx_stencil.cuh"

namespace cx {
namespace {

using namespace stencil;

// Each thread writes 16 bytes, or one element where rows or `dst` are not
// aligned to that: consecutive threads fill consecutive bytes of the link's
// packets (32 bytes per thread, in two stores, ran at 79 instead of 125 GB/s).
template <typename T, typename D, bool VEC>
__global__ void __launch_bounds__(256)
    read_field_kernel(const T *a, D *dst, int nx, int ny, long long pitch)
{
    pass_wait();
    constexpr int kUnit = VEC ? 16 / (int)sizeof(D) : 1;  // cells per thread
    const int units = nx / kUnit;
    const long long total = (long long)units * ny;
    for (long long q = blockIdx.x * 256LL + threadIdx.x; q < total; q += gridDim.x * 256LL) {
        const long long j = q / units;
        const int i = (int)(q - j * units) * kUnit;
        const T *row = a + j * pitch;
        D *p = dst + j * nx + i;
        if constexpr (!VEC) {
            *p = (D)Vec<T>::load1(row + pair_col(i));
        } else if constexpr (kUnit == 4) {
            T v[4];
            Vec<T>::load(row + i, v);
            *reinterpret_cast<float4 *>(p) = make_float4((float)v[0], (float)v[2], (float)v[1], (float)v[3]);
        } else {
            const long long c = pair_col(i);  // the next cell lies two elements on
            const D x = (D)Vec<T>::load1(row + c), y = (D)Vec<T>::load1(row + c + 2);
            *reinterpret_cast<double2 *>(p) = make_double2(x, y);
        }
    }
}

template <typename T, typename D>
cudaError_t launch_read(const void *a, void *dst, int nx, int ny, long long pitch, cudaStream_t st)
{
    const bool vec = nx % 4 == 0 && (uintptr_t)dst % 16 == 0;
    const long long units = (long long)nx * ny / (vec ? 16 / (int)sizeof(D) : 1);
    const long long blocks = (units + 255) / 256;
    const int grid = (int)(blocks < 152LL * 16 ? blocks : 152LL * 16);
    auto kern = vec ? read_field_kernel<T, D, true> : read_field_kernel<T, D, false>;
    return launch_pass(kern, grid, 256, 0, st, (const T *)a, (D *)dst, nx, ny, pitch);
}

using PointerAttributesFn = CUresult (*)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);

PointerAttributesFn pointer_attributes()
{
    static std::once_flag once;
    static PointerAttributesFn fn = nullptr;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PointerAttributesFn)f;
        cudaGetLastError();
    });
    return fn;
}

}  // namespace

void *pinned_view(void *host, size_t count, size_t elem)
{
    // a kernel stores whole elements: an array behind an odd-sized header goes
    // through the copies
    if ((uintptr_t)host % elem) return nullptr;
    const PointerAttributesFn get = pointer_attributes();
    if (!get) return nullptr;
    // one query: memory that CUDA does not know comes back as type 0
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                  CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    unsigned type = 0;
    CUdeviceptr p = 0, start = 0;
    size_t size = 0;
    void *values[] = {&type, &p, &start, &size};
    if (get(4, what, values, (CUdeviceptr)host) != CUDA_SUCCESS) return nullptr;
    if (type != CU_MEMORYTYPE_HOST || !p) return nullptr;
    // the whole array has to lie in the pinned allocation (one that does not is
    // left to the copies, which refuse it)
    return p % elem == 0 && p >= start && p + count * elem <= start + size ? (void *)p : nullptr;
}

cudaError_t launch_read_field(int prec, const void *field, int nx, int ny, long long pitch, void *dst,
                              int dtype, cudaStream_t st)
{
    if (prec == CX_PREC_F64)
        return dtype == CX_F64 ? launch_read<double, double>(field, dst, nx, ny, pitch, st)
                               : launch_read<double, float>(field, dst, nx, ny, pitch, st);
    return dtype == CX_F64 ? launch_read<float, double>(field, dst, nx, ny, pitch, st)
                           : launch_read<float, float>(field, dst, nx, ny, pitch, st);
}

}  // namespace cx
