// rows.cu -- copies between the solver's arrays and a caller's device memory:
// linear ones, and delta-f rows between the padded layout ([row][pitch]) and the
// packed [row][nnode] layout of fdtd_plasma_read_fields / write_fields.
//
// A cudaMemcpyAsync inside device memory occupies the stream for about six
// microseconds however small it is (reading E, H, J and delta f of 256 batched runs,
// 1024 copies of 0.05 - 2 MB: 6.2 ms); those of 16 KB to 16 MB run as a kernel that
// starts while the work before it finishes (3.1 ms).
//
// A strided cudaMemcpy2D of short rows runs far below the copy bandwidth (rows of
// 124 bytes, 1.2 M of them: 141 us; 64-byte rows, 33.5 M: 3.2 ms), so rows that are not
// padded go as one linear copy and padded rows through this kernel: one thread a
// unit, the widest one (16, 8, 4 or 2 bytes) that a row and both layouts are a
// multiple of, consecutive threads on consecutive units of the packed side, the
// row of a unit by one multiplication (exact below 2^31).  Bound by HBM
// (the same rows: 51 us, and 0.62 ms as a linear copy).
#include <algorithm>

#include "internal.cuh"

namespace fp {

namespace {

constexpr int kRowsUnroll = 4;

template <typename U, bool PACK>
__global__ void __launch_bounds__(256) k_rows_copy(U *__restrict__ dst, const U *__restrict__ src, uint32_t n,
                                                   uint32_t per_row, uint32_t pitch, uint32_t mul, int shift)
{
    const uint32_t i0 = blockIdx.x * (256u * kRowsUnroll) + threadIdx.x;
    U v[kRowsUnroll];
    int64_t at[kRowsUnroll];
#pragma unroll
    for (int q = 0; q < kRowsUnroll; ++q) {
        const uint32_t i = i0 + 256u * q;
        if (i >= n) continue;
        const uint32_t row = (uint32_t)(((uint64_t)i * mul) >> shift);
        at[q] = (int64_t)row * pitch + (i - row * per_row);
        v[q] = PACK ? __ldcs(src + at[q]) : __ldcs(src + i);
    }
#pragma unroll
    for (int q = 0; q < kRowsUnroll; ++q) {
        const uint32_t i = i0 + 256u * q;
        if (i >= n) continue;
        if (PACK) dst[i] = v[q];
        else dst[at[q]] = v[q];
    }
}

template <typename U>
__global__ void __launch_bounds__(256) k_copy(U *__restrict__ dst, const U *__restrict__ src, uint32_t n)
{
    pdl_enter();
    const uint32_t stride = gridDim.x * 256u * kRowsUnroll;
    for (uint32_t i0 = blockIdx.x * (256u * kRowsUnroll) + threadIdx.x; i0 < n; i0 += stride) {
        U v[kRowsUnroll];
#pragma unroll
        for (int q = 0; q < kRowsUnroll; ++q)
            if (i0 + 256u * q < n) v[q] = src[i0 + 256u * q];
#pragma unroll
        for (int q = 0; q < kRowsUnroll; ++q)
            if (i0 + 256u * q < n) dst[i0 + 256u * q] = v[q];
    }
}

template <typename U>
cudaError_t run_copy(cudaStream_t st, void *dst, const void *src, size_t bytes, const CopyHome &home)
{
    const uint32_t n = (uint32_t)(bytes / sizeof(U));
    const DeviceGuard guard(home.dev);
    return launch_pdl(k_copy<U>, dim3(copy_blocks(n, 256 * kRowsUnroll, home)), dim3(256), 0, st, static_cast<U *>(dst), static_cast<const U *>(src), n);
}

bool reaches(const void *p, const CopyHome &home)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) == cudaSuccess)
        return kernel_reaches(at.type == cudaMemoryTypeDevice, at.device, home);
    cudaGetLastError();
    return false;
}

template <typename U>
cudaError_t run(cudaStream_t st, void *dst, const void *src, int64_t rows, size_t row, size_t pitch, bool pack,
                const CopyHome &home)
{
    const DeviceGuard guard(home.dev);
    const uint32_t per = (uint32_t)(row / sizeof(U)), n = (uint32_t)(rows * per);
    // i / per = (i * mul) >> shift for every i < 2^31: mul = ceil(2^(31 + k) / per), 2^k >= per
    int k = 0;
    while ((1u << k) < per) ++k;
    const uint32_t mul = (uint32_t)((((uint64_t)1 << (31 + k)) + per - 1) / per);
    const uint32_t blocks = (n + 256 * kRowsUnroll - 1) / (256 * kRowsUnroll);
    U *d = static_cast<U *>(dst);
    const U *s = static_cast<const U *>(src);
    if (pack) k_rows_copy<U, true><<<blocks, 256, 0, st>>>(d, s, n, per, (uint32_t)(pitch / sizeof(U)), mul, 31 + k);
    else k_rows_copy<U, false><<<blocks, 256, 0, st>>>(d, s, n, per, (uint32_t)(pitch / sizeof(U)), mul, 31 + k);
    return cudaGetLastError();
}

}  // namespace

cudaError_t copy_linear(cudaStream_t st, void *theirs, void *ours, size_t bytes, cudaMemcpyKind kind, bool out,
                        const CopyHome &home)
{
    void *dst = out ? theirs : ours;
    const void *src = out ? ours : theirs;
    // up to 16 MB the six microseconds are more than the kernel takes; beyond, both run at the copy bandwidth.  The
    // smallest keep the plain copy: a call with the pointer's check and a launch is a microsecond longer on the
    // host, which bounds a program that reads a few kilobytes after every step (39 against 43 us a step and four
    // reads)
    if (kind == cudaMemcpyDeviceToDevice && bytes > 16384 && bytes <= (size_t)16 << 20 && reaches(theirs, home)) {
        size_t u = 16;
        while (u > 2 && (((uintptr_t)dst | (uintptr_t)src | bytes) & (u - 1))) u >>= 1;
        switch (u) {
        case 16: return run_copy<uint4>(st, dst, src, bytes, home);
        case 8: return run_copy<uint2>(st, dst, src, bytes, home);
        case 4: return run_copy<uint32_t>(st, dst, src, bytes, home);
        default:
            if (!(((uintptr_t)dst | (uintptr_t)src | bytes) & 1)) return run_copy<uint16_t>(st, dst, src, bytes, home);
        }
    }
    return cudaMemcpyAsync(dst, src, bytes, kind, st);
}

cudaError_t copy_rows(cudaStream_t st, void *packed, void *padded, int64_t rows, size_t row, size_t pitch,
                      cudaMemcpyKind kind, bool out, const CopyHome &home)
{
    void *dst = out ? packed : padded;
    const void *src = out ? padded : packed;
    if (row == pitch) return copy_linear(st, packed, padded, (size_t)rows * row, kind, out, home);
    size_t u = 16;
    while (u > 1 && (row % u || pitch % u || (uintptr_t)packed % u)) u >>= 1;
    if (kind == cudaMemcpyDeviceToDevice && rows > 0 && u >= 2 && (uint64_t)rows * (row / u) < ((uint64_t)1 << 31) &&
        reaches(packed, home)) {
        switch (u) {
        case 16: return run<uint4>(st, dst, src, rows, row, pitch, out, home);
        case 8: return run<uint2>(st, dst, src, rows, row, pitch, out, home);
        case 4: return run<uint32_t>(st, dst, src, rows, row, pitch, out, home);
        default: return run<uint16_t>(st, dst, src, rows, row, pitch, out, home);
        }
    }
    return out ? cudaMemcpy2DAsync(packed, row, padded, pitch, row, rows, kind, st)
               : cudaMemcpy2DAsync(padded, pitch, packed, row, row, rows, kind, st);
}

}  // namespace fp
