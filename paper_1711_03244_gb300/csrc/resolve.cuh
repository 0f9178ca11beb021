// Read-out of an accumulation map: the bordered map [g][nz+2][ny+2][nx+2] to the caller's
// unpadded [g][nz][ny][nx], optionally normalised (x inv_norm[label]), one value read and
// one written per voxel and gate.  Included by the single-run and the batch interface.
#pragma once

#include <algorithm>

#include "mcx_internal.h"

namespace mcxg {

// S: the map's type, P: the type of the product with inv_norm, T: the output's type.
template <typename T, typename S, typename P>
__device__ __forceinline__ T resolved(S v, const float *inv_norm, unsigned label)
{
    P d = (P)v;
    if (inv_norm) d *= (P)__ldg(inv_norm + label);
    return (T)d;
}

// (float)(v (double)inv) in integers, from the words of v and the bits of inv and with the two
// roundings of the FP64 way: the 53 x 24-bit product to 53 bits, then to 24, each to nearest
// even.  False unless inv is positive and finite and either v is zero or v, inv and the result
// are normal.
__host__ __device__ __forceinline__ bool fp64_product_to_fp32(unsigned vhi, unsigned vlo, unsigned inv, unsigned *out)
{
    const unsigned ev = vhi >> 20 & 0x7ffu, ei = inv >> 23;                // biased by 1023 and 127
    const unsigned m = inv << 8 | 0x80000000u;                             // inv's 24 bits, in 32
    const unsigned long long lo = (unsigned long long)vlo * m;
    unsigned long long s = (vhi & 0xfffffu | 0x100000u) * (unsigned long long)m + (lo >> 32);
    unsigned rest = (unsigned)lo;                                          // product = s 2^32 + rest
    int e = (int)(ev + ei) - 1023;                                         // the result's, biased by 127
    if (s >> 52) {
        ++e;
    } else {
        s = s << 1 | rest >> 31;
        rest <<= 1;
    }
    s += ((unsigned long long)rest + 0x7fffffffu + (unsigned)(s & 1u)) >> 32;
    // a carry out of either rounding moves into the exponent
    const unsigned q = (unsigned)((s + 0xfffffffu + (unsigned)(s >> 29 & 1u)) >> 29);
    // asked of the words: asked of the 64 bits, it bounded the read-out like an FP64 comparison
    // (256 x 256 x 128, 50 gates: 1.63 ms against 1.09)
    const bool zero = (vhi << 1 | vlo) == 0u && ei < 255u;
    *out = (vhi & 0x80000000u) | (zero ? 0u : ((unsigned)(e - 1) << 23) + q);
    return zero || (ev - 1u < 2046u && ei - 1u < 254u && (unsigned)(e - 1) < 253u);
}

// FP64 -> FP32 without the FP64 pipe, whose conversions and product bounded the read-out (2
// per clock and SM), and with its results: bit for bit, also where FP32 arithmetic would flush
// the parts of a split product.  What the integer way leaves out (results outside FP32's normal
// range, infinities, NaN) takes the FP64 one.  Zeros do not: a map's empty voxels lie among the
// others, and with a way of their own nearly every warp took both (64^3, 50 gates, half of the
// voxels empty: 84 us against 53).
template <>
__device__ __forceinline__ float resolved<float, double, double>(double v, const float *inv_norm, unsigned label)
{
    const float inv = inv_norm ? __ldg(inv_norm + label) : 1.f;
    unsigned f;
    if (fp64_product_to_fp32((unsigned)__double2hiint(v), (unsigned)__double2loint(v), __float_as_uint(inv), &f))
        return __uint_as_float(f);
    return (float)(v * (double)inv);
}

// One warp per line along x, four independent elements per lane: HBM-bound (layered tissue,
// 50 gates of 256x256x128, normalised FP64 -> FP32: 3.4 GB read, 1.7 GB written).
template <typename T, typename S, typename P>
__global__ void __launch_bounds__(256)
resolve_lines(const S *map, unsigned nx, unsigned ny, unsigned lines, unsigned n_gates, unsigned pnvox,
              const uint8_t *labels, const float *inv_norm, T *out)
{
    const unsigned lane = threadIdx.x & 31u, stride = gridDim.x * 8u;
    for (unsigned g = blockIdx.y; g < n_gates; g += gridDim.y)
        for (unsigned long long l64 = blockIdx.x * 8u + (threadIdx.x >> 5); l64 < lines; l64 += stride) {
            const unsigned l = (unsigned)l64, z = l / ny, y = l - z * ny;
            const size_t first = (size_t)padded_index(0, y, z, nx, ny);
            const S *src = map + (size_t)g * pnvox + first;
            const uint8_t *lab = labels + first;
            T *dst = out + ((size_t)g * lines + l) * nx;
            for (unsigned x0 = lane; x0 < nx; x0 += 128u) {
                S v[4];
                unsigned b[4];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (x0 + 32u * k < nx) {
                        v[k] = __ldcs(src + x0 + 32u * k);
                        b[k] = inv_norm ? __ldg(lab + x0 + 32u * k) : 0u;
                    }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (x0 + 32u * k < nx) __stcs(dst + x0 + 32u * k, resolved<T, S, P>(v[k], inv_norm, b[k]));
            }
        }
}

// Lines that leave many lanes of a warp idle: E elements per thread, 256 apart.  The divisions
// for a voxel's line bound the kernel; a plain FP64 -> FP32 conversion runs beside them (33 x
// 100 x 100, 20 gates: 29 us, in integers 33).
template <typename T, typename S, typename P, int E>
__global__ void __launch_bounds__(256)
resolve_flat(const S *map, unsigned nx, unsigned ny, unsigned nvox, unsigned n_gates, unsigned pnvox,
             const uint8_t *labels, const float *inv_norm, T *out)
{
    for (unsigned g = blockIdx.y; g < n_gates; g += gridDim.y) {
        const S *src = map + (size_t)g * pnvox;
        T *dst = out + (size_t)g * nvox;
        for (unsigned long long i0 = blockIdx.x * (256ull * E) + threadIdx.x; i0 < nvox; i0 += gridDim.x * (256ull * E)) {
            S v[E];
            unsigned b[E];
#pragma unroll
            for (int k = 0; k < E; ++k)
                if (i0 + 256u * k < nvox) {
                    const unsigned i = (unsigned)i0 + 256u * k, l = i / nx, z = l / ny;
                    const unsigned pv = (unsigned)padded_index(i - l * nx, l - z * ny, z, nx, ny);
                    v[k] = __ldcs(src + pv);
                    b[k] = inv_norm ? __ldg(labels + pv) : 0u;
                }
#pragma unroll
            for (int k = 0; k < E; ++k)
                if (i0 + 256u * k < nvox)
                    __stcs(dst + i0 + 256u * k, inv_norm ? resolved<T, S, P>(v[k], inv_norm, b[k]) : (T)v[k]);
        }
    }
}

template <typename T, typename S, typename P>
cudaError_t resolve_map(const S *map, unsigned nx, unsigned ny, unsigned nz, unsigned n_gates,
                        const uint8_t *labels, const float *inv_norm, T *out, cudaStream_t st)
{
    const unsigned lines = ny * nz, nvox = lines * nx;
    const unsigned pnvox = (nx + 2) * (ny + 2) * (nz + 2);
    const unsigned gy = std::min(n_gates, 64u);
    auto blocks = [&](unsigned long long n) { return dim3((unsigned)std::max(1ull, std::min(n, 152ull * 32u / gy)), gy); };
    // A warp per line where more than 3/4 of its lanes have a voxel.  FP64 -> FP32, normalised,
    // lines / flat: nx = 24 10.6 / 8.5 us, 33 49 / 33, 48 14.7 / 12.6, 64 (50 gates) 53 / 60,
    // 66 (256 x 256, 50 gates) 1.24 / 0.89 ms, 200 57 / 73 us, 256 (128, 50 gates) 1.11 / 1.71 ms
    if (4ull * nx > 3ull * ((nx + 31ull) / 32u * 32u))
        resolve_lines<T, S, P><<<blocks((lines + 7ull) / 8u), 256, 0, st>>>(map, nx, ny, lines, n_gates, pnvox, labels,
                                                                            inv_norm, out);
    else if ((unsigned long long)nvox * n_gates > 152ull * 2u * 1024u)
        resolve_flat<T, S, P, 4><<<blocks((nvox + 1023ull) / 1024u), 256, 0, st>>>(map, nx, ny, nvox, n_gates, pnvox,
                                                                                   labels, inv_norm, out);
    else      // too few for two such blocks per SM (16 x 60 x 60, 4 gates: 5.0 us against 6.2)
        resolve_flat<T, S, P, 1><<<blocks((nvox + 255ull) / 256u), 256, 0, st>>>(map, nx, ny, nvox, n_gates, pnvox,
                                                                                 labels, inv_norm, out);
    return cudaGetLastError();
}

}  // namespace mcxg
