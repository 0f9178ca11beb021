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

// (float)(v (double)inv) in integers, from the bits of v and inv and with the two roundings of
// the FP64 way: the 53 x 24-bit product to 53 bits, then to 24, each to nearest even.  False
// (nothing written) unless v and inv are normal, inv is positive and the result is normal.
__host__ __device__ __forceinline__ bool fp64_product_to_fp32(unsigned long long v, unsigned inv, unsigned *out)
{
    const unsigned ev = (unsigned)(v >> 52) & 0x7ffu, ei = inv >> 23;      // biased by 1023 and 127
    const unsigned m = inv << 8 | 0x80000000u;                             // inv's 24 bits, in 32
    const unsigned long long lo = (unsigned long long)(unsigned)v * m;
    unsigned long long s = ((v >> 32 & 0xfffffu) | 0x100000u) * (unsigned long long)m + (lo >> 32);
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
    if (ev - 1u >= 2046u || ei - 1u >= 254u || (unsigned)(e - 1) >= 253u) return false;
    *out = ((unsigned)(v >> 32) & 0x80000000u) | (((unsigned)(e - 1) << 23) + q);
    return true;
}

// FP64 -> FP32 without the FP64 pipe, whose conversions and product bounded the read-out (2
// per clock and SM), and with its results: bit for bit, also where FP32 arithmetic would flush
// the parts of a split product.  Zeros keep FP32's 0 x inv (NaN for an infinite inv); what else
// the integer way leaves out (results outside FP32's normal range, infinities, NaN) takes the
// FP64 one.
template <>
__device__ __forceinline__ float resolved<float, double, double>(double v, const float *inv_norm, unsigned label)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const float inv = inv_norm ? __ldg(inv_norm + label) : 1.f;
    unsigned f;
    if (fp64_product_to_fp32(b, __float_as_uint(inv), &f)) return __uint_as_float(f);
    if (!(b << 1)) return __uint_as_float((unsigned)(b >> 32)) * inv;
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

// lines too short for a warp: one element per thread
template <typename T, typename S, typename P>
__global__ void __launch_bounds__(256)
resolve_flat(const S *map, unsigned nx, unsigned ny, unsigned nvox, unsigned n_gates, unsigned pnvox,
             const uint8_t *labels, const float *inv_norm, T *out)
{
    const size_t total = (size_t)nvox * n_gates, stride = (size_t)gridDim.x * blockDim.x;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += stride) {
        const unsigned v = (unsigned)(i % nvox), g = (unsigned)(i / nvox);
        const size_t pv = (size_t)padded_index(v % nx, (v / nx) % ny, v / (nx * ny), nx, ny);
        out[i] = resolved<T, S, P>(map[(size_t)g * pnvox + pv], inv_norm, labels[pv]);
    }
}

// A warp per line from 24 voxels on (3/4 of its lanes at work).
template <typename T, typename S, typename P>
cudaError_t resolve_map(const S *map, unsigned nx, unsigned ny, unsigned nz, unsigned n_gates,
                        const uint8_t *labels, const float *inv_norm, T *out, cudaStream_t st)
{
    const unsigned lines = ny * nz, nvox = lines * nx;
    const unsigned pnvox = (nx + 2) * (ny + 2) * (nz + 2);
    if (nx >= 24) {
        const unsigned gy = std::min(n_gates, 64u);
        const unsigned gx = std::max(1u, std::min((unsigned)(((unsigned long long)lines + 7) / 8), 152u * 32u / gy));
        resolve_lines<T, S, P><<<dim3(gx, gy), 256, 0, st>>>(map, nx, ny, lines, n_gates, pnvox, labels, inv_norm, out);
    } else {
        const size_t blocks = ((size_t)nvox * n_gates + 255) / 256;
        resolve_flat<T, S, P><<<(unsigned)std::max<size_t>(1, std::min<size_t>(blocks, 152u * 16u)), 256, 0, st>>>(
            map, nx, ny, nvox, n_gates, pnvox, labels, inv_norm, out);
    }
    return cudaGetLastError();
}

}  // namespace mcxg
