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

// FP64 -> FP32 without the FP64 pipe, whose conversions and product bounded the read-out (2
// per clock and SM).  v = hi + lo with hi its leading 24 bits and lo the other 29 as 23 and a
// sticky bit, which rounds as they do: hi + lo is v correctly rounded.  The product with
// inv_norm keeps its rounding error (FMA) and lo's share, an error below 2^-46 before the one
// rounding.  Values outside FP32's middle range (and zeros) take the FP64 way.
template <>
__device__ __forceinline__ float resolved<float, double, double>(double v, const float *inv_norm, unsigned label)
{
    const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
    const unsigned ex = (h >> 20) & 0x7ffu;                       // biased by 1023
    const float inv = inv_norm ? __ldg(inv_norm + label) : 1.f;
    // |v| in [2^-60, 2^60), inv in [2^-60, 2^60)
    const unsigned ei = (__float_as_uint(inv) >> 23) & 0xffu;
    if (ex - (1023u - 60u) < 120u && ei - (127u - 60u) < 120u) {
        const unsigned sign = h & 0x80000000u, e8 = (ex - 896u) << 23;
        const float hi = __uint_as_float(sign | e8 | ((h & 0xfffffu) << 3) | (l >> 29));
        const unsigned r = (l & 0x1fffffffu) >> 5 | ((l & 0x1fu) ? 1u : 0u);
        const float lo = __uint2float_rn(r) * __uint_as_float(sign | (e8 - (47u << 23)));   // r 2^(ex - 1023 - 47)
        if (!inv_norm) return __fadd_rn(hi, lo);
        const float p = __fmul_rn(hi, inv);
        return __fadd_rn(p, __fmaf_rn(lo, inv, __fmaf_rn(hi, inv, -p)));
    }
    if (v == 0.0) return 0.f;
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
