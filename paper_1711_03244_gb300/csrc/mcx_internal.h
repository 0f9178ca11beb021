// Internal interface between the C-ABI layer (api.cu) and the photon-walk kernels
// (walk.cu).  Not part of the public ABI.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <cuda_runtime.h>

#include "../../include/mcx.h"

namespace mcxg {

constexpr int kMaxMedia = 256;       // label values 0..255
constexpr int kMaxDetMedia = 33;     // media rows allowed when detectors are present
constexpr int kMaxDet = 64;
constexpr int kRecBase = 12;         // detected-record words before the partial paths
constexpr int kClaimChunk = 32;      // default photon ids a warp claims per global atomic
constexpr int kHot = 4;              // voxels of a pencil beam summed per warp
constexpr float kHotMaxMus = 6.f;    // largest mus h at which they are
constexpr float kC0 = 299.792458f;   // mm/ns

// device status word bits
constexpr unsigned kStatusCapped = 1u;
constexpr unsigned kStatusDetOverflow = 2u;

// Per-run constants in the walk's precision R.
template <typename R>
struct RunConsts {
    R dt;                             // gate width, ns
    R inv_dt;                         // 1 / gate width
    R t_end;                          // n_gates * gate width, ns
    R src_pos[3];                     // voxel units
    R src_dir[3];                     // unit vector
    R src_e1[3], src_e2[3];           // Gaussian launch-plane basis
    R waist;                          // voxel units
    R rr_threshold;
    R rr_m;
    R rr_inv_m;
};

// One simulation of a batch (all lengths in its own voxel units).
struct BatchSim {
    const uint8_t *labels;            // [nz][ny][nx]
    float *fluence;                   // accum 0: [n_gates][nvox]
    double *fluence64;                // accum 2: [n_gates][nvox]
    double *tally;                    // [MCX_NTALLY], FP64 atomics
    unsigned long long first;         // first flattened photon index of this simulation
    unsigned long long n_photons;
    unsigned long long seed;
    int nx, ny, nz;
    unsigned nvox;                    // voxels of the padded volume (nx+2)(ny+2)(nz+2)
    unsigned sy, sz;                  // padded strides: nx + 2, (nx + 2)(ny + 2)
    int tab0;                         // first row of this simulation in the batch tables
    int src_kind;
    float src_pos[3], src_dir[3], src_e1[3], src_e2[3], waist;
};

struct WalkParams {
    // Volumes (labels and the accumulation maps) carry a one-voxel exterior border on every
    // side ([nz+2][ny+2][nx+2]) except in the allocation-free run, whose caller-owned
    // buffers are unpadded; nvox, sy and sz describe the layout actually used.
    const uint8_t *labels;            // [nz][ny][nx] (+ border)
    float *fluence;                   // [n_gates][nvox] absorbed weight; accum 1: [n_gates][nvox][2]
                                      // compensated (hi, lo) pairs, the two words adjacent
    double *fluence64;                // accum 2: [n_gates][nvox]; accum 1: the tile's FP64 map
    int tile_lo[4];                   // accum 1: tile origin (x, y, z, gate)
    int tile_size[4];                 // accum 1: tile extent; entries = product
    const void *tab_a;                // [n_media] MedA<R>: mus, 1/mus, mua (voxel units), c0/(n h)
    const void *tab_b;                // [n_media] MedB<R>: g, 1-g^2, 1+g^2, 1/(2g)
    const void *tab_n;                // [n_media] R: refractive index
    const void *tab_tpl;              // [n_media] R: ns per voxel length, n h / c0
    const float4 *det;                // [n_det] cx, cy, cz, r^2 in voxel units
    float *det_buf;                   // [max_detected][rec_stride] words
    unsigned long long *det_count;
    unsigned long long *photon_counter;
    mcx_exit *exits;                  // [exit_log]
    double *block_tally;              // [grid][MCX_NTALLY]
    unsigned long long *block_stats;  // [grid][MCX_NSTAT]
    unsigned *status;

    int nx, ny, nz;                   // the volume's voxels (without border)
    unsigned nvox;                    // voxels per gate of the maps (with border, if any)
    unsigned sy, sz;                  // linear strides of y and z in the labels and maps
    int src_kind;
    int n_media;
    int n_det;
    int rec_stride;
    unsigned n_gates;
    float h;                          // voxel edge, mm

    // per-run constants, given in both precisions so the walk never converts in its loop
    RunConsts<float> cf;
    RunConsts<double> cd;

    unsigned long long n_photons;
    unsigned long long photon_offset;
    unsigned long long seed;
    unsigned long long max_detected;
    unsigned long long exit_log;
    unsigned long long max_events;
    int reflect;
    int claim_static;                 // 1: static per-thread photon split
    unsigned claim_chunk;             // photon ids a warp claims per global atomic (>= lanes)
    unsigned lanes, warps;            // lanes per warp and warps per block that take photons;
                                      // set at the launch
    // pencil beam: the first voxels on its ray, as indices into the map's gate 0 (n_hot = 0:
    // every deposit goes to the map)
    int n_hot;
    unsigned hot[kHot];
    const BatchSim *sims;             // batch: [n_sims], ordered by `first`
    int n_sims;
};

struct LaunchShape {
    int grid, block, blocks_per_sm, regs;
    int warps;                        // warps per block that take photons; 0: as the launch finds
    int resident;                     // blocks that the device holds at once
};

// Expected events of the longest of N photon histories in a medium (ln_n = ln N), in a volume
// of mean side L, over a path of at most max_path: photons are lost at the rate mua + pi^2 /
// (L^2 mus') per unit path (absorption, and escape by diffusion from a cube of side L: the
// slowest mode's loss rate, mus' = mus (1 - g)), so the longest of N travels about ln N / rate;
// times the events per unit path (scatterings mus and voxel crossings 1 / h).
inline double longest_history(const float *prop, double h, double L, double ln_n, double max_path)
{
    const double mua = prop[0], mus = prop[1], musp = std::max(mus * (1.0 - prop[2]), 1e-6);
    const double rate = mua + 9.8696044 / (L * L * musp);
    return std::min(ln_n / std::max(rate, 1e-9), max_path) * (mus + 1.0 / h);
}

// What the grid's rule asks of a run's volumes: their longest history (over at most 650 mm),
// whether any of them scatters (mus h >= 0.5), their largest map.
struct GridVolumes {
    double longest = 0, map_bytes = 0;
    bool scatters = false;
    void add(unsigned nx, unsigned ny, unsigned nz, double h, unsigned n_media, const float *props,
             unsigned long long n_photons, unsigned n_gates)
    {
        const double L = h * ((double)nx + ny + nz) / 3.0, ln_n = std::log(std::max((double)n_photons, 2.0));
        for (unsigned m = 1; m < n_media; ++m) {
            longest = std::max(longest, longest_history(props + 4 * m, h, L, ln_n, 650.0));
            scatters |= props[4 * m + 1] * h >= 0.5;
        }
        map_bytes = std::max(map_bytes, (double)nx * ny * nz * n_gates * sizeof(double));
    }
};
enum class GridUse { Run, Compensated, Batch, F64 };

// The grid of a run of n photons whose caller gives none: as many warps per SM as the run
// keeps busy.  A run ends with its longest histories, and in that time every resident warp
// still issues the walk for the few lanes it has left; fewer warps take more photons each,
// stay full for longer and iterate faster.  Too few leave the issue slots idle, and sooner
// where label loads and deposits go past L2.  So 8, 16 and 24 warps per SM up to so many
// photons per lane, then all 32: with a map that stays in L2, with a larger one, and for a
// batch of such maps, whose histories differ most.  (Four warps pay in the FP64 walk only, which
// a few warps keep at its rate.)  The limits hold where the longest history is many times the
// mean, and shrink
//   with a window below 3 ns (650 mm of path in tissue), which cuts the longest histories and
//   not the mean (layers, 9.1e5 photons, 0.8 ns: 6.3 ms with all warps, 6.8 ms with half);
//   where photons cross voxel after voxel without scattering: they wait for label loads, which
//   only more warps hide (64 mm cube, mus 0.1/mm, 1e6 photons: 2.47 ms at 16 warps, 1.95 at 32);
//   in the compensated mode, whose sums wait for shared memory, and in batches with the longest
//   history's length (cube, mua 2/mm, 1e6 photons, compensated: 0.82 ms at 16 warps, 0.60 at
//   32; 24 such simulations of 8e5 photons in all: 1.06 and 0.81 ms).
constexpr double kGridSmallMap[4] = {0, 3.5, 13, 26}, kGridLargeMap[4] = {0, 3.5, 6.5, 13},
                 kGridBatch[4] = {0, 10, 20, 34}, kGridF64[4] = {2.6, 3.5, 13, 26},
                 kGridCompensated[4] = {0, 3.5, 6.5, 13};
constexpr double kGridMapBytes = 128e6;
// Measured kernel times, ms, at 32 / 24 / 16 / 8 / 4 warps per SM:
//   cube        2e4  4.23 /  4.22 /  3.93 /  3.93 /  3.75    1e5   7.41 /  6.82 /  5.40 /  4.62 /  5.41
//               3e5  9.73 /  7.93 /  6.61 /  7.57 / 10.9     1e6  14.0  / 13.2  / 13.2  / 17.6
//               1e7  81.0 / 83.0  / 94.7
//   B2a         1e5  2.96 /  2.78 /  2.58 /  2.57 /  2.83    3e5   4.07 /  3.53 /  3.16 /  3.58
//               1e6  5.91 /  5.36 /  5.52                    1e7  29.3  / 30.8  / 36.7
//   layers      3e5  6.59 /  5.90 /  6.28 /  8.28            1e6  12.3  / 12.1  / 13.9
//   ellipsoids (96 mm, mus about 19/mm) 5e5  17.9 / 14.3 / 11.1 / 9.96 / 13.0
//               2e6  24.9 / 21.3 / 19.7 / 24.1               5e6  40.0 / 37.2 / 37.9 / 52.5
//   batch of 16, 6e5 photons in all  13.7 / 11.1 / 9.15 / 8.66    1.2e6  15.4 / 12.9 / 10.8 / 12.4
//               2.5e6  18.6 / 15.9 / 15.5 / 21.3                  6.2e6  31.2 / 31.9 / 34.1
inline LaunchShape walk_grid(LaunchShape s, unsigned long long n, GridUse use, const GridVolumes &v, double window_ns)
{
    if (s.blocks_per_sm < 1) return s;
    const double *limits = use == GridUse::F64 ? kGridF64 : use == GridUse::Compensated ? kGridCompensated
                         : v.map_bytes > kGridMapBytes ? kGridLargeMap
                         : use == GridUse::Batch ? kGridBatch : kGridSmallMap;
    double scale = std::min(1.0, window_ns / 3.0);
    if (use == GridUse::Batch) scale *= std::min(1.0, v.longest / 4000.0);
    else if (!v.scatters) scale *= 0.25;
    if (use == GridUse::Compensated) scale *= std::min(1.0, v.longest / 2000.0);
    const int wpb = s.block / 32, most = s.blocks_per_sm * wpb;
    const int sms = s.grid / s.blocks_per_sm, warps[5] = {4, 8, 16, 24, most};
    int k = 0;
    while (k < 4 && (double)n > scale * limits[k] * (32.0 * sms * warps[k])) ++k;
    int want = warps[k];
    if (want > most) want = most;
    const int blocks = (want + wpb - 1) / wpb;
    s.grid = sms * blocks;
    s.warps = (want + blocks - 1) / blocks;
    return s;
}

// How a run's photons are shared out: the shape's warps, 32 lanes each, and the caller's
// claim size; where there are fewer photons than those lanes, each of the shape's warps
// takes its share in fewer lanes, or (a grid of the caller's) as few warps of each block as
// hold the block's share.  Blocks beyond those that the device holds at once do not count:
// they start when the others have ended, and find nothing left (a grid of 20 000 blocks, 5e4
// photons, with its shares counted over all of them: layers 4.7 -> 14.1 ms, cube 7.1 -> 13.7).
inline unsigned sharing_blocks(const LaunchShape &s)
{
    return (unsigned)(s.resident > 0 ? std::min(s.grid, s.resident) : s.grid);
}
inline unsigned sharing_warps(const LaunchShape &s)
{
    return s.warps > 0 ? (unsigned)s.warps : (unsigned)s.block / 32u;
}
inline bool shares_photons(unsigned long long n, const LaunchShape &s)
{
    return n < 32ull * sharing_warps(s) * sharing_blocks(s);
}
inline WalkParams shared_out(WalkParams p, const LaunchShape &s)
{
    const unsigned grid = sharing_blocks(s);
    p.lanes = 32;
    p.warps = sharing_warps(s);
    if (p.claim_static || !shares_photons(p.n_photons, s)) return p;
    // at most 32 warps' worth; counted in 64 bits, since a caller's grid may be of any size
    const unsigned per_block = p.n_photons ? (unsigned)((p.n_photons + grid - 1ull) / grid) : 1u;
    if (s.warps <= 0) p.warps = (per_block + 31u) / 32u;
    p.lanes = (per_block + p.warps - 1u) / p.warps;
    p.claim_chunk = p.lanes;
    return p;
}

// Walk precision: the FP32 product path, or the same kernel in FP64 (trajectory-parity
// diagnostic; FP64 runs at a small fraction of the FP32 rate on this part).
enum class Precision { F32 = 0, F64 = 1 };

// walk.cu
size_t walk_table_bytes(Precision prec, int n_media);   // bytes of the 4 tables together
void walk_fill_tables(Precision prec, int n_media, const float *props, float h, void *host_buf,
                      const void **tab_a_off, const void **tab_b_off, const void **tab_n_off,
                      const void **tab_tpl_off);        // offsets into the buffer
// accumulation modes (mcx_run_cfg.accum_mode)
enum { kAccPlain = 0, kAccCompensated = 1, kAccF64 = 2 };
constexpr int kTileMaxEntries = 6144;  // (gate, voxel) pairs per block tile, 48 KiB

cudaError_t walk_query_shape(bool detectors, Precision prec, int accum, int block, int n_media,
                             int n_det, int tile_entries, bool claim_static, LaunchShape *shape);
cudaError_t walk_launch(const WalkParams &p, Precision prec, int accum, const LaunchShape &shape,
                        cudaStream_t stream);
// batch walk: FP32 photon state, accumulation 0 or 2, no detectors or exit log
cudaError_t walk_batch_query_shape(int accum, int block, LaunchShape *shape);
// unpadded caller-owned volume and map (allocation-free run): FP32 walk, no detectors,
// accumulation 0 or 2
cudaError_t walk_query_shape_unpadded(int accum, int block, LaunchShape *shape);
cudaError_t walk_launch_unpadded(const WalkParams &p, int accum, const LaunchShape &shape,
                                 cudaStream_t stream);
cudaError_t walk_batch_launch(const WalkParams &p, int accum, const LaunchShape &shape,
                              cudaStream_t stream);
// Gaussian launch plane of a beam along unit vector d: e1 = normalise(d x z) (x when the
// beam is along z), e2 = d x e1.
inline void launch_plane(const double d[3], double e1[3], double e2[3])
{
    if (d[2] > 0.999999 || d[2] < -0.999999) {
        e1[0] = 1; e1[1] = 0; e1[2] = 0;
    } else {
        double n1 = d[0] * d[0] + d[1] * d[1];
        n1 = n1 > 0 ? 1.0 / __builtin_sqrt(n1) : 0.0;
        e1[0] = d[1] * n1; e1[1] = -d[0] * n1; e1[2] = 0;
    }
    e2[0] = d[1] * e1[2] - d[2] * e1[1];
    e2[1] = d[2] * e1[0] - d[0] * e1[2];
    e2[2] = d[0] * e1[1] - d[1] * e1[0];
}

// The voxels that an undeflected photon of a pencil beam crosses first, for the walk to sum
// per warp in shared memory (pos in voxel units; p's volume, strides and source kind set; pad
// = 1 for the bordered layout).  Every photon deposits into them, and the L2 adds to one
// address at about 3.6e8/s: that bounds a run whose photons are short.  Photons that scatter
// often are too slow to meet it, and the test in every face step would cost them 2%, so the
// rule asks for mus h <= 6 in every tissue (B1, mus h = 1, 1e7 photons: 27.3 -> 17.8 ms;
// B2a, 1 and 5: 33.8 -> 29.4 ms; two spheres, 10 / 5 / 1, 2e7 photons, with them: 151.7 ->
// 155.6 ms).  The list decides where a sum is kept, never what is added: a photon that
// rounding or refraction takes off the ray deposits as usual.
inline void find_hot_voxels(WalkParams &p, const double pos[3], const double dir[3], unsigned pad,
                            uint32_t n_media, const float *props, float h)
{
    p.n_hot = 0;
    if (p.src_kind != 0) return;
    for (uint32_t m = 1; m < n_media; ++m)
        if (!(props[4 * m + 1] * h <= kHotMaxMus)) return;
    const int dim[3] = {p.nx, p.ny, p.nz};
    double q[3];
    int c[3];
    for (int a = 0; a < 3; ++a) {
        const float x = (float)pos[a];
        if (!(x >= 0.f) || !(x <= (float)dim[a])) return;
        const float f = __builtin_floorf(x);
        c[a] = (int)f - ((x == f && dir[a] < 0) ? 1 : 0);
        q[a] = (double)x - c[a];
    }
    while (p.n_hot < kHot) {
        for (int a = 0; a < 3; ++a)
            if (c[a] < 0 || c[a] >= dim[a]) return;
        p.hot[p.n_hot++] = ((unsigned)c[2] + pad) * p.sz + ((unsigned)c[1] + pad) * p.sy + ((unsigned)c[0] + pad);
        double l = 1e300;
        int ax = 0;
        for (int a = 0; a < 3; ++a) {
            const double d = dir[a] > 0 ? (1.0 - q[a]) / dir[a] : (dir[a] < 0 ? -q[a] / dir[a] : 1e300);
            if (d < l) { l = d; ax = a; }
        }
        for (int a = 0; a < 3; ++a) q[a] += l * dir[a];
        c[ax] += dir[ax] > 0 ? 1 : -1;
        q[ax] = dir[ax] > 0 ? 0.0 : 1.0;
    }
}

// api.cu: the error text mcx_last_error(NULL) returns (per host thread)
void set_global_error(const std::string &msg);

cudaError_t debug_uniforms(uint64_t seed, uint64_t photon, uint64_t n, float *dev_out);
cudaError_t debug_primitive(int kind, uint64_t n, const float *dev_in, float *dev_out);

// Padded volume layout: index of voxel (x, y, z) of an nx x ny volume in its bordered copy.
__host__ __device__ inline unsigned long long padded_index(unsigned x, unsigned y, unsigned z,
                                                        unsigned nx, unsigned ny)
{
    return ((unsigned long long)(z + 1) * (ny + 2) + (y + 1)) * (nx + 2) + (x + 1);
}

}  // namespace mcxg
