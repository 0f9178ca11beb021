"""Rules that the library's host and device code share or that decide a launch, compiled for
the host and run on the CPU.  No GPU needed."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def compile_and_run(tmp_path, body):
    """Builds a host program from a body that may use the internal headers; returns its output."""
    from paper_1711_03244_gb300 import build
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text('#include "resolve.cuh"\n#include <cmath>\n#include <cstdio>\n#include <cstring>\n'
                   "#include <random>\nusing namespace mcxg;\n" + body)
    r = subprocess.run([build._nvcc(), "-O2", "-std=c++17", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                        str(src), "-o", str(exe)] + build.ARCH, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


# the read-out's integer product against the host's FP64 product and conversion: bits of every
# kind (0), factors of any size whose product is in FP32's range (1), with trailing zeros, as
# for ties (2), with a power of two and a value on or beside a midpoint of FP32 (3), and with a
# product on or beside such a midpoint (4)
@pytest.mark.parametrize("kind", range(5))
def test_readout_product_equals_fp64(tmp_path, kind):
    out = compile_and_run(tmp_path, "const int kind = %d;" % kind + r"""
int main()
{
    std::mt19937_64 r(1 + kind);
    size_t handled = 0, differ = 0, missed = 0;
    for (int k = 0; k < 10000000; ++k) {
        unsigned long long v = r();
        unsigned i = (unsigned)r();
        if (kind > 0) {
            const int ei = 1 + (int)(r() % 254), ev = (int)(r() % 256) - 2 - ei + 1023;
            v = (v & ~(0x7ffull << 52)) | ((unsigned long long)ev << 52);
            i = (i & 0x7fffffu) | (unsigned)ei << 23;
        }
        if (kind == 2) { v &= ~0ull << r() % 52; i &= ~0u << r() % 23; }
        if (kind == 3) { i &= ~0x7fffffu; v = ((v & ~0x1fffffffull) | 0x10000000ull) + r() % 3 - 1; }
        float f, want;
        double d;
        std::memcpy(&f, &i, 4);
        if (kind == 4) {
            const unsigned long long mid = 0x3ffull << 52 | (r() & 0x7fffffull) << 29 | 0x10000000ull;
            std::memcpy(&d, &mid, 8);
            d /= f;
            std::memcpy(&v, &d, 8);
            v += r() % 5 - 2;
        }
        std::memcpy(&d, &v, 8);
        want = (float)(d * (double)f);
        unsigned w, got;
        std::memcpy(&w, &want, 4);
        if (fp64_product_to_fp32((unsigned)(v >> 32), (unsigned)v, i, &got)) {
            ++handled;
            differ += got != w;
        } else {                            // left to the FP64 way: only at the ends of the range
            missed += f > 0 && std::isnormal(d) && std::isnormal(f) && std::isnormal(want) &&
                      std::fabs(want) > 0x1p-125f && std::fabs(want) < 0x1p125f;
        }
    }
    std::printf("%zu %zu %zu\n", handled, differ, missed);
    return 0;
}
""")
    handled, differ, missed = map(int, out.split())
    assert handled > (10000 if kind == 0 else 1000000) and differ == 0 and missed == 0


SHARE = r"""
static WalkParams shared(unsigned long long n, int grid, int block, int warps)
{
    LaunchShape s{};
    s.grid = grid;
    s.block = block;
    s.warps = warps;
    WalkParams p{};
    p.n_photons = n;
    p.claim_chunk = 32;
    return shared_out(p, s);
}
"""


def test_sharing_of_photons_is_in_range(tmp_path):
    """Every warp has 1 to 32 lanes and a claim for each, and those lanes hold all photons or
    are all that there are, whatever the photon count and the caller's grid: also where count
    and grid add up to more than 32 bits."""
    out = compile_and_run(tmp_path, SHARE + r"""
int main()
{
    size_t bad = 0, n_cases = 0;
    std::mt19937_64 r(1);
    const int grids[] = {1, 2, 152, 608, 4864, 20000, (1 << 24) + 1, 1 << 27, 0x7fffffff};
    const int blocks[] = {32, 64, 128, 224, 256};
    for (int grid : grids)
        for (int block : blocks)
            for (int warps = 0; warps <= block / 32; ++warps)
                for (int k = 0; k < 400; ++k) {
                    const unsigned long long edge[] = {0, 1, 1ull << 32, (1ull << 32) - grid, (1ull << 32) - grid + 1,
                                                       32ull * grid, 32ull * grid * (block / 32) - 1};
                    const unsigned long long n = k < 7 ? edge[k] : r() >> (20 + r() % 44);
                    const WalkParams p = shared(n, grid, block, warps);
                    const unsigned wpb = block / 32;
                    const bool range = p.warps >= 1 && p.warps <= wpb && p.lanes >= 1 && p.lanes <= 32 &&
                                       p.claim_chunk >= p.lanes && (warps == 0 || (int)p.warps == warps);
                    const bool all = (unsigned long long)p.warps * p.lanes * grid >= n ||
                                     (p.lanes == 32 && p.warps == (warps ? (unsigned)warps : wpb));
                    ++n_cases;
                    bad += !(range && all);
                }
    std::printf("%zu %zu\n", n_cases, bad);
    return 0;
}
""")
    cases, bad = map(int, out.split())
    assert cases > 50000 and bad == 0


def test_sharing_ignores_blocks_that_wait(tmp_path):
    """A grid of more blocks than the device holds shares photons out as one that just fills
    it; a smaller one by its own blocks."""
    out = compile_and_run(tmp_path, r"""
int main()
{
    size_t bad = 0;
    for (int block : {32, 64, 256})
        for (unsigned long long n = 0; n < 300000; n += 1 + n / 50)
            for (int grid : {1, 100, 607, 608, 609, 2000, 20000, 0x7fffffff}) {
                LaunchShape s{}, t{};
                s.block = t.block = block;
                s.resident = t.resident = 608;
                s.grid = grid;
                t.grid = grid < 608 ? grid : 608;
                WalkParams p{};
                p.n_photons = n;
                p.claim_chunk = 32;
                const WalkParams a = shared_out(p, s);
                t.resident = 0;
                const WalkParams b = shared_out(p, t);
                bad += a.warps != b.warps || a.lanes != b.lanes || a.claim_chunk != b.claim_chunk;
            }
    std::printf("%zu\n", bad);
    return 0;
}
""")
    assert int(out) == 0


def test_grid_rule(tmp_path):
    """The grid of a run whose caller gives none: within what the device holds, of warps that a
    block has, never smaller for more photons, and all of it from some count on; for every use,
    block size, map, medium and window."""
    out = compile_and_run(tmp_path, r"""
int main()
{
    size_t bad = 0, cases = 0, steps = 0;
    const float media[][4] = {{2.f, 5.f, 0.5f, 1.37f}, {0.01f, 10.f, 0.9f, 1.37f}, {0.01f, 0.1f, 0.9f, 1.37f},
                              {0.f, 0.f, 0.f, 1.f}, {0.f, 20.f, 0.f, 1.4f}};
    for (GridUse use : {GridUse::Run, GridUse::Compensated, GridUse::Batch, GridUse::F64})
        for (int block : {32, 64, 96, 128, 224, 256})
            for (int per_sm : {1, 2, 1024 / block})
                for (auto &m : media)
                    for (unsigned gates : {1u, 100000u})
                        for (double window : {1e-6, 0.1, 2.9, 5.0, 1e6}) {
                            int last = 0;
                            for (unsigned long long n = 0; n < (1ull << 40); n = 2 * n + 1 + n / 3) {
                                const float props[8] = {0, 0, 1, 1, m[0], m[1], m[2], m[3]};
                                GridVolumes v;
                                v.add(64, 60, 50, 1.0, 2, props, n, gates);
                                LaunchShape s{};
                                s.block = block;
                                s.blocks_per_sm = per_sm;
                                s.grid = s.resident = 152 * per_sm;
                                const LaunchShape t = walk_grid(s, n, use, v, window);
                                const int warps = t.warps * t.grid;
                                bad += t.grid < 152 || t.grid > s.grid || t.grid % 152 || t.warps < 1 ||
                                       t.warps > block / 32 || t.block != block || warps < last;
                                steps += warps > last;
                                last = warps;
                                ++cases;
                            }
                            bad += last != 152 * per_sm * (block / 32);
                        }
    std::printf("%zu %zu %zu\n", cases, steps, bad);
    return 0;
}
""")
    cases, steps, bad = map(int, out.split())
    assert bad == 0 and cases > 50000 and steps > 5000
