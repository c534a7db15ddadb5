// deck_band (csrc/terrain.cuh) on the host against the FP64 clearance penalty. Built and run by
// test_deck_band_cpu.py; the header's device functions compile as plain C++ with the few CUDA
// intrinsics they use written out below (IEEE operations; -ffp-contract=off).
//
//   deck_band_check <seed> <positions> <nodes per side> <box corner> <box side> <lowest node> <highest node> <ulps>
//
// Positions lie on a node line of the heightmap give or take <ulps> fp32 spacings (0: anywhere),
// with the clearance within 30 cm of the threshold. Prints how many were certain, how many of
// those differ from FP64 and how many of these flip the decision.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include <cuda_runtime.h>

static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __ddiv_rn(double a, double b) { return a / b; }
static inline double __dsqrt_rn(double a) { return std::sqrt(a); }
template <class T>
static inline T __ldg(const T* p) { return *p; }
template <class To, class From>
static inline To bits_of(From v) {
    To r;
    std::memcpy(&r, &v, sizeof r);
    return r;
}
static inline int __float_as_int(float v) { return bits_of<int>(v); }
static inline float __int_as_float(int v) { return bits_of<float>(v); }
static inline unsigned __float_as_uint(float v) { return bits_of<unsigned>(v); }
static inline float __uint_as_float(unsigned v) { return bits_of<float>(v); }
static inline double __hiloint2double(int hi, int lo) {
    return bits_of<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
}
template <class T>
static inline T min(T a, T b) { return a < b ? a : b; }
template <class T>
static inline T max(T a, T b) { return a > b ? a : b; }

#ifndef __noinline__
#define __noinline__
#endif
#include "terrain.cuh"

using namespace fmdp;

int main(int argc, char** argv) {
    if (argc != 9) return 2;
    const int seed = std::atoi(argv[1]), n = std::atoi(argv[2]), nodes = std::atoi(argv[3]);
    const double corner = std::atof(argv[4]), side = std::atof(argv[5]), lo = std::atof(argv[6]), hi = std::atof(argv[7]);
    const int ulps = std::atoi(argv[8]);
    std::mt19937_64 rng((uint64_t)seed);
    auto uniform = [&](double a, double b) { return a + (b - a) * (double)(rng() >> 11) * 0x1p-53; };
    std::vector<float> hm((size_t)nodes * nodes);
    for (float& h : hm) h = (float)uniform(lo, hi);
    static Model m;
    m.box[0] = corner, m.box[1] = corner + 7.3, m.box[2] = 0.0;
    m.box[3] = m.box[0] + side, m.box[4] = m.box[1] + 0.9 * side, m.box[5] = 5000.0;
    m.clearance = 60.0, m.deck = 1000.0;
    m.hm = hm.data(), m.hm_nx = m.hm_ny = nodes;
    m.hm_sx = (float)((nodes - 1) / (m.box[3] - m.box[0]));
    m.hm_sy = (float)((nodes - 1) / (m.box[4] - m.box[1]));
    const DeckGrid grid = deck_grid(m);
    long certain = 0, differ = 0, flips = 0;
    for (int i = 0; i < n; ++i) {
        double p[2];
        for (int a = 0; a < 2; ++a) {
            const double b0 = m.box[a], w = m.box[3 + a] - b0;
            p[a] = uniform(b0, b0 + w);
            // (a quarter of them on the grid's own border, where the cell is clamped)
            if (ulps > 0 && rng() % 2) {
                const int node = rng() % 4 ? (int)(rng() % nodes) : (rng() % 2 ? 0 : nodes - 1);
                p[a] = b0 + w * node / (nodes - 1);
                p[a] += uniform(-ulps, ulps) * std::fabs(p[a]) * 0x1p-23;
            }
        }
        const double z = terrain64(m, p[0], p[1]) + m.clearance + uniform(-0.3, 0.3);
        const float hx = (float)p[0], hy = (float)p[1], hz = (float)z;
        const float lx = (float)(p[0] - hx), ly = (float)(p[1] - hy), lz = (float)(z - hz);
        // the caller's fp32 position may be off by a rounding
        auto off = [&](float v) { return (rng() & 3) ? v : std::nextafter(v, (rng() & 1) ? INFINITY : -INFINITY); };
        TerrainCell t = terrain_cell(off(hx), off(hy), (float)m.box[0], (float)m.box[1], m.hm_sx, m.hm_sy, nodes, nodes);
        terrain_nodes(t, m.hm, nodes);
        const float got = deck_band(m, grid, t, hx, lx, hy, ly, hz, lz, 0);
        if (got < 0.f) continue;
        ++certain;
        const double c = z - terrain64(m, p[0], p[1]);
        const float want = c < m.clearance ? (float)(m.deck - c) : 0.f;
        differ += got != want;
        flips += (got > 0.f) != (want > 0.f);
    }
    std::printf("%ld %ld %ld\n", certain, differ, flips);
    return differ ? 1 : 0;
}
