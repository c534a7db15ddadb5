// FastMDP rollout with a lookahead window of W sub-steps (sm_103a).
//
// Sec. IV "Forward project" holds each action for W time steps of dt (the paper runs
// W = 10 at dt = 0.1 s), and the compute-value kernel (Alg. 9) keeps, per action, the
// largest value met along those W projected states. The state then advances by one step
// of dt to the chosen action's first projected state (Alg. 1, Delta_1). Here:
//   x_1 = s + move(a), x_j = x_(j-1) + move(a) (FP64, rounded at each sub-step);
//   value(x_j) = goal term - aggregate of the wells of the plans present at t + j (their
//                sample at t + j, velocity from t + j to t + j + 1) - hard-deck penalty;
//   Q(a) = max over j with x_j inside the box; a is valid when x_1 is inside.
//
// One CTA per request, 256 or 512 threads. A step is a chain of four short phases with a barrier after
// each; no unit is busy, so what counts is the length of each phase's instruction stream:
//   1. side by side: the projected states per (action, sub-step) with box test, goal terms as a
//      log2 offset from the goal term at s (from the exact identity d - d_s =
//      (|o|^2 - 2 G.o) / (d + d_s), G = goal - s, o the offset, which keeps fp32 accurate to
//      micrometres at any distance) and static wells; and a list of the plan samples (and, in
//      a co-simulation, the other aircraft) with a well that can reach a projected state,
//      collected by the other warps from the table's slices or from the spatial index;
//   2. the list's samples, shared out between the warps, lanes = actions: wells in fp32, d < R
//      in FP64 inside its band;
//   3. penalty and clearance per (action, sub-step): the W values g - N as (sign, log2 |g - N|),
//      so that a large penalty at one sub-step leaves the goal term's resolution at the others;
//   4. one warp: the best value per action, argmax (lowest index on ties), near-tie record,
//      exact FP64 advance, terminal tests.
// On GB300: 60 plans and W = 10, 8.1 us per step with every pair scored by the warp that found
// it and seven barriers, 5.3 us now; a co-simulation of 128 aircraft among 3000 plans, 23 us per
// step with every slot read and a grid barrier, 6.6 us now.
// Every decision that is a threshold (box, well radius, clearance, capture) is taken in
// FP64 with the oracle's operation order wherever fp32 could be on the wrong side.
#include <climits>
#include <cmath>

#include "fmdp_internal.cuh"
#include "terrain.cuh"

namespace fmdp {

namespace {

constexpr unsigned kFullMask = 0xffffffffu;

constexpr int kLookList = 1024;  // samples the list of a step holds (more are scored where they are found)

// A sample whose wells `wells` may reach a projected state of sub-step j: offset from s, velocity.
struct LookItem {
    float qx, qy, qz;
    int what;  // wells | j << 16 | kind << 24
    float vx, vy, vz;
    int ref;   // slot, index item (within the row) or aircraft
};
enum { kLookSlot, kLookIndex, kLookMember };

struct LookLayout {
    size_t ox, oy, oz, inb, rel, vsg, vlv, cmp, vls, keys, sums, stat, Dx, Dy, Dz, Dh, Dz2, list, misc, total;
};

__host__ __device__ inline LookLayout look_layout(int A, int W) {
    LookLayout L;
    const size_t AW = (size_t)A * W;
    size_t o = 0;
    auto al = [&](size_t a) { o = (o + a - 1) & ~(a - 1); };
    L.ox = o; o += AW * 4;    // offsets of the projected states from s (fp32)
    L.oy = o; o += AW * 4;
    L.oz = o; o += AW * 4;
    L.inb = o; o += AW * 4;   // projected state inside the box
    L.rel = o; o += AW * 4;   // log2 of the goal term at x_j minus log2 of the goal term at s
    L.vsg = o; o += AW * 4;   // value g - N at x_j: sign class (2 bits) and whether vlv is absolute
    L.vlv = o; o += AW * 4;   // log2 |g - N| (relative to n0, or absolute when penalty dominated)
    L.vls = o; o += AW * 4;   // log2 of the term scale max(g, N) relative to n0
    L.keys = o; o += AW * 4;  // float keys of the largest well log-value (MAX)
    al(8);
    L.cmp = o; o += AW * 8;   // what orders the values: class, log2 |g - N| relative to n0 (signed)
    L.sums = o; o += AW * 8;  // fixed-point sums of well values (SUM)
    L.stat = o; o += (size_t)kMaxStatic * 3 * 4;  // static-well centres minus s (fp32)
    al(16);
    L.Dx = o; o += kHeadings * 8;    // exact moves per heading (FP64)
    L.Dy = o; o += kHeadings * 8;
    L.Dz = o; o += kMaxActions * 8;  // exact climb per action (FP64)
    L.Dh = o; o += kHeadings * 4 * 4;     // the moves as double-float: xh, xl, yh, yl per heading
    L.Dz2 = o; o += kMaxActions * 2 * 4;  // climb as double-float
    al(16);
    L.list = o; o += kLookList * sizeof(LookItem);  // (then LookState, 16-byte aligned)
    L.misc = o; o += 1024;
    L.total = (o + 127) & ~size_t(127);
    return L;
}

// Per-step shared scalars.
struct LookState {
    double s[3];      // exact state
    double prev[3];   // state one step earlier (co-simulation velocity)
    double step, cap2;
    float shx, shy, shz, slx, sly, slz;  // s as double-float
    float Ghx, Ghy, Ghz, Glx, Gly, Glz;  // goal - s as double-float
    float phi;                           // log2 g(s) - n0
    // the step's number (co-simulation) and the step: written a barrier ahead of the step, because
    // its first phase already scores samples (those the list cannot take)
    int64_t step_no, t;
    int n0;                              // integer part of log2 of the goal term at s
    int h, k, done, status, near_ties;
    int tie_k, tie_a1, tie_a2;  // near-tie test of step tie_k still to do (tie_k < 0: none)
    int tie_n0;
    int tie_sg[kMaxActions];     // per action: sign class of Q (-1, 0, 1), -2 invalid
    float tie_T[kMaxActions];    // ... log2 of the term scale max(g, N), relative to tie_n0
    double tie_L[kMaxActions];   // ... log2 |Q|
    int64_t row0;     // ring row of t + 1 for the current step
    int n_list;       // samples found in this step (may exceed kLookList)
    int late;         // co-simulation: a wait for another aircraft's record expired
    alignas(16) float well[kMaxWells][4];  // tau, R^2, log2 gamma, log2 |r|
    float band[kMaxWells];
    float reach[kMaxWells];    // R
};
static_assert(sizeof(LookState) <= 1024, "see look_layout");

// Co-simulation: an aircraft's state at one step, as six 16-byte words {value, stamp}. The stamp
// (2 x last step it holds for, + 1 when flying) is in every word and a word is read and written
// as one access, so a reader needs no fence: it reads until every stamp is at least its step's.
// Two records per aircraft, by step parity: the one of step t is overwritten for step t + 2,
// by then every other aircraft has published step t + 1, so it has read step t.
struct LookRecord {
    double v[6];  // x, y, z, vx, vy, vz
    bool flying;
};
constexpr int64_t kStampForever = INT64_MAX / 4;
__device__ __forceinline__ void put_word(double* p, double v, int64_t stamp) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(__double_as_longlong(v)), "l"(stamp)
                 : "memory");
}
__device__ __forceinline__ int64_t get_word(const double* p, double& v) {
    long long x, stamp;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(x), "=l"(stamp)
                 : "l"(p)
                 : "memory");
    v = __longlong_as_double(x);
    return stamp;
}
// reads record p, once it holds for step `step` (counted from 1); false after about a second
__device__ __forceinline__ bool look_read(const double* p, int64_t step, LookRecord& r, bool patient) {
    const long long t0 = clock64();
    for (;;) {
        int64_t least = INT64_MAX;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const int64_t stamp = get_word(p + 2 * i, r.v[i]);
            least = min(least, stamp);
            if (i == 0) r.flying = stamp & 1;
        }
        if ((least >> 1) >= step) return true;
        if (clock64() - t0 > (1ll << 31)) return false;
        if (patient) __nanosleep(200);
    }
}

__device__ __forceinline__ unsigned long long look_sum_term(float l, float ref) {
    const float t = exp2f(l - ref) * kSumUnits;  // fixed point, 2^-kSumBits of the largest |r|
    return (unsigned long long)__float2ull_rn(t);
}

// |G|^2 of a double-float G as a double-float, and its fp32 root
__device__ __forceinline__ float lk_goal_dist(float Ghx, float Ghy, float Ghz, float Glx, float Gly, float Glz, float& Sh,
                                              float& Sl) {
    const float p0 = Ghx * Ghx, p1 = Ghy * Ghy, p2 = Ghz * Ghz;
    const float e0 = fmaf(Ghx, Ghx, -p0), e1 = fmaf(Ghy, Ghy, -p1), e2 = fmaf(Ghz, Ghz, -p2);
    float s1, t1, s2, t2;
    two_sum(p0, p1, s1, t1);
    two_sum(s1, p2, s2, t2);
    const float lo = t1 + t2 + e0 + e1 + e2 + 2.f * (Ghx * Glx + Ghy * Gly + Ghz * Glz);
    fast_two_sum(s2, lo, Sh, Sl);
    return Sh > 0.f ? sqrtf(Sh) : 0.f;
}
// log2 of the goal term |r_g| gamma^|G| at a state whose goal vector is the double-float G,
// split as n0 (integer) + phi (fraction in [0, 1))
__device__ __forceinline__ void lk_goal_log(const Model& m, float Ghx, float Ghy, float Ghz, float Glx, float Gly,
                                            float Glz, int& n0, float& phi) {
    const float lg_hi = (float)m.lg64, lg_lo = (float)(m.lg64 - (double)(float)m.lg64);
    const float l2r_hi = (float)m.log2rg, l2r_lo = (float)(m.log2rg - (double)(float)m.log2rg);
    float Sh, Sl;
    const float rt = lk_goal_dist(Ghx, Ghy, Ghz, Glx, Gly, Glz, Sh, Sl);
    const float rr = fmaf(-rt, rt, Sh);
    const float rl = rt > 0.f ? (rr + Sl) * (0.5f / rt) : 0.f;
    const float p = rt * lg_hi;
    const float pe = fmaf(rt, lg_hi, -p);
    const float lo2 = pe + rt * lg_lo + rl * lg_hi;
    float Lh, Le;
    two_sum(p, l2r_hi, Lh, Le);
    Le = Le + (lo2 + l2r_lo);
    float LH, LL;
    fast_two_sum(Lh, Le, LH, LL);
    float fl = floorf(LH);
    float fr = (LH - fl) + LL;
    if (fr >= 1.f) { fr -= 1.f; fl += 1.f; }
    if (fr < 0.f) { fr += 1.f; fl -= 1.f; }
    n0 = (int)fl;
    phi = fr;
}

// The exact FP64 projected state x_(j+1) of a move (Dxa, Dya, Dza) from s: j + 1 rounded
// additions, as the oracle forms it. Called only where an fp32 decision falls in its band.
__device__ __noinline__ void look_state_exact(const double* s, double Dxa, double Dya, double Dza, int j, double& x,
                                              double& y, double& z) {
    x = s[0];
    y = s[1];
    z = s[2];
    for (int i = 0; i <= j; ++i) {
        x = __dadd_rn(x, Dxa);
        y = __dadd_rn(y, Dya);
        z = __dadd_rn(z, Dza);
    }
}

// d < R for a plan well, in FP64 with the oracle's order of operations (no FMA).
__device__ __noinline__ bool look_well_exact(const Model& m, int w, const double* s, double Dxa, double Dya, double Dza,
                                             int j, float p1x, float p1y, float p1z, float p2x, float p2y, float p2z,
                                             bool has2) {
    double x, y, z;
    look_state_exact(s, Dxa, Dya, Dza, j, x, y, z);
    double vx = 0.0, vy = 0.0, vz = 0.0;
    if (has2) {
        vx = __ddiv_rn(__dsub_rn((double)p2x, (double)p1x), m.dt);
        vy = __ddiv_rn(__dsub_rn((double)p2y, (double)p1y), m.dt);
        vz = __ddiv_rn(__dsub_rn((double)p2z, (double)p1z), m.dt);
    }
    const double tau = m.w_tau64[w];
    const double cx = __dadd_rn((double)p1x, __dmul_rn(tau, vx));
    const double cy = __dadd_rn((double)p1y, __dmul_rn(tau, vy));
    const double cz = __dadd_rn((double)p1z, __dmul_rn(tau, vz));
    return norm3_64(__dsub_rn(x, cx), __dsub_rn(y, cy), __dsub_rn(z, cz)) < m.w_R64[w];
}

// d < R for a well of another aircraft of a co-simulated batch: centre = s_m + tau * v_m.
__device__ __noinline__ bool look_member_exact(const Model& m, int w, const double* s, double Dxa, double Dya,
                                               double Dza, int j, double sx, double sy, double sz, double vx,
                                               double vy, double vz) {
    double x, y, z;
    look_state_exact(s, Dxa, Dya, Dza, j, x, y, z);
    const double tau = m.w_tau64[w];
    const double cx = __dadd_rn(sx, __dmul_rn(tau, vx));
    const double cy = __dadd_rn(sy, __dmul_rn(tau, vy));
    const double cz = __dadd_rn(sz, __dmul_rn(tau, vz));
    return norm3_64(__dsub_rn(x, cx), __dsub_rn(y, cy), __dsub_rn(z, cz)) < m.w_R64[w];
}

__device__ __noinline__ bool look_static_exact(const Model& m, int w, const double* s, double Dxa, double Dya,
                                               double Dza, int j) {
    double x, y, z;
    look_state_exact(s, Dxa, Dya, Dza, j, x, y, z);
    const double* c = m.statics + 6 * w;
    return norm3_64(__dsub_rn(x, c[0]), __dsub_rn(y, c[1]), __dsub_rn(z, c[2])) < c[3];
}

__device__ __noinline__ float look_deck_exact(const Model& m, const double* s, double Dxa, double Dya, double Dza,
                                              int j) {
    double x, y, z;
    look_state_exact(s, Dxa, Dya, Dza, j, x, y, z);
    const double c = __dsub_rn(z, terrain64(m, x, y));
    return c < m.clearance ? (float)__dsub_rn(m.deck, c) : 0.f;
}

__device__ __noinline__ bool look_box_exact(const Model& m, const double* s, double Dxa, double Dya, double Dza,
                                            int j) {
    double x, y, z;
    look_state_exact(s, Dxa, Dya, Dza, j, x, y, z);
    return x >= m.box[0] && x <= m.box[3] && y >= m.box[1] && y <= m.box[4] && z >= m.box[2] && z <= m.box[5];
}

__device__ __noinline__ bool look_capture_exact(const double* s, const fmdp_request& req, double cap2) {
    const double ex = __dsub_rn(req.gx, s[0]), ey = __dsub_rn(req.gy, s[1]), ez = __dsub_rn(req.gz, s[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) <= cap2;
}

// Monotone 64-bit argmax key of a value held as (sign class, log2 |Q|): valid keys are > 0,
// Q > 0 above Q = 0 above Q < 0, and within a class ordered by Q (two low bits of log2 |Q|
// dropped).
__device__ __forceinline__ unsigned long long look_key(int sg, double L) {
    unsigned long long u = (unsigned long long)__double_as_longlong(L);
    u = (u >> 63) ? ~u : (u | 0x8000000000000000ull);  // increasing in L
    if (sg > 0) return (3ull << 62) | (u >> 2);
    if (sg == 0) return 2ull << 62;
    return (1ull << 62) | ((~u) >> 2);  // larger |Q| is a worse negative value
}

// Near-tie test of the two best actions from their (sign, log2 |Q|) and log2 scales:
// (Q1 - Q2) < 1e-4 * max(|Q1|, |Q2|, T1, T2), evaluated in the log domain.
__device__ __noinline__ bool look_near_tie(int s1, double L1, double T1, int s2, double L2, double T2) {
    double M = fmax(T1, T2);
    if (s1 != 0) M = fmax(M, L1);
    if (s2 != 0) M = fmax(M, L2);
    double gap;  // log2 (Q1 - Q2)
    if (s1 == s2) {
        if (s1 == 0) return true;
        const double hi = s1 > 0 ? L1 : L2, lo = s1 > 0 ? L2 : L1;  // Q1 >= Q2
        if (hi == lo) return true;
        gap = hi + (double)log2f(1.f - exp2f((float)(lo - hi)));
    } else if (s1 > 0 && s2 < 0) {
        const double hi = fmax(L1, L2), lo = fmin(L1, L2);
        gap = hi + (double)log2f(1.f + exp2f((float)(lo - hi)));
    } else {
        gap = s1 == 0 ? L2 : L1;  // one of them is zero
    }
    return gap < M - 13.287712379549449;  // log2(1e-4)
}

// Scores one sample (the same in every lane) for every action (lanes) at its sub-step. hn, Dxy,
// Dzf: the lane's heading after its turn and its move. Two wells at a time, without branches but
// for the band: a sample with five wells took 1500 cycles well by well, most of them waiting for
// one square root after the other.
struct LookScore {
    const LookState* st;
    int* keys;
    unsigned long long* sums;
    const double *Dx, *Dy, *Dz;
};
// d < R for one well of a sample whose edge lies in the fp32 band
__device__ __noinline__ bool look_band(const LookArgs& a, const LookScore& c, const LookItem& it, int w, int hn) {
    const Model& m = a.m;
    const LookState* st = c.st;
    const int lane = threadIdx.x & 31, j = (it.what >> 16) & 0xff, kind = it.what >> 24;
    bool in;
    if (kind == kLookMember) {
        const double* rc = a.mem + ((size_t)(st->step_no & 1) * a.n_req + it.ref) * 12;
        double v[6];
        for (int i = 0; i < 6; ++i) get_word(rc + 2 * i, v[i]);
        in = look_member_exact(m, w, st->s, c.Dx[hn], c.Dy[hn], c.Dz[lane], j, v[0], v[1], v[2], v[3], v[4], v[5]);
    } else {
        int64_t r1 = st->row0 + j;
        r1 -= r1 >= a.tab.T_win ? a.tab.T_win : 0;
        float4 P1, P2;
        if (kind == kLookIndex) {
            const float4* p = a.iv.items + ((size_t)r1 * a.tab.S_pad + it.ref) * 2;
            P1 = __ldcg(p);
            P2 = __ldcg(p + 1);
        } else {
            const size_t o1 = (size_t)r1 * a.tab.S_pad + it.ref;
            P1 = make_float4(a.tab.X[o1], a.tab.Y[o1], a.tab.Z[o1], 0.f);
            P2 = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
            if (st->t + j + 2 < a.tab.t_base + a.tab.T_win) {
                const int64_t r2 = r1 + 1 >= a.tab.T_win ? 0 : r1 + 1;
                const size_t o2 = (size_t)r2 * a.tab.S_pad + it.ref;
                P2 = make_float4(a.tab.X[o2], a.tab.Y[o2], a.tab.Z[o2], 0.f);
            }
        }
        in = look_well_exact(m, w, st->s, c.Dx[hn], c.Dy[hn], c.Dz[lane], j, P1.x, P1.y, P1.z, P2.x, P2.y, P2.z,
                             P2.x == P2.x);
    }
    return in;
}
__device__ __forceinline__ void look_score(const LookArgs& a, const LookScore& c, const LookItem& it, int hn, float4 Dxy,
                                           float2 Dzf) {
    const Model& m = a.m;
    const int lane = threadIdx.x & 31;
    if (lane >= m.A) return;
    const int j = (it.what >> 16) & 0xff;
    const float fj = (float)(j + 1);
    const float px = fmaf(fj, Dxy.x, fj * Dxy.y), py = fmaf(fj, Dxy.z, fj * Dxy.w), pz = fmaf(fj, Dzf.x, fj * Dzf.y);
    float mb = -INFINITY;
    unsigned long long sb = 0ull;
    unsigned bands = 0u;
    auto one = [&](int w, bool on) {
        const float4 k = *reinterpret_cast<const float4*>(c.st->well[w]);
        const float ux = px - fmaf(k.x, it.vx, it.qx), uy = py - fmaf(k.x, it.vy, it.qy), uz = pz - fmaf(k.x, it.vz, it.qz);
        const float d2 = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
        const bool band = fabsf(d2 - k.y) <= c.st->band[w];
        const bool in = on && !band && d2 < k.y;
        const float l = fmaf(sqrtf(d2), k.z, k.w);
        mb = fmaxf(mb, in ? l : -INFINITY);
        if (m.combine && in) sb += look_sum_term(l, m.sum_ref);
        bands |= on && band ? 1u << w : 0u;
    };
    for (unsigned left = (unsigned)it.what & 0xffffu; left;) {
        const int w0 = __ffs(left) - 1;
        left &= left - 1u;
        const int w1 = left ? __ffs(left) - 1 : w0;
        one(w0, true);
        one(w1, left != 0u);
        left &= left - 1u;
    }
    for (; bands; bands &= bands - 1u) {  // (rare)
        const int w = __ffs(bands) - 1;
        if (!look_band(a, c, it, w, hn)) continue;
        const float4 k = *reinterpret_cast<const float4*>(c.st->well[w]);
        const float ux = px - fmaf(k.x, it.vx, it.qx), uy = py - fmaf(k.x, it.vy, it.qy), uz = pz - fmaf(k.x, it.vz, it.qz);
        const float l = fmaf(sqrtf(fmaf(ux, ux, fmaf(uy, uy, uz * uz))), k.z, k.w);
        mb = fmaxf(mb, l);
        if (m.combine) sb += look_sum_term(l, m.sum_ref);
    }
    const int q = lane * a.W + j;
    if (mb > -INFINITY) atomicMax(&c.keys[q], float_key(mb));
    if (sb) atomicAdd(&c.sums[q], sb);
}
__device__ __noinline__ void look_score_over(const LookArgs& a, const LookScore& c, const LookItem& it, int hn, float4 Dxy,
                                             float2 Dzf) {
    look_score(a, c, it, hn, Dxy, Dzf);
}

}  // namespace

size_t lookahead_smem_bytes(int A, int W) { return look_layout(A, W).total; }

// NT 512: sixteen warps share out a step's samples and its projected states, one CTA per SM; 256 (for
// co-simulations, which all have to be resident): two CTAs per SM. Both leave 128 registers a thread;
// some 120 bytes of a thread's state are spilled.
template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) lookahead_kernel(const __grid_constant__ LookArgs a) {
    extern __shared__ __align__(128) unsigned char lsm[];
    const Model& m = a.m;
    const int A = m.A, W = a.W, AW = A * W;
    const LookLayout L = look_layout(A, W);
    float* ox = reinterpret_cast<float*>(lsm + L.ox);
    float* oy = reinterpret_cast<float*>(lsm + L.oy);
    float* oz = reinterpret_cast<float*>(lsm + L.oz);
    int* inb = reinterpret_cast<int*>(lsm + L.inb);
    float* rel = reinterpret_cast<float*>(lsm + L.rel);
    int* vsg = reinterpret_cast<int*>(lsm + L.vsg);
    float* vlv = reinterpret_cast<float*>(lsm + L.vlv);
    float* vls = reinterpret_cast<float*>(lsm + L.vls);
    int* keys = reinterpret_cast<int*>(lsm + L.keys);
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(lsm + L.sums);
    float* stc = reinterpret_cast<float*>(lsm + L.stat);
    double* Dx = reinterpret_cast<double*>(lsm + L.Dx);
    double* Dy = reinterpret_cast<double*>(lsm + L.Dy);
    double* Dz = reinterpret_cast<double*>(lsm + L.Dz);
    float* Dh = reinterpret_cast<float*>(lsm + L.Dh);    // [24][4]: xh, xl, yh, yl
    float* Dz2 = reinterpret_cast<float*>(lsm + L.Dz2);  // [32][2]: zh, zl
    float2* cmp = reinterpret_cast<float2*>(lsm + L.cmp);
    LookItem* list = reinterpret_cast<LookItem*>(lsm + L.list);
    LookState* st = reinterpret_cast<LookState*>(lsm + L.misc);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wi = blockIdx.x;
    if (wi >= a.n_req || (a.n_dev && wi >= *a.n_dev)) return;
    const int r = a.idx ? a.idx[wi] : wi;
    const fmdp_request req = a.reqs[r];
    float* traj = a.traj + (size_t)r * a.cap * 3;
    uint8_t* acts = a.acts + (size_t)r * a.cap;
    const int KEY_NONE = float_key(-INFINITY);
    const float inv_dt = (float)(1.0 / m.dt);
    const int S = a.S_scan;
    double* q_trace = a.trace ? a.q_trace + (size_t)r * a.cap * A : nullptr;
    double* st_trace = a.trace ? a.st_trace + (size_t)r * a.cap * 3 : nullptr;
    int32_t* hd_trace = a.trace ? a.hd_trace + (size_t)r * a.cap : nullptr;
    uint8_t* tie_trace = a.trace ? a.tie_trace + (size_t)r * a.cap : nullptr;
    // near-tie flag of a finished step, taken off the step's chain (one thread)
    auto deferred_tie = [&]() {
        if (st->tie_k < 0) return;
        bool tie = false;
        if (st->tie_a1 >= 0 && st->tie_a2 >= 0)
            tie = look_near_tie(st->tie_sg[st->tie_a1], st->tie_L[st->tie_a1],
                                __dadd_rn((double)st->tie_n0, (double)st->tie_T[st->tie_a1]), st->tie_sg[st->tie_a2],
                                st->tie_L[st->tie_a2], __dadd_rn((double)st->tie_n0, (double)st->tie_T[st->tie_a2]));
        if (a.trace) tie_trace[st->tie_k] = tie ? 1 : 0;
        st->near_ties += tie ? 1 : 0;
        st->tie_k = -1;
    };
    const float box0 = (float)m.box[0], box1 = (float)m.box[1], box2 = (float)m.box[2];
    const float box3 = (float)m.box[3], box4 = (float)m.box[4], box5 = (float)m.box[5];
    constexpr float kBoxBandL = 0.01f;  // metres from a box face: decided in FP64
    constexpr float kCapBandL = 0.5f;   // metres around the capture radius: decided in FP64

    // ---- prologue: heading table (the bearing turned by k * 15 degrees), climb moves
    if (tid < kHeadings) {
        const double dx = __dsub_rn(req.gx, req.ox), dy = __dsub_rn(req.gy, req.oy);
        const double Lh = __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
        double c0 = 1.0, s0 = 0.0;
        if (Lh > 0.0) {
            c0 = __ddiv_rn(dx, Lh);
            s0 = __ddiv_rn(dy, Lh);
        }
        double ck, sk;
        unit15(tid, ck, sk);
        const double C = __dsub_rn(__dmul_rn(c0, ck), __dmul_rn(s0, sk));
        const double Sn = __dadd_rn(__dmul_rn(s0, ck), __dmul_rn(c0, sk));
        const double step = __dmul_rn(req.speed_mps, m.dt);
        const double X = __dmul_rn(step, C), Y = __dmul_rn(step, Sn);
        Dx[tid] = X;
        Dy[tid] = Y;
        const float xh = (float)X, yh = (float)Y;
        Dh[4 * tid] = xh;
        Dh[4 * tid + 1] = (float)__dsub_rn(X, (double)xh);
        Dh[4 * tid + 2] = yh;
        Dh[4 * tid + 3] = (float)__dsub_rn(Y, (double)yh);
    }
    if (tid < kMaxActions) {
        const double dz = tid < A ? __dmul_rn(m.climb[tid], m.dt) : 0.0;
        Dz[tid] = dz;
        const float zh = (float)dz;
        Dz2[2 * tid] = zh;
        Dz2[2 * tid + 1] = (float)__dsub_rn(dz, (double)zh);
    }
    if (tid == 0) {
        st->s[0] = req.ox;
        st->s[1] = req.oy;
        st->s[2] = req.oz;
        st->h = 0;
        st->k = 0;
        st->n_list = 0;
        st->late = 0;
        st->near_ties = 0;
        st->tie_k = -1;
        st->step = __dmul_rn(req.speed_mps, m.dt);
        st->cap2 = __dmul_rn(st->step, st->step);
        traj[0] = (float)req.ox;
        traj[1] = (float)req.oy;
        traj[2] = (float)req.oz;
        st->prev[0] = req.ox;
        st->prev[1] = req.oy;
        st->prev[2] = req.oz;
        const double s0[3] = {req.ox, req.oy, req.oz}, g0[3] = {req.gx, req.gy, req.gz};
        float* sh = &st->shx;
        float* sl = &st->slx;
        float* gh = &st->Ghx;
        float* gl = &st->Glx;
        for (int c = 0; c < 3; ++c) {
            sh[c] = (float)s0[c];
            sl[c] = (float)__dsub_rn(s0[c], (double)sh[c]);
            const double G = __dsub_rn(g0[c], s0[c]);
            gh[c] = (float)G;
            gl[c] = (float)__dsub_rn(G, (double)gh[c]);
        }
        st->t = req.depart_step;
        st->step_no = req.depart_step - a.t_start + 1;
        int64_t row = (req.depart_step + 1) % a.tab.T_win;
        st->row0 = row < 0 ? row + a.tab.T_win : row;
        if (a.trace) {
            st_trace[0] = req.ox;
            st_trace[1] = req.oy;
            st_trace[2] = req.oz;
            hd_trace[0] = 0;
        }
        const double ex = __dsub_rn(req.gx, req.ox), ey = __dsub_rn(req.gy, req.oy), ez = __dsub_rn(req.gz, req.oz);
        const bool cap0 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) <= st->cap2;
        st->done = cap0 || req.horizon <= 0;
        st->status = cap0 ? kStatusCaptured : FMDP_REJ_HORIZON;
    }
    if (tid < m.n_wells) {
        st->well[tid][0] = m.w_tau[tid];
        st->well[tid][1] = m.w_R2[tid];
        st->well[tid][2] = m.w_lg[tid];
        st->well[tid][3] = m.w_L[tid];
        st->band[tid] = m.w_band[tid];
        st->reach[tid] = sqrtf(m.w_R2[tid]);
    }
    for (int q = tid; q < AW; q += NT) {
        keys[q] = KEY_NONE;
        sums[q] = 0ull;
    }
    __syncthreads();
    // largest horizontal + vertical move of one sub-step (culling bound)
    float lstep = 0.f;
    for (int q = 0; q < A; ++q) lstep = fmaxf(lstep, fabsf(Dz2[2 * q]));
    const float stepf = (float)st->step;
    lstep = sqrtf(stepf * stepf + lstep * lstep) * 1.0001f + 0.01f;
    // Wells of a plan sample (offset q from s, velocity v) that can reach a projected state
    // within rho of s: centre within R + rho + 1 m. A well left out is more than 1 m outside
    // its radius at every projected state, so no fp32 rounding or band decision can flip it.
    auto well_mask = [&](float qx, float qy, float qz, float vx, float vy, float vz, float rho) {
        unsigned msk = 0u;
        for (int w = 0; w < m.n_wells; ++w) {
            const float tau = st->well[w][0];
            const float cx = fmaf(tau, vx, qx), cy = fmaf(tau, vy, qy), cz = fmaf(tau, vz, qz);
            const float lim = st->reach[w] + rho + 1.f;
            if (fmaf(cx, cx, fmaf(cy, cy, cz * cz)) < lim * lim) msk |= 1u << w;
        }
        return msk;
    };

    // the (sub-step, slot) pairs of this warp's first turn, and from one turn to the next
    const int pair_j = S > 0 ? warp * 32 / S : 0, pair_i = warp * 32 - pair_j * S;
    const int turn_j = S > 0 ? NT / S : 0, turn_i = NT - turn_j * S;
    const bool act = lane < A;
    const DeckGrid grid = m.hm ? deck_grid(m) : DeckGrid{};
    const LookScore sc{st, keys, sums, Dx, Dy, Dz};
    // ---- co-simulation: records of the other aircraft (see LookRecord). Before it departs an
    // aircraft's record holds up to the step before, afterwards for ever; then its CTA is done.
    const int n_mem = a.cosim ? a.n_req : 0, n_wait = n_mem + (a.cosim ? a.absent : 0);
    auto record_of = [&](int64_t step, int who) { return a.mem + ((size_t)(step & 1) * n_mem + who) * 12; };
    auto publish = [&](int64_t step, int64_t until, bool flying) {  // lanes 0 .. 5 of warp 0
        if (tid < 6) {
            const double v = tid < 3 ? st->s[tid] : (st->k > 0 ? __ddiv_rn(__dsub_rn(st->s[tid - 3], st->prev[tid - 3]), m.dt) : 0.0);
            put_word(record_of(step, r) + 2 * tid, v, 2 * until + (flying ? 1 : 0));
        }
    };
    auto wait_all = [&](int64_t step) {  // every thread; false when a record did not come
        bool ok = true;
        LookRecord rec;
        for (int q = tid; q < n_wait; q += NT) {
            if (q == r) continue;
            // (the absent aircraft of the self-test: a record that nobody writes)
            ok = look_read(q < n_mem ? record_of(step, q) : a.mem + (size_t)2 * n_mem * 12, step, rec, true) && ok;
            if (!ok) break;
        }
        return __syncthreads_and(ok) != 0;
    };
    int64_t step_no = 0;  // the step's number from a.t_start, counted from 1
    bool late = false;
    if (a.cosim) {
        step_no = req.depart_step - a.t_start + 1;
        if (st->done || step_no > 1) {
            const int64_t until = st->done ? kStampForever : step_no - 1;
            publish(0, until, false);
            publish(1, until, false);
            // until it departs, step by step (each wait is bounded): every aircraft has reached the
            // step before when its record is replaced
            // (one that never flies only sees the others start)
            for (int64_t q = 1; !late && q < (st->done ? 2 : step_no); ++q) late = !wait_all(q);
        }
    }
    for (; !late && !st->done; ++step_no) {
        if (a.cosim) publish(step_no, step_no, true);
        const int k = st->k;
        const int64_t t = req.depart_step + k;
        const int64_t row0 = st->row0;  // ring row of t + 1
        // ---- 1. projected states and samples within reach, side by side
        if (tid == NT - 64) deferred_tie();  // the previous step's near-tie flag (FP64: 1900 cycles, off the chain here)
        if (tid == NT - 1) {
            int n0;
            float phi;
            lk_goal_log(m, st->Ghx, st->Ghy, st->Ghz, st->Glx, st->Gly, st->Glz, n0, phi);
            st->n0 = n0;
            st->phi = phi;
        }
        if (m.n_static > 0) {
            for (int w = tid; w < m.n_static; w += NT) {
                const double* c = m.statics + 6 * w;
                stc[3 * w] = (float)__dsub_rn(c[0], st->s[0]);
                stc[3 * w + 1] = (float)__dsub_rn(c[1], st->s[1]);
                stc[3 * w + 2] = (float)__dsub_rn(c[2], st->s[2]);
            }
            __syncthreads();
        }
        const int h0 = st->h;
        auto turned = [&](int ac) {
            int hn = h0 + m.dh[ac];
            hn += hn < 0 ? 24 : 0;
            return hn - (hn >= 24 ? 24 : 0);
        };
        const float shx = st->shx, shy = st->shy, shz = st->shz, slx = st->slx, sly = st->sly, slz = st->slz;
        const float Gx = st->Ghx + st->Glx, Gy = st->Ghy + st->Gly, Gz = st->Ghz + st->Glz;
        // fp32 offsets (j + 1) * move, box test, goal-term offset, static wells
        for (int q = tid; q < AW; q += NT) {
            const int ac = q / W, j = q - ac * W;
            const int hn = turned(ac);
            const float fj = (float)(j + 1);
            const float px = fmaf(fj, Dh[4 * hn], fj * Dh[4 * hn + 1]);
            const float py = fmaf(fj, Dh[4 * hn + 2], fj * Dh[4 * hn + 3]);
            const float pz = fmaf(fj, Dz2[2 * ac], fj * Dz2[2 * ac + 1]);
            ox[q] = px;
            oy[q] = py;
            oz[q] = pz;
            const float sx = shx + (slx + px), sy = shy + (sly + py), sz = shz + (slz + pz);
            const float mb = fminf(fminf(fminf(sx - box0, sy - box1), sz - box2), fminf(fminf(box3 - sx, box4 - sy), box5 - sz));
            int in;
            if (mb > kBoxBandL) in = 1;
            else if (mb < -kBoxBandL) in = 0;
            else in = look_box_exact(m, st->s, Dx[hn], Dy[hn], Dz[ac], j) ? 1 : 0;
            inb[q] = in;
            float Sh, Sl;
            const float ds = lk_goal_dist(st->Ghx, st->Ghy, st->Ghz, st->Glx, st->Gly, st->Glz, Sh, Sl);
            const float ex = Gx - px, ey = Gy - py, ez = Gz - pz;
            const float d = sqrtf(fmaf(ex, ex, fmaf(ey, ey, ez * ez)));
            const float num = fmaf(px, px, fmaf(py, py, pz * pz)) - 2.f * fmaf(Gx, px, fmaf(Gy, py, Gz * pz));
            const float den = d + ds;
            const float dd = den > 0.f ? num / den : 0.f;  // d(x_j) - d(s)
            rel[q] = dd * m.lg32;
            // static negative peaks (restricted volumes / terrain wells)
            float mbw = -INFINITY;
            unsigned long long sb = 0ull;
            for (int w = 0; w < m.n_static; ++w) {
                const float ux = px - stc[3 * w], uy = py - stc[3 * w + 1], uz = pz - stc[3 * w + 2];
                const float d2 = fmaf(ux, ux, fmaf(uy, uy, uz * uz));
                const float R2 = m.st_R2[w];
                bool inw = d2 < R2;
                if (fabsf(d2 - R2) <= m.st_band[w]) inw = look_static_exact(m, w, st->s, Dx[hn], Dy[hn], Dz[ac], j);
                if (inw) {
                    const float l = fmaf(sqrtf(d2), m.st_lg[w], m.st_L[w]);
                    mbw = fmaxf(mbw, l);
                    if (m.combine) sb += look_sum_term(l, m.sum_ref);
                }
            }
            if (mbw > -INFINITY) atomicMax(&keys[q], float_key(mbw));
            if (sb) atomicAdd(&sums[q], sb);
        }
        int hn_l = 0;  // this lane's action
        float4 Dxy_l = make_float4(0.f, 0.f, 0.f, 0.f);
        float2 Dzf_l = make_float2(0.f, 0.f);
        if (act) {
            hn_l = turned(lane);
            Dxy_l = *reinterpret_cast<const float4*>(Dh + 4 * hn_l);
            Dzf_l = *reinterpret_cast<const float2*>(Dz2 + 2 * lane);
        }
        // appends the lanes' samples that have wells in reach (a warp together); those that no
        // longer fit are scored at once
        auto add = [&](const LookItem& it, bool have) {
            const unsigned mask = __ballot_sync(kFullMask, have);
            if (!mask) return;
            int at = 0;
            if (lane == __ffs(mask) - 1) at = atomicAdd(&st->n_list, __popc(mask));
            at = __shfl_sync(kFullMask, at, __ffs(mask) - 1) + __popc(mask & ((1u << lane) - 1u));
            if (have && at < kLookList) list[at] = it;
#pragma unroll 1
            for (unsigned over = __ballot_sync(kFullMask, have && at >= kLookList); over; over &= over - 1u) {
                const int b = __ffs(over) - 1;
                LookItem o;
                o.qx = __shfl_sync(kFullMask, it.qx, b), o.qy = __shfl_sync(kFullMask, it.qy, b);
                o.qz = __shfl_sync(kFullMask, it.qz, b), o.what = __shfl_sync(kFullMask, it.what, b);
                o.vx = __shfl_sync(kFullMask, it.vx, b), o.vy = __shfl_sync(kFullMask, it.vy, b);
                o.vz = __shfl_sync(kFullMask, it.vz, b), o.ref = __shfl_sync(kFullMask, it.ref, b);
                look_score_over(a, sc, o, hn_l, Dxy_l, Dzf_l);
                __syncwarp();
            }
        };
        // a plan sample (P2.x NaN: the plan's last) as an item of sub-step j
        auto plan_item = [&](float4 P1, float4 P2, int j, int kind, int ref) {
            LookItem it;
            it.qx = (P1.x - shx) - slx, it.qy = (P1.y - shy) - sly, it.qz = (P1.z - shz) - slz;
            const bool has2 = P2.x == P2.x;
            it.vx = has2 ? (P2.x - P1.x) * inv_dt : 0.f;
            it.vy = has2 ? (P2.y - P1.y) * inv_dt : 0.f;
            it.vz = has2 ? (P2.z - P1.z) * inv_dt : 0.f;
            it.what = (int)well_mask(it.qx, it.qy, it.qz, it.vx, it.vy, it.vz, (float)(j + 1) * lstep) | j << 16 | kind << 24;
            it.ref = ref;
            return it;
        };
        const int64_t t_hi = a.tab.t_base + a.tab.T_win;
        if (a.by_index) {
            // one warp per sub-step (the last warps first: the first ones have the projected
            // states): the cells within reach, as in the one-step rollout, and the extra list
            const IndexView& iv = a.iv;
            for (int j = NT / 32 - 1 - warp; j < W; j += NT / 32) {
                const int64_t t1 = t + j + 1;
                if (t1 < a.tab.t_base || t1 >= t_hi) continue;
                int64_t r1 = row0 + j;
                r1 -= r1 >= a.tab.T_win ? a.tab.T_win : 0;
                const int32_t* cs_row = iv.cstart + r1 * ((int64_t)iv.ncell + 1);
                const float Rq = m.reach_base + (float)(j + 1) * lstep + m.tau_absmax * iv.vmax * 1.0001f + 2.f;
                const float x = shx + slx, y = shy + sly;
                auto cell_of = [&](float v, float o, int n) {
                    const float g = floorf((v - o) * iv.inv_cell);
                    return g < 0.f ? 0 : (g > (float)(n - 1) ? n - 1 : (int)g);
                };
                const int cx0 = cell_of(x - Rq, iv.x0, iv.ncx), cx1 = cell_of(x + Rq, iv.x0, iv.ncx);
                const int cy0 = cell_of(y - Rq, iv.y0, iv.ncy), cy1 = cell_of(y + Rq, iv.y0, iv.ncy);
                const int nrows = cy1 - cy0 + 1;
                int e0 = 0, e1 = 0;  // item ranges, one per lane (lane 31: the extra list)
                if (nrows < 32) {
                    if (lane < nrows) {
                        e0 = __ldcg(cs_row + (cy0 + lane) * iv.ncx + cx0);
                        e1 = __ldcg(cs_row + (cy0 + lane) * iv.ncx + cx1 + 1);
                    }
                } else if (lane == 0) {  // one range over full cell rows
                    e0 = __ldcg(cs_row + cy0 * iv.ncx);
                    e1 = __ldcg(cs_row + (cy1 + 1) * iv.ncx);
                }
                if (lane == 31) {
                    e0 = __ldcg(cs_row + iv.ncell);
                    e1 = e0 + __ldcg(iv.nextra + r1);
                }
                const int num = max(0, e1 - e0);
                int at = num;  // inclusive prefix of the ranges' item counts
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(kFullMask, at, o);
                    if (lane >= o) at += v;
                }
                const int total = __shfl_sync(kFullMask, at, 31), base = e0 - (at - num);
                const float4* items = iv.items + (size_t)r1 * a.tab.S_pad * 2;
                for (int i0 = 0; i0 < total; i0 += 32) {
                    const int i = i0 + lane;
                    int lo = 0;  // the range of item i: the first whose prefix exceeds i
#pragma unroll
                    for (int o = 16; o; o >>= 1) lo += __shfl_sync(kFullMask, at, lo + o - 1) <= i ? o : 0;
                    const int id = __shfl_sync(kFullMask, base, lo) + i;
                    LookItem it{};
                    bool have = false;
                    if (i < total) {
                        const float4 P1 = __ldcg(items + 2 * (size_t)id), P2 = __ldcg(items + 2 * (size_t)id + 1);
                        it = plan_item(P1, P2, j, kLookIndex, id);
                        have = tag_visible(__float_as_int(P1.w), INT_MAX) && (it.what & 0xffff);
                    }
                    add(it, have);
                }
            }
        } else {
            // every (sub-step, slot) pair, U per thread and turn: their loads are in flight together
            // (S is a multiple of 32, so a warp's slots lie in one slice)
            constexpr int U = 3;
            const int npairs = W * S;
            int j0 = pair_j, i0 = pair_i;
            const int j_lo = (int)max(a.tab.t_base - t - 1, (int64_t)0), j_hi = (int)min(t_hi - t - 1, (int64_t)W);
            const int row_i = (int)row0, T_win = a.tab.T_win;
            for (int base = warp * 32; base < npairs; base += U * NT) {
                float4 P1[U], P2[U];
                int js[U], is[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    js[u] = j0, is[u] = i0 + lane;
                    j0 += turn_j, i0 += turn_i;
                    if (i0 >= S) i0 -= S, ++j0;
                    P1[u] = P2[u] = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
                    if (base + u * NT < npairs && js[u] >= j_lo && js[u] < j_hi) {
                        int r1 = row_i + js[u];  // rows of t + j + 1 and t + j + 2 (j < T_win)
                        r1 -= r1 >= T_win ? T_win : 0;
                        const size_t o1 = (size_t)r1 * a.tab.S_pad + is[u];
                        P1[u] = make_float4(a.tab.X[o1], a.tab.Y[o1], a.tab.Z[o1], 0.f);
                        if (t + js[u] + 2 < t_hi) {
                            const size_t o2 = (size_t)(r1 + 1 >= T_win ? 0 : r1 + 1) * a.tab.S_pad + is[u];
                            P2[u] = make_float4(a.tab.X[o2], a.tab.Y[o2], a.tab.Z[o2], 0.f);
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (base + u * NT >= npairs) break;  // (the same in the whole warp)
                    LookItem it{};
                    bool have = P1[u].x == P1[u].x;
                    if (have) {
                        it = plan_item(P1[u], P2[u], js[u], kLookSlot, is[u]);
                        have = (it.what & 0xffff) != 0;
                    }
                    add(it, have);
                }
            }
        }
        // co-simulation: the wells of every other aircraft in flight, at its position at t plus tau
        // times its last move (the same peaks for every sub-step)
        for (int q0 = warp * 32; q0 < n_wait; q0 += NT) {
            const int q = q0 + lane;
            LookRecord rec;
            rec.flying = false;
            if (q < n_wait && q != r &&
                !look_read(q < n_mem ? record_of(step_no, q) : a.mem + (size_t)2 * n_mem * 12, step_no, rec, false)) {
                st->late = 1;
                rec.flying = false;
            }
            __syncwarp();
            LookItem it{};
            if (rec.flying) {
                it.qx = (float)__dsub_rn(rec.v[0], st->s[0]);
                it.qy = (float)__dsub_rn(rec.v[1], st->s[1]);
                it.qz = (float)__dsub_rn(rec.v[2], st->s[2]);
                it.vx = (float)rec.v[3], it.vy = (float)rec.v[4], it.vz = (float)rec.v[5];
                it.ref = q;
            }
            for (int j = 0; j < W; ++j) {
                const unsigned wells =
                    rec.flying ? well_mask(it.qx, it.qy, it.qz, it.vx, it.vy, it.vz, (float)(j + 1) * lstep) : 0u;
                it.what = (int)wells | j << 16 | kLookMember << 24;
                add(it, wells != 0u);
            }
        }
        __syncthreads();
        if (st->late) {  // (the same in every thread)
            late = true;
            break;
        }

        // ---- 2. the list, shared out between the warps
        const int n_list = min(st->n_list, kLookList);
        for (int e = warp; e < n_list; e += NT / 32) look_score(a, sc, list[e], hn_l, Dxy_l, Dzf_l);
        __syncthreads();

        // ---- 3. penalty + deck per (action, sub-step), as log2
        if (tid == 0) st->n_list = 0;
        for (int q = tid; q < AW; q += NT) {
            float P = 0.f;
            if (m.combine) {
                if (sums[q]) P = (float)((double)sums[q] * m.sum_scale);
            } else if (keys[q] != KEY_NONE) {
                P = exp2f(key_float(keys[q]));
            }
            keys[q] = KEY_NONE;  // for the next step
            if (m.combine) sums[q] = 0ull;
            float D = 0.f;
            if (m.hm) {
                const float sx = shx + (slx + ox[q]), sy = shy + (sly + oy[q]), sz = shz + (slz + oz[q]);
                const float c32 = sz - terrain32(m, sx, sy);
                if (fabsf(c32 - (float)m.clearance) <= kClrBand + kTerrBand) {
                    const int ac = q / W, hn = turned(ac), j = q - ac * W;
                    // the projected state as double-float: off from the exact one by a rounding per
                    // step and per sub-step
                    float hx = shx, lx = slx, hy = shy, ly = sly, hz = shz, lz = slz;
                    for (int i = 0; i <= j; ++i) {
                        df_add(hx, lx, Dh[4 * hn], Dh[4 * hn + 1]);
                        df_add(hy, ly, Dh[4 * hn + 2], Dh[4 * hn + 3]);
                        df_add(hz, lz, Dz2[2 * ac], Dz2[2 * ac + 1]);
                    }
                    TerrainCell tc = terrain_cell(hx, hy, box0, box1, m.hm_sx, m.hm_sy, m.hm_nx, m.hm_ny);
                    terrain_nodes(tc, m.hm, m.hm_nx);
                    D = deck_band(m, grid, tc, hx, lx, hy, ly, hz, lz, k + j);
                    if (D < 0.f) D = look_deck_exact(m, st->s, Dx[hn], Dy[hn], Dz[ac], j);
                } else if (c32 < (float)m.clearance) {
                    D = (float)m.deck - c32;
                }
            }
            const float N = P + D;
            const float ln = N > 0.f ? log2f(N) : -INFINITY;
            // the value g - N at x_j relative to 2^n0 (g = 2^(phi + rel), N = 2^(ln - n0))
            const float lg = st->phi + rel[q];
            int sg;
            float lv, lsc;
            bool vabs = false;
            if (ln == -INFINITY) {
                sg = 1;
                lv = lg;
                lsc = lg;
            } else {
                const float lnr = ln - (float)st->n0;
                const float x = lnr - lg;  // log2 (N / g)
                lsc = fmaxf(lg, lnr);
                if (x < -30.f) {
                    sg = 1;
                    lv = lg;
                } else if (x > 30.f) {
                    sg = -1;
                    lv = ln;
                    vabs = true;
                } else {
                    const float rr = exp2f(x);
                    if (rr < 1.f) {
                        sg = 1;
                        lv = lg + log2f(1.f - rr);
                    } else if (rr > 1.f) {
                        sg = -1;
                        lv = lg + log2f(rr - 1.f);
                    } else {
                        sg = 0;
                        lv = 0.f;
                    }
                }
            }
            vsg[q] = (sg + 1) | (vabs ? 4 : 0);
            vlv[q] = lv;
            vls[q] = lsc;
            // order of the values: by sign, then by size; a sub-step outside the box counts only as
            // the first
            const float lr = vabs ? lv - (float)st->n0 : lv;
            cmp[q] = make_float2(q % W > 0 && !inb[q] ? -2.f : (float)sg, sg > 0 ? lr : (sg < 0 ? -lr : 0.f));
        }
        __syncthreads();

        // ---- 4. per action (lanes): the largest value over its projected states inside the box.
        // Values are held relative to 2^n0 (n0: integer part of log2 of the goal term at s):
        // g = 2^(phi + rel), N = 2^(lN - n0); g - N as (sign, log2 |g - N|), which keeps the
        // goal term's resolution when N at another sub-step is larger by hundreds of binary
        // orders. Only the winner per action is turned into an absolute FP64 log2. Then argmax,
        // near-tie record, advance.
        if (warp == 0) {
            int sgl = -2;
            double Lkl = 0.0;
            unsigned long long kq = 0ull;
            const int n0 = st->n0;
            if (act) {
                const int q0 = lane * W;
                int bj = 0;
                float2 b = cmp[q0];
#pragma unroll 4
                for (int j = 1; j < W; ++j) {
                    const float2 v = cmp[q0 + j];
                    const bool better = v.x > b.x || (v.x == b.x && v.y > b.y);
                    bj = better ? j : bj;
                    b = better ? v : b;
                }
                const int bq = q0 + bj, code = vsg[bq];
                const float lv = vlv[bq];
                const int sg = (code & 3) - 1;
                Lkl = (code & 4) ? (double)lv : __dadd_rn((double)n0, (double)lv);
                if (inb[q0]) {
                    sgl = sg;
                    kq = look_key(sg, Lkl);
                }
                // for the near-tie flag, during the next step
                st->tie_sg[lane] = sgl;
                st->tie_L[lane] = Lkl;
                st->tie_T[lane] = vls[bq];
            }
            // the largest of the lanes' 64-bit keys, by halves
            auto largest = [&](unsigned long long v) {
                const unsigned hi = __reduce_max_sync(kFullMask, (unsigned)(v >> 32));
                const unsigned lo = __reduce_max_sync(kFullMask, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
                return (unsigned long long)hi << 32 | lo;
            };
            const unsigned long long mx = largest(kq);
            const unsigned bm = __ballot_sync(kFullMask, lane < A && kq == mx && mx != 0ull);
            const int a1 = bm ? __ffs(bm) - 1 : -1;
            const unsigned long long k2 = largest(lane < A && lane != a1 ? kq : 0ull);
            const unsigned b2 = __ballot_sync(kFullMask, lane < A && lane != a1 && kq == k2 && k2 != 0ull);
            const int a2 = b2 ? __ffs(b2) - 1 : -1;
            if (a.trace && lane < A)
                q_trace[(size_t)k * A + lane] = sgl == -2 ? -INFINITY : (sgl == 0 ? 0.0 : (double)sgl * exp2(Lkl));
            if (a1 < 0) {
                if (lane == 0) {
                    st->status = FMDP_REJ_NO_ACTION;
                    st->done = 1;
                }
            } else {
                // exact advance (FP64, the oracle's x_1) and its double-float copies: lanes 0 .. 2
                // take x, y, z
                const int hn = turned(a1), np = k + 1;
                float G = 0.f;
                if (lane < 3) {
                    const float* Df = lane < 2 ? Dh + 4 * hn + 2 * lane : Dz2 + 2 * a1;
                    const double D = (lane == 0 ? Dx : Dy)[hn], s0 = st->s[lane];
                    const double s1 = __dadd_rn(s0, lane < 2 ? D : Dz[a1]);
                    df_add((&st->shx)[lane], (&st->slx)[lane], Df[0], Df[1]);
                    df_add((&st->Ghx)[lane], (&st->Glx)[lane], -Df[0], -Df[1]);
                    G = (&st->Ghx)[lane] + (&st->Glx)[lane];
                    st->prev[lane] = s0;
                    st->s[lane] = s1;
                    traj[3 * np + lane] = (float)s1;
                    if (a.trace) st_trace[3 * np + lane] = s1;
                }
                const float gx = __shfl_sync(kFullMask, G, 0), gy = __shfl_sync(kFullMask, G, 1), gz = __shfl_sync(kFullMask, G, 2);
                __syncwarp();
                if (lane == 0) {
                    st->h = hn;
                    acts[k] = (uint8_t)a1;
                    if (a.trace) hd_trace[np] = hn;
                    st->k = np;
                    st->t = t + 1;
                    st->step_no = step_no + 1;
                    st->row0 = row0 + 1 == a.tab.T_win ? 0 : row0 + 1;
                    const float gd = sqrtf(gx * gx + gy * gy + gz * gz);
                    bool cap = false;
                    if (gd < stepf + kCapBandL) cap = look_capture_exact(st->s, req, st->cap2);
                    if (cap) {
                        st->status = kStatusCaptured;
                        st->done = 1;
                    } else if (np >= req.horizon) {
                        st->status = FMDP_REJ_HORIZON;
                        st->done = 1;
                    }
                }
            }
            if (lane == 0) {
                st->tie_k = k;  // tested during the next step (deferred_tie)
                st->tie_a1 = a1;
                st->tie_a2 = a2;
                st->tie_n0 = n0;
            }
        }
        __syncthreads();
    }
    if (a.cosim && !late && step_no > req.depart_step - a.t_start + 1) {
        // the record of the first step not flown, then, once every other aircraft has it or its own,
        // the other one
        publish(step_no, kStampForever, false);
        late = !wait_all(step_no);
        if (!late) publish(step_no + 1, kStampForever, false);
    }
    if (late && tid == 0) atomicExch(a.err, FMDP_ERR_TIMEOUT);
    if (tid == 0) {
        deferred_tie();
        RolloutOut o;
        o.n_points = st->k + 1;
        o.status = st->status;
        o.near_ties = st->near_ties;
        o.steps = st->k;
        a.out[r] = o;
    }
}

cudaError_t prepare_lookahead_kernel() {
    const int smem = (int)look_layout(kMaxActions, kMaxLookahead).total;
    const cudaError_t e = cudaFuncSetAttribute(lookahead_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(lookahead_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

int lookahead_max_resident(int A, int W) {
    int per_sm = 0, dev = 0, n_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lookahead_kernel<256>, 256, look_layout(A, W).total) !=
            cudaSuccess ||
        cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per_sm * n_sm;
}

cudaError_t launch_lookahead(const LookArgs& a, cudaStream_t s) {
    if (a.n_req <= 0) return cudaSuccess;
    const size_t smem = look_layout(a.m.A, a.W).total;
    if (!a.cosim) {
        // also with more requests than SMs: 256 requests at W = 10, 450 ms of rollouts in waves, 610
        // with 256 threads and two CTAs per SM (most waves are the last few requests' re-plans)
        lookahead_kernel<512><<<a.n_req, 512, smem, s>>>(a);
        return cudaGetLastError();
    }
    // co-simulation: every CTA must be resident at once (they wait for one another), two per SM
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.n_req, 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, lookahead_kernel<256>, a);
}

}  // namespace fmdp
