// One request planned against the spatial index by one CTA (included by rollout.cu).
//
// FastMDP's rollout is a chain: step k + 1 scores the successors of the state that step k
// chose. No throughput bounds it; what counts is the latency from one state to the next, and
// that is mostly the length of the instruction stream of the warps between the two. So the
// step's work is cut into short pieces that run side by side, and everything that does not
// depend on the newest state runs ahead of the chain or behind it:
//   control    (warp 0, lane a scores action a) goal term and box; then, with the folded
//              wells and the clearance, the action values and the argmax;
//   successor  (warp 1) each action's successor as a complete next state (double-float
//              position, goal vector, capture test; after it the goal-term split, which the
//              next step's values need last), in shared memory: the next step's state is the
//              winner's entry. It also publishes that state to the warps below;
//   terrain    (one warp of eight or more, else the control warp) the clearance penalties;
//   fold       (1 or 2 warps) the wells of the step's list, shared out between them;
//   helpers    each prepare the list of every n-th step, kAhead steps ahead, from the last
//              state known then: they read the index rows around it with a radius widened by
//              the steps in between, and keep the plan samples with a well that can reach a
//              successor of any state the aircraft may have by then (also the static
//              wells in reach). A sample left out has its wells more
//              than 1 m beyond their radii for every successor, so it adds an exact zero; a
//              kept one is scored with the state's own offsets, in the order of operations of
//              the full scan. The index
//              latency (row header, cell starts, items) is spent kAhead steps before its
//              result is needed;
//   recorder   behind the chain: the exact FP64 state (three rounded adds per step),
//              trajectory, actions, resume records and near-tie flags. The exact state is
//              read by the others only where a decision falls into an FP64 band.
// Per step control, successor and fold warps meet at two named barriers, each with one side
// arriving without waiting: A (the action chosen) and B (successors and wells ready). Lists
// and published states go through mbarriers, every wait bounded. Warps 4 and 8 share the
// control warp's issue slots, so they hold the light roles.
// On GB300, one request against 3000 plans: 1.65 us per step with two CTA barriers per step
// and the items staged raw in shared memory, 1.08 us with this; 20 000 plans (124 samples read
// and 36 kept per step): 2.5 and 1.86 us. (One warp doing control, successor and fold alone,
// without any barrier, took 1.6 and 3.0 us: some 700 instructions in one stream.) Of the 1900
// cycles of a step, 750 are the control warp's from A to B, next to the successor and fold
// warps' 900, and 850 to 1400 from B to the next A.
// Lists of samples rather than of sample-well pairs: at 36 samples per step the list warps take
// 8700 cycles instead of 15 700, and five of them keep up with the chain; the fold warps
// pick the wells in reach of the newest state when they read the list. A warp between the
// two that picks them cost the chain another hand-over: 1.18 and 2.1 us.

constexpr int kAhead = 6;    // steps between the state a list is made from and its use
constexpr int kSlots = 8;    // lists in shared memory (a power of two > kAhead)
constexpr int kPub = 16;     // published states in shared memory (a power of two)
constexpr int kRecLag = 10;  // steps the recorder may fall behind (< kPub)
constexpr int kMaxFold = 2;  // fold warps
constexpr int kMaxRanges = 8;  // item ranges of a query: up to 7 cell rows and the extra list
constexpr int kPatch = 8;    // heightmap patch: 8 x 8 nodes
constexpr int kBarChosen = 1, kBarReady = 2;  // named barriers A and B

enum PlanRole { kControl, kSuccessor, kTerrain, kFold, kRecorder, kHelper };
struct PlanRoles {
    int role, index, n_fold, n_help;  // index: which fold warp or helper
    // false: the successor warp records; the control warp does the terrain
    bool own_recorder, own_terrain;
};
// Roles of NW (4 .. 12) warps.
__device__ __forceinline__ PlanRoles plan_roles(int NW, int warp) {
    PlanRoles r;
    r.own_recorder = NW > 5;
    r.own_terrain = NW >= 8;
    // (one fold warp sets the pace among many plans: 64 rollouts among 20 000 plans by eight warps
    // 4.56 ms, 3.69 with two; by six, two would leave one list warp)
    r.n_fold = NW >= 7 ? 2 : 1;
    auto role_of = [&](int w) {
        if (w == 0) return kControl;
        if (w == 1) return kSuccessor;
        if (w == 2 || (w == 5 && r.n_fold > 1)) return kFold;
        if (w == 3 && r.own_terrain) return kTerrain;
        if (w == 4 && r.own_recorder) return kRecorder;
        return kHelper;
    };
    r.role = role_of(warp);
    r.n_help = r.index = 0;
    for (int w = 0; w < NW; ++w) {
        if (w < warp && role_of(w) == r.role) ++r.index;
        if (role_of(w) == kHelper) ++r.n_help;
    }
    return r;
}

// named barrier over `threads` threads: wait, or arrive without waiting
__device__ __forceinline__ void bar_wait(int id, int threads) {
    asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
    asm volatile("barrier.cta.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// plan samples a list holds: an eighth of options.index_stage_items (a step with more near ones
// is scored from the index by a fold warp)
__host__ __device__ inline int list_capacity(int icap) { return icap / 8 > 8 ? icap / 8 : 8; }

struct ListMeta {
    int n;            // near samples (may exceed the capacity: then none is used)
    int pub;          // table operations published before the row was read
    int abort;        // a wait of the helper expired
    unsigned stat_lo, stat_hi;  // static wells in reach
    int pad;
    long long row_off;          // first float4 of the row's items
    int beg[kMaxRanges], cnt[kMaxRanges];  // the row's item ranges (cnt 0: none)
};

// One published state: x, y, z as double-float; what the step that reached it chose.
struct PubState {
    float hx, hy, hz;
    int what;  // action | heading index << 8 | kPubDone | kPubNone
    float lx, ly, lz;
    int pub;   // table operations known to the step that reached it
};
constexpr int kPubDone = 1 << 16;  // the plan ends in this state
constexpr int kPubNone = 1 << 17;  // no action was taken (dead end or error)
constexpr int kNoAction = 0xff;

// A successor as a complete next state.
struct NextState {
    float hx, hy, hz;  // position, double-float
    int packed;        // captured << 5 | heading index
    float lx, ly, lz;
    float pad0;
    float Gx, Gy, Gz;  // goal - position
    float pad1;
};

struct IdxState {
    NextState next[2][kMaxActions];  // by step parity
    float2 split[2][kMaxActions];    // log2 of the goal term there: integer part (int bits), fraction
    float deck[kMaxActions];         // clearance penalties of the step's successors
    float patch[kPatch * kPatch];    // heightmap around the state before the last step (terrain warp)
    float fold_max[kMaxFold][kMaxActions];  // per action: largest log2 (|r| gamma^d) of a fold warp's wells
    unsigned long long fold_sum[kMaxFold][kMaxActions];  // SUM
    int best[2];     // action of step c (by c & 1), kNoAction: the plan ends without one
    int fold_abort;  // a fold warp's wait expired, or its list's helper gave up
    float4 well[kMaxWells];   // tau, R^2, log2 gamma, log2 |r|
    float2 reach[kMaxWells];  // tau, (R + largest successor offset + 1 m)^2
    double s64[kPub][3];      // exact states, written by the recorder
    float4 Dxy[kHeadings];    // the moves as double-float: xh, xl, yh, yl
    float2 Dzf[kMaxActions];  // climb: zh, zl
    double Dx[kHeadings], Dy[kHeadings], Dz[kMaxActions];
    PubState ps[kPub];
    float4 tie[kPub][kMaxActions];  // every action of a step: key, log2|Q|, log2 of the goal term, penalty
    // mbarriers: list ready; state published (for the helpers, for the recorder)
    uint64_t full[kSlots], seen[kPub], seen_rec[kPub];
    float stat_hi[kMaxStatic][3], stat_lo[kMaxStatic][3];  // static-well centres as double-float
    ListMeta meta[kSlots];
    double step, cap2;
    int rec_steps;            // steps the recorder has finished
    int stop;                 // no more lists are needed
    int captured0;            // the origin is inside the capture ball
    int status, n_points, steps, near_ties;
};

__host__ __device__ inline size_t idx_lists_offset() { return (sizeof(IdxState) + 127) & ~size_t(127); }
__host__ __device__ inline size_t idx_misc_offset(int icap) {
    return idx_lists_offset() + (size_t)kSlots * list_capacity(icap) * 2 * sizeof(float4);
}
// misc: the work-queue words of the persistent modes (48 bytes, see rollout_kernel)
__host__ __device__ inline size_t idx_smem_bytes(int icap) { return (idx_misc_offset(icap) + 48 + 127) & ~size_t(127); }

__device__ __forceinline__ bool idx_wait(uint64_t* bar, uint32_t parity) {
    return mbar_try_wait(bar, parity) || mbar_wait_bounded(bar, parity);
}
// A fold warp's wait for the list of step c. It may be ahead of the state by one step, so the plan
// can end while it waits: then true, and the barrier after it tells.
__device__ __forceinline__ bool idx_wait_list(IdxState* st, int c) {
    uint64_t* bar = &st->full[c & (kSlots - 1)];
    const uint32_t parity = (uint32_t)((c / kSlots) & 1);
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_test_wait(bar, parity)) {
        if (*(volatile int*)&st->stop) return true;
        if (clock64() - t0 > (1ll << 31)) return false;
    }
    return true;
}
// A helper's wait for a state: 1 published, 0 not needed any more (stop), -1 timed out.
__device__ __forceinline__ int idx_wait_state(IdxState* st, int state) {
    uint64_t* bar = &st->seen[(state - 1) & (kPub - 1)];
    const uint32_t parity = (uint32_t)(((state - 1) / kPub) & 1);
    if (mbar_try_wait(bar, parity)) return 1;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*(volatile int*)&st->stop) return 0;
        if (clock64() - t0 > (1ll << 31)) return -1;
    }
    return 1;
}

// What scoring a well needs of the state and this lane's action.
struct FoldLane {
    float shx, shy, shz, slx, sly, slz;  // the state, double-float
    float dxa, dya, dza;                 // the action's move
    float mloc;                          // largest log2 (|r| gamma^d) so far
    unsigned long long sloc;             // SUM: fixed-point sum
};

// Wells of a plan sample (offset q from the state, velocity v) whose centre is within reach of a
// successor.
__device__ __forceinline__ unsigned well_mask(const float2* reach, int n_wells, float qx, float qy, float qz, float vx,
                                              float vy, float vz) {
    unsigned msk = 0u;
#pragma unroll
    for (int w = 0; w < kMaxWells; ++w) {
        if (w >= n_wells) break;
        const float2 r = reach[w];
        const float cx = fmaf(r.x, vx, qx), cy = fmaf(r.x, vy, qy), cz = fmaf(r.x, vz, qz);
        if (fmaf(cx, cx, fmaf(cy, cy, cz * cz)) < r.y) msk |= 1u << w;
    }
    return msk;
}

// One well of a plan sample (offset q, velocity v) at this lane's successor; true when its edge
// lies within the FP32 band (to be decided in FP64). R2 < 0: no well. Without branches: a lone
// warp pays for a divergent region with more cycles than the square root costs.
__device__ __forceinline__ bool fold_well(FoldLane& f, float qx, float qy, float qz, float vx, float vy, float vz,
                                          const float4 well, bool use_sum, float sum_ref) {
    const float ex = f.dxa - fmaf(well.x, vx, qx);
    const float ey = f.dya - fmaf(well.x, vy, qy);
    const float ez = f.dza - fmaf(well.x, vz, qz);
    const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
    const float R2 = well.y, bw = kWellBand * R2;
    const bool in = d2 < R2 - bw;
    const float l = fmaf(approx_sqrt(d2), well.z, well.w);
    f.mloc = fmaxf(f.mloc, in ? l : -INFINITY);
    if (use_sum && in) f.sloc += sum_term(l, sum_ref);
    return d2 < R2 + bw && !in;
}

// The wells of one sample that lie in the FP32 band, decided in FP64 (exact state s64, exact move
// of the lane's action), then scored. item: the sample in the index.
__device__ __noinline__ void fold_band(const Model& m, const IdxState* st, const double* s64, double Dxa, double Dya,
                                       double Dza, const float4* item, unsigned band, float qx, float qy, float qz, float vx,
                                       float vy, float vz, FoldLane& f, bool use_sum) {
    const float4 P1 = __ldcg(item), P2 = __ldcg(item + 1);
    const bool has2 = P2.x == P2.x;
    for (; band; band &= band - 1u) {
        const int w = __ffs(band) - 1;
        if (!well_inside_exact(m, s64, Dxa, Dya, Dza, P1.x, P1.y, P1.z, has2 ? P2.x : 0.f, has2 ? P2.y : 0.f,
                               has2 ? P2.z : 0.f, has2, w))
            continue;
        const float4 k = st->well[w];
        const float ex = f.dxa - fmaf(k.x, vx, qx), ey = f.dya - fmaf(k.x, vy, qy), ez = f.dza - fmaf(k.x, vz, qz);
        const float l = fmaf(approx_sqrt(fmaf(ex, ex, fmaf(ey, ey, ez * ez))), k.z, k.w);
        f.mloc = fmaxf(f.mloc, l);
        if (use_sum) f.sloc += sum_term(l, m.sum_ref);
    }
}

// Scores the wells `wells` of one sample (position p, velocity v; the same in every lane) for
// every action. item: the sample in the index. exact: the exact state, asked for only in the band.
template <class Exact>
__device__ __forceinline__ void fold_sample(const Model& m, const IdxState* st, const Exact& exact, double Dxa, double Dya,
                                            double Dza, const float4* item, unsigned wells, float px, float py, float pz,
                                            float vx, float vy, float vz, bool act, FoldLane& f, bool use_sum) {
    const float qx = (px - f.shx) - f.slx, qy = (py - f.shy) - f.sly, qz = (pz - f.shz) - f.slz;
    unsigned band = 0u;
    while (wells) {  // two at a time: independent chains
        const int i = __ffs(wells) - 1;
        wells &= wells - 1u;
        const int j = wells ? __ffs(wells) - 1 : i;
        const float4 a = st->well[i];
        float4 b = st->well[j];
        if (!wells) b.y = -1.f;
        wells &= wells - 1u;
        if (fold_well(f, qx, qy, qz, vx, vy, vz, a, use_sum, m.sum_ref)) band |= 1u << i;
        if (fold_well(f, qx, qy, qz, vx, vy, vz, b, use_sum, m.sum_ref)) band |= 1u << j;
    }
    if (act && band) {  // (rare)
        FoldLane g = f;  // (a copy: the call takes addresses)
        fold_band(m, st, exact(), Dxa, Dya, Dza, item, band, qx, qy, qz, vx, vy, vz, g, use_sum);
        f.mloc = g.mloc;
        f.sloc = g.sloc;
    }
    __syncwarp();
}

// A plan sample of the index (lanes = items), for a query around a state: its velocity, and
// whether one of its wells can lie within `reach` (plus its own motion) of the state.
struct ItemLane {
    float px, py, pz, vx, vy, vz;
    bool near;
};
__device__ __forceinline__ ItemLane item_lane(const float4 P1, const float4 P2, bool have, int my_ord, float hx, float hy,
                                              float hz, float lx, float ly, float lz, float inv_dt, float tau_absmax,
                                              float reach) {
    ItemLane t;
    t.px = P1.x, t.py = P1.y, t.pz = P1.z;
    const bool next = P2.x == P2.x;
    t.vx = next ? (P2.x - P1.x) * inv_dt : 0.f;
    t.vy = next ? (P2.y - P1.y) * inv_dt : 0.f;
    t.vz = next ? (P2.z - P1.z) * inv_dt : 0.f;
    const float qx = (P1.x - hx) - lx, qy = (P1.y - hy) - ly, qz = (P1.z - hz) - lz;
    const float r = fmaf(tau_absmax, approx_sqrt(t.vx * t.vx + t.vy * t.vy + t.vz * t.vz), reach);
    // a later request's tentative plan, or a withdrawn one, is not in this request's table
    t.near = have && tag_visible(__float_as_int(P1.w), my_ord) && (qx * qx + qy * qy + qz * qz) < r * r;
    return t;
}

// A step whose near samples exceeded its list: a fold warp reads the query's items itself and
// scores the wells in reach (lanes = items, then lanes = actions).
__device__ __noinline__ void fold_overflow(const RolloutArgs& a, const IdxState* st, const ListMeta& M, int my_ord,
                                           float inv_dt, float reach0, const double* s64, double Dxa, double Dya,
                                           double Dza, bool act, FoldLane& f, bool use_sum, unsigned& pairs) {
    const Model& m = a.m;
    const int lane = threadIdx.x & 31;
    const float4* items = a.iv.items + M.row_off;
    FoldLane g = f;
    for (int q = 0; q < kMaxRanges; ++q) {
        for (int i0 = 0; i0 < M.cnt[q]; i0 += 32) {
            const int i = M.beg[q] + i0 + lane;
            const bool have = i0 + lane < M.cnt[q];
            float4 P1 = make_float4(0.f, 0.f, 0.f, 0.f), P2 = P1;
            if (have) {
                P1 = __ldcg(items + 2 * (size_t)i);
                P2 = __ldcg(items + 2 * (size_t)i + 1);
            }
            const ItemLane t = item_lane(P1, P2, have, my_ord, g.shx, g.shy, g.shz, g.slx, g.sly, g.slz, inv_dt,
                                         m.tau_absmax, reach0);
            const unsigned wells = t.near ? well_mask(st->reach, m.n_wells, (t.px - g.shx) - g.slx, (t.py - g.shy) - g.sly,
                                                      (t.pz - g.shz) - g.slz, t.vx, t.vy, t.vz)
                                          : 0u;
            pairs += __popc(wells);
            for (unsigned mask = __ballot_sync(kFull, wells != 0u); mask; mask &= mask - 1u) {
                const int b = __ffs(mask) - 1;
                const float px = __shfl_sync(kFull, t.px, b), py = __shfl_sync(kFull, t.py, b), pz = __shfl_sync(kFull, t.pz, b);
                const float vx = __shfl_sync(kFull, t.vx, b), vy = __shfl_sync(kFull, t.vy, b), vz = __shfl_sync(kFull, t.vz, b);
                fold_sample(m, st, [&] { return s64; }, Dxa, Dya, Dza, items + 2 * (size_t)__shfl_sync(kFull, i, b),
                            __shfl_sync(kFull, wells, b), px, py, pz, vx, vy, vz, act, g, use_sum);
            }
        }
    }
    f.mloc = g.mloc;
    f.sloc = g.sloc;
}

// Near-tie flag of step k0 + c (one warp).
template <bool GEN>
__device__ __forceinline__ void tie_step(const RolloutArgs& a, IdxState* st, int r, int k0, int c, int best) {
    const int lane = threadIdx.x & 31;
    const float4* t = st->tie[c & (kPub - 1)];
    const uint32_t qk = __float_as_uint(t[lane].x);
    const uint32_t k2nd = __reduce_max_sync(kFull, lane == best ? 0u : qk);
    const unsigned sm2 = __ballot_sync(kFull, qk == k2nd && k2nd != 0u && lane != best);
    const float4 t1 = t[best], t2 = t[sm2 ? __ffs(sm2) - 1 : best];
    if (lane == 0) {
        auto cls = [](float key) {  // see action_key
            const uint32_t u = __float_as_uint(key);
            return u > 0x80000000u ? 2 : (u == 0x80000000u ? 1 : 0);
        };
        // log2 max(g, N): a penalty of zero has no logarithm
        const float s1 = fmaxf(t1.z, t1.w > 0.f ? __log2f(t1.w) : -INFINITY);
        const float s2 = fmaxf(t2.z, t2.w > 0.f ? __log2f(t2.w) : -INFINITY);
        // two positive values whose logarithms differ by more than 3e-4 differ by more than twice the
        // bar (1 - 2^-3e-4 = 2.1e-4) of the larger one: no tie while that is about the scale
        const bool clear = cls(t1.x) == 2 && cls(t2.x) == 2 && t1.y - t2.y > 3e-4f && fmaxf(s1, s2) <= t1.y + 0.5f;
        const bool tie = sm2 && !clear && near_tie(cls(t1.x), cls(t2.x), t1.y, t2.y, s1, s2);
        if (tie) atomicAdd(&st->near_ties, 1);
        if (GEN && a.trace && r == 0) a.tie_trace[k0 + c] = tie ? 1 : 0;
        else if (a.pipe.ties) a.pipe.ties[(size_t)r * a.cap + k0 + c] = tie ? 1 : 0;
    }
    __syncwarp();
}

// Records step k0 + c (one warp; rs: the exact coordinate of lanes 0 .. 2).
template <bool GEN>
__device__ __forceinline__ void record_step(const RolloutArgs& a, IdxState* st, int r, int k0, int c, float* traj,
                                            uint8_t* acts, double& rs) {
    const int lane = threadIdx.x & 31;
    const PubState p = st->ps[(c + 1) & (kPub - 1)];
    if (p.what & kPubNone) return;
    const int k = k0 + c, np = k + 1;
    const int best = p.what & 0xff, hn = (p.what >> 8) & 0xff;
    if (lane < 3) {
        rs = __dadd_rn(rs, lane == 0 ? st->Dx[hn] : (lane == 1 ? st->Dy[hn] : st->Dz[best]));
        st->s64[(c + 1) & (kPub - 1)][lane] = rs;
    }
    __syncwarp();
    if (lane == 0) {
        __threadfence_block();
        *(volatile int*)&st->rec_steps = c + 1;
    }
    const size_t off = (size_t)r * a.cap;
    if (lane < 3) {
        traj[3 * (size_t)np + lane] = (float)rs;
        if (a.pipe.obs) a.pipe.st_s[3 * (off + np) + lane] = rs;
        if (GEN && a.trace && r == 0) a.st_trace[3 * (size_t)np + lane] = rs;
    }
    if (lane == 3) acts[k] = (uint8_t)best;
    if (GEN && a.trace && r == 0 && lane == 4) a.hd_trace[np] = hn;
    if (a.pipe.obs) {  // what a resumed plan and the host's influence test need
        if (lane == 5) a.pipe.obs[off + k] = p.pub;
        if (lane == 6) a.pipe.st_h[off + np] = (uint8_t)hn;
        if (lane >= 8 && lane < 14) {
            const int q = lane - 8;
            const float x = q == 0 ? p.hx : q == 1 ? p.lx : q == 2 ? p.hy : q == 3 ? p.ly : q == 4 ? p.hz : p.lz;
            a.pipe.st_df[6 * (off + np) + q] = x;
        }
    }
    tie_step<GEN>(a, st, r, k0, c, best);
}

// Plans request r with this CTA. Every thread calls it; all shared memory it uses is
// re-initialised, so a CTA can plan requests back to back. k0 > 0 (pipelined mode): the plan
// keeps its first k0 steps and resumes from its state at step k0, as stored by the run that
// planned them. tbase: the first step of the table window the plan reads. GEN: the general
// instance, with the uncommon features (phase clock stamps, trace, SUM combination, static wells).
template <bool GEN>
__device__ __forceinline__ void plan_indexed(const RolloutArgs& a, const int r, unsigned char* smem, const int64_t tbase,
                                             const int k0 = 0) {
    const Model& m = a.m;
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, NW = NT >> 5;
    const fmdp_request req = a.reqs[r];
    const int A = m.A;
    IdxState* st = reinterpret_cast<IdxState*>(smem);
    const int lcap = list_capacity(a.icap);
    float4* lists = reinterpret_cast<float4*>(smem + idx_lists_offset());
    float* traj = a.traj + (size_t)r * a.cap * 3;
    uint8_t* acts = a.acts + (size_t)r * a.cap;
    const size_t rec_off = (size_t)r * a.cap;
    // FCFS ordinal of this request: tentative plans of later requests are not part of its table
    const int32_t my_ord = a.pipe.on ? a.pipe.ord0 + r : INT_MAX;
    const PlanRoles R = plan_roles(NW, warp);
    const int n_meet = 32 * (2 + R.n_fold + (R.own_terrain ? 1 : 0));  // threads that meet at the named barriers

    // ---------------------------------------------------------------- prologue
    if (tid < kHeadings) {
        const double dx = __dsub_rn(req.gx, req.ox), dy = __dsub_rn(req.gy, req.oy);
        const double Lh = __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
        double c0 = 1.0, s0 = 0.0;
        if (Lh > 0.0) { c0 = __ddiv_rn(dx, Lh); s0 = __ddiv_rn(dy, Lh); }
        double ck, sk;
        unit15(tid, ck, sk);
        const double C = __dsub_rn(__dmul_rn(c0, ck), __dmul_rn(s0, sk));
        const double S = __dadd_rn(__dmul_rn(s0, ck), __dmul_rn(c0, sk));
        const double step = __dmul_rn(req.speed_mps, m.dt);
        const double X = __dmul_rn(step, C), Y = __dmul_rn(step, S);
        st->Dx[tid] = X;
        st->Dy[tid] = Y;
        const float xh = (float)X, yh = (float)Y;
        st->Dxy[tid] = make_float4(xh, (float)__dsub_rn(X, (double)xh), yh, (float)__dsub_rn(Y, (double)yh));
    }
    if (tid >= 32 && tid < 32 + kMaxActions) {
        const int q = tid - 32;
        const double dz = q < A ? __dmul_rn(m.climb[q], m.dt) : 0.0;
        st->Dz[q] = dz;
        const float zh = (float)dz;
        st->Dzf[q] = make_float2(zh, (float)__dsub_rn(dz, (double)zh));
    }
    if (tid >= 64 && tid < 64 + kSlots) mbar_init(&st->full[tid - 64], 1);
    if (tid >= 96 && tid < 96 + kPub) mbar_init(&st->seen[tid - 96], 1);
    if (tid >= 112 && tid < 112 + kPub) mbar_init(&st->seen_rec[tid - 112], 1);
    if (GEN)
        for (int q = tid; q < 3 * m.n_static; q += NT) {
            const double c = m.statics[6 * (q / 3) + q % 3];
            const float hi = (float)c;
            st->stat_hi[q / 3][q % 3] = hi;
            st->stat_lo[q / 3][q % 3] = (float)__dsub_rn(c, (double)hi);
        }
    if (tid == 0) {
        const double step = __dmul_rn(req.speed_mps, m.dt);
        st->step = step;
        st->cap2 = __dmul_rn(step, step);
        // a successor lies within step + max |climb| dt of the state; a well whose centre
        // is farther than R + that + 1 m misses every successor by more than 1 m
        float dzm = 0.f;
        for (int q = 0; q < A; ++q) dzm = fmaxf(dzm, fabsf((float)__dmul_rn(m.climb[q], m.dt)));
        for (int w = 0; w < m.n_wells; ++w) {
            const float lim = sqrtf(m.w_R2[w]) + (float)step + dzm + 1.f;
            st->well[w] = make_float4(m.w_tau[w], m.w_R2[w], m.w_lg[w], m.w_L[w]);
            st->reach[w] = make_float2(m.w_tau[w], lim * lim);
        }
        const double s0[3] = {req.ox, req.oy, req.oz};
        PubState p;
        if (k0 > 0) {  // the state as the step that reached it published it
            const size_t o = rec_off + k0;
            for (int q = 0; q < 3; ++q) st->s64[0][q] = a.pipe.st_s[3 * o + q];
            const float* df = a.pipe.st_df + 6 * o;
            p.hx = df[0], p.lx = df[1], p.hy = df[2], p.ly = df[3], p.hz = df[4], p.lz = df[5];
            p.what = (int)a.pipe.st_h[o] << 8;
            st->captured0 = 0;  // the run that planned these steps went on from step k0
        } else {
            for (int q = 0; q < 3; ++q) st->s64[0][q] = s0[q];
            p.hx = (float)s0[0], p.hy = (float)s0[1], p.hz = (float)s0[2];
            p.lx = (float)__dsub_rn(s0[0], (double)p.hx);
            p.ly = (float)__dsub_rn(s0[1], (double)p.hy);
            p.lz = (float)__dsub_rn(s0[2], (double)p.hz);
            p.what = 0;
            st->captured0 = capture_exact_at(s0[0], s0[1], s0[2], req, st->cap2) ? 1 : 0;
        }
        p.pub = INT_MAX;
        st->ps[0] = p;
        st->best[1] = 0;  // step 0 starts from next[1][0]
        st->fold_abort = 0;
        st->rec_steps = 0;
        st->stop = 0;
        st->near_ties = 0;
        traj[0] = (float)req.ox; traj[1] = (float)req.oy; traj[2] = (float)req.oz;
        if (GEN && a.trace && r == 0) {
            a.st_trace[0] = req.ox; a.st_trace[1] = req.oy; a.st_trace[2] = req.oz;
            a.hd_trace[0] = 0;
        }
    }
    mbar_fence_init();
    __syncthreads();
    if (k0 > 0) {  // near ties of the kept steps
        int nt = 0;
        for (int i = tid; i < k0; i += NT) nt += a.pipe.ties[rec_off + i];
        if (nt) atomicAdd(&st->near_ties, nt);
    }

    const float stepf = (float)st->step;
    float dzmax = 0.f;
    for (int i = 0; i < A; ++i) dzmax = fmaxf(dzmax, fabsf(st->Dzf[i].x));
    const float reach0 = m.reach_base + stepf + dzmax;
    const float inv_dt = (float)(1.0 / m.dt);
    const float box0 = (float)m.box[0], box1 = (float)m.box[1];
    const bool over = st->captured0 != 0 || (k0 == 0 && req.horizon <= 0);  // nothing to plan
    const bool timing = GEN && a.phase != nullptr;
    unsigned long long ph[6] = {0, 0, 0, 0, 0, 0};
    unsigned qe_items = 0u, qe_dnear = 0u, qe_wells = 0u;  // statistics: see RolloutArgs::qe_ctr

    if (over) {
        if (tid == 0) {
            st->status = st->captured0 ? kStatusCaptured : FMDP_REJ_HORIZON;
            st->n_points = 1;
            st->steps = 0;
        }
    } else if (R.role <= kFold) {
        // the exact state of step k0 + c, for a decision inside an FP64 band
        const volatile int* rec_steps = &st->rec_steps;
        auto wait_steps = [&](const volatile int* done, int c) {
            const long long t0 = clock64();
            while (*done < c)
                if (clock64() - t0 > (1ll << 31)) {
                    atomicExch(a.err, FMDP_ERR_TIMEOUT);
                    break;
                }
            __threadfence_block();
        };
        auto exact_state = [&](int c) -> const double* {
            wait_steps(rec_steps, c);
            return st->s64[c & (kPub - 1)];
        };
        const bool act = lane < A;
        const int my_dh = act ? m.dh[lane] : 0;
        const float2 my_dz = st->Dzf[lane];
        const bool has_goal = m.goal_reward > 0.0;
        const bool combine = GEN && m.combine != 0;
        const float lg32 = m.lg32, sum_ref = m.sum_ref;
        // heading index after this lane's action's turn, wrapped to [0, 24)
        auto turned = [&](int h) {
            int hn = h + my_dh;
            hn += hn < 0 ? 24 : 0;
            hn -= hn >= 24 ? 24 : 0;
            return hn;
        };

        // the clearance penalty of this lane's successor: heightmap nodes from the patch if there is one
        const float* __restrict__ hm = m.hm;
        const bool trace0 = GEN && a.trace && r == 0;
        DeckGrid grid{};
        if (hm && (R.role == kTerrain || (R.role == kControl && !R.own_terrain))) grid = deck_grid(m);
        auto deck_penalty = [&](int c, const NextState& s, const float4 D, int hn, int patch_x, int patch_y) {
            const float clr = (float)m.clearance;
            const float sx = s.hx + (s.lx + D.x), sy = s.hy + (s.ly + D.z), sz = s.hz + (s.lz + my_dz.x);
            TerrainCell tc = terrain_cell(sx, sy, box0, box1, m.hm_sx, m.hm_sy, m.hm_nx, m.hm_ny);
            const int px = tc.ix - patch_x, py = tc.iy - patch_y;
            if (patch_x >= 0 && (unsigned)px < kPatch - 1 && (unsigned)py < kPatch - 1) {
                const float* n = st->patch + py * kPatch + px;
                tc.h00 = n[0], tc.h10 = n[1], tc.h01 = n[kPatch], tc.h11 = n[kPatch + 1];
            } else {
                terrain_nodes(tc, hm, m.hm_nx);
            }
            const float cl = sz - terrain_height(tc);
            float Vd = cl < clr ? (float)m.deck - cl : 0.f;
            if (act && fabsf(cl - clr) < kClrBand) {
                float hx = s.hx, lx = s.lx, hy = s.hy, ly = s.ly, hz = s.hz, lz = s.lz;
                df_add(hx, lx, D.x, D.y);
                df_add(hy, ly, D.z, D.w);
                df_add(hz, lz, my_dz.x, my_dz.y);
                Vd = deck_band(m, grid, tc, hx, lx, hy, ly, hz, lz, k0 + c);
                if (Vd < 0.f) Vd = deck_exact(m, exact_state(c), st->Dx[hn], st->Dy[hn], st->Dz[lane]);
            }
            return Vd;
        };
        if (R.role == kTerrain) {
            // -------------------------------------------------------- terrain
            bar_arrive(kBarReady, n_meet);
            // the patch holds the cells of every successor two steps on from the state it is made for
            const bool fits = (int)(2.f * stepf * fmaxf(m.hm_sx, m.hm_sy)) + 1 <= kPatch / 2 - 1 && m.hm_nx >= kPatch &&
                              m.hm_ny >= kPatch;
            int patch_x = -1, patch_y = 0;
            auto load_patch = [&](float x, float y) {
                if (!hm || !fits) return;
                patch_x = min(max((int)floorf((x - box0) * m.hm_sx) - (kPatch / 2 - 1), 0), m.hm_nx - kPatch);
                patch_y = min(max((int)floorf((y - box1) * m.hm_sy) - (kPatch / 2 - 1), 0), m.hm_ny - kPatch);
                const float* q = hm + (size_t)(patch_y + (lane >> 3)) * m.hm_nx + patch_x + (lane & 7);
                const float u = __ldg(q), v = __ldg(q + 4 * (size_t)m.hm_nx);
                st->patch[lane] = u;
                st->patch[lane + 32] = v;
                __syncwarp();
            };
            load_patch(st->ps[0].hx, st->ps[0].hy);
            for (int c = 0;; ++c) {
                bar_wait(kBarChosen, n_meet);
                const int best = *(volatile int*)&st->best[(c + 1) & 1];
                if (best == kNoAction) break;
                const NextState s = st->next[(c + 1) & 1][best];
                if ((s.packed & 32) || k0 + c >= req.horizon) break;
                const int hn = turned(s.packed & 31);
                if (hm) st->deck[lane] = deck_penalty(c, s, st->Dxy[hn], hn, patch_x, patch_y);
                __syncwarp();
                bar_arrive(kBarReady, n_meet);
                load_patch(s.hx, s.hy);  // for the next step, while the control warp compares the actions
            }
        } else if (R.role == kSuccessor) {
            // -------------------------------------------------------- successor
            const float lg_hi = (float)m.lg64, lg_lo = (float)(m.lg64 - (double)(float)m.lg64);
            const float l2r_hi = has_goal ? (float)m.log2rg : 0.f;
            const float l2r_lo = has_goal ? (float)(m.log2rg - (double)(float)m.log2rg) : 0.f;
            float gh[3], gl[3];  // goal as double-float
            {
                const double g0[3] = {req.gx, req.gy, req.gz};
                for (int q = 0; q < 3; ++q) {
                    gh[q] = (float)g0[q];
                    gl[q] = (float)__dsub_rn(g0[q], (double)gh[q]);
                }
            }
            // the first state as an entry: its goal vector from FP64, or (a resumed plan) formed from
            // the double-float state exactly as a step forms it
            {
                const PubState p0 = st->ps[0];
                NextState n;
                n.hx = p0.hx, n.hy = p0.hy, n.hz = p0.hz, n.lx = p0.lx, n.ly = p0.ly, n.lz = p0.lz;
                float Gh[3], Gl[3];
                const float sh[3] = {p0.hx, p0.hy, p0.hz}, sl[3] = {p0.lx, p0.ly, p0.lz};
                const double g0[3] = {req.gx, req.gy, req.gz};
                for (int q = 0; q < 3; ++q) {
                    if (k0 > 0) {
                        Gh[q] = gh[q], Gl[q] = gl[q];
                        df_add(Gh[q], Gl[q], -sh[q], -sl[q]);
                    } else {
                        const double G = __dsub_rn(g0[q], st->s64[0][q]);
                        Gh[q] = (float)G;
                        Gl[q] = (float)__dsub_rn(G, (double)Gh[q]);
                    }
                }
                int n0;
                float phi;
                goal_log_split(Gh[0], Gh[1], Gh[2], Gl[0], Gl[1], Gl[2], lg_hi, lg_lo, l2r_hi, l2r_lo, n0, phi);
                n.Gx = Gh[0] + Gl[0], n.Gy = Gh[1] + Gl[1], n.Gz = Gh[2] + Gl[2];
                n.packed = p0.what >> 8;
                n.pad0 = n.pad1 = 0.f;
                if (lane == 0) {
                    st->next[1][0] = n;
                    st->split[1][0] = make_float2(__int_as_float(n0), phi);
                }
                __syncwarp();
                bar_arrive(kBarReady, n_meet);  // (the control warp waits for it once before its first step)
            }
            const double cap2 = st->cap2;
            double rs = !R.own_recorder && lane < 3 ? st->s64[0][lane] : 0.0;
            int recorded = 0;  // steps recorded (without a recorder warp)
            // state c for the helpers and the recorder (state 0 was published at the start)
            auto publish = [&](int c, const NextState& s, int best, bool done, bool none) {
                if (c == 0) return;
                if (lane == 0) {
                    PubState p;
                    p.hx = s.hx, p.hy = s.hy, p.hz = s.hz, p.lx = s.lx, p.ly = s.ly, p.lz = s.lz;
                    p.what = best | ((s.packed & 31) << 8) | (done ? kPubDone : 0) | (none ? kPubNone : 0);
                    p.pub = st->meta[(c - 1) & (kSlots - 1)].pub;
                    st->ps[c & (kPub - 1)] = p;
                    if (done) *(volatile int*)&st->stop = 1;
                }
                __syncwarp();
                if (lane < 2) mbar_arrive(lane == 0 ? &st->seen[(c - 1) & (kPub - 1)] : &st->seen_rec[(c - 1) & (kPub - 1)]);
                // the helpers that wait for a later state (at most n_help steps ahead) wake and see `stop`
                if (done && lane > 0 && lane < kPub) mbar_arrive(&st->seen[(c - 1 + lane) & (kPub - 1)]);
                __syncwarp();
            };
            float Gnhx = 0.f, Gnhy = 0.f, Gnhz = 0.f, Gnlx = 0.f, Gnly = 0.f, Gnlz = 0.f;  // of the last step's successors
            for (int c = 0;; ++c) {
                bar_wait(kBarChosen, n_meet);
                const int best = *(volatile int*)&st->best[(c + 1) & 1];
                const bool none = best == kNoAction;
                const NextState s = st->next[(c + 1) & 1][none ? 0 : best];
                const bool done = none || (s.packed & 32) || k0 + c >= req.horizon;  // captured, or out of steps
                bool told = false;
                if (!R.own_recorder) {  // (the exact state is this warp's work too, and others may need it now)
                    publish(c, s, best, done, none);
                    told = true;
                    for (; recorded < c; ++recorded) record_step<GEN>(a, st, r, k0, recorded, traj, acts, rs);
                    __syncwarp();
                }
                if (!done) {
                    const int hn = turned(s.packed & 31);
                    const float4 D = st->Dxy[hn];
                    NextState n;
                    n.hx = s.hx, n.hy = s.hy, n.hz = s.hz, n.lx = s.lx, n.ly = s.ly, n.lz = s.lz;
                    df_add(n.hx, n.lx, D.x, D.y);
                    df_add(n.hy, n.ly, D.z, D.w);
                    df_add(n.hz, n.lz, my_dz.x, my_dz.y);
                    // goal vector at the successor and its capture test
                    Gnhx = gh[0], Gnlx = gl[0], Gnhy = gh[1], Gnly = gl[1], Gnhz = gh[2], Gnlz = gl[2];
                    df_add(Gnhx, Gnlx, -n.hx, -n.lx);
                    df_add(Gnhy, Gnly, -n.hy, -n.ly);
                    df_add(Gnhz, Gnlz, -n.hz, -n.lz);
                    n.Gx = Gnhx + Gnlx, n.Gy = Gnhy + Gnly, n.Gz = Gnhz + Gnlz;
                    bool capn = false;
                    const bool close = act && approx_sqrt(n.Gx * n.Gx + n.Gy * n.Gy + n.Gz * n.Gz) < stepf + kCapBand;
                    if (!told && __any_sync(kFull, close)) {  // (the recorder must have this state to make it exact)
                        publish(c, s, best, done, none);
                        told = true;
                    }
                    if (close) {
                        const double* x = exact_state(c);
                        capn = capture_exact_at(__dadd_rn(x[0], st->Dx[hn]), __dadd_rn(x[1], st->Dy[hn]),
                                                __dadd_rn(x[2], st->Dz[lane]), req, cap2);
                    }
                    n.packed = (capn ? 32 : 0) | hn;
                    n.pad0 = n.pad1 = 0.f;
                    st->next[c & 1][lane] = n;
                    __syncwarp();
                    bar_arrive(kBarReady, n_meet);
                }
                // ---- off the chain: the state is published, and the goal term of the successors split
                if (!told) publish(c, s, best, done, none);
                if (done) break;
                int n0n;
                float phin;
                goal_log_split(Gnhx, Gnhy, Gnhz, Gnlx, Gnly, Gnlz, lg_hi, lg_lo, l2r_hi, l2r_lo, n0n, phin);
                st->split[c & 1][lane] = make_float2(__int_as_float(n0n), phin);
                __syncwarp();
            }
        } else if (R.role == kFold) {
            // -------------------------------------------------------- fold
            FoldLane f;
            f.dza = my_dz.x;
            bar_arrive(kBarReady, n_meet);
            for (int c = 0;; ++c) {
                // the step's list is there before the state it is scored for: this lane's first sample is
                // loaded ahead of the barrier (a list that never comes is reported after it)
                const bool ready =
                    __all_sync(kFull, idx_wait_list(st, c));
                const ListMeta& M = st->meta[c & (kSlots - 1)];
                const bool good = ready && !M.abort && M.n <= lcap;
                const int n_list = good ? M.n : 0;
                // sample i of this warp is entry i n_fold + index of the list
                const float4* L = lists + (size_t)(c & (kSlots - 1)) * lcap * 2 + 2 * R.index;
                float4 e0 = make_float4(0.f, 0.f, 0.f, 0.f), e1 = e0;
                if (lane * R.n_fold + R.index < n_list) {
                    e0 = L[2 * lane * R.n_fold];
                    e1 = L[2 * lane * R.n_fold + 1];
                }
                bar_wait(kBarChosen, n_meet);
                const int best = *(volatile int*)&st->best[(c + 1) & 1];
                if (best == kNoAction) break;
                const NextState* s = &st->next[(c + 1) & 1][best];
                const int packed = s->packed;
                if ((packed & 32) || k0 + c >= req.horizon) break;
                f.shx = s->hx, f.shy = s->hy, f.shz = s->hz, f.slx = s->lx, f.sly = s->ly, f.slz = s->lz;
                const int hn = turned(packed & 31);
                const float4 D = st->Dxy[hn];
                f.dxa = D.x, f.dya = D.z;
                f.mloc = -INFINITY;
                f.sloc = 0ull;
                if (!ready || M.abort) {
                    if (lane == 0) {
                        if (!ready) atomicExch(a.err, FMDP_ERR_TIMEOUT);
                        *(volatile int*)&st->fold_abort = 1;
                    }
                } else if (!good) {  // the list overflowed: one fold warp reads the query's items itself
                    if (R.index == 0) {
                        FoldLane g = f;  // (a copy: the call takes addresses)
                        unsigned pairs = 0u;
                        fold_overflow(a, st, M, my_ord, inv_dt, reach0, exact_state(c), st->Dx[hn], st->Dy[hn], st->Dz[lane],
                                      act, g, combine, pairs);
                        f.mloc = g.mloc;
                        f.sloc = g.sloc;
                        qe_wells += pairs;
                    }
                } else {
                    // lanes = samples for the reach test with this state, then lanes = actions
                    for (int b0 = 0; b0 * R.n_fold < n_list; b0 += 32) {
                        const bool have = (b0 + lane) * R.n_fold + R.index < n_list;
                        if (b0 > 0 && have) {
                            e0 = L[2 * (b0 + lane) * R.n_fold];
                            e1 = L[2 * (b0 + lane) * R.n_fold + 1];
                        }
                        unsigned wells = well_mask(st->reach, m.n_wells, (e0.x - f.shx) - f.slx, (e0.y - f.shy) - f.sly,
                                                   (e0.z - f.shz) - f.slz, e1.x, e1.y, e1.z);
                        wells = have ? wells : 0u;
                        qe_wells += __popc(wells);
                        for (unsigned mask = __ballot_sync(kFull, wells != 0u); mask; mask &= mask - 1u) {
                            const int b = __ffs(mask) - 1;
                            const float4* e = L + 2 * (b0 + b) * R.n_fold;
                            const float4 p = e[0], v = e[1];
                            fold_sample(m, st, [&] { return exact_state(c); }, st->Dx[hn], st->Dy[hn], st->Dz[lane],
                                        a.iv.items + M.row_off + 2 * (size_t)__float_as_int(p.w),
                                        __shfl_sync(kFull, wells, b), p.x, p.y, p.z, v.x, v.y, v.z, act, f, combine);
                        }
                    }
                }
                if (GEN && m.n_static > 0 && R.index == R.n_fold - 1 && act && ready && !M.abort) {  // static wells in reach
                    for (unsigned long long bits = ((unsigned long long)M.stat_hi << 32) | M.stat_lo; bits;
                         bits &= bits - 1ull) {
                        const int w = __ffsll((long long)bits) - 1;
                        const float qx = (st->stat_hi[w][0] - f.shx) + (st->stat_lo[w][0] - f.slx);
                        const float qy = (st->stat_hi[w][1] - f.shy) + (st->stat_lo[w][1] - f.sly);
                        const float qz = (st->stat_hi[w][2] - f.shz) + (st->stat_lo[w][2] - f.slz);
                        const float ex = f.dxa - qx, ey = f.dya - qy, ez = f.dza - qz;
                        const float d2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                        const float R2 = m.st_R2[w], bw = m.st_band[w];
                        if (!(d2 < R2 + bw)) continue;
                        if (!(d2 < R2 - bw) &&
                            !static_inside_exact(m, exact_state(c), st->Dx[hn], st->Dy[hn], st->Dz[lane], w))
                            continue;
                        const float l = fmaf(approx_sqrt(d2), m.st_lg[w], m.st_L[w]);
                        f.mloc = fmaxf(f.mloc, l);
                        if (combine) f.sloc += sum_term(l, sum_ref);
                    }
                }
                __syncwarp();
                st->fold_max[R.index][lane] = f.mloc;
                if (combine) st->fold_sum[R.index][lane] = f.sloc;
                __syncwarp();
                bar_arrive(kBarReady, n_meet);
            }
        } else {
            // -------------------------------------------------------- control
            const float box2 = (float)m.box[2], box3 = (float)m.box[3], box4 = (float)m.box[4], box5 = (float)m.box[5];
            const float sum_unit = exp2f(sum_ref - (float)kSumBits);  // value of one unit of the fixed-point sum
            int status = FMDP_REJ_HORIZON, steps = k0;
            bar_wait(kBarReady, n_meet);   // the first state's entry is written
            bar_arrive(kBarChosen, n_meet);
            int best = 0;
            for (int c = 0;; ++c) {
                const int k = k0 + c;
                const long long t0 = timing ? clock64() : 0;
                const NextState s = st->next[(c + 1) & 1][best];  // the winner's successor is the state
                if ((s.packed & 32) || k >= req.horizon) {
                    status = (s.packed & 32) ? kStatusCaptured : FMDP_REJ_HORIZON;
                    steps = k;
                    break;
                }
                const int hn = turned(s.packed & 31);
                const float4 D = st->Dxy[hn];
                const float dxa = D.x, dya = D.z, dza = my_dz.x;
                // goal distance change of the action
                const float Dl = goal_change(s.Gx, s.Gy, s.Gz, dxa, dya, dza);
                // successor estimate (fp32); box validity: exact comparison near a face
                const float sx = s.hx + (s.lx + dxa), sy = s.hy + (s.ly + dya), sz = s.hz + (s.lz + dza);
                const float mb = box_margin(sx, sy, sz, box0, box1, box2, box3, box4, box5);
                bool valid = mb > kBoxBand;
                if (act && fabsf(mb) <= kBoxBand)
                    valid = box_inside_exact(m, exact_state(c), st->Dx[hn], st->Dy[hn], st->Dz[lane]);
                // the recorder must not fall so far behind that its ring entries are overwritten
                if (c > kRecLag && *rec_steps < c - kRecLag) wait_steps(rec_steps, c - kRecLag);
                float Vd = 0.f;
                if (hm && !R.own_terrain) Vd = deck_penalty(c, s, D, hn, -1, 0);
                __syncwarp();
                const long long t1 = timing ? clock64() : 0;
                bar_wait(kBarReady, n_meet);  // B: successors, wells and clearance ready
                const long long t2 = timing ? clock64() : 0;
                const float2 split = st->split[(c + 1) & 1][best];
                const int n0 = __float_as_int(split.x);
                const float phi = split.y;
                const float sc0 = exp2f((float)-n0);  // 2^-n0 of the current state
                if (hm && R.own_terrain) Vd = st->deck[lane];
                float mloc = st->fold_max[0][lane];
                unsigned long long ssum = combine ? st->fold_sum[0][lane] : 0ull;
                if (R.n_fold > 1) {
                    mloc = fmaxf(mloc, st->fold_max[1][lane]);
                    if (combine) ssum += st->fold_sum[1][lane];
                }
                // ---- action values as (sign class, log2 |Q|) keys; Q = g - P - V (Alg. 1, Alg. 8)
                ActionValue v;
                float Nl;
                const float Lp = combine ? (ssum ? __log2f((float)ssum) + (sum_ref - (float)kSumBits) : -INFINITY) : mloc;
                action_value(combine, has_goal, ssum, Lp, Vd, sum_unit, phi, Dl, lg32, n0, sc0, v, Nl);
                const uint32_t qkey = (act && valid) ? action_key(v.cls, v.k2) : 0u;
                const uint32_t kmax = __reduce_max_sync(kFull, qkey);
                const unsigned bm = __ballot_sync(kFull, qkey == kmax && kmax != 0u);
                const bool none = !bm || *(volatile int*)&st->fold_abort != 0;
                best = none ? kNoAction : __ffs(bm) - 1;
                if (lane == 0) *(volatile int*)&st->best[c & 1] = best;
                // for the near-tie flag
                st->tie[c & (kPub - 1)][lane] =
                    make_float4(__uint_as_float(qkey), v.la, has_goal ? __fadd_rn(fmaf(Dl, lg32, phi), (float)n0) : -INFINITY, Nl);
                __syncwarp();
                bar_arrive(kBarChosen, n_meet);  // A: the next step
                if (trace0 && act)  // FP64 action values for the trace (not used for the decision)
                    a.q_trace[(size_t)k * A + lane] = valid ? trace_q(m, has_goal, n0, phi, Dl, Lp, ssum, Vd) : -INFINITY;
                if (timing) {
                    const long long t = clock64();
                    ph[0] += t1 - t0;
                    ph[2] += t2 - t1;
                    ph[3] += t - t2;
                }
                if (none) {
                    status = FMDP_REJ_NO_ACTION;
                    steps = k;
                    break;
                }
            }
            if (lane == 0) {
                st->status = status;
                st->steps = steps;
                st->n_points = steps + 1;
            }
        }
    } else if (R.role == kRecorder) {
        // ------------------------------------------------------------ behind the chain
        double rs = lane < 3 ? st->s64[0][lane] : 0.0;  // lanes 0 .. 2 carry the exact x, y, z
        for (int c = 0;; ++c) {
            if (!__all_sync(kFull, idx_wait(&st->seen_rec[c & (kPub - 1)], (uint32_t)((c / kPub) & 1)))) {
                if (lane == 0) atomicExch(a.err, FMDP_ERR_TIMEOUT);
                break;
            }
            const long long t0 = timing ? clock64() : 0;
            const int what = st->ps[(c + 1) & (kPub - 1)].what;
            if (what & kPubNone) break;
            record_step<GEN>(a, st, r, k0, c, traj, acts, rs);
            if (timing) ph[5] += clock64() - t0;
            if (what & kPubDone) break;
        }
    } else {
        // ------------------------------------------------------------ helpers
        const IndexView& iv = a.iv;
        const int64_t cst_len = (int64_t)iv.ncell + 1;
        const int32_t T_win = a.tab.T_win;
        const float delta = stepf + dzmax + 0.02f;  // largest distance between the states of two steps
        // a query covers every cell within this of the state it is made from (an item outside the
        // extra list moves no faster than vmax), one step's move included
        const float Rq = reach0 + m.tau_absmax * iv.vmax * 1.0001f + stepf + 2.0f;
        // steps whose rows lie in the table window: [c_lo, c_hi) of this run's steps
        const int64_t T1 = req.depart_step + k0 + 1;
        const int64_t lo64 = tbase - T1, hi64 = tbase + T_win - T1;
        const int c_lo = lo64 < 0 ? 0 : (lo64 > (1 << 30) ? 1 << 30 : (int)lo64);
        const int c_hi = hi64 < 0 ? 0 : (hi64 > (1 << 30) ? 1 << 30 : (int)hi64);
        int64_t row64 = (T1 + R.index) % T_win;
        int row = (int)(row64 < 0 ? row64 + T_win : row64);
        const int n_help = R.n_help;
        auto cell_of = [&](float v, float o, int n) {
            const float g = floorf((v - o) * iv.inv_cell);
            return g < 0.f ? 0 : (g > (float)(n - 1) ? n - 1 : (int)g);
        };
        // One or two list warps set the pace of the steps, so they read the bounds of their next list
        // before the items of this one: two loads that depend on one another beside two more. (They
        // start with a turn that only reads bounds.) 64 rollouts among 3000 plans, 128 threads: 2.96
        // to 2.55 ms. More of them are ahead of the chain anyway, and would ask from a state that is
        // several steps older, for more cells.
        const int early = n_help <= 2 ? n_help : 0;
        int lo_next = 0, hi_next = 0, pub_next = INT_MAX;
        int64_t off_next = 0;
        for (int c = R.index - early;; c += n_help) {
            const int from = max(c - kAhead, 0);  // the state the list is made from
            const int got = from > 0 ? __reduce_min_sync(kFull, idx_wait_state(st, from)) : 1;
            if (got < 0) {
                if (lane == 0) {
                    atomicExch(a.err, FMDP_ERR_TIMEOUT);
                    st->meta[c & (kSlots - 1)].abort = 1;
                    mbar_arrive(&st->full[c & (kSlots - 1)]);
                }
                break;
            }
            if (got == 0 || *(volatile int*)&st->stop) break;
            const long long t0 = timing ? clock64() : 0;
            const PubState p = st->ps[from & (kPub - 1)];
            const float x = p.hx + p.lx, y = p.hy + p.ly;
            const float margin = (float)(c - from) * delta;
            // ---- item ranges of the query, one per lane (the extra list last): lo to hi, or hi items
            int lo = 0, hi = 0, pub = INT_MAX;
            {
                const int cb = c + early;  // the list they are for
                if (cb >= c_lo && cb < c_hi) {
                    const int32_t* cs_row = iv.cstart + row * cst_len;
                    const float R = Rq + (float)max(cb - from - 1, 0) * stepf;
                    const int cx0 = cell_of(x - R, iv.x0, iv.ncx), cx1 = cell_of(x + R, iv.x0, iv.ncx);
                    const int cy0 = cell_of(y - R, iv.y0, iv.ncy), cy1 = cell_of(y + R, iv.y0, iv.ncy);
                    const int nrows = cy1 - cy0 + 1;
                    // L2 loads (.cg): the index may change while a persistent launch runs (extra lists
                    // published, rows rebuilt between launches), so nothing of it is kept in L1
                    if (nrows < kMaxRanges) {
                        if (lane < nrows) {
                            lo = __ldcg(cs_row + (cy0 + lane) * iv.ncx + cx0);
                            hi = __ldcg(cs_row + (cy0 + lane) * iv.ncx + cx1 + 1);
                        }
                    } else if (lane == 0) {  // one range over full cell rows
                        lo = __ldcg(cs_row + cy0 * iv.ncx);
                        hi = __ldcg(cs_row + (cy1 + 1) * iv.ncx);
                    }
                    if (lane == kMaxRanges - 1) {
                        // the count of published operations first (acquire), then the extra list's length:
                        // every operation counted is in the list this query reads
                        if (a.pipe.pub_seq) pub = ld_acquire_gpu(a.pipe.pub_seq);
                        lo = __ldcg(cs_row + iv.ncell);
                        hi = __ldcg(iv.nextra + row);
                    }
                }
            }
            int64_t row_off = (int64_t)row * a.tab.S_pad * 2;
            row += n_help;
            while (row >= T_win) row -= T_win;
            if (early) {  // this turn's list is the one the last turn's bounds are for
                const int64_t off = off_next;
                const int l = lo_next, h = hi_next, q = pub_next;
                off_next = row_off, lo_next = lo, hi_next = hi, pub_next = pub;
                if (c < 0) continue;
                row_off = off, lo = l, hi = h, pub = q;
            }
            ListMeta& M = st->meta[c & (kSlots - 1)];
            const int beg = lo, num = max(0, lane == kMaxRanges - 1 ? hi : hi - lo);
            pub = __shfl_sync(kFull, pub, kMaxRanges - 1);
            if (GEN && m.n_static > 0) {  // static wells that can reach a successor by then
                unsigned bits[2];
                for (int u = 0; u < 2; ++u) {
                    const int w = 32 * u + lane;
                    bool in = false;
                    if (w < m.n_static) {
                        const double* q = m.statics + 6 * w;
                        const float ex = (float)(q[0] - (double)x), ey = (float)(q[1] - (double)y),
                                    ez = (float)(q[2] - (double)(p.hz + p.lz));
                        const float lim = sqrtf(m.st_R2[w]) + delta + margin + 1.f;
                        in = ex * ex + ey * ey + ez * ez < lim * lim;
                    }
                    bits[u] = __ballot_sync(kFull, in);
                }
                if (lane == 0) M.stat_lo = bits[0], M.stat_hi = bits[1];
            }
            // ---- the items, as one flat list over the ranges
            int at = num;  // inclusive prefix of the ranges' item counts
            for (int o = 1; o < kMaxRanges; o <<= 1) {
                const int v = __shfl_up_sync(kFull, at, o);
                if (lane >= o) at += v;
            }
            const int total = __shfl_sync(kFull, at, kMaxRanges - 1);
            const int base = beg - (at - num);
            if (lane < kMaxRanges) M.beg[lane] = beg, M.cnt[lane] = num;
            __syncwarp();  // (the acquire above comes before the item reads of every lane)
            const float4* items = iv.items + row_off;
            float4* L = lists + (size_t)(c & (kSlots - 1)) * lcap * 2;
            int n_list = 0;
            // 32 U items at a time: loads, then tests (independent chains), then the near ones. One copy
            // of this for every length: on a full chip the warps' code, six roles side by side, waits
            // for instructions. 4000 rollouts among 20 000 plans: 55.8 ms with copies for 32, 64 and
            // 128 items, 40.5 with one for 64 (one for 32: 45, for 96: 50); one rollout: unchanged.
            // (152 CTAs: 65 and 78 % of the instruction cache's requests hit, 5.1 and 1.7 warps per
            // issue wait for an instruction.)
            constexpr int U = 2;
            for (int i0 = 0; i0 < total; i0 += 32 * U) {
                float4 P1[U], P2[U];
                int id[U];
                ItemLane t[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int i = i0 + 32 * u + lane;
                    int lo = 0;  // the range of item i: the first whose prefix exceeds i
#pragma unroll
                    for (int o = kMaxRanges / 2; o; o >>= 1) lo += __shfl_sync(kFull, at, lo + o - 1) <= i ? o : 0;
                    id[u] = __shfl_sync(kFull, base, lo) + i;
                    P1[u] = P2[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (i < total) {
                        P1[u] = __ldcg(items + 2 * (size_t)id[u]);
                        P2[u] = __ldcg(items + 2 * (size_t)id[u] + 1);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    t[u] = item_lane(P1[u], P2[u], i0 + 32 * u + lane < total, my_ord, p.hx, p.hy, p.hz, p.lx, p.ly, p.lz, inv_dt,
                                     m.tau_absmax, reach0 + margin);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned b = __ballot_sync(kFull, t[u].near);
                    const int pos = n_list + __popc(b & ((1u << lane) - 1u));
                    if (t[u].near && pos < lcap) {
                        L[2 * pos] = make_float4(t[u].px, t[u].py, t[u].pz, __int_as_float(id[u]));
                        L[2 * pos + 1] = make_float4(t[u].vx, t[u].vy, t[u].vz, 0.f);
                    }
                    n_list += __popc(b);
                }
            }
            if (lane == 0) {
                M.n = n_list;
                M.pub = pub;
                M.abort = 0;
                M.row_off = row_off;
                qe_items += (unsigned)total;
                qe_dnear += (unsigned)n_list;
                if (a.items_ctr && total > 0) atomicAdd(a.items_ctr, (unsigned long long)total);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&st->full[c & (kSlots - 1)]);
            // cell starts of this helper's next row, into L2 (its query lies near this one)
            if (!early && c >= c_lo && c < c_hi && lane < kMaxRanges - 1) {
                const int cy = cell_of(y + ((float)lane - 3.f) / iv.inv_cell, iv.y0, iv.ncy);
                const int32_t* q = iv.cstart + row * cst_len + cy * iv.ncx + cell_of(x, iv.x0, iv.ncx);
                asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
            }
            if (timing) ph[4] += clock64() - t0;
        }
    }
    __syncthreads();

    // ---------------------------------------------------------------- epilogue
    if (tid == 0) {
        RolloutOut o;
        o.n_points = st->n_points;
        o.status = st->status;
        o.near_ties = st->near_ties;
        o.steps = st->steps;
        a.out[r] = o;
    }
    if (timing && lane == 0)
        for (int i = 0; i < 6; ++i)
            if (ph[i]) atomicAdd(&a.phase[i], ph[i]);
    if (a.qe_ctr) {
        qe_items = __reduce_add_sync(kFull, qe_items);
        qe_dnear = __reduce_add_sync(kFull, qe_dnear);
        qe_wells = __reduce_add_sync(kFull, qe_wells);
        if (lane == 0) {
            if (qe_items) atomicAdd(&a.qe_ctr[0], (unsigned long long)qe_items);
            if (qe_dnear) atomicAdd(&a.qe_ctr[1], (unsigned long long)qe_dnear);
            if (qe_wells) atomicAdd(&a.qe_ctr[2], (unsigned long long)qe_wells);
        }
    }
    if (tid < kSlots) mbar_inval(&st->full[tid]);  // a next request initialises them again
    if (tid >= 32 && tid < 32 + kPub) mbar_inval(&st->seen[tid - 32]);
    if (tid >= 64 && tid < 64 + kPub) mbar_inval(&st->seen_rec[tid - 64]);
    __syncthreads();
}
