// Learned proposal kernels (sm_103a): training-set collection from FastMDP rollouts, the
// optimiser (loss and gradient: train.cu), and policy rollouts that run
// many requests in lock step through the MLP (mma.sync m16n8k16; the weights resident in a
// cluster's shared memory, or streamed by bulk copies past many rows). The network, its inputs
// and its loss are stated in plain FP64 in the oracle.
#include <climits>

#include "learned.cuh"

namespace fmdp {

namespace {

constexpr unsigned kFull = 0xffffffffu;

}  // namespace

// ------------------------------------------------------------------ training-set collection

// One block per request: headings from the recorded actions, then one warp per step. The
// heading recurrence runs in chunks of kHeadChunk steps (one shared array per chunk), so a
// rollout of any length writes one row per step: exactly the n_points - 1 rows the host
// counted for it.
constexpr int kHeadChunk = 2048;
__global__ void __launch_bounds__(256) collect_kernel(const __grid_constant__ CollectArgs a) {
    __shared__ float feat[8][kFeat];
    __shared__ unsigned long long skey[8][kSectors];
    __shared__ int8_t head[kHeadChunk];
    __shared__ int h_carry;
    const int r = blockIdx.x;
    if (r >= a.n) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const fmdp_request req = a.reqs[r];
    const int np = a.rout[r].n_points;
    const int steps = max(np - 1, 0);
    const uint8_t* act = a.acts + (size_t)r * a.cap;
    const float dx = (float)(req.gx - req.ox), dy = (float)(req.gy - req.oy);
    const float L = sqrtf(dx * dx + dy * dy);
    const float c0 = L > 0.f ? dx / L : 1.f, s0 = L > 0.f ? dy / L : 0.f;
    const float inv_dt = (float)(1.0 / a.m.dt);
    if (threadIdx.x == 0) h_carry = 0;
    for (int k0 = 0; k0 < steps; k0 += kHeadChunk) {
        const int k1 = min(steps, k0 + kHeadChunk);
        __syncthreads();  // the previous chunk's headings are no longer read
        if (threadIdx.x == 0) {
            int h = h_carry;
            for (int k = k0; k < k1; ++k) {
                head[k - k0] = (int8_t)h;
                h += a.m.dh[act[k]];
                h += h < 0 ? 24 : 0;
                h -= h >= 24 ? 24 : 0;
            }
            h_carry = h;
        }
        __syncthreads();
        for (int k = k0 + warp; k < k1; k += 8) {
            const float* p = a.traj + ((size_t)r * a.cap + k) * 3;
            float hc, hs;
            heading_cs(c0, s0, head[k - k0], hc, hs);
            const int64_t T1 = req.depart_step + k + 1;
            const int64_t row1 = T1 % a.tab.T_win;
            const bool held = T1 >= a.tab.t_base && T1 < a.tab.t_base + a.tab.T_win;
            warp_features(a.m, a.iv, a.tab, held ? (int)(row1 < 0 ? row1 + a.tab.T_win : row1) : -1, p[0], p[1], p[2], hc, hs,
                          (float)req.speed_mps, (float)req.gx, (float)req.gy, (float)req.gz, inv_dt, feat[warp],
                          skey[warp]);
            const size_t row = (size_t)a.row0[r] + k;
            for (int i = lane; i < kFeat; i += 32) a.X[row * kFeat + i] = __float2bfloat16_rn(feat[warp][i]);
            if (lane == 0) a.y[row] = act[k];
            __syncwarp();
        }
    }
}

cudaError_t launch_collect(const CollectArgs& a, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    collect_kernel<<<a.n, 256, 0, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ training rows and weights

__global__ void gather_rows_kernel(const __nv_bfloat16* X, const int32_t* idx, int M, __nv_bfloat16* out,
                                   const uint8_t* y, uint8_t* y_out) {
    const int row = blockIdx.x;
    if (row >= M) return;
    const int src = idx[row];
    for (int i = threadIdx.x; i < kFeat; i += blockDim.x) out[(size_t)row * kFeat + i] = X[(size_t)src * kFeat + i];
    if (threadIdx.x == 0) y_out[row] = y[src];
}
cudaError_t launch_gather_rows(const __nv_bfloat16* X, const int32_t* idx, int M, __nv_bfloat16* out,
                               const uint8_t* y, uint8_t* y_out, cudaStream_t s) {
    if (M <= 0) return cudaSuccess;
    gather_rows_kernel<<<M, 128, 0, s>>>(X, idx, M, out, y, y_out);
    return cudaGetLastError();
}

// (no step on the gradient of a batch whose kernels gave up a wait: *err is set then)
__global__ void adam_kernel(float* p, const float* g, float* m1, float* m2, size_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2, const int32_t* err) {
    if (*(volatile const int32_t*)err != 0) return;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float a = b1 * m1[i] + (1.f - b1) * gi;
        const float v = b2 * m2[i] + (1.f - b2) * gi * gi;
        m1[i] = a;
        m2[i] = v;
        p[i] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
    }
}
cudaError_t launch_adam(float* p, const float* g, float* m1, float* m2, size_t n, float lr, float b1, float b2,
                        float eps, int t, const int32_t* err, cudaStream_t s) {
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    adam_kernel<<<592, 256, 0, s>>>(p, g, m1, m2, n, lr, b1, b2, eps, c1, c2, err);
    return cudaGetLastError();
}

// bf16 copy of the weights in the chunked layout that the policy and the training kernels stream
__global__ void export_kernel(const float* p, __nv_bfloat16* Wp) {
    for (int l = 0; l < kLayers; ++l) {
        const int in = layer_in(l), out = layer_out(l), op = layer_out_pad(l);
        const float* W = p + param_offset_W(l);
        __nv_bfloat16* wp = Wp + wp_layer_offset(l);
        const size_t n = (size_t)in * op;
        for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
            const int i = (int)(e / op), j = (int)(e % op);
            const __nv_bfloat16 v = __float2bfloat16_rn(j < out ? W[(size_t)i * out + j] : 0.f);
            const int ch = i / kChunkK, kl = i % kChunkK;
            wp[(size_t)ch * wp_chunk_elems(l) + (size_t)j * kChunkPad + kl] = v;
        }
        // row padding of the chunked layout
        const size_t npad = (size_t)(in / kChunkK) * op * (kChunkPad - kChunkK);
        for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < npad; e += (size_t)gridDim.x * blockDim.x) {
            const size_t rowi = e / (kChunkPad - kChunkK), q = e % (kChunkPad - kChunkK);
            wp[rowi * kChunkPad + kChunkK + q] = __float2bfloat16_rn(0.f);
        }
    }
}
cudaError_t launch_export_weights(const float* p, __nv_bfloat16* Wp, cudaStream_t s) {
    export_kernel<<<296, 256, 0, s>>>(p, Wp);
    return cudaGetLastError();
}

// Largest step count the judge accepts for request q: (1 + slack) times the fewest steps
// that can reach the capture ball (radius one step): horizontal motion is exactly one step
// per step, vertical motion at most the largest climb.
__device__ __noinline__ double judge_step_bound(const fmdp_request& q, double dt, double climb_step, double slack) {
    const double step = q.speed_mps * dt;
    const double dh = sqrt((q.gx - q.ox) * (q.gx - q.ox) + (q.gy - q.oy) * (q.gy - q.oy));
    const double dz = fabs(q.gz - q.oz);
    double kmin = fmax(0.0, ceil(dh / step - 1.0));
    if (climb_step > 0.0) kmin = fmax(kmin, ceil((dz - step) / climb_step));
    return floor((1.0 + slack) * kmin + 1e-9);
}

// ------------------------------------------------------------------ policy rollouts

namespace {

// Policy rollouts are a chain of steps per request, and a step a chain of five small matrix
// products, so what counts is the latency of one step. A CTA that streams all weights (475 KB)
// past 16 rows in every step takes 48 000 cycles for it, 35 000 of them for the stream. Here
// the weights stay in the shared memory of a cluster: each of its four CTAs holds 64 columns of
// every hidden layer (119 KB) and multiplies all rows by them, each warp 8 columns; the
// activations of a layer are written to all four CTAs (distributed shared memory, one cluster
// barrier per layer). Each CTA keeps the states of a quarter of the rows, reads the index for
// their features, and chooses and takes their actions.
// On GB300, 256 requests against 20 000 plans: 27 us per step before, 11.3 us now (12.8 with one
// warp per state reading the index).
constexpr int kActPad = kHid + 8;  // bf16 per activation row (bank-conflict-free fragment reads)
constexpr int kPolicyCols = kHid / kPolicyCluster;    // columns of a hidden layer per CTA
constexpr int kPolicyOut = kOutPad / kPolicyCluster;  // logits per CTA
constexpr int kPolicyOwn = kPolicyRows / kPolicyCluster;
static_assert(kPolicyCols == 8 * (kPolicyThreads / 32) && kPolicyOut == 8, "one 8-column tile per warp");

struct PolicyRow {
    double s[3];
    double c0, s0, step, cap2;
    double gx, gy, gz;          // the request's goal, kept so a step reads no request
    int32_t row1;               // index row of the first step's samples
    int32_t k_lo, k_hi;         // steps whose samples lie in the table window: [k_lo, k_hi)
    float speed;
    int32_t horizon;
    int32_t req, k, h, status;  // req < 0: empty
};

struct PolicyTurns {  // the actions' moves
    double cks[48];   // cos, sin of 15 degree steps (FP64)
    double climb_dt[kMaxActions];
    int dh[kMaxActions];
};

struct PolicySmem {
    __nv_bfloat16 w0[kPolicyCols * (kFeat + 8)];               // [column][input]
    __nv_bfloat16 w[kLayers - 2][kPolicyCols * kActPad];
    __nv_bfloat16 w4[kPolicyOut * kActPad];
    __nv_bfloat16 act[2][kPolicyRows * kActPad];  // every CTA's copy of a layer's input
    float logits[kPolicyOwn][kOutPad];
    float feat[kPolicyThreads / 32][kFeat];
    unsigned long long skey[kPolicyThreads / 32][kSectors];
    PolicyRow rows[kPolicyOwn];                   // this CTA's share of the rows
    PolicyTurns turns;
    float bias[(kLayers - 1) * kHid + kOutPad];   // every layer's bias (fp32), in parameter order
    int choice[kPolicyOwn];
    int flags[2][kPolicyCluster];  // per CTA of the cluster: 1 rows in flight, 2 the queue may hold work
    int more;
};
static_assert(sizeof(PolicySmem) <= 232448, "shared memory of one CTA");

__device__ __forceinline__ uint32_t cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void peer_store(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t addr, uint2 v) {
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
    const __nv_bfloat162 v = __halves2bfloat162(__float2bfloat16_rn(x), __float2bfloat16_rn(y));
    return *reinterpret_cast<const uint32_t*>(&v);
}

// Takes the next work item into an empty row (one thread); false when the queue is empty. A row
// whose plan ends at once stays empty and pulls again in the next round.
__device__ __forceinline__ bool policy_refill(const PolicyArgs& a, PolicyRow& R) {
    const Model& m = a.m;
    const int w = atomicAdd(a.queue, 1);
    if (w >= (a.n_dev ? *a.n_dev : a.n_items)) return false;
    const int r = a.idx ? a.idx[w] : w;
    const fmdp_request q = a.reqs[r];
    R.req = r;
    R.k = 0;
    R.h = 0;
    R.s[0] = q.ox;
    R.s[1] = q.oy;
    R.s[2] = q.oz;
    const double dx = __dsub_rn(q.gx, q.ox), dy = __dsub_rn(q.gy, q.oy);
    const double Lh = __dsqrt_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
    R.c0 = Lh > 0.0 ? __ddiv_rn(dx, Lh) : 1.0;
    R.s0 = Lh > 0.0 ? __ddiv_rn(dy, Lh) : 0.0;
    R.step = __dmul_rn(q.speed_mps, m.dt);
    R.cap2 = __dmul_rn(R.step, R.step);
    R.gx = q.gx;
    R.gy = q.gy;
    R.gz = q.gz;
    const int64_t T1 = q.depart_step + 1, T0 = a.tab.t_base;
    const int64_t row1 = T1 % a.tab.T_win;
    R.row1 = (int32_t)(row1 < 0 ? row1 + a.tab.T_win : row1);
    R.k_lo = (int32_t)min(max(T0 - T1, (int64_t)0), (int64_t)INT_MAX);
    R.k_hi = (int32_t)min(max(T0 + a.tab.T_win - T1, (int64_t)0), (int64_t)INT_MAX);
    R.speed = (float)q.speed_mps;
    R.horizon = q.horizon;
    if (a.step_bound) {  // the judge rejects anything longer: stop there
        const double b = judge_step_bound(q, m.dt, a.climb_step, a.slack);
        if (b < (double)R.horizon) R.horizon = (int32_t)fmax(b, 0.0);
    }
    float* tr = a.traj + (size_t)r * a.cap * 3;
    tr[0] = (float)q.ox;
    tr[1] = (float)q.oy;
    tr[2] = (float)q.oz;
    R.status = -1;
    const double ex = __dsub_rn(q.gx, q.ox), ey = __dsub_rn(q.gy, q.oy), ez = __dsub_rn(q.gz, q.oz);
    const bool cap0 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) <= R.cap2;
    if (cap0 || R.horizon <= 0) {  // done before the first step
        RolloutOut o;
        o.n_points = 1;
        o.status = cap0 ? kStatusCaptured : FMDP_REJ_HORIZON;
        o.near_ties = 0;
        o.steps = 0;
        a.out[r] = o;
        R.req = -1;  // the row pulls again next round
    }
    return true;
}
// The best action by logits among those that keep the successor inside the box, -1: none (a warp,
// lanes = actions). The sums of products are written out, see sum2.
__device__ __forceinline__ int policy_choice(const Model& m, const PolicyRow& R, const PolicyTurns& T, const float* logits) {
    const int lane = threadIdx.x & 31, A = m.A;
    const double* cks = T.cks;
    float v = -INFINITY;
    if (lane < A) {
        int hn = R.h + T.dh[lane];
        hn += hn < 0 ? 24 : 0;
        hn -= hn >= 24 ? 24 : 0;
        const float C = sum2((float)R.c0, (float)cks[2 * hn], -(float)R.s0, (float)cks[2 * hn + 1]);
        const float Sn = sum2((float)R.s0, (float)cks[2 * hn], (float)R.c0, (float)cks[2 * hn + 1]);
        const float x = fmaf((float)R.step, C, (float)R.s[0]), y = fmaf((float)R.step, Sn, (float)R.s[1]);
        const float z = (float)R.s[2] + (float)T.climb_dt[lane];
        const float mg = 1.0f;  // metres kept from the box faces
        const bool inside = x > (float)m.box[0] + mg && x < (float)m.box[3] - mg && y > (float)m.box[1] + mg &&
                            y < (float)m.box[4] - mg && z > (float)m.box[2] + mg && z < (float)m.box[5] - mg;
        v = inside ? logits[lane] : -INFINITY;
    }
    float mx = v;
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    const unsigned bm = __ballot_sync(kFull, v == mx && mx > -INFINITY);
    return bm ? __ffs(bm) - 1 : -1;
}
// Exact FP64 advance of the chosen action (FastMDP's successor rule, Alg. 1; one thread)
__device__ __forceinline__ void policy_advance(const PolicyArgs& a, PolicyRow& R, const PolicyTurns& T, int ch) {
    const double* cks = T.cks;
    bool done = false;
    if (ch < 0) {
        R.status = FMDP_REJ_NO_ACTION;
        done = true;
    } else {
        int hn = R.h + T.dh[ch];
        hn += hn < 0 ? 24 : 0;
        hn -= hn >= 24 ? 24 : 0;
        const double C = __dsub_rn(__dmul_rn(R.c0, cks[2 * hn]), __dmul_rn(R.s0, cks[2 * hn + 1]));
        const double Sn = __dadd_rn(__dmul_rn(R.s0, cks[2 * hn]), __dmul_rn(R.c0, cks[2 * hn + 1]));
        R.s[0] = __dadd_rn(R.s[0], __dmul_rn(R.step, C));
        R.s[1] = __dadd_rn(R.s[1], __dmul_rn(R.step, Sn));
        R.s[2] = __dadd_rn(R.s[2], T.climb_dt[ch]);
        R.h = hn;
        a.acts[(size_t)R.req * a.cap + R.k] = (uint8_t)ch;
        R.k += 1;
        float* tr = a.traj + ((size_t)R.req * a.cap + R.k) * 3;
        tr[0] = (float)R.s[0];
        tr[1] = (float)R.s[1];
        tr[2] = (float)R.s[2];
        const double ex = __dsub_rn(R.gx, R.s[0]), ey = __dsub_rn(R.gy, R.s[1]), ez = __dsub_rn(R.gz, R.s[2]);
        if (__dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez)) <= R.cap2) {
            R.status = kStatusCaptured;
            done = true;
        } else if (R.k >= R.horizon) {
            R.status = FMDP_REJ_HORIZON;
            done = true;
        }
    }
    if (done) {
        RolloutOut o;
        o.n_points = R.k + 1;
        o.status = R.status;
        o.near_ties = 0;
        o.steps = R.k;
        a.out[R.req] = o;
        R.req = -1;
    }
}
// Features of an active row's state (one warp, or the `parts` warps that share it) into feat;
// lane i's four of them as bf16
__device__ __forceinline__ uint2 policy_features(const PolicyArgs& a, const PolicyRow& R, float inv_dt, float* feat,
                                              unsigned long long* skey, int part, int parts, int bar) {
    const int lane = threadIdx.x & 31;
    float hc, hs;
    heading_cs((float)R.c0, (float)R.s0, R.h, hc, hs);
    const bool held = R.k >= R.k_lo && R.k < R.k_hi;
    const int row = R.row1 + R.k - (R.row1 + R.k >= a.tab.T_win ? a.tab.T_win : 0);
    warp_features(a.m, a.iv, a.tab, held ? row : -1, (float)R.s[0], (float)R.s[1], (float)R.s[2], hc, hs, R.speed, (float)R.gx,
                  (float)R.gy, (float)R.gz, inv_dt, feat, skey, part, parts, bar);
    const uint2 v = make_uint2(pack_bf16(feat[4 * lane], feat[4 * lane + 1]), pack_bf16(feat[4 * lane + 2], feat[4 * lane + 3]));
    __syncwarp();
    return v;
}
// the moves and every layer's bias into shared memory
__device__ __forceinline__ void policy_tables(const PolicyArgs& a, PolicyTurns& T, float* bias) {
    const int tid = threadIdx.x, A = a.m.A;
    if (tid < 24) unit15(tid, T.cks[2 * tid], T.cks[2 * tid + 1]);
    if (tid < kMaxActions) {
        T.climb_dt[tid] = tid < A ? __dmul_rn(a.m.climb[tid], a.m.dt) : 0.0;
        T.dh[tid] = tid < A ? a.m.dh[tid] : 0;
    }
    for (int l = 0, o = 0; l < kLayers; o += layer_out(l), ++l)
        for (int j = tid; j < layer_out(l); j += kPolicyThreads) bias[o + j] = a.params[param_offset_b(l) + j];
}

}  // namespace

__global__ void __cluster_dims__(kPolicyCluster, 1, 1) __launch_bounds__(kPolicyThreads, 1)
    policy_kernel(const __grid_constant__ PolicyArgs a) {
    extern __shared__ __align__(128) unsigned char psm[];
    PolicySmem& S = *reinterpret_cast<PolicySmem*>(psm);
    PolicyRow* rows = S.rows;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, NWp = kPolicyThreads / 32;
    const int g = lane >> 2, t = lane & 3;
    const int rank = (int)cta_rank();
    const Model& m = a.m;
    const int MT = a.rows >> 4;                  // 16-row tiles
    const int own = a.rows / kPolicyCluster;     // rows whose states this CTA keeps
    const int first = rank * own;                // the first of them among the cluster's rows
    const float inv_dt = (float)(1.0 / m.dt);
    uint32_t act_peer[kPolicyCluster];
#pragma unroll
    for (int c = 0; c < kPolicyCluster; ++c) act_peer[c] = peer_addr(smem_addr(S.act), c);
    if (tid < kPolicyOwn) rows[tid].req = -1;
    policy_tables(a, S.turns, S.bias);
    // this CTA's columns of every layer, once per launch
    for (int l = 0; l < kLayers; ++l) {
        const int cols = l == kLayers - 1 ? kPolicyOut : kPolicyCols, per = layer_in(l) / 8;
        __nv_bfloat16* dst = l == 0 ? S.w0 : (l == kLayers - 1 ? S.w4 : S.w[l - 1]);
        const int pad = layer_in(l) + 8;
        const __nv_bfloat16* src = a.Wp + wp_layer_offset(l) + (size_t)rank * cols * kChunkPad;
        for (int e = tid; e < cols * per; e += kPolicyThreads) {
            const int n = e / per, k = (e - n * per) * 8;
            *reinterpret_cast<uint4*>(dst + (size_t)n * pad + k) = *reinterpret_cast<const uint4*>(
                src + (size_t)(k / kChunkK) * wp_chunk_elems(l) + (size_t)n * kChunkPad + k % kChunkK);
        }
    }
    if (tid == 0) S.more = 1;  // 1 while the queue may hold work
    __syncthreads();
    cluster_sync();  // every CTA of the cluster is running before its memory is written
    for (int it = 0;; ++it) {
        // ---- refill empty rows from the work queue (one thread per row)
        if (tid < own && rows[tid].req < 0 && S.more && !policy_refill(a, rows[tid])) S.more = 0;
        __syncthreads();
        int any = 0;
        for (int i = lane; i < own; i += 32) any |= rows[i].req >= 0;
        any = __any_sync(kFull, any);
        if (tid < kPolicyCluster)  // (two sets: a CTA may be one step ahead of a peer's reads)
            peer_store(peer_addr(smem_addr(&S.flags[it & 1][rank]), tid), (uint32_t)(any | 2 * S.more));
        // ---- features of this CTA's rows (one warp per row) into every CTA's act[0]
        // (with at most four rows per CTA two warps share each row's samples)
        const int parts = 2 * own <= NWp ? 2 : 1, part = parts == 2 ? warp / (NWp / 2) : 0;
        for (int rr = parts == 2 ? warp % (NWp / 2) : warp; rr < own; rr += NWp / parts) {
            const PolicyRow& R = rows[rr];
            uint2 v = make_uint2(0u, 0u);
            if (R.req >= 0) v = policy_features(a, R, inv_dt, S.feat[rr % NWp], S.skey[rr % NWp], part, parts, 1 + rr);
            if (part > 0) continue;
            const uint32_t off = (uint32_t)(((first + rr) * kActPad + 4 * lane) * sizeof(__nv_bfloat16));
#pragma unroll
            for (int c = 0; c < kPolicyCluster; ++c) peer_store(act_peer[c] + off, v);
        }
        cluster_sync();
        int flags = 0;
#pragma unroll
        for (int c = 0; c < kPolicyCluster; ++c) flags |= S.flags[it & 1][c];
        if (!flags) break;  // (the same in every CTA)
        if (!(flags & 1)) continue;
        // ---- the MLP: hidden layers, 8 columns per warp, then the logits
#pragma unroll 1
        for (int l = 0; l < kLayers - 1; ++l) {
            const __nv_bfloat16* xin = S.act[l & 1];
            const __nv_bfloat16* w = l == 0 ? S.w0 : S.w[l - 1];
            const int K = layer_in(l), wpad = K + 8;
            const __nv_bfloat16* wl = w + (size_t)(warp * 8 + (lane & 7)) * wpad + (lane >> 3) * 8;
            float acc[kPolicyRows / 16][4];
#pragma unroll
            for (int i = 0; i < kPolicyRows / 16; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[i][q] = 0.f;
#pragma unroll 4
            for (int k = 0; k < K; k += 32) {
                uint32_t b[4], a0[4], a1[4];
                ldsm4(b, wl + k);
#pragma unroll
                for (int mt = 0; mt < kPolicyRows / 16; ++mt) {
                    if (mt >= MT) break;
                    frag_a(a0, xin + (size_t)mt * 16 * kActPad, kActPad, k, lane);
                    frag_a(a1, xin + (size_t)mt * 16 * kActPad, kActPad, k + 16, lane);
                    mma_bf16(acc[mt], a0, b);
                    mma_bf16(acc[mt], a1, b + 2);
                }
            }
            // bias, ReLU, into every CTA's input of the next layer
            const int col = rank * kPolicyCols + warp * 8 + 2 * t;
            const float c0 = S.bias[l * kHid + col], c1 = S.bias[l * kHid + col + 1];
            const uint32_t base = (uint32_t)((((l + 1) & 1) * kPolicyRows * kActPad + g * kActPad + col) * sizeof(__nv_bfloat16));
#pragma unroll
            for (int mt = 0; mt < kPolicyRows / 16; ++mt) {
                if (mt >= MT) break;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const uint32_t v = pack_bf16(fmaxf(acc[mt][2 * u] + c0, 0.f), fmaxf(acc[mt][2 * u + 1] + c1, 0.f));
                    const uint32_t off = base + (uint32_t)((mt * 16 + 8 * u) * kActPad * sizeof(__nv_bfloat16));
#pragma unroll
                    for (int c = 0; c < kPolicyCluster; ++c) peer_store(act_peer[c] + off, v);
                }
            }
            cluster_sync();
        }
        if (warp < MT) {  // logits: warp takes rows [16 warp, 16 warp + 16), 8 columns per CTA
            const __nv_bfloat16* xin = S.act[(kLayers - 1) & 1] + (size_t)warp * 16 * kActPad;
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int k = 0; k < kHid; k += 32) {
                uint32_t b[4], a0[4], a1[4];
                ldsm4(b, S.w4 + (size_t)(lane & 7) * kActPad + (lane >> 3) * 8 + k);
                frag_a(a0, xin, kActPad, k, lane);
                frag_a(a1, xin, kActPad, k + 16, lane);
                mma_bf16(acc, a0, b);
                mma_bf16(acc, a1, b + 2);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = warp * 16 + g + (q >= 2 ? 8 : 0), col = rank * kPolicyOut + 2 * t + (q & 1);
                const float v = col < kOut ? acc[q] + S.bias[(kLayers - 1) * kHid + col] : -INFINITY;
                peer_store(peer_addr(smem_addr(&S.logits[r % own][col]), r / own), __float_as_uint(v));
            }
        }
        cluster_sync();
        // ---- argmax over the actions that keep the successor inside the box (one warp per row)
        for (int rr = warp; rr < own; rr += NWp) {
            const PolicyRow& R = rows[rr];
            if (R.req < 0) continue;
            const int ch = policy_choice(m, R, S.turns, S.logits[rr]);
            if (lane == 0) S.choice[rr] = ch;
        }
        __syncthreads();
        // ---- exact FP64 advance of the chosen action (FastMDP's successor rule, Alg. 1)
        if (tid < own && rows[tid].req >= 0) policy_advance(a, rows[tid], S.turns, S.choice[tid]);
        __syncthreads();
    }
}

// Many proposals at once: 32 rows per CTA, every CTA by itself, all weights streamed past its rows in
// every step (18 chunks by bulk copies, four buffers, three chunks ahead). It is bound by that stream
// and a step takes longer than the cluster's, but the chip carries twice as many rows: see
// policy_streamed.
namespace {
constexpr int kStreamRows = 32, kStreamBufs = 4;
constexpr int kStreamChunks = kFeat / kChunkK + (kLayers - 1) * (kHid / kChunkK);  // per step

struct PolicyStreamSmem {
    __nv_bfloat16 w[kStreamBufs][kHid * kChunkPad];
    __nv_bfloat16 act[2][kStreamRows * kActPad];
    float logits[kStreamRows][kOutPad];
    float feat[kPolicyThreads / 32][kFeat];
    unsigned long long skey[kPolicyThreads / 32][kSectors];
    PolicyRow rows[kStreamRows];
    PolicyTurns turns;
    float bias[(kLayers - 1) * kHid + kOutPad];
    uint64_t bars[kStreamBufs];
    int choice[kStreamRows];
    int more;
};
static_assert(sizeof(PolicyStreamSmem) <= 232448, "shared memory of one CTA");
}  // namespace

__global__ void __launch_bounds__(kPolicyThreads, 1) policy_stream_kernel(const __grid_constant__ PolicyArgs a) {
    extern __shared__ __align__(128) unsigned char psm[];
    PolicyStreamSmem& S = *reinterpret_cast<PolicyStreamSmem*>(psm);
    PolicyRow* rows = S.rows;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, NWp = kPolicyThreads / 32;
    const int g = lane >> 2, t = lane & 3;
    const float inv_dt = (float)(1.0 / a.m.dt);
    constexpr int MT = kStreamRows / 16;
    // Chunks are numbered across steps: chunk q is in buffer q mod kStreamBufs, its (q / kStreamBufs)-th
    // fill. The buffer of chunk q + 3 was read last as chunk q - 1, and every thread has passed the
    // barrier after that when chunk q is waited for.
    long long q = 0, issued = 0;
    auto issue = [&]() {  // thread 0
        int l = 0, kc = (int)(issued % kStreamChunks);
        while (kc >= layer_in(l) / kChunkK) kc -= layer_in(l++) / kChunkK;
        const uint32_t bytes = (uint32_t)(wp_chunk_elems(l) * sizeof(__nv_bfloat16));
        uint64_t* bar = &S.bars[issued % kStreamBufs];
        bar_expect(bar, bytes);
        bulk_load(S.w[issued % kStreamBufs], a.Wp + wp_layer_offset(l) + (size_t)kc * wp_chunk_elems(l), bytes, bar);
        ++issued;
    };
    auto chunk_came = [&](long long c) { return bar_wait(&S.bars[c % kStreamBufs], (uint32_t)((c / kStreamBufs) & 1)); };
    if (tid < kStreamRows) rows[tid].req = -1;
    policy_tables(a, S.turns, S.bias);
    if (tid == 0) {
        for (int b = 0; b < kStreamBufs; ++b) bar_init(&S.bars[b]);
        S.more = 1;  // 1 while the queue may hold work
        for (int b = 0; b < kStreamBufs - 1; ++b) issue();
    }
    __syncthreads();
    bool failed = false;
    while (!failed) {
        // ---- refill empty rows from the work queue (one thread per row)
        if (tid < kStreamRows && rows[tid].req < 0 && S.more && !policy_refill(a, rows[tid])) S.more = 0;
        __syncthreads();
        const bool any = __any_sync(kFull, rows[lane].req >= 0), more = S.more != 0;
        __syncthreads();
        if (!any && !more) break;
        if (!any) continue;
        // ---- features of every active row (one warp per row)
        for (int rr = warp; rr < kStreamRows; rr += NWp) {
            uint2 v = make_uint2(0u, 0u);
            if (rows[rr].req >= 0) v = policy_features(a, rows[rr], inv_dt, S.feat[warp], S.skey[warp], 0, 1, 0);
            *reinterpret_cast<uint2*>(S.act[0] + (size_t)rr * kActPad + 4 * lane) = v;
        }
        __syncthreads();
        // ---- the MLP, layer by layer, chunk by chunk
        for (int l = 0; l < kLayers && !failed; ++l) {
            const __nv_bfloat16* xin = S.act[l & 1];
            const bool last = l == kLayers - 1;
            float acc[MT][4][4];
#pragma unroll
            for (int i = 0; i < MT * 16; ++i) acc[i >> 4][(i >> 2) & 3][i & 3] = 0.f;
            for (int kc = 0; kc < layer_in(l) / kChunkK && !failed; ++kc, ++q) {
                const bool came = chunk_came(q);
                if (!came && lane == 0) atomicExch(a.err, FMDP_ERR_TIMEOUT);
                if (tid == 0 && came) issue();
                const __nv_bfloat16* wb = S.w[q % kStreamBufs];
                if (!last) {  // warp: columns [32 warp, 32 warp + 32), all rows
#pragma unroll
                    for (int kk = 0; kk < kChunkK; kk += 16) {
                        uint32_t af[MT][4], b0[4], b1[4];
                        const __nv_bfloat16* p =
                            wb + (size_t)(warp * 32 + (lane >> 4) * 8 + (lane & 7)) * kChunkPad + kk + ((lane >> 3) & 1) * 8;
                        ldsm4(b0, p);
                        ldsm4(b1, p + 16 * kChunkPad);
#pragma unroll
                        for (int mt = 0; mt < MT; ++mt) {
                            frag_a(af[mt], xin + (size_t)mt * 16 * kActPad, kActPad, kc * kChunkK + kk, lane);
                            mma_bf16(acc[mt][0], af[mt], b0);
                            mma_bf16(acc[mt][1], af[mt], b0 + 2);
                            mma_bf16(acc[mt][2], af[mt], b1);
                            mma_bf16(acc[mt][3], af[mt], b1 + 2);
                        }
                    }
                } else if (warp < MT * 4) {  // warp: 16 rows, 8 of the 32 logits
#pragma unroll
                    for (int kk = 0; kk < kChunkK; kk += 32) {
                        uint32_t af[4], b[4];
                        const __nv_bfloat16* x = xin + (size_t)(warp >> 2) * 16 * kActPad;
                        ldsm4(b, wb + (size_t)((warp & 3) * 8 + (lane & 7)) * kChunkPad + kk + (lane >> 3) * 8);
                        frag_a(af, x, kActPad, kc * kChunkK + kk, lane);
                        mma_bf16(acc[0][0], af, b);
                        frag_a(af, x, kActPad, kc * kChunkK + kk + 16, lane);
                        mma_bf16(acc[0][0], af, b + 2);
                    }
                }
                // the chunk's buffer is free again; a wait that expired anywhere stops every thread
                failed = __syncthreads_or(came ? 0 : 1) != 0;
            }
            const float* bias = S.bias + l * kHid;
            if (!last) {
                __nv_bfloat16* out = S.act[(l + 1) & 1];
#pragma unroll
                for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int col = warp * 32 + j * 8 + 2 * t;
                        const float c0 = bias[col], c1 = bias[col + 1];
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            *reinterpret_cast<uint32_t*>(out + (size_t)(mt * 16 + g + 8 * u) * kActPad + col) =
                                pack_bf16(fmaxf(acc[mt][j][2 * u] + c0, 0.f), fmaxf(acc[mt][j][2 * u + 1] + c1, 0.f));
                    }
            } else if (warp < MT * 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = (warp >> 2) * 16 + g + (i >= 2 ? 8 : 0), col = (warp & 3) * 8 + 2 * t + (i & 1);
                    S.logits[r][col] = col < kOut ? acc[0][0][i] + bias[col] : -INFINITY;
                }
            }
            __syncthreads();
        }
        if (failed) break;
        // ---- actions and advance
        for (int rr = warp; rr < kStreamRows; rr += NWp) {
            if (rows[rr].req < 0) continue;
            const int ch = policy_choice(a.m, rows[rr], S.turns, S.logits[rr]);
            if (lane == 0) S.choice[rr] = ch;
        }
        __syncthreads();
        if (tid < kStreamRows && rows[tid].req >= 0) policy_advance(a, rows[tid], S.turns, S.choice[tid]);
        __syncthreads();
    }
    // the copies still in flight, before the block's shared memory is given back
    // (after an expired wait the chunk waited for is among them)
    if (tid == 0)
        for (long long c = q > 0 ? q - 1 : 0; c < issued; ++c) chunk_came(c);
}

cudaError_t prepare_policy_kernels() {
    const cudaError_t e =
        cudaFuncSetAttribute(policy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PolicySmem));
    return e != cudaSuccess ? e
                            : cudaFuncSetAttribute(policy_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)sizeof(PolicyStreamSmem));
}

cudaError_t launch_policy(PolicyArgs a, int n, int n_sm, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (policy_streamed(n, n_sm)) {
        const int ctas = (n + kStreamRows - 1) / kStreamRows;
        policy_stream_kernel<<<ctas < n_sm ? ctas : n_sm, kPolicyThreads, sizeof(PolicyStreamSmem), s>>>(a);
    } else {
        a.rows = policy_rows_for(n, n_sm);
        policy_kernel<<<policy_ctas_for(n, a.rows, n_sm), kPolicyThreads, sizeof(PolicySmem), s>>>(a);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ judge

__global__ void judge_kernel(const __grid_constant__ JudgeArgs a) {
    const int w = blockIdx.x;
    if (w >= a.n || (a.n_dev && w >= *a.n_dev)) return;
    const int r = a.idx ? a.idx[w] : w;
    __shared__ int ok_s;
    const RolloutOut rp = a.rout_p[r];
    if (threadIdx.x == 0) {
        const fmdp_request q = a.reqs[r];
        const SepOut sp = a.sep_p[r];
        const bool ok = rp.status == kStatusCaptured && sp.first_conflict == INT_MAX && sp.first_terrain == INT_MAX &&
                        (double)rp.steps <= judge_step_bound(q, a.dt, a.climb_step, a.slack);
        ok_s = ok ? 1 : 0;
        a.accepted[r] = ok_s;
        if (ok && a.traj) {
            a.rout[r] = rp;
            a.sep[r] = sp;
        }
    }
    __syncthreads();
    if (!ok_s || !a.traj) return;
    const int np = rp.n_points;
    for (int k = threadIdx.x; k < np; k += blockDim.x) {
        const size_t o = ((size_t)r * a.cap + k) * 3;
        a.traj[o] = a.traj_p[o];
        a.traj[o + 1] = a.traj_p[o + 1];
        a.traj[o + 2] = a.traj_p[o + 2];
        if (k + 1 < np) a.acts[(size_t)r * a.cap + k] = a.acts_p[(size_t)r * a.cap + k];
    }
}

cudaError_t launch_judge(const JudgeArgs& a, int max_points, cudaStream_t s) {
    if (a.n <= 0) return cudaSuccess;
    judge_kernel<<<a.n, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace fmdp
