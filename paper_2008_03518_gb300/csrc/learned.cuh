// Learned proposal (no counterpart in the paper): a small MLP trained on FastMDP's action
// choices (Alg. 1, Sec. III) proposes a whole trajectory, which the separation check and a
// path-cost bound then judge; plain FastMDP is the fallback.
#pragma once

#include <cuda_bf16.h>

#include "fmdp_internal.cuh"

namespace fmdp {

constexpr int kFeat = 128;        // network inputs
constexpr int kHid = 256;         // hidden width (four hidden layers)
constexpr int kOut = 25;          // action logits
constexpr int kOutPad = 32;       // logits padded to four 8-wide tiles
constexpr int kLayers = 5;
constexpr int kSectors = 20;      // 10 azimuth sectors x (above, below)
constexpr int kOwn = 8;
constexpr float kRF = 1000.0f;    // metres: sectors see plan samples this close
constexpr int kChunkK = 64;       // weight rows per staged chunk (policy kernel)
constexpr int kChunkPad = 72;     // bf16 per staged row: 64 + 8 (bank-conflict-free reads)

__host__ __device__ constexpr int layer_in(int l) { return l == 0 ? kFeat : kHid; }
__host__ __device__ constexpr int layer_out(int l) { return l == kLayers - 1 ? kOut : kHid; }
__host__ __device__ constexpr int layer_out_pad(int l) { return l == kLayers - 1 ? kOutPad : kHid; }
// fp32 master parameters: per layer W (in x out, row-major) then b (out)
__host__ __device__ inline size_t param_offset_W(int l) {
    size_t o = 0;
    for (int i = 0; i < l; ++i) o += (size_t)layer_in(i) * layer_out(i) + layer_out(i);
    return o;
}
__host__ __device__ inline size_t param_offset_b(int l) { return param_offset_W(l) + (size_t)layer_in(l) * layer_out(l); }
__host__ __device__ inline size_t n_params_total() { return param_offset_W(kLayers); }
// policy weights: per layer, chunks of kChunkK input rows, each [out_pad][kChunkPad] bf16
// (out-major, the chunk's inputs contiguous: the column layout of the mma B operand)
__host__ __device__ inline size_t wp_chunk_elems(int l) { return (size_t)layer_out_pad(l) * kChunkPad; }
__host__ __device__ inline size_t wp_layer_offset(int l) {
    size_t o = 0;
    for (int i = 0; i < l; ++i) o += (size_t)(layer_in(i) / kChunkK) * wp_chunk_elems(i);
    return o;
}
__host__ __device__ inline size_t wp_total() { return wp_layer_offset(kLayers); }

// ---- tensor-core and bulk-copy steps shared by the network kernels
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void bar_init(uint64_t* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait (about a second of SM cycles); false on timeout
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
    const long long t0 = clock64();
    while (!bar_try(bar, parity))
        if (clock64() - t0 > (1ll << 31)) return false;
    return true;
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void ldsm4(uint32_t* r, const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p))
                 : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t* r, const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p))
                 : "memory");
}
// A fragment (16 rows x 16 k) of a row-major tile
__device__ __forceinline__ void frag_a(uint32_t* r, const __nv_bfloat16* tile, int pad, int k, int lane) {
    ldsm4(r, tile + (size_t)(lane & 15) * pad + k + (lane >> 4) * 8);
}

__device__ __forceinline__ uint32_t sample_hash(float x, float y, float z) {
    return __float_as_uint(x) ^ (__float_as_uint(y) * 2654435761u) ^ (__float_as_uint(z) * 40503u);
}
__device__ __forceinline__ float clampf(float v, float lo, float hi) { return fminf(fmaxf(v, lo), hi); }
// a b + c d with the first product fused, and sums of three squares: written out, because the
// features are inlined into several kernels and have to be the same bits in each (which product of
// a sum is fused would be the compiler's choice in each copy)
__device__ __forceinline__ float sum2(float a, float b, float c, float d) { return fmaf(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ float squares3(float x, float y, float z) { return fmaf(z, z, sum2(x, x, y, y)); }
// (one copy for every kernel, for the same reason)
static __device__ __noinline__ float feature_ground(const Model& m, float x, float y) { return terrain32(m, x, y); }
// Features of one state, computed by one warp into out[kFeat] (shared memory). s: position;
// (hc, hs): heading cos / sin; skey: kSectors words of scratch in shared memory. The order of
// reading and of the index's items does not change the result: each sector keeps its minimum of
// (squared distance, a hash of the sample's coordinates).
// row: the index row of the plan samples to read (the next step's), below 0 outside the table
// window. parts > 1: that many warps share one state's samples (part: this one; they meet at named
// barrier `bar`). With 16 proposals to a cluster of four CTAs every step waits for its densest
// state: two warps per state and the own state's features read while the cell bounds arrive took a
// step against 20 000 plans from 12.8 to 11.3 us.
__device__ inline void warp_features(const Model& m, const IndexView& iv, const TableView& tab, int row, float sx,
                                     float sy, float sz, float hc, float hs, float speed, float gx, float gy, float gz,
                                     float inv_dt, float* out, unsigned long long* skey, int part = 0, int parts = 1,
                                     int bar = 0) {
    const int lane = threadIdx.x & 31;
    auto meet = [&]() {
        if (parts == 1) __syncwarp();
        else asm volatile("barrier.cta.sync %0, %1;" ::"r"(bar), "r"(32 * parts) : "memory");
    };
    for (int i = lane + 32 * part; i < kFeat; i += 32 * parts) out[i] = 0.f;
    if (lane < kSectors && part == 0) skey[lane] = ~0ull;
    meet();
    const int32_t* cs_row = iv.cstart + max(row, 0) * (int64_t)(iv.ncell + 1);
    const float4* it = iv.items + (size_t)max(row, 0) * tab.S_pad * 2;
    auto cell_of = [&](float v, float o, int n) {
        const float f = floorf((v - o) * iv.inv_cell);
        return f < 0.f ? 0 : (f > (float)(n - 1) ? n - 1 : (int)f);
    };
    const int cx0 = cell_of(sx - kRF, iv.x0, iv.ncx), cx1 = cell_of(sx + kRF, iv.x0, iv.ncx);
    const int cy0 = cell_of(sy - kRF, iv.y0, iv.ncy), cy1 = cell_of(sy + kRF, iv.y0, iv.ncy);
    // The query's ranges: its cell rows (cells cx0..cx1 of a row are contiguous), then the
    // extra list. They are taken 16 at a time; lanes 2q and 2q + 1 load range q's bounds
    // together, and the lanes then share out the group's items as one flat list.
    const int nrows = cy1 - cy0 + 1;
    auto bounds = [&](int q0) {
        const int q = q0 + (lane >> 1);
        if (q < nrows) return cs_row[(cy0 + q) * iv.ncx + ((lane & 1) ? cx1 + 1 : cx0)];
        if (q == nrows) return (lane & 1) ? cs_row[iv.ncell] + iv.nextra[row] : cs_row[iv.ncell];
        return 0;
    };
    const int bounds0 = row >= 0 ? bounds(0) : 0;
    if (lane == 0 && part == parts - 1) {  // own state, while the bounds arrive
        const float z0 = (float)m.box[2], z1 = (float)m.box[5];
        out[0] = (sz - z0) / (z1 - z0);
        const float clr = m.hm ? sz - feature_ground(m, sx, sy) : sz - z0;
        out[1] = clampf(clr / 200.f, -1.f, 4.f);
        const float Gx = gx - sx, Gy = gy - sy, Gz = gz - sz;
        const float gf = sum2(Gx, hc, Gy, hs), gl = sum2(Gy, hc, -Gx, hs);
        const float gh = sqrtf(sum2(gf, gf, gl, gl));
        out[2] = clampf(gf / 5000.f, -4.f, 4.f);
        out[3] = clampf(gl / 5000.f, -4.f, 4.f);
        out[4] = clampf(Gz / 200.f, -4.f, 4.f);
        out[5] = fminf(gh / 20000.f, 4.f);
        out[6] = gh > 0.f ? gf / gh : 1.f;
        out[7] = gh > 0.f ? gl / gh : 0.f;
    }
    if (row < 0) {
        meet();
        return;
    }
    const float R2 = kRF * kRF;
    const unsigned full = 0xffffffffu;
    auto sector_of = [&](float rf, float rl, float rz) {
        const float az = atan2f(rl, rf);  // [-pi, pi]
        int k = (int)floorf((az + 3.14159265358979f) * (10.f / 6.28318530717959f));
        k = min(max(k, 0), 9);
        return k + (rz >= 0.f ? 10 : 0);
    };
    auto visit = [&](auto&& fn) {
        for (int q0 = 0; q0 <= nrows; q0 += 16) {
            const int v = q0 ? bounds(q0) : bounds0;
            int beg[16], start[17];
            start[0] = 0;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int b = __shfl_sync(full, v, 2 * k), e = __shfl_sync(full, v, 2 * k + 1);
                beg[k] = b;
                start[k + 1] = start[k] + (q0 + k <= nrows ? max(0, e - b) : 0);
            }
            const int total = start[16];
            for (int j = lane + 32 * part; j < total; j += 32 * parts) {
                // the range holding flat item j: the last k whose start is at or before j
                int i = beg[0] + j;
#pragma unroll
                for (int k = 1; k < 16; ++k)
                    if (j >= start[k]) i = beg[k] + (j - start[k]);
                fn(i);
            }
        }
    };
    // sector feature of the nearest sample P1 (and the same plan's next sample P2)
    auto emit = [&](float4 P1, float4 P2, float d2, int sec) {
        const float rx = P1.x - sx, ry = P1.y - sy, rz = P1.z - sz;
        const float rf = sum2(ry, hs, rx, hc), rl = sum2(ry, hc, -rx, hs);
        float vx = 0.f, vy = 0.f, vz = 0.f;
        if (P2.x == P2.x) {
            vx = (P2.x - P1.x) * inv_dt;
            vy = (P2.y - P1.y) * inv_dt;
            vz = (P2.z - P1.z) * inv_dt;
        }
        const float vf = sum2(vx, hc, vy, hs), vl = sum2(vy, hc, -vx, hs);
        const float w = 1.f - sqrtf(d2) / kRF;
        float* o = out + kOwn + 6 * sec;
        o[0] = rf * (1.f / 500.f) * w;
        o[1] = rl * (1.f / 500.f) * w;
        o[2] = rz * (1.f / 500.f) * w;
        o[3] = (vf - speed) * (1.f / 50.f) * w;
        o[4] = vl * (1.f / 50.f) * w;
        o[5] = vz * (1.f / 50.f) * w;
    };
    // key of sample P1: (squared distance, position hash), all-ones beyond R_F
    auto key_of = [&](float4 P1, float& d2, int& sec) {
        const float rx = P1.x - sx, ry = P1.y - sy, rz = P1.z - sz;
        d2 = squares3(rx, ry, rz);
        if (!(d2 < R2)) return ~0ull;
        sec = sector_of(sum2(rx, hc, ry, hs), sum2(ry, hc, -rx, hs), rz);
        return ((unsigned long long)__float_as_uint(d2) << 32) | sample_hash(P1.x, P1.y, P1.z);
    };
    // pass 1: every sector's least key; a lane keeps its first two in-range samples
    int ci0 = -1, ci1 = -1, cs0 = 0, cs1 = 0;
    float cd0 = 0.f, cd1 = 0.f;
    unsigned long long ck0 = 0, ck1 = 0;
    float4 cp0 = make_float4(0.f, 0.f, 0.f, 0.f), cp1 = cp0;
    bool over = false;
    visit([&](int i) {
        const float4 P1 = it[2 * (size_t)i];
        float d2;
        int sec;
        const unsigned long long key = key_of(P1, d2, sec);
        if (key == ~0ull) return;
        atomicMin(&skey[sec], key);
        if (ci0 < 0) {
            ci0 = i, cs0 = sec, cd0 = d2, ck0 = key, cp0 = P1;
        } else if (ci1 < 0) {
            ci1 = i, cs1 = sec, cd1 = d2, ck1 = key, cp1 = P1;
        } else {
            over = true;
        }
    });
    meet();
    // pass 2: the sector winners write their features
    if (!__any_sync(full, over)) {
        if (ci0 >= 0 && ck0 == skey[cs0]) emit(cp0, it[2 * (size_t)ci0 + 1], cd0, cs0);
        if (ci1 >= 0 && ck1 == skey[cs1]) emit(cp1, it[2 * (size_t)ci1 + 1], cd1, cs1);
    } else {
        visit([&](int i) {
            const float4 P1 = it[2 * (size_t)i];
            float d2;
            int sec;
            const unsigned long long key = key_of(P1, d2, sec);
            if (key != ~0ull && key == skey[sec]) emit(P1, it[2 * (size_t)i + 1], d2, sec);
        });
    }
    meet();
}

// fp32 cos / sin of the heading with index h (15 degree steps) turned from the bearing
// (c0, s0): the features' heading frame
__device__ __forceinline__ void heading_cs(float c0, float s0, int h, float& hc, float& hs) {
    const float a = (float)h * (3.14159265358979f / 12.f);
    float sk, ck;
    sincosf(a, &sk, &ck);
    hc = sum2(c0, ck, -s0, sk);
    hs = sum2(s0, ck, c0, sk);
}

// ---- device entry points (learned.cu)
struct CollectArgs {
    Model m;
    TableView tab;
    IndexView iv;
    const float* traj;          // [n][cap][3]
    const uint8_t* acts;        // [n][cap]
    int32_t cap;
    const RolloutOut* rout;
    const fmdp_request* reqs;
    const int64_t* row0;        // [n]: first training row of request r
    __nv_bfloat16* X;           // [rows][kFeat]
    uint8_t* y;                 // [rows]
    int32_t n;
};
cudaError_t launch_collect(const CollectArgs& a, cudaStream_t s);

// Loss and gradient of one batch (train.cu). Weight gradients are summed over kTrainSplit
// stretches of the batch at most, each into its own copy of the parameters.
constexpr int kTrainRows = 16;                 // rows per block of the forward / backward kernel
constexpr int kTrainSplit = 8;
constexpr int kTrainSums = 4 * kHid + kOutPad + 4;  // per block: output-gradient column sums, loss
struct TrainArgs {
    const float* Xf;           // fp32 features [M][kFeat], rounded to X by the kernel (or nullptr)
    __nv_bfloat16* X;          // bf16 features [M][kFeat]
    const uint8_t* y;          // labels
    int32_t M, n_valid;        // rows; actions
    const __nv_bfloat16* Wp;   // chunked bf16 weights
    const float* params;       // fp32 master parameters (biases)
    __nv_bfloat16* H;          // [4][M][kHid]: hidden activations
    __nv_bfloat16* dZ;         // [4][M][kHid] then [M][kOutPad]: gradients of the layers' outputs
    float* sums;               // [blocks][kTrainSums]
    float* part;               // [kTrainSplit][n_params_total()]
    float* grad;               // [n_params_total()]
    float* loss;               // the batch's mean loss is added
    int32_t* err;
};
inline int train_blocks(int M) { return (M + kTrainRows - 1) / kTrainRows; }
cudaError_t prepare_train_kernels();
cudaError_t launch_train(const TrainArgs& a, cudaStream_t s);
cudaError_t launch_gather_rows(const __nv_bfloat16* X, const int32_t* idx, int M, __nv_bfloat16* out,
                               const uint8_t* y, uint8_t* y_out, cudaStream_t s);
// Adam on the fp32 master parameters (nothing once *err is set), then the bf16 copy in the chunk
// layout
cudaError_t launch_adam(float* p, const float* g, float* m1, float* m2, size_t n, float lr, float b1, float b2,
                        float eps, int t, const int32_t* err, cudaStream_t s);
cudaError_t launch_export_weights(const float* p, __nv_bfloat16* Wp, cudaStream_t s);

// Policy rollouts: a cluster of CTAs carries up to kPolicyRows requests in lock step (one
// matrix row each), every CTA the features and states of its share of them, and refills a
// finished row from the work queue.
constexpr int kPolicyCluster = 4;
constexpr int kPolicyRows = 64;
constexpr int kPolicyThreads = 256;
struct PolicyArgs {
    Model m;
    TableView tab;
    IndexView iv;
    const __nv_bfloat16* Wp;  // chunked bf16 weights
    const float* params;      // fp32 master parameters (biases)
    const fmdp_request* reqs;
    const int32_t* idx;       // work items -> requests (nullptr: identity)
    int32_t n_items;
    const int32_t* n_dev;     // number of work items on the device (nullptr: n_items)
    int32_t* queue;           // work counter
    int32_t cap;
    float* traj;              // [n][cap][3]
    uint8_t* acts;            // [n][cap]
    RolloutOut* out;          // [n]
    int32_t* err;             // device error word
    int32_t rows;             // requests per cluster: a multiple of 16 up to kPolicyRows (set by the launch)
    // 1: stop a proposal at the judge's step bound (a longer one would be rejected anyway)
    int32_t step_bound;
    double slack, climb_step;
};
// rows per cluster for n work items on n_sm multiprocessors: as few 16-row tiles as give every
// item a row at once. A step against 200 plans takes 10 us with one tile, 13 with two, 20 with
// four: 600 requests take 12.1 ms by one tile, 620 take 15.2 by two (one tile, two rounds: 24).
inline int policy_rows_for(int n, int n_sm) {
    const int clusters = n_sm / kPolicyCluster > 0 ? n_sm / kPolicyCluster : 1;
    const int tiles = (n + 16 * clusters - 1) / (16 * clusters);
    return 16 * (tiles < 1 ? 1 : (tiles > kPolicyRows / 16 ? kPolicyRows / 16 : tiles));
}
inline int policy_ctas_for(int n, int rows, int n_sm) {
    const int clusters = n_sm / kPolicyCluster > 0 ? n_sm / kPolicyCluster : 1, want = (n + rows - 1) / rows;
    return kPolicyCluster * (want < clusters ? want : clusters);
}
// n work items by policy_stream_kernel instead, whose CTAs share nothing and carry 32 rows each (4864
// at once, the clusters 2432): past the clusters' first round of rows by a fifth. Among 3000 plans
// 2432 proposals take 35.0 ms by clusters, 3000 take 39.4, 5000 51 and 10 000 75; streamed 38.0 up to
// 4864 and 55 for 10 000. (20 000 plans: 42, 46, 60 and 96; 46.3 and 69.)
inline bool policy_streamed(int n, int n_sm) {
    const int clusters = n_sm / kPolicyCluster > 0 ? n_sm / kPolicyCluster : 1;
    return n > 6 * kPolicyRows * clusters / 5;
}
cudaError_t prepare_policy_kernels();
cudaError_t launch_policy(PolicyArgs a, int n, int n_sm, cudaStream_t s);  // n: the most work items there may be

// Judge: a proposal is accepted when it reaches the goal, passes the separation and
// terrain checks, and takes at most (1 + slack) times the fewest steps any trajectory
// needs to reach the goal (which bounds its cost gap to FastMDP's by the same factor).
// Accepted proposals are copied over the request's FastMDP buffers and flagged.
struct JudgeArgs {
    const fmdp_request* reqs;
    const int32_t* idx;
    const int32_t* n_dev;
    int32_t n;
    const float* traj_p;
    const uint8_t* acts_p;
    const RolloutOut* rout_p;
    const SepOut* sep_p;
    float* traj;              // nullptr: decide only, copy nothing
    uint8_t* acts;
    RolloutOut* rout;
    SepOut* sep;
    int32_t* accepted;        // [n]
    int32_t cap;
    double dt, slack;
    double climb_step;        // largest |climb| x dt of the action set
};
cudaError_t launch_judge(const JudgeArgs& a, int max_points, cudaStream_t s);

}  // namespace fmdp
