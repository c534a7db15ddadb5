// Loss and gradient of the proposal network on one batch (sm_103a), in three launches.
//
// What bounds it: 1.4 GFLOP at 2048 rows are a microsecond of tensor work; a chain of matrix
// products as launches of its own was bound by latency, since each product had few blocks, a
// serial sum of K in each and a pass through memory between any two (1.5 ms). Rows are
// independent of one another up to the weight gradients, so:
//   train_chain_kernel  one block per 16 rows runs all layers forward and backward on its
//                       rows with the activations in shared memory; the weights stream
//                       through four buffers by bulk copies, three chunks ahead. It is bound
//                       by that stream (34 chunks of 36 KB per block from L2);
//   train_dw_kernel     the weight gradients of all layers, H^T dZ, as 64 x 64 tiles; the batch
//                       is split over up to eight blocks per tile, because 60 tiles would
//                       leave most of the chip idle;
//   train_sum_kernel    adds the stretches, the blocks' column sums (bias gradients) and losses,
//                       in a fixed order.
// Every value that is rounded to bf16 (activations, output gradients) is summed over K
// ascending in steps of 16, as the m16n8k16 product takes them.
// On GB300, loss and gradient of 2048 rows from and to host memory: 1672 us before, 158 us now.
#include "learned.cuh"

namespace fmdp {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kTrainThreads = 256;
constexpr int kXPad = kFeat + 8, kHPad = kHid + 8;  // bf16 per row: conflict-free fragment reads
constexpr int kTrainBufs = 4;
constexpr int kChunkElems = kHid * kChunkPad;
constexpr int kFwdChunks = kFeat / kChunkK + (kLayers - 1) * (kHid / kChunkK);
constexpr int kBwdChunks = (kLayers - 1) * (kHid / kChunkK);

struct TrainSmem {
    __nv_bfloat16 w[kTrainBufs][kChunkElems];
    __nv_bfloat16 x[kTrainRows * kXPad];
    __nv_bfloat16 h[kLayers - 1][kTrainRows * kHPad];
    __nv_bfloat16 dz[2][kTrainRows * kHPad];
    float logits[kTrainRows][kOutPad + 1];  // then the gradients of the logits
    float loss[kTrainRows];
    uint64_t bars[kTrainBufs];
};
static_assert(sizeof(TrainSmem) <= 232448, "shared memory of one block");

// The q-th chunk of a block's weight stream: its layer and its 64 inputs. Forward: layer by
// layer; backward: the same chunks of layers 4 to 1 (each gives the gradients of 64 inputs).
__device__ __forceinline__ void train_chunk(int q, int& l, int& kc) {
    if (q < kFwdChunks) {
        l = q < 2 ? 0 : 1 + (q - 2) / 4;
        kc = q < 2 ? q : (q - 2) & 3;
    } else {
        l = kLayers - 1 - (q - kFwdChunks) / 4;
        kc = (q - kFwdChunks) & 3;
    }
}

// bf16 rows of a shared tile to global memory, 16 bytes per thread and turn
__device__ __forceinline__ void store_rows(__nv_bfloat16* dst, const __nv_bfloat16* src, int pad, int cols, int rows) {
    const int per = cols / 8;
    for (int e = threadIdx.x; e < rows * per; e += kTrainThreads) {
        const int r = e / per, c = (e - r * per) * 8;
        *reinterpret_cast<uint4*>(dst + (size_t)r * cols + c) = *reinterpret_cast<const uint4*>(src + (size_t)r * pad + c);
    }
}

}  // namespace

__global__ void __launch_bounds__(kTrainThreads, 1) train_chain_kernel(const __grid_constant__ TrainArgs a) {
    extern __shared__ __align__(128) unsigned char train_smem[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(train_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int row0 = blockIdx.x * kTrainRows, rows = min(kTrainRows, a.M - row0);
    float* sums = a.sums + (size_t)blockIdx.x * kTrainSums;
    const uint8_t* wp = reinterpret_cast<const uint8_t*>(a.Wp);
    auto issue = [&](int q) {  // thread 0
        int l, kc;
        train_chunk(q, l, kc);
        const uint32_t bytes = (uint32_t)(wp_chunk_elems(l) * sizeof(__nv_bfloat16));
        uint64_t* bar = &S.bars[q % kTrainBufs];
        bar_expect(bar, bytes);
        bulk_load(S.w[q % kTrainBufs], wp + (wp_layer_offset(l) + (size_t)kc * wp_chunk_elems(l)) * sizeof(__nv_bfloat16),
                  bytes, bar);
    };
    if (tid == 0) {
        for (int b = 0; b < kTrainBufs; ++b) bar_init(&S.bars[b]);
        for (int q = 0; q < kTrainBufs - 1; ++q) issue(q);
    }
    // the block's features (rows past the batch: zeros)
    for (int e = tid; e < kTrainRows * (kFeat / 4); e += kTrainThreads) {
        const int r = e / (kFeat / 4), c = (e % (kFeat / 4)) * 4;
        uint2 v = make_uint2(0u, 0u);
        if (r < rows) {
            __nv_bfloat16* X = a.X + (size_t)(row0 + r) * kFeat + c;
            if (a.Xf) {
                const float4 f = *reinterpret_cast<const float4*>(a.Xf + (size_t)(row0 + r) * kFeat + c);
                const __nv_bfloat162 lo = __halves2bfloat162(__float2bfloat16_rn(f.x), __float2bfloat16_rn(f.y));
                const __nv_bfloat162 hi = __halves2bfloat162(__float2bfloat16_rn(f.z), __float2bfloat16_rn(f.w));
                v = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                *reinterpret_cast<uint2*>(X) = v;
            } else {
                v = *reinterpret_cast<const uint2*>(X);
            }
        }
        *reinterpret_cast<uint2*>(S.x + (size_t)r * kXPad + c) = v;
    }
    __syncthreads();
    bool failed = false;
    int q = 0;  // chunk of the stream
    // waits for chunk q and starts the one three further on: its buffer's last reader was chunk
    // q - 1, and every thread has passed the barrier after that
    auto next_chunk = [&]() {
        if (!failed && !bar_wait(&S.bars[q % kTrainBufs], (uint32_t)((q / kTrainBufs) & 1))) failed = true;
        if (tid == 0 && q + kTrainBufs - 1 < kFwdChunks + kBwdChunks) issue(q + kTrainBufs - 1);
        return S.w[q % kTrainBufs];
    };
    // ---- forward
    for (int l = 0; l < kLayers; ++l) {
        const __nv_bfloat16* xin = l == 0 ? S.x : S.h[l - 1];
        const int pad = l == 0 ? kXPad : kHPad;
        const bool last = l == kLayers - 1;
        float acc[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
        for (int kc = 0; kc < layer_in(l) / kChunkK; ++kc, ++q) {
            const __nv_bfloat16* wb = next_chunk();
            if (!last) {  // warp: columns [32 warp, 32 warp + 32)
#pragma unroll
                for (int kk = 0; kk < kChunkK; kk += 16) {
                    uint32_t af[4], b0[4], b1[4];
                    frag_a(af, xin, pad, kc * kChunkK + kk, lane);
                    const __nv_bfloat16* p =
                        wb + (size_t)(warp * 32 + (lane >> 4) * 8 + (lane & 7)) * kChunkPad + kk + ((lane >> 3) & 1) * 8;
                    ldsm4(b0, p);
                    ldsm4(b1, p + 16 * kChunkPad);
                    mma_bf16(acc[0], af, b0);
                    mma_bf16(acc[1], af, b0 + 2);
                    mma_bf16(acc[2], af, b1);
                    mma_bf16(acc[3], af, b1 + 2);
                }
            } else if (warp < kOutPad / 8) {  // last layer: warp takes 8 columns
#pragma unroll
                for (int kk = 0; kk < kChunkK; kk += 32) {
                    uint32_t af[4], b[4];
                    ldsm4(b, wb + (size_t)(warp * 8 + (lane & 7)) * kChunkPad + kk + (lane >> 3) * 8);
                    frag_a(af, xin, pad, kc * kChunkK + kk, lane);
                    mma_bf16(acc[0], af, b);
                    frag_a(af, xin, pad, kc * kChunkK + kk + 16, lane);
                    mma_bf16(acc[0], af, b + 2);
                }
            }
            __syncthreads();
        }
        const float* bias = a.params + param_offset_b(l);
        if (!last) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int col = warp * 32 + j * 8 + 2 * t;
                const float c0 = bias[col], c1 = bias[col + 1];
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    *reinterpret_cast<__nv_bfloat162*>(S.h[l] + (size_t)(g + 8 * u) * kHPad + col) =
                        __halves2bfloat162(__float2bfloat16_rn(fmaxf(acc[j][2 * u] + c0, 0.f)),
                                           __float2bfloat16_rn(fmaxf(acc[j][2 * u + 1] + c1, 0.f)));
            }
            __syncthreads();
            store_rows(a.H + ((size_t)l * a.M + row0) * kHid, S.h[l], kHPad, kHid, rows);
        } else {
            if (warp < kOutPad / 8) {
#pragma unroll
                for (int i = 0; i < 4; ++i) S.logits[g + (i >= 2 ? 8 : 0)][warp * 8 + 2 * t + (i & 1)] = acc[0][i];
            }
            __syncthreads();
        }
    }
    // ---- mean softmax cross-entropy: lanes = actions, two rows per warp
    const float* bias = a.params + param_offset_b(kLayers - 1);
    for (int r = warp; r < kTrainRows; r += kTrainThreads / 32) {
        float gval = 0.f, loss = 0.f;
        if (r < rows) {
            const float z = lane < a.n_valid ? S.logits[r][lane] + (lane < kOut ? bias[lane] : 0.f) : -INFINITY;
            float mx = z;
            for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
            const float e = lane < a.n_valid ? expf(z - mx) : 0.f;
            float sum = e;
            for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
            const float p = e / sum;
            const int lab = a.y[row0 + r];
            if (lane < a.n_valid) gval = (p - (lane == lab ? 1.f : 0.f)) / (float)a.M;
            loss = __shfl_sync(kFull, -(logf(p)) / (float)a.M, lab);
        }
        S.logits[r][lane] = gval;
        S.dz[0][(size_t)r * kHPad + lane] = __float2bfloat16_rn(gval);
        if (lane == 0) S.loss[r] = loss;
    }
    __syncthreads();
    if (warp == 0) {
        float s = 0.f;
        for (int r = 0; r < kTrainRows; ++r) s += S.logits[r][lane];
        sums[(kLayers - 1) * kHid + lane] = s;
        if (lane == 0) {
            s = 0.f;
            for (int r = 0; r < kTrainRows; ++r) s += S.loss[r];
            sums[(kLayers - 1) * kHid + kOutPad] = s;
        }
    }
    store_rows(a.dZ + (size_t)(kLayers - 1) * a.M * kHid + (size_t)row0 * kOutPad, S.dz[0], kHPad, kOutPad, rows);
    // ---- backward: gradients of the inputs of layers 4 .. 1, masked by the ReLU below them
    for (int l = kLayers - 1; l > 0; --l) {
        const __nv_bfloat16* dz = S.dz[(kLayers - 1 - l) & 1];
        __nv_bfloat16* out = S.dz[(kLayers - l) & 1];
        const int K = layer_out_pad(l);
        for (int ic = 0; ic < kHid / kChunkK; ++ic, ++q) {
            const __nv_bfloat16* wb = next_chunk() + warp * 8;
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int k = 0; k < K; k += 32) {  // the chunk holds [output][64 inputs]: transposed loads
                uint32_t b[4], a0[4], a1[4];
                ldsm4_t(b, wb + (size_t)(k + lane) * kChunkPad);
                frag_a(a0, dz, kHPad, k, lane);
                frag_a(a1, dz, kHPad, k + 16, lane);
                mma_bf16(acc, a0, b);
                mma_bf16(acc, a1, b + 2);
            }
            const int col = ic * kChunkK + warp * 8 + 2 * t;
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(S.h[l - 1] + (size_t)(g + 8 * u) * kHPad + col);
                const float v0 = __low2float(h) > 0.f ? acc[2 * u] : 0.f, v1 = __high2float(h) > 0.f ? acc[2 * u + 1] : 0.f;
                *reinterpret_cast<__nv_bfloat162*>(out + (size_t)(g + 8 * u) * kHPad + col) =
                    __halves2bfloat162(__float2bfloat16_rn(v0), __float2bfloat16_rn(v1));
                s0 += v0;
                s1 += v1;
            }
            for (int o = 4; o < 32; o <<= 1) {
                s0 += __shfl_xor_sync(kFull, s0, o);
                s1 += __shfl_xor_sync(kFull, s1, o);
            }
            if (g == 0) *reinterpret_cast<float2*>(sums + (l - 1) * kHid + col) = make_float2(s0, s1);
            __syncthreads();
        }
        store_rows(a.dZ + ((size_t)(l - 1) * a.M + row0) * kHid, out, kHPad, kHid, rows);
    }
    if (failed) {  // the copies still in flight, before the block's shared memory is given back
        atomicExch(a.err, FMDP_ERR_TIMEOUT);
        for (int c = kFwdChunks + kBwdChunks - kTrainBufs; c < kFwdChunks + kBwdChunks; ++c)
            bar_wait(&S.bars[c % kTrainBufs], (uint32_t)((c / kTrainBufs) & 1));
    }
}

// Weight gradient of one 64 x 64 tile over one stretch of the batch: part[stretch] = H^T dZ.
namespace {
constexpr int kDwRows = 32;  // batch rows per step
constexpr int kDwPad = 72;   // bf16 per row: 64 + 8
// tiles: layer 0 2 x 4, layers 1 .. 3 4 x 4 each, layer 4 4 x 1 (32 columns)
constexpr int kDwTiles = (kFeat / 64) * 4 + 3 * 16 + 4;
}  // namespace
__global__ void __launch_bounds__(128) train_dw_kernel(const __grid_constant__ TrainArgs a, int k_per) {
    __shared__ __align__(16) __nv_bfloat16 As[3][kDwRows][kDwPad], Bs[3][kDwRows][kDwPad];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    int l, ti, tj;
    {
        const int b = blockIdx.x;
        if (b < 8) {
            l = 0, ti = b >> 2, tj = b & 3;
        } else if (b < kDwTiles - 4) {
            l = 1 + (b - 8) / 16, ti = ((b - 8) >> 2) & 3, tj = b & 3;
        } else {
            l = kLayers - 1, ti = b - (kDwTiles - 4), tj = 0;
        }
    }
    const int in = layer_in(l), ldz = layer_out_pad(l), out = layer_out(l);
    const __nv_bfloat16* A = (l == 0 ? a.X : a.H + (size_t)(l - 1) * a.M * kHid) + ti * 64;
    const __nv_bfloat16* B = a.dZ + (size_t)l * a.M * kHid + tj * 64;  // (layer 4's follow the others)
    const int k0 = blockIdx.y * k_per, k1 = min(a.M, k0 + k_per);
    const int n_step = (k1 - k0 + kDwRows - 1) / kDwRows;
    const int nb = min(64, ldz - tj * 64);  // columns of the tile: 64, or layer 4's 32
    // 32 rows x 64 columns of A and B, 16 bytes per copy; rows past the stretch: zeros
    auto load = [&](int step) {
        const int buf = step % 3;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = tid + u * 128, r = e >> 3, c = (e & 7) * 8, k = k0 + step * kDwRows + r;
            const bool ok = step < n_step && k < k1;
            const __nv_bfloat16* sa = A + (size_t)(ok ? k : 0) * in + c;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(&As[buf][r][c])), "l"(sa),
                         "r"(ok ? 16 : 0)
                         : "memory");
            const bool okb = ok && c < nb;
            const __nv_bfloat16* sb = B + (okb ? (size_t)k * ldz + c : 0);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(&Bs[buf][r][c])), "l"(sb),
                         "r"(okb ? 16 : 0)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[i][j][u] = 0.f;
    load(0);
    load(1);
    for (int step = 0; step < n_step; ++step) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();  // step's tiles are in; the buffer of step - 1 is free
        load(step + 2);
        const int buf = step % 3;
#pragma unroll
        for (int kk = 0; kk < kDwRows; kk += 16) {
            uint32_t af[2][4], bf[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i)  // stored [k][i]: transposed loads
                ldsm4_t(af[i], &As[buf][kk + (lane >> 4) * 8 + (lane & 7)][wm + i * 16 + ((lane >> 3) & 1) * 8]);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                ldsm4_t(bf[j], &Bs[buf][kk + ((lane >> 3) & 1) * 8 + (lane & 7)][wn + j * 16 + (lane >> 4) * 8]);
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j >> 1] + 2 * (j & 1));
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    float* P = a.part + (size_t)blockIdx.y * n_params_total() + param_offset_W(l);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int r = ti * 64 + wm + i * 16 + g + (u >= 2 ? 8 : 0);
                const int c = tj * 64 + wn + j * 8 + 2 * t + (u & 1);
                if (c < out) P[(size_t)r * out + c] = acc[i][j][u];
            }
}

// Blocks [0, w_blocks): the weight gradients' stretches added. The others: the bias gradients,
// 32 columns each, eight warps sharing out the chain kernel's blocks; the last of them also the
// loss.
namespace {
constexpr int kBiasBlocks = ((kLayers - 1) * kHid + kOutPad) / 32;
}
__global__ void __launch_bounds__(256) train_sum_kernel(const __grid_constant__ TrainArgs a, int stretches, int chain_blocks,
                                                        int w_blocks) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t P = n_params_total();
    if ((int)blockIdx.x < w_blocks) {
        for (size_t e = blockIdx.x * 256ull + tid; e < P; e += w_blocks * 256ull) {
            int l = 0;
            while (l < kLayers - 1 && e >= param_offset_W(l + 1)) ++l;
            if (e >= param_offset_b(l)) continue;  // (a bias)
            float v[kTrainSplit];
#pragma unroll
            for (int s = 0; s < kTrainSplit; ++s) v[s] = s < stretches ? a.part[s * P + e] : 0.f;
            float sum = v[0];
#pragma unroll
            for (int s = 1; s < kTrainSplit; ++s) sum += v[s];
            a.grad[e] = sum;
        }
        return;
    }
    __shared__ float part[8][33];
    const int b = blockIdx.x - w_blocks, col = b * 32 + lane;
    auto column = [&](int c) {  // sum of column c over the chain's blocks, in every warp-0 lane's own column
        float s = 0.f;
#pragma unroll 4
        for (int i = warp; i < chain_blocks; i += 8) s += a.sums[(size_t)i * kTrainSums + c];
        __syncthreads();
        part[warp][lane] = s;
        __syncthreads();
        s = 0.f;
        for (int w = 0; w < 8; ++w) s += part[w][lane];
        return s;
    };
    const float s = column(col);
    const int l = col / kHid, j = col - l * kHid;
    if (warp == 0 && j < layer_out(l)) a.grad[param_offset_b(l) + j] = s;
    if (b == kBiasBlocks - 1) {
        const float loss = column((kLayers - 1) * kHid + kOutPad);
        if (tid == 0) *a.loss += loss;
    }
}

cudaError_t prepare_train_kernels() {
    return cudaFuncSetAttribute(train_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
}

cudaError_t launch_train(const TrainArgs& a, cudaStream_t s) {
    if (a.M <= 0) return cudaSuccess;
    const int blocks = train_blocks(a.M);
    train_chain_kernel<<<blocks, kTrainThreads, sizeof(TrainSmem), s>>>(a);
    // A stretch of at least 128 rows: below that its partial sums cost more than they spread.
    int k_per = (a.M + kTrainSplit - 1) / kTrainSplit;
    k_per = (k_per < 128 ? 128 : k_per + kDwRows - 1) / kDwRows * kDwRows;
    const int stretches = (a.M + k_per - 1) / k_per;
    train_dw_kernel<<<dim3(kDwTiles, stretches), 128, 0, s>>>(a, k_per);
    const int w_blocks = 296;
    train_sum_kernel<<<w_blocks + kBiasBlocks, 256, 0, s>>>(a, stretches, blocks, w_blocks);
    return cudaGetLastError();
}

}  // namespace fmdp
