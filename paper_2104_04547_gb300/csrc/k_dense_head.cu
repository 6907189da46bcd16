// CNN dense layer and fusion head.
//
// CNN dense in FP32 (Section 3.3.1: flatten -> dense + ReLU): y[b][n] = ReLU(bias[n] + sum_k x[b][k] W[n][k]) with
// K = pooled voxels x channels (221,184 for the full-size model), a split-K product whose order of additions
// depends on K only: split s, its eight sub-slices of K, in each a chain of multiply-adds in k order; the eight
// chains are added in order, then a second kernel adds the splits.  So a pose's result does not depend on its batch,
// and two kernels can share the work by batch size:
//   * up to 16 poses the weight stream is the bound, and dense_stream_kernel keeps it flowing: a warp takes one
//     sub-slice of 32 weight rows, a lane per row, through a private ring of 16-byte asynchronous copies (up to 128 KB in
//     flight per SM with two CTAs), with no CTA barrier until the end;
//   * above that the multiply-adds are (7.2 GFLOP at 64 poses: 90 us at the FP32 rate, 42 us for the bytes), and
//     dense_tile_kernel gives each warp one sub-slice of a 64 x 64 (or 64 x 32) tile, a lane 8 x 16 outputs, reading
//     k-quads of rows as they lie in memory (a transpose would cost as many stores as the loads it saves).
// The line between them is where 16 sums per weight still fit a lane and cost less than the stream (23 of 33 us).
// The weight rows were permuted at model creation so that the flatten of the NDHWC pooled map is a plain row read.
// Measured with the reduction: 4 x 128 x 110,592 127 -> 21.5 us (58 MB, 2.7 TB/s; through the no-allocation entry, which
// takes these kernels up to 8 rows), 64 x 256 x 221,184 266 -> 197 us (36.8 TFLOP/s); the dense layer of the single-pose
// 24^3 model 100 -> 16 us, of the full-size model at 3 poses 256 -> 61 us.  Errors against float64 fell from 6e-7 to 2.4e-7 (chains of 256, not 2048).
//
// Fusion head (Section 3.3.3, Table V: fusion dense layers with SELU): one CTA
// per pose runs Linear -> SELU -> ... -> Linear on [cnn latent, sg latent].
#include "fusion_internal.cuh"

namespace fusion {

namespace {

constexpr int kDenseWarps = 8;            // sub-slices of a split, one warp each
constexpr int kDenseThreads = 32 * kDenseWarps;

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(ok ? 16 : 0));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N)); }

// K range [kb, ke) of warp q in split s: splits of kper (a multiple of 64), eight sub-slices each (empty past K).
__device__ __forceinline__ void dense_range(const DenseArgs &a, int q, int &kb, int &ke) {
    const int kper = ((a.K + a.splits - 1) / a.splits + 63) / 64 * 64, sub = kper / kDenseWarps;
    kb = blockIdx.y * kper + q * sub;
    ke = min(a.K, kb + sub);
}

// `rows` rows from r0 of a [.. limit][K] matrix, columns [k, k + KC) (zero past ke and past the last row), into a tile
// with rows of KC + 4 floats: a warp's 16-byte reads down eight rows then touch all banks.
template <int KC>
__device__ __forceinline__ void dense_stage(float *tile, const float *m, int r0, int rows, int limit, int K, int k, int ke,
                                            int lane) {
    for (int e = lane; e < rows * (KC / 4); e += 32) {
        const int r = e / (KC / 4), c = (e % (KC / 4)) * 4;
        const bool ok = r0 + r < limit && k + c < ke;       // ke is a multiple of 8: a quad is all in or all out
        cp_async16(tile + r * (KC + 4) + c, ok ? m + (size_t)(r0 + r) * K + k + c : m, ok);
    }
}

constexpr int kStreamRows = 32, kStreamKC = 16;
template <int BT>
struct StreamTile {
    static constexpr int STAGES = BT <= 4 ? 5 : BT <= 8 ? 4 : 3;       // the most that leave room for two CTAs on an SM
    static constexpr int LD = kStreamKC + 4, STAGE = (kStreamRows + BT) * LD, RING = STAGES * STAGE;   // floats, a warp's
};

template <int BT>
__global__ void __launch_bounds__(kDenseThreads, 2) dense_stream_kernel(DenseArgs a) {
    extern __shared__ __align__(16) float dsm[];
    launch_next();
    wait_prior();
    using S = StreamTile<BT>;
    constexpr int LD = S::LD, STAGE = S::STAGE, STAGES = S::STAGES;
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int n0 = blockIdx.x * kStreamRows;
    const float *x = a.x, *w = a.w;
    float *ring = dsm + q * S::RING;
    int kb, ke;
    dense_range(a, q, kb, ke);
    const int steps = ke > kb ? (ke - kb + kStreamKC - 1) / kStreamKC : 0;
    auto load = [&](int i) {
        if (i < steps) {
            float *st = ring + (i % STAGES) * STAGE;
            dense_stage<kStreamKC>(st, w, n0, kStreamRows, a.N, a.K, kb + i * kStreamKC, ke, lane);
            dense_stage<kStreamKC>(st + kStreamRows * LD, x, 0, BT, a.B, a.K, kb + i * kStreamKC, ke, lane);
        }
        cp_async_commit();
    };
    float acc[BT];
#pragma unroll
    for (int b = 0; b < BT; ++b) acc[b] = 0.f;
    for (int i = 0; i < STAGES - 1; ++i) load(i);
    for (int i = 0; i < steps; ++i) {
        load(i + STAGES - 1);
        cp_async_wait<STAGES - 1>();
        __syncwarp();
        const float *st = ring + (i % STAGES) * STAGE;
#pragma unroll
        for (int c = 0; c < kStreamKC; c += 4) {
            const float4 w4 = *reinterpret_cast<const float4 *>(st + lane * LD + c);
#pragma unroll
            for (int b = 0; b < BT; ++b) {
                const float4 x4 = *reinterpret_cast<const float4 *>(st + (kStreamRows + b) * LD + c);
                acc[b] = fmaf(x4.x, w4.x, acc[b]);
                acc[b] = fmaf(x4.y, w4.y, acc[b]);
                acc[b] = fmaf(x4.z, w4.z, acc[b]);
                acc[b] = fmaf(x4.w, w4.w, acc[b]);
            }
        }
        __syncwarp();                            // the stage is free for the copies of the next iteration
    }
    cp_async_wait<0>();
    __syncthreads();
    // the eight chains in order
    float *red = dsm;                            // [8][BT][32]
#pragma unroll
    for (int b = 0; b < BT; ++b) red[(q * BT + b) * 32 + lane] = acc[b];
    __syncthreads();
    for (int e = threadIdx.x; e < BT * 32; e += kDenseThreads) {
        const int b = e >> 5, n = n0 + (e & 31);
        float s = red[e];
#pragma unroll
        for (int j = 1; j < kDenseWarps; ++j) s += red[j * BT * 32 + e];
        if (b < a.B && n < a.N) a.part[((size_t)blockIdx.y * a.B + b) * a.N + n] = s;
    }
}

constexpr int kTileN = 64, kTileKC = 16;
template <int BT>
struct GemmTile {
    static constexpr int LD = kTileKC + 4, STAGE = (kTileN + BT) * LD, RING = 2 * STAGE;               // floats, a warp's
};

// BT poses (64 or 32): a lane's outputs are rows lane % 8 + 8 j and poses lane / 8 + 4 i.
template <int BT>
__global__ void __launch_bounds__(kDenseThreads, 1) dense_tile_kernel(DenseArgs a) {
    extern __shared__ __align__(16) float dsm[];
    launch_next();
    wait_prior();
    using S = GemmTile<BT>;
    constexpr int LD = S::LD, STAGE = S::STAGE, NI = BT / 4;
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int n0 = blockIdx.x * kTileN, b0 = blockIdx.z * BT;
    const int ln = lane & 7, lb = lane >> 3;
    const float *x = a.x, *w = a.w;
    float *ring = dsm + q * S::RING;
    int kb, ke;
    dense_range(a, q, kb, ke);
    const int steps = ke > kb ? (ke - kb + kTileKC - 1) / kTileKC : 0;
    auto load = [&](int i) {
        if (i < steps) {
            float *st = ring + (i & 1) * STAGE;
            dense_stage<kTileKC>(st, w, n0, kTileN, a.N, a.K, kb + i * kTileKC, ke, lane);
            dense_stage<kTileKC>(st + kTileN * LD, x, b0, BT, a.B, a.K, kb + i * kTileKC, ke, lane);
        }
        cp_async_commit();
    };
    float acc[NI][8];
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
    load(0);
    for (int s = 0; s < steps; ++s) {
        load(s + 1);
        cp_async_wait<1>();
        __syncwarp();
        const float *ws = ring + (s & 1) * STAGE + ln * LD, *xs = ring + (s & 1) * STAGE + (kTileN + lb) * LD;
#pragma unroll 1
        for (int c = 0; c < kTileKC; c += 4) {
            float4 wv[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) wv[j] = *reinterpret_cast<const float4 *>(ws + 8 * j * LD + c);
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const float4 xv = *reinterpret_cast<const float4 *>(xs + 4 * i * LD + c);
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xv.x, wv[j].x, acc[i][j]);
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xv.y, wv[j].y, acc[i][j]);
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xv.z, wv[j].z, acc[i][j]);
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(xv.w, wv[j].w, acc[i][j]);
            }
        }
        __syncwarp();
    }
    cp_async_wait<0>();
    __syncthreads();
    float *red = dsm;                            // [8][BT][64]
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) red[(q * BT + lb + 4 * i) * kTileN + ln + 8 * j] = acc[i][j];
    __syncthreads();
    for (int e = threadIdx.x; e < BT * kTileN; e += kDenseThreads) {
        const int b = b0 + e / kTileN, n = n0 + e % kTileN;
        float s = red[e];
#pragma unroll
        for (int j = 1; j < kDenseWarps; ++j) s += red[j * BT * kTileN + e];
        if (b < a.B && n < a.N) a.part[((size_t)blockIdx.y * a.B + b) * a.N + n] = s;
    }
}

// Sum of the split partials plus bias and activation: a block takes 32 outputs, its eight warps an eighth of the
// splits each (in order), and the eight sums are added in order, so the result does not depend on the batch.  Bound by
// the latency of its loads: one thread per output walked 108 partials in 14 rounds, a warp now holds its 14 in flight.
__global__ void __launch_bounds__(256) dense_reduce_kernel(DenseArgs a) {
    __shared__ float sums[8][32];
    launch_next();
    wait_prior();
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane, tot = a.B * a.N;
    const int per = (a.splits + 7) / 8, lo = q * per, hi = min(a.splits, lo + per);
    float s = 0.f;
    if (e < tot) {
        const float *p = a.part + e;
        for (int i = lo; i < hi; i += 16) {
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = i + j < hi ? p[(size_t)(i + j) * tot] : 0.f;
#pragma unroll
            for (int j = 0; j < 16; ++j) s += v[j];
        }
    }
    sums[q][lane] = s;
    __syncthreads();
    if (q == 0 && e < tot) {
#pragma unroll
        for (int j = 1; j < 8; ++j) s += sums[j][lane];
        s += a.bias[e % a.N];
        a.y[e] = a.relu ? fmaxf(s, 0.f) : s;
    }
}

__device__ __forceinline__ float selu(float x) {
    const float alpha = 1.6732632423543772848f, scale = 1.0507009873554804934f;
    return x > 0.f ? scale * x : scale * alpha * expm1f(x);
}

constexpr int kHeadThreads = 512;

// One dense layer of the head for one pose, all threads of the CTA: out[o] = act(b[o] + sum_k in[k] W[o][k])
// (weights stored transposed, [in][out]); act 0 = none, 1 = ReLU, 2 = SELU; `res` adds in[o] after the
// activation.  `in` and `out` are distinct shared-memory buffers.  A narrow layer splits its inputs into ks
// contiguous ranges (ks = 2, 4 or 8, as many as the CTA's threads allow), summed by different threads and
// added in range order after the bias, so its chains of dependent multiply-adds (and weight loads) are ks
// times shorter; the order depends only on the layer's shape.
__device__ void head_layer(const float *in, int fin, float *out, int fout, const float *wt, const float *bias,
                           int act, bool res) {
    __shared__ float part[kHeadThreads];
    int ks = 1;
    while (ks < 8 && fout * ks * 2 <= (int)blockDim.x) ks *= 2;
    if (ks == 1) {
        for (int o = threadIdx.x; o < fout; o += blockDim.x) {
            float s = bias[o];
            for (int k = 0; k < fin; ++k) s = fmaf(wt[(size_t)k * fout + o], in[k], s);
            if (act == 1) s = fmaxf(s, 0.f);
            else if (act == 2) s = selu(s);
            out[o] = res ? in[o] + s : s;
        }
        __syncthreads();
        return;
    }
    const int chunk = (fin + ks - 1) / ks;
    if ((int)threadIdx.x < fout * ks) {
        const int o = threadIdx.x % fout, q = threadIdx.x / fout;
        const int k1 = min(fin, (q + 1) * chunk);
        float s = 0.f;
        for (int k = q * chunk; k < k1; ++k) s = fmaf(wt[(size_t)k * fout + o], in[k], s);
        part[q * fout + o] = s;
    }
    __syncthreads();
    if ((int)threadIdx.x < fout) {
        const int o = threadIdx.x;
        float s = bias[o];
        for (int q = 0; q < ks; ++q) s += part[q * fout + o];
        if (act == 1) s = fmaxf(s, 0.f);
        else if (act == 2) s = selu(s);
        out[o] = res ? in[o] + s : s;
    }
    __syncthreads();
}

// Ask L2 for the CTA's share of a weight matrix's 128-byte lines (the head's weights, used by every CTA, are
// usually out of L2 after the convolutions' streams; each CTA otherwise walks them from DRAM in dependent rounds).
__device__ __forceinline__ void prefetch_share(const float *w, size_t n) {
    if (!w) return;
    const size_t lines = (n * 4 + 127) / 128;
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < lines; q += (size_t)gridDim.x * blockDim.x)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char *>(w) + q * 128));
}

// Coherent Fusion: fusion layers on [cnn, sg].  Mid-level: each latent through its branch layers (SELU
// after each), the two results appended after the latents, then the fusion layers.  Late: each latent
// through its own affinity stack (ReLU between, last linear), the mean of the two.
__global__ void __launch_bounds__(kHeadThreads) head_kernel(HeadArgs a) {
    __shared__ float v[3][kHeadMaxWidth];
    const int p = blockIdx.x;
    const int fin0 = a.Dc + a.G;
    {
        int fin = fin0;
        for (int br = 0; br < 2; ++br) {
            int bin = br == 0 ? a.Dc : a.G;
            for (int l = 0; l < a.n_branch[br]; ++l) {
                prefetch_share(a.bwt[br][l], (size_t)bin * a.bwidth[br][l]);
                bin = a.bwidth[br][l];
            }
            if (a.mode == FUSION_MID) fin += bin;
        }
        for (int l = 0; l < a.n_layers; ++l) {
            prefetch_share(a.wt[l], (size_t)fin * a.width[l]);
            fin = a.width[l];
        }
    }
    for (int i = threadIdx.x; i < fin0; i += blockDim.x)
        v[0][i] = i < a.Dc ? a.cnn[(size_t)p * a.Dc + i] : a.sg[(size_t)p * a.G + (i - a.Dc)];
    __syncthreads();
    if (a.mode == FUSION_LATE) {
        float aff[2];
        for (int br = 0; br < 2; ++br) {
            const float *in = v[0] + (br == 0 ? 0 : a.Dc);
            int fin = br == 0 ? a.Dc : a.G, cur = 1;
            for (int l = 0; l < a.n_branch[br]; ++l) {
                const bool last = l + 1 == a.n_branch[br];
                head_layer(in, fin, v[cur], a.bwidth[br][l], a.bwt[br][l], a.bb[br][l], last ? 0 : 1, false);
                in = v[cur];
                cur = cur == 1 ? 2 : 1;
                fin = a.bwidth[br][l];
            }
            aff[br] = in[0];
            __syncthreads();
        }
        if (threadIdx.x == 0) a.out[p] = 0.5f * (aff[0] + aff[1]);
        return;
    }
    int fin = fin0;
    if (a.mode == FUSION_MID) {
        for (int br = 0; br < 2; ++br) {
            const float *in = v[0] + (br == 0 ? 0 : a.Dc);
            int bin = br == 0 ? a.Dc : a.G, cur = 1;
            for (int l = 0; l < a.n_branch[br]; ++l) {
                head_layer(in, bin, v[cur], a.bwidth[br][l], a.bwt[br][l], a.bb[br][l], 2, false);
                in = v[cur];
                cur = cur == 1 ? 2 : 1;
                bin = a.bwidth[br][l];
            }
            for (int i = threadIdx.x; i < bin; i += blockDim.x) v[0][fin + i] = in[i];
            __syncthreads();
            fin += bin;
        }
    }
    int cur = 0;
    for (int l = 0; l < a.n_layers; ++l) {
        const int fout = a.width[l];
        const bool last = l + 1 == a.n_layers;
        const int nxt = cur == 0 ? 1 : 0;
        head_layer(v[cur], fin, v[nxt], fout, a.wt[l], a.b[l], last ? 0 : 2, !last && a.residual && fin == fout);
        cur = nxt;
        fin = fout;
    }
    if (threadIdx.x == 0) a.out[p] = v[cur][0];
}

}  // namespace

int dense_splits(int K) {
    int s = K / 2048;
    if (s < 1) s = 1;
    if (s > 128) s = 128;
    return s;
}

template <int BT>
static void launch_stream(const DenseArgs &a, cudaStream_t s) {
    const size_t ring = (size_t)kDenseWarps * StreamTile<BT>::RING * 4;      // covers the [8][BT][32] sums too
    cudaFuncSetAttribute(dense_stream_kernel<BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring);
    launch_kernel(dense_stream_kernel<BT>, dim3((a.N + kStreamRows - 1) / kStreamRows, a.splits), kDenseThreads, ring, s,
                  a.early, a);
}

template <int BT>
static void launch_tile(const DenseArgs &a, cudaStream_t s) {
    const size_t ring = (size_t)kDenseWarps * GemmTile<BT>::RING * 4;        // covers the [8][BT][64] sums too
    cudaFuncSetAttribute(dense_tile_kernel<BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring);
    launch_kernel(dense_tile_kernel<BT>, dim3((a.N + kTileN - 1) / kTileN, a.splits, (a.B + BT - 1) / BT), kDenseThreads,
                  ring, s, a.early, a);
}

void launch_dense(const DenseArgs &a, cudaStream_t s) {
    if (a.B <= 1) launch_stream<1>(a, s);
    else if (a.B <= 4) launch_stream<4>(a, s);
    else if (a.B <= 8) launch_stream<8>(a, s);
    else if (a.B <= 16) launch_stream<16>(a, s);
    else if (a.B <= 32) launch_tile<32>(a, s);
    else launch_tile<64>(a, s);
    launch_dense_reduce(a, s);
}

void launch_dense_reduce(const DenseArgs &a, cudaStream_t s) {
    const int tot = a.B * a.N;
    launch_kernel(dense_reduce_kernel, (tot + 31) / 32, 256, 0, s, a.early, a);
}

void launch_head(const HeadArgs &a, cudaStream_t s) {
    head_kernel<<<a.B, kHeadThreads, 0, s>>>(a);
}

}  // namespace fusion
