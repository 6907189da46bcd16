// FP32 dense layer for more than a few poses on the tcgen05 tensor cores: y = act(bias + x W^T) with x and W in FP32, each
// operand split into three BF16 parts (24 bits, no scale needed: BF16 has FP32's exponents).
//
// The multiply-adds soon bound the CUDA-core kernels (7.2 GFLOP at 64 x 256 x 221,184: 90 us at the FP32 rate,
// 197 us measured) while the bytes take 42 us.  Six products of the parts keep FP32's accuracy: w0 x0, then w0 x1, w1 x0,
// then w0 x2, w1 x1, w2 x0; the dropped ones are at most 2^-25 of |w x|.  Two things keep the tensor core's truncating
// additions from showing: the small products have accumulators of their own, and w0 x0 is summed four MMAs at a time,
// in six accumulators in turn, which four warps add up in FP32 registers.  (Six accumulators over a sixth of the K range
// each, 31 MMAs, erred 6.7e-7 on all-positive operands, the chains of multiply-adds 1.6e-7.)
//
// A CTA takes 128 output channels (MMA M) x 64 poses (N) x one K split; the splits give about one CTA per SM and their
// partials are added by dense_reduce_kernel.  Twelve warps stream W and x through a ring of 16-byte asynchronous copies
// (72 KB in flight, whole 128-byte lines per request) into slots that only the copying warp reads (no CTA barrier), split
// them and store the parts as K-major core matrices (the K chunks 32 bytes apart modulo the banks, so eight lanes' 16-byte stores touch all of them); a
// further warp issues the MMAs: per 16 of K, w0 x0 (N = 64), w0 [x1 x2], w1 [x0 x1] (N = 128) and w2 x0 (N = 64).  Tensor memory:
// columns [0, 384) the six sums of w0 x0, [384, 448) w0 x1 + w1 x0, [448, 512) the three smallest.
//
// Infinities and NaN: a first part is at most BF16's largest number, so that an infinity is its second part (its third is
// NaN), a large finite value still the sum of its parts, and an output that uses them the infinity or NaN of a chain of
// multiply-adds, once a sum of the smallest products that is not finite is left out.  (Recomputing such outputs by chains
// instead took 4.1 ms for one infinite weight and 13.6 ms for NaN operands at 64 x 256 x 221,184.)  A bounded wait that
// runs out (none should) has every output of the CTA computed by a plain chain over its K range.
//
// Bound: HBM and the latency of the copy - split - MMA chain: 64 x 256 x 221,184 takes 73 us (3.9 TB/s of the 283 MB; 266
// us for the split-K kernel of the CUDA cores that was here, 197 us for its successor), 17 x 128 x 110,592 27 us.  Error
// against float64 8.5e-8 on all-positive operands (split-K chains 1.4e-7 to 3.1e-7).
#include "fusion_internal.cuh"
#include "tc_ptx.cuh"

#include <algorithm>

namespace fusion {

namespace {

constexpr int kM = 128, kN = 64, kBK = 32;       // output channels, poses, K per stage
constexpr int kRing = 4;                         // raw stages
constexpr int kGroups = (kM + kN) / 8;           // groups of 8 rows x kBK, copied and split by a warp
constexpr int kConvWarps = kGroups / 2, kConv = 32 * kConvWarps;
constexpr int kThreads = kConv + 32 + 128;       // converters, the MMA warp, four totalling warps
constexpr uint32_t kRawStage = (kM + kN) * kBK * 4;
constexpr uint32_t kWChunk = kM * 16 + 32, kWPart = (kBK / 8) * kWChunk;      // 8 of K of one part; a part
constexpr uint32_t kXChunk = 3 * kN * 16 + 32, kX = (kBK / 8) * kXChunk;      // the three parts of x side by side
constexpr uint32_t kTile = 3 * kWPart + kX;
constexpr int kSums = 6;                         // accumulators of w0 x0, taken in turn
constexpr int kSumIters = 2;                     // stages per accumulator (4 MMAs)
constexpr uint32_t kSmem = kRing * kRawStage + 2 * kTile + (5 + 2 * kSums) * 8 + 16;
constexpr uint64_t kWaitNs = 1000000000ull;      // 1 s

__device__ __forceinline__ uint32_t pack(__nv_bfloat162 v) { return *reinterpret_cast<uint32_t *>(&v); }

// x -> bf16 parts p[0] + p[1] + p[2] of a pair of values, |p[0]| at most BF16's largest number.
__device__ __forceinline__ void split3(float a, float b, uint32_t (&p)[3]) {
    const __nv_bfloat16 top = __ushort_as_bfloat16(0x7F7F), bottom = __ushort_as_bfloat16(0xFF7F);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        if (i == 0) h = __hmax2(__hmin2(h, __nv_bfloat162(top, top)), __nv_bfloat162(bottom, bottom));
        p[i] = pack(h);
        a -= __uint_as_float(p[i] << 16);
        b -= __uint_as_float(p[i] & 0xffff0000u);
    }
}

__global__ void __launch_bounds__(kThreads, 1) dense_f32tc_kernel(DenseArgs a, int kper) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + kRing * kRawStage + 2 * kTile);   // [2]
    uint64_t *empty = full + 2;                                                            // [2]
    uint64_t *done = empty + 2;
    uint64_t *sum_full = done + 1, *sum_empty = sum_full + kSums;                          // [kSums]
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(sum_empty + kSums);
    volatile int *failed = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n0 = blockIdx.x * kM, b0 = blockIdx.z * kN;
    const int kbeg = blockIdx.y * kper, kend = min(a.K, kbeg + kper);
    const int iters = (kend - kbeg + kBK - 1) / kBK;
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) { tc::mbar_init(&full[i], kConv); tc::mbar_init(&empty[i], 1); }
        tc::mbar_init(done, 1);
        for (int i = 0; i < kSums; ++i) { tc::mbar_init(&sum_full[i], 1); tc::mbar_init(&sum_empty[i], 4); }
        *failed = 0;
        tc::fence_mbar_init();
    }
    if (warp == kConvWarps) tc::tmem_alloc(tmem_slot, 512);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tbase = *tmem_slot;
    const uint64_t deadline = tc::globaltimer() + kWaitNs;     // once the tensor memory is held: another kernel may have had it
    const int sums = (iters + kSumIters - 1) / kSumIters;

    if (warp < kConvWarps) {
        // ---- copy and split: row groups warp and warp + kConvWarps of [W's 16; x's 8] ----
        // A request copies four rows' 128-byte lines; lane's share of a group then is row lane / 4, K chunk lane % 4.
        // The quads of odd rows are stored in swapped pairs, so eight lanes' reads touch all banks.
        auto copy = [&](int it) {
            if (it < iters) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int g = warp + kConvWarps * i;
                    const bool is_w = g < kM / 8;
                    const int first = is_w ? n0 + g * 8 : b0 + g * 8 - kM, rows = is_w ? a.N : a.B;
                    const float *m = is_w ? a.w : a.x;
                    unsigned char *st = smem + (it % kRing) * kRawStage + g * (8 * kBK * 4);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int r = h * 4 + (lane >> 3), c4 = lane & 7, k = kbeg + it * kBK + c4 * 4;
                        const bool ok = first + r < rows && k < kend;           // kend is a multiple of 8
                        const float *p = m + (size_t)min(first + r, rows - 1) * a.K + (k < kend ? k : 0);
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                                         tc::smem_u32(st + r * (kBK * 4) + (c4 ^ (r & 1)) * 16)),
                                     "l"(p), "r"(ok ? 16 : 0));
                    }
                }
            }
            asm volatile("cp.async.commit_group;");
        };
        for (int it = 0; it < kRing - 1; ++it) copy(it);
        for (int it = 0; it < iters; ++it) {
            copy(it + kRing - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 1) : "memory");
            __syncwarp();
            const int buf = it & 1, r = lane >> 2, c = lane & 3;
            uint32_t p[2][4][3];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const unsigned char *st = smem + (it % kRing) * kRawStage + (warp + kConvWarps * i) * (8 * kBK * 4) + r * (kBK * 4);
                const float4 u = *reinterpret_cast<const float4 *>(st + ((2 * c) ^ (r & 1)) * 16);
                const float4 v = *reinterpret_cast<const float4 *>(st + ((2 * c + 1) ^ (r & 1)) * 16);
                split3(u.x, u.y, p[i][0]);
                split3(u.z, u.w, p[i][1]);
                split3(v.x, v.y, p[i][2]);
                split3(v.z, v.w, p[i][3]);
            }
            __syncwarp();                                   // the slots are free for the next copies
            if (!tc::mbar_wait(&empty[buf], ((it >> 1) & 1) ^ 1, deadline)) { *failed = 1; break; }
            unsigned char *tile = smem + kRing * kRawStage + buf * kTile;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int g = warp + kConvWarps * i;
                const bool is_w = g < kM / 8;
                unsigned char *dst = is_w ? tile + c * kWChunk + (g * 8 + r) * 16
                                          : tile + 3 * kWPart + c * kXChunk + (g * 8 - kM + r) * 16;
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    *reinterpret_cast<uint4 *>(dst + q * (is_w ? kWPart : (uint32_t)(kN * 16))) =
                        make_uint4(p[i][0][q], p[i][1][q], p[i][2][q], p[i][3][q]);
            }
            tc::fence_proxy_async();
            tc::mbar_arrive(&full[buf]);
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    } else if (warp == kConvWarps) {
        // ---- MMA warp, converged; one elected lane issues ----
        const uint32_t on = tc::elect_one();
        constexpr uint32_t I64 = tc::idesc_bf16(kM, kN), I128 = tc::idesc_bf16(kM, 2 * kN);
        const uint32_t small = tbase + kSums * kN;
        int acc = 0;                             // accumulator of w0 x0 in turn, and the parity of its turn
        uint32_t par = 0;
        for (int it = 0; it < iters; ++it) {
            const int buf = it & 1;
            const bool fresh = it % kSumIters == 0;
            bool ok = tc::mbar_wait(&full[buf], (it >> 1) & 1, deadline);
            if (fresh) ok = ok && tc::mbar_wait(&sum_empty[acc], par ^ 1, deadline);
            if (!__all_sync(0xffffffffu, ok) || __any_sync(0xffffffffu, *failed != 0)) { *failed = 1; break; }
            tc::tc_fence_after();
            const uint32_t t = tc::smem_u32(smem + kRing * kRawStage + buf * kTile);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk) {
                uint64_t w[3], x[3];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    w[q] = tc::desc_kmajor(t + q * kWPart + 2 * kk * kWChunk, kWChunk, 128);
                    x[q] = tc::desc_kmajor(t + 3 * kWPart + 2 * kk * kXChunk + q * kN * 16, kXChunk, 128);
                }
                if (on) {
                    tc::mma_bf16(small, w[0], x[1], I128, it > 0 || kk > 0);       // [w0 x1 | w0 x2]
                    tc::mma_bf16(small, w[1], x[0], I128, 1);                      // [w1 x0 | w1 x1]
                    tc::mma_bf16(small + kN, w[2], x[0], I64, 1);                  // w2 x0
                    tc::mma_bf16(tbase + acc * kN, w[0], x[0], I64, !fresh || kk > 0);
                }
            }
            if (on) tc::mma_commit(&empty[buf]);
            if (it % kSumIters == kSumIters - 1 || it == iters - 1) {
                if (on) tc::mma_commit(&sum_full[acc]);
                if (++acc == kSums) { acc = 0; par ^= 1; }
            }
        }
        if (on) tc::mma_commit(done);
        if (!__all_sync(0xffffffffu, tc::mbar_wait(done, 0, tc::globaltimer() + kWaitNs))) *failed = 1;
    } else {
        // ---- totals: lane quarter warp % 4, row = output channel ----
        const int quarter = warp & 3, n = n0 + quarter * 32 + lane;
        const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
        float tot[kN];
#pragma unroll
        for (int j = 0; j < kN; ++j) tot[j] = 0.f;
        auto add = [&](int col, bool finite_only) {
#pragma unroll
            for (int c = 0; c < kN; c += 16) {       // 16 at a time: 32 registers beside the totals would spill
                uint32_t v[16];
                tc::tmem_ld16(tbase + lanes + (uint32_t)(col + c), v);
                tc::tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const float t = __uint_as_float(v[j]);
                    if (!finite_only || fabsf(t) < INFINITY) tot[c + j] += t;
                }
            }
        };
        bool ok = true;
        for (int q = 0; q < sums && ok; ++q) {
            const int acc = q % kSums;
            // tensor-memory loads need all 32 lanes
            ok = __all_sync(0xffffffffu, tc::mbar_wait(&sum_full[acc], (q / kSums) & 1, deadline)) &&
                 !__any_sync(0xffffffffu, *failed != 0);
            if (!ok) break;
            tc::tc_fence_after();
            add(acc * kN, false);
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&sum_empty[acc]);
        }
        ok = __all_sync(0xffffffffu, ok && tc::mbar_wait(done, 0, deadline)) && !__any_sync(0xffffffffu, *failed != 0);
        if (ok) {
            tc::tc_fence_after();
            add((kSums + 1) * kN, true);
            add(kSums * kN, false);
        } else {
            *failed = 1;
        }
        if (n < a.N) {
#pragma unroll
            for (int j = 0; j < kN; ++j) {
                const int b = b0 + j;
                if (b >= a.B) break;
                float s = tot[j];
                if (!ok) {
                    const float *w = a.w + (size_t)n * a.K, *x = a.x + (size_t)b * a.K;
                    s = 0.f;
                    for (int k = kbeg; k < kend; ++k) s = fmaf(x[k], w[k], s);
                }
                a.part[((size_t)blockIdx.y * a.B + b) * a.N + n] = s;
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == kConvWarps) tc::tmem_dealloc(tbase, 512);
}

}  // namespace

void launch_dense_f32tc(DenseArgs a, size_t partials, int sms, cudaStream_t s) {
    // about one CTA per SM for 64 rows, no fewer than 512 of K each, in whole stages.  A function of N and K alone: a row's
    // sums do not depend on the rows beside it.  (More rows are more rounds of CTAs, each with its start and end, where a
    // split by the batch made each CTA's range longer: 128 rows x 128 x 110,592 48 -> 66 us, 65 x 256 x 221,184 130 -> 144.)
    const int mt = (a.N + kM - 1) / kM;
    const int want = std::max(1, std::min(sms / mt, (a.K + 511) / 512));
    const int kper = ((a.K + want - 1) / want + kBK - 1) / kBK * kBK;
    a.splits = (a.K + kper - 1) / kper;
    // rows whose partials fit (splits x N is under 128 x sms, or N with one split): a launch takes those
    size_t rows = std::max<size_t>(1, partials / ((size_t)a.splits * a.N));
    if (rows >= kN) rows = rows / kN * kN;
    cudaFuncSetAttribute(dense_f32tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    const int total = a.B;
    for (int b0 = 0; b0 < total; b0 += a.B) {
        a.B = (int)std::min<size_t>(rows, total - b0);
        dense_f32tc_kernel<<<dim3(mt, a.splits, (a.B + kN - 1) / kN), kThreads, kSmem, s>>>(a, kper);
        launch_dense_reduce(a, s);
        a.x += (size_t)a.B * a.K;
        a.y += (size_t)a.B * a.N;
    }
}

}  // namespace fusion
