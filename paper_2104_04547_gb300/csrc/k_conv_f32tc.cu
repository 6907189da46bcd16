// FP32 3D convolution on the tcgen05 tensor cores (Section 3.3.1, Table III): the FP32 path's convolutions as
// three FP16 products of two-part operands, at the accuracy of FP32 multiply-adds.
//
// Operands: x * s_x = x_hi + x_lo and w * s_w = w_hi + w_lo, each part FP16 (x_hi the rounded value, x_lo the
// rounded rest), with power-of-two scales (s_x per pose from its largest |x|, s_w per output channel) that put
// the largest magnitude in [2^14, 2^15), so the parts keep 22 bits and even values 2^-24 of the largest keep
// 14.  The sum is x_lo w_hi + x_hi w_lo + x_hi w_hi; the dropped x_lo w_lo is at most 2^-22 of a product.
// The FP16 products are exact in the MMA.  Scaling back is exact.
//
// What bounds the accuracy is the accumulation: the tensor core adds with truncation, so thousands of MMAs into
// one FP32 accumulator would lose more than the FP32 chain of multiply-adds they replace (21,952 terms per
// output in the full-size residual layers).  Hence the small products have accumulator columns of their own,
// added up once per tile (truncation there acts on values 2^-11 of the result's), and the large product is summed
// in intervals of at most kFlushTaps kernel offsets, after each of which epilogue warps add the interval's sums, in
// FP32 with rounding, to the outputs' totals in their registers.  Intervals and the order of every sum depend on the
// layer only (not on the tile or the batch), so a pose's result depends on nothing but the pose.
//
// Infinities and NaN: the scales are those of the finite values, an infinity's low part is 0 and sums of small products
// that are not finite are left out, so that x_hi w_hi alone gives an output what a chain of multiply-adds would: the
// infinity of its sign, NaN where two disagree, and every output whose terms are finite keeps its value.  (In a folded
// 7^3 first layer an infinity of features 16..18 meets the zero weights of slots read twice: outputs within a voxel of it
// along x are NaN, stored as 0.)
//
// Tiles: M = 128 voxels (16 x 8), T output slices and NT output channels per CTA.  Operand A is read from a
// TMA-loaded halo by sliding descriptors as in k_conv_tc.cu, weights stream in whole (ty, tx) groups.  The
// halo of x_lo is multiplied with w_hi (N = NT), the halo of x_hi with [w_hi | w_lo] (N = 2 NT), so one read of
// an A tile serves two products: an MMA takes the larger of N / 2 clocks and its operand reads (4 KB + 32 N bytes at
// 128 bytes a clock; measured 40, 48, 64, 128 clocks at N = 32, 64, 128, 256).  Each MMA serves one slice, so a
// slice's sums are added up while the next slices' MMAs run.
//
// Bound: those operand reads, 112 clocks per kernel offset, 16 channels and slice at NT = 64 against 96 of math.
// Measured, full-size residual layer (64 channels, 7^3): 8.46 ms -> 0.74 ms for one pose, 25.1 -> 1.6 ms for three
// against the FP32 multiply-add kernel (36 TFLOP/s).  Error against float64, 2-norm of the output's, over the layers of the
// 20^3, 24^3, paper-final and full-size models at 224 to 860 atoms: 1.4e-7 to 3.0e-7, of the multiply-adds 2.4e-7 to 1.4e-6,
// and smaller in every layer.
#include "fusion_internal.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdio>

namespace fusion {

namespace {

constexpr int kRing = 4;                       // tile indices the producer publishes ahead
constexpr int kFlushTaps = 14;                 // kernel offsets of the large product per interval
constexpr uint64_t kWaitNs = 1000000000ull;    // 1 s

// NT output channels, T output slices.  A slice's accumulators: NT columns of x_hi w_hi, NT of the small products.
template <int NT, int T>
struct Roles {
    static constexpr int UCOLS = 2 * NT;
    static constexpr int COLS = T * UCOLS;
    static constexpr int NI = 2;                                // MMA-issuing warps, each owns T / NI slices
    static constexpr int EG = 2;                                // epilogue groups of 4 warps; group e totals slices e, e + EG, ..
    static constexpr int OWN = T / EG;                          // slices an epilogue warp totals
    static constexpr int EPI0 = 1 + NI;
    static constexpr int THREADS = 32 * (EPI0 + 4 * EG);
};

struct Geo {
    int nbx, nby, nbz;     // tiles along x (8), y (16), z (T)
    int nphase;            // 1, or the 8 input parity phases of stride 2
    int ntap[2];           // taps per dimension of parity 0 / 1, or k
    int hd, hh, hw;        // halo extents
    uint32_t plane_bytes;  // one 8-channel plane of a plain-layout halo, 128-byte aligned
    uint32_t a_bytes;      // one halo buffer
    uint32_t lbo_a;        // bytes between the two K halves of a voxel row
    int ystep;             // 16-byte rows between y rows of the buffer
    uint32_t stage_bytes;  // one weight stage
    int gps[2];            // (ty, tx) groups per weight stage of the x_lo / x_hi product
    int nblk;              // blocks of NT output channels
    int flush_groups;      // (ty, tx) groups of the large product per interval
    int nbs, na, chunks;
};

struct Args {
    const uint8_t *w[2];   // arranged weights (conv_f32tc_arrange_weights): w_hi, and [w_hi | w_lo]
    size_t wblk;           // bytes of w[0] per block of NT output channels
    const float *inv_sw;   // [c_out] 1 / s_w
    const float *inv_sx;   // [B] 1 / s_x (this and the maps below from the launch's first pose on)
    const float *bias;     // [c_out]
    const float *xres;     // residual source [B][n_out]^3[c_out], or unused
    float *y;              // [B][n_out]^3[c_out]
    int c_out;
    float *amax;           // per-pose max |output| (atomic max; may be null)
    int n_out, k, stride, pad, residual, B, max_poses;
    int xpat, xt_n[2], xt_step[2], xt_start[2];   // x-folded first layer (see k_conv_tc.cu)
    int blocked;           // input layout: 0 NDHWC, 1 channel-blocked, 2 parity-split
    Geo g;
    unsigned *err;
    int stall;             // test of the bounded waits: the producer loads nothing
    int *tile_counter;     // [0] tiles handed out beyond each CTA's first, [1] CTAs done (both zero between launches)
};

__device__ __forceinline__ void phase_taps(const Args &a, int ph, int &pz, int &py, int &px, int &nz, int &ny,
                                           int &nx) {
    if (a.stride == 1) {
        pz = py = px = 0;
        nz = ny = nx = a.k;
    } else {
        pz = (ph >> 2) & 1;
        py = (ph >> 1) & 1;
        px = ph & 1;
        nz = a.g.ntap[pz];
        ny = a.g.ntap[py];
        nx = a.g.ntap[px];
    }
}

// (ty, tx) groups of chunk c, phase ph (0: the phase has no taps and is skipped by every role).
__device__ __forceinline__ int phase_groups(const Args &a, int c, int ph) {
    int pz, py, px, nz, ny, nx;
    phase_taps(a, ph, pz, py, px, nz, ny, nx);
    if (a.xpat) nx = a.xt_n[c];
    return nz > 0 ? ny * nx : 0;
}

// The MMAs of one slice over `cnt` (ty, tx) groups from (.., tx): ROWS = N B rows per kernel offset, tz = 0 stored
// last in a group.  What the tensor pipe waits for here is the issuing warp's scalar work, so a group's MMAs unroll to
// one add per operand each (NZ is a template parameter), the warp runs converged with one elected lane issuing (the
// operands then sit in uniform registers), and block bookkeeping has no divisions: 166 -> 111 clocks per MMA and
// issuing warp in the full-size residual layers (890 -> 610 thousand clocks of MMAs per 4-slice tile with two warps;
// the operand reads of N = 64 and 128 allow 48 and 64 per MMA, 615 thousand).
template <int NZ, int ROWS>
__device__ __forceinline__ void issue(uint32_t on, uint32_t dt, uint32_t al, uint32_t ah, uint32_t bl, uint32_t bh, int cnt, int tx,
                                      int nx, int xstep, uint32_t wrap, uint32_t row_zy, uint32_t idesc) {
#pragma unroll 1
    for (int i = 0; i < cnt; ++i) {
        uint32_t a = al;
#pragma unroll
        for (int tz = 0; tz < NZ; ++tz) {
            tc::mma_acc<false>(on, dt, a, ah, bl + (uint32_t)((NZ - 1 - tz) * ROWS), bh, idesc);
            a += row_zy;
        }
        bl += (uint32_t)(NZ * ROWS * 2);
        if (++tx == nx) { tx = 0; al += wrap; }
        else al += (uint32_t)xstep;
    }
}

template <int ROWS>
__device__ __forceinline__ void issue_nz(int nz, uint32_t on, uint32_t dt, uint32_t al, uint32_t ah, uint32_t bl, uint32_t bh, int cnt,
                                         int tx, int nx, int xstep, uint32_t wrap, uint32_t row_zy, uint32_t idesc) {
    switch (nz) {       // k and, at stride 2, (k + 1) / 2 and k / 2 for odd k <= 9
    case 1: issue<1, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    case 2: issue<2, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    case 3: issue<3, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    case 4: issue<4, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    case 5: issue<5, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    case 7: issue<7, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    default: issue<9, ROWS>(on, dt, al, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc); break;
    }
}

template <int NT, int T>
__global__ void __launch_bounds__(Roles<NT, T>::THREADS, 1) conv3d_f32tc_kernel(const __grid_constant__ CUtensorMap tmap,
                                                                                Args a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    using R = Roles<NT, T>;
    constexpr int UCOLS = R::UCOLS, COLS = R::COLS, NI = R::NI, EG = R::EG, OWN = R::OWN, EPI0 = R::EPI0;
    constexpr uint32_t TCOLS = COLS;
    static_assert(T % 2 == 0 && UCOLS <= 256 && TCOLS <= 512 && (TCOLS & (TCOLS - 1)) == 0, "accumulators fit tensor memory");
    const Geo &g = a.g;
    const uint32_t a_tx = 2u * (uint32_t)(g.hd * g.hh * g.hw) * 16u;
    unsigned char *sA = smem;
    unsigned char *sB = smem + g.na * g.a_bytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + g.nbs * g.stage_bytes);
    uint64_t *a_full = bars;                 // [2]
    uint64_t *a_empty = bars + 2;            // [2]
    uint64_t *b_full = bars + 4;             // [nbs]
    uint64_t *b_empty = b_full + g.nbs;      // [nbs]
    uint64_t *acc_full = b_empty + g.nbs;        // [T] an interval's MMAs of the slice are complete
    uint64_t *acc_empty = acc_full + T;   // [T] the epilogue has read and re-zeroed the slice
    uint64_t *mma_done = acc_empty + T;
    uint64_t *tile_full = mma_done + 1;      // [kRing]
    uint64_t *tile_empty = tile_full + kRing;
    int *tile_ring = reinterpret_cast<int *>(tile_empty + kRing);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tile_ring + kRing);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    // the shuffle tells the compiler that the warp index is uniform
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int n_tiles = g.nbx * g.nby * g.nbz * g.nblk * a.B;
    auto decode = [&](int t, int &x0, int &y0, int &z0, int &c0, int &b) {
        x0 = (t % g.nbx) * 8; t /= g.nbx;
        y0 = (t % g.nby) * 16; t /= g.nby;
        z0 = (t % g.nbz) * T; t /= g.nbz;
        c0 = (t % g.nblk) * NT;
        b = t / g.nblk;
    };

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) { tc::mbar_init(&a_full[i], 1); tc::mbar_init(&a_empty[i], NI); }
        for (int i = 0; i < g.nbs; ++i) { tc::mbar_init(&b_full[i], 1); tc::mbar_init(&b_empty[i], NI); }
        for (int i = 0; i < T; ++i) { tc::mbar_init(&acc_full[i], 1); tc::mbar_init(&acc_empty[i], 4); }
        tc::mbar_init(mma_done, NI);
        for (int i = 0; i < kRing; ++i) { tc::mbar_init(&tile_full[i], 1); tc::mbar_init(&tile_empty[i], NI + 4 * EG); }
        *abort_flag = 0;
        tc::fence_mbar_init();
    }
    if (warp == 1) tc::tmem_alloc(tmem_slot, TCOLS);
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tbase = *tmem_slot;
    if (warp >= EPI0 && warp < EPI0 + 4) {      // one warp per lane quarter zeroes the accumulators
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        for (uint32_t c = 0; c < TCOLS; c += 32u) tc::tmem_st32_zero(tbase + lane_base + c);
        tc::tmem_st_wait();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();

    auto fail = [&]() {
        *abort_flag = 1;
        atomicOr(a.err, FUSION_ERR_TIMEOUT);
    };

    int prod_ai = 0, prod_bi = 0;
    if (warp == 0 && lane == 0) {
        // ---------------- producer ----------------
        int &ai = prod_ai, &bi = prod_bi;
        int tile = blockIdx.x;
        for (int it = 0;; ++it) {
            const uint64_t deadline = tc::globaltimer() + kWaitNs;
            const int slot = it % kRing;
            if (!tc::mbar_wait(&tile_empty[slot], ((it / kRing) & 1) ^ 1, deadline, a.err, FUSION_ERR_TIMEOUT)) { fail(); break; }
            const bool done = tile >= n_tiles || *abort_flag;
            tile_ring[slot] = done ? -1 : tile;
            tc::mbar_arrive(&tile_full[slot]);
            if (done || a.stall) break;
            int x0, y0, z0, c0, b;
            decode(tile, x0, y0, z0, c0, b);
            size_t woff = (size_t)(c0 / NT) * a.wblk;   // stored channel block, chunk, phase, (ty, tx) group
            for (int c = 0; c < g.chunks && !*abort_flag; ++c) {
                for (int ph = 0; ph < g.nphase && !*abort_flag; ++ph) {
                    const int ngr = phase_groups(a, c, ph);
                    if (!ngr) continue;
                    int pz, py, px, nz, ny, nx;
                    phase_taps(a, ph, pz, py, px, nz, ny, nx);
                    // pass 0: x_lo with w_hi; pass 1: x_hi with [w_hi | w_lo]
                    bool ok = true;
                    for (int pass = 0; pass < 2 && ok; ++pass) {
                        const int buf = ai % g.na;
                        ok = tc::mbar_wait(&a_empty[buf], ((ai / g.na) & 1) ^ 1, deadline, a.err, FUSION_ERR_TIMEOUT);
                        if (!ok) { fail(); break; }
                        tc::mbar_expect_tx(&a_full[buf], a_tx);
                        unsigned char *dst = sA + buf * g.a_bytes;
                        const int bb = (pass == 0 ? a.max_poses : 0) + b;      // the low parts follow the high ones
                        const int S = a.stride;
                        if (a.blocked == 2) {
                            const int qx = px - a.pad, qy = py - a.pad, qz = pz - a.pad;
                            tc::tma_load_5d(dst, &tmap, &a_full[buf], (x0 + (qx >> 1)) * 8, 2 * c, y0 + (qy >> 1),
                                            z0 + (qz >> 1), bb * 8 + (qz & 1) * 4 + (qy & 1) * 2 + (qx & 1));
                        } else if (a.blocked) {
                            tc::tma_load_5d(dst, &tmap, &a_full[buf], (x0 - a.pad) * 8, 2 * c, y0 - a.pad, z0 - a.pad, bb);
                        } else {
                            for (int j = 0; j < 2; ++j)
                                tc::tma_load_5d(dst + j * g.plane_bytes, &tmap, &a_full[buf], c * 16 + j * 8,
                                                x0 * S + px - a.pad, y0 * S + py - a.pad, z0 * S + pz - a.pad, bb);
                        }
                        ++ai;
                        const uint32_t gbytes = (uint32_t)nz * NT * 32 * (pass + 1);
                        const uint8_t *wp = a.w[pass] + woff * (pass + 1);
                        for (int g0 = 0; g0 < ngr; g0 += g.gps[pass]) {
                            const int cnt = min(g.gps[pass], ngr - g0);
                            const int st = bi % g.nbs;
                            ok = tc::mbar_wait(&b_empty[st], ((bi / g.nbs) & 1) ^ 1, deadline, a.err, FUSION_ERR_TIMEOUT);
                            if (!ok) { fail(); break; }
                            const uint32_t bytes = (uint32_t)cnt * gbytes;
                            tc::mbar_expect_tx(&b_full[st], bytes);
                            tc::bulk_load(sB + st * g.stage_bytes, wp + (size_t)g0 * gbytes, bytes, &b_full[st]);
                            ++bi;
                        }
                    }
                    woff += (size_t)ngr * nz * NT * 32;
                }
            }
            tile = atomicAdd(a.tile_counter, 1) + (int)gridDim.x;
        }
    } else if (warp >= 1 && warp <= NI) {
        // ---------------- MMA issuer of slices w0, w0 + NI, .. ----------------
        // All lanes run the loops (the MMAs' operands are then in uniform registers); one issues.
        const int w0 = warp - 1;
        const uint32_t on = tc::elect_one();
        auto wait_all = [&](uint64_t *bar, uint32_t parity, uint64_t deadline) {
            return __all_sync(0xffffffffu, tc::mbar_wait(bar, parity, deadline, a.err, FUSION_ERR_TIMEOUT)) != 0;
        };
        int ai = 0;                        // halo buffers so far
        int st = 0;                        // weight stage in turn and its parity; parity of the interval
        uint32_t b_par = 0, acc_par = 0;
        const uint32_t sbo_a = (uint32_t)g.ystep * 16;
        const uint32_t row_zy = (uint32_t)g.hh * g.ystep;
        for (int it = 0;; ++it) {
            const uint64_t deadline = tc::globaltimer() + kWaitNs;
            const int slot = it % kRing;
            if (!wait_all(&tile_full[slot], (it / kRing) & 1, deadline)) { fail(); break; }
            const bool done = __any_sync(0xffffffffu, tile_ring[slot] < 0 || *abort_flag != 0);   // every lane has read the slot
            if (on) tc::mbar_arrive(&tile_empty[slot]);
            if (done) break;
            bool ok = true;
            for (int c = 0; c < g.chunks && ok; ++c) {
                for (int ph = 0; ph < g.nphase && ok; ++ph) {
                    const int ngr = phase_groups(a, c, ph);
                    if (!ngr) continue;
                    int pz, py, px, nz, ny, nx;
                    phase_taps(a, ph, pz, py, px, nz, ny, nx);
                    int xstep = 1, xstart = 0;
                    if (a.xpat) {
                        nx = a.xt_n[c];
                        xstep = a.xt_step[c];
                        xstart = a.xt_start[c];
                    }
                    bool fresh = true;         // the next block of MMAs starts an interval
                    for (int pass = 0; pass < 2 && ok; ++pass) {
                        const int buf = ai % g.na;
                        ok = wait_all(&a_full[buf], (ai / g.na) & 1, deadline);
                        if (!ok) { fail(); break; }
                        ++ai;
                        const uint64_t adesc0 = tc::desc_kmajor(tc::smem_u32(sA + buf * g.a_bytes), g.lbo_a, sbo_a);
                        const int rows = NT * (pass + 1);                      // B rows per kernel offset
                        const uint32_t idesc = tc::idesc_f16(128, NT) + (pass ? (uint32_t)(NT >> 3) << 17 : 0u);
                        const uint32_t lbo_b = (uint32_t)(nz * rows * 16);     // between the two 8-channel halves
                        const uint32_t wrap = (uint32_t)(g.ystep - xstep * (nx - 1));
                        // counters instead of divisions: a block's scalar work stands between its MMAs and the last block's
                        const int gps = g.gps[pass];
                        int tx = 0, left = g.flush_groups;                     // column of the next group; groups left in the interval
                        uint32_t at = (uint32_t)adesc0 + (uint32_t)xstart;     // its A address
                        const uint32_t ah = (uint32_t)(adesc0 >> 32);
                        for (int g0 = 0; g0 < ngr && ok; g0 += gps) {
                            ok = wait_all(&b_full[st], b_par, deadline);
                            if (!ok) { fail(); break; }
                            tc::tc_fence_after();
                            const uint64_t bdesc = tc::desc_kmajor(tc::smem_u32(sB + st * g.stage_bytes), lbo_b, 128);
                            const uint32_t bh = (uint32_t)(bdesc >> 32);
                            uint32_t bl = (uint32_t)bdesc;
                            // blocks of groups end where the stage does and, for x_hi, where an interval does
                            for (int todo = min(gps, ngr - g0), gdone = g0; todo > 0 && ok;) {
                                const int cnt = pass ? min(todo, left) : todo;
                                todo -= cnt;
                                gdone += cnt;
                                if (pass) left -= cnt;
                                const bool close = pass && (left == 0 || gdone == ngr);
                                for (int s = w0; s < T; s += NI) {
                                    if (fresh) {
                                        ok = wait_all(&acc_empty[s], acc_par ^ 1, deadline);
                                        if (!ok) { fail(); break; }
                                        tc::tc_fence_after();
                                    }
                                    // x_hi: columns [0, 2 NT) of the slice; x_lo w_hi joins the small products in [NT, 2 NT)
                                    const uint32_t dt = tbase + (uint32_t)(s * UCOLS);
                                    const uint32_t as = at + (uint32_t)(s * row_zy);
                                    if (pass) issue_nz<2 * NT>(nz, on, dt, as, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc);
                                    else issue_nz<NT>(nz, on, dt + NT, as, ah, bl, bh, cnt, tx, nx, xstep, wrap, row_zy, idesc);
                                    if (close && on) tc::mma_commit(&acc_full[s]);
                                }
                                bl += (uint32_t)(cnt * nz * rows * 2);
                                for (int i = 0; i < cnt; ++i) {
                                    if (++tx == nx) { tx = 0; at += wrap; }
                                    else at += (uint32_t)xstep;
                                }
                                fresh = close;
                                if (close) {
                                    left = g.flush_groups;
                                    acc_par ^= 1;
                                }
                            }
                            if (!ok) break;
                            if (on) tc::mma_commit(&b_empty[st]);
                            if (++st == g.nbs) { st = 0; b_par ^= 1; }
                        }
                        if (ok && on) tc::mma_commit(&a_empty[buf]);
                    }
                }
            }
            if (!ok) break;
        }
        if (on) tc::mma_commit(mma_done);
    } else if (warp >= EPI0) {
        // ---------------- epilogue: EG groups of one warp per lane quarter ----------------
        const int q = warp & 3;
        const int e0 = (warp - EPI0) >> 2;      // totals slices e0, e0 + EG, ..
        const int r = q * 32 + lane;            // M row = voxel of the slice
        const int h = r >> 3, w = r & 7;
        const uint32_t tsub = tbase + ((uint32_t)(q * 32) << 16);
        int iv = 0;
        int per_tile = 0;                       // intervals per tile
        for (int c = 0; c < g.chunks; ++c)
            for (int ph = 0; ph < g.nphase; ++ph) per_tile += (phase_groups(a, c, ph) + g.flush_groups - 1) / g.flush_groups;
        for (int it = 0;; ++it) {
            const uint64_t deadline = tc::globaltimer() + kWaitNs;
            const int slot = it % kRing;
            int tile = -1;
            if (lane == 0) {
                if (tc::mbar_wait(&tile_full[slot], (it / kRing) & 1, deadline, a.err, FUSION_ERR_TIMEOUT)) {
                    tile = tile_ring[slot];
                    tc::mbar_arrive(&tile_empty[slot]);
                } else {
                    fail();
                }
            }
            tile = __shfl_sync(0xffffffffu, tile, 0);
            if (tile < 0 || __any_sync(0xffffffffu, *abort_flag != 0)) break;
            float tot[OWN][NT];
#pragma unroll
            for (int o = 0; o < OWN; ++o)
#pragma unroll
                for (int j = 0; j < NT; ++j) tot[o][j] = 0.f;
            bool ok = true;
            for (int i = 0; i < per_tile && ok; ++i, ++iv) {
#pragma unroll
                for (int o = 0; o < OWN; ++o) {
                    const int s = e0 + EG * o;
                    // tensor-memory loads must be executed by all 32 lanes or by none
                    ok = ok && tc::mbar_wait(&acc_full[s], iv & 1, deadline, a.err, FUSION_ERR_TIMEOUT);
                    ok = __all_sync(0xffffffffu, ok) && !__any_sync(0xffffffffu, *abort_flag != 0);
                    if (ok) {
                        tc::tc_fence_after();
                        const uint32_t tu = tsub + (uint32_t)(s * UCOLS);
                        // 16 columns at a time: 32 more registers beside the totals would spill
                        auto add16 = [&](int col, int c16, bool finite_only) {
                            uint32_t v[16];
                            tc::tmem_ld16(tu + (uint32_t)(col + c16), v);
                            tc::tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 16; ++j) {
                                const float t = __uint_as_float(v[j]);
                                if (!finite_only || fabsf(t) < INFINITY) tot[o][c16 + j] += t;
                            }
                        };
                        auto zero = [&](int col) {
#pragma unroll
                            for (int c32 = 0; c32 < NT; c32 += 32) tc::tmem_st32_zero(tu + (uint32_t)(col + c32));
                        };
                        if (i == per_tile - 1) {      // the tile's small products are complete
#pragma unroll
                            for (int c16 = 0; c16 < NT; c16 += 16) add16(NT, c16, true);
                            zero(NT);
                        }
#pragma unroll
                        for (int c16 = 0; c16 < NT; c16 += 16) add16(0, c16, false);
                        zero(0);
                        tc::tmem_st_wait();
                        tc::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(&acc_empty[s]);
                    }
                }
            }
            if (!ok) { if (lane == 0) fail(); break; }
            int x0, y0, z0, c0, b;
            decode(tile, x0, y0, z0, c0, b);
            const int n = a.n_out, yy = y0 + h, xx = x0 + w;
            // 1 / s_x, a power of two as 1 / s_w is: before 1 / s_w where it is below 1 and after it elsewhere, so that no step
            // overflows, or goes below the normal range, where the result does not
            const float isx = a.inv_sx[b], sx_lo = fminf(isx, 1.f), sx_hi = fmaxf(isx, 1.f);
            float vmax = 0.f;
#pragma unroll
            for (int o = 0; o < OWN; ++o) {
                const int zz = z0 + e0 + EG * o;
                if (zz >= n || yy >= n || xx >= n) continue;
                const size_t at = ((((size_t)b * n + zz) * n + yy) * n + xx) * a.c_out + c0;
#pragma unroll
                for (int j4 = 0; j4 < NT / 4; ++j4) {
                    const float4 sw = __ldg(reinterpret_cast<const float4 *>(a.inv_sw + c0) + j4);
                    const float4 bs = __ldg(reinterpret_cast<const float4 *>(a.bias + c0) + j4);
                    const float *t = tot[o] + j4 * 4;
                    float4 v;
                    v.x = fmaxf(t[0] * sx_lo * sw.x * sx_hi + bs.x, 0.f);
                    v.y = fmaxf(t[1] * sx_lo * sw.y * sx_hi + bs.y, 0.f);
                    v.z = fmaxf(t[2] * sx_lo * sw.z * sx_hi + bs.z, 0.f);
                    v.w = fmaxf(t[3] * sx_lo * sw.w * sx_hi + bs.w, 0.f);
                    if (a.residual) {
                        const float4 x4 = __ldg(reinterpret_cast<const float4 *>(a.xres + at) + j4);
                        v.x += x4.x; v.y += x4.y; v.z += x4.z; v.w += x4.w;
                    }
                    vmax = fmaxf(vmax, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
                    reinterpret_cast<float4 *>(a.y + at)[j4] = v;
                }
            }
            if (a.amax) {
                if (vmax == INFINITY) {         // rare: the finite ones, from what this thread just stored
                    vmax = 0.f;
                    for (int o = 0; o < OWN; ++o) {
                        const int zz = z0 + e0 + EG * o;
                        if (zz >= n || yy >= n || xx >= n) continue;
                        const float *own = a.y + ((((size_t)b * n + zz) * n + yy) * n + xx) * a.c_out + c0;
                        for (int j = 0; j < NT; ++j) vmax = fmaxf(vmax, finite_abs(own[j]));
                    }
                }
                for (int o = 16; o > 0; o >>= 1) vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
                if (lane == 0 && vmax > 0.f) atomicMax(reinterpret_cast<unsigned *>(a.amax + b), __float_as_uint(vmax));
            }
        }
    }
    // every MMA must be complete before tensor memory is freed
    if (warp == 1) {
        if (lane == 0 && !tc::mbar_wait(mma_done, 0, tc::globaltimer() + kWaitNs)) fail();
        __syncwarp();
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0 && lane == 0) {
        // no copy issued by this CTA may still be landing in its shared memory
        const uint64_t dl = tc::globaltimer() + 100000000ull;
        for (int i = 0; i < g.na; ++i) {
            const int c = prod_ai > i ? (prod_ai - i + g.na - 1) / g.na : 0;
            if (c > 0 && !tc::mbar_wait(&a_full[i], (c - 1) & 1, dl)) atomicOr(a.err, FUSION_ERR_TIMEOUT);
        }
        for (int i = 0; i < g.nbs; ++i) {
            const int c = prod_bi > i ? (prod_bi - i + g.nbs - 1) / g.nbs : 0;
            if (c > 0 && !tc::mbar_wait(&b_full[i], (c - 1) & 1, dl)) atomicOr(a.err, FUSION_ERR_TIMEOUT);
        }
    }
    __syncthreads();
    if (warp == 1) tc::tmem_dealloc(tbase, TCOLS);
    // the last CTA to end resets the counters for the next launch
    if (tid == 0) {
        __threadfence();
        if (atomicInc(reinterpret_cast<unsigned *>(a.tile_counter + 1), gridDim.x - 1) == gridDim.x - 1) a.tile_counter[0] = 0;
    }
}

// ---- the two FP16 parts of a map -------------------------------------------

__device__ __forceinline__ float pow2(int e) { return __int_as_float((e + 127) << 23); }   // -126 <= e <= 127

// Exponent e of the pose's scale 2^e: the largest |x| lands in [2^14, 2^15) (a map of zeros: 0).
__device__ __forceinline__ int scale_exp(float am) {
    if (!(am > 0.f)) return 0;
    const int e = (int)((__float_as_uint(am) >> 23) & 0xFF) - 127;
    return min(14 - min(e, 127), 126);
}

__device__ __forceinline__ void split2(float x, float s, __half &hi, __half &lo) {
    const float t = x * s;                              // exact: s is a power of two
    hi = __float2half_rn(t);
    const float f = __half2float(hi);
    lo = isinf(f) || isnan(f) ? __float2half_rn(0.f) : __float2half_rn(t - f);
}

// One item: 8 channels (16 bytes of each part) of a voxel.  Channel block cb varies fastest across threads, so
// the reads are contiguous.  Bound by memory (4 bytes read and 4 written per element).
// Poses last to first, as the FP8 quantizers take them (the last ones are still in L2).
__global__ void __launch_bounds__(256) split_f16_kernel(SplitF16Args a) {
    const int b = gridDim.y - 1 - blockIdx.y;
    const int e = scale_exp(a.amax[b]);
    const float s = pow2(e);
    if (blockIdx.x == 0 && threadIdx.x == 0) a.inv_sx[b] = pow2(-e);
    const int n = a.n, nb = a.cp / 8;
    const size_t nv = (size_t)n * n * n, items = nv * nb;
    const float *xb = a.x + (size_t)b * nv * a.c;
    const size_t per_pose = nv * a.cp;
    __half *hi = a.out + (size_t)b * per_pose, *lo = hi + (size_t)a.max_poses * per_pose;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < items; i += (size_t)gridDim.x * blockDim.x) {
        const size_t v = i / nb;
        const int cb = (int)(i - v * nb);
        const size_t row = v / n;                  // (z, y)
        const int x = (int)(v - row * n);
        float f[8];
        if (a.fold_pad >= 0 && cb >= 2) {
            // x-folded second chunk: slot 3 s + c = channel 16 + c of voxel x - p + s, s < k (slot 15 unused)
            const int used = 3 * min(5, 2 * a.fold_pad + 1);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int sl = (cb - 2) * 8 + j, xs = x - a.fold_pad + sl / 3;
                f[j] = sl < used && xs >= 0 && xs < n ? xb[(row * n + xs) * a.c + 16 + sl % 3] : 0.f;
            }
        } else if (cb * 8 < a.c) {
            const float4 *src = reinterpret_cast<const float4 *>(xb + v * a.c + cb * 8);   // c is a multiple of 8
            const float4 p = src[0], q = src[1];
            f[0] = p.x; f[1] = p.y; f[2] = p.z; f[3] = p.w;
            f[4] = q.x; f[5] = q.y; f[6] = q.z; f[7] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) f[j] = 0.f;
        }
        __align__(16) __half h8[8], l8[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) split2(f[j], s, h8[j], l8[j]);
        size_t dst;
        if (a.layout == 2) {
            const size_t hn = (size_t)(n >> 1);
            const int yy = (int)(row % n), zz = (int)(row / n);
            const size_t p = (size_t)(zz & 1) * 4 + (yy & 1) * 2 + (x & 1);
            dst = ((((p * hn + (zz >> 1)) * hn + (yy >> 1)) * nb + cb) * hn + (x >> 1)) * 8;
        } else if (a.layout == 1) {
            dst = ((row * nb + cb) * n + x) * 8;
        } else {
            dst = v * a.cp + cb * 8;
        }
        *reinterpret_cast<uint4 *>(hi + dst) = *reinterpret_cast<const uint4 *>(h8);
        *reinterpret_cast<uint4 *>(lo + dst) = *reinterpret_cast<const uint4 *>(l8);
    }
}

__global__ void __launch_bounds__(256) amax_f32_kernel(const float *x, size_t per_pose, float *amax) {
    const int b = blockIdx.y;
    const float4 *src = reinterpret_cast<const float4 *>(x + (size_t)b * per_pose);
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < per_pose / 4; i += (size_t)gridDim.x * blockDim.x) {
        const float4 v = src[i];
        m = fmaxf(m, fmaxf(fmaxf(finite_abs(v.x), finite_abs(v.y)), fmaxf(finite_abs(v.z), finite_abs(v.w))));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(reinterpret_cast<unsigned *>(amax + b), __float_as_uint(m));
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        return static_cast<PFN_cuTensorMapEncodeTiled_v12000>(nullptr);
    }();
    return fn;
}

constexpr int kMaxVariants = 4;

}  // namespace

struct ConvF32TcPlan::Impl {
    struct Variant {
        CUtensorMap tmap;
        Geo g;
        int T;
        size_t smem;
        double tile_cost;       // clocks of a tile's MMAs per kernel offset and chunk, for choosing T
    } var[kMaxVariants];
    int n_var = 0;
    Args args{};
    int NT = 0, sms = 1;
    int *counter = nullptr;
    ~Impl() { if (counter) cudaFree(counter); }
};

ConvF32TcPlan::ConvF32TcPlan() : impl(new Impl()) {}
ConvF32TcPlan::~ConvF32TcPlan() { delete impl; }

int conv_f32tc_plan(ConvF32TcPlan &plan, const ConvF32TcSpec &sp, char *why, size_t why_len) {
    ConvF32TcPlan::Impl &P = *plan.impl;
    const int k = sp.k, stride = sp.stride, NT = conv_f32tc_block(sp.c_out);
    if (!NT) {
        snprintf(why, why_len, "c_out must be a multiple of 32");
        return -1;
    }
    if (sp.cin_pad % 16 != 0 || (stride != 1 && stride != 2) || (sp.blocked == 1 && stride != 1) ||
        (sp.blocked == 2 && (stride != 2 || sp.n_in % 2 != 0)) || (sp.fold && (sp.cin_pad != 32 || sp.blocked != 1))) {
        snprintf(why, why_len, "unsupported layout");
        return -1;
    }
    auto enc = get_encode();
    int dev = 0, sms = 0;
    if (!enc || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
        snprintf(why, why_len, "no TMA encoder or device");
        return -2;
    }
    P.sms = sms;
    P.NT = NT;
    P.n_var = 0;
    Args &A = P.args;
    A.w[0] = static_cast<const uint8_t *>(sp.w_hi);
    A.w[1] = static_cast<const uint8_t *>(sp.w_both);
    A.wblk = conv_tc_weight_bytes(sp.cin_pad, NT, k, stride, 2, sp.fold);
    A.c_out = sp.c_out;
    A.inv_sw = sp.inv_sw;
    A.inv_sx = sp.inv_sx;
    A.bias = sp.bias;
    A.xres = sp.xres;
    A.y = sp.y;
    A.n_out = sp.n_out;
    A.k = k;
    A.stride = stride;
    A.pad = k / 2;
    A.residual = sp.residual;
    A.max_poses = sp.max_poses;
    A.xpat = sp.fold ? 1 : 0;
    if (sp.fold) conv_tc_fold_pattern(1, k, A.xt_n, A.xt_step, A.xt_start);
    A.blocked = sp.blocked;
    A.err = sp.err;
    // T slices x 2 NT <= 512 columns, and smaller tiles for batches that would leave most SMs idle
    for (int T = 256 / NT; T >= 2 && P.n_var < kMaxVariants; T /= 2) {
        Geo g{};
        g.nbx = (sp.n_out + 7) / 8;
        g.nby = (sp.n_out + 15) / 16;
        g.nbz = (sp.n_out + T - 1) / T;
        g.nphase = stride == 1 ? 1 : 8;
        g.ntap[0] = stride == 1 ? k : (k + 1) / 2;
        g.ntap[1] = stride == 1 ? k : k / 2;
        const int nt = g.ntap[0];
        g.hd = T + nt - 1;
        g.hh = 16 + nt - 1;
        g.hw = 8 + nt - 1;
        const uint32_t vox = (uint32_t)(g.hd * g.hh * g.hw);
        g.plane_bytes = (vox * 16 + 127) / 128 * 128;
        if (sp.blocked) {
            g.a_bytes = (vox * 32 + 127) / 128 * 128;
            g.lbo_a = (uint32_t)g.hw * 16;
            g.ystep = 2 * g.hw;
        } else {
            g.a_bytes = 2 * g.plane_bytes;
            g.lbo_a = g.plane_bytes;
            g.ystep = g.hw;
        }
        if (g.hw * stride > 256 || g.hh * stride > 256 || g.hd * stride > 256 || (sp.blocked && g.hw * 8 > 256)) continue;
        g.flush_groups = std::max(1, kFlushTaps / nt);     // a function of the layer only: results do not depend on T
        g.chunks = sp.cin_pad / 16;
        g.nblk = sp.c_out / NT;
        g.nbs = 2;
        const uint32_t gbytes = (uint32_t)nt * NT * 32;            // a group of the x_lo product; twice that for x_hi
        const size_t bar_bytes = (size_t)(4 + 2 * g.nbs + 2 * T + 1 + 2 * kRing) * 8 + kRing * 4 + 16, limit = 227 * 1024;
        // about 57 KB of weights per stage (2 groups of x_hi in the 64-channel 7^3 layers), less where the halo
        // leaves no room
        g.gps[1] = std::min(nt * nt, std::max(1, (int)(57344u / (2 * gbytes))));
        auto bytes = [&](int na) {
            g.gps[0] = std::min(nt * nt, 2 * g.gps[1]);
            g.stage_bytes = ((uint32_t)g.gps[1] * 2 * gbytes + 127) / 128 * 128;
            return na * (size_t)g.a_bytes + (size_t)g.nbs * g.stage_bytes + bar_bytes;
        };
        while (g.gps[1] > 1 && bytes(1) > limit) --g.gps[1];
        if (bytes(1) > limit) continue;
        g.na = bytes(2) <= limit ? 2 : 1;
        ConvF32TcPlan::Impl::Variant &V = P.var[P.n_var];
        V.smem = bytes(g.na);
        V.g = g;
        V.T = T;
        // clocks of a slice's two MMAs per kernel offset: operand reads (4 KB + 32 bytes per row at 128 a clock) or math
        auto mma = [](int n) { return std::max(n * 0.5, (4096 + 32 * n) / 128.0); };
        // a tile costs its slices' MMAs plus about 0.4 of a slice for halo loads and hand-offs
        V.tile_cost = (T + 0.4) * (mma(NT) + mma(2 * NT));
        const cuuint64_t n = (cuuint64_t)sp.n_in, rowb = (cuuint64_t)sp.cin_pad * 2;
        cuuint64_t dims[5] = {(cuuint64_t)sp.cin_pad, n, n, n, 2 * (cuuint64_t)sp.max_poses};
        cuuint64_t strides[4] = {rowb, rowb * n, rowb * n * n, rowb * n * n * n};
        cuuint32_t box[5] = {8, (cuuint32_t)(g.hw * stride), (cuuint32_t)(g.hh * stride), (cuuint32_t)(g.hd * stride), 1};
        cuuint32_t estr[5] = {1, (cuuint32_t)stride, (cuuint32_t)stride, (cuuint32_t)stride, 1};
        if (sp.blocked) {
            const cuuint64_t blocks = (cuuint64_t)sp.cin_pad / 8, h = sp.blocked == 2 ? n / 2 : n;
            dims[0] = h * 8; dims[1] = blocks; dims[2] = h; dims[3] = h;
            dims[4] = 2 * (cuuint64_t)sp.max_poses * (sp.blocked == 2 ? 8 : 1);
            strides[0] = h * 16; strides[1] = blocks * h * 16; strides[2] = strides[1] * h; strides[3] = strides[2] * h;
            box[0] = (cuuint32_t)(g.hw * 8); box[1] = 2; box[2] = (cuuint32_t)g.hh; box[3] = (cuuint32_t)g.hd;
            for (int i = 0; i < 5; ++i) estr[i] = 1;
        }
        const CUresult r = enc(&V.tmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 5, const_cast<void *>(sp.x), dims, strides, box,
                               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            snprintf(why, why_len, "cuTensorMapEncodeTiled failed (%d)", (int)r);
            return -2;
        }
        ++P.n_var;
    }
    if (!P.n_var) {
        snprintf(why, why_len, "no tile fits shared memory");
        return -1;
    }
    if (!P.counter && (cudaMalloc(&P.counter, 2 * sizeof(int)) != cudaSuccess ||
                       cudaMemset(P.counter, 0, 2 * sizeof(int)) != cudaSuccess)) {
        cudaGetLastError();
        snprintf(why, why_len, "cannot allocate the tile counter");
        return -2;
    }
    A.tile_counter = P.counter;
    return 0;
}

int conv_f32tc_block(int c_out) { return c_out % 128 == 0 ? 128 : c_out % 64 == 0 ? 64 : c_out % 32 == 0 ? 32 : 0; }

template <int NT, int T>
static void launch_t(const ConvF32TcPlan::Impl &P, const ConvF32TcPlan::Impl::Variant &V, const Args &a, cudaStream_t s) {
    cudaFuncSetAttribute(conv3d_f32tc_kernel<NT, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)V.smem);
    const unsigned tiles = (unsigned)(V.g.nbx * V.g.nby * V.g.nbz * V.g.nblk) * (unsigned)a.B;
    const unsigned grid = std::min(tiles, (unsigned)P.sms);
    conv3d_f32tc_kernel<NT, T><<<grid, Roles<NT, T>::THREADS, V.smem, s>>>(V.tmap, a);
}

void conv_f32tc_stall_next(ConvF32TcPlan &plan) { plan.impl->args.stall = 1; }

ConvTile conv_f32tc_launch(ConvF32TcPlan &plan, int p0, int B, float *amax, cudaStream_t s) {
    ConvF32TcPlan::Impl &P = *plan.impl;
    // the tile with the shortest schedule: rounds of tiles over the SMs x a tile's MMA clocks
    int best = 0;
    double best_t = 1e300;
    for (int i = 0; i < P.n_var; ++i) {
        const Geo &g = P.var[i].g;
        const long long tiles = (long long)g.nbx * g.nby * g.nbz * g.nblk * B;
        const double t = (double)((tiles + P.sms - 1) / P.sms) * P.var[i].tile_cost;
        if (t < best_t) { best_t = t; best = i; }
    }
    const ConvF32TcPlan::Impl::Variant &V = P.var[best];
    Args a = P.args;
    a.g = V.g;
    a.B = B;
    a.amax = amax;
    // an output map has n_out^3 c_out floats, and so has a residual source (stride 1, c_in = c_out)
    const size_t maps = (size_t)p0 * a.n_out * a.n_out * a.n_out * a.c_out;
    a.inv_sx += p0;
    a.y += maps;
    if (a.residual) a.xres += maps;
    P.args.stall = 0;      // one launch only
    switch (P.NT * 16 + V.T) {
    case 32 * 16 + 8: launch_t<32, 8>(P, V, a, s); break;
    case 32 * 16 + 4: launch_t<32, 4>(P, V, a, s); break;
    case 32 * 16 + 2: launch_t<32, 2>(P, V, a, s); break;
    case 64 * 16 + 4: launch_t<64, 4>(P, V, a, s); break;
    case 64 * 16 + 2: launch_t<64, 2>(P, V, a, s); break;
    default: launch_t<128, 2>(P, V, a, s); break;
    }
    return {V.T, 1, 0, P.NT};
}

void launch_split_f16(const SplitF16Args &a, int B, cudaStream_t s) {
    const size_t items = (size_t)a.n * a.n * a.n * (a.cp / 8);
    const unsigned gx = (unsigned)std::min<size_t>((items + 255) / 256, 256);
    split_f16_kernel<<<dim3(gx, B), 256, 0, s>>>(a);
}

void launch_amax_f32(const float *x, int B, size_t per_pose, float *amax, cudaStream_t s) {
    const unsigned gx = (unsigned)std::max<size_t>(1, std::min<size_t>((per_pose / 4 + 255) / 256, 128));
    amax_f32_kernel<<<dim3(gx, B), 256, 0, s>>>(x, per_pose, amax);
}

}  // namespace fusion
