// fc_qvec.cu -- q_g = s~_g^T A s~_g for every grid point on the tensor cores.
//
// The screen (fc_screen.cu) needs, per inverse covariance A = M^-1, the
// vector q_g of Eq. 1 expanded around the centre v (s~_g = s_g - v).  With
// A = W^T W (W = L^-1, lower triangular, from the Cholesky factor of M),
//
//     q_g = || W s~_g ||^2 ,
//
// so q is the row-wise squared norm of the G x K x K product T = S~ W^T.  One
// CTA tile is 128 grid points; the tile's S~ rows (the screen's own B image,
// bf16 hi + lo) and the W image (bf16 hi + lo) meet on tcgen05 as
// hi*hi + lo*hi + hi*lo with binary32 accumulation in TMEM, and the epilogue
// squares and sums each row.  Every term left out is bounded from the
// realized norms of the split parts:
//
//     T - T^ = W_lo S_lo + r_W s~ + (W_hi + W_lo) r_S + accumulation error
//     ||T - T^||_2 <= E_g = |W_lo|_F |S_lo| + |r_W|_F |s~| + |W_hl|_F |r_S|
//                          + (3K+2) 1.02 2^-23 |W|_F |s~|
//
// so q_g lies in [(|T^| - E_g)^2, (|T^| + E_g)^2] with |T^| from the binary32
// sum of squares (relative error <= (K+2) 2^-24).  The stored pair is
// Qc = that sum and Qb = Qc - delta - q_rel_slack |Qc|, delta the larger
// distance to either end, so q >= Qb and q <= Qc + (Qc - Qb) as the screen
// and the probes require.
//
// Roles (one CTA per SM, persistent over (slot group, 128-point tile) items):
//   warps 0, 10..12  bulk-async copies: the group's W images when the group
//               changes (warp 0), then the S~ rows of each tile into a stage
//               ring, the producers taking the stages in turn
//   warp 1      TMEM allocation; one lane issues tcgen05.mma
//   warps 2..9  epilogue, two per TMEM lane quadrant: tcgen05.ld of the row,
//               sum of squares, certified bound, Qc / Qb / Qb3 stores
// Waits are bounded as in the screen (kDevTimeout, abort flag, TMEM freed).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <float.h>

#include <cstdint>

#include "fc_internal.cuh"
#include "fc_tc.cuh"

namespace fcdev {
namespace {

using namespace tc;

constexpr int kQM = 128;                 // grid points per tile (TMEM lanes)
constexpr uint32_t kQSlab = kQM * 16u;   // one 8-column slab of a tile's S~ rows
constexpr int kQTmemCols = 512;          // two accumulators of up to 256 columns
constexpr uint32_t kQSmemMax = 232448u;

__device__ __forceinline__ int64_t wimg_offset(int i, int c, int K) {
    // [2K/8 slabs][K rows][8 cols] bf16, hi columns 0..K-1, lo columns K..2K-1
    return (int64_t)(c >> 3) * (K * 8) + (i >> 3) * 64 + (i & 7) * 8 + (c & 7);
}

// W image of a slot: W = W_hi + W_lo + r_W split of the binary64 factor, and
// the Frobenius norms (rounded up) of W, W_lo, r_W and W_hi + W_lo.
__global__ void __launch_bounds__(256) k_wimage(const double* __restrict__ W64, const int32_t* __restrict__ slots,
                                                int nfit, int K, uint16_t* __restrict__ Wimg,
                                                float4* __restrict__ wnorm) {
    const int slot = slots[blockIdx.x];
    const double* W = W64 + (size_t)slot * nfit * nfit;
    uint16_t* img = Wimg + (size_t)slot * 2 * K * K;
    double sw = 0.0, sl = 0.0, sr = 0.0, sh = 0.0;
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
        const int i = e / K, j = e % K;
        const double w = (i < nfit && j < nfit) ? W[i * nfit + j] : 0.0;
        const __nv_bfloat16 h = __double2bfloat16(w);
        const double rem = w - (double)__bfloat162float(h);
        const __nv_bfloat16 l = __double2bfloat16(rem);
        const double lo = (double)__bfloat162float(l);
        const double hl = (double)__bfloat162float(h) + lo;
        const double r = rem - lo;
        sw = fma(w, w, sw);
        sl = fma(lo, lo, sl);
        sr = fma(r, r, sr);
        sh = fma(hl, hl, sh);
        img[wimg_offset(i, j, K)] = __bfloat16_as_ushort(h);
        img[wimg_offset(i, K + j, K)] = __bfloat16_as_ushort(l);
    }
    __shared__ double red[4][8];
    for (int o = 16; o > 0; o >>= 1) {
        sw += __shfl_xor_sync(0xffffffffu, sw, o);
        sl += __shfl_xor_sync(0xffffffffu, sl, o);
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        sh += __shfl_xor_sync(0xffffffffu, sh, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        red[0][warp] = sw;
        red[1][warp] = sl;
        red[2][warp] = sr;
        red[3][warp] = sh;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        for (int k = 0; k < 4; ++k)
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t[k] += red[k][w];
        auto up = [](double x) { return __double2float_ru(__dsqrt_ru(x) * (1.0 + 1e-12)); };
        wnorm[slot] = make_float4(up(t[0]), up(t[1]), up(t[2]), up(t[3]));
    }
}

// A group of up to m = 256 / K slots shares each S~ tile: their W images sit
// side by side as one B operand of N = m K columns, so one MMA chain gives the
// T tiles of every slot in the group and the tile is read once per group.
// W is lower triangular, so K step kk (16 columns of W) meets only the rows
// from 16 kk on.  The slots are interleaved in blocks of 16 rows (block b of
// slot i at rows (b m + i) 16), which makes those rows one contiguous range:
// the step's MMA takes N = m (K - 16 kk) columns from accumulator column
// 16 kk m on, a bit over half the products of the full square (K = 128: 9/16).
// What bounds it then is the issue of MMAs and copies (see the whole-warp roles
// in fc_tc.cuh) and the round trip of a stage, so the ring is as deep as shared
// memory allows and a stage holds kPer = 2 K steps (128 points of 64^3, K = 128,
// the covariance stage with its factorisations: 233 ms with full squares issued
// from one lane, 176 ms with triangles issued by whole warps, 163 ms with the
// packed images and two steps a stage, 208 ms with one; a wave of 152 groups of
// two slots over 262144 points 5.4 -> 3.3 ms, tensor pipe 58 % of the full
// squares before).  4 points of 16.7 million, K = 80: 51 -> 42 ms.
// The zero blocks are neither copied nor stored: K step kk keeps its four
// slabs (8 columns each, two hi, two lo) of m (K - 16 kk) rows back to back.
// S~ rows stream through a ring of stages of `per` K steps, each step four
// slabs of 128 rows (two hi, two lo).
struct QvecLayout {
    int K, m, stages, per;
    uint32_t w_bytes, s_bytes, off_s, off_bar, bytes;
};

constexpr int kQNumBars(int stages) { return 2 * stages + 2 + 2 + 2 + 1; }
constexpr int kQEpiWarps = 8;  // two per TMEM lane quadrant, splitting the group's slots
// Copy producers, taking the stages in turn: a stage of four 2 KB copies keeps
// one issuing thread busy for 430 ns (a wait, the expected bytes, 55 ns a
// copy), longer than the stage's MMAs take; four bring one every 107 ns.
constexpr int kQProducers = 4;
constexpr int kQThreads = 32 * (1 + kQEpiWarps + kQProducers);

inline QvecLayout qvec_layout(int K, int m, int stages, int per) {
    QvecLayout l{};
    const uint32_t nb = (uint32_t)K / 16;
    l.K = K;
    l.m = m;
    l.stages = stages;
    l.per = per;
    l.w_bytes = (uint32_t)m * (nb * (nb + 1) / 2) * 1024u;
    l.s_bytes = (uint32_t)per * 4u * kQSlab;
    l.off_s = l.w_bytes;
    l.off_bar = l.off_s + stages * l.s_bytes;
    l.bytes = l.off_bar + kQNumBars(stages) * 8 + 16 + 1024;
    return l;
}

// Items are (group, 128-point tile) pairs.  Groups run in waves of gridDim.x;
// a full wave gives every CTA one group whose tiles it walks in order, so all
// CTAs read the same region of the S~ image at about the same time and it is
// fetched from DRAM about once per wave.  A partial wave splits its items
// evenly.  Every role walks the same sequence; f returns false to stop.
template <class F>
__device__ __forceinline__ void qvec_items(int64_t n_groups, int64_t n_tq, F&& f) {
    for (int64_t v0 = 0; v0 < n_groups; v0 += gridDim.x) {
        const int64_t wg = (n_groups - v0 < (int64_t)gridDim.x) ? n_groups - v0 : (int64_t)gridDim.x;
        const int64_t tot = wg * n_tq;
        const int64_t ch = (tot + gridDim.x - 1) / gridDim.x;
        const int64_t a = (int64_t)blockIdx.x * ch;
        const int64_t b = (a + ch < tot) ? a + ch : tot;
        int64_t grp = v0 + a / n_tq, t = a % n_tq;
        for (int64_t it = a; it < b; ++it) {
            if (!f(grp, t)) return;
            if (++t == n_tq) {
                t = 0;
                ++grp;
            }
        }
    }
}

__global__ void __launch_bounds__(kQThreads, 1)
    k_qvec_tc(const uint16_t* __restrict__ Bt, const uint16_t* __restrict__ Wimg, const float4* __restrict__ wnorm,
              const float4* __restrict__ gnorm, const int32_t* __restrict__ slots, int n_slots, int64_t G,
              int64_t G_pad, int nfit, float* __restrict__ Qc, float* __restrict__ Qb, uint16_t* __restrict__ Qb3,
              int* __restrict__ status, QvecLayout lay) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_addr(smem);
    const int K = lay.K, M = lay.m, STAGES = lay.stages;
    uint64_t* bars = (uint64_t*)(smem + lay.off_bar);
    uint32_t* tmem_holder = (uint32_t*)(smem + lay.off_bar + kQNumBars(STAGES) * 8);
    volatile int* abort_flag = (volatile int*)(tmem_holder + 1);
    auto bar = [&](int i) { return smem_addr(&bars[i]); };
    const int S_FULL = 0, S_EMPTY = STAGES, W_FULL = 2 * STAGES, W_EMPTY = 2 * STAGES + 1,
              T_FULL = 2 * STAGES + 2, T_EMPTY = 2 * STAGES + 4, DONE = 2 * STAGES + 6;
    const int warp = uniform(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar(S_FULL + s), 1);
            mbar_init(bar(S_EMPTY + s), 1);
        }
        mbar_init(bar(W_FULL), 1);
        mbar_init(bar(W_EMPTY), 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(T_FULL + i), 1);
            mbar_init(bar(T_EMPTY + i), kQEpiWarps);
        }
        mbar_init(bar(DONE), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(tmem_holder)),
                     "r"(kQTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = uniform(*tmem_holder);
    const int64_t n_tq = G_pad / kQM;
    const int64_t n_groups = (n_slots + M - 1) / M;
    auto group_size = [&](int64_t grp) {
        const int64_t r = n_slots - grp * M;
        return (int)(r < M ? r : M);
    };
    const uint32_t tile_elems = 2u * K * kBN;      // bf16 elements of one 256-row B-image tile
    const int nb = K / 16, NC = (nb + lay.per - 1) / lay.per;  // K steps and stages of a tile

    // warp 0 and the warps after the epilogue's are producers 0, 1, ...
    // At most as many as there are stages: a producer that has filled stage n knows stage n - STAGES
    // consumed, and its next wait, for stage n + producers, tells phases apart by their parity only if
    // the use before the slot's last one is consumed too.
    const int n_prod = min(kQProducers, STAGES);
    const int prod = warp == 0 ? 0 : warp - (1 + kQEpiWarps);
    if ((warp == 0 || warp >= 2 + kQEpiWarps) && prod < n_prod) {
        // --------------------------------------------------------- producers
        const bool leader = elect_one();
        int turn = 0;  // whose stage the next one is
        uint32_t used = 0, phase = 0;  // slots this producer has filled, and the phase of its last fill
        int w_par = -1, w_loads = 0, s = 0;
        int64_t cur = -1;
        uint32_t ph = 0;
        bool ok = true;
        qvec_items(n_groups, n_tq, [&](int64_t grp, int64_t t) {
            if (grp != cur && prod == 0) {
                if (w_loads > 0 && !warp_wait(bar(W_EMPTY), (uint32_t)((w_loads - 1) & 1), abort_flag)) {
                    ok = false;
                    return false;
                }
                const int mg = group_size(grp);
                // 16-row blocks b >= kk of the slabs of K step kk: nb (nb + 1) / 2 blocks for each of the
                // step's four slabs, 256 bytes each
                if (leader) mbar_expect_tx(bar(W_FULL), (uint32_t)mg * (uint32_t)(nb * (nb + 1) / 2) * 4u * 256u);
                __syncwarp();
                // the lanes share the copies: lane l takes slabs l, l + 32, ...
                for (int i = 0; i < mg; ++i) {
                    const uint16_t* w = Wimg + (size_t)slots[grp * M + i] * 2 * K * K;
                    for (int j = lane; j < 2 * K / 8; j += 32) {
                        const int jj = j < K / 8 ? j : j - K / 8, kk = jj / 2;
                        const uint32_t slab = (uint32_t)(nb - kk) * M * 256u;
                        const uint32_t dst = sbase + (uint32_t)(kk * nb - kk * (kk - 1) / 2) * M * 1024u +
                                             (uint32_t)((j < K / 8 ? 0 : 2) + (jj & 1)) * slab;
                        for (int b = kk; b < nb; ++b)
                            bulk_g2s(dst + (uint32_t)((b - kk) * mg + i) * 256u, w + ((size_t)j * K + b * 16) * 8, 256u,
                                     bar(W_FULL));
                    }
                }
                __syncwarp();
                w_par = w_loads & 1;
                ++w_loads;
                cur = grp;
            }
            // rows (t & 1) * 128 .. +127 of B-image tile t / 2: one 2 KB run per 8-column slab
            const uint16_t* src = Bt + (t >> 1) * (int64_t)tile_elems + (t & 1) * (kQM * 8);
            for (int c = 0; c < NC; ++c) {
                const bool mine = turn == prod;
                if (++turn == n_prod) turn = 0;
                if (mine) {
                    if (!warp_wait(bar(S_EMPTY + s), ph ^ 1, abort_flag)) {
                        ok = false;
                        return false;
                    }
                    const uint32_t full = bar(S_FULL + s);
                    const int k_hi = min((c + 1) * lay.per, nb);
                    if (leader) {
                        mbar_expect_tx(full, (uint32_t)(k_hi - c * lay.per) * 4u * kQSlab);
                        uint32_t dst = sbase + lay.off_s + s * lay.s_bytes;
                        // hi slabs 2 kk, 2 kk + 1 and lo slabs K/8 + 2 kk, K/8 + 2 kk + 1 of each K step
                        const uint16_t* hi = src + (int64_t)(2 * c * lay.per) * (kBN * 8);
                        for (int kk = c * lay.per; kk < k_hi; ++kk) {
                            const uint16_t* lo = hi + (int64_t)(K / 8) * (kBN * 8);
                            bulk_g2s(dst, hi, kQSlab, full);
                            bulk_g2s(dst + kQSlab, hi + kBN * 8, kQSlab, full);
                            bulk_g2s(dst + 2 * kQSlab, lo, kQSlab, full);
                            bulk_g2s(dst + 3 * kQSlab, lo + kBN * 8, kQSlab, full);
                            hi += 2 * kBN * 8;
                            dst += 4 * kQSlab;
                        }
                    }
                    __syncwarp();
                    used |= 1u << s;
                    phase = (phase & ~(1u << s)) | (ph << s);
                }
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            return true;
        });
        if (!ok) {
            if (lane == 0) {
                *abort_flag = 1;
                atomicOr(status, kDevTimeout);
            }
            // let every copy this warp issued land before the CTA can exit
            if (w_par >= 0) mbar_wait(bar(W_FULL), (uint32_t)w_par, nullptr);
            for (int s = 0; s < STAGES; ++s)
                if ((used >> s) & 1u) mbar_wait(bar(S_FULL + s), (phase >> s) & 1u, nullptr, kDrainNs);
        }
    } else if (warp == 1) {
        // --------------------------------------------------------------- MMA
        const bool leader = elect_one();
        int w_uses = 0, s = 0, ab = 0, mg = 0;
        int64_t cur = -1;
        uint32_t ph = 0, aph = 0;
        bool ok = true;
        // Low words of the descriptors; the high word (row-group stride, version) is common.  The A
        // descriptors move with the ring.  Per K step the B descriptors go on by the step's four slabs,
        // which get m 16-row blocks shorter, and N and the accumulator column follow the triangle.
        const uint64_t dhi = smem_desc(0, 0, 128) & 0xffffffff00000000ull;
        const uint32_t a_lbo = (kQSlab >> 4) << 16, a_k = (4 * kQSlab) >> 4, a_lo_off = (2 * kQSlab) >> 4;
        const uint32_t a_first = ((sbase + lay.off_s) >> 4) | a_lbo, a_stage = lay.s_bytes >> 4;
        const uint32_t b_slab = (uint32_t)nb * M * 16u, b_less = (uint32_t)M * 16u;  // in 16-byte units
        qvec_items(n_groups, n_tq, [&](int64_t grp, int64_t) {
            if (grp != cur) {
                // the previous group's W images stay until every MMA issued so far has completed
                if (w_uses > 0 && leader) mma_commit(bar(W_EMPTY));
                __syncwarp();
                if (!warp_wait(bar(W_FULL), (uint32_t)(w_uses & 1), abort_flag)) {
                    ok = false;
                    return false;
                }
                ++w_uses;
                cur = grp;
                mg = group_size(grp);
            }
            if (!warp_wait(bar(T_EMPTY + ab), aph ^ 1, abort_flag)) {
                ok = false;
                return false;
            }
            const uint32_t id_k = (uint32_t)(2 * mg) << 17, d_k = 16u * mg;
            uint32_t d = tmem_base + (uint32_t)(ab * 256), id = idesc_bf16(kQM, mg * K), slab = b_slab,
                     bk = (sbase >> 4) | (b_slab << 16);
            for (int c = 0; c < NC; ++c) {
                if (!warp_wait(bar(S_FULL + s), ph, abort_flag)) {
                    ok = false;
                    return false;
                }
                tc_fence_after();
                uint32_t ak = a_first + (uint32_t)s * a_stage;
                const int k_hi = min((c + 1) * lay.per, nb);
                for (int kk = c * lay.per; kk < k_hi; ++kk) {
                    if (leader) {
                        mma_bf16(d, dhi | ak, dhi | bk, id, kk ? 1u : 0u);
                        mma_bf16(d, dhi | (ak + a_lo_off), dhi | bk, id, 1u);
                        mma_bf16(d, dhi | ak, dhi | (bk + 2 * slab), id, 1u);
                    }
                    ak += a_k;
                    bk += 4 * slab - (b_less << 16);
                    slab -= b_less;
                    id -= id_k;
                    d += d_k;
                }
                if (leader) mma_commit(bar(S_EMPTY + s));
                __syncwarp();
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            if (leader) mma_commit(bar(T_FULL + ab));
            __syncwarp();
            if (++ab == 2) { ab = 0; aph ^= 1u; }
            return true;
        });
        if (!ok && lane == 0) {
            *abort_flag = 1;
            atomicOr(status, kDevTimeout);
        }
        __syncwarp();
        if (leader) {
            mma_commit(bar(DONE));
            mbar_wait(bar(DONE), 0, nullptr);
        }
        __syncwarp();
    } else if (warp >= 2 && warp < 2 + kQEpiWarps) {
        // ---------------------------------------------------------- epilogue
        const int quad = warp & 3;
        const int half = (warp - 2) >> 2;  // slots half, half + 2, ... of each group
        const int row = quad * 32 + lane;
        const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
        const float gam = (float)(K + 2) * 5.9604645e-08f;
        const float acc = (float)(3 * K + 2) * 1.02f * 1.1920929e-07f;
        const float slack = q_rel_slack(nfit);
        int ab = 0, my_slot = 0;
        uint32_t aph = 0;
        int64_t cur = -1;
        float4 my_wn = make_float4(0.f, 0.f, 0.f, 0.f);
        qvec_items(n_groups, n_tq, [&](int64_t grp, int64_t t) {
            const int mg = group_size(grp);
            if (grp != cur) {  // lane i keeps the group's slot i and its norms
                cur = grp;
                my_slot = lane < mg ? slots[grp * M + lane] : 0;
                if (lane < mg) my_wn = wnorm[my_slot];
            }
            // everything the bound reads is on its way before the accumulator is waited for
            const int64_t g = t * kQM + row;
            const float4 gn = g < G ? gnorm[g] : make_float4(0.f, 0.f, 0.f, 0.f);
            const bool w_ok = mbar_wait(bar(T_FULL + ab), aph, abort_flag);
            if (!__all_sync(0xffffffffu, w_ok)) {
                if (lane == 0) {
                    *abort_flag = 1;
                    atomicOr(status, kDevTimeout);
                }
                return false;
            }
            tc_fence_after();
            const uint32_t tb = tmem_base + lane_base + (uint32_t)(ab * 256);
            auto release = [&]() {  // this warp has read its columns
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(T_EMPTY + ab));
            };
            if (half >= mg) release();
            for (int i = half; i < mg; i += 2) {
                // sum of squares of the slot's K columns
                float q4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
                for (int b = 0; b < K / 16; ++b) {
                    uint32_t r[16];
                    tmem_ld16(tb + (uint32_t)((b * mg + i) * 16), r);
                    tmem_wait(r);
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        q4[k & 3] = fmaf(__uint_as_float(r[k]), __uint_as_float(r[k]), q4[k & 3]);
                }
                if (i + 2 >= mg) release();  // before the bound's arithmetic and the stores
                const float q = (q4[0] + q4[1]) + (q4[2] + q4[3]);
                const int slot = __shfl_sync(0xffffffffu, my_slot, i);
                float4 wn;
                wn.x = __shfl_sync(0xffffffffu, my_wn.x, i);
                wn.y = __shfl_sync(0xffffffffu, my_wn.y, i);
                wn.z = __shfl_sync(0xffffffffu, my_wn.z, i);
                wn.w = __shfl_sync(0xffffffffu, my_wn.w, i);
                float qc = 0.0f, qb = 3.0e38f;
                if (g < G) {
                    const float E =
                        1.0001f * fmaf(wn.y, gn.y, fmaf(wn.z, gn.x, fmaf(wn.w, gn.z, acc * wn.x * gn.x)));
                    const float tlo = __fsqrt_rd(__fmul_rd(q, __fsub_rd(1.0f, gam)));
                    const float thi = __fsqrt_ru(__fmul_ru(q, __fadd_ru(1.0f, gam)));
                    const float lo = fmaxf(0.0f, __fsub_rd(tlo, E));
                    const float hi = __fadd_ru(thi, E);
                    const float delta = fmaxf(__fsub_ru(q, __fmul_rd(lo, lo)), __fsub_ru(__fmul_ru(hi, hi), q));
                    qc = q;
                    qb = __fsub_rd(__fsub_rd(q, delta), slack * q);
                }
                const size_t o = (size_t)slot * G_pad + g;
                Qc[o] = qc;
                Qb[o] = qb;
                store_qb3(Qb3 + o * 8, qb);
            }
            if (++ab == 2) { ab = 0; aph ^= 1u; }
            return true;
        });
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kQTmemCols)
                     : "memory");
    }
}

}  // namespace

bool qvec_tc_supported(int K) { return K >= 16 && K <= kMaxScreenK && K % 16 == 0; }

void launch_wimage(const double* W64, const int32_t* slots, int n, int nfit, int K, uint16_t* Wimg, float4* wnorm,
                   cudaStream_t st) {
    if (n <= 0) return;
    count_launch();
    k_wimage<<<n, 256, 0, st>>>(W64, slots, nfit, K, Wimg, wnorm);
}

// Widest group whose W images leave room for at least four stages (the
// producers' number, which they need).
static bool qvec_pick_layout(int K, int n, QvecLayout* out) {
    constexpr int kPer = 2, kMaxStages = 16;
    int m = 256 / K;
    if (m > n) m = n;
    for (; m >= 1; --m) {
        const int per = kPer < K / 16 ? kPer : K / 16;
        const QvecLayout one = qvec_layout(K, m, 1, per);
        if (one.bytes > kQSmemMax) continue;
        int stages = 1 + (int)((kQSmemMax - one.bytes) / (one.s_bytes + 16u));
        stages = stages > kMaxStages ? kMaxStages : stages;
        if (stages < 4) continue;
        *out = qvec_layout(K, m, stages, per);
        return true;
    }
    return false;
}

bool launch_qvec_tc(const uint16_t* Bt, const uint16_t* Wimg, const float4* wnorm, const float4* gnorm,
                    const int32_t* slots, int n, int64_t G, int64_t G_pad, int nfit, int K, float* Qc, float* Qb,
                    uint16_t* Qb3, int* status, int n_sm, cudaStream_t st) {
    if (n <= 0) return true;
    if (!qvec_tc_supported(K)) return false;
    QvecLayout lay{};
    if (!qvec_pick_layout(K, n, &lay)) return false;
    // the largest layout's, not this launch's: the limit is shared by every thread that launches the kernel
    cudaFuncSetAttribute(k_qvec_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQSmemMax);
    const int64_t groups = (n + lay.m - 1) / lay.m;
    const int64_t items = groups * (G_pad / kQM);
    const int grid = (int)(items < n_sm ? items : n_sm);
    count_launch();
    k_qvec_tc<<<grid, kQThreads, lay.bytes, st>>>(Bt, Wimg, wnorm, gnorm, slots, n, G, G_pad, nfit, Qc,
                                                              Qb, Qb3, status, lay);
    return true;
}

}  // namespace fcdev
