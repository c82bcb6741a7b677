// Eq. 1 window scores and the Section 4.2 importance I (before pooling), from
// the window queries' attention over the candidate tokens, recomputed on the
// tensor cores with the softmax statistics (m_r, Z_r) of the score kernel.
//
// Work unit: (sequence s, 128-token tile of candidates, group of up to 8 KV
// heads); the candidates are [0, L - w), or [0, L) when every position
// competes.  An item is one KV head h of a unit: S^T = K_tile Q_h^T on
// tcgen05.mma (M = 128 tokens, N = g*w query rows padded to 16, K = d) into a
// TMEM accumulator, so one epilogue thread owns one token and every query row
// of it:
//   A[r][t]   = 2^(s_rt * scale * log2(e) - m_r) / Z_r   (softmax over all visible keys)
//   G_h[q][t] = sum_j A[(q, j)][t]                       (GQA group sum, r = q * g + j)
//   P_O[h,t]  = (1/O)  sum_{q >= w-O}  G_h[q][t]
//   P_O'[h,t] = (1/O') sum_{q >= w-O'} G_h[q][t]
//   I[t]      = (1/O)  sum_{q >= w-O}  max_h G_h[q][t]
// The grid is persistent: a CTA walks units blockIdx.x, blockIdx.x + gridDim.x,
// ... and the items of its units in order.  Warp 0 streams K_h and Q_h with
// TMA into a ring of stages, warp 1 issues the MMAs into A accumulators (4 of
// N <= 128 columns, or 2 of N <= 256), and the epilogue is A groups of four
// warps (one per TMEM lane quadrant): group a takes the CTA's items a, a + A,
// ..., each thread all the query rows of its token, so every group streams
// through its own accumulator without waiting for the others.  The head maxima
// of G_h[q][t] meet in shared memory through atomicMax on the float bits
// (values are >= +0, so the integer order is the float order and the result
// does not depend on the order of the updates); the last group to finish a
// unit sums them into I (or, with several head groups per tile, writes them to
// a partial buffer that the heads kernel combines).  The raw rows go to the
// slot arrays; pooling happens in the heads kernel.
#include <cudaTypedefs.h>

#include "kvec_internal.cuh"
#include "sm100_ptx.cuh"
#include "tile_loads.cuh"

namespace kvec {

namespace {

constexpr int kWinThreads = 576;                      // warp 0 TMA, warp 1 MMA, warps 2..17 epilogue
constexpr int kMaxSmemWin = 232448;                   // opt-in shared memory per CTA on sm_103
constexpr int kKTileBytes = kTileT * kHeadDim * 2;    // 32 KB: two 64-column swizzled halves
constexpr int kMaxStages = 3;                         // deepest operand ring
constexpr int kWinReserveSms = 8;                     // SMs a window launch leaves to the other kernels

struct WinArgs {
    CUtensorMap kmap[kMaxGroup], qmap[kMaxGroup];
    Geometry G;
    int* err;
    Slot sl[kMaxGroup];
    const int* cu;                  // device cu_seqlens
    int upl;                        // units of a layer
    int Npad;                       // query rows padded to a multiple of 16 (MMA N)
    int kst;                        // operand stages
    int nacc;                       // accumulators = epilogue groups (4, or 2 when N > 128)
    int units;                      // (layer, sequence, candidate tile, head group) units of the launch
    uint32_t tmem_cols;
    int fault;                      // test of the error path (kvec_set_test_fault).  1: the first
                                    // accumulator is never signalled and its wait gives up early;
                                    // 2: a warp gives up on the head maxima buffer of its third unit
};

// Limit of the epilogue's wait for the withheld accumulator under the injected fault.
constexpr uint64_t kFaultWaitNs = 20000;

struct __align__(8) WinBars {
    uint64_t full[kMaxStages], empty[kMaxStages], acc_full[4], acc_empty[4];
    uint64_t mma_done;
    uint32_t tmem_base;
    volatile int abort_flag;
    volatile int gok[4][2];     // per group: the outcome of its accumulator wait, by item parity
    int done[2];                // per unit parity: groups finished with the unit
    volatile int ready[2];      // per unit parity: the local unit index whose maxima may use the buffer
    int last[4];                // per group: 1 if it finished a unit last
};

__host__ __device__ inline size_t stage_bytes(int Npad) { return (size_t)kKTileBytes + 2 * (size_t)Npad * 128; }

// Shared memory: stages | head maxima [2][O][128] | row statistics [4 groups][2][256] | barriers.
__host__ __device__ inline size_t win_smem_bytes(int Npad, int O, int kst) {
    return 1024 + (size_t)kst * stage_bytes(Npad) + 2 * (size_t)O * kTileT * sizeof(float) +
           4 * 2 * 256 * sizeof(float) + sizeof(WinBars);
}

__device__ __forceinline__ void win_abort(WinBars* bars, int* err) {
    bars->abort_flag = 1;
    atomicExch(err, 3);
}

// Unit u of a layer -> sequence s, candidate tile jt within it, head group ng, global
// candidate tile tg; sequence s owns ceil(Lc / 128) * NG consecutive units.
struct WinUnit {
    int s, jt, ng, tg, L, Lc, row0;
};

__device__ __forceinline__ bool decode_unit(const Geometry& G, const int* cu, int u, WinUnit& w) {
    int base = 0, tbase = 0;
    for (int b = 0; b < G.batch; ++b) {
        const int c0 = __ldg(&cu[b]), c1 = __ldg(&cu[b + 1]);
        const int Lc = c1 - c0 - G.wk;
        const int nt = Lc > 0 ? (Lc + kTileT - 1) / kTileT : 0;
        if (u < base + nt * G.NG) {
            const int local = u - base;
            w.s = b;
            w.jt = local / G.NG;
            w.ng = local - w.jt * G.NG;
            w.tg = tbase + w.jt;
            w.L = c1 - c0;
            w.Lc = Lc;
            w.row0 = c0 + w.jt * kTileT;
            return true;
        }
        base += nt * G.NG;
        tbase += nt;
    }
    return false;
}

// One head of this thread's token: the group sums G_h[q] of every window row q,
// added to po (q >= w-O) and poe (q >= w-O') and folded into the head maxima
// (q >= w-O).  Rows q < qmin come before the token (it lies in the window part,
// which only later rows see): their attention to it is 0.  GG > 0 is the group
// size g known at compile time: each 32-column chunk holds 32 / GG whole
// groups and runs as straight-line code.
template <int GG>
__device__ __forceinline__ void head_rows(uint32_t taddr, const float* __restrict__ rsb, int g, int w, int qmin,
                                          float sl2, int qO, int qOe, int* maxg_col, float& po, float& poe) {
    if constexpr (GG > 0) {
        constexpr int QPC = 32 / GG, CW = QPC * GG;
        for (int qb = 0; qb < w; qb += QPC) {
            const int c0 = qb * GG;
            float v[32];
            ptx::tmem_ld32(taddr + (uint32_t)c0, v);
            ptx::tmem_wait_ld();
            float pr[CW];
#pragma unroll
            for (int i = 0; i < CW; ++i) pr[i] = ptx::ex2(fmaf(v[i], sl2, -rsb[c0 + i]));
#pragma unroll
            for (int k = 0; k < QPC; ++k) {
                float gs = 0.f;
#pragma unroll
                for (int j = 0; j < GG; ++j) gs += pr[k * GG + j];
                const int q = qb + k;
                gs = q >= qmin ? gs : 0.f;
                if (q < w) {
                    if (q >= qOe) poe += gs;
                    if (q >= qO) {
                        po += gs;
                        atomicMax(maxg_col + (q - qO) * kTileT, __float_as_int(gs));
                    }
                }
            }
        }
    } else {
        float gs = 0.f;
        int q = 0, jq = 0;
        const int c_end = w * g;
        for (int c0 = 0; c0 < c_end; c0 += 32) {
            float v[32];
            ptx::tmem_ld32(taddr + (uint32_t)c0, v);
            ptx::tmem_wait_ld();
            const int n = min(32, c_end - c0);
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                if (i >= n) break;
                gs += ptx::ex2(fmaf(v[i], sl2, -rsb[c0 + i]));
                if (++jq == g) {
                    gs = q >= qmin ? gs : 0.f;
                    if (q >= qOe) poe += gs;
                    if (q >= qO) {
                        po += gs;
                        atomicMax(maxg_col + (q - qO) * kTileT, __float_as_int(gs));
                    }
                    gs = 0.f;
                    jq = 0;
                    ++q;
                }
            }
        }
    }
}

template <int GG>
__global__ void __launch_bounds__(kWinThreads, 1)
    window_kernel(const __grid_constant__ WinArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if (threadIdx.x == 0) {
        ptx::prefetch_tensormap(&A.kmap[0]);
        ptx::prefetch_tensormap(&A.qmap[0]);
        // The next launch on this stream (the next group's row statistics) reads
        // nothing this grid writes and does not wait for it: let it be scheduled.
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    }
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // Scalars and pointers in registers: values read through a reference to the
    // parameter block would be re-read after every asm statement that clobbers memory.
    const Geometry G = A.G;
    int* const err = A.err;
    const int upl = A.upl;
    const int* const cu_dev = A.cu;
    const int kst = A.kst, NA = A.nacc, units = A.units, fault = A.fault;
    const uint32_t tmem_cols = A.tmem_cols;
    const int Npad = A.Npad, R = G.R;
    const size_t sbytes = stage_bytes(Npad);
    int* maxg = reinterpret_cast<int*>(smem + kst * sbytes);             // [2][O][128] float bits
    float* rsm = reinterpret_cast<float*>(maxg + 2 * G.O * kTileT);      // [4][2][256] m_r + log2 Z_r
    WinBars* bars = reinterpret_cast<WinBars*>(rsm + 4 * 2 * 256);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u0 = blockIdx.x, ustep = gridDim.x;

    if (threadIdx.x == 32) {
        for (int i = 0; i < kst; ++i) {
            ptx::mbar_init(&bars->full[i], 1);
            ptx::mbar_init(&bars->empty[i], 1);
        }
        for (int i = 0; i < 4; ++i) {
            ptx::mbar_init(&bars->acc_full[i], 1);
            ptx::mbar_init(&bars->acc_empty[i], 4);   // one arrival per warp of the group
        }
        ptx::mbar_init(&bars->mma_done, 1);
        bars->abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            bars->done[i] = 0;
            bars->ready[i] = i;
        }
        ptx::fence_barrier_init();
    }
    for (int i = threadIdx.x; i < 2 * G.O * kTileT; i += blockDim.x) maxg[i] = 0;
    if (warp == 1) {
        ptx::tmem_alloc(&bars->tmem_base, tmem_cols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = bars->tmem_base;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const uint64_t policy = ptx::policy_evict_first();   // the K tiles' last use
            int it = 0;
            int fills[kMaxStages] = {0, 0, 0};
            for (int u = u0; u < units && !bars->abort_flag; u += ustep) {
                WinUnit wu;
                const int lay = u / upl;
                decode_unit(G, cu_dev, u - lay * upl, wu);
                const int h0 = wu.ng * G.HG, nh = min(G.HG, G.Hkv - h0);
                bool stop = false;
                for (int hh = 0; hh < nh; ++hh, ++it) {
                    const int st = it % kst, n = it / kst;
                    if (n > 0 && !ptx::mbar_wait_abortable(&bars->empty[st], (n - 1) & 1, &bars->abort_flag)) {
                        win_abort(bars, err);
                        stop = true;
                        break;
                    }
                    uint8_t* sk = smem + st * sbytes;
                    uint8_t* sq = sk + kKTileBytes;
                    const int h = h0 + hh;
                    ptx::mbar_arrive_expect_tx(&bars->full[st], (uint32_t)kKTileBytes + 2u * (uint32_t)R * 128u);
                    ptx::tma_load_3d(sk, &A.kmap[lay], &bars->full[st], 0, h, wu.row0, policy);
                    ptx::tma_load_3d(sk + kKTileBytes / 2, &A.kmap[lay], &bars->full[st], 64, h, wu.row0, policy);
                    load_queries(sq, Npad * 128, &A.qmap[lay], &bars->full[st], G, h, wu.s);
                    ++fills[st];
                }
                if (stop) break;
            }
            // Drain: every issued copy lands before the CTA may exit.
            for (int st = 0; st < kst; ++st)
                if (fills[st] > 0) ptx::mbar_wait(&bars->full[st], (fills[st] - 1) & 1, 50000000ull);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = ptx::idesc_bf16_f32(128, Npad);
            int it = 0;
            bool stop = false;
            for (int u = u0; u < units && !stop; u += ustep) {
                WinUnit wu;
                const int lay = u / upl;
                decode_unit(G, cu_dev, u - lay * upl, wu);
                const int nh = min(G.HG, G.Hkv - wu.ng * G.HG);
                for (int hh = 0; hh < nh; ++hh, ++it) {
                    const int st = it % kst, n = it / kst;
                    const int b = it % NA, ub = it / NA;
                    // Giving up on a stage in flight is safe: the producer drains its own loads.
                    if (bars->abort_flag || !ptx::mbar_wait_abortable(&bars->full[st], n & 1, &bars->abort_flag) ||
                        (ub > 0 && !ptx::mbar_wait_abortable(&bars->acc_empty[b], (ub - 1) & 1, &bars->abort_flag))) {
                        win_abort(bars, err);
                        stop = true;
                        break;
                    }
                    ptx::tc_fence_after();
                    const uint32_t sk = ptx::smem_u32(smem + st * sbytes), sq = sk + kKTileBytes;
                    const uint32_t d = tmem + (uint32_t)(b * Npad);
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const int half = kk >> 2, kin = kk & 3;
                        const uint64_t ad = ptx::smem_desc_k_sw128(sk + half * (kKTileBytes / 2) + kin * 32);
                        const uint64_t bd = ptx::smem_desc_k_sw128(sq + half * Npad * 128 + kin * 32);
                        ptx::mma_bf16(d, ad, bd, idesc, kk > 0 ? 1u : 0u);
                    }
                    ptx::mma_commit(&bars->empty[st]);
                    if (!(fault == 1 && it == 0)) ptx::mma_commit(&bars->acc_full[b]);
                }
            }
            ptx::mma_commit(&bars->mma_done);
        }
    } else if (warp < 2 + 4 * NA) {
        // ------------------------------------------------------------ epilogue
        const int grp = (warp - 2) >> 2;                  // accumulator / item group
        const int gtid = threadIdx.x - 64 - grp * 128;    // 0 .. 127 within the group
        const int quad = warp & 3;                        // TMEM lanes 32*quad .. +31
        const int tok = quad * 32 + lane;                 // token within the tile
        const int bar_id = 1 + grp;                       // named barrier of the group (128 threads)
        const int qO = G.w - G.O, qOe = G.w - G.Oe;
        const float invO = 1.f / (float)G.O, invOe = 1.f / (float)G.Oe;
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(grp * Npad);
        float* rs_g = rsm + grp * 2 * 256;
        // Row statistics come from the launch this grid is a programmatic
        // dependent of: wait for it before the first read.
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
        // This thread's rows (gtid, gtid + 128) of an item's statistics.
        auto fetch = [&](const float2* rowstat, int s, int h, float& a, float& b) {
            const float2* src = rowstat + ((size_t)s * G.Hkv + h) * R;
            a = b = 0.f;
            if (gtid < R) {
                const float2 m = __ldcg(src + gtid);
                a = m.x + __log2f(m.y);
            }
            if (gtid + 128 < R) {
                const float2 m = __ldcg(src + gtid + 128);
                b = m.x + __log2f(m.y);
            }
        };
        int it = 0, k = 0;   // it: CTA item index; k: this group's items so far
        bool failed = false;
        for (int u = u0, ul = 0; u < units; u += ustep, ++ul) {
            WinUnit wu;
            const int lay = u / upl;
            decode_unit(G, cu_dev, u - lay * upl, wu);
            const Slot& sl = A.sl[lay];
            const int h0 = wu.ng * G.HG, nh = min(G.HG, G.Hkv - h0);
            const int t = wu.jt * kTileT + tok;                  // token within the sequence
            const int qmin = t - (wu.L - G.w);                   // > 0 only for tokens in the window part
            const int buf = ul & 1;
            int* mg = maxg + buf * G.O * kTileT;
            // The head maxima buffer of this unit parity is free once the unit two
            // before has been folded into I (bounded wait on a flag of this CTA).  A warp
            // that gives up takes its group along: the barriers below have no limit.
            if (ul >= 2) {
                bool ok = true;
                if (lane == 0) {
                    const bool give_up = fault == 2 && gtid == 32;
                    const long long c0 = clock64();
                    while (give_up || bars->ready[buf] != ul) {
                        if (give_up || bars->abort_flag || clock64() - c0 > 600000000ll) {
                            win_abort(bars, err);
                            ok = false;
                            break;
                        }
                        __nanosleep(64);
                    }
                }
                if (ptx::named_bar_or(bar_id, 128, !ok)) break;
                __threadfence_block();
            }
            float pa = 0.f, pb = 0.f;
            int hh = (grp - it % NA + NA) % NA;   // the unit's first item for this group
            if (!failed && hh < nh) fetch(sl.rowstat, wu.s, h0 + hh, pa, pb);
            for (; hh < nh && !failed; hh += NA, ++k) {
                // gtid 0 waits for the accumulator and publishes the outcome to the
                // group with the statistics (one barrier per item).
                if (gtid == 0) {
                    const bool ok = !bars->abort_flag &&
                                    ptx::mbar_wait_abortable(&bars->acc_full[grp], k & 1, &bars->abort_flag,
                                                             fault == 1 && it + hh == 0 ? kFaultWaitNs : 200000000ull);
                    if (!ok) win_abort(bars, err);
                    bars->gok[grp][k & 1] = ok ? 1 : 0;
                }
                float* rsb = rs_g + (k & 1) * 256;
                rsb[gtid] = pa;
                rsb[gtid + 128] = pb;
                ptx::named_bar_sync(bar_id, 128);
                if (!bars->gok[grp][k & 1]) {
                    failed = true;
                    break;
                }
                if (hh + NA < nh) fetch(sl.rowstat, wu.s, h0 + hh + NA, pa, pb);   // next item's rows, in flight
                ptx::tc_fence_after();
                float po = 0.f, poe = 0.f;
                head_rows<GG>(tbase, rsb, G.g, G.w, qmin, G.sl2, qO, qOe, mg + tok, po, poe);
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(&bars->acc_empty[grp]);
                if (t < wu.Lc) {
                    const size_t row = (size_t)wu.s * G.Hkv + h0 + hh;
                    sl.rawO[row * G.ML + t] = po * invO;
                    sl.rawOe[row * G.ML + t] = poe * invOe;
                }
            }
            it += nh;
            if (failed) break;
            // This group is done with the unit: the last of the NA groups folds the
            // head maxima into I and frees the buffer for the unit two ahead.
            ptx::named_bar_sync(bar_id, 128);
            if (gtid == 0) {
                __threadfence_block();
                bars->last[grp] = atomicAdd(&bars->done[buf], 1) == NA - 1;
                __threadfence_block();
            }
            ptx::named_bar_sync(bar_id, 128);
            if (bars->last[grp]) {
                __threadfence_block();
                if (G.NG > 1) {
                    float* wp = sl.wpart + ((size_t)wu.tg * G.NG + wu.ng) * G.O * kTileT;
                    for (int q = 0; q < G.O; ++q) wp[q * kTileT + tok] = __int_as_float(mg[q * kTileT + tok]);
                } else if (t < wu.Lc) {
                    float ip = 0.f;
                    for (int q = 0; q < G.O; ++q) ip += __int_as_float(mg[q * kTileT + tok]);
                    sl.rawI[(size_t)wu.s * G.ML + t] = ip * invO;
                }
                for (int q = 0; q < G.O; ++q) mg[q * kTileT + tok] = 0;
                ptx::named_bar_sync(bar_id, 128);
                if (gtid == 0) {
                    bars->done[buf] = 0;
                    __threadfence_block();
                    bars->ready[buf] = ul + 2;
                }
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    if (warp == 1 && lane == 0) ptx::mbar_wait(&bars->mma_done, 0, 50000000ull);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 1) ptx::tmem_dealloc(tmem, tmem_cols);
}

// ---------------------------------------------------------------------------
// Tile-owning variant for O of 8 or 16 and a window that is a multiple of 8 (query
// tiles ordered by query head, Geometry::jm).
//
// A unit is T consecutive candidate tiles of one sequence and one head group, and
// the NA = T * P epilogue groups (one TMEM accumulator each) split it: group a owns
// tile a / P for the heads a % P, a % P + P, ... of the head group.  The query block
// Q_h is loaded once per (unit, head) into its own two-slot ring and serves the T
// tiles of the head, so the K ring holds 32 KB stages only.  A thread keeps the
// running maxima over its heads of its token's O last-row group sums in registers;
// with P > 1 the P groups of a tile meet in shared memory at the unit's end (the
// maximum does not depend on the order).  CTAs claim units from a per-launch
// counter.
//
// Each row sum adds its positions in ascending order, as window_kernel does.
// ---------------------------------------------------------------------------
constexpr int kTileOMax = 16;     // largest O of the tile-owning variant (register maxima)
// The paper's windows (w = O' = 32, O = 16): known at compile time, the epilogue's
// addresses are constants and no position is compared with a window's start, which
// takes 40 % of its instructions away (it bounds the kernel).
constexpr int kDefWindow = 32, kDefObs = 16;
constexpr int kMaxKStages = 6;
constexpr int kUnitSlots = 4;     // claimed units in flight inside a CTA
constexpr int kTileThreads = kWinThreads + 64;   // warps 18 and 19: a second MMA issuer and its producer
constexpr int kTileMmaWarp1 = 18, kTileTmaWarp1 = 19;

struct TileArgs {
    CUtensorMap kmap[kMaxGroup], qmap[kMaxGroup];
    Geometry G;
    int* err;
    int* claim;                     // the launch's unit counter, zero before the launch
    Slot sl[kMaxGroup];
    const int* cu;
    int upl;                        // units of a layer
    int Npad, kst, nacc, T, units, fault;
};

struct __align__(8) TileBars {
    uint64_t k_full[kMaxKStages], k_empty[kMaxKStages], q_full[2], q_empty[2], acc_full[4], acc_empty[4];
    uint64_t u_full[kUnitSlots], u_empty[kUnitSlots];
    uint64_t m_full[4], m_empty[4];  // per tile, P > 1: the other groups' maxima are there / have been read
    uint64_t mma_done;
    uint32_t tmem_base;
    volatile int abort_flag;
    volatile int unit[kUnitSlots];   // claimed unit (-1: no more work)
};

// Shared memory: K stages | query slots [2] | normalisers [4 groups][2][256] | maxima [3][O][128] (P > 1) | barriers.
__host__ __device__ inline size_t tile_smem_bytes(int Npad, int kst, bool shared_tiles) {
    return 1024 + (size_t)kst * kKTileBytes + 2 * (size_t)Npad * 256 + 4 * 2 * 256 * sizeof(float) +
           (shared_tiles ? 3 * kTileOMax * kTileT * sizeof(float) : 0) + sizeof(TileBars);
}

// Unit u of a layer -> sequence s, first candidate tile j0 of the unit, its tile count nt,
// head group ng, global candidate tile of j0.
struct TileUnit {
    int s, j0, nt, ng, tg0, L, Lc, row0;
};

__device__ __forceinline__ bool decode_tile_unit(const Geometry& G, const int* cu, int T, int u, TileUnit& w) {
    int base = 0, tbase = 0;
    for (int b = 0; b < G.batch; ++b) {
        const int c0 = __ldg(&cu[b]), c1 = __ldg(&cu[b + 1]);
        const int Lc = c1 - c0 - G.wk;
        const int ntile = Lc > 0 ? (Lc + kTileT - 1) / kTileT : 0;
        const int ngrp = (ntile + T - 1) / T;
        if (u < base + ngrp * G.NG) {
            const int local = u - base;
            const int tgi = local / G.NG;
            w.s = b;
            w.ng = local - tgi * G.NG;
            w.j0 = tgi * T;
            w.nt = min(T, ntile - w.j0);
            w.tg0 = tbase + w.j0;
            w.L = c1 - c0;
            w.Lc = Lc;
            w.row0 = c0 + w.j0 * kTileT;
            return true;
        }
        base += ngrp * G.NG;
        tbase += ntile;
    }
    return false;
}

// Group sums G_h[q] of eight window positions q0 .. q0 + 7 of this thread's token:
// sum over the query heads j of 2^(s * scale * log2 e - normaliser), columns
// j * w + q.  nrs: the normalisers.  GG > 0: the group size g, known at compile
// time (the columns of up to four query heads are loaded together).
template <int GG>
__device__ __forceinline__ void group_sums8(uint32_t taddr, const float* __restrict__ nrs, int g, int w, int q0, float sl2,
                                            float* gs) {
    auto add_head = [&](const float* v, int j, bool first) {
        const float4* n4 = reinterpret_cast<const float4*>(nrs + j * w + q0);
        const float4 na = n4[0], nb = n4[1];
        const float n[8] = {na.x, na.y, na.z, na.w, nb.x, nb.y, nb.z, nb.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float e = ptx::ex2(fmaf(v[k], sl2, -n[k]));
            gs[k] = first ? e : gs[k] + e;
        }
    };
    if constexpr (GG > 0) {
#pragma unroll
        for (int j0 = 0; j0 < GG; j0 += 4) {
            float v[4][8];
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
                if (j0 + jj < GG) ptx::tmem_ld8(taddr + (uint32_t)((j0 + jj) * w + q0), v[jj]);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
                if (j0 + jj < GG) add_head(v[jj], j0 + jj, j0 + jj == 0);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) gs[k] = 0.f;   // 0 + x is x: the sums start at +0 or above
        for (int j = 0; j < g; ++j) {
            float v[8];
            ptx::tmem_ld8(taddr + (uint32_t)(j * w + q0), v);
            ptx::tmem_wait_ld();
            add_head(v, j, false);
        }
    }
}

template <int GG, bool DW>
__global__ void __launch_bounds__(kTileThreads, 1) window_tiles_kernel(const __grid_constant__ TileArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    if (threadIdx.x == 0) {
        ptx::prefetch_tensormap(&A.kmap[0]);
        ptx::prefetch_tensormap(&A.qmap[0]);
        // The next launch on this stream (the next group's row statistics) reads
        // nothing this grid writes and does not wait for it: let it be scheduled.
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    }
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const Geometry G = A.G;
    int* const err = A.err;
    const int upl = A.upl;
    const int* const cu_dev = A.cu;
    const int kst = A.kst, NA = A.nacc, T = A.T, units = A.units, fault = A.fault;
    const int Npad = A.Npad, R = G.R, P = NA / T;
    // MMA issuers, each with its own part of the K ring (see score_kernel), and the
    // item's: by accumulator j * P + hh % P, even or odd.
    const int ni = kst >= 4 ? 2 : 1, half_ring = (kst + 1) / 2;
    auto ring_first = [&](int c) { return c == 0 ? 0 : half_ring; };
    auto ring_end = [&](int c) { return c == 0 && ni == 2 ? half_ring : kst; };
    auto issuer = [&](int j, int hh) { return ni == 1 ? 0 : (P == 1 ? j : hh) & 1; };
    uint8_t* sK = smem;                                      // kst x 32 KB
    uint8_t* sQ = sK + (size_t)kst * kKTileBytes;            // 2 slots x Npad x 256 B
    float* rsm = reinterpret_cast<float*>(sQ + 2 * (size_t)Npad * 256);   // [4][2][256]
    float* mbuf = rsm + 4 * 2 * 256;                         // [3][O][128], P > 1 only
    TileBars* bars = reinterpret_cast<TileBars*>(mbuf + (P > 1 ? 3 * kTileOMax * kTileT : 0));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 32) {
        for (int i = 0; i < kst; ++i) {
            ptx::mbar_init(&bars->k_full[i], 1);
            ptx::mbar_init(&bars->k_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            ptx::mbar_init(&bars->q_full[i], 1);
            ptx::mbar_init(&bars->q_empty[i], ni);
        }
        for (int i = 0; i < 4; ++i) {
            ptx::mbar_init(&bars->acc_full[i], 1);
            ptx::mbar_init(&bars->acc_empty[i], 4);   // one arrival per warp of the group
        }
        for (int i = 0; i < T; ++i) {
            ptx::mbar_init(&bars->m_full[i], 4 * (P > 1 ? P - 1 : 1));
            ptx::mbar_init(&bars->m_empty[i], 4);
        }
        for (int i = 0; i < kUnitSlots; ++i) {
            ptx::mbar_init(&bars->u_full[i], 1);
            ptx::mbar_init(&bars->u_empty[i], 2 * ni - 1 + 4 * NA);   // issuers, second producer, epilogue warps
        }
        ptx::mbar_init(&bars->mma_done, ni);
        bars->abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (warp == 1) {
        ptx::tmem_alloc(&bars->tmem_base, 512);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    auto give_up = [&]() {
        bars->abort_flag = 1;
        atomicExch(err, 3);
    };
    // The next claimed unit for a warp of the MMA issuer or the epilogue; -1: no more
    // work, -2: gave up.
    auto take_unit = [&](int di) {
        const int ds = di % kUnitSlots;
        if (!ptx::warp_wait(&bars->u_full[ds], (di / kUnitSlots) & 1, &bars->abort_flag)) {
            if (lane == 0) give_up();
            return -2;
        }
        const int u = ptx::warp_uniform(bars->unit[ds]);
        if (lane == 0) ptx::mbar_arrive(&bars->u_empty[ds]);
        return u;
    };
    auto uniform_unit = [&](int u, TileUnit& tu) {
        const int lay = u / upl;
        decode_tile_unit(G, cu_dev, T, u - lay * upl, tu);
        tu.s = ptx::warp_uniform(tu.s);
        tu.nt = ptx::warp_uniform(tu.nt);
        tu.ng = ptx::warp_uniform(tu.ng);
        tu.row0 = ptx::warp_uniform(tu.row0);
        return lay;
    };

    // The producer and the MMA issuer run as whole warps and elect a lane for the
    // instructions that one thread issues (see score_kernel).
    if (warp == 0 || warp == kTileTmaWarp1) {
        // ------------------------------------------------------------ TMA producers
        const int me = warp == kTileTmaWarp1 ? 1 : 0;
        const uint64_t policy = ptx::policy_evict_first();   // the K tiles' last use
        int qi = 0, st = ring_first(me);
        uint32_t kphase = 0u, filled = 0u;   // bit st: filled an odd number of times; filled at all
        bool stop = false;
        int next = 0;
        if (me == 0 && lane == 0) next = atomicAdd(A.claim, 1);
        for (int di = 0; !stop && me < ni; ++di) {
            int u;
            if (me == 0) {
                const int ds = di % kUnitSlots, nd = di / kUnitSlots;
                if (nd > 0 && !ptx::warp_wait(&bars->u_empty[ds], (nd - 1) & 1, &bars->abort_flag)) {
                    stop = true;
                    break;
                }
                u = ptx::warp_uniform(bars->abort_flag ? units : next);
                if (lane == 0) {
                    bars->unit[ds] = u < units ? u : -1;
                    ptx::mbar_arrive(&bars->u_full[ds]);
                }
                if (u >= units) break;
                if (lane == 0) next = atomicAdd(A.claim, 1);   // arrives while this unit is loaded
            } else {
                u = take_unit(di);
                if (u < 0) break;
            }
            TileUnit tu;
            const int lay = uniform_unit(u, tu);
            const int h0 = tu.ng * G.HG, nh = min(G.HG, G.Hkv - h0);
            for (int hh = 0; hh < nh && !stop; ++hh) {
                const int h = h0 + hh;
                if (me == 0) {
                    const int qs = qi & 1, nq = qi >> 1;
                    if (nq > 0 && !ptx::warp_wait(&bars->q_empty[qs], (nq - 1) & 1, &bars->abort_flag)) {
                        stop = true;
                        break;
                    }
                    if (ptx::elect_one()) {
                        ptx::mbar_arrive_expect_tx(&bars->q_full[qs], 2u * (uint32_t)R * 128u);
                        load_queries(sQ + (size_t)qs * Npad * 256, (uint32_t)Npad * 128u, &A.qmap[lay], &bars->q_full[qs], G, h,
                                     tu.s);
                    }
                    __syncwarp();
                    ++qi;
                }
                for (int j = 0; j < tu.nt; ++j) {
                    if (issuer(j, hh) != me) continue;
                    if (((filled >> st) & 1u) != 0u &&
                        !ptx::warp_wait(&bars->k_empty[st], ((kphase >> st) & 1u) ^ 1u, &bars->abort_flag)) {
                        stop = true;
                        break;
                    }
                    if (ptx::elect_one()) {
                        uint8_t* sk = sK + (size_t)st * kKTileBytes;
                        const int row = tu.row0 + j * kTileT;
                        ptx::mbar_arrive_expect_tx(&bars->k_full[st], (uint32_t)kKTileBytes);
                        ptx::tma_load_3d(sk, &A.kmap[lay], &bars->k_full[st], 0, h, row, policy);
                        ptx::tma_load_3d(sk + kKTileBytes / 2, &A.kmap[lay], &bars->k_full[st], 64, h, row, policy);
                    }
                    __syncwarp();
                    kphase ^= 1u << st;
                    filled |= 1u << st;
                    st = st + 1 == ring_end(me) ? ring_first(me) : st + 1;
                }
            }
        }
        if (stop && lane == 0) give_up();
        // Drain: every issued copy lands before the CTA may exit.
        for (int b = 0; b < kst; ++b)
            if ((filled >> b) & 1u) ptx::mbar_wait(&bars->k_full[b], ((kphase >> b) & 1u) ^ 1u, 50000000ull);
        for (int b = 0; b < 2 && b < qi; ++b)
            ptx::mbar_wait(&bars->q_full[b], ((qi - b + 1) / 2 - 1) & 1, 50000000ull);
    } else if (warp == 1 || warp == kTileMmaWarp1) {
        // ------------------------------------------------------------ MMA issuers
        const int me = warp == kTileMmaWarp1 ? 1 : 0;
        const uint32_t idesc = ptx::idesc_bf16_f32(128, Npad);
        const uint64_t qdesc = ptx::smem_desc_k_sw128(ptx::smem_u32(sQ)), kdesc = ptx::smem_desc_k_sw128(ptx::smem_u32(sK));
        const uint32_t qhalf = (uint32_t)Npad * 128u;
        int qi = 0, st = ring_first(me), first = 1;
        uint32_t kphase = 0u, used = 0u, aphase = 0u;   // per stage / accumulator
        bool stop = false;
        for (int di = 0; !stop && me < ni; ++di) {
            const int u = take_unit(di);
            if (u < 0) break;
            TileUnit tu;
            uniform_unit(u, tu);
            const int nh = min(G.HG, G.Hkv - tu.ng * G.HG);
            for (int hh = 0, hp = 0; hh < nh && !stop; ++hh, hp = hp + 1 == P ? 0 : hp + 1) {
                const int qs = qi & 1;
                if (!ptx::warp_wait(&bars->q_full[qs], (qi >> 1) & 1, &bars->abort_flag)) {
                    stop = true;
                    break;
                }
                for (int j = 0; j < tu.nt; ++j) {
                    const int b = j * P + hp;
                    if (issuer(j, hh) == me) {
                        // Giving up on a stage in flight is safe: the producer drains its own loads.
                        if (!ptx::warp_wait(&bars->k_full[st], (kphase >> st) & 1u, &bars->abort_flag) ||
                            (((used >> b) & 1u) != 0u &&
                             !ptx::warp_wait(&bars->acc_empty[b], ((aphase >> b) & 1u) ^ 1u, &bars->abort_flag))) {
                            stop = true;
                            break;
                        }
                        ptx::tc_fence_after();
                        if (ptx::elect_one()) {
                            const uint64_t kd = kdesc + (uint32_t)(st * (kKTileBytes >> 4)), qd = qdesc + (uint32_t)qs * (qhalf >> 3);
                            const uint32_t d = tmem + (uint32_t)(b * Npad);
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk) {
                                const uint32_t half = kk >> 2, kin = kk & 3;
                                ptx::mma_bf16(d, kd + half * (kKTileBytes >> 5) + kin * 2, qd + half * (qhalf >> 4) + kin * 2,
                                              idesc, kk > 0 ? 1u : 0u);
                            }
                            ptx::mma_commit(&bars->k_empty[st]);
                            if (!(fault && first)) ptx::mma_commit(&bars->acc_full[b]);
                        }
                        __syncwarp();
                        kphase ^= 1u << st;
                        used |= 1u << b;
                        aphase ^= 1u << b;
                        st = st + 1 == ring_end(me) ? ring_first(me) : st + 1;
                    }
                    first = 0;
                }
                if (ptx::elect_one()) ptx::mma_commit(&bars->q_empty[qs]);   // this issuer's products of the head
                __syncwarp();
                ++qi;
            }
        }
        if (stop && lane == 0) give_up();
        if (me < ni && ptx::elect_one()) ptx::mma_commit(&bars->mma_done);
        __syncwarp();
    } else if (warp < 2 + 4 * NA) {
        // ------------------------------------------------------------ epilogue
        const int grp = (warp - 2) >> 2;                  // accumulator
        const int tile = grp / P, par = grp - tile * P;   // tile of the unit, heads par, par + P, ...
        const int gtid = threadIdx.x - 64 - grp * 128;
        const int quad = warp & 3;
        const int tok = quad * 32 + lane;
        const int w = DW ? kDefWindow : G.w, g = GG > 0 ? GG : G.g, O = DW ? kDefObs : G.O, Oe = DW ? kDefWindow : G.Oe;
        const int qO = w - O, qOe = w - Oe;
        const float invO = 1.f / (float)O, invOe = 1.f / (float)Oe;
        const float sl2 = G.sl2;
        const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(grp * Npad);
        float* rs_g = rsm + grp * 2 * 256;
        // This thread's columns of an item, gtid and gtid + 128: their rows in the statistics.
        const int r0 = gtid % w * g + gtid / w, r1 = (gtid + 128) % w * g + (gtid + 128) / w;
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
        auto fetch = [&](const float2* rowstat, int s, int h, float& a, float& b) {
            const float2* src = rowstat + ((size_t)s * G.Hkv + h) * R;
            a = b = 0.f;
            if (gtid < R) {
                const float2 m = __ldcg(src + r0);
                a = m.x + __log2f(m.y);
            }
            if (gtid + 128 < R) {
                const float2 m = __ldcg(src + r1);
                b = m.x + __log2f(m.y);
            }
        };
        uint32_t k = 0u, meets = 0u;   // items of this group and meetings of its tile's groups so far
        bool failed = false;           // this warp gave up on a wait
        for (int di = 0;; ++di) {
            const int u = failed ? -2 : take_unit(di);
            // The group's warps leave together: whoever gave up says so at the next
            // group barrier, where all of them hear it.
            if (ptx::named_bar_or(1 + grp, 128, u == -2) || u < 0) break;
            const int lay = u / upl;
            TileUnit tu;
            decode_tile_unit(G, cu_dev, T, u - lay * upl, tu);
            if (tile >= tu.nt) continue;   // this group's tile is past the sequence's last
            const Slot& sl = A.sl[lay];
            const float2* rowstat = sl.rowstat;
            const int h0 = tu.ng * G.HG, nh = min(G.HG, G.Hkv - h0);
            const int t0 = (tu.j0 + tile) * kTileT, t = t0 + tok;
            // Rows q < qmin come before the token (it lies in the window part, a candidate
            // only when every position is one): their attention to it is 0.
            const int qmin = t - (tu.L - w);
            const bool masked = G.wk == 0 && t0 + kTileT - 1 > tu.L - w;
            float mx[kTileOMax];
#pragma unroll
            for (int i = 0; i < kTileOMax; ++i) mx[i] = 0.f;
            float pa = 0.f, pb = 0.f;
            if (par < nh) fetch(rowstat, tu.s, h0 + par, pa, pb);
            for (int hh = par; hh < nh; hh += P, ++k) {
                // The group's threads exchange the normalisers while the accumulator fills.
                float* nrs = rs_g + (k & 1u) * 256;
                nrs[gtid] = pa;
                nrs[gtid + 128] = pb;
                // One warp of the group polls, the others wait in the barrier (a polling
                // warp takes issue slots from those that compute).
                bool ok = true;
                if (gtid < 32) {
                    ok = ptx::warp_wait(&bars->acc_full[grp], k & 1u, &bars->abort_flag,
                                        fault && k == 0u && grp == 0 ? kFaultWaitNs : 200000000ull);
                    if (!ok && lane == 0) give_up();
                }
                failed = ptx::named_bar_or(1 + grp, 128, !ok);
                if (failed) break;
                if (hh + P < nh) fetch(rowstat, tu.s, h0 + hh + P, pa, pb);   // the next head's rows, in flight
                ptx::tc_fence_after();
                float po = 0.f, poe = 0.f;
                float gs[8];
                auto sums = [&](int q0) {
                    group_sums8<GG>(tbase, nrs, g, w, q0, sl2, gs);
                    if (masked) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) gs[i] = q0 + i < qmin ? 0.f : gs[i];
                    }
                };
                for (int q0 = qOe & ~7; q0 < qO; q0 += 8) {
                    sums(q0);
                    if (q0 >= qOe) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) poe += gs[i];
                    } else {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (q0 + i >= qOe) poe += gs[i];
                    }
                }
#pragma unroll
                for (int c = 0; c < kTileOMax / 8; ++c) {
                    const int q0 = qO + 8 * c;
                    if (q0 >= w) break;
                    sums(q0);
                    if (q0 + 8 >= w) {   // the accumulator is in registers
                        ptx::tc_fence_before();
                        __syncwarp();
                        if (lane == 0) ptx::mbar_arrive(&bars->acc_empty[grp]);
                    }
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float x = gs[i];
                        if (q0 + i >= qOe) poe += x;
                        po += x;
                        mx[8 * c + i] = fmaxf(mx[8 * c + i], x);
                    }
                }
                if (t < tu.Lc) {
                    const size_t row = (size_t)tu.s * G.Hkv + h0 + hh;
                    sl.rawO[row * G.ML + t] = po * invO;
                    sl.rawOe[row * G.ML + t] = poe * invOe;
                }
            }
            if (failed) continue;
            if (P > 1) {
                // The P groups of the tile: their maxima meet in the first one's registers.
                float* mb = mbuf + (size_t)(tile * (P - 1)) * kTileOMax * kTileT + tok;
                int ok = 1;
                if (lane == 0) {
                    if (par > 0)
                        ok = meets == 0u || ptx::mbar_wait_abortable(&bars->m_empty[tile], (meets - 1u) & 1u, &bars->abort_flag);
                    else
                        ok = ptx::mbar_wait_abortable(&bars->m_full[tile], meets & 1u, &bars->abort_flag);
                    if (!ok) give_up();
                }
                ++meets;
                if (!__shfl_sync(0xffffffffu, ok, 0)) {
                    failed = true;
                    continue;
                }
                __syncwarp();   // what lane 0 waited for is there for every lane
                if (par > 0) {
#pragma unroll
                    for (int i = 0; i < kTileOMax; ++i) mb[((par - 1) * kTileOMax + i) * kTileT] = mx[i];
                } else {
                    for (int o = 0; o < P - 1; ++o)
#pragma unroll
                        for (int i = 0; i < kTileOMax; ++i) mx[i] = fmaxf(mx[i], mb[(o * kTileOMax + i) * kTileT]);
                }
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(par > 0 ? &bars->m_full[tile] : &bars->m_empty[tile]);
            }
            if (par > 0) continue;
            // I[t] = (1/O) sum over the last O rows of the maxima over the heads (or
            // this head group's maxima, combined by the heads kernel).
            if (G.NG > 1) {
                float* wp = sl.wpart + ((size_t)(tu.tg0 + tile) * G.NG + tu.ng) * O * kTileT;
#pragma unroll
                for (int i = 0; i < kTileOMax; ++i)
                    if (i < O) wp[i * kTileT + tok] = mx[i];
            } else if (t < tu.Lc) {
                float ip = 0.f;
#pragma unroll
                for (int i = 0; i < kTileOMax; ++i)
                    if (i < O) ip += mx[i];
                sl.rawI[(size_t)tu.s * G.ML + t] = ip * invO;
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    if (warp == 1 && lane == 0) ptx::mbar_wait(&bars->mma_done, 0, 50000000ull);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 1) ptx::tmem_dealloc(tmem, 512);
}

int npad_of(int R) { return (R + 15) & ~15; }

int kst_for(int Npad, int O) {
    int k = kMaxStages;
    while (k > 1 && win_smem_bytes(Npad, O, k) > (size_t)kMaxSmemWin) --k;
    return k;
}

// Units of a layer: (sequence, candidate tile, head group).
int units_of(const Geometry& g) { return g.win_tiles * g.NG; }

}  // namespace

size_t window_smem_bytes(const Geometry& g) {
    const int Npad = npad_of(g.R);
    return win_smem_bytes(Npad, g.O, kst_for(Npad, g.O));
}

cudaError_t configure_window(const Geometry& g) {
    // Per-function attribute shared by every handle: the opt-in maximum (every
    // geometry's stage count is chosen to fit it).
    (void)g;
    cudaError_t e = cudaSuccess;
    for (auto fn : {window_kernel<0>, window_kernel<1>, window_kernel<2>, window_kernel<4>, window_kernel<7>,
                    window_kernel<8>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmemWin);
    for (auto fn : {window_tiles_kernel<0, true>, window_tiles_kernel<1, true>, window_tiles_kernel<2, true>,
                    window_tiles_kernel<4, true>, window_tiles_kernel<7, true>, window_tiles_kernel<8, true>,
                    window_tiles_kernel<0, false>, window_tiles_kernel<1, false>, window_tiles_kernel<2, false>,
                    window_tiles_kernel<4, false>, window_tiles_kernel<8, false>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmemWin);
    return e;
}

namespace {

// SMs of a window grid: a few are left to the selection chain and the other
// layers' kernels.
int usable_sms(int num_sms) { return num_sms > 2 * kWinReserveSms ? num_sms - kWinReserveSms : num_sms; }

int tile_kst_for(int Npad, bool shared_tiles) {
    int k = kMaxKStages;
    while (k > 1 && tile_smem_bytes(Npad, k, shared_tiles) > (size_t)kMaxSmemWin) --k;
    return k;
}

// A layer's units of the tile-owning variant: groups of T candidate tiles per sequence and head group.
int tile_units_of(const Geometry& g, const int* cu_host, int T) {
    int units = 0;
    for (int b = 0; b < g.batch; ++b) {
        const int Lc = cu_host[b + 1] - cu_host[b] - g.wk;
        const int nt = Lc > 0 ? (Lc + kTileT - 1) / kTileT : 0;
        units += (nt + T - 1) / T * g.NG;
    }
    return units;
}

// Candidate tiles per unit: with more of them the query blocks are loaded less
// often (32 KB for every T tiles of 32 KB), with fewer there are more units; the
// most that still give every usable SM a unit.
int tile_unit_tiles(const Geometry& g, int nl, int usable) {
    int T = npad_of(g.R) <= 128 ? 4 : 2;
    while (T > 1 && tile_units_of(g, g.cu_host, T) * nl < usable) T /= 2;
    return T;
}

template <class Args>
void set_layers(Args* a, const ScorePlan& sp, const Geometry& g, const Group& gr, const Scratch& sc) {
    for (int l = 0; l < gr.nl; ++l) {
        a->kmap[l] = sp.kmap[l];
        a->qmap[l] = sp.qmap[l];
        a->sl[l] = gr.sl[l];
    }
    a->G = g;
    a->err = sc.err;
    a->cu = gr.io[0].cu;
}

cudaError_t launch_window_tiles(const ScorePlan& sp, const Geometry& g, const Group& gr, const Scratch& sc,
                                int* claim, cudaStream_t st, bool after_own_launch) {
    TileArgs a{};
    set_layers(&a, sp, g, gr, sc);
    const int usable = usable_sms(sp.num_sms);
    a.claim = claim + 1;
    a.Npad = npad_of(g.R);
    a.nacc = a.Npad <= 128 ? 4 : 2;   // nacc * Npad <= 512 TMEM columns
    a.T = tile_unit_tiles(g, gr.nl, usable);
    a.kst = tile_kst_for(a.Npad, a.T < a.nacc);
    a.upl = tile_units_of(g, g.cu_host, a.T);
    a.units = gr.nl * a.upl;
    a.fault = test_fault() == 1 ? 1 : 0;
    const size_t smem = tile_smem_bytes(a.Npad, a.kst, a.T < a.nacc);
    const int grid = a.units < usable ? a.units : usable;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kTileThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = after_own_launch ? 1 : 0;
    const bool dw = g.w == kDefWindow && g.Oe == kDefWindow && g.O == kDefObs;
    const auto launch = [&](auto with_dw, auto without) {
        return dw ? cudaLaunchKernelEx(&cfg, with_dw, a) : cudaLaunchKernelEx(&cfg, without, a);
    };
    switch (g.g) {
        case 1: return launch(window_tiles_kernel<1, true>, window_tiles_kernel<1, false>);
        case 2: return launch(window_tiles_kernel<2, true>, window_tiles_kernel<2, false>);
        case 4: return launch(window_tiles_kernel<4, true>, window_tiles_kernel<4, false>);
        case 7: return launch(window_tiles_kernel<7, true>, window_tiles_kernel<0, false>);
        case 8: return launch(window_tiles_kernel<8, true>, window_tiles_kernel<8, false>);
        default: return launch(window_tiles_kernel<0, true>, window_tiles_kernel<0, false>);
    }
}

}  // namespace

bool tile_variant_fits(const Geometry& g) { return g.w % 8 == 0 && (g.O == 8 || g.O == kTileOMax); }

int window_grid_size(const ScorePlan& sp, const Geometry& g, int nl) {
    if (g.win_tiles == 0) return 0;
    const int usable = usable_sms(sp.num_sms);
    const int units = g.jm ? tile_units_of(g, g.cu_host, tile_unit_tiles(g, nl, usable)) : units_of(g);
    return units * nl < usable ? units * nl : usable;
}

cudaError_t launch_window(const ScorePlan& sp, const Geometry& g, const Group& gr, const Scratch& sc, int* claim,
                          cudaStream_t st, bool after_own_launch) {
    if (g.win_tiles == 0) return cudaSuccess;
    if (g.jm) return launch_window_tiles(sp, g, gr, sc, claim, st, after_own_launch);
    WinArgs a{};
    set_layers(&a, sp, g, gr, sc);
    a.Npad = npad_of(g.R);
    a.kst = kst_for(a.Npad, g.O);
    a.nacc = a.Npad <= 128 ? 4 : 2;   // nacc * Npad <= 512 TMEM columns
    a.upl = units_of(g);
    a.units = gr.nl * a.upl;
    a.fault = test_fault();
    a.tmem_cols = 512;   // one CTA per SM; a 32-column load past the last group's columns stays inside
    const size_t smem = win_smem_bytes(a.Npad, g.O, a.kst);
    // Persistent: at most one CTA per SM.
    const int usable = usable_sms(sp.num_sms);
    const int grid = a.units < usable ? a.units : usable;
    // after_own_launch: the previous kernel on the stream is this layer's
    // row-statistics launch and no event wait stands between them; the launch is
    // then its programmatic dependent and waits (griddepcontrol.wait) right
    // before reading the statistics.
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kWinThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = after_own_launch ? 1 : 0;
    switch (g.g) {
        case 1: return cudaLaunchKernelEx(&cfg, window_kernel<1>, a);
        case 2: return cudaLaunchKernelEx(&cfg, window_kernel<2>, a);
        case 4: return cudaLaunchKernelEx(&cfg, window_kernel<4>, a);
        case 7: return cudaLaunchKernelEx(&cfg, window_kernel<7>, a);
        case 8: return cudaLaunchKernelEx(&cfg, window_kernel<8>, a);
        default: return cudaLaunchKernelEx(&cfg, window_kernel<0>, a);
    }
}

}  // namespace kvec
