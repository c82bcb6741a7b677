// Softmax statistics of the window queries' attention over every visible key
// (the denominators of the attention A that Eq. 1 averages): for each query
// row r of KV head h, the row max m_r of s = <q_r, k_t> * scale (log2 units)
// and Z_r = sum_t 2^(s_rt - m_r), causal on the window part.
//
// Persistent, warp-specialised, one CTA per SM; a launch serves a group of
// layers, and its CTAs claim chunks of a layer's consecutive work items
// (sequence s, KV head h, 128-token tile j) from a per-launch counter, so a CTA
// that starts late (its SM held by other kernels) takes fewer chunks instead of
// delaying the launch:
//   warp 0      TMA producer: the KV head's g*w query rows (once per (s,h) of a
//               chunk, two buffers) and a ring of 128-token K tiles, both
//               128-byte swizzled; warp 19 loads the K tiles of the second issuer;
//   warps 1, 18 issue tcgen05.mma (M = 128 query rows per M-block, N = 128 tokens,
//               K = 128 = d) into TMEM accumulators, the even ones and the odd ones:
//               an issuer's waits and commits take as long as the products, which
//               run meanwhile for the other one's item.  Each has its own part of
//               the K ring (a ring with two readers that skip each other's stages
//               would let one of them take a phase for another two further on);
//               with fewer than four stages there is one issuer;
//   warps 2..17 epilogue: groups of warps, one per TMEM accumulator, each
//               taking every NB-th item of a chunk; one thread per query row and
//               all 128 columns of the item: tcgen05.ld of its logits, their sum
//               of 2^(s - max), merged online into the thread's running
//               (max, sum) of the group's items of one (s, h) inside the chunk.
// No stage waits for a chunk's end: the producer claims the next chunk while it
// loads this one, its K tiles follow each other through the ring whatever chunk
// they belong to, and every warp of the epilogue takes the chunks from the hand-
// over slots by itself.  At the end of a segment (a run of one (s, h) inside a
// chunk) each group writes one (max, sum) partial per row; rowstat_kernel merges
// the groups' and then the segments' partials of a (s, h) into (m_r, Z_r).  The
// segments and the groups' shares are fixed by the chunk boundaries, not by which
// CTA claimed a chunk, so the results do not depend on the schedule.
// The window kernel recomputes the logits with these statistics.
#include <cudaTypedefs.h>

#include <algorithm>

#include "kvec_internal.cuh"
#include "sm100_ptx.cuh"
#include "tile_loads.cuh"

namespace kvec {

namespace {

constexpr int kKStages = 6;                           // deepest K ring (fewer when shared memory is short)
constexpr int kMaxSmem = 232448;                      // opt-in shared memory per CTA on sm_103
constexpr int kKStageBytes = kTileT * kHeadDim * 2;   // 32 KB: two 64-column swizzled halves
constexpr int kKHalfBytes = kTileT * 128;             // 16 KB
constexpr uint32_t kTmemCols = 512;

constexpr int kSeqCache = 64;   // sequences whose first items the CTA keeps in shared memory

// Position of work item i of a layer: sequence s, KV head h, tile j.  Items are
// ordered (s, h, j); sequence s owns ntiles(s) * Hkv consecutive items.  A role
// walks a chunk's items in order, so the walker decodes once and then steps.
struct ItemWalker {
    const int* cu;
    const int* first;             // [batch] first item of every sequence, or null (batch > kSeqCache)
    int batch, Hkv;
    int s, h, j, ntiles;
    int row0, L;                  // cu[s], L_s

    __device__ __forceinline__ void enter_sequence() {
        row0 = __ldg(&cu[s]);
        L = __ldg(&cu[s + 1]) - row0;
        ntiles = tiles_of(L);
    }
    __device__ __forceinline__ void init(int i) {
        int base = 0;
        if (first) {
            for (s = 0; s + 1 < batch && i >= first[s + 1]; ++s) {}
            base = first[s];
            enter_sequence();
        } else {
            for (s = 0; s < batch; ++s) {
                enter_sequence();
                if (i < base + ntiles * Hkv) break;
                base += ntiles * Hkv;
            }
        }
        const int local = i - base;
        h = local / ntiles;
        j = local - h * ntiles;
    }
    __device__ __forceinline__ bool last_of_head() const { return j + 1 == ntiles; }
    __device__ __forceinline__ int head() const { return s * Hkv + h; }
    __device__ __forceinline__ void next() {
        if (++j < ntiles) return;
        j = 0;
        if (++h < Hkv) return;
        h = 0;
        if (++s < batch) enter_sequence();
    }
};

constexpr int kScoreReserveSms = 8;      // SMs a score launch leaves to the other kernels
constexpr int kChunkLarge = 12;          // (sequence, head, tile) items per claim when there are enough
constexpr int kChunkSmall = 8;           // items per claim otherwise
constexpr int kChunkSlots = 4;           // claimed chunks in flight inside a CTA

// MMA issuers of a ring of kst K stages, and the first stage and number of stages
// of an issuer's part.
__host__ __device__ constexpr int issuers(int kst) { return kst >= 4 ? 2 : 1; }
__device__ __forceinline__ int ring_first(int kst, int c) { return c == 0 ? 0 : (kst + 1) / 2; }
__device__ __forceinline__ int ring_end(int kst, int c) { return c == 0 && issuers(kst) == 2 ? (kst + 1) / 2 : kst; }

struct ScoreArgs {
    CUtensorMap kmap[kMaxGroup], qmap[kMaxGroup];
    Geometry G;
    const int* cu;                 // device cu_seqlens
    int* err;
    int nl;       // layers
    int W;        // work items of a layer
    int kst;      // K ring depth
    int* claim;   // the launch's chunk counter, zero before the launch
    int chunk;    // items per claim
    int by_item;  // layout of the partials (partials_by_item)
    int fault;    // test of the error path (kvec_set_test_fault): one epilogue warp gives up on its first chunk
    float2* segpart[kMaxGroup];
};

constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kScoreThreads = 64 + kEpiThreads + 64;
constexpr int kScoreRegThreads = 896;
static_assert(kScoreThreads <= kScoreRegThreads, "the launch bound");
constexpr int kMmaWarp1 = 2 + kEpiWarps;   // the second issuer
constexpr int kTmaWarp1 = 3 + kEpiWarps;   // its producer

struct __align__(8) Barriers {
    uint64_t k_full[kKStages], k_empty[kKStages];
    uint64_t q_full[2], q_empty[2];
    uint64_t acc_full[4], acc_empty[4];
    uint64_t c_full[kChunkSlots], c_empty[kChunkSlots];
    uint64_t mma_done;
    uint32_t tmem_base;
    volatile int abort_flag;
    volatile int chunk[kChunkSlots];   // claimed chunk (-1: no more work)
    int first[kSeqCache];              // first item of every sequence
};

__device__ __forceinline__ void raise_abort(Barriers* bars, int* err) {
    bars->abort_flag = 1;
    atomicExch(err, 3);
}

__device__ __forceinline__ void merge_partial(float& M, float& Z, float2 o) {
    if (o.x == -INFINITY) return;
    if (o.x > M) {
        Z = Z * ptx::ex2(M - o.x) + o.y;
        M = o.x;
    } else {
        Z += o.y * ptx::ex2(o.x - M);
    }
}

// MB: 128-row M-blocks per KV head (R <= 128 * MB).  The 16 epilogue warps form
// NB = 4 / MB groups of 4 * MB warps, one group per TMEM accumulator.
// Compiled for kScoreRegThreads threads, i.e. for 72 registers (nothing spills): of
// the register file 19456 are left, so that row statistics, pooling and gather CTAs
// run beside a score CTA that stays for its whole grid, instead of on the few SMs
// without one.  With the 96 that 640 threads may have: ragged batch of 8 prompts 2217 us
// (72: 2098), 16 short prompts 1052 (985), 32 layers of 8192 tokens 388 (371), of 32768
// 1087 (1046).  The window kernel spills below 96 (given log-sum-exps 1277 -> 1308).
template <int MB>
__global__ void __launch_bounds__(kScoreRegThreads, 1) score_kernel(const __grid_constant__ ScoreArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    // 1024-byte alignment for the swizzled operand tiles.
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // Scalars and pointers in registers: values read through a reference to the
    // parameter block would be re-read after every asm statement that clobbers memory.
    const Geometry G = A.G;
    int* const err = A.err;
    const int W = A.W, kst = A.kst;
    const int chunk_items = A.chunk;
    const int per_layer = (W + chunk_items - 1) / chunk_items;   // chunks of a layer
    const int nchunks = A.nl * per_layer;
    int* const claim = A.claim;
    const int ni = issuers(kst);   // MMA issuers
    const int R = G.R;
    const uint32_t qhalf = (uint32_t)R * 128u;            // bytes of a query buffer's half (64 columns)
    uint8_t* sQ = smem;                                   // 2 buffers x 2 halves x R rows x 128 B
    uint8_t* sK = sQ + 4 * qhalf;                         // kst x 32 KB
    Barriers* bars = reinterpret_cast<Barriers*>(sK + kst * kKStageBytes);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NB = 4 / MB;                             // TMEM accumulator buffers

    if (warp == 0 && lane == 0) {
        ptx::prefetch_tensormap(&A.kmap[0]);
        ptx::prefetch_tensormap(&A.qmap[0]);
        // The next launch on this stream (the next group's statistics) reads
        // nothing this grid writes: let it be scheduled as SMs free up.
        asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    }
    if (threadIdx.x == 32) {
        for (int s = 0; s < kst; ++s) {
            ptx::mbar_init(&bars->k_full[s], 1);
            ptx::mbar_init(&bars->k_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(&bars->q_full[b], 1);
            ptx::mbar_init(&bars->q_empty[b], ni);
        }
        for (int b = 0; b < 4; ++b) {
            ptx::mbar_init(&bars->acc_full[b], 1);
            ptx::mbar_init(&bars->acc_empty[b], 4 * MB);  // one arrival per warp of the group
        }
        for (int c = 0; c < kChunkSlots; ++c) {
            ptx::mbar_init(&bars->c_full[c], 1);
            ptx::mbar_init(&bars->c_empty[c], 2 * ni - 1 + kEpiWarps);   // issuers, second producer, epilogue warps
        }
        ptx::mbar_init(&bars->mma_done, ni);
        bars->abort_flag = 0;
        ptx::fence_barrier_init();
    }
    if (threadIdx.x >= 64 && threadIdx.x - 64 < min(G.batch, kSeqCache)) {
        const int s = threadIdx.x - 64;
        int base = 0;
        for (int b = 0; b < s; ++b) base += tiles_of(__ldg(&A.cu[b + 1]) - __ldg(&A.cu[b])) * G.Hkv;
        bars->first[s] = base;
    }
    if (warp == 1) {
        ptx::tmem_alloc(&bars->tmem_base, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = bars->tmem_base;
    ItemWalker p;
    p.cu = A.cu;
    p.first = G.batch <= kSeqCache ? bars->first : nullptr;
    p.batch = G.batch;
    p.Hkv = G.Hkv;

    // The producer and the MMA issuer run as whole warps, so that what they compute
    // stays uniform, and elect a lane for the instructions that one thread issues.
    // (Run by lane 0 alone, each tcgen05.mma and TMA instruction had its operands
    // moved to uniform registers one by one: 1,700 cycles an item for the MMA issuer.)
    auto uniform_init = [&](int i0) {
        p.init(i0);
        p.s = ptx::warp_uniform(p.s);
        p.h = ptx::warp_uniform(p.h);
        p.j = ptx::warp_uniform(p.j);
        p.ntiles = ptx::warp_uniform(p.ntiles);
        p.row0 = ptx::warp_uniform(p.row0);
    };
    auto uniform_next = [&]() {
        if (++p.j < p.ntiles) return;
        p.j = 0;
        if (++p.h < p.Hkv) return;
        p.h = 0;
        if (++p.s < p.batch) {
            p.enter_sequence();
            p.ntiles = ptx::warp_uniform(p.ntiles);
            p.row0 = ptx::warp_uniform(p.row0);
        }
    };
    if (warp == 0 || warp == kTmaWarp1) {
        // ------------------------------------------------------------ TMA producers
        const int me = warp == kTmaWarp1 ? 1 : 0;
        const uint64_t policy = ptx::policy_evict_normal();   // the window kernel reads K again
        int qloads = 0, st = ring_first(kst, me), di = 0;
        uint32_t kphase = 0u, filled = 0u;   // bit st: filled an odd number of times; filled at all
        int next = 0;
        if (me == 0 && lane == 0) next = atomicAdd(claim, 1);
        bool stop = false;
        while (!stop && me < ni) {
            const int ds = di % kChunkSlots, nd = di / kChunkSlots;
            int c;
            if (me == 0) {
                // Hand the claimed chunk to the other roles, and claim the next one: its
                // number arrives while this one is loaded.
                if (nd > 0 && !ptx::warp_wait(&bars->c_empty[ds], (nd - 1) & 1, &bars->abort_flag)) {
                    stop = true;
                    break;
                }
                c = ptx::warp_uniform(bars->abort_flag ? nchunks : next);
                if (lane == 0) {
                    bars->chunk[ds] = c < nchunks ? c : -1;
                    ptx::mbar_arrive(&bars->c_full[ds]);
                }
                if (c >= nchunks) break;
                if (lane == 0) next = atomicAdd(claim, 1);
            } else {
                if (!ptx::warp_wait(&bars->c_full[ds], nd & 1, &bars->abort_flag)) {
                    stop = true;
                    break;
                }
                c = ptx::warp_uniform(bars->chunk[ds]);
                if (lane == 0) ptx::mbar_arrive(&bars->c_empty[ds]);
                if (c < 0) break;
            }
            ++di;
            const int lay = c / per_layer, i0 = (c - lay * per_layer) * chunk_items, i1 = min(W, i0 + chunk_items);
            const CUtensorMap* kmap = &A.kmap[lay];
            const CUtensorMap* qmap = &A.qmap[lay];
            int prev_sh = -1;   // the query rows are loaded again at every chunk's start
            uniform_init(i0);
            for (int i = i0; i < i1; ++i) {
                if (me == 0 && p.head() != prev_sh) {
                    const int qs = qloads & 1, nq = qloads >> 1;
                    if (nq > 0 && !ptx::warp_wait(&bars->q_empty[qs], (nq - 1) & 1, &bars->abort_flag)) {
                        stop = true;
                        break;
                    }
                    if (ptx::elect_one()) {
                        ptx::mbar_arrive_expect_tx(&bars->q_full[qs], 2u * qhalf);
                        load_queries(sQ + qs * 2 * qhalf, qhalf, qmap, &bars->q_full[qs], G, p.h, p.s);
                    }
                    __syncwarp();
                    ++qloads;
                    prev_sh = p.head();
                }
                if (ni == 1 || ((i - i0) & 1) == me) {   // the item's issuer (NB is even)
                    if (((filled >> st) & 1u) != 0u &&
                        !ptx::warp_wait(&bars->k_empty[st], ((kphase >> st) & 1u) ^ 1u, &bars->abort_flag)) {
                        stop = true;
                        break;
                    }
                    if (ptx::elect_one()) {
                        uint8_t* dst = sK + st * kKStageBytes;
                        const int row = p.row0 + p.j * kTileT;
                        ptx::mbar_arrive_expect_tx(&bars->k_full[st], (uint32_t)kKStageBytes);
                        ptx::tma_load_3d(dst, kmap, &bars->k_full[st], 0, p.h, row, policy);
                        ptx::tma_load_3d(dst + kKHalfBytes, kmap, &bars->k_full[st], 64, p.h, row, policy);
                    }
                    __syncwarp();
                    kphase ^= 1u << st;
                    filled |= 1u << st;
                    st = st + 1 == ring_end(kst, me) ? ring_first(kst, me) : st + 1;
                }
                uniform_next();
            }
        }
        if (stop && lane == 0) raise_abort(bars, err);
        // Drain: every issued copy lands before the CTA may exit (query buffer b was
        // filled ceil((qloads - b) / 2) times).
        for (int b = 0; b < kst; ++b)
            if ((filled >> b) & 1u) ptx::mbar_wait(&bars->k_full[b], ((kphase >> b) & 1u) ^ 1u, 50000000ull);
        for (int b = 0; b < 2 && b < qloads; ++b)
            ptx::mbar_wait(&bars->q_full[b], ((qloads - b + 1) / 2 - 1) & 1, 50000000ull);
    } else if (warp == 1 || warp == kMmaWarp1) {
        // ------------------------------------------------------------ MMA issuers
        const int me = warp == kMmaWarp1 ? 1 : 0;
        const uint32_t idesc = ptx::idesc_bf16_f32(128, kTileT);
        const uint64_t qdesc = ptx::smem_desc_k_sw128(ptx::smem_u32(sQ)), kdesc = ptx::smem_desc_k_sw128(ptx::smem_u32(sK));
        int qk = 0, st = ring_first(kst, me), di = 0;
        uint32_t kphase = 0u, used = 0u, aphase = 0u;   // per stage / accumulator
        bool stop = false;
        while (!stop && me < ni) {
            const int ds = di % kChunkSlots;
            if (!ptx::warp_wait(&bars->c_full[ds], (di / kChunkSlots) & 1, &bars->abort_flag)) {
                stop = true;
                break;
            }
            const int c = ptx::warp_uniform(bars->chunk[ds]);
            if (lane == 0) ptx::mbar_arrive(&bars->c_empty[ds]);
            ++di;
            if (c < 0) break;
            const int i0 = (c % per_layer) * chunk_items, i1 = min(W, i0 + chunk_items);
            int prev_sh = -1, qs = 0, buf = 0;
            uniform_init(i0);
            for (int i = i0; i < i1; ++i) {
                if (p.head() != prev_sh) {
                    qs = qk & 1;
                    if (!ptx::warp_wait(&bars->q_full[qs], (qk >> 1) & 1, &bars->abort_flag)) {
                        stop = true;
                        break;
                    }
                    ++qk;
                    prev_sh = p.head();
                }
                const bool seg_end = i + 1 >= i1 || p.last_of_head();
                if (ni == 1 || (buf & 1) == me) {
                    // Giving up on a stage in flight is safe: the producer drains its own loads.
                    if (!ptx::warp_wait(&bars->k_full[st], (kphase >> st) & 1u, &bars->abort_flag) ||
                        (((used >> buf) & 1u) != 0u &&
                         !ptx::warp_wait(&bars->acc_empty[buf], ((aphase >> buf) & 1u) ^ 1u, &bars->abort_flag))) {
                        stop = true;
                        break;
                    }
                    ptx::tc_fence_after();
                    if (ptx::elect_one()) {
                        const uint64_t kd = kdesc + (uint32_t)(st * (kKStageBytes >> 4)), qd = qdesc + (uint32_t)qs * (qhalf >> 3);
#pragma unroll
                        for (int m = 0; m < MB; ++m) {
                            const uint32_t d = tmem + (uint32_t)(buf * 128 * MB + m * 128);
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk) {
                                const uint32_t half = kk >> 2, kin = kk & 3;
                                ptx::mma_bf16(d, qd + half * (qhalf >> 4) + m * 1024 + kin * 2,
                                              kd + half * (kKHalfBytes >> 4) + kin * 2, idesc, kk > 0 ? 1u : 0u);
                            }
                        }
                        ptx::mma_commit(&bars->k_empty[st]);
                        ptx::mma_commit(&bars->acc_full[buf]);
                    }
                    __syncwarp();
                    kphase ^= 1u << st;
                    used |= 1u << buf;
                    aphase ^= 1u << buf;
                    st = st + 1 == ring_end(kst, me) ? ring_first(kst, me) : st + 1;
                }
                if (seg_end) {   // this issuer's products of the segment, if any, are the last of its query rows
                    if (ptx::elect_one()) ptx::mma_commit(&bars->q_empty[qs]);
                    __syncwarp();
                }
                buf = buf + 1 == NB ? 0 : buf + 1;
                uniform_next();
            }
        }
        if (stop && lane == 0) raise_abort(bars, err);
        if (me < ni && ptx::elect_one()) ptx::mma_commit(&bars->mma_done);
        __syncwarp();
    } else {
        // ------------------------------------------------------------ epilogue
        // NB groups of GW = 4 * MB warps; group a takes the items a, a + NB, ... of
        // every chunk from its own accumulator, so the groups work on different
        // items at once (one group's TMEM loads and barrier waits overlap the
        // others' ex2).  Warp k of a group reads TMEM lanes 32*(warp % 4) .. +31
        // (the lane quadrant its warp id allows) of M-block k / 4: one thread per
        // query row, all 128 columns of the item.
        constexpr int GW = 4 * MB;
        const int ew = warp - 2;
        const int grp = ew / GW;
        const int m = (ew % GW) >> 2;
        const int quad = warp & 3;
        const int row = m * 128 + quad * 32 + lane;   // query head j of the group at window position q
        const bool vrow = row < R;
        const int q = !vrow ? 0 : G.jm ? row % G.w : row / G.g;
        float seg_m = -INFINITY, seg_z = 0.f;
        // Relative to the segment's running reference seg_m, 2^(s - seg_m) sums the
        // same mass as an online max/rescale without a max pass.  32 columns of the
        // row, four sums of every fourth.
        auto sum32 = [&](const float* v) {
            const uint64_t sl2 = ptx::pack_f32x2(G.sl2, G.sl2), ref = ptx::pack_f32x2(-seg_m, -seg_m);
            uint64_t z01 = 0ull, z23 = 0ull;   // packed pairs: the roundings are the scalar operations'
#pragma unroll
            for (int c = 0; c < 32; c += 4) {
                const uint64_t a = ptx::fma_f32x2(ptx::pack_f32x2(v[c], v[c + 1]), sl2, ref);
                const uint64_t b = ptx::fma_f32x2(ptx::pack_f32x2(v[c + 2], v[c + 3]), sl2, ref);
                z01 = ptx::add_f32x2(z01, ptx::pack_f32x2(ptx::ex2(ptx::lo_f32(a)), ptx::ex2(ptx::hi_f32(a))));
                z23 = ptx::add_f32x2(z23, ptx::pack_f32x2(ptx::ex2(ptx::lo_f32(b)), ptx::ex2(ptx::hi_f32(b))));
            }
            return (ptx::lo_f32(z01) + ptx::hi_f32(z01)) + (ptx::lo_f32(z23) + ptx::hi_f32(z23));
        };
        // The same, `lim` of the columns visible (<= 0: none), for any of them: a sum
        // far above the reference (not below 2^64) and the segment's first columns
        // take the exact path.
        auto chunk = [&](const float* v, int lim) {
            if (lim <= 0) return;
            if (lim >= 32 && seg_m != -INFINITY) {
                const float z = sum32(v);
                if (z < 0x1p64f) {
                    seg_z += z;
                    if (seg_z >= 0x1p40f) {
                        // Keep the sum bounded: move a power of two into the reference.
                        const int k = ilogbf(seg_z);
                        seg_m += (float)k;
                        seg_z = ldexpf(seg_z, -k);
                    }
                    return;
                }
            }
            float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 32; ++c)
                if (c < lim) m4[c & 3] = fmaxf(m4[c & 3], v[c]);
            const float mu = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * G.sl2;
            float z4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int c = 0; c < 32; ++c)
                if (c < lim) z4[c & 3] += ptx::ex2(fmaf(v[c], G.sl2, -mu));
            merge_partial(seg_m, seg_z, make_float2(mu, (z4[0] + z4[1]) + (z4[2] + z4[3])));
        };

        int di = 0;
        uint32_t nb = 0u;   // items of this group so far
        bool aborted = false;
        while (!aborted) {
            // Each warp takes the next claimed chunk by itself (-1: no more work); the
            // group's warps go on with it or, when one of them gave up, leave together (the
            // barrier of an item would wait without a limit for a warp that has left).
            const int ds = di % kChunkSlots;
            int c = -1;
            bool got = true;
            if (lane == 0) {
                got = !(A.fault && ew == 1 && di == 0) &&
                      ptx::mbar_wait_abortable(&bars->c_full[ds], (di / kChunkSlots) & 1, &bars->abort_flag);
                if (got) {
                    c = bars->chunk[ds];
                    ptx::mbar_arrive(&bars->c_empty[ds]);
                } else {
                    raise_abort(bars, err);
                }
            }
            c = __shfl_sync(0xffffffffu, c, 0);
            if (ptx::named_bar_or(1 + grp, 32 * GW, !got)) break;
            ++di;
            if (c < 0) break;
            const int lay = c / per_layer, cl = c - lay * per_layer;
            const int i0 = cl * chunk_items, i1 = min(W, i0 + chunk_items);
            // The segment of chunk cl and head sh is number cl + sh of the layer: one of
            // the two grows from a segment to the next.
            float2* const segpart = A.segpart[lay];
            p.init(i0);
            int f = i0;   // the segment's first item
            for (int i = i0; i < i1; ++i) {
                if ((i - i0) % NB == grp) {
                    // One warp of the group polls, the others wait in the barrier (a
                    // polling warp takes issue slots from those that compute).
                    bool ok = true;
                    if (ew % GW == 0) {
                        ok = ptx::warp_wait(&bars->acc_full[grp], nb & 1u, &bars->abort_flag);
                        if (!ok && lane == 0) raise_abort(bars, err);
                    }
                    if (ptx::named_bar_or(1 + grp, 32 * GW, !ok)) {
                        aborted = true;
                        break;
                    }
                    ++nb;
                    ptx::tc_fence_after();
                    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(grp * 128 * MB + m * 128);
                    const int t0 = p.j * kTileT;
                    const int last = vrow ? min(p.L - 1, p.L - G.w + q) : -1;   // causal on the window part
                    const int nvalid = max(0, min(kTileT, last - t0 + 1));
                    // Four times 32 columns, straight through: the next columns' TMEM load
                    // is in flight while these are summed.  The sums count when every
                    // row of the warp has a reference that they stay near (all but a
                    // segment's first item and its last tile); else the columns are
                    // read again and taken one by one.
                    bool plain = nvalid == kTileT && seg_m != -INFINITY;
                    if (__all_sync(0xffffffffu, plain || !vrow)) {
                        float va[32], vb[32], z[4];
                        ptx::tmem_ld32(taddr, va);
                        ptx::tmem_wait_ld();
                        ptx::tmem_ld32(taddr + 32, vb);
                        z[0] = sum32(va);
                        ptx::tmem_wait_ld();
                        ptx::tmem_ld32(taddr + 64, va);
                        z[1] = sum32(vb);
                        ptx::tmem_wait_ld();
                        ptx::tmem_ld32(taddr + 96, vb);
                        z[2] = sum32(va);
                        ptx::tmem_wait_ld();
                        z[3] = sum32(vb);
                        const float s0 = seg_z + z[0], s1 = s0 + z[1], s2 = s1 + z[2], s3 = s2 + z[3];
                        plain = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])) < 0x1p64f &&
                                fmaxf(fmaxf(s0, s1), fmaxf(s2, s3)) < 0x1p40f && s3 == s3;
                        plain = __all_sync(0xffffffffu, plain || !vrow);
                        if (plain) seg_z = s3;
                    } else {
                        plain = false;
                    }
                    if (!plain) {
#pragma unroll 1
                        for (int c = 0; c < kTileT; c += 32) {
                            float v[32];
                            ptx::tmem_ld32(taddr + (uint32_t)c, v);
                            ptx::tmem_wait_ld();
                            chunk(v, nvalid - c);
                        }
                    }
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(&bars->acc_empty[grp]);
                }
                if (i + 1 >= i1 || p.last_of_head()) {   // the segment ends
                    // By item: the group's first item of the segment, if it has one (a
                    // chunk starts at a multiple of NB).
                    const int slot = A.by_item ? f + ((grp - f) & (NB - 1)) : (cl + p.head()) * NB + grp;
                    if (vrow && (!A.by_item || slot <= i)) segpart[(size_t)slot * R + row] = make_float2(seg_m, seg_z);
                    f = i + 1;
                    seg_m = -INFINITY;
                    seg_z = 0.f;
                }
                p.next();
            }
        }
    }

    // ---------------------------------------------------------------- teardown
    if (warp == 1 && lane == 0) ptx::mbar_wait(&bars->mma_done, 0, 50000000ull);
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    if (warp == 1) ptx::tmem_dealloc(tmem, kTmemCols);
}

// (m_r, Z_r) of every row of (s, h) from the score kernel's partials: its
// segments lie in the consecutive chunks that hold its items, the groups' partials
// of a segment merge first, then the segments in item order.  Grid (Hkv, batch,
// layers), one thread per row, as the score kernel orders them.
template <int NB>
__global__ void __launch_bounds__(256) rowstat_kernel(const __grid_constant__ Geometry G, const __grid_constant__ Group A,
                                                      int chunk, int by_item, int* claim, int wait_prev) {
    // The window launch that follows may start; it waits for this grid.
    if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    // wait_prev: a programmatic dependent of the score launch right before it on
    // the stream, whose partials are read only after that grid has completed.
    // Otherwise the partials come through a full dependency and the stream's
    // previous kernel (if a programmatic predecessor at all) is not waited for.
    const int h = blockIdx.x, s = blockIdx.y, lay = blockIdx.z, r = threadIdx.x;
    const int* __restrict__ cu = A.io[0].cu;   // an input: read before the wait
    int ib = 0;
    for (int b = 0; b < s; ++b) ib += tiles_of(__ldg(&cu[b + 1]) - __ldg(&cu[b])) * G.Hkv;
    const int nt = tiles_of(__ldg(&cu[s + 1]) - __ldg(&cu[s]));
    if (wait_prev) asm volatile("griddepcontrol.wait;\n" ::: "memory");
    // The score grid has completed: its chunk counter is free for the next launch.
    if (h == 0 && s == 0 && lay == 0 && r == 0) *claim = 0;
    if (r >= G.R) return;
    const int sh = s * G.Hkv + h;
    ib += h * nt;
    const int seg0 = ib / chunk + sh, seg1 = (ib + nt - 1) / chunk + sh;
    const float2* src = A.segpart[lay] + r;
    float M = -INFINITY, Z = 0.f;
    constexpr int kSegs = 16 / NB;   // segments whose loads are issued together
    for (int g0 = seg0; g0 <= seg1; g0 += kSegs) {
        float2 pz[kSegs][NB];
#pragma unroll
        for (int k = 0; k < kSegs; ++k)
#pragma unroll
            for (int a = 0; a < NB; ++a) {
                const int c0 = (g0 + k - sh) * chunk, f = max(c0, ib), f1 = min(c0 + chunk, ib + nt);
                const int slot = by_item ? f + ((a - f) & (NB - 1)) : (g0 + k) * NB + a;
                pz[k][a] = g0 + k <= seg1 && (!by_item || slot < f1) ? __ldcg(&src[(size_t)slot * G.R])
                                                                     : make_float2(-INFINITY, 0.f);
            }
#pragma unroll
        for (int k = 0; k < kSegs; ++k) {
            float ms = pz[k][0].x, zs = pz[k][0].y;
#pragma unroll
            for (int a = 1; a < NB; ++a) merge_partial(ms, zs, pz[k][a]);
            merge_partial(M, Z, make_float2(ms, zs));
        }
    }
    const int q = G.jm ? r % G.w : r / G.g, j = G.jm ? r / G.w : r - q * G.g;
    A.sl[lay].rowstat[(size_t)sh * G.R + q * G.g + j] = make_float2(M, Z);
}

// Row statistics from the caller's log-sum-exp of each window query row (the
// denominator its prefill attention already computed): row r = q * g + j of KV
// head h is query head h * g + j at window position q.  Grid (Hkv, batch, layers).
__global__ void __launch_bounds__(256) rowstat_lse_kernel(const __grid_constant__ Geometry G,
                                                          const __grid_constant__ Group A) {
    // The window launch that follows may start; it waits for this grid before reading.
    if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int h = blockIdx.x, s = blockIdx.y, lay = blockIdx.z, r = threadIdx.x;
    if (r >= G.R) return;
    const int q = r / G.g, j = r - q * G.g;
    const float v = __ldg(&A.io[lay].lse[((size_t)s * G.w + q) * G.Hq + h * G.g + j]);
    A.sl[lay].rowstat[((size_t)s * G.Hkv + h) * G.R + r] = make_float2(v * 1.4426950408889634f, 1.f);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

int mblocks(const Geometry& g) { return g.R > 128 ? 2 : 1; }

// Two query buffers of R rows, the K ring, the barriers.  (An M-block's rows past R
// are whatever follows the buffer; their accumulator rows are not read.)
size_t smem_bytes_with(const Geometry& g, int kst) {
    return 1024 + 4 * (size_t)g.R * 128 + (size_t)kst * kKStageBytes + sizeof(Barriers);
}

int kstages_for(const Geometry& g) {
    int kst = kKStages;
    while (kst > 2 && smem_bytes_with(g, kst) > (size_t)kMaxSmem) --kst;
    return kst;
}

// A layer's partials lie by segment and group (slot segment * NB + group, every one
// written), or by item where that takes less room, i.e. with fewer than about eight
// tiles a head: in the slot of the group's first item of the segment.
size_t partial_slots(const Geometry& g, size_t tiles) {
    return (tiles * g.Hkv / kChunkSmall + 1 + (size_t)g.batch * g.Hkv) * (4 / mblocks(g));
}

int partials_by_item(const Geometry& g, size_t tiles) { return tiles * g.Hkv < partial_slots(g, tiles); }

size_t smem_bytes_for(const Geometry& g) { return smem_bytes_with(g, kstages_for(g)); }

}  // namespace

size_t score_smem_bytes(const Geometry& g) { return smem_bytes_for(g); }

size_t score_partial_bytes(const Geometry& g, size_t tiles) {
    return std::min(tiles * g.Hkv, partial_slots(g, tiles)) * g.R * sizeof(float2);
}

cudaError_t configure_score(const Geometry& g) {
    // Per-function attribute shared by every handle: the largest supported geometry.
    size_t need = 0;
    for (int R = 8; R <= 256; R += 8) {
        Geometry gr = g;
        gr.R = R;
        if (smem_bytes_for(gr) > need) need = smem_bytes_for(gr);
    }
    cudaError_t e = cudaFuncSetAttribute(score_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(score_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
    return e;
}

cudaError_t plan_score(const Geometry& g, const Group& gr, int num_sms, ScorePlan* plan) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    for (int l = 0; l < gr.nl; ++l) {
        {
            cuuint64_t dims[3] = {(cuuint64_t)kHeadDim, (cuuint64_t)g.Hkv, (cuuint64_t)g.total_tokens};
            cuuint64_t strides[2] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)g.Hkv * kHeadDim * 2};
            cuuint32_t box[3] = {64, 1, (cuuint32_t)kTileT};
            cuuint32_t es[3] = {1, 1, 1};
            if (enc(&plan->kmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(gr.io[l].k), dims,
                    strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        }
        {
            // A KV head's rows in one box, or a box for each query head (load_queries).
            cuuint64_t dims[4] = {(cuuint64_t)kHeadDim, (cuuint64_t)g.Hq, (cuuint64_t)g.w, (cuuint64_t)g.batch};
            cuuint64_t strides[3] = {(cuuint64_t)kHeadDim * 2, (cuuint64_t)g.Hq * kHeadDim * 2,
                                     (cuuint64_t)g.w * g.Hq * kHeadDim * 2};
            cuuint32_t box[4] = {64, (cuuint32_t)(g.jm ? 1 : g.g), (cuuint32_t)g.w, 1};
            cuuint32_t es[4] = {1, 1, 1, 1};
            if (enc(&plan->qmap[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(gr.io[l].q), dims,
                    strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
                return cudaErrorInvalidValue;
        }
    }
    plan->items = g.total_tiles * g.Hkv;
    // At most all but kScoreReserveSms SMs (the rest run the window, heads and
    // selection kernels of neighbouring layers, which cannot share an SM with a
    // score CTA) and at most one CTA per chunk.
    const int usable = num_sms > 2 * kScoreReserveSms ? num_sms - kScoreReserveSms : num_sms;
    // Chunks of kChunkLarge items when one layer's still give every usable SM one,
    // else of kChunkSmall (measured: larger chunks reload the query rows less
    // often, smaller ones leave fewer SMs idle on small layers).  The rule looks at
    // one layer, so that a row's statistics do not depend on how many layers
    // share a launch.
    plan->chunk = plan->items / kChunkLarge >= usable ? kChunkLarge : kChunkSmall;
    const int nchunks = (plan->items + plan->chunk - 1) / plan->chunk * gr.nl;
    plan->grid = nchunks < usable ? nchunks : usable;
    plan->by_item = partials_by_item(g, g.total_tiles);
    plan->threads = kScoreThreads;
    plan->mb = mblocks(g);
    plan->smem = smem_bytes_for(g);
    plan->num_sms = num_sms;
    return cudaSuccess;
}

namespace {

cudaLaunchConfig_t launch_config(dim3 grid, int threads, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr,
                                 bool programmatic) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = programmatic ? 1 : 0;
    return cfg;
}

}  // namespace

cudaError_t launch_rowstat(const ScorePlan& plan, const Geometry& g, const Group& gr, int* claim, cudaStream_t st,
                           bool programmatic, bool after_score) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config(dim3(g.Hkv, g.batch, gr.nl), 256, 0, st, &attr, programmatic);
    if (plan.mb == 2) return cudaLaunchKernelEx(&cfg, rowstat_kernel<2>, g, gr, plan.chunk, plan.by_item, claim, after_score ? 1 : 0);
    return cudaLaunchKernelEx(&cfg, rowstat_kernel<4>, g, gr, plan.chunk, plan.by_item, claim, after_score ? 1 : 0);
}

cudaError_t launch_rowstat_lse(const Geometry& g, const Group& gr, cudaStream_t st, bool programmatic) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config(dim3(g.Hkv, g.batch, gr.nl), 256, 0, st, &attr, programmatic);
    return cudaLaunchKernelEx(&cfg, rowstat_lse_kernel, g, gr);
}

cudaError_t launch_score(const ScorePlan& plan, const Geometry& g, const Group& gr, const Scratch& sc, int* claim,
                         cudaStream_t st, bool after_own_launch) {
    ScoreArgs a{};
    for (int l = 0; l < gr.nl; ++l) {
        a.kmap[l] = plan.kmap[l];
        a.qmap[l] = plan.qmap[l];
        a.segpart[l] = gr.segpart[l];
    }
    a.G = g;
    a.cu = gr.io[0].cu;
    a.err = sc.err;
    a.nl = gr.nl;
    a.W = plan.items;
    a.kst = kstages_for(g);
    a.claim = claim;
    a.chunk = plan.chunk;
    a.by_item = plan.by_item;
    a.fault = test_fault() == 2 ? 1 : 0;
    // after_own_launch: the previous kernel on the stream is the previous
    // group's launch, whose results this grid does not read; the launch is then
    // its programmatic dependent and never executes griddepcontrol.wait.
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = launch_config(dim3(plan.grid), plan.threads, plan.smem, st, &attr, after_own_launch);
    if (plan.mb == 2) return cudaLaunchKernelEx(&cfg, score_kernel<2>, a);
    return cudaLaunchKernelEx(&cfg, score_kernel<1>, a);
}

}  // namespace kvec
