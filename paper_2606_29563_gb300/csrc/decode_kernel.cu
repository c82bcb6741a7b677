// One decoding step of attention over the compacted KV cache that the
// selection leaves behind.  Section 4.1: after the per-head top-B selection the
// keys and values of the kept tokens are the cache the subsequent decoding
// steps read; Section 5.3 measures decoding over it.  For sequence s and query
// head hq (KV head h = hq / g):
//   out[s][hq] = sum_{j < n_s} softmax_j(scale * <q[s][hq], k[s][h][j]>) v[s][h][j].
//
// Every K/V row is read once: HBM-bound when there are many rows, bound by one
// memory latency and the launch when there are few.  Each warp works on its
// own: it streams blocks of eight rows (2 KB of K, 2 KB of V) through a private
// cp.async ring, so no block barrier stands between loads and arithmetic.  The
// logits of a block and of up to eight query heads are one m16n8k16 tile (half
// of its rows unused; bf16 products with fp32 sums, the operands' own type), so
// no dot product is summed over lanes; tcgen05 tiles of 64 rows and more would
// leave most of this shape empty.  The online softmax rescales only when a
// maximum moves, and the fp32 weights meet the value rows in packed fp32 pairs
// (fma.rn.f32x2), a half-warp per row.
//
// The warps of a CTA merge in shared memory, the CTAs of a (sequence, KV head)
// over distributed shared memory: one launch does the whole step.
//
// Measured (one GB300, caches larger than L2, CUDA graph of many calls), against
// the 64-row tiles with five block barriers each that this replaced: 64
// sequences x 8 KV heads x 1024-2048 rows, g = 4: 179 -> 68 us per call
// (5.9 TB/s, 86 % of the measured copy rate; bound by HBM), g = 8: 281 -> 104 us
// (3.9 TB/s; bound by the fp32 pair multiply-adds of the weighted rows); one
// sequence x 512 rows, g = 4: 7.1 -> 4.7 us (launch, lengths, one load latency,
// two merges).  With fp32 dot products summed over lanes in place of the matrix
// tile: 75, 124 and 4.7 us.
#include "kvec_internal.cuh"
#include "sm100_ptx.cuh"

#include <cooperative_groups.h>

namespace kvec {

namespace {

namespace cg = cooperative_groups;

constexpr int kDecBlock = 8;                          // cached rows per ring stage
constexpr int kDecStageBytes = 2 * kDecBlock * kHeadDim * 2;   // K rows, then V rows
constexpr int kDecMaxSplits = 8;                      // CTAs per (sequence, KV head): a portable cluster
// The maximum before the first logit: the lowest finite value, so that a logit of minus
// infinity gets the weight 2^-inf = 0 there too, and not 2^(-inf + inf).
constexpr float kNoLogit = -3.402823466e38f;

struct DecArgs {
    const __nv_bfloat16* q;      // [batch][Hq][d]
    const __nv_bfloat16* k;      // [batch][Hkv][cap][d]
    const __nv_bfloat16* v;
    const int* lens;             // [batch]
    float* out;                  // [batch][Hq][d]
    int Hq, Hkv, g, cap;
    float sl2;                   // softmax scale * log2(e)
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    // src_bytes 0: sixteen zero bytes are written and src is not read.
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Four 8x8 bf16 matrices, one row address per lane.
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t* r) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// d += A B for the upper eight rows of a 16 x 16 A tile (the lower eight are zero).
__device__ __forceinline__ void mma_rows8(float* d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi) {
    [[maybe_unused]] float z2, z3;
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %5}, {%7, %8}, "
        "{%9, %10, %11, %11};\n"
        : "=f"(d[0]), "=f"(d[1]), "=f"(z2), "=f"(z3)
        : "r"(a_lo), "r"(0u), "r"(a_hi), "r"(b_lo), "r"(b_hi), "f"(d[0]), "f"(d[1]), "f"(0.f));
}

// The two bf16 of a word as an fp32 pair.
__device__ __forceinline__ uint64_t bf16x2_pair(uint32_t w) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "r"(w << 16), "r"(w & 0xffff0000u));
    return r;
}

// GP: query heads per KV head, padded to a power of two.  NW: warps, ST: ring
// stages per warp, NC: CTAs per SM.
template <int GP_, int NW_, int ST_, int NC_>
struct DecConfig {
    static constexpr int GP = GP_, NW = NW_, ST = ST_, NC = NC_;
    static constexpr int kThreads = 32 * NW;
    static constexpr int kRing = NW * ST * kDecStageBytes;
    static constexpr int kAcc = NW * GP * kHeadDim * 4;   // the warps' outputs, over the ring
    static constexpr int kSmem = kRing > kAcc ? kRing : kAcc;
};

template <class C>
__global__ void __launch_bounds__(C::kThreads, C::NC) decode_kernel(const __grid_constant__ DecArgs A) {
    constexpr int GP = C::GP, ST = C::ST, kDecWarps = C::NW, kDecThreads = C::kThreads;
    extern __shared__ __align__(128) uint8_t dec_smem[];
    __shared__ __align__(16) uint64_t sw[kDecWarps][kDecBlock][GP < 2 ? 2 : GP];   // a block's weights, as pairs (p, p)
    __shared__ float wm[kDecWarps][GP], wl[kDecWarps][GP];          // the warps' maxima and sums
    __shared__ __align__(16) float co[GP][kHeadDim];                // this CTA's outputs, unnormalised
    __shared__ float cm[GP], cl[GP];
    cg::cluster_group cluster = cg::this_cluster();
    const int splits = (int)cluster.num_blocks(), sp = (int)cluster.block_rank();
    const int h = blockIdx.y, s = blockIdx.z;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int half = lane >> 4, l16 = lane & 15;
    const int g = A.g, cap = A.cap;
    // A launch after another decoding step may have started early: its inputs
    // are read only once everything before it has completed.
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    const int n = min(max(__ldg(&A.lens[s]), 0), cap);
    // Blocks of eight rows, an even contiguous share per CTA, dealt to its warps.
    const int nb = (n + kDecBlock - 1) / kDecBlock;
    const int b_end = (int)((long long)nb * (sp + 1) / splits);
    const int b0 = (int)((long long)nb * sp / splits) + warp;
    const size_t kv_base = ((size_t)s * A.Hkv + h) * (size_t)cap * kHeadDim;
    const __nv_bfloat16* kg = A.k + kv_base + l16 * 8;
    const __nv_bfloat16* vg = A.v + kv_base + l16 * 8;
    const uint32_t ring = ptx::smem_u32(dec_smem) + warp * ST * kDecStageBytes;
    // Row 2 i + half of the block, i < 4.  The 16-byte pieces of K row r are
    // permuted by r, so that the eight rows of a matrix load lie in different banks.
    auto load = [&](int st, int b) {
        const uint32_t dst = ring + st * kDecStageBytes;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 2 * i + half, row = b * kDecBlock + r;
            const bool in = row < n;                       // zeros past the valid rows, never read
            const size_t ofs = (size_t)(in ? row : 0) * kHeadDim;
            cp_async16(dst + r * 256 + ((l16 ^ r) << 4), kg + ofs, in ? 16u : 0u);
            cp_async16(dst + 2048 + r * 256 + (l16 << 4), vg + ofs, in ? 16u : 0u);
        }
    };
#pragma unroll
    for (int i = 0; i < ST - 1; ++i) {
        if (b0 + i * kDecWarps < b_end) load(i, b0 + i * kDecWarps);
        cp_async_commit();
    }
    // The group's query rows as the tile's column operand (zeros past g): head
    // lane / 4, dims 16 kk + 2 (lane % 4) and the next, and the same eight higher.
    uint32_t qb[8][2];
    {
        const int j = lane >> 2;
        const uint32_t* qr = reinterpret_cast<const uint32_t*>(A.q + ((size_t)s * A.Hq + h * g + (j < g ? j : 0)) * kHeadDim) +
                             (lane & 3);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
            qb[kk][0] = j < g ? __ldg(qr + 8 * kk) : 0u;
            qb[kk][1] = j < g ? __ldg(qr + 8 * kk + 4) : 0u;
        }
    }
    uint64_t acc[GP][4];   // this lane's eight dims of the outputs, over its half-warp's rows
#pragma unroll
    for (int j = 0; j < GP; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[j][c] = 0ull;
    // This lane's logits: row lane / 4 of the block, heads j0 and j0 + 1.
    const int xr = lane >> 2, j0 = 2 * (lane & 3);
    float m[2] = {kNoLogit, kNoLogit}, l[2] = {0.f, 0.f};
    int st = 0;
    for (int b = b0; b < b_end; b += kDecWarps) {
        cp_async_wait<ST - 2>();
        __syncwarp();
        const uint32_t src = ring + st * kDecStageBytes;
        // Logits: rows lane & 7, pieces 4 kq + lane / 8 (two steps of 16 dims a load); two sums, added.
        float xa[2] = {0.f, 0.f}, xb[2] = {0.f, 0.f};
#pragma unroll
        for (int kq = 0; kq < 4; ++kq) {
            uint32_t a[4];
            ldmatrix_x4(src + (lane & 7) * 256 + (((4 * kq + (lane >> 3)) ^ (lane & 7)) << 4), a);
            mma_rows8(xa, a[0], a[1], qb[2 * kq][0], qb[2 * kq][1]);
            mma_rows8(xb, a[2], a[3], qb[2 * kq + 1][0], qb[2 * kq + 1][1]);
        }
        // Online softmax of the block.
        const bool valid = b * kDecBlock + xr < n;
        float x[2], mn[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            x[c] = valid ? (xa[c] + xb[c]) * A.sl2 : -INFINITY;
            float t = x[c];
            t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 4));
            t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 8));
            t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, 16));
            mn[c] = fmaxf(m[c], t);
        }
        if (__any_sync(0xffffffffu, mn[0] != m[0] || mn[1] != m[1])) {
            float corr[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                corr[c] = ptx::ex2(m[c] - mn[c]);   // 0 from kNoLogit on
                l[c] *= corr[c];
                m[c] = mn[c];
            }
#pragma unroll
            for (int j = 0; j < GP; ++j) {
                const float cj = __shfl_sync(0xffffffffu, corr[j & 1], j >> 1);
                const uint64_t c2 = ptx::pack_f32x2(cj, cj);
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[j][c] = ptx::mul_f32x2(acc[j][c], c2);
            }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            x[c] = ptx::ex2(x[c] - m[c]);
            l[c] += x[c];
        }
        if (j0 < GP) {
            sw[warp][xr][j0] = ptx::pack_f32x2(x[0], x[0]);
            sw[warp][xr][j0 + 1] = ptx::pack_f32x2(x[1], x[1]);
        }
        __syncwarp();
        // Weighted value rows, row 2 i + half.
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 2 * i + half;
            const uint4 w = ptx::ld_shared_v4(src + 2048 + r * 256 + (l16 << 4));
            const uint64_t v0 = bf16x2_pair(w.x), v1 = bf16x2_pair(w.y), v2 = bf16x2_pair(w.z), v3 = bf16x2_pair(w.w);
#pragma unroll
            for (int j = 0; j < GP; ++j) {
                const uint64_t p2 = sw[warp][r][j];
                acc[j][0] = ptx::fma_f32x2(p2, v0, acc[j][0]);
                acc[j][1] = ptx::fma_f32x2(p2, v1, acc[j][1]);
                acc[j][2] = ptx::fma_f32x2(p2, v2, acc[j][2]);
                acc[j][3] = ptx::fma_f32x2(p2, v3, acc[j][3]);
            }
        }
        // The next block for the stage that the previous step left (every lane has
        // passed this step's __syncwarp, so that step's reads are done).
        const int nxt = st == 0 ? ST - 1 : st - 1;
        if (b + (ST - 1) * kDecWarps < b_end) load(nxt, b + (ST - 1) * kDecWarps);
        cp_async_commit();
        st = st + 1 == ST ? 0 : st + 1;
    }
    cp_async_wait<0>();
    __syncthreads();   // every warp is done with the ring
    // The warp's sums over its rows, and its outputs (both half-warps hold every dim).
    float* wacc = reinterpret_cast<float*>(dec_smem) + (size_t)warp * GP * kHeadDim;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 4);
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 8);
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 16);
        if (lane < 4 && j0 + c < GP) {
            wm[warp][j0 + c] = m[c];
            wl[warp][j0 + c] = l[c];
        }
    }
#pragma unroll
    for (int j = 0; j < GP; ++j) {
        float f[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            f[2 * c] = ptx::lo_f32(acc[j][c]);
            f[2 * c + 1] = ptx::hi_f32(acc[j][c]);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) f[c] += __shfl_xor_sync(0xffffffffu, f[c], 16);
        const float4 o = half ? make_float4(f[4], f[5], f[6], f[7]) : make_float4(f[0], f[1], f[2], f[3]);
        *reinterpret_cast<float4*>(wacc + j * kHeadDim + l16 * 8 + half * 4) = o;
    }
    __syncthreads();
    // The CTA's (max, sum, output) per head.
    for (int i = tid; i < g * kHeadDim; i += kDecThreads) {
        const int j = i / kHeadDim, c = i - j * kHeadDim;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) M = fmaxf(M, wm[w][j]);
        float L = 0.f, O = 0.f;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) {
            if (wm[w][j] == kNoLogit) continue;   // no row with a logit above minus infinity
            const float e = ptx::ex2(wm[w][j] - M);
            L = fmaf(e, wl[w][j], L);
            O = fmaf(e, reinterpret_cast<const float*>(dec_smem)[((size_t)w * GP + j) * kHeadDim + c], O);
        }
        if (splits == 1) {
            A.out[((size_t)s * A.Hq + h * g + j) * kHeadDim + c] = L > 0.f ? O / L : 0.f;
        } else {
            co[j][c] = O;
            if (c == 0) {
                cm[j] = M;
                cl[j] = L;
            }
        }
    }
    if (splits == 1) return;
    cluster.sync();
    // CTA r merges query heads r, r + splits, ... over the cluster:
    // out = sum_c 2^(m_c - M) o_c / sum_c 2^(m_c - M) l_c, zeros for an empty cache
    // (and where every logit is minus infinity).
    for (int i = tid; sp + (i / kHeadDim) * splits < g; i += kDecThreads) {
        const int j = sp + (i / kHeadDim) * splits, c = i % kHeadDim;
        float mc[kDecMaxSplits], M = -INFINITY;
#pragma unroll
        for (int r = 0; r < kDecMaxSplits; ++r) {
            mc[r] = r < splits ? *cluster.map_shared_rank(&cm[j], r) : -INFINITY;
            M = fmaxf(M, mc[r]);
        }
        float L = 0.f, O = 0.f;
#pragma unroll
        for (int r = 0; r < kDecMaxSplits; ++r) {
            if (mc[r] <= kNoLogit) continue;
            const float e = ptx::ex2(mc[r] - M);
            L = fmaf(e, *cluster.map_shared_rank(&cl[j], r), L);
            O = fmaf(e, *cluster.map_shared_rank(&co[j][c], r), O);
        }
        A.out[((size_t)s * A.Hq + h * g + j) * kHeadDim + c] = L > 0.f ? O / L : 0.f;
    }
    cluster.sync();   // no CTA leaves while another still reads its shared memory
}

using Dec1 = DecConfig<1, 8, 3, 2>;
using Dec2 = DecConfig<2, 8, 3, 2>;
using Dec4 = DecConfig<4, 8, 3, 2>;
using Dec8 = DecConfig<8, 8, 3, 2>;

template <class C>
cudaError_t configure_one() {
    return cudaFuncSetAttribute(decode_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmem);
}

// CTAs per (sequence, KV head): the largest cluster that still fits the device's
// resident CTAs in one wave, with more than 32 rows to a CTA.  Measured, in us
// per call (g = 4): 64 pairs x 128-256 rows 5.3 / 6.2 / 5.5 / 9.8 with 1 / 2 / 4 /
// 8 CTAs (two waves at 8); 128 pairs x 256-512 rows 10.5 / 9.9 / 13.3 / 20.4; 8
// pairs x 512 rows 7.0 / 6.0 / 4.7 / 4.7, x 64 rows 2.9 / 3.8 / 3.8 / 4.2.
template <class C>
cudaError_t launch_one(const DecArgs& a, int batch, int num_sms, cudaStream_t st) {
    int splits = 1;
    while (splits < kDecMaxSplits && (long long)batch * a.Hkv * splits * 2 <= C::NC * num_sms &&
           a.cap > 32 * 2 * splits)
        splits *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(splits, a.Hkv, batch);
    cfg.blockDim = dim3(C::kThreads);
    cfg.dynamicSmemBytes = C::kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, decode_kernel<C>, a);
}

}  // namespace

cudaError_t configure_decode() {
    cudaError_t e = configure_one<Dec1>();
    if (e == cudaSuccess) e = configure_one<Dec2>();
    if (e == cudaSuccess) e = configure_one<Dec4>();
    if (e == cudaSuccess) e = configure_one<Dec8>();
    return e;
}

cudaError_t launch_decode(const DecodeIO& io, int num_sms, cudaStream_t st) {
    DecArgs a{};
    a.q = io.q;
    a.k = io.k;
    a.v = io.v;
    a.lens = io.lens;
    a.out = io.out;
    a.Hq = io.Hq;
    a.Hkv = io.Hkv;
    a.g = io.Hq / io.Hkv;
    a.cap = io.cap;
    a.sl2 = io.scale * 1.4426950408889634f;
    if (a.g <= 1) return launch_one<Dec1>(a, io.batch, num_sms, st);
    if (a.g <= 2) return launch_one<Dec2>(a, io.batch, num_sms, st);
    if (a.g <= 4) return launch_one<Dec4>(a, io.batch, num_sms, st);
    return launch_one<Dec8>(a, io.batch, num_sms, st);
}

}  // namespace kvec
