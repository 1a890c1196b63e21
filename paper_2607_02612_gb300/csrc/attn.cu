// Size-aware attention over a ragged batch: the transformer block that consumes a compacted
// batch (Algorithm 1, Block_b), with the proportional attention of ToMe so that a merged
// token of size s weighs like the s tokens it replaced.  For every sample, head h and query
// row m of the sample:
//   out[m, h] = sum_j softmax_j(q_m . k_j / sqrt(dh) + log s_j) v_j.
//
// One CTA per (pair of query tiles, head, sample), dh = 64, bf16; a query tile is 128 rows and has a
// warpgroup of its own, one thread per row.  One more warp per tile issues its tensor-core products; the
// query tiles and blocks of 64 keys (K and V rows) come by TMA through a ring of four stages (128-byte
// swizzle; Q and K are K-major operands; V, rows of keys with the dims contiguous, is the MN-major B
// operand of the second product as it lies).  Per tile and key block: S = Q K^T (M = 128, N = keys
// rounded up to 16) into tensor-memory columns [0, 64) of the tile; the thread of a row reads it, forms
// P = 2^(S scale + log2 s_j - m) (ex2.approx), adds its float32 sum and writes P as bf16 over S's first 32
// columns; O += P V (A = P from tensor memory) accumulates in columns [64, 128), and the next block's S
// follows it in the same issue order, so one barrier per block tells the warpgroup that its S is
// ready and its O complete.
//
// The shift is m = max_j S scale + max_j log2 s_j over the blocks so far (an upper bound of the row
// maximum within log2(max s / min s), so sizes within a factor 2^100 of each other keep every probability a
// normal float); where it grows, the warp rescales its rows of O and their sums.  P is rounded to bf16
// (the operand type of the second product), the sum is taken before that; the row's largest
// probabilities end as 2^0, exact in bf16 (letting the shift lag, to rescale rarely, raised the error
// against 64 bits at 577 tokens from 2.2e-3 to 2.3e-3).
//
// What bounds it: the softmax's instructions (about six issue slots per logit and row of 32) and, for short
// samples, the way to the first product (metadata, barriers, loads: 5 of 15 thousand cycles at 197
// tokens); two CTAs (four warpgroups) per SM hide each other's waits for the products.  The forms before
// it, one CTA per (head, sample) with block-wide barriers between load, product, softmax and product,
// idled in them, and samples past 256 tokens formed S twice (a pass for the maximum).  256 samples of
// 100 to 197 tokens x 6 heads: 62 -> 43 us; 128 of 577 x 16 heads: 769 -> 307 us (0.57 PFLOP/s; 317 with
// the loops over key blocks and rows unrolled by the compiler).
// Measured and not taken: halves of 32 keys with two S buffers (495 us at 577 tokens: twice the barriers),
// a first pass for the maximum with two S buffers (440), the shift allowed to lag by 2^8 (309).
//
// Every wait on an mbarrier is bounded; on a timeout the CTA raises FUSION_DEV_TIMEOUT, skips
// its outputs, waits (bounded) for the operations it started and frees its tensor memory.
#include "launch.h"
#include "tc.cuh"

namespace fz {
namespace {

constexpr int kAttnDh = 64;
constexpr int kAttnMaxN = FUSION_ATTN_MAX_TOKENS;
constexpr uint32_t kQTileBytes = 128 * 128;   // 128 rows x 64 bf16
constexpr int kKeyBlock = 64;
constexpr uint32_t kKeyBytes = kKeyBlock * 128;   // 64 key rows (K or V)
constexpr int kStages = 4;      // K and V blocks in flight, at most
constexpr uint32_t kTileCols = 128;           // tensor-memory columns of a query tile: S (P over it), O at 64

__device__ __forceinline__ float ex2(float x) {   // 2^x, one MUFU instruction (2^-inf = 0)
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// max(a, b, c) in one instruction (three-source max.f32 of sm_100 and later); exact
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
struct AttnMaps {
    CUtensorMap b128, b64, b32, b8;   // qkv rows, boxes of 64 dims x 128 / 64 / 32 / 8 rows, 128-byte swizzle
};

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
// D (tensor memory) += A (tensor memory, 128 lanes x 16 bf16 packed in 8 columns) x B (shared memory).
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{ .reg .pred p; setp.ne.b32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p; }" ::"r"(tmem_d),
        "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}


__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t *r) {   // no wait: tmem_ld_wait
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Stages of the K and V rings: all of the call's blocks, up to four.
__host__ __device__ inline int attn_stages(int max_tokens) {
    const int nb = (max_tokens + kKeyBlock - 1) / kKeyBlock;
    return nb < kStages ? nb : kStages;
}
// Position in a ring of n stages: the stage, and the parity of its current use.
struct RingPos {
    int st = 0;
    uint32_t par = 0;
    __device__ __forceinline__ void next(int n) {
        if (++st == n) {
            st = 0;
            par ^= 1u;
        }
    }
};

// mbar_wait by a whole warp, with one outcome.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity) {
    return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity));
}

// q: query tiles; k, v: key / value blocks landed; s: a tile's S complete (and its O up to the block
// before); free: a stage's products done (each tile's); p: a tile's S replaced by P
struct AttnBars {
    unsigned long long q[2], drain[2], k[kStages], v[kStages], s[2], free[kStages], p[2];
};

// The softmax of one block for one row: S (64 logits in v) -> P over S's first columns; returns the sum
// of the probabilities as an (even, odd) pair.  kSized: log2 sizes from lz, else all zero.
template <bool kSized>
__device__ __forceinline__ float2 block_probs(const uint32_t (&v)[64], uint32_t taddr, const float *lz, float m) {
    constexpr float kScale2 = 0.18033688011112042f;   // log2(e) / sqrt(64)
    float2 sum = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        uint32_t pk[8];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
            const int j = 16 * c + e;
            const float2 sv = make_float2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
            float2 x;
            if constexpr (kSized)
                x = __fadd2_rn(__ffma2_rn(sv, make_float2(kScale2, kScale2), *reinterpret_cast<const float2 *>(lz + j)),
                               make_float2(-m, -m));
            else
                x = __ffma2_rn(sv, make_float2(kScale2, kScale2), make_float2(-m, -m));
            const float2 pr = make_float2(ex2(x.x), ex2(x.y));
            sum = __fadd2_rn(sum, pr);
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(pr.x, pr.y);
            pk[e >> 1] = *reinterpret_cast<const uint32_t *>(&b2);
        }
        tmem_st8(taddr + 8u * c, pk);
    }
    return sum;
}

// NWG: query tiles (warpgroups) per CTA.
template <int NWG>
__global__ void __launch_bounds__(NWG * 160, NWG == 2 ? 2 : 3)
    k_attn_tc(const __grid_constant__ AttnMaps maps, AttnParams p, int n_part) {
    extern __shared__ unsigned char sm_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) AttnBars bar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail, s_kv;             // s_kv: key blocks whose loads were issued
    __shared__ float red_max[NWG * 4], red_min[NWG * 4];
    __shared__ __align__(16) float lsz[kAttnMaxN];   // log2 of the key sizes

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == NWG * 4 && lane < 4)   // the descriptors travel while the sample's metadata loads
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.b128 + lane)) : "memory");
    const int part = blockIdx.x % n_part, h = blockIdx.x / n_part, i = blockIdx.y;
    const int B = device_batch(p.in);
    if (B < 0) {
        if (blockIdx.x == 0 && i == 0 && tid == 0) raise_status(p.status, FUSION_DEV_BAD_BATCH);
        return;
    }
    if (i >= B) return;
    const int o0 = p.in.offsets[i], n = p.in.offsets[i + 1] - o0;
    if (o0 < 0 || n < 1 || n > p.in.max_tokens || n > kAttnMaxN || (long long)o0 + n > p.in.max_rows) {
        if (blockIdx.x == 0 && tid == 0) raise_status(p.status, FUSION_DEV_BAD_OFFSETS);
        return;
    }
    const int row0 = part * NWG * 128;            // this CTA's first query row
    if (row0 >= n) return;
    const int nw = min(NWG, (n - row0 + 127) >> 7);   // its query tiles
    const int H = p.heads;
    const int nb = (n + kKeyBlock - 1) / kKeyBlock;
    unsigned char *Q = sm, *Kr = sm + NWG * kQTileBytes;
    const int ns = attn_stages(p.in.max_tokens);
    unsigned char *Vr = Kr + ns * kKeyBytes;

    // (values that a whole warp shares, through shuffles, and elected lanes: the compiler then keeps the
    // copies' and products' operands in uniform registers; a product took 100 cycles to issue from a lane
    // picked by its index, 40 this way)
    const int n_u = __shfl_sync(0xFFFFFFFFu, n, 0), o0_u = __shfl_sync(0xFFFFFFFFu, o0, 0);
    auto rows = [&](unsigned char *dst, int x, int y0, int cnt, unsigned long long *b) {   // cnt: multiple of 8
        mbar_expect_tx(smem_addr(b), (uint32_t)cnt * 128u);
        if (cnt == 128) return tma_load_2d(smem_addr(dst), &maps.b128, x, y0, smem_addr(b));
        int r = 0;
#pragma unroll 1
        for (; r + 64 <= cnt; r += 64) tma_load_2d(smem_addr(dst + r * 128), &maps.b64, x, y0 + r, smem_addr(b));
#pragma unroll 1
        for (; r + 32 <= cnt; r += 32) tma_load_2d(smem_addr(dst + r * 128), &maps.b32, x, y0 + r, smem_addr(b));
#pragma unroll 1
        for (; r < cnt; r += 8) tma_load_2d(smem_addr(dst + r * 128), &maps.b8, x, y0 + r, smem_addr(b));
    };
    auto block_rows = [&](int j) { return (min(kKeyBlock, n_u - j * kKeyBlock) + 7) & ~7; };
    auto load_k = [&](int j, int st) {
        rows(Kr + st * kKeyBytes, (H + h) * kAttnDh, o0_u + j * kKeyBlock, block_rows(j), &bar.k[st]);
    };
    auto load_v = [&](int j, int st) {
        rows(Vr + st * kKeyBytes, (2 * H + h) * kAttnDh, o0_u + j * kKeyBlock, block_rows(j), &bar.v[st]);
    };
    auto load_q = [&](int w) {
        rows(Q + w * kQTileBytes, h * kAttnDh, o0_u + row0 + 128 * w, (min(128, n_u - row0 - 128 * w) + 7) & ~7, &bar.q[w]);
    };
    if (warp == NWG * 4) {   // the barriers, one per lane
        if (lane < (int)(sizeof(AttnBars) / 8))
            mbar_init(smem_addr(&bar.q[0] + lane), lane < 6 + 2 * kStages ? 1 : lane < 6 + 3 * kStages ? nw : 128);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (lane == 0) {
            s_fail = 0;
            s_kv = min(nb, ns);
        }
        __syncwarp();
    }
    if (warp == NWG * 4) {   // the first blocks at once (the second issuing warp allocates meanwhile)
        const int n0 = min((n_u + kKeyBlock - 1) / kKeyBlock, ns);
        if (elect_one()) {
#pragma unroll 1
            for (int j = 0; j < n0; ++j) {
                load_k(j, j);
#pragma unroll 1
                for (int w = 0; j == 0 && w < nw; ++w) load_q(w);
                load_v(j, j);
            }
        }
        __syncwarp();
    }
    if (warp == NWG * 5 - 1) {   // the last of the issuing warps
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                     "r"(NWG * kTileCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp < NWG * 4) {   // log2 of the key sizes meanwhile, four loads of a thread in flight
        float lmax = -INFINITY, lmin = INFINITY;
#pragma unroll 1
        for (int j0 = tid; j0 < nb * kKeyBlock; j0 += NWG * 512) {
            float sz[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = j0 + k * NWG * 128;
                sz[k] = j < n && p.sizes ? p.sizes[o0 + j] : 1.0f;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = j0 + k * NWG * 128;
                if (j >= nb * kKeyBlock) break;
                const float l = log2f(sz[k]);   // 0 past the sample
                lsz[j] = l;
                if (j < n) {
                    lmax = fmaxf(lmax, l);
                    lmin = fminf(lmin, l == l ? l : -1.0f);   // (a NaN is a size too: not ignored as the minimum would)
                }
            }
        }
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            lmax = fmaxf(lmax, __shfl_xor_sync(0xFFFFFFFFu, lmax, o));
            lmin = fminf(lmin, __shfl_xor_sync(0xFFFFFFFFu, lmin, o));
        }
        if (lane == 0) {
            red_max[warp] = lmax;
            red_min[warp] = lmin;
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base;

    if (warp >= NWG * 4 && warp - NWG * 4 < nw) {
        // ---- products of tile w ----------------------------------------------------------------------
        // S of block 0; then per block O += P V, followed by the next block's S
        const int w = __shfl_sync(0xFFFFFFFFu, warp, 0) - NWG * 4;
        const int nb_u = (n_u + kKeyBlock - 1) / kKeyBlock;
        const uint32_t d = __shfl_sync(0xFFFFFFFFu, tmem, 0) + w * kTileCols;
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
        const uint64_t qd = sw128_desc(smem_addr(Q + w * kQTileBytes));
        const uint64_t kd0 = sw128_desc(smem_addr(Kr)), vd0 = sw128_desc(smem_addr(Vr));   // (in 16-byte units)
        auto keys_of = [&](int j) { return (min(kKeyBlock, n_u - j * kKeyBlock) + 15) & ~15; };   // the MMA granularity
        auto s_product = [&](int j, int st, uint32_t dst) {
            const uint64_t kd = kd0 + (uint32_t)st * (kKeyBytes >> 4);
            const uint32_t id = idesc | ((uint32_t)(keys_of(j) >> 3) << 17);
#pragma unroll
            for (int k = 0; k < 4; ++k) umma_bf16(dst, qd + 2u * k, kd + 2u * k, id, k ? 1u : 0u);
        };
        bool ok = warp_wait(smem_addr(&bar.q[w]), 0);
        RingPos kp, vp, rf;   // stages of block j + 1's K, of block j's V, and of the block to refill next
        int next = min(nb_u, ns);
#pragma unroll 1
        for (int j = -1; ok && j < nb_u; ++j) {
            const int cnt = min(kKeyBlock, n_u - j * kKeyBlock), np = (cnt + 15) & ~15;
            if (j >= 0) {
                ok = warp_wait(smem_addr(&bar.v[vp.st]), vp.par);
                if (ok && cnt < np) {
                    // V rows past the sample (another sample's rows or stale memory) read as zero in P V (both
                    // tiles' warps write these zeros)
#pragma unroll 1
                    for (int c = lane; c < (np - cnt) * 8; c += 32)
                        reinterpret_cast<uint4 *>(Vr + vp.st * kKeyBytes + (size_t)cnt * 128)[c] = make_uint4(0u, 0u, 0u, 0u);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor core
                    __syncwarp();
                }
            }
            if (ok && j + 1 < nb_u) ok = warp_wait(smem_addr(&bar.k[kp.st]), kp.par);
            if (ok && j >= 0) ok = warp_wait(smem_addr(&bar.p[w]), (uint32_t)j & 1u);
            if (elect_one() && ok) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (j >= 0) {
                    // B = V as it lies: MN-major (bit 16), 8-key swizzle atoms 1024 bytes apart
                    const uint64_t vd = vd0 + (uint32_t)vp.st * (kKeyBytes >> 4);
                    const uint32_t id = idesc | (1u << 16) | ((uint32_t)(kAttnDh >> 3) << 17);
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        if (kk * 16 < np) umma_bf16_ts(d + 64u, d + 8u * kk, vd + 128u * kk, id, (j | kk) ? 1u : 0u);
                }
                if (j + 1 < nb_u) s_product(j + 1, kp.st, d);
                umma_commit(smem_addr(&bar.s[w]));
                if (j >= 0) umma_commit(smem_addr(&bar.free[vp.st]));   // this block's K and V are read
                // the last tile's lane refills the stage of the block before (both tiles are past it, or nearly)
                if (w == nw - 1 && j >= 1 && next < nb_u) {
                    ok = mbar_wait(smem_addr(&bar.free[rf.st]), rf.par);
                    if (ok) {
                        load_k(next, rf.st);
                        load_v(next, rf.st);
                        rf.next(ns);
                        s_kv = ++next;
                    }
                }
            }
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (j + 1 < nb_u) kp.next(ns);
            if (j >= 0) vp.next(ns);
        }
        if (!ok) atomicOr(&s_fail, 2);
    } else if (warp < nw * 4) {
        // ---- softmax: one thread per query row ---------------------------------------------------
        const int w = warp >> 2, r = tid & 127;
        const bool here = row0 + 128 * w + 32 * (warp & 3) < n;   // warp-uniform: a warp of rows past the sample idles
        const uint32_t taddr = tmem + w * kTileCols + ((uint32_t)((warp & 3) * 32) << 16);
        float lszmax = red_max[0], lszmin = red_min[0];
#pragma unroll
        for (int k = 1; k < NWG * 4; ++k) {
            lszmax = fmaxf(lszmax, red_max[k]);
            lszmin = fminf(lszmin, red_min[k]);
        }
        const bool sized = lszmax != 0.0f || lszmin != 0.0f;
        constexpr float kScale2 = 0.18033688011112042f;   // log2(e) / sqrt(64)
        // the shift; the largest S so far, at least the lowest finite value: a row whose first blocks are -inf
        // (infinite inputs, an overflowing product) has probabilities of zero there, not of -inf - (-inf)
        float m = 0.0f, mraw = -3.402823466e38f;
        float2 lsum = make_float2(0.0f, 0.0f);   // even and odd keys
        bool ok = true;
#pragma unroll 1
        for (int j = 0; ok && j < nb; ++j) {
            ok = warp_wait(smem_addr(&bar.s[w]), (uint32_t)j & 1u);   // S of block j, and O up to the block before
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (ok && here) {
                const int cnt = n - j * kKeyBlock;
                uint32_t v[64];
                tmem_ld32(taddr, v);
                tmem_ld32(taddr + 32u, v + 32);
                tmem_ld_wait();
                if (cnt < kKeyBlock) {   // keys past the sample: probability 2^-inf = 0
#pragma unroll
                    for (int e = 0; e < 64; ++e) v[e] = e < cnt ? v[e] : 0xFF800000u;
                }
                float a[4] = {mraw, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                for (int e = 0; e < 64; e += 8)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        a[q] = max3(a[q], __uint_as_float(v[e + 2 * q]), __uint_as_float(v[e + 2 * q + 1]));
                const float mx = fmaxf(max3(a[0], a[1], a[2]), a[3]);
                const float mn = fmaf(mx, kScale2, lszmax), f = ex2(m - mn);   // the shift follows the largest S
                const bool grows = j > 0 && __any_sync(0xFFFFFFFFu, mx > mraw);
                m = mn;
                mraw = mx;
                const float2 ps = sized ? block_probs<true>(v, taddr, lsz + j * kKeyBlock, m)
                                        : block_probs<false>(v, taddr, nullptr, m);
                if (grows) {   // and the rows of O and their sums follow the shift (after P: S's registers are free)
                    lsum = __fmul2_rn(lsum, make_float2(f, f));
                    uint32_t o[64];
                    tmem_ld32(taddr + 64u, o);
                    tmem_ld32(taddr + 96u, o + 32);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 64; e += 8) {
                        uint32_t o8[8];
#pragma unroll
                        for (int q = 0; q < 8; q += 2) {
                            const float2 y = __fmul2_rn(make_float2(__uint_as_float(o[e + q]), __uint_as_float(o[e + q + 1])),
                                                        make_float2(f, f));
                            o8[q] = __float_as_uint(y.x);
                            o8[q + 1] = __float_as_uint(y.y);
                        }
                        tmem_st8(taddr + 64u + e, o8);
                    }
                }
                lsum = __fadd2_rn(lsum, ps);
                tmem_st_wait();
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(smem_addr(&bar.p[w]));
        }
        if (ok) ok = warp_wait(smem_addr(&bar.s[w]), (uint32_t)nb & 1u);   // the last block's O
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) atomicOr(&s_fail, 4);
        if (ok && here) {
            // ---- O / row sum -> bf16, through the tile's Q rows (read by now), eight lanes per row ----
            uint32_t o[64];
            tmem_ld32(taddr + 64u, o);
            tmem_ld32(taddr + 96u, o + 32);
            tmem_ld_wait();
            const float inv = 1.0f / (lsum.x + lsum.y);
            unsigned char *qt = Q + w * kQTileBytes;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                uint32_t q4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 y = __fmul2_rn(
                        make_float2(__uint_as_float(o[8 * c + 2 * e]), __uint_as_float(o[8 * c + 2 * e + 1])),
                        make_float2(inv, inv));
                    const __nv_bfloat162 b2 = __floats2bfloat162_rn(y.x, y.y);
                    q4[e] = *reinterpret_cast<const uint32_t *>(&b2);
                }
                *reinterpret_cast<uint4 *>(qt + r * 128 + ((c ^ (r & 7)) << 4)) = make_uint4(q4[0], q4[1], q4[2], q4[3]);
            }
            __syncwarp();
            __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(p.out) + (size_t)h * kAttnDh;
            const int rw = 32 * (warp & 3) + (lane >> 3), c = lane & 7;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int rr = rw + 4 * k, mrow = row0 + 128 * w + rr;
                if (mrow < n)
                    *reinterpret_cast<uint4 *>(out + (size_t)(o0 + mrow) * H * kAttnDh + c * 8) =
                        *reinterpret_cast<const uint4 *>(qt + rr * 128 + ((c ^ (rr & 7)) << 4));
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (s_fail != 0 && warp == NWG * 4) {   // let everything this CTA started finish before it leaves
        if (lane == 0) {
            raise_status(p.status, FUSION_DEV_TIMEOUT);
#pragma unroll 1
            for (int j = max(0, s_kv - ns); j < s_kv; ++j) {
                (void)mbar_wait(smem_addr(&bar.k[j % ns]), (uint32_t)(j / ns) & 1u);
                (void)mbar_wait(smem_addr(&bar.v[j % ns]), (uint32_t)(j / ns) & 1u);
            }
#pragma unroll 1
            for (int w = 0; w < nw; ++w) (void)mbar_wait(smem_addr(&bar.q[w]), 0);
        }
        __syncwarp();
    }
    if (s_fail != 0) {   // uniform: each issuing thread drains its own products (a commit covers only those, and
                         // the election picks the same lane every time)
        if (warp >= NWG * 4 && warp - NWG * 4 < nw && elect_one()) {
            umma_commit(smem_addr(&bar.drain[warp - NWG * 4]));
            (void)mbar_wait(smem_addr(&bar.drain[warp - NWG * 4]), 0);
        }
        __syncthreads();
    }
    if (warp == NWG * 5 - 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(NWG * kTileCols) : "memory");
}

template <int NWG>
cudaError_t launch_tiles(const AttnMaps &maps, const AttnParams &p, cudaStream_t s) {
    const int n_part = ceil_div(p.in.max_tokens, NWG * 128);
    const size_t smem = 1024 + (size_t)NWG * kQTileBytes + 2 * (size_t)attn_stages(p.in.max_tokens) * kKeyBytes;
    cudaError_t e = cudaFuncSetAttribute(k_attn_tc<NWG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_attn_tc<NWG>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    k_attn_tc<NWG><<<dim3((unsigned)(p.heads * n_part), (unsigned)p.in.max_batch), NWG * 160, smem, s>>>(maps, p, n_part);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_attention(const AttnParams &p, cudaStream_t s) {
    if (p.in.max_batch == 0 || p.heads == 0) return cudaSuccess;
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    AttnMaps maps;
    CUtensorMap *dst[4] = {&maps.b128, &maps.b64, &maps.b32, &maps.b8};
    for (int b = 0; b < 4; ++b) {
        cuuint64_t dims[2] = {(cuuint64_t)3 * p.heads * kAttnDh, (cuuint64_t)p.in.max_rows};
        cuuint64_t strides[1] = {(cuuint64_t)3 * p.heads * kAttnDh * 2};
        cuuint32_t box[2] = {64, b == 0 ? 128u : b == 1 ? 64u : b == 2 ? 32u : 8u};
        cuuint32_t estr[2] = {1, 1};
        if (enc(dst[b], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(p.qkv), dims,
                strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    // one query tile per CTA where the call's samples have one
    return p.in.max_tokens <= 128 ? launch_tiles<1>(maps, p, s) : launch_tiles<2>(maps, p, s);
}

}  // namespace fz
