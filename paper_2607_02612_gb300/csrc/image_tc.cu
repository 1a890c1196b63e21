// Per-sample merge -> prune -> gather for bf16 tokens on the 5th-generation tensor
// cores (tcgen05) with TMA, for samples of at most 257 tokens (|A|, |B| <= 128).
//
// One CTA of 256 threads per input sample (128 threads for large batches of small samples; small
// batches: up to four CTAs per sample, each a range of the output columns).  The keys of half A (even positions) and
// half B (odd positions) arrive by TMA tensor loads in K-blocks of 64 dims, 128-byte
// swizzled: K-block kb of a half is a [rows][128 B] tile, 16-byte chunk j of row t
// stored at chunk position j ^ (t % 8).  Tensor maps per parity of the global row index
// (every other row of the token matrix) cover boxes of a whole half, 64, 32 and 8 rows, so any
// half of any sample loads in whole 8-row groups and few copies.  The K-blocks stream through a ring
// of stages (the whole sample stays resident when it fits).
//
// An elected lane of warp 0 produces (TMA), one of warp 1 issues tcgen05.mma (M = 128 A rows, N = |B|
// rounded up to 16, K = 16 per instruction, f32 accumulation in tensor memory), and
// every thread accumulates the squared norm of one A or B row from the same stages.
// A stage is released when the MMAs that read it completed (tcgen05.commit) and all
// warps are done with it.  The epilogue reads S from tensor memory, one A row per
// thread (two warpgroups split the columns), forms cos = dot * inv|a| * inv|b| and
// keeps the largest value with the lowest B index.  Everything after the decisions
// (top-r, merged set, sums, pruning, gather) is the shared finish phase.
//
// Every wait on an mbarrier is bounded; on a timeout the CTA raises
// FUSION_DEV_TIMEOUT, skips its outputs and frees its tensor memory.
#include <cuda.h>

#include <algorithm>

#include "sample.cuh"
#include "tc.cuh"

namespace fz {
namespace {

constexpr int kSms = 152;
constexpr int kMaxStages = 16;

struct TcMaps {
    CUtensorMap e32, o32, e8, o8;   // even / odd rows, boxes of 32 / 8 rows x 64 dims
    // larger boxes: 256 / 128 rows (k_image_tc_tiled); a whole half of max_tokens / 64 rows (k_image_tc)
    CUtensorMap e256, o256, e128, o128;
    // even / odd rows seen as (64 dims, row, K-block) with the K-block stride 128 B: a box of
    // 8 rows x all K-blocks lands as [K-block][8 rows][128 B], one 1 KB swizzle atom per K-block
    CUtensorMap ge, go;
};

// ss + sc += part, Neumaier-compensated.
__device__ __forceinline__ void neumaier_add(float &ss, float &sc, float part) {
    const float t = __fadd_rn(ss, part);
    sc = __fadd_rn(sc, fabsf(ss) >= fabsf(part) ? __fadd_rn(__fsub_rn(ss, t), part) : __fadd_rn(__fsub_rn(part, t), ss));
    ss = t;
}
// Sum of squares of the 8 bf16 values of a 16-byte chunk.
__device__ __forceinline__ float chunk_sq(uint4 v) {
    float f[8];
    chunk_to_f(v, f);
    float part = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; ++e) part = fmaf(f[e], f[e], part);
    return part;
}

// Chunk c of input token pos for the finish phase, wherever the sample's rows are: one type
// for every layout, so the finish phase is compiled once (its code is fetched cold after every
// flush of L2, and a second copy for another layout made stages slower).
//   rows in global memory (g != null): chunk c of token pos at g + pos * rb + 16 c;
//   rows in shared memory: CLS from its staged copy; row r of a half (positions 2, 4, ... or
//   1, 3, ...) at h + (r / 8) G + (r % 8) 128, its 16-byte chunk c (c / 8) K + 16 ((c % 8) ^
//   (r % 8)) further (ring: h = the half's base in stage 0, G = 1024, K = kbs; grouped layout:
//   h = the half's first group, G = n_kb KB, K = 1024).
// The branch is uniform over the CTA.
struct RowLoader {
    const unsigned char *g;   // the sample's first row in global memory, or null
    uint32_t rb;               // bytes of a token row
    const unsigned char *cls, *hA, *hB;
    uint32_t G, K;
    __device__ __forceinline__ uint4 operator()(int pos, int c) const {
        if (g) return ldg16(g + (size_t)pos * rb + (size_t)c * 16);
        if (pos == 0) return *reinterpret_cast<const uint4 *>(cls + (size_t)c * 16);
        const bool isB = pos & 1;
        const unsigned r = (unsigned)(isB ? (pos - 1) >> 1 : (pos - 2) >> 1);
        const unsigned x = r & 7u, cc = (unsigned)c;
        const unsigned char *base = (isB ? hB : hA) + (size_t)(r >> 3) * G + (size_t)(cc >> 3) * K;
        return *reinterpret_cast<const uint4 *>(base + x * 128u + (((cc & 7u) ^ x) << 4));
    }
};

// The ring of K-block stages of one sample, sized for it: S stages of kbs bytes, K-block kb
// in stage kb % S with half A at the stage's start and half B after rowsA rows.  The boxes of
// one K-block: half A then half B, in 32-row boxes while 32 rows remain, then 8-row boxes.
struct Ring {
    int S, rowsA, rowsB, npad, nbA, per_kb;
    uint32_t kbs;
};
// The boxes of n rows: one of `full` rows where that is n rounded up to 8 (the longest samples of a call,
// all of a uniform one), else 64, 32 and 8 rows.  A copy costs its issuing thread about 200 cycles.
__device__ __forceinline__ int box_count(int n, int full) {
    return ((n + 7) & ~7) == full ? 1 : (n >> 6) + ((n >> 5) & 1) + (((n & 31) + 7) >> 3);
}
__device__ __forceinline__ Ring ring_for(int nA, int nB, int nkb, const TcGeometry &g) {
    Ring R;
    R.rowsA = (nA + 7) & ~7;
    R.rowsB = (nB + 7) & ~7;
    R.npad = (nB + 15) & ~15;   // MMA N: |B| rounded up to 16
    R.kbs = (uint32_t)(R.rowsA + R.rowsB) * 128u;
    // An MMA reads 128 A rows and npad B rows from a stage, past its end when the sample is
    // small, which stays inside the buffer.
    const uint32_t reach = (uint32_t)max(16384, (R.rowsA + R.npad) * 128);
    int S = min(min(nkb, kMaxStages), (int)(g.stage_region / R.kbs));
    while (S > 1 && (uint32_t)(S - 1) * R.kbs + reach > g.usable) --S;
    R.S = S;
    R.nbA = box_count(nA, g.full_rows);
    R.per_kb = R.nbA + box_count(nB, g.full_rows);
    return R;
}
// Box b of K-block kb of the sample whose rows start at `start` (half A: positions 2, 4, ...,
// half B: 1, 3, ..., each contiguous in the even or odd row view).
__device__ __forceinline__ void issue_box(const TcMaps &maps, const Ring &R, const TcGeometry &g, int start, int nA,
                                          int nB, unsigned char *sm, unsigned long long *bar_full, int kb, int b) {
    const int st = kb % R.S;
    const int half = b >= R.nbA ? 1 : 0;
    const int q = half ? b - R.nbA : b, n = half ? nB : nA;
    const bool odd = half ? ((start + 1) & 1) : ((start + 2) & 1);
    const int n64 = n >> 6, n32 = (n >> 5) & 1;
    int row0 = 0;
    const CUtensorMap *map;
    if (((n + 7) & ~7) == g.full_rows) {
        map = odd ? &maps.o256 : &maps.e256;
    } else if (q < n64) {
        row0 = q * 64;
        map = odd ? &maps.o128 : &maps.e128;
    } else if (q - n64 < n32) {
        row0 = n64 * 64;
        map = odd ? &maps.o32 : &maps.e32;
    } else {
        row0 = (n >> 5) * 32 + (q - n64 - n32) * 8;
        map = odd ? &maps.o8 : &maps.e8;
    }
    const int y = half ? (start + 1) >> 1 : (start + 2) >> 1;
    const uint32_t dst = smem_addr(sm + (half ? (size_t)R.rowsA * 128 : (size_t)0) + (size_t)st * R.kbs + (size_t)row0 * 128);
    tma_load_2d(dst, map, kb * 64, y + row0, smem_addr(&bar_full[st]));
}
// Every barrier a ring can use, from the lanes of one warp at kernel entry: the fence that publishes
// the initialisation waits for a thread's outstanding memory operations, so it runs before the
// warp has issued any.
template <int NT>
__device__ __forceinline__ void ring_barriers_init(unsigned long long *bar_full, unsigned long long *bar_empty,
                                                   unsigned long long *bar_done, unsigned long long *bar_drain) {
    const int lane = threadIdx.x & 31;
    static_assert(kMaxStages == 16, "a full and an empty barrier per lane pair");
    mbar_init(smem_addr(lane < 16 ? &bar_full[lane] : &bar_empty[lane - 16]), lane < 16 ? 1 : 1 + NT / 32);
    if (lane < 2) mbar_init(smem_addr(lane == 0 ? bar_done : bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// From the 32 lanes of one warp, once the barriers are initialised and that is visible to the
// warp: the first min(S, nkb) K-blocks.
__device__ __forceinline__ void ring_start(const TcMaps &maps, const Ring &R, const TcGeometry &g, int start, int nA, int nB, int nkb,
                                           unsigned char *sm, unsigned long long *bar_full) {
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const int S0 = min(R.S, nkb);
    if (lane < S0) mbar_expect_tx(smem_addr(&bar_full[lane]), R.kbs);
#pragma unroll 1
    for (int t = lane; t < S0 * R.per_kb; t += 32)
        issue_box(maps, R, g, start, nA, nB, sm, bar_full, t / R.per_kb, t % R.per_kb);
}
// A sample that fits in shared memory, grouped: half A in 8-row groups g at g * nkb KB, each
// group [K-block][8 rows][128 B], half B after it the same way, all behind bar_full[0]; one box
// per group (the K-block ring needs per_kb boxes per K-block).  The rows of the last group past
// the half belong to the next sample or lie past the tensor (zero fill) and are never used.
// From the 32 lanes of one warp, once the barriers are initialised and that is visible to it.
__device__ __forceinline__ void group_start(const TcMaps &maps, const Ring &R, int start, int nkb, unsigned char *sm,
                                            unsigned long long *bar_full) {
    const int lane = threadIdx.x & 31;
    const int GA = R.rowsA >> 3, GB = R.rowsB >> 3;
    const uint32_t gstride = (uint32_t)nkb * 1024u;
    __syncwarp();
    if (lane == 0) mbar_expect_tx(smem_addr(&bar_full[0]), (uint32_t)(GA + GB) * gstride);
    const bool oddA = (start + 2) & 1, oddB = (start + 1) & 1;
    const int yA = (start + 2) >> 1, yB = (start + 1) >> 1;
#pragma unroll 1
    for (int b = lane; b < GA + GB; b += 32) {
        const bool isB = b >= GA;
        const int q = isB ? b - GA : b;
        const CUtensorMap *map = (isB ? oddB : oddA) ? &maps.go : &maps.ge;
        const uint32_t dst = smem_addr(sm + (size_t)(isB ? GA + q : q) * gstride);
        tma_load_3d(dst, map, 0, (isB ? yB : yA) + 8 * q, 0, smem_addr(&bar_full[0]));
    }
}
// The sample's token sizes and scores and its CLS row into shared memory (cp.async, one
// group; waited for in meta_init_rest).
template <int NT>
__device__ __forceinline__ void prefetch_own(const ImageParams &p, int start, int N, const MetaPtrs &m, uint4 *cls) {
#pragma unroll 1
    for (int pos = threadIdx.x; pos < N; pos += NT) {
        cp_async4(&m.tsize[pos], p.sizes + start + pos);
        if (p.scores) cp_async4(&m.tscore[pos], p.scores + start + pos);
    }
    const uint4 *row = reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(p.x) + (long long)start * p.dim);
#pragma unroll 1
    for (int c = threadIdx.x; c < p.dim / 8; c += NT) cp_async16(&cls[c], row + c);
    cp_async_commit();
}

// NT 256: two CTAs per SM; 128 (large batches of samples of at most 129 tokens): four.
template <int NT>
__global__ void __launch_bounds__(NT, NT == 128 ? 4 : 2)
    k_image_tc(const __grid_constant__ TcMaps maps, ImageParams p, TcGeometry g) {
    extern __shared__ unsigned char sm_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) unsigned long long bar_full[kMaxStages], bar_empty[kMaxStages], bar_done, bar_drain;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail;
    __shared__ unsigned long long half_best[NT == 256 ? 128 : 1];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // Tensor memory first: an SM admits another CTA of a kernel that allocates tensor
    // memory only once the resident one has given up its allocation permit.
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                     "r"(g.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the tensor maps' descriptors travel while the sample's metadata loads
    if (tid >= 32 && tid < 36) {
        const CUtensorMap *mp = tid == 32 ? &maps.e32 : tid == 33 ? &maps.o32 : tid == 34 ? &maps.e8 : &maps.o8;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(mp)) : "memory");
    }
    // the ring's barriers, before this warp issues any memory operation (warp 0 issues the
    // tokens' loads after a CTA barrier: the fused plan's, or the one below)
    if (warp == 2) ring_barriers_init<NT>(bar_full, bar_empty, &bar_done, &bar_drain);
    if (g.grouped && (tid == 38 || tid == 39))
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tid == 38 ? &maps.ge : &maps.go)) : "memory");
    if (tid == 0) s_fail = 0;   // visible after the barriers below, before any other write
    const int nkb = g.n_kb;
    MetaPtrs m(sm, meta_layout(p.in.max_tokens, g.meta_base));
    uint4 *cls = reinterpret_cast<uint4 *>(sm + g.cls_base);
    // launched as a programmatic dependent of the exit check: everything above (tensor memory,
    // barriers, descriptor prefetch) and the plan's loads of this call's own inputs overlap that
    // kernel's end; the exit mask is read after `griddepcontrol.wait` (without a programmatic
    // predecessor the wait returns at once)
    SampleInfo s;
    const int part = g.parts > 1 ? (int)(blockIdx.x % (unsigned)g.parts) : 0;
    if (!sample_begin<NT>(p, g.parts > 1 ? blockIdx.x / g.parts : blockIdx.x, s, true)) {   // uniform over the CTA
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(g.tmem_cols)
                         : "memory");
        return;
    }
    if (!p.fused_plan) __syncthreads();   // uniform: the fused plan has barriers of its own
    const bool dec = s.decide;
    const Ring R = ring_for(s.nA, s.nB, nkb, g);
    const int S = R.S, npad = R.npad;
    const uint32_t kbs = R.kbs;
    unsigned char *regA = sm;                         // stage st, half A: regA + st * kbs
    unsigned char *regB = sm + (size_t)R.rowsA * 128;  // stage st, half B: regB + st * kbs (ring layout)
    auto produce = [&](int kb) {   // a whole K-block from one thread
        mbar_expect_tx(smem_addr(&bar_full[kb % S]), kbs);
#pragma unroll 1
        for (int b = 0; b < R.per_kb; ++b) issue_box(maps, R, g, s.start, s.nA, s.nB, sm, bar_full, kb, b);
    };

    // the sample's sizes, scores and CLS row first (a few KB that would otherwise queue behind the
    // bulk loads), then its tokens: the grouped layout or the ring's first stages (warp 0)
    prefetch_own<NT>(p, s.start, s.N, m, cls);
    const bool grouped = g.grouped && S >= nkb;   // the layout of this sample (uniform)
    const uint32_t gstride = (uint32_t)nkb * 1024u;
    unsigned char *gB = sm + (size_t)(R.rowsA >> 3) * gstride;   // grouped layout: half B
    if (warp == 0 && dec) {
        if (grouped)
            group_start(maps, R, s.start, nkb, sm, bar_full);
        else
            ring_start(maps, R, g, s.start, s.nA, s.nB, nkb, sm, bar_full);
    }
    meta_init_rest<NT>(p, s, m);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    if (dec) {
        const uint32_t tmem = tmem_base;

        // instruction descriptor: f32 accumulator, bf16 A and B, K-major, N = |B| rounded to 16, M = 128
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(npad >> 3) << 17) | (8u << 24);
        // Squared row norms: for a sample that stays resident, after all stages landed with
        // kT threads per row; otherwise one thread per row, K-block by K-block as the ring turns.
        const bool resident = S >= nkb;
        const int splitA = NT == 256 ? 128 : s.nA;   // 128 threads: nA + nB <= 128
        const bool isA = tid < splitA;
        const int row = isA ? tid : tid - splitA;
        const bool has_row = !resident && row < (isA ? s.nA : s.nB);
        float ss = 0.0f, sc = 0.0f;
        // A lane whose wait gave up goes on through the loop without waiting, because the others meet it there (an
        // election, a warp barrier); it only does nothing that needs what it waited for.  (A vote after every wait
        // instead: long samples 136 -> 140 us, four stages of 8192 images 298 -> 302.)
        bool ok = true;
        int issued = grouped ? 1 : min(S, nkb);   // stages whose copies were issued (the count of warp 0's elected lane)
        if (grouped) {   // everything behind one barrier; all products at once
            ok = mbar_wait(smem_addr(&bar_full[0]), 0u);
            if (warp == 1 && elect_one() && ok) {
                const uint32_t a0 = smem_addr(sm), b0 = smem_addr(gB);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
                for (int kb = 0; kb < nkb; ++kb)
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        umma_bf16(tmem, sw128_desc_sbo(a0 + kb * 1024 + k * 32, gstride),
                                  sw128_desc_sbo(b0 + kb * 1024 + k * 32, gstride), idesc, (kb | k) ? 1u : 0u);
                umma_commit(smem_addr(&bar_done));
            }
        }
#pragma unroll 1
        for (int kb = 0; kb < (grouped ? 0 : nkb); ++kb) {
            const int st = kb % S;
            const uint32_t par = (uint32_t)(kb / S) & 1u;
            ok = ok && mbar_wait(smem_addr(&bar_full[st]), par);
            if (warp == 1 && elect_one() && ok) {
                const uint32_t a0 = smem_addr(regA + (size_t)st * kbs), b0 = smem_addr(regB + (size_t)st * kbs);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    umma_bf16(tmem, sw128_desc(a0 + k * 32), sw128_desc(b0 + k * 32), idesc, (kb | k) ? 1u : 0u);
                umma_commit(smem_addr(&bar_empty[st]));
                if (kb == nkb - 1) umma_commit(smem_addr(&bar_done));
            }
            if (has_row) {   // squared norm of this thread's row, chunk by chunk
                const unsigned char *base = (isA ? regA : regB) + (size_t)st * kbs + row * 128;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    neumaier_add(ss, sc, chunk_sq(*reinterpret_cast<const uint4 *>(base + ((j ^ (row & 7)) << 4))));
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&bar_empty[st]));
            if (warp == 0 && kb + S < nkb) {   // refill this stage once everyone is done with it
                ok = ok && mbar_wait(smem_addr(&bar_empty[st]), par);
                if (elect_one() && ok) {
                    produce(kb + S);
                    ++issued;
                }
                __syncwarp();
            }
        }
        if (!ok) atomicOr(&s_fail, 1);
        int nrow = row;        // row of this thread: A rows, then B rows
        bool owner = has_row;  // writes the row's inverse norm
        if (resident) {   // uniform over the CTA: every lane reaches the shuffles
            // kT threads per row (the largest power of two up to 8 that fits), each taking
            // every kT-th chunk of the row; the partial sums meet by shuffles
            const int R = s.nA + s.nB;
            const int kT = R <= NT / 8 ? 8 : R <= NT / 4 ? 4 : R <= NT / 2 ? 2 : 1;
            const int r = tid / kT, part = tid % kT;
            if (r < R) {
                const bool rA = r < s.nA;
                const int rr = rA ? r : r - s.nA;
                const unsigned char *base = grouped ? (rA ? sm : gB) + (size_t)(rr >> 3) * gstride + (rr & 7) * 128
                                                    : (rA ? regA : regB) + (size_t)rr * 128;
                const uint32_t kstep = grouped ? 1024u : kbs;   // bytes from one K-block of the row to the next
#pragma unroll 1
                for (int c = part; c < nkb * 8; c += kT)
                    neumaier_add(ss, sc, chunk_sq(*reinterpret_cast<const uint4 *>(
                                             base + (size_t)(c >> 3) * kstep + (((c & 7) ^ (rr & 7)) << 4))));
            }
            for (int mk = 1; mk < kT; mk <<= 1) {   // kT divides 32: groups stay inside a warp
                const float oss = __shfl_xor_sync(0xFFFFFFFFu, ss, mk), osc = __shfl_xor_sync(0xFFFFFFFFu, sc, mk);
                neumaier_add(ss, sc, oss);
                sc = __fadd_rn(sc, osc);
            }
            owner = r < R && part == 0;
            nrow = r;
        } else if (has_row) {
            nrow = isA ? row : s.nA + row;
        }
        if (owner) {
            const float sq = __fadd_rn(ss, sc);
            if (!isfinite(sq)) raise_status(p.status, FUSION_DEV_NONFINITE);
            const float inv = 1.0f / fmaxf(sqrtf(sq), 1e-12f);
            if (nrow < s.nA)
                m.inv_a[nrow] = inv;
            else
                m.inv_b[nrow - s.nA] = inv;
        }
        __syncthreads();
        bool mma_ok = s_fail == 0 && mbar_wait(smem_addr(&bar_done), 0);
        if (!mma_ok) atomicOr(&s_fail, 2);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        __syncthreads();
        if (s_fail == 0) {
            // epilogue: thread -> A row (tid % 128); the two warpgroups take the low / high columns
            const int wg = tid >> 7;
            const int r = tid & 127;
            const int half_cols = NT == 256 ? ((npad / 16 + 1) / 2) * 16 : npad;
            const int c_lo = wg ? half_cols : 0, c_hi = wg ? npad : half_cols;
            const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16);
            const float ia = r < s.nA ? m.inv_a[r] : 0.0f;
            // the largest cosine of the thread's columns and its lowest column: the columns go up,
            // so a strict comparison keeps the first of equal values (and -0 equals +0)
            float bv = -INFINITY;
            int bi = -1;
#pragma unroll 1
            for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
                uint32_t v[16];
                tmem_ld16(lane_addr + (uint32_t)c0, v);
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int col = c0 + e;
                    if (col < s.nB) {
                        const float cs = (__uint_as_float(v[e]) * ia) * m.inv_b[col];
                        if (cs > bv || bi < 0) {
                            bv = cs;
                            bi = col;
                        }
                    }
                }
            }
            const unsigned long long bk = (r < s.nA && bi >= 0) ? rank_key(bv, bi) : 0ull;
            if constexpr (NT == 256) {
                if (wg == 1) half_best[r] = bk;
                __syncthreads();
                if (wg == 0 && r < s.nA) {
                    const unsigned long long o = half_best[r];
                    m.best[r] = o > bk ? o : bk;
                }
            } else if (r < s.nA) {
                m.best[r] = bk;
            }
        } else {
            // a wait gave up: let the copies and products in flight land (bounded) before the
            // shared and tensor memory are released
            if (warp == 0 && elect_one()) {
                raise_status(p.status, FUSION_DEV_TIMEOUT);
#pragma unroll 1
                for (int q = max(0, issued - S); q < issued; ++q)
                    (void)mbar_wait(smem_addr(&bar_full[q % S]), (uint32_t)(q / S) & 1u);
            }
            if (warp == 1 && elect_one()) {   // the lane that issued the products: a commit covers only its own
                umma_commit(smem_addr(&bar_drain));
                (void)mbar_wait(smem_addr(&bar_drain), 0u);
            }
        }
        __syncthreads();
        if (s_fail == 0) select_top_r<NT>(s, m);
    }

    if (s_fail == 0) {
        const uint32_t rb = (uint32_t)p.dim * 2u;   // bytes of a token row
        RowLoader ld{reinterpret_cast<const unsigned char *>(p.x) + (size_t)s.start * rb, rb,
                     reinterpret_cast<const unsigned char *>(cls), nullptr, nullptr, 0u, 0u};
        if (dec && S >= nkb && p.keys_alias) {   // the whole sample is in shared memory
            ld.g = nullptr;
            ld.hA = sm;
            ld.hB = grouped ? gB : regB;
            ld.G = grouped ? gstride : 1024u;
            ld.K = grouped ? 1024u : kbs;
        }
        if (finish_decide<NT>(p, s, m)) {
            if (part == 0) write_index_outputs<NT>(p, s, m);
            const int w = p.dim / 8;
            write_rows<__nv_bfloat16, NT>(p, s, m, ld, w * part / g.parts, w * (part + 1) / g.parts);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(g.tmem_cols)
                     : "memory");
}

// ---------------------------------------------------------------------------
// Samples whose halves exceed one tile (|A| or |B| above 128; ViT-L/16 at 384: 288 x 288 x
// 1024): one CTA of 512 threads per SM, 512 tensor-memory columns.  Half A lies in M-tiles of 128
// rows (up to four), half B in passes of at most 512 / M-tiles columns (a multiple of 16, at most 256), so
// that the accumulators of all M-tiles of a pass fit tensor memory.  Per pass the K-blocks of (all A
// rows, the pass's B rows) stream by TMA through the ring (stage q = pass q / n_kb, K-block q % n_kb); the
// epilogue keeps each A row's best column over the passes.  Row norms, one thread per row: A during
// the first pass, a pass's B rows during it.
//
// Bound by DRAM while it streams: A is read once per pass and B once.  One pass per M-tile, which reads
// B once per M-tile (three times at 288 x 288, the second and third mostly from DRAM: a wave's first
// tiles are larger than L2), took 58 us for the three tiles of 128 samples; the whole call takes 15 us less in this order (159 -> 144).
// ---------------------------------------------------------------------------
constexpr int kTiledMaxStages = 8;
constexpr int kTiledThreads = 512;

__global__ void __launch_bounds__(kTiledThreads, 1)
    k_image_tc_tiled(const __grid_constant__ TcMaps maps, ImageParams p, TcGeometry g) {
    extern __shared__ unsigned char sm_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) unsigned long long bar_full[kTiledMaxStages], bar_empty[kTiledMaxStages], bar_done, bar_drain;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail;
    __shared__ unsigned long long part_best[kTiledThreads];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                     "r"(g.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid >= 32 && tid < 36) {
        const CUtensorMap *mp = tid == 32 ? &maps.e32 : tid == 33 ? &maps.o32 : tid == 34 ? &maps.e8 : &maps.o8;
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(mp)) : "memory");
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");   // as in k_image_tc: the exit check's grid first
    SampleInfo s;
    if (!sample_begin<kTiledThreads>(p, blockIdx.x, s)) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(g.tmem_cols)
                         : "memory");
        return;
    }
    const bool dec = s.decide;
    const int nkb = g.n_kb;
    int issued = 0;   // stages issued (the count of warp 0's elected lane; the warp issues the first ones)
    const int nM = max(1, (s.nA + 127) >> 7);       // M-tiles of half A
    const int rowsA = (s.nA + 7) & ~7;
    const int npad = (s.nB + 15) & ~15;             // columns of the product
    const int nblk = min(256, g.tmem_cols / nM & ~15);   // columns of a pass and M-tile
    const int nP = (npad + nblk - 1) / nblk;
    // stage: [A rows][a pass's B rows] x 128 B; an MMA reads 128 A rows from a tile's start, and up to a
    // pass's columns of B rows
    const uint32_t aBytes = (uint32_t)rowsA * 128u;
    const uint32_t kbs = aBytes + (uint32_t)min(nblk, (s.nB + 7) & ~7) * 128u;
    const uint32_t reach = max((uint32_t)nM * 16384u, aBytes + (uint32_t)min(nblk, npad) * 128u);
    const int nq = nP * nkb;
    int S = min(min(nq, kTiledMaxStages), (int)(g.stage_region / kbs));
    while (S > 1 && (uint32_t)(S - 1) * kbs + reach > g.usable) --S;
    const int yB = (s.start + 1) >> 1, yA0 = (s.start + 2) >> 1;
    const bool oddA = (s.start + 2) & 1, oddB = (s.start + 1) & 1;
    // boxes of stage q: the A rows, then the B rows of its pass
    auto pass_rows = [&](int ps) { return min(nblk, s.nB - ps * nblk); };
    // 256- and 128-row boxes while they fit, then 32, then 8: a copy costs its issuing thread about 200
    // cycles, and 32-row boxes alone (13 per stage at 288 x 288) held the ring to 1.75 us per stage
    auto nboxes = [&](int n) { return (n >> 8) + ((n >> 7) & 1) + ((n >> 5) & 3) + (((n & 31) + 7) >> 3); };
    auto stage_tx = [&](int ps) { return (uint32_t)(rowsA + ((pass_rows(ps) + 7) & ~7)) * 128u; };
    auto issue_box = [&](int q, int b) {
        const int st = q % S, ps = q / nkb, kb = q - ps * nkb;
        const int nbA = nboxes(s.nA);
        const bool half = b >= nbA;   // B rows
        const int qq = half ? b - nbA : b;
        const int n = half ? pass_rows(ps) : s.nA;
        const bool odd = half ? oddB : oddA;
        const int n256 = n >> 8, n128 = (n >> 7) & 1, n32 = (n >> 5) & 3;
        int row0, u = qq;
        const CUtensorMap *map;
        if (u < n256) {
            row0 = u * 256;
            map = odd ? &maps.o256 : &maps.e256;
        } else if ((u -= n256) < n128) {
            row0 = n256 * 256;
            map = odd ? &maps.o128 : &maps.e128;
        } else if ((u -= n128) < n32) {
            row0 = (n >> 7) * 128 + u * 32;
            map = odd ? &maps.o32 : &maps.e32;
        } else {
            row0 = (n >> 5) * 32 + (u - n32) * 8;
            map = odd ? &maps.o8 : &maps.e8;
        }
        unsigned char *base = sm + (size_t)st * kbs + (half ? aBytes : 0u);
        tma_load_2d(smem_addr(base + (size_t)row0 * 128), map, kb * 64, (half ? yB + ps * nblk : yA0) + row0,
                    smem_addr(&bar_full[st]));
    };
    auto boxes_of = [&](int q) { return nboxes(s.nA) + nboxes(pass_rows(q / nkb)); };
    auto produce = [&](int q) {
        mbar_expect_tx(smem_addr(&bar_full[q % S]), stage_tx(q / nkb));
        const int nb = boxes_of(q);
        for (int b = 0; b < nb; ++b) issue_box(q, b);
    };

    MetaPtrs m(sm, meta_layout(p.in.max_tokens, g.meta_base));
    meta_prefetch<kTiledThreads>(p, s, m);
    if (warp == 0) {
        if (lane == 0) s_fail = 0;
        if (dec) {
            if (lane < S) {
                mbar_init(smem_addr(&bar_full[lane]), 1);
                mbar_init(smem_addr(&bar_empty[lane]), 1 + kTiledThreads / 32);
            }
            if (lane == 31) mbar_init(smem_addr(&bar_done), 1);
            if (lane == 30) mbar_init(smem_addr(&bar_drain), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            issued = min(S, nq);
            for (int q = 0; q < min(S, nq); ++q) {   // each stage's boxes from all lanes
                if (lane == 0) mbar_expect_tx(smem_addr(&bar_full[q]), stage_tx(q / nkb));
                __syncwarp();
                const int nb = boxes_of(q);
                for (int b = lane; b < nb; b += 32) issue_box(q, b);
            }
        }
    }
    meta_init_rest<kTiledThreads>(p, s, m);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

    if (dec) {
        const uint32_t tmem = tmem_base;
        // norms: a thread takes the rows tid, tid + 512 of (all A rows, this pass's B rows); |A| + nblk < 1024
        constexpr int kRows = 2;
        bool ok = true;
        for (int a = tid; a < s.nA; a += kTiledThreads) m.best[a] = 0ull;   // (each row's threads meet at barriers below)
        for (int ps = 0; ps < nP && ok; ++ps) {
            const int nB_p = pass_rows(ps), cols = (nB_p + 15) & ~15;
            const int nrA = ps == 0 ? s.nA : 0, nr = nrA + nB_p;
            float ss[kRows] = {}, sc[kRows] = {};
            for (int kb = 0; kb < nkb; ++kb) {
                const int q = ps * nkb + kb;
                const int st = q % S;
                const uint32_t par = (uint32_t)(q / S) & 1u;
                ok = ok && mbar_wait(smem_addr(&bar_full[st]), par);   // (as in k_image_tc)
                const unsigned char *stA = sm + (size_t)st * kbs, *stB = stA + aBytes;
                if (warp == 1 && elect_one() && ok) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(cols >> 3) << 17) | (8u << 24);
                    for (int mt = 0; mt < nM; ++mt) {
                        const uint32_t a0 = smem_addr(stA + (size_t)mt * 16384), b0 = smem_addr(stB);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            umma_bf16(tmem + (uint32_t)(mt * nblk), sw128_desc(a0 + k * 32), sw128_desc(b0 + k * 32), idesc,
                                      (kb | k) ? 1u : 0u);
                    }
                    umma_commit(smem_addr(&bar_empty[st]));
                    if (kb == nkb - 1) umma_commit(smem_addr(&bar_done));
                }
#pragma unroll
                for (int u = 0; u < kRows; ++u) {
                    const int r = tid + u * kTiledThreads;
                    if (r < nr) {
                        const bool isA = r < nrA;
                        const int rr = isA ? r : r - nrA;
                        const unsigned char *rb = (isA ? stA : stB) + rr * 128;
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            neumaier_add(ss[u], sc[u], chunk_sq(*reinterpret_cast<const uint4 *>(rb + ((j ^ (rr & 7)) << 4))));
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&bar_empty[st]));
                if (warp == 0 && q + S < nq) {   // refill this stage (possibly with the next pass's K-block)
                    ok = ok && mbar_wait(smem_addr(&bar_empty[st]), par);
                    if (elect_one() && ok) {
                        produce(q + S);
                        ++issued;
                    }
                    __syncwarp();
                }
            }
            if (!ok) atomicOr(&s_fail, 1);
#pragma unroll
            for (int u = 0; u < kRows; ++u) {
                const int r = tid + u * kTiledThreads;
                if (r < nr) {
                    const float sq = __fadd_rn(ss[u], sc[u]);
                    if (!isfinite(sq)) raise_status(p.status, FUSION_DEV_NONFINITE);
                    const float inv = 1.0f / fmaxf(sqrtf(sq), 1e-12f);
                    if (r < nrA)
                        m.inv_a[r] = inv;
                    else
                        m.inv_b[ps * nblk + r - nrA] = inv;
                }
            }
            __syncthreads();
            const bool mma_ok = s_fail == 0 && mbar_wait(smem_addr(&bar_done), (uint32_t)ps & 1u);
            if (!mma_ok) atomicOr(&s_fail, 2);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            __syncthreads();
            if (s_fail != 0) {
                ok = false;
                break;
            }
            // epilogue of the pass, M-tile by M-tile: thread -> A row (tid % 128); the four warpgroups split
            // the columns
            const int wg = tid >> 7, r = tid & 127;
            const int part_cols = ((cols / 16 + 3) / 4) * 16;
            const int c_lo = min(cols, wg * part_cols), c_hi = min(cols, c_lo + part_cols);
            for (int mt = 0; mt < nM; ++mt) {
                const uint32_t lane_addr = tmem + (uint32_t)(mt * nblk) + ((uint32_t)((warp & 3) * 32) << 16);
                const int arow = mt * 128 + r;
                const float ia = arow < s.nA ? m.inv_a[arow] : 0.0f;
                float bv = -INFINITY;   // as in k_image_tc: strict comparison over rising columns
                int bi = -1;
                for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
                    uint32_t v[16];
                    tmem_ld16(lane_addr + (uint32_t)c0, v);
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int col = ps * nblk + c0 + e;
                        if (c0 + e < nB_p) {
                            const float cs = (__uint_as_float(v[e]) * ia) * m.inv_b[col];
                            if (cs > bv || bi < 0) {
                                bv = cs;
                                bi = col;
                            }
                        }
                    }
                }
                part_best[tid] = (arow < s.nA && bi >= 0) ? rank_key(bv, bi) : 0ull;
                __syncthreads();
                if (wg == 0 && arow < s.nA) {   // (the larger key: the lower column among equal values)
                    unsigned long long o = m.best[arow];
#pragma unroll
                    for (int k = 0; k < 4; ++k) o = part_best[k * 128 + r] > o ? part_best[k * 128 + r] : o;
                    m.best[arow] = o;
                }
                __syncthreads();   // part_best is reused
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();   // the next pass's products overwrite the accumulators after this
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        if (s_fail != 0) {
            // a wait gave up: let the copies and products in flight land (bounded) before the
            // shared and tensor memory are released
            if (warp == 0 && elect_one()) {
                raise_status(p.status, FUSION_DEV_TIMEOUT);
                for (int q = max(0, issued - S); q < issued; ++q)
                    (void)mbar_wait(smem_addr(&bar_full[q % S]), (uint32_t)(q / S) & 1u);
            }
            if (warp == 1 && elect_one()) {   // the lane that issued the products: a commit covers only its own
                umma_commit(smem_addr(&bar_drain));
                (void)mbar_wait(smem_addr(&bar_drain), 0u);
            }
        } else {
            select_top_r<kTiledThreads>(s, m);
        }
        __syncthreads();
    }
    if (s_fail == 0) {
        const GlobalLoader<__nv_bfloat16> gl{reinterpret_cast<const __nv_bfloat16 *>(p.x), (long long)s.start, p.dim};
        finish_sample<__nv_bfloat16, kTiledThreads>(p, s, m, gl);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(g.tmem_cols)
                     : "memory");
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int ceil8(int v) { return (v + 7) & ~7; }

}  // namespace

namespace {
// Geometry of k_image_tc_tiled: one CTA per SM, a ring of [all A rows | a pass's B rows] stages.
TcGeometry tiled_geometry(int max_tokens, int kdim) {
    TcGeometry g{};
    const int nAmax = (max_tokens - 1) / 2, nBmax = max_tokens / 2;
    const int npad_max = (nBmax + 15) & ~15;
    g.tiled = 1;
    g.n_kb = kdim / 64;
    g.tmem_cols = 512;
    // the largest stage and the furthest read from its start over all samples of at most max_tokens: with
    // one M-tile less a pass has more columns
    size_t per_stage = 0, reach = 0;
#pragma unroll 1
    for (int nM = 1; nM <= (nAmax + 127) / 128; ++nM) {
        const int nblk = std::min(256, 512 / nM & ~15);
        const size_t a = (size_t)ceil8(std::min(nAmax, nM * 128)) * 128;
        per_stage = std::max(per_stage, a + (size_t)std::min(nblk, ceil8(nBmax)) * 128);
        reach = std::max({reach, (size_t)nM * 16384, a + (size_t)std::min(nblk, npad_max) * 128});
    }
    // one CTA per SM: all of its shared memory, the metadata at the end; at least two stages (shorter
    // samples of the call have more, from their own sizes): up to 962 tokens (64 samples of 960 tokens, d =
    // 384: 140 us, on the general kernel 699).  The stages end where the metadata begin: copies write whole
    // stages, and what a product reads past them feeds only unused rows and columns.
    const size_t usable = (227 * 1024 - 6144 - 1024) / 1024 * 1024;   // static shared memory, alignment
    const size_t meta = meta_layout(max_tokens, 0).total;
    if (2 * per_stage + meta > usable || per_stage + reach > usable) return TcGeometry{};
    g.meta_base = (uint32_t)((usable - meta) / 16 * 16);
    g.stage_region = g.meta_base;
    g.stages = (int)(g.stage_region / per_stage);
    g.usable = (uint32_t)usable;
    g.smem = g.usable + 1024;
    g.ok = 1;
    return g;
}
}  // namespace

TcGeometry image_tc_geometry(int dtype, int max_tokens, int kdim, int dim, long long max_rows, int do_merge,
                             int stage_budget_kb, int max_batch) {
    TcGeometry g{};
    if (dtype != FUSION_BF16 || !do_merge || kdim % 64 != 0 || max_rows < 2) return g;
    const int nAmax = (max_tokens - 1) / 2, nBmax = max_tokens / 2;
    if (nAmax > 128 || nBmax > 128) return tiled_geometry(max_tokens, kdim);
    g.n_kb = kdim / 64;
    g.full_rows = ceil8(nBmax > 0 ? nBmax : 1);
    g.kb_a = (uint32_t)ceil8(nAmax > 0 ? nAmax : 1) * 128u;
    g.kb_b = (uint32_t)ceil8(nBmax > 0 ? nBmax : 1) * 128u;
    int cols = 32;
    while (cols < ((nBmax + 15) & ~15)) cols <<= 1;
    g.tmem_cols = cols;
    const size_t per_stage = g.kb_a + g.kb_b;
    // the largest read from a stage base: 128 A rows, or half A and npad B rows
    const size_t npad_max = (size_t)((nBmax + 15) & ~15);
    const size_t reach = std::max<size_t>(16384, g.kb_a + npad_max * 128);
    // More samples than two CTAs per SM hold, each with at most 128 rows: CTAs of 128 threads with
    // four K-block stages, as many per SM as fit (the samples' chains of latencies overlap; a sample that does
    // not stay in shared memory is gathered from L2).  8192 samples of 9 to 65 tokens, d = 384, four stages
    // that keep 40 % each, per-sample kernels 452 -> 318 us; at 304 samples a CTA of 256 threads finishes its
    // sample sooner and every sample has one at once.  Where a sample's rows pass 68 KB, the few
    // samples past 304 may start as short ones end (305 samples of 2 to 65 tokens, d = 1024, merged: 256 threads 42
    // us, 128 46; 340 of them 53, 47; 305 of 2 to 33 tokens 33, 35).  Three CTAs per SM (100 tokens from d = 384)
    // do not halve the waves: they serve one wave of their own, up to 456 samples, and, with narrower rows, the
    // batches with a plan kernel (100 tokens, d = 384, merged, 256 / 128 threads: 400 samples 48 / 36 us, 500 52 /
    // 58, 608 54 / 62, 1100 93 / 87; d = 768: 500 samples 72 / 96).
    constexpr int kWave = 2 * kSms;
    if (max_batch > kWave && max_tokens <= 129) {
        auto small = [&](int S) {
            const size_t meta_base = (size_t)S * per_stage;
            return std::max(meta_layout(max_tokens, meta_base).total + (size_t)dim * 2, (size_t)(S - 1) * per_stage + reach);
        };
        const int S = std::min(g.n_kb, 4);
        for (int per_sm = 4; per_sm >= 3; --per_sm) {
            // 228 KB per SM, 1 KB of it reserved per CTA, 1 KB of alignment slack and the static arrays
            if (small(S) + 1024 + 1536 + 1024 > (size_t)228 * 1024 / per_sm) continue;
            const bool past_wave = max_batch > kWave + kWave / 16;
            if (per_sm == 4 ? 2 * dim * max_tokens > 68 * 1024 && !past_wave
                            : !past_wave || (max_batch > 3 * kSms && (max_batch <= kFusedPlanMaxBatch || dim > 384)))
                break;
            g.threads = 128;
            g.stages = S;
            g.stage_region = (uint32_t)(S * per_stage);
            g.meta_base = g.stage_region;
            g.cls_base = (uint32_t)meta_layout(max_tokens, g.meta_base).total;
            g.usable = (uint32_t)small(S);
            g.smem = g.usable + 1024;
            g.ok = 1;
            return g;
        }
    }
    g.threads = 256;
    size_t budget = (size_t)stage_budget_kb * 1024;
    if (budget > 227 * 1024 - 4096) budget = 227 * 1024 - 4096;   // room for static shared memory
    // usable bytes for S stages at max_tokens: the ring, the metadata, the CLS row (dim bf16)
    auto need = [&](int S) {
        const size_t meta_base = (size_t)S * per_stage + 2048;
        return std::max(meta_layout(max_tokens, meta_base).total + (size_t)dim * 2, (size_t)(S - 1) * per_stage + reach);
    };
    int S = g.n_kb < kMaxStages ? g.n_kb : kMaxStages;
    while (S > 2 && need(S) + 1024 > budget) --S;
    if (need(S) + 1024 > budget) return g;
    g.stages = S;
    g.stage_region = (uint32_t)(S * per_stage);
    g.meta_base = (uint32_t)(S * per_stage + 2048);
    g.cls_base = (uint32_t)meta_layout(max_tokens, g.meta_base).total;
    g.usable = (uint32_t)need(S);
    // The grouped layout for samples that fit: an MMA reads 128 A rows, 16 groups of n_kb KB from
    // the start of the buffer, and up to one group past half B (npad rows), so the buffer must
    // cover both; when the budget allows it, it does.
    const size_t gstride = (size_t)g.n_kb * 1024;
    const size_t g_need = std::max({(size_t)g.usable, 16 * gstride, (size_t)g.stage_region + gstride});
    if (g_need + 1024 <= budget) {
        g.grouped = 1;
        g.usable = (uint32_t)g_need;
    }
    g.smem = g.usable + 1024;
    g.ok = 1;
    return g;
}

cudaError_t launch_image_tc(const ImageParams &p, const TcGeometry &geometry, cudaStream_t s, bool pdl) {
    if (p.in.max_batch == 0) return cudaSuccess;
    // A small batch leaves SMs idle: up to four CTAs per sample, each making the sample's decisions (its
    // keys come from L2 after the first) and writing a quarter of the columns; nothing is exchanged.  The
    // gather and the means are 6 of the 24 us of one 197-token sample on its SM.
    TcGeometry g = geometry;
    g.parts = 1;
    // (a launch gate may stop a single CTA: its samples keep one)
    while (!p.gate && !g.tiled && g.parts < 4 && (long long)p.in.max_batch * (g.parts + 1) <= 2 * kSms && p.dim / 8 / (g.parts + 1) >= 8)
        ++g.parts;
    EncodeTiledFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    TcMaps maps{};
    const cuuint64_t rows_even = (cuuint64_t)((p.in.max_rows + 1) / 2), rows_odd = (cuuint64_t)(p.in.max_rows / 2);
    const char *keys = reinterpret_cast<const char *>(p.keys);
    CUtensorMap *const dsts[8] = {&maps.e32, &maps.o32, &maps.e8, &maps.o8, &maps.e256, &maps.o256, &maps.e128, &maps.o128};
    const int box[4] = {32, 8, g.tiled ? 256 : g.full_rows, g.tiled ? 128 : 64};
    for (int i = 0; i < 8; ++i) {
        const int odd = i & 1, box_rows = box[i >> 1];
        cuuint64_t dims[2] = {(cuuint64_t)p.kdim, odd ? rows_odd : rows_even};
        cuuint64_t strides[1] = {(cuuint64_t)p.kdim * 2 * 2};   // every other row
        cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
        cuuint32_t estr[2] = {1, 1};
        CUtensorMap *dst = dsts[i];
        void *base = const_cast<char *>(keys + (odd ? (size_t)p.kdim * 2 : 0));
        if (enc(dst, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
#pragma unroll 1
    for (int odd = 0; odd < 2 && g.grouped; ++odd) {   // (64 dims, row, K-block), box 8 rows x all K-blocks
        cuuint64_t dims[3] = {64, odd ? rows_odd : rows_even, (cuuint64_t)(p.kdim / 64)};
        cuuint64_t strides[2] = {(cuuint64_t)p.kdim * 2 * 2, 128};
        cuuint32_t box[3] = {64, 8, (cuuint32_t)(p.kdim / 64)};
        cuuint32_t estr[3] = {1, 1, 1};
        void *base = const_cast<char *>(keys + (odd ? (size_t)p.kdim * 2 : 0));
        if (enc(odd ? &maps.go : &maps.ge, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    auto kernel = g.tiled ? k_image_tc_tiled : g.threads == 128 ? k_image_tc<128> : k_image_tc<256>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem);
    if (e != cudaSuccess) return e;
    // the largest shared-memory carveout, so that both CTAs of an SM are resident from the start
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.in.max_batch * (unsigned)g.parts);
    cfg.blockDim = dim3(g.tiled ? kTiledThreads : g.threads);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, maps, p, g);
}

}  // namespace fz
