// Per-sample merge -> prune -> gather for float32 tokens: the similarity on FFMA with the key dims
// streamed through two to six cp.async stages, so that several CTAs share an SM (large batches of small
// samples), and clusters of CTAs per sample (small batches of long ones).
//
// A cluster of CL CTAs owns a sample.  Each takes a run of 16-row strips of half A against all of half
// B: warp tiles of 16 x 16 (a thread 2 rows x 4 columns, 6 shared-memory wavefronts per 32 FFMA), the
// accumulators in registers over the whole key width.  The row maxima go to every CTA of the cluster,
// each repeats the decisions (they are short), rank 0 writes the index outputs and every CTA a range of
// columns of the token rows.
//
// Sums are formed as the general kernel (image.cu) forms them, bit for bit: dot products in partial
// sums of 16 dims, squared norms per block of `kc` dims with chunk c of a block in lane c % 32.
//
// Bound by the chain of latencies of one sample (loads, FFMA, decisions, gather) and, with enough
// samples, by issue slots (8192 images of 65 tokens: 55 % busy; 29 % of the instructions are the similarity's FFMA).
// The general kernel keeps a whole sample in shared memory where it can, has one CTA
// of 512 threads per SM (its 128 registers) and gives 16 x 32 strips to warps, of which 65 tokens have two.  It stays
// the faster one for many batches of longer samples (image_f32_geometry has the rule).
// Measured, general kernel -> this one: 3277 of 8192 samples of 65 tokens, d = 384, continuing: 606 -> 219
// us (and 69 -> 29 us for the 210 that the fourth stage of that chain keeps); 8 samples of 197 tokens,
// keys of their own, clusters of 8, the stage with its exit check: 117 -> 45 us.  All with cold caches.
#include <cooperative_groups.h>

#include "sample.cuh"

namespace cg = cooperative_groups;

namespace fz {
namespace {

__host__ __device__ inline uint32_t stage_row(int kd) { return (uint32_t)(kd + 4) * 4u; }   // bytes; 16 (mod 32): 8 rows conflict-free

// The oldest of the S stages in flight has landed (this thread's part of it).
__device__ __forceinline__ void wait_stage(int S) {
    switch (S) {
    case 2: asm volatile("cp.async.wait_group 1;\n" ::: "memory"); break;
    case 3: asm volatile("cp.async.wait_group 2;\n" ::: "memory"); break;
    case 4: asm volatile("cp.async.wait_group 3;\n" ::: "memory"); break;
    case 5: asm volatile("cp.async.wait_group 4;\n" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 5;\n" ::: "memory"); break;   // kMaxStagesF32
    }
}
constexpr int kMaxStagesF32 = 6;

// NT threads; TPW warp tiles held in registers per pass; NP > 0: squared norms summed from the stages,
// NP rows per 16 threads (kd = 64, norm blocks of whole stages), else read again from global memory (L2).
template <int NT, int TPW, int NP>
__global__ void __launch_bounds__(NT, NT == 128 ? 4 : TPW == 1 ? 1 : 2) k_merge_f32(ImageParams p, F32Geometry g) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int kW = NT / 32;
    const int CL = g.cluster;
    const int rank = CL > 1 ? (int)(blockIdx.x % (unsigned)CL) : 0;
    SampleInfo s;
    if (!sample_begin<NT>(p, CL > 1 ? blockIdx.x / CL : blockIdx.x, s)) return;   // the same in every CTA of the cluster
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr bool kSplit = NP > 0 && NT == 256;
    const int kdim = p.kdim, kd = kSplit ? 64 : g.kd;
    const uint32_t rs = stage_row(kd);
    // this CTA's strips of half A
    const int strips = (s.nA + 15) / 16, per = (strips + CL - 1) / CL;
    const int a0 = min(s.nA, rank * per * 16), na = min(s.nA, a0 + per * 16) - a0;
    const uint32_t stage_bytes = (uint32_t)(g.rows_a + g.rows_b) * rs;
    unsigned char *const st0 = sm;
    const int S = g.stages;
    MetaPtrs m(sm, meta_layout(p.in.max_tokens, (size_t)S * stage_bytes));
    const float *keys = reinterpret_cast<const float *>(p.keys);

    const int n_stage = (kdim + kd - 1) / kd;
    const int rows = na + s.nB;
    // stage q: dims [q kd, ..) of the CTA's A rows, then of all B rows
    auto issue = [&](int q) {
        unsigned char *dst = st0 + (q % S) * stage_bytes;
        const int nch = min(kd, kdim - q * kd) / 4;
        int row = tid / nch, c = tid - row * nch;
        const int rstep = NT / nch, cstep = NT - rstep * nch;
        while (row < rows) {
            const bool isA = row < na;
            const int tok = isA ? a0 + row : row - na;
            const long long grow = s.start + (isA ? 2 + 2 * tok : 1 + 2 * tok);
            cp_async16(dst + (uint32_t)(isA ? row : g.rows_a + tok) * rs + c * 16, keys + grow * kdim + q * kd + c * 4);
            row += rstep;
            c += cstep;
            if (c >= nch) {
                c -= nch;
                ++row;
            }
        }
        cp_async_commit();
    };
    // a pass begins with S stages in flight; every stage is one commit group, empty past the last
    auto start = [&] {
#pragma unroll 1
        for (int q = 0; q < S; ++q) {
            if (q < n_stage) issue(q);
            else cp_async_commit();
        }
    };
    const int MT = (na + 15) / 16, NG = (s.nB + 15) / 16, tiles = MT * NG;
    const int n_pass = (tiles + kW * TPW - 1) / (kW * TPW);
    const bool sim = s.decide && na > 0;
    if (sim) start();
    meta_init<NT>(p, s, m);
    __syncthreads();
    if (s.decide) {
        // A thread's two rows and four columns of a tile.  kSplit (kd = 64): half of the warp sums the even
        // 16-dim blocks, the other half the odd ones, of 4 rows x 4 columns per thread (8 shared-memory
        // loads per 64 FFMA; 2 rows x 4 columns of every block take 12), and they swap the partial sums of
        // each other's rows: every sum is formed from the same terms in the same order.  8 samples of 197
        // tokens in clusters of 8, the stage: 49.1 -> 47.3 us.  Not with 128 threads, where the registers are
        // needed for the CTAs of an SM: the chain of stages on 8192 samples 518 us instead of 516 at four CTAs,
        // 554 instead of 537 at five.
        const int h = lane >> 4, t4 = lane & 3;
        const int g8 = kSplit ? ((lane >> 2) & 3) + 8 * h : lane >> 2;
        constexpr int kRowStep = kSplit ? 4 : 8;
        float nlo[NP > 0 ? NP : 1], nhi[NP > 0 ? NP : 1];
#pragma unroll
        for (int k = 0; k < (NP > 0 ? NP : 1); ++k) nlo[k] = nhi[k] = 0.0f;
#pragma unroll 1
        for (int pass = 0; sim && pass < n_pass; ++pass) {
            if (pass > 0) start();
            float acc[TPW][2][4];
#pragma unroll
            for (int w = 0; w < TPW; ++w)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[w][i][e] = 0.0f;
#pragma unroll 1
            for (int q = 0; q < n_stage; ++q) {
                wait_stage(S);
                __syncthreads();
                const unsigned char *st = st0 + (q % S) * stage_bytes;
                const int kw = min(kd, kdim - q * kd);   // a multiple of 16
#pragma unroll
                for (int w = 0; w < TPW; ++w) {
                    const int tile = (pass * TPW + w) * kW + warp;
                    if (tile >= tiles) continue;
                    const int mt = tile / NG, ng = tile - mt * NG;
                    // rows past the halves read stale or unwritten shared memory inside the stage: their
                    // products are never used
                    if constexpr (kSplit) {
                        const unsigned char *rb = st + (uint32_t)(g.rows_a + ng * 16 + t4) * rs + h * 64;
                        const unsigned char *own = st + (uint32_t)(mt * 16 + g8) * rs + h * 64;
                        const unsigned char *oth = st + (uint32_t)(mt * 16 + (g8 ^ 8)) * rs + h * 64;
#pragma unroll 1
                        for (int k0 = 0; k0 < kw; k0 += 32) {
                            const bool odd = k0 + 16 < kw;   // uniform: a second block
                            float t[4][4] = {};
                            if (h == 0 || odd) {
#pragma unroll
                                for (int kk = 0; kk < 16; kk += 4) {
                                    const uint32_t o = (uint32_t)(k0 + kk) * 4;
                                    float4 a[4];
                                    a[0] = *reinterpret_cast<const float4 *>(own + o);
                                    a[1] = *reinterpret_cast<const float4 *>(own + 4 * rs + o);
                                    a[2] = *reinterpret_cast<const float4 *>(oth + o);
                                    a[3] = *reinterpret_cast<const float4 *>(oth + 4 * rs + o);
#pragma unroll
                                    for (int e = 0; e < 4; ++e) {
                                        const float4 b = *reinterpret_cast<const float4 *>(rb + (uint32_t)(4 * e) * rs + o);
#pragma unroll
                                        for (int i = 0; i < 4; ++i) {
                                            t[i][e] = fmaf(a[i].x, b.x, t[i][e]);
                                            t[i][e] = fmaf(a[i].y, b.y, t[i][e]);
                                            t[i][e] = fmaf(a[i].z, b.z, t[i][e]);
                                            t[i][e] = fmaf(a[i].w, b.w, t[i][e]);
                                        }
                                    }
                                }
                            }
                            __syncwarp();
#pragma unroll
                            for (int i = 0; i < 2; ++i)
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    const float got = __shfl_xor_sync(0xFFFFFFFFu, t[i + 2][e], 16);
                                    acc[w][i][e] += h ? got : t[i][e];
                                    if (odd) acc[w][i][e] += h ? t[i][e] : got;
                                }
                        }
                        continue;
                    }
                    const unsigned char *ra = st + (uint32_t)(mt * 16 + g8) * rs;
                    const unsigned char *rb = st + (uint32_t)(g.rows_a + ng * 16 + t4) * rs;
#pragma unroll 1
                    for (int k0 = 0; k0 < kw; k0 += 16) {
                        float t[2][4] = {};
#pragma unroll
                        for (int kk = 0; kk < 16; kk += 4) {
                            const uint32_t o = (uint32_t)(k0 + kk) * 4;
                            const float4 va = *reinterpret_cast<const float4 *>(ra + o);
                            const float4 vb = *reinterpret_cast<const float4 *>(ra + 8 * rs + o);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float4 b = *reinterpret_cast<const float4 *>(rb + (uint32_t)(4 * e) * rs + o);
                                t[0][e] = fmaf(va.x, b.x, t[0][e]);
                                t[1][e] = fmaf(vb.x, b.x, t[1][e]);
                                t[0][e] = fmaf(va.y, b.y, t[0][e]);
                                t[1][e] = fmaf(vb.y, b.y, t[1][e]);
                                t[0][e] = fmaf(va.z, b.z, t[0][e]);
                                t[1][e] = fmaf(vb.z, b.z, t[1][e]);
                                t[0][e] = fmaf(va.w, b.w, t[0][e]);
                                t[1][e] = fmaf(vb.w, b.w, t[1][e]);
                            }
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i)
#pragma unroll
                            for (int e = 0; e < 4; ++e) acc[w][i][e] += t[i][e];
                    }
                }
                if constexpr (NP > 0) {   // chunk c = 16 qb + l of the norm block: lane c % 32 of the general kernel's sum
                    const int l = tid & 15, r0 = tid >> 4;
                    const int per_block = (p.kc + kd - 1) / kd, qb = q % per_block;   // stages of a norm block
                    if (pass == 0 && l * 4 < kw) {
#pragma unroll
                        for (int k = 0; k < NP; ++k) {
                            const int row = r0 + k * (NT / 16);
                            if (row >= rows) continue;
                            const float4 f = *reinterpret_cast<const float4 *>(
                                st + (uint32_t)(row < na ? row : g.rows_a + row - na) * rs + l * 16);
                            float v = (qb & 1) ? nhi[k] : nlo[k];
                            v = fmaf(f.x, f.x, v);
                            v = fmaf(f.y, f.y, v);
                            v = fmaf(f.z, f.z, v);
                            v = fmaf(f.w, f.w, v);
                            if (qb & 1) nhi[k] = v;
                            else nlo[k] = v;
                        }
                    }
                    if (pass == 0 && (qb == per_block - 1 || q == n_stage - 1)) {   // the block's sum joins the row's
#pragma unroll
                        for (int k = 0; k < NP; ++k) {
                            float v = nlo[k] + nhi[k];
#pragma unroll
                            for (int o = 8; o >= 1; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
                            const int row = r0 + k * (NT / 16);
                            if (l == 0 && row < rows) {
                                float *ss = row < na ? m.inv_a + a0 + row : m.inv_b + row - na;
                                *ss = q < per_block ? v : *ss + v;
                            }
                            nlo[k] = nhi[k] = 0.0f;
                        }
                    }
                }
                __syncthreads();   // everyone is done with this stage
                if (q + S < n_stage) issue(q + S);
                else cp_async_commit();   // an empty group keeps the count
            }
            if (pass == 0) {
                // inverse norms of the CTA's A rows and of the B rows
                auto put = [&](int row, float v) {
                    if (!isfinite(v)) raise_status(p.status, FUSION_DEV_NONFINITE);
                    const float inv = 1.0f / fmaxf(sqrtf(v), 1e-12f);
                    if (row < na) m.inv_a[a0 + row] = inv;
                    else m.inv_b[row - na] = inv;
                };
                if constexpr (NP > 0) {
#pragma unroll 1
                    for (int row = tid; row < rows; row += NT)   // after the last stage's barrier
                        put(row, row < na ? m.inv_a[a0 + row] : m.inv_b[row - na]);
                } else {
                    // four rows at a time, so that their loads are in flight together
#pragma unroll 1
                    for (int row0 = warp; row0 < rows; row0 += 4 * kW) {
                        const float4 *src[4];
                        float v[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const int row = min(row0 + u * kW, rows - 1), tok = row < na ? a0 + row : row - na;
                            src[u] = reinterpret_cast<const float4 *>(
                                keys + (long long)(s.start + (row < na ? 2 + 2 * tok : 1 + 2 * tok)) * kdim);
                            v[u] = 0.0f;
                        }
#pragma unroll 1
                        for (int k0 = 0; k0 < kdim; k0 += p.kc) {
                            const int nch = min(p.kc, kdim - k0) / 4;
                            float sq[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 2
                            for (int c = lane; c < nch; c += 32)
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    const float4 f = __ldg(src[u] + k0 / 4 + c);
                                    sq[u] = fmaf(f.x, f.x, sq[u]);
                                    sq[u] = fmaf(f.y, f.y, sq[u]);
                                    sq[u] = fmaf(f.z, f.z, sq[u]);
                                    sq[u] = fmaf(f.w, f.w, sq[u]);
                                }
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
#pragma unroll
                                for (int o = 16; o >= 1; o >>= 1) sq[u] += __shfl_xor_sync(0xFFFFFFFFu, sq[u], o);
                                v[u] += sq[u];
                            }
                        }
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            if (lane == u && row0 + u * kW < rows) put(row0 + u * kW, v[u]);
                    }
                }
                __syncthreads();
            }
            // cosine and row maximum with the lowest column on ties: every tile leaves its 16 rows' maxima in
            // the stages (all read by now), a thread per row takes the largest (no
            // slower and no faster than 64-bit atomic maxima, and no entries to clear).
            unsigned long long *tile_best = reinterpret_cast<unsigned long long *>(st0);
            const int tile0 = pass * TPW * kW;
#pragma unroll
            for (int w = 0; w < TPW; ++w) {
                const int tile = (pass * TPW + w) * kW + warp;
                if (tile >= tiles) continue;
                const int mt = tile / NG, ng = tile - mt * NG;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int row = mt * 16 + g8 + kRowStep * i;
                    unsigned long long bk = 0ull;
                    if (row < na) {
                        const float ia = m.inv_a[a0 + row];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int col = ng * 16 + t4 + 4 * e;
                            if (col < s.nB) {
                                const unsigned long long k = rank_key((acc[w][i][e] * ia) * m.inv_b[col], col);
                                bk = k > bk ? k : bk;
                            }
                        }
                    }
                    unsigned long long o = __shfl_xor_sync(0xFFFFFFFFu, bk, 1);
                    bk = o > bk ? o : bk;
                    o = __shfl_xor_sync(0xFFFFFFFFu, bk, 2);
                    bk = o > bk ? o : bk;
                    if (t4 == 0) tile_best[(tile - tile0) * 16 + g8 + kRowStep * i] = bk;   // 0 for rows past the CTA's share
                }
            }
            __syncthreads();
            const int tile1 = min(tiles, tile0 + TPW * kW);
#pragma unroll 1
            for (int a = tid; a < na; a += NT) {
                const int t0 = (a >> 4) * NG;
                unsigned long long o = m.best[a0 + a];
#pragma unroll 1
                for (int t = max(t0, tile0); t < min(t0 + NG, tile1); ++t) {
                    const unsigned long long b = tile_best[(t - tile0) * 16 + (a & 15)];
                    o = b > o ? b : o;
                }
                m.best[a0 + a] = o;
            }
            __syncthreads();   // the next pass's copies overwrite the stages
        }
        if (CL > 1) {   // this CTA's row maxima to the others
            cg::cluster_group cl = cg::this_cluster();
            cl.sync();   // every CTA has initialised its maxima
#pragma unroll 1
            for (int t = tid; t < na * (CL - 1); t += NT) {
                const int k = t / na, a = a0 + t - k * na;
                *cl.map_shared_rank(m.best + a, k < rank ? k : k + 1) = m.best[a];
            }
            cl.sync();   // all maxima here; no CTA reads another's shared memory after this
        }
        select_top_r<NT>(s, m);
    }
    const GlobalLoader<float> ld{reinterpret_cast<const float *>(p.x), (long long)s.start, p.dim};
    if (!finish_decide<NT>(p, s, m)) return;
    if (rank == 0) write_index_outputs<NT>(p, s, m);
    const int w = p.dim / 4;
    write_rows<float, NT>(p, s, m, ld, w * rank / CL, w * (rank + 1) / CL);
}

template <int NT, int TPW, int NP>
cudaError_t launch(const ImageParams &p, const F32Geometry &g, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_merge_f32<NT, TPW, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_merge_f32<NT, TPW, NP>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)p.in.max_batch * (unsigned)g.cluster);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = g.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = g.cluster > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k_merge_f32<NT, TPW, NP>, p, g);
}

constexpr int kSmallTokens = 65;   // four 16 x 16 tiles: four warps, one tile each

}  // namespace

F32Geometry image_f32_geometry(const ImageParams &p) {
    F32Geometry g{};
    const int nA = (p.in.max_tokens - 1) / 2, nB = p.in.max_tokens / 2;
    const int N = p.in.max_tokens, B = p.in.max_batch;
    const bool small = N <= kSmallTokens;
    const int strips = ceil_div(nA > 0 ? nA : 1, 16), cols = ceil_div(nB > 0 ? nB : 1, 16);
    // CTAs per sample (portable cluster sizes), each with a strip at least; a gate may stop a single CTA, which a
    // cluster cannot.  A cluster lies in one GPC: 15 clusters of 8, 36 of 4 or 76 of 2 have an SM per CTA at once,
    // twice as many share SMs (cudaOccupancyMaxActiveClusters), and one more begins a second wave (76 samples of
    // 100 tokens, d = 384, in clusters of 4 82 us, of 2 50).
    auto fits = [&](int cl, int most) { return !p.gate && cl <= strips + 1 && B <= most; };
    // With an SM each they are the fastest form measured, except that pairs have half of the general kernel's
    // threads per SM for the decisions, which samples with narrow keys spend their time on once a warp has more than
    // a tile (76 samples of 300 tokens, d = 48: 64 us, general kernel 51).
    const bool narrow = p.kdim < 192, one_tile = N <= kSmallTokens + 1;
    // Two per SM gain less: where the similarity is nearly all of the time (60 samples of 197 tokens, d = 192:
    // clusters of 4 59 us, of 2 68; 100 tokens 48 and 36; past 600 tokens the stages are 16 dims: 700 tokens, d =
    // 384, 627 and 502), in pairs where a pass's 64 tiles are three quarters used (100 samples, d = 384: 577 tokens
    // 566 us, general kernel 620; 257 tokens 141 and 126) ...
    const int pair_tiles = ceil_div(strips, 2) * cols;
    const bool full = 4 * pair_tiles >= 3 * 64 * ceil_div(pair_tiles, 64);
    const bool four = N > 150 && N <= 600, two = four && !narrow && full;
    // ... and in a call with an exit check, whose samples that leave free the SMs (half of the batch continuing:
    // 20 samples of 197 tokens, d = 384, clusters of 8 52 us, of 4 77; 100 of 100 tokens pairs 51 us, general kernel
    // 62; everyone continuing 73 and 60 of the 77 that the call took before either), up to where the whole batch
    // would be slower than the general kernel and the exit check before were (64 samples of 65 to 130 tokens, d = 48:
    // clusters of 4 40 us, 36 before; 152 of 50 to 100 tokens, d = 384, merge and exit check, pairs 70 us, 66 before).
    const bool exits = p.plan_args.exit_mask != nullptr && !narrow;
    const bool exit2 = exits && !one_tile && N <= 600 && (N <= 129 ? p.kdim < 768 && B <= 114 : N <= 197 || full);
    g.cluster = fits(8, exits ? 30 : 15) ? 8
                : fits(4, four || exits ? 72 : 36) ? 4
                : fits(2, two || exit2 ? 152 : narrow && pair_tiles > 8 ? 0 : 76) ? 2
                : 1;
    // One CTA per sample with more than eight tiles: 256 threads against the general kernel's 512, but two CTAs
    // per SM where that has one.  In a wave of at most 152 samples each CTA is alone and slower (300 tokens,
    // d = 384: 354 us, general kernel 203); between 153 and 304 it needs one wave instead of two (197 tokens,
    // d = 384, 200 samples: 180 us, general kernel 202), from 305 to 456 two against three (340 samples 333,
    // 289); past that the waves even out (608 samples of 100 tokens, d = 384: 159, 175) until the long samples'
    // decisions take over (257 tokens, d = 192, half of 608 continuing: 215, 191).  How many continue is known here
    // only without an exit check and without a device count; else 153 to 456 samples may leave one wave, which
    // costs nothing up to 80 tokens and d = 384 (100 of 200 samples: 73 us, at the start's general kernel 72).
    const bool known = !p.in.batch && !p.plan_args.exit_mask;
    const bool few_waves = (known && B <= 2 * 152) || (N <= 80 && !narrow && p.kdim <= 384);
    if (g.cluster == 1 && !one_tile && !(N <= 197 && B > 152 && (B > 3 * 152 || few_waves))) return g;
    g.rows_a = ceil_div(strips, g.cluster) * 16;
    g.rows_b = cols * 16;
    auto need = [&](int kd, int S) {
        return meta_layout(p.in.max_tokens, (size_t)S * (g.rows_a + g.rows_b) * stage_row(kd)).total;
    };
    g.small = small;
    // two CTAs per SM where 16 dims allow it; a batch that leaves SMs idle has each to itself, and more
    // stages (a loop of six 64-dim stages took 12.4 of the kernel's 30 us with two in flight, most of it the
    // wait for them)
    const bool alone = B <= (g.cluster == 4 ? 36 : 152 / g.cluster);
    const size_t most = 224 * 1024;
    for (size_t budget : {alone ? most : (size_t)110 * 1024, most})
        for (int kd = 64; kd >= 16; kd /= 2) {
            if (need(kd, 2) > budget) continue;
            g.kd = kd;
            g.stages = 2;
            const int n_stage = ceil_div(p.kdim, kd);
            while (alone && g.stages < kMaxStagesF32 && g.stages < n_stage && need(kd, g.stages + 1) <= most) ++g.stages;
            g.smem = need(kd, g.stages);
            g.ok = 1;
            return g;
        }
    return g;
}

cudaError_t launch_image_f32(const ImageParams &p, const F32Geometry &g, cudaStream_t s) {
    if (p.in.max_batch == 0) return cudaSuccess;
    // norms from the stages: whole stages per norm block, at most 8 rows per 16 threads
    const bool norms = g.kd == 64 && (p.kc == p.kdim || p.kc % 64 == 0);
    if (g.small && g.cluster == 1) return norms ? launch<128, 1, 8>(p, g, s) : launch<128, 1, 0>(p, g, s);
    if ((g.rows_a / 16) * (g.rows_b / 16) <= 8)   // a tile per warp
        return norms && g.rows_a + g.rows_b <= 128 ? launch<256, 1, 8>(p, g, s) : launch<256, 1, 0>(p, g, s);
    return launch<256, 8, 0>(p, g, s);
}

}  // namespace fz
