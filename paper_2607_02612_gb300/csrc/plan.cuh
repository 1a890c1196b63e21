// The per-call plan: validates the ragged batch, decides which samples continue,
// computes every sample's output token count and scans them into the output
// offsets.  Output counts follow from the inputs alone: merging removes
// r_eff = clamp(r, 0, floor(P/2)) tokens (Sec. III-C) and pruning then keeps
// 1 + ceil(rho * P') (Sec. III-E), so the scan needs no merge decision.
#pragma once

#include "common.cuh"

namespace fz {

struct PlanArgs {
    Ragged in;
    int merge;                 // counts include merging
    int prune;                 // counts include pruning
    const int *r;              // [*] merge counts (by original id)
    const float *rho;          // [*] keep ratios (by original id)
    const uint8_t *exit_mask;  // [B] 1 = exits (leaves the batch); NULL = all continue
    int *offsets_out;          // [max_batch + 1]
    int *ids_out;              // [max_batch] or NULL
    int *batch_out;            // device scalar or NULL
    // batches above the fused plan's bound (scratch in the workspace):
    int *cnt;                  // [max_batch]: output rows of every input sample, -1 if gone
    int4 *agg;                 // [tiles of pt samples]: survivors and rows before the tile (x, y)
    int *plan;                 // [4]: ok flag, survivor count
    int *counter;              // zero between calls
    int pt;                    // samples per tile (32 or 64)
    int *status;
};

constexpr int kPlanRhoNonfinite = 1 << 30;   // a continuing sample's keep ratio is NaN or infinite

// The plan of a batch above the fused plan's bound, in tiles of pt samples.  plan_tile, one warp:
// a tile's output counts and its totals.  plan_scan, one block once every tile is done: the totals
// become exclusive prefixes, and the batch-level outputs are written.  The per-sample kernel adds
// the prefix inside its tile itself (sample_live), so no serial pass over the samples remains:
// one block over 8192 samples took about 20 us, the tiles run beside one another in the kernel that
// makes the exit decisions and the scan of 128 totals takes about 2.
//
// plan_count: the output rows of sample i if it continues (its merge and prune counts are inputs of
// the call, so a kernel can take them before it knows who continues), 0 with `bits` set when its
// offsets or id are malformed.
__device__ __forceinline__ int plan_count(const PlanArgs &a, int i, int &bits) {
    const int o0 = a.in.offsets[i], o1 = a.in.offsets[i + 1];
    const int id = a.in.ids ? a.in.ids[i] : i;
    const int N = o1 - o0;
    const bool ok = o0 >= 0 && N >= 1 && N <= a.in.max_tokens && (long long)o1 <= a.in.max_rows;
    const bool id_ok = id >= 0 && id < a.in.max_batch;
    if (!ok) bits |= FUSION_DEV_BAD_OFFSETS;
    if (!id_ok) bits |= FUSION_DEV_BAD_IDS;
    if (!ok || !id_ok) return 0;
    int c = N;
    if (a.merge) c -= merge_count(a.r[id], N - 1);
    if (a.prune) {
        bool f = false;
        c = 1 + keep_count(a.rho[id], c - 1, f);
        if (f) bits |= kPlanRhoNonfinite;
    }
    return c;
}

// Tile t of the plan by one warp: lane and lane + 32 bring their samples' counts (-1: gone, or
// beyond the batch count B) and bits.
__device__ __forceinline__ void plan_tile(const PlanArgs &a, int t, int B, const int (&c)[2], int bits) {
    const int lane = threadIdx.x & 31;
    int surv = 0, rows = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = lane + 32 * h, i = t * a.pt + k;
        if (k >= a.pt || i >= B) continue;
        a.cnt[i] = c[h];
        if (c[h] >= 0) {
            ++surv;
            rows += c[h];
        }
    }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        surv += __shfl_xor_sync(0xFFFFFFFFu, surv, m);
        rows += __shfl_xor_sync(0xFFFFFFFFu, rows, m);
        bits |= __shfl_xor_sync(0xFFFFFFFFu, bits, m);
    }
    if (lane == 0) a.agg[t] = make_int4(surv, rows, bits, 0);
}

// Run by one block (any size, a multiple of 32); B: the device batch count, -1 when out of range.
__device__ inline void plan_scan(const PlanArgs &a, int B) {
    __shared__ int wsum[2][32], s_bad;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nw = blockDim.x >> 5;
    if (t == 0) s_bad = 0;
    __syncthreads();
    const int tiles = B > 0 ? (B + a.pt - 1) / a.pt : 0;
    int base_s = 0, base_r = 0;
#pragma unroll 1
    for (int t0 = 0; t0 < tiles; t0 += blockDim.x) {
        int4 v = make_int4(0, 0, 0, 0);
        if (t0 + t < tiles) v = __ldcg(a.agg + t0 + t);
        if (v.z) atomicOr(&s_bad, v.z);
        int is = v.x, ir = v.y;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int ys = __shfl_up_sync(0xFFFFFFFFu, is, o), yr = __shfl_up_sync(0xFFFFFFFFu, ir, o);
            if (lane >= o) {
                is += ys;
                ir += yr;
            }
        }
        if (lane == 31) {
            wsum[0][w] = is;
            wsum[1][w] = ir;
        }
        __syncthreads();
        int ps = base_s, pr = base_r, ts = 0, tr = 0;
#pragma unroll 1
        for (int k = 0; k < nw; ++k) {
            if (k < w) {
                ps += wsum[0][k];
                pr += wsum[1][k];
            }
            ts += wsum[0][k];
            tr += wsum[1][k];
        }
        if (t0 + t < tiles) a.agg[t0 + t] = make_int4(ps + is - v.x, pr + ir - v.y, 0, 0);
        base_s += ts;
        base_r += tr;
        __syncthreads();   // wsum is reused by the next round
    }
    if (t == 0) {
        const int bits = s_bad & ~kPlanRhoNonfinite;
        const bool bad = B < 0 || bits != 0;
        a.offsets_out[bad ? 0 : base_s] = bad ? 0 : base_r;
        if (a.batch_out) *a.batch_out = bad ? 0 : base_s;
        a.plan[0] = bad ? 0 : 1;
        a.plan[1] = bad ? 0 : base_s;
        if (B < 0) raise_status(a.status, FUSION_DEV_BAD_BATCH);
        if (bits) raise_status(a.status, bits);
        if (s_bad & kPlanRhoNonfinite) raise_status(a.status, FUSION_DEV_NONFINITE);
    }
}

}  // namespace fz
