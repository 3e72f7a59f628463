// Dual routing (expert gate top-k + per-expert bit-width choice, Section 3.2) and the stable
// grouping of assignments by (expert, width); its histogram is B_{j,k} of Section 3.4.3.
#include "d2moe_common.cuh"
#include "tc_common.cuh"
#include "group_block.cuh"

#include <type_traits>

namespace {

constexpr int MAX_TOPK = 8;
constexpr int MAX_E_PER_LANE = 8;        // up to 256 experts

// fp32 dot product in the pinned order: lane l accumulates elements l, l+32, ... with one fused
// multiply-add each, then a butterfly reduction with offsets 16, 8, 4, 2, 1.
__device__ __forceinline__ float dot_pinned(const __nv_bfloat16* __restrict__ a,
                                            const __nv_bfloat16* __restrict__ b, int d, int lane) {
    float acc = 0.0f;
    for (int i = lane; i < d; i += 32)
        acc = fmaf(__bfloat162float(a[i]), __bfloat162float(b[i]), acc);
    for (int off = 16; off; off >>= 1) acc = acc + __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
}

// One warp: the gate of one token from its logits (lane l holds the logits of experts l, l + 32, ...).
// k rounds of arg-max over the remaining logits, ties to the lower index (shuffle reduction); softmax over
// all experts, gathered at the selected ones.  Outputs in every lane: sel[s], w[s] (not renormalised) and
// their sum; a NaN or an infinity among the logits raises D2MOE_DEV_NONFINITE.
__device__ __forceinline__ void gate_select(const float (&lg)[MAX_E_PER_LANE], int E, int k, int lane,
                                            int (&sel)[MAX_TOPK], float (&w)[MAX_TOPK], float& wsum,
                                            int32_t* __restrict__ device_status) {
    bool bad = false;
#pragma unroll
    for (int m = 0; m < MAX_E_PER_LANE; ++m)
        if (lane + 32 * m < E && !isfinite(lg[m])) bad = true;
    if (__any_sync(0xffffffffu, bad) && lane == 0 && device_status) atomicOr(device_status, D2MOE_DEV_NONFINITE);

    unsigned taken = 0;
    float selv[MAX_TOPK];
#pragma unroll
    for (int s = 0; s < MAX_TOPK; ++s) {
        sel[s] = 0; selv[s] = 0.0f;
        if (s < k) {
            float bv = -INFINITY; int bi = 0x7fffffff;
#pragma unroll
            for (int m = 0; m < MAX_E_PER_LANE; ++m) {
                const int e = lane + 32 * m;
                if (e < E && !((taken >> m) & 1u)) {
                    if (bi == 0x7fffffff || lg[m] > bv) { bv = lg[m]; bi = e; }
                }
            }
            for (int off = 16; off; off >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
                const bool take = (oi != 0x7fffffff) &&
                                  (bi == 0x7fffffff || ov > bv || (ov == bv && oi < bi));
                if (take) { bv = ov; bi = oi; }
            }
            sel[s] = bi; selv[s] = bv;
            if ((bi & 31) == lane) taken |= 1u << (bi >> 5);
        }
    }
    const float mx = selv[0];
    float part = 0.0f;
#pragma unroll
    for (int m = 0; m < MAX_E_PER_LANE; ++m)
        if (lane + 32 * m < E) part += expf(lg[m] - mx);
    for (int off = 16; off; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
    wsum = 0.0f;
#pragma unroll
    for (int s = 0; s < MAX_TOPK; ++s) {
        w[s] = 0.0f;
        if (s < k) { w[s] = expf(selv[s] - mx) / part; wsum += w[s]; }
    }
}

// One warp per token.
__global__ void __launch_bounds__(128)
route_kernel(MoeDims D, const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ gate_w,
             const float* __restrict__ logits_in, const __nv_bfloat16* __restrict__ bit_w,
             const int8_t* __restrict__ forced, RouteBufs R, int32_t* __restrict__ keys,
             int32_t* __restrict__ device_status) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= D.T) return;
    const int E = D.E;
    const __nv_bfloat16* xt = x + (size_t)t * D.d;

    float lg[MAX_E_PER_LANE];
#pragma unroll
    for (int m = 0; m < MAX_E_PER_LANE; ++m) lg[m] = -INFINITY;
    if (logits_in) {
#pragma unroll
        for (int m = 0; m < MAX_E_PER_LANE; ++m) {
            const int e = lane + 32 * m;
            if (e < E) lg[m] = logits_in[(size_t)t * E + e];
        }
    } else {
        for (int e = 0; e < E; ++e) {
            const float v = dot_pinned(xt, gate_w + (size_t)e * D.d, D.d, lane);
#pragma unroll
            for (int m = 0; m < MAX_E_PER_LANE; ++m)
                if (m == (e >> 5) && lane == (e & 31)) lg[m] = v;
        }
    }
    int sel[MAX_TOPK];
    float w[MAX_TOPK];
    float wsum;
    gate_select(lg, E, D.k, lane, sel, w, wsum, device_status);

    // bit-width choice per selected expert
#pragma unroll
    for (int s = 0; s < MAX_TOPK; ++s) {
        if (s < D.k) {
            const int a = t * D.k + s;
            int kk;
            if (forced) {
                kk = forced[a];
                if (kk < 0 || kk >= D.K) {
                    if (lane == 0 && device_status) atomicOr(device_status, D2MOE_DEV_BAD_INDEX);
                    kk = kk < 0 ? 0 : D.K - 1;
                }
            } else {
                float best = 0.0f; kk = 0;
                for (int c = 0; c < D.K; ++c) {
                    const float u = dot_pinned(xt, bit_w + ((size_t)sel[s] * D.K + c) * D.d, D.d, lane);
                    if (c == 0 || u > best) { best = u; kk = c; }
                }
            }
            if (lane == 0) {
                R.topk_idx[a] = sel[s];
                R.topk_w[a] = D.renormalize ? w[s] / wsum : w[s];
                R.bit_idx[a] = (int8_t)kk;
                keys[a] = sel[s] * D.K + kk;
            }
        }
    }
}

// Bit-width choice of every (token, selected expert) pair for many tokens: eight lanes per pair, which read the token's row and
// the expert's width rows straight from memory (8 bytes per load: lane q carries the chains 4q .. 4q + 3 of the pinned order), four
// rows at a time.  No shared memory and no barrier, so that all pairs are in flight; bound by the rows' trip from L2.
// (Staged in shared memory by a block per token, three barriers each: 65 us for 9000 pairs of 3 rows x 2048.)
__global__ void __launch_bounds__(128)
width_router_kernel(MoeDims D, const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ bit_w, RouteBufs R,
                    int32_t* __restrict__ keys) {
    pdl_enter();
    const int q = threadIdx.x & 7, a = blockIdx.x * 16 + (threadIdx.x >> 3);
    const int ac = min(a, D.A - 1), t = ac / D.k, e = R.topk_idx[ac];
    const uint2* xr = reinterpret_cast<const uint2*>(x + (size_t)t * D.d) + q;
    const __nv_bfloat16* w0 = bit_w + (size_t)e * D.K * D.d;
    float best = 0.0f;
    int kk = 0;
    for (int c0 = 0; c0 < D.K; c0 += 4) {
        const uint2* wr[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) wr[r] = reinterpret_cast<const uint2*>(w0 + (size_t)min(c0 + r, D.K - 1) * D.d) + q;
        const int nr = min(4, D.K - c0);
        float acc[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[r][j] = 0.0f;
        const int steps = D.d / 32;
#pragma unroll 8
        for (int i = 0; i < steps; ++i) {
            const uint2 xv = xr[8 * i];
            const float xf[4] = {__uint_as_float(xv.x << 16), __uint_as_float(xv.x & 0xffff0000u),
                                 __uint_as_float(xv.y << 16), __uint_as_float(xv.y & 0xffff0000u)};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (r < nr) {
                    const uint2 wv = wr[r][8 * i];
                    acc[r][0] = fmaf(xf[0], __uint_as_float(wv.x << 16), acc[r][0]);
                    acc[r][1] = fmaf(xf[1], __uint_as_float(wv.x & 0xffff0000u), acc[r][1]);
                    acc[r][2] = fmaf(xf[2], __uint_as_float(wv.y << 16), acc[r][2]);
                    acc[r][3] = fmaf(xf[3], __uint_as_float(wv.y & 0xffff0000u), acc[r][3]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {             // butterfly: chain distance 16, 8, 4 is lane distance 4, 2, 1; 2 and 1 are the lane's own
#pragma unroll
            for (int off = 4; off; off >>= 1)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[r][j] += __shfl_xor_sync(0xffffffffu, acc[r][j], off);
            const float v = (acc[r][0] + acc[r][2]) + (acc[r][1] + acc[r][3]);
            if (c0 + r < D.K && (c0 + r == 0 || v > best)) { best = v; kk = c0 + r; }
        }
    }
    if (q == 0 && a < D.A) {
        R.bit_idx[a] = (int8_t)kk;
        keys[a] = e * D.K + kk;
    }
}

// Grouping of large loads: a stable counting sort over the grid.  Block b owns a contiguous run of assignments and takes it 512
// at a time, one per thread; an assignment's rank among the earlier ones of its key inside the run comes from a match instruction
// (inside its warp) and one array of running counts in shared memory, to which the warps add in order, one after the other.
// Pass 1 leaves the ranks in inv_perm and the run's histogram in hist[b]; pass 2 adds the counts of the earlier runs and of the
// smaller keys.
// (Before: one warp per key walked all assignments, twice: 62 us for 9000 assignments on 192 keys.)
constexpr int GS_THREADS = 512, GS_MAX_RUNS = 64;
__global__ void __launch_bounds__(GS_THREADS)
run_rank_kernel(int A, int n_keys, int run, const int32_t* __restrict__ keys, int32_t* __restrict__ rank, int32_t* __restrict__ hist) {
    pdl_enter();
    extern __shared__ int32_t s_run[];            // [n_keys] counts of the run so far, then one warp's turn at a time
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < n_keys; i += GS_THREADS) s_run[i] = 0;
    __syncthreads();
    const int a0 = blockIdx.x * run, a1 = min(A, a0 + run);
    for (int base = a0; base < a1; base += GS_THREADS) {
        const int a = base + threadIdx.x;
        const int key = a < a1 ? keys[a] : -1 - lane;                  // dead lanes match nobody
        const unsigned same = __match_any_sync(0xffffffffu, key);
        const int mine = __popc(same & ((1u << lane) - 1u));
        // the warps add their counts in order (stable): sixteen short turns per 512 assignments
        int before = 0;
        for (int w = 0; w < GS_THREADS / 32; ++w) {
            if (w == warp) {
                if (a < a1) before = s_run[key];
                __syncwarp();
                if (a < a1 && mine == 0) s_run[key] = before + __popc(same);
            }
            __syncthreads();
        }
        if (a < a1) rank[a] = before + mine;
    }
    for (int i = threadIdx.x; i < n_keys; i += GS_THREADS) hist[(size_t)blockIdx.x * n_keys + i] = s_run[i];
}

__global__ void __launch_bounds__(GS_THREADS)
run_place_kernel(int A, int n_keys, int run, int n_runs, const int32_t* __restrict__ keys, const int32_t* __restrict__ hist,
                 int32_t* __restrict__ group_off, int32_t* __restrict__ perm, int32_t* inv_perm) {
    pdl_enter();
    extern __shared__ int32_t s_place[];          // [n_keys] first position of this run's assignments of a key
    __shared__ int s_warp[GS_THREADS / 32];
    __shared__ int s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int k0 = 0; k0 < n_keys; k0 += GS_THREADS) {
        const int key = k0 + threadIdx.x;
        int total = 0, earlier = 0;
        if (key < n_keys)
            for (int r = 0; r < n_runs; ++r) {
                const int c = hist[(size_t)r * n_keys + key];
                if (r == (int)blockIdx.x) earlier = total;
                total += c;
            }
        int incl = total;                         // block-wide exclusive scan of the keys' totals
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += o;
        }
        if (lane == 31) s_warp[warp] = incl;
        __syncthreads();
        int carry = s_carry;
        for (int w = 0; w < warp; ++w) carry += s_warp[w];
        const int off = carry + incl - total;
        if (key < n_keys) {
            s_place[key] = off + earlier;
            if (blockIdx.x == 0) group_off[key] = off;
        }
        __syncthreads();
        if (threadIdx.x == GS_THREADS - 1) s_carry = carry + incl;
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) group_off[n_keys] = A;
    const int a0 = blockIdx.x * run, a1 = min(A, a0 + run);
    for (int a = a0 + threadIdx.x; a < a1; a += GS_THREADS) {
        const int p = s_place[keys[a]] + inv_perm[a];
        perm[p] = a;
        inv_perm[a] = p;
    }
}

// Small and mid-sized loads: histogram, scan and scatter in one launch.  Every block stages all keys in shared
// memory and counts every key itself (32 warps, a key per warp at a time), so no block waits for another;
// block b then writes the groups of the keys b, b + grid, ...  One block for decode-sized loads, a few
// blocks for a prefill batch of a few thousand assignments on a few dozen keys.  A warp walks the staged keys
// with ballots, which keeps the assignments of a key in order: the same stable order as the other kernels'.
// smem: A keys + n_keys + 1 ints.
__global__ void __launch_bounds__(1024)
group_block_kernel(int A, int n_keys, const int32_t* __restrict__ keys, int32_t* __restrict__ group_off,
                 int32_t* __restrict__ perm, int32_t* __restrict__ inv_perm) {
    pdl_enter();
    extern __shared__ int32_t s_grp[];
    group_block_body(A, n_keys, keys, group_off, perm, inv_perm, s_grp, blockIdx.x, gridDim.x);
}

// One block, counting sort: up to a few thousand assignments on up to 512 keys (see group_block.cuh).
__global__ void __launch_bounds__(1024)
group_sort_kernel(int A, int n_keys, const int32_t* __restrict__ keys, int32_t* __restrict__ group_off,
                  int32_t* __restrict__ perm, int32_t* __restrict__ inv_perm) {
    pdl_enter();
    extern __shared__ int32_t s_grp[];
    group_sort_body(A, n_keys, keys, group_off, perm, inv_perm, s_grp);
}

// Same dot product with both vectors already in shared memory.
__device__ __forceinline__ float dot_pinned_smem(const __nv_bfloat16* a, const __nv_bfloat16* b, int d, int lane) {
    float acc = 0.0f;
#pragma unroll 8
    for (int i = lane; i < d; i += 32)
        acc = fmaf(__bfloat162float(a[i]), __bfloat162float(b[i]), acc);
    for (int off = 16; off; off >>= 1) acc = acc + __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
}

// Copies d elements (a multiple of 8; both ends 16-byte aligned) into shared memory with asynchronous 16-byte copies:
// every copy of a block is in flight at once (one trip to memory instead of one per few registers).  The data may
// be read after stage_wait() and a barrier.
__device__ __forceinline__ void stage_row(__nv_bfloat16* dst, const __nv_bfloat16* __restrict__ src, int d) {
    const uint4* s = reinterpret_cast<const uint4*>(src);
    const uint32_t t = smem_u32(dst);
    for (int i = threadIdx.x; i < d / 8; i += blockDim.x)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(t + 16u * (uint32_t)i), "l"(s + i) : "memory");
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Dot products of one row with NR others, all in shared memory, by 16 lanes: lane p of the half-warp carries the chains 2p and
// 2p + 1 of the pinned order (elements 2p, 2p + 1 of every 32), so an operand is one 4-byte load per 32 elements and the
// row's word is used NR times.  Afterwards the butterfly: chain distance 16, 8, 4, 2 is lane distance 8, 4, 2, 1;
// distance 1 is the lane's own pair.  d a multiple of 32.
template <int NR>
__device__ __forceinline__ void dots_halfwarp(const uint32_t* x, const uint32_t* const (&wr)[NR], int d, float (&out)[NR]) {
    const int p = threadIdx.x & 15;
    float acc[NR][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r][0] = acc[r][1] = 0.0f;
#pragma unroll 8
    for (int i = 0; i < d / 32; ++i) {
        const uint32_t xw = x[16 * i + p];
        const float x0 = __uint_as_float(xw << 16), x1 = __uint_as_float(xw & 0xffff0000u);
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const uint32_t v = wr[r][16 * i + p];
            acc[r][0] = fmaf(x0, __uint_as_float(v << 16), acc[r][0]);
            acc[r][1] = fmaf(x1, __uint_as_float(v & 0xffff0000u), acc[r][1]);
        }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
#pragma unroll
        for (int off = 8; off; off >>= 1) {
            acc[r][0] += __shfl_xor_sync(0xffffffffu, acc[r][0], off);
            acc[r][1] += __shfl_xor_sync(0xffffffffu, acc[r][1], off);
        }
        out[r] = acc[r][0] + acc[r][1];
    }
}

// Gate logits as a tiled product: a block takes 4 XT tokens x 2 WT experts, a half-warp forms XT x WT of them in registers (same
// lane layout and order as above), columns stream through shared memory 256 at a time, STAGES chunks in flight.
//   XT = WT = 4, two stages (nine blocks share an SM).  Bound: fp32 issue (a multiply-add, half a conversion and a quarter of a
// shared load per product).  1500 tokens x 64 experts x 2048: 62 us before (one dot per warp, two 2-byte shared loads per product).
//   XT = WT = 1, eight stages, for a handful of tokens: the other tile would be mostly padding, whose products a half-warp
// would walk through all the same (56 instructions per 32 columns against 8).
constexpr int GATE_COLS = 256;
constexpr int GATE_PITCH = GATE_COLS / 2 + 4;           // words per row: four rows on, the other half of the banks
template <int XT, int WT, int STAGES>
__global__ void __launch_bounds__(128)
gate_logits_kernel(int T, int E, int d, const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ gate_w,
                   float* __restrict__ logits) {
    pdl_enter();
    constexpr int TB = 4 * XT, ROWS = TB + 2 * WT;
    static_assert(XT * WT <= 16, "a lane of the half-warp writes each product");
    __shared__ __align__(16) uint32_t sm[STAGES][ROWS][GATE_PITCH];
    const int hw = threadIdx.x >> 4, p = threadIdx.x & 15;
    const int tb = blockIdx.x * TB, eb = blockIdx.y * (2 * WT);
    const int n_chunks = (d + GATE_COLS - 1) / GATE_COLS;
    auto stage = [&](int c) {
        if (c < n_chunks) {
            const int c0 = c * GATE_COLS, n16 = min(GATE_COLS, d - c0) / 8;
            for (int i = threadIdx.x; i < ROWS * (GATE_COLS / 8); i += 128) {
                const int r = i / (GATE_COLS / 8), k = i % (GATE_COLS / 8);
                if (k >= n16) continue;
                // rows past the end repeat the last one; their results are dropped
                const __nv_bfloat16* src = r < TB ? x + (size_t)min(tb + r, T - 1) * d : gate_w + (size_t)min(eb + r - TB, E - 1) * d;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(&sm[c % STAGES][r][4 * k])), "l"(src + c0 + 8 * k) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll 1
    for (int c = 0; c < STAGES - 1; ++c) stage(c);
    float acc[XT][WT][2];
#pragma unroll
    for (int t = 0; t < XT; ++t)
#pragma unroll
        for (int r = 0; r < WT; ++r) acc[t][r][0] = acc[t][r][1] = 0.0f;
    const int xr = (hw & 3) * XT, wr = TB + (hw >> 2) * WT;
    for (int c = 0; c < n_chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncthreads();                          // chunk c is there; the stage refilled next has been read
        stage(c + STAGES - 1);
        const uint32_t (*b)[GATE_PITCH] = sm[c % STAGES];
        const int steps = min(GATE_COLS, d - c * GATE_COLS) / 32;
#pragma unroll 4
        for (int i = 0; i < steps; ++i) {
            float xv[XT][2], wv[WT][2];
#pragma unroll
            for (int t = 0; t < XT; ++t) {
                const uint32_t v = b[xr + t][16 * i + p];
                xv[t][0] = __uint_as_float(v << 16); xv[t][1] = __uint_as_float(v & 0xffff0000u);
            }
#pragma unroll
            for (int r = 0; r < WT; ++r) {
                const uint32_t u = b[wr + r][16 * i + p];
                wv[r][0] = __uint_as_float(u << 16); wv[r][1] = __uint_as_float(u & 0xffff0000u);
            }
#pragma unroll
            for (int t = 0; t < XT; ++t)
#pragma unroll
                for (int r = 0; r < WT; ++r) {
                    acc[t][r][0] = fmaf(xv[t][0], wv[r][0], acc[t][r][0]);
                    acc[t][r][1] = fmaf(xv[t][1], wv[r][1], acc[t][r][1]);
                }
        }
    }
#pragma unroll
    for (int t = 0; t < XT; ++t)
#pragma unroll
        for (int r = 0; r < WT; ++r) {
#pragma unroll
            for (int off = 8; off; off >>= 1) {
                acc[t][r][0] += __shfl_xor_sync(0xffffffffu, acc[t][r][0], off);
                acc[t][r][1] += __shfl_xor_sync(0xffffffffu, acc[t][r][1], off);
            }
            const int tt = tb + xr + t, ee = eb + wr - TB + r;
            if (p == WT * t + r && tt < T && ee < E) logits[(size_t)tt * E + ee] = acc[t][r][0] + acc[t][r][1];
        }
}

// One block (8 warps) per token: the same results as route_kernel, with the token row and batches of
// EB weight rows staged in shared memory by 16-byte loads (the pinned summation order makes a lane
// walk a row with stride 32, which is slow straight from global memory); warp w takes row w of a batch.
// WIDTHS: supplied by the caller (a kernel of its own: the code for choosing them costs such a call 1 us of instruction fetch), chosen
// from the width rows of all selected experts staged at once, or from batches of EB rows (apart from the former, whose 64
// registers leave four blocks on an SM, this one's 48 five) or by the kernel behind it.
enum { WIDTHS_SUPPLIED, WIDTHS_AT_ONCE, WIDTHS_BATCHED };
template <int WIDTHS>
__global__ void __launch_bounds__(256, WIDTHS == WIDTHS_AT_ONCE ? 4 : 5)
route_block_kernel(MoeDims D, const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ gate_w,
                   const float* __restrict__ logits_in, const __nv_bfloat16* __restrict__ bit_w,
                   const int8_t* __restrict__ forced, RouteBufs R, int32_t* __restrict__ keys,
                   int32_t* __restrict__ device_status, int EB, int xs_elems, int ws_elems, int slot_pitch) {
    pdl_enter();
    extern __shared__ __align__(16) uint8_t rsm[];
    // EB == 0: nothing is staged (logits and widths supplied); xs_elems, ws_elems: elements of the token row's place and of the staging
    // area behind it
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(rsm);
    __nv_bfloat16* ws = xs + xs_elems;
    float* lg_s = reinterpret_cast<float*>(ws + ws_elems);               // [E]
    float* u_s = lg_s + D.E;                                             // [k * K]
    int* sel_s = reinterpret_cast<int*>(u_s + MAX_TOPK * 8);             // [k]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x;
    const int E = D.E;

    if (EB) stage_row(xs, x + (size_t)t * D.d, D.d);
    if (logits_in) {
        for (int e = threadIdx.x; e < E; e += blockDim.x) lg_s[e] = logits_in[(size_t)t * E + e];
        stage_wait();
        __syncthreads();
    } else {
        for (int eb = 0; eb < E; eb += EB) {
            const int n = min(EB, E - eb);
            stage_row(ws, gate_w + (size_t)eb * D.d, n * D.d);       // the n rows are contiguous: one copy loop
            stage_wait();
            __syncthreads();
            for (int r = warp; r < n; r += 8) {
                const float v = dot_pinned_smem(xs, ws + (size_t)r * D.d, D.d, lane);
                if (lane == 0) lg_s[eb + r] = v;
            }
            __syncthreads();
        }
    }

    float w[MAX_TOPK];
    float wsum = 0.0f;
    int sel[MAX_TOPK];
    if (warp == 0) {
        float lg[MAX_E_PER_LANE];
#pragma unroll
        for (int m = 0; m < MAX_E_PER_LANE; ++m) {
            const int e = lane + 32 * m;
            lg[m] = e < E ? lg_s[e] : -INFINITY;
        }
        gate_select(lg, E, D.k, lane, sel, w, wsum, device_status);
        if (lane == 0) {
#pragma unroll
            for (int s = 0; s < MAX_TOPK; ++s)
                if (s < D.k) sel_s[s] = sel[s];
        }
    }
    __syncthreads();

    const bool later = WIDTHS == WIDTHS_BATCHED && slot_pitch < 0;     // the widths are chosen by the next kernel
    if constexpr (WIDTHS == WIDTHS_AT_ONCE) {   // the width rows of all selected experts at once, a half-warp per slot, four widths at a time
        for (int s = 0; s < D.k; ++s)         // (odd slots half a bank row on: the two half-warps of a warp meet no conflict)
            stage_row(ws + (size_t)s * slot_pitch, bit_w + (size_t)sel_s[s] * D.K * D.d, D.K * D.d);
        stage_wait();
        __syncthreads();
        if (D.k * D.K <= (int)(blockDim.x >> 4)) {                             // few rows: a half-warp each (shortest chain)
            const int row = min((int)(threadIdx.x >> 4), D.k * D.K - 1), s = row / D.K, c = row - s * D.K;
            const uint32_t* wr[1] = {reinterpret_cast<const uint32_t*>(ws + (size_t)s * slot_pitch + (size_t)c * D.d)};
            float v[1];
            dots_halfwarp<1>(reinterpret_cast<const uint32_t*>(xs), wr, D.d, v);
            if ((threadIdx.x & 15) == 0 && (int)(threadIdx.x >> 4) < D.k * D.K) u_s[row] = v[0];
        } else
        for (int sb = 0; sb < D.k; sb += (int)(blockDim.x >> 4)) {
            const int s = min(sb + (int)(threadIdx.x >> 4), D.k - 1);
            if (sb + (int)(threadIdx.x >> 5) * 2 >= D.k) break;               // nothing for this warp
            for (int c0 = 0; c0 < D.K; c0 += 4) {
                const uint32_t* wr[4];
#pragma unroll
                for (int r = 0; r < 4; ++r)       // past the end: the last row again, result dropped
                    wr[r] = reinterpret_cast<const uint32_t*>(ws + (size_t)s * slot_pitch + (size_t)min(c0 + r, D.K - 1) * D.d);
                float v[4];
                dots_halfwarp<4>(reinterpret_cast<const uint32_t*>(xs), wr, D.d, v);
                const int p = threadIdx.x & 15;
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (p == r && c0 + r < D.K) u_s[s * D.K + c0 + r] = v[r];
            }
        }
        __syncthreads();
    } else if (WIDTHS == WIDTHS_BATCHED && !later) {   // bit-width router logits of the selected experts: rows (slot s, width c)
        const int n_rows = D.k * D.K;
        for (int rb = 0; rb < n_rows; rb += EB) {
            const int n = min(EB, n_rows - rb);
            for (int r = 0; r < n; ++r) {
                const int s = (rb + r) / D.K, c = (rb + r) - s * D.K;
                stage_row(ws + (size_t)r * D.d, bit_w + ((size_t)sel_s[s] * D.K + c) * D.d, D.d);
            }
            stage_wait();
            __syncthreads();
            for (int r = warp; r < n; r += 8) {
                const float v = dot_pinned_smem(xs, ws + (size_t)r * D.d, D.d, lane);
                if (lane == 0) u_s[rb + r] = v;
            }
            __syncthreads();
        }
    }

    if (warp == 0 && lane == 0) {
#pragma unroll
        for (int s = 0; s < MAX_TOPK; ++s) {
            if (s < D.k) {
                const int a = t * D.k + s;
                int kk = 0;
                if (WIDTHS == WIDTHS_SUPPLIED) {
                    kk = forced[a];
                    if (kk < 0 || kk >= D.K) {
                        if (device_status) atomicOr(device_status, D2MOE_DEV_BAD_INDEX);
                        kk = kk < 0 ? 0 : D.K - 1;
                    }
                } else if (!later) {
                    float best = u_s[s * D.K];
                    for (int c = 1; c < D.K; ++c)
                        if (u_s[s * D.K + c] > best) { best = u_s[s * D.K + c]; kk = c; }
                }
                R.topk_idx[a] = sel[s];
                R.topk_w[a] = D.renormalize ? w[s] / wsum : w[s];
                if (later) continue;
                R.bit_idx[a] = (int8_t)kk;
                keys[a] = sel[s] * D.K + kk;
            }
        }
    }
}

}  // namespace

cudaError_t launch_route(const MoeDims& D, const __nv_bfloat16* x, const __nv_bfloat16* gate_w,
                         const float* logits_in, const __nv_bfloat16* bit_w, const int8_t* forced,
                         const RouteBufs& R, float* logits_ws, int32_t* keys_ws, int32_t* hist_ws, int hist_ints,
                         int32_t* device_status, cudaStream_t st, bool* defer_small_group) {
    const int warps_per_block = 4;
    const int n_keys = D.E * D.K;
    // block-per-token kernel when the token row plus at least one weight row fit in shared memory
    const size_t row_bytes = (size_t)D.d * 2;
    const size_t tail_bytes = (size_t)(D.E + MAX_TOPK * 8 + MAX_TOPK) * 4 + 64;
    const size_t budget = 200 * 1024;
    int EB = row_bytes + tail_bytes < budget ? (int)((budget - row_bytes - tail_bytes) / row_bytes) : 0;
    if (EB > 8) EB = 8;
    if (EB >= 1 && D.d % 8 == 0) {
        if (!logits_in && logits_ws && d2moe_gate_is_tiled(D.d, D.E, D.T, forced != nullptr)) {
            const bool few = D.T <= 8;
            dim3 grid(few ? (D.T + 3) / 4 : (D.T + 15) / 16, few ? (D.E + 1) / 2 : (D.E + 7) / 8);
            launch_chained(few ? gate_logits_kernel<1, 1, 8> : gate_logits_kernel<4, 4, 2>, dim3(grid), dim3(128), 0, st, D.T, D.E, D.d, x, gate_w, logits_ws);
            logits_in = logits_ws;
            gate_w = nullptr;
        }
        // staging area: EB gate rows (or width rows, batch by batch), or the width rows of all selected experts
        if (logits_in && forced) EB = 0;
        const size_t slots_bytes = (size_t)D.k * ((size_t)D.K * row_bytes + 64);
        const bool fits = slots_bytes + row_bytes + tail_bytes <= 110 * 1024;                  // half of what an SM has
        // Many pairs of token and expert with the logits at hand: one warp per token selects, the widths are chosen by a kernel of
        // their own.  Its chain of d / 32 loads takes 29 us at d = 4096 whatever the number of pairs, which the staged
        // forms reach at 3000 pairs (8 experts x 4096, top-2: 1024 tokens 29 staged, 36 so; 2048 tokens 47, 39), 2300 where the rows
        // are staged batch by batch (17 experts x 8192, 6 widths).
        const bool later = logits_in && !forced && D.A >= (fits ? 2560 : 2048);
        if (later) EB = 0;
        int slot_pitch = later ? -1 : 0;
        if (!forced && !later && fits) {
            // All width rows at once need one trip to memory, batches of EB several; but they may leave fewer blocks on an SM.
            const int rows = D.k * D.K, sms = device_sm_count();
            auto resident = [&](size_t area) { const long long n = 228 * 1024 / (long long)(row_bytes + area + tail_bytes + 1024); return (int)(n < 8 ? n : 8); };
            const int all = resident(!logits_in && slots_bytes < EB * row_bytes ? EB * row_bytes : slots_bytes), batched = resident(EB * row_bytes);
            // 4 rows and fewer behind the gate's rows: the batch is one as well, and a warp per row is faster than half a one
            // (dense layer of 4096, 2048 tokens: 44 against 49 us).  More rows than a batch: all at once while the tokens are one wave of
            // blocks, beyond that if the trips saved outweigh the blocks lost (64 experts x 2048, top-6, 3 widths: 256 tokens 19
            // against 23, 768 tokens 39 against 37; 16 x 1024, top-4, 4 widths: 768 tokens 19 against 30).
            const bool at_once = rows <= EB ? logits_in || rows > 4
                                            : D.T <= (long long)sms * all || (rows + EB - 1) / EB * all > batched;
            if (at_once) slot_pitch = D.K * D.d + 32;
        }
        size_t ws_elems = !EB ? 0 : slot_pitch > 0 ? (size_t)D.k * slot_pitch : (size_t)EB * D.d;
        if (EB && !logits_in && ws_elems < (size_t)EB * D.d) ws_elems = (size_t)EB * D.d;
        const size_t smem = (EB ? row_bytes : 0) + 2 * ws_elems + tail_bytes;
        // logits and widths both supplied: no dot products, one warp per token does the selection
        const int threads = !EB ? 32 : (logits_in && slot_pitch > 0) ? 128 : 256;
        auto launch = [&](auto widths) -> cudaError_t {
            constexpr auto kern = &route_block_kernel<decltype(widths)::value>;
            cudaError_t e = ensure_dynamic_smem<kern>((int)smem);
            if (e != cudaSuccess) return e;
            launch_chained(kern, dim3(D.T), dim3(threads), smem, st, D, x, gate_w, logits_in, bit_w, forced, R, keys_ws, device_status, EB,
                           EB ? D.d : 0, (int)ws_elems, slot_pitch);
            return cudaSuccess;
        };
        const cudaError_t e = forced ? launch(std::integral_constant<int, WIDTHS_SUPPLIED>{})
                            : slot_pitch > 0 ? launch(std::integral_constant<int, WIDTHS_AT_ONCE>{}) : launch(std::integral_constant<int, WIDTHS_BATCHED>{});
        if (e != cudaSuccess) return e;
        if (later) launch_chained(width_router_kernel, dim3((D.A + 15) / 16), dim3(128), 0, st, D, x, bit_w, R, keys_ws);
    } else
    launch_chained(route_kernel, dim3((D.T + warps_per_block - 1) / warps_per_block), dim3(warps_per_block * 32), 0, st, 
        D, x, gate_w, logits_in, bit_w, forced, R, keys_ws, device_status);
    // few assignments and keys: histogram, scan and scatter in one single-block launch
    const bool small = d2moe_group_is_small(D.A, n_keys);
    // the caller runs the single-block grouping in front of its next kernel (one launch instead of two)
    if ((small || d2moe_group_is_sortable(D.A, n_keys)) && defer_small_group) { *defer_small_group = true; return cudaGetLastError(); }
    if (!small && d2moe_group_is_sortable(D.A, n_keys)) {
        const int threads = D.A >= 2048 ? 1024 : 512;
        const size_t gsm = group_sort_smem_ints(D.A, n_keys, threads / 32) * 4;
        cudaError_t e = ensure_dynamic_smem<&group_sort_kernel>((int)gsm);
        if (e != cudaSuccess) return e;
        launch_chained(group_sort_kernel, dim3(1), dim3(threads), gsm, st, D.A, n_keys, keys_ws, R.group_off, R.perm, R.inv_perm);
        return cudaGetLastError();
    }
    if (small || d2moe_group_is_mid(D.A, n_keys)) {
        const size_t gsm = (size_t)(((D.A + 31) & ~31) + n_keys + 1) * 4;
        cudaError_t e = ensure_dynamic_smem<&group_block_kernel>((int)gsm);
        if (e != cudaSuccess) return e;
        const int blocks = small ? 1 : (n_keys < 16 ? n_keys : 16);
        launch_chained(group_block_kernel, dim3(blocks), dim3(1024), gsm, st, D.A, n_keys, keys_ws, R.group_off, R.perm, R.inv_perm);
        return cudaGetLastError();
    }
    // runs of at least 512 assignments, as many as the histogram space holds
    long long n_runs = hist_ints / n_keys < GS_MAX_RUNS ? hist_ints / n_keys : GS_MAX_RUNS;
    if (n_runs > (D.A + GS_THREADS - 1) / GS_THREADS) n_runs = (D.A + GS_THREADS - 1) / GS_THREADS;
    const int run = (int)(((D.A + n_runs - 1) / n_runs + GS_THREADS - 1) / GS_THREADS * GS_THREADS);
    n_runs = (D.A + run - 1) / run;
    launch_chained(run_rank_kernel, dim3((unsigned)n_runs), dim3(GS_THREADS), (size_t)n_keys * 4, st, D.A, n_keys, run, keys_ws, R.inv_perm, hist_ws);
    launch_chained(run_place_kernel, dim3((unsigned)n_runs), dim3(GS_THREADS), (size_t)n_keys * 4, st, D.A, n_keys, run, (int)n_runs, keys_ws, hist_ws,
                   R.group_off, R.perm, R.inv_perm);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// d2moe_route_static_scratch: the routing call for callers that cannot hand over a workspace.
//
// Its scratch (the per-assignment sort keys and the (expert, width) histogram that d2moe_route keeps
// in the caller's workspace) lives in one file-scope device array, so the call needs no allocation
// of any kind.  The array is part of the library image: every GPU that loads the library holds these
// bytes until the process exits.
// ------------------------------------------------------------------------------------------------
#include <mutex>

#define D2MOE_STATIC_SCRATCH_BYTES ((D2MOE_STATIC_MAX_ASSIGNMENTS + D2MOE_STATIC_MAX_KEYS) * 4)

static __device__ __align__(256) unsigned char g_route_scratch[D2MOE_STATIC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_addr[kMaxDevices] = {};   // device address of g_route_scratch, per device ordinal
}  // namespace

extern "C" d2moe_status d2moe_route_static_scratch(const d2moe_config* c, int64_t T, const void* x,
                                                   const void* gate_w, const float* logits, const void* bit_w,
                                                   const int8_t* forced, int32_t* topk_idx, float* topk_w,
                                                   int8_t* bit_idx, int32_t* perm, int32_t* inv_perm,
                                                   int32_t* group_off, int32_t* device_status, void* stream) {
    d2moe_status s = d2moe_check_config(c);
    if (s != D2MOE_OK) return s;
    if (T < 0) return D2MOE_ERR_SHAPE;
    // the fixed scratch bounds the problem: say so instead of overrunning it
    if (T * c->top_k > D2MOE_STATIC_MAX_ASSIGNMENTS || c->n_experts * c->n_bits > D2MOE_STATIC_MAX_KEYS)
        return D2MOE_ERR_WORKSPACE;
    if (!topk_idx || !topk_w || !bit_idx || !perm || !inv_perm || !group_off) return D2MOE_ERR_NULL;
    if (T > 0 && !x) return D2MOE_ERR_NULL;
    if ((gate_w == nullptr) == (logits == nullptr)) return D2MOE_ERR_NULL;
    if ((bit_w == nullptr) == (forced == nullptr)) return D2MOE_ERR_NULL;

    // In host code `g_route_scratch` is only a handle for the symbol, not an address a kernel can
    // use.  The device address is looked up once per device, with that device current, and kept.
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return D2MOE_ERR_CUDA;
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_scratch_mutex);
        if (!g_scratch_addr[dev]) {
            void* addr = nullptr;
            if (cudaGetSymbolAddress(&addr, g_route_scratch) != cudaSuccess || !addr) return D2MOE_ERR_CUDA;
            g_scratch_addr[dev] = addr;
        }
        scratch = g_scratch_addr[dev];
    }

    cudaStream_t st = (cudaStream_t)stream;
    const int n_keys = c->n_experts * c->n_bits;
    if (T == 0) {
        cudaError_t e = cudaMemsetAsync(group_off, 0, (size_t)(n_keys + 1) * 4, st);
        return e == cudaSuccess ? D2MOE_OK : D2MOE_ERR_CUDA;
    }
    MoeDims D;
    D.T = (int)T; D.d = c->d_model; D.F = c->d_ffn; D.E = c->n_experts; D.k = c->top_k;
    D.n_shared = c->n_shared; D.g = c->group_size; D.K = c->n_bits;
    for (int i = 0; i < 8; ++i) D.bits[i] = i < c->n_bits ? c->bits[i] : 0;
    D.A = (int)(T * c->top_k);
    D.A_tot = D.A + (int)(T * c->n_shared);
    D.renormalize = c->renormalize;
    // Nothing in the scratch has to start at zero: the key of every assignment and the count of every
    // (expert, width) pair are written before they are read, so the previous call's contents are inert.
    int32_t* keys = reinterpret_cast<int32_t*>(scratch);
    int32_t* hist = keys + D2MOE_STATIC_MAX_ASSIGNMENTS;
    RouteBufs R{topk_idx, topk_w, bit_idx, perm, inv_perm, group_off};
    launch_chain_begin();
    cudaError_t e = launch_route(D, (const __nv_bfloat16*)x, (const __nv_bfloat16*)gate_w, logits,
                                 (const __nv_bfloat16*)bit_w, forced, R, nullptr, keys, hist, D2MOE_STATIC_MAX_KEYS, device_status, st);
    return e == cudaSuccess ? D2MOE_OK : D2MOE_ERR_CUDA;
}
