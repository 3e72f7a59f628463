// MWQ quantization + packing (Section 3.3.1, Eq. 2, Eq. 4, Eq. 5, Algorithm 1) and the unpack test hooks.
//
// All fp32 operations follow the definition's order with one IEEE rounding per operation and no contraction, so that
// codes, scales and offsets are reproducible bit for bit.
#include "d2moe_common.cuh"
#include "tc_common.cuh"

namespace {

constexpr int PACK_THREADS = 256;

__global__ void pack_header_kernel(PackHeader* h, PackLayout L, int n_bits,
                                   int b0, int b1, int b2, int b3, int b4, int b5, int b6, int b7) {
    uint32_t* words = reinterpret_cast<uint32_t*>(h);
    for (int i = threadIdx.x; i < D2MOE_HEADER_BYTES / 4; i += blockDim.x) words[i] = 0u;   // the maxima start at zero
    __syncwarp();
    if (threadIdx.x == 0) {
        h->magic = D2MOE_MAGIC; h->version = D2MOE_LAYOUT_VERSION;
        h->rows = L.rows; h->cols = L.cols; h->g = L.g; h->n_bits = n_bits;
        int b[8] = {b0, b1, b2, b3, b4, b5, b6, b7};
        for (int i = 0; i < 8; ++i) h->bits[i] = b[i];
        h->scale_mode = L.scale_mode;
    }
}

// ---- pieces shared by the packing kernels ------------------------------------------------------

// float <-> int with the same order (a zero below its positive twin), so that a group's extremes take one integer
// warp reduction each
__device__ __forceinline__ int ordered(float f) { const int i = __float_as_int(f); return i ^ ((i >> 31) & 0x7fffffff); }
__device__ __forceinline__ float unordered(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// Eq. 2: base scale (rounded up) and offset (rounded down) of a group from its extremes
__device__ __forceinline__ __half2 group_meta(float wmin, float wmax, float levels) {
    const __half lo_h = __float2half_rd(wmin);
    __half s1_h = __float2half_ru(__fdiv_rn(__fsub_rn(wmax, __half2float(lo_h)), levels));
    if (__half2float(s1_h) == 0.0f) s1_h = __float2half_rn(6.103515625e-05f);      // 2^-14
    return __halves2half2(s1_h, lo_h);                                            // low half = s1, high half = lo
}

// rint of the correctly rounded quotient t / s1, clamped to the base code: the product with the reciprocal is within
// 1e-4 of the quotient (quotients reach 255, the two roundings are 2^-23 each), so only a value that close to a
// half needs the division itself
__device__ __forceinline__ float base_code(float t, float s1, float inv, float levels) {
    const float a = t * inv;
    float q = rintf(a);
    if (fabsf(a - q) > 0.4998f) q = rintf(__fdiv_rn(t, s1));
    return fminf(fmaxf(q, 0.0f), levels);
}

// Two fp32 operations in one instruction (each lane rounds on its own, exactly as the scalar form)
__device__ __forceinline__ unsigned long long pair(float a, float b) {
    return ((unsigned long long)__float_as_uint(b) << 32) | __float_as_uint(a);
}
__device__ __forceinline__ float first(unsigned long long v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float second(unsigned long long v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// one residual step of Eq. 4 for one element: adds +-sj by the sign of the residual (a zero counts as positive: `w` is
// never -0, so an exact residual is +0) and shifts the residual's sign bit into the code (complemented by the caller)
__device__ __forceinline__ void residual_step(float w, float sj, float& wh, float& rs, uint32_t& code) {
    code = __funnelshift_l(__float_as_uint(rs), code, 1);
    wh = __fadd_rn(wh, __uint_as_float(__float_as_uint(sj) | (__float_as_uint(rs) & 0x80000000u)));
    rs = __fsub_rn(w, wh);
}

// Stored words of eight consecutive operand cells (32 codes, `cell[i]`: four top-width codes in the cell's byte order)
// of row r of a packed block, into `blk` (the block's image).  q: which eight cells of the row.
template <int GS>
__device__ __forceinline__ void store_fields(const PackLayout& L, uint8_t* blk, int r, int q, const uint32_t (&cell)[8]) {
#pragma unroll 1
    for (int j = 0; j < L.n_seg; ++j) {
        const int sh = L.seg_shift[j];
        uint8_t* seg = blk + L.seg_off[j];
        // cell c's field to bit `to` of its bytes: one rotation, then the field is merged under a constant mask
        auto at = [&](int c, int to) { return __funnelshift_l(cell[c], cell[c], (to - sh) & 31); };
        if (L.seg_sw[j] == 4) {
            uint32_t v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = (at(2 * i, 0) & 0x0F0F0F0Fu) | (at(2 * i + 1, 4) & 0xF0F0F0F0u);
            *reinterpret_cast<uint4*>(seg + (q * D2MOE_TILE_ROWS + r) * 16) = make_uint4(v[0], v[1], v[2], v[3]);
        } else if (L.seg_sw[j] == 2) {
            uint32_t v[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                v[i] = at(4 * i, 0) & 0x03030303u;
#pragma unroll
                for (int u = 1; u < 4; ++u) v[i] |= at(4 * i + u, 2 * u) & (0x03030303u << (2 * u));
            }
            constexpr int CS = GS / 4 < 16 ? GS / 4 : 16;
            const int ob = 8 * q;
            *reinterpret_cast<uint2*>(seg + ((ob / CS) * D2MOE_TILE_ROWS + r) * CS + ob % CS) = make_uint2(v[0], v[1]);
        } else if (L.seg_sw[j] == 1) {
            uint32_t v = at(0, 0) & 0x01010101u;
#pragma unroll
            for (int i = 1; i < 8; ++i) v |= at(i, i) & (0x01010101u << i);
            constexpr int CS = GS / 8 < 16 ? GS / 8 : 16;
            const int ob = 4 * q;
            *reinterpret_cast<uint32_t*>(seg + ((ob / CS) * D2MOE_TILE_ROWS + r) * CS + ob % CS) = v;
        } else {
            *reinterpret_cast<uint4*>(seg + (2 * q * D2MOE_TILE_ROWS + r) * 16) = make_uint4(cell[0], cell[1], cell[2], cell[3]);
            *reinterpret_cast<uint4*>(seg + ((2 * q + 1) * D2MOE_TILE_ROWS + r) * 16) = make_uint4(cell[4], cell[5], cell[6], cell[7]);
        }
    }
}

// the matrix's largest scale and largest |W|, kept in the header: a block writes only what exceeds the value it sees
// (the maxima only grow, so a stale value costs an atomic, never a result)
__device__ __forceinline__ void raise_maxima(uint8_t* packed, unsigned s1_bits, unsigned wabs_bits) {
    PackHeader* h = reinterpret_cast<PackHeader*>(packed);
    if (s1_bits > *(volatile uint32_t*)&h->s1_max_bits) atomicMax(&h->s1_max_bits, s1_bits);
    if (wabs_bits > *(volatile uint32_t*)&h->wabs_max_bits) atomicMax(&h->wabs_max_bits, wabs_bits);
}

// byte of element k inside its operand cell: order 0, 2, 1, 3
__device__ __forceinline__ int cell_byte(int k) { return ((k & 1) << 1) | ((k >> 1) & 1); }

__host__ __device__ constexpr int pack_cell_stride(int gs) { return gs + 16; }      // bytes per row of the cell buffer (16: no bank conflicts)

// Last phase of a packing block: the codes of its 64 rows (cell buffer) become the stored fields of the block's image in
// shared memory, which leaves as one run of 16-byte stores; the block's extremes go to the header.
template <int GS>
__device__ __forceinline__ void pack_finish(const PackLayout& L, uint8_t* packed, uint8_t* blk, const uint8_t* cells, uint8_t* image,
                                            unsigned s1_max, unsigned wabs_max) {
    __shared__ unsigned s_max[2];
    constexpr int NQ = GS / 32;                            // runs of eight cells per row
    if (threadIdx.x < 2) s_max[threadIdx.x] = 0u;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && s1_max) { atomicMax(&s_max[0], s1_max); atomicMax(&s_max[1], wabs_max); }
    for (int i = threadIdx.x; i < D2MOE_TILE_ROWS * NQ; i += PACK_THREADS) {
        const int r = i & (D2MOE_TILE_ROWS - 1), q = i / D2MOE_TILE_ROWS;
        const uint4* src = reinterpret_cast<const uint4*>(cells + r * pack_cell_stride(GS) + 32 * q);
        const uint4 a = src[0], b = src[1];
        const uint32_t cell[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        store_fields<GS>(L, image, r, q, cell);
    }
    __syncthreads();
    const uint4* src = reinterpret_cast<const uint4*>(image);
    uint4* dst = reinterpret_cast<uint4*>(blk);
    for (int i = threadIdx.x; i < L.block_bytes / 16; i += PACK_THREADS) dst[i] = src[i];
    if (threadIdx.x == 0) raise_maxima(packed, s_max[0], s_max[1]);
}

// Tied scales.  One block per packed block (64 rows x one group); a lane owns whole operand cells (four consecutive
// elements: one 16-byte load, one cell word), LPR lanes per row; the loads of PB passes are in flight at once and the
// scales of their rows are formed together, one row per lane.
//   Residual steps: with s_j = s1 / 2^(j+1) the sum of the +-s_j is exact in fp32 (11 + 7 bits), so the code's low bits are
// read off that sum at the end instead of being shifted in, and a step is one logic instruction and three packed fp32
// additions per two weights.  q s1 is exact too (8 + 11 bits), so lo + q s1 is one fused operation.  The base code needs
// no clamp: lo is rounded down and s1 up, so a quotient lies in [0, levels + 2^-15].
// Bound: instruction issue (75 % of the slots, DRAM 25 %).  14336 x 4096, {2,3,4,8}: 0.626 -> 0.134 ms.
template <int GS>
__global__ void __launch_bounds__(PACK_THREADS)
pack_tied_kernel(PackLayout L, const float* __restrict__ W, uint8_t* __restrict__ packed) {
    constexpr int LPR = GS / 4 < 32 ? GS / 4 : 32;         // lanes per row
    constexpr int V = GS / (4 * LPR);                      // cells per lane
    constexpr int RPW = 32 / LPR;                          // rows a warp takes per pass
    constexpr int PASSES = D2MOE_TILE_ROWS / (8 * RPW);
    constexpr int PB = PASSES < 4 ? PASSES : (V == 1 ? 4 : 2);
    extern __shared__ __align__(16) uint8_t smem[];
    uint8_t* cells = smem;
    uint8_t* image = smem + D2MOE_TILE_ROWS * pack_cell_stride(GS);
    const int G = blockIdx.x, rt = blockIdx.y;
    uint8_t* blk = packed + d2moe_block_offset(L, rt, G);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / LPR, l = lane % LPR;
    const float levels = (float)((1 << L.b1) - 1);
    const int n_lv = L.top - L.b1;
    const bool aligned = (reinterpret_cast<uintptr_t>(W) & 15) == 0;
    const float two_nl = (float)(1 << n_lv);
    const unsigned long long magic = pair(12582912.0f, 12582912.0f), minus_magic = pair(-12582912.0f, -12582912.0f);
    const unsigned long long zero2 = pair(0.0f, 0.0f), minus_one = pair(-1.0f, -1.0f);
    const unsigned long long nl2 = pair(two_nl, two_nl), half2_ = pair(0.5f * (two_nl - 1.0f), 0.5f * (two_nl - 1.0f));
    unsigned s1_max = 0, wabs_max = 0;

#pragma unroll 1
    for (int p0 = 0; p0 < PASSES; p0 += PB) {
        float w[PB][V][4];
        int mn[PB], mx[PB];
#pragma unroll
        for (int b = 0; b < PB; ++b) {
            const long long row = (long long)rt * D2MOE_TILE_ROWS + ((p0 + b) * 8 + warp) * RPW + sub;
            const float* src = W + row * (long long)L.cols + (long long)G * GS;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (row < L.rows) {
                    const int k = 4 * (l + LPR * v);
                    if (aligned) f = *reinterpret_cast<const float4*>(src + k);
                    else f = make_float4(src[k], src[k + 1], src[k + 2], src[k + 3]);
                }
                w[b][v][0] = f.x; w[b][v][1] = f.y; w[b][v][2] = f.z; w[b][v][3] = f.w;
            }
        }
#pragma unroll
        for (int b = 0; b < PB; ++b) {
            float fmn = w[b][0][0], fmx = fmn;
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int i = 0; i < 4; ++i) { fmn = fminf(fmn, w[b][v][i]); fmx = fmaxf(fmx, w[b][v][i]); }
            mn[b] = ordered(fmn); mx[b] = ordered(fmx);
            if constexpr (LPR == 32) {
                mn[b] = __reduce_min_sync(0xffffffffu, mn[b]);
                mx[b] = __reduce_max_sync(0xffffffffu, mx[b]);
            } else {
#pragma unroll
                for (int off = LPR / 2; off; off >>= 1) {
                    mn[b] = min(mn[b], __shfl_xor_sync(0xffffffffu, mn[b], off));
                    mx[b] = max(mx[b], __shfl_xor_sync(0xffffffffu, mx[b], off));
                }
            }
        }
        // lane (sub, l) forms the scale and offset of its row in pass l % PB
        int my_mn = mn[0], my_mx = mx[0];
#pragma unroll
        for (int b = 1; b < PB; ++b)
            if (l % PB == b) { my_mn = mn[b]; my_mx = mx[b]; }
        const float wmin = unordered(my_mn), wmax = unordered(my_mx);
        const __half2 my_meta = group_meta(wmin, wmax, levels);
        const float my_inv = __frcp_rn(__low2float(my_meta));
        const int my_r = ((p0 + l % PB) * 8 + warp) * RPW + sub;
        const bool my_live = (long long)rt * D2MOE_TILE_ROWS + my_r < L.rows;            // padding rows: zero codes, zero meta
        if (l < PB) {
            reinterpret_cast<uint32_t*>(image)[my_r] = my_live ? as_u32(my_meta) : 0u;
            if (my_live) {
                s1_max = max(s1_max, __float_as_uint(__low2float(my_meta)));
                wabs_max = max(wabs_max, __float_as_uint(fmaxf(fabsf(wmin), fabsf(wmax))));
            }
        }
        // two rows at a time
#pragma unroll
        for (int b0 = 0; b0 < PB; b0 += 2) {
            unsigned long long wc[2][V][2], q[2][V][2], wh[2][V][2], rs[2][V][2], sum[2][V][2];
            float sj[2], inv[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const __half2 meta = as_h2(__shfl_sync(0xffffffffu, as_u32(my_meta), sub * LPR + b0 + h));
                inv[h] = __shfl_sync(0xffffffffu, my_inv, sub * LPR + b0 + h);
                const float s1 = __low2float(meta), lo = __high2float(meta);
                const unsigned long long s1_2 = pair(s1, s1), lo_2 = pair(lo, lo), mlo_2 = pair(-lo, -lo), inv_2 = pair(inv[h], inv[h]);
#pragma unroll
                for (int v = 0; v < V; ++v)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        wc[h][v][i] = add2(pair(w[b0 + h][v][2 * i], w[b0 + h][v][2 * i + 1]), zero2);   // -0 becomes +0: see residual_step
                        const unsigned long long t = add2(wc[h][v][i], mlo_2), a = mul2(t, inv_2);
                        q[h][v][i] = add2(add2(a, magic), minus_magic);                                  // rint
                        const unsigned long long d = fma2(q[h][v][i], minus_one, a);
                        if (fmaxf(fabsf(first(d)), fabsf(second(d))) > 0.4998f)                           // close to a half: the quotient itself decides
                            q[h][v][i] = pair(rintf(__fdiv_rn(first(t), s1)), rintf(__fdiv_rn(second(t), s1)));
                        wh[h][v][i] = fma2(q[h][v][i], s1_2, lo_2);
                        rs[h][v][i] = fma2(wh[h][v][i], minus_one, wc[h][v][i]);
                        sum[h][v][i] = zero2;
                    }
                sj[h] = __fmul_rn(s1, 0.25f);                                    // s_1 = s1 * 2^-2
            }
#pragma unroll 1
            for (int j = 0; j < n_lv; ++j) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t sb = __float_as_uint(sj[h]);
#pragma unroll
                    for (int v = 0; v < V; ++v)
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const unsigned long long st = pair(__uint_as_float(sb | ((uint32_t)rs[h][v][i] & 0x80000000u)),
                                                               __uint_as_float(sb | ((uint32_t)(rs[h][v][i] >> 32) & 0x80000000u)));
                            wh[h][v][i] = add2(wh[h][v][i], st);
                            sum[h][v][i] = add2(sum[h][v][i], st);
                            rs[h][v][i] = fma2(wh[h][v][i], minus_one, wc[h][v][i]);
                        }
                    sj[h] = __fmul_rn(sj[h], 0.5f);
                }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = ((p0 + b0 + h) * 8 + warp) * RPW + sub;
                // (a one-bit base whose range exceeds fp16: the scale is infinite, its reciprocal 0, no residual a number, every bit 0)
                const bool live = (long long)rt * D2MOE_TILE_ROWS + r < L.rows && inv[h] > 0.0f;
                const unsigned long long k2 = pair(inv[h] * two_nl, inv[h] * two_nl);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    uint32_t c[4];
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        // code = q 2^n + (sum / s1 2^(n+1) + 2^n - 1) / 2: a whole number up to rounding errors below 1e-4
                        const unsigned long long z = add2(fma2(q[h][v][i], nl2, fma2(sum[h][v][i], k2, half2_)), magic);
                        c[2 * i] = (uint32_t)z; c[2 * i + 1] = (uint32_t)(z >> 32);
                    }
                    // the low bytes, in the cell's order 0, 2, 1, 3
                    const uint32_t cell = __byte_perm(__byte_perm(c[0], c[2], 0x0040), __byte_perm(c[1], c[3], 0x0040), 0x5410);
                    *reinterpret_cast<uint32_t*>(cells + r * pack_cell_stride(GS) + 4 * (l + LPR * v)) = live ? cell : 0u;
                }
            }
        }
    }
    s1_max = __reduce_max_sync(0xffffffffu, s1_max);
    wabs_max = __reduce_max_sync(0xffffffffu, wabs_max);
    pack_finish<GS>(L, packed, blk, cells, image, s1_max, wabs_max);
}

// Free per-step scales, R rows of one group by one warp: the lane holds elements k = lane, lane + 32, ... of every row
// (`w`), as the pinned sums demand (32 strided partial sums, then a butterfly).  For every residual step the R sums are
// reduced together: each exchange halves the rows a lane still carries, which adds the same pairs as a butterfly per
// row and leaves one quotient per lane instead of R.  dw / den: the weights of Eq. 5 and their sum (USE_E), else the
// group's length (a power of two: the quotient is an exact product).  Outputs: `code` (top-width codes), `wh` (the
// values they stand for), `meta`; emit(row, level, scale) is called by lane 0.
template <int E, int R, bool USE_E, typename Emit>
__device__ __forceinline__ void free_codes(const float (&w)[R][E], float levels, int n_lv, const float (&dw)[E], float den,
                                           float (&wh)[R][E], uint32_t (&code)[R][E], __half2 (&meta)[R], unsigned& wabs_max, Emit emit) {
    static_assert(R == 1 || R == 2 || R == 4, "rows per step");
    const int lane = threadIdx.x & 31;
    auto quotient_lane = [](int r) { return R == 4 ? (r >> 1) * 16 + (r & 1) * 8 : r * 16; };
    float rs[R][E];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float fmn = INFINITY, fmx = -INFINITY;               // (compensated weights that are no numbers count for neither)
#pragma unroll
        for (int e = 0; e < E; ++e) { fmn = fminf(fmn, w[r][e]); fmx = fmaxf(fmx, w[r][e]); }
        const float wmin = unordered(__reduce_min_sync(0xffffffffu, ordered(fmn))), wmax = unordered(__reduce_max_sync(0xffffffffu, ordered(fmx)));
        meta[r] = group_meta(wmin, wmax, levels);
        wabs_max = max(wabs_max, __float_as_uint(fmaxf(fabsf(wmin), fabsf(wmax))));
        const float s1 = __low2float(meta[r]), lo = __high2float(meta[r]), inv = __frcp_rn(s1);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float wc = __fadd_rn(w[r][e], 0.0f);
            const float q = base_code(__fsub_rn(wc, lo), s1, inv, levels);
            code[r][e] = (uint32_t)q;
            wh[r][e] = __fadd_rn(lo, __fmul_rn(q, s1));
            rs[r][e] = __fsub_rn(wc, wh[r][e]);
        }
    }
    int numbers = 0;                                         // steps whose scale is a number, of the row this lane forms the quotient of
#pragma unroll 1
    for (int j = 0; j < n_lv; ++j) {
        float part[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            part[r] = 0.0f;
#pragma unroll
            for (int e = 0; e < E; ++e) part[r] = __fadd_rn(part[r], USE_E ? __fmul_rn(fabsf(rs[r][e]), dw[e]) : fabsf(rs[r][e]));
        }
        float v;
        if constexpr (R == 4) {                              // lanes with bit 4 clear keep rows 0, 1, the others rows 2, 3
            const bool up = lane & 16;
            const float a = __shfl_xor_sync(0xffffffffu, up ? part[0] : part[2], 16);
            const float b = __shfl_xor_sync(0xffffffffu, up ? part[1] : part[3], 16);
            const float k0 = __fadd_rn(up ? part[2] : part[0], a), k1 = __fadd_rn(up ? part[3] : part[1], b);
            const bool up8 = lane & 8;
            v = __fadd_rn(up8 ? k1 : k0, __shfl_xor_sync(0xffffffffu, up8 ? k0 : k1, 8));
        } else if constexpr (R == 2) {
            const bool up = lane & 16;
            v = __fadd_rn(up ? part[1] : part[0], __shfl_xor_sync(0xffffffffu, up ? part[0] : part[1], 16));
            v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 8));
        } else {
            v = __fadd_rn(part[0], __shfl_xor_sync(0xffffffffu, part[0], 16));
            v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 8));
        }
#pragma unroll
        for (int off = 4; off; off >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, off));
        const float mean = USE_E ? __fdiv_rn(v, den) : __fmul_rn(v, 1.0f / (32 * E));
        const float sv = __half2float(__float2half_rn(mean));
        if constexpr (USE_E) numbers += sv == sv;            // (a plain mean is a number whenever the residuals are)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float sj = __shfl_sync(0xffffffffu, sv, quotient_lane(r));
            if (lane == 0) emit(r, j, __float2half_rn(sj));
#pragma unroll
            for (int e = 0; e < E; ++e) residual_step(__fadd_rn(w[r][e], 0.0f), sj, wh[r][e], rs[r][e], code[r][e]);
        }
    }
    const uint32_t flip = (1u << n_lv) - 1u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // A residual that is no number gives the bit 0.  That is every residual from the base on if the base scale is infinite (a
        // one-bit base whose range exceeds fp16), and those after the first step whose scale is no number (a group whose
        // weights of Eq. 5 are all zero; a step's bit is decided before its scale counts).
        const int stand = USE_E ? __shfl_sync(0xffffffffu, numbers, quotient_lane(r)) + 1 : n_lv;
        const uint32_t keep = __hisinf(__low2half(meta[r])) ? 0u : ~0u << max(n_lv - stand, 0);
#pragma unroll
        for (int e = 0; e < E; ++e) code[r][e] = (code[r][e] ^ flip) & keep;
    }
}

// Free scales, no error compensation.  One block per packed block; a warp takes four rows at a time.  col_energy
// (optional) weights the scale fit of Eq. 5.  Bound: instruction issue (about 60 per weight for a 2 -> 8 bit list).
template <int GS, bool USE_E>
__global__ void __launch_bounds__(PACK_THREADS)
pack_free_kernel(PackLayout L, const float* __restrict__ W, uint8_t* __restrict__ packed, const float* __restrict__ col_energy) {
    constexpr int E = GS / 32, R = E > 4 ? 2 : 4;
    extern __shared__ __align__(16) uint8_t smem[];
    uint8_t* cells = smem;
    uint8_t* image = smem + D2MOE_TILE_ROWS * pack_cell_stride(GS);
    const int G = blockIdx.x, rt = blockIdx.y;
    uint8_t* blk = packed + d2moe_block_offset(L, rt, G);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float levels = (float)((1 << L.b1) - 1);
    const int n_lv = L.top - L.b1;
    float dw[E], den = 1.0f;
    if constexpr (USE_E) {
        float d = 0.0f;
#pragma unroll
        for (int e = 0; e < E; ++e) { dw[e] = col_energy[(long long)G * GS + lane + 32 * e]; d = __fadd_rn(d, dw[e]); }
        for (int off = 16; off; off >>= 1) d = __fadd_rn(d, __shfl_xor_sync(0xffffffffu, d, off));
        den = d;
    }
    unsigned s1_max = 0, wabs_max = 0;
#pragma unroll 1
    for (int r0 = warp * R; r0 < D2MOE_TILE_ROWS; r0 += 8 * R) {
        float w[R][E], wh[R][E];
        uint32_t code[R][E];
        __half2 meta[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long row = (long long)rt * D2MOE_TILE_ROWS + r0 + r;
#pragma unroll
            for (int e = 0; e < E; ++e) w[r][e] = row < L.rows ? W[row * (long long)L.cols + (long long)G * GS + lane + 32 * e] : 0.0f;
        }
        free_codes<E, R, USE_E>(w, levels, n_lv, dw, den, wh, code, meta, wabs_max, [&](int r, int lv, __half s) {
            const bool live = (long long)rt * D2MOE_TILE_ROWS + r0 + r < L.rows;
            *reinterpret_cast<__half*>(image + d2moe_level_offset(L, lv, r0 + r)) = live ? s : __ushort_as_half(0);
        });
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const bool live = (long long)rt * D2MOE_TILE_ROWS + r0 + r < L.rows;  // padding rows: zero codes, meta and scales
            uint8_t* dst = cells + (r0 + r) * pack_cell_stride(GS);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int k = lane + 32 * e;
                dst[(k & ~3) + cell_byte(k)] = live ? (uint8_t)code[r][e] : (uint8_t)0;
            }
            if (lane == 0) {
                reinterpret_cast<__half2*>(image)[r0 + r] = live ? meta[r] : __halves2half2(__ushort_as_half(0), __ushort_as_half(0));
                if (live) s1_max = max(s1_max, __float_as_uint(__low2float(meta[r])));
            }
        }
    }
    pack_finish<GS>(L, packed, blk, cells, image, s1_max, wabs_max);
}

// Calibration-aware packing with error compensation (Algorithm 1), all groups of the matrix in one launch.
//
// A row never meets another row: W[r, c] loses E[r, j] H^c[j, c] for all earlier columns j, in ascending order, each one
// fp32 multiply and one fp32 subtract (the pinned order).  So the update is taken "left-looking": a warp owns R rows and
// walks the groups; for a group it starts from the original weights, subtracts the products of ALL earlier groups' E in
// one ascending pass with the sums in registers, quantizes the group, and leaves the group's E in W's own columns, where
// only this warp reads it again.  Nothing is written twice and no group waits for a launch.  (One pass over all later
// columns per group instead reads and writes the whole matrix once per group and starts 2 n_groups kernels.)
// The panel H^c[0..b, b..b+g) streams through shared memory in chunks of CAL_KC rows (two or three of them, cp.async), the
// warp's E chunk is transposed into shared memory.
// Bound: fp32 instruction issue, two instructions per (weight, earlier column): 6.4 ms for 14336 x 4096.
// Measured there (one B200): 9.2 ms; one pass over all later columns per group, two launches each, took 64.8 ms.
// Registers: a lane owns E neighbouring columns of each of the R rows as packed pairs (one instruction per two products);
// the pinned order of the scale fit wants columns lane, lane + 32, ..., so a finished group goes through a row buffer.
constexpr int CAL_KC = 32;

template <int GS, int R>
struct CalShape {
    static constexpr int E = GS / 32;                                      // columns per lane
    // With one or two rows a warp (few rows in all) a scheduler has a warp or two and the copies are what a chunk waits for: three
    // chunks in flight and all loads of a chunk's products ahead of them.  (256 x 4096, group size 128: 1970 us with two
    // chunks and four products unrolled, now 1420; 128 x 14336: 23.2 -> 16.7 ms.)
    static constexpr int STAGES = R >= 4 ? 2 : 3;
    static constexpr int UNROLL = R == 1 ? 32 : (R == 2 ? 16 : 4);
    // floats per warp: the E chunk [CAL_KC][R], the finished rows [R][GS], the cells of one row
    static constexpr int WARP_FLOATS = CAL_KC * R + R * GS + GS / 4;
};

template <int GS, int R>
__global__ void __launch_bounds__(R >= 4 ? 640 : 1024, 1)
pack_calibrated_kernel(PackLayout L, float* W, const float* __restrict__ hc, const float* __restrict__ col_energy,
                       uint8_t* __restrict__ packed, int n_warp_tiles, float one) {
    using C = CalShape<GS, R>;
    constexpr int E = C::E;
    constexpr int STAGES = C::STAGES, UNROLL = C::UNROLL;
    extern __shared__ __align__(16) uint8_t smem[];
    float* hs = reinterpret_cast<float*>(smem);                            // [STAGES][CAL_KC][GS]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    float* es = hs + STAGES * CAL_KC * GS + warp * C::WARP_FLOATS;
    float* rows_s = es + CAL_KC * R;
    uint32_t* cs = reinterpret_cast<uint32_t*>(rows_s + R * GS);
    const float levels = (float)((1 << L.b1) - 1);
    const int n_lv = L.top - L.b1;
    const bool hc_aligned = (reinterpret_cast<uintptr_t>(hc) & 15) == 0;
    const unsigned long long one2 = pair(one, one);                        // 1.0f, not known at compile time
    unsigned s1_max = 0, wabs_max = 0;
    auto col = [&](int e) { return E >= 4 ? 4 * lane + (e & 3) + 128 * (e >> 2) : E * lane + e; };   // the lane's columns

    // warp tile of this warp: tiles are dealt to the blocks warp by warp, so that every block gets its share
    for (int base = 0; base < n_warp_tiles; base += gridDim.x * n_warps) {
        const int tile = base + warp * gridDim.x + blockIdx.x;
        const long long row0 = (long long)tile * R;
        const bool mine = tile < n_warp_tiles;
#pragma unroll 1
        for (int G = 0; G < L.n_groups; ++G) {
            const int b = G * GS;
            float w[R][E];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int e = 0; e < E; ++e) w[r][e] = mine && row0 + r < L.rows ? W[(row0 + r) * (long long)L.cols + b + col(e)] : 0.0f;
            int fill = 0, drain = 0;                                       // stages the next chunk goes to and the next one read is in
            auto stage = [&](int k0) {                                     // rows k0 .. k0 + CAL_KC of the panel, if it has them
                const uint32_t dst = smem_u32(hs + fill * CAL_KC * GS);
                if (++fill == STAGES) fill = 0;
                const float* src = hc + (long long)k0 * L.cols + b;
                if (k0 >= b) {
                } else if (hc_aligned) {
                    for (int i = threadIdx.x; i < CAL_KC * GS / 4; i += blockDim.x)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * i), "l"(src + (long long)(i / (GS / 4)) * L.cols + 4 * (i % (GS / 4))) : "memory");
                } else {
                    for (int i = threadIdx.x; i < CAL_KC * GS; i += blockDim.x)
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * i), "l"(src + (long long)(i / GS) * L.cols + i % GS) : "memory");
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            float ev[R];
            auto load_e = [&](int k0) {                                    // E of columns k0 .. k0 + 31, one column per lane
#pragma unroll
                for (int r = 0; r < R; ++r) ev[r] = mine && row0 + r < L.rows ? W[(row0 + r) * (long long)L.cols + k0 + lane] : 0.0f;
            };
#pragma unroll 1
            for (int c = 0; c < STAGES - 1; ++c) stage(c * CAL_KC);
            if (b > 0) load_e(0);
            for (int k0 = 0; k0 < b; k0 += CAL_KC) {
                __syncwarp();
#pragma unroll
                for (int r = 0; r < R; ++r) es[lane * R + r] = -ev[r];
                asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
                __syncthreads();                                           // the chunk is there, the one before it has been read
                stage(k0 + (STAGES - 1) * CAL_KC);
                if (k0 + CAL_KC < b) load_e(k0 + CAL_KC);
                const float* hp = hs + drain * CAL_KC * GS;
                if (++drain == STAGES) drain = 0;
                if (!mine) continue;                                       // such a warp only helps with the copies
#pragma unroll UNROLL
                for (int k = 0; k < CAL_KC; ++k) {
                    // (-e) h rounds to -(e h), so that adding it is the subtraction of the definition.  The assembler contracts a
                    // packed product and a packed sum into one fused operation (one rounding: other bits), so the sum is
                    // written as product x one + w, which rounds the same and leaves it nothing to contract.
                    // (E is read one word at a time: a broadcast of 16 bytes takes the shared-memory pipe four cycles, like four.)
                    float h[E];
                    if constexpr (E >= 4) {
#pragma unroll
                        for (int e = 0; e < E; e += 4)
                            *reinterpret_cast<float4*>(h + e) = *reinterpret_cast<const float4*>(hp + k * GS + 4 * lane + 32 * e);
                    } else if constexpr (E == 2) *reinterpret_cast<float2*>(h) = *reinterpret_cast<const float2*>(hp + k * GS + 2 * lane);
                    else h[0] = hp[k * GS + lane];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float me = es[k * R + r];
                        if constexpr (E == 1) w[r][0] = __fadd_rn(w[r][0], __fmul_rn(me, h[0]));
                        else {
#pragma unroll
                            for (int e = 0; e < E; e += 2) {
                                const unsigned long long v = fma2(mul2(pair(me, me), pair(h[e], h[e + 1])), one2, pair(w[r][e], w[r][e + 1]));
                                w[r][e] = first(v); w[r][e + 1] = second(v);
                            }
                        }
                    }
                }
            }
            if (mine) {
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int e = 0; e < E; ++e) rows_s[r * GS + col(e)] = w[r][e];
            }
            __syncthreads();                                               // the last chunk has been read by every warp

            // quantize the group: one row at a time (a few percent of the work)
            float dw[E], den = (float)GS, hd[E];
            if (col_energy) {
                float d = 0.0f;
#pragma unroll
                for (int e = 0; e < E; ++e) { dw[e] = col_energy[b + lane + 32 * e]; d = __fadd_rn(d, dw[e]); }
                for (int off = 16; off; off >>= 1) d = __fadd_rn(d, __shfl_xor_sync(0xffffffffu, d, off));
                den = d;
            }
            const bool keep_error = G + 1 < L.n_groups;
#pragma unroll
            for (int e = 0; e < E; ++e) hd[e] = keep_error ? hc[(long long)(b + lane + 32 * e) * (L.cols + 1)] : 1.0f;
            if (!mine) continue;
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const long long row = row0 + r;
                if (row >= L.rows_pad) break;
                const int rt = (int)(row / D2MOE_TILE_ROWS), rr = (int)(row % D2MOE_TILE_ROWS);
                uint8_t* blk = packed + d2moe_block_offset(L, rt, G);
                const bool live = row < L.rows;                            // padding rows: zero codes, meta and scales
                float w1[1][E], wh[1][E];
                uint32_t code[1][E];
                __half2 meta[1];
#pragma unroll
                for (int e = 0; e < E; ++e) w1[0][e] = rows_s[r * GS + lane + 32 * e];
                auto emit = [&](int, int lv, __half s) {
                    *reinterpret_cast<__half*>(blk + d2moe_level_offset(L, lv, rr)) = live ? s : __ushort_as_half(0);
                };
                if (col_energy) free_codes<E, 1, true>(w1, levels, n_lv, dw, den, wh, code, meta, wabs_max, emit);
                else free_codes<E, 1, false>(w1, levels, n_lv, dw, den, wh, code, meta, wabs_max, emit);
                if (lane == 0) {
                    reinterpret_cast<__half2*>(blk)[rr] = live ? meta[0] : __halves2half2(__ushort_as_half(0), __ushort_as_half(0));
                    if (live) s1_max = max(s1_max, __float_as_uint(__low2float(meta[0])));
                }
                __syncwarp();
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int k = lane + 32 * e;
                    reinterpret_cast<uint8_t*>(cs)[(k & ~3) + cell_byte(k)] = live ? (uint8_t)code[0][e] : (uint8_t)0;
                    if (keep_error && live)                                // E = (W - W_hat) / H^c[j, j], in place of the group's weights
                        W[row * (long long)L.cols + b + k] = __fdiv_rn(__fsub_rn(w1[0][e], wh[0][e]), hd[e]);
                }
                __syncwarp();
                if (lane < GS / 32) {
                    uint32_t cell[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) cell[i] = cs[8 * lane + i];
                    store_fields<GS>(L, blk, rr, lane, cell);
                }
            }
        }
    }
    if (lane == 0 && s1_max) raise_maxima(packed, s1_max, wabs_max);
}

__global__ void unpack_kernel(PackLayout L, const uint8_t* __restrict__ packed, int bits,
                              uint8_t* __restrict__ codes, float* __restrict__ scale,
                              float* __restrict__ offset) {
    const long long n = (long long)L.rows * L.cols;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int row = (int)(idx / L.cols), col = (int)(idx - (long long)row * L.cols);
        const int rt = row / D2MOE_TILE_ROWS, r = row - rt * D2MOE_TILE_ROWS;
        const int G = col / L.g, k = col - G * L.g;
        const uint8_t* blk = packed + d2moe_block_offset(L, rt, G);
        unsigned code = 0;
        for (int j = 0; j < L.n_seg; ++j) {
            int bitpos;
            const int wo = d2moe_elem_word(L, j, r, k, &bitpos);
            const uint32_t word = *reinterpret_cast<const uint32_t*>(blk + wo);
            code |= ((word >> bitpos) & ((1u << L.seg_w[j]) - 1u)) << L.seg_shift[j];
        }
        codes[idx] = (uint8_t)(code >> (L.top - bits));
        if (k == 0) {
            const __half2 m = reinterpret_cast<const __half2*>(blk)[r];
            if (scale) scale[(long long)row * L.n_groups + G] = __low2float(m);
            if (offset) offset[(long long)row * L.n_groups + G] = __high2float(m);
        }
    }
}

// scale_mode 1: the free scale of every residual step, s_extra[row, G, level]
__global__ void unpack_scales_kernel(PackLayout L, const uint8_t* __restrict__ packed, float* __restrict__ s_extra) {
    const int n_lv = L.top - L.b1;
    const long long n = (long long)L.rows * L.n_groups * n_lv;
    for (long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x; idx < n;
         idx += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(idx % n_lv);
        const long long rg = idx / n_lv;
        const int G = (int)(rg % L.n_groups), row = (int)(rg / L.n_groups);
        const int rt = row / D2MOE_TILE_ROWS, r = row - rt * D2MOE_TILE_ROWS;
        const uint8_t* blk = packed + d2moe_block_offset(L, rt, G);
        s_extra[idx] = __half2float(*reinterpret_cast<const __half*>(blk + d2moe_level_offset(L, l, r)));
    }
}

}  // namespace

static cudaError_t launch_header(const PackLayout& L, const int* bits, int n_bits, uint8_t* packed, cudaStream_t st) {
    int b[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int i = 0; i < n_bits; ++i) b[i] = bits[i];
    pack_header_kernel<<<1, 32, 0, st>>>(reinterpret_cast<PackHeader*>(packed), L, n_bits,
                                         b[0], b[1], b[2], b[3], b[4], b[5], b[6], b[7]);
    return cudaGetLastError();
}

template <int GS>
static cudaError_t launch_pack_gs(const PackLayout& L, const float* W, const float* col_energy, uint8_t* packed, cudaStream_t st) {
    const dim3 grid(L.n_groups, L.n_rt);
    const int smem = D2MOE_TILE_ROWS * pack_cell_stride(GS) + L.block_bytes;
    if (L.scale_mode == 0) {
        cudaError_t e = ensure_dynamic_smem<&pack_tied_kernel<GS>>(smem);
        if (e != cudaSuccess) return e;
        pack_tied_kernel<GS><<<grid, PACK_THREADS, smem, st>>>(L, W, packed);
    } else if (col_energy) {
        cudaError_t e = ensure_dynamic_smem<&pack_free_kernel<GS, true>>(smem);
        if (e != cudaSuccess) return e;
        pack_free_kernel<GS, true><<<grid, PACK_THREADS, smem, st>>>(L, W, packed, col_energy);
    } else {
        cudaError_t e = ensure_dynamic_smem<&pack_free_kernel<GS, false>>(smem);
        if (e != cudaSuccess) return e;
        pack_free_kernel<GS, false><<<grid, PACK_THREADS, smem, st>>>(L, W, packed, nullptr);
    }
    return cudaGetLastError();
}

static cudaError_t launch_pack_any(const PackLayout& L, const float* W, const float* col_energy, uint8_t* packed, cudaStream_t st) {
    switch (L.g) {
        case 32: return launch_pack_gs<32>(L, W, col_energy, packed, st);
        case 64: return launch_pack_gs<64>(L, W, col_energy, packed, st);
        case 128: return launch_pack_gs<128>(L, W, col_energy, packed, st);
        default: return launch_pack_gs<256>(L, W, col_energy, packed, st);
    }
}

template <int GS, int R>
static cudaError_t launch_calibrated_gs(const PackLayout& L, float* W, const float* hc, const float* col_energy, uint8_t* packed,
                                        int grid, cudaStream_t st) {
    const int tiles = (L.rows_pad + R - 1) / R, max_warps = R >= 4 ? 20 : 32;
    int warps = (tiles + grid - 1) / grid;
    warps = warps < 8 ? 8 : (warps > max_warps ? max_warps : warps);      // at least eight share the panel's copies
    const int smem = (CalShape<GS, R>::STAGES * CAL_KC * GS + warps * CalShape<GS, R>::WARP_FLOATS) * 4;
    cudaError_t e = ensure_dynamic_smem<&pack_calibrated_kernel<GS, R>>(smem);
    if (e != cudaSuccess) return e;
    pack_calibrated_kernel<GS, R><<<grid, 32 * warps, smem, st>>>(L, W, hc, col_energy, packed, tiles, 1.0f);
    return cudaGetLastError();
}

// Rows per warp: the whole matrix is one wave of warps where it fits, so what counts is the number of rows on the busiest
// scheduler (an SM has four); equal counts go to the larger R (fewer shared-memory reads per product).
template <int GS>
static cudaError_t launch_calibrated_any(const PackLayout& L, float* W, const float* hc, const float* col_energy, uint8_t* packed,
                                         cudaStream_t st) {
    const int grid = device_sm_count();
    const int cand[4] = {1, 2, 4, 5};
    int best = 4;
    long long best_cost = -1;
    for (int R : cand) {
        const long long tiles = (L.rows_pad + R - 1) / R, per_sm = (tiles + grid - 1) / grid;
        const long long cost = (per_sm + 3) / 4 * R;
        if (GS == 256 && R == 5) continue;                                 // registers
        if (best_cost < 0 || cost <= best_cost) { best = R; best_cost = cost; }
    }
    if constexpr (GS != 256)
        if (best == 5) return launch_calibrated_gs<GS, 5>(L, W, hc, col_energy, packed, grid, st);
    if (best == 4) return launch_calibrated_gs<GS, 4>(L, W, hc, col_energy, packed, grid, st);
    if (best == 2) return launch_calibrated_gs<GS, 2>(L, W, hc, col_energy, packed, grid, st);
    return launch_calibrated_gs<GS, 1>(L, W, hc, col_energy, packed, grid, st);
}

cudaError_t launch_pack_calibrated(const PackLayout& L, const int* bits, int n_bits, float* W, const float* hc,
                                   const float* col_energy, uint8_t* packed, cudaStream_t st) {
    cudaError_t err = launch_header(L, bits, n_bits, packed, st);
    if (err != cudaSuccess) return err;
    if (!hc) return launch_pack_any(L, W, col_energy, packed, st);         // no compensation: every group on its own
    switch (L.g) {
        case 32: return launch_calibrated_any<32>(L, W, hc, col_energy, packed, st);
        case 64: return launch_calibrated_any<64>(L, W, hc, col_energy, packed, st);
        case 128: return launch_calibrated_any<128>(L, W, hc, col_energy, packed, st);
        default: return launch_calibrated_any<256>(L, W, hc, col_energy, packed, st);
    }
}

cudaError_t launch_pack(const PackLayout& L, const int* bits, int n_bits, const float* W, uint8_t* packed,
                        cudaStream_t st) {
    cudaError_t err = launch_header(L, bits, n_bits, packed, st);
    if (err != cudaSuccess) return err;
    return launch_pack_any(L, W, nullptr, packed, st);
}

cudaError_t launch_unpack_scales(const PackLayout& L, const uint8_t* packed, float* s_extra, cudaStream_t st) {
    const long long n = (long long)L.rows * L.n_groups * (L.top - L.b1);
    if (n == 0) return cudaSuccess;
    int blocks = (int)((n + 255) / 256 < 148 * 16 ? (n + 255) / 256 : 148 * 16);
    unpack_scales_kernel<<<blocks, 256, 0, st>>>(L, packed, s_extra);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const PackLayout& L, const uint8_t* packed, int bits, uint8_t* codes,
                          float* scale, float* offset, cudaStream_t st) {
    long long n = (long long)L.rows * L.cols;
    int blocks = (int)((n + 255) / 256 < 148 * 16 ? (n + 255) / 256 : 148 * 16);
    if (blocks < 1) blocks = 1;
    unpack_kernel<<<blocks, 256, 0, st>>>(L, packed, bits, codes, scale, offset);
    return cudaGetLastError();
}
