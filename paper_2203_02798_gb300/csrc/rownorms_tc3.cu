// rownorms_tc3.cu -- row norms x_i = alpha ||A_i B||^2 + beta x_i to FP32
// accuracy on tcgen05 (dense A, d <= 256).
//
// A and B are scaled by powers of two, columns of A by s_j and columns of B
// by 1 / t_l with the rows of B taking 1 / s_j, so that a typical entry of A
// is about 2^10 and the largest of each column of B 128 .. 256.  Each scaled
// entry is then split into three bf16 terms,
//     y = hi + mid + lo,   hi = the bf16 rounding of the nearest integer,
// so that the products hi hi are whole numbers: their sum over K <= 256 is
// exact in the FP32 accumulator while it stays below 2^24, which the tensor
// pipe (it rounds toward zero) would otherwise spoil by some 2^-19.  The
// products hi mid, mid hi, hi lo, lo hi and mid mid, 2^-8 of the first or less,
// go to a second accumulator; (acc0 + acc1) t_l is squared and summed in the
// epilogue.  (Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012, with the
// first slice on a fixed grid.)
//
// That holds for rows within a factor of about 30 of the typical row.  A row is put
// on a list, and the CUDA-core kernel does the listed rows, where the second
// accumulator may hold more than 2^-5 of the norm (there the terms left out are as
// large as FP32's roundings), where an accumulator reaches 2^24, and where the sum
// is not finite or near FP32's bottom.  A column's own acc1 may cancel, so that its
// share is taken from all columns.  The norm has to be 2^10 times what remainders
// of 1/12 each, squared, in A's entries would give on average, and 2^10 times the sum
// of the acc1^2 with the weight (t_l^2) that B's remainders have on average.
//
// One persistent CTA pair per two SMs (cta_group::2, M = 256): each CTA keeps
// half of every K-chunk's B tile, three bf16 slices of it, beside a ring of
// 24 KB stages (128 rows x 32 K, three slices).  Warps: 0-7 epilogue (two per
// TMEM lane quarter), 8 MMA issue (even CTA), 9-19 converters (32- or 64-row
// pieces: 16-byte loads, scale, split, 64-byte-swizzled stores).  Up to 128 columns
// the accumulators are double-buffered.  750,001 x 200 times 200 x 200:
// 0.37 ms against 1.98 on CUDA cores; errors 3.2e-8 (root mean square, relative)
// against 6.7e-8.
#include "tc_common.cuh"

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

namespace {

constexpr int kRows = 128, kKC = 32, kMaxQ = 8;
constexpr int kEpiWarps = 8, kMmaWarp = 8, kConv0 = 9, kConvWarps = 11;
constexpr int kThreads = (kConv0 + kConvWarps) * 32;
constexpr uint32_t kSlice = kRows * kKC * 2;          // one bf16 tile of a stage: 8 KB
constexpr uint32_t kStage = 3 * kSlice;
// Pieces a converter warp works in.  64 rows: loads, then waits for its stage,
// then splits and stores; 16 loads a lane in flight keep A streaming.  Early, 32
// rows: has the piece split, in registers, before it waits, and the next one's
// loads on their way.  With B's image beside it the ring has three stages at 200
// columns, and the time from a stage's release to its refill is what the MMAs wait
// for (750,001 x 200 times 200 x 200: 372 us early, 439 late; 500,000 x 256
// triangular, four stages, 235 and 256).  With five stages and more (1M x 128
// times 128 x 128) it is A: 203 early, 166 late.
template <bool kEarly>
struct Piece {
    static constexpr int kRowsOf = kEarly ? 32 : 64, kQuads = kRowsOf / 4, kParts = kRows / kRowsOf;
};
constexpr int kEarlyStages = 4;
constexpr int kMaxStages = 8, kMinStages = 3;
constexpr size_t kSmemLimit = 232448;
constexpr uint32_t kTail = 1024;                      // barriers, and four floats at its end
constexpr uint32_t kXchg = 4 * kRows * 4;             // the epilogue halves' exchange
constexpr size_t kExtra = 1024 + kTail + 2 * 256 * 4 + kXchg;
constexpr int kSampleGroups = 64, kSampleRows = 8;

struct Rn3Params {
    const float* A;
    int64_t lda, n;
    float* x;
    float alpha, beta;
    int d, c, nq, npad, ntiles, stages, nbuf;
    uint32_t n0[kMaxQ], nn[kMaxQ], hoff[kMaxQ];
    uint32_t hb;              // bytes of one slice of a CTA's half of B
    const uint8_t* img;       // [half][slice][hb]
    const float *s, *t;       // column scales of A, result scales of B's columns
    const float *norm, *rest; // of B's scaled columns: sum of squares, and of the remainders after hi
    int *list, *count;        // rows left to the CUDA-core kernel (*count < 0: all)
    int* flag;
};

__device__ __forceinline__ float pow2f(int e) { return __uint_as_float((uint32_t)(min(max(e, -126), 127) + 127) << 23); }
__device__ __forceinline__ int exponent(float v) { return (int)(__float_as_uint(v) >> 23) - 127; }   // v > 0

// s_j: 2^10 over the power of two below the median, over 64 groups of 8
// consecutive rows spread over A, of the largest |a_ij| (a few outlying rows
// do not move it; a column that is mostly zero takes its largest, one with no
// nonzero in the sample is left at 0: scale_of()).  *count: 0, or -1 where more than
// two thirds of the sampled rows are so far from the typical one, by their first 32
// columns, that their norms would be left to the CUDA cores (rows 2^-6 of it or
// 2^6 times): these then do all rows at once (750,001 x 200 times 200 x 200 with 85%
// of the rows scaled by 1e-4: 2,487 us with the tensor-core pass before them).
constexpr int kUnitWarps = 32;
__global__ void __launch_bounds__(kUnitWarps * 32) rn3_units_kernel(const float* __restrict__ A, int64_t lda, int64_t n, int d,
                                                                  float* __restrict__ s, int* __restrict__ count) {
    pdl_enter(A, s, count);
    __shared__ float gm[kSampleGroups][33];
    __shared__ float med[32];
    __shared__ int far;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = (int)blockIdx.x * 32 + lane;
    constexpr int kGroups = kSampleGroups / kUnitWarps;   // of a warp
    float v[kGroups][kSampleRows];
    if (threadIdx.x == 0) far = 0;
#pragma unroll
    for (int k = 0; k < kGroups; ++k) {
        const int g = w + k * kUnitWarps;
        const int64_t r0 = (n - kSampleRows) * g / (kSampleGroups - 1);
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < kSampleRows; ++i) v[k][i] = j < d ? fabsf(__ldg(A + (r0 + i) * lda + j)) : 0.f;
#pragma unroll
        for (int i = 0; i < kSampleRows; ++i) m = fmaxf(m, v[k][i]);
        gm[g][lane] = m;
    }
    __syncthreads();
    float mx = 0.f;
    for (int g = 0; g < kSampleGroups; ++g) mx = fmaxf(mx, gm[g][lane]);
    for (int g = w; g < kSampleGroups; g += kUnitWarps) {
        const float v = gm[g][lane];
        int rank = 0;
        for (int h = 0; h < kSampleGroups; ++h) rank += gm[h][lane] < v || (gm[h][lane] == v && h < g);
        if (rank == kSampleGroups / 2) med[lane] = v;
    }
    __syncthreads();
    const float m = med[lane] > 0.f ? med[lane] : mx;
    const float sj = m > 0.f ? (m <= 3.402823466e38f ? pow2f(10 - exponent(m)) : 1.f) : 0.f;
    if (w == 0 && j < 256) s[j] = sj;
    if (blockIdx.x != 0) return;
    // the sampled rows' largest scaled entries: 2^10 .. 2^12 in a typical row
    int out = 0;
#pragma unroll
    for (int k = 0; k < kGroups; ++k)
#pragma unroll
        for (int i = 0; i < kSampleRows; ++i) {
            float r = v[k][i] * sj;
#pragma unroll
            for (int o = 16; o; o >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, o));
            out += r > 0.f && (r < 16.f || r > 262144.f);
        }
    if (lane == 0) atomicAdd(&far, out);
    __syncthreads();
    if (threadIdx.x == 0) *count = 3 * far > 2 * kSampleGroups * kSampleRows ? -1 : 0;
}

// The scale of a column: its own, or the largest of all where the sample had no
// nonzero, which leaves its row of B, scaled by 1 / s_j, the least weight.  (At
// scale 1 it had the most: B's columns were then scaled by an entry that next to
// no row uses, and every row was left to the CUDA cores, 2,752 us at 750,001 x 200
// times 200 x 200.)
__device__ __forceinline__ float scale_of(float sj, float smax) { return sj > 0.f ? sj : smax > 0.f ? smax : 1.f; }

// scaled value y (an integer part below 2^24) as hi + mid + lo
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    float2 r;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}
__device__ __forceinline__ uint32_t to_bf16x2(float2 v) {   // v.x in the low half
    uint32_t h;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(v.y), "f"(v.x));
    return h;
}
__device__ __forceinline__ float2 neg_bf16x2(uint32_t h) {
    return make_float2(-__uint_as_float(h << 16), -__uint_as_float(h & 0xFFFF0000u));
}
__device__ __forceinline__ void split3(float2 y, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    constexpr float kMagic = 12582912.f;   // 1.5 * 2^23: y + magic has the nearest integer in its low bits
    hi = to_bf16x2(add2(add2(y, make_float2(kMagic, kMagic)), make_float2(-kMagic, -kMagic)));
    const float2 r = add2(y, neg_bf16x2(hi));
    mid = to_bf16x2(r);
    lo = to_bf16x2(add2(r, neg_bf16x2(mid)));
}

// The image of B: 8 columns a block.  Column l (0-based in this pass, column
// c0 + l of B) is scaled so that its largest |b_jl| / s_j is in [128, 256).
__global__ void __launch_bounds__(256) rn3_image_kernel(const float* __restrict__ B, int ldb, int c0, const Rn3Params p,
                                                        const float* __restrict__ sample, float* __restrict__ scale,
                                                        uint8_t* __restrict__ img, float* __restrict__ t,
                                                        float* __restrict__ norm, float* __restrict__ rest) {
    pdl_enter(B, sample, scale, img, t, norm, rest);
    __shared__ float red[32][9], red1[32][9], s[256], wmax[8];
    {
        const float own = sample[threadIdx.x];
        float m = own;
#pragma unroll
        for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
        __syncthreads();
        for (int w = 0; w < 8; ++w) m = fmaxf(m, wmax[w]);
        s[threadIdx.x] = scale_of(own, m);
        if (blockIdx.x == 0) scale[threadIdx.x] = s[threadIdx.x];
        __syncthreads();
    }
    const int col = threadIdx.x & 7, part = threadIdx.x >> 3, l = (int)blockIdx.x * 8 + col;
    float m = 0.f;
    if (l < p.c)
        for (int j = part; j < p.d; j += 32) m = fmaxf(m, fabsf(__ldg(B + (int64_t)j * ldb + c0 + l)) / s[j]);
    red[part][col] = m;
    __syncthreads();
    for (int k = 0; k < 32; ++k) m = fmaxf(m, red[k][col]);
    const int e = (m > 0.f && m <= 3.402823466e38f) ? exponent(m) : 0;
    const float f = pow2f(7 - e);
    if (part == 0) t[l] = pow2f(e - 7);
    float nb = 0.f, rb = 0.f;
    for (int i = part; i < p.nq * (kKC / 2); i += 32) {
        const int q = i / (kKC / 2), kl = (i % (kKC / 2)) * 2, r = l - (int)p.n0[q];
        if (r < 0) continue;
        const int k = kKC * q + kl;
        const float b0 = (k < p.d && l < p.c) ? __ldg(B + (int64_t)k * ldb + c0 + l) / s[k] * f : 0.f;
        const float b1 = (k + 1 < p.d && l < p.c) ? __ldg(B + (int64_t)(k + 1) * ldb + c0 + l) / s[k + 1] * f : 0.f;
        uint32_t w[3];
        split3(make_float2(b0, b1), w[0], w[1], w[2]);
        const float2 rem = add2(make_float2(b0, b1), neg_bf16x2(w[0]));
        nb += b0 * b0 + b1 * b1;
        rb += rem.x * rem.x + rem.y * rem.y;
        const int hn = (int)p.nn[q] / 2, h = r / hn;
        const uint32_t off = (uint32_t)h * 3 * p.hb + p.hoff[q] + tc::sw64_offset((uint32_t)(r - h * hn), (uint32_t)kl);
#pragma unroll
        for (int z = 0; z < 3; ++z) *reinterpret_cast<uint32_t*>(img + off + (uint32_t)z * p.hb) = w[z];
    }
    __syncthreads();
    red[part][col] = nb;
    red1[part][col] = rb;
    __syncthreads();
    if (part == 0) {
        for (int k = 1; k < 32; ++k) {
            nb += red[k][col];
            rb += red1[k][col];
        }
        norm[l] = nb;
        rest[l] = rb;
    }
}

// Lane l: float4 number l + 32 i of a piece of 4 Q rows x 32 columns (row l / 8 +
// 4 i, columns 4 (l % 8) ..).
template <bool VEC, int Q>
__device__ __forceinline__ void load_piece(const Rn3Params& p, int64_t row0, int q, int lane, float4 (&v)[Q]) {
    const int k = kKC * q + 4 * (lane & 7);
    const int64_t r0 = row0 + (lane >> 3);
    if (VEC && row0 + 4 * Q <= p.n && kKC * q + kKC <= p.d) {
        const float* src = p.A + r0 * p.lda + k;
        const int64_t step = 4 * p.lda;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                         : "=f"(v[i].x), "=f"(v[i].y), "=f"(v[i].z), "=f"(v[i].w) : "l"(src));
            src += step;
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int64_t row = r0 + 4 * i;
        if (row >= p.n || k >= p.d) continue;
        const float* src = p.A + row * p.lda + k;
        if (VEC) {   // d a multiple of 4: the quad is whole
            v[i] = __ldg(reinterpret_cast<const float4*>(src));
        } else {
            v[i].x = __ldg(src);
            if (k + 1 < p.d) v[i].y = __ldg(src + 1);
            if (k + 2 < p.d) v[i].z = __ldg(src + 2);
            if (k + 3 < p.d) v[i].w = __ldg(src + 3);
        }
    }
}

// Scale and split a quad: its three terms.
__device__ __forceinline__ void split_quad(float4 s, float4 v, uint2 (&w)[3]) {
    split3(mul2(make_float2(v.x, v.y), make_float2(s.x, s.y)), w[0].x, w[1].x, w[2].x);
    split3(mul2(make_float2(v.z, v.w), make_float2(s.z, s.w)), w[0].y, w[1].y, w[2].y);
}
// Store a piece, quad i's terms by terms(i, w): rows 4 Q part + l / 8 + 4 i of the
// stage's K-major 64-byte-swizzled tiles (two base offsets a lane, as the swizzle
// phase of a row depends on i's parity alone).
template <int Q, class F>
__device__ __forceinline__ void store_piece(uint8_t* stage, int part, int lane, const F& terms) {
    const uint32_t l8 = (uint32_t)lane >> 3, c4 = (uint32_t)lane & 7u;
    const uint32_t lane_part = (uint32_t)part * (4u * Q * 64u) + l8 * 64u + (c4 & 1u) * 8u;
    uint8_t* const even = stage + lane_part + ((((c4 >> 1) ^ (l8 >> 1)) & 3u) << 4);
    uint8_t* const odd = stage + lane_part + 256u + ((((c4 >> 1) ^ (2u + (l8 >> 1))) & 3u) << 4);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        uint8_t* const dst = ((i & 1) ? odd : even) + (i >> 1) * 512;
        uint2 w[3];
        terms(i, w);
#pragma unroll
        for (int z = 0; z < 3; ++z) *reinterpret_cast<uint2*>(dst + z * kSlice) = w[z];
    }
}

__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
    int ok = 0;
    if ((threadIdx.x & 31) == 0) ok = tc::mbar_wait(bar, parity, abort) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

template <bool VEC, bool kEarly>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) rownorm_tc3_kernel(const Rn3Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    const int S = p.stages;
    const uint32_t rank = tc::cluster_ctarank();
    const int cid = (int)tc::cluster_id_x(), ncl = (int)tc::nclusters_x();
    uint8_t* sB = smem + S * kStage;                       // this CTA's half of B: three slices
    uint64_t* bars = reinterpret_cast<uint64_t*>(sB + 3 * p.hb);
    uint64_t* full = bars;                       // [S] even CTA: stage filled in both CTAs (2 kParts arrivals)
    uint64_t* empty = bars + kMaxStages;         // [S] stage consumed (multicast commit)
    uint64_t* tfull = bars + 2 * kMaxStages;     // [2] accumulators done (multicast commit)
    uint64_t* tempty = tfull + 2;                // [2] even CTA: accumulators read in both (16 arrivals)
    uint64_t* fin = tfull + 4;                   // all MMAs complete (multicast commit)
    uint64_t* xfull = fin + 1;                   // [4 quarters][4] second half's sums written (1 arrival)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(xfull + 16);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* stored = const_cast<int*>(abort) + 1;   // [S] pieces stored per stage (in use order)
    float* ss = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kTail);   // [256] column scales of A
    float* ts = ss + 256;                                                              // [256] result scales
    float* xchg = ts + 256;                                                            // [4][128]
    float* need = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bars) + kTail) - 4;   // [2] halves of the columns:
    float* weigh = need + 2;                                                                // [2] what a row needs (below)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            tc::mbar_init(full + s, 2 * Piece<kEarly>::kParts);
            tc::mbar_init(empty + s, 1);
            stored[s] = 0;
        }
        for (int a = 0; a < 2; ++a) {
            tc::mbar_init(tfull + a, 1);
            tc::mbar_init(tempty + a, 2 * kEpiWarps);
        }
        tc::mbar_init(fin, 1);
        for (int k = 0; k < 16; ++k) tc::mbar_init(xfull + k, 1);
        *abort = 0;
        tc::fence_mbar_init();
    }
    const uint8_t* img = p.img;
    pdl_enter(img);
    if (*(volatile const int*)p.count < 0) return;   // (both CTAs of every pair) the CUDA cores do all rows
    for (int j = threadIdx.x; j < 256; j += kThreads) {
        ss[j] = p.s[j];
        ts[j] = j < p.npad ? p.t[j] : 0.f;
    }
    if (warp < 2) {
        // need: 2^10 / 12 of what unit entries of the scaled A give; weigh: the
        // mean of t_l^2 over B's columns by their remainders
        float unit = 0.f, rest = 0.f, rest1 = 0.f;
        for (int l = 32 * warp + lane; l < p.npad; l += 64) {
            const float t = p.t[l];
            unit += t * t * p.norm[l];
            rest += t * t * p.rest[l];
            rest1 += p.rest[l];
        }
        unit = warp_sum(unit);
        rest = warp_sum(rest);
        rest1 = warp_sum(rest1);
        if (lane == 0) {
            need[warp] = unit * (1024.f / 12.f);
            weigh[warp] = rest1 > 0.f ? rest / rest1 : 0.f;
        }
    }
    if (warp == kMmaWarp) {
        tc::tmem_alloc_pair(tmem_slot, 512u);
        tc::tmem_relinquish_pair();
    }
    {   // this CTA's half of B
        const uint4* src = reinterpret_cast<const uint4*>(img + (size_t)rank * 3 * p.hb);
        uint4* dst = reinterpret_cast<uint4*>(sB);
        const uint32_t n16 = (3 * p.hb) >> 4;
        for (uint32_t i = threadIdx.x; i < n16; i += kThreads) dst[i] = __ldg(src + i);
    }
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    tc::cluster_sync();   // barriers of both CTAs initialised, B halves in place
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const int my_tiles = (cid < p.ntiles) ? (p.ntiles - 1 - cid) / ncl + 1 : 0;
    const uint32_t acc1 = p.nbuf == 2 ? 128u : 256u;   // the second accumulator's column

    if (warp < kEpiWarps) {
        // ------------------------------------------------------------ epilogue
        // quarter warp % 4 of the rows; half warp / 4: column blocks of 32 of its parity
        const int quarter = warp & 3, half = warp >> 2, lr = quarter * 32 + lane;
        for (int i = 0; i < my_tiles; ++i) {
            const int b = p.nbuf == 2 ? i & 1 : 0;
            const uint32_t par = (uint32_t)(p.nbuf == 2 ? i >> 1 : i) & 1u;
            if (!warp_wait(tfull + b, par, abort)) break;
            tc::fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + 256u * (uint32_t)b;
            float sum[4] = {0.f, 0.f, 0.f, 0.f}, s1[2] = {0.f, 0.f}, mx = 0.f;
            for (int col = 32 * half; col < p.npad; col += 64) {
                uint32_t v0[32], v1[32];
                tc::tmem_ld_32x32b_x32(taddr + (uint32_t)col, v0);
                tc::tmem_ld_32x32b_x32(taddr + acc1 + (uint32_t)col, v1);
                tc::tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 32; e += 4) {   // (four squares at a time: fewer roundings into the running sums)
                    float q = 0.f;
#pragma unroll
                    for (int k = e; k < e + 4; ++k) {
                        const float a1 = __uint_as_float(v1[k]), a = __uint_as_float(v0[k]) + a1, y = a * ts[col + k];
                        q = k == e ? y * y : fmaf(y, y, q);
                        mx = fmaxf(mx, fabsf(a));
                        s1[k & 1] = fmaf(a1, a1, s1[k & 1]);
                    }
                    sum[(e >> 2) & 3] += q;
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) {
                if (rank == 0) tc::mbar_arrive(tempty + b);
                else tc::mbar_arrive_cluster(tempty + b, 0);
            }
            float tot = sum[0], low = 0.f;   // the last sums with compensation: one rounding, not three
#pragma unroll
            for (int k = 1; k < 4; ++k) comp_add(tot, low, sum[k]);
            if (half == 1) tot += low;
            // outside the split's range: NaN, which no sum within it is (2^-10; 2^-110 unless all zero)
            if (!((s1[0] + s1[1]) * weigh[half] <= 9.765625e-4f * tot && mx < 16777216.f &&
                  (tot >= fmaxf(need[half], 7.703719778e-34f) || mx == 0.f)))
                tot = __uint_as_float(0x7FC00000u);
            // The second half's sum goes to the first through shared memory.
            // Four cells a row: the second half is at most two tiles ahead (the
            // MMAs of a tile wait for both halves of the one two before).
            float* const cell = xchg + (i & 3) * kRows + lr;
            uint64_t* const xbar = xfull + 4 * quarter + (i & 3);
            if (half == 1) {
                *cell = tot;
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(xbar);
            } else {
                if (!warp_wait(xbar, (uint32_t)(i >> 2) & 1u, abort)) break;
                comp_add(tot, low, *cell);
                tot += low;   // (NaN where a sum was not finite)
                const int64_t row = ((int64_t)cid + (int64_t)i * ncl) * (2 * kRows) + rank * kRows + lr;
                if (row < p.n) {
                    if (tot <= 3.402823466e38f) p.x[row] = (p.beta != 0.f) ? fmaf(p.alpha, tot, p.beta * p.x[row]) : p.alpha * tot;
                    else p.list[atomicAdd(p.count, 1)] = (int)row;
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------ MMA issue (even CTA)
        // the whole warp goes along, one elected lane issues (uniform descriptors)
        if (rank == 0) {
            const uint64_t da0 = tc::desc_sw64_kmajor(tc::smem_u32(smem)), db0 = tc::desc_sw64_kmajor(tc::smem_u32(sB));
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int i = 0; i < my_tiles && ok; ++i) {
                const int b = p.nbuf == 2 ? i & 1 : 0;
                const uint32_t par = (uint32_t)(p.nbuf == 2 ? i >> 1 : i) & 1u;
                ok = __all_sync(0xffffffffu, tc::mbar_wait_cluster(tempty + b, par ^ 1u, abort));
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t d0 = tmem + 256u * (uint32_t)b;
#pragma unroll
                for (int q = 0; q < kMaxQ; ++q) {
                    if (q >= p.nq) break;
                    ok = __all_sync(0xffffffffu, tc::mbar_wait_cluster(full + s, ph, abort));
                    if (!ok) break;
                    tc::fence_after_sync();
                    if (tc::elect_one()) {
                        const uint32_t idesc = tc::idesc_bf16_f32(2 * kRows, p.nn[q]);
                        const uint32_t t0 = d0 + p.n0[q], t1 = t0 + acc1;
                        const uint64_t as = da0 + ((uint32_t)s * kStage >> 4), bs = db0 + (p.hoff[q] >> 4);
                        constexpr int kPA[6] = {0, 0, 1, 0, 2, 1}, kPB[6] = {0, 1, 0, 2, 0, 1};
#pragma unroll
                        for (int kk = 0; kk < kKC / 16; ++kk)
#pragma unroll
                            for (int z = 0; z < 6; ++z)
                                tc::mma_bf16_pair(z ? t1 : t0, as + ((kPA[z] * kSlice + 32u * kk) >> 4),
                                                  bs + ((kPB[z] * p.hb + 32u * kk) >> 4), idesc,
                                                  z < 2 ? (q | kk) != 0 : 1);
                        tc::mma_commit_pair(empty + s);
                        if (q + 1 == p.nq) tc::mma_commit_pair(tfull + b);
                    }
                    __syncwarp();
                    if (++s == S) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (tc::elect_one()) tc::mma_commit_pair(fin);
            __syncwarp();
        }
        if (lane == 0) {
            // both CTAs: the last multicast commit has landed here, so no
            // arrival is still on its way when the CTA leaves
            volatile int never = 0;
            tc::mbar_wait(fin, 0, &never);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ converters
        // piece pc: part pc % kParts of chunk g = pc / kParts = (tile g / nq, K-chunk g % nq);
        // the uses of each stage are claimed in piece order (stored[s])
        constexpr int kQuads = Piece<kEarly>::kQuads, kParts = Piece<kEarly>::kParts;
        const int total = my_tiles * p.nq * kParts;
        float4 v[kQuads];
        const auto load = [&](int pc) {
            const int g = pc / kParts, t = g / p.nq, q = g - t * p.nq;
            load_piece<VEC, kQuads>(p, ((int64_t)cid + (int64_t)t * ncl) * (2 * kRows) + rank * kRows + (pc % kParts) * 4 * kQuads,
                                    q, lane, v);
        };
        if (kEarly && warp - kConv0 < total) load(warp - kConv0);
        for (int pc = warp - kConv0; pc < total; pc += kConvWarps) {
            const int g = pc / kParts, q = g % p.nq, u = g / S, s = g - u * S;
            const float4 sc = *reinterpret_cast<const float4*>(ss + kKC * q + 4 * (lane & 7));
            uint2 early[kEarly ? kQuads : 1][3];
            if constexpr (kEarly) {
#pragma unroll
                for (int i = 0; i < kQuads; ++i) split_quad(sc, v[i], early[i]);
                if (pc + kConvWarps < total) load(pc + kConvWarps);
            } else {
                load(pc);
            }
            int ok = 1;
            if (lane == 0)
                ok = tc::counter_wait(reinterpret_cast<volatile int*>(stored + s), kParts * u, abort) &&
                     tc::mbar_wait(empty + s, ((uint32_t)u & 1u) ^ 1u, abort);
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            store_piece<kQuads>(smem + (size_t)s * kStage, pc % kParts, lane, [&](int i, uint2 (&w)[3]) {
                if constexpr (kEarly) {
#pragma unroll
                    for (int z = 0; z < 3; ++z) w[z] = early[i][z];
                } else {
                    split_quad(sc, v[i], w);
                }
            });
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                if (rank == 0) tc::mbar_arrive(full + s);
                else tc::mbar_arrive_cluster(full + s, 0);
                atomicAdd(stored + s, 1);
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::cluster_sync();   // no CTA leaves while its peer may still arrive on its barriers
    if (warp == kMmaWarp) {
        tc::fence_after_sync();
        tc::tmem_dealloc_pair(tmem, 512u);
    }
    if (threadIdx.x == 0 && *abort) set_flag(p.flag, LSK_FLAG_TIMEOUT);
}

// Columns c0 .. c0 + c of B in one pass; false if B's image leaves no ring.
bool pass_plan(int64_t d, int64_t c, int upper_tri, Rn3Params& p) {
    p.d = (int)d;
    p.c = (int)c;
    p.nq = (int)((d + kKC - 1) / kKC);
    p.npad = (int)((c + 31) / 32) * 32;
    p.nbuf = p.npad <= 128 ? 2 : 1;
    uint32_t off = 0;
    for (int q = 0; q < kMaxQ; ++q) {
        p.n0[q] = (upper_tri && q < p.nq) ? (uint32_t)(kKC * q) : 0u;
        p.nn[q] = q < p.nq ? (uint32_t)p.npad - p.n0[q] : 0u;
        p.hoff[q] = off;
        off += (p.nn[q] / 2) * (kKC * 2);
    }
    p.hb = off;
    const int64_t room = (int64_t)kSmemLimit - (int64_t)kExtra - 3 * (int64_t)p.hb;
    p.stages = (int)std::min<int64_t>(kMaxStages, room / (int64_t)kStage);
    return p.stages >= kMinStages;
}
size_t smem_of(const Rn3Params& p) { return (size_t)p.stages * kStage + 3 * (size_t)p.hb + kExtra; }

// passes over A (0: not this kernel) and the columns of each
int passes_of(const lsk_mat* A, int64_t c, int upper_tri, double beta, int64_t* per) {
    if (A->kind != LSK_DENSE || A->d < 1 || A->d > 256 || c < 1 || c > 256) return 0;
    // below this the CUDA-core kernel's one launch is shorter than the scales,
    // the image and the ring's set-up (at 2^30: 40 against 50 us at 65,537 x 128 x
    // 128 triangular, 50 against 62 at 262,145 x 64 x 64, 60 against 77 at 17,000 x
    // 256 x 256)
    if (A->n * A->d * c < (int64_t)1 << 30) return 0;
    Rn3Params p{};
    *per = c;
    if (pass_plan(A->d, c, upper_tri, p)) return 1;
    // a wide general B goes in two halves; the second adds to x, which a listed
    // row's recomputation could not take back
    if (upper_tri || beta != 0.0) return 0;
    *per = (c / 2 + 31) / 32 * 32;
    return pass_plan(A->d, *per, 0, p) ? 2 : 0;
}

size_t image_bytes(const lsk_mat* A, int64_t c, int upper_tri) {
    Rn3Params p{};
    pass_plan(A->d, c, upper_tri, p);
    return ws_round(6 * (size_t)p.hb);
}

using Rn3Kernel = void (*)(const Rn3Params);
Rn3Kernel kernel_of(bool vec, int stages) {
    if (!vec) return rownorm_tc3_kernel<false, false>;
    return stages <= kEarlyStages ? rownorm_tc3_kernel<true, true> : rownorm_tc3_kernel<true, false>;
}
// clusters that fit on the device at once (cached per device, kernel and size)
int pair_clusters(Rn3Kernel kernel, size_t smem) {
    static std::mutex mu;
    static std::map<std::tuple<int, const void*, size_t>, int> cache;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    const void* fn = (const void*)kernel;
    const auto key = std::make_tuple(dev, fn, smem);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    int n = 0;
    if (allow_dynamic_smem(fn) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2, 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) n = 0;
    }
    cudaGetLastError();
    cache[key] = n;
    return n;
}

}  // namespace

size_t rownorms_tc3_workspace_bytes(const lsk_mat* A, int64_t c, int upper_tri) {
    int64_t per = 0;
    const int np = passes_of(A, c, upper_tri, 0.0, &per);
    if (!np) return 0;
    return image_bytes(A, per, upper_tri) + 5 * ws_round(256 * 4) + ws_round((size_t)np * A->n * 4) + ws_round(4);
}

// False: not this kernel's shape.  True: launched (*e its status); rows
// list[0 .. *count) of x, or all of them where *count < 0, are then left to the
// caller.
bool rownorms_tc3_launch(const lsk_mat* A, const float* B, int64_t c, float alpha, float beta, int upper_tri, float* x,
                         void* ws, int* flag, cudaStream_t st, const int** list, const int** count, cudaError_t* e) {
    int64_t per = 0;
    const int np = passes_of(A, c, upper_tri, beta, &per);
    if (!np) return false;
    const bool vec = (A->d % 4 == 0) && (A->ld % 4 == 0) && (((uintptr_t)A->values & 15) == 0);
    WsCarver wc{(char*)ws, 0};
    uint8_t* img = wc.take<uint8_t>(image_bytes(A, per, upper_tri));
    float* sample = wc.take<float>(256);
    float* s = wc.take<float>(256);
    float* t = wc.take<float>(256);
    float* norm = wc.take<float>(256);
    float* rest = wc.take<float>(256);
    int* rows = wc.take<int>((size_t)np * A->n);
    int* cnt = wc.take<int>(1);
    LSK_PROF("rownorm_tc_prep", st) launch_pdl(rn3_units_kernel, 8, kUnitWarps * 32, 0, 1, st, (const float*)A->values, A->ld, A->n,
                                             (int)A->d, sample, cnt);
    for (int k = 0; k < np; ++k) {
        Rn3Params p{};
        const int64_t c0 = k * per, ck = std::min<int64_t>(per, c - c0);
        if (!pass_plan(A->d, ck, upper_tri, p)) {
            *e = cudaErrorNotSupported;
            return true;
        }
        p.A = (const float*)A->values;
        p.lda = A->ld;
        p.n = A->n;
        p.x = x;
        p.alpha = alpha;
        p.beta = k ? 1.f : beta;
        p.ntiles = (int)((A->n + 2 * kRows - 1) / (2 * kRows));
        p.img = img;
        p.s = s;
        p.t = t;
        p.norm = norm;
        p.rest = rest;
        p.list = rows;
        p.count = cnt;
        p.flag = flag;
        const size_t smem = smem_of(p);
        const Rn3Kernel kernel = kernel_of(vec, p.stages);
        const int ncl = std::min(p.ntiles, pair_clusters(kernel, smem));
        if (ncl <= 0) {
            if (k == 0) return false;
            *e = cudaErrorNotSupported;
            return true;
        }
        LSK_PROF("rownorm_tc_prep", st) launch_pdl(rn3_image_kernel, p.npad / 8, 256, 0, 1, st, B, (int)c, (int)c0, p, sample, s, img, t, norm, rest);
        LSK_PROF("rownorm_dense_tc3", st) launch_pdl(kernel, 2 * ncl, kThreads, smem, 1, st, p);
    }
    *list = rows;
    *count = cnt;
    *e = cudaGetLastError();
    return true;
}
