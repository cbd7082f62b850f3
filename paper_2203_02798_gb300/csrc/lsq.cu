// lsq.cu -- sketch-and-precondition least squares (Alg. 12).
//
// Alg. 12 leaves the "parallel preconditioned iterative method" open; the
// reading used here is a preconditioned Krylov solve with N = R^-1 from the
// sketch, wrapped in FP64 iterative refinement:
//     r_t = b - A x_t   (FP64, A's FP32 values taken exactly)
//     g_t = N^T A^T r_t (FP64, from the same pass)
//     eta_t = ||A^T r_t|| / ||A^T b||          stop when eta_t <= tol
//     z = CG(N^T A^T A N, g_t) to inner_tol;  x_{t+1} = x_t + N z   (FP64)
// The inner solve is conjugate gradients on the preconditioned normal
// equations (CGLS, Hestenes & Stiefel 1952), mathematically the same Krylov
// iterates as LSQR on min ||A N y - r_t||, but with the right-hand side g_t
// formed in FP64: its FP32 products are then relative to the correction
// being sought, not to r_t, so a refinement step gains ~inner_tol even when
// the residual is large (LSQR's FP32 vectors carry r_t and stall at about
// eps32 sqrt(n) there).  Each CG iteration makes ONE pass over A: the block
// that forms u_i = A_i p immediately adds u_i A_i^T into its partial of A^T u
// while the row is still in registers.  The FP64 residual pass likewise forms
// r_i and accumulates r_i A_i^T in the same read.  Scalars live on the
// device; the host reads them back every few iterations for the stop test.
#include "lsk_internal.cuh"

#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <new>
#include <string.h>
#include <utility>

namespace cg = cooperative_groups;

namespace {

struct CgState {
    double atb_norm, eta;
    double rho, rho0;   // ||s||^2 now and at the start of the inner solve
    int done, it;
    int pe;             // p holds 2^-pe N p_cg
};

constexpr int kPassThreads = 256;

// The passes and the vector step of the inner solve alternate some 130 times, so
// each is launched programmatically: the next one's blocks start (and load what
// no kernel of the solve writes) while it finishes; everything the previous
// kernel writes is read after pdl_wait, with __ldcg (a load the compiler may not
// take for one of constant memory and move ahead of the wait).

// ---- FP32 pairs: x = h + l carries ~48 bits at the FP32 rate (FP64 runs at
// 1/64 of it here).  Products by FMA, sums by Knuth's TwoSum; a dot product
// kept this way is the "Dot2" of Ogita, Rump & Oishi (SIAM J. Sci. Comput. 26,
// 2005): as accurate as one computed in twice the working precision.
__device__ __forceinline__ float2 to_pair(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}
// (h, l) += a * (xh + xl)
__device__ __forceinline__ void pair_fma(float& h, float& l, float a, float xh, float xl) {
    const float p = a * xh;
    const float e = fmaf(a, xl, fmaf(a, xh, -p));
    const float s = h + p;
    const float t = s - h;
    l += ((h - (s - t)) + (p - t)) + e;
    h = s;
}
// (h, l) += (h2, l2)
__device__ __forceinline__ void pair_add(float& h, float& l, float h2, float l2) {
    const float s = h + h2;
    const float t = s - h;
    l += ((h - (s - t)) + (h2 - t)) + l2;
    h = s;
}

// (double)a by integer instructions: the conversion instruction issues on the FP64
// pipe, which the residual passes keep full with their products.
__device__ __forceinline__ double to_double(float a) {
    const uint32_t mag = __float_as_uint(a) & 0x7fffffffu;
    const bool small = mag < 0x00800000u;                                  // zero or subnormal: scaled up first
    const uint32_t bits = __float_as_uint(small ? a * 16777216.f : a);     // 2^24
    const uint32_t bias = mag >= 0x7f800000u ? 0x70000000u : small ? (896u - 24u) << 20 : 896u << 20;
    const uint32_t hi = (((uint32_t)((int32_t)bits >> 3)) & 0x8fffffffu) + (mag ? bias : 0u);
    return __hiloint2double((int)hi, (int)(bits << 29));
}

// Sum each of RB per-lane values over groups of L lanes: at every step a lane
// keeps half of its values and hands over the other half, so the RB sums cost
// about RB + 3 exchanges instead of 5 RB.  On return the sum of value r is in
// the lanes of the group whose bit log2(L) - 1 - b is bit b of r (sum_lane,
// sum_index).
template <int RB, int L>
__device__ __forceinline__ int sum_lane(int r) {
    int l = 0;
#pragma unroll
    for (int b = 0; (1 << b) < RB; ++b) l |= ((r >> b) & 1) * (L >> (b + 1));
    return l;
}
template <int RB, int L>
__device__ __forceinline__ int sum_index(int lane) {
    int r = 0;
#pragma unroll
    for (int b = 0; (1 << b) < RB; ++b) r |= (lane & (L >> (b + 1))) ? 1 << b : 0;
    return r;
}
template <int RB, int L, class T>
__device__ __forceinline__ T warp_sum_rows(T (&v)[RB], int lane) {
    int o = L / 2;
#pragma unroll
    for (int m = RB; m > 1; m >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int r = 0; r < m / 2; ++r) {   // even values stay in the lower lanes
            const T keep = up ? v[2 * r + 1] : v[2 * r];
            const T give = up ? v[2 * r] : v[2 * r + 1];
            v[r] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    T t = v[0];
    for (; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}
// ---- dense passes, d <= 256 --------------------------------------------------
// A warp takes RB x (32 / L) rows at a time: L lanes own a row, each E entries
// of it -- kVec: E / 4 runs of four columns (16-byte loads; d, lda multiples
// of 4, A 16-byte aligned), else columns L apart -- and the next rows' loads
// are in flight while it computes.
template <int L, int E, int RB, bool kVec>
struct DenseRows {
    static constexpr int kRpl = 32 / L;            // rows a load instruction covers
    static constexpr int kRows = RB * kRpl;        // rows a warp takes at a time
    float a[RB][E];
    static __device__ __forceinline__ int col(int li, int e) { return kVec ? 4 * (li + L * (e / 4)) + e % 4 : li + L * e; }
    __device__ __forceinline__ void load(const float* __restrict__ A, int64_t lda, int64_t n, int d, int64_t i0, int lane) {
        const int sub = lane / L, li = lane % L;
        const float* row = A + (i0 + sub) * lda;
        const int64_t rs = (int64_t)kRpl * lda;
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const bool in = i0 + r * kRpl + sub < n;
            if constexpr (kVec) {
#pragma unroll
                for (int v = 0; v < E / 4; ++v) {
                    const int c = 4 * (li + L * v);
                    const float4 t = (in && c < d) ? __ldg(reinterpret_cast<const float4*>(row + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    a[r][4 * v] = t.x;
                    a[r][4 * v + 1] = t.y;
                    a[r][4 * v + 2] = t.z;
                    a[r][4 * v + 3] = t.w;
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int c = li + L * e;
                    a[r][e] = (in && c < d) ? __ldg(row + c) : 0.f;
                }
            }
            row += rs;
        }
    }
    __device__ __forceinline__ void take(const DenseRows& o) {
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int e = 0; e < E; ++e) a[r][e] = o.a[r][e];
    }
};

// r = b - A x and partial sums of A^T r in one read of A, in FP64 (x == nullptr:
// r = b).  Two FMAs an entry at 2 lanes a cycle and SM bound it: 140 us for
// 316,227 x 128, and half of that for the first pass, whose x is zero; the three
// passes of a solve take 390.  With a conversion instruction an entry on the same
// pipe a pass took 471; FP32 pairs took 57 but hold 48 bits, and FP32's range.
template <int L, int E, int RB, bool kVec>
__global__ void __launch_bounds__(kPassThreads, 2) resid_dense_rows_kernel(
    const float* __restrict__ A, int64_t lda, int64_t n, int d, const double* __restrict__ b,
    const double* __restrict__ x, double* __restrict__ qpart) {
    using Rows = DenseRows<L, E, RB, kVec>;
    __shared__ double qs[(kPassThreads / 32) * Rows::kRpl][L * E];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane / L, li = lane % L;
    double xr[E], q[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int j = Rows::col(li, e);
        xr[e] = x && j < d ? x[j] : 0.0;
        q[e] = 0.0;
    }
    const int mine = sum_index<RB, L>(lane) * Rows::kRpl + sub;   // the row whose sum this lane receives
    const int64_t step = (int64_t)gridDim.x * (kPassThreads / 32) * Rows::kRows;
    int64_t i0 = ((int64_t)blockIdx.x * (kPassThreads / 32) + w) * Rows::kRows;
    Rows cur, nxt;
    double bn = 0.0;
    if (i0 < n) {
        cur.load(A, lda, n, d, i0, lane);
        if (i0 + mine < n) bn = b[i0 + mine];
    }
    for (; i0 < n; i0 += step) {
        double ri = bn;   // rows past n: zero
        if (i0 + step < n) {
            nxt.load(A, lda, n, d, i0 + step, lane);
            bn = i0 + step + mine < n ? b[i0 + step + mine] : 0.0;
        }
        if (x) {
            double dot[RB];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                dot[r] = 0.0;
#pragma unroll
                for (int e = 0; e < E; ++e) dot[r] = fma(to_double(cur.a[r][e]), xr[e], dot[r]);
            }
            ri -= warp_sum_rows<RB, L>(dot, lane);
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const double rr = __shfl_sync(0xffffffffu, ri, sub * L + sum_lane<RB, L>(r));
#pragma unroll
            for (int e = 0; e < E; ++e) q[e] = fma(to_double(cur.a[r][e]), rr, q[e]);
        }
        cur.take(nxt);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) qs[w * Rows::kRpl + sub][Rows::col(li, e)] = q[e];
    __syncthreads();
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        double t = 0.0;
        for (int z = 0; z < (kPassThreads / 32) * Rows::kRpl; ++z) t += qs[z][j];
        qpart[(int64_t)blockIdx.x * d + j] = t;
    }
}

// u = A p: partial sums of u^2 (pairs) and of A^T u; u is used while its rows
// are in registers and not kept.  Passes alternate their direction (rev): where
// A is larger than L2, the rows one pass reads last are still there for the
// next (119 us a pass against 153 at 900,000 x 256, 25 against 30 at 316,227 x
// 128; 40 us there with one row group in flight and u read and written).
template <int L, int E, int RB, bool kVec>
__global__ void __launch_bounds__(kPassThreads, 2) cg_pass_dense_rows_kernel(
    const float* __restrict__ A, int64_t lda, int64_t n, int d, const float* __restrict__ p,
    const CgState* __restrict__ st, int rev, float* __restrict__ qpart, double* __restrict__ sspart) {
    using Rows = DenseRows<L, E, RB, kVec>;
    __shared__ float qs[(kPassThreads / 32) * Rows::kRpl][L * E];
    __shared__ double ssw[kPassThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane / L, li = lane % L;
    const int64_t groups = (n + Rows::kRows - 1) / Rows::kRows, step = (int64_t)gridDim.x * (kPassThreads / 32);
    int64_t g = (int64_t)blockIdx.x * (kPassThreads / 32) + w;
    Rows cur, nxt;
    if (g < groups) cur.load(A, lda, n, d, (rev ? groups - 1 - g : g) * Rows::kRows, lane);
    pdl_wait();
    pdl_launch_next();
    if (__ldcg(&st->done)) return;
    float pr[E], q[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int j = Rows::col(li, e);
        pr[e] = j < d ? __ldcg(p + j) : 0.f;
        q[e] = 0.f;
    }
    float sh = 0.f, sl = 0.f;
    for (; g < groups; g += step) {
        const int64_t gn = g + step;
        if (gn < groups) nxt.load(A, lda, n, d, (rev ? groups - 1 - gn : gn) * Rows::kRows, lane);
        float dot[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            dot[r] = 0.f;
#pragma unroll
            for (int e = 0; e < E; ++e) dot[r] = fmaf(cur.a[r][e], pr[e], dot[r]);
        }
        const float u = warp_sum_rows<RB, L>(dot, lane);   // rows past n are zero
        pair_fma(sh, sl, u, u, 0.f);
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            const float ui = __shfl_sync(0xffffffffu, u, sub * L + sum_lane<RB, L>(r));
#pragma unroll
            for (int e = 0; e < E; ++e) q[e] = fmaf(cur.a[r][e], ui, q[e]);
        }
        cur.take(nxt);
    }
#pragma unroll
    for (int e = 0; e < E; ++e) qs[w * Rows::kRpl + sub][Rows::col(li, e)] = q[e];
    // each row's u is in L / RB lanes: one of them counts
    const double ss = warp_sum((lane & (L / RB - 1)) == 0 ? (double)sh + (double)sl : 0.0);
    if (lane == 0) ssw[w] = ss;
    __syncthreads();
    for (int j = threadIdx.x; j < d; j += blockDim.x) {
        float t = 0.f;
        for (int z = 0; z < (kPassThreads / 32) * Rows::kRpl; ++z) t += qs[z][j];
        qpart[(int64_t)blockIdx.x * d + j] = t;
    }
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int z = 0; z < kPassThreads / 32; ++z) t += ssw[z];
        sspart[blockIdx.x] = t;
    }
}

// ---- CSR: both products of a pass without atomics ---------------------------
// A solve makes some 60 passes over the same matrix, so its rows are cut into
// tiles of `rows_per` rows once and each tile's entries also stored sorted by
// column (local row, value).  A pass then forms u = A p on a tile from the CSR
// entries (segments: rows) and A^T u from the sorted ones (segments:
// columns; the CSR arrays were checked by the sketch): in both, the block multiplies a
// coalesced run of entries by the
// vector's values in shared memory and sums the segments from there.  With
// one thread per row and shared-memory float atomics (compare-and-swap loops)
// for A^T u, a pass took 35 us at 500,000 x 256 and 2.6 M entries; this takes 15,
// and building the tiles 45 once.
constexpr int kTileRowsMax = 4096;
constexpr int kTilesPerSm = 3;
// Entries are taken six quads a thread at a time (16-byte loads, all in flight
// before any product), 6,144 to a run: what 80 registers a thread, and with them
// three blocks an SM, leave room for.  A tile with more takes its entries run by run,
// each of them another round of loads and barriers: at 500,000 x 256 (456 tiles, one
// wave) a pass takes 14.8 us with 2,200 entries a tile, 18.4 with 5,500, 21.7 with
// 6,800 (two runs), 26.0 with 11,500 and 34.1 with 13,200 (three).
constexpr int kQuads = 6;
constexpr int kTileEntries = kQuads * 4 * kPassThreads;

struct CsrTiles {
    int64_t n, d, ntiles;
    int rows_per;
    const float* V;
    const int32_t* J;
    const int64_t* I;
    int32_t* cptr;     // ntiles x (d + 1): column offsets inside each tile
    float* tval;       // nnz
    uint16_t* trow;    // nnz
};

__global__ void __launch_bounds__(kPassThreads) csr_tiles_kernel(CsrTiles t, int64_t nnz) {
    extern __shared__ int cnt[];                     // d
    __shared__ uint16_t rid[kTileEntries];           // row of each entry of the run in hand
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t r0 = (int64_t)blockIdx.x * t.rows_per;
    const int rows = (int)min((int64_t)t.rows_per, t.n - r0);
    const int d = (int)t.d;
    for (int j = threadIdx.x; j < d; j += blockDim.x) cnt[j] = 0;
    __syncthreads();
    const int64_t base = t.I[r0], end = min(t.I[r0 + rows], nnz);
#pragma unroll 8
    for (int64_t e = base + threadIdx.x; e < end; e += kPassThreads)
        atomicAdd(&cnt[min((uint32_t)__ldg(t.J + e), (uint32_t)(d - 1))], 1);
    __syncthreads();
    if (w == 0) {   // exclusive scan
        int32_t* out = t.cptr + (int64_t)blockIdx.x * (d + 1);
        int run = 0;
        for (int j0 = 0; j0 < d; j0 += 32) {
            const int j = j0 + lane;
            const int v = j < d ? cnt[j] : 0;
            int s = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int up = __shfl_up_sync(0xffffffffu, s, o);
                if (lane >= o) s += up;
            }
            if (j < d) {
                cnt[j] = run + s - v;
                out[j] = run + s - v;
            }
            run += __shfl_sync(0xffffffffu, s, 31);
        }
        if (lane == 0) out[d] = run;
    }
    for (int64_t c0 = base; c0 < end; c0 += kTileEntries) {
        const int m = (int)min((int64_t)kTileEntries, end - c0);
        __syncthreads();
        for (int r = threadIdx.x; r < rows; r += kPassThreads) {
            const int k0 = (int)max(t.I[r0 + r] - c0, (int64_t)0), k1 = (int)min(t.I[r0 + r + 1] - c0, (int64_t)m);
            for (int k = k0; k < k1; ++k) rid[k] = (uint16_t)r;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = threadIdx.x; k < m; k += kPassThreads) {
            const float v = __ldg(t.V + c0 + k);
            const int pos = atomicAdd(&cnt[min((uint32_t)__ldg(t.J + c0 + k), (uint32_t)(d - 1))], 1);
            t.tval[base + pos] = v;
            t.trow[base + pos] = rid[k];
        }
    }
}

// out[s] += sum over the entries e of segment s of val[e] vec[idx[e]], for the
// segments [ptr[s], ptr[s + 1]) of a run of entries.  The run starts at a
// multiple of four (`shift` entries before the first segment); 2^lg lanes a
// segment.  Sums are float, or double in the residual pass.
__device__ __forceinline__ float seg_mul(float v, float x) { return v * x; }
__device__ __forceinline__ double seg_mul(float v, double x) { return to_double(v) * x; }

__device__ __forceinline__ int4 idx_quad(const int32_t* p) { return __ldg(reinterpret_cast<const int4*>(p)); }
__device__ __forceinline__ int4 idx_quad(const uint16_t* p) {
    const ushort4 t = __ldg(reinterpret_cast<const ushort4*>(p));
    return make_int4(t.x, t.y, t.z, t.w);
}

struct EntryQuads {
    float4 v[kQuads];
    int4 j[kQuads];
};

// Entries [e0, e0 + 6144) of the run, e0 a multiple of four, up to `end` of
// the arrays (vec4: both are 16-byte aligned; the last quad may be ragged).
template <class Idx>
__device__ __forceinline__ void load_quads(EntryQuads& r, const float* __restrict__ val, const Idx* __restrict__ idx,
                                           int64_t e0, int64_t end, bool vec4) {
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
        const int64_t e = e0 + 4 * (threadIdx.x + q * kPassThreads);
        r.v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        r.j[q] = make_int4(0, 0, 0, 0);
        if (vec4 && e + 4 <= end) {
            r.v[q] = __ldg(reinterpret_cast<const float4*>(val + e));
            r.j[q] = idx_quad(idx + e);
        } else if (e < end) {
            r.v[q].x = val[e];
            r.j[q].x = idx[e];
            if (e + 1 < end) r.v[q].y = val[e + 1], r.j[q].y = idx[e + 1];
            if (e + 2 < end) r.v[q].z = val[e + 2], r.j[q].z = idx[e + 2];
            if (e + 3 < end) r.v[q].w = val[e + 3], r.j[q].w = idx[e + 3];
        }
    }
}

template <class T>
__device__ __forceinline__ void mul_quads(const EntryQuads& r, const T* vec, int nvec, T* prod, int m) {
    const uint32_t top = (uint32_t)(nvec - 1);
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
        const int e = 4 * (threadIdx.x + q * kPassThreads);
        if (e >= m) continue;
        const T a = seg_mul(r.v[q].x, vec[min((uint32_t)r.j[q].x, top)]), b = seg_mul(r.v[q].y, vec[min((uint32_t)r.j[q].y, top)]);
        const T c = seg_mul(r.v[q].z, vec[min((uint32_t)r.j[q].z, top)]), f = seg_mul(r.v[q].w, vec[min((uint32_t)r.j[q].w, top)]);
        if constexpr (sizeof(T) == sizeof(float)) {
            *reinterpret_cast<float4*>(prod + e) = make_float4(a, b, c, f);
        } else {
            *reinterpret_cast<double2*>(prod + e) = make_double2(a, b);
            *reinterpret_cast<double2*>(prod + e + 2) = make_double2(c, f);
        }
    }
}

template <class T>
__device__ __forceinline__ void sum_segments(const T* prod, int c0, int m, int shift, const int32_t* ptr, int nseg,
                                             int lg, T* out) {
    const int G = 1 << lg, sub = threadIdx.x & (G - 1);
    for (int s0 = 0; s0 < nseg; s0 += kPassThreads >> lg) {
        const int s = s0 + (threadIdx.x >> lg);
        T t = 0;
        int k0 = 0, k1 = 0;
        if (s < nseg) {
            k0 = max(ptr[s] + shift, c0);
            k1 = min(ptr[s + 1] + shift, c0 + m);
            for (int k = k0 + sub; k < k1; k += G) t += prod[k - c0];
        }
        for (int o = G >> 1; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (k1 > k0 && sub == 0) out[s] += t;
    }
}

__device__ __forceinline__ int seg_lanes(int nseg) {   // log2 of the lanes a segment
    int lg = 0;
    while (lg < 5 && (nseg << (lg + 1)) <= kPassThreads) ++lg;
    return lg;
}

// T = float: u = A p and partial sums of A^T u, ||u||^2.
// T = double: r = b - A x and partial sums of A^T r.
template <class T>
__global__ void __launch_bounds__(kPassThreads, kTilesPerSm) tile_pass_kernel(CsrTiles t, const float* __restrict__ p,
                                                                 const double* __restrict__ x,
                                                                 const double* __restrict__ b,
                                                                 const CgState* __restrict__ st,
                                                                 void* __restrict__ qpart, double* __restrict__ sspart) {
    constexpr bool kResid = sizeof(T) == sizeof(double);
    extern __shared__ __align__(16) unsigned char tile_sh[];
    __shared__ double ssw[kPassThreads / 32];
    const int d = (int)t.d;
    T* prod = reinterpret_cast<T*>(tile_sh);
    T* vec = prod + kTileEntries;            // p or x
    T* q = vec + d;
    T* u = q + d;
    int32_t* rptr = reinterpret_cast<int32_t*>(u + t.rows_per);   // rows_per + 1
    int32_t* cptr = rptr + t.rows_per + 1;                        // d + 1
    // the first run's entries do not depend on the previous kernel
    const bool vec4 = ((reinterpret_cast<uintptr_t>(t.V) | reinterpret_cast<uintptr_t>(t.J)) & 15) == 0;
    EntryQuads r;
    int64_t base = 0, base4 = 0, end = 0;
    if (blockIdx.x < t.ntiles) {
        const int64_t r0 = (int64_t)blockIdx.x * t.rows_per;
        base = t.I[r0];
        end = t.I[min(r0 + t.rows_per, t.n)];
        base4 = base & ~(int64_t)3;
        load_quads(r, t.V, t.J, base4, end, vec4);
    }
    pdl_wait();
    pdl_launch_next();
    if (!kResid && __ldcg(&st->done)) return;
    for (int j = threadIdx.x; j < d; j += kPassThreads) {
        if constexpr (kResid) vec[j] = x[j];
        else vec[j] = __ldcg(p + j);
        q[j] = 0;
    }
    float sh = 0.f, sl = 0.f;
    for (int64_t tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x) {
        const int64_t r0 = tile * t.rows_per;
        const int rows = (int)min((int64_t)t.rows_per, t.n - r0);
        if (tile != blockIdx.x) {
            base = t.I[r0];
            end = t.I[r0 + rows];
            base4 = base & ~(int64_t)3;
            load_quads(r, t.V, t.J, base4, end, vec4);
        }
        const int count = (int)(end - base4), shift = (int)(base - base4);
        __syncthreads();   // the last tile's readers of rptr, cptr, u
        for (int i = threadIdx.x; i <= rows; i += kPassThreads) {
            rptr[i] = (int32_t)(t.I[r0 + i] - base);
            if (i < rows) u[i] = 0;
        }
        for (int j = threadIdx.x; j <= d; j += kPassThreads) cptr[j] = t.cptr[tile * (d + 1) + j];
        __syncthreads();
        const int lgr = seg_lanes(rows), lgd = seg_lanes(d);
        for (int c0 = 0; c0 < count; c0 += kTileEntries) {
            const int m = min(kTileEntries, count - c0);
            if (c0) load_quads(r, t.V, t.J, base4 + c0, end, vec4);
            mul_quads(r, vec, d, prod, m);
            if (c0 + kTileEntries >= count) load_quads(r, t.tval, t.trow, base4, end, true);   // for the next product
            __syncthreads();
            sum_segments(prod, c0, m, shift, rptr, rows, lgr, u);
            __syncthreads();
        }
        for (int i = threadIdx.x; i < rows; i += kPassThreads) {
            if constexpr (kResid) u[i] = b[r0 + i] - u[i];
            else pair_fma(sh, sl, u[i], u[i], 0.f);
        }
        __syncthreads();
        for (int c0 = 0; c0 < count; c0 += kTileEntries) {
            const int m = min(kTileEntries, count - c0);
            if (c0) load_quads(r, t.tval, t.trow, base4 + c0, end, true);
            mul_quads(r, u, rows, prod, m);
            __syncthreads();
            sum_segments(prod, c0, m, shift, cptr, d, lgd, q);
            __syncthreads();
        }
    }
    __syncthreads();
    for (int j = threadIdx.x; j < d; j += kPassThreads) {
        reinterpret_cast<T*>(qpart)[(int64_t)blockIdx.x * d + j] = q[j];
    }
    if constexpr (!kResid) {
        const double ss = warp_sum((double)sh + (double)sl);
        if ((threadIdx.x & 31) == 0) ssw[threadIdx.x >> 5] = ss;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int z = 0; z < kPassThreads / 32; ++z) s += ssw[z];
            sspart[blockIdx.x] = s;
        }
    }
}

// ---- FP64 residual + A^T r, dense, d > 256: warp per row -------------------
__global__ void __launch_bounds__(kPassThreads) resid64_dense_kernel(
    const float* __restrict__ A, int64_t lda, int64_t n, int64_t d, const double* __restrict__ b,
    const double* __restrict__ x, double* __restrict__ qpart) {
    extern __shared__ double sh[];   // x (d) then per-warp q (8 * d)
    double* xs = sh;
    double* qs = sh + d;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t j = threadIdx.x; j < d; j += blockDim.x) xs[j] = x[j];
    for (int64_t j = threadIdx.x; j < 8 * d; j += blockDim.x) qs[j] = 0.0;
    __syncthreads();
    double* qw = qs + w * d;
    const int64_t wid = (int64_t)blockIdx.x * 8 + w, nw = (int64_t)gridDim.x * 8;
    for (int64_t i = wid; i < n; i += nw) {
        const float* row = A + i * lda;
        double dot = 0.0;
        for (int64_t j = lane; j < d; j += 32) dot = fma((double)row[j], xs[j], dot);
        dot = warp_sum(dot);
        const double ri = b[i] - dot;
        for (int64_t j = lane; j < d; j += 32) qw[j] = fma((double)row[j], ri, qw[j]);
    }
    __syncthreads();
    for (int64_t j = threadIdx.x; j < d; j += blockDim.x) {
        double s = 0.0;
        for (int t = 0; t < 8; ++t) s += qs[t * d + j];
        qpart[(int64_t)blockIdx.x * d + j] = s;
    }
}

// ---- FP64 residual + A^T r, CSR: thread per row ----------------------------
__global__ void __launch_bounds__(kPassThreads) resid64_csr_kernel(
    const float* __restrict__ V, const int32_t* __restrict__ J, const int64_t* __restrict__ I,
    int64_t n, int64_t nnz, int64_t d, const double* __restrict__ b, const double* __restrict__ x,
    double* __restrict__ qpart, int* flag) {
    extern __shared__ double sh[];
    double* xs = sh;
    double* qs = sh + d;
    for (int64_t j = threadIdx.x; j < d; j += blockDim.x) {
        xs[j] = x[j];
        qs[j] = 0.0;
    }
    __syncthreads();
    bool bad = false;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t k0 = I[i], k1 = I[i + 1];
        double dot = 0.0;
        const bool ok = !(k0 < 0 || k1 < k0 || k1 > nnz);
        if (!ok) bad = true;
        if (ok)
            for (int64_t p = k0; p < k1; ++p) {
                const int32_t j = J[p];
                if (j >= 0 && j < d) dot = fma((double)V[p], xs[j], dot);
                else bad = true;
            }
        const double ri = b[i] - dot;
        if (ok)
            for (int64_t p = k0; p < k1; ++p) {
                const int32_t j = J[p];
                if (j >= 0 && j < d) atomicAdd(&qs[j], (double)V[p] * ri);
            }
    }
    if (bad) set_flag(flag, LSK_FLAG_BAD_CSR);
    __syncthreads();
    for (int64_t j = threadIdx.x; j < d; j += blockDim.x) qpart[(int64_t)blockIdx.x * d + j] = qs[j];
}

// u = A p: partial sums of u^2 and of A^T u.  Dense, any d: warp per row.
__global__ void __launch_bounds__(kPassThreads) cg_pass_dense_kernel(
    const float* __restrict__ A, int64_t lda, int64_t n, int64_t d, const float* __restrict__ p,
    const CgState* __restrict__ st, float* __restrict__ qpart, double* __restrict__ sspart) {
    extern __shared__ float shf[];   // p (d) then per-warp q (8 * d)
    pdl_wait();
    pdl_launch_next();
    if (__ldcg(&st->done)) return;
    float* ps = shf;
    float* qs = shf + d;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t j = threadIdx.x; j < d; j += blockDim.x) ps[j] = __ldcg(p + j);
    for (int64_t j = threadIdx.x; j < 8 * d; j += blockDim.x) qs[j] = 0.f;
    __syncthreads();
    float* qw = qs + w * d;
    double ss = 0.0;
    const int64_t wid = (int64_t)blockIdx.x * 8 + w, nw = (int64_t)gridDim.x * 8;
    for (int64_t i = wid; i < n; i += nw) {
        const float* row = A + i * lda;
        float dot = 0.f;
        for (int64_t j = lane; j < d; j += 32) dot = fmaf(row[j], ps[j], dot);
        dot = warp_sum(dot);
        const float ui = dot;
        ss = fma((double)ui, (double)ui, ss);
        for (int64_t j = lane; j < d; j += 32) qw[j] = fmaf(row[j], ui, qw[j]);
    }
    __syncthreads();
    for (int64_t j = threadIdx.x; j < d; j += blockDim.x) {
        float s = 0.f;
        for (int t = 0; t < 8; ++t) s += qs[t * d + j];
        qpart[(int64_t)blockIdx.x * d + j] = s;
    }
    __shared__ double ssw[8];
    if (lane == 0) ssw[w] = ss;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int t = 0; t < 8; ++t) s += ssw[t];
        sspart[blockIdx.x] = s;
    }
}

// ---- inner solve: CG on the preconditioned normal equations ----------------
// N^T A^T A N z = g with g = N^T A^T r formed in FP64 by the residual pass.
// The pass kernels form u = A N p_cg, A^T u and ||u||^2 in FP32 / pairs; the
// d-vectors (z, s, p_cg) stay in FP64.  Unlike LSQR on min ||A N y - r||,
// whose FP32 n-vectors carry r itself (mostly orthogonal to range(A) when the
// residual is large), every FP32 quantity here is relative to the correction
// being sought, so each refinement step gains ~inner_tol whatever the size of
// the residual.
//
// The work between two passes -- sum the blocks' partials, w = N^T (A^T u),
// z += a p_cg, s -= a w, p_cg = s + b p_cg, p = N p_cg -- is a chain of two
// d x d products and two dot products.  One block took 84 us for it at d = 128
// (FP64 issues at 2 lanes a cycle per SM, and its reads of N were serial),
// twice the pass itself.  Here a cluster of 16 CTAs (or the largest one that the
// device can place, cg_vec_ctas) runs it in one launch:
// for d <= 256 every warp owns one row of N^T and one of N, as FP32 pairs
// in registers before anything is waited for (with FP64 products each of the
// two took 4,800 of the step's 25,000 cycles at d = 256), one more warp a CTA
// does the scalars, and the two vectors that each step needs whole are
// exchanged through distributed shared memory: 9 us a step.  Where d is more
// than the warps of the cluster, N is read from L2 in FP64.
//
// p is handed to the pass scaled by a power of two that brings ||A p|| near one,
// taken from ||s||: the pass squares u = A p in FP32, and ||u|| follows the scale
// of b and falls by ten orders during a solve, so that without it u^2 left FP32's
// range for b of 1e-13 and less or 1e18 and more.  The scaling is exact and undone
// in the step length.
// kStart: the residual pass's FP64 partials, eta and the start of a solve, three
// or four times in all, with N in FP64.
constexpr int kVecCtas = 16, kVecThreads = 512;   // CTAs at most (2 at least)
constexpr int kVecBlock = kVecThreads + 32;   // one more warp for the scalars

__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }   // |e| < 1023

// the lane's eight entries of a row of N (or N^T) times v, summed over the warp
__device__ __forceinline__ double row_dot(const float2 (&n)[8], const float2* v, int d, int lane, int c_lo, int c_hi) {
    float h = 0.f, l = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c >= c_lo && c <= c_hi) {
            const float2 x = v[min(lane + 32 * c, d - 1)];
            l = fmaf(n[c].y, x.x, l);
            pair_fma(h, l, n[c].x, x.x, x.y);
        }
#pragma unroll
    for (int o = 16; o; o >>= 1) pair_add(h, l, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o));
    return (double)h + (double)l;
}

template <bool kStart>
__global__ void __launch_bounds__(kVecBlock, 1) cg_vec_kernel(const void* __restrict__ part_, const double* __restrict__ sspart,
                                                           int nblocks, int d, const double* __restrict__ N,
                                                           const double* __restrict__ Nt, const float2* __restrict__ N2,
                                                           const float2* __restrict__ Nt2, int first, double inner_tol,
                                                           CgState* st, double* __restrict__ s, double* __restrict__ pc,
                                                           double* __restrict__ z, float* __restrict__ p) {
    using T = typename std::conditional<kStart, double, float>::type;
    const T* part = reinterpret_cast<const T*>(part_);
    // Another CTA's shared memory may be written once that CTA is known to run:
    // every CTA arrives here, the wait before the first such store finds them
    // all there.
    cg::cluster_group cl = cg::this_cluster();
    auto started = cl.barrier_arrive();
    __shared__ double qv[1024], sv[1024], pv[1024];
    __shared__ float2 v2[256];      // the vector being multiplied, as pairs (d <= 256)
    __shared__ T red[kVecThreads];
    __shared__ double gv[kVecCtas]; // the CTAs' shares of ||u||^2
    __shared__ double sc[3];        // step length, beta, the scale of p
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, cta = (int)cl.block_rank(), ctas = (int)gridDim.x;
    const int warps = ctas * (kVecThreads / 32);
    const bool scalar_warp = tid >= kVecThreads, small = N2 != nullptr;   // a row a warp
    const int gw = scalar_warp ? d : w * ctas + cta;   // rows gw, gw + warps, ... of N^T and N
    float2 nt[8], nn[8];
    if (small && gw < d) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int i = lane + 32 * c;
            nt[c] = i <= gw ? __ldg(Nt2 + gw * d + i) : make_float2(0.f, 0.f);
            nn[c] = (i >= gw && i < d) ? __ldg(N2 + gw * d + i) : make_float2(0.f, 0.f);
        }
    }
    pdl_wait();
    pdl_launch_next();
    cl.barrier_wait(std::move(started));
    // everything the pass and the previous step left is loaded at once
    const int done = kStart ? 0 : __ldcg(&st->done);
    const double rho = kStart ? 0.0 : __ldcg(&st->rho);
    const int pe = kStart ? 0 : __ldcg(&st->pe);
    // the partials of this CTA's columns: ng threads a column, then a tree
    const int cpc = (d + ctas - 1) / ctas, j0 = cta * cpc, nc = max(0, min(cpc, d - j0));
    int ng = 1;
    while (2 * ng * cpc <= kVecThreads) ng *= 2;
    const int col = tid % cpc, grp = tid / cpc;
    T acc = 0;
    double zj = 0.0, sj = 0.0, pj = 0.0;   // d <= 256: this warp's entry
    double g = 0.0;
    if (!scalar_warp) {
        if (grp < ng && col < nc) {
            const T* src = part + j0 + col;
            for (int q = grp; q < nblocks; q += 10 * ng) {   // ten loads in flight
                T v[10];
#pragma unroll
                for (int k = 0; k < 10; ++k) v[k] = q + k * ng < nblocks ? __ldcg(src + (int64_t)(q + k * ng) * d) : (T)0;
#pragma unroll
                for (int k = 0; k < 10; ++k) acc += v[k];
            }
        }
        if (!kStart) {
            for (int j = tid; j < d; j += kVecThreads) pv[j] = __ldcg(pc + j);
            if (small && gw < d) {
                zj = __ldcg(z + gw);
                sj = __ldcg(s + gw);
                pj = __ldcg(pc + gw);
            }
        }
        red[tid] = acc;
    } else if (!kStart) {
        for (int q = cta + ctas * lane; q < nblocks; q += ctas * 32) g += __ldcg(sspart + q);
        g = warp_sum(g);
        if (lane < ctas) cl.map_shared_rank(gv, lane)[cta] = g;
    }
    __syncthreads();
    for (int m = ng >> 1; m; m >>= 1) {
        if (grp < m) red[tid] += red[tid + m * cpc];
        __syncthreads();
    }
    for (int e = tid; e < nc * ctas; e += kVecBlock)
        cl.map_shared_rank(qv, e / nc)[j0 + e % nc] = (double)red[e % nc];
    cl.sync();   // qv = A^T u (or A^T r) and gv in every CTA
    if (done) return;   // the same in every CTA: written only after the second cluster barrier
    if (small) {
        if (tid < d) v2[tid] = to_pair(qv[tid]);
        __syncthreads();
    }
    double t = 0.0;
    if (scalar_warp) {
        if (!kStart) {
            double G = lane < ctas ? gv[lane] : 0.0;
            G = warp_sum(G);
            const double m = pow2d(-pe);
            if (lane == 0) sc[0] = G > 0.0 ? rho * m * m / G : 0.0;
        } else if (cta == 0) {   // eta = ||A^T r|| / ||A^T b||
            double a2 = 0.0;
            for (int j = lane; j < d; j += 32) a2 = fma(qv[j], qv[j], a2);
            a2 = warp_sum(a2);
            if (lane == 0) {
                const double atrn = sqrt(a2), atb = first ? atrn : st->atb_norm;
                st->atb_norm = atb;
                st->eta = atb > 0.0 ? atrn / atb : 0.0;
            }
        }
    } else if (small && gw < d) {
        t = row_dot(nt, v2, d, lane, 0, gw >> 5);   // (N^T q)_gw
    }
    __syncthreads();
    const double a = kStart ? 0.0 : sc[0], as = kStart ? 0.0 : a * pow2d(pe);   // as: for the scaled A^T u
    if (!scalar_warp)
        for (int j = gw; j < d; j += warps) {
            if (!small) {
                t = 0.0;
                for (int i = lane; i <= j; i += 32) t = fma(Nt[(int64_t)j * d + i], qv[i], t);
                t = warp_sum(t);
                if (!kStart) {
                    zj = __ldcg(z + j);
                    sj = __ldcg(s + j);
                    pj = pv[j];
                }
            }
            const double snew = kStart ? t : fma(-as, t, sj);
            if (lane == 0) {
                s[j] = snew;
                z[j] = kStart ? 0.0 : fma(a, pj, zj);
            }
            if (lane < ctas) cl.map_shared_rank(sv, lane)[j] = snew;
        }
    cl.sync();   // sv = the new s in every CTA
    if (scalar_warp) {
        double r2 = 0.0;
        for (int j = lane; j < d; j += 32) r2 = fma(sv[j], sv[j], r2);
        r2 = warp_sum(r2);
        if (lane == 0) {
            sc[1] = (!kStart && rho > 0.0) ? r2 / rho : 0.0;
            // 2^e: ||s|| rounded down to a power of two, e half the exponent of ||s||^2
            const int e = ((__double2hiint(r2) >> 20) - 1023) >> 1;   // [-512, 512]
            sc[2] = pow2d(-e);
            if (cta == 0) {
                st->rho = r2;
                st->pe = e;
                if (kStart) {
                    st->rho0 = r2;
                    st->it = 0;
                    st->done = r2 == 0.0 ? 1 : 0;
                } else {
                    st->it += 1;
                    if (a == 0.0 || r2 <= inner_tol * inner_tol * st->rho0) st->done = 1;
                }
            }
        }
    }
    __syncthreads();
    const double bta = sc[1], ps = sc[2];
    for (int j = tid; j < d; j += kVecBlock) {
        const double v = kStart ? sv[j] : fma(bta, pv[j], sv[j]);
        pv[j] = v;
        if (small) v2[j] = to_pair(v * ps);
        if (cta == 0) pc[j] = v;
    }
    __syncthreads();
    if (scalar_warp) return;
    for (int i = gw; i < d; i += warps) {   // p = N p_cg
        if (small) {
            t = row_dot(nn, v2, d, lane, gw >> 5, (d - 1) >> 5);
        } else {
            t = 0.0;
            for (int j = i + lane; j < d; j += 32) t = fma(N[(int64_t)i * d + j], pv[j], t);
            t = warp_sum(t) * ps;
        }
        if (lane == 0) p[i] = (float)t;
    }
}

// N^T, and both as pairs for d <= 256 (converting them in every step would
// cost more FP64-pipe cycles than the products)
__global__ void __launch_bounds__(256) factor_forms_kernel(const double* __restrict__ N, int d, double* __restrict__ Nt,
                                                           float2* __restrict__ N2, float2* __restrict__ Nt2) {
    __shared__ double tile[32][33];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5, i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
    for (int k = y; k < 32; k += 8)
        if (i0 + k < d && j0 + x < d) {
            const double v = N[(int64_t)(i0 + k) * d + j0 + x];
            tile[k][x] = v;
            if (N2) N2[(i0 + k) * d + j0 + x] = to_pair(v);
        }
    __syncthreads();
    for (int k = y; k < 32; k += 8)
        if (j0 + k < d && i0 + x < d) {
            const double v = tile[x][k];
            Nt[(int64_t)(j0 + k) * d + i0 + x] = v;
            if (Nt2) Nt2[(j0 + k) * d + i0 + x] = to_pair(v);
        }
}

// x <- x + N y (FP64), one warp a row.
__global__ void __launch_bounds__(256) update_x_kernel(const double* __restrict__ N64, int64_t d,
                                                       const double* __restrict__ y, double* __restrict__ x) {
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= d) return;
    double s = 0.0;
    for (int64_t j = i + lane; j < d; j += 32) s = fma(N64[i * d + j], y[j], s);
    s = warp_sum(s);
    if (lane == 0) x[i] += s;
}

template <bool kStart>
bool cg_vec_places(int ctas) {
    // more than 8 CTAs a cluster are above the portable size: opt in (idempotent, the same value always)
    if (cudaFuncSetAttribute(cg_vec_kernel<kStart>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas, 1, 1);
    cfg.blockDim = dim3(kVecBlock, 1, 1);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, cg_vec_kernel<kStart>, &cfg) == cudaSuccess && n > 0;
}
// CTAs of the step's cluster: the most that the current device can place (a
// device or a partition of one may have no processing cluster of 16 free SMs).
int cg_vec_ctas() {
    int ctas = kVecCtas;
    while (ctas > 2 && !(cg_vec_places<true>(ctas) && cg_vec_places<false>(ctas))) ctas >>= 1;
    cudaGetLastError();
    return ctas;
}

template <bool kStart>
cudaError_t launch_vec(int ctas, const void* part, const double* sspart, int nblocks, int64_t d, const double* N, const double* Nt,
                       const float2* N2, const float2* Nt2, int first, double inner_tol, CgState* S, double* s, double* pc, double* z, float* p,
                       cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    LSK_PROF("lsq_small", st) e = launch_pdl(cg_vec_kernel<kStart>, ctas, kVecBlock, 0, ctas, st, part, sspart,
                                             nblocks, (int)d, N, Nt, N2, Nt2, first, inner_tol, S, s, pc, z, p);
    return e;
}

constexpr int kMaxPassBlocks = 2432;   // >= 8 x the SM count of any sm_103 part

// Blocks of a pass over A: two per SM of the d <= 256 kernels are resident, and
// fewer blocks leave fewer partials to sum; each covers two row groups or more.
int pass_grid(const lsk_mat* A, int sm_count) {
    const int64_t n = A->n;
    const bool rows_kernel = A->kind == LSK_DENSE && A->d <= 256;
    const int64_t per_block = rows_kernel ? (kPassThreads / 32) * (A->d <= 32 ? 32 : A->d <= 64 ? 16 : 8) * 2 : kPassThreads * 2;
    int64_t g = (n + per_block - 1) / per_block;
    const int64_t cap = std::min<int64_t>(rows_kernel ? 2 * sm_count : 8 * sm_count, kMaxPassBlocks);
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

template <int L, int E, int RB, bool kVec>
void launch_rows_pass(const lsk_mat* A, int nb, const float* p, const CgState* S, int rev, float* qpart,
                      double* sspart, cudaStream_t st) {
    LSK_PROF("lsq_pass", st) launch_pdl(cg_pass_dense_rows_kernel<L, E, RB, kVec>, nb, kPassThreads, 0, 1, st,
                                        (const float*)A->values, A->ld, A->n, (int)A->d, p, S, rev, qpart, sspart);
}

// 16-byte loads of whole rows: d and ld multiples of 4, values 16-byte aligned
bool rows_vec4(const lsk_mat* A) {
    return A->d % 4 == 0 && A->ld % 4 == 0 && (reinterpret_cast<uintptr_t>(A->values) & 15) == 0;
}

void cg_pass_dense(const lsk_mat* A, int nb, const float* p, const CgState* S, int rev, float* qpart, double* sspart,
                   cudaStream_t st) {
    const int64_t d = A->d;
    if (d > 256)
        LSK_PROF("lsq_pass", st) launch_pdl(cg_pass_dense_kernel, nb, kPassThreads, (size_t)9 * d * 4, 1, st,
                                            (const float*)A->values, A->ld, A->n, d, p, S, qpart, sspart);
    else if (rows_vec4(A)) {
        if (d <= 32) launch_rows_pass<8, 4, 8, true>(A, nb, p, S, rev, qpart, sspart, st);
        else if (d <= 64) launch_rows_pass<16, 4, 8, true>(A, nb, p, S, rev, qpart, sspart, st);
        else if (d <= 128) launch_rows_pass<32, 4, 8, true>(A, nb, p, S, rev, qpart, sspart, st);
        else launch_rows_pass<32, 8, 4, true>(A, nb, p, S, rev, qpart, sspart, st);
    } else {
        if (d <= 32) launch_rows_pass<32, 1, 16, false>(A, nb, p, S, rev, qpart, sspart, st);
        else if (d <= 64) launch_rows_pass<32, 2, 16, false>(A, nb, p, S, rev, qpart, sspart, st);
        else if (d <= 128) launch_rows_pass<32, 4, 8, false>(A, nb, p, S, rev, qpart, sspart, st);
        else launch_rows_pass<32, 8, 4, false>(A, nb, p, S, rev, qpart, sspart, st);
    }
}

template <int L, int E, int RB, bool kVec>
void launch_resid(const lsk_mat* A, int nb, const double* b, const double* x, double* qpart, cudaStream_t st) {
    LSK_PROF("lsq_resid64", st) resid_dense_rows_kernel<L, E, RB, kVec><<<nb, kPassThreads, 0, st>>>(
        (const float*)A->values, A->ld, A->n, (int)A->d, b, x, qpart);
}

// dense b - A x and the blocks' partial sums of A^T (b - A x)
// (x == nullptr: x = 0, d <= 256 only)
cudaError_t resid_dense(const lsk_mat* A, int nb, const double* b, const double* x, double* qpart, cudaStream_t st) {
    const int64_t d = A->d;
    if (d > 256) {
        const size_t sh = (size_t)9 * d * 8;
        if (sh > 48 * 1024) {
            const cudaError_t e = allow_dynamic_smem(resid64_dense_kernel);
            if (e != cudaSuccess) return e;
        }
        LSK_PROF("lsq_resid64", st) resid64_dense_kernel<<<nb, kPassThreads, sh, st>>>((const float*)A->values, A->ld,
                                                                                       A->n, d, b, x, qpart);
    } else if (rows_vec4(A)) {
        if (d <= 32) launch_resid<8, 4, 4, true>(A, nb, b, x, qpart, st);
        else if (d <= 64) launch_resid<8, 8, 4, true>(A, nb, b, x, qpart, st);
        else if (d <= 128) launch_resid<16, 8, 4, true>(A, nb, b, x, qpart, st);
        else launch_resid<32, 8, 4, true>(A, nb, b, x, qpart, st);
    } else {
        if (d <= 32) launch_resid<32, 1, 8, false>(A, nb, b, x, qpart, st);
        else if (d <= 64) launch_resid<32, 2, 8, false>(A, nb, b, x, qpart, st);
        else if (d <= 128) launch_resid<32, 4, 4, false>(A, nb, b, x, qpart, st);
        else launch_resid<32, 8, 4, false>(A, nb, b, x, qpart, st);
    }
    return cudaGetLastError();
}

// ---- CSR tiles: plan, workspace ----------------------------------------------
CsrTiles tiles_plan(const lsk_mat* A, int sm_count) {
    CsrTiles t{};
    t.n = A->n;
    t.d = A->d;
    int64_t rp = (A->n + kTilesPerSm * (int64_t)sm_count - 1) / (kTilesPerSm * (int64_t)sm_count);
    rp = std::max<int64_t>(32, std::min<int64_t>(rp, kTileRowsMax));
    t.rows_per = (int)rp;
    t.ntiles = (A->n + rp - 1) / rp;
    t.V = (const float*)A->values;
    t.J = A->colidx;
    t.I = A->rowptr;
    return t;
}
size_t tiles_smem(const CsrTiles& t, size_t elem) {
    return (kTileEntries + 2 * (size_t)t.d + t.rows_per) * elem + (t.rows_per + t.d + 2) * 4 + 16;
}
size_t tiles_bytes(const lsk_mat* A, int sm_count) {
    const CsrTiles t = tiles_plan(A, sm_count);
    return ws_round((size_t)t.ntiles * (t.d + 1) * 4) + ws_round((size_t)A->nnz * 4) + ws_round((size_t)A->nnz * 2);
}

}  // namespace

// atr = A^T (b - A x) in FP64 (the residual pass of the refinement loop,
// reduced in block order); x == nullptr means x = 0.
namespace {
__global__ void sum_qpart_kernel(const double* __restrict__ qpart, int nblocks, int64_t d, double* __restrict__ atr) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int z = 0; z < nblocks; ++z) s += qpart[(int64_t)z * d + j];
        atr[j] = s;
    }
}
}  // namespace

size_t atr64_workspace_bytes(const lsk_mat* A) {
    const int nb = kMaxPassBlocks;
    return ws_round((size_t)nb * A->d * 8) + ws_round((size_t)A->d * 8) + 1024;
}

cudaError_t atr64_launch(const lsk_mat* A, const double* b, const double* x, double* atr, void* ws, int* flag,
                         int sm_count, cudaStream_t st) {
    const int64_t n = A->n, d = A->d;
    const int nb = pass_grid(A, sm_count);
    WsCarver wc{(char*)ws, 0};
    double* qpart = wc.take<double>((size_t)nb * d);
    double* zero = wc.take<double>(d);
    cudaError_t e = cudaSuccess;
    if (!x && !(A->kind == LSK_DENSE && d <= 256)) {
        if ((e = cudaMemsetAsync(zero, 0, (size_t)d * 8, st)) != cudaSuccess) return e;
        x = zero;
    }
    if (A->kind == LSK_DENSE) {
        if ((e = resid_dense(A, nb, b, x, qpart, st)) != cudaSuccess) return e;
    } else {
        const size_t sh = (size_t)2 * d * 8;
        if (sh > 48 * 1024 && (e = allow_dynamic_smem(resid64_csr_kernel)) != cudaSuccess) return e;
        LSK_PROF("lsq_resid64", st) resid64_csr_kernel<<<nb, kPassThreads, sh, st>>>(
            (const float*)A->values, A->colidx, A->rowptr, n, A->nnz, d, b, x, qpart, flag);
    }
    LSK_PROF("lsq_small", st) sum_qpart_kernel<<<(unsigned)((d + 255) / 256), 256, 0, st>>>(qpart, nb, d, atr);
    return cudaGetLastError();
}

// Pinned copies of the solver's state for the lagged stopping test.
struct LsqHost {
    CgState* state;       // two, pinned
    cudaEvent_t ev[2];
    int ctas;             // of the step's cluster
    cudaError_t read(int slot, const CgState* S, cudaStream_t st) {
        const cudaError_t e = cudaMemcpyAsync(state + slot, S, sizeof(CgState), cudaMemcpyDeviceToHost, st);
        return e != cudaSuccess ? e : cudaEventRecord(ev[slot], st);
    }
    cudaError_t wait(int slot) { return cudaEventSynchronize(ev[slot]); }
};

void lsq_host_free(lsk_ctx* ctx) {
    LsqHost* h = ctx->lsq_host;
    if (!h) return;
    for (cudaEvent_t ev : h->ev)
        if (ev) cudaEventDestroy(ev);
    if (h->state) cudaFreeHost(h->state);
    delete h;
    ctx->lsq_host = nullptr;
}

namespace {
LsqHost* lsq_host(lsk_ctx* ctx) {
    if (ctx->lsq_host) return ctx->lsq_host;
    ctx->lsq_host = new (std::nothrow) LsqHost();
    LsqHost* h = ctx->lsq_host;
    if (!h) return nullptr;
    if (cudaMallocHost(&h->state, 2 * sizeof(CgState)) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev[1], cudaEventDisableTiming) != cudaSuccess) {
        lsq_host_free(ctx);
        return nullptr;
    }
    h->ctas = cg_vec_ctas();
    return h;
}
}  // namespace

size_t lsq_workspace_bytes(const lsk_mat* A, int sm_count) {
    const int64_t d = A->d;
    const int nb = kMaxPassBlocks;
    return ws_round(sizeof(CgState)) + 4 * ws_round((size_t)d * 8) + 3 * ws_round((size_t)d * d * 8) +
           ws_round((size_t)nb * d * 8) + ws_round((size_t)nb * 8) + ws_round((size_t)d * 4) +
           (A->kind == LSK_CSR ? tiles_bytes(A, sm_count) : 0) + 4096;
}

int lsq_run(lsk_ctx* ctx, const lsk_mat* A, const double* b, double* x, const lsk_lsq_opts* o,
            const double* Rinv64, void* ws, lsk_lsq_info* info) {
    cudaStream_t st = ctx->stream;
    const int64_t d = A->d;
    const bool dense = A->kind == LSK_DENSE;
    WsCarver wc{(char*)ws, 0};
    LsqHost* host = lsq_host(ctx);
    if (!host) return LSK_ERR_CUDA;
    const int ctas = ctx->lsq_ctas > 0 ? std::min(ctx->lsq_ctas, host->ctas) : host->ctas;
    CgState* S = wc.take<CgState>(1);
    double* y = wc.take<double>(d);
    double* cg_s = wc.take<double>(d);
    double* cg_p = wc.take<double>(d);
    double* Nt = wc.take<double>((size_t)d * d);   // N^T
    float2 *N2 = nullptr, *Nt2 = nullptr;
    if (d <= 256 && d <= ctas * (kVecThreads / 32)) {   // a row a warp
        N2 = wc.take<float2>((size_t)d * d);
        Nt2 = wc.take<float2>((size_t)d * d);
    }
    double* qpart64 = wc.take<double>((size_t)kMaxPassBlocks * d);
    double* sspart = wc.take<double>(kMaxPassBlocks);
    float* p = wc.take<float>(d);
    float* qpart32 = reinterpret_cast<float*>(qpart64);   // reused by the FP32 pass

    CgState h{};
    cudaError_t e = cudaMemsetAsync(x, 0, (size_t)d * 8, st);
    if (e != cudaSuccess) return LSK_ERR_CUDA;
    const dim3 tg((unsigned)((d + 31) / 32), (unsigned)((d + 31) / 32));
    LSK_PROF("lsq_small", st) factor_forms_kernel<<<tg, 256, 0, st>>>(Rinv64, (int)d, Nt, N2, Nt2);
    int nb = pass_grid(A, ctx->sm_count);
    CsrTiles t{};
    size_t sh32 = 0, sh64 = 0;
    if (!dense) {
        t = tiles_plan(A, ctx->sm_count);
        t.cptr = wc.take<int32_t>((size_t)t.ntiles * (d + 1));
        t.tval = wc.take<float>((size_t)A->nnz);
        t.trow = wc.take<uint16_t>((size_t)A->nnz);
        sh32 = tiles_smem(t, sizeof(float));
        sh64 = tiles_smem(t, sizeof(double));
        if (allow_dynamic_smem(tile_pass_kernel<float>) != cudaSuccess ||
            allow_dynamic_smem(tile_pass_kernel<double>) != cudaSuccess)
            return LSK_ERR_CUDA;
        nb = (int)std::max<int64_t>(1, std::min<int64_t>(t.ntiles, kTilesPerSm * (int64_t)ctx->sm_count));
        if (t.ntiles > 0)
            LSK_PROF("lsq_tiles", st) csr_tiles_kernel<<<(unsigned)t.ntiles, kPassThreads, (size_t)d * 4, st>>>(t, A->nnz);
    }
    int total_it = 0, refinements = 0, status = LSK_ERR_NOT_CONVERGED;
    double eta = INFINITY;
    for (int step = 0; step <= o->max_refine; ++step) {
        if (dense) {
            if (resid_dense(A, nb, b, step == 0 && d <= 256 ? nullptr : x, qpart64, st) != cudaSuccess) return LSK_ERR_CUDA;
        } else {
            LSK_PROF("lsq_resid64", st) tile_pass_kernel<double><<<nb, kPassThreads, sh64, st>>>(t, nullptr, x, b, S, qpart64, sspart);
        }
        if (launch_vec<true>(ctas, qpart64, sspart, nb, d, Rinv64, Nt, nullptr, nullptr, step == 0 ? 1 : 0, 0.0, S, cg_s, cg_p, y, p, st) != cudaSuccess)
            return LSK_ERR_CUDA;
        e = cudaMemcpyAsync(&h, S, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return LSK_ERR_CUDA;
        eta = h.eta;
        refinements = step;
        if (!(eta > o->tol)) {
            status = LSK_OK;
            break;
        }
        if (step == o->max_refine) break;
        // the inner solve need only reduce its residual by the factor left to
        // reach tol (with a margin of 20), and never by less than inner_tol
        double stop_rel = 0.05 * o->tol / eta;
        if (stop_rel < o->inner_tol) stop_rel = o->inner_tol;
        if (stop_rel > 0.5) stop_rel = 0.5;
        // The stopping test lags: iterations are queued four at a time with a
        // copy of the state behind each four, and the host waits for the copy
        // two batches back, so the GPU always has work queued (kernels queued
        // past the end return at once).
        int queued = 0;
        for (int batch = 0; queued < o->max_iter; ++batch) {
            if (batch >= 2) {
                if ((e = host->wait(batch & 1)) != cudaSuccess) return LSK_ERR_CUDA;
                if (host->state[batch & 1].done) break;
            }
            for (int k = 0; k < 4 && queued < o->max_iter; ++k, ++queued) {
                if (dense)
                    cg_pass_dense(A, nb, p, S, queued & 1, qpart32, sspart, st);
                else
                    LSK_PROF("lsq_pass", st) launch_pdl(tile_pass_kernel<float>, nb, kPassThreads, sh32, 1, st, t, (const float*)p,
                                                        (const double*)nullptr, (const double*)nullptr, (const CgState*)S,
                                                        (void*)qpart32, sspart);
                if (launch_vec<false>(ctas, qpart32, sspart, nb, d, Rinv64, Nt, N2, Nt2, 0, stop_rel, S, cg_s, cg_p, y, p, st) != cudaSuccess)
                    return LSK_ERR_CUDA;
            }
            if ((e = host->read(batch & 1, S, st)) != cudaSuccess) return LSK_ERR_CUDA;
        }
        e = cudaMemcpyAsync(&h, S, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return LSK_ERR_CUDA;
        total_it += h.it;
        LSK_PROF("lsq_small", st) update_x_kernel<<<(unsigned)((d + 7) / 8), 256, 0, st>>>(Rinv64, d, y, x);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return LSK_ERR_CUDA;
    if (info) {
        info->iters = total_it;
        info->refinements = refinements;
        info->eta = eta;
        info->status = status;
    }
    return status;
}
