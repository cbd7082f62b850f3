// jlt.cu -- Gaussian sketch of a CSR matrix, C = G A (Alg. 4, csrjlt).
//
// G is m x n with entries z / sqrt(m) drawn like the Gaussian stage's G
// (Philox-4x32-10 + Box-Muller, bfloat16-rounded in the BF16 mode) on
// counter stream 3, with column index = row index of A.  As in Alg. 4 each
// block owns a range of rows of G and keeps its slice of C, d x jb, in shared
// memory; the row ranges of A are split over blocks too (split-K) and the
// partial slices are summed in a fixed order.
//
// A block takes its rows of A a chunk at a time:
//   1. its threads draw the jb x R entries of G of the chunk into shared
//      memory (four a Philox call, one 16-byte store), whatever A holds;
//   2. the chunk's nonzeros, 256 at a time, are sorted by column mod the
//      number of groups, stably (warp matches and a scan, no atomics);
//   3. group g of jb / 2 threads (two rows each) adds G[:, row] A[row, col] into C[:, col] for its
//      own columns: no two groups touch the same entry of C, and each entry's
//      additions run in row order.
// Three blocks of 8 warps share an SM, so that one draws while another sorts or
// adds.  With one thread per row of G drawing for itself (values swapped inside
// quads by shuffles) a 128-row slice left 8 warps an SM to hide the draws'
// latency behind; 500,000 x 200 with 1.0 M nonzeros, m = 400: 2.75 ms against
// 0.65 ms.
#include "lsk_internal.cuh"

#include <algorithm>

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kItems = 4;          // Philox calls per thread and chunk
constexpr int kMaxRows = 256;      // rows of A in a chunk

struct JltParams {
    const float* V;
    const int32_t* J;
    const int64_t* I;
    int64_t n, nnz, rows_per_split, rows_per_part;
    int parts;                     // partials a split
    int d, m, jb, lg, rows;        // rows of G a block, log2 of the threads a group, rows of A a chunk
    uint32_t nq_inv;               // ceil(2^16 / (jb / 4))
    uint32_t k0, k1;
    float scale;
    int bf16;
    float* part;
    int* flag;
};

// shared memory: C [d][jb], G [rows][jb], the sorted batch, row pointers
__host__ __device__ inline size_t jlt_smem(int64_t d, int jb, int rows) {
    return (size_t)d * jb * 4 + (size_t)rows * jb * 4 + kThreads * 8 + (size_t)(rows + 1) * 4 + kThreads * 2 + 64;
}

__global__ void __launch_bounds__(kThreads, 3) csrjlt_kernel(const JltParams p) {
    extern __shared__ __align__(16) float cs[];                       // [d][jb]
    float* gs = cs + (size_t)p.d * p.jb;                              // [rows][jb]
    uint2* list = reinterpret_cast<uint2*>(gs + p.rows * p.jb);       // (col << 16 | row, value) sorted by group
    int32_t* rp = reinterpret_cast<int32_t*>(list + kThreads);        // row offsets of the chunk
    uint16_t* rid = reinterpret_cast<uint16_t*>(rp + p.rows + 1);     // row of each entry of the batch
    __shared__ int hist[kWarps][64], start[65];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int jb = p.jb, nq = jb >> 2, ngroups = kThreads >> p.lg;
    const int grp = t >> p.lg, jj = 2 * (t & ((1 << p.lg) - 1));   // rows jj, jj + 1 of the slice
    const int j0 = (int)blockIdx.x * jb;
    const int64_t r0 = (int64_t)blockIdx.y * p.rows_per_split, r1 = min(p.n, r0 + p.rows_per_split);
    for (int x = t; x < p.d * jb; x += kThreads) cs[x] = 0.f;
    bool bad = false;
    for (int k = 0; k < p.parts; ++k) {
        const int64_t rb = r0 + k * p.rows_per_part, re = min(r1, rb + p.rows_per_part);
        for (int64_t ra = rb; ra < re; ra += p.rows) {
            const int nr = (int)min((int64_t)p.rows, re - ra);
            const int64_t nz0 = p.I[ra], nz1 = p.I[ra + nr];
            const bool span_ok = nz0 >= 0 && nz1 >= nz0 && nz1 <= p.nnz;
            if (!span_ok) {
                bad = true;
                continue;   // the same for every thread
            }
            // the first batch's entries and the row pointers arrive under the draws
            int32_t col = 0;
            float val = 0.f;
            if (nz0 + t < nz1) {
                col = __ldg(p.J + nz0 + t);
                val = __ldg(p.V + nz0 + t);
            }
            __syncthreads();   // the last chunk's readers
            for (int r = t; r <= nr; r += kThreads) {
                const int64_t k = p.I[ra + r];
                if (k < nz0 || k > nz1) bad = true;
                rp[r] = (int32_t)(min(max(k, nz0), nz1) - nz0);
            }
#pragma unroll
            for (int i = 0; i < kItems; i += 2) {
                float4 z[2];
                int at[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const uint32_t item = (uint32_t)(t + kThreads * (i + u)), r = (item * p.nq_inv) >> 16, q = item - r * nq;
                    at[u] = (int)r < nr ? (int)(r * jb + 4 * q) : -1;
                    z[u] = gauss4((uint64_t)ra + r, (uint32_t)(j0 >> 2) + q, p.k0, p.k1, 3u);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float4 g = make_float4(z[u].x * p.scale, z[u].y * p.scale, z[u].z * p.scale, z[u].w * p.scale);
                    if (p.bf16) g = make_float4(bf16_round(g.x), bf16_round(g.y), bf16_round(g.z), bf16_round(g.w));
                    if (at[u] >= 0) *reinterpret_cast<float4*>(gs + at[u]) = g;
                }
            }
            const int count = (int)(nz1 - nz0);
            for (int b0 = 0; b0 < count; b0 += kThreads) {
                if (b0) {
                    col = 0;
                    val = 0.f;
                    if (b0 + t < count) {
                        col = __ldg(p.J + nz0 + b0 + t);
                        val = __ldg(p.V + nz0 + b0 + t);
                    }
                }
                rid[t] = 0xFFFFu;
                for (int x = t; x < kWarps * 64; x += kThreads) (&hist[0][0])[x] = 0;
                __syncthreads();   // G, rp written; the last batch's list read
                for (int r = t; r < nr; r += kThreads) {
                    const int e0 = max(rp[r] - b0, 0), e1 = min(rp[r + 1] - b0, kThreads);
                    if (rp[r + 1] < rp[r]) bad = true;
                    for (int e = e0; e < e1; ++e) rid[e] = (uint16_t)r;
                }
                bool in = b0 + t < count;
                if (in && (col < 0 || col >= p.d)) {
                    bad = true;
                    in = false;
                }
                const int g = in ? col & (ngroups - 1) : 64;
                const uint32_t same = __match_any_sync(0xffffffffu, g);
                const int rank = __popc(same & ((1u << lane) - 1u));
                if (in && rank == 0) hist[w][g] = __popc(same);
                __syncthreads();
                if (w == 0) {   // start[g]: exclusive sums over the groups; hist: over the warps of a group
                    int run = 0;
                    for (int h = 0; h < ngroups; h += 32) {
                        const int gg = h + lane;
                        int s = 0;
                        if (gg < ngroups)
#pragma unroll
                            for (int x = 0; x < kWarps; ++x) {
                                const int c = hist[x][gg];
                                hist[x][gg] = s;
                                s += c;
                            }
                        int inc = s;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int up = __shfl_up_sync(0xffffffffu, inc, o);
                            if (lane >= o) inc += up;
                        }
                        if (gg < ngroups) start[gg] = run + inc - s;
                        run += __shfl_sync(0xffffffffu, inc, 31);
                    }
                    if (lane == 0) start[ngroups] = run;
                }
                __syncthreads();
                if (in) {
                    const uint32_t r = rid[t];   // 0xFFFF: no row covers it (bad is set)
                    list[start[g] + hist[w][g] + rank] =
                        make_uint2(((uint32_t)col << 16) | (r == 0xFFFFu ? 0u : r), r == 0xFFFFu ? 0u : __float_as_uint(val));
                }
                __syncthreads();
                if (jj < jb) {
                    int q = start[grp];
                    const int q1 = start[grp + 1];
                    for (; q + 1 < q1; q += 2) {   // two at a time
                        const uint2 a = list[q], b = list[q + 1];
                        float2* ca = reinterpret_cast<float2*>(cs + (a.x >> 16) * jb + jj);
                        float2* cb = reinterpret_cast<float2*>(cs + (b.x >> 16) * jb + jj);
                        const float2 ga = *reinterpret_cast<const float2*>(gs + (a.x & 0xFFFFu) * jb + jj);
                        const float2 gb = *reinterpret_cast<const float2*>(gs + (b.x & 0xFFFFu) * jb + jj);
                        const float va = __uint_as_float(a.y), vb = __uint_as_float(b.y);
                        float2 xa = *ca, xb = *cb;
                        xa.x = fmaf(ga.x, va, xa.x);
                        xa.y = fmaf(ga.y, va, xa.y);
                        if (ca == cb) xb = xa;
                        else *ca = xa;
                        xb.x = fmaf(gb.x, vb, xb.x);
                        xb.y = fmaf(gb.y, vb, xb.y);
                        *cb = xb;
                    }
                    if (q < q1) {
                        const uint2 a = list[q];
                        float2* ca = reinterpret_cast<float2*>(cs + (a.x >> 16) * jb + jj);
                        const float2 ga = *reinterpret_cast<const float2*>(gs + (a.x & 0xFFFFu) * jb + jj);
                        const float va = __uint_as_float(a.y);
                        float2 xa = *ca;
                        xa.x = fmaf(ga.x, va, xa.x);
                        xa.y = fmaf(ga.y, va, xa.y);
                        *ca = xa;
                    }
                }
            }
        }
        // part[split, k][col][j]: consecutive threads, consecutive addresses, each
        // thread the entries that it adds to (cleared for the next rows)
        __syncthreads();
        const int64_t at = (int64_t)blockIdx.y * p.parts + k;
        for (int c = grp; c < p.d; c += ngroups)
            for (int e = 0; e < 2; ++e)
                if (jj < jb) {
                    if (j0 + jj + e < p.m) p.part[(at * p.d + c) * p.m + j0 + jj + e] = cs[c * jb + jj + e];
                    cs[c * jb + jj + e] = 0.f;
                }
    }
    if (bad) set_flag(p.flag, LSK_FLAG_BAD_CSR);
}

// C[j][col] = sum over parts of part[][col][j]: a block takes 32 entries, warp g
// adds the parts g, g + kReduceWarps, ... of them with compensation (eight loads in
// flight), then the warps' sums are added in order.
template <int kReduceWarps>
__global__ void __launch_bounds__(32 * kReduceWarps) csrjlt_reduce_kernel(const float* __restrict__ part, int nparts, int d,
                                                                          int m, float* __restrict__ C) {
    __shared__ double acc[kReduceWarps][32];
    const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t total = (int64_t)d * m, x = (int64_t)blockIdx.x * 32 + lane;
    float s = 0.f, c = 0.f;
    if (x < total)
        for (int b = g; b < nparts; b += 8 * kReduceWarps) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                v[k] = b + k * kReduceWarps < nparts ? part[(b + k * kReduceWarps) * total + x] : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) comp_add(s, c, v[k]);
        }
    acc[g][lane] = (double)s + (double)c;
    if (!comp_ok(s, c)) {
        double t = 0.0;
        for (int b = g; b < nparts; b += kReduceWarps) t += (double)part[(int64_t)b * total + x];
        acc[g][lane] = t;
    }
    __syncthreads();
    if (g == 0 && x < total) {
        double t = 0.0;
        for (int k = 0; k < kReduceWarps; ++k) t += acc[k][lane];
        C[(x % m) * d + x / m] = (float)t;
    }
}

struct JltPlan {
    int jb, lg, rows, jblocks, nsplit, parts;   // (parts: partials a split)
    int64_t rows_per_split, rows_per_part;
    size_t smem;
};

// Rows of G a block: up to 64, fewer where a slice of C that wide would leave
// fewer than three blocks on an SM (d > 230) -- but at least 16, so that a
// nonzero's bookkeeping is shared by that many rows.
bool jlt_plan(int64_t n, int64_t d, int64_t m, int sm_count, JltPlan& p) {
    if (d < 1 || m < 1 || m > (1 << 20) || d > 1527) return false;
    const size_t smem_sm = 227 * 1024;
    int cap = 64;
    const auto rows_of = [](int jb) { return std::min(kMaxRows, kItems * kThreads / (jb / 4)); };
    while (cap > 16 && 3 * (jlt_smem(d, cap, rows_of(cap)) + 3072) > smem_sm) cap >>= 1;
    const int64_t jblocks = (m + cap - 1) / cap;
    p.jb = (int)(((m + jblocks - 1) / jblocks + 3) / 4 * 4);
    p.jblocks = (int)((m + p.jb - 1) / p.jb);
    p.lg = 2;   // a thread adds two rows; at most 64 groups
    while ((2 << p.lg) < p.jb) ++p.lg;
    p.rows = rows_of(p.jb);
    p.smem = jlt_smem(d, p.jb, p.rows);
    // one wave: as many row splits as resident blocks allow
    int64_t per_sm = (int64_t)(smem_sm / (p.smem + 3072));
    per_sm = std::max<int64_t>(1, std::min<int64_t>(per_sm, 3));
    int64_t ns = std::max<int64_t>(1, (int64_t)sm_count * per_sm / p.jblocks);
    ns = std::max<int64_t>(1, std::min<int64_t>(ns, (n + 511) / 512));
    // Partials: the error is that of the FP32 chain of products of an entry within
    // one, so a block stores its slice every thousand rows of A or more, as many
    // partials in all as 160 KB an SM hold (with one a split, 500,000 x 32 with
    // 1% nonzeros, m = 400, was 1.7e-7 off in 505 us; 0.9e-7 in 524 now).
    const int64_t want = std::max<int64_t>(ns, (int64_t)sm_count * (160 << 10) / (d * m * 4));
    const int64_t sub = std::max<int64_t>(1, std::min<int64_t>((want + ns - 1) / ns, (n / ns + 1023) / 1024));
    const int64_t chunks = std::max<int64_t>(1, ((n + ns - 1) / ns + p.rows - 1) / p.rows);   // of a split
    p.rows_per_split = chunks * p.rows;
    p.rows_per_part = (chunks + sub - 1) / sub * p.rows;
    p.parts = (int)((p.rows_per_split + p.rows_per_part - 1) / p.rows_per_part);
    p.nsplit = (int)std::max<int64_t>(1, (n + p.rows_per_split - 1) / p.rows_per_split);
    return true;
}

}  // namespace

bool jlt_supported(int64_t d, int64_t m) {
    JltPlan p;
    return jlt_plan(1024, d, m, 152, p);
}

size_t jlt_workspace_bytes(int64_t n, int64_t d, int64_t m, int sm_count) {
    JltPlan p;
    if (!jlt_plan(n, d, m, sm_count, p)) return 0;
    return ws_round((size_t)p.nsplit * p.parts * d * m * 4);
}

cudaError_t jlt_launch(const lsk_mat* A, int64_t m, uint64_t seed, int32_t prec, float* C, void* ws, int* flag,
                       int sm_count, cudaStream_t st) {
    const int64_t n = A->n, d = A->d;
    JltPlan q;
    if (!jlt_plan(n, d, m, sm_count, q)) return cudaErrorNotSupported;
    if (n == 0) return cudaMemsetAsync(C, 0, (size_t)m * d * 4, st);
    JltParams p{};
    p.V = (const float*)A->values;
    p.J = A->colidx;
    p.I = A->rowptr;
    p.n = n;
    p.nnz = A->nnz;
    p.rows_per_split = q.rows_per_split;
    p.rows_per_part = q.rows_per_part;
    p.parts = q.parts;
    p.d = (int)d;
    p.m = (int)m;
    p.jb = q.jb;
    p.lg = q.lg;
    p.rows = q.rows;
    p.nq_inv = (65536u + (uint32_t)(q.jb / 4) - 1) / (uint32_t)(q.jb / 4);
    p.k0 = (uint32_t)seed;
    p.k1 = (uint32_t)(seed >> 32);
    p.scale = (float)(1.0 / sqrt((double)m));
    p.bf16 = prec == LSK_PREC_BF16 ? 1 : 0;
    p.part = (float*)ws;
    p.flag = flag;
    cudaError_t e;
    // (at any size: the default limit, 48 KB, counts the kernel's static arrays too)
    if ((e = allow_dynamic_smem(csrjlt_kernel)) != cudaSuccess) return e;
    LSK_PROF("csrjlt", st) csrjlt_kernel<<<dim3((unsigned)q.jblocks, (unsigned)q.nsplit), kThreads, q.smem, st>>>(p);
    const int64_t total = d * m;
    const bool many = q.nsplit * q.parts > 256;   // (128 loads in flight an entry, or 32)
    LSK_PROF("csrjlt_reduce", st) (many ? csrjlt_reduce_kernel<16> : csrjlt_reduce_kernel<4>)<<<(unsigned)((total + 31) / 32), many ? 512 : 128, 0, st>>>(
        p.part, q.nsplit * q.parts, (int)d, (int)m, C);
    return cudaGetLastError();
}
