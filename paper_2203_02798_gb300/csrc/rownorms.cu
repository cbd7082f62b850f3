// rownorms.cu -- x <- alpha * diag(A B B^T A^T) + beta * x (csrsqn / rmsqn).
//
// dense (rmsqn): a block owns 128 rows of A and sweeps the columns of B in
//   tiles of 64; each product tile A_blk * B_tile stays in registers, is
//   squared and summed into per-row partials, so A*B never exists outside
//   registers (the memory-efficient form of Alg. 8 for dense A).  When B is
//   upper triangular (B = R^-1) the k-loop of column tile [c0, c0+64) stops
//   at c0+64, skipping the zero blocks.  This is the CUDA-core (SIMT) path of
//   LSK_PREC_FP32: A that is small, wide or unaligned, and the rows that the
//   tensor-core path (rownorms_tc3.cu) leaves; BF16 and TF32 are in rownorms_tc.cu.
// CSR (csrsqn, Alg. 8): Btilde = B B^T is formed once (FP32, 16 x 16 output
//   tiles); then one thread per row, or with more than three nonzeros a row one
//   lane per nonzero, evaluates
//   sum_{p,q in row} v_p v_q Btilde[J_p, J_q] using the symmetry of Btilde.
#include "lsk_internal.cuh"

#include <algorithm>

namespace {

constexpr int RM = 128;   // rows of A per block
constexpr int RN = 64;    // columns of B per tile
constexpr int RK = 16;    // reduction step
constexpr int RMP = RM + 4;

// The rows list[0 .. rows), rows <= kShort gridDim.x, each block kShort of them, a
// thread to a column (c, d <= 256).  One tile of 128 rows takes an SM 45 us at 256 x
// 256, the rest of the GPU idle: 20,000 x 256 with a few listed rows 87 us, 49 this
// way.  (Not inlined: the tiles' loop keeps its registers.)
constexpr int kShort = 4;
__device__ __noinline__ void short_list(const float* __restrict__ A, int64_t lda, int rows, int d,
                                        const float* __restrict__ B, int c, float alpha, float beta,
                                        float* __restrict__ x, const int* __restrict__ list, float* a, float* part) {
    if ((int)blockIdx.x >= rows) return;
    const int tid = threadIdx.x;
#pragma unroll
    for (int r = 0; r < kShort; ++r) {       // a: [d][kShort]
        const int i = (int)blockIdx.x + r * (int)gridDim.x;
        if (tid < d) a[tid * kShort + r] = i < rows ? __ldg(A + (int64_t)__ldg(list + i) * lda + tid) : 0.f;
    }
    __syncthreads();
    float y[kShort] = {};
    if (tid < c) {
#pragma unroll 8
        for (int k = 0; k < d; ++k) {
            const float b = __ldg(B + (int64_t)k * c + tid);
            const float4 v = *reinterpret_cast<const float4*>(a + k * kShort);
            y[0] = fmaf(v.x, b, y[0]);
            y[1] = fmaf(v.y, b, y[1]);
            y[2] = fmaf(v.z, b, y[2]);
            y[3] = fmaf(v.w, b, y[3]);
        }
    }
#pragma unroll
    for (int r = 0; r < kShort; ++r) {       // part: [8 warps][kShort]
        const float q = warp_sum(y[r] * y[r]);
        if ((tid & 31) == 0) part[(tid >> 5) * kShort + r] = q;
    }
    __syncthreads();
    const int i = (int)blockIdx.x + tid * (int)gridDim.x;
    if (tid < kShort && i < rows) {
        float q = 0.f;
        for (int w = 0; w < 8; ++w) q += part[w * kShort + tid];
        float* const xi = x + __ldg(list + i);
        *xi = (beta != 0.f) ? fmaf(alpha, q, beta * *xi) : alpha * q;
    }
}

// thread (ty, tx) = (tid / 16, tid % 16): rows 8*ty..8*ty+7, cols 4*tx..4*tx+3.
// kList: the rows list[0 .. *count) of A and x only (all where *count < 0), a
// persistent grid.
template <bool kList, bool kPdl = true>
__global__ void __launch_bounds__(256) rownorm_dense_kernel(
    const float* __restrict__ A, int64_t lda, int64_t n, int64_t d, const float* __restrict__ B,
    int64_t c, int upper_tri, float alpha, float beta, float* __restrict__ x, const int* __restrict__ list,
    const int* __restrict__ count) {
    if constexpr (kPdl) pdl_enter(A, B, x, list, count);
    __shared__ __align__(16) float As[RK][RMP];
    __shared__ __align__(16) float Bs[RK][RN];
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    const bool all = !kList || *count < 0;
    const int64_t rows = all ? n : (int64_t)*count;
    const auto row_of = [&](int64_t i) { return all ? i : (int64_t)__ldg(list + i); };
    const bool brief = kList && !all && rows <= (int64_t)kShort * gridDim.x && c <= 256 && d <= 256;
    int64_t i0 = (int64_t)blockIdx.x * RM;
    if (!kList || (i0 < rows && !brief)) do {
        float rowsum[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) rowsum[a] = 0.f;
        // a thread loads the same eight rows of every chunk
        int64_t at[kList ? 8 : 1];
        if constexpr (kList) {
#pragma unroll
            for (int t = 0; t < (RM * RK) / 256; ++t) {
                const int64_t i = i0 + tid / RK + (256 / RK) * t;
                at[t] = i < rows ? row_of(i) * lda : 0;
            }
        }

        for (int64_t c0 = 0; c0 < c; c0 += RN) {
            const int64_t kmax = upper_tri ? min(d, c0 + RN) : d;
            float acc[8][4];
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
            for (int64_t k0 = 0; k0 < kmax; k0 += RK) {
#pragma unroll
                for (int t = 0; t < (RM * RK) / 256; ++t) {
                    const int idx = tid + 256 * t;
                    const int row = idx / RK, kk = idx % RK;
                    const int64_t i = i0 + row, kx = k0 + kk;
                    const int64_t row_at = kList ? at[kList ? t : 0] : i * lda;
                    As[kk][row] = (i < rows && kx < kmax) ? __ldg(A + row_at + kx) : 0.f;
                }
#pragma unroll
                for (int t = 0; t < (RK * RN) / 256; ++t) {
                    const int idx = tid + 256 * t;
                    const int kk = idx / RN, cc = idx % RN;
                    const int64_t kx = k0 + kk, cx = c0 + cc;
                    Bs[kk][cc] = (kx < kmax && cx < c) ? __ldg(B + kx * c + cx) : 0.f;
                }
                __syncthreads();
#pragma unroll
                for (int kk = 0; kk < RK; ++kk) {
                    const float4 a0 = *reinterpret_cast<const float4*>(&As[kk][8 * ty]);
                    const float4 a1 = *reinterpret_cast<const float4*>(&As[kk][8 * ty + 4]);
                    const float4 bv = *reinterpret_cast<const float4*>(&Bs[kk][4 * tx]);
                    const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                    const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
                    for (int a = 0; a < 8; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(av[a], bb[b], acc[a][b]);
                }
                __syncthreads();
            }
#pragma unroll
            for (int a = 0; a < 8; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) rowsum[a] = fmaf(acc[a][b], acc[a][b], rowsum[a]);
        }
        // the 16 threads of a half-warp share rows: reduce across tx
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            float v = rowsum[a];
#pragma unroll
            for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            rowsum[a] = v;
        }
        if (tx == 0) {
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const int64_t i = i0 + 8 * ty + a;
                if (i < rows) {
                    float* const xi = x + row_of(i);
                    *xi = (beta != 0.f) ? fmaf(alpha, rowsum[a], beta * *xi) : alpha * rowsum[a];
                }
            }
        }
        if (!kList) return;   // one tile a block
        i0 += (int64_t)gridDim.x * RM;
    } while (i0 < rows);
    if (brief) short_list(A, lda, (int)rows, (int)d, B, (int)c, alpha, beta, x, list, &As[0][0], &Bs[0][0]);
}

// Btilde[a][b] = sum_j B[a][j] B[b][j], FP32, 16 x 16 output tiles (one
// output per thread, two accumulation chains).
__device__ __forceinline__ void bbt_body(const float* __restrict__ B, int64_t d, int64_t c, float* __restrict__ M,
                                         int64_t a0, int64_t b0) {
    __shared__ float Ba[16][17], Bb[16][17];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc0 = 0.f, acc1 = 0.f;
    for (int64_t j0 = 0; j0 < c; j0 += 16) {
        const int64_t ja = j0 + tx;
        Ba[ty][tx] = (a0 + ty < d && ja < c) ? __ldg(B + (a0 + ty) * c + ja) : 0.f;
        Bb[ty][tx] = (b0 + ty < d && ja < c) ? __ldg(B + (b0 + ty) * c + ja) : 0.f;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            acc0 = fmaf(Ba[ty][j], Bb[tx][j], acc0);
            acc1 = fmaf(Ba[ty][j + 1], Bb[tx][j + 1], acc1);
        }
        __syncthreads();
    }
    if (a0 + ty < d && b0 + tx < d) M[(a0 + ty) * d + b0 + tx] = acc0 + acc1;
}
__global__ void __launch_bounds__(256) bbt_kernel(const float* __restrict__ B, int64_t d, int64_t c,
                                                  float* __restrict__ M) {
    pdl_enter(B, M);
    bbt_body(B, d, c, M, (int64_t)blockIdx.y * 16, (int64_t)blockIdx.x * 16);
}
// B B^T of many problems in one launch: problem g's 16 x 16 tiles are blocks
// off[g] .. off[g + 1] - 1, row-major over the tile grid
__global__ void __launch_bounds__(256) bbt_grouped_kernel(const BbtJob* __restrict__ jobs, const int* __restrict__ off,
                                                          int count) {
    const int g = group_of(off, count, blockIdx.x);
    const BbtJob& j = jobs[g];
    const int64_t tiles = (j.d + 15) / 16, t = (int64_t)blockIdx.x - __ldg(off + g);
    bbt_body(j.B, j.d, j.c, j.M, (t / tiles) * 16, (t % tiles) * 16);
}

// x_i = alpha a_i M a_i^T + beta x_i, a row a thread.  Launched plainly, as is the
// form below: blocks sent out beside B B^T pile up on some SMs and read through
// pointers that the compiler knows nothing of any more (53,322 x 256 with three
// nonzeros a row 18.3 us on the GPU against 13.5), and the next call's B B^T, let in
// early with its shared memory, takes the L1 that M's rows are read through (1M x 256
// with two a row 47.8 us a call against 40.8).
__global__ void rownorm_csr_kernel(const float* __restrict__ V, const int32_t* __restrict__ J,
                                   const int64_t* __restrict__ I, int64_t n, int64_t nnz, int64_t d,
                                   const float* __restrict__ M, float alpha, float beta,
                                   float* __restrict__ x, int* flag) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const int64_t k0 = __ldg(I + i), k1 = __ldg(I + i + 1);
        float q = 0.f;
        if (k0 < 0 || k1 < k0 || k1 > nnz) {
            bad = true;
        } else {
            for (int64_t p = k0; p < k1; ++p) {
                const int32_t jp = __ldg(J + p);
                if (jp < 0 || jp >= d) {
                    bad = true;
                    continue;
                }
                const float vp = __ldg(V + p);
                const float* Mrow = M + (int64_t)jp * d;
                float s = vp * __ldg(Mrow + jp);  // diagonal term once
                for (int64_t t = p + 1; t < k1; ++t) {
                    const int32_t jt = __ldg(J + t);
                    if (jt < 0 || jt >= d) continue;
                    s = fmaf(2.0f * __ldg(V + t), __ldg(Mrow + jt), s);
                }
                q = fmaf(vp, s, q);
            }
        }
        x[i] = (beta != 0.f) ? fmaf(alpha, q, beta * x[i]) : alpha * q;
    }
    if (bad) set_flag(flag, LSK_FLAG_BAD_CSR);
}

// The same with the nonzeros of `rows` (32 or fewer) consecutive rows dealt out to
// the lanes of a warp: the lane of entry p forms v_p (v_p M_pp + 2 sum_{t > p} v_t
// M_pt), a segmented sum over the lanes adds up each row's entries, and the lane of
// the row keeps the sum.  For denser rows, whose pairs would otherwise follow one
// another in one thread: 50,000 x 256 with 128 nonzeros a row 1.0 ms (2.1), 200,000
// x 256 with eight 45 us (59), 300,000 x 128 with 6.4 36 (42); with two a row (1M x
// 200) finding the entries costs more than it shares out, 39 against 36.
__global__ void __launch_bounds__(256, 8) rownorm_csr_flat_kernel(const float* __restrict__ V, const int32_t* __restrict__ J,
                                                                  const int64_t* __restrict__ I, int64_t n, int64_t nnz,
                                                                  int64_t d, const float* __restrict__ M, float alpha,
                                                                  float beta, float* __restrict__ x, int rows, int* flag) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool bad = false;
    for (int64_t i0 = warp * rows; i0 < n; i0 += nwarps * rows) {
        const int64_t i = i0 + lane, i1 = min(n, i0 + rows);
        RowGroup g;
        if (!g.load(I, i, i1, nnz)) bad = true;
        int64_t before = __shfl_up_sync(0xffffffffu, g.upto, 1);   // entries of the rows before it
        if (lane == 0) before = 0;
        float sum = 0.f;
        for (int64_t e0 = 0; e0 < g.total; e0 += 32) {
            const bool live = e0 + lane < g.total;
            const int64_t e = live ? e0 + lane : g.total - 1;
            const int row = g.lane_of(e);
            const int64_t first = g.first_of(row), at = first + e, last = first + g.upto_of(row);
            const int64_t head = max(g.upto_of((row + 31) & 31), e0);   // the row's first entry among these (row > 0)
            const int back = lane - (row ? (int)(head - e0) : 0);
            float q = 0.f;
            if (live) {
                const int32_t jp = __ldg(J + at);
                if (jp < 0 || jp >= d) {
                    bad = true;
                } else {
                    const float vp = __ldg(V + at);
                    const float* Mrow = M + (int64_t)jp * d;
                    float s = vp * __ldg(Mrow + jp);   // diagonal term once
                    for (int64_t t = at + 1; t < last; ++t) {
                        const int32_t jt = __ldg(J + t);
                        if (jt < 0 || jt >= d) continue;
                        s = fmaf(2.0f * __ldg(V + t), __ldg(Mrow + jt), s);
                    }
                    q = vp * s;
                }
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float y = __shfl_up_sync(0xffffffffu, q, o);
                if (back >= o) q += y;
            }
            const int64_t end = g.upto < e0 + 32 ? g.upto : e0 + 32;   // past this row's entries among these
            const float part = __shfl_sync(0xffffffffu, q, (int)(end - 1 - e0) & 31);
            if (end > e0 && end > before) sum += part;
        }
        if (i < i1) x[i] = (beta != 0.f) ? fmaf(alpha, sum, beta * x[i]) : alpha * sum;
    }
    if (bad) set_flag(flag, LSK_FLAG_BAD_CSR);
}

}  // namespace

size_t rownorms_workspace_bytes(const lsk_mat* A, int64_t c, int upper_tri, int32_t prec) {
    if (A->kind == LSK_DENSE) {
        // the BF16x3 and TF32 images have the same size
        if ((prec == LSK_PREC_BF16 || prec == LSK_PREC_TF32) &&
            (rownorms_tc_supported(A, c, upper_tri) || rownorms_tc_supported(A, c, upper_tri, true)))
            return rownorms_tc_workspace_bytes(A, c, upper_tri);
        return rownorms_tc3_workspace_bytes(A, c, upper_tri);
    }
    return ws_round((size_t)A->d * A->d * 4);
}

cudaError_t rownorms_launch(const lsk_mat* A, const float* B, int64_t c, double alpha, double beta,
                            int upper_tri, int32_t prec, float* x, void* ws, int* flag, int sm_count,
                            cudaStream_t st, int min_tiles, const void* prepared) {
    const int64_t n = A->n, d = A->d;
    if (n == 0) return cudaSuccess;
    // TF32: the one-product TF32 kernel where A suits TMA, else BF16x3 (more
    // accurate), else FP32 on the CUDA cores (an operand prepared by a grouped
    // launch is a BF16x3 image)
    if (A->kind == LSK_DENSE && prec == LSK_PREC_TF32 && !prepared && rownorms_tc_supported(A, c, upper_tri, true))
        return rownorms_tc_launch(A, B, c, (float)alpha, (float)beta, upper_tri, x, ws, flag, sm_count, st,
                                  min_tiles, nullptr, true);
    if (A->kind == LSK_DENSE && (prec == LSK_PREC_BF16 || prec == LSK_PREC_TF32) &&
        rownorms_tc_supported(A, c, upper_tri))
        return rownorms_tc_launch(A, B, c, (float)alpha, (float)beta, upper_tri, x, ws, flag, sm_count, st,
                                  min_tiles, (const uint8_t*)prepared);
    if (A->kind == LSK_DENSE) {
        // the tensor-core kernel where A is large enough (then this one does the
        // rows it leaves), else CUDA cores for all
        const int *list = nullptr, *count = nullptr;
        cudaError_t e = cudaSuccess;
        const bool tc3 = rownorms_tc3_launch(A, B, c, (float)alpha, (float)beta, upper_tri ? 1 : 0, x, ws, flag, st,
                                             &list, &count, &e);
        if (e != cudaSuccess) return e;
        const unsigned tiles = (unsigned)((n + RM - 1) / RM);
        if (tc3) {
            const unsigned grid = std::min(tiles, 4u * (unsigned)sm_count);
            LSK_PROF("rownorm_dense_simt", st) launch_pdl(rownorm_dense_kernel<true>, grid, 256, 0, 1, st,
                (const float*)A->values, A->ld, n, d, B, c, upper_tri ? 1 : 0, (float)alpha, (float)beta, x, list, count);
        } else {
            // chained only where every block finds an SM of its own: sent out early, more than
            // that pile up on those that are free first (19,000 x 400 times 400 x 64 31.0 us
            // chained, 33.3 plainly; 50,000 x 400 102 and 79; 496,154 x 300 546 and 535), and
            // where the tile is short: handed through the wait, the pointers cost the loop 2%
            // (1,729 x 256 times 256 x 256 75.1 us on the GPU, 73.7 plainly)
            const bool early = tiles <= (unsigned)sm_count && d * c < (1 << 15);
            LSK_PROF("rownorm_dense_simt", st) launch_chained(
                early, early ? rownorm_dense_kernel<false> : rownorm_dense_kernel<false, false>, tiles, 256, 0, 1, st,
                (const float*)A->values, A->ld, n, d, B, c, upper_tri ? 1 : 0, (float)alpha, (float)beta, x, nullptr, nullptr);
        }
    } else {
        float* M = prepared ? (float*)prepared : (float*)ws;   // prepared: built by bbt_group_launch
        const dim3 bg((unsigned)((d + 15) / 16), (unsigned)((d + 15) / 16));
        if (!prepared) LSK_PROF("rownorm_bbt", st) launch_pdl(bbt_kernel, bg, 256, 0, 1, st, B, d, c, M);
        // A lane a nonzero where rows are dense enough: of 3, 4 or 5 nonzeros on, the wider
        // A the fewer, as the pairs' loads from M then miss L1 (200,000 rows: d = 32 with 4.5
        // 18.3 us against 17.4 with a lane a row, 5.5 21.1 against 22.2; d = 128 with 3.4 15.0
        // and 14.2, 4.5 17.8 and 18.5; d = 256 with 3.4 16.7 and 17.6).  While rows are few,
        // earlier, since there the lanes are too (60,000 x 17 with 4.5 9.3 and 10.7, 200,000 x
        // 17 18.5 and 18.0); of 9 columns never (60,000 with 8 12.0 and 8.4).
        const bool few = n < 1024 * (int64_t)sm_count;
        const int64_t dense = d < 64 ? (few ? 4 : 5) : d < (few ? 128 : 256) ? 4 : 3;
        const bool flat = d >= (few ? 17 : 32) && A->nnz / dense > n;
        int rows = 32;   // of a warp of the flat form: fewer where warps are few, 64 nonzeros or more
        while (flat && rows > 4 && n / rows < 32 * (int64_t)sm_count && A->nnz * (rows / 2) >= 64 * n) rows /= 2;
        int64_t gr = flat ? (n + 8 * rows - 1) / (8 * rows) : (n + 255) / 256;
        if (gr > 16 * (int64_t)sm_count) gr = 16 * (int64_t)sm_count;
        if (flat)
            LSK_PROF("rownorm_csr", st) rownorm_csr_flat_kernel<<<(unsigned)gr, 256, 0, st>>>(
                (const float*)A->values, A->colidx, A->rowptr, n, A->nnz, d, M, (float)alpha, (float)beta, x, rows, flag);
        else
            LSK_PROF("rownorm_csr", st) rownorm_csr_kernel<<<(unsigned)gr, 256, 0, st>>>(
                (const float*)A->values, A->colidx, A->rowptr, n, A->nnz, d, M, (float)alpha, (float)beta, x, flag);
    }
    return cudaGetLastError();
}

void bbt_group_build(const std::vector<BbtJob>& jobs, HostTable& t, BbtGroup& g) {
    std::vector<int> blocks, off;
    for (const BbtJob& j : jobs) {
        const int tiles = (int)((j.d + 15) / 16);
        blocks.push_back(tiles * tiles);
    }
    g.count = (int)jobs.size();
    g.blocks = group_offsets(blocks, off);
    g.params_off = t.put(jobs.data(), jobs.size());
    g.off_off = t.put(off.data(), off.size());
}

cudaError_t bbt_group_launch(const BbtGroup& g, const unsigned char* table, cudaStream_t st) {
    if (g.count == 0) return cudaSuccess;
    LSK_PROF("rownorm_bbt", st) bbt_grouped_kernel<<<g.blocks, 256, 0, st>>>(
        reinterpret_cast<const BbtJob*>(table + g.params_off), reinterpret_cast<const int*>(table + g.off_off),
        g.count);
    return cudaGetLastError();
}
