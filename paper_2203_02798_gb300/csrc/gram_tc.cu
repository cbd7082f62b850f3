// gram_tc.cu -- Gram matrix C = alpha A^T A + beta C of a dense A on tcgen05.
//
// The dense form of Alg. 5 / Alg. 7 (rows of A produce partial Gram matrices
// that are then summed), with the partial of a block of rows formed on the
// tensor cores.  Precision: A is split into bfloat16 pairs, a = hi + lo, and
//     A^T A ~= hi^T hi + hi^T lo + lo^T hi        (FP32 accumulation in TMEM)
// (the dropped lo^T lo term is ~2^-17 relative to |a_i||a_j|).
//
// Persistent kernel, one CTA per SM; CTA c takes the slices c, c + grid, ...
// of kSliceRows = 1024 rows each, so no FP32 accumulator sums more than
// 3 x 1024 products (the tensor cores' FP32 accumulation biases long
// all-positive sums, such as the diagonal, at the 1e-5 level by 2048 rows).
// After each slice the epilogue warps read the accumulator out of TMEM, hand
// it back to the MMAs at once, and add it into the CTA's running FP32 partial
// in global memory with fire-and-forget vector reductions (one writer per
// address, in program order, so the sums are deterministic); a second kernel
// adds the CTAs' partials in order with a compensated FP32 sum, then forms
// alpha * sum + beta * C.  Warps:
//   0 .. kWorkers-1
//               workers: each owns every kWorkers-th piece of 8 rows (a
//               quarter of a 32-row chunk) and works alone: 16-byte loads of
//               whole rows, a bf16 hi / lo split, and 8-byte stores into the
//               stage's MN-major tiles (no transpose: a row-major chunk of A
//               is MN-major for both operands of A^T A, the instruction
//               descriptor's transpose bits say so).  The uses of each ring
//               stage are claimed in piece order;
//   kWorkers    lane 0 issues, for each 128-column M tile t, the products
//               with columns 128 t .. npad - 1 as the N operand (the same
//               shared-memory tile is both operands; only the upper block
//               triangle is computed);
//   then 8      epilogue: accumulator t is read by the warps whose TMEM lane
//               quarter covers it.
// TMEM holds the two accumulators (N = npad and npad - 128 columns).  Waits
// are bounded; a timeout sets the TIMEOUT flag.
#include "tc_common.cuh"

#include <algorithm>

namespace {

constexpr int kKC = 32;            // rows of A per chunk (the K of the MMAs)
constexpr int kMT = 128;           // rows of an MMA tile (columns of A)
// warp roles: kWorkers workers, one MMA warp, kEpiWarps epilogue warps
template <int W, int E, int PR = 8>
struct GramShape {
    static constexpr int kPieceRows = PR;   // rows of one worker piece
    static constexpr int kPieces = 32 / PR; // pieces per 32-row chunk
    static constexpr int kWorkers = W;
    static constexpr int kMmaWarp = W;
    static constexpr int kEpi0 = W + 1;
    static constexpr int kEpiWarps = E;   // 4 (both accumulators each) or 8 (one each)
    static constexpr int kThreads = (W + 1 + E) * 32;
};
constexpr int kMaxStages = 8;
constexpr int kSliceRows = 1024;   // rows per slice (FP32 accumulation length bound)
constexpr size_t kSmemLimit = 232448;

struct GrParams {
    const float* A;
    int64_t lda, n;
    int d, npad, slices, vec;   // vec: 16-byte loads
    float* part;       // [gridDim][npad][npad] running partials, zeroed before the launch
    int* flag;
};

// Stage layout, per bf16 tile (hi, then lo): MN-major 128-byte-swizzled atoms
// of 8 rows of A (K) x 64 columns of A (M / N), atom (column block mb, row
// group kg) at mb x 1024 + kg x kSbo(npad).  The column blocks run to a whole
// number of 128-column MMA tiles, so an M = 128 operand never reads past its
// tile (columns past d hold zeros, past npad they feed accumulator rows that
// are never read).
__host__ __device__ constexpr uint32_t mn_blocks(int npad) { return 2u * (uint32_t)((npad + kMT - 1) / kMT); }
__host__ __device__ constexpr uint32_t kSbo(int npad) { return mn_blocks(npad) * 1024u; }   // next 8 rows
__host__ __device__ constexpr uint32_t half_bytes(int npad) { return kSbo(npad) * (kKC / 8); }  // one bf16 tile
__host__ __device__ constexpr uint32_t stage_bytes(int npad) { return 2 * half_bytes(npad); }   // hi + lo
// ring depth that fits next to the barriers
__host__ __device__ constexpr int stages_of(int npad) {
    return (int)((232448 - 2048) / stage_bytes(npad)) < kMaxStages ? (int)((232448 - 2048) / stage_bytes(npad))
                                                                     : kMaxStages;
}

// Rows row0 .. row0 + 7 of A (zeros at and past r_end or d), lane t: float4
// number t + 32 h of each row (columns 4 t + 128 h .. + 3): 512 contiguous
// bytes a row per warp instruction.
template <int NPAD>
__device__ __forceinline__ void load_row(const GrParams& p, int64_t row, int64_t r_end, int lane,
                                         float4 (&v)[(NPAD + kMT - 1) / kMT]) {
    constexpr int H = (NPAD + kMT - 1) / kMT;
    const float* src = p.A + row * p.lda;
#pragma unroll
    for (int h = 0; h < H; ++h) {
        const int c = 4 * lane + kMT * h;
        v[h] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < r_end && c < p.d) {
            if (p.vec && c + 3 < p.d) {
                asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                             : "=f"(v[h].x), "=f"(v[h].y), "=f"(v[h].z), "=f"(v[h].w)
                             : "l"(src + c));
            } else {
                v[h].x = __ldg(src + c);
                v[h].y = c + 1 < p.d ? __ldg(src + c + 1) : 0.f;
                v[h].z = c + 2 < p.d ? __ldg(src + c + 2) : 0.f;
                v[h].w = c + 3 < p.d ? __ldg(src + c + 3) : 0.f;
            }
        }
    }
}
// The eight rows from row0 on, v[r] the row r + turn, modulo 8; rows of whole
// 16-byte quads that are all in range go without per-row checks (the registers of
// lanes past d, zero before, are left as they are).
template <int NPAD>
__device__ __forceinline__ void load_piece_quads(const GrParams& p, int64_t row0, int64_t r_end, int lane, int turn,
                                                 float4 (&v)[8][(NPAD + kMT - 1) / kMT]) {
    constexpr int H = (NPAD + kMT - 1) / kMT;
    if (p.vec && (p.d & 3) == 0 && row0 + 8 <= r_end) {
        const char* const src0 = reinterpret_cast<const char*>(p.A + row0 * p.lda + 4 * lane);
        const int64_t step = p.lda * 4;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const char* const src = src0 + ((r + turn) & 7) * step;
#pragma unroll
            for (int h = 0; h < H; ++h)
                if (4 * lane + kMT * h < p.d)
                    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                                 : "=f"(v[r][h].x), "=f"(v[r][h].y), "=f"(v[r][h].z), "=f"(v[r][h].w)
                                 : "l"(src + 4 * kMT * h));
        }
    } else {
#pragma unroll
        for (int r = 0; r < 8; ++r) load_row<NPAD>(p, row0 + ((r + turn) & 7), r_end, lane, v[r]);
    }
}
template <int NPAD, int PR>
__device__ __forceinline__ void load_piece(const GrParams& p, int64_t row0, int64_t r_end, int lane,
                                           float4 (&v)[PR][(NPAD + kMT - 1) / kMT]) {
#pragma unroll
    for (int r = 0; r < PR; ++r) load_row<NPAD>(p, row0 + r, r_end, lane, v[r]);
}

// Split the piece into bf16 hi / lo and store it as rows PR part .. PR part +
// PR - 1 of the chunk: row k of the chunk is row k % 8 of the atoms of row
// group k / 8; columns 4 t .. 4 t + 3 go to atom (c / 64, k / 8), 16-byte
// chunk ((c % 64) / 8) ^ (k % 8), bytes 8 (t % 2) .. +7.  Sixteen lanes fill
// one 128-byte atom row: two wavefronts a warp instruction.
template <int NPAD, int PR>
__device__ __forceinline__ void store_piece(uint8_t* th, uint8_t* tl, int part, int lane,
                                            const float4 (&v)[PR][(NPAD + kMT - 1) / kMT]) {
    constexpr int H = (NPAD + kMT - 1) / kMT;
    const uint32_t c0 = 4u * (uint32_t)lane;
    const uint32_t k0 = (uint32_t)(PR * part);
    uint8_t* const bh = th + (k0 >> 3) * kSbo(NPAD);
    uint8_t* const bl = tl + (k0 >> 3) * kSbo(NPAD);
#pragma unroll
    for (int r = 0; r < PR; ++r) {
        const uint32_t rr = (k0 & 7u) + (uint32_t)r;   // row in the atom
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const uint32_t c = c0 + kMT * h;
            const uint32_t off = (c >> 6) * 1024u + rr * 128u + (((((c & 63u) >> 3) ^ rr) & 7u) << 4) + (c & 7u) * 2u;
            uint2 hi, lo;
            tc::split_bf16x2(v[r][h].x, v[r][h].y, hi.x, lo.x);
            tc::split_bf16x2(v[r][h].z, v[r][h].w, hi.y, lo.y);
            *reinterpret_cast<uint2*>(bh + off) = hi;
            *reinterpret_cast<uint2*>(bl + off) = lo;
        }
    }
}

// NPAD (d rounded up to 32) is a template parameter: every index split below
// is then a division by a constant.
template <int NPAD, class SH>
__global__ void __launch_bounds__(SH::kThreads, 1) gram_tc_kernel(const GrParams p) {
    constexpr int kWorkers = SH::kWorkers, kMmaWarp = SH::kMmaWarp, kEpi0 = SH::kEpi0, kEpiWarps = SH::kEpiWarps;
    constexpr int kPieceRows = SH::kPieceRows, kPieces = SH::kPieces;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int kStages = stages_of(NPAD);
    const uint32_t sbytes = stage_bytes(NPAD);
    uint8_t* stages = smem;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * sbytes);
    uint64_t* full = bars;                 // [kStages] (kPieces arrivals)
    uint64_t* empty = bars + kStages;      // [kStages] (MMA commit)
    uint64_t* done = bars + 2 * kStages;   // slice accumulated       (MMA commit)
    uint64_t* drained = done + 1;          // accumulator read        (epilogue warp arrivals)
    uint64_t* fin = done + 2;              // every MMA complete      (MMA commit)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* stored = const_cast<int*>(abort) + 1;   // [kStages] pieces stored per stage (in use order)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int ntiles = (NPAD + kMT - 1) / kMT;   // 1 or 2 M tiles
    const int nepi = 4 * (ntiles < kEpiWarps / 4 ? ntiles : kEpiWarps / 4);   // epilogue warps in use
    const int my_slices = ((int)blockIdx.x < p.slices) ? (p.slices - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(full + s, kPieces);
            tc::mbar_init(empty + s, 1);
            stored[s] = 0;
        }
        tc::mbar_init(done, 1);
        tc::mbar_init(drained, nepi);
        tc::mbar_init(fin, 1);
        *abort = 0;
        tc::fence_mbar_init();
    }
    // accumulator t at column 256 t: N = npad (t = 0), npad - 128 (t = 1)
    constexpr uint32_t tcols = ntiles == 2 ? 512u : NPAD <= 32 ? 32u : NPAD <= 64 ? 64u : 128u;
    if (warp == kMmaWarp) {
        tc::tmem_alloc(tmem_slot, tcols);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    if (warp < kWorkers) {
        // the CTA's chunks in order: slice z (rows from (blockIdx.x + z grid)
        // 1024) holds chunks 32 z .. 32 z + 31; only the matrix's last slice
        // is short
        int my_chunks = my_slices * (kSliceRows / kKC);
        if (my_slices > 0 && (int)blockIdx.x + (my_slices - 1) * (int)gridDim.x == p.slices - 1) {
            const int64_t last_rows = p.n - (int64_t)(p.slices - 1) * kSliceRows;
            my_chunks -= kSliceRows / kKC - (int)((last_rows + kKC - 1) / kKC);
        }
        constexpr int H = (NPAD + kMT - 1) / kMT;
        const int npieces = my_chunks * kPieces;
        // piece pc: chunk h = pc / kPieces of the CTA's sequence, rows
        // kPieceRows (pc % kPieces) .. of it
        const auto rows_of = [&](int pc, int64_t& row0, int64_t& r_end) {
            const int h = pc / kPieces;
            const int z = h / (kSliceRows / kKC), cz = h % (kSliceRows / kKC);
            const int64_t r_begin = ((int64_t)blockIdx.x + (int64_t)z * gridDim.x) * kSliceRows;
            r_end = min(p.n, r_begin + kSliceRows);
            row0 = r_begin + (int64_t)cz * kKC + (pc % kPieces) * kPieceRows;
        };
        // claim piece pc's stage (in piece order), store it, arrive
        const auto put = [&](int pc, const float4 (&v)[kPieceRows][H]) -> bool {
            const int h = pc / kPieces, s = h % kStages, u = h / kStages;
            int ok = 1;
            if (lane == 0) {
                ok = tc::counter_wait(reinterpret_cast<volatile int*>(stored + s), kPieces * u, abort) &&
                     tc::mbar_wait(empty + s, ((uint32_t)u & 1u) ^ 1u, abort);
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
            uint8_t* th = stages + (size_t)s * sbytes;
            store_piece<NPAD, kPieceRows>(th, th + half_bytes(NPAD), pc % kPieces, lane, v);
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tc::mbar_arrive(full + s);
                atomicAdd(stored + s, 1);
            }
            return true;
        };
        // one piece in registers: load it, claim its stage, store it (two
        // 4-row pieces in flight a warp measured no faster)
        int64_t row0, r_end;
        float4 v[kPieceRows][H];
        for (int pc = warp; pc < npieces; pc += kWorkers) {
            rows_of(pc, row0, r_end);
            load_piece<NPAD, kPieceRows>(p, row0, r_end, lane, v);
            if (!put(pc, v)) break;
        }
    } else if (warp == kMmaWarp) {
        // the whole warp goes along and an elected lane issues, so that the
        // descriptors stay in uniform registers
        const uint64_t d0 = tc::desc_sw128_mnmajor(tc::smem_u32(stages), 1024u, kSbo(NPAD));
        bool okm = true;
        int s = 0;
        uint32_t ph = 0;
        for (int z = 0; z < my_slices && okm; ++z) {
            const int64_t r_begin = ((int64_t)blockIdx.x + (int64_t)z * gridDim.x) * kSliceRows;
            const int64_t r_end = min(p.n, r_begin + kSliceRows);
            const int nchunks = (int)((r_end - r_begin + kKC - 1) / kKC);
            // the previous slice's accumulator has been read out
            if (z > 0) okm = __all_sync(0xffffffffu, tc::mbar_wait(drained, (uint32_t)(z - 1) & 1u, abort));
            tc::fence_after_sync();
            for (int g = 0; g < nchunks && okm; ++g) {
                okm = __all_sync(0xffffffffu, tc::mbar_wait(full + s, ph, abort));
                if (!okm) break;
                tc::fence_after_sync();
                if (tc::elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < kKC / 16; ++kk) {
                        // 16 rows = two 8-row groups
                        const uint64_t dk = d0 + (((uint32_t)s * sbytes + 2u * kSbo(NPAD) * kk) >> 4);
#pragma unroll
                        for (int t = 0; t < ntiles; ++t) {
                            const uint32_t idesc = tc::idesc_bf16_f32_mn(128, (uint32_t)(NPAD - t * kMT));
                            const uint32_t dt = tmem + 256u * t;
                            const uint64_t dh = dk + (t * 2048u >> 4), dl = dh + (half_bytes(NPAD) >> 4);   // columns from 128 t
                            tc::mma_bf16(dt, dh, dh, idesc, (g | kk) != 0);
                            tc::mma_bf16(dt, dh, dl, idesc, 1);
                            tc::mma_bf16(dt, dl, dh, idesc, 1);
                        }
                    }
                    tc::mma_commit(empty + s);
                    if (g + 1 == nchunks) tc::mma_commit(done);
                }
                __syncwarp();
                if (++s == kStages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
        if (tc::elect_one()) tc::mma_commit(fin);
        __syncwarp();
        volatile int never = 0;
        tc::mbar_wait(fin, 0, &never);
        __syncwarp();
    } else if (warp - kEpi0 < nepi) {
        // epilogue warp e: TMEM lane quarter q = warp % 4, accumulators
        // t = e / 4, e / 4 + nepi / 4, ...
        const int e = warp - kEpi0, q = warp & 3;
        for (int z = 0; z < my_slices; ++z) {
            int okw = 0;
            if (lane == 0) okw = tc::mbar_wait(done, (uint32_t)z & 1u, abort) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, okw, 0)) break;
            tc::fence_after_sync();
            // the accumulator is handed back as soon as it is in registers; the
            // adds into the running partial are fire-and-forget reductions (one
            // writer per address, in program order: deterministic)
            for (int t = e >> 2; t < ntiles; t += nepi >> 2) {
                const int row = t * kMT + q * 32 + lane;   // column a of A
                const int ncols = NPAD - t * kMT;        // columns b = t*128 .. npad-1
                // by columns: a warp's 32 rows are one 128-byte line
                float* dst = p.part + ((int64_t)blockIdx.x * NPAD + t * kMT) * NPAD + row;
                // 64 columns per TMEM round trip (ncols is a multiple of 32)
                for (int col = 0; col < ncols; col += 64) {
                    uint32_t va[32], vb[32];
                    const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(256 * t + col);
                    const bool two = col + 32 < ncols;
                    tc::tmem_ld_32x32b_x32(ta, va);
                    if (two) tc::tmem_ld_32x32b_x32(ta + 32u, vb);
                    tc::tmem_ld_wait();
                    if (t + (nepi >> 2) >= ntiles && col + 64 >= ncols) {
                        tc::fence_before_sync();
                        __syncwarp();
                        if (lane == 0) tc::mbar_arrive(drained);
                    }
                    if (row < p.d) {
#pragma unroll
                        for (int k = 0; k < 64; ++k)
                            if (k < 32 || two)
                                asm volatile("red.global.add.f32 [%0], %1;" ::"l"(dst + (int64_t)(col + k) * NPAD),
                                             "f"(__uint_as_float(k < 32 ? va[k] : vb[k - 32])) : "memory");
                    }
                }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, tcols);
    }
    if (threadIdx.x == 0 && *abort) set_flag(p.flag, LSK_FLAG_TIMEOUT);
}

// C[a][b] = alpha * sum_c part[c][min][max] + beta * C[a][b]: the CTAs'
// partials in order, compensated FP32 sum (Neumaier), alpha and beta in FP64.
__global__ void gram_tc_reduce_kernel(const float* __restrict__ part, int slices, int d, int npad, double alpha,
                                      double beta, float* __restrict__ C) {
    const int64_t len = (int64_t)d * d, plen = (int64_t)npad * npad;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < len; e += stride) {
        int b = (int)(e / d), a = (int)(e % d);   // C[b][a] (symmetric)
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int64_t idx = (int64_t)b * npad + a;   // the partial's columns, a <= b
        float s = 0.f, c = 0.f;
        for (int z = 0; z < slices; ++z) {
            const float x = part[(int64_t)z * plen + idx];
            const float t = s + x;
            c += (fabsf(s) >= fabsf(x)) ? (s - t) + x : (x - t) + s;
            s = t;
        }
        double v = alpha * ((double)s + (double)c);
        if (beta != 0.0) v += beta * (double)C[e];
        C[e] = (float)v;
    }
}

size_t smem_bytes(int npad) {
    return (size_t)stages_of(npad) * stage_bytes(npad) + 1024 + 256;
}

}  // namespace

bool gram_tc_supported(const lsk_mat* A) {
    return A->kind == LSK_DENSE && A->d >= 1 && A->d <= 256 && smem_bytes((int)((A->d + 31) / 32) * 32) <= kSmemLimit;
}

template <int NPAD, class SH>
cudaError_t launch_shape(const GrParams& p, int grid, cudaStream_t st) {
    const size_t smem = smem_bytes(NPAD);
    cudaError_t e = allow_dynamic_smem(gram_tc_kernel<NPAD, SH>);
    if (e != cudaSuccess) return e;
    LSK_PROF("gram_tc", st) gram_tc_kernel<NPAD, SH><<<grid, SH::kThreads, smem, st>>>(p);
    return cudaGetLastError();
}
// 15 workers and 4 epilogue warps (each reading both accumulators): 640
// threads, 96 registers a thread (11 workers with 8 epilogue warps measured
// 1.3% slower at 4M x 256)
template <int NPAD>
cudaError_t launch_npad(const GrParams& p, int grid, cudaStream_t st) {
    return launch_shape<NPAD, GramShape<15, 4>>(p, grid, st);
}

// one running partial per CTA of the persistent grid
int grid_of(const lsk_mat* A, int sm_count) {
    const int64_t slices = (A->n + kSliceRows - 1) / kSliceRows;
    return (int)(slices < sm_count ? slices : sm_count);
}

size_t gram_tc_workspace_bytes(const lsk_mat* A, int sm_count) {
    const int g = grid_of(A, sm_count);
    const size_t npad = (size_t)((A->d + 31) / 32) * 32;
    return ws_round((size_t)(g > 0 ? g : 1) * npad * npad * 4);
}

cudaError_t gram_tc_launch(const lsk_mat* A, double alpha, double beta, float* C, void* ws, int* flag, int sm_count,
                           cudaStream_t st) {
    if (!gram_tc_supported(A)) return cudaErrorNotSupported;
    GrParams p;
    p.A = (const float*)A->values;
    p.lda = A->ld;
    p.n = A->n;
    p.d = (int)A->d;
    p.npad = (int)((A->d + 31) / 32) * 32;
    p.slices = (int)((A->n + kSliceRows - 1) / kSliceRows);
    p.vec = (A->ld % 4 == 0) && (((uintptr_t)A->values & 15) == 0);
    p.part = (float*)ws;
    p.flag = flag;
    const int grid = grid_of(A, sm_count);
    const int64_t len = A->d * A->d;
    int64_t rg = (len + 255) / 256;
    if (rg > 8 * (int64_t)sm_count) rg = 8 * (int64_t)sm_count;
    cudaError_t e;
    if (grid > 0) {
        e = cudaMemsetAsync(p.part, 0, (size_t)grid * p.npad * p.npad * 4, st);
        if (e != cudaSuccess) return e;
        switch (p.npad) {
            case 32: e = launch_npad<32>(p, grid, st); break;
            case 64: e = launch_npad<64>(p, grid, st); break;
            case 96: e = launch_npad<96>(p, grid, st); break;
            case 128: e = launch_npad<128>(p, grid, st); break;
            case 160: e = launch_npad<160>(p, grid, st); break;
            case 192: e = launch_npad<192>(p, grid, st); break;
            case 224: e = launch_npad<224>(p, grid, st); break;
            default: e = launch_npad<256>(p, grid, st); break;
        }
        if (e != cudaSuccess) return e;
    }
    LSK_PROF("gram_reduce", st) gram_tc_reduce_kernel<<<(unsigned)rg, 256, 0, st>>>(p.part, grid, p.d, p.npad, alpha, beta, C);
    return cudaGetLastError();
}

namespace {

// ---- the FP32 form -------------------------------------------------------------
// C to FP32 accuracy from bf16 products.  Every entry is split as
//     x = hi + mid + lo,   hi = x rounded to a multiple of the column's unit,
//                          mid, lo = bf16 roundings of what is left,
// where the unit is a power of two a fixed number of bits below the column's
// largest recent entry.  hi then has at most eight significant bits and the
// sums of hi hi over a segment of rows are whole numbers of units^2 up to 2^24:
// exact in the FP32 accumulator, so the tensor pipe's accumulation, which rounds
// toward zero, has nothing to round there.  This is the error-free splitting of
// Ozaki, Ogita, Oishi & Rump (Numer. Algorithms 59, 2012) with the first slice
// on a fixed grid.  The other products but lo lo (hi mid, hi lo, mid lo, both
// ways round, and mid mid) go to a second accumulator, a small part of the
// first, where that rounding no longer matters.  The unit is only a choice of
// rounding: an entry above the maximum seen (the first rows of the CTA, then a
// quarter of each segment and of the one before, or, where these show none, the
// largest ever) costs exactness in its segment, no more.  Warps note what they see
// while others split, so that equal calls may differ in the last bits.  Entries below
// 2^-8 of their column's unit keep 16 bits: the error is small against the norms
// of the two columns, but not entry by entry against sum |a_ij a_ik|.  A CTA adds up
// to kChain segments in FP32, the two accumulators apart, and starts another partial
// for the next ones, so that the error does not grow with its rows (offset entries,
// 16M x 64, 103 segments: 2.2e-8 in one chain, 1.8e-8 in five; CUDA cores 1.8e-8); all
// partials are summed with compensation.  Frobenius errors against FP64: 1.9e-8 at
// 1M x 256 (2.9e-8 for the CUDA-core kernel; storing C in FP32 alone costs 1.85e-8),
// 4.5e-8 against 2.5e-7 with five rows scaled x100.  A column below 2^-48 (its
// small products would leave FP32's range) or a diagonal whose sum might leave it
// sets *redo, and the CUDA-core kernel, which adds up in FP64, forms C.
//
// Work: a job is a 128-column panel of C's rows against the columns from the
// panel's first on (d > 128: two jobs, N = npad and npad - 128; the SMs are
// shared out by N), so each CTA's two accumulators (2 N <= 512 columns) fill
// its TMEM.  Each CTA takes a contiguous range of rows.  At 1M x 256
// the eight products over the block triangle are 0.41 ms of the tensor pipe's
// measured rate; the call takes 0.57 to 0.60 ms, this kernel 0.55 of it (CUDA cores:
// 4.20), bound by shared-memory bandwidth (the MMAs' operands and the workers' stores keep its data pipe
// full).  What it took: MMAs issued by an elected lane of a warp that runs
// along, so that the descriptors stay in uniform registers (else issue takes 120
// cycles an MMA), few flushes, and partials stored by columns.

// Unit and segment.  Segments of seg_chunks 32-row chunks are summed in TMEM,
// then added to the CTA's partial in FP32.  With the column's maximum at
// 128 .. 256 units a segment of 256 rows stays exact, with 64 .. 128 units one of
// 1,024.  Up to 1,024 rows a CTA take the finer unit (few rows to average the
// roundings of lo over); more rows the longer segments, since every flush of
// the accumulators costs L2 reductions (1.5 GB of them at 1M x 256 with 256-row
// segments: 0.13 ms).
constexpr int kChain = 24, kMaxSlabs = 64;   // (2.5 GB of partials at most)
struct Gr3Params {
    GrParams a;          // A, lda, n, d, vec, part, flag
    int chunks;          // 32-row chunks of A
    int ctas[2];         // CTAs of the two jobs (ctas[1] = 0 for d <= 128)
    int seg_chunks;
    int slabs, chain;    // partials a CTA, and the segments of each
    uint32_t magic_add;  // exponent of 1.5 * 2^23 units above the column maximum's, and the 1.5
    int* redo;
};

__host__ __device__ constexpr uint32_t stage3_bytes(int npad) { return 3 * half_bytes(npad); }
__host__ __device__ constexpr int stages3_of(int npad) {
    return (int)((232448 - 6144) / stage3_bytes(npad)) < kMaxStages ? (int)((232448 - 6144) / stage3_bytes(npad)) : kMaxStages;
}
__host__ __device__ constexpr uint32_t tmem3_cols(int npad) { return npad <= 32 ? 64u : npad <= 64 ? 128u : npad <= 128 ? 256u : 512u; }
// FP32 words of one partial: two planes of 128 x N
__host__ __device__ constexpr size_t part3_floats(int npad) { return 2u * kMT * (size_t)npad; }

// two FP32 additions in one instruction (the low word is the first of the pair)
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

// The three bf16 terms of the pair v; m: 1.5 * 2^23 units of its columns
// (x + m has x's nearest multiple of the unit in its low bits).
__device__ __forceinline__ void split3_grid(float2 v, float2 m, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
    hi = to_bf16x2(add2(add2(v, m), make_float2(-m.x, -m.y)));
    const float2 r = add2(v, neg_bf16x2(hi));
    mid = to_bf16x2(r);
    lo = to_bf16x2(add2(r, neg_bf16x2(mid)));
}

// 1.5 * 2^23 units for a column whose largest |entry| has these bits (add: magic_add)
__device__ __forceinline__ float unit_magic(uint32_t max_bits, uint32_t add) {
    return __uint_as_float((max_bits & 0x7F800000u) + add);
}
__device__ __forceinline__ uint4 ld_shared4(const uint32_t* p) {
    uint4 v;
    asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(tc::smem_u32(p)));
    return v;
}
// where the rows of chunk c's pieces begin in a lane's registers: the two rows that
// are looked at (store_piece3) are other ones from chunk to chunk, so that no
// pattern of rows hides from them
__device__ __forceinline__ int turn_of(int c) { return (int)(((uint32_t)c * 0x9E3779B1u) >> 30) * 2; }
__device__ __forceinline__ uint32_t max_abs_bf16x2(uint32_t m, uint32_t h) {   // per half: max(m, |h|), m >= 0
    const __nv_bfloat162 r = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&m), __habs2(*reinterpret_cast<__nv_bfloat162*>(&h)));
    return *reinterpret_cast<const uint32_t*>(&r);
}

// Split a piece and store it as row group `part` of the stage's three tiles;
// mx[h]: the largest |hi| of the lane's columns (bf16 pairs) in its first two rows.
template <int NPAD>
__device__ __forceinline__ void store_piece3(uint8_t* tile, int part, int lane, const float4 (&v)[8][(NPAD + kMT - 1) / kMT],
                                             const float4 (&mg)[(NPAD + kMT - 1) / kMT], uint2 (&mx)[(NPAD + kMT - 1) / kMT]) {
    constexpr int H = (NPAD + kMT - 1) / kMT;
    const uint32_t c0 = 4u * (uint32_t)lane;
    uint8_t* const b = tile + (uint32_t)part * kSbo(NPAD);
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const uint32_t c = c0 + kMT * h;
            const uint32_t off = (c >> 6) * 1024u + r * 128u + (((((c & 63u) >> 3) ^ (uint32_t)r) & 7u) << 4) + (c & 7u) * 2u;
            uint2 hi, mid, lo;
            split3_grid(make_float2(v[r][h].x, v[r][h].y), make_float2(mg[h].x, mg[h].y), hi.x, mid.x, lo.x);
            split3_grid(make_float2(v[r][h].z, v[r][h].w), make_float2(mg[h].z, mg[h].w), hi.y, mid.y, lo.y);
            if (r < 2) {
                mx[h].x = max_abs_bf16x2(r ? mx[h].x : 0u, hi.x);
                mx[h].y = max_abs_bf16x2(r ? mx[h].y : 0u, hi.y);
            }
            *reinterpret_cast<uint2*>(b + off) = hi;
            *reinterpret_cast<uint2*>(b + half_bytes(NPAD) + off) = mid;
            *reinterpret_cast<uint2*>(b + 2 * half_bytes(NPAD) + off) = lo;
        }
}

// One CTA of a job: the panel of p's first 128 columns against all of p's
// columns (NPAD of them, padded), 32-row chunks [g0, g1), partial into `part`.
template <int NPAD, class SH>
__device__ __forceinline__ void gram_tc3_body(const GrParams& p, const Gr3Params& q, int g0, int g1, float* part, uint8_t* smem) {
    constexpr int kWorkers = SH::kWorkers, kMmaWarp = SH::kMmaWarp;
    constexpr int H = (NPAD + kMT - 1) / kMT;
    constexpr int kStages = stages3_of(NPAD);
    constexpr uint32_t sbytes = stage3_bytes(NPAD);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * sbytes);
    uint64_t* full = bars;                 // [kStages] (4 arrivals: the pieces of a chunk)
    uint64_t* empty = bars + kStages;      // [kStages] (MMA commit)
    uint64_t* done = bars + 2 * kStages;   // segment accumulated     (MMA commit)
    uint64_t* drained = done + 1;          // accumulators read       (4 epilogue warps)
    uint64_t* fin = done + 2;              // every MMA complete      (MMA commit)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    uint32_t* cmax = reinterpret_cast<uint32_t*>(smem + kStages * sbytes + 1024);   // largest |entry| of the columns, as bits:
                                                                                    // [2] segments (even, odd), [1] earlier ones
    static_assert(2 * kMaxStages * 8 + 64 <= 1024, "the barriers fit before the maxima");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nchunks = g1 - g0, nseg = (nchunks + q.seg_chunks - 1) / q.seg_chunks;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            tc::mbar_init(full + s, 4);
            tc::mbar_init(empty + s, 1);
        }
        tc::mbar_init(done, 1);
        tc::mbar_init(drained, 4);
        tc::mbar_init(fin, 1);
        *abort = 0;
        tc::fence_mbar_init();
    }
    constexpr int kCols = kMT * H;
    for (int j = threadIdx.x; j < 3 * kCols; j += SH::kThreads) cmax[j] = 0u;
    if (warp == kMmaWarp) {
        tc::tmem_alloc(tmem_slot, tmem3_cols(NPAD));
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;

    // Worker w owns rows 8 (w % 4) .. of the chunks w / 4, w / 4 + 4, ...: a piece
    // in registers (two where they fit), the next one's loads in flight.
    constexpr int NB = H == 1 ? 2 : 1;
    float4 v[NB][8][H];
    const int grp = warp & 3, c0 = warp >> 2;
    const int64_t row_base = (int64_t)g0 * kKC + grp * 8, r_end = min(p.n, (int64_t)g1 * kKC);
    if (warp < kWorkers) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
#pragma unroll
            for (int r = 0; r < 8; ++r)
#pragma unroll
                for (int h = 0; h < H; ++h) v[b][r][h] = make_float4(0.f, 0.f, 0.f, 0.f);
            load_piece_quads<NPAD>(p, row_base + (int64_t)(c0 + 4 * b) * kKC, r_end, lane, turn_of(c0 + 4 * b), v[b]);
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {   // the first rows give the columns' units
            float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 t = v[0][i][h];
                m.x = fmaxf(m.x, fabsf(t.x));
                m.y = fmaxf(m.y, fabsf(t.y));
                m.z = fmaxf(m.z, fabsf(t.z));
                m.w = fmaxf(m.w, fabsf(t.w));
            }
            uint32_t* c = cmax + 4 * lane + kMT * h;
            atomicMax(c, __float_as_uint(m.x));
            atomicMax(c + 1, __float_as_uint(m.y));
            atomicMax(c + 2, __float_as_uint(m.z));
            atomicMax(c + 3, __float_as_uint(m.w));
        }
    }
    __syncthreads();

    if (warp < kWorkers) {
        uint32_t* const cm = cmax + 4 * lane;
        // split row group `grp` of chunk c into its stage
        const auto put = [&](int c, const float4 (&t)[8][H]) -> bool {
            const int z = c / q.seg_chunks;   // the unit: the largest entry of this segment so far and of the last
            uint32_t* const cur = cm + (z & 1) * kCols;
            uint32_t* const last = cm + (~z & 1) * kCols;
            if (z > 0 && c % q.seg_chunks == 0 && grp == 0)
#pragma unroll
                for (int i = 0; i < H; ++i)
#pragma unroll
                    for (int k = 0; k < 4; ++k) atomicMax(cm + 2 * kCols + kMT * i + k, atomicExch(cur + kMT * i + k, 0u));
            float4 mg[H];
            uint2 mx[H];
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const uint4 b = ld_shared4(cur + kMT * i), d = ld_shared4(last + kMT * i);   // other warps may be raising these
                uint4 u = make_uint4(max(b.x, d.x), max(b.y, d.y), max(b.z, d.z), max(b.w, d.w));
                if (!u.x || !u.y || !u.z || !u.w) {
                    const uint4 o = ld_shared4(cm + 2 * kCols + kMT * i);
                    u = make_uint4(u.x ? u.x : o.x, u.y ? u.y : o.y, u.z ? u.z : o.z, u.w ? u.w : o.w);
                }
                mg[i] = make_float4(unit_magic(u.x, q.magic_add), unit_magic(u.y, q.magic_add), unit_magic(u.z, q.magic_add),
                                    unit_magic(u.w, q.magic_add));
            }
            const int s = c % kStages;
            int okl = 1;
            if (lane == 0) okl = tc::mbar_wait(empty + s, ((uint32_t)(c / kStages) & 1u) ^ 1u, abort) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, okl, 0)) return false;
            store_piece3<NPAD>(smem + (size_t)s * sbytes, grp, lane, t, mg, mx);
            tc::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(full + s);
#pragma unroll
            for (int i = 0; i < H; ++i) {   // tell the other warps (a quarter of the rows look)
                const uint4 b = ld_shared4(cur + kMT * i);
                const uint32_t m[4] = {mx[i].x << 16, mx[i].x & 0xFFFF0000u, mx[i].y << 16, mx[i].y & 0xFFFF0000u};
                const uint32_t o[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (m[k] > o[k]) atomicMax(cur + kMT * i + k, m[k]);
            }
            return true;
        };
        for (int c = c0; c < nchunks; c += 4 * NB) {
            if (!put(c, v[0])) break;
            load_piece_quads<NPAD>(p, row_base + (int64_t)(c + 4 * NB) * kKC, r_end, lane, turn_of(c + 4 * NB), v[0]);
            if constexpr (NB == 2) {
                if (c + 4 >= nchunks || !put(c + 4, v[1])) break;
                load_piece_quads<NPAD>(p, row_base + (int64_t)(c + 12) * kKC, r_end, lane, turn_of(c + 12), v[1]);
            }
        }
    } else {
        // Accumulator warps: TMEM lane quarter warp % 4 (rows of the panel);
        // lane 0 of the first also issues the MMAs (the accumulators fill TMEM,
        // so a segment's MMAs start when the last one's sums are read out).
        const uint32_t base = tc::smem_u32(smem);
        constexpr uint32_t idesc = tc::idesc_bf16_f32_mn(128, (uint32_t)NPAD);
        const uint32_t acc0 = tmem, acc1 = tmem + (uint32_t)NPAD;
        const int quarter = warp & 3, row = quarter * 32 + lane;
        float diag = 0.f;   // of this CTA's rows so far
        bool okm = true;
        int s = 0;
        uint32_t ph = 0;
        // the descriptors of stage 0, first 16 rows; the others differ in the
        // start address alone (16-byte units, bits 0 .. 13)
        const uint64_t d0 = tc::desc_sw128_mnmajor(base, 1024u, kSbo(NPAD));
        for (int z = 0; z < nseg; ++z) {
            if (warp == kMmaWarp) {   // the whole warp goes along, so descriptors stay in uniform registers
                if (z > 0) okm = tc::mbar_wait(drained, (uint32_t)(z - 1) & 1u, abort);
                tc::fence_after_sync();
                const int ng = min(q.seg_chunks, nchunks - z * q.seg_chunks);
                for (int g = 0; g < ng && okm; ++g) {
                    okm = __all_sync(0xffffffffu, tc::mbar_wait(full + s, ph, abort));
                    if (!okm) break;
                    tc::fence_after_sync();
                    if (tc::elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < kKC / 16; ++kk) {
                            // 16 rows = two 8-row groups
                            const uint64_t dh = d0 + (((uint32_t)s * sbytes + 2u * kSbo(NPAD) * kk) >> 4);
                            const uint64_t dm = dh + (half_bytes(NPAD) >> 4), dl = dm + (half_bytes(NPAD) >> 4);
                            tc::mma_bf16(acc0, dh, dh, idesc, (g | kk) != 0);
                            tc::mma_bf16(acc1, dh, dm, idesc, (g | kk) != 0);
                            tc::mma_bf16(acc1, dm, dh, idesc, 1);
                            tc::mma_bf16(acc1, dh, dl, idesc, 1);
                            tc::mma_bf16(acc1, dl, dh, idesc, 1);
                            tc::mma_bf16(acc1, dm, dm, idesc, 1);
                            tc::mma_bf16(acc1, dm, dl, idesc, 1);
                            tc::mma_bf16(acc1, dl, dm, idesc, 1);
                        }
                        tc::mma_commit(empty + s);
                        if (g + 1 == ng) tc::mma_commit(done);
                    }
                    __syncwarp();
                    if (++s == kStages) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            int okw = okm;
            if (lane == 0 && okm) okw = tc::mbar_wait(done, (uint32_t)z & 1u, abort) ? 1 : 0;
            if (!__shfl_sync(0xffffffffu, okw, 0)) break;
            tc::fence_after_sync();
            const int slab = z / q.chain;
            const bool first = slab * q.chain == z;
            for (int col = 0; col < NPAD; col += 32) {
                uint32_t va[32], vb[32];
                const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)col;
                tc::tmem_ld_32x32b_x32(ta, va);
                tc::tmem_ld_32x32b_x32(ta + (uint32_t)NPAD, vb);
                tc::tmem_ld_wait();
                if (col == quarter * 32) {
                    // the diagonal, which bounds every sum of its row and column: the
                    // CTAs' (some 300 at most) stay within FP32's range below 2^117 each
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (i == lane) diag += __uint_as_float(va[i]) + __uint_as_float(vb[i]);
                    if (!(diag <= 1.66153499e35f)) atomicOr(q.redo, 1);
                }
                if (col + 32 >= NPAD) {
                    tc::fence_before_sync();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(drained);
                }
                // the partial is stored by columns: a warp's 32 rows are one
                // 128-byte line (row-major v4 reductions, a line a lane, took
                // 7,700 cycles a flush at N = 128)
                float* dst = part + (size_t)slab * part3_floats(NPAD) + (size_t)col * kMT + row;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (first) {   // (one thread an address: the first segment stores, later ones add)
                        dst[i * kMT] = __uint_as_float(va[i]);
                        dst[(NPAD + i) * kMT] = __uint_as_float(vb[i]);
                    } else {
                        asm volatile("red.global.add.f32 [%0], %1;" ::"l"(dst + i * kMT), "f"(__uint_as_float(va[i])) : "memory");
                        asm volatile("red.global.add.f32 [%0], %1;" ::"l"(dst + (NPAD + i) * kMT), "f"(__uint_as_float(vb[i])) : "memory");
                    }
                }
            }
        }
        for (int y = (nseg + q.chain - 1) / q.chain; y < q.slabs; ++y)   // (a CTA of fewer segments than others)
            for (int i = 0; i < 2 * NPAD; ++i) part[(size_t)y * part3_floats(NPAD) + (size_t)i * kMT + row] = 0.f;
        if (warp == kMmaWarp) {   // also when a wait gave up: every MMA issued is complete before TMEM goes
            if (tc::elect_one()) tc::mma_commit(fin);
            __syncwarp();
            volatile int never = 0;
            tc::mbar_wait(fin, 0, &never);
        }
        __syncwarp();
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, tmem3_cols(NPAD));
    }
    for (int j = threadIdx.x; j < kCols; j += SH::kThreads) {
        const uint32_t m = max(max(cmax[j], cmax[kCols + j]), cmax[2 * kCols + j]);
        if (m != 0u && m < 0x27800000u) atomicOr(q.redo, 1);   // below 2^-48
    }
    if (threadIdx.x == 0 && *abort) set_flag(p.flag, LSK_FLAG_TIMEOUT);
}

using Shape3 = GramShape<16, 3>;   // 16 workers, 4 accumulator warps

template <int NPAD>
__global__ void __launch_bounds__(Shape3::kThreads, 1) gram_tc3_kernel(const Gr3Params p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    const int job = (int)blockIdx.x >= p.ctas[0];
    const int64_t c = (int)blockIdx.x - (job ? p.ctas[0] : 0), nc = job ? p.ctas[1] : p.ctas[0];
    const int g0 = (int)(p.chunks * c / nc), g1 = (int)(p.chunks * (c + 1) / nc);
    float* part = p.a.part + p.slabs * (job ? p.ctas[0] * part3_floats(NPAD) + c * part3_floats(NPAD - kMT) : c * part3_floats(NPAD));
    if constexpr (NPAD > kMT) {
        if (job) {
            GrParams b = p.a;
            b.A += kMT;
            b.d -= kMT;
            gram_tc3_body<NPAD - kMT, Shape3>(b, p, g0, g1, part, smem);
            return;
        }
    }
    gram_tc3_body<NPAD, Shape3>(p.a, p, g0, g1, part, smem);
}

// C[a][b] = C[b][a] = alpha sum + beta C for a <= b: a block takes 32
// consecutive entries; thread (g, x) adds both planes of the partials g, g + 8,
// ... of entry x as FP32 pairs, then the 8 group sums are added in order.
template <typename OutT>
__global__ void __launch_bounds__(256) gram_tc3_reduce_kernel(const float* __restrict__ part, int ctas0, int ctas1, int d,
                                                              int npad, const int* __restrict__ redo, double alpha,
                                                              double beta, OutT* __restrict__ C) {
    __shared__ double acc[8][33];
    if (*redo) return;
    const int x = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int e = (int)blockIdx.x * 32 + x;
    const int b = e / d, a = e % d;
    const bool upper = e < d * d && a <= b;
    float s = 0.f, c = 0.f;
    if (upper) {
        const int job = a >= kMT, w = job ? npad - kMT : npad, n = job ? ctas1 : ctas0;   // (partials of all CTAs)
        const size_t one = part3_floats(w), plane = (size_t)kMT * w;
        const float* src = part + (job ? ctas0 * part3_floats(npad) : 0) + (size_t)(b - job * kMT) * kMT + (a - job * kMT);
        for (int z = g; z < n; z += 32) {   // eight loads in flight
            float v[8];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool in = z + 8 * k < n;
                v[2 * k] = in ? src[(z + 8 * k) * one] : 0.f;
                v[2 * k + 1] = in ? src[(z + 8 * k) * one + plane] : 0.f;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) comp_add(s, c, v[k]);
        }
    }
    acc[g][x] = (double)s + (double)c;
    __syncthreads();
    if (g == 0 && upper) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += acc[k][x];
        const double ab = alpha * t;
        C[(size_t)a * d + b] = (OutT)(beta != 0.0 ? ab + beta * (double)C[(size_t)a * d + b] : ab);
        if (a != b) C[(size_t)b * d + a] = (OutT)(beta != 0.0 ? ab + beta * (double)C[(size_t)b * d + a] : ab);
    }
}

struct Gr3Plan {
    int npad, chunks, ctas[2], seg_chunks, slabs, chain;
    size_t part_bytes;
};
// The SMs are shared out between the two jobs by a chunk's cost: 6 N cycles of
// products, or the split of a 128-column panel (some 450) where N is small.
Gr3Plan gram_tc3_plan(const lsk_mat* A, int sm_count) {
    Gr3Plan q{};
    q.npad = (int)((A->d + 31) / 32) * 32;
    q.chunks = (int)((A->n + kKC - 1) / kKC);
    if (q.npad > kMT) {
        const int w0 = 6 * q.npad, w1 = std::max(6 * (q.npad - kMT), 450);
        q.ctas[1] = std::max(1, (sm_count * w1 + (w0 + w1) / 2) / (w0 + w1));
        q.ctas[0] = std::max(1, sm_count - q.ctas[1]);
    } else {
        q.ctas[0] = sm_count;
    }
    for (int j = 0; j < 2; ++j) q.ctas[j] = std::min(q.ctas[j], q.chunks);
    q.seg_chunks = q.chunks <= 32 * q.ctas[0] ? 8 : 32;   // (at most 1,024 rows a CTA: the finer unit)
    const int fewest = q.npad > kMT ? std::min(q.ctas[0], q.ctas[1]) : q.ctas[0];   // CTAs of a job
    const int64_t most = ((q.chunks + fewest - 1) / fewest + q.seg_chunks - 1) / q.seg_chunks;   // segments of a CTA
    q.slabs = (int)std::max<int64_t>(1, std::min<int64_t>((most + kChain - 1) / kChain, kMaxSlabs));
    q.chain = (int)((most + q.slabs - 1) / q.slabs);
    q.part_bytes = q.slabs * (q.ctas[0] * part3_floats(q.npad) * 4 + (q.npad > kMT ? q.ctas[1] * part3_floats(q.npad - kMT) * 4 : 0));
    return q;
}

template <int NPAD>
cudaError_t launch_tc3(const Gr3Params& p, cudaStream_t st) {
    size_t smem = stages3_of(NPAD) * (size_t)stage3_bytes(NPAD);
    if constexpr (NPAD > kMT) smem = std::max(smem, stages3_of(NPAD - kMT) * (size_t)stage3_bytes(NPAD - kMT));
    smem += 6144;
    cudaError_t e = allow_dynamic_smem(gram_tc3_kernel<NPAD>);
    if (e != cudaSuccess) return e;
    LSK_PROF("gram_tc3", st) gram_tc3_kernel<NPAD><<<p.ctas[0] + p.ctas[1], Shape3::kThreads, smem, st>>>(p);
    return cudaGetLastError();
}

}  // namespace

// Dense A with d <= 256 and at least 2^19 entries: the CUDA-core kernel's two
// launches are the shorter chain below (21 against 29 us at 2,048 x 32, 29
// against 28 at 10,000 x 50, 65 against 42 at 10,000 x 256).
bool gram_tc3_supported(const lsk_mat* A) {
    return A->kind == LSK_DENSE && A->d >= 1 && A->d <= 256 && A->n * A->d >= (int64_t)1 << 19;
}

size_t gram_tc3_workspace_bytes(const lsk_mat* A, int sm_count) {
    return ws_round(gram_tc3_plan(A, sm_count).part_bytes) + ws_round(sizeof(int));
}

// alpha A^T A + beta C, or nothing with **redo != 0 where a column is out of
// the splitting's range (the caller then runs the CUDA-core kernels, which return
// at once when *redo is 0)
template <typename OutT>
cudaError_t gram_tc3_launch(const lsk_mat* A, double alpha, double beta, OutT* C, void* ws, int* flag, int sm_count,
                            cudaStream_t st, const int** redo) {
    const Gr3Plan q = gram_tc3_plan(A, sm_count);
    WsCarver wc{(char*)ws, 0};
    Gr3Params p{};
    p.a.A = (const float*)A->values;
    p.a.lda = A->ld;
    p.a.n = A->n;
    p.a.d = (int)A->d;
    p.a.npad = q.npad;
    p.a.vec = (A->ld % 4 == 0) && (((uintptr_t)A->values & 15) == 0);
    p.a.part = wc.take<float>(q.part_bytes / 4);
    p.a.flag = flag;
    p.redo = wc.take<int>(1);
    *redo = p.redo;
    p.chunks = q.chunks;
    p.ctas[0] = q.ctas[0];
    p.ctas[1] = q.ctas[1];
    p.seg_chunks = q.seg_chunks;
    p.slabs = q.slabs;
    p.chain = q.chain;
    p.magic_add = ((q.seg_chunks == 8 ? 16u : 17u) << 23) + 0x400000u;
    cudaError_t e = cudaMemsetAsync(p.redo, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    switch (q.npad) {
        case 32: e = launch_tc3<32>(p, st); break;
        case 64: e = launch_tc3<64>(p, st); break;
        case 96: e = launch_tc3<96>(p, st); break;
        case 128: e = launch_tc3<128>(p, st); break;
        case 160: e = launch_tc3<160>(p, st); break;
        case 192: e = launch_tc3<192>(p, st); break;
        case 224: e = launch_tc3<224>(p, st); break;
        default: e = launch_tc3<256>(p, st); break;
    }
    if (e != cudaSuccess) return e;
    LSK_PROF("gram_reduce", st) gram_tc3_reduce_kernel<OutT><<<(unsigned)((A->d * A->d + 31) / 32), 256, 0, st>>>(
        p.a.part, q.slabs * q.ctas[0], q.slabs * q.ctas[1], (int)A->d, q.npad, p.redo, alpha, beta, C);
    return cudaGetLastError();
}
template cudaError_t gram_tc3_launch<float>(const lsk_mat*, double, double, float*, void*, int*, int, cudaStream_t, const int**);
template cudaError_t gram_tc3_launch<double>(const lsk_mat*, double, double, double*, void*, int*, int, cudaStream_t, const int**);
