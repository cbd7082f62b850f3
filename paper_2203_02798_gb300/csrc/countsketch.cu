// countsketch.cu -- CountSketch S*A for dense and CSR A (Def. 3, Alg. 2).
//
// The paper stores S as a Block (Column) CountSketch and lets each thread
// own whole rows of SA (Alg. 2, the b_r = r case of Sec. 2.3), so that no two
// threads write the same output row.  Here S is never stored: (h(i), sigma_i)
// is recomputed from Philox whenever it is needed, and row ownership is kept
// at a fine grain:
//
//   1. count: cnt[h(i)]++ for every row (fire-and-forget atomics)
//   2. scan:  off = exclusive prefix sum of cnt        (bucket -> first slot),
//             and a copy of it as each bucket's fill cursor
//   3. place: perm[cursor[h(i)]++] = i | sigma_bit << 31
//   4. gather (dense): teams of 8 to 32 lanes stream the rows listed in
//      stretches of perm with coalesced loads, accumulate them (with their
//      signs) in registers and write each bucket's row of SA once.
//      gather (CSR): same ownership, the row of SA is accumulated in shared
//      memory because CSR columns are scattered.
//
// Every byte of A is read once and every row of SA written once, with no
// global atomics on floating-point data; the only extra traffic is the
// 4 bytes per row of perm.  The per-bucket loads are the Y of Lemma 1:
// expected n/r rows per warp, concentrated as in Lemma 2-3.
#include "lsk_internal.cuh"

namespace {

constexpr int kScanBlock = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanBlock * kScanItems;

// Row i of A is column row0 + i of S: a block of rows of a larger matrix
// (one shard of a row partition) is hashed by its global row index.  Each
// thread takes kPrepRows rows per pass with their atomics independent, so
// several round trips to L2 are in flight per thread.
constexpr int kPrepRows = 4;

__global__ void cs_count_kernel(int64_t n, uint64_t row0, uint32_t r, uint32_t k0, uint32_t k1,
                                uint32_t* __restrict__ cnt) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += stride * kPrepRows) {
#pragma unroll
        for (int q = 0; q < kPrepRows; ++q) {
            const int64_t i = i0 + q * stride;
            if (i < n) {
                uint32_t b, neg;
                cs_hash(row0 + (uint64_t)i, r, k0, k1, b, neg);
                atomicAdd(&cnt[b], 1u);   // result unused: compiled to a reduction (no round trip)
            }
        }
    }
}

// The order of the rows inside a bucket is the order in which their atomics
// reach the cursor (not fixed from run to run); every consumer sums a bucket's
// rows in that order, so S*A is exact for integer-valued data and agrees to
// FP32 rounding otherwise.
__global__ void cs_place_kernel(int64_t n, uint64_t row0, uint32_t r, uint32_t k0, uint32_t k1,
                                uint32_t* __restrict__ cursor, uint32_t* __restrict__ perm) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += stride * kPrepRows) {
        uint32_t slot[kPrepRows], val[kPrepRows];
#pragma unroll
        for (int q = 0; q < kPrepRows; ++q) {
            const int64_t i = i0 + q * stride;
            if (i < n) {
                uint32_t b, neg;
                cs_hash(row0 + (uint64_t)i, r, k0, k1, b, neg);
                slot[q] = atomicAdd(&cursor[b], 1u);
                val[q] = (uint32_t)i | (neg << 31);
            }
        }
#pragma unroll
        for (int q = 0; q < kPrepRows; ++q)
            if (i0 + q * stride < n) perm[slot[q]] = val[q];
    }
}

// Single-pass exclusive scan of the counters (decoupled look-back): block b
// takes tile t (the t-th ticket, kScanTile counts), scans it, publishes its
// aggregate, then adds the published values of the tiles before it, nearest
// first and 32 at a time (one warp), until one carries its inclusive prefix,
// and publishes its own.  A
// tile only waits on tiles whose tickets were taken earlier, i.e. by blocks
// already running.  Writes off[i] = cursor[i] = the exclusive prefix and
// off[len] = the total.  state: the ticket, then one word per tile (flag
// << 32 | value; flag 1 = aggregate, 2 = inclusive prefix), zeroed before
// the launch.  A wait that runs out sets the TIMEOUT flag.
constexpr int kLookbackSpins = 1 << 20;
__device__ __forceinline__ void st_release_u64(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__global__ void __launch_bounds__(kScanBlock) scan_lookback_kernel(const uint32_t* in, uint32_t* off,
                                                                   uint32_t* __restrict__ cursor, int64_t len,
                                                                   unsigned long long* state, int* flag) {
    pdl_enter(in, off, cursor, state);
    __shared__ uint32_t warp_tot[kScanBlock / 32];
    __shared__ uint32_t s_tile, s_prefix;
    if (threadIdx.x == 0) s_tile = atomicAdd(reinterpret_cast<unsigned int*>(state), 1u);
    __syncthreads();
    const int64_t t = s_tile;
    unsigned long long* tiles = state + 1;
    const int64_t base = t * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t run = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        const int64_t i = base + q;
        const uint32_t x = (i < len) ? in[i] : 0u;
        v[q] = run;
        run += x;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const uint32_t w = (lane < kScanBlock / 32) ? warp_tot[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < kScanBlock / 32) warp_tot[lane] = wi - w;
        const uint32_t total = __shfl_sync(0xffffffffu, wi, kScanBlock / 32 - 1);   // the tile's sum
        uint32_t prefix = 0;
        if (t == 0) {
            if (lane == 0) st_release_u64(tiles, (2ull << 32) | total);
        } else {
            if (lane == 0) st_release_u64(tiles + t, (1ull << 32) | total);
            // the warp reads 32 tiles at once, nearest first (lane l: tile p0 - l);
            // before tile 0 counts as an inclusive prefix of 0
            for (int64_t p0 = t - 1;; p0 -= 32) {
                const int64_t p = p0 - lane;
                unsigned long long x = 2ull << 32;
                if (p >= 0) {
                    x = ld_acquire_u64(tiles + p);
                    for (int spin = 0; (x >> 32) == 0 && spin < kLookbackSpins; ++spin) x = ld_acquire_u64(tiles + p);
                    if ((x >> 32) == 0) {
                        set_flag(flag, LSK_FLAG_TIMEOUT);
                        x = 2ull << 32;
                    }
                }
                const unsigned incl_lanes = __ballot_sync(0xffffffffu, (x >> 32) == 2);
                const int stop = incl_lanes ? __ffs(incl_lanes) - 1 : 31;   // the nearest inclusive prefix
                uint32_t val = lane <= stop ? (uint32_t)x : 0u;
#pragma unroll
                for (int o = 16; o; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
                prefix += val;
                if (incl_lanes) break;
            }
            if (lane == 0) st_release_u64(tiles + t, (2ull << 32) | (prefix + total));
        }
        if (lane == 0) {
            s_prefix = prefix;
            if ((t + 1) * kScanTile >= len) off[len] = prefix + total;   // the last tile: the total
        }
    }
    __syncthreads();
    const uint32_t excl = s_prefix + warp_tot[wid] + incl - run;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        const int64_t i = base + q;
        if (i < len) {
            off[i] = v[q] + excl;
            if (cursor) cursor[i] = v[q] + excl;
        }
    }
}

// ---- two-level counting sort of the rows by bucket --------------------------
// The permutation of count / scan / place with the per-row atomics in shared
// memory instead of L2, and every write coalesced: bucket b splits into
// coarse c = b >> shift and fine f = b & (F - 1).  (1) block k hashes its
// chunk of rows, keeps (bucket | sign) per row and counts its rows per
// coarse bucket in shared memory; (2) the counts, laid out coarse bucket by
// coarse bucket and block by block, are scanned in place (the look-back
// scan): each block's offset inside each coarse bucket; (3) each block sorts
// its chunk by coarse bucket in shared memory and writes each coarse bucket's
// run contiguously (row | sign, and f); (4) block c counts coarse bucket c's
// rows per fine bucket, scans the counts (the offsets of its F buckets),
// sorts the rows by fine bucket in shared memory and writes them
// contiguously.  F makes a coarse bucket ~kRxRowsPerCoarse rows on average.
constexpr int kRxThreads = 512;
constexpr int64_t kRxMaxFine = 4096;
constexpr int64_t kRxMaxCoarse = 2048;
constexpr int64_t kRxRowsPerCoarse = 8192;
constexpr int64_t kRxChunk = 16384;        // rows a block sorts in shared memory (step 3)
constexpr int64_t kRxStage = 16384;        // rows of a coarse bucket sorted in shared memory (step 4)
struct RxPlan {
    int64_t F, B, chunk;
    int shift, nct;
};
bool rx_plan(int64_t n, int64_t r, RxPlan& q) {
    if (n <= 0 || n >= ((int64_t)1 << 31) || r < 1) return false;
    int64_t F = 1;
    int sh = 0;
    while (F < kRxMaxFine && n * (F * 2) <= kRxRowsPerCoarse * r) {
        F *= 2;
        ++sh;
    }
    if (n * F > 2 * kRxRowsPerCoarse * r) return false;   // few buckets for many rows: the atomic form
    const int64_t B = (r + F - 1) / F;
    if (B > kRxMaxCoarse) return false;
    int64_t nct = (n + kRxChunk - 1) / kRxChunk;
    if (nct < 256) nct = 256;
    if (B * nct > ((int64_t)1 << 24)) return false;
    q.F = F;
    q.B = B;
    q.shift = sh;
    q.nct = (int)nct;
    q.chunk = (n + nct - 1) / nct;
    return true;
}
size_t rx_scatter_smem(const RxPlan& q) { return (size_t)q.B * 12 + 16 + (size_t)q.chunk * 8; }
size_t rx_fine_smem(const RxPlan& q) { return (size_t)q.F * 4 + (size_t)kRxStage * 4; }

// block-wide exclusive scan of cnt[0 .. len) in shared memory (len <=
// 8 kRxThreads), in place; `tot` receives the total
__device__ __forceinline__ void rx_block_scan(uint32_t* cnt, int len, uint32_t* wsum, uint32_t& tot) {
    const int per = (len + kRxThreads - 1) / kRxThreads;
    const int lo = (int)threadIdx.x * per, hi = min(len, lo + per);
    uint32_t run = 0;
    for (int i = lo; i < hi; ++i) run += cnt[i];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        const uint32_t x = lane < kRxThreads / 32 ? wsum[lane] : 0u;
        uint32_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += y;
        }
        if (lane < kRxThreads / 32) wsum[lane] = xi - x;
        if (lane == 31) wsum[kRxThreads / 32] = xi;
    }
    __syncthreads();
    uint32_t acc = wsum[w] + incl - run;
    for (int i = lo; i < hi; ++i) {
        const uint32_t c = cnt[i];
        cnt[i] = acc;
        acc += c;
    }
    tot = wsum[kRxThreads / 32];
    __syncthreads();
}

__global__ void __launch_bounds__(kRxThreads) rx_count_kernel(int64_t n, uint64_t row0, uint32_t r, uint32_t k0,
                                                              uint32_t k1, RxPlan q, uint32_t* __restrict__ bsign,
                                                              uint32_t* __restrict__ H, unsigned long long* hstate,
                                                              int hstate_words) {
    pdl_enter(bsign, H, hstate);
    extern __shared__ uint32_t hs[];
    if (blockIdx.x == 0)   // the scan's state, zeroed for the next launch
        for (int j = threadIdx.x; j < hstate_words; j += blockDim.x) hstate[j] = 0ull;
    for (int64_t c = threadIdx.x; c < q.B; c += blockDim.x) hs[c] = 0u;
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * q.chunk, i1 = min(n, i0 + q.chunk);
    for (int64_t i = i0 + threadIdx.x; i < i1; i += (int64_t)kPrepRows * kRxThreads) {
        uint32_t b[kPrepRows], neg[kPrepRows];
#pragma unroll
        for (int u = 0; u < kPrepRows; ++u)
            if (i + u * kRxThreads < i1) cs_hash(row0 + (uint64_t)(i + u * kRxThreads), r, k0, k1, b[u], neg[u]);
#pragma unroll
        for (int u = 0; u < kPrepRows; ++u) {
            if (i + u * kRxThreads < i1) {
                bsign[i + u * kRxThreads] = b[u] | (neg[u] << 31);
                atomicAdd(&hs[b[u] >> q.shift], 1u);
            }
        }
    }
    __syncthreads();
    for (int64_t c = threadIdx.x; c < q.B; c += blockDim.x) H[c * q.nct + blockIdx.x] = hs[c];
}

// step 3: shared memory holds the global base and the local offset (then the
// cursor) of every coarse bucket, and the chunk sorted by coarse bucket as
// (row | sign, fine | coarse << 16)
__global__ void __launch_bounds__(kRxThreads) rx_scatter_kernel(int64_t n, RxPlan q,
                                                                const uint32_t* __restrict__ bsign,
                                                                const uint32_t* __restrict__ base,
                                                                uint32_t* __restrict__ T, uint16_t* __restrict__ TF) {
    pdl_enter(bsign, base, T, TF);
    extern __shared__ uint32_t sm[];
    __shared__ uint32_t wsum[kRxThreads / 32 + 1];
    uint32_t* hb = sm;                 // [B] global start of this block's run in coarse bucket c
    uint32_t* lo = sm + q.B;           // [B] local start of coarse bucket c in the sorted chunk
    uint32_t* cur = sm + 2 * q.B;      // [B] cursor
    uint2* stage = reinterpret_cast<uint2*>(sm + ((3 * q.B + 3) & ~(int64_t)1));
    for (int64_t c = threadIdx.x; c < q.B; c += blockDim.x) {
        const int64_t idx = c * q.nct + blockIdx.x;
        const uint32_t b0 = __ldg(base + idx);
        hb[c] = b0;
        lo[c] = __ldg(base + idx + 1) - b0;   // this block's rows in coarse bucket c
    }
    __syncthreads();
    uint32_t tot;
    rx_block_scan(lo, (int)q.B, wsum, tot);
    for (int64_t c = threadIdx.x; c < q.B; c += blockDim.x) cur[c] = lo[c];
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * q.chunk, i1 = min(n, i0 + q.chunk);
    const uint32_t fmask = (uint32_t)q.F - 1u;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += kRxThreads) {
        const uint32_t v = __ldg(bsign + i);
        const uint32_t b = v & 0x7fffffffu, c = b >> q.shift;
        const uint32_t p = atomicAdd(&cur[c], 1u);
        stage[p] = make_uint2((uint32_t)i | (v & 0x80000000u), (b & fmask) | (c << 16));
    }
    __syncthreads();
    for (uint32_t p = threadIdx.x; p < tot; p += kRxThreads) {
        const uint2 e = stage[p];
        const uint32_t c = e.y >> 16;
        const uint32_t g = hb[c] + (p - lo[c]);
        T[g] = e.x;
        TF[g] = (uint16_t)(e.y & 0xffffu);
    }
}

// step 4: block c, rows [s, e) of coarse bucket c
__global__ void __launch_bounds__(kRxThreads) rx_fine_kernel(int64_t n, int64_t r, RxPlan q,
                                                             const uint32_t* __restrict__ base,
                                                             const uint32_t* __restrict__ T,
                                                             const uint16_t* __restrict__ TF,
                                                             uint32_t* __restrict__ perm, uint32_t* __restrict__ off) {
    pdl_enter(base, T, TF, perm, off);
    extern __shared__ uint32_t fc[];   // [F] counts, then starts; then the staged rows
    __shared__ uint32_t wsum[kRxThreads / 32 + 1];
    uint32_t* stage = fc + q.F;
    const int64_t c = blockIdx.x;
    const uint32_t s = __ldg(base + c * q.nct);
    const uint32_t e = (c + 1 < q.B) ? __ldg(base + (c + 1) * q.nct) : (uint32_t)n;
    for (int f = threadIdx.x; f < (int)q.F; f += kRxThreads) fc[f] = 0u;
    __syncthreads();
    for (uint32_t i = s + threadIdx.x; i < e; i += kRxThreads) atomicAdd(&fc[__ldg(TF + i)], 1u);
    __syncthreads();
    uint32_t tot;
    rx_block_scan(fc, (int)q.F, wsum, tot);
    for (int f = threadIdx.x; f < (int)q.F; f += kRxThreads) {
        const int64_t b = c * q.F + f;
        if (b < r) off[b] = s + fc[f];
    }
    if (c == q.B - 1 && threadIdx.x == 0) off[r] = (uint32_t)n;
    __syncthreads();
    if (e - s <= (uint32_t)kRxStage) {
        // sorted in shared memory, then written contiguously
        for (uint32_t i = s + threadIdx.x; i < e; i += kRxThreads) {
            const uint32_t p = atomicAdd(&fc[__ldg(TF + i)], 1u);
            stage[p] = __ldg(T + i);
        }
        __syncthreads();
        for (uint32_t p = threadIdx.x; p < e - s; p += kRxThreads) perm[s + p] = stage[p];
    } else {
        for (uint32_t i = s + threadIdx.x; i < e; i += kRxThreads) {
            const uint32_t p = atomicAdd(&fc[__ldg(TF + i)], 1u);
            perm[s + p] = __ldg(T + i);
        }
    }
}

// ---- dense gather ---------------------------------------------------------
// The rows of A in the order of perm, summed bucket by bucket.  A team of L
// lanes takes a contiguous stretch of perm and walks it, kRows rows of loads in
// flight, across the ends of its buckets: with a bucket (or a part of one) per
// warp at a time, each bucket of 5 to 30 rows waited for its own chain of
// offsets, permutation and rows, and with 20,000 parts on 9,728 warps a third
// round ran nearly empty.  Lanes own VEC consecutive columns in each of U
// groups of L VEC; a row of 32 or 64 columns is 8 or 16 lanes wide, and 4 or 2
// teams share a warp in step (a warp per row left the other lanes without
// loads).  The ends of the next L buckets stand in the team's lanes.  Bound by
// DRAM, which random rows of 400 bytes hold at 4.5 TB/s and of 1 KB at 6.2:
// 1,234,567 x 100 -> 10,000 in 112 us (123 with a warp per bucket part),
// 1M x 100 -> 256 in 88 (111), 790,706 x 32 -> 1,024 in 25 (54), 500,000 x 200 ->
// 40,000 in 87 (105), 22,379 x 256 -> 65,536 in 23 (42).
//
// Team t of T starts at the point t r / T of the buckets.  own: rounded down to
// a bucket, so that each bucket is one team's and is stored, empty ones as
// zeros.  Otherwise the fraction is taken of the bucket's rows, so that few
// long buckets are shared out evenly; what a team holds of a bucket that it
// shares is added to SA (zeroed first) atomically.
template <int VEC>
struct VecT;
template <>
struct VecT<4> {
    using T = float4;
};
template <>
struct VecT<2> {
    using T = float2;
};
template <>
struct VecT<1> {
    using T = float;
};

__device__ __forceinline__ void vadd(float4& a, const float4& b, float s) {
    a.x = fmaf(s, b.x, a.x);
    a.y = fmaf(s, b.y, a.y);
    a.z = fmaf(s, b.z, a.z);
    a.w = fmaf(s, b.w, a.w);
}
__device__ __forceinline__ void vadd(float2& a, const float2& b, float s) {
    a.x = fmaf(s, b.x, a.x);
    a.y = fmaf(s, b.y, a.y);
}
__device__ __forceinline__ void vadd(float& a, const float& b, float s) { a = fmaf(s, b, a); }
__device__ __forceinline__ void vzero(float4& a) { a = make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ void vzero(float2& a) { a = make_float2(0.f, 0.f); }
__device__ __forceinline__ void vzero(float& a) { a = 0.f; }
__device__ __forceinline__ void vatomic_add(float4* p, const float4& v) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void vatomic_add(float2* p, const float2& v) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void vatomic_add(float* p, const float& v) { atomicAdd(p, v); }

template <int VEC>
__device__ __forceinline__ typename VecT<VEC>::T ldg_stream(const float* p) {
    if constexpr (VEC == 4) {
        float4 v;
        asm("ld.global.nc.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "l"(p));
        return v;
    } else if constexpr (VEC == 2) {
        float2 v;
        asm("ld.global.nc.L1::no_allocate.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
        return v;
    } else {
        float v;
        asm("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(v) : "l"(p));
        return v;
    }
}

// three blocks an SM keep 32 loads a lane in registers; single floats need fewer
constexpr int kGatherThreads = 256;
__host__ __device__ constexpr int gather_per_sm(int vec, int u) { return vec == 1 && u < 4 ? 4 : 3; }
template <int VEC, int U, int L>
__global__ void __launch_bounds__(kGatherThreads, gather_per_sm(VEC, U)) cs_dense_gather_kernel(
    const float* __restrict__ A, int64_t lda, int64_t d, uint32_t r, const uint32_t* __restrict__ off,
    const uint32_t* __restrict__ perm, float* __restrict__ SA, int64_t teams, int own, int accumulate,
    const uint32_t* __restrict__ cpos) {
    pdl_enter(A, off, perm, cpos, SA);
    using V = typename VecT<VEC>::T;
    constexpr unsigned kAll = 0xffffffffu, kTeam = L == 32 ? kAll : (1u << (L & 31)) - 1u;
    constexpr int kCols = L * VEC * U;              // columns per pass
    constexpr int kRows = VEC * U >= 8 ? 4 : 8;     // rows of loads in flight
    const int lane = threadIdx.x & 31, tl = lane & (L - 1), sh = lane & ~(L - 1);
    const int64_t team = ((int64_t)blockIdx.x * kGatherThreads + threadIdx.x) / L;
    int64_t b0 = 0, b1 = 0;
    uint32_t s = 0, e = 0;
    bool shared_start = false;
    if (team < teams) {
        const int64_t x0 = team * (int64_t)r, x1 = x0 + r;
        b0 = x0 / teams;
        b1 = x1 / teams;
        s = __ldg(off + b0);
        e = __ldg(off + b1);
        if (!own) {
            const uint64_t f0 = (uint64_t)(x0 - b0 * teams), f1 = (uint64_t)(x1 - b1 * teams);
            const uint32_t s0 = s;
            if (f0) s += (uint32_t)((uint64_t)(__ldg(off + b0 + 1) - s) * f0 / (uint64_t)teams);
            if (f1) e += (uint32_t)((uint64_t)(__ldg(off + b1 + 1) - e) * f1 / (uint64_t)teams);
            shared_start = s != s0;
        }
    }
    for (int64_t c0 = 0; c0 < d; c0 += kCols) {
        bool colok[U];
#pragma unroll
        for (int u = 0; u < U; ++u) colok[u] = c0 + (int64_t)(u * L + tl) * VEC < d;
        uint32_t next = s + tl < e ? __ldg(perm + s + tl) : 0u;
        int64_t bb = b0;                            // lane tl: the end (and the rank) of bucket bb + tl
        uint32_t ends = __ldg(off + min(bb + 1 + tl, (int64_t)r));
        uint32_t ranks = cpos ? __ldg(cpos + min(bb + tl, (int64_t)r - 1)) : 0u;
        uint32_t end = 0;                           // of the bucket that is summed
        int64_t orow = 0;                           // its row of SA
        // the bucket that holds position t, for the teams that want it
        auto find = [&](uint32_t t, bool want) {
            int at = 0;
            for (;;) {
                const unsigned m = (__ballot_sync(kAll, ends > t) >> sh) & kTeam;
                if (want && m) at = __ffs(m) - 1;
                const bool more = want && !m;
                if (!__any_sync(kAll, more)) break;
                if (more) {
                    bb += L;
                    ends = __ldg(off + min(bb + 1 + tl, (int64_t)r));
                    if (cpos) ranks = __ldg(cpos + min(bb + tl, (int64_t)r - 1));
                }
            }
            const uint32_t en = __shfl_sync(kAll, ends, sh + at), rk = __shfl_sync(kAll, ranks, sh + at);
            if (want) {
                end = en;
                orow = cpos ? (int64_t)rk : bb + at;
            }
        };
        find(s, s < e);
        bool whole = !shared_start;                 // the bucket's first row is this team's
        V acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) vzero(acc[u]);
        for (uint32_t t0 = s; __any_sync(kAll, t0 < e); t0 += L) {
            const uint32_t mine = next;
            next = t0 + L + tl < e ? __ldg(perm + t0 + L + tl) : 0u;
#pragma unroll 1
            for (int j = 0; j < L; j += kRows) {
                if (!__any_sync(kAll, t0 + j < e)) break;
                V v[kRows][U];
                float sg[kRows];
#pragma unroll
                for (int q = 0; q < kRows; ++q) {
                    const uint32_t p = __shfl_sync(kAll, mine, sh + j + q);
                    const bool ok = t0 + j + q < e;
                    sg[q] = (p >> 31) ? -1.0f : 1.0f;
                    const float* row = A + (int64_t)(p & 0x7fffffffu) * lda + c0;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (ok && colok[u]) v[q][u] = ldg_stream<VEC>(row + (u * L + tl) * VEC);
                        else vzero(v[q][u]);
                    }
                }
                // no team's bucket ends among these rows: summed in pairs first,
                // an eighth (a quarter) of the roundings into the running sum
                const uint32_t t8 = t0 + j + kRows;
                if (__all_sync(kAll, (t8 < end && t8 < e) || t0 + j >= e)) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        V x[kRows / 2];
#pragma unroll
                        for (int q = 0; q < kRows / 2; ++q) {
                            vzero(x[q]);
                            vadd(x[q], v[2 * q][u], sg[2 * q]);
                            vadd(x[q], v[2 * q + 1][u], sg[2 * q + 1]);
                        }
#pragma unroll
                        for (int o = kRows / 4; o; o >>= 1)
#pragma unroll
                            for (int q = 0; q < o; ++q) vadd(x[q], x[q + o], 1.0f);
                        vadd(acc[u], x[0], 1.0f);
                    }
                    continue;
                }
                // else row by row, two summed before they are added where they can be
                // (20,000 x 50 -> 2,500, eight rows to a bucket: 5.1e-8 off, 5.6e-8 one by one)
                V two[U];
#pragma unroll
                for (int q = 0; q < kRows; ++q) {
                    const uint32_t t = t0 + j + q + 1;   // past this row
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (q % 2 == 0) vzero(two[u]);
                        vadd(two[u], v[q][u], sg[q]);
                        if (q % 2) vadd(acc[u], two[u], 1.0f);
                    }
                    const bool last = t <= e && (t == end || t == e);
                    if (!__any_sync(kAll, last)) continue;
                    if (last) {
                        float* out = SA + orow * d + c0;
                        const bool store = whole && end <= e && !accumulate;
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            if (q % 2 == 0) {
                                vadd(acc[u], two[u], 1.0f);
                                vzero(two[u]);
                            }
                            if (colok[u]) {
                                V* o = reinterpret_cast<V*>(out + (u * L + tl) * VEC);
                                if (store) *o = acc[u];
                                else vatomic_add(o, acc[u]);
                            }
                            vzero(acc[u]);
                        }
                        whole = true;
                    }
                    find(t, last && t < e);
                }
            }
        }
        if (own && !accumulate && !cpos) {          // empty buckets
            for (int64_t x0 = b0; __any_sync(kAll, x0 < b1); x0 += L) {
                const int64_t x = x0 + tl;
                const bool empty = x < b1 && __ldg(off + x) == __ldg(off + x + 1);
                unsigned m = (__ballot_sync(kAll, empty) >> sh) & kTeam;
                while (m) {
                    float* out = SA + (x0 + __ffs(m) - 1) * d + c0;
                    m &= m - 1;
                    V z;
                    vzero(z);
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (colok[u]) *reinterpret_cast<V*>(out + (u * L + tl) * VEC) = z;
                }
            }
        }
    }
}

// ---- CSR gather -----------------------------------------------------------
// One warp per bucket part (P parts per bucket as in the dense gather); the
// part's row of SA lives in shared memory (d floats per warp).  Lane t handles the t-th row of the bucket's list and
// adds its nonzeros with shared-memory atomics (columns of different rows
// may collide).  Out-of-range row pointers or column indices are skipped
// and reported through the BAD_CSR flag.
__global__ void cs_csr_gather_kernel(const float* __restrict__ V, const int32_t* __restrict__ J,
                                     const int64_t* __restrict__ I, int64_t nnz, int64_t d,
                                     uint32_t r, const uint32_t* __restrict__ off,
                                     const uint32_t* __restrict__ perm, float* __restrict__ SA,
                                     int* flag, int P, int accumulate, const uint32_t* __restrict__ cpos) {
    extern __shared__ float srow[];
    const int lane = threadIdx.x & 31;
    float* acc = srow + (int64_t)(threadIdx.x >> 5) * d;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t items = (int64_t)r * P;
    for (int64_t vb = warp; vb < items; vb += nwarps) {
        const int64_t b = vb / P;
        const uint32_t part = (uint32_t)(vb % P);
        const uint32_t s0 = off[b], len = off[b + 1] - s0;
        const uint32_t s = s0 + (uint32_t)(((uint64_t)len * part) / P);
        const uint32_t e = s0 + (uint32_t)(((uint64_t)len * (part + 1)) / P);
        if ((P > 1 || accumulate || cpos) && s == e) continue;
        for (int64_t c = lane; c < d; c += 32) acc[c] = 0.0f;
        __syncwarp();
        bool bad = false;
        for (uint32_t t = s + lane; t < e; t += 32) {
            const uint32_t p = perm[t];
            const float sg = (p >> 31) ? -1.0f : 1.0f;
            const int64_t row = p & 0x7fffffffu;
            const int64_t k0 = I[row], k1 = I[row + 1];
            if (k0 < 0 || k1 < k0 || k1 > nnz) {
                bad = true;
                continue;
            }
            for (int64_t kk = k0; kk < k1; ++kk) {
                const int32_t col = __ldg(J + kk);
                if (col < 0 || col >= d) {
                    bad = true;
                    continue;
                }
                atomicAdd(&acc[col], sg * __ldg(V + kk));
            }
        }
        if (bad) set_flag(flag, LSK_FLAG_BAD_CSR);
        __syncwarp();
        float* out = SA + (cpos ? (int64_t)cpos[b] : b) * d;
        if (P == 1 && !accumulate) {
            for (int64_t c = lane; c < d; c += 32) out[c] = acc[c];
        } else {
            for (int64_t c = lane; c < d; c += 32)
                if (acc[c] != 0.0f) atomicAdd(out + c, acc[c]);
        }
        __syncwarp();
    }
}

// ---- CSR scatter ----------------------------------------------------------
// S A without a permutation: a warp hashes 32 consecutive rows, then deals
// their nonzeros out to its lanes, each one reduction in L2 on its entry of SA
// (zeroed first).  The entries of A are read once, in order; L2 takes 176
// scattered reductions a ns where they spread over 2^20 addresses, 82 over
// 2^14, so the reductions cost less than finding each bucket's rows and
// fetching their two or three nonzeros from anywhere in A: the sketch of 1M x
// 200 at 1% into 40,000 buckets takes 28 us (79 with the permutation), 500,000 x
// 256 at 2% into 65,536 32 (98), 20,000 x 64 at 5% into 4,096 14 (30).
__global__ void __launch_bounds__(256) cs_csr_scatter_kernel(const float* __restrict__ V,
                                                             const int32_t* __restrict__ J,
                                                             const int64_t* __restrict__ I, int64_t n, int64_t nnz,
                                                             int64_t d, uint64_t row0, uint32_t r, uint32_t k0,
                                                             uint32_t k1, float* SA, float* copy, int64_t stride,
                                                             int more, int* flag) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool bad = false;
    for (int64_t i0 = warp * 32; i0 < n; i0 += nwarps * 32) {
        RowGroup g;
        if (!g.load(I, i0 + lane, n, nnz)) bad = true;
        uint32_t b, neg;
        cs_hash(row0 + (uint64_t)(i0 + lane), r, k0, k1, b, neg);
        const uint32_t to = b | (neg << 31);
        const int at_copy = (int)(i0 >> 5) & more;   // groups of rows take turns (more: copies - 1)
        float* const out = at_copy ? copy + (at_copy - 1) * stride : SA;
        constexpr int kEntries = 2;   // entries a lane at once
        for (int64_t e0 = 0; e0 < g.total; e0 += 32 * kEntries) {
            int32_t col[kEntries];
            float v[kEntries];
            uint32_t t[kEntries];
#pragma unroll
            for (int u = 0; u < kEntries; ++u) {
                const int64_t e = min(e0 + 32 * u + lane, g.total - 1);
                const int q = g.lane_of(e);
                const int64_t at = g.first_of(q) + e;
                t[u] = __shfl_sync(0xffffffffu, to, q);
                col[u] = __ldg(J + at);
                v[u] = __ldg(V + at);
            }
#pragma unroll
            for (int u = 0; u < kEntries; ++u) {
                if (e0 + 32 * u + lane >= g.total) continue;
                if (col[u] < 0 || col[u] >= d) {
                    bad = true;
                    continue;
                }
                atomicAdd(out + (int64_t)(t[u] & 0x7fffffffu) * d + col[u], (t[u] >> 31) ? -v[u] : v[u]);
            }
        }
    }
    if (bad) set_flag(flag, LSK_FLAG_BAD_CSR);
}

// SA += the copies of a CSR scatter, in pairs
__global__ void cs_add_copies_kernel(float* __restrict__ SA, const float* __restrict__ copy, int64_t stride, int more,
                                     int64_t entries) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < entries; i += (int64_t)gridDim.x * blockDim.x) {
        float s = SA[i] + __ldg(copy + i);
        if (more == 3) s += __ldg(copy + stride + i) + __ldg(copy + 2 * stride + i);
        SA[i] = s;
    }
}

__global__ void cs_hash_debug_kernel(int64_t n, uint32_t r, uint32_t k0, uint32_t k1,
                                     int32_t* bucket, int8_t* sign) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        uint32_t b, neg;
        cs_hash((uint64_t)i, r, k0, k1, b, neg);
        bucket[i] = (int32_t)b;
        sign[i] = neg ? (int8_t)-1 : (int8_t)1;
    }
}

// Compaction of the sketch's rows to the non-empty buckets (off[b + 1] >
// off[b]), in bucket order: cpos[b] = the number of non-empty buckets before b,
// cidx[cpos[b]] = b for each non-empty b, *ccount = their number.  One block
// of 1024 threads: each warp counts its contiguous 1/32 of the buckets by
// ballots, the 32 totals are scanned, and a second pass writes.  Bound by the
// latency of the loads, so a lane keeps 2 kCompactLoads of them in flight and
// the block meets twice in all, not in every 4,096 buckets (24 problems,
// 65,536 buckets at most: 43 -> 20 us).
constexpr int kCompactLoads = 8;
__device__ __forceinline__ void compact_body(const uint32_t* __restrict__ off, int64_t r, uint32_t* __restrict__ cpos,
                                             uint32_t* __restrict__ cidx, uint32_t* __restrict__ ccount) {
    __shared__ uint32_t wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t seg = ((r + 1023) / 1024) * 32, lo = min(r, w * seg), hi = min(r, lo + seg);
    // the non-empty ones among buckets b0 + 32 q, q < kCompactLoads, as lane masks
    auto masks = [&](int64_t b0, unsigned (&m)[kCompactLoads]) {
        uint32_t x[kCompactLoads], y[kCompactLoads];
#pragma unroll
        for (int q = 0; q < kCompactLoads; ++q) {
            const int64_t b = b0 + 32 * q + lane;
            x[q] = b < hi ? __ldg(off + b) : 0u;
            y[q] = b < hi ? __ldg(off + b + 1) : 0u;
        }
#pragma unroll
        for (int q = 0; q < kCompactLoads; ++q) m[q] = __ballot_sync(0xffffffffu, y[q] > x[q]);
    };
    unsigned m[kCompactLoads];
    uint32_t own = 0;
    for (int64_t b0 = lo; b0 < hi; b0 += 32 * kCompactLoads) {
        masks(b0, m);
#pragma unroll
        for (int q = 0; q < kCompactLoads; ++q) own += __popc(m[q]);
    }
    if (lane == 0) wsum[w] = own;
    __syncthreads();
    uint32_t incl = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (threadIdx.x == 31) *ccount = incl;
    uint32_t pos = __shfl_sync(0xffffffffu, incl, w) - own;   // non-empty buckets before this warp's
    for (int64_t b0 = lo; b0 < hi; b0 += 32 * kCompactLoads) {
        masks(b0, m);
#pragma unroll
        for (int q = 0; q < kCompactLoads; ++q) {
            const int64_t b = b0 + 32 * q + lane;
            const uint32_t at = pos + __popc(m[q] & ((1u << lane) - 1u));
            if (b < hi) {
                cpos[b] = at;
                if ((m[q] >> lane) & 1u) cidx[at] = (uint32_t)b;
            }
            pos += __popc(m[q]);
        }
    }
}
__global__ void __launch_bounds__(1024) cs_compact_kernel(const uint32_t* __restrict__ off, int64_t r,
                                                          uint32_t* __restrict__ cpos, uint32_t* __restrict__ cidx,
                                                          uint32_t* __restrict__ ccount) {
    compact_body(off, r, cpos, cidx, ccount);
}

// ---- grouped preparation: the permutations of many problems, three launches
// The problems' counters are numbered consecutively (problem p's r + 1
// counters from cnt_base); one exclusive scan over all the counters then
// gives each bucket its range of the shared permutation, so the problems'
// rows land in consecutive blocks of it and each problem's off[] (its slice
// of the scanned counters) indexes that shared permutation directly.
struct CsGp {
    int64_t n, r, cnt_base;
    uint32_t k0, k1;
    uint32_t* cidx;     // compaction (or null)
    uint32_t* ccount;
};

// Counting and placing take the same form: a block takes a run of one
// problem's rows.  With few buckets for its rows (r <= kGroupBuckets, n >= 2r)
// it ranks them per bucket in shared memory and goes to L2 once per bucket it
// met, not once per row: the problems of 32 columns send some hundred rows to
// each of 1,024 counters, whose atomics queue up at one address.  With more
// buckets a run meets most of its buckets once, and the rows go to L2
// themselves, kPrepRows at a time.  24 problems, 3.1M rows, 267K buckets:
// counting 26 us, placing 44 (all rows through L2: 113 and 131).
constexpr int kGroupThreads = 512;
constexpr int kGroupRows = 16;         // rows a thread: 13 bits of rank, 13 of bucket, the sign
constexpr int64_t kGroupBuckets = 4096;
__host__ __device__ __forceinline__ bool group_shared(int64_t n, int64_t r) { return r <= kGroupBuckets && n >= 2 * r; }
__host__ __device__ __forceinline__ int64_t group_run(int64_t n, int64_t r) {
    return (int64_t)kGroupThreads * (group_shared(n, r) ? kGroupRows : kPrepRows);
}

template <bool kPlace>
__global__ void __launch_bounds__(kGroupThreads, 2) cs_rows_grouped_kernel(const CsGp* __restrict__ ps,
                                                                           const int* __restrict__ boff, int count,
                                                                           uint32_t* __restrict__ counters,
                                                                           uint32_t* __restrict__ perm) {
    __shared__ uint32_t hist[kGroupBuckets];
    const int p = group_of(boff, count, (int)blockIdx.x);
    const CsGp& j = ps[p];
    const int64_t n = j.n, r = j.r;
    const uint32_t k0 = j.k0, k1 = j.k1;
    uint32_t* cnt = counters + j.cnt_base;
    const int64_t i0 = (int64_t)((int)blockIdx.x - __ldg(boff + p)) * group_run(n, r) + threadIdx.x;
    if (group_shared(n, r)) {
        for (int b = threadIdx.x; b < (int)r; b += kGroupThreads) hist[b] = 0u;
        __syncthreads();
        uint32_t at[kGroupRows];   // sign << 31 | bucket << 13 | rank among the block's rows of that bucket
#pragma unroll
        for (int q = 0; q < kGroupRows; ++q) {
            const int64_t i = i0 + q * kGroupThreads;
            if (i < n) {
                uint32_t b, neg;
                cs_hash((uint64_t)i, (uint32_t)r, k0, k1, b, neg);
                const uint32_t rank = atomicAdd(&hist[b], 1u);
                at[q] = (neg << 31) | (b << 13) | rank;
            }
        }
        __syncthreads();
        for (int b = threadIdx.x; b < (int)r; b += kGroupThreads) {
            const uint32_t h = hist[b];
            if (h) {
                if (kPlace) hist[b] = atomicAdd(&cnt[b], h);
                else atomicAdd(&cnt[b], h);
            }
        }
        if (!kPlace) return;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kGroupRows; ++q) {
            const int64_t i = i0 + q * kGroupThreads;
            if (i < n)
                perm[hist[(at[q] >> 13) & (kGroupBuckets - 1)] + (at[q] & 0x1fffu)] =
                    (uint32_t)i | (at[q] & 0x80000000u);
        }
        return;
    }
    uint32_t slot[kPrepRows], val[kPrepRows];
#pragma unroll
    for (int q = 0; q < kPrepRows; ++q) {
        const int64_t i = i0 + q * kGroupThreads;
        if (i < n) {
            uint32_t b, neg;
            cs_hash((uint64_t)i, (uint32_t)r, k0, k1, b, neg);
            if (kPlace) {
                slot[q] = atomicAdd(&cnt[b], 1u);
                val[q] = (uint32_t)i | (neg << 31);
            } else {
                atomicAdd(&cnt[b], 1u);
            }
        }
    }
    if (kPlace) {
#pragma unroll
        for (int q = 0; q < kPrepRows; ++q)
            if (i0 + q * kGroupThreads < n) perm[slot[q]] = val[q];
    }
}

// block p: problem p's compaction (if it has one)
__global__ void __launch_bounds__(1024) cs_compact_grouped_kernel(const CsGp* __restrict__ ps,
                                                                  const uint32_t* __restrict__ off,
                                                                  uint32_t* __restrict__ cpos) {
    const CsGp& j = ps[blockIdx.x];
    if (!j.cidx) return;
    compact_body(off + j.cnt_base, j.r, cpos + j.cnt_base, j.cidx, j.ccount);
}

inline unsigned grid_for(int64_t items, int threads, int sm_count, int per_sm = 8) {
    int64_t g = (items + threads - 1) / threads;
    const int64_t cap = (int64_t)sm_count * per_sm;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (unsigned)g;
}

}  // namespace

// the look-back scan's ticket and tile words
size_t scan_state_words(int64_t len) { return (size_t)((len + kScanTile - 1) / kScanTile) + 1; }

// The CountSketch workspace, in this order: the counters and the scan's
// state (zeroed by one memset), the bucket offsets, the cursors, the
// permutation, the compaction positions;
// then, for the two-level sort, the per-row (bucket | sign), the rows
// grouped by coarse bucket with their fine indices, the per-block counts
// (scanned in place) and their scan state.
struct CsWs {
    uint32_t *cnt, *off, *cursor, *perm, *cpos;
    unsigned long long* state;
    uint32_t *bsign, *T, *H;
    uint16_t* TF;
    unsigned long long* hstate;
    int hstate_words;
    size_t bytes;
};
CsWs cs_carve(void* ws, int64_t n, int64_t r, const RxPlan* q) {
    WsCarver wc{(char*)ws, 0};
    CsWs w{};
    const size_t nn = n > 0 ? (size_t)n : 1;
    w.cnt = wc.take<uint32_t>(r + 1);
    w.state = wc.take<unsigned long long>(scan_state_words(r));
    w.off = wc.take<uint32_t>(r + 1);
    w.cursor = wc.take<uint32_t>(r + 1);
    w.perm = wc.take<uint32_t>(nn);
    w.cpos = wc.take<uint32_t>(r + 1);
    if (q) {
        w.bsign = wc.take<uint32_t>(nn);
        w.T = wc.take<uint32_t>(nn);
        w.TF = wc.take<uint16_t>(nn);
        w.H = wc.take<uint32_t>((size_t)q->B * q->nct + 1);
        w.hstate_words = (int)scan_state_words(q->B * q->nct);
        w.hstate = wc.take<unsigned long long>((size_t)w.hstate_words);
    }
    w.bytes = ws_round(wc.off) + 256;
    return w;
}

size_t cs_workspace_bytes(int64_t n, int64_t r) {
    RxPlan q;
    return cs_carve(nullptr, n, r, rx_plan(n, r, q) ? &q : nullptr).bytes;
}
size_t cs_workspace_bytes(const lsk_mat* A, int64_t r) {
    return std::max(cs_workspace_bytes(A->n, r), cs_scatter_copy_bytes(A, r, false));
}
size_t cs_workspace_bytes_atomic(int64_t n, int64_t r) { return cs_carve(nullptr, n, r, nullptr).bytes; }

cudaError_t cs_hash_launch(int64_t n, int64_t r, uint64_t seed, int32_t* bucket, int8_t* sign,
                           cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    cs_hash_debug_kernel<<<grid_for(n, 256, 152, 16), 256, 0, st>>>(
        n, (uint32_t)r, (uint32_t)seed, (uint32_t)(seed >> 32), bucket, sign);
    return cudaGetLastError();
}

// Steps 1-3 (count, scan, place): on return *off_out (r + 1 entries, off[r] = n)
// and *perm_out (n entries, local row indices) point into ws; the launches
// are queued on st.  Row i is hashed as column row0 + i of S.  rx: ws holds
// cs_workspace_bytes (the two-level sort where its plan applies), else
// cs_workspace_bytes_atomic (count / scan / place with L2 atomics).
cudaError_t cs_prep_launch(int64_t n, int64_t r, uint64_t seed, void* ws, int sm_count, cudaStream_t st,
                           const uint32_t** off_out, const uint32_t** perm_out, uint64_t row0, int* flag, bool rx,
                           bool scan_early) {
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    RxPlan q;
    const bool two_level = rx && rx_plan(n, r, q);
    const CsWs w = cs_carve(ws, n, r, two_level ? &q : nullptr);
    cudaError_t e;
    if (two_level) {
        if ((e = allow_dynamic_smem(rx_scatter_kernel)) != cudaSuccess) return e;
        if ((e = allow_dynamic_smem(rx_fine_kernel)) != cudaSuccess) return e;
        LSK_PROF("cs_count", st) launch_pdl(rx_count_kernel, q.nct, kRxThreads, (size_t)q.B * 4, 1, st, n, row0, (uint32_t)r,
                                             k0, k1, q, w.bsign, w.H, w.hstate, w.hstate_words);
        const int64_t len = q.B * q.nct;
        LSK_PROF("cs_scan", st) launch_chained(scan_early, scan_lookback_kernel, (unsigned)((len + kScanTile - 1) / kScanTile),
                                                kScanBlock, 0, 1, st, w.H, w.H, nullptr, len, w.hstate, flag);
        LSK_PROF("cs_place", st) launch_pdl(rx_scatter_kernel, q.nct, kRxThreads, rx_scatter_smem(q), 1, st, n, q, w.bsign, w.H,
                                             w.T, w.TF);
        // Not early: its blocks would wait where the scatter's leave room, several on an SM
        // (60,000 x 128 -> 16,384 26.8 us on the GPU, 23.3 this way, 20,000 x 50 -> 2,500 19.6 and
        // 17.7; a call 28.3 and 27.0, 25.2 and 24.3).
        LSK_PROF("cs_fine", st) rx_fine_kernel<<<(unsigned)q.B, kRxThreads, rx_fine_smem(q), st>>>(n, r, q, w.H, w.T, w.TF,
                                                                                                w.perm, w.off);
        *off_out = w.off;
        *perm_out = w.perm;
        return cudaGetLastError();
    }
    // the counters and the scan's state are contiguous: one memset
    e = cudaMemsetAsync(w.cnt, 0, (size_t)((char*)(w.state + scan_state_words(r)) - (char*)w.cnt), st);
    if (e != cudaSuccess) return e;
    if (n > 0) LSK_PROF("cs_count", st) cs_count_kernel<<<grid_for(n, 256, sm_count), 256, 0, st>>>(n, row0, (uint32_t)r, k0, k1, w.cnt);
    const unsigned tiles = (unsigned)((r + kScanTile - 1) / kScanTile);
    LSK_PROF("cs_scan", st) launch_chained(scan_early, scan_lookback_kernel, tiles, kScanBlock, 0, 1, st, w.cnt, w.off, w.cursor, r, w.state, flag);
    if (n > 0) {
        LSK_PROF("cs_place", st) cs_place_kernel<<<grid_for(n, 256, sm_count), 256, 0, st>>>(n, row0, (uint32_t)r, k0, k1, w.cursor, w.perm);
    }
    *off_out = w.off;
    *perm_out = w.perm;
    return cudaGetLastError();
}

// Parts of a bucket in the permutation's form: enough warps to stream A when there
// are few buckets, while each part keeps several rows (one part a bucket when
// compacting).
static int csr_parts(int64_t n, int64_t r, bool compact) {
    int P = 1;
    while (!compact && P < 32 && r * P < 16384 && n >= r * P * 8) P *= 2;
    return P;
}

// Matrices that the reductions of a CSR sketch are added to: one where the
// permutation's form sums an entry in one chain too, or where an entry has half a
// nonzero or fewer.  Of split buckets the partial sums are shorter chains, and two
// or four (all but the first in the workspace, added to it at the end) keep theirs as
// short: 200,000 x 64 -> 4,096 with 4 nonzeros to an entry is 4.5e-8 off with one,
// 4.2e-8 with two and by the permutation, 15 to an entry 7.7e-8, 5.8e-8 with four and
// 5.9e-8 (21 us, 14 with one, 45 by the permutation; 33, 25 and 70).
static int scatter_copies(const lsk_mat* A, int64_t r) {
    const int64_t entries = r * A->d;
    if (csr_parts(A->n, r, false) == 1 || 2 * A->nnz <= entries) return 1;
    return A->nnz / 4 <= entries ? 2 : 4;
}
size_t cs_scatter_copy_bytes(const lsk_mat* A, int64_t r, bool compact) {
    return cs_scatters(A, r, compact) ? (scatter_copies(A, r) - 1) * ws_round((size_t)r * A->d * 4) : 0;
}

// Every CSR sketch but a compacted one (which needs the buckets' counts), one of
// so few entries that the reductions queue up at their addresses (2^14), one
// that sums more than 16 nonzeros to an entry (there the permutation's form rounds
// less: r = 64 of 1M x 256 at 5%, 781 to an entry, 1.4e-7 against 5.0e-7 at 269 and 130
// us), and one whose copies would be large (16 MB each).
bool cs_scatters(const lsk_mat* A, int64_t r, bool compact) {
    const int64_t entries = r * A->d;
    return A->kind == LSK_CSR && !compact && entries >= (1 << 14) && r < ((int64_t)1 << 31) && A->nnz / 16 <= entries &&
           (scatter_copies(A, r) == 1 || entries <= (1 << 22));
}

cudaError_t cs_csr_scatter_launch(const lsk_mat* A, int64_t r, uint64_t seed, float* SA, float* copy, int* flag,
                                  int sm_count, cudaStream_t st, uint64_t row0, bool accumulate) {
    cudaError_t e;
    if (!accumulate && (e = cudaMemsetAsync(SA, 0, (size_t)r * A->d * 4, st)) != cudaSuccess) return e;
    if (A->n <= 0) return cudaSuccess;
    const int64_t entries = r * A->d, stride = (int64_t)ws_round((size_t)entries * 4) / 4;
    const int copies = scatter_copies(A, r);
    if (copies > 1 && (e = cudaMemsetAsync(copy, 0, (size_t)stride * 4 * (copies - 1), st)) != cudaSuccess) return e;
    LSK_PROF("cs_csr_scatter", st) cs_csr_scatter_kernel<<<grid_for(A->n, 256, sm_count, 32), 256, 0, st>>>(
        (const float*)A->values, A->colidx, A->rowptr, A->n, A->nnz, A->d, row0, (uint32_t)r, (uint32_t)seed,
        (uint32_t)(seed >> 32), SA, copy, stride, copies - 1, flag);
    if (copies > 1)
        LSK_PROF("cs_csr_scatter", st) cs_add_copies_kernel<<<grid_for(entries, 256, sm_count), 256, 0, st>>>(SA, copy, stride,
                                                                                                           copies - 1, entries);
    return cudaGetLastError();
}

cudaError_t cs_launch(const lsk_mat* A, int64_t r, uint64_t seed, float* SA, void* ws, int* flag,
                      int sm_count, cudaStream_t st, uint64_t row0, bool accumulate, uint32_t* cidx,
                      uint32_t* ccount, bool rx) {
    const int64_t n = A->n;
    const bool compact = cidx != nullptr && ccount != nullptr && !accumulate;
    // (without rx: a workspace of fixed size, which has no room for a second copy beyond its own)
    const size_t copy = cs_scatter_copy_bytes(A, r, compact);
    if (cs_scatters(A, r, compact) && (rx || copy <= cs_workspace_bytes_atomic(n, r)))
        return cs_csr_scatter_launch(A, r, seed, SA, (float*)ws, flag, sm_count, st, row0, accumulate);
    const uint32_t* off = nullptr;
    const uint32_t* perm = nullptr;
    // (the scan of many rows of CSR A plainly: 237,676 x 300 with 30 nonzeros a row -> 464 87.9
    // us on the GPU early, 82.3 plainly, 500,000 x 100 with ten -> 1,000 79.5 and 73.0; a call of
    // 44,670 x 32 -> 349 30.5 and 32.7)
    cudaError_t e = cs_prep_launch(n, r, seed, ws, sm_count, st, &off, &perm, row0, flag, rx,
                                   A->kind == LSK_DENSE || n < (1 << 17));
    if (e != cudaSuccess) return e;
    uint32_t* cpos = nullptr;
    if (compact) {
        cpos = cs_carve(ws, n, r, nullptr).cpos;   // the same place in either form
        LSK_PROF("cs_compact", st) cs_compact_kernel<<<1, 1024, 0, st>>>(off, r, cpos, cidx, ccount);
    }
    return cs_gather_launch(A, r, off, perm, cpos, SA, flag, sm_count, st, accumulate);
}

cudaError_t cs_gather_launch(const lsk_mat* A, int64_t r, const uint32_t* off, const uint32_t* perm,
                             const uint32_t* cpos, float* SA, int* flag, int sm_count, cudaStream_t st,
                             bool accumulate, bool early) {
    const int64_t n = A->n, d = A->d;
    cudaError_t e = cudaSuccess;
    const bool compact = cpos != nullptr;
    const int acc = accumulate ? 1 : 0;   // add into SA (shared buckets add atomically either way)
    if (A->kind == LSK_DENSE) {
        const float* Av = (const float*)A->values;
        const uintptr_t at = (uintptr_t)Av | (uintptr_t)SA | (uintptr_t)(4 * d) | (uintptr_t)(4 * A->ld);
        const int vec = (at & 15) == 0 ? 4 : (at & 7) == 0 ? 2 : 1;
        const int L = vec == 4 ? (d <= 32 ? 8 : d <= 64 ? 16 : 32) : 32;
        // Odd widths above 64 in one pass of four floats a lane: two passes follow every
        // chain of permutation and rows twice (1M x 101 -> 10,201 136 us, 113 in one; 30,000
        // x 127 -> 16,384 28.3 and 26.3).
        const int U = L < 32 ? 1 : vec == 4 ? (d <= 128 ? 1 : 2) : vec == 2 ? (d <= 64 ? 1 : 2) : d <= 32 ? 1 : d <= 64 ? 2 : 4;
        // one wave of teams, of four rows or four buckets (to store, empty ones too) at
        // least: with eight and sixteen 1,000 x 101 -> 3,000 took 19.8 us, 15.5 now
        const int64_t wave = (int64_t)sm_count * gather_per_sm(vec, U) * kGatherThreads / L;
        int64_t teams = std::max<int64_t>(1, std::min(wave, std::max((n + 3) / 4, (r + 3) / 4)));
        // one or two buckets a team where that makes them 16 rows at most: whole ones need
        // no zeroed SA
        if (!compact && r >= 2 && r < 2 * teams && n <= 8 * r) teams = r <= wave ? r : r / 2;
        // Whole buckets per team where each has eight of them, two that are short, or
        // one: the rows are then shared out to about an eighth, or to a few
        // dozen rows, and SA need not be zeroed.  A compacted SA holds no rows
        // for the empty buckets to zero, and its buckets are short.
        const int own = compact || r >= 8 * teams || (r >= 2 * teams && n <= 32 * r) || teams == r ? 1 : 0;
        if (!own && !accumulate && (e = cudaMemsetAsync(SA, 0, (size_t)r * d * 4, st)) != cudaSuccess) return e;
        const unsigned grid = (unsigned)((teams * L + kGatherThreads - 1) / kGatherThreads);
        // A long gather's blocks are not sent out while the permutation's last kernel
        // runs (without a memset of SA between the two): waiting beside that kernel's
        // blocks they cost more than they save.  1M x 200 -> 65,536 233 us against 190,
        // 300,000 x 100 -> 10,000 54 against 49, 100,000 x 256 -> 8,192 40 against 39;
        // 50,000 x 100 -> 10,000 26 against 29, 33,333 x 256 -> 65,536 33 against 36.
        if (own && n * d >= (1 << 24)) early = false;
        auto launch = [&](auto kernel) {
            LSK_PROF("cs_dense_gather", st) launch_chained(early, kernel, grid, kGatherThreads, 0, 1, st, Av, A->ld, d,
                                                           (uint32_t)r, off, perm, SA, teams, own, acc, cpos);
        };
        if (L == 8) launch(cs_dense_gather_kernel<4, 1, 8>);
        else if (L == 16) launch(cs_dense_gather_kernel<4, 1, 16>);
        else if (vec == 4 && U == 1) launch(cs_dense_gather_kernel<4, 1, 32>);
        else if (vec == 4) launch(cs_dense_gather_kernel<4, 2, 32>);
        else if (vec == 2 && U == 1) launch(cs_dense_gather_kernel<2, 1, 32>);
        else if (vec == 2) launch(cs_dense_gather_kernel<2, 2, 32>);
        else if (U == 1) launch(cs_dense_gather_kernel<1, 1, 32>);
        else if (U == 2) launch(cs_dense_gather_kernel<1, 2, 32>);
        else launch(cs_dense_gather_kernel<1, 4, 32>);
    } else {
        // shared-memory row per warp: pick warps per block to fit 200 KB
        int warps = 8;
        while (warps > 1 && (size_t)warps * d * 4 > 200 * 1024) warps >>= 1;
        const size_t smem = (size_t)warps * d * 4;
        if (smem > 200 * 1024) return cudaErrorInvalidValue;
        const int P = csr_parts(n, r, compact);
        if (P > 1 && !accumulate && (e = cudaMemsetAsync(SA, 0, (size_t)r * d * 4, st)) != cudaSuccess) return e;
        const int64_t warps_needed = r * P;
        if (smem > 48 * 1024) {
            e = allow_dynamic_smem(cs_csr_gather_kernel);
            if (e != cudaSuccess) return e;
        }
        const int threads = warps * 32;
        int64_t g = (warps_needed + warps - 1) / warps;
        const int64_t cap = (int64_t)sm_count * 32 / warps * 2;
        if (g > cap) g = cap;
        if (g < 1) g = 1;
        LSK_PROF("cs_csr_gather", st) cs_csr_gather_kernel<<<(unsigned)g, threads, smem, st>>>(
            (const float*)A->values, A->colidx, A->rowptr, A->nnz, d, (uint32_t)r, off, perm, SA, flag, P, acc, cpos);
    }
    return cudaGetLastError();
}

size_t cs_group_ws_bytes(int64_t rows, int64_t counters) {
    return ws_round((size_t)(counters + 1) * 4) * 4 + ws_round((size_t)(rows > 0 ? rows : 1) * 4) +
           ws_round(scan_state_words(counters) * 8) + 2048;
}

void cs_group_build(std::vector<CsJob>& jobs, void* ws, HostTable& t, CsGroup& g) {
    std::vector<CsGp> ps(jobs.size());
    std::vector<int> blocks(jobs.size()), boff;
    int64_t cb = 0;
    g.any_compact = false;
    g.rows = 0;
    for (size_t i = 0; i < jobs.size(); ++i) {
        CsJob& j = jobs[i];
        j.cnt_base = cb;
        ps[i] = CsGp{j.n, j.r, cb, (uint32_t)j.seed, (uint32_t)(j.seed >> 32), j.cidx, j.ccount};
        const int64_t run = group_run(j.n, j.r);
        blocks[i] = (int)((j.n + run - 1) / run);
        g.rows += j.n;
        cb += j.r + 1;
        g.any_compact = g.any_compact || j.cidx != nullptr;
    }
    g.count = (int)jobs.size();
    g.blocks = group_offsets(blocks, boff);
    g.counters = cb;
    WsCarver wc{(char*)ws, 0};
    g.cnt = wc.take<uint32_t>((size_t)g.counters);
    g.state = wc.take<unsigned long long>(scan_state_words(g.counters));
    g.off = wc.take<uint32_t>((size_t)g.counters + 1);
    g.cursor = wc.take<uint32_t>((size_t)g.counters);
    g.cpos = wc.take<uint32_t>((size_t)g.counters);
    g.perm = wc.take<uint32_t>((size_t)(g.rows > 0 ? g.rows : 1));
    g.params_off = t.put(ps.data(), ps.size());
    g.boff_off = t.put(boff.data(), boff.size());
}

cudaError_t cs_group_launch(const CsGroup& g, const unsigned char* table, int* flag, cudaStream_t st) {
    if (g.count == 0) return cudaSuccess;
    const CsGp* ps = reinterpret_cast<const CsGp*>(table + g.params_off);
    const int* boff = reinterpret_cast<const int*>(table + g.boff_off);
    // the counters and the scan's state are contiguous: one memset
    cudaError_t e = cudaMemsetAsync(
        g.cnt, 0, (size_t)((char*)(g.state + scan_state_words(g.counters)) - (char*)g.cnt), st);
    if (e != cudaSuccess) return e;
    if (g.blocks > 0)
        LSK_PROF("cs_count", st) cs_rows_grouped_kernel<false><<<g.blocks, kGroupThreads, 0, st>>>(
            ps, boff, g.count, g.cnt, nullptr);
    LSK_PROF("cs_scan", st) launch_pdl(scan_lookback_kernel, (unsigned)((g.counters + kScanTile - 1) / kScanTile), kScanBlock,
                                        0, 1, st, g.cnt, g.off, g.cursor, g.counters, g.state, flag);
    if (g.blocks > 0)
        LSK_PROF("cs_place", st) cs_rows_grouped_kernel<true><<<g.blocks, kGroupThreads, 0, st>>>(
            ps, boff, g.count, g.cursor, g.perm);
    if (g.any_compact)
        LSK_PROF("cs_compact", st) cs_compact_grouped_kernel<<<g.count, 1024, 0, st>>>(ps, g.off, g.cpos);
    return cudaGetLastError();
}
