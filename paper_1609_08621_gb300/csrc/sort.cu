// Device-wide exclusive scan and stable LSD radix sort of (63-bit Morton key, index) pairs.
//
// The sort produces the "hierarchically sorted order" of the particles (Sec. 3.1):
// particles ordered by Morton key, ties kept in input order (the sort is stable and
// starts from the identity permutation).  8 passes of 8-bit digits; each pass is a
// per-tile digit histogram, an exclusive scan of the (digit, tile) counts in
// digit-major order (a block per digit), and a stable scatter that ranks keys within the tile with
// warp match masks and stages the tile in shared memory so that global writes are
// runs of equal digits.
#include <utility>

#include "fmm_internal.cuh"

#define SCAN_THREADS 1024
#define SCAN_ITEMS 4
#define SCAN_TILE (SCAN_THREADS * SCAN_ITEMS)

#define RS_THREADS 256
#define RS_WARPS (RS_THREADS / 32)
#define RS_ITEMS 8  // tree phase of a 384^3 / 128^3 box: 26.8 / 1.40 ms with 8, 27.3 / 1.42 with 12, 28.4 / 1.45 with 16
#define RS_TILE (RS_THREADS * RS_ITEMS)

// inclusive block scan of one value per thread (blockDim.x multiple of 32, <= 1024)
__device__ __forceinline__ unsigned int block_inclusive_scan(unsigned int v, unsigned int* sh /* 32 */,
                                                             unsigned int* total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned int t = __shfl_up_sync(FMM_FULL_MASK, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        unsigned int s = lane < nw ? sh[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned int t = __shfl_up_sync(FMM_FULL_MASK, s, o);
            if (lane >= o) s += t;
        }
        sh[lane] = s;
    }
    __syncthreads();
    unsigned int add = w > 0 ? sh[w - 1] : 0u;
    if (total) *total = sh[nw - 1];
    __syncthreads();
    return v + add;
}

// this thread's four values of the tile, zeros past n; one 16-byte load where the tile is aligned for it
__device__ __forceinline__ uint4 scan_load(const unsigned int* __restrict__ in, long long base, long long n)
{
    if (base + 3 < n && (reinterpret_cast<size_t>(in) & 15) == 0) return *reinterpret_cast<const uint4*>(in + base);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (base < n) v.x = in[base];
    if (base + 1 < n) v.y = in[base + 1];
    if (base + 2 < n) v.z = in[base + 2];
    if (base + 3 < n) v.w = in[base + 3];
    return v;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(const unsigned int* __restrict__ in, long long n,
                                                              unsigned int* __restrict__ part)
{
    __shared__ unsigned int sh[32];
    const uint4 v = scan_load(in, (long long)blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_ITEMS, n);
    unsigned int tot;
    block_inclusive_scan(v.x + v.y + v.z + v.w, sh, &tot);
    if (threadIdx.x == 0) part[blockIdx.x] = tot;
}

// exclusive scan of the per-tile sums in place, one block, any length
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_parts(unsigned int* __restrict__ part, long long np)
{
    __shared__ unsigned int sh[32];
    long long per = fmm_ceil_div(np, SCAN_THREADS);
    long long b = (long long)threadIdx.x * per, e = b + per < np ? b + per : np;
    unsigned int s = 0;
    for (long long i = b; i < e; i++) s += part[i];
    unsigned int incl = block_inclusive_scan(s, sh, nullptr);
    unsigned int run = incl - s;
    for (long long i = b; i < e; i++) {
        unsigned int v = part[i];
        part[i] = run;
        run += v;
    }
}

// The tile's values from the sums of the tiles before it: part[blockIdx.x] where k_scan_parts has run
// (SCANNED), else added up here; the last tile writes the total.
template <bool SCANNED>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_down(const unsigned int* in, unsigned int* out, long long n,
                                                            const unsigned int* __restrict__ part,
                                                            unsigned int* __restrict__ total)
{
    __shared__ unsigned int sh[32];
    const long long base = (long long)blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_ITEMS;
    const uint4 v = scan_load(in, base, n);
    unsigned int before = 0;
    if (SCANNED) {
        before = part[blockIdx.x];
    } else if (blockIdx.x > 0) {
        unsigned int p = 0;
        for (int i = threadIdx.x; i < (int)blockIdx.x; i += SCAN_THREADS) p += part[i];
        block_inclusive_scan(p, sh, &before);
    }
    const unsigned int s = v.x + v.y + v.z + v.w, incl = block_inclusive_scan(s, sh, nullptr), run = before + incl - s;
    const uint4 r = make_uint4(run, run + v.x, run + v.x + v.y, run + v.x + v.y + v.z);
    if (base + 3 < n && (reinterpret_cast<size_t>(out) & 15) == 0) {
        *reinterpret_cast<uint4*>(out + base) = r;
    } else {
        if (base < n) out[base] = r.x;
        if (base + 1 < n) out[base + 1] = r.y;
        if (base + 2 < n) out[base + 2] = r.z;
        if (base + 3 < n) out[base + 3] = r.w;
    }
    if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == SCAN_THREADS - 1) *total = before + incl;
}

static cudaError_t ensure_u32(unsigned int** p, long long* cap, long long need)
{
    if (need <= *cap) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    cudaError_t e = cudaMalloc(p, (size_t)need * sizeof(unsigned int));
    if (e == cudaSuccess) *cap = need;
    return e;
}

// scratch of fmm_scan_exclusive for scans of up to n values, allocated ahead (graph capture)
cudaError_t fmm_scan_reserve(DevTree& t, long long n)
{
    return ensure_u32(&t.scan_part, &t.cap_scan_part, fmm_ceil_div(n, SCAN_TILE));
}

// Exclusive scan: one launch for a single tile, two while a tile can add up the sums before it itself
// (up to SCAN_DIRECT of them, two per thread), three beyond.  Every launch costs about 2.5 us of a
// small solve, which scans six times.
#define SCAN_DIRECT (2 * SCAN_THREADS)
cudaError_t fmm_scan_exclusive(const unsigned int* in, unsigned int* out, long long n, unsigned int* total_dev,
                               DevTree& t, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    long long nb = fmm_ceil_div(n, SCAN_TILE);
    cudaError_t e = ensure_u32(&t.scan_part, &t.cap_scan_part, nb);
    if (e != cudaSuccess) return e;
    if (nb > 1) k_scan_reduce<<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, t.scan_part);
    if (nb > SCAN_DIRECT) {
        k_scan_parts<<<1, SCAN_THREADS, 0, s>>>(t.scan_part, nb);
        k_scan_down<true><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, out, n, t.scan_part, total_dev);
    } else {
        k_scan_down<false><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, out, n, t.scan_part, total_dev);
    }
    t.n_launches += nb == 1 ? 1 : nb > SCAN_DIRECT ? 3 : 2;
    return cudaGetLastError();
}

// ---------------------------------------------------------------- radix sort

__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const unsigned long long* __restrict__ kin, long long n,
                                                        int shift, unsigned int* __restrict__ hist, int nblk,
                                                        unsigned int* __restrict__ tot)
{
    __shared__ unsigned int c[RS_WARPS * 256];
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    for (int i = tid; i < RS_WARPS * 256; i += RS_THREADS) c[i] = 0;
    __syncthreads();
    const long long t0 = (long long)blockIdx.x * RS_TILE + (long long)w * 32 * RS_ITEMS;
    // one count per key with shared-memory atomics into the warp's own counters (matching lanes first, as
    // the scatter must to rank them, costs more than the conflicts it saves)
#pragma unroll
    for (int r = 0; r < RS_ITEMS; r++) {
        const long long i = t0 + r * 32 + lane;
        if (i < n) atomicAdd(&c[w * 256 + (unsigned int)((kin[i] >> shift) & 255u)], 1u);
    }
    __syncthreads();
    unsigned int s = 0;
#pragma unroll
    for (int ww = 0; ww < RS_WARPS; ww++) s += c[ww * 256 + tid];
    hist[(long long)tid * nblk + blockIdx.x] = s;
    if (s) atomicAdd(tot + tid, s);  // keys of this digit in all tiles
}

// First output position of every (digit, tile): a block per digit, from the digits' totals and the
// exclusive scan of the digit's row of counts, in place.
__global__ void __launch_bounds__(SCAN_THREADS) k_rs_scan(unsigned int* __restrict__ hist, int nblk,
                                                          const unsigned int* __restrict__ tot)
{
    __shared__ unsigned int sh[32];
    const int tid = threadIdx.x;
    unsigned int run;  // keys before this digit, then before this round's tiles
    block_inclusive_scan(tid < (int)blockIdx.x ? tot[tid] : 0u, sh, &run);
    unsigned int* const row = hist + (long long)blockIdx.x * nblk;
    for (int b = 0; b < nblk; b += SCAN_THREADS) {
        const unsigned int v = b + tid < nblk ? row[b + tid] : 0u;
        unsigned int sum;
        const unsigned int incl = block_inclusive_scan(v, sh, &sum);
        if (b + tid < nblk) row[b + tid] = run + incl - v;
        run += sum;
    }
}

__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const unsigned long long* __restrict__ kin,
                                                           const unsigned int* __restrict__ vin,
                                                           unsigned long long* __restrict__ kout,
                                                           unsigned int* __restrict__ vout, long long n, int shift,
                                                           const unsigned int* __restrict__ offs, int nblk)
{
    extern __shared__ __align__(16) unsigned char rs_smem[];
    unsigned long long* sk = reinterpret_cast<unsigned long long*>(rs_smem);
    unsigned int* sv = reinterpret_cast<unsigned int*>(sk + RS_TILE);
    unsigned int* wcnt = sv + RS_TILE;          // RS_WARPS * 256
    unsigned int* dstart = wcnt + RS_WARPS * 256;  // 256
    unsigned int* gbase = dstart + 256;         // 256
    unsigned int* sh = gbase + 256;             // 32
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const long long tile0 = (long long)blockIdx.x * RS_TILE;
    for (int i = tid; i < RS_WARPS * 256; i += RS_THREADS) wcnt[i] = 0;
    gbase[tid] = offs[(long long)tid * nblk + blockIdx.x];
    __syncthreads();
    unsigned long long k[RS_ITEMS];
    unsigned int v[RS_ITEMS], lp[RS_ITEMS];
    const unsigned int lt = fmm_lanemask_lt();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; r++) {
        long long i = tile0 + (long long)w * 32 * RS_ITEMS + r * 32 + lane;
        bool ok = i < n;
        k[r] = ok ? kin[i] : 0ull;
        v[r] = ok ? vin[i] : 0u;
        unsigned int d = ok ? (unsigned int)((k[r] >> shift) & 255u) : 256u;
        unsigned int peers = __match_any_sync(FMM_FULL_MASK, d);
        unsigned int rank = __popc(peers & lt);
        unsigned int before = ok ? wcnt[w * 256 + d] : 0u;
        __syncwarp();
        if (ok && rank == 0) wcnt[w * 256 + d] = before + __popc(peers);
        __syncwarp();
        lp[r] = before + rank;
    }
    __syncthreads();
    // per digit: exclusive scan over warps; block total
    unsigned int run = 0;
#pragma unroll
    for (int ww = 0; ww < RS_WARPS; ww++) {
        unsigned int c = wcnt[ww * 256 + tid];
        wcnt[ww * 256 + tid] = run;
        run += c;
    }
    unsigned int incl = block_inclusive_scan(run, sh, nullptr);
    dstart[tid] = incl - run;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ITEMS; r++) {
        long long i = tile0 + (long long)w * 32 * RS_ITEMS + r * 32 + lane;
        if (i < n) {
            unsigned int d = (unsigned int)((k[r] >> shift) & 255u);
            unsigned int pos = dstart[d] + wcnt[w * 256 + d] + lp[r];
            sk[pos] = k[r];
            sv[pos] = v[r];
        }
    }
    __syncthreads();
    long long rem = n - tile0;
    int cnt = rem < RS_TILE ? (int)rem : RS_TILE;
    for (int i = tid; i < cnt; i += RS_THREADS) {
        unsigned long long kk = sk[i];
        unsigned int d = (unsigned int)((kk >> shift) & 255u);
        unsigned long long g = (unsigned long long)gbase[d] + (unsigned long long)(i - (int)dstart[d]);
        kout[g] = kk;
        vout[g] = sv[i];
    }
}

// A sort of at most RS_SMALL keys in one block, all passes in shared memory: warp w holds keys
// [32 I w, 32 I (w + 1)), ranks its own with match masks, and the digits' starts come from one block
// scan over (digit, quarter of the warps).  Eight passes of a 4096-particle box take one launch instead
// of 40 (or 24 with the digit rows scanned by one kernel).
#define RS_SMALL 8192
#define RS_SMALL_THREADS 1024
struct SortSmall {
    unsigned long long k[RS_SMALL];
    unsigned int v[RS_SMALL];
    unsigned short cnt[32 * 256];  // [warp][digit]
    unsigned int sh[32];
};
template <int I>
__global__ void __launch_bounds__(RS_SMALL_THREADS) k_rs_small(unsigned long long* key, unsigned int* val, int n, int passes)
{
    extern __shared__ __align__(16) unsigned char rs_smem[];
    SortSmall& S = *reinterpret_cast<SortSmall*>(rs_smem);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const unsigned int lt = fmm_lanemask_lt();
    for (int i = tid; i < n; i += RS_SMALL_THREADS) {
        S.k[i] = key[i];
        S.v[i] = val[i];
    }
    for (int pass = 0; pass < passes; pass++) {
        const int shift = 8 * pass;
        for (int i = tid; i < 32 * 256 / 2; i += RS_SMALL_THREADS) reinterpret_cast<unsigned int*>(S.cnt)[i] = 0u;
        __syncthreads();
        unsigned long long k[I];
        unsigned int v[I], rank[I];
#pragma unroll
        for (int r = 0; r < I; r++) {
            const int i = (w * I + r) * 32 + lane;
            const bool ok = i < n;
            k[r] = ok ? S.k[i] : 0ull;
            v[r] = ok ? S.v[i] : 0u;
            const unsigned int d = ok ? (unsigned int)((k[r] >> shift) & 255u) : 256u;
            const unsigned int peers = __match_any_sync(FMM_FULL_MASK, d);
            const unsigned int before = ok ? S.cnt[w * 256 + d] : 0u;
            __syncwarp();
            if (ok && (peers & lt) == 0) S.cnt[w * 256 + d] = (unsigned short)(before + __popc(peers));
            __syncwarp();
            rank[r] = before + __popc(peers & lt);
        }
        __syncthreads();
        // thread (digit, quarter): starts of its 8 warps' keys of the digit
        const int d = tid >> 2, q = (tid & 3) * 8;
        unsigned int c[8], sum = 0;
#pragma unroll
        for (int u = 0; u < 8; u++) {
            c[u] = S.cnt[(q + u) * 256 + d];
            sum += c[u];
        }
        unsigned int run = block_inclusive_scan(sum, S.sh, nullptr) - sum;
#pragma unroll
        for (int u = 0; u < 8; u++) {
            S.cnt[(q + u) * 256 + d] = (unsigned short)run;
            run += c[u];
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < I; r++) {
            if ((w * I + r) * 32 + lane < n) {
                const unsigned int p = S.cnt[w * 256 + ((k[r] >> shift) & 255u)] + rank[r];
                S.k[p] = k[r];
                S.v[p] = v[r];
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < n; i += RS_SMALL_THREADS) {
        key[i] = S.k[i];
        val[i] = S.v[i];
    }
}

static size_t rs_smem_bytes()
{
    return (size_t)RS_TILE * 8 + (size_t)RS_TILE * 4 + (RS_WARPS * 256 + 256 + 256 + 32) * 4;
}

// Lets the sort's kernels use their shared memory on the current device.
static std::atomic<unsigned long long> g_rs_attr{0}, g_rs1_attr{0}, g_rs2_attr{0}, g_rs4_attr{0}, g_rs8_attr{0};
cudaError_t fmm_sort_prepare()
{
    cudaError_t e = fmm_smem_attr_once(k_rs_scatter, (int)rs_smem_bytes(), g_rs_attr);
    if (e == cudaSuccess) e = fmm_smem_attr_once(k_rs_small<1>, (int)sizeof(SortSmall), g_rs1_attr);
    if (e == cudaSuccess) e = fmm_smem_attr_once(k_rs_small<2>, (int)sizeof(SortSmall), g_rs2_attr);
    if (e == cudaSuccess) e = fmm_smem_attr_once(k_rs_small<4>, (int)sizeof(SortSmall), g_rs4_attr);
    if (e == cudaSuccess) e = fmm_smem_attr_once(k_rs_small<8>, (int)sizeof(SortSmall), g_rs8_attr);
    return e;
}

// Scratch entries the sort needs for n keys: digit counts (256 per tile), and the digits' totals of
// up to 8 passes.
long long fmm_sort_hist_entries(long long n) { return 256LL * fmm_ceil_div(n, RS_TILE); }
long long fmm_sort_part_entries(long long n)
{
    (void)n;
    return 256LL * 8;
}

cudaError_t fmm_sort_ensure(DevTree& t, long long n)
{
    cudaError_t e = ensure_u32(&t.hist, &t.cap_hist, fmm_sort_hist_entries(n) + fmm_sort_part_entries(n));
    if (e != cudaSuccess) return e;
    return fmm_sort_prepare();
}

// Stable LSD sort of n (key, value) pairs on the low 8 * passes key bits (passes even, at most 8): the
// result is back in ka / va; kb / vb are scratch of the same size, hist and tot of the sizes above.
// Nothing is allocated here; fmm_sort_prepare must have run on the current device.  Returns the
// launches in *launches.
cudaError_t fmm_radix_sort_kv_scratch(unsigned long long* ka, unsigned long long* kb, unsigned int* va,
                                      unsigned int* vb, long long n, int passes, unsigned int* hist,
                                      unsigned int* tot, int* launches, cudaStream_t s)
{
    *launches = 0;
    if (n <= 1) return cudaSuccess;
    if (n <= RS_SMALL) {
        const size_t smem = sizeof(SortSmall);
        const int per = (int)fmm_ceil_div(n, RS_SMALL_THREADS);
        if (per <= 1) k_rs_small<1><<<1, RS_SMALL_THREADS, smem, s>>>(ka, va, (int)n, passes);
        else if (per <= 2) k_rs_small<2><<<1, RS_SMALL_THREADS, smem, s>>>(ka, va, (int)n, passes);
        else if (per <= 4) k_rs_small<4><<<1, RS_SMALL_THREADS, smem, s>>>(ka, va, (int)n, passes);
        else k_rs_small<8><<<1, RS_SMALL_THREADS, smem, s>>>(ka, va, (int)n, passes);
        *launches = 1;
        return cudaGetLastError();
    }
    const int nblk = (int)fmm_ceil_div(n, RS_TILE);
    cudaError_t e = cudaMemsetAsync(tot, 0, sizeof(unsigned int) * 256 * (size_t)passes, s);
    if (e != cudaSuccess) return e;
    for (int pass = 0; pass < passes; pass++) {
        const int shift = 8 * pass;
        k_rs_hist<<<nblk, RS_THREADS, 0, s>>>(ka, n, shift, hist, nblk, tot + 256 * pass);
        k_rs_scan<<<256, SCAN_THREADS, 0, s>>>(hist, nblk, tot + 256 * pass);
        k_rs_scatter<<<nblk, RS_THREADS, rs_smem_bytes(), s>>>(ka, va, kb, vb, n, shift, hist, nblk);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    *launches = 3 * passes;
    return cudaGetLastError();
}

cudaError_t fmm_radix_sort_kv(unsigned long long* ka, unsigned long long* kb, unsigned int* va, unsigned int* vb,
                              long long n, int passes, DevTree& t, cudaStream_t s)
{
    cudaError_t e = fmm_sort_ensure(t, n);
    if (e != cudaSuccess) return e;
    int launches = 0;
    e = fmm_radix_sort_kv_scratch(ka, kb, va, vb, n, passes, t.hist, t.hist + fmm_sort_hist_entries(n), &launches, s);
    t.n_launches += launches;
    return e;
}

// sorts t.key / t.idx (n elements) on all 64 key bits
cudaError_t fmm_radix_sort(DevTree& t, long long n, cudaStream_t s)
{
    return fmm_radix_sort_kv(t.key, t.key_alt, t.idx, t.idx_alt, n, 8, t, s);
}
