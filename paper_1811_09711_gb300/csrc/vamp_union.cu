// vamp_union.cu -- interval tables of the union pass (vamp_union.cuh) and
// its kernel variants.
//
// After every change of the grids (creation, rebinning, state upload) the
// tables are rebuilt from the FP64 master grids, coordinate by coordinate:
//   k_union_images  image of every edge under its channel's map,
//                   v = φ_c(ξ_{c,k,j}) in FP64 (the forward map's formula),
//                   rounded up to FP32: for an FP32 p, p >= v32 exactly when
//                   p >= v, so comparing p with the images decides the bin
//                   as comparing φ_c^{-1}(p) with the edges does;
//   k_union_sort    the K (n+1) images of a coordinate in order, by merging
//                   the K rows two by two; the distinct ones: U_k;
//   k_union_cells   for each of UNION_CELLS equal cells [q/L, (q+1)/L) the
//                   count of U_k values <= q/L and the count inside the cell;
//   k_union_rows    for each interval [U_k[u], U_k[u+1]) and channel c the
//                   FP32 density 1/(nΔx) of the bin of row (c, k) whose image
//                   holds it: the largest j <= n-1 with image_j <= U_k[u]
//                   (bin 0 below the first image), from the lookup block.
// For the collider (d = 14, K = 64, n = 100) they take 5, 22, 7 and 19 us, the
// first three bounded by latency and the last by writing 23 MB of densities.
// A bitonic sort, two searches per cell and a search per density took 70, 18
// and 49; placing every image by a search in its neighbour list at each merge
// 48, in every other channel's row 49; a thread filling the cells up to its
// value's successor 75 to 125, long gaps being filled by one thread.
#include "vamp_union.cuh"

#include <algorithm>

namespace vamp {

namespace {

__global__ void k_union_images(Params P)
{
    const int d = P.d, K = P.K, n1 = P.n + 1;
    const int64_t tot = (int64_t)d * K * n1;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(t % n1);
        const int c = (int)((t / n1) % K);
        const int k = (int)(t / ((int64_t)n1 * K));
        const double e = P.edges64[((size_t)c * d + k) * n1 + j];
        const ChanHdr<double>& h = *reinterpret_cast<const ChanHdr<double>*>(P.lk64 + (size_t)c * P.lay64.bytes);
        const int s = map_slot(h, k);
        const double v = s >= 0 ? edge_image(h, s, e) : e;
        P.uImg[t] = __double2float_ru(v);  // [k][c][j]
    }
}

constexpr int SORT_THREADS = 1024;

__device__ __forceinline__ int pow2_floor(int v) { return 1 << (31 - __clz(v)); }

// One block per coordinate; dynamic shared memory: the K (n+1) images twice.
__global__ void __launch_bounds__(SORT_THREADS, 1) k_union_sort(Params P)
{
    extern __shared__ float sv[];
    __shared__ int wsum[SORT_THREADS / 32];
    const int k = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int K = P.K, n1 = P.n + 1, m = K * n1;
    float *src = sv, *dst = sv + m;
    // The rows are sorted as they come; a running maximum keeps them so where
    // the forward map's rounding turned two neighbours round (the merges below
    // and the walk of k_union_rows rest on it).
    for (int c = wid; c < K; c += SORT_THREADS / 32) {
        float* img = P.uImg + (size_t)k * m + (size_t)c * n1;
        float top = -INFINITY;
        for (int j0 = 0; j0 < n1; j0 += 32) {
            const int j = j0 + lane;
            const float raw = j < n1 ? img[j] : -INFINITY;
            float v = fmaxf(raw, top);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) v = fmaxf(v, __shfl_up_sync(0xffffffffu, v, o));
            top = __shfl_sync(0xffffffffu, v, 31);
            if (j < n1) {
                src[c * n1 + j] = v;
                if (v != raw) img[j] = v;
            }
        }
    }
    __syncthreads();
    // Neighbouring lists of w values merge into one, equal values of the left
    // list first.  Each thread makes a run of outputs: where the two lists
    // stand at its start by a search along the diagonal, then value by value.
    // The runs have odd length, so that a warp's accesses spread over the banks.
    const int per = ((m + SORT_THREADS - 1) / SORT_THREADS) | 1;
    const int i0 = min(tid * per, m), i1 = min(i0 + per, m);
    for (int w = n1; w < m; w *= 2) {
        for (int o = i0; o < i1;) {
            const int p0 = o / (2 * w) * (2 * w), t = o - p0;
            const int la = min(w, m - p0), lb = min(w, m - p0 - la), end = min(i1, p0 + la + lb);
            const float *A = src + p0, *B = A + la;
            int lo = max(0, t - lb), hi = min(t, la);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (A[mid] <= B[t - 1 - mid]) lo = mid + 1; else hi = mid;
            }
            int i = lo, j = t - lo;
            for (; o < end; ++o) {
                const bool left = j >= lb || (i < la && !(B[j] < A[i]));
                dst[o] = left ? A[i] : B[j];
                if (left) ++i; else ++j;
            }
        }
        __syncthreads();
        float* t = src;
        src = dst;
        dst = t;
    }
    // distinct values, in order: a block scan of the runs' counts
    int cnt = 0;
    for (int i = i0; i < i1; ++i) cnt += (i == 0 || src[i] != src[i - 1]) ? 1 : 0;
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int w = wsum[lane];
        int iw = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, iw, o);
            if (lane >= o) iw += y;
        }
        wsum[lane] = iw;  // inclusive prefix of the warp totals
    }
    __syncthreads();
    int pos = (wid ? wsum[wid - 1] : 0) + incl - cnt;
    const int nu = wsum[SORT_THREADS / 32 - 1];
    for (int i = i0; i < i1; ++i)
        if (i == 0 || src[i] != src[i - 1]) dst[pos++] = src[i];
    __syncthreads();
    if (tid == 0) P.uNU[k] = nu;
    float* U = P.uU + (size_t)k * P.uMax;
    for (int i = tid; i < nu; i += SORT_THREADS) U[i] = dst[i];
}

constexpr int CELL_THREADS = 1024;
constexpr int CELLS_PER_BLOCK = 4 * CELL_THREADS;

// Block (cell range, coordinate).  Value i is counted from the first cell
// boundary at or above it on, and lies inside the cell before that boundary
// unless it is on it; a running maximum of i+1 over the cells is the count at
// or below their starts.  The last cell of all takes every value above its
// start.
__global__ void __launch_bounds__(CELL_THREADS) k_union_cells(Params P)
{
    __shared__ __align__(16) int le[CELLS_PER_BLOCK], in[CELLS_PER_BLOCK];
    __shared__ int wtop[CELL_THREADS / 32];
    const int k = blockIdx.y, q0 = blockIdx.x * CELLS_PER_BLOCK, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nu = P.uNU[k];
    const float* U = P.uU + (size_t)k * P.uMax;
    const float L = (float)UNION_CELLS;  // a power of two: the products are exact
    reinterpret_cast<int4*>(le)[tid] = make_int4(0, 0, 0, 0);
    reinterpret_cast<int4*>(in)[tid] = make_int4(0, 0, 0, 0);
    __syncthreads();
    int before = 0;
    for (int i = tid; i < nu; i += CELL_THREADS) {
        const float x = fminf(fmaxf(U[i] * L, -1.f), L + 1.f);
        const int a = (int)ceilf(x) - q0, b = (int)floorf(x) - q0;
        if (a <= 0) before = i + 1;
        else if (a < CELLS_PER_BLOCK) atomicMax(&le[a], i + 1);
        if (b != a && b >= 0 && b < CELLS_PER_BLOCK) atomicAdd(&in[b], 1);
    }
    if (before) atomicMax(&le[0], before);
    __syncthreads();
    int4 v = reinterpret_cast<int4*>(le)[tid];
    const int4 w = reinterpret_cast<int4*>(in)[tid];
    v.y = max(v.x, v.y);
    v.z = max(v.y, v.z);
    v.w = max(v.z, v.w);
    int top = v.w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, top, o);
        if (lane >= o) top = max(top, y);
    }
    if (lane == 31) wtop[wid] = top;
    __syncthreads();
    if (wid == 0) {
        int y = wtop[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int z = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y = max(y, z);
        }
        wtop[lane] = y;
    }
    __syncthreads();
    int pre = __shfl_up_sync(0xffffffffu, top, 1);
    if (lane == 0) pre = 0;
    if (wid) pre = max(pre, wtop[wid - 1]);
    v.x = max(v.x, pre);
    v.y = max(v.y, pre);
    v.z = max(v.z, pre);
    v.w = max(v.w, pre);
    uint4 out = make_uint4((uint32_t)v.x | ((uint32_t)w.x << 16), (uint32_t)v.y | ((uint32_t)w.y << 16),
                           (uint32_t)v.z | ((uint32_t)w.z << 16), (uint32_t)v.w | ((uint32_t)w.w << 16));
    if (q0 + 4 * tid + 3 == UNION_CELLS - 1) out.w = (uint32_t)v.w | ((uint32_t)(nu - v.w) << 16);
    reinterpret_cast<uint4*>(P.uC + (size_t)k * UNION_CELLS + q0)[tid] = out;
}

constexpr int ROWS_THREADS = 1024;
constexpr int ROWS_GROUPS = ROWS_THREADS / UNION_SLOTS;
constexpr int ROWS_PER_BLOCK = 512;

// Block (u-range, coordinate); dynamic shared memory: the K (n+1) images and
// the K n densities of the coordinate.  A thread walks one channel through
// consecutive intervals, its bin moving on from one to the next.
__global__ void __launch_bounds__(ROWS_THREADS) k_union_rows(Params P)
{
    extern __shared__ float im[];
    const int k = blockIdx.y;
    const int nu = P.uNU[k];
    const int u0 = blockIdx.x * ROWS_PER_BLOCK;
    if (u0 >= nu) return;
    const int K = P.K, n = P.n, n1 = n + 1, m = K * n1;
    const BlkLayout& L = P.lay32;
    float* den = im + m;
    const float* src = P.uImg + (size_t)k * m;
    for (int i = threadIdx.x; i < m; i += ROWS_THREADS) im[i] = src[i];
    for (int c = threadIdx.x >> 5; c < K; c += ROWS_THREADS / 32) {
        const float* dn = reinterpret_cast<const float*>(P.lk32 + (size_t)c * L.bytes + L.H + (size_t)k * L.R +
                                                         (size_t)L.Es * sizeof(float));
        for (int j = threadIdx.x & 31; j < n; j += 32) den[c * n + j] = dn[j];
    }
    __syncthreads();
    constexpr int PER = ROWS_PER_BLOCK / ROWS_GROUPS;
    const int c = threadIdx.x % UNION_SLOTS, a = u0 + threadIdx.x / UNION_SLOTS * PER, b = min(nu, a + PER);
    if (a >= b) return;
    const float* U = P.uU + (size_t)k * P.uMax;
    float* out = P.uD + ((size_t)k * P.uMax + a) * UNION_SLOTS + c;
    if (c >= K) {
        for (int u = a; u < b; ++u, out += UNION_SLOTS) *out = 0.f;
        return;
    }
    const float* e = im + c * n1;
    const float* dn = den + c * n;
    // largest j in [0, n-1] with e[j] <= U[a] (0 if none)
    int j = 0;
    const float xa = __ldg(U + a);
    for (int s = pow2_floor(n); s; s >>= 1)
        if (j + s < n && e[j + s] <= xa) j += s;
#pragma unroll 4
    for (int u = a; u < b; ++u, out += UNION_SLOTS) {
        const float x = __ldg(U + u);
        while (j < n - 1 && e[j + 1] <= x) ++j;
        *out = dn[j];
    }
}

}  // namespace

bool union_fits(int fp32, int d, int K, int n, int stratified)
{
    return fp32 && !stratified && d >= 1 && K >= 1 && K <= UNION_SLOTS && K * (n + 1) <= UNION_MAXV;
}

size_t union_bytes(int d, int K, int n)
{
    const size_t m = (size_t)K * (n + 1);
    auto a256 = [](size_t v) { return (v + 255) & ~size_t(255); };
    return a256(d * m * 4) + a256(d * m * 4) + a256((size_t)d * 4) + a256((size_t)d * UNION_CELLS * 4) +
           a256(d * m * UNION_SLOTS * 4);
}

void bind_union(Params& P, unsigned char* base)
{
    const size_t m = (size_t)P.K * (P.n + 1);
    const int d = P.d;
    auto a256 = [](size_t v) { return (v + 255) & ~size_t(255); };
    P.uMax = (int)m;
    if (!base) {
        P.uImg = P.uU = P.uD = nullptr;
        P.uNU = nullptr;
        P.uC = nullptr;
        return;
    }
    unsigned char* q = base;
    P.uImg = reinterpret_cast<float*>(q); q += a256(d * m * 4);
    P.uU = reinterpret_cast<float*>(q); q += a256(d * m * 4);
    P.uNU = reinterpret_cast<int*>(q); q += a256((size_t)d * 4);
    P.uC = reinterpret_cast<uint32_t*>(q); q += a256((size_t)d * UNION_CELLS * 4);
    P.uD = reinterpret_cast<float*>(q);
}

cudaError_t launch_union_build(const Params& P, cudaStream_t s)
{
    const int d = P.d, m = P.K * (P.n + 1);
    const size_t sort_smem = (size_t)m * 8, rows_smem = (size_t)(m + P.K * P.n) * 4;
    cudaError_t e = ensure_smem((const void*)k_union_sort, sort_smem);
    if (e == cudaSuccess) e = ensure_smem((const void*)k_union_rows, rows_smem);
    if (e != cudaSuccess) return e;
    const int64_t tot = (int64_t)d * m;
    k_union_images<<<(unsigned)std::min<int64_t>((tot + 255) / 256, 4096), 256, 0, s>>>(P);
    k_union_sort<<<d, SORT_THREADS, sort_smem, s>>>(P);
    k_union_cells<<<dim3(UNION_CELLS / CELLS_PER_BLOCK, d), CELL_THREADS, 0, s>>>(P);
    k_union_rows<<<dim3((m + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK, d), ROWS_THREADS, rows_smem, s>>>(P);
    return cudaGetLastError();
}

size_t union_pass_smem(const Params& P, const PassVariant& v, int mode)
{
    const int DM = v.D > 0 ? v.D : (v.dhi > 0 ? v.dhi : DMAX);
    return (size_t)union_smem_layout(DM, P.d, P.n, mode).bytes;
}

void add_pass_variants_union(std::vector<PassVariant>& v)
{
    v.push_back(make_union_variant<14, 100, 2>());
    v.push_back(make_union_variant<0, 0, 2>());
}

}  // namespace vamp
