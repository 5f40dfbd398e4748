// vamp_kernels.cu -- the small kernels around the pass kernel (vamp_pass.cuh):
//
//   k_begin_pass      integer call allocation N_c, prefix P_c (§3.4); cells of a
//                     pseudo-stratified pass (§3.3); clears the accumulators
//   k_strat_q         Σ over a channel's cells of the squared cell sums (§3.3)
//   k_finish_pass     per-channel means/variances, pass result, combination
//   k_pass_result     pass result into a caller's device array (asynchronous pass)
//   k_refine          VEGAS rebinning of every (channel, axis) row (Eqs. 14, 15),
//                     with the channel equivalences pooled in (§3.5)
//   k_update_alpha    channel-weight update (Eq. 25)
//   k_derive          lookup-block rows: densities 1/(n Δx), cell tables, FP32 copies
//   k_gen_prepare / k_gen_scan / k_gen_copy   generation bookkeeping
//   k_eval<T>         per-call diagnostics for parity tests
//   k_batch_*         the same steps for every instance of a batch or server tick
#include "vamp_device.cuh"
#include "vamp_internal.h"

#include <algorithm>

namespace vamp {

// ---------------------------------------------------------------------------
// allocation (R6: N_c = max(N_min, floor(α_c N)) for α_c > 0)
// ---------------------------------------------------------------------------
// Pseudo-stratified sampling (§3.3): the largest m in [1, 2^20] with
// 2 m^d <= N (exact integer search).
__device__ int64_t strat_cells_per_axis(int64_t N, int d)
{
    int64_t lo = 1, hi = 1 << 20;
    while (lo < hi) {
        const int64_t mid = (lo + hi + 1) / 2;
        int64_t prod = 2;
        for (int k = 0; k < d && prod <= N; ++k) {
            if (prod > N / mid) { prod = N + 1; break; }
            prod *= mid;
        }
        if (prod <= N) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Inclusive scan of v over the block (all threads; at most 1024), and the sum
// over the block through `total`.  tmp: 33 words of shared memory.
template <typename V>
__device__ __forceinline__ V block_scan(V v, V* tmp, V* total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const V y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    __syncthreads();  // tmp is free again
    if (lane == 31) tmp[wid] = v;
    __syncthreads();
    if (wid == 0) {
        V w = lane < nw ? tmp[lane] : V(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const V y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) tmp[lane] = w;
        if (lane == nw - 1) tmp[32] = w;
    }
    __syncthreads();
    *total = tmp[32];
    return v + (wid > 0 ? tmp[wid - 1] : V(0));
}

// Sum over the block in a fixed order, to every thread.
__device__ __forceinline__ double block_sum(double v, double* tmp)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) tmp[wid] = v;
    __syncthreads();
    double s = 0.0;
    for (int q = 0; q < nw; ++q) s += tmp[q];
    return s;
}

// Two sums at once.
__device__ __forceinline__ void block_sum2(double& u, double& v, double (*tmp)[2])
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        u += __shfl_xor_sync(0xffffffffu, u, o);
        v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    if (lane == 0) { tmp[wid][0] = u; tmp[wid][1] = v; }
    __syncthreads();
    u = v = 0.0;
    for (int q = 0; q < nw; ++q) { u += tmp[q][0]; v += tmp[q][1]; }
}

__device__ __forceinline__ double lanes_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Called by every thread of one block (a multiple of 32 threads), a channel a
// thread: with one thread walking the channels the allocation of K = 64 took
// 12 us, the pass results 35 and the weights 19.
__device__ void begin_pass_dev(const Params& P, int64_t N)
{
    __shared__ long long tmp[33];
    long long acc = 0, cells = 0;
    for (int c0 = 0; c0 < P.K; c0 += blockDim.x) {
        const int c = c0 + (int)threadIdx.x;
        long long nc = 0, m = 1, s = 0, C = 1;
        if (c < P.K) {
            if (P.alpha[c] > 0.0) {
                nc = (long long)floor(P.alpha[c] * (double)N);
                if (nc < P.n_min) nc = P.n_min;
            }
            if (P.stratified) {
                // whole cells: n_r per axis, C = n_r^d cells, s = floor(N_c / C)
                s = nc;
                if (nc >= 2) {
                    m = strat_cells_per_axis(nc, P.d);
                    for (int k = 0; k < P.d; ++k) C *= m;
                    s = nc / C;
                }
                nc = s * C;
                P.nr[c] = m;
                P.spc[c] = s;
            }
            P.Nc[c] = nc;
        }
        long long tot;
        const long long incl = block_scan(c < P.K ? nc : 0ll, tmp, &tot);
        if (c < P.K) P.Pc[c + 1] = acc + incl;
        acc += tot;
        if (P.stratified) {
            const long long ci = block_scan(c < P.K ? C : 0ll, tmp, &tot);
            if (c < P.K) P.coff[c + 1] = cells + ci;
            cells += tot;
        }
    }
    if (threadIdx.x == 0) {
        P.Pc[0] = 0;
        if (P.stratified) P.coff[0] = 0;
        P.sc->n_total = acc;
        P.sc->wmax_bits = 0ull;
    }
}

// Stratified passes: Q_c = Σ over the channel's cells of the squared cell
// sums (Qc is zero before), `parts` blocks of 256 threads per channel: one
// block alone took 211 us for the 5e5 cells of a 1e6-call channel.
constexpr int STRAT_PARTS = 32;

__device__ void strat_q_channel(const Params& P, int c, int part, int parts)
{
    __shared__ double tmp[33];
    const int64_t a = P.coff[c], len = P.coff[c + 1] - a;
    const int64_t lo = a + len * part / parts, hi = a + len * (part + 1) / parts;
    double s = 0.0;
    for (int64_t q = lo + threadIdx.x; q < hi; q += blockDim.x) {
        const double v = P.cellsum[q];
        s += v * v;
    }
    s = block_sum(s, tmp);
    if (threadIdx.x == 0 && hi > lo) atomicAdd(&P.Qc[c], s);
}

__global__ void k_strat_q(Params P)
{
    strat_q_channel(P, blockIdx.x, blockIdx.y, gridDim.y);
}

// Block 0 allocates; with clear != 0 all blocks clear the pass accumulators
// (and `cells` cell sums).
__global__ void k_begin_pass(Params P, int64_t N, int clear, int64_t cells)
{
    if (clear) {
        const int64_t nd = (int64_t)P.K * P.d * P.n, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x,
                      nt = (int64_t)gridDim.x * blockDim.x;
        for (int64_t q = t0; q < nd; q += nt) P.D[q] = 0.0;
        for (int64_t q = t0; q < 2 * P.K; q += nt) P.csum[q] = 0.0;
        if (P.stratified) {
            for (int64_t q = t0; q < cells; q += nt) P.cellsum[q] = 0.0;
            for (int64_t q = t0; q < P.K; q += nt) P.Qc[q] = 0.0;
        }
    }
    if (blockIdx.x == 0) begin_pass_dev(P, N);
}

// ---------------------------------------------------------------------------
// pass result (Eqs. 10, 11 per channel on shifted sums; Eq. 23; R8, R9)
// ---------------------------------------------------------------------------
// Called by every thread of one block: per-channel values and their sums by
// all, the combination of the passes by the first warp.
__device__ void finish_pass_dev(const Params& P, int combine)
{
    __shared__ double tmp[32][2];
    Scalars* sc = P.sc;
    double I = 0.0, V = 0.0;
    // this lane's share of the history of passes, fetched while the channels' sums are on their way
    const int h = sc->n_hist;
    const unsigned long long wbits = sc->wmax_bits;
    double cnt = 0.0, nzero = 0.0, zI = 0.0, sw = 0.0, swi = 0.0;
    auto take = [&](double hI, double hV) {
        cnt += 1.0;
        if (hV <= 0.0) { nzero += 1.0; zI += hI; }
        else { const double iv = 1.0 / hV; sw += iv; swi += hI * iv; }
    };
    if (threadIdx.x < 32)
        for (int q = threadIdx.x; q < h; q += 32)
            if (sc->hist_comb[q]) take(sc->hist_I[q], sc->hist_V[q]);
    for (int c = threadIdx.x; c < P.K; c += blockDim.x) {
        const int64_t nci = P.Nc[c];
        if (nci == 0) { P.Ic[c] = P.Vc[c] = P.Wc[c] = 0.0; P.shift[c] = 0.0; continue; }
        const double Nc = (double)nci, al = P.alpha[c];
        const double m1 = P.csum[2 * c] / Nc, m2 = P.csum[2 * c + 1] / Nc;
        const double Ic = P.shift[c] + m1;
        double Vv = 0.0;
        if (!P.stratified) {
            if (nci > 1) Vv = (m2 - m1 * m1) * Nc / (Nc - 1.0);
        } else if (P.spc[c] >= 2) {
            // mean over the channel's cells of the cells' sample variances
            const double s = (double)P.spc[c], C = (double)(P.coff[c + 1] - P.coff[c]);
            Vv = (P.csum[2 * c + 1] - P.Qc[c] / s) / (C * (s - 1.0));
        }
        if (Vv < 0.0) Vv = 0.0;
        P.Ic[c] = Ic;
        P.Vc[c] = Vv;
        P.Wc[c] = (m2 - m1 * m1) + Ic * Ic;
        P.shift[c] = Ic;  // R13: the next pass's sums are taken about this mean
        I += al * Ic;
        V += al * al * Vv / Nc;
    }
    block_sum2(I, V, tmp);
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    if (lane == 0 && h < 1024) {
        sc->hist_I[h] = I;
        sc->hist_V[h] = V;
        sc->hist_comb[h] = combine;
        sc->n_hist = h + 1;
        if (combine) take(I, V);
    }
    // inverse-variance combination of the flagged passes
    cnt = lanes_sum(cnt);
    double cI = 0.0, cS = 0.0, chi = 0.0;
    if (cnt > 0.0) {
        nzero = lanes_sum(nzero);
        if (nzero > 0.0) {
            cI = lanes_sum(zI) / nzero;
        } else {
            sw = lanes_sum(sw);
            cI = lanes_sum(swi) / sw;
            cS = sqrt(1.0 / sw);
            if (cnt > 1.0) {
                double ch = 0.0;
                for (int q = lane; q < h; q += 32) {
                    if (!sc->hist_comb[q]) continue;
                    const double dI = sc->hist_I[q] - cI;
                    ch += dI * dI / sc->hist_V[q];
                }
                if (lane == 0 && h < 1024 && combine) ch += (I - cI) * (I - cI) / V;
                chi = lanes_sum(ch) / (cnt - 1.0);
            }
        }
    }
    if (lane != 0) return;
    const double wmax = __longlong_as_double((long long)wbits);
    sc->wmax_gen = wmax;
    sc->res[0] = I;
    sc->res[1] = V;
    sc->res[2] = wmax;
    sc->res[3] = wmax > 0.0 ? I / wmax : 0.0;
    sc->res[4] = 0.0; // n_calls is taken from n_total on the host
    sc->res[5] = cI;
    sc->res[6] = cS;
    sc->res[7] = chi;
}

__global__ void k_finish_pass(Params P, int combine)
{
    finish_pass_dev(P, combine);
}

// Result of the last pass into a caller's device array (asynchronous form):
// integral, variance, w_max, efficiency, N', combined, its σ, χ²/dof, flags.
__global__ void k_pass_result(Params P, double* out)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const Scalars* sc = P.sc;
    for (int q = 0; q < 8; ++q) out[q] = sc->res[q];
    out[4] = (double)sc->n_total;
    out[8] = (double)sc->err;
}

// ---------------------------------------------------------------------------
// lookup blocks of one grid row (Eq. 12 densities, FP32 copies, cell tables)
// ---------------------------------------------------------------------------
// One warp derives grid row `row` from its edges e64 (global or shared memory).
// q0: n+1 ints of warp scratch.
template <typename T>
__device__ __forceinline__ void derive_row_t(const Params& P, const BlkLayout& L, unsigned char* lk, int row,
                                             int lane, const double* e64, int* q0)
{
    const int n = P.n, d = P.d;
    const int c = row / d, k = row % d;
    unsigned char* r = lk + (size_t)c * L.bytes + L.H + (size_t)k * L.R;
    T* e = reinterpret_cast<T*>(r);
    T* dnr = reinterpret_cast<T*>(r + L.Es * sizeof(T));
    unsigned char* tb = r + (L.Es + L.Dn) * sizeof(T);
    // FP64 rows of mapped coordinates hold the images φ_c(ξ_j) of the edges
    // (clamped at 0, the forward map's formula): a bin of x = φ_c^{-1}(p) is
    // the bin whose image holds p, so the FP64 lookups compare p itself; the
    // forward map reads the edges from the master grid
    const ChanHdr<T>& h = *reinterpret_cast<const ChanHdr<T>*>(lk + (size_t)c * L.bytes);
    int slot = -1;
    if constexpr (sizeof(T) == 8) slot = map_slot(h, k);
    const bool over_x = slot >= 0;
    const int Lc = 1 << L.lshift;
    for (int j = lane; j <= n; j += 32) {
        const double x = e64[j];
        double v = x;
        if constexpr (sizeof(T) == 8)
            if (over_x) v = edge_image(h, slot, x);
        const T ev = (T)(v > 0.0 ? v : 0.0);
        e[j] = ev;
        // first cell boundary q/L at or above the edge (over x in the FP64 rows
        // of mapped coordinates; scaling by L is exact)
        const double tq = ceil((over_x ? x : (double)ev) * (double)Lc);
        q0[j] = tq > (double)(Lc + 1) ? Lc + 1 : (int)tq;
        const int jb = j < n ? j : n - 1;  // entry n repeats bin n-1
        const double dx = (double)n * (e64[jb + 1] - e64[jb]);
        if constexpr (sizeof(T) == 8) {
            // 1 / (n Δx), rounded to 53 bits (a subnormal Δx as the division has it)
            reinterpret_cast<uint64_t*>(dnr)[j] =
                dx >= 2.3e-308 ? sf_pack(sf_norm(sf_rcp(sf_from_double(dx)))) : sf_pack_double(1.0 / dx);
        } else {
            dnr[j] = (T)(1.0 / dx);
        }
    }
    __syncwarp();
    // tb[q] = largest j in [0, n-1] with edge j <= q/L, for q = 0..L: bin j
    // takes the boundaries from its own edge's up to the next edge's; span =
    // the most edges (of 1..n-1) inside one cell
    int span = 0;
    for (int j = lane; j < n; j += 32) {
        const int a = j == 0 ? 0 : q0[j], b = j == n - 1 ? Lc + 1 : min(q0[j + 1], Lc + 1);
        for (int q = a; q < b; ++q) tb[q] = (unsigned char)j;
        if (j > 0 && a >= 1 && a <= Lc) {
            int run = 1;
            while (j + run <= n - 1 && q0[j + run] == a) ++run;
            span = max(span, run);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) span = max(span, __shfl_xor_sync(0xffffffffu, span, o));
    if (lane == 0) {
        tb[Lc + 1] = (unsigned char)min(span, 255);
        // this row's bit of the channel's slow-row mask (each row owns its bit)
        unsigned int* slow = reinterpret_cast<unsigned int*>(lk + (size_t)c * L.bytes + offsetof(ChanHdr<T>, slow));
        if (span > 1 && !over_x) atomicOr(slow, 1u << k);
        else atomicAnd(slow, ~(1u << k));
    }
    __syncwarp();
}

// A context's passes read the blocks of its own precision only.
__device__ __forceinline__ void derive_row(const Params& P, int row, int lane, const double* e64, int* q0)
{
    if (P.fp32) derive_row_t<float>(P, P.lay32, P.lk32, row, lane, e64, q0);
    else derive_row_t<double>(P, P.lay64, P.lk64, row, lane, e64, q0);
}

// The forms of α_c that the pass kernels read beside alpha[c].
__device__ __forceinline__ void store_alpha(const Params& P, int c, double a)
{
    P.alpha32[c] = (float)a;
    P.alphaN[c] = a * reinterpret_cast<const ChanHdr<double>*>(P.lk64 + (size_t)c * P.lay64.bytes)->gN;
}

__global__ void k_derive(Params P, double w_max, int n_hist)
{
    extern __shared__ int dq0[];
    const int rows = P.K * P.d;
    const int lane = threadIdx.x & 31;
    int* q0 = dq0 + (threadIdx.x >> 5) * (P.n + 1);
    const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int nw = gridDim.x * (blockDim.x >> 5);
    for (int row = w; row < rows; row += nw) derive_row(P, row, lane, P.edges64 + (size_t)row * (P.n + 1), q0);
    if (blockIdx.x == 0) {
        for (int c = threadIdx.x; c < P.K; c += blockDim.x) store_alpha(P, c, P.alpha[c]);
        if (threadIdx.x == 0 && w_max >= 0.0) P.sc->wmax_gen = w_max;
        if (threadIdx.x == 0 && n_hist >= 0) P.sc->n_hist = n_hist;
    }
}

// ---------------------------------------------------------------------------
// rebinning, one warp per (channel, axis) row (Eqs. 14, 15; R2-R4)
// ---------------------------------------------------------------------------
// ((r - 1) / ln r)^a for r in (0, 1): logarithms and powers on 64-bit mantissas
// (an FP64 log and pow are some 150 operations of the FP64 pipe a bin, half of
// the rebinning of the collider's 896 rows).  Nothing is rounded to a double
// before the result, whose error is that rounding's and 2^-58 (grid_alpha 1.5).
// Above 1/2, which one bin of a row can be, and below a normal number the FP64
// log.
__device__ __forceinline__ double rebin_measure(double r, double a)
{
    Sf num, den;
    if (r <= 0.5 && r >= 2.3e-308) {
        bool neg;
        const Sf x = sf_from_double(r);
        den = sf_mul(sf_log2(x, neg), Sf{0xb17217f7d1cf79acull, -64});  // -ln r
        num = Sf{0ull - (x.e > -128 ? x.m >> (-64 - x.e) : 1ull), -64};  // 1 - r
    } else {
        den = sf_from_double(-log(r));
        num = sf_from_double(1.0 - r);
    }
    return sf_to_double(sf_pow(sf_norm(sf_mul(num, sf_rcp(sf_norm(den)))), a));
}

// Doubles of warp scratch of refine_row_dev.
__host__ __device__ constexpr int refine_scratch(int n) { return 5 * n + 4; }

// One warp rebins grid row `row` of P; ws = refine_scratch(n) doubles.
__device__ void refine_row_dev(const Params& P, int row, int lane, double* ws)
{
    const int n = P.n;
    double* Dj = ws;
    double* m = Dj + n;
    double* C = m + n;          // n+1
    double* eo = C + n + 1;     // n+1
    double* en = eo + n + 1;    // n+1
    const double* Din = P.D + (size_t)row * n;
    double* e = P.edges64 + (size_t)row * (n + 1);
    for (int j = lane; j < n; j += 32) Dj[j] = Din[j];
    if (P.eq_off) {
        // channel equivalences (§3.5): the pass's d-values of the equivalent
        // rows, added in list order (identity j, invert n-1-j, symmetric the
        // mean of both); an invariant axis takes unit weights
        const int q0 = P.eq_off[row], q1 = P.eq_off[row + 1];
        bool invariant = false;
        for (int q = q0; q < q1; ++q) {
            const int ent = P.eq_ent[q], kind = ent & 3;
            const double* src = P.D + (size_t)(ent >> 2) * n;
            if (kind == VAMP_EQ_INVARIANT) { invariant = true; continue; }
            for (int j = lane; j < n; j += 32) {
                double t;
                if (kind == VAMP_EQ_IDENTITY) t = src[j];
                else if (kind == VAMP_EQ_INVERT) t = src[n - 1 - j];
                else t = __dmul_rn(0.5, __dadd_rn(src[j], src[n - 1 - j]));
                Dj[j] = __dadd_rn(Dj[j], t);
            }
        }
        if (invariant)
            for (int j = lane; j < n; j += 32) Dj[j] = 1.0;
    }
    for (int j = lane; j <= n; j += 32) eo[j] = e[j];
    __syncwarp();
    if (P.smooth && n >= 2) {
        for (int j = lane; j < n; j += 32) {
            double t;
            if (j == 0) t = (Dj[0] + Dj[1]) / 2.0;
            else if (j == n - 1) t = (Dj[n - 2] + Dj[n - 1]) / 2.0;
            else t = (Dj[j - 1] + Dj[j] + Dj[j + 1]) / 3.0;
            m[j] = t;
        }
        __syncwarp();
        for (int j = lane; j < n; j += 32) Dj[j] = m[j];
        __syncwarp();
    }
    double S = 0.0;
    for (int j = lane; j < n; j += 32) {
        const double w = sqrt(Dj[j]);  // ω_j
        Dj[j] = w;
        S += w;
    }
    S = lanes_sum(S);
    // axis kept (R2), lookup blocks unchanged; likewise where a d-value is
    // infinite (a weight above 1.3e154 is finite, its square is not), which
    // leaves no ratio between the bins
    if (!(S > 0.0 && S < INFINITY)) return;
    for (int j = lane; j < n; j += 32) {
        const double r = Dj[j] / S;
        double mj;
        if (r == 0.0) mj = 0.0;
        else if (fabs(r - 1.0) < 1e-12) mj = 1.0;
        else mj = rebin_measure(r, P.grid_alpha);
        m[j] = mj;
    }
    __syncwarp();
    // The cumulative of m in bin order, by one lane: C never falls, and stays
    // the same to the last bit over bins with m = 0, so that the search below
    // ends in a bin with m > 0.  (A scan by the lanes adds in another order for
    // each j; its C moves by an ulp over empty bins, and 1 to 10 % of
    // mirror-symmetric rows with empty bins then divided by their m = 0.)
    if (lane == 0) {
        double acc = 0.0;
        C[0] = 0.0;
#pragma unroll 8
        for (int j = 0; j < n; ++j) {
            acc += m[j];
            C[j + 1] = acc;
        }
    }
    __syncwarp();
    const double M = C[n];
    if (!(M > 0.0)) return;
    for (int i = lane; i <= n; i += 32) {
        double ne;
        if (i == 0) ne = 0.0;
        else if (i == n) ne = 1.0;
        else {
            const double t = (double)i * M / (double)n;
            int lo = 1, hi = n; // smallest j in [1, n] with C[j] >= t
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (C[mid] >= t) hi = mid; else lo = mid + 1;
            }
            const int j = lo;
            const double fr = (t - C[j - 1]) / m[j - 1];
            ne = __dadd_rn(eo[j - 1], __dmul_rn(fr, __dsub_rn(eo[j], eo[j - 1])));
        }
        e[i] = ne;
        en[i] = ne;
    }
    __syncwarp();
    derive_row(P, row, lane, en, reinterpret_cast<int*>(Dj));  // n + 1 ints over Dj and m
}

__global__ void __launch_bounds__(REFINE_WARPS * 32) k_refine(Params P)
{
    extern __shared__ double rs[];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int row = blockIdx.x * REFINE_WARPS + wid;
    if (row >= P.K * P.d) return;
    refine_row_dev(P, row, lane, rs + (size_t)wid * refine_scratch(P.n));
}

// ---------------------------------------------------------------------------
// channel weights (Eq. 25 with R5)
// ---------------------------------------------------------------------------
// ω^β on 64-bit mantissas (about 2^-57 and the rounding, as long as the power
// lies within 2^±128); by pow beyond, and where ω or β is not a normal number.
__device__ __forceinline__ double omega_power(double w, double beta)
{
    if (w >= 2.3e-308 && w < INFINITY && fabs(beta) >= 2.3e-308) {
        const Sf u = sf_pow(sf_from_double(w), beta);
        if (u.e + 63 >= -128 && u.e + 63 < 128) return sf_to_double(u);
    }
    return pow(w, beta);
}

// Called by every thread of one block, a channel a thread (Acum holds the
// terms α_c ω_c^β and then the new weights between the sums).
__device__ void update_alpha_dev(const Params& P)
{
    __shared__ double tmp[33], tmp2[32][2];
    const int K = P.K;
    auto omega = [&](int c) { return P.omega_mode ? P.Wc[c] : P.Vc[c]; };
    double SU = 0.0, MU = 0.0;
    for (int c = threadIdx.x; c < K; c += blockDim.x) {
        const double a = P.alpha[c], w = omega(c);
        double u = 0.0;
        if (a > 0.0 && P.Nc[c] > 0 && w > 0.0) {
            u = a * omega_power(w, P.beta);
            SU += u;
            MU += a;
        }
        P.Acum[c] = u;
    }
    block_sum2(SU, MU, tmp2);
    double tot = 0.0;
    for (int c = threadIdx.x; c < K; c += blockDim.x) {
        double a = P.alpha[c];
        if (a > 0.0 && P.Nc[c] > 0) {
            if (omega(c) > 0.0) a = P.Acum[c] / SU * MU;
            else if (P.Ic[c] == 0.0) a = 0.0;  // every call of the channel gave w = 0
        }
        P.Acum[c] = a;  // new weights, normalised below
        tot += a;
    }
    tot = block_sum(tot, tmp);
    for (int c = threadIdx.x; c < K; c += blockDim.x) {
        if (tot > 0.0) P.alpha[c] = P.Acum[c] / tot;
        store_alpha(P, c, P.alpha[c]);
    }
}

__global__ void k_update_alpha(Params P)
{
    update_alpha_dev(P);
}

// ---------------------------------------------------------------------------
// generation bookkeeping
// ---------------------------------------------------------------------------
constexpr int SMALL_BLOCK = 256;  // most threads of the one-block kernels

// Cumulative α in channel order, by one thread: A_c never falls and stays the
// same where α_c = 0, so that no call draws a channel that is switched off (in
// the sums of a scan by lanes such a channel's A_c could lie an ulp higher).
// Once per generation: K additions from shared memory.
__global__ void k_gen_prepare(Params P)
{
    __shared__ double a[SMALL_BLOCK], sum[SMALL_BLOCK];
    const int nt = blockDim.x;
    double acc = 0.0;
    for (int c0 = 0; c0 < P.K; c0 += nt) {
        const int c = c0 + (int)threadIdx.x, m = min(nt, P.K - c0);
        if (c < P.K) a[threadIdx.x] = P.alpha[c];
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll 8
            for (int q = 0; q < m; ++q) {
                acc += a[q];
                sum[q] = acc;
            }
        }
        __syncthreads();
        if (c < P.K) P.Acum[c] = sum[threadIdx.x];
        __syncthreads();
    }
    if (threadIdx.x == 0) P.sc->gen_bmax_bits = 0ull;
}

// Exclusive prefix of the per-chunk counts, how many to take, calls used; the
// batch's maximum weight into w_max for the next batch (wmax_cut keeps the
// bound that this batch was accepted against).
__global__ void k_gen_scan(Params P, PassArgs G, int64_t remaining)
{
    __shared__ long long tmp[33];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int nb = (int)G.nchunks;
    const int per = (nb + nt - 1) / nt;
    const int b0 = min(nb, tid * per), b1 = min(nb, b0 + per);
    long long s = 0;
    for (int b = b0; b < b1; ++b) s += G.counts[b];
    long long total;
    long long off = block_scan(s, tmp, &total) - s;
    const long long take = total < remaining ? total : remaining;
    if (tid == 0) {
        Scalars* sc = P.sc;
        sc->gen_total = total;
        sc->gen_take = take;
        sc->gen_over = 0;
        if (!(take == remaining && take > 0)) sc->gen_used = G.batch;
        const double bm = __longlong_as_double((long long)sc->gen_bmax_bits), cut = sc->wmax_gen;
        sc->wmax_cut = cut;
        if (bm > cut) sc->wmax_gen = bm;
        sc->gen_bmax_bits = 0ull;
    }
    for (int b = b0; b < b1; ++b) {
        const long long cnt = G.counts[b];
        G.offsets[b] = off;
        // the chunk holding the last taken record decides the calls used
        if (take == remaining && take > 0 && off < take && take <= off + cnt) {
            const long long r = take - 1 - off;
            P.sc->gen_used = (long long)G.callidx[(int64_t)b * G.chunk + r] + 1;
        }
        off += cnt;
    }
}

__global__ void k_gen_copy(Params P, PassArgs G, unsigned char* out)
{
    const int b = blockIdx.x;
    const long long off = G.offsets[b], cnt = G.counts[b], take = P.sc->gen_take;
    if (off >= take) return;
    const long long ncopy = min(cnt, take - off);
    const int words = G.rec_bytes / 8;
    const unsigned long long* src =
        reinterpret_cast<const unsigned long long*>(G.staging + (int64_t)b * G.chunk * G.rec_bytes);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(out + off * G.rec_bytes);
    const double wmax = P.sc->wmax_cut;
    int over = 0;
    for (long long q = threadIdx.x; q < ncopy * words; q += blockDim.x) dst[q] = src[q];
    for (long long r = threadIdx.x; r < ncopy; r += blockDim.x) {
        const double w = *reinterpret_cast<const double*>(G.staging + ((int64_t)b * G.chunk + r) * G.rec_bytes +
                                                          (G.rec_bytes - 8));
        over += (fabs(w) > wmax);
    }
    if (over) atomicAdd(reinterpret_cast<unsigned long long*>(&P.sc->gen_over), (unsigned long long)over);
}

// ---------------------------------------------------------------------------
// diagnostics: one call per thread, lookup blocks read from global memory
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_eval(Params P, EvalArgs A)
{
    using SH = Shape<T, 0, 0>;
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= A.count) return;
    const SH sh(Prec<T>::lay(P), P.d, P.n);
    const int d = P.d;
    const uint32_t call = A.call0 + (uint32_t)q;
    uint32_t X[DMAX + 4];
    int c;
    if (A.mode == 0) {
        call_words<DMAX + 4>(P, call, A.field, d, X);
        c = find_channel(P.Pc, P.K, (int64_t)call);
    } else {
        call_words<DMAX + 4>(P, call, A.field, d + 2, X);
        uint32_t xc = 0u;
        for (int k = 0; k < DMAX + 4; ++k)
            if (k == d) xc = X[k];
        c = choose_channel(P, unif64(xc));
    }
    T p1[1][DMAX], x[DMAX], g[1], f[1], Aq[1];
    int jf[DMAX];
    uint32_t dig[DMAX], nr = 1u;
    const bool strat = A.mode == 0 && P.stratified;
    if (strat) {
        nr = (uint32_t)P.nr[c];
        uint32_t cell = (uint32_t)(((int64_t)call - P.Pc[c]) / P.spc[c]);
        for (int k = 0; k < DMAX; ++k) {
            dig[k] = cell % nr;
            cell /= nr;
        }
    }
    SoftCall<DMAX> soft;
    if constexpr (sizeof(T) == 8) {
        double own;
        soft_forward(P, sh, c, X, p1[0], jf, own, soft, strat ? dig : nullptr, nr, x);
        Aq[0] = soft.A;
        g[0] = P.alphaN[c] * own;
    } else {
        T owngJ;
        forward_call<T>(P, sh, c, X, x, p1[0], jf, owngJ, Aq[0], strat ? dig : nullptr, nr);
        g[0] = Prec<T>::alpha(P, c) * owngJ;
    }
    f[0] = P.matching ? T(0) : integrand_peaks<T, DMAX>(P, d, p1[0], Aq[0]);
    int* bins = A.bins + (size_t)q * P.K * d;
    for (int c2 = 0; c2 < P.K; ++c2) {
        const T a = Prec<T>::alpha(P, c2);
        const bool lookups = a != T(0) && c2 != c;
        const unsigned char* blk = Prec<T>::lk(P) + (size_t)c2 * sh.bytes();
        if constexpr (sizeof(T) == 8) {
            double gt, ft;
            soft_channel<true>(P, sh, blk, lookups, p1[0], soft, gt, ft, bins + c2 * d);
            if (lookups) g[0] += P.alphaN[c2] * gt;
            if (P.matching) f[0] += reinterpret_cast<const ChanHdr<double>*>(blk)->fN * ft;
        } else {
            const bool skip[1] = {false};
            channel_body<T, 1, true>(P, sh, blk, a, lookups, P.matching != 0, p1, Aq, skip, g, f, bins + c2 * d);
        }
        if (a == T(0))
            for (int k = 0; k < d; ++k) bins[c2 * d + k] = -1;
        else if (c2 == c)
            for (int k = 0; k < d; ++k) bins[c2 * d + k] = jf[k];
    }
    const T w = g[0] > T(0) ? f[0] / g[0] : T(0);
    for (int k = 0; k < d; ++k) {
        A.x[(size_t)q * d + k] = (double)x[k];
        A.p[(size_t)q * d + k] = (double)p1[0][k];
        A.jf[(size_t)q * d + k] = jf[k];
    }
    A.fgwc[4 * q + 0] = (double)f[0];
    A.fgwc[4 * q + 1] = (double)g[0];
    A.fgwc[4 * q + 2] = (double)w;
    A.fgwc[4 * q + 3] = (double)c;
}

// ---------------------------------------------------------------------------
// many instances: the small steps of one iteration, one block (or warp) per
// instance (or grid row)
// ---------------------------------------------------------------------------
__global__ void k_batch_begin(MultiArgs M)
{
    const int i = blockIdx.x;
    if (i >= M.n_inst) return;
    const Params& P = M.inst[i];
    begin_pass_dev(P, M.ncalls[i]);
    const size_t nd = (size_t)P.K * P.d * P.n;
    for (size_t q = threadIdx.x; q < nd; q += blockDim.x) P.D[q] = 0.0;
    for (int q = threadIdx.x; q < 2 * P.K; q += blockDim.x) P.csum[q] = 0.0;
    if (P.stratified) {
        // the cells of this pass (first cell of each channel set above)
        __syncthreads();
        const int64_t ncell = P.coff[P.K];
        for (int64_t q = threadIdx.x; q < ncell; q += blockDim.x) P.cellsum[q] = 0.0;
        for (int q = threadIdx.x; q < P.K; q += blockDim.x) P.Qc[q] = 0.0;
    }
}

// Stratified instances: Q_c per (instance, channel) pair, STRAT_PARTS blocks each.
__global__ void k_batch_strat_q(MultiArgs M)
{
    const int pair = blockIdx.x;
    int lo = 0, hi = M.n_inst - 1;  // instance of the pair
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (M.pair_off[mid] <= pair) lo = mid; else hi = mid - 1;
    }
    const Params& P = M.inst[lo];
    if (!P.stratified) return;
    strat_q_channel(P, pair - M.pair_off[lo], blockIdx.y, gridDim.y);
}

// Work items: every (instance, channel) pair with N_c calls gives
// ceil(N_c / item_calls) items; exclusive prefix over the pairs.
__global__ void k_batch_items(MultiArgs M)
{
    __shared__ long long tmp[33];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int per = (M.npairs + nt - 1) / nt;
    const int p0 = min(M.npairs, tid * per), p1 = min(M.npairs, p0 + per);
    auto items_of = [&](int pr) -> long long {
        int lo = 0, hi = M.n_inst - 1; // instance with pair_off[i] <= pr
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (M.pair_off[mid] <= pr) lo = mid; else hi = mid - 1;
        }
        const long long nc = M.inst[lo].Nc[pr - M.pair_off[lo]];
        return (nc + M.item_calls - 1) / M.item_calls;
    };
    long long s = 0;
    for (int pr = p0; pr < p1; ++pr) s += items_of(pr);
    long long total;
    long long off = block_scan(s, tmp, &total) - s;
    if (tid == 0) {
        M.ctl->total = total;
        M.ctl->next = 0;
        M.pair_prefix[M.npairs] = total;
    }
    for (int pr = p0; pr < p1; ++pr) {
        M.pair_prefix[pr] = off;
        off += items_of(pr);
    }
}

// one block per instance
__global__ void k_batch_finish(MultiArgs M)
{
    const int i = blockIdx.x;
    if (i >= M.n_inst) return;
    const Params& P = M.inst[i];
    finish_pass_dev(P, (int)M.iter[i] >= M.combine_from[i] ? 1 : 0);
    if (threadIdx.x != 0) return;
    double* r = M.results + (size_t)i * 9;
    for (int q = 0; q < 8; ++q) r[q] = P.sc->res[q];
    r[4] = (double)P.sc->n_total;
    r[8] = (double)P.sc->err;
}

__global__ void __launch_bounds__(REFINE_WARPS * 32) k_batch_refine(MultiArgs M)
{
    extern __shared__ double rs[];
    if (!(M.it->adapt & 1)) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int row = blockIdx.x * REFINE_WARPS + wid;
    if (row >= M.nrows) return;
    int lo = 0, hi = M.n_inst - 1; // instance with row_off[i] <= row
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (M.row_off[mid] <= row) lo = mid; else hi = mid - 1;
    }
    refine_row_dev(M.inst[lo], row - M.row_off[lo], lane, rs + (size_t)wid * refine_scratch(M.max_n));
}

// one block per instance
__global__ void k_batch_alpha(MultiArgs M)
{
    if (!(M.it->adapt & 2)) return;
    const int i = blockIdx.x;
    if (i < M.n_inst) update_alpha_dev(M.inst[i]);
}

cudaError_t launch_batch_begin(const MultiArgs& M, cudaStream_t s)
{
    k_batch_begin<<<M.n_inst, 256, 0, s>>>(M);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_batch_items<<<1, 1024, 0, s>>>(M);
    return cudaGetLastError();
}

cudaError_t launch_batch_after(const MultiArgs& M, cudaStream_t s)
{
    cudaError_t e;
    if (M.any_strat) {
        k_batch_strat_q<<<dim3(M.npairs, STRAT_PARTS), 256, 0, s>>>(M);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    k_batch_finish<<<M.n_inst, 64, 0, s>>>(M);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int blocks = (M.nrows + REFINE_WARPS - 1) / REFINE_WARPS;
    k_batch_refine<<<blocks, REFINE_WARPS * 32, (size_t)REFINE_WARPS * refine_scratch(M.max_n) * sizeof(double), s>>>(M);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_batch_alpha<<<M.n_inst, 64, 0, s>>>(M);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// self-test of the bounded wait: one CTA arms an mbarrier for a copy that is
// never issued, waits with the pass kernels' wait routine and a short limit,
// and records that it gave up (flag bit 0) and the cycles it waited
// ---------------------------------------------------------------------------
__global__ void k_wait_selftest(long long limit, unsigned int* flag, long long* cycles)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    const long long t0 = clock64();
    const bool ok = mbar_wait_bounded(&bar, 0u, limit);  // nothing completes phase 0
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!ok) atomicOr(flag, ERR_TIMEOUT);
        *cycles = clock64() - t0;
    }
}

cudaError_t launch_wait_selftest(long long limit, unsigned int* flag, long long* cycles, cudaStream_t s)
{
    k_wait_selftest<<<1, 64, 0, s>>>(limit, flag, cycles);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------
// Threads of the one-block kernels: a channel a thread up to 256.
static int small_block(int K) { return std::min(SMALL_BLOCK, (K + 31) / 32 * 32); }

cudaError_t launch_begin_pass(const Params& P, int64_t N, cudaStream_t s, int clear, int64_t cells)
{
    // a block for every 4096 words to clear, up to two per SM
    const int64_t words = clear ? (int64_t)P.K * P.d * P.n + (P.stratified ? cells : 0) : 0;
    const int blocks = (int)std::min<int64_t>(304, std::max<int64_t>(1, words / 4096));
    k_begin_pass<<<blocks, 256, 0, s>>>(P, N, clear, cells);
    return cudaGetLastError();
}

cudaError_t launch_strat_q(const Params& P, cudaStream_t s)
{
    k_strat_q<<<dim3(P.K, STRAT_PARTS), 256, 0, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_finish_pass(const Params& P, int combine, cudaStream_t s)
{
    k_finish_pass<<<1, small_block(P.K), 0, s>>>(P, combine);
    return cudaGetLastError();
}

cudaError_t launch_derive(const Params& P, cudaStream_t s, double w_max, int n_hist)
{
    const int rows = P.K * P.d;
    const int blocks = min((rows + 3) / 4, 1024);
    k_derive<<<blocks, 128, (size_t)4 * (P.n + 1) * sizeof(int), s>>>(P, w_max, n_hist);
    return cudaGetLastError();
}

cudaError_t launch_refine(const Params& P, cudaStream_t s)
{
    const int rows = P.K * P.d;
    const int blocks = (rows + REFINE_WARPS - 1) / REFINE_WARPS;
    const size_t sm = (size_t)REFINE_WARPS * refine_scratch(P.n) * sizeof(double);
    k_refine<<<blocks, REFINE_WARPS * 32, sm, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_pass_result(const Params& P, double* out, cudaStream_t s)
{
    k_pass_result<<<1, 32, 0, s>>>(P, out);
    return cudaGetLastError();
}

cudaError_t launch_update_alpha(const Params& P, cudaStream_t s)
{
    k_update_alpha<<<1, small_block(P.K), 0, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_gen_prepare(const Params& P, cudaStream_t s)
{
    k_gen_prepare<<<1, small_block(P.K), 0, s>>>(P);
    return cudaGetLastError();
}

cudaError_t launch_gen_finish(const Params& P, const PassArgs& G, int64_t remaining, unsigned char* out,
                              cudaStream_t s)
{
    k_gen_scan<<<1, 1024, 0, s>>>(P, G, remaining);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_gen_copy<<<(unsigned)G.nchunks, 256, 0, s>>>(P, G, out);
    return cudaGetLastError();
}

cudaError_t launch_eval(const Params& P, int fp32, const EvalArgs& A, cudaStream_t s)
{
    const int blocks = (A.count + 127) / 128;
    if (fp32) k_eval<float><<<blocks, 128, 0, s>>>(P, A);
    else k_eval<double><<<blocks, 128, 0, s>>>(P, A);
    return cudaGetLastError();
}

}  // namespace vamp
