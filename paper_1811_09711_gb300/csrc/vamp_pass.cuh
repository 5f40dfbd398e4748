// vamp_pass.cuh -- the persistent pass kernel, templated on precision, mode
// (0 integration, 1 generation), calls per thread and problem shape.
//
// Each CTA owns a contiguous range of calls (integration: split further at
// channel boundaries so that its d-value accumulators in shared memory
// belong to one channel) or a strided set of call chunks (generation), and
// processes them in batches of PASS_THREADS*CPT calls:
//   A  per call: Philox words, channel (integration: the segment's; generation:
//      drawn from α), forward map x_c -> p on the channel's grid, its own term
//      α_c g_c/φ'_c of g(p), Gaussian exponent sum (and the integrand when the
//      peaks are not the channels' maps);
//   B  every channel's term of g(p) (Eq. 30) and the matching integrand peak,
//      with the channels' lookup blocks streamed through shared memory in
//      tiles (cp.async.bulk, two buffers, bounded mbarrier waits);
//   C  w = f/g: per-channel shifted sums, d-values D_{c,k,j} += w² (Eq. 15),
//      max |weight| (integration); accept u w_max < |w| and ordered compaction
//      of the event records (generation).
#pragma once

#include "vamp_device.cuh"
#include "vamp_internal.h"

namespace vamp {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}


struct SmemHead {
    uint64_t bar[2];
    int abort;
    int pad;
    double red[3][PASS_THREADS / 32];
    int wcnt[PASS_THREADS / 32];
    int woff[PASS_THREADS / 32];
    int round_total;
};
static_assert(sizeof(SmemHead) <= SMEM_HEAD, "shared-memory head too large");

// Per-thread state of the CPT calls of one batch.
template <typename T, int CPT, int DM>
struct Calls {
    T p[CPT][DM], g[CPT], f[CPT], Aexp[CPT];
    bool valid[CPT];
    int cq[CPT];
    uint32_t jp[CPT][(DM + 3) / 4];
    uint32_t xacc[CPT];
};

// Cell sums of a stratified batch: the call at local index l (from the
// channel's first call) belongs to cell coff + l / spc.
struct CellSums {
    double* sum;     // nullptr: importance sampling
    int64_t l0;      // local index of the batch's first call
    int64_t spc;     // calls per cell
    int64_t coff;    // first cell of the channel
};

// Calls of an integration batch: warp w takes the 32 CPT calls from 32 CPT w
// on, so that a short batch leaves whole warps without calls, and they skip
// it (the 1e4-call pass of a d = 4 problem has 33 calls per CTA).
template <int CPT>
__device__ __forceinline__ int warp_first()
{
    return (int)(threadIdx.x >> 5) * (32 * CPT);
}
template <int CPT>
__device__ __forceinline__ int call_of(int q)
{
    return warp_first<CPT>() + q * 32 + (int)(threadIdx.x & 31);
}

// f / g, 0 where g is not positive.  FP64: by the integer reciprocal, the FP64
// division (ten operations of that pipe) where g is not a normal number or f
// not finite.
__device__ __forceinline__ double call_weight(float f, float g) { return g > 0.f ? (double)(f / g) : 0.0; }
__device__ __forceinline__ double call_weight(double f, double g)
{
    const uint64_t b = sf_bits(g), a = sf_bits(f) & 0x7fffffffffffffffull;
    if (b - 0x0010000000000000ull < 0x7fe0000000000000ull && a < 0x7ff0000000000000ull) return sf_div(f, g);
    return g > 0.0 ? f / g : 0.0;
}

// The larger of wm >= 0 and |w|, and whether w is finite, from the bits (an FP64
// compare takes the pipe that the sums need).
__device__ __forceinline__ double max_abs(double wm, double w)
{
    const long long a = __double_as_longlong(wm), b = __double_as_longlong(w) & 0x7fffffffffffffffll;
    return __longlong_as_double(a > b ? a : b);
}
__device__ __forceinline__ bool finite_bits(double w)
{
    return ((unsigned)__double2hiint(w) & 0x7ff00000u) != 0x7ff00000u;
}

// Phase A: Philox words, channel, forward map on the channel's grid, own
// term of g(p), Gaussian exponent sum; the integrand when peaks are not the
// channels' maps.  Call q of this thread is base + call_of(q) (integration)
// or base + q*PASS_THREADS + tid (generation, whose records are in that order).
template <typename T, int MODE, int CPT, class SH>
__device__ __forceinline__ void phase_a(const Params& P, const SH& sh, uint32_t field, int64_t base, int64_t end,
                                        int cseg, Calls<T, CPT, SH::DM>& C, SoftCall<SH::DM>* soft = nullptr)
{
    constexpr int DM = SH::DM;
    const int d = sh.d();
    const int tid = threadIdx.x;
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        const int64_t i = base + (MODE == 0 ? call_of<CPT>(q) : q * PASS_THREADS + tid);
        C.valid[q] = i < end;
        uint32_t X[DM + 4];
        call_words<DM + 4>(P, (uint32_t)(C.valid[q] ? i : base), field, MODE == 0 ? d : d + 2, X);
        int c;
        if (MODE == 0) {
            c = cseg;
            C.xacc[q] = 0u;
        } else {
            uint32_t xc = 0u, xa = 0u;
#pragma unroll
            for (int k = 0; k < DM + 4; ++k) {
                if (k == d) xc = X[k];
                if (k == d + 1) xa = X[k];
            }
            c = choose_channel(P, unif64(xc));
            C.xacc[q] = xa;
        }
        C.cq[q] = c;
        int jf[DM];
        uint32_t dig[DM], nr = 1u;
        const bool strat = MODE == 0 && SH::kStrat && P.stratified;
        if (strat) {
            // cell of the call and its base-n_r digits (§3.3)
            nr = (uint32_t)P.nr[c];
            uint32_t cell = (uint32_t)((C.valid[q] ? i : base) - P.Pc[c]) / (uint32_t)P.spc[c];  // both < 2^32
#pragma unroll
            for (int k = 0; k < DM; ++k) {
                dig[k] = 0u;
                if (sh.has(k)) {
                    const uint32_t up = cell / nr;
                    dig[k] = cell - up * nr;
                    cell = up;
                }
            }
        }
        if constexpr (sizeof(T) == 8) {
            double own;
            if (strat) soft_forward(P, sh, c, X, C.p[q], jf, own, *soft, dig, nr);
            else soft_forward(P, sh, c, X, C.p[q], jf, own, *soft);
            C.Aexp[q] = soft->A;
            C.g[q] = __ldg(P.alphaN + c) * own;
        } else {
            T x[DM], owngJ, Aq;
            if (strat) forward_call<T>(P, sh, c, X, x, C.p[q], jf, owngJ, Aq, dig, nr);
            else forward_call<T>(P, sh, c, X, x, C.p[q], jf, owngJ, Aq);
            C.Aexp[q] = Aq;
            C.g[q] = Prec<T>::alpha(P, c) * owngJ;
        }
#pragma unroll
        for (int w = 0; w < (DM + 3) / 4; ++w) {
            uint32_t v = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (4 * w + b < DM) v |= (uint32_t)(jf[4 * w + b] & 0xff) << (8 * b);
            C.jp[q][w] = v;
        }
        C.f[q] = P.matching ? T(0) : integrand_peaks<T, DM>(P, d, C.p[q], C.Aexp[q]);
    }
}

// Phase B for one staged tile: channels t*tile .. of the tile buffer tb.
template <typename T, int MODE, int CPT, class SH>
__device__ __forceinline__ void tile_compute(const Params& P, const SH& sh, const unsigned char* tb, int t, int tile,
                                             int cseg, Calls<T, CPT, SH::DM>& C, const SoftCall<SH::DM>* soft)
{
    const int S = sh.bytes();
    const int cnt = min(tile, P.K - t * tile);
    for (int cl = 0; cl < cnt; ++cl) {
        const int c2 = t * tile + cl;
        const unsigned char* blk = tb + (size_t)cl * S;
        if constexpr (sizeof(T) == 8) {
            const double a = __ldg(P.alphaN + c2);
            const bool lookups = (a != 0.0) && !(MODE == 0 && c2 == cseg);
            double gt, ft;
            soft_channel<false>(P, sh, blk, lookups, C.p[0], *soft, gt, ft, nullptr);
            if (lookups && !(MODE == 1 && C.cq[0] == c2)) C.g[0] += a * gt;
            if (P.matching) C.f[0] += reinterpret_cast<const ChanHdr<double>*>(blk)->fN * ft;
        } else {
            bool skip[CPT];
            const T a = Prec<T>::alpha(P, c2);
            const bool lookups = (a != T(0)) && !(MODE == 0 && c2 == cseg);
#pragma unroll
            for (int q = 0; q < CPT; ++q) skip[q] = (MODE == 1) && (C.cq[q] == c2);
            channel_body<T, CPT, false>(P, sh, blk, a, lookups, P.matching != 0, C.p, C.Aexp, skip, C.g, C.f, nullptr);
        }
    }
}

// Word i of a small register array, by a chain of selects (no local memory).
template <int W>
__device__ __forceinline__ uint32_t pick(const uint32_t (&a)[W], int i)
{
    uint32_t v = a[0];
#pragma unroll
    for (int t = 1; t < W; ++t) v = i == t ? a[t] : v;
    return v;
}

// Phase C of an integration batch: shifted sums, max weight and the d-values
// (Eq. 15) of the segment's channel in shared memory (FP64 atomics, which
// retry on collisions), in 2^dshift copies (plan_tiles).  Unless the shape has
// many bins per axis (a lane's bins then rarely collide), lane l adds its d
// terms in the rotated axis order l, l+1, ... (mod d), so that at any step the
// lanes of a warp hit different rows, and lanes that share a row (l, l+d, ...)
// different copies.
template <typename T, int CPT, class SH>
__device__ __forceinline__ void phase_c_int(const SH& sh, const Calls<T, CPT, SH::DM>& C, double sft, double* Ds,
                                            int dshift, double& s1, double& s2, double& wm, bool& bad,
                                            const CellSums cs = CellSums{nullptr, 0, 1, 0})
{
    constexpr int DM = SH::DM;
    const int d = sh.d(), n = sh.n(), lane = threadIdx.x & 31;
    constexpr bool kRotate = !(SH::kN && SH::NBC >= 64);
    const int rot = kRotate ? lane % d : 0;
    double* Dl = Ds + ((kRotate ? lane / d : lane) & ((1 << dshift) - 1));
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        if (!C.valid[q]) continue;
        double w = call_weight(C.f[q], C.g[q]);
        if (!finite_bits(w)) { bad = true; w = 0.0; }
        const double dv = w - sft;
        s1 += dv;
        s2 += dv * dv;
        if (cs.sum)  // stratified: the sum of the call's cell
            atomicAdd(&cs.sum[cs.coff + (uint32_t)(cs.l0 + call_of<CPT>(q)) / (uint32_t)cs.spc], dv);
        wm = max_abs(wm, w);  // signed integrands: w_max bounds |w|
        const double w2 = w * w;
#pragma unroll
        for (int s = 0; s < DM; ++s) {
            if (sh.has(s)) {
                int k = s;
                uint32_t v = C.jp[q][s >> 2];
                if (kRotate) {
                    k = s + rot;
                    if (k >= d) k -= d;
                    v = pick(C.jp[q], k >> 2);
                }
                atomicAdd(&Dl[(k * n + (int)((v >> (8 * (k & 3))) & 0xff)) << dshift], w2);
            }
        }
    }
}

// Phase C of a generation batch (chunk `chunk`, calls from `base`): accept iff
// u w_max < |w| and write the accepted records of the chunk in call order
// (ballot within a warp, warp offsets through shared memory), then the
// chunk's count.  Every thread of the CTA takes part.
template <typename T, int CPT, class SH>
__device__ __forceinline__ void phase_c_gen(const Params& P, const PassArgs& A, const SH& sh,
                                            const Calls<T, CPT, SH::DM>& C, int64_t chunk, int64_t base,
                                            int* wcnt, int* woff, int* round_total, double& wm, bool& bad)
{
    constexpr int DM = SH::DM;
    constexpr int B = PASS_THREADS * CPT;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const double wmax = P.sc->wmax_gen;
    int running = 0;
    const int64_t cbase = chunk * B;
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        double w = 0.0;
        bool acc = false;
        if (C.valid[q]) {
            w = call_weight(C.f[q], C.g[q]);
            if (!finite_bits(w)) { bad = true; w = 0.0; }
            wm = max_abs(wm, w);
            acc = unif64(C.xacc[q]) * wmax < fabs(w);  // the event keeps the sign of w
        }
        const unsigned bal = __ballot_sync(0xffffffffu, acc);
        if (lane == 0) wcnt[wid] = __popc(bal);
        __syncthreads();
        if (tid == 0) {
            int s = 0;
            for (int w2 = 0; w2 < PASS_THREADS / 32; ++w2) { woff[w2] = s; s += wcnt[w2]; }
            *round_total = s;
        }
        __syncthreads();
        if (acc) {
            const int pos = running + woff[wid] + __popc(bal & ((1u << lane) - 1u));
            const int64_t slot = cbase + pos;
            // record {float p[d]; zero pad to 8 bytes; double w}: 8-byte
            // stores (records are 8-byte multiples at 8-byte offsets)
            unsigned char* rec = A.staging + slot * A.rec_bytes;
            float2* pf2 = reinterpret_cast<float2*>(rec);
#pragma unroll
            for (int k = 0; k < DM; k += 2)
                if (sh.has(k))
                    pf2[k >> 1] = make_float2((float)C.p[q][k],
                                              (k + 1 < DM && sh.has(k + 1)) ? (float)C.p[q][k + 1] : 0.0f);
            *reinterpret_cast<double*>(rec + A.rec_bytes - 8) = w;
            A.callidx[slot] = (uint32_t)(base + (int64_t)q * PASS_THREADS + tid);
        }
        running += *round_total;
        __syncthreads();
    }
    if (tid == 0) A.counts[chunk] = running;
}

// Flush of a segment: block sums of (s1, s2) and the d-values to global.
__device__ __forceinline__ void flush_segment(const Params& P, SmemHead& H, int cseg, int dn, double* Ds,
                                              int dshift, double s1, double s2)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0) { H.red[0][wid] = s1; H.red[1][wid] = s2; }
    __syncthreads();
    if (tid == 0) {
        double a = 0.0, bb = 0.0;
        for (int q = 0; q < PASS_THREADS / 32; ++q) { a += H.red[0][q]; bb += H.red[1][q]; }
        atomicAdd(&P.csum[2 * cseg], a);
        atomicAdd(&P.csum[2 * cseg + 1], bb);
    }
    double* Dg = P.D + (size_t)cseg * dn;
    for (int q = tid; q < dn; q += PASS_THREADS) {
        double v = 0.0;
        for (int r = 0; r < 1 << dshift; ++r) v += Ds[(q << dshift) + ((r + tid) & ((1 << dshift) - 1))];
        if (v != 0.0) atomicAdd(&Dg[q], v);
    }
    __syncthreads();
}

// Block maximum of wm into *dst (non-negative doubles compare as bits).
__device__ __forceinline__ void block_max_to(SmemHead& H, double wm, unsigned long long* dst)
{
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    wm = warp_max(wm);
    if (lane == 0) H.red[2][wid] = wm;
    __syncthreads();
    if (tid == 0) {
        double m = 0.0;
        for (int q = 0; q < PASS_THREADS / 32; ++q) m = fmax(m, H.red[2][q]);
        atomicMax(dst, (unsigned long long)__double_as_longlong(m));
    }
}

template <typename T, int MODE, int CPT, class SH>
__device__ __forceinline__ void pass_body(const Params& P, const PassArgs& A)
{
    constexpr int DM = SH::DM;
    extern __shared__ __align__(128) unsigned char smem[];
    SmemHead& H = *reinterpret_cast<SmemHead*>(smem);
    unsigned char* buf0 = smem + SMEM_HEAD;
    const SH sh(Prec<T>::lay(P), P.d, P.n);
    const int S = sh.bytes();
    const size_t tile_bytes = (size_t)A.tile * S;
    const size_t tiles_bytes = (A.ntiles > 1 ? 2 : 1) * tile_bytes;
    double* Ds = reinterpret_cast<double*>(buf0 + tiles_bytes);
    const int d = sh.d(), n = sh.n(), dn = d * n, K = P.K;
    int dshift = A.dshift;
    const int tid = threadIdx.x;
    constexpr int B = PASS_THREADS * CPT;
    const unsigned char* lk = Prec<T>::lk(P);
    SoftCall<DM> soft;  // FP64: what the channel loop needs of the call

    // ---- work of this CTA ---------------------------------------------------
    int64_t r0 = 0, r1 = 0;
    int64_t nbatch = 0;
    if (MODE == 0) {
        const int64_t N = P.sc->n_total;
        // whole warps of calls, so that a small pass has few half-empty ones
        r0 = (N * blockIdx.x / gridDim.x) & ~int64_t(31);
        r1 = blockIdx.x + 1 < gridDim.x ? (N * (blockIdx.x + 1) / gridDim.x) & ~int64_t(31) : N;
        // copies only as far as the calls outnumber the words to clear and sum
        while (dshift > 0 && r1 - r0 < (int64_t)(4 * n) << dshift) --dshift;
        int64_t i = r0;
        while (i < r1) {
            const int c = find_channel(P.Pc, K, i);
            const int64_t e = min(r1, P.Pc[c + 1]);
            nbatch += (e - i + B - 1) / B;
            i = e;
        }
    } else {
        const int64_t nch = A.nchunks;
        nbatch = blockIdx.x < nch ? (nch - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    }
    if (nbatch == 0) return;
    const int ntiles = A.ntiles;
    const bool streaming = ntiles > 2;
    const int64_t total_uses = streaming ? nbatch * ntiles : ntiles;

    auto issue = [&](int64_t u) {
        const int t = (int)(u % ntiles);
        const int cnt = min(A.tile, K - t * A.tile);
        fence_proxy_async_smem();
        bulk_load(buf0 + (u & 1) * tile_bytes, lk + (size_t)t * tile_bytes, (uint32_t)(cnt * S), &H.bar[u & 1]);
    };
    if (tid == 0) {
        mbar_init(&H.bar[0], 1);
        mbar_init(&H.bar[1], 1);
        H.abort = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0) {
        issue(0);
        if (total_uses > 1) issue(1);
    }
    int64_t u = 0;              // next tile use to consume
    int64_t issued = total_uses > 1 ? 2 : 1;
    double wm = 0.0, s1 = 0.0, s2 = 0.0;
    bool bad = false;

    // integration segment state
    int64_t i0 = r0;
    int cseg = -1;
    int64_t seg_end = 0;
    double sft = 0.0;
    // generation chunk state
    int64_t chunk = blockIdx.x;

    for (int64_t bt = 0; bt < nbatch; ++bt) {
        int64_t base, end;
        if (MODE == 0) {
            if (i0 >= seg_end || cseg < 0) {
                // new segment of one channel: reset the shared d-values
                cseg = find_channel(P.Pc, K, i0);
                seg_end = min(r1, P.Pc[cseg + 1]);
                sft = P.shift[cseg];
                for (int q = tid; q < dn << dshift; q += PASS_THREADS) Ds[q] = 0.0;
                s1 = s2 = 0.0;
                __syncthreads();
            }
            base = i0;
            end = min(seg_end, i0 + B);
        } else {
            base = chunk * B;
            end = min(A.batch, base + B);
        }

        // ---- phase A: own channel forward map, integrand --------------------
        Calls<T, CPT, DM> C;
        const bool live = MODE == 1 || base + warp_first<CPT>() < end;  // some call of this warp
        if (live) phase_a<T, MODE, CPT>(P, sh, A.field, base, end, cseg, C, &soft);

        // ---- phase B: every channel's term of g(p) (and the matching peaks) --
        for (int t = 0; t < ntiles; ++t) {
            // streaming: use u lives in buffer u%2 (phase u/2); otherwise tile t
            // stays in buffer t after the first batch
            const int b = streaming ? (int)(u & 1) : t;
            if (streaming || bt == 0) {
                if (!mbar_wait_bounded(&H.bar[b], streaming ? (uint32_t)((u >> 1) & 1) : 0u)) {
                    atomicOr(&P.sc->err, ERR_TIMEOUT);
                    H.abort = 1;
                }
            }
            if (live && !H.abort)
                tile_compute<T, MODE, CPT>(P, sh, buf0 + b * tile_bytes, t, A.tile, cseg, C, &soft);
            __syncthreads();
            if (H.abort) goto drain;
            if (streaming && tid == 0 && issued < total_uses) {
                issue(issued);
                ++issued;
            }
            ++u;
        }

        // ---- phase C: weights and accumulation ------------------------------
        if (MODE == 0) {
            if (live)
                phase_c_int<T, CPT>(sh, C, sft, Ds, dshift, s1, s2, wm, bad,
                                    (SH::kStrat && P.stratified)
                                        ? CellSums{P.cellsum, base - P.Pc[cseg], P.spc[cseg], P.coff[cseg]}
                                        : CellSums{nullptr, 0, 1, 0});
            i0 = end;
            if (i0 >= seg_end) {
                // end of the segment: flush its sums and d-values
                flush_segment(P, H, cseg, dn, Ds, dshift, s1, s2);
                s1 = s2 = 0.0;
            }
        } else {
            phase_c_gen<T, CPT>(P, A, sh, C, chunk, base, H.wcnt, H.woff, &H.round_total, wm, bad);
            chunk += gridDim.x;
        }
    }

    // ---- CTA totals --------------------------------------------------------
    if (bad) atomicOr(&P.sc->err, ERR_NONFINITE);
    block_max_to(H, wm, MODE == 0 ? &P.sc->wmax_bits : &P.sc->gen_bmax_bits);
    return;

drain:
    // a wait gave up: let this CTA's copies in flight land (bounded), then exit
    if (tid == 0) {
        if (streaming) {
            for (int64_t v = u; v < issued; ++v) mbar_wait_bounded(&H.bar[v & 1], (uint32_t)((v >> 1) & 1));
        } else {
            for (int64_t v = u; v < issued; ++v) mbar_wait_bounded(&H.bar[v], 0u);
        }
    }
    __syncthreads();
}

template <typename T, int MODE, int CPT, int D_, int NB_, int MINB>
__global__ void __launch_bounds__(PASS_THREADS, MINB) k_pass(Params P, PassArgs A)
{
    pass_body<T, MODE, CPT, Shape<T, D_, NB_>>(P, A);
}

// Any number of bins, d in [DLO_, DHI_]: the row loops unroll to DHI_ and the
// first DLO_ rows need no test.  With the loops of the any-d form (16 rows) the
// FP64 pass took 589 against 484 us at d = 8 (K = 6, 1e6 calls) and 59.7
// against 55.6 ms at d = 14 (K = 64, 1e7 calls): fewer registers and less code.
template <typename T, int MODE, int CPT, int DLO_, int DHI_, int MINB>
__global__ void __launch_bounds__(PASS_THREADS, MINB) k_pass_dims(Params P, PassArgs A)
{
    pass_body<T, MODE, CPT, Shape<T, 0, 0, DHI_, DLO_>>(P, A);
}

// Registers the integration and generation kernels of one (T, CPT, D, NB,
// CTAs per SM), or of one (T, CPT, range of d).
template <typename T, int CPT, int D_, int NB_, int MINB>
cudaError_t pass_launch_t(const Params& P, int mode, const PassArgs& A, int grid, size_t smem, cudaStream_t s)
{
    if (mode) k_pass<T, 1, CPT, D_, NB_, MINB><<<grid, PASS_THREADS, smem, s>>>(P, A);
    else k_pass<T, 0, CPT, D_, NB_, MINB><<<grid, PASS_THREADS, smem, s>>>(P, A);
    return cudaGetLastError();
}

template <typename T, int CPT, int DLO_, int DHI_, int MINB>
cudaError_t pass_launch_dims(const Params& P, int mode, const PassArgs& A, int grid, size_t smem, cudaStream_t s)
{
    if (mode) k_pass_dims<T, 1, CPT, DLO_, DHI_, MINB><<<grid, PASS_THREADS, smem, s>>>(P, A);
    else k_pass_dims<T, 0, CPT, DLO_, DHI_, MINB><<<grid, PASS_THREADS, smem, s>>>(P, A);
    return cudaGetLastError();
}

template <typename T, int CPT, int DLO_, int DHI_, int MINB = 2>
PassVariant make_variant_dims()
{
    PassVariant v;
    v.fp32 = sizeof(T) == 4;
    v.cpt = CPT;
    v.D = v.NB = 0;
    v.dlo = DLO_;
    v.dhi = DHI_;
    v.minb = MINB;
    v.family = "k_pass";
    v.fn[0] = (const void*)k_pass_dims<T, 0, CPT, DLO_, DHI_, MINB>;
    v.fn[1] = (const void*)k_pass_dims<T, 1, CPT, DLO_, DHI_, MINB>;
    v.launch = &pass_launch_dims<T, CPT, DLO_, DHI_, MINB>;
    return v;
}

template <typename T, int CPT, int D_, int NB_, int MINB = 2>
PassVariant make_variant()
{
    PassVariant v;
    v.fp32 = sizeof(T) == 4;
    v.cpt = CPT;
    v.D = D_;
    v.NB = NB_;
    v.minb = MINB;
    v.family = "k_pass";
    v.fn[0] = (const void*)k_pass<T, 0, CPT, D_, NB_, MINB>;
    v.fn[1] = (const void*)k_pass<T, 1, CPT, D_, NB_, MINB>;
    v.launch = &pass_launch_t<T, CPT, D_, NB_, MINB>;
    return v;
}

}  // namespace vamp
