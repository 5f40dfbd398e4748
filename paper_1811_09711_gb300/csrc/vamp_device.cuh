// vamp_device.cuh -- device-side building blocks of the sampling hot path.
//
// One call of the doubly adaptive multi-channel integrator (§3.5 work order):
//   r (Philox words) -> x_c = G_c^{-1}(r) on the selected channel's grid
//   -> p = φ_c(x_c) -> f(p) -> for every channel c': x_c' = φ_c'^{-1}(p),
//   bin lookup on grid c', g_c'(x_c') / φ'_c' -> g(p) (Eq. 30) -> w = f/g.
// Everything is templated on the evaluation type T: double (FP64 path) or
// float (FP32-eval path).  Sums are always FP64 (in the kernels).
//
// Grid data of one channel lives in one contiguous "lookup block" so that a
// tile of channels can be staged into shared memory with one bulk copy:
//   [header: map constants of the channel]
//   [row 0: edges (Es) | densities 1/(nΔx) (Dn) | cell table (Ts bytes)] [row 1] ...
// The cell table of a row splits [0,1) into L = 2^lshift equal cells and
// stores for cell q the bin containing q/L (byte L+1 holds the row's span:
// the most bins any cell overlaps), so a lookup starts next to its answer.
// Density entry n repeats entry n-1, so that a probe of edge ξ_n = 1 by a
// point at (or rounded past) 1 needs no bounds check: it lands on entry n
// with the last bin's density.  In the FP64 blocks the densities are packed
// numbers (vamp_soft64.cuh), and the rows of mapped coordinates hold the
// images φ_c(ξ_j) of the edges: the maps are increasing, so the bin of
// φ_c^{-1}(p) is the bin whose image holds p, decided with no inverse map; the
// cell table of such a row is over x, entered with an FP32 inverse map.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "vamp_soft64.cuh"

namespace vamp {

constexpr int DMAX = 16;      // largest supported dimension
constexpr int MAXMAP = 4;     // mapped coordinates per channel / peak
constexpr int MAX_BINS = 256; // largest supported bins per axis (table entries are bytes)

enum : int { MAP_ID = 0, MAP_BW = 1, MAP_POW = 2 };
enum : unsigned { ERR_NONFINITE = 1u, ERR_TIMEOUT = 2u };

// Map constants of one channel or peak (used from global memory by the
// non-matching integrand path and by the host).
template <typename T>
struct MapRec {
    int32_t nmap;
    uint32_t mask;      // bit k: coordinate k is mapped
    uint64_t slotpack;  // 4 bits per coordinate: its slot
    int32_t kind[MAXMAP];
    T m[MAXMAP];        // Breit-Wigner mass
    T G[MAXMAP];        // Breit-Wigner width Γ
    T invG[MAXMAP];     // 1/Γ
    T A[MAXMAP];        // atan((1-m)/Γ) + atan(m/Γ)
    T GinvA[MAXMAP];    // Γ/A
    T invA[MAXMAP];     // 1/A
    T t0[MAXMAP];       // atan(m/Γ)
    T del[MAXMAP];      // power-law factor offset δ
    T invPowN[MAXMAP];  // 1 / (5((1+δ)^0.2 - δ^0.2))
    T wz;               // peak weight x Z^-(d - nmap) (Gaussian normalisation)
};

// Slot constants inside a lookup-block header.
enum : int { SP_M = 0, SP_G, SP_A, SP_G2, SP_INVG, SP_GINVA, SP_INVA, SP_T0, SP_DEL, SP_INVPOWN, SP_N };

// Header of a lookup block: what the channel loop needs about channel c'.
template <typename T>
struct ChanHdr {
    uint32_t mask;       // bit k: coordinate k is mapped
    uint32_t kinds;      // byte s: map kind of slot s
    uint64_t slotpack;   // 4 bits per coordinate: its slot
    T wz;                // matching peak: weight x Z^-(d - nmap)
    uint32_t slow;       // bit k: some cell of row k overlaps more than two bins (kept by the derive kernel)
    uint32_t pad[(16 - (sizeof(T) + 4) % 16) % 16 / 4];
    T sp[MAXMAP][SP_N];  // per slot: m, Γ, A, Γ², 1/Γ, Γ/A, 1/A, atan(m/Γ), δ, 1/powN
};
// FP64: the mapped coordinates as a list, and what does not depend on the
// call folded into two constants.
template <>
struct alignas(16) ChanHdr<double> {
    uint32_t slow;       // bit k: some cell of (unmapped) row k overlaps more than two bins
    uint32_t mmask;      // bit k: coordinate k has a Breit-Wigner or power-law map
    double gN;           // Π_BW Γ/A x 0.2^(number of power-law slots), times α the constant of the term of g(p)
    double fN;           // wz Π_BW Γ/A Π_POW 1/powN: the constant of the matching peak
    uint32_t nslot;      // Breit-Wigner and power-law slots
    uint32_t bw;         // 1: some are Breit-Wigner; 2: of widths far from 1
    // bw = 2: gN and fN are 2^-ge of the above, and the denominators' product
    // is divided by 2^ge, so that neither leaves the range of a double where
    // their ratio does not (0 otherwise)
    int32_t ge;
    uint8_t sk[MAXMAP];  // their coordinate | kind << 4
    double c0[MAXMAP], c1[MAXMAP];    // Breit-Wigner: m, Γ²; power law: δ
    double fw[MAXMAP][3];             // Breit-Wigner: Γ, A, atan(m/Γ)
    float pinvG[MAXMAP], pt0[MAXMAP], pscale[MAXMAP];  // FP32 inverse map to cells: (atan(dp/Γ) + t0) scale; x scale
};
static_assert(sizeof(ChanHdr<float>) % 16 == 0 && sizeof(ChanHdr<double>) % 16 == 0, "header not 16-byte sized");

// Byte layout of one channel's lookup block for element type T.
struct BlkLayout {
    int H;         // header bytes
    int Es;        // edges per row (>= n+1, padded)
    int Dn;        // densities per row (>= n+1, padded; entry n repeats entry n-1)
    int Ts;        // table bytes per row (>= L+2, padded)
    int R;         // row stride in bytes
    int lshift;    // L = 2^lshift cells per row
    int bytes;     // block size (multiple of 16)
};

// Device-resident scalars of one context.  The head (up to `n_hist`) is
// what the host copies back after a pass or a generation batch.
struct Scalars {
    int64_t n_total;                 // Σ N_c of the current pass
    unsigned long long wmax_bits;    // max weight of the pass (non-negative double bits)
    unsigned int err;                // ERR_* flags
    unsigned int pad0;
    double wmax_gen;                 // w_max used by generation
    double res[8];                   // pass result, vamp_pass_result order (n_calls slot unused)
    // generation batch bookkeeping
    unsigned long long gen_bmax_bits;
    long long gen_total;             // accepted in this batch
    long long gen_take;              // taken from this batch
    long long gen_used;              // calls consumed in this batch
    long long gen_over;              // overweights among taken
    double wmax_cut;                 // w_max that this batch was accepted against
    // history of passes for the combination of iterations
    int32_t n_hist;
    int32_t pad1;
    double hist_I[1024];
    double hist_V[1024];
    int32_t hist_comb[1024];
};

// All pointers and sizes a kernel needs (passed by value).
struct Params {
    int d, K, n, P;
    int fp32;              // evaluation precision of the passes
    uint32_t map_any, pow_any;  // bit k: some channel has a Breit-Wigner or power-law map (a power-law map) on k
    int gauss_sum;         // the Gaussian factor of one coordinate can leave the packed range: exponents are summed
    int matching;          // peaks are the channels' maps (integrand fused into the channel loop)
    uint32_t key0, key1, request;
    int64_t n_min;
    double grid_alpha, beta;
    int smooth, omega_mode;
    // maps (host order, for the non-matching integrand)
    const MapRec<double>* pk64;
    const MapRec<float>* pk32;
    // Gaussian factor in log2 units: a_k = (p_k - centre)^2 * gk2
    double gcen, gk2;
    float gcen_f, gk2_f;
    // lookup blocks
    unsigned char* lk64;   // [K][lay64.bytes]
    unsigned char* lk32;   // [K][lay32.bytes]
    BlkLayout lay64, lay32;
    // state
    double* edges64;   // [K][d][n+1] FP64 master grid
    double* alpha;     // [K]
    float* alpha32;    // [K]
    double* alphaN;    // [K] α times the header's gN (kept with alpha32)
    double* shift;     // [K]
    double* Acum;      // [K] cumulative α for generation
    int64_t* Nc;       // [K]
    int64_t* Pc;       // [K+1]
    double* D;         // [K][d][n]
    double* csum;      // [K][2]: Σ (w - s_c), Σ (w - s_c)^2
    double* Ic;        // [K]
    double* Vc;        // [K]
    double* Wc;        // [K]
    Scalars* sc;
    // pseudo-stratified sampling (§3.3), when stratified != 0
    int stratified;
    int64_t* nr;       // [K] cells per r axis
    int64_t* spc;      // [K] calls per cell
    int64_t* coff;     // [K+1] first cell of each channel
    double* Qc;        // [K] Σ over the channel's cells of (Σ_cell (w - s_c))^2
    double* cellsum;   // [Σ cells] Σ_cell (w - s_c) of the pass (context-owned, grows)
    // channel equivalences (§3.5): the bin weights that rebin grid row r are
    // D[r] plus the terms eq_ent[eq_off[r] .. eq_off[r+1]) in list order, each
    // (source row << 2 | kind); null without equivalences
    int n_eq_ent;
    const int32_t* eq_off;   // [K*d + 1]
    const int32_t* eq_ent;   // [n_eq_ent]
    // interval tables of the FP32-eval union pass (null unless that kernel
    // is in use; rebuilt whenever the grids change): for coordinate k the
    // sorted distinct values U_k of every channel's edge images φ_c(ξ_{c,k,j})
    // (rounded up to FP32), a cell index over them, and for each interval
    // [U_k[u], U_k[u+1]) the bin densities of all channels (UNION_SLOTS wide)
    int uMax;          // row stride of uImg / uU / uD: K (n+1)
    float* uImg;       // [d][K][n+1] edge images per coordinate and channel
    float* uU;         // [d][uMax] sorted distinct images (first uNU[k] valid)
    int* uNU;          // [d]
    uint32_t* uC;      // [d][UNION_CELLS]: count of U_k <= q/L (low 16 bits), values inside the cell (high 16)
    float* uD;         // [d][uMax][UNION_SLOTS] densities of every channel on each interval
};

constexpr int UNION_SLOTS = 64;        // channels per density row of the union tables
constexpr int UNION_LCELLS = 16;       // log2 of the cells per coordinate of the union search
constexpr int UNION_CELLS = 1 << UNION_LCELLS;
constexpr int UNION_MAXV = 16384;      // largest K (n+1) the union tables take (16-bit indices, one sort block)

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 10 rounds of the
// multiply-xor round function with Weyl key schedule.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) { k0 += W0; k1 += W1; }
        const uint32_t lo0 = M0 * c.x, hi0 = __umulhi(M0, c.x);
        const uint32_t lo1 = M1 * c.z, hi1 = __umulhi(M1, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

// Words 0..nw-1 of one call (counter = call, block, field, request).
template <int NWMAX>
__device__ __forceinline__ void call_words(const Params& P, uint32_t call, uint32_t field, int nw,
                                           uint32_t (&X)[NWMAX])
{
#pragma unroll
    for (int b = 0; b < (NWMAX + 3) / 4; ++b) {
        if (4 * b < nw) {
            const uint4 o = philox4x32_10(make_uint4(call, (uint32_t)b, field, P.request), P.key0, P.key1);
            if (4 * b + 0 < NWMAX) X[4 * b + 0] = o.x;
            if (4 * b + 1 < NWMAX) X[4 * b + 1] = o.y;
            if (4 * b + 2 < NWMAX) X[4 * b + 2] = o.z;
            if (4 * b + 3 < NWMAX) X[4 * b + 3] = o.w;
        }
    }
}

// u = (X + 1/2) 2^-32 in (0, 1), exact in FP64.
__device__ __forceinline__ double unif64(uint32_t X) { return ((double)X + 0.5) * 0x1p-32; }

// ---------------------------------------------------------------------------
// Precision traits.
// ---------------------------------------------------------------------------
template <typename T> struct Prec;

template <> struct Prec<double> {
    static __device__ __forceinline__ const unsigned char* lk(const Params& P) { return P.lk64; }
    static __device__ __forceinline__ const BlkLayout& lay(const Params& P) { return P.lay64; }
    static __device__ __forceinline__ const MapRec<double>* pk(const Params& P) { return P.pk64; }
    static __device__ __forceinline__ double alpha(const Params& P, int c) { return P.alpha[c]; }
    static __device__ __forceinline__ double gcen(const Params& P) { return P.gcen; }
    static __device__ __forceinline__ double gk2(const Params& P) { return P.gk2; }
    // in-bin fraction of the forward map: the exact 33-bit value
    static __device__ __forceinline__ double frac(uint64_t low33) { return sf_frac33(low33); }
    // x = ξ_j + frac (ξ_{j+1} - ξ_j), rounded as two separate operations
    static __device__ __forceinline__ double lerp(double e0, double e1, double fr)
    {
        return __dadd_rn(e0, __dmul_rn(fr, __dsub_rn(e1, e0)));
    }
    static __device__ __forceinline__ double tan_(double v) { return sf_tan(v); }
    // v^(-1/5) for a normal v > 0 (Newton's method for the inverse fifth
    // root): with v = m 2^E, m in [1, 2), write -E = 5a + r (r in 0..4), so
    // v^(-1/5) = 2^a w^(-1/5) with w = m 2^-r in [1/16, 2).  The seed
    // 2^(-0.2 log2 w) comes from the FP32 special-function approximations
    // (relative error about 1e-7); two division-free Newton steps for
    // y^-5 = w, y <- y (6 - w y^5) / 5, each squaring the relative error,
    // bring it to a few units in the last place.
    static __device__ __forceinline__ double rinv5(double v)
    {
        const long long b = __double_as_longlong(v);
        const int ne = 1023 - (int)((b >> 52) & 0x7ff);  // -E
        const int a = ne >= 0 ? ne / 5 : -((4 - ne) / 5);
        const int r = ne - 5 * a;
        const double w = __longlong_as_double((b & 0x000FFFFFFFFFFFFFll) | ((long long)(1023 - r) << 52));
        float s;
        float l;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"((float)w));  // w is normal
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(-0.2f * l));
        double y = (double)s;
#pragma unroll
        for (int it = 0; it < 2; ++it) {
            const double y2 = y * y, y4 = y2 * y2;
            y = y * fma(-w, y4 * y, 6.0) * 0.2;
        }
        return y * __longlong_as_double((long long)(1023 + a) << 52);  // times 2^a
    }
    // v^-0.8 = (v^(-1/5))^4
    static __device__ __forceinline__ double powm08(double v)
    {
        const double y = rinv5(v), y2 = y * y;
        return y2 * y2;
    }
    static __device__ __forceinline__ double exp2_(double v) { return exp2(v); }
    static __device__ __forceinline__ double tiny() { return 2.2250738585072014e-308; }
    // e <= x for the non-negative edges: compare bit patterns (integer pipe)
    static __device__ __forceinline__ bool le(double e, double x)
    {
        return __double_as_longlong(e) <= __double_as_longlong(x);
    }
    // floor(x L) for x clamped to [0, 1), from the bit pattern with integer
    // operations only (the FP64 pipe is the scarce one): x = m 2^(e-52) with
    // the 53-bit significand m, so floor(x 2^lshift) = m >> (52 - e - lshift)
    static __device__ __forceinline__ int cell(double x, int lshift)
    {
        const long long b = __double_as_longlong(x);
        if (b <= 0) return 0;                                    // x <= 0 (or -0)
        if (b >= 0x3FF0000000000000ll) return (1 << lshift) - 1; // x >= 1
        const int e = (int)(b >> 52) - 1023;                     // e <= -1
        const int sh = 52 - e - lshift;
        const unsigned long long m = (unsigned long long)(b & 0xFFFFFFFFFFFFFll) | (1ull << 52);
        return sh >= 64 ? 0 : (int)(m >> sh);
    }
};

template <> struct Prec<float> {
    static __device__ __forceinline__ const unsigned char* lk(const Params& P) { return P.lk32; }
    static __device__ __forceinline__ const BlkLayout& lay(const Params& P) { return P.lay32; }
    static __device__ __forceinline__ const MapRec<float>* pk(const Params& P) { return P.pk32; }
    static __device__ __forceinline__ float alpha(const Params& P, int c) { return P.alpha32[c]; }
    static __device__ __forceinline__ float gcen(const Params& P) { return P.gcen_f; }
    static __device__ __forceinline__ float gk2(const Params& P) { return P.gk2_f; }
    // top 24 bits of the 33-bit fraction (exact conversion)
    static __device__ __forceinline__ float frac(uint64_t low33) { return (float)(uint32_t)(low33 >> 9) * 0x1p-24f; }
    static __device__ __forceinline__ float lerp(float e0, float e1, float fr) { return fmaf(fr, e1 - e0, e0); }
    static __device__ __forceinline__ float tan_(float v) { return tanf(v); }
    static __device__ __forceinline__ float atan_(float v) { return atanf(v); }
    // 2^v by the ex2.approx instruction (relative error about 2^-22; flushes
    // results below the normal range to zero, where the factors it scales
    // are negligible)
    static __device__ __forceinline__ float ex2(float v)
    {
        float r;
        asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
        return r;
    }
    // log2 v by the lg2.approx instruction, flush-to-zero form: the
    // arguments here are 0 or normal numbers (coordinates are sums and
    // products of uniform fractions and bin widths, and the power map
    // floors p at the smallest normal), on which it equals the form with
    // subnormal support and skips that form's rescaling steps
    static __device__ __forceinline__ float lg2(float v)
    {
        float r;
        asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
        return r;
    }
    static __device__ __forceinline__ float pow02(float v) { return ex2(0.2f * lg2(v)); }
    static __device__ __forceinline__ float powm08(float v) { return ex2(-0.8f * lg2(v)); }
    static __device__ __forceinline__ float exp2_(float v) { return ex2(v); }
    // Jacobian factors of the FP32-eval form: a (1/b) by the div.approx
    // instruction (within 2 ulp for |b| in [2^-126, 2^126]), flush-to-zero
    // form: the denominators and quotients that occur here are normal
    static __device__ __forceinline__ float div(float a, float b)
    {
        float r;
        asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
        return r;
    }
    static __device__ __forceinline__ float tiny() { return 1.17549435e-38f; }
    static __device__ __forceinline__ bool le(float e, float x) { return e <= x; }
    // floor(x L) of x clamped to [0, 1], in [0, L]: x L + 2^23 rounded toward
    // zero is exact and its low mantissa bits are the integer part
    static __device__ __forceinline__ int cell(float x, int lshift)
    {
        const float y = __fmaf_rz(__saturatef(x), (float)(1 << lshift), 0x1p23f);
        return (int)(__float_as_uint(y) - 0x4B000000u);  // y - 2^23 (bit pattern of 2^23 is 0x4B000000)
    }
};

// ---------------------------------------------------------------------------
// Shape policy: D_, NB_ > 0 fix the dimension and the bins at compile time
// (all block offsets become constants); 0 means "read from the layout".
// With D_ = 0 the dimension is only known to lie in [DLO_, DMAX_]: loops run
// to DMAX_ and rows below DLO_ need no test (no branch in the unrolled loop).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int ceil_log2(int v) { return v <= 1 ? 0 : 1 + ceil_log2((v + 1) / 2); }
__host__ __device__ constexpr int round_up(int v, int m) { return (v + m - 1) / m * m; }

template <typename T>
__host__ __device__ constexpr BlkLayout make_layout_c(int d, int n)
{
    const int per16 = 16 / (int)sizeof(T);
    const int es = round_up(n + 1, per16), dn = round_up(n + 1, per16);
    // about four cells per bin: on adapted grids nearly every row then has
    // no cell overlapping more than two bins (the single-probe lookup)
    const int ls = ceil_log2(n) + 2;
    const int ts = round_up((1 << ls) + 2, 16);
    const int h = (int)sizeof(ChanHdr<T>);
    const int r = (es + dn) * (int)sizeof(T) + ts;
    return BlkLayout{h, es, dn, ts, r, ls, h + d * r};
}

template <typename T, int D_, int NB_, int DMAX_ = DMAX, int DLO_ = 1>
struct Shape {
    static constexpr bool kD = D_ > 0, kN = NB_ > 0;
    static constexpr int DM = kD ? D_ : DMAX_;  // unrolled loop bound
    static constexpr int DLO = kD ? D_ : DLO_;  // rows below this always exist
    static constexpr int NBC = NB_;              // compile-time bins (0: runtime)
    // pseudo-stratified passes run only in the fully generic shape (the
    // specialised kernels are compiled without that code)
    static constexpr bool kStrat = !kD && !kN && DMAX_ == DMAX && DLO_ == 1;
    static constexpr BlkLayout C = make_layout_c<T>(kD ? D_ : 1, kN ? NB_ : 1);
    const BlkLayout L;
    const int d_rt, n_rt;
    __device__ __forceinline__ Shape(const BlkLayout& l, int d, int n) : L(l), d_rt(d), n_rt(n) {}
    __device__ __forceinline__ int d() const { return kD ? D_ : d_rt; }
    __device__ __forceinline__ bool has(int k) const { return k < DLO || k < d(); }
    __device__ __forceinline__ int n() const { return kN ? NB_ : n_rt; }
    __device__ __forceinline__ int H() const { return kN ? C.H : L.H; }
    __device__ __forceinline__ int R() const { return kN ? C.R : L.R; }
    __device__ __forceinline__ int dens_off() const { return kN ? C.Es * (int)sizeof(T) : L.Es * (int)sizeof(T); }
    __device__ __forceinline__ int tab_off() const { return kN ? (C.Es + C.Dn) * (int)sizeof(T) : (L.Es + L.Dn) * (int)sizeof(T); }
    __device__ __forceinline__ int lshift() const { return kN ? C.lshift : L.lshift; }
    __device__ __forceinline__ int bytes() const { return kN && kD ? C.bytes : L.bytes; }
    __device__ __forceinline__ const unsigned char* row(const unsigned char* blk, int k) const
    {
        return blk + H() + k * R();
    }
};

// Slot of coordinate k among a channel's Breit-Wigner and power-law maps, -1
// if it has none.
__device__ __forceinline__ int map_slot(const ChanHdr<double>& h, int k)
{
    for (int s = 0; s < (int)h.nslot; ++s)
        if ((h.sk[s] & 15) == k) return s;
    return -1;
}

// Image φ(x) of a grid edge under slot s, by the forward map's formula.
__device__ __forceinline__ double edge_image(const ChanHdr<double>& h, int s, double x)
{
    if ((h.sk[s] >> 4) == MAP_BW) return h.c0[s] + h.fw[s][0] * Prec<double>::tan_(h.fw[s][1] * x - h.fw[s][2]);
    const double x2 = x * x, x4 = x2 * x2, v = x4 * x;
    return v < Prec<double>::tiny() ? Prec<double>::tiny() : v;
}

// Bin of x in a row whose cells overlap at most two bins: the cell's table
// entry, plus one if x reaches the next edge.
template <typename T, class SH>
__device__ __forceinline__ int lookup_fast(const SH& sh, const unsigned char* row, T x)
{
    const T* e = reinterpret_cast<const T*>(row);
    const int j = row[sh.tab_off() + Prec<T>::cell(x, sh.lshift())];
    return j + (Prec<T>::le(e[j + 1], x) ? 1 : 0);
}

// Largest j in [0, n-1] with e[j] <= x (the oracle's bin rule), starting at
// the table entry of x's cell.  A point at or past ξ_n = 1 may return n,
// whose density entry repeats bin n-1's.
template <typename T, class SH>
__device__ __forceinline__ int lookup(const SH& sh, const unsigned char* row, int span, T x)
{
    const T* e = reinterpret_cast<const T*>(row);
    const int q = Prec<T>::cell(x, sh.lshift());
    int j = row[sh.tab_off() + q];
    const int nm1 = sh.n() - 1;
    if (span <= 1) {
        j += Prec<T>::le(e[j + 1], x) ? 1 : 0;
    } else {
        for (int s = 1 << (31 - __clz(span)); s > 0; s >>= 1) {
            const int t = j + s;
            if (t <= nm1 && Prec<T>::le(e[t], x)) j = t;
        }
    }
    return j;
}

// Forward bin j and in-bin fraction of a stratified call from the integer t
// below n n_r 2^33: t = (j n_r + rest) 2^33 + low, fraction (rest 2^33 + low) /
// (n_r 2^33) to about 2^-53 by the integer reciprocal of n_r.  (64-bit integer
// and FP64 divisions here were a third of a d = 4 stratified pass.)
template <typename T>
__device__ __forceinline__ T strat_fraction(uint64_t t, uint32_t nr, Sf inv_nr, int& j)
{
    const uint32_t hi = (uint32_t)(t >> 33), q = hi / nr;  // below n n_r < 2^28
    j = (int)q;
    if (nr == 1u) return Prec<T>::frac(t & ((1ull << 33) - 1ull));
    const uint64_t rem = ((uint64_t)(hi - q * nr) << 33) | (t & ((1ull << 33) - 1ull));
    if (rem == 0ull) return T(0);
    const int z = __clzll((long long)rem);
    return (T)sf_to_double(sf_norm(sf_mul(Sf{rem << z, -z}, Sf{inv_nr.m, inv_nr.e - 33})));
}

// ---------------------------------------------------------------------------
// Forward map of the selected channel (lookup block in global memory):
// r -> x_c -> p, the own term g_c(x_c)/φ'_c(x_c) and the Gaussian exponent
// sum of p (log2 units).  FP32; the FP64 form is soft_forward.
// ---------------------------------------------------------------------------
template <typename T, class SH>
__device__ __forceinline__ void forward_call(const Params& P, const SH& sh, int c, const uint32_t* X,
                                             T (&x)[SH::DM], T (&p)[SH::DM], int (&jf)[SH::DM], T& own_gJ,
                                             T& asum_all, const uint32_t* dig = nullptr, uint32_t nr = 1u)
{
    const int d = sh.d(), n = sh.n();
    const unsigned char* blk = Prec<T>::lk(P) + (size_t)c * sh.bytes();
    const Sf inv_nr = dig ? sf_rcp(sf_from_double((double)nr)) : Sf{0, 0};
    T g = T(1);
#pragma unroll
    for (int k = 0; k < SH::DM; ++k) {
        if (sh.has(k)) {
            int j;
            T fr;
            if (dig) {
                // stratified call: r_k = (a_k + u_k) / n_r, from the integer
                // (2^33 a_k + 2X + 1) n over n_r 2^33 (n_r = 1: the line below)
                const uint64_t t = (((uint64_t)dig[k] << 33) + 2ull * X[k] + 1ull) * (uint64_t)n;
                fr = strat_fraction<T>(t, nr, inv_nr, j);
            } else {
                const uint64_t t = (2ull * X[k] + 1ull) * (uint64_t)n;
                j = (int)(t >> 33);
                fr = Prec<T>::frac(t & ((1ull << 33) - 1ull));
            }
            const unsigned char* row = sh.row(blk, k);
            const T* e = reinterpret_cast<const T*>(row);
            x[k] = Prec<T>::lerp(__ldg(e + j), __ldg(e + j + 1), fr);
            jf[k] = j;
            g *= __ldg(reinterpret_cast<const T*>(row + sh.dens_off()) + j);
        } else {
            x[k] = T(0);
            jf[k] = 0;
        }
    }
    const ChanHdr<T>* h = reinterpret_cast<const ChanHdr<T>*>(blk);
    const uint32_t mask = __ldg(&h->mask), kinds = __ldg(&h->kinds);
    const uint64_t slotpack = __ldg(&h->slotpack);
    T J = T(1), A = T(0);
    const T gc = Prec<T>::gcen(P), k2 = Prec<T>::gk2(P);
#pragma unroll
    for (int k = 0; k < SH::DM; ++k) {
        p[k] = x[k];
        if (sh.has(k)) {
            if ((mask >> k) & 1u) {
                const int s = (int)((slotpack >> (4 * k)) & 0xFu);
                const int kind = (kinds >> (8 * s)) & 0xff;
                const T* sp = h->sp[s];
                if (kind == MAP_BW) {
                    const T mass = __ldg(sp + SP_M), G = __ldg(sp + SP_G), A_ = __ldg(sp + SP_A);
                    p[k] = mass + G * Prec<T>::tan_(A_ * x[k] - __ldg(sp + SP_T0));
                    const T dp = p[k] - mass;
                    J *= Prec<T>::div(__ldg(sp + SP_GINVA), dp * dp + __ldg(sp + SP_G2));
                } else if (kind == MAP_POW) {
                    const T x2 = x[k] * x[k], x4 = x2 * x2;
                    T pk = x4 * x[k];
                    if (pk < Prec<T>::tiny()) pk = Prec<T>::tiny();
                    p[k] = pk;
                    J *= Prec<T>::div(T(1), T(5) * x4);
                }
            }
            const T u = p[k] - gc;
            A += u * u * k2;
        }
    }
    own_gJ = g * J;
    asum_all = A;
}

// ---------------------------------------------------------------------------
// One channel c' (block in shared or global memory) against CPT calls: the
// inner loop of Eq. 30, fused with the matching integrand peak when with_f:
//   g_q += α_c' g_c'(φ_c'^{-1}(p_q)) / φ'_c'   (lookups and not skip_q)
//   f_q += wz_c' 2^-(A_q - Σ_mapped a_k) Π_mapped factor(p_k)
// REC records the bin indices of call 0 into bins[0..d-1].
// ---------------------------------------------------------------------------
// Rows of one channel against CPT calls: bin densities (gp), Jacobians of the
// mapped coordinates (J), matching-peak factors (F) and Gaussian exponents of
// the mapped coordinates (as).  FAST: every row's cells overlap at most two
// bins, so one edge probe settles each bin and the unrolled row loop has no
// branch other than the mapped-coordinate test; otherwise rows are tested
// one by one and only the spanning ones search.
// (FP32; the FP64 form is soft_channel below.)
template <typename T, int CPT, bool REC, bool FAST, class SH>
__device__ __forceinline__ void channel_rows(const Params& P, const SH& sh, const unsigned char* blk, bool with_f,
                                             const T (&p)[CPT][SH::DM], T (&J)[CPT], T (&F)[CPT], T (&gp)[CPT],
                                             T (&as)[CPT], int* bins)
{
    const int d = sh.d();
    const ChanHdr<T>& h = *reinterpret_cast<const ChanHdr<T>*>(blk);
    const uint32_t mask = h.mask, kinds = h.kinds, slow = h.slow;
    const uint64_t slotpack = h.slotpack;
    const T gc = Prec<T>::gcen(P), k2 = Prec<T>::gk2(P);
#pragma unroll
    for (int k = 0; k < SH::DM; ++k) {
        if (sh.has(k)) {
            T xk[CPT];
#pragma unroll
            for (int q = 0; q < CPT; ++q) xk[q] = p[q][k];
            if ((mask >> k) & 1u) {
                const int s = (int)((slotpack >> (4 * k)) & 0xFu);
                const int kind = (kinds >> (8 * s)) & 0xff;
                const T* sp = h.sp[s];
                if (kind == MAP_BW) {
                    const T mass = sp[SP_M], G2 = sp[SP_G2], invG = sp[SP_INVG], GinvA = sp[SP_GINVA],
                            invA = sp[SP_INVA], t0 = sp[SP_T0];
#pragma unroll
                    for (int q = 0; q < CPT; ++q) {
                        const T dp = p[q][k] - mass;
                        const T jfac = Prec<T>::div(GinvA, dp * dp + G2);
                        J[q] *= jfac;
                        F[q] *= jfac;
                        xk[q] = (Prec<T>::atan_(dp * invG) + t0) * invA;
                        const T u = p[q][k] - gc;
                        as[q] += u * u * k2;
                    }
                } else if (kind == MAP_POW) {
                    const T del = sp[SP_DEL], ipn = sp[SP_INVPOWN];
#pragma unroll
                    for (int q = 0; q < CPT; ++q) {
                        const T xx = Prec<T>::pow02(p[q][k]);
                        const T x2 = xx * xx;
                        J[q] *= Prec<T>::div(T(1), T(5) * (x2 * x2));
                        xk[q] = xx;
                        if (with_f) F[q] *= Prec<T>::powm08(p[q][k] + del) * ipn;
                        const T u = p[q][k] - gc;
                        as[q] += u * u * k2;
                    }
                }
            }
            // every channel's rows are probed; the terms of the own channel
            // and of switched-off channels are dropped by the caller
            const unsigned char* row = sh.row(blk, k);
            const T* dn = reinterpret_cast<const T*>(row + sh.dens_off());
            if (FAST) {
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
                    const int j = lookup_fast<T>(sh, row, xk[q]);
                    if (REC && q == 0) bins[k] = min(j, sh.n() - 1);
                    gp[q] *= dn[j];
                }
            } else if (!((slow >> k) & 1u)) {
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
                    const int j = lookup_fast<T>(sh, row, xk[q]);
                    if (REC && q == 0) bins[k] = min(j, sh.n() - 1);
                    gp[q] *= dn[j];
                }
            } else {
                const int sp = row[sh.tab_off() + (1 << sh.lshift()) + 1];
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
                    const int j = lookup<T>(sh, row, sp, xk[q]);
                    if (REC && q == 0) bins[k] = min(j, sh.n() - 1);
                    gp[q] *= dn[j];
                }
            }
        }
    }
}

template <typename T, int CPT, bool REC, class SH>
__device__ __forceinline__ void channel_body(const Params& P, const SH& sh, const unsigned char* blk, T alpha_c,
                                             bool lookups, bool with_f, const T (&p)[CPT][SH::DM],
                                             const T (&A)[CPT], const bool (&skip)[CPT], T (&g)[CPT],
                                             T (&f)[CPT], int* bins)
{
    const ChanHdr<T>& h = *reinterpret_cast<const ChanHdr<T>*>(blk);
    T J[CPT], F[CPT], gp[CPT], as[CPT];
#pragma unroll
    for (int q = 0; q < CPT; ++q) { J[q] = T(1); F[q] = T(1); gp[q] = T(1); as[q] = T(0); }
    if (h.slow == 0u) channel_rows<T, CPT, REC, true>(P, sh, blk, with_f, p, J, F, gp, as, bins);
    else channel_rows<T, CPT, REC, false>(P, sh, blk, with_f, p, J, F, gp, as, bins);
    const T wz = h.wz;
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        if (lookups && !skip[q]) g[q] += alpha_c * gp[q] * J[q];
        if (with_f) f[q] += wz * Prec<T>::exp2_(as[q] - A[q]) * F[q];
    }
}

// ---------------------------------------------------------------------------
// The FP64 form of the channel loop, on the integer pipe (vamp_soft64.cuh).
// Same terms as channel_body: g += α_c g_c(φ_c^{-1}(p)) / φ'_c, f += the
// matching peak.  What bounded it before: the FP64 pipe, 76 % busy with about
// 5 200 operations a call on the collider (d = 14, K = 64), 134 ms per 1e7
// calls.  Here the FP64 pipe keeps, per channel, p - m and (p - m)² + Γ² of
// each Breit-Wigner slot, p + δ of each power-law slot and the two sums.
// ---------------------------------------------------------------------------
// Per call, for all channels: the cell of p_k in an unmapped row's table (the
// same for every channel), and for coordinates that some channel maps the
// Gaussian factor 2^(a_k) that its peak must not have (its exponent a_k, where
// P.gauss_sum is set) and p_k^(-4/5).  The arrays that the slots index by coordinate live in local memory (coalesced
// there, and read at most 4 times a channel).
template <int DM>
struct SoftCall {
    int q[DM];
    double p[DM];
    uint64_t E[DM], W[DM];
    Sf e0;     // 2^-(Σ a_k), the Gaussian factors of all coordinates (1 where P.gauss_sum)
    double A;  // Σ a_k
};

// One packed factor onto acc; the exponents' biases are added by the caller.
__device__ __forceinline__ void soft_factor(uint64_t& acc, int& ae, uint64_t w)
{
    acc = sf_mulhi(acc, w & ~2047ull);
    ae += (int)((uint32_t)w & 2047u);
}

// Forward map of a call of channel c (lookup block and master grid in global
// memory) and what the channel loop needs of it: p, the forward bins jf, the
// own term g_c/φ'_c without the constant gN, and S.  An FP64 operation stands
// only where a coordinate's value is formed: the fraction, the edges'
// interpolation, (p - centre)² and the map's ends; the tangent, the densities
// and the own Jacobian (its denominators, and the p^(-4/5) that the channels
// share) are on the integer pipe.  With FP64 throughout, a d = 8 call of six
// channels kept the FP64 pipe busy for 250 operations, half of them here, and
// the pass (1e6 calls) took 482 us.
// digit (stratified calls, else null): the cell's base-n_r digits.  x_out (may
// be null) receives x.
template <class SH>
__device__ __forceinline__ void soft_forward(const Params& P, const SH& sh, int c, const uint32_t* X,
                                             double (&p)[SH::DM], int (&jf)[SH::DM], double& own,
                                             SoftCall<SH::DM>& S, const uint32_t* digit = nullptr, uint32_t nr = 1u,
                                             double* x_out = nullptr)
{
    const int d = sh.d(), n = sh.n();
    const unsigned char* blk = P.lk64 + (size_t)c * sh.bytes();
    const ChanHdr<double>* h = reinterpret_cast<const ChanHdr<double>*>(blk);
    const double* e0 = P.edges64 + (size_t)c * d * (size_t)(n + 1);
    const Sf inv_nr = digit ? sf_rcp(sf_from_double((double)nr)) : Sf{0, 0};
    uint64_t acc = 1ull << 63;
    int ae = 0;  // acc 2^(ae - 1022 d - 63)
#pragma unroll
    for (int k = 0; k < SH::DM; ++k) {
        jf[k] = 0;
        if (sh.has(k)) {
            double fr;
            if (digit) {
                // stratified call: r_k = (a_k + u_k) / n_r, from the integer
                // (2^33 a_k + 2X + 1) n over n_r 2^33 (n_r = 1: the line below)
                const uint64_t t = (((uint64_t)digit[k] << 33) + 2ull * X[k] + 1ull) * (uint64_t)n;
                fr = strat_fraction<double>(t, nr, inv_nr, jf[k]);
            } else {
                const uint64_t t = (2ull * X[k] + 1ull) * (uint64_t)n;
                jf[k] = (int)(t >> 33);
                fr = sf_frac33(t & ((1ull << 33) - 1ull));
            }
            const double* e = e0 + (size_t)k * (n + 1) + jf[k];
            S.p[k] = Prec<double>::lerp(__ldg(e), __ldg(e + 1), fr);
            if (x_out) x_out[k] = S.p[k];
            soft_factor(acc, ae, __ldg(reinterpret_cast<const unsigned long long*>(sh.row(blk, k) + sh.dens_off()) + jf[k]));
        }
        if (k % 8 == 7 || k == SH::DM - 1) sf_norm(acc, ae);
    }
    const Sf one{1ull << 63, -63};
    Sf den{1ull << 63, -63 - __ldg(&h->ge)}, G = one;
    const int ns = (int)__ldg(&h->nslot);
#pragma unroll 1
    for (int s = 0; s < ns; ++s) {
        const int w = __ldg(&h->sk[s]), k = w & 15;
        const double x = S.p[k];
        if ((w >> 4) == MAP_BW) {
            const double* sp = h->fw[s];
            const double t = __ldg(sp) * Prec<double>::tan_(__ldg(sp + 1) * x - __ldg(sp + 2));  // p - m, before p is rounded
            const double pk = __ldg(&h->c0[s]) + t, dp = pk - __ldg(&h->c0[s]);
            den = sf_mul(den, sf_from_any(dp * dp + __ldg(&h->c1[s])));
            S.p[k] = pk;
        } else {
            const double x2 = x * x, x4 = x2 * x2;
            double pk = x4 * x;
            if (pk < Prec<double>::tiny()) pk = Prec<double>::tiny();
            G = sf_mul(G, sf_rcp(sf_from_any(x4)));  // (p^(-4/5) from x: p may have been floored)
            S.p[k] = pk;
        }
    }
    const Sf y = sf_rcp(sf_norm(den));
    own = sf_to_double(sf_norm(sf_mul(sf_mul(Sf{acc, ae - 1022 * d - 63}, sf_norm(G)), y)));
    // Gaussian exponents, cells, and the factors of the coordinates that some
    // channel maps
    const double gc = P.gcen, k2 = P.gk2;
    double A = 0.0;
#pragma unroll
    for (int k = 0; k < SH::DM; ++k) {
        p[k] = 0.0;
        if (sh.has(k)) {
            p[k] = S.p[k];
            S.q[k] = Prec<double>::cell(p[k], sh.lshift());
            const double u = p[k] - gc, u2 = u * u;
            A += u2;
            if ((P.map_any >> k) & 1u) S.E[k] = sf_bits(u2);
        }
    }
    A *= k2;
    for (uint32_t m = P.map_any; m; m &= m - 1u) {
        const int k = __ffs(m) - 1;
        if (P.matching) {
            const double a = sf_from_bits(S.E[k]) * k2;
            S.E[k] = P.gauss_sum ? sf_bits(a) : sf_pack(sf_exp2(a));
        }
        if ((P.pow_any >> k) & 1u) S.W[k] = sf_pack(sf_powm08(S.p[k]));
    }
    S.A = A;
    S.e0 = P.matching && !P.gauss_sum ? sf_exp2(-A) : one;
}

// Largest j' in [j, n] with e[j'] <= x, for e[j] <= x: three edges at a time,
// since a search from the right cell seldom goes further.  (Doubling steps
// after the first three cost 2 to 4 % of every pass, collider 52.9 -> 54.0 ms, for 4 %
// of a pass over rows with 52 edges in a cell.)
__device__ __forceinline__ int soft_search(const double* e, int j, int n, double x)
{
    for (;;) {
        const int a = Prec<double>::le(e[min(j + 1, n)], x) ? 1 : 0, b = Prec<double>::le(e[min(j + 2, n)], x) ? 1 : 0,
                  c = Prec<double>::le(e[min(j + 3, n)], x) ? 1 : 0;
        j += a + b + c;
        if (!c || j >= n) return min(j, n);
    }
}

// atan t within 1.7e-6: the least-squares odd polynomial of degree 11 on
// [0, 1], with atan t = pi/2 - atan(1/t) above.  A starting point of searches.
__device__ __forceinline__ float atan_start(float t)
{
    const float a = fabsf(t), u = a > 1.f ? sf_rcpf(a) : a, v = u * u;
    float y = fmaf(v, -0.011719031f, 0.052647073f);
    y = fmaf(y, v, -0.116426215f);
    y = fmaf(y, v, 0.19354026f);
    y = fmaf(y, v, -0.3326228f);
    y = fmaf(y, v, 0.99997723f) * u;
    y = a > 1.f ? 1.57079633f - y : y;
    return copysignf(y, t);
}

// Product of a channel's Breit-Wigner denominators for widths far from 1 (they
// need not be normal numbers), divided by 2^ge.  In a loop of its own: tests
// and powers of two in the loop over all slots took 0.6 of the collider's 53 ms.
__device__ __forceinline__ Sf far_denominators(const ChanHdr<double>& h, const double* p)
{
    Sf den{1ull << 63, -63 - h.ge};
#pragma unroll 1
    for (uint32_t s = 0; s < h.nslot; ++s) {
        if ((h.sk[s] >> 4) != MAP_BW) continue;
        const double dp = p[h.sk[s] & 15] - h.c0[s];
        den = sf_mul(den, sf_from_any(dp * dp + h.c1[s]));
    }
    return den;
}

// Channel c' (block in shared or global memory) against one call: its term of
// g(p) without the constant α gN, and of f without fN.  bins (REC): the bin of
// every row.  At most eight factors follow one another without normalising
// (each loses at most one of the 64 bits).
template <bool REC, class SH>
__device__ __forceinline__ void soft_channel(const Params& P, const SH& sh, const unsigned char* blk, bool lookups,
                                             const double (&p)[SH::DM], const SoftCall<SH::DM>& S, double& gt,
                                             double& ft, int* bins)
{
    const bool with_f = P.matching != 0, gauss_sum = P.gauss_sum != 0;
    const ChanHdr<double>& h = *reinterpret_cast<const ChanHdr<double>*>(blk);
    const uint32_t mmask = h.mmask;
    const int n = sh.n();
    uint64_t acc = 1ull << 63;
    int ae = 0;  // acc 2^(ae - 1022 d - 63) once every row is in
    if (lookups) {
        const uint32_t slow = h.slow;
#pragma unroll
        for (int k = 0; k < SH::DM; ++k) {
            if (sh.has(k) && !((mmask >> k) & 1u)) {
                const unsigned char* row = sh.row(blk, k);
                const double* e = reinterpret_cast<const double*>(row);
                int j = row[sh.tab_off() + S.q[k]];
                j += Prec<double>::le(e[j + 1], p[k]) ? 1 : 0;
                if ((slow >> k) & 1u) j = soft_search(e, j, n, p[k]);  // a cell of more than two bins
                if (REC) bins[k] = min(j, n - 1);  // (entry n of the densities repeats the last)
                soft_factor(acc, ae, reinterpret_cast<const uint64_t*>(row + sh.dens_off())[j]);
            }
            if (k % 8 == 7 || k == SH::DM - 1) sf_norm(acc, ae);
        }
    }
    // den: Breit-Wigner denominators; G: p^(-4/5); F: the peak's factors
    const Sf one{1ull << 63, -63};
    Sf den = one, G = one, F = S.e0;
    double as = 0.0;
#pragma unroll 1
    for (uint32_t s = 0; s < h.nslot; ++s) {
        const int k = h.sk[s] & 15;
        const double pk = S.p[k];
        float xc;  // cell of the FP32 inverse map
        if ((h.sk[s] >> 4) == MAP_BW) {
            const double dp = pk - h.c0[s];
            den = sf_mul(den, sf_from_double(dp * dp + h.c1[s]));
            xc = (atan_start(sf_to_float(dp) * h.pinvG[s]) + h.pt0[s]) * h.pscale[s];
        } else {
            if (with_f) F = sf_mul(F, sf_powm08(pk + h.c0[s]));
            G = sf_mul(G, sf_unpack(S.W[k]));
            const uint64_t b = sf_bits(pk);
            const float lg = sf_lg2f((float)(((uint32_t)(b >> 29) & 0x7fffffu) | 0x800000u)) + (float)((int)((int64_t)b >> 52) - 1046);
            xc = sf_ex2f(0.2f * lg) * h.pscale[s];  // (p < 0, by rounding at a map's lower end, gives cell 0)
        }
        if (with_f) {
            if (gauss_sum) as += sf_from_bits(S.E[k]);
            else F = sf_mul(F, sf_unpack(S.E[k]));
        }
        if (lookups) {
            const unsigned char* row = sh.row(blk, k);
            const double* e = reinterpret_cast<const double*>(row);
            const int L = 1 << sh.lshift();
            int j = row[sh.tab_off() + min(max((int)(xc - 0.02f), 0), L)];
            j = soft_search(e, j, n, pk);
            if (REC) bins[k] = min(j, n - 1);
            soft_factor(acc, ae, reinterpret_cast<const uint64_t*>(row + sh.dens_off())[j]);
        }
    }
    Sf y = one;
    if (h.bw) {
        if (h.bw > 1u) den = far_denominators(h, S.p);
        y = sf_rcp(sf_norm(den));
    }
    if (with_f && gauss_sum) F = sf_mul(sf_norm(F), sf_exp2(as - S.A));
    gt = ft = 0.0;
    if (lookups) {
        sf_norm(acc, ae);
        gt = sf_to_double(sf_norm(sf_mul(sf_mul(Sf{acc, ae - 1022 * sh.d() - 63}, G), y)));
    }
    if (with_f) ft = sf_to_double(sf_norm(sf_mul(sf_norm(F), y)));
}

// Integrand of a non-matching problem: loop over its own peaks.
template <typename T, int DM>
__device__ __forceinline__ T integrand_peaks(const Params& P, int d, const T (&p)[DM], T A)
{
    const MapRec<T>* pks = Prec<T>::pk(P);
    const T gc = Prec<T>::gcen(P), k2 = Prec<T>::gk2(P);
    T f = T(0);
    for (int q = 0; q < P.P; ++q) {
        const MapRec<T>& r = pks[q];
        const uint32_t mask = r.mask;
        T v = T(1), as = T(0);
#pragma unroll
        for (int k = 0; k < DM; ++k) {
            if (k < d && ((mask >> k) & 1u)) {
                const int s = (int)((r.slotpack >> (4 * k)) & 0xFu);
                if (r.kind[s] == MAP_BW) {
                    const T dp = p[k] - r.m[s];
                    v *= r.GinvA[s] / (dp * dp + r.G[s] * r.G[s]);
                } else if (r.kind[s] == MAP_POW) {
                    v *= Prec<T>::powm08(p[k] + r.del[s]) * r.invPowN[s];
                }
                const T u = p[k] - gc;
                as += u * u * k2;
            }
        }
        f += r.wz * Prec<T>::exp2_(as - A) * v;
    }
    return f;
}

// Channel of a generation call: min{c : u A_K < A_c} on the cumulative α.
__device__ __forceinline__ int choose_channel(const Params& P, double u)
{
    const double tgt = u * P.Acum[P.K - 1];
    int lo = 0, hi = P.K - 1; // first c with tgt < A_c
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (tgt < P.Acum[mid]) hi = mid; else lo = mid + 1;
    }
    if (!(tgt < P.Acum[lo])) { // rounding: last live channel
        for (int c = P.K - 1; c >= 0; --c)
            if (P.alpha[c] > 0.0) return c;
    }
    return lo;
}

__device__ __forceinline__ int find_channel(const int64_t* Pc, int K, int64_t i)
{
    int lo = 0, hi = K - 1; // largest c with Pc[c] <= i
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (Pc[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// Bulk-copy staging (cp.async.bulk + mbarrier), with bounded waits.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// One thread: expect `bytes` on bar and start the copy global -> shared.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits for phase `parity` of bar; gives up after `limit` SM cycles (by
// default 2^31, about a second) and returns false, so that no wait can hang
// the GPU.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long limit = 1ll << 31)
{
    if (mbar_test(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_test(bar, parity)) {
        if (clock64() - t0 > limit) return false;
    }
    return true;
}

}  // namespace vamp
