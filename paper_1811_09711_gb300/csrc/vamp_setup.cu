// vamp_setup.cu -- host-side setup shared by vamp_create and the
// allocation-free entry point: validation of a vamp_config, derived
// constants of the maps and the Gaussian factor, lookup-block layout and
// headers, placement of the per-problem arrays, pass-kernel variants.
#include "vamp_device.cuh"
#include "vamp_internal.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

namespace vamp {

namespace {

bool check_maps(const vamp_map_desc* m, int cnt, int d, std::string& why)
{
    for (int q = 0; q < cnt; ++q) {
        const vamp_map_desc& r = m[q];
        if (r.n_mapped < 0 || r.n_mapped > MAXMAP) { why = "n_mapped out of range"; return false; }
        unsigned seen = 0;
        for (int s = 0; s < r.n_mapped; ++s) {
            const int k = r.coord[s];
            if (k < 0 || k >= d) { why = "mapped coordinate out of range"; return false; }
            if (seen & (1u << k)) { why = "coordinate mapped twice"; return false; }
            seen |= 1u << k;
            if (r.kind[s] == VAMP_MAP_BW) {
                if (!(r.b[s] > 0.0) || !std::isfinite(r.a[s]) || !std::isfinite(r.b[s])) {
                    why = "Breit-Wigner width must be > 0";
                    return false;
                }
            } else if (r.kind[s] == VAMP_MAP_POW) {
                if (!(r.b[s] >= 0.0) || !std::isfinite(r.b[s])) { why = "power-law delta must be >= 0"; return false; }
            } else if (r.kind[s] != VAMP_MAP_ID) {
                why = "unknown map kind";
                return false;
            }
        }
    }
    return true;
}

bool same_maps(const vamp_map_desc& a, const vamp_map_desc& b)
{
    if (a.n_mapped != b.n_mapped) return false;
    for (int s = 0; s < a.n_mapped; ++s)
        if (a.coord[s] != b.coord[s] || a.kind[s] != b.kind[s] || a.a[s] != b.a[s] || a.b[s] != b.b[s])
            return false;
    return true;
}

// Breit-Wigner constants: A = ∫_0^1 Γ/((p-m)²+Γ²) dp, t0 = atan(m/Γ);
// power law: 1 / ∫_0^1 (p+δ)^-0.8 dp.
double bw_A(double m, double G) { return std::atan((1.0 - m) / G) + std::atan(m / G); }
double pow_invN(double del) { return 1.0 / (5.0 * (std::pow(1.0 + del, 0.2) - std::pow(del, 0.2))); }

template <typename T>
MapRec<T> make_rec(const vamp_map_desc& r, double weight, double zinv, int d)
{
    MapRec<T> o;
    std::memset(&o, 0, sizeof o);
    o.nmap = r.n_mapped;
    o.wz = (T)(weight * std::pow(zinv, (double)(d - r.n_mapped)));
    for (int s = 0; s < r.n_mapped; ++s) {
        const int k = r.coord[s];
        o.mask |= 1u << k;
        o.slotpack |= (uint64_t)s << (4 * k);
        o.kind[s] = r.kind[s];
        if (r.kind[s] == VAMP_MAP_BW) {
            const double m = r.a[s], G = r.b[s], A = bw_A(m, G);
            o.m[s] = (T)m;
            o.G[s] = (T)G;
            o.invG[s] = (T)(1.0 / G);
            o.A[s] = (T)A;
            o.GinvA[s] = (T)(G / A);
            o.invA[s] = (T)(1.0 / A);
            o.t0[s] = (T)std::atan(m / G);
        } else if (r.kind[s] == VAMP_MAP_POW) {
            o.del[s] = (T)r.b[s];
            o.invPowN[s] = (T)pow_invN(r.b[s]);
        }
    }
    return o;
}

void make_hdr32(const vamp_map_desc& r, double weight, double zinv, int d, unsigned char* out)
{
    ChanHdr<float> h;
    std::memset(&h, 0, sizeof h);
    h.wz = (float)(weight * std::pow(zinv, (double)(d - r.n_mapped)));
    for (int s = 0; s < r.n_mapped; ++s) {
        const int k = r.coord[s];
        h.mask |= 1u << k;
        h.slotpack |= (uint64_t)s << (4 * k);
        h.kinds |= (uint32_t)(r.kind[s] & 0xff) << (8 * s);
        float* sp = h.sp[s];
        if (r.kind[s] == VAMP_MAP_BW) {
            const double m = r.a[s], G = r.b[s], A = bw_A(m, G);
            sp[SP_M] = (float)m;
            sp[SP_G] = (float)G;
            sp[SP_A] = (float)A;
            sp[SP_G2] = (float)(G * G);
            sp[SP_INVG] = (float)(1.0 / G);
            sp[SP_GINVA] = (float)(G / A);
            sp[SP_INVA] = (float)(1.0 / A);
            sp[SP_T0] = (float)std::atan(m / G);
        } else if (r.kind[s] == VAMP_MAP_POW) {
            sp[SP_DEL] = (float)r.b[s];
            sp[SP_INVPOWN] = (float)pow_invN(r.b[s]);
        }
    }
    std::memcpy(out, &h, sizeof h);
}

// m 2^e times v, with |m| in [1/2, 1) (m alone where the product is 0 or not finite).
void scale_by(double& m, int32_t& e, double v)
{
    int q = 0;
    m *= std::isfinite(v) ? std::frexp(v, &q) : v;
    e += q;
    if (!std::isfinite(m) || m == 0.0) return;
    m = std::frexp(m, &q);
    e += q;
}

// The slots with a factor, and the constants of the channel's terms (SoftCall).
void make_hdr64(const vamp_map_desc& r, double weight, double zinv, int d, int lshift, unsigned char* out)
{
    ChanHdr<double> h;
    std::memset(&h, 0, sizeof h);
    int32_t ge = 0, fe = 0, far = 0;
    h.gN = h.fN = 1.0;
    scale_by(h.fN, fe, weight * std::pow(zinv, (double)(d - r.n_mapped)));
    for (int s = 0; s < r.n_mapped; ++s) {
        const int kind = r.kind[s], q = (int)h.nslot;
        if (kind != MAP_BW && kind != MAP_POW) continue;
        h.mmask |= 1u << r.coord[s];
        h.sk[q] = (uint8_t)(r.coord[s] | kind << 4);
        // cells of the row's table per unit of the FP32 inverse map.  A search
        // starts 0.02 cells before it, more than its error (2.2e-6 of the
        // angle, and 2.4e-5 of a small one) above A = 0.3; below, that error is
        // taken off as well (d = 8, n = 256, two wide or outlying maps a
        // channel, 1e6 calls: 553 us; from bin 0 on 1 640)
        const double cells = (double)(1 << lshift);
        if (kind == MAP_BW) {
            const double m = r.a[s], G = r.b[s], A = bw_A(m, G), t0 = std::atan(m / G);
            h.bw = 1;
            far += std::abs(std::ilogb(G));
            h.c0[q] = m;
            h.c1[q] = G * G;
            h.fw[q][0] = G;
            h.fw[q][1] = A;
            h.fw[q][2] = t0;
            scale_by(h.gN, ge, G / A);
            scale_by(h.fN, fe, G / A);
            h.pinvG[q] = (float)(1.0 / G);
            const double tmax = std::max(std::fabs(m), std::fabs(1.0 - m)) / G;
            h.pt0[q] = (float)(A > 0.3 ? t0 : t0 - std::min(2.5e-6, 3e-5 * tmax));
            h.pscale[q] = (float)(cells / A);
        } else {
            h.c0[q] = r.b[s];
            scale_by(h.gN, ge, 0.2);
            scale_by(h.fN, fe, pow_invN(r.b[s]));
            h.pscale[q] = (float)cells;
        }
        ++h.nslot;
    }
    // without these constants the terms of g(p) and f reach 2^far further than
    // with them; beyond 2^511 a Γ² is no normal number
    if (far > 100) {
        h.bw = 2;
        h.ge = ge;
        h.fN = std::ldexp(h.fN, fe - ge);
    } else {
        h.gN = std::ldexp(h.gN, ge);
        h.fN = std::ldexp(h.fN, fe);
    }
    std::memcpy(out, &h, sizeof h);
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

}  // namespace

bool build_setup(const vamp_config* cfg, Params& pr, Setup& S, std::string& why)
{
    if (!cfg) { why = "cfg is NULL"; return false; }
    const int d = cfg->d, K = cfg->n_channels, n = cfg->n_bins, P = cfg->n_peaks;
    if (d < 1 || d > DMAX) { why = "d must be in 1..16"; return false; }
    if (K < 1 || P < 1) { why = "need at least one channel and one peak"; return false; }
    if (n < 1 || n > MAX_BINS) { why = "n_bins must be in 1..256"; return false; }
    if (!cfg->channels || !cfg->peaks || !cfg->peak_weight) { why = "descriptor pointers are NULL"; return false; }
    if (!check_maps(cfg->channels, K, d, why) || !check_maps(cfg->peaks, P, d, why)) return false;
    if (!(cfg->gauss_sigma >= 0.0) || !std::isfinite(cfg->gauss_sigma)) { why = "gauss_sigma must be >= 0"; return false; }
    if (!(cfg->grid_alpha > 0.0) || !std::isfinite(cfg->beta)) { why = "grid_alpha must be > 0"; return false; }
    if (cfg->n_min < 1 || cfg->n_min > int64_t(0xffffffff)) { why = "n_min must be in 1..2^32-1"; return false; }
    if (cfg->gen_batch < 0 || cfg->gen_batch > (int64_t(1) << 24)) { why = "gen_batch out of range"; return false; }
    if (cfg->precision != VAMP_PREC_FP64 && cfg->precision != VAMP_PREC_FP32_EVAL) { why = "bad precision"; return false; }
    if (cfg->stratified != 0 && cfg->stratified != 1) { why = "stratified must be 0 or 1"; return false; }
    if (cfg->n_equiv < 0 || cfg->n_equiv > 65536 || (cfg->n_equiv > 0 && !cfg->equiv)) {
        why = "n_equiv must be in 0..65536 with a table"; return false;
    }
    if (cfg->n_equiv > 0 && (int64_t)K * d >= (int64_t(1) << 28)) { why = "too many grid rows for equivalences"; return false; }
    for (int e = 0; e < cfg->n_equiv; ++e) {
        const int32_t* r = cfg->equiv + (size_t)e * (2 + 2 * d);
        if (r[0] < 0 || r[0] >= K || r[1] < 0 || r[1] >= K) { why = "equivalence names a channel out of range"; return false; }
        unsigned seen = 0;
        for (int k = 0; k < d; ++k) {
            if (r[2 + k] < 0 || r[2 + k] >= d || (seen >> r[2 + k] & 1u)) {
                why = "equivalence axes must be a permutation of 0..d-1"; return false;
            }
            seen |= 1u << r[2 + k];
            if (r[2 + d + k] < VAMP_EQ_IDENTITY || r[2 + d + k] > VAMP_EQ_INVARIANT) {
                why = "equivalence kind must be 0..3"; return false;
            }
        }
    }
    for (int q = 0; q < P; ++q)
        if (!std::isfinite(cfg->peak_weight[q])) { why = "peak weights must be finite"; return false; }

    S.d = d; S.K = K; S.n = n; S.P = P;
    S.fp32 = cfg->precision == VAMP_PREC_FP32_EVAL;
    pr.d = d; pr.K = K; pr.n = n; pr.P = P;
    pr.fp32 = S.fp32;
    pr.key0 = (uint32_t)(cfg->seed & 0xffffffffu);
    pr.key1 = (uint32_t)(cfg->seed >> 32);
    pr.request = cfg->request_id;
    pr.n_min = cfg->n_min;
    pr.grid_alpha = cfg->grid_alpha;
    pr.beta = cfg->beta;
    pr.smooth = cfg->smooth;
    pr.omega_mode = cfg->omega_mode;
    pr.stratified = cfg->stratified;
    // equivalences regrouped by target grid row, list order kept (§3.5)
    S.eq_off.assign(cfg->n_equiv > 0 ? (size_t)K * d + 1 : 0, 0);
    S.eq_ent.clear();
    if (cfg->n_equiv > 0) {
        for (int row = 0; row < K * d; ++row) {
            const int c = row / d, k = row % d;
            S.eq_off[row] = (int32_t)S.eq_ent.size();
            for (int e = 0; e < cfg->n_equiv; ++e) {
                const int32_t* r = cfg->equiv + (size_t)e * (2 + 2 * d);
                if (r[0] == c) S.eq_ent.push_back(((r[1] * d + r[2 + k]) << 2) | r[2 + d + k]);
            }
        }
        S.eq_off[(size_t)K * d] = (int32_t)S.eq_ent.size();
    }
    pr.n_eq_ent = (int)S.eq_ent.size();
    // Gaussian factor exp(-(p-c)²/(2σ²)) / Z written as 2^-((p-c)² gk2) / Z,
    // gk2 = log2(e) / (2σ²); σ = 0 switches it off (factor 1)
    S.zinv = 1.0;
    pr.gcen = 0.0; pr.gk2 = 0.0; pr.gcen_f = 0.f; pr.gk2_f = 0.f;
    pr.gauss_sum = 0;
    if (cfg->gauss_sigma > 0.0) {
        const double s = cfg->gauss_sigma, cc = cfg->gauss_centre;
        double Z;
        if (cfg->gauss_norm == VAMP_GAUSS_NORM_REAL_LINE) Z = s * std::sqrt(2.0 * M_PI);
        else Z = s * std::sqrt(M_PI / 2.0) * (std::erf((1.0 - cc) / (s * M_SQRT2)) + std::erf(cc / (s * M_SQRT2)));
        S.zinv = 1.0 / Z;
        pr.gcen = cc;
        pr.gk2 = M_LOG2E / (2.0 * s * s);
        // a coordinate's exponent reaches this (or is no number, which the sum
        // carries on); packed numbers hold up to 2^960
        const double amax = std::max(cc * cc, (1.0 - cc) * (1.0 - cc)) * pr.gk2;
        pr.gauss_sum = !(amax <= 900.0);
        pr.gcen_f = (float)cc;
        pr.gk2_f = (float)pr.gk2;
    }
    pr.matching = P == K;
    for (int q = 0; pr.matching && q < K; ++q)
        if (!same_maps(cfg->channels[q], cfg->peaks[q])) pr.matching = 0;
    pr.map_any = pr.pow_any = 0;
    for (int q = 0; q < K; ++q)
        for (int t = 0; t < cfg->channels[q].n_mapped; ++t) {
            const int kind = cfg->channels[q].kind[t];
            if (kind != VAMP_MAP_ID) pr.map_any |= 1u << cfg->channels[q].coord[t];
            if (kind == VAMP_MAP_POW) pr.pow_any |= 1u << cfg->channels[q].coord[t];
        }
    pr.lay64 = make_layout_c<double>(d, n);
    pr.lay32 = make_layout_c<float>(d, n);

    S.hdr64.assign((size_t)K * pr.lay64.H, 0);
    S.hdr32.assign((size_t)K * pr.lay32.H, 0);
    for (int q = 0; q < K; ++q) {
        // with matching peaks the channel header carries the peak weight too
        const double w = pr.matching ? cfg->peak_weight[q] : 0.0;
        make_hdr64(cfg->channels[q], w, S.zinv, d, pr.lay64.lshift, S.hdr64.data() + (size_t)q * pr.lay64.H);
        make_hdr32(cfg->channels[q], w, S.zinv, d, S.hdr32.data() + (size_t)q * pr.lay32.H);
    }
    S.pk64.assign((size_t)P * sizeof(MapRec<double>), 0);
    S.pk32.assign((size_t)P * sizeof(MapRec<float>), 0);
    for (int q = 0; q < P; ++q) {
        const MapRec<double> r64 = make_rec<double>(cfg->peaks[q], cfg->peak_weight[q], S.zinv, d);
        const MapRec<float> r32 = make_rec<float>(cfg->peaks[q], cfg->peak_weight[q], S.zinv, d);
        std::memcpy(S.pk64.data() + (size_t)q * sizeof r64, &r64, sizeof r64);
        std::memcpy(S.pk32.data() + (size_t)q * sizeof r32, &r32, sizeof r32);
    }
    return true;
}

Arena plan_arena(const Params& P)
{
    Arena A{};
    const size_t K = (size_t)P.K, rows = K * P.d;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += a256(bytes); return o; };
    // the state that callers read and write, and the scalars: one range
    A.edges64 = take(rows * (P.n + 1) * 8);
    A.alpha = take(K * 8);
    A.shift = take(K * 8);
    A.sc = take(sizeof(Scalars));
    A.lk64 = take(K * P.lay64.bytes);
    A.lk32 = take(K * P.lay32.bytes);
    A.alpha32 = take(K * 4);
    A.alphan = take(K * 8);
    A.acum = take(K * 8);
    A.nc = take(K * 8);
    A.pc = take((K + 1) * 8);
    A.D = take(rows * P.n * 8);
    A.csum = take(2 * K * 8);
    A.ic = take(K * 8);
    A.vc = take(K * 8);
    A.wc = take(K * 8);
    A.pk64 = take((size_t)P.P * sizeof(MapRec<double>));
    A.pk32 = take((size_t)P.P * sizeof(MapRec<float>));
    A.nr = take(K * 8);
    A.spc = take(K * 8);
    A.coff = take((K + 1) * 8);
    A.qc = take(K * 8);
    A.eqoff = take(P.n_eq_ent > 0 ? (rows + 1) * 4 : 0);
    A.eqent = take((size_t)P.n_eq_ent * 4);
    A.bytes = off;
    return A;
}

void bind_arena(Params& P, unsigned char* b, const Arena& A)
{
    P.edges64 = (double*)(b + A.edges64);
    P.lk64 = b + A.lk64;
    P.lk32 = b + A.lk32;
    P.alpha = (double*)(b + A.alpha);
    P.alpha32 = (float*)(b + A.alpha32);
    P.alphaN = (double*)(b + A.alphan);
    P.shift = (double*)(b + A.shift);
    P.Acum = (double*)(b + A.acum);
    P.Nc = (int64_t*)(b + A.nc);
    P.Pc = (int64_t*)(b + A.pc);
    P.D = (double*)(b + A.D);
    P.csum = (double*)(b + A.csum);
    P.Ic = (double*)(b + A.ic);
    P.Vc = (double*)(b + A.vc);
    P.Wc = (double*)(b + A.wc);
    P.pk64 = (const MapRec<double>*)(b + A.pk64);
    P.pk32 = (const MapRec<float>*)(b + A.pk32);
    P.sc = (Scalars*)(b + A.sc);
    P.nr = (int64_t*)(b + A.nr);
    P.spc = (int64_t*)(b + A.spc);
    P.coff = (int64_t*)(b + A.coff);
    P.Qc = (double*)(b + A.qc);
    P.cellsum = nullptr;  // sized per pass by the context
    P.eq_off = P.n_eq_ent > 0 ? (const int32_t*)(b + A.eqoff) : nullptr;
    P.eq_ent = P.n_eq_ent > 0 ? (const int32_t*)(b + A.eqent) : nullptr;
}

cudaError_t upload_setup(const Params& P, const Setup& S, cudaStream_t s, bool both)
{
    cudaError_t e = cudaSuccess;
    if (both || !P.fp32)
        e = cudaMemcpy2DAsync(P.lk64, P.lay64.bytes, S.hdr64.data(), P.lay64.H, P.lay64.H, P.K,
                              cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && (both || P.fp32))
        e = cudaMemcpy2DAsync(P.lk32, P.lay32.bytes, S.hdr32.data(), P.lay32.H, P.lay32.H, P.K,
                              cudaMemcpyHostToDevice, s);
    // peaks of their own (matching ones are in the channels' headers)
    if (e == cudaSuccess && !P.matching && !P.fp32)
        e = cudaMemcpyAsync((void*)P.pk64, S.pk64.data(), S.pk64.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && !P.matching && P.fp32)
        e = cudaMemcpyAsync((void*)P.pk32, S.pk32.data(), S.pk32.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && P.n_eq_ent > 0)
        e = cudaMemcpyAsync((void*)P.eq_off, S.eq_off.data(), S.eq_off.size() * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && P.n_eq_ent > 0)
        e = cudaMemcpyAsync((void*)P.eq_ent, S.eq_ent.data(), S.eq_ent.size() * 4, cudaMemcpyHostToDevice, s);
    return e;
}

// D-value copies: the lanes of a warp that add to the same axis at a step use
// different ones, so that calls of one bin rarely meet at one word (an FP64
// add in shared memory is a compare-and-swap loop: a d = 4, n = 20 pass went
// through it 36 times per add with one copy).  Every segment clears and sums
// the copies that it uses, so the plan keeps them within 16 KB and a segment of
// few calls takes fewer (vamp_pass.cuh): with 32 KB, all used by every segment,
// the 32-problem batch went from 8.65 to 9.99 ms.
TilePlan plan_tiles(size_t S, int K, int dn, size_t fixed, size_t budget)
{
    const size_t most = 16 * 1024, one = (size_t)dn * 8;
    int ds = 5;
    while (ds > 0 && ((one << ds) > most || fixed + 2 * S + (one << ds) > budget)) --ds;
    const size_t d = one << ds;
    const size_t room = budget > fixed + d ? budget - fixed - d : 0;
    TilePlan p{};
    p.dshift = ds;
    p.tile = (size_t)K * S <= room ? K : (int)std::max<size_t>(1, std::min<size_t>((size_t)K, room / (2 * S)));
    const size_t tiles = (size_t)(p.tile < K ? 2 : 1) * p.tile * S;
    p.smem_int = fixed + tiles + d;
    p.smem_gen = fixed + tiles;
    return p;
}

TilePlan pass_smem(const Params& P, int fp32, int minb)
{
    const size_t S = (size_t)(fp32 ? P.lay32.bytes : P.lay64.bytes);
    // per-CTA share of the SM's shared memory, less the per-CTA reservation
    int dev = 0, per_sm = 0, reserved = 0;
    size_t budget = TILE_BUDGET;
    if (minb > 2 && cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) == cudaSuccess)
        budget = std::min(budget, (size_t)(per_sm / minb - reserved));
    return plan_tiles(S, P.K, P.d * P.n, SMEM_HEAD, budget);
}

std::vector<const PassVariant*> pass_candidates(int fp32, int d, int n, int stratified, int K)
{
    static std::vector<PassVariant> all;
    static std::once_flag once;
    std::call_once(once, [] {
        add_pass_variants_f32_generic(all);
        add_pass_variants_f32_shapes(all);
        add_pass_variants_f32_dims(all);
        add_pass_variants_f64(all);
        add_pass_variants_f64_dims(all);
        add_pass_variants_union(all);
        add_pass_variants_union_dims(all);
    });
    const bool uni = K > 0 && union_fits(fp32, d, K, n, stratified);
    std::vector<const PassVariant*> out;
    for (int u = 0; u <= (uni ? 1 : 0); ++u)          // staged-tile kernels, then union kernels
        for (int fit = stratified ? 2 : 0; fit < 3; ++fit)  // exact shape, range of d, any shape
            for (const PassVariant& v : all) {
                if (v.fp32 != fp32 || v.uni != u) continue;
                const int is = v.D > 0 ? 0 : (v.dhi > 0 ? 1 : 2);
                if (is != fit || (is == 0 && (v.D != d || v.NB != n)) || (is == 1 && (d < v.dlo || d > v.dhi))) continue;
                out.push_back(&v);
            }
    return out;
}

cudaError_t ensure_smem(const void* fn, size_t bytes)
{
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess && fa.maxDynamicSharedSizeBytes < (int)bytes)
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    return e;
}

}  // namespace vamp
