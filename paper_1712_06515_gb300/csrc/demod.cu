// Detector-frame ("demodulation") CrossCorr: the statistic the resampled method
// replaces (Sec. II: Eqs. fourier-transform-def, normalized-z-bin, total-data-eq,
// geometric-filter, norm-cc, textbook-cc-rho), evaluated at the plan's output
// frequencies on the same data, so the two methods can be compared on one GPU.
//
//   crosscorr_demod_prepare: short Fourier transforms of every locked T_sft block, only
//     the bins a signal in the band can reach (direct DFT with an exact integer twiddle
//     index), normalised to unit variance, and per SFT the filter weights
//     a^ = sqrt(2 T_sft / S) a(t_K), b^ likewise (S = 2 sigma^2 dt);
//   crosscorr_demod_search: per template an FP64 pass gives, per locked SFT (a list in
//     time order built by the prepare call), the signal's bin position and phase as
//     linear functions of the output bin; one thread per (template, output bin) then
//     walks the SFTs in time order, forms
//     y_K = sum_m (-1)^m sinc(kappa_Km) z_Km exp(-i Phi_K) (= Xi_K z_K exp(-i Phi_K); here and in
//     Xi_K with every sinc times pi / 4, which cancels in rho) and
//     sums Gamma_KL 2 Re(conj(y_K) y_L) over every earlier SFT L within T_max, with the
//     normalisation sum (Xi_K Xi_L Gamma_KL)^2 alongside; rho = raw / sqrt(2 den).  Two
//     forms of that sum: the method's pair loop (demod_pair_kernel, one term per pair,
//     each unordered pair once) and the separable form (demod_sep_kernel: Gamma_KL is a
//     sum of products of a K factor and an L factor, so running sums over the partners
//     give the same value in O(1) per SFT).
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace cc {
cc_status set_inputs(cc_plan* plan, const void* const* x_dev);

namespace {

constexpr int SFT_THREADS = 256;
constexpr int DM_MAX_SFT_SAMPLES = 16384;   // T_sft / dt staged in shared memory
constexpr size_t DM_RING_BUDGET = 160 * 1024;
constexpr size_t DM_SEP_RING = 40 * 1024;   // separable form: block-sum ring per CTA (R_s <= 10)

struct DemodTiming {   // per (template, locked SFT): 32 bytes
    float A0, A1;       // signal bin position x - 1/2 = A0 + df A1 (df = f - f_h of the output bin)
    float C0, C1;       // heterodyned phase (cycles) = C0 + kbar C1 with kbar = 128 kh + kl:
    float C128, pad0;   //   C0 + kh C128 + kl C1 (mod 1); pad0, pad1: the SFT's a^, b^
    float pad1, pad2;   //   divided by sqrt(10); pad2: its row of SFT bins, X n_blk + l (int bits)
};

// What the separable kernel does when the list reaches a new block, from the list alone
// (crosscorr_demod_prepare): bits 0-1 DM_*, bit 2: the partial sums join the compensated totals,
// bits 3-16 and 17-30: the ring slots of the finished and of the new block.
enum { DM_SAME = 0, DM_STEP = 1, DM_REFRESH = 2, DM_EMPTY = 3 };
constexpr int DM_LIST_PAD = 8;   // padding entries of the per-entry tables

// DFT bins m_lo .. m_lo + nbins - 1 of one T_sft block of detector X, normalised to unit
// variance, each times (-1)^m: the two-bin interpolation's alternating sign
// (-1)^m0 (s0 z_m0 - s1 z_(m0+1)) is then s0 z'_m0 + s1 z'_(m0+1).  Zero for gaps.  Also the
// block's filter weights (a^, b^, locked).
__global__ void __launch_bounds__(SFT_THREADS)
sft_kernel(DevParams p, int nsft, int m_lo, int nbins, int n_blk, const float2* __restrict__ tw,
           float2* __restrict__ z, float4* __restrict__ wts) {
    extern __shared__ __align__(16) float2 xs[];
    const int l = blockIdx.x, X = blockIdx.y;
    float2* zo = z + ((size_t)X * n_blk + l) * (nbins + 2);   // two zero columns end a row
    if (threadIdx.x < 2) zo[nbins + threadIdx.x] = make_float2(0.f, 0.f);
    const float2 sw = (l < (int)p.n_sig[X]) ? __ldg(p.sigw[X] + l) : make_float2(0.f, 0.f);
    const bool locked = sw.x > 0.f;
    if (threadIdx.x == 0) {
        float ah = 0.f, bh = 0.f;
        if (locked) {
            // a, b at the mid-time (linear in the table, end intervals extrapolated)
            const double tm = (double)l * nsft + 0.5 * nsft;
            const double fr = (tm - (double)p.ab_j0) / (double)p.n_ab_step;
            int64_t i = (int64_t)floor(fr);
            const int64_t nab = p.n_ab[X];
            i = i < 0 ? 0 : (i > nab - 2 ? nab - 2 : i);
            const double f = fr - (double)i;
            const double a = __ldg(p.atab[X] + i) + f * (__ldg(p.atab[X] + i + 1) - __ldg(p.atab[X] + i));
            const double b = __ldg(p.btab[X] + i) + f * (__ldg(p.btab[X] + i + 1) - __ldg(p.btab[X] + i));
            const double sc = sqrt((double)nsft * (double)sw.y);   // sqrt(2 T_sft / S) = sqrt(nsft / sigma^2)
            ah = (float)(sc * a);
            bh = (float)(sc * b);
        }
        wts[(size_t)X * n_blk + l] = make_float4(ah, bh, locked ? 1.f : 0.f, 0.f);
    }
    if (!locked) {
        for (int i = threadIdx.x; i < nbins; i += blockDim.x) zo[i] = make_float2(0.f, 0.f);
        return;
    }
    const float2* __restrict__ x = p.x[X] + (size_t)l * nsft;
    for (int j = threadIdx.x; j < nsft; j += blockDim.x) xs[j] = __ldg(x + j);
    __syncthreads();
    const float norm = sqrtf(sw.y / (float)nsft);   // dt sqrt(2 / (T_sft S)) = 1 / (sigma sqrt(nsft))
    for (int i = threadIdx.x; i < nbins; i += blockDim.x) {
        const int m = m_lo + i;
        const int step = ((m % nsft) + nsft) % nsft;     // exp(-2 pi i j m / nsft) = tw[(j m) mod nsft]
        int idx = 0;
        float2 acc = make_float2(0.f, 0.f);
        for (int j = 0; j < nsft; ++j) {
            const float2 w = tw[idx];
            const float2 v = xs[j];
            acc.x = fmaf(v.x, w.x, fmaf(-v.y, w.y, acc.x));
            acc.y = fmaf(v.x, w.y, fmaf(v.y, w.x, acc.y));
            idx += step;
            idx -= idx >= nsft ? nsft : 0;
        }
        const float sn = (m & 1) ? -norm : norm;         // stored times (-1)^m (see below)
        zo[i] = make_float2(acc.x * sn, acc.y * sn);
    }
}

// Per (template, detector, SFT block): the signal's heterodyned bin position and phase as
// functions of the output bin, in FP64 reduced to FP32 pieces.
__device__ DemodTiming demod_timing(const DevParams& p, const cc_template& T, int nsft, int l, int X, double df0,
                                    double dK) {
    const double tmid = ((double)l * nsft + 0.5 * nsft) * p.dt;   // relative to t0
    // Delta_X(t) and its slope (linear interpolation of the table)
    const double u = (tmid - p.eph_t0[X]) * p.inv_eph_dt[X];
    int64_t i = (int64_t)floor(u);
    const int64_t n = p.n_eph[X];
    i = i < 0 ? 0 : (i > n - 2 ? n - 2 : i);
    const double d0 = __ldg(p.ssb[X] + i), d1 = __ldg(p.ssb[X] + i + 1);
    const double dl = d0 + (u - (double)i) * (d1 - d0);
    const double ddl = (d1 - d0) * p.inv_eph_dt[X];
    // binary delay R/c at t_SSB and its rate (Eqs. t-ssb-equation, tau-equation,
    // Kepler-equation), dtau/dt = (1 + Delta') (1 - dR/du / c)
    const Orbit o = make_orbit(p, T);
    const double u_ssb = tmid + dl, om = 6.283185307179586 * o.invP;
    double R, dR;
    if (o.e == 0.0) {
        double s, c;
        sincospi(2.0 * ((u_ssb - o.tasc_rel) * o.invP), &s, &c);
        R = o.a_p * s;
        dR = o.a_p * om * c;
    } else {
        double xm = (u_ssb - o.tp_rel) * o.invP;
        xm -= floor(xm);
        const double M = 6.283185307179586 * xm;
        double E = M + o.e * sinpi(2.0 * xm), sE, cE;
        sincos_rad(E, &sE, &cE);
        for (int it = 0; it < N_KEPLER_ITER; ++it) {
            E -= (E - o.e * sE - M) / (1.0 - o.e * cE);
            sincos_rad(E, &sE, &cE);
        }
        R = o.a_p * (o.sinw * (cE - o.e) + o.cosw * o.sq * sE);
        dR = o.a_p * (-o.sinw * sE + o.cosw * o.sq * cE) * om / (1.0 - o.e * cE);
    }
    const double d = dl - R;                                           // tau - t
    const double dtau = (1.0 + ddl) * (1.0 - dR);
    const double Tsft = nsft * p.dt;
    DemodTiming r;
    // x = (f (dtau - 1) + df) T_sft with f = f_h + df
    r.A0 = (float)(p.f_h * (dtau - 1.0) * Tsft - 0.5);
    r.A1 = (float)(dtau * Tsft);
    // phase f tau - f_h t = f_h d + df (t + d), df = df0 + kbar dK
    const double tau = tmid + d;
    const double c0 = p.f_h * d + df0 * tau;
    const double c1 = dK * tau, c128 = 128.0 * dK * tau;
    r.C0 = (float)(c0 - floor(c0));
    r.C1 = (float)(c1 - floor(c1));
    r.C128 = (float)(c128 - floor(c128));
    r.pad0 = r.pad1 = r.pad2 = 0.f;
    return r;
}

// The search kernels' records: one per locked SFT of the time-ordered list, the timing of
// demod_timing with the SFT's filter weights (divided by sqrt(10)) and its row of bins in
// the spare words; two padding records (no bins) follow the list.
__global__ void demod_timing_list_kernel(DevParams p, const cc_template* __restrict__ tm, int nsft, int n_blk,
                                         double df0, double dK, const int* __restrict__ list, int n_list,
                                         const float4* __restrict__ wts, DemodTiming* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t t = blockIdx.y;
    if (i >= n_list + 2) return;
    DemodTiming r;
    if (i >= n_list) {                                 // padding: no bins (x far below the band)
        r.A0 = -1.0e9f;
        r.A1 = r.C0 = r.C1 = r.C128 = r.pad0 = r.pad1 = 0.f;
        r.pad2 = __int_as_float(0);
    } else {
        const int key = __ldg(list + i);
        const int l = key >> 2, X = key & 3;
        r = demod_timing(p, tm[t], nsft, l, X, df0, dK);
        const float4 wk = __ldg(wts + (size_t)X * n_blk + l);
        r.pad0 = wk.x * 0.316227766016837933f;         // a^ / sqrt(10)
        r.pad1 = wk.y * 0.316227766016837933f;
        r.pad2 = __int_as_float(X * n_blk + l);
    }
    out[(size_t)t * (n_list + 2) + i] = r;
}

// The same statistic in separable form.  The geometric filter Gamma_KL = (a^_K a^_L +
// b^_K b^_L) / 10 splits into a factor of K times one of L, so the pair sum of SFT K over
// its partners L is 2 Re(conj(y_K) (a^_K SA + b^_K SB)) / 10 with SA = sum_L a^_L y_L and
// SB = sum_L b^_L y_L, and the normalisation term Xi_K^2 (a^_K^2 UAA + 2 a^_K b^_K UAB +
// b^_K^2 UBB) / 100 with UAA = sum_L Xi_L^2 a^_L^2, UAB = sum_L Xi_L^2 a^_L b^_L,
// UBB = sum_L Xi_L^2 b^_L^2: O(1) per SFT instead of one term per partner.  The partners
// of (block l, detector X) are every detector of blocks l - R_s .. l - 1 (window sums W)
// and the earlier detectors of block l (running sums P).  W moves by adding the finished
// block's sums s_l and subtracting s_(l - R_s), and is recomputed exactly every few blocks
// so that rounding cannot drift.  s_(l - R_s) comes from a per-thread ring of block sums in
// shared memory when R_s is small (RING), otherwise it is recomputed from the SFT bins.
// Results equal the per-pair loop's up to FP32 rounding.
struct SepSums {     // (paired operations: the kernel is bound by instruction issue)
    float2 ay, by;   // sum a^ y, sum b^ y
    float2 u;        // sum Xi^2 a^^2, sum Xi^2 a^ b^
    float ubb;       // sum Xi^2 b^^2
};

__device__ __forceinline__ void sep_zero(SepSums& a) {
    a.ay = a.by = a.u = make_float2(0.f, 0.f);
    a.ubb = 0.f;
}

__device__ __forceinline__ void sep_add(SepSums& a, const SepSums& b) {
    a.ay = cadd(a.ay, b.ay);
    a.by = cadd(a.by, b.by);
    a.u = cadd(a.u, b.u);
    a.ubb += b.ubb;
}

__device__ __forceinline__ void sep_sub(SepSums& a, const SepSums& b) {
    a.ay = csub(a.ay, b.ay);
    a.by = csub(a.by, b.by);
    a.u = csub(a.u, b.u);
    a.ubb -= b.ubb;
}

// An SFT's factors, the same for every bin (a^, b^ over sqrt(10)): (a^, a^), (b^, b^),
// (a^^2, a^ b^), b^^2.
struct SftW {
    float2 a, b, u;
    float bb;
};

__device__ __forceinline__ SftW sft_w(float a, float b) {
    return SftW{make_float2(a, a), make_float2(b, b), make_float2(a * a, a * b), b * b};
}

// One SFT's contribution (a^ y, b^ y, Xi^2 a^^2, Xi^2 a^ b^, Xi^2 b^^2) to the sums
__device__ __forceinline__ void sep_add_sft(SepSums& s, float2 y, float xi2, const SftW& w) {
    s.ay = __ffma2_rn(w.a, y, s.ay);
    s.by = __ffma2_rn(w.b, y, s.by);
    s.u = make_float2(fmaf(xi2, w.u.x, s.u.x), fmaf(xi2, w.u.y, s.u.y));
    s.ubb = fmaf(xi2, w.bb, s.ubb);
}

// One SFT's inputs, fetched ahead of its arithmetic: h = x - m - 1/2 in [-1/2, 1/2] of the
// signal bin position x between bins m and m + 1, the heterodyne phase in cycles reduced to
// [-1/2, 1/2], and the two stored bins (zero when out of the band).
struct SftIn {
    float h, cyc;
    float2 z0, z1;
};

// The two sinc weights of kappa = -f and 1 - f, f = h + 1/2, times pi / 4: with
// g(h) = cos(pi h) / (1 - 4 h^2), an entire even function, sinc(f) = (4 / pi) g (1/2 - h) and
// sinc(1 - f) = (4 / pi) g (1/2 + h); the common factor cancels in rho.  g = 1 + u P(u), u = h^2, P of
// degree four by least squares at Chebyshev nodes, one coefficient after the other rounded to FP32
// and the rest fitted again: 2.5e-10 from g on |h| <= 1/2.  In FP32 the sincs are within 9e-8 (a
// series for one and a quotient for the other: 1.4e-7).
__device__ __forceinline__ float2 sinc_weights(float h) {
    const float u = h * h;
    float g = -0.000398144301f;
    g = fmaf(g, u, 0.00628934102f);
    g = fmaf(g, u, -0.0572400875f);
    g = fmaf(g, u, 0.319502473f);
    g = fmaf(g, u, -0.934802175f);
    g = fmaf(g, u, 1.f);
    const float k = 0.5f * g;
    return make_float2(fmaf(-h, g, k), fmaf(h, g, k));
}

// The demodulated bin y (the two-bin sinc interpolation, rotated by the heterodyne phase) and
// the interpolation weight Xi^2.  The rotation takes the phase in [-1/2, 1/2] cycles to the fast
// sine/cosine, whose absolute error there (2^-21.4) is far below the statistic's FP32 rounding.
__device__ __forceinline__ float2 sft_y(const SftIn& q, float& xi2) {
    const float2 s = sinc_weights(q.h);
    xi2 = fmaf(s.x, s.x, s.y * s.y);
    const float2 u = make_float2(fmaf(s.x, q.z0.x, s.y * q.z1.x), fmaf(s.x, q.z0.y, s.y * q.z1.y));
    float sn, cs;
    __sincosf(6.28318530717958648f * q.cyc, &sn, &cs);
    return make_float2(fmaf(u.x, cs, u.y * sn), fmaf(u.y, cs, -u.x * sn));
}

// One record of the list: timing, weights and row of SFT i.
struct SepRec {
    float4 t0;   // A0, A1, C0, C1
    float4 t1;   // C128, a^, b^, row (int bits)
};

// x - 1/2 rounded to the nearest integer m by adding 1.5 x 2^23 (|x| < 2^22 for any real SFT; a
// tie gives f = 0 or 1 with the same weights on the same bins), m also read from the sum's bits.
__device__ __forceinline__ void rec_fetch(SftIn& q, const SepRec& r, float df, float kh, float kl, int m_lo,
                                          int nbins, const float2* __restrict__ z) {
    constexpr float MAGIC = 12582912.f;
    const float xs = fmaf(df, r.t0.y, r.t0.x), t = xs + MAGIC;
    q.h = xs - (t - MAGIC);
    const int i = __float_as_int(t) - (0x4b400000 + m_lo);
    const int c = (unsigned)i < (unsigned)(nbins - 1) ? i : nbins;   // the zero columns
    const float cyc = fmaf(kl, r.t0.w, fmaf(kh, r.t1.x, r.t0.z));
    q.cyc = cyc - rintf(cyc);
    const float2* zr = z + (size_t)(unsigned)__float_as_int(r.t1.w) * (unsigned)(nbins + 2) + c;
    q.z0 = __ldg(zr);
    q.z1 = __ldg(zr + 1);
}

// A thread takes SB output bins of one template (a CTA's threads apart) and walks the list of
// locked SFTs in time order (gaps never enter the loop): what is the same for every bin -- the
// records, the weights' products, the list's control words -- is read and formed once for them.
// The filter weights come scaled by 1/sqrt(10), so Gamma_KL = a^'_K a^'_L + b^'_K b^'_L and the
// factors 1/10 and 1/100 drop out (the pair sum is then half the statistic's raw sum).
// V holds the sums over SFT K's partners so far (window W plus the current block); block
// sums go to the window when the block index changes: one step adds s_l and subtracts
// s_(l - R_s); a jump over empty blocks, and every 4 (R_s + 1) steps, sums the window
// exactly.  Records and control words reach shared memory by cp.async, SG at a time, one group
// ahead; SFT i + 1's bins load while SFT i is summed.  What bounds it: instruction issue (66 %
// active with the twelve warps whose rings fit an SM, about 110 instructions per SFT and 32 bins): 16
// templates on 120 days 28.8 ms, 44.9 with one bin a thread.
constexpr int SB = 2, SG = 16;

template <bool RING>
__global__ void __launch_bounds__(128) demod_sep_kernel(DevParams p, int m_lo, int nbins, int n_blk, int Rs,
                                 const float2* __restrict__ z, const DemodTiming* __restrict__ recs, int n_list,
                                 const int* __restrict__ boff, const int* __restrict__ list, const int* __restrict__ ctl,
                                 const double* __restrict__ dfreq, const int64_t* __restrict__ kbar, int64_t t_base,
                                 float* __restrict__ rho) {
    extern __shared__ __align__(16) float sring[];     // RING: [R_s + 1][7 words][SB][nthr] block sums, thread-private
    __shared__ __align__(16) float4 s_rec[3][SG][2];
    __shared__ __align__(16) int s_ctl[3][SG];
    const int nthr = blockDim.x, tid = threadIdx.x, rst = SB * nthr;
    const int64_t t = t_base + blockIdx.y;
    const int k0 = blockIdx.x * rst + tid;
    const DemodTiming* rt = recs + (size_t)(t - t_base) * (n_list + 2);
    if (n_list == 0) {                                 // no locked SFT
        for (int q = 0; q < SB; ++q)
            if (k0 + q * nthr < (int)p.N_f) rho[(size_t)t * p.N_f + k0 + q * nthr] = 0.f;
        return;
    }
    if (RING)
        for (int j = 0; j < (Rs + 1) * 7 * SB; ++j) sring[(size_t)j * nthr + tid] = 0.f;
    // threads past the last bin compute bin 0's statistic and store nothing
    float df[SB], kh[SB], kl[SB];
#pragma unroll
    for (int q = 0; q < SB; ++q) {
        const int k = k0 + q * nthr < (int)p.N_f ? k0 + q * nthr : 0;
        df[q] = (float)__ldg(dfreq + k);
        const int64_t kb = __ldg(kbar + k);
        kh[q] = (float)(kb >> 7);
        kl[q] = (float)(kb & 127);
    }
    auto ring_get = [&](int slot, int q) {
        const float* r = sring + slot * 7 * rst;
        const float2* r2 = (const float2*)r + q * nthr + tid;
        return SepSums{r2[0], r2[rst], r2[2 * rst], r[6 * rst + q * nthr + tid]};
    };
    auto ring_put = [&](int slot, int q, const SepSums& v) {
        float* r = sring + slot * 7 * rst;
        float2* r2 = (float2*)r + q * nthr + tid;
        r2[0] = v.ay;
        r2[rst] = v.by;
        r2[2 * rst] = v.u;
        r[6 * rst + q * nthr + tid] = v.ubb;
    };
    // block j's sums from its SFT bins (no ring)
    auto block_sums = [&](int j, int q, SepSums& sj) {
        sep_zero(sj);
        const int e = __ldg(boff + j + 1);
        for (int i = __ldg(boff + j); i < e; ++i) {
            const float4* r4 = (const float4*)(rt + i);
            const SepRec r{__ldg(r4), __ldg(r4 + 1)};
            SftIn in;
            rec_fetch(in, r, df[q], kh[q], kl[q], m_lo, nbins, z);
            float xi2;
            const float2 y = sft_y(in, xi2);
            sep_add_sft(sj, y, xi2, sft_w(r.t1.y, r.t1.z));
        }
    };
    // group n (entries n SG ..) into buffer n mod 3; past the list: the padding record, no control
    auto stage = [&](int n) {
        if (tid < 2 * SG + SG / 4) {
            if (tid < 2 * SG) {
                const int i = min(n * SG + (tid >> 1), n_list);
                const uint32_t d = (uint32_t)__cvta_generic_to_shared(&s_rec[n % 3][tid >> 1][tid & 1]);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"((const float4*)(rt + i) + (tid & 1)) : "memory");
            } else if (n * SG < n_list) {
                const uint32_t d = (uint32_t)__cvta_generic_to_shared(&s_ctl[n % 3][4 * (tid - 2 * SG)]);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(ctl + n * SG + 4 * (tid - 2 * SG)) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float raw[SB], rawc[SB], den[SB], denc[SB];
    // the pair and normalisation terms go to plain FP32 partial sums that join the
    // compensated totals at most every 64 SFTs (at a block change)
    float raw_p[SB], den_p[SB];
    SepSums W[SB], V[SB];
    SftIn F[SB];
    stage(0);
    stage(1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int q = 0; q < SB; ++q) {
        raw[q] = rawc[q] = den[q] = denc[q] = raw_p[q] = den_p[q] = 0.f;
        sep_zero(W[q]);
        sep_zero(V[q]);
        rec_fetch(F[q], SepRec{s_rec[0][0][0], s_rec[0][0][1]}, df[q], kh[q], kl[q], m_lo, nbins, z);
    }
    const int groups = (n_list + SG - 1) / SG;
    for (int n = 0, buf = 0; n < groups; ++n) {
        const int next = buf == 2 ? 0 : buf + 1;
        // group n + 1's records are needed by this group's last fetch
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();                               // and every thread has left group n - 1's buffer
        stage(n + 2);
        const int cnt = min(SG, n_list - n * SG);
#pragma unroll 2
        for (int e = 0; e < cnt; ++e) {
            const float4 w4 = s_rec[buf][e][1];
            const SftW w = sft_w(w4.y, w4.z);
            const int cw = s_ctl[buf][e];
            const float4* nr = e + 1 < SG ? s_rec[buf][e + 1] : s_rec[next][0];
            float2 y[SB];
            float xi2[SB];
#pragma unroll
            for (int q = 0; q < SB; ++q) {
                y[q] = sft_y(F[q], xi2[q]);
                rec_fetch(F[q], SepRec{nr[0], nr[1]}, df[q], kh[q], kl[q], m_lo, nbins, z);
            }
            const int op = cw & 3;
            if (op != DM_SAME) {                       // the block before is complete: the new block's window
                const int from = (cw >> 3) & 0x3fff, to = (cw >> 17) & 0x3fff;
                const int i = n * SG + e;
                if (Rs == 0) {
                } else if (RING) {
#pragma unroll
                    for (int q = 0; q < SB; ++q) {
                        SepSums Pb = V[q];             // the finished block's sums
                        sep_sub(Pb, W[q]);
                        ring_put(from, q, Pb);
                    }
                    if (op == DM_STEP) {               // slot `to` holds s_(l - R_s - 1)
#pragma unroll
                        for (int q = 0; q < SB; ++q) {
                            W[q] = V[q];
                            sep_sub(W[q], ring_get(to, q));
                        }
                    } else {
                        const int l = __ldg(list + i) >> 2, lcur = __ldg(list + i - 1) >> 2;
                        SepSums zero;
                        sep_zero(zero);
                        const int nz = min(l - lcur - 1, Rs + 1);   // empty blocks lcur + 1 .. l - 1
#pragma unroll
                        for (int q = 0; q < SB; ++q) {
                            int s = from;
                            for (int j = 1; j <= nz; ++j) {
                                s = s == Rs ? 0 : s + 1;
                                ring_put(s, q, zero);
                            }
                            sep_zero(W[q]);
                            for (int j = 0; j <= Rs; ++j)
                                if (j != to) sep_add(W[q], ring_get(j, q));
                        }
                    }
                } else if (op == DM_EMPTY) {           // every block of the new window is empty
#pragma unroll
                    for (int q = 0; q < SB; ++q) sep_zero(W[q]);
                } else {
                    const int l = __ldg(list + i) >> 2, lcur = __ldg(list + i - 1) >> 2;
#pragma unroll
                    for (int q = 0; q < SB; ++q) {
                        SepSums sj;
                        if (op == DM_STEP) {           // blocks lcur - R_s .. l - R_s - 1 leave
                            W[q] = V[q];
                            for (int j = max(0, lcur - Rs); j < l - Rs; ++j) {
                                block_sums(j, q, sj);
                                sep_sub(W[q], sj);
                            }
                        } else {                       // blocks l - R_s .. lcur (those after are empty)
                            SepSums Wn = V[q];
                            sep_sub(Wn, W[q]);
                            for (int j = max(0, l - Rs); j < lcur; ++j) {
                                block_sums(j, q, sj);
                                sep_add(Wn, sj);
                            }
                            W[q] = Wn;
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < SB; ++q) {
                    V[q] = W[q];
                    if (cw & 4) {
                        kahan_add(raw[q], rawc[q], raw_p[q]);
                        kahan_add(den[q], denc[q], den_p[q]);
                        raw_p[q] = den_p[q] = 0.f;
                    }
                }
            }
            const float ab2 = 2.f * w.u.y;
#pragma unroll
            for (int q = 0; q < SB; ++q) {
                const float2 g = __ffma2_rn(w.a, V[q].ay, __fmul2_rn(w.b, V[q].by));
                raw_p[q] = fmaf(y[q].x, g.x, fmaf(y[q].y, g.y, raw_p[q]));   // Re(conj(y) g)
                const float nq = fmaf(w.u.x, V[q].u.x, fmaf(ab2, V[q].u.y, w.bb * V[q].ubb));
                den_p[q] = fmaf(xi2[q], nq, den_p[q]);
                sep_add_sft(V[q], y[q], xi2[q], w);
            }
        }
        buf = next;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int q = 0; q < SB; ++q) {
        kahan_add(raw[q], rawc[q], raw_p[q]);
        kahan_add(den[q], denc[q], den_p[q]);
        // rho = (2 raw) / sqrt(2 den)
        if (k0 + q * nthr < (int)p.N_f)
            rho[(size_t)t * p.N_f + k0 + q * nthr] = den[q] > 0.f ? 1.41421356237309505f * raw[q] * rsqrtf(den[q]) : 0.f;
    }
}

// The method's pair loop: one thread per (template, output bin) over the locked SFTs in time
// order (the separable kernel's records), PT consecutive SFTs at a time.  The partners of SFT i
// are the entries of the list from the first one of block l_i - R_s up to i - 1, so those of a
// tile of PT SFTs are a contiguous range before the tile plus pairs inside it (start: the first
// partner of each entry).  A ring of the
// last NR = (R_s + 1) Q entries holds, per entry, the thread's y and Xi^2 (thread-private columns
// of shared memory) and the SFT's prescaled filter weights (shared); per tile the CTA forms
// Gamma_KL = a^'_K a^'_L + b^'_K b^'_L of every ring entry against the PT SFTs (zero where it is
// not a partner), and every thread reads each entry once for PT pairs: four shared-memory
// wavefronts per PT pairs and warp, where one SFT at a time took four per pair and bound the
// kernel.  Bound now by issue (66 to 70 %) and shared memory (60 % of its wavefronts): 16
// templates on 30 days 12.6 ms, 12.9 without paired operations, 30.2 one SFT at a time.  Records reach shared memory by cp.async three tiles ahead, the SFT bins registers
// one tile ahead.
constexpr int PT = 4;   // (the ring's loop is written for four)

template <int NT>
__global__ void __launch_bounds__(NT, 768 / NT) demod_pair_kernel(DevParams p, int m_lo, int nbins, int n_blk, int Rs,
                                                            const float2* __restrict__ z,
                                                            const DemodTiming* __restrict__ recs, int n_list,
                                                            const int* __restrict__ start, const double* __restrict__ dfreq,
                                                            const int64_t* __restrict__ kbar, int64_t t_base,
                                                            float* __restrict__ rho) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int nthr = NT;
    const int tid = threadIdx.x;
    const int NR = (Rs + 1) * p.Q;
    float4* sg = (float4*)sm;                          // [NR] Gamma of the tile's SFTs against each ring entry
    float4* sq = sg + NR;                              // [NR] their squares
    float4* rec4 = sq + NR;                            // [4 tiles][PT][2] records
    float* sin_ = (float*)(rec4 + 4 * PT * 2);         // [PT (PT - 1) / 2] Gamma of the pairs inside the tile, padded to 8
    float2* rab = (float2*)(sin_ + 8);                 // [NR] (a^', b^')
    float2* ry = rab + NR + (NR & 1);                  // [NR][nthr] y
    float* rx = (float*)(ry + (size_t)NR * nthr);      // [NR][nthr] Xi^2
    __shared__ int s_lo;
    const int64_t t = t_base + blockIdx.y;
    const int k = blockIdx.x * nthr + tid;
    const bool act = k < (int)p.N_f;
    const float4* rt = (const float4*)(recs + (size_t)(t - t_base) * (n_list + 2));
    if (n_list == 0) {
        if (act) rho[(size_t)t * p.N_f + k] = 0.f;
        return;
    }
    // records of tile n (padding past the list: no bins, no weight) into slot n mod 4
    auto stage = [&](int n) {
        if (tid < 2 * PT) {
            const int i = min(n * PT + (tid >> 1), n_list);
            const uint32_t d = (uint32_t)__cvta_generic_to_shared(rec4 + (n & 3) * PT * 2 + tid);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(rt + 2 * i + (tid & 1)) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto rec = [&](int i) { return SepRec{rec4[((i / PT) & 3) * PT * 2 + (i % PT) * 2], rec4[((i / PT) & 3) * PT * 2 + (i % PT) * 2 + 1]}; };
    stage(0);
    stage(1);
    stage(2);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const float df = (float)__ldg(dfreq + (act ? k : 0));
    const int64_t kb = __ldg(kbar + (act ? k : 0));
    const float kh = (float)(kb >> 7), kl = (float)(kb & 127);
    float raw = 0.f, rawc = 0.f, den = 0.f, denc = 0.f;
    SftIn F[PT];
#pragma unroll
    for (int q = 0; q < PT; ++q) rec_fetch(F[q], rec(q), df, kh, kl, m_lo, nbins, z);
    int slot0 = 0;                                     // ring slot of the tile's first SFT
    for (int n = 0; n * PT < n_list; ++n) {
        const int i0 = n * PT;
        const int have = min(i0, NR);                  // ring entries before the tile
        // the tile's first entries of the windows, and Gamma against the ring
        for (int j = tid; j < have + 8; j += nthr) {
            if (j < have) {
                const int e = i0 - 1 - j;              // j-th entry before the tile
                int s = slot0 - 1 - j;
                s += s < 0 ? NR : 0;
                const float2 ab = rab[s];
                float g[PT];
#pragma unroll
                for (int q = 0; q < PT; ++q) {
                    const float4 r1 = rec4[(n & 3) * PT * 2 + 2 * q + 1];
                    g[q] = e >= __ldg(start + i0 + q) ? fmaf(r1.y, ab.x, r1.z * ab.y) : 0.f;
                }
                sg[s] = make_float4(g[0], g[1], g[2], g[3]);
                sq[s] = make_float4(g[0] * g[0], g[1] * g[1], g[2] * g[2], g[3] * g[3]);
            } else if (j < have + 6) {                 // pairs (q, r), r < q, of the tile: index q (q - 1) / 2 + r
                const int c = j - have, q = c < 1 ? 1 : c < 3 ? 2 : 3, r = c - q * (q - 1) / 2;
                const float4 a = rec4[(n & 3) * PT * 2 + 2 * q + 1], b = rec4[(n & 3) * PT * 2 + 2 * r + 1];
                sin_[c] = i0 + r >= __ldg(start + i0 + q) ? fmaf(a.y, b.y, a.z * b.z) : 0.f;
            } else if (j == have + 6) {
                s_lo = __ldg(start + i0);
            }
        }
        stage(n + 3);
        asm volatile("cp.async.wait_group 2;" ::: "memory");   // tile n + 1's records
        __syncthreads();
        float2 y[PT];
        float xi[PT];
#pragma unroll
        for (int q = 0; q < PT; ++q) y[q] = sft_y(F[q], xi[q]);
        // the tile's sums, two SFTs to a paired operation
        float2 r01 = make_float2(0.f, 0.f), r23 = r01, n01 = r01, n23 = r01;
        const float2 x01 = make_float2(y[0].x, y[1].x), x23 = make_float2(y[2].x, y[3].x);
        const float2 y01 = make_float2(y[0].y, y[1].y), y23 = make_float2(y[2].y, y[3].y);
#pragma unroll
        for (int q = 0; q < PT; ++q) rec_fetch(F[q], rec(i0 + PT + q), df, kh, kl, m_lo, nbins, z);
        const int cnt = i0 - max(s_lo, i0 - have);
        // the range in the ring, in up to two runs of consecutive slots
        auto run = [&](int s0, int m) {
            const float2* cy = ry + s0 * nthr + tid;
            const float* cx = rx + s0 * nthr + tid;
#pragma unroll 4
            for (int j = 0; j < m; ++j) {
                const float4 g = sg[s0 + j], h = sq[s0 + j];
                const float2 yl = cy[j * nthr];
                const float xl = cx[j * nthr];
                const float2 lx = make_float2(yl.x, yl.x), ly = make_float2(yl.y, yl.y), l2 = make_float2(xl, xl);
                r01 = __ffma2_rn(make_float2(g.x, g.y), __ffma2_rn(x01, lx, __fmul2_rn(y01, ly)), r01);
                r23 = __ffma2_rn(make_float2(g.z, g.w), __ffma2_rn(x23, lx, __fmul2_rn(y23, ly)), r23);
                n01 = __ffma2_rn(make_float2(h.x, h.y), l2, n01);
                n23 = __ffma2_rn(make_float2(h.z, h.w), l2, n23);
            }
        };
        const int s = slot0 - cnt;
        if (s < 0) {
            run(s + NR, -s);
            run(0, slot0);
        } else {
            run(s, cnt);
        }
        // pairs inside the tile, then the ring takes its SFTs
        float pr[PT] = {r01.x, r01.y, r23.x, r23.y}, pq[PT] = {n01.x, n01.y, n23.x, n23.y};
#pragma unroll
        for (int q = 1; q < PT; ++q)
#pragma unroll
            for (int r = 0; r < q; ++r) {
                const float g = sin_[q * (q - 1) / 2 + r];
                pr[q] = fmaf(g, fmaf(y[q].x, y[r].x, y[q].y * y[r].y), pr[q]);
                pq[q] = fmaf(g * g, xi[r], pq[q]);
            }
        int w = slot0;
#pragma unroll
        for (int q = 0; q < PT; ++q) {
            kahan_add(raw, rawc, pr[q]);
            kahan_add(den, denc, xi[q] * pq[q]);
            if (NR >= PT || q >= PT - NR) {            // (a ring shorter than the tile keeps its last SFTs)
                ry[(size_t)w * nthr + tid] = y[q];
                rx[(size_t)w * nthr + tid] = xi[q];
                if (tid == q) {
                    const float4 r1 = rec4[(n & 3) * PT * 2 + 2 * q + 1];
                    rab[w] = make_float2(r1.y, r1.z);
                }
            }
            w = w + 1 == NR ? 0 : w + 1;
        }
        slot0 = w;
        __syncthreads();
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // rho = (2 raw) / sqrt(2 den)
    if (act) rho[(size_t)t * p.N_f + k] = den > 0.f ? 1.41421356237309505f * raw * rsqrtf(den) : 0.f;
}

// R_s = floor(T_max / T_sft): blocks back that hold partners; whether the separable form keeps
// their sums in its shared-memory ring.
int demod_blocks_back(const cc_plan* plan) {
    const double Tsft = (double)llround(plan->cfg.T_sft / plan->cfg.dt) * plan->cfg.dt;
    return (int)std::floor(plan->cfg.T_max / Tsft + 1e-9);
}
bool demod_sep_ring(int Rs) { return (size_t)(Rs + 1) * 7 * 128 * sizeof(float) <= DM_SEP_RING; }

}  // namespace
}  // namespace cc

using namespace cc;

extern "C" cc_status crosscorr_demod_prepare(cc_plan* plan, const void* const* x_dev, int32_t n_bin,
                                             double doppler_max, void* stream) {
    CC_NVTX_RANGE("crosscorr_demod_prepare");
    if (!plan) return fail(CC_ERR_INVALID, "plan is null");
    if (n_bin != 2) return fail(CC_ERR_UNSUPPORTED, "demodulation search implemented for n_bin = 2");
    if (!(doppler_max >= 0) || doppler_max > 0.01) return fail(CC_ERR_INVALID, "doppler_max must be in [0, 0.01]");
    if (doppler_max == 0) doppler_max = 5e-4;
    int64_t nsft = 0;
    {
        const double r = plan->cfg.T_sft / plan->cfg.dt;
        nsft = (int64_t)llround(r);
    }
    if (nsft < 2 || nsft > DM_MAX_SFT_SAMPLES) return fail(CC_ERR_UNSUPPORTED, "T_sft / dt must be 2..16384");
    cc_status s = set_inputs(plan, x_dev);
    if (s != CC_OK) return s;
    const DevParams& p = plan->dp;
    const int64_t n_blk = p.N_t / nsft;
    if (n_blk < 1) return fail(CC_ERR_INVALID, "series shorter than one SFT");
    // bins a signal of the band can reach: |f - f_h| <= max |df| plus Doppler and the kernel
    double dmin = 1e300, dmax = -1e300;
    for (double f : plan->freq) {
        dmin = std::min(dmin, f - plan->cfg.f_h);
        dmax = std::max(dmax, f - plan->cfg.f_h);
    }
    const double Tsft = nsft * plan->cfg.dt;
    const double wing = doppler_max * (plan->cfg.f_h + std::max(std::fabs(dmin), std::fabs(dmax))) * Tsft;
    const int m_lo = (int)std::floor(dmin * Tsft - wing) - 2;
    const int m_hi = (int)std::ceil(dmax * Tsft + wing) + 2;
    const int nbins = m_hi - m_lo + 1;
    if (nbins > nsft) return fail(CC_ERR_UNSUPPORTED, "band plus Doppler wider than an SFT");
    // device arrays (plan-owned; replaced on a new prepare)
    cudaError_t e;
    for (void* ptr : {plan->demod_z, plan->demod_w, plan->demod_tw})
        if (ptr) cudaFree(ptr);
    plan->demod_z = plan->demod_w = plan->demod_tw = nullptr;
    plan->demod_ready = false;
    std::vector<float2> tw(nsft);
    for (int64_t j = 0; j < nsft; ++j) {
        const double a = -2.0 * M_PI * (double)j / (double)nsft;
        tw[j] = make_float2((float)cos(a), (float)sin(a));
    }
    if ((e = cudaMalloc(&plan->demod_tw, sizeof(float2) * nsft)) != cudaSuccess ||
        (e = cudaMalloc(&plan->demod_z, sizeof(float2) * (size_t)p.Q * n_blk * (nbins + 2))) != cudaSuccess ||
        (e = cudaMalloc(&plan->demod_w, sizeof(float4) * (size_t)p.Q * n_blk)) != cudaSuccess)
        return cuda_fail(e, "demodulation SFT allocation");
    cudaStream_t st = (cudaStream_t)stream;
    if ((e = cudaMemcpyAsync(plan->demod_tw, tw.data(), sizeof(float2) * nsft, cudaMemcpyHostToDevice, st)) !=
        cudaSuccess)
        return cuda_fail(e, "demodulation twiddles");
    const size_t smem = sizeof(float2) * nsft;
    if (smem > 48 * 1024 &&
        (e = cudaFuncSetAttribute(sft_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return cuda_fail(e, "sft smem attribute");
    sft_kernel<<<dim3((unsigned)n_blk, (unsigned)p.Q), SFT_THREADS, smem, st>>>(
        p, (int)nsft, m_lo, nbins, (int)n_blk, (const float2*)plan->demod_tw, (float2*)plan->demod_z,
        (float4*)plan->demod_w);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "sft_kernel launch");
    // host copies the search needs: output bins' df (FP64) and kbar
    if (!plan->demod_df) {
        if ((e = cudaMalloc(&plan->demod_df, sizeof(double) * plan->N_f)) != cudaSuccess ||
            (e = cudaMalloc(&plan->demod_kbar, sizeof(int64_t) * plan->N_f)) != cudaSuccess)
            return cuda_fail(e, "demodulation bin tables");
        std::vector<double> df(plan->N_f);
        for (int64_t i = 0; i < plan->N_f; ++i)
            df[i] = (plan->f_r - 0.5 / plan->cfg.dt) + (double)plan->kbar[i] / plan->T_FFT;
        if ((e = cudaMemcpy(plan->demod_df, df.data(), sizeof(double) * plan->N_f, cudaMemcpyHostToDevice)) !=
                cudaSuccess ||
            (e = cudaMemcpy(plan->demod_kbar, plan->kbar.data(), sizeof(int64_t) * plan->N_f,
                            cudaMemcpyHostToDevice)) != cudaSuccess)
            return cuda_fail(e, "demodulation bin tables");
    }
    // the locked SFTs in time order (key 4 l + X) and each block's first entry, for the
    // separable form
    {
        std::vector<float4> w((size_t)p.Q * n_blk);
        if ((e = cudaMemcpyAsync(w.data(), plan->demod_w, sizeof(float4) * w.size(), cudaMemcpyDeviceToHost, st)) !=
                cudaSuccess ||
            (e = cudaStreamSynchronize(st)) != cudaSuccess)
            return cuda_fail(e, "demodulation SFT weights");
        std::vector<int> list, boff(n_blk + 1);
        for (int64_t l = 0; l < n_blk; ++l) {
            boff[l] = (int)list.size();
            for (int X = 0; X < p.Q; ++X)
                if (w[(size_t)X * n_blk + l].z != 0.f) list.push_back((int)(4 * l + X));
        }
        boff[n_blk] = (int)list.size();
        // per entry: its first partner, and the separable kernel's control word (a refresh after
        // 4 (R_s + 1) single-block steps: the FP32 rounding of the running sums cannot drift
        // further; totals at most every 64 SFTs)
        const int Rs = demod_blocks_back(plan), refresh = 4 * (Rs + 1);
        const bool ring = demod_sep_ring(Rs);
        std::vector<int> start(list.size() + DM_LIST_PAD, (int)list.size()), ctl(list.size() + 2 * SG, 0);
        int steps = 0, nacc = 0;
        for (size_t i = 0; i < list.size(); ++i, ++nacc) {
            const int l = list[i] >> 2;
            start[i] = boff[std::max(0, l - Rs)];
            const int lcur = i ? list[i - 1] >> 2 : l;
            if (l == lcur) continue;
            int op = DM_SAME;
            if (Rs == 0) {
                op = DM_STEP;
            } else if (ring) {
                op = l == lcur + 1 && ++steps < refresh ? DM_STEP : DM_REFRESH;
            } else {
                op = l - lcur > Rs ? DM_EMPTY : ++steps < refresh ? DM_STEP : DM_REFRESH;
            }
            if (op != DM_STEP) steps = 0;
            const bool flush = steps == 0 || nacc >= 64;
            if (flush) nacc = 0;
            ctl[i] = op | (flush ? 4 : 0);
            if (ring) ctl[i] |= lcur % (Rs + 1) << 3 | l % (Rs + 1) << 17;
        }
        for (void* ptr : {plan->demod_list, plan->demod_boff, plan->demod_start, plan->demod_ctl})
            if (ptr) cudaFree(ptr);
        plan->demod_list = plan->demod_boff = plan->demod_start = plan->demod_ctl = nullptr;
        if ((e = cudaMalloc(&plan->demod_list, sizeof(int) * std::max<size_t>(1, list.size()))) != cudaSuccess ||
            (e = cudaMalloc(&plan->demod_boff, sizeof(int) * boff.size())) != cudaSuccess ||
            (e = cudaMalloc(&plan->demod_start, sizeof(int) * start.size())) != cudaSuccess ||
            (e = cudaMalloc(&plan->demod_ctl, sizeof(int) * ctl.size())) != cudaSuccess ||
            (e = cudaMemcpy(plan->demod_start, start.data(), sizeof(int) * start.size(), cudaMemcpyHostToDevice)) !=
                cudaSuccess ||
            (e = cudaMemcpy(plan->demod_ctl, ctl.data(), sizeof(int) * ctl.size(), cudaMemcpyHostToDevice)) != cudaSuccess ||
            (!list.empty() && (e = cudaMemcpy(plan->demod_list, list.data(), sizeof(int) * list.size(),
                                              cudaMemcpyHostToDevice)) != cudaSuccess) ||
            (e = cudaMemcpy(plan->demod_boff, boff.data(), sizeof(int) * boff.size(), cudaMemcpyHostToDevice)) !=
                cudaSuccess)
            return cuda_fail(e, "demodulation SFT list");
        plan->demod_nlist = (int)list.size();
    }
    plan->demod_nsft = (int)nsft;
    plan->demod_m_lo = m_lo;
    plan->demod_nbins = nbins;
    plan->demod_nblk = (int)n_blk;
    plan->demod_ready = true;
    return CC_OK;
}

extern "C" cc_status crosscorr_plan_set_demod_form(cc_plan* plan, int form) {
    if (!plan) return fail(CC_ERR_INVALID, "plan is null");
    if (form != CC_DEMOD_PAIRS && form != CC_DEMOD_SEPARABLE) return fail(CC_ERR_INVALID, "unknown demodulation form");
    plan->demod_form = form;
    return CC_OK;
}

extern "C" cc_status crosscorr_demod_search(cc_plan* plan, const cc_template* t_dev, int64_t n_t, float* rho_dev,
                                            void* stream) {
    CC_NVTX_RANGE("crosscorr_demod_search");
    if (!plan) return fail(CC_ERR_INVALID, "plan is null");
    if (n_t < 0) return fail(CC_ERR_INVALID, "n_t must be >= 0");
    if (!plan->demod_ready) return fail(CC_ERR_INVALID, "call crosscorr_demod_prepare first");
    if (n_t == 0) return CC_OK;
    if (!t_dev || !rho_dev) return fail(CC_ERR_INVALID, "null device pointer");
    const DevParams& p = plan->dp;
    const int n_blk = plan->demod_nblk, nsft = plan->demod_nsft;
    const int Rs = demod_blocks_back(plan);
    const int W = (Rs + 1) * p.Q;
    const bool sep = plan->demod_form == CC_DEMOD_SEPARABLE;
    const int n_list = plan->demod_nlist;
    // separable form: the ring of block sums while 128 bins of it stay within DM_SEP_RING
    const bool sep_ring = sep && demod_sep_ring(Rs);
    int nthr = sep ? 128 : 256;
    auto ring_bytes = [&](int nt) {
        return sep ? (sep_ring ? (size_t)(Rs + 1) * 7 * SB * nt * sizeof(float) : 0)
                   : (size_t)W * nt * 12 + (size_t)W * 40 + 8 + 4 * PT * 32 + 32;
    };
    const int bins = sep ? SB : 1;   // output bins of a thread
    while (nthr > 32 && ring_bytes(nthr) > DM_RING_BUDGET) nthr /= 2;
    // the limit counts the ring itself, 32 threads' columns and the weights; the tile's Gamma tables
    // (28 bytes an entry more) find room beside it
    if (!sep && (size_t)W * (32 * 12 + 12) > DM_RING_BUDGET)
        return fail(CC_ERR_UNSUPPORTED, "T_max / T_sft too large for the pair ring");
    // timing records for a batch of templates: the list of locked SFTs plus two padding
    const size_t per_t = sizeof(DemodTiming) * ((size_t)n_list + 2);
    const int64_t batch = std::max<int64_t>(1, std::min<int64_t>({n_t, (int64_t)((size_t)2 << 30) / (int64_t)per_t, 65535}));
    auto kernel = [&](int nt) -> const void* {
        if (sep) return sep_ring ? (const void*)demod_sep_kernel<true> : (const void*)demod_sep_kernel<false>;
        switch (nt) {
            case 256: return (const void*)demod_pair_kernel<256>;
            case 192: return (const void*)demod_pair_kernel<192>;
            case 128: return (const void*)demod_pair_kernel<128>;
            case 96: return (const void*)demod_pair_kernel<96>;
            case 64: return (const void*)demod_pair_kernel<64>;
            default: return (const void*)demod_pair_kernel<32>;
        }
    };
    {
        // CTA size (every thread does the same work, in whole waves of the first batch): the least
        // waves x warps resident on an SM, a wave of few warps counted as one of eleven (its time
        // is the latency of a thread's steps; the separable form's two bins a thread fill the
        // issue slots from there on)
        int dev = 0, sms = 152;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        int64_t best = -1;
        for (int nt : {256, 192, 128, 112, 96, 80, 64, 48}) {
            if (sep ? nt > 128 : nt == 112 || nt == 80 || nt == 48) continue;
            if (ring_bytes(nt) > DM_RING_BUDGET) continue;
            if (ring_bytes(nt) > 48 * 1024 &&
                cudaFuncSetAttribute(kernel(nt), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring_bytes(nt)) != cudaSuccess)
                continue;
            int occ = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel(nt), nt, ring_bytes(nt)) != cudaSuccess || occ < 1)
                continue;
            const int64_t ctas = (plan->N_f + (int64_t)bins * nt - 1) / ((int64_t)bins * nt) * std::min(batch, n_t);
            const int64_t est = (ctas + (int64_t)occ * sms - 1) / ((int64_t)occ * sms) * std::max(11, occ * ((nt + 31) / 32));
            if (best < 0 || est < best) {
                best = est;
                nthr = nt;
            }
        }
    }
    cc_status s = ensure_workspace(plan, per_t * batch);
    if (s != CC_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    const size_t smem = ring_bytes(nthr);
    if (smem > 48 * 1024 &&
        (e = cudaFuncSetAttribute(kernel(nthr), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return cuda_fail(e, "demodulation smem attribute");
    const double df0 = plan->f_r - 0.5 / plan->cfg.dt, dK = 1.0 / plan->T_FFT;
    for (int64_t t0 = 0; t0 < n_t; t0 += batch) {
        const int64_t nb = std::min(batch, n_t - t0);
        if (n_list > 0) {
            demod_timing_list_kernel<<<dim3((unsigned)((n_list + 2 + 127) / 128), (unsigned)nb), 128, 0, st>>>(
                p, t_dev + t0, nsft, n_blk, df0, dK, (const int*)plan->demod_list, n_list,
                (const float4*)plan->demod_w, (DemodTiming*)plan->ws);
            count_launch();
        }
        cudaEvent_t ev0, ev1;   // diagnostic timing of the pair loop (crosscorr_plan_set_kernel_timing)
        timing_pair(plan, &ev0, &ev1);
        if (ev0) cudaEventRecord(ev0, st);
        const dim3 grid((unsigned)((plan->N_f + (int64_t)bins * nthr - 1) / ((int64_t)bins * nthr)), (unsigned)nb);
        const float2* zp = (const float2*)plan->demod_z;
        const DemodTiming* rp = (const DemodTiming*)plan->ws;
        const int *bo = (const int*)plan->demod_boff, *li = (const int*)plan->demod_list, *ct = (const int*)plan->demod_ctl,
                  *sp = (const int*)plan->demod_start;
        const double* dfp = (const double*)plan->demod_df;
        const int64_t* kp = (const int64_t*)plan->demod_kbar;
        void* as[] = {(void*)&p, (void*)&plan->demod_m_lo, (void*)&plan->demod_nbins, (void*)&n_blk, (void*)&Rs, (void*)&zp,
                      (void*)&rp, (void*)&n_list, (void*)&bo, (void*)&li, (void*)&ct, (void*)&dfp, (void*)&kp, (void*)&t0,
                      (void*)&rho_dev};
        void* ap[] = {(void*)&p, (void*)&plan->demod_m_lo, (void*)&plan->demod_nbins, (void*)&n_blk, (void*)&Rs, (void*)&zp,
                      (void*)&rp, (void*)&n_list, (void*)&sp, (void*)&dfp, (void*)&kp, (void*)&t0, (void*)&rho_dev};
        if ((e = cudaLaunchKernel(kernel(nthr), grid, dim3((unsigned)nthr), sep ? as : ap, smem, st)) != cudaSuccess)
            return cuda_fail(e, "demodulation launch");
        count_launch();
        if (ev1) cudaEventRecord(ev1, st);
    }
    e = cudaGetLastError();
    return e == cudaSuccess ? CC_OK : cuda_fail(e, "demodulation launch");
}
