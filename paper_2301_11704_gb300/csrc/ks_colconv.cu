// ks_colconv.cu -- the column form of the s-contraction: D_t (or W^-1 D_t^T W)
// applied to one real column of a curve per CTA, the whole convolution in
// registers and one CTA's shared memory (Ashtari & Schneider, arXiv 2301.11704,
// eq. rational_diff_matrix, Sec. V.C.1).
//
// D_t u is -sin^2(theta) / S times the theta-derivative q of the 2P-periodic even
// extension of the column, and -W^-1 D_t^T W r (r zero on the end rows) the same
// with the odd extension.  Both are taken from the differences of neighbouring
// sections, d_m = x_{m+1} - x_m (m < P), whose extension is odd or even about the
// midpoint:
//   q_j = sum_{m<P} (g[j-m] - s g[j+m+1]) d_m,   s = +1 (even) or -1 (odd),
//   g[l] = (1/2P) sum_{|k|<P} kappa_k cos((pi k/P)(l - 1/2)),  kappa_k = k / (2 sin(pi k/2P)).
// kappa varies only from P/pi to P/2, so rounding in the transforms stays relative
// to q; a convolution of x itself multiplies the rounding of its highest
// frequencies by P (in FP32 at N_s = 16384 the error of D_t u is 1.6e-7 this way
// and 4e-5 that way; the differences of FP32 neighbours are nearly exact).
//
// The sum is a Toeplitz and a Hankel convolution whose products have exponents in
// [-P, 2P).  Both are taken modulo x^L = i at a power of two L >= P + 1: a real
// product's exponents in [0, L) then land in the real part and those in [L, 2L)
// and [-L, 0) in the imaginary part (right-angle convolution), so no zero padding
// is needed, and as every evaluation point w_k = e^(-2 pi i (k + 1/4) / L) is on the
// unit circle the reversed sequence of a real column is the conjugate of its
// transform:
//   Y_k = T_k Z_k + s H_k conj(Z_k),   q = Re of the inverse transform,
// with Z_k = sum_m d_m w_k^m, T_k = sum_l g[l] w_k^l (-P < l <= P) and
// H_k = -sum_n g[n+1] w_k^n (0 <= n < 2P).  One complex transform of L points forward
// and one back per real column, each value Z_k used where it is (no partner at -k).
//
// Why this split: the columns are independent, so a column per CTA fills the GPU
// from N_x = 64 on, a column's working set (8 L bytes in FP32) never leaves its
// SM, and the epilogue of the descent step holds the updated sections in the
// registers the next forward transform starts from: a step's two contractions
// are one launch that reads R, A and U once and writes U and D_t u once.  The
// fields of such a curve are column-major ([W][pitch] words), so that these
// accesses are contiguous.
#include <cmath>
#include <type_traits>

#include <cooperative_groups.h>

#include "ks_rfft.cuh"

namespace ks {

namespace {

// The transform of each length (B: of batched curves).  FP32: 16 values per thread, 32
// from L = 8192 on (two exchanges instead of three: 35.7 against 43.6 us a step's
// contraction at 256 x 8000), 8 at L = 256 and 512 and for single curves up to 2048,
// which are bound by the latency of a column's chain (L = 1024: 10.7 against 12.9 us; the
// 256-curve batch, bound by throughput, takes 0.74 ms a step with 8 and 0.57 with
// 16), and 4 at L = 128, a warp.  FP64: few values, to give every quarter of an SM's FP64
// pipes a warp: 2 to 8, 16 at L = 8192.
template <typename T, int L, bool B = false>
struct CcPlan : CcPlan<T, L, false> {};
template <> struct CcPlan<float, 128, false> { using F = RegFft<float, 128, 4, true, false, 4, 4, 4, 2>; };
template <> struct CcPlan<float, 256, false> { using F = RegFft<float, 256, 8, true, false, 8, 8, 4>; };
template <> struct CcPlan<float, 512, false> { using F = RegFft<float, 512, 8, true, false, 8, 8, 8>; };
template <> struct CcPlan<float, 1024, false> { using F = RegFft<float, 1024, 8, true, false, 8, 8, 4, 4>; };
template <> struct CcPlan<float, 1024, true> { using F = RegFft<float, 1024, 16, true, false, 16, 16, 4>; };
template <> struct CcPlan<float, 2048, false> { using F = RegFft<float, 2048, 8, true, false, 8, 8, 8, 4>; };
template <> struct CcPlan<float, 2048, true> { using F = RegFft<float, 2048, 16, true, false, 16, 16, 8>; };
template <> struct CcPlan<float, 4096, false> { using F = RegFft<float, 4096, 16, true, false, 16, 16, 16>; };
template <> struct CcPlan<float, 8192, false> { using F = RegFft<float, 8192, 32, true, false, 32, 32, 8>; };
template <> struct CcPlan<float, 16384, false> { using F = RegFft<float, 16384, 32, true, false, 32, 32, 16>; };
template <> struct CcPlan<double, 128, false> { using F = RegFft<double, 128, 2, true, true, 2, 2, 2, 2, 2, 2, 2>; };
template <> struct CcPlan<double, 256, false> { using F = RegFft<double, 256, 2, true, true, 2, 2, 2, 2, 2, 2, 2, 2>; };
template <> struct CcPlan<double, 512, false> { using F = RegFft<double, 512, 4, true, true, 4, 4, 4, 4, 2>; };
template <> struct CcPlan<double, 1024, false> { using F = RegFft<double, 1024, 8, true, true, 8, 8, 4, 4>; };
template <> struct CcPlan<double, 2048, false> { using F = RegFft<double, 2048, 8, true, true, 8, 8, 8, 4>; };
template <> struct CcPlan<double, 4096, false> { using F = RegFft<double, 4096, 8, true, true, 8, 8, 8, 8>; };
template <> struct CcPlan<double, 8192, false> { using F = RegFft<double, 8192, 16, true, true, 16, 16, 8, 4>; };

// The split form (a column over a cluster of CS CTAs): the transform of one class of
// L / CS frequencies.  A warp's FP64 instruction takes about 64 cycles on its quarter
// of the SM, so the plans give every quarter a warp: 2 values per thread at 256, 4 at 512
// and 1024, 8 at 2048 and 4096.
template <int Q>
struct CxPlan;
template <> struct CxPlan<256> { using F = RegFft<double, 256, 2, true, true, 2, 2, 2, 2, 2, 2, 2, 2>; };
template <> struct CxPlan<512> { using F = RegFft<double, 512, 4, true, true, 4, 4, 4, 4, 2>; };
template <> struct CxPlan<1024> { using F = RegFft<double, 1024, 4, true, true, 4, 4, 4, 4, 4>; };
template <> struct CxPlan<2048> { using F = RegFft<double, 2048, 8, true, true, 8, 8, 8, 4>; };
template <> struct CxPlan<4096> { using F = RegFft<double, 4096, 8, true, true, 8, 8, 8, 8>; };

// fn(plan, cluster size) for the split form of length L over cs CTAs (cx_size's pairs)
template <typename Fn>
auto cx_dispatch(int L, int cs, Fn &&fn, decltype(fn(typename CxPlan<256>::F(), std::integral_constant<int, 2>())) none)
{
    const std::integral_constant<int, 2> two;
    const std::integral_constant<int, 4> four;
    switch (L / cs) {
    case 256: return cs == 2 ? fn(typename CxPlan<256>::F(), two) : fn(typename CxPlan<256>::F(), four);
    case 512: return cs == 2 ? fn(typename CxPlan<512>::F(), two) : fn(typename CxPlan<512>::F(), four);
    case 1024: return cs == 2 ? fn(typename CxPlan<1024>::F(), two) : fn(typename CxPlan<1024>::F(), four);
    case 2048: return cs == 2 ? fn(typename CxPlan<2048>::F(), two) : fn(typename CxPlan<2048>::F(), four);
    case 4096: if (cs == 2) return fn(typename CxPlan<4096>::F(), two); break;
    default: break;
    }
    return none;
}

template <typename T, bool B, typename Fn>
auto cc_dispatch(int L, Fn &&fn, decltype(fn(typename CcPlan<T, 128, B>::F())) none)
{
    switch (L) {
    case 128: return fn(typename CcPlan<T, 128, B>::F());
    case 256: return fn(typename CcPlan<T, 256, B>::F());
    case 512: return fn(typename CcPlan<T, 512, B>::F());
    case 1024: return fn(typename CcPlan<T, 1024, B>::F());
    case 2048: return fn(typename CcPlan<T, 2048, B>::F());
    case 4096: return fn(typename CcPlan<T, 4096, B>::F());
    case 8192: return fn(typename CcPlan<T, 8192, B>::F());
    case 16384:
        if constexpr (sizeof(T) == 4) return fn(typename CcPlan<T, 16384, B>::F());
        break;
    default: break;
    }
    return none;
}

// Sum of a thread's E terms w(r) g(r)^2 in FP32 storage: a compensated FP32 pair (Knuth's
// TwoSum), which keeps the sum of the FP32 terms to about 2^-46 without the FP64 pipe (its
// issue rate is a small fraction of the FP32 one).  The terms keep the range of g: w
// reaches S P / pi, so w g^2 leaves FP32's long before g^2 does.  They are scaled by the
// power of two that brings the largest g^2 to [1, 4), and the sum is scaled back in FP64.
// (Terms out of range to FP64 behind a branch took 5 to 9% of a step of the short plans,
// whose chain waits for instructions at each jump; the scaling 0 to 1.3%.)
template <int E, typename W, typename G>
__device__ __forceinline__ double sum_terms(W &&w, G &&g)
{
    float m[E];
#pragma unroll
    for (int r = 0; r < E; ++r) m[r] = fabsf(g(r));
#pragma unroll
    for (int o = E / 2; o > 0; o >>= 1)
#pragma unroll
        for (int r = 0; r < o; ++r) m[r] = fmaxf(m[r], m[r + o]);
    // the scale's exponent field: 2^(127 - e) for the field e of the largest
    const int f = max(254 - (int)(__float_as_uint(m[0]) >> 23), 1);
    const float scale = __uint_as_float((unsigned)f << 23);
    float hi = 0.f, lo = 0.f;
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const float q = g(r) * scale, t = w(r) * (q * q), s = __fadd_rn(hi, t), b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(t, b)));
        hi = s;
    }
    // (an infinite sum has no second part)
    const float inf = __int_as_float(0x7f800000);
    return __longlong_as_double((long long)(1023 + 2 * (127 - f)) << 52) * ((double)hi + (double)(fabsf(hi) < inf ? lo : 0.f));
}

// The product's factors at one frequency: with s = +1, Y = (a x + b y, c x + d y) for
// Z = (x, y), a = T.x + H.x, b = H.y - T.y, c = T.y + H.y, d = T.x - H.x; s = -1 swaps a
// with d and b with -c.
template <typename T>
struct alignas(16) SpecPair {
    cpx<T> t, h;   // (a, b), (c, d)
    __device__ __forceinline__ cpx<T> times(cpx<T> z, bool even) const
    {
        if (even) return {t.x * z.x + t.y * z.y, h.x * z.x + h.y * z.y};
        return {h.y * z.x - h.x * z.y, t.x * z.y - t.y * z.x};
    }
};
__device__ __forceinline__ SpecPair<float> ldc_spec(const SpecPair<float> *p)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return {{v.x, v.y}, {v.z, v.w}};
}
__device__ __forceinline__ SpecPair<double> ldc_spec(const SpecPair<double> *p)
{
    const double2 *q = reinterpret_cast<const double2 *>(p), t = __ldg(q), h = __ldg(q + 1);
    return {{t.x, t.y}, {h.x, h.y}};
}

// Deferred form: the FP64 reduction of a step's row phase (rows_finish in
// ks_device.cuh), by the CTA of a column that is held at zero (it has no transform to
// do): sums the row_parts partials in a fixed order, takes the convergence decision,
// publishes it in sc->decided, records the scalars and advances step, tau and lambda.
// A warp's FP64 instruction takes about 64 cycles, so the sums the decision needs come
// first and the roots and the quotient only where the tolerance asks for them; the
// record follows.  A kernel boundary used to expose all of it (4 us at N_s = 1024);
// the other CTAs' first transform covers it.
template <int NT>
__device__ __forceinline__ void cc_decide(const CurveDev &c, int tid)
{
    constexpr int FW = NT / 32 < 4 ? NT / 32 : 4;   // warps that sum
    __shared__ double red[FW][5];
    DevScalars *sc = c.sc;
    const int w = tid >> 5, lane = tid & 31, P = c.P;
    // J^2 and the two sums of J_arc
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    const double tol = sc->tol;
    const int conv = sc->conv;
    const bool withheld = sc->wait_cycles < 0;   // test hook: every column's wait runs out
    if (w < FW) {
#pragma unroll 4
        for (int b = w * 32 + lane; b < c.row_parts; b += FW * 32) {
            const double *p = c.bpart + (size_t)b * 5;
            a0 += __ldcg(p);
            a1 += __ldcg(p + 1);
            a2 += __ldcg(p + 2);
        }
        // halve the values at the first two levels: value 2 (lane bit 4) + (lane bit 3)
        const bool b4 = (lane & 16) != 0, b3 = (lane & 8) != 0;
        const double x0 = (b4 ? a2 : a0) + __shfl_xor_sync(0xffffffffu, b4 ? a0 : a2, 16);
        const double x1 = a1 + __shfl_xor_sync(0xffffffffu, a1, 16);
        double x = (b3 ? x1 : x0) + __shfl_xor_sync(0xffffffffu, b3 ? x0 : x1, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((lane & 7) == 0) red[w][lane >> 3] = x;   // 0: J^2, 1 (and 3): numerator, 2: denominator
    }
    __syncthreads();
    if (w != 0) return;
    double r = 0.0;
    if (lane < 3)
#pragma unroll
        for (int k = 0; k < FW; ++k) r += red[k][lane];
    const double j2 = __shfl_sync(0xffffffffu, r, 0), num = __shfl_sync(0xffffffffu, r, 1), den = __shfl_sync(0xffffffffu, r, 2);
    auto publish = [&](bool stop) {
        if (lane == 0 && !withheld)
            asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(&sc->decided), "r"(stop ? 2 : 1) : "memory");
    };
    // without a tolerance: finite, with no quotient (den = 0 gives J_arc = 0) unless it may overflow
    const bool quick = tol <= 0 && isfinite(j2) && (fabs(num) < 1e300 * den);
    if (quick) publish(false);
    // |l d|^2 and <d, r>
    double b0 = 0.0, b1 = 0.0;
#pragma unroll 4
    for (int b = lane; b < c.row_parts; b += 32) {
        const double *p = c.bpart + (size_t)b * 5;
        b0 += __ldcg(p + 4);
        b1 += __ldcg(p + 3);
    }
    const double d2 = warp_sum(b0), dl = warp_sum(b1);
    const double root = sqrt(lane == 1 ? d2 : j2);   // both roots at once
    const double J = __shfl_sync(0xffffffffu, root, 0), Dnorm = __shfl_sync(0xffffffffu, root, 1);
    const double Jarc = den > 0 ? num / den : 0.0, dJdl = -2.0 * dl;
    const bool bad = !isfinite(j2) || !isfinite(Jarc);
    bool done = bad;
    if (!bad && tol > 0) done = (conv == 0 ? Jarc : (conv == 1 ? J : (Dnorm > 0 ? J / Dnorm : J))) < tol;
    if (!quick) publish(done);
    if (lane != 0) return;
    const double lamd = sc->lambda_next;
    sc->J2 = j2;
    sc->Jarc = Jarc;
    sc->dJdl = dJdl;
    sc->Dnorm = Dnorm;
    sc->u2_plus = __ldcg(c.rowsc + 0);
    sc->f2_plus = __ldcg(c.rowsc + 3);
    sc->u2_minus = __ldcg(c.rowsc + 4 * (size_t)P + 0);
    sc->f2_minus = __ldcg(c.rowsc + 4 * (size_t)P + 3);
    if (bad) sc->status = 5;
    if (!done) {
        sc->lambda_next = sc->lambda_free ? lamd - sc->dtau_lambda * dJdl : lamd;
        sc->step += 1;
        sc->tau += sc->dtau;
        sc->g2_pending = 1;
    } else {
        sc->done = 1;   // (sc->active stays: the CTAs of this launch all see the same gate)
    }
}

__device__ __forceinline__ int cc_decided(const DevScalars *sc)
{
    int d;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(d) : "l"(&sc->decided) : "memory");
    return d;
}

// The wait for it where a first look (d) found none: CTA 0 decides, which starts first and
// waits for nobody; bounded all the same.  A step that is not decided in time is not
// applied and flagged as error 6; where only some columns gave up they differ by a step
// from the others, and the curve has to be initialised again.
__device__ __forceinline__ bool cc_wait(DevScalars *sc, int d)
{
    if (d == 0) {
        const long long t0 = clock64(), lim = wait_bound(*sc);
        while ((d = cc_decided(sc)) == 0 && clock64() - t0 < lim) {}
        if (d == 0) atomicExch(&sc->err, 6);
    }
    return d == 1;
}

// DEFER: a single curve's step (mode GM_STEP) after a row phase that left its reduction
// here; else GM_GRAD, GM_STORE and in a batch (BATCH) GM_STEP, with their own last-CTA
// reduction.
template <class F, bool DEFER, bool BATCH = false>
__device__ __forceinline__ void cc_body(const CurveDev &c, int mode, int discrete, int gate, int col, int ncol)
{
    using T = typename F::type;
    constexpr int E = F::E, NT = F::NT, U128 = 32 / E;   // stage-0 element r carries e^(-2 pi i r / 4E)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *buf = (cpx<T> *)smem_raw;
    __shared__ double wsum[NT / 32];
    __shared__ T edge[E * (NT / 32)];
    __shared__ int am_last;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    DevScalars *sc = c.sc;
    const cpx<T> *tw = as_global((const cpx<T> *)c.cctw);
    const SpecPair<T> *spec = as_global((const SpecPair<T> *)c.ccs);
    auto sync = [] {
        if constexpr (NT == 32) __syncwarp();
        else __syncthreads();
    };
    __shared__ int go;
    // tables by loads that the compiler may move (ahead of stores, out of the loop over the
    // contractions) or, where the registers do not hold their values early, not
    constexpr bool HOIST = DEFER && E <= 16;
    auto tab = [](const T *p) { return HOIST ? ldc(p) : *as_global(p); };
    pdl_wait();
    if ((DEFER || gate) && !sc->active) return;
    const int P = c.P, ns = c.ns;
    const size_t co = (size_t)col * c.pitch;
    T *D = as_global((T *)c.D + co), *U = as_global((T *)c.U + co), *G = as_global((T *)c.G + co);
    const T *A = as_global((const T *)c.A + co), *R = as_global((const T *)c.R + co);
    const T *wt = (const T *)c.wt, *rowscale = (const T *)c.ccr;
    const bool step = DEFER || (BATCH && mode == GM_STEP);
    double partsum = 0.0;

    // the first contraction's column: section n + 1 beside n
    const T *X = (!DEFER && mode == GM_STORE) ? U : R;
    const bool live = col_live(col, c.sym, c.hs);
    T x0[E], x1[E];
#pragma unroll
    for (int r = 0; r < E; ++r) {
        const int n = tid + NT * r;
        const bool ok = live && n < P;
        x0[r] = ok ? X[n] : T(0);
        x1[r] = ok ? X[n + 1] : T(0);
    }
    if (!live) {
        if (DEFER && col == 1 - c.hs) cc_decide<NT>(c, tid);
        // held at zero by the subspace (or the mean's imaginary part)
        if (mode == GM_STORE || step)
            for (int j = tid; j < ns; j += NT) D[j] = T(0);
        if (mode == GM_GRAD)
            for (int j = tid; j < ns; j += NT) G[j] = T(0);
    } else {
        cpx<T> v[E];
        // element r carries the quarter twist e^(-2 pi i r / 4E)
        auto put = [&](int r, T z) { v[r] = {z * cos128<T>(U128 * r), -(z * sin128<T>(U128 * r))}; };
        auto get = [&](int r) { return v[r].x * cos128<T>(U128 * r) - v[r].y * sin128<T>(U128 * r); };
        auto contract = [&](bool even, bool first) {
            F::template dif<false, HOIST>(v, buf, tw, tid, sync);
            asm volatile("" ::: "memory");   // the spectra are not loaded ahead of the transform
            // the step's decision, for the epilogue (published by the barriers of dit())
            int d = 1;
            if (DEFER && first && tid == 0) d = cc_decided(sc);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const SpecPair<T> p = HOIST ? ldc_spec(spec + e * NT + tid) : spec[e * NT + tid];
                v[e] = p.times(v[e], even);
            }
            if (DEFER && first && tid == 0) go = cc_wait(sc, d);
            F::template dit<true, HOIST>(v, buf, tw, tid, sync);
        };
#pragma unroll
        for (int r = 0; r < E; ++r) put(r, x1[r] - x0[r]);
        // epilogue operands that fit the registers are loaded across the transforms
        constexpr bool EARLY = E * sizeof(T) <= 64 && NT < 1024;
        T a[EARLY ? E : 1], u[EARLY ? E : 1];
        if (EARLY && mode != GM_STORE) {
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const int n = tid + NT * r;
                a[EARLY ? r : 0] = n < ns ? A[n] : T(0);
                u[EARLY ? r : 0] = (step && n < ns) ? U[n] : T(0);
            }
        }
        // one or two contractions (a descent step: the update, then D_t u of the updated
        // column) through the same code: unrolled into two copies it outgrew the
        // instruction caches (the warps' largest stall at L = 16384)
        bool even = !discrete;
        bool store = !DEFER && mode == GM_STORE;
#pragma unroll 1
        for (;;) {
            contract(even, !store);
            if (store) {
                constexpr int CH = E < 8 ? E : 8;   // row scales loaded a group ahead of the stores
                T rs[CH];
                auto fetch = [&](int r0) {
#pragma unroll
                    for (int i = 0; i < CH; ++i) rs[i] = tid + NT * (r0 + i) < ns ? tab(rowscale + tid + NT * (r0 + i)) : T(0);
                };
                fetch(0);
#pragma unroll
                for (int r0 = 0; r0 < E; r0 += CH) {
                    T rc[CH];
#pragma unroll
                    for (int i = 0; i < CH; ++i) rc[i] = rs[i];
                    if (r0 + CH < E) fetch(r0 + CH);
#pragma unroll
                    for (int i = 0; i < CH; ++i)
                        if (tid + NT * (r0 + i) < ns) D[tid + NT * (r0 + i)] = rc[i] * get(r0 + i);
                }
                break;
            }
            if constexpr (DEFER) {
                if (!go) return;
            }
            const T lam = (T)sc->lambda, dtp = (T)sc->dtau * ((const T *)c.prec_imex)[col_mode(col, c.hs)];
            // sections whose loads are issued together, a group ahead of the stores
            constexpr int CH = EARLY ? E : 4;
            double sum = 0.0;
            T wk[EARLY ? E : 1];
            T rs[CH], w[CH], av[CH], uv[CH];
            auto fetch = [&](int r0) {
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    const int n = tid + NT * (r0 + i);
                    const bool ok = n < ns;
                    rs[i] = ok ? tab(rowscale + n) : T(0);
                    w[i] = ok ? tab(wt + n) : T(0);
                    av[i] = EARLY ? a[EARLY ? r0 + i : 0] : (ok ? A[n] : T(0));
                    uv[i] = EARLY ? u[EARLY ? r0 + i : 0] : ((step && ok) ? U[n] : T(0));
                }
            };
            fetch(0);
#pragma unroll
            for (int r0 = 0; r0 < E; r0 += CH) {
                T rc[CH], wc[CH], ac[CH], uc[CH];
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    rc[i] = rs[i];
                    wc[i] = w[i];
                    ac[i] = av[i];
                    uc[i] = uv[i];
                }
                if (r0 + CH < E) fetch(r0 + CH);
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    const int n = tid + NT * (r0 + i), r = r0 + i;
                    const bool interior = n > 0 && n < P;
                    const T y = rc[i] * get(r);
                    const T g = interior ? -(ac[i] + lam * y) : T(0);
                    if constexpr (sizeof(T) == 8) {
                        sum += wc[i] * (g * g);
                    } else {   // v[r] has been read
                        v[r].y = g;
                        if (EARLY) wk[EARLY ? r : 0] = wc[i];
                    }
                    if (step) {
                        const T un = uc[i] + dtp * g;   // the end rows unchanged (g = 0)
                        if (interior) U[n] = un;
                        v[r].x = un;
                    } else if (n < ns) {
                        G[n] = g;
                    }
                }
            }
            if constexpr (sizeof(T) == 4) {
                auto weight = [&](int r) { return EARLY ? wk[EARLY ? r : 0] : tid + NT * r < ns ? tab(wt + tid + NT * r) : T(0); };
                sum = sum_terms<E>(weight, [&](int r) { return v[r].y; });
            }
            partsum = (col_mode(col, c.hs) == 0 ? 1.0 : 2.0) * sum;
            if (!step) break;
            // the differences of the updated column: section n + 1 is the next lane's, for a
            // warp's last lane the next warp's first (through `edge`)
            if (lane == 0) {
#pragma unroll
                for (int r = 0; r < E; ++r) edge[r * (NT / 32) + warp] = v[r].x;
            }
            sync();
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const T nx = __shfl_down_sync(0xffffffffu, v[r].x, 1);
                const int q = r * (NT / 32) + warp + 1;
                const T up = lane < 31 ? nx : (q < E * (NT / 32) ? edge[q] : T(0));
                put(r, tid + NT * r < P ? up - v[r].x : T(0));
            }
            even = true;
            store = true;
        }
    }
    if (!DEFER && mode == GM_STORE) return;

    // ---- FP64 |G|^2: a partial per column, summed in column order by the last CTA or,
    // deferred, beside the next row phase
    partsum = warp_sum(partsum);
    if constexpr (DEFER) {   // a partial per warp
        if (lane == 0) c.tile[col * (NT / 32) + warp] = partsum;
        return;
    }
    if (lane == 0) wsum[warp] = partsum;
    sync();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < NT / 32; ++w) t += wsum[w];
        c.tile[col] = t;
    }
    if (!last_cta_arrive(&sc->cnt_gemm, (unsigned)ncol, am_last)) return;
    if (warp == 0) {
        double t = 0.0;
        for (int b = lane; b < ncol; b += 32) t += __ldcg(c.tile + b);
        t = warp_sum(t);
        if (lane == 0) {
            sc->G2 = c.L * t;
            if (step) {
                sc->step += 1;
                sc->tau += sc->dtau;
                sc->lambda = sc->lambda_next;
            }
            sc->cnt_gemm = 0;
        }
    }
}

// Bound: at few sections the chain of a column's stages and their barriers (N_x = 64,
// N_s = 1024 FP32, both contractions of a step and its reduction: 10.8 us, where the
// clustered four-step kernel took 21.3); at many, issue slots (N_x = 256, N_s = 16384:
// 70 us, half of the issue slots used, FMA pipe 35%, 50 MB read from DRAM where the
// three-launch form took 132 + 69 us); in FP64 the FP64 pipes (83% busy in a batch).
// Up to 128 registers a thread: at 32 values per thread the transform's 64 registers
// of data, its twiddles and the epilogue about fit.
template <class F, bool DEFER>
__global__ void __launch_bounds__(F::NT, F::NT >= 512 ? 1 : 512 / F::NT)
    k_cc(const __grid_constant__ CurveDev c, int mode, int discrete, int gate)
{
    // CTA 0 takes the column held at zero (1, the imaginary part of the mean; in sine
    // storage 0, the mean), whose CTA decides in the deferred form
    const int b = blockIdx.x, col = c.hs || b > 1 ? b : 1 - b;
    cc_body<F, DEFER>(c, mode, discrete, gate, col, gridDim.x);
}

// ---- the split form: a column over a cluster of CS CTAs.  CTA `rank` takes the class
// of frequencies CS k + rank, a transform of Q = L / CS points of the column folded
// into them,
//   z_rank[n] = sum_p d[n + p Q] e^(-2 pi i phi (n + p Q) / Q),  phi = (4 rank + 1) / 4 CS,  n < Q,
// and owns the sections [rank Q, (rank + 1) Q): the classes' parts of q at n + p Q go to
// CTA p through distributed shared memory, the updated sections to every CTA.  For
// FP64 curves of few columns, whose CTAs would leave most SMs idle while each is
// bound by its FP64 pipes: N_x = 64, N_s = 552 over two CTAs a step in 45 us, over one
// in 64 (143 before the column form); the pipes of the SMs in use are then 77% busy.
// DEFER: a step (mode GM_STEP); else GM_GRAD or GM_STORE.
template <class F, int CS>
constexpr size_t cx_bytes() { return F::BYTES + ((size_t)(CS - 1) * F::L + CS * F::L + 1) * sizeof(typename F::type); }

template <class F, int CS, bool DEFER>
__global__ void __launch_bounds__(F::NT) k_cx(const __grid_constant__ CurveDev c, int mode, int discrete, int gate)
{
    namespace cg = cooperative_groups;
    using T = typename F::type;
    constexpr int E = F::E, NT = F::NT, Q = F::L;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *buf = (cpx<T> *)smem_raw;
    T *xb = (T *)(smem_raw + F::BYTES), *ub = xb + (CS - 1) * Q;   // the other classes' parts; the updated column
    __shared__ double wsum[NT / 32];
    __shared__ int go, am_last;
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = blockIdx.x / CS, rank = blockIdx.x % CS, col = c.hs || b > 1 ? b : 1 - b, ncta = gridDim.x;
    DevScalars *sc = c.sc;
    auto sync = [] { __syncthreads(); };
    auto barrier = [] {   // release / acquire over the cluster
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    };
    pdl_wait();
    if ((DEFER || gate) && !sc->active) return;   // the same for the whole grid
    const int P = c.P, ns = c.ns;
    const size_t co = (size_t)col * c.pitch;
    T *D = as_global((T *)c.D + co), *U = as_global((T *)c.U + co), *G = as_global((T *)c.G + co);
    const T *A = as_global((const T *)c.A + co), *R = as_global((const T *)c.R + co);
    const T *wt = as_global((const T *)c.wt), *rowscale = as_global((const T *)c.ccr);
    const cpx<T> *tw = as_global((const cpx<T> *)c.cctw + (size_t)rank * F::TW);
    const SpecPair<T> *spec = as_global((const SpecPair<T> *)c.ccs + (size_t)rank * Q);
    double partsum = 0.0;

    if (!col_live(col, c.sym, c.hs)) {   // held at zero (the whole cluster)
        if (DEFER && rank == 0 && col == 1 - c.hs) cc_decide<NT>(c, tid);
        if (DEFER || mode == GM_STORE)
            for (int j = rank * NT + tid; j < ns; j += CS * NT) D[j] = T(0);
        if (mode == GM_GRAD)
            for (int j = rank * NT + tid; j < ns; j += CS * NT) G[j] = T(0);
    } else {
        // every CTA of the cluster has started, before the first remote write
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        const T *X = (!DEFER && mode == GM_STORE) ? U : R;
        T d[CS][E];
#pragma unroll
        for (int p = 0; p < CS; ++p)
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const int n = tid + NT * r + Q * p;
                d[p][r] = n < P ? X[n + 1] - X[n] : T(0);
            }
        const int n0 = rank * Q + tid;   // this thread's sections: n0 + NT r
        T a[E], u[E];
        if (mode != GM_STORE) {
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const int n = n0 + NT * r;
                a[r] = n < ns ? A[n] : T(0);
                u[r] = (DEFER && n < ns) ? U[n] : T(0);
            }
        }
        cpx<T> v[E];
        auto by_rank = [&](auto &&f) {   // f(the class as a constant)
            if (rank == 0) f(std::integral_constant<int, 0>());
            else if (rank == 1) f(std::integral_constant<int, 1>());
            else if constexpr (CS > 2) {
                if (rank == 2) f(std::integral_constant<int, 2>());
                else f(std::integral_constant<int, 3>());
            }
        };
        bool even = !discrete, store = !DEFER && mode == GM_STORE, first = true;
#pragma unroll 1
        for (;;) {
            by_rank([&](auto rk) {
                constexpr int U128 = 32 * (4 * decltype(rk)::value + 1) / (CS * E);
                static_assert(U128 * CS * E == 32 * (4 * decltype(rk)::value + 1), "the twists are multiples of 1/128 turn");
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    v[r] = {T(0), T(0)};
#pragma unroll
                    for (int p = 0; p < CS; ++p) {
                        v[r].x += d[p][r] * cos128<T>(U128 * (r + E * p));
                        v[r].y -= d[p][r] * sin128<T>(U128 * (r + E * p));
                    }
                }
            });
            F::template dif<false>(v, buf, tw, tid, sync);
            int dec = 1;
            if (DEFER && first && rank == 0 && tid == 0) dec = cc_decided(sc);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const SpecPair<T> p = spec[e * NT + tid];
                v[e] = p.times(v[e], even);
            }
            F::template dit<true>(v, buf, tw, tid, sync);
            if (first) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (DEFER && first && rank == 0 && tid == 0) {
                // one answer for the cluster: no CTA leaves while another writes to it
                const int answer = cc_wait(sc, dec);
                for (int p = 0; p < CS; ++p) *cluster.map_shared_rank(&go, p) = answer;
            }
            // this class's part of q at its own sections, and at the others' to their CTAs
            T y[E];
            by_rank([&](auto rk) {
                constexpr int C = decltype(rk)::value, U128 = 32 * (4 * C + 1) / (CS * E);
#pragma unroll
                for (int p = 0; p < CS; ++p) {
                    T *dst = p == C ? nullptr : cluster.map_shared_rank(xb, p) + (C < p ? C : C - 1) * Q;
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        const T q = v[r].x * cos128<T>(U128 * (r + E * p)) - v[r].y * sin128<T>(U128 * (r + E * p));
                        if (p == C) y[r] = q;
                        else dst[tid + NT * r] = q;
                    }
                }
            });
            barrier();
            if (DEFER && first && !go) return;
#pragma unroll
            for (int r = 0; r < E; ++r) {
#pragma unroll
                for (int q = 0; q < CS - 1; ++q) y[r] += xb[q * Q + tid + NT * r];
                const int n = n0 + NT * r;
                y[r] *= n < ns ? rowscale[n] : T(0);
            }
            if (store) {
#pragma unroll
                for (int r = 0; r < E; ++r)
                    if (n0 + NT * r < ns) D[n0 + NT * r] = y[r];
                break;
            }
            const T lam = (T)sc->lambda, dtp = (T)sc->dtau * ((const T *)c.prec_imex)[col_mode(col, c.hs)];
            double sum = 0.0;
#pragma unroll
            for (int r = 0; r < E; ++r) {
                const int n = n0 + NT * r;
                const bool interior = n > 0 && n < P;
                const T g = interior ? -(a[r] + lam * y[r]) : T(0);
                sum += (n < ns ? wt[n] : T(0)) * (g * g);
                if (DEFER) {
                    u[r] += dtp * g;   // the end rows unchanged (g = 0)
                    if (interior) U[n] = u[r];
                } else if (n < ns) {
                    G[n] = g;
                }
            }
            partsum = (col_mode(col, c.hs) == 0 ? 1.0 : 2.0) * sum;
            if constexpr (!DEFER) break;
#pragma unroll
            for (int p = 0; p < CS; ++p) {
                T *dst = cluster.map_shared_rank(ub, p);
#pragma unroll
                for (int r = 0; r < E; ++r) dst[n0 + NT * r] = u[r];
            }
            barrier();
#pragma unroll
            for (int p = 0; p < CS; ++p)
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    const int n = tid + NT * r + Q * p;
                    d[p][r] = n < P ? ub[n + 1] - ub[n] : T(0);
                }
            even = true;
            store = true;
            first = false;
        }
    }
    if (!DEFER && mode == GM_STORE) return;
    partsum = warp_sum(partsum);
    if constexpr (DEFER) {
        if (lane == 0) c.tile[(col * CS + rank) * (NT / 32) + warp] = partsum;
        return;
    }
    if (lane == 0) wsum[warp] = partsum;
    __syncthreads();
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < NT / 32; ++w) t += wsum[w];
        c.tile[col * CS + rank] = t;
    }
    if (!last_cta_arrive(&sc->cnt_gemm, (unsigned)ncta, am_last)) return;
    if (warp == 0) {
        double t = 0.0;
        for (int k = lane; k < ncta; k += 32) t += __ldcg(c.tile + k);
        t = warp_sum(t);
        if (lane == 0) {
            sc->G2 = c.L * t;
            sc->cnt_gemm = 0;
        }
    }
}

// Batched curves: work item (curve, column) per CTA, the curves of one length.  A step
// of the 256-curve batch (N_x 32 to 128, N_s 256 to 2048), contractions and row phase:
// FP32 0.555 ms (1.49 with the four-step form), bound by issue slots and shared memory;
// FP64 11.6 ms (17.1), by the FP64 pipes.
template <class F>
__global__ void __launch_bounds__(F::NT, F::NT >= 512 ? 1 : 512 / F::NT) k_cc_batch(const CurveDev *cv, const int2 *items,
                                                                                    int mode, int discrete, int gate)
{
    const int2 it = items[blockIdx.x];
    const CurveDev &c = cv[it.x];
    cc_body<F, false, true>(c, mode, discrete, gate, it.y, c.W);
}

__global__ void k_cc_finish(const __grid_constant__ CurveDev c)
{
    finish_g2(c, 256);
    if (threadIdx.x == 0) c.sc->lambda = c.sc->lambda_next;
}

// ---- set-up: twiddles, and the spectra T_k and H_k (with the inverse transform's
// 1/L) in the order dif() leaves, in FP64.  With L = A B, n = B n1 + n2 and
// k = k1 + A k2 the sum over n splits into A terms and B terms per value:
//   S[k1][n2] = w^(n2 (k1 + 1/4)) sum_n1 f[B n1 + n2] e^(-2 pi i n1 (k1 + 1/4) / A)
//   X[k1 + A k2] = sum_n2 S[k1][n2] e^(-2 pi i n2 k2 / B)
// of the kernel f folded modulo x^L = i (exponents n + L times -i, n - L times i).

// g[0 .. 2P] (FP64, in the physical scratch) is the running sum of the even
// extension's derivative kernel, g[l+1] - g[l] = (-1)^l cot(pi l / 2P) / 2 (g[1] = g[0]),
// up to a constant that follows from sum_{l<2P} g[l] = kappa_0 = P / pi; g[1 - l] = g[l].
// First the increments and the other tables (row scales -sin^2(theta) / S and, for
// FP32 storage, the quadrature weights in it), then the sum by one CTA.
// Set-up kernels run over curves: one (by value), or the batch's (blockIdx.y).
struct CurveSet {
    CurveDev one;
    const CurveDev *many;   // with `index`: the curves of one length
    const int *index;
    __device__ const CurveDev &get() const { return many ? many[index ? index[blockIdx.y] : blockIdx.y] : one; }
    CurveSet from(int o) const { return {one, many && !index ? many + o : many, index ? index + o : index}; }
};
constexpr int GRID_Y = 32768;   // curves per launch

template <typename T>
__global__ void __launch_bounds__(256) k_cc_tables(const __grid_constant__ CurveSet cs)
{
    const CurveDev &c = cs.get();
    if (!c.cc) return;
    const int P = c.P;
    double *g = (double *)c.X;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < c.ns; i += gridDim.x * blockDim.x) {
        const bool end = i == 0 || i == P;
        double s, co;
        sincospi((double)i / (2.0 * P), &s, &co);
        if (i < P) g[i + 1] = i ? (i & 1 ? -0.5 : 0.5) * co / s : 0.0;   // g[i+1] - g[i]
        sincospi((double)i / (double)P, &s, &co);
        ((T *)c.ccr)[i] = end ? T(0) : (T)(-s * s / c.S);
        if (sizeof(T) == 4) ((T *)c.wt)[i] = end ? T(0) : (T)((M_PI / (double)P) * c.S / (s * s));
    }
}

__global__ void __launch_bounds__(1024) k_cc_kernel(const __grid_constant__ CurveSet cs)
{
    const CurveDev &c = cs.get();
    if (!c.cc) return;
    __shared__ double wpre[32], wtot[32];
    const int P = c.P, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ch = (P + 1023) / 1024, q0 = 1 + tid * ch, q1 = min(P + 1, q0 + ch);
    double *g = (double *)c.X;
    double a = 0.0;
    for (int q = q0; q < q1; ++q) a += g[q];
    // exclusive sums over the threads: within the warp, then over the warps
    double inc = a;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) wpre[warp] = inc;
    __syncthreads();
    double base = 0.0;
    for (int w = 0; w < warp; ++w) base += wpre[w];
    double v = base + (inc - a), sum = 0.0;
    for (int q = q0; q < q1; ++q) {
        v += g[q];
        g[q] = v;
        sum += v;
    }
    sum = warp_sum(sum);
    if (lane == 0) wtot[warp] = sum;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < 32; ++w) t += wtot[w];
    const double c0 = (P / M_PI - 2.0 * t) / (2.0 * P);
    for (int q = q0; q < q1; ++q) {
        const double x = g[q] + c0;
        g[q] = x;
        g[2 * P + 1 - q] = x;
        if (q == 1) g[0] = x;
    }
}

__global__ void __launch_bounds__(256) k_cc_specA(const __grid_constant__ CurveSet cs, int L, int A)
{
    const CurveDev &c = cs.get();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *wA = (double2 *)smem_raw;   // e^(-2 pi i p / 4A), p < 4A
    for (int p = threadIdx.x; p < 4 * A; p += blockDim.x) {
        double s, co;
        sincospi(2.0 * (double)p / (double)(4 * A), &s, &co);
        wA[p] = make_double2(co, -s);
    }
    __syncthreads();
    const int B = L / A, P = c.P, twoP = 2 * P;
    const double *g = (const double *)c.X;
    double2 *S = (double2 *)c.ccx;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2 * L) return;
    const int kind = idx / L, k1 = (idx % L) / B, n2 = idx % B;
    double re = 0.0, im = 0.0;
    for (int n1 = 0; n1 < A; ++n1) {
        const int n = B * n1 + n2;
        double gr = 0.0, gi = 0.0;
        if (kind == 0) {   // Toeplitz: lags n <= P, and n - L > -P (g[n - L] = g[1 + L - n])
            if (n <= P) gr = g[n];
            if (n > L - P) gi = g[1 + L - n];
        } else {           // Hankel: n and n + L below 2P
            if (n < twoP) gr = -g[n + 1];
            if (n + L < twoP) gi = g[n + L + 1];
        }
        const double2 w = wA[(n1 * (4 * k1 + 1)) & (4 * A - 1)];
        re += gr * w.x - gi * w.y;
        im += gr * w.y + gi * w.x;
    }
    double s, co;
    sincospi(2.0 * (double)((long long)n2 * (4 * k1 + 1)) / (4.0 * (double)L), &s, &co);
    S[(size_t)kind * L + (size_t)k1 * B + n2] = make_double2(re * co + im * s, im * co - re * s);
}

template <class F, int CS>
__global__ void __launch_bounds__(256) k_cc_specB(const __grid_constant__ CurveSet cs, int A)
{
    const CurveDev &c = cs.get();
    using T = typename F::type;
    constexpr int L = F::L * CS;   // CS classes of F::L frequencies
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *wB = (double2 *)smem_raw;   // e^(-2 pi i p / B)
    const int B = L / A;
    for (int p = threadIdx.x; p < B; p += blockDim.x) {
        double s, co;
        sincospi(2.0 * (double)p / (double)B, &s, &co);
        wB[p] = make_double2(co, -s);
    }
    __syncthreads();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < L) {
        const int rank = idx / F::L, e = (idx % F::L) / F::NT, t = idx % F::NT;
        const int k = CS * F::freq(t, e) + rank, k1 = k % A, k2 = k / A;
        const double2 *S = (const double2 *)c.ccx + (size_t)k1 * B;
        double2 x[2];
#pragma unroll
        for (int kind = 0; kind < 2; ++kind) {
            double re = 0.0, im = 0.0;
            for (int n2 = 0; n2 < B; ++n2) {
                const double2 w = wB[(n2 * k2) & (B - 1)], y = S[(size_t)kind * L + n2];
                re += y.x * w.x - y.y * w.y;
                im += y.x * w.y + y.y * w.x;
            }
            x[kind] = make_double2(re / L, im / L);
        }
        SpecPair<T> o;   // T in x[0], H in x[1]
        o.t = {(T)(x[0].x + x[1].x), (T)(x[1].y - x[0].y)};
        o.h = {(T)(x[0].y + x[1].y), (T)(x[0].x - x[1].x)};
        ((SpecPair<T> *)c.ccs)[rank * F::L + e * F::NT + t] = o;
    }
    if (idx < F::TW * CS) {
        long long num, den;
        F::tw_entry(idx % F::TW, idx / F::TW, CS, num, den);
        double s, co;
        sincospi(2.0 * (double)num / (double)den, &s, &co);
        ((cpx<T> *)c.cctw)[idx] = {(T)co, (T)(-s)};
    }
}


template <typename... KArgs, typename... Args>
cudaError_t cc_launch(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, kern, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t setup_tables(const CurveSet &cs, int n, int ns_max, cudaStream_t st)
{
    for (int o = 0; o < n; o += GRID_Y) {
        const CurveSet part = cs.from(o);
        const int k = n - o < GRID_Y ? n - o : GRID_Y;
        k_cc_tables<T><<<dim3((ns_max + 255) / 256, k), 256, 0, st>>>(part);
        k_cc_kernel<<<dim3(1, k), 1024, 0, st>>>(part);
    }
    return cudaGetLastError();
}

template <class F, int CS>
cudaError_t setup_spectra(const CurveSet &cs, int nc, cudaStream_t st)
{
    constexpr int L = F::L * CS;
    int A = 1;
    while (A * A < L) A <<= 1;
    const int B = L / A, n = L > F::TW * CS ? L : F::TW * CS;
    for (int o = 0; o < nc; o += GRID_Y) {
        const CurveSet part = cs.from(o);
        const int k = nc - o < GRID_Y ? nc - o : GRID_Y;
        k_cc_specA<<<dim3((2 * L + 255) / 256, k), 256, (size_t)4 * A * sizeof(double2), st>>>(part, L, A);
        k_cc_specB<F, CS><<<dim3((n + 255) / 256, k), 256, (size_t)B * sizeof(double2), st>>>(part, A);
    }
    return cudaGetLastError();
}

template <typename T>
cudaError_t setup_t(const CurveDev &c, cudaStream_t st)
{
    const CurveSet cs = {c, nullptr, nullptr};
    cudaError_t e = setup_tables<T>(cs, 1, c.ns, st);
    if (e != cudaSuccess) return e;
    if (c.ccl > 1)
        return cx_dispatch(
            c.cc, c.ccl, [&](auto f, auto k) { return setup_spectra<decltype(f), decltype(k)::value>(cs, 1, st); },
            cudaErrorInvalidValue);
    return cc_dispatch<T, false>(c.cc, [&](auto f) { return setup_spectra<decltype(f), 1>(cs, 1, st); }, cudaErrorInvalidValue);
}

cudaError_t run_cx(const CurveDev &c, int mode, int discrete, int gate, cudaStream_t st)
{
    return cx_dispatch(
        c.cc, c.ccl,
        [&](auto f, auto cs) {
            using F = decltype(f);
            constexpr int CS = decltype(cs)::value;
            const auto kern = c.defer && mode == GM_STEP ? k_cx<F, CS, true> : k_cx<F, CS, false>;
            cudaError_t e = set_smem(kern, cx_bytes<F, CS>());
            if (e != cudaSuccess) return e;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(c.W * CS);
            cfg.blockDim = dim3(F::NT);
            cfg.dynamicSmemBytes = cx_bytes<F, CS>();
            cfg.stream = st;
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[0].val.programmaticStreamSerializationAllowed = 1;
            attr[1].id = cudaLaunchAttributeClusterDimension;
            attr[1].val.clusterDim.x = CS;
            attr[1].val.clusterDim.y = 1;
            attr[1].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 2;
            e = cudaLaunchKernelEx(&cfg, kern, c, mode, discrete, gate);
            return e != cudaSuccess ? e : cudaGetLastError();
        },
        cudaErrorInvalidValue);
}

template <typename T>
cudaError_t run_t(const CurveDev &c, int mode, int discrete, int gate, cudaStream_t st)
{
    return cc_dispatch<T, false>(
        c.cc,
        [&](auto f) {
            using F = decltype(f);
            const bool defer = c.defer && mode == GM_STEP;
            const auto kern = defer ? k_cc<F, true> : k_cc<F, false>;
            const cudaError_t e = set_smem(kern, F::BYTES);
            if (e != cudaSuccess) return e;
            return cc_launch(kern, c.W, F::NT, F::BYTES, st, c, mode, discrete, gate);
        },
        cudaErrorInvalidValue);
}

template <typename T>
cudaError_t batch_t(int L, const CurveDev *cv, const int2 *items, int nitems, int mode, int discrete, int gate,
                    cudaStream_t st)
{
    return cc_dispatch<T, true>(
        L,
        [&](auto f) {
            using F = decltype(f);
            const cudaError_t e = set_smem(k_cc_batch<F>, F::BYTES);
            if (e != cudaSuccess) return e;
            return cc_launch(k_cc_batch<F>, nitems, F::NT, F::BYTES, st, cv, items, mode, discrete, gate);
        },
        cudaErrorInvalidValue);
}

}  // namespace

size_t cc_twiddles(int L, int prec, int cs, int batched)
{
    if (cs > 1) return cx_dispatch(L, cs, [](auto f, auto) { return (size_t)decltype(f)::TW; }, (size_t)0) * cs;
    const auto n = [](auto f) { return (size_t)decltype(f)::TW; };
    if (batched) return prec ? cc_dispatch<float, true>(L, n, (size_t)0) : cc_dispatch<double, true>(L, n, (size_t)0);
    return prec ? cc_dispatch<float, false>(L, n, (size_t)0) : cc_dispatch<double, false>(L, n, (size_t)0);
}

int cc_warps(int L, int prec, int cs)
{
    if (cs > 1) return cx_dispatch(L, cs, [](auto f, auto) { return decltype(f)::NT / 32; }, 0) * cs;
    const auto n = [](auto f) { return decltype(f)::NT / 32; };
    return prec ? cc_dispatch<float, false>(L, n, 0) : cc_dispatch<double, false>(L, n, 0);
}

cudaError_t launch_setup_cc(const CurveDev &c, cudaStream_t st)
{
    return c.prec ? setup_t<float>(c, st) : setup_t<double>(c, st);
}

cudaError_t launch_setup_cc_tables(int prec, const CurveDev *cv, int nb, int ns_max, cudaStream_t st)
{
    const CurveSet cs = {CurveDev{}, cv, nullptr};
    return prec ? setup_tables<float>(cs, nb, ns_max, st) : setup_tables<double>(cs, nb, ns_max, st);
}

cudaError_t launch_setup_cc_spectra(int prec, int L, const CurveDev *cv, const int *index, int n, cudaStream_t st)
{
    const CurveSet cs = {CurveDev{}, cv, index};
    auto run = [&](auto f) { return setup_spectra<decltype(f), 1>(cs, n, st); };
    return prec ? cc_dispatch<float, true>(L, run, cudaErrorInvalidValue) : cc_dispatch<double, true>(L, run, cudaErrorInvalidValue);
}

cudaError_t launch_cc(const CurveDev &c, int mode, int discrete, int gate, cudaStream_t st)
{
    // a single curve's step is deferred (the implicit scheme has GM_GRAD in its place)
    if (mode != GM_GRAD && mode != GM_STORE && !(mode == GM_STEP && c.defer)) return cudaErrorInvalidValue;
    if (c.ccl > 1) return run_cx(c, mode, discrete, gate, st);
    return c.prec ? run_t<float>(c, mode, discrete, gate, st) : run_t<double>(c, mode, discrete, gate, st);
}

cudaError_t launch_cc_finish(const CurveDev &c, cudaStream_t st)
{
    k_cc_finish<<<1, 256, 0, st>>>(c);
    return cudaGetLastError();
}

cudaError_t launch_cc_batch(int prec, int L, const CurveDev *cv, const int2 *items, int nitems, int mode, int discrete,
                            int gate, cudaStream_t st)
{
    if (nitems <= 0) return cudaSuccess;
    return prec ? batch_t<float>(L, cv, items, nitems, mode, discrete, gate, st)
                : batch_t<double>(L, cv, items, nitems, mode, discrete, gate, st);
}

}  // namespace ks
