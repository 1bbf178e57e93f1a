// ks_rows_cm.cu -- the x-direction kernels of curves whose fields are column-major
// ([W][pitch] words of the storage type, the layout of the column form of the
// s-contraction, ks_colconv.cu): the row phase of one evaluation (Ashtari &
// Schneider, arXiv 2301.11704, eq. KSE, eq. KSE_residual, eq. KSE_G; the formulas
// stand beside rows_body in ks_device.cuh) and the transforms between physical
// curves ([N_s][N], row-major) and spectral fields.
//
// A CTA takes SEC consecutive sections.  Their tiles of the fields come in as
// runs of SEC words per column (64 bytes at 16 FP32 or 8 FP64 sections) and go out
// the same way, through a padded [section][word] tile in shared memory whose
// column accesses and row accesses both fall in distinct banks.  Two real sections
// are packed into one complex transform of N points, held by N / E threads in
// registers (ks_rfft.cuh): the physical section u stays in registers between the
// products, and a transform crosses shared memory once to three times.
//
// Bound: at few sections the chain of a warp (N = 64, N_s = 1024 FP32 8.5 us alone, the
// row-major warp transforms 12.8; N = 128, N_s = 4096 10.8 and 18.0); at many, the
// shared-memory pipe and the round trips to memory between its phases (N = 256,
// N_s = 16384 36 us and 66, 67 MB of fields at 1.9 TB/s); in FP64 the FP64 pipes (N = 64,
// N_s = 4096 42 us and 64).
#include <type_traits>

#include "ks_dfloat.cuh"
#include "ks_rfft.cuh"

namespace ks {

namespace {

// V = 0: the plan of batches and of single curves that fill the chip with it; V = 1, 2:
// fewer values per thread, for single curves of few sections (cm_warps, cm_spread).
// V = 0 at N = 128 in FP32: 8 values, 16 were slower at every size (a step with 8 and
// with 16: 17.0 and 20.2 us at N_s = 4096, 47.9 and 49.7 at 16384, a batch of 256 curves
// 0.555 and 0.567 ms).
template <typename T, int N, int V = 0>
struct RowFft;
template <> struct RowFft<float, 8> { using F = RegFft<float, 8, 2, false, true, 2, 2, 2>; };
template <> struct RowFft<float, 16> { using F = RegFft<float, 16, 4, false, true, 4, 4>; };
template <> struct RowFft<float, 32> { using F = RegFft<float, 32, 8, false, true, 8, 4>; };
template <> struct RowFft<float, 64> { using F = RegFft<float, 64, 8, false, true, 8, 8>; };
template <> struct RowFft<float, 128> { using F = RegFft<float, 128, 8, false, true, 8, 8, 2>; };
template <> struct RowFft<float, 256> { using F = RegFft<float, 256, 16, false, true, 16, 16>; };
template <> struct RowFft<float, 32, 1> { using F = RegFft<float, 32, 2, false, true, 2, 2, 2, 2, 2>; };
template <> struct RowFft<float, 64, 1> { using F = RegFft<float, 64, 2, false, true, 2, 2, 2, 2, 2, 2>; };
template <> struct RowFft<float, 128, 1> { using F = RegFft<float, 128, 4, false, true, 4, 4, 4, 2>; };
template <> struct RowFft<float, 256, 1> { using F = RegFft<float, 256, 8, false, true, 8, 8, 4>; };
template <> struct RowFft<float, 32, 2> { using F = RegFft<float, 32, 4, false, true, 4, 4, 2>; };
template <> struct RowFft<float, 64, 2> { using F = RegFft<float, 64, 4, false, true, 4, 4, 4>; };
// FP64, N = 32 to 128: 4 values per thread: a warp's FP64 instruction holds its pipe for
// about 64 cycles whatever the size of the curve, so the work is spread over warps
template <> struct RowFft<double, 32> { using F = RegFft<double, 32, 4, false, true, 4, 4, 2>; };
template <> struct RowFft<double, 64> { using F = RegFft<double, 64, 4, false, true, 4, 4, 4>; };
template <> struct RowFft<double, 128> { using F = RegFft<double, 128, 4, false, true, 4, 4, 4, 2>; };
// and 2 where there is less than a warp per pipe with 4 (a third of the steps of a
// pair's chain, a fifth more instructions in all)
template <> struct RowFft<double, 32, 1> { using F = RegFft<double, 32, 2, false, true, 2, 2, 2, 2, 2>; };
template <> struct RowFft<double, 64, 1> { using F = RegFft<double, 64, 2, false, true, 2, 2, 2, 2, 2, 2>; };
// double-float, and the FP64 lengths not listed above: 2, 4 and from N = 32 on 8 values
// per thread
template <typename T> struct RowFft<T, 8> { using F = RegFft<T, 8, 2, false, true, 2, 2, 2>; };
template <typename T> struct RowFft<T, 16> { using F = RegFft<T, 16, 4, false, true, 4, 4>; };
template <typename T> struct RowFft<T, 32> { using F = RegFft<T, 32, 8, false, true, 8, 4>; };
template <typename T> struct RowFft<T, 64> { using F = RegFft<T, 64, 8, false, true, 8, 8>; };
template <typename T> struct RowFft<T, 128> { using F = RegFft<T, 128, 8, false, true, 8, 8, 2>; };
template <typename T> struct RowFft<T, 256> { using F = RegFft<T, 256, 8, false, true, 8, 8, 4>; };

// Shared-memory plan of a CTA of SEC sections: the transform's twiddles, the
// exchange buffers of its section pairs, NTILE tiles [SEC][N + 2].
template <typename Tc, typename Ts, int N, int SEC, int V = 0>
struct CmCfg {
    using F = typename RowFft<Tc, N, V>::F;
    static constexpr int E = F::E, LPS = F::NT, PAIRS = SEC / 2, NTHR = PAIRS * LPS, HE = E / 2, TS = N + 2;
    static_assert(NTHR >= 32, "whole warps");
    // the buffers of the pairs of one wavefront (128 bytes) in distinct banks
    static constexpr int WAVE = 128 / (int)sizeof(cpx<Tc>);
    static constexpr int BUFS = F::BUF + ((LPS < WAVE ? LPS : 0) - F::BUF % WAVE + WAVE) % WAVE;
    static constexpr size_t TWB = (size_t)F::TW * sizeof(cpx<Tc>), BUFB = (size_t)PAIRS * BUFS * sizeof(cpx<Tc>),
                            TILE = ((size_t)SEC * TS * sizeof(Ts) + 15) / 16 * 16;
    static constexpr size_t bytes(int tiles) { return (TWB + 15) / 16 * 16 + (BUFB + 15) / 16 * 16 + tiles * TILE; }
    static __device__ __forceinline__ cpx<Tc> *tw(unsigned char *s) { return (cpx<Tc> *)s; }
    static __device__ __forceinline__ cpx<Tc> *buf(unsigned char *s) { return (cpx<Tc> *)(s + (TWB + 15) / 16 * 16); }
    static __device__ __forceinline__ Ts *tile(unsigned char *s, int i)
    {
        return (Ts *)(s + (TWB + 15) / 16 * 16 + (BUFB + 15) / 16 * 16 + i * TILE);
    }
};

// The twiddle tables of the stages from e^(-2 pi i t / N), given as w(t) for t < N / 2.
template <class F, int N, int NTHR, int I = 0, typename W>
__device__ __forceinline__ void row_twiddles(cpx<typename F::type> *tw, W &&w)
{
    if constexpr (I + 1 < F::NST) {
        for (int e = threadIdx.x; e < F::rad(I) * F::lr(I); e += NTHR) {
            const int t = ((e / F::lr(I)) * (e % F::lr(I)) * (N / F::sub(I))) & (N - 1);
            cpx<typename F::type> v = w(t & (N / 2 - 1));
            if (t >= N / 2) v = {-v.x, -v.y};
            tw[F::tw_off(I) + e] = v;
        }
        row_twiddles<F, N, NTHR, I + 1>(tw, w);
    }
}

template <typename T>
struct alignas(16) Vec16 {
    static constexpr int CW = 16 / (int)sizeof(T);
    T v[CW];
};

// A tile's 16-byte chunks (CW sections of one column): item i of a thread is chunk
// (tid + NTHR i) % CPC of column (tid + NTHR i) / CPC.
template <typename T, int N, int SEC, int NTHR>
struct CmTile {
    static constexpr int CW = Vec16<T>::CW, CPC = SEC / CW, ITEMS = (N * CPC + NTHR - 1) / NTHR, TS = N + 2;
    Vec16<T> x[ITEMS];
    __device__ __forceinline__ void fetch(const T *f, int pitch, int W, int m0)
    {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = threadIdx.x + NTHR * i, col = e / CPC;
            if (col < W) x[i] = *reinterpret_cast<const Vec16<T> *>(f + (size_t)col * pitch + m0 + (e % CPC) * CW);
        }
    }
    // into the tile; the sections past the curve as zeros (their words in the pitch are not set)
    __device__ __forceinline__ void put(T *tile, int W, int hs, int m0, int ns) const
    {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = threadIdx.x + NTHR * i, col = e / CPC, s0 = (e % CPC) * CW;
            if (col >= W) continue;
#pragma unroll
            for (int q = 0; q < CW; ++q) {
                const T v = m0 + s0 + q < ns ? x[i].v[q] : T(0);
                if (hs) *reinterpret_cast<cpx<T> *>(tile + (s0 + q) * TS + 2 * col) = {T(0), v};
                else tile[(s0 + q) * TS + col] = v;
            }
        }
    }
    static __device__ __forceinline__ void store(const T *tile, T *f, int pitch, int W, int hs, int m0)
    {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int e = threadIdx.x + NTHR * i, col = e / CPC, s0 = (e % CPC) * CW;
            if (col >= W) continue;
            Vec16<T> o;
#pragma unroll
            for (int q = 0; q < CW; ++q) o.v[q] = tile[(s0 + q) * TS + (hs ? 2 * col + 1 : col)];
            *reinterpret_cast<Vec16<T> *>(f + (size_t)col * pitch + m0 + s0) = o;
        }
    }
};

// The packed spectrum Z = A + i B (over all N frequencies) of two sections, in the
// layout of stage 0, from their tile rows.
template <class F, int N, typename T>
__device__ __forceinline__ void pack_pair(cpx<T> (&v)[F::E], const T *ra, const T *rb, int t)
{
    constexpr int H = N / 2, HE = F::E / 2;
#pragma unroll
    for (int r = 0; r < HE; ++r) {
        const int k = t + F::NT * r;
        cpx<T> a = *reinterpret_cast<const cpx<T> *>(ra + 2 * k), b = *reinterpret_cast<const cpx<T> *>(rb + 2 * k);
        if (k == 0) a.y = b.y = T(0);
        v[r] = {a.x - b.y, a.y + b.x};
    }
#pragma unroll
    for (int r = HE; r < F::E; ++r) {
        const int k = t + F::NT * r, j = N - k;
        if (k == H) {
            v[r] = {T(0), T(0)};
            continue;
        }
        const cpx<T> a = *reinterpret_cast<const cpx<T> *>(ra + 2 * j), b = *reinterpret_cast<const cpx<T> *>(rb + 2 * j);
        v[r] = {a.x + b.y, b.x - a.y};
    }
}

// Half spectra of the two sections at frequency j from the packed transform in buf.
template <class F, int N, typename T>
__device__ __forceinline__ void unpack_pair(const cpx<T> *buf, int j, cpx<T> &A, cpx<T> &B)
{
    const cpx<T> wj = buf[F::ph(j)], wn = buf[F::ph((N - j) & (N - 1))];
    const T h = T(0.5) / T(N);
    A = {(wj.x + wn.x) * h, (wj.y - wn.y) * h};
    B = {(wj.y + wn.y) * h, (wn.x - wj.x) * h};
    if (j == 0) A.y = B.y = T(0);
}

template <typename T, int N, int SEC, int V = 0>
__device__ __forceinline__ void rows_cm_body(const CurveDev &c, int mode, int blk, int nblk, StepArm arm)
{
    using C = CmCfg<T, T, N, SEC, V>;
    using F = typename C::F;
    constexpr int E = C::E, LPS = C::LPS, HE = C::HE, NTHR = C::NTHR, TS = C::TS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *tw = C::tw(smem_raw);
    T *tu = C::tile(smem_raw, 0), *td = C::tile(smem_raw, 1);
    __shared__ T term[SEC][5];
    __shared__ int am_last;
    const int tid = threadIdx.x, pr = tid / LPS, t = tid % LPS;
    cpx<T> *buf = C::buf(smem_raw) + (size_t)pr * C::BUFS;
    DevScalars *sc = c.sc;
    const int ns = c.ns, P = c.P, hs = c.hs, W = c.W, pitch = c.pitch, m0 = blk * SEC;
    const int sa = 2 * pr, sb = sa + 1, ma = m0 + sa, mb = m0 + sb;
    auto sync = [] { __syncwarp(); };   // a pair's threads are in one warp

    // tables written at set-up, before the predecessor has finished
    row_twiddles<F, N, NTHR>(tw, [&](int k) { return ldc((const cpx<T> *)c.twid + k); });
    T kv[HE], av[HE];
#pragma unroll
    for (int i = 0; i < HE; ++i) {
        kv[i] = ldc((const T *)c.kj + t + LPS * i);
        av[i] = ldc((const T *)c.aj + t + LPS * i);
    }
    const T wsec = (t < 2 && ma + t < ns) ? ((const T *)c.wt)[ma + t] : T(0);   // section a in thread 0, b in thread 1
    double lamd;
    pdl_wait();
    {
        CmTile<T, N, SEC, NTHR> xu, xd;
        xu.fetch(as_global((const T *)c.U), pitch, W, m0);
        xd.fetch(as_global((const T *)c.D), pitch, W, m0);
        // the gate and lambda; an armed call starts from the current step with `done`
        // cleared, and block 0 records the limit (as in rows_body)
        const int g_done = arm.on ? 0 : sc->done;
        const long long g_step = sc->step, g_limit = arm.on ? g_step + arm.nsteps : sc->limit;
        lamd = c.defer ? sc->lambda_next : sc->lambda;
        if (arm.on && blk == 0 && tid == 0) {
            sc->limit = g_limit;
            sc->tol = arm.tol;
            sc->done = 0;
            sc->status = 0;
        }
        if (mode == ROWS_STEP && (g_done || g_step >= g_limit)) {
            if (blk == 0 && tid == 0) sc->active = 0;
            return;
        }
        if (c.defer && blk == 0 && tid == 0) {
            sc->active = 1;
            sc->decided = 0;
            sc->lambda = lamd;
        }
        xu.put(tu, W, hs, m0, ns);
        xd.put(td, W, hs, m0, ns);
    }
    const T lam = (T)lamd;
    __syncthreads();

    T *ua = tu + sa * TS, *ub = tu + sb * TS, *da = td + sa * TS, *db = td + sb * TS;
    cpx<T> v[E], u[E];
    pack_pair<F, N>(v, ua, ub, t);
    F::template dif<true>(v, buf, tw, t, sync);          // u_a + i u_b on the grid
#pragma unroll
    for (int e = 0; e < E; ++e) {
        u[e] = v[e];
        v[e] = {u[e].x * u[e].x, u[e].y * u[e].y};
    }
    F::template dit<false>(v, buf, tw, t, sync);         // DFT of u_a^2 + i u_b^2
    F::template store<0>(v, buf, t);
    sync();
    const bool in0 = ma > 0 && ma < P, in1 = mb > 0 && mb < P;
    // pairs with an end section also sum |u|^2 and |f|^2 (a rare warp; uniform in it)
    const bool ends = __any_sync(0xffffffffu, !(in0 && in1) && ma < ns);
    T s[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // |r|^2, |d|^2, <d, r> of section a, then of b
    T se[4] = {0, 0, 0, 0};              // |u|^2, |f|^2 of a, then of b
    cpx<T> ra[HE], rb[HE];
#pragma unroll
    for (int i = 0; i < HE; ++i) {
        const int j = t + LPS * i;
        cpx<T> wa, wb;
        unpack_pair<F, N>(buf, j, wa, wb);
        const T a = av[i], hk = T(0.5) * kv[i];
        cpx<T> xa = *reinterpret_cast<cpx<T> *>(ua + 2 * j), xb = *reinterpret_cast<cpx<T> *>(ub + 2 * j);
        cpx<T> ya = *reinterpret_cast<cpx<T> *>(da + 2 * j), yb = *reinterpret_cast<cpx<T> *>(db + 2 * j);
        if (j == 0) xa.y = xb.y = ya.y = yb.y = T(0);
        cpx<T> fa = {hk * wa.y - a * xa.x, -hk * wa.x - a * xa.y};
        cpx<T> fb = {hk * wb.y - a * xb.x, -hk * wb.x - a * xb.y};
        ra[i] = in0 ? project(cpx<T>{fa.x - lam * ya.x, fa.y - lam * ya.y}, j, c.sym) : cpx<T>{0, 0};
        rb[i] = in1 ? project(cpx<T>{fb.x - lam * yb.x, fb.y - lam * yb.y}, j, c.sym) : cpx<T>{0, 0};
        if (j == 0) { ra[i].y = 0; rb[i].y = 0; fa.y = 0; fb.y = 0; }
        // half the Parseval sums (weights 1/2 at j = 0, 1 elsewhere)
        const T h = T(0.5);
        auto norm = [&](T acc, cpx<T> p, cpx<T> q) {
            const T v = i == 0 ? p.x * q.x + p.y * q.y : T(0);
            return i == 0 ? acc + (t == 0 ? h * v : v) : acc + p.x * q.x + p.y * q.y;
        };
        s[0] = norm(s[0], ra[i], ra[i]);
        s[1] = norm(s[1], ya, ya);
        s[2] = norm(s[2], ya, ra[i]);
        s[3] = norm(s[3], rb[i], rb[i]);
        s[4] = norm(s[4], yb, yb);
        s[5] = norm(s[5], yb, rb[i]);
        if (ends) {
            se[0] = norm(se[0], xa, xa);
            se[1] = norm(se[1], fa, fa);
            se[2] = norm(se[2], xb, xb);
            se[3] = norm(se[3], fb, fb);
        }
        // r^ out through the tile (u^ is read for the last time here)
        *reinterpret_cast<cpx<T> *>(ua + 2 * j) = ra[i];
        *reinterpret_cast<cpx<T> *>(ub + 2 * j) = rb[i];
    }
    if (mode != ROWS_COST) {
    sync();   // every partner value has been read
    // the packed spectrum of i k r^ -> r_x on the grid -> DFT of u r_x
#pragma unroll
    for (int i = 0; i < HE; ++i) {
        const int j = t + LPS * i;
        const T k = kv[i];
        const cpx<T> a = {-k * ra[i].y, k * ra[i].x}, b = {-k * rb[i].y, k * rb[i].x};
        buf[F::ph(j)] = {a.x - b.y, a.y + b.x};
        if (j > 0) buf[F::ph(N - j)] = {a.x + b.y, b.x - a.y};
    }
    if (t == 0) buf[F::ph(N / 2)] = {T(0), T(0)};
    sync();
    F::template load<0>(v, buf, t);
    F::template dif<true>(v, buf, tw, t, sync);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = {u[e].x * v[e].x, u[e].y * v[e].y};
    F::template dit<false>(v, buf, tw, t, sync);
    F::template store<0>(v, buf, t);
    sync();
#pragma unroll
    for (int i = 0; i < HE; ++i) {
        const int j = t + LPS * i;
        cpx<T> pa, pb;
        unpack_pair<F, N>(buf, j, pa, pb);
        const T a = av[i];
        // A^ out through D_t u's tile (its values at j were read by this thread)
        cpx<T> oa = project(cpx<T>{pa.x - a * ra[i].x, pa.y - a * ra[i].y}, j, c.sym);
        cpx<T> ob = project(cpx<T>{pb.x - a * rb[i].x, pb.y - a * rb[i].y}, j, c.sym);
        if (j == 0) oa.y = ob.y = T(0);
        *reinterpret_cast<cpx<T> *>(da + 2 * j) = oa;
        *reinterpret_cast<cpx<T> *>(db + 2 * j) = ob;
    }
    }
    // per-section norms |q_m|^2 = L sum_j c_j |q^_j|^2.  The eight sums are halved at the
    // first butterfly levels (a lane keeps the half its bit selects, one addition per
    // value and level), then added whole; value v ends in the lanes whose leading
    // bits are v's.
    {
        constexpr int LV = LPS >= 8 ? 3 : 2;
        int n = 8;
#pragma unroll
        for (int l = 0; l < LV; ++l) {
            const int o = LPS >> (l + 1);
            const bool up = (t & o) != 0;
            n >>= 1;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < n) {
                    const T keep = up ? s[n + i] : s[i], give = up ? s[i] : s[n + i];
                    s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
        }
#pragma unroll
        for (int o = LPS >> (LV + 1); o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
        // thread 0 forms section a's five terms of the cost, thread 1 section b's; the square
        // roots of |r|^2 and |d|^2 in threads 0, 1 and 2, 3 at once
        const int sec = t & 1, v0 = 3 * sec;
        auto val = [&](int v) {   // value v of this pair
            const int src = LPS >= 8 ? v * (LPS / 8) : (v >> 1) * (LPS / 4);
            const T x = __shfl_sync(0xffffffffu, s[0], src, LPS);
            if constexpr (LPS >= 8) return x;
            const T y = __shfl_sync(0xffffffffu, s[1], src, LPS);
            return (v & 1) ? y : x;
        };
        const T Lt = T(2) * (T)c.L, nr = Lt * val(v0), nd = Lt * val(v0 + 1), ndr = Lt * val(v0 + 2);
        const T root = sqrt((t & 2) ? nd : nr);
        const T sr = __shfl_sync(0xffffffffu, root, sec, LPS), sd = __shfl_sync(0xffffffffu, root, 2 + sec, LPS);
        if (t < 2) {
            const T alt = fabs(lam), w = (t ? in1 : in0) ? wsec : T(0);
            T *o = term[sa + t];
            o[0] = w * nr;                     // J^2
            o[1] = w * sr * alt * sd;          // J_arc numerator
            o[2] = w * alt * sd;               // J_arc denominator
            o[3] = w * ndr;                    // <d, r>_W
            o[4] = w * (T)(lamd * lamd) * nd;  // |l d|_W^2
        }
        if (ends) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int o = LPS / 2; o > 0; o >>= 1) se[q] += __shfl_xor_sync(0xffffffffu, se[q], o);
            if (t < 2 && ma + t < ns && !(t ? in1 : in0)) {   // an end section: |u|^2 and |f|^2
                c.rowsc[(size_t)(ma + t) * 4 + 0] = (double)(Lt * (t ? se[2] : se[0]));
                c.rowsc[(size_t)(ma + t) * 4 + 3] = (double)(Lt * (t ? se[3] : se[1]));
            }
        }
    }
    __syncthreads();
    if (mode != ROWS_COST) {
        CmTile<T, N, SEC, NTHR>::store(tu, as_global((T *)c.R), pitch, W, hs, m0);
        CmTile<T, N, SEC, NTHR>::store(td, as_global((T *)c.A), pitch, W, hs, m0);
    }
    if (tid < 32) {
        // the CTA's sums over its sections in FP64: value q in lanes 4 q .. 4 q + 3, a quarter
        // of the sections each (few FP64 instructions: each takes about 64 cycles)
        const int q = tid >> 2;
        double x = 0.0;
        if (q < 5) {
            x = (double)term[(tid & 3) * (SEC / 4)][q];
#pragma unroll
            for (int i = 1; i < SEC / 4; ++i) x += (double)term[(tid & 3) * (SEC / 4) + i][q];
        }
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        x += __shfl_xor_sync(0xffffffffu, x, 2);
        if ((tid & 3) == 0 && q < 5) c.bpart[(size_t)blk * 5 + q] = x;
    }
    if (c.defer && mode == ROWS_STEP) return;   // the contraction sums the partials
    if (!last_cta_arrive(&sc->cnt_rows, (unsigned)nblk, am_last)) return;
    rows_finish<NTHR>(c, mode, nblk, true, arm);
}

// FP32: 16 warps per SM at 16 values a thread (128 registers): N = 256 and N_s = 16384
// in 1.7 waves instead of 2.2.  20 at fewer (96 registers, no spills to speak of).
template <typename T, int N, int SEC, int V>
__global__ void __launch_bounds__(CmCfg<T, T, N, SEC, V>::NTHR,
                                  sizeof(T) == 4 && N >= 128 ? (N == 128 || V ? 640 : 512) / CmCfg<T, T, N, SEC, V>::NTHR : 1)
    k_rows_cm(const __grid_constant__ CurveDev c, int mode, StepArm arm)
{
    if ((int)blockIdx.x == c.row_blocks) {   // the extra CTA of the deferred form
        pdl_wait();
        finish_g2(c, CmCfg<T, T, N, SEC, V>::NTHR);
        return;
    }
    rows_cm_body<T, N, SEC, V>(c, mode, blockIdx.x, c.row_blocks, arm);
}

template <typename T, int N, int SEC>
__global__ void __launch_bounds__(CmCfg<T, T, N, SEC>::NTHR) k_rows_cm_batch(const CurveDev *cv, const int2 *items, int mode)
{
    const int2 it = items[blockIdx.x];
    const CurveDev &c = cv[it.x];
    rows_cm_body<T, N, SEC>(c, mode, it.y, c.row_blocks, StepArm{0, 0.0, 0});
}

// e^(-2 pi i k / N), k < N / 2, in the transform's type (FP32: the nearest values, not
// the row phase's pairs of modulus 1: a state read back has the smaller error with them)
template <typename T>
__device__ __forceinline__ cpx<T> row_root(const CurveDev &c, int k)
{
    if constexpr (std::is_same<T, dfloat>::value) {
        const float4 w = ((const float4 *)c.twdf)[k];
        return {dfloat(w.x, w.y), dfloat(w.z, w.w)};
    } else if constexpr (sizeof(T) == 4) {
        const float4 w = ((const float4 *)c.twdf)[k];
        return {w.x, w.z};
    } else {
        return ((const cpx<T> *)c.twid64)[k];
    }
}

// Physical (input type Ti) -> spectral, transformed in Tc, rounded per coefficient
// to the storage type To.
template <typename Ti, typename Tc, typename To, int N, int SEC>
__global__ void __launch_bounds__(CmCfg<Tc, To, N, SEC>::NTHR) k_row_fwd_cm(const __grid_constant__ CurveDev c,
                                                                            const Ti *phys, To *spec, SetScalars set)
{
    using C = CmCfg<Tc, To, N, SEC>;
    using F = typename C::F;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<Tc> *tw = C::tw(smem_raw);
    To *tile = C::tile(smem_raw, 0);
    const int tid = threadIdx.x, pr = tid / C::LPS, t = tid % C::LPS, m0 = blockIdx.x * SEC, ns = c.ns;
    const int sa = 2 * pr, ma = m0 + sa;
    cpx<Tc> *buf = C::buf(smem_raw) + (size_t)pr * C::BUFS;
    auto sync = [] { __syncwarp(); };
    row_twiddles<F, N, C::NTHR>(tw, [&](int k) { return row_root<Tc>(c, k); });
    pdl_wait();
    if (set.on && blockIdx.x == 0 && tid == 0) set_scalars(c.sc, set.lambda, set.tau);
    cpx<Tc> v[F::E];
#pragma unroll
    for (int e = 0; e < F::E; ++e) {   // the grid index in the digit order dit() starts from
        const int n = F::freq(t, e);
        v[e] = {ma < ns ? (Tc)phys[(size_t)ma * N + n] : Tc(0), ma + 1 < ns ? (Tc)phys[(size_t)(ma + 1) * N + n] : Tc(0)};
    }
    __syncthreads();
    F::template dit<false>(v, buf, tw, t, sync);
    F::template store<0>(v, buf, t);
    sync();
#pragma unroll
    for (int i = 0; i < C::HE; ++i) {
        const int j = t + C::LPS * i;
        cpx<Tc> A, B;
        unpack_pair<F, N>(buf, j, A, B);
        A = project(A, j, c.sym);
        B = project(B, j, c.sym);
        *reinterpret_cast<cpx<To> *>(tile + sa * C::TS + 2 * j) = {(To)A.x, (To)A.y};
        *reinterpret_cast<cpx<To> *>(tile + (sa + 1) * C::TS + 2 * j) = {(To)B.x, (To)B.y};
    }
    __syncthreads();
    CmTile<To, N, SEC, C::NTHR>::store(tile, spec, c.pitch, c.W, c.hs, m0);
}

// Trial curves (eq. KSE_initial_curve with a = 0, plus the perturbation) of a batch's
// column-form curves straight into the spectral state, in FP64: work item (curve, row
// block) per CTA.  The sections' factors (tanh and the sines) are formed once per
// section.  amps: npert per curve; vp: the curves' [npert][N] fields, curve i's at voff[i].
template <typename To, int N, int SEC>
__global__ void __launch_bounds__(CmCfg<double, To, N, SEC>::NTHR)
    k_trial_batch_cm(const CurveDev *cv, const int2 *items, int npert, const double *amps, const double *vp, const int *voff)
{
    using C = CmCfg<double, To, N, SEC>;
    using F = typename C::F;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double fac[SEC][2 + MAX_PERT];
    cpx<double> *tw = C::tw(smem_raw);
    To *tile = C::tile(smem_raw, 0);
    const int2 it = items[blockIdx.x];
    const CurveDev &c = cv[it.x];
    const int tid = threadIdx.x, pr = tid / C::LPS, t = tid % C::LPS, m0 = it.y * SEC, ns = c.ns, P = c.P;
    const int sa = 2 * pr;
    cpx<double> *buf = C::buf(smem_raw) + (size_t)pr * C::BUFS;
    auto sync = [] { __syncwarp(); };
    row_twiddles<F, N, C::NTHR>(tw, [&](int k) { return row_root<double>(c, k); });
    for (int e = tid; e < SEC * (1 + npert); e += C::NTHR) {
        const int s = e / (1 + npert), q = e % (1 + npert), m = m0 + s;
        if (q == 0) {
            double sn, co, h = m == 0 ? 1.0 : -1.0;
            if (m > 0 && m < P) {
                sincospi((double)m / (double)P, &sn, &co);
                h = tanh(c.s0 + c.S * co / sn);
            }
            fac[s][0] = m < ns ? 0.5 * (1.0 + h) : 0.0;
            fac[s][1] = m < ns ? 0.5 * (1.0 - h) : 0.0;
        } else {
            double sn = 0.0, co;
            if (m > 0 && m < P) sincospi((double)(((long long)q * m) % (2LL * P)) / (double)P, &sn, &co);
            fac[s][1 + q] = amps[(size_t)it.x * npert + q - 1] * sn;
        }
    }
    __syncthreads();
    const double *up = c.ends, *um = c.ends + N, *v0 = vp + voff[it.x];
    cpx<double> v[F::E];
#pragma unroll
    for (int e = 0; e < F::E; ++e) {   // the grid index in the digit order dit() starts from
        const int n = F::freq(t, e);
        const double a = up[n], b = um[n];
        v[e] = {fac[sa][0] * a + fac[sa][1] * b, fac[sa + 1][0] * a + fac[sa + 1][1] * b};
        for (int p = 0; p < npert; ++p) {
            const double x = v0[p * N + n];
            v[e].x += fac[sa][2 + p] * x;
            v[e].y += fac[sa + 1][2 + p] * x;
        }
    }
    F::template dit<false>(v, buf, tw, t, sync);
    F::template store<0>(v, buf, t);
    sync();
#pragma unroll
    for (int i = 0; i < C::HE; ++i) {
        const int j = t + C::LPS * i;
        cpx<double> A, B;
        unpack_pair<F, N>(buf, j, A, B);
        A = project(A, j, c.sym);
        B = project(B, j, c.sym);
        *reinterpret_cast<cpx<To> *>(tile + sa * C::TS + 2 * j) = {(To)A.x, (To)A.y};
        *reinterpret_cast<cpx<To> *>(tile + (sa + 1) * C::TS + 2 * j) = {(To)B.x, (To)B.y};
    }
    __syncthreads();
    CmTile<To, N, SEC, C::NTHR>::store(tile, (To *)c.U, c.pitch, c.W, c.hs, m0);
}

template <typename T, int N, int SEC>
__global__ void __launch_bounds__(CmCfg<T, T, N, SEC>::NTHR) k_row_inv_cm(const __grid_constant__ CurveDev c, const T *spec,
                                                                          T *phys, int scale_mode)
{
    using C = CmCfg<T, T, N, SEC>;
    using F = typename C::F;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cpx<T> *tw = C::tw(smem_raw);
    T *tile = C::tile(smem_raw, 0);
    const int tid = threadIdx.x, pr = tid / C::LPS, t = tid % C::LPS, m0 = blockIdx.x * SEC, ns = c.ns, P = c.P;
    const int sa = 2 * pr, ma = m0 + sa, mb = ma + 1;
    cpx<T> *buf = C::buf(smem_raw) + (size_t)pr * C::BUFS;
    auto sync = [] { __syncwarp(); };
    CmTile<T, N, SEC, C::NTHR> x;
    row_twiddles<F, N, C::NTHR>(tw, [&](int k) { return row_root<T>(c, k); });
    pdl_wait();
    x.fetch(spec, c.pitch, c.W, m0);
    x.put(tile, c.W, c.hs, m0, ns);
    T fa = 1, fb = 1;
    if (scale_mode == 1) {   // Euclidean gradient: -2 dx w_m, zero on the end rows
        const double dx = c.L / (double)N;
        fa = (ma >= ns || ma == 0 || ma == P) ? T(0) : (T)(-2.0 * dx * c.w[ma]);
        fb = (mb >= ns || mb == P) ? T(0) : (T)(-2.0 * dx * c.w[mb]);
    }
    __syncthreads();
    cpx<T> v[F::E];
    pack_pair<F, N>(v, tile + sa * C::TS, tile + (sa + 1) * C::TS, t);
    F::template dif<true>(v, buf, tw, t, sync);
#pragma unroll
    for (int e = 0; e < F::E; ++e) {
        const int n = F::freq(t, e);
        if (ma < ns) phys[(size_t)ma * N + n] = fa * v[e].x;
        if (mb < ns) phys[(size_t)mb * N + n] = fb * v[e].y;
    }
}

template <typename... KArgs, typename... Args>
cudaError_t cm_launch(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, bool pdl, Args... args)
{
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, kern, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// FP64 single curves on the plan of 2 values per thread: about a warp or less for each
// of the SMs' 608 quarters (a warp holds one pair at N = 64, two at N = 32).  An FP64
// instruction holds a quarter's pipe, so a second warp there would wait for the first.
bool cm_spread(int nx, int ns) { return (nx == 64 && ns <= 1216) || (nx == 32 && ns <= 2432); }

// The section counts built: 4 (FP64), 8 and 16, where a CTA has at least one warp.
template <typename T, int N, int SEC>
constexpr bool cm_built()
{
    return SEC >= (sizeof(T) == 4 ? 8 : 4) && RowFft<T, N>::F::NT * SEC / 2 >= 32;
}
// f(N, SEC) as constants for the smallest count built that is at least sec (16 always is)
template <typename T, typename Fn>
cudaError_t cm_dispatch(int n, int sec, Fn &&f)
{
    return dispatch_n(n, [&](auto nn) {
        constexpr int NN = decltype(nn)::value;
        if constexpr (cm_built<T, NN, 4>())
            if (sec <= 4) return f(nn, std::integral_constant<int, 4>{});
        if constexpr (cm_built<T, NN, 8>())
            if (sec <= 8) return f(nn, std::integral_constant<int, 8>{});
        return f(nn, std::integral_constant<int, 16>{});
    });
}

// Warps of a single curve's row phase on a plan.  FP32 curves run on the plan of the
// fewest values per thread that has at most CM_WARPS of them, 8 per SM: below that the
// phase is one wave bound by the chain of a warp and by the first pass through its code,
// both of which shrink with the values per thread; above, by the instructions in all,
// which grow.  Graph step in us on the finer / the coarser plan: N = 64, 2 and 4 values,
// 9.4 / 9.9 at N_s = 1024, 11.7 / 11.9 at 2048, 15.5 / 14.8 at 3000; 4 and 8 values,
// 15.2 / 15.4 at 4096, 26.0 / 25.9 at 6000; N = 128, 4 and 8 values, 10.6 / 12.2 at 1024,
// 17.2 / 16.6 at 3000; N = 256, 8 and 16 values, 14.4 / 18.0 at 1024, 17.1 / 20.0 at 2048,
// 24.9 / 25.0 at 4096, 96.6 / 94.9 at 16384.
constexpr int CM_WARPS = 1216;
template <typename T, int N, int V>
constexpr int cm_warps(int ns)
{
    return (ns + 1) / 2 * RowFft<T, N, V>::F::NT / 32;
}

template <typename T, int N, int SEC, int V>
cudaError_t rows_run(const CurveDev &c, int mode, cudaStream_t st, StepArm arm)
{
    using C = CmCfg<T, T, N, SEC, V>;
    return cm_launch(k_rows_cm<T, N, SEC, V>, c.row_blocks + c.defer, C::NTHR, C::bytes(2), st, true, c, mode, arm);
}

template <typename T>
cudaError_t rows_t(const CurveDev &c, int mode, cudaStream_t st, StepArm arm)
{
    if constexpr (sizeof(T) == 8) {
        if (cm_spread(c.nx, c.ns))
            return c.nx == 32 ? rows_run<T, 32, 4, 1>(c, mode, st, arm) : rows_run<T, 64, 4, 1>(c, mode, st, arm);
    }
    return cm_dispatch<T>(c.nx, c.rsec, [&](auto nn, auto ss) {
        constexpr int N = decltype(nn)::value, SEC = decltype(ss)::value;
        if constexpr (sizeof(T) == 4 && N >= 32)
            if (cm_warps<T, N, 1>(c.ns) <= CM_WARPS) return rows_run<T, N, SEC, 1>(c, mode, st, arm);
        if constexpr (sizeof(T) == 4 && (N == 32 || N == 64))
            if (cm_warps<T, N, 2>(c.ns) <= CM_WARPS) return rows_run<T, N, SEC, 2>(c, mode, st, arm);
        return rows_run<T, N, SEC, 0>(c, mode, st, arm);
    });
}

template <typename T>
cudaError_t rows_batch_t(int N_, int sec, const CurveDev *cv, const int2 *items, int nitems, int mode, cudaStream_t st)
{
    return cm_dispatch<T>(N_, sec, [&](auto nn, auto ss) {
        constexpr int N = decltype(nn)::value, SEC = decltype(ss)::value;
        using C = CmCfg<T, T, N, SEC>;
        return cm_launch(k_rows_cm_batch<T, N, SEC>, nitems, C::NTHR, C::bytes(2), st, true, cv, items, mode);
    });
}

template <typename Ti, typename Tc, typename To>
cudaError_t fwd_t(const CurveDev &c, const void *phys, void *spec, SetScalars set, cudaStream_t st)
{
    return cm_dispatch<float>(c.nx, 8, [&](auto nn, auto ss) {
        constexpr int N = decltype(nn)::value, SEC = decltype(ss)::value;
        using C = CmCfg<Tc, To, N, SEC>;
        return cm_launch(k_row_fwd_cm<Ti, Tc, To, N, SEC>, (c.ns + SEC - 1) / SEC, C::NTHR, C::bytes(1), st, true, c,
                         (const Ti *)phys, (To *)spec, set);
    });
}

template <typename T>
cudaError_t inv_t(const CurveDev &c, const void *spec, void *phys, int scale_mode, cudaStream_t st)
{
    return cm_dispatch<float>(c.nx, 8, [&](auto nn, auto ss) {
        constexpr int N = decltype(nn)::value, SEC = decltype(ss)::value;
        using C = CmCfg<T, T, N, SEC>;
        return cm_launch(k_row_inv_cm<T, N, SEC>, (c.ns + SEC - 1) / SEC, C::NTHR, C::bytes(1), st, true, c,
                         (const T *)spec, (T *)phys, scale_mode);
    });
}

}  // namespace

int cm_sections(int nx, int ns, int prec, int want, int single)
{
    if (single && !prec && cm_spread(nx, ns)) return 4;
    int got = 0;
    auto pick = [&](auto, auto ss) {
        got = decltype(ss)::value;
        return cudaSuccess;
    };
    if (prec) cm_dispatch<float>(nx, want, pick);
    else cm_dispatch<double>(nx, want, pick);
    return got;
}

cudaError_t launch_rows_cm(const CurveDev &c, int mode, cudaStream_t st, StepArm arm)
{
    return c.prec ? rows_t<float>(c, mode, st, arm) : rows_t<double>(c, mode, st, arm);
}

cudaError_t launch_rows_cm_batch(int prec, int N, int sec, const CurveDev *cv, const int2 *items, int nitems, int mode,
                                 cudaStream_t st)
{
    if (nitems <= 0) return cudaSuccess;
    return prec ? rows_batch_t<float>(N, sec, cv, items, nitems, mode, st)
                : rows_batch_t<double>(N, sec, cv, items, nitems, mode, st);
}

template <typename T>
static cudaError_t trial_batch_t(int N_, int sec, const CurveDev *cv, const int2 *items, int nitems, int npert,
                                 const double *amps, const double *vp, const int *voff, cudaStream_t st)
{
    return cm_dispatch<T>(N_, sec, [&](auto nn, auto ss) {
        constexpr int N = decltype(nn)::value, SEC = decltype(ss)::value;
        using C = CmCfg<double, T, N, SEC>;
        return cm_launch(k_trial_batch_cm<T, N, SEC>, nitems, C::NTHR, C::bytes(1), st, false, cv, items, npert, amps, vp,
                         voff);
    });
}

cudaError_t launch_trial_batch_cm(int prec, int N, int sec, const CurveDev *cv, const int2 *items, int nitems, int npert,
                                  const double *amps, const double *vp, const int *voff, cudaStream_t st)
{
    if (nitems <= 0) return cudaSuccess;
    return prec ? trial_batch_t<float>(N, sec, cv, items, nitems, npert, amps, vp, voff, st)
                : trial_batch_t<double>(N, sec, cv, items, nitems, npert, amps, vp, voff, st);
}

cudaError_t launch_row_fwd_x_cm(const CurveDev &c, void *spec, cudaStream_t st)
{
    const SetScalars none = {0.0, 0.0, 0};
    return c.prec ? fwd_t<double, double, float>(c, c.X, spec, none, st) : fwd_t<double, double, double>(c, c.X, spec, none, st);
}

cudaError_t launch_row_fwd_cm(const CurveDev &c, const void *phys, void *spec, SetScalars set, cudaStream_t st)
{
    return c.prec ? fwd_t<float, dfloat, float>(c, phys, spec, set, st) : fwd_t<double, double, double>(c, phys, spec, set, st);
}

cudaError_t launch_row_inv_cm(const CurveDev &c, const void *spec, void *phys, int scale_mode, cudaStream_t st)
{
    return c.prec ? inv_t<float>(c, spec, phys, scale_mode, st) : inv_t<double>(c, spec, phys, scale_mode, st);
}

}  // namespace ks
