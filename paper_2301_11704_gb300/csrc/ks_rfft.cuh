// ks_rfft.cuh -- register transforms: a DFT of L = E x NT points by NT threads,
// E complex values per thread, as a chain of in-register DFTs of radix up to 32
// with one exchange through shared memory between two of them.
//
// Why this shape.  A transform whose radix-2 stages cross lanes by shuffles, or
// whose radix-4 stages each pass through shared memory, is bound by the L1 pipe
// (a shuffle of 4 bytes and a shared access cost the same there): log2(L) - 3
// crossings of the whole line.  With radices of 8 to 32 in registers a line of
// 256 crosses once, of 4096 twice, of 16384 (32 x 32 x 16) twice.
//
// The stages are in place: stage i reads and writes the same positions of the
// buffer in the same thread, so one barrier per exchange is enough (after the
// writes).  dif() takes the values in the layout of stage 0 (element tid + NT r in
// register r) and leaves them in the layout of the last stage; dit() goes back.
// Between them the transformed index stays in the digit order of the stages, in
// which the tables of a pointwise product are stored.
#pragma once

#include "ks_device.cuh"

namespace ks {

// A pointer into global memory (the fields' and tables' addresses come in a struct:
// without this the compiler takes them for generic ones, which may alias the
// exchanges in shared memory and cannot be read ahead of them).
template <typename T>
__device__ __forceinline__ T *as_global(T *p)
{
    __builtin_assume(__isGlobal(p));
    return p;
}
// Loads of tables written at set-up.
template <typename T>
__device__ __forceinline__ T ldc(const T *p) { return __ldg(p); }
__device__ __forceinline__ cpx<float> ldc(const cpx<float> *p)
{
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cpx<double> ldc(const cpx<double> *p)
{
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}

// cos(2 pi e / 128); folds to a literal once the caller's loops are unrolled
template <typename T>
__device__ constexpr T cos128(int e)
{
    e &= 127;
    if (e > 64) e = 128 - e;
    const bool neg = e > 32;
    if (neg) e = 64 - e;
    double v = 0.0;
    switch (e) {
    case 0: v = 1.0; break;
    case 1: v = 0.99879545620517239271; break;
    case 2: v = 0.99518472667219688624; break;
    case 3: v = 0.98917650996478097345; break;
    case 4: v = 0.98078528040323044913; break;
    case 5: v = 0.9700312531945439926; break;
    case 6: v = 0.95694033573220886494; break;
    case 7: v = 0.94154406518302077841; break;
    case 8: v = 0.92387953251128675613; break;
    case 9: v = 0.90398929312344333159; break;
    case 10: v = 0.88192126434835502971; break;
    case 11: v = 0.8577286100002720699; break;
    case 12: v = 0.83146961230254523708; break;
    case 13: v = 0.80320753148064490981; break;
    case 14: v = 0.77301045336273696081; break;
    case 15: v = 0.74095112535495909118; break;
    case 16: v = 0.7071067811865475244; break;
    case 17: v = 0.67155895484701840063; break;
    case 18: v = 0.63439328416364549822; break;
    case 19: v = 0.59569930449243334347; break;
    case 20: v = 0.55557023301960222474; break;
    case 21: v = 0.51410274419322172659; break;
    case 22: v = 0.47139673682599764856; break;
    case 23: v = 0.42755509343028209432; break;
    case 24: v = 0.38268343236508977173; break;
    case 25: v = 0.33688985339222005069; break;
    case 26: v = 0.29028467725446236764; break;
    case 27: v = 0.24298017990326388995; break;
    case 28: v = 0.19509032201612826785; break;
    case 29: v = 0.14673047445536175166; break;
    case 30: v = 0.098017140329560601994; break;
    case 31: v = 0.049067674327418014255; break;
    default: v = 0.0; break;
    }
    return T(neg ? -v : v);
}
template <typename T>
__device__ constexpr T sin128(int e) { return cos128<T>(e - 32); }

// v e^(-2 pi i e / 128), or its conjugate factor when inv; e a constant after unrolling
template <typename T>
__device__ __forceinline__ cpx<T> mul128(cpx<T> v, int e, bool inv)
{
    if (inv) e = -e;
    e &= 127;
    if (e == 0) return v;
    if (e == 32) return {v.y, -v.x};
    if (e == 64) return {-v.x, -v.y};
    if (e == 96) return {-v.y, v.x};
    const T h = cos128<T>(16);
    if (e == 16) return {h * (v.x + v.y), h * (v.y - v.x)};
    if (e == 48) return {h * (v.y - v.x), -h * (v.x + v.y)};
    if (e == 80) return {-h * (v.x + v.y), h * (v.x - v.y)};
    if (e == 112) return {h * (v.x - v.y), h * (v.x + v.y)};
    const T c = cos128<T>(e), s = sin128<T>(e);
    return {v.x * c + v.y * s, v.y * c - v.x * s};
}

// R-point DFT in registers, natural order in and out, unscaled (e^(-...), or
// e^(+...) when INV): 2, 4 directly, the others as A x B.
template <typename T, int R, bool INV>
__device__ __forceinline__ void dft(cpx<T> (&v)[R])
{
    if constexpr (R == 2) {
        const cpx<T> a = v[0], b = v[1];
        v[0] = {a.x + b.x, a.y + b.y};
        v[1] = {a.x - b.x, a.y - b.y};
    } else if constexpr (R == 4) {
        const cpx<T> t0 = {v[0].x + v[2].x, v[0].y + v[2].y}, t1 = {v[0].x - v[2].x, v[0].y - v[2].y};
        const cpx<T> t2 = {v[1].x + v[3].x, v[1].y + v[3].y}, t3 = {v[1].x - v[3].x, v[1].y - v[3].y};
        v[0] = {t0.x + t2.x, t0.y + t2.y};
        v[2] = {t0.x - t2.x, t0.y - t2.y};
        if constexpr (INV) {
            v[1] = {t1.x - t3.y, t1.y + t3.x};
            v[3] = {t1.x + t3.y, t1.y - t3.x};
        } else {
            v[1] = {t1.x + t3.y, t1.y - t3.x};
            v[3] = {t1.x - t3.y, t1.y + t3.x};
        }
    } else {
        constexpr int A = R == 8 ? 2 : 4, B = R / A;
        cpx<T> u[R];   // [n2][k1]
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) {
            cpx<T> t[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) t[n1] = v[B * n1 + n2];
            dft<T, A, INV>(t);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) u[n2 * A + k1] = mul128(t[k1], n2 * k1 * (128 / R), INV);
        }
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            cpx<T> t[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) t[n2] = u[n2 * A + k1];
            dft<T, B, INV>(t);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = t[k2];
        }
    }
}

// The plan of a transform: L points, the product of the radices Rs, E per thread, the
// first radix E.
// PH: a transform at the frequencies k + 1/4 (the twiddles of stage 0 carry
// the quarter; its radix part, e^(-2 pi i r / 4 R1) on element r, is the caller's).
// FULL: every twiddle is tabulated; else (FP32) a radix-R stage keeps 4 + R/4 - 1
// of them and forms the others by one product (a fifth of the loads at R = 32;
// one more rounding).
template <typename T, int L_, int E_, bool PH, bool FULL, int... Rs>
struct RegFft {
    using type = T;
    static constexpr int L = L_, E = E_, NT = L_ / E_;
    static constexpr int NST = sizeof...(Rs);   // stages
    static __host__ __device__ constexpr int rad(int i)
    {
        const int r[] = {Rs...};
        return r[i];
    }
    static_assert((Rs * ...) == L && rad(0) == E && NST >= 2, "the radices make up the length");
    static __host__ __device__ constexpr int sub(int i) { return i == 0 ? L : sub(i - 1) / rad(i - 1); }
    static __host__ __device__ constexpr int lr(int i) { return sub(i) / rad(i); }   // butterflies of a sub-transform
    // tabulated factors of a stage's butterfly, and where the stage's table starts
    static __host__ __device__ constexpr int ent(int i)
    {
        return (FULL || rad(i) <= 4) ? rad(i) : 4 + rad(i) / 4 - 1;
    }
    static __host__ __device__ constexpr int tw_off(int i) { return i == 0 ? 0 : tw_off(i - 1) + ent(i - 1) * lr(i - 1); }
    static constexpr int TW = tw_off(NST - 1);   // the last stage has none
    // padded buffer: the strided accesses of the later stages (stride rad(last)
    // or runs of lr(i) elements) fall in distinct banks
    static constexpr int PSH = sizeof(T) == 4 ? 4 : 3;
    static constexpr bool PAD2 = sizeof(T) == 4 && L > 256 && lr(1) == 8 && sub(1) == 256;
    static __host__ __device__ constexpr int ph(int p)
    {
        int q = p + (p >> PSH);
        if constexpr (PAD2) q += (p >> 8) * 8;
        return q;
    }
    static constexpr int BUF = L + (L >> PSH) + (PAD2 ? (L >> 8) * 8 : 0);
    static constexpr size_t BYTES = (size_t)BUF * sizeof(cpx<T>);

    // table entry p is e^(-2 pi i num / den); with PH the frequencies are k + (4 c + 1) / 4 cs
    // (k + 1/4 for the one class of cs = 1)
    static __host__ __device__ void tw_entry(int p, int c, int cs, long long &num, long long &den)
    {
        int i = 0;
        while (i + 1 < NST - 1 && p >= tw_off(i + 1)) ++i;
        const int rel = p - tw_off(i), kk = rel / lr(i), o = rel % lr(i);
        const bool a = FULL || rad(i) <= 4 || kk < 4;
        const int k4 = a ? 4 * cs * kk + ((PH && i == 0) ? 4 * c + 1 : 0) : 16 * cs * (kk - 3);
        num = (long long)o * k4;
        den = 4LL * cs * sub(i);
    }
    // the frequency index k of register e of thread t after dif()
    static __host__ __device__ int freq(int t, int e)
    {
        constexpr int RL = rad(NST - 1);
        int q = t + NT * (e / RL);   // sub-transform of the last stage: digits k1, k2, (k3)
        int k = e % RL, w = L / RL;
        k *= w;
        for (int i = NST - 2; i >= 0; --i) {
            w /= rad(i);
            k += (q % rad(i)) * w;
            q /= rad(i);
        }
        return k;
    }

    template <int I>
    static __device__ __forceinline__ int pos0(int tid, int b)
    {
        const int q = tid + NT * b;
        if constexpr (I == 0) return q;
        else return (q / lr(I)) * sub(I) + q % lr(I);
    }
    template <int I>
    static __device__ __forceinline__ void load(cpx<T> (&v)[E], const cpx<T> *buf, int tid)
    {
#pragma unroll
        for (int b = 0; b < E / rad(I); ++b) {
            // p and lr r have no bit in common, so their places in the padded buffer add: one
            // address per butterfly, the elements at constant offsets
            const cpx<T> *q = buf + ph(pos0<I>(tid, b));
#pragma unroll
            for (int r = 0; r < rad(I); ++r) v[b * rad(I) + r] = q[ph(lr(I) * r)];
        }
    }
    template <int I>
    static __device__ __forceinline__ void store(const cpx<T> (&v)[E], cpx<T> *buf, int tid)
    {
#pragma unroll
        for (int b = 0; b < E / rad(I); ++b) {
            cpx<T> *q = buf + ph(pos0<I>(tid, b));
#pragma unroll
            for (int r = 0; r < rad(I); ++r) q[ph(lr(I) * r)] = v[b * rad(I) + r];
        }
    }
    template <int I, bool CONJ, bool NC>
    static __device__ __forceinline__ void twiddle(cpx<T> (&v)[E], const cpx<T> *tw, int tid)
    {
        constexpr int R = rad(I), KA = (FULL || R <= 4) ? R : 4;
        constexpr bool P0 = PH && I == 0;
        auto get = [](const cpx<T> *p) {
            if constexpr (NC) return ldc(p);
            else return *p;
        };
#pragma unroll
        for (int b = 0; b < E / R; ++b) {
            const cpx<T> *t = tw + tw_off(I) + (tid + NT * b) % lr(I);
            cpx<T> ta[KA];
#pragma unroll
            for (int k = P0 ? 0 : 1; k < KA; ++k) {
                ta[k] = get(t + k * lr(I));
                if (CONJ) ta[k].y = -ta[k].y;
            }
#pragma unroll
            for (int kb = 0; kb < R / KA; ++kb) {
                cpx<T> tb = {T(1), T(0)};
                if (kb > 0) {
                    tb = get(t + (KA + kb - 1) * lr(I));
                    if (CONJ) tb.y = -tb.y;
                }
#pragma unroll
                for (int k = 0; k < KA; ++k) {
                    cpx<T> &x = v[b * R + kb * KA + k];
                    if (k == 0 && !P0) {
                        if (kb > 0) x = cmul(x, tb);
                    } else {
                        x = cmul(x, kb > 0 ? cmul(ta[k], tb) : ta[k]);
                    }
                }
            }
        }
    }
    template <int I, bool INV>
    static __device__ __forceinline__ void butterflies(cpx<T> (&v)[E])
    {
        constexpr int R = rad(I);
#pragma unroll
        for (int b = 0; b < E / R; ++b) {
            cpx<T> t[R];
#pragma unroll
            for (int r = 0; r < R; ++r) t[r] = v[b * R + r];
            dft<T, R, INV>(t);
#pragma unroll
            for (int r = 0; r < R; ++r) v[b * R + r] = t[r];
        }
    }
    template <bool INV, bool NC, int I, typename Sync>
    static __device__ __forceinline__ void dif_from(cpx<T> (&v)[E], cpx<T> *buf, const cpx<T> *tw, int tid, Sync &&sync)
    {
        if constexpr (I > 0) load<I>(v, buf, tid);
        butterflies<I, INV>(v);
        if constexpr (I + 1 < NST) {
            twiddle<I, INV, NC>(v, tw, tid);
            store<I>(v, buf, tid);
            sync();
            dif_from<INV, NC, I + 1>(v, buf, tw, tid, sync);
        }
    }
    // layout of stage 0 -> layout of the last stage (NC: the twiddles by loads of the
    // read-only path, which the compiler may move)
    template <bool INV, bool NC = false, typename Sync>
    static __device__ __forceinline__ void dif(cpx<T> (&v)[E], cpx<T> *buf, const cpx<T> *tw, int tid, Sync &&sync)
    {
        dif_from<INV, NC, 0>(v, buf, tw, tid, sync);
    }
    template <bool INV, bool NC, int I, typename Sync>
    static __device__ __forceinline__ void dit_from(cpx<T> (&v)[E], cpx<T> *buf, const cpx<T> *tw, int tid, Sync &&sync)
    {
        if constexpr (I + 1 < NST) {
            load<I>(v, buf, tid);
            twiddle<I, INV, NC>(v, tw, tid);
        }
        butterflies<I, INV>(v);
        if constexpr (I > 0) {
            store<I>(v, buf, tid);
            sync();
            dit_from<INV, NC, I - 1>(v, buf, tw, tid, sync);
        }
    }
    // layout of the last stage -> layout of stage 0
    template <bool INV, bool NC = false, typename Sync>
    static __device__ __forceinline__ void dit(cpx<T> (&v)[E], cpx<T> *buf, const cpx<T> *tw, int tid, Sync &&sync)
    {
        dit_from<INV, NC, NST - 1>(v, buf, tw, tid, sync);
    }
};

}  // namespace ks
