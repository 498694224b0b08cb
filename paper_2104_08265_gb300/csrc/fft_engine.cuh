// Device FFT engine: register DFTs and mixed-radix Stockham passes over shared memory.
//
// A plan factors N into a few radices R <= 25 (composite radices such as 20 or 24 are
// transformed entirely in registers), so that a 6000-point transform takes three
// shared-memory passes.  Pass p (Ns = product of the earlier radices) reads
// x[j + r N/R], r < R, multiplies by exp(-+2 pi i r (j mod Ns) / (Ns R)), applies the
// R-point DFT and writes y[(j / Ns) Ns R + (j mod Ns) + r Ns]; the result is in natural
// order.  B = 2^LOGB independent sequences are transformed together; element (c, i) of the
// batch lives at buf[pad(i) * B + c], where pad() inserts one slot every 16 elements so
// that the stride-R writes of early passes do not pile onto one shared-memory bank.
//
// Plans come in two forms: a runtime plan (FftPlan: any length that factors into radices <= 25)
// and a compile-time plan (all strides and divisors constants).  A batch of sequences ping-pongs
// between two buffers (run_plan); a single sequence is transformed in place in one buffer
// (run_plan_inplace, run_plan_fixed).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "async_copy.cuh"
#include "dft_roots.cuh"
#include "rng.cuh"
#include "wcsim_internal.cuh"

namespace wcsim {

__host__ __device__ __forceinline__ int pad16(int i) { return i + (i >> 4); }
__host__ __device__ __forceinline__ int padded_len(int n) { return n + (n >> 4) + 1; }

// ------------------------------------------------------------------ complex helpers
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * w (forward) or a * conj(w) (inverse)
template <bool INV>
__device__ __forceinline__ float2 twiddle(float2 a, float2 w)
{
    return INV ? make_float2(a.x * w.x + a.y * w.y, a.y * w.x - a.x * w.y) : cmul(a, w);
}
// -i a (forward) or +i a (inverse)
template <bool INV>
__device__ __forceinline__ float2 rot(float2 a)
{
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// ------------------------------------------------------------------ small DFTs
template <bool INV>
__device__ __forceinline__ void dft4v(float2& v0, float2& v1, float2& v2, float2& v3)
{
    const float2 s02 = cadd(v0, v2), d02 = csub(v0, v2);
    const float2 s13 = cadd(v1, v3), d13 = rot<INV>(csub(v1, v3));
    v0 = cadd(s02, s13);
    v2 = csub(s02, s13);
    v1 = cadd(d02, d13);
    v3 = csub(d02, d13);
}

template <bool INV>
__device__ __forceinline__ void dft3v(float2* v)
{
    const float s3 = 0.866025403784438647f;
    const float2 t = cadd(v[1], v[2]);
    const float2 d = rot<INV>(cscale(csub(v[1], v[2]), s3));
    const float2 m = make_float2(v[0].x - 0.5f * t.x, v[0].y - 0.5f * t.y);
    v[0] = cadd(v[0], t);
    v[1] = cadd(m, d);
    v[2] = csub(m, d);
}

template <bool INV>
__device__ __forceinline__ void dft5v(float2* v)
{
    const float c1 = 0.309016994374947424f, c2 = -0.809016994374947424f;
    const float s1 = 0.951056516295153572f, s2 = 0.587785252292473129f;
    const float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
    const float2 d1 = csub(v[1], v[4]), d2 = csub(v[2], v[3]);
    const float2 v0 = v[0];
    const float2 a1 = make_float2(v0.x + c1 * t1.x + c2 * t2.x, v0.y + c1 * t1.y + c2 * t2.y);
    const float2 a2 = make_float2(v0.x + c2 * t1.x + c1 * t2.x, v0.y + c2 * t1.y + c1 * t2.y);
    const float2 b1 = rot<INV>(make_float2(s1 * d1.x + s2 * d2.x, s1 * d1.y + s2 * d2.y));
    const float2 b2 = rot<INV>(make_float2(s2 * d1.x - s1 * d2.x, s2 * d1.y - s1 * d2.y));
    v[0] = cadd(v0, cadd(t1, t2));
    v[1] = cadd(a1, b1);
    v[4] = csub(a1, b1);
    v[2] = cadd(a2, b2);
    v[3] = csub(a2, b2);
}

template <bool INV>
__device__ __forceinline__ void dft7v(float2* v)
{
    // cos / sin (2 pi m / 7), m = 1, 2, 3
    const float c[3] = {0.623489801858733530f, -0.222520933956314404f, -0.900968867902419126f};
    const float s[3] = {0.781831482468029809f, 0.974927912181823607f, 0.433883739117558120f};
    float2 t[3], d[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        t[p] = cadd(v[p + 1], v[6 - p]);
        d[p] = csub(v[p + 1], v[6 - p]);
    }
    const float2 v0 = v[0];
    v[0] = cadd(v0, cadd(t[0], cadd(t[1], t[2])));
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
        float2 a = v0, b = make_float2(0.f, 0.f);
#pragma unroll
        for (int p = 1; p <= 3; ++p) {
            const int m = (p * k) % 7;
            const float cm = (m <= 3) ? c[m - 1] : c[7 - m - 1];
            const float sm = (m <= 3) ? s[m - 1] : -s[7 - m - 1];
            a.x += cm * t[p - 1].x; a.y += cm * t[p - 1].y;
            b.x += sm * d[p - 1].x; b.y += sm * d[p - 1].y;
        }
        const float2 rb = rot<INV>(b);
        v[k] = cadd(a, rb);
        v[7 - k] = csub(a, rb);
    }
}

template <bool INV>
__device__ __forceinline__ void dft8v(float2* v)
{
    const float h = 0.707106781186547524f;
    dft4v<INV>(v[0], v[2], v[4], v[6]);
    dft4v<INV>(v[1], v[3], v[5], v[7]);
    float2 o1 = v[3], o2 = v[5], o3 = v[7];
    o1 = INV ? make_float2(h * (o1.x - o1.y), h * (o1.x + o1.y))
             : make_float2(h * (o1.x + o1.y), h * (o1.y - o1.x));
    o2 = rot<INV>(o2);
    o3 = INV ? make_float2(-h * (o3.x + o3.y), h * (o3.x - o3.y))
             : make_float2(h * (o3.y - o3.x), -h * (o3.x + o3.y));
    const float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

template <bool INV>
__device__ __forceinline__ void dft16v(float2* v)
{
    // X[k1 + 4 k2] = sum_b w16^(b k1) w4^(b k2) Y_b[k1],  Y_b = DFT4 of v[b + 4 a] over a
#pragma unroll
    for (int b = 0; b < 4; ++b) dft4v<INV>(v[b], v[b + 4], v[b + 8], v[b + 12]);
    const float cs[4] = {1.0f, 0.923879532511286756f, 0.707106781186547524f, 0.382683432365089772f};
#pragma unroll
    for (int b = 1; b < 4; ++b)
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1) {
            const int m = b * k1;
            const int q = m / 4, rr = m % 4;
            const float cr = cs[rr], sr = (rr == 0) ? 0.0f : cs[4 - rr];
            float cm, sm;
            if (q == 0) { cm = cr; sm = sr; }
            else if (q == 1) { cm = -sr; sm = cr; }
            else { cm = -cr; sm = -sr; }
            v[b + 4 * k1] = cmul(v[b + 4 * k1], make_float2(cm, INV ? sm : -sm));
        }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4v<INV>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
    float2 o[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) o[k1 + 4 * k2] = v[4 * k1 + k2];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = o[i];
}

// First factor of a composite radix for the Cooley-Tukey split R = A * B.
template <int R>
struct Split {
    static constexpr int A = (R % 16 == 0 && R != 16) ? 16
                           : (R % 8 == 0 && R != 8) ? 8
                           : (R % 4 == 0 && R != 4) ? 4
                           : (R % 2 == 0) ? 2
                           : (R % 3 == 0) ? 3
                           : (R % 5 == 0) ? 5 : 7;
    static constexpr int B = R / A;
};

// In-register R-point DFT, natural order in and out.  Composite R: n = B n1 + n2,
// k = k1 + A k2;  A-point DFTs over n1, twiddle exp(-+2 pi i n2 k1 / R), B-point DFTs over n2.
template <int R, bool INV>
__device__ __forceinline__ void dft(float2* v)
{
    if constexpr (R == 1) {
    } else if constexpr (R == 2) {
        const float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (R == 3) {
        dft3v<INV>(v);
    } else if constexpr (R == 4) {
        dft4v<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 5) {
        dft5v<INV>(v);
    } else if constexpr (R == 7) {
        dft7v<INV>(v);
    } else if constexpr (R == 8) {
        dft8v<INV>(v);
    } else if constexpr (R == 16) {
        dft16v<INV>(v);
    } else {
        constexpr int A = Split<R>::A, B = Split<R>::B;
        float2 y[R];
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) {
            float2 t[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) t[n1] = v[B * n1 + n2];
            dft<A, INV>(t);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) {
                float2 x = t[k1];
                if (n2 * k1 != 0) {
                    const float c = Roots<R>::c((n2 * k1) % R), s = Roots<R>::s((n2 * k1) % R);
                    x = INV ? make_float2(x.x * c - x.y * s, x.x * s + x.y * c)
                            : make_float2(x.x * c + x.y * s, x.y * c - x.x * s);
                }
                y[n2 * A + k1] = x;
            }
        }
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) {
            float2 t[B];
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) t[n2] = y[n2 * A + k1];
            dft<B, INV>(t);
#pragma unroll
            for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = t[k2];
        }
    }
}

// ------------------------------------------------------------------ shared-memory access
template <int LOGB>
struct SmemLd {
    static constexpr bool kShared = true;
    const float2* p;
    __device__ __forceinline__ float2 operator()(int c, int i) const { return p[(pad16(i) << LOGB) + c]; }
    __device__ __forceinline__ float2 at(int c, int pi) const { return p[(pi << LOGB) + c]; }
};
template <int LOGB>
struct SmemSt {
    static constexpr bool kShared = true;
    float2* p;
    __device__ __forceinline__ void operator()(int c, int i, float2 v) const { p[(pad16(i) << LOGB) + c] = v; }
    __device__ __forceinline__ void at(int c, int pi, float2 v) const { p[(pi << LOGB) + c] = v; }
};

// First-pass source over an unpadded shared buffer (a staged input): element (c, i) at
// p[(i << LOGB) + c].  The first pass reads x[j + r N/R] with consecutive j on consecutive
// lanes, which needs no padding to stay free of bank conflicts.
template <int LOGB>
struct FlatLd {
    const float2* p;
    __device__ __forceinline__ float2 operator()(int c, int i) const { return p[(i << LOGB) + c]; }
};

template <class T, class = void>
struct IsShared { static constexpr bool value = false; };
template <class T>
struct IsShared<T, decltype((void)T::kShared)> { static constexpr bool value = T::kShared; };

struct PassArgs {
    int n, ns;
    uint32_t ns_magic;
    const float2* tw;
};

// One Stockham pass of radix R over a batch of 2^LOGB sequences.
template <int R, bool INV, int LOGB, class Ld, class St>
__device__ __forceinline__ void pass_r(const Ld& ld, const St& st, const PassArgs& a)
{
    const int nb = a.n / R;
    const int total = nb << LOGB;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int c = idx & ((1 << LOGB) - 1);
        const int j = idx >> LOGB;
        const int q = (a.ns == 1) ? j : (int)__umulhi((uint32_t)j, a.ns_magic);
        const int k = j - q * a.ns;
        float2 v[R];
        // Padded shared indices: pad16(j + r nb) = pad16(j) + r (nb + nb / 16) when 16 | nb.
        if constexpr (IsShared<Ld>::value) {
            if ((nb & 15) == 0) {
                const int p0 = pad16(j), ps = nb + (nb >> 4);
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = ld.at(c, p0 + r * ps);
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = ld(c, j + r * nb);
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = ld(c, j + r * nb);
        }
        if (k > 0) {
            const float2* t = a.tw + k;
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = twiddle<INV>(v[r], __ldg(t + (r - 1) * a.ns));
        }
        dft<R, INV>(v);
        const int o = q * a.ns * R + k;
        // pad16(o + r ns) = pad16(o) + r (ns + ns / 16) when 16 | ns; a radix-16 first pass
        // (ns = 1, o = 16 q) writes 16 consecutive padded slots.
        if constexpr (IsShared<St>::value) {
            if ((a.ns & 15) == 0 || (R == 16 && a.ns == 1)) {
                const int p0 = pad16(o), ps = (a.ns == 1) ? 1 : a.ns + (a.ns >> 4);
#pragma unroll
                for (int r = 0; r < R; ++r) st.at(c, p0 + r * ps, v[r]);
            } else {
#pragma unroll
                for (int r = 0; r < R; ++r) st(c, o + r * a.ns, v[r]);
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) st(c, o + r * a.ns, v[r]);
        }
    }
}

// Radices a plan may use (every one has a pass_r instantiation below).
#define WCSIM_FOR_EACH_RADIX(X) \
    X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(10) X(12) X(14) X(15) X(16) X(20) X(24) X(25)

template <bool INV, int LOGB, class Ld, class St>
__device__ __forceinline__ void pass_any(int R, const Ld& ld, const St& st, const PassArgs& a)
{
    switch (R) {
#define WCSIM_CASE(RR) case RR: pass_r<RR, INV, LOGB>(ld, st, a); break;
        WCSIM_FOR_EACH_RADIX(WCSIM_CASE)
#undef WCSIM_CASE
        default: {   // R == 1: a copy
            for (int idx = threadIdx.x; idx < (a.n << LOGB); idx += blockDim.x) {
                const int c = idx & ((1 << LOGB) - 1), i = idx >> LOGB;
                st(c, i, ld(c, i));
            }
        }
    }
}

// Stage the input of an inverse real-pair transform: z[k] = X0[k] + i X1[k], k < n, for two
// Hermitian spectra given by their halves k < nh at columns w0, w1 of blocked slabs s0, s1
// (X1 = 0 when !has1), into the unpadded shared buffer z (read back through FlatLd).  Each
// stored element is read once and also gives the mirror z[n - k] (conj X0 + i conj X1);
// loads are issued in batches of kU per thread before their stores.  With amp (k < nh) the
// noise A(k) xi_w(k) of Eq. 1 is added to each half spectrum on the way (xi from noise_xi,
// key seed, wires w0 and w1).  Ends without a barrier.
__device__ __forceinline__ void stage_herm_pair(const float2* __restrict__ s0,
                                                const float2* __restrict__ s1, int w0, int w1,
                                                bool has1, int n_w, int nh, int n, float2* z,
                                                const float* __restrict__ amp = nullptr,
                                                uint64_t seed = 0, uint32_t plane_id = 0)
{
    constexpr int kU = 6;
    for (int base = threadIdx.x; base < nh; base += kU * blockDim.x) {
        float2 a[kU], b[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int kk = base + u * blockDim.x;
            a[u] = b[u] = make_float2(0.f, 0.f);
            if (kk < nh) {
                a[u] = ld_fresh(s0 + blk_index(kk, w0, n_w));
                if (has1) b[u] = ld_fresh(s1 + blk_index(kk, w1, n_w));
            }
        }
        if (amp) {
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int kk = base + u * blockDim.x;
                if (kk < nh) {
                    const float A = __ldg(amp + kk);
                    const float2 x0 = noise_xi((uint32_t)w0, kk, n, plane_id, seed);
                    a[u].x = fmaf(A, x0.x, a[u].x);
                    a[u].y = fmaf(A, x0.y, a[u].y);
                    if (has1) {
                        const float2 x1 = noise_xi((uint32_t)w1, kk, n, plane_id, seed);
                        b[u].x = fmaf(A, x1.x, b[u].x);
                        b[u].y = fmaf(A, x1.y, b[u].y);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int kk = base + u * blockDim.x;
            if (kk < nh) {
                z[kk] = make_float2(a[u].x - b[u].y, a[u].y + b[u].x);
                if (kk > 0 && n - kk >= nh) z[n - kk] = make_float2(a[u].x + b[u].y, b[u].x - a[u].y);
            }
        }
    }
}

// Ticks 2q and 2q + 1 of a transform in z (16-byte aligned); PAD: z is padded (run_plan; the two lie
// in one group of 16).
template <bool PAD>
__device__ __forceinline__ float4 tick_pair(const float2* z, int q)
{
    if constexpr (PAD) {
        const float2 *p = z + pad16(2 * q), a = p[0], b = p[1];
        return make_float4(a.x, a.y, b.x, b.y);
    } else {
        return reinterpret_cast<const float4*>(z)[q];
    }
}

// Write the two real rows of an inverse real-pair transform held in z (16-byte aligned; row 0 in
// .x, row 1 in .y; o1 ignored when !has1; PAD: z is padded), ticks t < n_t.  With vec (rows 8-byte
// aligned, n_t even) a thread takes 2 ticks: consecutive lanes read consecutive 16 bytes of shared
// memory, free of bank conflicts, and write 8 bytes of each row (four ticks per thread, with 16-byte
// stores, read 32 bytes apart: the inverse FFT of dL/dS took 144 us with it).
template <bool PAD>
__device__ __forceinline__ void store_real_pair(const float2* z, float* __restrict__ o0,
                                                float* __restrict__ o1, int n_t, bool has1,
                                                bool vec)
{
    if (vec) {
        float2* p0 = reinterpret_cast<float2*>(o0);
        float2* p1 = reinterpret_cast<float2*>(o1);
        for (int q = threadIdx.x; q < (n_t >> 1); q += blockDim.x) {
            const float4 a = tick_pair<PAD>(z, q);
            p0[q] = make_float2(a.x, a.z);
            if (has1) p1[q] = make_float2(a.y, a.w);
        }
    } else {
        for (int t = threadIdx.x; t < n_t; t += blockDim.x) {
            const float2 v = z[PAD ? pad16(t) : t];
            o0[t] = v.x;
            if (has1) o1[t] = v.y;
        }
    }
}

// store_real_pair for a residual: o = M - target (one FP32 subtraction of the value
// store_real_pair would write) for rows 0 (.x, target t0) and 1 (.y, t1); returns this
// thread's FP32 sum of the squared residuals it wrote.  vec: rows and targets 8-byte aligned,
// n_t even.
template <bool PAD>
__device__ __forceinline__ float store_residual_pair(const float2* z, float* __restrict__ o0,
                                                    float* __restrict__ o1,
                                                    const float* __restrict__ t0,
                                                    const float* __restrict__ t1, int n_t,
                                                    bool has1, bool vec)
{
    float ss = 0.0f;
    if (vec) {
        // the targets' 8-byte loads in batches of kU per row, issued before their use
        constexpr int kU = 6;
        const int nq = n_t >> 1;
        const float2 zero = make_float2(0.f, 0.f);
        for (int base = threadIdx.x; base < nq; base += kU * blockDim.x) {
            float2 ta[kU], tb[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int q = base + u * blockDim.x;
                ta[u] = tb[u] = zero;
                if (q < nq) {
                    ta[u] = __ldg(reinterpret_cast<const float2*>(t0) + q);
                    if (has1) tb[u] = __ldg(reinterpret_cast<const float2*>(t1) + q);
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int q = base + u * blockDim.x;
                if (q < nq) {
                    const float4 a = tick_pair<PAD>(z, q);
                    const float2 r0 = make_float2(__fsub_rn(a.x, ta[u].x), __fsub_rn(a.z, ta[u].y));
                    reinterpret_cast<float2*>(o0)[q] = r0;
                    ss += r0.x * r0.x + r0.y * r0.y;
                    if (has1) {
                        const float2 r1 = make_float2(__fsub_rn(a.y, tb[u].x), __fsub_rn(a.w, tb[u].y));
                        reinterpret_cast<float2*>(o1)[q] = r1;
                        ss += r1.x * r1.x + r1.y * r1.y;
                    }
                }
            }
        }
    } else {
        for (int t = threadIdx.x; t < n_t; t += blockDim.x) {
            const float2 v = z[PAD ? pad16(t) : t];
            const float r0 = __fsub_rn(v.x, t0[t]);
            o0[t] = r0;
            ss += r0 * r0;
            if (has1) {
                const float r1 = __fsub_rn(v.y, t1[t]);
                o1[t] = r1;
                ss += r1 * r1;
            }
        }
    }
    return ss;
}

// ADC code of waveform value m: clamp(floor(fl(fl(g m) + p) + 1/2), 0, top), each step one
// correctly rounded FP32 operation.
__device__ __forceinline__ uint16_t adc_code(float m, float g, float p, float top)
{
    const float x = __fadd_rn(__fmul_rn(g, m), p);
    const float c = floorf(__fadd_rn(x, 0.5f));
    return (uint16_t)fminf(fmaxf(c, 0.0f), top);
}

// store_real_pair for ADC codes: row 0 (.x) to o0, row 1 (.y) to o1, uint16.  With vec (rows
// 4-byte aligned, n_t even) a thread writes 2 codes per row with one 4-byte store.
template <bool PAD>
__device__ __forceinline__ void store_real_pair_adc(const float2* z, uint16_t* __restrict__ o0,
                                                    uint16_t* __restrict__ o1, int n_t, bool has1,
                                                    bool vec, float g, float p, float top)
{
    if (vec) {
        uint32_t* p0 = reinterpret_cast<uint32_t*>(o0);
        uint32_t* p1 = reinterpret_cast<uint32_t*>(o1);
        auto pack = [&](float u, float v) {
            return (uint32_t)adc_code(u, g, p, top) | ((uint32_t)adc_code(v, g, p, top) << 16);
        };
        for (int q = threadIdx.x; q < (n_t >> 1); q += blockDim.x) {
            const float4 a = tick_pair<PAD>(z, q);
            p0[q] = pack(a.x, a.z);
            if (has1) p1[q] = pack(a.y, a.w);
        }
    } else {
        for (int t = threadIdx.x; t < n_t; t += blockDim.x) {
            const float2 v = z[PAD ? pad16(t) : t];
            o0[t] = adc_code(v.x, g, p, top);
            if (has1) o1[t] = adc_code(v.y, g, p, top);
        }
    }
}

// All passes of plan p.  The first pass reads through `first` (global memory or a shared
// buffer outside X/Y), later passes ping-pong between X and Y.  Returns the buffer holding
// the transform; ends with a block barrier.
template <bool INV, int LOGB, class FirstLd>
__device__ __forceinline__ float2* run_plan(const FftPlan& p, const FirstLd& first, float2* X, float2* Y)
{
    float2* dst = X;
    for (int i = 0; i < p.npass; ++i) {
        const PassArgs a = {p.n, p.ns[i], p.ns_magic[i], p.tw + p.tw_off[i]};
        dst = (i & 1) ? Y : X;
        if (i == 0) {
            pass_any<INV, LOGB>(p.radix[0], first, SmemSt<LOGB>{dst}, a);
        } else {
            const float2* src = (i & 1) ? X : Y;
            pass_any<INV, LOGB>(p.radix[i], SmemLd<LOGB>{src}, SmemSt<LOGB>{dst}, a);
        }
        __syncthreads();
    }
    return dst;
}

// ------------------------------------------------------------------ in-place plans
// A single sequence in one shared buffer: in each pass every thread first loads the inputs of all
// its butterflies into registers, the block synchronises, and the outputs are written over the
// same buffer (one buffer per sequence instead of two, for more CTAs per SM).  The layout between
// two passes pads each group of ns R outputs of the first by one slot when the group is even, so
// that the first pass's stride-R writes spread over the banks; the groups divide the next pass's
// strides, so every address is base + r step, with one base per butterfly (a pad of one slot per
// 16 elements takes three operations per element where 16 does not divide the strides: a
// 6250-point transform of 8000 rows took 184 us with it).  The input and the result are unpadded.
//
// A pass of the runtime plan reads its length and stride at run time; a fixed one has them as
// template parameters.
struct RtPass {
    static constexpr bool kFew = false;
    int n, ns, T;
    uint32_t magic;
    const float2* tw;
    bool last;
    __device__ __forceinline__ int div_ns(int j) const
    {
        return ns == 1 ? j : (int)__umulhi((uint32_t)j, magic);
    }
};
template <int N, int NS, int THREADS, bool LAST>
struct FixedPass {
    static constexpr int n = N, ns = NS, T = THREADS;
    static constexpr bool last = LAST, kFew = true;
    const float2* tw;
    __device__ __forceinline__ int div_ns(int j) const { return j / NS; }
};

// Apply the twiddles w^(r k), r = 1 .. R - 1, of a pass to v[1 ..]; tw the pass's table (entry
// (r - 1) ns + k = w^(r k)).  FEW, radix 15: only the entries of r = 1, 5 and 10 are read and the
// rest formed as products of them (w^(3k) = w^(5k) conj(w^(2k)) and so on, each at most three
// roundings away from correctly rounded table values), 3 table entries instead of 14.
template <int R, bool INV, bool FEW>
__device__ __forceinline__ void apply_twiddles(float2* v, const float2* __restrict__ tw, int ns,
                                               uint32_t k)
{
    if constexpr (R == 15 && FEW) {
        const float2 a = __ldg(tw + k), b = __ldg(tw + 4 * ns + k), c = __ldg(tw + 9 * ns + k);
        const float2 na = make_float2(a.x, -a.y);                  // conj: w^(-k)
        const float2 a2 = cmul(a, a), na2 = make_float2(a2.x, -a2.y);
        const float2 a3 = cmul(b, na2), a4 = cmul(b, na);
        float2 w[15];
        w[1] = a;            w[2] = a2;            w[3] = a3;            w[4] = a4;
        w[5] = b;            w[6] = cmul(b, a);    w[7] = cmul(b, a2);   w[8] = cmul(c, na2);
        w[9] = cmul(c, na);  w[10] = c;            w[11] = cmul(c, a);   w[12] = cmul(c, a2);
        w[13] = cmul(c, a3); w[14] = cmul(c, a4);
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = twiddle<INV>(v[r], w[r]);
    } else {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = twiddle<INV>(v[r], __ldg(tw + (r - 1) * ns + k));
    }
}

// The twiddles w^(r k) to va and their conjugates to vb.  Radix 15 reads the entries of r = 1, 2,
// 5, 10 and 14 and forms the others as products of two of them: both halves of a pair see one
// error here, which no longer averages out between them, so it is kept at one product.
template <int R>
__device__ __forceinline__ void pair_twiddles(float2* va, float2* vb, const float2* __restrict__ tw,
                                              int ns, uint32_t k)
{
    float2 w[R];
    if constexpr (R == 15) {
        const float2 a = __ldg(tw + k), a2 = __ldg(tw + ns + k), b = __ldg(tw + 4 * ns + k);
        const float2 c = __ldg(tw + 9 * ns + k), e = __ldg(tw + 13 * ns + k);
        const float2 na = make_float2(a.x, -a.y), na2 = make_float2(a2.x, -a2.y);
        w[1] = a;            w[2] = a2;            w[3] = cmul(b, na2);  w[4] = cmul(b, na);
        w[5] = b;            w[6] = cmul(b, a);    w[7] = cmul(b, a2);   w[8] = cmul(c, na2);
        w[9] = cmul(c, na);  w[10] = c;            w[11] = cmul(c, a);   w[12] = cmul(c, a2);
        w[13] = cmul(e, na); w[14] = e;
    } else {
#pragma unroll
        for (int r = 1; r < R; ++r) w[r] = __ldg(tw + (r - 1) * ns + k);
    }
#pragma unroll
    for (int r = 1; r < R; ++r) {
        va[r] = twiddle<false>(va[r], w[r]);
        vb[r] = twiddle<true>(vb[r], w[r]);
    }
}

// One in-place pass of radix R, at most NI butterflies per thread; the block has P.T threads.
// Ends with a block barrier.
template <int R, bool INV, int NI, class P>
__device__ __forceinline__ void pass_inplace(float2* buf, const P& p)
{
    const int nb = p.n / R, ns = p.ns;
    const int pad_in = (ns > 1 && (ns & 1) == 0) ? 1 : 0;
    const int pad_out = (!p.last && ((ns * R) & 1) == 0) ? 1 : 0;
    const int rd_step = nb + pad_in * p.div_ns(nb);
    float2 v[NI][R];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int j = threadIdx.x + i * p.T;
        if (j < nb) {
            const float2* src = buf + j + pad_in * p.div_ns(j);
#pragma unroll
            for (int r = 0; r < R; ++r) v[i][r] = src[r * rd_step];
        } else {
            // (unset, the values would be carried from one pass of the plan's loop to the next,
            // and those of every radix stay live)
#pragma unroll
            for (int r = 0; r < R; ++r) v[i][r] = make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int j = threadIdx.x + i * p.T;
        if (j < nb) {
            const int q = p.div_ns(j), k = j - q * ns;
            if (k > 0) apply_twiddles<R, INV, P::kFew>(v[i], p.tw, ns, (uint32_t)k);
            dft<R, INV>(v[i]);
            float2* dst = buf + q * (ns * R + pad_out) + k;
#pragma unroll
            for (int r = 0; r < R; ++r) dst[r * ns] = v[i][r];
        }
    }
    __syncthreads();
}

// The last pass of a forward transform of a real pair z = x0 + i x1, with the two half spectra
// taken apart in registers: X0(k) = (Z(k) + conj Z(n - k)) / 2 to f[k] and X1(k) = (Z(k) - conj
// Z(n - k)) / 2i to f[o1 + k], k <= n / 2.  With nb = n / R butterflies, outputs a + r nb of
// butterfly a mirror those of butterfly nb - a, so a thread takes both (units a = 0 .. nb / 2, NI
// per thread).  The twiddles of nb - a are those of a conjugated times W_R^r, and the factor W_R^r
// turns its outputs by one: with v_b the transform without it, Z(n - a - r nb) = v_b[(R - r) mod R]
// for every a, a = 0 (butterfly 0 twice) and a = nb / 2 included (whose values are written twice).
// This saves writing the transform and reading it back, a fifth of the kernel's shared-memory
// traffic.  f may overlap buf.  Ends without a barrier.
template <int R, int NI, class P>
__device__ __forceinline__ void last_pass_pairs(const float2* buf, const P& p, float2* f, int o1)
{
    const int nb = p.n / R, units = nb / 2 + 1;
    const int pad_in = (p.ns > 1 && (p.ns & 1) == 0) ? 1 : 0;
    const int rd_step = nb + pad_in;                   // ns == nb: one group
    float2 va[NI][R], vb[NI][R];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int a = threadIdx.x + i * p.T;
        if (a < units) {
            const float2 *sa = buf + a, *sb = buf + (a ? nb - a : 0);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                va[i][r] = sa[r * rd_step];
                vb[i][r] = sb[r * rd_step];
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) va[i][r] = vb[i][r] = make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int a = threadIdx.x + i * p.T;
        if (a < units) {
            if (a > 0) pair_twiddles<R>(va[i], vb[i], p.tw, p.ns, (uint32_t)a);
            dft<R, false>(va[i]);
            dft<R, false>(vb[i]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 u = va[i][r], w = vb[i][(R - r) % R];
                const float2 x0 = make_float2(0.5f * (u.x + w.x), 0.5f * (u.y - w.y));
                const float2 x1 = make_float2(0.5f * (u.y + w.y), 0.5f * (w.x - u.x));
                if (r <= (R - 1) / 2) {                // k = a + r nb <= n / 2
                    f[a + r * nb] = x0;
                    f[o1 + a + r * nb] = x1;
                } else {                               // n - k, the conjugates
                    f[(R - r) * nb - a] = make_float2(x0.x, -x0.y);
                    f[o1 + (R - r) * nb - a] = make_float2(x1.x, -x1.y);
                }
            }
        }
    }
}

// The first pass of an inverse transform of a real pair, z(k) = X0(k) + i X1(k), from the two half
// spectra: load(k, x0, x1) gives X0(k), X1(k), k <= n / 2, and z(n - k) = conj X0(k) + i conj
// X1(k).  Inputs a + r nb of butterfly a mirror those of butterfly nb - a, so a thread that takes
// both (units a = 0 .. nb / 2) reads each half-spectrum value once, all of them before the first
// butterfly, and nothing is staged in shared memory.  Ends with a block barrier.
template <int R, int NI, class P, class Load>
__device__ __forceinline__ void first_pass_pairs(float2* buf, const P& p, const Load& load)
{
    const int nb = p.n / R, units = nb / 2 + 1;
    const int pad = (!p.last && (R & 1) == 0) ? 1 : 0;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int a = threadIdx.x + i * p.T;
        if (a >= units) break;
        float2 va[R], vb[R];
#pragma unroll
        for (int r = 0; r <= (R - 1) / 2; ++r) load(a + r * nb, va[r], vb[R - 1 - r]);
#pragma unroll
        for (int r = 0; r < R / 2; ++r) load((r + 1) * nb - a, vb[r], va[R - 1 - r]);
        // (x0, x1) -> z(k) and z(n - k)
        auto pair = [](float2& u, float2& w) {
            const float2 x0 = u, x1 = w;
            u = make_float2(x0.x - x1.y, x0.y + x1.x);
            w = make_float2(x0.x + x1.y, x1.x - x0.y);
        };
#pragma unroll
        for (int r = 0; r <= (R - 1) / 2; ++r) pair(va[r], vb[R - 1 - r]);
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            pair(vb[r], va[R - 1 - r]);
            if (2 * (r + 1) == R && a == 0) va[R - 1 - r] = vb[r];     // k = n / 2 as it stands
        }
        dft<R, true>(va);
        float2* dst = buf + a * (R + pad);
#pragma unroll
        for (int r = 0; r < R; ++r) dst[r] = va[r];
        if (a > 0) {
            dft<R, true>(vb);
            dst = buf + (nb - a) * (R + pad);
#pragma unroll
            for (int r = 0; r < R; ++r) dst[r] = vb[r];
        }
    }
    __syncthreads();
}

// Units of butterflies a and nb - a of radix R that a thread holds at once (32 complex values);
// none above radix 16.
__host__ __device__ constexpr int row_pair_units(int R) { return 16 / R; }

// The passes of the compile-time plan (R0, R1, R2) for a block of exactly T threads, [FIRST, END)
// of them.
template <bool INV, int R0, int R1, int R2, int T, int FIRST = 0, int END = 3>
__device__ __forceinline__ void run_plan_fixed(const FftPlan& p, float2* X)
{
    constexpr int N = R0 * R1 * R2;
    constexpr int N0 = (N / R0 + T - 1) / T, N1 = (N / R1 + T - 1) / T, N2 = (N / R2 + T - 1) / T;
    if constexpr (FIRST <= 0 && END > 0)
        pass_inplace<R0, INV, N0>(X, FixedPass<N, 1, T, false>{p.tw + p.tw_off[0]});
    if constexpr (FIRST <= 1 && END > 1)
        pass_inplace<R1, INV, N1>(X, FixedPass<N, R0, T, false>{p.tw + p.tw_off[1]});
    if constexpr (FIRST <= 2 && END > 2)
        pass_inplace<R2, INV, N2>(X, FixedPass<N, R0 * R1, T, true>{p.tw + p.tw_off[2]});
}

// Butterflies of radix R that a thread of a runtime plan holds at once: at most 32 complex values
// (64 registers).
__host__ __device__ constexpr int row_butterflies(int R) { return R > 16 ? 1 : 32 / R; }

__device__ __forceinline__ RtPass rt_pass(const FftPlan& p, int i)
{
    return {p.n, p.ns[i], (int)blockDim.x, p.ns_magic[i], p.tw + p.tw_off[i], i + 1 == p.npass};
}

// Passes [first, end) of the runtime plan p, for a block of row_threads(p) threads.  (A plan of
// one point has radix 1 and nothing to do.)
template <bool INV>
__device__ __forceinline__ void run_plan_inplace(const FftPlan& p, float2* X, int first, int end)
{
    for (int i = first; i < end; ++i) {
        const RtPass a = rt_pass(p, i);
        switch (p.radix[i]) {
#define WCSIM_CASE(RR) case RR: pass_inplace<RR, INV, row_butterflies(RR)>(X, a); break;
            WCSIM_FOR_EACH_RADIX(WCSIM_CASE)
#undef WCSIM_CASE
        }
    }
}

// Threads of a row kernel for plan p: every pass fits its butterflies, at least 128 (so that a
// short transform still has the warps to hide its shared-memory latency), whole warps.
__host__ inline int row_threads(const FftPlan& p)
{
    int t = 128;
    for (int i = 0; i < p.npass; ++i) {
        const int nb = p.n / p.radix[i], ni = row_butterflies(p.radix[i]);
        const int need = (nb + ni - 1) / ni;
        if (need > t) t = need;
    }
    return (t + 31) & ~31;
}

// Row-kernel instances: the compile-time 6000-point plan (radices 16, 25, 15; 256 threads); the
// runtime plan in place, for blocks of up to 384, 448 and 704 threads; and the runtime plan between
// two buffers (run_plan, 256 threads).  The in-place ones keep 72 (448) to 80 registers per thread, so
// that registers and shared memory give out together: 24 warps per SM at 6000 points, 26 at 9600,
// where two buffers leave 8 to 16.  What they pay for it is code: every pass unrolls the butterflies
// that a thread holds (the runtime ones spill 48 to 200 bytes per thread, that of 448 threads 192 to
// 836), and a kernel of one wave or two spends much of its time fetching instructions.
enum RowVariant : int { kRow6000 = 0, kRow384, kRow448, kRow704, kRowTwo, kRowVariants };
__host__ __device__ constexpr int row_max_threads(int v)
{
    return v == kRow384 ? 384 : v == kRow448 ? 448 : v == kRow704 ? 704 : 256;
}
__host__ __device__ constexpr int row_min_ctas(int v)
{
    return v == kRow6000 ? 3 : v == kRow704 ? 1 : 2;
}

__host__ inline bool is_plan6000(const FftPlan& p)
{
    return p.n == 6000 && p.npass == 3 && p.radix[0] == 16 && p.radix[1] == 25 && p.radix[2] == 15;
}

// Block of an in-place row kernel for plan p over `ctas` CTAs: what the plan needs; 256 threads at least
// when the CTAs are few for the SMs (a short transform's staging and stores are then what a CTA waits
// for), or instead of 128 from 3500 points on (9600 rows of 4096 points 134 -> 127 us, 2500 of 3840
// 53.6 -> 47.9; of 3072 points 94 -> 107, the other way round).
__host__ inline int row_block(const FftPlan& p, int64_t ctas)
{
    const int t = row_threads(p);
    if (t < 256 && (ctas < 4 * (int64_t)sm_count() || (t == 128 && p.n > 3500))) return 256;
    return t;
}

// Whether pass i of plan p, its first or last, can run on units of two mirrored butterflies: the
// block that the other passes ask for holds them all.
__host__ inline bool row_pairs(const FftPlan& p, int i)
{
    if (is_plan6000(p)) return true;
    const int u = row_pair_units(p.radix[i]);
    return p.radix[i] > 1 && u > 0 && p.n / p.radix[i] / 2 + 1 <= u * row_threads(p);
}

// Radices with units of two butterflies.
#define WCSIM_FOR_EACH_PAIR_RADIX(X) \
    X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(10) X(12) X(14) X(15) X(16)

// Forward transform of the real pair staged in X.  pairs (row_pairs of the last pass): the two half
// spectra in f and f + o1, which may overlap X, without a final barrier; else the transform in X.
template <int V>
__device__ __forceinline__ void run_row_forward(const FftPlan& p, float2* X, bool pairs, float2* f,
                                                int o1)
{
    if constexpr (V == kRow6000) {
        run_plan_fixed<false, 16, 25, 15, 256, 0, 2>(p, X);
        if (pairs)
            last_pass_pairs<15, 1>(X, FixedPass<6000, 400, 256, true>{p.tw + p.tw_off[2]}, f, o1);
        else
            run_plan_fixed<false, 16, 25, 15, 256, 2, 3>(p, X);
    } else {
        run_plan_inplace<false>(p, X, 0, pairs ? p.npass - 1 : p.npass);
        if (pairs) {
            const RtPass a = rt_pass(p, p.npass - 1);
            switch (p.radix[p.npass - 1]) {
#define WCSIM_CASE(RR) case RR: last_pass_pairs<RR, row_pair_units(RR)>(X, a, f, o1); break;
                WCSIM_FOR_EACH_PAIR_RADIX(WCSIM_CASE)
#undef WCSIM_CASE
            }
        }
    }
}

// Inverse transform of the pair staged in X, in X.
template <int V>
__device__ __forceinline__ void run_row_inverse(const FftPlan& p, float2* X)
{
    if constexpr (V == kRow6000) run_plan_fixed<true, 16, 25, 15, 256>(p, X);
    else run_plan_inplace<true>(p, X, 0, p.npass);
}

// Inverse transform of the real pair with half spectra at columns w0 and w0 + 1 (X1 = 0 when
// !has1) of the blocked slab s into X, without staging them (row_pairs of the first pass).  It
// loads with the few hundred threads that hold units: where the grid is many times the resident
// CTAs that is faster (dL/dS of the 960 x 6000 plane 144 -> 126 us), where a launch is about one
// wave the longer chain of a CTA shows (the frame's own inverse, 480 CTAs: 27 -> 37 us, so that
// kernel stages).
template <int V>
__device__ __forceinline__ void run_row_inverse_pairs(const FftPlan& p, float2* X,
                                                      const float2* __restrict__ s, int w0,
                                                      bool has1, int n_w)
{
    const float2* col = s + (int64_t)w0 * kBlockCols;
    auto load = [&](int k, float2& x0, float2& x1) {
        const float2* q = col + (int64_t)(k >> 2) * n_w * kBlockCols + (k & 3);
        x0 = __ldg(q);
        x1 = has1 ? __ldg(q + kBlockCols) : make_float2(0.f, 0.f);
    };
    if constexpr (V == kRow6000) {
        first_pass_pairs<16, 1>(X, FixedPass<6000, 1, 256, false>{p.tw}, load);
        run_plan_fixed<true, 16, 25, 15, 256, 1, 3>(p, X);
    } else {
        const RtPass a = rt_pass(p, 0);
        switch (p.radix[0]) {
#define WCSIM_CASE(RR) case RR: first_pass_pairs<RR, row_pair_units(RR)>(X, a, load); break;
            WCSIM_FOR_EACH_PAIR_RADIX(WCSIM_CASE)
#undef WCSIM_CASE
        }
        run_plan_inplace<true>(p, X, 1, p.npass);
    }
}

// Shared bytes of an in-place row kernel for plan p: n complex values and one pad per even group of
// the passes' layouts (at least padded_len(n), which the flat rows of the TMA stores are sized to).
__host__ inline size_t row_plan_smem(const FftPlan& p)
{
    int len = padded_len(p.n);
    for (int i = 0; i + 1 < p.npass; ++i) {
        const int group = p.ns[i] * p.radix[i];
        if ((group & 1) == 0 && p.n + p.n / group > len) len = p.n + p.n / group;
    }
    return (size_t)len * sizeof(float2);
}

// How a row transform of plan p over `ctas` CTAs is launched.  pairs: the spectra of S and the inverse
// of dL/dS may take mirrored butterflies together.
enum RowUse : int { kRowForward, kRowFrame, kRowGrid };
struct RowLaunch {
    RowVariant variant;
    int threads;
    size_t smem;
    bool pairs;
};

// In place or between two buffers?  In place puts more CTAs on an SM and can pair butterflies; two
// buffers run a fraction of the code, which a launch of one round or two spends most of its time
// fetching.  So the rounds that the CTAs take either way decide, up to 6000 points (above 6700 two
// buffers leave one CTA per SM; between, in place is ahead).  Times between two buffers over times in
// place, 64 to 960 wires x 10 rows, 512 to 5760 points:
// - the frame's inverse: 0.75 to 0.97 where two buffers need no more rounds, 1.1 to 1.3 where they do;
// - spectra of S and inverse of dL/dS: 0.65 to 1.0 where a second round in place is a small one (480
//   CTAs, at 160 threads 640 to 800), 1.0 to 1.8 else.  Two buffers may take 6/5 the rounds for the
//   spectra, 8/5 up to 4200 points, 2 from 3000 there without pairs where there is a second round (4000
//   points, 1280 CTAs: 0.93), and 8/5 for the inverse; from four rounds in place on they never do;
// - except that passes of radix 16 and more, without pairs, gain nothing in place (4096 points: 0.91 to
//   0.97 at any size).
__host__ inline RowLaunch row_launch(const FftPlan& p, int64_t ctas, RowUse use, bool pairs)
{
    if (is_plan6000(p)) return {kRow6000, 256, row_plan_smem(p), pairs};
    pairs = pairs && row_pairs(p, use == kRowForward ? p.npass - 1 : 0);
    const int t = row_block(p, ctas);
    const RowVariant v = t <= 384 ? kRow384 : t <= 448 ? kRow448 : kRow704;
    const size_t one = row_plan_smem(p), two = 2 * (size_t)padded_len(p.n) * sizeof(float2);
    const size_t sm = 228 * 1024, reserved = 1024;              // shared memory of an SM, and per CTA
    auto rounds = [&](int per_regs, size_t bytes) {
        const int64_t fit = (int64_t)(sm / (bytes + reserved));
        const int64_t per = (fit < per_regs ? (fit > 0 ? fit : 1) : per_regs) * sm_count();
        return (ctas + per - 1) / per;
    };
    // warps per SM by registers: 6 per quarter at 80 registers, 7 at 72
    const int64_t r1 = rounds((v == kRow448 ? 28 : 24) / (t / 32), one), r2 = rounds(2, two);
    bool use_two = false;
    if (use == kRowFrame) {
        use_two = p.n <= 6000 && r2 <= r1;
    } else if (p.n <= 6000 && r1 <= 3) {
        const int fifths = use == kRowGrid ? 8 : p.n > 4200 ? 6 : !pairs && r1 > 1 && p.n > 3000 ? 10 : 8;
        use_two = 5 * r2 <= fifths * r1;
    }
    if (use == kRowForward && !pairs && p.n <= 6700) {
        bool large = true;
        for (int i = 0; i < p.npass; ++i) large = large && p.radix[i] >= 16;
        use_two = use_two || large;
    }
    if (use_two) return {kRowTwo, 256, two, false};
    return {v, t, one, pairs};
}

// The instance of kernel template K for variant v.
#define WCSIM_ROW_KERNEL(K, v)                                                                    \
    ((v) == kRow6000 ? K<kRow6000> : (v) == kRow384 ? K<kRow384> : (v) == kRow448 ? K<kRow448>    \
     : (v) == kRow704 ? K<kRow704> : K<kRowTwo>)

}  // namespace wcsim
