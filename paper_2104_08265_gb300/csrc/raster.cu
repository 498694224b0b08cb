// Drift, rasterization, fluctuation and scatter-add of depos into the impact x tick grid
// (Sec. 2.1.1 "rasterization" and "scatter adding"; drift and diffusion as in Fig. 2;
// fluctuation with a Box-Muller normal as in Sec. 4.3.1).
//
// Work split.  A warp owns a run of consecutive depos (4 to 32, chosen by the number of depos).
// Its lanes take the bin decision of one depo each and park what the rasterization needs of it in
// shared memory; then each group of 8 lanes takes the warp's depos one by one (the four groups of
// a warp work on four depos side by side): its lanes form the 1D weights of the patch (rows and ticks
// together) in shared memory, each from a series about the bin's centre, or where bins are wide
// against sigma from differences of one erfc per bin edge, and stride over (row, 4-tick group) items.
// Warps never wait for one another.
// An item draws one Philox block for its four ticks when fluctuating (four Box-Muller
// normals), forms Q' w_p w_t per bin and adds the four values into the grid with one
// vector reduction.  The exact binomial fluctuation (an instance of its own) strides over
// single bins instead: each draw walks its bin's CDF, and neighbouring ticks, whose walks
// cost alike, then run side by side in a group.  With renormalisation the weights of each
// axis are divided by the mass of its unclipped n-sigma window (folded into the per-depo
// scale of the decision).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "async_copy.cuh"
#include "binomial.cuh"
#include "depo_common.cuh"
#include "rng.cuh"
#include "wcsim_internal.cuh"

namespace wcsim {
namespace {

constexpr int kRasterWarps = 4; // warps per block
constexpr int kWmax = 32;       // weights per axis held per patch tile

// Exact binomial fluctuation of the bin (row r, tick k) with mean v: x ~ Binomial(N, p) with
// N = rint(Q') whole electrons and p = v / Q', drawn by inversion at the 23-bit uniform of
// word k mod 4 of the bin's Philox block (the block the normal approximation uses).  A bin
// whose variance N p (1 - p) exceeds 65536, or N above 2^24, takes the normal
// approximation instead.
__device__ __forceinline__ float binomial_bin(const RasterConsts& c, float qatt, uint32_t id, int k,
                                              int64_t r, float v, float inv_q, const float* stirl)
{
    const uint4 x = philox_rounds<0>(make_uint4((uint32_t)(k >> 2), (uint32_t)r, id, c.plane_id),
                                     c.keys);
    const int e = k & 3;
    const float n = rintf(qatt);
    const float p = fminf(1.0f, v * inv_q);
    if (n > 16777216.0f || n * p * (1.0f - p) > 65536.0f) {
        float z[4];
        box_muller4(x, z);
        const float ze = e == 0 ? z[0] : e == 1 ? z[1] : e == 2 ? z[2] : z[3];
        const float var = v * (1.0f - v * inv_q);
        return fmaxf(0.0f, fmaf(sqrt_fast(var), ze, v));
    }
    if (n == 0.0f) return 0.0f;
    if (p >= 1.0f) return n;
    const uint32_t w = e == 0 ? x.x : e == 1 ? x.y : e == 2 ? x.z : x.w;
    return binomial_inverse(n, p, uniform23(w), stirl);
}

// What the lanes of a group need of one depo, formed once by the lane that decides it.  Bin edge e
// of the window (e bins above its first) lies at u = ((off + e) - frac) s, off the window's first
// bin relative to the floor of the position (exact in FP32 below 2^24 bins).  A point (sigma == 0,
// all weight in the window's one bin) has its edges far out on either side of that bin's centre: the
// bin is the next one (off == 1) for a position so little below an edge that frac rounds up to 1.
//
// Bin masses come in two forms.  In general they are differences of erfc at the edges.  Where the
// bins are not wide against sigma, the mass about a bin's centre c (in units of sqrt(2) sigma,
// half width s / 2) is
//   1/2 (erf(c + s/2) - erf(c - s/2)) = erf(s/2) e^(-c^2) sum_k A_k / A_0 (c s)^(2k) / (2k)!,
//   A_k = int_0^1 x^(2k) e^(-(s x / 2)^2) dx,
// (the even part of e^(-2 c x) in the integral of e^(-(c + x)^2)): one exponential and ten terms,
// all positive, per bin, with no cancellation, where the erfc form takes two edges and loses the
// digits their difference cancels.  `series` marks a depo whose bins all have (c s)^2 <= 20 and
// s <= 2.8 on both axes (sigma above about half a bin at 3 sigma), where ten terms and the
// recurrence below leave less than 5e-8.
// Instructions per four depos (960 x 6000 plane, warp counts): 400 with erfc, 170 with the series.
constexpr int kTerms = 10;
struct __align__(16) PatchDepo {
    int32_t r_lo, nr, k_lo, nt;      // window; nr == 0: the depo adds nothing
    float off_p, frac_p, s_p, qw;
    float off_t, frac_t, s_t, inv_q;
    float qatt;
    uint32_t id;
    int32_t series;
    float pad;
    float term[2][kTerms + 2];       // series_terms of the ticks and of the rows
};

// (float)k, by the 32-bit conversion where it holds k.
__device__ __forceinline__ float offset_float(int64_t k)
{
    const int32_t k32 = (int32_t)k;
    return (int64_t)k32 == k ? (float)k32 : (float)k;
}

__device__ __forceinline__ void edge_axis(float sigma, float bin, float off, float frac, float& f,
                                          float& s)
{
    const bool point = !(sigma > 0.0f);
    s = point ? 1e30f : bin / (1.41421356237309505f * sigma);
    f = point ? off + 0.5f : frac;
}

// Series terms of one axis: term[0] = erf(s / 2), the mass of a bin about the mean, to which the
// series comes down at c = 0, and term[k] = A_k / (A_0 (2k)!), with A_k by the downward recurrence
// A_k = (e^(-h^2) + 2 h^2 A_(k+1)) / (2k + 1), h = s / 2, from the first terms of its own
// expansion at k = 10.  What scales a whole patch is rounded once, scale and bias included: a
// frame sums patches over many bins, where such errors add up and those of single bins average
// out.
__device__ __forceinline__ void series_terms(float s, float scale, float bias, float* term)
{
    constexpr float kInvFact[kTerms] = {1.0f, 5.0e-1f, 4.1666666666667e-2f, 1.3888888888889e-3f,
                                        2.4801587301587e-5f, 2.7557319223986e-7f,
                                        2.0876756987868e-9f, 1.1470745597729e-11f,
                                        4.7794773323874e-14f, 1.5619206968586e-16f};   // 1 / (2k)!
    const float h2 = 0.25f * s * s, g = 2.0f * h2, e = expf(-h2);
    float A[kTerms];
    float a = e * (1.0f / 21.0f) * (1.0f + g * (1.0f / 23.0f) * (1.0f + g * (1.0f / 25.0f)));
#pragma unroll
    for (int k = kTerms - 1; k >= 0; --k) {
        a = fmaf(g, a, e) * (1.0f / (2 * k + 1));
        A[k] = a;
    }
    const float r = 1.0f / A[0];
    const float m = erff(0.5f * s), t0 = scale * m;
    term[0] = t0 + fmaf(t0, bias, fmaf(scale, m, -t0));      // scale m (1 + bias), rounded once
#pragma unroll
    for (int k = 1; k < kTerms; ++k) term[k] = A[k] * (r * kInvFact[k]);
}

__device__ __forceinline__ bool series_axis(float off, float n, float frac, float s)
{
    const float c = fmaxf(fabsf((off + 0.5f) - frac), fabsf((off + (n - 0.5f)) - frac)) * s;
    return c * s <= 4.47f && s <= 2.8f;   // sqrt(20); s far above for a point
}

// ex2.approx truncates: its mean relative error measured -2e-8 over (-1/4, 0), -3.2e-8 over
// (-1, 0) and -5.0e-8 over (-7, 0).  Weighted by the masses, and with the rounding of log2 e, the
// two factors of a bin took 7.7e-8 off the total of a patch (48,000 patches against 64 bits),
// which the row factor puts back.
constexpr float kEx2Bias = 7.7e-8f;

template <int MODE>
__device__ __forceinline__ void make_patch(const RasterConsts& c, const Decision& r, PatchDepo& out)
{
    PatchDepo p;
    if (!r.ok || !(r.qatt > 0.0f)) {                      // nothing, or Q' underflowed
        out.nr = 0;
        return;
    }
    p.r_lo = r.r_lo;
    p.nr = r.r_hi - r.r_lo + 1;
    p.k_lo = r.k_lo;
    p.nt = r.k_hi - r.k_lo + 1;
    p.off_p = offset_float((int64_t)r.r_lo - r.i0p);
    p.off_t = offset_float((int64_t)r.k_lo - r.i0t);
    edge_axis(r.sp, c.dp_f, p.off_p, r.frac_p, p.frac_p, p.s_p);
    edge_axis(r.st, c.dt_f, p.off_t, r.frac_t, p.frac_t, p.s_t);
    p.qw = r.qw;
    p.qatt = r.qatt;
    p.inv_q = 1.0f / r.qatt;
    p.id = r.id;
    // the exact binomial keeps the erfc form: its integer draws then stay as they are
    p.series = MODE != 2 && series_axis(p.off_p, (float)p.nr, p.frac_p, p.s_p) &&
               series_axis(p.off_t, (float)p.nt, p.frac_t, p.s_t);
    if (MODE != 2 && p.series) {
        series_terms(p.s_t, 1.0f, 0.0f, p.term[0]);
        series_terms(p.s_p, p.qw, kEx2Bias, p.term[1]);
    }
    out = p;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Shared memory of one warp: its depos, then per group of lanes the weights of a patch tile.  A
// row record is the row's weight (MODE 1: with the row's words of the
// Philox second round), a quad record the weights of the four ticks 4 (q_lo + i) .. (zero outside
// the window; MODE 1: with the quad's Philox words), read with 16-byte loads.
constexpr int kMaxQuads = (kWmax + 3 + 3) / 4;

template <int MODE>
struct TileLayout {
    static constexpr int kRow = MODE == 1 ? 4 : 1;       // floats per row record
    static constexpr int kQuad = MODE == 1 ? 8 : 4;      // floats per quad record
    static constexpr int kGroupBytes = kMaxQuads * kQuad * 4 + kWmax * kRow * 4;
};

__host__ __device__ constexpr int raster_warp_smem(int mode, int depos_per_warp, int lanes_per_depo)
{
    return depos_per_warp * (int)sizeof(PatchDepo) +
           (32 / lanes_per_depo) * (mode == 1 ? TileLayout<1>::kGroupBytes : TileLayout<0>::kGroupBytes);
}

// The depos [base, base + dpw) of one event, dpw <= 32, by one warp: each lane decides one, then
// each group of G lanes rasterizes one depo at a time.  MODE is the fluctuation mode (0 mean, 1
// normal approximation, 2 exact binomial).
template <int G, int MODE>
__device__ __forceinline__ void rasterize_warp(const RasterConsts& c, const DepoArrays& d,
                                               float* __restrict__ grid, int* flags, int64_t base,
                                               int dpw, unsigned char* smem, const float* stirl)
{
    static_assert(G == 8 || G == 16 || G == 32, "lanes per depo");
    using L = TileLayout<MODE>;
    constexpr int NG = 32 / G;
    const int lane = threadIdx.x & 31, gl = lane % G, grp = lane / G;
    // the lanes of this group within its warp
    const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << (G & 31)) - 1u) << (lane & ~(G - 1)));
    PatchDepo* dep = reinterpret_cast<PatchDepo*>(smem);
    if (lane < dpw) {
        const int64_t i = base + lane;
        Decision r;
        r.ok = 0;
        if (i < d.n) {
            r = decide(c, d, i, flags, true);
            if (r.ok) r.id = d.id[i];
        }
        make_patch<MODE>(c, r, dep[lane]);
    }
    __syncwarp();
    // 16-byte reductions need 4-tick groups to start on 16-byte boundaries
    const bool vec4 = ((c.n_ticks & 3) == 0) && ((reinterpret_cast<uintptr_t>(grid) & 15) == 0);
    float* quad = reinterpret_cast<float*>(smem + dpw * sizeof(PatchDepo) + grp * L::kGroupBytes);
    float* row = quad + kMaxQuads * L::kQuad;

#pragma unroll 1
    for (int i = grp; i < dpw; i += NG) {
        const PatchDepo& pd = dep[i];
        const int nr_all = pd.nr, nt_all = pd.nt;
        const float off_p = pd.off_p, frac_p = pd.frac_p, s_p = pd.s_p, qw = pd.qw;
        const float off_t = pd.off_t, frac_t = pd.frac_t, s_t = pd.s_t, inv_q = pd.inv_q;

#pragma unroll 1
        for (int32_t ra = 0; ra < nr_all; ra += kWmax) {
            const int nr = min(kWmax, nr_all - ra), r0 = pd.r_lo + ra;
#pragma unroll 1
            for (int32_t ka = 0; ka < nt_all; ka += kWmax) {
                const int nt = min(kWmax, nt_all - ka), k0 = pd.k_lo + ka;
                const int q_lo = k0 >> 2, nq = ((k0 + nt - 1) >> 2) - q_lo + 1;
                const int koff = k0 & 3;                   // slot of tick k0
                for (int q = gl; q < nq; q += G) {
                    *reinterpret_cast<float4*>(quad + L::kQuad * q) = make_float4(0.f, 0.f, 0.f, 0.f);
                    if constexpr (MODE == 1)
                        *reinterpret_cast<uint4*>(quad + L::kQuad * q + 4) =
                            philox_quad(c.keys, c.plane_id, pd.id, (uint32_t)(q_lo + q));
                }
                __syncwarp(gmask);
                // the weight w of tick ka + i (row < 0) or of row ra + row into its record
                auto put = [&](int i, int row_i, float w) {
                    if (row_i < 0) {
                        const int p = i + koff;
                        quad[L::kQuad == 4 ? p : (p >> 2) * L::kQuad + (p & 3)] = w;
                    } else if constexpr (MODE == 1) {
                        const uint64_t h = philox_row(c.keys, pd.id, (uint32_t)(r0 + row_i));
                        *reinterpret_cast<float4*>(row + 4 * row_i) =
                            make_float4(w, __uint_as_float((uint32_t)(h >> 32)),
                                        __uint_as_float((uint32_t)h), 0.0f);
                    } else {
                        row[row_i] = w;
                    }
                };
                if (MODE != 2 && pd.series) {
                    const float bt = off_t + ((float)ka + 0.5f), bp = off_p + ((float)(ra - nt) + 0.5f);
                    for (int e = gl; e < nt + nr; e += G) {
                        const bool tick = e < nt;
                        const float4* tm = reinterpret_cast<const float4*>(pd.term[tick ? 0 : 1]);
                        const float sc = tick ? s_t : s_p;
                        const float cc = (((tick ? bt : bp) + (float)e) - (tick ? frac_t : frac_p)) * sc;
                        const float cs = cc * sc, y = cs * cs;
                        const float4 t0 = tm[0], t1 = tm[1], t2 = tm[2];
                        float p = fmaf(y, t2.y, t2.x);
                        p = fmaf(y, p, t1.w);
                        p = fmaf(y, p, t1.z);
                        p = fmaf(y, p, t1.y);
                        p = fmaf(y, p, t1.x);
                        p = fmaf(y, p, t0.w);
                        p = fmaf(y, p, t0.z);
                        p = fmaf(y, p, t0.y);
                        p = fmaf(y, p, 1.0f);
                        put(e, tick ? -1 : e - nt,
                            t0.x * (p * ex2_ftz(cc * (cc * -1.44269504088896341f))));
                    }
                } else {
                    // One erfc per bin edge, signed by the side of the mean it lies on: the nt + 1
                    // tick edges, then the nr + 1 row edges, each lane's next edge in the next
                    // lane (G - 1 bins per round).  The mass of a bin from its signed edge terms
                    // a, b (span_mass's three cases) is half their difference, plus 1 when the
                    // mean lies between them.
                    const float bt = off_t + (float)ka, bp = off_p + (float)(ra - (nt + 1));
                    for (int e0 = 0; e0 <= nr + nt; e0 += G - 1) {
                        const int e = e0 + gl;
                        const bool tick = e <= nt;
                        const float u = (((tick ? bt : bp) + (float)e) - (tick ? frac_t : frac_p)) *
                                        (tick ? s_t : s_p);
                        const float a = copysignf(erfcf(fabsf(u)), u);
                        const float b = __shfl_down_sync(gmask, a, 1, G);
                        if (gl == G - 1 || e == nt || e > nr + nt) continue;
                        float w = 0.5f * (a - b);
                        if (__float_as_int(a) < 0 && __float_as_int(b) >= 0) w += 1.0f;
                        put(e, tick ? -1 : e - (nt + 1), tick ? w : w * qw);
                    }
                }
                __syncwarp(gmask);
                if constexpr (MODE == 2) {
                    // one bin per lane: neighbouring ticks cost alike, so the group's lanes
                    // walk their CDFs side by side, and no lane chains four draws
                    const float inv_nt = 1.0f / (float)nt;
                    for (int b = gl; b < nr * nt; b += G) {
                        const int ir = (int)(((float)b + 0.5f) * inv_nt);
                        const int ik = b - ir * nt;
                        const int64_t r = r0 + ir;
                        const float v = row[ir] * quad[ik + koff];
                        if (!(v > 0.0f)) continue;
                        atomicAdd(grid + r * c.n_ticks + (k0 + ik),
                                  binomial_bin(c, pd.qatt, pd.id, k0 + ik, r, v, inv_q, stirl));
                    }
                    __syncwarp(gmask);
                    continue;
                }
                // (row, 4-tick group) items, G apart: the row and group of an item advance by
                // G / nq and G mod nq (no division per item)
                const float inv_nq = rcp_approx((float)nq);
                const int step_r = (int)(((float)G + 0.5f) * inv_nq), step_q = G - step_r * nq;
                float* tile = grid + (int64_t)r0 * c.n_ticks + 4 * q_lo;
                auto items = [&](auto fast) {
                    int ir = (int)(((float)gl + 0.5f) * inv_nq), iq = gl - ir * nq;
#pragma unroll 1
                    while (ir < nr) {
                        const float4 t4 = *reinterpret_cast<const float4*>(quad + L::kQuad * iq);
                        float v[4];
                        if constexpr (MODE == 1) {
                            // normal approximation to Binomial(Q', mean / Q'); zero-mean bins
                            // (outside the window) stay zero
                            const float4 rr = *reinterpret_cast<const float4*>(row + 4 * ir);
                            const uint4 qq = *reinterpret_cast<const uint4*>(quad + 8 * iq + 4);
                            v[0] = rr.x * t4.x; v[1] = rr.x * t4.y; v[2] = rr.x * t4.z; v[3] = rr.x * t4.w;
                            fluctuate4<decltype(fast)::value>(
                                philox_rest(qq, __float_as_uint(rr.y), __float_as_uint(rr.z), c.keys), inv_q, v);
                        } else {
                            const float w = row[ir];
                            v[0] = w * t4.x; v[1] = w * t4.y; v[2] = w * t4.z; v[3] = w * t4.w;
                        }
                        float* dst = tile + (int64_t)ir * c.n_ticks + 4 * iq;
                        if (vec4) {
                            atomicAdd(reinterpret_cast<float4*>(dst), make_float4(v[0], v[1], v[2], v[3]));
                        } else {
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if ((unsigned)(4 * iq + e - koff) < (unsigned)nt) atomicAdd(dst + e, v[e]);
                        }
                        ir += step_r;
                        iq += step_q;
                        if (iq >= nq) { iq -= nq; ++ir; }
                    }
                };
                if (MODE != 1 || fluctuate_fast(inv_q)) items(std::true_type{});
                else if constexpr (MODE == 1) items(std::false_type{});
                __syncwarp(gmask);
            }
        }
    }
}

// The binomial's small-count table in shared memory.
template <int MODE>
__device__ __forceinline__ void load_stirling(const RasterConsts& c, float* s_stirl)
{
    if constexpr (MODE == 2) {
        if (threadIdx.x == 0) {
#pragma unroll
            for (int m = 0; m < 16; ++m) s_stirl[m] = c.stirl[m];    // constant indices: no local copy
        }
        __syncthreads();
    }
}

template <int G, int MODE>
__global__ void __launch_bounds__(kRasterWarps * 32, MODE == 2 ? 8 : 10)
k_rasterize(RasterConsts c, DepoArrays d, float* __restrict__ grid, int* flags, int dpw)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ float s_stirl[MODE == 2 ? 16 : 1];
    after_previous_kernel();
    load_stirling<MODE>(c, s_stirl);
    const int warp = threadIdx.x >> 5;
    rasterize_warp<G, MODE>(c, d, grid, flags, ((int64_t)blockIdx.x * kRasterWarps + warp) * dpw, dpw,
                            smraw + warp * raster_warp_smem(MODE, dpw, G), s_stirl);
}

// Every event of a batch in one launch, each with its plane's own constants.  A warp's share of depos
// is a piece, a block's worth of pieces one item of block_start, in the events' order.  The constants
// are read through the event's index, and a round key that the compiler then holds costs a register:
// formed from the key instead, the kernel keeps 64 registers and 32 warps per SM.  (Warps that popped
// their pieces from a queue held 96, 20 warps per SM: 16 events of 2000 to 20000 depos on 480 x 2000
// and 800 x 6000 planes 180 us with fluctuation, this 94; 12 mixed events 349 / 229.)
// MODE kMixed: events with the normal fluctuation and without.
constexpr int kMixed = 3;
template <int G, int MODE>
__global__ void __launch_bounds__(kRasterWarps * 32, 8)
k_rasterize_events(const __grid_constant__ BatchPlanes q, int dpw)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ float s_stirl[MODE == 2 ? 16 : 1];
    load_stirling<MODE>(q.c[0], s_stirl);
    const int warp = threadIdx.x >> 5;
    const int64_t piece = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const int item = (int)(piece / kRasterWarps);
    int e = 0;
    while (e + 1 < q.n && q.block_start[e + 1] <= item) ++e;
    RasterConsts c = q.c[e];
    c.keys.set(c.keys.k0[0], c.keys.k1[0]);
    const int64_t base = (piece - (int64_t)q.block_start[e] * kRasterWarps) * dpw;
    constexpr int kOne = MODE == kMixed ? 1 : MODE;
    unsigned char* tile = smraw + warp * raster_warp_smem(kOne, dpw, G);
    if constexpr (MODE == kMixed) {
        if (c.fluctuate == 0) {
            rasterize_warp<G, 0>(c, q.d[e], q.grid[e], q.flags[e], base, dpw, tile, s_stirl);
            return;
        }
    }
    rasterize_warp<G, kOne>(c, q.d[e], q.grid[e], q.flags[e], base, dpw, tile, s_stirl);
}

// Sum over the G lanes of a lane group (mask: the group's lanes), in every lane of it.
template <int G>
__device__ __forceinline__ float group_sum(float v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
    return v;
}

// Renormalisation factors of one depo for the adjoint: 1 / T and the telescoped dT/dmu,
// dT/dsigma per axis (rows, then ticks), T the unclipped window's mass between its outer
// edges: dT/dmu = -(phi(B') - phi(A')) / sigma, dT/dsigma = -(B' phi(B') - A' phi(A')) /
// sigma.  The identity (1, 0, 0) when renormalisation is off or sigma == 0.
__device__ __forceinline__ void renorm_factors(const RasterConsts& c, const Decision& r, float* f)
{
    f[0] = 1.0f; f[1] = 0.0f; f[2] = 0.0f;
    f[3] = 1.0f; f[4] = 0.0f; f[5] = 0.0f;
    if (!c.renorm || !r.ok) return;
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
        const float sg = ax ? r.st : r.sp;
        if (!(sg > 0.0f)) continue;
        const float bin = ax ? c.dt_f : c.dp_f;
        const float s = bin / (1.41421356237309505f * sg);
        const float hw = __fmul_rn(__fmul_rn(c.nsig, sg), ax ? c.inv_dt_f : c.inv_dp_f);
        const float frac = ax ? r.frac_t : r.frac_p;
        const float ua = outer_edge_u(frac, hw, s, false), ub = outer_edge_u(frac, hw, s, true);
        const float pa = 0.398942280401432678f * expf(-ua * ua);
        const float pb = 0.398942280401432678f * expf(-ub * ub);
        const float isg = 1.0f / sg;
        f[3 * ax + 0] = 1.0f / span_mass(ua, ub, erfcf(fabsf(ua)), erfcf(fabsf(ub)));
        f[3 * ax + 1] = -(pb - pa) * isg;
        f[3 * ax + 2] = -1.41421356237309505f * (ub * pb - ua * pa) * isg;
    }
}

// What the adjoint's lanes need of one depo (edges as in PatchDepo); after its patch, the terms of
// the three global sums.
struct __align__(16) AdjointDepo {
    int32_t r_lo, nr, k_lo, nt;      // window; nr == 0: the depo adds nothing
    float off_p, frac_p, s_p, isp;   // isp, ist: 1 / sigma, 0 for a point
    float off_t, frac_t, s_t, ist;
    float qatt, att, sp, st;         // Q', Q' / Q, the sigmas
    float a_q, dsl, dst, pad;        // dL/dQ', dL/dsigma_L, dL/dsigma_T
    float rn[8];                     // renorm_factors
};
constexpr int kAdjointQuad = 12;     // floats per quad record: weights, dw/dmu, dw/dsigma
constexpr int kAdjointGroup = kMaxQuads * kAdjointQuad * 4 + kWmax * 16;   // bytes per group

__host__ __device__ constexpr int adjoint_warp_smem(int depos_per_warp)
{
    return depos_per_warp * (int)sizeof(AdjointDepo) + 4 * kAdjointGroup;
}

// Adjoint of drift and rasterization, split as the rasterizer: a warp decides its own dpw depos,
// then each group of 8 lanes takes one at a time: it recomputes the patch weights and their mu /
// sigma derivatives (one erfc and one normal pdf per bin edge, each lane's next edge in the next
// lane), gathers dL/dS over the patch and applies the chain rule through Q' = Q exp(-t_d / tau),
// t_a = t + t_d and sigma = sqrt(2 D t_d).  The global sums are reduced per block in FP64.
// Bound by instructions: a block whose first two warps decided for eight, kept the edge terms in
// shared memory (58 KB per block, three blocks per SM) and divided for every item's row took 70 us
// on 100k depos of the 960 x 6000 plane, this 56 us (2000 depos 12.5 / 8.8 us).  Depos per warp: 16
// above 64k depos, 8 above 16k, else 4.  The order of every sum over a patch is as it was: the per-depo
// results keep their bits.
template <bool RN>
__global__ void __launch_bounds__(kRasterWarps * 32, 8)
k_depo_adjoint(RasterConsts c, DepoArrays d, const float* __restrict__ dgrid, DepoGrads g,
               int* flags, int dpw)
{
    constexpr int G = 8;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gl = lane % G, grp = lane / G;
    const unsigned gmask = ((1u << G) - 1u) << (lane & ~(G - 1));
    unsigned char* wsm = smraw + warp * adjoint_warp_smem(dpw);
    AdjointDepo* dep = reinterpret_cast<AdjointDepo*>(wsm);
    const int64_t base = ((int64_t)blockIdx.x * kRasterWarps + warp) * dpw;
    if (lane < dpw) {
        AdjointDepo p;
        p.nr = 0;
        p.nt = 0;
        p.qatt = p.att = p.a_q = p.dsl = p.dst = p.sp = p.st = 0.0f;
        const int64_t i = base + lane;
        if (i < d.n) {
            const Decision r = decide(c, d, i, flags);
            if (RN) renorm_factors(c, r, p.rn);
            if (r.ok && r.qatt > 0.0f) {
                p.r_lo = r.r_lo;
                p.nr = r.r_hi - r.r_lo + 1;
                p.k_lo = r.k_lo;
                p.nt = r.k_hi - r.k_lo + 1;
                p.off_p = offset_float((int64_t)r.r_lo - r.i0p);
                p.off_t = offset_float((int64_t)r.k_lo - r.i0t);
                edge_axis(r.sp, c.dp_f, p.off_p, r.frac_p, p.frac_p, p.s_p);
                edge_axis(r.st, c.dt_f, p.off_t, r.frac_t, p.frac_t, p.s_t);
                p.isp = (r.sp > 0.0f) ? 1.0f / r.sp : 0.0f;
                p.ist = (r.st > 0.0f) ? 1.0f / r.st : 0.0f;
                p.qatt = r.qatt;
                p.att = r.qatt / d.q[i];
                p.sp = r.sp;
                p.st = r.st;
            }
        }
        dep[lane] = p;
    }
    __syncwarp();
    float* quad = reinterpret_cast<float*>(wsm + dpw * sizeof(AdjointDepo) + grp * kAdjointGroup);
    float* row = quad + kMaxQuads * kAdjointQuad;
    const bool vec4 = ((c.n_ticks & 3) == 0) && ((reinterpret_cast<uintptr_t>(dgrid) & 15) == 0);

#pragma unroll 1
    for (int i = grp; i < dpw; i += 32 / G) {
        const int64_t gi = base + i;
        if (gi >= d.n) break;
        AdjointDepo& pd = dep[i];
        const int nr_all = pd.nr, nt_all = pd.nt;
        const float off_p = pd.off_p, frac_p = pd.frac_p, s_p = pd.s_p, isp = pd.isp;
        const float off_t = pd.off_t, frac_t = pd.frac_t, s_t = pd.s_t, ist = pd.ist;
        float a_q = 0.f, a_pm = 0.f, a_ps = 0.f, a_tm = 0.f, a_ts = 0.f;
#pragma unroll 1
        for (int32_t ra = 0; ra < nr_all; ra += kWmax) {
            const int nr = min(kWmax, nr_all - ra), r0 = pd.r_lo + ra;
#pragma unroll 1
            for (int32_t ka = 0; ka < nt_all; ka += kWmax) {
                const int nt = min(kWmax, nt_all - ka), k0 = pd.k_lo + ka;
                const int q_lo = k0 >> 2, nq = ((k0 + nt - 1) >> 2) - q_lo + 1;
                const int koff = k0 & 3;               // slot of tick k0
                for (int q = gl; q < 3 * nq; q += G)
                    *reinterpret_cast<float4*>(quad + 4 * q) = make_float4(0.f, 0.f, 0.f, 0.f);
                __syncwarp(gmask);
                // w = Phi(b') - Phi(a'); dw/dmu = -(phi(b') - phi(a')) / sigma;
                // dw/dsigma = -(b' phi(b') - a' phi(a')) / sigma, with b' = sqrt(2) ub.
                // Renormalised weights w / T and their derivatives by the quotient rule,
                // (dw - (w / T) dT) / T.
                const float bt = off_t + (float)ka, bp = off_p + (float)(ra - (nt + 1));
                for (int e0 = 0; e0 <= nr + nt; e0 += G - 1) {
                    const int e = e0 + gl;
                    const bool tick = e <= nt;
                    const float u = (((tick ? bt : bp) + (float)e) - (tick ? frac_t : frac_p)) *
                                    (tick ? s_t : s_p);
                    const float ph = 0.398942280401432678f * expf(-u * u), up = u * ph;
                    const float a = copysignf(erfcf(fabsf(u)), u);
                    const float b = __shfl_down_sync(gmask, a, 1, G);
                    const float phb = __shfl_down_sync(gmask, ph, 1, G);
                    const float upb = __shfl_down_sync(gmask, up, 1, G);
                    if (gl == G - 1 || e == nt || e > nr + nt) continue;
                    float w = 0.5f * (a - b);
                    if (__float_as_int(a) < 0 && __float_as_int(b) >= 0) w += 1.0f;
                    const float is = tick ? ist : isp;
                    const float m = -(phb - ph), sg = -1.41421356237309505f * (upb - up);
                    float wn = w, wm = m * is, ws = sg * is;
                    if (RN) {
                        const float* rn = pd.rn + (tick ? 3 : 0);
                        wn = w * rn[0];
                        wm = (m * is - wn * rn[1]) * rn[0];
                        ws = (sg * is - wn * rn[2]) * rn[0];
                    }
                    if (tick) {
                        const int p = e + koff;
                        float* q = quad + (p >> 2) * kAdjointQuad + (p & 3);
                        q[0] = wn;
                        q[4] = wm;
                        q[8] = ws;
                    } else {
                        *reinterpret_cast<float4*>(row + 4 * (e - (nt + 1))) = make_float4(wn, wm, ws, 0.f);
                    }
                }
                __syncwarp(gmask);
                if (vec4) {
                    // (row, 4-tick group) items, one 16-byte load of dL/dS each
                    const float inv_nq = rcp_approx((float)nq);
                    const int step_r = (int)(((float)G + 0.5f) * inv_nq), step_q = G - step_r * nq;
                    int ir = (int)(((float)gl + 0.5f) * inv_nq), iq = gl - ir * nq;
                    const float* tile = dgrid + (int64_t)r0 * c.n_ticks + 4 * q_lo;
#pragma unroll 1
                    while (ir < nr) {
                        const float4 sv = __ldg(reinterpret_cast<const float4*>(
                            tile + (int64_t)ir * c.n_ticks + 4 * iq));
                        const float4* q4 = reinterpret_cast<const float4*>(quad + kAdjointQuad * iq);
                        const float4 w4 = q4[0], m4 = q4[1], g4 = q4[2];
                        const float4 rw = *reinterpret_cast<const float4*>(row + 4 * ir);
                        const float A = sv.x * w4.x + sv.y * w4.y + sv.z * w4.z + sv.w * w4.w;
                        const float B = sv.x * m4.x + sv.y * m4.y + sv.z * m4.z + sv.w * m4.w;
                        const float C = sv.x * g4.x + sv.y * g4.y + sv.z * g4.z + sv.w * g4.w;
                        a_q += rw.x * A;
                        a_pm += rw.y * A;
                        a_ps += rw.z * A;
                        a_tm += rw.x * B;
                        a_ts += rw.x * C;
                        ir += step_r;
                        iq += step_q;
                        if (iq >= nq) { iq -= nq; ++ir; }
                    }
                } else {
                    const float inv_nt = 1.0f / (float)nt;
                    for (int b = gl; b < nr * nt; b += G) {
                        const int ir = (int)(((float)b + 0.5f) * inv_nt);
                        const int ik = b - ir * nt, p = ik + koff;
                        const float sv = __ldg(dgrid + (int64_t)(r0 + ir) * c.n_ticks + (k0 + ik));
                        const float* q = quad + (p >> 2) * kAdjointQuad + (p & 3);
                        const float pw = row[4 * ir], tw = q[0];
                        a_q += sv * pw * tw;
                        a_pm += sv * row[4 * ir + 1] * tw;
                        a_ps += sv * row[4 * ir + 2] * tw;
                        a_tm += sv * pw * q[4];
                        a_ts += sv * pw * q[8];
                    }
                }
                __syncwarp(gmask);
            }
        }
        a_q = group_sum<G>(a_q, gmask);
        a_pm = group_sum<G>(a_pm, gmask);
        a_ps = group_sum<G>(a_ps, gmask);
        a_tm = group_sum<G>(a_tm, gmask);
        a_ts = group_sum<G>(a_ts, gmask);
        if (gl == 0) {
            const float qa = pd.qatt;
            const float dst = qa * a_ps, dsl = qa * a_ts * c.inv_v;
            if (g.dq) g.dq[gi] = a_q * pd.att;
            if (g.dp) g.dp[gi] = qa * a_pm;
            if (g.dt) g.dt[gi] = qa * a_tm;
            if (g.dsl) g.dsl[gi] = dsl;
            if (g.dst) g.dst[gi] = dst;
            pd.a_q = a_q;
            pd.dsl = dsl;
            pd.dst = dst;
        }
    }
    if (!g.dglobal) return;
    __syncthreads();
    // The global sums, by one warp for the whole block (FP64 is scarce on this part: one
    // warp instruction per 32 depos).  sigma = sqrt(2 D t_d) gives dsigma/dD = sigma / (2 D)
    // (sigma_L = v sigma_t in mm); dQ'/dtau = Q' t_d / tau^2.  Products of two FP32 values
    // are exact in FP64.
    if (warp == 0) {
        double a0 = 0.0, a1 = 0.0, a2 = 0.0;
        for (int i = lane; i < kRasterWarps * dpw; i += 32) {
            const int64_t gi = (int64_t)blockIdx.x * kRasterWarps * dpw + i;
            const AdjointDepo& p = reinterpret_cast<const AdjointDepo*>(
                smraw + (i / dpw) * adjoint_warp_smem(dpw))[i % dpw];
            if (!(p.qatt > 0.0f)) continue;
            a0 += (double)p.dsl * (double)p.st;
            a1 += (double)p.dst * (double)p.sp;
            a2 += (double)p.a_q * (double)p.qatt * d.td[gi];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, o);
            a1 += __shfl_xor_sync(0xffffffffu, a1, o);
            a2 += __shfl_xor_sync(0xffffffffu, a2, o);
        }
        if (lane == 0) {
            if (c.DL > 0.0) atomicAdd(g.dglobal + 0, a0 * c.v / (2.0 * c.DL));
            if (c.DT > 0.0) atomicAdd(g.dglobal + 1, a1 / (2.0 * c.DT));
            atomicAdd(g.dglobal + 2, a2 / (c.tau * c.tau));
        }
    }
}

__global__ void k_windows(RasterConsts c, DepoArrays d, int32_t* __restrict__ out, int* flags)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= d.n) return;
    Decision r = decide(c, d, i, flags);
    int4 v = r.ok ? make_int4(r.r_lo, r.r_hi, r.k_lo, r.k_hi) : make_int4(-1, -1, -1, -1);
    reinterpret_cast<int4*>(out)[i] = v;
}

}  // namespace

// Tiles that can be set by hand or tried by the autotuner: depos per 8 warps (per 256 threads),
// lanes per depo.
bool raster_tile_supported(int depos_per_block, int lanes_per_depo)
{
    if (lanes_per_depo != 8 && lanes_per_depo != 16 && lanes_per_depo != 32) return false;
    // 4 depos per warp at least, 8 with more lanes each; and raster_tile's own for the exact binomial
    const int lo = lanes_per_depo == 8 ? 32 : 64;
    if ((depos_per_block == 8 && lanes_per_depo == 32) || (depos_per_block == 16 && lanes_per_depo == 16)) return true;
    return depos_per_block >= lo && depos_per_block <= 256 && (depos_per_block & (depos_per_block - 1)) == 0;
}

RasterTile raster_tile(const RasterConsts& c, int64_t n_depos)
{
    // (so many depos that a launch of fewer per warp would have too many blocks)
    if (n_depos > (1ll << 30)) return {16, 8};
    if (c.depos_per_block > 0) return {c.depos_per_block / 8, c.lanes_per_depo};
    // One depo per warp for the exact binomial's long serial walks (2000 depos: 76 us against 210 with
    // 4 x 8 lanes), two above 64k depos.  Along tracks, 1 x 32 / 2 x 16 / 4 x 8: 100k 1301 / 1231 / 1266
    // us, 300k 3699 / 3408 / 3371; strewn evenly 1272 / 1524 / 1826 and 3734 / 4410 / 5148, so that more
    // than two never pay.
    if (c.fluctuate == 2) return n_depos > 65536 ? RasterTile{2, 16} : RasterTile{1, 32};
    // Else 8 lanes per depo, and more depos per warp (fewer, better filled decisions) as soon as there
    // are warps enough for every SM.  With fluctuation, 4 / 8 / 16 depos per warp: 2000 depos 7.6 / 10.8 /
    // 17.2 us, 10k along tracks 7.9 / 8.3 / 10.8, 12.5k 9.2 / 8.3 / 11.5, 30k 24.3 / 24.4 / 26.1, 100k 58.5 /
    // 56.0 / 58.0, 300k 148 / 132 / 128, 1M 466 / 404 / 378; 32 is slower throughout.  On the mean path, and
    // where depos reach few bins, the decision is more of the work (5000 depos along tracks 5.0 / 5.2 us, 8000
    // 5.9 / 5.6, 12.5k 7.5 / 6.2, before the warps decided for themselves 6.5; 30k points 10.3 / 7.9, 7.4).  Rows that are not 16-byte
    // aligned, whose patches are added bin by bin, behave alike along tracks (5998 ticks: 12.5k 14.3 / 12.6 /
    // 15.5, 250k 195 / 172 / 159), and are nearly indifferent for evenly strewn depos (200k 159 / 161 / 165).
    return {n_depos > 196608 ? 16 : n_depos > (c.fluctuate ? 11000 : 7000) ? 8 : 4, 8};
}

int rasterize_blocks(int64_t n_depos, int depos_per_warp)
{
    const int kd = kRasterWarps * depos_per_warp;
    return (int)((n_depos + kd - 1) / kd);
}

// One launch of the instance for `lanes` and the fluctuation mode.
#define WCSIM_RASTER_DISPATCH(KERNEL, lanes, mode, ...)                                        \
    do {                                                                                       \
        if (lanes == 8) {                                                                      \
            if (mode == 2) { auto k = KERNEL<8, 2>; __VA_ARGS__; }                             \
            else if (mode == 1) { auto k = KERNEL<8, 1>; __VA_ARGS__; }                        \
            else { auto k = KERNEL<8, 0>; __VA_ARGS__; }                                       \
        } else if (lanes == 16) {                                                              \
            if (mode == 2) { auto k = KERNEL<16, 2>; __VA_ARGS__; }                            \
            else if (mode == 1) { auto k = KERNEL<16, 1>; __VA_ARGS__; }                       \
            else { auto k = KERNEL<16, 0>; __VA_ARGS__; }                                      \
        } else {                                                                               \
            if (mode == 2) { auto k = KERNEL<32, 2>; __VA_ARGS__; }                            \
            else if (mode == 1) { auto k = KERNEL<32, 1>; __VA_ARGS__; }                       \
            else { auto k = KERNEL<32, 0>; __VA_ARGS__; }                                      \
        }                                                                                      \
    } while (0)

cudaError_t launch_rasterize(const RasterConsts& c, const DepoArrays& d, float* grid,
                             int* flags, cudaStream_t s)
{
    if (d.n <= 0) return cudaSuccess;
    const RasterTile t = raster_tile(c, d.n);
    const unsigned blocks = (unsigned)rasterize_blocks(d.n, t.depos_per_warp);
    const int smem = kRasterWarps * raster_warp_smem(c.fluctuate, t.depos_per_warp, t.lanes_per_depo);
    WCSIM_RASTER_DISPATCH(k_rasterize, t.lanes_per_depo, c.fluctuate,
        return launch_chained(c.chained != 0, k, blocks, kRasterWarps * 32, smem, s, c, d, grid,
                              flags, t.depos_per_warp));
    return cudaSuccess;
}

cudaError_t launch_rasterize_events(const BatchPlanes& q, const RasterTile& t, cudaStream_t s)
{
    const int blocks = q.n > 0 ? q.block_start[q.n] : 0;
    if (blocks <= 0) return cudaSuccess;
    const int mode = q.c[0].fluctuate;
    for (int e = 1; e < q.n; ++e) {
        if (q.c[e].fluctuate == mode) continue;
        if (mode == 2 || q.c[e].fluctuate == 2) return cudaErrorInvalidValue;
        auto k = t.lanes_per_depo == 8 ? k_rasterize_events<8, kMixed>
                 : t.lanes_per_depo == 16 ? k_rasterize_events<16, kMixed> : k_rasterize_events<32, kMixed>;
        k<<<(unsigned)blocks, kRasterWarps * 32,
            kRasterWarps * raster_warp_smem(1, t.depos_per_warp, t.lanes_per_depo), s>>>(q, t.depos_per_warp);
        return cudaGetLastError();
    }
    // one warp per block for the exact binomial, whose walks differ much in length (16 events of 2000
    // to 20000 depos: 2043 us, with four 2096)
    const int warps = mode == 2 ? 1 : kRasterWarps;
    const int smem = warps * raster_warp_smem(mode, t.depos_per_warp, t.lanes_per_depo);
    WCSIM_RASTER_DISPATCH(k_rasterize_events, t.lanes_per_depo, mode,
        k<<<(unsigned)blocks * (kRasterWarps / warps), warps * 32, smem, s>>>(q, t.depos_per_warp));
    return cudaGetLastError();
}

cudaError_t launch_depo_adjoint(const RasterConsts& c, const DepoArrays& d, const float* dgrid,
                                const DepoGrads& g, int* flags, cudaStream_t s)
{
    if (d.n <= 0) return cudaSuccess;
    const int dpw = d.n > 65536 ? 16 : d.n > 16384 ? 8 : 4;
    const unsigned blocks = (unsigned)rasterize_blocks(d.n, dpw);
    const int smem = kRasterWarps * adjoint_warp_smem(dpw);
    if (c.renorm) k_depo_adjoint<true><<<blocks, kRasterWarps * 32, smem, s>>>(c, d, dgrid, g, flags, dpw);
    else k_depo_adjoint<false><<<blocks, kRasterWarps * 32, smem, s>>>(c, d, dgrid, g, flags, dpw);
    return cudaGetLastError();
}

cudaError_t launch_windows(const RasterConsts& c, const DepoArrays& d, int32_t* out,
                           int* flags, cudaStream_t s)
{
    if (d.n <= 0) return cudaSuccess;
    const int64_t blocks = (d.n + 255) / 256;
    k_windows<<<(unsigned)blocks, 256, 0, s>>>(c, d, out, flags);
    return cudaGetLastError();
}

}  // namespace wcsim
