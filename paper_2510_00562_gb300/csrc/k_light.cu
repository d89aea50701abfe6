// K2 (the light pass of one P-PDS iteration), the exact radix search for the
// l1 thresholds, state conversion kernels and the standalone l1 projection.
//
// K2 finishes Algorithm 1 once the l1 thresholds tau_s, tau_t are known:
//   s+ = P_{B1,alpha}(s~) = soft(s~, tau_s),  t+ = soft(t~, tau_t),
//   s' = 2 s+ - s,  t' = 2 t+ - t,
//   y3+ = y3 + g3 D_v t'                                   (needs row i+1)
//   y4' = y4 + g4 (u' + s' + t'),  q = y4' - g4 v,
// and reduces ||q||^2: the l2-ball step of Algorithm 1 (Eq. 23 through
// Moreau's identity, Eq. 3) is y4+ = (1 - c) q with c = min(1, eps g4 / ||q||),
// which the next iteration applies when it reads q.  It also reduces the two
// norms of the stopping rule (Eq. 28).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "gsstv_internal.cuh"
#include "gsstv_l1.cuh"

namespace gsstv {
namespace {

constexpr int NT = 256;
constexpr int K2_ROWS = 8;   // rows per thread strip in K2

template <typename T> struct Vec4;
template <> struct Vec4<float> {
    static __device__ __forceinline__ float4 ld(const float* p) { return *reinterpret_cast<const float4*>(p); }
    static __device__ __forceinline__ void st(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
};
template <> struct Vec4<__nv_bfloat16> {
    static __device__ __forceinline__ float4 ld(const __nv_bfloat16* p) {
        uint2 r = *reinterpret_cast<const uint2*>(p);
        float2 a = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&r.x));
        float2 b = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&r.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float4 v) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        uint2 r;
        r.x = *reinterpret_cast<unsigned*>(&a);
        r.y = *reinterpret_cast<unsigned*>(&b);
        *reinterpret_cast<uint2*>(p) = r;
    }
};
template <> struct Vec4<__half> {
    static __device__ __forceinline__ float4 ld(const __half* p) {
        uint2 r = *reinterpret_cast<const uint2*>(p);
        float2 a = __half22float2(*reinterpret_cast<__half2*>(&r.x));
        float2 b = __half22float2(*reinterpret_cast<__half2*>(&r.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    static __device__ __forceinline__ void st(__half* p, float4 v) {
        __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
        uint2 r;
        r.x = *reinterpret_cast<unsigned*>(&a);
        r.y = *reinterpret_cast<unsigned*>(&b);
        *reinterpret_cast<uint2*>(p) = r;
    }
};
// four stores of a quad, stochastically rounded for 16-bit storage
template <typename T>
__device__ __forceinline__ void st4S(T* p, const float4& v, SRStream& sr) {
    if constexpr (std::is_same<T, float>::value) {
        *reinterpret_cast<float4*>(p) = v;
    } else {
        stS(p, v.x, sr); stS(p + 1, v.y, sr); stS(p + 2, v.z, sr); stS(p + 3, v.w, sr);
    }
}

__device__ __forceinline__ float comp(const float4& v, int k) {
    return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w;
}
__device__ __forceinline__ void set_comp(float4& v, int k, float x) {
    if (k == 0) v.x = x; else if (k == 1) v.y = x; else if (k == 2) v.z = x; else v.w = x;
}

// ---------------------------------------------------------------------------
// K2
// ---------------------------------------------------------------------------
template <typename T>
struct K2Args {
    Geom g;
    const T *u, *u_n, *s, *t, *y3, *q;
    const float* v;
    T *s_n, *t_n, *y3_n, *q_n;
    IterParams p;
    Scal* sc;
    double* part;       // 3 doubles per CTA
    SlabPart sp;        // the bands updated, and this launch's CTAs among the stage's
    int windows;        // 1: the first CTA places the next windows
};

// A thread's part of the three norms |q|^2, |u+ - u|^2, |u|^2.
struct K2Norms {
    Kahan q, du, u;
};

// The norms of the strips, in the order of the block.
struct K2NormsStrip {
    KahanSum q, du, u;
};

// The rows of one strip per thread and item, top to bottom, t' of the row below
// carried over: 16-bit storage, whose rounding streams follow the strips, and
// float32 with its sums in their fixed order (a thread's Kahan sums over a strip
// of four columns: the last place of the l2-ball scale).
template <typename T>
__device__ __forceinline__ void k2_strips(const K2Args<T>& a, const int bid, const int nblk, K2NormsStrip& N) {
    const Geom g = a.g;
    const IterParams& P = a.p;
    const float cs = (float)(1.0 - a.sc->c[P.parity]);
    const float tau_s = (float)a.sc->ctl[0].tau;
    const float tau_t = (float)a.sc->ctl[1].tau;
    const unsigned it32 = (unsigned)a.sc->iter;       // seeds the 16-bit rounding streams
    const int quads = g.p2 / 4;
    const int strips = (g.n1 + K2_ROWS - 1) / K2_ROWS;
    const long long items = (long long)(a.sp.o1 - a.sp.o0) * strips * quads;
    for (long long it = bid * (long long)NT + threadIdx.x; it < items; it += (long long)nblk * NT) {
        const int qd = (int)(it % quads);
        const long long rest = it / quads;
        const int strip = (int)(rest % strips);
        const int b = a.sp.o0 + (int)(rest / strips);
        const int j = qd * 4;
        const int i_s = strip * K2_ROWS;
        const int i_own = min(i_s + K2_ROWS, g.n1);            // own rows [i_s, i_own)
        const int i_last = min(i_s + K2_ROWS, g.n1 - 1);       // plus one halo row if any
        float4 y3m = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i_s >= 1) y3m = Vec4<T>::ld(a.y3 + g.at(b, i_s - 1, j));
        float4 tprev = y3m, y3prev = y3m;
        for (int i = i_s; i <= i_last; ++i) {
            const long long o = g.at(b, i, j);
            const float4 s4 = Vec4<T>::ld(a.s + o), t4 = Vec4<T>::ld(a.t + o);
            const float4 y34 = Vec4<T>::ld(a.y3 + o), q4 = Vec4<T>::ld(a.q + o);
            const bool own = i < i_own;
            float4 u0 = make_float4(0, 0, 0, 0), u1 = u0, v4 = u0;
            if (own) {
                u0 = Vec4<T>::ld(a.u + o);
                u1 = Vec4<T>::ld(a.u_n + o);
                v4 = *reinterpret_cast<const float4*>(a.v + o);
            }
            float4 sp4, tp4, qn4, tb4, y3n4;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float y4 = __fmul_rn(cs, comp(q4, k));
                float xs, xt;
                s_t_tilde(comp(s4, k), comp(t4, k), comp(y34, k), comp(y3m, k), comp(q4, k), cs, i,
                          g.n1, P.gamma_s, P.gamma_t, xs, xt);
                const float sp = soft(xs, tau_s), tp = soft(xt, tau_t);
                const float sb = 2.f * sp - comp(s4, k), tb = 2.f * tp - comp(t4, k);
                set_comp(sp4, k, sp);
                set_comp(tp4, k, tp);
                set_comp(tb4, k, tb);
                // y3 of the row above, now that t' of this row is known
                set_comp(y3n4, k, comp(y3prev, k) + P.gamma_y3 * (tb - comp(tprev, k)));
                if (own) {
                    const float uo = comp(u0, k), un = comp(u1, k);
                    const float ub = 2.f * un - uo;
                    const float y4p = y4 + P.gamma_y4 * (ub + sb + tb);
                    const float qn = y4p - P.gamma_y4 * comp(v4, k);
                    set_comp(qn4, k, qn);
                    if (j + k < g.n2) {
                        N.q.add(qn * qn);
                        const float du = un - uo;
                        N.du.add(du * du);
                        N.u.add(uo * uo);
                    }
                }
            }
            SRStream sr((unsigned)o, it32, 5u);
            if (i > i_s) st4S(a.y3_n + o - g.p2, y3n4, sr);
            if (own) {
                st4S(a.s_n + o, sp4, sr);
                st4S(a.t_n + o, tp4, sr);
                st4S(a.q_n + o, qn4, sr);
            }
            y3m = y34;
            y3prev = y34;
            tprev = tb4;
        }
        // the last row has D_v t' = 0: y3 is unchanged there
        if (i_own == g.n1) {
            SRStream sr((unsigned)g.at(b, g.n1 - 1, j), it32, 6u);
            st4S(a.y3_n + g.at(b, g.n1 - 1, j), y3prev, sr);
        }
    }
}

// float32: one row of four columns per thread and item, every load of the item
// issued at once (t' of the row below is computed again from its t, y3, q,
// which the neighbouring rows' threads read too: cache hits).  A persistent
// grid walks the cube in memory order, so that no wave of CTAs is left half
// empty.  (The strips above, one thread marching down 8 rows, were bound by
// the latency of 9 dependent row loads on small cubes, 20 us whatever the
// size up to 128 x 128 x 64, and left their third wave a quarter full at
// 256 x 256 x 128, 80 us.)
// big: the block's shared sums that take a thread's partials before they could
// overflow float.
__device__ __forceinline__ void k2_rows(const K2Args<float>& a, const int bid, const int nblk, K2Norms& N, double* big) {
    const Geom g = a.g;
    const IterParams& P = a.p;
    const unsigned quads = (unsigned)g.p2 / 4u, n1 = (unsigned)g.n1;
    const unsigned total = (unsigned)(a.sp.o1 - a.sp.o0) * n1 * quads;     // < 2^30 for any cube that fits
    const unsigned row0 = (unsigned)a.sp.o0 * n1;
    const float cs = (float)(1.0 - a.sc->c[P.parity]);
    const float tau_s = (float)a.sc->ctl[0].tau;
    const float tau_t = (float)a.sc->ctl[1].tau;
    for (unsigned e = (unsigned)bid * NT + threadIdx.x; e < total; e += (unsigned)nblk * NT) {
        const unsigned r = e / quads;
        const int j = (int)(e - r * quads) * 4;
        const unsigned row = row0 + r;                                      // b * n1 + i
        const int i = (int)(row % n1);
        const long long o = (long long)row * g.p2 + j;
        const bool dn = i < g.n1 - 1;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 s4 = Vec4<float>::ld(a.s + o), t4 = Vec4<float>::ld(a.t + o);
        const float4 y34 = Vec4<float>::ld(a.y3 + o), q4 = Vec4<float>::ld(a.q + o);
        const float4 u0 = Vec4<float>::ld(a.u + o), u1 = Vec4<float>::ld(a.u_n + o);
        const float4 v4 = Vec4<float>::ld(a.v + o);
        const float4 yu4 = i >= 1 ? Vec4<float>::ld(a.y3 + o - g.p2) : zero;
        const float4 td4 = dn ? Vec4<float>::ld(a.t + o + g.p2) : zero;
        const float4 yd4 = dn ? Vec4<float>::ld(a.y3 + o + g.p2) : zero;
        const float4 qd4 = dn ? Vec4<float>::ld(a.q + o + g.p2) : zero;
        float4 sp4, tp4, qn4, y3n4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float y4 = __fmul_rn(cs, comp(q4, k));
            float xs, xt, xsd, xtd;
            s_t_tilde(comp(s4, k), comp(t4, k), comp(y34, k), comp(yu4, k), comp(q4, k), cs, i, g.n1, P.gamma_s,
                      P.gamma_t, xs, xt);
            const float sp = soft(xs, tau_s), tp = soft(xt, tau_t);
            const float sb = 2.f * sp - comp(s4, k), tb = 2.f * tp - comp(t4, k);
            set_comp(sp4, k, sp);
            set_comp(tp4, k, tp);
            // t' of the row below (the last row has D_v t' = 0: y3 is unchanged there)
            s_t_tilde(0.f, comp(td4, k), comp(yd4, k), comp(y34, k), comp(qd4, k), cs, i + 1, g.n1, P.gamma_s,
                      P.gamma_t, xsd, xtd);
            const float tbd = 2.f * soft(xtd, tau_t) - comp(td4, k);
            set_comp(y3n4, k, dn ? comp(y34, k) + P.gamma_y3 * (tbd - tb) : comp(y34, k));
            const float uo = comp(u0, k), un = comp(u1, k);
            const float ub = 2.f * un - uo;
            const float y4p = y4 + P.gamma_y4 * (ub + sb + tb);
            const float qn = y4p - P.gamma_y4 * comp(v4, k);
            set_comp(qn4, k, qn);
            if (j + k < g.n2) {
                N.q.add(qn * qn);
                const float du = un - uo;
                N.du.add(du * du);
                N.u.add(uo * uo);
            }
        }
        if (fmaxf(fmaxf(N.q.s, N.du.s), N.u.s) > 1e36f) {
            atomicAdd(big, N.q.value());
            atomicAdd(big + 1, N.du.value());
            atomicAdd(big + 2, N.u.value());
            N = K2Norms();
        }
        Vec4<float>::st(a.y3_n + o, y3n4);
        Vec4<float>::st(a.s_n + o, sp4);
        Vec4<float>::st(a.t_n + o, tp4);
        Vec4<float>::st(a.q_n + o, qn4);
    }
}

// The next windows of the threshold search, placed beside K2 by a CTA of its own
// (one warp per vector): K1 needs them, K2 does not, and in the search launch
// they stood 5 us in K2's way (code that runs once, in FP64).
__device__ __forceinline__ void k2_windows(Scal* sc) {
    if ((threadIdx.x & 31) || threadIdx.x >= 64) return;
    L1Ctl& c = sc->ctl[threadIdx.x >> 5];
    if (!c.pend) return;
    c.pend = 0;
    l1_place_window(c, c.tau, c.rec_m, c.rec_w, c.rec_hit != 0, c.rec_hist != 0);
}

// The CTA `bid` of `nblk` that share one cube's K2 (a launch of its own, or
// the cube's share of a batch launch).  CTA -1, where the launch has one, places
// the next windows.
template <typename T, bool STRIPS = !std::is_same<T, float>::value>
__device__ __forceinline__ void k2_body(const K2Args<T>& a, const int bid, const int nblk) {
    constexpr int NW = NT / 32;
    if (bid < 0) {
        k2_windows(a.sc);
        return;
    }
    __shared__ double red_d[64];
    __shared__ int is_last;
    const IterParams& P = a.p;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cta = a.sp.cta_base + bid;
    const int ncta = a.sp.cta_total > 0 ? a.sp.cta_total : nblk;
    if constexpr (!STRIPS) {
        __shared__ double big[3];
        if (threadIdx.x < 3) big[threadIdx.x] = 0.0;
        __syncthreads();
        K2Norms N;
        k2_rows(a, bid, nblk, N, big);
        // the CTA's norms: float pairs through each warp (no lane's sum is
        // above 1e36), the warps' in FP64 by three lanes
        const Kahan* k3[3] = {&N.q, &N.du, &N.u};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float h, l;
            warp_sum_pair(*k3[k], h, l);
            if (lane == 0) red_d[k * NW + wid] = (double)h + (double)l;
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            double r = big[threadIdx.x];
            for (int k = 0; k < NW; ++k) r += red_d[threadIdx.x * NW + k];
            a.part[3 * cta + threadIdx.x] = r;
            __threadfence();
        }
    } else {
        K2NormsStrip N;
        k2_strips(a, bid, nblk, N);
        const double q2 = block_sum(N.q.value(), red_d);
        const double du2 = block_sum(N.du.value(), red_d);
        const double u2 = block_sum(N.u.value(), red_d);
        if (threadIdx.x == 0) {
            a.part[3 * cta] = q2;
            a.part[3 * cta + 1] = du2;
            a.part[3 * cta + 2] = u2;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = (atomicAdd(&a.sc->k2_ticket, 1u) == (unsigned)(ncta - 1));
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    double s0 = 0, s1 = 0, s2 = 0;
    if constexpr (!STRIPS) {
        // one warp per norm sums the CTAs' partials
        if (wid < 3) {
            double r = 0.0;
#pragma unroll 4
            for (int k = lane; k < ncta; k += 32) r += __ldcg(a.part + 3 * k + wid);
            r = warp_sum(r);
            if (lane == 0) red_d[wid] = r;
        }
        __syncthreads();
        s0 = red_d[0];
        s1 = red_d[1];
        s2 = red_d[2];
    } else {
        for (int k = threadIdx.x; k < ncta; k += NT) {
            s0 += __ldcg(a.part + 3 * k);
            s1 += __ldcg(a.part + 3 * k + 1);
            s2 += __ldcg(a.part + 3 * k + 2);
        }
        s0 = block_sum(s0, red_d);
        s1 = block_sum(s1, red_d);
        s2 = block_sum(s2, red_d);
    }
    if (threadIdx.x == 0) {
        Scal* sc = a.sc;
        double c = 1.0;
        if (!isfinite(s0) || !isfinite(s1) || !isfinite(s2)) {
            sc->error |= 1;
        } else if (s0 > 0.0) {
            c = fmin(1.0, P.eps * (double)P.gamma_y4 / sqrt(s0));
        }
        sc->c[P.parity ^ 1] = c;
        sc->q2 = s0;
        sc->du2 = s1;
        sc->u2 = s2;
        sc->iter++;
        sc->k2_ticket = 0;
        sc->search = SearchSync();
        // the stopping rule of a batch cube (Eq. 28, or the pass cap): on the
        // device, so that a batch runs as one graph without host polling
        if (P.max_iter > 0) {
            const bool at_check = P.tol > 0.0 && P.check_every > 0 && sc->iter % P.check_every == 0;
            const bool conv = at_check && s2 > 0.0 && sqrt(s1 / s2) < P.tol;
            if (conv || sc->iter >= P.max_iter) {
                sc->done = 1;
                sc->stop_parity = P.parity ^ 1;
                if (P.live) atomicSub(P.live, 1);
            }
        }
    }
}

template <typename T, bool STRIPS>
__global__ void __launch_bounds__(NT, 3) k2_light(const K2Args<T> a) {
    k2_body<T, STRIPS>(a, (int)blockIdx.x - a.windows, (int)gridDim.x - a.windows);
}

// ---------------------------------------------------------------------------
// value sources of the radix search: the cube's s~, t~ or a flat vector
// ---------------------------------------------------------------------------
template <typename T>
struct CubeSrc {
    using Sum = KahanSum;       // of a retry pass above its window (reproduced, as K1's)
    Geom g;
    const T *s, *t, *y3, *q;
    const Scal* sc;
    int parity;
    float gs, gt;
    int o0, nb;         // the stored bands [o0, o0 + nb) this launch visits
    // Calls f(valid, |s~|, |t~|) for every voxel this thread owns, four
    // columns at a time in row order; every lane of a warp makes the same
    // number of calls (warp-collective work inside f is allowed).  want_s /
    // want_t: whether the pass needs |s~| / |t~| (uniform over the launch); the
    // inputs of a vector not wanted are not read, and its value passed to f is
    // meaningless.
    // The thread takes items first + its index, then every stride (both in
    // threads, the stride a multiple of 32; threads at or past it take none).
    template <typename F>
    __device__ void visit(const unsigned first, const unsigned stride, F&& f, const bool want_s,
                          const bool want_t) const {
        const float cs = (float)(1.0 - sc->c[parity]);
        const unsigned quads = (unsigned)g.p2 / 4u;
        const unsigned n1 = (unsigned)g.n1;
        const unsigned total = (unsigned)nb * n1 * quads;       // < 2^31 for any cube that fits
        const unsigned row0 = (unsigned)o0 * n1;
        const bool mine = first + threadIdx.x < stride;
        for (unsigned base = first; base < total; base += stride) {
            const unsigned item = base + threadIdx.x;
            const bool live = mine && item < total;
            const unsigned row = row0 + (live ? item / quads : 0u);   // b * n1 + i
            const int j = (int)(item - (row - row0) * quads) * 4;
            const int i = (int)(row % n1);
            float4 s4 = make_float4(0, 0, 0, 0), t4 = s4, y34 = s4, yu4 = s4, q4 = s4;
            if (live) {
                const long long o = (long long)row * g.p2 + j;
                if (want_s) s4 = Vec4<T>::ld(s + o);
                if (want_t) {
                    t4 = Vec4<T>::ld(t + o);
                    y34 = Vec4<T>::ld(y3 + o);
                    if (i >= 1) yu4 = Vec4<T>::ld(y3 + o - g.p2);
                }
                q4 = Vec4<T>::ld(q + o);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float xs = 0.f, xt = 0.f;
                const bool valid = live && j + k < g.n2;
                if (valid)
                    s_t_tilde(comp(s4, k), comp(t4, k), comp(y34, k), comp(yu4, k), comp(q4, k), cs, i, g.n1,
                              gs, gt, xs, xt);
                f(valid, fabsf(xs), fabsf(xt));
            }
        }
    }
};

struct FlatSrc {
    using Sum = Kahan;          // tau is a result in FP64
    const float* x;
    long long n;
    template <typename F>
    __device__ void visit(const unsigned first, const unsigned stride, F&& f, bool, bool) const {
        long long done = 0;
        if (!(reinterpret_cast<unsigned long long>(x) & 15ull)) {
            // four values per thread and two loads in flight
            const float4* x4 = reinterpret_cast<const float4*>(x);
            const long long quads = n >> 2;
            done = quads << 2;
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            const bool mine = first + threadIdx.x < stride;
            for (long long base = first; base < quads; base += 2ll * stride) {
                const long long l0 = base + threadIdx.x, l1 = l0 + stride;
                const bool v0 = mine && l0 < quads, v1 = mine && l1 < quads;
                const float4 q0 = v0 ? __ldg(x4 + l0) : zero, q1 = v1 ? __ldg(x4 + l1) : zero;
#pragma unroll
                for (int k = 0; k < 4; ++k) f(v0, fabsf(comp(q0, k)), 0.f);
#pragma unroll
                for (int k = 0; k < 4; ++k) f(v1, fabsf(comp(q1, k)), 0.f);
            }
        }
        for (long long base = done + first; base < n; base += stride) {
            const long long l = base + threadIdx.x;
            const bool valid = first + threadIdx.x < stride && l < n;
            f(valid, valid ? fabsf(x[l]) : 0.f, 0.f);
        }
    }
};

// One value in 32 of a flat vector: of every whole block of 1024 a run of 32,
// its place hashed (a fixed stride could fall in step with the data).
struct SampleSrc {
    using Sum = Kahan;
    const float* x;
    long long n;            // sampled values, a multiple of 32
    template <typename F>
    __device__ void visit(const unsigned first, const unsigned stride, F&& f, bool, bool) const {
        for (long long base = first; base < n; base += stride) {
            const long long e = base + threadIdx.x;
            const bool valid = first + threadIdx.x < stride && e < n;
            const unsigned run = ((unsigned)(e >> 5) * 2654435761u) >> 27;
            const long long l = ((e >> 5) << 10) + 32u * run + (e & 31);
            f(valid, valid ? fabsf(__ldg(x + l)) : 0.f, 0.f);
        }
    }
};

struct SearchArgs {
    Scal* sc;
    L1Work w;
    int nvec;        // 2 for the cube (s, t), 1 for a flat vector
    int cta_base = 0, cta_total = 0;   // this launch's CTAs among the stage's (0: alone)
    __device__ int total(int nblk) const { return cta_total > 0 ? cta_total : nblk; }
};

// Radix histogram pass of one level for every vector that needs it.
template <typename Src>
__device__ __forceinline__ void radix_count(const Src& src, const SearchArgs& a, const int level, const int bid,
                                            const int nblk) {
    extern __shared__ __align__(16) unsigned hsm[];   // [2][2048] counts, low and high residue halves
    const int want = NEED_RADIX0 + level;
    bool need[2];
    need[0] = a.sc->ctl[0].need == want;
    need[1] = a.nvec > 1 && a.sc->ctl[1].need == want;
    if (!need[0] && !need[1]) return;
    const RadixLevel lv{level};
    const int nb = lv.nbins();
    // 32-bit shared bins: count, and the residue split into its low and high
    // 10 bits so that a CTA's sums stay below 2^32 (it sees at most 2^21
    // values per vector, each half below 2^10); every add is fire-and-forget,
    // so no lane waits on a result
    unsigned* hc = hsm;
    unsigned* hrl = hsm + 2 * kHistBins;
    unsigned* hrh = hsm + 4 * kHistBins;
    for (int k = threadIdx.x; k < 6 * kHistBins; k += blockDim.x) hsm[k] = 0;
    __syncthreads();
    const unsigned pre0 = a.sc->ctl[0].prefix, pre1 = a.sc->ctl[1].prefix;
    auto insert = [&](int v, bool take, unsigned key) {
        if (take) {
            const int bn = v * kHistBins + lv.bin(key);
            const unsigned r = lv.residue(key);
            atomicAdd(hc + bn, 1u);
            if (r) {
                atomicAdd(hrl + bn, r & 1023u);
                atomicAdd(hrh + bn, r >> 10);
            }
        }
    };
    src.visit(bid * blockDim.x, nblk * blockDim.x, [&](bool valid, float x0, float x1) {
        if (need[0]) {
            const unsigned key = __float_as_uint(x0);
            insert(0, valid && lv.inside(key, pre0), key);
        }
        if (need[1]) {
            const unsigned key = __float_as_uint(x1);
            insert(1, valid && lv.inside(key, pre1), key);
        }
    }, need[0], need[1]);
    __syncthreads();
    for (int k = threadIdx.x; k < 2 * kHistBins; k += blockDim.x) {
        if ((k % kHistBins) >= nb) continue;
        if (hc[k]) atomicAdd(a.w.hcnt + k, (unsigned long long)hc[k]);
        const unsigned long long res = ((unsigned long long)hrh[k] << 10) + hrl[k];
        if (res) atomicAdd(a.w.hres + k, res);
    }
}

// Selects the bracket of one level once every CTA has counted; one whole block.
__device__ __forceinline__ void radix_finish(const SearchArgs& a, const int level) {
    __shared__ double sh_d[NT];
    __shared__ unsigned long long sh_u[NT];
    __shared__ int sh_i[1];
    const int want = NEED_RADIX0 + level;
    const RadixLevel lv{level};
    bool need[2];
    need[0] = a.sc->ctl[0].need == want;
    need[1] = a.nvec > 1 && a.sc->ctl[1].need == want;
    for (int v = 0; v < 2; ++v) {
        if (!need[v]) continue;
        l1_radix_select(a.sc->ctl[v], lv, a.w.hcnt + v * kHistBins, a.w.hres + v * kHistBins,
                        a.sc->radius[v], sh_d, sh_u, sh_i);
    }
    for (int k = threadIdx.x; k < 2 * kHistBins; k += blockDim.x) { a.w.hcnt[k] = 0; a.w.hres[k] = 0; }
}

// A level in a launch of its own; the last CTA selects the bracket.
template <typename Src>
__device__ __forceinline__ void radix_body(const Src& src, const SearchArgs& a, const int level, const int bid,
                                           const int nblk) {
    __shared__ int is_last;
    const int want = NEED_RADIX0 + level;
    if (a.sc->ctl[0].need != want && !(a.nvec > 1 && a.sc->ctl[1].need == want)) return;
    radix_count(src, a, level, bid, nblk);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(&a.sc->fb_ticket, 1u) == (unsigned)(a.total(nblk) - 1));
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    radix_finish(a, level);
    if (threadIdx.x == 0) a.sc->fb_ticket = 0;
}

template <typename Src>
__global__ void __launch_bounds__(NT) k_radix(const Src src, const SearchArgs a, const int level) {
    radix_body(src, a, level, blockIdx.x, gridDim.x);
}

// Candidates of one CTA collected in shared memory and appended to the global
// lists with one atomic per vector at the end of the pass (a warp-level global
// atomic per candidate serialises on the counter once windows are wide).
// What overflows the shared buffer goes straight to the global list.
constexpr int kBlkCand = 1024;           // per vector in a 256-thread CTA's static shared memory
struct BlockCand {
    float* buf[2];
    unsigned cap;
    unsigned* cnt;     // [2]
    unsigned* base;    // [2]
    // the lists' key histograms over the windows (null: not kept)
    unsigned* nh[2] = {nullptr, nullptr};
    unsigned* nbinned = nullptr;
    NarrowGeom ng[2];
    __device__ void init() {
        if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
        __syncthreads();
    }
    // keep vector v's list histogram over the key window (lo, hi]
    __device__ void keep_hist(const L1Work& w, int v, float lo, float hi) {
        ng[v] = narrow_geom(__float_as_uint(lo), __float_as_uint(hi));
        nh[v] = w.nh && ng[v].ok ? w.nh + v * 3 * kNarrowBins : nullptr;
        nbinned = w.nbinned;
    }
    // values past the buffer go straight to the global list and its histogram
    __device__ void append(int v, bool take, float x, float* gcand, unsigned* gcnt) {
        const unsigned mask = __ballot_sync(0xffffffffu, take);
        if (mask == 0) return;
        const int lane = threadIdx.x & 31;
        const int leader = __ffs(mask) - 1;
        unsigned b = 0;
        if (lane == leader) b = atomicAdd(cnt + v, (unsigned)__popc(mask));
        b = __shfl_sync(0xffffffffu, b, leader);
        const unsigned k = b + __popc(mask & ((1u << lane) - 1u));
        if (take && k < cap) buf[v][k] = x;
        if (b + __popc(mask) > cap) {
            const bool over = take && k >= cap;
            append_candidate(over, x, gcand, gcnt);
            if (over && nh[v]) {
                narrow_add(nh[v], ng[v], __float_as_uint(x));
                atomicAdd(nbinned + v, 1u);
            }
        }
    }
    // whole block; before the pass's completion ticket
    __device__ void flush(float* const* gcand, Scal* sc) {
        __syncthreads();
        if (threadIdx.x < 2) {
            const unsigned n = min(cnt[threadIdx.x], cap);
            base[threadIdx.x] = n ? atomicAdd(&sc->acc[threadIdx.x].m, n) : 0u;
        }
        __syncthreads();
        for (int v = 0; v < 2; ++v) {
            const unsigned n = min(cnt[v], cap);
            for (unsigned k = threadIdx.x; k < n; k += blockDim.x)
                if (base[v] + k < kCandCap) gcand[v][base[v] + k] = buf[v][k];
        }
    }
    // after flush: counts the buffered candidates of vector v into the list's
    // key histogram (kept by keep_hist)
    __device__ void bin(int v) {
        if (!nh[v]) return;
        const unsigned n = min(cnt[v], cap);
        for (unsigned k = threadIdx.x; k < n; k += blockDim.x) narrow_add(nh[v], ng[v], __float_as_uint(buf[v][k]));
        if (threadIdx.x == 0 && n) atomicAdd(nbinned + v, n);
    }
};
// The buffers: the static ones, or `store` (cap floats per vector).
struct CandStore {
    float* p = nullptr;
    unsigned cap = 0;
};
#define GSSTV_BLOCK_CAND(name, store)                                                                  \
    __shared__ float name##_buf[2][kBlkCand];                                                          \
    __shared__ unsigned name##_cnt[2], name##_base[2];                                                 \
    BlockCand name{{store.p ? store.p : name##_buf[0], store.p ? store.p + store.cap : name##_buf[1]}, \
                   store.p ? store.cap : (unsigned)kBlkCand, name##_cnt, name##_base};                 \
    name.init()

// Gathers the bracket bin of every vector that needs it (finish_body
// finishes tau).
template <typename Src>
__device__ __forceinline__ void gather_body(const Src& src, const SearchArgs& a, const int bid, const int nblk,
                                            const CandStore store = CandStore()) {
    bool need[2];
    need[0] = a.sc->ctl[0].need == NEED_GATHER;
    need[1] = a.nvec > 1 && a.sc->ctl[1].need == NEED_GATHER;
    if (!need[0] && !need[1]) return;
    const float lo0 = a.sc->ctl[0].g_lo, hi0 = a.sc->ctl[0].g_hi;
    const float lo1 = a.sc->ctl[1].g_lo, hi1 = a.sc->ctl[1].g_hi;
    GSSTV_BLOCK_CAND(bc, store);
    if (need[0]) bc.keep_hist(a.w, 0, lo0, hi0);
    if (need[1]) bc.keep_hist(a.w, 1, lo1, hi1);
    src.visit(bid * blockDim.x, nblk * blockDim.x, [&](bool valid, float x0, float x1) {
        if (need[0]) bc.append(0, valid && x0 > lo0 && x0 <= hi0, x0, a.w.cand[0], &a.sc->acc[0].m);
        if (need[1]) bc.append(1, valid && x1 > lo1 && x1 <= hi1, x1, a.w.cand[1], &a.sc->acc[1].m);
    }, need[0], need[1]);
    bc.flush(a.w.cand, a.sc);
    bc.bin(0);
    bc.bin(1);
}

template <typename Src>
__global__ void __launch_bounds__(NT) k_gather(const Src src, const SearchArgs a) {
    gather_body(src, a, blockIdx.x, gridDim.x);
}

// One windowed pass after K1's window missed: count and sum of |x| above the
// retry window and its values as candidates (finish_body runs Michelot's
// finish; a second miss leaves the threshold to the radix passes).  Per-CTA
// partial sums go to pn / ps (the stencil pass's partial arrays, free by now).
template <typename Src>
__device__ __forceinline__ void window_body(const Src& src, const SearchArgs& a, unsigned long long* pn, double* ps,
                                            const int bid, const unsigned stride,
                                            const CandStore store = CandStore()) {
    __shared__ double red_d[64];
    __shared__ unsigned long long red_u[64];
    bool need[2];
    need[0] = a.sc->ctl[0].need == NEED_WINDOW;
    need[1] = a.nvec > 1 && a.sc->ctl[1].need == NEED_WINDOW;
    if (!need[0] && !need[1]) return;
    const float lo0 = a.sc->ctl[0].g_lo, hi0 = a.sc->ctl[0].g_hi;
    const float lo1 = a.sc->ctl[1].g_lo, hi1 = a.sc->ctl[1].g_hi;
    WinAcc<typename Src::Sum> w0, w1;
    GSSTV_BLOCK_CAND(bc, store);
    if (need[0]) bc.keep_hist(a.w, 0, lo0, hi0);
    if (need[1]) bc.keep_hist(a.w, 1, lo1, hi1);
    src.visit(bid * blockDim.x, stride, [&](bool valid, float x0, float x1) {
        if (need[0]) {
            // (a flat vector's NaN counts as above, so that the window misses and
            // the radix passes decide)
            const bool hi = valid && (std::is_same<Src, FlatSrc>::value ? !(x0 <= hi0) : x0 > hi0);
            if (hi) { w0.n++; w0.s.add(x0); }
            bc.append(0, valid && !hi && x0 > lo0, x0, a.w.cand[0], &a.sc->acc[0].m);
        }
        if (need[1]) {
            const bool hi = valid && x1 > hi1;
            if (hi) { w1.n++; w1.s.add(x1); }
            bc.append(1, valid && !hi && x1 > lo1, x1, a.w.cand[1], &a.sc->acc[1].m);
        }
    }, need[0], need[1]);
    bc.flush(a.w.cand, a.sc);
    bc.bin(0);
    bc.bin(1);
    float2* pbuf = reinterpret_cast<float2*>(red_d);
    const unsigned long long n0 = block_sum(w0.n, red_u), n1 = block_sum(w1.n, red_u);
    const double s0 = block_sum_pair(w0.s, pbuf), s1 = block_sum_pair(w1.s, pbuf);
    const int cta = a.cta_base + bid;
    if (threadIdx.x == 0) {
        pn[2 * cta] = n0; pn[2 * cta + 1] = n1;
        ps[2 * cta] = s0; ps[2 * cta + 1] = s1;
    }
}

template <typename Src>
__global__ void __launch_bounds__(NT) k_window(const Src src, const SearchArgs a, unsigned long long* pn,
                                               double* ps) {
    window_body(src, a, pn, ps, blockIdx.x, gridDim.x * blockDim.x);
}

// The finish of K1's window (mode 2), of the retry window (mode 0) or of the
// gathered radix bracket (mode 1) of vector v, if it needs it: one CTA of kFinishThreads threads,
// the candidates staged in its shared memory when they fit (kFinishStage
// floats), narrowed on the float keys and finished by Michelot's step (see
// l1_window_finish).  A single CTA walking a list of a few hundred thousand
// candidates is bound by the latency of its loads, so it runs apart from the
// main pass with the most threads a CTA can have, and the vectors' searches
// (independent) run in CTAs of their own.  parts: the main pass's CTAs (mode
// 0: their count and sum above the window in pn / ps, two per CTA; mode 2:
// K1's four per CTA, the window's and the histogram's above-range statistics
// of both vectors).
constexpr int kFinishThreads = 1024;
constexpr unsigned kFinishStage = 32768;

// tau inside the window (lo, hi] of m values by one warp: 0 found, 1 below, 2
// above or no number (as l1_window_finish), -1 not settled.  Newton's steps on phi
// from the window's middle, where the window was predicted around: from the right
// of the root a step lands left of it, from there they do not pass it, so that the
// counts fall, and a repeated count means the active set is the root's.  (A count
// that rises again has met a value equal to tau but for its rounding.)  Sums that
// overflow give a tau that is no number.
__device__ __forceinline__ bool window_settled(int it, unsigned c, unsigned prev) {
    return c == prev || (it > 2 && c > prev);
}
__device__ __forceinline__ int warp_window(const float* x, unsigned m, double n_hi, double s_hi, float lo, float hi,
                                           double r, double* tau_out) {
    const unsigned lane = threadIdx.x & 31u;
    if (!(s_hi - n_hi * (double)hi - r <= 0.0)) return 2;
    float tf = -INFINITY;                                 // first the sum of all values: phi at lo
    unsigned prev = 0xffffffffu;
#pragma unroll 1
    for (int it = 0; it < 200; ++it) {
        Kahan k;
        unsigned c = 0;
#pragma unroll 1
        for (unsigned e = lane; e < m; e += 32u) {
            const float y = x[e];
            const bool in = y > tf;
            k.add(in ? y : 0.f);
            c += in ? 1u : 0u;
        }
        c = __reduce_add_sync(0xffffffffu, c);
        float h = k.s, l = -k.c;
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
            pair_add(h, l, oh, ol);
        }
        const double num = s_hi + ((double)h + (double)l) - r, den = n_hi + (double)c;
        if (it == 0) {
            if (num - den * (double)lo < 0.0) {           // phi(lo) < 0: inside the ball, or a miss below
                *tau_out = 0.0;
                return lo <= 0.f ? 0 : 1;
            }
            tf = 0.5f * (lo + hi);
        } else {
            const double tau = num / den;
            tf = __double2float_rd(tau);
            if (window_settled(it, c, prev)) {
                *tau_out = tau;
                return isfinite(tau) ? 0 : -1;
            }
            prev = c;
        }
    }
    return -1;
}

// The same by the whole block on m values in shared memory (a finish through the
// narrowing took 34 us and more; 157x203x61: a pass 139 -> 131 us).
__device__ __forceinline__ int block_window(const float* x, unsigned m, double n_hi, double s_hi, float lo, float hi,
                                            double r, double* tau_out) {
    __shared__ float2 part[32];
    __shared__ unsigned cnt[32];
    __shared__ float sh_tf;
    __shared__ int sh_state;                              // 0 go on, 1 found, 2 inside the ball, 3 below, 4 above, 5 no number
    __shared__ double sh_tau;
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float tf = -INFINITY;
    unsigned prev = 0xffffffffu;
#pragma unroll 1
    for (int it = 0; it < 200; ++it) {
        Kahan k;
        unsigned c = 0;
#pragma unroll 4
        for (unsigned e = threadIdx.x; e < m; e += blockDim.x) {
            const float y = x[e];
            const bool in = y > tf;
            k.add(in ? y : 0.f);
            c += in ? 1u : 0u;
        }
        c = __reduce_add_sync(0xffffffffu, c);
        float h = k.s, l = -k.c;
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
            pair_add(h, l, oh, ol);
        }
        if (lane == 0) { part[wid] = make_float2(h, l); cnt[wid] = c; }
        __syncthreads();
        if (wid == 0) {
            h = lane < nw ? part[lane].x : 0.f;
            l = lane < nw ? part[lane].y : 0.f;
            c = __reduce_add_sync(0xffffffffu, lane < nw ? cnt[lane] : 0u);
#pragma unroll 1
            for (int o = 16; o > 0; o >>= 1) {
                const float oh = __shfl_xor_sync(0xffffffffu, h, o), ol = __shfl_xor_sync(0xffffffffu, l, o);
                pair_add(h, l, oh, ol);
            }
            const double num = s_hi + ((double)h + (double)l) - r, den = n_hi + (double)c;
            int state = 0;
            double tau = 0.0;
            if (it == 0) {
                tf = 0.5f * (lo + hi);
                if (!(s_hi - n_hi * (double)hi - r <= 0.0)) state = 4;
                else if (num - den * (double)lo < 0.0) state = lo <= 0.f ? 2 : 3;
            } else {
                tau = num / den;
                tf = __double2float_rd(tau);
                if (window_settled(it, c, prev)) state = isfinite(tau) ? 1 : 5;
                prev = c;
            }
            if (lane == 0) { sh_tf = tf; sh_state = state; sh_tau = tau; }
        }
        __syncthreads();
        tf = sh_tf;
        if (sh_state) break;
        __syncthreads();
    }
    const int state = sh_state;
    *tau_out = state == 2 ? 0.0 : sh_tau;
    return state == 3 ? 1 : state == 4 ? 2 : state == 1 || state == 2 ? 0 : -1;
}

// K1's window of vector v, after the fused pass: the CTAs' counts and sums
// above the window summed, tau found on the candidates (l1_window_finish); on
// a miss, K1's sampled histogram (when it was on) brackets tau for one retry
// pass, else the next window is placed from the bounds the miss gives or the
// radix passes run.  The whole block; K1's partials: pn / ps, four per CTA.
__device__ __noinline__ int k1_window_finish(const SearchArgs& a, const unsigned long long* pn, const double* ps,
                                              int parts, const int v, float* fstage, unsigned* scr, double* red_d,
                                              unsigned long long* red_u) {
    __shared__ int sh_flag;
    __shared__ int sh_rc;
    L1Ctl& C = a.sc->ctl[v];
    // everything the finish starts from in one round of loads: the scalars, the
    // first candidates, and in warp 0 K1's partials (one per SM; one warp, so
    // that the FP64 additions, scarce on this part, are not issued by every warp)
    const double r = __ldcg(&a.sc->radius[v]);
    const int win = __ldcg(&a.sc->k1_win[v]), hist_w = __ldcg(&a.sc->k1_hist[v]), hist_left = __ldcg(&C.hist_left);
    const unsigned m = __ldcg(&a.sc->acc[v].m), nbin = a.w.nh ? __ldcg(a.w.nbinned + v) : 0u;
    const float tlo_f = __ldcg(&C.theta_lo), thi_f = __ldcg(&C.theta_hi);
    const float x0 = __ldcg(a.w.cand[v] + threadIdx.x);          // (the list holds kCandCap floats)
    unsigned n = 0;                                              // (fewer than 2^32 voxels)
    double s = 0.0;
    if (threadIdx.x < 32) {
#pragma unroll 5
        for (int k = threadIdx.x; k < parts; k += 32) {
            n += (unsigned)__ldcg(pn + 4 * k + v);
            s += __ldcg(ps + 4 * k + v);
        }
    }
    fstage[threadIdx.x] = x0;
    if (!(__double_as_longlong(r) > 0)) {
        if (threadIdx.x == 0) {
            C.tau = __int_as_float(0x7f800000);
            C.have_tau = 1;
            C.need = NEED_NONE;
            C.window_ok = 0;
        }
        return NEED_NONE;
    }
    if (!win) {
        if (threadIdx.x == 0) {
            C.need = NEED_RADIX0; C.prefix = 0; C.n_above = 0; C.s_above = 0.0; C.exact_runs++;
        }
        return NEED_RADIX0;
    }
    const bool hist_v = hist_w != 0;
    __syncthreads();
    if (threadIdx.x < 32) {
        n = __reduce_add_sync(0xffffffffu, n);
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        // A window of few values (the steady state): warp 0 finds tau alone.
        // This launch runs its code once, so the instruction fetches are what
        // it waits for (the same steps took 21 us after passes that stay in L2
        // and 34 us after larger ones): short loops over all the values beat the
        // narrowing by the list's histogram up to here.
        double tau = 0.0;
        const int rc = m > (unsigned)kFinishThreads ? -1 : warp_window(fstage, m, (double)n, s, tlo_f, thi_f, r, &tau);
        if (threadIdx.x == 0) {
            sh_rc = rc;
            red_d[0] = s;
            red_u[0] = n;
            red_d[1] = tau;
            red_d[2] = (double)n;
        }
    }
    __syncthreads();
    if (m > (unsigned)kFinishThreads && m <= kFinishStage) {
        double tau = 0.0;
        const float* cand = a.w.cand[v];
#pragma unroll 8
        for (unsigned e = threadIdx.x + kFinishThreads; e < m; e += kFinishThreads) fstage[e] = __ldcg(cand + e);
        __syncthreads();
        const int rc = block_window(fstage, m, red_d[2], red_d[0], tlo_f, thi_f, r, &tau);
        if (threadIdx.x == 0) { sh_rc = rc; red_d[1] = tau; }
        __syncthreads();
    }
    if (sh_rc == 0) {
        if (threadIdx.x == 0) {
            l1_record_tau(C, red_d[1], (double)m, (double)thi_f - (double)tlo_f, true);
            atomicAdd(reinterpret_cast<unsigned long long*>(&C.hits), 1ull);
            // (counted down where K1 keeps the histogram: float32 storage)
            if (hist_left > 0 && win == 1) C.hist_left = hist_left - 1;
            a.sc->acc[v].m = 0;
        }
        if (nbin) {
            uint4* h4 = reinterpret_cast<uint4*>(a.w.nh + v * 3 * kNarrowBins);
            for (int k = threadIdx.x; k < 2 * kNarrowBins / 4; k += kFinishThreads) h4[k] = make_uint4(0u, 0u, 0u, 0u);
            if (threadIdx.x == 0) a.w.nbinned[v] = 0u;
        }
        if (hist_v) a.w.khist[v * kK1Bins + threadIdx.x] = 0u;
        return NEED_NONE;
    }
    n = (unsigned)red_u[0];
    s = red_d[0];
    __syncthreads();
    const double tlo = tlo_f, thi = thi_f;
    double tau = 0.0;
    WinInfo wi;
    const int miss = l1_window_finish((double)n, s, a.w.cand[v], m, tlo, thi, r, &tau, red_d, red_u, &wi, fstage,
                                      kFinishStage, scr, m > 0u && nbin == m ? a.w.nh + v * 3 * kNarrowBins : nullptr,
                                      a.w.nbinned + v);
    narrow_clear(a.w, v);
    int hist_hit = 0;
    float h_lo = 0.f, h_hi = 0.f;
    double h_m = 0.0;
    if (miss && hist_v) {
        unsigned long long hn = 0;
        double hs = 0.0;
        for (int k = threadIdx.x; k < parts; k += blockDim.x) {
            hn += __ldcg(pn + 4 * k + 2 + v);
            hs += __ldcg(ps + 4 * k + 2 + v);
        }
        hn = block_sum(hn, red_u);
        hs = block_sum(hs, red_d);
        hist_hit = l1_hist_bracket(a.w.khist + v * kK1Bins, C.hbase, (double)hn, hs, r, (double)kHistSample,
                                   &h_lo, &h_hi, &h_m, &sh_flag, reinterpret_cast<unsigned*>(fstage));
    }
    if (hist_v) {
        __syncthreads();
        for (int k = threadIdx.x; k < kK1Bins; k += blockDim.x) a.w.khist[v * kK1Bins + k] = 0u;
    }
    if (threadIdx.x == 0) {
        if (!miss) {
            l1_record_tau(C, tau, (double)min(m, kCandCap), thi - tlo, true);
            C.hits++;
            if (hist_left > 0 && win == 1) C.hist_left = hist_left - 1;
        } else if (hist_hit) {
            C.prefix = 0; C.n_above = 0; C.s_above = 0.0;
            C.need = NEED_WINDOW;
            C.g_lo = h_lo;
            C.g_hi = h_hi;
            C.hist_left = kHistPasses;
        } else {
            l1_after_miss(C, miss, wi, (double)n, m, tlo, thi);
        }
        a.sc->acc[v].m = 0;
    }
    __syncthreads();
    return -1;
}

constexpr size_t kFinishSmem = kFinishStage * sizeof(float) + 3 * kNarrowBins * sizeof(unsigned);
__device__ __forceinline__ int finish_body(const SearchArgs& a, int mode, const unsigned long long* pn,
                                            const double* ps, int parts, const int v) {
    extern __shared__ __align__(16) float fstage[];         // kFinishStage floats + the narrowing scratch
    __shared__ double red_d[64];
    __shared__ unsigned long long red_u[64];
    const int want = mode == 0 ? NEED_WINDOW : NEED_GATHER;
    unsigned* scr = reinterpret_cast<unsigned*>(fstage + kFinishStage);
    if (v >= a.nvec) return -1;
    if (mode == 2) return k1_window_finish(a, pn, ps, parts, v, fstage, scr, red_d, red_u);
    {
        L1Ctl& C = a.sc->ctl[v];
        if (C.need != want) return -1;                      // uniform over the CTA
        const double r = a.sc->radius[v];
        const unsigned m = __ldcg(&a.sc->acc[v].m);
        const double lo = C.g_lo, hi = C.g_hi;
        double n = 0.0, sm = 0.0;
        if (mode == 0) {
            unsigned long long nn = 0;
            double ss = 0.0;
            for (int k = threadIdx.x; k < parts; k += blockDim.x) {
                nn += __ldcg(pn + 2 * k + v);
                ss += __ldcg(ps + 2 * k + v);
            }
            n = (double)block_sum(nn, red_u);
            sm = block_sum(ss, red_d);
        } else {
            n = (double)C.n_above;
            sm = C.s_above;
        }
        double tau = 0.0;
        const int rc = l1_window_finish(n, sm, a.w.cand[v], m, lo, hi, r, &tau, red_d, red_u, nullptr, fstage,
                                        kFinishStage, scr, narrow_pre(a.w, v, m), a.w.nbinned + v);
        narrow_clear(a.w, v);
        if (threadIdx.x == 0) {
            if (mode == 0) {
                if (rc == 0) {
                    l1_record_tau(C, tau, (double)min(m, kCandCap), hi - lo, false);
                    C.retry_hits++;
                } else {
                    C.need = NEED_RADIX0; C.prefix = 0; C.n_above = 0; C.s_above = 0.0;
                    C.exact_runs++;
                }
            } else {
                if (rc == 2 && n > 0.0) {
                    // the root lies between the largest value of the bin and
                    // the next bin's edge: every value of the bin is inactive
                    tau = (sm - r) / n;
                } else if (rc != 0) {
                    atomicOr(&a.sc->error, 2);
                }
                l1_record_tau(C, tau, (double)min(m, kCandCap), hi - lo, false);
            }
            a.sc->acc[v].m = 0;
        }
        __syncthreads();
    }
    return -1;
}

// After K1's window finish (mode 2) in a graph: the last of the launch's
// CTAs opens the conditional node of the search launches when a cube still
// needs a search (one thread, so that no two calls race).  need_any() reads the
// cubes' flags after every CTA's have landed.
template <typename F>
__device__ __forceinline__ void finish_gate(Scal* counter, unsigned total, cudaGraphConditionalHandle cond,
                                            F&& need_any) {
    __shared__ int last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&counter->fin_ticket, 1u) == total - 1u;
    }
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        counter->fin_ticket = 0u;
        const unsigned need = need_any() ? 1u : 0u;
        if (need) counter->gate_opens++;
        cudaGraphSetConditional(cond, need);
    }
}
__device__ __forceinline__ bool scal_needs_search(const Scal* s) {
    return !__ldcg(&s->done) && (__ldcg(&s->ctl[0].need) != NEED_NONE || __ldcg(&s->ctl[1].need) != NEED_NONE);
}

// one CTA per vector; gated: a graph's conditional node waits on this launch
__global__ void __launch_bounds__(kFinishThreads) k_search_finish(const SearchArgs a, int mode,
                                                                   const unsigned long long* pn,
                                                                   const double* ps, int parts, int gated,
                                                                   cudaGraphConditionalHandle cond) {
    finish_body(a, mode, pn, ps, parts, blockIdx.x);
    if (gated) finish_gate(a.sc, gridDim.x, cond, [&] { return scal_needs_search(a.sc); });
}

// ---------------------------------------------------------------------------
// the threshold search of a pass in one launch
// ---------------------------------------------------------------------------
// Between K1 and K2: the finish of K1's window (two CTAs, one per vector) and,
// when a vector's window missed, the retry, radix and gather passes on all CTAs.
// The stages follow one another inside the launch.  (With the search launches in
// a conditional graph node, every pass paid 8.5 us between the finish and K2 for
// the node alone, opened or not; passes launched one by one paid for seven
// launches that returned at once.)
//
// A stage is a number of items that CTAs draw from a counter; the CTA that
// completes a stage's last item decides the next stage and publishes it.  A CTA
// only ever waits for items that running CTAs hold, so the launch needs no
// co-residency and may share the GPU with others of its kind.  K2 clears the
// counters for the next pass.  Waits are bounded.
enum { ST_FINISH = 0, ST_WINDOW, ST_WINDOW_END, ST_RADIX0, ST_RADIX1, ST_RADIX2, ST_GATHER, ST_GATHER_END, ST_EXIT };
static_assert(ST_GATHER_END < kSearchStages, "counters per stage");

struct SearchShape {
    int parts;              // K1's partials (-1: no K1, the first stage is set already)
    unsigned win_threads;   // threads that share the retry pass (a multiple of 256)
    int win_items, pass_items;
    int count;              // count the passes that searched (graph launches)
};

__device__ __forceinline__ unsigned search_stage(const SearchSync* y) {
    unsigned w;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(&y->stage) : "memory");
    return w;
}

// The stage after `st` from the vectors' needs (thread 0).
__device__ __forceinline__ int search_next(const SearchArgs& a, int st) {
    if (st == ST_WINDOW) return ST_WINDOW_END;
    if (st == ST_GATHER) return ST_GATHER_END;
    int next = ST_EXIT;
    for (int v = 0; v < a.nvec; ++v) {
        const int need = __ldcg(&a.sc->ctl[v].need);
        const int s = need == NEED_WINDOW ? ST_WINDOW : need == NEED_RADIX0 ? ST_RADIX0 : need == NEED_RADIX1 ? ST_RADIX1
                    : need == NEED_RADIX2 ? ST_RADIX2 : need == NEED_GATHER ? ST_GATHER : ST_EXIT;
        if (s > st) next = min(next, s);
    }
    return next;
}

template <typename Src>
__device__ __forceinline__ void search_body(const Src& src, const SearchArgs& a, unsigned long long* pn, double* ps,
                                            const SearchShape& h, const int bid) {
    extern __shared__ __align__(16) float fstage[];
    __shared__ int sh_stage, sh_item, sh_last;
    // an item's candidates wait in the finish's stage, free in these stages: 152
    // CTAs with 1024 places a vector overflowed into single atomics on the global
    // list (a retry pass of 512x512x224 appends 180-360 thousand)
    const CandStore store{fstage, kFinishStage / 2};
    SearchSync* y = &a.sc->search;
    auto publish = [&](int next) {                       // (thread 0)
        __threadfence();
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&y->stage), "r"((unsigned)next) : "memory");
    };
    // whole block: an item of stage st is done; the last of n publishes the next stage
    auto complete = [&](int st, int n) {
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            sh_last = atomicAdd(&y->done[st], 1u) == (unsigned)(n - 1);
            __threadfence();
        }
        __syncthreads();
        if (!sh_last) return;
        if (st >= ST_RADIX0 && st <= ST_RADIX2) {
            __threadfence();
            radix_finish(a, st - ST_RADIX0);
            __threadfence();
            __syncthreads();
        }
        if (threadIdx.x == 0) publish(search_next(a, st));
    };
    if (h.parts >= 0 && bid < a.nvec) {
        // the finishes' count carries in its upper half whether a vector still
        // needs a search, so that the usual pass reads nothing back
        const bool need = finish_body(a, 2, pn, ps, h.parts, bid) != NEED_NONE;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            const unsigned was = atomicAdd(&y->done[ST_FINISH], need ? 0x10001u : 1u);
            if ((was & 0xffffu) == (unsigned)(a.nvec - 1)) {
                __threadfence();
                const int next = need || (was >> 16) ? search_next(a, ST_FINISH) : (int)ST_EXIT;
                if (next != ST_EXIT && h.count) a.sc->gate_opens++;
                publish(next);
            }
        }
    }
    for (int st = ST_FINISH;;) {
        if (threadIdx.x == 0) {
            unsigned w = search_stage(y);
            for (unsigned k = 0; w <= (unsigned)st && k < kSearchSpinLimit; ++k) {
                __nanosleep(100);
                w = search_stage(y);
            }
            if (w <= (unsigned)st) {
                atomicOr(&a.sc->error, 4);
                w = ST_EXIT;
            }
            sh_stage = (int)w;
        }
        __syncthreads();
        st = sh_stage;
        if (st >= ST_EXIT) return;
        const int n = st == ST_WINDOW ? h.win_items : st == ST_WINDOW_END || st == ST_GATHER_END ? a.nvec : h.pass_items;
        for (;;) {
            if (threadIdx.x == 0) sh_item = (int)atomicAdd(&y->next[st], 1u);
            __syncthreads();
            const int item = sh_item;
            if (item >= n) break;
            if (st == ST_WINDOW) window_body(src, a, pn, ps, item, h.win_threads, store);
            else if (st == ST_WINDOW_END) finish_body(a, 0, pn, ps, h.win_items, item);
            else if (st == ST_GATHER) gather_body(src, a, item, n, store);
            else if (st == ST_GATHER_END) finish_body(a, 1, pn, ps, 0, item);
            else radix_count(src, a, st - ST_RADIX0, item, n);
            complete(st, n);
        }
        __syncthreads();
    }
}

template <typename Src>
__global__ void __launch_bounds__(kFinishThreads) k_search(const Src src, const SearchArgs a, unsigned long long* pn,
                                                           double* ps, const SearchShape h) {
    search_body(src, a, pn, ps, h, blockIdx.x);
}

// The standalone projection between its two searches: tau of the sample (1 / scale
// of the values) places the window of one pass over all of them.  0.5 % about
// tau is several standard deviations of the sample's for vectors this long; a
// miss costs the radix passes.  A sample inside its ball says nothing about a
// root near zero: the radix passes run at once.
__global__ void k_flat_window(Scal* sc, double radius, double scale) {
    if (threadIdx.x != 0) return;
    L1Ctl& c = sc->ctl[0];
    sc->radius[0] = radius;
    sc->search = SearchSync();
    sc->acc[0].m = 0u;
    c.prefix = 0; c.n_above = 0; c.s_above = 0.0;
    if (c.tau > 0.0 && isfinite(c.tau)) {
        double hw = 0.005 * c.tau;
        if (c.dens > 0.0) hw = fmin(hw, 0.25 * (double)kCandCap / (c.dens * scale));
        c.g_lo = __double2float_rd(c.tau - hw);
        c.g_hi = __double2float_ru(c.tau + hw);
        c.need = NEED_WINDOW;
        sc->search.stage = ST_WINDOW;
    } else {
        c.need = NEED_RADIX0;
        sc->search.stage = ST_RADIX0;
    }
}

// The standalone projection of at most kSmallProject values by one CTA: with everything a candidate the finish's steps are the whole
// search.  (4096 values took 59 us in the radix stages, whose code runs once.)  As
// there, a NaN leaves the vector as it is and an infinity makes tau infinite.
// The block's sums are float pairs, so values whose sum could pass the largest
// float (2^13 of them at 2^112 and more) are scaled by 2^-32 first: exact, but for
// bits below 2^-200 of the largest value.
constexpr unsigned kSmallProject = 8192;
constexpr float kProjectHuge = 0x1p112f, kProjectDown = 0x1p-32f;
static_assert(kSmallProject <= 1u << 13, "a sum of values below kProjectHuge stays a float");
__global__ void __launch_bounds__(1024) k_project_small(const float* x, float* out, unsigned n, double radius,
                                                        double* tau_out) {
    __shared__ float xs[kSmallProject];
    __shared__ double sh_tau;
    bool nan = false, inf = false, huge = false;
    for (unsigned e = threadIdx.x; e < n; e += blockDim.x) {
        const float y = x[e];
        xs[e] = fabsf(y);
        nan = nan || y != y;
        inf = inf || fabsf(y) == INFINITY;
        huge = huge || fabsf(y) >= kProjectHuge;
    }
    nan = __syncthreads_or(nan);
    inf = __syncthreads_or(inf);
    huge = __syncthreads_or(huge);
    double tau = nan ? 0.0 : (double)INFINITY;
    if (radius > 0.0 && !nan && !inf) {
        double down = 1.0;
        if (huge) {
            down = (double)kProjectDown;
            for (unsigned e = threadIdx.x; e < n; e += blockDim.x) xs[e] *= kProjectDown;
            __syncthreads();
        }
        tau = block_window(xs, n, 0.0, 0.0, 0.f, 0.f, radius * down, &tau) == 0 ? tau / down : (double)NAN;
    }
    if (radius == 0.0) tau = (double)INFINITY;
    if (threadIdx.x == 0) {
        sh_tau = tau;
        *tau_out = tau;
    }
    __syncthreads();
    tau = sh_tau;
    const float tf = (float)tau;
    const bool on = tau > 0.0;
    for (unsigned e = threadIdx.x; e < n; e += blockDim.x) {
        const float y = x[e];
        out[e] = on ? soft(y, tf) : y;
    }
}

// out = soft(x, tau) for the standalone projection
__global__ void __launch_bounds__(NT) k_apply_flat(const float* x, float* out, long long n, const Scal* sc) {
    const double tau = sc->ctl[0].tau;
    const float tf = (float)tau;
    const bool on = tau > 0.0;
    long long done = 0;
    if (!((reinterpret_cast<unsigned long long>(x) | reinterpret_cast<unsigned long long>(out)) & 15ull)) {
        const float4* x4 = reinterpret_cast<const float4*>(x);
        float4* o4 = reinterpret_cast<float4*>(out);
        const long long quads = n >> 2;
        done = quads << 2;
        for (long long l = blockIdx.x * (long long)NT + threadIdx.x; l < quads; l += (long long)gridDim.x * NT) {
            float4 q = x4[l];
            if (on) q = make_float4(soft(q.x, tf), soft(q.y, tf), soft(q.z, tf), soft(q.w, tf));
            o4[l] = q;
        }
    }
    for (long long l = done + blockIdx.x * (long long)NT + threadIdx.x; l < n; l += (long long)gridDim.x * NT)
        out[l] = on ? soft(x[l], tf) : x[l];
}

// ---------------------------------------------------------------------------
// layout conversion: (ncubes, n3, n1, *) arrays between pitches and types
// ---------------------------------------------------------------------------
// Cube by cube, 32 x 8 threads: a warp takes 32 columns of one row, blocks in
// y walk the rows (no division per element).
template <typename S, typename D>
__global__ void __launch_bounds__(256) k_convert(const S* src, long long src_pitch, long long src_cube, D* dst,
                                                 long long dst_pitch, long long dst_cube, int n1, int n2, int n3,
                                                 int ncubes, const double* scale) {
    const float f = scale ? (float)(1.0 - *scale) : 1.f;
    const long long rows = (long long)n3 * n1;
    for (int cb = 0; cb < ncubes; ++cb) {
        for (long long row = blockIdx.y * 8ll + threadIdx.y; row < rows; row += gridDim.y * 8ll) {
            const S* s = src + cb * src_cube + row * src_pitch;
            D* d = dst + cb * dst_cube + row * dst_pitch;
            for (int j = blockIdx.x * 32 + threadIdx.x; j < n2; j += gridDim.x * 32) {
                const float x = ldT(s + j);
                stT(d + j, scale ? f * x : x);
            }
        }
    }
}

// The same for float32 rows whose pitches, width and bases are multiples of
// four floats: one float4 per thread and row (more bytes in flight).
__global__ void __launch_bounds__(256) k_convert4(const float4* src, long long src_pitch, long long src_cube,
                                                  float4* dst, long long dst_pitch, long long dst_cube,
                                                  long long rows, int w4, int ncubes, const double* scale) {
    const float f = scale ? (float)(1.0 - *scale) : 1.f;
    for (int cb = 0; cb < ncubes; ++cb) {
        for (long long row = blockIdx.y * 8ll + threadIdx.y; row < rows; row += gridDim.y * 8ll) {
            const float4* s = src + cb * src_cube + row * src_pitch;
            float4* d = dst + cb * dst_cube + row * dst_pitch;
            for (int j = blockIdx.x * 32 + threadIdx.x; j < w4; j += gridDim.x * 32) {
                float4 x = __ldg(s + j);
                if (scale) { x.x *= f; x.y *= f; x.z *= f; x.w *= f; }
                d[j] = x;
            }
        }
    }
}

// All 21 float32 cubes of a state in one launch (grid z = cube), float4 rows;
// the last cube (q) is scaled by 1 - c into y4.
struct CubeCopy4 {
    const float4* src;
    float4* dst;
    int scaled;
};
struct StateCopy4 {
    CubeCopy4 c[21];
    long long rows, src_pitch, dst_pitch;   // pitches in float4
    int w4;
    const double* scale;
};

__global__ void __launch_bounds__(256) k_unpack_state4(const StateCopy4 a) {
    const CubeCopy4 cc = a.c[blockIdx.z];
    const float f = cc.scaled ? (float)(1.0 - *a.scale) : 1.f;
    for (long long row = blockIdx.y * 8ll + threadIdx.y; row < a.rows; row += gridDim.y * 8ll) {
        const float4* s = cc.src + row * a.src_pitch;
        float4* d = cc.dst + row * a.dst_pitch;
        for (int j = blockIdx.x * 32 + threadIdx.x; j < a.w4; j += gridDim.x * 32) {
            float4 x = __ldg(s + j);
            if (cc.scaled) { x.x *= f; x.y *= f; x.z *= f; x.w *= f; }
            d[j] = x;
        }
    }
}

int grid_for(long long n) {
    long long b = (n + NT - 1) / NT;
    return (int)std::max(1ll, std::min(b, device_sms() * 16ll));
}

// voxels a part's launch visits
long long part_voxels(const Geom& g, const SlabPart& sp) {
    return (long long)(sp.o1 - sp.o0) * g.n1 * g.n2;
}

// CTAs of K2 that fit the GPU at once (its launch bounds), beside the one that
// places the windows
int k2_resident() { return 3 * device_sms() - 1; }

int k2_grid_part(bool strips, const Geom& g, const SlabPart& sp) {
    const long long nb = sp.o1 - sp.o0;
    if (strips) return grid_for(nb * ((g.n1 + K2_ROWS - 1) / K2_ROWS) * (g.p2 / 4));
    const long long ctas = (nb * g.n1 * (g.p2 / 4) + NT - 1) / NT;
    return (int)std::max(1ll, std::min<long long>(ctas, k2_resident()));
}

int radix_grid_n(long long n) {
    // enough CTAs that none sees more than 2^21 values (the shared bins are 32-bit)
    const long long min_ctas = (n + (1ll << 21) - 1) >> 21;
    return (int)std::max<long long>(std::min(grid_for(n), device_sms() * 3), min_ctas);
}

int gather_grid_n(long long n) { return std::min(grid_for(n), device_sms() * 4); }

template <typename T>
int launch_k2_t(const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc, double* part,
                int part_cap, const SlabPart& sp, cudaStream_t st) {
    K2Args<T> a;
    a.g = g;
    a.u = (const T*)b.u; a.u_n = (const T*)b.u_n; a.s = (const T*)b.s; a.t = (const T*)b.t;
    a.y3 = (const T*)b.y3; a.q = (const T*)b.q; a.v = b.v;
    a.s_n = (T*)b.s_n; a.t_n = (T*)b.t_n; a.y3_n = (T*)b.y3_n; a.q_n = (T*)b.q_n;
    a.p = p;
    a.sc = sc;
    a.part = part;
    a.sp = sp;
    a.windows = sp.cta_total == 0 ? 1 : 0;                 // (a slab's windows are placed by the finish)
    constexpr bool f32 = std::is_same<T, float>::value;
    const bool strips = !f32 || p.fixed_sums;
    const int ctas = std::min(k2_grid_part(strips, g, sp), part_cap) + a.windows;
    if (strips) k2_light<T, true><<<ctas, NT, 0, st>>>(a);
    else if constexpr (f32) k2_light<T, false><<<ctas, NT, 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template <typename Src>
int launch_radix_src(const Src& src, long long n, const SearchArgs& a, int level, cudaStream_t st) {
    const size_t smem = 6 * kHistBins * sizeof(unsigned);
    k_radix<Src><<<radix_grid_n(n), NT, smem, st>>>(src, a, level);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template <typename T>
CubeSrc<T> make_cube_src(const Geom& g, const IterBufs& b, const IterParams& p, const Scal* sc,
                         const SlabPart& sp) {
    CubeSrc<T> c;
    c.g = g;
    c.s = (const T*)b.s; c.t = (const T*)b.t; c.y3 = (const T*)b.y3; c.q = (const T*)b.q;
    c.sc = sc;
    c.parity = p.parity;
    c.gs = p.gamma_s;
    c.gt = p.gamma_t;
    c.o0 = sp.o0;
    c.nb = sp.o1 - sp.o0;
    return c;
}

SearchArgs cube_args(Scal* sc, const L1Work& w, const SlabPart& sp) {
    SearchArgs a{sc, w, 2};
    a.cta_base = sp.cta_base;
    a.cta_total = sp.cta_total;
    return a;
}

template <typename T>
int launch_fallback_t(int level, const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc,
                      const L1Work& w, const SlabPart& sp, cudaStream_t st) {
    const CubeSrc<T> src = make_cube_src<T>(g, b, p, sc, sp);
    return launch_radix_src(src, part_voxels(g, sp), cube_args(sc, w, sp), level, st);
}

template <typename T>
int launch_gather_t(const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc, const L1Work& w,
                    const SlabPart& sp, cudaStream_t st) {
    const CubeSrc<T> src = make_cube_src<T>(g, b, p, sc, sp);
    k_gather<CubeSrc<T>><<<gather_grid_n(part_voxels(g, sp)), NT, 0, st>>>(src, cube_args(sc, w, sp));
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int window_grid_n(long long n, int part_cap) {
    return std::max(1, std::min({grid_for(n), device_sms() * 4, part_cap}));
}

template <typename T>
int launch_window_t(const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc, const L1Work& w,
                    int part_cap, const SlabPart& sp, cudaStream_t st) {
    const CubeSrc<T> src = make_cube_src<T>(g, b, p, sc, sp);
    const int grid = window_grid_n(part_voxels(g, sp), part_cap);
    k_window<CubeSrc<T>><<<grid, NT, 0, st>>>(src, cube_args(sc, w, sp), w.k1_n, w.k1_s);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// the shape of a cube's search launch.  win_ctas: 256-thread CTAs that the retry
// pass is split by; a radix item sees at most 2^21 values (its shared bins are
// 32-bit).
SearchShape search_shape(long long voxels, int win_ctas, int parts, int count, int ctas) {
    SearchShape h;
    h.parts = parts;
    h.win_threads = 256u * (unsigned)win_ctas;
    h.win_items = (win_ctas * 256 + kFinishThreads - 1) / kFinishThreads;
    h.pass_items = (int)std::max<long long>(ctas, (voxels + (1ll << 21) - 1) >> 21);
    h.count = count;
    return h;
}

template <typename T>
int launch_search_t(const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc, const L1Work& w, int part_cap,
                    int parts, int count, cudaStream_t st) {
    const SlabPart whole = whole_cube(g);
    const CubeSrc<T> src = make_cube_src<T>(g, b, p, sc, whole);
    const int win = window_grid_n(part_voxels(g, whole), part_cap);
    const int ctas = std::max(2, (win * 256 + kFinishThreads - 1) / kFinishThreads);
    const SearchShape h = search_shape(part_voxels(g, whole), win, parts, count, ctas);
    k_search<CubeSrc<T>><<<ctas, kFinishThreads, kFinishSmem, st>>>(src, cube_args(sc, w, whole), w.k1_n, w.k1_s, h);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

template <typename S, typename D>
int launch_convert(const S* src, long long sp, long long sc_, D* dst, long long dp, long long dc,
                   const Geom& g, int ncubes, const double* scale, cudaStream_t st) {
    const long long rows = (long long)g.n3 * g.n1;
    if constexpr (std::is_same<S, float>::value && std::is_same<D, float>::value) {
        const bool a16 = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0;
        if (a16 && sp % 4 == 0 && dp % 4 == 0 && sc_ % 4 == 0 && dc % 4 == 0 && g.n2 % 4 == 0) {
            const int w4 = g.n2 / 4;
            const int gx = std::min((w4 + 31) / 32, 64);
            const long long gy = std::max(1ll, std::min({(rows + 7) / 8, (device_sms() * 16ll) / gx, 65535ll}));
            k_convert4<<<dim3(gx, (unsigned)gy), dim3(32, 8), 0, st>>>(
                reinterpret_cast<const float4*>(src), sp / 4, sc_ / 4, reinterpret_cast<float4*>(dst), dp / 4,
                dc / 4, rows, w4, ncubes, scale);
            return cudaGetLastError() == cudaSuccess ? 0 : -3;
        }
    }
    const int gx = std::min((g.n2 + 31) / 32, 64);
    const long long gy = std::max(1ll, std::min({(rows + 7) / 8, (device_sms() * 16ll) / gx, 65535ll}));
    k_convert<S, D><<<dim3(gx, (unsigned)gy), dim3(32, 8), 0, st>>>(src, sp, sc_, dst, dp, dc, g.n1, g.n2, g.n3,
                                                                    ncubes, scale);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// ---------------------------------------------------------------------------
// batches: one launch of a stage for many cubes (float32 storage)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int batch_cube_of(const int* start, int n, int blk) {
    int lo = 0, hi = n - 1;                 // the last cube whose first CTA is <= blk
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= blk) lo = mid; else hi = mid - 1;
    }
    return lo;
}

struct SearchCube {
    CubeSrc<float> src;
    SearchArgs a;
    unsigned long long* pn;
    double* ps;
    SearchShape h;
};
struct SearchBatchTab {
    int n;
    int start[kBatchMax + 1];
    SearchCube c[kBatchMax];
};
struct K2BatchTab {
    int n;
    int start[kBatchMax + 1];
    K2Args<float> c[kBatchMax];
};

// The search of every cube of a batch.  The first CTAs are two per cube, its
// window's finishes; the rest help the cubes that start[] gives them to.
__global__ void __launch_bounds__(kFinishThreads) k_search_batch(const __grid_constant__ SearchBatchTab t) {
    const int k = (int)blockIdx.x - 2 * t.n;
    const int c = k < 0 ? (int)blockIdx.x >> 1 : batch_cube_of(t.start, t.n, k);
    const SearchCube& q = t.c[c];
    if (__ldcg(&q.a.sc->done)) return;
    search_body(q.src, q.a, q.pn, q.ps, q.h, k < 0 ? (int)blockIdx.x & 1 : 2);
}
__global__ void __launch_bounds__(NT, 3) k2_batch(const __grid_constant__ K2BatchTab t) {
    const int c = batch_cube_of(t.start, t.n, blockIdx.x);
    // the cube's arguments in shared memory: by value they did not fit the
    // registers beside an item's eleven quads (28 bytes spilled)
    __shared__ __align__(16) unsigned words[sizeof(K2Args<float>) / 4];
    const K2Args<float>& a = *reinterpret_cast<const K2Args<float>*>(words);
    static_assert(sizeof(K2Args<float>) % 4 == 0, "copied in words");
    for (unsigned k = threadIdx.x; k < sizeof(words) / 4; k += NT)
        words[k] = reinterpret_cast<const unsigned*>(&t.c[c])[k];
    __syncthreads();
    if (__ldcg(&a.sc->done)) return;
    k2_body(a, (int)blockIdx.x - t.start[c] - 1, t.start[c + 1] - t.start[c] - 1);
}

}  // namespace

int device_sms() {
    constexpr int kMaxDev = 64;
    constexpr int kFallback = 152;     // GB300, if the query fails
    static std::once_flag once[kMaxDev];
    static int sms[kMaxDev];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        return kFallback;
    }
    std::call_once(once[dev], [dev] {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
            cudaGetLastError();
            n = kFallback;
        }
        sms[dev] = n;
    });
    return sms[dev];
}

int light_configure(int storage) {
    const int smem = 6 * kHistBins * sizeof(unsigned);
    cudaError_t e = cudaErrorInvalidValue;
    switch (storage) {
        case 0: e = cudaFuncSetAttribute(k_radix<CubeSrc<float>>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
        case 1: e = cudaFuncSetAttribute(k_radix<CubeSrc<__nv_bfloat16>>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
        case 2: e = cudaFuncSetAttribute(k_radix<CubeSrc<__half>>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem); break;
    }
    if (e != cudaSuccess) return -3;
    e = cudaFuncSetAttribute(k_radix<FlatSrc>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return -3;
    switch (storage) {
        case 0: e = cudaFuncSetAttribute(k_search<CubeSrc<float>>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinishSmem); break;
        case 1: e = cudaFuncSetAttribute(k_search<CubeSrc<__nv_bfloat16>>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinishSmem); break;
        case 2: e = cudaFuncSetAttribute(k_search<CubeSrc<__half>>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinishSmem); break;
    }
    if (e != cudaSuccess) return -3;
    e = cudaFuncSetAttribute(k_search_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinishSmem);
    return e == cudaSuccess ? 0 : -3;
}

int launch_search(int storage, const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc, const L1Work& w,
                  int part_cap, int parts, int count, cudaStream_t st) {
    switch (storage) {
        case 0: return launch_search_t<float>(g, b, p, sc, w, part_cap, parts, count, st);
        case 1: return launch_search_t<__nv_bfloat16>(g, b, p, sc, w, part_cap, parts, count, st);
        case 2: return launch_search_t<__half>(g, b, p, sc, w, part_cap, parts, count, st);
    }
    return -1;
}

int launch_search_finish(int mode, Scal* sc, const L1Work& w, int nvec, const unsigned long long* pn,
                         const double* ps, int parts, cudaStream_t st, int gated,
                         cudaGraphConditionalHandle cond) {
    SearchArgs a{sc, w, nvec};
    k_search_finish<<<nvec, kFinishThreads, kFinishSmem, st>>>(a, mode, pn, ps, parts, gated, cond);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

// (the partials of a float32 cube serve both of its grids)
int k2_grid_ctas(int storage, const Geom& g) {
    const int strips = k2_grid_part(true, g, whole_cube(g));
    return storage != 0 ? strips : std::max(strips, k2_grid_part(false, g, whole_cube(g)));
}

int window_grid(const Geom& g, const SlabPart& sp, int part_cap) {
    return window_grid_n(part_voxels(g, sp), part_cap);
}
int radix_grid(const Geom& g, const SlabPart& sp) { return radix_grid_n(part_voxels(g, sp)); }
int gather_grid(const Geom& g, const SlabPart& sp) { return gather_grid_n(part_voxels(g, sp)); }
int k2_grid(const Geom& g, const SlabPart& sp, int part_cap) { return std::min(k2_grid_part(false, g, sp), part_cap); }

int launch_k2(int storage, const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc,
              double* part, int part_cap, const SlabPart& sp, cudaStream_t st) {
    switch (storage) {
        case 0: return launch_k2_t<float>(g, b, p, sc, part, part_cap, sp, st);
        case 1: return launch_k2_t<__nv_bfloat16>(g, b, p, sc, part, part_cap, sp, st);
        case 2: return launch_k2_t<__half>(g, b, p, sc, part, part_cap, sp, st);
    }
    return -1;
}


int launch_fallback(int storage, int level, const Geom& g, const IterBufs& b, const IterParams& p,
                    Scal* sc, const L1Work& w, const SlabPart& sp, cudaStream_t st) {
    switch (storage) {
        case 0: return launch_fallback_t<float>(level, g, b, p, sc, w, sp, st);
        case 1: return launch_fallback_t<__nv_bfloat16>(level, g, b, p, sc, w, sp, st);
        case 2: return launch_fallback_t<__half>(level, g, b, p, sc, w, sp, st);
    }
    return -1;
}

int launch_gather(int storage, const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc,
                  const L1Work& w, const SlabPart& sp, cudaStream_t st) {
    switch (storage) {
        case 0: return launch_gather_t<float>(g, b, p, sc, w, sp, st);
        case 1: return launch_gather_t<__nv_bfloat16>(g, b, p, sc, w, sp, st);
        case 2: return launch_gather_t<__half>(g, b, p, sc, w, sp, st);
    }
    return -1;
}

int launch_window(int storage, const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc,
                  const L1Work& w, int part_cap, const SlabPart& sp, cudaStream_t st) {
    switch (storage) {
        case 0: return launch_window_t<float>(g, b, p, sc, w, part_cap, sp, st);
        case 1: return launch_window_t<__nv_bfloat16>(g, b, p, sc, w, part_cap, sp, st);
        case 2: return launch_window_t<__half>(g, b, p, sc, w, part_cap, sp, st);
    }
    return -1;
}

// Whether a vector still needs a threshold search after the cooperative K1, which
// finishes its window itself: sets the condition of the graph node that holds the
// search launches.
__global__ void k_search_gate(Scal* sc, cudaGraphConditionalHandle cond) {
    if (threadIdx.x != 0) return;
    const unsigned need = scal_needs_search(sc) ? 1u : 0u;
    if (need) sc->gate_opens++;
    cudaGraphSetConditional(cond, need);
}

int launch_search_gate(Scal* sc, cudaGraphConditionalHandle cond, cudaStream_t st) {
    k_search_gate<<<1, 32, 0, st>>>(sc, cond);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

constexpr double kHelperVoxels = 32768;        // fewer are not worth a CTA's start
int launch_search_batch(const BatchCube* cubes, int n, cudaStream_t st) {
    if (n < 1 || n > kBatchMax) return -1;
    static_assert(sizeof(SearchBatchTab) <= 32000, "kernel parameter space");
    SearchBatchTab t{};
    t.n = n;
    double all = 0.0;
    for (int c = 0; c < n; ++c) all += (double)cubes[c].g.cube;
    // Helpers in proportion to the cubes, three times the SMs in all: they follow the
    // other cubes' CTAs on the SMs as those end.  (With one CTA per SM in all, the
    // finishes of 64 cubes left 24 to help: the first 32 passes of 64 cubes of 0.05 to
    // 59 million voxels took 7.9 ms each in the search, 1.5 with twice the SMs, 1.3
    // with three times, 1.2 with four; of 8 such cubes 0.265, 0.230, 0.223, 0.244.)
    const double helpers = 3.0 * device_sms();
    int total = 0;
    for (int c = 0; c < n; ++c) {
        const BatchCube& q = cubes[c];
        const SlabPart whole = whole_cube(q.g);
        const long long vox = part_voxels(q.g, whole);
        SearchCube& e = t.c[c];
        e.src = make_cube_src<float>(q.g, q.b, q.p, q.sc, whole);
        e.a = cube_args(q.sc, q.l1, whole);
        e.pn = q.l1.k1_n;
        e.ps = q.l1.k1_s;
        t.start[c] = total;
        const int share = (int)std::min(helpers * ((double)q.g.cube / all), 1.0 + (double)vox / kHelperVoxels);
        e.h = search_shape(vox, window_grid_n(vox, q.k1_ctas), q.k1.ctas, 1, 2 + share);
        total += share;
    }
    t.start[n] = total;
    k_search_batch<<<2 * n + total, kFinishThreads, kFinishSmem, st>>>(t);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_k2_batch(const BatchCube* cubes, int n, cudaStream_t st) {
    if (n < 1 || n > kBatchMax) return -1;
    static_assert(sizeof(K2BatchTab) <= 32000, "kernel parameter space");
    K2BatchTab t{};
    t.n = n;
    int total = 0;
    // CTAs shared out by size (each cube at least one): up to eight times as many as
    // fit the GPU, as long as a thread has about five quads.  With those that fit it
    // once, rounded up per cube, a few ran a whole CTA's time after the rest (64 cubes
    // of 0.05 to 59 million voxels: once 3.13, twice 2.81, four times 2.57, eight
    // 2.47, sixteen 2.42 ms; 16 of 0.29 million: 47, 41, 47, 63, 71 us).
    double all = 0.0;
    for (int c = 0; c < n; ++c) all += (double)cubes[c].g.cube;
    const double waves = std::min(8.0, std::max(1.0, all / (20.0 * NT * k2_resident())));
    for (int c = 0; c < n; ++c) {
        const BatchCube& q = cubes[c];
        K2Args<float>& a = t.c[c];
        a.g = q.g;
        a.u = (const float*)q.b.u; a.u_n = (const float*)q.b.u_n; a.s = (const float*)q.b.s;
        a.t = (const float*)q.b.t; a.y3 = (const float*)q.b.y3; a.q = (const float*)q.b.q; a.v = q.b.v;
        a.s_n = (float*)q.b.s_n; a.t_n = (float*)q.b.t_n; a.y3_n = (float*)q.b.y3_n; a.q_n = (float*)q.b.q_n;
        a.p = q.p;
        a.sc = q.sc;
        a.part = q.k2_part;
        a.sp = whole_cube(q.g);
        t.start[c] = total;
        const int share = (int)std::ceil(waves * k2_resident() * ((double)q.g.cube / all));
        a.windows = 1;
        total += std::max(1, std::min({share, k2_grid_part(false, q.g, a.sp), q.k2_cap})) + 1;
    }
    t.start[n] = total;
    k2_batch<<<total, NT, 0, st>>>(t);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int k1_batch_configure();

int batch_configure() {
    if (k1_batch_configure() != 0) return -3;
    const cudaError_t e = cudaFuncSetAttribute(k_search_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFinishSmem);
    return e == cudaSuccess ? 0 : -3;
}

int launch_copy_f32(const float* src, long long src_pitch, long long src_cube, float* dst, long long dst_pitch,
                    long long dst_cube, int n1, int n2, int nbands, int ncubes, const double* scale,
                    cudaStream_t st) {
    if (nbands <= 0 || ncubes <= 0) return 0;
    Geom g{};
    g.n1 = n1; g.n2 = n2; g.n3 = nbands;
    return launch_convert(src, src_pitch, src_cube, dst, dst_pitch, dst_cube, g, ncubes, scale, st);
}

// dense float32 (ncubes, n3, n1, n2)  ->  pitched storage cubes
int launch_pack(int storage, const float* src, void* dst, const Geom& g, int ncubes, cudaStream_t st) {
    const long long sp = g.n2, scb = (long long)g.n3 * g.n1 * g.n2;
    switch (storage) {
        case 0: return launch_convert(src, sp, scb, (float*)dst, g.p2, g.cube, g, ncubes, nullptr, st);
        case 1: return launch_convert(src, sp, scb, (__nv_bfloat16*)dst, g.p2, g.cube, g, ncubes, nullptr, st);
        case 2: return launch_convert(src, sp, scb, (__half*)dst, g.p2, g.cube, g, ncubes, nullptr, st);
    }
    return -1;
}

// pitched float32 (the handle's v)  ->  pitched storage cube
int launch_pitched_to_storage(int storage, const float* src, void* dst, const Geom& g, cudaStream_t st) {
    switch (storage) {
        case 0: return launch_convert(src, g.p2, g.cube, (float*)dst, g.p2, g.cube, g, 1, nullptr, st);
        case 1: return launch_convert(src, g.p2, g.cube, (__nv_bfloat16*)dst, g.p2, g.cube, g, 1, nullptr, st);
        case 2: return launch_convert(src, g.p2, g.cube, (__half*)dst, g.p2, g.cube, g, 1, nullptr, st);
    }
    return -1;
}

// dense float32 (n3, n1, n2)  ->  pitched float32
int launch_dense_to_pitched(const float* src, float* dst, const Geom& g, cudaStream_t st) {
    return launch_convert(src, (long long)g.n2, (long long)g.n3 * g.n1 * g.n2, dst, g.p2, g.cube, g, 1,
                          nullptr, st);
}

int launch_unpack(int storage, const void* src, float* dst, const Geom& g, int ncubes, cudaStream_t st) {
    const long long dp = g.n2, dcb = (long long)g.n3 * g.n1 * g.n2;
    switch (storage) {
        case 0: return launch_convert((const float*)src, g.p2, g.cube, dst, dp, dcb, g, ncubes, nullptr, st);
        case 1: return launch_convert((const __nv_bfloat16*)src, g.p2, g.cube, dst, dp, dcb, g, ncubes, nullptr, st);
        case 2: return launch_convert((const __half*)src, g.p2, g.cube, dst, dp, dcb, g, ncubes, nullptr, st);
    }
    return -1;
}

int launch_unpack_state(int storage, const void* const src[9], float* const dst[9], const double* c,
                        const Geom& g, cudaStream_t st) {
    static const int ncubes[9] = {1, 1, 1, 6, 6, 2, 2, 1, 1};
    if (storage != 0 || g.n2 % 4 != 0) return 1;
    StateCopy4 a;
    const long long dense = (long long)g.n3 * g.n1 * g.n2;
    int k = 0;
    for (int f = 0; f < 9; ++f) {
        if (((reinterpret_cast<uintptr_t>(src[f]) | reinterpret_cast<uintptr_t>(dst[f])) & 15) != 0) return 1;
        for (int cb = 0; cb < ncubes[f]; ++cb, ++k) {
            a.c[k].src = reinterpret_cast<const float4*>(static_cast<const float*>(src[f]) + cb * g.cube);
            a.c[k].dst = reinterpret_cast<float4*>(dst[f] + cb * dense);
            a.c[k].scaled = f == 8;
        }
    }
    a.rows = (long long)g.n3 * g.n1;
    a.src_pitch = g.p2 / 4;
    a.dst_pitch = g.n2 / 4;
    a.w4 = g.n2 / 4;
    a.scale = c;
    const int gx = std::min((a.w4 + 31) / 32, 64);
    const long long gy = std::max(1ll, std::min({(a.rows + 7) / 8, (device_sms() * 16ll) / (gx * 21ll), 65535ll}));
    k_unpack_state4<<<dim3(gx, (unsigned)gy, 21), dim3(32, 8), 0, st>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int launch_scale_unpack(int storage, const void* q, const double* c, float* dst, const Geom& g,
                        cudaStream_t st) {
    const long long dp = g.n2, dcb = (long long)g.n3 * g.n1 * g.n2;
    switch (storage) {
        case 0: return launch_convert((const float*)q, g.p2, g.cube, dst, dp, dcb, g, 1, c, st);
        case 1: return launch_convert((const __nv_bfloat16*)q, g.p2, g.cube, dst, dp, dcb, g, 1, c, st);
        case 2: return launch_convert((const __half*)q, g.p2, g.cube, dst, dp, dcb, g, 1, c, st);
    }
    return -1;
}

// ---------------------------------------------------------------------------
// standalone projection of a flat device vector onto an l1 ball
// ---------------------------------------------------------------------------
// Scratch of the standalone projection: stream-ordered, from a memory pool of the
// library's own on each device that keeps at most 8 MB between calls (a pair of
// cudaMalloc and cudaFree took 0.15 ms of every call).  Without a pool, cudaMalloc.
struct PoolScratch {
    void* p = nullptr;
    cudaStream_t st;
    bool pooled = false;
    explicit PoolScratch(cudaStream_t s) : st(s) {}
    static cudaMemPool_t pool() {
        constexpr int kMaxDev = 64;
        static std::once_flag once[kMaxDev];
        static cudaMemPool_t pools[kMaxDev];
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return nullptr;
        std::call_once(once[dev], [dev] {
            cudaMemPoolProps props{};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t q = nullptr;
            unsigned long long keep = 8ull << 20;
            if (cudaMemPoolCreate(&q, &props) != cudaSuccess ||
                cudaMemPoolSetAttribute(q, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
                if (q) cudaMemPoolDestroy(q);
                q = nullptr;
                cudaGetLastError();
            }
            pools[dev] = q;
        });
        return pools[dev];
    }
    bool get(size_t bytes) {
        const cudaMemPool_t q = pool();
        if (q) {
            if (cudaMallocFromPoolAsync(&p, bytes, q, st) == cudaSuccess) {
                pooled = true;
                return true;
            }
            cudaGetLastError();
        }
        if (cudaMalloc(&p, bytes) == cudaSuccess) return true;
        cudaGetLastError();
        p = nullptr;
        return false;
    }
    ~PoolScratch() {
        if (!p) return;
        if (pooled) cudaFreeAsync(p, st);
        else cudaFree(p);
    }
};

// Vectors from this length on are searched by a sample and one pass.
constexpr long long kSampleFrom = 1ll << 21;

// One allocation holds the scratch.  A vector of at most kSmallProject values is
// one CTA's; a short one is searched by the radix
// stages of one launch; a long one by those stages on a sample of 1/32, which
// place the window of one pass over all values (58.7 M values: a call with three
// radix passes and a gather over all of them took 1290 us, now 544: sample 89,
// pass 168, output 66 us, and 484 with pooled scratch; 4096 values in seven
// launches and four allocations 357
// us, now 52).
int l1_project_standalone(const float* x, long long n, double radius, float* out, double* tau,
                          cudaStream_t st) {
    PoolScratch scr(st);
    if (n <= (long long)kSmallProject) {
        double t = 0.0;
        if (!scr.get(sizeof(double))) return -2;
        k_project_small<<<1, 1024, 0, st>>>(x, out, (unsigned)n, radius, (double*)scr.p);
        const bool ok = cudaGetLastError() == cudaSuccess &&
                        cudaMemcpyAsync(&t, scr.p, sizeof(t), cudaMemcpyDeviceToHost, st) == cudaSuccess;
        if (cudaStreamSynchronize(st) != cudaSuccess || !ok) return -3;
        if (std::isnan(t)) return -6;
        if (tau) *tau = t;
        return 0;
    }
    const bool sampled = n >= kSampleFrom && radius > 0.0;
    if (cudaFuncSetAttribute(k_search<FlatSrc>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinishSmem) != cudaSuccess ||
        cudaFuncSetAttribute(k_search<SampleSrc>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFinishSmem) != cudaSuccess)
        return -3;
    const size_t parts = 4 * (size_t)device_sms(), b_hist = 2 * kHistBins * sizeof(unsigned long long);
    // (a gathered bracket holds at most kGatherMax values, a window kCandCap)
    const size_t b_cand = (sampled ? (size_t)kCandCap : (size_t)kGatherMax) * sizeof(float);
    const size_t b_nh = 6 * kNarrowBins * sizeof(unsigned);
    size_t off = 0;
    auto take = [&](size_t b) { const size_t o = off; off += (b + 255) / 256 * 256; return o; };
    const size_t o_sc = take(sizeof(Scal)), o_cnt = take(b_hist), o_res = take(b_hist), o_nh = take(b_nh),
                 o_nb = take(2 * sizeof(unsigned)), o_zero = off, o_pn = take(parts * 8), o_ps = take(parts * 8),
                 o_cand = take(b_cand);
    if (!scr.get(off)) return -2;
    char* mem = (char*)scr.p;
    Scal* sc = reinterpret_cast<Scal*>(mem + o_sc);
    L1Work w{};
    w.hcnt = reinterpret_cast<unsigned long long*>(mem + o_cnt);
    w.hres = reinterpret_cast<unsigned long long*>(mem + o_res);
    w.nh = reinterpret_cast<unsigned*>(mem + o_nh);
    w.nbinned = reinterpret_cast<unsigned*>(mem + o_nb);
    w.cand[0] = w.cand[1] = reinterpret_cast<float*>(mem + o_cand);
    unsigned long long* pn = reinterpret_cast<unsigned long long*>(mem + o_pn);
    double* ps = reinterpret_cast<double*>(mem + o_ps);
    const SearchArgs a{sc, w, 1};
    auto search = [&](const auto& src, long long cnt) {
        const int win = window_grid_n(cnt, 4 * device_sms());
        const int ctas = (win * 256 + kFinishThreads - 1) / kFinishThreads;
        k_search<<<ctas, kFinishThreads, kFinishSmem, st>>>(src, a, pn, ps, search_shape(cnt, win, -1, 0, ctas));
    };
    int rc = 0;
    Scal h{};
    const long long ns = (n >> 10) << 5;
    const double scale = sampled ? (double)n / (double)ns : 1.0;
    h.radius[0] = radius / scale;
    h.ctl[0].need = radius > 0.0 ? NEED_RADIX0 : NEED_NONE;
    h.ctl[0].tau = radius > 0.0 ? 0.0 : (double)INFINITY;
    h.search.stage = ST_RADIX0;
    if (cudaMemsetAsync(mem, 0, o_zero, st) != cudaSuccess ||
        cudaMemcpyAsync(sc, &h, sizeof(Scal), cudaMemcpyHostToDevice, st) != cudaSuccess)
        rc = -3;
    if (rc == 0) {
        if (sampled) {
            search(SampleSrc{x, ns}, ns);
            k_flat_window<<<1, 32, 0, st>>>(sc, radius, scale);
        }
        if (radius > 0.0) search(FlatSrc{x, n}, n);
        k_apply_flat<<<grid_for(n), NT, 0, st>>>(x, out, n, sc);
        if (cudaGetLastError() != cudaSuccess) rc = -3;
    }
    if (rc == 0) {
        if (cudaMemcpyAsync(&h, sc, sizeof(Scal), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            rc = -3;
        else if (h.error) rc = -6;
        else if (tau) *tau = h.ctl[0].tau;
    }
    cudaStreamSynchronize(st);
    return rc;
}

}  // namespace gsstv

// ---------------------------------------------------------------------------
// Allocation-free l1-ball projection.
//
// Same kernels as gsstv_project_l1ball, but every scratch byte (controller
// block, radix histograms, candidate buffer) lives in one file-scope device
// array instead of cudaMalloc'd memory, for callers that are not allowed to
// allocate device memory.  The candidate buffer here holds
// GSSTV_NOALLOC_MAX_N values; a radix bracket never holds more values than
// the whole input, so every n <= GSSTV_NOALLOC_MAX_N fits, and larger n are
// refused.
// ---------------------------------------------------------------------------
#include <mutex>

#include "gsstv.h"

namespace gsstv {
namespace {

constexpr size_t kNaScal = (sizeof(Scal) + 255) / 256 * 256;
constexpr size_t kNaHist = 2 * kHistBins * sizeof(unsigned long long);
constexpr size_t kNaCand = (size_t)GSSTV_NOALLOC_MAX_N * sizeof(float);
constexpr size_t kNaBytes = kNaScal + 2 * kNaHist + kNaCand;

// The scratch array: on every device that loads this library, until exit.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

constexpr int kMaxDevices = 64;
unsigned char* g_na_ptr[kMaxDevices] = {};     // device address of the array, per device
std::mutex g_na_mutex;

__global__ void k_noalloc_init(Scal* sc, double radius) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        Scal z;
        memset(&z, 0, sizeof(z));
        z.radius[0] = radius;
        z.ctl[0].need = radius > 0.0 ? NEED_RADIX0 : NEED_NONE;
        z.ctl[0].tau = radius > 0.0 ? 0.0 : (double)__int_as_float(0x7f800000);
        *sc = z;
    }
}

// Resolves the array's device address on the current device (first call on
// that device only) and configures the kernels it launches.
int noalloc_setup(unsigned char** base) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -3;
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return -3;
        if (light_configure(0) != 0) return -3;
        g_na_ptr[dev] = (unsigned char*)p;
    }
    *base = g_na_ptr[dev];
    return 0;
}

}  // namespace

int l1_project_noalloc(const float* x, long long n, double radius, float* out, double* tau,
                       cudaStream_t st) {
    unsigned char* base = nullptr;
    if (noalloc_setup(&base) != 0) return -3;
    Scal* sc = reinterpret_cast<Scal*>(base);
    L1Work w{};
    w.hcnt = reinterpret_cast<unsigned long long*>(base + kNaScal);
    w.hres = reinterpret_cast<unsigned long long*>(base + kNaScal + kNaHist);
    w.cand[0] = w.cand[1] = reinterpret_cast<float*>(base + kNaScal + 2 * kNaHist);
    // the previous call's contents stay in the array: clear what must start at zero
    k_noalloc_init<<<1, 32, 0, st>>>(sc, radius);
    if (cudaGetLastError() != cudaSuccess) return -3;
    if (cudaMemsetAsync(w.hcnt, 0, 2 * kNaHist, st) != cudaSuccess) return -3;
    const FlatSrc src{x, n};
    const SearchArgs a{sc, w, 1};
    for (int level = 0; level < 3; ++level)
        if (launch_radix_src(src, n, a, level, st) != 0) return -3;
    k_gather<FlatSrc><<<gather_grid_n(n), NT, 0, st>>>(src, a);
    k_search_finish<<<1, kFinishThreads, kFinishSmem, st>>>(a, 1, nullptr, nullptr, 0, 0, 0);
    k_apply_flat<<<grid_for(n), NT, 0, st>>>(x, out, n, sc);
    if (cudaGetLastError() != cudaSuccess) return -3;
    double t = 0.0;
    int err = 0;
    if (cudaMemcpyAsync(&t, &sc->ctl[0].tau, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&err, &sc->error, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return -3;
    if (err) return -6;
    if (tau) *tau = t;
    return 0;
}

}  // namespace gsstv

extern "C" int gsstv_project_l1ball_noalloc(const float* d_x, int64_t n, double radius, float* d_out,
                                            double* tau_out, void* stream) {
    if (!d_x || !d_out || n < 0 || !(radius >= 0.0) || !std::isfinite(radius)) return GSSTV_ERR_ARG;
    if (n > GSSTV_NOALLOC_MAX_N) return GSSTV_ERR_ARG;
    if (n == 0) { if (tau_out) *tau_out = 0.0; return GSSTV_OK; }
    const int rc = gsstv::l1_project_noalloc(d_x, (long long)n, radius, d_out, tau_out, (cudaStream_t)stream);
    return rc == 0 ? GSSTV_OK : rc == -6 ? GSSTV_ERR_INTERNAL : GSSTV_ERR_CUDA;
}
