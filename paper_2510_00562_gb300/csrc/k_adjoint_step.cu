// One pass of Algorithm 1 transposed, for a single vector-Jacobian product.  The
// derivatives and the array layouts are those of k_adjoint.cu, which transposes
// whole runs in place.
//
// Three launches (four where the dual step runs set by set), nothing
// synchronises the host:
//   SUMS  every global sum of the pass.  The l1 adjoints need S and |A|, sums
//         over s1bar = s+_bar + 2 g4 qbar and t1bar, and
//         qbar = (1 - f) y4+_bar + f (q^ . y4+_bar)/|q| q  (f = eps g4/|q|) is
//         linear in y4+_bar and q with scalars this same pass finds, so the
//         sums of sign(s+) s+_bar, sign(s+) y4+_bar, sign(s+) q (and for t)
//         give S without a pass after the l2 step.  Its last block turns the
//         sums into the scalars the other launches read.
//   CUBE  one voxel at a time: the l2 step, the transposed dual ascents and
//         extrapolations of u, s, t, the box, the l1 adjoints, y4; G_bar and
//         a_t_bar to memory for the next launch.  Reads neighbours only of
//         y1, y2, y3, which it does not write.
//   DUAL  w1, w2 and y1, y2 (and y3): the group-shrink adjoints a_w on a tile
//         and a one-pixel ring in shared memory, then L^T of them onto the
//         duals.  The two sets (w1, y1), (w2, y2) are independent; within a
//         set the ring reads neighbours that other blocks write, so each set's
//         output is never its input (see launch_adjoint_single).
//
// Against the five launches of k_adjoint.cu this moves 91 words a voxel instead
// of 126 (512x256x64, 8.4 M voxels: SUMS 93, CUBE 203, DUAL 393 us, 4.4 TB/s in
// all, against 1085 us).  Without the next rows asked into L2 the three took 120,
// 222 and 451 us.  Runs keep the five launches: their parameter adjoints are FP64
// outputs summed over the passes, and sums split otherwise move them by 1e-7.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "gsstv_adjoint.cuh"

namespace gsstv {
namespace {

// sums of one reverse pass: |q|^2, q . y4_bar, |a_s|_1, |a_t|_1, the sums of
// sign(s+) s+_bar, sign(s+) y4_bar, sign(s+) q, the same for t (with the
// transposed D_v in place), and the sizes of the active sets
enum { QQ = 0, QB, L1S, L1T, SS, SY, SQ, ST, TY4, TQ, NS, NT_, NSUM };
constexpr int kSlots = 16;                        // NSUM padded to a power of two

// device memory of the sums; zero before the first pass, and each pass leaves
// sums and ticket zero for the next
struct AdjScal {
    double sum[kSlots];
    float l2act, fk, qs;          // l2 ball active; eps g4/|q|; (q^ . y4_bar)/|q|
    float in_s, in_t, ks, kt;     // inside the l1 balls; S/|A| of s and t
    unsigned ticket;
};
static_assert(sizeof(AdjScal) <= kAdjScalBytes, "scalars of the reverse pass");

struct AdjArgs {
    Dims d;
    SV x, x1, b1;                 // state k, state k+1, adjoint of state k+1
    SW b;                         // adjoint of state k (written; u, s, t, y3, y4 may be b1's)
    const float* v;
    float* vbar;                  // += adjoint of v
    double* pbar;                 // += adjoints of eps, alpha, beta, omega
    AdjScal* sc;
    float *gbar, *atb;            // temporaries (N each): G_bar, a_t_bar
    int len;                      // DUAL: bands per block
    float g_u, g_w1, g_w2, g_s, g_t, g1, g2, g3, g4, th1, th2, mu_lo, mu_hi;
    double eps, alpha, beta, g4d, g_w1d;
};

// Float partial sums over a thread's voxels, moved into float pairs every 32
// terms: float alone drifts over hundreds of terms, and FP64 issue is scarce on
// this part.  A thread whose sums come near what a block's float pairs can hold
// (kSpill: twice it from each of at most 2^9 threads is still a float) adds them to
// the block's doubles `big` instead, so that the range is FP64's.
constexpr float kSpill = 0x1p116f;
template <int K>
struct Partial {
    float f[K], hi[K], lo[K];
    int n;
    double* big;                  // K sums of the block, in shared memory
    __device__ __forceinline__ explicit Partial(double* b) : n(0), big(b) {
#pragma unroll
        for (int k = 0; k < K; ++k) f[k] = hi[k] = lo[k] = 0.f;
    }
    __device__ __forceinline__ void step() {
        if (++n == 32) flush();
    }
    // the float sums into the pairs at once
    __device__ __forceinline__ void fold() {
#pragma unroll
        for (int k = 0; k < K; ++k) { pair_add(hi[k], lo[k], f[k], 0.f); f[k] = 0.f; }
    }
    __device__ __forceinline__ void flush() {
        float top = 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k) top = fmaxf(top, fmaxf(fabsf(hi[k]), fabsf(f[k])));
        if (top > kSpill) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                atomicAdd(big + k, ((double)hi[k] + (double)lo[k]) + (double)f[k]);
                hi[k] = lo[k] = f[k] = 0.f;
            }
        }
        fold();
        n = 0;
    }
};

// q = y4 + g4 (u' + s' + t') - g4 v at voxel l = (b, i, j)
__device__ __forceinline__ float q_at(const AdjArgs& a, long long l, int b, int i, int j) {
    const float up = 2.f * rd(a.x1.u, l) - rd(a.x.u, l), sp = 2.f * rd(a.x1.s, l) - rd(a.x.s, l),
                tp = 2.f * rd(a.x1.t, l) - rd(a.x.t, l);
    const float v = rd(a.v, ((long long)b * a.d.n1 + i) * a.d.vp + j);
    return rd(a.x.y4, l) + a.g4 * (up + sp + tp) - a.g4 * v;
}

// The row that a warp takes next, asked into L2 while it works on this one: lane
// k asks for the line of array k (the warps in flight alone, at 56-64 registers a
// thread, left the memory half idle).
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
struct NextRow {
    const float* p = nullptr;     // this lane's array at the warp's first column
    long long pitch = 0;
    template <int K>
    __device__ __forceinline__ NextRow(const float* const (&arr)[K], const Dims& d, const float* v) {
        const int k = threadIdx.x;                       // (blocks of 32 x 8)
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (k == q) p = arr[q];
        pitch = d.n2;
        if (k == K) { p = v; pitch = d.vp; }
        if (p) p += min((int)(blockIdx.x * BX), d.n2 - 1);
    }
    __device__ __forceinline__ void ask(const Dims& d, int row) const {
        const int next = row + (int)gridDim.y * BY;
        if (p && next < d.rows) prefetch_l2(p + next * pitch);
    }
};

// SUMS: every global sum of the pass (see the top of the file), and by the
// last block the scalars that follow from them.  Bound by HBM: 13 reads per
// voxel.
__global__ void __launch_bounds__(NTA, 4) k_adj_sums(const AdjArgs a) {
    __shared__ float2 part[BY][kSlots];
    __shared__ double big[NSUM];
    __shared__ bool last;
    const int tid = threadIdx.y * BX + threadIdx.x;
    if (tid < NSUM) big[tid] = 0.0;
    __syncthreads();
    Partial<NSUM> p(big);
    const float* const arr[12] = {a.x.u, a.x.s, a.x.t, a.x.y3, a.x.y4, a.x1.u, a.x1.s, a.x1.t,
                                  a.b1.s, a.b1.t, a.b1.y3, a.b1.y4};
    const NextRow nx(arr, a.d, a.v);
    for_voxels(a.d, [&](int b, int i, int j, long long l, auto in) {
        constexpr bool IN = decltype(in)::value;
        nx.ask(a.d, b * a.d.n1 + i);
        const float q = q_at(a, l, b, i, j);
        const float y4 = rd(a.x.y4, l), yb = rd(a.b1.y4, l);
        const float s1 = rd(a.x1.s, l), t1 = rd(a.x1.t, l);
        const float bs = rd(a.b1.s, l), bt = rd(a.b1.t, l) + 2.f * a.g3 * dvT<IN>(a.b1.y3, a.d, l, i);
        p.f[QQ] = fmaf(q, q, p.f[QQ]);
        p.f[QB] = fmaf(q, yb, p.f[QB]);
        p.f[L1S] += fabsf(rd(a.x.s, l) - a.g_s * y4);
        p.f[L1T] += fabsf(rd(a.x.t, l) - a.g_t * (dvT<IN>(a.x.y3, a.d, l, i) + y4));
        const bool as = s1 != 0.f, at = t1 != 0.f, ps = s1 > 0.f, pt = t1 > 0.f;
        p.f[SS] += as ? (ps ? bs : -bs) : 0.f;
        p.f[SY] += as ? (ps ? yb : -yb) : 0.f;
        p.f[SQ] += as ? (ps ? q : -q) : 0.f;
        p.f[NS] += as ? 1.f : 0.f;
        p.f[ST] += at ? (pt ? bt : -bt) : 0.f;
        p.f[TY4] += at ? (pt ? yb : -yb) : 0.f;
        p.f[TQ] += at ? (pt ? q : -q) : 0.f;
        p.f[NT_] += at ? 1.f : 0.f;
        p.step();
    });
    p.flush();
    // the warp's sums, halving the slots a lane holds at each exchange: lane
    // pair 2k, 2k + 1 ends with the total of the slot in its upper lane bits
    const int lane = threadIdx.x;
    float hi[kSlots], lo[kSlots];
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
        hi[k] = k < NSUM ? p.hi[k < NSUM ? k : 0] : 0.f;
        lo[k] = k < NSUM ? p.lo[k < NSUM ? k : 0] : 0.f;
    }
#pragma unroll
    for (int half = kSlots / 2, o = 16; half > 0; half >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const float oh = __shfl_xor_sync(0xffffffffu, up ? hi[k] : hi[k + half], o);
            const float ol = __shfl_xor_sync(0xffffffffu, up ? lo[k] : lo[k + half], o);
            if (up) { hi[k] = hi[k + half]; lo[k] = lo[k + half]; }
            pair_add(hi[k], lo[k], oh, ol);
        }
    }
    {
        const float oh = __shfl_xor_sync(0xffffffffu, hi[0], 1), ol = __shfl_xor_sync(0xffffffffu, lo[0], 1);
        pair_add(hi[0], lo[0], oh, ol);
    }
    if (!(lane & 1)) part[threadIdx.y][lane >> 1] = make_float2(hi[0], lo[0]);
    __syncthreads();
    if (tid < NSUM) {
        float h = part[0][tid].x, e = part[0][tid].y;
#pragma unroll
        for (int k = 1; k < BY; ++k) pair_add(h, e, part[k][tid].x, part[k][tid].y);
        atomicAdd(a.sc->sum + tid, ((double)h + (double)e) + big[tid]);
        __threadfence();
    }
    __syncthreads();
    if (tid == 0) last = atomicAdd(&a.sc->ticket, 1u) == gridDim.x * gridDim.y - 1u;
    __syncthreads();
    if (!last || tid != 0) return;
    __threadfence();
    double r[NSUM];
#pragma unroll
    for (int k = 0; k < NSUM; ++k) {
        r[k] = __ldcg(a.sc->sum + k);
        a.sc->sum[k] = 0.0;
    }
    a.sc->ticket = 0u;
    // the l2 step: y4+ = (1 - c) q
    const double nq = sqrt(r[QQ]);
    const bool act = nq > a.eps * a.g4d;
    const double qdot = act ? r[QB] / nq : 0.0;                 // q^ . y4_bar+
    const double f = act ? a.eps * a.g4d / nq : 0.0, g = act ? qdot / nq : 0.0;
    a.sc->l2act = act ? 1.f : 0.f;
    a.sc->fk = (float)f;
    a.sc->qs = (float)g;
    if (act) a.pbar[0] += -a.g4d * qdot;
    // S/|A| of the l1 adjoints (the ball inactive: the adjoint passes)
    auto mean = [&](double s, double sy, double sq, double n) {
        if (!(n > 0.0)) return 0.0;
        return (act ? s + 2.0 * a.g4d * ((1.0 - f) * sy + f * g * sq) : s) / n;
    };
    const bool is = r[L1S] <= a.alpha, it = r[L1T] <= a.beta;
    const double ks = is ? 0.0 : mean(r[SS], r[SY], r[SQ], r[NS]), kt = it ? 0.0 : mean(r[ST], r[TY4], r[TQ], r[NT_]);
    a.sc->in_s = is ? 1.f : 0.f;
    a.sc->in_t = it ? 1.f : 0.f;
    a.sc->ks = (float)ks;
    a.sc->kt = (float)kt;
    if (!is) a.pbar[1] += ks;
    if (!it) a.pbar[2] += kt;
}

// CUBE: the l2 step, transposed dual ascents, extrapolations of u, s, t, box,
// l1 adjoints, y4.  18 reads and 7 writes per voxel (the neighbours come from
// cache).
__global__ void __launch_bounds__(NTA, 4) k_adj_cube(const AdjArgs a) {
    const Dims& d = a.d;
    const bool l2act = __ldg(&a.sc->l2act) != 0.f;
    const float fk = __ldg(&a.sc->fk), qs = __ldg(&a.sc->qs);
    const bool in_s = __ldg(&a.sc->in_s) != 0.f, in_t = __ldg(&a.sc->in_t) != 0.f;
    const float ks = __ldg(&a.sc->ks), kt = __ldg(&a.sc->kt);
    const float* const arr[17] = {a.x.u, a.x.s, a.x.t, a.x.y4, a.x1.u, a.x1.s, a.x1.t, a.b1.u, a.b1.s, a.b1.t,
                                  a.b1.y1, a.b1.y1 + d.N, a.b1.y2, a.b1.y2 + d.N, a.b1.y3, a.b1.y4, a.vbar};
    const NextRow nx(arr, d, a.v);
    for_voxels(d, [&](int b, int i, int j, long long l, auto in) {
        constexpr bool IN = decltype(in)::value;
        nx.ask(d, b * d.n1 + i);
        // loads of the buffers that this kernel also writes (in place), first
        const float y4b = a.b1.y4[l], bu = a.b1.u[l], bs = a.b1.s[l], bt = a.b1.t[l], vb = a.vbar[l];
        const float u1 = rd(a.x1.u, l), s1 = rd(a.x1.s, l), t1 = rd(a.x1.t, l);
        const float qbar = l2act ? y4b - fk * (y4b - q_at(a, l, b, i, j) * qs) : 0.f;
        const float ub_ = a.g4 * qbar + a.g2 * dsT_dT<IN>(a.b1.y2, d, l, b, i, j) + a.g1 * dT<IN>(a.b1.y1, d, l, i, j);
        const float sb_ = a.g4 * qbar;
        const float tb_ = a.g4 * qbar + a.g3 * dvT<IN>(a.b1.y3, d, l, i);
        // u+ = box(a_u): the adjoint passes where mu_lo < u+ < mu_hi
        const float u1bar = bu + 2.f * ub_;
        const float aub = (u1 > a.mu_lo && u1 < a.mu_hi) ? u1bar : 0.f;
        const float gb = -a.g_u * aub;
        const float s1bar = bs + 2.f * sb_, t1bar = bt + 2.f * tb_;
        const float asb = in_s ? s1bar : (s1 != 0.f ? s1bar - (s1 > 0.f ? ks : -ks) : 0.f);
        const float atb = in_t ? t1bar : (t1 != 0.f ? t1bar - (t1 > 0.f ? kt : -kt) : 0.f);
        a.vbar[l] = vb - a.g4 * qbar;
        a.b.u[l] = -ub_ + aub;
        a.gbar[l] = gb;
        a.atb[l] = atb;
        a.b.s[l] = -sb_ + asb;
        a.b.t[l] = -tb_ + atb;
        a.b.y4[l] = qbar + (gb - a.g_s * asb - a.g_t * atb);
    });
}

// ---------------------------------------------------------------------------
// DUAL
// ---------------------------------------------------------------------------
// A block owns a 32 x 16 tile of one set and marches over a.len bands: 16
// warps of one voxel per thread, and two warps for the ring of a_w that L^T
// reads around the tile (grid 0 above and right, grid 1 below and left, grid 2
// below and right: 49 lanes with one position per grid).  a_w goes to shared
// memory (two buffers, so one barrier per band), its sums over L^T onto the
// duals.  Writing a_w to memory and reading it back in a launch of its own took
// 24 more words per voxel.  A band needs 28 loads per thread before anything
// can be computed; two blocks per SM (56 registers) keep them in flight while
// the other block computes.
constexpr int DTX = 32, DTY = 16, DTILE = 16, DNT = 32 * (DTILE + 2);
constexpr int DSW = 36, DPL = (DTY + 2) * DSW;    // a_w planes with the ring; row pitch spreads a column over banks
static_assert(DTX * DTY == 32 * DTILE, "one voxel per tile thread");

// One set's arrays.
struct DualSet {
    const float *w, *y, *bw, *by;                 // state k; adjoint of state k+1
    float *ow, *oy;                               // adjoint of state k
    float gw, gy, thr;
};

// The group shrink's adjoint at x = w + g L y with threshold thr: (pv, ph) the
// adjoint of w+; gives the adjoint of x, returns the radial part (the
// derivative in the threshold is its negative).
__device__ __forceinline__ float shrink_adj(float xv, float xh, float pv, float ph, float thr, float& av, float& ah) {
    const float n = sqrtf(xv * xv + xh * xh);
    av = ah = 0.f;
    if (!(n > thr)) return 0.f;
    const float rn = 1.f / n;
    const float xhv = xv * rn, xhh = xh * rn;
    const float dot = xhv * pv + xhh * ph;
    const float k2 = thr * rn, k1 = 1.f - k2;
    av = k1 * pv + k2 * xhv * dot;
    ah = k1 * ph + k2 * xhh * dot;
    return dot;
}

// Which neighbours of (i, j) D leaves nonzero: entries of y_v at rows i-1, i
// and columns j, j+1, of y_h at rows i, i+1 and columns j-1, j; the position
// itself with mv, mh (not on the last row / column).
struct Nbr {
    bool mv, mh, up, dn, lf, rt;                  // last row/column; rows i-1, i+1, columns j-1, j+1 exist
    __device__ __forceinline__ Nbr(const Dims& d, int i, int j) {
        mv = i < d.n1 - 1; mh = j < d.n2 - 1;
        up = i >= 1; dn = i + 1 < d.n1; lf = j >= 1; rt = j + 1 < d.n2;
    }
};
// L y at (i, j) (p: the voxel's address in y's vertical plane, N to the
// horizontal one): out[k], k = 2 grid + component.  A neighbour is read only
// where it exists and D leaves it nonzero.
template <bool IN>
__device__ __forceinline__ void L_at(const float* p, long long N, int n2, const Nbr& m, float out[6]) {
    const float* h = p + N;
    const float v00 = IN || m.mv ? __ldg(p) : 0.f, vm0 = IN || m.up ? __ldg(p - n2) : 0.f,
                v01 = IN || (m.mv && m.rt) ? __ldg(p + 1) : 0.f, vm1 = IN || (m.up && m.rt) ? __ldg(p - n2 + 1) : 0.f;
    const float h00 = IN || m.mh ? __ldg(h) : 0.f, h0m = IN || m.lf ? __ldg(h - 1) : 0.f,
                h10 = IN || (m.dn && m.mh) ? __ldg(h + n2) : 0.f, h1m = IN || (m.dn && m.lf) ? __ldg(h + n2 - 1) : 0.f;
    out[0] = v00;
    out[1] = IN || m.mv ? 0.25f * (h00 + h0m + h10 + h1m) : 0.f;
    out[2] = IN || m.mh ? 0.25f * (v00 + vm0 + v01 + vm1) : 0.f;
    out[3] = h00;
    out[4] = 0.5f * (v00 + vm0);
    out[5] = 0.5f * (h00 + h0m);
}

// The tile's voxels.
template <int SET, bool IN>
__device__ __forceinline__ void dual_tile(const AdjArgs& a, const DualSet& S, float* sm, double* big, int i0, int j0,
                                          int b0, int b1) {
    const Dims& d = a.d;
    const long long N = d.N;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = i0 + wid, j = j0 + lane;
    const bool valid = IN || (i < d.n1 && j < d.n2);
    const Nbr m(d, i, j);
    long long l = valid ? (long long)b0 * d.plane + (long long)i * d.n2 + j : 0;
    float* own = sm + (wid + 1) * DSW + lane + 1;
    Partial<1> om(big);
    float gn[3] = {0.f, 0.f, 0.f};                // SET 1: G_bar of the next band at (0,0), (1,0), (0,1)
    auto load_g = [&](long long lg, float g[3]) {
        const float* p = a.gbar + lg;
        g[0] = __ldg(p);
        g[1] = IN || m.mv ? __ldg(p + d.n2) : 0.f;
        g[2] = IN || m.mh ? __ldg(p + 1) : 0.f;
    };
    if (SET == 1 && valid) load_g(l, gn);
    // this row of the next band asked into L2 while this band is worked on: lane
    // k for plane k of w, the adjoint of w, y and the adjoint of y; lanes 16 up
    // for the row's other end (rows need not start on a line)
    const float* ask;
    {
        const int k = lane & 15;
        ask = k < 6 ? S.w + k * N : k < 12 ? S.bw + (k - 6) * N : k < 14 ? S.y + (k - 12) * N : S.by + (k - 14) * N;
        ask += (long long)(b0 + 1) * d.plane + (long long)min(i, d.n1 - 1) * d.n2 + min(j0 + (lane & 16 ? 31 : 0), d.n2 - 1);
    }
    for (int b = b0; b < b1; ++b, l += d.plane) {
        if (b + 1 < b1) prefetch_l2(ask);
        ask += d.plane;
        float* buf = own + ((b - b0) & 1) * (6 * DPL);
        float byv = 0.f, byh = 0.f, dg0 = 0.f, dg1 = 0.f;
        if (valid) {
            float w[6], bw[6], lb[6], lx[6], g[3];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                w[k] = __ldg(S.w + l + k * N);
                bw[k] = __ldg(S.bw + l + k * N);
            }
            L_at<IN>(S.by + l, N, d.n2, m, lb);
            L_at<IN>(S.y + l, N, d.n2, m, lx);
            byv = IN || m.mv ? lb[0] : __ldg(S.by + l);
            byh = IN || m.mh ? lb[3] : __ldg(S.by + l + N);
            if constexpr (SET == 0) {
                load_g(l, g);
                // y3 -= g_t D_v a_t_bar
                const float at = __ldg(a.atb + l), b3 = a.b1.y3[l];
                const float dvat = IN || m.mv ? __ldg(a.atb + l + d.n2) - at : 0.f;
                a.b.y3[l] = b3 - a.g_t * dvat;
            } else {
                // D_s G_bar
                const float c0 = gn[0], c1 = gn[1], c2 = gn[2];
                const bool nxt = b < d.n3 - 1;
                if (nxt) load_g(l + d.plane, gn);
                g[0] = nxt ? gn[0] - c0 : 0.f;
                g[1] = nxt ? gn[1] - c1 : 0.f;
                g[2] = nxt ? gn[2] - c2 : 0.f;
            }
            dg0 = IN || m.mv ? g[1] - g[0] : 0.f;
            dg1 = IN || m.mh ? g[2] - g[0] : 0.f;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float wbv = -S.gy * lb[2 * q], wbh = -S.gy * lb[2 * q + 1];      // adjoint of w'
                const float pv = bw[2 * q] + 2.f * wbv, ph = bw[2 * q + 1] + 2.f * wbh; // total of w+
                float av, ah;
                const float dot = shrink_adj(w[2 * q] + S.gw * lx[2 * q], w[2 * q + 1] + S.gw * lx[2 * q + 1], pv, ph,
                                             S.thr, av, ah);
                if (SET == 0) om.f[0] -= dot;
                S.ow[l + (2 * q) * N] = -wbv + av;
                S.ow[l + (2 * q + 1) * N] = -wbh + ah;
                // L^T takes zero where L's output is structurally zero (the
                // buffers start zero)
                if (IN || (q == 0 ? m.mv : q == 1 ? m.mh : true)) {
                    buf[(2 * q) * DPL] = av;
                    buf[(2 * q + 1) * DPL] = ah;
                }
            }
            if (SET == 0) {
                om.fold();                        // (float sums of three terms, as where a thread has one voxel)
                om.step();
            }
        }
        __syncthreads();
        if (valid) {
            auto W = [&](int k, int di, int dj) { return buf[k * DPL + di * DSW + dj]; };
            const float gv = IN || m.mv ? W(0, 0, 0) + 0.25f * (W(2, 0, 0) + W(2, 1, 0) + W(2, 0, -1) + W(2, 1, -1)) +
                                              0.5f * (W(4, 0, 0) + W(4, 1, 0))
                                        : 0.f;
            const float gh = IN || m.mh ? 0.25f * (W(1, 0, 0) + W(1, 0, 1) + W(1, -1, 0) + W(1, -1, 1)) + W(3, 0, 0) +
                                              0.5f * (W(5, 0, 0) + W(5, 0, 1))
                                        : 0.f;
            S.oy[l] = byv + (dg0 + S.gw * gv);
            S.oy[l + N] = byh + (dg1 + S.gw * gh);
        }
    }
    if (SET == 0) {
        // the adjoint of omega: -g_w1 times the sum of the radial parts
        om.flush();
        float h = om.hi[0], e = om.lo[0];
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, h, o), oe = __shfl_xor_sync(0xffffffffu, e, o);
            pair_add(h, e, oh, oe);
        }
        if (lane == 0) {
            sm[12 * DPL + 2 * wid] = h;
            sm[12 * DPL + 2 * wid + 1] = e;
        }
    }
}

// The ring's positions.
template <int SET, bool IN>
__device__ __forceinline__ void dual_ring(const AdjArgs& a, const DualSet& S, float* sm, int b0, int b1,
                                          const int (&ri)[3], const int (&rj)[3], const int (&ko)[3], bool has) {
    const Dims& d = a.d;
    const long long N = d.N;
    const int n2 = d.n2;
    // grid 0 is structurally zero on the last row, grid 1 on the last column
    bool on[3];
    long long l[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        on[q] = has && (IN || (ri[q] >= 0 && ri[q] < d.n1 && rj[q] >= 0 && rj[q] < d.n2 &&
                               (q != 0 || ri[q] < d.n1 - 1) && (q != 1 || rj[q] < d.n2 - 1)));
        l[q] = on[q] ? (long long)b0 * d.plane + (long long)ri[q] * n2 + rj[q] : 0;
    }
    const Nbr m0(d, ri[0], rj[0]), m1(d, ri[1], rj[1]), m2(d, ri[2], rj[2]);
    // (L y)_v, (L y)_h at the position of each grid
    auto L3 = [&](const float* y, float o[6]) {
        {   // grid 0: y_v itself, the four-point mean of y_h
            const float *v = y + l[0], *h = v + N;
            o[0] = on[0] ? __ldg(v) : 0.f;
            const float h00 = on[0] && (IN || m0.mh) ? __ldg(h) : 0.f, h0m = on[0] && (IN || m0.lf) ? __ldg(h - 1) : 0.f,
                        h10 = on[0] && (IN || m0.mh) ? __ldg(h + n2) : 0.f,
                        h1m = on[0] && (IN || m0.lf) ? __ldg(h + n2 - 1) : 0.f;
            o[1] = 0.25f * (h00 + h0m + h10 + h1m);
        }
        {   // grid 1: the four-point mean of y_v, y_h itself
            const float *v = y + l[1], *h = v + N;
            const float v00 = on[1] && (IN || m1.mv) ? __ldg(v) : 0.f, vm0 = on[1] && (IN || m1.up) ? __ldg(v - n2) : 0.f,
                        v01 = on[1] && (IN || m1.mv) ? __ldg(v + 1) : 0.f,
                        vm1 = on[1] && (IN || m1.up) ? __ldg(v - n2 + 1) : 0.f;
            o[2] = 0.25f * (v00 + vm0 + v01 + vm1);
            o[3] = on[1] ? __ldg(h) : 0.f;
        }
        {   // grid 2: the centred means
            const float *v = y + l[2], *h = v + N;
            const float v00 = on[2] && (IN || m2.mv) ? __ldg(v) : 0.f, vm0 = on[2] && (IN || m2.up) ? __ldg(v - n2) : 0.f;
            const float h00 = on[2] && (IN || m2.mh) ? __ldg(h) : 0.f, h0m = on[2] && (IN || m2.lf) ? __ldg(h - 1) : 0.f;
            o[4] = 0.5f * (v00 + vm0);
            o[5] = 0.5f * (h00 + h0m);
        }
    };
    for (int b = b0; b < b1; ++b) {
        float* buf = sm + ((b - b0) & 1) * (6 * DPL);
        float w[6], bw[6], lb[6], lx[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            w[k] = on[k / 2] ? __ldg(S.w + l[k / 2] + k * N) : 0.f;
            bw[k] = on[k / 2] ? __ldg(S.bw + l[k / 2] + k * N) : 0.f;
        }
        L3(S.by, lb);
        L3(S.y, lx);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float wbv = -S.gy * lb[2 * q], wbh = -S.gy * lb[2 * q + 1];
            const float pv = bw[2 * q] + 2.f * wbv, ph = bw[2 * q + 1] + 2.f * wbh;
            float av, ah;
            shrink_adj(w[2 * q] + S.gw * lx[2 * q], w[2 * q + 1] + S.gw * lx[2 * q + 1], pv, ph, S.thr, av, ah);
            if (on[q]) {
                buf[(2 * q) * DPL + ko[q]] = av;
                buf[(2 * q + 1) * DPL + ko[q]] = ah;
            }
            l[q] += on[q] ? d.plane : 0;
        }
        __syncthreads();
    }
}

template <int SET>
__device__ __forceinline__ void dual_block(const AdjArgs& a, float* sm, double* big, int tiles_x, int run) {
    const Dims& d = a.d;
    DualSet S;
    S.w = SET ? a.x.w2 : a.x.w1; S.y = SET ? a.x.y2 : a.x.y1;
    S.bw = SET ? a.b1.w2 : a.b1.w1; S.by = SET ? a.b1.y2 : a.b1.y1;
    S.ow = SET ? a.b.w2 : a.b.w1; S.oy = SET ? a.b.y2 : a.b.y1;
    S.gw = SET ? a.g_w2 : a.g_w1; S.gy = SET ? a.g2 : a.g1; S.thr = SET ? a.th2 : a.th1;
    const int ty = blockIdx.x / tiles_x, tx = blockIdx.x - ty * tiles_x;
    const int i0 = ty * DTY, j0 = tx * DTX;
    const int b0 = run * a.len, b1 = min(d.n3, b0 + a.len);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto inside = [&](int i, int j) { return i >= 1 && i <= d.n1 - 2 && j >= 1 && j <= d.n2 - 2; };
    if (wid < DTILE) {
        if (__all_sync(0xffffffffu, inside(i0 + wid, j0 + lane))) dual_tile<SET, true>(a, S, sm, big, i0, j0, b0, b1);
        else dual_tile<SET, false>(a, S, sm, big, i0, j0, b0, b1);
    } else {
        const int q = wid - DTILE;
        // grid 0 at (-1, c), grids 1, 2 at (DTY, c) for a column c; grids 0, 2
        // at (r, DTX), grid 1 at (r, -1) for a row r; the corners (-1, DTX) of
        // grid 0 and (DTY, -1) of grid 1.  Each warp takes half of each.
        const bool has = lane < (q == 0 ? 25 : 24);
        int r[3], c[3], ko[3];
        if (lane < 8) {
            r[0] = r[1] = r[2] = 8 * q + lane;
            c[0] = c[2] = DTX;
            c[1] = -1;
        } else {
            r[0] = -1;
            r[1] = r[2] = DTY;
            c[0] = lane < 24 ? 16 * q + lane - 8 : DTX;
            c[1] = c[2] = lane < 24 ? c[0] : -1;
        }
        bool in = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            ko[k] = (r[k] + 1) * DSW + c[k] + 1;
            r[k] += i0;
            c[k] += j0;
            in = in && inside(r[k], c[k]);
        }
        if (__all_sync(0xffffffffu, in || !has)) dual_ring<SET, true>(a, S, sm, b0, b1, r, c, ko, has);
        else dual_ring<SET, false>(a, S, sm, b0, b1, r, c, ko, has);
    }
    if (SET == 0) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const float* red = sm + 12 * DPL;
            float h = red[0], e = red[1];
            for (int k = 1; k < DTILE; ++k) pair_add(h, e, red[2 * k], red[2 * k + 1]);
            atomicAdd(a.pbar + 3, a.g_w1d * (((double)h + (double)e) + *big));
        }
    }
}

// blocks: (tile, run of bands x set), sets set0 .. set0 + nset - 1
__global__ void __launch_bounds__(DNT, 2) k_adj_dual(const AdjArgs a, int tiles_x, int set0, int nset) {
    __shared__ float sm[12 * DPL + 2 * DTILE];
    __shared__ double big;
    if (threadIdx.x == 0) big = 0.0;
    for (int k = threadIdx.x; k < 12 * DPL; k += DNT) sm[k] = 0.f;
    __syncthreads();
    const int run = blockIdx.y / nset, set = set0 + (blockIdx.y - run * nset);
    if (set == 0) dual_block<0>(a, sm, &big, tiles_x, run);
    else dual_block<1>(a, sm, &big, tiles_x, run);
}

// Launch facts of one device: SM count and resident blocks of each kernel.
struct StepInfo {
    int sms = 0;
    int res[3] = {0, 0, 0};
};

int resident_of(const void* fn, int threads) {
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, threads, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return std::max(1, nb);
}

// blocks of 32 x 8 threads: columns in x, persistent over the rows in y
dim3 step_grid(const Dims& d, int resident, int sms) {
    const int gx = (d.n2 + BX - 1) / BX;
    const long long rb = ((long long)d.rows + BY - 1) / BY;
    const long long want = std::max(1ll, (long long)sms * std::max(1, resident) / gx);
    return dim3(gx, (unsigned)std::min({rb, want, 65535ll}));
}

// Bands per block of DUAL: the split whose waves of `slots` resident blocks
// march the fewest bands, a block's own start (pointers, clearing its shared
// memory, the first loads' latency) counted as most of a band.
int dual_len(const Dims& d, long long tiles, int nset, int slots) {
    int best_len = d.n3, prev = 0;
    double best = 1e300;
    for (int runs = 1; runs <= d.n3; ++runs) {
        const int len = (d.n3 + runs - 1) / runs;
        if (len == prev) continue;
        prev = len;
        const long long nruns = (d.n3 + len - 1) / len;
        if (nruns * nset > 65535) break;
        const double cost = (double)((tiles * nset * nruns + slots - 1) / slots) * (len + 0.7);
        if (cost < best * (1.0 - 1e-12)) { best = cost; best_len = len; }
    }
    return best_len;
}

// Resident blocks of each kernel and the SM count, filled once per device
// (std::call_once: concurrent first calls from several host threads wait for
// the one that fills it).
const StepInfo& step_info() {
    constexpr int kMaxDev = 64;
    static StepInfo info[kMaxDev + 1];          // the last entry: device query failed
    static std::once_flag once[kMaxDev + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) {
        cudaGetLastError();
        dev = kMaxDev;
    }
    StepInfo& a = info[dev];
    std::call_once(once[dev], [&a] {
        a.res[0] = resident_of((const void*)k_adj_sums, NTA);
        a.res[1] = resident_of((const void*)k_adj_cube, NTA);
        a.res[2] = resident_of((const void*)k_adj_dual, DNT);
        a.sms = device_sms();
    });
    return a;
}

}  // namespace

size_t adjoint_step_bytes(long long n) {
    return (size_t)adj_stride(n) * 2 * sizeof(float) + kAdjScalBytes;
}
size_t adjoint_spare_bytes(long long n) { return (size_t)adj_stride(n) * 8 * sizeof(float); }

int launch_adjoint_single(int n1, int n2, int n3, const float* const x[9], const float* const x1[9],
                        const float* const b1[9], float* const bo[9], void* spare, const float* v, int v_pitch,
                        float* vbar, double* pbar, void* work, const double prm[16], cudaStream_t st) {
    const StepInfo& info = step_info();
    const int* res = info.res;
    AdjArgs a;
    a.d.n1 = n1; a.d.n2 = n2; a.d.n3 = n3; a.d.vp = v_pitch;
    a.d.rows = n3 * n1;
    a.d.plane = (long long)n1 * n2;
    a.d.N = (long long)n1 * n2 * n3;
    const long long N = a.d.N;
    a.x = SV{x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7], x[8]};
    a.x1 = SV{x1[0], x1[1], x1[2], x1[3], x1[4], x1[5], x1[6], x1[7], x1[8]};
    a.b1 = SV{b1[0], b1[1], b1[2], b1[3], b1[4], b1[5], b1[6], b1[7], b1[8]};
    a.b = SW{bo[0], bo[1], bo[2], bo[3], bo[4], bo[5], bo[6], bo[7], bo[8]};
    a.v = v;
    a.vbar = vbar;
    a.pbar = pbar;
    // each region on a 256-byte boundary (the sums are doubles): G_bar, a_t_bar;
    // in place, the spare set (w: 6 regions, y: 2; their planes at the cube stride N)
    float* f = (float*)work;
    const long long P = adj_stride(N);
    a.gbar = f; a.atb = f + P;
    a.sc = (AdjScal*)(f + 2 * P);
    a.g_u = (float)prm[0]; a.g_w1 = (float)prm[1]; a.g_w2 = (float)prm[2]; a.g_s = (float)prm[3];
    a.g_t = (float)prm[4]; a.g1 = (float)prm[5]; a.g2 = (float)prm[6]; a.g3 = (float)prm[7];
    a.g4 = (float)prm[8]; a.th1 = (float)prm[9]; a.th2 = (float)prm[10];
    a.mu_lo = (float)prm[11]; a.mu_hi = (float)prm[12];
    a.eps = prm[13]; a.alpha = prm[14]; a.beta = prm[15];
    a.g4d = prm[8]; a.g_w1d = prm[1];
    if (N == 0) return 0;
    const dim3 blk(BX, BY);
    k_adj_sums<<<step_grid(a.d, res[0], info.sms), blk, 0, st>>>(a);
    k_adj_cube<<<step_grid(a.d, res[1], info.sms), blk, 0, st>>>(a);
    const int tx = (n2 + DTX - 1) / DTX;
    const long long tiles = (long long)tx * ((n1 + DTY - 1) / DTY);
    auto dual = [&](int set0, int nset) {
        a.len = dual_len(a.d, tiles, nset, info.sms * res[2]);
        const dim3 grid((unsigned)tiles, (unsigned)(((n3 + a.len - 1) / a.len) * nset));
        k_adj_dual<<<grid, DNT, 0, st>>>(a, tx, set0, nset);
    };
    if (!spare) {
        dual(0, 2);
    } else {
        // in place: a set's inputs copied to the spare set first
        float *spare_w = (float*)spare, *spare_y = spare_w + 6 * P;
        for (int s = 0; s < 2; ++s) {
            const float *&w = s ? a.b1.w2 : a.b1.w1, *&y = s ? a.b1.y2 : a.b1.y1;
            if (cudaMemcpyAsync(spare_w, w, 6 * N * sizeof(float), cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
                cudaMemcpyAsync(spare_y, y, 2 * N * sizeof(float), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
                return -3;
            w = spare_w;
            y = spare_y;
            dual(s, 1);
        }
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace gsstv
