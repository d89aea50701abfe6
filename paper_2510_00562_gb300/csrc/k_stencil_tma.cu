// K1, the fused stencil pass of one P-PDS iteration (Algorithm 1).
//
// For each band: the u step and u' of the next band; the w1, w2 group
// soft-thresholds and w' on the tile plus a one-pixel ring; the y1, y2 ascent;
// the window statistics of the l1 threshold search.
//
// Every tile runs the same code, with the masks of the image border.  Interior
// tiles once had code of their own without masks: the two loops did not fit the
// instruction cache that the two SMs of a pair share, and wherever a border tile
// and an interior one ran on a pair both took 2.3 to 3.1 us a band step instead
// of 2.0 (264x176x184 358 us a launch and 274 with one code, 176x104x94 111 and
// 75, 256x256x128 263 and 237, bfloat16 512x512x224 2464 and 2364; sizes with few
// such pairs 2 % slower to 3 % faster).
//
// One persistent CTA per SM works through (tile, band run) items, in the order
// in which neighbouring tiles run at the same time over the same bands (their
// halos then meet in L2).  Its warps have roles:
//   16 tile warps   one voxel of the 16 x 32 tile per thread;
//   2 ring warps    the one-pixel ring of w' and of u' (49 positions).  The
//                   ascent reads on the ring only grid 0 above and right of the
//                   tile, grid 1 below and left, grid 2 below and right, so 49
//                   lanes with one position per grid cover it: the work of a
//                   tile warp without its stores, and no tile warp does ring
//                   work on top of its own before the band barrier;
//   load warps      bring each band's planes into shared-memory rings, as far
//                   ahead as slots are free and across item boundaries: one
//                   warp of bulk tensor (TMA) copies for float32 storage, two
//                   of 8-byte cp.async for 16-bit storage (the planes stay
//                   16-bit in shared memory and are widened as they are read).
// Full / empty mbarriers per slot couple the load warps to the others.  Every
// wait is bounded; a wait that gives up raises a flag that ends the CTA.
//
// Band step, one barrier phase per band (an mbarrier with an arrival per
// warp, so that arriving and waiting are apart): the dual ascent of the
// previous band (it reads the w' and u' that the previous phase published);
// the w steps and u' of the next band; arrive; the window statistics of the
// next band, which nobody waits for, fill the time until the others arrive.
// Each thread keeps the four y values of its own voxel that the ascent needs,
// and D^T y2 of the previous band at its own u' position, in registers.
//
// What bounds it: instruction issue (63 % of the slots) and the latency of 18
// warps' dependency chains (0.88 of the copy bandwidth at 512x512x224, 0.77 at
// 256x256x128, where the split into whole items leaves 12 % of the band steps idle).
#include <algorithm>
#include <vector>
#include <cmath>
#include <type_traits>

#include "gsstv_internal.cuh"
#include "gsstv_l1.cuh"
#include "gsstv_tma.cuh"

namespace gsstv {

// ---------------------------------------------------------------------------
// host: tensor maps
// ---------------------------------------------------------------------------
namespace {
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn() {
    static EncodeFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
    }
    return fn;
}
}  // namespace

// A 3-D tiled map over `ncubes` stacked pitched float32 cubes of geometry g, of
// which the first n1 rows and n2 columns of each band exist (zero fill outside),
// box (box_x, box_y, 1).  Returns 0 on success.
static int tma_encode_cubes(CUtensorMap* map, const void* base, const Geom& g, int n1, int n2, int ncubes, int box_x,
                            int box_y) {
    EncodeFn fn = encode_fn();
    if (!fn) return -3;
    const CUtensorMapDataType dt = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    cuuint64_t dims[3] = {(cuuint64_t)n2, (cuuint64_t)n1, (cuuint64_t)g.n3 * (cuuint64_t)ncubes};
    cuuint64_t strides[2] = {(cuuint64_t)g.p2 * 4u, (cuuint64_t)g.p2 * 4u * g.n1};
    cuuint32_t box[3] = {(cuuint32_t)box_x, (cuuint32_t)box_y, 1u};
    cuuint32_t estr[3] = {1u, 1u, 1u};
    const CUresult r = fn(map, dt, 3, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -3;
}

namespace {


constexpr int pad128(int b) { return (b + 127) / 128 * 128; }

constexpr int TY = 16, TX = 32;
constexpr int OX = 4;                    // left halo columns: staged rows start 16-byte (16-bit: 8-byte) aligned
constexpr int SW = TX + 2 * OX;          // width of the staged planes
constexpr int YR = TY + 4, WR = TY + 2, UR = TY + 1, UC = TX + 1;
constexpr int kTileWarps = 16, kRingWarps = 2, kConsWarps = kTileWarps + kRingWarps;
constexpr int kCandBuf = 256;            // window candidates buffered per item and vector
constexpr int kMaxRun = 4064;            // bands per item at most (16-bit histogram counters, see k1_plan)
static_assert(TY * TX == 32 * kTileWarps, "one tile voxel per tile thread");

template <typename T>
struct Lay {
    static constexpr bool F32 = std::is_same<T, float>::value;
    static constexpr int LW = F32 ? 1 : 2;               // load warps
    static constexpr int NT = 32 * (kConsWarps + LW);
    static constexpr int ES = (int)sizeof(T);
    static constexpr int Y_B = pad128(YR * SW * ES);
    static constexpr int W_B = pad128(WR * SW * ES);
    static constexpr int U_B = pad128(UR * SW * ES);
    static constexpr int S_B = pad128(TY * TX * ES);
    static constexpr int Y3_B = pad128((TY + 1) * TX * ES);
    static constexpr int YG_B = 4 * Y_B + 2 * U_B + 2 * S_B + Y3_B;
    static constexpr int WG_B = 12 * W_B;
    // ring depths: y-group, w, u'.  float32 w' overwrites w in place, so a w
    // slot is held one band longer (until the ascent has read it); 16-bit
    // storage keeps float32 w' in two slots of its own
    static constexpr int NYS = 3, NWS = F32 ? 4 : 3, NUS = 3, NPS = F32 ? 0 : 2;
    static constexpr int UP1 = UR * UC;                  // floats of one u' plane
    static constexpr int WPL = pad128(WR * SW * 4) / 4;  // floats of one w' plane
    static constexpr int OFF_WG = NYS * YG_B;
    static constexpr int OFF_WP = OFF_WG + NWS * WG_B;
    static constexpr int OFF_UP = OFF_WP + NPS * 12 * WPL * 4;
    static constexpr int OFF_CB = OFF_UP + pad128(NUS * UP1 * 4);
    static constexpr int OFF_HIST = OFF_CB + 4 * kCandBuf * 4;    // K1 histogram: 2 x kK1Bins packed 16-bit counts
    static constexpr int OFF_BAR = OFF_HIST + kK1Bins * 4;
    // 16-bit: the window's values of three bands (see Ordered)
    static constexpr int OFF_X = pad128(OFF_BAR + (2 * NYS + 2 * NWS + 1) * 8);
    static constexpr int SMEM = F32 ? OFF_BAR + (2 * NYS + 2 * NWS + 1) * 8 : OFF_X + NUS * TY * TX * 8;
    // element offsets inside a y-group slot, and between raw planes
    static constexpr int YPL = Y_B / ES, WRAW = W_B / ES;
    static constexpr int O_U = 4 * YPL, O_Q = O_U + U_B / ES, O_S = O_Q + U_B / ES, O_T = O_S + S_B / ES,
                         O_Y3 = O_T + S_B / ES;
    // dynamic plus the kernel's static shared memory within the 227 KB a CTA may use
    static_assert(SMEM + 512 <= 227 * 1024, "shared memory");
    static_assert(!F32 || WPL == WRAW, "w' in place");
};

template <typename T>
struct K1Args {
    Geom g;
    const T *u, *q, *s, *t, *y3, *y1, *y2, *w1, *w2;
    T *u_n, *w1_n, *w2_n, *y1_n, *y2_n;
    IterParams p;
    Scal* sc;
    L1Work l1;
    int chunk;          // bands per item
    int unit;           // sums in a fixed order: bands per piece (chunk is a multiple of it)
    SlabPart sp;
};

// Window of the l1 threshold search for this launch (see gsstv_l1.cuh), and
// the histograms of |s~|, |t~| near the predicted thresholds when they are on.
struct K1Win {
    bool s, t;
    float lo_s, hi_s, lo_t, hi_t;
    bool hs, ht;
    unsigned hb_s, hb_t;
};

// A thread's count and sum of sampled values above the histogram's range.
struct K1Acc {
    unsigned n = 0;
    float s = 0.f;
};

// A thread's window statistics (a CTA covers at most a few thousand voxels per
// thread slot, so 32-bit counts suffice), the compensated sums of s and t packed.
struct K1Stat {
    unsigned n_s = 0, n_t = 0;
    float2 ks = make_float2(0.f, 0.f), kc = make_float2(0.f, 0.f);
    K1Acc top_s, top_t;
};

// 16-bit storage: the sums above the windows in the order and the pieces of the
// cooperative kernel (a thread's sum over `unit` bands of the tile's rows r and
// r + 8, row r before row r + 8 at each band), so that both kernels find the
// same thresholds: a threshold one float ulp off flips random roundings of a
// 16-bit iterate.  The warps of rows 0-7 add up what all 16 rows' warps leave
// in shared memory, one band late; finished pieces join a float pair.  (Sums
// split otherwise, with a histogram and exact additions, moved one threshold in
// 32 passes of a 256x256x200 float16 solve by an ulp and the result by up to a
// float16 place, and a pass took the same time.  It takes 0.80 ms, 1.47 in the
// cooperative kernel's launches; at 512x512x224 bfloat16 3.3 and 6.05 ms.)
//
// float32 storage with the sums in their fixed order (FIX, gsstv_set_fixed_sums):
// a thread's Kahan sum over `unit` bands of its own voxel, in one launch shape for
// every run.  A solve sums more exactly and splits as the SMs are filled best; the
// thresholds of the two differ by 1e-10, which rounds to another float once in some
// hundred passes, and the FP64 adjoints of a run of 9 to 40 passes then moved by
// 1e-8 to 9e-6 (5 of 40 runs).
struct Ordered {
    KahanSum s, t;
    float hs = 0.f, ls = 0.f, ht = 0.f, lt = 0.f;
    __device__ __forceinline__ void add(float2 x) {            // a component below zero: not above its window
        if (x.x >= 0.f) s.add(x.x);
        if (x.y >= 0.f) t.add(x.y);
    }
    __device__ __forceinline__ void close() {
        pair_add(hs, ls, s.s, -s.c);
        pair_add(ht, lt, t.s, -t.c);
        s = t = KahanSum();
    }
    // a piece's packed sums of the two vectors
    __device__ __forceinline__ void close(float2& ks, float2& kc) {
        pair_add(hs, ls, ks.x, -kc.x);
        pair_add(ht, lt, ks.y, -kc.y);
        ks = kc = make_float2(0.f, 0.f);
    }
};

// A position in a ring of N slots and the phase parity of its next use.
template <int N>
struct Ring {
    int slot = 0;
    unsigned ph = 0;
    __device__ __forceinline__ void next() {
        if (++slot == N) { slot = 0; ph ^= 1u; }
    }
};

// Bounded wait that also gives up once another warp of the CTA has.
__device__ __forceinline__ bool k1_wait(uint64_t* bar, unsigned parity, volatile int* abort) {
    if (mbar_try_wait(bar, parity)) return true;
    for (unsigned k = 0; k < kMbarSpinLimit; ++k) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((k & 255u) == 255u && *abort) return false;
    }
    *abort = 1;
    return false;
}

// Appends the lanes' window candidates to the CTA's shared buffer (one
// shared-memory atomic per warp); values past its end go straight to the
// global list (and are not counted into its key histogram, so that the finish
// then bins the list itself: counting them here made K1 2 % slower).  `cnt`
// keeps counting past the buffer.
__device__ __forceinline__ void append_shared(bool take, float x, float* buf, unsigned* cnt, float* cand,
                                              unsigned* gcnt) {
    const unsigned mask = __ballot_sync(0xffffffffu, take);
    if (mask == 0) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(mask) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(cnt, (unsigned)__popc(mask));
    base = __shfl_sync(0xffffffffu, base, leader);
    const unsigned k = base + __popc(mask & ((1u << lane) - 1u));
    if (take && k < (unsigned)kCandBuf) buf[k] = x;
    if (base + __popc(mask) > (unsigned)kCandBuf) {
        const bool over = take && k >= (unsigned)kCandBuf;
        append_candidate(over, x, cand, gcnt);
    }
}

// One warp: the buffered candidates of vector v join the global list (one
// atomic) and its key histogram over the window, which the finish then narrows
// without another pass over the candidates.
__device__ __forceinline__ void flush_candidates(int v, float* buf, unsigned* cnt, Scal* sc, const L1Work& l1,
                                              float lo, float hi) {
    const int lane = threadIdx.x & 31;
    const unsigned n = min(*cnt, (unsigned)kCandBuf);
    if (n == 0) return;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&sc->acc[v].m, n);
    base = __shfl_sync(0xffffffffu, base, 0);
    const NarrowGeom ng = narrow_geom(__float_as_uint(lo), __float_as_uint(hi));
    unsigned* h = l1.nh && ng.ok ? l1.nh + v * 3 * kNarrowBins : nullptr;
    for (unsigned k = lane; k < n; k += 32u) {
        const float x = buf[k];
        if (base + k < kCandCap) l1.cand[v][base + k] = x;
        if (h) narrow_add(h, ng, __float_as_uint(x));
    }
    __syncwarp();
    if (lane == 0) {
        if (h) atomicAdd(l1.nbinned + v, n);
        *cnt = 0u;
    }
    __syncwarp();
}

// Counts x into the CTA's histogram (bins of the float key >> kHistShift from
// hb; two 16-bit counters per shared word), or into the above-range
// accumulator; values below the range are not needed.
__device__ __forceinline__ void hist_add(bool on, float x, unsigned hb, unsigned* h, K1Acc& top) {
    const unsigned kb = __float_as_uint(x) >> kHistShift;
    const unsigned bin = kb - hb;                    // below the range wraps to a large value
    const bool in = on && bin < (unsigned)kK1Bins;
    if (in) atomicAdd(h + (bin >> 1), (bin & 1u) ? 65536u : 1u);
    // above the range: an estimate from a sample, a plain sum suffices
    const bool up = on && !in && kb >= hb + (unsigned)kK1Bins;
    top.n += up ? 1u : 0u;
    top.s += up ? x : 0.f;
}

// Packed FP32 pairs (two lanes per instruction on sm_100 and later), used for
// the (vertical, horizontal) pairs of the stencil; each lane rounds exactly as
// the scalar operation would.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, f2(-1.f, -1.f), a); }

// What a CTA's warps share: shared-memory regions and barriers.
template <typename T>
struct Sm {
    unsigned char* sm;
    uint64_t *yfull, *yempty, *wfull, *wempty, *evt;
    unsigned* ccnt;
    int* abort;
    __device__ __forceinline__ Sm(unsigned char* p, unsigned* c, int* ab) : sm(p), ccnt(c), abort(ab) {
        using L = Lay<T>;
        yfull = reinterpret_cast<uint64_t*>(p + L::OFF_BAR);
        yempty = yfull + L::NYS;
        wfull = yempty + L::NYS;
        wempty = wfull + L::NWS;
        evt = wempty + L::NWS;
    }
    __device__ __forceinline__ T* yg(int slot) const { return reinterpret_cast<T*>(sm + slot * Lay<T>::YG_B); }
    __device__ __forceinline__ T* wg(int slot) const {
        return reinterpret_cast<T*>(sm + Lay<T>::OFF_WG + slot * Lay<T>::WG_B);
    }
    // w' of a band: in place of w (float32), or the band's slot of its own
    __device__ __forceinline__ float* wp(int wslot, int pslot) const {
        if constexpr (Lay<T>::F32) return reinterpret_cast<float*>(wg(wslot));
        else return reinterpret_cast<float*>(sm + Lay<T>::OFF_WP) + pslot * (12 * Lay<T>::WPL);
    }
    __device__ __forceinline__ float* up(int slot) const {
        return reinterpret_cast<float*>(sm + Lay<T>::OFF_UP) + slot * Lay<T>::UP1;
    }
    // candidates of vector v of an even or odd item: filled during the item,
    // emptied while the next one fills the other
    __device__ __forceinline__ float* cbuf(int v, int odd) const {
        return reinterpret_cast<float*>(sm + Lay<T>::OFF_CB) + (2 * odd + v) * kCandBuf;
    }
    __device__ __forceinline__ unsigned* cnt(int v, int odd) const { return ccnt + 2 * odd + v; }
    // 16-bit: |s~|, |t~| of one band where they are above their windows, else -1
    __device__ __forceinline__ float2* above(int slot) const {
        return reinterpret_cast<float2*>(sm + Lay<T>::OFF_X) + slot * (TY * TX);
    }
    __device__ __forceinline__ unsigned* hist() const { return reinterpret_cast<unsigned*>(sm + Lay<T>::OFF_HIST); }
};

// One item: a tile's first row and column, and its bands [b0, b1).
struct Item {
    int i0, j0, b0, b1;
};
template <typename T>
__device__ __forceinline__ Item item_of(const K1Args<T>& a, int it, int gx, int gy) {
    const int bx = it % gx, r = it / gx;
    const int by = r % gy, bz = r / gy;
    Item m;
    m.i0 = by * TY;
    m.j0 = bx * TX;
    m.b0 = a.sp.o0 + bz * a.chunk;
    m.b1 = min(a.sp.o1, m.b0 + a.chunk);
    return m;
}

// Ring positions and phases of a warp that consumes bands (kept across items).
template <typename T>
struct Cons {
    Ring<Lay<T>::NYS> y;        // the next band's y-group
    Ring<Lay<T>::NWS> w;        // the current band's w
    int us = 0, ps = 0;         // u' slot of the next band, w' slot of the current one (16-bit)
    unsigned ev = 0;            // parity of the next barrier phase
    __device__ __forceinline__ void arrive(const Sm<T>& S) {
        // float32: slots freed by this phase are reloaded by TMA: order this
        // thread's generic accesses before those async-proxy writes
        if constexpr (Lay<T>::F32) fence_proxy_async_smem();
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(S.evt);
    }
    __device__ __forceinline__ bool wait(const Sm<T>& S) {
        const bool ok = k1_wait(S.evt, ev, S.abort);
        ev ^= 1u;
        return __all_sync(0xffffffffu, ok);
    }
};

// D^T y2 of one band at row gi, column gj of the image, from global memory (y2
// of the band at yv, yh): what D_s^T needs of the band before an item's first
template <typename T>
__device__ __forceinline__ float dty_global(const T* yv, const T* yh, int gi, int gj, const Geom& g) {
    const long long k = (long long)gi * g.p2 + gj;
    if (gi >= g.n1 || gj >= g.n2) return 0.f;
    float d = 0.f;
    if (gi >= 1) d += ldT(yv + k - g.p2);
    if (gi <= g.n1 - 2) d -= ldT(yv + k);
    if (gj >= 1) d += ldT(yh + k - 1);
    if (gj <= g.n2 - 2) d -= ldT(yh + k);
    return d;
}

// u step (Eq. 21) and u' of one band at tile position (r, c) in [0, TY] x
// [0, TX]: u' goes to upb, D^T y2 of the band replaces gprev (that of the
// band before); returns u+.  gb: the band's place in the whole cube.
template <typename T>
__device__ __forceinline__ float u_item(const K1Args<T>& a, const T* ys, float* upb, int gb, int r, int c, int gi,
                                        int gj, float cs, float& gprev) {
    using L = Lay<T>;
    constexpr int YPL = L::YPL;
    const Geom& g = a.g;
    const IterParams& P = a.p;
    const int kc = r * UC + c;
    if (gi >= g.n1 || gj >= g.n2) { upb[kc] = 0.f; gprev = 0.f; return 0.f; }
    const int k = (r + 2) * SW + (c + OX);
    float d1, gcur;                                 // D^T y1 and D^T y2 of the band
    {
        const T *v1 = ys + k, *h1 = ys + YPL + k, *v2 = ys + 2 * YPL + k, *h2 = ys + 3 * YPL + k;
        const float2 d = sub2(add2(sub2(f2(ldT(v1 - SW), ldT(v2 - SW)), f2(ldT(v1), ldT(v2))),
                                   f2(ldT(h1 - 1), ldT(h2 - 1))), f2(ldT(h1), ldT(h2)));
        d1 = d.x;
        gcur = d.y;
    }
    // D_s^T at the band's place in the whole cube (Neumann at its ends)
    float dst_ = 0.f;
    if (gb >= 1) dst_ += gprev;
    if (gb <= a.sp.n3g - 2) dst_ -= gcur;
    const int ku = r * SW + (c + OX);
    const float y4 = cs * ldT(ys + L::O_Q + ku);
    const float u = ldT(ys + L::O_U + ku);
    const float un = fminf(fmaxf(u - P.gamma_u * (d1 + dst_ + y4), P.mu_lo), P.mu_hi);
    upb[kc] = 2.f * un - u;
    gprev = gcur;
    return un;
}

// The eight dual entries that L reads at a grid position.
struct YN {
    float v00, vm0, v01, vm1, h00, h0m, h10, h1m;
};
template <typename T>
__device__ __forceinline__ YN load_yn(const T* yv, const T* yh) {
    YN y;
    y.v00 = ldT(yv); y.vm0 = ldT(yv - SW); y.v01 = ldT(yv + 1); y.vm1 = ldT(yv - SW + 1);
    y.h00 = ldT(yh); y.h0m = ldT(yh - 1); y.h10 = ldT(yh + SW); y.h1m = ldT(yh + SW - 1);
    return y;
}

// (L_v, L_h) at the three grids of one position: the dual entries themselves,
// the four-point means and the centred means.
__device__ __forceinline__ void l_pairs(const YN& y, bool mv, bool mh, float2 (&Lg)[3]) {
    // (v, h) pairs: the centred means 0.5 (v00 + vm0), 0.5 (h00 + h0m), and
    // the four-point means 0.25 (v00 + vm0 + v01 + vm1), 0.25 (h00 + h0m + h10 + h1m)
    float2 sum = add2(f2(y.v00, y.h00), f2(y.vm0, y.h0m));
    Lg[2] = mul2(sum, f2(0.5f, 0.5f));
    sum = add2(add2(sum, f2(y.v01, y.h10)), f2(y.vm1, y.h1m));
    const float2 four = mul2(sum, f2(0.25f, 0.25f));
    Lg[0] = f2(mv ? y.v00 : 0.f, mv ? four.y : 0.f);
    Lg[1] = f2(mh ? four.x : 0.f, mh ? y.h00 : 0.f);
}

// w step of one set (0 = w1, 1 = w2) from L y at each grid's position and the
// six w values wk (k = 2 grid + component): w+ replaces wk, w' goes to the
// set's planes 2 grid, 2 grid + 1 of wp at offset kw[grid] where L's output is
// not structurally zero (on[grid]), zero elsewhere: L^T then reads w' unmasked.
template <int SET, typename T>
__device__ __forceinline__ void w_step(const IterParams& P, const float2 (&Lg)[3], float (&wk)[6], float* wp,
                                       const int (&kw)[3], const bool (&on)[3]) {
    constexpr int WPL = Lay<T>::WPL;
    const float gam = SET ? P.gamma_w2 : P.gamma_w1;
    const float thr = SET ? P.thr_w2 : P.thr_w1;
#pragma unroll
    for (int gr = 0; gr < 3; ++gr) {
        const float wv = wk[2 * gr], wh = wk[2 * gr + 1];
        const float2 x = fma2(f2(gam, gam), Lg[gr], f2(wv, wh));
        const float xv = x.x, xh = x.y;
        // Eq. 24: max(1 - thr / ||x||, 0) x
        float sc;
        if constexpr (Lay<T>::F32) {
            // 1 / ||x|| from rsqrt
            const float n2 = xv * xv + xh * xh;
            sc = n2 > thr * thr ? fmaxf(1.f - thr * rsqrtf(n2), 0.f) : 0.f;
        } else {
            const float n = sqrtf(xv * xv + xh * xh);
            sc = n > thr ? 1.f - thr / n : 0.f;
        }
        const float2 nn = mul2(f2(sc, sc), x);
        wk[2 * gr] = nn.x;
        wk[2 * gr + 1] = nn.y;
        const float nv = 2.f * nn.x - wv, nh = 2.f * nn.y - wh;
        wp[(6 * SET + 2 * gr) * WPL + kw[gr]] = on[gr] ? nv : 0.f;
        wp[(6 * SET + 2 * gr + 1) * WPL + kw[gr]] = on[gr] ? nh : 0.f;
    }
}

// ---------------------------------------------------------------------------
// tile warps: one item
// ---------------------------------------------------------------------------
template <typename T, bool FIX, bool HIST>
__device__ __forceinline__ bool tile_item(const K1Args<T>& a, const Sm<T>& S, const Item& m, Cons<T>& C, K1Stat& A,
                                          Ordered& O, const K1Win& W, float cs, int turn) {
    using L = Lay<T>;
    constexpr int YPL = L::YPL, WPL = L::WPL, WRAW = L::WRAW;
    const Geom& g = a.g;
    const IterParams& P = a.p;
    const int tid = threadIdx.x;
    const unsigned cube = (unsigned)g.cube;        // 6 cubes < 2^32 elements (checked at handle creation)
    const unsigned plane = (unsigned)g.n1 * (unsigned)g.p2;
    const int r_t = tid / TX, c_t = tid % TX;
    const int gi = m.i0 + r_t, gj = m.j0 + c_t;
    const bool valid = gi < g.n1 && gj < g.n2;
    const unsigned o_t = valid ? (unsigned)gi * (unsigned)g.p2 + (unsigned)gj : 0u;
    const int ky = (r_t + 2) * SW + (c_t + OX), kw = (r_t + 1) * SW + (c_t + OX);
    const bool mv = gi < g.n1 - 1, mh = gj < g.n2 - 1;
    const unsigned it32 = L::F32 ? 0u : (unsigned)a.sc->iter;      // seeds the 16-bit rounding streams

    // ---- dual ascent of y1, y2 at this thread's voxel of band tb ----
    // Reads the band's completed w' (wp) and u' of the band (upb) and the next
    // (upn); yc: the voxel's y1 (v, h), y2 (v, h) of band tb.
    auto t_item = [&](int tb, const float* wp, const float* upb, const float* upn, const float (&yc)[4]) {
        if (!valid) return;
        const bool nxt = tb + 1 < g.n3;
        const int kc = r_t * UC + c_t;
        const float u0 = upb[kc];
        // (vertical, horizontal) pairs: D u' and D D_s u' at the voxel
        const float2 ub = f2(upb[kc + UC], upb[kc + 1]);
        const float2 du_ = sub2(ub, f2(u0, u0));
        const float2 du = f2(mv ? du_.x : 0.f, mh ? du_.y : 0.f);
        const float d0 = upn[kc] - u0;
        const float2 dd_ = sub2(sub2(f2(upn[kc + UC], upn[kc + 1]), ub), f2(d0, d0));
        const float2 dd = f2(nxt && mv ? dd_.x : 0.f, nxt && mh ? dd_.y : 0.f);
        const float* wk = wp + kw;
        float2 lt[2];                                    // (L^T w')_v, (L^T w')_h of each set
#pragma unroll
        for (int set = 0; set < 2; ++set) {
            auto Wk = [&](int k, int dr, int dc) { return wk[(6 * set + k) * WPL + dr * SW + dc]; };
            // v: W0 + 0.25 (W2(0,0) + W2(1,0) + W2(0,-1) + W2(1,-1)) + 0.5 (W4(0,0) + W4(1,0))
            // h: W3 + 0.25 (W1(0,0) + W1(0,1) + W1(-1,0) + W1(-1,1)) + 0.5 (W5(0,0) + W5(0,1))
            const float2 s4 = add2(add2(add2(f2(Wk(2, 0, 0), Wk(1, 0, 0)), f2(Wk(2, 1, 0), Wk(1, 0, 1))),
                                        f2(Wk(2, 0, -1), Wk(1, -1, 0))),
                                   f2(Wk(2, 1, -1), Wk(1, -1, 1)));
            const float2 s2 = add2(f2(Wk(4, 0, 0), Wk(5, 0, 0)), f2(Wk(4, 1, 0), Wk(5, 0, 1)));
            const float2 gg = fma2(f2(0.5f, 0.5f), s2, fma2(f2(0.25f, 0.25f), s4, f2(Wk(0, 0, 0), Wk(3, 0, 0))));
            lt[set] = f2(mv ? gg.x : 0.f, mh ? gg.y : 0.f);
        }
        const unsigned ob = (unsigned)tb * plane + o_t;
        const float2 y1 = fma2(f2(P.gamma_y1, P.gamma_y1), sub2(du, lt[0]), f2(yc[0], yc[1]));
        const float2 y2 = fma2(f2(P.gamma_y2, P.gamma_y2), sub2(dd, lt[1]), f2(yc[2], yc[3]));
        if constexpr (L::F32) {
            a.y1_n[ob] = y1.x;
            a.y1_n[cube + ob] = y1.y;
            a.y2_n[ob] = y2.x;
            a.y2_n[cube + ob] = y2.y;
        } else {
            SRStream sr(ob, it32, 3u);
            stS(a.y1_n + ob, y1.x, sr);
            stS(a.y1_n + (cube + ob), y1.y, sr);
            stS(a.y2_n + ob, y2.x, sr);
            stS(a.y2_n + (cube + ob), y2.y, sr);
        }
    };

    // ---- l1 window statistics of s~, t~ at this thread's voxel ----
    auto stats = [&](const T* ys, int b) {
        float xs = 0.f, xt = 0.f;
        if (valid) {
            // s~ = s - g_s y4, t~ = t - g_t (D_v^T y3 + y4), each product and
            // difference rounded once as in s_t_tilde (the light pass computes
            // the same values), the (s, t) pair packed
            const float qv = ldT(ys + L::O_Q + r_t * SW + (c_t + OX));
            const float y3v = ldT(ys + L::O_Y3 + (r_t + 1) * TX + c_t);
            const float y3u = gi >= 1 ? ldT(ys + L::O_Y3 + r_t * TX + c_t) : 0.f;
            const float y4 = __fmul_rn(cs, qv);
            const float dvt = __fsub_rn(y3u, gi <= g.n1 - 2 ? y3v : 0.f);
            const float2 mm = mul2(f2(P.gamma_s, P.gamma_t), f2(y4, __fadd_rn(dvt, y4)));
            const float2 x = sub2(f2(ldT(ys + L::O_S + r_t * TX + c_t), ldT(ys + L::O_T + r_t * TX + c_t)), mm);
            xs = x.x;
            xt = x.y;
        }
        // an inactive window has lo = hi = +inf: nothing is counted or taken
        const float x_s = fabsf(xs), x_t = fabsf(xt);
        const bool hs = valid && x_s > W.hi_s, ht = valid && x_t > W.hi_t;
        A.n_s += hs ? 1u : 0u;
        A.n_t += ht ? 1u : 0u;
        if constexpr (!L::F32) {
            S.above(C.us)[tid] = f2(hs ? x_s : -1.f, ht ? x_t : -1.f);
        } else {
            // both vectors' compensated sums in packed pairs; a value not
            // taken adds zero, which leaves the represented sum unchanged
            const float2 x2 = f2(hs ? x_s : 0.f, ht ? x_t : 0.f);
            if constexpr (FIX) {
                const float2 y2 = sub2(x2, A.kc);
                const float2 t2 = add2(A.ks, y2);
                A.kc = sub2(sub2(t2, A.ks), y2);
                A.ks = t2;
            } else {
                const float2 t2 = add2(A.ks, x2);
                const float2 b2 = sub2(t2, A.ks);
                A.kc = sub2(A.kc, add2(sub2(A.ks, sub2(t2, b2)), sub2(x2, b2)));
                A.ks = t2;
            }
        }
        const bool cs_ = valid && !hs && x_s > W.lo_s, ct_ = valid && !ht && x_t > W.lo_t;
        if (__ballot_sync(0xffffffffu, cs_ || ct_)) {     // most warps have no candidate
            append_shared(cs_, x_s, S.cbuf(0, turn & 1), S.cnt(0, turn & 1), a.l1.cand[0], &a.sc->acc[0].m);
            append_shared(ct_, x_t, S.cbuf(1, turn & 1), S.cnt(1, turn & 1), a.l1.cand[1], &a.sc->acc[1].m);
        }
        if constexpr (HIST) {
            // a 1/32 sample: a warp (one row of the tile) counts its 32 voxels
            // at one band in 32, the band rotating with the row and the tile
            // so that every band is sampled; the branch is warp-uniform, so
            // the other 31 band steps cost one test
            if ((((unsigned)b + 7u * (unsigned)r_t + 5u * (unsigned)(m.i0 >> 4) + 3u * (unsigned)(m.j0 >> 5)) & 31u) == 0u) {
                hist_add(W.hs && valid, x_s, W.hb_s, S.hist(), A.top_s);
                hist_add(W.ht && valid, x_t, W.hb_t, S.hist() + kK1Bins / 2, A.top_t);
            }
        }
    };
    const bool win = W.s || W.t;
    auto store_u = [&](unsigned ob, float un) {
        if constexpr (L::F32) a.u_n[ob] = un;
        else { SRStream sr(ob, it32, 2u); stS(a.u_n + ob, un, sr); }
    };

    // ---- band march, one barrier phase per band ----
    // The step before the first band computes u' of the first band only; it
    // shares the loop's code so that a launch fetches one copy of it (with
    // separate code for the first steps and the last ascent, a launch of a few
    // bands per CTA spent most of its time on instruction fetches).  u' of the
    // band past the cube's last one is computed from a stale slot and not
    // stored (its values are never used).
    float gprev = 0.f;
    if (m.b0 > 0) {
        const T* yv = a.y2 + (unsigned)(m.b0 - 1) * plane;
        gprev = dty_global(yv, yv + cube, gi, gj, g);
    }
    float yprev[4] = {0.f, 0.f, 0.f, 0.f};
    const int w_last = C.w.slot == 0 ? L::NWS - 1 : C.w.slot - 1;    // the previous item's last w
    int wslot_prev = w_last, ys_slot = 0, us_cur = 0, us_prev = 0;
    int piece = 0;
#pragma unroll 1
    for (int b = m.b0 - 1;; ++b) {
        const bool body = b >= m.b0, has_next = b + 1 < g.n3;
        if (b > m.b0) t_item(b - 1, S.wp(wslot_prev, C.ps ^ 1), S.up(us_prev), S.up(us_cur), yprev);
        if (b == m.b1) break;
        bool ok = true;
        if (body) ok = k1_wait(S.wfull + C.w.slot, C.w.ph, S.abort);
        if (has_next) ok = k1_wait(S.yfull + C.y.slot, C.y.ph, S.abort) && ok;
        if (!__all_sync(0xffffffffu, ok)) return false;    // warp-uniform: the statistics use warp votes
        const unsigned ob = (unsigned)b * plane + o_t;
        if (body) {
            const T* ys = S.yg(ys_slot);
            const T* wraw = S.wg(C.w.slot) + kw;
            float* wp = S.wp(C.w.slot, C.ps) + kw;
            if (!valid) {
#pragma unroll
                for (int k = 0; k < 12; ++k) wp[k * WPL] = 0.f;
            } else {
                // every operand before the first store (the compiler cannot
                // tell the shared-memory regions apart)
                float w1[6], w2[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    w1[k] = ldT(wraw + k * WRAW);
                    w2[k] = ldT(wraw + (6 + k) * WRAW);
                }
                const YN ya = load_yn(ys + ky, ys + YPL + ky);
                const YN yb = load_yn(ys + 2 * YPL + ky, ys + 3 * YPL + ky);
                yprev[0] = ya.v00; yprev[1] = ya.h00; yprev[2] = yb.v00; yprev[3] = yb.h00;
                // staged as zero where D is structurally zero (see
                // k1_tma_maps): the ascent leaves the stored values there
                if (!mv) { yprev[0] = ldT(a.y1 + ob); yprev[2] = ldT(a.y2 + ob); }
                if (!mh) { yprev[1] = ldT(a.y1 + (cube + ob)); yprev[3] = ldT(a.y2 + (cube + ob)); }
                float2 La[3], Lb[3];
                l_pairs(ya, mv, mh, La);
                l_pairs(yb, mv, mh, Lb);
                const int k3[3] = {0, 0, 0};
                const bool on[3] = {mv, mh, true};
                w_step<0, T>(P, La, w1, wp, k3, on);
                w_step<1, T>(P, Lb, w2, wp, k3, on);
                if constexpr (L::F32) {
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        a.w1_n[k * cube + ob] = w1[k];
                        a.w2_n[k * cube + ob] = w2[k];
                    }
                } else {
                    SRStream s1(ob, it32, 4u), s2(ob, it32, 5u);
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        stS(a.w1_n + (k * cube + ob), w1[k], s1);
                        stS(a.w2_n + (k * cube + ob), w2[k], s2);
                    }
                }
            }
        }
        const T* yn = S.yg(C.y.slot);
        const float un = u_item(a, yn, S.up(C.us), b + 1 + a.sp.band0, r_t, c_t, gi, gj, cs, gprev);
        C.arrive(S);
        const bool more = b + 1 < m.b1;
        if (valid && more) store_u(ob + plane, un);
        if (win && more) {
            stats(yn, b + 1);
            if constexpr (FIX) {
                if (++piece == a.unit || b + 2 == m.b1) { O.close(A.ks, A.kc); piece = 0; }
            }
        }
        if (!C.wait(S)) return false;
        if constexpr (!L::F32) {
            // band b, whose values every warp left before this phase (the slot
            // is written again two phases on)
            if (win && body && tid < TY * TX / 2) {
                const float2* x = S.above(us_cur) + tid;
                O.add(x[0]);
                O.add(x[TY * TX / 2]);
                if (++piece == a.unit || !more) { O.close(); piece = 0; }
            }
        }
        if (tid == 0) {
            // what every warp has finished with by now
            if (body) mbar_arrive(S.yempty + ys_slot);
            if (!more && has_next) mbar_arrive(S.yempty + C.y.slot);
            if (!L::F32) {
                if (body) mbar_arrive(S.wempty + C.w.slot);
            } else if (body ? b > m.b0 : turn > 0) {
                mbar_arrive(S.wempty + wslot_prev);
            }
        }
        us_prev = us_cur;
        us_cur = C.us;
        C.us = C.us == L::NUS - 1 ? 0 : C.us + 1;
        ys_slot = C.y.slot;
        if (has_next) C.y.next();
        if (body) {
            wslot_prev = C.w.slot;
            C.w.next();
            C.ps ^= 1;
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// ring warps: one item
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ bool ring_item(const K1Args<T>& a, const Sm<T>& S, const Item& m, Cons<T>& C, float cs) {
    using L = Lay<T>;
    constexpr int YPL = L::YPL, WRAW = L::WRAW;
    const Geom& g = a.g;
    const IterParams& P = a.p;
    const int q = (threadIdx.x >> 5) - kTileWarps, lane = threadIdx.x & 31;
    // w ring, a position per grid (row, column): grid 0 at (-1, c) and grids
    // 1, 2 at (TY, c) for a column c of the tile; grids 0, 2 at (r, TX) and
    // grid 1 at (r, -1) for a row r; the corners (-1, TX) of grid 0 and
    // (TY, -1) of grid 1.  A column of the ring walks rows 40 floats apart, so
    // rows r and r + 4 fall in one shared-memory bank: each warp takes half
    // the rows and half the columns.
    const bool has_w = lane < (q == 0 ? 25 : 24), has_u = has_w;
    int pr[3], pc[3];
    if (lane < 8) {
        pr[0] = pr[1] = pr[2] = 8 * q + lane;
        pc[0] = pc[2] = TX;
        pc[1] = -1;
    } else if (lane < 24) {
        pr[0] = -1;
        pr[1] = pr[2] = TY;
        pc[0] = pc[1] = pc[2] = 16 * q + lane - 8;
    } else {
        pr[0] = -1;
        pr[1] = pr[2] = TY;
        pc[0] = TX;
        pc[1] = pc[2] = -1;
    }
    // u' ring: the right column's rows and the row below
    const int ur = lane < 8 ? 8 * q + lane : TY, uc = lane < 8 ? TX : lane < 24 ? 16 * q + lane - 8 : TX;
    const int ui = m.i0 + ur, uj = m.j0 + uc;
    int gi[3], gj[3], ky[3], kw[3];
    bool in[3];                 // inside the image, and L's output not structurally zero
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        gi[k] = m.i0 + pr[k];
        gj[k] = m.j0 + pc[k];
        ky[k] = (pr[k] + 2) * SW + (pc[k] + OX);
        kw[k] = (pr[k] + 1) * SW + (pc[k] + OX);
        in[k] = gi[k] >= 0 && gi[k] < g.n1 && gj[k] >= 0 && gj[k] < g.n2;
    }
    const bool mv = gi[0] < g.n1 - 1, mh = gj[1] < g.n2 - 1;
    in[0] = in[0] && mv;
    in[1] = in[1] && mh;
    // L y of one set at the three positions (as l_pairs; the planes read
    // outside a position's grid stay in the staged boxes)
    auto ring_L = [&](const T* yv, const T* yh, float2 (&Lg)[3]) {
        auto V = [&](int k, int dr, int dc) { return ldT(yv + ky[k] + dr * SW + dc); };
        auto H = [&](int k, int dr, int dc) { return ldT(yh + ky[k] + dr * SW + dc); };
        const float h4 = 0.25f * (((H(0, 0, 0) + H(0, 0, -1)) + H(0, 1, 0)) + H(0, 1, -1));
        const float v4 = 0.25f * (((V(1, 0, 0) + V(1, -1, 0)) + V(1, 0, 1)) + V(1, -1, 1));
        Lg[0] = f2(mv ? V(0, 0, 0) : 0.f, mv ? h4 : 0.f);
        Lg[1] = f2(mh ? v4 : 0.f, mh ? H(1, 0, 0) : 0.f);
        Lg[2] = f2(0.5f * (V(2, 0, 0) + V(2, -1, 0)), 0.5f * (H(2, 0, 0) + H(2, 0, -1)));
    };

    float gprev = 0.f;
    if (has_u && m.b0 > 0) {
        const T* yv = a.y2 + (long long)(m.b0 - 1) * g.n1 * g.p2;
        gprev = dty_global(yv, yv + g.cube, ui, uj, g);
    }
    int ys_slot = 0;
#pragma unroll 1
    for (int b = m.b0 - 1; b < m.b1; ++b) {
        const bool body = b >= m.b0, has_next = b + 1 < g.n3;
        bool ok = true;
        if (body) ok = k1_wait(S.wfull + C.w.slot, C.w.ph, S.abort);
        if (has_next) ok = k1_wait(S.yfull + C.y.slot, C.y.ph, S.abort) && ok;
        if (!__all_sync(0xffffffffu, ok)) return false;
        if (body && has_w) {
            const T* ys = S.yg(ys_slot);
            const T* wraw = S.wg(C.w.slot);
            float* wp = S.wp(C.w.slot, C.ps);
            float w1[6], w2[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                w1[k] = ldT(wraw + k * WRAW + kw[k / 2]);
                w2[k] = ldT(wraw + (6 + k) * WRAW + kw[k / 2]);
            }
            float2 La[3], Lb[3];
            ring_L(ys, ys + YPL, La);
            ring_L(ys + 2 * YPL, ys + 3 * YPL, Lb);
            w_step<0, T>(P, La, w1, wp, kw, in);
            w_step<1, T>(P, Lb, w2, wp, kw, in);
        }
        if (has_u && has_next)
            u_item(a, S.yg(C.y.slot), S.up(C.us), b + 1 + a.sp.band0, ur, uc, ui, uj, cs, gprev);
        C.arrive(S);
        if (!C.wait(S)) return false;
        C.us = C.us == L::NUS - 1 ? 0 : C.us + 1;
        ys_slot = C.y.slot;
        if (has_next) C.y.next();
        if (body) {
            C.w.next();
            C.ps ^= 1;
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// load warps
// ---------------------------------------------------------------------------
// The groups of an item in the order they are asked for: each band's y-group
// and w, and the y-group of the band after the last (for its u').  issue_y
// (band, slot), issue_w(band, slot) fill a slot; wait_empty(bar, parity) waits
// for it to be free.  Returns false when a wait gave up.
template <typename T, typename FY, typename FW, typename FE>
__device__ __forceinline__ bool load_item(const Item& m, const Geom& g, Ring<Lay<T>::NYS>& y, Ring<Lay<T>::NWS>& w,
                                          const Sm<T>& S, FY&& issue_y, FW&& issue_w, FE&& wait_empty) {
    const int blast = min(m.b1, g.n3 - 1);
#pragma unroll 1
    for (int b = m.b0; b <= blast; ++b) {
        if (!wait_empty(S.yempty + y.slot, y.ph ^ 1u)) return false;
        issue_y(b, y.slot);
        y.next();
        if (b == m.b1) break;
        if (!wait_empty(S.wempty + w.slot, w.ph ^ 1u)) return false;
        issue_w(b, w.slot);
        w.next();
    }
    return true;
}

// float32: one thread issues bulk tensor copies
// (ny, nw: groups issued)
__device__ __forceinline__ void load_tma(const K1Maps& M, const K1Args<float>& a, const Sm<float>& S, int bid, int nblk,
                                         int items, int gx, int gy, unsigned& ny, unsigned& nw) {
    using L = Lay<float>;
    // bytes each group's copies deliver
    constexpr unsigned YG_TX = 4u * (4u * YR * SW + 2u * UR * SW + 2u * TY * TX + (TY + 1u) * TX);
    constexpr unsigned WG_TX = 4u * 12u * WR * SW;
    Ring<L::NYS> y;
    Ring<L::NWS> w;
    const Geom& g = a.g;
    bool ok = true;
    for (int it = bid; it < items && ok; it += nblk) {
        const Item m = item_of(a, it, gx, gy);
        ok = load_item<float>(
            m, g, y, w, S,
            [&](int band, int slot) {
                unsigned char* s = reinterpret_cast<unsigned char*>(S.yg(slot));
                uint64_t* bar = S.yfull + slot;
                mbar_arrive_expect_tx(bar, YG_TX);
                // (a cube of one row / column has no vertical / horizontal
                // differences: start past its map's one row / aligned column)
                const int iv = g.n1 > 1 ? m.i0 - 2 : 16, jh = g.n2 > 1 ? m.j0 - OX : 64;
                tma_load_3d(s + 0 * L::Y_B, &M.y1v, m.j0 - OX, iv, band, bar);
                tma_load_3d(s + 1 * L::Y_B, &M.y1h, jh, m.i0 - 2, band, bar);
                tma_load_3d(s + 2 * L::Y_B, &M.y2v, m.j0 - OX, iv, band, bar);
                tma_load_3d(s + 3 * L::Y_B, &M.y2h, jh, m.i0 - 2, band, bar);
                tma_load_3d(s + 4 * L::O_U, &M.u, m.j0 - OX, m.i0, band, bar);
                tma_load_3d(s + 4 * L::O_Q, &M.q, m.j0 - OX, m.i0, band, bar);
                tma_load_3d(s + 4 * L::O_S, &M.s, m.j0, m.i0, band, bar);
                tma_load_3d(s + 4 * L::O_T, &M.t, m.j0, m.i0, band, bar);
                tma_load_3d(s + 4 * L::O_Y3, &M.y3, m.j0, m.i0 - 1, band, bar);
                ny++;
            },
            [&](int band, int slot) {
                unsigned char* s = reinterpret_cast<unsigned char*>(S.wg(slot));
                uint64_t* bar = S.wfull + slot;
                mbar_arrive_expect_tx(bar, WG_TX);
                for (int k = 0; k < 6; ++k)
                    tma_load_3d(s + k * L::W_B, &M.w1, m.j0 - OX, m.i0 - 1, k * g.n3 + band, bar);
                for (int k = 0; k < 6; ++k)
                    tma_load_3d(s + (6 + k) * L::W_B, &M.w2, m.j0 - OX, m.i0 - 1, k * g.n3 + band, bar);
                nw++;
            },
            [&](uint64_t* bar, unsigned parity) { return k1_wait(bar, parity, S.abort); });
    }
}

// Waits (bounded) for the copies in flight to land, before the CTA gives its
// shared memory back after a wait gave up.
__device__ __forceinline__ void drain_tma(const Sm<float>& S, unsigned ny, unsigned nw) {
    using L = Lay<float>;
    for (unsigned k = 0; k < (unsigned)L::NYS && k < ny; ++k)
        (void)mbar_wait(S.yfull + (ny - 1u - k) % L::NYS, ((ny - 1u - k) / L::NYS) & 1u);
    for (unsigned k = 0; k < (unsigned)L::NWS && k < nw; ++k)
        (void)mbar_wait(S.wfull + (nw - 1u - k) % L::NWS, ((nw - 1u - k) / L::NWS) & 1u);
}

// 16-bit: the load warps copy 8 bytes (four columns) per lane and instruction, the
// first n of them from src and zero after (outside the image); a slot's full barrier counts every load thread.
__device__ __forceinline__ void cp8(void* dst, const void* src, int n) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
}
template <typename T>
__device__ __forceinline__ void load_async(const K1Args<T>& a, const Sm<T>& S, int bid, int nblk, int items, int gx,
                                           int gy) {
    using L = Lay<T>;
    constexpr int NL = 32 * L::LW;
    Ring<L::NYS> y;
    Ring<L::NWS> w;
    const Geom& g = a.g;
    const int lt = threadIdx.x - 32 * kConsWarps;
    const long long plane = (long long)g.n1 * g.p2;
    auto done = [&](uint64_t* bar) {
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
    };
    for (int it = bid; it < items; it += nblk) {
        const Item m = item_of(a, it, gx, gy);
        // `n` planes of `rows` rows from (row0, col0), `quads` quads a row:
        // plane k from base(k), into dst + k * stride; nr, nc: the image's rows
        // and columns, the rest is zero
        auto planes = [&](int n, int rows, int quads, int row0, int col0, T* dst, int stride, int nr, int nc,
                          auto&& base) {
            for (int e = lt; e < rows * quads; e += NL) {
                const int r = e / quads, c = 4 * (e - r * quads);
                const int gi = row0 + r, gj = col0 + c;
                const bool in = gi >= 0 && gi < nr && gj >= 0 && gj < nc;
                const int bytes = in ? min(nc - gj, 4) * L::ES : 0;
                const long long o = in ? (long long)gi * g.p2 + gj : 0;
                T* d = dst + r * 4 * quads + c;
                for (int k = 0; k < n; ++k) cp8(d + k * stride, base(k) + o, bytes);
            }
        };
        const bool ok = load_item<T>(
            m, g, y, w, S,
            [&](int band, int slot) {
                T* s = S.yg(slot);
                const long long bo = band * plane;
                // (y_v without the last row, y_h without the last column, as in k1_tma_maps)
                planes(2, YR, SW / 4, m.i0 - 2, m.j0 - OX, s, 2 * L::YPL, g.n1 - 1, g.n2,
                       [&](int k) { return (k ? a.y2 : a.y1) + bo; });
                planes(2, YR, SW / 4, m.i0 - 2, m.j0 - OX, s + L::YPL, 2 * L::YPL, g.n1, g.n2 - 1,
                       [&](int k) { return (k ? a.y2 : a.y1) + g.cube + bo; });
                planes(2, UR, SW / 4, m.i0, m.j0 - OX, s + L::O_U, L::O_Q - L::O_U, g.n1, g.n2,
                       [&](int k) { return (k ? a.q : a.u) + bo; });
                planes(2, TY, TX / 4, m.i0, m.j0, s + L::O_S, L::O_T - L::O_S, g.n1, g.n2,
                       [&](int k) { return (k ? a.t : a.s) + bo; });
                planes(1, TY + 1, TX / 4, m.i0 - 1, m.j0, s + L::O_Y3, 0, g.n1, g.n2, [&](int) { return a.y3 + bo; });
                done(S.yfull + slot);
            },
            [&](int band, int slot) {
                const long long bo = band * plane;
                planes(12, WR, SW / 4, m.i0 - 1, m.j0 - OX, S.wg(slot), L::WRAW, g.n1, g.n2,
                       [&](int k) { return (k < 6 ? a.w1 + k * g.cube : a.w2 + (k - 6) * g.cube) + bo; });
                done(S.wfull + slot);
            },
            [&](uint64_t* bar, unsigned parity) { return __all_sync(0xffffffffu, k1_wait(bar, parity, S.abort)); });
        if (!ok) break;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// One CTA of K1: items bid, bid + nblk, ... of the gx x gy x gz items (tiles
// by band runs) of one cube.
template <typename T, bool FIX = false>
__device__ __forceinline__ void k1_run(const K1Maps* maps, const K1Args<T>& a, const int bid, const int nblk,
                                       const int gx, const int gy, const int gz) {
    using L = Lay<T>;
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ unsigned ccnt[4];
    __shared__ int abort_flag;
    __shared__ float wred[kTileWarps * 12];
    const IterParams& P = a.p;
    const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
    const int items = gx * gy * gz;
    const Sm<T> S(sm, ccnt, &abort_flag);
    if (tid == 0) {
        const unsigned full = L::F32 ? 1u : 32u * L::LW;
        for (int k = 0; k < L::NYS; ++k) { mbar_init(S.yfull + k, full); mbar_init(S.yempty + k, 1); }
        for (int k = 0; k < L::NWS; ++k) { mbar_init(S.wfull + k, full); mbar_init(S.wempty + k, 1); }
        mbar_init(S.evt, kConsWarps);
        mbar_fence_init();
        for (int k = 0; k < 4; ++k) ccnt[k] = 0u;
        abort_flag = 0;
    }
    for (int k = tid; k < kK1Bins; k += L::NT) S.hist()[k] = 0u;
    __syncthreads();

    K1Win W;
    W.s = !P.tau_exact && a.sc->radius[0] > 0.0 && a.sc->ctl[0].window_ok;
    W.t = !P.tau_exact && a.sc->radius[1] > 0.0 && a.sc->ctl[1].window_ok;
    W.lo_s = W.s ? a.sc->ctl[0].theta_lo : INFINITY; W.hi_s = W.s ? a.sc->ctl[0].theta_hi : INFINITY;
    W.lo_t = W.t ? a.sc->ctl[1].theta_lo : INFINITY; W.hi_t = W.t ? a.sc->ctl[1].theta_hi : INFINITY;
    // the histograms: on after a recent miss
    W.hb_s = a.sc->ctl[0].hbase;
    W.hb_t = a.sc->ctl[1].hbase;
    // (float32 storage only: 16-bit storage searches as the cooperative kernel does;
    // sums in a fixed order: only where a piece fits the counters)
    const bool keep = L::F32 && (!FIX || a.unit * (TY * TX) <= 65535);
    W.hs = keep && W.s && a.sc->ctl[0].hist_left > 0 && hist_base_ok(W.hb_s);
    W.ht = keep && W.t && a.sc->ctl[1].hist_left > 0 && hist_base_ok(W.hb_t);
    const bool hist = W.hs || W.ht;
    K1Stat A;
    Ordered O;
    unsigned ny = 0, nw = 0;
    if (wid < kTileWarps) {
        const float cs = (float)(1.0 - a.sc->c[P.parity]);      // y4 = (1 - c) q
        Cons<T> C;
        int turn = 0;
        for (int it = bid; it < items; it += nblk, ++turn) {
            const Item m = item_of(a, it, gx, gy);
            const bool ok = hist ? tile_item<T, FIX, L::F32>(a, S, m, C, A, O, W, cs, turn)
                                 : tile_item<T, FIX, false>(a, S, m, C, A, O, W, cs, turn);
            if (!ok) break;
        }
    } else if (wid < kConsWarps) {
        const float cs = (float)(1.0 - a.sc->c[P.parity]);
        const int v = wid - kTileWarps;                         // warps 0, 1: vector v's candidates
        const bool mine = v == 0 ? W.s : v == 1 && W.t;
        Cons<T> C;
        int turn = 0;
        for (int it = bid; it < items; it += nblk, ++turn) {
            const Item m = item_of(a, it, gx, gy);
            if (!ring_item<T>(a, S, m, C, cs)) break;
            if (mine)
                flush_candidates(v, S.cbuf(v, turn & 1), S.cnt(v, turn & 1), a.sc, a.l1, v ? W.lo_t : W.lo_s,
                                 v ? W.hi_t : W.hi_s);
        }
    } else {
        if constexpr (L::F32) {
            if (lane == 0) load_tma(*maps, a, S, bid, nblk, items, gx, gy, ny, nw);
            __syncwarp();
        } else {
            load_async<T>(a, S, bid, nblk, items, gx, gy);
        }
    }
    __syncthreads();
    if (abort_flag) {                                           // a load never arrived
        if (tid == 0) atomicOr(&a.sc->error, 4);
        if constexpr (L::F32)
            if (tid == 32 * kConsWarps) drain_tma(S, ny, nw);
    }

    // this CTA among every CTA of the pass stage (all slabs of a split cube)
    const int cta = a.sp.cta_base + bid;
    if (W.s || W.t) {
        if (hist) {
            // the histogram joins the global one (unpacked, nonzero bins only)
            for (int k = tid; k < kK1Bins; k += L::NT) {
                const unsigned w = S.hist()[k];
                const int v = k / (kK1Bins / 2), b = 2 * (k - v * (kK1Bins / 2));
                unsigned* gh = a.l1.khist + v * kK1Bins + b;
                if (w & 0xffffu) atomicAdd(gh, w & 0xffffu);
                if (w >> 16) atomicAdd(gh + 1, w >> 16);
            }
        }
        // the CTA's window statistics (counts and sums above the windows) and
        // the histograms' above-range statistics, reduced together: 32-bit
        // counts and float-pair sums through the tile warps, then through
        // warp 0 (no FP64 outside one thread)
        if constexpr (!L::F32 || FIX) {
            A.ks = f2(O.hs, O.ht);
            A.kc = f2(-O.ls, -O.lt);
        }
        unsigned n4[4] = {A.n_s, A.n_t, A.top_s.n, A.top_t.n};
        float hi4[4] = {A.ks.x, A.ks.y, A.top_s.s, A.top_t.s};
        float lo4[4] = {-A.kc.x, -A.kc.y, 0.f, 0.f};
        auto reduce = [&](int from) {
            for (int o = from; o > 0; o >>= 1) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    n4[q] += __shfl_xor_sync(0xffffffffu, n4[q], o);
                    const float bh = __shfl_xor_sync(0xffffffffu, hi4[q], o);
                    const float bl = __shfl_xor_sync(0xffffffffu, lo4[q], o);
                    pair_add(hi4[q], lo4[q], bh, bl);
                }
            }
        };
        if (wid < kTileWarps) {
            reduce(16);
            if (lane == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    wred[wid * 12 + q] = __uint_as_float(n4[q]);
                    wred[wid * 12 + 4 + q] = hi4[q];
                    wred[wid * 12 + 8 + q] = lo4[q];
                }
            }
        }
        __syncthreads();
        if (wid == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                n4[q] = lane < kTileWarps ? __float_as_uint(wred[lane * 12 + q]) : 0u;
                hi4[q] = lane < kTileWarps ? wred[lane * 12 + 4 + q] : 0.f;
                lo4[q] = lane < kTileWarps ? wred[lane * 12 + 8 + q] : 0.f;
            }
            reduce(kTileWarps / 2);
            if (lane == 0) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    a.l1.k1_n[4 * cta + q] = n4[q];
                    a.l1.k1_s[4 * cta + q] = (double)hi4[q] + (double)lo4[q];
                }
            }
        }
    }
    // what this pass counted, for the finishing launch that follows (every
    // CTA agrees; the first writes it)
    if (cta == 0 && tid == 0) {
        constexpr int on = L::F32 ? 1 : 2;                      // 2: no histogram is ever kept
        a.sc->k1_win[0] = W.s ? on : 0; a.sc->k1_win[1] = W.t ? on : 0;
        a.sc->k1_hist[0] = W.hs; a.sc->k1_hist[1] = W.ht;
    }
}

__global__ void __launch_bounds__(Lay<float>::NT, 1) k1_tma(const __grid_constant__ K1Maps maps,
                                                            const __grid_constant__ K1Args<float> a, int gx, int gy,
                                                            int gz) {
    k1_run<float>(&maps, a, blockIdx.x, gridDim.x, gx, gy, gz);
}
__global__ void __launch_bounds__(Lay<float>::NT, 1) k1_tma_fixed(const __grid_constant__ K1Maps maps,
                                                                  const __grid_constant__ K1Args<float> a, int gx,
                                                                  int gy, int gz) {
    k1_run<float, true>(&maps, a, blockIdx.x, gridDim.x, gx, gy, gz);
}
template <typename T>
__global__ void __launch_bounds__(Lay<T>::NT, 1) k1_half(const __grid_constant__ K1Args<T> a, int gx, int gy, int gz) {
    k1_run<T>(nullptr, a, blockIdx.x, gridDim.x, gx, gy, gz);
}

// K1 over many cubes in one launch: the cube of a CTA from a table of first
// CTAs, its arguments from the table, its tensor maps from device memory.
struct K1BatchTab {
    int n;
    int start[kBatchMax + 1];
    int gx[kBatchMax], gy[kBatchMax], gz[kBatchMax];
    const K1Maps* maps[kBatchMax];
    K1Args<float> args[kBatchMax];
};

__device__ __forceinline__ int batch_cube_of(const int* start, int n, int blk) {
    int lo = 0, hi = n - 1;                 // the last cube whose first CTA is <= blk
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= blk) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(Lay<float>::NT, 1) k1_tma_batch(const __grid_constant__ K1BatchTab t) {
    const int c = batch_cube_of(t.start, t.n, blockIdx.x);
    // the cube's arguments where they lie, in the constant bank: a copy of them
    // went to local memory (96 registers are all in use), and its loads lengthened
    // every band step (464 against 306 us a launch for eight cubes of 0.05 to
    // 4.2 million voxels)
    const K1Args<float>& a = t.args[c];
    if (__ldcg(&a.sc->done)) return;        // this cube has stopped
    const K1Maps* maps = t.maps[c];
    if (threadIdx.x == 32 * kConsWarps) {
        // the cube's tensor maps sit in global memory (the copies' descriptors)
        tma_prefetch_map(&maps->y1v); tma_prefetch_map(&maps->y1h); tma_prefetch_map(&maps->y2v);
        tma_prefetch_map(&maps->y2h); tma_prefetch_map(&maps->w1); tma_prefetch_map(&maps->w2); tma_prefetch_map(&maps->u); tma_prefetch_map(&maps->q);
        tma_prefetch_map(&maps->s); tma_prefetch_map(&maps->t); tma_prefetch_map(&maps->y3);
    }
    k1_run<float>(maps, a, blockIdx.x - t.start[c], t.start[c + 1] - t.start[c], t.gx[c], t.gy[c], t.gz[c]);
}

// ---------------------------------------------------------------------------
// host: how a cube is split
// ---------------------------------------------------------------------------
// Band steps that an item costs beyond its bands: u' of its first band, the
// copies of the bands before and after it, and the wait for its first planes.
constexpr double kItemCost = 1.5;

int tiles_of(const Geom& g) { return ((g.n2 + TX - 1) / TX) * ((g.n1 + TY - 1) / TY); }

// Band steps of the slowest of `ctas` CTAs when `tiles` tiles of nb bands run
// as items of len bands.
double run_cost(int nb, int tiles, int len, int ctas) {
    const long long items = (long long)tiles * ((nb + len - 1) / len);
    return (double)((items + ctas - 1) / ctas) * (len + kItemCost);
}

// The fewest runs of nb bands that are shorter than len (past nb where none is): the
// next split to look at, so that a launch's plan takes some 2 sqrt(nb) steps.
int next_split(int nb, int len) { return len > 1 ? (nb + len - 2) / (len - 1) : nb + 1; }

// Bands per item for `ctas` persistent CTAs: the split of the bands (in multiples
// of unit) whose slowest CTA does the fewest band steps.
int best_run(int nb, int tiles, int ctas, int unit = 1) {
    int best_len = std::min(nb, kMaxRun);
    double best = 1e30;
    int prev = 0;
    for (int runs = 1, next; runs <= nb; runs = next) {
        int len = (nb + runs - 1) / runs;
        next = next_split(nb, len);
        len = (len + unit - 1) / unit * unit;
        if (len == prev || (len > kMaxRun && unit == 1)) continue;
        prev = len;
        const double c = run_cost(nb, tiles, len, ctas);
        if (c < best * (1.0 - 1e-12)) { best = c; best_len = len; }
    }
    return best_len;
}

// One launch's split: bands per item and CTAs.  One CTA per SM, and more only
// for cubes so large that a CTA's sampled histogram could pass its 16-bit
// counters (an item counts at most 512 voxels for every 32 of its bands).
struct Plan {
    int chunk, gz, ctas;
};
Plan k1_plan(const Geom& g, int nb, int chunk, int ctas) {
    Plan p;
    const int tiles = tiles_of(g);
    p.chunk = chunk >= 1 && chunk <= std::min(nb, kMaxRun) ? chunk : best_run(nb, tiles, ctas);
    p.gz = (nb + p.chunk - 1) / p.chunk;
    const long long items = (long long)tiles * p.gz;
    const long long per = std::max(1, 127 / ((p.chunk + 31) / 32));       // items a CTA may count
    p.ctas = (int)std::min(items, std::max((long long)ctas, (items + per - 1) / per));
    return p;
}

// 16-bit storage: items of whole pieces of the window's sums (no histogram, so
// no limit on the run or the items a CTA takes).
Plan k1_plan_half(const Geom& g, int nb) {
    Plan p;
    const int tiles = tiles_of(g);
    p.chunk = best_run(nb, tiles, device_sms(), k1_coop_chunk(g));
    p.gz = (nb + p.chunk - 1) / p.chunk;
    p.ctas = (int)std::min<long long>((long long)tiles * p.gz, device_sms());
    return p;
}

// float32 sums in their fixed order: the bands of a piece.  Runs of at least 8
// bands, or all of fewer, chosen as if each piece were a CTA of its own: the split
// whose last wave leaves the least of the SMs idle, a CTA's start counted as 1.5
// bands.  Part of what the sums are, so it follows no measurement.
int fixed_piece(int nb, int tiles) {
    const double sms = (double)device_sms();
    int len_best = nb;
    double best = 1e30;
    for (int runs = 1, next; runs <= std::max(1, nb / 8); runs = next) {
        const int len = (nb + runs - 1) / runs;
        next = next_split(nb, len);
        const double units = (double)tiles * ((nb + len - 1) / len);
        const double waves = std::ceil(units / sms);
        const double waste = (waves - units / sms) / waves + 1.5 / len;
        if (waste < best - 1e-12) { best = waste; len_best = len; }
    }
    return len_best;
}
// Items of whole pieces; with a histogram (see k1_run) within its counters as in k1_plan.
Plan k1_plan_fixed(const Geom& g, int nb) {
    Plan p;
    const int tiles = tiles_of(g), unit = fixed_piece(nb, tiles);
    p.chunk = best_run(nb, tiles, device_sms(), unit);
    if (unit * (TY * TX) <= 65535) p.chunk = std::min(p.chunk, kMaxRun / unit * unit);
    p.gz = (nb + p.chunk - 1) / p.chunk;
    const long long items = (long long)tiles * p.gz;
    const long long per = std::max(1, 127 / ((p.chunk + 31) / 32));
    p.ctas = (int)std::min(items, std::max((long long)device_sms(), (items + per - 1) / per));
    return p;
}
Plan k1_plan_of(int storage, const Geom& g, int nb, int chunk, int fixed_sums) {
    return storage != 0 ? k1_plan_half(g, nb) : fixed_sums ? k1_plan_fixed(g, nb) : k1_plan(g, nb, chunk, device_sms());
}

}  // namespace

// CTAs of the largest launch any run length gives: the per-CTA statistics
// arrays are sized for it.
int k1_tma_ctas(const Geom& g) {
    return std::max(device_sms(), tiles_of(g) * ((g.n3 + std::min(8, g.n3) - 1) / std::min(8, g.n3)));
}

// Run lengths worth timing: those of at least 8 bands (all of them when there are
// fewer), the model's choice first, then the next best by its estimate, at most
// `cap` distinct lengths.
int k1_tma_chunk_candidates(const Geom& g, int* out, int cap) {
    const int tiles = tiles_of(g), sms = device_sms();
    std::vector<std::pair<double, int>> c;
    for (int runs = 1; runs <= std::max(1, g.n3 / 8); ++runs) {
        const int len = (g.n3 + runs - 1) / runs;
        if (len > kMaxRun || (!c.empty() && c.back().second == len)) continue;
        c.push_back({run_cost(g.n3, tiles, len, sms), len});
    }
    std::stable_sort(c.begin(), c.end(), [](const auto& x, const auto& y) { return x.first < y.first; });
    const int first = best_run(g.n3, tiles, sms);
    int n = 0;
    if (cap > 0 && first >= std::min(8, g.n3)) out[n++] = first;
    for (const auto& e : c)
        if (n < cap && e.second != first) out[n++] = e.second;
    return n;
}

int k1_tma_configure(int storage) {
    cudaError_t e = cudaErrorInvalidValue;
    switch (storage) {
        case 0:
            e = cudaFuncSetAttribute(k1_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<float>::SMEM);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k1_tma_fixed, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<float>::SMEM);
            break;
        case 1: e = cudaFuncSetAttribute(k1_half<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<__nv_bfloat16>::SMEM); break;
        case 2: e = cudaFuncSetAttribute(k1_half<__half>, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<__half>::SMEM); break;
    }
    return e == cudaSuccess ? 0 : -3;
}

// tensor maps over the current-parity buffers of one iteration (float32)
int k1_tma_maps(const Geom& g, const IterBufs& b, K1Maps* m) {
    int rc = 0;
    // y_v without its last row and y_h without its last column (where D is
    // structurally zero and L and D^T read them as zero): the copies' zero fill
    // then masks them, and no load in the kernel needs a test
    const float *y1 = (const float*)b.y1, *y2 = (const float*)b.y2;
    const int rv = std::max(g.n1 - 1, 1), ch = std::max(g.n2 - 1, 1);
    rc |= tma_encode_cubes(&m->y1v, y1, g, rv, g.n2, 1, SW, YR);
    rc |= tma_encode_cubes(&m->y1h, y1 + g.cube, g, g.n1, ch, 1, SW, YR);
    rc |= tma_encode_cubes(&m->y2v, y2, g, rv, g.n2, 1, SW, YR);
    rc |= tma_encode_cubes(&m->y2h, y2 + g.cube, g, g.n1, ch, 1, SW, YR);
    rc |= tma_encode_cubes(&m->w1, b.w1, g, g.n1, g.n2, 6, SW, WR);
    rc |= tma_encode_cubes(&m->w2, b.w2, g, g.n1, g.n2, 6, SW, WR);
    rc |= tma_encode_cubes(&m->u, b.u, g, g.n1, g.n2, 1, SW, UR);
    rc |= tma_encode_cubes(&m->q, b.q, g, g.n1, g.n2, 1, SW, UR);
    rc |= tma_encode_cubes(&m->s, b.s, g, g.n1, g.n2, 1, TX, TY);
    rc |= tma_encode_cubes(&m->t, b.t, g, g.n1, g.n2, 1, TX, TY);
    rc |= tma_encode_cubes(&m->y3, b.y3, g, g.n1, g.n2, 1, TX, TY + 1);
    return rc ? -3 : 0;
}

int k1_tma_part_chunk(const Geom& g, const SlabPart& sp, int chunk) {
    return sp.o1 > sp.o0 ? k1_plan(g, sp.o1 - sp.o0, chunk, device_sms()).chunk : 0;
}

int k1_tma_grid(int storage, const Geom& g, const SlabPart& sp, int chunk, int fixed_sums) {
    return sp.o1 > sp.o0 ? k1_plan_of(storage, g, sp.o1 - sp.o0, chunk, fixed_sums).ctas : 0;
}

namespace {
template <typename T>
K1Args<T> k1_args(const Geom& g, const IterBufs& b, const IterParams& p, Scal* sc, const L1Work& w, int chunk,
                  const SlabPart& sp) {
    K1Args<T> a;
    a.g = g;
    a.u = (const T*)b.u; a.q = (const T*)b.q; a.s = (const T*)b.s; a.t = (const T*)b.t; a.y3 = (const T*)b.y3;
    a.y1 = (const T*)b.y1; a.y2 = (const T*)b.y2; a.w1 = (const T*)b.w1; a.w2 = (const T*)b.w2;
    a.u_n = (T*)b.u_n; a.w1_n = (T*)b.w1_n; a.w2_n = (T*)b.w2_n; a.y1_n = (T*)b.y1_n; a.y2_n = (T*)b.y2_n;
    a.p = p;
    a.sc = sc;
    a.l1 = w;
    a.chunk = chunk;
    a.unit = 0;
    a.sp = sp;
    return a;
}
}  // namespace

// How the cubes of a batch share the SMs.  Within a number of CTAs, each cube gets
// the fewest with which none of its CTAs does more than some number of band steps,
// the same for all cubes (bisection on it).  With one CTA per SM that number is the
// launch's time: best for a few cubes.  Many cubes leave most SMs with less than it
// (a small cube's CTA ends early and nothing follows), so that several times as many
// CTAs, which follow one another on the SMs, are weighed against it: their total
// steps spread over the SMs, half a CTA for the last ones, a start for each.  (64
// cubes of 0.05 to 59 million voxels: one CTA per SM 17.2 ms a launch, 16 times that
// 10.6; the 8 cubes of 0.05 to 4.2 million: 0.27 and 0.36 ms.)
constexpr double kCtaCost = 2.0;              // band steps that a CTA's start costs

void k1_batch_plan(BatchCube* cubes, int n) {
    const int sms = device_sms();
    struct Run { int len; long long items; };
    std::vector<std::vector<Run>> runs(n);
    double all = 0.0;
    for (int c = 0; c < n; ++c) {
        const BatchCube& q = cubes[c];
        const int nb = q.g.n3, tiles = tiles_of(q.g);
        const bool own = q.k1_chunk >= 1 && q.k1_chunk <= nb;      // the cube's own (autotuned) run
        for (int k = 1, len; k <= nb; k = own ? nb + 1 : next_split(nb, len)) {
            len = own ? q.k1_chunk : (nb + k - 1) / k;
            if (len <= kMaxRun) runs[c].push_back({len, (long long)tiles * ((nb + len - 1) / len)});
        }
        all += (double)tiles * (nb + kItemCost);
    }
    // the fewest CTAs with which cube c stays within `steps` band steps, and its run
    auto fewest = [&](int c, double steps, Run* best) -> long long {
        long long ctas = 1ll << 40;
        for (const Run& r : runs[c]) {
            const long long per = (long long)(steps / (r.len + kItemCost));
            if (per < 1) continue;
            const long long k = (r.items + per - 1) / per;
            if (k < ctas) { ctas = k; *best = r; }
        }
        return ctas;
    };
    std::vector<Plan> plan(n), best_plan(n);
    double best = 1e300;
    for (int wave = 1; wave <= 32; wave *= 2) {
        const long long budget = (long long)wave * std::max(sms, n);
        double lo = 0.0, hi = 1.0 + 2.0 * all;
        Run r{1, 1};
        for (int k = 0; k < 40 && hi - lo > 1e-3 * hi; ++k) {
            const double mid = 0.5 * (lo + hi);
            long long sum = 0;
            for (int c = 0; c < n && sum <= budget; ++c) sum += fewest(c, mid, &r);
            if (sum <= budget) hi = mid; else lo = mid;
        }
        double total = 0.0;
        for (int c = 0; c < n; ++c) {
            const BatchCube& q = cubes[c];
            r = Run{std::min(q.g.n3, kMaxRun), 1};
            // (the statistics of a cube's CTAs have k1_ctas places)
            const int want = (int)std::max(1ll, std::min({fewest(c, hi, &r), budget, (long long)q.k1_ctas}));
            plan[c] = k1_plan(q.g, q.g.n3, r.len, want);
            total += (double)tiles_of(q.g) * plan[c].gz * (plan[c].chunk + kItemCost) + kCtaCost * plan[c].ctas;
        }
        const double t = wave == 1 ? hi + kCtaCost : total / sms + 0.5 * hi;
        if (t < best) { best = t; best_plan.swap(plan); }
    }
    for (int c = 0; c < n; ++c) cubes[c].k1 = K1Split{best_plan[c].chunk, best_plan[c].gz, best_plan[c].ctas};
}

int launch_k1_batch(const BatchCube* cubes, int n, cudaStream_t st) {
    if (n < 1 || n > kBatchMax) return -1;
    static_assert(sizeof(K1BatchTab) <= 32000, "kernel parameter space");
    K1BatchTab t{};
    t.n = n;
    int total = 0;
    for (int c = 0; c < n; ++c) {
        const BatchCube& q = cubes[c];
        t.args[c] = k1_args<float>(q.g, q.b, q.p, q.sc, q.l1, q.k1.chunk, whole_cube(q.g));
        const int tx = (q.g.n2 + TX - 1) / TX, ty = (q.g.n1 + TY - 1) / TY;
        t.gx[c] = tx; t.gy[c] = ty; t.gz[c] = q.k1.gz;
        t.maps[c] = q.maps;
        t.start[c] = total;
        total += q.k1.ctas;
    }
    t.start[n] = total;
    k1_tma_batch<<<total, Lay<float>::NT, Lay<float>::SMEM, st>>>(t);
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

int k1_batch_configure() {
    const cudaError_t e = cudaFuncSetAttribute(k1_tma_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<float>::SMEM);
    return e == cudaSuccess ? 0 : -3;
}

int launch_k1_tma(int storage, const Geom& g, const K1Maps& m, const IterBufs& b, const IterParams& p,
                  Scal* sc, const L1Work& w, int chunk, const SlabPart& sp, cudaStream_t st) {
    const int nb = sp.o1 - sp.o0;
    if (nb <= 0 || sp.o0 < 0 || sp.o1 > g.n3) return -1;
    const Plan pl = k1_plan_of(storage, g, nb, chunk, p.fixed_sums);
    const int gx = (g.n2 + TX - 1) / TX, gy = (g.n1 + TY - 1) / TY;
    auto half = [&](auto zero) {
        using T = decltype(zero);
        K1Args<T> args = k1_args<T>(g, b, p, sc, w, pl.chunk, sp);
        args.unit = k1_coop_chunk(g);
        k1_half<T><<<pl.ctas, Lay<T>::NT, Lay<T>::SMEM, st>>>(args, gx, gy, pl.gz);
    };
    switch (storage) {
        case 0: {
            K1Args<float> args = k1_args<float>(g, b, p, sc, w, pl.chunk, sp);
            args.unit = p.fixed_sums ? fixed_piece(nb, gx * gy) : 0;
            if (p.fixed_sums) k1_tma_fixed<<<pl.ctas, Lay<float>::NT, Lay<float>::SMEM, st>>>(m, args, gx, gy, pl.gz);
            else k1_tma<<<pl.ctas, Lay<float>::NT, Lay<float>::SMEM, st>>>(m, args, gx, gy, pl.gz);
            break;
        }
        case 1: half(__nv_bfloat16()); break;
        case 2: half(__half()); break;
        default: return -1;
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -3;
}

}  // namespace gsstv
