// Warp-wide walk along listmode events on 3D grids: two lanes per voxel plane,
// images held as z pairs.
//
// Images.  The image the events read and the accumulator they add to hold
// one 8-byte pair per voxel: (value of voxel j, value of voxel j + nx*ny).  A
// sample of an x- or y-principal event has its z neighbours in one pair, so it
// takes two 8-byte gathers and two 8-byte vector atomics instead of four
// scalar ones, and both families use the one image.  Where the rows and
// columns are multiples of 4 the pairs of a slice are stored in 4 x 4 bricks
// (one 128-byte line) of 2 x 2 sectors (32 bytes), x fastest at each level,
// so that lines along x, y or between touch equally few of them; other grids
// keep rows (lmh::PairLay).
//
// Lanes.  A warp takes an event's voxel planes along its principal axis
// sixteen per pass: lanes 2j and 2j + 1 sit on plane j of the pass, on the
// voxels A and A + 1 of the first secondary axis.  What bounds these kernels is
// the path from the SM to L2: one cycle per 128-byte line that a gather
// touches and per 32-byte sector that an atomic touches.  With one plane per
// lane the 32 planes of a request drift over 1 + 32 s rows (s: slope in A),
// for A and again for A + 1; sixteen planes with both neighbours touch 2 + 16 s
// rows once.
//
// Two events are in flight per warp: their gathers are issued back to back,
// one shuffle tree reduces both sums and the dual step runs once for both (a
// half-warp each).  The events' parameters are staged in shared memory, one
// 64-byte record each, with what does not depend on the lane worked out by
// the staging lane (one event per lane).
#pragma once
#include "lm_internal.h"

namespace lmw {

using namespace lmk;
using lmh::TOF_TAB_N;

constexpr float MAGIC = 12582912.0f;    // 1.5 * 2^23: adding it leaves a float whose unit in the last place is 1
constexpr unsigned MAGIC_BITS = 0x4B400000u;
constexpr int PASSES = 4;               // planes kept in registers: 4 passes of 16
constexpr int TAB_PAD = TOF_TAB_N + 2;  // table entries -1 .. TOF_TAB_N
constexpr unsigned NONE = 0xFFFFFFFFu;  // byte offset of a lane without a sample

// One event of a chunk.
struct alignas(16) Rec {
    float4 g0;      // ua0, sa, ub0, sb: secondary coordinates at plane i are ua0 + i sa, ub0 + i sb
    float4 g1;      // tau0, dtau (TOF coordinate, mm); c_e step / mu_e; S_e
    float4 d;       // c_e step, s_e, y_e, mu_e
    int i0;         // the first plane
    unsigned meta;  // planes (15 bits), principal axis (2), REC_INNER, place in the chunk (5 bits from 20)
    int pad[2];
};

constexpr unsigned REC_INNER = 1u << 17;  // every sample has its four neighbours inside the grid

// Where a sample's TOF weight comes from.
enum Tof {
    NO_TOF,      // weight 1
    TOF_TABLE,   // linear interpolation of the state's table (data updates)
    TOF_SERIES,  // standalone projections: second-order expansion about the nearest node of the block's own table
    TOF_ERF,     // the same without a table: the two lanes of a plane take one erf each
};

// Nodes of the block's own table over [0, W] (the kernel is even).  The
// expansion's remainder, dt^3 |w'''| / 48 with dt = W / SERIES_N, is 2.7e-8 of
// the peak at the widest cut it serves and 0.7e-9 at 3 sigma, less than the
// rounding of an erf; wider cuts take TOF_ERF.  Measured against 64 bits over 1e6
// samples at 3 sigma: largest error 5.1e-8, rms 1.3e-8 (an erf difference per
// sample: 5.4e-8, 1.7e-8); whole calls over 357 143 events on the 200 x 200 x 96
// grid: forward 124 us, back 144 us (with TOF_ERF 157 and 163 us).
constexpr int SERIES_N = 1024;
constexpr float SERIES_SIGMAS = 10.0f;

// The TOF table in shared memory as (value, slope) pairs, with one entry of
// margin at either end: the table coordinate of a sample with |tau| <= W is
// within rounding of [0, TOF_TAB_N].
__device__ __forceinline__ void fill_tab(float2* s_tab, const float* __restrict__ tab)
{
#pragma unroll 4
    for (int k = threadIdx.x; k < TAB_PAD; k += blockDim.x) {
        const float a = __ldg(tab + min(max(k - 1, 0), TOF_TAB_N));
        const float b = __ldg(tab + min(k, TOF_TAB_N));
        s_tab[k] = make_float2(a, b - a);
    }
}

// The block's own table: weight and its first two Taylor coefficients (per
// mm, per mm^2).  erf where its arguments are small and erfc in the tail, each
// where it is the more accurate.  Ends with a barrier.
__device__ __forceinline__ void make_series(float4* s_ser, const Geo& G)
{
    const float hb = 0.5f * G.bin, dt = G.W / (float)SERIES_N, g = 0.564189584f * G.inv_s;  // 1/sqrt(pi)
    for (int k = threadIdx.x; k <= SERIES_N; k += blockDim.x) {
        const float p = fmaf(dt, (float)k, hb) * G.inv_s, q = fmaf(dt, (float)k, -hb) * G.inv_s;
        const float w = 0.5f * (q > 0.5f ? erfcf(q) - erfcf(p) : erff(p) - erff(q));
        const float ep = expf(-p * p), eq = expf(-q * q);
        s_ser[k] = make_float4(w, g * (ep - eq), g * G.inv_s * (q * eq - p * ep), 0.0f);
    }
    __syncthreads();
}

// Trims the plane range of a traversal (lor_setup widens it by a plane on
// each side) to the planes with a sample: |tau| <= W and a neighbour inside
// the grid.  The coordinates are monotone in the plane, so these planes are
// consecutive and the two ends decide for all; evaluated with the walk's own
// arithmetic.  *inner: every sample has its four neighbours inside the grid.
__device__ __forceinline__ bool plane_counts(const Geo& G, const Lor& L, int i)
{
    const float fi = (float)i;
    if (G.tof_on && !(fabsf(fmaf(fi, L.dtau, L.tau0)) <= G.W)) return false;
    const float fa = floorf(fmaf(fi, L.sa, L.ua0)), fb = floorf(fmaf(fi, L.sb, L.ub0));
    return fa >= -1.0f && fa < (float)L.nA && fb >= -1.0f && fb < (float)L.nB;
}

__device__ __forceinline__ void trim(const Geo& G, Lor& L, bool* inner)
{
    int lo = L.i0, hi = L.i0 + L.cnt - 1;
    while (lo <= hi && !plane_counts(G, L, lo)) ++lo;
    while (hi > lo && !plane_counts(G, L, hi)) --hi;
    L.i0 = lo;
    L.cnt = hi - lo + 1;
    bool in = L.cnt > 0 && L.k != 2;
    for (int e = 0; e < 2; ++e) {
        const float fi = (float)(e ? hi : lo);
        const float fa = floorf(fmaf(fi, L.sa, L.ua0)), fb = floorf(fmaf(fi, L.sb, L.ub0));
        in = in && fa >= 0.0f && fa < (float)(L.nA - 1) && fb >= 0.0f && fb < (float)(L.nB - 1);
    }
    *inner = in;
}

// Constants of the calling lane and of the launch.
struct Lane {
    float fpl;           // plane within a pass
    int pl;
    int par;             // 0: voxel A, 1: voxel A + 1
    float sgn, off;      // weight along A: off + sgn * frac
    unsigned tab;        // shared-memory address of table entry or node 0, minus that of the MAGIC bits
    float W, inv_dt;     // TOF_TABLE: coordinate (tau + W) inv_dt; TOF_SERIES: |tau| inv_dt
    float dt;            // TOF_SERIES: node spacing (W / 2^10, exact)
    float hb, inv_s;     // TOF_ERF: the lane's edge of the bin, (tau + hb) inv_s
};

__device__ __forceinline__ Lane make_lane()
{
    Lane l;
    const int lane = threadIdx.x & 31;
    l.pl = lane >> 1;
    l.fpl = (float)l.pl;
    l.par = lane & 1;
    l.sgn = l.par ? 1.0f : -1.0f;
    l.off = l.par ? 0.0f : 1.0f;
    return l;
}

__device__ __forceinline__ Lane table_lane(const float2* s_tab, float W)
{
    Lane l = make_lane();
    l.tab = (unsigned)__cvta_generic_to_shared(s_tab) + 8u - (MAGIC_BITS << 3);
    l.W = W;
    l.inv_dt = (float)TOF_TAB_N / (2.0f * W);
    return l;
}

// TOF_SERIES and TOF_ERF (which has no table).
__device__ __forceinline__ Lane op_lane(const float4* s_ser, const Geo& G)
{
    Lane l = make_lane();
    l.tab = (unsigned)__cvta_generic_to_shared(s_ser) - (MAGIC_BITS << 4);
    l.dt = G.W / (float)SERIES_N;
    l.inv_dt = (float)SERIES_N / G.W;
    l.hb = (l.par ? -0.5f : 0.5f) * G.bin;
    l.inv_s = G.inv_s;
    return l;
}

// Packs a traversal into a record (the per-event values are the caller's).
__device__ __forceinline__ void rec_path(const float4& g0, float tau0, float dtau, int i0, int cnt, int k, bool inner,
                                         int place, Rec& r)
{
    r.g0 = g0;
    r.g1.x = tau0;
    r.g1.y = dtau;
    r.i0 = i0;
    r.meta = (unsigned)cnt | ((unsigned)k << 15) | (inner ? REC_INNER : 0u) | ((unsigned)place << 20);
}

// The samples of one event held by a lane: byte offset of its pair (NONE: no
// sample) and the weights of the pair's halves, without the sample length
// and c_e, which are the event's.
struct Held {
    unsigned off[PASSES];
    float q0[PASSES], q1[PASSES];
};

// TOF weight at plane fi from the shared-memory table.
__device__ __forceinline__ float tof_at(const Lane& l, float tau0, float dtau, float fi)
{
    const float tau = fmaf(fi, dtau, tau0);
    const float u = __fmul_rn(__fadd_rn(tau, l.W), l.inv_dt);
    const float tv = __fadd_rd(u, MAGIC);
    const float f = u - (tv - MAGIC);
    float t0, t1;
    asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(t0), "=f"(t1) : "r"(l.tab + (__float_as_uint(tv) << 3)));
    return fmaf(f, t1, t0);
}

// Byte offset along one axis of the pair image (see PairLay).
struct AxisLay {
    unsigned c1, c2, c3;
};
__device__ __forceinline__ unsigned along(const AxisLay& a, unsigned i)
{
    return i * a.c1 + (i & 2u) * a.c2 + (i & 1u) * a.c3;
}

// The same from the block's own table.
__device__ __forceinline__ float tof_series(const Lane& l, float tau0, float dtau, float fi)
{
    const float tau = fabsf(fmaf(fi, dtau, tau0));
    const float tv = fmaf(tau, l.inv_dt, MAGIC);
    const float f = fmaf(MAGIC - tv, l.dt, tau);  // from the node, without a rounding of the coordinate
    float w, s, c, z;
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(w), "=f"(s), "=f"(c), "=f"(z)
        : "r"(l.tab + (__float_as_uint(tv) << 4)));
    return fmaf(f, fmaf(f, c, s), w);
}

// The same by the pair of lanes of a plane, each with the erf of one edge of
// the bin (tof_weight's arithmetic).  All lanes of the warp take part.
__device__ __forceinline__ float tof_erf(const Lane& l, float tau0, float dtau, float fi)
{
    const float tau = fmaf(fi, dtau, tau0);
    const float e = erff((tau + l.hb) * l.inv_s);
    const float o = __shfl_xor_sync(FULL, e, 1);
    return 0.5f * (l.par ? o - e : e - o);
}

// Straight-line walk of NP passes of an x- or y-principal event: all gathers
// are in flight before the first is used.  Passes from CHECK on may lie
// beyond the event's planes: their lanes repeat the last plane's coordinates
// (which keeps the table index in range) without a sample.  INNER: all
// neighbours are inside the grid; otherwise a neighbour outside weighs 0, and
// a sample whose slice B is below the grid takes the first half of slice 0.
// SAFE: a voxel of weight 0 does not enter (it may hold an infinity or NaN).
// Returns the lane's part of sum w x / (c_e step).
template <int NP, int CHECK, bool INNER, Tof TOF, bool GATHER, bool SAFE>
__device__ __forceinline__ float walk(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r, int p0,
                                      const char* __restrict__ img, Held& h)
{
    const float4 g0 = r.g0;
    const float tau0 = r.g1.x, dtau = r.g1.y;
    const unsigned m = r.meta;
    const int cnt = (int)(m & 0x7FFFu);
    const bool kx = ((m >> 15) & 3u) == 0u;
    const AxisLay pa = {kx ? P.x1 : P.y1, kx ? P.x2 : P.y2, kx ? P.x3 : P.y3};
    const AxisLay aa = {kx ? P.y1 : P.x1, kx ? P.y2 : P.x2, kx ? P.y3 : P.x3};
    // MAGIC_BITS is a multiple of 4: it only enters the linear terms
    const unsigned base = along(pa, (unsigned)(r.i0 + l.pl + 16 * p0)) - MAGIC_BITS * (aa.c1 + P.zs);
    const float fp = (float)(r.i0 + 16 * p0) + l.fpl, flast = (float)(r.i0 + cnt - 1);
    float2 x[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        bool in = p < CHECK || l.pl + 16 * (p0 + p) < cnt;
        const float fi = p < CHECK ? fp + (float)(16 * p) : fminf(fp + (float)(16 * p), flast);
        const float w = TOF == TOF_TABLE    ? tof_at(l, tau0, dtau, fi)
                        : TOF == TOF_SERIES ? tof_series(l, tau0, dtau, fi)
                        : TOF == TOF_ERF    ? tof_erf(l, tau0, dtau, fi)
                                            : 1.0f;
        const float ua = fmaf(fi, g0.y, g0.x);
        const float ta = __fadd_rd(ua, MAGIC);
        const float fa = ua - (ta - MAGIC);
        const float ub = fmaf(fi, g0.w, g0.z);
        const float tb = __fadd_rd(ub, MAGIC);
        const float fb = ub - (tb - MAGIC);
        const float wa = fmaf(l.sgn, fa, l.off) * w;
        unsigned off = base + 16u * p * pa.c1 + along(aa, __float_as_uint(ta) + (unsigned)l.par) + __float_as_uint(tb) * P.zs;
        // (not wa - wa fb: at the grid's faces the small weight is all there is of a sample)
        float q1 = wa * fb, q0 = wa * (1.0f - fb);
        if (!INNER) {
            const int ia = (int)(__float_as_uint(ta) - MAGIC_BITS) + l.par;
            const int ib = (int)(__float_as_uint(tb) - MAGIC_BITS);
            in = in && (unsigned)ia < (unsigned)(kx ? G.n[1] : G.n[0]);
            if (ib < 0) {
                off += P.zs;
                q0 = q1;
                q1 = 0.0f;
            } else if (ib + 1 >= G.n[2]) {
                q1 = 0.0f;
            }
        }
        if (!INNER || p >= CHECK) {
            off = in ? off : NONE;
            q0 = in ? q0 : 0.0f;
            q1 = in ? q1 : 0.0f;
        }
        h.off[p] = off;
        h.q0[p] = q0;
        h.q1[p] = q1;
        if (GATHER) {
            x[p] = make_float2(0.0f, 0.0f);
            if ((INNER && p < CHECK) || off != NONE) x[p] = __ldg(reinterpret_cast<const float2*>(img + off));
            if (SAFE) {
                if (q0 == 0.0f) x[p].x = 0.0f;
                if (q1 == 0.0f) x[p].y = 0.0f;
            }
        }
    }
    float acc = 0.0f;
    if (GATHER) {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            acc = fmaf(h.q0[p], x[p].x, acc);
            acc = fmaf(h.q1[p], x[p].y, acc);
        }
    }
    return acc;
}

// A z-principal event (B along y: its neighbours are two rows, each the first
// half of a pair).  BACK: adds b times the weights to acc, else returns the
// lane's part of sum w x / (c_e step).  Few events of a short scanner, most of
// one that is longer than wide: U planes per lane at a time, so that 2 U gathers
// are in flight.
template <Tof TOF, bool BACK, int U>
__device__ __forceinline__ float walk_z(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r,
                                        const char* __restrict__ img, char* acc, float b)
{
    const float4 g0 = r.g0;
    const float tau0 = r.g1.x, dtau = r.g1.y;
    const int cnt = (int)(r.meta & 0x7FFFu), i0 = r.i0;
    const AxisLay ax = {P.x1, P.x2, P.x3}, ay = {P.y1, P.y2, P.y3};
    float s = 0.0f;
    for (int j0 = 0; j0 < cnt; j0 += 16 * U) {
        unsigned o0[U], o1[U];
        float q0[U], q1[U];
#pragma unroll
        for (int p = 0; p < U; ++p) {
            const int jp = j0 + 16 * p + l.pl, j = min(jp, cnt - 1);  // (keeps the table index in range)
            const float fi = (float)(i0 + j);
            const float w = TOF == TOF_TABLE    ? tof_at(l, tau0, dtau, fi)
                            : TOF == TOF_SERIES ? tof_series(l, tau0, dtau, fi)
                            : TOF == TOF_ERF    ? tof_weight(G, TOF_BIN, fmaf(fi, dtau, tau0))
                                                : 1.0f;
            const float ua = fmaf(fi, g0.y, g0.x), fla = floorf(ua);
            const float ub = fmaf(fi, g0.w, g0.z), flb = floorf(ub), fb = ub - flb;
            const int ia = (int)fla + l.par, iy = (int)flb;
            const bool in = jp < cnt && (unsigned)ia < (unsigned)G.n[0];
            const float wa = fmaf(l.sgn, ua - fla, l.off) * w;
            q0[p] = in && (unsigned)iy < (unsigned)G.n[1] ? wa * (1.0f - fb) : 0.0f;
            q1[p] = in && (unsigned)(iy + 1) < (unsigned)G.n[1] ? wa * fb : 0.0f;
            const unsigned o = along(ax, (unsigned)ia) + (unsigned)(i0 + j) * P.zs;
            o0[p] = o + along(ay, (unsigned)iy);
            o1[p] = o + along(ay, (unsigned)iy + 1u);
        }
        if (BACK) {
#pragma unroll
            for (int p = 0; p < U; ++p) {
                if (q0[p] != 0.0f) atomicAdd(reinterpret_cast<float*>(acc + o0[p]), q0[p] * b);
                if (q1[p] != 0.0f) atomicAdd(reinterpret_cast<float*>(acc + o1[p]), q1[p] * b);
            }
        } else {
            float x0[U], x1[U];
#pragma unroll
            for (int p = 0; p < U; ++p) {
                x0[p] = q0[p] != 0.0f ? __ldg(reinterpret_cast<const float*>(img + o0[p])) : 0.0f;
                x1[p] = q1[p] != 0.0f ? __ldg(reinterpret_cast<const float*>(img + o1[p])) : 0.0f;
            }
#pragma unroll
            for (int p = 0; p < U; ++p) s = fmaf(q1[p], x1[p], fmaf(q0[p], x0[p], s));
        }
    }
    return s;
}

// The same as a call, for kernels that meet such events among the others.
template <Tof TOF, bool BACK>
__device__ __noinline__ float walk_z_call(const Lane l, const Geo& G, const lmh::PairLay& P, const Rec& r,
                                          const char* __restrict__ img, char* acc, float b)
{
    return walk_z<TOF, BACK, 4>(l, G, P, r, img, acc, b);
}

template <bool SAFE>
__device__ __forceinline__ float times(float q, float b)
{
    return SAFE && q == 0.0f ? 0.0f : q * b;
}

__device__ __forceinline__ bool z_principal(const Rec& r) { return ((r.meta >> 15) & 3u) == 2u; }

// Forward part of one x- or y-principal event.  Planes beyond the held ones
// (finer grids) are walked sixteen at a time.
template <Tof TOF, bool SAFE = false>
__device__ __forceinline__ float forward(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r,
                                         const char* __restrict__ img, Held& h)
{
    const unsigned m = r.meta;
    const int cnt = (int)(m & 0x7FFFu);
    if (cnt == 0) return 0.0f;
    float acc;
    if ((m & REC_INNER) && cnt > 32) {
        if (cnt > 48) acc = walk<4, 3, true, TOF, true, SAFE>(l, G, P, r, 0, img, h);
        else acc = walk<3, 2, true, TOF, true, SAFE>(l, G, P, r, 0, img, h);
    } else {
        acc = walk<4, 0, false, TOF, true, SAFE>(l, G, P, r, 0, img, h);
    }
    for (int p = PASSES; 16 * p < cnt; ++p) {
        Held t;
        acc += walk<1, 0, false, TOF, true, SAFE>(l, G, P, r, p, img, t);
    }
    return acc;
}

// Back-projection part of one x- or y-principal event: b is its value times the sample length.
// SAFE: nothing is added where the weight is 0 (b may be an infinity or NaN).
template <Tof TOF, bool SAFE = false>
__device__ __forceinline__ void backward(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r,
                                         const Held& h, float b, char* acc)
{
    const int cnt = (int)(r.meta & 0x7FFFu);
#pragma unroll
    for (int p = 0; p < PASSES; ++p)
        if (16 * p < cnt && h.off[p] != NONE)
            atomicAdd(reinterpret_cast<float2*>(acc + h.off[p]), make_float2(times<SAFE>(h.q0[p], b), times<SAFE>(h.q1[p], b)));
    for (int p = PASSES; 16 * p < cnt; ++p) {
        Held t;
        walk<1, 0, false, TOF, false, false>(l, G, P, r, p, nullptr, t);
        if (t.off[0] != NONE)
            atomicAdd(reinterpret_cast<float2*>(acc + t.off[0]), make_float2(times<SAFE>(t.q0[0], b), times<SAFE>(t.q1[0], b)));
    }
}

// Projection of one event of any principal axis.
template <Tof TOF>
__device__ __forceinline__ float gather(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r,
                                        const char* __restrict__ img)
{
    Held h;
    return z_principal(r) ? walk_z_call<TOF, false>(l, G, P, r, img, nullptr, 0.0f)
                          : forward<TOF, true>(l, G, P, r, img, h);
}

// Back-projection of one event of any principal axis that was not walked forward before.
template <Tof TOF>
__device__ __forceinline__ void spread(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r, float b, char* acc)
{
    const unsigned m = r.meta;
    const int cnt = (int)(m & 0x7FFFu);
    if (cnt == 0) return;
    if (z_principal(r)) {
        walk_z_call<TOF, true>(l, G, P, r, nullptr, acc, b);
        return;
    }
    Held h;
    if (m & REC_INNER) walk<PASSES, 0, true, TOF, false, false>(l, G, P, r, 0, nullptr, h);
    else walk<PASSES, 0, false, TOF, false, false>(l, G, P, r, 0, nullptr, h);
    backward<TOF, true>(l, G, P, r, h, b, acc);
}

// Sums of two events over the warp in one tree: lanes 0-15 return the first
// event's, lanes 16-31 the second's.
__device__ __forceinline__ float reduce2(float a0, float a1)
{
    const bool lo = (threadIdx.x & 16) == 0;
    float mine = lo ? a0 : a1;
    mine += __shfl_xor_sync(FULL, lo ? a1 : a0, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mine += __shfl_xor_sync(FULL, mine, o);
    return mine;
}

// Events per work item of a launch over `count` events: two per warp of the
// launch at least (a pair is the unit of the walk), at most 32 (a warp's
// staging), about four items per warp in between.
__device__ __forceinline__ int chunk_of(int64_t count, int64_t warps)
{
    const int64_t c = count / (4 * warps);
    return c >= 32 ? 32 : (c <= 2 ? 2 : (int)c & ~1);
}

// One x- or y-principal event pass by pass: its sum with every voxel and without
// those of weight 0, and its back-projection without them.
template <Tof TOF>
__device__ __forceinline__ void forward_both(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r,
                                             const char* __restrict__ img, float& plain, float& safe)
{
    plain = safe = 0.0f;
#pragma unroll 1
    for (int p = 0; 16 * p < (int)(r.meta & 0x7FFFu); ++p) {
        Held t;
        walk<1, 0, false, TOF, false, false>(l, G, P, r, p, nullptr, t);
        if (t.off[0] == NONE) continue;
        const float2 x = __ldg(reinterpret_cast<const float2*>(img + t.off[0]));
        plain = fmaf(t.q1[0], x.y, fmaf(t.q0[0], x.x, plain));
        if (t.q0[0] != 0.0f) safe = fmaf(t.q0[0], x.x, safe);
        if (t.q1[0] != 0.0f) safe = fmaf(t.q1[0], x.y, safe);
    }
}

template <Tof TOF>
__device__ __forceinline__ void spread_small(const Lane& l, const Geo& G, const lmh::PairLay& P, const Rec& r, float b,
                                             char* acc)
{
#pragma unroll 1
    for (int p = 0; 16 * p < (int)(r.meta & 0x7FFFu); ++p) {
        Held t;
        walk<1, 0, false, TOF, false, false>(l, G, P, r, p, nullptr, t);
        if (t.off[0] != NONE)
            atomicAdd(reinterpret_cast<float2*>(acc + t.off[0]), make_float2(times<true>(t.q0[0], b), times<true>(t.q1[0], b)));
    }
}

__device__ __forceinline__ bool finite(float v) { return fabsf(v) <= 3.402823466e38f; }

}  // namespace lmw
