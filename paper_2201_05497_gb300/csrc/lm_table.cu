// Data update of Alg. 2 (forward projection of the subset's events, the
// closed-form dual step of Eq. (proxD), back-projection of the dual change
// divided by mu) from a stored traversal table.
//
// The direct event kernel (lm_project.cu) sets up every event's traversal
// from the crystal table on each visit.  This path computes each event's
// traversal (reading 1 of the projector: principal axis, trimmed plane range,
// affine secondary coordinates, TOF coordinate, sample length), 1/(P^LM 1)_e
// and mu_e once per state (trav_build), so a data update reads 40 bytes of
// table per event, and walks the events over z-pair images (lm_walk.cuh).
//
// Measured on the 200 x 200 x 96 grid (GB300, CUDA events around the launch,
// Monte Carlo events): 7 143 events 14.5 us, 50 000 33 us, 357 143 136 us, 1.07e6
// 356 us; one plane per lane over two image layouts and two accumulators took 200 us
// at 357 143.  ncu at 357 143 events: with the pairs in rows 71 % of the SM-to-L2
// request cycles (17.1 M lines gathered + 19.5 M sectors added to), issue 42 %, 176
// us; in bricks 9.2 M + 16.0 M: instructions and requests now bound it about
// equally (profiles/ev_table_kernel_data_update_3d_short.txt).
// Ordering the events by direction and place moved it by less than 10 % in
// either direction, and one-plane-per-lane with the same pairs was no faster.
// Per sample the positions and weights are the direct kernel's (lor_setup; see
// build_table for the rounding of the TOF coordinate).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "lm_walk.cuh"

using namespace lmk;

namespace lmh {

bool trav_capable(const lm_grid* g)
{
    if (g->n[2] < 2 || g->n[1] < 2) return false;
    for (int d = 0; d < 3; ++d)
        if (g->n[d] >= (1 << 15)) return false;
    return true;
}

TravLayout trav_layout(const lm_grid* g, int64_t N)
{
    (void)g;
    TravLayout L;
    std::memset(&L, 0, sizeof(L));
    const size_t n = (size_t)std::max<int64_t>(N, 1);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += align_up(bytes);
        return o;
    };
    L.r0 = take(n * 16);
    L.r1 = take(n * 16);
    L.meta = take(n * 8);
    L.total = off + 256;
    return L;
}

}  // namespace lmh

namespace {

using lmh::TOF_TAB_N;

// Packed plane range of a table entry: i0 (15 bits), planes (15 bits, 0 =
// inert event), principal axis (2 bits); an entry whose samples all have
// their four neighbours inside the grid has a negative sample length.
__device__ __forceinline__ unsigned pack_meta(int i0, int cnt, int k)
{
    return (unsigned)i0 | ((unsigned)cnt << 15) | ((unsigned)k << 30);
}

// One thread per event: the traversal of reading 1 (lor_setup, the direct
// kernel's own set-up) trimmed to its planes with a sample, 1/(P^LM 1)_e with
// (P^LM 1)_e = c_e times the sum over the event's samples of the in-grid
// bilinear weights times TOF weight times sample length (0 where that sum is
// 0: S_e = 0, an inert event), and mu_e.
__global__ void trav_build_kernel(const Geo G, const int32_t* __restrict__ det1, const int32_t* __restrict__ det2,
                                  const int16_t* __restrict__ tofb, const float* __restrict__ corr,
                                  const uint16_t* __restrict__ mu, int64_t N, const float* __restrict__ tab,
                                  float4* __restrict__ r0, float4* __restrict__ r1, int2* __restrict__ meta, bool stored)
{
    __shared__ float s_tab[TOF_TAB_N + 1];
    for (int k = threadIdx.x; k <= TOF_TAB_N; k += blockDim.x) s_tab[k] = tab[k];
    __syncthreads();
    const float inv_dt = (float)TOF_TAB_N / (2.0f * G.W);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < N; e += (int64_t)gridDim.x * blockDim.x) {
        const int d1 = det1[e], d2 = det2[e], m = (int)tofb[e];
        bool ok = d1 >= 0 && d1 < G.n_det && d2 >= 0 && d2 < G.n_det && d1 != d2 && m >= -G.M && m <= G.M;
        Lor L;
        ok = ok && lor_setup(G, d1, d2, m, TOF_BIN, true, L, stored);
        float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
        unsigned mw = 0u;
        if (ok) {
            lmh::lor_strides(G, L.k, true, L);  // extents (and strides) of the secondary axes
            bool inner;
            lmw::trim(G, L, &inner);
            if (L.cnt > 0) {
                float acc1 = 0.0f;
                for (int i = L.i0; i < L.i0 + L.cnt; ++i) {
                    Smp s;
                    if (lmh::sample_tab<false>(G, L, s_tab, inv_dt, i, s)) acc1 += wsum<false>(s);
                }
                const float p1 = (corr ? corr[e] : 1.0f) * acc1;
                a = make_float4(L.ua0, L.sa, L.ub0, L.sb);
                b = make_float4(L.tau0, L.dtau, inner ? -L.step : L.step, p1 > 0.0f ? 1.0f / p1 : 0.0f);
                mw = pack_meta(L.i0, L.cnt, L.k);
            }
        }
        r0[e] = a;
        r1[e] = b;
        meta[e] = make_int2((int)mw, __float_as_int((float)mu[e]));
    }
}

// Staged events of a chunk: the first `main` are x- or y-principal, the others
// up to `all` z-principal.
struct Staged {
    int main, all;
};

// Stages the events [e0, e0 + nev) that have samples into `rec` (lanes load
// their event's entry and fields coalesced, with the streaming cache policy:
// each is read once per update).  MODE EV_FWD also stages the events without
// samples (their projection is 0).
template <int MODE>
__device__ __forceinline__ Staged stage(const lmh::TabArgs& A, int64_t e0, int nev, lmw::Rec* rec)
{
    const int lane = threadIdx.x & 31;
    const int64_t e = e0 + lane;
    const bool in = lane < nev;
    const int2 mt = in ? __ldcs(A.meta + e) : make_int2(0, 0);
    const unsigned mw = (unsigned)mt.x;
    const unsigned cnt = (mw >> 15) & 0x7FFFu;
    const bool mine = in && (MODE != lmh::EV_DATA || cnt != 0u), zp = (mw >> 30) == 2u;
    const unsigned mask = __ballot_sync(FULL, mine && !zp), zmask = __ballot_sync(FULL, mine && zp);
    if (mine) {
        const unsigned below = (1u << lane) - 1u;
        lmw::Rec& r = rec[zp ? __popc(mask) + __popc(zmask & below) : __popc(mask & below)];
        const float4 g1 = __ldcs(A.r1 + e);
        const float mu = __int_as_float(mt.y), step = fabsf(g1.z);
        const float cs = (A.corr ? __ldcs(A.corr + e) : 1.0f) * step;
        lmw::rec_path(__ldcs(A.r0 + e), g1.x, g1.y, (int)(mw & 0x7FFFu), (int)cnt, (int)(mw >> 30), g1.z < 0.0f, lane,
                      r);
        r.g1.z = cs / mu;
        r.g1.w = A.gamma_rho * g1.w;  // S_e = gamma rho / (P^LM 1)_e
        r.d = make_float4(cs, MODE == lmh::EV_FWD ? 0.0f : __ldcs(A.contam + e),
                          MODE == lmh::EV_DATA ? __ldcs(A.y + e) : 0.0f, mu);
    }
    __syncwarp();
    return {__popc(mask), __popc(mask) + __popc(zmask)};
}

// Staged events [lo, hi), two at a time: forward projection of both, one
// reduction, the per-event step (MODE EV_DATA: Eq. (proxD); EV_FWD: the
// projection itself) in a half-warp each, and the back-projection of both.  Z:
// z-principal events.  They have a loop of their own because a call or a
// second walk in this one costs all events registers (64 per thread, and an
// event's samples take 12): spilling them made an update 12 to 50 % longer.
// An event with a value that is not finite is left undone and *bad set: a voxel of
// weight 0 may hold an infinity (see table_again; walk_z reads and writes no
// such voxels).  A projection that is not finite leaves no finite dual change.
template <int MODE, bool Z>
__device__ __forceinline__ void table_pairs(const lmh::TabArgs& A, const lmw::Lane& l, int64_t e0, int lo, int hi,
                                            const lmw::Rec* rec, int* bad)
{
    const int lane = threadIdx.x & 31;
    const char* img = reinterpret_cast<const char*>(A.xp);
    char* acc = reinterpret_cast<char*>(A.acc);
    for (int b = lo; b < hi; b += 2) {
        lmw::Held h0, h1;
        float a0, a1 = 0.0f;
        const bool two = b + 1 < hi;
        if (Z) {
            a0 = lmw::walk_z<lmw::TOF_TABLE, false, 2>(l, A.G, A.lay, rec[b], img, nullptr, 0.0f);
            if (two) a1 = lmw::walk_z<lmw::TOF_TABLE, false, 2>(l, A.G, A.lay, rec[b + 1], img, nullptr, 0.0f);
        } else {
            a0 = lmw::forward<lmw::TOF_TABLE>(l, A.G, A.lay, rec[b], img, h0);
            if (two) a1 = lmw::forward<lmw::TOF_TABLE>(l, A.G, A.lay, rec[b + 1], img, h1);
        }
        const lmw::Rec& R = rec[b + (two ? lane >> 4 : 0)];
        const float4 dd = R.d;
        const bool valid = lane < 16 || two;
        const bool first = valid && (lane & 15) == 0;
        const float J = lmw::reduce2(a0, a1);                 // (P^LM x)_e = c_e step J
        const int64_t e = e0 + (R.meta >> 20);
        if (MODE == lmh::EV_FWD) {
            if (first) A.out[e] = dd.x * J;
            if (!Z && !lmw::finite(J)) *bad = 1;
            continue;
        }
        // dual step of Eq. (proxD) with the listmode step mu_e S_e
        const float Se = R.g1.w;
        const float a = fmaf(Se, fmaf(dd.x, J, dd.y), dd.z);  // y + S (P^LM x + s)
        const float yp = prox_dstar(a, dd.w * Se);
        const bool ok = Z || lmw::finite(yp);
        if (first && ok) __stcs(A.y + e, yp);
        float bval = R.g1.z * (yp - dd.z);                    // c step (y+ - y) / mu
        if (!valid || !ok) bval = 0.0f;
        if (!ok) *bad = 1;
        const float b0 = __shfl_sync(FULL, bval, 0), b1 = __shfl_sync(FULL, bval, 16);
        if (Z) {
            if (b0 != 0.0f) lmw::walk_z<lmw::TOF_TABLE, true, 2>(l, A.G, A.lay, rec[b], nullptr, acc, b0);
            if (b1 != 0.0f) lmw::walk_z<lmw::TOF_TABLE, true, 2>(l, A.G, A.lay, rec[b + 1], nullptr, acc, b1);
        } else {
            if (b0 != 0.0f) lmw::backward<lmw::TOF_TABLE>(l, A.G, A.lay, rec[b], h0, b0, acc);
            if (b1 != 0.0f) lmw::backward<lmw::TOF_TABLE>(l, A.G, A.lay, rec[b + 1], h1, b1, acc);
        }
    }
}

// Once more through a chunk for the events that table_pairs left undone, those
// whose dual step is still not finite, one at a time, without the voxels of weight
// 0 in either direction.  Run by a block that met such an event, after its last
// chunk, and as little code as does it: inside the loop over the chunks its
// registers, or a call's, cost every event 12 to 25 %.
template <int MODE>
__device__ __forceinline__ void table_again(const lmh::TabArgs& A, const lmw::Lane& l, int64_t e0, int n,
                                            const lmw::Rec* rec)
{
#pragma unroll 1
    for (int b = 0; b < n; ++b) {
        const lmw::Rec& R = rec[b];
        const int64_t e = e0 + (R.meta >> 20);
        const bool first = (threadIdx.x & 31) == 0;
        float plain, safe, v;
        lmw::forward_both<lmw::TOF_TABLE>(l, A.G, A.lay, R, reinterpret_cast<const char*>(A.xp), plain, safe);
        plain = warp_sum(plain);
        safe = warp_sum(safe);
        if (MODE == lmh::EV_FWD) {
            if (first && !lmw::finite(plain)) A.out[e] = R.d.x * safe;
            continue;
        }
        if (lmw::finite(prox_dstar(fmaf(R.g1.w, fmaf(R.d.x, plain, R.d.y), R.d.z), R.d.w * R.g1.w))) continue;
        const float yp = prox_dstar(fmaf(R.g1.w, fmaf(R.d.x, safe, R.d.y), R.d.z), R.d.w * R.g1.w);
        if (first) __stcs(A.y + e, yp);
        v = R.g1.z * (yp - R.d.z);
        if (v != 0.0f) lmw::spread_small<lmw::TOF_TABLE>(l, A.G, A.lay, R, v, reinterpret_cast<char*>(A.acc));
    }
    __syncwarp();
}

template <int MODE>
__device__ __forceinline__ void table_chunk(const lmh::TabArgs& A, const lmw::Lane& l, int64_t e0, const Staged& n,
                                            const lmw::Rec* rec, int* bad)
{
    table_pairs<MODE, false>(A, l, e0, 0, n.main, rec, bad);
    table_pairs<MODE, true>(A, l, e0, n.main, n.all, rec, bad);
    __syncwarp();
}

constexpr int TAB_THREADS = 512;
constexpr int TAB_WARPS = TAB_THREADS / 32;
constexpr size_t TAB_SMEM = lmw::TAB_PAD * sizeof(float2) + (size_t)TAB_WARPS * 32 * sizeof(lmw::Rec);

// One subset (or event range) from the traversal table.  Block b takes the
// chunks b, b + blocks, ...; its warps draw them from a counter in shared
// memory (a global counter served one draw in about 2.5 ns, which held
// launches with small chunks back: 75 us for 50 000 events, against 22 us).
template <int MODE>
__global__ void __launch_bounds__(TAB_THREADS, 2) ev_table_kernel(const __grid_constant__ lmh::TabArgs A)
{
    extern __shared__ float4 s_dyn[];
    __shared__ int s_next, s_bad;
    float2* s_tab = reinterpret_cast<float2*>(s_dyn);
    int64_t eb = A.e_begin, ee = A.e_end;
    if (A.seq != nullptr) {
        const int sel = A.seq[A.u];
        if (sel >= A.n_subsets) return;
        eb = A.sub_off[sel];
        ee = A.sub_off[sel + 1];
    }
    const int64_t count = ee - eb;
    const int CH = lmw::chunk_of(count, (int64_t)gridDim.x * TAB_WARPS);
    const int64_t nch = count > 0 ? (count + CH - 1) / CH : 0;
    const int warp = threadIdx.x >> 5;
    lmw::Rec* rec = reinterpret_cast<lmw::Rec*>(s_tab + lmw::TAB_PAD) + warp * 32;
    int64_t c = (int64_t)warp * gridDim.x + blockIdx.x;
    Staged n = {0, 0};
    if (c < nch) n = stage<MODE>(A, eb + c * CH, (int)min((int64_t)CH, count - c * CH), rec);
    if (threadIdx.x == 0) {
        s_next = TAB_WARPS;
        s_bad = 0;
    }
    lmw::fill_tab(s_tab, A.tof_tab);
    __syncthreads();
    const lmw::Lane l = lmw::table_lane(s_tab, A.G.W);
    while (c < nch) {
        table_chunk<MODE>(A, l, eb + c * CH, n, rec, &s_bad);
        int k = 0;
        if ((threadIdx.x & 31) == 0) k = atomicAdd(&s_next, 1);
        c = (int64_t)__shfl_sync(FULL, k, 0) * gridDim.x + blockIdx.x;
        if (c < nch) n = stage<MODE>(A, eb + c * CH, (int)min((int64_t)CH, count - c * CH), rec);
    }
    __syncthreads();
    if (s_bad)
        for (c = (int64_t)warp * gridDim.x + blockIdx.x; c < nch; c += (int64_t)TAB_WARPS * gridDim.x) {
            n = stage<MODE>(A, eb + c * CH, (int)min((int64_t)CH, count - c * CH), rec);
            table_again<MODE>(A, l, eb + c * CH, n.main, rec);
        }
}

// The data updates of every active frame of a batch at update u, from their
// traversal tables: the work items are the chunks of each frame's
// selected subset (frames at a prior update have none: their dual step runs
// in the image pass), found through a prefix table in shared memory.
__global__ void __launch_bounds__(TAB_THREADS, 2) ev_table_batch_kernel(const __grid_constant__ lmh::BatchTabArgs B)
{
    extern __shared__ float4 s_dyn[];
    float2* s_tab = reinterpret_cast<float2*>(s_dyn);
    __shared__ long long s_pre[lmh::BATCH_MAX + 1];
    __shared__ long long s_eb[lmh::BATCH_MAX];
    __shared__ long long s_ee[lmh::BATCH_MAX];
    __shared__ int s_next, s_bad;
    const int cap = B.cap;
    if (threadIdx.x < cap) {
        const int s = threadIdx.x;
        long long eb = 0, ee = 0;
        if (B.active[s]) {
            const lmh::TabArgs& A = B.slots[s];
            const int sel = B.seqs[(size_t)s * B.seq_stride + B.u];
            if (sel < A.n_subsets) {
                eb = A.sub_off[sel];
                ee = A.sub_off[sel + 1];
            }
        }
        s_eb[s] = eb;
        s_ee[s] = ee;
    }
    if (threadIdx.x == 0) s_next = s_bad = 0;
    lmw::fill_tab(s_tab, B.tof_tab);
    __syncthreads();
    long long events = 0;
    for (int s = 0; s < cap; ++s) events += s_ee[s] - s_eb[s];
    const int CH = lmw::chunk_of(events, (long long)gridDim.x * TAB_WARPS);
    if (threadIdx.x == 0) {
        s_pre[0] = 0;
        for (int s = 0; s < cap; ++s) s_pre[s + 1] = s_pre[s] + (s_ee[s] - s_eb[s] + CH - 1) / CH;
    }
    __syncthreads();
    const long long total = s_pre[cap];
    const lmw::Lane l = lmw::table_lane(s_tab, B.tof_W);
    lmw::Rec* rec = reinterpret_cast<lmw::Rec*>(s_tab + lmw::TAB_PAD) + (threadIdx.x >> 5) * 32;
    for (;;) {
        int k = 0;
        if ((threadIdx.x & 31) == 0) k = atomicAdd(&s_next, 1);
        const long long c = (long long)__shfl_sync(FULL, k, 0) * gridDim.x + blockIdx.x;
        if (c >= total) break;
        int s = 0;
        while (s_pre[s + 1] <= c) ++s;
        const lmh::TabArgs& A = B.slots[s];
        const int64_t e0 = s_eb[s] + (c - s_pre[s]) * CH;
        const Staged n = stage<lmh::EV_DATA>(A, e0, (int)min((long long)CH, s_ee[s] - e0), rec);
        table_chunk<lmh::EV_DATA>(A, l, e0, n, rec, &s_bad);
    }
    __syncthreads();
    if (!s_bad) return;
    for (long long c = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; c < total; c += (long long)TAB_WARPS * gridDim.x) {
        int s = 0;
        while (s_pre[s + 1] <= c) ++s;
        const lmh::TabArgs& A = B.slots[s];
        const int64_t e0 = s_eb[s] + (c - s_pre[s]) * CH;
        const Staged n = stage<lmh::EV_DATA>(A, e0, (int)min((long long)CH, s_ee[s] - e0), rec);
        table_again<lmh::EV_DATA>(A, l, e0, n.main, rec);
    }
}

// Standalone projections (lm_fwd, lm_back) by the same walk, the traversals set
// up by the staging lanes.  357 143 events on the 200 x 200 x 96 grid, whole calls
// (with the pair image, or the accumulator's clearing and fold): ev_kernel / this:
// forward 165 / 124 us, back 317 / 144 us.
constexpr size_t OP_RECS = (size_t)TAB_WARPS * 32 * sizeof(lmw::Rec);
constexpr size_t OP_SMEM = OP_RECS + (lmw::SERIES_N + 1) * sizeof(float4);  // TOF_SERIES; the others: OP_RECS

template <int MODE, lmw::Tof TOF>
__global__ void __launch_bounds__(TAB_THREADS, 2) op_walk_kernel(const __grid_constant__ lmh::OpArgs A)
{
    constexpr bool TOF_ON = TOF != lmw::NO_TOF;
    extern __shared__ float4 s_dyn[];
    __shared__ int s_next;
    float4* s_ser = s_dyn + OP_RECS / sizeof(float4);
    const Geo& G = A.G;
    const int lane = threadIdx.x & 31;
    const int CH = lmw::chunk_of(A.n, (int64_t)gridDim.x * TAB_WARPS);
    const int64_t nch = (A.n + CH - 1) / CH;
    lmw::Rec* rec = reinterpret_cast<lmw::Rec*>(s_dyn) + (threadIdx.x >> 5) * 32;
    if (threadIdx.x == 0) s_next = 0;
    if (TOF == lmw::TOF_SERIES) lmw::make_series(s_ser, G);
    else __syncthreads();
    const lmw::Lane l = lmw::op_lane(s_ser, G);
    const char* img = reinterpret_cast<const char*>(A.xp);
    char* acc = reinterpret_cast<char*>(A.acc);
    for (;;) {
        int k = 0;
        if (lane == 0) k = atomicAdd(&s_next, 1);
        const int64_t c = (int64_t)__shfl_sync(FULL, k, 0) * gridDim.x + blockIdx.x;
        if (c >= nch) break;
        const int64_t e0 = c * CH;
        const int nev = (int)min((int64_t)CH, A.n - e0);
        if (lane < nev) {
            const int64_t e = e0 + lane;
            const int d1 = A.det1[e], d2 = A.det2[e], m = TOF_ON ? (int)A.tof[e] : 0;
            bool ok = d1 >= 0 && d1 < G.n_det && d2 >= 0 && d2 < G.n_det && d1 != d2 && (!TOF_ON || (m >= -G.M && m <= G.M));
            Lor L;
            bool inner = false;
            ok = ok && lor_setup(G, d1, d2, m, TOF_ON ? TOF_BIN : TOF_NONE, false, L);
            if (ok) lmw::trim(G, L, &inner);
            lmw::Rec& r = rec[lane];
            if (ok) lmw::rec_path(make_float4(L.ua0, L.sa, L.ub0, L.sb), L.tau0, L.dtau, L.i0, L.cnt, L.k, inner, lane, r);
            else lmw::rec_path(make_float4(0.0f, 0.0f, 0.0f, 0.0f), 0.0f, 0.0f, 0, 0, 0, false, lane, r);
            r.d.x = (A.corr ? A.corr[e] : 1.0f) * (ok ? L.step : 0.0f);
            r.d.y = MODE == lmh::EV_BACK ? A.v[e] : 0.0f;
        }
        __syncwarp();
        for (int b = 0; b < nev; b += 2) {
            const bool two = b + 1 < nev;
            if (MODE == lmh::EV_FWD) {
                float a1 = 0.0f;
                const float a0 = lmw::gather<TOF>(l, G, A.lay, rec[b], img);
                if (two) a1 = lmw::gather<TOF>(l, G, A.lay, rec[b + 1], img);
                const float J = lmw::reduce2(a0, a1);
                const int w = lane >> 4;
                if ((lane & 15) == 0 && (w == 0 || two)) A.out[e0 + b + w] = rec[b + w].d.x * J;
            } else {
                for (int w = 0; w < (two ? 2 : 1); ++w) {
                    const lmw::Rec& r = rec[b + w];
                    const float bv = r.d.x * r.d.y;
                    if (bv != 0.0f) lmw::spread<TOF>(l, G, A.lay, r, bv, acc);
                }
            }
        }
        __syncwarp();
    }
}

// img += the pair accumulator.
__global__ void __launch_bounds__(256) pair_fold_kernel(float* __restrict__ img, const char* __restrict__ acc, int nx,
                                                        int ny, int64_t V, const lmh::PairLay P)
{
    const int64_t nxy = (int64_t)nx * ny;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < V; j += (int64_t)gridDim.x * blockDim.x) {
        const int z = (int)(j / nxy), r = (int)(j - z * nxy), y = r / nx;
        const unsigned o = P.at((unsigned)(r - y * nx), (unsigned)y, (unsigned)z);
        img[j] += *reinterpret_cast<const float*>(acc + o) +
                  (z > 0 ? *reinterpret_cast<const float*>(acc + (o - P.zs) + 4) : 0.0f);
    }
}

// x (x fastest) as z pairs (x_j, x_{j + nx*ny}), 0 above the last slice.
__global__ void __launch_bounds__(256) pair_image_kernel(const float* __restrict__ x, char* __restrict__ xp, int nx,
                                                         int ny, int64_t V, const lmh::PairLay P)
{
    const int64_t nxy = (int64_t)nx * ny;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < V; j += (int64_t)gridDim.x * blockDim.x) {
        const int z = (int)(j / nxy), r = (int)(j - z * nxy), y = r / nx;
        *reinterpret_cast<float2*>(xp + P.at((unsigned)(r - y * nx), (unsigned)y, (unsigned)z)) =
            make_float2(x[j], j + nxy < V ? x[j + nxy] : 0.0f);
    }
}

}  // namespace

namespace lmh {

PairLay pair_layout(const lm_grid* g, bool rows)
{
    PairLay P;
    const unsigned nx = (unsigned)g->n[0], ny = (unsigned)g->n[1];
    P.x1 = 8u;
    P.y1 = 8u * nx;
    P.x2 = P.x3 = P.y2 = P.y3 = 0u;
    P.zs = 8u * nx * ny;
    P.brick = !rows && nx % 4 == 0 && ny % 4 == 0;
    if (P.brick) {
        P.x1 = 32u;
        P.x2 = 0u - 16u;
        P.x3 = 0u - 24u;
        P.y2 = 32u - 8u * nx;
        P.y3 = 16u - 8u * nx;
    }
    return P;
}

void launch_pair_image(const lm_grid* g, const PairLay& P, const float* x, float* xp, cudaStream_t st)
{
    const int64_t V = nvox(g);
    const int grid = (int)std::min<int64_t>((V + 255) / 256, (int64_t)num_sms() * 16);
    pair_image_kernel<<<grid, 256, 0, st>>>(x, (char*)xp, g->n[0], g->n[1], V, P);
    count_launch();
}

int trav_build(const Geo& G, const lm_events& ev, const uint16_t* mu, const float* tof_tab, const TravLayout& L,
               char* base, bool stored, cudaStream_t st)
{
    LM_CHECK(G.tof_on && tof_tab != nullptr, LM_ERR_INVALID_ARG, "the traversal table needs TOF data");
    if (ev.n <= 0) return LM_OK;
    const int grid = std::max<int64_t>(1, std::min<int64_t>((ev.n + 255) / 256, (int64_t)num_sms() * 8));
    trav_build_kernel<<<grid, 256, 0, st>>>(G, ev.det1, ev.det2, ev.tof, ev.corr, mu, ev.n, tof_tab,
                                            (float4*)(base + L.r0), (float4*)(base + L.r1), (int2*)(base + L.meta),
                                            stored);
    count_launch();
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

// Before every launch: the attribute belongs to the current device's copy of
// the kernel, so a flag kept by the process would serve the first device only.
template <class F>
static void table_smem(F* kernel)
{
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAB_SMEM);
}

template <class F>
static int table_blocks(F* kernel)
{
    int b = 0;
    table_smem(kernel);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, TAB_THREADS, TAB_SMEM) != cudaSuccess || b < 1) b = 1;
    return num_sms() * b;
}

// Resident blocks of the table kernels (all modes have the same bounds).
int table_grid()
{
    static int nb = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        nb = std::min(table_blocks(ev_table_kernel<EV_DATA>),
                      std::min(table_blocks(ev_table_kernel<EV_FWD>), table_blocks(ev_table_batch_kernel)));
    });
    return nb;
}

int launch_table_batch(const BatchTabArgs& b, cudaStream_t st)
{
    table_smem(ev_table_batch_kernel);
    ev_table_batch_kernel<<<table_grid(), TAB_THREADS, TAB_SMEM, st>>>(b);
    count_launch();
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

template <class F>
static int launch_op_kernel(F* kernel, size_t smem, const OpArgs& a, cudaStream_t st)
{
    int b = 0;
    LM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, TAB_THREADS, smem) != cudaSuccess || b < 1) b = 1;
    kernel<<<num_sms() * b, TAB_THREADS, smem, st>>>(a);
    count_launch();
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

template <int MODE>
static int launch_op_mode(const OpArgs& a, cudaStream_t st)
{
    if (!a.G.tof_on) return launch_op_kernel(op_walk_kernel<MODE, lmw::NO_TOF>, OP_RECS, a, st);
    const float sigmas = a.G.W * a.G.inv_s * 1.41421356f;
    return sigmas <= lmw::SERIES_SIGMAS * 1.00001f
               ? launch_op_kernel(op_walk_kernel<MODE, lmw::TOF_SERIES>, OP_SMEM, a, st)
               : launch_op_kernel(op_walk_kernel<MODE, lmw::TOF_ERF>, OP_RECS, a, st);
}

int launch_op(int mode, const OpArgs& a, cudaStream_t st)
{
    return mode == EV_FWD ? launch_op_mode<EV_FWD>(a, st) : launch_op_mode<EV_BACK>(a, st);
}

void launch_pair_fold(const lm_grid* g, const PairLay& P, float* img, const float* acc, cudaStream_t st)
{
    const int64_t V = nvox(g);
    const int grid = (int)std::min<int64_t>((V + 255) / 256, (int64_t)num_sms() * 16);
    pair_fold_kernel<<<grid, 256, 0, st>>>(img, (const char*)acc, g->n[0], g->n[1], V, P);
    count_launch();
}

int launch_table(int mode, const TabArgs& a, cudaStream_t st)
{
    const int grid = table_grid();
    switch (mode) {
    case EV_DATA:
        table_smem(ev_table_kernel<EV_DATA>);
        ev_table_kernel<EV_DATA><<<grid, TAB_THREADS, TAB_SMEM, st>>>(a);
        break;
    case EV_FWD:
        table_smem(ev_table_kernel<EV_FWD>);
        ev_table_kernel<EV_FWD><<<grid, TAB_THREADS, TAB_SMEM, st>>>(a);
        break;
    default: set_error("unknown traversal-table mode %d", mode); return LM_ERR_INVALID_ARG;
    }
    count_launch();
    LM_CUDA(cudaGetLastError());
    return LM_OK;
}

}  // namespace lmh
