// Combinatorial forward search (Sec. 2.2) as layer-synchronous rounds of three kernels.
//
// All seeds of all events advance together, one step of their layer plan per round (the
// paper's search processes every candidate of a layer before the next, Sec. 3.1).  A seed owns
// 8 candidate slots; per round:
//   k_move    one thread per live child, taken from a compacted work list: its state from its
//             parent's prediction and its hit (the Joseph update, a11), then the propagation to the
//             round's layer with Jacobian, transport and material (a4-a7);
//   k_find    one thread per child that crossed the layer: the eta-phi window (a8) and the chi2 of
//             each hit inside it (a9).  Writes the candidate's own children: its best hits (chi2
//             asc, hit id asc) and its non-hit child;
//   k_merge   eight lanes per seed: the N best children over the seed's candidates (a10), their
//             descriptors (parent slot, hit), (parent slot, hit) for the trail, the next work lists.
// k_start makes each seed the first child of its slot 0; k_finish gives each seed's best child its
// state and walks the trail back for its hit list (a13).
//
// Why three kernels: k_move computes (128 registers a thread, 16 warps per SM), k_find waits for
// chains of small loads and k_merge for short lists, and both need warps.  A child's state exists in
// registers only: its update and its propagation follow each other in k_move, one thread per child,
// and only predictions go through HBM.  The former round (propagation and window in one kernel, then
// merge and update by eight lanes per seed, 18.5 of 32 lanes active, states and predictions both
// written, records one after another) took 21.6 ms for 64 Phase-2-like events (1.28M seeds, 58M
// crossed steps) and 0.90 ms for one; one kernel for update, propagation and window 17.2 ms (its 128
// registers also held the window's chains of loads to 16 warps); these three 15.45 and 0.65 ms:
// k_move 7.3 ms, k_find 3.1, k_merge 4.3 of the 64 events.  k_move is bound by issue and latency
// together (50% issue active, 29% of DRAM), k_find and k_merge by their dependent loads.
//
// No kernel waits on another block; every loop is bounded by a list length, a window's bin range or
// the Newton iteration limit.  The kernels of a search are chained by programmatic dependent
// launches: a kernel's blocks start and load the geometry while the one before it ends.
#include "internal.h"
#include "launch.cuh"

#include <cstring>

namespace mk {

namespace {

constexpr int kGroup = 8;   // slots (lanes) per seed, >= MKGB_MAX_CANDS
constexpr int kThreads = 128;
constexpr float kBig = 3.0e38f;
constexpr int kQueue = 8;
constexpr int kDiskBit = 16;   // in a child list's header beside the number of hits: its layer is a disk
constexpr unsigned kFull = 0xffffffffu;

// ---- slot records: words of F, moved as 16-byte vectors

__device__ __forceinline__ void unpack16(const float4& v, float* f) { f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
__device__ __forceinline__ void unpack16(const double2& v, double* f) { f[0] = v.x; f[1] = v.y; }
__device__ __forceinline__ float4 pack16(const float* f) { return make_float4(f[0], f[1], f[2], f[3]); }
__device__ __forceinline__ double2 pack16(const double* f) { return make_double2(f[0], f[1]); }
template <class F> struct Vec16;
template <> struct Vec16<float> { using T = float4; };
template <> struct Vec16<double> { using T = double2; };

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Slots are laid out in tiles of 32 seeds: the 16-byte words of an array run over the seeds of a tile,
// then over the eight slots, then over the words of a record.  A warp of k_move or k_merge, whose slots
// come from a few neighbouring seeds, then touches about eight 128-byte lines per 16-byte load; with
// one record after another each lane touched a line of its own, and the L1 handles one line per cycle
// (~700 lines per warp of the update and propagation: 570 us a round of 640k seeds, 520 us in tiles).
constexpr int kTile = 32;
__host__ __device__ constexpr int tile_slots(int n_seeds) { return (n_seeds + kTile - 1) / kTile * (kTile * kGroup); }
// Place of slot sl = seed * kGroup + slot in an array of one 16-byte word (or one int) per slot.
__device__ __forceinline__ int slot_at(int sl) {
    return (sl & ~(kTile * kGroup - 1)) | (sl & (kGroup - 1)) * kTile | ((sl / kGroup) & (kTile - 1));
}
// Place of word j of slot sl in an array of N words per slot.
template <int N> __device__ __forceinline__ int64_t word_at(int sl, int j) {
    return ((int64_t)(sl / (kTile * kGroup)) * N + j) * (kTile * kGroup) + (sl & (kGroup - 1)) * kTile +
           ((sl / kGroup) & (kTile - 1));
}

// Words of a slot's record: a state (hi/lo positions, k, phi, theta, 21 covariance words, theta's and
// phi's low parts) or a prediction (the same with 15 surface-frame covariance words).
constexpr int kStateWords = 32, kPredWords = 28;
static_assert(kStateWords == kSeedStateStride, "seed records are read as state records");
template <class F> constexpr int rec_vecs() { return (int)(kStateWords * sizeof(F) / 16); }

template <class F, int W> __device__ __forceinline__ void load_rec(const unsigned char* __restrict__ base, int sl, F* f) {
    using V = typename Vec16<F>::T;
    constexpr int per = 16 / sizeof(F);
    const V* v = reinterpret_cast<const V*>(base) + word_at<rec_vecs<F>()>(sl, 0);
#pragma unroll
    for (int j = 0; j < W / per; ++j) unpack16(v[j * (kTile * kGroup)], f + per * j);
}

template <class F, int W> __device__ __forceinline__ void store_rec(unsigned char* __restrict__ base, int sl, const F* f) {
    using V = typename Vec16<F>::T;
    constexpr int per = 16 / sizeof(F);
    V* v = reinterpret_cast<V*>(base) + word_at<rec_vecs<F>()>(sl, 0);
#pragma unroll
    for (int j = 0; j < W / per; ++j) v[j * (kTile * kGroup)] = pack16(f + per * j);
}

template <class F> __device__ __forceinline__ void unpack_pred(const F* f, PredT<F>& q) {
    q.xh = f[0]; q.yh = f[1]; q.zh = f[2]; q.xl = f[3]; q.yl = f[4]; q.zl = f[5];
    q.k = f[6]; q.phi = f[7]; q.th = f[8];
#pragma unroll
    for (int i = 0; i < 15; ++i) q.c[i] = f[9 + i];
    q.tl = f[24];
    q.pl = f[25];
}

template <class F> __device__ __forceinline__ void store_state_rec(unsigned char* base, int sl, const StateT<F>& t) {
    F f[kStateWords];
    f[0] = t.xh; f[1] = t.yh; f[2] = t.zh; f[3] = t.xl; f[4] = t.yl; f[5] = t.zl;
    f[6] = t.k; f[7] = t.phi; f[8] = t.th;
#pragma unroll
    for (int i = 0; i < 21; ++i) f[9 + i] = t.c[i];
    f[30] = t.tl; f[31] = t.pl;
    store_rec<F, kStateWords>(base, sl, f);
}

// A prediction's record also holds the direction at the crossing (sin phi, cos phi, sin theta, cos
// theta, as propagate_core returns it), for k_find.
template <class F>
__device__ __forceinline__ void store_pred_rec(unsigned char* base, int sl, const PredT<F>& q, const F dir[4]) {
    F f[kStateWords];
    f[0] = q.xh; f[1] = q.yh; f[2] = q.zh; f[3] = q.xl; f[4] = q.yl; f[5] = q.zl;
    f[6] = q.k; f[7] = q.phi; f[8] = q.th;
#pragma unroll
    for (int i = 0; i < 15; ++i) f[9 + i] = q.c[i];
    f[24] = q.tl; f[25] = q.pl;
#pragma unroll
    for (int i = 0; i < 4; ++i) f[26 + i] = dir[i];
    f[30] = F(0); f[31] = F(0);
    store_rec<F, kStateWords>(base, sl, f);
}

// The words of a prediction that the window and the chi2 take: positions, the
// position covariance, the direction.
template <class F>
__device__ __forceinline__ void load_pred_rec(const unsigned char* __restrict__ base, int sl, PredT<F>& q, F dir[4]) {
    using V = typename Vec16<F>::T;
    constexpr int per = 16 / sizeof(F);
    const V* v = reinterpret_cast<const V*>(base) + word_at<rec_vecs<F>()>(sl, 0);
    F f[kStateWords];
#pragma unroll
    for (int j = 0; j < kStateWords / per; ++j)
        if (j * per < 12 || j * per >= 24) unpack16(v[j * (kTile * kGroup)], f + per * j);
        else
#pragma unroll
            for (int i = 0; i < per; ++i) f[per * j + i] = F(0);
    unpack_pred(f, q);
#pragma unroll
    for (int i = 0; i < 4; ++i) dir[i] = f[26 + i];
}

// The record of a seed (one after another, in the seeds' own order).
template <class F> __device__ __forceinline__ void load_seed_rec(const F* __restrict__ r, F* f) {
    using V = typename Vec16<F>::T;
    constexpr int per = 16 / sizeof(F);
#pragma unroll
    for (int j = 0; j < kStateWords / per; ++j) unpack16(reinterpret_cast<const V*>(r)[j], f + per * j);
}

// slot meta: (score, chi2 sum, nfound | nholes << 8 | stopped << 16, alive)
__device__ __forceinline__ int4 pack_meta(float score, float chi2s, int nfound, int nholes, bool stopped, bool alive) {
    return make_int4(__float_as_int(score), __float_as_int(chi2s), nfound | (nholes << 8) | ((int)stopped << 16),
                     (int)alive);
}

// Appends v to list (count at *cnt) for the lanes with pred set: one atomic per warp.
__device__ __forceinline__ void warp_append(bool pred, int v, int* list, int* cnt) {
    const unsigned m = __ballot_sync(kFull, pred);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(cnt, __popc(m));
    base = __shfl_sync(kFull, base, leader);
    if (pred) list[base + __popc(m & ((1u << lane) - 1u))] = v;
}

__device__ __forceinline__ void load_geom_smem(const DevGeom* __restrict__ gp, DevGeom& g) {
    const int4* src = reinterpret_cast<const int4*>(gp);
    int4* dst = reinterpret_cast<int4*>(&g);
    for (int i = threadIdx.x; i < (int)(sizeof(DevGeom) / 16); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
}

// Adds the threads' work counts to the call's counters, one atomic per warp and count.  A thread's own
// counts are below kCountCap, so that a warp's sum fits 32 bits (64-bit counts took registers that
// k_move and k_find do not have): a thread takes at most 2^31 slots / 9,728 threads of the smallest
// launch, with 8 updates or a few dozen Newton iterations each; k_find, whose windows can hold any
// number of hits, adds its counts to the call's counters whenever they reach the cap.
constexpr int kCountCap = 1 << 26;
__device__ __forceinline__ void add_counters(unsigned long long* counters, int c0, int c1, int c2, int c3, int c4) {
    const int c[5] = {c0, c1, c2, c3, c4};
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const long long sum = (long long)__reduce_add_sync(kFull, c[k]);
        if ((threadIdx.x & 31) == 0 && sum) atomicAdd(counters + k, (unsigned long long)sum);
    }
}

struct BuildArgs {
    const DevGeom* geom;
    DevParams P;
    HitStore H;
    SeedStore S;
    BuildOutDev out;
    BuildWork w;
    unsigned long long* counters;
    int slots;       // slots of the arrays (whole tiles)
    int nfound0;     // hits a track has when its search starts (3 seed hits forwards, 0 backwards)
};

// Child descriptor (one int4 per slot): parent slot | kind << 4 | disk << 8, its hit (K_HIT) or the
// seed (K_SEED), its score, its missed layers.  disk: the parent's prediction lies
// on a disk.
__device__ __forceinline__ int4 pack_child(int parent, int kind, bool disk, int q, float score, int nholes) {
    return make_int4(parent | (kind << 4) | ((int)disk << 8), q, __float_as_int(score), nholes);
}
__device__ __forceinline__ int child_parent(const int4& d) { return d.x & 15; }
__device__ __forceinline__ int child_kind(const int4& d) { return (d.x >> 4) & 15; }
__device__ __forceinline__ int child_surface(const int4& d) {
    return (d.x >> 8) & 1 ? MKGB_DISK : MKGB_BARREL;
}

template <class F> __device__ __forceinline__ const F* seed_states(const SeedStore& S) {
    if constexpr (sizeof(F) == 4) return S.state;
    else return S.state64;
}

// ---- round 0: the child in slot 0 of every seed with work is the seed itself
__global__ void __launch_bounds__(kThreads) k_start(BuildArgs a) {
    next_kernel_may_start();
    wait_for_last_kernel();
    const DevGeom* __restrict__ g = a.geom;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;   // seed position in the (event, eta, phi) order
    bool work = false;
    if (i < a.S.n) {
        const int seed = a.S.order[i];
        const int4 inf = a.S.info[seed];
        int pos = 0, start = 0, nsteps = 0, event = 0;
        if (inf.w == 0) {
            const int pb = g->plan_off[inf.x];
            start = inf.y;
            pos = pb + start;
            nsteps = g->plan_off[inf.x + 1] - pos;
            if (nsteps < 0) nsteps = 0;
            event = inf.z;
        }
        a.w.sinfo[i] = make_int4(pos, start, nsteps, event);
        a.w.fin[i] = -1;
        work = nsteps > 0;
        const int4 dead = make_int4(0, 0, 0, 0);
#pragma unroll
        for (int c = 1; c < kGroup; ++c) a.w.meta[0][slot_at(i * kGroup + c)] = dead;
        a.w.meta[0][slot_at(i * kGroup)] = work ? pack_meta(0.0f, 0.0f, a.nfound0, 0, false, true) : dead;
        if (work) a.w.child[slot_at(i * kGroup)] = pack_child(0, K_SEED, false, seed, 0.0f, 0);
    }
    warp_append(work, i * kGroup, a.w.live[0], a.w.counts + 0);
    warp_append(work, i, a.w.seeds[0], a.w.counts + 2);
}

// The update of a child redone in FP64 from its parent's FP32 prediction, narrowed (mixed
// precision, growth G3).  False: the update failed.
__device__ __noinline__ bool update_fp64(int surface, const Pred& pq, const float4* __restrict__ pay, int id,
                                         State& t) {
    PredT<double> qd;
    qd.xh = pq.xh; qd.yh = pq.yh; qd.zh = pq.zh; qd.xl = pq.xl; qd.yl = pq.yl; qd.zl = pq.zl;
    qd.k = pq.k; qd.phi = pq.phi; qd.th = pq.th; qd.tl = pq.tl; qd.pl = pq.pl;
#pragma unroll
    for (int q = 0; q < 15; ++q) qd.c[q] = pq.c[q];
    double m[3], v[6];
    load_hit(pay, id, m, v, nullptr);
    StateT<double> td;
    const bool ok = kalman_update(surface, qd, m[0], m[1], m[2], v, td);
    if (ok) narrow_state(td, t);
    return ok;
}

// The state of a child from its record words f (its parent's prediction, or its own state for a
// child that did not cross the parent's layer or is a seed).  Returns 0, 1 (the update failed) or 2
// (an innovation covariance that FP32 cannot resolve: to be redone by update_fp64).
template <class F>
__device__ __forceinline__ int child_state(const BuildArgs& a, const int4& d, const F* f, const F m[3], const F v[6],
                                           StateT<F>& t) {
    const int kind = child_kind(d);
    if (kind != K_HIT && kind != K_MISS) {
        t.xh = f[0]; t.yh = f[1]; t.zh = f[2]; t.xl = f[3]; t.yl = f[4]; t.zl = f[5];
        t.k = f[6]; t.phi = f[7]; t.th = f[8];
#pragma unroll
        for (int q = 0; q < 21; ++q) t.c[q] = f[9 + q];
        t.tl = f[30];
        t.pl = f[31];
        return 0;
    }
    PredT<F> pq;
    unpack_pred(f, pq);
    const int surface = child_surface(d);
    if (kind == K_HIT) {
        float kap = 0.0f;
        if (!kalman_update(surface, pq, m[0], m[1], m[2], v, t, &kap)) return 1;
        return sizeof(F) == 4 && a.P.kappa_fp64 > 0.0f && kap > a.P.kappa_fp64 ? 2 : 0;
    }
    pred_to_state(surface, pq, t);
    return 0;
}

// ---- a11 and a4-a7 for every live child of round tau: its state, then its way to the next layer

// REDO: the children whose update the first launch left to FP64 (the
// round's redo list).  BWD: the backward search (Sec. 2.2), crossing the layers behind the candidate.
template <class F, int TH, int MINB, bool BWD = false, bool REDO = false>
__global__ void __launch_bounds__(TH, MINB) k_move(BuildArgs a, int tau) {
    __shared__ DevGeom g;
    next_kernel_may_start();
    if (!REDO) load_geom_smem(a.geom, g);
    wait_for_last_kernel();
    const int cur = tau & 1, nxt = cur ^ 1;
    const int n = REDO ? a.w.counts[4] : a.w.counts[cur];
    if (REDO) {
        if (n == 0) return;
        load_geom_smem(a.geom, g);
    }
    const int* __restrict__ list = REDO ? a.w.redo : a.w.live[cur];
    if (!REDO && blockIdx.x == 0 && threadIdx.x == 0) {   // lists filled by this round's k_merge
        a.w.counts[nxt] = 0;
        a.w.counts[2 + nxt] = 0;
    }
    const DevParams& P = a.P;
    const unsigned char* __restrict__ prev = a.w.rec[nxt];
    unsigned char* __restrict__ rec = a.w.rec[cur];
    int c_steps = 0, c_newton = 0, c_failed = 0;
    const int stride = gridDim.x * TH;
    // the descriptor of the next child is loaded one child ahead: it names the record to read
    const int4 none = make_int4(0, 0, 0, 0);
    // the redo list is dealt out to the SMs one by one, like every FP64 redo (k_fit.cu)
    const int lane0 = REDO ? blockIdx.x + gridDim.x * threadIdx.x : threadIdx.x;
    const int base0 = REDO ? 0 : blockIdx.x * TH;
    const int first = base0 + lane0;
    int sl_next = first < n ? list[first] : 0;
    int4 d_next = first < n ? a.w.child[slot_at(sl_next)] : none;
    for (int base = base0; base < n; base += stride) {
        // the warps of a block start a child together: they share the fetches of the loop's code
        __syncthreads();
        const int idx = base + lane0;
        const int sl = sl_next;
        const int4 d = d_next;
        bool crossed = false;
        int4 si = none;
        StateT<F> t;
        int fail = 4;   // no child
        if (idx < n) {
            si = a.w.sinfo[sl / kGroup];
            F f[kStateWords];
            F m[3] = {F(0), F(0), F(0)}, v[6] = {F(0), F(0), F(0), F(0), F(0), F(0)};
            if (child_kind(d) == K_SEED)
                load_seed_rec(seed_states<F>(a.S) + (int64_t)d.y * kSeedStateStride, f);
            else
                load_rec<F, kStateWords>(prev, (sl & ~(kGroup - 1)) | child_parent(d), f);
            if (child_kind(d) == K_HIT) load_hit(a.H.pay, d.y, m, v, nullptr);
            if (idx + (int64_t)stride < n) {
                sl_next = list[idx + stride];
                d_next = a.w.child[slot_at(sl_next)];
            }
            if constexpr (REDO) {
                Pred pq;
                unpack_pred(f, pq);
                fail = update_fp64(child_surface(d), pq, a.H.pay, d.y, t) ? 0 : 3;
            } else {
                fail = child_state(a, d, f, m, v, t);
            }
        }
        // children with and without a hit go on together (without this the compiler makes a copy of
        // the rest for each kind: 17.7 of 32 lanes active instead of 28)
        __syncwarp();
        // the next child's record and hit on their way to the L2 (64-event search 15.8 -> 15.45 ms)
        if (!REDO && idx + (int64_t)stride < n && child_kind(d_next) != K_SEED) {
            const char* r = reinterpret_cast<const char*>(prev) +
                            16 * word_at<rec_vecs<F>()>((sl_next & ~(kGroup - 1)) | child_parent(d_next), 0);
#pragma unroll
            for (int j = 0; j < rec_vecs<F>(); ++j) prefetch_l2(r + 16 * j * (kTile * kGroup));
            if (child_kind(d_next) == K_HIT) prefetch_l2(a.H.pay + 3 * (int64_t)d_next.y);
        }
        int nh_kind = K_NONE;
        if (fail == 0) {
            const DevLayer& L = g.layers[g.plan[si.x + tau]];
            PredT<F> q;
            F dir[4];
            int newton = 0;
            const int r = propagate_core<F, F, BWD>(L, g.cB, P.material, t, t.c, q, q.c, newton, dir);
            c_newton += newton;
            crossed = r > 0;
            if (crossed) {
                store_pred_rec(rec, sl, q, dir);
                ++c_steps;
            } else if (r == 0) {   // not crossed: the next child is this state
                nh_kind = K_SKIP;
                store_state_rec(rec, sl, t);
            }
        } else if (fail == 2) {   // redone in FP64 by the round's second launch
            a.w.redo[atomicAdd(a.w.counts + 4, 1)] = sl;
        } else if (fail != 4) {   // the child is dropped
            a.w.meta[cur][slot_at(sl)].w = 0;
            c_failed += fail == 1;
        }
        // (a crossed layer's list is k_find's)
        if (!crossed && fail != 4) a.w.ls[word_at<2>(sl, 0)] = make_int4(0, nh_kind, d.z, 0);
        warp_append(crossed, sl, a.w.found, a.w.counts + 5);
    }
    add_counters(a.counters, c_steps, 0, -c_failed, 0, c_newton);
}

// ---- a8-a9 for every candidate that crossed its layer in round tau
//
// Apart from k_move because the two want different things: this one waits for chains of small
// loads (bin bounds, hits, their measurements) and needs many warps, that one computes and needs
// registers.  It reads five of the record's eight words.
template <class F, int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) k_find(BuildArgs a, int tau) {
    __shared__ DevGeom g;
    // per-thread sorted list of hit children (chi2 asc, id asc), one column per thread
    __shared__ float s_x2[kGroup][TH];
    __shared__ int s_id[kGroup][TH];
    __shared__ int s_q[kQueue][TH];   // ids of the hits inside the window, waiting for their chi2
    next_kernel_may_start();
    load_geom_smem(a.geom, g);
    wait_for_last_kernel();
    const int tx = threadIdx.x;
    const int cur = tau & 1;
    const DevParams& P = a.P;
    const int n = a.w.counts[5];
    int c_chi2 = 0, c_tested = 0;
    const int stride = gridDim.x * TH;
    for (int idx = blockIdx.x * TH + tx; idx < n; idx += stride) {
        const int sl = a.w.found[idx];
        const int4 d = a.w.child[slot_at(sl)];
        const int4 si = a.w.sinfo[sl / kGroup];
        PredT<F> q;
        F dir[4];
        load_pred_rec(a.w.rec[cur], sl, q, dir);
        const DevLayer& L = g.layers[g.plan[si.x + tau]];
        const float score = __int_as_float(d.z);
        const bool miss = d.w < P.max_holes;
        const int nh_kind = miss ? K_MISS : K_STOP;
        const float nh_score = miss ? score - P.score_hole : score;
        int n_h = 0;
        const FrameT<F> fr = frame_of(L.kind, q.xh, q.yh, dir[0], dir[1], dir[2], dir[3]);
        const WindowT<F> w = window(L, P, q, fr);
        const float eps = 1e-5f;
        const float fe0 = (w.eta - w.deta - eps - L.eta_lo) * L.eta_scale;
        const float fe1 = (w.eta + w.deta + eps - L.eta_lo) * L.eta_scale;
        const int e0 = fe0 >= 0.0f ? (int)fminf(floorf(fe0), (float)(L.n_eta - 1)) : 0;
        const int e1 = fe1 >= 0.0f ? (int)fminf(floorf(fe1), (float)(L.n_eta - 1)) : 0;
        const float pscale = L.n_phi * (1.0f / kTwoPi);
        const int f0 = (int)floorf((w.phi - w.dphi - eps + kPi) * pscale);
        const int f1 = (int)floorf((w.phi + w.dphi + eps + kPi) * pscale);
        int nf = f1 - f0 + 1;
        int fa = f0 % L.n_phi;
        if (fa < 0) fa += L.n_phi;
        if (nf >= L.n_phi) {
            nf = L.n_phi;
            fa = 0;
        }
        const int run1 = min(nf, L.n_phi - fa), run2 = nf - run1;
        const int64_t bb = (int64_t)si.w * g.bins_per_event + L.bin_base;
        // the window's bins are ranges of hits, one or two (around phi = pi) per eta row; the bounds
        // of the next range are loaded while the hits of this one are tested, two at a time, and
        // the hits inside the window are queued, so that the lanes of a warp meet at the chi2
        const int nr = run2 > 0 ? 2 : 1, n_ranges = (e1 - e0 + 1) * nr;
        auto bounds = [&](int rg, int& q0, int& q1) {
            const int64_t at = bb + (int64_t)(e0 + (rg >> (nr - 1))) * L.n_phi + ((rg & (nr - 1)) ? 0 : fa);
            q0 = __ldg(a.H.bin_start + at);
            q1 = __ldg(a.H.bin_start + at + ((rg & (nr - 1)) ? run2 : run1));
        };
        auto inside = [&](const float4& ep) {
            return fabs(F(ep.x) - w.eta) <= w.deta && fabs(wrap_pi(F(ep.y) - w.phi)) <= w.dphi;
        };
        int rg = 0, hq = 0, q1 = 0, hq_next = 0, q1_next = 0;
        if (n_ranges > 0) bounds(0, hq_next, q1_next);
        for (bool more = true; more;) {
            int nq = 0;
            while (nq < kQueue) {
                if (hq >= q1) {
                    if (rg >= n_ranges) {
                        more = false;
                        break;
                    }
                    hq = hq_next;
                    q1 = q1_next;
                    if (++rg < n_ranges) bounds(rg, hq_next, q1_next);
                    continue;
                }
                const bool two = hq + 1 < q1 && nq + 1 < kQueue;
                const float4 ep0 = __ldg(a.H.hb + hq), ep1 = __ldg(a.H.hb + hq + (int)two);
                c_tested += 1 + two;
                if (inside(ep0)) s_q[nq++][tx] = __float_as_int(ep0.z);
                if (two && inside(ep1)) s_q[nq++][tx] = __float_as_int(ep1.z);
                hq += 1 + two;
            }
            c_chi2 += nq;
            for (int jq = 0; jq < nq; ++jq) {
                const int id = s_q[jq][tx];
                F mh[3], vh[6];
                F x2f;
                load_hit(a.H.pay, id, mh, vh, nullptr);
                const bool okx = chi2_hit(fr, q, mh[0], mh[1], mh[2], vh, x2f);
                if (!okx || !(x2f < F(P.chi2_cut))) continue;
                const float x2 = float(x2f);   // scores and child order in FP32
                // insert into the sorted list (kept to its first kGroup entries)
                int j = n_h < kGroup ? n_h : kGroup - 1;
                if (n_h == kGroup && !(x2 < s_x2[j][tx] || (x2 == s_x2[j][tx] && id < s_id[j][tx]))) continue;
                while (j > 0 && (x2 < s_x2[j - 1][tx] || (x2 == s_x2[j - 1][tx] && id < s_id[j - 1][tx]))) {
                    s_x2[j][tx] = s_x2[j - 1][tx];
                    s_id[j][tx] = s_id[j - 1][tx];
                    --j;
                }
                s_x2[j][tx] = x2;
                s_id[j][tx] = id;
                if (n_h < kGroup) ++n_h;
            }
        }
        // the child list: its header and first two hits, the other hits apart
        int4* lrec = a.w.ls + word_at<2>(sl, 0);
        lrec[0] = make_int4(n_h | (L.kind == MKGB_DISK ? kDiskBit : 0), nh_kind, __float_as_int(nh_score), 0);
        for (int j = 0; j < n_h; j += 2) {
            const int4 e = make_int4(__float_as_int(s_x2[j][tx]), s_id[j][tx],
                                     __float_as_int(j + 1 < n_h ? s_x2[j + 1][tx] : kBig),
                                     j + 1 < n_h ? s_id[j + 1][tx] : 0);
            if (j == 0)
                lrec[kTile * kGroup] = e;
            else
                a.w.ls_more[word_at<3>(sl, j / 2 - 1)] = e;
        }
        if (c_tested >= kCountCap) {   // (c_chi2 is no larger; one window adds at most its layer's hits)
            atomicAdd(a.counters + 1, (unsigned long long)c_chi2);
            atomicAdd(a.counters + 3, (unsigned long long)c_tested);
            c_chi2 = 0;
            c_tested = 0;
        }
    }
    add_counters(a.counters, 0, c_chi2, 0, c_tested, 0);
}

// ---- a10 for every seed with a live candidate in round tau
//
// Eight lanes per seed, lane = parent slot.  Every child of the seed puts its key (score, then parent
// slot, then place in the parent's list) into shared memory and counts the keys above its own: that
// count is its slot among the N best, so a parent's lane writes its kept children straight from its
// registers, with no exchange of their contents and no round per rank.  64 registers (12 bytes spilled)
// for 32 warps per SM.  64 events: 4.3 ms (4.8 with a walk over the keys per child); eight lanes
// exchanging keys and contents by shuffles, a round per rank: 7.4 ms; one thread per seed with its eight
// best in registers: 3.8 ms, but 1.3 times the whole search of one event (0.86 against 0.66 ms), where
// the latency of a thread's serial lists counts.
constexpr int kNoHit = 15;   // place of the child without a hit
constexpr int kSeedKeys = kGroup * (kGroup + 1);
__device__ __forceinline__ unsigned long long child_key(float score, int slot, int place) {
    unsigned u = __float_as_uint(score);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)u << 32) | (unsigned)(0xffff - (slot << 4 | place));
}

template <class F, int TH, int MINB>
__global__ void __launch_bounds__(TH, MINB) k_merge(BuildArgs a, int tau) {
    __shared__ unsigned long long s_key[TH / kGroup][kSeedKeys];
    __shared__ int s_cnt[2][TH / 32], s_base[2];
    next_kernel_may_start();
    wait_for_last_kernel();
    const int cur = tau & 1, nxt = cur ^ 1;
    const DevParams& P = a.P;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, slot = lane & 7, gbase = lane & ~7;
    unsigned long long* keys = s_key[threadIdx.x / kGroup];
    const int n = a.w.counts[2 + cur];
    const int* __restrict__ list = a.w.seeds[cur];
    if (blockIdx.x == 0 && threadIdx.x == 0) {   // the redo list and k_find's list of the next round
        a.w.counts[4] = 0;
        a.w.counts[5] = 0;
    }
    int c_upd = 0;
    const int gstride = gridDim.x * (TH / kGroup);
    for (int bg = blockIdx.x * (TH / kGroup); bg < n; bg += gstride) {   // uniform over the block
        const int gi = bg + wid * 4 + (lane >> 3);
        const bool gact = gi < n;
        const int i = list[gact ? gi : bg];
        const int nsteps = a.w.sinfo[i].z;
        const int sl = i * kGroup + slot;
        // all of the slot's words at once (those of an empty slot are not used)
        const int4 mt = a.w.meta[cur][slot_at(sl)];
        int4 e0 = make_int4(0, K_NONE, 0, 0), e1 = e0;
        if (mt.w != 0) {
            e0 = a.w.ls[word_at<2>(sl, 0)];
            e1 = a.w.ls[word_at<2>(sl, 1)];
        }
        const float score = __int_as_float(mt.x);
        const bool alive = gact && mt.w != 0, stopped = ((mt.z >> 16) & 1) != 0;
        const bool searched = alive && !stopped;
        const int n_h = searched ? e0.x & (kDiskBit - 1) : 0;
        const int nh_kind = !alive ? K_NONE : stopped ? K_CARRY : e0.y;
        const float nh_score = stopped ? score : __int_as_float(e0.z);
        const bool disk = (e0.x & kDiskBit) != 0;
        const bool has_nh = nh_kind != K_NONE;
        auto hit_entry = [&](int j) {   // (chi2, id) of the parent's j-th hit
            if (j == 0) return make_int2(e1.x, e1.y);
            if (j == 1) return make_int2(e1.z, e1.w);
            return reinterpret_cast<const int2*>(a.w.ls_more + word_at<3>(sl, j / 2 - 1))[j & 1];
        };
        auto hit_score = [&](int j) { return score + P.score_hit - __int_as_float(hit_entry(j).x); };

        // ---- the seed's children and the slots they take
        const int cnt = n_h + (int)has_nh;
        int end = cnt;
#pragma unroll
        for (int d = 1; d < kGroup; d <<= 1) {
            const int o = __shfl_up_sync(kFull, end, d, kGroup);
            if (slot >= d) end += o;
        }
        const int total = __shfl_sync(kFull, end, kGroup - 1, kGroup);
        for (int j = 0; j < n_h; ++j) keys[end - cnt + j] = child_key(hit_score(j), slot, j);
        if (has_nh) keys[end - 1] = child_key(nh_score, slot, kNoHit);
        __syncwarp();
        // most parents have one hit child and one without: both are ranked in one walk over the keys
        const unsigned long long k_first = n_h > 0 ? keys[end - cnt] : ~0ull, k_nh = has_nh ? keys[end - 1] : ~0ull;
        int r_first = 0, nh_slot = 0;
        for (int q = 0; q < total; ++q) {
            const unsigned long long k = keys[q];
            r_first += k > k_first;
            nh_slot += k > k_nh;
        }
        int kept_hits = 0;         // the first of the parent's hits are kept, at these slots (4 bits each)
        unsigned hit_slots = 0, kept = 0, live = 0;
        for (int j = 0; j < n_h; ++j) {
            int r = r_first;
            if (j > 0) {
                const unsigned long long kj = keys[end - cnt + j];
                r = 0;
                for (int q = 0; q < total; ++q) r += keys[q] > kj;
            }
            if (r >= P.max_cands) break;   // the others come after it
            hit_slots |= (unsigned)r << (4 * j);
            live |= 1u << r;
            ++kept_hits;
        }
        c_upd += kept_hits;
        const bool nh_kept = nh_slot < P.max_cands && has_nh;
        const bool nh_stop = nh_kept && nh_kind == K_STOP;
        kept = live | (nh_kept ? 1u << nh_slot : 0u);
        if (nh_kept && (nh_kind == K_MISS || nh_kind == K_SKIP)) live |= 1u << nh_slot;
        const bool more = gact && tau + 1 < nsteps;
        const unsigned used = nh_kept && nh_kind == K_CARRY ? 1u << ((mt.z >> 18) & 7) : 0u;   // stop records in use
        const unsigned all_kept = __reduce_or_sync(kFull, kept << gbase);
        const unsigned all_live = __reduce_or_sync(kFull, more ? live << gbase : 0u);
        const unsigned all_used = __reduce_or_sync(kFull, used << gbase);
        const unsigned all_stop = __ballot_sync(kFull, nh_stop);   // (also the end of the keys' use)
        const unsigned seed_kept = (all_kept >> gbase) & 0xffu;
        const bool p_seed = more && seed_kept != 0 && slot == 0;
        const unsigned ms = __ballot_sync(kFull, p_seed);
        if (lane == 0) {
            s_cnt[0][wid] = __popc(all_live);
            s_cnt[1][wid] = __popc(ms);
        }
        __syncthreads();
        int bl = 0, bs = 0, tl = 0, ts = 0;
#pragma unroll
        for (int q = 0; q < TH / 32; ++q) {
            bl += q < wid ? s_cnt[0][q] : 0;
            bs += q < wid ? s_cnt[1][q] : 0;
            tl += s_cnt[0][q];
            ts += s_cnt[1][q];
        }
        if (threadIdx.x == 0) {   // the block's two list reservations, in flight during the writes below
            s_base[0] = tl ? atomicAdd(a.w.counts + nxt, tl) : 0;
            s_base[1] = ts ? atomicAdd(a.w.counts + 2 + nxt, ts) : 0;
        }

        // ---- the kept children: descriptors, meta, trail
        auto put = [&](int r, int kind, float child_score, int4 cm, int code, int hq) {
            const int cs = i * kGroup + r;
            const int at = slot_at(cs);
            a.w.child[at] = pack_child(slot, kind, disk, hq, child_score, (cm.z >> 8) & 0xff);
            a.w.meta[nxt][at] = cm;
            a.w.trail[(int64_t)tau * a.slots + at] = ((code + 4) << 3) | slot;
        };
        const float chi2s = __int_as_float(mt.y);
        const int nfound = mt.z & 0xff, nholes = (mt.z >> 8) & 0xff;
        for (int j = 0; j < kept_hits; ++j) {   // (a child whose update fails is dropped by the next k_move)
            const int2 e = hit_entry(j);
            const float sc = hit_score(j);
            put((hit_slots >> (4 * j)) & 15, K_HIT, sc,
                pack_meta(sc, chi2s + __int_as_float(e.x), nfound + 1, nholes, false, true), e.y, e.y);
        }
        if (nh_kept) {
            const bool stop = nh_kind == K_STOP || nh_kind == K_CARRY;
            int4 cm = pack_meta(nh_score, chi2s, nfound, nholes + (nh_kind == K_MISS), stop, true);
            if (nh_kind == K_CARRY) cm.z |= mt.z & (15 << 17);
            if (nh_kind == K_STOP) {   // the prediction where it stopped is put aside for the search's end
                unsigned free = ~(all_used >> gbase) & 0xffu;
                for (int q = __popc((all_stop >> gbase) & ((1u << slot) - 1u)); q > 0; --q) free &= free - 1;
                const int k = __ffs(free) - 1;
                cm.z |= ((int)disk << 17) | (k << 18);
                F f[kPredWords];
                load_rec<F, kPredWords>(a.w.rec[cur], sl, f);
                store_rec<F, kPredWords>(a.w.stop, i * kGroup + k, f);
            }
            put(nh_slot, nh_kind, nh_score, cm,
                nh_kind == K_MISS ? MKGB_HIT_MISS : nh_kind == K_SKIP ? MKGB_HIT_SKIP : MKGB_HIT_STOP, 0);
        }
        if (gact && !((seed_kept >> slot) & 1)) a.w.meta[nxt][slot_at(sl)] = make_int4(0, 0, 0, 0);
        if (gact && slot == 0 && !p_seed) a.w.fin[i] = tau + 1;

        // ---- next-round lists, in the seeds' and slots' order: a block's 32 seeds stay together, or the
        // lists, and with them the tiles that a warp of the next round touches, would come apart in
        // pieces of a warp's four seeds (27.6 ms per 64-event search)
        __syncthreads();
        const unsigned below = (1u << lane) - 1u;
        if ((all_live >> lane) & 1) a.w.live[nxt][s_base[0] + bl + __popc(all_live & below)] = sl;
        if (p_seed) a.w.seeds[nxt][s_base[1] + bs + __popc(ms & below)] = i;
    }
    // a hit child that is kept counts as an update: k_move and k_finish take back the ones that fail
    add_counters(a.counters, 0, 0, c_upd, 0, 0);
}

// ---- best candidate per seed and its hit list (a13); one thread per seed.  REDO: the seeds that the
// first launch left because the last update of their best candidate is one for FP64.
template <class F, bool REDO>
__global__ void __launch_bounds__(kThreads) k_finish(BuildArgs a) {
    if (!REDO) next_kernel_may_start();
    wait_for_last_kernel();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (REDO ? a.w.counts[4] : a.S.n)) return;
    if (REDO) i = a.w.redo[i];
    const int rounds = a.w.fin[i];   // rounds searched, -1 none
    const int seed = a.S.order[i];
    int4 mt = make_int4(0, 0, 0, 0);
    int best = -1;
    StateT<F> t;
    // the last round's children still have to take their hits: the best one, the next if that fails
    for (int r = 0; rounds > 0 && best < 0 && r < kGroup; ++r) {
        const int cs = i * kGroup + r;
        mt = a.w.meta[rounds & 1][slot_at(cs)];
        if (mt.w == 0) continue;
        F f[kStateWords];
        F m[3] = {F(0), F(0), F(0)}, v[6] = {F(0), F(0), F(0), F(0), F(0), F(0)};
        int4 d = pack_child(0, K_MISS, (mt.z >> 17) & 1, 0, 0.0f, 0);   // stopped: its record is a prediction
        if ((mt.z >> 16) & 1) {
            load_rec<F, kStateWords>(a.w.stop, i * kGroup + ((mt.z >> 18) & 7), f);
        } else {
            d = a.w.child[slot_at(cs)];
            load_rec<F, kStateWords>(a.w.rec[(rounds & 1) ^ 1], i * kGroup + child_parent(d), f);
            if (child_kind(d) == K_HIT) load_hit(a.H.pay, d.y, m, v, nullptr);
        }
        int fail = child_state(a, d, f, m, v, t);
        if (fail == 2) {
            if constexpr (REDO) {
                Pred q;
                unpack_pred(f, q);
                fail = update_fp64(child_surface(d), q, a.H.pay, d.y, t) ? 0 : 1;
            } else {
                a.w.redo[atomicAdd(a.w.counts + 4, 1)] = i;
                return;
            }
        }
        if (fail == 0) best = r;
        else if (fail == 1) atomicAdd(a.counters + 2, ~0ull);   // k_merge counted its update (- 1)
    }
    int* hrow = a.out.hits + (int64_t)seed * a.out.max_plan;
    int* orow = a.out.ovl ? a.out.ovl + (int64_t)seed * a.out.max_plan : nullptr;
    float* po = a.out.params + 6 * (int64_t)seed;
    float* co = a.out.cov + 21 * (int64_t)seed;
    int q0 = a.out.max_plan, q1 = a.out.max_plan;   // steps of the row that the search covered
    if (best >= 0) {
        store_state6(t, po, co);
        a.out.chi2[seed] = __int_as_float(mt.y);
        a.out.score[seed] = __int_as_float(mt.x);
        a.out.nfound[seed] = mt.z & 0xff;
        a.out.nholes[seed] = (mt.z >> 8) & 0xff;
        const int4 si = a.w.sinfo[i];
        q0 = si.y;
        q1 = si.y + min(rounds, si.z);
        int s_ = best;
        for (int tau = min(rounds, si.z) - 1; tau >= 0; --tau) {
            const int64_t at = (int64_t)tau * a.slots + slot_at(i * kGroup + s_);
            const int v = a.w.trail[at];
            const int code = (v >> 3) - 4;
            hrow[si.y + tau] = code;
            s_ = v & 7;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 6; ++q) po[q] = 0.0f;
#pragma unroll
        for (int q = 0; q < 21; ++q) co[q] = 0.0f;
        a.out.chi2[seed] = 0.0f;
        a.out.score[seed] = -INFINITY;
        a.out.nfound[seed] = 0;
        a.out.nholes[seed] = 0;
    }
    for (int q = 0; q < a.out.max_plan; ++q) {
        const bool covered = q >= q0 && q < q1;
        if (!covered) hrow[q] = MKGB_HIT_PRE;
        if (orow) orow[q] = -1;   // no module hits, no overlap hits
    }
}

int resident_grid(const void* kernel, int n_sms, int threads = kThreads) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    return n_sms * per_sm;
}

}  // namespace

namespace {

// Carves the work buffers out of one allocation (256-byte aligned pieces); with base == nullptr
// only the total size is computed.
size_t layout_build_work(char* base, int n_seeds, int max_plan_len, int word_bytes, BuildWork* w) {
    const size_t ns = (size_t)n_seeds, slots = tile_slots(n_seeds), wb = (size_t)word_bytes;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* r = base ? base + off : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return r;
    };
    BuildWork t = {};
    t.rec[0] = reinterpret_cast<unsigned char*>(take(slots * kStateWords * wb));
    t.rec[1] = reinterpret_cast<unsigned char*>(take(slots * kStateWords * wb));
    t.stop = reinterpret_cast<unsigned char*>(take(slots * kStateWords * wb));
    t.meta[0] = reinterpret_cast<int4*>(take(slots * 16));
    t.meta[1] = reinterpret_cast<int4*>(take(slots * 16));
    t.child = reinterpret_cast<int4*>(take(slots * 16));
    t.ls = reinterpret_cast<int4*>(take(slots * 32));
    t.ls_more = reinterpret_cast<int4*>(take(slots * 48));
    t.live[0] = reinterpret_cast<int*>(take(slots * 4));
    t.live[1] = reinterpret_cast<int*>(take(slots * 4));
    t.seeds[0] = reinterpret_cast<int*>(take(ns * 4));
    t.seeds[1] = reinterpret_cast<int*>(take(ns * 4));
    t.sinfo = reinterpret_cast<int4*>(take(ns * 16));
    t.fin = reinterpret_cast<int*>(take(ns * 4));
    t.trail = reinterpret_cast<int*>(take(slots * (size_t)max_plan_len * 4));
    t.redo = reinterpret_cast<int*>(take(slots * 4));
    t.found = reinterpret_cast<int*>(take(slots * 4));
    t.counts = reinterpret_cast<int*>(take(32));
    if (w) *w = t;
    return off;
}

// Start records of the backward search (Sec. 2.2): per track its state on its innermost found
// layer (p, c: 6 + 21 floats), the region from its eta as for a seed, and the first step of the
// geometry's reversed plan after that layer (info = (region, start, event, status); status 1
// when the layer is not in the plan or no layer lies inside it); the search order is the input
// order.
__global__ void __launch_bounds__(kThreads) k_bw_seed(const DevGeom* __restrict__ g, DevParams P, int n,
                                                      const float* __restrict__ p, const float* __restrict__ c,
                                                      const int* __restrict__ first_layer,
                                                      const int* __restrict__ event, float* state, int4* info,
                                                      int* order) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float* o = state + (int64_t)i * kSeedStateStride;
    const float* pi = p + 6 * (int64_t)i;
    const float* ci = c + 21 * (int64_t)i;
    o[0] = pi[0]; o[1] = pi[1]; o[2] = pi[2]; o[3] = 0.0f; o[4] = 0.0f; o[5] = 0.0f;
    o[6] = pi[3]; o[7] = pi[4]; o[8] = pi[5];
#pragma unroll
    for (int q = 0; q < 21; ++q) o[9 + q] = ci[q];
    o[30] = 0.0f; o[31] = 0.0f;
    const float eta = -logf(tanf(0.5f * pi[5]));
    int region = 0;
    if (g->n_regions > 1 && !(fabsf(eta) < P.barrel_eta_max)) region = eta > 0.0f ? 1 : 2;
    if (region >= g->n_regions) region = 0;
    int start = -1;
    const int pb = g->plan_off[region], len = g->plan_off[region + 1] - pb;
    for (int k = 0; k < len; ++k)   // g holds the reversed plans
        if (g->plan[pb + k] == first_layer[i]) start = k + 1;
    const bool ok = start > 0 && start < len;
    info[i] = make_int4(region, ok ? start : 0, event[i], ok ? 0 : 1);
    order[i] = i;
}

// Launch shapes of the round kernels (threads per block, minimum resident blocks per SM), one of
// which the autotuner picks: k_move x k_find.  The resident grid of each shape is computed once,
// before any capture.
//
// The FP64 redo: one block of 256 threads per SM.  Its list is empty or short at the default kappa_fp64
// (a block of 64 or of 512 threads does it as well), but a caller may lower that until every child is on
// it: searches of 160,000 seeds at 2^24, 2^8 and 1 took 2.38, 7.4 and 37.6 ms with blocks of 64 threads,
// 2.37, 3.7 and 9.6 with 256, 2.39, 3.7 and 9.4 with 512.
template <class F, int TH, int MINB, bool BWD, bool REDO = false> struct MoveShape {
    static int grid(int n_sms) {
        static int g = 0;
        if (!g) g = resident_grid((const void*)k_move<F, TH, MINB, BWD, REDO>, n_sms, TH);
        return g;
    }
    static void launch(cudaStream_t st, const BuildArgs& a, int tau, int n_sms) {
        launch_next(k_move<F, TH, MINB, BWD, REDO>, REDO ? n_sms : grid(n_sms), TH, st, true, a, tau);
    }
};
template <class F, int TH, int MINB> struct FindShape {
    static int grid(int n_sms) {
        static int g = 0;
        if (!g) g = resident_grid((const void*)k_find<F, TH, MINB>, n_sms, TH);
        return g;
    }
    static void launch(cudaStream_t st, const BuildArgs& a, int tau, int n_sms) {
        launch_next(k_find<F, TH, MINB>, grid(n_sms), TH, st, true, a, tau);
    }
};
template <class F, int TH, int MINB> struct MergeShape {
    static int grid(int n_sms) {
        static int g = 0;
        if (!g) g = resident_grid((const void*)k_merge<F, TH, MINB>, n_sms, TH);
        return g;
    }
    static void launch(cudaStream_t st, const BuildArgs& a, int tau, int n_sms) {
        launch_next(k_merge<F, TH, MINB>, grid(n_sms), TH, st, true, a, tau);
    }
};

// find_shape: k_move as blocks of 128 x 5, 128 x 4 (the default), 256 x 2, 64 x 8, 64 x 10, 128 x 3
// (threads x resident blocks per SM): searches of 64 events 15.91, 15.45, 15.63, 15.48, 15.92 and 16.44
// ms (125 registers at 16 warps per SM, no spills; 96 and 116 bytes spilled at 20; 139 at 12).
// select_shape: k_find as 128 x 6 (80 registers), 64 x 12, 128 x 8 (64 registers, 20 bytes spilled): 15.45,
// 15.50 and 15.34 ms, one event 0.647, 0.649 and 0.670.
template <class F, bool BWD, class Do> void with_move_shape(int shape, Do&& f) {
    if constexpr (sizeof(F) == 8) {
        f(MoveShape<F, 128, 1, BWD>());
    } else if constexpr (BWD) {   // the backward search: one shape
        f(MoveShape<F, 128, 4, BWD>());
    } else {
        switch (shape) {
            case 0: f(MoveShape<F, 128, 5, BWD>()); break;
            case 2: f(MoveShape<F, 256, 2, BWD>()); break;
            case 3: f(MoveShape<F, 64, 8, BWD>()); break;
            case 4: f(MoveShape<F, 64, 10, BWD>()); break;
            case 5: f(MoveShape<F, 128, 3, BWD>()); break;
            default: f(MoveShape<F, 128, 4, BWD>()); break;
        }
    }
}
template <class F, class Do> void with_find_shape(int shape, Do&& f) {
    if constexpr (sizeof(F) == 8) {
        f(FindShape<F, 128, 2>());
    } else {
        switch (shape) {
            case 1: f(FindShape<F, 64, 12>()); break;
            case 2: f(FindShape<F, 128, 8>()); break;
            default: f(FindShape<F, 128, 6>()); break;
        }
    }
}

template <class F, bool BWD = false>
cudaError_t launch_rounds(cudaStream_t st, const BuildArgs& a, int n, int max_plan_len, int n_sms, int find_shape,
                          int select_shape) {
    cudaError_t e = cudaMemsetAsync(a.w.counts, 0, 32, st);
    if (e != cudaSuccess) return e;
    const int nb = (n + kThreads - 1) / kThreads;
    k_start<<<nb, kThreads, 0, st>>>(a);
    for (int tau = 0; tau < max_plan_len; ++tau) {
        with_move_shape<F, BWD>(find_shape, [&](auto s) { decltype(s)::launch(st, a, tau, n_sms); });
        if constexpr (sizeof(F) == 4) {
            if (a.P.kappa_fp64 > 0.0f && tau > 0) MoveShape<F, 256, 1, BWD, true>::launch(st, a, tau, n_sms);
        }
        with_find_shape<F>(select_shape, [&](auto s) { decltype(s)::launch(st, a, tau, n_sms); });
        MergeShape<F, 256, 4>::launch(st, a, tau, n_sms);
    }
    launch_next(k_finish<F, false>, nb, kThreads, st, true, a);
    if constexpr (sizeof(F) == 4) {
        if (a.P.kappa_fp64 > 0.0f) launch_next(k_finish<F, true>, nb, kThreads, st, true, a);
    }
    return cudaGetLastError();
}

// The resident grids of every shape, asked for outside any capture.
template <class F, bool BWD> void prime_shapes_of(int n_sms) {
    for (int q = 0; q < 6; ++q) with_move_shape<F, BWD>(q, [&](auto s) { decltype(s)::grid(n_sms); });
    for (int q = 0; q < 3; ++q) with_find_shape<F>(q, [&](auto s) { decltype(s)::grid(n_sms); });
    MergeShape<F, 256, 4>::grid(n_sms);
}
template <class F> void prime_shapes(int n_sms) {
    prime_shapes_of<F, false>(n_sms);
    if constexpr (sizeof(F) == 4) prime_shapes_of<F, true>(n_sms);
}

cudaError_t enqueue_rounds(cudaStream_t st, const BuildArgs& a, int n, int max_plan_len, int n_sms, int find_shape,
                           int select_shape, bool backward = false) {
    if (a.w.mod)   // module hits loaded
        return launch_mod_rounds(st, a.geom, max_plan_len, a.P, a.H, a.S, a.out, a.w.mod, a.counters, n_sms, find_shape,
                                 select_shape, backward);
    if (backward) return launch_rounds<float, true>(st, a, n, max_plan_len, n_sms, find_shape, select_shape);
    // MKGB_FP64: the plain all-FP64 comparison path (same rounds, every Kalman step in FP64)
    if (a.P.precision == MKGB_FP64)
        return launch_rounds<double>(st, a, n, max_plan_len, n_sms, find_shape, select_shape);
    return launch_rounds<float>(st, a, n, max_plan_len, n_sms, find_shape, select_shape);
}

bool capturable(cudaStream_t st) {
    if (st == nullptr || st == cudaStreamLegacy || st == cudaStreamPerThread) return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) return false;
    return cs == cudaStreamCaptureStatusNone;   // inside a caller's capture: plain launches join it
}

}  // namespace

size_t build_work_bytes(int n_seeds, int max_plan_len, int precision, bool modular) {
    if (modular) return mod_work_bytes(n_seeds, max_plan_len, precision);
    return layout_build_work(nullptr, n_seeds, max_plan_len, precision == MKGB_FP64 ? 8 : 4, nullptr);
}

BuildWork carve_build_work(void* base, int n_seeds, int max_plan_len, int precision, bool modular) {
    BuildWork w;
    memset(&w, 0, sizeof(w));
    if (modular)
        w.mod = base;
    else
        layout_build_work(static_cast<char*>(base), n_seeds, max_plan_len, precision == MKGB_FP64 ? 8 : 4, &w);
    return w;
}

// The search of one call as a CUDA graph: the ~90 launches of the rounds (counters reset, k_start,
// per plan step k_move twice, k_find and k_merge, k_finish twice) are captured once and replayed while the
// arguments, the launch shapes and the stream stay the same.
struct BuildGraph {
    cudaGraphExec_t exec = nullptr;
    BuildArgs key;
    int n = -1, max_plan = -1, find_shape = -1, select_shape = -1;
    cudaStream_t st = nullptr;
    bool disabled = false;
};

BuildGraph* build_graph_create() { return new BuildGraph(); }

void build_graph_destroy(BuildGraph* gph) {
    if (!gph) return;
    if (gph->exec) cudaGraphExecDestroy(gph->exec);
    delete gph;
}

cudaError_t launch_build(cudaStream_t st, const DevGeom* g, int max_plan_len, DevParams P, HitStore H, SeedStore S,
                         BuildOutDev out, BuildWork w, unsigned long long* counters, int n_sms, int find_shape,
                         int select_shape, BuildGraph* gph, bool backward) {
    if (S.n == 0) return cudaSuccess;
    BuildArgs a;
    memset(&a, 0, sizeof(a));   // padding included: the graph cache compares arguments bytewise
    a.geom = g; a.P = P; a.H = H; a.S = S; a.out = out; a.w = w; a.counters = counters; a.slots = tile_slots(S.n);
    a.nfound0 = backward ? 0 : 3;
    if (w.mod)
        prime_mod_shapes(a.P.precision, n_sms);
    else if (a.P.precision == MKGB_FP64)
        prime_shapes<double>(n_sms);
    else
        prime_shapes<float>(n_sms);
    if (backward) {   // plain launches (the search's graph cache serves the forward search)
        if (P.precision == MKGB_FP64) return cudaErrorInvalidValue;
        return enqueue_rounds(st, a, S.n, max_plan_len, n_sms, find_shape, select_shape, true);
    }
    if (!gph || gph->disabled || !capturable(st))
        return enqueue_rounds(st, a, S.n, max_plan_len, n_sms, find_shape, select_shape);
    const bool same = gph->exec && gph->st == st && gph->n == S.n && gph->max_plan == max_plan_len &&
                      gph->find_shape == find_shape && gph->select_shape == select_shape &&
                      memcmp(&gph->key, &a, sizeof(a)) == 0;
    if (!same) {
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) {
            gph->disabled = true;
            return enqueue_rounds(st, a, S.n, max_plan_len, n_sms, find_shape, select_shape);
        }
        const cudaError_t le = enqueue_rounds(st, a, S.n, max_plan_len, n_sms, find_shape, select_shape);
        e = cudaStreamEndCapture(st, &graph);
        if (le != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return le;
        }
        if (e != cudaSuccess) return e;
        if (gph->exec) {
            cudaGraphExecDestroy(gph->exec);
            gph->exec = nullptr;
        }
        e = cudaGraphInstantiate(&gph->exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            gph->exec = nullptr;
            return e;
        }
        gph->key = a;
        gph->st = st;
        gph->n = S.n;
        gph->max_plan = max_plan_len;
        gph->find_shape = find_shape;
        gph->select_shape = select_shape;
    }
    return cudaGraphLaunch(gph->exec, st);
}

cudaError_t launch_bw_seed(cudaStream_t st, const DevGeom* g, DevParams P, int n, const float* p, const float* c,
                           const int* first_layer, const int* event, float* state, int4* info, int* order) {
    if (n == 0) return cudaSuccess;
    k_bw_seed<<<(n + kThreads - 1) / kThreads, kThreads, 0, st>>>(g, P, n, p, c, first_layer, event, state, info,
                                                                  order);
    return cudaGetLastError();
}

}  // namespace mk
