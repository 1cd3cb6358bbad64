// Derivative of the fit's total chi2 (growth row G1 of the fit over a known assignment, Sec. 4).
//
// d(sum of the predicted chi2 over tracks and layers) / d(per-layer alignment, per-layer material
// thickness scale, per-track starting parameters).  Alignment of layer l moves its hits,
// h' = h + d_l + w_l x (h - c_l), with c_l the origin for a cylinder and (0, 0, z_l) for a disk;
// the layer surfaces stay nominal.  The thickness scale multiplies x/X0 of the layer.
//
// The kernels run the FP32 fit step (fit_step below) on dual numbers (dual.cuh) carrying KD
// directional derivatives.
//
// Reverse sweep (the default, k_fit_adjoint, launched twice): a plain FP32 pass stores the input state
// of every step (a checkpoint per layer); then, from the last step back to the first, the step is
// redone from its checkpoint with its 34 inputs (27 state words, 6 alignment, 1 thickness scale)
// seeded KD at a time, and the adjoint of its output (d total / d output, starting at zero after
// the last step; the step's own chi2 enters with weight 1) is contracted with the output
// derivatives: d total / d input = dchi2_j / d input + lambda . d out / d input.  The state part
// becomes the adjoint for the previous step, the layer part is summed per layer, and the adjoint
// at the first step's input is d chi2 / d p0.  Cost ~ L x ceil(34 / KD) dual steps per track.
//
// k_fit_grad (forward mode): all 6 + 7 L parameters of a track are seeded KD at a time over a
// whole fit, ceil((6 + 7 L) / KD) fits per track (about 4x the work of the reverse sweep at 22
// layers) but no checkpoint memory.
//
// Per-layer derivatives are summed in shared memory per block, then added to the global arrays.
#include "internal.h"

namespace mk {

namespace {

constexpr int kThreads = 64;
constexpr int KD = 2;   // derivative directions per pass (at 4 the dual state spilled 1.4 KB of stack per thread)
using D = Dual<float, KD>;

__device__ __forceinline__ void load_geom(const DevGeom* __restrict__ gp, DevGeom& g) {
    const int4* src = reinterpret_cast<const int4*>(gp);
    int4* dst = reinterpret_cast<int4*>(&g);
    for (int i = threadIdx.x; i < (int)(sizeof(DevGeom) / 16); i += blockDim.x) dst[i] = src[i];
}

__device__ __forceinline__ D seeded(float v, int comp, int base) {
    D r(v);
    const int k = comp - base;
    if (k >= 0 && k < KD) r.d[k] = 1.0f;
    return r;
}

// A module hit's chi2 and update on its module's plane (Sec. 3.1) with the alignment
// displacement dm in the residual; 0 ok, 1 plane not reached, 3 update failed.  Not inlined: the
// dual-number kernels keep their registers for the layers without modules.
template <class T>
__device__ __noinline__ int grad_module_update(int kind, const PredT<T>& q, const float4* __restrict__ mods, int mod,
                                               float cB, T mx, T my, T mz, const T v[6], const T dm[3], StateT<T>& t,
                                               T& x2) {
    PredT<T> qp;
    FrameT<T> fp;
    if (!to_module_plane(kind, q, mods, mod, cB, qp, fp)) return 1;
    if (!chi2_hit(fp, qp, mx, my, mz, v, x2, dm) || !kalman_update_f(fp, qp, mx, my, mz, v, t, nullptr, dm))
        return 3;
    return 0;
}

// One step of the fit in scalar T: propagate to layer l (its thickness scaled by xs), then, with
// hit h >= 0, chi2 and update with the hit displaced by the alignment al (the displacement
// d + w x (h - c) enters the residual, not the FP32 hit position, whose ulp at 1 m is 0.08 um);
// h < 0 propagates only.  Returns 0 (ok; x2 = the step's chi2) or the fit's status code.
template <class T, bool MOD>
__device__ __forceinline__ int fit_step(const DevGeom& g, const DevParams& P, const float4* __restrict__ pay,
                                        int64_t n_hits, int l, int h, StateT<T>& t, const T al[6], const T& xs,
                                        T& x2) {
    const DevLayer& L = g.layers[l];
    PredT<T> q;
    int newton = 0;
    const int r = propagate_core<T, T>(L, g.cB, P.material, t, t.c, q, q.c, newton, nullptr, &xs);
    if (r != 1) return r == 0 ? 1 : 2;
    if (h >= n_hits) return 4;
    x2 = T(0.0f);
    if (h < 0) {
        pred_to_state(L.kind, q, t);
        return 0;
    }
    float mf[3], vf[6];
    int md = -1;
    if constexpr (MOD)
        load_hit(pay, h, mf, vf, nullptr, &md);
    else
        load_hit(pay, h, mf, vf, nullptr);
    const float cz = L.kind == MKGB_DISK ? L.pos : 0.0f;
    const T r0(mf[0]), r1(mf[1]), r2(mf[2] - cz);
    const T dm[3] = {al[0] + (al[4] * r2 - al[5] * r1), al[1] + (al[5] * r0 - al[3] * r2),
                     al[2] + (al[3] * r1 - al[4] * r0)};
    const T mx(mf[0]), my(mf[1]), mz(mf[2]);
    T v[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) v[c] = T(vf[c]);
    if (MOD && md >= 0) {   // a module hit, on its module's plane (not reached: status 1, as the fit)
        const int rm = grad_module_update(L.kind, q, g.mods, md, g.cB, mx, my, mz, v, dm, t, x2);
        if (rm == 1) pred_to_state(L.kind, q, t);
        return rm;
    }
    if (!chi2_hit(L.kind, q, mx, my, mz, v, x2, dm) || !kalman_update(L.kind, q, mx, my, mz, v, t, nullptr, dm))
        return 3;
    return 0;
}

template <bool MOD>
__global__ void __launch_bounds__(kThreads) k_fit_grad(const DevGeom* __restrict__ gp, DevParams P,
                                                       const float4* __restrict__ pay, int64_t n_hits, int n,
                                                       int max_steps, const int* __restrict__ layers,
                                                       const int* __restrict__ hits, const float* __restrict__ p0,
                                                       const float* __restrict__ c0, const float* __restrict__ align,
                                                       const float* __restrict__ xscale, float* __restrict__ chi2_out,
                                                       float* __restrict__ d_p0, float* __restrict__ d_align,
                                                       float* __restrict__ d_xscale, int* __restrict__ status_out) {
    __shared__ DevGeom g;
    __shared__ float acc[MKGB_MAX_LAYERS * 7];
    load_geom(gp, g);
    for (int q = threadIdx.x; q < MKGB_MAX_LAYERS * 7; q += blockDim.x) acc[q] = 0.0f;
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const int* lrow = layers + (int64_t)i * max_steps;
        const int* hrow = hits + (int64_t)i * max_steps;
        int nl = 0;
        while (nl < max_steps && lrow[nl] >= 0 && lrow[nl] < g.n_layers) ++nl;
        const int ncomp = 6 + 7 * nl;
        const float* pi = p0 + 6 * (int64_t)i;
        const float* ci = c0 + 21 * (int64_t)i;
        int status = 0;
        float chi2v = 0.0f;
        for (int base = 0; base < ncomp && status == 0; base += KD) {
            StateT<D> t;
            t.xh = seeded(pi[0], 0, base); t.yh = seeded(pi[1], 1, base); t.zh = seeded(pi[2], 2, base);
            t.xl = D(0.0f); t.yl = D(0.0f); t.zl = D(0.0f);
            t.k = seeded(pi[3], 3, base); t.phi = seeded(pi[4], 4, base); t.th = seeded(pi[5], 5, base);
#pragma unroll 1
            for (int q = 0; q < 21; ++q) t.c[q] = D(ci[q]);
            D sum(0.0f);
            for (int j = 0; j < nl; ++j) {
                const int l = lrow[j];
                const int cj = 6 + 7 * j;
                const float* al = align + 6 * l;
                D ald[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) ald[c] = seeded(al[c], cj + c, base);
                const D xs = seeded(xscale[l], cj + 6, base);
                D x2;
                status = fit_step<D, MOD>(g, P, pay, n_hits, l, hrow[j], t, ald, xs, x2);
                if (status != 0) break;
                sum += x2;
            }
            if (status != 0) break;
            if (base == 0) chi2v = sum.v;
#pragma unroll
            for (int k = 0; k < KD; ++k) {
                const int comp = base + k;
                if (comp >= ncomp) break;
                if (comp < 6) {
                    d_p0[6 * (int64_t)i + comp] = sum.d[k];
                } else {
                    const int j = (comp - 6) / 7, qq = (comp - 6) % 7;
                    atomicAdd(acc + lrow[j] * 7 + qq, sum.d[k]);
                }
            }
        }
        if (status != 0) {
            chi2v = 0.0f;
#pragma unroll
            for (int c = 0; c < 6; ++c) d_p0[6 * (int64_t)i + c] = 0.0f;
        }
        chi2_out[i] = chi2v;
        if (status_out) status_out[i] = status;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < g.n_layers * 7; q += blockDim.x) {
        const float v = acc[q];
        if (v != 0.0f) {
            const int l = q / 7, c = q % 7;
            atomicAdd(c < 6 ? d_align + 6 * l + c : d_xscale + l, v);
        }
    }
}

// Checkpoint of a step's input state: 32 floats (hi positions, lo positions, k, phi, theta, 21
// covariance words, theta's and phi's low parts), record j of track i at ((j * n + i) * 32).
__device__ __forceinline__ void store_ck(float* __restrict__ p, const State& t) {
    float4* v = reinterpret_cast<float4*>(p);
    v[0] = make_float4(t.xh, t.yh, t.zh, t.xl);
    v[1] = make_float4(t.yl, t.zl, t.k, t.phi);
    v[2] = make_float4(t.th, t.c[0], t.c[1], t.c[2]);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[3 + q] = make_float4(t.c[3 + 4 * q], t.c[4 + 4 * q], t.c[5 + 4 * q], t.c[6 + 4 * q]);
    v[7] = make_float4(t.c[19], t.c[20], t.tl, t.pl);
}

__device__ __forceinline__ void load_ck(const float* __restrict__ p, State& t) {
    const float4* v = reinterpret_cast<const float4*>(p);
    float4 a = v[0];
    t.xh = a.x; t.yh = a.y; t.zh = a.z; t.xl = a.w;
    a = v[1];
    t.yl = a.x; t.zl = a.y; t.k = a.z; t.phi = a.w;
    a = v[2];
    t.th = a.x; t.c[0] = a.y; t.c[1] = a.z; t.c[2] = a.w;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        a = v[3 + q];
        t.c[3 + 4 * q] = a.x; t.c[4 + 4 * q] = a.y; t.c[5 + 4 * q] = a.z; t.c[6 + 4 * q] = a.w;
    }
    a = v[7];
    t.c[19] = a.x; t.c[20] = a.y; t.tl = a.z; t.pl = a.w;
}

// Inputs of one step, in the adjoint's order: x, y, z, k, phi, theta, the 21 covariance words,
// the layer's 6 alignment parameters, its thickness scale.
constexpr int kStateIn = 27, kStepIn = 34;

// Keys of the reverse sweep's order: steps of the track (the longest first) and how many of them
// cross disks.
constexpr int kAdjKeyLen = 64, kAdjKeyDisks = 32, kAdjKeys = kAdjKeyLen * kAdjKeyDisks;

__global__ void __launch_bounds__(256) k_adj_order(int n, const int4* __restrict__ trk,
                                                   const int* __restrict__ key_off, int* __restrict__ order) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int4 t = trk[i];
    order[key_off[t.z] + t.w] = i;
}

// The sweep's bound is the fetch of its own code: a dual step is ~12,000 straight-line
// instructions (200 KB, more than the instruction cache), and 255 registers leave room for eight
// warps.  With one thread per track and all passes each warp walked through that code on its own
// (no_instruction 2.1-4.9 of the stall cycles per issue, issue active 21%).  So the eight warps of
// a block share the passes of a step (17 at KD = 2), start each round of them together and share
// the fetches; a small batch spreads over eight times as many warps.  The tracks are taken in the
// order of their length and layer kinds, so that the lanes of a warp walk the same steps (31 of 32
// active instead of 21, and no round for the few long tracks of a block), longest first.
// 1 to kAdjWide groups of 32 tracks per block: four make 68 passes for 8 warps (9 rounds, 94%
// busy), one 3 rounds (71%); the launch takes the number with the fewest rounds over all blocks.
// 100k tracks, 12 layers each, of the misaligned endcap: 23.4 ms with one thread per track; passes
// shared by the warps 14.5, rounds started together 12.3, in order 9.5, the directions seeded by index
// 8.9 ms (one direction per pass, KD = 1 with 12 warps of 168 registers, 12.1); 1,001 tracks: 5.71 ->
// 0.74 ms.
//
// plain: the pass that writes the checkpoints, one thread per track, the input of every step stored;
// trk and the keys' counts for the order are its results too.  It is a launch of the same kernel, not
// a kernel of its own, because the compiler rounds the step's FP32 operations differently there (0.3%
// of the tracks' first steps in the last bit), which d/dp0 of ill-conditioned tracks turns into up to
// 1.2e-3 of its norm over a batch; in one function with the dual step its values have been the same
// through every rearrangement of the sweep.  (255 registers instead of 119 cost it 0.1 ms of 100k
// tracks' 8.9.)
constexpr int kAdjWarps = 8, kAdjThreads = 32 * kAdjWarps;
constexpr int kAdjPasses = (kStepIn + KD - 1) / KD;
constexpr int kAdjWide = 4;   // groups of 32 tracks per block where the batch fills the device

template <bool MOD>
__global__ void __launch_bounds__(kAdjThreads, 1) k_fit_adjoint(
    const DevGeom* __restrict__ gp, DevParams P, const float4* __restrict__ pay, int64_t n_hits, int n,
    int max_steps, const int* __restrict__ layers, const int* __restrict__ hits, const float* __restrict__ align,
    const float* __restrict__ xscale, float* __restrict__ chi2_out, float* __restrict__ d_p0,
    float* __restrict__ d_align, float* __restrict__ d_xscale, int* __restrict__ status_out, int4* trk,
    const int* __restrict__ order, float* ck, int groups, bool plain, const float* __restrict__ p0,
    const float* __restrict__ c0, int* key_counts) {
    __shared__ DevGeom g;
    __shared__ float acc[MKGB_MAX_LAYERS * 7];
    __shared__ int s_nl[32 * kAdjWide];   // steps to redo; 0 once a redone step has failed
    __shared__ int s_status[32 * kAdjWide];
    __shared__ int s_id[32 * kAdjWide];
    __shared__ int s_max;
    // d total / d (state after the step), of the step at hand and of the one before it:
    // [2][kStateIn][tracks]
    extern __shared__ float s_lam[];
    const int tracks = 32 * groups;
    load_geom(gp, g);
    for (int q = threadIdx.x; q < MKGB_MAX_LAYERS * 7; q += blockDim.x) acc[q] = 0.0f;
    if (plain) {
        __syncthreads();
        const int i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i < n) {
            const int* lrow = layers + (int64_t)i * max_steps;
            const int* hrow = hits + (int64_t)i * max_steps;
            int nl = 0;
            while (nl < max_steps && lrow[nl] >= 0 && lrow[nl] < g.n_layers) ++nl;
            State t;
            {
                const float* pi = p0 + 6 * (int64_t)i;
                const float* ci = c0 + 21 * (int64_t)i;
                t.xh = pi[0]; t.yh = pi[1]; t.zh = pi[2];
                t.xl = 0.0f; t.yl = 0.0f; t.zl = 0.0f;
                t.k = pi[3]; t.phi = pi[4]; t.th = pi[5];
#pragma unroll
                for (int q = 0; q < 21; ++q) t.c[q] = ci[q];
            }
            int status = 0, disks = 0;
            float chi2v = 0.0f;
            for (int j = 0; j < nl && status == 0; ++j) {
                const int l = lrow[j];
                disks += g.layers[l].kind == MKGB_DISK;
                store_ck(ck + ((int64_t)j * n + i) * 32, t);
                float x2 = 0.0f;
                status = fit_step<float, MOD>(g, P, pay, n_hits, l, hrow[j], t, align + 6 * l, xscale[l], x2);
                chi2v += x2;
            }
            chi2_out[i] = chi2v;
            const int len = status == 0 ? nl : 0;
            const int key = (kAdjKeyLen - 1 - min(len, kAdjKeyLen - 1)) * kAdjKeyDisks + min(disks, kAdjKeyDisks - 1);
            trk[i] = make_int4(nl, status, key, atomicAdd(key_counts + key, 1));
        }
        return;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t i0 = (int64_t)blockIdx.x * tracks; i0 < n; i0 += (int64_t)gridDim.x * tracks) {
        __syncthreads();   // the geometry and acc are set; the last tracks' adjoints are written out
        if (threadIdx.x == 0) s_max = 0;
        __syncthreads();
        for (int u = threadIdx.x; u < tracks; u += kAdjThreads) {
            const int id = i0 + u < n ? order[i0 + u] : 0;
            const int4 tr = i0 + u < n ? trk[id] : make_int4(0, 0, 0, 0);
            s_id[u] = id;
            s_status[u] = tr.y;
            s_nl[u] = tr.y == 0 ? tr.x : 0;
            atomicMax(&s_max, s_nl[u]);
        }
        for (int q = threadIdx.x; q < kStateIn * tracks; q += kAdjThreads) s_lam[q] = 0.0f;
        __syncthreads();
        int cur = 0;
        for (int j = s_max - 1; j >= 0; --j, cur ^= 1) {
            const float* lam = s_lam + cur * kStateIn * tracks;
            float* next = s_lam + (cur ^ 1) * kStateIn * tracks;
#pragma unroll 1
            for (int w0 = 0; w0 < groups * kAdjPasses; w0 += kAdjWarps) {
                __syncthreads();   // the warps start a pass together
                const int w = w0 + wid;
                if (w >= groups * kAdjPasses) continue;
                const int ps = w % kAdjPasses, u = (w / kAdjPasses) * 32 + lane;
                const int64_t i = s_id[u];
                const bool on = j < s_nl[u];
                const int l = on ? layers[i * max_steps + j] : 0, h = on ? hits[i * max_steps + j] : -1;
                const int base = ps * KD;
                float out[KD];
#pragma unroll
                for (int k = 0; k < KD; ++k) out[k] = 0.0f;
                // without a hit the alignment has no effect: skip passes that seed only it
                const bool idle = h < 0 && base >= kStateIn + 1 && base + KD <= kStepIn - 1;
                if (on && !idle) {
                    State t0;
                    load_ck(ck + ((int64_t)j * n + i) * 32, t0);
                    const float* al = align + 6 * l;
                    StateT<D> td;
                    td.xh = seeded(t0.xh, 0, base);
                    td.yh = seeded(t0.yh, 1, base);
                    td.zh = seeded(t0.zh, 2, base);
                    td.xl = D(t0.xl); td.yl = D(t0.yl); td.zl = D(t0.zl);
                    td.k = seeded(t0.k, 3, base);
                    td.phi = seeded(t0.phi, 4, base);
                    td.th = seeded(t0.th, 5, base);
                    td.tl = D(t0.tl);
                    td.pl = D(t0.pl);
#pragma unroll
                    for (int q = 0; q < 21; ++q) td.c[q] = seeded(t0.c[q], 6 + q, base);
                    D ald[6];
#pragma unroll
                    for (int c = 0; c < 6; ++c) ald[c] = seeded(al[c], kStateIn + c, base);
                    const D xs = seeded(xscale[l], kStepIn - 1, base);
                    D x2;
                    if (fit_step<D, MOD>(g, P, pay, n_hits, l, h, td, ald, xs, x2) != 0) {
                        s_status[u] = 5;   // the redone step failed where the plain pass did not
                    } else {
#pragma unroll
                        for (int k = 0; k < KD; ++k) {
                            float a = x2.d[k];
                            a = fmaf(lam[u], td.xh.d[k] + td.xl.d[k], a);
                            a = fmaf(lam[tracks + u], td.yh.d[k] + td.yl.d[k], a);
                            a = fmaf(lam[2 * tracks + u], td.zh.d[k] + td.zl.d[k], a);
                            a = fmaf(lam[3 * tracks + u], td.k.d[k], a);
                            a = fmaf(lam[4 * tracks + u], td.phi.d[k] + td.pl.d[k], a);
                            a = fmaf(lam[5 * tracks + u], td.th.d[k] + td.tl.d[k], a);
#pragma unroll
                            for (int q = 0; q < 21; ++q) a = fmaf(lam[(6 + q) * tracks + u], td.c[q].d[k], a);
                            out[k] = a;
                        }
                    }
                }
#pragma unroll
                for (int k = 0; k < KD; ++k) {
                    const int comp = base + k;
                    if (comp < kStateIn)
                        next[comp * tracks + u] = out[k];
                    else if (comp < kStepIn && out[k] != 0.0f)
                        atomicAdd(acc + l * 7 + (comp - kStateIn), out[k]);
                }
            }
            __syncthreads();   // the step's adjoints are complete
            for (int u = threadIdx.x; u < tracks; u += kAdjThreads)
                if (s_status[u] != 0) s_nl[u] = 0;
            __syncthreads();
        }
        for (int u = threadIdx.x; u < tracks && i0 + u < n; u += kAdjThreads) {
            const int status = s_status[u];
            const int64_t i = s_id[u];
#pragma unroll
            for (int c = 0; c < 6; ++c) d_p0[6 * i + c] = status == 0 ? s_lam[(cur * kStateIn + c) * tracks + u] : 0.0f;
            if (status != 0) chi2_out[i] = 0.0f;
            if (status_out) status_out[i] = status;
        }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < g.n_layers * 7; q += blockDim.x) {
        const float v = acc[q];
        if (v != 0.0f) {
            const int l = q / 7, c = q % 7;
            atomicAdd(c < 6 ? d_align + 6 * l + c : d_xscale + l, v);
        }
    }
}

}  // namespace

size_t fit_grad_scratch_bytes(int n, int max_steps) {
    return (size_t)n * (128 * (size_t)(max_steps > 0 ? max_steps : 1) + 16 + 4) + 4 * (kAdjKeys + 4);
}

cudaError_t launch_fit_grad(cudaStream_t st, const DevGeom* g, DevParams P, const float4* pay, int64_t n_hits, int n,
                            int max_steps, const int* layers, const int* hits, const float* p0, const float* c0,
                            const float* align, const float* xscale, float* chi2_out, float* d_p0, float* d_align,
                            float* d_xscale, int* status_out, float* ck, int n_sms, bool modular) {
    if (n == 0) return cudaSuccess;
    const int blocks = (n + kThreads - 1) / kThreads;
    if (ck) {
        auto adjoint = modular ? k_fit_adjoint<true> : k_fit_adjoint<false>;
        // after the checkpoints: per track (steps, status, key, rank), the keys' counts, the order
        int4* trk = reinterpret_cast<int4*>(ck + (size_t)32 * n * (max_steps > 0 ? max_steps : 1));
        int* key_counts = reinterpret_cast<int*>(trk + n);
        int* order = key_counts + kAdjKeys + 4;
        cudaError_t e = cudaMemsetAsync(key_counts, 0, 4 * kAdjKeys, st);
        if (e != cudaSuccess) return e;
        adjoint<<<blocks, kThreads, 0, st>>>(g, P, pay, n_hits, n, max_steps, layers, hits, align, xscale, chi2_out, d_p0,
                                             d_align, d_xscale, status_out, trk, nullptr, ck, 1, true, p0, c0,
                                             key_counts);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if ((e = exclusive_scan(st, key_counts, key_counts, kAdjKeys, nullptr)) != cudaSuccess) return e;   // one block
        k_adj_order<<<(n + 255) / 256, 256, 0, st>>>(n, trk, key_counts, order);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        // groups per block: the fewest rounds of passes over all blocks of an SM
        int groups = 1, need = 0, best = 0;
        for (int gr = 1; gr <= kAdjWide; ++gr) {
            const int nb = (n + 32 * gr - 1) / (32 * gr);
            const int rounds = (nb + n_sms - 1) / n_sms * ((gr * kAdjPasses + kAdjWarps - 1) / kAdjWarps);
            if (gr == 1 || rounds < best) {
                best = rounds;
                groups = gr;
                need = nb;
            }
        }
        adjoint<<<need < n_sms ? need : n_sms, kAdjThreads, 2 * kStateIn * 32 * groups * sizeof(float), st>>>(
            g, P, pay, n_hits, n, max_steps, layers, hits, align, xscale, chi2_out, d_p0, d_align, d_xscale,
            status_out, trk, order, ck, groups, false, nullptr, nullptr, nullptr);
        return cudaGetLastError();
    }
    auto forward = modular ? k_fit_grad<true> : k_fit_grad<false>;
    forward<<<blocks, kThreads, 0, st>>>(g, P, pay, n_hits, n, max_steps, layers, hits, p0, c0, align, xscale,
                                         chi2_out, d_p0, d_align, d_xscale, status_out);
    return cudaGetLastError();
}

}  // namespace mk
