// Discrete adjoint over dense rows: the same map and formulas as
// psst_adjoint.cu, for networks of up to 128 neurons with per-pair gates.
//
// One cluster of two CTAs per network.  Rank 0 recomputes segment c - 1
// forward from its checkpoint with the dense kernel's stage (psst_dense.cuh:
// the forward kernel's own operations, so the recomputed trajectory is the
// forward's) and stores for every stage what the sweep needs, every
// exponential and division already done: per neuron (V, m, h, n), the closing
// slopes and the slopes' derivatives by V, the synaptic conductance and the
// slope of V; per pair a T + b, the slope of r's derivative by V, dG/ds and G.
// Rank 1 sweeps segment c backward from those records, copied into shared
// memory one step ahead.
//
// Sweep.  Pairs sit in slots sorted by type, each type padded to a multiple of
// 4; eight neighbouring threads share four slots, thread l holding the weights
// from these pairs to neurons 32 q + 4 l .. + 3 in registers, and beside each
// weight its gradient's partial sum.  The last two warps hold the neurons, two
// per thread, with their state in registers.  A stage is
//   1. neuron warps: the potential's adjoint of the stage after it (its base
//      and its pairs' terms), kb_V, q = kb_V / C, and z_t = q (V - E_t) for
//      every synapse type t into shared memory; pair warps, meanwhile: the
//      gradients' multiply-adds G_p z_i of the stage after it;
//   2. pair warps: C_p = sum_i w_ip z_i (one 16-byte load of z feeds 16
//      multiply-adds), the exchange among the eight threads, the pairs'
//      adjoints; neuron warps, meanwhile: the gates' adjoints and the
//      parameter gradients,
// with one barrier after each.  Every few steps the gradients' partial sums
// go to two-float totals (FOLD_STEPS).
//
// Bound: the chain of a sweep stage (two barriers, sums, exchange) on 64
// networks of 120 neurons, the recompute's stage on small ones.  It replaces,
// for these networks, four phases per stage with rate functions on the chain,
// gathers for the column sums and a pass over all weight gradients in global
// memory per step (psst_adjoint.cu, kept for larger networks, duplicated
// synapses and per-synapse gates).  Adjoint of 200 steps, us per step, before /
// now: 64 lobes of 120 neurons 20 / 7.6, one of 37 neurons 14 / 3.6; with the
// forward, 8565 -> 2730 us per pass and (300 steps) 6497 -> 2110.
#include <cuda_runtime.h>

#include <type_traits>

#include "psst_dense.cuh"
#include "psst_device.cuh"
#include "psst_internal.h"
#include "psst_syn.cuh"

namespace psst {

namespace {

// Steps whose weight-gradient terms run up in FP32 before they join the
// two-float totals: at most a quarter of a segment (one rounding per stage and
// at most four stages a step: no more than the one per step of a sum over the
// whole segment, as psst_adjoint.cu forms it).  Weight gradients of 8 lobes,
// 200 steps, from the float64 ones with 4 / 8 / 16 / 32 steps: 2.26 / 2.27 /
// 2.31 / 2.46e-7; 64 lobes, forward and adjoint: 2741 / 2654 / 2619 / 2607 us.
constexpr int FOLD_STEPS = 8;

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// (Without .aligned, for the same reason as bar_all below.)
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ void copy16(int o, const float4 *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dsm + o)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The CTA's barrier, met by the sweep's pair warps and neuron warps at
// different places of their code.  (barrier.sync, not bar.sync, which is the
// aligned form: lanes without a neuron or past a copy's end need not have
// reconverged with the others of their warp.)
__device__ __forceinline__ void bar_all() { asm volatile("barrier.sync 0;" ::: "memory"); }

// ---------------------------------------------------------------- recompute

template <int QR>
struct Recompute {
    const NetView &v;
    const AdjDenseView &av;
    const AdjDensePlan &pl;
    const AdjDenseLayout &lay;
    const float *stab;
    int b, n0, N, nt, C, np, Nw, TR, l8, row0, row, i0, u1, u2, ns;
    bool has_row, writes;
    long long sbase, step0;
    float4 w[QR][4];
    NeuronPrm P;

    __device__ void load_weights() {
        const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, nq = pl.nq;
        const long long *rp = v.row_ptr + n0;
        const uint32_t *gcode = v.syn_code + sbase;
        const float *gw = v.weight + sbase;
        const unsigned short *pcol = av.col + (long long)n0 * nt;
#pragma unroll
        for (int q = 0; q < QR; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) w[q][r] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int c = tid; c < 2 * C; c += nthr) F1(lay.g + 4 * c) = 0.0f;
        for (int q = tid; q < nq; q += nthr) {
            int t = 0;
            while (t + 1 < nt && q >= pl.tq[t + 1]) ++t;
            F1(lay.eq + 4 * q) = stab[t * ST_COLS + SP_E];
        }
        if (tid < ns) {
            const StageRT s = stage_rt(v, tid, v.dt);
            F4(lay.sc + 16 * tid) = make_float4(s.c.w, s.c.cn, s.c.fin, s.c.finl);
        }
        const int SR = pl.rows;  // a multiple of 4
        for (int r0 = 0; r0 < N; r0 += SR) {
            const int nr = min(SR, N - r0), nr4 = (nr + 3) & ~3;
            for (int q = tid; q < nr4 * (C >> 2); q += nthr) F4(lay.stage + 16 * q) = make_float4(0.f, 0.f, 0.f, 0.f);
            __syncthreads();
            for (int i = tid >> 5; i < nr; i += nthr >> 5)
                for (long long k = rp[r0 + i] - sbase + lane; k < rp[r0 + i + 1] - sbase; k += 32)
                    F1(lay.stage + 4 * (i * C + pcol[gcode[k] & 0xFFFFFFu])) = gw[k];
            __syncthreads();
            if (row0 >= r0 && row0 < r0 + nr) {
                const int src = lay.stage + 4 * (row0 - r0) * C + 16 * l8;
#pragma unroll
                for (int q = 0; q < QR; ++q)
#pragma unroll
                    for (int r = 0; r < 4; ++r) w[q][r] = F4(src + 4 * r * C + 128 * q);
                for (int q = QR; q < nq; ++q)
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        F4(lay.xw + 16 * ((4 * (q - QR) + r) * TR + tid)) = F4(src + 4 * r * C + 128 * q);
            }
            __syncthreads();
        }
        if (row0 >= N && tid < TR)
            for (int q = 0; q < 4 * (nq - QR); ++q) F4(lay.xw + 16 * (q * TR + tid)) = make_float4(0.f, 0.f, 0.f, 0.f);
        if (has_row) P = load_neuron_prm(v, n0 + row);
        for (int i = tid; i < Nw; i += nthr) {
            F1(lay.inp + 8 * i) = i < N ? v.i_const[n0 + i] : 0.0f;
            F1(lay.inp + 8 * i + 4) = i < N && v.pulse_amp ? v.pulse_amp[n0 + i] : 0.0f;
        }
        for (int p = tid; p < np; p += nthr) {
            const int4 pr = av.pair[pl.pair0 + p];
            const int j = pr.x / nt, t = pr.x - j * nt;
            *(int4 *)(dsm + lay.pinfo + 16 * p) = make_int4(4 * j, (t << 24) | (4 * pr.w), pr.z, 0);
        }
        __syncthreads();
    }

    // Segment c into buffer c mod 2.
    __device__ void segment(int c, int nsteps, float *seg, long long seg_buf) {
        const int tid = threadIdx.x, nthr = blockDim.x, nq = pl.nq;
        const int k0 = c * av.ckpt_every, k1 = min(k0 + av.ckpt_every, nsteps);
        const float *y = av.ck + (long long)c * av.dim, *yl = av.ck_lo + (long long)c * av.dim;
        const float *gV = y + n0, *gVl = yl + n0, *gr = y + 4 * v.N + sbase, *grl = yl + 4 * v.N + sbase;
        float V = 0.0f, y0 = 0.0f, ylo = 0.0f, acc = 0.0f;
        if (has_row) {
            y0 = V = gV[row];
            ylo = gVl[row];
        }
        for (int i = tid; i < Nw; i += nthr) {
            const bool own = i < N;
            F1(lay.vst + 4 * i) = F1(lay.vst + 4 * (Nw + i)) = own ? gV[i] : 0.0f;
            float g[3];
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                const long long at = (long long)(x + 1) * v.N + i;
                g[x] = own ? gV[at] : 0.0f;
                F4(lay.gst + 16 * (x * Nw + i)) = make_float4(g[x], own ? gVl[at] : 0.0f, 0.0f, g[x]);
            }
            F4(lay.ys + 16 * i) = make_float4(g[0], g[1], g[2], 0.0f);
        }
        for (int p = tid; p < np; p += nthr) {
            const int rep = av.pair[pl.pair0 + p].y;
            const int4 info = *(const int4 *)(dsm + lay.pinfo + 16 * p);
            const float r = gr[rep], rl = grl[rep];
            F4(lay.pst + 16 * p) = make_float4(r, rl, 0.0f, 0.0f);
            *(float2 *)(dsm + lay.pacc + 8 * p) = make_float2(0.0f, 0.0f);
            float g = __fadd_rn(r, rl);
            if (p >= pl.np1) {
                const float s = gr[v.S + rep], sl = grl[v.S + rep];
                F4(lay.pst2 + 32 * (p - pl.np1)) = make_float4(s, sl, 0.0f, 0.0f);
                F4(lay.pst2 + 32 * (p - pl.np1) + 16) = make_float4(0.f, 0.f, 0.f, 0.f);
                g = second_gate(__fadd_rn(s, sl), stab[(info.y >> 24) * ST_COLS + SP_KD]);
            }
            F1(lay.g + (info.y & 0xFFFFFF)) = bounded(g);
        }
        __syncthreads();
        const int SF = adj_stage_floats(N, pl.Mp);
        float *rec = seg + (long long)(c & 1) * seg_buf;
        const long long pon = v.pulse_on[b], poff = v.pulse_off[b];
        int vc = lay.vst, vn = lay.vst + 4 * Nw, yc = lay.ys, yn = lay.ys + 16 * Nw, gc = lay.g, gn = lay.g + 4 * C;
        const float4 c0 = F4(lay.sc);
        StageCoef cf{c0.x, c0.y, c0.z, c0.w};
        float iext = 0.0f;
        auto stage = [&](auto last, int next) {
            constexpr bool LAST = decltype(last)::value;
#pragma unroll 1
            for (int p = u1; p < pl.np1; p += nthr) {
                float4 st = F4(lay.pst + 16 * p);
                const int4 info = *(const int4 *)(dsm + lay.pinfo + 16 * p);
                float2 a = *(const float2 *)(dsm + lay.pacc + 8 * p);
                const float *sp = stab + (info.y >> 24) * ST_COLS;
                const float T = transmitter(F1(vc + info.x), sp), a_ = __fmul_rn(sp[SP_A], T);
                const float bb = __fadd_rn(a_, sp[SP_B]), r = F1(gc + (info.y & 0xFFFFFF));  // G = r
                *(float4 *)(rec + 12 * N + 4 * info.z) =
                    make_float4(bb, a_ * (1.0f - T) * (sp[SP_KP] * 0.693147181f) * (1.0f - r), 0.0f, r);
                F1(gn + (info.y & 0xFFFFFF)) = bounded(pair_unit<LAST>(cf, a_, bb, st, a));
                F4(lay.pst + 16 * p) = st;
                *(float2 *)(dsm + lay.pacc + 8 * p) = a;
            }
#pragma unroll 1
            for (int p2 = u2; p2 < pl.np2; p2 += nthr) {
                const int p = pl.np1 + p2;
                float4 st = F4(lay.pst + 16 * p), q = F4(lay.pst2 + 32 * p2), z = F4(lay.pst2 + 32 * p2 + 16);
                const int4 info = *(const int4 *)(dsm + lay.pinfo + 16 * p);
                float2 a = *(const float2 *)(dsm + lay.pacc + 8 * p);
                const float *sp = stab + (info.y >> 24) * ST_COLS;
                const float T = transmitter(F1(vc + info.x), sp), a_ = __fmul_rn(sp[SP_A], T);
                const float bb = __fadd_rn(a_, sp[SP_B]);
                // this stage's r and s from their maps
                const float r = __fadd_rn(st.x, __fadd_rn(fmaf(st.w, st.x, st.z), st.y));
                const float s = __fadd_rn(q.x, __fadd_rn(fmaf(z.x, q.x, fmaf(q.w, st.x, q.z)), q.y));
                const float s2 = s * s, den = fmaf(s2, s2, sp[SP_KD]);
                *(float4 *)(rec + 12 * N + 4 * info.z) =
                    make_float4(bb, a_ * (1.0f - T) * (sp[SP_KP] * 0.693147181f) * (1.0f - r),
                                __fdiv_rn(4.0f * s2 * s * sp[SP_KD], den * den), F1(gc + (info.y & 0xFFFFFF)));
                const float r0 = st.x, sP = st.z, sQ = st.w;
                pair_unit<LAST>(cf, a_, bb, st, a);
                F1(gn + (info.y & 0xFFFFFF)) = bounded(pair_unit2<LAST>(cf, sp, r0, sP, sQ, q, z));
                F4(lay.pst + 16 * p) = st;
                *(float2 *)(dsm + lay.pacc + 8 * p) = a;
                F4(lay.pst2 + 32 * p2) = q;
                F4(lay.pst2 + 32 * p2 + 16) = z;
            }
#pragma unroll 1
            for (int i = i0; i < Nw; i += nthr) {
                const float Vi = F1(vc + 4 * i), e = rate_e(Vi);
                const int o = lay.gst + 16 * i;
                float4 m = F4(o), h = F4(o + 16 * Nw), n = F4(o + 32 * Nw);
                const float am = alpha_m(Vi, e), bm = beta_m(Vi), ah = alpha_h(Vi), bh = beta_h(e), an = alpha_n(Vi, e),
                            bn = beta_n(Vi);
                if (i < N) {
                    *(float4 *)(rec + 4 * i) = make_float4(Vi, m.w, h.w, n.w);
                    float *ls = rec + 4 * N + 4 * i, *gd = rec + 8 * N + 4 * i;
                    ls[0] = am + bm;
                    ls[1] = ah + bh;
                    ls[2] = an + bn;
                    gd[0] = slope_m(Vi, e, am, bm, m.w);
                    gd[1] = slope_h(ah, bh, h.w);
                    gd[2] = slope_n(Vi, e, an, bn, n.w);
                }
                gate_update<LAST>(cf, am, bm, m);
                gate_update<LAST>(cf, ah, bh, h);
                gate_update<LAST>(cf, an, bn, n);
                F4(o) = m;
                F4(o + 16 * Nw) = h;
                F4(o + 32 * Nw) = n;
                F4(yn + 16 * i) = make_float4(m.w, h.w, n.w, 0.0f);
            }
            if (tid < TR) {
                const float4 V4 = F4(vc + 4 * row0);
                const int g0 = gc + 16 * l8;
                float I[4] = {}, A[4] = {};
#pragma unroll
                for (int q = 0; q < QR; ++q) quad(w[q], F4(g0 + 128 * q), F1(lay.eq + 4 * q), V4, I, A);
#pragma unroll 1
                for (int q = QR; q < nq; ++q) {
                    const int x = lay.xw + 16 * (4 * (q - QR) * TR + tid);
                    const float4 wq[4] = {F4(x), F4(x + 16 * TR), F4(x + 32 * TR), F4(x + 48 * TR)};
                    quad(wq, F4(g0 + 128 * q), F1(lay.eq + 4 * q), V4, I, A);
                }
                const float isyn = row_sum(I, l8), As = row_sum(A, l8);
                const float4 yy = F4(yc + 16 * row);
                const float d = __fmul_rn(__fsub_rn(ionic_rest(P, V, yy.x, yy.y, yy.z, iext), isyn), P.invC);
                const float ac = fmaf(cf.w, d, acc);
                if (!LAST) {
                    acc = ac;
                    V = ext_stage(y0, ylo, cf.cn, d);
                } else {
                    ext_step(y0, ylo, cf.fin, cf.finl, ac);
                    acc = 0.0f;
                    V = y0;
                }
                if (writes) {
                    F1(vn + 4 * row) = V;
                    rec[4 * N + 4 * row + 3] = As;
                    rec[8 * N + 4 * row + 3] = d;
                }
            }
            const float4 c4 = F4(lay.sc + 16 * next);
            cf = StageCoef{c4.x, c4.y, c4.z, c4.w};
            __syncthreads();
            int t = vc;
            vc = vn;
            vn = t;
            t = yc;
            yc = yn;
            yn = t;
            t = gc;
            gc = gn;
            gn = t;
            rec += SF;
        };
        for (int n = k0; n < k1; ++n) {
            const long long step = step0 + n;
            if (has_row)
                iext = input_current(v, F1(lay.inp + 8 * row), F1(lay.inp + 8 * row + 4), step >= pon && step < poff,
                                     (long long)n0 + row, step);
#pragma unroll 1
            for (int s = 0; s < ns - 1; ++s) stage(std::false_type{}, s + 1);
            stage(std::true_type{}, 0);
        }
    }
};

// ---------------------------------------------------------------- sweep

template <int Q>
__device__ void sweep_run(const NetView &v, const AdjDenseView &av, const AdjDensePlan &pl, const AdjDenseLayout &lay,
                          const float *stab, const float2 *cc, int b, int n0, int N, long long sbase, long long step0,
                          int nsteps, int ns, const float *seg, long long seg_buf) {
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, nt = v.n_stypes, Mp = pl.Mp, TP = 2 * Mp;
    const long long *rp = v.row_ptr + n0;
    const uint32_t *gcode = v.syn_code + sbase;
    const float *gw = v.weight + sbase;
    const unsigned short *pslot = av.slot + (long long)n0 * nt;
    // own slots (threads below TP, whole warps)
    const int l8 = tid & 7, s0 = (tid >> 3) * 4, slot = s0 + 2 * (l8 & 1) + (l8 >> 1 & 1);
    int type = 0;
    while (type + 1 < nt && s0 >= pl.ts[type + 1]) ++type;
    const float *sp = stab + type * ST_COLS;
    float4 w[Q][4], ga[Q][4];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) w[q][r] = ga[q][r] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int a0 = 0; a0 < Mp; a0 += pl.slots) {
        const int na = min(pl.slots, Mp - a0);
        for (int q = tid; q < na * 8 * Q; q += nthr) F4(lay.buf + 16 * q) = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        for (int i = tid >> 5; i < N; i += nthr >> 5)
            for (long long k = rp[i] - sbase + lane; k < rp[i + 1] - sbase; k += 32) {
                const int a = (int)pslot[gcode[k] & 0xFFFFFFu] - a0;
                if (a >= 0 && a < na) F1(lay.buf + 4 * (a * 32 * Q + i)) = gw[k];
            }
        __syncthreads();
        if (s0 >= a0 && s0 < a0 + na)
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) w[q][r] = F4(lay.buf + 4 * ((s0 - a0 + r) * 32 * Q + 32 * q + 4 * l8));
        __syncthreads();
    }
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = tid; q < 2 * nt * 8 * Q; q += nthr) F4(lay.z + 16 * q) = zero4;
    for (int i = tid; i < N * nt; i += nthr) *(int *)(dsm + lay.pidx + 4 * i) = lay.uvc + 4 * Mp;
    for (int p = tid; p <= Mp; p += nthr) F1(lay.uvc + 4 * p) = 0.0f;
    __syncthreads();
    for (int p = tid; p < pl.np1 + pl.np2; p += nthr) {
        const int4 pr = av.pair[pl.pair0 + p];
        const int j = pr.x / nt, t = pr.x - j * nt;
        *(int *)(dsm + lay.pidx + 4 * (t * N + j)) = lay.uvc + 4 * pr.z;
    }
    // totals of the weight gradients: high and low parts, [Q][4][2][TP]
    float4 *gt = (float4 *)av.gtot + pl.grad_off;
    if (tid < TP)
        for (int k = 0; k < 8 * Q; ++k) gt[(long long)k * TP + tid] = zero4;
    __syncthreads();

    const int SF = adj_stage_floats(N, Mp), step_bytes = 4 * ns * SF, nvec = ns * SF / 4, zb = 128 * Q * nt;
    const int ckpt = av.ckpt_every, nseg = (nsteps + ckpt - 1) / ckpt;
    const int fold_steps = max(1, min(FOLD_STEPS, min(ckpt, nsteps) / 4));
    if (tid < TP) {
        // ---- pair warps: the sums over each slot's neurons, the pairs'
        // adjoints; the gradients' multiply-adds while the neuron warps
        // prepare the next stage (z is double-buffered by stage)
        float2 lam = make_float2(0.0f, 0.0f), yp = lam, ys = lam;  // own slot's (r, s) adjoints (threads l8 < 4)
        const int z0 = lay.z + 4 * (type * 32 * Q + 4 * l8);
        int since = 0, zc = 0;
        auto fold = [&]() {
#pragma unroll
            for (int q = 0; q < Q; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float4 *at = gt + (long long)(2 * (4 * q + r)) * TP + tid;
                    float4 hi = at[0], lo = at[TP];
                    ext_add(hi.x, lo.x, ga[q][r].x);
                    ext_add(hi.y, lo.y, ga[q][r].y);
                    ext_add(hi.z, lo.z, ga[q][r].z);
                    ext_add(hi.w, lo.w, ga[q][r].w);
                    at[0] = hi;
                    at[TP] = lo;
                    ga[q][r] = zero4;
                }
        };
        for (int c = nseg - 1; c >= 0; --c) {
            const int k0 = c * ckpt, k1 = min(k0 + ckpt, nsteps);
            const float4 *src = (const float4 *)(seg + (long long)(c & 1) * seg_buf);
            auto fetch = [&](int n) {
                for (int q = tid; q < nvec; q += TP)
                    copy16(lay.buf + (n & 1) * step_bytes + 16 * q, src + (long long)(n - k0) * nvec + q);
                copy_commit();
            };
            fetch(k1 - 1);
            copy_wait();
            bar_all();
            for (int n = k1 - 1; n >= k0; --n) {
                if (n > k0) fetch(n - 1);
#pragma unroll 1
                for (int st = ns - 1; st >= 0; --st) {
                    const int pb = lay.buf + (n & 1) * step_bytes + 4 * st * SF + 48 * N;
                    const float2 k = cc[st];  // h b_s, h a_{s+1}
                    const float kbr = fmaf(k.x, lam.x, k.y * yp.x), kbs = fmaf(k.x, lam.y, k.y * yp.y);
                    bar_all();
                    const int z1 = z0 + zc;
                    float Cs[4] = {};
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const float4 z = F4(z1 + 128 * q);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            Cs[r] = fmaf(w[q][r].x, z.x, Cs[r]);
                            Cs[r] = fmaf(w[q][r].y, z.y, Cs[r]);
                            Cs[r] = fmaf(w[q][r].z, z.z, Cs[r]);
                            Cs[r] = fmaf(w[q][r].w, z.w, Cs[r]);
                        }
                    }
                    const float4 pd = F4(pb + 16 * slot);  // a T + b, dr'/dV, dG/ds, G
                    const float Cp = row_sum(Cs, l8);
                    if (l8 < 4) F1(lay.uvc + 4 * slot) = kbr * pd.y;
                    float ur = -pd.x * kbr, us = 0.0f;
                    if (sp[SP_KIND] != 0.0f) {
                        ur = fmaf(sp[SP_K3], kbs, ur);
                        us = -Cp * pd.z - sp[SP_K4] * kbs;
                    } else {
                        ur -= Cp;
                    }
                    ys.x += ur;
                    ys.y += us;
                    yp = make_float2(ur, us);
                    if (st == 0) {
                        lam.x += ys.x;
                        lam.y += ys.y;
                        yp = ys = make_float2(0.0f, 0.0f);
                        copy_wait();
                    }
                    // (read before the barrier: the next step's copy into this
                    // buffer may start as soon as one warp has passed it)
                    float G[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) G[r] = F1(pb + 16 * (s0 + r) + 12);
                    bar_all();
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const float4 z = F4(z1 + 128 * q);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            ga[q][r].x = fmaf(G[r], z.x, ga[q][r].x);
                            ga[q][r].y = fmaf(G[r], z.y, ga[q][r].y);
                            ga[q][r].z = fmaf(G[r], z.z, ga[q][r].z);
                            ga[q][r].w = fmaf(G[r], z.w, ga[q][r].w);
                        }
                    }
                    zc = zb - zc;
                }
                if (++since == fold_steps) {
                    fold();
                    since = 0;
                }
            }
            bar_all();  // the last records are read before the next segment's arrive
            cluster_sync();
        }
        fold();
    } else {
        // ---- neuron warps: two neurons per thread, their state in registers
        struct Neuron {
            float4 lam, yp, ys;  // adjoints of (V, m, h, n), of the later stage's values (V: base), their sums
            NeuronPrm P;
            float2 g[9];         // parameter gradients, two-float
            float q, kb[3];
            int u[4];            // offsets of its pairs' terms
            float dl, dl_prev;
        };
        Neuron a[2];
        const int ln = tid - TP;
        bool own[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const int i = ln + 64 * x;
            own[x] = ln < 64 && i < N;
            Neuron &o = a[x];
            o.lam = o.yp = o.ys = zero4;
            o.P = load_neuron_prm(v, n0 + (own[x] ? i : 0));
#pragma unroll
            for (int y = 0; y < 9; ++y) o.g[y] = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int t = 0; t < 4; ++t)
                o.u[t] = own[x] && t < nt ? *(const int *)(dsm + lay.pidx + 4 * (t * N + i)) : lay.uvc + 4 * Mp;
            o.dl = o.dl_prev = o.q = 0.0f;
        }
        float E[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) E[t] = stab[min(t, nt - 1) * ST_COLS + SP_E];
        const int stride = v.rec_stride;
        int frame = av.n_frames - 1;
        if (stride > 0 && (step0 + nsteps) % stride == 0 && frame >= 0) {
#pragma unroll
            for (int x = 0; x < 2; ++x)
                if (own[x]) a[x].lam.x = av.dLdV[(long long)frame * v.N + n0 + ln + 64 * x];
            --frame;
        }
        // the potential's adjoint at the stage last swept: its base and its pairs' terms
        auto potential = [&](const Neuron &o) {
            const float u0 = F1(o.u[0]), u1 = F1(o.u[1]), u2 = F1(o.u[2]), u3 = F1(o.u[3]);
            return (((o.yp.x + u0) + u1) + u2) + u3;
        };
        // lam_n = lam + the stages' adjoints of the step just swept (+ the frame at its start)
        auto finish_step = [&](Neuron &o, float dl) {
            o.lam.x += o.ys.x + potential(o) + dl;
            o.lam.y += o.ys.y;
            o.lam.z += o.ys.z;
            o.lam.w += o.ys.w;
            o.ys = o.yp = zero4;
        };
        bool started = false;
        int zc = 0;
        for (int c = nseg - 1; c >= 0; --c) {
            const int k0 = c * ckpt, k1 = min(k0 + ckpt, nsteps);
            bar_all();
            for (int n = k1 - 1; n >= k0; --n) {
                const bool at_frame = stride > 0 && n > 0 && (step0 + n) % stride == 0 && frame >= 0;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    a[x].dl_prev = a[x].dl;
                    a[x].dl = at_frame && own[x] ? av.dLdV[(long long)frame * v.N + n0 + ln + 64 * x] : 0.0f;
                }
                if (at_frame) --frame;
#pragma unroll 1
                for (int st = ns - 1; st >= 0; --st) {
                    const int sb = lay.buf + (n & 1) * step_bytes + 4 * st * SF;
                    const float2 k = cc[st];
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if (!own[x]) continue;
                        Neuron &o = a[x];
                        const int i = ln + 64 * x;
                        if (st < ns - 1) {
                            o.yp.x = potential(o);
                            o.ys.x += o.yp.x;
                        } else if (started) {
                            finish_step(o, o.dl_prev);
                        }
                        o.q = fmaf(k.x, o.lam.x, k.y * o.yp.x) * o.P.invC;
                        const float V = F1(sb + 16 * i);
                        const int z = lay.z + zc + 4 * i;
#pragma unroll
                        for (int t = 0; t < 4; ++t)
                            if (t < nt) F1(z + 128 * Q * t) = bounded(o.q * (V - E[t]));
                    }
                    bar_all();
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        if (!own[x]) continue;
                        // the gates' adjoints, the base of the potential's, the parameter gradients
                        Neuron &o = a[x];
                        const int i = ln + 64 * x;
                        const float4 y = F4(sb + 16 * i), ls = F4(sb + 16 * (N + i)), gd = F4(sb + 16 * (2 * N + i));
                        const float q = o.q, V = y.x, m = y.y, h = y.z, nn = y.w;
                        const float kbm = fmaf(k.x, o.lam.y, k.y * o.yp.y), kbh = fmaf(k.x, o.lam.z, k.y * o.yp.z),
                                    kbn = fmaf(k.x, o.lam.w, k.y * o.yp.w);
                        const NeuronPrm &P = o.P;
                        const float dNa = V - P.ENa, dK = V - P.EK, dL = V - P.EL, dKL = V - P.EKL;
                        const float m2h = m * m * h, m3h = m2h * m, n3 = nn * nn * nn, n4 = n3 * nn;
                        const float um = -q * P.gNa * 3.0f * m2h * dNa - kbm * ls.x;
                        const float uh = -q * P.gNa * m * m * m * dNa - kbh * ls.y;
                        const float un = -q * P.gK * 4.0f * n3 * dK - kbn * ls.z;
                        float base = q * (-(P.gNa * m3h + P.gK * n4 + P.gL + P.gKL) - ls.w);
                        base = fmaf(kbm, gd.x, base);
                        base = fmaf(kbh, gd.y, base);
                        base = fmaf(kbn, gd.z, base);
                        o.yp = make_float4(base, um, uh, un);
                        o.ys.y += um;
                        o.ys.z += uh;
                        o.ys.w += un;
                        auto add = [&](int j, float term) { ext_add(o.g[j].x, o.g[j].y, term); };
                        add(NP_C, -q * gd.w);
                        add(NP_GNA, -q * m3h * dNa);
                        add(NP_GK, -q * n4 * dK);
                        add(NP_GL, -q * dL);
                        add(NP_GKL, -q * dKL);
                        add(NP_ENA, q * P.gNa * m3h);
                        add(NP_EK, q * P.gK * n4);
                        add(NP_EL, q * P.gL);
                        add(NP_EKL, q * P.gKL);
                    }
                    bar_all();
                    zc = zb - zc;
                }
                started = true;
            }
            bar_all();
            cluster_sync();
        }
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            if (!own[x]) continue;
            Neuron &o = a[x];
            const int i = ln + 64 * x;
            finish_step(o, o.dl);
#pragma unroll
            for (int y = 0; y < 9; ++y)
                av.gp_neuron[(long long)(n0 + i) * 9 + y] = (double)o.g[y].x + (double)o.g[y].y;
            av.grad_y0[n0 + i] = o.lam.x;
            av.grad_y0[v.N + n0 + i] = o.lam.y;
            av.grad_y0[2 * v.N + n0 + i] = o.lam.z;
            av.grad_y0[3 * v.N + n0 + i] = o.lam.w;
        }
    }
    __syncthreads();
    // weight gradients in CSR order
    for (int i = tid >> 5; i < N; i += nthr >> 5)
        for (long long k = rp[i] - sbase + lane; k < rp[i + 1] - sbase; k += 32) {
            const int s = pslot[gcode[k] & 0xFFFFFFu], t = (s >> 2) * 8 + ((i & 31) >> 2);
            const float *g = (const float *)(gt + (long long)(2 * (4 * (i >> 5) + (s & 3))) * TP + t) + (i & 3);
            av.grad_w[sbase + k] = -(g[0] + g[4 * TP]);
        }
}

template <int Q>
__global__ void __launch_bounds__(ADJ_DENSE_THREADS) adj_dense_kernel(NetView v, AdjDenseView av, long long step0,
                                                                      int nsteps) {
    __shared__ float stab[PSST_MAX_SYN_TYPES * ST_COLS];
    __shared__ float2 cc[4];
    load_syn_table(v.sparams, v.n_stypes, stab);
    const int tid = threadIdx.x, nthr = blockDim.x, ns = method_stages(v);
    if (tid < ns) {
        // h b_s and h a_{s+1} of the method
        const float dt = v.dt;
        float2 k = make_float2((tid == 1 || tid == 2) ? dt / 3.0f : dt / 6.0f, tid == 2 ? dt : 0.5f * dt);
        if (v.method == PSST_METHOD_EULER) k = make_float2(dt, 0.0f);
        if (v.method == PSST_METHOD_TABLEAU) k = make_float2(v.rk_beta * v.rk_w[tid] * dt, tid < 3 ? v.rk_c[tid] * dt : 0.0f);
        cc[tid] = k;
    }
    __syncthreads();
    const int b = blockIdx.x / 2;
    const AdjDensePlan &pl = av.plan[b];
    const int n0 = v.net_off[b], N = v.net_off[b + 1] - n0, nt = v.n_stypes;
    const long long sbase = v.row_ptr[n0];
    constexpr int QR = Q + 1;
    const AdjDenseLayout lay =
        make_adj_layout(N, nt, pl.Mp, pl.np1 + pl.np2, pl.np2, pl.nq, QR, Q, ns, pl.rows, pl.slots);
    float *seg = av.seg + pl.seg_off;
    const long long seg_buf = (long long)min(av.ckpt_every, nsteps) * ns * adj_stage_floats(N, pl.Mp);
    const int nseg = (nsteps + av.ckpt_every - 1) / av.ckpt_every;
    if (cluster_rank() == 0) {
        const int np = pl.np1 + pl.np2, Nw = (N + 31) & ~31, W1 = (pl.np1 + 31) & ~31, i0 = nthr - 1 - tid;
        const int l8 = tid & 7, row0 = (tid >> 3) * 4, row = row0 + 2 * (l8 & 1) + (l8 >> 1 & 1);
        Recompute<QR> rc{v, av, pl, lay, stab, b, n0, N, nt, 32 * pl.nq, np, Nw, dense_row_threads(N), l8, row0, row, i0,
                         ((i0 - Nw) % nthr + nthr) % nthr, ((i0 - Nw - W1) % nthr + nthr) % nthr, ns, row < N,
                         row < N && l8 < 4, sbase, step0, {}, {}};
        rc.load_weights();
        // one segment ahead of the sweep; the cluster barrier hands each buffer over
        for (int c = nseg - 1; c >= -1; --c) {
            if (c >= 0) rc.segment(c, nsteps, seg, seg_buf);
            cluster_sync();
        }
    } else {
        cluster_sync();
        sweep_run<Q>(v, av, pl, lay, stab, cc, b, n0, N, sbase, step0, nsteps, ns, seg, seg_buf);
    }
}

}  // namespace

cudaError_t adj_dense_launch(const NetView &v, const AdjDenseView &av, int Q, int threads, int smem, long long step0,
                             int nsteps, int n_types, float *grad_np, cudaStream_t stream) {
    void (*kern)(NetView, AdjDenseView, long long, int) = Q == 1   ? adj_dense_kernel<1>
                                                          : Q == 2 ? adj_dense_kernel<2>
                                                          : Q == 3 ? adj_dense_kernel<3>
                                                                   : adj_dense_kernel<4>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * v.n_nets);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kern, v, av, step0, nsteps);
    if (e != cudaSuccess) return e;
    return adj_reduce(v, av.gp_neuron, n_types, grad_np, stream);
}

}  // namespace psst
