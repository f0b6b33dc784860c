// Integration of small and medium networks with per-pair gates whose synapses
// are held as dense rows in registers (RK4, Euler or a tableau).
//
// One cluster of `cl` CTAs (1, 2 or 4) owns a network for all steps of a
// launch and each CTA a block of its rows.  Eight neighbouring threads share
// four rows (postsynaptic neurons): thread l of the eight holds the weights
// of all four rows in the columns 32 q + 4 l .. + 3 of every quad q, absent
// synapses as zeros.  Columns are the used (presynaptic neuron, type) pairs,
// sorted by synapse type, each type padded to a multiple of 32.  A stage's
// synaptic sums are then products of registers with the gate table: one
// conflict-free 16-byte load of four gates feeds 16 multiply-adds, with no
// index and no gather (one row per thread, with broadcast loads, was bound by
// the loads: 47 multiply-adds per cycle and SM; packed two-column multiply-
// adds run at the rate of two single ones here).  Each quad's sum a of a row
// adds a (V - E) to the row's current; the eight threads' currents are
// exchanged so that each ends with one row's (two threads per row, equal
// bits), which updates the row's potential from registers.  A thread's first
// QR quads live in registers, the rest in shared memory (`xw`); the order of
// the sums depends on neither, nor on the cluster size or block size, so
// results do not.
//
// Everything a stage reads was finished by the stage before: the gate of a
// pair at stage s + 1 is an affine map of its step-start gate whose
// coefficients need only the potentials of stage s (psst_cta.cu).  So the
// gate table is computed one stage ahead, beside the synaptic sums, and one
// barrier per stage suffices.  The gate table has three buffers: the CTAs of
// a cluster push their pairs' next gates to every CTA, arrive at the cluster
// barrier and only then go on to the gates and the sums; a CTA two stages
// ahead in pushing is impossible, so the buffer it writes is never one still
// read.
//
// Bound: instruction issue (60% of the slots with the 12 warps of a
// 180-neuron CTA, 5,180 warp instructions a stage, 3,270 of them on the FMA
// pipe; a quad of 16 multiply-adds is 26, 24 of them there and two loads);
// alone on its SM, the chain of one stage (rates, or sums, exchange and
// potential: about 500 cycles).  Measured against the work-item kernel
// (psst_cta.cu), us per RK4 step, work items / dense rows: antennal lobe 6.5 /
// 3.1; at 30% connectivity 300 neurons alone 7.9 / 4.3, 608 networks of 60
// neurons 5.4 / 3.9, of 120 12.0 / 8.2, of 150 14.9 / 14.0, 304 of 180 10.9 /
// 8.8, of 250 20.8 / 17.9, of 300 32.5 / 25.9.  Its cost does not fall with the
// connectivity, the work items' does: the planner chooses (choose_dense in
// psst_api.cu).
#include <cuda_runtime.h>

#include <type_traits>

#include "psst_dense.cuh"
#include "psst_device.cuh"
#include "psst_internal.h"
#include "psst_syn.cuh"

namespace psst {

namespace {

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// (Without .aligned: warps arrive from loops whose lanes leave at different
// times, and only this form is defined for lanes that have not reconverged.)
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// x into the float at offset o of every CTA of the cluster.
__device__ __forceinline__ void put(int o, int cl, float x) {
    if (cl == 1) {
        F1(o) = x;
        return;
    }
    const unsigned laddr = (unsigned)__cvta_generic_to_shared(dsm + o);
    for (int q = 0; q < cl; ++q) {
        unsigned raddr;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(laddr), "r"(q));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(raddr), "f"(x) : "memory");
    }
}

template <int QR>
__device__ __forceinline__ void dense_run(const NetView &v, const int b, const DensePlan &pl, long long step0,
                                          int nsteps, int cl, const float *stab) {
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const int rank = cl > 1 ? (int)cluster_rank() : 0;
    const int n0 = v.net_off[b], nt = v.n_stypes;
    const int nq = pl.nq, C = 32 * nq;
    const int r_lo = pl.split[rank], nown = pl.split[rank + 1] - r_lo;
    // own pairs: np1 of first order, then np2 of second order
    const int p_lo = v.pair_off[b] + pl.psplit[rank], np1 = pl.psec[rank] - pl.psplit[rank];
    const int np2 = pl.psplit[rank + 1] - pl.psec[rank], np = np1 + np2;
    const int Nw = (nown + 31) & ~31, TR = dense_row_threads(nown);  // TR: threads that hold rows (whole warps)
    const DenseLayout lay = make_dense_layout(nown, np1, np2, nq, QR, pl.stage_rows);

    const long long sbase = v.row_ptr[n0];
    const float *gw = v.weight + sbase;
    const uint32_t *gcode = v.syn_code + sbase;
    const unsigned short *pcol = v.pair_col + (long long)n0 * nt;
    const long long *rp = v.row_ptr + n0 + r_lo;
    float *gV = v.state + n0 + r_lo, *gVl = v.state_lo ? v.state_lo + n0 + r_lo : nullptr;
    float *gr = v.state + 4 * v.N + sbase;
    float *grl = v.state_lo ? v.state_lo + 4 * v.N + sbase : nullptr;

    // ---- own rows: weights in registers, state and parameters of one neuron
    const int l8 = tid & 7, row0 = (tid >> 3) * 4, row = row0 + 2 * (l8 & 1) + (l8 >> 1 & 1);
    const bool has_row = row < nown, writes = has_row && l8 < 4;
    float4 w[QR][4];
#pragma unroll
    for (int q = 0; q < QR; ++q)
#pragma unroll
        for (int r = 0; r < 4; ++r) w[q][r] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c = tid; c < 3 * C; c += nthr) F1(lay.g + 4 * c) = 0.0f;
    for (int q = tid; q < nq; q += nthr) {
        int t = 0;
        while (t + 1 < nt && q >= pl.tq[t + 1]) ++t;
        F1(lay.eq + 4 * q) = stab[t * ST_COLS + SP_E];
    }
    const int ns = method_stages(v);
    if (tid < ns) {
        const StageRT s = stage_rt(v, tid, v.dt);
        F4(lay.sc + 16 * tid) = make_float4(s.c.w, s.c.cn, s.c.fin, s.c.finl);
    }
    const int SR = pl.stage_rows;  // a multiple of 4
    for (int r0 = 0; r0 < nown; r0 += SR) {
        const int nr = min(SR, nown - r0), nr4 = (nr + 3) & ~3;
        for (int q = tid; q < nr4 * (C >> 2); q += nthr) F4(lay.stage + 16 * q) = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        for (int i = tid >> 5; i < nr; i += nthr >> 5) {
            const long long k0 = rp[r0 + i] - sbase, k1 = rp[r0 + i + 1] - sbase;
            for (long long k = k0 + lane; k < k1; k += 32)
                F1(lay.stage + 4 * (i * C + pcol[gcode[k] & 0xFFFFFFu])) = gw[k];
        }
        __syncthreads();
        if (row0 >= r0 && row0 < r0 + nr) {
            const int src = lay.stage + 4 * (row0 - r0) * C + 16 * l8;
#pragma unroll
            for (int q = 0; q < QR; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) w[q][r] = F4(src + 4 * r * C + 128 * q);
            for (int q = QR; q < nq; ++q)
#pragma unroll
                for (int r = 0; r < 4; ++r) F4(lay.xw + 16 * ((4 * (q - QR) + r) * TR + tid)) = F4(src + 4 * r * C + 128 * q);
        }
        __syncthreads();
    }
    if (row0 >= nown && tid < TR)  // threads past the last row: their quads in shared memory are read too
        for (int q = 0; q < 4 * (nq - QR); ++q) F4(lay.xw + 16 * (q * TR + tid)) = make_float4(0.f, 0.f, 0.f, 0.f);
    NeuronPrm P = {};
    float V = 0.0f, y0 = 0.0f, ylo = 0.0f, acc = 0.0f;
    if (has_row) {
        y0 = V = gV[row];
        ylo = gVl ? gVl[row] : 0.0f;
        P = load_neuron_prm(v, n0 + r_lo + row);
    }
    for (int i = tid; i < Nw; i += nthr) {
        const bool own = i < nown;
        F1(lay.vst + 4 * i) = F1(lay.vst + 4 * (Nw + i)) = own ? gV[i] : 0.0f;
        F1(lay.inp + 8 * i) = own ? v.i_const[n0 + r_lo + i] : 0.0f;
        F1(lay.inp + 8 * i + 4) = own && v.pulse_amp ? v.pulse_amp[n0 + r_lo + i] : 0.0f;
        float g[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const long long at = (long long)(x + 1) * v.N + i;
            g[x] = own ? gV[at] : 0.0f;
            F4(lay.gst + 16 * (x * Nw + i)) = make_float4(g[x], own && gVl ? gVl[at] : 0.0f, 0.0f, g[x]);
        }
        F4(lay.ys + 16 * i) = make_float4(g[0], g[1], g[2], 0.0f);
    }
    if (cl > 1) {
        // no push before every CTA has cleared its table
        cluster_arrive();
        cluster_wait();
    }
    // own pairs: step-start gates from one synapse of each, stage-0 gates
    for (int p = tid; p < np; p += nthr) {
        const int2 pr = v.dense_pair[p_lo + p];
        const int j = pr.x / nt, t = pr.x - j * nt, col = pcol[pr.x];
        const float r = gr[pr.y], rl = grl ? grl[pr.y] : 0.0f;
        F4(lay.pst + 16 * p) = make_float4(r, rl, 0.0f, 0.0f);
        *(float2 *)(dsm + lay.pacc + 8 * p) = make_float2(0.0f, 0.0f);
        *(int2 *)(dsm + lay.pinfo + 8 * p) = make_int2(4 * (j - r_lo), (t << 24) | (4 * col));
        float g = __fadd_rn(r, rl);
        if (p >= np1) {
            const float s = gr[v.S + pr.y], sl = grl ? grl[v.S + pr.y] : 0.0f;
            F4(lay.pst2 + 32 * (p - np1)) = make_float4(s, sl, 0.0f, 0.0f);
            F4(lay.pst2 + 32 * (p - np1) + 16) = make_float4(0.f, 0.f, 0.f, 0.f);
            g = second_gate(__fadd_rn(s, sl), stab[t * ST_COLS + SP_KD]);
        }
        put(lay.g + 4 * col, cl, bounded(g));
    }
    __syncthreads();
    if (cl > 1) {
        cluster_arrive();
        cluster_wait();
    }

    // each thread's first neuron (highest threads first), first-order pair
    // (on the threads below) and second-order pair (below those): with enough
    // threads every warp has one kind of work
    const int i0 = nthr - 1 - tid, W1 = (np1 + 31) & ~31;
    const int u1 = ((i0 - Nw) % nthr + nthr) % nthr, u2 = ((i0 - Nw - W1) % nthr + nthr) % nthr;
    const long long pon = v.pulse_on[b], poff = v.pulse_off[b];
    int vc = lay.vst, vn = lay.vst + 4 * Nw;                      // stage potential: this stage's, the next's
    int yc = lay.ys, yn = lay.ys + 16 * Nw;                       // stage gates m, h, n
    int gc = lay.g, gn = lay.g + 4 * C, gx = lay.g + 8 * C;       // gate table: this stage's, the next's, the last's
    int rec_phase = v.rec_stride > 0 ? (int)((step0 + 1) % v.rec_stride) : -1;
    const float4 c0 = F4(lay.sc);
    StageCoef cf{c0.x, c0.y, c0.z, c0.w};
    float iext = 0.0f;
    long long rec_at = 0;
    // one stage; next: the index of the stage after it
    auto stage = [&](auto last, int next, bool rec_now) {
        constexpr bool LAST = decltype(last)::value;
        // next gates of the own pairs
#pragma unroll 1
        for (int p = u1; p < np1; p += nthr) {
            float4 st = F4(lay.pst + 16 * p);
            const int2 info = *(const int2 *)(dsm + lay.pinfo + 8 * p);
            float2 a = *(const float2 *)(dsm + lay.pacc + 8 * p);
            const float g = pair_unit<LAST>(cf, stab + (info.y >> 24) * ST_COLS, F1(vc + info.x), st, a);
            put(gn + (info.y & 0xFFFFFF), cl, bounded(g));
            F4(lay.pst + 16 * p) = st;
            *(float2 *)(dsm + lay.pacc + 8 * p) = a;
        }
#pragma unroll 1
        for (int p2 = u2; p2 < np2; p2 += nthr) {
            const int p = np1 + p2;
            float4 st = F4(lay.pst + 16 * p), q = F4(lay.pst2 + 32 * p2), z = F4(lay.pst2 + 32 * p2 + 16);
            const int2 info = *(const int2 *)(dsm + lay.pinfo + 8 * p);
            float2 a = *(const float2 *)(dsm + lay.pacc + 8 * p);
            const float *sp = stab + (info.y >> 24) * ST_COLS;
            const float r0 = st.x, sP = st.z, sQ = st.w;
            pair_unit<LAST>(cf, sp, F1(vc + info.x), st, a);
            put(gn + (info.y & 0xFFFFFF), cl, bounded(pair_unit2<LAST>(cf, sp, r0, sP, sQ, q, z)));
            F4(lay.pst + 16 * p) = st;
            *(float2 *)(dsm + lay.pacc + 8 * p) = a;
            F4(lay.pst2 + 32 * p2) = q;
            F4(lay.pst2 + 32 * p2 + 16) = z;
        }
        if (cl > 1) {
            __syncwarp();
            cluster_arrive();
        }
        // gates m, h, n of the owned neurons
#pragma unroll 1
        for (int i = i0; i < Nw; i += nthr) {
            const float Vi = F1(vc + 4 * i), e = rate_e(Vi);
            const int o = lay.gst + 16 * i;
            float4 m = F4(o), h = F4(o + 16 * Nw), n = F4(o + 32 * Nw);
            gate_update<LAST>(cf, alpha_m(Vi, e), beta_m(Vi), m);
            gate_update<LAST>(cf, alpha_h(Vi), beta_h(e), h);
            gate_update<LAST>(cf, alpha_n(Vi, e), beta_n(Vi), n);
            F4(o) = m;
            F4(o + 16 * Nw) = h;
            F4(o + 32 * Nw) = n;
            F4(yn + 16 * i) = make_float4(m.w, h.w, n.w, 0.0f);
        }
        if (tid < TR) {
            const float4 V4 = F4(vc + 4 * row0);
            const int g0 = gc + 16 * l8;
            float I[4] = {};
#pragma unroll
            for (int q = 0; q < QR; ++q) quad(w[q], F4(g0 + 128 * q), F1(lay.eq + 4 * q), V4, I);
#pragma unroll 2
            for (int q = QR; q < nq; ++q) {
                const int x = lay.xw + 16 * (4 * (q - QR) * TR + tid);
                const float4 wq[4] = {F4(x), F4(x + 16 * TR), F4(x + 32 * TR), F4(x + 48 * TR)};
                quad(wq, F4(g0 + 128 * q), F1(lay.eq + 4 * q), V4, I);
            }
            const float isyn = row_sum(I, l8);
            const float4 y = F4(yc + 16 * row);
            const float d = __fmul_rn(__fsub_rn(ionic_rest(P, V, y.x, y.y, y.z, iext), isyn), P.invC);
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
                if (LAST && rec_now) v.rec[rec_at + row] = V;
            }
        }
        const float4 c4 = F4(lay.sc + 16 * next);
        cf = StageCoef{c4.x, c4.y, c4.z, c4.w};
        __syncthreads();
        if (cl > 1) cluster_wait();
        int t = vc;
        vc = vn;
        vn = t;
        t = yc;
        yc = yn;
        yn = t;
        t = gc;
        gc = gn;
        gn = gx;
        gx = t;
    };
    for (int itn = 0; itn < nsteps; ++itn) {
        const long long step = step0 + itn;
        const bool rec_now = rec_phase == 0;
        if (rec_phase >= 0) rec_phase = rec_phase + 1 == v.rec_stride ? 0 : rec_phase + 1;
        if (rec_now) rec_at = (((step + 1) / v.rec_stride - 1) % v.rec_cap) * v.N + n0 + r_lo;
        if (has_row)
            iext = input_current(v, F1(lay.inp + 8 * row), F1(lay.inp + 8 * row + 4), step >= pon && step < poff,
                                 (long long)n0 + r_lo + row, step);
#pragma unroll 1
        for (int s = 0; s < ns - 1; ++s) stage(std::false_type{}, s + 1, false);
        stage(std::true_type{}, 0, rec_now);
    }

    // ---- write back: final gates to every CTA (by column), then the owned
    // neurons and the owned rows' synapses
    if (cl > 1) {
        // a peer may still read its table in its last sum
        cluster_arrive();
        cluster_wait();
    }
    for (int p = tid; p < np; p += nthr) {
        const float4 st = F4(lay.pst + 16 * p);
        const int o = lay.g + ((*(const int2 *)(dsm + lay.pinfo + 8 * p)).y & 0xFFFFFF);
        put(o, cl, st.x);
        put(o + 4 * C, cl, st.y);
        if (p >= np1) {
            const float4 q = F4(lay.pst2 + 32 * (p - np1));
            put(o + 8 * C, cl, q.x);
            put(o + 12 * C, cl, q.y);
        }
    }
    __syncthreads();
    if (cl > 1) {
        cluster_arrive();
        cluster_wait();
    }
    {
        const long long k0 = rp[0] - sbase, k1 = rp[nown] - sbase;
        for (long long k = k0 + tid; k < k1; k += nthr) {
            const uint32_t code = gcode[k];
            const int o = lay.g + 4 * pcol[code & 0xFFFFFFu];
            const bool sec = second_order(stab, code);
            gr[k] = F1(o);
            if (sec) gr[v.S + k] = F1(o + 8 * C);
            if (grl) {
                grl[k] = F1(o + 4 * C);
                if (sec) grl[v.S + k] = F1(o + 12 * C);
            }
        }
    }
    bool bad = false;
    if (writes) {
        bad = !isfinite(y0);
        gV[row] = y0;
        if (gVl) gVl[row] = ylo;
    }
    for (int i = tid; i < nown; i += nthr) {
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            const long long at = (long long)(x + 1) * v.N + i;
            const float4 st = F4(lay.gst + 16 * (x * Nw + i));
            bad |= !isfinite(st.x);
            gV[at] = st.x;
            if (gVl) gVl[at] = st.y;
        }
    }
    if (bad) set_error(v.err, PSST_ERR_NONFINITE);
}

template <int QR, int MAXT>
__global__ void __launch_bounds__(MAXT) dense_kernel(NetView v, const int *list, const DensePlan *plans,
                                                     long long step0, int nsteps, int cl) {
    __shared__ float stab[PSST_MAX_SYN_TYPES * ST_COLS];
    load_syn_table(v.sparams, v.n_stypes, stab);
    __syncthreads();
    const int b = list[blockIdx.x / cl];
    dense_run<QR>(v, b, plans[b], step0, nsteps, cl, stab);
}

typedef void (*DenseKernel)(NetView, const int *, const DensePlan *, long long, int, int);

DenseKernel dense_function(int qr) {
    switch (qr) {
#define PSST_DENSE(QR, MAXT) \
    case QR: return dense_kernel<QR, MAXT>;
        PSST_DENSE_VARIANTS(PSST_DENSE)
#undef PSST_DENSE
    default: return nullptr;
    }
}

}  // namespace

cudaError_t dense_prepare(int qr, int max_smem) {
    const DenseKernel k = dense_function(qr);
    if (!k) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
}

cudaError_t dense_launch(const NetView &v, const ClassLaunch &c, long long step0, int nsteps, cudaStream_t stream) {
    const DenseKernel k = dense_function(c.qr);
    if (!k) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(c.n_nets * c.cl);
    cfg.blockDim = dim3(c.block);
    cfg.dynamicSmemBytes = (size_t)c.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c.cl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c.cl > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, v, c.list, c.dplans, step0, nsteps, c.cl);
}

}  // namespace psst
