// Building blocks of the kernels that hold synapses as dense rows in registers
// (psst_dense.cu, psst_adjdense.cu): shared memory by byte offset, the stage
// updates of a gate variable and of a gate pair, the sums of four rows over a
// quad of columns and their exchange among the eight threads of a row group.
#pragma once

#include "psst_device.cuh"
#include "psst_syn.cuh"

namespace psst {

extern __shared__ __align__(16) unsigned char dsm[];

// Shared memory at byte offset o.
__device__ __forceinline__ float &F1(int o) { return *(float *)(dsm + o); }
__device__ __forceinline__ float4 &F4(int o) { return *(float4 *)(dsm + o); }

// One gate variable with rates al, be: st (step-start value, its remainder,
// the step's running sum, stage value) advanced by one stage, the step's last
// if LAST, with the operations of neuron_gates (psst_syn.cuh).  Running sums
// start a step at 0 here and everywhere below: the first stage's term w d is
// fma(w, d, 0).
template <bool LAST>
__device__ __forceinline__ void gate_update(const StageCoef &c, float al, float be, float4 &st) {
    const float d = fmaf(al, __fsub_rn(1.0f, st.w), -__fmul_rn(be, st.w));
    const float ac = fmaf(c.w, d, st.z);
    if (!LAST) {
        st.z = ac;
        st.w = ext_stage(st.x, st.y, c.cn, d);
    } else {
        ext_step(st.x, st.y, c.fin, c.finl, ac);
        st.z = 0.0f;
        st.w = st.x;
    }
}

// One pair's r from a_ = a T and bb = a T + b at its neuron's potential: st
// (step-start gate, remainder, stage map P, Qm), acc the step's running sums,
// with the operations of coef_update, pair_step and pair_gate; returns the
// next stage's r.
template <bool LAST>
__device__ __forceinline__ float pair_unit(const StageCoef &c, float a_, float bb, float4 &st, float2 &acc) {
    const float kP = fmaf(-bb, st.z, a_), kQ = fmaf(-bb, st.w, -bb);
    const float aP = fmaf(c.w, kP, acc.x);
    const float aQ = fmaf(c.w, kQ, acc.y);
    if (!LAST) {
        acc = make_float2(aP, aQ);
        st.z = __fmul_rn(c.cn, kP);
        st.w = __fmul_rn(c.cn, kQ);
        return __fadd_rn(st.x, __fadd_rn(fmaf(st.w, st.x, st.z), st.y));
    }
    ext_add(st.x, st.y, fmaf(step_end(c, aQ), st.x, step_end(c, aP)));
    st.z = st.w = 0.0f;
    acc = make_float2(0.0f, 0.0f);
    return __fadd_rn(st.x, st.y);
}

template <bool LAST>
__device__ __forceinline__ float pair_unit(const StageCoef &c, const float *sp, float V, float4 &st, float2 &acc) {
    const float a_ = __fmul_rn(sp[SP_A], transmitter(V, sp));
    return pair_unit<LAST>(c, a_, __fadd_rn(a_, sp[SP_B]), st, acc);
}

__device__ __forceinline__ float second_gate(float s, float Kd) {
    const float s2 = __fmul_rn(s, s), s4 = __fmul_rn(s2, s2);
    return __fdiv_rn(s4, __fadd_rn(s4, Kd));
}

// The second gate of a second-order pair (r0 its step-start r, P and Qm this
// stage's map of r): q (step-start s, remainder, stage map U, X), z (map Zm,
// running sums); returns the next stage's G = s^4 / (s^4 + Kd).
template <bool LAST>
__device__ __forceinline__ float pair_unit2(const StageCoef &c, const float *sp, float r0, float P, float Qm, float4 &q,
                                            float4 &z) {
    const float K3 = sp[SP_K3], K4 = sp[SP_K4];
    const float kU = fmaf(K3, P, __fmul_rn(-K4, q.z)), kX = fmaf(K3, Qm, fmaf(-K4, q.w, K3));
    const float kZ = fmaf(-K4, z.x, -K4);
    const float aU = fmaf(c.w, kU, z.y);
    const float aX = fmaf(c.w, kX, z.z);
    const float aZ = fmaf(c.w, kZ, z.w);
    float s;
    if (!LAST) {
        z = make_float4(__fmul_rn(c.cn, kZ), aU, aX, aZ);
        q.z = __fmul_rn(c.cn, kU);
        q.w = __fmul_rn(c.cn, kX);
        s = __fadd_rn(q.x, __fadd_rn(fmaf(z.x, q.x, fmaf(q.w, r0, q.z)), q.y));
    } else {
        ext_add(q.x, q.y, fmaf(step_end(c, aZ), q.x, fmaf(step_end(c, aX), r0, step_end(c, aU))));
        q.z = q.w = 0.0f;
        z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        s = __fadd_rn(q.x, q.y);
    }
    return second_gate(s, sp[SP_KD]);
}

// Four rows' currents over one quad of columns with reversal potential E.
__device__ __forceinline__ void quad(const float4 (&w)[4], float4 g, float E, const float4 &V, float (&I)[4]) {
    const float Vr[4] = {V.x, V.y, V.z, V.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float a = __fmul_rn(w[r].x, g.x);
        a = fmaf(w[r].y, g.y, a);
        a = fmaf(w[r].z, g.z, a);
        a = fmaf(w[r].w, g.w, a);
        I[r] = fmaf(a, __fsub_rn(Vr[r], E), I[r]);
    }
}

// The same with the rows' synaptic conductances in A.
__device__ __forceinline__ void quad(const float4 (&w)[4], float4 g, float E, const float4 &V, float (&I)[4],
                                     float (&A)[4]) {
    const float Vr[4] = {V.x, V.y, V.z, V.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float a = __fmul_rn(w[r].x, g.x);
        a = fmaf(w[r].y, g.y, a);
        a = fmaf(w[r].z, g.z, a);
        a = fmaf(w[r].w, g.w, a);
        I[r] = fmaf(a, __fsub_rn(Vr[r], E), I[r]);
        A[r] = __fadd_rn(A[r], a);
    }
}

// The largest finite number in place of one that is not finite.  Absent synapses
// are weights of 0: with such a gate in the table they add 0 to their rows and
// not NaN, while a present synapse drives its neuron out as well.  (Two versions
// of the sums, with and without absent synapses, made a stage 5 to 18% longer, a
// look through the row's synapses 5 to 10%.)
__device__ __forceinline__ float bounded(float x) { return fmaxf(fminf(x, 3.402823466e38f), -3.402823466e38f); }

// Sum over the eight threads of a row group: thread l gets row
// 2 (l & 1) + (l >> 1 & 1).
__device__ __forceinline__ float row_sum(const float (&a)[4], int l) {
    const bool b0 = l & 1, b1 = l & 2;
    float x0 = __shfl_xor_sync(0xffffffffu, b0 ? a[0] : a[2], 1);
    float x1 = __shfl_xor_sync(0xffffffffu, b0 ? a[1] : a[3], 1);
    x0 = __fadd_rn(b0 ? a[2] : a[0], x0);
    x1 = __fadd_rn(b0 ? a[3] : a[1], x1);
    const float y = __shfl_xor_sync(0xffffffffu, b1 ? x0 : x1, 2);
    x0 = __fadd_rn(b1 ? x1 : x0, y);
    return __fadd_rn(x0, __shfl_xor_sync(0xffffffffu, x0, 4));
}

}  // namespace psst
