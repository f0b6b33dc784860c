// Host-side declarations shared by the CUDA translation units of the library.
#pragma once

#include <cuda_runtime.h>

#include "psst_device.cuh"

namespace psst {

// One launch of the CTA/cluster kernel: the networks of one size class.
struct ClassLaunch {
    int cl;               // CTAs per network (1, 2 or 4)
    int n_nets;           // networks in the class
    int block, smem;      // CTA size, dynamic shared memory
    const int *list;      // [n_nets] device: network indices, largest first
    const NetPlan *plans; // [all nets] device
    int lrep_cap;         // per-pair gates: at most 2^lrep_cap copies of the gate table (autotuned)
    int qr;               // dense kernel: quads per thread in registers (0: the item kernel)
    int rows;             // dense kernel: threads that hold rows (the smallest block)
    const DensePlan *dplans; // dense kernel: [all nets] device
};

// Dense kernel (psst_dense.cu): quads per thread held in registers and the
// largest block of each compiled variant.  An SM quarter holds 512 registers
// per lane, so the block sizes with 6, 5, 4, 3 and 2 warps a quarter leave
// 80, 96, 128, 168 and 255 registers a thread: 16 per quad and about 55 for
// everything else.  A quad in shared memory costs four 16-byte loads more and
// shows: a network of 300 neurons on 4 CTAs takes 4.1 us per step with all 10
// quads in registers, 5.6 with 2 (240 neurons on 2: 4.6 with 6 of 8, 5.6 with 1).
#define PSST_DENSE_VARIANTS(X) \
    X(1, 768) X(2, 640) X(3, 512) X(4, 512) X(5, 384) X(6, 384) X(7, 384) X(8, 256) X(9, 256) X(10, 256)
cudaError_t dense_prepare(int qr, int max_smem);
cudaError_t dense_launch(const NetView &v, const ClassLaunch &c, long long step0, int nsteps, cudaStream_t stream);

// CTA/cluster batched kernel (psst_cta.cu).
int cta_static_smem();
cudaError_t cta_prepare(int cl, int max_smem);
cudaError_t pair_check(const NetView &v, uint8_t *out, int smem, cudaStream_t stream);
cudaError_t cta_launch(const NetView &v, const ClassLaunch &c, long long step0, int nsteps, cudaStream_t stream);

// Networks without synapses, one thread per neuron (psst_indep.cu).
cudaError_t indep_launch(const NetView &v, const int *ind_neuron, const int *ind_net, int count, long long step0,
                         int nsteps, cudaStream_t stream);

// Grid-wide single-network kernel (psst_grid.cu).
cudaError_t grid_occupancy(int block, int smem, int *blocks_per_sm);
cudaError_t grid_launch(const NetView &v, const GridView &g, long long step0, int nsteps, int grid, int block,
                        int smem, cudaStream_t stream);

// Discrete adjoint (psst_adjoint.cu).
long long adj_smem_need(int N, int nt, int n_items, int K, int n_citems, int KC);
// Floats one step keeps in an adjoint segment buffer (its stages: RK4 four,
// Euler one, a tableau rk_ns).
long long adj_segment_floats(int method, int rk_ns, int N, int nt);
cudaError_t adj_launch(const NetView &v, const AdjView &av, long long step0, int nsteps, int smem, int n_types,
                       float *grad_np, cudaStream_t stream);


// The adjoint over dense rows (psst_adjdense.cu): networks of at most
// 32 x ADJ_DENSE_Q neurons and ADJ_DENSE_TYPES synapse types whose pair slots
// (two threads each) leave ADJ_DENSE_NEURONS of the threads to the neurons; Q:
// quads of neurons per pair row.
constexpr int ADJ_DENSE_Q = 4, ADJ_DENSE_TYPES = 4, ADJ_DENSE_THREADS = 384, ADJ_DENSE_NEURONS = 64;
cudaError_t adj_dense_launch(const NetView &v, const AdjDenseView &av, int Q, int threads, int smem, long long step0,
                             int nsteps, int n_types, float *grad_np, cudaStream_t stream);
// Sum of the per-neuron parameter gradients into the neuron-type table.
cudaError_t adj_reduce(const NetView &v, const double *gp_neuron, int n_types, float *grad_np, cudaStream_t stream);

}  // namespace psst
