// sp_kernels.h -- host-callable launchers of the kernels in sp_kernels.cu.
#pragma once
#include <cuda_runtime.h>

#include "sp_device.cuh"

namespace sp {

cudaError_t launch_reset(const RegionArgs &a, cudaStream_t st);
// 16 cost-model features per region of the launch into X [total][16].
cudaError_t launch_features(const RegionArgs &a, const float4 *simf, const unsigned long long *prev_trace, float *X,
                            cudaStream_t st);
// The region kernel of a base with a worker count: regions per CTA, CTAs per SM
// (none: it does not fit) and dynamic shared memory.
struct RegionConfig {
    int groups = 1, ctas_per_sm = 0;
    size_t smem = 0;
};
cudaError_t region_config(int threads, int B, int imp_units, RegionConfig *c);
cudaError_t launch_region(const RegionArgs &a, int threads, int B, int groups, size_t smem, int grid, cudaStream_t st);
cudaError_t launch_sweep(const float2 *phi_in, float2 *phi_out, float4 *pc, const int n[3],
                         const LevelCoef *coef, int lvl, PhysConst q, cudaStream_t st);
// Two levels of the whole grid in one pass, from one copy of the state to
// another (sp_columns.cu); coef: of the first of them.  columns_pay: whether
// that is faster than two one-level sweeps of this grid.
bool columns_pay(const float2 *phi, const float4 *pc, const int n[3], int sm_count);
cudaError_t launch_columns(const float2 *phi_in, const float4 *pc_in, float2 *phi_out, float4 *pc_out, const int n[3],
                           const LevelCoef *coef, PhysConst q, int sm_count, cudaStream_t st);
// Diagnostics of a stored state (sp_diag.cu): energy terms and winding counts
// in one pass, and the map of plaquette windings [3][sites].
struct DiagOut {
    double energy[3];      // kinetic, gradient, potential
    long long winding[7];  // pierced plaquettes by normal axis, sum |w|, sum w by normal axis
};
size_t diag_scratch_bytes(const int n[3]);
cudaError_t launch_diag(const float2 *phi, const float4 *pc, const int n[3], double inv_dx2, double eta2,
                        double half_lambda_a2, void *scratch, DiagOut *out, cudaStream_t st);
cudaError_t launch_winding_map(const float2 *phi, const int n[3], signed char *map, cudaStream_t st);

}  // namespace sp

namespace sp {
// The base-32 cluster kernel (sp_octant.cu): shared memory per CTA, the
// number of 8-CTA clusters that fit the device, its launch and worker count.
size_t region_oct_smem_bytes(int imp_units, int face_units);
cudaError_t region_oct_clusters(size_t smem, int *clusters);
cudaError_t launch_region_oct(const RegionArgs &a, size_t smem, int clusters, cudaStream_t st);
int region_oct_workers();
}  // namespace sp

namespace sp {
struct LatticeTables;
// The 4-cube lattice kernels (sp_lattice.cu): how a size runs with a worker
// count (regions per CTA, CTAs per SM, dynamic shared memory; no CTA: it does
// not fit), the per-call reset (ticket counter, error word, layer epoch) and
// the launch of `grid` CTAs.
struct LatConfig {
    bool resident = false;  // the kernel with the whole cell list in shared memory
    int groups = 1, ctas_per_sm = 0;
    size_t smem = 0;
};
bool lattice_valid_threads(int threads);
bool lattice_ring_faster(int s, int threads, bool few);  // few: regions of a layer
bool lattice_ring_brief(int s, long long n_steps, long long per_layer, int sms);
cudaError_t lattice_config(const LatticeTables &t, int threads, bool ring, LatConfig *c);
cudaError_t launch_lattice_reset(Ctl *ctl, int layers, cudaStream_t st);
cudaError_t launch_lattice(const LatArgs &a, int threads, size_t smem, int grid, cudaStream_t st);
}  // namespace sp
