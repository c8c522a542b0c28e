// Interface of the tiled (TMA-staged, order-streamed) half-step kernel.
#pragma once
#include <string>
#include <vector>

#include "host_math.h"

namespace starmap {

struct TiledPlan;

struct TiledGeometry {
    void* base[4];
    long cstride[4];
    int nx[4], ny[4], K[4];
    int cp[4];                         // row pitch of the decay coefficients and sources
    long pitch, rows;
    int p[2];
    int N;
    int variant = 0;                   // tile height: 0 = 10 rows, 1 = 5 rows
    int shape = -1;                    // tile shape, or -1 for the one the height, order and grid ask for
                                       // (the instances of a batch share one: tiled_batch_shape)
};

// Tile height the tiled kernel uses for order N on nx x ny points when
// nothing else decides.
int tiled_default_variant(int N, int nx, int ny);

bool tiled_supported(int system, int N, int precision);
// Host only: the stage list of pass P (parity of its outputs) as global
// components (4 per stage: input R, input I, output R, output I; -1 absent),
// its coefficient rows (16 floats per input, each value twice) and the
// component finalised at each finalising event (-1: absent I).
int tiled_schedule(int N, int P, bool frozen_top, double dx, double dy, std::vector<int>& stages,
                   std::vector<float>& coef, std::vector<int>& fin, std::string& err);
int tiled_create(const TiledGeometry& geo, TiledPlan** out);
// frozen[j] != 0: component j is read but never written (closure moments)
int tiled_update(TiledPlan* plan, const SystemMatrices& sys, const std::vector<int>& comp_class,
                 const std::vector<int>& src_slot, const std::vector<void*>& src_dev,
                 const std::vector<char>& frozen, double dx, double dy);
void tiled_set_coef(TiledPlan* plan, int g, void* coef, int nclasses);
int tiled_pass(TiledPlan* plan, bool odd, int which, void* stream);
// Temporally fused step: one launch applies the full even update and then
// the full odd update, tile by tile (fused_kernel.cuh), reading one buffer
// set and writing the other.  base1: the second set's grid bases (the same
// layout as the first).  The fused parameters follow every table rebuild.
int tiled_fused_setup(TiledPlan* plan, void* const base1[4]);
bool tiled_fused_ready(TiledPlan* plan);
// dir 0: set 0 -> set 1; dir 1: set 1 -> set 0.  The caller refreshes the
// boundary copies of the written odd grids afterwards.
int tiled_fused_step(TiledPlan* plan, int dir, void* stream);
// Read and clear the bounded-wait failure flag (synchronises the stream).
int tiled_poll(TiledPlan* plan, void* stream);
const char* tiled_error(TiledPlan* plan);
void tiled_destroy(TiledPlan* plan);

// Batched passes over several plans (one persistent launch per pass).
size_t tiled_params_bytes();
// Copy the plan's four pass parameter blocks (index 2 P + which) to host4.
int tiled_export_params(TiledPlan* plan, void* host4);
int tiled_smem_bytes(TiledPlan* plan, int P);
void tiled_tile_grid(TiledPlan* plan, int* tiles_x, int* tiles_y);
int tiled_stage_count(TiledPlan* plan, int P);
// Self-test of the bounded wait (an mbarrier nothing arrives at); *gave_up = 1
// when the wait expired and raised the flag as it must.
int tiled_wait_selftest(int* gave_up);
// Microseconds that the end of two producers takes that gave up some stages apart.
int tiled_drain_selftest(int* us);
// The tile shape of a batch's kernel: for a tile height and its highest order.
int tiled_batch_shape(int variant, int max_N);
// Resident CTAs per SM of that kernel with smem_bytes of dynamic shared memory.
int tiled_batch_ctas(int smem_bytes, int shape);
// Allow it smem_bytes of dynamic shared memory.
int tiled_batch_prepare(int smem_bytes, int shape);
// items: device array of int4 (instance, first tile, tile count, stride),
// each the tiles first, first + stride, ... of one instance; CTA b runs
// items off[b] .. off[b + 1] - 1 (off: grid + 1 device ints); params: device array
// of 4 * instances parameter blocks (instance i, parity P, which at
// 4 i + 2 P + which).
int tiled_batch_pass(const void* params, const void* items, const int* off, int P, int which, int grid,
                     int smem_bytes, int shape, void* stream);

}  // namespace starmap
