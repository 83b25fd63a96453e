// Tiled FP32 reverse kernels of a freely rotating body (lks_free3d.cu).
#pragma once

#include "lks_kernels.h"

namespace lks {

constexpr int kFreeTile = 8;          // cells per tile edge
constexpr int kFreeDesignCtas = 304;  // design-point kernel: two CTAs per SM, striding over the tiles

// Shared memory of the kernels; Geo::free_tiled tells whether a handle may run them, free_*_pays whether
// they are the faster ones for its body box.
bool prepare_free3d();
int free_tiles(const Geo& g);
bool free_cell_pays(const Geo& g);
bool free_design_pays(const Geo& g);
void launch_adj_cell_free(const Geo& g, const Ctrl* ctrl, const Dof* it, const float* kref, const float* boxstore, int nbox,
                          float* Lb, long long lstride, float* acc, float* scratch, int k, int di, cudaStream_t st);
int free_design_ctas(const Geo& g);
void launch_adj_design_free(const Geo& g, Ctrl* ctrl, const Dof* it, const float* kref, const float* scratch, double* dkref,
                            void* partials, int k, int di, cudaStream_t st);

}  // namespace lks
