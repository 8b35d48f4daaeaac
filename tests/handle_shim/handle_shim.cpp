// Test-only shim: reaches into mesh and batch handles of the loaded libhgks.so, to put its
// scratch and launch shapes into states that no public call produces on demand.
#include <cstring>
#include "../../paper_2304_09485_gb300/csrc/batch_impl.h"

using namespace hgks;

// as in batch_capi.cu
struct hgks_batch_s {
  Batch *B;
};

// every byte of the reconstruction coefficients: 0xff makes NaNs
extern "C" int hx_fill_coef(hgks_mesh h, int byte) {
  Mesh &m = *mesh_of(h);
  const size_t rows = m.d.hex ? ShapeOf<HexShape>::COEF : ShapeOf<TetShape>::COEF;
  return cudaMemset(m.s.coef, byte, sizeof(double) * rows * m.N) != cudaSuccess;
}
extern "C" int hx_fill_batch_coef(hgks_batch b, int byte) {
  Mesh &m = b->B->m;
  const size_t rows = m.d.hex ? ShapeOf<HexShape>::COEF : ShapeOf<TetShape>::COEF;
  return cudaMemset(m.s.coef, byte, sizeof(double) * rows * m.N) != cudaSuccess;
}

// block shapes of k_recon and k_flux, as the autotuner sets them
extern "C" void hx_batch_shape(hgks_batch b, int recon, int flux) {
  b->B->m.s.blk_recon = recon;
  b->B->m.s.blk_flux = flux;
}

// a one-launch GMRES whose barriers expect `extra` arrivals beyond its blocks and give up after `polls`
extern "C" void hx_barrier(hgks_mesh h, unsigned extra, unsigned polls) {
  mesh_of(h)->s.grid_extra = extra;
  mesh_of(h)->s.grid_polls = polls;
}

// the record of a grid barrier that gave up
extern "C" int hx_set_stuck(hgks_mesh h) {
  const int64_t one = 1;
  return cudaMemcpy(mesh_of(h)->s.hs + kHsStuck, &one, sizeof(one), cudaMemcpyHostToDevice) != cudaSuccess;
}

// the largest mesh of the one-launch FP64 GMRES: 0 for separate launches
extern "C" void hx_grid_cells(hgks_mesh h, int cells) { mesh_of(h)->s.grid_cells = cells; }

// whether the mesh keeps a captured step
extern "C" int hx_captured(hgks_mesh h) {
  const StepGraph *g = mesh_of(h)->graph;
  return g && g->exec;
}
