// Host-side declarations shared by the C ABI and the kernel launchers.
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>
#include <cuda_runtime.h>

#include "pps_device.cuh"

struct pps_params;

namespace pps {

// The order in which pass two of the insert adds contributions up (add_ordered
// in pps_kernels.cu says why).
enum AddOrder : int {
  kAnyOrder = 0,       // no order: the sums' FP32 rounding may take any of its values
  kRowsBackwards = 1,  // rows of 32 vertices, from the end of the stream
  kPairsForwards = 2,  // pairs of neighbouring vertices, from its start
};

// Launch geometry of the persistent filter kernel for one call.
struct FusedPlan {
  int grid = 0;       // CTAs
  int block = 0;      // threads per CTA
  int batch = 2;      // vertices per lane per insert step (2 or 4)
  uint32_t tile = 0;  // vertices per warp tile
  bool temporal = false;  // kernel variants: a table with a history
  bool evict = false;     // ... an evicting one
  bool neigh = false;     // ... the neighborhood search
  bool kv = false;        // ... vertices with key variants
  bool sweep = false;     // zero the whole slot table first, not the frame's slots at the end
  size_t swept = 0;       // slots the launch zeroes, or may find left over and have to zero
  int merge = 2;      // merging of equal keys within a warp (pps_tuning.merge)
  bool backwards = false;  // insert from the end of the vertex stream
  AddOrder order = kAnyOrder;
};

// One view of a batched launch: its table, key constants, vertices and
// outputs, and its place in the batch's tile space.
struct ViewDesc {
  KeyConst kc;
  TableDev t;
  VertexPtrs v;
  OutPtrs o;
  unsigned long long n;
  uint32_t tile_base;  // first tile of this view in the batch
  uint32_t ntiles;
  int blended;  // blend this view's cells (temporal table and blending requested)
  int sweep;    // zero this view's slot table by a sweep first
  int ordered;  // add contributions up in the order of kPairsForwards
};

struct MultiPlan {
  int grid = 0, block = 0, batch = 2;
  uint32_t tile = 0;  // vertices per warp tile
};

// Plan / launch the batched persistent kernel over `total_tiles` warp tiles of
// `tile` vertices (`swept`: slots of all tables) of the views in device memory (`views`, nviews entries);
// `ctrl` carries the grid barrier, `stash` (total_tiles
// tiles) the vertices' cell ids.
cudaError_t plan_multi(size_t total_tiles, uint32_t tile, size_t swept, bool temporal, int batch,
                       int block, MultiPlan* plan);
cudaError_t launch_multi(const ViewDesc* views, uint32_t nviews, uint32_t total_tiles, Ctrl* ctrl,
                         bool temporal, bool ordered, float alpha, const MultiPlan& plan,
                         uint32_t* stash, cudaStream_t st);
// The additions' order on frames of table t that are blended (`backwards`: ones
// whose contributions have always been added up from the end of the stream).
AddOrder add_order(const TableDev& t, bool backwards);
bool sweep_pays_host(const TableDev& t, size_t vertices);

// `wide`: ids of this insert may take all 32 bits, so that the stash has no bit
// left for a cell's creator.
cudaError_t launch_insert(const KeyConst& kc, const TableDev& t, const VertexPtrs& v, size_t n,
                          uint32_t* stash, uint32_t* id_out, uint32_t unit_base, bool wide, int batch,
                          int merge, cudaStream_t st);
cudaError_t launch_query(const KeyConst& kc, const TableDev& t, const VertexPtrs& v, size_t n,
                         const uint32_t* id_in, const OutPtrs& o, bool blended, uint32_t id_limit,
                         cudaStream_t st);
cudaError_t launch_keys(const KeyConst& kc, const VertexPtrs& v, size_t n, uint32_t* h_out,
                        uint32_t* f_out, cudaStream_t st);
cudaError_t launch_blend(const KeyConst& kc, const TableDev& t, uint32_t ntiles, float alpha,
                         cudaStream_t st);
// Empty the slots: those of the split path's frame of `ntiles` tiles, or all of
// them where a launch left its own (Ctrl::left, which the caller resets).
cudaError_t launch_clear(const TableDev& t, uint32_t ntiles, cudaStream_t st);
// Evicting history: lower every entry's priority by `by` (epoch rebase).
cudaError_t launch_hist_age(const TableDev& t, uint32_t by, cudaStream_t st);
// Multi-level accumulation: vertices with fine status LOWCOUNT take the
// coarse resolution's value, count and status COARSE (unless the coarse
// insert overflowed).  `fine_status` may alias o.status.
cudaError_t launch_combine_coarse(size_t n, const uint8_t* fine_status, const OutPtrs& coarse,
                                  const OutPtrs& o, cudaStream_t st);
cudaError_t launch_count_nonzero(const void* base, uint32_t stride, uint32_t off, uint32_t width,
                                 uint64_t n, unsigned long long* out, cudaStream_t st);
// Fill in the geometry of a plan whose kernel variant and batch are set
// (tiles whose id ranges span at most max_cells cells).
cudaError_t plan_fused(size_t n, size_t max_cells, FusedPlan* plan);
cudaError_t launch_fused(const KeyConst& kc, const TableDev& t, const VertexPtrs& v, size_t n,
                         const OutPtrs& o, bool blend, float alpha, const FusedPlan& plan, uint32_t* stash, uint32_t* nq, cudaStream_t st);

int sm_count();   // multiprocessors of the device
// The split path hands out cell ids in units: ids per unit, and units that one
// insert of n vertices takes.
int split_unit_ids();
size_t split_units(size_t n);
// ... of the persistent kernels, for a launch over n vertices
uint32_t fused_tile(size_t n, int batch);
// Cells that the tiles' id ranges span (tiles of `tile` vertices).
size_t fused_cells(size_t n, uint32_t tile, int batch);
bool aligned16(const void* p);

int record_error(int code, const char* msg);  // message for pps_last_error()
const char* last_error_text();                // the message pps_last_error() returns
std::string device_error_text(unsigned int word);  // the bits of a device error word
// Checks of table parameters shared by pps_create and pps_filter_noalloc
// (PPS_OK, or PPS_EINVAL with the reason recorded for pps_last_error()).
int check_params(const pps_params* p);

// Self-test of the tensor-core kernels' bounded mbarrier wait (pps_mlp.cu).
// One CTA of the learned fallback's evaluation over `tiles` tiles per group, in
// which the thread of row `row` gives up its wait for the output layer; `mem`:
// selftest_infer_bytes() zeroed bytes, 16-byte aligned.
constexpr uint32_t kSelftestVertices = 3 * 512;
size_t selftest_infer_bytes();
cudaError_t launch_selftest_infer(int row, uint32_t tiles, void* mem, unsigned int* err, cudaStream_t st);
cudaError_t launch_selftest_mbar(unsigned long long limit_ns, unsigned int* err, cudaStream_t st);

}  // namespace pps

struct pps_table;

namespace pps {
int table_for_batch(pps_table* t, ViewDesc* vd, int* batch, int* block, bool* temporal);
int table_reserve(pps_table* t, size_t cells, cudaStream_t st);
const TableDev& table_dev(const pps_table* t);

}  // namespace pps
