// Batched filtering of several views (see pps_batch_create in include/pps.h).
//
// A view that fills the GPU by itself is filtered by a persistent launch of its
// own, whose kernel finds the view's pointers and key constants in its
// parameters.  The smaller views share one persistent launch, replayed from a
// CUDA graph, that keeps the descriptor of the view a warp works on in shared
// memory; that costs instructions and registers, but the views pay for the
// barriers and the uneven ends of the phases once.  Eight equal views, shared
// launch against one each: 640,000 vertices a view 277 and 350 us, 1.14 M 447 and
// 427, 2.56 M 961 and 918, 4.55 M 1,616 and 1,269, 10.2 M 4,048 and 3,041.
//
// Per frame only the views' cameras and the frame number change.  For the
// shared launch they live in a descriptor array in device memory, uploaded by a
// copy node at the start of the graph from a pinned host buffer; two buffers
// (and two instantiated graphs) alternate so that filling the next frame's
// descriptors never races with the copy of the previous one.
#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "pps.h"
#include "pps_internal.h"

struct pps_batch {
  struct OwnView {  // a view with a launch of its own
    uint32_t index;  // of its camera
    pps_table* table;
    pps::ViewDesc vd;
    pps::FusedPlan plan;
  };
  int device = 0;
  std::vector<OwnView> own;
  std::vector<pps::ViewDesc> base;  // views of the shared launch, without camera and frame
  std::vector<uint32_t> index;      // of their cameras
  std::vector<pps_table*> tables;   // theirs
  uint32_t total_tiles = 0;
  bool temporal = false;
  bool ordered = false;  // a view of the shared launch adds its contributions up in order
  float alpha = 0.f;
  pps::MultiPlan plan;
  pps::ViewDesc* dviews[2] = {nullptr, nullptr};
  pps::ViewDesc* hviews[2] = {nullptr, nullptr};
  pps::Ctrl* ctrl = nullptr;
  uint32_t* gstash = nullptr;
  cudaGraphExec_t exec[2] = {nullptr, nullptr};
  cudaEvent_t done[2] = {nullptr, nullptr};
  unsigned long long runs = 0;
};

namespace {

// From this many vertices on a view gets a launch of its own.
constexpr size_t kOwnLaunch = size_t{1} << 20;

int bfail(int code, const std::string& msg) { return pps::record_error(code, msg.c_str()); }

void release(pps_batch* b) {
  for (int k = 0; k < 2; ++k) {
    if (b->exec[k]) cudaGraphExecDestroy(b->exec[k]);
    if (b->done[k]) cudaEventDestroy(b->done[k]);
    cudaFree(b->dviews[k]);
    cudaFreeHost(b->hviews[k]);
  }
  cudaFree(b->ctrl);
  cudaFree(b->gstash);
}

}  // namespace

extern "C" {

int pps_batch_create(pps_batch** out, const pps_view* views, uint32_t nviews, int blend,
                     float alpha) {
  if (!out || !views || nviews == 0 || nviews > 4096) return bfail(PPS_EINVAL, "bad views");
  *out = nullptr;
  pps_batch* b = new (std::nothrow) pps_batch();
  if (!b) return bfail(PPS_ENOMEM, "host allocation failed");
  cudaGetDevice(&b->device);
  b->alpha = alpha;
  int batch = 2, block = 512;
  size_t total = 0, own_words = 0, swept = 0;
  for (uint32_t i = 0; i < nviews; ++i) {
    const pps_view& v = views[i];
    if (!v.table || !v.out.r || !v.out.g || !v.out.b || (v.n && (!v.v.px || !v.v.py || !v.v.pz ||
        !v.v.nx || !v.v.ny || !v.v.nz || !v.v.r || !v.v.g || !v.v.b))) {
      delete b;
      return bfail(PPS_EINVAL, "view " + std::to_string(i) + ": table, vertices and r, g, b required");
    }
    if (v.v.dist || v.v.extra) {
      delete b;
      return bfail(PPS_EINVAL, "view " + std::to_string(i) + ": batched views take no dist or extra arrays");
    }
    pps::ViewDesc vd{};
    bool tmp = false;
    int bw = 2, blk = 512;
    if (int rc = pps::table_for_batch(v.table, &vd, &bw, &blk, &tmp)) {
      delete b;
      return rc;
    }
    if (i == 0) {
      batch = bw;
      block = blk;
    }
    vd.v = pps::VertexPtrs{v.v.px, v.v.py, v.v.pz, v.v.nx, v.v.ny, v.v.nz, v.v.r, v.v.g, v.v.b,
                           v.v.id, v.v.id_base, v.v.stream_id, v.v.dist, v.v.extra};
    vd.o = pps::OutPtrs{v.out.r, v.out.g, v.out.b, v.out.count, v.out.status};
    vd.n = v.n;
    vd.blended = blend && tmp ? 1 : 0;
    vd.sweep = pps::sweep_pays_host(vd.t, v.n) ? 1 : 0;
    vd.ordered = vd.blended && pps::add_order(vd.t, false) != pps::kAnyOrder ? 1 : 0;
    if (v.n >= kOwnLaunch) {
      pps::FusedPlan plan;
      plan.merge = 2;
      plan.temporal = vd.blended != 0;
      plan.sweep = vd.sweep != 0;
      plan.swept = static_cast<size_t>(vd.t.mask) + 1;
      if (vd.ordered) plan.order = pps::kPairsForwards;
      b->own.push_back(pps_batch::OwnView{i, v.table, vd, plan});
      own_words = std::max<size_t>(own_words, v.n);
    } else {
      b->temporal = b->temporal || tmp;
      b->ordered = b->ordered || vd.ordered;
      total += v.n;
      swept += static_cast<size_t>(vd.t.mask) + 1;
      b->base.push_back(vd);
      b->index.push_back(i);
      b->tables.push_back(v.table);
    }
  }
  if (blend && (!(alpha <= 1.0f) || alpha != alpha)) {
    delete b;
    return bfail(PPS_EINVAL, "alpha must be finite and <= 1");
  }
  const uint32_t tile = pps::fused_tile(total, batch);
  for (pps::ViewDesc& vd : b->base) {
    vd.tile_base = b->total_tiles;
    vd.ntiles = static_cast<uint32_t>((vd.n + tile - 1) / tile);
    b->total_tiles += vd.ntiles;
  }
  cudaError_t e = cudaSuccess;
  for (pps_batch::OwnView& w : b->own) {
    w.plan.batch = batch;
    if (e == cudaSuccess) e = pps::plan_fused(w.vd.n, ~size_t{0}, &w.plan);
  }
  const uint32_t nshared = static_cast<uint32_t>(b->base.size());
  // room for the cell ids of each view's tiles
  int rc = PPS_OK;
  for (size_t i = 0; i < b->own.size() && e == cudaSuccess && !rc; ++i)
    rc = pps::table_reserve(b->own[i].table, pps::fused_cells(b->own[i].vd.n, b->own[i].plan.tile, batch), nullptr);
  for (size_t i = 0; i < nshared && e == cudaSuccess && !rc; ++i)
    rc = pps::table_reserve(b->tables[i], pps::fused_cells(b->base[i].n, tile, batch), nullptr);
  if (rc) {
    delete b;
    return rc;
  }
  const int graphs = nshared ? 2 : 0;
  if (e == cudaSuccess && nshared)
    e = pps::plan_multi(b->total_tiles, tile, swept, b->temporal, batch, block, &b->plan);
  const size_t bytes = nshared * sizeof(pps::ViewDesc);
  for (int k = 0; k < graphs && e == cudaSuccess; ++k) {
    e = cudaMalloc(&b->dviews[k], bytes);
    if (e == cudaSuccess) e = cudaMallocHost(&b->hviews[k], bytes);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&b->done[k], cudaEventDisableTiming);
    if (e == cudaSuccess) std::memcpy(b->hviews[k], b->base.data(), bytes);
  }
  if (e == cudaSuccess) e = cudaMalloc(&b->ctrl, sizeof(pps::Ctrl));
  if (e == cudaSuccess) e = cudaMemset(b->ctrl, 0, sizeof(pps::Ctrl));
  // the launches follow one another, so they share the stash
  const size_t words = std::max(own_words, static_cast<size_t>(b->total_tiles) * tile);
  if (e == cudaSuccess && words) e = cudaMalloc(&b->gstash, words * sizeof(uint32_t));
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  // capture: descriptor upload, the persistent kernel
  cudaStream_t cs = nullptr;
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  for (int k = 0; k < graphs && e == cudaSuccess; ++k) {
    cudaGraph_t g = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) e = cudaMemcpyAsync(b->dviews[k], b->hviews[k], bytes, cudaMemcpyHostToDevice, cs);
    if (e == cudaSuccess)
      e = pps::launch_multi(b->dviews[k], nshared, b->total_tiles, b->ctrl, b->temporal, b->ordered, alpha,
                            b->plan, b->gstash, cs);
    cudaError_t e2 = cudaStreamEndCapture(cs, &g);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec[k], g, 0);
    if (g) cudaGraphDestroy(g);
  }
  if (cs) cudaStreamDestroy(cs);
  if (e != cudaSuccess) {
    release(b);
    delete b;
    cudaGetLastError();
    return bfail(e == cudaErrorMemoryAllocation ? PPS_ENOMEM : PPS_ECUDA,
                 std::string("pps_batch_create: ") + cudaGetErrorString(e));
  }
  *out = b;
  return PPS_OK;
}

int pps_batch_run(pps_batch* b, const pps_camera* cams, uint32_t frame, void* stream) {
  if (!b || !cams) return bfail(PPS_EINVAL, "NULL argument");
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != b->device)
    return bfail(PPS_EINVAL, "the batch's device is not the current device");
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  auto aim = [&](pps::KeyConst& kc, const pps_camera& cam) {
    kc.cam[0] = cam.pos[0];
    kc.cam[1] = cam.pos[1];
    kc.cam[2] = cam.pos[2];
    kc.frame = frame;
    pps::set_round_keys(kc);
  };
  cudaError_t e = cudaSuccess;
  if (!b->base.empty()) {
    const int k = static_cast<int>(b->runs & 1);
    // the buffer's previous upload must have completed before it is refilled
    if (b->runs >= 2) e = cudaEventSynchronize(b->done[k]);
    if (e == cudaSuccess) {
      for (size_t i = 0; i < b->base.size(); ++i) {
        pps::ViewDesc vd = b->base[i];
        vd.t = pps::table_dev(b->tables[i]);  // another call on the table may have moved its arrays
        aim(vd.kc, cams[b->index[i]]);
        b->hviews[k][i] = vd;
      }
      e = cudaGraphLaunch(b->exec[k], st);
    }
    if (e == cudaSuccess) e = cudaEventRecord(b->done[k], st);
  }
  for (size_t i = 0; i < b->own.size() && e == cudaSuccess; ++i) {
    const pps::ViewDesc& vd = b->own[i].vd;
    pps::KeyConst kc = vd.kc;
    aim(kc, cams[b->own[i].index]);
    e = pps::launch_fused(kc, pps::table_dev(b->own[i].table), vd.v, vd.n, vd.o, vd.blended != 0, b->alpha, b->own[i].plan, b->gstash,
                          nullptr, st);
  }
  if (e != cudaSuccess) return bfail(PPS_ECUDA, std::string("pps_batch_run: ") + cudaGetErrorString(e));
  ++b->runs;
  return PPS_OK;
}

int pps_batch_destroy(pps_batch* b) {
  if (!b) return PPS_OK;
  cudaDeviceSynchronize();
  release(b);
  delete b;
  return PPS_OK;
}

}  // extern "C"
