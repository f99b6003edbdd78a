// C-ABI layer, batches (Section 4's many maps): the LPT-ordered work plan of many fields and its
// CUDA graph (memsets, persistent kernels per launch shape and mass mode, float-float re-evaluation).
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "rs_host.h"

using rsdev::FieldDev;
using rsdev::ShootDesc;
using namespace rshost;

struct rs_batch {
  int device;
  int n_fields;
  // work items grouped by (launch shape, mass mode): one persistent kernel per group; group
  // g = kMassModes * cfg + mass (rsdev::MassMode)
  static constexpr int kMassModes = 3;
  static constexpr int kGroups = kMassModes * rsint::kNumCfg;
  int n_items[kGroups];
  int item_offset[kGroups];
  int grid[kGroups];
  ShootDesc* d_descs;
  int2* d_items;
  int* d_counter;
  uint2* d_rc_list;
  unsigned int* d_rc_count;
  unsigned int rc_cap;
  cudaGraph_t graph;
  cudaGraphExec_t exec;
};

namespace {

// Per-ray cost of a field: one interaction per lens plus a fixed epilogue of about so many interactions.
constexpr double kEpilogue = 64.0;
double item_lenses(const rs_field* f) { return (double)f->n_lens + kEpilogue; }

}  // namespace

extern "C" {

// ------------------------------------------------------------------------------------------------ batch

int rs_batch_create_shaped(int n_fields, const rs_field_t* fields, const rs_ray_grid* grids, const rs_window* windows,
                           uint32_t* const* d_counts, uint64_t* d_out_of_window, const int* shapes, rs_batch_t* out) {
  if (!out) return fail(RS_EINVAL, "out is NULL");
  *out = nullptr;
  if (n_fields <= 0) return fail(RS_EINVAL, "n_fields must be >= 1");
  if (!fields || !grids || !windows || !d_counts) return fail(RS_EINVAL, "NULL array argument");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  int rc;
  std::vector<ShootDesc> descs(n_fields);
  struct Item {
    double cost;
    int field;
    int tile;
  };
  constexpr int G = rs_batch::kGroups;
  std::vector<Item> items[G];
  int64_t n_total = 0;
  double work = 0.0, work_lenses = 0.0, most = 0.0;  // in interactions: all fields, times their lenses, the largest
  int64_t most_n0 = 1;
  for (int k = 0; k < n_fields; ++k) {
    if (!fields[k]) return fail(RS_EINVAL, "fields[%d] is NULL", k);
    if (fields[k]->device != dev) return fail(RS_EINVAL, "fields[%d] lives on another device", k);
    if ((rc = check_grid(&grids[k])) != RS_OK) return rc;
    if ((rc = check_window(&windows[k])) != RS_OK) return rc;
    if (!d_counts[k]) return fail(RS_EINVAL, "d_counts[%d] is NULL", k);
    if ((rc = fill_desc(fields[k], &grids[k], 0, grids[k].n[1], &windows[k], d_counts[k],
                        d_out_of_window ? d_out_of_window + k : nullptr, &descs[k])) != RS_OK)
      return rc;
    const double w = (double)descs[k].n_rows * (double)descs[k].n0 * item_lenses(fields[k]);
    work += w;
    work_lenses += w * (double)fields[k]->n_lens;
    if (w > most) {
      most = w;
      most_n0 = descs[k].n0;
    }
  }
  // without shapes of the caller's: the shape of a plain call of as many rays through a field as make the whole
  // batch's work, since the fields share the SMs.  Two fields of 1000 lenses x 200^2 rays: 73 us by lens count alone, 61
  // so.  Batches of less than kOneShape large CTAs per SM take one shape for all fields of a mass mode, by their mean
  // lens count: a second group's CTAs wait for the first one's.  One shape / a shape per field, us, uneven fields of so
  // many large CTAs per SM: 8.4 487 / 538, 15 (masses) 1314 / 1382, 17 591 / 552, 25 2769 / 2770, 36 1214 / 1212.
  constexpr double kOneShape = 16.0;
  const double mean_lenses = work > 0.0 ? work_lenses / work : 0.0;
  const double mean_rays = work / (mean_lenses + kEpilogue);
  const bool one_shape = mean_rays < kOneShape * 1024.0 * num_sms(dev);
  for (int k = 0; k < n_fields; ++k) {
    const int64_t n0 = descs[k].n0, nr = descs[k].n_rows;
    const int mass = fields[k]->dev.has_mass;
    int cfg = rsint::kDefaultCfg;
    if (!shapes && n0 > 0) {
      const double lenses = one_shape ? mean_lenses : (double)fields[k]->n_lens;
      const int64_t row = one_shape ? most_n0 : n0;
      const double rows = std::ceil(work / (lenses + kEpilogue) / (double)row);
      cfg = pick_cfg(fields[k], lenses, (int64_t)std::min(rows, 0x1p40), row, true);
    }
    if (shapes) {
      const int* sh = shapes + 4 * k;
      cfg = rsint::find_cfg(sh[0], sh[1], sh[2], sh[3]);
      if (cfg < 0)
        return fail(RS_EINVAL, "shapes[%d] = (%d, %d, %d, %d) is not a compiled launch shape", k, sh[0], sh[1], sh[2],
                    sh[3]);
    }
    if (mass == rsdev::kWideMass) cfg = rsint::kDefaultCfg;
    const int grp = rs_batch::kMassModes * cfg + mass;
    const int warps = rsint::kCfgs[cfg].block / 32;
    const int64_t seg = 32 * (int64_t)rsint::kCfgs[cfg].rpt;
    if (n0 == 0 || nr == 0) continue;
    const int64_t ncol = (n0 + seg - 1) / seg;
    const int64_t nt = ((nr + warps - 1) / warps) * ncol;
    if (n_total + nt >= ((int64_t)1 << 31)) return fail(RS_EOVERFLOW, "too many work items");
    n_total += nt;
    for (int64_t t = 0; t < nt; ++t) {
      const int64_t trow = t / ncol, tcol = t - trow * ncol;
      const int64_t rows = std::min<int64_t>(warps, nr - trow * warps);
      const int64_t cols = std::min<int64_t>(seg, n0 - tcol * seg);
      const double cost = (double)(rows * cols) * item_lenses(fields[k]);
      items[grp].push_back({cost, k, (int)t});
    }
  }
  std::vector<int2> h_items;
  rs_batch* b = new (std::nothrow) rs_batch();
  if (!b) return fail(RS_ENOMEM, "host allocation failed");
  b->device = dev;
  b->n_fields = n_fields;
  for (int grp = 0; grp < G; ++grp) {
    std::stable_sort(items[grp].begin(), items[grp].end(),
                     [](const Item& x, const Item& y) { return x.cost > y.cost; });
    b->item_offset[grp] = (int)h_items.size();
    b->n_items[grp] = (int)items[grp].size();
    for (const Item& it : items[grp]) h_items.push_back(make_int2(it.field, it.tile));
    b->grid[grp] = 0;
    if (b->n_items[grp] == 0) continue;
    int bps = 0;
    if (rsint::batch_blocks_per_sm(grp / rs_batch::kMassModes, grp % rs_batch::kMassModes, &bps) != cudaSuccess || bps < 1) bps = 1;
    // no more CTAs than items: the block scheduler spreads them over the SMs, where idle CTAs of one SM would race
    // for two or three items each (one field of 3000 lenses x 300^2 rays, 150 items for 456 CTAs: 299 us with all of
    // them, 153 so)
    b->grid[grp] = std::min(num_sms(dev) * bps, b->n_items[grp]);
  }
  auto cleanup = [&]() {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    cudaFree(b->d_descs);
    cudaFree(b->d_items);
    cudaFree(b->d_counter);
    cudaFree(b->d_rc_list);
    cudaFree(b->d_rc_count);
    delete b;
  };
  if (g_certify) {
    int64_t total = 0;
    for (int k = 0; k < n_fields; ++k) total += descs[k].n_rows * descs[k].n0;
    b->rc_cap = rsint::recheck_capacity(total);
  }
  if ((e = dev_alloc(&b->d_descs, sizeof(ShootDesc) * n_fields)) != cudaSuccess ||
      (e = dev_alloc(&b->d_items, sizeof(int2) * std::max<size_t>(1, h_items.size()))) != cudaSuccess ||
      (e = dev_alloc(&b->d_counter, G * sizeof(int))) != cudaSuccess ||
      (b->rc_cap > 0 && (e = dev_alloc(&b->d_rc_list, sizeof(uint2) * (size_t)b->rc_cap)) != cudaSuccess) ||
      (b->rc_cap > 0 && (e = dev_alloc(&b->d_rc_count, sizeof(unsigned int))) != cudaSuccess)) {
    rc = cuda_fail(e, "cudaMalloc (batch)");
    cleanup();
    return rc;
  }
  for (int k = 0; k < n_fields; ++k) {
    descs[k].field_id = k;
    descs[k].rc_list = b->d_rc_list;
    descs[k].rc_count = b->d_rc_count;
    descs[k].rc_cap = b->rc_cap;
  }
  if ((e = cudaMemcpy(b->d_descs, descs.data(), sizeof(ShootDesc) * n_fields, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (!h_items.empty() &&
       (e = cudaMemcpy(b->d_items, h_items.data(), sizeof(int2) * h_items.size(), cudaMemcpyHostToDevice)) != cudaSuccess)) {
    rc = cuda_fail(e, "cudaMemcpy (batch descriptors)");
    cleanup();
    return rc;
  }
  // Capture: zero every map and counter, then the persistent kernel.
  cudaStream_t cs;
  if ((e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking)) != cudaSuccess) {
    rc = cuda_fail(e, "cudaStreamCreate");
    cleanup();
    return rc;
  }
  e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    for (int k = 0; k < n_fields && e == cudaSuccess; ++k)
      e = cudaMemsetAsync(d_counts[k], 0, sizeof(uint32_t) * (size_t)windows[k].npix[0] * (size_t)windows[k].npix[1], cs);
    if (e == cudaSuccess && d_out_of_window) e = cudaMemsetAsync(d_out_of_window, 0, sizeof(uint64_t) * n_fields, cs);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->d_counter, 0, G * sizeof(int), cs);
    if (e == cudaSuccess && b->rc_cap > 0) e = cudaMemsetAsync(b->d_rc_count, 0, sizeof(unsigned int), cs);
    // groups in decreasing order of their largest item (each group's items are already LPT-ordered)
    std::vector<int> order;
    for (int grp = 0; grp < G; ++grp)
      if (b->n_items[grp] > 0) order.push_back(grp);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return items[x][0].cost > items[y][0].cost; });
    // the groups are independent: one branch of the graph each, so that a group's CTAs start where another
    // group's last ones leave SMs idle
    std::vector<cudaStream_t> side(order.size(), nullptr);
    std::vector<cudaEvent_t> done(order.size(), nullptr);
    cudaEvent_t fork = nullptr;
    if (e == cudaSuccess && order.size() > 1) {
      e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
      if (e == cudaSuccess) e = cudaEventRecord(fork, cs);
    }
    for (size_t i = 0; i < order.size() && e == cudaSuccess; ++i) {
      const int grp = order[i];
      cudaStream_t bs = cs;
      if (i > 0) {
        e = cudaStreamCreateWithFlags(&side[i], cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done[i], cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(side[i], fork, 0);
        bs = side[i];
      }
      if (e == cudaSuccess)
        e = rsint::launch_batch(grp / rs_batch::kMassModes, grp % rs_batch::kMassModes, b->d_descs,
                                b->d_items + b->item_offset[grp], b->n_items[grp], b->d_counter + grp, b->grid[grp],
                                bs);
      if (e == cudaSuccess && i > 0) e = cudaEventRecord(done[i], bs);
    }
    for (size_t i = 1; i < order.size() && e == cudaSuccess; ++i) e = cudaStreamWaitEvent(cs, done[i], 0);
    if (e == cudaSuccess && b->rc_cap > 0)
      e = rsint::launch_recheck(nullptr, b->d_descs, b->d_rc_list, b->d_rc_count, b->rc_cap, recheck_grid(dev), cs);
    cudaError_t e2 = cudaStreamEndCapture(cs, &b->graph);
    if (e == cudaSuccess) e = e2;
    for (size_t i = 1; i < order.size(); ++i) {
      if (done[i]) cudaEventDestroy(done[i]);
      if (side[i]) cudaStreamDestroy(side[i]);
    }
    if (fork) cudaEventDestroy(fork);
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
  cudaStreamDestroy(cs);
  if (e != cudaSuccess) {
    rc = cuda_fail(e, "batch graph capture");
    cleanup();
    return rc;
  }
  *out = b;
  return RS_OK;
}

int rs_batch_create(int n_fields, const rs_field_t* fields, const rs_ray_grid* grids, const rs_window* windows,
                    uint32_t* const* d_counts, uint64_t* d_out_of_window, rs_batch_t* out) {
  return rs_batch_create_shaped(n_fields, fields, grids, windows, d_counts, d_out_of_window, nullptr, out);
}

int rs_batch_launch(rs_batch_t b, void* stream) {
  if (!b) return fail(RS_EINVAL, "batch is NULL");
  int cur = -1;
  cudaGetDevice(&cur);
  if (cur != b->device) return fail(RS_EINVAL, "batch lives on device %d but device %d is current", b->device, cur);
  cudaError_t e = cudaGraphLaunch(b->exec, reinterpret_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
  return RS_OK;
}

int rs_batch_destroy(rs_batch_t b) {
  if (!b) return RS_OK;
  DeviceGuard g(b->device);
  cudaDeviceSynchronize();
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  cudaFree(b->d_descs);
  cudaFree(b->d_items);
  cudaFree(b->d_counter);
  cudaFree(b->d_rc_list);
  cudaFree(b->d_rc_count);
  delete b;
  return RS_OK;
}

int rs_shoot_batch(int n_fields, const rs_field_t* fields, const rs_ray_grid* grids, const rs_window* windows,
                   uint32_t* const* d_counts, uint64_t* d_out_of_window, void* stream) {
  rs_batch_t b = nullptr;
  int rc = rs_batch_create(n_fields, fields, grids, windows, d_counts, d_out_of_window, &b);
  if (rc != RS_OK) return rc;
  rc = rs_batch_launch(b, stream);
  cudaError_t e = cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(stream));
  rs_batch_destroy(b);
  if (rc != RS_OK) return rc;
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize (batch)");
  return RS_OK;
}

}  // extern "C"
