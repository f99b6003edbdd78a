// Culled shooting (the interactive zoom of Section 4: a sub-window of the source plane re-shot at
// higher resolution): rays are grouped in cells of 8 x 8; a cell is skipped when a rigorous bound
// shows that none of its rays can land in the window, and the others are shot with the same per-ray
// arithmetic as rs_shoot, so the counts and the out-of-window count equal those of rs_shoot.
//
// Bound for a cell with ray box centre c and circumradius rho (every ray x = c + h of the cell has |h| <= rho),
// lenses at distance d_i = |c - x_i| > rho.  In complex notation conj(alpha(z)) = f(z) = sum_i m_i / (z - z_i), and
// 1 / (w + h) = 1 / w - h / w^2 + h^2 / (w^2 (w + h)) with w = c - z_i gives
//   |f(c + h) - f(c) - f'(c) h| <= rho^2 sum_i m_i / (d_i^2 (d_i - rho)) = rho^2 B,    f'(c) = -sum_i m_i / w_i^2.
// So with q1 = sum_i m_i (dx^2 - dy^2) / d^4, q2 = sum_i 2 m_i dx dy / d^4 the cell's source positions are
//   y1 = lam1 c1 - alpha1(c) + (lam1 + q1) h1 + q2 h2 +- rho^2 B,   y2 = lam2 c2 - alpha2(c) + q2 h1 + (lam2 - q1) h2 +- rho^2 B,
// and sum_i m_i / |x - x_i| <= sum_i m_i / (d_i - rho) = S bounds the rounding of every ray of the cell.  A cell
// whose box misses the window on some axis is skipped and its rays are counted out of window.  A cell with a lens
// within 1.02 rho of c has no finite bound and is always shot.  The bound is applied to cells of 64 x 64 rays first,
// then to the 16 x 16 cells of the kept ones and to the 8 x 8 cells of those.
//
// x4 zoom of the 1e4-lens map, 4.12e6 rays in the window: 8.52e6 rays shot with cells of 16 x 16 and no linear term
// (|alpha(x) - alpha(c)| <= rho sum m / (d (d - rho))), 6.78e6 with it -- most of the rest in cells a few rho from a
// lens, whose area shrinks with the cell's -- hence the cells of 8 x 8: 5.08e6.
#include <algorithm>

#include "rs_internal.h"

namespace {

using namespace rsdev;

constexpr int kCell = 8;         // rays per side of the cells that are shot
constexpr int kMid = 16;         // of the second level
constexpr int kCoarse = 64;      // and of the first
constexpr int kCullBlock = 256;  // threads per CTA of the bound kernel
constexpr int kCullSmThreads = 512;  // threads per SM up to which a cell's sums are shared

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void fold(float& hi, float& lo, float p) {
  const float t = __fadd_rn(hi, p);
  const float bp = __fsub_rn(t, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bp)), __fsub_rn(p, bp)));
  hi = t;
}

// Threads that share a cell's sums (a power of two up to a warp): as many as keep all cells' threads within `threads`,
// so that a level of few cells still fills the chip, and leave each thread 64 lenses or more (each has the float64
// bound of its cell to work out as well).  With one thread per cell a level takes as long as one thread's walk over
// all lenses, however few its cells are: 30000 lenses, 500^2 rays 1.17 ms for each of the three levels, call 5.58 ->
// 2.53 ms; 64 lenses a thread against none at 60 lenses, 3600^2 rays 94 against 160 us.
__host__ __device__ __forceinline__ int cull_lanes(int64_t cells, int64_t threads, int n_lens) {
  int lanes = 1;
  while (lanes < 32 && cells * (2 * lanes) <= threads && n_lens >= 128 * lanes) lanes *= 2;
  return lanes;
}

__device__ __forceinline__ double sum_over_lanes(double v, int lanes) {
  for (int o = 1; o < lanes; o *= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// cull_lanes threads per cell: the bound sums over all lenses (tiles staged in shared memory), then
// the cell's source-plane box against the window.  Kept cells are appended to `out`; skipped cells add
// their rays to the out-of-window count.  The first level takes every cell of the call (parent == nullptr), the
// others the split x split cells of every kept cell of the level before.
// Three CTAs per SM, 80 registers: at the four that the compiler aims at the lens loop spills (x4 zoom of 1e4 lenses, a
// lower level: 1.17 ms, 0.85 so).
template <bool MASS>
__global__ void __launch_bounds__(kCullBlock, 3)
    cull_kernel(const ShootDesc d, int cell_rays, int64_t n_cx, int64_t n_cells, const unsigned* __restrict__ parent,
                const unsigned* __restrict__ parent_count, int64_t n_px, int split, int64_t threads, double hi0,
                double hi1, unsigned* __restrict__ out, unsigned* __restrict__ out_count, unsigned long long* __restrict__ n_shot) {
  __shared__ float4 s_lens[kCullBlock];
  __shared__ float s_mass[kCullBlock];
  const int64_t n_cy = (d.n_rows + cell_rays - 1) / cell_rays;
  const int children = split * split;
  if (parent != nullptr) n_cells = (int64_t)*parent_count * children;
  const int lanes = cull_lanes(n_cells, threads, d.f.n_lens);
  if ((int64_t)blockIdx.x * kCullBlock >= n_cells * lanes) return;  // CTA-uniform: no cells left
  const int64_t c = ((int64_t)blockIdx.x * kCullBlock + threadIdx.x) >> (__ffs(lanes) - 1);
  const int share = (int)threadIdx.x & (lanes - 1);  // the thread takes lenses share, share + lanes, ...
  int64_t cx, cy;
  bool ok = c < n_cells;
  if (parent != nullptr) {
    const int64_t p = parent[ok ? c / children : 0];
    const int sub = (int)(c % children);
    const int64_t py = p / n_px, px = p - py * n_px;
    cx = px * split + sub % split;
    cy = py * split + sub / split;
    ok = ok && cx < n_cx && cy < n_cy;
  } else {
    cy = c / n_cx;
    cx = c - cy * n_cx;
  }
  if (!ok) cx = cy = 0;
  const int64_t i0 = cx * cell_rays, i1 = min(i0 + cell_rays, d.n0) - 1;
  const int64_t r0 = cy * cell_rays, r1 = min(r0 + cell_rays, d.n_rows) - 1;
  const float xa1 = ray_coord(i0, d.sp0, d.or0), xb1 = ray_coord(i1, d.sp0, d.or0);
  const float xa2 = ray_coord(d.j_begin + r0, d.sp1, d.or1), xb2 = ray_coord(d.j_begin + r1, d.sp1, d.or1);
  const float c1 = 0.5f * (xa1 + xb1), c2 = 0.5f * (xa2 + xb2);
  const double h1 = fmax((double)c1 - (double)xa1, (double)xb1 - (double)c1);
  const double h2 = fmax((double)c2 - (double)xa2, (double)xb2 - (double)c2);
  const float rho = (float)(sqrt(h1 * h1 + h2 * h2) * (1.0 + 0x1p-20)) + 1e-30f;
  const float rho_gap = 0.02f * rho;  // d - rho <= 0.02 rho: no usable bound
  float a1h = 0.f, a1l = 0.f, a2h = 0.f, a2l = 0.f, bh = 0.f, bl = 0.f, sh = 0.f, sl = 0.f;
  float q1h = 0.f, q1l = 0.f, q2h = 0.f, q2l = 0.f;
  bool near = false;
  const int n = d.f.n_lens;
  for (int t0 = 0; t0 < n; t0 += kCullBlock) {
    __syncthreads();
    const int l = t0 + threadIdx.x;
    if (l < n) {
      s_lens[threadIdx.x] = d.f.lens4[l];
      if (MASS) s_mass[threadIdx.x] = d.f.mass2[l].x;
    }
    __syncthreads();
    const int cnt = min(kCullBlock, n - t0);
    for (int g = 0; g < cnt; g += 32 * lanes) {  // at most 32 terms of the thread
      float pa1 = 0.f, pa2 = 0.f, pb = 0.f, ps = 0.f, pq1 = 0.f, pq2 = 0.f;
      auto term = [&](int q) {
        const float4 L = s_lens[q];
        const float dx = c1 - L.x, dy = c2 - L.z;
        const float dy2 = dy * dy;
        const float d2 = fmaf(dx, dx, dy2);
        const float rs = rsqrt_approx(d2);
        const float gap = fmaf(d2, rs, -rho);  // d - rho
        near |= !(gap > rho_gap);  // NaN (a lens on the centre) counts as near
        const float r2 = rs * rs;
        float mi = r2, mg = rcp_approx(gap);
        if (MASS) {
          const float m = s_mass[q];
          mi *= m;
          mg *= m;
        }
        pa1 = fmaf(mi, dx, pa1);
        pa2 = fmaf(mi, dy, pa2);
        const float mq = mi * r2;
        pq1 = fmaf(mq, fmaf(dx, dx, -dy2), pq1);
        pq2 = fmaf(mq, dx * dy, pq2);
        ps += mg;
        pb = fmaf(mg, r2, pb);
      };
      if (lanes == 1 && g + 32 <= cnt) {
#pragma unroll 8
        for (int q = g; q < g + 32; ++q) term(q);
      } else {
        const int end = min(g + 32 * lanes, cnt);
#pragma unroll 4
        for (int q = g + share; q < end; q += lanes) term(q);
      }
      fold(a1h, a1l, pa1);
      fold(a2h, a2l, pa2);
      fold(q1h, q1l, pq1);
      fold(q2h, q2l, pq2);
      fold(bh, bl, pb);
      fold(sh, sl, ps);
    }
  }
  ok = ok && share == 0;  // one thread speaks for the cell
  const unsigned rays = ok ? (unsigned)((i1 - i0 + 1) * (r1 - r0 + 1)) : 0u;  // at most 64 x 64
  bool keep = true;
  near = sum_over_lanes(near ? 1.0 : 0.0, lanes) > 0.0;
  const double sum_s = sum_over_lanes((double)sh + (double)sl, lanes);
  const double sum_b = sum_over_lanes((double)bh + (double)bl, lanes);
  const double A1 = sum_over_lanes((double)a1h + (double)a1l, lanes);
  const double A2 = sum_over_lanes((double)a2h + (double)a2l, lanes);
  const double Q1 = sum_over_lanes((double)q1h + (double)q1l, lanes);
  const double Q2 = 2.0 * sum_over_lanes((double)q2h + (double)q2l, lanes);
  if (!near) {
    // terms carry a few 2^-22 relative (approximate reciprocal square root and reciprocal, the gap's
    // cancellation when d is near 1.02 rho: <= 2^-15), sums of 32 float terms ~2^-19 of their
    // absolute sum: inflate B and S by 2^-8
    const double S = sum_s * (1.0 + 0x1p-8);
    const double B = (double)rho * (double)rho * sum_b * (1.0 + 0x1p-8);
    // alpha(c) error <= ~2^-18.4 S, a ray's float32 error <= 72 u S = 2^-17.8 S, the linear term's error <= rho 2^-18
    // sum m / d^2 <= 2^-20 S per coefficient (rho (d - rho) <= d^2 / 4): together below 2^-16 S, taken twice; and
    // float64 roundings
    const double x1m = fmax(fabs((double)xa1), fabs((double)xb1)), x2m = fmax(fabs((double)xa2), fabs((double)xb2));
    const double M = B + 0x1p-15 * S +
                     0x1p-40 * (fabs(d.f.lam1) * x1m + fabs(d.f.lam2) * x2m + fabs(A1) + fabs(A2) + B + 1.0 +
                                fabs(d.lo0) + fabs(d.lo1) + fabs(hi0) + fabs(hi1));
    const double y1 = d.f.lam1 * (double)c1 - A1, y2 = d.f.lam2 * (double)c2 - A2;
    const double e1 = (fabs(d.f.lam1 + Q1) * h1 + fabs(Q2) * h2) * (1.0 + 0x1p-40) + M;
    const double e2 = (fabs(Q2) * h1 + fabs(d.f.lam2 - Q1) * h2) * (1.0 + 0x1p-40) + M;
    const bool finite = isfinite(e1) && isfinite(e2) && isfinite(A1) && isfinite(A2);
    keep = !finite || !(y1 + e1 < d.lo0 || y1 - e1 > hi0 || y2 + e2 < d.lo1 || y2 - e2 > hi1);
  }
  // one append and one count per warp: neighbouring cells stay together in the list
  const int lane = threadIdx.x & 31;
  const unsigned kept = __ballot_sync(0xffffffffu, ok && keep);
  const unsigned shot = __reduce_add_sync(0xffffffffu, keep ? rays : 0u);
  const unsigned missed = __reduce_add_sync(0xffffffffu, keep ? 0u : rays);
  unsigned slot = 0;
  if (lane == 0) {
    if (kept != 0u) slot = atomicAdd(out_count, (unsigned)__popc(kept));
    if (n_shot && shot != 0u) atomicAdd(n_shot, (unsigned long long)shot);
    if (d.oow && missed != 0u) atomicAdd(d.oow, (unsigned long long)missed);
  }
  slot = __shfl_sync(0xffffffffu, slot, 0);
  if (ok && keep) out[slot + (unsigned)__popc(kept & ((1u << lane) - 1u))] = (unsigned)(cy * n_cx + cx);
}

// Kept cells: a CTA of four warps shoots sixteen cells per pass; eight lanes share a cell, lane l of them holding
// its row l (eight columns).  The list holds cells of 8 x 8, or (n_mx > 0, cells per row) of 16 x 16, whose four
// children are then all shot.  The per-ray arithmetic is rs_shoot's (per-ray squared distances instead of the shared
// row table give bitwise the same values).
template <int MASS>
__global__ void __launch_bounds__(128, 2) shoot_cells_kernel(const ShootDesc d, int64_t n_cx, int64_t n_mx,
                                                             const unsigned* __restrict__ list,
                                                             const unsigned* __restrict__ n_kept) {
  constexpr int RPT = kCell, CELLS = 128 / kCell;
  __shared__ LensSmem<rsint::kTile, 1> sm;
  __shared__ NearSmem<rsint::kTile, CELLS, 128, RPT> ns;  // one near-lens box per cell
  PipeState ps;
  pipe_init(sm.bar, ps);
  constexpr unsigned CHILDREN = (kMid / kCell) * (kMid / kCell);
  const unsigned count = *n_kept * (n_mx > 0 ? CHILDREN : 1u);
  const int lane = threadIdx.x & 31, own = threadIdx.x / kCell, row = threadIdx.x % kCell;
  for (unsigned base = blockIdx.x * (unsigned)CELLS; base < count; base += gridDim.x * (unsigned)CELLS) {  // CTA-uniform
    const unsigned slot = base + (unsigned)own;
    bool cell_ok = slot < count;
    const unsigned at = cell_ok ? slot : count - 1;
    int64_t cx, cy;
    if (n_mx > 0) {
      const int64_t mid = (int64_t)list[at / CHILDREN];
      const int64_t my = mid / n_mx, mx = mid - my * n_mx;
      cx = mx * 2 + (at & 1u);
      cy = my * 2 + ((at >> 1) & 1u);
      if (cx >= n_cx || cy * kCell >= d.n_rows) {  // past the last column or row: no rays
        cell_ok = false;
        cx = mx * 2;
        cy = my * 2;
      }
    } else {
      const int64_t cell = (int64_t)list[at];
      cy = cell / n_cx;
      cx = cell - cy * n_cx;
    }
    const int64_t jrel = cy * kCell + row;
    const bool row_ok = cell_ok && jrel < d.n_rows;
    const int64_t j = d.j_begin + (jrel < d.n_rows ? jrel : d.n_rows - 1);
    const float x2r = ray_coord(j, d.sp1, d.or1);
    const int64_t i_base = cx * kCell;
    float x1[RPT], x2[RPT];
    bool valid[RPT];
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      int64_t i = i_base + k;
      valid[k] = row_ok && i < d.n0;
      if (i >= d.n0) i = d.n0 - 1;
      x1[k] = ray_coord(i, d.sp0, d.or0);
      x2[k] = x2r;
    }
    if (row == 0) {
      // the cell's ray box (coordinates grow with the grid index)
      const int64_t ia = cx * kCell, ib = min(ia + kCell, d.n0) - 1;
      const int64_t ja = cy * kCell, jb = min(ja + kCell, d.n_rows) - 1;
      near_set_box(ns, own, ray_coord(ia, d.sp0, d.or0), ray_coord(ib, d.sp0, d.or0),
                   ray_coord(d.j_begin + ja, d.sp1, d.or1), ray_coord(d.j_begin + jb, d.sp1, d.or1));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      float u0 = ns.box[0][0], u1 = ns.box[0][1], u2 = ns.box[0][2], u3 = ns.box[0][3];
      for (int c = 1; c < CELLS; ++c) {
        u0 = fminf(u0, ns.box[c][0]);
        u1 = fmaxf(u1, ns.box[c][1]);
        u2 = fminf(u2, ns.box[c][2]);
        u3 = fmaxf(u3, ns.box[c][3]);
      }
      ns.ubox[0] = u0;
      ns.ubox[1] = u1;
      ns.ubox[2] = u2;
      ns.ubox[3] = u3;
    }
    __syncthreads();  // every box is set before the first lens tile is searched
    float a1h[RPT], a1l[RPT], a2h[RPT], a2l[RPT], sig[RPT], tn[RPT];
    if (!deflect_pairs<RPT, rsint::kTile, MASS, false, 1>(d.f, x1, x2, a1h, a1l, a2h, a2l, sig, tn, sm, ps, &ns))
      return;
    bin_rays<RPT, RPT, 1>(d, x1, x2, a1h, a1l, a2h, a2l, sig, tn, valid, jrel, i_base, lane);
  }
}

}  // namespace

namespace rsint {

static int64_t cells_of(int64_t n_rows, int64_t n0, int side) {
  return ((n_rows + side - 1) / side) * ((n0 + side - 1) / side);
}
int64_t cull_cells(int64_t n_rows, int64_t n0) { return cells_of(n_rows, n0, kCell); }
int64_t cull_coarse_cells(int64_t n_rows, int64_t n0) { return cells_of(n_rows, n0, kCoarse); }
int64_t cull_mid_cells(int64_t n_rows, int64_t n0) { return cells_of(n_rows, n0, kMid); }

template <bool MASS>
static void launch_cull_m(const rsdev::ShootDesc& d, double hi0, double hi1, unsigned* coarse, unsigned* n_coarse,
                          unsigned* mid, unsigned* n_mid, unsigned* list, unsigned* n_kept, unsigned long long* n_shot,
                          int sms, cudaStream_t s) {
  const auto across = [&](int side) { return (d.n0 + side - 1) / side; };
  const int64_t threads = (int64_t)sms * kCullSmThreads;
  // CTAs of a level of `cells` cells at most; where few cells are left, their lanes fill up to `threads`
  const auto blocks = [&](int64_t cells) {
    const int64_t t = std::max(cells, std::min(cells * cull_lanes(1, threads, d.f.n_lens), threads));
    return (unsigned)((t + kCullBlock - 1) / kCullBlock);
  };
  const int64_t n1 = cull_coarse_cells(d.n_rows, d.n0);
  constexpr int S2 = kCoarse / kMid, S3 = kMid / kCell;
  // the lower levels are launched for all cells the level above could keep; CTAs beyond what it kept leave at once
  cull_kernel<MASS><<<blocks(n1), kCullBlock, 0, s>>>(d, kCoarse, across(kCoarse), n1, nullptr, nullptr, 0, 1, threads,
                                                      hi0, hi1, coarse, n_coarse, nullptr);
  cull_kernel<MASS><<<blocks(n1 * S2 * S2), kCullBlock, 0, s>>>(d, kMid, across(kMid), 0, coarse, n_coarse,
                                                                across(kCoarse), S2, threads, hi0, hi1, mid, n_mid,
                                                                list ? nullptr : n_shot);
  if (list == nullptr) return;
  cull_kernel<MASS><<<blocks(cull_mid_cells(d.n_rows, d.n0) * S3 * S3), kCullBlock, 0, s>>>(
      d, kCell, across(kCell), 0, mid, n_mid, across(kMid), S3, threads, hi0, hi1, list, n_kept, n_shot);
}

cudaError_t launch_cull(const rsdev::ShootDesc& d, double hi0, double hi1, unsigned* coarse, unsigned* n_coarse,
                        unsigned* mid, unsigned* n_mid, unsigned* list, unsigned* n_kept, unsigned long long* n_shot,
                        int sms, cudaStream_t s) {
  if (cull_coarse_cells(d.n_rows, d.n0) <= 0) return cudaSuccess;
  if (d.f.has_mass)
    launch_cull_m<true>(d, hi0, hi1, coarse, n_coarse, mid, n_mid, list, n_kept, n_shot, sms, s);
  else
    launch_cull_m<false>(d, hi0, hi1, coarse, n_coarse, mid, n_mid, list, n_kept, n_shot, sms, s);
  return cudaGetLastError();
}

cudaError_t launch_shoot_cells(const rsdev::ShootDesc& d, bool mid_cells, const unsigned* list, const unsigned* n_kept,
                               int grid, cudaStream_t s) {
  const int64_t n_cx = (d.n0 + kCell - 1) / kCell, n_mx = mid_cells ? (d.n0 + kMid - 1) / kMid : 0;
  if (d.f.has_mass == rsdev::kWideMass)
    shoot_cells_kernel<rsdev::kWideMass><<<grid, 128, 0, s>>>(d, n_cx, n_mx, list, n_kept);
  else if (d.f.has_mass)
    shoot_cells_kernel<rsdev::kMass><<<grid, 128, 0, s>>>(d, n_cx, n_mx, list, n_kept);
  else
    shoot_cells_kernel<rsdev::kUnitMass><<<grid, 128, 0, s>>>(d, n_cx, n_mx, list, n_kept);
  return cudaGetLastError();
}

}  // namespace rsint
