// Listed-ray traces (rs_trace): source positions, deflections and error bands of the float32 path, bit for bit
// what the shoot kernels compute for those rays.
//
// Two ways to the same bits:
//   * trace_kernel: a thread sums all lenses for its four rays.  512 rays a CTA, so it fills the chip only with
//     1e5 rays or more (4096 rays, 1e5 lenses, error bands: 23.2 ms, eight CTAs).
//   * the split path: the float32 partial sum of a 64-lens group depends on nothing but the ray and the group, so
//     all (ray, group) partials are formed independently (trace_part_kernel: one warp per 128 rays and group) into
//     a workspace, and only their fold into the two-float accumulators, a few additions per group, runs in lens
//     order (trace_fold_kernel: one lane per ray pair and sum).  Large fields run in chunks of groups, the
//     accumulators carried in the workspace.  The same 4096 rays: 0.30 ms, bound by the partials' FMA work (4.1e8
//     interactions) and by the serial fold where rays are few (10 rays, 1e6 lenses: 0.9 ms, was 79).
#include <algorithm>
#include <type_traits>

#include "rs_internal.h"

namespace {

using namespace rsdev;

// Outputs of ray r at (x1, x2): Eq. 6 in float64, and the band half-width from sig and the largest-term bound tn.
__device__ __forceinline__ void trace_store(const FieldDev& f, int64_t r, float x1, float x2, double a1, double a2,
                                            float sig, float tn, double* __restrict__ y, double* __restrict__ alpha,
                                            double* __restrict__ err) {
  y[2 * r] = __dsub_rn(__dmul_rn(f.lam1, (double)x1), a1);
  y[2 * r + 1] = __dsub_rn(__dmul_rn(f.lam2, (double)x2), a2);
  if (alpha != nullptr) {
    alpha[2 * r] = a1;
    alpha[2 * r + 1] = a2;
  }
  if (err != nullptr) {
    const double b = (double)band_halfwidth(sig, tn, f.lamabs, x1, x2);
    err[2 * r] = b;
    err[2 * r + 1] = b;
  }
}

template <int BLOCK, int RPT, int TILE, int MASS>
__global__ void __launch_bounds__(BLOCK)
    trace_kernel(const FieldDev f, double or0, double or1, double sp0, double sp1, const int64_t* __restrict__ ij,
                 int64_t k, double* __restrict__ y, double* __restrict__ alpha, double* __restrict__ err) {
  __shared__ LensSmem<TILE> sm;
  PipeState ps;
  pipe_init(sm.bar, ps);
  const int64_t base = (int64_t)blockIdx.x * (BLOCK * RPT);
  float x1[RPT], x2[RPT];
  bool valid[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    int64_t r = base + (int64_t)q * BLOCK + threadIdx.x;
    valid[q] = r < k;
    if (!valid[q]) r = k - 1;
    x1[q] = ray_coord(ij[2 * r], sp0, or0);
    x2[q] = ray_coord(ij[2 * r + 1], sp1, or1);
  }
  double a1[RPT], a2[RPT];
  float sig[RPT];
  if (!deflect<RPT, TILE, MASS, false, 1>(f, x1, x2, a1, a2, sig, sm, ps)) return;
#pragma unroll
  for (int q = 0; q < RPT; ++q) {
    if (!valid[q]) continue;
    const int64_t r = base + (int64_t)q * BLOCK + threadIdx.x;
    // the ray's largest-term bound over every lens: the value the shoot kernels reach through
    // their near-lens search
    const float tn = err != nullptr ? near_term_all<MASS>(f, x1[q], x2[q]) : 0.f;
    trace_store(f, r, x1[q], x2[q], a1[q], a2[q], sig[q], tn, y, alpha, err);
  }
}


// ---- split path --------------------------------------------------------------------------------

static_assert(kRenorm == 4 * kGroup, "the fold renormalises after every fourth group");
constexpr int kRb = 128;         // rays of a ray block: 32 lanes x 4 rays (two packed pairs)
constexpr int kPartTile = 256;   // lenses of a CTA of trace_part_kernel: four groups
constexpr int kStateWords = 6;   // per ray pair: H1, L1, H2, L2, SS, AB

// Workspace of a call of n_rb ray blocks, in this order (16-byte multiples): ray coordinates, the largest near
// term of each ray, the accumulators and the partials of one chunk of groups.
struct TraceWs {
  float2* xy;       // [n_rb][128]
  float* tmax;      // [n_rb][128]
  uint64_t* state;  // [n_rb][2 pairs][kStateWords][32 lanes]
  uint64_t* part;   // [groups of a chunk][n_rb][2 pairs][P1, P2][32 lanes]
};

size_t trace_fixed_bytes(int64_t n_rb) {
  return (size_t)n_rb * (kRb * (sizeof(float2) + sizeof(float)) + 2 * kStateWords * 32 * sizeof(uint64_t));
}
size_t trace_group_bytes(int64_t n_rb) { return (size_t)n_rb * 2 * 2 * 32 * sizeof(uint64_t); }

__global__ void trace_init_kernel(double or0, double or1, double sp0, double sp1, const int64_t* __restrict__ ij,
                                  int64_t k, int64_t n_pad, float2* __restrict__ xy, float* __restrict__ tmax) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_pad) return;
  const int64_t s = r < k ? r : k - 1;
  xy[r] = make_float2(ray_coord(ij[2 * s], sp0, or0), ray_coord(ij[2 * s + 1], sp1, or1));
  tmax[r] = 0.f;
}

// Partials of groups g0 + 4 blockIdx.x .. + 3 (at most ng of the chunk) for the ray blocks 4 blockIdx.y .. + 3.
// NEAR: also the largest near term of each ray; a warp looks at a group's near terms only when one of its
// rays came within h of a lens of the group.
template <int MASS, bool NEAR>
__global__ void __launch_bounds__(128)
    trace_part_kernel(const FieldDev f, int64_t n_rb, int g0, int ng, const float2* __restrict__ xy,
                      uint64_t* __restrict__ part, float* __restrict__ tmax) {
  __shared__ __align__(16) float4 s_lens[kPartTile];
  __shared__ __align__(16) float2 s_mass[kPartTile];
  const int gl0 = (int)blockIdx.x * (kPartTile / kGroup);  // the CTA's first group of the chunk
  const int l0 = (g0 + gl0) * kGroup;
  const int cnt = min(min(kPartTile, (ng - gl0) * kGroup), f.n_lens - l0);
  for (int l = threadIdx.x; l < cnt; l += 128) {
    s_lens[l] = __ldg(f.lens4 + l0 + l);
    if (MASS != kUnitMass) s_mass[l] = __ldg(f.mass2 + l0 + l);
  }
  __syncthreads();
  const uint32_t lbase = smem_u32(s_lens), mbase = smem_u32(s_mass);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t rb0 = (int64_t)blockIdx.y * 4;
  const int nrb = (int)min((int64_t)4, n_rb - rb0);
  const int tasks = nrb * ((cnt + kGroup - 1) / kGroup);
  for (int t = warp; t < tasks; t += 4) {
    const int64_t rb = rb0 + t % nrb;
    const int g = t / nrb;
    float x1[4], x2[4], mn[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 p = __ldg(xy + rb * kRb + lane + 32 * k);
      x1[k] = p.x;
      x2[k] = p.y;
      mn[k] = __int_as_float(0x7f800000);
    }
    uint64_t X1[2], X2[2], P1[2] = {0ull, 0ull}, P2[2] = {0ull, 0ull};
    pack_rays<4>(x1, x2, X1, X2);
    const int gc = min(kGroup, cnt - g * kGroup);
    using TR = std::conditional_t<NEAR, MinTrack, NoTrack>;
    TR tr{};
    if constexpr (NEAR) tr.r2 = mn;
    if (gc == kGroup) {
#pragma unroll
      for (int p4 = 0; p4 < kGroup / 8; ++p4)
        lens_block<4, kPartTile, MASS, false>(lbase, 0u, mbase, 0u, g * kGroup + p4 * 8, X1, X2, P1, P2, tr);
    } else {
      lens_group_partial<4, kPartTile, MASS, false>(lbase, 0u, mbase, 0u, g * kGroup, gc, X1, X2, P1, P2, tr);
    }
    uint64_t* o = part + ((size_t)(gl0 + g) * n_rb + rb) * 128 + lane;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      o[q * 64] = P1[q];
      o[q * 64 + 32] = P2[q];
    }
    if constexpr (NEAR) {
      const bool near = mn[0] <= kNearH2 || mn[1] <= kNearH2 || mn[2] <= kNearH2 || mn[3] <= kNearH2;
      if (__any_sync(0xffffffffu, near)) {
        float tn[4] = {0.f, 0.f, 0.f, 0.f};
        for (int l = g * kGroup; l < g * kGroup + gc; ++l) {
          const float4 L = s_lens[l];
          const float m = MASS != kUnitMass ? s_mass[l].x : 1.f;
#pragma unroll
          for (int k = 0; k < 4; ++k) tn[k] = fmaxf(tn[k], near_term(x1[k], x2[k], L.x, L.z, m));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)  // non-negative floats order as their bits
          if (tn[k] > 0.f) atomicMax(reinterpret_cast<int*>(tmax + rb * kRb + lane + 32 * k), __float_as_int(tn[k]));
      }
    }
  }
}

// Folds the ng groups of a chunk (first: group g0 of the field) into the accumulators of ray pair (block, q) =
// blockIdx.x: warp 0 the first axis, warp 1 the second, warp 2 the band sums.  Serial in the groups, so bound by
// latency: a ring in shared memory keeps 64 groups in flight ahead of the fold.  The last chunk ends in the outputs.
__global__ void __launch_bounds__(96)
    trace_fold_kernel(const FieldDev f, int64_t n_rb, int g0, int ng, const uint64_t* __restrict__ part,
                      uint64_t* __restrict__ state, int last, const float2* __restrict__ xy,
                      const float* __restrict__ tmax, int64_t k, double* __restrict__ y, double* __restrict__ alpha,
                      double* __restrict__ err) {
  constexpr int AHEAD = 16;   // groups of a stage: a multiple of the renormalisation period (four groups)
  constexpr int STAGES = 5;   // stages of the ring, all but one in flight
  __shared__ __align__(16) uint64_t ring[STAGES][AHEAD][64];  // [group][P1 of 32 lanes, P2 of 32 lanes]
  __shared__ uint64_t s_acc[kStateWords][32];
  const int role = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t rb = (int64_t)blockIdx.x >> 1;
  const int q = (int)(blockIdx.x & 1);
  uint64_t* st = state + (size_t)blockIdx.x * kStateWords * 32 + role * 64 + lane;
  uint64_t a = 0ull, b = 0ull;  // H and L of the axis, or SS and AB
  if (g0 > 0) {
    a = st[0];
    b = st[32];
  }
  const uint64_t* p = part + (size_t)rb * 128 + q * 64;
  const size_t step = (size_t)n_rb * 128;
  const int whole = min(ng, f.n_lens / kGroup - g0);  // whole groups of the chunk: renormalised as in the shoot
  auto fetch = [&](int stage) {
    for (int i = threadIdx.x; i < AHEAD * 32; i += 96) {  // 16-byte pieces, 32 a group
      const int g = stage * AHEAD + i / 32;
      if (g < ng)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         smem_u32(&ring[stage % STAGES][i / 32][2 * (i % 32)])),
                     "l"(p + (size_t)g * step + 2 * (i % 32))
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int t = 0; t < STAGES - 1; ++t) fetch(t);
  for (int t = 0; t * AHEAD < ng; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();        // stage t has arrived, and every warp is done with stage t - 1
    fetch(t + STAGES - 1);  // into the slot of stage t - 1
    const uint64_t(*u)[64] = ring[t % STAGES];
    const int g = t * AHEAD;
    auto band = [&](int j) {
      const uint64_t p1 = u[j][lane], p2 = u[j][32 + lane];
      a = f2_fma(p1, p1, a);
      a = f2_fma(p2, p2, a);
      b = f2_add_x(b, f2_add_x(f2_abs(p1), f2_abs(p2)));
    };
    auto axis = [&](int j, bool renorm) {
      twosum_accumulate(a, b, u[j][role * 32 + lane]);
      if (renorm) renormalise(a, b);
    };
    // a whole stage has no branch between its groups, so that their additions overlap
    if (g + AHEAD > whole) {
      for (int j = 0; j < AHEAD && g + j < ng; ++j)
        if (role == 2)
          band(j);
        else
          axis(j, (j & 3) == 3 && g + j < whole);
    } else if (role == 2) {
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) band(j);
    } else {
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) axis(j, (j & 3) == 3);
    }
  }
  if (!last) {
    st[0] = a;
    st[32] = b;
    return;
  }
  s_acc[2 * role][lane] = a;
  s_acc[2 * role + 1][lane] = b;
  __syncthreads();
  if (role != 0) return;
  DeflectAcc<1> acc;
  acc.H1[0] = s_acc[0][lane];
  acc.L1[0] = s_acc[1][lane];
  acc.H2[0] = s_acc[2][lane];
  acc.L2[0] = s_acc[3][lane];
  acc.SS[0] = s_acc[4][lane];
  acc.AB[0] = s_acc[5][lane];
  float a1h[2], a1l[2], a2h[2], a2l[2], sig[2];
  deflect_finish<2>(acc, a1h, a1l, a2h, a2l, sig);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int64_t r = rb * kRb + lane + 32 * (2 * q + h);
    if (r >= k) continue;
    const float2 x = xy[r];
    trace_store(f, r, x.x, x.y, (double)a1h[h] + (double)a1l[h], (double)a2h[h] + (double)a2l[h], sig[h],
                err != nullptr ? fmaxf(f.mcap, tmax[r]) : 0.f, y, alpha, err);
  }
}

template <int MASS, bool NEAR>
void launch_part(const FieldDev& f, int64_t n_rb, int g0, int ng, const TraceWs& w, cudaStream_t s) {
  const dim3 grid((unsigned)((ng + kPartTile / kGroup - 1) / (kPartTile / kGroup)), (unsigned)((n_rb + 3) / 4));
  trace_part_kernel<MASS, NEAR><<<grid, 128, 0, s>>>(f, n_rb, g0, ng, w.xy, w.part, w.tmax);
}

}  // namespace

namespace rsint {

cudaError_t launch_trace(const rsdev::FieldDev& f, double or0, double or1, double sp0, double sp1,
                         const int64_t* ij, int64_t k, double* y, double* alpha, double* err, cudaStream_t s) {
  constexpr int B = 128, R = 4;
  if (k <= 0) return cudaSuccess;
  const int64_t grid = (k + B * R - 1) / (B * R);
  if (f.has_mass == rsdev::kWideMass)
    trace_kernel<B, R, kTile, rsdev::kWideMass>
        <<<(unsigned)grid, B, 0, s>>>(f, or0, or1, sp0, sp1, ij, k, y, alpha, err);
  else if (f.has_mass)
    trace_kernel<B, R, kTile, rsdev::kMass><<<(unsigned)grid, B, 0, s>>>(f, or0, or1, sp0, sp1, ij, k, y, alpha, err);
  else
    trace_kernel<B, R, kTile, rsdev::kUnitMass><<<(unsigned)grid, B, 0, s>>>(f, or0, or1, sp0, sp1, ij, k, y, alpha, err);
  return cudaGetLastError();
}

// Groups of a chunk: as many whole tiles as the workspace bound leaves room for.
int64_t trace_chunk_groups(int64_t n_rb, int64_t n_groups) {
  const int64_t fit = (int64_t)(kTraceSplitBytes / trace_group_bytes(n_rb));
  constexpr int64_t kTileGroups = kPartTile / kGroup;
  return std::min((n_groups + kTileGroups - 1) / kTileGroups * kTileGroups,
                  std::max(kTileGroups, fit / kTileGroups * kTileGroups));
}

size_t trace_split_bytes(int n_lens, int64_t k) {
  const int64_t n_rb = (std::min(k, kTraceSplitRays) + kRb - 1) / kRb;
  const int64_t n_groups = ((int64_t)n_lens + kGroup - 1) / kGroup;
  return trace_fixed_bytes(n_rb) + (size_t)trace_chunk_groups(n_rb, n_groups) * trace_group_bytes(n_rb);
}

// At most kTraceSplitRays rays.
static void trace_split_block(const rsdev::FieldDev& f, double or0, double or1, double sp0, double sp1,
                              const int64_t* ij, int64_t k, double* y, double* alpha, double* err, void* ws,
                              cudaStream_t s) {
  const int64_t n_rb = (k + kRb - 1) / kRb, n_groups = ((int64_t)f.n_lens + kGroup - 1) / kGroup;
  const int64_t chunk = trace_chunk_groups(n_rb, n_groups);
  TraceWs w;
  char* b = reinterpret_cast<char*>(ws);
  w.xy = reinterpret_cast<float2*>(b);
  w.tmax = reinterpret_cast<float*>(w.xy + n_rb * kRb);
  w.state = reinterpret_cast<uint64_t*>(w.tmax + n_rb * kRb);
  w.part = w.state + n_rb * 2 * kStateWords * 32;
  trace_init_kernel<<<(unsigned)n_rb, kRb, 0, s>>>(or0, or1, sp0, sp1, ij, k, n_rb * kRb, w.xy, w.tmax);
  for (int64_t g0 = 0; g0 < n_groups; g0 += chunk) {
    const int ng = (int)std::min(chunk, n_groups - g0);
    const bool near = err != nullptr;
    if (f.has_mass == rsdev::kWideMass)
      near ? launch_part<kWideMass, true>(f, n_rb, (int)g0, ng, w, s)
           : launch_part<kWideMass, false>(f, n_rb, (int)g0, ng, w, s);
    else if (f.has_mass)
      near ? launch_part<kMass, true>(f, n_rb, (int)g0, ng, w, s) : launch_part<kMass, false>(f, n_rb, (int)g0, ng, w, s);
    else
      near ? launch_part<kUnitMass, true>(f, n_rb, (int)g0, ng, w, s)
           : launch_part<kUnitMass, false>(f, n_rb, (int)g0, ng, w, s);
    trace_fold_kernel<<<(unsigned)(2 * n_rb), 96, 0, s>>>(f, n_rb, (int)g0, ng, w.part, w.state,
                                                          g0 + chunk >= n_groups ? 1 : 0, w.xy, w.tmax, k, y, alpha,
                                                          err);
  }
}

cudaError_t launch_trace_split(const rsdev::FieldDev& f, double or0, double or1, double sp0, double sp1,
                               const int64_t* ij, int64_t k, double* y, double* alpha, double* err, void* ws,
                               cudaStream_t s) {
  // blocks of rays, one after the other through the same workspace
  for (int64_t r = 0; r < k; r += kTraceSplitRays)
    trace_split_block(f, or0, or1, sp0, sp1, ij + 2 * r, std::min(kTraceSplitRays, k - r), y + 2 * r,
                      alpha ? alpha + 2 * r : nullptr, err ? err + 2 * r : nullptr, ws, s);
  return cudaGetLastError();
}

}  // namespace rsint
