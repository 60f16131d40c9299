// CUDA kernels of the DPD fluid step for sm_103a.
//
// One step, every stage a kernel over the packed particle slots (the force
// kernels are in force.cu):
//   1. integrate_bin  kick (completing the previous step), kick, drift, wrap
//                     (Sec. 3.1 item 5, Eq. 1); cell (x slice) of the new
//                     position and its arrival rank by an atomic count
//                     (Sec. 3.2); with the full stencil the previous step's
//                     force kernel can do this instead (fused);
//   2. scan           exclusive scan of the cell counts into cell starts
//                     (one pass for one tile, two up to 2048 tiles, else three:
//                     tile sums, scan of the tile sums, apply);
//   3. bin_keys       full stencil: record each slot's old index at its
//                     arrival position;
//   4. bin_scatter    move position and velocity to the new slot: full
//                     stencil ranked by old index inside the cell (a stable
//                     counting sort), half stencil by arrival rank;
//   5. force          pair forces of Eqs. 2-5 over the 27 neighbouring cells
//                     (full stencil) or 13 cells + own cell with Newton's third
//                     law (half stencil, Sec. 3.2), plus the body force.
// All arithmetic is FP32; statistics sum in FP64 above each thread.
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

#include "dpd_device.cuh"
#include "kernels.h"

namespace dpd {

constexpr int kBinThreads = 256;
static inline int blocks_for(long long n, int t) { return (int)((n + t - 1) / t); }
constexpr float kSqrt3Scale = (float)(1.7320508075688772 / 16777216.0);  // sqrt(3) 2^-24


// ------------------------------------------------------------------ load
__global__ void k_load(Packed P, int slot0, int n, const float *__restrict__ pos3,
                       const float *__restrict__ vel3, float Lx, float Ly, float Lz,
                       const int32_t *__restrict__ species, int nspec) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  load_particle(P, i, pos3, vel3, Lx, Ly, Lz, species, nspec, P.pos[slot0 + i], P.vel[slot0 + i]);
}

// ------------------------------------------------------- integrate + count
template <bool SINGLE>
__global__ void __launch_bounds__(kBinThreads) k_integrate_bin(Packed P, bool move) {
  step_begin();
  const int p = blockIdx.x * kBinThreads + threadIdx.x;
  int b = 0;
  if constexpr (!SINGLE) b = find_box_warp(P.pbase, P.nbox, min(p, P.ntot - 1));
  if (p >= P.ntot) return;
  const BoxDev B = box_of<SINGLE>(P, b);
  const bool mv = move && P.st[b].remaining > 0;
  const float4 f = mv ? P.frc[p] : make_float4(0.f, 0.f, 0.f, 0.f);
  // a stopped box (a step with nothing left to take) keeps its slots and forces
  integrate_one(P, B, p, P.pos[p], P.vel[p], f.x, f.y, f.z, mv, P.st[b].pending != 0,
                move && !mv);
}

// Row a1 of the half stencil's larger sets, split so that the reorder finishes
// it: this kernel kicks the velocities and clears the forces where they are,
// and counts the cells of the new positions without storing these; the
// reorder (k_drift_scatter) drifts the old position again with the stored
// velocity, the same operations and so the same bits, and writes to the other
// pair of position and velocity arrays.  Both kernels are bound by HBM: a
// step moves 152 B a particle (48 + 36 here, 36 + 32 there) in place of the 176
// of k_integrate_bin and k_bin_scatter.
template <bool SINGLE>
__global__ void __launch_bounds__(kBinThreads) k_kick_bin(Packed P) {
  const int p = blockIdx.x * kBinThreads + threadIdx.x;
  int b = 0;
  if constexpr (!SINGLE) b = find_box_warp(P.pbase, P.nbox, min(p, P.ntot - 1));
  if (p >= P.ntot) return;
  const BoxDev B = box_of<SINGLE>(P, b);
  const bool mv = P.st[b].remaining > 0;  // a stopped box keeps its slots and forces
  float4 x = P.pos[p], v = P.vel[p];
  if (mv) {
    const float4 f = P.frc[p];
    kick(B, v, f.x, f.y, f.z, P.st[b].pending != 0);
    drift(P, B, x, v);
  }
  const int cx = cell_axis(x.x, B.invh[0], B.n[0]);
  const int cy = cell_axis(x.y, B.invh[1], B.n[1]);
  const int cz = cell_axis(x.z, B.invh[2], B.n[2]);
  const int c = B.cellBase + (cz * B.n[1] + cy) * B.n[0] + cx;
  if (mv) {
    v.w = __int_as_float(pack_cell(cx, cy, cz));
    P.vel[p] = v;
    P.frc[p] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (!DPD_IN_BOUNDS(c >= 0 && c < P.ncell, P.err)) return;
  P.slotIn[p] = atomicAdd(P.count + c, 1);
}

// ------------------------------------------------------------------ scan
__device__ __forceinline__ int warp_incl_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Exclusive block scan of one value per thread; returns the block total in *total.
template <int NT>
__device__ __forceinline__ int block_excl_scan(int v, int *total) {
  __shared__ int wsum[NT / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int incl = warp_incl_scan(v);
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int s = (lane < NT / 32) ? wsum[lane] : 0;
    s = warp_incl_scan(s);
    if (lane < NT / 32) wsum[lane] = s;
  }
  __syncthreads();
  const int before = (warp > 0) ? wsum[warp - 1] : 0;
  *total = wsum[NT / 32 - 1];
  __syncthreads();
  return before + incl - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int *__restrict__ count,
                                                              int *__restrict__ bsum) {
  step_begin();
  const int4 *c4 =
      reinterpret_cast<const int4 *>(count) + (size_t)blockIdx.x * (kScanTile / 4) + threadIdx.x;
  int s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems / 4; ++k) {
    const int4 q = c4[k * kScanThreads];
    s += q.x + q.y + q.z + q.w;
  }
  int total;
  block_excl_scan<kScanThreads>(s, &total);
  if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

// Exclusive scan of the tile sums in place (one block).
__global__ void __launch_bounds__(1024) k_scan_bsum(int *__restrict__ bsum, int ntile) {
  const int per = (ntile + 1023) / 1024;
  const int b0 = threadIdx.x * per;
  int s = 0;
  for (int k = 0; k < per; ++k)
    if (b0 + k < ntile) s += bsum[b0 + k];
  int total;
  int run = block_excl_scan<1024>(s, &total);
  for (int k = 0; k < per; ++k)
    if (b0 + k < ntile) {
      const int v = bsum[b0 + k];
      bsum[b0 + k] = run;
      run += v;
    }
}

// sum_tiles: bsum holds the tiles' sums, and each block adds up those before
// its own; otherwise it holds their exclusive scan.
__global__ void __launch_bounds__(kScanThreads)
    k_scan_apply(Packed P, bool advance, bool sum_tiles) {
  step_begin();
  // A warp takes consecutive 128-cell rounds, four cells a lane, so that every
  // load and store is a whole line (16 cells a lane left half-written sectors)
  // at the cost of a warp scan a round.  The scan's stage (event times) of an
  // L = 8 box 7.6 -> 6.5 us, L = 64 12.9 -> 10.6, L = 96 15.2 -> 13.0; a step of
  // an L = 12 box 10.7 -> 10.05 us (half), of an L = 128 box 831 -> 826.
  constexpr int R = kScanItems / 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const size_t i0 = (size_t)blockIdx.x * (kScanTile / 4) + warp * (32 * R) + lane;
  int4 *c4 = reinterpret_cast<int4 *>(P.count) + i0;
  int4 *s4 = reinterpret_cast<int4 *>(P.start) + i0;
  int4 q[R];
#pragma unroll
  for (int k = 0; k < R; ++k) q[k] = c4[32 * k];
#pragma unroll
  for (int k = 0; k < R; ++k) c4[32 * k] = make_int4(0, 0, 0, 0);  // for the next rebuild
  int first[R], sum = 0;  // cells before this lane's in the warp's rounds
#pragma unroll
  for (int k = 0; k < R; ++k) {
    const int t = q[k].x + q[k].y + q[k].z + q[k].w;
    const int incl = warp_incl_scan(t);
    first[k] = sum + incl - t;
    sum += __shfl_sync(0xffffffffu, incl, 31);
  }
  int total;
  int run = block_excl_scan<kScanThreads>(lane == 0 ? sum : 0, &total);
  run = __shfl_sync(0xffffffffu, run, 0);  // the warps before this one
  if (sum_tiles) {
    int before = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += kScanThreads) before += P.bsum[k];
    block_excl_scan<kScanThreads>(before, &total);
    run += total;
  } else {
    run += P.bsum[blockIdx.x];
  }
#pragma unroll
  for (int k = 0; k < R; ++k) {
    int4 o;
    o.x = run + first[k];
    o.y = o.x + q[k].x;
    o.z = o.y + q[k].y;
    o.w = o.z + q[k].z;
    s4[32 * k] = o;
  }
  if (advance && blockIdx.x == 0) {
    for (int b = threadIdx.x; b < P.nbox; b += kScanThreads) {
      BoxState st = P.st[b];
      if (st.remaining > 0) {
        st.step += 1;
        st.remaining -= 1;
        st.pending = 1;
        st.adv = 1;
      } else {
        st.adv = 0;
      }
      P.st[b] = st;
    }
  }
}

// ---------------------------------------------------------------- reorder
__global__ void __launch_bounds__(kBinThreads) k_bin_keys(Packed P) {
  const int p = blockIdx.x * kBinThreads + threadIdx.x;
  step_begin();
  if (p < P.ntot) bin_key(P, p);
}

template <bool STABLE>
__global__ void __launch_bounds__(kBinThreads) k_bin_scatter(Packed P, bool zero_frc) {
  const int p = blockIdx.x * kBinThreads + threadIdx.x;
  step_begin();
  if (p < P.ntot) bin_scatter<STABLE>(P, p, zero_frc);
}

// The reorder after k_kick_bin, by arrival rank, into pos2 and vel2.
template <bool SINGLE>
__global__ void __launch_bounds__(kBinThreads) k_drift_scatter(Packed P) {
  const int p = blockIdx.x * kBinThreads + threadIdx.x;
  int b = 0;
  if constexpr (!SINGLE) b = find_box_warp(P.pbase, P.nbox, min(p, P.ntot - 1));
  if (p >= P.ntot) return;
  const BoxDev B = box_of<SINGLE>(P, b);
  const bool moved = P.st[b].adv != 0;
  float4 x = P.pos[p];
  const float4 v = P.vel[p];
  int dst = p;
  if (moved) {
    int cx, cy, cz;
    unpack_cell(__float_as_int(v.w), cx, cy, cz);
    const int c = B.cellBase + (cz * B.n[1] + cy) * B.n[0] + cx;
    if (!DPD_IN_BOUNDS(c >= 0 && c < P.ncell, P.err)) return;
    dst = P.start[c] + P.slotIn[p];
    if (!DPD_IN_BOUNDS(dst >= 0 && dst < P.start[c + 1] && dst < P.ntot, P.err)) return;
    drift(P, B, x, v);
  }
  P.pos2[dst] = x;
  P.vel2[dst] = v;
}

// ------------------------------------------------------------------ stats
constexpr int kStatsThreads = 256;

// Sum of two unevaluated pairs hi + lo of FP32 numbers, as such a pair: the
// high parts are added error-free (TwoSum), the low parts and that error go
// into the new low part, then the pair is renormalised (Dekker's Fast2Sum).
// The result carries about 2^-44 of the operands' magnitude as error.
__device__ __forceinline__ void pair_add(float &hi, float &lo, float bh, float bl) {
  const float s = hi + bh;
  const float bv = s - hi;
  float e = (hi - (s - bv)) + (bh - bv);
  e += lo + bl;
  hi = s + e;
  lo = e - (hi - s);
}

// The last block of a box to finish also sums the box's work items and writes
// its totals, and the error word, to pinned host memory, in place of a second
// kernel and two copies: dpd_get_stats of an L = 8 box 28.0 -> 21.2 us.
__global__ void __launch_bounds__(kStatsThreads)
    k_stats(Packed P, const StatsWork *__restrict__ work, const int *__restrict__ wbeg, double *out,
            int *__restrict__ done, double *__restrict__ host_sums,
            unsigned *__restrict__ host_err) {
  const StatsWork w = work[blockIdx.x];
  const BoxDev &B = P.boxes[w.box];
  const BoxState S = P.st[w.box];
  const float h = S.pending ? B.hdt_m : 0.0f;
  // Each thread sums its particles' FP32 values as unevaluated pairs
  // hi + lo of FP32 numbers (the error-free TwoSum transformation: each
  // addition's rounding error is carried in lo).  The warp and the block
  // combine those pairs as pairs, and only the block's total is converted
  // to FP64: every FP64 operation per particle or per lane is avoided,
  // since FP64 runs at a small fraction of the FP32 rate on this part.
  // Everything above the block (work items, boxes) is summed in FP64.
  constexpr int F = kStatsFields - 1;
  float hi[F] = {0.f, 0.f, 0.f, 0.f, 0.f};
  float lo[F] = {0.f, 0.f, 0.f, 0.f, 0.f};
  auto two_sum = [&](int k, float x) {
    const float t = hi[k] + x;
    const float xv = t - hi[k];
    lo[k] += (hi[k] - (t - xv)) + (x - xv);
    hi[k] = t;
  };
#pragma unroll 4
  for (int p = w.begin + threadIdx.x; p < w.end; p += kStatsThreads) {
    float4 v = P.vel[p];
    const float4 f = P.frc[p];
    v.x = fmaf(h, f.x, v.x);
    v.y = fmaf(h, f.y, v.y);
    v.z = fmaf(h, f.z, v.z);
    two_sum(0, v.x);
    two_sum(1, v.y);
    two_sum(2, v.z);
    two_sum(3, fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z)));
    two_sum(4, f.w);
  }
#pragma unroll
  for (int k = 0; k < F; ++k)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      pair_add(hi[k], lo[k], __shfl_down_sync(0xffffffffu, hi[k], o),
               __shfl_down_sync(0xffffffffu, lo[k], o));
  constexpr int NW = kStatsThreads / 32;
  static_assert(NW <= 32 && (NW & (NW - 1)) == 0, "block of 1 to 32 warps, a power of two");
  __shared__ float2 red[F][NW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int k = 0; k < F; ++k) red[k][warp] = make_float2(hi[k], lo[k]);
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < F; ++k) {
      float2 r = (lane < NW) ? red[k][lane] : make_float2(0.f, 0.f);
#pragma unroll
      for (int o = NW / 2; o > 0; o >>= 1)
        pair_add(r.x, r.y, __shfl_down_sync(0xffffffffu, r.x, o),
                 __shfl_down_sync(0xffffffffu, r.y, o));
      if (lane == 0) out[(size_t)blockIdx.x * kStatsFields + k] = (double)r.x + (double)r.y;
    }
    if (lane == 0) out[(size_t)blockIdx.x * kStatsFields + F] = (double)(w.end - w.begin);
  }
  __shared__ bool last;
  const int w0 = wbeg[w.box], w1 = wbeg[w.box + 1];
  if (threadIdx.x == 0) {
    __threadfence();  // this block's sums before its count
    last = atomicAdd(done + w.box, 1) == w1 - w0 - 1;
  }
  __syncthreads();
  if (!last) return;
  // Per-box totals in a fixed order (strided sums, then a tree), so that they
  // do not depend on the other boxes nor on which block is last.
  __threadfence();
  __shared__ double box[kStatsFields][kStatsThreads];
  const int t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < kStatsFields; ++k) {
    double acc[2] = {0.0, 0.0};
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll 4
      for (int i = w0 + t + h * kStatsThreads; i < w1; i += 2 * kStatsThreads)
        acc[h] += __ldcg(out + (size_t)i * kStatsFields + k);
    box[k][t] = acc[0] + acc[1];
  }
  __syncthreads();
  for (int h = kStatsThreads / 2; h > 0; h >>= 1) {
    if (t < h)
#pragma unroll
      for (int k = 0; k < kStatsFields; ++k) box[k][t] += box[k][t + h];
    __syncthreads();
  }
  if (t < kStatsFields) host_sums[(size_t)w.box * kStatsFields + t] = box[t][0];
  if (t == 0) {
    done[w.box] = 0;  // for the next read-out
    *host_err = *P.err;
  }
}

// ----------------------------------------------------------------- gather
// host_err (may be null): the last block to finish also writes the error word
// to pinned host memory, in place of a copy behind the kernel.
__global__ void k_gather(Packed P, int box, int slot0, int n, float *__restrict__ pos3,
                         float *__restrict__ vel3, float *__restrict__ frc3,
                         int *__restrict__ done, unsigned *__restrict__ host_err) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) {
    const int p = slot0 + k;
    const float4 x = P.pos[p];
    const int id = (int)(__float_as_uint(x.w) & kIdMask);
    if (id >= n) {
      atomicOr(P.err, kErrNonFinite);
    } else {
      const float4 f = P.frc[p];
      if (pos3) {
        pos3[3 * id] = x.x;
        pos3[3 * id + 1] = x.y;
        pos3[3 * id + 2] = x.z;
      }
      if (vel3) {
        const float h = P.st[box].pending ? P.boxes[box].hdt_m : 0.0f;
        const float4 v = P.vel[p];
        vel3[3 * id] = fmaf(h, f.x, v.x);
        vel3[3 * id + 1] = fmaf(h, f.y, v.y);
        vel3[3 * id + 2] = fmaf(h, f.z, v.z);
      }
      if (frc3) {
        frc3[3 * id] = f.x;
        frc3[3 * id + 1] = f.y;
        frc3[3 * id + 2] = f.z;
      }
    }
  }
  if (!host_err) return;
  __syncthreads();  // this block's error bits
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(done, 1) == (int)gridDim.x - 1) {
      *done = 0;  // for the next read-out
      *host_err = atomicOr(P.err, 0u);
    }
  }
}

// -------------------------------------------------------------- debug rng
__global__ void k_debug_rng(const uint32_t *__restrict__ lo, const uint32_t *__restrict__ hi,
                            long long n, uint32_t slo, uint32_t shi, uint32_t klo, uint32_t khi,
                            int noise, uint32_t *__restrict__ out, uint32_t *__restrict__ out1,
                            float *__restrict__ xi) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const uint2 u = pair_words(lo[k], hi[k], slo, shi, klo, khi);
  out[k] = u.x;
  if (out1) out1[k] = u.y;
  if (xi) xi[k] = noise ? gauss_xi(u.x, u.y) : __fmul_rn(noise_int(u.x), kSqrt3Scale);
}

// ------------------------------------------------------ served-form kernels
// Initial state of a new box drawn on the device from its seed: positions
// uniform in [0, L), velocities Maxwellian (Box-Muller) with variance kT/m.
// Philox-4x32-10 with key (seed lo, seed hi ^ 0x5EED0001) on counters
// (id, 0, 0, 0) and (id, 1, 0, 0); this only samples an initial condition.
__device__ __forceinline__ void philox4(uint32_t c0, uint32_t c1, uint32_t k0, uint32_t k1,
                                        uint32_t out[4]) {
  uint32_t c2 = 0u, c3 = 0u;
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += kPhiloxW0;
      k1 += kPhiloxW1;
    }
    const uint32_t hi0 = __umulhi(kPhiloxM0, c0), lo0 = kPhiloxM0 * c0;
    const uint32_t hi1 = __umulhi(kPhiloxM1, c2), lo1 = kPhiloxM1 * c2;
    const uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  out[0] = c0;
  out[1] = c1;
  out[2] = c2;
  out[3] = c3;
}

__device__ __forceinline__ float unit_open(uint32_t u) {  // (0, 1)
  return ((float)(u >> 8) + 0.5f) * (1.0f / 16777216.0f);
}

__global__ void k_init_box(Packed P, int slot0, int n, float Lx, float Ly, float Lz, float vscale,
                           uint32_t seed_lo, uint32_t seed_hi) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t a[4], b[4];
  philox4((uint32_t)i, 0u, seed_lo, seed_hi ^ 0x5EED0001u, a);
  philox4((uint32_t)i, 1u, seed_lo, seed_hi ^ 0x5EED0001u, b);
  float x = unit_open(a[0]) * Lx, y = unit_open(a[1]) * Ly, z = unit_open(a[2]) * Lz;
  x = x < Lx ? x : 0.f;
  y = y < Ly ? y : 0.f;
  z = z < Lz ? z : 0.f;
  const float r1 = sqrtf(-2.0f * logf(unit_open(b[0])));
  const float r2 = sqrtf(-2.0f * logf(unit_open(b[2])));
  float s1, c1, s2, c2;
  sincospif(2.0f * unit_open(b[1]), &s1, &c1);
  sincospif(2.0f * unit_open(b[3]), &s2, &c2);
  P.pos[slot0 + i] = make_float4(x, y, z, __int_as_float(i));
  P.vel[slot0 + i] = make_float4(vscale * r1 * c1, vscale * r1 * s1, vscale * r2 * c2, 0.f);
}

// Remove the mean velocity of one box: one block sums in a fixed order (FP64),
// then every thread subtracts.
__global__ void __launch_bounds__(1024) k_zero_momentum(Packed P, int slot0, int n) {
  __shared__ double red[3][32];
  __shared__ float mean[3];
  double s[3] = {0, 0, 0};
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float4 v = P.vel[slot0 + i];
    s[0] += v.x;
    s[1] += v.y;
    s[2] += v.z;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double t = s[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) red[k][warp] = t;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += red[threadIdx.x][w];
    mean[threadIdx.x] = (float)(n > 0 ? t / n : 0.0);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    float4 v = P.vel[slot0 + i];
    v.x -= mean[0];
    v.y -= mean[1];
    v.z -= mean[2];
    P.vel[slot0 + i] = v;
  }
}

// Move surviving boxes to their new slot ranges: new slot q of new box b
// takes old slot src0[b] + (q - newbase[b]) (src0 < 0: a new box, skipped).
__global__ void k_repack(const float4 *__restrict__ opos, const float4 *__restrict__ ovel,
                         float4 *__restrict__ npos, float4 *__restrict__ nvel,
                         const int *__restrict__ newbase, const int *__restrict__ src0, int nbox,
                         int ntot) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= ntot) return;
  const int b = find_box(newbase, nbox, q);
  const int s0 = src0[b];
  if (s0 < 0) return;
  const int src = s0 + (q - newbase[b]);
  npos[q] = opos[src];
  nvel[q] = ovel[src];
}

// Statistics sample of every box whose step is a multiple of `every` and
// past its window start: per work item FP64 partials of sum v^2, sum r.F^C
// (frc.w, each pair counted twice) and per-slab sums of the flow-axis
// velocity with their counts.  The last block of a box to finish adds the
// box's partials (in work order) to its accumulators: acc[b] = {samples,
// sum v^2, sum frc.w, slab sums[nbins], slab counts[nbins]}.  It runs behind
// every step, so its cost on the steps that no box samples is its launch: a
// second kernel for the accumulators took 3.2 us a step.
__global__ void __launch_bounds__(256)
    k_sample(Packed P, const StatsWork *__restrict__ work, const int *__restrict__ wbeg,
             const long long *__restrict__ from, int every, int nbins, double *__restrict__ part,
             double *__restrict__ acc, int *__restrict__ done) {
  extern __shared__ double sbin[];  // 2 * nbins: sums then counts
  const StatsWork w = work[blockIdx.x];
  const BoxState S = P.st[w.box];
  const int fields = 3 + 2 * nbins;
  double *out = part + (size_t)blockIdx.x * fields;
  const bool take = S.adv && every > 0 && (long long)S.step > from[w.box] &&
                    (S.step % (unsigned long long)every) == 0ull;
  if (!take) return;  // the same for all blocks of a box
  for (int k = threadIdx.x; k < 2 * nbins; k += blockDim.x) sbin[k] = 0.0;
  __syncthreads();
  const BoxDev B = P.boxes[w.box];
  const float h = S.pending ? B.hdt_m : 0.0f;
  const float Lg = B.L[B.fb_grad];
  double v2 = 0.0, vir = 0.0;
  for (int p = w.begin + threadIdx.x; p < w.end; p += blockDim.x) {
    const float4 x = P.pos[p];
    float4 v = P.vel[p];
    const float4 f = P.frc[p];
    v.x = fmaf(h, f.x, v.x);
    v.y = fmaf(h, f.y, v.y);
    v.z = fmaf(h, f.z, v.z);
    v2 += (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z;
    vir += (double)f.w;
    if (nbins > 0) {
      const float xg = (B.fb_grad == 0) ? x.x : (B.fb_grad == 1) ? x.y : x.z;
      const float vf = (B.fb_flow == 0) ? v.x : (B.fb_flow == 1) ? v.y : v.z;
      int bin = (int)(xg / Lg * nbins);
      bin = min(max(bin, 0), nbins - 1);
      atomicAdd(&sbin[bin], (double)vf);
      atomicAdd(&sbin[nbins + bin], 1.0);
    }
  }
  __shared__ double red[2][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v2 += __shfl_down_sync(0xffffffffu, v2, o);
    vir += __shfl_down_sync(0xffffffffu, vir, o);
  }
  if (lane == 0) {
    red[0][warp] = v2;
    red[1][warp] = vir;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, c = 0.0;
    for (int q = 0; q < (int)(blockDim.x / 32); ++q) {
      a += red[0][q];
      c += red[1][q];
    }
    out[1] = a;
    out[2] = c;
  }
  for (int k = threadIdx.x; k < 2 * nbins; k += blockDim.x) out[3 + k] = sbin[k];
  __shared__ bool last;
  __threadfence();  // this block's partials before its count
  __syncthreads();
  const int w0 = wbeg[w.box], w1 = wbeg[w.box + 1];
  if (threadIdx.x == 0) last = atomicAdd(done + w.box, 1) == w1 - w0 - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  double *a = acc + (size_t)w.box * fields;
  for (int k = threadIdx.x; k < fields; k += blockDim.x) {
    double s = 0.0;
    if (k == 0)
      s = 1.0;
    else
      for (int i = w0; i < w1; ++i) s += __ldcg(part + (size_t)i * fields + k);
    a[k] += s;
  }
  if (threadIdx.x == 0) done[w.box] = 0;  // for the next sample or read-out
}

// ================================================================ launchers

cudaError_t launch_load(const Packed &P, int slot0, int n, const float *pos3, const float *vel3,
                        float Lx, float Ly, float Lz, cudaStream_t s, const int32_t *species,
                        int nspec) {
  if (n <= 0) return cudaSuccess;
  k_load<<<blocks_for(n, 256), 256, 0, s>>>(P, slot0, n, pos3, vel3, Lx, Ly, Lz, species, nspec);
  return cudaGetLastError();
}

// Scan of the cell counts.  One tile needs no sums of others.  Up to
// kScanSumTiles tiles each block of the last pass adds up the sums before its
// own (at most 8 KB, from L2) instead of waiting for a launch that scans
// them, which took 2 to 4 us: the scan's stage went from 13.7 to 7.7 us for
// an L = 8 box, 13.7 to 10.8 us at L = 24 and 15.1 to 12.9 us at L = 64
// (event times, with the gaps between launches).  Beyond that the sums are
// scanned by one block.
constexpr int kScanSumTiles = 2048;
static void launch_scan(const Packed &P, bool advance, bool early, cudaStream_t s) {
  const int nt = scan_tiles(P.ncell);
  if (nt > 1) launch_step_kernel(early, k_scan_reduce, nt, kScanThreads, 0, s, P.count, P.bsum);
  if (nt > kScanSumTiles) k_scan_bsum<<<1, 1024, 0, s>>>(P.bsum, nt);
  launch_step_kernel(early, k_scan_apply, nt, kScanThreads, 0, s, P, advance,
                     nt <= kScanSumTiles);
}

static void launch_integrate(const Packed &P, bool move, bool early, cudaStream_t s) {
  const int gb = blocks_for(P.ntot, kBinThreads);
  if (P.nbox == 1)
    launch_step_kernel(early, k_integrate_bin<true>, gb, kBinThreads, 0, s, P, move);
  else
    launch_step_kernel(early, k_integrate_bin<false>, gb, kBinThreads, 0, s, P, move);
}

// The full stencil's key pass.
static void launch_keys(const Packed &P, bool early, cudaStream_t s) {
  launch_step_kernel(early, k_bin_keys, blocks_for(P.ntot, kBinThreads), kBinThreads, 0, s, P);
}

// half: by arrival rank, clearing the forces for the half stencil's sums.
static void launch_scatter(const Packed &P, bool half, bool early, cudaStream_t s) {
  const int gb = blocks_for(P.ntot, kBinThreads);
  if (half)
    launch_step_kernel(early, k_bin_scatter<false>, gb, kBinThreads, 0, s, P, true);
  else
    launch_step_kernel(early, k_bin_scatter<true>, gb, kBinThreads, 0, s, P, false);
}

cudaError_t launch_step(const Packed &P, bool move, bool advance, const StepConfig &cfg,
                        cudaStream_t s, bool fused_in, bool fuse_out) {
  if (P.ntot <= 0) return cudaSuccess;
  const bool half = cfg.stencil == 1;
  const bool early = cfg.rows && P.ntot <= kEarlySlots &&
                     rows_pay(P, half, cfg.nbands > 0 ? cfg.band[0].gen : 0);
  // fused_in: row a1 of this step ran in the previous step's force kernel
  if (!fused_in) launch_integrate(P, move, early, s);
  launch_scan(P, advance, early, s);
  if (!half) launch_keys(P, early, s);
  launch_scatter(P, half, early, s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_force(P, cfg, s, fuse_out && cfg.stencil == 0);
}

bool swap_pays(const Packed &P, const StepConfig &cfg) {
  return cfg.stencil == 1 && P.ntot > kSwapSlots;
}

static void launch_kick(const Packed &P, cudaStream_t s) {
  const int gb = blocks_for(P.ntot, kBinThreads);
  if (P.nbox == 1)
    k_kick_bin<true><<<gb, kBinThreads, 0, s>>>(P);
  else
    k_kick_bin<false><<<gb, kBinThreads, 0, s>>>(P);
}

static void launch_drift(Packed &P, cudaStream_t s) {
  const int gb = blocks_for(P.ntot, kBinThreads);
  if (P.nbox == 1)
    k_drift_scatter<true><<<gb, kBinThreads, 0, s>>>(P);
  else
    k_drift_scatter<false><<<gb, kBinThreads, 0, s>>>(P);
  std::swap(P.pos, P.pos2);
  std::swap(P.vel, P.vel2);
}

cudaError_t launch_step_swapped(Packed &P, const StepConfig &cfg, cudaStream_t s) {
  if (P.ntot <= 0) return cudaSuccess;
  launch_kick(P, s);
  launch_scan(P, true, false, s);
  launch_drift(P, s);
  cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_force(P, cfg, s);
}

cudaError_t launch_step_timed(Packed &P, const StepConfig &cfg, bool swap, cudaStream_t s,
                              cudaEvent_t *ev) {
  if (P.ntot <= 0) return cudaSuccess;
  const bool half = cfg.stencil == 1;
  cudaError_t e;
  if ((e = cudaEventRecord(ev[0], s)) != cudaSuccess) return e;
  if (swap)
    launch_kick(P, s);
  else
    launch_integrate(P, true, false, s);
  if ((e = cudaEventRecord(ev[1], s)) != cudaSuccess) return e;
  launch_scan(P, true, false, s);
  if ((e = cudaEventRecord(ev[2], s)) != cudaSuccess) return e;
  if (!half) launch_keys(P, false, s);
  if ((e = cudaEventRecord(ev[3], s)) != cudaSuccess) return e;
  if (swap)
    launch_drift(P, s);
  else
    launch_scatter(P, half, false, s);
  if ((e = cudaEventRecord(ev[4], s)) != cudaSuccess) return e;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_force(P, cfg, s)) != cudaSuccess) return e;
  return cudaEventRecord(ev[5], s);
}

cudaError_t launch_stats(const Packed &P, const StatsWork *work, int nwork, const int *wbeg,
                         double *part, int *done, double *host_sums, unsigned *host_err,
                         cudaStream_t s) {
  if (nwork <= 0) return cudaSuccess;
  k_stats<<<nwork, kStatsThreads, 0, s>>>(P, work, wbeg, part, done, host_sums, host_err);
  return cudaGetLastError();
}

cudaError_t launch_gather(const Packed &P, int box, int slot0, int n, float *pos3, float *vel3,
                          float *frc3, cudaStream_t s, int *done, unsigned *host_err) {
  if (n <= 0) return cudaSuccess;
  k_gather<<<blocks_for(n, 256), 256, 0, s>>>(P, box, slot0, n, pos3, vel3, frc3, done, host_err);
  return cudaGetLastError();
}

cudaError_t launch_debug_rng(const uint32_t *lo, const uint32_t *hi, long long n, uint64_t step,
                             uint64_t seed, int noise, uint32_t *out, uint32_t *out1, float *xi,
                             cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_debug_rng<<<blocks_for(n, 256), 256, 0, s>>>(lo, hi, n, (uint32_t)step,
                                                 (uint32_t)(step >> 32), (uint32_t)seed,
                                                 (uint32_t)(seed >> 32), noise, out, out1, xi);
  return cudaGetLastError();
}

}  // namespace dpd

namespace dpd {

cudaError_t launch_init_box(const Packed &P, int slot0, int n, float Lx, float Ly, float Lz,
                            float vscale, uint64_t seed, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_init_box<<<blocks_for(n, 256), 256, 0, s>>>(P, slot0, n, Lx, Ly, Lz, vscale, (uint32_t)seed,
                                                 (uint32_t)(seed >> 32));
  k_zero_momentum<<<1, 1024, 0, s>>>(P, slot0, n);
  return cudaGetLastError();
}

cudaError_t launch_repack(const float4 *opos, const float4 *ovel, float4 *npos, float4 *nvel,
                          const int *newbase, const int *src0, int nbox, int ntot,
                          cudaStream_t s) {
  if (ntot <= 0) return cudaSuccess;
  k_repack<<<blocks_for(ntot, 256), 256, 0, s>>>(opos, ovel, npos, nvel, newbase, src0, nbox,
                                                  ntot);
  return cudaGetLastError();
}

cudaError_t launch_sample(const Packed &P, const StatsWork *work, int nwork, const int *wbeg,
                          const long long *from, int every, int nbins, double *part, double *acc,
                          int *done, cudaStream_t s) {
  if (nwork <= 0 || every <= 0) return cudaSuccess;
  k_sample<<<nwork, 256, 2 * nbins * sizeof(double), s>>>(P, work, wbeg, from, every, nbins, part,
                                                          acc, done);
  return cudaGetLastError();
}

}  // namespace dpd
