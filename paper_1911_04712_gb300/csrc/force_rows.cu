// Row-parallel force kernels for small sets (pair forces, Sec. 2.1 Eqs. 2-5,
// over the cell list of Sec. 3.2).  A block owns 32 target slots and has one
// warp per stencil row: warp r scans row r for the 32 targets at once, the
// lists of all rows are gathered into one queue, every thread of the block
// evaluates pairs of the queue, and with the full stencil each target then
// adds its pairs' results in row and slot order: the order, and so the bits,
// of the direct routine.
//
// What bounds it: latency.  A set of a few thousand particles is a handful
// of warps per SM, and the direct routine has each of them walk nine rows
// and evaluate up to twenty pairs one after the other, most of the time
// waiting for one load.  Here a step's chain is one row scan, about two pair
// evaluations and one ordered sum.  Force stage at rho = 3, direct against
// row-parallel: N = 1,536 full 28.6 -> 10.2 us, half 18.4 -> 8.2; N = 55,296
// (rho = 4) full 41.3 -> 33.1, half 23.9 -> 18.3.  rows_pay says where the lines
// cross.
#include <cuda_runtime.h>

#include <cstdint>

#include "dpd_device.cuh"
#include "force_direct.cuh"
#include "kernels.h"

namespace dpd {

namespace {

constexpr int kRowsUnroll = 4;  // candidates loaded per iteration
// List places of one target in one row, and of a block's queue: at rho = 8
// the own row holds 10 neighbours of 34, so that denser boxes need the longer
// lists, which cost the others resident blocks.
constexpr int kRowsCap = 24, kRowsCapDense = 40;
constexpr int kRowsQueue = 1728, kRowsQueueDense = 2880;  // half of it for the half stencil
// Resident blocks an SM the registers are held to.  With eight candidates an
// iteration, the long lists and no bound (72 registers, three and five blocks)
// an L = 24, rho = 4 box stepped in 40.0 us (full) and 22.6 (half), with these
// in 35.9 and 21.4; an L = 12, rho = 3 box in 14.9 / 11.3 and 14.7 / 11.3.
constexpr int kRowsBlocksFull = 4, kRowsBlocksHalf = 6;
constexpr unsigned kAll = 0xffffffffu;

// Which boxes (rows_pay).
constexpr int kRowsMaxHalf = 262144;
constexpr int kRowsMaxFull = 65536, kRowsMaxFullDense = 106496;  // dense: above 5 per cell
constexpr int kRowsMaxFullGeneral = 90112, kRowsMaxFullGeneralDense = 139264;
constexpr int kRowsMaxPerCell = 12;
bool slots_per_cell_at_most(const Packed &P, int n) {
  return (long long)P.ntot * kSlicesX <= (long long)n * P.ncell;
}

template <bool HALF, bool DENSE>
struct RowsShared {
  static constexpr int kRows = HALF ? 5 : 9, kThreads = 32 * kRows;
  static constexpr int kCap = DENSE ? kRowsCapDense : kRowsCap;
  static constexpr int kQueue = (DENSE ? kRowsQueueDense : kRowsQueue) / (HALF ? 2 : 1);
  float4 own_pos[32], own_vel[32];
  union {
    uint32_t list[kCap * kThreads];  // entry k of thread t at k * kThreads + t
    float4 res[HALF ? 1 : kQueue];       // after the lists were gathered
  };
  uint32_t queue[kQueue];                // list entries: rows in order, lanes in order
  uint8_t who[kQueue];                   // their targets' lanes
  uint16_t off[kRows][32], cnt[kRows][32];
  int row_total[kRows];
  int overflow;
};

// A force to its particle's place in an n x 3 array.
__device__ __forceinline__ void store3(float *__restrict__ out3, const float4 &pi,
                                       const float4 &f) {
  float *o = out3 + 3 * (size_t)(__float_as_uint(pi.w) & kIdMask);
  o[0] = f.x;
  o[1] = f.y;
  o[2] = f.z;
}

template <bool HALF, int GEN, bool DENSE>
__global__ void __launch_bounds__(RowsShared<HALF, DENSE>::kThreads,
                                  HALF ? kRowsBlocksHalf : kRowsBlocksFull)
    k_force_rows(Packed P, bool fuse, float *__restrict__ out3) {
  using Sh = RowsShared<HALF, DENSE>;
  constexpr int NT = Sh::kThreads, U = kRowsUnroll, CAP = Sh::kCap;
  extern __shared__ float4 rows_smem[];
  Sh &W = *reinterpret_cast<Sh *>(rows_smem);
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
  const int p0 = (int)blockIdx.x * 32, p = p0 + lane;
  const bool real = p < P.ntot;
  const BoxDev &B = P.single;
  step_begin();
  const BoxState S = P.st[0];
  const bool alive = real && S.adv && DPD_IN_BOUNDS(p >= 0 && p < P.ntot, P.err);
  float4 pi = make_float4(0.f, 0.f, 0.f, 0.f), vi = pi;
  if (alive) {
    pi = P.pos[p];
    vi = P.vel[p];
  }
  if (row == 0) {
    W.own_pos[lane] = pi;
    W.own_vel[lane] = vi;
  }
  if (tid == 0) W.overflow = 0;

  // ---- this warp's row (rows as in the direct routine)
  int cnt = 0;
  bool over = false;
  if (alive) {
    const int dz = HALF ? (row < 2 ? 0 : 1) : row / 3 - 1;
    const int dy = HALF ? (row == 0 ? 0 : (row == 1 ? 1 : row - 3)) : row - 3 * (row / 3) - 1;
    const float Lx = B.L[0], Ly = B.L[1], Lz = B.L[2];
    const int nx = B.n[0], ny = B.n[1], nz = B.n[2];
    int cx, cy, cz;
    unpack_cell(__float_as_int(vi.w), cx, cy, cz);
    const int xlo = __float2int_rd((pi.x - B.xwin) * B.invh[0]);
    const int xhi = __float2int_rd((pi.x + B.xwin) * B.invh[0]);
    int z = cz + dz, y = cy + dy;
    float az = pi.z, jsz = 0.f, ay = pi.y, jsy = 0.f;
    uint32_t code = 0;
    if (z < 0) {
      z += nz;
      jsz = Lz;
      code |= kCodeJZ;
    } else if (z >= nz) {
      z -= nz;
      az = pi.z - Lz;
      code |= kCodeIZ;
    }
    if (y < 0) {
      y += ny;
      jsy = Ly;
      code |= kCodeJY;
    } else if (y >= ny) {
      y -= ny;
      ay = pi.y - Ly;
      code |= kCodeIY;
    }
    const int rowbase = B.cellBase + (z * ny + y) * nx;
    const bool own = HALF && row == 0;
    const int lo = own ? cx : xlo, hi = xhi;
    if (DPD_IN_BOUNDS(rowbase >= 0 && rowbase + nx <= P.ncell && lo >= -nx && lo <= hi &&
                          hi < 2 * nx, P.err)) {
      const int nseg = (lo < 0 || hi >= nx) ? 2 : 1;
      // both ends of both parts at once: [s0, s1) and, across an x face, [0, s2)
      const int s0 = lo < 0 ? lo + nx : lo, s1 = (lo < 0 || hi >= nx) ? nx : hi + 1;
      const int s2 = lo < 0 ? hi + 1 : hi - nx + 1;
      int j0 = own ? p + 1 : __ldg(P.start + rowbase + s0);
      int j1 = __ldg(P.start + rowbase + s1);
      int k0 = 0, k1 = 0;
      if (nseg == 2) {
        k0 = __ldg(P.start + rowbase);
        k1 = __ldg(P.start + rowbase + s2);
      }
      if (!DPD_IN_BOUNDS(j0 >= 0 && j0 <= j1 && j1 <= P.ntot && k0 >= 0 && k0 <= k1 &&
                             k1 <= P.ntot, P.err))
        j0 = j1 = k0 = k1 = 0;
      const uint32_t rc2m1 = __float_as_uint(B.rc2) - 1u;
#pragma unroll 1
      for (int sg = 0; sg < nseg && !over; ++sg) {
        float ax = pi.x, jsx = 0.f;
        uint32_t c = code;
        int a0 = j0, a1 = j1;
        if (lo < 0) {  // slices lo + nx .. nx - 1 as r_j - L, then 0 .. hi
          if (sg == 0) {
            jsx = Lx;
            c |= kCodeJX;
          } else {
            a0 = k0;
            a1 = k1;
          }
        } else if (sg == 1) {  // lo .. nx - 1, then 0 .. hi - nx seen from r_i - L
          a0 = k0;
          a1 = k1;
          ax = pi.x - Lx;
          c |= kCodeIX;
        }
        const int stop = scan_range<true, NT, CAP, U>(P.pos, a0, a1, ax, ay, az, jsx, jsy, jsz,
                                                      rc2m1, c, W.list + tid, cnt);
        over = stop >= 0 && (stop < a1 || sg + 1 < nseg);
      }
    }
  }

  // ---- places in the queue: rows in order, lanes in order
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kAll, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) W.row_total[row] = incl;
  __syncthreads();
  if (over) W.overflow = 1;
  int base = 0, total = 0;
#pragma unroll
  for (int r = 0; r < Sh::kRows; ++r) {
    const int n = W.row_total[r];
    base += r < row ? n : 0;
    total += n;
  }
  const int off = base + incl - cnt;
  W.off[row][lane] = (uint16_t)off;
  W.cnt[row][lane] = (uint16_t)cnt;
  if (total <= Sh::kQueue)
    for (int k = 0; k < cnt; ++k) {
      W.queue[off + k] = W.list[k * NT + tid];
      W.who[off + k] = (uint8_t)lane;
    }
  __syncthreads();

  if (W.overflow || total > Sh::kQueue) {
    // a denser place than the lists hold: the direct routine, by one warp
    if (row == 0) {
      force_direct<HALF, NT, CAP, false, GEN>(P, P.single, S, p, alive, W.list + tid, nullptr,
                                                nullptr, false, fuse, real);
      if (out3 && alive) store3(out3, pi, P.frc[p]);
    }
    return;
  }

  // ---- evaluate the queue
#pragma unroll 1
  for (int q = tid; q < total; q += NT) {
    const uint32_t e = W.queue[q];
    const int o = W.who[q], j = (int)(e & kSlotMask);
    if (!DPD_IN_BOUNDS(j < P.ntot, P.err)) continue;
    const float4 pj = __ldg(P.pos + j), vj = __ldg(P.vel + j);
    const float4 qi = W.own_pos[o], ui = W.own_vel[o];
    float dx, dy, dz;
    pair_vector(B, e, qi, pj, dx, dy, dz);
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float4 g = pair_force<GEN>(B, dx, dy, dz, r2, ui, vj, __float_as_uint(qi.w),
                                       __float_as_uint(pj.w), (uint32_t)S.step,
                                       (uint32_t)(S.step >> 32));
    if constexpr (HALF) {
      atomicAdd(P.frc + j, make_float4(-g.x, -g.y, -g.z, g.w));
      atomicAdd(P.frc + (p0 + o), g);
    } else {
      W.res[q] = g;
    }
  }

  if constexpr (!HALF) __syncthreads();
  if (row != 0) return;
  float fx = 0.f, fy = 0.f, fz = 0.f, vir = 0.f;
  if constexpr (!HALF) {
#pragma unroll 1
    for (int r = 0; r < Sh::kRows; ++r) {
      const int q0 = W.off[r][lane], q1 = q0 + W.cnt[r][lane];
#pragma unroll 4
      for (int q = q0; q < q1; ++q) {
        const float4 g = W.res[q];
        fx += g.x;
        fy += g.y;
        fz += g.z;
        vir += g.w;
      }
    }
  }
  finish_force<HALF>(P, B, S, p, pi, vi, alive, real, fuse, fx, fy, fz, vir);
  if (out3 && alive) store3(out3, pi, P.frc[p]);  // this thread's own store
}

template <bool HALF, int GEN, bool DENSE>
cudaError_t launch_one(const Packed &P, bool fuse, cudaStream_t s, float *out3) {
  using Sh = RowsShared<HALF, DENSE>;
  return launch_step_kernel(P.ntot <= kEarlySlots, k_force_rows<HALF, GEN, DENSE>,
                            (P.ntot + 31) / 32, Sh::kThreads, sizeof(Sh), s, P, fuse, out3);
}

template <bool HALF, int GEN>
cudaError_t launch_one(const Packed &P, bool fuse, cudaStream_t s, float *out3) {
  return slots_per_cell_at_most(P, 7) ? launch_one<HALF, GEN, false>(P, fuse, s, out3)
                                      : launch_one<HALF, GEN, true>(P, fuse, s, out3);
}

template <bool HALF, int GEN>
cudaError_t prepare_one() {
  cudaError_t e = cudaFuncSetAttribute(k_force_rows<HALF, GEN, false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(RowsShared<HALF, false>));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_force_rows<HALF, GEN, true>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)sizeof(RowsShared<HALF, true>));
}

}  // namespace

// The row-parallel kernels win while the direct kernels leave the GPU waiting.
// A step, direct against row-parallel (us):
//   full  N = 40,960 (rho 10) 78.3 / 47.0; 65,856 (rho 3) 40.5 / 38.3; 81,000 (rho 3)
//         43.0 / 44.1; 105,456 (rho 6) 73.0 / 65.5; 106,480 (rho 10) 103.9 / 98.3;
//         279,936 (rho 6) 137.6 / 146.2
//   half  N = 40,960 (rho 10) 42.5 / 28.4; 192,000 (rho 3) 46.6 / 41.3; 255,552 (rho 3)
//         52.6 / 51.2; 331,776 (rho 3) 62.0 / 63.9; 552,960 (rho 5) 117.1 / 120.9
// and the general kernels (Gaussian noise; several species)
//   full  N = 65,856 (rho 3) 46.1 / 38.9; 42.6 / 38.5, 98,304 (rho 3) 55.2 / 50.2; 49.1 /
//         49.8, 116,346 (rho 3, uneven edges) 57.5 / 63.9, 138,240 (rho 10) 167.6 / 128.0;
//         140.6 / 124.9
//   half  N = 255,552 (rho 3) 55.5 / 53.1; 54.6 / 52.0, 331,776 (rho 3) 66.4 / 66.5; 64.6 / 65.1.
// Above about 12 particles per cell the lists overflow too often.
bool rows_pay(const Packed &P, bool half, bool general) {
  const bool dense = !slots_per_cell_at_most(P, 5);
  int most = kRowsMaxHalf;
  if (!half && general)
    most = dense ? kRowsMaxFullGeneralDense : kRowsMaxFullGeneral;
  else if (!half)
    most = dense ? kRowsMaxFullDense : kRowsMaxFull;
  return P.nbox == 1 && P.ntot <= most && slots_per_cell_at_most(P, kRowsMaxPerCell);
}

cudaError_t prepare_rows() {
  cudaError_t e = cudaSuccess;
  for (cudaError_t (*one)() :
       {prepare_one<false, 0>, prepare_one<false, 1>, prepare_one<false, 2>, prepare_one<false, 3>,
        prepare_one<true, 0>, prepare_one<true, 1>, prepare_one<true, 2>, prepare_one<true, 3>})
    if (e == cudaSuccess) e = one();
  return e;
}

template <bool HALF>
static cudaError_t launch_gen(const Packed &P, int gen, bool fuse, cudaStream_t s, float *out3) {
  switch (gen) {
    case 0: return launch_one<HALF, 0>(P, fuse, s, out3);
    case kGenGauss: return launch_one<HALF, kGenGauss>(P, fuse, s, out3);
    case kGenSpecies: return launch_one<HALF, kGenSpecies>(P, fuse, s, out3);
    default: return launch_one<HALF, kGenGauss | kGenSpecies>(P, fuse, s, out3);
  }
}

cudaError_t launch_force_rows(const Packed &P, bool half, int gen, bool fuse, cudaStream_t s,
                              float *out3) {
  if (P.nbox != 1 || (half && (fuse || out3))) return cudaErrorInvalidValue;
  return half ? launch_gen<true>(P, gen, fuse, s, out3) : launch_gen<false>(P, gen, fuse, s, out3);
}

}  // namespace dpd
