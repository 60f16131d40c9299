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
//
// Places denser than the lists or the queue hold are done in rounds by the whole
// block (dense_full, dense_half).  One warp with the direct routine, as before,
// leaves the block's other warps idle: a step of 65,000 particles in a drop of 15
// per cell in an otherwise empty box took 275 us with the full stencil (104 in
// rounds, 100 by the direct kernel), of 260,000 with the half stencil 364 (139;
// 143); of 16,000 in a drop of 20 per cell 52 and 30 us in rounds, 100 and 52 by
// the direct kernels.  The slowest against the direct kernel are full-stencil boxes
// at the upper end with every particle in a drop of 10 to 12 per cell: 96 to 80.
#include <cuda_runtime.h>

#include <cstdint>
#include <iterator>

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
constexpr int kRowsQueue = 1728, kRowsQueueDense = 2880, kRowsQueueDenseHalf = 1440;
// Resident blocks an SM the registers are held to.  With eight candidates an
// iteration, the long lists and no bound (72 registers, three and five blocks)
// an L = 24, rho = 4 box stepped in 40.0 us (full) and 22.6 (half), with these
// in 35.9 and 21.4; an L = 12, rho = 3 box in 14.9 / 11.3 and 14.7 / 11.3.
constexpr int kRowsBlocksFull = 4, kRowsBlocksHalf = 6;
constexpr unsigned kAll = 0xffffffffu;

bool slots_per_cell_at_most(const Packed &P, double n) {
  return (double)P.ntot * kSlicesX <= n * P.ncell;
}

template <bool HALF, bool DENSE>
struct RowsShared {
  static constexpr int kRows = HALF ? 5 : 9, kThreads = 32 * kRows;
  static constexpr int kCap = DENSE ? kRowsCapDense : kRowsCap;
  static constexpr int kQueue = !DENSE ? kRowsQueue : HALF ? kRowsQueueDenseHalf : kRowsQueueDense;
  float4 own_pos[32], own_vel[32];
  union {
    uint32_t list[kCap * kThreads];  // entry k of thread t at k * kThreads + t
    float4 res[HALF ? 1 : kQueue];   // after the lists were gathered
  };
  uint32_t queue[kQueue];            // list entries: warps in order, lanes in order
  uint8_t who[kQueue];               // their targets' lanes
  uint16_t off[kRows][32], cnt[kRows][32];
  int row_total[kRows];
  int overflow;                      // a list was not enough
};

// A force to its particle's place in an n x 3 array.
__device__ __forceinline__ void store3(float *__restrict__ out3, const float4 &pi,
                                       const float4 &f) {
  float *o = out3 + 3 * (size_t)(__float_as_uint(pi.w) & kIdMask);
  o[0] = f.x;
  o[1] = f.y;
  o[2] = f.z;
}

// One stencil row of this lane's target, if it has one (rows as in the direct
// routine): appends the neighbours among its candidates, in slot order, to a
// list.  PART: among the candidates b .. e - 1 that `part(size, b, e)` names, of
// `size` in all.  True if it did not get through: it took `taken` candidates until
// the list was full, or (LIMIT) none, since the warp has more than `most`.
template <bool HALF, bool PART, bool LIMIT, int NT, int CAP, typename F>
__device__ __forceinline__ bool scan_row(const Packed &P, const BoxDev &B, int row, int p,
                                         const float4 &pi, const float4 &vi, bool alive, F part,
                                         int most, uint32_t *lst, int &cnt, int &size,
                                         int &taken) {
  const float Lx = B.L[0], Ly = B.L[1], Lz = B.L[2];
  float az = pi.z, jsz = 0.f, ay = pi.y, jsy = 0.f;
  uint32_t code = 0;
  int nseg = 0, j0 = 0, j1 = 0, k0 = 0, k1 = 0;  // slots [j0, j1), then [k0, k1) across an x face
  bool low = false, over = false;                // low: it is the lower face
  if (alive) {
    const int dz = HALF ? (row < 2 ? 0 : 1) : row / 3 - 1;
    const int dy = HALF ? (row == 0 ? 0 : (row == 1 ? 1 : row - 3)) : row - 3 * (row / 3) - 1;
    const int nx = B.n[0], ny = B.n[1], nz = B.n[2];
    int cx, cy, cz;
    unpack_cell(__float_as_int(vi.w), cx, cy, cz);
    const int xlo = __float2int_rd((pi.x - B.xwin) * B.invh[0]);
    const int xhi = __float2int_rd((pi.x + B.xwin) * B.invh[0]);
    int z = cz + dz, y = cy + dy;
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
      low = lo < 0;
      nseg = (lo < 0 || hi >= nx) ? 2 : 1;
      // both ends of both parts at once: [s0, s1) and, across an x face, [0, s2)
      const int s0 = lo < 0 ? lo + nx : lo, s1 = (lo < 0 || hi >= nx) ? nx : hi + 1;
      const int s2 = lo < 0 ? hi + 1 : hi - nx + 1;
      j0 = own ? p + 1 : __ldg(P.start + rowbase + s0);
      j1 = __ldg(P.start + rowbase + s1);
      if (nseg == 2) {
        k0 = __ldg(P.start + rowbase);
        k1 = __ldg(P.start + rowbase + s2);
      }
      if (!DPD_IN_BOUNDS(j0 >= 0 && j0 <= j1 && j1 <= P.ntot && k0 >= 0 && k0 <= k1 &&
                             k1 <= P.ntot, P.err))
        j0 = j1 = k0 = k1 = 0;
    }
  }
  if constexpr (PART) {
    const int nj = j1 - j0;
    size = nj + k1 - k0;
    int b, e;
    part(size, b, e);
    e = min(e, size);
    b = min(b, e);
    j1 = j0 + min(e, nj);
    j0 += min(b, nj);
    k1 = k0 + max(e - nj, 0);
    k0 += max(b - nj, 0);
  }
  if constexpr (LIMIT)
    if (__reduce_add_sync(kAll, j1 - j0 + k1 - k0) > most) return true;
  const uint32_t rc2m1 = __float_as_uint(B.rc2) - 1u;
#pragma unroll 1
  for (int sg = 0; sg < nseg && !over; ++sg) {
    float ax = pi.x, jsx = 0.f;
    uint32_t c = code;
    int a0 = j0, a1 = j1;
    if (low) {  // slices lo + nx .. nx - 1 as r_j - L, then 0 .. hi
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
    const int stop = scan_range<true, NT, CAP, kRowsUnroll>(P.pos, a0, a1, ax, ay, az, jsx, jsy,
                                                            jsz, rc2m1, c, lst, cnt);
    over = stop >= 0 && (stop < a1 || sg + 1 < nseg);
    if (HALF && over) taken = min(stop, a1) - a0 + (sg ? j1 - j0 : 0);
  }
  return over;
}

// The lists' places in the queue, warps in order, lanes in order, and the
// entries in them.  Returns their number, or -1 where the queue cannot hold them
// (nothing is queued).  over: a list was not enough, which W.overflow keeps.
template <typename Sh>
__device__ __forceinline__ int queue_lists(Sh &W, int cnt, bool over) {
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
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
      W.queue[off + k] = W.list[k * Sh::kThreads + tid];
      W.who[off + k] = (uint8_t)lane;
    }
  __syncthreads();
  return total > Sh::kQueue ? -1 : total;
}

// The queue's pairs, by all threads.
template <bool HALF, int GEN, typename Sh>
__device__ __forceinline__ void evaluate_queue(const Packed &P, const BoxDev &B, const BoxState &S,
                                               Sh &W, int p0, int total) {
#pragma unroll 1
  for (int q = threadIdx.x; q < total; q += Sh::kThreads) {
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
}

// Adds the results to this lane's target in queue order (full stencil).
template <typename Sh>
__device__ __forceinline__ void add_results(const Sh &W, float4 &f) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int r = 0; r < Sh::kRows; ++r) {
    const int q0 = W.off[r][lane], q1 = q0 + W.cnt[r][lane];
#pragma unroll 4
    for (int q = q0; q < q1; ++q) {
      const float4 g = W.res[q];
      f.x += g.x;
      f.y += g.y;
      f.z += g.z;
      f.w += g.w;
    }
  }
}

// A denser place than the lists or the queue hold, half stencil, whose sums have
// no order: after the first lists (queued and evaluated already, if `queued`),
// the lists as they are for fewer targets at a time, and then on from where each
// list was full.
template <int GEN, bool DENSE>
__device__ __forceinline__ void dense_half(const Packed &P, const BoxDev &B, const BoxState &S,
                                           RowsShared<true, DENSE> &W, bool queued, int cnt,
                                           bool over, int taken) {
  using Sh = RowsShared<true, DENSE>;
  constexpr int NT = Sh::kThreads, CAP = Sh::kCap;
  static_assert(4 * Sh::kRows * CAP <= Sh::kQueue, "the queue holds four targets' lists");
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
  const int p0 = (int)blockIdx.x * 32;
  const float4 pi = W.own_pos[lane], vi = W.own_vel[lane];
  int done = 0, size;
  for (;;) {
#pragma unroll 1
    for (int first = queued ? 32 : 0, m = 16; first < 32;) {
      const int total = queue_lists(W, lane >= first && lane < first + m ? cnt : 0, false);
      if (total < 0) {
        m >>= 1;
        continue;
      }
      evaluate_queue<true, GEN>(P, B, S, W, p0, total);
      first += m;
    }
    if (!W.overflow) return;
    __syncthreads();  // all have looked
    if (tid == 0) W.overflow = 0;
    done += taken;
    cnt = taken = 0;
    over = scan_row<true, true, false, NT, CAP>(
        P, B, row, p0 + lane, pi, vi, over,
        [=](int n, int &b, int &e) {
          b = done;
          e = n;
        },
        0, W.list + tid, cnt, size, taken);
    const int total = queue_lists(W, cnt, over);
    queued = total >= 0;
    if (queued) evaluate_queue<true, GEN>(P, B, S, W, p0, total);
  }
}

// Full stencil: the candidates of a warp above which its lists or the queue
// overflow more often than not, so that it does not try.
template <bool DENSE>
constexpr int kRowMost = 32 * (DENSE ? 54 : 30);

// The same for the full stencil, whose sums keep row and slot order: a plane's
// three rows at a time, three warps to a row; where that is too much, one row at
// a time, a ninth to each warp; where that is, parts that their lists and their
// share of the queue hold even if every candidate is a neighbour.
template <int GEN, bool DENSE>
__device__ __forceinline__ void dense_full(const Packed &P, const BoxDev &B, const BoxState &S,
                                           RowsShared<false, DENSE> &W, bool alive, float4 &f) {
  using Sh = RowsShared<false, DENSE>;
  constexpr int NT = Sh::kThreads, CAP = Sh::kCap;
  constexpr int kPart = Sh::kQueue / NT, kRound = kPart * Sh::kRows;
  static_assert(kPart >= 1 && kPart <= CAP - kRowsUnroll, "a part's list never fills");
  // the middle plane's and the middle row's limits; twice as many for the others
  constexpr int kThirdMost = DENSE ? 1070 : 640, kNinthMost = Sh::kQueue / 9 * 2;
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
  const int p0 = (int)blockIdx.x * 32;
  const float4 pi = W.own_pos[lane], vi = W.own_vel[lane];
  int size = 0;
  auto round = [&](int r, int most, auto part) -> bool {
    __syncthreads();  // the results, in the lists' memory, have been added
    if (tid == 0) W.overflow = 0;
    int cnt = 0, taken;
    const bool over = scan_row<false, true, true, NT, CAP>(P, B, r, p0 + lane, pi, vi, alive, part,
                                                           most, W.list + tid, cnt, size, taken);
    const int total = queue_lists(W, cnt, over);
    if (total < 0 || W.overflow) return false;
    evaluate_queue<false, GEN>(P, B, S, W, p0, total);
    __syncthreads();
    if (row == 0) add_results(W, f);
    return true;
  };
  auto split = [&](int r, int k, int parts, int most) -> bool {
    return round(r, most, [=](int n, int &b, int &e) {
      const int each = (n + parts - 1) / parts;
      b = k * each;
      e = b + each;
    });
  };
#pragma unroll 1
  for (int r0 = 0; r0 < Sh::kRows; r0 += 3) {
    if (split(r0 + row / 3, row % 3, 3, r0 == 3 ? kThirdMost : 2 * kThirdMost)) continue;
#pragma unroll 1
    for (int r = r0; r < r0 + 3; ++r) {
      if (split(r, row, Sh::kRows, r == 4 ? kNinthMost : 2 * kNinthMost)) continue;
      const int n = size;  // the same for all warps, which hold the same targets
#pragma unroll 1
      for (int q0 = 0; __any_sync(kAll, q0 < n); q0 += kRound)
        round(r, NT * kPart, [=](int, int &b, int &e) {
          b = q0 + row * kPart;
          e = b + kPart;
        });
    }
  }
}

template <bool HALF, int GEN, bool DENSE>
__global__ void __launch_bounds__(RowsShared<HALF, DENSE>::kThreads,
                                  HALF ? kRowsBlocksHalf : kRowsBlocksFull)
    k_force_rows(Packed P, bool fuse, float *__restrict__ out3) {
  using Sh = RowsShared<HALF, DENSE>;
  constexpr int NT = Sh::kThreads, CAP = Sh::kCap;
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

  // This warp's row, then the queue of all rows.  The limit costs the plain full
  // kernel half a per cent and saves a dense place a scan for nothing; the general
  // ones 1.5 per cent at rho = 1, so that they go without.
  constexpr bool kLimit = !HALF && GEN == 0;
  int cnt = 0, size, taken = 0;
  const bool over =
      scan_row<HALF, false, kLimit, NT, CAP>(P, B, row, p, pi, vi, alive, 0, kRowMost<DENSE>,
                                             W.list + tid, cnt, size, taken);
  const int total = queue_lists(W, cnt, over);
  const bool fits = total >= 0 && !W.overflow;
  float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (HALF) {
    if (total >= 0) evaluate_queue<HALF, GEN>(P, B, S, W, p0, total);
    if (!fits) dense_half<GEN, DENSE>(P, B, S, W, total >= 0, cnt, over, taken);
    if (row != 0) return;
  } else if (fits) {
    evaluate_queue<HALF, GEN>(P, B, S, W, p0, total);
    __syncthreads();
    if (row != 0) return;
    add_results(W, f);
  } else {
    dense_full<GEN, DENSE>(P, B, S, W, alive, f);
    if (row != 0) return;
  }
  // read again, not kept in registers through the queue: the full kernel spilled
  // (59,259 particles, rho = 1: 30.0 us a step; 28.1 so)
  pi = W.own_pos[lane];
  vi = W.own_vel[lane];
  finish_force<HALF>(P, B, S, p, pi, vi, alive, real, fuse, f.x, f.y, f.z, f.w);
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

// The row-parallel kernels win while the direct kernels leave the GPU waiting: the
// slots up to which they serve a box, by its slots per cell.  A step, row-parallel
// over direct, on both sides of each line (percent; rho of the box, thousand slots):
//   full     rho 1    plain 94 (55), 107 (69); Gauss 98 (59), 104 (69); species 94 (55),
//                     108 (69)
//            rho 1.5  96 (59), 105 (70); 92 (59), 101 (70); 97 (59), 106 (70)
//            rho 2    95 (60), 102 (72); 99 (86), 103 (93); 100 (72), 105 (79)
//            rho 3    97 (73), 101 (81); 98 (128), 96 (140); 98 (81), 101 (89)
//            rho 5    98 (110), 104 (135); 85 (149); 92 (122), 98 (135)
//            rho 6    91 (118), 97 (146); 79 (146); 93 (146)
//            rho 7.3  98 (101), 106 (114); 86 (144); 99 (114), 100 (144)
//            rho 8    91 (85), 101 (97); 82 (140); 97 (140)
//            rho 10   92 (106), 96 (138); 75 (138); 90 (138)
//   half     rho 1    94 (79), 103 (110); 99 (91), 101 (110); 99 (91), 101 (110)
//            rho 1.5  100 (128), 104 (156); 97 (128), 101 (156); 99 (128), 103 (156)
//            rho 2    98 (250), 102 (297); 95 (250), 99 (297); 96 (250), 99 (297)
//            rho 3    98 (255), 101 (292); 96 (255), 100 (292); 96 (255), 99 (292)
//            rho 10   92 (244), 97 (298); 91 (244), 95 (298); 90 (244), 94 (298)
// Where a line lies below the crossing, the boxes in between stay on the direct
// kernel they had.  Above about 12 slots per cell the lists overflow too often.
bool rows_pay(const Packed &P, bool half, int gen) {
  struct Limit {
    double per_cell;
    int plain, gauss, other;  // other: several species, or both
  };
  static constexpr Limit kFull[] = {{1.75, 57344, 57344, 57344},   {3.5, 65536, 90112, 73728},
                                    {5.0, 65536, 90112, 90112},    {7.0, 106496, 139264, 139264},
                                    {9.5, 90112, 139264, 139264},  {12.0, 106496, 139264, 139264}};
  static constexpr Limit kHalf[] = {{1.75, 90112, 90112, 90112}, {12.0, 262144, 262144, 262144}};
  const Limit *l = half ? kHalf : kFull, *end = half ? std::end(kHalf) : std::end(kFull);
  while (l != end && !slots_per_cell_at_most(P, l->per_cell)) ++l;
  if (P.nbox != 1 || l == end) return false;
  return P.ntot <= (gen == 0 ? l->plain : gen == kGenGauss ? l->gauss : l->other);
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
