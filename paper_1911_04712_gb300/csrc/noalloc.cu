// dpd_forces_noalloc: pair forces on a caller-provided state without any
// device allocation.
//
// Some callers cannot allocate device memory at the point where they need
// forces: code running inside a host callback or a custom allocator, a
// framework that has handed every byte of device memory to its own pool,
// or a real-time loop that must not hit cudaMalloc's implicit device
// synchronisation.  This entry point serves them: all the scratch it needs
// (float4 copies of the state, the cell counts and starts, the reorder keys)
// lives in one file-scope static device array of fixed size, reserved when
// the library is loaded and held by every GPU that loads it until the
// process exits.  The caller passes only its inputs and its output.
//
// The array's name is a host-side stand-in in host code, not a device
// address; the device address is looked up with cudaGetSymbolAddress once
// per device, on that device's first call (so that first call should come
// before any stream capture).  Every call shares the one array and leaves
// its contents behind; the counts that must start at zero are cleared at the
// start of each call.  Calls whose work overlaps on the GPU (different
// streams, or different host threads) race on the array and must be
// serialised by the caller.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <mutex>

#include "dpd.h"
#include "engine.h"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace dpd {

namespace {

constexpr int kNaMaxParticles = DPD_NOALLOC_MAX_PARTICLES;
constexpr int kNaMaxCells = DPD_NOALLOC_MAX_CELLS;
constexpr int kNaMaxSlices = kNaMaxCells * kSlicesX;  // entries of the cell list
constexpr int kNaScanTiles = (kNaMaxSlices + 1 + kScanTile - 1) / kScanTile;
constexpr size_t kNaCellCap = (size_t)kNaScanTiles * kScanTile;

constexpr size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
constexpr size_t kOffPos = 0;
constexpr size_t kOffVel = kOffPos + align256(sizeof(float4) * kNaMaxParticles);
constexpr size_t kOffFrc = kOffVel + align256(sizeof(float4) * kNaMaxParticles);
constexpr size_t kOffPos2 = kOffFrc + align256(sizeof(float4) * kNaMaxParticles);
constexpr size_t kOffVel2 = kOffPos2 + align256(sizeof(float4) * kNaMaxParticles);
constexpr size_t kOffCellOf = kOffVel2 + align256(sizeof(float4) * kNaMaxParticles);
constexpr size_t kOffSlotIn = kOffCellOf + align256(sizeof(int) * kNaMaxParticles);
constexpr size_t kOffKey = kOffSlotIn + align256(sizeof(int) * kNaMaxParticles);
constexpr size_t kOffCount = kOffKey + align256(sizeof(int) * kNaMaxParticles);
constexpr size_t kOffStart = kOffCount + align256(sizeof(int) * kNaCellCap);
constexpr size_t kOffBsum = kOffStart + align256(sizeof(int) * kNaCellCap);
constexpr size_t kOffState = kOffBsum + align256(sizeof(int) * kNaScanTiles);
constexpr size_t kOffErr = kOffState + align256(sizeof(BoxState));
constexpr size_t kScratchBytes = kOffErr + align256(sizeof(unsigned));

}  // namespace

// The scratch: about 3.5 MB for 32768 particles and 32767 cells (two x slices each).
static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// The whole rebuild of one call in one launch: counts and error word cleared,
// the inputs loaded and counted (Sec. 3.2), scan, keys and reorder, by one
// thread-block cluster whose barriers stand where the separate kernels have
// launches.  What bounds a call is launches: for n = 1,536 eight or nine small
// kernels took 35 us on the GPU; this one takes 10.9 and the force kernel 7.4, a
// call among others 17.9 on the GPU and 21 with the host's work.
constexpr int kNaBlocks = 8;  // the portable cluster size
constexpr int kNaThreads = 1024;
constexpr int kNaAll = kNaBlocks * kNaThreads;
constexpr int kNaQuads = (int)(kNaCellCap / 4 + kNaAll - 1) / kNaAll;  // per thread, at most

__global__ void __cluster_dims__(kNaBlocks, 1, 1) __launch_bounds__(kNaThreads, 1)
    k_noalloc_bin(Packed P, const float *__restrict__ pos3, const float *__restrict__ vel3,
                  unsigned long long step) {
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ int wsum[32];
  __shared__ int block_total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gt = (int)blockIdx.x * kNaThreads + tid;
  const int quads_all = scan_tiles(P.ncell) * (kScanTile / 4);
  const int quads = (quads_all + kNaAll - 1) / kNaAll;  // a run of cells per thread
  int4 *c4 = reinterpret_cast<int4 *>(P.count) + (size_t)gt * quads;
  int4 *s4 = reinterpret_cast<int4 *>(P.start) + (size_t)gt * quads;
  for (int k = 0; k < quads && gt * quads + k < quads_all; ++k) c4[k] = make_int4(0, 0, 0, 0);
  if (gt == 0) {
    *P.st = BoxState{step, 0ll, 0, 1};
    *P.err = 0u;
  }
  cluster.sync();

  const BoxDev &B = P.single;
  for (int i = gt; i < P.ntot; i += kNaAll) {
    float4 x, v;
    load_particle(P, i, pos3, vel3, B.L[0], B.L[1], B.L[2], nullptr, 1, x, v);
    integrate_one(P, B, i, x, v, 0.f, 0.f, 0.f, false, false);
  }
  cluster.sync();

  // exclusive scan of the counts
  int4 q[kNaQuads];
  int sum = 0;
#pragma unroll
  for (int k = 0; k < kNaQuads; ++k) {
    q[k] = make_int4(0, 0, 0, 0);
    if (k < quads && gt * quads + k < quads_all) q[k] = c4[k];
    sum += q[k].x + q[k].y + q[k].z + q[k].w;
  }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += t;
    }
    wsum[lane] = w;
    if (lane == 31) block_total = w;
  }
  cluster.sync();
  int other = 0;  // totals of the blocks before this one
  if (lane < (int)cluster.block_rank()) other = *cluster.map_shared_rank(&block_total, lane);
  int run = incl - sum + (warp > 0 ? wsum[warp - 1] : 0) + __reduce_add_sync(0xffffffffu, other);
#pragma unroll
  for (int k = 0; k < kNaQuads; ++k)
    if (k < quads && gt * quads + k < quads_all) {
      int4 o;
      o.x = run;
      o.y = o.x + q[k].x;
      o.z = o.y + q[k].y;
      o.w = o.z + q[k].z;
      s4[k] = o;
      run = o.w + q[k].w;
    }
  cluster.sync();

  for (int p = gt; p < P.ntot; p += kNaAll) bin_key(P, p);
  cluster.sync();
  for (int p = gt; p < P.ntot; p += kNaAll) bin_scatter<true>(P, p, false);
}

// Device address of the scratch on each device, looked up once per device
// and kept for the life of the process (a cudaDeviceReset, which may load
// the module again at another address, is not supported).
static unsigned char *scratch_address(int device, int *status) {
  static std::mutex mu;
  static unsigned char *addr[64] = {nullptr};
  std::lock_guard<std::mutex> g(mu);
  if (device < 0 || device >= 64) {
    *status = set_error(DPD_ERR_CUDA, "device ordinal %d out of range", device);
    return nullptr;
  }
  if (!addr[device]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e == cudaSuccess) e = prepare_device();  // launch attributes of the force kernels
    if (e != cudaSuccess || !p) {
      *status = set_error(DPD_ERR_CUDA, "preparing dpd_forces_noalloc: %s",
                          cudaGetErrorString(e));
      return nullptr;
    }
    addr[device] = static_cast<unsigned char *>(p);
  }
  *status = DPD_OK;
  return addr[device];
}

}  // namespace dpd

extern "C" int dpd_forces_noalloc(int64_t n, const float *pos, const float *vel,
                                  const double box[3], double a, double gamma, double kT,
                                  double rc, double dt, uint64_t seed, uint64_t step,
                                  float *force, void *stream) {
  using namespace dpd;
  clear_error();
  if (!box) return set_error(DPD_ERR_ARG, "null box");
  if (n < 0) return set_error(DPD_ERR_ARG, "negative particle count");
  if (n > kNaMaxParticles)
    return set_error(DPD_ERR_ARG,
                     "dpd_forces_noalloc handles at most %d particles (got %lld); use the "
                     "allocating context API for larger systems",
                     kNaMaxParticles, (long long)n);
  BoxParams bp{};
  for (int k = 0; k < 3; ++k) bp.L[k] = box[k];
  bp.a = a;
  bp.gamma = gamma;
  bp.kT = kT;
  bp.rc = rc;
  bp.dt = dt;
  bp.mass = 1.0;
  bp.kexp = 1.0;
  bp.fb_flow = 2;
  bp.seed = seed;
  int nc[3];
  int rc_ = check_params(bp, nc);
  if (rc_) return rc_;
  const int64_t ncell = (int64_t)nc[0] * nc[1] * nc[2];  // x slices of the cells
  if (ncell > kNaMaxSlices)
    return set_error(DPD_ERR_ARG,
                     "dpd_forces_noalloc handles at most %d cells (box has %lld); use the "
                     "allocating context API for larger boxes",
                     kNaMaxCells, (long long)(ncell / kSlicesX));
  if (n == 0) return DPD_OK;
  if (!pos || !vel || !force) return set_error(DPD_ERR_ARG, "null device pointer");

  int dev = -1;
  DPD_CUDA_TRY(cudaGetDevice(&dev));
  int status = DPD_OK;
  unsigned char *base = scratch_address(dev, &status);
  if (!base) return status;

  cudaStream_t s = (cudaStream_t)stream;
  Packed P{};
  P.pos = reinterpret_cast<float4 *>(base + kOffPos);
  P.vel = reinterpret_cast<float4 *>(base + kOffVel);
  P.frc = reinterpret_cast<float4 *>(base + kOffFrc);
  P.pos2 = reinterpret_cast<float4 *>(base + kOffPos2);
  P.vel2 = reinterpret_cast<float4 *>(base + kOffVel2);
  P.cellOf = reinterpret_cast<int *>(base + kOffCellOf);
  P.slotIn = reinterpret_cast<int *>(base + kOffSlotIn);
  P.keyTmp = reinterpret_cast<int *>(base + kOffKey);
  P.count = reinterpret_cast<int *>(base + kOffCount);
  P.start = reinterpret_cast<int *>(base + kOffStart);
  P.bsum = reinterpret_cast<int *>(base + kOffBsum);
  P.boxes = nullptr;
  P.pbase = nullptr;
  P.st = reinterpret_cast<BoxState *>(base + kOffState);
  P.err = reinterpret_cast<unsigned *>(base + kOffErr);
  P.ntot = (int)n;
  P.ncell = (int)ncell;
  P.nbox = 1;
  P.single = make_box_dev(bp, 0, 0, (int)n);

  k_noalloc_bin<<<kNaBlocks, kNaThreads, 0, s>>>(P, pos, vel, (unsigned long long)step);
  DPD_CUDA_TRY(cudaGetLastError());
  if (rows_pay(P, false, 0)) {
    DPD_CUDA_TRY(launch_force_rows(P, false, 0, false, s, force));
  } else {
    DPD_CUDA_TRY(launch_force(P, StepConfig{}, s));
    DPD_CUDA_TRY(launch_gather(P, 0, 0, (int)n, nullptr, nullptr, force, s));
  }
#if defined(DPD_CHECKED) && DPD_CHECKED
  // checked build: read the error word back (the normal build does not wait)
  unsigned h = 0;
  DPD_CUDA_TRY(cudaMemcpyAsync(&h, P.err, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  DPD_CUDA_TRY(cudaStreamSynchronize(s));
  if (h & kErrBounds)
    return set_error(DPD_ERR_INTERNAL, "a kernel's index check failed (checked build)");
#endif
  return DPD_OK;
}
