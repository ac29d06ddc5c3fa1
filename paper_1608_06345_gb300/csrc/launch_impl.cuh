// Launcher templates: pick the step shape, set up and launch the kernels of
// one (lattice, storage type, compute type).
#pragma once

#include <algorithm>
#include <atomic>

#include "runtime.h"

namespace lbm {

template <class C>
const Args<C>& args_of(const Instance* inst) {
  if constexpr (std::is_same<C, double>::value) return inst->ad;
  else return inst->af;
}

// Launches a kernel that starts with wait_for_previous_kernel(): it is set up
// while the stream's previous kernel drains, so a chain of steps does not pay
// the whole launch latency in between.  Measured, us per step, without and
// with (plain launches; replayed graph): D2Q37 FP32 300 x 7 5.2 -> 3.2; 3.1 ->
// 2.9, 1000 x 16 5.6 -> 3.0; 3.0 -> 2.8, 256^2 8.2 -> 5.6; 5.9 -> 5.4.  Letting
// the next kernel's blocks in as soon as this one's have all started
// (griddepcontrol.launch_dependents) packs small grids onto few SMs: 1000 x 16
// 4.8.
template <class... P, class... A>
cudaError_t launch_next(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
  if (e != cudaSuccess) cudaGetLastError();  // the caller gets it; a later launch's check must not
  return e;
}

// dynamic shared memory of a step shape: none (STAGE 0, 6), h only (STAGE 3),
// g and h (STAGE 1)
template <int LAT, class S, int STAGE, int BX>
constexpr size_t step_smem() {
  if constexpr (STAGE == 9) return sizeof(unsigned) * (Lat<LAT>::Q - (Lat<LAT>::Q + 1) / 2) * BX;
  return (STAGE == 0 || STAGE == 6) ? 0 : (STAGE == 3 ? 1 : 2) * sizeof(S) * Lat<LAT>::Q * BX;
}

// the dynamic shared-memory opt-in is a per-device function attribute: set
// it once per device (bit d of the mask) for each kernel instance; the mask
// is atomic because host threads may launch concurrently (setting the
// attribute twice is harmless)
template <int LAT, class S, class C, int STAGE, int BX, int MINB, bool IDX32, int ROWS>
cudaError_t step_smem_opt_in(size_t smem) {
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !(configured.load(std::memory_order_acquire) & (1ull << dev))) {
    e = cudaFuncSetAttribute(k_step<LAT, S, C, STAGE, BX, MINB, IDX32, ROWS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_release);
  }
  return cudaSuccess;
}

// rows of a 3D grid that lie within 3 cells of a y or z face
inline long long boundary_rows(int ny, int nz) { return (long long)ny * nz - (long long)(ny - 6) * (nz - 6); }

template <int LAT, class S, class C, int STAGE, int BX, int MINB = 1, bool IDX32 = false>
cudaError_t launch_step_v(const Instance* inst, const void* src, void* dst, const Args<C>& a,
                          bool configure_only = false) {
  constexpr size_t smem = step_smem<LAT, S, STAGE, BX>();
  const unsigned gx = (unsigned)((inst->n[0] + BX - 1) / BX);
  // a 3D grid with interior rows whose byte offsets fit 32 bits (the ROW
  // path): with FP32 storage and 32-bit element indices one launch whose
  // every block takes the ROW path's code with block-uniform row shift
  // tables; otherwise an interior and a boundary launch (measured: the
  // uniform launch is the faster for FP32 storage, the split for 16-bit)
  constexpr long long E = IsS16<S>::value ? 2 * (long long)sizeof(S) : (long long)sizeof(S);
  constexpr bool UNIFORM = Lat<LAT>::D == 3 && IDX32 && sizeof(S) == 4 && !IsS16<S>::value;
  const int ny = inst->n[1], nz = inst->n[2];
  const bool split = Lat<LAT>::D == 3 && ny >= 7 && nz >= 7 && inst->N * E < (1LL << 32) &&
                     boundary_rows(ny, nz) <= 65535;
  // (the choice is made at compile time where it can be, so that no kernel
  // instance is built that a launch never reaches)
  if constexpr (smem != 0) {
    cudaError_t e;
    if constexpr (UNIFORM) {
      e = split ? step_smem_opt_in<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsUniform>(smem)
                : step_smem_opt_in<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsAll>(smem);
    } else {
      e = split ? step_smem_opt_in<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsInterior>(smem)
                : step_smem_opt_in<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsAll>(smem);
      if (e == cudaSuccess && split) e = step_smem_opt_in<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsBoundary>(smem);
    }
    if (e != cudaSuccess) return e;
  }
  if (configure_only) return cudaSuccess;
  const S* s = static_cast<const S*>(src);
  S* d = static_cast<S*>(dst);
  if constexpr (UNIFORM) {
    if (split) {
      return launch_next(k_step<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsUniform>, dim3(gx, (unsigned)ny, (unsigned)nz), BX, smem, inst->stream,
                         s, d, a);
    }
  } else if constexpr (Lat<LAT>::D == 3) {
    if (split) {
      cudaError_t e = launch_next(k_step<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsInterior>,
                                  dim3(gx, (unsigned)(ny - 6), (unsigned)(nz - 6)), BX, smem, inst->stream, s, d, a);
      if (e != cudaSuccess) return e;
      return launch_next(k_step<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsBoundary>, dim3(gx, (unsigned)boundary_rows(ny, nz), 1), BX, smem, inst->stream,
                         s, d, a);
    }
  }
  if constexpr (Lat<LAT>::D == 2 && IDX32 && sizeof(S) < 8) {
    // Rows that are no multiple of 32 cells.  FP32 storage: always (us per
    // step, row-wise and flat: 300 x 7 2.9 / 2.8, 333^2 10.4 / 7.7, 500^2 25.3 /
    // 24.6).  16-bit storage is near its issue bound, so only where the rows
    // start off the 32-byte sectors (8 pairs) and the state leaves the 126 MB
    // of L2: 2999 x 1777 275 / 252; 3000 x 1776, on the sectors, 246 / 252;
    // 2999 x 100, in L2, 14.3 / 15.1.
    const bool flat = IsS16<S>::value ? inst->n[0] % 8 != 0 && 2 * inst->buf_bytes > 126000000
                                      : inst->n[0] % 32 != 0;
    if (flat && inst->N <= 0x7fffffffLL - BX)
      return launch_next(k_step<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsFlat>,
                         dim3((unsigned)((inst->N + BX - 1) / BX), 1, 1), BX, smem, inst->stream, s, d, a);
  }
  return launch_next(k_step<LAT, S, C, STAGE, BX, MINB, IDX32, kRowsAll>, dim3(gx, (unsigned)ny, (unsigned)nz), BX, smem, inst->stream,
                     s, d, a);
}

// Buffers whose element indices (2Q ps; Q ps pairs for 16-bit storage) stay
// below 2^32 index in unsigned 32-bit arithmetic, which takes fewer integer
// instructions per load and store (4096^2 D2Q37 and 256^3 D3Q107 both do)
template <int LAT, class S, class C, int STAGE, int BX, int MINB = 1>
cudaError_t launch_step_t(const Instance* inst, const void* src, void* dst, const Args<C>& a,
                          bool configure_only = false) {
  const long long planes = IsS16<S>::value ? Lat<LAT>::Q : 2LL * Lat<LAT>::Q;
  if (planes * inst->ps < (1LL << 32))
    return launch_step_v<LAT, S, C, STAGE, BX, MINB, true>(inst, src, dst, a, configure_only);
  return launch_step_v<LAT, S, C, STAGE, BX, MINB, false>(inst, src, dst, a, configure_only);
}

// the velocity-split step: 32 cells per block, P warps (static shared memory only)
template <int LAT, class S, class C, int P, int MINB, bool SHARE = false>
cudaError_t launch_step_split(const Instance* inst, const void* src, void* dst, const Args<C>& a,
                              bool configure_only = false) {
  if (configure_only) return cudaSuccess;
  const dim3 grid((unsigned)((inst->n[0] + 31) / 32), (unsigned)inst->n[1], (unsigned)inst->n[2]);
  return launch_next(k_step_split<LAT, S, C, P, MINB, SHARE>, grid, dim3(32, P), 0, inst->stream,
                     static_cast<const S*>(src), static_cast<S*>(dst), a);
}

// the mirror-pair step (stage 8): BX threads, BX / 2 cells per block; HS
// stages h in shared memory (FP32/FP64 storage)
template <int LAT, class S, class C, int BX, int MINB, bool HS, bool IDX32>
cudaError_t launch_step_mirror_v(const Instance* inst, const void* src, void* dst, const Args<C>& a,
                                 bool configure_only) {
  constexpr size_t smem = HS ? sizeof(S) * ((Lat<LAT>::Q - 1) / 2) * BX : 0;
  if constexpr (smem > 48 * 1024) {
    // per-device shared-memory opt-in, as in launch_step_v
    static std::atomic<unsigned long long> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(configured.load(std::memory_order_acquire) & (1ull << dev))) {
      e = cudaFuncSetAttribute(k_step_mirror<LAT, S, C, BX, MINB, IDX32, HS>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_release);
    }
  }
  if (configure_only) return cudaSuccess;
  const dim3 grid((unsigned)((inst->n[0] + BX / 2 - 1) / (BX / 2)), (unsigned)inst->n[1], (unsigned)inst->n[2]);
  return launch_next(k_step_mirror<LAT, S, C, BX, MINB, IDX32, HS>, grid, BX, smem, inst->stream,
                     static_cast<const S*>(src), static_cast<S*>(dst), a);
}

template <int LAT, class S, class C, int BX, int MINB, bool HS>
cudaError_t launch_step_mirror(const Instance* inst, const void* src, void* dst, const Args<C>& a,
                               bool configure_only = false) {
  const long long planes = IsS16<S>::value ? Lat<LAT>::Q : 2LL * Lat<LAT>::Q;
  if (planes * inst->ps < (1LL << 32))
    return launch_step_mirror_v<LAT, S, C, BX, MINB, HS, true>(inst, src, dst, a, configure_only);
  return launch_step_mirror_v<LAT, S, C, BX, MINB, HS, false>(inst, src, dst, a, configure_only);
}

// Candidate shapes of the step per (lattice, storage), tried by the
// autotuner: (stage, cells per block, minimum resident blocks per SM requested
// from the compiler, which caps registers).  Index 0 picks by the grid's size
// among shapes of one rounding (pick), and takes two steps per launch where
// that is the faster way (has_pair_t); its row is what a large grid takes.
// The other indices are the kernel that their row names, on every grid:
//   D2Q37 FP32:        (0,128,4) (0,256,2) (0,64,8) (0,128,1)
//   D2Q37 16-bit:      (6,128,8) (6,128,7) (6,128,6) (6,256,3) (0,128,4) (0,64,8)
//   D2Q37 FP64:        (0,128,1) (0,256,1) (0,64,1)  (4,32,4)  (7,32,4)
//   D3Q107 FP32:       (3,128,3) (3,64,6)  (3,32,12) (4,32,6)  (8,32,8)  (8,64,4)  (3,128,3)
//   D3Q107 FP64:       (7,32,3)  (4,32,3)  (4,32,2)  (7,32,3)
//   D3Q107 16-bit:     (6,64,6)  (9,256,2) (6,32,12) (4,32,6)  (8,32,10) (8,32,12) (6,128,3)
// Stage 4 is the velocity-split step: 4 warps per block of 32 cells; stage 7
// the same with the per-cell coefficients formed once by warp 0 and shared.
// Stage 8 is the mirror-pair step: two lanes per cell (c and -c of every
// pair), h staged in shared memory for FP32.  Stage 9 holds half the 16-bit
// pairs packed in registers and stages the other half in shared memory.  In FP32 the
// moments of stages 4, 7 and 8 are summed in another order, so their results
// differ from the other shapes' by rounding; in FP64 every shape sums them in
// the order of stage 4.  Index 0's shapes have the rounding of the batched
// pool's, so a pooled instance's result is bitwise that of a lone one.
struct ShapeRow {
  int stage, bx, minb;
  bool operator==(const ShapeRow& o) const { return stage == o.stage && bx == o.bx && minb == o.minb; }
};

template <int LAT, class S>
struct StepShapes {
  static constexpr int count =
      (LAT == 0) ? (sizeof(S) == 8 ? 5 : (sizeof(S) == 2 ? 6 : 4)) : (sizeof(S) == 8 ? 4 : 7);
  static ShapeRow get(int k) {
    static const ShapeRow s2[4] = {{0, 128, 4}, {0, 256, 2}, {0, 64, 8}, {0, 128, 1}};
    static const ShapeRow s2h[6] = {{6, 128, 8}, {6, 128, 7}, {6, 128, 6}, {6, 256, 3}, {0, 128, 4}, {0, 64, 8}};
    static const ShapeRow s2d[5] = {{0, 128, 1}, {0, 256, 1}, {0, 64, 1}, {4, 32, 4}, {7, 32, 4}};
    static const ShapeRow s3f[7] = {{3, 128, 3}, {3, 64, 6}, {3, 32, 12}, {4, 32, 6}, {8, 32, 8}, {8, 64, 4}, {3, 128, 3}};
    static const ShapeRow s3d[4] = {{7, 32, 3}, {4, 32, 3}, {4, 32, 2}, {7, 32, 3}};
    static const ShapeRow s3h[7] = {{6, 64, 6}, {9, 256, 2}, {6, 32, 12}, {4, 32, 6}, {8, 32, 10}, {8, 32, 12}, {6, 128, 3}};
    if (LAT == 0) return sizeof(S) == 8 ? s2d[k] : (sizeof(S) == 2 ? s2h[k] : s2[k]);
    return sizeof(S) == 4 ? s3f[k] : (sizeof(S) == 8 ? s3d[k] : s3h[k]);
  }
  // the shape of one step of this instance with index k
  static ShapeRow pick(const Instance* inst, int k) {
    if (k != 0) return get(k);
    if constexpr (LAT == 0 && sizeof(S) == 8) {
      // a tube of a few blocks waits on one thread's chain of 560 FP64
      // instructions per cell: split it while every SM has at most two
      // 32-cell blocks (1000 x 4: 22.6 -> 9.4 us; 1000 x 16, 512 blocks:
      // 22.8 us, split 30.2)
      if ((long long)((inst->n[0] + 31) / 32) * inst->n[1] <= 2LL * device_sms()) return {4, 32, 4};
    } else if constexpr (LAT == 1 && sizeof(S) < 8) {
      // Blocks of 32 cells where they leave a seventh fewer threads past the
      // row ends than blocks of 64 (us per step, 64 and 32 cells: FP32 32^3
      // 14.6 / 7.7, 96^3 291 / 271).  The line leaves out rows of 193 cells,
      // 256 and 224 threads, where the two are level: FP32 860 / 856, FP16
      // storage 193 x 96 x 96 352 / 363, BF16 380 / 376.  Else 128 cells with
      // FP32 storage where they pad no more (256 x 128 x 128 1221 -> 1190, 193
      // x 130 x 97 860 -> 830, 112 x 96 x 80 286 -> 267).
      auto padded = [&](int bx) { return (inst->n[0] + bx - 1) / bx * bx; };
      constexpr int stage = sizeof(S) == 4 ? 3 : 6;
      if (7 * padded(32) <= 6 * padded(64)) return {stage, 32, 12};
      if (sizeof(S) == 4 && padded(128) == padded(64)) return {stage, 128, 3};
      return {stage, 64, 6};
    }
    // D3Q107 FP64: the split with shared coefficients is the fastest at every
    // size (one thread per cell with cp.async staging 1000 x 16 x 16 983 ->
    // 779 us, 256 x 128 x 128 14.1 -> 12.7 ms, 32^3 273 -> 116)
    return get(0);
  }
};

template <int LAT, class S>
int shape_count_t() { return StepShapes<LAT, S>::count; }

template <int LAT, class S>
void shape_get_t(const Instance* inst, int k, int* stage, int* bx, int* minb) {
  const ShapeRow r = inst ? StepShapes<LAT, S>::pick(inst, k) : StepShapes<LAT, S>::get(k);
  *stage = r.stage;
  *bx = r.bx;
  *minb = r.minb;
}

template <int LAT, class S, class C>
cudaError_t launch_step_shape(const Instance* inst, const void* src, void* dst, bool configure_only = false) {
  const Args<C>& a = args_of<C>(inst);
  const ShapeRow r = StepShapes<LAT, S>::pick(inst, inst->shape.index);
  if constexpr (LAT == 0 && sizeof(S) == 8) {
    if (r == ShapeRow{0, 128, 1}) return launch_step_t<LAT, S, C, 0, 128>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 256, 1}) return launch_step_t<LAT, S, C, 0, 256>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 64, 1}) return launch_step_t<LAT, S, C, 0, 64>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{4, 32, 4}) return launch_step_split<LAT, S, C, 4, 4>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{7, 32, 4}) return launch_step_split<LAT, S, C, 4, 4, true>(inst, src, dst, a, configure_only);
  } else if constexpr (LAT == 0 && sizeof(S) == 2) {
    if (r == ShapeRow{6, 128, 8}) return launch_step_t<LAT, S, C, 6, 128, 8>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{6, 128, 7}) return launch_step_t<LAT, S, C, 6, 128, 7>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{6, 128, 6}) return launch_step_t<LAT, S, C, 6, 128, 6>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{6, 256, 3}) return launch_step_t<LAT, S, C, 6, 256, 3>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 128, 4}) return launch_step_t<LAT, S, C, 0, 128, 4>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 64, 8}) return launch_step_t<LAT, S, C, 0, 64, 8>(inst, src, dst, a, configure_only);
  } else if constexpr (LAT == 0) {
    if (r == ShapeRow{0, 128, 4}) return launch_step_t<LAT, S, C, 0, 128, 4>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 256, 2}) return launch_step_t<LAT, S, C, 0, 256, 2>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 64, 8}) return launch_step_t<LAT, S, C, 0, 64, 8>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{0, 128, 1}) return launch_step_t<LAT, S, C, 0, 128, 1>(inst, src, dst, a, configure_only);
  } else if constexpr (sizeof(S) == 4) {
    if (r == ShapeRow{3, 128, 3}) return launch_step_t<LAT, S, C, 3, 128, 3>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{3, 64, 6}) return launch_step_t<LAT, S, C, 3, 64, 6>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{3, 32, 12}) return launch_step_t<LAT, S, C, 3, 32, 12>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{4, 32, 6}) return launch_step_split<LAT, S, C, 4, 6>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{8, 32, 8}) return launch_step_mirror<LAT, S, C, 64, 8, true>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{8, 64, 4}) return launch_step_mirror<LAT, S, C, 128, 4, true>(inst, src, dst, a, configure_only);
  } else if constexpr (sizeof(S) == 8) {
    if (r == ShapeRow{7, 32, 3}) return launch_step_split<LAT, S, C, 4, 3, true>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{4, 32, 3}) return launch_step_split<LAT, S, C, 4, 3>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{4, 32, 2}) return launch_step_split<LAT, S, C, 4, 2>(inst, src, dst, a, configure_only);
  } else {
    if (r == ShapeRow{6, 64, 6}) return launch_step_t<LAT, S, C, 6, 64, 6>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{9, 256, 2}) return launch_step_t<LAT, S, C, 9, 256, 2>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{6, 32, 12}) return launch_step_t<LAT, S, C, 6, 32, 12>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{4, 32, 6}) return launch_step_split<LAT, S, C, 4, 6>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{8, 32, 10}) return launch_step_mirror<LAT, S, C, 64, 10, false>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{8, 32, 12}) return launch_step_mirror<LAT, S, C, 64, 12, false>(inst, src, dst, a, configure_only);
    if (r == ShapeRow{6, 128, 3}) return launch_step_t<LAT, S, C, 6, 128, 3>(inst, src, dst, a, configure_only);
  }
  return cudaErrorInvalidConfiguration;  // no row is without a kernel
}

// ---------------------------------------------------------------------------
// two steps in one launch
// ---------------------------------------------------------------------------
// Whether steps go two per launch: shape index 0 leaves the choice open, and it
// is the faster way.  Measured against the share of pair_grid: 0.44 (384^2)
// 0.79 of the single step's speed, 0.57 (512^2) 1.03, 0.60 (100 x 6000) 1.18,
// 0.72 (768^2) 1.15, 0.80 (1024^2) 1.19, 0.94 (4096^2) 1.25.
template <int LAT, class S, class C>
bool has_pair_t(const Instance* inst) {
  if constexpr (LAT == 0 && std::is_same<S, float>::value) {
    return inst->shape.index == 0 && inst->pair.share >= 0.6;
  } else {
    return false;
  }
}

template <bool IDX32>
cudaError_t launch_pair_v(const Instance* inst, const void* src, void* dst, bool configure_only) {
  auto kern = k_step_pair<IDX32>;
  constexpr size_t smem = PairRing::bytes(2);
  static std::atomic<unsigned long long> configured{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !(configured.load(std::memory_order_acquire) & (1ull << dev))) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_release);
  }
  if (configure_only) return cudaSuccess;
  const PairGrid& g = inst->pair;
  return launch_next(kern, dim3((unsigned)g.strips, (unsigned)g.bands), 4 * kPairW, smem, inst->stream,
                     static_cast<const float*>(src), static_cast<float*>(dst), inst->af, g.width, inst->wait_tries);
}

template <int LAT, class S, class C>
cudaError_t launch_pair_t(const Instance* inst, const void* src, void* dst, bool configure_only) {
  if constexpr (LAT == 0 && std::is_same<S, float>::value) {
    if (2LL * Lat<LAT>::Q * inst->ps < (1LL << 32)) return launch_pair_v<true>(inst, src, dst, configure_only);
    return launch_pair_v<false>(inst, src, dst, configure_only);
  } else {
    return cudaErrorInvalidConfiguration;
  }
}

template <int LAT, class S, class C>
cudaError_t launch_step_pair(const Instance* inst, const void* src, void* dst) {
  return launch_pair_t<LAT, S, C>(inst, src, dst, false);
}

// sets the kernel attributes of the shape, and of the two-step kernel where
// the instance takes it, on the current device without launching (done
// before a graph capture)
template <int LAT, class S, class C>
cudaError_t configure_step_t(const Instance* inst) {
  if (has_pair_t<LAT, S, C>(inst)) {
    const cudaError_t e = launch_pair_t<LAT, S, C>(inst, nullptr, nullptr, true);
    if (e != cudaSuccess) return e;
  }
  return launch_step_shape<LAT, S, C>(inst, nullptr, nullptr, true);
}

template <int LAT, class S, class C>
cudaError_t launch_step_plain(const Instance* inst, const void* src, void* dst) {
  return launch_step_shape<LAT, S, C>(inst, src, dst, false);
}

// the finite-difference step (lam = dt/dx)
template <int LAT, class S, class C, int BX, int BY, int BZ, int MINB>
cudaError_t launch_step_fd_tile(const Instance* inst, const void* src, void* dst, double lam) {
  const dim3 grid((unsigned)((inst->n[0] + BX - 1) / BX), (unsigned)((inst->n[1] + BY - 1) / BY),
                  (unsigned)((inst->n[2] + BZ - 1) / BZ));
  return launch_next(k_step_fd_tile<LAT, S, C, BX, BY, BZ, MINB>, grid, dim3(BX, BY, BZ), 0, inst->stream,
                     static_cast<const S*>(src), static_cast<S*>(dst), args_of<C>(inst), static_cast<C>(lam * inst->table.r));
}
// one thread per cell holding its 2Q values, BX cells of a row per block
template <int LAT, class S, class C, int BX>
cudaError_t launch_step_fd_row(const Instance* inst, const void* src, void* dst, double lam) {
  const dim3 grid((unsigned)((inst->n[0] + BX - 1) / BX), (unsigned)inst->n[1], (unsigned)inst->n[2]);
  return launch_next(k_step_fd<LAT, S, C, BX>, grid, BX, 0, inst->stream,
                     static_cast<const S*>(src), static_cast<S*>(dst), args_of<C>(inst), static_cast<C>(lam * inst->table.r));
}

// The faster of the two per lattice, storage and size (large grids: figures at
// k_step_fd_tile).  us per step, tile / row.
//   A tile's block is long and large, so grids of few tiles leave SMs idle that
// the row kernel's smaller blocks would use: D3Q107 FP32 64 x 64 x 6 (24576
// cells) 60 / 36, 40 x 100 x 5 (20000) 59 / 36, 1000 x 4 x 4 (16000) 59 / 37,
// 32^3 (32768) 74 / 72, 2000 x 4 x 4 (32000) 54 / 57, 40^3 88 / 137; FP16
// storage 40 x 100 x 5 45 / 31, 32^3 57 / 63; FP64 32^3 (128 tiles) 553 / 380,
// 48^3 (432) 878 / 1238; D2Q37 FP16 storage 256^2 (256 tiles) 13.1 / 11.1, 512^2
// (1024) 27.1 / 29.6.
//   Nor does it pay where the grid is so thin along y or z that its tiles hold
// more threads without a cell than the row kernel's blocks, by a factor that
// depends on the tile's gain on full ones: D3Q107 FP32 2.8 (1000 x 9 x 5) 80 /
// 113, 3.5 (4000 x 3 x 3) 66 / 59, 3.8 (300 x 300 x 1) 230 / 168, 32 (20000 x 1 x
// 1) 194 / 34; FP16 storage 1.28 (300 x 300 x 3) 308 / 345, 1.31 (1000 x 40 x
// 3) 187 / 138, 1.5 (300 x 5 x 300) 518 / 448, 32 (20000 x 1 x 1) 171 / 28; D2Q37 FP16 storage
// 2 (100000 x 4) 46 / 53, 4 (100000 x 2) 31 / 24, 8 (100000 x 1) 26 / 13.  FP64 is
// bound by the FP64 pipe, whose time is that of the warps with a cell (16 x 2 of
// a tile, 32 of a row): 1.06 times as many (300 x 9 x 300) 6740 / 7189, 1.09 (1000
// x 9 x 5) 561 / 619, 1.27 (300 x 3 x 300) 2797 / 2412, 2 (20000 x 1 x 1) 563 / 219.
template <int LAT, class S, class C>
cudaError_t launch_step_fd_t(const Instance* inst, const void* src, void* dst, double lam) {
  auto blocks = [&](long long bx, int by, int bz) {
    return (inst->n[0] + bx - 1) / bx * ((inst->n[1] + by - 1) / by) * ((inst->n[2] + bz - 1) / bz);
  };
  if constexpr (LAT == 0) {
    if constexpr (IsS16<S>::value) {
      const long long tiles = blocks(32, 8, 1);
      if (tiles >= 3 * device_sms() && tiles * 256 <= 2 * 128 * blocks(128, 1, 1))
        return launch_step_fd_tile<LAT, S, C, 32, 8, 1, 3>(inst, src, dst, lam);
    }
    return launch_step_fd_row<LAT, S, C, 128>(inst, src, dst, lam);
  } else {
    if constexpr (sizeof(S) == 8) {
      const long long tiles = blocks(16, 4, 4);
      if (tiles >= 2 * device_sms() && 10 * blocks(16, 2, 1) <= 11 * blocks(32, 1, 1) &&
          2 * tiles * 256 <= 5 * 64 * blocks(64, 1, 1))
        return launch_step_fd_tile<LAT, S, C, 16, 4, 4, 2>(inst, src, dst, lam);
    } else {
      const long long tiles = blocks(16, 8, 4), row = 64 * blocks(64, 1, 1);
      if (inst->N >= 200LL * device_sms() && 10 * tiles * 512 <= (IsS16<S>::value ? 13 : 30) * row)
        return launch_step_fd_tile<LAT, S, C, 16, 8, 4, 2>(inst, src, dst, lam);
    }
    return launch_step_fd_row<LAT, S, C, 64>(inst, src, dst, lam);
  }
}

// pool: the shape of the batched step per (lattice, storage)
template <int LAT, class S>
struct PoolShape {
  static constexpr int kStage = (LAT == 0) ? 0 : (sizeof(S) == 4 ? 3 : (sizeof(S) == 8 ? 1 : 6));
  static constexpr int kBX = (LAT == 0) ? 128 : 64;
  // resident blocks per SM asked of the compiler, as in the step's shapes
  // (D2Q37 FP32 took 138 registers, 3 blocks; 20 tubes of up to 12000 x 4 cells
  // served in 11.0 -> 10.4 ms with 4)
  static constexpr int kMinB = sizeof(S) == 8 ? 1 : (LAT == 0 ? 4 : 6);
};

template <int LAT, class S, class C>
cudaError_t launch_pool_step_t(const PoolLaunch& pl) {
  using PS = PoolShape<LAT, S>;
  auto kern = k_pool_step<LAT, S, C, PS::kStage, PS::kBX, PS::kMinB>;
  // the shared-memory opt-in was set by pool_grid_t at pool creation (outside
  // any stream capture)
  const size_t smem = step_smem<LAT, S, PS::kStage, PS::kBX>();
  return launch_next(kern, pl.grid, PS::kBX, smem, pl.stream,
                     static_cast<const PoolSlot<C>*>(pl.slots), pl.tiles, pl.ntiles);
}

template <class C>
cudaError_t launch_pool_advance_t(const PoolLaunch& pl) {
  const int t = 128;
  return launch_next(k_pool_advance<C>, (pl.nslots + t - 1) / t, t, 0, pl.stream,
                     static_cast<PoolSlot<C>*>(pl.slots), pl.nslots);
}

// persistent grid of the batched step: resident blocks per SM x SMs
template <int LAT, class S, class C>
int pool_grid_t() {
  using PS = PoolShape<LAT, S>;
  const size_t smem = step_smem<LAT, S, PS::kStage, PS::kBX>();
  auto kern = k_pool_step<LAT, S, C, PS::kStage, PS::kBX, PS::kMinB>;
  if (smem && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return 0;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PS::kBX, smem) != cudaSuccess) return 0;
  return sms * (per_sm > 0 ? per_sm : 1);
}

template <int LAT, class S>
constexpr int pool_tile_cells() { return PoolShape<LAT, S>::kBX; }

inline unsigned blocks_for(long long N, int t) { return (unsigned)((N + t - 1) / t); }


template <int LAT, class S, class C>
cudaError_t launch_init_t(const Instance* inst, void* dst, const double* rho, const double* u, const double* T) {
  constexpr int kT = 128;
  if (inst->N == 0) return cudaSuccess;
  k_init<LAT, S, C><<<blocks_for(inst->N, kT), kT, 0, inst->stream>>>(static_cast<S*>(dst), rho, u, T, inst->N,
                                                                      args_of<C>(inst), inst->rho0, inst->T0);
  return cudaGetLastError();
}


template <int LAT, class S, class C>
cudaError_t launch_moments_t(const Instance* inst, const void* src, double* rho, double* u, double* T) {
  constexpr int kT = 128;
  if (inst->N == 0) return cudaSuccess;
  k_moments<LAT, S, C><<<blocks_for(inst->N, kT), kT, 0, inst->stream>>>(
      static_cast<const S*>(src), rho, u, T, inst->N, args_of<C>(inst), inst->rho0, inst->T0);
  return cudaGetLastError();
}


// Blocks of 64 threads while the grid takes no more of them than there are
// partials (262144 cells at 4 cells per thread, 65536 in FP64), so that few
// cells are spread over many SMs; else two blocks of 256 per SM, all resident
// at once.  us per launch (k_conserve_partial), one block of 256 threads per
// 256 cells up to 6 per SM -> this: D2Q37 FP32 4000 cells 20.7 -> 14.6, 300^2
// 24.1 -> 18.6, 300000 cells 41.2 -> 32.9, 1024^2 96.5 -> 60.4, 2048^2 211 ->
// 203; FP16 storage 600000 cells 63.7 -> 39.2, 2048^2 182 -> 179; FP64 40000 cells
// 26.8 -> 18.6; D3Q107 FP32 48000 cells 40.0 -> 34.1, 128 x 128 x 127 377 ->
// 297.
template <int LAT, class S>
cudaError_t launch_conserve_t(const Instance* inst, const void* src, double* partial, int* nblocks) {
  constexpr int V = totals_load<S>();
  const S* s = static_cast<const S*>(src);
  if (inst->N <= 64LL * V * kRedMaxBlocks) {
    *nblocks = (int)((inst->N + 64 * V - 1) / (64 * V));
    k_conserve_partial<LAT, S, 64><<<*nblocks, 64, 0, inst->stream>>>(s, inst->N, inst->ad, inst->af, partial);
  } else {
    *nblocks = std::min(2 * device_sms(), kRedMaxBlocks);
    k_conserve_partial<LAT, S, 256><<<*nblocks, 256, 0, inst->stream>>>(s, inst->N, inst->ad, inst->af, partial);
  }
  return cudaGetLastError();
}


}  // namespace lbm
