// Host-side launch wrappers of the device kernels (one translation unit per
// precision instantiates them).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "lbm_layout.h"

namespace lbmk {

// Strip widths of a tiling (threads per CTA of the step kernels).
inline bool valid_bx(int bx) { return bx == 32 || bx == 64 || bx == 128; }

// Strip widths the staged kernel also runs, for cases whose whole row is
// one strip of that width (their own chains, see lbm_api.cu).
inline bool row_bx(int bx) { return bx == 96 || bx == 192 || bx == 256; }

// PLAIN, here and below: in FP64, the kernels without the short forms of
// lbm_math.cuh (strips of 32, 64 and 128 columns), which handles with reverse
// mode run.  A template and not a branch: a launch-uniform branch cost the
// register kernel its registers (1536 x 1024 with walls 817 -> 906 us per step).
// tma: use the staged kernel (every case must have nx a multiple
// of 16 bytes of T and nx >= 4), else the register-pipelined kernel.
template <typename T, bool PLAIN>
cudaError_t launch_step(const StepArgs<T>& a, int bx, bool coupled, int mode, bool tma,
                        int n_items, cudaStream_t s);

// Persistent register-path kernel (cooperative launch): nsteps steps in one
// launch; grid = min(n_items, co-resident CTAs).  count/gen: grid-barrier
// words (zero-initialised, device).
template <typename T, bool PLAIN>
cudaError_t launch_persistent(const StepArgs<T>& a, int bx, bool coupled, int n_items,
                              int nsteps, int flip, unsigned int* count, unsigned int* gen,
                              cudaStream_t s);

// Variants of the chip-resident kernel: nt threads per CTA with r nodes each,
// pc cells of shared memory (nodes and their two-node surround), nx rim
// triples at most, per_sm CTAs per SM.  The first that holds a batch runs it.
// Measured, us per step over 256 steps:
//   FP32 coupled     128x64  256x128  384x192  512x256
//   256 x 1, 2/SM     1.68     2.05      -        -     (more CTAs: rims overlap)
//   512 x 1, 1/SM     1.71     2.18      -        -
//   512 x 2, 1/SM     1.77     2.24     2.60     3.73
//   448 x 2, 1/SM     1.73     2.23     2.97     4.26
//   896 x 1, 1/SM     1.85     2.34     2.73     4.02   (72 registers)
// The vortex holds twice the nodes (g alone): 256^2 2.31 with 512 x 1, 512^2
// 4.28 with 896 x 2.  FP64 is bound by its pipe (128x64: 14.2, 256x128: 26.5);
// spare threads change nothing there.
struct ResVariant {
  int nt, r, pc, nx, per_sm;
};
constexpr int kResVariants = 2;
constexpr ResVariant kRes32[kResVariants] = {{256, 1, 448, 384, 2}, {512, 2, 1296, 640, 1}};
constexpr ResVariant kRes64[kResVariants] = {{256, 1, 448, 384, 1}, {256, 2, 704, 512, 1}};
constexpr ResVariant kRes32V[kResVariants] = {{512, 1, 784, 512, 1}, {896, 2, 2304, 768, 1}};
constexpr ResVariant kRes64V[kResVariants] = {{512, 1, 784, 512, 1}, {512, 2, 1296, 768, 1}};
constexpr ResVariant res_variant(bool f64, bool coupled, int v) {
  return coupled ? (f64 ? kRes64[v] : kRes32[v]) : (f64 ? kRes64V[v] : kRes32V[v]);
}

// Chip-resident kernel (cooperative launch of ntiles CTAs).
template <typename T, bool PLAIN>
cudaError_t launch_resident(const StepArgs<T>& a, bool coupled, int variant,
                            const ResTile* tiles, int ntiles, const ResRun& run, cudaStream_t s);

// Whether ntiles CTAs of a variant are co-resident on the current device
// (also allows the variant's dynamic shared memory; before the first launch).
template <typename T, bool PLAIN>
bool resident_fits(bool coupled, int variant, int ntiles);

// Allow the dynamic shared memory of every TMA kernel variant on the current
// device (call once per device before the first launch or graph capture).
template <typename T, bool PLAIN>
cudaError_t prepare_tma();

// Dynamic shared memory of the TMA kernel variant (0 if not available).
template <typename T>
size_t tma_smem_bytes(int bx, bool coupled, int mode);

// Initial state of every case in one launch over the work items (bx columns
// per CTA); src: per-case device-readable pointers to phi0 and u0.
template <typename T>
cudaError_t launch_init_items(const CaseDev<T>* cases, const Item* items, int n_items, int bx,
                              const InitSrc* src, double beta4, double kappa, double lambda,
                              int vortex, double vU, int parity, cudaStream_t s);

// buf: the 9-plane buffer with plane stride P (walls: bounce-back positions)
template <typename T>
cudaError_t launch_plane_import(T* buf, int64_t P, const double* src, int i, int nx, int ny,
                                int walls, cudaStream_t s);
template <typename T>
cudaError_t launch_plane_export(double* dst, const T* buf, int64_t P, int i, int nx, int ny,
                                int walls, cudaStream_t s);
// moving-wall term of f plane i at the wall rows, added (sign 1) or removed (-1)
template <typename T>
cudaError_t launch_wall_f_fix(double* v, const CaseDev<T>& cd, int par, int i, double sign,
                              cudaStream_t s);
// One case's snapshot (lbm_snapshot layout) in one launch; lo may be null.
template <typename T>
cudaError_t launch_snapshot(const T* f, const T* g, const T* J, const T* lo, int64_t P,
                            int64_t n, T* out, cudaStream_t s);
template <typename T>
cudaError_t launch_copy_to_T(T* dst, const double* src, int64_t n, cudaStream_t s);
template <typename T>
cudaError_t launch_copy_to_f64(double* dst, const T* src, int64_t n, cudaStream_t s);
template <typename T>
cudaError_t launch_add_lo_f64(double* v, const T* lo, int64_t n, cudaStream_t s);
template <typename T>
cudaError_t launch_lo_from_f64(T* lo, const T* hi, const double* v, int64_t n, cudaStream_t s);

// Per-item partial volumes (labelled regions) of the state in buffer parity;
// with end.ticket also the per-case sums, by the CTA that finishes last.
template <typename T>
cudaError_t launch_volume_partial(const CaseDev<T>* cases, const Item* items, int n_items,
                                  int bx, int parity, double* part, const VolumeEnd& end,
                                  cudaStream_t s);

// Per-case sums of the item partials (written by the step kernel's fused
// volume or by launch_volume_partial): the cases case_ids[0..ncases), or
// cases 0..ncases-1 with case_ids null.
template <typename T>
cudaError_t launch_volume_final(const CaseDev<T>* cases, const int* case_ids, int ncases,
                                const double* part, double* out, const int64_t* t, int64_t toff,
                                int64_t slots, int64_t stride, cudaStream_t s);

cudaError_t launch_clock(int64_t* t, int64_t n, cudaStream_t s);
cudaError_t launch_set_clock(int64_t* t, int64_t value, cudaStream_t s);

}  // namespace lbmk
