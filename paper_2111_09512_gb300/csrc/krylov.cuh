// Launchers of the FP64 Krylov kernels (flexible GMRES, reductions, the
// minimal-residual step of the Schur complement smoother).
#pragma once

#include <cuda_runtime.h>

#include "device.cuh"

namespace silu {

// ---- Krylov (FP64, one right-hand side) --------------------------------
// Block partial sums are written to part[0..nparts); every consumer reduces
// them in the same fixed order, so results are bitwise reproducible.
int krylov_parts(int n);
cudaError_t launch_dot_part(int n, const double* a, const double* b, double* part, cudaStream_t s);
// h = sum(part_in); if hout: *hout = h; w -= h vi; part_out = partials of w.vnext (or |w|^2 if vnext null)
cudaError_t launch_mgs_step(int n, const double* part_in, double* hout, double* w, const double* vi,
                            const double* vnext, double* part_out, int sms, cudaStream_t s);
// h = sqrt(sum(part_in)); *hout = h; vout = w / h (skipped if h == 0)
cudaError_t launch_normalize(int n, const double* part_in, double* hout, const double* w, double* vout,
                             cudaStream_t s);
// The end of Arnoldi step j: h = sqrt(sum(part_in)), vout = w / h (skipped if
// h == 0), and the Givens update of column j of H (row-major (m+1) x m,
// leading dimension m; rows 0..j hold h_0..h_j); res[0] = |g_{j+1}|, res[1] = h
cudaError_t launch_normalize_givens(int n, const double* part_in, const double* w, double* vout, int j, int m,
                                    double* H, double* cs, double* sn, double* g, double* res, cudaStream_t s);
// solve the jend x jend triangle, then x += sum_k y_k Z_k
cudaError_t launch_update_x(int n, int jend, int m, const double* H, const double* g, double* y, const double* Z,
                            double* x, cudaStream_t s);
// y = (sum(part_num) / sum(part_den)) s (0 when the denominator sums to 0); both
// partial arrays written by launch_dot_part over n rows
cudaError_t launch_mr_step(int n, const double* part_num, const double* part_den, const double* sv, double* y,
                           cudaStream_t s);
// q = w / h entry by entry, by the normalisations' division (a self-test).
cudaError_t launch_divide(int64_t n, const double* w, const double* h, double* q, cudaStream_t s);
// One Arnoldi step in one launch (kernels_arnoldi.cu): w against columns 0..j
// of V (stride n) by modified Gram-Schmidt, column j of H, V_{j+1} and the
// Givens update, with the bits of launch_dot_part, launch_mgs_step,
// launch_normalize_givens; w is only read.  scratch:
// arnoldi_bytes(n), this workspace's alone.  For sizes and restart lengths
// that fit (arnoldi_fits); a wait that gives up sets value 16 of *env.err.
// Each j runs at most once between two calls of arnoldi_reset, which belongs
// at the start of every restart cycle.
size_t arnoldi_bytes(int n);
cudaError_t arnoldi_reset(int n, int m, void* scratch, const LaunchEnv& env, cudaStream_t s);
// Make a wait of the exchange run out and leave entries in scratch that the
// next cycle's first step would take for its own.
cudaError_t launch_exchange_selftest(int n, void* scratch, int* err, cudaStream_t s);
cudaError_t arnoldi_prepare(LaunchEnv& env);
bool arnoldi_fits(int n, int m, const LaunchEnv& env);
cudaError_t launch_arnoldi(int n, int j, int m, const double* w, double* V, double* H, double* cs, double* sn,
                           double* g, double* res, void* scratch, const LaunchEnv& env, cudaStream_t s);
// *out = sqrt(sum(part_in)) for partials written by a launch over n rows
cudaError_t launch_norm_final(int n, const double* part_in, double* out, cudaStream_t s);

}  // namespace silu
