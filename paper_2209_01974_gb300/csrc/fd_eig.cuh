// The symmetric eigensolver's task description (fd_eig.cu): one matrix of a
// batch, its work arrays and outputs.
#pragma once

#include <stddef.h>

#include "fd_internal.cuh"

namespace fdi {

constexpr int EIG_BLOCK = 8;

struct EigTask {
  const double* H;      // n x n symmetric, row-major
  double* w;            // n eigenvalues, ascending
  double* Qout;         // n x n, eigenvectors as columns
  const int* active;    // nullptr, or skip the matrix when *active == 0
  const int* flags;     // nullptr, or skip it when *flags & flag_mask
  int flag_mask;
  int n, np;            // order, padded to a multiple of 16
  double *A0, *A1, *Q;  // np x np
  double* J;            // np / 16 rotations of 16 x 16
  int* shift;
};

int eig_padded(int n);
size_t eig_work_doubles(int n);
// fills n, np and the work pointers from `work` (eig_work_doubles(n) doubles)
void eig_task_layout(EigTask* t, int n, double* work);
size_t eig_part_floats(const fd_ctx* ctx, int n_inst);
// all matrices tasks_dev[0 .. n_inst) (device array; orders at most n_max) in
// one cooperative launch; part: eig_part_floats(ctx, n_inst) device floats
fd_status eig_batch(fd_ctx* ctx, const EigTask* tasks_dev, int n_inst, int n_max, int max_sweeps, float* part);

}  // namespace fdi
