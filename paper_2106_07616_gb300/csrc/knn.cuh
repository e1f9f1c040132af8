// knn.cuh -- internal interface of the cloud builder.
#pragma once
#include <stddef.h>

#include "common.cuh"

namespace rbffd {

struct KnnLayout {
  int m;              // cells at most
  size_t off_bbox, off_cnt, off_grid, off_cell, off_start, off_sums, off_pts;
  size_t zero_bytes;  // the first bytes, zeroed before a search
  size_t bytes;
};

int knn_workspace_bytes(int n, KnnLayout *lay);
// Lx, Ly: periods of the axes (0: bounded).
int knn_run(rbffd_ctx *ctx, void *ws, const KnnLayout &lay, int n, const double *x,
            const double *y, const int8_t *tag, int q, int32_t *idx, double Lx, double Ly);

}  // namespace rbffd
