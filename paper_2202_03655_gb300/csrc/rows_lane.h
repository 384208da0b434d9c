// Lane-per-point row writer of FP32 factors with few columns (rows_lane.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "../../include/hdf.h"

namespace hdf {
struct DeviceTables;
struct FactorChoice;
namespace dev { struct Center; }

struct RowsLanePlan {
    int ngrp = 0, ndeg = 0, nF0 = 0, nFp = 0, lane_floats = 0, rs = 0, pairs = 0;
    size_t smem = 0;
    std::vector<int> tab;
    std::vector<float> rc;
};
bool rows_lane_plan(int d, int L, const FactorChoice& fc, const DeviceTables& tb, RowsLanePlan& out);
hdf_status rows_lane(const RowsLanePlan& pl, const double* x, int64_t n, int d, const dev::Center& c, double inv2R, int L,
                     const DeviceTables& tb, const float* cA, const float* cB, float* U, cudaStream_t st);
}  // namespace hdf
