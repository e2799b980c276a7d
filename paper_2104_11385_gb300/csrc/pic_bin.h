// pic_bin.h -- box binning of caller-owned particles (shared by pic_bin.cu and
// its allocation-free variant).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/pic_api.h"

struct BinGeom {
    int dim;
    int n[3], bsz[3], nb[3];
    double d[3], inv[3];  // cell sizes and their reciprocals
    float rbsz[3];        // reciprocals of the box extents
    int nboxes;
};

constexpr int kBinHistMax = 8192;  // boxes of a histogram in shared memory: 32 KB
constexpr int kBinPer = 16;        // positions per thread that the shared scatter ranks at a time

// The shared histograms of the counts pay when adding them up takes at most a
// quarter of the global atomics they save (16.8 M positions in 4096 boxes: 803 ->
// 704 us per call; 100 thousand positions there stay with the global ones, 31 us).
inline bool bin_count_in_shared(int nboxes, int64_t np, int ctas) { return nboxes <= kBinHistMax && np >= 4ll * ctas * nboxes; }
// The shared scatter needs work for several CTAs of 1024 threads as well: below 16
// chunks it leaves the chip idle, and the global one, which ranks within warps, is
// faster (8 boxes, 10 / 30 / 100 thousand positions per call: 42 / 50 / 52 us against
// 28 / 28 / 30; 300 thousand, the first it takes: 53 against 35, or with 64 boxes
// 57 against 77).
inline bool bin_scatter_in_shared(int nboxes, int64_t np, int ctas) {
    return bin_count_in_shared(nboxes, np, ctas) && np >= 16ll * kBinPer * 1024;
}

pic_status pic_bin_validate(const pic_grid_desc* grid, const double* x, const double* y,
                            const double* z, int64_t np, const int64_t* box_off_out,
                            const int64_t* perm_out, BinGeom* g, std::string* err);
// box_off: nboxes+1 int64 (output, also the histogram); cursor: nboxes int32 scratch
cudaError_t pic_bin_launch(const BinGeom& g, const double* x, const double* y, const double* z,
                           int64_t np, int64_t* box_off, int64_t* perm, int32_t* cursor,
                           cudaStream_t st);
// streaming multiprocessors of the current device (defined in pic_particles.cu)
int pic_sm_count();
// records the message returned by pic_last_error(NULL) on this thread
pic_status pic_record_error(pic_status st, const char* msg);
