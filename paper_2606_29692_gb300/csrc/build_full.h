// Plan and launches of the full-space Hamiltonian build (build_full.cu).
#pragma once

#include "common.h"

namespace tq {

constexpr int BUILD_SMALL_RANK = 6;            // tables of at most 64 entries: one kept mask per group
constexpr int BUILD_MAX_RANK = 10;             // runs of a wide group (1024 entries each)
constexpr uint32_t BUILD_WIDE = 0xffffffffu;   // BuildGroup::low of a wide group (b[0]: its index)

// A group with one table: parity masks b (unused: 0), the table indices of
// the row bits 0..2 (8 bits each), and the table's first entry.
struct alignas(16) BuildGroup {
    uint32_t b[BUILD_SMALL_RANK];
    uint32_t low, tab;
};

// Terms t0 .. t1-1 of one group, whose Z-masks lie in the span of
// b[0..m-1]; g: the group if it is small, else -1.
struct BuildRun {
    int t0, t1, m, tab, g;
    uint32_t b[BUILD_MAX_RANK];
    uint32_t low[3];
};

struct BuildSeg {
    int rows, pairs, half, max_row;
};
struct BuildOffsets {
    long long rows, pairs, half;
};

struct BuildTotals {
    long long rows, pairs, half;
    unsigned long long amb;
    int max_row, pad;
};

// The host's plan (all vectors are uploaded as they are).
struct BuildPlan {
    std::vector<BuildGroup> rec;     // [G]
    std::vector<BuildRun> runs;      // one per small group, one or more per wide group, in group order
    std::vector<uint32_t> comb;      // [terms] coordinates of the term's Z-mask in its run's basis
    std::vector<uint32_t> wx;        // [W] masks of the wide groups
    std::vector<int> woff, wend;     // [W] their runs
    std::vector<uint32_t> hx;        // [H] distinct x >> 3, ascending
    std::vector<int> hoff;           // [H + 1] first group of each
    std::vector<uint32_t> sib;       // [levels H] size of the sibling subtree at each level
    int levels = 0;
    int n_entries = 0;               // table entries of all runs
    std::vector<int> dorder, dbin;   // diagonal terms sorted by their low 8 Z bits, and the bins [257]
};
BuildPlan plan_build(int nq, const std::vector<uint32_t>& gx, const std::vector<int>& goff,
                     const std::vector<uint32_t>& tz, const std::vector<uint32_t>& dz);

// The plan on the device.
struct BuildView {
    int G, W, H, levels;
    const uint32_t* gx;
    const BuildGroup* rec;
    const uint2* keep;       // [G] kept entries of the group's table (small groups)
    const uint2* amb;        // [G] kept entries near the drop tolerance
    const BuildRun* runs;
    const double* T;         // tables, float64 and rounded to float32
    const float* Tf;
    const uint32_t* wx;
    const int *woff, *wend;
    const uint32_t* hx;
    const int* hoff;
    const uint32_t* sib;
    int half_bit;            // lowest of the HALF_CLASSES top index bits, or 0: no half pass
    int cls[HALF_CLASSES];   // first group whose mask has a bit at or above half_bit + j
};

int build_segments(long long B);
// tol and amb: the drop tolerance and the ambiguity bound as the bits of a
// non-negative double.  keep / amb_mask: one mask per group, zeroed.
int launch_build_tables(const BuildView& v, int n_runs, const uint32_t* comb, const double* tc, double* T, float* Tf,
                        unsigned long long tol, unsigned long long amb, uint2* keep, uint2* amb_mask,
                        cudaStream_t s);
int launch_build_diag(long long D, const int* dbin, const uint32_t* dz, const double* dc, double* diag, int sms,
                      cudaStream_t s);
// hcls, hptr: the half pass's tables (null when v.half_bit is 0).
int launch_build_count(const BuildView& v, long long D, long long B, unsigned long long tol, unsigned long long amb,
                       int* rowcnt, int* blkcnt, int* halfcnt, BuildSeg* seg, BuildOffsets* off, BuildTotals* tot,
                       int* rowptr, int* xptr, uint2* hcls, int* hptr, cudaStream_t s);
int launch_build_fill(const BuildView& v, long long D, long long B, long long nnz, unsigned long long tol, int prec,
                      const int* rowptr, int* col, void* val, const int* xptr, uint32_t* xmask, void* xval, int sms,
                      cudaStream_t s);

}  // namespace tq
