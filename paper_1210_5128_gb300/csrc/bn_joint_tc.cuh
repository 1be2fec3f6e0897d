// bn_joint_tc.cuh -- joint count tables of the largest sets on the tensor cores
// (bn_joint_tc.cu), called by the table build.
#pragma once

#include <vector>

#include "bn_internal.cuh"

namespace bn {

struct TcJoint {
    int n, m, mw, size;            // sets of `size` nodes, 4 or 5
    int nh;                        // variants of the configuration sums (parent sets), or 0
    const uint8_t* arity;          // device
    const uint32_t* packed;        // device, [n][mw]
    const fx128* lut[4];           // device, [m + 1]: lgamma terms of a cell count and of the
                                   // variants' configuration counts, one table for every set
    fx128* G;                      // device, by rank over sets of at most k + 1 nodes
    fx128* H;                      // device, [nh][H_stride] by rank over sets of at most k
    int64_t H_stride;
    uint32_t* status;
    uint8_t* scratch;              // joint_tc_scratch bytes
};

// the work of one (n, k, arities): row tiles of pairs, column tiles of low sets
struct TcPlan {
    std::vector<uint32_t> pairs, rowinfo, mt_first, nt_start;
    uint32_t items = 0;
};

// plans the sets of `size` nodes (luts tables); false where the histogram kernel is better
bool joint_tc_plan(int n, int m, int size, int luts, const uint8_t* arity_host, TcPlan* P);
size_t joint_tc_scratch(const TcPlan& P, int m);
// the plan's lists to the scratch block; the host may wait for the stream's work before it
int joint_tc_upload(const TcPlan& P, uint8_t* scratch, cudaStream_t s);
int launch_joint_tc(const TcJoint& J, const TcPlan& P, cudaStream_t s);

}  // namespace bn
