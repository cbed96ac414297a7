// The tensor-core path of the FP64 precision (fp64_tc.cu).
#pragma once
#include <vector>

#include "gw_internal.cuh"

namespace gw {

// whether a q point's FP64 polarization takes the sliced path; the groups of q points that share
// launches, and a group's workspace
bool oz_pol_eligible(int64_t K);
std::vector<std::vector<int>> oz_pol_groups(const std::vector<int>& qs, const int64_t* K, const int* nb,
                                            int nw);
size_t oz_pol_workspace(const std::vector<int>& group, const int64_t* K, const int* nb, int nw, int sm);
// P of one group. The workspace's first 256 bytes then hold one int per q of the group that is
// odd when that q's input needs the FP64 kernel (its P is untouched).
int oz_pol(const std::vector<int>& group, const PolQ* qs, double pref, int nw, const OmegaArr& om,
           bool accumulate, void* ws, size_t ws_bytes, cudaStream_t s, const DeviceCtx& ctx,
           PolOpts& o);

// Pair coefficients c_p (FP64) of every q. The workspace's first 4 nq bytes then hold one int per q
// that is odd when that q needs the FP64 kernel (its c is to be overwritten).
size_t oz_pair_workspace(int nq, const int64_t* npair, const int* nb, int nw, int sm);
int oz_pair(int nq, const int64_t* npair, const int* nb, const void* const* Msig, int nw,
            const double* const* Wc, double* const* c, void* ws, size_t ws_bytes, cudaStream_t s,
            const DeviceCtx& ctx);

}  // namespace gw
