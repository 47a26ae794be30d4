// A connected configuration of the wide row form (tc.cu), read from the
// sample's connected list.
#pragma once

#include <cstdint>

namespace nqs {

// One configuration of a group: sigma with sites i and j exchanged (-1: as
// it is), rolled along x: its column c is sigma's column c + roll.
struct WideCfg {
    int16_t i, j, roll, pad;
};

// Entry k of the list's nconn exchanges (ci, cj) on N sites. The checked
// build tests k before it reads the list and the sites before they index the
// sample: an entry out of range is the sample itself.
__device__ inline WideCfg wide_entry(const int16_t *ci, const int16_t *cj, int k, int nconn, int N, int *err) {
    const WideCfg sample{-1, -1, 0, 0};
    if (!NQS_INDEX_OK(k >= 0 && k < nconn, err)) return sample;
    const WideCfg c{ci[k], cj[k], 0, 0};
    return NQS_INDEX_OK(c.i >= 0 && c.i < N && c.j >= 0 && c.j < N, err) ? c : sample;
}

}  // namespace nqs
