// gj_factor_small.cuh -- factor construction of small relations in one launch.
#pragma once

#include "gj_state.cuh"

namespace gj {

// Rows up to which a relation is built by one CTA, and the words the build
// reports: groups, 1 if it was built (0: the key does not fit a word beside
// the row id), then min and max of every key column.
constexpr int64_t SF_MAX = 12 * 1024;
constexpr int SF_OUT = 2 + 2 * MAX_KEYS;

// A relation of 1 .. SF_MAX rows; F's order is set and its arrays are
// allocated (perm, gstart, gkey at the relation's rows, payloads).
struct SmallFactor {
    const Relation *R;
    Factor *F;
    int32_t *out;          // device, SF_OUT words
};
cudaError_t small_factors(Ctx &c, const std::vector<SmallFactor> &f);

}  // namespace gj
