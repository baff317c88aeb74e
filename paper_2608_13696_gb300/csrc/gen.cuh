// Descriptor-driven group-by kernel (gen.cu): launch interface.
#pragma once

#include "groupby.cuh"

namespace rel {

// Group-by (p as fill_params left it, layers set): every row into a CTA-shared table of about `est` groups when that
// fits, merged into the global table; else straight into the global table.
rel_status gb_launch_gen(const GbParams& p, int64_t est, cudaStream_t st);
// Distinct qualifying keys: hdr->aux counts the keys claimed in the set
// p.tkeys (2^p.log2_slots slots), hdr->n_side the rows with key INT64_MIN.
// beside as for distinct_launch.
rel_status gb_launch_gen_set(const GbParams& p, bool beside, cudaStream_t st);

}  // namespace rel
