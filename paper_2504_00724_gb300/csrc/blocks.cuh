// How the FP64 sweep stages an SMO-2 block's inverse rows: in two parts, one stage each.
#pragma once

#include <cstddef>

#include "fixed.cuh"

namespace ccm {
namespace dev {

// Extended rows of the first part: half of them, rounded up to an even number (the second part's copy
// starts on 16 bytes) and so never fewer than the second part's.
CCM_HD int block_split(int ne) { return ne < 2 ? ne : ((ne + 1) / 2 + 1) & ~1; }

// bytes of the bulk copy of `rows` rows of nc columns
CCM_HD unsigned block_copy_bytes(int rows, int nc, int es) { return (unsigned)(((long)rows * nc * es + 15) & ~15L); }

// bytes that a stage needs for any block of at most max_ext extended and max_core core rows, whole
// or (parts) any part of it: the first part is the longer one, and longest at max_ext
inline size_t block_stage_bytes(int max_ext, int max_core, int es, bool parts) {
  return block_copy_bytes(parts ? block_split(max_ext) : max_ext, max_core, es);
}

}  // namespace dev
}  // namespace ccm
