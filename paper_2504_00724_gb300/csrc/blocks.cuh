// How the FP64 sweep stages an SMO-2 block's inverse rows: in two parts, one stage each.
#pragma once

#include <cstddef>

#ifdef __CUDACC__
#define CCM_HDC __host__ __device__ constexpr
#else
#define CCM_HDC constexpr
#endif

namespace ccm {
namespace dev {

// extended rows of the first part: about half, even (the second part's copy starts on 16 bytes)
CCM_HDC int block_split(int ne) { return (ne / 2 + 1) & ~1; }

// bytes of the bulk copy of `rows` rows of nc columns
CCM_HDC unsigned block_copy_bytes(int rows, int nc, size_t es) { return (unsigned)(((long)rows * nc * es + 15) & ~15L); }

// bytes that a stage needs for any block of at most max_ext extended and max_core core rows, whole
// or (parts) any part of it: the second part is the longer one where ne = 4 k + 1, and the longer
// part does not get shorter as ne grows
inline size_t block_stage_bytes(int max_ext, int max_core, int es, bool parts) {
  const int first = block_split(max_ext), second = max_ext - first;
  return block_copy_bytes(parts ? (first > second ? first : second) : max_ext, max_core, es);
}

}  // namespace dev
}  // namespace ccm
