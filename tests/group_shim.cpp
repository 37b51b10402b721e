// Test shim: the layout constants of fused groups (paper_2010_07284_gb300/
// csrc/vl_internal.h), compiled with the host compiler by
// tests/test_group_vectors.py.
#include "vl_internal.h"

extern "C" int group_threads() { return vl::EXEC_THREADS; }
extern "C" int group_segment() { return vl::GROUP_SEG; }
extern "C" int group_row_vecs(int tile_words) { return vl::group_vecs(tile_words); }
