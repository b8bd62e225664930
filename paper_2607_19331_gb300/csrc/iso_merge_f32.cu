// iso_merge_f32.cu -- the merge pass over binary32 experts (iso_merge.cu holds
// the code; a second translation unit halves the build time).
#define ISO_MERGE_XT float
#include "iso_merge.cu"
