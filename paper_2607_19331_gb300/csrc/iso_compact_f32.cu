// iso_compact_f32.cu -- the compact-candidate passes over binary32 experts
// (iso_compact.cu holds the code).
#define ISO_COMPACT_XT float
#include "iso_compact.cu"
