// pz_line_bwd4.cu -- the far-wing reverse pass with all three damping families (see pz_line_bwd.cu).
#define PZ_BWD_FOUR true
#define PZ_BWD_LAUNCH launch_far_bwd4
#include "pz_line_bwd.cu"
