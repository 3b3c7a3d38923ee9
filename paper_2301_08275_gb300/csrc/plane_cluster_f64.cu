// plane_cluster_f64.cu - complex128 instances of the on-chip 2D step (plane_cluster.cu).
#define GPE_PLANE_R double
#define GPE_PLANE_LAUNCH launch_plane_f64
#include "plane_cluster.cu"
