// The forward query of float32 models (k_fwd.cuh).
#define SRN_FWD_LAUNCH launch_forward_f32
#define SRN_FWD_NODES forward_nodes_f32
namespace srn { namespace { constexpr bool kF32 = true; } }
#include "k_fwd.cuh"
