// The forward query of BF16 models (k_fwd.cuh).
#define SRN_FWD_LAUNCH launch_forward_bf16
#define SRN_FWD_NODES forward_nodes_bf16
namespace srn { namespace { constexpr bool kF32 = false; } }
#include "k_fwd.cuh"
