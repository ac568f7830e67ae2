// The forward query of float32 models with K = 16 features (k_fwd.cuh).
namespace srn { namespace { constexpr bool kF32 = true; constexpr int kK = 16; } }
#include "k_fwd.cuh"
