// The forward query of BF16 models with K = 16 features (k_fwd.cuh).
namespace srn { namespace { constexpr bool kF32 = false; constexpr int kK = 16; } }
#include "k_fwd.cuh"
