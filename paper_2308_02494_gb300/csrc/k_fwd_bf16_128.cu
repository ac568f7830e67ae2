// The forward query of BF16 models with K = 128 features (k_fwd.cuh).
namespace srn { namespace { constexpr bool kF32 = false; constexpr int kK = 128; } }
#include "k_fwd.cuh"
