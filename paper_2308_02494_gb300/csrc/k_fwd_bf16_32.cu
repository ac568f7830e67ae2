// The forward query of BF16 models with K = 32 features (k_fwd.cuh).
namespace srn { namespace { constexpr bool kF32 = false; constexpr int kK = 32; } }
#include "k_fwd.cuh"
