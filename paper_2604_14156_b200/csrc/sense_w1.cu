// The sensing launch for up to 32 groups.
#include "sense_kernel.cuh"

namespace cs {

template SenseFn sense_fn_kc<1>(int, SenseKind, bool);

}  // namespace cs
