// The sensing launch for 65 to 96 groups.
#include "sense_kernel.cuh"

namespace cs {

template SenseFn sense_fn_kc<3>(int, SenseKind, bool);

}  // namespace cs
