// The sensing launch for 33 to 64 groups.
#include "sense_kernel.cuh"

namespace cs {

template SenseFn sense_fn_kc<2>(int, SenseKind, bool);

}  // namespace cs
