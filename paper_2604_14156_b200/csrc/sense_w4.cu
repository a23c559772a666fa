// The sensing launch for 97 to 128 groups.
#include "sense_kernel.cuh"

namespace cs {

template SenseFn sense_fn_kc<4>(int, SenseKind, bool);

}  // namespace cs
