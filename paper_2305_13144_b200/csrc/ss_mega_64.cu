// The decode step's instantiations for heads of 64: a module of its own, since the first kernel of a module that a process
// launches loads all of it.  With all sixteen instantiations in one module the first context of a process took 22 ms, now 10.
#include "ss_decode_mega.cuh"

namespace ss {

const void* mega_kernel_64(int rows, bool trace) { return mega_kernel_of<64>(rows, trace); }

}  // namespace ss
