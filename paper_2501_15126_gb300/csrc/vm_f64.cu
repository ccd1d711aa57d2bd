// vm_f64.cu -- the eliminated walk from program images, one arithmetic (vm_impl.cuh).
#include "vm_impl.cuh"

namespace perm {
GenericFns vm_fns_f64() { return vm_make_fns<pk::VmF64>(); }
}  // namespace perm
