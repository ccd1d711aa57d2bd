// vm_dd.cu -- the eliminated walk from program images, one arithmetic (vm_impl.cuh).
#include "vm_impl.cuh"

namespace perm {
GenericFns vm_fns_dd() { return vm_make_fns<pk::VmDD>(); }
}  // namespace perm
