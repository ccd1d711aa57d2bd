// vm_exact.cu -- the eliminated walk from program images, exact rings (vm_impl.cuh).
#include "vm_impl.cuh"
#include "vm.hpp"

namespace perm {
GenericFns vm_fns_f64();
GenericFns vm_fns_dd();
GenericFns vm_fns(int kind) {
    switch (kind >> 1) {
    case 0: return kind & 1 ? vm_fns_dd() : vm_fns_f64();
    case 2: return vm_make_fns<pk::VmExact<2>>();
    case 3: return vm_make_fns<pk::VmExact<3>>();
    case 4: return vm_make_fns<pk::VmExact<4>>();
    case 5: return vm_make_fns<pk::VmExact<5>>();
    case 6: return vm_make_fns<pk::VmExact<6>>();
    default: return GenericFns();
    }
}
}  // namespace perm
