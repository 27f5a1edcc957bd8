// Resident step kernels, f64 storage.
#include "resident.inl"
namespace lbmfvm_fv {
LBMFVM_RESIDENT_INSTANTIATE(double)
}
