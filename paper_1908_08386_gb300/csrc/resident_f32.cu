// Resident step kernels, f32 storage.
#include "resident.inl"
namespace lbmfvm_fv {
LBMFVM_RESIDENT_INSTANTIATE(float)
}
