// Resident step kernels, 16-bit storage.
#include "resident.inl"
namespace lbmfvm_fv {
LBMFVM_RESIDENT_INSTANTIATE(__half)
LBMFVM_RESIDENT_INSTANTIATE(__nv_bfloat16)
}
