// Resident step kernels, ds storage.
#include "resident.inl"
namespace lbmfvm_fv {
LBMFVM_RESIDENT_INSTANTIATE(lbmfvm_dev::dsf)
}
