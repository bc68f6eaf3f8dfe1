// fft_float_zt.cu -- the float passes over z and t with the filter.
#include "fft_dispatch.h"
#include "fft_fixed.cuh"

namespace lgf {
namespace {
template <int NZ, int NTT> ZtKernel entry() {
  if constexpr (NZ * NTT <= kZtSites) {
    using Z = ZtTile<NZ, NTT>;
    return {(const void *)k_fx_zt<float, NZ, NTT>, Z::C, Z::threads, Z::smem};
  }
  return {};
}
template <int NZ> ZtKernel by_nt(int nt) {
  switch (nt) {
    case 8: return entry<NZ, 8>();
    case 16: return entry<NZ, 16>();
    case 24: return entry<NZ, 24>();
    case 32: return entry<NZ, 32>();
    case 48: return entry<NZ, 48>();
    default: return entry<NZ, 64>();
  }
}
}  // namespace
ZtKernel fft_float_zt(int nz, int nt) {
  switch (nz) {
    case 8: return by_nt<8>(nt);
    case 16: return by_nt<16>(nt);
    case 24: return by_nt<24>(nt);
    case 32: return by_nt<32>(nt);
    case 48: return by_nt<48>(nt);
    default: return by_nt<64>(nt);
  }
}
}  // namespace lgf
