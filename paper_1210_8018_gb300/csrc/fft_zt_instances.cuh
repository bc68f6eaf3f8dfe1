// fft_zt_instances.cuh -- the table of the passes over z and t with the filter, for the translation units of the
// two arithmetic types.
#pragma once
#include "fft_dispatch.h"
#include "fft_fixed.cuh"

namespace lgf {
namespace {
template <typename T, int NZ, int NTT> ZtKernel zt_entry() {
  if constexpr (zt_faster<T>(NZ, NTT)) {
    using Z = ZtTile<T, NZ, NTT>;
    return {(const void *)k_fx_zt<T, NZ, NTT>, Z::C, Z::threads, Z::smem};
  }
  return {};
}
template <typename T, int NZ> ZtKernel zt_by_nt(int nt) {
  switch (nt) {
    case 8: return zt_entry<T, NZ, 8>();
    case 16: return zt_entry<T, NZ, 16>();
    case 24: return zt_entry<T, NZ, 24>();
    case 32: return zt_entry<T, NZ, 32>();
    case 48: return zt_entry<T, NZ, 48>();
    default: return zt_entry<T, NZ, 64>();
  }
}
}  // namespace
}  // namespace lgf
