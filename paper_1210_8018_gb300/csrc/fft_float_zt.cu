// fft_float_zt.cu -- the float passes over z and t with the filter.
#include "fft_zt_instances.cuh"

namespace lgf {
ZtKernel fft_float_zt(int nz, int nt) {
  switch (nz) {
    case 8: return zt_by_nt<float, 8>(nt);
    case 16: return zt_by_nt<float, 16>(nt);
    case 24: return zt_by_nt<float, 24>(nt);
    case 32: return zt_by_nt<float, 32>(nt);
    case 48: return zt_by_nt<float, 48>(nt);
    default: return zt_by_nt<float, 64>(nt);
  }
}
}  // namespace lgf
