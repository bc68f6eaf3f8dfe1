// fft_df64_zt.cu -- the df64 passes over z and t with the filter.
#include "fft_zt_instances.cuh"

namespace lgf {
ZtKernel fft_df64_zt_long(int nz, int nt);  // fft_df64_zt_long.cu
ZtKernel fft_df64_zt(int nz, int nt) {
  switch (nz) {
    case 8: return zt_by_nt<df64, 8>(nt);
    case 16: return zt_by_nt<df64, 16>(nt);
    default: return fft_df64_zt_long(nz, nt);
  }
}
}  // namespace lgf
