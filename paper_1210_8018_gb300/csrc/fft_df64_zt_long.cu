// fft_df64_zt_long.cu -- the df64 passes over z and t for Nz above 16 (compiled apart).
#include "fft_zt_instances.cuh"

namespace lgf {
ZtKernel fft_df64_zt_long(int nz, int nt) {
  switch (nz) {
    case 32: return zt_by_nt<df64, 32>(nt);
    case 64: return zt_by_nt<df64, 64>(nt);
    default: return {};  // 24 and 48: none is faster (zt_faster)
  }
}
}  // namespace lgf
