// fft_dispatch.h -- kernel-pointer tables of the FFT passes. The passes are instantiated per arithmetic
// type in their own translation units (fft_float.cu, fft_double.cu, fft_df64_*.cu) so that the library
// compiles in parallel; the host code launches them through these pointers with cudaLaunchKernel.
#pragma once
#include <type_traits>

#include "df64.cuh"

namespace lgf {

// Specialised pass (fft_fixed.cuh): kind 1 = xy plane (mode 0 forward, 1 inverse), kind 2 = columns
// (mode 0 forward, 1 inverse, 2 forward + filter + inverse) with C in {16, 32}; N in {8,16,24,32,48,64};
// kind 3 = the float column pass with the filter held in registers (k_fx_tfilter64: N = 64, C = 32, mode 2);
// kind 4 = the float 64 x 64 xy plane pass held in registers (k_fx_plane64; mode 0 forward, 1 inverse).
template <typename FT> const void *fft_fixed_kernel(int kind, int mode, int N, int C);
// The pass over z and t with the filter (k_fx_zt) in float and df64 for extents of the table, with its columns per
// block, threads and shared memory; no kernel where the column passes are faster (zt_faster).
struct ZtKernel {
  const void *kernel;
  int C, threads;
  size_t smem;
};
ZtKernel fft_float_zt(int nz, int nt);
ZtKernel fft_df64_zt(int nz, int nt);
// Measured per iteration, with the events of the timing mode, against the three column passes. Float: 16 x 32
// (16^3 x 32) 16 against 35 us, 32 x 32 (32^4) 44 / 68, 32 x 48 (48^2 x 32 x 48) 155 / 181, 32 x 64 (64^2 x 32 x 64)
// 289 / 323; but 48 x 48 (48^4) 299 / 277, 64 x 64 (64^4) 621 / 572. df64: 16 x 16 (16^4) 20 / 39, 32 x 32 (32^4)
// 121 / 149, 16 x 64 (32^2 x 16 x 64) 120 / 170; but 32 x 48 296 / 258, and with radix 3 24 x 24 (24^4) 77 / 79,
// 24 x 48 (24^3 x 48) 150 / 129.
template <typename FT> constexpr bool zt_faster(int nz, int nt) {
  if (std::is_same<FT, float>::value) return nz * nt <= 2048;
  return nz * nt <= 1024 && (nz & (nz - 1)) == 0 && (nt & (nt - 1)) == 0;
}
// Generic pass (fft.cuh, k_fft_pass).
template <typename FT> const void *fft_generic_kernel();

// Packed fields per block of the column pass with the filter (kind 2, mode 2): one (small tiles, more
// resident blocks), except in IEEE double, where four fields share the weights of the FP64 pipe.
template <typename FT> constexpr int filter_fields_per_block() { return std::is_same<FT, double>::value ? 4 : 1; }

// Passes that prefetch the next tile into registers while the current one is transformed: the float z
// passes (forward, inverse; measured at 64^4: 0.19 -> 0.17 ms per pass). The xy pass and the t pass with
// the filter gained nothing from it in float (the t pass lost resident blocks to the extra registers),
// and the double-float and double passes are bound by arithmetic: those take one tile per block.
template <typename FT, int KIND, int MODE> __host__ __device__ constexpr bool prefetch_tiles() {
  return std::is_same<FT, float>::value && KIND == 2 && MODE != 2;
}

}  // namespace lgf
