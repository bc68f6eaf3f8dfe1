// fft.cuh -- hand-written batched 4D FFT with the Fourier-acceleration filter of Algorithm 1.
//
// Each packed Delta field (4 per site, see site_kernels.cuh) is transformed by a sequence of
// "passes". A pass stages a tile of the field in shared memory -- whole xy planes or lattice rows, or the
// full extent of one or two lattice axes times C neighbouring columns -- transforms the tile along
// those axes and writes it back. The forward transform is an in-place mixed-radix decimation-in-
// frequency FFT, which leaves the spectrum in digit-reversed order; the filter reads the frequency of
// each position from tables, and the inverse runs the exact inverse stages (decimation in time) in
// reverse order, which restores natural order. No permutation pass is needed. The filter
// w(k) = p^2_max / (V p^2(k)), w(0) = 0, is applied inside the last forward pass, which then runs the
// inverse along its own axes before writing (Algorithm 1: FFT forward, p^2_max/p^2, FFT backward,
// normalize).
//
// DIF stage (block length L, radix R, M = L/R), for each block and each j in [0, M):
//   y_r' = w_L^{j r'} * sum_r x[j + M r] w_R^{r r'},   stored at j + M r',   w_n = exp(-2 pi i / n).
// The inverse stage undoes it exactly up to the factor R.
#pragma once
#include "site_kernels.cuh"

namespace lgf {

constexpr int kMaxStages = 8;

struct AxisFFT {
  int N;                  // axis length
  int nst;                // number of stages
  int R[kMaxStages];      // radix of each DIF stage, in forward order
};

// n / d for n d < 2^32 by one high multiplication (m = ceil(2^32 / d); d = 1 has m = 0): the lengths of a
// general lattice are known only at run time, and the hardware has no integer division.
struct FastDiv {
  unsigned d, m;
};
inline FastDiv fast_div(unsigned d) {
  return FastDiv{d, d == 1 ? 0u : (unsigned)((((unsigned long long)1 << 32) + d - 1) / d)};
}
__device__ __forceinline__ unsigned div_by(unsigned n, FastDiv f) { return f.m ? __umulhi(n, f.m) : n; }

// The transform of a tile along one of its axes: npen pencils of N elements `estride` apart, pencil p
// starting at (p / A) B + (p % A) S.
struct AxisPhase {
  int mu;                    // lattice axis
  int nst, R[kMaxStages];    // radix of each DIF stage, in forward order
  FastDiv M[kMaxStages];     // block length of each stage over its radix
  int N, npen, A, B, S, estride;
  FastDiv dpen, dA;
};

// One pass: tiles of one packed field are staged in shared memory and transformed along one or two axes.
//   columns (rowform 0): C neighbouring columns by `rows` rows, element (row, c) of the tile at
//     base(q) + row rstride with q = tile C + c, base(q) = (q % nin) + (q / nin) ostride; ncol columns;
//   rows (rowform 1): `rows` consecutive lattice rows of nx elements (whole xy planes, or rows alone).
struct PassDesc {
  int rowform;
  int rows, C, logC, pitch;
  unsigned ncol, nin;
  int64_t ostride, rstride;
  unsigned nrow;
  FastDiv dnx;
  int nax;
  AxisPhase ph[2];
  int mode;     // 0 forward, 1 inverse, 2 forward + filter + inverse
  int nblocks;  // tiles per field
};

struct FFTTables {
  // Not read by a kernel any more, but the specialised passes are slower without it, with the same registers (the
  // float t pass at 64^4 255 us against 231, df64 z passes at 24^3 x 48 35 against 28): what it changes is the place
  // of the arguments behind it.
  AxisFFT ax[4];
  const void *tw[4];        // per lattice axis: N complex twiddles w_N^j (T)
  const double *p2part[4];  // per lattice axis: 4 sin^2(pi k(pos)/N) for the frequency at position pos
  double wscale;            // p^2_max / V
  const void *weights;      // w of every site in the transform's type (the general passes), or null
  int n[4];
};

// Butterfly sums. In double-float the pair is not renormalised after each addition (TwoSum of the high
// parts plus the low parts: 8 operations instead of 11); the twiddle multiplication renormalises, so the
// low part grows by at most a few ulps of the high part between multiplications. The transform's error
// stays ~2^-45 of the field norm, far below what the filter (which only sets the step direction) needs.
template <typename T> __device__ __forceinline__ cx<T> badd(cx<T> a, cx<T> b) { return a + b; }
template <typename T> __device__ __forceinline__ cx<T> bsub(cx<T> a, cx<T> b) { return a - b; }
__device__ __forceinline__ df64 df64_add_unnormalised(df64 x, df64 y) {
  const df64 s = two_sum(x.hi, y.hi);
  return {s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo))};
}
template <> __device__ __forceinline__ cx<df64> badd(cx<df64> a, cx<df64> b) {
  return {df64_add_unnormalised(a.r, b.r), df64_add_unnormalised(a.i, b.i)};
}
template <> __device__ __forceinline__ cx<df64> bsub(cx<df64> a, cx<df64> b) {
  return {df64_add_unnormalised(a.r, -b.r), df64_add_unnormalised(a.i, -b.i)};
}

// ---------------- register DFTs (R points, forward sign -1 or inverse sign +1) ----------------
template <typename T, bool INV> __device__ __forceinline__ cx<T> mul_mi(cx<T> a) {
  // forward: multiply by -i; inverse: by +i
  return INV ? cx<T>{-a.i, a.r} : cx<T>{a.i, -a.r};
}

template <typename T, bool INV> __device__ __forceinline__ void dft2(cx<T> *v) {
  const cx<T> a = v[0], b = v[1];
  v[0] = badd(a, b);
  v[1] = bsub(a, b);
}

template <typename T, bool INV> __device__ __forceinline__ void dft3(cx<T> *v) {
  const T h = kconst<T>(0.86602540378443864676);  // sqrt(3)/2
  const cx<T> s = v[1] + v[2], d = v[1] - v[2];
  const T half = kconst<T>(0.5);
  const cx<T> a = {v[0].r - half * s.r, v[0].i - half * s.i};
  const cx<T> b = scale(mul_mi<T, INV>(d), h);  // forward: -i (sqrt3/2) (x1 - x2)
  v[0] = v[0] + s;
  v[1] = a + b;
  v[2] = a - b;
}

template <typename T, bool INV> __device__ __forceinline__ void dft4(cx<T> *v) {
  const cx<T> s02 = badd(v[0], v[2]), d02 = bsub(v[0], v[2]), s13 = badd(v[1], v[3]);
  const cx<T> d13 = mul_mi<T, INV>(bsub(v[1], v[3]));
  v[0] = badd(s02, s13);
  v[2] = bsub(s02, s13);
  v[1] = badd(d02, d13);
  v[3] = bsub(d02, d13);
}

template <typename T, bool INV> __device__ __forceinline__ void dft5(cx<T> *v) {
  const T c1 = kconst<T>(0.30901699437494742410), c2 = kconst<T>(-0.80901699437494742410);  // cos 2pi/5, 4pi/5
  const T s1 = kconst<T>(0.95105651629515357212), s2 = kconst<T>(0.58778525229247312917);   // sin 2pi/5, 4pi/5
  const cx<T> a1 = v[1] + v[4], b1 = v[1] - v[4], a2 = v[2] + v[3], b2 = v[2] - v[3];
  const cx<T> x0 = v[0];
  v[0] = x0 + a1 + a2;
  const cx<T> r1 = {x0.r + c1 * a1.r + c2 * a2.r, x0.i + c1 * a1.i + c2 * a2.i};
  const cx<T> r2 = {x0.r + c2 * a1.r + c1 * a2.r, x0.i + c2 * a1.i + c1 * a2.i};
  // forward: y1 = r1 - i(s1 b1 + s2 b2), y4 = r1 + i(...); y2 = r2 - i(s2 b1 - s1 b2), y3 = r2 + i(...)
  const cx<T> q1 = mul_mi<T, INV>(cx<T>{s1 * b1.r + s2 * b2.r, s1 * b1.i + s2 * b2.i});
  const cx<T> q2 = mul_mi<T, INV>(cx<T>{s2 * b1.r - s1 * b2.r, s2 * b1.i - s1 * b2.i});
  v[1] = r1 + q1;
  v[4] = r1 - q1;
  v[2] = r2 + q2;
  v[3] = r2 - q2;
}

template <typename T, bool INV> __device__ __forceinline__ void dft8(cx<T> *v) {
  cx<T> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  dft4<T, INV>(e);
  dft4<T, INV>(o);
  const T h = kconst<T>(0.70710678118654752440);  // 1/sqrt(2)
  // twiddles w8^k, k = 0..3 (forward w8 = (1 - i)/sqrt 2)
  const cx<T> o1 = INV ? cx<T>{h * (o[1].r - o[1].i), h * (o[1].r + o[1].i)}
                       : cx<T>{h * (o[1].r + o[1].i), h * (o[1].i - o[1].r)};
  const cx<T> o2 = mul_mi<T, INV>(o[2]);
  const cx<T> o3 = INV ? cx<T>{-h * (o[3].r + o[3].i), h * (o[3].r - o[3].i)}
                       : cx<T>{h * (o[3].i - o[3].r), -h * (o[3].r + o[3].i)};
  v[0] = badd(e[0], o[0]);
  v[4] = bsub(e[0], o[0]);
  v[1] = badd(e[1], o1);
  v[5] = bsub(e[1], o1);
  v[2] = badd(e[2], o2);
  v[6] = bsub(e[2], o2);
  v[3] = badd(e[3], o3);
  v[7] = bsub(e[3], o3);
}

template <typename T, int R, bool INV> __device__ __forceinline__ void dft(cx<T> *v) {
  if constexpr (R == 2) dft2<T, INV>(v);
  else if constexpr (R == 3) dft3<T, INV>(v);
  else if constexpr (R == 4) dft4<T, INV>(v);
  else if constexpr (R == 5) dft5<T, INV>(v);
  else dft8<T, INV>(v);
}

// One stage over every pencil of the tile. Work item w -> (pencil p, butterfly beta) with the pencil
// varying fastest, so that consecutive threads touch consecutive words (or rows of odd pitch) of the tile.
template <typename T, int R, bool INV>
__device__ __forceinline__ void fft_stage(cx<T> *tile, const cx<T> *tw, const AxisPhase &ph, FastDiv dM) {
  const unsigned M = dM.d;
  const unsigned L = M * R;
  const unsigned twstep = ph.N / L;  // w_L^e = w_N^(e N/L)
  const unsigned items = ph.npen * (ph.N / R);
  const int step = M * ph.estride;
#pragma unroll 1
  for (unsigned w = threadIdx.x; w < items; w += blockDim.x) {
    const unsigned beta = div_by(w, ph.dpen), p = w - beta * ph.npen;
    const unsigned a = div_by(p, ph.dA);
    const unsigned blk = div_by(beta, dM), j = beta - blk * M;
    cx<T> *q = tile + (int)(a * ph.B + (p - a * ph.A) * ph.S + (blk * L + j) * ph.estride);
    cx<T> v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = q[r * step];
    // (a stage with M = 1 has j = 0 and unit twiddles: no multiplications; M is uniform per stage)
    if constexpr (!INV) {
      dft<T, R, false>(v);
      if (M > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = v[r] * tw[j * r * twstep];
      }
    } else {
      if (M > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = v[r] * conjg(tw[j * r * twstep]);
      }
      dft<T, R, true>(v);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) q[r * step] = v[r];
  }
}

template <typename T, bool INV>
__device__ __forceinline__ void fft_stage_any(int R, cx<T> *tile, const cx<T> *tw, const AxisPhase &ph, FastDiv dM) {
  switch (R) {
    case 2: fft_stage<T, 2, INV>(tile, tw, ph, dM); break;
    case 3: fft_stage<T, 3, INV>(tile, tw, ph, dM); break;
    case 4: fft_stage<T, 4, INV>(tile, tw, ph, dM); break;
    case 5: fft_stage<T, 5, INV>(tile, tw, ph, dM); break;
    default: fft_stage<T, 8, INV>(tile, tw, ph, dM); break;
  }
}

// Full forward (DIF, digit-reversed output) or inverse (DIT, natural output) transform along one axis.
template <typename T, bool INV>
__device__ __forceinline__ void fft_axis(cx<T> *tile, const cx<T> *tw, const AxisPhase &ph) {
#pragma unroll 1
  for (int i = 0; i < ph.nst; ++i) {
    const int k = INV ? ph.nst - 1 - i : i;
    fft_stage_any<T, INV>(ph.R[k], tile, tw, ph, ph.M[k]);
    __syncthreads();
  }
}

// Filter weight of every site for the general passes, w = p^2_max / (V p^2), 0 at p = 0: in double, rounded
// once. Kept as a table because p^2 at a (digit-reversed) position and its quotient cost three 64-bit
// divisions and one FP64 division per element when they are formed inside the pass.
template <typename T>
__global__ void k_filter_weights(T *__restrict__ W, int64_t V, FFTTables tb) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  unsigned r = (unsigned)s;
  const unsigned px = r % (unsigned)tb.n[0];
  r /= (unsigned)tb.n[0];
  const unsigned py = r % (unsigned)tb.n[1];
  r /= (unsigned)tb.n[1];
  const unsigned pz = r % (unsigned)tb.n[2], pt = r / (unsigned)tb.n[2];
  const double p2 = __ldg(tb.p2part[0] + px) + __ldg(tb.p2part[1] + py) + __ldg(tb.p2part[2] + pz) +
                    __ldg(tb.p2part[3] + pt);
  W[s] = p2 == 0.0 ? kconst<T>(0.0) : convert<T>(tb.wscale / p2);
}

// The pass kernel. blockIdx.x: tile, blockIdx.y: packed field. Shared memory: the tile, then the
// twiddle tables of the transformed axes.
// The fields of the lattices that come here mostly fit the L2, and what bounds a pass is issue and the latency
// of its phases. Index arithmetic is one high multiplication per division, a thread of a column tile keeps its
// column, and the filter's weight is one load. Measured per launch against passes with run-time division and
// weights formed in place (ncu: 3-4% of DRAM, 25-58% of the SM, the FP64 pipe 40% busy with the weights):
// 30x20x24x36 float, z and t with the filter 166 -> 39 us, xy 60 -> 24 us; 18x12x10x15 double-float, 66 -> 19 us
// and 19 -> 11 us. The operations and their order are those of the earlier passes: the same bits.
template <typename T>
__global__ void __launch_bounds__(512) k_fft_pass(T *__restrict__ data, int64_t V, const __grid_constant__ PassDesc pd,
                                                 const __grid_constant__ FFTTables tb, const Ctrl *ctrl,
                                                 int check_active, int tkid) {
  follow_on();
  data += (int64_t)blockIdx.z * 4 * V * 2;
  ctrl += blockIdx.z;
  if (!should_run<T>(ctrl, check_active)) return;
  count_run(ctrl, tkid);
  using V2 = typename vec2<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T> *tile = reinterpret_cast<cx<T> *>(smem_raw);
  cx<T> *twb = tile + pd.rows * pd.pitch;
  const cx<T> *tw[2] = {twb, twb + pd.ph[0].N};
  for (int a = 0; a < pd.nax; ++a) {
    const cx<T> *src = reinterpret_cast<const cx<T> *>(tb.tw[pd.ph[a].mu]);
    cx<T> *dst = twb + (a ? pd.ph[0].N : 0);
    for (int k = threadIdx.x; k < pd.ph[a].N; k += blockDim.x) dst[k] = src[k];
  }
  V2 *field = reinterpret_cast<V2 *>(data + (int64_t)blockIdx.y * V * 2);
  // this thread's column (column form), or the tile's run of elements (row form)
  const int c = threadIdx.x & (pd.C - 1), row0 = threadIdx.x >> pd.logC, rstep = blockDim.x >> pd.logC;
  int64_t base = 0;
  int rows = pd.rows, nel = 0;
  if (pd.rowform) {
    const unsigned r0 = blockIdx.x * (unsigned)pd.rows;
    nel = (int)min((unsigned)pd.rows, pd.nrow - r0) * (int)pd.dnx.d;
    base = (int64_t)r0 * pd.dnx.d;
    for (int e = threadIdx.x; e < pd.rows * (int)pd.dnx.d; e += blockDim.x) {
      const unsigned r = div_by(e, pd.dnx), x = e - r * pd.dnx.d;
      V2 v = {};
      if (e < nel) v = ldv(field + base + e);
      tile[r * pd.pitch + x] = from_vec<T>(v);
    }
  } else {
    const unsigned q = blockIdx.x * (unsigned)pd.C + c;
    if (q >= pd.ncol) rows = 0;  // columns beyond the last: zeros in the tile, nothing stored
    base = (int64_t)(q % pd.nin) + (int64_t)(q / pd.nin) * pd.ostride;
#pragma unroll 4
    for (int r = row0; r < pd.rows; r += rstep) {
      V2 v = {};
      if (r < rows) v = ldv(field + base + r * pd.rstride);
      tile[r * pd.pitch + c] = from_vec<T>(v);
    }
  }
  __syncthreads();
  if (pd.mode != 1) {
    for (int a = 0; a < pd.nax; ++a) fft_axis<T, false>(tile, tw[a], pd.ph[a]);
  }
  if (pd.mode == 2) {
    // only column passes end with the filter; the weight is read at the site's own index
    const T *W = reinterpret_cast<const T *>(tb.weights);
#pragma unroll 4
    for (int r = row0; r < rows; r += rstep) {
      cx<T> &v = tile[r * pd.pitch + c];
      v = scale(v, W[base + r * pd.rstride]);
    }
    __syncthreads();
  }
  if (pd.mode != 0) {
    for (int a = pd.nax - 1; a >= 0; --a) fft_axis<T, true>(tile, tw[a], pd.ph[a]);
  }
  if (pd.rowform) {
    for (int e = threadIdx.x; e < nel; e += blockDim.x) {
      const unsigned r = div_by(e, pd.dnx), x = e - r * pd.dnx.d;
      field[base + e] = to_vec<T>(tile[r * pd.pitch + x]);
    }
  } else {
    for (int r = row0; r < rows; r += rstep) field[base + r * pd.rstride] = to_vec<T>(tile[r * pd.pitch + c]);
  }
}

}  // namespace lgf
