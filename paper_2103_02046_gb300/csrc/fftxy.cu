// FP64-path transforms along x and y, around the fused z solve (zsolve_df.cu): forward, the charged
// block of the doubled mesh to its x-y spectrum in the planes z < n_z; inverse, the potential's x-y
// spectrum to the potential on the mesh's nodes.
//
// A library transform of a plane does all of its rows and columns in FP64, on two FP64 lanes per
// clock and SM. Here only the rows y < n_y are transformed along x (the others are zero on the way
// in and not read on the way out), and the first pass of a column that is half zero and the last
// pass of one that is half wanted do half of the work.
//
// Forward in double-float, on the FP32 pipes: its rounding errors, about 2^-49 of the values met,
// are multiplied by the Green's function, which falls with k, before they reach the potential. The
// inverse in FP64: what rounds there is the potential itself, a few hundred times larger than the
// differences between nodes that make the force. With the inverse in double-float too the error of
// the forces against 64 bits was 3.3e-13 instead of 1.8e-13 (400,000 particles on 128^3).
//
// x: two rows, y and y + 1, make one complex column (row y + i times row y + 1), whose spectrum Z
// gives theirs as (Z(k) + conj Z(-k)) / 2 and (Z(k) - conj Z(-k)) / 2i; back the same way.
// y: columns of consecutive kx in one plane, in place.
// A block holds 1024 points (128 threads, an 8-point butterfly each a pass) for lengths up to 128,
// so that a 64^3 mesh still makes several blocks an SM, and 2048 for longer ones, whose columns
// then stand 128 bytes wide in memory up to length 256.
//
// 64^3 mesh: 13 + 12 us forward (x, y), 31 + 19 us back; 128^3: 50 + 65 and 192 + 109 us. The inverse
// is bound by the FP64 unit. With cuFFT in their place a gradient of 4096 particles on 64^3 (103
// solves) took 36.0 ms instead of 21.9, an evaluation of 2,097,152 particles on 128^3 5.02 ms instead
// of 4.03.
#include <algorithm>
#include <cmath>

#include "dfft.cuh"

namespace p3m {
namespace {

// a block's share: threads, columns of length N
inline int xy_threads(int N) { return N <= 128 ? 128 : 256; }
inline int log2_of(int N) {
  int l = 0;
  while ((1 << l) < N) ++l;
  return l;
}
inline size_t xy_smem(int N) {
  const int cols = 8 * xy_threads(N) / N;
  return sizeof(CD) * (static_cast<size_t>(cols) * dcolumn(N) + N);
}

__device__ __forceinline__ F2 halved(F2 a) { return F2{0.5f * a.hi, 0.5f * a.lo}; }

// Rows of the charged block -> their spectra, spec[(z My + y) Hx + kx], y < n_y, z < n_z.
__global__ void __launch_bounds__(256, 3)
    k_xfwd_df(Geom g, int logN, int padN, const double* __restrict__ q,
              const CD* __restrict__ tw_g, const unsigned long long* __restrict__ bound,
              CD* __restrict__ spec) {
  extern __shared__ CD sm[];
  const int N = 1 << logN, threads = blockDim.x;
  const int logC = 3 + 31 - __clz(threads) - logN;  // columns (pairs of rows) to a block
  const int C = 1 << logC, tpc = N >> 3;
  CD* A = sm;
  CD* tw = sm + C * padN;
  const int nx = g.n[0], ny = g.n[1], My = g.M[1], Hx = N / 2 + 1;
  const int nyb = (ny + 2 * C - 1) / (2 * C);
  const int z = blockIdx.x / nyb, y0 = (blockIdx.x - z * nyb) * 2 * C;
  const int tid = threadIdx.x;
  for (int t = tid; t < N; t += threads) tw[t] = tw_g[t];
  const double sc = bound ? w_scale(*bound) : 1.0;
  // the first pass reads the lower half only
  for (int idx = tid; idx < (C << (logN - 1)); idx += threads) {
    const int x = idx & (N / 2 - 1), cc = idx >> (logN - 1), y = y0 + 2 * cc;
    const double* row = q + (static_cast<size_t>(z) * My + y) * N + x;
    CD v = cd_zero();
    if (x < nx) {
      if (y < ny) v.x = dfm::split_double(bound ? sc * row[0] : row[0]);
      if (y + 1 < ny) v.y = dfm::split_double(bound ? sc * row[N] : row[N]);
    }
    A[cc * padN + dpad(x)] = v;
  }
  __syncthreads();
  const int c = tid / tpc;
  dcolumn_fft<true>(A + c * padN, logN, tid - c * tpc, tpc, tw);
  for (int idx = tid; idx < C * Hx; idx += threads) {
    const int cc = idx / Hx, k = idx - cc * Hx, y = y0 + 2 * cc;
    if (y >= ny) continue;
    const CD a = A[cc * padN + dpad(k)], b = A[cc * padN + dpad((N - k) & (N - 1))];
    CD* out = spec + (static_cast<size_t>(z) * My + y) * Hx + k;
    out[0] = CD{halved(dadd(a.x, b.x)), halved(dsub(a.y, b.y))};
    if (y + 1 < ny) out[Hx] = CD{halved(dadd(a.y, b.y)), halved(dsub(b.x, a.x))};
  }
}

// The way back: spectra of the rows y < n_y, z < n_z -> the potential on the nodes.
__global__ void __launch_bounds__(256, 3)
    k_xinv(Geom g, int logN, int padN, const CZ* __restrict__ spec,
              const CZ* __restrict__ tw_g, const unsigned long long* __restrict__ bound,
              double* __restrict__ phi) {
  extern __shared__ CZ smz[];
  const int N = 1 << logN, threads = blockDim.x;
  const int logC = 3 + 31 - __clz(threads) - logN;
  const int C = 1 << logC, tpc = N >> 3;
  CZ* A = smz;
  CZ* tw = smz + C * padN;
  const int nx = g.n[0], ny = g.n[1], My = g.M[1], Hx = N / 2 + 1;
  const int nyb = (ny + 2 * C - 1) / (2 * C);
  const int z = blockIdx.x / nyb, y0 = (blockIdx.x - z * nyb) * 2 * C;
  const int tid = threadIdx.x;
  for (int t = tid; t < N; t += threads) tw[t] = tw_g[t];
  for (int idx = tid; idx < C * Hx; idx += threads) {
    const int cc = idx / Hx, k = idx - cc * Hx, y = y0 + 2 * cc;
    const CZ* in = spec + (static_cast<size_t>(z) * My + y) * Hx + k;
    CZ a{}, b{};
    if (y < ny) a = in[0];
    if (y + 1 < ny) b = in[Hx];
    if (k == 0 || k == N / 2) {  // real for a real row
      A[cc * padN + dpad(k)] = CZ{a.x, b.x};
    } else {
      A[cc * padN + dpad(k)] = CZ{a.x - b.y, a.y + b.x};
      A[cc * padN + dpad(N - k)] = CZ{a.x + b.y, b.x - a.y};
    }
  }
  __syncthreads();
  const int c = tid / tpc;
  dcolumn_fft<false>(A + c * padN, logN, tid - c * tpc, tpc, tw);
  const double sc = bound ? w_unscale(*bound) : 1.0;
  for (int idx = tid; idx < (C << (logN - 1)); idx += threads) {
    const int x = idx & (N / 2 - 1), cc = idx >> (logN - 1), y = y0 + 2 * cc;
    if (x >= nx || y >= ny) continue;
    const CZ v = A[cc * padN + dpad(x)];
    double* row = phi + (static_cast<size_t>(z) * My + y) * N + x;
    row[0] = bound ? sc * v.x : v.x;
    if (y + 1 < ny) row[N] = bound ? sc * v.y : v.y;
  }
}

// Columns along y of the planes z < n_z, in place: forward from the rows y < n_y to all ky, or back
// from all ky to the rows y < n_y.
template <bool kForward, typename E>
__global__ void __launch_bounds__(256, 3)
    k_ycols(Geom g, int logN, int padN, E* __restrict__ spec, const E* __restrict__ tw_g) {
  extern __shared__ float4 smy[];
  static_assert(sizeof(E) == sizeof(float4), "16-byte elements");
  E* sm = reinterpret_cast<E*>(smy);
  const int N = 1 << logN, threads = blockDim.x;
  const int logC = 3 + 31 - __clz(threads) - logN;
  const int C = 1 << logC, tpc = N >> 3;
  E* A = sm;
  E* tw = sm + C * padN;
  const int ny = g.n[1], Hx = g.M[0] / 2 + 1, cols = g.n[2] * Hx;
  const int tid = threadIdx.x, mine = tid & (C - 1);
  // column number col0 + cc counts (z, kx), kx fastest: no block is part empty but the last
  const int col = blockIdx.x * C + mine;
  const int z = col / Hx, kx = col - z * Hx;
  E* base = spec + static_cast<size_t>(z) * N * Hx + kx;
  for (int t = tid; t < N; t += threads) tw[t] = tw_g[t];
  const int in = kForward ? N / 2 : N, out = kForward ? N : N / 2;
  for (int y = tid >> logC; y < in; y += threads >> logC)
    A[mine * padN + dpad(y)] = (col < cols && (!kForward || y < ny))
                                   ? base[static_cast<size_t>(y) * Hx]
                                   : c_zero<E>();
  __syncthreads();
  const int c = tid / tpc;
  dcolumn_fft<kForward>(A + c * padN, logN, tid - c * tpc, tpc, tw);
  if (col >= cols) return;
  for (int y = tid >> logC; y < out; y += threads >> logC)
    if (kForward || y < ny) base[static_cast<size_t>(y) * Hx] = A[mine * padN + dpad(y)];
}

// tables of e^{-2 pi i t / M} (zsolve_df_setup): Mz, Mx, My in double-float, Mx, My in FP64
const CD* table_df(const p3m_ctx* c, int axis) {
  return reinterpret_cast<const CD*>(c->ztw) + c->g.M[2] + (axis == 1 ? c->g.M[0] : 0);
}
const CZ* table_fp64(const p3m_ctx* c, int axis) {
  return reinterpret_cast<const CZ*>(c->ztw) + c->g.M[2] + c->g.M[0] + c->g.M[1] +
         (axis == 1 ? c->g.M[0] : 0);
}

unsigned x_blocks(const p3m_ctx* c) {
  const int rows = 2 * (8 * xy_threads(c->g.M[0]) / c->g.M[0]);
  return static_cast<unsigned>((c->g.n[1] + rows - 1) / rows * c->g.n[2]);
}
unsigned y_blocks(const p3m_ctx* c) {
  const int C = 8 * xy_threads(c->g.M[1]) / c->g.M[1];
  const int cols = c->g.n[2] * (c->g.M[0] / 2 + 1);
  return static_cast<unsigned>((cols + C - 1) / C);
}

}  // namespace

bool fftxy_length(int N) { return N >= 16 && N <= 2048 && (N & (N - 1)) == 0; }

bool fftxy_supported(const p3m_ctx* c) {
  return c->zsolve_df && fftxy_length(c->g.M[0]) && fftxy_length(c->g.M[1]);
}

cudaError_t fftxy_setup(p3m_ctx* c) {
  cudaError_t e = cudaSuccess;
  auto room = [&](auto kern) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(xy_smem(2048)));
  };
  room(k_xfwd_df);
  room(k_xinv);
  room(k_ycols<true, CD>);
  room(k_ycols<false, CZ>);
  c->fftxy = e == cudaSuccess;
  return e;
}

void launch_fftxy_forward(const p3m_ctx* c, bool scaled) {
  const Geom& g = c->g;
  CD* spec = static_cast<CD*>(c->qhat);
  k_xfwd_df<<<x_blocks(c), xy_threads(g.M[0]), xy_smem(g.M[0]), c->work>>>(
      g, log2_of(g.M[0]), dcolumn(g.M[0]), static_cast<const double*>(c->qpad), table_df(c, 0),
      scaled ? c->wbound : nullptr, spec);
  k_ycols<true, CD><<<y_blocks(c), xy_threads(g.M[1]), xy_smem(g.M[1]), c->work>>>(
      g, log2_of(g.M[1]), dcolumn(g.M[1]), spec, table_df(c, 1));
}

void launch_fftxy_inverse(const p3m_ctx* c, bool scaled) {
  const Geom& g = c->g;
  CZ* spec = static_cast<CZ*>(c->phihat);
  k_ycols<false, CZ><<<y_blocks(c), xy_threads(g.M[1]), xy_smem(g.M[1]), c->work>>>(
      g, log2_of(g.M[1]), dcolumn(g.M[1]), spec, table_fp64(c, 1));
  k_xinv<<<x_blocks(c), xy_threads(g.M[0]), xy_smem(g.M[0]), c->work>>>(
      g, log2_of(g.M[0]), dcolumn(g.M[0]), spec, table_fp64(c, 0),
      scaled ? c->wbound : nullptr, static_cast<double*>(c->phireal));
}

}  // namespace p3m
