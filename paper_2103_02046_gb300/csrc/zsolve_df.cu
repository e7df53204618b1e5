// FP64-path long-range solve along z, fused and in double-float arithmetic: for each (kx, ky)
// column of the x-y transformed charge, the forward transform along z, the Green's-function
// multiply of eq. (phi_L) with the cathode image term of eq. (GreenFunc_planar_cathode), and the
// inverse transform of the potential spectrum, keeping only the n_z planes that the x-y inverse
// transform reads. The FP64 path's numbers enter and leave as doubles; inside, every real is an
// unevaluated sum hi + lo of two FP32 numbers (about 48 significant bits), so the butterflies
// run on GB300's FP32 pipes instead of its scarce FP64 units, with a rounding error of a few
// 1e-15 per operation (the FP64 path's bound against the oracle is 1e-12).
//
// Mesh layout as in the FP32 fused solve: element (z, ky, kx) of a spectrum at (z My + ky) Hx +
// kx, Hx = Mx/2 + 1; the charge is non-zero only in planes z < n_z <= Mz / 2. With
// base = Kf Q - Ki Q(-kz) (Ki absent without the cathode), phihat = base.
//
// Transforms: power-of-two Mz in [16, 2048], radix-8 Stockham autosort passes (then one radix-4
// or radix-2 pass when log2 Mz is not a multiple of 3) in shared memory; twiddles from a table
// computed in extended precision on the host and split into double-float. A block holds
// C = 2048 / Mz columns (one 8-point butterfly per thread and pass, 256 threads), taken from the whole
// (ky, kx) plane, since rows of Mx/2 + 1 columns would leave one block in five (64^3 mesh) nearly empty.
// The Green's spectra are held in double-float from context creation on, and the charge spectrum
// comes in double-float from fftxy.cu or is split by integer operations, so that no FP64 instruction
// runs per element but the final conversion.
//
// Bound by latency and shared memory: barriers between passes at 24 warps an SM. 128^3 mesh: 384 us
// with columns a multiple of 16 bytes x 32 apart (bank conflicts on two of three wavefronts), 128
// registers and two blocks an SM; 283 us with columns an odd number of elements apart and 16-byte
// accesses; 240 us with 80 registers and three blocks.
#include <algorithm>
#include <cmath>
#include <vector>

#include "dfft.cuh"

namespace p3m {
namespace {

constexpr long double kTwoPiL = 6.283185307179586476925286766559005768L;
constexpr int kDThreads = 256;
constexpr int kDElems = 2048;  // columns per block x Mz

// One block: C consecutive columns, counted (ky, kx) with kx fastest (consecutive in memory; no block
// is part empty but the last). kDF: the charge spectrum comes in double-float (fftxy.cu).
template <bool kDF>
__global__ void __launch_bounds__(kDThreads, 3)
    k_zsolve_df(Geom g, int logN, int padN, const void* __restrict__ qhat,
                const F2* __restrict__ kf, const CD* __restrict__ ki,
                const CD* __restrict__ tw_g, double2* __restrict__ phihat,
                double* __restrict__ energy) {
  extern __shared__ CD zd[];
  const int N = 1 << logN;
  const int logC = 11 - logN;  // C = 2048 / N
  const int C = 1 << logC;
  const int tpc = N >> 3;      // threads per column
  CD* A = zd;                  // the columns, then their spectra, then the potential
  CD* tw = zd + C * padN;      // e^{-2 pi i t / N}, t < N
  const int Hx = g.M[0] / 2 + 1, My = g.M[1], nz = g.n[2];
  const int plane = My * Hx, col0 = static_cast<int>(blockIdx.x) << logC;
  const int tid = threadIdx.x;
  for (int t = tid; t < N; t += kDThreads) tw[t] = tw_g[t];
  // the charged planes z < n_z of the columns, zero above
  for (int idx = tid; idx < kDElems; idx += kDThreads) {
    const int z = idx >> logC, k = col0 + (idx & (C - 1));
    const size_t at = static_cast<size_t>(z) * plane + k;
    CD v = cd_zero();
    if (z < nz && k < plane) {
      if constexpr (kDF)
        v = static_cast<const CD*>(qhat)[at];
      else
        v = cd_split(static_cast<const double2*>(qhat)[at]);
    }
    A[(idx & (C - 1)) * padN + dpad(z)] = v;
  }
  __syncthreads();
  const int c = tid / tpc, i0 = tid - c * tpc;
  CD* col = A + c * padN;
  dcolumn_fft<true>(col, logN, i0, tpc, tw);
  // Green's-function multiply, kz paired with -kz (the image term reads Q(-kz))
  double e = 0.0;
  const int nmul = (N / 2 + 1) << logC;  // (kz, -kz) pairs x columns
  for (int idx = tid; idx < nmul; idx += kDThreads) {
    const int cc = idx & (C - 1), kz = idx >> logC;
    const int kz2 = (N - kz) & (N - 1);
    const int k = col0 + cc;
    if (k >= plane) continue;
    CD* cl = A + cc * padN;
    const CD a = cl[dpad(kz)], b = cl[dpad(kz2)];
    const size_t ia = static_cast<size_t>(kz) * plane + k,
                 ib = static_cast<size_t>(kz2) * plane + k;
    const F2 fa = kf[ia], fb = kf[ib];
    CD ba{dfm::mul(a.x, fa), dfm::mul(a.y, fa)};
    CD bb{dfm::mul(b.x, fb), dfm::mul(b.y, fb)};
    if (ki) {
      ba = cd_sub(ba, cd_mul(ki[ia], b));
      bb = cd_sub(bb, cd_mul(ki[ib], a));
    }
    if (energy) {
      const int kxx = k % Hx;
      const double wx = (kxx == 0 || 2 * kxx == g.M[0]) ? 1.0 : 2.0;
      double ee = wx * (d_of(dadd(dfm::mul(a.x, ba.x), dfm::mul(a.y, ba.y))));
      if (kz2 != kz) ee += wx * d_of(dadd(dfm::mul(b.x, bb.x), dfm::mul(b.y, bb.y)));
      e += ee;
    }
    cl[dpad(kz)] = ba;
    if (kz2 != kz) cl[dpad(kz2)] = bb;
  }
  __syncthreads();
  dcolumn_fft<false>(col, logN, i0, tpc, tw);
  // the planes z < n_z of the potential spectrum
  for (int idx = tid; idx < (nz << logC); idx += kDThreads) {
    const int z = idx >> logC, cc = idx & (C - 1);
    const int k = col0 + cc;
    if (k >= plane) continue;
    phihat[static_cast<size_t>(z) * plane + k] = cd_to(A[cc * padN + dpad(z)]);
  }
  if (energy) {
    for (int o = 16; o > 0; o >>= 1) e += __shfl_down_sync(0xffffffffu, e, o);
    if ((tid & 31) == 0 && e != 0.0) atomicAdd(energy, e);
  }
}

// The Green's spectra, FP64 as built, to double-float in place (8 bytes each either way), once
// at context creation: the fused solve is then their only reader.
__global__ void k_spectra_to_df(double* __restrict__ v, size_t n) {
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (i < n) {
    const F2 d = dfm::split_double_fp64(v[i]);
    reinterpret_cast<F2*>(v)[i] = d;
  }
}

size_t zsolve_df_smem_bytes(int N) {
  return sizeof(CD) * (static_cast<size_t>(kDElems / N) * dcolumn(N) + N);
}

}  // namespace

bool zsolve_df_supported(const p3m_ctx* c) {
  // Lengths below 64 only with the x-y transforms of fftxy.cu (which scale what they pass on into
  // FP32's exponents): on a 16^3 mesh the solve is then five kernels of a few microseconds instead of
  // cuFFT's nine and the multiply.
  const int* M = c->g.M;
  if (c->fp32 || c->det || c->g.pm_bc == 2 || !fftxy_length(M[2])) return false;
  return M[2] >= 64 || (fftxy_length(M[0]) && fftxy_length(M[1]));
}

cudaError_t zsolve_df_setup(p3m_ctx* c) {
  const int N = c->g.M[2];
  // the tables of Mz, Mx, My in double-float, then those of Mx, My in FP64
  std::vector<float> tw;
  std::vector<double> tz;
  for (int axis : {2, 0, 1})
    for (int t = 0, M = c->g.M[axis]; t < M; ++t) {
      // in extended precision: the angle's rounding in FP64 alone is worth several ulp
      const long double ang = -kTwoPiL * t / M;
      for (long double v : {std::cos(ang), std::sin(ang)}) {
        const float h = static_cast<float>(v);
        tw.push_back(h);
        tw.push_back(static_cast<float>(v - h));
        if (axis != 2) tz.push_back(static_cast<double>(v));
      }
    }
  static_assert(sizeof(CD) == 4 * sizeof(float), "complex double-float layout");
  const size_t tw_bytes = sizeof(float) * tw.size(), tz_bytes = sizeof(double) * tz.size();
  cudaError_t e = cudaMalloc(&c->ztw, tw_bytes + tz_bytes);
  if (e == cudaSuccess) e = cudaMemcpy(c->ztw, tw.data(), tw_bytes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(reinterpret_cast<char*>(c->ztw) + tw_bytes, tz.data(), tz_bytes,
                   cudaMemcpyHostToDevice);
  auto room = [&](auto kern) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               static_cast<int>(zsolve_df_smem_bytes(N)));
  };
  room(k_zsolve_df<false>);
  room(k_zsolve_df<true>);
  // the spectra: n_cplx reals (free kernel) and n_cplx complex values (image kernel)
  auto convert = [&](void* p, size_t n) {
    if (p == nullptr || e != cudaSuccess) return;
    k_spectra_to_df<<<static_cast<unsigned>((n + 255) / 256), 256, 0, c->work>>>(
        static_cast<double*>(p), n);
    e = cudaGetLastError();
  };
  convert(c->khat_f, c->n_cplx);
  convert(c->khat_i, 2 * c->n_cplx);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->work);
  return e;
}

void launch_zsolve_df(const p3m_ctx* c, bool want_energy) {
  const Geom& g = c->g;
  const int N = g.M[2];
  int logN = 0;
  while ((1 << logN) < N) ++logN;
  const int C = kDElems / N;
  const int64_t cols = static_cast<int64_t>(g.M[0] / 2 + 1) * g.M[1];
  const unsigned blocks = static_cast<unsigned>((cols + C - 1) / C);
  double* en = want_energy ? c->energy_acc + 1 : nullptr;
  auto kern = c->fftxy ? k_zsolve_df<true> : k_zsolve_df<false>;
  kern<<<blocks, kDThreads, zsolve_df_smem_bytes(N), c->work>>>(
      g, logN, dcolumn(N), c->qhat, static_cast<const F2*>(c->khat_f),
      static_cast<const CD*>(c->khat_i), reinterpret_cast<const CD*>(c->ztw),
      static_cast<double2*>(c->phihat), en);
}

}  // namespace p3m
