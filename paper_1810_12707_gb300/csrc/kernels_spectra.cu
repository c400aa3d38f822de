// kernels_spectra.cu -- shell spectra and velocity-derivative statistics of one instance (paper,
// section "for hydrodynamic flow": theta' = <(du_i/dx_i)^2>^(1/2) and the skewness
// S_3 = <(du_1/dx_1)^3> / <(du_1/dx_1)^2>^(3/2); kinetic and magnetic energy spectra), with the
// kinetic and magnetic helicities and the largest |div B| on the grid.
//
// The velocity u = m / rho exists only on the grid, so one fused x pass brings rho and m to real
// rows (inverse x), divides, and sends u back (forward x); the y and z column passes then give the
// truncated spectrum u_hat.  A mode k belongs to shell s = round(|k|), decided exactly in integer
// arithmetic: (2s - 1)^2 <= 4|k|^2 < (2s + 1)^2 (|k|^2 is an integer, so no mode lies on a shell
// boundary).  Warps walk the rows of the truncated half spectrum and add each shell's run of k_x to
// their own bins in a fixed order, so the spectra are bitwise reproducible.
#include "fft_device.cuh"
#include "fp64_util.cuh"
#include "launch_util.cuh"

namespace mhd {

namespace {

constexpr int kMaxThreads = 384;

constexpr int pairs_for(int n) { return (n / 8) >= 16 ? 1 : 16 / (n / 8); }

constexpr int threads_for(int tpp, int pencils) {
  int g = kMaxThreads / tpp;
  if (g > pencils) g = pencils;
  int t = g * tpp;
  return (t + 31) / 32 * 32;
}

}  // namespace

// rho, m (fields 0..3 of `in`, [f][z][y][kx <= K] after the inverse y pass) -> u = m / rho on the
// grid -> forward x -> out [3][z][y][kx <= K].  Two real rows per complex pencil, as in the flux
// pass; a block owns PAIRS row pairs (256^3 1.39 -> 0.90 ms with the rows straight from and to their
// spectra and corrected quotients for the divisions).
template <int N>
__global__ void __launch_bounds__(kMaxThreads) velocity_x_kernel(const cplx64 *__restrict__ in,
                                                                  cplx64 *__restrict__ out,
                                                                  const TwFx *__restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx64 *sm = reinterpret_cast<cplx64 *>(smem_raw);
  constexpr int P = pencil_pitch<cplx64>(N), TPP = tpp_for<N, 8>();
  constexpr int PAIRS = pairs_for(N);
  constexpr size_t NN = (size_t)N * N;
  constexpr int NX = (N - 1) / 3 + 1;
  const size_t row0 = (size_t)blockIdx.x * PAIRS * 2;
  const int nthr = blockDim.x;
  const int g = threadIdx.x / TPP, t = threadIdx.x - g * TPP, G = nthr / TPP;

  for (int base = 0; base < 4 * PAIRS; base += G) {
    const int id = base + g;
    const bool active = g < G && id < 4 * PAIRS;
    const int f = active ? id % 4 : 0, p = active ? id / 4 : 0;
    RowPair<N, cplx64, 8> x;
    x.load(in + ((size_t)f * NN + row0 + 2 * p) * NX, t, active);
    rows_inverse<N, cplx64, 8, false>(sm + (active ? id : 0) * P, t, active, x, tw);
  }
  __syncthreads();

  for (int q = threadIdx.x; q < PAIRS * N; q += nthr) {
    const int p = q / N, j = q - p * N;
    cplx64 *b = sm + p * 4 * P + sm_idx<cplx64>(j);
    const cplx64 rho = b[0];
    if (rcp3_covers(rho.re) && rcp3_covers(rho.im)) {
      const double i0 = rcp3(rho.re), i1 = rcp3(rho.im);
#pragma unroll
      for (int f = 1; f < 4; ++f) {
        const cplx64 m = b[f * P];
        b[f * P] = cplx64{quotient(m.re, rho.re, i0), quotient(m.im, rho.im, i1)};
      }
    } else {
      for (int f = 1; f < 4; ++f) {
        const cplx64 m = b[f * P];
        b[f * P] = cplx64{m.re / rho.re, m.im / rho.im};
      }
    }
  }
  __syncthreads();

  for (int base = 0; base < 3 * PAIRS; base += G) {
    const int id = base + g;
    const bool active = g < G && id < 3 * PAIRS;
    const int f = active ? id % 3 : 0, p = active ? id / 3 : 0;
    // (scale 2^-1: the split's factor 1/2)
    rows_forward<N, cplx64, 8, true>(sm + (active ? p * 4 + 1 + f : 0) * P, t, active,
                                     out + ((size_t)f * NN + row0 + 2 * p) * NX, tw, -1, [](cplx64 v) { return v; });
  }
}

// Re(conj(f) . (i k x f)) of one mode: with t = k x f, (i t)_a = (-Im t_a, Re t_a).
__device__ __forceinline__ double curl_dot(double kx, double ky, double kz, cplx64 fx, cplx64 fy, cplx64 fz) {
  const cplx64 tx{ky * fz.re - kz * fy.re, ky * fz.im - kz * fy.im};
  const cplx64 ty{kz * fx.re - kx * fz.re, kz * fx.im - kx * fz.im};
  const cplx64 tz{kx * fy.re - ky * fx.re, kx * fy.im - ky * fx.im};
  return (fx.im * tx.re - fx.re * tx.im) + (fy.im * ty.re - fy.re * ty.im) + (fz.im * tz.re - fz.re * tz.im);
}

// Shell sums.  uh, bh: 3 truncated spectra each (stride `spec`); per shell s the five sums
// (sum w |u_hat|^2 / 2, sum w |B_hat|^2 / 2, sum w |k . u_hat|^2, sum w Re(conj(u_hat) . i k x u_hat),
// sum w Re(conj(B_hat) . i k x B_hat) / |k|^2), with w = 1 on the k_x = 0 plane and 2 elsewhere (the
// half spectrum stands for k and -k).  By Parseval the last two are the shell's shares of the kinetic
// helicity <u . curl u> and of the magnetic helicity <A . B>, A_hat = i k x B_hat / |k|^2 (Coulomb
// gauge, A_hat(0) = 0).  dh = i k_x u_hat_x and gh = i k . B_hat on every mode.
// A warp takes 32 consecutive k_x of one (k_z, k_y) row, so that every lane has a mode and the FP64
// pipe, which bounds this, works on full warps; along a row the shells come in order, so each
// shell's lanes are a run whose sums one lane per quantity adds up from shared memory into the warp's
// own bins.  The warps' rows, the runs and the blocks' sums are added in a fixed order.  A thread per
// row and shell, the earlier form, kept a quarter of its lanes busy: 256^3 1.43 -> 0.545 ms.
constexpr int kShellWarps = 4;
__global__ void __launch_bounds__(32 * kShellWarps) shell_kernel(const cplx64 *__restrict__ uh,
                                                                 const cplx64 *__restrict__ bh,
                                                                 cplx64 *__restrict__ dh, cplx64 *__restrict__ gh,
                                                                 double *__restrict__ part, int K, int ns) {
  extern __shared__ double shell_sm[];  // [warp][5 ns] bins, [warp][32][5] terms
  __shared__ int shell_of[kShellWarps][32];
  const int NX = K + 1, NK = 2 * K + 1;
  const size_t spec = (size_t)NK * NK * NX;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double *bins = shell_sm + (size_t)warp * 5 * ns;
  double *term = shell_sm + (size_t)kShellWarps * 5 * ns + warp * 160;
  for (int i = lane; i < 5 * ns; i += 32) bins[i] = 0.0;
  __syncwarp();
  const int chunks = (NX + 31) / 32, items = NK * NK * chunks;
  for (int it = blockIdx.x * kShellWarps + warp; it < items; it += gridDim.x * kShellWarps) {
    const int r = it / chunks, kxi = (it - r * chunks) * 32 + lane;
    const int kzi = kept_wave(r / NK, K), kyi = kept_wave(r % NK, K);
    const bool valid = kxi <= K;
    const int k2 = kxi * kxi + kyi * kyi + kzi * kzi;
    // round(|k|): the integer s with (2s - 1)^2 <= 4 |k|^2 < (2s + 1)^2
    int s = (int)(sqrtf((float)k2) + 0.5f);
    while ((2 * s + 1) * (2 * s + 1) <= 4 * k2) ++s;
    while (s > 0 && (2 * s - 1) * (2 * s - 1) > 4 * k2) --s;
    if (valid) {
      const size_t m = (size_t)r * NX + kxi;
      const double kx = kxi, ky = kyi, kz = kzi;
      const double w = kxi == 0 ? 1.0 : 2.0;
      const cplx64 ux = uh[m], uy = uh[spec + m], uz = uh[2 * spec + m];
      const cplx64 bx = bh[m], by = bh[spec + m], bz = bh[2 * spec + m];
      double *e = term + 5 * lane;
      e[0] = 0.5 * w * (ux.re * ux.re + ux.im * ux.im + uy.re * uy.re + uy.im * uy.im + uz.re * uz.re + uz.im * uz.im);
      e[1] = 0.5 * w * (bx.re * bx.re + bx.im * bx.im + by.re * by.re + by.im * by.im + bz.re * bz.re + bz.im * bz.im);
      const double dr = kx * ux.re + ky * uy.re + kz * uz.re, di = kx * ux.im + ky * uy.im + kz * uz.im;
      e[2] = w * (dr * dr + di * di);
      dh[m] = cplx64{-kx * ux.im, kx * ux.re};
      e[3] = w * curl_dot(kx, ky, kz, ux, uy, uz);
      const double k2d = k2 > 0 ? (double)k2 : 1.0, c = w * curl_dot(kx, ky, kz, bx, by, bz);
      e[4] = k2 > 0 ? quotient(c, k2d, rcp3(k2d)) : 0.0;
      const double gr = kx * bx.re + ky * by.re + kz * bz.re, gi = kx * bx.im + ky * by.im + kz * bz.im;
      gh[m] = cplx64{-gi, gr};
    }
    shell_of[warp][lane] = s;
    const int before = __shfl_up_sync(0xffffffffu, s, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, valid && (lane == 0 || s != before));
    const int count = __popc(__ballot_sync(0xffffffffu, valid));
    __syncwarp();
    const int runs = __popc(heads);
    for (int i = lane; i < 5 * runs; i += 32) {
      const int j = i / 5, q = i - 5 * j;
      const int first = __fns(heads, 0, j + 1), end = j + 1 < runs ? (int)__fns(heads, 0, j + 2) : count;
      double v = term[5 * first + q];
      for (int l = first + 1; l < end; ++l) v += term[5 * l + q];
      bins[5 * shell_of[warp][first] + q] += v;
    }
    __syncwarp();
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 5 * ns; i += blockDim.x) {
    double v = shell_sm[i];
#pragma unroll
    for (int w = 1; w < kShellWarps; ++w) v += shell_sm[(size_t)w * 5 * ns + i];
    part[(size_t)blockIdx.x * 5 * ns + i] = v;
  }
}

// out[i] = sum over the blocks of part[block][i], i < n: 32 sums per block, 8 threads each, in a fixed
// order.
__global__ void __launch_bounds__(256) shell_sum_kernel(const double *__restrict__ part, int blocks, int n,
                                                        double *__restrict__ out) {
  __shared__ double red[8][32];
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + l;
  double v = 0.0;
  if (i < n)
    for (int b = w; b < blocks; b += 8) v += part[(size_t)b * n + i];
  red[w][l] = v;
  __syncthreads();
  if (w == 0 && i < n) {
    for (int k = 1; k < 8; ++k) v += red[k][l];
    out[i] = v;
  }
}

// part[block][2] = (sum d^2, sum d^3) over a fixed grid-stride share of the n values of d.
__global__ void __launch_bounds__(256) moments_kernel(const double *__restrict__ d, size_t n, double *__restrict__ part) {
  __shared__ double red[32];
  double s2 = 0.0, s3 = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double v = d[i];
    s2 += v * v;
    s3 += v * v * v;
  }
  const double a = block_sum(s2, red);
  const double b = block_sum(s3, red);
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = a;
    part[2 * blockIdx.x + 1] = b;
  }
}

// part[block] = max |v| over a fixed grid-stride share of the n values of v (a NaN is kept): on the
// magnitudes' bits, which order as the magnitudes do with NaNs above infinity.  FP64 comparisons held
// this to 0.9 TB/s (256^3 0.150 -> 0.100 ms).
__global__ void __launch_bounds__(256) absmax_kernel(const double *__restrict__ v, size_t n, double *__restrict__ part) {
  __shared__ unsigned long long red[8];
  unsigned long long m = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(v[i]) & 0x7fffffffffffffffull);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = max(m, red[w]);
    part[blockIdx.x] = __longlong_as_double((long long)m);
  }
}

namespace {

template <int N>
cudaError_t velocity_n(const cplx64 *in, cplx64 *out, const Dims &d, const TwFx *tw, cudaStream_t s) {
  constexpr int PAIRS = pairs_for(N);
  const int blocks = N * N / (2 * PAIRS);
  const int threads = threads_for(tpp_for<N, 8>(), 4 * PAIRS);
  const size_t smem = (size_t)4 * PAIRS * pencil_pitch<cplx64>(N) * sizeof(cplx64);
  if (smem > 48 * 1024) {
    cudaError_t e = ensure_smem<velocity_x_kernel<N>>((int)smem);
    if (e != cudaSuccess) return e;
  }
  velocity_x_kernel<N><<<blocks, threads, smem, s>>>(in, out, tw);
  return cudaGetLastError();
}

}  // namespace

int num_shells(int k) {
  // round(sqrt(3) k): the largest s with (2s - 1)^2 <= 12 k^2
  int s = 0;
  while ((long long)(2 * s + 1) * (2 * s + 1) <= 12LL * k * k) ++s;
  return s + 1;
}

cudaError_t launch_velocity_x(const cplx64 *in, cplx64 *out, const Dims &d, const TwFx *tw, cudaStream_t s) {
  switch (d.n) {
    case 16: return velocity_n<16>(in, out, d, tw, s);
    case 32: return velocity_n<32>(in, out, d, tw, s);
    case 64: return velocity_n<64>(in, out, d, tw, s);
    case 128: return velocity_n<128>(in, out, d, tw, s);
    case 256: return velocity_n<256>(in, out, d, tw, s);
    case 512: return velocity_n<512>(in, out, d, tw, s);
    case 1024: return velocity_n<1024>(in, out, d, tw, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_shells(const cplx64 *uh, const cplx64 *bh, cplx64 *dh, cplx64 *gh, double *part, int blocks,
                          const Dims &d, cudaStream_t s) {
  const int ns = num_shells(d.k), n = 5 * ns;
  const size_t smem = (size_t)kShellWarps * (n + 160) * sizeof(double);
  if (smem > 48 * 1024) {
    cudaError_t e = ensure_smem<shell_kernel>((int)smem);
    if (e != cudaSuccess) return e;
  }
  shell_kernel<<<blocks, 32 * kShellWarps, smem, s>>>(uh, bh, dh, gh, part + n, d.k, ns);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  shell_sum_kernel<<<(n + 31) / 32, 256, 0, s>>>(part + n, blocks, n, part);
  return cudaGetLastError();
}

cudaError_t launch_absmax(const double *v, size_t n, double *part, int blocks, cudaStream_t s) {
  absmax_kernel<<<blocks, 256, 0, s>>>(v, n, part);
  return cudaGetLastError();
}

cudaError_t launch_moments(const double *v, size_t n, double *part, int blocks, cudaStream_t s) {
  moments_kernel<<<blocks, 256, 0, s>>>(v, n, part);
  return cudaGetLastError();
}

}  // namespace mhd
