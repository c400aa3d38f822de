// kernels_col.cu -- FFT passes along a strided axis (y or z) of the truncated spectral layout.
//
// The data of one pass is viewed as [nslab][L][C]: the transform runs along L for each of the
// nslab * C columns; the C columns of a slab are contiguous in memory.  A block takes TC
// consecutive columns of one slab, so every row of the tile is one coalesced segment of TC complex
// values.  The tile is transposed into shared memory as TC pencils of length N (tile_pitch apart,
// which spreads consecutive pencils over the banks), transformed by TC groups of N/VPT threads, and
// written back.
//   inverse (DIR = +1): L = 2K + 1 kept rows in, scattered to their FFT indices with the rest of
//                       the pencil zero (the 2/3-rule truncation), all N rows out;
//   forward (DIR = -1): N rows in, only the 2K + 1 kept rows out, times `scale`.
// Used for: inverse z (state -> z), inverse y, forward y, forward z (-> truncated spectra).
#include "fft_device.cuh"
#include "launch_util.cuh"

#include <type_traits>

namespace mhd {

// Double-float passes at N >= 512 stage the twiddle table (N values, 8 KB at 512) in shared
// memory behind the tile: 4-6 % faster per pass at 512^3 than 16-byte L1 loads per butterfly
// element; at 256^3 the copy per block cost more than it saved.
template <typename CC, int N>
constexpr bool tws_staged() { return std::is_same<CC, cdf>::value && N >= 512; }
template <typename CC, int N>
constexpr size_t tws_bytes() { return tws_staged<CC, N>() ? (size_t)N * sizeof(CC) : 0; }

// Where a thread's rows l = l0 + i TPP (l0 < TPP) lie in a pencil: kept index l at FFT index l, or
// l + N - NK above K, or (all rows) FFT index l.  Addresses are at constant offsets from two base
// pointers where TPP is a multiple of the pad's period; only the row group that straddles K needs
// a selection.
template <int N, int TPP, typename CC>
struct KeptRows {
  static constexpr int K = (N - 1) / 3, UP = N - (2 * K + 1);
  static constexpr bool kConst = TPP % sm_pad<CC>() == 0;
  CC *pen, *lo, *hi;
  unsigned l0;
  __device__ __forceinline__ KeptRows(CC *p, unsigned l) : pen(p), l0(l) {
    lo = p + sm_at<CC>(l);
    hi = p + sm_at<CC>(l + (unsigned)(UP % sm_pad<CC>())) + sm_idx<CC>(UP - UP % sm_pad<CC>());
  }
  template <bool Kept>
  __device__ __forceinline__ CC *row(int i) const {
    const int d = i * TPP;
    if constexpr (!kConst) {
      const unsigned l = l0 + d;
      return pen + sm_at<CC>(Kept && l > (unsigned)K ? l + UP : l);
    } else {
      if (!Kept || d + TPP - 1 <= K) return lo + sm_idx<CC>(d);
      if (d > K) return hi + sm_idx<CC>(d);
      return (l0 + d > (unsigned)K ? hi : lo) + sm_idx<CC>(d);
    }
  }
};

// Distance between a tile's pencils.  The tile's loads and stores go through shared memory with a
// row's tc columns in consecutive lanes, so the L = 128 / element size lanes of one wavefront cover
// max(1, L / tc) consecutive elements of min(tc, L) pencils: a pitch of L / tc modulo L puts them on
// distinct banks (1 for tc >= L).  With the odd pitch of the x passes every access of the tiles
// narrower than L had two-way conflicts: 28 % of the wavefronts of the 256^3 mixed passes.  Groups of
// less than L threads (the smallest grids) keep the odd pitch, their stages have several pencils in a
// wavefront.
template <int N, int TPP, typename CC>
__host__ __device__ __forceinline__ int tile_pitch(int tc) {
  constexpr int L = sm_pad<CC>(), base = sm_idx<CC>(N);
  if constexpr (TPP < L) return base | 1;
  const int want = tc >= L ? 1 : L / tc;  // modulo L
  return base + (want + L - base % L) % L;
}

// CI, CO: element types in and out; CC: type of the transform arithmetic (= the output's).
// A block has TC = 2^tsh columns and TC * N/VPT threads: thread (l0, c) = (tid >> tsh, tid & (TC-1))
// moves rows l0, l0 + N/VPT, ... of column c, so consecutive threads touch consecutive columns of a
// row (coalesced) and no index needs a division.
// VPT: values per thread of the transform (8, or 16 for FP32), so N / VPT threads per column.
// One tile (TC columns of one slab): work item w = slab * ntiles + tile.
template <int N, int DIR, typename CI, typename CO, typename CC, int VPT, typename TW>
__device__ __forceinline__ void col_fft_tile(const CI *__restrict__ in, CO *__restrict__ out, unsigned w, int ntiles,
                                             int tsh, int cols, typename scale_of<CC>::type scale,
                                             const TW *__restrict__ tw, CC *sm) {
  constexpr int TPP = tpp_for<N, VPT>();
  const int P = tile_pitch<N, TPP, CC>(1 << tsh);
  constexpr int K = (N - 1) / 3;  // the 2/3-rule cut-off, fixed by N
  constexpr int NK = 2 * K + 1;
  constexpr int LIN = DIR > 0 ? NK : N;
  constexpr int LOUT = DIR > 0 ? N : NK;
  const int tc = 1 << tsh;
  const int tile = (int)(w % (unsigned)ntiles);
  const size_t slab = w / (unsigned)ntiles;
  const int c = threadIdx.x & (tc - 1);
  const int l0 = threadIdx.x >> tsh;  // 0 .. TPP-1
  const int col = tile * tc + c;
  const bool col_ok = col < cols;

  const CI *src = in + slab * (size_t)LIN * cols + col;
  CC *pen = sm + c * P;
  // fully unrolled (the trip count is a constant), so all of a thread's loads are in flight at once
  constexpr int NLD = (LIN + TPP - 1) / TPP;
  CC v[NLD];
#pragma unroll
  for (int i = 0; i < NLD; ++i) {
    const int l = l0 + i * TPP;
    v[i] = CC{0, 0};
    if (col_ok && (LIN % TPP == 0 || i + 1 < NLD || l < LIN)) v[i] = c_cvt<CC>(src[(size_t)l * cols]);
  }
  const KeptRows<N, TPP, CC> at(pen, (unsigned)l0);
#pragma unroll
  for (int i = 0; i < NLD; ++i) {
    if (LIN % TPP == 0 || i + 1 < NLD || l0 + i * TPP < LIN) *at.template row<(DIR > 0)>(i) = v[i];
  }
  if (DIR > 0) {
    // of the FFT indices K+1 .. N-K-1, outside the kept set, those that the transform reads
    for (unsigned l = l0; l < (unsigned)pencil_zero_count<N>(); l += TPP)
      pen[sm_at<CC>(pencil_zero<N>(l))] = CC{0, 0};
  }
  // double-float at N >= 512: the twiddle table staged in shared memory behind the pencils
  constexpr bool kTws = tws_staged<CC, N>();
  const TW *twp = tw;
  if constexpr (kTws) {
    CC *tws = sm + tc * P;
    for (int i = threadIdx.x; i < N; i += blockDim.x) tws[i] = tw[i];
    twp = tws;
  }
  __syncthreads();

  const int pencil = threadIdx.x / TPP;
  const int t = threadIdx.x - pencil * TPP;
  const bool active = pencil < tc && tile * tc + pencil < cols;
  // fixed-point transforms take `scale`, a power of two there, into their results' exponents
  constexpr bool kFx = std::is_same<TW, TwFx>::value;
  int scale2 = 0;
  if constexpr (kFx && DIR < 0) scale2 = (int)fx_exp(fx_hi(scale)) - 1023;
  pencil_fft<N, DIR, CC, VPT, (DIR > 0), kTws, kFx>(sm + (active ? pencil : 0) * P, t, active, twp,
                                                     scale2);  // inverse: zero-padded
  __syncthreads();  // the store loop reads every pencil

  if (col_ok) {
    CO *dst = out + slab * (size_t)LOUT * cols + col;
    // the double-float inverse passes keep their 64 registers (4 blocks per SM) with a short unroll:
    // 512^3 inverse y 3.24 ms against 3.52
    constexpr int kStoreUnroll = std::is_same<CC, cdf>::value && DIR > 0 ? 2 : 16;
    constexpr int NST = (LOUT + TPP - 1) / TPP;
#pragma unroll(kStoreUnroll)
    for (int i = 0; i < NST; ++i) {
      const int l = l0 + i * TPP;
      if (LOUT % TPP == 0 || i + 1 < NST || l < LOUT) {
        CC v = *at.template row<(DIR < 0)>(i);
        if (!kFx && DIR < 0 && scale != (typename scale_of<CC>::type)1) v = c_scale(v, scale);
        dst[(size_t)l * cols] = c_store(c_cvt<CO>(v));
      }
    }
  }
}

template <int N, int DIR, typename CI, typename CO, typename CC, int VPT, typename TW>
__global__ void col_fft_kernel(const CI *__restrict__ in, CO *__restrict__ out, int ntiles, int tsh,
                               int cols, typename scale_of<CC>::type scale, const TW *__restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  col_fft_tile<N, DIR, CI, CO, CC, VPT, TW>(in, out, blockIdx.x, ntiles, tsh, cols, scale, tw,
                                        reinterpret_cast<CC *>(smem_raw));
}

// FP64 passes and double-float forward passes: the same tile with 4 blocks of 256 threads per SM
// (64 registers a thread).  Against the 3 blocks that 66 to 74 registers allow: FP64 at 512^3
// inverse y 4.57 -> 3.97 ms, forward y 7.81 -> 6.60 ms; double-float forward y 8 % faster.  (The
// double-float inverse passes measured slower so and keep col_fft_kernel.)
template <int N, int DIR, typename CI, typename CO, typename CC, int VPT, typename TW>
__global__ void __launch_bounds__(256, 4) col_fft_kernel_b4(const CI *__restrict__ in, CO *__restrict__ out,
                                                           int ntiles, int tsh, int cols,
                                                           typename scale_of<CC>::type scale,
                                                           const TW *__restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  col_fft_tile<N, DIR, CI, CO, CC, VPT, TW>(in, out, blockIdx.x, ntiles, tsh, cols, scale, tw,
                                        reinterpret_cast<CC *>(smem_raw));
}

// The kernel a pass launches.
template <int N, int DIR, typename CI, typename CO, int VPT, typename TW = typename tw_of<CO>::type>
constexpr auto col_kernel() {
  if constexpr ((std::is_same<CO, cdf>::value && DIR < 0) || std::is_same<TW, TwFx>::value)
    return col_fft_kernel_b4<N, DIR, CI, CO, CO, VPT, TW>;
  else return col_fft_kernel<N, DIR, CI, CO, CO, VPT, TW>;
}

// The same pass as a persistent kernel: a grid of (SMs x resident blocks) takes tiles from the
// work counter ctr[0] until all `total` are done; ctr[1] counts the blocks that have finished, and
// the last one resets both for the next launch (every block has taken its last tile by then; no
// block waits on another).  Each tile's arithmetic is the one col_fft_kernel does.
template <int N, int DIR, typename CI, typename CO, typename CC, int VPT, typename TW>
__global__ void col_fft_persistent_kernel(const CI *__restrict__ in, CO *__restrict__ out, int ntiles, int tsh,
                                          int cols, typename scale_of<CC>::type scale, const TW *__restrict__ tw,
                                          unsigned total, unsigned *ctr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned next;
  for (;;) {
    if (threadIdx.x == 0) next = atomicAdd(ctr, 1u);
    __syncthreads();
    const unsigned w = next;
    if (w >= total) break;
    col_fft_tile<N, DIR, CI, CO, CC, VPT, TW>(in, out, w, ntiles, tsh, cols, scale, tw, reinterpret_cast<CC *>(smem_raw));
    __syncthreads();  // the tile's shared memory and `next` are free again
  }
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(ctr + 1, 1u) == gridDim.x - 1) {
      ctr[0] = 0u;
      ctr[1] = 0u;
    }
  }
}

namespace {

// Columns per block: enough that a tile row is at least 128 bytes and a block at least 128
// threads, but not more than the columns there are; 16-byte values (FP64 and double-float) at most
// 256 threads a block (the width the autotuner picks for them at N >= 512 on GB300).
int pick_tc(int tpp, int cols, size_t elem) {
  int tc = 8;
  while (tc * tpp < 128 && tc < 64) tc *= 2;
  while (tc * tpp > 1024) tc /= 2;
  while (elem >= 16 && tc > 1 && tc * tpp > 256) tc /= 2;
  while (tc > 1 && tc / 2 >= cols) tc /= 2;  // no more than one power of two above `cols`
  return tc;
}

// log2 of the largest power of two <= v (v >= 1)
int floor_log2(int v) {
  int s = 0;
  while ((2 << s) <= v) ++s;
  return s;
}

// Largest thread count a launch of this instantiation may use (its registers bound it below 1024).
template <int N, int DIR, typename CI, typename CO, int VPT, typename TW = typename tw_of<CO>::type>
int col_max_threads() {
  static int cached = 0;
  if (cached == 0) {
    cudaFuncAttributes a;
    cached = cudaFuncGetAttributes(&a, col_kernel<N, DIR, CI, CO, VPT, TW>()) == cudaSuccess ? a.maxThreadsPerBlock
                                                                                               : 256;
  }
  return cached;
}

// Resident blocks per SM of a persistent launch (per instantiation and block shape).
template <auto Fn>
int resident_blocks(int threads, size_t smem) {
  static int cached_threads = -1, cached = 1;
  static size_t cached_smem = 0;
  if (threads != cached_threads || smem != cached_smem) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Fn, threads, smem) != cudaSuccess) {
      cudaGetLastError();
      per_sm = 1;
    }
    cached = per_sm > 0 ? per_sm : 1;
    cached_threads = threads;
    cached_smem = smem;
  }
  return cached;
}

int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, v = 0;
    sms = (cudaGetDevice(&dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0) ? v : 1;
  }
  return sms;
}

template <int N, int DIR, typename CI, typename CO, int VPT, typename TW = typename tw_of<CO>::type>
cudaError_t launch_col_v(const CI *in, CO *out, int nslab, int cols, double scale, const TW *tw,
                         cudaStream_t s, int tile, unsigned *ctr) {
  constexpr int TPP = tpp_for<N, VPT>();
  int tc = tile > 0 ? tile : pick_tc(TPP, cols, sizeof(CO));
  const int max_threads = col_max_threads<N, DIR, CI, CO, VPT, TW>();
  while (tc > 1 && tc * TPP > max_threads) tc /= 2;
  if (tc < 1) tc = 1;
  const int tsh = floor_log2(tc);  // a requested width that is not a power of two is rounded down
  tc = 1 << tsh;
  const int ntiles = (cols + tc - 1) / tc;
  const size_t smem = (size_t)tc * tile_pitch<N, TPP, CO>(tc) * sizeof(CO) + tws_bytes<CO, N>();
  const long long blocks = (long long)nslab * ntiles;
  if (blocks <= 0) return cudaSuccess;
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  if (ctr != nullptr) {
    constexpr auto kfn = col_fft_persistent_kernel<N, DIR, CI, CO, CO, VPT, TW>;
    if (smem > 48 * 1024) {
      cudaError_t e = ensure_smem<kfn>((int)smem);
      if (e != cudaSuccess) return e;
    }
    long long grid = (long long)sm_count() * resident_blocks<kfn>(tc * TPP, smem);
    if (grid > blocks) grid = blocks;
    kfn<<<(unsigned)grid, tc * TPP, smem, s>>>(in, out, ntiles, tsh, cols, (typename scale_of<CO>::type)scale, tw,
                                               (unsigned)blocks, ctr);
    return cudaGetLastError();
  }
  if (smem > 48 * 1024) {
    cudaError_t e = ensure_smem<col_kernel<N, DIR, CI, CO, VPT, TW>()>((int)smem);
    if (e != cudaSuccess) return e;
  }
  return launch_after(col_kernel<N, DIR, CI, CO, VPT, TW>(), dim3((unsigned)blocks), dim3(tc * TPP), smem, s, in, out,
                      ntiles, tsh, cols, (typename scale_of<CO>::type)scale, tw);
}

// Radix of a column pass: `vpt` 8 or 16 (FP32 only); 0 picks the library default (radix 8, and
// radix 16 for FP32 at N >= 512, where it measured faster).
template <int N, int DIR, typename CI, typename CO, typename TW>
cudaError_t launch_col_n(const CI *in, CO *out, int nslab, int cols, double scale, const TW *tw,
                         cudaStream_t s, int tile, int vpt, unsigned *ctr) {
  if constexpr (sizeof(CO) == 8) {
    if (vpt == 16 || (vpt == 0 && N >= 512))
      return launch_col_v<N, DIR, CI, CO, 16, TW>(in, out, nslab, cols, scale, tw, s, tile, ctr);
  }
  return launch_col_v<N, DIR, CI, CO, 8, TW>(in, out, nslab, cols, scale, tw, s, tile, ctr);
}

template <int DIR, typename CI, typename CO, typename TW>
cudaError_t launch_col(const CI *in, CO *out, int n, int nslab, int cols, double scale, const TW *tw,
                       cudaStream_t s, int tile, int vpt, unsigned *ctr = nullptr) {
  switch (n) {
    case 16: return launch_col_n<16, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    case 32: return launch_col_n<32, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    case 64: return launch_col_n<64, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    case 128: return launch_col_n<128, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    case 256: return launch_col_n<256, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    case 512: return launch_col_n<512, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    case 1024: return launch_col_n<1024, DIR>(in, out, nslab, cols, scale, tw, s, tile, vpt, ctr);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

int col_max_tile_df(int n, int dir) {
  auto pick = [&](auto tag_n) -> int {
    constexpr int N = decltype(tag_n)::value;
    const int t = dir > 0 ? col_max_threads<N, +1, cdf, cdf, 8>() : col_max_threads<N, -1, cdf, cdf, 8>();
    int tc = 1;
    while (tc * 2 * tpp_for<N, 8>() <= t && tc < 64) tc *= 2;
    return tc;
  };
  switch (n) {
    case 16: return pick(std::integral_constant<int, 16>());
    case 32: return pick(std::integral_constant<int, 32>());
    case 64: return pick(std::integral_constant<int, 64>());
    case 128: return pick(std::integral_constant<int, 128>());
    case 256: return pick(std::integral_constant<int, 256>());
    case 512: return pick(std::integral_constant<int, 512>());
    case 1024: return pick(std::integral_constant<int, 1024>());
    default: return 1;
  }
}

int col_max_tile(int n, int dir, bool fp64, bool mixed_in, int vpt) {
  const bool r16 = !fp64 && vpt == 16;
  auto pick = [&](auto tag_n) -> int {
    constexpr int N = decltype(tag_n)::value;
    int t;
    if (fp64) t = dir > 0 ? col_max_threads<N, +1, cplx64, cplx64, 8>() : col_max_threads<N, -1, cplx64, cplx64, 8>();
    else if (dir > 0 && mixed_in) t = col_max_threads<N, +1, cplx64, cplx32, 8>();
    else if (dir > 0) t = r16 ? col_max_threads<N, +1, cplx32, cplx32, 16>() : col_max_threads<N, +1, cplx32, cplx32, 8>();
    else t = r16 ? col_max_threads<N, -1, cplx32, cplx32, 16>() : col_max_threads<N, -1, cplx32, cplx32, 8>();
    const int tpp = r16 ? tpp_for<N, 16>() : tpp_for<N, 8>();
    int tc = 1;
    while (tc * 2 * tpp <= t && tc < 64) tc *= 2;
    return tc;
  };
  switch (n) {
    case 16: return pick(std::integral_constant<int, 16>());
    case 32: return pick(std::integral_constant<int, 32>());
    case 64: return pick(std::integral_constant<int, 64>());
    case 128: return pick(std::integral_constant<int, 128>());
    case 256: return pick(std::integral_constant<int, 256>());
    case 512: return pick(std::integral_constant<int, 512>());
    case 1024: return pick(std::integral_constant<int, 1024>());
    default: return 1;
  }
}

cudaError_t launch_col_inverse(const cplx64 *in, cplx64 *out, int n, int nslab, int cols,
                               const TwFx *tw, cudaStream_t s, int tile, int, unsigned *ctr) {
  return launch_col<+1>(in, out, n, nslab, cols, 1.0, tw, s, tile, 8, ctr);
}
cudaError_t launch_col_inverse(const cplx64 *in, cplx32 *out, int n, int nslab, int cols,
                               const cplx32 *tw, cudaStream_t s, int tile) {
  return launch_col<+1>(in, out, n, nslab, cols, 1.0, tw, s, tile, 8);
}
cudaError_t launch_col_inverse(const cplx32 *in, cplx32 *out, int n, int nslab, int cols,
                               const cplx32 *tw, cudaStream_t s, int tile, int vpt, unsigned *ctr) {
  return launch_col<+1>(in, out, n, nslab, cols, 1.0, tw, s, tile, vpt, ctr);
}
cudaError_t launch_col_forward(const cplx64 *in, cplx64 *out, int n, int nslab, int cols,
                               double scale, const TwFx *tw, cudaStream_t s, int tile, int, unsigned *ctr) {
  return launch_col<-1>(in, out, n, nslab, cols, scale, tw, s, tile, 8, ctr);
}
cudaError_t launch_col_forward(const cplx64 *in, cplx64 *out, int n, int nslab, int cols,
                               double scale, const cplx64 *tw, cudaStream_t s) {
  return launch_col<-1>(in, out, n, nslab, cols, scale, tw, s, 0, 8);
}
cudaError_t launch_col_forward(const cplx32 *in, cplx32 *out, int n, int nslab, int cols,
                               double scale, const cplx32 *tw, cudaStream_t s, int tile, int vpt, unsigned *ctr) {
  return launch_col<-1>(in, out, n, nslab, cols, scale, tw, s, tile, vpt, ctr);
}
cudaError_t launch_col_inverse(const cdf *in, cdf *out, int n, int nslab, int cols, const cdf *tw, cudaStream_t s,
                               int tile, int, unsigned *ctr) {
  return launch_col<+1>(in, out, n, nslab, cols, 1.0, tw, s, tile, 8, ctr);
}
cudaError_t launch_col_forward(const cdf *in, cdf *out, int n, int nslab, int cols, double scale, const cdf *tw,
                               cudaStream_t s, int tile, int, unsigned *ctr) {
  return launch_col<-1>(in, out, n, nslab, cols, scale, tw, s, tile, 8, ctr);
}

}  // namespace mhd
