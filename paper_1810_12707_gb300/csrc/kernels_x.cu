// kernels_x.cu -- passes along the contiguous x axis, where real-space data exists.
//
// Two real rows of the same field are transformed together as one complex pencil
// z = f_row0 + i f_row1.  Inverse (half spectrum -> real rows): with the truncated half spectra
// X0, X1 (kx = 0..K), Z[k] = X0[k] + i X1[k] and Z[N-k] = conj(X0[k]) + i conj(X1[k]) for
// 1 <= k <= K, Z[0] = Re X0[0] + i Re X1[0] (the Hermitian part), zero elsewhere; the real parts
// of the inverse FFT are row 0 and the imaginary parts row 1.  Forward (real rows -> half
// spectra): Z = FFT(row0 + i row1), X0[k] = (Z[k] + conj Z[N-k]) / 2 and
// X1[k] = -i (Z[k] - conj Z[N-k]) / 2, kept for k = 0..K only.
//
// The flux passes store 2 X0 and 2 X1 (the factor 1/2 of the split is left to the assembly, which
// scales the product spectra by 1/(2 N^3): a power of two, so the results are the same bits).
// The flux kernel is the fused pass of the method: the 7 state fields of a block's rows are
// brought to the grid, the 12 products of the RHS are formed pointwise in shared memory (no
// real-space array ever reaches HBM), and their forward transforms leave as truncated half
// spectra.  Rows are indexed r = z*N + y; a block owns PAIRS consecutive row pairs.
#include "cfl_screen.cuh"
#include "fft_device.cuh"
#include "fp64_util.cuh"
#include "launch_util.cuh"
#include "tma_util.cuh"

#include <type_traits>

namespace mhd {

namespace {

constexpr int kMaxThreads = 384;

constexpr int pairs_for(int n) { return (n / 8) >= 16 ? 1 : 16 / (n / 8); }

constexpr int threads_for(int tpp, int pencils, int max_threads = kMaxThreads) {
  // groups of tpp threads (one pencil each), at most max_threads threads, a multiple of 32
  int g = max_threads / tpp;
  if (g < 1) g = 1;
  if (g > pencils) g = pencils;
  int t = g * tpp;
  return (t + 31) / 32 * 32;
}

// Block size of the flux pass: where one row pair fills a block (N >= 128), 4 groups, which take the 7
// and 12 pencils in 2 + 3 rounds with one group idle in one of them (12 groups left 5 idle for the
// fields, 8 left 4 idle for the last products).  128^3 double-float 0.303 -> 0.210 ms against 192
// threads, 256^3 mixed 0.408 -> 0.346 against 128, 512^3 mixed 4.45 -> 4.41 against 192.  Below, where
// few blocks have to hide each other's latency, one group per product (at most 192 threads): 64 threads
// measured 0.059 against 0.049 ms for one 64^3 FP64 instance.
constexpr int flux_max_threads(int n, int tpp) {
  return n < 128 || n > 512 ? kMaxThreads : 4 * tpp;
}
// Values per thread of the flux pass's transforms: FP32 at N <= 256 uses radix 16 (measured
// faster at 64^3 and 256^3); larger FP32 grids and FP64 use radix 8.
template <int N, typename C>
constexpr int flux_vpt() { return sizeof(C) == 8 && N <= 256 ? 16 : 8; }
template <int N, typename C>
constexpr int flux_threads() {
  return threads_for(tpp_for<N, flux_vpt<N, C>()>(), 12 * pairs_for(N),
                     flux_max_threads(N, tpp_for<N, flux_vpt<N, C>()>()));
}
// Blocks per SM the register allocation is sized for: about 170 registers a thread in FP64, 85 in
// FP32 with radix 8 and 128 with radix 16 (its 16 values per thread).
template <int N, typename C>
constexpr int flux_min_blocks() {
  const int budget = sizeof(C) == 8 ? (flux_vpt<N, C>() == 16 ? 512 : 768)
                                    : (N == 512 ? 512 : 384);
  const int b = budget / flux_threads<N, C>();
  return b < 1 ? 1 : b;
}

// Whether a group loads its next row pair before it transforms one: not where the registers that
// holds cost more than the loads' latency (double-float 256^3 1.85 -> 1.81 ms, 512^3 17.6 -> 16.4; FP64
// 512^3 20.5 -> 19.8, but 256^3 2.31 -> 2.33; not compared at 1024^3).
template <int N, typename C>
constexpr bool flux_ahead() { return std::is_same<C, cplx64>::value ? N != 512 : !std::is_same<C, cdf>::value; }

// Run the FFT of `np` pencils (pencil id -> shared-memory pointer `ptr(id)`) with every group of
// N/VPT threads of the block taking one pencil at a time.  Each pencil is touched by its group only,
// so the stages synchronise per group; one block barrier closes the whole transform.
// Every inverse (DIR = +1) transform here starts from a truncated half spectrum, so its pencil is
// zero-padded by the 2/3 rule (see pencil_fft).
// DP, scale2: see pencil_fft.
template <int N, int DIR, int VPT, bool DP = false, typename Ptr, typename TW>
__device__ __forceinline__ void fft_pencils(int np, Ptr ptr, const TW *__restrict__ tw, int scale2 = 0) {
  using C = typename std::remove_pointer<decltype(ptr(0))>::type;
  constexpr int TPP = tpp_for<N, VPT>();
  const int G = blockDim.x / TPP;
  const int g = threadIdx.x / TPP, t = threadIdx.x - g * TPP;
  for (int base = 0; base < np; base += G) {
    const int id = base + g;
    const bool active = g < G && id < np;
    pencil_fft<N, DIR, C, VPT, (DIR > 0), false, DP>(ptr(active ? id : 0), t, active, tw, scale2);
  }
  __syncthreads();  // the callers' next phase reads every pencil
}

}  // namespace

// ------------------------------------------------------------------------------------------
// Fused flux pass
// ------------------------------------------------------------------------------------------
// C: complex type of the data and of all arithmetic (cplx64 or cplx32); the CFL maxima are
// combined in FP64.
// bgrid (nullable): the grid magnetic field is also written out, [inst][3][N^3] in the data's
// precision, for the tracer push.
// One work item w = (instance, block of PAIRS row pairs); `sm` the block's dynamic shared memory,
// `red` 32 doubles of shared scratch for the block maximum.
template <int N, typename C>
__device__ __forceinline__ void flux_x_item(const C *__restrict__ in, C *__restrict__ out,
                                            const PhysDev *__restrict__ phys,
                                            unsigned long long *__restrict__ smax_bits, int K, int blocks_per_inst,
                                            const typename tw_of<C>::type *__restrict__ tw,
                                            typename grid_of<C>::type *__restrict__ bgrid, unsigned w, C *sm, double *red) {
  constexpr int KT = (N - 1) / 3;  // the 2/3-rule cut-off, fixed by N
  using R = typename C::value_type;
  constexpr int P = pencil_pitch<C>(N);
  constexpr int PAIRS = pairs_for(N);
  constexpr size_t NN = (size_t)N * N;
  constexpr int NX = KT + 1;
  const int inst = (int)(w / (unsigned)blocks_per_inst);
  const int bl = (int)(w - (unsigned)inst * (unsigned)blocks_per_inst);
  const size_t row0 = (size_t)bl * PAIRS * 2;
  // the launch uses exactly this many threads, so every loop below has a constant trip count
  constexpr int nthr = flux_threads<N, C>();

  // 1. inverse transforms of the 7 state fields: pencil (p, f) at sm + (p * 12 + f) * P, each by one
  // group, which loads its next row pair while it transforms one
  constexpr int VPT = flux_vpt<N, C>(), TPP = tpp_for<N, VPT>(), G = nthr / TPP;
  const int g = threadIdx.x / TPP, t = threadIdx.x - g * TPP;
  {
    auto src = [&](int id) {
      return in + ((size_t)(inst * 7 + id % 7) * NN + row0 + 2 * (id / 7)) * NX;
    };
    RowPair<N, C, VPT> x;
    if constexpr (flux_ahead<N, C>()) x.load(src(g < 7 * PAIRS ? g : 0), t, g < 7 * PAIRS);
#pragma unroll 1
    for (int base = 0; base < 7 * PAIRS; base += G) {
      const int id = base + g;
      const bool active = id < 7 * PAIRS, more = id + G < 7 * PAIRS;
      C *pen = sm + (active ? (id / 7) * 12 + id % 7 : 0) * P;
      if constexpr (flux_ahead<N, C>()) {
        RowPair<N, C, VPT> next;
        if (base + G < 7 * PAIRS) next.load(src(more ? id + G : 0), t, more);
        rows_inverse<N, C, VPT, false>(pen, t, active, x, tw);
        x = next;
      } else {
        x.load(src(active ? id : 0), t, active);
        rows_inverse<N, C, VPT, false>(pen, t, active, x, tw);
      }
    }
  }
  __syncthreads();

  // 3. products on the grid (real part: row 0, imaginary part: row 1)
  constexpr bool kDF = std::is_same<C, cdf>::value;
  using SM = typename std::conditional<kDF, double, R>::type;  // type of the CFL maximum
  SM smax = 0;
  // FP64 and double-float: exact speeds only where they can raise the published maximum
  float screen = 0.f;
  if constexpr (sizeof(SM) == 8) {
    const double lb = __longlong_as_double((long long)*reinterpret_cast<volatile unsigned long long *>(smax_bits + inst));
    screen = cfl_screen(lb);
  }
  if constexpr (kDF) {
    // double-float products.  The grid values leave the inverse transforms unnormalised; near a
    // zero of a field (a stagnation point) their low part can exceed the high part, and the
    // square of such a pair, which drops lo^2, can come out negative.  So they are renormalised
    // first (then |lo| <= ulp(hi) / 2 and every square is >= 0), as are the velocity components
    // before the exact speed is formed.  The screening estimate takes the high parts alone (FP32
    // products of normalised values, within an ulp); the exact speed is taken in FP64 from the
    // double-float squares, at the points that pass.
    const double csd = phys[inst].cs;
    const dfr cs2 = dfr_from_double(csd * csd);
    for (int q = threadIdx.x; q < PAIRS * N; q += nthr) {
      const int p = q / N, j = q - p * N;
      C *b = sm + p * 12 * P + sm_idx<C>(j);
      dfr v[2][7];
#pragma unroll
      for (int f = 0; f < 7; ++f) {
        const C c = b[f * P];
        v[0][f] = dfr_norm(c.re);
        v[1][f] = dfr_norm(c.im);
      }
      if (bgrid != nullptr) {
        constexpr size_t N3 = NN * N;
        double *g = bgrid + (size_t)inst * 3 * N3 + (row0 + 2 * p) * N + j;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          g[c * N3] = dfr_to_double(v[0][4 + c]);
          g[c * N3 + N] = dfr_to_double(v[1][4 + c]);
        }
      }
      dfr *bd = reinterpret_cast<dfr *>(b);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const dfr rho = v[h][0];
        const dfr mx = v[h][1], my = v[h][2], mz = v[h][3];
        const dfr bx = v[h][4], by = v[h][5], bz = v[h][6];
        const dfr ir = dfr_rcp(rho);
        const dfr ux = mx * ir, uy = my * ir, uz = mz * ir;
        const dfr bxx = bx * bx, byy = by * by, bzz = bz * bz;
        const dfr b2 = bxx + byy + bzz;
        const dfr hb = dfr_scale2(b2, 0.5f);
        bd[2 * 0 * P + h] = mx * ux + hb - bxx;   // T_xx
        bd[2 * 1 * P + h] = my * uy + hb - byy;   // T_yy
        bd[2 * 2 * P + h] = mz * uz + hb - bzz;   // T_zz
        bd[2 * 3 * P + h] = mx * uy - bx * by;    // T_xy
        bd[2 * 4 * P + h] = mx * uz - bx * bz;    // T_xz
        bd[2 * 5 * P + h] = my * uz - by * bz;    // T_yz
        bd[2 * 6 * P + h] = uy * bz - uz * by;    // E_x
        bd[2 * 7 * P + h] = uz * bx - ux * bz;    // E_y
        bd[2 * 8 * P + h] = ux * by - uy * bx;    // E_z
        bd[2 * 9 * P + h] = ux;
        bd[2 * 10 * P + h] = uy;
        bd[2 * 11 * P + h] = uz;
        if (cfl_may_raise(ux.hi, uy.hi, uz.hi, cs2.hi, b2.hi, ir.hi, screen)) {
          const dfr nx = dfr_norm(ux), ny = dfr_norm(uy), nz = dfr_norm(uz);
          const dfr u2 = dfr_norm(nx * nx + ny * ny + nz * nz), c2 = dfr_norm(cs2 + b2 * ir);
          const double s = sqrt(dfr_to_double(u2)) + sqrt(dfr_to_double(c2));
          smax = (s != s || s > smax) ? s : smax;  // keeps a NaN once seen
        }
      }
    }
  } else {
  const R cs2 = (R)(phys[inst].cs * phys[inst].cs);
  const float cs2f = (float)cs2;
  for (int q = threadIdx.x; q < PAIRS * N; q += nthr) {
    const int p = q / N, j = q - p * N;
    C *b = sm + p * 12 * P + sm_idx<C>(j);
    R v[2][7];
#pragma unroll
    for (int f = 0; f < 7; ++f) {
      const C c = b[f * P];
      v[0][f] = c.re;
      v[1][f] = c.im;
    }
    if (bgrid != nullptr) {
      constexpr size_t N3 = NN * N;
      R *g = bgrid + (size_t)inst * 3 * N3 + (row0 + 2 * p) * N + j;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        g[c * N3] = v[0][4 + c];
        g[c * N3 + N] = v[1][4 + c];
      }
    }
    R *bd = reinterpret_cast<R *>(b);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const R rho = v[h][0];
      const R mx = v[h][1], my = v[h][2], mz = v[h][3];
      const R bx = v[h][4], by = v[h][5], bz = v[h][6];
      R ir;
      if constexpr (sizeof(R) == 8) ir = rcp_any(rho);
      else ir = (R)1 / rho;
      const R ux = mx * ir, uy = my * ir, uz = mz * ir;
      const R b2 = bx * bx + by * by + bz * bz;
      const R hb = (R)0.5 * b2;
      // component h of pencil f at this point is bd[2 * f * P + h]
      bd[2 * 0 * P + h] = mx * ux + hb - bx * bx;   // T_xx
      bd[2 * 1 * P + h] = my * uy + hb - by * by;   // T_yy
      bd[2 * 2 * P + h] = mz * uz + hb - bz * bz;   // T_zz
      bd[2 * 3 * P + h] = mx * uy - bx * by;        // T_xy
      bd[2 * 4 * P + h] = mx * uz - bx * bz;        // T_xz
      bd[2 * 5 * P + h] = my * uz - by * bz;        // T_yz
      bd[2 * 6 * P + h] = uy * bz - uz * by;        // E_x
      bd[2 * 7 * P + h] = uz * bx - ux * bz;        // E_y
      bd[2 * 8 * P + h] = ux * by - uy * bx;        // E_z
      bd[2 * 9 * P + h] = ux;
      bd[2 * 10 * P + h] = uy;
      bd[2 * 11 * P + h] = uz;
      if constexpr (sizeof(R) == 8) {
        if (cfl_may_raise(ux, uy, uz, cs2f, b2, ir, screen)) {
          const R s = sqrt(ux * ux + uy * uy + uz * uz) + sqrt(cs2 + b2 * ir);
          smax = (s != s || s > smax) ? s : smax;  // keeps a NaN once seen
        }
      } else {
        const R s = sqrt(ux * ux + uy * uy + uz * uz) + sqrt(cs2 + b2 * ir);
        smax = (s != s || s > smax) ? s : smax;
      }
    }
  }
  }
  __syncthreads();

  // 4. forward transforms of the 12 products, their kept half spectra to memory
#pragma unroll 1
  for (int base = 0; base < 12 * PAIRS; base += G) {
    const int id = base + g;
    const bool active = id < 12 * PAIRS;
    const int f = id % 12, p = id / 12;
    rows_forward<N, C, VPT, false>(sm + (active ? id : 0) * P, t, active,
                                   out + ((size_t)(inst * 12 + f) * NN + row0 + 2 * p) * NX, tw, 0,
                                   [](C v) { return c_store(v); });
  }

  const SM m = block_nan_max(smax, reinterpret_cast<SM *>(red));
  if (threadIdx.x == 0) atomicMax(smax_bits + inst, max_bits((double)m));
}

template <int N, typename C>
__global__ void __launch_bounds__((flux_threads<N, C>()), (flux_min_blocks<N, C>()))
    flux_x_kernel(const C *__restrict__ in, C *__restrict__ out, const PhysDev *__restrict__ phys,
                  unsigned long long *__restrict__ smax_bits, int K, int blocks_per_inst,
                  const typename tw_of<C>::type *__restrict__ tw,
                  typename grid_of<C>::type *__restrict__ bgrid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  after_previous();
  flux_x_item<N, C>(in, out, phys, smax_bits, K, blocks_per_inst, tw, bgrid, blockIdx.x,
                    reinterpret_cast<C *>(smem_raw), red);
}

// The same pass as a persistent kernel (batched small grids): a grid of resident blocks takes
// work items from ctr[0] until all `total` are done; ctr[1] counts finished blocks and the last
// one resets both (no block waits on another).  Each item computes what flux_x_kernel computes.
template <int N, typename C>
__global__ void __launch_bounds__((flux_threads<N, C>()), (flux_min_blocks<N, C>()))
    flux_x_persistent_kernel(const C *__restrict__ in, C *__restrict__ out, const PhysDev *__restrict__ phys,
                             unsigned long long *__restrict__ smax_bits, int K, int blocks_per_inst,
                             const typename tw_of<C>::type *__restrict__ tw, typename grid_of<C>::type *__restrict__ bgrid, unsigned total,
                             unsigned *ctr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  __shared__ unsigned next;
  for (;;) {
    if (threadIdx.x == 0) next = atomicAdd(ctr, 1u);
    __syncthreads();
    const unsigned w = next;
    if (w >= total) break;
    flux_x_item<N, C>(in, out, phys, smax_bits, K, blocks_per_inst, tw, bgrid, w, reinterpret_cast<C *>(smem_raw),
                      red);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(ctr + 1, 1u) == gridDim.x - 1) {
      ctr[0] = 0u;
      ctr[1] = 0u;
    }
  }
}

// ------------------------------------------------------------------------------------------
// Fused flux pass, persistent and pipelined (one row pair per iteration, N >= 128, FP32)
// ------------------------------------------------------------------------------------------
// Each block walks over row pairs (pair = blockIdx.x, + gridDim.x, ...).  The 7 state rows of
// the next pair (one contiguous chunk of 2 * NX complex values per field) are fetched with bulk
// asynchronous copies into the other of two staging buffers while the current pair is
// transformed, so the copy engine keeps HBM busy during the FFT work.  The arithmetic, its order
// and the results are those of flux_x_kernel.  A wait for a copy that does not complete within
// `wait_polls` polls (kWaitPolls unless a caller lowers it; 0 gives up at once) sets *err = 1.
// Before the block returns, thread 0 then waits, with the full limit kWaitPolls each, for BOTH
// copies the block may still have in flight -- the one it gave up on and the prefetch of the
// next row pair -- so that no bulk copy lands in shared memory after the block has released it;
// if one of those waits also runs out, *err = 2.

template <int N, typename C>
__global__ void __launch_bounds__(kMaxThreads, 1)
    flux_x_pipe_kernel(const C *__restrict__ in, C *__restrict__ out, const PhysDev *__restrict__ phys,
                       unsigned long long *__restrict__ smax_bits, int K, long long total_pairs,
                       const typename tw_of<C>::type *__restrict__ tw, int *err, uint32_t wait_polls) {
  constexpr int KT = (N - 1) / 3;  // the 2/3-rule cut-off, fixed by N
  using R = typename C::value_type;
  extern __shared__ __align__(128) unsigned char smem_pipe[];
  __shared__ __align__(8) uint64_t mbar[2];
  constexpr int P = pencil_pitch<C>(N);
  constexpr long long PPI = (long long)N * N / 2;  // row pairs per instance
  constexpr size_t NN = (size_t)N * N;
  constexpr int NX = KT + 1;
  const int chunk = 2 * NX;  // complex values of one field's row pair
  const uint32_t chunk_bytes = (uint32_t)(chunk * sizeof(C));
  C *stage = reinterpret_cast<C *>(smem_pipe);
  C *sm = stage + ((2 * 7 * chunk * sizeof(C) + 127) / 128 * 128) / sizeof(C);
  const int nthr = blockDim.x;

  auto issue = [&](long long pr, int b) {
    const int inst = (int)(pr / PPI);
    const size_t row0 = (size_t)(pr - (long long)inst * PPI) * 2;
    mbar_arrive_expect_tx(&mbar[b], 7 * chunk_bytes);
    for (int f = 0; f < 7; ++f)
      bulk_g2s(stage + (size_t)(b * 7 + f) * chunk, in + ((size_t)(inst * 7 + f) * NN + row0) * NX, chunk_bytes,
               &mbar[b]);
  };

  if (threadIdx.x == 0) {
    mbar_init(&mbar[0], 1);
    mbar_init(&mbar[1], 1);
    fence_mbar_init();
  }
  __syncthreads();
  long long pair = blockIdx.x;
  if (threadIdx.x == 0 && pair < total_pairs) issue(pair, 0);
  int issued_next = 0;
  for (int iter = 0; pair < total_pairs; pair += gridDim.x, ++iter) {
    const int buf = iter & 1;
    const long long nxt = pair + gridDim.x;
    if (threadIdx.x == 0) {
      issued_next = nxt < total_pairs;
      if (issued_next) {
        fence_proxy_async();
        issue(nxt, buf ^ 1);
      }
    }
    const bool ok = mbar_wait(&mbar[buf], (iter >> 1) & 1, wait_polls);
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) {
        atomicExch(err, 1);
        // drain: the copy into stage[buf] that the wait gave up on, and the prefetch into
        // stage[buf ^ 1] issued above; the block's shared memory stays allocated while thread 0
        // is still running
        bool drained = mbar_wait(&mbar[buf], (iter >> 1) & 1, kWaitPolls);
        if (issued_next) drained = mbar_wait(&mbar[buf ^ 1], ((iter + 1) >> 1) & 1, kWaitPolls) && drained;
        if (!drained) atomicExch(err, 2);
      }
      return;
    }
    const int inst = (int)(pair / PPI);
    const size_t row0 = (size_t)(pair - (long long)inst * PPI) * 2;
    const int tx = launder(threadIdx.x);

    // 1. pack the 7 fields of this row pair from the staging buffer
    const C *st = stage + (size_t)buf * 7 * chunk;
    for (int q = tx; q < 7 * NX; q += nthr) {
      const int k = q % NX, f = q / NX;
      const C x0 = st[f * chunk + k], x1 = st[f * chunk + NX + k];
      C *pen = sm + f * P;
      if (k == 0) {
        pen[0] = C{x0.re, x1.re};
      } else {
        pen[sm_idx<C>(k)] = C{x0.re - x1.im, x0.im + x1.re};
        pen[sm_idx<C>(N - k)] = C{x0.re + x1.im, x1.re - x0.im};
      }
    }
    constexpr int NZ = pencil_zero_count<N>();
    for (unsigned q = tx; q < (unsigned)(7 * NZ); q += nthr) {
      const unsigned z = q % NZ, f = q / NZ;
      sm[f * P + sm_at<C>(pencil_zero<N>(z))] = C{0, 0};
    }
    __syncthreads();

    // 2. inverse transforms of the 7 fields
    fft_pencils<N, +1, (flux_vpt<N, C>())>(7, [&](int id) { return sm + id * P; }, tw);

    // 3. products on the grid
    const R cs2 = (R)(phys[inst].cs * phys[inst].cs);
    R smax = 0;
    for (int j = tx; j < N; j += nthr) {
      C *b = sm + sm_idx<C>(j);
      R v[2][7];
#pragma unroll
      for (int f = 0; f < 7; ++f) {
        const C c = b[f * P];
        v[0][f] = c.re;
        v[1][f] = c.im;
      }
      R *bd = reinterpret_cast<R *>(b);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const R rho = v[h][0];
        const R mx = v[h][1], my = v[h][2], mz = v[h][3];
        const R bx = v[h][4], by = v[h][5], bz = v[h][6];
        const R ir = (R)1 / rho;
        const R ux = mx * ir, uy = my * ir, uz = mz * ir;
        const R b2 = bx * bx + by * by + bz * bz;
        const R hb = (R)0.5 * b2;
        bd[2 * 0 * P + h] = mx * ux + hb - bx * bx;
        bd[2 * 1 * P + h] = my * uy + hb - by * by;
        bd[2 * 2 * P + h] = mz * uz + hb - bz * bz;
        bd[2 * 3 * P + h] = mx * uy - bx * by;
        bd[2 * 4 * P + h] = mx * uz - bx * bz;
        bd[2 * 5 * P + h] = my * uz - by * bz;
        bd[2 * 6 * P + h] = uy * bz - uz * by;
        bd[2 * 7 * P + h] = uz * bx - ux * bz;
        bd[2 * 8 * P + h] = ux * by - uy * bx;
        bd[2 * 9 * P + h] = ux;
        bd[2 * 10 * P + h] = uy;
        bd[2 * 11 * P + h] = uz;
        const R s = sqrt(ux * ux + uy * uy + uz * uz) + sqrt(cs2 + b2 * ir);
        smax = (s != s || s > smax) ? s : smax;
      }
    }
    __syncthreads();

    // 4. forward transforms of the 12 products
    fft_pencils<N, -1, (flux_vpt<N, C>())>(12, [&](int id) { return sm + id * P; }, tw);

    // 5. unpack and store
      for (int q = tx; q < 12 * NX; q += nthr) {
      const int k = q % NX, f = q / NX;
      const C *pen = sm + f * P;
      const C z = pen[sm_idx<C>(k)], zc = pen[sm_idx<C>((N - k) & (N - 1))];
      C *dst = out + ((size_t)(inst * 12 + f) * NN + row0) * NX;
      dst[k] = C{z.re + zc.re, z.im - zc.im};
      dst[NX + k] = C{z.im + zc.im, zc.re - z.re};
    }

    // CFL maximum of this pair: warp maximum, one atomic per warp
    R m = smax;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = nan_max(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(smax_bits + inst, max_bits((double)m));
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// Forward x transform of an initial state (m = rho u formed first)
// ------------------------------------------------------------------------------------------
// The real fields are FP64; C = cplx64 transforms in FP64, C = cdf splits each value (and the FP64
// product rho u) into double-float pairs and transforms in double-float.
__device__ __forceinline__ void x_load(double v, double &r) { r = v; }
__device__ __forceinline__ void x_load(double v, dfr &r) { r = dfr_from_double(v); }
__device__ __forceinline__ double x_store(double v) { return v; }
__device__ __forceinline__ double x_store(dfr v) { return dfr_to_double(v); }

// One group of N/8 threads per pencil (field f = id mod 7, row pair id / 7), kXThreads threads a block:
// every thread's values of the two rows are the inputs of its first stage, and the last stage's
// results go out from registers, so the fields' groups share nothing but the density rows (from L1)
// and no block barrier.  One block of all 7 fields, the earlier form, left 5 of its 6 groups idle for
// the seventh field at N = 512 and packed through shared memory: FP64 256^3 set 1.68 -> 0.50 ms, get
// 1.75 -> 0.51 ms; IEEE set 2.92 -> 2.55 ms.
constexpr int kXThreads = 256;
template <int N>
constexpr int x_groups() { return kXThreads / tpp_for<N, 8>(); }

// The 7 real fields as three arrays (rho; 3 of one vector; 3 of the other) with field stride `stride`.
template <typename T>
struct Fields7 {
  T *a, *b, *c;
  size_t stride;
  __device__ __forceinline__ T *field(int f) const {
    return f == 0 ? a : f < 4 ? b + (f - 1) * stride : c + (f - 4) * stride;
  }
};

// Rows from `row_begin` on (even); the real arrays hold rows from `row_begin` (field stride N^3 for
// whole fields, less for a slab of z-planes).
template <int N, typename C, typename TW>
__global__ void __launch_bounds__(kXThreads) set_x_kernel(Fields7<const double> in, C *__restrict__ out,
                                                          const TW *__restrict__ tw, size_t row_begin, int pencils) {
  using R = typename C::value_type;
  constexpr int NX = (N - 1) / 3 + 1, TPP = tpp_for<N, 8>(), P = pencil_pitch<C>(N);
  constexpr size_t NN = (size_t)N * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  const int g = threadIdx.x / TPP, t = threadIdx.x - g * TPP;
  const int id = blockIdx.x * x_groups<N>() + g;
  const bool active = id < pencils;
  const int f = active ? id % 7 : 0;
  const size_t pair = active ? id / 7 : 0;

  C x[8];
  const double *src = in.field(f) + 2 * pair * N + t;
  double v0[8], v1[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    v0[r] = active ? src[r * TPP] : 0.0;
    v1[r] = active ? src[N + r * TPP] : 0.0;
  }
  if (f >= 1 && f < 4) {  // m = rho u
    const double *rho = in.a + 2 * pair * N + t;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v0[r] = rho[r * TPP] * v0[r];
      v1[r] = rho[N + r * TPP] * v1[r];
    }
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    R a, b;
    x_load(v0[r], a);
    x_load(v1[r], b);
    x[r] = C{a, b};
  }
  // the split's factor 1/2: in fixed point a step of the results' exponents
  constexpr bool kFx = std::is_same<TW, TwFx>::value;
  rows_forward_from<N, C, kFx>(x, reinterpret_cast<C *>(smem_raw) + g * P, t, active,
                               out + (f * NN + row_begin + 2 * pair) * NX, tw, -1,
                               [](C v) { return c_store(c_scale(v, (typename scale_of<C>::type)0.5)); });
}

// ------------------------------------------------------------------------------------------
// Inverse x transform to real rows
// ------------------------------------------------------------------------------------------
// Rows from `row_begin` on; `out` holds rows from `row_begin`; nf fields.  Pencils as in set_x_kernel.
template <int N, typename C>
__global__ void __launch_bounds__(kXThreads) get_x_kernel(const C *__restrict__ in, Fields7<double> out, int nf,
                                                          const typename tw_of<C>::type *__restrict__ tw,
                                                          size_t row_begin, int pencils) {
  constexpr int NX = (N - 1) / 3 + 1, TPP = tpp_for<N, 8>(), P = pencil_pitch<C>(N);
  constexpr size_t NN = (size_t)N * N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  const int g = threadIdx.x / TPP, t = threadIdx.x - g * TPP;
  const int id = blockIdx.x * x_groups<N>() + g;
  const bool active = id < pencils;
  const int f = active ? id % nf : 0;
  const size_t pair = active ? id / nf : 0;
  RowPair<N, C, 8> x;
  x.load(in + (f * NN + row_begin + 2 * pair) * NX, t, active);
  reg_of<C, typename tw_of<C>::type> z[8];
  FxScale sc{};
  rows_inverse<N, C, 8, true, true>(reinterpret_cast<C *>(smem_raw) + g * P, t, active, x, tw, z, &sc);
  if (active) {
    double *dst = out.field(f) + 2 * pair * N + t;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      double v0, v1;
      if constexpr (std::is_same<C, cplx64>::value) {
        const uint32_t be = sc.ek + (uint32_t)sc.shift + 1u;
        v0 = fx_to_double_dp(z[r].re, be);
        v1 = fx_to_double_dp(z[r].im, be);
      } else {
        v0 = x_store(z[r].re);
        v1 = x_store(z[r].im);
      }
      dst[r * TPP] = v0;
      dst[N + r * TPP] = v1;
    }
    if constexpr (std::is_same<C, cplx64>::value) {
      if (sc.bad) {
        const double f = fx_bad_factor(sc.ek);
#pragma unroll 1
        for (int r = 0; r < 16; ++r) dst[r * TPP] *= f;  // N = 8 TPP: both rows
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// Inverse x transform of the state with grid diagnostics
// ------------------------------------------------------------------------------------------
// A block owns PAIRS row pairs and one group per pencil (7 PAIRS of them) where 448 threads hold them.
// The sums' constant factors are applied once per thread.  Bound by the FP64 pipe: per point one
// reciprocal, three corrected quotients, three roots, a logarithm and about 20 more instructions
// (fp64_util.cuh; 256^3 7.15 -> 3.96 ms against divisions, library roots and 7 pencils on 6 groups).
constexpr int kDiagThreads = 448;
template <int N>
__global__ void __launch_bounds__(kDiagThreads) diag_x_kernel(const cplx64 *__restrict__ in,
                                                              const PhysDev *__restrict__ phys,
                                                              double *__restrict__ part,
                                                              const TwFx *__restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx64 *sm = reinterpret_cast<cplx64 *>(smem_raw);
  __shared__ double red[32];
  constexpr int P = pencil_pitch<cplx64>(N), TPP = tpp_for<N, 8>();
  constexpr int PAIRS = pairs_for(N);
  constexpr size_t NN = (size_t)N * N;
  constexpr int NX = (N - 1) / 3 + 1;
  const size_t row0 = (size_t)blockIdx.x * PAIRS * 2;
  const int nthr = blockDim.x;

  const int g = threadIdx.x / TPP, t = threadIdx.x - g * TPP, G = nthr / TPP;
  for (int base = 0; base < 7 * PAIRS; base += G) {
    const int id = base + g;
    const bool active = g < G && id < 7 * PAIRS;
    const int f = active ? id % 7 : 0, p = active ? id / 7 : 0;
    RowPair<N, cplx64, 8> x;
    x.load(in + ((size_t)f * NN + row0 + 2 * p) * NX, t, active);
    rows_inverse<N, cplx64, 8, false>(sm + (active ? id : 0) * P, t, active, x, tw);
  }
  __syncthreads();

  const double cs2 = phys[0].cs * phys[0].cs;
  double acc[6] = {0, 0, 0, 0, 0, 0};
  double smax = 0.0;
  for (int q = threadIdx.x; q < PAIRS * N; q += nthr) {
    const int p = q / N, j = q - p * N;
    const cplx64 *b = sm + p * 7 * P + sm_idx<cplx64>(j);
    double v[2][7];
#pragma unroll
    for (int f = 0; f < 7; ++f) {
      const cplx64 c = b[f * P];
      v[0][f] = c.re;
      v[1][f] = c.im;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double rho = v[h][0];
      const double bx = v[h][4], by = v[h][5], bz = v[h][6];
      const double b2 = bx * bx + by * by + bz * bz;
      double ux, uy, uz, c2;
      if (rcp3_covers(rho)) {
        const double ir = rcp3(rho);
        ux = quotient(v[h][1], rho, ir);
        uy = quotient(v[h][2], rho, ir);
        uz = quotient(v[h][3], rho, ir);
        c2 = fma(b2, ir, cs2);
      } else {
        ux = v[h][1] / rho;
        uy = v[h][2] / rho;
        uz = v[h][3] / rho;
        c2 = cs2 + b2 / rho;
      }
      const double u2 = ux * ux + uy * uy + uz * uz;
      const double su = sqrt3(u2);
      acc[0] = fma(rho, u2, acc[0]);
      acc[1] += b2;
      acc[2] = fma(rho, log(rho), acc[2]);
      acc[3] = fma(ux, bx, fma(uy, by, fma(uz, bz, acc[3])));
      acc[4] += su;
      acc[5] += sqrt3(b2);
      smax = nan_max(smax, su + sqrt3(c2));
    }
  }
  acc[0] *= 0.5;
  acc[1] *= 0.5;
  acc[2] *= cs2;
  for (int i = 0; i < 6; ++i) {
    const double s = block_sum(acc[i], red);
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * 8 + i] = s;
  }
  const double m = block_nan_max(smax, red);
  if (threadIdx.x == 0) {
    part[(size_t)blockIdx.x * 8 + 6] = m;
    part[(size_t)blockIdx.x * 8 + 7] = 0.0;
  }
}

// ------------------------------------------------------------------------------------------
// Launchers
// ------------------------------------------------------------------------------------------
namespace {

template <int N, typename C>
cudaError_t flux_n(const C *in, C *out, const PhysDev *phys, unsigned long long *part, const Dims &d,
                   const typename tw_of<C>::type *tw, cudaStream_t s, int *err, typename grid_of<C>::type *bgrid,
                   uint32_t wait_polls, unsigned *ctr) {
  constexpr int PAIRS = pairs_for(N);
  if constexpr (PAIRS == 1 && sizeof(C) == 8) {
    if (bgrid != nullptr) err = nullptr;  // the pipelined variant does not write the grid field
    const int chunk = 2 * (d.k + 1);
    const size_t stage_bytes = (2 * 7 * chunk * sizeof(C) + 127) / 128 * 128;
    const size_t smem = stage_bytes + (size_t)12 * pencil_pitch<C>(N) * sizeof(C);
    if (err != nullptr && smem <= 200 * 1024) {
      cudaError_t e = ensure_smem<flux_x_pipe_kernel<N, C>>((int)smem);
      if (e != cudaSuccess) return e;
      const int threads = threads_for(tpp_for<N, flux_vpt<N, C>()>(), 12);
      int per_sm = 0, dev = 0, sms = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, flux_x_pipe_kernel<N, C>, threads, smem);
      if (e != cudaSuccess) return e;
      if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
      if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
      const long long total = (long long)d.batch * N * N / 2;
      long long blocks = (long long)sms * (per_sm > 0 ? per_sm : 1);
      if (blocks > total) blocks = total;
      flux_x_pipe_kernel<N, C><<<(unsigned)blocks, threads, smem, s>>>(in, out, phys, part, d.k, total, tw, err,
                                                                          wait_polls);
      return cudaGetLastError();
    }
  }
  const int bpi = N * N / (2 * PAIRS);
  const int threads = flux_threads<N, C>();
  const size_t smem = (size_t)12 * PAIRS * pencil_pitch<C>(N) * sizeof(C);
  if (smem > 48 * 1024) {
    cudaError_t e = ensure_smem<flux_x_kernel<N, C>>((int)smem);
    if (e != cudaSuccess) return e;
  }
  const long long blocks = (long long)bpi * d.batch;
  if (ctr != nullptr) {
    constexpr auto kfn = flux_x_persistent_kernel<N, C>;
    if (smem > 48 * 1024) {
      cudaError_t e = ensure_smem<kfn>((int)smem);
      if (e != cudaSuccess) return e;
    }
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, threads, smem);
    if (e != cudaSuccess) return e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    long long grid = (long long)sms * (per_sm > 0 ? per_sm : 1);
    if (grid > blocks) grid = blocks;
    kfn<<<(unsigned)grid, threads, smem, s>>>(in, out, phys, part, d.k, bpi, tw, bgrid, (unsigned)blocks, ctr);
    return cudaGetLastError();
  }
  return launch_after(flux_x_kernel<N, C>, dim3((unsigned)blocks), dim3(threads), smem, s, in, out, phys, part, d.k,
                      bpi, tw, bgrid);
}

template <int N, typename C, typename TW>
cudaError_t set_n(const double *rho, const double *u, const double *b, C *out, const Dims &d,
                  const TW *tw, cudaStream_t s, size_t row_begin, size_t nrows, size_t fstride) {
  if (row_begin % 2 || nrows % 2) return cudaErrorInvalidValue;
  const long long pencils = 7LL * (long long)(nrows / 2);
  if (pencils == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((pencils + x_groups<N>() - 1) / x_groups<N>());
  const size_t smem = (size_t)x_groups<N>() * pencil_pitch<C>(N) * sizeof(C);  // below 48 KB for every N
  return launch_after(set_x_kernel<N, C, TW>, dim3(blocks), dim3(kXThreads), smem, s,
                      Fields7<const double>{rho, u, b, fstride}, out, tw, row_begin, (int)pencils);
}

template <int N, typename C>
cudaError_t get_n(const C *in, double *a, double *b, double *c, int nf, const Dims &d,
                  const typename tw_of<C>::type *tw, cudaStream_t s, size_t row_begin, size_t nrows, size_t fstride) {
  if (row_begin % 2 || nrows % 2 || nf < 1 || nf > 7) return cudaErrorInvalidValue;
  const long long pencils = (long long)nf * (long long)(nrows / 2);
  if (pencils == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((pencils + x_groups<N>() - 1) / x_groups<N>());
  const size_t smem = (size_t)x_groups<N>() * pencil_pitch<C>(N) * sizeof(C);
  return launch_after(get_x_kernel<N, C>, dim3(blocks), dim3(kXThreads), smem, s, in, Fields7<double>{a, b, c, fstride},
                      nf, tw, row_begin, (int)pencils);
}

template <int N>
cudaError_t diag_n(const cplx64 *in, const PhysDev *phys, double *part, const Dims &d,
                   const TwFx *tw, cudaStream_t s) {
  constexpr int PAIRS = pairs_for(N);
  const int blocks = N * N / (2 * PAIRS);
  const int threads = threads_for(tpp_for<N, 8>(), 7 * PAIRS, kDiagThreads);
  const size_t smem = (size_t)7 * PAIRS * pencil_pitch<cplx64>(N) * sizeof(cplx64);
  if (smem > 48 * 1024) {
    cudaError_t e = ensure_smem<diag_x_kernel<N>>((int)smem);
    if (e != cudaSuccess) return e;
  }
  diag_x_kernel<N><<<blocks, threads, smem, s>>>(in, phys, part, tw);
  return cudaGetLastError();
}

}  // namespace

#define MHD_DISPATCH_N(n, call)     \
  switch (n) {                      \
    case 16: { constexpr int N = 16; return call; }     \
    case 32: { constexpr int N = 32; return call; }     \
    case 64: { constexpr int N = 64; return call; }     \
    case 128: { constexpr int N = 128; return call; }   \
    case 256: { constexpr int N = 256; return call; }   \
    case 512: { constexpr int N = 512; return call; }   \
    case 1024: { constexpr int N = 1024; return call; } \
    default: return cudaErrorInvalidValue;              \
  }

int flux_x_blocks_per_instance(int n) { return n * n / (2 * pairs_for(n)); }
int diag_x_blocks(int n) { return n * n / (2 * pairs_for(n)); }

cudaError_t launch_flux_x(const cplx64 *in, cplx64 *out, const PhysDev *phys, unsigned long long *smax_bits,
                          const Dims &d, const TwFx *tw, cudaStream_t s, int *err, double *bgrid,
                          uint32_t wait_polls, unsigned *ctr) {
  MHD_DISPATCH_N(d.n, (flux_n<N>(in, out, phys, smax_bits, d, tw, s, err, bgrid, wait_polls, ctr)));
}

cudaError_t launch_flux_x(const cplx32 *in, cplx32 *out, const PhysDev *phys, unsigned long long *smax_bits,
                          const Dims &d, const cplx32 *tw, cudaStream_t s, int *err, float *bgrid,
                          uint32_t wait_polls, unsigned *ctr) {
  MHD_DISPATCH_N(d.n, (flux_n<N>(in, out, phys, smax_bits, d, tw, s, err, bgrid, wait_polls, ctr)));
}

cudaError_t launch_flux_x(const cdf *in, cdf *out, const PhysDev *phys, unsigned long long *smax_bits, const Dims &d,
                          const cdf *tw, cudaStream_t s, int *, double *bgrid, uint32_t, unsigned *ctr) {
  MHD_DISPATCH_N(d.n, (flux_n<N>(in, out, phys, smax_bits, d, tw, s, nullptr, bgrid, kWaitPolls, ctr)));
}

cudaError_t launch_set_x(const double *rho, const double *u, const double *b, cplx64 *out,
                         const Dims &d, const TwFx *tw, cudaStream_t s) {
  const size_t nn = (size_t)d.n * d.n;
  MHD_DISPATCH_N(d.n, (set_n<N>(rho, u, b, out, d, tw, s, 0, nn, nn * d.n)));
}

cudaError_t launch_set_x_rows(const double *rho, const double *u, const double *b, cplx64 *out, const Dims &d,
                              const TwFx *tw, cudaStream_t s, size_t row_begin, size_t nrows, size_t fstride) {
  MHD_DISPATCH_N(d.n, (set_n<N>(rho, u, b, out, d, tw, s, row_begin, nrows, fstride)));
}

cudaError_t launch_set_x(const double *rho, const double *u, const double *b, cplx64 *out,
                         const Dims &d, const cplx64 *tw, cudaStream_t s) {
  const size_t nn = (size_t)d.n * d.n;
  MHD_DISPATCH_N(d.n, (set_n<N>(rho, u, b, out, d, tw, s, 0, nn, nn * d.n)));
}

cudaError_t launch_set_x_rows(const double *rho, const double *u, const double *b, cplx64 *out, const Dims &d,
                              const cplx64 *tw, cudaStream_t s, size_t row_begin, size_t nrows, size_t fstride) {
  MHD_DISPATCH_N(d.n, (set_n<N>(rho, u, b, out, d, tw, s, row_begin, nrows, fstride)));
}

cudaError_t launch_get_x(const cplx64 *in, double *out, int nfields, const Dims &d,
                         const TwFx *tw, cudaStream_t s) {
  const size_t nn = (size_t)d.n * d.n;
  const size_t n3 = nn * d.n;
  MHD_DISPATCH_N(d.n, (get_n<N>(in, out, out + n3, out + 4 * n3, nfields, d, tw, s, 0, nn, n3)));
}

cudaError_t launch_get_x(const cplx64 *in, double *a, double *b, double *c, const Dims &d, const TwFx *tw,
                         cudaStream_t s) {
  const size_t nn = (size_t)d.n * d.n;
  MHD_DISPATCH_N(d.n, (get_n<N>(in, a, b, c, 7, d, tw, s, 0, nn, nn * d.n)));
}

cudaError_t launch_get_x(const cdf *in, double *a, double *b, double *c, const Dims &d, const cdf *tw,
                         cudaStream_t s) {
  const size_t nn = (size_t)d.n * d.n;
  MHD_DISPATCH_N(d.n, (get_n<N>(in, a, b, c, 7, d, tw, s, 0, nn, nn * d.n)));
}

cudaError_t launch_get_x_rows(const cplx64 *in, double *out, int nfields, const Dims &d, const TwFx *tw,
                              cudaStream_t s, size_t row_begin, size_t nrows, size_t fstride) {
  MHD_DISPATCH_N(d.n, (get_n<N>(in, out, out + fstride, out + 4 * fstride, nfields, d, tw, s, row_begin, nrows, fstride)));
}

cudaError_t launch_set_x_rows(const double *rho, const double *u, const double *b, cdf *out, const Dims &d,
                              const cdf *tw, cudaStream_t s, size_t row_begin, size_t nrows, size_t fstride) {
  MHD_DISPATCH_N(d.n, (set_n<N>(rho, u, b, out, d, tw, s, row_begin, nrows, fstride)));
}

cudaError_t launch_get_x_rows(const cdf *in, double *out, int nfields, const Dims &d, const cdf *tw, cudaStream_t s,
                              size_t row_begin, size_t nrows, size_t fstride) {
  MHD_DISPATCH_N(d.n, (get_n<N>(in, out, out + fstride, out + 4 * fstride, nfields, d, tw, s, row_begin, nrows, fstride)));
}

cudaError_t launch_diag_x(const cplx64 *in, const PhysDev *phys, double *part, const Dims &d,
                          const TwFx *tw, cudaStream_t s) {
  MHD_DISPATCH_N(d.n, (diag_n<N>(in, phys, part, d, tw, s)));
}

}  // namespace mhd
