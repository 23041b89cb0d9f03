// bp_spectrum.cu -- angular power spectrum of a flat-sky map (Section 5.3: the FFT of the map,
// binned in logarithmic multipole bins).
//
//   a(l) = dtheta^2 sum_pixels f(theta) e^{-i l.theta},  C(l) = |a(l)|^2 / (nx ny dtheta^2),
//   l = 2 pi (kx / (nx dtheta), ky / (ny dtheta)) for the integer frequencies kx, ky,
// averaged over the modes whose |l| falls in each bin [edges[b], edges[b+1]).
//
//  k_fft_rows     two map rows (FP32 map + lo plane) as the real and imaginary part of one FP64
//                 FFT, separated by its symmetry; only the frequencies kx = 0 .. nx / 2 are kept
//                 (the others are their conjugates), written transposed, two rows = 32 bytes
//  k_fft_bin      the FFT along y of one frequency kx, the power of every mode and the sums per
//                 bin: for a given kx, |l|^2 grows with |ky|, so each bin is a range of |ky|
//                 whose ends are found by binary search (FP64, explicitly rounded |l|^2 against
//                 the squared edges); columns 0 < kx < nx / 2 count twice
//  k_bin_reduce   per bin: the column partials summed in a fixed tree, divided by the mode count
//
// The FFT: 8 points per thread in registers, Stockham passes of radix 8 (the first of radix 2,
// 4 or 8) exchanged through padded shared memory.  The twiddles are fused into the radix-2
// butterflies of a pass, t = u + w v and 2 u - t: 6 FP64 instructions instead of 8.  What bounds
// it: the FP64 pipe (about 2 operations per SM and cycle on this GPU; the real-input transform
// of a 4096^2 map needs 34 instructions per point in each of its two half-size passes, 0.9 ms).
// Measured at 4096^2: 1.30 ms for the whole call (4.59 ms with a complex transform of every row
// and column in radix-2 passes through shared memory, host twiddles on each call).
//
// Everything is FP64 (the FFT costs ~5 n log2 n flops per map, small next to the pastes), so
// the bins agree with an FP64 reference to rounding and each mode's bin is decided exactly
// as the reference decides it.
#include <cmath>
#include <type_traits>
#include <vector>

#include "bp_internal.cuh"

namespace {

constexpr int MAX_BINS = 256;
constexpr int LG_MAX = 13;           // up to 8192 points
constexpr int TWN = 1 << LG_MAX;     // twiddle table: e^{-2 pi i k / TWN}, k < TWN

struct Edges {
  double e2[MAX_BINS + 1];  // squared bin edges (a kernel argument: no upload)
};

// t = u + w v, v = u - w v (as 2 u - t)
__device__ __forceinline__ void bfly(double2& u, double2& v, double2 w) {
  double2 t;
  t.x = fma(w.x, v.x, fma(-w.y, v.y, u.x));
  t.y = fma(w.x, v.y, fma(w.y, v.x, u.y));
  v = make_double2(fma(2.0, u.x, -t.x), fma(2.0, u.y, -t.y));
  u = t;
}
// the same for w = 1 and for w = -i
__device__ __forceinline__ void bfly1(double2& u, double2& v) {
  const double2 t = make_double2(u.x + v.x, u.y + v.y);
  v = make_double2(u.x - v.x, u.y - v.y);
  u = t;
}
__device__ __forceinline__ void bflyi(double2& u, double2& v) {
  const double2 t = make_double2(u.x + v.y, u.y - v.x);
  v = make_double2(u.x - v.y, u.y + v.x);
  u = t;
}
__device__ __forceinline__ double2 times_mi(double2 w) { return make_double2(w.y, -w.x); }

// 8-point DFT of x_m w^m (w1 = w, w2 = w^2, w4 = w^4, w1r = w e^{-i pi / 4}), in place and in
// natural order
__device__ __forceinline__ void dft8(double2 (&v)[8], double2 w1, double2 w2, double2 w4,
                                     double2 w1r) {
#pragma unroll
  for (int m = 0; m < 4; ++m) bfly(v[m], v[m + 4], w4);  // even half (a), odd half (b)
  bfly(v[0], v[2], w2);
  bfly(v[1], v[3], w2);
  const double2 w2i = times_mi(w2);
  bfly(v[4], v[6], w2i);
  bfly(v[5], v[7], w2i);
  bfly(v[0], v[1], w1);             // X0, X4
  bfly(v[2], v[3], times_mi(w1));   // X2, X6
  bfly(v[4], v[5], w1r);            // X1, X5
  bfly(v[6], v[7], times_mi(w1r));  // X3, X7
  const double2 x4 = v[1], x2 = v[2], x6 = v[3], x1 = v[4], x5 = v[5], x3 = v[6];
  v[1] = x1;
  v[2] = x2;
  v[3] = x3;
  v[4] = x4;
  v[5] = x5;
  v[6] = x6;
}
__device__ __forceinline__ void dft8_first(double2 (&v)[8]) {  // w = 1
  // e^{-i pi / 4}, one component rounded up and the other down: rounded alike, its modulus is
  // 7e-17 above 1, which raises every power by as much
  constexpr double SU = 0x1.6a09e667f3bcdp-1, SD = 0x1.6a09e667f3bccp-1;
#pragma unroll
  for (int m = 0; m < 4; ++m) bfly1(v[m], v[m + 4]);
  bfly1(v[0], v[2]);
  bfly1(v[1], v[3]);
  bflyi(v[4], v[6]);
  bflyi(v[5], v[7]);
  bfly1(v[0], v[1]);
  bflyi(v[2], v[3]);
  bfly(v[4], v[5], make_double2(SU, -SD));
  bfly(v[6], v[7], make_double2(-SD, -SU));
  const double2 x4 = v[1], x2 = v[2], x6 = v[3], x1 = v[4], x5 = v[5], x3 = v[6];
  v[1] = x1;
  v[2] = x2;
  v[3] = x3;
  v[4] = x4;
  v[5] = x5;
  v[6] = x6;
}

template <int LG>
struct Fft {
  static constexpr int N = 1 << LG;
  static constexpr int E = LG < 3 ? N : 8;  // points per thread
  static constexpr int T = N / E;           // threads per transform
  // transforms per CTA: at least 64 threads
  static constexpr int F = T >= 64 ? 1 : 64 / T;
  static constexpr int PADN = N + (N >> 3);  // doubles of a padded array
  static __device__ __forceinline__ int at(int p) { return p + (p >> 3); }
  static size_t smem() { return (size_t)F * 2 * PADN * sizeof(double); }

  // Transform of v[m] = x[j + m T] (thread j): v[m] = X[j + m T] on return.  Every thread of the
  // CTA calls it; re, im: this transform's shared arrays.
  static __device__ __forceinline__ void run(double2 (&v)[E], int j, double* re, double* im,
                                             const double2* __restrict__ tw) {
    if constexpr (LG == 1) {
      bfly1(v[0], v[1]);
    } else if constexpr (LG == 2) {
      bfly1(v[0], v[2]);
      bfly1(v[1], v[3]);
      bfly1(v[0], v[1]);
      bflyi(v[2], v[3]);
      const double2 t = v[1];
      v[1] = v[2];
      v[2] = t;
    } else {
      constexpr int R0 = LG % 3 == 0 ? 8 : (LG % 3 == 1 ? 2 : 4);
      // first pass, no twiddles; the results in order of increasing output position
      if constexpr (R0 == 8) {
        dft8_first(v);
      } else if constexpr (R0 == 2) {
#pragma unroll
        for (int s = 0; s < 4; ++s) bfly1(v[s], v[s + 4]);
      } else {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          bfly1(v[s], v[s + 4]);
          bfly1(v[s + 2], v[s + 6]);
          bfly1(v[s], v[s + 2]);
          bflyi(v[s + 4], v[s + 6]);
        }
      }
      if constexpr (LG > 3) {
        // butterfly q = j + s T wrote outputs R0 q .. R0 q + R0 - 1
        auto put = [&](int p, const double2& x) {
          re[at(p)] = x.x;
          im[at(p)] = x.y;
        };
        if constexpr (R0 == 8) {
#pragma unroll
          for (int m = 0; m < 8; ++m) put(8 * j + m, v[m]);
        } else if constexpr (R0 == 2) {
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            put(2 * (j + s * T), v[s]);
            put(2 * (j + s * T) + 1, v[s + 4]);
          }
        } else {
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            const int o = 4 * (j + s * T);
            put(o, v[s]);
            put(o + 1, v[s + 4]);
            put(o + 2, v[s + 2]);
            put(o + 3, v[s + 6]);
          }
        }
        int ns = R0;  // the size of the sub-transforms done so far
#pragma unroll
        for (int pass = 0; pass < (LG - (LG % 3 == 0 ? 3 : LG % 3)) / 3; ++pass) {
          __syncthreads();
#pragma unroll
          for (int m = 0; m < 8; ++m) v[m] = make_double2(re[at(j + m * T)], im[at(j + m * T)]);
          const int e = j & (ns - 1);
          const int i1 = e * (TWN / 8 / ns);
          dft8(v, __ldg(tw + i1), __ldg(tw + 2 * i1), __ldg(tw + 4 * i1), __ldg(tw + i1 + TWN / 8));
          if (ns * 8 < N) {
            __syncthreads();
            const int o = ((j - e) << 3) + e;
#pragma unroll
            for (int m = 0; m < 8; ++m) {
              re[at(o + m * ns)] = v[m].x;
              im[at(o + m * ns)] = v[m].y;
            }
          }
          ns *= 8;
        }
      }
    }
  }
};

// Two rows a, a + 1 of the map as one complex transform; out[kx][row], kx = 0 .. N / 2
template <int LG>
__global__ void __launch_bounds__(Fft<LG>::T* Fft<LG>::F, Fft<LG>::N <= 4096 ? 2 : 1)
    k_fft_rows(const float* __restrict__ map, const float* __restrict__ lo, int ny,
               const double2* __restrict__ tw, double2* __restrict__ out) {
  using P = Fft<LG>;
  constexpr int N = P::N, T = P::T;
  extern __shared__ double s_d[];
  const int j = threadIdx.x % T, f = threadIdx.x / T;
  double *re = s_d + (size_t)f * 2 * P::PADN, *im = re + P::PADN;
  const int pair = blockIdx.x * P::F + f;
  const bool live = 2 * pair < ny;
  const int64_t a = live ? 2 * pair : 0;
  const float *m0 = map + a * N, *m1 = m0 + N;
  const float *l0 = lo ? lo + a * N : nullptr, *l1 = lo ? l0 + N : nullptr;
  double2 v[P::E];
#pragma unroll
  for (int m = 0; m < P::E; ++m) {
    const int i = j + m * T;
    v[m] = make_double2((double)m0[i] + (l0 ? (double)l0[i] : 0.0),
                        (double)m1[i] + (l1 ? (double)l1[i] : 0.0));
  }
  P::run(v, j, re, im, tw);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < P::E; ++m) {
    re[P::at(j + m * T)] = v[m].x;
    im[P::at(j + m * T)] = v[m].y;
  }
  __syncthreads();
  // Z = X + i Y with X, Y the rows' transforms: X[k] = (Z[k] + conj Z[N - k]) / 2,
  // Y[k] = (Z[k] - conj Z[N - k]) / 2 i
  if (!live) return;
  auto put = [&](int k, double2 z) {
    const int kn = (N - k) & (N - 1);
    const double2 c = make_double2(re[P::at(kn)], im[P::at(kn)]);
    double2* o = out + (int64_t)k * ny + a;
    o[0] = make_double2(0.5 * (z.x + c.x), 0.5 * (z.y - c.y));
    o[1] = make_double2(0.5 * (z.y + c.y), 0.5 * (c.x - z.x));
  };
#pragma unroll
  for (int m = 0; m < P::E / 2; ++m) put(j + m * T, v[m]);
  if (j == 0) put(N / 2, v[P::E / 2]);
}

// Column kx of the row transforms (kx = 0 .. nx / 2): FFT along y, then the sums of |a|^2 over
// the bins of the modes (kx, ky), twice for the columns that stand for -kx as well
template <int LG>
__global__ void __launch_bounds__(Fft<LG>::T* Fft<LG>::F, Fft<LG>::N <= 4096 ? 2 : 1)
    k_fft_bin(const double2* __restrict__ in, int nx, const double2* __restrict__ tw,
              double inv_lx, double inv_ly, double c2, Edges E, int nb, double* psum, int* pcnt) {
  using P = Fft<LG>;
  constexpr int N = P::N, T = P::T, F = P::F;
  extern __shared__ double s_d[];
  __shared__ short s_f[F][MAX_BINS + 1];  // first |ky| at or above each edge
  const int j = threadIdx.x % T, f = threadIdx.x / T;
  double *re = s_d + (size_t)f * 2 * P::PADN, *im = re + P::PADN;
  const int ncol = nx / 2 + 1, col0 = blockIdx.x * F;
  const int kx = min(col0 + f, ncol - 1);
  double2 v[P::E];
#pragma unroll
  for (int m = 0; m < P::E; ++m) v[m] = in[(int64_t)kx * N + j + m * T];
  // |l|^2 = c2 ((kx / Lx)^2 + (ky / Ly)^2), every operation rounded as written; it does not
  // decrease with |ky|
  auto kx2 = [&](int ff) {
    const int k = min(col0 + ff, ncol - 1), fx = k < nx / 2 ? k : k - nx;
    const double ux = __dmul_rn((double)fx, inv_lx);
    return __dmul_rn(ux, ux);
  };
  auto l2 = [&](double ux2, int ky) {
    const double uy = __dmul_rn((double)ky, inv_ly);
    return __dmul_rn(c2, __dadd_rn(ux2, __dmul_rn(uy, uy)));
  };
  if constexpr (F > 1) {  // short columns: every |l|^2 once, in the transforms' arrays
    for (int q = threadIdx.x; q < F * (N / 2 + 1); q += blockDim.x) {
      const int ff = q / (N / 2 + 1), k = q % (N / 2 + 1);
      s_d[(size_t)ff * 2 * P::PADN + k] = l2(kx2(ff), k);
    }
    __syncthreads();
  }
  // every (column, b) with b < n, a thread each (no divisions)
  auto each = [&](int n, auto&& fn) {
    for (int ff = 0, b = threadIdx.x;; b += blockDim.x) {
      for (; b >= n; b -= n)
        if (++ff == F) return;
      fn(ff, b);
    }
  };
  each(nb + 1, [&](int ff, int b) {
    const double ux2 = F > 1 ? 0.0 : kx2(ff), e2 = E.e2[b];
    const double* s_l = s_d + (size_t)ff * 2 * P::PADN;
    int lo = 0, hi = N / 2 + 1;  // the answer is in [lo, hi]
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((F > 1 ? s_l[mid] : l2(ux2, mid)) >= e2) hi = mid; else lo = mid + 1;
    }
    s_f[ff][b] = (short)lo;
  });
  if constexpr (F > 1) __syncthreads();
  P::run(v, j, re, im, tw);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < P::E; ++m)
    re[P::at(j + m * T)] = fma(v[m].x, v[m].x, v[m].y * v[m].y);
  __syncthreads();
  // |ky| in the bin's range, ky and -ky (one mode at 0 and at N / 2)
  auto put = [&](int ff, int b, double s) {
    const int k0 = s_f[ff][b], k1 = s_f[ff][b + 1];
    const int k = col0 + ff, w = k > 0 && k < nx / 2 ? 2 : 1;
    const int ends = (k0 == 0 && k1 > 0 ? 1 : 0) + (k0 <= N / 2 && k1 > N / 2 ? 1 : 0);
    psum[(int64_t)k * nb + b] = w * s;
    pcnt[(int64_t)k * nb + b] = w * (2 * (k1 - k0) - ends);
  };
  // Short columns, several per CTA: a thread per (column, bin), Kahan sums.  (A warp each left two
  // warps 960 turns at 64 columns and 30 bins.  A map of 512 x 2: 482 us before, 47 now; 512 x 128
  // with 256 bins: 310 and 53 us.)
  if (F > 1 && (N < 256 || nb > 64)) {  // (256 rows, 30 bins: a warp each is 2 us faster)
    each(nb, [&](int ff, int b) {
      if (col0 + ff >= ncol) return;
      const double* p = s_d + (size_t)ff * 2 * P::PADN;
      double s = 0.0, c = 0.0;
      for (int k = s_f[ff][b]; k < s_f[ff][b + 1]; ++k) {
        const double v = p[P::at(k)] + (k > 0 && k < N / 2 ? p[P::at(N - k)] : 0.0);
        const double y = v - c, t = s + y;
        c = (t - s) - y;
        s = t;
      }
      put(ff, b, s);
    });
    return;
  }
  // a warp per (column, bin)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int ff = 0; ff < F && col0 + ff < ncol; ++ff) {
    const double* p = s_d + (size_t)ff * 2 * P::PADN;
    for (int b = wid; b < nb; b += nw) {
      const int k0 = s_f[ff][b], k1 = s_f[ff][b + 1];
      double s = 0.0;
      for (int k = k0 + lane; k < k1; k += 32) {
        s += p[P::at(k)];
        if (k > 0 && k < N / 2) s += p[P::at(N - k)];
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) put(ff, b, s);
    }
  }
}

// One block per bin: rows summed lane-strided, then a fixed shared-memory tree (the same
// order on every run).
constexpr int BR_THREADS = 256;
__global__ void __launch_bounds__(BR_THREADS)
    k_bin_reduce(const double* __restrict__ psum, const int* __restrict__ pcnt, int nrows, int nb,
                 double norm, double* cl, int64_t* nmodes) {
  __shared__ double s_s[BR_THREADS];
  __shared__ long long s_c[BR_THREADS];
  const int b = blockIdx.x, t = threadIdx.x;
  double s = 0.0;
  long long c = 0;
  for (int r = t; r < nrows; r += BR_THREADS) {
    s += psum[(int64_t)r * nb + b];
    c += pcnt[(int64_t)r * nb + b];
  }
  s_s[t] = s;
  s_c[t] = c;
  __syncthreads();
  for (int o = BR_THREADS / 2; o > 0; o >>= 1) {
    if (t < o) {
      s_s[t] += s_s[t + o];
      s_c[t] += s_c[t + o];
    }
    __syncthreads();
  }
  if (t == 0) {
    // norm times the mean in one rounding: the quotient and what it leaves
    // (1e-16 of it, so that an FP32 reciprocal does for what it leaves)
    const double n = (double)s_c[0], q = s_s[0] / n;
    const double rest = fma(-q, n, s_s[0]) * (double)(1.0f / (float)n);
    cl[b] = s_c[0] > 0 ? fma(norm, q, norm * rest) : 0.0;
    if (nmodes) nmodes[b] = s_c[0];
  }
}

template <int LG>
int launch_rows(bp_ctx* ctx, const float* map, const float* lo, int ny, const double2* tw,
                double2* out) {
  using P = Fft<LG>;
  BP_CUDA(ctx, cudaFuncSetAttribute(k_fft_rows<LG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)P::smem()));
  k_fft_rows<LG><<<(ny / 2 + P::F - 1) / P::F, P::T * P::F, P::smem(), ctx->stream>>>(map, lo, ny,
                                                                                    tw, out);
  BP_LAUNCH_CHECK(ctx, "fft rows");
  return BP_OK;
}

template <int LG>
int launch_bins(bp_ctx* ctx, const double2* in, int nx, const double2* tw, double inv_lx,
                double inv_ly, double c2, const Edges& E, int nb, double* psum, int* pcnt) {
  using P = Fft<LG>;
  BP_CUDA(ctx, cudaFuncSetAttribute(k_fft_bin<LG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)P::smem()));
  k_fft_bin<LG><<<(nx / 2 + 1 + P::F - 1) / P::F, P::T * P::F, P::smem(), ctx->stream>>>(
      in, nx, tw, inv_lx, inv_ly, c2, E, nb, psum, pcnt);
  BP_LAUNCH_CHECK(ctx, "fft bins");
  return BP_OK;
}

// Calls f(std::integral_constant<int, lg>) for the runtime lg in [1, LG_MAX]
template <int LG = 1, typename Fn>
int with_lg(int lg, Fn f) {
  if constexpr (LG < LG_MAX) {
    if (lg != LG) return with_lg<LG + 1>(lg, f);
  }
  return f(std::integral_constant<int, LG>{});
}

// The context's twiddle table, uploaded on its first use (synchronises then)
int twiddles(bp_ctx* ctx, const double2** tw) {
  if (!ctx->fft_tw) {
    std::vector<double2> h(TWN);
    for (int k = 0; k < TWN; ++k)
      h[k] = make_double2(cos(-2.0 * bpc::PI * k / TWN), sin(-2.0 * bpc::PI * k / TWN));
    void* d = nullptr;
    BP_CUDA(ctx, cudaMalloc(&d, TWN * sizeof(double2)));
    cudaError_t e = cudaMemcpyAsync(d, h.data(), TWN * sizeof(double2), cudaMemcpyHostToDevice,
                                    ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) {
      cudaFree(d);
      return bp_cuda_check(ctx, e, "twiddle upload");
    }
    ctx->fft_tw = d;
  }
  *tw = static_cast<const double2*>(ctx->fft_tw);
  return BP_OK;
}

int log2_exact(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return (1 << l) == n ? l : -1;
}

}  // namespace

extern "C" int bp_power_spectrum(bp_ctx* ctx, const float* map, const float* lo, int nx, int ny,
                                 double dtheta, int nb, const double* edges, double* cl,
                                 int64_t* nmodes) {
  if (!ctx) return BP_EINVAL;
  const int lgx = log2_exact(nx), lgy = log2_exact(ny);
  if (lgx < 1 || lgy < 1 || nx > 8192 || ny > 8192)
    return bp_fail(ctx, BP_EINVAL, "bp_power_spectrum: nx, ny must be powers of two in [2, 8192]");
  if (!(dtheta > 0)) return bp_fail(ctx, BP_EINVAL, "bp_power_spectrum: dtheta <= 0");
  if (nb < 1 || nb > MAX_BINS) return bp_fail(ctx, BP_EINVAL, "bp_power_spectrum: nb outside [1, 256]");
  if (!map || !edges || !cl) return bp_fail(ctx, BP_EINVAL, "bp_power_spectrum: null pointer");
  for (int b = 0; b < nb; ++b)
    if (!(edges[b] >= 0.0) || !(edges[b + 1] > edges[b]))
      return bp_fail(ctx, BP_EINVAL, "bp_power_spectrum: edges must increase from >= 0");
  int r;
  const size_t ncell = (size_t)nx * ny;
  const int ncol = nx / 2 + 1;
  const double2* tw;
  if ((r = twiddles(ctx, &tw))) return r;
  double2* A;  // row transforms, transposed
  if ((r = bp_ws(ctx, WS_PART, (size_t)ncol * ny * sizeof(double2), (void**)&A))) return r;
  double* psum;
  if ((r = bp_ws(ctx, WS_MISC3, (size_t)ncol * nb * (8 + 4), (void**)&psum))) return r;
  int* pcnt = reinterpret_cast<int*>(psum + (size_t)ncol * nb);
  Edges E;
  for (int b = 0; b <= MAX_BINS; ++b) E.e2[b] = b <= nb ? edges[b] * edges[b] : 0.0;
  const double inv_lx = 1.0 / (nx * dtheta), inv_ly = 1.0 / (ny * dtheta);
  const double c2 = 4.0 * bpc::PI * bpc::PI;
  const double norm = dtheta * dtheta / (double)ncell;
  if ((r = with_lg(lgx, [&](auto lg) { return launch_rows<lg()>(ctx, map, lo, ny, tw, A); })))
    return r;
  if ((r = with_lg(lgy, [&](auto lg) {
         return launch_bins<lg()>(ctx, A, nx, tw, inv_lx, inv_ly, c2, E, nb, psum, pcnt);
       })))
    return r;
  k_bin_reduce<<<nb, BR_THREADS, 0, ctx->stream>>>(psum, pcnt, ncol, nb, norm, cl, nmodes);
  BP_LAUNCH_CHECK(ctx, "bin reduce");
  return BP_OK;
}
