// bp_hsml.cu -- SPH smoothing lengths (Section 3.4: the cubic kernel Eq. SPH_kernel and the
// effective neighbour number N_ngb).  h_i solves
//   N_eff(h) = (4 pi / 3) h^3 sum_j W(|r_i - r_j|, h) = (32/3) sum_j w(|r_i - r_j| / h) = N_ngb,
// the sum over every particle, i itself included; N_eff grows monotonically with h.
//
// The particles are put in Hilbert-curve order of their positions quantised to 21 bits per
// axis over the bounding cube.  Every 32 consecutive particles are a leaf with its bounding box,
// every 32 leaves (then every 32 nodes) a node with the box of theirs.  Light-cone particles span
// four decades of density (halo cores to voids): the boxes follow it, which cells of one size
// per search cannot (a halo's core in a corner of a cell is tested whole).  The Hilbert curve has
// no jumps, so its runs of 32 are compact: a particle's sphere meets 16 leaves, 25 with the
// Z-curve's.
//
//  k_bbox          bounding box of the positions (order-independent min / max)
//  k_curve         63-bit curve key of every particle, as a low and a high 32-bit word
//  radix sorts     stable sort by the low word, then by the high word (bp_sort.cu):
//                  k_curve_mid carries the high words into the first order,
//                  k_curve_final the particle ids and float4 positions into the last
//  k_tree          boxes of one level from the positions, or from the level below
//  k_hs_start      first search radius of every particle, a thread each
//  k_hsml_group    one warp per 8 particles: one search of the tree for all of them; four
//                  particles' lists at a time solve N_eff(h) = N_ngb
//  k_hsml          one warp per particle: the few that the groups leave, and large N_ngb; the
//                  particles within R compacted into shared memory by ballot; R grows until
//                  N_eff(R) >= N_ngb, then N_eff(h) = N_ngb is solved in (0, R] by Newton
//                  inside a bisection bracket.
// Every list is in tree order and every sum lane-strided plus a fixed shuffle tree:
// deterministic.
//
// What bounds it: instruction issue (60 % of the slots in k_hsml_group, the rest is waiting for
// leaves from L2).  4e6 light-cone particles, N_ngb = 64: 15.0 ms in all (30.4 ms with a warp per
// particle that tests the Z-curve cells around it, found by binary searches: 6100 instructions
// per particle, 1400 particles tested).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "bp_internal.cuh"

namespace {

constexpr int HS_CAP_MAX = 2048;      // twice the largest N_ngb
// Candidates of a warp's particle in k_hsml.  One that overflows streams its sums over the tree,
// a millisecond or two by itself.  Among few particles that is the call's tail (5e4: k_hsml 1.5 ms
// at 2048, 0.2 ms at 4096); among many, warps in flight count more (4e6: 5.5 ms and 8.4 ms).
constexpr int HS_CAP_FEW = 4096;
constexpr int64_t HS_MANY = 1 << 20;
constexpr int HS_CAP = 2048;          // candidate distances per warp (shared memory)
constexpr int HS_MAX_ROUNDS = 48;     // radius updates per particle
constexpr int HS_QBITS = 21;          // quantisation bits per axis (63-bit keys)
constexpr int HS_SCAN_CAPS = 16;      // particles worth one search, in buffer capacities
constexpr float HS_FAR = 1.5f;        // a guess is looked at above this many leaf diagonals
// The groups.  A search shared by 8 or 16 particles costs the same (13.6 ms at 4e6 particles,
// 32: 15 ms; at 5e4, 8 leaves more warps: 0.22 and 0.33 ms).  Lists of 2 N_ngb to 3 N_ngb: 13.6
// ms, 4 N_ngb 15.5 ms (fewer warps per SM).  Starts of 0.3 N_ngb to 0.5 N_ngb particles: 13.6 to
// 14.3 ms (the median distance in a box overestimates a sphere's: these hold 0.8 to 1.4 N_ngb).
constexpr int HG_NGB_MAX = 128;       // largest N_ngb (above, few warps fit)
constexpr int HG_SIZE = 8;            // particles per group (a power of two, <= 32)
constexpr int HG_ROUNDS = 6;          // radius updates per group
constexpr int HG_LEAVES = 96;         // leaves of a group
constexpr float HG_LIST = 2.5f;       // candidates of a particle, in N_ngb
constexpr float HG_START = 0.35f;     // first radius: HG_START N_ngb particles
constexpr float HS_KNORM = 32.0f / 3.0f;

struct Cube {  // quantisation q = floor((v - v0) * inv_s), cells of side s at level 0
  float x0, y0, z0, inv_s, s;
};

__device__ __forceinline__ unsigned ordered(float v) {  // monotone float -> uint map
  unsigned u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float unordered(unsigned u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// bb[0..2] = ordered min of x, y, z; bb[3..5] = ordered max
__global__ void k_bbox(int64_t n, const float* __restrict__ x, const float* __restrict__ y,
                       const float* __restrict__ z, unsigned* bb) {
  unsigned mn[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, mx[3] = {0u, 0u, 0u};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned v[3] = {ordered(x[i]), ordered(y[i]), ordered(z[i])};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      mn[a] = min(mn[a], v[a]);
      mx[a] = max(mx[a], v[a]);
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    for (int o = 16; o > 0; o >>= 1) {
      mn[a] = min(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
      mx[a] = max(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
    }
  }
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      atomicMin(&bb[a], mn[a]);
      atomicMax(&bb[3 + a], mx[a]);
    }
  }
}

// monotone quantisation to [0, 2^21), explicitly rounded so that every evaluation agrees
__device__ __forceinline__ uint32_t quant(float v, float v0, float inv_s) {
  const float t = __fmul_rn(__fsub_rn(v, v0), inv_s);
  constexpr float QMAX = (float)((1u << HS_QBITS) - 1);
  if (!(t > 0.f)) return 0u;
  if (t >= QMAX) return (1u << HS_QBITS) - 1u;
  return (uint32_t)t;  // truncation = floor for t > 0
}

// the 21 bits of v moved to every third bit (bit b -> bit 3b)
__device__ __forceinline__ uint64_t spread3(uint32_t v) {
  uint64_t x = v & 0x1fffffu;
  x = (x | (x << 32)) & 0x1f00000000ffffull;
  x = (x | (x << 16)) & 0x1f0000ff0000ffull;
  x = (x | (x << 8)) & 0x100f00f00f00f00full;
  x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
  x = (x | (x << 2)) & 0x1249249249249249ull;
  return x;
}

// Position on the 3-D Hilbert curve of 2^21 cells per axis (Skilling 2004, "Programming the
// Hilbert curve": from the top bit down, the sub-cube's axes are reflected or exchanged so that
// the curve leaves every octant next to the one that it enters, then the bits are Gray coded).
__device__ __forceinline__ uint64_t hilbert(uint32_t x, uint32_t y, uint32_t z) {
  uint32_t c[3] = {x, y, z};
#pragma unroll 1
  for (uint32_t bit = 1u << (HS_QBITS - 1); bit > 1; bit >>= 1) {
    const uint32_t low = bit - 1;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const uint32_t swap = (c[a] & bit) ? 0u : (c[0] ^ c[a]) & low;
      const uint32_t flip = (c[a] & bit) ? low : 0u;
      c[0] ^= swap | flip;
      if (a) c[a] ^= swap;
    }
  }
  c[1] ^= c[0];
  c[2] ^= c[1];
  uint32_t t = 0;  // bit b: the parity of the bits of c[2] above b
  for (uint32_t bit = 1u << (HS_QBITS - 1); bit > 1; bit >>= 1)
    if (c[2] & bit) t ^= bit - 1;
  return (spread3(c[0] ^ t) << 2) | (spread3(c[1] ^ t) << 1) | spread3(c[2] ^ t);
}

__global__ void k_curve(int64_t n, const float* __restrict__ x, const float* __restrict__ y,
                         const float* __restrict__ z, Cube c, uint32_t* klo, uint32_t* khi,
                         uint32_t* vals) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t key = hilbert(quant(x[i], c.x0, c.inv_s), quant(y[i], c.y0, c.inv_s),
                               quant(z[i], c.z0, c.inv_s));
  klo[i] = (uint32_t)key;
  khi[i] = (uint32_t)(key >> 32);
  vals[i] = (uint32_t)i;
}

// after the sort by low words (values v1): the high words in that order, identity values
__global__ void k_curve_mid(int64_t n, const uint32_t* __restrict__ khi,
                             const uint32_t* __restrict__ v1, uint32_t* khi1, uint32_t* vals) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  khi1[k] = khi[v1[k]];
  vals[k] = (uint32_t)k;
}

// after the stable sort by high words (values v2 into the first order)
__global__ void k_curve_final(int64_t n, const float* __restrict__ x,
                               const float* __restrict__ y, const float* __restrict__ z,
                               const uint32_t* __restrict__ v1, const uint32_t* __restrict__ v2,
                               uint32_t* ids, float4* pos) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) {  // the last leaf's empty places: within no radius
    if (k < ((n + 31) & ~(int64_t)31)) pos[k] = make_float4(INFINITY, INFINITY, INFINITY, 0.f);
    return;
  }
  const uint32_t i = v1[v2[k]];
  ids[k] = i;
  pos[k] = make_float4(x[i], y[i], z[i], 0.f);
}

// squared distance, rounded the same way wherever it is evaluated
__device__ __forceinline__ float dist2(const float4& o, const float4& p) {
  const float dx = __fsub_rn(o.x, p.x), dy = __fsub_rn(o.y, p.y), dz = __fsub_rn(o.z, p.z);
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// Sums over candidates at distances r of the 3-D cubic spline of Eq. SPH_kernel without
// 8 / (pi h^3), and of its h derivative: with x = r / h, u = (1 - x)_+ and v = (1/2 - x)_+ the
// spline is w = 2 u^3 - 8 v^3, and -x w' follows from the same powers, since x = 1 - u where
// u > 0 and 1/2 - v where v > 0.
struct Sums {
  float u3 = 0.f, v3 = 0.f, u2 = 0.f, v2 = 0.f;
  __device__ __forceinline__ void add(float r, float ih) {
    const float x = r * ih, u = __saturatef(1.0f - x), v = __saturatef(0.5f - x);
    const float uu = u * u, vv = v * v;
    u3 = fmaf(uu, u, u3);
    v3 = fmaf(vv, v, v3);
    u2 += uu;
    v2 += vv;
  }
  // N_eff and dN_eff / dh over `width` lanes
  __device__ __forceinline__ void total(int width, float ih, float& f, float& df) const {
    float s = 2.0f * u3 - 8.0f * v3, ds = 6.0f * (u2 - u3) - 24.0f * (0.5f * v2 - v3);
    for (int o = width / 2; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      ds += __shfl_xor_sync(0xffffffffu, ds, o);
    }
    f = HS_KNORM * s;
    df = HS_KNORM * ds * ih;
  }
};

// N_eff(h) and dN_eff/dh over the warp's candidates: distances buf[0..nc), or (FIRST) squares
// that are replaced by their roots
template <bool FIRST>
__device__ __forceinline__ void neff(float* buf, int nc, float h, int lane, float& f, float& df) {
  const float ih = 1.0f / h;
  Sums t;
#pragma unroll 2
  for (int j = lane; j < nc; j += 32) {
    if (FIRST) buf[j] = sqrtf(buf[j]);
    t.add(buf[j], ih);
  }
  t.total(32, ih, f, df);
}

// ---- tree ----------------------------------------------------------------------------------
constexpr int TREE_MAX = 7;  // 32^7 > 2^32 particles
struct Tree {  // level 0: boxes of 32 particles; level l: of 32 boxes of level l - 1
  const float4* lo[TREE_MAX];
  const float4* hi[TREE_MAX];
  uint32_t cnt[TREE_MAX];
  int top;  // the level of at most 32 boxes
};

// boxes of 32 consecutive boxes (or points, plo == phi) each, one warp per box
__global__ void k_tree(int64_t n, const float4* __restrict__ plo, const float4* __restrict__ phi,
                       float4* lo, float4* hi) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (32 * w >= n) return;
  const int64_t i = 32 * w + lane < n ? 32 * w + lane : n - 1;
  const float4 a = plo[i], b = phi[i];
  const auto umin = [](float v) { return unordered(__reduce_min_sync(0xffffffffu, ordered(v))); };
  const auto umax = [](float v) { return unordered(__reduce_max_sync(0xffffffffu, ordered(v))); };
  const float4 mn = make_float4(umin(a.x), umin(a.y), umin(a.z), 0.f);
  const float4 mx = make_float4(umax(b.x), umax(b.y), umax(b.z), 0.f);
  if (lane == 0) {
    lo[w] = mn;
    hi[w] = mx;
  }
}

// Depth first over the leaves whose boxes come within sqrt(R2) of the box [lo, hi] (a point:
// lo == hi): leaves(node, hits, box lo, box hi) for every lowest node with some, until it
// returns false; its leaf 32 node + lane is one of them if bit lane of hits is set.  Rounding
// is monotone and the gaps are squared and summed as in dist2, so no particle with dist2 < R2
// is in a leaf left out.  Every lane tests one of a node's 32 children.
template <class Leaves>
__device__ __forceinline__ void search(const Tree& t, const float3& lo, const float3& hi, float R2,
                                       int lane, Leaves&& leaves) {
  float4 bl, bh;
  const auto test = [&](int l, uint32_t node) -> unsigned {
    const uint32_t c = node * 32 + lane;
    bool hit = false;
    if (c < t.cnt[l]) {
      bl = t.lo[l][c];
      bh = t.hi[l][c];
      const float4 g = make_float4(fmaxf(fmaxf(bl.x - hi.x, lo.x - bh.x), 0.f),
                                   fmaxf(fmaxf(bl.y - hi.y, lo.y - bh.y), 0.f),
                                   fmaxf(fmaxf(bl.z - hi.z, lo.z - bh.z), 0.f), 0.f);
      hit = dist2(g, make_float4(0.f, 0.f, 0.f, 0.f)) < R2;
    }
    return __ballot_sync(0xffffffffu, hit);
  };
  unsigned mask[TREE_MAX];
  uint32_t node[TREE_MAX];
  int l = t.top;
  uint32_t at = 0;
  for (;;) {
    const unsigned m = test(l, at);
    if (l == 0) {
      if (m && !leaves(at, m, bl, bh)) return;
    } else {
      mask[l] = m;
      node[l] = at;
      --l;
    }
    // the next node at level l: a child of the deepest one with some left
    while (l < t.top && mask[l + 1] == 0) ++l;
    if (l == t.top) return;
    at = node[l + 1] * 32 + __ffs(mask[l + 1]) - 1;
    mask[l + 1] &= mask[l + 1] - 1;
  }
}

// the sums of neff over a search, for the rare particle whose candidates overflow the buffer (a
// dense clump near the kernel's edge)
__device__ __forceinline__ void neff_stream(const Tree& t, const float4* __restrict__ pos,
                                            const float4& p, float R, float h, int lane,
                                            float& f, float& df) {
  const float ih = 1.0f / h;
  const float3 c = make_float3(p.x, p.y, p.z);
  Sums sum;
  search(t, c, c, R * R, lane, [&](uint32_t node, unsigned hits, const float4&, const float4&) {
    for (; hits; hits &= hits - 1)
      sum.add(sqrtf(dist2(pos[((uint64_t)node * 32 + __ffs(hits) - 1) * 32 + lane], p)), ih);
    return true;
  });
  sum.total(32, ih, f, df);
}

// ---- groups of particles -------------------------------------------------------------------
// neff of a quarter warp's list; steps: of 8 candidates, the most any quarter needs
template <bool FIRST>
__device__ __forceinline__ void neff_quarter(float* l, int len, int steps, float h, int sub,
                                             float& f, float& df) {
  const float ih = 1.0f / h;
  Sums t;
#pragma unroll 2
  for (int i = 0; i < steps; ++i) {
    const int j = 8 * i + sub;
    float d = INFINITY;
    if (j < len) {
      d = l[j];
      if (FIRST) l[j] = d = sqrtf(d);
    }
    t.add(d, ih);
  }
  t.total(8, ih, f, df);
}

// one Newton step on ln N_eff(ln h) = ln n_ngb (nearly linear) from x inside the bisection
// bracket [lo, hi]; h: the answer so far; step: the length of the last step if it was one of
// Newton's, else infinite (as at first); false: this step is the last.  A step that is not half as
// long as Newton's last becomes a bisection: with a clump between x and the root, Newton can jump
// to and fro between its two sides, both within the bracket, for ever (light-cone particles, N_ngb
// = 200: 3 in 1e5).  The bracket includes its ends: a step that rounds to none has converged.
__device__ __forceinline__ bool newton(float n_ngb, float f, float df, float& x, float& lo,
                                       float& hi, float& h, float& step) {
  const float F = f - n_ngb;
  if (F < 0.f) lo = x; else hi = x;
  h = x;
  if (fabsf(F) <= 1e-6f * n_ngb) return false;
  float xn = (df > 0.f) ? x * __expf(__logf(n_ngb / f) * f / (x * df)) : 0.f;
  const bool in = xn >= lo && xn <= hi && fabsf(xn - x) < 0.5f * step && xn > 0.f;
  if (!in) xn = 0.5f * (lo + hi);
  const float s = fabsf(xn - x);
  step = in ? s : INFINITY;
  // what a Newton step leaves is of the order of its square; next to it the FP32 sums' rounding
  // is the larger part (stopping at 1e-6 instead leaves the same errors, at 0.6 more steps)
  const bool last = s <= (in ? 2e-4f : 1e-6f) * x || hi - lo <= 1e-6f * hi;
  h = x = xn;
  return !last;
}

// First radius of every particle (curve order), a thread each: 1.25 x the caller's guess, or
// from the distances to the particles around it on the curve (spatial neighbours, mostly).  A
// guess far above the size of the particle's leaf (32 particles), and above four times what those
// distances give, would only be searched in vain, thousands of particles a time: it is left.
// (1e5 particles, N_ngb = 64, with and without this: guesses of h 0.68 and 0.67 ms, of 10 h 1.3 and
// 8.1 ms, of 1000 h 1.2 and 129 ms.)  Not with so few particles that h can be any multiple of
// their extent.
__global__ void __launch_bounds__(128)
    k_hs_start(int64_t n, const float4* __restrict__ pos, const uint32_t* __restrict__ ids, Cube cb,
               float n_ngb, const float* __restrict__ guess, float* R0) {
  __shared__ float4 s_c[4][64];
  __shared__ float s_d[4][64 * 32];
  constexpr unsigned ALL = 0xffffffffu;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t k0 = (int64_t)blockIdx.x * 128 + 32 * w, k = k0 + lane;
  if (k0 >= n) return;  // whole warps leave together
  const int64_t kk = k < n ? k : n - 1;
  const float4 p = pos[kk];
  float R = 0.f;
  if (guess) {
    const float gv = guess[ids[kk]];
    if (gv > 0.f && isfinite(gv)) R = 1.25f * gv;
  }
  float far = INFINITY;
  if (guess && n_ngb < (float)n) {
    const auto extent = [&](float v) {
      const unsigned o = ordered(v);
      return unordered(__reduce_max_sync(ALL, o)) - unordered(__reduce_min_sync(ALL, o));
    };
    const float4 e = make_float4(extent(p.x), extent(p.y), extent(p.z), 0.f);
    far = HS_FAR * sqrtf(dist2(e, make_float4(0.f, 0.f, 0.f, 0.f))) * cbrtf(n_ngb / 64.0f);
  }
  if (__any_sync(ALL, R == 0.f || R > far)) {
    // the median distance to the 64 particles around the warp's on the curve, scaled to
    // hold HG_START N_ngb particles at that density
    const int W = n < 64 ? (int)n : 64;
    int64_t j0 = k0 - 16;
    if (j0 > n - W) j0 = n - W;
    if (j0 < 0) j0 = 0;
    float* list = s_d[w] + lane;
    for (int j = lane; j < W; j += 32) s_c[w][j] = pos[j0 + j];
    __syncwarp();
    float m = 0.f;
    for (int j = 0; j < W; ++j) {
      const float d2 = dist2(s_c[w][j], p);
      list[j * 32] = d2;
      m = fmaxf(m, d2);
    }
    // bisection on the bit patterns, from 2^-16 of the largest: 1/8 octave of d^2
    uint32_t b = __float_as_uint(m), a = b > (16u << 23) ? b - (16u << 23) : 0u;
#pragma unroll 1
    for (int it = 0; it < 7; ++it) {
      const uint32_t c = a + ((b - a) >> 1);
      const float cf = __uint_as_float(c);
      int cnt = 0;
#pragma unroll 8
      for (int j = 0; j < W; ++j) cnt += list[j * 32] <= cf;
      if (2 * cnt > W) b = c; else a = c;
    }
    const float E =
        fmaxf(sqrtf(__uint_as_float(b)) * cbrtf(2.0f * HG_START * n_ngb / (float)W), cb.s);
    if (R == 0.f || (R > far && R > 4.0f * E)) R = E;
  }
  if (k < n) R0[k] = R;
}

// A full list of squares l[0..m) within R.  N_eff of some of the candidates is a lower bound of
// N_eff, so a radius at which it reaches N_ngb bounds h from above: R and the list shrink to
// such a radius (false: R itself is too short for that).
__device__ __forceinline__ bool shrink(float* l, int& m, float& R, float n_ngb, int lane) {
  float x = R, best = R;
#pragma unroll 1
  for (int it = 0; it < 3; ++it) {
    const float ih = 1.0f / x;
    Sums t;
    for (int j = lane; j < m; j += 32) t.add(sqrtf(l[j]), ih);
    float f, df;
    t.total(32, ih, f, df);
    if (f >= n_ngb) {
      best = x;
      x *= 1.01f * cbrtf(n_ngb / f);
      if (!(x < best)) break;
    } else {
      if (it == 0) return false;
      x = 0.5f * (x + best);
    }
  }
  R = best;
  int q = 0;
  for (int j0 = 0; j0 < m; j0 += 32) {
    const int j = j0 + lane;
    const float d2 = j < m ? l[j] : INFINITY;
    const bool in = d2 < best * best;
    const unsigned msk = __ballot_sync(0xffffffffu, in);
    if (in) l[q + __popc(msk & ((1u << lane) - 1u))] = d2;  // (never ahead of the reads)
    q += __popc(msk);
    __syncwarp();
  }
  m = q;
  return true;
}

// One warp per group of consecutive particles: the leaves near any of them are collected once
// (a group whose leaves are too many is halved), then every particle tests those leaves' boxes
// and the particles of the ones it meets, 32 at a time, and four particles' lists are solved
// together, a quarter warp each: an evaluation costs its instructions and two rounds of
// shuffles for four particles at once.
__global__ void __launch_bounds__(32)
    k_hsml_group(int64_t n, const float4* __restrict__ pos, const Tree tree,
                 const uint32_t* __restrict__ ids, const float* __restrict__ R0, float n_ngb,
                 int cap, float* h_out, uint32_t* left_k, float* left_R,
                 unsigned long long* n_left) {
  extern __shared__ float s_dyn[];
  constexpr unsigned ALL = 0xffffffffu;
  __shared__ float s_box[6][HG_LEAVES];
  __shared__ uint32_t s_leaf[HG_LEAVES];
  const int lane = threadIdx.x, sub = lane & 7, quarter = lane >> 3;
  const unsigned below = (1u << lane) - 1u;
  const int64_t k = (int64_t)blockIdx.x * HG_SIZE + lane;  // lanes of particles: the first ones
  bool act = lane < HG_SIZE && k < n;
  const int64_t kk = act ? k : n - 1;
  const float4 p = pos[kk];
  const uint32_t id = ids[kk];
  float R = R0[kk];
  auto leave = [&](bool out) {  // to the kernel of a warp per particle
    const unsigned pm = __ballot_sync(ALL, out);
    if (!pm) return;
    unsigned long long at = 0;
    if (lane == 0) at = atomicAdd(n_left, (unsigned long long)__popc(pm));
    at = __shfl_sync(ALL, at, 0);
    if (out) {
      const unsigned long long q = at + __popc(pm & below);
      left_k[q] = (uint32_t)k;
      left_R[q] = R;
      act = false;
    }
  };
  for (int round = 0; round < HG_ROUNDS && __any_sync(ALL, act); ++round) {
    int a = 0, s = HG_SIZE;
    while (a < HG_SIZE) {
      const bool part = act && lane >= a && lane < a + s;
      unsigned todo = __ballot_sync(ALL, part);
      const int na = __popc(todo);
      if (na == 0) {
        a += s;
        s = a & -a;
        continue;
      }
      // the participants' box and largest radius
      float3 lo, hi;
      const auto umin = [&](float v) {
        return unordered(__reduce_min_sync(ALL, part ? ordered(v) : 0xffffffffu));
      };
      const auto umax = [&](float v) {
        return unordered(__reduce_max_sync(ALL, part ? ordered(v) : 0u));
      };
      lo.x = umin(p.x); lo.y = umin(p.y); lo.z = umin(p.z);
      hi.x = umax(p.x); hi.y = umax(p.y); hi.z = umax(p.z);
      const float Rm = umax(R), Rm2 = Rm * Rm;
      // the leaves within Rm of the box
      int nleaf = 0;
      search(tree, lo, hi, Rm2, lane, [&](uint32_t node, unsigned hits, const float4& bl,
                                          const float4& bh) {
        const int at = nleaf + __popc(hits & below);
        if ((hits >> lane & 1u) && at < HG_LEAVES) {
          s_leaf[at] = (node * 32 + lane) * 32;
          s_box[0][at] = bl.x; s_box[1][at] = bl.y; s_box[2][at] = bl.z;
          s_box[3][at] = bh.x; s_box[4][at] = bh.y; s_box[5][at] = bh.z;
        }
        nleaf += __popc(hits);
        return nleaf <= HG_LEAVES;
      });
      __syncwarp();
      if (nleaf > HG_LEAVES) {  // too many for one group: halves, then the other kernel
        if (s > 1) s >>= 1;
        else {
          leave(part);
          a += s;
          s = a & -a;
        }
        continue;
      }
      // every participant's candidates, up to four lists at a time
      while (todo) {
        int mine_l = 0, len = 0, steps = 0;  // this quarter's particle and list
        bool has = false;
        for (int q = 0; q < 4 && todo; ++q) {
          const int b = __ffs(todo) - 1;
          todo &= todo - 1;
          const float4 pb = make_float4(__shfl_sync(ALL, p.x, b), __shfl_sync(ALL, p.y, b),
                                        __shfl_sync(ALL, p.z, b), 0.f);
          float Rb = __shfl_sync(ALL, R, b), R2 = Rb * Rb;
          float* l = s_dyn + q * (cap + 72);  // lists 8 banks apart (cap: a multiple of 32)
          int m = 0;
          for (int l0 = 0; l0 < nleaf; l0 += 32) {
            const int j = l0 + lane;
            bool hit = false;
            if (j < nleaf) {
              const float4 gap = make_float4(
                  fmaxf(fmaxf(s_box[0][j] - pb.x, pb.x - s_box[3][j]), 0.f),
                  fmaxf(fmaxf(s_box[1][j] - pb.y, pb.y - s_box[4][j]), 0.f),
                  fmaxf(fmaxf(s_box[2][j] - pb.z, pb.z - s_box[5][j]), 0.f), 0.f);
              hit = dist2(gap, make_float4(0.f, 0.f, 0.f, 0.f)) < R2;
            }
            unsigned hits = __ballot_sync(ALL, hit);
            auto take = [&](const float4& c) {
              const float d2 = dist2(c, pb);
              const unsigned msk = __ballot_sync(ALL, d2 < R2);
              if (d2 < R2) l[m + __popc(msk & below)] = d2;  // (m <= cap: 64 places more)
              m += __popc(msk);
            };
            while (hits) {  // two leaves at a time: their loads overlap
              const float4 c0 = pos[s_leaf[l0 + __ffs(hits) - 1] + lane];
              hits &= hits - 1;
              const bool two = hits != 0;
              const float4 c1 = pos[two ? s_leaf[l0 + __ffs(hits) - 1] + lane : 0];
              hits &= hits - 1;
              take(c0);
              if (two) take(c1);
              if (m > cap) {
                __syncwarp();
                if (shrink(l, m, Rb, n_ngb, lane)) R2 = Rb * Rb;
                if (lane == b) R = Rb;
                if (m > cap) {  // a dense clump at the edge
                  hits = 0;
                  l0 = nleaf;
                }
              }
            }
          }
          if (quarter == q) {
            mine_l = b;
            len = m;
            has = true;
          }
          steps = max(steps, (m + 7) >> 3);
        }
        __syncwarp();
        float* l = s_dyn + quarter * (cap + 72);
        const float Rq = __shfl_sync(ALL, R, mine_l);
        float f, df;
        neff_quarter<true>(l, len, steps, Rq, sub, f, df);
        __syncwarp();
        const bool found = has && f >= n_ngb;
        bool run = found && f - n_ngb >= 1e-6f * n_ngb;
        float h = Rq, xlo = 0.f, xhi = Rq, step = INFINITY;
        float x = run ? fminf(Rq, fmaxf(0.5f * Rq, Rq * cbrtf(n_ngb / f))) : Rq;
        const float f_R = f;
        for (int it = 0; it < 40 && __any_sync(ALL, run); ++it) {
          neff_quarter<false>(l, len, steps, x, sub, f, df);
          if (run) run = newton(n_ngb, f, df, x, xlo, xhi, h, step);
        }
        // back to the particles' lanes
        bool gone = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int b = __shfl_sync(ALL, has ? mine_l : -1, 8 * q);
          const bool ok = __shfl_sync(ALL, (int)found, 8 * q);
          const float hb = __shfl_sync(ALL, h, 8 * q), fb = __shfl_sync(ALL, f_R, 8 * q);
          const int lb = __shfl_sync(ALL, len, 8 * q);
          if (lane == b) {
            if (ok && lb <= cap) {
              h_out[id] = hb;
              act = false;
            } else if (lb > cap) {
              gone = true;
              if (ok) R = 1.0001f * hb;  // (an upper bound of h, nearly)
            } else {  // not enough within R: grow
              R *= fminf(fmaxf(1.1f * cbrtf(n_ngb / fmaxf(fb, 1e-3f)), 1.15f), 4.0f);
            }
          }
        }
        leave(gone);
        __syncwarp();
      }
      a += s;
      s = a & -a;
    }
  }
  leave(act);
}

// One warp per particle: every particle of a call with a large N_ngb (a block each, as far as the
// grid goes), or the ones that the groups
// left (5 % in a light-cone: field particles with a halo at the edge of their kernel, hundreds of
// candidates of little weight), fetched one by one.
__global__ void __launch_bounds__(32)
    k_hsml(int64_t n, const float4* __restrict__ pos, const Tree tree,
           const uint32_t* __restrict__ ids, float n_ngb, int cap, const float* __restrict__ R0,
           const uint32_t* __restrict__ left_k, const float* __restrict__ left_R,
           const unsigned long long* n_left, unsigned long long* next, float* h_out,
           int64_t* nfail) {
  extern __shared__ float s_dyn[];
  const int lane = threadIdx.x;
  float* buf = s_dyn;
  // every particle, or the ones the groups left
  const int64_t todo = left_k ? (int64_t)*n_left : n;
  for (int64_t item = blockIdx.x;; item += gridDim.x) {
    if (left_k) {  // (their work varies by orders of magnitude)
      unsigned long long q = 0;
      if (lane == 0) q = atomicAdd(next, 1ull);
      item = (int64_t)__shfl_sync(0xffffffffu, q, 0);
    }
    if (item >= todo) break;
    const int64_t k = left_k ? left_k[item] : item;
    const float4 p = pos[k];
    const float3 pc = make_float3(p.x, p.y, p.z);
    const uint32_t id = ids[k];
    float R = left_k ? left_R[item] : R0[k];
    float r_short = 0.f, r_over = INFINITY;  // N_eff too small at r_short; too many at r_over
    float cut = 0.63f;  // next cut of a radius with far too many particles
    float h = __int_as_float(0x7fc00000);
    bool done = false;
    for (int round = 0; round < HS_MAX_ROUNDS && !done; ++round) {
      const float R2 = R * R;
      // the particles within R, in tree order
      uint32_t off = 0;
      search(tree, pc, pc, R2, lane, [&](uint32_t node, unsigned hits, const float4&,
                                         const float4&) {
        while (hits) {  // four leaves at a time: their loads overlap
          float d2[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            d2[q] = INFINITY;
            if (hits) d2[q] = dist2(pos[((uint64_t)node * 32 + __ffs(hits) - 1) * 32 + lane], p);
            hits &= hits - 1;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const bool in = d2[q] < R2;
            const unsigned m = __ballot_sync(0xffffffffu, in);
            const uint32_t at = off + __popc(m & ((1u << lane) - 1u));
            if (in && at < (uint32_t)cap) buf[at] = d2[q];
            off += __popc(m);
          }
        }
        return off <= (uint32_t)(HS_SCAN_CAPS * cap);
      });
      __syncwarp();
      if (off > (uint32_t)(HS_SCAN_CAPS * cap)) {  // far too many: try a smaller radius first
        const float Rn = (r_short > 0.f ? 0.63f : cut) * R;
        if (Rn > r_short) {  // (how many is not known: the cuts get deeper until one is too deep)
          cut = fmaxf(cut * cut, 0.02f);
          R = Rn;
          __syncwarp();
          continue;
        }
      }
      // too many candidates: shrink towards the last short radius while that bracket is wide,
      // else stream the sums over the cube at this radius
      const bool stream = off > (uint32_t)cap;
      if (stream && !(r_short > 0.f && R <= 1.3f * r_short) && round < HS_MAX_ROUNDS - 8) {
        r_over = R;
        R = fmaxf(r_short, R * cbrtf(0.5f * cap / (float)off));
        if (!(R > r_short)) R = 0.5f * (r_short + r_over);
        continue;
      }
      const int total = (int)off;
      float f, df;
      if (stream) neff_stream(tree, pos, p, R, R, lane, f, df);
      else neff<true>(buf, total, R, lane, f, df);
      if (f < n_ngb) {  // not enough within R: grow
        r_short = R;
        float grow = 1.1f * cbrtf(n_ngb / fmaxf(f, 1e-3f));
        grow = fminf(fmaxf(grow, 1.15f), 4.0f);
        R = fminf(R * grow, 0.5f * (R + r_over));
        if (!(R > r_short)) R = r_short * 1.15f;
        __syncwarp();
        continue;
      }
      // N_eff(R) >= n_ngb: the root in (0, R]
      h = R;
      if (f - n_ngb >= 1e-6f * n_ngb) {
        float lo = 0.f, hi = R, step = INFINITY;
        float x = fminf(R, fmaxf(0.5f * R, R * cbrtf(n_ngb / f)));
        for (int it = 0; it < 40; ++it) {
          if (stream) neff_stream(tree, pos, p, R, x, lane, f, df);
          else neff<false>(buf, total, x, lane, f, df);
          if (!newton(n_ngb, f, df, x, lo, hi, h, step)) break;
        }
      }
      done = true;
      __syncwarp();
    }
    if (lane == 0) {
      h_out[id] = done ? h : __int_as_float(0x7fc00000);
      if (!done) atomicAdd((unsigned long long*)nfail, 1ull);
    }
    __syncwarp();
  }
}

}  // namespace

extern "C" int bp_smoothing_lengths(bp_ctx* ctx, int64_t n, const float* x, const float* y,
                                    const float* z, double n_ngb, const float* h_guess,
                                    float* h_out) {
  if (!ctx) return BP_EINVAL;
  if (n < 0) return bp_fail(ctx, BP_EINVAL, "bp_smoothing_lengths: n < 0");
  if (n == 0) return BP_OK;
  if (!x || !y || !z || !h_out) return bp_fail(ctx, BP_EINVAL, "bp_smoothing_lengths: null pointer");
  if (!(n_ngb > 32.0 / 3.0) || !(n_ngb <= HS_CAP_MAX / 2))
    return bp_fail(ctx, BP_EINVAL, "bp_smoothing_lengths: n_ngb must be in (32/3, %d]",
                   HS_CAP_MAX / 2);
  if (32.0 / 3.0 * (double)n <= n_ngb)
    return bp_fail(ctx, BP_ERANGE, "bp_smoothing_lengths: %lld particles cannot reach n_ngb",
                   (long long)n);
  if (n >= ((int64_t)1 << 32))
    return bp_fail(ctx, BP_ERANGE, "bp_smoothing_lengths: n >= 2^32");
  int r;
  // bounding box
  unsigned* bb;
  if ((r = bp_ws(ctx, WS_MISC2, 64, (void**)&bb))) return r;
  const unsigned init[8] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u, 0u, 0u};
  BP_CUDA(ctx, cudaMemcpyAsync(bb, init, sizeof(init), cudaMemcpyHostToDevice, ctx->stream));
  k_bbox<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4 * ctx->num_sms), 256, 0, ctx->stream>>>(
      n, x, y, z, bb);
  BP_LAUNCH_CHECK(ctx, "bbox");
  unsigned hb[8];
  BP_CUDA(ctx, cudaMemcpyAsync(hb, bb, sizeof(hb), cudaMemcpyDeviceToHost, ctx->stream));
  BP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  auto unord = [](unsigned u) {
    u = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
    float f;
    memcpy(&f, &u, 4);
    return (double)f;
  };
  double lo[3], ext[3];
  for (int a = 0; a < 3; ++a) {
    lo[a] = unord(hb[a]);
    ext[a] = unord(hb[3 + a]) - lo[a];
    if (!std::isfinite(lo[a]) || !std::isfinite(ext[a]))
      return bp_fail(ctx, BP_EINVAL, "bp_smoothing_lengths: non-finite positions");
  }
  // quantisation cube: the bounding box's largest side split into 2^21 level-0 cells
  double D = std::max(ext[0], std::max(ext[1], ext[2]));
  if (!(D > 0.0)) D = 1.0;
  Cube cb;
  cb.x0 = (float)lo[0];
  cb.y0 = (float)lo[1];
  cb.z0 = (float)lo[2];
  cb.inv_s = (float)((double)(1u << HS_QBITS) / (D * (1.0 + 1e-6)));
  cb.s = (float)(1.0 / (double)cb.inv_s);
  // curve order: sort by the low key words, then stably by the high words
  uint32_t *A, *B, *C, *Dv, *E, *F, *G;
  if ((r = bp_ws(ctx, WS_KEYS0, (size_t)n * 4, (void**)&A))) return r;
  if ((r = bp_ws(ctx, WS_VALS0, (size_t)n * 4, (void**)&B))) return r;
  if ((r = bp_ws(ctx, WS_KEYS1, (size_t)n * 4, (void**)&C))) return r;
  if ((r = bp_ws(ctx, WS_VALS1, (size_t)n * 4, (void**)&Dv))) return r;
  if ((r = bp_ws(ctx, WS_COUNTS, (size_t)n * 4, (void**)&E))) return r;
  if ((r = bp_ws(ctx, WS_UNITS, (size_t)n * 4, (void**)&F))) return r;
  if ((r = bp_ws(ctx, WS_OFFS, (size_t)n * 4, (void**)&G))) return r;
  const unsigned nb = (unsigned)((n + 255) / 256);
  k_curve<<<nb, 256, 0, ctx->stream>>>(n, x, y, z, cb, A, E, B);
  BP_LAUNCH_CHECK(ctx, "curve keys");
  uint32_t *klo_s, *v1;
  if ((r = bp_radix_sort_pairs(ctx, A, B, C, Dv, n, 32, &klo_s, &v1))) return r;
  uint32_t* t0 = (klo_s == A) ? C : A;  // the pair the first sort's result does not occupy
  uint32_t* t1 = (klo_s == A) ? Dv : B;
  k_curve_mid<<<nb, 256, 0, ctx->stream>>>(n, E, v1, F, G);
  BP_LAUNCH_CHECK(ctx, "curve high words");
  uint32_t *khi_s, *v2;
  if ((r = bp_radix_sort_pairs(ctx, F, G, t0, t1, n, 3 * HS_QBITS - 32, &khi_s, &v2))) return r;
  float4* pos;
  if ((r = bp_ws(ctx, WS_HPAR, (size_t)((n + 31) & ~(int64_t)31) * sizeof(float4),
                 (void**)&pos))) return r;
  k_curve_final<<<nb, 256, 0, ctx->stream>>>(n, x, y, z, v1, v2, E, pos);
  BP_LAUNCH_CHECK(ctx, "curve order");
  // boxes, level by level
  Tree tree;
  memset(&tree, 0, sizeof(tree));
  int64_t off[TREE_MAX], boxes = 0;
  for (int64_t c = (n + 31) / 32, l = 0;; c = (c + 31) / 32, ++l) {
    tree.cnt[l] = (uint32_t)c;
    tree.top = (int)l;
    off[l] = boxes;
    boxes += c;
    if (c <= 32) break;
  }
  float4* box;
  if ((r = bp_ws(ctx, WS_TILES, (size_t)boxes * 2 * sizeof(float4), (void**)&box))) return r;
  for (int l = 0; l <= tree.top; ++l) {
    const int64_t m = l ? tree.cnt[l - 1] : n;
    k_tree<<<(unsigned)((tree.cnt[l] + 3) / 4), 128, 0, ctx->stream>>>(
        m, l ? tree.lo[l - 1] : pos, l ? tree.hi[l - 1] : pos, box + off[l],
        box + boxes + off[l]);
    BP_LAUNCH_CHECK(ctx, "tree");
    tree.lo[l] = box + off[l];
    tree.hi[l] = box + boxes + off[l];
  }
  // (the sorts' arrays are free again; E holds the ids)
  k_hs_start<<<(unsigned)((n + 127) / 128), 128, 0, ctx->stream>>>(
      n, pos, E, cb, (float)n_ngb, h_guess, (float*)F);
  BP_LAUNCH_CHECK(ctx, "first radii");
  const int cap = n < HS_MANY ? HS_CAP_FEW : HS_CAP;
  const size_t smem = cap * sizeof(float);
  BP_CUDA(ctx, cudaFuncSetAttribute(k_hsml, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem));
  BP_CUDA(ctx, cudaMemsetAsync(ctx->d_counter + 5, 0, sizeof(int64_t), ctx->stream));
  const uint32_t* left_k = nullptr;
  const float* left_R = nullptr;
  unsigned long long* n_left = (unsigned long long*)(ctx->d_counter + 8);
  int64_t blocks = n;
  if (n_ngb <= HG_NGB_MAX) {
    const int gcap = ((int)(HG_LIST * n_ngb) + 31) & ~31;
    const size_t gsmem = (size_t)4 * (gcap + 72) * sizeof(float);
    BP_CUDA(ctx, cudaFuncSetAttribute(k_hsml_group, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)gsmem));
    BP_CUDA(ctx, cudaMemsetAsync(n_left, 0, 2 * sizeof(*n_left), ctx->stream));
    k_hsml_group<<<(unsigned)((n + HG_SIZE - 1) / HG_SIZE), 32, gsmem, ctx->stream>>>(
        n, pos, tree, E, (const float*)F, (float)n_ngb, gcap, h_out, A, (float*)B, n_left);
    BP_LAUNCH_CHECK(ctx, "smoothing lengths of groups");
    left_k = A;
    left_R = (const float*)B;
    blocks = std::min(blocks, (int64_t)ctx->num_sms * 26);  // (they fetch their particles)
  }
  k_hsml<<<bp_item_grid(blocks), 32, smem, ctx->stream>>>(
      n, pos, tree, E, (float)n_ngb, cap, (const float*)F, left_k, left_R, n_left, n_left + 1,
      h_out, ctx->d_counter + 5);
  BP_LAUNCH_CHECK(ctx, "smoothing lengths");
  BP_CUDA(ctx, cudaMemcpyAsync(ctx->h_pinned + 5, ctx->d_counter + 5, sizeof(int64_t),
                               cudaMemcpyDeviceToHost, ctx->stream));
  BP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (ctx->h_pinned[5] > 0)
    return bp_fail(ctx, BP_ENOCONV, "bp_smoothing_lengths: %lld particles did not converge",
                   (long long)ctx->h_pinned[5]);
  return BP_OK;
}
