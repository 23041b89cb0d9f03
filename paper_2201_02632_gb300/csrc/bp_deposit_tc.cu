// bp_deposit_tc.cu -- the particle deposit (Section 3.4: the separable pixel-integrated
// kernel f_ij and the integrated SPH kernel) on the fifth-generation tensor cores.
//
// For one 64 x 64 pixel tile and a slab of 16 particles k the y and b contributions are
//   Y[j, i] += sum_k (Y_k wy_k(j)) wx_k(i),     B[j, i] += sum_k (B_k wy_k(j)) wx_k(i),
// a rank-16 update, i.e. one 128 x 64 x 16 GEMM with the y rows and b rows stacked in M:
//   A[r, k] = Y_k wy_k(r)  (r < 64),   B_k wy_k(r - 64)  (r >= 64);    Bop[i, k] = wx_k(i).
// A cell weight is the difference of the integrated kernel at the cell's two edges, in
// the split representation of bp_wsplit_inv (w(u) left of the particle, w(u) - 1 = -w(-u)
// right of it, plus 1 for the cell holding the particle).  The edge value uses the
// truncated-power form of the piecewise quartic: with a = |u|,
//   w_left(a) = (2/3) max(1 - a, 0)^4 - (8/3) max(1/2 - a, 0)^4,
// which is the inner piece 1/2 - (4/3) a + (8/3) a^3 - 2 a^4 below a = 1/2, the outer piece
// (2/3)(1 - a)^4 above and zero beyond a = 1: no branch and no piece selection (two
// saturating FMAs, four multiplies and a sign flip).
//
// Products are formed by kind::f16 MMAs on FP16 operands: each FP32 operand is scaled by a
// power of two and split into an FP16 head (11 significant bits) and the FP16 rounding of the
// exact rest, a b ~ ah bh + ah bt + at bh (three MMAs; about 1e-6 relative error per product).
// The column weights (at most 1) are scaled by 2^14; the A rows by 2^s per accumulation
// group, s chosen from the group's largest |Y| (|B| for the b rows) so that the largest
// value lies in [2^14, 2^15): far below the FP16 maximum, and contributions that would fall
// below the FP16 normal range are below 2^-28 of the group's largest.  A group is two halves
// of TC_HS slabs (96 particles), each accumulated in FP32 in tensor memory; their sum, its
// scale undone exactly, is folded into a compensated (sum, compensation) pair by Kahan's
// summation, also kept in tensor memory.
//
// One CTA of 24 warps per SM, persistent over work units; no CTA barrier in the loop, every
// hand-over through mbarriers:
//  - 18 producer warps.  A warp takes a slab of 16 particles (one MMA K-step) at a time, every
//    18th of the CTA: its lanes turn the records (held in registers, loaded two slabs ahead)
//    into per-(particle, axis) fields, publish the largest |Y|, |B| of its next slab for that
//    group's scale, and fill the slab in four rounds of four particles.  A half warp evaluates
//    one particle's integrated kernel at four consecutive edges per lane (the fifth from the
//    neighbour), differences, scales and splits them and stores 8 bytes of each 128-byte
//    operand row: MN-major operands, so that a lane's cells are contiguous, the stores have no
//    bank conflicts and the arithmetic runs on packed pairs (add / mul / fma.f32x2).  The cell
//    holding the particle's centre (difference + 1) is written afterwards by one lane per
//    (particle, axis).  h = 0 becomes an infinite kernel scale (a nearest-grid-point weight
//    without a branch) and a slot past the unit's end a particle far outside the tile.  A slab
//    without y skips the y rows (zeroed once).
//  - 2 MMA warps, one thread each, issue the slabs' MMAs in slab order, so that every
//    accumulator sums its particles in a fixed order; each takes a half of every group, with an
//    accumulator of its own (the issuing thread is the serial part: one warp alone held the CTA
//    to 700 cycles per slab).
//  - 4 fold warps fold the finished groups (three accumulator pairs in rotation) and write the
//    finished tile out; the first also fetches the units, two ahead.
// The 17 slabs (12 KB each) rotate among the warps, so a warp waits only for the MMAs 17 slabs
// back.  What bounds it: instruction issue (72% of the issue slots used on the 4e6-particle
// cone, 24 warps per SM; 104 warp instructions per (tile, particle) pair), the fixed-latency and
// FP32-pipe stalls between them, then 10% of the producers' time waiting for a free slab.
// Measured, k_deposit_tc on the 4e6-particle cone and on the 5e8-particle cone: 3.44 and 195.6
// ms with two CTAs of eight warps filling K-major stages of 64 particles together (each MMA
// batch waited for the slowest of eight warps); 3.07 ms with slabs owned by one warp, MN-major;
// 2.80 and 156 ms with the round loop rolled (the unrolled body missed the instruction cache);
// 2.66 and 145 ms with packed pairs; 2.54 and 140.4 ms with the 24 specialised warps.
// Accumulating groups of 128 particles singly (four fold warps, half the additions) is 1%
// slower and less exact (relative L2 error against 64 bits 3.4e-7 against 2.8e-7).
//
// TMEM (512 columns x 128 lanes): accumulator pair p at [128 p, 128 p + 128), HI = [384, 448)
// (sums), LO = [448, 512) (compensations).  Lane r is tile row r of y (r < 64) or of b (r >= 64);
// column i is tile column i.
//
// Every wait is bounded; on a timeout the CTA sets *err, stops taking work, waits (bounded)
// for its MMAs in flight and frees its tensor memory.
#include <cuda_fp16.h>

#include "bp_internal.cuh"
#include "bp_tc.cuh"

namespace {

constexpr int TC_TS = 64;        // tile side (pixels)
constexpr int TC_PW = 16;        // particles of a slab: one MMA K-step
constexpr int TC_PROD = 18;      // producer warps
constexpr int TC_MMA = 2;        // MMA warps (a half of each accumulation group each)
constexpr int TC_FOLD = 4;       // fold warps (one per tensor-memory lane quarter)
constexpr int TC_FOLD0 = TC_PROD + TC_MMA;  // the first fold warp
constexpr int TC_WARPS = TC_FOLD0 + TC_FOLD;
constexpr int TC_THREADS = 32 * TC_WARPS;
static_assert(TC_FOLD0 % 4 == 0, "a fold warp owns the tensor-memory lanes of warp id % 4");
constexpr int TC_SLABS = 17;     // slabs in rotation
constexpr int TC_HS = 6;         // slabs of an FP32 accumulation (half a group)
constexpr int TC_GS = TC_MMA * TC_HS;  // slabs of a group: one accumulation per MMA warp
constexpr int TC_ACC = 3;        // accumulator pairs in rotation
constexpr int TC_ACOLS = TC_MMA * TC_TS;  // columns of a pair
constexpr int TC_SLOTS = 16;     // group-scale slots in rotation
constexpr int TC_UNITS = 4;      // work units in the ring
constexpr int TC_SB = 14;        // the column weights' scale exponent
constexpr uint32_t TC_COLS = 512;
constexpr uint32_t COL_HI = TC_ACC * TC_ACOLS, COL_LO = COL_HI + TC_TS;
static_assert(COL_LO + TC_TS <= TC_COLS, "tensor memory");
constexpr uint32_t TC_IDESC = bptc::idesc_f16(128, TC_TS) | bptc::IDESC_A_MN | bptc::IDESC_B_MN;
constexpr float KT = BP_KT;
constexpr float KS = BP_KS;
constexpr float NGP_IH = 1.0e38f;  // 1/h of a particle with h = 0
constexpr float FAR = -1.0e6f;     // tile position of an empty slot
#ifndef TC_SLEEP_NS
#define TC_SLEEP_NS 20000  // a waiting warp sleeps (it wakes when the phase completes)
#endif

// One warp's operands of 16 particles, MN-major: a row is the 64 cells of one particle (128
// bytes of FP16, 16-byte chunk c of particle k at chunk c ^ (k % 8)), 8 particles make a
// 1024-byte atom.  A has two 64-row blocks (y, then b) 2048 bytes apart.
struct alignas(1024) TcSlab {
  unsigned char a_hi[4096];
  unsigned char a_lo[4096];
  unsigned char b_hi[2048];
  unsigned char b_lo[2048];
};

// Fields of one particle (derived by the owning warp at the start of a batch).
struct TcField {
  float4 pos[2];  // per axis: minus the particle's pixel relative to the tile (twice, a packed
                  // pair) and minus its fraction (twice)
  float4 k;       // KT / h, KS / h, Y, B
  float2 e64;     // edge value at 64 (x, y)
  float2 pad;
};

// A work unit as the fetching warp leaves it in the ring; len < 0: no more units.
struct TcUnit {
  int64_t begin;
  int len, tile, slot, pad;
};

struct TcSmem {
  TcSlab slab[TC_SLABS];
  TcField fld[TC_PROD][TC_PW];   // fields of each producer warp's slab
  float2 wmax[TC_SLOTS][TC_GS];  // per group slot and slab: the largest |Y|, |B|
  TcUnit unit[TC_UNITS];
  uint64_t full[TC_SLABS];    // per slab: its warp wrote the operands
  uint64_t empty[TC_SLABS];   // per slab: its MMAs completed (tcgen05.commit)
  uint64_t accf[TC_ACC];      // per accumulator: its group's MMAs completed
  uint64_t acce[TC_ACC];      // per accumulator: the fold warps took its group
  uint64_t gready[TC_SLOTS];  // per group slot: the maxima of every slab are published
  uint64_t ufull[TC_UNITS], uempty[TC_UNITS];  // unit written / read by every other warp
  uint64_t fin;               // every MMA of the CTA completed
  uint32_t issued[TC_MMA];    // groups whose halves each MMA warp issued
  uint32_t state[TC_SLABS];   // per slab: 2 x the times it was filled, + 1: its y rows are zero
  uint32_t tmem;
  int abort;
};

static_assert(sizeof(TcSmem) + 1024 <= 232448, "deposit shared memory");

// Test and limit settings of the bounded waits.
struct TcWaitCfg {
  uint32_t polls;
  uint64_t ns;
  const int* stall_flag;  // non-null: every warp first waits on this flag (nothing sets it)
  uint32_t stall_polls;
};

// Edge value in the split representation (bp_edge_split).
__device__ __forceinline__ float edge_split(float dx, float k1, float k2) {
  return bp_edge_split(dx, k1, k2);
}

// 2^e as an FP32 value, -126 <= e <= 127
__device__ __forceinline__ float exp2i(int e) { return __int_as_float((e + 127) << 23); }

// Scale exponent of a group whose largest magnitude is m: m 2^s in [2^14, 2^15) (m normal),
// 0 for m = 0 or NaN; s <= 100 (a subnormal m is taken as 2^-126).
__device__ __forceinline__ int group_exp(float m) {
  if (!(m > 0.f)) return 0;
  const int e = ((__float_as_int(m) >> 23) & 0xff) - 127;
  return min(14 - max(e, -126), 100);
}

// x, y (|x|, |y| < 2^15) as FP16 heads and the FP16 roundings of their exact rests, packed in
// pairs (x in the low half)
__device__ __forceinline__ void split_f16x2(float x, float y, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 hf = __half22float2(h);
  const __half2 t = __floats2half2_rn(__fsub_rn(x, hf.x), __fsub_rn(y, hf.y));
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&t);
}

// The values of four cells (e: cells 0 and 2, o: cells 1 and 3) times s, split and stored as 8
// bytes of the head and tail rows
__device__ __forceinline__ void split_store4(unsigned char* hi, unsigned char* lo, int off,
                                             float2 e, float2 o, float s) {
  const float2 ss = make_float2(s, s);
  e = bptc::mul2(e, ss);
  o = bptc::mul2(o, ss);
  const __half2 h0 = __floats2half2_rn(e.x, o.x), h1 = __floats2half2_rn(e.y, o.y);
  const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
  const float2 te = bptc::sub2(e, make_float2(f0.x, f1.x));
  const float2 to = bptc::sub2(o, make_float2(f0.y, f1.y));
  const __half2 l0 = __floats2half2_rn(te.x, to.x), l1 = __floats2half2_rn(te.y, to.y);
  *reinterpret_cast<uint2*>(hi + off) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0),
                                                   *reinterpret_cast<const uint32_t*>(&h1));
  *reinterpret_cast<uint2*>(lo + off) = make_uint2(*reinterpret_cast<const uint32_t*>(&l0),
                                                   *reinterpret_cast<const uint32_t*>(&l1));
}

// Two edge values (bp_edge_split of each, the unclipped steps on packed pairs) at edges L (tile
// coordinates, integers), pos = (-pixel, -pixel, -fraction, -fraction).
__device__ __forceinline__ float2 edge2(float2 L, float4 pos, float k1, float k2) {
  const float2 d = bptc::add2(bptc::add2(L, make_float2(pos.x, pos.y)), make_float2(pos.z, pos.w));
  const float2 t = make_float2(__saturatef(fmaf(-k1, fabsf(d.x), KT)),
                               __saturatef(fmaf(-k1, fabsf(d.y), KT)));
  const float2 s = make_float2(__saturatef(fmaf(-k2, fabsf(d.x), 0.5f * KS)),
                               __saturatef(fmaf(-k2, fabsf(d.y), 0.5f * KS)));
  const float2 A = bptc::mul2(t, t), B = bptc::mul2(s, s);
  const float2 C = bptc::mul2(B, B);
  const float2 v = bptc::fma2(A, A, make_float2(-C.x, -C.y));
  constexpr int SG = (int)0x80000000;
  return make_float2(__int_as_float(__float_as_int(v.x) ^ (~__float_as_int(d.x) & SG)),
                     __int_as_float(__float_as_int(v.y) ^ (~__float_as_int(d.y) & SG)));
}

// The edge differences of cells 4 li .. 4 li + 3 of one axis (li the lane's index in its half
// warp, le = (4 li, 4 li + 2)), as cells (0, 2) and (1, 3): each lane evaluates its four left
// edges and takes edge 4 li + 4 from its neighbour (the last lane: the particle's stored edge
// 64).  The cell holding the centre is one short here (its weight is written by the centre
// pass).
__device__ __forceinline__ void axis_diffs(int li, float2 le, float2 lo_, float4 pos, float k1,
                                           float k2, float e64, float2& e, float2& o) {
  const float2 ve = edge2(le, pos, k1, k2);   // edges 0 and 2
  const float2 vo = edge2(lo_, pos, k1, k2);  // edges 1 and 3
  const float t = __shfl_down_sync(0xffffffffu, ve.x, 1, 16);
  const float n = li < 15 ? t : e64;
  e = bptc::sub2(vo, ve);
  o = make_float2(ve.y - vo.x, n - vo.y);
}

__global__ void __launch_bounds__(TC_THREADS, 1)
    k_deposit_tc(const float4* __restrict__ rec, const uint32_t* __restrict__ pvals,
                 const BpUnit* __restrict__ units, const int64_t* __restrict__ n_units_ptr,
                 int64_t* counter, int nx, int ny, int ntx, float* ymap, float* bmap,
                 float* ylo, float* blo, float* partials, int* err, TcWaitCfg wc) {
  using namespace bptc;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment by pointer arithmetic on the shared array (keeps shared accesses)
  TcSmem& S = *reinterpret_cast<TcSmem*>(smem_raw +
                                         ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (w == 0) {
    tmem_alloc(&S.tmem, TC_COLS);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int q = 0; q < TC_SLABS; ++q) {
      mbar_init(&S.full[q], 1);
      mbar_init(&S.empty[q], 1);
      S.state[q] = 0u;
    }
    for (int q = 0; q < TC_ACC; ++q) {
      mbar_init(&S.accf[q], TC_MMA);
      mbar_init(&S.acce[q], TC_FOLD);
    }
    for (int q = 0; q < TC_UNITS; ++q) {
      mbar_init(&S.ufull[q], 1);
      mbar_init(&S.uempty[q], TC_WARPS);
    }
    for (int q = 0; q < TC_SLOTS; ++q) mbar_init(&S.gready[q], TC_GS);
    mbar_init(&S.fin, TC_MMA);
    fence_mbar_init();
    S.issued[0] = S.issued[1] = 0u;
    S.abort = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = S.tmem;
  auto fail = [&]() {
    *reinterpret_cast<volatile int*>(&S.abort) = 1;
    if (lane == 0) atomicExch(err, 1);
  };
  // test hook: a bounded wait on a flag that nothing sets, before any MMA is issued
  if (wc.stall_flag) {
    bool ok = false;
    for (uint32_t it = 0; it < wc.stall_polls && !ok; ++it)
      ok = *reinterpret_cast<const volatile int*>(wc.stall_flag) != 0;
    if (!__all_sync(0xffffffffu, ok)) fail();
  }
  __syncthreads();
  // bounded wait on an mbarrier phase, warp-collective; false (and the CTA aborts) on a timeout
  // or when another warp aborted
  auto wait_bar = [&](uint64_t* bar, uint32_t parity) -> bool {
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) {
      const uint64_t t0 = global_ns();
      for (uint32_t it = 1; it < wc.polls && !ok; ++it) {
        ok = mbar_try_wait_sleep(bar, parity, TC_SLEEP_NS);
        if (!ok && (*reinterpret_cast<volatile int*>(&S.abort) ||
                    ((it & 7) == 0 && global_ns() - t0 > wc.ns)))
          break;
      }
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) fail();
    return ok;
  };
  // unit uu of this CTA (every warp but the fetching one reads the ring in order); false at the
  // end or on an abort
  auto next_unit = [&](uint32_t uu, TcUnit& U) -> bool {
    const int ub = (int)(uu % TC_UNITS);
    if (!wait_bar(&S.ufull[ub], (uu / TC_UNITS) & 1)) return false;
    U = S.unit[ub];
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.uempty[ub]);
    return U.len >= 0;
  };
  const bool start_ok = *reinterpret_cast<volatile int*>(&S.abort) == 0;

  if (w >= TC_PROD && w < TC_FOLD0) {
    // ---------------------------------------------------------------- MMA warps
    // Issues each slab's three MMAs (K = 16) in slab order, so that every accumulator sums its
    // particles in a fixed order.  One thread runs the whole loop: its instructions are the
    // serial chain that every slab passes through, so there are as few as possible, and the two
    // MMA warps take the two halves of each group, with an accumulator each.
    if (lane == 0 && start_ok) {
      auto wait1 = [&](uint64_t* bar, uint32_t parity) -> bool {
        if (mbar_try_wait(bar, parity)) return true;
        const uint64_t t0 = global_ns();
        for (uint32_t it = 1; it < wc.polls; ++it) {
          if (mbar_try_wait_sleep(bar, parity, TC_SLEEP_NS)) return true;
          if (*reinterpret_cast<volatile int*>(&S.abort) ||
              ((it & 7) == 0 && global_ns() - t0 > wc.ns))
            break;
        }
        *reinterpret_cast<volatile int*>(&S.abort) = 1;
        atomicExch(err, 1);
        return false;
      };
      const uint64_t dah0 = desc_mn128(smem_u32(S.slab[0].a_hi), 2048);
      constexpr uint64_t AL = sizeof(S.slab[0].a_hi) >> 4;  // to a_lo, in descriptor units
      constexpr uint64_t BH = 2 * AL, BL = BH + (sizeof(S.slab[0].b_hi) >> 4);  // b_hi, b_lo
      uint32_t slot = 0, use = 0;  // the next slab's place in the rotation
      uint32_t acc = 0, ause = 0;  // the next group's accumulator
      const int m = w - TC_PROD;  // this warp takes half m of every group
      uint32_t groups = 0;        // groups so far
      // before this warp's half of group n: the other warp issued its halves of the groups
      // before n - 1 (m = 0) or n (m = 1)
      auto wait_issued = [&](uint32_t n) -> bool {
        const uint32_t need = n + m < 1 ? 0 : n + m - 1;
        const volatile uint32_t* c = &S.issued[1 - m];
        if (*c >= need) return true;
        const uint64_t t0 = global_ns();
        for (uint32_t it = 1; *c < need; ++it) {
          __nanosleep(50);
          if (it >= wc.polls || *reinterpret_cast<volatile int*>(&S.abort) ||
              ((it & 63) == 0 && global_ns() - t0 > wc.ns)) {
            *reinterpret_cast<volatile int*>(&S.abort) = 1;
            atomicExch(err, 1);
            return false;
          }
        }
        return true;
      };
      for (uint32_t uu = 0;; ++uu) {
        const int ub = (int)(uu % TC_UNITS);
        if (!wait1(&S.ufull[ub], (uu / TC_UNITS) & 1)) break;
        const int len = S.unit[ub].len;
        mbar_arrive(&S.uempty[ub]);
        if (len < 0) break;
        bool go = true;
        int left = (len + TC_PW - 1) / TC_PW;
        while (left > 0 && go) {  // one group
          // the slabs before this warp's half, of the half, and after it
          const int n0 = min(left, m * TC_HS), n = min(left - n0, TC_HS);
          const int n2 = min(left - n0 - n, TC_GS - n0 - n);
          left -= n0 + n + n2;
          slot += (uint32_t)n0;
          if (slot >= TC_SLABS) {
            slot -= TC_SLABS;
            ++use;
          }
          // the other warp's halves before the last one are issued: every slab of this half has
          // then been filled as often as its place in the rotation says, and the parity wait
          // below cannot mistake an older phase for it
          go = wait_issued(groups) && (ause == 0 || wait1(&S.acce[acc], (ause - 1) & 1));
          const uint32_t dt = tm + acc * TC_ACOLS + (uint32_t)(m * TC_TS);
          for (int k = 0; k < n && go; ++k) {
            go = wait1(&S.full[slot], use & 1);
            if (!go) break;
            tc_fence_after();
            const uint64_t da = dah0 + (uint64_t)(slot * (uint32_t)(sizeof(TcSlab) >> 4));
            mma_f16(dt, da, da + BH, TC_IDESC, k > 0 ? 1u : 0u);
            mma_f16(dt, da, da + BL, TC_IDESC, 1u);
            mma_f16(dt, da + AL, da + BH, TC_IDESC, 1u);
            mma_commit(&S.empty[slot]);
            if (++slot == TC_SLABS) {
              slot = 0;
              ++use;
            }
          }
          if (go) mma_commit(&S.accf[acc]);  // an empty half: once the MMAs before are done
          slot += (uint32_t)n2;
          if (slot >= TC_SLABS) {
            slot -= TC_SLABS;
            ++use;
          }
          ++groups;
          *reinterpret_cast<volatile uint32_t*>(&S.issued[m]) = groups;
          if (++acc == TC_ACC) {
            acc = 0;
            ++ause;
          }
        }
        if (!go) break;
      }
    }
    __syncwarp();
    // every issued MMA must finish (bounded) before the tensor memory is released
    if (lane == 0) mma_commit(&S.fin);
    __syncwarp();
    mbar_wait_bounded_sleep(&S.fin, 0, wc.polls, wc.ns, TC_SLEEP_NS);
  } else if (w >= TC_FOLD0) {
    // ---------------------------------------------------------------- fold warps
    // Warp q of the four owns tensor-memory lanes 32 q .. + 31 (rows of y for q < 2, of b
    // above): it folds every finished group into the (sum, compensation) pair and writes the
    // finished tile out.  The first one also fetches the units, two ahead.
    const int q = w & 3;
    const uint32_t lanes = tm + ((uint32_t)(32 * q) << 16);
    const int64_t n_units = *n_units_ptr;
    uint32_t uc = 0;  // units fetched
    bool done = false;
    auto fetch = [&]() -> bool {
      const int ub = (int)(uc % TC_UNITS);
      if (done) return true;
      if (uc >= TC_UNITS && !wait_bar(&S.uempty[ub], ((uc / TC_UNITS) - 1) & 1)) return false;
      int64_t u = 0;
      if (lane == 0) u = (int64_t)atomicAdd((unsigned long long*)counter, 1ull);
      u = __shfl_sync(0xffffffffu, u, 0);
      TcUnit U = {0, -1, 0, 0, 0};
      if (u < n_units) {
        const BpUnit B = units[u];
        U.begin = B.begin;
        U.len = (int)(B.end - B.begin);  // a unit holds at most 2^30 pairs
        U.tile = B.tile;
        U.slot = B.slot;
      } else {
        done = true;
      }
      if (lane == 0) {
        S.unit[ub] = U;
        mbar_arrive(&S.ufull[ub]);
      }
      __syncwarp();
      ++uc;
      return true;
    };
    const bool fetcher = w == TC_FOLD0;
    bool go = start_ok && (!fetcher || (fetch() && fetch()));
    uint32_t g = 0, acc = 0, ause = 0;  // the next group
    TcUnit U;
    for (uint32_t uu = 0; go && next_unit(uu, U); ++uu) {
      if (fetcher && !fetch()) break;
      const int ns = (U.len + TC_PW - 1) / TC_PW;
      for (int i = 0; i < ns; i += TC_GS, ++g) {
        if (!wait_bar(&S.accf[acc], ause & 1)) {
          go = false;
          break;
        }
        tc_fence_after();
        // the group's scale for these rows, undone: exact (a power of two)
        float m = 0.f;
        const int nv = min(TC_GS, ns - i);
        for (int k = 0; k < nv; ++k) {
          const float2 v = S.wmax[g % TC_SLOTS][k];
          m = fmaxf(m, q < 2 ? v.x : v.y);
        }
        const float us = exp2i(-group_exp(m) - TC_SB);
        const float2 us2 = make_float2(us, us);
        const uint32_t dcol = acc * TC_ACOLS;
        const bool two = nv > TC_HS;  // the second half holds slabs
        const bool first = i == 0;
#pragma unroll 1
        for (int h = 0; h < TC_TS; h += 16) {
          float x[16], x1[16], hi[16], lo[16];
          tmem_ld16(lanes + dcol + h, x);
          if (two) {
            tmem_ld16(lanes + dcol + TC_TS + h, x1);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) x1[j] = 0.f;
          }
          if (!first) {
            tmem_ld16(lanes + COL_HI + h, hi);
            tmem_ld16(lanes + COL_LO + h, lo);
          }
          tmem_wait_ld();
          if (first) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              hi[j] = __fmul_rn(__fadd_rn(x[j], x1[j]), us);
              lo[j] = 0.f;
            }
          } else {  // Kahan's summation
#pragma unroll
            for (int j = 0; j < 16; j += 2) {
              const float2 h2 = make_float2(hi[j], hi[j + 1]);
              // v us is exact: the fused form rounds once, like the sum
              const float2 v = add2(make_float2(x[j], x[j + 1]), make_float2(x1[j], x1[j + 1]));
              const float2 y = fma2(v, us2, make_float2(lo[j], lo[j + 1]));
              const float2 t = add2(h2, y);
              const float2 l2 = sub2(y, sub2(t, h2));
              hi[j] = t.x;
              hi[j + 1] = t.y;
              lo[j] = l2.x;
              lo[j + 1] = l2.y;
            }
          }
          tmem_st16(lanes + COL_HI + h, hi);
          tmem_st16(lanes + COL_LO + h, lo);
        }
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.acce[acc]);
        if (++acc == TC_ACC) {
          acc = 0;
          ++ause;
        }
      }
      if (!go) break;
      // the tile's rows 32 q .. + 31 of y or b: into the map, or as a partial tile
      const int x0 = (U.tile % ntx) * TC_TS, y0 = (U.tile / ntx) * TC_TS;
      const int r = 32 * q + lane;
      const bool is_b = r >= TC_TS;
      const int jr = r & (TC_TS - 1);
      // Eight pixels of the map and of its compensation at a time, so that their loads overlap:
      // pixel by pixel (a store may alias the next pixel's load) a tile took 60 us, which is what
      // a map of few particles costs.  1e5 particles on 4096^2 pixels: 0.62 ms (1.67 ms; two CTAs
      // per SM of eight warps, all of them writing, 1.33 ms), 2e7: 2.4 ms (3.3 ms).
#pragma unroll 1
      for (int h = 0; h < TC_TS; h += 8) {
        float hi[8], lo[8];
        tmem_ld8(lanes + COL_HI + h, hi);
        tmem_ld8(lanes + COL_LO + h, lo);
        tmem_wait_ld();
        if (U.slot < 0) {
          const int gy = y0 + jr, left = nx - (x0 + h);  // columns of the map from here on
          if (gy < ny) {
            float* map = is_b ? bmap : ymap;
            float* mlo = is_b ? blo : ylo;
            const int64_t p0 = (int64_t)gy * nx + x0 + h;
            float m[8], l[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              m[j] = j < left ? map[p0 + j] : 0.f;
              l[j] = j < left ? mlo[p0 + j] : 0.f;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (j >= left) continue;
              const int64_t p = p0 + j;
              if (!BP_DCHECK(p >= 0 && p < (int64_t)nx * ny, err + BP_DBG_SLOT, 401)) continue;
              float sm, e;
              bp_two_sum(m[j], hi[j], sm, e);
              map[p] = sm;
              mlo[p] = l[j] + (lo[j] + e);
            }
          }
        } else {
          if (!BP_DCHECK(jr * TC_TS + h + 8 <= TC_TS * TC_TS, err + BP_DBG_SLOT, 402)) continue;
          float* P = partials + (int64_t)U.slot * 4 * TC_TS * TC_TS +
                     (is_b ? 2 : 0) * TC_TS * TC_TS + jr * TC_TS + h;
#pragma unroll
          for (int j = 0; j < 8; j += 4) {
            *reinterpret_cast<float4*>(P + j) = make_float4(hi[j], hi[j + 1], hi[j + 2], hi[j + 3]);
            *reinterpret_cast<float4*>(P + TC_TS * TC_TS + j) =
                make_float4(lo[j], lo[j + 1], lo[j + 2], lo[j + 3]);
          }
        }
      }
    }
  } else if (start_ok) {
    // ---------------------------------------------------------------- producer warps
    // Warp w fills the slabs whose number (counted over the CTA's units) is w modulo TC_PROD.
    const int li = lane & 15, hw = lane >> 4;
    const float2 le = make_float2((float)(4 * li), (float)(4 * li + 2));
    const float2 lo2 = make_float2((float)(4 * li + 1), (float)(4 * li + 3));
    // byte offset of this lane's 8 bytes in particle row hw; rows 2 q + hw: XOR of the chunk
    // bits with 2 q % 8, plus the row and atom offsets
    const int off0 = (((li >> 1) ^ hw) << 4) + (li & 1) * 8;
    constexpr float sw = (float)(1 << TC_SB);
    uint32_t s0 = 0, g0 = 0;  // slabs and groups of the units before
    // bounded wait until slab `slot` was filled `use` times: its last but one use is then
    // consumed, so that the parity wait on the last one cannot mistake an older phase for it
    auto wait_filled = [&](uint32_t slot, uint32_t use) -> bool {
      bool ok = true;
      const volatile uint32_t* st = &S.state[slot];
      if ((*st >> 1) < use) {
        const uint64_t t0 = global_ns();
        for (uint32_t it = 1; (*st >> 1) < use; ++it) {
          __nanosleep(100);
          if (it >= wc.polls || *reinterpret_cast<volatile int*>(&S.abort) ||
              ((it & 63) == 0 && global_ns() - t0 > wc.ns)) {
            ok = false;
            break;
          }
        }
      }
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) fail();
      return ok;
    };
    bool ok = true;
    TcUnit U;
    for (uint32_t uu = 0; ok && next_unit(uu, U); ++uu) {
      const int x0 = (U.tile % ntx) * TC_TS, y0 = (U.tile / ntx) * TC_TS;
      const int len = U.len;
      const int ns = (len + TC_PW - 1) / TC_PW;
      const uint32_t* uvals = pvals + U.begin;
      // publishes the largest |Y| and |B| of slab i (lane: |Y| of particle li in the lower half
      // warp, |B| in the upper); the last slab arrives for the missing ones of its group
      auto publish = [&](int i, float4 r) {
        float m = fabsf(hw ? r.x : r.w);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        const uint32_t gs = (g0 + (uint32_t)(i / TC_GS)) % TC_SLOTS;
        float* dst = &S.wmax[gs][i % TC_GS].x;
        if (li == 0) dst[hw] = m;
        __syncwarp();
        if (lane == 0)
          mbar_arrive_n(&S.gready[gs], i + 1 == ns ? (uint32_t)(TC_GS - i % TC_GS) : 1u);
      };
      int i = (int)((w + TC_PROD - s0 % TC_PROD) % TC_PROD);
      uint32_t seq = s0 + (uint32_t)i, slot = seq % TC_SLABS, use = seq / TC_SLABS;
      // half record hw of particle li of the slab: this slab's (r0) and the next one's (r1), and
      // the particle index of the one after
      const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
      constexpr int STEP = TC_PW * TC_PROD;
      float4 r0 = zero4, r1 = zero4;
      uint32_t pv = 0;
      {
        const int q = TC_PW * i + li;
        const uint32_t pa = q < len ? uvals[q] : 0u;
        const uint32_t pb = q + STEP < len ? uvals[q + STEP] : 0u;
        if (q + 2 * STEP < len) pv = uvals[q + 2 * STEP];
        if (q < len) r0 = rec[2 * (int64_t)pa + hw];
        if (q + STEP < len) r1 = rec[2 * (int64_t)pb + hw];
      }
      if (i < ns) publish(i, r0);
      for (; i < ns && ok; i += TC_PROD) {
        const int q = TC_PW * i + li;
        // 1. the slab's fields, one (particle, axis) per lane: particle li, axis hw
        float4 a = make_float4(FAR, 0.5f, KT, KS);  // empty slot: far outside the tile
        int kc = -(1 << 30);
        float sig = 0.f;  // Y (lower half warp) or B (upper) of the lane's particle
        {
          // lower half: fx, fy, hp, Y; upper half: B, kind, ix, iy
          const float other = __shfl_xor_sync(0xffffffffu, hw ? r0.z : r0.y, 16);
          const float hp = __shfl_sync(0xffffffffu, r0.z, li);
          float e64 = 0.f;
          if (q < len) {
            float f = hw ? other : r0.x;
            const int pr = __float_as_int(hw ? r0.w : other) - (hw ? y0 : x0);
            const bool ngp = !(hp > 0.f);
            const float ih = ngp ? NGP_IH : __frcp_rn(hp);
            if (ngp && !(f > 0.f)) f = 1.0e-30f;  // exactly on an edge: the cell to its right
            a = make_float4((float)pr, f, KT * ih, KS * ih);
            kc = pr + (f > 0.f ? 0 : -1);
            e64 = edge_split(__fsub_rn(__fsub_rn((float)TC_TS, a.x), a.y), a.z, a.w);
            sig = hw ? r0.x : r0.w;
          }
          TcField& F = S.fld[w][li];
          F.pos[hw] = make_float4(-a.x, -a.x, -a.y, -a.y);
          if (hw == 0) *reinterpret_cast<float2*>(&F.k) = make_float2(a.z, a.w);
          (&F.k.z)[hw] = sig;
          (&F.e64.x)[hw] = e64;
        }
        const bool has_y = __any_sync(0xffffffffu, !hw && sig != 0.f);
        // 2. the next slab's maxima, and the records of the one after on their way
        if (i + TC_PROD < ns) publish(i + TC_PROD, r1);
        r0 = r1;
        r1 = zero4;
        {
          const int qn = q + 2 * STEP;
          if (qn < len) r1 = rec[2 * (int64_t)pv + hw];
          if (qn + STEP < len) pv = uvals[qn + STEP];
        }
        __syncwarp();
        // 3. four rounds of four particles, two at a time (one per half warp): the edge
        // differences in registers; before the first store the group's scales, once all its
        // slabs' maxima are published, and the slab, free once the MMAs of its last use are
        // done; then scaled, split and stored.  A rolled loop: the unrolled body overflowed
        // the instruction cache.
        TcSlab& T = S.slab[slot];
        float sy = 1.f, sb = 1.f;
#pragma unroll 1
        for (int qq = 0; qq < 4; ++qq) {
          float2 xe[2], xo[2], ye[2], yo[2];  // column and row differences
          float Yk[2], Bk[2];
#pragma unroll
          for (int t = 0; t < 2; ++t) {  // particle 4 qq + 2 t + hw
            const TcField& F = S.fld[w][4 * qq + 2 * t + hw];
            const float4 k = F.k;
            const float2 e64 = F.e64;
            axis_diffs(li, le, lo2, F.pos[0], k.x, k.y, e64.x, xe[t], xo[t]);
            axis_diffs(li, le, lo2, F.pos[1], k.x, k.y, e64.y, ye[t], yo[t]);
            Yk[t] = k.z;
            Bk[t] = k.w;
          }
          if (qq == 0) {
            const uint32_t g = g0 + (uint32_t)(i / TC_GS);
            ok = wait_bar(&S.gready[g % TC_SLOTS], (g / TC_SLOTS) & 1) &&
                 (use == 0 || (wait_filled(slot, use) && wait_bar(&S.empty[slot], (use - 1) & 1)));
            if (!ok) break;
            // slabs past the unit's end have no maxima
            const int nv = min(TC_GS, ns - i / TC_GS * TC_GS);
            float2 v = S.wmax[g % TC_SLOTS][min(li, nv - 1)];
            static_assert(TC_GS <= 16, "one lane of sixteen per slab of the group");
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
              v.x = fmaxf(v.x, __shfl_xor_sync(0xffffffffu, v.x, o));
              v.y = fmaxf(v.y, __shfl_xor_sync(0xffffffffu, v.y, o));
            }
            sy = exp2i(group_exp(v.x));
            sb = exp2i(group_exp(v.y));
            const bool yz = *reinterpret_cast<volatile uint32_t*>(&S.state[slot]) & 1u;
            if (!has_y && !yz) {  // 16 particles without y after some with: zero rows once
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                *reinterpret_cast<uint4*>(T.a_hi + 16 * (16 * j + li) + hw * (int)sizeof(T.a_hi)) =
                    make_uint4(0, 0, 0, 0);
              }
            }
            __syncwarp();
          }
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            // rows k = 4 qq + 2 t (+ hw): chunk bits XOR k % 8, row and atom offsets
            const int off = (off0 ^ ((((qq & 1) * 4 + 2 * t) << 4))) +
                            ((qq & 1) * 4 + 2 * t + hw) * 128 + (qq >> 1) * 1024;
            split_store4(T.b_hi, T.b_lo, off, xe[t], xo[t], sw);
            split_store4(T.a_hi + 2048, T.a_lo + 2048, off, ye[t], yo[t], __fmul_rn(Bk[t], sb));
            if (has_y) split_store4(T.a_hi, T.a_lo, off, ye[t], yo[t], __fmul_rn(Yk[t], sy));
          }
        }
        if (!ok) break;
        __syncwarp();
        // 4. the centre pass: lane (particle li, axis hw) writes the whole weight of the cell
        // holding its centre over the edge difference stored above
        if (kc >= 0 && kc < TC_TS) {
          const float v0 = edge_split(__fsub_rn(__fsub_rn((float)kc, a.x), a.y), a.z, a.w);
          const float v1 = edge_split(__fsub_rn(__fsub_rn((float)(kc + 1), a.x), a.y), a.z, a.w);
          const float wc0 = (v1 - v0) + 1.f;
          const int off = (li >> 3) * 1024 + (li & 7) * 128 + (((kc >> 3) ^ (li & 7)) << 4) +
                          (kc & 7) * 2;
          uint32_t h, l;
          if (hw == 0) {
            split_f16x2(__fmul_rn(wc0, sw), 0.f, h, l);
            *reinterpret_cast<unsigned short*>(T.b_hi + off) = (unsigned short)h;
            *reinterpret_cast<unsigned short*>(T.b_lo + off) = (unsigned short)l;
          } else {
            const float Yc = S.fld[w][li].k.z;
            split_f16x2(__fmul_rn(wc0, __fmul_rn(sig, sb)), __fmul_rn(wc0, __fmul_rn(Yc, sy)), h,
                        l);
            *reinterpret_cast<unsigned short*>(T.a_hi + 2048 + off) = (unsigned short)h;
            *reinterpret_cast<unsigned short*>(T.a_lo + 2048 + off) = (unsigned short)l;
            if (has_y) {
              *reinterpret_cast<unsigned short*>(T.a_hi + off) = (unsigned short)(h >> 16);
              *reinterpret_cast<unsigned short*>(T.a_lo + off) = (unsigned short)(l >> 16);
            }
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          *reinterpret_cast<volatile uint32_t*>(&S.state[slot]) =
              (uint32_t)(((use + 1) << 1) | (has_y ? 0u : 1u));
          mbar_arrive(&S.full[slot]);
        }
        slot += TC_PROD - TC_SLABS;
        ++use;
        if (slot >= TC_SLABS) {
          slot -= TC_SLABS;
          ++use;
        }
      }
      s0 += (uint32_t)ns;
      g0 += (uint32_t)((ns + TC_GS - 1) / TC_GS);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (w == 0) tmem_dealloc(tm, TC_COLS);
}

}  // namespace

// Launches the tensor-core deposit over the work units; the tile side is 64.  One CTA per SM
// (its shared memory and all tensor-memory columns), capped by max_units.  Sets the context's
// device flag 0 on a timed-out wait.
int bp_deposit_tc_launch(bp_ctx* ctx, const float* assigned, const uint32_t* vals,
                         const BpUnit* units, const int64_t* n_units_dev, int64_t* counter,
                         int64_t max_units, const bp_map_geom* g, float* ymap, float* bmap,
                         float* ylo, float* blo, float* partials) {
  const int ntx = (g->nx + TC_TS - 1) / TC_TS;
  const size_t smem = sizeof(TcSmem) + 1024;
  BP_CUDA(ctx, cudaFuncSetAttribute(k_deposit_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem));
  int64_t grid = ctx->num_sms;
  if (grid > max_units) grid = max_units;
  if (grid < 1) grid = 1;
  TcWaitCfg wc;
  wc.polls = 1u << 26;
  wc.ns = 2000000000ull;  // 2 s
  wc.stall_flag = nullptr;
  wc.stall_polls = 0;
  if (ctx->test_stall_polls > 0) {  // test of the timeout path: flag 2 is zero and stays zero
    BP_CUDA(ctx, cudaMemsetAsync(ctx->d_flags + 2, 0, sizeof(int), ctx->stream));
    wc.stall_flag = ctx->d_flags + 2;
    wc.stall_polls = (uint32_t)ctx->test_stall_polls;
  }
  BP_CUDA(ctx, cudaMemsetAsync(ctx->d_flags, 0, sizeof(int), ctx->stream));
  k_deposit_tc<<<(unsigned)grid, TC_THREADS, smem, ctx->stream>>>(
      reinterpret_cast<const float4*>(assigned), vals, units, n_units_dev, counter, g->nx, g->ny,
      ntx, ymap, bmap, ylo, blo, partials, ctx->d_flags, wc);
  BP_LAUNCH_CHECK(ctx, "deposit (tensor cores)");
  return BP_OK;
}

// Reads the device flag the tensor-core deposit sets on a timed-out wait (synchronises
// the context's stream).
int bp_deposit_tc_check(bp_ctx* ctx) {
  int* h = reinterpret_cast<int*>(ctx->h_pinned + 3);
  BP_CUDA(ctx, cudaMemcpyAsync(h, ctx->d_flags, sizeof(int), cudaMemcpyDeviceToHost,
                               ctx->stream));
  BP_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  if (*h) return bp_fail(ctx, BP_ETIMEOUT, "deposit: a tensor-core wait timed out");
  return BP_OK;
}

// Loads the tensor-core deposit kernel (CUDA loads modules lazily: its first launch would
// otherwise load its code into device memory).
int bp_deposit_tc_preload(bp_ctx* ctx) {
  cudaFuncAttributes a;
  BP_CUDA(ctx, cudaFuncGetAttributes(&a, k_deposit_tc));
  return BP_OK;
}
