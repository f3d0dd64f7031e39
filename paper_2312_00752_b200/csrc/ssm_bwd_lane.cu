// Backward selective scan for everything the tuned bf16 / N = 16 kernel does not take (mathematics as in ssm_bwd.cu:
// adjoint of Eq. 2a/2b with skip term and gate, states recomputed from checkpoints, Section 3.3; inputs, alignment and
// time split as in ssm_lane.cuh).
//
// Main sweep.  A lane holds 8 of 16 states of 2 adjacent channels (local channel q of lane l is channel l ^ q, its states
// are 8 (l & 1) ..), so the sums over n are reduce-scattered with one xor-shuffle and every lane finishes the channel with
// its own number.  Time runs backwards in blocks of 8 steps = one checkpoint: a forward sweep rebuilds the states and keeps
// those after the odd steps in registers, the reverse sweep walks pairs of steps and rebuilds the even one.  dB / dC terms
// are summed over the warp's channels through a transposing pass over shared memory every 4 steps, in a fixed order.
// With N > 16 a team of N / 16 warps shares the rows of a piece, each warp with its own group of 16 states; the three sums
// over n of a step meet in shared memory once per block.
//
// Time split.  As in the forward kernel, over the teams of a block and the blocks of a cluster: a first sweep of the
// lam / mu recurrence alone (a lane per channel) gives the adjoint that leaves every piece, the fold runs from the last
// piece to the first.  That is for little work (one launch); with more, the launch is cut into segments that fill whole
// waves and the first sweep is a kernel of its own at four warps per sub-partition instead of two (plan_lane_bwd).
//
// Bound (counters): latency at two warps per sub-partition (255 registers).  Issue slots 40 to 44 % in use, FMA pipe 31 to
// 46 %, special-function unit 11 to 35 %; per issued instruction a warp waits 1.0 to 1.2 cycles for fixed latencies, 0.6 to
// 0.9 for shared memory and special functions and, a block's body being near the size of the instruction cache, 0.2
// (float32, N = 64) to 0.7 (bf16 rows at odd addresses, complex states) for instructions, hence rolled loops around it;
// 315 warp instructions per warp and step at float32 (2, 2048, 1536).  Measured against the generic
// kernel, backward call: float32 (2, 2048, 1536), N = 16: 485 -> 174 us; bf16 (3, 1237, 1001): 430 -> 125 us; bf16
// (1, 2048, 5120), N = 64: 3003 -> 824 us; float32 (1, 256, 64): 207 -> 14 us.
#include <type_traits>

#include "ssm_lane.cuh"

namespace ssm {

namespace {

namespace cg = cooperative_groups;

constexpr float kLn2 = 0.6931471805599453f;

// Shared memory of a block, in bytes: per team the raw rows and the per-step values of a block of 8 steps; per warp B and
// C of the block, two checkpoints, the transposing buffer (also: tiles of the first sweep, what leaves a piece, dA), the
// sums over n (N > 16); per chain A * log2(e) and the sums of delta
template <typename IO, int NG, bool VEC, bool ROLLED = false>
struct BwdLaneSmem {
  static constexpr int NP = 16 * NG, kTeams = kLaneWarps / NG;
  static constexpr int kPitch = (VEC || sizeof(IO) == 4) ? 32 * (int)sizeof(IO) : 80;   // bytes of a raw row
  static constexpr int kRaw = kLB * kPitch;                   // one tensor
  static constexpr int kTeam = 4 * kRaw + 2 * kLB * 32 * 16;
  static_assert(2 * kLB * 32 * 16 >= NP * 128, "the totals of a chain fit where the per-step values go");
  static constexpr int kRed = 4 * 32 * 4 * 16;
  static constexpr int kWarp = 2 * kLB * 16 * 4 + 2 * 4 * 32 * 16 + kRed + (NG > 1 ? kLB * 32 * 16 : 0) + (ROLLED ? kLB / 2 * 4 * 32 * 16 : 0);
  static constexpr int kChain = NP * 128 + 128 + kTeams * 128;
  static __host__ __device__ constexpr int bytes(int chains) { return kTeams * kTeam + kLaneWarps * kWarp + chains * kChain + kLaneWarps * 256; }
};

__device__ __forceinline__ void cp_async4(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void cp_async16_bytes(void* dst, const void* src, int bytes) {   // (bytes < 16: zero-filled)
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}

// Raw rows: the 32 channels of a block of 8 steps of x, delta, z, dout, copied asynchronously.  Rows that are not 16-byte
// aligned go word by word, the words of the 8 rows dealt out over the lanes; a bf16 row piece that starts at an odd element
// is copied from the word it starts in and read with a shift of one element.  Blocks are 8 rows apart, an even number of
// elements, so what a lane copies of a block is at the same offsets in every block and in all four tensors.  If one of the
// tensors is not even aligned to a word, elements are copied one by one.
enum { kElements = 0, kWords = 1, kVectors = 2 };   // how rows are copied
template <typename IO, int ROWS>
struct RawRows {
  static constexpr bool VEC = ROWS == kVectors;
  static constexpr int kPitch = BwdLaneSmem<IO, 1, VEC>::kPitch;
  static constexpr int kRowWords = sizeof(IO) == 4 ? 32 : 17; // words of a row (not VEC)
  static constexpr int kCopies = VEC ? LaneRows<IO, true>::NV : (kLB * kRowWords + 31) / 32;
  unsigned off[kCopies];   // bytes from the first element of the block's rows (plus 2 if a row may start half a word in)
  unsigned dst[kCopies];   // bytes in the tile | row << 16 (a row past the block: nothing to copy) | half a word << 12
  int shift_even, shift_odd;   // elements by which rows of even / odd number are shifted in the tile
  static constexpr unsigned kBack = VEC ? 0u : 2u;
  // first: element index (in the tensor) of the first row's first channel
  __device__ __forceinline__ int shift(int t) const { return ROWS == kWords && sizeof(IO) == 2 ? ((t & 1) ? shift_odd : shift_even) : 0; }
  __device__ __forceinline__ void setup(size_t first, int D, int lane, int cols) {
    shift_even = (int)(first & 1);
    shift_odd = (int)((first + D) & 1);
    if constexpr (ROWS == kElements) return;
#pragma unroll
    for (int i = 0; i < kCopies; ++i) {
      const int q = lane + 32 * i;
      if constexpr (VEC) {
        using R = LaneRows<IO, true>;
        const int row = q / R::VPR, col = q % R::VPR * R::EPV;
        off[i] = (unsigned)(row * D + col) * (unsigned)sizeof(IO);
        dst[i] = (unsigned)q * 16u | (unsigned)(col < cols ? row : kLB) << 16;
      } else {
        // (the last word of a row piece may be half: what lies behind the row may lie behind the tensor)
        const int row = q / kRowWords, w = q % kRowWords, sh = shift(row), bytes = (cols + sh) * (int)sizeof(IO) - w * 4;
        off[i] = (unsigned)(row * D - sh) * (unsigned)sizeof(IO) + (unsigned)w * 4u + kBack;
        dst[i] = (unsigned)(row * kPitch + w * 4) | (bytes == 2 ? 1u << 12 : 0u) | (unsigned)(bytes > 0 ? row : kLB) << 16;
      }
    }
  }
  __device__ __forceinline__ void issue(unsigned char* tile, const IO* base, int D, int lane, int cols, int live
                                        SSM_DEBUG_ARGS(const IO* tensor, size_t count, int* status)) const {
    if constexpr (ROWS == kElements) {
#pragma unroll 1
      for (int t = 0; t < live; ++t) {
        SSM_GUARD_SPAN(base + (size_t)t * D, cols, tensor, count, status, return)
        if (lane < cols) reinterpret_cast<IO*>(tile + t * kPitch)[lane] = base[(size_t)t * D + lane];
      }
      return;
    }
    const IO* const from = reinterpret_cast<const IO*>(reinterpret_cast<const char*>(base) - kBack);
#pragma unroll
    for (int i = 0; i < kCopies; ++i) {
      if ((int)(dst[i] >> 16) < live) {
        unsigned char* const to = tile + (dst[i] & 0xfffu);
        SSM_GUARD((dst[i] & 0xfffu) + (VEC ? 16 : 4) <= (BwdLaneSmem<IO, 1, VEC>::kRaw), status, continue)
        SSM_GUARD_SPAN(reinterpret_cast<const char*>(at_bytes(from, off[i])), VEC ? 16 : 4 - (int)(dst[i] >> 11 & 2u), tensor,
                       count * sizeof(IO), status, continue)
        if constexpr (VEC) cp_async16(to, at_bytes(from, off[i]), true);
        else cp_async4(to, at_bytes(from, off[i]), 4 - (int)(dst[i] >> 11 & 2u));
      }
    }
  }
  __device__ __forceinline__ float get(const unsigned char* tile, int t, int lane) const {
    using RawT = typename LaneRaw<IO>::T;
    return LaneRaw<IO>::widen(reinterpret_cast<const RawT*>(tile + t * kPitch)[lane + shift(t)]);
  }
};

// Slot of channel `lane` in the 32 results of row t: permuted so that neither the stores (a row of all lanes) nor the
// 16-byte gathers of the flush (8 or 4 channels of a row per lane) hit a bank twice.
__device__ __forceinline__ int out_slot(int t, int c) { return (c & 24) | ((c ^ ((c >> 3) + 4 * (t & 1))) & 7); }

// What a lane carries along a piece: constants of its 16 recurrences, the adjoint, the dA sums.
struct LaneChain {
  float2 A2[2][4], mu[2][4], dA[2][4];   // A2: A * log2(e)
  float Dk, dD, dbias;
};

// the decays of a lane's 8 rows (complex: pairs k and k + 2 are real and imaginary parts, k = 0, 1)
template <bool AP, bool CPLX>
__device__ __forceinline__ void lane_decays(float dt, const float2 (&A2)[4], float2 (&a)[4]) {
  if constexpr (CPLX) {
    cexp_pair(dt, A2[0], A2[2], a[0], a[2]);
    cexp_pair(dt, A2[1], A2[3], a[1], a[3]);
  } else if constexpr (AP) {
    const float a0 = ex2_approx(dt * A2[0].x), r = ex2_approx(dt * (A2[0].y - A2[0].x)), r2 = r * r, r4 = r2 * r2;
    a[0] = make_float2(a0, a0 * r);
    a[1] = f2mul(a[0], f2dup(r2));
    a[2] = f2mul(a[0], f2dup(r4));
    a[3] = f2mul(a[1], f2dup(r4));
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 e = f2mul(f2dup(dt), A2[k]);
      a[k] = make_float2(ex2_approx(e.x), ex2_approx(e.y));
    }
  }
}
// a u + v and a u for the lane's rows, and (conj a) u
template <bool CPLX>
__device__ __forceinline__ void lane_mul_add(const float2 (&a)[4], const float2 (&u)[4], const float2 (&v)[4], float2 (&out)[4]) {
  if constexpr (CPLX) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float2 ur = u[k], ui = u[k + 2];
      out[k] = f2fma(f2neg(a[k + 2]), ui, f2fma(a[k], ur, v[k]));
      out[k + 2] = f2fma(a[k + 2], ur, f2fma(a[k], ui, v[k + 2]));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = f2fma(a[k], u[k], v[k]);
  }
}
template <bool CPLX>
__device__ __forceinline__ void lane_mul_conj(const float2 (&a)[4], const float2 (&u)[4], float2 (&out)[4]) {
  if constexpr (CPLX) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float2 ur = u[k], ui = u[k + 2];
      out[k] = f2fma(a[k + 2], ui, f2mul(a[k], ur));
      out[k + 2] = f2fma(f2neg(a[k + 2]), ur, f2mul(a[k], ui));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = f2mul(a[k], u[k]);
  }
}
// sum over the lane's rows of w A, in units of 1 / ln 2 (A as staged)
template <bool CPLX>
__device__ __forceinline__ float lane_dot_a(const float2 (&w)[4], const float2 (&A2)[4], float2 part) {
  // part: the sum over pairs 0, 1 (real parts) on entry
  if constexpr (CPLX) {
    const float2 im = f2fma(w[3], A2[3], f2mul(w[2], A2[2]));
    return fmaf(im.x + im.y, 1.f / kLn2, part.x + part.y);
  } else {
    const float2 all = f2fma(w[3], A2[3], f2fma(w[2], A2[2], part));
    return all.x + all.y;
  }
}
__device__ __forceinline__ void load8(const float* row, float2 (&v)[4]) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(row + 4 * k);
    v[2 * k] = make_float2(a.x, a.y);
    v[2 * k + 1] = make_float2(a.z, a.w);
  }
}

// Results of one (step, channel) from the three sums over n.  v1 = (dt, dt', u, u'), v2 = (ds, ds', gp, dstep) of the lane.
__device__ __forceinline__ float3 finish_step(LaneChain& lc, float4 v1, float4 v2, float y, float lb, float wa, bool live) {
  const float dx = fmaf(v1.x, lb, v2.x * lc.Dk);
  const float dd = fmaf(v1.z, lb, wa * kLn2) * v2.w;   // (v2.w: derivative of the step size by its pre-activation)
  const float dz = v2.z * fmaf(lc.Dk, v1.z, y);
  lc.dD = fmaf(v2.x, v1.z, lc.dD);
  lc.dbias += live ? dd : 0.f;
  return make_float3(dx, dd, dz);
}

// One block of 8 steps of one group of 16 states.  ROLLED: loops over the steps, states after the odd steps in sh
// [4][vectors as in ck][32] instead of registers.  t1 / t2: per-step values; fB / fC: rows of 16 states; ck: the states
// before the block; part_dB / part_dC: first row of this block in the partial sums (stride N); emit(t, y, lb, wa, v1, v2)
// takes the sums over the 16 states for the lane's own channel.
template <bool AP, bool CPLX, bool ROLLED, typename Emit>
__device__ __forceinline__ void lane_block(LaneChain& lc, const float4* t1, const float4* t2, const float* fB, const float* fC,
                                           const float4* ck, float4* sh, float4* red, float* part_dB, float* part_dC, int N, int n_live,
                                           int live, int lane, Emit&& emit
                                           SSM_DEBUG_ARGS(const float* parts, size_t part_count, int* status)) {
  const int j = lane & 1;
  float2 hist[ROLLED ? 1 : kLB / 2][2][4];
  constexpr int kUnroll = ROLLED ? 1 : kLB;
  {
    float2 h[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float4 v = ck[(2 * q + k) * 32 + lane];
        h[q][2 * k] = make_float2(v.x, v.y);
        h[q][2 * k + 1] = make_float2(v.z, v.w);
      }
#pragma unroll kUnroll
    for (int t = 0; t < kLB; ++t) {
      const float4 v = t1[t * 32 + lane];
      float2 Bv[4];
      load8(fB + t * 16 + 8 * j, Bv);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float dt = q ? v.y : v.x, u = q ? v.w : v.z;
        float2 a[4];
        lane_decays<AP, CPLX>(dt, lc.A2[q], a);
        const float2 du2 = f2dup(dt * u);
        float2 bx[4], hn[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) bx[k] = f2mul(du2, Bv[k]);
        lane_mul_add<CPLX>(a, h[q], bx, hn);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          h[q][k] = hn[k];
          if (!ROLLED && (t & 1)) hist[ROLLED ? 0 : t >> 1][q][k] = hn[k];
        }
      }
      if (ROLLED && (t & 1)) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 lo = h[i >> 1][2 * (i & 1)], hi = h[i >> 1][2 * (i & 1) + 1];
          sh[(t >> 1) * 128 + i * 32 + lane] = make_float4(lo.x, lo.y, hi.x, hi.y);
        }
      }
    }
  }
#pragma unroll kUnroll
  for (int m = kLB / 2 - 1; m >= 0; --m) {
    // pair k of channel q of a lane's states, as the checkpoint holds them
    auto pair_of = [&](const float4* st, int q, int k) {
      const float4 v = st[(2 * q + (k >> 1)) * 32 + lane];
      return (k & 1) ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
    };
    // ---- odd step 2m + 1: its state is hist[m]; its w = mu h_{t-1} waits for the even step's state
    const int to = 2 * m + 1, te = 2 * m;
    const float4 v1o = t1[to * 32 + lane], v2o = t2[to * 32 + lane];
    float yo[2], lo[2];
    const int swz = (lane >> 1) & 3;   // (conflict-free 16-byte stores: 4 vectors per lane)
    {
      float2 Bv[4], Cv[4], dBt[4], dCt[4];
      load8(fB + to * 16 + 8 * j, Bv);
      load8(fC + to * 16 + 8 * j, Cv);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float dt = q ? v1o.y : v1o.x, u = q ? v1o.w : v1o.z, ds = q ? v2o.y : v2o.x;
        float2 a[4];
        lane_decays<AP, CPLX>(dt, lc.A2[q], a);
        // (complex: the staged C is its conjugate and the readout twice a real part, so lam = 2 ds conj(C) + mu; the
        // imaginary rows of dC come out with the other sign)
        const float2 ds2 = f2dup(CPLX ? 2.f * ds : ds), du2 = f2dup(dt * u);
        float2 yv = make_float2(0.f, 0.f), lb = yv, lam[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 hc = ROLLED ? pair_of(sh + m * 128, q, k) : hist[ROLLED ? 0 : m][q][k];
          lam[k] = f2fma(Cv[k], ds2, lc.mu[q][k]);
          dCt[k] = q == 0 ? f2mul(ds2, hc) : f2fma(ds2, hc, dCt[k]);
          dBt[k] = q == 0 ? f2mul(lam[k], du2) : f2fma(lam[k], du2, dBt[k]);
          lb = f2fma(lam[k], Bv[k], lb);
          yv = f2fma(Cv[k], hc, yv);
        }
        lane_mul_conj<CPLX>(a, lam, lc.mu[q]);
        yo[q] = yv.x + yv.y;
        lo[q] = lb.x + lb.y;
      }
      float4* rrow = red + (to & 3) * 128 + lane * 4;
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        rrow[v ^ swz] = make_float4(dBt[2 * v].x, dBt[2 * v].y, dBt[2 * v + 1].x, dBt[2 * v + 1].y);
        rrow[(2 + v) ^ swz] = make_float4(dCt[2 * v].x, dCt[2 * v].y, dCt[2 * v + 1].x, dCt[2 * v + 1].y);
      }
    }
    yo[0] += __shfl_xor_sync(0xffffffffu, yo[1], 1);
    lo[0] += __shfl_xor_sync(0xffffffffu, lo[1], 1);
    // ---- even step 2m: its state is rebuilt from the one before it
    const float4 v1e = t1[te * 32 + lane], v2e = t2[te * 32 + lane];
    float ye[2], le[2], we[2], wo[2];
    {
      float2 Bv[4], Cv[4], dBt[4], dCt[4];
      load8(fB + te * 16 + 8 * j, Bv);
      load8(fC + te * 16 + 8 * j, Cv);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const float dt = q ? v1e.y : v1e.x, u = q ? v1e.w : v1e.z, ds = q ? v2e.y : v2e.x;
        float2 a[4];
        lane_decays<AP, CPLX>(dt, lc.A2[q], a);
        const float2 ds2 = f2dup(CPLX ? 2.f * ds : ds), du2 = f2dup(dt * u), dte2 = f2dup(dt), dto2 = f2dup(q ? v1o.y : v1o.x);
        float2 yv = make_float2(0.f, 0.f), lb = yv, hpp[4], he[4], bx[4], w1[4], lam[4], w0[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          // the state before the even step: the history entry before, or the checkpoint
          if (ROLLED) hpp[k] = pair_of(m > 0 ? sh + (m - 1) * 128 : ck, q, k);
          else if (m > 0) hpp[k] = hist[!ROLLED && m > 0 ? m - 1 : 0][q][k];
          else hpp[k] = pair_of(ck, q, k);
          bx[k] = f2mul(du2, Bv[k]);
        }
        lane_mul_add<CPLX>(a, hpp, bx, he);
        lane_mul_conj<CPLX>(he, lc.mu[q], w1);   // the odd step's w = conj(h_{t-1}) mu_t
        wo[q] = lane_dot_a<CPLX>(w1, lc.A2[q], f2fma(w1[1], lc.A2[q][1], f2mul(w1[0], lc.A2[q][0])));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          lc.dA[q][k] = f2fma(w1[k], dto2, lc.dA[q][k]);
          lam[k] = f2fma(Cv[k], ds2, lc.mu[q][k]);
          dCt[k] = q == 0 ? f2mul(ds2, he[k]) : f2fma(ds2, he[k], dCt[k]);
          dBt[k] = q == 0 ? f2mul(lam[k], du2) : f2fma(lam[k], du2, dBt[k]);
          lb = f2fma(lam[k], Bv[k], lb);
          yv = f2fma(Cv[k], he[k], yv);
        }
        lane_mul_conj<CPLX>(a, lam, lc.mu[q]);
        lane_mul_conj<CPLX>(hpp, lc.mu[q], w0);
        we[q] = lane_dot_a<CPLX>(w0, lc.A2[q], f2fma(w0[1], lc.A2[q][1], f2mul(w0[0], lc.A2[q][0])));
#pragma unroll
        for (int k = 0; k < 4; ++k) lc.dA[q][k] = f2fma(w0[k], dte2, lc.dA[q][k]);
        ye[q] = yv.x + yv.y;
        le[q] = lb.x + lb.y;
      }
      float4* rrow = red + (te & 3) * 128 + lane * 4;
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        rrow[v ^ swz] = make_float4(dBt[2 * v].x, dBt[2 * v].y, dBt[2 * v + 1].x, dBt[2 * v + 1].y);
        rrow[(2 + v) ^ swz] = make_float4(dCt[2 * v].x, dCt[2 * v].y, dCt[2 * v + 1].x, dCt[2 * v + 1].y);
      }
    }
    ye[0] += __shfl_xor_sync(0xffffffffu, ye[1], 1);
    le[0] += __shfl_xor_sync(0xffffffffu, le[1], 1);
    we[0] += __shfl_xor_sync(0xffffffffu, we[1], 1);
    wo[0] += __shfl_xor_sync(0xffffffffu, wo[1], 1);
    __syncwarp();   // all lanes have read the two rows of t2: their slots may take results
    emit(to, CPLX ? 2.f * yo[0] : yo[0], lo[0], wo[0], v1o, v2o);
    emit(te, CPLX ? 2.f * ye[0] : ye[0], le[0], we[0], v1e, v2e);
    if (m % 2 == 0) {
      // dB / dC of steps 2m .. 2m + 3: every lane sums one float4 of one step over the 16 lane pairs, ascending
      __syncwarp();
      const int s = lane >> 3, o = lane & 7, which = o >> 2, n0 = 4 * (o & 3);
      const int jo = n0 >> 3, v = which * 2 + ((n0 >> 2) & 1);
      const float4* rs = red + s * 128;
      float2 lo, hi;
#pragma unroll
      for (int gg = 0; gg < 16; ++gg) {
        const int l = gg * 2 + jo;
        const float4 x = rs[l * 4 + (v ^ (gg & 3))];
        lo = gg == 0 ? make_float2(x.x, x.y) : __fadd2_rn(lo, make_float2(x.x, x.y));
        hi = gg == 0 ? make_float2(x.z, x.w) : __fadd2_rn(hi, make_float2(x.z, x.w));
      }
      float4 acc = make_float4(lo.x, lo.y, hi.x, hi.y);
      if constexpr (CPLX) {
        // four real or four imaginary rows to four columns: the lanes of a half exchange two values each
        const bool im = o & 1;
        if (im && which) acc = make_float4(-acc.x, -acc.y, -acc.z, -acc.w);
        const float gx = __shfl_xor_sync(0xffffffffu, im ? acc.x : acc.z, 1), gy = __shfl_xor_sync(0xffffffffu, im ? acc.y : acc.w, 1);
        acc = im ? make_float4(gx, acc.z, gy, acc.w) : make_float4(acc.x, gx, acc.y, gy);
      }
      const int row = 2 * m + s;
      if (row < live && n0 < n_live) {
        float* dst = (which ? part_dC : part_dB) + (size_t)row * N + n0;
        SSM_GUARD_SPAN(dst, min(n_live - n0, 4), parts, part_count, status, dst = const_cast<float*>(parts))
        if (n_live - n0 >= 4) {   // (then N is a multiple of 4)
          *reinterpret_cast<float4*>(dst) = acc;
        } else {
          dst[0] = acc.x;
          if (n_live - n0 > 1) dst[1] = acc.y;
        }
      }
      __syncwarp();
    }
  }
}

// The lam / mu recurrence alone over steps [t_begin, t_end) of one chain, last to first, from mu (a lane per channel, states
// 16 gi ..): what it leaves and the sum of delta.  a_log2: A * log2(e) of the 16 states [16][32]; tiles: 2048 floats.
template <typename IO, bool VEC, bool CPLX>
__device__ __forceinline__ void adjoint_sweep(const BwdParams& p, int N, int gi, size_t row_b, int t_begin, int t_end, int c0, int lane,
                                              const float* a_log2, bool ap, float bias, bool cvec, float* tiles, float2 (&mu)[8],
                                              float& dsum) {
  const IO* __restrict__ gd = static_cast<const IO*>(p.delta);
  const IO* __restrict__ gz = static_cast<const IO*>(p.z);
  const IO* __restrict__ gg = static_cast<const IO*>(p.dout);
  const IO* __restrict__ gC = static_cast<const IO*>(p.C);
  const int D = p.D, cols = min(32, D - c0);
  const bool has_z = gz != nullptr;
  const int t_last = t_begin + (t_end - t_begin - 1) / kLB * kLB;
  LaneRows<IO, VEC> rd, rz, rg;
  LaneQuad<IO> qC;
  constexpr int kTile = kLB * 32 * (int)sizeof(IO) / 4;
  auto fetch = [&](int t0) {
    const size_t base = (row_b + t0) * D + c0;
    const int last = t_end - 1 - t0, r = lane >> 2, n = 16 * gi + 4 * (lane & 3);
    SSM_GUARD((lane_rows_exist<IO, VEC>((int)(row_b / p.L), p.batch, t0, last, p.L, c0, cols, D)), p.abort, return)
    rd.load(gd + base, D, lane, last, cols);
    if (has_z) rz.load(gz + base, D, lane, last, cols);
    rg.load(gg + base, D, lane, last, cols);
    qC.load(gC + (row_b + t0 + r) * N + n, r <= last ? N - n : 0, cvec);
  };
  if (!has_z) rz.zero();
  fetch(t_last);
  float2 A2[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) A2[k] = make_float2(a_log2[(2 * k) * 32 + lane], a_log2[(2 * k + 1) * 32 + lane]);
  const float zoff = has_z ? 0.f : 1.f;
  auto run = [&](auto ap_tag) {
    constexpr bool AP = decltype(ap_tag)::value;
    int buf = 0;
    float dlost = 0.f;
#pragma unroll 1
    for (int t0 = t_last; t0 >= t_begin; t0 -= kLB, buf ^= 1) {
      float* const tb = tiles + buf * 1024;
      IO* const td = reinterpret_cast<IO*>(tb);
      IO* const tz = reinterpret_cast<IO*>(tb + kTile);
      IO* const tg = reinterpret_cast<IO*>(tb + 2 * kTile);
      float* const tC = tb + 3 * 256;
      rd.put(td, lane);
      rz.put(tz, lane);
      rg.put(tg, lane);
      put_quad<CPLX>(tC, lane, qC.widen(), -1.f);
      float dt[kLB], ds[kLB];
      if constexpr (VEC) {
        __syncwarp();
        if (t0 > t_begin) fetch(t0 - kLB);
      }
#pragma unroll
      for (int t = 0; t < kLB; ++t) {
        dt[t] = rd.get(td, t, lane) + bias;
        const float z = rz.get(tz, t, lane);
        ds[t] = rg.get(tg, t, lane) * fmaf(z, sigmoid_fast(z), zoff);
      }
      if constexpr (!VEC) {
        if (t0 > t_begin) fetch(t0 - kLB);
        __syncwarp();
      }
      if (p.softplus) {
#pragma unroll
        for (int t = 0; t < kLB; ++t) dt[t] = lane_softplus<IO>(dt[t]);
      }
      if (t_end - t0 < kLB) {   // rows past the end are identity steps
#pragma unroll
        for (int t = 0; t < kLB; ++t) {
          dt[t] = t < t_end - t0 ? dt[t] : 0.f;
          ds[t] = t < t_end - t0 ? ds[t] : 0.f;
        }
      }
      add_steps<CPLX>(dt, dsum, dlost);
      // decays and C ds of a step are prepared one step ahead of the recurrence that consumes them
      float2 aN[2][8], cN[2][8];
      auto front = [&](int t, float2 (&a)[8], float2 (&cd)[8]) {
        if constexpr (CPLX) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const int k = (kk & 1) + 4 * (kk >> 1);
            cexp_pair(dt[t], A2[k], A2[k + 2], a[k], a[k + 2]);
          }
        } else if constexpr (AP) {
          const float a0 = ex2_approx(dt[t] * A2[0].x), r = ex2_approx(dt[t] * (A2[0].y - A2[0].x)), r2 = r * r, r4 = r2 * r2,
                      r8 = r4 * r4;
          a[0] = make_float2(a0, a0 * r);
          a[1] = f2mul(a[0], f2dup(r2));
          a[2] = f2mul(a[0], f2dup(r4));
          a[3] = f2mul(a[1], f2dup(r4));
#pragma unroll
          for (int k = 0; k < 4; ++k) a[4 + k] = f2mul(a[k], f2dup(r8));
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float2 e = f2mul(f2dup(dt[t]), A2[k]);
            a[k] = make_float2(ex2_approx(e.x), ex2_approx(e.y));
          }
        }
        load16(tC + t * 16, cd);
      };
      front(kLB - 1, aN[(kLB - 1) & 1], cN[(kLB - 1) & 1]);
#pragma unroll
      for (int t = kLB - 1; t >= 0; --t) {
        if (t > 0) front(t - 1, aN[(t - 1) & 1], cN[(t - 1) & 1]);
        const float2 ds2 = f2dup(CPLX ? 2.f * ds[t] : ds[t]);
        if constexpr (CPLX) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const int k = (kk & 1) + 4 * (kk >> 1);
            const float2 ar = aN[t & 1][k], ai = aN[t & 1][k + 2];
            const float2 lr = f2fma(cN[t & 1][k], ds2, mu[k]), li = f2fma(cN[t & 1][k + 2], ds2, mu[k + 2]);
            mu[k] = f2fma(ai, li, f2mul(ar, lr));
            mu[k + 2] = f2fma(f2neg(ai), lr, f2mul(ar, li));
          }
        } else {
#pragma unroll
          for (int k = 0; k < 8; ++k) mu[k] = f2mul(aN[t & 1][k], f2fma(cN[t & 1][k], ds2, mu[k]));
        }
      }
    }
  };
  if constexpr (sizeof(IO) == 2 && !CPLX) {
    if (ap) run(std::true_type{});
    else run(std::false_type{});
  } else {
    run(std::false_type{});
  }
}

// whether the 16 states 16 gi .. of every lane's channel have their A in arithmetic progression (bf16 io only: the decays
// are then products of rounded exponentials)
template <typename IO>
__device__ __forceinline__ bool lane_progression(const float* a_log2, int N, int gi, int general_A, int lane) {
  bool ap = sizeof(IO) == 2 && !general_A && N - 16 * gi >= 16;
  const float* a = a_log2 + lane;
  const float a0 = a[0], step = a[32] - a0, tol = 1e-6f * fabsf(a[32 * 15]);
  ap = ap && step <= 0.f;   // (as in ssm_fwd_lane.cu)
#pragma unroll
  for (int k = 2; k < 16; ++k) ap = ap && fabsf(a[32 * k] - (a0 + (float)k * step)) <= tol;
  return __all_sync(0xffffffffu, ap);
}

// First pass of a launch split in time: one warp per (chain, group of 16 states), the adjoint that leaves the segment (the
// main kernel folds what leaves the segments behind its own).
// Latency-bound, so capped for four warps per sub-partition (float32 rows in flight take more registers: three).
template <typename IO, bool VEC, bool CPLX>
__global__ void __launch_bounds__(kLaneWarps * 32, sizeof(IO) == 4 ? 3 : 4) ssm_bwd_lane_local_kernel(const BwdParams p, const int N, const int ng) {
  __shared__ __align__(16) float s_tiles[kLaneWarps][2048];
  __shared__ float s_A[kLaneWarps][16 * 32];
  dependency_wait();
  const int bwarp = uniform_warp(), lane = threadIdx.x & 31;
  const int D = p.D, groups = (D + 31) / 32, nseg = p.nseg - 1;   // (nobody wants what leaves the first segment)
  const int item = blockIdx.x * kLaneWarps + bwarp;
  const int gi = item % ng, chain = item / ng;
  if (chain >= p.batch * nseg * groups) return;
  const int grp = chain % groups, bs = chain / groups, seg = bs % nseg + 1, b = bs / nseg;
  const int c_own = grp * 32 + lane, c_ld = min(c_own, D - 1);
  const int t_begin = seg * p.seg_steps, t_end = min(p.L, t_begin + p.seg_steps);
  float* const sA = s_A[bwarp];
  for (int n = 0; n < 16; ++n) {
    const int col = lane_col<CPLX>(16 * gi + n);
    sA[n * 32 + lane] = col < N ? p.A[(size_t)c_ld * N + col] * lane_a_scale<CPLX>(n) : 0.f;
  }
  const float bias = p.delta_bias != nullptr ? p.delta_bias[c_ld] : 0.f;
  const bool cvec = N >= 4 && (reinterpret_cast<uintptr_t>(p.C) & (4 * sizeof(IO) - 1)) == 0;
  const bool ap = !CPLX && lane_progression<IO>(sA, N, gi, p.general_A, lane);
  float2 mu[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) mu[k] = make_float2(0.f, 0.f);
  float dsum = 0.f;
  adjoint_sweep<IO, VEC, CPLX>(p, N, gi, (size_t)b * p.L, t_begin, t_end, grp * 32, lane, sA, ap, bias, cvec, s_tiles[bwarp], mu, dsum);
  // [batch][segment][channel group][row][32], rows as in shared memory
  const size_t at = ((size_t)b * p.nseg + seg) * groups + grp;
  SSM_GUARD(at < (size_t)p.batch * p.nseg * groups && gi < ng, p.abort, return)
  float* const dst = p.seg_local + (at * ng + gi) * 512 + lane;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    dst[64 * k] = mu[k].x;
    dst[64 * k + 32] = mu[k].y;
  }
  if (gi == 0) p.seg_dsum[at * 32 + lane] = dsum;
}

// CPLX: complex states, as in ssm_fwd_lane.cu
template <typename IO, int NG, int ROWS, bool CPLX, bool ROLLED>
__global__ void __launch_bounds__(kLaneWarps * 32, 2) ssm_bwd_lane_kernel(const BwdParams p, const LaneSplit sp, const int N) {
  constexpr bool VEC = ROWS == kVectors;
  using SM = BwdLaneSmem<IO, NG, VEC, ROLLED>;
  constexpr int NP = SM::NP, kTeams = SM::kTeams;
  extern __shared__ __align__(16) unsigned char smem[];
  dependency_wait();
  const int bwarp = uniform_warp(), lane = threadIdx.x & 31;
  const int W = sp.warps, CL = sp.cluster;      // pieces of a chain in this block, blocks of the chain
  const int team = bwarp / NG, gi = bwarp % NG; // gi: this warp's group of 16 states
  const int sub = div_pow2(team, W), tw = team - sub * W;      // which chain of the block, which of its pieces here
  const int per_block = div_pow2(kTeams, W);
  SSM_GUARD(W * per_block == kTeams && SM::bytes(per_block) <= dynamic_smem_bytes() && cluster_rank() < CL, p.abort, return)
  unsigned char* const sTeam = smem + team * SM::kTeam;
  unsigned char* const rX = sTeam;
  unsigned char* const rD = rX + SM::kRaw;
  unsigned char* const rZ = rD + SM::kRaw;
  unsigned char* const rG = rZ + SM::kRaw;
  float4* const t1 = reinterpret_cast<float4*>(rG + SM::kRaw);
  float4* const t2 = t1 + kLB * 32;
  unsigned char* const sWarps = smem + kTeams * SM::kTeam;
  auto warp_base = [&](int w) { return reinterpret_cast<float*>(sWarps + w * SM::kWarp); };
  float* const fB = warp_base(bwarp);
  float* const fC = fB + kLB * 16;
  float4* const ck = reinterpret_cast<float4*>(fC + kLB * 16);   // [2][4][32]
  float4* const red = ck + 2 * 128;
  float4* const ex = red + 4 * 128;                              // NG > 1: [kLB][32]
  float4* const sh = red + 4 * 128 + (NG > 1 ? kLB * 32 : 0);    // ROLLED: states after the odd steps of a block
  // what leaves piece w of this chain, states 16 gi .. of it: in the transposing buffer of its warp
  auto leaving = [&](int w, int n) {
    return warp_base((sub * W + w) * NG + (n >> 4)) + 2 * kLB * 16 + 2 * 128 * 4 + (n & 15) * 32;
  };
  float* const sChain = reinterpret_cast<float*>(sWarps + kLaneWarps * SM::kWarp + sub * SM::kChain);
  float* const sA = sChain;                  // [NP][32]
  float* const sTotDs = sA + NP * 32;        // [32]
  float* const sDs = sTotDs + 32;            // [kTeams][32]
  float* const sTot = reinterpret_cast<float*>(smem + sub * W * SM::kTeam + 4 * SM::kRaw);   // [NP][32], where t1 and t2 go later
  float* const sAcc = reinterpret_cast<float*>(sWarps + kLaneWarps * SM::kWarp + per_block * SM::kChain);   // [warps][2][32]

  const IO* __restrict__ gx = static_cast<const IO*>(p.x);
  const IO* __restrict__ gd = static_cast<const IO*>(p.delta);
  const IO* __restrict__ gz = static_cast<const IO*>(p.z);
  const IO* __restrict__ gg = static_cast<const IO*>(p.dout);
  const IO* __restrict__ gB = static_cast<const IO*>(p.B);
  const IO* __restrict__ gC = static_cast<const IO*>(p.C);

  const int D = p.D, groups = (D + 31) / 32;
  const int rank = cluster_rank();
  const int nseg = p.nseg, chains = p.batch * nseg * groups;
  const int chain_id = cluster_index() * per_block + sub;
  const int chain = min(chain_id, chains - 1);
  const int bs = chain / groups, grp = chain - bs * groups;
  const int b = nseg == 1 ? bs : bs / nseg, seg = bs - b * nseg;
  const int c_own = grp * 32 + lane, cols = min(32, D - grp * 32);
  const bool valid = c_own < D;
  const int c_ld = valid ? c_own : D - 1;
  const int seg_t0 = seg * p.seg_steps, seg_end = min(p.L, seg_t0 + p.seg_steps);
  const int t_begin = chain_id < chains ? min(seg_end, seg_t0 + (rank * W + tw) * sp.piece) : seg_end;
  const int t_end = min(seg_end, t_begin + sp.piece);
  const bool live_piece = t_begin < t_end;
  const bool has_z = gz != nullptr;
  const bool bvec = N >= 4 && (reinterpret_cast<uintptr_t>(p.B) & (4 * sizeof(IO) - 1)) == 0;
  const bool cvec = N >= 4 && (reinterpret_cast<uintptr_t>(p.C) & (4 * sizeof(IO) - 1)) == 0;
  const size_t row_b = (size_t)b * p.L;
  const int t_last = live_piece ? t_begin + (t_end - t_begin - 1) / kLB * kLB : t_begin;   // first step of the last block
  auto team_sync = [&] {
    if constexpr (NG == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(32 * NG) : "memory");
  };

  for (int n = tw * NG + gi; n < NP; n += W * NG) {
    const int col = lane_col<CPLX>(n);
    sA[n * 32 + lane] = col < N ? p.A[(size_t)c_ld * N + col] * lane_a_scale<CPLX>(n) : 0.f;
  }
  const float bias = p.delta_bias != nullptr ? p.delta_bias[c_ld] : 0.f;
  // four of the 16 states of row lane / 4 of a block of B or C; rows past the end are zero
  auto quad = [&](LaneQuad<IO>& q, const IO* src, int t0, bool vec) {
    const int r = lane >> 2, n = 16 * gi + 4 * (lane & 3);
    SSM_GUARD(t0 + r >= t_end || n >= N || (row_b + t0 + r) * N + n + min(N - n, 4) <= (size_t)p.batch * p.L * N, p.abort, return)
    q.load(src + (row_b + t0 + r) * N + n, t0 + r < t_end ? N - n : 0, vec);
  };
  __syncthreads();
  const bool ap = !CPLX && lane_progression<IO>(sA + gi * 512, N, gi, p.general_A, lane);

  const bool split = W * CL > 1;
  // ---- first sweep: the adjoint that leaves the piece with nothing flowing in (a lane per channel, 16 states)
  float dsum = 0.f;
  if (split) {
    float2 mu[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) mu[k] = make_float2(0.f, 0.f);
    if (live_piece && rank * W + tw > 0) {   // (nobody wants what leaves the first piece)
      adjoint_sweep<IO, VEC, CPLX>(p, N, gi, row_b, t_begin, t_end, grp * 32, lane, sA + gi * 512, ap, bias, cvec,
                             reinterpret_cast<float*>(red), mu, dsum);
      __syncwarp();
    }
    float* const e = leaving(tw, 16 * gi) + lane;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      e[64 * k] = mu[k].x;
      e[64 * k + 32] = mu[k].y;
    }
    if (gi == 0) sDs[tw * 32 + lane] = dsum;
  }

  // ---- rows of the main sweep: each warp of the team copies its share of the four tensors
  RawRows<IO, ROWS> rr;
  rr.setup((row_b + t_begin) * D + grp * 32, D, lane, cols);
  auto issue_rows = [&](int t0) {
    const size_t base = (row_b + t0) * D + grp * 32;
    const int live = min(kLB, t_end - t0);
    if (0 % NG == gi) rr.issue(rX, gx + base, D, lane, cols, live SSM_DEBUG_ARGS(gx, (size_t)p.batch * p.L * D, p.abort));
    if (1 % NG == gi) rr.issue(rD, gd + base, D, lane, cols, live SSM_DEBUG_ARGS(gd, (size_t)p.batch * p.L * D, p.abort));
    if (2 % NG == gi && has_z) rr.issue(rZ, gz + base, D, lane, cols, live SSM_DEBUG_ARGS(gz, (size_t)p.batch * p.L * D, p.abort));
    if (3 % NG == gi) rr.issue(rG, gg + base, D, lane, cols, live SSM_DEBUG_ARGS(gg, (size_t)p.batch * p.L * D, p.abort));
  };
  // the states before a block, for the lane's two channels and 8 states: vectors [2 q + k][lane]
  const bool ck_vec = p.ckpt_tiled && (reinterpret_cast<uintptr_t>(p.ckpt) & 15) == 0;
  const int n_own = 16 * gi + 8 * (lane & 1);   // first of the lane's states
  const int NC = lane_ckpt_rows<CPLX>(N);
  const float* const ck_own = p.ckpt + ckpt_offset(1, b, p.nck, 0, D, NC, grp * 32, 0) + (size_t)(n_own >> 2) * 128;
  const size_t ck_step = ckpt_floats_per_step(1, D, NC);
  int ck_bytes[2][2];   // 16, or 0 where the channel or the states do not exist
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < 2; ++k) ck_bytes[q][k] = (lane ^ q) < cols && n_own + 4 * k < NC ? 16 : 0;
  auto issue_ckpt = [&](int t0, float4* dst) {
    const int kc = t0 / kCkptSteps;
    const float* const src = ck_own + (size_t)kc * ck_step;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float4* at = dst + (2 * q + k) * 32 + lane;
        SSM_GUARD(!ck_bytes[q][k] || ckpt_offset(p.ckpt_tiled, b, p.nck, kc, D, NC, grp * 32 + (lane ^ q), n_own + 4 * k) + min(4, NC) <=
                                         (size_t)p.batch * p.nck * ckpt_floats_per_step(p.ckpt_tiled, D, NC), p.abort, continue)
        SSM_GUARD(!ck_vec || src + k * 128 + (lane ^ q) * 4 == p.ckpt + ckpt_offset(1, b, p.nck, kc, D, NC, grp * 32 + (lane ^ q), n_own + 4 * k),
                  p.abort, continue)
        if (ck_vec) {
          cp_async16_bytes(at, ck_bytes[q][k] ? src + k * 128 + (lane ^ q) * 4 : p.ckpt, ck_bytes[q][k]);
        } else {
#pragma unroll 1
          for (int i = 0; i < 4; ++i) {
            const int n = n_own + 4 * k + i;
            const float x = (lane ^ q) < cols && n < NC ? p.ckpt[ckpt_offset(p.ckpt_tiled, b, p.nck, kc, D, NC, grp * 32 + (lane ^ q), n)] : 0.f;
            reinterpret_cast<float*>(at)[i] = x;
          }
        }
      }
    }
  };
  LaneQuad<IO> qB, qC;
  if (live_piece) {
    issue_rows(t_last);
    issue_ckpt(t_last, ck);
    quad(qB, gB, t_last, bvec);
    quad(qC, gC, t_last, cvec);
  }
  cp_async_commit();

  // ---- fold over the pieces, last to first
  LaneChain lc;
  lc.Dk = p.Dskip != nullptr && valid ? p.Dskip[c_ld] : 0.f;
  lc.dD = lc.dbias = 0.f;
  if (split) {
    __syncthreads();
    // (a complex adjoint: rows n and n + 4)
    constexpr int kRow2 = 4 * 32;
    for (int n = tw * NG + gi; n < NP; n += W * NG) {
      if (CPLX && (n & 4)) continue;
      const float a2 = sA[n * 32 + lane], ai = CPLX ? sA[n * 32 + kRow2 + lane] : 0.f;
      float2 pre = make_float2(0.f, 0.f);
      float ds = 0.f;
      float2 l[kTeams];
      float d[kTeams];
#pragma unroll
      for (int w = kTeams - 1; w >= 0; --w) {   // (all loaded before the first is used)
        const float* const at = leaving(w < W ? w : 0, n) + lane;
        l[w] = make_float2(*at, CPLX ? at[kRow2] : 0.f);
        d[w] = sDs[(w < W ? w : 0) * 32 + lane];
      }
#pragma unroll
      for (int w = kTeams - 1; w >= 0; --w) {
        if (w < W) {
          float* const at = leaving(w, n) + lane;
          *at = pre.x;
          if (CPLX) at[kRow2] = pre.y;
          const float2 q = CPLX ? cexp_apply<true>(d[w], a2, ai, pre) : make_float2(ex2_approx(a2 * d[w]) * pre.x, 0.f);
          pre = make_float2(q.x + l[w].x, q.y + l[w].y);
          ds += d[w];
        }
      }
      sTot[n * 32 + lane] = pre.x;
      if (CPLX) sTot[n * 32 + kRow2 + lane] = pre.y;
      if (n == 0) sTotDs[lane] = ds;
    }
    if (CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    for (int n = tw * NG + gi; n < NP; n += W * NG) {
      if (CPLX && (n & 4)) continue;
      const int col = lane_col<CPLX>(n);
      const float a2 = sA[n * 32 + lane], ai = CPLX ? sA[n * 32 + kRow2 + lane] : 0.f;
      auto step = [&](float d, float2 v) {
        return CPLX ? cexp_apply<true>(d, a2, ai, v) : make_float2(ex2_approx(a2 * d) * v.x, 0.f);
      };
      float2 M = make_float2(0.f, 0.f);
      if (p.mu_in != nullptr && col < N) {
        M.x = p.mu_in[((size_t)b * D + c_ld) * N + col];
        if (CPLX) M.y = p.mu_in[((size_t)b * D + c_ld) * N + col + 1];
      }
      float2 rt[kLaneMaxCluster];
      float rds[kLaneMaxCluster];
#pragma unroll
      for (int r = kLaneMaxCluster - 1; r > 0; --r) {   // (all requested before the first is used)
        if (r > rank && r < CL) {
          const float* const tot = cg::this_cluster().map_shared_rank(sTot, r) + n * 32 + lane;
          rt[r] = make_float2(tot[0], CPLX ? tot[kRow2] : 0.f);
          rds[r] = cg::this_cluster().map_shared_rank(sTotDs, r)[lane];
        }
      }
#pragma unroll
      for (int r = kLaneMaxCluster - 1; r > 0; --r) {
        if (r > rank && r < CL) {
          const float2 q = step(rds[r], M);
          M = make_float2(q.x + rt[r].x, q.y + rt[r].y);
        }
      }
      float2 l[kTeams];
      float cum[kTeams];
      float sum = 0.f;
#pragma unroll
      for (int w = kTeams - 1; w >= 0; --w) {
        const float* const at = leaving(w < W ? w : 0, n) + lane;
        l[w] = make_float2(*at, CPLX ? at[kRow2] : 0.f);
        cum[w] = sum;
        if (w < W) sum += sDs[w * 32 + lane];
      }
#pragma unroll
      for (int w = kTeams - 1; w >= 0; --w) {
        if (w < W) {
          float* const at = leaving(w, n) + lane;
          const float2 q = step(cum[w], M);
          *at = l[w].x + q.x;
          if (CPLX) at[kRow2] = l[w].y + q.y;
        }
      }
    }
    if (CL > 1) cg::this_cluster().sync();   // (also: no block leaves while another still reads its totals)
    else __syncthreads();
  }
  // a launch split into segments: fold what leaves the segments behind this one, last to first
  const bool behind = p.nseg > 1 && seg < p.nseg - 1;
  if (behind) {
    float M[16];
#pragma unroll
    for (int n = 0; n < 16; ++n) {
      const int col = lane_col<CPLX>(16 * gi + n);
      M[n] = p.mu_in != nullptr && col < N ? p.mu_in[((size_t)b * D + c_ld) * N + col] : 0.f;
    }
    const float* const a = sA + gi * 512 + lane;
    // (the values of several segments requested before the first is used: one by one the fold took 7000 cycles of a block's
    // 230000 at 12 segments)
    constexpr int kAhead = CPLX ? 2 : 4;
#pragma unroll 1
    for (int sg = p.nseg - 1; sg > seg; sg -= kAhead) {
      float l[kAhead][16], ds[kAhead];
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        const size_t at = ((size_t)b * p.nseg + max(sg - i, seg + 1)) * groups + grp;
        const float* const src = p.seg_local + (at * NG + gi) * 512 + lane;
        ds[i] = p.seg_dsum[at * 32 + lane];
#pragma unroll
        for (int n = 0; n < 16; ++n) l[i][n] = src[32 * n];
      }
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        if (sg - i > seg) {
#pragma unroll
          for (int n = 0; n < 16; ++n) {
            if constexpr (CPLX) {
              if (n & 4) continue;
              const float2 q = cexp_apply<true>(ds[i], a[32 * n], a[32 * n + 128], make_float2(M[n], M[n + 4]));
              M[n] = q.x + l[i][n];
              M[n + 4] = q.y + l[i][n + 4];
            } else {
              M[n] = fmaf(ex2_approx(a[32 * n] * ds[i]), M[n], l[i][n]);
            }
          }
        }
      }
    }
    float* const to = leaving(tw, 16 * gi) + lane;
#pragma unroll
    for (int n = 0; n < 16; ++n) to[32 * n] = M[n];
    __syncwarp();
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int cl = lane ^ q;
    const bool ok = grp * 32 + cl < D;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int n = 16 * gi + 8 * (lane & 1) + k;
      float m = 0.f;
      if (split || behind) m = ok ? leaving(tw, n)[cl] : 0.f;
      else if (p.mu_in != nullptr && ok && lane_col<CPLX>(n) < N) m = p.mu_in[((size_t)b * D + grp * 32 + cl) * N + lane_col<CPLX>(n)];
      reinterpret_cast<float*>(lc.mu[q])[k] = m;
      reinterpret_cast<float*>(lc.A2[q])[k] = sA[n * 32 + cl];
      reinterpret_cast<float*>(lc.dA[q])[k] = 0.f;
    }
  }
  __syncwarp();

  // ---- main sweep
  IO* const ox = static_cast<IO*>(p.dx);
  IO* const od = static_cast<IO*>(p.ddelta);
  IO* const oz = static_cast<IO*>(p.dz);
  const size_t bln = (size_t)p.batch * p.L * N;
  // what this lane writes of a block: bytes from the block's first element, first slot (a multiple of 8 but for the
  // permutation of its low bits) and row
  constexpr int kVecs = kLB / NG * LaneRows<IO, true>::VPR, kFlush = VEC ? (kVecs + 31) / 32 : 1;
  unsigned fl_off[kFlush], fl_slot[kFlush];
  if constexpr (VEC) {
    using R = LaneRows<IO, true>;
#pragma unroll
    for (int i = 0; i < kFlush; ++i) {
      const int q = lane + 32 * i, t = gi * (kLB / NG) + q / R::VPR, col = q % R::VPR * R::EPV;
      fl_off[i] = (unsigned)(t * D + col) * (unsigned)sizeof(IO);
      fl_slot[i] = (unsigned)(t * 32 + (col & 24)) | (unsigned)(out_slot(t, col) & 7) | (unsigned)(q < kVecs && col < cols ? t : kLB) << 16;
    }
  }
  auto sweep = [&](auto ap_tag) {
    constexpr bool AP = decltype(ap_tag)::value;
    int st = 0;
#pragma unroll 1
    for (int t0 = t_last; t0 >= t_begin; t0 -= kLB, st ^= 1) {
      const int live = min(kLB, t_end - t0);
      const size_t row0 = row_b + t0, base = row0 * D + grp * 32;
      cp_async_wait_all();
      put_quad<CPLX>(fB, lane, qB.widen(), 1.f);
      put_quad<CPLX>(fC, lane, qC.widen(), -1.f);   // (complex: conj C)
      team_sync();   // the rows of all warps of the team have landed
      // per-step values of the rows, each warp its share: step size, input, gate terms.  Two rows at a time, their loads and
      // arithmetic before the first store, which no later load may pass (it was a fifth of a block's time, 2270 of 10700 cycles at
      // float32 (2, 2048, 1536), with a row's stores before the next row's loads).  Not more, and with complex states one: the
      // body of a block is near the size of the instruction cache or beyond it (main kernel at float32 (2, 2048, 1536) 133.0 us
      // before, 130.4 with two rows, 131.0 with four, 133.0 with eight; bf16 (3, 1237, 1001) 97.0, 95.3 with two; complex, whole
      // backward, the same within 1 % in two orders of the problems: bf16 (2, 2048, 1536) 489 before, 479 with one row, 497 with
      // two, float32 (2, 2048, 1001) 360, 352, 363; small ones 1 to 2 % the other way, (2, 1000, 300) 101.1, 101.0, 99.4).
      constexpr int kOwn = kLB / NG, kAtOnce = CPLX ? 1 : 2;
      static_assert(kOwn % kAtOnce == 0, "whole groups of rows");
#pragma unroll 1
      for (int i0 = 0; i0 < kOwn; i0 += kAtOnce) {
        const int tb = gi * kOwn + i0;
        float dt[kAtOnce], uu[kAtOnce], ds[kAtOnce], gp[kAtOnce], step[kAtOnce];
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) {
          dt[i] = rr.get(rD, tb + i, lane) + bias;
          uu[i] = rr.get(rX, tb + i, lane);
          ds[i] = rr.get(rG, tb + i, lane);
          gp[i] = 0.f;
          step[i] = 1.f;
        }
        if (has_z) {
          float z[kAtOnce];
#pragma unroll
          for (int i = 0; i < kAtOnce; ++i) z[i] = rr.get(rZ, tb + i, lane);
#pragma unroll
          for (int i = 0; i < kAtOnce; ++i) {
            const float g = ds[i], sg = sigmoid_fast(z[i]);
            ds[i] = g * z[i] * sg;
            gp[i] = g * sg * fmaf(z[i], 1.f - sg, 1.f);
          }
        }
        if (p.softplus) {
#pragma unroll
          for (int i = 0; i < kAtOnce; ++i) {
            const float dv = dt[i];
            dt[i] = lane_softplus<IO>(dv);
            step[i] = sizeof(IO) == 4 ? 1.f / (1.f + __expf(-dv)) : sigmoid_from_softplus(dt[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) {
          const bool ok = valid && tb + i < live;
          dt[i] = ok ? dt[i] : 0.f;
          uu[i] = ok ? uu[i] : 0.f;
          ds[i] = ok ? ds[i] : 0.f;
          gp[i] = ok ? gp[i] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < kAtOnce; ++i) {
          t1[(tb + i) * 32 + lane] = make_float4(dt[i], __shfl_xor_sync(0xffffffffu, dt[i], 1), uu[i], __shfl_xor_sync(0xffffffffu, uu[i], 1));
          t2[(tb + i) * 32 + lane] = make_float4(ds[i], __shfl_xor_sync(0xffffffffu, ds[i], 1), gp[i], step[i]);
        }
      }
      team_sync();
      if (t0 > t_begin) {
        issue_rows(t0 - kLB);
        issue_ckpt(t0 - kLB, ck + (st ^ 1) * 128);
        quad(qB, gB, t0 - kLB, bvec);
        quad(qC, gC, t0 - kLB, cvec);
      }
      cp_async_commit();
      auto put = [&](int t, float3 r) { t2[t * 32 + out_slot(t, lane)] = make_float4(r.x, r.y, r.z, 0.f); };
      float* const part_dB = p.dBC_part + (size_t)grp * 2 * bln + row0 * N + 16 * gi;
      lane_block<AP, CPLX, ROLLED>(lc, t1, t2, fB, fC, ck + st * 128, sh, red, part_dB, part_dB + bln, N, N - 16 * gi, live, lane,
                     [&](int t, float y, float lb, float wa, float4 v1, float4 v2) {
                       if constexpr (NG == 1) put(t, finish_step(lc, v1, v2, y, lb, wa, t < live));
                       else ex[t * 32 + lane] = make_float4(y, lb, wa, 0.f);
                     } SSM_DEBUG_ARGS(p.dBC_part, (size_t)groups * 2 * bln, p.abort));
      if constexpr (NG > 1) {
        team_sync();
#pragma unroll
        for (int i = 0; i < kLB / NG; ++i) {
          const int t = gi * (kLB / NG) + i;
          float y = 0.f, lb = 0.f, wa = 0.f;
#pragma unroll
          for (int w = 0; w < NG; ++w) {   // (ascending groups of states)
            const float4 v = reinterpret_cast<const float4*>(warp_base(team * NG + w) + 2 * kLB * 16 + 2 * 128 * 4 + 4 * 128 * 4)[t * 32 + lane];
            y += v.x;
            lb += v.y;
            wa += v.z;
          }
          const float4 v1 = t1[t * 32 + lane], v2 = t2[t * 32 + lane];
          __syncwarp();
          put(t, finish_step(lc, v1, v2, y, lb, wa, t < live));
        }
      }
      // the rows this warp finished: 16-byte stores, or one channel per lane
      __syncwarp();
      if constexpr (VEC) {
        using R = LaneRows<IO, true>;
#pragma unroll
        for (int i = 0; i < kFlush; ++i) {
          if ((int)(fl_slot[i] >> 16) < min(live, kLB)) {
            const float4* const from = t2 + (fl_slot[i] & 0xfff8u);
            SSM_GUARD((fl_slot[i] & 0xfff8u) + 8 <= kLB * 32, p.abort, continue)
            SSM_GUARD_SPAN(at_bytes(ox + base, fl_off[i]), R::EPV, ox, (size_t)p.batch * p.L * D, p.abort, continue)
            const int x = fl_slot[i] & 7;
            __align__(16) IO vx[R::EPV], vd[R::EPV], vz[R::EPV];
#pragma unroll
            for (int k = 0; k < R::EPV; ++k) {
              const float4 v = from[k ^ x];
              vx[k] = float_to_io<IO>(v.x);
              vd[k] = float_to_io<IO>(v.y);
              vz[k] = float_to_io<IO>(v.z);
            }
            *reinterpret_cast<uint4*>(at_bytes(ox + base, fl_off[i])) = *reinterpret_cast<const uint4*>(vx);
            *reinterpret_cast<uint4*>(at_bytes(od + base, fl_off[i])) = *reinterpret_cast<const uint4*>(vd);
            if (oz != nullptr) *reinterpret_cast<uint4*>(at_bytes(oz + base, fl_off[i])) = *reinterpret_cast<const uint4*>(vz);
          }
        }
      } else if (valid) {
        unsigned at = (unsigned)(gi * (kLB / NG) * D + lane) * (unsigned)sizeof(IO);
#pragma unroll 2
        for (int i = 0; i < kLB / NG; ++i, at += (unsigned)D * (unsigned)sizeof(IO)) {
          const int t = gi * (kLB / NG) + i;
          if (t >= live) break;
          SSM_GUARD_SPAN(at_bytes(ox + base, at), 1, ox, (size_t)p.batch * p.L * D, p.abort, break)
          const float4 v = t2[t * 32 + out_slot(t, lane)];
          *at_bytes(ox + base, at) = float_to_io<IO>(v.x);
          *at_bytes(od + base, at) = float_to_io<IO>(v.y);
          if (oz != nullptr) *at_bytes(oz + base, at) = float_to_io<IO>(v.z);
        }
      }
    }
  };
  if (live_piece) {
    if constexpr (sizeof(IO) == 2 && !CPLX) {
      if (ap) sweep(std::true_type{});
      else sweep(std::false_type{});
    } else {
      sweep(std::false_type{});
    }
  }
  cp_async_wait_all();
  __syncwarp();

  // ---- sums over time: added over the pieces of the chain in this block, in order, one partial sum per block
  {
    float* const e = leaving(tw, 16 * gi);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < 8; ++k) e[(8 * (lane & 1) + k) * 32 + (lane ^ q)] = reinterpret_cast<float*>(lc.dA[q])[k];
    sAcc[bwarp * 64 + lane] = lc.dD;
    sAcc[bwarp * 64 + 32 + lane] = lc.dbias;
    // (the first step's piece: the adjoint that leaves it is the gradient of the initial state)
    if (p.dh0 != nullptr && seg == 0 && rank == 0 && tw == 0 && chain_id < chains) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int c = grp * 32 + (lane ^ q);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int n = 16 * gi + 8 * (lane & 1) + k;
          const int col = lane_col<CPLX>(n);
          if (c < D && col < N) p.dh0[((size_t)b * D + c) * N + col] = reinterpret_cast<float*>(lc.mu[q])[k];
        }
      }
    }
  }
  __syncthreads();
  if (valid && chain_id < chains) {
    const size_t part = ((size_t)b * p.nseg + seg) * CL + rank;
    SSM_GUARD(part < (size_t)p.batch * p.nseg * CL, p.abort, return)
    for (int n = tw * NG + gi; n < NP; n += W * NG) {
      const int col = lane_col<CPLX>(n);
      float v = 0.f;
      for (int w = 0; w < W; ++w) v += leaving(w, n)[lane];
      if (col < N) p.dA_part[(part * D + c_own) * N + col] = v;
    }
    if (tw == 0 && gi == 0) {
      float dD = 0.f, db = 0.f;
      for (int w = 0; w < W * NG; ++w) {
        dD += sAcc[(sub * W * NG + w) * 64 + lane];
        db += sAcc[(sub * W * NG + w) * 64 + 32 + lane];
      }
      p.dD_part[part * D + c_own] = dD;
      if (p.dbias_part != nullptr) p.dbias_part[part * D + c_own] = db;
    }
  }
}

template <typename IO, int NG, int ROWS, bool CPLX, bool ROLLED>
cudaError_t launch_bwd_lane_main(const Plan& plan, const BwdParams& p, int N, cudaStream_t s) {
  using SM = BwdLaneSmem<IO, NG, ROWS == kVectors, ROLLED>;
  auto kern = ssm_bwd_lane_kernel<IO, NG, ROWS, CPLX, ROLLED>;
  const long long chains = (long long)p.batch * plan.nseg * ((p.D + 31) / 32);
  const LaneSplit sp = plan.split;
  const int per_block = SM::kTeams / sp.warps;
  KernelLimits lim;
  const cudaError_t e = kernel_limits(reinterpret_cast<const void*>(kern), 32 * kLaneWarps, SM::bytes(SM::kTeams), &lim);
  if (e != cudaSuccess) return e;
  return launch_dependent(kern, (unsigned)((chains + per_block - 1) / per_block * sp.cluster), 32 * kLaneWarps, SM::bytes(per_block), sp.cluster, s, p, sp, N);
}

template <typename IO, int NG, int ROWS, bool CPLX>
cudaError_t launch_bwd_lane_n(const Plan& plan, const BwdParams& p, int N, int mode, cudaStream_t s) {
  if (mode == kBwdLocal) {
    const long long items = (long long)p.batch * (plan.nseg - 1) * ((p.D + 31) / 32) * NG;
    if (items <= 0) return cudaSuccess;
    return launch_dependent(ssm_bwd_lane_local_kernel<IO, ROWS == kVectors, CPLX>, (unsigned)((items + kLaneWarps - 1) / kLaneWarps), kLaneWarps * 32, 0, 1, s, p, N, NG);
  }
  // A piece of one block runs the block's code once, so its time is that of fetching the code: with loops over the steps, and
  // the states after the odd steps in shared memory instead of registers, that is a quarter of it (float32 (1, 256, 64): main
  // kernel 13.6 -> 12.0 us; with two blocks per piece the loops cost what they save).  Its shared memory leaves room for one
  // block per SM, so only for grids that then still run at once (float32 (2, 256, 256), 16 clusters of 8: 25.5 -> 34.6 us a
  // pass): eight clusters of 8, smaller clusters on three quarters of the SMs, or a block per SM.  (The occupancy query
  // gives 15 clusters of 8, 33 of 4 and 74 of 2 at once; between the lines and these nothing was timed.)
  if constexpr (NG == 1 && !CPLX) {
    const LaneSplit sp = plan.split;
    const int per_block = kLaneWarps / sp.warps, most = sp.cluster == 8 ? 64 : sp.cluster > 1 ? 112 : kNumSMs;
    const long long chains = (long long)p.batch * ((p.D + 31) / 32), blocks = (chains + per_block - 1) / per_block * sp.cluster;
    if (plan.nseg == 1 && sp.piece <= kLB && blocks <= most) return launch_bwd_lane_main<IO, NG, ROWS, CPLX, true>(plan, p, N, s);
  }
  return launch_bwd_lane_main<IO, NG, ROWS, CPLX, false>(plan, p, N, s);
}

template <typename IO, int NG, bool CPLX>
cudaError_t launch_bwd_lane_vec(const Plan& plan, const BwdParams& p, int N, int mode, cudaStream_t s) {
  uintptr_t in = 0, out = 0;
  for (const void* q : {p.x, p.delta, p.z, p.dout}) in |= reinterpret_cast<uintptr_t>(q);
  for (const void* q : {p.dx, p.ddelta, p.dz}) out |= reinterpret_cast<uintptr_t>(q);
  if ((size_t)p.D * sizeof(IO) % 16 == 0 && ((in | out) & 15) == 0) return launch_bwd_lane_n<IO, NG, kVectors, CPLX>(plan, p, N, mode, s);
  if constexpr (sizeof(IO) == 2) {
    if (in & 3) return launch_bwd_lane_n<IO, NG, kElements, CPLX>(plan, p, N, mode, s);
  }
  return launch_bwd_lane_n<IO, NG, kWords, CPLX>(plan, p, N, mode, s);
}

template <typename IO, bool CPLX>
cudaError_t launch_bwd_lane_io(const Plan& plan, const BwdParams& p, int N, int mode, cudaStream_t s) {
  if (N <= 16) return launch_bwd_lane_vec<IO, 1, CPLX>(plan, p, N, mode, s);
  if (N <= 32) return launch_bwd_lane_vec<IO, 2, CPLX>(plan, p, N, mode, s);
  return launch_bwd_lane_vec<IO, 4, CPLX>(plan, p, N, mode, s);
}

}  // namespace

bool bwd_lane_applicable(const BwdParams& p) { return !p.zoh && !p.static_B && !p.static_C; }

cudaError_t launch_bwd_lane(const ssm_problem_t& prob, const Plan& plan, const BwdParams& p, int mode, cudaStream_t s) {
  const bool bf = prob.io_dtype == SSM_BF16;
  if (prob.flags & SSM_FLAG_COMPLEX)
    return bf ? launch_bwd_lane_io<__nv_bfloat16, true>(plan, p, 2 * prob.N, mode, s) : launch_bwd_lane_io<float, true>(plan, p, 2 * prob.N, mode, s);
  return bf ? launch_bwd_lane_io<__nv_bfloat16, false>(plan, p, prob.N, mode, s) : launch_bwd_lane_io<float, false>(plan, p, prob.N, mode, s);
}

}  // namespace ssm
