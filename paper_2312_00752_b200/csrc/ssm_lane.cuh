// Pieces shared by the lane-per-channel kernels (ssm_fwd_lane.cu, ssm_bwd_lane.cu): element loads and stores of either io
// dtype at any alignment, the staging of B and C, and the split of a chain over the warps of a cluster.
//
// These kernels take what the tuned bf16 / N = 16 kernels do not: float32 io, any D and any pointer alignment, any
// N (states are handled 16 at a time; N < 16 is padded with states that stay zero).  x, delta, z, dout go straight from
// global memory to the lane that owns the channel (a warp's 32 lanes read one contiguous row piece, so no alignment
// beyond the element's is needed), one batch of 8 steps ahead of its use; only B and C, which every lane needs, pass
// through shared memory.
//
// A chain is 32 adjacent channels of one batch entry (of one time segment of the launch, if the launch is split in
// time).  When the chains alone cannot fill the GPU a chain is cut in time between the W warps of a block and the blocks
// of a cluster: every warp sweeps its piece from a zero state, the (decay, end state) pairs are folded through
// (distributed) shared memory, and every warp sweeps its piece again from the true state.  That costs what the summary
// launch of a time split costs, but no carry launch and no round trip through global memory, and pieces may be as short
// as one batch.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "ssm_common.cuh"

namespace ssm {

constexpr int kLB = kCkptSteps;   // steps per batch of the lane kernels (= checkpoint spacing)
constexpr int kLaneChannels = 32; // channels per chain

// Blocks always have kLaneWarps warps (a warp's place in its block decides its SM sub-partition, so smaller blocks would
// pile up on one); with fewer warps on a chain than that a block holds several chains.
constexpr int kLaneWarps = 4, kLaneMaxCluster = 8;
// Split with the shortest estimated run.  `extra`: cost of the first sweep over a piece relative to the second; `fixed`: what a
// block costs besides its steps (set-up and fold, in steps); `teams`:
// pieces a block holds (a piece is swept by one warp, or by a team of warps that share its states); `cost`: the estimate,
// in steps of a lone warp.
LaneSplit choose_lane_split(long long chains, int steps, float extra, float fixed, int blocks_per_sm, int teams, float* cost = nullptr);

// Time split of the lane backward kernel for a problem whose teams have kLaneWarps / teams warps (ssm_api.cu); pl->bwd_groups
// is set.
void plan_lane_bwd(const ssm_problem_t& p, int teams, Plan* pl, float* cost);
cudaError_t launch_fwd_lane(const ssm_problem_t& prob, const Plan& plan, const FwdParams& p, int mode, cudaStream_t s);
cudaError_t launch_bwd_lane(const ssm_problem_t& prob, const Plan& plan, const BwdParams& p, int mode, cudaStream_t s);

#ifdef __CUDACC__
template <typename IO>
struct LaneRaw;
template <>
struct LaneRaw<float> {
  using T = float;
  static __device__ __forceinline__ T load(const float* p) { return __ldg(p); }
  static __device__ __forceinline__ float widen(T v) { return v; }
};
template <>
struct LaneRaw<__nv_bfloat16> {
  using T = unsigned short;
  static __device__ __forceinline__ T load(const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const unsigned short*>(p)); }
  static __device__ __forceinline__ float widen(T v) { return __uint_as_float((uint32_t)v << 16); }
};

// Four adjacent elements of a B / C row, still in the io dtype.  `n` of them exist; vec: the row pieces are aligned to
// four elements.
template <typename IO>
struct LaneQuad;
template <>
struct LaneQuad<float> {
  float4 v;
  __device__ __forceinline__ void zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ void load(const float* p, int n, bool vec) {
    v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n >= 4 && vec) {
      v = __ldg(reinterpret_cast<const float4*>(p));
    } else {
      if (n > 0) v.x = __ldg(p);
      if (n > 1) v.y = __ldg(p + 1);
      if (n > 2) v.z = __ldg(p + 2);
      if (n > 3) v.w = __ldg(p + 3);
    }
  }
  __device__ __forceinline__ float4 widen() const { return v; }
};
template <>
struct LaneQuad<__nv_bfloat16> {
  uint2 v;
  __device__ __forceinline__ void zero() { v = make_uint2(0u, 0u); }
  __device__ __forceinline__ void load(const __nv_bfloat16* p, int n, bool vec) {
    v = make_uint2(0u, 0u);
    if (n >= 4 && vec) {
      v = __ldg(reinterpret_cast<const uint2*>(p));
    } else {
      const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
      if (n > 0) v.x = __ldg(q);
      if (n > 1) v.x |= (uint32_t)__ldg(q + 1) << 16;
      if (n > 2) v.y = __ldg(q + 2);
      if (n > 3) v.y |= (uint32_t)__ldg(q + 3) << 16;
    }
  }
  __device__ __forceinline__ float4 widen() const { return make_float4(bf16lo(v.x), bf16hi(v.x), bf16lo(v.y), bf16hi(v.y)); }
};

// The warp index, in a form the compiler can see is the same in all lanes
// (a warp reduction lands in a uniform register, so addresses built on it cost no vector instructions)
__device__ __forceinline__ int uniform_warp() { return __reduce_max_sync(0xffffffffu, (int)(threadIdx.x >> 5)); }

template <typename T>
__device__ __forceinline__ T* at_bytes(T* base, unsigned bytes) {
  using C = typename std::conditional<std::is_const<T>::value, const char, char>::type;
  return reinterpret_cast<T*>(reinterpret_cast<C*>(base) + bytes);
}

// A batch of 8 rows of 32 channels of one tensor, in flight from global memory.  VEC (rows are 16-byte aligned): the warp
// reads it with 16-byte loads, 8 / EPV x 32 lanes of them per row, and passes it through shared memory to the lanes that
// own the channels; otherwise every lane reads its own channel row by row.
template <typename IO, bool VEC>
struct LaneRows {
  static constexpr int EPV = 16 / (int)sizeof(IO);   // elements of a 16-byte vector
  static constexpr int VPR = 32 / EPV;               // vectors of a row piece
  static constexpr int NV = kLB * VPR / 32;          // vectors per lane
  using RawT = typename LaneRaw<IO>::T;
  uint4 v[VEC ? NV : 1];
  RawT r[VEC ? 1 : kLB];
  // base: first row of the batch and first channel of the group; `last`: last row that exists (rows past it repeat it);
  // `cols`: channels of the group that exist (lanes past them read existing ones)
  __device__ __forceinline__ void load(const IO* base, int D, int lane, int last, int cols) {
    if constexpr (VEC) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const int q = lane + 32 * i, row = min(q / VPR, last), col = min(q % VPR * EPV, cols - EPV);
        v[i] = __ldg(reinterpret_cast<const uint4*>(base + (size_t)row * D + col));
      }
    } else {
      const IO* p = base + min(lane, cols - 1);
      if (last >= kLB - 1) {
#pragma unroll
        for (int t = 0; t < kLB; ++t) r[t] = LaneRaw<IO>::load(at_bytes(p, (unsigned)t * (unsigned)D * (unsigned)sizeof(IO)));
      } else {
#pragma unroll
        for (int t = 0; t < kLB; ++t)
          r[t] = LaneRaw<IO>::load(at_bytes(p, (unsigned)min(t, last) * (unsigned)D * (unsigned)sizeof(IO)));
      }
    }
  }
  __device__ __forceinline__ void zero() {
    if constexpr (VEC) {
#pragma unroll
      for (int i = 0; i < NV; ++i) v[i] = make_uint4(0u, 0u, 0u, 0u);
    } else {
#pragma unroll
      for (int t = 0; t < kLB; ++t) r[t] = RawT(0);
    }
  }
  // rows `live` .. of the batch (not VEC: they are zeroed in the tile there)
  __device__ __forceinline__ void zero_from(int live) {
#pragma unroll
    for (int t = 0; t < kLB; ++t)
      if (t >= live) r[t] = RawT(0);
  }
  // into the tile [kLB][32] (VEC only)
  __device__ __forceinline__ void put(IO* tile, int lane) const {
    if constexpr (VEC) {
#pragma unroll
      for (int i = 0; i < NV; ++i) reinterpret_cast<uint4*>(tile)[lane + 32 * i] = v[i];
    }
  }
  // this lane's value of row t
  __device__ __forceinline__ float get(const IO* tile, int t, int lane) const {
    if constexpr (VEC) return LaneRaw<IO>::widen(reinterpret_cast<const RawT*>(tile)[t * 32 + lane]);
    else return LaneRaw<IO>::widen(r[t]);
  }
};
// (bounds-checking build) whether a batch from row t0 with `last` as in LaneRows::load, and `cols` channels from c0, exist
template <typename IO, bool VEC>
__device__ __forceinline__ bool lane_rows_exist(int b, int batch, int t0, int last, int L, int c0, int cols, int D) {
  return b >= 0 && b < batch && t0 >= 0 && last >= 0 && t0 + min(last, kLB - 1) < L && c0 >= 0 &&
         cols >= (VEC ? LaneRows<IO, VEC>::EPV : 1) && c0 + cols <= D;
}
// The way back: results of a batch, collected in a tile (VEC) and written with 16-byte stores, or written one by one.
template <typename IO, bool VEC>
struct LaneOut {
  using R = LaneRows<IO, VEC>;
  static __device__ __forceinline__ void put(IO* tile, IO* base, int D, int t, int lane, bool ok, float v) {
    if constexpr (VEC) tile[t * 32 + lane] = float_to_io<IO>(v);
    else if (ok) *at_bytes(base + lane, (unsigned)t * (unsigned)D * (unsigned)sizeof(IO)) = float_to_io<IO>(v);
  }
  // after a __syncwarp
  static __device__ __forceinline__ void flush(const IO* tile, IO* base, int D, int lane, int live, int cols) {
    if constexpr (VEC) {
#pragma unroll
      for (int i = 0; i < R::NV; ++i) {
        const int q = lane + 32 * i, row = q / R::VPR, col = q % R::VPR * R::EPV;
        if (row < live && col < cols)
          *reinterpret_cast<uint4*>(base + (size_t)row * D + col) = reinterpret_cast<const uint4*>(tile)[q];
      }
    }
  }
};

// step size from the staged value: float32 io keeps the precise logarithm
template <typename IO>
__device__ __forceinline__ float lane_softplus(float v) {
  if constexpr (sizeof(IO) == 4) return softplus_precise(v);
  else return softplus_fast(v);
}

// which cluster this block belongs to (the block itself in a launch without clusters), and its place there
__device__ __forceinline__ int cluster_index() {
  unsigned v;
  asm("mov.u32 %0, %%clusterid.x;" : "=r"(v));
  return (int)v;
}
__device__ __forceinline__ int cluster_rank() {
  unsigned v;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
  return (int)v;
}
__device__ __forceinline__ unsigned dynamic_smem_bytes() {
  unsigned v;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
  return v;
}
// x / w for w = 1, 2 or 4
__device__ __forceinline__ int div_pow2(int x, int w) { return x >> (w >> 1); }

// ---- complex states (SSM_FLAG_COMPLEX) in the lane kernels.  N complex states are 2 N columns of the same arrays; a group
// of 16 rows holds 8 of them as two halves of 4 real parts and their 4 imaginary parts, so that packed arithmetic works on
// pairs of real parts and pairs of imaginary parts.  lane_col: the column (re, im interleaved) of row n.
template <bool CPLX>
__device__ __forceinline__ int lane_col(int n) {
  return CPLX ? (n & ~7) + 2 * (n & 3) + ((n >> 2) & 1) : n;
}
// rows (and columns) of a channel's checkpoint
template <bool CPLX>
__host__ __device__ __forceinline__ int lane_ckpt_rows(int N) { return CPLX && N < 8 ? 8 : N; }
// what a row of A is multiplied with when it is staged: real parts for ex2, imaginary parts stay in radians (scaled to turns
// they would carry a rounding of their own, the same in every step of a channel)
template <bool CPLX>
__device__ __forceinline__ float lane_a_scale(int n) { return CPLX && (n & 4) ? 1.f : kLog2e; }
// Four columns of B or C (quad v of a batch of rows of 16 NG) into the staged rows; im_sign: of imaginary parts
template <bool CPLX>
__device__ __forceinline__ void put_quad(float* rows, int v, float4 q, float im_sign) {
  if constexpr (CPLX) {
    // columns 4 v .. 4 v + 3 are two complex states: real parts next to each other, imaginary parts 4 rows on
    float* const at = rows + (v >> 1) * 8 + (v & 1) * 2;
    *reinterpret_cast<float2*>(at) = make_float2(q.x, q.z);
    *reinterpret_cast<float2*>(at + 4) = make_float2(im_sign * q.y, im_sign * q.w);
  } else {
    *reinterpret_cast<float4*>(rows + 4 * v) = q;
  }
}

// Angles are reduced to half a turn the way of Cody and Waite: k whole turns off the unrounded product dt Im A, 2 pi as the
// sum of a number of 8 bits (so that k times it is exact up to k = 2^16) and a rest.
constexpr float kInvTurn = 0.15915494309189534f, kTurnHi = 6.28125f, kTurnLo = 0.0019353071795864769f;
__device__ __forceinline__ float reduce_angle(float s, float aim) {
  const float k = rintf(s * aim * kInvTurn);
  return fmaf(k, -kTurnLo, fmaf(s, aim, k * -kTurnHi));
}
// exp(dt A) for a pair of complex states: magnitude by ex2, phase by sin and cos of the reduced angle.  (Six packed operations
// for the reduction.  With Im A staged in turns, which takes six as well, the state of float32 (8, 512, 2400), N = 8, Re A = 0
// turned by 560 rad was off by 7.0e-5, against 6.3e-5 this way and with each product rounded.)
__device__ __forceinline__ void cexp_pair(float dt, float2 are, float2 aim, float2& ar, float2& ai) {
  const float2 d = f2dup(dt), e = f2mul(d, are);
  const float2 m = make_float2(ex2_approx(e.x), ex2_approx(e.y));
  constexpr float kRound = 12582912.f;   // 1.5 * 2^23: adding it rounds to a whole number
  const float2 k = __fadd2_rn(f2fma(f2mul(d, aim), f2dup(kInvTurn), f2dup(kRound)), f2dup(-kRound));
  const float2 r = f2fma(k, f2dup(-kTurnLo), f2fma(d, aim, f2mul(k, f2dup(-kTurnHi))));
  ar = f2mul(m, make_float2(__cosf(r.x), __cosf(r.y)));
  ai = f2mul(m, make_float2(__sinf(r.x), __sinf(r.y)));
}
__device__ __forceinline__ float2 f2neg(float2 v) { return make_float2(-v.x, -v.y); }
// (re, im) <- exp(s A) (re, im) (conjugate: exp(s conj A)), A as staged
template <bool CONJ>
__device__ __forceinline__ float2 cexp_apply(float s, float are, float aim, float2 v) {
  const float m = ex2_approx(s * are), r = reduce_angle(s, aim);
  const float c = m * __cosf(r), n = (CONJ ? -m : m) * __sinf(r);
  return make_float2(fmaf(c, v.x, -n * v.y), fmaf(c, v.y, n * v.x));
}

// sum += the step sizes of a batch.  Complex: the sum turns the state of a whole piece at once, so its rounding counts as
// often as the piece has radians; it is kept to one rounding by Kahan's compensation (`lost`: what the last addition dropped).
template <bool CPLX>
__device__ __forceinline__ void add_steps(const float (&dt)[kLB], float& sum, float& lost) {
  if constexpr (CPLX) {
    const float batch = ((dt[0] + dt[1]) + (dt[2] + dt[3])) + ((dt[4] + dt[5]) + (dt[6] + dt[7]));
    const float y = batch - lost, t = sum + y;
    lost = (t - sum) - y;
    sum = t;
  } else {
#pragma unroll
    for (int t = 0; t < kLB; ++t) sum += dt[t];
  }
}

// 16 floats of a shared-memory row as packed pairs
__device__ __forceinline__ void load16(const float* row, float2 (&v)[8]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(row + 4 * k);
    v[2 * k] = make_float2(a.x, a.y);
    v[2 * k + 1] = make_float2(a.z, a.w);
  }
}
#endif

}  // namespace ssm
