// Forward selective scan, one lane per channel, for everything the tuned bf16 / N = 16 kernel does not take and for the
// problems with too few chains to fill the GPU (mathematics and modes as in ssm_fwd.cu; layout and time split: ssm_lane.cuh).
//
// A lane owns one channel and 16 of its states at a time as packed float2 pairs, so the readout sum over n stays in the
// thread.  With N > 16 the groups of 16 states of a batch run one after the other, their state parked in shared memory;
// everything that belongs to the channel (step size, input, gate, rounding) is done once.
//
// Bound (counters): the special-function unit with its one exponential per state, 70 % busy at float32 (2, 2048, 1536), 67 %
// at bf16 (3, 1237, 1001), 68 % with complex states at (2, 2048, 1536), 62 % at float32 (1, 2048, 2560), N = 64 (two warps per
// sub-partition: the states of four groups take the shared memory).  The issue slots are 35 to 50 % in use.  So the registers
// are capped for three warps per sub-partition and a chain is split in time until they are there.
// Measured against the generic kernel with its summary and carry launches: float32 (2, 2048, 1536), N = 16: 262 -> 75 us;
// bf16 (3, 1237, 1001), N = 16: 268 -> 49 us; float32 (1, 256, 64): 126 -> 7.6 us.  bf16 N = 32 and 64 with enough channels run
// in ssm_fwd_team.cu.
#include <type_traits>

#include "ssm_lane.cuh"

namespace ssm {

namespace {

namespace cg = cooperative_groups;

// shared memory of a block, in floats: per warp, the tiles of two batches (x, delta, z; B, C widened), the output tile,
// the state, the sum of delta; per chain, A * log2(e), the chain's totals over this block (for the other blocks of the
// cluster) and its sum of delta
template <typename IO, int NG>
struct FwdLaneSmem {
  static constexpr int NP = 16 * NG;              // padded states
  static constexpr int kTile = kLB * 32 * (int)sizeof(IO) / 4;
  static constexpr int kBuf = 3 * kTile + 2 * kLB * NP;   // one batch: x | delta | z | B | C
  static constexpr int kIO = 2 * kBuf + kTile;    // floats per warp
  static constexpr int kState = NP * 32;          // floats per warp
  static constexpr int kChain = 2 * kState + 32;  // floats per chain
  static __host__ __device__ constexpr size_t bytes(int warps, int chains) {
    return sizeof(float) * ((size_t)warps * (kIO + kState + 32) + (size_t)chains * kChain);
  }
};

// CPLX: complex states (N is then the number of columns, twice that of states; layout of the rows: lane_col)
template <typename IO, int NG, bool VEC, bool CPLX>
__global__ void __launch_bounds__(kLaneWarps * 32, 3) ssm_fwd_lane_kernel(const FwdParams p, const LaneSplit sp, const int N, const int mode) {
  using SM = FwdLaneSmem<IO, NG>;
  constexpr int NP = SM::NP;
  const bool full = mode == kFwdFull, summary = mode == kFwdSummary;
  extern __shared__ __align__(16) float smem[];
  dependency_wait();
  const int bwarp = uniform_warp(), lane = threadIdx.x & 31;
  const int W = sp.warps, CL = sp.cluster;
  constexpr int nwarps = kLaneWarps;
  SSM_GUARD(W * (nwarps / W) == nwarps && SM::bytes(nwarps, nwarps / W) <= dynamic_smem_bytes() && cluster_rank() < CL, p.abort, return)
  const int sub = div_pow2(bwarp, W), warp = bwarp - sub * W;   // sub: which chain of the block
  float* const sIO = smem + (size_t)bwarp * SM::kIO;
  float* const sE = smem + (size_t)nwarps * SM::kIO + (size_t)sub * W * SM::kState;         // [W][NP][32]
  float* const sDs = smem + (size_t)nwarps * (SM::kIO + SM::kState) + sub * W * 32;         // [W][32]
  float* const sA = smem + (size_t)nwarps * (SM::kIO + SM::kState + 32) + (size_t)sub * SM::kChain;   // [NP][32]
  float* const sTot = sA + SM::kState;                                                      // [NP][32]
  float* const sTotDs = sTot + SM::kState;                                                  // [32]
  float* const sH = sE + (size_t)warp * SM::kState;                 // this warp's states

  const IO* __restrict__ gx = static_cast<const IO*>(p.x);
  const IO* __restrict__ gd = static_cast<const IO*>(p.delta);
  const IO* __restrict__ gz = static_cast<const IO*>(p.z);
  const IO* __restrict__ gB = static_cast<const IO*>(p.B);
  const IO* __restrict__ gC = static_cast<const IO*>(p.C);
  IO* __restrict__ gout = static_cast<IO*>(p.out);

  const int D = p.D;
  const int groups = (D + 31) / 32;
  const int rank = cluster_rank();
  const int chains = p.batch * p.nseg * groups;
  const int chain_id = cluster_index() * div_pow2(nwarps, W) + sub;
  const int chain = min(chain_id, chains - 1);
  const int bs = chain / groups, grp = chain - bs * groups;
  const int b = p.nseg == 1 ? bs : bs / p.nseg, seg = bs - b * p.nseg;
  const int c_own = grp * 32 + lane;
  const bool valid = c_own < D;
  const int c_ld = valid ? c_own : D - 1;       // lanes past the last channel read it along and store nothing
  const int seg_t0 = seg * p.seg_steps;
  const int seg_end = min(p.L, seg_t0 + p.seg_steps);
  const int piece0 = (rank * W + warp) * sp.piece;
  const int t_begin = chain_id < chains ? min(seg_end, seg_t0 + piece0) : seg_end;   // (a spare warp has no steps)
  const int t_end = min(seg_end, t_begin + sp.piece);
  const bool split = W * CL > 1;
  const bool bvec = (reinterpret_cast<uintptr_t>(p.B) & (4 * sizeof(IO) - 1)) == 0;
  const bool cvec = (reinterpret_cast<uintptr_t>(p.C) & (4 * sizeof(IO) - 1)) == 0;
  // (the caller's buffer has any float's alignment; off the 16-byte grid the launch takes the variant without VEC)
  const bool ck_vec = VEC || (reinterpret_cast<uintptr_t>(p.ckpt) & 15) == 0;
  const bool has_z = full && gz != nullptr;
  const int cols = min(32, D - grp * 32);
  const int NC = lane_ckpt_rows<CPLX>(N);

  // One batch in flight from global memory.  read: with z and C.
  LaneRows<IO, VEC> rx, rd, rz;
  LaneQuad<IO> qB[NG], qC[NG];
  const size_t row_b = (size_t)b * p.L;
  if (!has_z) rz.zero();
  auto prefetch = [&](int t0, bool read) {
    const size_t base = (row_b + t0) * D + grp * 32, baseBC = (row_b + t0) * N;
    const int last = t_end - 1 - t0;
    SSM_GUARD((lane_rows_exist<IO, VEC>(b, p.batch, t0, last, p.L, grp * 32, cols, D)), p.abort, return)
    rd.load(gd + base, D, lane, last, cols);
    rx.load(gx + base, D, lane, last, cols);
    if (read && has_z) rz.load(gz + base, D, lane, last, cols);
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const int v = lane + 32 * i, n = 4 * (v % (4 * NG));
      const unsigned o = (unsigned)(min(v / (4 * NG), last) * N + n);
      qB[i].load(gB + baseBC + o, N - n, bvec && N >= 4);
      if (read) qC[i].load(gC + baseBC + o, N - n, cvec && N >= 4);
    }
  };
  // The first batch is requested before anything else is set up.  What leaves the last piece of the launch is wanted by
  // the summary mode only.
  const bool live_piece = t_begin < t_end;
  const bool first_sweep = (split || summary) && (summary || rank * W + warp < W * CL - 1);
  if (live_piece) prefetch(t_begin, full && !first_sweep);

  for (int n = warp; n < NP; n += W) {
    const int col = lane_col<CPLX>(n);
    sA[n * 32 + lane] = col < N ? p.A[(size_t)c_ld * N + col] * lane_a_scale<CPLX>(n) : 0.f;
  }
  __syncthreads();
  float2 A2[8];
  float2 h[8];
  // which groups of 16 have their A in arithmetic progression (falling only: a rising one starts from its smallest decay,
  // which underflows for large steps, and padded states, which continue it, would come to grow)
  unsigned ap_mask = 0;
  if (sizeof(IO) == 2 && !CPLX && !p.general_A) {
#pragma unroll 1
    for (int g = 0; g < NG; ++g) {
      const float* a = sA + g * 512 + lane;
      const int live = min(16, N - 16 * g);
      const float a0 = a[0], step = live > 1 ? a[32] - a0 : 0.f;
      const float tol = 1e-6f * fabsf(a[32 * (live - 1)]);
      bool ok = step <= 0.f;
#pragma unroll
      for (int k = 2; k < 16; ++k) ok = ok && (k >= live || fabsf(a[32 * k] - (a0 + (float)k * step)) <= tol);
      if (__all_sync(0xffffffffu, ok)) ap_mask |= 1u << g;
    }
  }
  if constexpr (NG == 1) {
#pragma unroll
    for (int k = 0; k < 8; ++k) A2[k] = make_float2(sA[(2 * k) * 32 + lane], sA[(2 * k + 1) * 32 + lane]);
  }
  const float bias = p.delta_bias != nullptr ? p.delta_bias[c_ld] : 0.f;
  const float Dk = (full && p.Dskip != nullptr) ? p.Dskip[c_ld] : 0.f;
  const float gate_off = has_z ? 0.f : 1.f;
  float dsum = 0.f, dlost = 0.f;

  auto load_h = [&](int g) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      h[k] = make_float2(sH[(g * 16 + 2 * k) * 32 + lane], sH[(g * 16 + 2 * k + 1) * 32 + lane]);
  };
  auto store_h = [&](int g) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      sH[(g * 16 + 2 * k) * 32 + lane] = h[k].x;
      sH[(g * 16 + 2 * k + 1) * 32 + lane] = h[k].y;
    }
  };

  // One sweep over the warp's piece, whose first batch has been requested.  READ: with readout, gate and output; else the
  // state only.
  auto sweep = [&](auto read_tag, bool write_ckpt) {
    constexpr bool READ = decltype(read_tag)::value;
    if (!live_piece) return;
    int buf = 0;
#pragma unroll 1
    for (int t0 = t_begin; t0 < t_end; t0 += kLB, buf ^= 1) {
      float* const sBuf = sIO + buf * SM::kBuf;
      IO* const tx = reinterpret_cast<IO*>(sBuf);
      IO* const td = reinterpret_cast<IO*>(sBuf + SM::kTile);
      IO* const tz = reinterpret_cast<IO*>(sBuf + 2 * SM::kTile);
      IO* const to = reinterpret_cast<IO*>(sIO + 2 * SM::kBuf);
      float* const fB = sBuf + 3 * SM::kTile;
      float* const fC = fB + kLB * NP;
      const int live = t_end - t0;
      if (live < kLB) {   // rows past the end are identity steps (below), and zero times infinity is not zero
#pragma unroll
        for (int i = 0; i < NG; ++i)
          if ((lane + 32 * i) / (4 * NG) >= live) qB[i].zero();
        if constexpr (!VEC) rx.zero_from(live);
      }
      rd.put(td, lane);
      rx.put(tx, lane);
      if constexpr (VEC) {
        if (live < kLB) {
          __syncwarp();
#pragma unroll 1
          for (int t = live; t < kLB; ++t) tx[t * 32 + lane] = float_to_io<IO>(0.f);
        }
      }
      if constexpr (READ) rz.put(tz, lane);
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const int v = lane + 32 * i;
        put_quad<CPLX>(fB, v, qB[i].widen(), 1.f);
        if constexpr (READ) put_quad<CPLX>(fC, v, qC[i].widen(), -1.f);   // (complex: conj C, what the real part of C h wants)
      }
      if constexpr (VEC) {
        __syncwarp();
        if (t0 + kLB < t_end) prefetch(t0 + kLB, READ);
      }
      float dt[kLB], u[kLB], zf[READ ? kLB : 1], y[READ ? kLB : 1];
#pragma unroll
      for (int t = 0; t < kLB; ++t) {
        dt[t] = rd.get(td, t, lane) + bias;
        u[t] = rx.get(tx, t, lane);
        if constexpr (READ) {
          zf[t] = rz.get(tz, t, lane);
          y[t] = CPLX ? 0.f : Dk * u[t];
        }
      }
      if constexpr (!VEC) {
        if (t0 + kLB < t_end) prefetch(t0 + kLB, READ);
        __syncwarp();
      }
      if (p.softplus) {
#pragma unroll
        for (int t = 0; t < kLB; ++t) dt[t] = lane_softplus<IO>(dt[t]);
      }
      if (live < kLB) {
#pragma unroll
        for (int t = 0; t < kLB; ++t) dt[t] = t < live ? dt[t] : 0.f;
      }
      if constexpr (!READ) add_steps<CPLX>(dt, dsum, dlost);

#pragma unroll 1
      for (int g = 0; g < NG; ++g) {
        if constexpr (NG > 1) load_h(g);
        if (write_ckpt) {
          const int kc = t0 / kCkptSteps;
          if (SSM_IN_RANGE(kc < p.nck, p.abort)) {
            if (NC >= 4) {   // (lanes past the last channel fill the padding of the tiled layout)
              float* dst = p.ckpt + ckpt_offset(1, b, p.nck, kc, D, NC, c_own, 16 * g);
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                if (16 * g + 4 * k < NC) {
                  SSM_GUARD_SPAN(dst + 128 * k, 4, p.ckpt, (size_t)p.batch * p.nck * ckpt_floats_per_step(1, D, NC), p.abort, continue)
                  const float4 q = make_float4(h[2 * k].x, h[2 * k].y, h[2 * k + 1].x, h[2 * k + 1].y);
                  if (ck_vec) {
                    *reinterpret_cast<float4*>(dst + 128 * k) = q;
                  } else {
                    dst[128 * k] = q.x;
                    dst[128 * k + 1] = q.y;
                    dst[128 * k + 2] = q.z;
                    dst[128 * k + 3] = q.w;
                  }
                }
              }
            } else if (valid) {
              float* dst = p.ckpt + ckpt_offset(0, b, p.nck, kc, D, N, c_own, 0);
              SSM_GUARD_SPAN(dst, N, p.ckpt, (size_t)p.batch * p.nck * ckpt_floats_per_step(0, D, N), p.abort, return)
              dst[0] = h[0].x;
              if (N > 1) dst[1] = h[0].y;
            }
          }
        }
        // Decays, input terms and C of a step do not depend on the state: they are prepared one step ahead of the
        // recurrence that consumes them.
        auto run = [&](auto ap_tag) {
          constexpr bool AP = decltype(ap_tag)::value;
          float a0s = 0.f, rs = 0.f;
          if constexpr (AP) {
            a0s = sA[(16 * g) * 32 + lane];
            rs = N - 16 * g > 1 ? sA[(16 * g + 1) * 32 + lane] - a0s : 0.f;
          } else if constexpr (NG > 1) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              A2[k] = make_float2(sA[(16 * g + 2 * k) * 32 + lane], sA[(16 * g + 2 * k + 1) * 32 + lane]);
          }
          float e0[AP ? kLB : 1], e1[AP ? kLB : 1];
#pragma unroll
          for (int t = 0; t < kLB; ++t) {
            if constexpr (AP) {
              e0[t] = ex2_approx(dt[t] * a0s);
              e1[t] = ex2_approx(dt[t] * rs);
            }
          }
          // general A: the exponentials of a step are taken AH steps ahead of its recurrence, between the multiply-adds of
          // the steps before it (complex: pairs k and k + 2 are real and imaginary parts, k = 0, 1, 4, 5).  Four steps'
          // exponentials ahead of four recurrences are no slower, since the other warps of the sub-partition fill in
          // (float32 (2, 2048, 1536) 73.8 us against 74.7, bf16 (1, 2048, 5120), N = 64, trained A 476.7 against 473.6); two
          // steps ahead are worth 1 % in complex states (222.8 -> 220.5 us) and nothing elsewhere
          constexpr int AH = CPLX ? 2 : 1, NA = AH + 1;
          float2 aN[NA][8], bxN[2][8], CvN[2][READ ? 8 : 1];
          auto exps = [&](int t, float2 (&a)[8]) {
            const float dtt = dt[t];
            if constexpr (CPLX) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const int k = (kk & 1) + 4 * (kk >> 1);
                cexp_pair(dtt, A2[k], A2[k + 2], a[k], a[k + 2]);
              }
            } else {
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const float2 e = f2mul(f2dup(dtt), A2[k]);
                a[k] = make_float2(ex2_approx(e.x), ex2_approx(e.y));
              }
            }
          };
          if constexpr (!AP) {
#pragma unroll
            for (int t = 0; t < AH; ++t) exps(t, aN[t]);
          }
          auto front = [&](int t, float2 (&a)[8], float2 (&bx)[8], float2 (&Cv)[READ ? 8 : 1]) {
            load16(fB + t * NP + 16 * g, bx);
            if constexpr (READ) load16(fC + t * NP + 16 * g, Cv);
            if constexpr (AP) {
              const float a0 = e0[t], rr = e1[t], r2 = rr * rr, r4 = r2 * r2, r8 = r4 * r4;
              a[0] = make_float2(a0, a0 * rr);
              a[1] = f2mul(a[0], f2dup(r2));
              a[2] = f2mul(a[0], f2dup(r4));
              a[3] = f2mul(a[1], f2dup(r4));
#pragma unroll
              for (int k = 0; k < 4; ++k) a[4 + k] = f2mul(a[k], f2dup(r8));
            }
            const float2 du2 = f2dup(dt[t] * u[t]);
#pragma unroll
            for (int k = 0; k < 8; ++k) bx[k] = f2mul(du2, bx[k]);
          };
          front(0, aN[0], bxN[0], CvN[0]);
#pragma unroll
          for (int t = 0; t < kLB; ++t) {
            if constexpr (!AP) {
              if (t + AH < kLB) exps(t + AH, aN[(t + AH) % NA]);
            }
            if (t + 1 < kLB) front(t + 1, aN[(t + 1) % NA], bxN[(t + 1) & 1], CvN[(t + 1) & 1]);
            float2 yv = make_float2(0.f, 0.f), yw = yv;
            if constexpr (CPLX) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const int k = (kk & 1) + 4 * (kk >> 1);
                const float2 ar = aN[t % NA][k], ai = aN[t % NA][k + 2], hr = h[k], hi = h[k + 2];
                h[k] = f2fma(f2neg(ai), hi, f2fma(ar, hr, bxN[t & 1][k]));
                h[k + 2] = f2fma(ai, hr, f2fma(ar, hi, bxN[t & 1][k + 2]));
              }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              if constexpr (!CPLX) h[k] = f2fma(aN[t % NA][k], h[k], bxN[t & 1][k]);
              if constexpr (READ) {
                if (k & 1) yw = f2fma(CvN[t & 1][k], h[k], yw);
                else yv = f2fma(CvN[t & 1][k], h[k], yv);
              }
            }
            if constexpr (READ) y[t] += (yv.x + yw.x) + (yv.y + yw.y);
          }
        };
        if constexpr (sizeof(IO) == 2 && !CPLX) {
          if (ap_mask >> g & 1) run(std::true_type{});
          else run(std::false_type{});
        } else {
          run(std::false_type{});
        }
        if constexpr (NG > 1) store_h(g);
      }
      if constexpr (READ) {
        IO* const bo = gout + (row_b + t0) * D + grp * 32;
        SSM_GUARD_SPAN(bo + (size_t)(min(live, kLB) - 1) * D, cols, gout, (size_t)p.batch * p.L * D, p.abort, return)
#pragma unroll
        for (int t = 0; t < kLB; ++t) {
          // without z its rows are zero: silu(0) = 0, and gate_off = 1 takes its place
          const float yt = CPLX ? fmaf(Dk, u[t], 2.f * y[t]) : y[t];   // (s = 2 Re(sum C h) + D x)
          const float v = yt * fmaf(zf[t], sigmoid_fast(zf[t]), gate_off);
          LaneOut<IO, VEC>::put(to, bo, D, t, lane, valid && t < live, v);
        }
        if constexpr (VEC) {
          __syncwarp();
          LaneOut<IO, VEC>::flush(to, bo, D, lane, live, cols);
        }
      }
    }
  };

  // ---- first sweep and the fold over the pieces (only if the chain or the launch is split)
  const size_t seg_row = ((size_t)b * p.nseg + seg) * D;
  if (split || summary) {
#pragma unroll
    for (int k = 0; k < 8; ++k) h[k] = make_float2(0.f, 0.f);
    if constexpr (NG > 1) {
      for (int g = 0; g < NG; ++g) store_h(g);
    }
    if (first_sweep) sweep(std::false_type{}, false);
    if (first_sweep && live_piece && !summary) prefetch(t_begin, full);
    if constexpr (NG == 1) store_h(0);
    sDs[warp * 32 + lane] = dsum;
    __syncthreads();
    // exclusive fold over the block's pieces from a zero inflow, and the block's totals (a complex state: rows n and n + 4)
    constexpr int kRow2 = 4 * 32;
    for (int n = warp; n < NP; n += W) {
      if (CPLX && (n & 4)) continue;
      const float a2 = sA[n * 32 + lane], ai = CPLX ? sA[n * 32 + kRow2 + lane] : 0.f;
      float2 pre = make_float2(0.f, 0.f);
      float ds = 0.f;
      float2 e[kLaneWarps];
      float d[kLaneWarps];
#pragma unroll
      for (int w = 0; w < kLaneWarps; ++w) {   // (all loaded before the first is used)
        const float* const at = sE + (size_t)(w < W ? w : 0) * SM::kState + n * 32 + lane;
        e[w] = make_float2(*at, CPLX ? at[kRow2] : 0.f);
        d[w] = sDs[(w < W ? w : 0) * 32 + lane];
      }
#pragma unroll
      for (int w = 0; w < kLaneWarps; ++w) {
        if (w < W) {
          float* const at = sE + (size_t)w * SM::kState + n * 32 + lane;
          *at = pre.x;
          if (CPLX) at[kRow2] = pre.y;
          const float2 q = CPLX ? cexp_apply<false>(d[w], a2, ai, pre) : make_float2(ex2_approx(a2 * d[w]) * pre.x, 0.f);
          pre = make_float2(q.x + e[w].x, q.y + e[w].y);
          ds += d[w];
        }
      }
      sTot[n * 32 + lane] = pre.x;
      if (CPLX) sTot[n * 32 + kRow2 + lane] = pre.y;
      if (n == 0) sTotDs[lane] = ds;
    }
    if (CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    // add the inflow of the block: the segment's start state behind the totals of the blocks before it
    for (int n = warp; n < NP; n += W) {
      if (CPLX && (n & 4)) continue;
      const int col = lane_col<CPLX>(n);
      const float a2 = sA[n * 32 + lane], ai = CPLX ? sA[n * 32 + kRow2 + lane] : 0.f;
      auto step = [&](float d, float2 v) {
        return CPLX ? cexp_apply<false>(d, a2, ai, v) : make_float2(ex2_approx(a2 * d) * v.x, 0.f);
      };
      float2 H = make_float2(0.f, 0.f);
      if (p.h_start != nullptr && col < N) {
        H.x = p.h_start[(seg_row + c_ld) * N + col];
        if (CPLX) H.y = p.h_start[(seg_row + c_ld) * N + col + 1];
      }
      float2 rt[kLaneMaxCluster - 1];
      float ds_all = 0.f, rds[kLaneMaxCluster - 1];
#pragma unroll
      for (int r = 0; r < kLaneMaxCluster - 1; ++r) {   // (all requested before the first is used)
        if (r < rank) {
          const float* const tot = cg::this_cluster().map_shared_rank(sTot, r) + n * 32 + lane;
          rt[r] = make_float2(tot[0], CPLX ? tot[kRow2] : 0.f);
          rds[r] = cg::this_cluster().map_shared_rank(sTotDs, r)[lane];
        }
      }
#pragma unroll
      for (int r = 0; r < kLaneMaxCluster - 1; ++r) {
        if (r < rank) {
          const float2 q = step(rds[r], H);
          H = make_float2(q.x + rt[r].x, q.y + rt[r].y);
          ds_all += rds[r];
        }
      }
      if (summary && rank == CL - 1 && valid && col < N && chain_id < chains) {   // (never complex: no launch is split)
        const float d = sTotDs[lane];
        p.seg_end[(seg_row + c_own) * N + col] = step(d, H).x + sTot[n * 32 + lane];
        if (n == 0) p.seg_dsum[seg_row + c_own] = ds_all + d;
      }
      float2 e[kLaneWarps];
      float cum[kLaneWarps + 1];
      cum[0] = 0.f;
#pragma unroll
      for (int w = 0; w < kLaneWarps; ++w) {
        const float* const at = sE + (size_t)(w < W ? w : 0) * SM::kState + n * 32 + lane;
        e[w] = make_float2(*at, CPLX ? at[kRow2] : 0.f);
        cum[w + 1] = cum[w] + sDs[(w < W ? w : 0) * 32 + lane];
      }
#pragma unroll
      for (int w = 0; w < kLaneWarps; ++w) {
        if (w < W) {
          float* const at = sE + (size_t)w * SM::kState + n * 32 + lane;
          const float2 q = step(cum[w], H);
          *at = e[w].x + q.x;
          if (CPLX) at[kRow2] = e[w].y + q.y;
        }
      }
    }
    if (CL > 1) cg::this_cluster().sync();   // (also: no block leaves while another still reads its totals)
    else __syncthreads();
    if constexpr (NG == 1) load_h(0);
  } else {
    for (int n = 0; n < NP; ++n) {
      const int col = lane_col<CPLX>(n);
      sH[n * 32 + lane] = (p.h_start != nullptr && col < N) ? p.h_start[(seg_row + c_ld) * N + col] : 0.f;
    }
    if constexpr (NG == 1) load_h(0);
  }
  if (summary) return;

  // ---- the sweep proper
  if (full) sweep(std::true_type{}, p.ckpt != nullptr);
  else sweep(std::false_type{}, true);
  if (full && p.h_last != nullptr && valid && t_begin < t_end && t_end == p.L) {
    if constexpr (NG == 1) store_h(0);
    for (int n = 0; n < NP; ++n) {
      const int col = lane_col<CPLX>(n);
      if (col < N) p.h_last[((size_t)b * D + c_own) * N + col] = sH[n * 32 + lane];
    }
  }
}

template <typename IO, int NG, bool VEC, bool CPLX>
cudaError_t launch_fwd_lane_n(const Plan& plan, const FwdParams& p, int N, int mode, cudaStream_t s) {
  auto kern = ssm_fwd_lane_kernel<IO, NG, VEC, CPLX>;
  const int steps = plan.nseg > 1 ? plan.seg_steps : p.L;
  const long long chains = (long long)p.batch * plan.nseg * ((p.D + 31) / 32);
  const LaneSplit sp = choose_lane_split(chains, steps, 0.75f, 25.f, NG > 2 ? 2 : 3, kLaneWarps);
  const int per_block = kLaneWarps / sp.warps;
  const size_t smem = FwdLaneSmem<IO, NG>::bytes(kLaneWarps, per_block);
  KernelLimits lim;
  const cudaError_t e = kernel_limits(reinterpret_cast<const void*>(kern), 32 * kLaneWarps, FwdLaneSmem<IO, NG>::bytes(kLaneWarps, kLaneWarps), &lim);
  if (e != cudaSuccess) return e;
  return launch_dependent(kern, (unsigned)((chains + per_block - 1) / per_block * sp.cluster), 32 * kLaneWarps, smem, sp.cluster, s, p, sp, N, mode);
}

template <typename IO, int NG, bool CPLX>
cudaError_t launch_fwd_lane_vec(const Plan& plan, const FwdParams& p, int N, int mode, cudaStream_t s) {
  // 16-byte row pieces need aligned rows and at least one whole vector of channels; checkpoints that are not aligned go
  // with rows that are not, so that the common variant carries no test (it cost 1 % at bf16 (1, 2048, 5120), N = 64)
  bool vec = (size_t)p.D * sizeof(IO) % 16 == 0;
  for (const void* q : {p.x, p.delta, p.z, (const void*)p.out, (const void*)p.ckpt}) vec = vec && (reinterpret_cast<uintptr_t>(q) & 15) == 0;
  return vec ? launch_fwd_lane_n<IO, NG, true, CPLX>(plan, p, N, mode, s) : launch_fwd_lane_n<IO, NG, false, CPLX>(plan, p, N, mode, s);
}

template <typename IO, bool CPLX>
cudaError_t launch_fwd_lane_io(const Plan& plan, const FwdParams& p, int N, int mode, cudaStream_t s) {
  if (N <= 16) return launch_fwd_lane_vec<IO, 1, CPLX>(plan, p, N, mode, s);
  if (N <= 32) return launch_fwd_lane_vec<IO, 2, CPLX>(plan, p, N, mode, s);
  return launch_fwd_lane_vec<IO, 4, CPLX>(plan, p, N, mode, s);
}

}  // namespace

LaneSplit choose_lane_split(long long chains, int steps, float extra, float fixed, int blocks_per_sm, int teams, float* cost) {
  // run time of 1, 2, 3 warps on a sub-partition relative to one (measured on these kernels)
  static const float slow[4] = {1.0f, 1.0f, 1.5f, 2.1f};
  LaneSplit best{1, 1, (steps + kLB - 1) / kLB * kLB};
  float best_t = 0.f;
  for (int cl = 1; cl <= kLaneMaxCluster; cl *= 2) {
    for (int w = cl > 1 ? teams : 1; w <= teams; w *= 2) {
      const int pieces = cl * w;
      const int piece = ((steps + pieces - 1) / pieces + kLB - 1) / kLB * kLB;
      if (pieces > 1 && (long long)piece * (pieces - w) >= steps) continue;   // the last block would be idle
      const long long blocks = (chains * w + teams - 1) / teams * cl;
      const long long per = (blocks + kNumSMs - 1) / kNumSMs;     // blocks on the fullest SM
      // (blocks of a last wave that is not full start as soon as any block ends: between the whole and the exact number)
      const float exact = (float)blocks / (float)(kNumSMs * blocks_per_sm);
      const float waves = exact <= 1.f ? 1.f : 0.5f * (exact + (float)((per + blocks_per_sm - 1) / blocks_per_sm));
      const float block = (float)piece * (pieces > 1 ? 1.f + extra : 1.f) + (pieces > 1 ? fixed : 0.5f * fixed) + (cl > 1 ? 0.3f * fixed : 0.f);
      const float t = block * slow[per < blocks_per_sm ? per : blocks_per_sm] * waves;
      if (best_t == 0.f || t < best_t) {
        best_t = t;
        best = LaneSplit{w, cl, piece};
      }
    }
  }
  if (cost != nullptr) *cost = best_t;
  return best;
}

bool fwd_lane_applicable(const FwdParams& p) {
  return !p.zoh && !p.static_B && !p.static_C;
}

cudaError_t launch_fwd_lane(const ssm_problem_t& prob, const Plan& plan, const FwdParams& p, int mode, cudaStream_t s) {
  const bool bf = prob.io_dtype == SSM_BF16;
  if (prob.flags & SSM_FLAG_COMPLEX)
    return bf ? launch_fwd_lane_io<__nv_bfloat16, true>(plan, p, 2 * prob.N, mode, s) : launch_fwd_lane_io<float, true>(plan, p, 2 * prob.N, mode, s);
  return bf ? launch_fwd_lane_io<__nv_bfloat16, false>(plan, p, prob.N, mode, s) : launch_fwd_lane_io<float, false>(plan, p, prob.N, mode, s);
}

}  // namespace ssm
