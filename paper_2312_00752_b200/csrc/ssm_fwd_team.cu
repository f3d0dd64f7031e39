// Forward selective scan for more than 16 states: a team of N / 16 warps per chain of 32 channels (bf16 io, 16-byte aligned
// rows; mathematics as in ssm_fwd.cu).  A lane owns a channel and 16 of its states, as in ssm_fwd_warp.cu, so each warp of the
// team is such a warp for its own 16 states; only what belongs to the channel is shared.
//
// Time goes in tiles of 32 steps.  The warps of a team deal the rows of a tile among themselves: each copies its share
// (16-byte cp.async, two tiles ahead), turns its rows of the next tile into (step size, step size times input) pairs and
// finishes its rows of the tile before (sum of the team's partial readouts, skip term, gate, rounding).  Pairs and partial
// readouts pass through shared memory, double-buffered, behind one barrier of the team per tile.
//
// Schedule: that of ssm_fwd_warp.cu (WarpSched) with a team in the place of a warp.
//
// Bound: as the tuned kernel, the arithmetic and the latencies of a lone warp per sub-partition (a block fills an SM's shared
// memory; counters at (1, 2048, 5120), N = 64: issue slots 40 %, FMA pipe 42 %, fixed latencies 0.79 cycles per instruction; with
// A off the progression the special-function unit 56 %, 1.38 cycles); what a team adds to a step (pairs and readouts through shared memory, the barrier) is about what the gate saves.
// Tiles of 32 steps because the rows passes are chains of latencies that a tile pays once (with 8 steps per barrier 304 us at
// (1, 2048, 5120), N = 64).  There: 201 us, 271 with A off the progression, against 332 and 460 for the lane kernel, which
// sweeps each piece twice and parks the states of three groups in shared memory.  For 16 states split over two or four warps the
// same scheme was slower than one warp (130M width, batch 8: 245 us against 175): 48 instructions per warp and step for 4
// states, 74 for all 16.
#include <type_traits>

#include "ssm_lane.cuh"

namespace ssm {

namespace {

constexpr int kTT = 32;      // steps per tile
constexpr int kStages = 4;   // tiles of rows in shared memory: being finished, computed on, prepared, on their way
using bf16 = __nv_bfloat16;

template <int T>
struct TeamSmem {
  static constexpr int N = 16 * T, R = kTT / T;   // rows of a tile that are a warp's
  uint4 x[kStages][kTT][4], d[kStages][kTT][4], z[kStages][kTT][4];   // 32 channels
  uint4 B[kStages][kTT][2 * T], C[kStages][kTT][2 * T];
  float2 pair[2][kTT][32];        // (step size, step size times input)
  float part[2][T][kTT][32];      // partial readouts
  float4 wide[T][2][2][kTT][4];   // per warp: B and C of its 16 states as floats
};

template <int T>
__global__ void __launch_bounds__(128, 1) ssm_fwd_team_kernel(const FwdParams p, const WarpSched sc) {
  using SM = TeamSmem<T>;
  constexpr int N = SM::N, R = SM::R, TB = 4 / T;   // TB: teams of a block
  extern __shared__ __align__(16) unsigned char smem_raw[];
  dependency_wait();
  const int bwarp = uniform_warp(), lane = threadIdx.x & 31;
  const int team = bwarp / T, w = bwarp - team * T, tid = w * 32 + lane;   // thread of the team
  SM& sm = reinterpret_cast<SM*>(smem_raw)[team];
  auto team_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(32 * T) : "memory"); };

  const bf16* __restrict__ gx = static_cast<const bf16*>(p.x);
  const bf16* __restrict__ gd = static_cast<const bf16*>(p.delta);
  const bf16* __restrict__ gz = static_cast<const bf16*>(p.z);
  const bf16* __restrict__ gB = static_cast<const bf16*>(p.B);
  const bf16* __restrict__ gC = static_cast<const bf16*>(p.C);
  bf16* __restrict__ gout = static_cast<bf16*>(p.out);
  const int D = p.D, L = p.L, groups = (D + 31) / 32;
  const bool has_z = gz != nullptr, has_out = gout != nullptr;
  const int worker = blockIdx.x * TB + team;
  const WorkList wl = make_worklist(sc, worker);
  for (int pi = 0; pi < wl.count; ++pi) {
    int chain, from, to;
    get_piece(wl, sc.tiles, pi, chain, from, to);
    const int b = chain / groups, grp = chain - b * groups;
    const int c_own = grp * 32 + lane;
    const bool valid = c_own < D;
    const int c_ld = valid ? c_own : D - 1;   // lanes past the last channel read it along and store nothing
    const int t_from = from * kTT, t_to = min(L, to * kTT);
    const size_t row_b = (size_t)b * L;

    // ---- rows: this thread's vectors of a tile
    constexpr int XI = kTT * 4 / (32 * T), BI = kTT * 2 * T / (32 * T);   // of x (and delta, z), of B (and C)
    auto issue = [&](int t0) {
      if (t0 < t_to) {
        const int st = t0 / kTT % kStages;
#pragma unroll
        for (int i = 0; i < XI; ++i) {
          const int row = tid / 4 + i * 8 * T, col = tid % 4;
          const bool ok = t0 + row < L && grp * 32 + col * 8 < D;
          const size_t at = ok ? (row_b + t0 + row) * D + grp * 32 + col * 8 : 0;
          SSM_GUARD(at + 8 <= (size_t)p.batch * L * D, p.abort, continue)
          cp_async16(&sm.x[st][row][col], gx + at, ok);
          cp_async16(&sm.d[st][row][col], gd + at, ok);
          cp_async16(&sm.z[st][row][col], (has_z ? gz : gx) + at, ok && has_z);
        }
#pragma unroll
        for (int i = 0; i < BI; ++i) {
          const int row = tid / (2 * T) + i * 16, col = tid % (2 * T);
          const bool ok = t0 + row < L;
          const size_t at = ok ? (row_b + t0 + row) * N + col * 8 : 0;
          SSM_GUARD(at + 8 <= (size_t)p.batch * L * N, p.abort, continue)
          cp_async16(&sm.B[st][row][col], gB + at, ok);
          cp_async16(&sm.C[st][row][col], gC + at, ok);
        }
      }
      cp_async_commit();
    };
    issue(t_from);
    issue(t_from + kTT);

    // ---- constants and the start state
    float2 A2[8], h[8];
    bool ap = !p.general_A;
    {
      float av[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) av[i] = p.A[(size_t)c_ld * N + 16 * w + i];
      const float step = av[1] - av[0], tol = 1e-6f * fabsf(av[15]);
      ap = ap && step <= 0.f;   // (as in ssm_fwd_warp.cu)
#pragma unroll
      for (int k = 2; k < 16; ++k) ap = ap && fabsf(av[k] - (av[0] + (float)k * step)) <= tol;
#pragma unroll
      for (int k = 0; k < 8; ++k) A2[k] = make_float2(av[2 * k] * kLog2e, av[2 * k + 1] * kLog2e);
    }
    ap = __all_sync(0xffffffffu, ap);
    const float a0s = A2[0].x, rs = A2[0].y - A2[0].x;
    const float bias = p.delta_bias != nullptr ? p.delta_bias[c_ld] : 0.f;
    const float Dk = p.Dskip != nullptr ? p.Dskip[c_ld] : 0.f;
    const float gate_off = has_z ? 0.f : 1.f;
    const size_t ck_stride = ckpt_floats_per_step(1, D, N);
    float* ck = p.ckpt != nullptr ? p.ckpt + ckpt_offset(1, b, p.nck, t_from / kCkptSteps, D, N, c_own, 16 * w) : nullptr;
    if (sc.handoff != nullptr) {   // (chains are shared)
      // the earlier part of this chain belongs to the team before; if any warp's wait gives up, the team leaves together
      const int gave_up = from > 0 && !wait_handoff(sc, worker * T + w, lane);
      int any;
      asm volatile("{.reg .pred a, b; setp.ne.s32 a, %1, 0; bar.red.or.pred b, %2, %3, a; selp.s32 %0, 1, 0, b;}"
                   : "=r"(any) : "r"(gave_up), "r"(1 + team), "r"(32 * T) : "memory");
      if (any) {
        cp_async_wait_all();
        return;
      }
    }
    if (from > 0) {
      const float4* const hb = sc.handoff + ((size_t)(worker * T + w) * 32 + lane) * 4;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 v = __ldcg(hb + k);
        h[2 * k] = make_float2(v.x, v.y);
        h[2 * k + 1] = make_float2(v.z, v.w);
      }
    } else {
      const float* const hs = p.h_start != nullptr ? p.h_start + ((size_t)b * D + c_ld) * N + 16 * w : nullptr;
#pragma unroll
      for (int i = 0; i < 16; ++i) reinterpret_cast<float*>(h)[i] = hs != nullptr ? hs[i] : 0.f;
    }

    auto at_lane = [&](const uint4* row) { return LaneRaw<bf16>::widen(reinterpret_cast<const unsigned short*>(row)[lane]); };
    // Eight rows at a time, loads before stores: a load may not pass an earlier store.
    constexpr int RC = R < 8 ? R : 8;
    // this warp's rows of the tile from t0 into pairs; B and C of its states widened
    auto prepare = [&](int t0, int buf) {
      const int st = t0 / kTT % kStages;
#pragma unroll 1
      for (int r0 = w * R; r0 < w * R + R; r0 += RC) {
        float x[RC], dt[RC];
#pragma unroll
        for (int r = 0; r < RC; ++r) {
          x[r] = at_lane(sm.x[st][r0 + r]);
          dt[r] = at_lane(sm.d[st][r0 + r]) + bias;
        }
        if (p.softplus) {
#pragma unroll
          for (int r = 0; r < RC; ++r) dt[r] = softplus_fast(dt[r]);
        }
#pragma unroll
        for (int r = 0; r < RC; ++r) {
          const float v = t0 + r0 + r < L ? dt[r] : 0.f;   // (rows past the end are identity steps; their x is zero)
          sm.pair[buf][r0 + r][lane] = make_float2(v, v * x[r]);
        }
      }
      uint2 q[2][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {   // rows lane / 4 + 8 i, states 4 (lane % 4) ..
        q[0][i] = reinterpret_cast<const uint2*>(sm.B[st][lane / 4 + 8 * i])[4 * w + lane % 4];
        q[1][i] = reinterpret_cast<const uint2*>(sm.C[st][lane / 4 + 8 * i])[4 * w + lane % 4];
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          sm.wide[w][buf][c][lane / 4 + 8 * i][lane % 4] = make_float4(bf16lo(q[c][i].x), bf16hi(q[c][i].x), bf16lo(q[c][i].y), bf16hi(q[c][i].y));
    };
    // this warp's rows of the tile from t0: sum of the partial readouts, skip term, gate
    auto finish = [&](int t0, int buf) {
      if (!has_out) return;
      const int st = t0 / kTT % kStages;
#pragma unroll 1
      for (int r0 = w * R; r0 < w * R + R; r0 += RC) {
        bf16* o = gout + (row_b + t0 + r0) * D + c_ld;
        float y[RC], x[RC], z[RC];
#pragma unroll
        for (int r = 0; r < RC; ++r) {
          y[r] = sm.part[buf][0][r0 + r][lane];
#pragma unroll
          for (int i = 1; i < T; ++i) y[r] += sm.part[buf][i][r0 + r][lane];
          x[r] = at_lane(sm.x[st][r0 + r]);
          z[r] = at_lane(sm.z[st][r0 + r]);
        }
#pragma unroll
        for (int r = 0; r < RC; ++r) {
          const float v = fmaf(Dk, x[r], y[r]) * fmaf(z[r], sigmoid_fast(z[r]), gate_off);   // (without z: silu(0) = 0, and gate_off takes its place)
          if (valid && t0 + r0 + r < L) {
            SSM_GUARD_SPAN(o, 1, gout, (size_t)p.batch * L * D, p.abort, continue)
            *o = __float2bfloat16_rn(v);
          }
          o += D;
        }
      }
    };

    // Eight steps from row r0 of the tile, as in ssm_fwd_warp.cu: exponentials first (general A: of four steps at a time),
    // B, C, decays and input terms of a step one step ahead of its state update, the readout one step behind.
    auto compute = [&](int buf, int r0, auto ap_tag) {
      constexpr bool AP = decltype(ap_tag)::value;
      constexpr int GB = AP ? 8 : 4;
#pragma unroll
      for (int g0 = 0; g0 < kLB; g0 += GB) {
        float du[GB], e0[AP ? GB : 1], e1[AP ? GB : 1];
        float2 af[AP ? 1 : GB][AP ? 1 : 8];
#pragma unroll
        for (int t = 0; t < GB; ++t) {
          const float2 v = sm.pair[buf][r0 + g0 + t][lane];
          du[t] = v.y;
          if constexpr (AP) {
            e0[t] = ex2_approx(v.x * a0s);
            e1[t] = ex2_approx(v.x * rs);
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float2 e = f2mul(f2dup(v.x), A2[k]);
              af[t][k] = make_float2(ex2_approx(e.x), ex2_approx(e.y));
            }
          }
        }
        float2 aN[2][8], bxN[2][8], CvN[3][8];
        auto front = [&](int t, float2 (&a)[8], float2 (&bx)[8], float2 (&Cv)[8]) {
          load16(reinterpret_cast<const float*>(sm.wide[w][buf][0][r0 + g0 + t]), bx);
          load16(reinterpret_cast<const float*>(sm.wide[w][buf][1][r0 + g0 + t]), Cv);
          if constexpr (AP) {
            const float a0 = e0[t], rr = e1[t], r2 = rr * rr, r4 = r2 * r2, r8 = r4 * r4;
            a[0] = make_float2(a0, a0 * rr);
            a[1] = f2mul(a[0], f2dup(r2));
            a[2] = f2mul(a[0], f2dup(r4));
            a[3] = f2mul(a[1], f2dup(r4));
#pragma unroll
            for (int k = 0; k < 4; ++k) a[4 + k] = f2mul(a[k], f2dup(r8));
          } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) a[k] = af[t][k];
          }
          const float2 du2 = f2dup(du[t]);
#pragma unroll
          for (int k = 0; k < 8; ++k) bx[k] = f2mul(du2, bx[k]);
        };
        float y[GB];
        float2 hp[8];
        auto readout = [&](int t, const float2 (&hh)[8]) {
          float2 yv = f2mul(CvN[t % 3][0], hh[0]), yw = f2mul(CvN[t % 3][1], hh[1]);
#pragma unroll
          for (int k = 2; k < 8; ++k) {
            if (k & 1) yw = f2fma(CvN[t % 3][k], hh[k], yw);
            else yv = f2fma(CvN[t % 3][k], hh[k], yv);
          }
          y[t] = (yv.x + yw.x) + (yv.y + yw.y);
        };
        front(0, aN[0], bxN[0], CvN[0]);
#pragma unroll
        for (int t = 0; t < GB; ++t) {
          if (t + 1 < GB) front(t + 1, aN[(t + 1) & 1], bxN[(t + 1) & 1], CvN[(t + 1) % 3]);
#pragma unroll
          for (int k = 0; k < 8; ++k) hp[k] = h[k];
#pragma unroll
          for (int k = 0; k < 8; ++k) h[k] = f2fma(aN[t & 1][k], h[k], bxN[t & 1][k]);
          if (t > 0) readout(t - 1, hp);
          if (t == GB - 1) readout(t, h);
        }
#pragma unroll
        for (int t = 0; t < GB; ++t) sm.part[buf][w][r0 + g0 + t][lane] = y[t];
      }
    };

    asm volatile("cp.async.wait_group 1;" ::: "memory");
    team_sync();
    prepare(t_from, 0);
    cp_async_wait_all();
    team_sync();
    int buf = 0;
#pragma unroll 1
    for (int t0 = t_from; t0 < t_to; t0 += kTT, buf ^= 1) {
      issue(t0 + 2 * kTT);   // (into the rows of the tile that was finished before the last barrier)
      if (t0 > t_from) finish(t0 - kTT, buf ^ 1);
      if (t0 + kTT < t_to) prepare(t0 + kTT, buf ^ 1);
#pragma unroll 1
      for (int r0 = 0; r0 < kTT && t0 + r0 < t_to; r0 += kLB) {
        if (ck != nullptr) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {   // (lanes past the last channel fill the padding of the tiled layout)
            SSM_GUARD_SPAN(ck + 128 * k, 4, p.ckpt, (size_t)p.batch * p.nck * ckpt_floats_per_step(1, D, N), p.abort, continue)
            *reinterpret_cast<float4*>(ck + 128 * k) = make_float4(h[2 * k].x, h[2 * k].y, h[2 * k + 1].x, h[2 * k + 1].y);
          }
          ck += ck_stride;
        }
        if (ap) compute(buf, r0, std::true_type{});
        else compute(buf, r0, std::false_type{});
      }
      cp_async_wait_all();   // (the rows of the tile after the next have landed)
      team_sync();
    }
    finish((t_to - 1) / kTT * kTT, buf ^ 1);
    if (to < sc.tiles) {
      // the rest of this chain belongs to the next team
      float4* const hb = sc.handoff + ((size_t)((worker + 1) * T + w) * 32 + lane) * 4;
#pragma unroll
      for (int k = 0; k < 4; ++k) __stcg(hb + k, make_float4(h[2 * k].x, h[2 * k].y, h[2 * k + 1].x, h[2 * k + 1].y));
      publish_handoff(sc, (worker + 1) * T + w - 1, lane);
    } else if (p.h_last != nullptr && valid) {
      float* const dst = p.h_last + ((size_t)b * D + c_own) * N + 16 * w;
#pragma unroll
      for (int i = 0; i < 16; ++i) dst[i] = reinterpret_cast<const float*>(h)[i];
    }
    team_sync();   // all warps are done with this piece's shared memory
  }
}

template <int T>
cudaError_t launch_team(const FwdParams& p, cudaStream_t s) {
  constexpr int TB = 4 / T;
  auto kern = ssm_fwd_team_kernel<T>;
  const size_t smem = sizeof(TeamSmem<T>) * TB;
  KernelLimits lim{};
  const cudaError_t e = kernel_limits(reinterpret_cast<const void*>(kern), 128, smem, &lim);
  if (e != cudaSuccess) return e;
  WarpSched sc{};
  sc.chains = p.batch * ((p.D + 31) / 32);
  sc.tiles = (p.L + kTT - 1) / kTT;
  // as many teams as there are SM sub-partitions, sharing chains, or a team per chain where that is fewer
  const int resident = lim.sms * TB;
  sc.workers = sc.chains;
  if (sc.chains > resident && lim.per_sm > 0 && p.handoff != nullptr && p.max_workers >= resident * T) sc.workers = resident;
  const long long total = (long long)sc.chains * sc.tiles;
  sc.quota = (int)((total + sc.workers - 1) / sc.workers);
  sc.spin_limit = p.test_withhold ? 1000 : 1 << 22;
  sc.withhold = p.test_withhold;
  if (sc.workers < sc.chains) {
    sc.flags = p.flags;
    sc.abort = p.abort;
    sc.handoff = p.handoff;
  }
  return launch_dependent(kern, (unsigned)((sc.workers + TB - 1) / TB), 128, smem, 1, s, p, sc);
}

}  // namespace

// Pointers the team kernel takes (shapes: team_fwd in ssm_api.cu).
bool fwd_team_applicable(const FwdParams& p) {
  for (const void* q : {p.x, p.delta, p.z, p.B, p.C, (const void*)p.ckpt, (const void*)p.handoff})
    if (reinterpret_cast<uintptr_t>(q) & 15) return false;
  return true;
}

cudaError_t launch_fwd_team(const ssm_problem_t& prob, const FwdParams& p, cudaStream_t s) {
  return prob.N == 32 ? launch_team<2>(p, s) : launch_team<4>(p, s);
}

}  // namespace ssm
