// Kernels and launch helpers shared by the library's translation units:
// the per-grasp shared-memory layout, the batched-QP kernel, the fused
// step kernel and the several-job kernel.  bodex.cu holds the C ABI and the
// small kernels; qp.cu, fused_m3.cu, fused_m4.cu, fused_m5.cu,
// fused_multi.cu and fused_multi_pull.cu instantiate the heavy kernels, so
// that nvcc compiles them in parallel.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <map>
#include <mutex>
#include <string>

#include "../../include/bodex.h"
#include "bodex_device.cuh"

namespace bodex {
// error state of the C ABI (bodex.cu)
int fail(int code, const std::string& msg);
int cuda_fail(cudaError_t e, const char* where);
int launch_err(const char* what);
}  // namespace bodex

using namespace bodex;

// ============================================================================ shared-memory layout
constexpr int CTA_LANES = 96;

__host__ __device__ constexpr int align4(int v) { return (v + 3) & ~3; }

template <int M>
struct Lay {
  static constexpr int NV = 3 * M, NC = 9 * M + 1, NVP = (NV + 3) & ~3;
  // K^-1 block per grasp (packed upper triangle in whole float4s); the
  // stride is skewed (== 20 mod 32 words) so that lanes of two or three
  // grasps in one warp hit disjoint banks.
  static constexpr int KT = 4 * Admm<M>::NTRI4;
  static constexpr int KS = KT + ((20 - KT % 32) + 32) % 32;
  static constexpr int CTW = 24;  // floats per contact record
  static constexpr int oG = 0;
  static constexpr int oK = align4(oG + 6 * NV);  // K^-1 setup scratch (16-byte aligned)
  static constexpr int oCT = oK + WoodburyScratch<M, double>::floats;
  // per-lane record of the QP outputs: r_j (6; read as a float4 and a
  // float2 by the dE/dG reduction, so records start on 16-byte boundaries),
  // two pad words, then y_j
  static constexpr int RYW = 8 + NVP;
  static constexpr int oRY = oCT + CTW * M;
  static constexpr int oQ = oRY + SMAX * RYW;
  static constexpr int oDG = oQ + SMAX;
  static constexpr int oCB = oDG + 6 * NV;
  static constexpr int oX = oCB + M * (6 + MAXCHAIN);
  static constexpr int oAM = oX + MAXD;
  static constexpr int oAV = oAM + MAXD;
  static constexpr int oJW = oAV + MAXD;  // chain joint axes/points, M x MAXCHAIN x 6
  static constexpr int oGC = oJW + M * MAXCHAIN * 6;  // collision gradient [MAXD], energy by lane [SMAX]
  static constexpr int oSC = oGC + MAXD + SMAX;
  // collision scratch: link frames in the K^-1 setup scratch, sphere centres
  // and slot sums in the r / Q / dE/dG block (both dead before A4)
  static constexpr int COLL_FR = WoodburyScratch<M, double>::floats;
  static constexpr int COLL_CS = SMAX * RYW + SMAX + 6 * NV;
  // per-grasp stride == 12 (mod 32) words: the two or three grasps that
  // share a warp then map the same offset to different banks
  static constexpr int PER = align4(oSC + 4) + ((12 - align4(oSC + 4) % 32) + 32) % 32;
  static constexpr int HAND_WORDS = align4((int)(sizeof(HandDev) / 4));
  static size_t bytes(int gpb) { return 4u * (size_t)(HAND_WORDS + gpb * (KS + PER)); }
};

// Contact record in shared memory: c(3) p(3) n(3) phi g(3) h(6) cell(3) degenerate.
__device__ __forceinline__ void store_ct(float* r, const ContactGeo& k) {
  for (int a = 0; a < 3; ++a) {
    r[a] = k.c[a];
    r[3 + a] = k.p[a];
    r[6 + a] = k.n[a];
    r[10 + a] = k.g[a];
    r[19 + a] = __int_as_float(k.cell[a]);
  }
  r[9] = k.phi;
  for (int e = 0; e < 6; ++e) r[13 + e] = k.h[e];
  r[22] = __int_as_float(k.degenerate);
}
__device__ __forceinline__ ContactGeo load_ct(const float* r) {
  ContactGeo k;
  for (int a = 0; a < 3; ++a) {
    k.c[a] = r[a];
    k.p[a] = r[3 + a];
    k.n[a] = r[6 + a];
    k.g[a] = r[10 + a];
    k.cell[a] = __float_as_int(r[19 + a]);
  }
  k.phi = r[9];
  for (int e = 0; e < 6; ++e) k.h[e] = r[13 + e];
  k.degenerate = __float_as_int(r[22]);
  return k;
}

__device__ __forceinline__ void copy_hand_to_smem(const HandDev* src, float* dst) {
  const int* s = reinterpret_cast<const int*>(src);
  int* d = reinterpret_cast<int*>(dst);
  const int words = (int)(sizeof(HandDev) / 4);
  for (int i = threadIdx.x; i < words; i += blockDim.x) d[i] = __ldg(s + i);
}

__device__ __forceinline__ bool finite3(const float* v) {
  return isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]);
}

// ============================================================================ per-grasp QP setup (shared by kernels)
// K^-1 of every grasp of the CTA (Woodbury form, all lanes); must be called
// by every thread of the CTA (contains barriers).
// Double precision when the host asks for it (solves that iterate to a
// tight residual target), single precision otherwise; the branch is
// uniform per launch.
template <int M, bool UNROLL = false, bool ENTRIES = false>
__device__ inline void setup_kinv(bool active, int lane, int S, const float* Gs, float* scratch, float* Kinv,
                                  const AdmmCfg& cfg) {
  if (cfg.fp64_setup) setup_kinv_woodbury<M, double, false, ENTRIES>(active, lane, S, Gs, scratch, Kinv, cfg);
  else setup_kinv_woodbury<M, float, UNROLL, ENTRIES>(active, lane, S, Gs, scratch, Kinv, cfg);
}

// ============================================================================ kernel: batched QP
// One QP per thread, the grasps' K^-1 shared by their QPs.  QPs converge
// after very different iteration counts (at 1e-5 on the paper geometry the
// median is 400, the slowest of a warp's 32 about 3100), and a warp runs
// until its last QP stops.  So at every residual check the QPs still running
// are repacked, through shared memory, into the lowest warps of the CTA: a
// warp whose QPs all stopped waits at the barrier and issues nothing while
// the others iterate.  A QP carries its iterate, -q, its iteration count and
// its slot (grasp, wrench); K^-1, G and rho stay with the grasp.
// The last QPs of a CTA (at most 32 / m a warp: 18 of 96 for m = 5) run in
// the wide form (Wide, bodex_device.cuh), m lanes each, over as few warps as
// hold them, repacked as they finish: alone on its scheduler a QP's iteration
// is bound by its chain of dependent instructions, and the slowest QPs run
// thousands.  With the rows of K^-1 in registers and every warp taking
// groups the 49,152 five-contact QPs take 1.85 ms (2.45 with the rows in
// shared memory and the last six QPs on warp 0).  A batch small enough runs
// in the wide form from the start (run_qp): 67 grasps of four contacts with
// the elliptic cone 2.31 -> 1.67 ms.
//
// Shared memory: alpha K^-1 per grasp (stride as in the fused kernel), the
// per-grasp block (G, Woodbury scratch, votes, rho), the parking area (one
// record per QP) and one count per warp.
template <int M, int CONE>
struct LayQP {
  static constexpr int NV = 3 * M, NC = CONE == CONE_SOC ? 4 * M + 1 : 9 * M + 1;
  static constexpr int KS = Lay<M>::KS;
  static constexpr int oG = 0;
  static constexpr int oK = align4(6 * NV);  // Woodbury scratch (16-byte aligned)
  static constexpr int oVote = oK + WoodburyScratch<M, double>::floats;
  static constexpr int oRho = oVote + SMAX;  // the grasp's rho; oRho + 1: its rho before the last vote
  static constexpr int PER0 = align4(oRho + 2);
  static constexpr int PER = PER0 + ((12 - PER0 % 32) + 32) % 32;
  // parked QP: y, w, -q, then (iterations, slot); an odd count of float4s
  // per record keeps eight consecutive records on distinct banks
  static constexpr int pW = align4(NV), pM = pW + align4(NC), pI = pM + align4(NV);
  static constexpr int PW0 = pI + 4;
  static constexpr int PW = (PW0 / 4) % 2 ? PW0 : PW0 + 4;
  static constexpr int QPW = Wide<M, CONE>::QPW, WPC = Wide<M, CONE>::WPC;  // wide form: QPs per warp, w rows per contact
  static size_t bytes(int gpb, int s) { return 4u * ((size_t)gpb * (KS + PER) + (size_t)gpb * s * PW + 32); }
};

template <int M, int CONE, bool ADAPT>
__global__ void __launch_bounds__(CTA_LANES, 4) qp_solve_kernel(const float* __restrict__ Gin, int B,
                                                                const float* __restrict__ T, int S, int GPB,
                                                                AdmmCfg cfg, int warm, float* yio, float* zio, float* lio,
                                                                float* Qout, int32_t* iters_out, int32_t* status_out,
                                                                float* res_out) {
  using L = LayQP<M, CONE>;
  constexpr int NV = L::NV, NC = L::NC;
  extern __shared__ __align__(16) float smem[];
  // setup role of this thread: lane `lane` of grasp gl of the CTA
  const int gl = threadIdx.x / S, lane = threadIdx.x % S;
  const bool role = (gl < GPB) && (blockIdx.x * GPB + gl < B);
  float* const park = smem + GPB * (L::KS + L::PER);
  int* const wcount = reinterpret_cast<int*>(park + GPB * S * L::PW);
  auto kin = [&](int g) { return smem + g * L::KS; };
  auto per = [&](int g) { return smem + GPB * L::KS + g * L::PER; };
  if (role) {
    const size_t b = (size_t)blockIdx.x * GPB + gl;
    for (int e = lane; e < 6 * NV; e += S) per(gl)[L::oG + e] = Gin[b * 6 * NV + e];
    if (lane == 0) per(gl)[L::oRho] = per(gl)[L::oRho + 1] = cfg.rho;
  }
  __syncthreads();
  setup_kinv<M>(role, lane, S, per(gl) + L::oG, per(gl) + L::oK, kin(gl), cfg);
  constexpr bool adaptive = ADAPT;  // cfg.eps > 0 and cfg.adapt
  const int check = cfg.eps > 0.f ? cfg.check : cfg.iters;  // without a target: residuals once, at the end
  const size_t q0 = (size_t)blockIdx.x * GPB * S;         // first QP of the CTA
  // the QP this thread runs: slot p = g * S + j of the CTA (at first its own), -1 for none
  int p = role ? (int)threadIdx.x : -1;
  int it = 0;
  float y[NV], w[NC], mq[NV];
  if (p >= 0) {
    float t[6];
#pragma unroll
    for (int r = 0; r < 6; ++r) t[r] = T[lane * 6 + r];
    neg_q<M>(per(gl) + L::oG, t, cfg.beta, mq);
    const size_t q = q0 + p;
    if (warm) {
#pragma unroll
      for (int a = 0; a < NV; ++a) y[a] = yio[q * NV + a];
#pragma unroll
      for (int r = 0; r < NC; ++r) w[r] = zio[q * NC + r] + lio[q * NC + r] / cfg.rho;
    } else {
#pragma unroll
      for (int a = 0; a < NV; ++a) y[a] = 0.f;
#pragma unroll
      for (int r = 0; r < NC; ++r) w[r] = 0.f;
    }
  }
  // Q, iterations, residuals and status of slot pp at the point yy
  auto finish = [&](int pp, const float (&yy)[NV], float rp, float rd, bool conv) {
    const int g = pp / S, j = pp % S;
    const size_t q = q0 + pp;
    const float* Gg = per(g) + L::oG;
    float Q = 0.f;
    bool fin = true;
#pragma unroll
    for (int r = 0; r < 6; ++r) {
      float s = cfg.beta * T[j * 6 + r];
#pragma unroll
      for (int a = 0; a < NV; ++a) s = fmaf(-Gg[r * NV + a], yy[a], s);
      Q = fmaf(s, s, Q);
    }
#pragma unroll
    for (int a = 0; a < NV; ++a) {
      fin = fin && isfinite(yy[a]);
      Q = fmaf(cfg.eps_reg * yy[a], yy[a], Q);  // regularised value when eps_reg > 0
    }
    Qout[q] = Q;
    if (iters_out) iters_out[q] = it;
    if (res_out) {
      res_out[2 * q] = rp;
      res_out[2 * q + 1] = rd;
    }
    int st = 0;
    if (!fin || !isfinite(Q)) st |= BODEX_ST_NONFINITE;
    if (cfg.eps > 0.f && !conv) st |= BODEX_ST_NOT_CONVERGED;
    if (status_out) status_out[q] = st;
  };
  // y, z = Pi(w) and lam = rho (w - Pi(w)) of the one-lane form, then the rest
  auto finish_lane = [&](int pp, float rp, float rd, bool conv) {
    const size_t q = q0 + pp;
    const float rho = per(pp / S)[L::oRho];
#pragma unroll
    for (int a = 0; a < NV; ++a) yio[q * NV + a] = y[a];
#pragma unroll
    for (int r = 0; r < NC; ++r) {
      const float pr = CONE == CONE_SOC ? proj_row_soc<M>(w, r, cfg.gamma) : proj_row<M>(w[r], r, cfg.gamma);
      zio[q * NC + r] = pr;
      lio[q * NC + r] = rho * (w[r] - pr);
    }
    finish(pp, y, rp, rd, conv);
  };
  // parking record r: the iterate, -q, the iteration count and the slot
  auto park_store = [&](int r) {
    float* rec = park + r * L::PW;
#pragma unroll
    for (int a = 0; a < NV; ++a) rec[a] = y[a];
#pragma unroll
    for (int k = 0; k < NC; ++k) rec[L::pW + k] = w[k];
#pragma unroll
    for (int a = 0; a < NV; ++a) rec[L::pM + a] = mq[a];
    reinterpret_cast<int*>(rec)[L::pI] = it;
    reinterpret_cast<int*>(rec)[L::pI + 1] = p;
  };
  auto park_load = [&](int r) {
    const float* rec = park + r * L::PW;
#pragma unroll
    for (int a = 0; a < NV; ++a) y[a] = rec[a];
#pragma unroll
    for (int k = 0; k < NC; ++k) w[k] = rec[L::pW + k];
#pragma unroll
    for (int a = 0; a < NV; ++a) mq[a] = rec[L::pM + a];
    it = reinterpret_cast<const int*>(rec)[L::pI];
    p = reinterpret_cast<const int*>(rec)[L::pI + 1];
  };
  // adaptive rho, one decision per grasp (lane 0 of its setup role): rho
  // moves by the geometric mean of its running QPs' proposals when that is
  // more than 5x (clamped to [1e-6, 1e6]); returns whether it moved
  auto decide = [&]() -> bool {
    if (!(role && lane == 0)) return false;
    float* pg = per(gl);
    float sh = 0.f;
    int cnt = 0;
    for (int j = 0; j < S; ++j) {
      const float v = pg[L::oVote + j];
      sh += v;
      cnt += v != 0.f;
    }
    const float cur = pg[L::oRho];
    float nxt = cur;
    if (cnt > 0 && fabsf(sh / cnt) > 1.6094379f)  // log 5
      nxt = fminf(fmaxf(cur * __expf(sh / cnt), 1e-6f), 1e6f);
    pg[L::oRho + 1] = cur;
    pg[L::oRho] = nxt;
    return nxt != cur;
  };
  // K^-1 of the grasps whose rho moved (every thread; barriers inside)
  auto rebuild = [&]() {
    AdmmCfg cl = cfg;
    bool upd = false;
    if (role) {
      cl.rho = per(gl)[L::oRho];
      upd = cl.rho != per(gl)[L::oRho + 1];
    }
    setup_kinv<M>(upd, lane, S, per(gl) + L::oG, per(gl) + L::oK, kin(gl), cl);
  };
  const int warp = threadIdx.x / 32, wl = threadIdx.x % 32;
  const int nw = min(32, (int)blockDim.x - 32 * warp);
  const unsigned wmask = nw == 32 ? 0xffffffffu : (1u << nw) - 1u;  // this warp's threads
  int warps = (blockDim.x + 31) / 32;                                  // warps that hold running QPs
  const int wide_warps = blockDim.x / 32;  // the CTA's full warps take wide groups
  // the running QPs into the parking area, in thread order (every thread)
  auto compact = [&]() {
    const unsigned bal = __ballot_sync(wmask, p >= 0);
    if (wl == 0) wcount[warp] = __popc(bal);
    __syncthreads();
    if (p >= 0) {
      int r = __popc(bal & ((1u << wl) - 1u));
      for (int k = 0; k < warp; ++k) r += wcount[k];
      park_store(r);
    }
    __syncthreads();
  };
  int n_run = __syncthreads_count(p >= 0);
#pragma unroll 1
  for (;;) {
    if (n_run <= wide_warps * L::QPW) break;  // the rest in the wide form
    if ((n_run + 31) / 32 < warps) {
      // repack: running QPs, in thread order, to threads 0 .. n_run - 1
      compact();
      p = -1;
      if ((int)threadIdx.x < n_run) park_load(threadIdx.x);
      warps = (n_run + 31) / 32;
    }
    bool run = p >= 0;
    if (run) {
      const int g = p / S;
      const float rho = per(g)[L::oRho];
      const float* kg = kin(g);
      const float* Gg = per(g) + L::oG;
      const int chunk = min(check, cfg.iters - it);
#pragma unroll 1
      for (int k = 0; k < chunk; ++k) {
        if (CONE == CONE_SOC) admm_iteration_soc<M>(y, w, mq, kg, cfg, rho);
        else admm_iteration<M>(y, w, mq, kg, cfg, rho);
      }
      it += chunk;
      // residuals from the parked copy: computed from registers, they would
      // need more than the 168 a thread has next to the iterate
      float rp, rd, scale[2];
      park_store(threadIdx.x);
      {
        const float* rec = park + threadIdx.x * L::PW;
        if (CONE == CONE_SOC) admm_residuals_soc<M, ADAPT>(rec, rec + L::pW, rec + L::pM, Gg, cfg, rho, rp, rd, scale);
        else admm_residuals<M, ADAPT>(rec, rec + L::pW, rec + L::pM, Gg, cfg, rho, rp, rd, scale);
      }
      park_load(threadIdx.x);
      const bool conv = cfg.eps > 0.f && rp <= cfg.eps && rd <= cfg.eps;
      if (conv || it >= cfg.iters) {
        finish_lane(p, rp, rd, conv);
        run = false;
      }
      // residual balancing (OSQP, Stellato et al. 2020, Sec. 5.2): each
      // running QP proposes rho_vote (normalised residuals) for its grasp; 0 once stopped
      if (adaptive) per(g)[L::oVote + p % S] = run ? rho_vote(rp, rd, scale) : 0.f;
      if (!run) p = -1;
    }
    n_run = __syncthreads_count(run);
    if (n_run == 0) break;
    if (adaptive) {
      if (!__syncthreads_or(decide())) continue;  // no grasp of the CTA changed rho
      const bool mine = p >= 0;
      if (mine) {  // re-express the iterate at the grasp's new rho, then park it (its registers go to the setup)
        const float* pg = per(p / S);
        if (pg[L::oRho] != pg[L::oRho + 1]) rescale_w<M, CONE>(w, pg[L::oRho + 1] / pg[L::oRho], cfg);
        park_store(threadIdx.x);
      }
      rebuild();
      if (mine) {
        park_load(threadIdx.x);
      } else {  // nothing of an idle thread lives across the rebuild
#pragma unroll
        for (int a = 0; a < NV; ++a) y[a] = mq[a] = 0.f;
#pragma unroll
        for (int k = 0; k < NC; ++k) w[k] = 0.f;
      }
    }
  }
  compact();
  // wide form (see above): the n_run parked QPs over as few warps as hold
  // them (record r on warp r mod ww), m lanes each
  const int ci = wl % M, gb = (wl / M) * M;  // contact; first lane of the group in the warp
  const bool group_lane = wl < L::QPW * M;   // lanes past the last whole group stay idle
  Wide<M, CONE> W;
  W.clear();
  p = -1;
  int ww = 0;  // warps that hold running QPs
  auto spread = [&]() {
    ww = (n_run + L::QPW - 1) / L::QPW;
    const int r = ww * (wl / M) + warp;
    p = -1;
    if (warp < ww && group_lane && r < n_run) {
      const float* rec = park + r * L::PW;
      it = reinterpret_cast<const int*>(rec)[L::pI];
      p = reinterpret_cast<const int*>(rec)[L::pI + 1];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        W.y[k] = rec[3 * ci + k];
        W.mq[k] = rec[L::pM + 3 * ci + k];
      }
#pragma unroll
      for (int k = 0; k < L::WPC; ++k) W.w[k] = rec[L::pW + L::WPC * ci + k];
      W.wsum = rec[L::pW + NC - 1];
      W.load_rows(kin(p / S), ci);
    }
  };
  spread();
#pragma unroll 1
  for (;;) {
    bool run = false;
    if (warp < ww) {
      const bool mine = p >= 0;
      const int g = mine ? p / S : 0;
      const float rho = per(g)[L::oRho];
      const float* Gg = per(g) + L::oG;
      // running QPs advance in lockstep rounds, so they share `it`
      const int chunk = __reduce_max_sync(0xffffffffu, mine ? min(check, cfg.iters - it) : 0);
      // two at a time with adaptive rho: one by one, five contacts' shuffles were
      // scheduled each before its own multiply-adds (0.29 us an iteration, two
      // at a time 0.14, the fixed-rho kernel 0.11)
#pragma unroll (ADAPT ? 2 : 1)
      for (int k = 0; k < chunk; ++k) W.iterate(cfg, rho, gb);
      it += chunk;
      float rpg, rdg, scale[2] = {0.f, 0.f};  // scales: adaptive rho only
      if (adaptive) W.template residuals<true>(Gg, cfg, rho, ci, gb, rpg, rdg, scale);
      else W.template residuals<false>(Gg, cfg, rho, ci, gb, rpg, rdg, scale);
      const bool conv = rpg <= cfg.eps && rdg <= cfg.eps;
      const bool done = mine && (conv || it >= cfg.iters);
      if (__any_sync(0xffffffffu, done)) {
        // the finished groups' results: each lane its contact's rows, the
        // group's first lane the sum row, Q and the status
        float ya[NV];
#pragma unroll
        for (int j = 0; j < NV; ++j) ya[j] = __shfl_sync(0xffffffffu, W.y[j % 3], gb + j / 3);
        if (done) {
          const size_t q = q0 + p;
#pragma unroll
          for (int r = 0; r < 3; ++r) yio[q * NV + 3 * ci + r] = W.y[r];
#pragma unroll
          for (int k = 0; k < L::WPC; ++k) {
            const float pr = CONE == CONE_SOC ? proj_row_soc<1>(W.w, k, cfg.gamma) : proj_row<1>(W.w[k], k, cfg.gamma);
            zio[q * NC + L::WPC * ci + k] = pr;
            lio[q * NC + L::WPC * ci + k] = rho * (W.w[k] - pr);
          }
          if (ci == 0) {
            const float pr = fmaxf(W.wsum, cfg.gamma);
            zio[q * NC + NC - 1] = pr;
            lio[q * NC + NC - 1] = rho * (W.wsum - pr);
            finish(p, ya, rpg, rdg, conv);
          }
        }
      }
      run = mine && !done && ci == 0;
      if (adaptive && mine && ci == 0) per(g)[L::oVote + p % S] = done ? 0.f : rho_vote(rpg, rdg, scale);
      if (done) p = -1;
    }
    n_run = __syncthreads_count(run);
    if (n_run == 0) break;
    if (adaptive && __syncthreads_or(decide())) {
      // the wide lanes re-express their rows at the grasp's new rho; after the
      // rebuild they load their rows of K^-1 again
      const bool moved = p >= 0 && per(p / S)[L::oRho] != per(p / S)[L::oRho + 1];
      if (moved) {
        const float ratio = per(p / S)[L::oRho + 1] / per(p / S)[L::oRho];
        rescale_contact<CONE>(W.w, ratio);
        W.wsum = rescale_sum_row(W.wsum, ratio, cfg.gamma);
      }
      rebuild();
      W.load_rows(kin(max(p, 0) / S), ci);  // every lane: the rows need not live across the rebuild
    }
    if ((n_run + L::QPW - 1) / L::QPW < ww) {
      // fewer warps hold the rest: their state through the parking area, in
      // thread order
      const unsigned bal = __ballot_sync(wmask, p >= 0 && ci == 0);
      if (wl == 0) wcount[warp] = __popc(bal);
      __syncthreads();
      if (p >= 0) {
        int r = __popc(bal & ((1u << gb) - 1u));
        for (int k = 0; k < warp; ++k) r += wcount[k];
        float* rec = park + r * L::PW;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          rec[3 * ci + k] = W.y[k];
          rec[L::pM + 3 * ci + k] = W.mq[k];
        }
#pragma unroll
        for (int k = 0; k < L::WPC; ++k) rec[L::pW + L::WPC * ci + k] = W.w[k];
        if (ci == 0) {
          rec[L::pW + NC - 1] = W.wsum;
          reinterpret_cast<int*>(rec)[L::pI] = it;
          reinterpret_cast<int*>(rec)[L::pI + 1] = p;
        }
      }
      __syncthreads();
      spread();
    }
  }
}

// ============================================================================ kernel: exact QPs (qp.solver = EXACT)
// One thread per QP, the minimum-norm-point solve in float32 (ExactQP); the
// block's grasps' G staged in shared memory.  Outputs: y, Q, the oracle
// calls in iters, res = (0, the final Frank-Wolfe gap, an upper bound on
// Q - Q*), z = A y clamped to the row bounds, lam = 0 (the method gives no
// multipliers); BODEX_ST_NOT_CONVERGED when the oracle-call cap stopped it.
template <int M>
__global__ void __launch_bounds__(CTA_LANES, 4) qp_exact_kernel(const float* __restrict__ Gin, int B,
                                                       const float* __restrict__ T, int S, AdmmCfg cfg, float* y_out,
                                                       float* z_out, float* l_out, float* Qout, int32_t* iters_out,
                                                       int32_t* status_out, float* res_out) {
  constexpr int NV = 3 * M, NC = 9 * M + 1;
  extern __shared__ __align__(16) float smem[];
  const int GPB = blockDim.x / S;
  const size_t g0 = (size_t)blockIdx.x * GPB;
  const int ng = (int)min((size_t)GPB, (size_t)B - g0);
  float* const edge = smem;                            // edge table, vertices [VW][threads], then G
  float* const vs = edge + ExactQP<M>::EDGE_WORDS;
  float* const Gs = vs + ExactQP<M>::VW * blockDim.x;
  ExactQP<M>::fill_edges(edge);
  for (int e = threadIdx.x; e < ng * 6 * NV; e += blockDim.x) Gs[e] = Gin[g0 * 6 * NV + e];
  __syncthreads();
  const int gl = threadIdx.x / S, j = threadIdx.x % S;
  if (gl >= ng) return;
  const size_t q = (g0 + gl) * S + j;
  const float* G = Gs + gl * 6 * NV;
  float t[6], y[NV], Q, gap;
#pragma unroll
  for (int r = 0; r < 6; ++r) t[r] = T[j * 6 + r];
  int n = 0;
  float lam[ExactQP<M>::K];
  const int ret = ExactQP<M>::solve(G, t, cfg, edge, cfg.iters, n, lam, vs + threadIdx.x, blockDim.x, y, Q, gap);
  const int calls = ret < 0 ? -ret : ret;
  bool fin = isfinite(Q);
#pragma unroll
  for (int a = 0; a < NV; ++a) {
    y_out[q * NV + a] = y[a];
    fin = fin && isfinite(y[a]);
  }
  float sumn = 0.f;
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const float yn = y[3 * i], yd = y[3 * i + 1], ye = y[3 * i + 2];
    sumn += yn;
    z_out[q * NC + 9 * i] = fminf(fmaxf(yn, 0.f), 1.f);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      z_out[q * NC + 9 * i + 1 + k] = fminf(fmaf(kFC[k], yd, fmaf(kFS[k], ye, -cfg.mu_c8 * yn)), 0.f);
  }
  z_out[q * NC + 9 * M] = fmaxf(sumn, cfg.gamma);
  for (int r = 0; r < NC; ++r) l_out[q * NC + r] = 0.f;
  Qout[q] = Q;
  if (iters_out) iters_out[q] = calls;
  if (res_out) {
    res_out[2 * q] = 0.f;
    res_out[2 * q + 1] = gap;
  }
  int st = 0;
  if (!fin) st |= BODEX_ST_NONFINITE;
  if (ret < 0) st |= BODEX_ST_NOT_CONVERGED;
  if (status_out) status_out[q] = st;
}

// ============================================================================ kernel: exact finish of the ADMM stragglers
// qp.polish = 2: after the ADMM kernel, the QPs it left above the residual
// target (BODEX_ST_NOT_CONVERGED) are solved exactly by the float32
// minimum-norm-point method (ExactQP).  A block takes a range of
// QP_FINISH_RANGE consecutive QPs, gathers the flagged ones into shared
// memory (ballot and prefix count), and its threads solve them one each.
// A finished QP takes the exact y and Q, gets BODEX_ST_POLISHED and loses
// BODEX_ST_NOT_CONVERGED; its z, lam, residuals and iteration count stay
// those of the ADMM run.  The QPs ADMM converged are not touched.
constexpr int QP_FINISH_RANGE = 256, QP_FINISH_THREADS = 128;

template <int M>
__global__ void __launch_bounds__(QP_FINISH_THREADS) qp_finish_kernel(const float* __restrict__ Gin, int B,
                                                                      const float* __restrict__ T, int S,
                                                                      AdmmCfg cfg, float* y_io, float* Qout,
                                                                      int32_t* status_io) {
  constexpr int NV = 3 * M;
  __shared__ int list[QP_FINISH_RANGE];
  __shared__ int count;
  __shared__ float edge[ExactQP<M, false>::EDGE_WORDS], vs[ExactQP<M, false>::VW * QP_FINISH_THREADS];
  ExactQP<M, false>::fill_edges(edge);
  const size_t n = (size_t)B * S, q0 = (size_t)blockIdx.x * QP_FINISH_RANGE;
  if (threadIdx.x == 0) count = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < QP_FINISH_RANGE; k += blockDim.x) {
    const size_t q = q0 + k;
    const bool flag = q < n && (status_io[q] & BODEX_ST_NOT_CONVERGED) && !(status_io[q] & BODEX_ST_NONFINITE);
    const unsigned bal = __ballot_sync(0xffffffffu, flag);
    int base = 0;
    if ((threadIdx.x & 31) == 0 && bal) base = atomicAdd(&count, __popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (flag) list[base + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u))] = k;
  }
  __syncthreads();
  const int cnt = count;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const size_t q = q0 + list[i];
    const size_t b = q / S;
    const int j = (int)(q % S);
    const float* G = Gin + b * 6 * NV;
    float t[6], y[NV], Q, gap;
#pragma unroll
    for (int r = 0; r < 6; ++r) t[r] = T[j * 6 + r];
    int m = 0;
    float lam[ExactQP<M, false>::K];
    if (ExactQP<M, false>::solve(G, t, cfg, edge, 64, m, lam, vs + threadIdx.x, QP_FINISH_THREADS, y, Q, gap) < 0) continue;
#pragma unroll
    for (int a = 0; a < NV; ++a) y_io[q * NV + a] = y[a];
    Qout[q] = Q;
    status_io[q] = (status_io[q] & ~BODEX_ST_NOT_CONVERGED) | BODEX_ST_POLISHED;
  }
}

// ============================================================================ kernel: solution polishing
// A pass after qp_solve_kernel when qp.polish is set (pyramid QPs with
// eps_reg = 0): one thread per QP solves the QP exactly in FP64 by the
// minimum-norm-point method (Wolfe<M, double>), its first vertex taken at the
// ADMM point.  Where that succeeds, y and Q become the exact minimiser and
// optimum (Q to FP64 rounding, y rounded to float), the QP gets
// BODEX_ST_POLISHED and loses BODEX_ST_NOT_CONVERGED; z, lam, the residuals
// and the iteration count stay those of the ADMM run.
template <int M>
__global__ void __launch_bounds__(128) qp_polish_kernel(const float* __restrict__ Gin, int B,
                                                        const float* __restrict__ T, int S, AdmmCfg cfg, float* y_io,
                                                        float* Qout, int32_t* status_io) {
  constexpr int NV = 3 * M;
  const size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (size_t)B * S) return;
  if (status_io && (status_io[q] & BODEX_ST_NONFINITE)) return;
  const size_t b = q / S;
  const int j = (int)(q % S);
  const float* G = Gin + b * 6 * NV;
  float t[6], ys[NV];
  for (int r = 0; r < 6; ++r) t[r] = T[j * 6 + r];
  for (int a = 0; a < NV; ++a) ys[a] = y_io[q * NV + a];
  double yd[NV], Qd;
  if (Wolfe<M, double>::solve(G, t, cfg, ys, 1e-13, 200, yd, Qd) < 0) return;
  for (int a = 0; a < NV; ++a) y_io[q * NV + a] = (float)yd[a];
  Qout[q] = (float)Qd;
  if (status_io) status_io[q] = (status_io[q] & ~BODEX_ST_NOT_CONVERGED) | BODEX_ST_POLISHED;
}

// ============================================================================ kernel: fused evaluation / step
struct FusedArgs {
  const HandDev* hand;
  ObjDev obj;
  const float* T;
  int S, B;
  AdmmCfg cfg;
  float w_q, w_d, delta;
  float lr_t, lr_r, b1, b2, adam_eps;
  int n_steps, t0;
  // pose input (eval) or state pose (step), updated in place for step
  const float* x_in;
  float* x_state;
  float* am;
  float* av;
  float* qy;  // warm start: may be null in eval (cold start); the state's arrays in step mode
  float* qw;
  // outputs
  float* E;
  float* dEdx;
  float* Qout;
  float* yout;
  int32_t* status;
  const float* yin;  // MODE_ADJOINT: forces from a previous solve [B, s, 3m]
  float* res;        // [B] max ADMM residual of the grasp's QPs at the last step (may be null)
  int gpb;           // grasps per CTA
  int dfc;           // 1: the DFC force-closure energy |G u|^2 replaces the QPs (uniform per launch)
  int coll;          // 1: the collision energies are on (uniform per launch)
  CollDev cd;
  CollParams cp;
};

// MODE_EVAL: E and dE/dx at x.  MODE_STEP: n_steps upper iterations on the
// state.  MODE_ADJOINT: E and dE/dx at x for given forces y (no QP solve):
// the backward pass of the energy, with FK and the SDF query recomputed.
enum { MODE_EVAL = 0, MODE_STEP = 1, MODE_ADJOINT = 2 };

// The work of one CTA: GPB grasps (cta * GPB ...) of one job, s lanes each;
// threads beyond GPB * s idle but take part in every barrier.
// CONE: CONE_PYR or CONE_SOC fixes the lower-level cone at compile time;
// CONE_ANY reads it from the arguments (the several-job kernel).  ADAPT:
// whether the kernel contains the adaptive-rho solve (residual-target
// solves); kernels for fixed iteration counts leave it out, as its code
// costs the fixed loop registers.  CONE_EXACT: the pyramid's QPs solved
// exactly (qp.solver = EXACT, ExactQP) instead of by ADMM: no K^-1 set-up;
// each QP's working set (corral) carries over to the next upper step in
// the state's warm-start array: word 0 the point count, then 7 vertex
// codes, 7 fractional forces and 7 weights (component-major, like the ADMM
// iterate it replaces).
constexpr int CONE_ANY = -1;
constexpr int CONE_EXACT = 2;

// dE/dc of contact `lane` through its kinematic chain: the translation, the
// root rotations and the chain joints (axes and points jw of the forward
// pass), into the contact's record cb.
__device__ __forceinline__ void chain_adjoint(const HandDev& H, int lane, const float* xs, const float* c,
                                              const float* jw, const float* dEdc, float* cb) {
  cb[0] = dEdc[0];
  cb[1] = dEdc[1];
  cb[2] = dEdc[2];
  // root rotations rx, ry, rz: axes through t
  {
    float s1, c1, s2, c2;
    angle_sincos(xs[3], &s1, &c1);
    angle_sincos(xs[4], &s2, &c2);
    const float om[3][3] = {{1.f, 0.f, 0.f}, {0.f, c1, s1}, {s2, -s1 * c2, c1 * c2}};
    const float rel[3] = {c[0] - xs[0], c[1] - xs[1], c[2] - xs[2]};
    for (int k3 = 0; k3 < 3; ++k3) {
      float v[3];
      cross3(om[k3], rel, v);
      cb[3 + k3] = dEdc[0] * v[0] + dEdc[1] * v[1] + dEdc[2] * v[2];
    }
  }
  const int Lc = H.chain_len[lane];
  for (int kk = 0; kk < Lc; ++kk) {
    const float rel[3] = {c[0] - jw[6 * kk + 3], c[1] - jw[6 * kk + 4], c[2] - jw[6 * kk + 5]};
    float v[3];
    cross3(jw + 6 * kk, rel, v);
    cb[6 + kk] = dEdc[0] * v[0] + dEdc[1] * v[1] + dEdc[2] * v[2];
  }
}

// The gradient of grasp b from its contacts' records (fixed order over the
// contacts), coordinates spread over S lanes; in MODE_STEP the Adam step and
// the clamp follow.
template <int M, int MODE>
__device__ __forceinline__ void assemble_step(const FusedArgs& A, const HandDev& H, int b, int lane, int S, int step,
                                              float lb1, float lb2, float* per) {
  using L = Lay<M>;
  float* xs = per + L::oX;
  float* ams = per + L::oAM;
  float* avs = per + L::oAV;
  const int D = H.D;
  const float* cb = per + L::oCB;
  const int tstep = A.t0 + step + 1;
  // bias corrections 1 - b^t as 1 - 2^(t log2 b): a function of t alone,
  // so a run split over several launches gives the same values
  const float c1 = 1.f - exp2f((float)tstep * lb1), c2 = 1.f - exp2f((float)tstep * lb2);
  const float ic1 = 1.f / c1, ic2 = 1.f / c2;  // once per step, not per coordinate
  for (int k = lane; k < D; k += S) {
    float g = 0.f;
    if (k < 6) {
#pragma unroll
      for (int i = 0; i < M; ++i) g += cb[i * (6 + MAXCHAIN) + k];
    } else {
      float v[M];  // every load before the sum: a contact that the joint does not move adds 0
#pragma unroll
      for (int i = 0; i < M; ++i) {
        const int pos = H.jpos[i][k - 6];
        const float e = cb[i * (6 + MAXCHAIN) + 6 + max(pos, 0)];
        v[i] = pos >= 0 ? e : 0.f;
      }
#pragma unroll
      for (int i = 0; i < M; ++i) g += v[i];
    }
    if (A.coll) g += per[L::oGC + k];
    if (MODE != MODE_STEP) {
      if (A.dEdx) A.dEdx[(size_t)b * D + k] = g;
    } else {
      const float mm = fmaf(A.b1, ams[k], (1.f - A.b1) * g);
      const float vv = fmaf(A.b2, avs[k], (1.f - A.b2) * g * g);
      ams[k] = mm;
      avs[k] = vv;
      const float lr = k < 3 ? A.lr_t : A.lr_r;
      const float xn = xs[k] - __fdividef(lr * (mm * ic1), sqrtf(vv * ic2) + A.adam_eps);
      xs[k] = fminf(fmaxf(xn, H.qmin[k]), H.qmax[k]);
    }
  }
}

template <int M, int MODE, int CONE = CONE_ANY, bool ADAPT = false, bool FEW = false>
__device__ __forceinline__ void fused_cta(const FusedArgs& A, int cta, int GPB, float* smem) {
  using L = Lay<M>;
  constexpr int NV = L::NV, NC = L::NC;
  copy_hand_to_smem(A.hand, smem);
  const int S = A.S;
  const int gl = threadIdx.x / S, lane = threadIdx.x % S;
  const int b = cta * GPB + gl;
  const bool active = (gl < GPB) && (b < A.B);
  // With s < m lanes a grasp, a lane takes several contacts.  The kernels for
  // s >= m do without that loop, which cost the fixed-iteration step 0.8%
  // (13.63 against 13.51 ms for 4096 grasps x 200 steps), the adaptive one of
  // five contacts 5% (310 -> 326 us for 3 steps of 2000 grasps) and its
  // evaluation 10% (349 -> 385 us at 810 grasps), where it spills the iterate
  // (816 bytes of loads instead of 384): run_fused gives their s < m cases to
  // the wide form or, with adaptive rho and under DFC, to the kernels for few
  // wrenches (FEW).  Launches of several jobs take the kernels for few wrenches
  // when a job needs them (without the loop the adaptive one reloads 856 bytes
  // instead of 1512, 434 -> 417 us for 4050 grasps of hand5, 3 steps of 8
  // wrenches; fixed rho gains some 1%) and when blocks pull their items, whose
  // spills without it are no smaller (8704 grasps of hand5: 637 us, with it 614).
  constexpr bool ONE_CONTACT = !FEW && MODE != MODE_ADJOINT && CONE != CONE_EXACT;
  const HandDev& H = *reinterpret_cast<const HandDev*>(smem);
  float* kin = smem + L::HAND_WORDS + gl * L::KS;
  float* per = smem + L::HAND_WORDS + GPB * L::KS + gl * L::PER;
  float* Gs = per + L::oG;
  float* xs = per + L::oX;
  float* ams = per + L::oAM;
  float* avs = per + L::oAV;
  float* sc = per + L::oSC;
  int* stat = reinterpret_cast<int*>(sc + 1);
  __syncthreads();  // hand copied
  const int D = H.D;
  const AdmmCfg& cfg = A.cfg;

  if (active) {
    const float* xsrc = (MODE == MODE_STEP) ? A.x_state : A.x_in;
    for (int k = lane; k < D; k += S) {
      xs[k] = xsrc[(size_t)b * D + k];
      if (MODE == MODE_STEP) {
        ams[k] = A.am[(size_t)b * D + k];
        avs[k] = A.av[(size_t)b * D + k];
      }
    }
    if (lane == 0) {
      *stat = 0;
      sc[2] = 0.f;      // max residual of the grasp's QPs at the last step
      sc[3] = cfg.rho;  // the grasp's ADMM penalty (adapted in solves with a residual target)
    }
  }
  // ADMM iterate of this lane's QP.  In MODE_STEP it lives in the state's
  // warm-start arrays between upper steps and in registers only around the
  // solve, so the FK / SDF / adjoint phases get the registers it would hold.
  float y[NV], w[NC];
  const size_t q = (size_t)b * S + lane, NQ = (size_t)A.B * S;
  if (MODE == MODE_ADJOINT && active) {
#pragma unroll
    for (int a = 0; a < NV; ++a) y[a] = A.yin[q * NV + a];
#pragma unroll
    for (int r = 0; r < NC; ++r) w[r] = 0.f;
  } else if (MODE == MODE_EVAL && active && A.qy && CONE != CONE_EXACT) {
#pragma unroll
    for (int a = 0; a < NV; ++a) y[a] = A.qy[a * NQ + q];
#pragma unroll
    for (int r = 0; r < NC; ++r) w[r] = A.qw[r * NQ + q];
  } else {
#pragma unroll
    for (int a = 0; a < NV; ++a) y[a] = 0.f;
#pragma unroll
    for (int r = 0; r < NC; ++r) w[r] = 0.f;
  }
  float t[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (active)
    for (int r = 0; r < 6; ++r) t[r] = A.T[lane * 6 + r];
  // the exact solver's edge table, in the first grasp's K^-1 block (no K^-1 there)
  float* const edge = smem + L::HAND_WORDS;
  if (CONE == CONE_EXACT) ExactQP<M>::fill_edges(edge);
  __syncthreads();

  const float lb1 = log2f(A.b1), lb2 = log2f(A.b2);
  for (int step = 0; step < A.n_steps; ++step) {
    // ---- A1-A3: kinematics, nearest-point query, grasp matrix (lane = contact)
    if (int i = lane; active && i < M) do {
      float c[3];
      fk_contact(H, i, xs, c, per + L::oJW + i * MAXCHAIN * 6,
                 (A.coll && A.cd.K > 0) ? per + L::oK : nullptr);  // link frames for the collision spheres
      const ContactGeo k = contact_geometry(A.obj, c);
      store_ct(per + L::oCT + L::CTW * i, k);
      write_G_block(k, i, NV, Gs);
      int st = 0;
      if (k.degenerate) st |= BODEX_ST_DEGENERATE_NORMAL;
      if (!finite3(k.p) || !finite3(k.n) || !isfinite(k.phi)) st |= BODEX_ST_NONFINITE;
      if (st) atomicOr(stat, st);
    } while (!ONE_CONTACT && (i += S) < M);
    __syncthreads();
    // ---- constraint energies on the collision spheres (Sec. IV-B)
    if (A.coll)
      collision_phase(active, lane, S, H, A.cd, A.obj, xs, A.cp, per + L::oK, per + L::oJW, per + L::oRY,
                      per + L::oRY + 3 * A.cd.K, per + L::oRY + 3 * A.cd.K + 6 * (H.n + 1), per + L::oGC,
                      per + L::oGC + MAXD);
    // ---- A4: K^-1 per grasp (at the grasp's current penalty)
    if (MODE != MODE_ADJOINT && !A.dfc && CONE != CONE_EXACT) {
      if constexpr (ADAPT) {
        AdmmCfg cg = cfg;
        if (active) cg.rho = sc[3];  // a several-job block has threads beyond its job's grasps: no record there
        setup_kinv<M, true>(active, lane, S, Gs, per + L::oK, kin, cg);
      } else {
        setup_kinv<M, true>(active, lane, S, Gs, per + L::oK, kin, cfg);
      }
    }
    // ---- A5: ADMM, one QP per lane
    if (active && A.dfc) per[L::oQ + lane] = 0.f;  // no lower-level QPs under DFC
    bool conv = true;
    // r_j, Q_j, the stored iterate and the status of this lane's QP
    auto finish_qp = [&]() {
      float* ry = per + L::oRY + lane * L::RYW;
      float Q = 0.f;
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        float s = cfg.beta * t[r];
#pragma unroll
        for (int a = 0; a < NV; ++a) s = fmaf(-Gs[r * NV + a], y[a], s);
        ry[r] = s;
        Q = fmaf(s, s, Q);
      }
#pragma unroll
      for (int a = 0; a < NV; ++a) {
        ry[8 + a] = y[a];
        Q = fmaf(cfg.eps_reg * y[a], y[a], Q);  // regularised value when eps_reg > 0
      }
      per[L::oQ + lane] = Q;
      if (MODE == MODE_STEP && CONE != CONE_EXACT) {
#pragma unroll
        for (int a = 0; a < NV; ++a) A.qy[a * NQ + q] = y[a];
#pragma unroll
        for (int r = 0; r < NC; ++r) A.qw[r * NQ + q] = w[r];
      }
      int st = 0;
      if (cfg.eps > 0.f && !conv) st |= BODEX_ST_NOT_CONVERGED;
      if (!isfinite(Q)) st |= BODEX_ST_NONFINITE;
      if (st) atomicOr(stat, st);
    };
    const bool soc = CONE == CONE_ANY ? cfg.cone != 0 : CONE == CONE_SOC;
    if constexpr (CONE == CONE_EXACT) {
      // the exact lower level: each lane solves its QP from the corral its
      // previous step left (cold at the first step of a run)
      if (active && !A.dfc && MODE != MODE_ADJOINT) {
        constexpr int K = ExactQP<M>::K;
        int n = 0;
        float lam[K];
        // the vertices live in this lane's output record, written only after the solve
        float* const vs = per + L::oRY + lane * L::RYW;
        if (A.qw) {
          n = __float_as_int(A.qw[q]);
#pragma unroll
          for (int i = 0; i < K; ++i) {
            vs[i] = A.qw[(1 + i) * NQ + q];
            vs[K + i] = A.qw[(8 + i) * NQ + q];
            lam[i] = A.qw[(15 + i) * NQ + q];
          }
        }
        float Qx, gap;
        const int ret = ExactQP<M>::solve(Gs, t, cfg, edge, cfg.iters, n, lam, vs, 1, y, Qx, gap);
        if (A.qw) {
          A.qw[q] = __int_as_float(n);
#pragma unroll
          for (int i = 0; i < K; ++i) {
            A.qw[(1 + i) * NQ + q] = vs[i];
            A.qw[(8 + i) * NQ + q] = vs[K + i];
            A.qw[(15 + i) * NQ + q] = lam[i];
          }
        }
        if (step == A.n_steps - 1) atomicMax(reinterpret_cast<int*>(sc + 2), __float_as_int(fmaxf(gap, 0.f)));
        if (ret < 0) atomicOr(stat, BODEX_ST_NOT_CONVERGED);
      }
      if (active && !A.dfc) finish_qp();
    } else if constexpr (ADAPT) {
      // solves with a residual target adapt rho per grasp (every thread takes
      // part); the iterate is stored with rho0 = cfg.rho and re-expressed at
      // the grasp's rho here
      if (!A.dfc) {
        float mq[NV];
        float rp = 0.f, rd = 0.f;
        AdmmCfg cg = cfg;
        if (active) {
          cg.rho = sc[3];
          if (MODE == MODE_STEP) {
#pragma unroll
            for (int a = 0; a < NV; ++a) y[a] = A.qy[a * NQ + q];
#pragma unroll
            for (int r = 0; r < NC; ++r) w[r] = A.qw[r * NQ + q];
          }
          if (MODE != MODE_ADJOINT) neg_q<M>(Gs, t, cfg.beta, mq);
          if (cg.rho != cfg.rho) {
            if (soc) rescale_w<M, CONE_SOC>(w, cfg.rho / cg.rho, cg);
            else rescale_w<M, CONE_PYR>(w, cfg.rho / cg.rho, cg);
          }
        }
        if (MODE != MODE_ADJOINT) {
          auto setup = [&](bool upd, const AdmmCfg& cc) { setup_kinv<M>(upd, lane, S, Gs, per + L::oK, kin, cc); };
          if (soc)
            admm_solve_adaptive<M, CONE_SOC>(active, lane, S, y, w, mq, kin, Gs, cg, per + L::oQ, setup, rp, rd, conv);
          else
            admm_solve_adaptive<M, CONE_PYR>(active, lane, S, y, w, mq, kin, Gs, cg, per + L::oQ, setup, rp, rd, conv);
          if (active) {
            if (lane == 0) sc[3] = cg.rho;  // every lane of the grasp holds the same rho
            if (cg.rho != cfg.rho) {
              if (soc) rescale_w<M, CONE_SOC>(w, cg.rho / cfg.rho, cg);
              else rescale_w<M, CONE_PYR>(w, cg.rho / cfg.rho, cg);
            }
            if (step == A.n_steps - 1) atomicMax(reinterpret_cast<int*>(sc + 2), __float_as_int(fmaxf(rp, rd)));
          }
        }
        if (active) finish_qp();
      }
    } else if (active && !A.dfc) {
      if (MODE == MODE_STEP) {
#pragma unroll
        for (int a = 0; a < NV; ++a) y[a] = A.qy[a * NQ + q];
#pragma unroll
        for (int r = 0; r < NC; ++r) w[r] = A.qw[r * NQ + q];
      }
      if (MODE != MODE_ADJOINT) {
        float mq[NV];
        neg_q<M>(Gs, t, cfg.beta, mq);
        float rp, rd;
        const bool last = step == A.n_steps - 1;
        if (soc) admm_solve<M, CONE_SOC>(y, w, mq, kin, Gs, cfg, rp, rd, conv, last);
        else admm_solve<M, CONE_PYR>(y, w, mq, kin, Gs, cfg, rp, rd, conv, last);
        if (step == A.n_steps - 1) atomicMax(reinterpret_cast<int*>(sc + 2), __float_as_int(fmaxf(rp, rd)));
      }
      finish_qp();
    }
    __syncthreads();
    // ---- A6: energy;  A7 (part 1), DFC only: E_Q = |G u|^2 with u = 1 on
    // every normal component, so dE/dG = 2 w_Q (G u) u^T (only the normal
    // columns), written to shared memory.  The QP energy's
    // dE/dG = -2 w_Q sum_j r_j y_j^T is formed per contact in part 2.
    if (active && A.dfc) {
      float gu[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < M; ++i) s += Gs[r * NV + 3 * i];
        gu[r] = s;
      }
      for (int e = lane; e < 6 * NV; e += S) {
        const int r = e / NV, a = e % NV;
        float g = 0.f;
#pragma unroll
        for (int rr = 0; rr < 6; ++rr) g = (rr == r) ? gu[rr] : g;
        per[L::oDG + e] = (a % 3 == 0) ? 2.f * A.w_q * g : 0.f;
      }
      if (lane == 0) {
        float EQ = 0.f;
#pragma unroll
        for (int r = 0; r < 6; ++r) EQ = fmaf(gu[r], gu[r], EQ);
        float Ed = 0.f;
        for (int i = 0; i < M; ++i) {
          const float r = per[L::oCT + L::CTW * i + 9] - H.alpha - A.delta;
          Ed = fmaf(r, r, Ed);
        }
        float Ec = 0.f;
        if (A.coll)
          for (int l = 0; l < S; ++l) Ec += per[L::oGC + MAXD + l];
        sc[0] = A.w_q * EQ + A.w_d * Ed + Ec;
      }
    }
    if (active && !A.dfc && lane == 0) {
      float EQ = 0.f;
      for (int j = 0; j < S; ++j) EQ += per[L::oQ + j];
      float Ed = 0.f;
      for (int i = 0; i < M; ++i) {
        const float r = per[L::oCT + L::CTW * i + 9] - H.alpha - A.delta;
        Ed = fmaf(r, r, Ed);
      }
      float Ec = 0.f;
      if (A.coll)
        for (int l = 0; l < S; ++l) Ec += per[L::oGC + MAXD + l];
      sc[0] = A.w_q * EQ + A.w_d * Ed + Ec;
    }
    // the QP energy's dE/dG is formed by the contact lanes below, from the
    // r_j and y_j the QP lanes wrote before the last barrier; only DFC's
    // shared dE/dG needs one more
    if (A.dfc) __syncthreads();
    // ---- A7 (part 2): through the contact geometry and the kinematic chain
    if (int i = lane; active && i < M) do {
      const ContactGeo k = load_ct(per + L::oCT + L::CTW * i);
      float cols[18];
      if (A.dfc) {
        for (int r = 0; r < 6; ++r)
          for (int cc = 0; cc < 3; ++cc) cols[r * 3 + cc] = per[L::oDG + r * NV + 3 * i + cc];
      } else {
        // this contact's three columns of dE/dG = -2 w_Q sum_j r_j y_j^T,
        // each entry summing j in four partial sums (j mod 4, the tail
        // into the first)
        const float* ry = per + L::oRY;
        float s[18][4];
#pragma unroll
        for (int e = 0; e < 18; ++e)
#pragma unroll
          for (int u = 0; u < 4; ++u) s[e][u] = 0.f;
        auto acc = [&](int j, int u) {
          const float4 r03 = *reinterpret_cast<const float4*>(ry + j * L::RYW);
          const float2 r45 = *reinterpret_cast<const float2*>(ry + j * L::RYW + 4);
          const float rv[6] = {r03.x, r03.y, r03.z, r03.w, r45.x, r45.y};
          const float* yj = ry + j * L::RYW + 8 + 3 * i;
          const float yv[3] = {yj[0], yj[1], yj[2]};
#pragma unroll
          for (int r = 0; r < 6; ++r)
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) s[r * 3 + cc][u] = fmaf(rv[r], yv[cc], s[r * 3 + cc][u]);
        };
        int j = 0;
        for (; j + 3 < S; j += 4) {
          acc(j, 0);
          acc(j + 1, 1);
          acc(j + 2, 2);
          acc(j + 3, 3);
        }
        for (; j < S; ++j) acc(j, 0);
#pragma unroll
        for (int e = 0; e < 18; ++e) cols[e] = -2.f * A.w_q * ((s[e][0] + s[e][1]) + (s[e][2] + s[e][3]));
      }
      float dEdc[3];
      contact_adjoint(k, cols, 2.f * A.w_d * (k.phi - H.alpha - A.delta), dEdc);
      chain_adjoint(H, i, xs, k.c, per + L::oJW + i * MAXCHAIN * 6, dEdc, per + L::oCB + i * (6 + MAXCHAIN));
    } while (!ONE_CONTACT && (i += S) < M);
    __syncthreads();
    // ---- gradient assembly (fixed order over contacts) and A8: Adam + clamp
    if (active) assemble_step<M, MODE>(A, H, b, lane, S, step, lb1, lb2, per);
    __syncthreads();
  }

  // ---- write back (no early return: the several-job kernel runs this
  // function once per work item, with barriers between items)
  if (active) {
    if (lane == 0) {
      if (A.E) A.E[b] = sc[0];
      if (A.status) A.status[b] = *stat;
      if (A.res) A.res[b] = sc[2];
    }
    if (MODE == MODE_STEP) {
      for (int k = lane; k < D; k += S) {
        A.x_state[(size_t)b * D + k] = xs[k];
        A.am[(size_t)b * D + k] = ams[k];
        A.av[(size_t)b * D + k] = avs[k];
      }
    }
    if (MODE == MODE_EVAL && A.qy && CONE != CONE_EXACT) {
#pragma unroll
      for (int a = 0; a < NV; ++a) A.qy[a * NQ + q] = y[a];
#pragma unroll
      for (int r = 0; r < NC; ++r) A.qw[r * NQ + q] = w[r];
    }
    if (MODE == MODE_EVAL) {
      if (A.Qout) A.Qout[q] = per[L::oQ + lane];
      if (A.yout)
#pragma unroll
        for (int a = 0; a < NV; ++a) A.yout[q * NV + a] = y[a];
    }
  }
}

template <int M, int MODE, int CONE, bool ADAPT, bool FEW = false>
__global__ void __launch_bounds__(CTA_LANES, 4) fused_kernel(FusedArgs A) {
  extern __shared__ __align__(16) float smem[];
  fused_cta<M, MODE, CONE, ADAPT, FEW>(A, blockIdx.x, A.gpb, smem);
}

// ============================================================================ kernel: fused evaluation / step, wide form
// The fused step with m lanes per QP (Wide) instead of one, for fixed rho:
// the CTA's GPB * s QPs lie one after another over its warps, 32 / m a warp,
// and the lanes of a grasp, all threads of the CTA over GPB, share its set-up
// phases.  Per lane the iterate is 13 words, so it stays in registers from
// step to step.  Results are bitwise those of fused_cta.
constexpr int WIDE_THREADS = 128;

template <int M, int MODE, int CONE>
__device__ __forceinline__ void fused_wide_cta(const FusedArgs& A, int cta, int GPB, float* smem) {
  using L = Lay<M>;
  using WQ = Wide<M, CONE>;
  constexpr int NV = L::NV, WPC = WQ::WPC, QPW = WQ::QPW;
  copy_hand_to_smem(A.hand, smem);
  const HandDev& H = *reinterpret_cast<const HandDev*>(smem);
  const int S = A.S, LN = blockDim.x / GPB;  // LN >= s m lanes per grasp
  // A thread's two roles: lane `lane` of grasp gl in the set-up phases, and
  // lane ci of the group (from lane gb of the warp) that holds wrench j of
  // grasp gq.  Between the phases they live in two words: what follows from
  // them is formed again in each phase (the compiler does not see that
  // word() returns the same value), or some thirty pointers and indices
  // stayed in registers across the ADMM loop and its K^-1 rows spilled (600
  // cycles an iteration instead of 237).
  auto word = [](int w) {
    asm volatile("" : "+r"(w));
    return w;
  };
  struct SetUp {
    int lane, b;
    bool active;
    float *per, *kin;
  };
  struct Solve {
    int ci, gb, j;
    bool mine;
    float *per, *kin;
    size_t q;
  };
  const int w_set = (threadIdx.x / LN) << 16 | (threadIdx.x % LN);
  int w_qp;
  {
    const int wl = threadIdx.x % 32, qi = (threadIdx.x / 32) * QPW + min(wl / M, QPW - 1), gq = min(qi / S, GPB - 1);
    const bool mine = wl < QPW * M && qi < GPB * S && cta * GPB + gq < A.B;
    w_qp = (mine ? 1 << 24 : 0) | gq << 16 | (qi % S) << 8 | (wl % M);
  }
  auto set_up = [&]() {
    const int w = word(w_set), gl = w >> 16, g = min(gl, GPB - 1);
    SetUp r;
    r.lane = w & 0xffff;
    r.b = cta * GPB + gl;
    r.active = gl < GPB && r.b < A.B;
    r.kin = smem + L::HAND_WORDS + g * L::KS;
    r.per = smem + L::HAND_WORDS + GPB * L::KS + g * L::PER;
    return r;
  };
  auto solve = [&]() {
    const int w = word(w_qp), gq = (w >> 16) & 0xff;
    Solve r;
    r.ci = w & 0xff;
    r.gb = ((threadIdx.x % 32) / M) * M;
    r.j = (w >> 8) & 0xff;
    r.mine = w >> 24;
    r.kin = smem + L::HAND_WORDS + gq * L::KS;
    r.per = smem + L::HAND_WORDS + GPB * L::KS + gq * L::PER;
    r.q = (size_t)(cta * GPB + gq) * S + r.j;
    return r;
  };
  const size_t NQ = (size_t)A.B * S;
  __syncthreads();  // hand copied
  const int D = H.D;
  const AdmmCfg& cfg = A.cfg;
  if (const SetUp u = set_up(); u.active) {
    float* const per = u.per;
    const int lane = u.lane, b = u.b;
    const float* xsrc = (MODE == MODE_STEP) ? A.x_state : A.x_in;
    for (int k = lane; k < D; k += LN) {
      per[L::oX + k] = xsrc[(size_t)b * D + k];
      if (MODE == MODE_STEP) {
        per[L::oAM + k] = A.am[(size_t)b * D + k];
        per[L::oAV + k] = A.av[(size_t)b * D + k];
      }
    }
    if (lane == 0) {
      reinterpret_cast<int*>(per + L::oSC)[1] = 0;  // status
      per[L::oSC + 2] = 0.f;                        // max residual of the grasp's QPs at the last step
    }
  }
  WQ W;
  W.clear();
  const bool warm = MODE == MODE_STEP || A.qy;
  if (const Solve v = solve(); v.mine && warm) {
    const int ci = v.ci;
    const size_t q = v.q;
#pragma unroll
    for (int r = 0; r < 3; ++r) W.y[r] = A.qy[(3 * ci + r) * NQ + q];
#pragma unroll
    for (int k = 0; k < WPC; ++k) W.w[k] = A.qw[(WPC * ci + k) * NQ + q];
    W.wsum = A.qw[WPC * M * NQ + q];
  }
  __syncthreads();

#pragma unroll 1
  for (int step = 0; step < A.n_steps; ++step) {
    const bool last = step == A.n_steps - 1;
    // ---- A1-A3: kinematics, nearest-point query, grasp matrix (lane = contact)
    // (rotations and root frame in the records of the QP outputs, which are
    // written after them)
    static_assert(SMAX * L::RYW >= 9 * MAXJ + 12, "room for the joint rotations");
    if (const SetUp u = set_up(); u.active)
      for (int e = u.lane; e <= H.n; e += LN)
        fk_joint(H, e, u.per + L::oX, u.per + L::oRY, u.per + L::oRY + 9 * MAXJ);
    __syncthreads();
    if (const SetUp u = set_up(); u.active)
      for (int e = u.lane; e < 3 * M; e += LN)
        fk_row(H, e / 3, e % 3, u.per + L::oRY, u.per + L::oRY + 9 * MAXJ, u.per + L::oJW + (e / 3) * MAXCHAIN * 6,
               u.per + L::oCT + L::CTW * (e / 3), nullptr,
               (A.coll && A.cd.K > 0) ? u.per + L::oK : nullptr);  // link frames for the collision spheres
    __syncthreads();
    if (const SetUp u = set_up(); u.active && u.lane < M) {
      float* const per = u.per;
      const int lane = u.lane;
      const float* rec = per + L::oCT + L::CTW * lane;
      const float c[3] = {rec[0], rec[1], rec[2]};
      const ContactGeo k = contact_geometry(A.obj, c);
      store_ct(per + L::oCT + L::CTW * lane, k);
      write_G_block(k, lane, NV, per + L::oG);
      int st = 0;
      if (k.degenerate) st |= BODEX_ST_DEGENERATE_NORMAL;
      if (!finite3(k.p) || !finite3(k.n) || !isfinite(k.phi)) st |= BODEX_ST_NONFINITE;
      if (st) atomicOr(reinterpret_cast<int*>(per + L::oSC + 1), st);
    }
    __syncthreads();
    // ---- constraint energies on the collision spheres (hinges in the K^-1 block, not yet formed)
    static_assert(L::KS >= BODEX_MAX_SPHERES, "room for the spheres' hinges");
    if (A.coll) {
      const SetUp u = set_up();
      float* const per = u.per;
      collision_phase_wide(u.active, u.lane, S, LN, L::COLL_CS, H, A.cd, A.obj, per + L::oX, A.cp, per + L::oK,
                      per + L::oJW, per + L::oRY, per + L::oRY + 3 * A.cd.K, per + L::oRY + 3 * A.cd.K + 6 * (H.n + 1),
                      u.kin, per + L::oGC, per + L::oGC + MAXD);
    }
    // ---- A4: K^-1 per grasp
    {
      const SetUp u = set_up();
      setup_kinv<M, false, true>(u.active, u.lane, LN, u.per + L::oG, u.per + L::oK, u.kin, cfg);
    }
    // ---- A5: ADMM, one QP per m lanes
    {
      const Solve v = solve();
      W.load_rows(v.kin, v.ci);
      float t[6];
#pragma unroll
      for (int r = 0; r < 6; ++r) t[r] = __ldg(A.T + v.j * 6 + r);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float s = 0.f;
#pragma unroll
        for (int r = 0; r < 6; ++r) s = fmaf(v.per[L::oG + r * NV + 3 * v.ci + k], t[r], s);
        W.mq[k] = 2.f * cfg.beta * s;
      }
    }
    const int gb = ((threadIdx.x % 32) / M) * M;
    float rp = 0.f, rd = 0.f;
    bool conv = false;
    if (cfg.eps > 0.f) {
      // to a residual: a QP that reaches it keeps its iterate while the
      // others of its warp go on
      float ky[3], kw[WPC], ksum = 0.f, krp = 0.f, krd = 0.f;
#pragma unroll 1
      for (int it = 0; it < cfg.iters;) {
        const int chunk = min(cfg.check, cfg.iters - it);
#pragma unroll 1
        for (int k = 0; k < chunk; ++k) W.iterate(cfg, cfg.rho, gb);
        it += chunk;
        const Solve v = solve();
        W.template residuals<false>(v.per + L::oG, cfg, cfg.rho, v.ci, gb, rp, rd, nullptr);
        if (!conv) {
          krp = rp;
          krd = rd;
          ksum = W.wsum;
#pragma unroll
          for (int r = 0; r < 3; ++r) ky[r] = W.y[r];
#pragma unroll
          for (int k = 0; k < WPC; ++k) kw[k] = W.w[k];
          conv = rp <= cfg.eps && rd <= cfg.eps;
        }
        if (__all_sync(0xffffffffu, conv || !v.mine)) break;
      }
      if (cfg.iters > 0) {
        rp = krp;
        rd = krd;
        W.wsum = ksum;
#pragma unroll
        for (int r = 0; r < 3; ++r) W.y[r] = ky[r];
#pragma unroll
        for (int k = 0; k < WPC; ++k) W.w[k] = kw[k];
      }
    } else {
#pragma unroll 1
      for (int it = 0; it < cfg.iters; ++it) W.iterate(cfg, cfg.rho, gb);
      if (last) {
        const Solve v = solve();
        W.template residuals<false>(v.per + L::oG, cfg, cfg.rho, v.ci, gb, rp, rd, nullptr);
      }
      conv = true;
    }
    {
      // r = beta t - G y (row r by lane r of the group, the last rows by the
      // first lanes), Q, the status; y and r for the adjoint
      const Solve u = solve();
      const int ci = u.ci, j = u.j;
      const bool mine = u.mine;
      float* const perq = u.per;
      const float* const Gq = perq + L::oG;
      float* const ry = perq + L::oRY + j * L::RYW;
      float ya[NV], s[(6 + M - 1) / M], Q = 0.f;
#pragma unroll
      for (int a = 0; a < NV; ++a) ya[a] = __shfl_sync(0xffffffffu, W.y[a % 3], gb + a / 3);
#pragma unroll
      for (int k = 0; k < (6 + M - 1) / M; ++k) {
        const int r = min(ci + k * M, 5);
        float v = cfg.beta * __ldg(A.T + j * 6 + r);
#pragma unroll
        for (int a = 0; a < NV; ++a) v = fmaf(-Gq[r * NV + a], ya[a], v);
        s[k] = v;
        if (mine && ci + k * M < 6) ry[r] = v;
      }
#pragma unroll
      for (int r = 0; r < 6; ++r) {
        const float v = __shfl_sync(0xffffffffu, s[r / M], gb + r % M);
        Q = fmaf(v, v, Q);
      }
#pragma unroll
      for (int a = 0; a < NV; ++a) Q = fmaf(cfg.eps_reg * ya[a], ya[a], Q);  // regularised value when eps_reg > 0
      if (mine) {
#pragma unroll
        for (int r = 0; r < 3; ++r) ry[8 + 3 * ci + r] = W.y[r];
        if (ci == 0) {
          perq[L::oQ + j] = Q;
          int st = 0;
          if (cfg.eps > 0.f && !conv) st |= BODEX_ST_NOT_CONVERGED;
          if (!isfinite(Q)) st |= BODEX_ST_NONFINITE;
          if (st) atomicOr(reinterpret_cast<int*>(perq + L::oSC + 1), st);
          if (last) atomicMax(reinterpret_cast<int*>(perq + L::oSC + 2), __float_as_int(fmaxf(rp, rd)));
        }
      }
    }
    __syncthreads();
    // ---- A6: energy (the last lane);  A7 (part 1): dE/dG = -2 w_Q sum_j r_j y_j^T,
    // three columns of one row and contact a task, each entry summing j in
    // four partial sums (j mod 4, the tail into the first)
    if (const SetUp u = set_up(); u.active) {
      float* const per = u.per;
      for (int e = u.lane; e < 6 * M; e += LN) {
        const int i = e / 6, r = e % 6;
        const float* rec = per + L::oRY;
        float s[3][4];
#pragma unroll
        for (int cc = 0; cc < 3; ++cc)
#pragma unroll
          for (int u = 0; u < 4; ++u) s[cc][u] = 0.f;
        auto acc = [&](int jj, int u) {
          const float rv = rec[jj * L::RYW + r];
#pragma unroll
          for (int cc = 0; cc < 3; ++cc) s[cc][u] = fmaf(rv, rec[jj * L::RYW + 8 + 3 * i + cc], s[cc][u]);
        };
        int jj = 0;
        for (; jj + 3 < S; jj += 4) {
          acc(jj, 0);
          acc(jj + 1, 1);
          acc(jj + 2, 2);
          acc(jj + 3, 3);
        }
        for (; jj < S; ++jj) acc(jj, 0);
#pragma unroll
        for (int cc = 0; cc < 3; ++cc)
          per[L::oDG + 18 * i + 3 * r + cc] = -2.f * A.w_q * ((s[cc][0] + s[cc][1]) + (s[cc][2] + s[cc][3]));
      }
      if (u.lane == LN - 1) {
        float EQ = 0.f;
        for (int k = 0; k < S; ++k) EQ += per[L::oQ + k];
        float Ed = 0.f;
        for (int i = 0; i < M; ++i) {
          const float r = per[L::oCT + L::CTW * i + 9] - H.alpha - A.delta;
          Ed = fmaf(r, r, Ed);
        }
        float Ec = 0.f;
        if (A.coll)
          for (int l = 0; l < S; ++l) Ec += per[L::oGC + MAXD + l];
        per[L::oSC] = A.w_q * EQ + A.w_d * Ed + Ec;
      }
    }
    __syncthreads();
    // ---- A7 (part 2): through the contact geometry and the kinematic chain
    if (const SetUp u = set_up(); u.active && u.lane < M) {
      float* const per = u.per;
      const int lane = u.lane;
      const ContactGeo k = load_ct(per + L::oCT + L::CTW * lane);
      float cols[18];
#pragma unroll
      for (int e = 0; e < 18; ++e) cols[e] = per[L::oDG + 18 * lane + e];
      float dEdc[3];
      contact_adjoint(k, cols, 2.f * A.w_d * (k.phi - H.alpha - A.delta), dEdc);
      chain_adjoint(H, lane, per + L::oX, k.c, per + L::oJW + lane * MAXCHAIN * 6, dEdc, per + L::oCB + lane * (6 + MAXCHAIN));
    }
    __syncthreads();
    // ---- gradient assembly and A8: Adam + clamp
    if (const SetUp u = set_up(); u.active)
      assemble_step<M, MODE>(A, H, u.b, u.lane, LN, step, log2f(A.b1), log2f(A.b2), u.per);
    __syncthreads();
  }

  if (const SetUp u = set_up(); u.active) {
    const float* const per = u.per;
    const int lane = u.lane, b = u.b;
    if (lane == 0) {
      if (A.E) A.E[b] = per[L::oSC];
      if (A.status) A.status[b] = __float_as_int(per[L::oSC + 1]);
      if (A.res) A.res[b] = per[L::oSC + 2];
    }
    if (MODE == MODE_STEP)
      for (int k = lane; k < D; k += LN) {
        A.x_state[(size_t)b * D + k] = per[L::oX + k];
        A.am[(size_t)b * D + k] = per[L::oAM + k];
        A.av[(size_t)b * D + k] = per[L::oAV + k];
      }
  }
  if (const Solve v = solve(); v.mine) {
    const int ci = v.ci;
    const size_t q = v.q;
    if (warm) {
#pragma unroll
      for (int r = 0; r < 3; ++r) A.qy[(3 * ci + r) * NQ + q] = W.y[r];
#pragma unroll
      for (int k = 0; k < WPC; ++k) A.qw[(WPC * ci + k) * NQ + q] = W.w[k];
      if (ci == 0) A.qw[WPC * M * NQ + q] = W.wsum;
    }
    if (MODE == MODE_EVAL) {
      if (A.Qout && ci == 0) A.Qout[q] = v.per[L::oQ + v.j];
      if (A.yout)
#pragma unroll
        for (int r = 0; r < 3; ++r) A.yout[q * NV + 3 * ci + r] = W.y[r];
    }
  }
}

template <int M, int MODE, int CONE>
__global__ void __launch_bounds__(WIDE_THREADS, 4) fused_wide_kernel(FusedArgs A) {
  extern __shared__ __align__(16) float smem[];
  fused_wide_cta<M, MODE, CONE>(A, blockIdx.x, A.gpb, smem);
}

// ============================================================================ kernel: several jobs in one launch
// Jobs with different hand templates (m = 3, 4, 5), objects, batch sizes,
// wrench sets and step counts share one launch, every job's 200 (or n)
// upper steps inside it.  A work item is one tile of one job (the grasps of
// one CTA of that job's own launch).  Two schedules (step_params
// .work_pulling):
//   * one CTA per item, items numbered job by job in the caller's order:
//     the hardware's block scheduler hands them to SMs as slots free up;
//   * a persistent grid (PULL) of as many CTAs as fit on the GPU at once,
//     items numbered job by job in decreasing order of cost (steps x
//     wrenches x ADMM work per iteration, or steps x wrenches x contacts for
//     the exact solve): each CTA takes the next item from one global counter
//     (atomicAdd; zeroed by the host on the launch's stream before the
//     launch) until none is left.  Measured slower on the mixed-template
//     batch (the item loop costs the step registers: 488 bytes of spills at
//     the 168-register cap), so it is not the default.
// The job table travels in the kernel parameters.
struct MultiArgs {
  int n_jobs;
  int total;                            // work items
  int* counter;                         // next work item (device, zeroed before the launch)
  int m[BODEX_MAX_JOBS];
  int order_job[BODEX_MAX_JOBS];        // the jobs in the order of their items
  int order_begin[BODEX_MAX_JOBS + 1];  // first item of the k-th job in that order
  int rows, cols;                       // rows > 0: of each rows * cols blocks, b, b + cols, b + 2 cols ... take consecutive items
  FusedArgs job[BODEX_MAX_JOBS];
};

static_assert(sizeof(MultiArgs) <= 32000, "job table must fit in the kernel parameter space");

// Some job has fewer wrenches than contacts.
inline bool few_wrenches(const MultiArgs& A) {
  for (int j = 0; j < A.n_jobs; ++j)
    if (A.job[j].S < A.m[j]) return true;
  return false;
}

// Work item w: the k-th job in the item order, the tile w - order_begin[k].
template <bool ADAPT, bool EXACT, bool FEW>
__device__ __forceinline__ void multi_item(const MultiArgs& A, int w, float* smem) {
  constexpr int CN = EXACT ? CONE_EXACT : CONE_ANY;
  int k = 0;
  while (k + 1 < A.n_jobs && w >= A.order_begin[k + 1]) ++k;
  const int j = A.order_job[k];
  const FusedArgs& J = A.job[j];
  const int cta = w - A.order_begin[k];
  switch (A.m[j]) {
    case 3: fused_cta<3, MODE_STEP, CN, ADAPT, FEW>(J, cta, J.gpb, smem); break;
    case 4: fused_cta<4, MODE_STEP, CN, ADAPT, FEW>(J, cta, J.gpb, smem); break;
    default: fused_cta<5, MODE_STEP, CN, ADAPT, FEW>(J, cta, J.gpb, smem); break;
  }
}

// The same in the wide form (fixed rho, no pulling): every job's tile is one
// grasp, blocks as wide as the widest job needs; a warp that a job leaves
// without QPs still shares its set-up phases.  Taken where its estimate (form_time) is
// the shorter one: six jobs of three hands, 12 wrenches, 50
// steps of 50 iterations take 912 us instead of 1772 with 200 grasps
// together, 1321 (1873) with 900, 2396 (2553) with 1600; with 2000 the
// one-lane form is ahead, 2586 against 2691.  (A warp without QPs also runs
// every iteration, on zeros.)
template <int CONE>
__global__ void __launch_bounds__(WIDE_THREADS, 4) multi_wide_kernel(const __grid_constant__ MultiArgs A) {
  extern __shared__ __align__(16) float smem[];
  int k = 0;
  while (k + 1 < A.n_jobs && (int)blockIdx.x >= A.order_begin[k + 1]) ++k;
  const int j = A.order_job[k], cta = (int)blockIdx.x - A.order_begin[k];
  const FusedArgs& J = A.job[j];
  switch (A.m[j]) {
    case 3: fused_wide_cta<3, MODE_STEP, CONE>(J, cta, 1, smem); break;
    case 4: fused_wide_cta<4, MODE_STEP, CONE>(J, cta, 1, smem); break;
    default: fused_wide_cta<5, MODE_STEP, CONE>(J, cta, 1, smem); break;
  }
}

// FEW: some job may have fewer wrenches than contacts (see fused_cta).
template <bool ADAPT, bool EXACT = false, bool PULL = false, bool FEW = true>
__global__ void __launch_bounds__(CTA_LANES, 4) multi_kernel(const __grid_constant__ MultiArgs A) {
  extern __shared__ __align__(16) float smem[];
  if constexpr (!PULL) {
    int w = (int)blockIdx.x;
    if (EXACT && A.rows > 0) {
      // in waves of rows x cols blocks; column c of a wave has `rows` items,
      // or, in the last one, one fewer from column `full` on
      const int size = A.rows * A.cols, w0 = w / size * size, n = min(size, A.total - w0), i = w - w0;
      const int rows = (n + A.cols - 1) / A.cols, full = n - A.cols * (rows - 1), c = i % A.cols, r = i / A.cols;
      w = w0 + (c < full ? c * rows + r : full * rows + (c - full) * (rows - 1) + r);
    }
    multi_item<ADAPT, EXACT, FEW>(A, w, smem);  // one item per CTA, no loop
  } else {
    __shared__ int item;
#pragma unroll 1
    for (;;) {
      if (threadIdx.x == 0) item = atomicAdd(A.counter, 1);
      __syncthreads();
      const int w = item;
      __syncthreads();  // every thread has read the item before thread 0 takes the next
      if (w >= A.total) break;
      multi_item<ADAPT, EXACT, FEW>(A, w, smem);
      __syncthreads();  // shared memory is free for the next item
    }
  }
}

// ============================================================================ launch helpers
namespace bodex {

// Grasps per CTA: 96 lanes / s, capped by the shared memory one CTA may use.
template <int M>
inline int gpb_for(int s) {
  constexpr size_t kMaxSmem = 227 * 1024;
  const size_t per = 4u * (size_t)(Lay<M>::KS + Lay<M>::PER);
  const size_t fit = (kMaxSmem - 4u * Lay<M>::HAND_WORDS) / per;
  return std::max(1, std::min(CTA_LANES / s, (int)fit));
}

// Grasps per CTA of the batched QP kernel: 96 lanes / s, capped by its
// shared memory.
template <int M, int CONE>
inline int qp_gpb(int s) {
  constexpr size_t kMaxSmem = 227 * 1024;
  using L = LayQP<M, CONE>;
  const size_t per = 4u * (size_t)(L::KS + L::PER + s * L::PW);
  return std::max(1, std::min(CTA_LANES / s, (int)((kMaxSmem - 128) / per)));
}

// Grasps per CTA: the requested count (autotuner), else the default,
// never more than fit in 96 lanes and in shared memory.
template <int M>
inline int pick_gpb(int s, int requested) {
  const int cap = gpb_for<M>(s);
  return requested > 0 ? std::min(requested, cap) : cap;
}

// Multiprocessors of the current device (152 on a GB300).
inline int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
    (void)cudaGetLastError();
    n = 152;
  }
  return n;
}

// Threads of a wide CTA with gpb grasps: 32 / m QPs a warp.
template <int M>
inline int wide_threads(int gpb, int s) {
  constexpr int QPW = 32 / M;
  return 32 * ((gpb * s + QPW - 1) / QPW);
}

// Grasps per CTA of the wide fused step: one while the batch takes at most
// two warps a scheduler (the shortest steps), else the count that leaves the
// fewest lanes idle, the smallest on ties.
template <int M>
inline int wide_tile(int s, int B, int sms) {
  if ((long long)B * wide_threads<M>(1, s) <= 8LL * 32 * sms) return 1;
  int best = 1;
  for (int g = 2; wide_threads<M>(g, s) <= WIDE_THREADS && g <= gpb_for<M>(s); ++g)
    if (wide_threads<M>(g, s) * best < wide_threads<M>(best, s) * g) best = g;
  return best;
}

// Which form a fused step takes: the one whose estimated time is shorter (the
// results are bitwise the same).  Both are latency-bound steps that rise with
// the warps on the busiest scheduler, u = 1..4, and with every further wave of
// blocks: a bound in QPs per SM alone, fitted at 12 wrenches, was wrong by up
// to 1.8 times for others (five contacts, 16 wrenches, 94 QPs an SM: 116 -> 157
// us for 6 steps of 20 iterations, as the wide form's blocks of 3 warps take a
// second wave there; elliptic cone, 174 QPs, 3 iterations: 89 -> 159).
// Measured at 23 batch sizes of 8 to 238 QPs an SM, s = m, 8, 12 and 16, 3 to
// 150 iterations, with and without collision energies, us:
//   - an iteration, one lane per QP, by u: three contacts 0.17, 0.34, 0.51 (a
//     block has 3 warps, an SM at most 4 blocks); wide 0.09, 0.15, 0.20, 0.27;
//   - the set-up of a wave of blocks: a constant, and a part that grows with
//     the grasps and, wide, the warps an SM holds; the collision energies'
//     part of a one-lane block is spread over the s lanes of a grasp;
//   - a later wave of the wide form overlaps the one before: 0.75 to 0.99 of
//     its own time (its last blocks start as the first ones end).
// The wide form is taken below 0.93 of the one-lane estimate.  Over the 6624
// measured pairs that is within 0.6% of always taking the faster form, in the
// mean; the worst choice that is slower than one lane loses 9% (three
// contacts, 16 wrenches, 10 iterations).
struct FormCost {
  double set, grasp, warp, inv_s;             // set-up of a wave: set + grasp * grasps/SM + warp * warps/SM + inv_s / s
  double coll, coll_grasp, coll_warp, coll_inv_s;  // the same with the collision energies
  double pyr[4], soc[4];                      // one ADMM iteration by warps on the busiest scheduler
};
inline const FormCost& form_cost(bool wide, int m) {
  static const FormCost lane[3] = {
      {8.55, 0.07, 0, 0, 13.0, 0.19, 0, 47, {0.173, 0.335, 0.51, 0.51}, {0.465, 0.566, 0.68, 0.68}},
      {9.2, 0.11, 0, 0, 18.6, 0.25, 0, 92, {0.27, 0.495, 0.75, 0.75}, {0.68, 0.84, 1.02, 1.02}},
      {10.7, 0.10, 0, 0, 22.0, 0.19, 0, 147, {0.405, 0.70, 1.05, 1.05}, {1.03, 1.19, 1.41, 1.41}}};
  static const FormCost lanes[3] = {
      {7.07, 0.08, 0.09, 0, 11.7, 0.37, -0.05, 0, {0.089, 0.145, 0.203, 0.271}, {0.197, 0.232, 0.33, 0.40}},
      {7.18, 0.20, 0.11, 0, 16.1, 1.38, -0.27, 0, {0.103, 0.158, 0.236, 0.318}, {0.207, 0.244, 0.30, 0.36}},
      {7.35, 0.22, 0.12, 0, 18.6, 2.24, -0.43, 0, {0.117, 0.18, 0.26, 0.353}, {0.235, 0.278, 0.34, 0.42}}};
  return (wide ? lanes : lane)[m - 3];
}

// One job's part of a launch: `blocks` blocks of gpb grasps.
struct FormLoad {
  int m, s, gpb, blocks, steps;
};

// Blocks of a step kernel that an SM holds at once (by registers, 16 warps of
// the wide form or 12, and by shared memory).
inline int resident_blocks(bool wide, int threads, size_t bytes) {
  constexpr size_t kSmemPerSM = 228 * 1024, kReserved = 1024;  // 1 KB of every block is the system's
  return std::max(1, std::min((wide ? 16 : 12) / ((threads + 31) / 32), (int)(kSmemPerSM / (bytes + kReserved))));
}

// Estimated time of a launch of n jobs' blocks, `threads` wide with `bytes`
// of shared memory each, us.
inline double form_time(bool wide, const FormLoad* job, int n, int threads, size_t bytes, const AdmmCfg& c, bool coll,
                        int sms) {
  const int wpb = (threads + 31) / 32, resident = resident_blocks(wide, threads, bytes);
  // with a residual target the QPs of a warp rarely all stop early; beyond
  // 300 iterations the set-up no longer matters
  const double iters = c.eps > 0.f ? std::min(c.iters, 300) : c.iters;
  long long total = 0;
  int counts = 0;  // a bit per contact count
  for (int k = 0; k < n; ++k) {
    total += job[k].blocks;
    counts |= 1 << job[k].m;
  }
  const bool mixed = counts == (1 << 3 | 1 << 4 | 1 << 5);
  double t = 0;
  bool first = true;
  long long begun = 0;  // blocks of the waves so far
  for (long long per = (total + sms - 1) / sms; per > 0; first = false) {
    const int r = (int)std::min<long long>(per, resident), warps = r * wpb, u = std::min((warps + 3) / 4, 4);
    per -= r;
    double mean = 0, longest = 0;
    begun += (long long)r * sms;
    long long end = 0;  // of the k-th job's blocks, which start in the order of the jobs
    for (int k = 0; k < n; ++k) {
      const FormCost& f = form_cost(wide, job[k].m);
      const double g = (double)r * job[k].gpb;
      double v = coll ? f.coll + f.coll_grasp * g + f.coll_warp * warps + f.coll_inv_s / job[k].s
                      : f.set + f.grasp * g + f.warp * warps + f.inv_s / job[k].s;
      v = job[k].steps * (v + iters * (c.cone ? f.soc : f.pyr)[u - 1]);
      mean += v * job[k].blocks / total;
      end += job[k].blocks;
      if (wide || end > begun - (long long)r * sms) longest = std::max(longest, v);
    }
    // The launch ends with its longest blocks: in the one-lane form the
    // longest of the last wave's jobs (three jobs of hand5 and one of hand3,
    // 8 wrenches, cone, 4050 grasps: the last wave is hand3's alone, 272 us
    // where the wide form takes 366); in the wide form, whose waves of small
    // blocks drift apart with unequal step counts, the longest of all.
    double wave = per > 0 ? mean : longest;
    // three contact counts on an SM: the wide form's many small blocks run
    // three kernels' code at once (measured against the estimates: 1.13 to
    // 1.26 with four warps a scheduler, 1.08 below, 1.06 for the cone)
    if (wide && mixed) wave *= c.cone ? 1.06 : u == 4 ? 1.2 : 1.08;
    if (wide && !first) wave *= (c.cone ? 0.75 : 0.8) + 0.06 * (u - 1) + (coll ? 0.1 : 0.0);
    t += wave;
  }
  return t;
}

template <int M>
inline bool wide_pays(const FusedArgs& A, int sms) {
  const int g1 = pick_gpb<M>(A.S, 0), gw = wide_tile<M>(A.S, A.B, sms);
  const FormLoad lane = {M, A.S, g1, (A.B + g1 - 1) / g1, 1}, lanes = {M, A.S, gw, (A.B + gw - 1) / gw, 1};
  return form_time(true, &lanes, 1, wide_threads<M>(gw, A.S), Lay<M>::bytes(gw), A.cfg, A.coll != 0, sms) <
         0.93 * form_time(false, &lane, 1, g1 * A.S, Lay<M>::bytes(g1), A.cfg, A.coll != 0, sms);
}

// Raises the kernel's dynamic shared-memory limit when needed, once per
// device and size (so that launches recorded into a CUDA graph issue no
// attribute calls after the first).
template <class K>
inline int ensure_smem(K kernel, size_t bytes) {
  // A launch reports errors through cudaGetLastError; clear what an earlier,
  // already reported failure may have left behind (sticky device faults are
  // returned again by the next call regardless).
  (void)cudaGetLastError();
  if (bytes <= 48 * 1024) return BODEX_OK;
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, size_t> configured;  // (kernel, device) -> bytes
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = -1;
  const auto key = std::make_pair(reinterpret_cast<const void*>(kernel), dev);
  std::lock_guard<std::mutex> lock(mu);
  auto it = configured.find(key);
  if (it != configured.end() && it->second >= bytes) return BODEX_OK;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return cuda_fail(e, "cudaFuncSetAttribute");
  }
  configured[key] = bytes;
  return BODEX_OK;
}

}  // namespace bodex

// The kernel of a step or an evaluation.
using FusedKernel = void (*)(FusedArgs);
template <int M, int MODE>
inline FusedKernel fused_for(bool wide, bool exact, bool few, bool adapt, bool soc) {
  if (wide) return soc ? fused_wide_kernel<M, MODE, CONE_SOC> : fused_wide_kernel<M, MODE, CONE_PYR>;
  if (exact) return fused_kernel<M, MODE, CONE_EXACT, false>;
  if (few)  // adaptive rho, or DFC, which skips the lower level
    return soc ? fused_kernel<M, MODE, CONE_SOC, true, true> : fused_kernel<M, MODE, CONE_PYR, true, true>;
  if (adapt) return soc ? fused_kernel<M, MODE, CONE_SOC, true> : fused_kernel<M, MODE, CONE_PYR, true>;
  return soc ? fused_kernel<M, MODE, CONE_SOC, false> : fused_kernel<M, MODE, CONE_PYR, false>;
}

template <int M>
inline int run_fused(int mode, const FusedArgs& A0, cudaStream_t st) {
  if (A0.B == 0) return BODEX_OK;
  FusedArgs A = A0;
  const bool soc = A.cfg.cone != 0;
  const bool adapt = A.cfg.eps > 0.f && A.cfg.adapt;
  const bool few = A.S < M;  // fewer wrenches than contacts (ONE_CONTACT)
  // the wide form: ADMM at a fixed rho, where it pays and no tile is asked
  // for, and fewer wrenches than contacts
  bool wide = mode != MODE_ADJOINT && A.cfg.solver != BODEX_QP_EXACT && !adapt && !A.dfc;
  if (wide) {
    const int sms = sm_count();
    wide = few || (A0.gpb <= 0 && wide_pays<M>(A, sms));
    if (wide) A.gpb = wide_tile<M>(A.S, A.B, sms);
  }
  if (!wide) A.gpb = pick_gpb<M>(A.S, A0.gpb);
  const int gpb = A.gpb;
  const size_t bytes = Lay<M>::bytes(gpb);
  const dim3 grid((A.B + gpb - 1) / gpb), block(wide ? wide_threads<M>(gpb, A.S) : gpb * A.S);
  const bool exact = A.cfg.solver == BODEX_QP_EXACT;
  const FusedKernel kernel = mode == MODE_ADJOINT ? fused_kernel<M, MODE_ADJOINT, CONE_PYR, false>  // no lower-level solve
                             : mode == MODE_STEP  ? fused_for<M, MODE_STEP>(wide, exact, few, adapt, soc)
                                                  : fused_for<M, MODE_EVAL>(wide, exact, few, adapt, soc);
  if (int r = ensure_smem(kernel, bytes)) return r;
  kernel<<<grid, block, bytes, st>>>(A);
  return launch_err("fused_kernel launch");
}

// Puts the code of every step kernel of M contacts on the current device.
template <int M>
inline int load_steps() {
  for (int k = 0; k < 32; ++k) {
    cudaFuncAttributes a;
    const cudaError_t e =
        cudaFuncGetAttributes(&a, fused_for<M, MODE_STEP>(k & 1, (k & 2) != 0, (k & 4) != 0, (k & 8) != 0, (k & 16) != 0));
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncGetAttributes(step kernel)");
  }
  return BODEX_OK;
}

template <int M>
inline int run_qp(const float* G, int B, const float* T, int s, const AdmmCfg& cfg, int warm, float* y, float* z,
           float* lam, float* Q, int32_t* iters, int32_t* status, float* res, cudaStream_t st) {
  if (B == 0) return BODEX_OK;
  if (cfg.solver == BODEX_QP_EXACT) {
    const int gpb = std::max(1, CTA_LANES / s);
    const size_t bytes = 4u * (size_t)(ExactQP<M>::EDGE_WORDS + gpb * (s * ExactQP<M>::VW + 6 * 3 * M));
    qp_exact_kernel<M><<<(B + gpb - 1) / gpb, gpb * s, bytes, st>>>(G, B, T, s, cfg, y, z, lam, Q, iters, status,
                                                                    res);
    return launch_err("qp_exact_kernel launch");
  }
  // A small batch runs in the wide form from its first iteration, one grasp
  // a block, while that takes at most two warps a scheduler: up to there an
  // iteration is latency (see Wide).  Larger batches start with one QP a lane.
  constexpr int QPW = Wide<M, CONE_PYR>::QPW;
  const int wide_warps = (s + QPW - 1) / QPW;
  const bool wide = (long long)B * wide_warps <= 8LL * sm_count();
  const int gpb = wide ? 1 : cfg.cone ? qp_gpb<M, CONE_SOC>(s) : qp_gpb<M, CONE_PYR>(s);
  const int threads = wide ? 32 * wide_warps : gpb * s;
  const size_t bytes = cfg.cone ? LayQP<M, CONE_SOC>::bytes(gpb, s) : LayQP<M, CONE_PYR>::bytes(gpb, s);
  const bool adapt = cfg.eps > 0.f && cfg.adapt;
  auto go = [&](auto kernel) -> int {
    if (int r = ensure_smem(kernel, bytes)) return r;
    kernel<<<(B + gpb - 1) / gpb, threads, bytes, st>>>(G, B, T, s, gpb, cfg, warm, y, z, lam, Q, iters, status, res);
    return launch_err("qp_solve_kernel launch");
  };
  if (cfg.cone) return adapt ? go(qp_solve_kernel<M, CONE_SOC, true>) : go(qp_solve_kernel<M, CONE_SOC, false>);
  {
    const int r = adapt ? go(qp_solve_kernel<M, CONE_PYR, true>) : go(qp_solve_kernel<M, CONE_PYR, false>);
    if (r) return r;
    if (cfg.polish == 1 && cfg.eps_reg == 0.f) {
      const size_t n = (size_t)B * s;
      qp_polish_kernel<M><<<(unsigned)((n + 127) / 128), 128, 0, st>>>(G, B, T, s, cfg, y, Q, status);
      return launch_err("qp_polish_kernel launch");
    }
    if (cfg.polish == 2 && cfg.eps_reg == 0.f && cfg.eps > 0.f && status) {
      const size_t n = (size_t)B * s;
      qp_finish_kernel<M><<<(unsigned)((n + QP_FINISH_RANGE - 1) / QP_FINISH_RANGE), QP_FINISH_THREADS, 0, st>>>(
          G, B, T, s, cfg, y, Q, status);
      return launch_err("qp_finish_kernel launch");
    }
    return BODEX_OK;
  }
}

// Launchers, one translation unit each (fused_m*.cu, qp.cu, fused_multi*.cu).
int launch_fused_m3(int mode, const FusedArgs& A, cudaStream_t st);
int launch_fused_m4(int mode, const FusedArgs& A, cudaStream_t st);
int launch_fused_m5(int mode, const FusedArgs& A, cudaStream_t st);
int load_steps_m3();
int load_steps_m4();
int load_steps_m5();
int launch_qp(int m, const float* G, int B, const float* T, int s, const AdmmCfg& cfg, int warm, float* y, float* z,
              float* lam, float* Q, int32_t* iters, int32_t* status, float* res, cudaStream_t st);
int launch_multi(bool adapt, bool exact, const MultiArgs& MA, size_t bytes, cudaStream_t st);
int launch_multi_pull(bool adapt, bool exact, const MultiArgs& MA, size_t bytes, cudaStream_t st);
int launch_multi_wide(bool soc, const MultiArgs& MA, int threads, size_t bytes, cudaStream_t st);
