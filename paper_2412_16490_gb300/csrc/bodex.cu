// BODex coarse-stage hot path for GB300 (sm_103a): the C ABI declared in
// include/bodex.h and its small kernels (kinematics, refinement, metrics);
// the heavy kernels live in bodex_kernels.cuh and are compiled in their own
// translation units.
//
// Kernel layout.  One CTA holds GPB grasps and s lanes (threads) per grasp,
// GPB * s = 96 threads for s = 6 or 12.  Lane j of a grasp owns the QP of
// desired wrench t_j and keeps its ADMM iterate (y: 3m, w: 9m+1 floats) in
// registers; the grasp's G and explicit K^-1 sit in shared memory and are
// read by all of its lanes.  Lanes 0..m-1 also own one contact each for the
// kinematics, the SDF query and the adjoint.  The fused step kernel runs
// every upper iteration of a launch back to back without leaving the CTA:
// pose, Adam moments and warm starts never return to HBM between steps.

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/bodex.h"
#include "bodex_device.cuh"
#include "bodex_kernels.cuh"

using namespace bodex;

// ============================================================================ error state
namespace {
thread_local std::string g_err;
}  // namespace

namespace bodex {
int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}
int cuda_fail(cudaError_t e, const char* where) {
  return fail(BODEX_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}
int launch_err(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, what);
  return BODEX_OK;
}
}  // namespace bodex

#define BODEX_CUDA(call)                                    \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(e_, #call);     \
  } while (0)

namespace {
cudaStream_t as_stream(void* s) { return static_cast<cudaStream_t>(s); }
}  // namespace

struct bodex_hand_s {
  HandDev host;
  HandDev* dev = nullptr;
  float* tips = nullptr;  // [m, S, 3] fingertip surface samples (refinement)
  void* coll_mem = nullptr;  // collision spheres (one allocation behind coll's pointers)
  CollDev coll{};
};
struct bodex_object_s {
  ObjDev dev;
  float* grid = nullptr;
};
struct bodex_state_s {
  int B = 0, s = 0, m = 0, D = 0;
  float* x = nullptr;
  float* am = nullptr;
  float* av = nullptr;
  // ADMM warm start, component-major ([3m][B s] and [9m+1][B s]) so that the
  // fused kernel's per-step loads and stores are coalesced across lanes
  float* qy = nullptr;
  float* qw = nullptr;
  float* res = nullptr;  // [B] max QP residual at the last step of the last launch
  int* work = nullptr;   // work-item counter of a several-job launch led by this state
  int t = 0;
};

// ============================================================================ kernel: FK + contacts + G
// One thread per contact, FkTile<M>::GPB grasps a block: poses come in and
// the grasp matrices (18 floats a contact, spread over six rows) go out
// through shared memory, so that both are coalesced.  With one thread per
// grasp, walking its contacts in turn and storing 90 floats at a stride of
// 360 bytes, a batch of 16,384 five-finger poses was 512 warps of mostly
// waiting threads: 28 us.
template <int M>
struct FkTile {
  static constexpr int THREADS = 128, GPB = THREADS / M;
};

template <int M>
__global__ void __launch_bounds__(FkTile<M>::THREADS) fk_contacts_kernel(const HandDev* __restrict__ hand, ObjDev obj,
                                                          const float* __restrict__ x, int B, float* c_w,
                                                          float* p_out, float* n_out, float* phi_out, float* G_out,
                                                          int32_t* cell_out, int32_t* status_out) {
  constexpr int NV = 3 * M, GPB = FkTile<M>::GPB;
  __shared__ __align__(16) float hs[Lay<M>::HAND_WORDS];
  __shared__ float xs[GPB * MAXD];
  __shared__ float Gs[GPB * 6 * NV];
  __shared__ int stat[GPB];
  copy_hand_to_smem(hand, hs);
  const HandDev& H = *reinterpret_cast<const HandDev*>(hs);
  const int D = __ldg(&hand->D);
  const int b0 = blockIdx.x * GPB, ng = min(GPB, B - b0);
  if ((int)threadIdx.x < GPB) stat[threadIdx.x] = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < ng * D; e += blockDim.x) {
    const float v = x[(size_t)b0 * D + e];
    xs[e] = v;
    if (!isfinite(v)) atomicOr(stat + e / D, BODEX_ST_NONFINITE);
  }
  __syncthreads();
  const int gl = threadIdx.x / M, i = threadIdx.x % M;
  if (gl < ng) {
    const int b = b0 + gl;
    float c[3];
    fk_contact(H, i, xs + gl * D, c, nullptr);
    const ContactGeo k = contact_geometry(obj, c);
    int st = 0;
    if (k.degenerate) st |= BODEX_ST_DEGENERATE_NORMAL;
    if (!finite3(k.p) || !finite3(k.n) || !isfinite(k.phi)) st |= BODEX_ST_NONFINITE;
    if (st) atomicOr(stat + gl, st);
    write_G_block(k, i, NV, Gs + gl * 6 * NV);
    const size_t o = ((size_t)b * M + i) * 3;
    const float gc[3] = {obj.gcx, obj.gcy, obj.gcz};
    for (int a = 0; a < 3; ++a) {
      if (c_w) c_w[o + a] = k.c[a];
      if (p_out) p_out[o + a] = k.p[a] + gc[a];
      if (n_out) n_out[o + a] = k.n[a];
      if (cell_out) cell_out[o + a] = k.cell[a];
    }
    if (phi_out) phi_out[(size_t)b * M + i] = k.phi;
  }
  __syncthreads();
  if (G_out)
    for (int e = threadIdx.x; e < ng * 6 * NV; e += blockDim.x) G_out[(size_t)b0 * 6 * NV + e] = Gs[e];
  if (status_out && (int)threadIdx.x < ng) status_out[b0 + threadIdx.x] = stat[threadIdx.x];
}

// ============================================================================ kernel: refinement epilogue
// Fine / final stages (Sec. IV-C, Eqs. (10)-(11)) in SDF form, no QP.  Per
// contact: c^f = the fingertip sample with the smallest phi (lowest index on
// ties), p^f its nearest object point, c^{f'} = R_i s_{k*} + T_i with the
// sample's link-frame coordinates held fixed (the Detach of Eq. (11)), and
//   E = w_d sum |c^{f'} - (p^f + delta n_out)|^2 + w_qp sum |c^{f'} - p^c|^2
// with p^f, n_out and the coarse-stage points p^c treated as constants.
// delta is the pre-grasp margin (Sec. IV-D): 1 cm in the fine stage, 0 in
// the final one.  Lanes 0..m-1 own a contact's adjoint, all lanes of a grasp
// share the gradient assembly and Adam, and no block barrier stands between
// steps.  Two forms:
//   - a warp per grasp: all 32 lanes share each fingertip's samples (160
//     queries a grasp and step with 32 samples), the chains are walked by
//     three lanes a contact, one row of the frames each, and the lowest sample
//     is found by two warp reductions.  A step of 4096 five-finger grasps in a
//     64^3 grid takes 14.3 us, with eight lanes 34.6: those are bound by the
//     latency of 32 queries in a row;
//   - eight lanes per grasp: a lane walks its contact's chain and samples.  A
//     warp holds four grasps' serial parts, so where the queries are few or
//     cheap and the batch fills the GPU it is the shorter one: 16,384 grasps
//     with 7 samples 24 us a step instead of 42, on a sphere object with 32
//     samples 14.0 instead of 23.2.
// warp_per_grasp chooses.  Both find the same sample and give the same bits.
struct RefineArgs {
  const HandDev* hand;
  const float* tips;
  ObjDev obj;
  int B;
  const float* pc;
  float delta, w_d, w_qp;
  float lr_t, lr_r, b1, b2, adam_eps;
  int n_steps, t0;
  int S;  // samples per fingertip
  float* x;
  float* am;
  float* av;
  float* E;
  int32_t* kstar;
  int32_t* status;
};

// The refinement and metrics kernels: blocks of 128 threads, LANES (32 or 8) a grasp.
constexpr int RF_THREADS = 128;

// The fingertip sample with the smallest phi over the warp, lowest index on
// ties (0 if none compares below infinity): T is the contact's link frame.
// phi receives the smallest value (infinity if none).
__device__ __forceinline__ int lowest_sample(const Tf& T, const float* __restrict__ tip, int S, const ObjDev& obj,
                                             float& phi) {
  const int lane = threadIdx.x % 32;
  float best = INFINITY;
  int kbest = 0;
  for (int k = lane; k < S; k += 32) {
    const float sk[3] = {__ldg(tip + 3 * k), __ldg(tip + 3 * k + 1), __ldg(tip + 3 * k + 2)};
    float ck[3];
    tf_point(T, sk, ck);
    const float ph = sdf_query(obj, ck).phi;
    if (ph < best) {
      best = ph;
      kbest = k;
    }
  }
  // two warp reductions (five shuffles and compares of a pair each before):
  // the smallest value as an integer of the same order, then the lowest index
  // that has it; adding 0 makes the two zeros one
  const int v = __float_as_int(best + 0.f);
  const unsigned key = (unsigned)(v ^ ((v >> 31) | (int)0x80000000));
  const unsigned lo = __reduce_min_sync(0xffffffffu, key);
  kbest = __reduce_min_sync(0xffffffffu, key == lo ? kbest : 0x7fffffff);
  phi = __int_as_float((lo & 0x80000000u) ? (int)(lo ^ 0x80000000u) : (int)~lo);
  return phi < INFINITY ? kbest : 0;
}

// A link frame in shared memory, 12 words.
__device__ __forceinline__ void load_frame(const float* f, Tf& T) {
#pragma unroll
  for (int e = 0; e < 9; ++e) T.R[e] = f[e];
  T.t[0] = f[9];
  T.t[1] = f[10];
  T.t[2] = f[11];
}

// Contact i's samples walked by one lane: the smallest phi (infinity if none
// compares below it) and the lowest index that has it.
__device__ __forceinline__ int lowest_sample_lane(const Tf& T, const float* __restrict__ tip, int S, const ObjDev& obj,
                                                  float& phi) {
  phi = INFINITY;
  int kbest = 0;
  for (int k = 0; k < S; ++k) {
    const float sk[3] = {__ldg(tip + 3 * k), __ldg(tip + 3 * k + 1), __ldg(tip + 3 * k + 2)};
    float ck[3];
    tf_point(T, sk, ck);
    const float ph = sdf_query(obj, ck).phi;
    if (ph < phi) {
      phi = ph;
      kbest = k;
    }
  }
  return kbest;
}

template <int M, int LANES>
__global__ void __launch_bounds__(RF_THREADS) refine_kernel(RefineArgs A) {
  constexpr bool WARP = LANES == 32;  // else a lane walks its contact's chain and samples
  constexpr int HW = Lay<M>::HAND_WORDS, GPB = RF_THREADS / LANES;
  constexpr int CBW = 6 + MAXCHAIN;
  constexpr int oEi = 3 * MAXD + M * CBW + M * MAXCHAIN * 6 + (WARP ? M * 12 : 0);
  constexpr int oRQ = oEi + M + 1;  // joint rotations and the root frame (WARP)
  constexpr int PER = align4(oRQ + (WARP ? 9 * MAXJ + 12 : 0) + 4);
  __shared__ __align__(16) float smem[HW + GPB * PER];
  copy_hand_to_smem(A.hand, smem);
  const int gl = threadIdx.x / LANES, lane = threadIdx.x % LANES;
  const int b_mine = blockIdx.x * GPB + gl;
  const int b = WARP ? b_mine : min(b_mine, A.B - 1);  // eight lanes past the last grasp repeat it and write nothing
  const HandDev& H = *reinterpret_cast<const HandDev*>(smem);
  float* per = smem + HW + gl * PER;
  float* xs = per;
  float* ams = per + MAXD;
  float* avs = per + 2 * MAXD;
  float* cb = per + 3 * MAXD;
  float* jwall = cb + M * CBW;
  float* frames = jwall + M * MAXCHAIN * 6;  // WARP
  float* Ei = per + oEi;
  int* stat = reinterpret_cast<int*>(Ei + M);
  __syncthreads();
  if (b_mine - (int)(threadIdx.x % 32) / LANES >= A.B) return;  // whole warps; no block barrier below
  const int D = H.D, S = H.S;
  for (int k = lane; k < D; k += LANES) {
    xs[k] = A.x[(size_t)b * D + k];
    ams[k] = A.am[(size_t)b * D + k];
    avs[k] = A.av[(size_t)b * D + k];
  }
  if (lane == 0) *stat = 0;
  __syncwarp();
  int kbest = 0;
  for (int step = 0; step < A.n_steps; ++step) {
    float* const jw = jwall + (lane < M ? lane : 0) * MAXCHAIN * 6;
    if constexpr (WARP) {
      for (int e = lane; e <= H.n; e += 32) fk_joint(H, e, xs, per + oRQ, per + oRQ + 9 * MAXJ);
      __syncwarp();
      if (lane < 3 * M)
        fk_row(H, lane / 3, lane % 3, per + oRQ, per + oRQ + 9 * MAXJ, jwall + (lane / 3) * MAXCHAIN * 6, nullptr,
               frames + 12 * (lane / 3), nullptr);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < M; ++i) {
        Tf T;
        load_frame(frames + 12 * i, T);
        float phi;
        const int k = lowest_sample(T, A.tips + (size_t)i * S * 3, S, A.obj, phi);
        if (lane == i) kbest = k;
      }
    }
    if (lane < M) {
      Tf T;
      if constexpr (WARP) {
        load_frame(frames + 12 * lane, T);
      } else {
        fk_link(H, lane, xs, T, jw);
        float phi;
        kbest = lowest_sample_lane(T, A.tips + (size_t)lane * S * 3, S, A.obj, phi);
      }
      const float* tip = A.tips + (size_t)lane * S * 3;
      const float sk[3] = {__ldg(tip + 3 * kbest), __ldg(tip + 3 * kbest + 1), __ldg(tip + 3 * kbest + 2)};
      float cf[3];
      tf_point(T, sk, cf);
      const ContactGeo k = contact_geometry(A.obj, cf);
      const float gc[3] = {A.obj.gcx, A.obj.gcy, A.obj.gcz};
      const float* pci = A.pc + ((size_t)b * M + lane) * 3;
      float dEdc[3], e = 0.f;
      for (int a = 0; a < 3; ++a) {
        const float target = k.p[a] + gc[a] - A.delta * k.n[a];
        const float da = cf[a] - target, db = cf[a] - pci[a];
        e += A.w_d * da * da + A.w_qp * db * db;
        dEdc[a] = 2.f * A.w_d * da + 2.f * A.w_qp * db;
      }
      Ei[lane] = e;
      if (k.degenerate) atomicOr(stat, BODEX_ST_DEGENERATE_NORMAL);
      if (!isfinite(e)) atomicOr(stat, BODEX_ST_NONFINITE);
      chain_adjoint(H, lane, xs, cf, jw, dEdc, cb + lane * CBW);
    }
    __syncwarp();
    {
      const int tstep = A.t0 + step + 1;
      const float c1 = 1.f - exp2f((float)tstep * log2f(A.b1)), c2 = 1.f - exp2f((float)tstep * log2f(A.b2));
      if (lane == 0 && A.E) {
        float e = 0.f;
        for (int i = 0; i < M; ++i) e += Ei[i];
        per[PER - 1] = e;
      }
      for (int k = lane; k < D; k += LANES) {
        float g = 0.f;
        if (k < 6) {
#pragma unroll
          for (int i = 0; i < M; ++i) g += cb[i * CBW + k];
        } else {
          float v[M];  // every load before the sum: a contact that the joint does not move adds 0
#pragma unroll
          for (int i = 0; i < M; ++i) {
            const int pos = H.jpos[i][k - 6];
            const float e = cb[i * CBW + 6 + max(pos, 0)];
            v[i] = pos >= 0 ? e : 0.f;
          }
#pragma unroll
          for (int i = 0; i < M; ++i) g += v[i];
        }
        const float mm = fmaf(A.b1, ams[k], (1.f - A.b1) * g);
        const float vv = fmaf(A.b2, avs[k], (1.f - A.b2) * g * g);
        ams[k] = mm;
        avs[k] = vv;
        const float lr = k < 3 ? A.lr_t : A.lr_r;
        const float xn = xs[k] - lr * (mm / c1) / (sqrtf(vv / c2) + A.adam_eps);
        xs[k] = fminf(fmaxf(xn, H.qmin[k]), H.qmax[k]);
      }
    }
    __syncwarp();
  }
  if (!WARP && b_mine >= A.B) return;
  for (int k = lane; k < D; k += LANES) {
    A.x[(size_t)b * D + k] = xs[k];
    A.am[(size_t)b * D + k] = ams[k];
    A.av[(size_t)b * D + k] = avs[k];
  }
  if (lane < M && A.kstar && A.n_steps > 0) A.kstar[(size_t)b * M + lane] = kbest;
  if (lane == 0) {
    if (A.E) A.E[b] = per[PER - 1];
    if (A.status) A.status[b] = *stat;
  }
}

// ============================================================================ kernel: contact metrics
// Contact Distance Consistency (Sec. V-B): d_i = the signed distance of
// fingertip i, the smallest phi over its surface samples (phi(c_i) - alpha
// for a hand without samples); cdc = max_i d_i - min_i d_i.  In the two forms
// of the refinement: with a warp per grasp 4096 five-finger poses with 32
// samples take 20 us (eight lanes 37), 16,384 poses 48 (60); with eight lanes
// 16,384 poses with 7 samples 22 (35).
struct MetricsArgs {
  const HandDev* hand;
  const float* tips;  // [m, S, 3] or null
  ObjDev obj;
  int B;
  int S;  // samples per fingertip, 0 without
  const float* x;
  float* d;    // [B, m]
  float* cdc;  // [B], may be null
};

template <int M, int LANES>
__global__ void __launch_bounds__(RF_THREADS) metrics_kernel(MetricsArgs A) {
  constexpr bool WARP = LANES == 32;
  constexpr int HW = Lay<M>::HAND_WORDS, GPB = RF_THREADS / LANES;
  constexpr int oRQ = align4(MAXD) + 12 * M;  // joint rotations and the root frame (WARP)
  constexpr int PER = WARP ? oRQ + 9 * MAXJ + 12 : align4(MAXD);
  __shared__ __align__(16) float smem[HW + GPB * PER];
  copy_hand_to_smem(A.hand, smem);
  const int gl = threadIdx.x / LANES, lane = threadIdx.x % LANES;
  const int b_mine = blockIdx.x * GPB + gl;
  const int b = WARP ? b_mine : min(b_mine, A.B - 1);  // eight lanes past the last grasp repeat it and write nothing
  const HandDev& H = *reinterpret_cast<const HandDev*>(smem);
  float* xs = smem + HW + gl * PER;
  float* frames = xs + align4(MAXD);  // WARP
  __syncthreads();
  if (b_mine - (int)(threadIdx.x % 32) / LANES >= A.B) return;  // whole warps; no block barrier below
  const int D = H.D, S = A.tips ? H.S : 0;
  for (int k = lane; k < D; k += LANES) xs[k] = A.x[(size_t)b * D + k];
  __syncwarp();
  float d = 0.f;
  if constexpr (WARP) {  // S > 0
    for (int e = lane; e <= H.n; e += 32) fk_joint(H, e, xs, xs + oRQ, xs + oRQ + 9 * MAXJ);
    __syncwarp();
    if (lane < 3 * M)
      fk_row(H, lane / 3, lane % 3, xs + oRQ, xs + oRQ + 9 * MAXJ, nullptr, nullptr, frames + 12 * (lane / 3), nullptr);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < M; ++i) {
      Tf T;
      load_frame(frames + 12 * i, T);
      float phi;
      (void)lowest_sample(T, A.tips + (size_t)i * S * 3, S, A.obj, phi);
      if (lane == i) d = phi;
    }
  } else if (lane < M) {
    Tf T;
    fk_link(H, lane, xs, T, nullptr);
    if (S > 0) {
      (void)lowest_sample_lane(T, A.tips + (size_t)lane * S * 3, S, A.obj, d);
    } else {
      float c[3];
      tf_point(T, H.clocal[lane], c);
      d = sdf_query(A.obj, c).phi - H.alpha;
    }
  }
  // spread over the grasp's fingers (in its lowest eight lanes)
  float lo = lane < M ? d : INFINITY, hi = lane < M ? d : -INFINITY;
#pragma unroll
  for (int off = 4; off >= 1; off >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
  }
  if (!WARP && b_mine >= A.B) return;
  if (lane < M) A.d[(size_t)b * M + lane] = d;
  if (lane == 0 && A.cdc) A.cdc[b] = hi - lo;
}

// ============================================================================ host helpers
namespace {

int check_qp_params(const bodex_qp_params* p, int m) {
  if (!p) return fail(BODEX_ERR_INVALID, "null qp params");
  if (!(p->gamma >= 0.f) || p->gamma > (float)m)
    return fail(BODEX_ERR_INFEASIBLE, "gamma must lie in [0, m]");
  if (!(p->rho > 0.f) || !(p->sigma >= 0.f) || !(p->alpha > 0.f && p->alpha < 2.f) || p->max_iter < 0 ||
      !(p->mu >= 0.f))
    return fail(BODEX_ERR_INVALID, "invalid ADMM parameters");
  if (p->cone != BODEX_CONE_PYRAMID && p->cone != BODEX_CONE_ELLIPTIC)
    return fail(BODEX_ERR_INVALID, "cone must be BODEX_CONE_PYRAMID or BODEX_CONE_ELLIPTIC");
  if (p->solver != BODEX_QP_ADMM && p->solver != BODEX_QP_EXACT)
    return fail(BODEX_ERR_INVALID, "solver must be BODEX_QP_ADMM or BODEX_QP_EXACT");
  if (p->polish < 0 || p->polish > 2) return fail(BODEX_ERR_INVALID, "polish must be 0, 1 or 2");
  if (p->solver == BODEX_QP_EXACT && (p->cone != BODEX_CONE_PYRAMID || p->eps_reg != 0.f || p->max_iter < 1))
    return fail(BODEX_ERR_INVALID, "the exact solver needs the pyramid cone, eps_reg = 0 and max_iter >= 1");
  return BODEX_OK;
}

int dispatch_fused(int m, int mode, const FusedArgs& A, cudaStream_t st) {
  switch (m) {
    case 3: return launch_fused_m3(mode, A, st);
    case 4: return launch_fused_m4(mode, A, st);
    case 5: return launch_fused_m5(mode, A, st);
    default: return fail(BODEX_ERR_INVALID, "m must be 3, 4 or 5");
  }
}

template <int M>
int run_fk(const bodex_hand_s* h, const bodex_object_s* o, const float* x, int B, float* c_w, float* p, float* n,
           float* phi, float* G, int32_t* cell, int32_t* status, cudaStream_t st) {
  if (B == 0) return BODEX_OK;
  (void)cudaGetLastError();
  fk_contacts_kernel<M><<<(B + FkTile<M>::GPB - 1) / FkTile<M>::GPB, FkTile<M>::THREADS, 0, st>>>(h->dev, o->dev, x, B, c_w, p, n, phi, G, cell, status);
  return launch_err("fk_contacts_kernel launch");
}

}  // namespace

namespace {
// Whether refinement and metrics take a warp per grasp: above a number of
// samples a finger that grows with the grasps an SM holds (g) until the batch
// fills the GPU.  Measured at 64 to 65,536 grasps and 1 to 128 samples, us a
// step, eight lanes -> a warp.  64^3 grid, five fingers: 2000 grasps, 2
// samples 5.9 -> 7.6, 4: 7.6 -> 7.7, 8: 11.1 -> 7.9; 5000 grasps, 10: 16.5 ->
// 17.9 (four fingers 13.9 -> 15.7); 6000 grasps, 8: 14.6 -> 18.9, 12: 19.2 ->
// 19.3, 16: 24.1 -> 19.9; 65,536 grasps, 12: 136 -> 165, 16: 194 -> 170 (three
// fingers 16: 83 -> 107, 24: 115 -> 113, and 20,000 grasps with 20 44 -> 35; the
// metrics cross at some 18 for every hand, 28,000 grasps of three fingers with
// 20 take 56 -> 44 us; hence `most`).  Sphere, whose queries are
// arithmetic alone: 2000 grasps, 12: 4.3 -> 4.4, 24: 5.3 -> 4.3; 6000, 32: 8.0
// -> 9.9, 48: 9.5 -> 11.4, 64: 11.6 -> 11.3; 65,536, 64: 76 -> 102, 128: 128
// -> 127.  More than 32 samples are two and more rounds of the warp.
template <int M>
bool warp_per_grasp(const ObjDev& obj, int S, int B, double most) {
  const double g = (double)B / sm_count(), rounds = S > 32 ? 0.8 * S : S;
  return rounds > (obj.kind == 0 ? std::min(std::max(1.0, g), 80.0) : std::min(std::max(2.0, 0.31 * g), most));
}

template <int M>
int run_refine(const RefineArgs& A, cudaStream_t st) {
  (void)cudaGetLastError();
  if (warp_per_grasp<M>(A.obj, A.S, A.B, std::min(19.0, 64.0 / M)))
    refine_kernel<M, 32><<<(A.B + RF_THREADS / 32 - 1) / (RF_THREADS / 32), RF_THREADS, 0, st>>>(A);
  else
    refine_kernel<M, 8><<<(A.B + RF_THREADS / 8 - 1) / (RF_THREADS / 8), RF_THREADS, 0, st>>>(A);
  return launch_err("refine_kernel launch");
}

template <int M>
int run_metrics(const MetricsArgs& A, cudaStream_t st) {
  (void)cudaGetLastError();
  if (warp_per_grasp<M>(A.obj, A.S, A.B, 19.0))
    metrics_kernel<M, 32><<<(A.B + RF_THREADS / 32 - 1) / (RF_THREADS / 32), RF_THREADS, 0, st>>>(A);
  else
    metrics_kernel<M, 8><<<(A.B + RF_THREADS / 8 - 1) / (RF_THREADS / 8), RF_THREADS, 0, st>>>(A);
  return launch_err("metrics_kernel launch");
}
}  // namespace

// ============================================================================ hand collision spheres
// Shared-memory room the fused kernel has for the collision scratch of one
// grasp (sphere centres and per-slot sums), by contact count.
static int coll_room(int m) {
  switch (m) {
    case 3: return Lay<3>::COLL_CS;
    case 4: return Lay<4>::COLL_CS;
    default: return Lay<5>::COLL_CS;
  }
}
static int frame_room(int m) {
  switch (m) {
    case 3: return Lay<3>::COLL_FR;
    case 4: return Lay<4>::COLL_FR;
    default: return Lay<5>::COLL_FR;
  }
}

// Orders the spheres by slot (link, then the root), bounds each slot's
// spheres, lists the slot pairs allowed for self-penetration, and uploads
// them in one allocation.  Pair rule: spheres on different links, except a
// link and its nearest ancestor link that carries spheres (the root counts).
static int upload_spheres(bodex_hand_s* h, const bodex_hand_desc* d) {
  const int K = d->n_spheres, n = h->host.n;
  if (K == 0) return BODEX_OK;
  if (K < 0 || K > BODEX_MAX_SPHERES) return fail(BODEX_ERR_INVALID, "n_spheres out of range");
  if (!d->sphere_link || !d->sphere_local || !d->sphere_radius)
    return fail(BODEX_ERR_INVALID, "null sphere array in hand descriptor");
  std::vector<int> slot(K);
  for (int k = 0; k < K; ++k) {
    const int L = d->sphere_link[k];
    if (L < -1 || L >= n) return fail(BODEX_ERR_INVALID, "sphere_link out of range");
    if (!(d->sphere_radius[k] > 0.f)) return fail(BODEX_ERR_INVALID, "sphere_radius must be > 0");
    slot[k] = L < 0 ? n : L;
  }

  if (3 * K + 9 * (n + 1) > coll_room(h->host.m) || 12 * (n + 1) > frame_room(h->host.m))
    return fail(BODEX_ERR_INVALID, "too many collision spheres and joints for this contact count");
  // the collision phase takes its link frames from the contact kinematics
  for (int k = 0; k < K; ++k) {
    const int L = d->sphere_link[k];
    bool on_chain = L < 0;
    for (int i = 0; i < h->host.m && !on_chain; ++i) on_chain = h->host.jpos[i][L] >= 0;
    if (!on_chain) return fail(BODEX_ERR_INVALID, "a sphere link lies on no contact chain");
  }
  std::vector<int> order(K);
  for (int k = 0; k < K; ++k) order[k] = k;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return slot[a] < slot[b]; });
  std::vector<char> has(n, 0);
  for (int k = 0; k < K; ++k)
    if (d->sphere_link[k] >= 0) has[d->sphere_link[k]] = 1;
  auto eff_parent = [&](int L) {  // -1: the root; -2: none (L is the root)
    if (L < 0) return -2;
    int p = h->host.parent[L];
    while (p >= 0 && !has[p]) p = h->host.parent[p];
    return p;
  };
  std::vector<float4> sph(K);
  std::vector<int> slot_start(n + 2, 0);
  for (int a = 0; a < K; ++a) {
    const int ka = order[a];
    sph[a] = make_float4(d->sphere_local[3 * ka], d->sphere_local[3 * ka + 1], d->sphere_local[3 * ka + 2],
                         d->sphere_radius[ka]);
    ++slot_start[slot[ka] + 1];
  }
  for (int L = 0; L <= n; ++L) slot_start[L + 1] += slot_start[L];
  // bounding sphere of each slot's spheres (centre: their mean), and the
  // slot pairs allowed for self-penetration
  std::vector<float4> sbound(n + 1, make_float4(0.f, 0.f, 0.f, 0.f));
  for (int L = 0; L <= n; ++L) {
    const int k0 = slot_start[L], k1 = slot_start[L + 1];
    if (k0 == k1) continue;
    double c[3] = {0, 0, 0};
    for (int k = k0; k < k1; ++k) {
      c[0] += sph[k].x;
      c[1] += sph[k].y;
      c[2] += sph[k].z;
    }
    for (double& v : c) v /= (k1 - k0);
    double R = 0;
    for (int k = k0; k < k1; ++k) {
      const double dx = sph[k].x - c[0], dy = sph[k].y - c[1], dz = sph[k].z - c[2];
      R = std::max(R, std::sqrt(dx * dx + dy * dy + dz * dz) + sph[k].w);
    }
    sbound[L] = make_float4((float)c[0], (float)c[1], (float)c[2], (float)(R * (1.0 + 1e-5)) + 1e-6f);
  }
  auto link_of = [&](int L) { return L == n ? -1 : L; };
  std::vector<int> spstart(n + 2, 0), spartners;
  for (int L = 0; L <= n; ++L) {
    for (int L2 = 0; L2 <= n; ++L2) {
      if (L2 == L || slot_start[L] == slot_start[L + 1] || slot_start[L2] == slot_start[L2 + 1]) continue;
      const int la = link_of(L), lb = link_of(L2);
      if (eff_parent(la) == lb || eff_parent(lb) == la) continue;
      spartners.push_back(L2);
    }
    spstart[L + 1] = (int)spartners.size();
  }
  const size_t b_sph = sizeof(float4) * K, b_sb = sizeof(float4) * (n + 1), b_ss = sizeof(int) * (n + 2),
               b_sp = sizeof(int) * (n + 2), b_pa = sizeof(int) * std::max<size_t>(1, spartners.size());
  const size_t o_sb = b_sph, o_ss = o_sb + b_sb, o_sp = o_ss + b_ss, o_pa = o_sp + b_sp;
  const size_t o_sl = o_pa + b_pa;  // each sphere's slot, in slot order
  std::vector<int> sphere_slot(K);
  for (int a = 0; a < K; ++a) sphere_slot[a] = slot[order[a]];
  std::vector<char> blob(o_sl + sizeof(int) * K);
  std::memcpy(blob.data() + o_sl, sphere_slot.data(), sizeof(int) * K);
  std::memcpy(blob.data(), sph.data(), b_sph);
  std::memcpy(blob.data() + o_sb, sbound.data(), b_sb);
  std::memcpy(blob.data() + o_ss, slot_start.data(), b_ss);
  std::memcpy(blob.data() + o_sp, spstart.data(), b_sp);
  if (!spartners.empty()) std::memcpy(blob.data() + o_pa, spartners.data(), sizeof(int) * spartners.size());
  if (cudaMalloc(&h->coll_mem, blob.size()) != cudaSuccess) {
    h->coll_mem = nullptr;
    return fail(BODEX_ERR_OOM, "cudaMalloc collision spheres");
  }
  cudaError_t e = cudaMemcpy(h->coll_mem, blob.data(), blob.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy collision spheres");
  char* base = static_cast<char*>(h->coll_mem);
  h->coll.K = K;
  h->coll.sph = reinterpret_cast<const float4*>(base);
  h->coll.sbound = reinterpret_cast<const float4*>(base + o_sb);
  h->coll.slot_start = reinterpret_cast<const int*>(base + o_ss);
  h->coll.spstart = reinterpret_cast<const int*>(base + o_sp);
  h->coll.spartners = reinterpret_cast<const int*>(base + o_pa);
  h->coll.sphere_slot = reinterpret_cast<const int*>(base + o_sl);
  return BODEX_OK;
}

extern "C" int bodex_hand_destroy(bodex_hand_t h);

// ============================================================================ C ABI
extern "C" {

const char* bodex_last_error(void) { return g_err.c_str(); }
const char* bodex_version(void) { return "bodex-gb300 0.1 (sm_103a)"; }

int bodex_step_tile(int m, int s, int requested, int* grasps_per_cta) {
  if (!grasps_per_cta || s < 1 || s > SMAX || requested < 0)
    return fail(BODEX_ERR_INVALID, "bodex_step_tile: s outside 1..16, requested < 0 or null output");
  switch (m) {
    case 3: *grasps_per_cta = pick_gpb<3>(s, requested); break;
    case 4: *grasps_per_cta = pick_gpb<4>(s, requested); break;
    case 5: *grasps_per_cta = pick_gpb<5>(s, requested); break;
    default: return fail(BODEX_ERR_INVALID, "bodex_step_tile: m must be 3, 4 or 5");
  }
  return BODEX_OK;
}

int bodex_sync(void* stream) {
  BODEX_CUDA(cudaStreamSynchronize(as_stream(stream)));
  return BODEX_OK;
}

int bodex_hand_create(const bodex_hand_desc* d, bodex_hand_t* out) {
  if (!d || !out) return fail(BODEX_ERR_INVALID, "null argument");
  *out = nullptr;
  const int n = d->n_joints, m = d->n_contacts;
  if (n < 1 || n > MAXJ) return fail(BODEX_ERR_INVALID, "n_joints out of range");
  if (m < 3 || m > MAXM) return fail(BODEX_ERR_INVALID, "n_contacts must be 3..5");
  if (!d->parent || !d->offset || !d->axis || !d->qmin || !d->qmax || !d->contact_link || !d->contact_local)
    return fail(BODEX_ERR_INVALID, "null array in hand descriptor");
  HandDev H;
  std::memset(&H, 0, sizeof(H));
  H.n = n;
  H.m = m;
  H.D = 6 + n;
  H.alpha = d->contact_radius;
  H.S = d->n_tip_samples;
  for (int j = 0; j < n; ++j) {
    H.parent[j] = d->parent[j];
    if (H.parent[j] >= j || H.parent[j] < -1) return fail(BODEX_ERR_INVALID, "parent[j] must be -1 or < j");
    for (int e = 0; e < 12; ++e) H.offset[j][e] = d->offset[12 * j + e];
    for (int e = 0; e < 3; ++e) H.axis[j][e] = d->axis[3 * j + e];
  }
  for (int k = 0; k < 6 + n; ++k) {
    H.qmin[k] = d->qmin[k];
    H.qmax[k] = d->qmax[k];
    if (!(H.qmin[k] <= H.qmax[k])) return fail(BODEX_ERR_INFEASIBLE, "qmin > qmax");
  }
  for (int i = 0; i < MAXM; ++i)
    for (int j = 0; j < MAXJ; ++j) H.jpos[i][j] = -1;
  for (int i = 0; i < m; ++i) {
    H.clink[i] = d->contact_link[i];
    if (H.clink[i] < 0 || H.clink[i] >= n) return fail(BODEX_ERR_INVALID, "contact_link out of range");
    for (int a = 0; a < 3; ++a) H.clocal[i][a] = d->contact_local[3 * i + a];
    int chain[MAXJ], L = 0;
    for (int j = H.clink[i]; j >= 0; j = H.parent[j]) chain[L++] = j;
    if (L > MAXCHAIN) return fail(BODEX_ERR_INVALID, "contact chain longer than BODEX_MAX_CHAIN");
    H.chain_len[i] = L;
    for (int k = 0; k < L; ++k) {
      H.chain[i][k] = chain[L - 1 - k];
      H.jpos[i][chain[L - 1 - k]] = (int8_t)k;
    }
  }
  if (H.S < 0 || (H.S > 0 && !d->tip_samples)) return fail(BODEX_ERR_INVALID, "tip samples missing");
  bodex_hand_s* h = new bodex_hand_s();
  h->host = H;
  cudaError_t e = cudaMalloc(&h->dev, sizeof(HandDev));
  if (e != cudaSuccess) {
    delete h;
    return fail(BODEX_ERR_OOM, "cudaMalloc hand");
  }
  if (H.S > 0) {
    const size_t bytes = (size_t)m * H.S * 3 * sizeof(float);
    e = cudaMalloc(&h->tips, bytes);
    if (e != cudaSuccess) {
      cudaFree(h->dev);
      delete h;
      return fail(BODEX_ERR_OOM, "cudaMalloc tip samples");
    }
    e = cudaMemcpy(h->tips, d->tip_samples, bytes, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
      cudaFree(h->tips);
      cudaFree(h->dev);
      delete h;
      return cuda_fail(e, "cudaMemcpy tip samples");
    }
  }
  e = cudaMemcpy(h->dev, &h->host, sizeof(HandDev), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    if (h->tips) cudaFree(h->tips);
    cudaFree(h->dev);
    delete h;
    return cuda_fail(e, "cudaMemcpy hand");
  }
  if (int r = upload_spheres(h, d)) {
    bodex_hand_destroy(h);
    return r;
  }
  *out = h;
  return BODEX_OK;
}

int bodex_hand_destroy(bodex_hand_t h) {
  if (!h) return BODEX_OK;
  if (h->tips) cudaFree(h->tips);
  if (h->coll_mem) cudaFree(h->coll_mem);
  cudaFree(h->dev);
  delete h;
  return BODEX_OK;
}

int bodex_object_create(const bodex_object_desc* d, void* stream, bodex_object_t* out) {
  if (!d || !out) return fail(BODEX_ERR_INVALID, "null argument");
  *out = nullptr;
  bodex_object_s* o = new bodex_object_s();
  std::memset(&o->dev, 0, sizeof(ObjDev));
  if (d->kind == 0) {
    if (!(d->radius > 0.f)) {
      delete o;
      return fail(BODEX_ERR_INVALID, "sphere radius must be > 0");
    }
    o->dev.kind = 0;
    o->dev.cx = d->center[0];
    o->dev.cy = d->center[1];
    o->dev.cz = d->center[2];
    o->dev.r = d->radius;
    o->dev.gcx = d->center[0];
    o->dev.gcy = d->center[1];
    o->dev.gcz = d->center[2];
  } else if (d->kind == 1) {
    const int N = d->n;
    if (N < 2 || !(d->h > 0.f) || !d->values) {
      delete o;
      return fail(BODEX_ERR_INVALID, "grid needs n >= 2, h > 0 and values");
    }
    const size_t cnt = (size_t)N * N * N;
    o->dev.kind = 1;
    o->dev.N = N;
    o->dev.h = d->h;
    o->dev.inv_h = 1.0f / d->h;
    o->dev.ox = d->origin[0];
    o->dev.oy = d->origin[1];
    o->dev.oz = d->origin[2];
    // gravity centre: mean of the node positions inside the object (double)
    double sx = 0, sy = 0, sz = 0;
    long long inside = 0;
    for (int iz = 0; iz < N; ++iz)
      for (int iy = 0; iy < N; ++iy)
        for (int ix = 0; ix < N; ++ix)
          if (d->values[((size_t)iz * N + iy) * N + ix] < 0.f) {
            sx += (double)d->origin[0] + (double)d->h * ix;
            sy += (double)d->origin[1] + (double)d->h * iy;
            sz += (double)d->origin[2] + (double)d->h * iz;
            ++inside;
          }
    if (inside > 0) {
      o->dev.gcx = (float)(sx / inside);
      o->dev.gcy = (float)(sy / inside);
      o->dev.gcz = (float)(sz / inside);
    } else {
      const double half = 0.5 * (double)d->h * (N - 1);
      o->dev.gcx = (float)(d->origin[0] + half);
      o->dev.gcy = (float)(d->origin[1] + half);
      o->dev.gcz = (float)(d->origin[2] + half);
    }
    cudaError_t e = cudaMalloc(&o->grid, cnt * sizeof(float));
    if (e != cudaSuccess) {
      delete o;
      return fail(BODEX_ERR_OOM, "cudaMalloc grid");
    }
    e = cudaMemcpyAsync(o->grid, d->values, cnt * sizeof(float), cudaMemcpyHostToDevice, as_stream(stream));
    if (e != cudaSuccess) {
      cudaFree(o->grid);
      delete o;
      return cuda_fail(e, "cudaMemcpyAsync grid");
    }
    o->dev.grid = o->grid;
  } else {
    delete o;
    return fail(BODEX_ERR_INVALID, "object kind must be 0 (sphere) or 1 (grid)");
  }
  *out = o;
  return BODEX_OK;
}

int bodex_object_destroy(bodex_object_t o) {
  if (!o) return BODEX_OK;
  if (o->grid) cudaFree(o->grid);
  delete o;
  return BODEX_OK;
}

int bodex_object_gravity_centre(bodex_object_t o, float out[3]) {
  if (!o || !out) return fail(BODEX_ERR_INVALID, "null argument");
  out[0] = o->dev.gcx;
  out[1] = o->dev.gcy;
  out[2] = o->dev.gcz;
  return BODEX_OK;
}

int bodex_fk_contacts(bodex_hand_t h, bodex_object_t o, const float* x, int B, float* c_w, float* p, float* n,
                      float* phi, float* G, int32_t* cell, int32_t* status, void* stream) {
  if (!h || !o || (!x && B > 0) || B < 0) return fail(BODEX_ERR_INVALID, "null handle/pose or B < 0");
  cudaStream_t st = as_stream(stream);
  switch (h->host.m) {
    case 3: return run_fk<3>(h, o, x, B, c_w, p, n, phi, G, cell, status, st);
    case 4: return run_fk<4>(h, o, x, B, c_w, p, n, phi, G, cell, status, st);
    case 5: return run_fk<5>(h, o, x, B, c_w, p, n, phi, G, cell, status, st);
  }
  return fail(BODEX_ERR_INVALID, "unsupported m");
}

int bodex_qp_solve_batch(const float* G, int B, int m, const float* T, int s, const bodex_qp_params* params,
                         float* y, float* z, float* lam, float* Q, int32_t* iters, int32_t* status, float* res,
                         void* stream) {
  if (B < 0 || s < 1 || s > SMAX) return fail(BODEX_ERR_INVALID, "B < 0 or s outside 1..16");
  if (B > 0 && (!G || !T || !y || !z || !lam || !Q)) return fail(BODEX_ERR_INVALID, "null array");
  if (int r = check_qp_params(params, m)) return r;
  if (params->strict && !status) return fail(BODEX_ERR_INVALID, "strict mode needs a status array");
  if (params->polish == 2 && !status) return fail(BODEX_ERR_INVALID, "polish = 2 needs a status array");
  AdmmCfg cfg = admm_cfg(*params);
  // K^-1 in FP64 for any residual target: an FP32 K^-1 raises the ADMM floor
  // (on the paper batch 98.2% instead of 99.5% of the QPs reach 1e-5)
  cfg.fp64_setup = params->eps_abs > 0.f ? 1 : 0;
  cudaStream_t st = as_stream(stream);
  if (m < 3 || m > 5) return fail(BODEX_ERR_INVALID, "m must be 3, 4 or 5");
  const int r = launch_qp(m, G, B, T, s, cfg, params->warm, y, z, lam, Q, iters, status, res, st);
  if (r || !params->strict || B == 0) return r;
  std::vector<int32_t> hs((size_t)B * s);
  BODEX_CUDA(cudaMemcpyAsync(hs.data(), status, hs.size() * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  BODEX_CUDA(cudaStreamSynchronize(st));
  for (int32_t v : hs)
    if (v & BODEX_ST_NOT_CONVERGED) return fail(BODEX_ERR_NOT_CONVERGED, "a QP missed eps_abs");
  return BODEX_OK;
}

int bodex_state_create(bodex_hand_t h, int B, int s, bodex_state_t* out) {
  if (!h || !out || B < 0 || s < 1 || s > SMAX) return fail(BODEX_ERR_INVALID, "bad state arguments");
  *out = nullptr;
  bodex_state_s* S = new bodex_state_s();
  S->B = B;
  S->s = s;
  S->m = h->host.m;
  S->D = h->host.D;
  const size_t nx = (size_t)B * S->D, ny = (size_t)B * s * 3 * S->m, nw = (size_t)B * s * (9 * S->m + 1);
  float** bufs[6] = {&S->x, &S->am, &S->av, &S->qy, &S->qw, &S->res};
  const size_t cnt[6] = {nx, nx, nx, ny, nw, (size_t)B};
  for (int k = 0; k < 6; ++k) {
    if (cnt[k] == 0) continue;
    if (cudaMalloc(bufs[k], cnt[k] * sizeof(float)) != cudaSuccess) {
      for (int j = 0; j < k; ++j) cudaFree(*bufs[j]);
      delete S;
      return fail(BODEX_ERR_OOM, "cudaMalloc state");
    }
    cudaMemset(*bufs[k], 0, cnt[k] * sizeof(float));
  }
  if (cudaMalloc(&S->work, sizeof(int)) != cudaSuccess) {
    for (int k = 0; k < 6; ++k) cudaFree(*bufs[k]);
    delete S;
    return fail(BODEX_ERR_OOM, "cudaMalloc state");
  }
  *out = S;
  return BODEX_OK;
}

int bodex_state_destroy(bodex_state_t S) {
  if (!S) return BODEX_OK;
  cudaFree(S->work);
  cudaFree(S->res);
  cudaFree(S->x);
  cudaFree(S->am);
  cudaFree(S->av);
  cudaFree(S->qy);
  cudaFree(S->qw);
  delete S;
  return BODEX_OK;
}

int bodex_state_set_pose(bodex_state_t S, const float* x, void* stream) {
  if (!S || (!x && S->B > 0)) return fail(BODEX_ERR_INVALID, "null argument");
  if (S->B == 0) return BODEX_OK;
  cudaStream_t st = as_stream(stream);
  const size_t nx = (size_t)S->B * S->D;
  BODEX_CUDA(cudaMemcpyAsync(S->x, x, nx * sizeof(float), cudaMemcpyDeviceToDevice, st));
  BODEX_CUDA(cudaMemsetAsync(S->am, 0, nx * sizeof(float), st));
  BODEX_CUDA(cudaMemsetAsync(S->av, 0, nx * sizeof(float), st));
  BODEX_CUDA(cudaMemsetAsync(S->qy, 0, (size_t)S->B * S->s * 3 * S->m * sizeof(float), st));
  BODEX_CUDA(cudaMemsetAsync(S->qw, 0, (size_t)S->B * S->s * (9 * S->m + 1) * sizeof(float), st));
  S->t = 0;
  return BODEX_OK;
}

int bodex_state_get_pose(bodex_state_t S, float* x, void* stream) {
  if (!S || (!x && S->B > 0)) return fail(BODEX_ERR_INVALID, "null argument");
  if (S->B == 0) return BODEX_OK;
  BODEX_CUDA(cudaMemcpyAsync(x, S->x, (size_t)S->B * S->D * sizeof(float), cudaMemcpyDeviceToDevice,
                             as_stream(stream)));
  return BODEX_OK;
}

int bodex_state_get_residual(bodex_state_t S, float* res, void* stream) {
  if (!S || (!res && S->B > 0)) return fail(BODEX_ERR_INVALID, "null argument");
  if (S->B == 0) return BODEX_OK;
  BODEX_CUDA(cudaMemcpyAsync(res, S->res, (size_t)S->B * sizeof(float), cudaMemcpyDeviceToDevice,
                             as_stream(stream)));
  return BODEX_OK;
}

int bodex_state_get_adam(bodex_state_t S, float* m, float* v, int* step, void* stream) {
  if (!S) return fail(BODEX_ERR_INVALID, "null state");
  const size_t nx = (size_t)S->B * S->D * sizeof(float);
  if (m && nx) BODEX_CUDA(cudaMemcpyAsync(m, S->am, nx, cudaMemcpyDeviceToDevice, as_stream(stream)));
  if (v && nx) BODEX_CUDA(cudaMemcpyAsync(v, S->av, nx, cudaMemcpyDeviceToDevice, as_stream(stream)));
  if (step) *step = S->t;
  return BODEX_OK;
}

static int fill_args(FusedArgs& A, bodex_hand_t h, bodex_object_t o, const float* T, int s, int B,
                     const bodex_step_params* p) {
  if (!h || !o || !p || !T || s < 1 || s > SMAX || B < 0) return fail(BODEX_ERR_INVALID, "bad arguments");
  if (int r = check_qp_params(&p->qp, h->host.m)) return r;
  std::memset(&A, 0, sizeof(A));
  A.hand = h->dev;
  A.obj = o->dev;
  A.T = T;
  A.S = s;
  A.B = B;
  A.cfg = admm_cfg(p->qp);
  A.w_q = p->energy.w_q;
  A.w_d = p->energy.w_d;
  A.delta = p->energy.delta;
  A.lr_t = p->lr_t;
  A.lr_r = p->lr_r;
  A.b1 = p->b1;
  A.b2 = p->b2;
  A.adam_eps = p->adam_eps;
  // a tight residual target moves ADMM's fixed point with the backward
  // error of K^-1: build it in double there
  A.cfg.fp64_setup = (p->qp.eps_abs > 0.f && p->qp.eps_abs <= 2e-6f) ? 1 : 0;
  A.gpb = p->grasps_per_cta;
  if (p->energy.kind != BODEX_ENERGY_QP && p->energy.kind != BODEX_ENERGY_DFC)
    return fail(BODEX_ERR_INVALID, "energy.kind must be BODEX_ENERGY_QP or BODEX_ENERGY_DFC");
  A.dfc = p->energy.kind == BODEX_ENERGY_DFC;
  const bodex_energy_params& e = p->energy;
  if (!(e.eta_pen >= 0.f) || !(e.eta_lim >= 0.f)) return fail(BODEX_ERR_INVALID, "eta_pen and eta_lim must be >= 0");
  A.coll = (e.w_pen != 0.f || e.w_self != 0.f || e.w_lim != 0.f) ? 1 : 0;
  A.cd = h->coll;
  A.cp = CollParams{e.w_pen, e.w_self, e.w_lim, e.eta_pen, e.eta_lim};
  return BODEX_OK;
}

int bodex_energy_grad(bodex_hand_t h, bodex_object_t o, const float* x, int B, const float* T, int s,
                      const bodex_step_params* params, bodex_state_t warm, float* E, float* dEdx, float* Q,
                      float* y, int32_t* status, void* stream) {
  FusedArgs A;
  if (int r = fill_args(A, h, o, T, s, B, params)) return r;
  if (B > 0 && (!x || !E)) return fail(BODEX_ERR_INVALID, "null x or E");
  if (warm && (warm->B != B || warm->s != s || warm->m != h->host.m))
    return fail(BODEX_ERR_INVALID, "warm state shape mismatch");
  A.n_steps = 1;
  A.x_in = x;
  A.qy = warm ? warm->qy : nullptr;
  A.qw = warm ? warm->qw : nullptr;
  A.E = E;
  A.dEdx = dEdx;
  A.Qout = Q;
  A.yout = y;
  A.status = status;
  return dispatch_fused(h->host.m, MODE_EVAL, A, as_stream(stream));
}

int bodex_energy_adjoint(bodex_hand_t h, bodex_object_t o, const float* x, int B, const float* T, int s,
                         const bodex_step_params* params, const float* y, float* E, float* dEdx, int32_t* status,
                         void* stream) {
  FusedArgs A;
  if (int r = fill_args(A, h, o, T, s, B, params)) return r;
  if (B > 0 && (!x || !y || !dEdx)) return fail(BODEX_ERR_INVALID, "null x, y or dEdx");
  A.n_steps = 1;
  A.x_in = x;
  A.yin = y;
  A.E = E;
  A.dEdx = dEdx;
  A.status = status;
  return dispatch_fused(h->host.m, MODE_ADJOINT, A, as_stream(stream));
}

int bodex_step(bodex_hand_t h, bodex_object_t o, bodex_state_t S, const float* T, int s, int n_steps,
               const bodex_step_params* params, float* E_last, int32_t* status, void* stream) {
  if (!S) return fail(BODEX_ERR_INVALID, "null state");
  FusedArgs A;
  if (int r = fill_args(A, h, o, T, s, S->B, params)) return r;
  if (S->s != s || S->m != h->host.m) return fail(BODEX_ERR_INVALID, "state shape mismatch");
  if (n_steps < 0) return fail(BODEX_ERR_INVALID, "n_steps < 0");
  if (n_steps == 0) return BODEX_OK;
  A.n_steps = n_steps;
  A.t0 = S->t;
  A.x_state = S->x;
  A.am = S->am;
  A.av = S->av;
  A.qy = S->qy;
  A.qw = S->qw;
  A.E = E_last;
  A.status = status;
  A.res = S->res;
  const int r = dispatch_fused(h->host.m, MODE_STEP, A, as_stream(stream));
  if (r == BODEX_OK) S->t += n_steps;
  return r;
}

int bodex_step_multi(const bodex_job* jobs, int n_jobs, const bodex_step_params* params, void* stream) {
  if (n_jobs < 0 || n_jobs > BODEX_MAX_JOBS || (n_jobs > 0 && !jobs) || !params)
    return fail(BODEX_ERR_INVALID, "n_jobs must be 0..BODEX_MAX_JOBS with a job array");
  MultiArgs* MA = new MultiArgs();  // ~15 KB: kept off the host stack
  std::memset(MA, 0, sizeof(MultiArgs));
  size_t bytes = 0;
  int total = 0, nj = 0;
  // the wide form for all jobs or none: ADMM at a fixed rho, no tile or
  // pulling asked for, where its estimated time is shorter (form_time)
  const bool exact = params->qp.solver == BODEX_QP_EXACT;
  const bool adapt = !exact && params->qp.eps_abs > 0.f && params->qp.adaptive_rho;
  const bool soc = params->qp.cone != BODEX_CONE_PYRAMID;
  bool wide = !exact && !adapt && params->energy.kind != BODEX_ENERGY_DFC && params->grasps_per_cta <= 0 && !params->work_pulling;
  int threads = 0;
  size_t wide_bytes = 0;
  FormLoad lane[BODEX_MAX_JOBS], lanes[BODEX_MAX_JOBS];
  int lane_threads = 0;
  bool coll = false;
  int take[BODEX_MAX_JOBS], tiles[BODEX_MAX_JOBS];
  double cost[BODEX_MAX_JOBS];
  for (int j = 0; j < n_jobs; ++j) {
    const bodex_job& J = jobs[j];
    bodex_state_t S = J.state;
    if (!J.hand || !J.obj || !S) {
      delete MA;
      return fail(BODEX_ERR_INVALID, "job with a null handle");
    }
    if (S->s != J.s || S->m != J.hand->host.m || S->D != J.hand->host.D || J.n_steps < 0) {
      delete MA;
      return fail(BODEX_ERR_INVALID, "job state shape mismatch or n_steps < 0");
    }
    if (S->B == 0 || J.n_steps == 0) continue;
    FusedArgs& A = MA->job[nj];
    if (int r = fill_args(A, J.hand, J.obj, J.T, J.s, S->B, params)) {
      delete MA;
      return r;
    }
    const int m = J.hand->host.m;
    int gpb = 0;
    size_t b = 0;
    switch (m) {
      case 3: gpb = pick_gpb<3>(J.s, A.gpb); b = Lay<3>::bytes(gpb); break;
      case 4: gpb = pick_gpb<4>(J.s, A.gpb); b = Lay<4>::bytes(gpb); break;
      default: gpb = pick_gpb<5>(J.s, A.gpb); b = Lay<5>::bytes(gpb); break;
    }
    A.gpb = gpb;
    A.n_steps = J.n_steps;
    A.t0 = S->t;
    A.x_state = S->x;
    A.am = S->am;
    A.av = S->av;
    A.qy = S->qy;
    A.qw = S->qw;
    A.E = J.E_last;
    A.status = J.status;
    A.res = S->res;
    MA->m[nj] = m;
    switch (m) {
      case 3: threads = std::max(threads, wide_threads<3>(1, J.s)); wide_bytes = std::max(wide_bytes, Lay<3>::bytes(1)); break;
      case 4: threads = std::max(threads, wide_threads<4>(1, J.s)); wide_bytes = std::max(wide_bytes, Lay<4>::bytes(1)); break;
      default: threads = std::max(threads, wide_threads<5>(1, J.s)); wide_bytes = std::max(wide_bytes, Lay<5>::bytes(1)); break;
    }
    tiles[nj] = (S->B + gpb - 1) / gpb;
    lane[nj] = {m, J.s, gpb, tiles[nj], J.n_steps};
    lanes[nj] = {m, J.s, 1, S->B, J.n_steps};
    lane_threads = std::max(lane_threads, gpb * J.s);
    coll = A.coll != 0;
    // cost of one tile: steps x wrenches x (ADMM work per iteration, 26 m + 9 m^2 + ...,
    // taken as m^2; or m for the exact solve, whose oracle is linear in m)
    cost[nj] = (double)J.n_steps * J.s * (exact ? m : m * m);
    total += tiles[nj];
    bytes = std::max(bytes, b);
    take[nj] = j;
    ++nj;
  }
  if (wide && nj > 0) {
    const int sms = sm_count();
    const AdmmCfg& c = MA->job[0].cfg;
    wide = form_time(true, lanes, nj, threads, wide_bytes, c, coll, sms) <
           0.96 * form_time(false, lane, nj, lane_threads, bytes, c, coll, sms);
  }
  if (wide) {
    total = 0;
    for (int k = 0; k < nj; ++k) {
      MA->job[k].gpb = 1;
      total += tiles[k] = MA->job[k].B;
    }
  }
  MA->n_jobs = nj;
  MA->total = total;
  int r = BODEX_OK;
  if (nj > 0) {
    // work items job by job: the costliest job's tiles first (stable on
    // ties) for the pulling schedule, the caller's order otherwise (but see
    // the exact QPs below)
    const bool pull = params->work_pulling != 0;
    int ord[BODEX_MAX_JOBS];
    for (int k = 0; k < nj; ++k) ord[k] = k;
    if (pull) std::stable_sort(ord, ord + nj, [&](int a, int b2) { return cost[a] > cost[b2]; });
    // Exact QPs: the solver's code for two or three contact counts on one SM
    // misses the instruction cache.  So the items go count by count, and up to
    // some two waves the blocks of an SM in a wave (block b goes to SM b mod
    // the number of SMs) take consecutive ones; beyond, the SMs drift apart.
    // Five jobs of three hands, 5 steps of 12 wrenches: 4864 grasps together
    // took 1.51 times as long in the caller's order as the former solver at two
    // blocks an SM, and take 0.51; 3800: 1.46 and 0.55; 6100: 1.03 and 0.61.
    // Two hands, 4600 grasps: 1.09 and 0.70.
    if (exact && !pull) {
      bool counts[MAXM + 1] = {};
      for (int k = 0; k < nj; ++k) counts[MA->m[k]] = true;
      if (counts[3] + counts[4] + counts[5] > 1) {
        std::stable_sort(ord, ord + nj, [&](int a, int b2) { return MA->m[a] > MA->m[b2]; });
        const int sms = sm_count(), rows = resident_blocks(false, CTA_LANES, bytes);
        if (total <= 2.25 * rows * sms) {
          MA->rows = rows;
          MA->cols = sms;
        }
      }
    }
    int acc = 0;
    for (int k = 0; k < nj; ++k) {
      MA->order_job[k] = ord[k];
      MA->order_begin[k] = acc;
      acc += tiles[ord[k]];
    }
    MA->order_begin[nj] = acc;
    // the item counter lives with the first job's state (calls that share a
    // state are serialised by the caller, so no two launches share it)
    MA->counter = jobs[take[0]].state->work;
    cudaStream_t st = as_stream(stream);
    if (pull) {
      const cudaError_t e = cudaMemsetAsync(MA->counter, 0, sizeof(int), st);
      if (e != cudaSuccess) {
        delete MA;
        return cuda_fail(e, "cudaMemsetAsync(work counter)");
      }
    }
    r = wide   ? launch_multi_wide(soc, *MA, threads, wide_bytes, st)
        : pull ? launch_multi_pull(adapt, exact, *MA, bytes, st)
               : launch_multi(adapt, exact, *MA, bytes, st);
    if (r == BODEX_OK)
      for (int k = 0; k < nj; ++k) jobs[take[k]].state->t += jobs[take[k]].n_steps;
  }
  delete MA;
  return r;
}

// ============================================================================ refinement ABI
extern "C" int bodex_refine(bodex_hand_t h, bodex_object_t o, bodex_state_t S, const float* p_coarse, int n_steps,
                            float delta, float w_qp, const bodex_step_params* p, float* E_last, int32_t* kstar,
                            int32_t* status, void* stream) {
  if (!h || !o || !S || !p) return fail(BODEX_ERR_INVALID, "null argument");
  if (h->host.S <= 0 || !h->tips) return fail(BODEX_ERR_INVALID, "hand has no fingertip samples");
  if (S->m != h->host.m || S->D != h->host.D) return fail(BODEX_ERR_INVALID, "state shape mismatch");
  if (n_steps < 0) return fail(BODEX_ERR_INVALID, "n_steps < 0");
  if (S->B > 0 && !p_coarse) return fail(BODEX_ERR_INVALID, "null p_coarse");
  if (n_steps == 0 || S->B == 0) return BODEX_OK;
  RefineArgs A;
  std::memset(&A, 0, sizeof(A));
  A.hand = h->dev;
  A.tips = h->tips;
  A.obj = o->dev;
  A.B = S->B;
  A.pc = p_coarse;
  A.delta = delta;
  A.w_d = p->energy.w_d;
  A.w_qp = w_qp;
  A.lr_t = p->lr_t;
  A.lr_r = p->lr_r;
  A.b1 = p->b1;
  A.b2 = p->b2;
  A.adam_eps = p->adam_eps;
  A.n_steps = n_steps;
  A.t0 = S->t;
  A.S = h->host.S;
  A.x = S->x;
  A.am = S->am;
  A.av = S->av;
  A.E = E_last;
  A.kstar = kstar;
  A.status = status;
  int r;
  switch (h->host.m) {
    case 3: r = run_refine<3>(A, as_stream(stream)); break;
    case 4: r = run_refine<4>(A, as_stream(stream)); break;
    case 5: r = run_refine<5>(A, as_stream(stream)); break;
    default: return fail(BODEX_ERR_INVALID, "unsupported m");
  }
  if (r == BODEX_OK) S->t += n_steps;
  return r;
}

extern "C" int bodex_contact_metrics(bodex_hand_t h, bodex_object_t o, const float* x, int B, float* d, float* cdc,
                                     void* stream) {
  if (!h || !o) return fail(BODEX_ERR_INVALID, "null handle");
  if (B < 0) return fail(BODEX_ERR_INVALID, "B < 0");
  if (B > 0 && (!x || !d)) return fail(BODEX_ERR_INVALID, "null x or d");
  if (B == 0) return BODEX_OK;
  MetricsArgs A;
  std::memset(&A, 0, sizeof(A));
  A.hand = h->dev;
  A.tips = (h->host.S > 0) ? h->tips : nullptr;
  A.obj = o->dev;
  A.B = B;
  A.S = A.tips ? h->host.S : 0;
  A.x = x;
  A.d = d;
  A.cdc = cdc;
  switch (h->host.m) {
    case 3: return run_metrics<3>(A, as_stream(stream));
    case 4: return run_metrics<4>(A, as_stream(stream));
    case 5: return run_metrics<5>(A, as_stream(stream));
    default: return fail(BODEX_ERR_INVALID, "unsupported m");
  }
}

// ============================================================================ squeeze pose
// x_s = 2 x - x_p (Sec. IV-D), elementwise over B * D floats; 2 x is exact
// in float, so the one rounding gives the same value as the formula.
__global__ void __launch_bounds__(256) squeeze_kernel(const float* __restrict__ x, const float* __restrict__ xp,
                                                      size_t n, float* __restrict__ xs) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    xs[i] = fmaf(2.f, x[i], -xp[i]);
}

extern "C" int bodex_squeeze_pose(const float* x, const float* x_p, int B, int D, float* x_s, void* stream) {
  if (B < 0 || D < 1) return fail(BODEX_ERR_INVALID, "B < 0 or D < 1");
  if (B > 0 && (!x || !x_p || !x_s)) return fail(BODEX_ERR_INVALID, "null array");
  if (B == 0) return BODEX_OK;
  const size_t n = (size_t)B * D;
  const unsigned blocks = (unsigned)std::min<size_t>((n + 255) / 256, 4096);
  (void)cudaGetLastError();
  squeeze_kernel<<<blocks, 256, 0, as_stream(stream)>>>(x, x_p, n, x_s);
  return launch_err("squeeze_kernel launch");
}

// ============================================================================ allocation-free step
// Some callers cannot allocate device memory once they are running: a robot
// controller that reserves everything at start-up so that its control loop
// has bounded latency, an application whose memory pool owns the whole
// device and forbids cudaMalloc, or a plug-in hosted by such a process.
// bodex_step_noalloc serves them.  The per-grasp state that bodex_step keeps
// in a bodex_state_t (Adam moments and the ADMM warm start of every QP) lives
// instead in the fixed array below, which every GPU that loads this library
// holds until the process exits.  The caller still passes the poses, the
// wrenches and the outputs.
namespace {
constexpr size_t kNoallocScratchFloats = size_t(1) << 20;  // 4 MiB per device
constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mu;
float* g_noalloc_addr[kNoallocMaxDevices] = {};
bool g_noalloc_loaded[kNoallocMaxDevices][MAXM + 1] = {};  // the step kernels of m contacts
}  // namespace

static __device__ __align__(256) float g_noalloc_scratch[kNoallocScratchFloats];

// Device address of the scratch array on the current device.  Host code may
// not use the symbol itself (it names a host-side stand-in), so the address
// is looked up once per device, with that device current, and cached.  The
// first call with a contact count also loads every step kernel of that count:
// which one runs depends on the batch, the wrenches and the parameters, and
// lazy loading would take device memory at the first launch of each (2 MB at
// the first large batch after a warm-up with a small one).
static int noalloc_scratch(int m, float** out) {
  int dev = 0;
  BODEX_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoallocMaxDevices) return fail(BODEX_ERR_INVALID, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    g_noalloc_addr[dev] = static_cast<float*>(p);
  }
  if (!g_noalloc_loaded[dev][m]) {
    if (int r = m == 3 ? load_steps_m3() : m == 4 ? load_steps_m4() : load_steps_m5()) return r;
    g_noalloc_loaded[dev][m] = true;
  }
  *out = g_noalloc_addr[dev];
  return BODEX_OK;
}

extern "C" int bodex_step_noalloc(bodex_hand_t h, bodex_object_t o, float* x, int B, const float* T, int s,
                                  int n_steps, const bodex_step_params* params, float* E_last, int32_t* status,
                                  void* stream) {
  FusedArgs A;
  if (int r = fill_args(A, h, o, T, s, B, params)) return r;
  if (B > 0 && !x) return fail(BODEX_ERR_INVALID, "null x");
  if (n_steps < 0) return fail(BODEX_ERR_INVALID, "n_steps < 0");
  const size_t D = (size_t)h->host.D, m = (size_t)h->host.m;
  auto up = [](size_t v) { return (v + 63) & ~size_t(63); };  // 256-byte aligned regions
  const size_t nA = up((size_t)B * D), nY = up((size_t)B * s * 3 * m), nW = up((size_t)B * s * (9 * m + 1));
  const size_t need = 2 * nA + nY + nW;
  if (need > kNoallocScratchFloats)
    return fail(BODEX_ERR_INVALID,
                "bodex_step_noalloc: B * (2 (6+n) + s (12 m + 1)) floats exceed its fixed 4 MiB scratch "
                "(1048576 floats); use bodex_state_create + bodex_step for larger batches");
  if (n_steps == 0 || B == 0) return BODEX_OK;
  float* base = nullptr;
  if (int r = noalloc_scratch((int)m, &base)) return r;
  cudaStream_t st = as_stream(stream);
  // the array keeps the previous call's contents: Adam moments and warm
  // starts must start at zero
  BODEX_CUDA(cudaMemsetAsync(base, 0, need * sizeof(float), st));
  A.n_steps = n_steps;
  A.t0 = 0;
  A.x_state = x;
  A.am = base;
  A.av = base + nA;
  A.qy = base + 2 * nA;
  A.qw = base + 2 * nA + nY;
  A.E = E_last;
  A.status = status;
  return dispatch_fused((int)m, MODE_STEP, A, st);
}

}  // extern "C"
