// adjoint.cu -- discrete adjoint of the lattice Boltzmann time step for
// inflow-parameter assimilation (arXiv:2508.18202 Sec. 1 and 2.4 motivate the
// assimilation; the paper itself does not differentiate the solver).
//
// Forward model of one time step n -> n + 1 (BGK, Sec. 2.2, Eq.
// deterministicLBE):
//   f*(x) = C(f^n(x))                       local collision
//   f^{n+1} = A f* + b(theta, n + 1)        streaming and link rules, linear in
//                                           f*, plus the moving-wall term
//                                           b_i = 6 w_i (c_i . u_in(z)) r(n+1)
//                                           on inflow links.
// With J = sum_p |u(x_p, T) - u*_p|^2 and lambda^n = dJ/df^n:
//   lambda^T   = dJ/df^T (probe cells only)
//   lambda*^n  = A^T lambda^{n+1}            (gather over the deliveries of
//                                            each post-collision population)
//   lambda^n   = (dC/df(f^n))^T lambda*^n
//   dJ/dtheta  = sum_n sum_inflow links lambda^{n+1}_i(x) db_i/dtheta.
// The forward states f^n of a segment are recomputed from checkpoints taken
// every L steps (about sqrt(T) checkpoints of about sqrt(T) steps each).
//
// All arrays are FP32 populations g = f - w in natural layout [19][pitch];
// the gradient and the loss accumulate in FP64.
#include <cuda_runtime.h>
#include <stdint.h>

#include "lbm_device.cuh"
#include "sclbm_internal.h"

namespace sclbm {
namespace {

// Blocks of 128 cells: a state stays in L2 and a launch is a few waves, so
// small blocks keep the last wave short.  The leading blocks take the listed
// cells: the outlet's stand one to a row, so a quarter of the bulk warps would
// run their long path for one lane; at the launch's end their chain of
// dependent loads would be its tail (17.3 ms a gradient).  Only warps with a moving-wall or
// specular link carry its terms.  One gradient of 300 steps on 128 x 64 x 48
// (forward, recompute and reverse sweep): 15.3 -> 11.3 ms; of 200 on 61 x 33 x 21: 3.80 -> 3.07 ms.
constexpr int kAdjThreads = 128;
constexpr int kAdjListed = 32;  // listed cells of a block: scattered accesses, 32 sectors a load, spread over the SMs

// The block's cell: a bulk cell (link word in lw, kLinkSolid where there is
// none to do), or a listed one with its record in L.
__device__ __forceinline__ bool adj_cell(const DevDomain& D, int* c, LinkWord* lw, ListedRef* L) {
  const unsigned lead = (unsigned)((D.nb + kAdjListed - 1) / kAdjListed);
  if (blockIdx.x >= lead) {
    *c = (int)((blockIdx.x - lead) * kAdjThreads + threadIdx.x);
    *lw = *c < (int)D.ncell ? __ldg(D.link + *c) : kLinkSolid;
    if (*lw & kLinkSlow) *lw = kLinkSolid;
    return false;
  }
  const int li = (int)(blockIdx.x * kAdjListed + threadIdx.x);
  const bool some = threadIdx.x < kAdjListed && li < (int)D.nb;
  *c = some ? __ldg(D.bcell + li) : 0;
  *lw = some ? 0 : kLinkSolid;
  *L = listed_ref(D, some ? li : 0);
  return true;
}

// One FP32 time step of one node, two arrays, push form.
__global__ void __launch_bounds__(kAdjThreads) adj_forward_kernel(const __grid_constant__ StepParams P, AdjArgs A,
                                                                  const float* src, float* dst, float r1) {
  const DevDomain& D = P.dom[A.domain];
  const int pc = (int)D.pitch, sy = D.nx, sz = D.nx * D.ny;
  int c;
  LinkWord lw;
  ListedRef L;
  const bool listed = adj_cell(D, &c, &lw, &L);
  const bool general = __any_sync(0xffffffffu, !(lw & kLinkSolid) && (lw & kLinkGeneral));
  if (lw & kLinkSolid) return;
  float g[kQ];
#pragma unroll
  for (int i = 0; i < kQ; ++i) g[i] = src[i * pc + c];
  collide_p<float, true>(P, g);
  Node<float> N;
  N.g = dst;
  N.bout = nullptr;
  N.uinf = A.uin;
  N.uind = nullptr;
  const Wind<float> w1{1.f, 0.f, r1};  // steady inflow: the ramp alone
  float ux = 0.f, uy = 0.f, uz = 0.f;
  if (listed) {
    if (L.word(kWordPushMove)) inflow_velocity<float>(N, L.word(kWordZ), w1, ux, uy, uz);
    listed_push<float>(L, dst, ux, uy, uz, r1, g);
  } else if (general) {
    wall_velocity<float>(N, lw, c / sz, w1, ux, uy, uz);
    mask_push<float, true>(dst + c, lw, pc, sy, sz, ux, uy, uz, r1, g);
  } else {
    mask_push<float, false>(dst + c, lw, pc, sy, sz, 0.f, 0.f, 0.f, 0.f, g);
  }
}

// Loss at the probes and the adjoint seed lambda^T = dJ/df^T
// (dJ/df_m = sum_a 2 (u_a - u*_a) (c_ma - u_a) / rho).
__global__ void adj_loss_kernel(const __grid_constant__ StepParams P, AdjArgs A, const float* f, float* lam) {
  const DevDomain& D = P.dom[A.domain];
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= A.n_probes) return;
  const int* q = A.probes + 3 * p;
  const long long c = q[0] + (long long)D.nx * (q[1] + (long long)D.ny * q[2]);
  double rho = 0.0, j[3] = {0.0, 0.0, 0.0};
  for (int i = 0; i < kQ; ++i) {
    const double fi = (double)f[(long long)i * D.pitch + c] + c_lat.wd[i];
    rho += fi;
    j[0] += c_lat.cx[i] * fi;
    j[1] += c_lat.cy[i] * fi;
    j[2] += c_lat.cz[i] * fi;
  }
  const double u[3] = {j[0] / rho, j[1] / rho, j[2] / rho};
  double e[3], loss = 0.0;
  for (int a = 0; a < 3; ++a) {
    e[a] = u[a] - A.target[3 * p + a];
    loss += e[a] * e[a];
    A.u_probe[3 * p + a] = u[a];
  }
  atomicAdd(A.accum, loss);
  for (int m = 0; m < kQ; ++m) {
    const double cm[3] = {(double)c_lat.cx[m], (double)c_lat.cy[m], (double)c_lat.cz[m]};
    double v = 0.0;
    for (int a = 0; a < 3; ++a) v += 2.0 * e[a] * (cm[a] - u[a]) / rho;
    lam[(long long)m * D.pitch + c] = (float)v;
  }
}

// One reverse step: lambda^n from lambda^{n+1} and the forward state f^n;
// accumulates the inflow-parameter gradient of level n + 1 (ramp r1).
__global__ void __launch_bounds__(kAdjThreads) adj_step_kernel(const __grid_constant__ StepParams P, AdjArgs A,
                                                               const float* f, const float* lam_next, float* lam,
                                                               float r1) {
  const DevDomain& D = P.dom[A.domain];
  const int pc = (int)D.pitch, sy = D.nx, sz = D.nx * D.ny;
  int c;
  LinkWord lw;
  ListedRef L;
  const bool listed = adj_cell(D, &c, &lw, &L);
  const bool some = !(lw & kLinkSolid);
  const bool moving = __any_sync(0xffffffffu, some && (lw & kLinkVel));
  const bool specular = __any_sync(0xffffffffu, some && (lw & kLinkSpec));
  float g0 = 0.0f, g1 = 0.0f;  // the cell's share of the gradient
  if (some) {
    float ls[kQ];
    // lambda*_k(x) = the sum of lambda^{n+1} over the slots the forward
    // step delivers f*_k(x) to (the transpose of the push rules), and the
    // moving-wall terms' share of dJ/dtheta: sum over the slots that receive
    // a term 6 w_i (c_i . u_in(z)) r(n + 1) of lambda^{n+1} there times the
    // term's derivative (summed per cell in FP32, over cells in FP64)
    if (!listed) {
      // each f*_k goes to the one slot the forward push writes (stream,
      // bounce-back, moving wall, specular lid)
      const LinkMasks m(lw);
#pragma unroll
      for (int k = 0; k < kQ; ++k) {
        const int stream = k * pc + (CX(k) + CY(k) * sy + CZ(k) * sz);
        int off = stream + LinkMasks::bit(m.wall, OPP(k)) * (OPP(k) * pc - stream);
        if (SPECZ(k) && specular)
          off += LinkMasks::bit(m.spec, OPP(k)) * (REFL(k, 2) * pc + (CX(k) + CY(k) * sy) - OPP(k) * pc);
        ls[k] = lam_next[c + (k == 0 ? 0 : off)];
      }
      if (moving) {
        const int z = c / sz;
        const float4 du0 = A.du[z], du1 = A.du[D.nz + z];
#pragma unroll
        for (int k = 1; k < kQ; ++k)
          if (LinkMasks::bit(m.move, OPP(k))) {  // lands in the own slot i = opp(k) with the term of link i
            const int i = OPP(k);
            const float pre = 6.0f * W<float>(i) * r1 * ls[k];
            g0 += pre * cdot<float>(i, du0.x, du0.y, du0.z);
            g1 += pre * cdot<float>(i, du1.x, du1.y, du1.z);
          }
      }
    } else {
      // listed cell: the deliveries of its compiled record; an outlet copy
      // stored to a slot the cell's own primary delivery also wrote
      // replaces it (listed_push writes the copies last)
      const int z = L.word(kWordZ);
      const float4 du0 = A.du[z], du1 = A.du[D.nz + z];
      constexpr int kCopies = kOutletPops * kOutletCopies;
      int32_t ex[kCopies];
#pragma unroll
      for (int e = 0; e < kCopies; ++e) ex[e] = L.word(kWordExtra + e);
      const uint32_t mm = (uint32_t)L.word(kWordPushMove);
#pragma unroll
      for (int k = 0; k < kQ; ++k) {
        const int d = L.word(kWordDst + k);
        bool replaced = false;
#pragma unroll
        for (int e = 0; e < kCopies; ++e) replaced |= ex[e] == d;
        const float v = (d >= 0 && !replaced) ? lam_next[d] : 0.0f;
        ls[k] = v;
        if ((mm >> k) & 1u) {
          const int i = OPP(k);
          const float pre = 6.0f * W<float>(i) * r1 * v;
          g0 += pre * cdot<float>(i, du0.x, du0.y, du0.z);
          g1 += pre * cdot<float>(i, du1.x, du1.y, du1.z);
        }
      }
      constexpr int kPops[kOutletPops] = {2, 8, 10, 12, 14};
#pragma unroll
      for (int e = 0; e < kOutletPops; ++e)
#pragma unroll
        for (int m = 0; m < kOutletCopies; ++m) {
          const int d = ex[e * kOutletCopies + m];
          if (d >= 0) ls[kPops[e]] += lam_next[d];
        }
    }
    // forward state of this level (the shifted populations: rho = 1 + sum g)
    float g[kQ];
#pragma unroll
    for (int i = 0; i < kQ; ++i) g[i] = f[i * pc + c];
    float m0, jx, jy, jz;
    flow_sums<float>(g, m0, jx, jy, jz);
    const float inv = recip(1.0f + m0);
    const float ux = jx * inv, uy = jy * inv, uz = jz * inv;
    const float usq = ux * ux + uy * uy + uz * uz;
    const float om = P.omega0;
    // alpha = sum_i ls_i df^eq_i/drho, beta_a = sum_i ls_i df^eq_i/dj_a: the
    // opposite pair (i, i + 1) shares (c_i . u)^2, so with its weighted sum s
    // and difference d of ls
    //   alpha += s (1 - 4.5 cu^2 + 1.5 u^2),  beta += c_i (3 d + 9 cu s) - 3 u s
    const float base = 1.0f + 1.5f * usq;
    float sw = W<float>(0) * ls[0], al = sw * base, bx = 0.0f, by = 0.0f, bz = 0.0f;
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
      const float s = W<float>(i) * (ls[i] + ls[i + 1]), d = W<float>(i) * (ls[i] - ls[i + 1]);
      const float cu = cdot<float>(i, ux, uy, uz);
      al += s * (base - 4.5f * cu * cu);
      sw += s;
      const float t = 3.0f * d + 9.0f * cu * s;
      if (CX(i)) bx += CX(i) > 0 ? t : -t;
      if (CY(i)) by += CY(i) > 0 ? t : -t;
      if (CZ(i)) bz += CZ(i) > 0 ? t : -t;
    }
    sw *= 3.0f;
    bx = om * (bx - sw * ux), by = om * (by - sw * uy), bz = om * (bz - sw * uz), al *= om;
    const float keep = 1.0f - om;
    lam[c] = keep * ls[0] + al;
#pragma unroll
    for (int m = 1; m < kQ; m += 2) {
      const float cb = cdot<float>(m, bx, by, bz);
      lam[m * pc + c] = keep * ls[m] + (al + cb);
      lam[(m + 1) * pc + c] = keep * ls[m + 1] + (al - cb);
    }
  }
  // warps without a moving-wall contribution skip the FP64 reduction
  if (!__any_sync(0xffffffffu, g0 != 0.0f || g1 != 0.0f)) return;
  double gr0 = (double)g0, gr1 = (double)g1;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gr0 += __shfl_xor_sync(0xffffffffu, gr0, o);
    gr1 += __shfl_xor_sync(0xffffffffu, gr1, o);
  }
  if ((threadIdx.x & 31) == 0 && (gr0 != 0.0 || gr1 != 0.0)) {
    atomicAdd(A.accum + 1, gr0);
    atomicAdd(A.accum + 2, gr1);
  }
}

__global__ void fill_zero_kernel(float* p, long long n) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x)
    p[k] = 0.0f;
}

// Blocks of a sweep's launch: the listed cells', then the bulk ones'.
unsigned adj_blocks(const DevDomain& D) {
  return (unsigned)((D.ncell + kAdjThreads - 1) / kAdjThreads + (D.nb + kAdjListed - 1) / kAdjListed);
}

}  // namespace

int launch_adj_forward(const StepParams& P, const AdjArgs& A, const float* src, float* dst, float r1,
                       void* stream) {
  const DevDomain& D = P.dom[A.domain];
  adj_forward_kernel<<<adj_blocks(D), kAdjThreads, 0, (cudaStream_t)stream>>>(P, A, src, dst, r1);
  return (int)cudaGetLastError();
}

int launch_adj_loss(const StepParams& P, const AdjArgs& A, const float* f, float* lam, void* stream) {
  adj_loss_kernel<<<(A.n_probes + 63) / 64, 64, 0, (cudaStream_t)stream>>>(P, A, f, lam);
  return (int)cudaGetLastError();
}

int launch_adj_step(const StepParams& P, const AdjArgs& A, const float* f, const float* lam_next, float* lam,
                    float r1, void* stream) {
  const DevDomain& D = P.dom[A.domain];
  adj_step_kernel<<<adj_blocks(D), kAdjThreads, 0, (cudaStream_t)stream>>>(P, A, f, lam_next, lam, r1);
  return (int)cudaGetLastError();
}

int launch_fill_zero(float* p, long long n, void* stream) {
  fill_zero_kernel<<<(unsigned)((n + 255) / 256 < 152 * 32 ? (n + 255) / 256 : 152 * 32), 256, 0,
                     (cudaStream_t)stream>>>(p, n);
  return (int)cudaGetLastError();
}

}  // namespace sclbm
