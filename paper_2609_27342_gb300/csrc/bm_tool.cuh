// Rigid tool step of a substep: wrench history, interval-averaged motion and
// the frame of the next substep, computed beside the particle kernels.
#pragma once
#include <math.h>
#include <stddef.h>

#include "bm_device.cuh"
#include "bm_internal.cuh"

namespace {

__device__ __forceinline__ const DevSeg *seg_at(const DevScene &sc, long long step) {
  long long acc = 0;
  for (int i = 0; i < sc.nseg; ++i) {
    acc += sc.seg[i].n_steps;
    if (step < acc) return &sc.seg[i];
  }
  return nullptr;
}

// The tool step by one warp on the shared-memory copy of the scene record:
// wrench history, interval-averaged rigid tool step, and the frame of the
// next substep.  Float64 operations are slow here (about 2 lanes per clock
// and SM), so each component of a vector or matrix is its own lane's, in the
// expression of the one-thread code: a serial thread spent most of the
// kernel's 16.5 us (a 16,000-particle scene) on some 400 of them; 9.2 us now.
__device__ __forceinline__ double matmul_at(const double A[9], const double B[9], int k) {
  const int i = k / 3, j = k % 3;
  return A[3 * i] * B[j] + A[3 * i + 1] * B[3 + j] + A[3 * i + 2] * B[6 + j];
}

struct ToolTmp {
  double Fa[3], Ta[3], th[3], A[9], Iw[9], K[9], Rinc[9];
};

// Frame of substep sc.step, by one warp: prescribed twist, cut, D reset, blade axes
// (prepare_substep in bm_kernels.cu restates it).
__device__ __forceinline__ void prepare_substep_warp(DevScene &sc, ToolTmp &T, int lane) {
  if (!sc.has_blade) {
    if (lane == 0) {
      sc.cut = -1;
      sc.reset_D = 0;
    }
    return;
  }
  const DevSeg *sg = seg_at(sc, sc.step);
  const int cut = sg ? sg->cut_id : -1;
  const bool dynamic = sc.mass > 0.0;
  const int reset = (cut >= 0 && cut != sc.cur_cut) ? 1 : 0;
  if (!dynamic && sg && lane < 3) {
    sc.vB[lane] = sg->v[lane];
    sc.wB[lane] = sg->w[lane];
  }
  if (lane == 0) {
    sc.cut = cut;
    sc.reset_D = reset;
  }
  // edge point and blade axes: lane 3 q + i holds component i of vector q
  if (lane < 12) {
    const int q = lane / 3, i = lane % 3;
    const double *v = q == 0 ? sc.edgeT : q == 1 ? sc.nT : q == 2 ? sc.eT : sc.dT;
    const double y = __dadd_rn(__dadd_rn(__dmul_rn(sc.R[3 * i], v[0]), __dmul_rn(sc.R[3 * i + 1], v[1])),
                               __dmul_rn(sc.R[3 * i + 2], v[2]));
    double *o = q == 0 ? sc.dxe : q == 1 ? sc.dn : q == 2 ? sc.de : sc.dd;
    o[i] = q == 0 ? __dadd_rn(sc.xB[i], y) : y;
  }
  __syncwarp();
  if (lane < 3) {
    const int i = lane, j = (lane + 1) % 3, k = (lane + 2) % 3;
    const double rj = __dsub_rn(sc.dxe[j], sc.xB[j]), rk = __dsub_rn(sc.dxe[k], sc.xB[k]);
    const double wr = __dsub_rn(__dmul_rn(sc.wB[j], rk), __dmul_rn(sc.wB[k], rj));
    sc.dve[i] = __dadd_rn(sc.vB[i], wr);
  }
  if (dynamic && lane < 9) T.A[lane] = matmul_at(sc.R, sc.Ib_inv, lane);
  __syncwarp();
  if (reset) {  // a new cut begins: keep its plane for the cut faces
    if (lane < 3) sc.cutpl[cut][lane] = sc.dn[lane];
    if (lane == 3) {
      sc.cutpl[cut][3] = __dadd_rn(__dadd_rn(__dmul_rn(sc.dn[0], sc.dxe[0]), __dmul_rn(sc.dn[1], sc.dxe[1])),
                                   __dmul_rn(sc.dn[2], sc.dxe[2]));
      sc.cutpl_set |= 1u << cut;
    }
  }
  if (lane < 3) {
    const int i = lane;
    sc.fxe[i] = (float)sc.dxe[i];
    sc.fn[i] = (float)sc.dn[i];
    sc.fe[i] = (float)sc.de[i];
    sc.fd[i] = (float)sc.dd[i];
    sc.fve[i] = (float)sc.dve[i];
    sc.fc[i] = (float)(sc.dxe[i] - sc.half_height * sc.dd[i]);
    sc.fxB[i] = (float)sc.xB[i];
    sc.fvB[i] = (float)sc.vB[i];
    sc.fwB[i] = (float)sc.wB[i];
  }
  if (lane == 3) {
    sc.fhext[0] = (float)sc.half_thick;
    sc.fhext[1] = (float)sc.half_len;
    sc.fhext[2] = (float)sc.half_height;
    sc.fL = (float)sc.L_d;
    sc.fmu_s = (float)sc.mu_s;
    sc.fmu_d = (float)sc.mu_d;
    sc.finv_mass = dynamic ? (float)(1.0 / sc.mass) : 0.f;
  }
  if (lane < 9) {  // world inverse inertia R Ib^-1 R^T
    const int i = lane / 3, j = lane % 3;
    sc.fIinv[lane] =
        dynamic ? (float)(T.A[3 * i] * sc.R[3 * j] + T.A[3 * i + 1] * sc.R[3 * j + 1] + T.A[3 * i + 2] * sc.R[3 * j + 2])
                : 0.f;
  }
}

__device__ __forceinline__ void tool_step(const World &w, DevScene &sc, ToolTmp &T, const double W[6], int lane) {
  if (sc.has_blade) {
    const long long st = sc.step;
    if (st < sc.hist_cap && lane < 6) w.whist[(size_t)(sc.hist_begin + st) * 6 + lane] = W[lane];
    const int cnt = sc.acc_cnt + 1;
    if (lane < 3) {
      sc.accF[lane] += W[lane];
      sc.accT[lane] += W[3 + lane];
    }
    __syncwarp();
    if (cnt >= sc.rigid_interval) {
      const double H = sc.dt_d * cnt;
      if (lane < 3) {
        T.Fa[lane] = sc.accF[lane] / cnt;
        T.Ta[lane] = sc.accT[lane] / cnt;
      }
      if (sc.mass > 0.0) {
        const DevSeg *tg = seg_at(sc, st);
        if (lane < 9) T.A[lane] = matmul_at(sc.R, sc.Ib_inv, lane);
        __syncwarp();
        if (lane < 9) {
          const int i = lane / 3, j = lane % 3;
          T.Iw[lane] = T.A[3 * i] * sc.R[3 * j] + T.A[3 * i + 1] * sc.R[3 * j + 1] + T.A[3 * i + 2] * sc.R[3 * j + 2];
        }
        __syncwarp();
        if (lane < 3) {
          const int k = lane;
          const double dw = T.Iw[3 * k] * T.Ta[0] + T.Iw[3 * k + 1] * T.Ta[1] + T.Iw[3 * k + 2] * T.Ta[2];
          const double vt = tg ? tg->v[k] : 0.0, wt = tg ? tg->w[k] : 0.0;
          sc.vB[k] += H * (sc.kv * (vt - sc.vB[k]) + T.Fa[k] / sc.mass);
          sc.wB[k] += H * (sc.kv * (wt - sc.wB[k]) + dw);
        }
      }
      __syncwarp();
      if (lane < 3) T.th[lane] = H * sc.wB[lane];
      __syncwarp();
      // rotation increment exp(th): I + sin a K + (1 - cos a) K^2
      const double th0 = T.th[0], th1 = T.th[1], th2 = T.th[2];
      const double a = sqrt(th0 * th0 + th1 * th1 + th2 * th2);
      if (a > 0) {
        const double k0 = th0 / a, k1 = th1 / a, k2 = th2 / a;
        if (lane == 0) {
          T.K[0] = T.K[4] = T.K[8] = 0;
          T.K[1] = -k2;
          T.K[2] = k1;
          T.K[3] = k2;
          T.K[5] = -k0;
          T.K[6] = -k1;
          T.K[7] = k0;
        }
        __syncwarp();
        if (lane < 9) {
          const double sa = sin(a), ca = 1.0 - cos(a);
          double r = (lane % 4 == 0) ? 1.0 : 0.0;
          r += sa * T.K[lane] + ca * matmul_at(T.K, T.K, lane);
          T.Rinc[lane] = r;
        }
      } else if (lane < 9) {
        T.Rinc[lane] = (lane % 4 == 0) ? 1.0 : 0.0;
      }
      __syncwarp();
      const double Rn = lane < 9 ? matmul_at(T.Rinc, sc.R, lane) : 0.0;
      __syncwarp();
      if (lane < 9) sc.R[lane] = Rn;
      if (lane < 3) {
        sc.xB[lane] += H * sc.vB[lane];
        sc.lastW[lane] = T.Fa[lane];
        sc.lastW[3 + lane] = T.Ta[lane];
        sc.accF[lane] = sc.accT[lane] = 0.0;
      }
    }
    __syncwarp();
    if (lane == 0) {
      sc.acc_cnt = cnt >= sc.rigid_interval ? 0 : cnt;
      if (sc.cut >= 0) sc.cur_cut = sc.cut;
    }
  }
  if (lane == 0) {
    sc.step++;
    if (sc.stop_at >= 0 && sc.step >= sc.stop_at) sc.frozen = 1;
  }
  __syncwarp();
  prepare_substep_warp(sc, T, lane);
}

// The tool step of a scene, by one CTA of another kernel: it needs the wrench
// partials, which P2G has left, and nothing later in the substep; k_fupd still
// reads this substep's frame, so the result goes to the scene's record in
// scenes_next and commit_tool takes it over when the particles are done.  As a
// kernel of its own after k_fupd it was 9.2 us of a 16,000-particle scene's 98 us
// substep and 16 of the 256-scene batch's 1,460.
struct ToolS {
  DevScene sc;
  ToolTmp T;
  double part[6][8], W[6];
};

// the part of the record that the tool step writes, in words
constexpr int kToolWord0 = (int)(offsetof(DevScene, xB) / sizeof(int));
constexpr int kToolWords = (int)(offsetof(DevScene, err) / sizeof(int)) - kToolWord0;

__device__ __forceinline__ void next_tool(const World &w, int sid, ToolS &S) {
  DevScene &g = w.scenes[sid];
  // the labels of the last substep are in the slot table; k_fupd sets this anew
  if (threadIdx.x == 0) g.label_pending = 0;
  if (g.frozen) return;  // a scene that has taken its substeps: nothing moves
  // the scene record into shared memory (coalesced), so that the tool step
  // and frame below read and write it at shared-memory latency
  static_assert(sizeof(DevScene) % sizeof(double) == 0, "the scene record copies as doubles");
  for (int i = threadIdx.x; i < (int)(sizeof(DevScene) / sizeof(double)); i += blockDim.x)
    reinterpret_cast<double *>(&S.sc)[i] = reinterpret_cast<const double *>(&g)[i];
  // this substep's per-brick wrench partials: 256 strides over the bricks, a
  // fixed shuffle tree over each 32 of them, then the eight in order (the
  // same sums for every node tile size, the CTA's thread count)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int v = wid; v < 8; v += nw) {
    double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (g.has_blade) {
      const double2 *q = reinterpret_cast<const double2 *>(w.wpart) + (size_t)g.brick_begin * 3;
      const int nb = g.n_brick;
      int j = 32 * v + lane;
      for (; j + 256 < nb; j += 512) {  // two strides' loads in flight
        double2 a[3], b[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          a[k] = q[(size_t)j * 3 + k];
          b[k] = q[(size_t)(j + 256) * 3 + k];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          acc[2 * k] = acc[2 * k] + a[k].x + b[k].x;
          acc[2 * k + 1] = acc[2 * k + 1] + a[k].y + b[k].y;
        }
      }
      if (j < nb)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double2 a = q[(size_t)j * 3 + k];
          acc[2 * k] += a.x;
          acc[2 * k + 1] += a.y;
        }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      double y = acc[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) y += __shfl_down_sync(FULL, y, o);
      if (lane == 0) S.part[k][v] = y;
    }
  }
  __syncthreads();
  if (wid == 0) {
    if (lane < 6) {
      double t = 0.0;
      for (int i = 0; i < 8; ++i) t += S.part[lane][i];
      S.W[lane] = t;
    }
    __syncwarp();
    tool_step(w, S.sc, S.T, S.W, lane);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kToolWords; i += blockDim.x)
    reinterpret_cast<int *>(w.scenes_next + sid)[kToolWord0 + i] = reinterpret_cast<const int *>(&S.sc)[kToolWord0 + i];
}

// take over the tool step that next_tool has left (one CTA; no other CTA of
// the launch may read the record's tool block, step or frozen)
__device__ __forceinline__ void commit_tool(const World &w, int sid) {
  const bool frozen = w.scenes[sid].frozen != 0;
  __syncthreads();
  if (frozen) return;
  for (int i = threadIdx.x; i < kToolWords; i += blockDim.x)
    reinterpret_cast<int *>(w.scenes + sid)[kToolWord0 + i] =
        reinterpret_cast<const int *>(w.scenes_next + sid)[kToolWord0 + i];
}

// Leading CTAs of G2P that take the scenes' tool steps; 0: k_musl_node does.
// A tool step takes about as long as G2P in a small scene and longer than its
// k_musl_node (6 us); a 477,000-particle scene's k_musl_node is 18 us with it, 14
// without.  For the 256-scene batch the two places measure the same (1,447 and
// 1,449 us a substep), and there k_musl_node's CTAs hold less of an SM.
constexpr int G2P_TOOLS = 152;
inline int g2p_tools(const LaunchSet &ls) { return ls.n_scenes <= G2P_TOOLS ? ls.n_scenes : 0; }

}  // namespace
