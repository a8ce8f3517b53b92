// sm_103a kernels of one TLMPM cutting substep (arXiv 2609.27342, Sec. III).
//
// Particles are sorted brick-major (4x4x4 reference base cells per brick) and
// every particle-side kernel runs one CTA per brick:
//   k_p2g_brick  contact (Eq. 12, 14-16), cutting progress (Eq. 5), side
//                labels for the next substep (Eq. 3, 4, 6), neo-Hookean
//                stress, and the brick's share of the per-code P2G sums
//                (Eq. 2) in its 6x6x6 node tile, in shared memory
//   k_p2g_node   per node: the <= 8 overlapping brick tiles summed in brick
//                order, coupling (Eq. 8), grid update (Eq. 9)
//   k_g2p_musl   G2P (Eq. 17), x update, the brick's share of the MUSL
//                re-scatter
//   k_musl_node  per node: MUSL sums, coupling, v*
//   k_fupd       F update, commit of the new side labels
//   k_recount, k_slot_*, k_brick_tiles, k_count_tiles
//                compact logical-grid slots (Sec. III-G) after label changes
// The tool step (bm_tool.cuh: wrench, rigid motion, next frame) runs as extra
// CTAs of G2P or k_musl_node.  The brick kernels here take any scene;
// bm_lattice.cu has their forms for lattice bodies.
//   k_pair_*     material-material contact (Eq. 10-13): the rebuild test,
//                spatial hash and candidate lists, and the pair impulses,
//                ahead of P2G
// No atomics touch floating-point sums: every sum is taken in a fixed order,
// so a scene gives bit-identical results alone or inside any batch.
//
// All arithmetic is float32 except the tool state and the near-threshold
// fallback of the side-label predicate, which is float64 with explicitly
// rounded operations so it reproduces a plain double-precision evaluation.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include "bm_device.cuh"
#include "bm_internal.cuh"
#include "bm_tool.cuh"


namespace {

// --------------------------------------------------------------------------
// k_p2g_brick: the brick's share of P2G (Eq. 2) into its node tile, per
// logical grid, from the particles' A, J, v staged in shared memory.
// --------------------------------------------------------------------------
// G groups of BT threads: G = 1, or an even number
template <int PPC, int G>
struct K2S {
  static constexpr int NP = (G + 1) / 2;  // passes side by side, two groups each
  BrickTile T;
  float part[18][PPC * BR3];   // the brick's particles (fx, v, A, J), [particle-in-cell][cell]
  union {
    float sz[NP][7][3][TZ];    // the passes' (node, z-offset) sums
    float wrc[6][G > 1 ? PPC * BR3 : 1];  // before: each particle's reaction wrench (G > 1)
  };
  unsigned long long cmask[BR3];  // several codes: which of the brick's codes each cell's particles carry
  float red[6][BT / 32];       // wrench partials of the warps
  int cs[BR3 + 1];
  uint8_t pid[PPC * BR3];      // several codes: code index of each particle
};

// Which of the brick's codes each cell's particles carry (threads of z-offset
// 0), from the [particle-in-cell][cell] staging of the code indices.
__device__ __forceinline__ void cell_codes(const uint8_t *pid, const int *cs, unsigned long long *cmask) {
  const int c = threadIdx.x;
  if (c >= BR3) return;
  const int n = cs[c + 1] - cs[c];
  unsigned long long m = 0;
  for (int j = 0; j < n; ++j) {
    const int b = pid[pic(j, c)];
    if (b < BM_BRICK_CODES) m |= 1ull << b;
  }
  cmask[c] = m;
}

// The brick's particles into shared memory, transposed to
// [particle-in-cell][cell] so that the (cell, z-offset) threads read
// consecutive words: the fractional offset, v, and the P2G inputs A and J
// that pre_particle computes from x, v, F, D, u_t and the codes.  The caller
// provides the barrier that publishes it.
template <int PPC, int G, bool INELASTIC>
__device__ void stage_particles(const World &w, const DevScene &sc, const int4 &bt, bool coded, K2S<PPC, G> &S,
                                float wr[6], bool &clamped, bool &anyc) {
  const PPool &P = w.P;
  // each thread fetches its next particle's flag one iteration ahead, so the
  // loads of D and u_t it gates do not wait on it
  uint8_t tf_next = (int)threadIdx.x < bt.w ? P.tflag[bt.z + threadIdx.x] : 0;
  for (int i = threadIdx.x; i < bt.w; i += blockDim.x) {
    const int p = bt.z + i;
    const uint8_t tf = tf_next;
    if (i + (int)blockDim.x < bt.w) tf_next = P.tflag[p + blockDim.x];
    const float x[3] = {P.x[0][p], P.x[1][p], P.x[2][p]};
    const float v[3] = {P.v[0][p], P.v[1][p], P.v[2][p]};
    const int id = P.cid[p];
    const uint2 code = id < BM_BRICK_CODES ? S.T.bcode[id] : make_uint2(0u, 0u);
    const float f0 = P.fx[0][p], f1 = P.fx[1][p], f2 = P.fx[2][p];
    float A[9], J[3];
    if (G == 1) {
      pre_particle<INELASTIC>(sc, P, p, tf, x, v, code.x, code.y, A, J, wr, clamped, anyc);
    } else {
      float wp[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      pre_particle<INELASTIC>(sc, P, p, tf, x, v, code.x, code.y, A, J, wp, clamped, anyc);
      if (sc.has_blade)
#pragma unroll
        for (int k = 0; k < 6; ++k) S.wrc[k][i] = wp[k];
    }
    const int c = cell_of(S.cs, i);
    const int si = pic(i - S.cs[c], c);
    S.part[0][si] = f0;
    S.part[1][si] = f1;
    S.part[2][si] = f2;
    S.part[3][si] = v[0];
    S.part[4][si] = v[1];
    S.part[5][si] = v[2];
#pragma unroll
    for (int k = 0; k < 9; ++k) S.part[6 + k][si] = A[k];
    S.part[15][si] = J[0];
    S.part[16][si] = J[1];
    S.part[17][si] = J[2];
    if (coded) S.pid[si] = (uint8_t)id;
  }
}

template <int PPC, int MB, bool INELASTIC, int G>
__global__ void __launch_bounds__(BT * G, MB) k_p2g_brick(World w, LaunchSet ls) {
  chain_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  K2S<PPC, G> &S = *reinterpret_cast<K2S<PPC, G> *>(smraw);
  const int4 bt = ls.btiles[blockIdx.x];  // scene, pool brick, first particle, count
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (sc.frozen || sc.lattice) return;
  constexpr int NT = BT * G, NP = K2S<PPC, G>::NP;
  const int tid = threadIdx.x, grp = tid / BT;
  const int lb = bt.y - sc.brick_begin;
  const BrickInfo B(w, bt, PPC * BR3);
  const bool several = B.nbc > 1;
  const int *csg = w.N.cell_start + sc.cell_begin + lb * BR3;
  for (int i = tid; i <= BR3; i += NT) S.cs[i] = csg[i] - bt.z;
  brick_tile(w, bt.y, B.nbc, S.T, NT);
  __syncthreads();
  float wr[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  bool clamped = false, anyc = false;
  stage_particles<PPC, G, INELASTIC>(w, sc, bt, several, S, wr, clamped, anyc);
  if (clamped) atomicOr(&scm.err, BM_ERRBIT_INVERTED);
  if (!B.uniform) brick_slots<true>(w, S.T, B.nbc, B.pbase, NT);
  if (sc.has_blade) {
    if (G > 1) {
      __syncthreads();
      stride_wrench(S.wrc[0], PPC * BR3, bt.w, wr);
    }
    brick_wrench(w, bt.y, wr, anyc, S.red);
  }
  __syncthreads();
  if (several) {
    cell_codes(S.pid, S.cs, S.cmask);
    __syncthreads();
  }

  // ---- one pass per code of the brick ----
  // Each thread sums, for its cell and one z-offset, m N, m v N and
  // A grad N + N J over the cell's particles with the pass's code; the warp
  // reduces the sums along x and y (xy_reduce), the z stage collects the
  // layers, and each tile node adds its <= 3 layer sums and writes the slot
  // of the pass's code.  Every float sum has one owner: no atomics, and each
  // partial-sum entry is written exactly once.
  const int c = tid % BR3, oz = tid % BT / BR3;
  const int cx = c & 3, cy = (c >> 2) & 3, cz = c >> 4;
  const int n_c = S.cs[c + 1] - S.cs[c];
  const unsigned long long codes = several ? S.cmask[c] : 0ull;
  const bool filt = (codes & (codes - 1)) != 0;  // the cell's particles carry several codes
  for (int b0 = 0; b0 < B.npass; b0 += NP) {
    // G > 1: an even group takes the momentum sums of its pass, the next the force sums
    const int b = b0 + grp / 2;
    const bool has = n_c > 0 && b < B.npass && (!several || ((codes >> b) & 1u));
    float(*sz)[3][TZ] = S.sz[grp / 2];
    // two walks over the cell's particles, each reducing its own values, so
    // that fewer sums are live at once: (m N, m v N), then A grad N + N J
    if (b < B.npass && (G == 1 || grp % 2 == 0)) {
      float a[3][3][4];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
          for (int f = 0; f < 4; ++f) a[i][j][f] = 0.f;
      if (has) {
        for (int j = 0; j < n_c; ++j) {
          const int si = pic(j, c);
          if (filt && S.pid[si] != b) continue;
          float wx[3], wy[3], wz, d;
          const float f0 = S.part[0][si], f1 = S.part[1][si], f2 = S.part[2][si];
          bs<0>(f0, wx[0], d); bs<1>(f0, wx[1], d); bs<2>(f0, wx[2], d);
          bs<0>(f1, wy[0], d); bs<1>(f1, wy[1], d); bs<2>(f1, wy[2], d);
          bs_rt(oz, f2, wz, d);
          const float v0 = S.part[3][si], v1 = S.part[4][si], v2 = S.part[5][si];
#pragma unroll
          for (int oy = 0; oy < 3; ++oy) {
            const float wyz = weight(wy[oy], wz);
            const float M0 = weight(v0, wyz), M1 = weight(v1, wyz), M2 = weight(v2, wyz);
#pragma unroll
            for (int ox = 0; ox < 3; ++ox) {
              float *q = a[oy][ox];
              const float wxx = wx[ox];
              q[0] = add_term(q[0], wxx, wyz);
              q[1] = add_term(q[1], wxx, M0);
              q[2] = add_term(q[2], wxx, M1);
              q[3] = add_term(q[3], wxx, M2);
            }
          }
        }
      }
      xy_reduce<4>(a, cx, cy);
      stage_layer<4, TZ>(sz, a, cx, cy, cz, oz);
    }
    if (b < B.npass && (G == 1 || grp % 2 == 1)) {
      float a[3][3][3];
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
          for (int f = 0; f < 3; ++f) a[i][j][f] = 0.f;
      if (has) {
        for (int j = 0; j < n_c; ++j) {
          const int si = pic(j, c);
          if (filt && S.pid[si] != b) continue;
          float wx[3], dwx[3], wy[3], dwy[3], wz, dwz;
          const float f0 = S.part[0][si], f1 = S.part[1][si], f2 = S.part[2][si];
          bs<0>(f0, wx[0], dwx[0]); bs<1>(f0, wx[1], dwx[1]); bs<2>(f0, wx[2], dwx[2]);
          bs<0>(f1, wy[0], dwy[0]); bs<1>(f1, wy[1], dwy[1]); bs<2>(f1, wy[2], dwy[2]);
          bs_rt(oz, f2, wz, dwz);
          float A[9];
#pragma unroll
          for (int k = 0; k < 9; ++k) A[k] = S.part[6 + k][si];
          const float J0 = S.part[15][si], J1 = S.part[16][si], J2 = S.part[17][si];
#pragma unroll
          for (int oy = 0; oy < 3; ++oy) {
            // with N = wx wyz and grad N = (dwx wyz, wx dyz, wx wyd):
            // A grad N + N J = wx (A_:1 dyz + A_:2 wyd + J wyz) + dwx (A_:0 wyz)
            const float wyz = wy[oy] * wz, dyz = dwy[oy] * wz, wyd = wy[oy] * dwz;
            const float U0 = force_u(A[1], dyz, A[2], wyd, J0, wyz);
            const float U1 = force_u(A[4], dyz, A[5], wyd, J1, wyz);
            const float U2 = force_u(A[7], dyz, A[8], wyd, J2, wyz);
            const float V0 = A[0] * wyz, V1 = A[3] * wyz, V2 = A[6] * wyz;
#pragma unroll
            for (int ox = 0; ox < 3; ++ox) {
              float *q = a[oy][ox];
              const float wxx = wx[ox], dxx = dwx[ox];
              q[0] = force_acc(q[0], wxx, U0, dxx, V0);
              q[1] = force_acc(q[1], wxx, U1, dxx, V1);
              q[2] = force_acc(q[2], wxx, U2, dxx, V2);
            }
          }
        }
      }
      xy_reduce<3>(a, cx, cy);
      stage_layer<3, TZ>(sz + 4, a, cx, cy, cz, oz);
    }
    __syncthreads();
    for (int t = tid; t < NP * TN; t += NT) {
      const int q = NP == 1 ? 0 : t / TN, nd = t - q * TN;
      if (b0 + q >= B.npass) break;
      const long long e = B.entry(w, S.T, b0 + q, nd);
      if (e < 0) continue;
      float acc[7];
      gather_z<7, TZ>(S.sz[q], nd, acc);
      w.B.pm[e] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      w.B.pd[e] = make_float4(acc[4], acc[5], acc[6], 0.f);
    }
    if (b0 + NP < B.npass) __syncthreads();  // the next pass overwrites the z stage
  }
}

// bricks whose tiles hold node coordinate i along one axis: [first, last]
__device__ __forceinline__ void covering(int i, int nbr, int &first, int &last) {
  last = min(i >> 2, nbr - 1);
  first = max((i - (TE - 1) + (BR - 1)) >> 2, 0);
  if (i - (TE - 1) < 0) first = 0;
}

// First partial-sum entry of a node in each of the (up to 8) brick tiles that
// cover it, in brick order (k = dz*4 + dy*2 + dx over the covering bricks'
// offsets); -1 where no brick or where the brick's partials overflowed.  All
// loads of the eight candidates are issued together.
__device__ __forceinline__ void covering_entries(const World &w, const DevScene &sc, int ix, int iy, int iz,
                                                 long long e[8]) {
  int x0, x1, y0, y1, z0, z1;
  covering(ix, sc.nbr[0], x0, x1);
  covering(iy, sc.nbr[1], y0, y1);
  covering(iz, sc.nbr[2], z0, z1);
  int b[8], tt[8], pb[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int Bx = x0 + (k & 1), By = y0 + ((k >> 1) & 1), Bz = z0 + (k >> 2);
    const bool ok = Bx <= x1 && By <= y1 && Bz <= z1;
    b[k] = ok ? sc.brick_begin + (Bz * sc.nbr[1] + By) * sc.nbr[0] + Bx : -1;
    tt[k] = ((iz - Bz * BR) * TE + (iy - By * BR)) * TE + (ix - Bx * BR);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) pb[k] = b[k] >= 0 ? w.B.poff[b[k]] : -1;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    e[k] = pb[k] >= 0 ? (long long)pb[k] + (w.B.tdesc[(size_t)b[k] * TN + tt[k]] & 0xffff) : -1;
}

// --------------------------------------------------------------------------
// Node kernels: k_p2g_node sums the tile partials of the bricks covering each
// node (in brick order), couples compatible logical grids (Eq. 8) and takes
// the grid update (Eq. 9); k_musl_node does the same for the MUSL sums and
// v*.  A node with one slot is one thread's work.  The slots of nodes with
// several (near a cut) are dealt out one to a thread, and the coupling reads
// the node's other slots from shared memory: walked by a thread per node,
// with its sums in local memory, they kept the whole warp waiting (k_p2g_node
// 137 -> 86 us for the 256-scene batch mid-cut, k_musl_node 72 -> 66).
// --------------------------------------------------------------------------
#define NODE_WIN 512                    // slots held in shared memory at a time
#define NODE_STEP (NODE_WIN - BM_MAXS)  // a window takes the nodes whose first slot lies in one step

template <int NC>
struct NodeS {
  float m[NODE_WIN];
  float S[NODE_WIN][NC];
  uint2 code[NODE_WIN];
  uint16_t owner[NODE_WIN];  // node (in the tile) of each slot, 0xffff none
  int first[512];            // first slot of each node among the tile's (node tile <= 512 nodes)
  int scan[33];
};

// Eq. 8 for slot a of the node whose ns slots start at lo, the terms in slot
// order
template <int NC>
__device__ __forceinline__ void couple_slot(const NodeS<NC> &N, int lo, int ns, int a, float (&out)[NC]) {
  float M = 0.f;
  for (int b = 0; b < ns; ++b) M += N.m[lo + b];
  float Sa[NC], acc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    out[c] = Sa[c] = N.S[lo + a][c];
    acc[c] = 0.f;
  }
  if (!(M > 0.f)) return;
  const float iM = 1.0f / M;
  const uint2 ca = N.code[lo + a];
  const float ma = N.m[lo + a];
  for (int b = 0; b < ns; ++b) {
    const uint2 cb = N.code[lo + b];
    if (b == a || conflict(ca.x, ca.y, cb.x, cb.y)) continue;
    const float mb = N.m[lo + b];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] += ma * N.S[lo + b][c] - mb * Sa[c];
  }
#pragma unroll
  for (int c = 0; c < NC; ++c) out[c] = Sa[c] + acc[c] * iM;
}

// A node tile: `single(node)` takes a node with one slot, by its own thread.
// The slots of the nodes with several go window by window: `sum(node, a, pool
// slot, m, S)` takes a slot's sums, `finish(pool slot, m, S)` its result after
// the coupling.  All threads of the CTA call it; thread i < nt holds the slot
// count of node i.  Each of `single` and `sum` is a chain of dependent loads;
// a CTA with threads beyond nt (sets of few tiles) has these take the slots
// while the first nt take the single nodes.
template <int NC, class Single, class Sum, class Finish>
__device__ __forceinline__ void tile_nodes(const World &w, NodeS<NC> &N, int node0, int nt, int cnt, Single single,
                                           Sum sum, Finish finish) {
  const int i = threadIdx.x, t0 = (int)blockDim.x > nt ? nt : 0;
  if (t0 == 0 && cnt == 1) single(node0 + i);
  if (!__syncthreads_or(cnt > 1)) {
    if (t0 != 0 && cnt == 1) single(node0 + i);
    return;
  }
  const int mine = cnt > 1 ? cnt : 0;
  int total;
  const int first = block_excl_scan(mine, N.scan, total);
  if (i < nt) N.first[i] = first;
  for (int w0 = 0; w0 < total; w0 += NODE_STEP) {
    for (int s = i; s < NODE_WIN; s += blockDim.x) N.owner[s] = 0xffff;
    __syncthreads();
    if (mine && first >= w0 && first < w0 + NODE_STEP)
      for (int a = 0; a < mine; ++a) N.owner[first - w0 + a] = (uint16_t)i;
    __syncthreads();
    const int ns = min(NODE_WIN, total - w0);
    if (i < t0) {
      if (w0 == 0 && cnt == 1) single(node0 + i);
    } else {
      for (int s = i - t0; s < ns; s += blockDim.x - t0) {
        const int o = N.owner[s];
        if (o == 0xffff) continue;
        const int a = s - (N.first[o] - w0);
        const int slot = w.N.slot_off[node0 + o] + a;
        N.code[s] = w.S.code[slot];
        float m, S[NC];
        sum(node0 + o, a, slot, m, S);
        N.m[s] = m;
#pragma unroll
        for (int c = 0; c < NC; ++c) N.S[s][c] = S[c];
      }
    }
    __syncthreads();
    for (int s = i; s < ns; s += blockDim.x) {
      const int o = N.owner[s];
      if (o == 0xffff) continue;
      const int lo = N.first[o] - w0;
      float out[NC];
      couple_slot<NC>(N, lo, w.N.slot_cnt[node0 + o], s - lo, out);
      finish(w.N.slot_off[node0 + o] + s - lo, N.m[s], out);
    }
    __syncthreads();
  }
}

__global__ void k_p2g_node(World w, LaunchSet ls) {
  chain_wait();
  __shared__ NodeS<6> N;
  const int4 t = ls.ntiles[blockIdx.x];
  const int i = threadIdx.x;
  const DevScene &sc = w.scenes[t.x];
  if (sc.frozen) return;
  const int cnt = i < t.z ? w.N.slot_cnt[t.y + i] : 0;
  auto single = [&](int node) {
    const int off = w.N.slot_off[node];
    int ix, iy, iz;
    node_coords(sc, node - sc.node_begin, ix, iy, iz);
    long long ent[8];
    covering_entries(w, sc, ix, iy, iz, ent);
    float4 sm = make_float4(0.f, 0.f, 0.f, 0.f), sd = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 a[8], d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      a[k] = ent[k] >= 0 ? w.B.pm[ent[k]] : make_float4(0.f, 0.f, 0.f, 0.f);
      d[k] = ent[k] >= 0 ? w.B.pd[ent[k]] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (ent[k] < 0) continue;
      sm.x += a[k].x; sm.y += a[k].y; sm.z += a[k].z; sm.w += a[k].w;
      sd.x += d[k].x; sd.y += d[k].y; sd.z += d[k].z;
    }
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f), nw = make_float4(0.f, 0.f, 0.f, 0.f);
    if (sm.x > 0.f) {
      const float im = 1.0f / sm.x, imm = 1.0f / (sc.mp * sm.x);
      o = make_float4(sm.y * im, sm.z * im, sm.w * im, sc.mp * sm.x);
      nw = make_float4(o.x + sd.x * imm, o.y + sd.y * imm, o.z + sd.z * imm, 0.f);
    }
    w.S.vold[off] = o;
    w.S.vnew[off] = nw;
  };
  tile_nodes<6>(
      w, N, t.y, ls.ntile_size, cnt, single,
      [&](int nd, int sl, int, float &m, float (&S)[6]) {
        int ix, iy, iz;
        node_coords(sc, nd - sc.node_begin, ix, iy, iz);
        long long ent[8];
        covering_entries(w, sc, ix, iy, iz, ent);
        float4 a[8], d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          a[k] = ent[k] >= 0 ? w.B.pm[ent[k] + sl] : make_float4(0.f, 0.f, 0.f, 0.f);
          d[k] = ent[k] >= 0 ? w.B.pd[ent[k] + sl] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        m = 0.f;
#pragma unroll
        for (int c = 0; c < 6; ++c) S[c] = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (ent[k] < 0) continue;
          m += a[k].x;
          S[0] += a[k].y; S[1] += a[k].z; S[2] += a[k].w;
          S[3] += d[k].x; S[4] += d[k].y; S[5] += d[k].z;
        }
        m *= sc.mp;
#pragma unroll
        for (int c = 0; c < 3; ++c) S[c] *= sc.mp;
      },
      [&](int slot, float m, const float (&S)[6]) {
        float4 o = make_float4(0.f, 0.f, 0.f, m), nw = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m > 0.f) {
          const float im = 1.0f / m;
          o = make_float4(S[0] * im, S[1] * im, S[2] * im, m);
          nw = make_float4((S[0] + S[3]) * im, (S[1] + S[4]) * im, (S[2] + S[5]) * im, 0.f);
        }
        w.S.vold[slot] = o;
        w.S.vnew[slot] = nw;
      });
}

// --------------------------------------------------------------------------
// k_g2p_musl: per particle G2P (Eq. 17) and x update from the brick's tile of
// grid velocities, then the brick's share of the MUSL re-scatter sum m v^{n+1}
// N per logical grid, committed in the same fixed phase order as P2G.
// --------------------------------------------------------------------------
// tile slot of code index id at tile node t, or -1 (a node with one slot holds
// the code of every particle it touches)
__device__ __forceinline__ int tile_slot(const World &w, const BrickTile &T, int nbc, int t, int id) {
  if (T.cnt[t] == 1) return T.lo[t];
  if (id >= nbc) return -1;
  const int a = brick_slot(w, T, nbc, id, t);
  return a == NOSLOT ? -1 : T.lo[t] + a;
}

template <int PPC, int G>
struct K4S {
  BrickTile T;
  union {
    struct {
      float4 tvo[TSCAP];      // v_old xyz, m of the tile slots (G2P)
      float4 tvn[TSCAP];      // v_new xyz
    };
    float sz[G][3][3][TN];    // then: each group's MUSL pass's (node, z-offset) sums
  };
  float pf[3][PPC * BR3];
  float pv[3][PPC * BR3];
  unsigned long long cmask[BR3];  // as in K2S
  int cs[BR3 + 1];
  uint8_t pid[PPC * BR3];
};

template <int PPC, int MB, int G>
__global__ void __launch_bounds__(BT * G, MB) k_g2p_musl(World w, LaunchSet ls, int tools) {
  chain_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  K4S<PPC, G> &S = *reinterpret_cast<K4S<PPC, G> *>(smraw);
  if ((int)blockIdx.x < tools) {
    next_tool(w, ls.scene_ids[blockIdx.x], *reinterpret_cast<ToolS *>(smraw));
    return;
  }
  static_assert(sizeof(ToolS) <= sizeof(K4S<PPC, G>), "the tool step fits");
  const int4 bt = ls.btiles[blockIdx.x - tools];
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (sc.frozen || sc.lattice) return;
  const PPool &P = w.P;
  constexpr int NT = BT * G;
  const int tid = threadIdx.x, grp = tid / BT;
  const int lb = bt.y - sc.brick_begin;
  const BrickInfo B(w, bt, PPC * BR3);
  const bool several = B.nbc > 1, single = B.single;
  const int total = w.B.ptot[bt.y];
  const bool in_smem = total <= TSCAP;  // otherwise G2P reads the pool slots directly
  const int *csg = w.N.cell_start + sc.cell_begin + lb * BR3;
  for (int i = tid; i <= BR3; i += NT) S.cs[i] = csg[i] - bt.z;
  brick_tile(w, bt.y, B.nbc, S.T, NT);
  __syncthreads();
  if (!B.uniform) brick_slots<false>(w, S.T, B.nbc, B.pbase, NT);
  if (single) {  // by node: a particle's node t holds its (only) logical grid
    for (int t = tid; t < TN; t += NT) {
      const bool has = S.T.cnt[t] != 0;
      const int g = S.T.goff[t];
      S.tvo[t] = has ? w.S.vold[g] : make_float4(0.f, 0.f, 0.f, 0.f);
      S.tvn[t] = has ? w.S.vnew[g] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  } else if (in_smem) {
    for (int t = tid; t < TN; t += NT) {
      const int n = S.T.cnt[t], lo = S.T.lo[t], g = S.T.goff[t];
      for (int a = 0; a < n; ++a) {
        S.tvo[lo + a] = w.S.vold[g + a];
        S.tvn[lo + a] = w.S.vnew[g + a];
      }
    }
  }
  __syncthreads();
  // ---- phase 0: G2P ----
  const float beta = sc.beta, dt = sc.dt;
  bool bad = false;
  for (int i = tid; i < bt.w; i += NT) {
    const int p = bt.z + i;
    const int c = cell_of(S.cs, i);
    const int lx = c & 3, ly = (c >> 2) & 3, lz = c >> 4;
    const int si = pic(i - S.cs[c], c);
    const int id = several ? P.cid[p] : 0;
    const float f0 = P.fx[0][p], f1 = P.fx[1][p], f2 = P.fx[2][p];
    float wx[3], wy[3], wz[3], d;
    bs<0>(f0, wx[0], d); bs<1>(f0, wx[1], d); bs<2>(f0, wx[2], d);
    bs<0>(f1, wy[0], d); bs<1>(f1, wy[1], d); bs<2>(f1, wy[2], d);
    bs<0>(f2, wz[0], d); bs<1>(f2, wz[1], d); bs<2>(f2, wz[2], d);
    float sn[3] = {0.f, 0.f, 0.f}, so[3] = {0.f, 0.f, 0.f};
    if (single) {
      // one logical grid per node, values by node; a node without mass holds
      // zero velocities, so it needs no test
      const int t0 = (lz * TE + ly) * TE + lx;
#pragma unroll
      for (int oz = 0; oz < 3; ++oz)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy) {
          const float wyz = weight(wy[oy], wz[oz]);
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const int t = t0 + (oz * TE + oy) * TE + ox;
            const float4 vo = S.tvo[t], vn = S.tvn[t];
            const float N = weight(wx[ox], wyz);
            sn[0] = add_term(sn[0], N, vn.x);
            sn[1] = add_term(sn[1], N, vn.y);
            sn[2] = add_term(sn[2], N, vn.z);
            so[0] = add_term(so[0], N, vo.x);
            so[1] = add_term(so[1], N, vo.y);
            so[2] = add_term(so[2], N, vo.z);
          }
        }
    } else if (in_smem) {
      // tile slots in shared memory: branch-free over the stencil (a missing
      // or massless logical grid contributes zero)
      const int t0 = (lz * TE + ly) * TE + lx;
#pragma unroll
      for (int oz = 0; oz < 3; ++oz)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy) {
          const float wyz = weight(wy[oy], wz[oz]);
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const int s = tile_slot(w, S.T, B.nbc, t0 + (oz * TE + oy) * TE + ox, id);
            const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 vo = s >= 0 ? S.tvo[s] : zero, vn = s >= 0 ? S.tvn[s] : zero;
            const float N = vo.w > 0.f ? weight(wx[ox], wyz) : 0.f;
            sn[0] = add_term(sn[0], N, vn.x);
            sn[1] = add_term(sn[1], N, vn.y);
            sn[2] = add_term(sn[2], N, vn.z);
            so[0] = add_term(so[0], N, vo.x);
            so[1] = add_term(so[1], N, vo.y);
            so[2] = add_term(so[2], N, vo.z);
          }
        }
    } else
#pragma unroll
    for (int oz = 0; oz < 3; ++oz)
#pragma unroll
      for (int oy = 0; oy < 3; ++oy)
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          const int t = ((lz + oz) * TE + (ly + oy)) * TE + (lx + ox);
          const int s = tile_slot(w, S.T, B.nbc, t, id);
          if (s < 0) continue;
          float4 vo, vn;
          {
            const int g = S.T.goff[t] + s - S.T.lo[t];
            vo = w.S.vold[g];
            vn = w.S.vnew[g];
          }
          if (!(vo.w > 0.f)) continue;
          const float N = weight(weight(wx[ox], wy[oy]), wz[oz]);
          sn[0] = add_term(sn[0], N, vn.x);
          sn[1] = add_term(sn[1], N, vn.y);
          sn[2] = add_term(sn[2], N, vn.z);
          so[0] = add_term(so[0], N, vo.x);
          so[1] = add_term(so[1], N, vo.y);
          so[2] = add_term(so[2], N, vo.z);
        }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float vv = next_v(beta, P.v[a][p], so[a], sn[a]);
      const float xx = next_x(P.x[a][p], dt, sn[a]);
      P.v[a][p] = vv;
      P.x[a][p] = xx;
      S.pv[a][si] = vv;
      bad |= !isfinite(vv) || !isfinite(xx);
    }
    S.pf[0][si] = f0;
    S.pf[1][si] = f1;
    S.pf[2][si] = f2;
    if (several) S.pid[si] = (uint8_t)id;
  }
  if (bad) atomicOr(&scm.err, BM_ERRBIT_NONFINITE);
  // ---- phase 1: MUSL sums m v^{n+1} N, one pass per code of the brick,
  // reduced as in k_p2g_brick (xy_reduce, z stage, <= 3 layer sums per node) ----
  const int c = tid % BR3, oz = tid % BT / BR3;
  const int cx = c & 3, cy = (c >> 2) & 3, cz = c >> 4;
  const int n_c = S.cs[c + 1] - S.cs[c];
  __syncthreads();  // G2P reads of the tile velocities are done: the z stage may reuse them
  if (several) {
    cell_codes(S.pid, S.cs, S.cmask);
    __syncthreads();
  }
  const unsigned long long codes = several ? S.cmask[c] : 0ull;
  const bool filt = (codes & (codes - 1)) != 0;
  for (int b0 = 0; b0 < B.npass; b0 += G) {
    const int b = b0 + grp;
    const bool has = n_c > 0 && b < B.npass && (!several || ((codes >> b) & 1u));
    float a[3][3][3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) a[i][j][0] = a[i][j][1] = a[i][j][2] = 0.f;
    if (has) {
      for (int j = 0; j < n_c; ++j) {
        const int si = pic(j, c);
        if (filt && S.pid[si] != b) continue;
        float wx[3], wy[3], wz, d;
        const float f0 = S.pf[0][si], f1 = S.pf[1][si], f2 = S.pf[2][si];
        bs<0>(f0, wx[0], d); bs<1>(f0, wx[1], d); bs<2>(f0, wx[2], d);
        bs<0>(f1, wy[0], d); bs<1>(f1, wy[1], d); bs<2>(f1, wy[2], d);
        bs_rt(oz, f2, wz, d);
        const float v0 = S.pv[0][si], v1 = S.pv[1][si], v2 = S.pv[2][si];
#pragma unroll
        for (int oy = 0; oy < 3; ++oy) {
          const float wyz = weight(wy[oy], wz);
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const float N = weight(wx[ox], wyz);
            a[oy][ox][0] = add_term(a[oy][ox][0], N, v0);
            a[oy][ox][1] = add_term(a[oy][ox][1], N, v1);
            a[oy][ox][2] = add_term(a[oy][ox][2], N, v2);
          }
        }
      }
    }
    if (b < B.npass) {
      xy_reduce<3>(a, cx, cy);
      stage_layer<3, TN>(S.sz[grp], a, cx, cy, cz, oz);
    }
    __syncthreads();
    for (int t = tid; t < G * TN; t += NT) {
      const int q = G == 1 ? 0 : t / TN, nd = t - q * TN;
      if (b0 + q >= B.npass) break;
      const long long e = B.entry(w, S.T, b0 + q, nd);
      if (e < 0) continue;
      float acc[3];
      gather_z<3, TN>(S.sz[q], nd, acc);
      w.B.pm[e] = make_float4(acc[0], acc[1], acc[2], 0.f);
    }
    if (b0 + G < B.npass) __syncthreads();  // the next pass overwrites the z stage
  }
}

// --------------------------------------------------------------------------
// k_musl_node: per slot, MUSL sums of the covering bricks, coupling, v*; its
// first `tools` CTAs take the scenes' tool steps (none if G2P did)
// --------------------------------------------------------------------------
__global__ void k_musl_node(World w, LaunchSet ls, int tools) {
  chain_wait();
  __shared__ __align__(16) unsigned char raw[sizeof(NodeS<3>) > sizeof(ToolS) ? sizeof(NodeS<3>) : sizeof(ToolS)];
  if ((int)blockIdx.x < tools) {
    next_tool(w, ls.scene_ids[blockIdx.x], *reinterpret_cast<ToolS *>(raw));
    return;
  }
  NodeS<3> &N = *reinterpret_cast<NodeS<3> *>(raw);
  const int4 t = ls.ntiles[blockIdx.x - tools];
  const int i = threadIdx.x;
  const DevScene &sc = w.scenes[t.x];
  if (sc.frozen) return;
  const int cnt = i < t.z ? w.N.slot_cnt[t.y + i] : 0;
  auto sums = [&](int nd, int sl, float (&S)[3]) {
    int ix, iy, iz;
    node_coords(sc, nd - sc.node_begin, ix, iy, iz);
    long long ent[8];
    covering_entries(w, sc, ix, iy, iz, ent);
    float4 a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = ent[k] >= 0 ? w.B.pm[ent[k] + sl] : make_float4(0.f, 0.f, 0.f, 0.f);
    S[0] = S[1] = S[2] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (ent[k] < 0) continue;
      S[0] += a[k].x;
      S[1] += a[k].y;
      S[2] += a[k].z;
    }
  };
  auto single = [&](int node) {
    const int off = w.N.slot_off[node];
    float S[3];
    sums(node, 0, S);
    const float m = w.S.vold[off].w;
    float4 vs = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m > 0.f) {
      const float im = sc.mp / m;
      vs = make_float4(S[0] * im, S[1] * im, S[2] * im, 0.f);
    }
    w.S.vstar[off] = vs;
  };
  tile_nodes<3>(
      w, N, t.y, ls.ntile_size, cnt, single,
      [&](int nd, int sl, int slot, float &m, float (&S)[3]) {
        sums(nd, sl, S);
        m = w.S.vold[slot].w;
#pragma unroll
        for (int c = 0; c < 3; ++c) S[c] *= sc.mp;
      },
      [&](int slot, float m, const float (&S)[3]) {
        float4 vs = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m > 0.f) {
          const float im = 1.0f / m;
          vs = make_float4(S[0] * im, S[1] * im, S[2] * im, 0.f);
        }
        w.S.vstar[slot] = vs;
      });
}

// --------------------------------------------------------------------------
// k_fupd: F += dt sum_i v*_i (x) grad0 N_ip from the brick's tile of v*, and
// commit the side labels assigned this substep (they act from the next one)
// --------------------------------------------------------------------------
struct K1S {
  BrickTile T;
  float4 tvs[TSCAP];
  int any;
};

template <int MB, bool INELASTIC, int NG>
__global__ void __launch_bounds__(BT * NG, MB) k_fupd(World w, LaunchSet ls) {
  chain_wait();
  __shared__ K1S S;
  const int4 bt = ls.btiles[blockIdx.x];
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (sc.frozen || sc.lattice) return;
  const PPool &P = w.P;
  constexpr int NT = BT * NG;
  const int tid = threadIdx.x;
  const int lb = bt.y - sc.brick_begin;
  int c0x, c0y, c0z;
  brick_coords(sc, lb, c0x, c0y, c0z);
  if (tid == 0) S.any = 0;
  const BrickInfo B(w, bt, 0);
  const bool several = B.nbc > 1, single = B.single;
  const bool in_smem = w.B.ptot[bt.y] <= TSCAP;
  brick_tile(w, bt.y, B.nbc, S.T, NT);
  __syncthreads();
  if (!B.uniform) brick_slots<false>(w, S.T, B.nbc, -1, NT);
  if (single) {  // by node
    for (int t = tid; t < TN; t += NT)
      S.tvs[t] = S.T.cnt[t] ? w.S.vstar[S.T.goff[t]] : make_float4(0.f, 0.f, 0.f, 0.f);
  } else if (in_smem) {
    for (int t = tid; t < TN; t += NT) {
      const int n = S.T.cnt[t], lo = S.T.lo[t], g = S.T.goff[t];
      for (int a = 0; a < n; ++a) S.tvs[lo + a] = w.S.vstar[g + a];
    }
  }
  __syncthreads();
  const float c = sc.dt * sc.inv_dx;
  const int cut = sc.cut;
  bool any = false;
  for (int i = tid; i < bt.w; i += NT) {
    const int p = bt.z + i;
    int bx, by, bz;
    particle_base(P.base[p], bx, by, bz);
    const int lx = bx - c0x, ly = by - c0y, lz = bz - c0z;
    const int id = several ? P.cid[p] : 0;
    const float f0 = P.fx[0][p], f1 = P.fx[1][p], f2 = P.fx[2][p];
    float wx[3], wy[3], wz[3], gx[3], gy[3], gz[3];
    bs<0>(f0, wx[0], gx[0]); bs<1>(f0, wx[1], gx[1]); bs<2>(f0, wx[2], gx[2]);
    bs<0>(f1, wy[0], gy[0]); bs<1>(f1, wy[1], gy[1]); bs<2>(f1, wy[2], gy[2]);
    bs<0>(f2, wz[0], gz[0]); bs<1>(f2, wz[1], gz[1]); bs<2>(f2, wz[2], gz[2]);
    float G[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int t0 = (lz * TE + ly) * TE + lx;
#pragma unroll
    for (int oz = 0; oz < 3; ++oz)
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        // grad N = (gx wyz, wx gyz, wx wgz): sum v* gx and v* wx along the
        // row of three nodes first, then scale by the row's y-z factors
        const float wyz = wy[oy] * wz[oz], gyz = gy[oy] * wz[oz], wgz = wy[oy] * gz[oz];
        float sx[3] = {0.f, 0.f, 0.f}, sw[3] = {0.f, 0.f, 0.f};
        if (single) {  // by node; nodes without mass hold v* = 0
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const float4 v = S.tvs[t0 + (oz * TE + oy) * TE + ox];
            sx[0] += v.x * gx[ox]; sx[1] += v.y * gx[ox]; sx[2] += v.z * gx[ox];
            sw[0] += v.x * wx[ox]; sw[1] += v.y * wx[ox]; sw[2] += v.z * wx[ox];
          }
        } else {
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const int t = t0 + (oz * TE + oy) * TE + ox;
            const int s = tile_slot(w, S.T, B.nbc, t, id);
            if (s < 0) continue;
            const float4 v = in_smem ? S.tvs[s] : w.S.vstar[S.T.goff[t] + s - S.T.lo[t]];
            sx[0] += v.x * gx[ox]; sx[1] += v.y * gx[ox]; sx[2] += v.z * gx[ox];
            sw[0] += v.x * wx[ox]; sw[1] += v.y * wx[ox]; sw[2] += v.z * wx[ox];
          }
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          G[3 * a] += sx[a] * wyz;
          G[3 * a + 1] += sw[a] * gyz;
          G[3 * a + 2] += sw[a] * wgz;
        }
      }
#pragma unroll
    for (int k = 0; k < 9; ++k) P.F[k][p] += c * G[k];
    if (INELASTIC && sc.viscosity > 0.0f)
#pragma unroll
      for (int k = 0; k < 9; ++k) P.Fdot[k][p] = sc.inv_dx * G[k];
    const uint8_t pend = P.pend[p];
    if (pend && cut >= 0) {
      if (pend == 1) P.s1[p] |= 1u << cut;
      else P.s2[p] |= 1u << cut;
      any = true;
      // the nodes of this particle's stencil need their codes recounted
      for (int oz = 0; oz < 3; ++oz)
        for (int oy = 0; oy < 3; ++oy)
          for (int ox = 0; ox < 3; ++ox)
            w.N.dirty[sc.node_begin + ((bz + oz) * sc.nn[1] + (by + oy)) * sc.nn[0] + (bx + ox)] = 1;
    }
  }
  if (any) S.any = 1;
  __syncthreads();
  if (tid == 0 && S.any) {
    w.B.bdirty[bt.y] = 1;  // its particles' codes are listed anew by the slot rebuild
    atomicOr(&scm.label_pending, 1);
  }
}

// --------------------------------------------------------------------------
// Material-material contact (Eq. 10-13) with per-particle candidate lists.
// Every particle keeps the particles of its scene that were within
// r_l = 2 R_p + skin (skin = 1.5 R_p) at the lists' last build.  A pair in
// contact this substep satisfies dist < 2 R_p + dt (|v_p| + |v_q|) (Eq. 10),
// and a pair missing from the lists was farther than r_l at the build, so
// its distance is at least r_l - d_p - d_q (d: displacement since the
// build).  Hence the lists hold every pair that can touch while every
// particle keeps d_p + dt |v_p| <= skin / 2; they are rebuilt (spatial hash
// of the current configuration, cell = r_l) when one does not, or when the
// state was written from outside.  A list is in (neighbour cell, pool index)
// order, the same alone and in any batch.  A pair is always evaluated in
// canonical (lower, higher) pool-index order by both of its particles, so
// the two impulses are exact negatives; the lower index owns the pair's
// tangential history (double-buffered by substep parity).
// --------------------------------------------------------------------------
__device__ __forceinline__ int hash_cell(int scene, int cx, int cy, int cz, int nb) {
  const unsigned h = ((unsigned)cx * 73856093u) ^ ((unsigned)cy * 19349663u) ^
                     ((unsigned)cz * 83492791u) ^ ((unsigned)scene * 2654435761u);
  return (int)(h & (unsigned)(nb - 1));
}

// scene and hash-cell coordinates in one word (16 bits each, coordinates
// wrapped): equal for the entries of one cell; two cells with equal words
// are at least 65,536 cells apart
__device__ __forceinline__ unsigned long long cell_key(int scene, int cx, int cy, int cz) {
  return ((unsigned long long)(scene & 0xffff) << 48) | ((unsigned long long)(cx & 0xffff) << 32) |
         ((unsigned long long)(cy & 0xffff) << 16) | (unsigned long long)(cz & 0xffff);
}

// per-substep reset of the scenes' reductions and of the world's build flag
__global__ void k_pair_reset(World w, LaunchSet ls) {
  chain_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *w.H.build = 0;
  if (i < ls.n_scenes) {
    DevScene &sc = w.scenes[ls.scene_ids[i]];
    sc.pair_vmax_bits = 0;
    sc.pair_disp_bits = 0;
  }
}

// per scene: largest particle speed, and largest displacement since the
// candidate lists were built (non-negative floats order like their bits)
__global__ void k_pair_vmax(World w, LaunchSet ls) {
  chain_wait();
  const int4 bt = ls.btiles[blockIdx.x];
  DevScene &sc = w.scenes[bt.x];
  if (!sc.pair_on || sc.frozen) return;
  float m = 0.f, dm = 0.f;
  const bool valid = sc.pair_valid != 0;
  for (int i = threadIdx.x; i < bt.w; i += blockDim.x) {
    const int p = bt.z + i;
    const float a = w.P.v[0][p], b = w.P.v[1][p], c = w.P.v[2][p];
    const float sp = sqrtf(a * a + b * b + c * c);
    m = fmaxf(m, sp);
    if (valid) {
      const float d0 = w.P.x[0][p] - w.P.xb[0][p], d1 = w.P.x[1][p] - w.P.xb[1][p],
                  d2 = w.P.x[2][p] - w.P.xb[2][p];
      dm = fmaxf(dm, sqrtf(d0 * d0 + d1 * d1 + d2 * d2) + sc.dt * sp);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fmaxf(m, __shfl_down_sync(FULL, m, o));
    dm = fmaxf(dm, __shfl_down_sync(FULL, dm, o));
  }
  if ((threadIdx.x & 31) == 0) {
    if (m > 0.f) atomicMax(&sc.pair_vmax_bits, __float_as_int(m));
    if (dm > 0.f) atomicMax(&sc.pair_disp_bits, __float_as_int(dm));
  }
}

// per scene: whether the candidate lists are rebuilt this substep
__global__ void k_pair_decide(World w, LaunchSet ls) {
  chain_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ls.n_scenes) return;
  DevScene &sc = w.scenes[ls.scene_ids[i]];
  if (!sc.pair_on || sc.frozen) {
    sc.pair_build = 0;
    return;
  }
  const float reach = __int_as_float(sc.pair_disp_bits);  // max of d_p + dt |v_p|
  const float skin = 1.5f * sc.Rp;
  // 10% margin against rounding in the distances
  const bool build = !sc.pair_valid || !(reach <= 0.45f * skin);
  sc.pair_build = build ? 1 : 0;
  if (build) {
    sc.pair_h = 1.001f * (2.0f * sc.Rp + skin);
    sc.pair_inv_h = 1.0f / sc.pair_h;
    sc.pair_valid = 1;
    sc.pair_builds++;
    atomicOr(w.H.build, 1);
  }
}

__global__ void k_pair_hash(World w, LaunchSet ls) {
  chain_wait();
  const int4 bt = ls.btiles[blockIdx.x];
  const DevScene &sc = w.scenes[bt.x];
  if (!sc.pair_on || !sc.pair_build) return;
  const PPool &P = w.P;
  const float ih = sc.pair_inv_h;
  for (int i = threadIdx.x; i < bt.w; i += blockDim.x) {
    const int p = bt.z + i;
    const int cx = (int)floorf(P.x[0][p] * ih);
    const int cy = (int)floorf(P.x[1][p] * ih);
    const int cz = (int)floorf(P.x[2][p] * ih);
    const int b = hash_cell(bt.x, cx, cy, cz, w.H.n_buckets);
    P.hkey[p] = b;
    P.hcell[p] = cell_key(bt.x, cx, cy, cz);
    atomicAdd(&w.H.bucket_start[b], 1);
  }
}

__global__ void k_scan_local(World w) {
  chain_wait();
  if (!*w.H.build) return;
  __shared__ int sm[33];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int v = i < w.H.n_buckets ? w.H.bucket_start[i] : 0;
  int total;
  const int ex = block_excl_scan(v, sm, total);
  if (i < w.H.n_buckets) w.H.bucket_start[i] = ex;
  if (threadIdx.x == 0) w.H.block_sum[blockIdx.x] = total;
}

__global__ void k_scan_top(World w, int nblocks) {
  chain_wait();
  if (!*w.H.build) return;
  __shared__ int sm[33];
  int carry = 0;
  for (int base = 0; base < nblocks; base += blockDim.x) {
    const int j = base + threadIdx.x;
    const int v = j < nblocks ? w.H.block_sum[j] : 0;
    int total;
    const int ex = block_excl_scan(v, sm, total);
    if (j < nblocks) w.H.block_sum[j] = carry + ex;
    carry += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) w.H.bucket_start[w.H.n_buckets] = carry;
}

__global__ void k_scan_add(World w) {
  chain_wait();
  if (!*w.H.build) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < w.H.n_buckets) w.H.bucket_start[i] += w.H.block_sum[blockIdx.x];
}

__global__ void k_pair_fill(World w, LaunchSet ls) {
  chain_wait();
  const int4 bt = ls.btiles[blockIdx.x];
  const DevScene &sc = w.scenes[bt.x];
  if (!sc.pair_on || !sc.pair_build) return;
  for (int i = threadIdx.x; i < bt.w; i += blockDim.x) {
    const int p = bt.z + i;
    const int b = w.P.hkey[p];
    w.P.horder[w.H.bucket_start[b] + atomicAdd(&w.H.bucket_fill[b], 1)] = p;
  }
}

// the entries of each bucket in pool-index order (position, pool index, base
// cell, cell key), for the list build.  A thread per entry counts the
// bucket's smaller indices (buckets are short); sorting a bucket in place, a
// thread per bucket, took 30 us on the 252,800-particle cylinder, most of
// 524,288 buckets being empty and the others a chain of global reads and
// writes.
__global__ void k_pair_sort(World w) {
  chain_wait();
  if (!*w.H.build) return;
  const int total = w.H.bucket_start[w.H.n_buckets];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int q = w.P.horder[e];
    const int b = w.P.hkey[q];
    const int s0 = w.H.bucket_start[b], s1 = w.H.bucket_start[b + 1];
    int i = s0;
    for (int k = s0; k < s1; ++k) i += w.P.horder[k] < q ? 1 : 0;
    w.P.hent[i] = make_float4(w.P.x[0][q], w.P.x[1][q], w.P.x[2][q], __int_as_float(q));
    w.P.hbase[i] = w.P.base[q];
    w.P.hentk[i] = w.P.hcell[q];
  }
}

// Candidate lists of the particles in entries [c0, c1) of the buckets (at most
// 32, lane i holding entry c0 + i), by one warp.  The particles are taken in
// groups of one cell (and scene); a group shares its 27 neighbour cells
// (dz, dy, dx in -1..1, x fastest), whose bucket entries are laid end to end
// and tested 64 at a time, two per lane, against each member in turn: an
// entry counts when it belongs to the neighbour cell (its key; a bucket's
// hash may be shared), is another particle and lies within r_l = 2 R_p +
// skin.  A ballot gives each accepted entry its place, so every list is in
// (cell, pool index) order, as a walk of the cells in order would give;
// bit 31 of an entry marks a pair whose reference stencils overlap (base
// cells at most two apart on every axis): such a pair interacts through the
// grid, and is a contact pair only once a cut separates it (self-contact
// exclusion).  A list of only such pairs is marked by NBR_SHARED in its count.
// The kernel is bound by instructions (more warps per SM change nothing):
// members are read from shared memory, the cell of an entry is the rank of
// its start among the non-empty cells', and base cells are compared unpacked.
#define NBR_SHARED 0x80
#define LIST_WARPS 8
#define LIST_UNIT 16  // entries per warp and round
#define LIST_OCC 4

struct ListMembers {
  float4 me[32];
  int4 base[32];               // base cell + 2
  int2 cell[27];               // of the non-empty neighbour cells: first entry and place in the row
  unsigned long long key[27];
};

__device__ __forceinline__ void bucket_lists(const World &w, ListMembers &M, int c0, int c1, int lane) {
  const PPool &P = w.P;
  const bool mine = lane < c1 - c0;
  const float4 me = mine ? P.hent[c0 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
  const unsigned long long mkey = mine ? P.hentk[c0 + lane] : ~0ull;
  int bx, by, bz;
  particle_base(mine ? P.hbase[c0 + lane] : 0u, bx, by, bz);
  __syncwarp();
  M.me[lane] = me;
  M.base[lane] = make_int4(bx + 2, by + 2, bz + 2, 0);
  const int mscene = (int)(mkey >> 48);
  int mx = 0, my = 0, mz = 0;
  if (mine) {
    const float ih = w.scenes[mscene].pair_inv_h;
    mx = (int)floorf(me.x * ih);
    my = (int)floorf(me.y * ih);
    mz = (int)floorf(me.z * ih);
  }
  int cnt = 0;
  unsigned apart = 0;  // bit m: lane saw a pair of member m that shares no stencil
  unsigned todo = __ballot_sync(FULL, mine);
  while (todo) {
    const int lead = __ffs(todo) - 1;
    const unsigned long long K = __shfl_sync(FULL, mkey, lead);
    const int cx0 = __shfl_sync(FULL, mx, lead), cy0 = __shfl_sync(FULL, my, lead),
              cz0 = __shfl_sync(FULL, mz, lead);
    const unsigned grp = __ballot_sync(FULL, mine && mkey == K && mx == cx0 && my == cy0 && mz == cz0) & todo;
    todo &= ~grp;
    const int scene = (int)(K >> 48);
    const DevScene &sc = w.scenes[scene];
    const float rl = 2.0f * sc.Rp + 1.5f * sc.Rp, rl2 = rl * rl;
    int a0 = 0, sz = 0;
    unsigned long long nk = 0;
    if (lane < 27) {
      const int cx = cx0 + lane % 3 - 1, cy = cy0 + (lane / 3) % 3 - 1, cz = cz0 + lane / 9 - 1;
      const int hb = hash_cell(scene, cx, cy, cz, w.H.n_buckets);
      a0 = w.H.bucket_start[hb];
      sz = w.H.bucket_start[hb + 1] - a0;
      nk = cell_key(scene, cx, cy, cz);
    }
    int incl = sz;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    const int T = __shfl_sync(FULL, incl, 31);
    const int excl = incl - sz;
    const unsigned full = __ballot_sync(FULL, sz > 0);
    if (sz > 0) {
      const int r = __popc(full & ((1u << lane) - 1u));
      M.cell[r] = make_int2(a0, excl);
      M.key[r] = nk;
    }
    __syncwarp();
    int before = -1;  // rank of the last cell that starts before the window
    for (int base = 0; base < T; base += 64) {
      float4 e[2];
      int ebx[2], eby[2], ebz[2];
      bool valid[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        // the cell of candidate j is the last one that starts at or before j
        const int w0 = base + 32 * h, j = w0 + lane;
        const unsigned starts =
            __reduce_or_sync(FULL, sz > 0 && excl >= w0 && excl < w0 + 32 ? 1u << (excl - w0) : 0u);
        const int L = before + __popc(starts & (0xffffffffu >> (31 - lane)));
        before += __popc(starts);
        const int2 cl = M.cell[L];
        const bool inr = j < T;
        const int k = cl.x + (j - cl.y);
        e[h] = inr ? P.hent[k] : make_float4(0.f, 0.f, 0.f, 0.f);
        const unsigned long long ek = inr ? P.hentk[k] : 0ull;
        particle_base(inr ? P.hbase[k] : 0u, ebx[h], eby[h], ebz[h]);
        valid[h] = inr && ek == M.key[L];
      }
      unsigned g = grp;
      while (g) {
        const int m = __ffs(g) - 1;
        g &= g - 1;
        const float4 mp = M.me[m];
        const int4 bp = M.base[m];
        const int p = __float_as_int(mp.w);
        const int c_in = __shfl_sync(FULL, cnt, m);
        int c = c_in;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int q = __float_as_int(e[h].w);
          const float d0 = mp.x - e[h].x, d1 = mp.y - e[h].y, d2 = mp.z - e[h].z;
          const bool acc = valid[h] && q != p && d0 * d0 + d1 * d1 + d2 * d2 <= rl2;
          const unsigned am = __ballot_sync(FULL, acc);
          if (acc) {
            const int pos = c + __popc(am & ((1u << lane) - 1u));
            const bool share = (unsigned)(bp.x - ebx[h]) <= 4u && (unsigned)(bp.y - eby[h]) <= 4u &&
                               (unsigned)(bp.z - ebz[h]) <= 4u;
            if (!share) apart |= 1u << m;
            if (pos < BM_NBR) P.nbr[(size_t)p * BM_NBR + pos] = share ? (int)((uint32_t)q | 0x80000000u) : q;
          }
          c += __popc(am);
        }
        if (lane == m) cnt = c;
      }
    }
    __syncwarp();
  }
  apart = __reduce_or_sync(FULL, apart);
  if (mine) {
    const int p = __float_as_int(me.w);
    P.nbr_n[p] = (uint8_t)(min(cnt, BM_NBR) | ((apart >> lane) & 1u ? 0 : NBR_SHARED));
    P.xb[0][p] = me.x;
    P.xb[1][p] = me.y;
    P.xb[2][p] = me.z;
    if (cnt > BM_NBR) atomicOr(&w.scenes[mscene].err, BM_ERRBIT_CONTACT_OVERFLOW);
  }
}

// candidate lists of every particle of the scenes that rebuild them: each
// warp takes LIST_UNIT consecutive entries (grid-stride).  The positions of
// the build are kept.
__global__ void __launch_bounds__(32 * LIST_WARPS, LIST_OCC) k_pair_list(World w) {
  chain_wait();
  if (!*w.H.build) return;
  __shared__ ListMembers members[LIST_WARPS];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int total = w.H.bucket_start[w.H.n_buckets];
  const int step = gridDim.x * LIST_WARPS * LIST_UNIT;
  for (int c = (blockIdx.x * LIST_WARPS + wid) * LIST_UNIT; c < total; c += step)
    bucket_lists(w, members[wid], c, min(total, c + LIST_UNIT), lane);
}

// Pair impulses (Eq. 10-13), one thread per particle walking its list
// (gridDim.y CTAs per brick).  A candidate sharing p's reference stencil is
// skipped unless the two are on opposite sides of a cut, before its state
// is read; a particle without labels is on no side, so such candidates of it
// are skipped unread, and a list of nothing else (NBR_SHARED) is not walked.
__global__ void k_pair(World w, LaunchSet ls) {
  chain_wait();
  const int4 bt = ls.btiles[blockIdx.x];
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (!sc.pair_on || sc.frozen) return;
  const PPool &P = w.P;
  const int rb = (int)(sc.step & 1), wb = rb ^ 1;
  const float dt = sc.dt, R2 = 2.0f * sc.Rp;
  const float meff = sc.mp * sc.mp / (sc.mp + sc.mp);
  bool over = false;
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < bt.w; i += blockDim.x * gridDim.y) {
    const int p = bt.z + i;
    const float xp[3] = {P.x[0][p], P.x[1][p], P.x[2][p]};
    const float vp[3] = {P.v[0][p], P.v[1][p], P.v[2][p]};
    const uint32_t a1 = P.s1[p], a2 = P.s2[p];
    float J[3] = {0.f, 0.f, 0.f};
    int cnt = 0;
    const int nn8 = P.nbr_n[p];
    const bool uncut = (a1 | a2) == 0u;
    const int n = uncut && (nn8 & NBR_SHARED) ? 0 : nn8 & (NBR_SHARED - 1);
    const int *lst = P.nbr + (size_t)p * BM_NBR;
    for (int k = 0; k < n; ++k) {
      const int ent = lst[k];
      const int q = ent & 0x7fffffff;
      if (ent < 0 && (uncut || !conflict(a1, a2, P.s1[q], P.s2[q]))) continue;  // self-contact exclusion
      const float xq[3] = {P.x[0][q], P.x[1][q], P.x[2][q]};
      const float vq[3] = {P.v[0][q], P.v[1][q], P.v[2][q]};
      const bool plo = p < q;
      const int lo = plo ? p : q, hi = plo ? q : p;
      const float *xl = plo ? xp : xq, *xh = plo ? xq : xp;
      const float *vl = plo ? vp : vq, *vh = plo ? vq : vp;
      const float d[3] = {xl[0] - xh[0], xl[1] - xh[1], xl[2] - xh[2]};
      const float dist = sqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
      if (!(dist > 0.f)) continue;
      const float id = 1.0f / dist;
      const float nn[3] = {d[0] * id, d[1] * id, d[2] * id};
      const float vr[3] = {vl[0] - vh[0], vl[1] - vh[1], vl[2] - vh[2]};
      const float vn = vr[0] * nn[0] + vr[1] * nn[1] + vr[2] * nn[2];
      const float dhat = R2 - (dist + fminf(dt * vn, 0.0f));  // Eq. 10
      if (!(dhat > 0.f)) continue;
      const float fn = sc.s_n * meff / (dt * dt) * dhat;  // Eq. 11
      float uh[3] = {0.f, 0.f, 0.f};
      for (int h = 0; h < BM_HIST; ++h) {
        const int pt = P.hist_partner[rb][(size_t)lo * BM_HIST + h];
        if (pt < 0) break;
        if (pt == hi) {
          const float *u = P.hist_u[rb] + ((size_t)lo * BM_HIST + h) * 3;
          uh[0] = u[0];
          uh[1] = u[1];
          uh[2] = u[2];
          break;
        }
      }
      float ft[3], un[3];
      friction(uh, nn, vr, fn, meff, dt, sc.gamma_k, sc.gamma_c, sc.pair_mu_s, sc.pair_mu_d, ft, un);
      const float Jv[3] = {dt * (fn * nn[0] + ft[0]), dt * (fn * nn[1] + ft[1]), dt * (fn * nn[2] + ft[2])};
      if (plo) {  // Eq. 13: +J on the lower index, -J on the higher
        J[0] += Jv[0];
        J[1] += Jv[1];
        J[2] += Jv[2];
        if (cnt < BM_HIST) {
          P.hist_partner[wb][(size_t)p * BM_HIST + cnt] = hi;
          float *u = P.hist_u[wb] + ((size_t)p * BM_HIST + cnt) * 3;
          u[0] = un[0];
          u[1] = un[1];
          u[2] = un[2];
          ++cnt;
        } else {
          over = true;
        }
      } else {
        J[0] -= Jv[0];
        J[1] -= Jv[1];
        J[2] -= Jv[2];
      }
    }
    if (cnt < BM_HIST) P.hist_partner[wb][(size_t)p * BM_HIST + cnt] = -1;
    P.J[0][p] = J[0];
    P.J[1][p] = J[1];
    P.J[2][p] = J[2];
  }
  if (over) atomicOr(&scm.err, BM_ERRBIT_CONTACT_OVERFLOW);
}

// --------------------------------------------------------------------------
// frames outside a substep (float64, a thread per scene): of the scenes as
// they are, and after a tool state was set.  prepare_substep_warp (bm_tool.cuh)
// in the same operations, so that setting a tool to the state it is in changes
// no bit; with the warp form here too, k_musl_node, which carries the tool step,
// is compiled to a slower kernel (14.5 -> 16.2 us for a 477,000-particle scene).
// --------------------------------------------------------------------------
__device__ void matvec_rn(const double M[9], const double x[3], double y[3]) {
  for (int i = 0; i < 3; ++i)
    y[i] = __dadd_rn(__dadd_rn(__dmul_rn(M[3 * i], x[0]), __dmul_rn(M[3 * i + 1], x[1])),
                     __dmul_rn(M[3 * i + 2], x[2]));
}

__device__ void matmul_d(const double A[9], const double B[9], double C[9]) {
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      C[3 * i + j] = A[3 * i] * B[j] + A[3 * i + 1] * B[3 + j] + A[3 * i + 2] * B[6 + j];
}

__device__ void world_inv_inertia(const DevScene &sc, double Iw[9]) {
  double RT[9], tmp[9];
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) RT[3 * i + j] = sc.R[3 * j + i];
  matmul_d(sc.R, sc.Ib_inv, tmp);
  matmul_d(tmp, RT, Iw);
}

// Sets up substep sc.step: prescribed twist, cut, D reset, blade frame.
__device__ void prepare_substep(DevScene &sc) {
  if (!sc.has_blade) {
    sc.cut = -1;
    sc.reset_D = 0;
    return;
  }
  const DevSeg *sg = seg_at(sc, sc.step);
  const int cut = sg ? sg->cut_id : -1;
  const bool dynamic = sc.mass > 0.0;
  if (!dynamic && sg)
    for (int i = 0; i < 3; ++i) {
      sc.vB[i] = sg->v[i];
      sc.wB[i] = sg->w[i];
    }
  sc.cut = cut;
  sc.reset_D = (cut >= 0 && cut != sc.cur_cut) ? 1 : 0;
  double t[3];
  matvec_rn(sc.R, sc.edgeT, t);
  for (int i = 0; i < 3; ++i) sc.dxe[i] = __dadd_rn(sc.xB[i], t[i]);
  matvec_rn(sc.R, sc.nT, sc.dn);
  matvec_rn(sc.R, sc.eT, sc.de);
  matvec_rn(sc.R, sc.dT, sc.dd);
  double r[3] = {__dsub_rn(sc.dxe[0], sc.xB[0]), __dsub_rn(sc.dxe[1], sc.xB[1]),
                 __dsub_rn(sc.dxe[2], sc.xB[2])};
  double wr[3] = {__dsub_rn(__dmul_rn(sc.wB[1], r[2]), __dmul_rn(sc.wB[2], r[1])),
                  __dsub_rn(__dmul_rn(sc.wB[2], r[0]), __dmul_rn(sc.wB[0], r[2])),
                  __dsub_rn(__dmul_rn(sc.wB[0], r[1]), __dmul_rn(sc.wB[1], r[0]))};
  for (int i = 0; i < 3; ++i) sc.dve[i] = __dadd_rn(sc.vB[i], wr[i]);
  if (sc.reset_D) {  // a new cut begins: keep its plane for the cut faces
    for (int i = 0; i < 3; ++i) sc.cutpl[cut][i] = sc.dn[i];
    sc.cutpl[cut][3] = __dadd_rn(__dadd_rn(__dmul_rn(sc.dn[0], sc.dxe[0]), __dmul_rn(sc.dn[1], sc.dxe[1])),
                                 __dmul_rn(sc.dn[2], sc.dxe[2]));
    sc.cutpl_set |= 1u << cut;
  }
  for (int i = 0; i < 3; ++i) {
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
  sc.fhext[0] = (float)sc.half_thick;
  sc.fhext[1] = (float)sc.half_len;
  sc.fhext[2] = (float)sc.half_height;
  sc.fL = (float)sc.L_d;
  sc.fmu_s = (float)sc.mu_s;
  sc.fmu_d = (float)sc.mu_d;
  if (dynamic) {
    double Iw[9];
    world_inv_inertia(sc, Iw);
    for (int k = 0; k < 9; ++k) sc.fIinv[k] = (float)Iw[k];
    sc.finv_mass = (float)(1.0 / sc.mass);
  } else {
    for (int k = 0; k < 9; ++k) sc.fIinv[k] = 0.f;
    sc.finv_mass = 0.f;
  }
}

__global__ void k_prepare(World w, LaunchSet ls) {
  chain_wait();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= ls.n_scenes) return;
  prepare_substep(w.scenes[ls.scene_ids[idx]]);
}

// tool states {x_B, R, v_B, omega_B} of several scenes, then their frames
__global__ void k_set_tools(World w, const int *ids, int n, const double *states) {
  chain_wait();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  DevScene &sc = w.scenes[ids[idx]];
  const double *q = states + (size_t)idx * 18;
  for (int k = 0; k < 3; ++k) sc.xB[k] = q[k];
  for (int k = 0; k < 9; ++k) sc.R[k] = q[3 + k];
  for (int k = 0; k < 3; ++k) {
    sc.vB[k] = q[12 + k];
    sc.wB[k] = q[15 + k];
  }
  prepare_substep(sc);
}

__global__ void k_get_wrenches(World w, const int *ids, int n, double *out) {
  chain_wait();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n) return;
  const DevScene &sc = w.scenes[ids[idx]];
  for (int k = 0; k < 6; ++k) out[(size_t)idx * 6 + k] = sc.lastW[k];
}

// --------------------------------------------------------------------------
// logical-grid slot table (rebuilt after label changes)
// --------------------------------------------------------------------------


// Recount of the distinct codes at one node, by one warp: lane l < 27 holds
// base cell (i - l % 3, j - l / 3 % 3, k - l / 9) of the node's stencil, and
// the node's codes are found in ascending order of the key (mask2 << 32 |
// mask1) as repeated warp-wide minima over the lanes' particles of the keys
// above the last one found.  Returns the count.
// KR: particles per cell whose label keys a lane keeps in registers across
// the passes (8 or 16, the launch set's largest cell)
template <int KR>
__device__ __forceinline__ int recount_node(const World &w, DevScene &sc, int nd, int lane) {
  const int *cs = w.N.cell_start + sc.cell_begin;
  int ix, iy, iz;
  node_coords(sc, nd - sc.node_begin, ix, iy, iz);
  int p0 = 0, p1 = 0;
  if (lane < 27) {
    const int bx = ix - lane % 3, by = iy - (lane / 3) % 3, bz = iz - lane / 9;
    if (bx >= 0 && by >= 0 && bz >= 0 && bx < sc.nb[0] && by < sc.nb[1] && bz < sc.nb[2]) {
      const int c = cell_index(sc, bx, by, bz);
      p0 = cs[c];
      p1 = cs[c + 1];
    }
  }
  int cnt = 0;
  bool over = false;
  unsigned long long last = 0;
  bool first = true;
  // a cell of up to KR particles keeps its keys in registers across the
  // passes (the all-ones key is never a code: a cut has one side per particle)
  const bool inreg = p1 - p0 <= KR;
  unsigned long long kr[KR];
#pragma unroll
  for (int j = 0; j < KR; ++j)
    kr[j] = (inreg && p0 + j < p1) ? ((unsigned long long)w.P.s2[p0 + j] << 32) | w.P.s1[p0 + j] : ~0ull;
  for (;;) {
    unsigned long long m = ~0ull;
    if (inreg) {
#pragma unroll
      for (int j = 0; j < KR; ++j)
        if ((first || kr[j] > last) && kr[j] < m) m = kr[j];
    } else {
      for (int p = p0; p < p1; ++p) {
        const unsigned long long k = ((unsigned long long)w.P.s2[p] << 32) | w.P.s1[p];
        if ((first || k > last) && k < m) m = k;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(FULL, m, o);
      m = y < m ? y : m;
    }
    if (m == ~0ull) break;
    if (cnt < BM_MAXS) {
      if (lane == 0) w.N.tmp_codes[(size_t)nd * BM_MAXS + cnt] = make_uint2((uint32_t)m, (uint32_t)(m >> 32));
      ++cnt;
    } else {
      over = true;
      break;
    }
    last = m;
    first = false;
  }
  if (lane == 0) {
    if (over) atomicOr(&sc.err, BM_ERRBIT_SLOT_OVERFLOW);
    w.N.ncodes[nd] = (uint8_t)cnt;
    w.N.dirty[nd] = 0;
  }
  return cnt;
}

// Recount of a tile's dirty nodes (all of them when forced) by the warps of
// gridDim.y CTAs, ahead of k_slot_count<.., true>.
template <int KR>
__global__ void k_recount(World w, LaunchSet ls, int force) {
  chain_wait();
  const int4 t = ls.ntiles[blockIdx.x];
  DevScene &sc = w.scenes[t.x];
  if (!force && !sc.label_pending) return;
  const int lane = threadIdx.x & 31;
  const int warp = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5), nw = gridDim.y * (blockDim.x >> 5);
  for (int li = warp; li < t.z; li += nw)
    if (force || w.N.dirty[t.y + li]) recount_node<KR>(w, sc, t.y + li, lane);
}

// Slot counts of a node tile's nodes and their sum.
__device__ __forceinline__ void count_tile(const World &w, const int4 &t, int *sm) {
  const int i = threadIdx.x;
  int cnt = 0;
  if (i < t.z) {
    cnt = w.N.ncodes[t.y + i];
    w.N.slot_cnt[t.y + i] = (uint8_t)cnt;
  }
  int total;
  block_excl_scan(cnt, sm, total);
  if (i == 0) w.N.tile_sum[t.w] = total;
}

// The same with the nodes next to a newly labelled particle (dirty) recounted
// first, a warp each; the others keep their distinct codes from the last
// rebuild.
template <int KR>
__global__ void k_slot_count(World w, LaunchSet ls, int force) {
  chain_wait();
  const int4 t = ls.ntiles[blockIdx.x];
  DevScene &sc = w.scenes[t.x];
  if (!force && !sc.label_pending) return;
  __shared__ int sm[33];
  __shared__ int dlist[512];   // node tile <= 512 nodes
  __shared__ int ndirty;
  const int i = threadIdx.x;
  if (i == 0) ndirty = 0;
  __syncthreads();
  if (i < t.z && (force != 0 || w.N.dirty[t.y + i] != 0)) dlist[atomicAdd(&ndirty, 1)] = i;
  __syncthreads();
  const int lane = i & 31, wid = i >> 5, nw = blockDim.x >> 5;
  for (int j = wid; j < ndirty; j += nw) recount_node<KR>(w, sc, t.y + dlist[j], lane);
  __syncthreads();
  count_tile(w, t, sm);
}

// per brick: slot count and first tile slot of each tile node, and the
// tile's slot total (after the per-node counts are final)
// (one warp per brick: lane l takes the tile's nodes 7l .. 7l + 6, an
// exclusive warp scan orders them)
#define BTILE_WARPS 8  // bricks per CTA of k_brick_tiles

// Distinct codes of a brick's particles and each particle's index in
// the list (one warp; a lane keeps the codes of its particles lane + 32 j in
// registers).  The next code is that of the lowest particle not yet listed,
// so the list is in first-occurrence order.
// (PER: 32 PER particles at most)
template <int PER>
__device__ __forceinline__ int list_brick_codes(const World &w, DevScene &sc, const int4 &bt, int lane) {
  uint32_t a[PER], b[PER];
  unsigned todo = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = lane + 32 * j;
    a[j] = b[j] = 0;
    if (i < bt.w) {
      a[j] = w.P.s1[bt.z + i];
      b[j] = w.P.s2[bt.z + i];
      todo |= 1u << j;
    }
  }
  int n = 0;
  for (;;) {
    const int first = todo ? lane + 32 * (__ffs(todo) - 1) : INT_MAX;
    const int lead = __reduce_min_sync(FULL, first);
    if (lead == INT_MAX) break;
    if (n == BM_BRICK_CODES) {
      if (lane == 0) atomicOr(&sc.err, BM_ERRBIT_SLOT_OVERFLOW);
#pragma unroll
      for (int j = 0; j < PER; ++j)
        if ((todo >> j) & 1u) w.P.cid[bt.z + lane + 32 * j] = 0xff;
      break;
    }
    const uint32_t ka = w.P.s1[bt.z + lead], kb = w.P.s2[bt.z + lead];
    if (lane == 0) w.B.bcode[(size_t)bt.y * BM_BRICK_CODES + n] = make_uint2(ka, kb);
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (((todo >> j) & 1u) && a[j] == ka && b[j] == kb) {
        w.P.cid[bt.z + lane + 32 * j] = (uint8_t)n;
        todo &= ~(1u << j);
      }
    ++n;
  }
  return n;
}

template <int PPC>
__device__ __forceinline__ void brick_tile_slots(const World &w, const LaunchSet &ls, int bi, int lane, int force) {
  if (bi >= ls.n_btiles) return;
  const int4 bt = ls.btiles[bi];
  DevScene &sc = w.scenes[bt.x];
  if (!force && !sc.label_pending) return;
  int ncode;
  if (force || w.B.bdirty[bt.y]) {
    ncode = list_brick_codes<PPC * BR3 / 32>(w, sc, bt, lane);
    if (lane == 0) w.B.bdirty[bt.y] = 0;
  } else {
    ncode = w.B.binfo[bt.y] & 0xff;
  }
  int c0x, c0y, c0z;
  brick_coords(sc, bt.y - sc.brick_begin, c0x, c0y, c0z);
  constexpr int PER = (TN + 31) / 32;  // 7
  int cnt[PER];
  int mine = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int t = lane * PER + j;
    cnt[j] = 0;
    if (t < TN) {
      const int nx = c0x + t % TE, ny = c0y + (t / TE) % TE, nz = c0z + t / (TE * TE);
      if (nx < sc.nn[0] && ny < sc.nn[1] && nz < sc.nn[2])
        cnt[j] = w.N.ncodes[sc.node_begin + (nz * sc.nn[1] + ny) * sc.nn[0] + nx];
    }
    mine += cnt[j];
  }
  bool several = false;
#pragma unroll
  for (int j = 0; j < PER; ++j) several |= cnt[j] > 1;
  const bool single = !__any_sync(FULL, several);
  if (lane == 0) w.B.binfo[bt.y] = ncode | (single ? 256 : 0);
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += y;
  }
  int ex = incl - mine;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int t = lane * PER + j;
    if (t < TN) w.B.tdesc[(size_t)bt.y * TN + t] = ex | (cnt[j] << 16);
    ex += cnt[j];
  }
  if (lane == 31) w.B.ptot[bt.y] = incl;
}

// Exclusive sums of v[0..n) by one CTA, each thread a run of consecutive
// values, so that the CTA scans once however many there are: `out(j, sum
// before j, v[j])`.  Returns the total.  (In steps of a value per thread, two
// barriers each, a 477,000-particle scene's 1,000 bricks kept k_slot_fill at 12 us.)
template <class Out>
__device__ __forceinline__ int cta_offsets(const int *v, int n, int *sm, Out out) {
  const int per = (n + blockDim.x - 1) / blockDim.x;
  const int j0 = threadIdx.x * per, j1 = min(j0 + per, n);
  int mine = 0;
#pragma unroll 4
  for (int j = j0; j < j1; ++j) mine += v[j];
  int total;
  int before = block_excl_scan(mine, sm, total);
  for (int j = j0; j < j1; ++j) {
    const int q = v[j];
    out(j, before, q);
    before += q;
  }
  return total;
}

// slot offsets of a scene's node tiles (one CTA): exclusive sums in place
__device__ __forceinline__ void tile_offsets(const World &w, DevScene &sc, int *sm) {
  int *ts = w.N.tile_sum + sc.ntile_begin;
  const int total = cta_offsets(ts, sc.n_ntile, sm, [&](int j, int before, int) { ts[j] = before; });
  if (threadIdx.x == 0) {
    sc.n_slots = total;
    if (total > sc.slot_cap) atomicOr(&sc.err, BM_ERRBIT_SLOT_OVERFLOW);
  }
}

// partial-sum ranges of a scene's bricks (one CTA)
__device__ __forceinline__ void brick_ranges(const World &w, DevScene &sc, int *sm) {
  bool pover = false;
  cta_offsets(w.B.ptot + sc.brick_begin, sc.n_brick, sm, [&](int j, int before, int v) {
    const bool fits = before + v <= sc.ppool_cap;
    w.B.poff[sc.brick_begin + j] = fits ? sc.ppool_begin + before : -1;
    pover |= !fits;
  });
  if (pover) atomicOr(&sc.err, BM_ERRBIT_SLOT_OVERFLOW);
}

// Sums over a scene stand between the counts and the slots: a CTA per scene
// takes them beside the work that does not wait for them, the tiles' in the
// launch of the bricks' tiles, the bricks' in that of the slots.  (A launch of
// its own for both was 3 us of a 16,000-particle scene, 8 of the 256-scene
// batch and 10 of a 477,000-particle scene.)
template <int PPC>
__global__ void __launch_bounds__(32 * BTILE_WARPS) k_brick_tiles(World w, LaunchSet ls, int force) {
  chain_wait();
  if ((int)blockIdx.x < ls.n_scenes) {
    __shared__ int sm[33];
    DevScene &sc = w.scenes[ls.scene_ids[blockIdx.x]];
    if (force || sc.label_pending) tile_offsets(w, sc, sm);
    return;
  }
  brick_tile_slots<PPC>(w, ls, (blockIdx.x - ls.n_scenes) * BTILE_WARPS + (threadIdx.x >> 5), threadIdx.x & 31,
                        force);
}

// After k_recount: the counts of the node tiles and, in further CTAs, the
// tiles of the bricks, which wait for the nodes' codes alone.
template <int PPC>
__global__ void __launch_bounds__(512) k_count_tiles(World w, LaunchSet ls, int force) {
  chain_wait();
  if ((int)blockIdx.x < ls.n_ntiles) {
    __shared__ int sm[33];
    const int4 t = ls.ntiles[blockIdx.x];
    if (force || w.scenes[t.x].label_pending) count_tile(w, t, sm);
    return;
  }
  brick_tile_slots<PPC>(w, ls, (blockIdx.x - ls.n_ntiles) * (blockDim.x >> 5) + (threadIdx.x >> 5),
                        threadIdx.x & 31, force);
}

// Slots of the nodes, and in the first n_scenes CTAs the bricks' partial-sum
// ranges and the commit of the tool step (not when forced: no substep).
// OFFSETS: tile_sum holds the tiles' slot offsets (tile_offsets), otherwise
// their counts, which each CTA sums up to its own tile.
template <bool OFFSETS>
__global__ void k_slot_fill(World w, LaunchSet ls, int force) {
  chain_wait();
  __shared__ int sm[33];
  if ((int)blockIdx.x < ls.n_scenes) {
    const int sid = ls.scene_ids[blockIdx.x];
    DevScene &sc = w.scenes[sid];
    if (force || sc.label_pending) brick_ranges(w, sc, sm);
    if (!force) commit_tool(w, sid);
    return;
  }
  const int4 t = ls.ntiles[blockIdx.x - ls.n_scenes];
  DevScene &sc = w.scenes[t.x];
  if (!force && !sc.label_pending) return;
  const int i = threadIdx.x;
  const int node = t.y + i;
  const int cnt = i < t.z ? (int)w.N.slot_cnt[node] : 0;
  int total;
  const int ex = block_excl_scan(cnt, sm, total);
  int tile0;
  if (OFFSETS) {
    tile0 = w.N.tile_sum[t.w];
  } else {
    int before = 0;
    for (int j = sc.ntile_begin + i; j < t.w; j += blockDim.x) before += w.N.tile_sum[j];
    __syncthreads();
    block_excl_scan(before, sm, tile0);
    if (t.w == sc.ntile_begin + sc.n_ntile - 1 && i == 0) {
      sc.n_slots = tile0 + total;
      if (tile0 + total > sc.slot_cap) atomicOr(&sc.err, BM_ERRBIT_SLOT_OVERFLOW);
    }
  }
  if (i < t.z) {
    int off = tile0 + ex;
    const bool fits = off + cnt <= sc.slot_cap;
    if (!fits) {
      w.N.slot_cnt[node] = 0;
      off = 0;
    } else {
      for (int a = 0; a < cnt; ++a)
        w.S.code[sc.slot_begin + off + a] = w.N.tmp_codes[(size_t)node * BM_MAXS + a];
    }
    w.N.slot_off[node] = sc.slot_begin + off;
    // the node's first slot in the tile table of every brick whose tile covers it
    int ix, iy, iz, x0, x1, y0, y1, z0, z1;
    node_coords(sc, node - sc.node_begin, ix, iy, iz);
    covering(ix, sc.nbr[0], x0, x1);
    covering(iy, sc.nbr[1], y0, y1);
    covering(iz, sc.nbr[2], z0, z1);
    for (int Bz = z0; Bz <= z1; ++Bz)
      for (int By = y0; By <= y1; ++By)
        for (int Bx = x0; Bx <= x1; ++Bx) {
          const int b = sc.brick_begin + (Bz * sc.nbr[1] + By) * sc.nbr[0] + Bx;
          const int tt = ((iz - Bz * BR) * TE + (iy - By * BR)) * TE + (ix - Bx * BR);
          w.B.tgoff[(size_t)b * TN + tt] = sc.slot_begin + off;
        }
  }
}

// --------------------------------------------------------------------------
// state I/O between pool order and the caller's order
// --------------------------------------------------------------------------
__device__ __forceinline__ void io_field(const World &w, int scene_slot, int p, int o, int field, void *buf,
                                         int to_pool) {
  const PPool &P = w.P;
  float *fb = (float *)buf;
  uint32_t *ub = (uint32_t *)buf;
  switch (field) {
    case 0:  // X (from fx and base cannot reproduce X exactly: kept separately)
      break;
    case 1:
      for (int a = 0; a < 3; ++a) {
        if (to_pool) P.x[a][p] = fb[3 * o + a];
        else fb[3 * o + a] = P.x[a][p];
      }
      break;
    case 2:
      for (int a = 0; a < 3; ++a) {
        if (to_pool) P.v[a][p] = fb[3 * o + a];
        else fb[3 * o + a] = P.v[a][p];
      }
      break;
    case 3:
      for (int a = 0; a < 9; ++a) {
        if (to_pool) P.F[a][p] = fb[9 * o + a];
        else fb[9 * o + a] = P.F[a][p];
      }
      break;
    case 4:
      if (to_pool) {
        P.D[p] = fb[o];
        P.tflag[p] = 1;  // may be nonzero: the next P2G reads it
      } else {
        fb[o] = P.D[p];
      }
      break;
    case 5:
      for (int a = 0; a < 3; ++a) {
        if (to_pool) P.ut[a][p] = fb[3 * o + a];
        else fb[3 * o + a] = P.ut[a][p];
      }
      if (to_pool) P.tflag[p] = 1;
      break;
    case 7:
      if (to_pool) P.s1[p] = ub[o];
      else ub[o] = P.s1[p];
      break;
    case 8:
      if (to_pool) P.s2[p] = ub[o];
      else ub[o] = P.s2[p];
      break;
    case 9:    // pair history partners (read only): caller indices, -1 ends the list
    case 10: {  // pair history spring displacements (read only)
      if (to_pool || !P.hist_partner[0]) break;
      const int rb = (int)(w.scenes[scene_slot].step & 1);  // the buffer the next substep reads
      bool live = true;
      for (int h = 0; h < BM_HIST; ++h) {
        const int pt = live ? P.hist_partner[rb][(size_t)p * BM_HIST + h] : -1;
        live = pt >= 0;
        if (field == 9) {
          ((int *)buf)[(size_t)o * BM_HIST + h] = live ? P.perm[pt] : -1;
        } else {
          const float *u = P.hist_u[rb] + ((size_t)p * BM_HIST + h) * 3;
          for (int a = 0; a < 3; ++a) fb[((size_t)o * BM_HIST + h) * 3 + a] = live ? u[a] : 0.0f;
        }
      }
      break;
    }
  }
}

__global__ void k_io(World w, int scene_slot, int p_begin, int n, int field, void *buf, int to_pool) {
  chain_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int p = p_begin + i;
  io_field(w, scene_slot, p, w.P.perm[p], field, buf, to_pool);
}

struct ReadSet {
  void *buf[BM_NUM_FIELDS];
  int field[BM_NUM_FIELDS];
};

// blockIdx.y: which of the requested fields
__global__ void k_read(World w, int scene_slot, int p_begin, int n, ReadSet r) {
  chain_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int p = p_begin + i;
  io_field(w, scene_slot, p, w.P.perm[p], r.field[blockIdx.y], r.buf[blockIdx.y], 0);
}

__global__ void k_code(World w, int p_begin, int n, int64_t *out) {
  chain_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int p = p_begin + i;
  const uint32_t a = w.P.s1[p], b = w.P.s2[p];
  int64_t c = 0, pw = 1;
  for (int k = 0; k < BM_MAX_CUTS; ++k) {
    const int d = ((a >> k) & 1u) ? 1 : (((b >> k) & 1u) ? 2 : 0);
    c += d * pw;
    pw *= 3;
  }
  out[w.P.perm[p]] = c;
}

}  // namespace

// ----------------------------------------------------------------------------
// launchers
// ----------------------------------------------------------------------------
cudaError_t bm_launch_prepare(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.n_scenes == 0) return cudaSuccess;
  chain_launch(k_prepare, dim3((unsigned)((ls.n_scenes + 63) / 64)), 64, 0, st, w, ls);
  return cudaGetLastError();
}

// k_tool and k_slot_scan have no launch (k_musl_node, k_brick_tiles and
// k_slot_fill do their work) and so no time of their own
const char *const bm_kernel_names[BM_NUM_KERNELS] = {
    "k_p2g_brick", "k_p2g_node", "k_g2p_musl", "k_musl_node", "k_fupd",
    "k_tool", "k_slot_count", "k_slot_scan", "k_slot_fill", "k_brick_tiles",
    "k_pair_clear", "k_pair_hash", "k_scan_local", "k_scan_top", "k_scan_add", "k_pair_fill",
    "k_pair_sort", "k_pair", "k_pair_list"};

// ev (optional): 2 * BM_NUM_KERNELS events recorded around each launch
static inline void rec(cudaEvent_t *ev, int k, int after, cudaStream_t st) {
  if (ev) cudaEventRecord(ev[2 * k + after], st);
}

// New labels fall on a few node tiles.  While the tiles are too few to fill
// the chip, their dirty nodes are shared out over several CTAs per tile in a
// launch of their own; beyond that (four CTAs on each of 152 SMs) a tile's own
// CTA recounts them.  16,000-particle scene 15.7 us in one launch -> 5 in two; 3,887 nodes
// all recounted after a restore 24 -> 7 us; the 256-scene batch takes 47 us
// in one launch.
#define RECOUNT_CTAS (4 * 152)
template <int PPC>
static void launch_slots(const World &w, const LaunchSet &ls, cudaStream_t st, int force, cudaEvent_t *ev) {
  rec(ev, 6, 0, st);
  if (ls.n_ntiles > RECOUNT_CTAS) {
    chain_launch(k_slot_count<PPC>, dim3(ls.n_ntiles), ls.ntile_size, 0, st, w, ls, force);
    rec(ev, 6, 1, st);
    rec(ev, 9, 0, st);
    const int tgrid = (ls.n_btiles + BTILE_WARPS - 1) / BTILE_WARPS;
    chain_launch(k_brick_tiles<PPC>, dim3(ls.n_scenes + tgrid), 32 * BTILE_WARPS, 0, st, w, ls, force);
    rec(ev, 9, 1, st);
    rec(ev, 8, 0, st);
    chain_launch(k_slot_fill<true>, dim3(ls.n_scenes + ls.n_ntiles), ls.ntile_size, 0, st, w, ls, force);
  } else {
    const int parts = min(max(RECOUNT_CTAS / ls.n_ntiles, 1), 16), nw = ls.ntile_size / 32;
    chain_launch(k_recount<PPC>, dim3((unsigned)ls.n_ntiles, (unsigned)parts), 256, 0, st, w, ls, force);
    chain_launch(k_count_tiles<PPC>, dim3(ls.n_ntiles + (ls.n_btiles + nw - 1) / nw), ls.ntile_size, 0, st, w, ls,
                 force);
    rec(ev, 6, 1, st);
    rec(ev, 8, 0, st);
    chain_launch(k_slot_fill<false>, dim3(ls.n_scenes + ls.n_ntiles), ls.ntile_size, 0, st, w, ls, force);
  }
  rec(ev, 8, 1, st);
}
static cudaError_t launch_rebuild(const World &w, const LaunchSet &ls, cudaStream_t st, int force,
                                  cudaEvent_t *ev) {
  if (ls.n_ntiles == 0) return cudaSuccess;
  if (ls.ppc16) launch_slots<16>(w, ls, st, force, ev);
  else launch_slots<8>(w, ls, st, force, ev);
  return cudaGetLastError();
}

cudaError_t bm_launch_rebuild(const World &w, const LaunchSet &ls, cudaStream_t st, int force) {
  return launch_rebuild(w, ls, st, force, nullptr);
}

// Brick-kernel occupancy: the minimum resident CTAs per SM each brick kernel
// is compiled for (launch bounds), chosen per kernel (fewer CTAs leave more
// registers per thread, more CTAs hide more latency).  A launch variant v in [0, 27) picks choice
// v % 3 for k_p2g_brick, (v / 3) % 3 for k_g2p_musl and v / 9 for k_fupd;
// choice 0 is each kernel's default.  The arithmetic is the same in every
// variant, so results are bit-identical; the batch autotuner picks one.
template <int C, bool INELASTIC> struct OccP2G;
template <> struct OccP2G<0, false> { static constexpr int v = 4; };
template <> struct OccP2G<1, false> { static constexpr int v = 3; };
template <> struct OccP2G<2, false> { static constexpr int v = 2; };
template <> struct OccP2G<0, true> { static constexpr int v = 3; };  // the inelastic stress needs the registers
template <> struct OccP2G<1, true> { static constexpr int v = 2; };
template <> struct OccP2G<2, true> { static constexpr int v = 4; };
template <int C> struct OccG2P;
template <> struct OccG2P<0> { static constexpr int v = 5; };
template <> struct OccG2P<1> { static constexpr int v = 4; };
template <> struct OccG2P<2> { static constexpr int v = 6; };
template <int C> struct OccFupd;
template <> struct OccFupd<0> { static constexpr int v = 7; };
template <> struct OccFupd<1> { static constexpr int v = 5; };
template <> struct OccFupd<2> { static constexpr int v = 6; };

// dynamic shared memory of the brick kernels, and the largest shared-memory
// carveout, so that the CTAs per SM their launch bounds aim at fit
template <class K>
static cudaError_t brick_smem(K *kernel, int bytes) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
}

template <int PPC, int C>
static cudaError_t set_smem_attrs() {
  cudaError_t e = brick_smem(k_p2g_brick<PPC, OccP2G<C, false>::v, false, 1>, (int)sizeof(K2S<PPC, 1>));
  if (e == cudaSuccess) e = brick_smem(k_p2g_brick<PPC, OccP2G<C, true>::v, true, 1>, (int)sizeof(K2S<PPC, 1>));
  if (e == cudaSuccess) e = brick_smem(k_g2p_musl<PPC, OccG2P<C>::v, 1>, (int)sizeof(K4S<PPC, 1>));
  return e;
}

template <int PPC>
static cudaError_t set_wide_smem_attrs() {
  cudaError_t e = brick_smem(k_p2g_brick<PPC, 1, false, WIDE>, (int)sizeof(K2S<PPC, WIDE>));
  if (e == cudaSuccess) e = brick_smem(k_p2g_brick<PPC, 1, true, WIDE>, (int)sizeof(K2S<PPC, WIDE>));
  if (e == cudaSuccess) e = brick_smem(k_g2p_musl<PPC, 1, WIDE>, (int)sizeof(K4S<PPC, WIDE>));
  return e;
}

cudaError_t bm_kernels_init() {
  static cudaError_t status = cudaErrorNotReady;
  static int device = -1;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (device == dev && status == cudaSuccess) return status;
  if (e == cudaSuccess) e = set_smem_attrs<8, 0>();
  if (e == cudaSuccess) e = set_smem_attrs<8, 1>();
  if (e == cudaSuccess) e = set_smem_attrs<8, 2>();
  if (e == cudaSuccess) e = set_smem_attrs<16, 0>();
  if (e == cudaSuccess) e = set_smem_attrs<16, 1>();
  if (e == cudaSuccess) e = set_smem_attrs<16, 2>();
  if (e == cudaSuccess) e = set_wide_smem_attrs<8>();
  if (e == cudaSuccess) e = set_wide_smem_attrs<16>();
  if (e == cudaSuccess) e = bm_lattice_init();
  status = e;
  device = dev;
  return e;
}

template <int PPC, int MB, int G>
static void launch_p2g(const World &w, const LaunchSet &ls, cudaStream_t st) {
  chain_launch(k_p2g_brick<PPC, MB, false, G>, dim3(ls.n_btiles), BT * G, sizeof(K2S<PPC, G>), st, w, ls);
}
template <int PPC, int MB, int G>
static void launch_p2g_inelastic(const World &w, const LaunchSet &ls, cudaStream_t st) {
  chain_launch(k_p2g_brick<PPC, MB, true, G>, dim3(ls.n_btiles), BT * G, sizeof(K2S<PPC, G>), st, w, ls);
}

template <int PPC, int C>
static void launch_p2g(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.any_inelastic) launch_p2g_inelastic<PPC, OccP2G<C, true>::v, 1>(w, ls, st);
  else launch_p2g<PPC, OccP2G<C, false>::v, 1>(w, ls, st);
}

template <int PPC, int MB, int G>
static void launch_g2p(const World &w, const LaunchSet &ls, cudaStream_t st) {
  const int tools = ls.any_lattice ? 0 : g2p_tools(ls);  // the lattice form's if both run
  chain_launch(k_g2p_musl<PPC, MB, G>, dim3(tools + ls.n_btiles), BT * G, sizeof(K4S<PPC, G>), st, w, ls, tools);
}

template <int MB, int G>
static void launch_fupd(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.any_inelastic) chain_launch(k_fupd<MB, true, G>, dim3(ls.n_btiles), BT * G, 0, st, w, ls);
  else chain_launch(k_fupd<MB, false, G>, dim3(ls.n_btiles), BT * G, 0, st, w, ls);
}

// Whether the general kernels take their wide form (WIDE).  One wide CTA fills
// an SM, so its time is that of the waves of 152 bricks, some 20 us a substep
// each, hardly depending on a brick's particles; the narrow form holds 600
// bricks at once and takes a round for every 192 particles of a brick.  So a set
// of sparse bricks goes over to the narrow form earlier.  Substep, us, narrow /
// wide, bodies mid-cut of b bricks with p particles in a brick:
//   p  33: b 125  61 /  53, 175  60 /  61, 245  62 /  69
//   p 150: b 175  87 /  65, 245  86 /  75, 343  89 /  87, 392  92 /  93
//   p 320: b 245  98 /  75, 343 102 /  88, 512 109 / 109, 648 112 / 127
//   p 650: b 245 154 /  96, 392 165 / 124, 576 182 / 159, 729 203 / 194
// and sets of one-brick scenes, every brick cut:
//   p  64: b 100  73 /  71, 200  84 / 104, 600 122 / 201
//   p 216: b 100  88 /  72, 200 107 / 114, 300 113 / 122
//   p 512: b 200 122 / 115, 300 130 / 124, 400 147 / 164
// The kernels' CTAs of the set's lattice bricks leave at once, but a wide one
// holds the SM meanwhile, so beyond 608 bricks in all two waves are the limit
// and beyond 1,216 none: b jittered bricks of 16,000-particle scenes among n,
// narrow / wide: b 54 n 648 171 / 132, n 3,456 410 / 394, n 13,554 1,208 / 1,338;
// b 216 n 1,080 213 / 199, n 3,456 411 / 414; b 432 n 864 204 / 213.
static bool wide_general(const LaunchSet &ls) {
  const int most = ls.n_btiles <= 4 * 152 ? 4 : ls.n_btiles <= 8 * 152 ? 2 : 0;
  const int waves = 1 + ls.gen_particles / ls.gen_bricks / 128;
  return ls.gen_bricks <= 152 * (waves < most ? waves : most);
}

template <int PPC>
static void launch_p2g_general(const World &w, const LaunchSet &ls, cudaStream_t st) {
  const int c = ls.variant % 3;
  if (wide_general(ls)) {
    if (ls.any_inelastic) launch_p2g_inelastic<PPC, 1, WIDE>(w, ls, st);
    else launch_p2g<PPC, 1, WIDE>(w, ls, st);
  } else if (c == 0) launch_p2g<PPC, 0>(w, ls, st);
  else if (c == 1) launch_p2g<PPC, 1>(w, ls, st);
  else launch_p2g<PPC, 2>(w, ls, st);
}

template <int PPC>
static void launch_g2p_general(const World &w, const LaunchSet &ls, cudaStream_t st) {
  const int c = (ls.variant / 3) % 3;
  if (wide_general(ls)) launch_g2p<PPC, 1, WIDE>(w, ls, st);
  else if (c == 0) launch_g2p<PPC, OccG2P<0>::v, 1>(w, ls, st);
  else if (c == 1) launch_g2p<PPC, OccG2P<1>::v, 1>(w, ls, st);
  else launch_g2p<PPC, OccG2P<2>::v, 1>(w, ls, st);
}

static void launch_fupd_general(const World &w, const LaunchSet &ls, cudaStream_t st) {
  const int c = ls.variant / 9;
  if (wide_general(ls)) launch_fupd<1, WIDE>(w, ls, st);
  else if (c == 0) launch_fupd<OccFupd<0>::v, 1>(w, ls, st);
  else if (c == 1) launch_fupd<OccFupd<1>::v, 1>(w, ls, st);
  else launch_fupd<OccFupd<2>::v, 1>(w, ls, st);
}

// Threads of a node tile's CTA beyond its nodes, for sets of few tiles (sets of
// many are bound by the loads themselves: 256-scene batch, 16,000 tiles,
// 1,451 -> 1,592 us a substep).  k_p2g_node of a cut 16,000-particle scene 10.1 ->
// 6.2 us, k_musl_node 8.8 -> 6.2; a 477,000-particle scene of some 500 tiles
// 141 -> 139 us a substep.
#define NODE_TEAM_TILES (4 * 152)
#define NODE_TEAM 256
static int node_threads(const LaunchSet &ls) {
  return ls.ntile_size + (ls.n_ntiles <= NODE_TEAM_TILES ? NODE_TEAM : 0);
}

// Each brick kernel in its lattice and its general form, as the set's scenes
// need (each form returns at once for the other's scenes).
static void launch_bricks(const World &w, const LaunchSet &ls, cudaStream_t st, cudaEvent_t *ev) {
  rec(ev, 0, 0, st);
  if (ls.any_lattice) bm_launch_p2g_lat(w, ls, st);
  if (ls.any_general) {
    if (ls.ppc16) launch_p2g_general<16>(w, ls, st);
    else launch_p2g_general<8>(w, ls, st);
  }
  rec(ev, 0, 1, st);
  rec(ev, 1, 0, st);
  chain_launch(k_p2g_node, dim3(ls.n_ntiles), node_threads(ls), 0, st, w, ls);
  rec(ev, 1, 1, st);
  rec(ev, 2, 0, st);
  if (ls.any_lattice) bm_launch_g2p_lat(w, ls, st);
  if (ls.any_general) {
    if (ls.ppc16) launch_g2p_general<16>(w, ls, st);
    else launch_g2p_general<8>(w, ls, st);
  }
  rec(ev, 2, 1, st);
  rec(ev, 3, 0, st);
  const int tools = g2p_tools(ls) ? 0 : ls.n_scenes;
  chain_launch(k_musl_node, dim3(tools + ls.n_ntiles), node_threads(ls), 0, st, w, ls, tools);
  rec(ev, 3, 1, st);
  rec(ev, 4, 0, st);
  if (ls.any_lattice) bm_launch_fupd_lat(w, ls, st);
  if (ls.any_general) launch_fupd_general(w, ls, st);
  rec(ev, 4, 1, st);
}

static void launch_pairs(const World &w, const LaunchSet &ls, cudaStream_t st, cudaEvent_t *ev) {
  const int nb = w.H.n_buckets;
  const int nblk = (nb + 1023) / 1024;
  rec(ev, 10, 0, st);
  chain_launch(k_pair_reset, dim3((ls.n_scenes + 255) / 256), 256, 0, st, w, ls);
  chain_launch(k_pair_vmax, dim3(ls.n_btiles), BT, 0, st, w, ls);
  chain_launch(k_pair_decide, dim3((ls.n_scenes + 63) / 64), 64, 0, st, w, ls);
  cudaMemsetAsync(w.H.bucket_start, 0, sizeof(int) * ((size_t)nb + 1), st);
  cudaMemsetAsync(w.H.bucket_fill, 0, sizeof(int) * (size_t)nb, st);
  rec(ev, 10, 1, st);
  rec(ev, 11, 0, st);
  chain_launch(k_pair_hash, dim3(ls.n_btiles), BT, 0, st, w, ls);
  rec(ev, 11, 1, st);
  rec(ev, 12, 0, st);
  chain_launch(k_scan_local, dim3(nblk), 1024, 0, st, w);
  rec(ev, 12, 1, st);
  rec(ev, 13, 0, st);
  chain_launch(k_scan_top, dim3(1), 1024, 0, st, w, nblk);
  rec(ev, 13, 1, st);
  rec(ev, 14, 0, st);
  chain_launch(k_scan_add, dim3(nblk), 1024, 0, st, w);
  rec(ev, 14, 1, st);
  rec(ev, 15, 0, st);
  chain_launch(k_pair_fill, dim3(ls.n_btiles), BT, 0, st, w, ls);
  rec(ev, 15, 1, st);
  rec(ev, 16, 0, st);
  chain_launch(k_pair_sort, dim3((nb / 2 + 255) / 256), 256, 0, st, w);  // at least a thread per particle
  rec(ev, 16, 1, st);
  rec(ev, 18, 0, st);
  chain_launch(k_pair_list, dim3(152 * LIST_OCC), 32 * LIST_WARPS, 0, st, w);
  rec(ev, 18, 1, st);
  rec(ev, 17, 0, st);
  chain_launch(k_pair, dim3(ls.n_btiles, 4), 128, 0, st, w, ls);
  rec(ev, 17, 1, st);
}

cudaError_t bm_launch_substep_ev(const World &w, const LaunchSet &ls, cudaStream_t st, cudaEvent_t *ev) {
  if (ls.n_btiles == 0) return cudaSuccess;
  if (ls.any_pair && w.H.n_buckets > 0) launch_pairs(w, ls, st, ev);
  launch_bricks(w, ls, st, ev);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_rebuild(w, ls, st, 0, ev);
}

cudaError_t bm_launch_substep(const World &w, const LaunchSet &ls, cudaStream_t st) {
  return bm_launch_substep_ev(w, ls, st, nullptr);
}

cudaError_t bm_launch_io(const World &w, int scene_slot, int p_begin, int n, int field, void *buf,
                         int to_pool, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  chain_launch(k_io, dim3((unsigned)((n + 255) / 256)), 256, 0, st, w, scene_slot, p_begin, n, field, buf, to_pool);
  return cudaGetLastError();
}

cudaError_t bm_launch_read(const World &w, int scene_slot, int p_begin, int n, uint32_t mask, void *const *buf,
                           cudaStream_t st) {
  ReadSet r{};
  int k = 0;
  for (int f = 0; f < BM_NUM_FIELDS; ++f)
    if (mask & (1u << f)) {
      r.buf[k] = buf[f];
      r.field[k++] = f;
    }
  if (n == 0 || k == 0) return cudaSuccess;
  chain_launch(k_read, dim3((unsigned)(n + 255) / 256, (unsigned)k), 256, 0, st, w, scene_slot, p_begin, n, r);
  return cudaGetLastError();
}

cudaError_t bm_launch_set_tools(const World &w, const int *scene_ids, int n, const double *states,
                                cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  chain_launch(k_set_tools, dim3((unsigned)((n + 63) / 64)), 64, 0, st, w, scene_ids, n, states);
  return cudaGetLastError();
}

cudaError_t bm_launch_get_wrenches(const World &w, const int *scene_ids, int n, double *out,
                                   cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  chain_launch(k_get_wrenches, dim3((unsigned)((n + 63) / 64)), 64, 0, st, w, scene_ids, n, out);
  return cudaGetLastError();
}

cudaError_t bm_launch_code(const World &w, int p_begin, int n, int64_t *out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  chain_launch(k_code, dim3((unsigned)((n + 255) / 256)), 256, 0, st, w, p_begin, n, out);
  return cudaGetLastError();
}
