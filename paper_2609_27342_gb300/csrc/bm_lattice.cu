// Brick kernels for scenes whose particles sit on a lattice: P2G, G2P + MUSL
// and the F update, bit for bit the sums of the general kernels
// (bm_kernels.cu) with the work that lattice particles share done once.
//
// A scene takes this path when along each axis the particles of a base-cell
// layer lie on at most two planes, no two particles share a place, and a
// cell's particles are listed in (x, y, z) plane order (DevScene::lattice,
// decided once at creation); a jittered or scanned body, a cell of more than
// 2 x 2 x 2 particles or another order takes the general kernels.  A brick
// then has 8 x 8 x 8 places whose weights are those of 8 planes per axis:
//   * weights come from a table of 24 planes instead of being formed from
//     each particle's offsets by each of the threads that use them, and a
//     particle's 12 B of offsets and 8 B of codes are not read;
//   * the scatter (P2G, MUSL) gives a thread one cell and one z offset, as in
//     the general kernels, with the cell's 8 particles unrolled: 16-byte
//     reads of a particle's inputs, and two of its components (or its mass and
//     a component) in one instruction;
//   * the gather (G2P) gives a thread the two particles of one cell that
//     differ in z: each node's values are read once for both;
//   * the F update forms the sums along x once per (node row, x plane) and
//     not once per particle.
// The kernels are bound by instructions and shared-memory reads, not by DRAM
// (78, 47 and 57 B per particle).  Two other forms were measured and left:
// one axis at a time for the whole brick (7 multiply-adds per particle and
// value; P2G 0.39 ms) rounds differently, and an x-row of cells per thread
// (no shuffles, but 9 reads per particle; P2G 0.97 ms) is slower.
// Every sum keeps the general kernels' terms and order (a cell's particles,
// then the cells along x, y and z, nearest first).  That matters beyond
// tidiness: a position that rounds differently can decide a stick-slip or
// label threshold differently, so equal sums keep whole trajectories equal.
// Pairs of float32 operations are issued as one (fma.rn.f32x2 and the like),
// each half rounded as the scalar operation.
//
// Bricks with several codes run one pass per code of the brick (BPool::bcode,
// PPool::cid, kept up to date by the slot rebuild); empty places and other
// codes' particles are skipped.
#include "bm_device.cuh"
#include "bm_internal.cuh"
#include "bm_tool.cuh"

namespace {

constexpr int LP = BM_LAT_POS;     // particle places of a brick

// B-spline weights of one particle plane: w0 w1 w2 d0 | d1 d2
struct __align__(16) PlaneW {
  float4 a;
  float4 b;
};

__device__ __forceinline__ void plane_w(const PlaneW &p, float (&w)[3]) {
  const float4 a = p.a;
  w[0] = a.x;
  w[1] = a.y;
  w[2] = a.z;
}
__device__ __forceinline__ void plane_wd(const PlaneW &p, float (&w)[3], float (&d)[3]) {
  const float4 a = p.a;
  const float2 b = *reinterpret_cast<const float2 *>(&p.b);
  w[0] = a.x;
  w[1] = a.y;
  w[2] = a.z;
  d[0] = a.w;
  d[1] = b.x;
  d[2] = b.y;
}
// weight and derivative of node offset o (runtime)
__device__ __forceinline__ float plane_w1(const PlaneW &p, int o) { return o == 0 ? p.a.x : o == 1 ? p.a.y : p.a.z; }
__device__ __forceinline__ float plane_d1(const PlaneW &p, int o) { return o == 0 ? p.a.w : o == 1 ? p.b.x : p.b.y; }

// two float32 values in one register pair: one instruction, each half rounded
// as the scalar operation
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f2 r, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r)); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// force_u and force_acc (bm_device.cuh) of two components
__device__ __forceinline__ f2 force_u2(f2 A1, f2 dyz, f2 A2, f2 wyd, f2 J, f2 wyz) {
  return fma2(J, wyz, fma2(A1, dyz, mul2(A2, wyd)));
}
__device__ __forceinline__ f2 force_acc2(f2 q, f2 w, f2 U, f2 d, f2 V) { return add2(q, fma2(w, U, mul2(d, V))); }

// the brick's node tile and the weights of its planes
struct LatTile : BrickTile {
  PlaneW wt[3][8];
};

// Tile and weights of brick `brick` (nt threads); ends without a barrier.
__device__ __forceinline__ void lat_tile(const World &w, int brick, int nbc, LatTile &T, int nt) {
  brick_tile(w, brick, nbc, T, nt);
  const int tid = threadIdx.x;
  if (tid >= nt - 24) {
    const int k = tid - (nt - 24);
    const float f = w.B.lf[(size_t)brick * 24 + k];
    float a[3], d[3];
    bs<0>(f, a[0], d[0]);
    bs<1>(f, a[1], d[1]);
    bs<2>(f, a[2], d[2]);
    T.wt[k >> 3][k & 7].a = make_float4(a[0], a[1], a[2], d[0]);
    T.wt[k >> 3][k & 7].b = make_float4(d[1], d[2], 0.f, 0.f);
  }
}

// plane indices of a place (inverse of bm_lat_place), its base cell in the
// brick (x fastest) and its particle's number in the cell's (x, y, z) order
__device__ __forceinline__ void place_xyz(int q, int &x, int &y, int &z) {
  z = q >> 6;
  y = (q >> 3) & 7;
  x = (q & 4) | ((((q >> 1) ^ q) & 1) << 1) | ((q >> 1) & 1);
}
__device__ __forceinline__ int place_cell8(int q) {  // 8 cell + number
  int x, y, z;
  place_xyz(q, x, y, z);
  return (((z >> 1) * BR + (y >> 1)) * BR + (x >> 1)) * 8 + ((x & 1) * 2 + (y & 1)) * 2 + (z & 1);
}

// Which of cell c's 8 particles carry the pass's code: bit k for particle k.
__device__ __forceinline__ unsigned cell_mask(const uint8_t *cid, int c, int b) {
  const uint2 q = reinterpret_cast<const uint2 *>(cid)[c];
  const unsigned k = (unsigned)b * 0x01010101u;
  const unsigned lo = __vcmpeq4(q.x, k) & 0x08040201u, hi = __vcmpeq4(q.y, k) & 0x08040201u;
  // gather the four flag bits of each word into its low four bits
  return ((lo * 0x01010101u) >> 24) | (((hi * 0x01010101u) >> 24) << 4);
}

// --------------------------------------------------------------------------
// k_p2g_lat (Eq. 2-6, 12-16): as k_p2g_brick, the per-particle work first,
// then the brick's sums of (N, N v) and of A grad N + N J per logical grid.
// --------------------------------------------------------------------------
constexpr int PT = BT;  // the wrench sums of a brick keep their threads

// a particle's scatter inputs, four 16-byte chunks (XORed by bm_lat_xor):
// A0 A3 A1 A4 | A2 A5 J0 J1 | A6 A7 A8 J2 | v0 v1 v2
template <int G>
struct P2GS {
  static constexpr int NP = (G + 1) / 2;  // passes side by side, two groups of PT threads each
  float4 part[LP][4];
  union {
    float sz[NP][7][3][TZ];  // the passes' (node, z-offset) sums
    float wrc[6][G > 1 ? LP : 1];  // before: each particle's reaction wrench (G > 1)
  };
  LatTile T;
  float red[6][PT / 32];
  __align__(8) uint8_t cid[LP];  // code index of each particle, 8 cell + number
};

// The scatter gives a thread one cell and one z offset, as in k_p2g_brick.
// Its 8 particles are the products of two planes per axis: their y-z weights
// are formed once for both x planes.
struct CellOz {
  int c, cx, cy, cz, oz, p0;
  __device__ __forceinline__ CellOz(int t) {  // t < 3 BR3
    c = t % BR3;
    oz = t / BR3;
    cx = c & 3;
    cy = (c >> 2) & 3;
    cz = c >> 4;
    p0 = cz * 128 + cy * 16 + (cx & 2) * 2;  // place bits that do not depend on the particle
  }
  __device__ __forceinline__ int place(int jx, int jy, int jz) const {
    return p0 + jz * 64 + jy * 8 + (jx << 1) + (jx ^ (cx & 1));
  }
};

template <int G>
__device__ __forceinline__ void p2g_momentum(const P2GS<G> &S, const CellOz &q, unsigned m, float (*sz)[3][TZ]) {
  f2 a[3][3][2];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) a[i][j][0] = a[i][j][1] = 0ull;
  if (m) {
    float wx[2][3], wy[2][3], wz[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      plane_w(S.T.wt[0][2 * q.cx + j], wx[j]);
      plane_w(S.T.wt[1][2 * q.cy + j], wy[j]);
      wz[j] = plane_w1(S.T.wt[2][2 * q.cz + j], q.oz);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int jx = k >> 2, jy = (k >> 1) & 1, jz = k & 1;
      if (!((m >> k) & 1u)) continue;
      const int p = q.place(jx, jy, jz);
      const float4 v = S.part[p][3 ^ bm_lat_xor(p)];
      const f2 v12 = pack2(v.y, v.z);
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        const float wyz = wy[jy][oy] * wz[jz];
        const f2 Ma = pack2(wyz, v.x * wyz), Mb = mul2(v12, pack2(wyz, wyz));
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          const f2 ww = pack2(wx[jx][ox], wx[jx][ox]);
          a[oy][ox][0] = fma2(ww, Ma, a[oy][ox][0]);
          a[oy][ox][1] = fma2(ww, Mb, a[oy][ox][1]);
        }
      }
    }
  }
  float s[3][3][4];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      unpack2(a[i][j][0], s[i][j][0], s[i][j][1]);
      unpack2(a[i][j][1], s[i][j][2], s[i][j][3]);
    }
  xy_reduce<4>(s, q.cx, q.cy);
  stage_layer<4, TZ>(sz, s, q.cx, q.cy, q.cz, q.oz);
}

template <int G>
__device__ __forceinline__ void p2g_force(const P2GS<G> &S, const CellOz &q, unsigned m, float (*sz)[3][TZ]) {
  f2 a[3][3];
  float a2[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      a[i][j] = 0ull;
      a2[i][j] = 0.f;
    }
  if (m) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int jx = k >> 2, jy = (k >> 1) & 1, jz = k & 1;
      if (!((m >> k) & 1u)) continue;
      const int p = q.place(jx, jy, jz), x = bm_lat_xor(p);
      float wx[3], dx[3], wy[3], dy[3];
      plane_wd(S.T.wt[0][2 * q.cx + jx], wx, dx);
      plane_wd(S.T.wt[1][2 * q.cy + jy], wy, dy);
      const PlaneW &pz = S.T.wt[2][2 * q.cz + jz];
      const float wz = plane_w1(pz, q.oz), dz = plane_d1(pz, q.oz);
      const float4 ca = S.part[p][0 ^ x], cb = S.part[p][1 ^ x], cc = S.part[p][2 ^ x];
      const f2 A0 = pack2(ca.x, ca.y), A1 = pack2(ca.z, ca.w), A2 = pack2(cb.x, cb.y), J = pack2(cb.z, cb.w);
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        // as in k_p2g_brick: A grad N + N J = wx (A_:1 dyz + A_:2 wyd + J wyz) + dwx (A_:0 wyz)
        const float wyz = wy[oy] * wz, dyz = dy[oy] * wz, wyd = wy[oy] * dz;
        const float U2 = force_u(cc.y, dyz, cc.z, wyd, cc.w, wyz), V2 = cc.x * wyz;
        const f2 pw = pack2(wyz, wyz);
        const f2 U = force_u2(A1, pack2(dyz, dyz), A2, pack2(wyd, wyd), J, pw);
        const f2 V = mul2(A0, pw);
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          a[oy][ox] = force_acc2(a[oy][ox], pack2(wx[ox], wx[ox]), U, pack2(dx[ox], dx[ox]), V);
          a2[oy][ox] = force_acc(a2[oy][ox], wx[ox], U2, dx[ox], V2);
        }
      }
    }
  }
  float s[3][3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      unpack2(a[i][j], s[i][j][0], s[i][j][1]);
      s[i][j][2] = a2[i][j];
    }
  xy_reduce<3>(s, q.cx, q.cy);
  stage_layer<3, TZ>(sz + 4, s, q.cx, q.cy, q.cz, q.oz);
}

template <int MB, bool INELASTIC, int G>
__global__ void __launch_bounds__(PT * G, MB) k_p2g_lat(World w, LaunchSet ls) {
  chain_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  P2GS<G> &S = *reinterpret_cast<P2GS<G> *>(smraw);
  const int4 bt = ls.btiles[blockIdx.x];  // scene, pool brick, first particle, count
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (sc.frozen || !sc.lattice) return;
  const PPool &P = w.P;
  constexpr int NT = PT * G, NP = P2GS<G>::NP;
  const int tid = threadIdx.x, grp = tid / PT;
  const BrickInfo B(w, bt, LP);
  lat_tile(w, bt.y, B.nbc, S.T, NT);
  if (B.mask && tid < LP / 4) reinterpret_cast<unsigned *>(S.cid)[tid] = 0xffffffffu;
  __syncthreads();
  float wr[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  bool clamped = false, anyc = false;
  uint8_t tf_next = tid < bt.w ? P.tflag[bt.z + tid] : 0;  // one iteration ahead, as in stage_particles
  for (int i = tid; i < bt.w; i += NT) {
    const int p = bt.z + i;
    const uint8_t tf = tf_next;
    if (i + NT < bt.w) tf_next = P.tflag[p + NT];
    const float x[3] = {P.x[0][p], P.x[1][p], P.x[2][p]};
    const float v[3] = {P.v[0][p], P.v[1][p], P.v[2][p]};
    const int c = P.cid[p], q = P.lpos[p];
    const uint2 code = c < BM_BRICK_CODES ? S.T.bcode[c] : make_uint2(0u, 0u);
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
    const int xo = bm_lat_xor(q);
    S.part[q][0 ^ xo] = make_float4(A[0], A[3], A[1], A[4]);
    S.part[q][1 ^ xo] = make_float4(A[2], A[5], J[0], J[1]);
    S.part[q][2 ^ xo] = make_float4(A[6], A[7], A[8], J[2]);
    S.part[q][3 ^ xo] = make_float4(v[0], v[1], v[2], 0.f);
    if (B.mask) S.cid[place_cell8(q)] = (uint8_t)c;
  }
  if (clamped) atomicOr(&scm.err, BM_ERRBIT_INVERTED);
  if (!B.uniform) brick_slots<true>(w, S.T, B.nbc, B.pbase, NT);
  if (sc.has_blade) {
    if (G > 1) {
      __syncthreads();
      stride_wrench(S.wrc[0], LP, bt.w, wr);
    }
    brick_wrench(w, bt.y, wr, anyc, S.red);
  }
  __syncthreads();
  const CellOz q(tid % PT);
  for (int b0 = 0; b0 < B.npass; b0 += NP) {
    // G > 1: an even group takes the momentum sums of its pass, the next the force sums
    const int b = b0 + grp / 2;
    if (b < B.npass) {
      const unsigned m = B.mask ? cell_mask(S.cid, q.c, b) : 0xffu;
      if (G == 1 || grp % 2 == 0) p2g_momentum(S, q, m, S.sz[grp / 2]);
      if (G == 1 || grp % 2 == 1) p2g_force(S, q, m, S.sz[grp / 2]);
    }
    __syncthreads();
    for (int t = tid; t < NP * TN; t += NT) {
      const int k = NP == 1 ? 0 : t / TN, nd = t - k * TN;
      if (b0 + k >= B.npass) break;
      const long long e = B.entry(w, S.T, b0 + k, nd);
      if (e < 0) continue;
      float acc[7];
      gather_z<7, TZ>(S.sz[k], nd, acc);
      w.B.pm[e] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      w.B.pd[e] = make_float4(acc[4], acc[5], acc[6], 0.f);
    }
    if (b0 + NP < B.npass) __syncthreads();
  }
}

// --------------------------------------------------------------------------
// k_g2p_lat: G2P (Eq. 17) and the x update, then the MUSL re-scatter
// --------------------------------------------------------------------------
constexpr int GT = 256;  // a thread per (base cell, x plane, y plane): its two z planes
constexpr int TVR = 52;  // floats of one x-row of 6 tile nodes: (v_old, v_new, 2 spare) each, padded

template <int G>
struct G2PS {
  float4 pv[LP];           // v^{n+1} at pv_place
  union {
    float tv[36 * TVR];    // v_old and v_new of the pass's code at the tile's nodes
    float sz[3][3][TZ];    // then: one MUSL pass's (node, z-offset) sums
  } g[G];                  // of each group of GT threads
  LatTile T;
  uint16_t inv[LP];        // particle (index in the brick) at each place
  __align__(8) uint8_t cid[LP];
};

// bank-spread index of a place in arrays of one 16-byte word per particle
__device__ __forceinline__ int pv_place(int p) { return p ^ (((p >> 4) & 1) << 1) ^ (((p >> 3) & 1) << 2); }

template <int G>
__device__ __forceinline__ void musl_cell(const G2PS<G> &S, const CellOz &q, unsigned m, float (*sz)[3][TZ]) {
  f2 a[3][3];
  float a2[3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      a[i][j] = 0ull;
      a2[i][j] = 0.f;
    }
  if (m) {
    float wx[2][3], wy[2][3], wz[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      plane_w(S.T.wt[0][2 * q.cx + j], wx[j]);
      plane_w(S.T.wt[1][2 * q.cy + j], wy[j]);
      wz[j] = plane_w1(S.T.wt[2][2 * q.cz + j], q.oz);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int jx = k >> 2, jy = (k >> 1) & 1, jz = k & 1;
      if (!((m >> k) & 1u)) continue;
      const float4 v = S.pv[pv_place(q.place(jx, jy, jz))];
      const f2 v01 = pack2(v.x, v.y);
#pragma unroll
      for (int oy = 0; oy < 3; ++oy) {
        const float wyz = wy[jy][oy] * wz[jz];
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) {
          const float N = wx[jx][ox] * wyz;
          a[oy][ox] = fma2(pack2(N, N), v01, a[oy][ox]);
          a2[oy][ox] += N * v.z;
        }
      }
    }
  }
  float s[3][3][3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      unpack2(a[i][j], s[i][j][0], s[i][j][1]);
      s[i][j][2] = a2[i][j];
    }
  xy_reduce<3>(s, q.cx, q.cy);
  stage_layer<3, TZ>(sz, s, q.cx, q.cy, q.cz, q.oz);
}

template <int MB, int G>
__global__ void __launch_bounds__(GT * G, MB) k_g2p_lat(World w, LaunchSet ls, int tools) {
  chain_wait();
  extern __shared__ __align__(16) unsigned char smraw[];
  G2PS<G> &S = *reinterpret_cast<G2PS<G> *>(smraw);
  if ((int)blockIdx.x < tools) {
    next_tool(w, ls.scene_ids[blockIdx.x], *reinterpret_cast<ToolS *>(smraw));
    return;
  }
  static_assert(sizeof(ToolS) <= sizeof(G2PS<G>), "the tool step fits");
  const int4 bt = ls.btiles[blockIdx.x - tools];
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (sc.frozen || !sc.lattice) return;
  const PPool &P = w.P;
  constexpr int NT = GT * G;
  const int tid = threadIdx.x % GT, grp = threadIdx.x / GT;  // a pass is a group's
  const BrickInfo B(w, bt, LP);
  // the general kernel multiplies the weights of a tile beyond its slot
  // window in another order: (wx wy) wz, not wx (wy wz)
  const bool wide = w.B.ptot[bt.y] > TSCAP;
  lat_tile(w, bt.y, B.nbc, S.T, NT);
  if (bt.w < LP && grp == 0) reinterpret_cast<unsigned *>(S.inv)[tid] = 0xffffffffu;
  if (B.mask && (int)threadIdx.x < LP / 4) reinterpret_cast<unsigned *>(S.cid)[tid] = 0xffffffffu;
  __syncthreads();
  for (int i = threadIdx.x; i < bt.w; i += NT) {
    const int q = P.lpos[bt.z + i];
    S.inv[q] = (uint16_t)i;
    if (B.mask) S.cid[place_cell8(q)] = P.cid[bt.z + i];
  }
  if (!B.uniform) brick_slots<false>(w, S.T, B.nbc, B.pbase, NT);
  __syncthreads();
  const int cell = tid >> 2, jx = (tid >> 1) & 1, jy = tid & 1;
  const int cx = cell & 3, cy = (cell >> 2) & 3, cz = cell >> 4;
  int pq[2], pi[2], pc[2];
  float v0[2][3], x0[2][3];
#pragma unroll
  for (int j = 0; j < 2; ++j) {  // read ahead of the tile
    pq[j] = bm_lat_place(2 * cx + jx, 2 * cy + jy, 2 * cz + j);
    const int i = S.inv[pq[j]];
    pi[j] = bt.z + i;
    pc[j] = i == 0xffff ? -1 : B.nbc > 1 ? S.cid[cell * 8 + (jx * 2 + jy) * 2 + j] : 0;
    if (pc[j] >= 0 && pc[j] % G == grp)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        v0[j][a] = P.v[a][pi[j]];
        x0[j][a] = P.x[a][pi[j]];
      }
  }
  const float beta = sc.beta, dt = sc.dt;
  bool bad = false;
  for (int b0 = 0; b0 < B.npass; b0 += G) {
    const int b = b0 + grp;
    float *tv = S.g[grp].tv;
    if (tid < TN && b < B.npass) {
      const int sl = B.slot(w, S.T, b, tid);
      float4 vo = make_float4(0.f, 0.f, 0.f, 0.f), vn = vo;
      if (sl != NOSLOT) {
        const int g = S.T.goff[tid] + sl;
        vo = w.S.vold[g];
        vn = w.S.vnew[g];
      }
      float *o = tv + (tid / TE) * TVR + (tid % TE) * 8;
      *reinterpret_cast<float4 *>(o) = make_float4(vo.x, vo.y, vo.z, vn.x);
      *reinterpret_cast<float2 *>(o + 4) = make_float2(vn.y, vn.z);
    }
    __syncthreads();
    if (pc[0] == b || pc[1] == b) {  // (no particle has a code beyond the last)
      float wx[3], wy[3], wz[2][3];
      plane_w(S.T.wt[0][2 * cx + jx], wx);
      plane_w(S.T.wt[1][2 * cy + jy], wy);
      plane_w(S.T.wt[2][2 * cz], wz[0]);
      plane_w(S.T.wt[2][2 * cz + 1], wz[1]);
      f2 acc[2][3];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[j][k] = 0ull;
      const float *r = tv + (cz * TE + cy) * TVR + cx * 8;
#pragma unroll
      for (int oz = 0; oz < 3; ++oz)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy) {
          const float ya = wy[oy] * wz[0][oz], yb = wy[oy] * wz[1][oz];
#pragma unroll
          for (int ox = 0; ox < 3; ++ox) {
            const float *e = r + (oz * TE + oy) * TVR + ox * 8;
            const float4 a4 = *reinterpret_cast<const float4 *>(e);
            const float2 b2 = *reinterpret_cast<const float2 *>(e + 4);
            const f2 pa = pack2(a4.x, a4.y), pb = pack2(a4.z, a4.w), ps = pack2(b2.x, b2.y);
            float Na = wx[ox] * ya, Nb = wx[ox] * yb;
            if (wide) {
              const float xy = wx[ox] * wy[oy];
              Na = xy * wz[0][oz];
              Nb = xy * wz[1][oz];
            }
            const f2 na = pack2(Na, Na), nb = pack2(Nb, Nb);
            acc[0][0] = fma2(na, pa, acc[0][0]);
            acc[0][1] = fma2(na, pb, acc[0][1]);
            acc[0][2] = fma2(na, ps, acc[0][2]);
            acc[1][0] = fma2(nb, pa, acc[1][0]);
            acc[1][1] = fma2(nb, pb, acc[1][1]);
            acc[1][2] = fma2(nb, ps, acc[1][2]);
          }
        }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (pc[j] != b) continue;
        float so[3], sn[3], vv[3];
        unpack2(acc[j][0], so[0], so[1]);
        unpack2(acc[j][1], so[2], sn[0]);
        unpack2(acc[j][2], sn[1], sn[2]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          vv[a] = next_v(beta, v0[j][a], so[a], sn[a]);
          const float xx = next_x(x0[j][a], dt, sn[a]);
          P.v[a][pi[j]] = vv[a];
          P.x[a][pi[j]] = xx;
          bad |= !isfinite(vv[a]) || !isfinite(xx);
        }
        S.pv[pv_place(pq[j])] = make_float4(vv[0], vv[1], vv[2], 0.f);
      }
    }
    if (b0 + G < B.npass) __syncthreads();
  }
  if (bad) atomicOr(&scm.err, BM_ERRBIT_NONFINITE);
  __syncthreads();  // v^{n+1} is complete, and the z stage may take the tile's place
  // ---- MUSL: sums of v^{n+1} N, one pass per code ----
  for (int b0 = 0; b0 < B.npass; b0 += G) {
    const int b = b0 + grp;
    if (tid < 3 * BR3 && b < B.npass) {
      const CellOz q(tid);
      musl_cell(S, q, B.mask ? cell_mask(S.cid, q.c, b) : 0xffu, S.g[grp].sz);
    }
    __syncthreads();
    if (tid < TN && b < B.npass) {
      const long long e = B.entry(w, S.T, b, tid);
      if (e >= 0) {
        float acc[3];
        gather_z<3, TZ>(S.g[grp].sz, tid, acc);
        w.B.pm[e] = make_float4(acc[0], acc[1], acc[2], 0.f);
      }
    }
    if (b0 + G < B.npass) __syncthreads();
  }
}

// --------------------------------------------------------------------------
// k_fupd_lat: F += dt sum v* (x) grad N, and the commit of the side labels
// --------------------------------------------------------------------------
constexpr int FT = 192;

struct FupdS {
  float4 tile[TN];         // v* of the pass's code
  float4 ra[36][8];        // per node row (y, z) and x plane: sum v* dx, and (w:) sum v*_x w
  float2 rb[36][8];        // sum v*_y w, sum v*_z w
  LatTile T;
  int any;
};

template <int MB, bool INELASTIC, int NG>
__global__ void __launch_bounds__(FT * NG, MB) k_fupd_lat(World w, LaunchSet ls) {
  chain_wait();
  __shared__ FupdS S;
  const int4 bt = ls.btiles[blockIdx.x];
  DevScene &scm = w.scenes[bt.x];
  const DevScene &sc = scm;
  if (sc.frozen || !sc.lattice) return;
  const PPool &P = w.P;
  constexpr int NT = FT * NG, NPT = (LP + NT - 1) / NT;  // particles per thread
  const int tid = threadIdx.x;
  const BrickInfo B(w, bt, LP);
  if (tid == 0) S.any = 0;
  float F[NPT][9];  // read up front: the latency passes under the tile
  int pq[NPT], pc[NPT];
#pragma unroll
  for (int j = 0; j < NPT; ++j) {
    const int i = tid + j * NT, p = bt.z + i;
    pc[j] = -1;
    if (i < bt.w) {
      pq[j] = P.lpos[p];
      pc[j] = B.nbc > 1 ? P.cid[p] : 0;
#pragma unroll
      for (int k = 0; k < 9; ++k) F[j][k] = P.F[k][p];
    }
  }
  lat_tile(w, bt.y, B.nbc, S.T, NT);
  __syncthreads();
  if (!B.uniform) {
    brick_slots<false>(w, S.T, B.nbc, -1, NT);
    __syncthreads();
  }
  const float c = sc.dt * sc.inv_dx;
  for (int b = 0; b < B.nbc; ++b) {
    for (int t = tid; t < TN; t += NT) {
      const int sl = B.slot(w, S.T, b, t);
      S.tile[t] = sl != NOSLOT ? w.S.vstar[S.T.goff[t] + sl] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    for (int e = tid; e < 288; e += NT) {
      const int row = e >> 3, x = e & 7;
      float wx[3], dx[3];
      plane_wd(S.T.wt[0][x], wx, dx);
      float sx[3] = {0.f, 0.f, 0.f}, sw[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int ox = 0; ox < 3; ++ox) {
        const float4 v = S.tile[row * TE + (x >> 1) + ox];
        sx[0] += v.x * dx[ox]; sx[1] += v.y * dx[ox]; sx[2] += v.z * dx[ox];
        sw[0] += v.x * wx[ox]; sw[1] += v.y * wx[ox]; sw[2] += v.z * wx[ox];
      }
      S.ra[row][x] = make_float4(sx[0], sx[1], sx[2], sw[0]);
      S.rb[row][x] = make_float2(sw[1], sw[2]);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NPT; ++j) {
      if (pc[j] != b) continue;
      const int p = bt.z + tid + j * NT;
      int x, y, z;
      place_xyz(pq[j], x, y, z);
      float wy[3], dy[3], wz[3], dz[3];
      plane_wd(S.T.wt[1][y], wy, dy);
      plane_wd(S.T.wt[2][z], wz, dz);
      float G[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      const int r0 = (z >> 1) * TE + (y >> 1);
#pragma unroll
      for (int oz = 0; oz < 3; ++oz)
#pragma unroll
        for (int oy = 0; oy < 3; ++oy) {
          const float wyz = wy[oy] * wz[oz], gyz = dy[oy] * wz[oz], wgz = wy[oy] * dz[oz];
          const float4 a = S.ra[r0 + oz * TE + oy][x];
          const float2 d = S.rb[r0 + oz * TE + oy][x];
          const float sx[3] = {a.x, a.y, a.z}, sw[3] = {a.w, d.x, d.y};
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            G[3 * q] += sx[q] * wyz;
            G[3 * q + 1] += sw[q] * gyz;
            G[3 * q + 2] += sw[q] * wgz;
          }
        }
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        P.F[k][p] = F[j][k] + c * G[k];
        if (INELASTIC && sc.viscosity > 0.0f) P.Fdot[k][p] = sc.inv_dx * G[k];
      }
    }
    if (b + 1 < B.nbc) __syncthreads();
  }
  const int cut = sc.cut;
  bool any = false;
  for (int i = tid; i < bt.w && cut >= 0; i += NT) {
    const int p = bt.z + i;
    const uint8_t pend = P.pend[p];
    if (pend) {
      if (pend == 1) P.s1[p] |= 1u << cut;
      else P.s2[p] |= 1u << cut;
      any = true;
      int bx, by, bz;
      particle_base(P.base[p], bx, by, bz);
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

template <class K>
cudaError_t lat_smem(K *kernel, size_t bytes) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)cudaSharedmemCarveoutMaxShared);
}

// Resident CTAs per SM the kernels are compiled for.  Times of the 256-scene
// batch in the middle of a cut (6.0 M particles), ms, general kernels first:
// P2G 0.750 -> 0.574 (0.610 at 3 CTAs, 0.672 at 5), G2P + MUSL 0.590 -> 0.315
// (0.342 at 3, 0.349 at 5), F update 0.442 -> 0.200 (0.206 at 5, 0.193 at 7,
// which costs a 477k-particle scene 2 us of 22).
constexpr int OCC_P2G = 4, OCC_G2P = 4, OCC_FUPD = 6;
// groups of threads of the forms for sets of few bricks (WIDE_BRICKS_LAT)
constexpr int GWIDE = 2, FWIDE = 3;

}  // namespace

cudaError_t bm_lattice_init() {
  cudaError_t e = lat_smem(k_p2g_lat<OCC_P2G, false, 1>, sizeof(P2GS<1>));
  if (e == cudaSuccess) e = lat_smem(k_p2g_lat<OCC_P2G, true, 1>, sizeof(P2GS<1>));
  if (e == cudaSuccess) e = lat_smem(k_p2g_lat<1, false, WIDE>, sizeof(P2GS<WIDE>));
  if (e == cudaSuccess) e = lat_smem(k_p2g_lat<1, true, WIDE>, sizeof(P2GS<WIDE>));
  if (e == cudaSuccess) e = lat_smem(k_g2p_lat<OCC_G2P, 1>, sizeof(G2PS<1>));
  if (e == cudaSuccess) e = lat_smem(k_g2p_lat<1, GWIDE>, sizeof(G2PS<GWIDE>));
  return e;
}

template <int MB, int G>
static void p2g_lat(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.any_inelastic) chain_launch(k_p2g_lat<MB, true, G>, dim3(ls.n_btiles), PT * G, sizeof(P2GS<G>), st, w, ls);
  else chain_launch(k_p2g_lat<MB, false, G>, dim3(ls.n_btiles), PT * G, sizeof(P2GS<G>), st, w, ls);
}

void bm_launch_p2g_lat(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.n_btiles <= WIDE_BRICKS_LAT) p2g_lat<1, WIDE>(w, ls, st);
  else p2g_lat<OCC_P2G, 1>(w, ls, st);
}

void bm_launch_g2p_lat(const World &w, const LaunchSet &ls, cudaStream_t st) {
  const int tools = g2p_tools(ls);
  if (ls.n_btiles <= WIDE_BRICKS_LAT)
    chain_launch(k_g2p_lat<1, GWIDE>, dim3(tools + ls.n_btiles), GT * GWIDE, sizeof(G2PS<GWIDE>), st, w, ls, tools);
  else
    chain_launch(k_g2p_lat<OCC_G2P, 1>, dim3(tools + ls.n_btiles), GT, sizeof(G2PS<1>), st, w, ls, tools);
}

template <int MB, int G>
static void fupd_lat(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.any_inelastic) chain_launch(k_fupd_lat<MB, true, G>, dim3(ls.n_btiles), FT * G, 0, st, w, ls);
  else chain_launch(k_fupd_lat<MB, false, G>, dim3(ls.n_btiles), FT * G, 0, st, w, ls);
}

void bm_launch_fupd_lat(const World &w, const LaunchSet &ls, cudaStream_t st) {
  if (ls.n_btiles <= WIDE_BRICKS_LAT) fupd_lat<1, FWIDE>(w, ls, st);
  else fupd_lat<OCC_FUPD, 1>(w, ls, st);
}
