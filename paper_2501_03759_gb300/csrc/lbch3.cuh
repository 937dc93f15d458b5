// 3D time step on the D3Q15 lattice (the C-ABI of include/lbch3.h), included at the
// end of lbch_api.cu.
//
// A step with general relaxation rates is three kernels over the periodic grid:
//   phi3_kernel      f_in,i(x) = f*_i(x - c_i); phi = sum_i f_in,i            (Eqs. 17, 22)
//   mu3_kernel       grad phi, lap phi (Eq. 26, D3Q15 weights), n, gamma(n) (Eqs. 3, 6),
//                    Q (Eq. 15 reading), w, mu_alpha (Eq. 16), then
//                    mu_beta = (gamma - 1) f - div Q + eps (lap w - f' w)     (Eqs. 13, 16)
//   collide3_kernel  g = grad mu_beta; MRT collision in the Eq. 24 moment basis;
//                    store f* (Eqs. 17-19, 25)
// phi3 and collide3 run one thread per node, x across threads. mu3 sweeps z through an
// x-y tile: each plane of phi and of (Q, w) passes once through shared memory and every
// thread keeps its column's partial stencil sums in registers.
//
// With s_k = 1 for every moment but phi and j, Eq. 17 reads of a node's populations only phi and
// j (and, to close the rest population, the sum of the moving ones). A run of steps then keeps
// the state in moment form, f_0, a = sum_{i >= 1} f_i, j_x, j_y, j_z and phi = f_0 + a:
//   gather3_kernel           once per run: the sums of the pulled populations
//   mu3_kernel               as above, from phi
//   stream3_kernel<false>    collide, and stream into the next step's sums (in shared memory)
//   stream3_kernel<true>     in the last step: collide and store f*
// The populations are read and written once per run instead of twice read and once written per
// step: 52 bytes per node and step pass through stream3 (28 read, 24 written) and 12 through mu3,
// against about 205 for the three kernels (256^3 on GB300: 0.760 ms per step for those, 0.45 ms here).
#pragma once

#include "lbch3_plan.h"

namespace lbch3 {

// Eq. 21a (c = 1) and Eq. 21b.
__host__ __device__ __forceinline__ constexpr int cx(int i) {
  return (i == 1 || i == 7 || i == 9 || i == 11 || i == 14) ? 1 : ((i == 2 || i == 8 || i == 10 || i == 12 || i == 13) ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int cy(int i) {
  return (i == 3 || i == 7 || i == 9 || i == 12 || i == 13) ? 1 : ((i == 4 || i == 8 || i == 10 || i == 11 || i == 14) ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr int cz(int i) {
  return (i == 5 || i == 7 || i == 10 || i == 11 || i == 13) ? 1 : ((i == 6 || i == 8 || i == 9 || i == 12 || i == 14) ? -1 : 0);
}
__host__ __device__ __forceinline__ constexpr double wgt(int i) {
  return i == 0 ? 2.0 / 9.0 : (i <= 6 ? 1.0 / 9.0 : 1.0 / 72.0);
}

// Row k of the Eq. 24 moment basis at velocity i, as the function of c it names.
__host__ __device__ __forceinline__ constexpr int mrow(int k, int i) {
  const int x = cx(i), y = cy(i), z = cz(i), c2 = x * x + y * y + z * z;
  return k == 0 ? 1
       : k == 1 ? c2 - 2
       : k == 2 ? (15 * c2 * c2 - 55 * c2 + 32) / 2
       : k == 3 ? x
       : k == 4 ? (5 * c2 - 13) * x / 2
       : k == 5 ? y
       : k == 6 ? (5 * c2 - 13) * y / 2
       : k == 7 ? z
       : k == 8 ? (5 * c2 - 13) * z / 2
       : k == 9 ? 3 * x * x - c2
       : k == 10 ? y * y - z * z
       : k == 11 ? x * y
       : k == 12 ? y * z
       : k == 13 ? x * z
       : x * y * z;
}

// The basis as a compile-time table, so that every entry the collision uses is a
// literal after unrolling (rows, and their squared norms for M^-1 = M^T diag(1/|M_k|^2)).
struct Basis3 {
  int m[15][15];
  int norm[15];
};
__host__ __device__ constexpr Basis3 make_basis3() {
  Basis3 b{};
  for (int k = 0; k < 15; ++k) {
    b.norm[k] = 0;
    for (int i = 0; i < 15; ++i) {
      b.m[k][i] = mrow(k, i);
      b.norm[k] += b.m[k][i] * b.m[k][i];
    }
  }
  return b;
}
constexpr Basis3 kBasis3 = make_basis3();
template <int K, int I>
struct MR {
  static constexpr int v = kBasis3.m[K][I];
};
template <int K>
struct MN {
  static constexpr int v = kBasis3.norm[K];
};

struct Grid3 {
  int nx, ny, nz;
  int segs;      // x segments of NX3 nodes per row (node kernels)
  long long ps;  // plane stride (elements)
};

constexpr int NX3 = 128;  // threads per block of the node kernels, along x

struct Consts3 {
  float k, kq, kiso, beta4, beta12, alpha, a16, eps, cw, cfp, cnk;
  float s[15];
};

__device__ __forceinline__ int wrapi(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }
__device__ __forceinline__ int modn(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// A node and the offsets of its neighbours (x fastest; 32-bit, since n < 2^31).
struct Site {
  int x, y, z, id;
  int xo[3];     // x - 1, x, x + 1 (periodic)
  int ro[3][3];  // (z + dz) ny nx + (y + dy) nx for dy, dz in {-1, 0, 1} (periodic)
  __device__ __forceinline__ int at(int dx, int dy, int dz) const { return ro[dy + 1][dz + 1] + xo[dx + 1]; }
};

// The node of this thread in node-kernel block b (x segment fastest, then y, then z);
// false past the end of the row.
__device__ __forceinline__ bool site_of(const Grid3& g, int b, Site& s) {
  const int seg = b % g.segs, row = b / g.segs;
  s.x = seg * NX3 + (int)threadIdx.x;
  if (s.x >= g.nx) return false;
  s.y = row % g.ny;
  s.z = row / g.ny;
  s.xo[0] = s.x == 0 ? g.nx - 1 : s.x - 1;
  s.xo[1] = s.x;
  s.xo[2] = s.x + 1 == g.nx ? 0 : s.x + 1;
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) s.ro[dy + 1][dz + 1] = (wrapi(s.z + dz, g.nz) * g.ny + wrapi(s.y + dy, g.ny)) * g.nx;
  s.id = s.ro[1][1] + s.x;
  return true;
}

// Gradient (Eq. 26a) and Laplacian (Eq. 26b) from the centre value c and the
// neighbour values t[i] = v(x + c_i), i = 1..14. The gradient pairs opposite
// velocities (c_{2j} = -c_{2j-1} in Eq. 21a), so each term is an exact difference and a
// locally uniform field gives exactly zero; the Laplacian sums differences from c.
__device__ __forceinline__ void grad_lap(float c, const float (&t)[15], float& gx, float& gy, float& gz, float& lap) {
  float sx = 0.0f, sy = 0.0f, sz = 0.0f, sl = 0.0f;
#pragma unroll
  for (int i = 1; i < 15; i += 2) {
    const float d = t[i] - t[i + 1];
    const float w = (float)(3.0 * wgt(i));
    if (cx(i) != 0) sx = fmaf(w * cx(i), d, sx);
    if (cy(i) != 0) sy = fmaf(w * cy(i), d, sy);
    if (cz(i) != 0) sz = fmaf(w * cz(i), d, sz);
    sl = fmaf(2.0f * w, (t[i] - c) + (t[i + 1] - c), sl);
  }
  gx = sx;
  gy = sy;
  gz = sz;
  lap = sl;
}

__device__ __forceinline__ void stencil(const float* __restrict__ v, const Site& s, float& gx, float& gy, float& gz,
                                        float& lap) {
  float t[15];
#pragma unroll
  for (int i = 1; i < 15; ++i) t[i] = v[s.at(cx(i), cy(i), cz(i))];
  grad_lap(v[s.id], t, gx, gy, gz, lap);
}

// Population load with a 256-byte L2 fetch (.L2::256B): a block's 128 threads read 512
// contiguous bytes of each plane row (0.7636 -> 0.7602 ms per 256^3 step on GB300).
__device__ __forceinline__ float ld_pop(const float* p) {
  float v;
  asm("ld.global.nc.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
// The same in a kernel that launch_dep starts: a plain load that stays behind wait_previous().
__device__ __forceinline__ float ld_pop_dep(const float* p) {
  float v;
  asm volatile("ld.global.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}

__global__ void __launch_bounds__(NX3) phi3_kernel(const float* __restrict__ f, Grid3 g, float* __restrict__ phi) {
  Site s;
  if (!site_of(g, blockIdx.x, s)) return;
  float p = 0.0f;
#pragma unroll
  for (int i = 0; i < 15; ++i) p += ld_pop(f + (long long)i * g.ps + s.at(-cx(i), -cy(i), -cz(i)));
  phi[s.id] = p;
}

// ---------------------------------------------------------------- mu3_kernel

using lbch::cp_async4;

constexpr int MU_TX = 30, MU_TY = 14;                // mu_beta outputs per plane and tile
constexpr int MU_QX = MU_TX + 2, MU_QY = MU_TY + 2;  // (Q, w) region: one thread per column
constexpr int MU_PX = MU_TX + 4, MU_PY = MU_TY + 4;  // phi region
constexpr int MU_THREADS = 32 * MU_QY;
constexpr int MU_PHI_PER_THREAD = (MU_PX * MU_PY + MU_THREADS - 1) / MU_THREADS;
constexpr int MU_RING = 6;  // planes in shared memory: MU_RING - 1 in flight ahead of the sweep
static_assert(MU_QX == 32, "one lane per (Q, w) column");

// The work of mu3_kernel and stream3_kernel: tiles_x * tiles tiles of x-y, each a column of nz
// planes cut into segments of len planes; block b takes tile b % tiles of segment b / tiles. Blocks
// that run together then sweep the same planes of neighbouring tiles, and what they share, the halos
// and the 32-byte sectors that a tile's edge cuts, is still in L2. (256^3: equal runs of a (tile, z) list instead, where neighbours were dozens
// of planes apart, took 440 us a stream3 launch instead of 229, and 890 instead of 332 the last one.)
struct MuTiles {
  int tiles_x, tiles;
  int len;
};

// Anisotropic quantities at one node from its phi, grad phi and lap phi: Q (reading of
// Eq. 15 under LBCH_Q_LITERAL / LBCH_MU_NESTED), w = lap phi - f (Eq. 9; 0 for the
// linear regularisation), mu_alpha (Eq. 16) and the local part of mu_beta.
struct Aniso {
  float qx, qy, qz, w, mua, a;
};
__device__ __forceinline__ Aniso aniso(const Consts3& c, float p, float dx, float dy, float dz, float lap) {
  Aniso r;
  const float g2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
  const bool ok = g2 >= 1e-12f;  // n = 0, gamma = 1 below this
  const float rs = lbch::rsqrt_normal(ok ? g2 : 1.0f);
  const float n1 = dx * rs, n2 = dy * rs, n3 = dz * rs;  // Eq. 3
  const float n1s = n1 * n1, n2s = n2 * n2, n3s = n3 * n3;
  const float S4 = fmaf(n1s, n1s, fmaf(n2s, n2s, n3s * n3s));
  const float gm1 = ok ? c.alpha * fmaf(4.0f, S4, -3.0f) : 0.0f;  // gamma - 1, Eq. 6
  const float t = ok ? c.kq * c.a16 * (g2 * rs) : 0.0f;         // k_q |grad phi| 16 alpha
  const float kg = fmaf(c.k, gm1, c.kiso);
  r.qx = fmaf(kg, dx, t * (n1 * (n1s - S4)));  // P grad_n gamma = 16 alpha n (n^2 - sum n^4)
  r.qy = fmaf(kg, dy, t * (n2 * (n2s - S4)));
  r.qz = fmaf(kg, dz, t * (n3 * (n3s - S4)));
  const float p2 = p * p;
  const float fb = c.beta4 * p * (p2 - 1.0f);
  const float fp = fmaf(c.beta12, p2, -c.beta4);
  r.w = fmaf(-c.cw, fb, lap);
  r.mua = fmaf(-c.k, lap, fb);
  r.a = fmaf(gm1, fb, fmaf(-c.cfp * fp, r.w, c.cnk * lap));
  return r;
}

// Stencil weights of Eq. 26 on D3Q15: 3 w_i for the gradient, 6 w_i for the Laplacian.
constexpr float G1 = 3.0f / 9.0f, G7 = 3.0f / 72.0f, L1 = 6.0f / 9.0f, L7 = 6.0f / 72.0f;

// What one plane p of phi gives the stencils at (x, y): the centre c, the in-plane axis
// terms of the gradient and Laplacian at (x, y, p), and the sums over the four in-plane
// diagonal neighbours (x +- 1, y +- 1, p) that the corner velocities of planes p -+ 1
// use: X = sum s_x v, Y = sum s_y v, S = sum v. Differences and pair sums are formed
// first, so a locally uniform field gives exact zeros.
struct PhiPlane {
  float c, gx, gy, lap, X, Y, S;
};
__device__ __forceinline__ PhiPlane phi_plane(const float (*v)[MU_PX], int rx, int ry) {
  PhiPlane r;
  const float c = v[ry][rx], e = v[ry][rx + 1], w = v[ry][rx - 1], n = v[ry + 1][rx], s = v[ry - 1][rx];
  const float ne = v[ry + 1][rx + 1], nw = v[ry + 1][rx - 1], se = v[ry - 1][rx + 1], sw = v[ry - 1][rx - 1];
  r.c = c;
  r.gx = G1 * (e - w);
  r.gy = G1 * (n - s);
  r.lap = L1 * (((e - c) + (w - c)) + ((n - c) + (s - c)));
  r.X = (ne - nw) + (se - sw);
  r.Y = (ne - se) + (nw - sw);
  r.S = (ne + nw) + (se + sw);
  return r;
}

// The same for one plane of (Q_x, Q_y, Q_z, w): in-plane parts of div Q and lap w, the
// diagonal sums X = sum s_x Q_x, Y = sum s_y Q_y, Z = sum Q_z, W = sum w, and the centre
// Q_z and w.
struct QPlane {
  float div, lapw, X, Y, Z, W, qz, w;
};
__device__ __forceinline__ QPlane q_plane(const float (*q)[MU_QY][MU_QX], int rx, int ry) {
  QPlane r;
  const float (*Qx)[MU_QX] = q[0];
  const float (*Qy)[MU_QX] = q[1];
  const float (*Qz)[MU_QX] = q[2];
  const float (*W)[MU_QX] = q[3];
  const float wc = W[ry][rx];
  r.div = G1 * ((Qx[ry][rx + 1] - Qx[ry][rx - 1]) + (Qy[ry + 1][rx] - Qy[ry - 1][rx]));
  r.lapw = L1 * (((W[ry][rx + 1] - wc) + (W[ry][rx - 1] - wc)) + ((W[ry + 1][rx] - wc) + (W[ry - 1][rx] - wc)));
  r.X = (Qx[ry + 1][rx + 1] - Qx[ry + 1][rx - 1]) + (Qx[ry - 1][rx + 1] - Qx[ry - 1][rx - 1]);
  r.Y = (Qy[ry + 1][rx + 1] - Qy[ry - 1][rx + 1]) + (Qy[ry + 1][rx - 1] - Qy[ry - 1][rx - 1]);
  r.Z = (Qz[ry + 1][rx + 1] + Qz[ry + 1][rx - 1]) + (Qz[ry - 1][rx + 1] + Qz[ry - 1][rx - 1]);
  r.W = (W[ry + 1][rx + 1] + W[ry + 1][rx - 1]) + (W[ry - 1][rx + 1] + W[ry - 1][rx - 1]);
  r.qz = Qz[ry][rx];
  r.w = wc;
  return r;
}

// A block sweeps z through an x-y tile; thread (lane, warp) owns the column (x0 - 1 + lane,
// y0 - 1 + warp) of the (Q, w) region. Each plane of phi and of (Q, w) passes through shared memory
// once; the thread keeps what the planes below contributed to its column's stencils in registers:
//   phi plane p arrives             ->  grad phi, lap phi, Q, w, mu_alpha on plane t = p - 1
//   (Q, w) plane t, one plane later ->  mu_beta on plane t - 1 (interior columns)
// so one barrier per plane serves both (two buffers of (Q, w)), and the two halves of an iteration
// are independent. phi planes arrive by cp.async MU_RING - 1 planes ahead. Bound by instruction
// issue: the loop runs three planes per iteration, in which the planes' registers change roles
// instead of being moved, and rings and offsets step by additions: 37.1 -> 31.1 M warp instructions
// on 128^3, 48.7 -> 42.7 us (256^3, with the shorter segments of MuTiles: 236 -> 223 us).
__global__ void __launch_bounds__(MU_THREADS, 2) mu3_kernel(const float* phi, Grid3 g, Consts3 c,
                                                            MuTiles mt, float* __restrict__ mua,
                                                            float* __restrict__ mub) {
  lbch::begin_dependents();
  __shared__ float sphi[MU_RING][MU_PY][MU_PX];
  __shared__ float sq[2][4][MU_QY][MU_QX];
  static_assert(MU_RING == 6, "two iterations of three planes");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tile = blockIdx.x % mt.tiles, z0 = blockIdx.x / mt.tiles * mt.len, z1 = min(g.nz, z0 + mt.len);
  const int x0 = (tile % mt.tiles_x) * MU_TX, y0 = (tile / mt.tiles_x) * MU_TY;
  const int plane = g.ny * g.nx;
  const int gx = x0 - 1 + lane, gy = y0 - 1 + warp;  // this column
  const bool out = lane >= 1 && lane <= MU_TX && warp >= 1 && warp <= MU_TY && gx < g.nx && gy < g.ny;
  int src_off[MU_PHI_PER_THREAD];  // in-plane offset of each element this thread copies
#pragma unroll
  for (int j = 0; j < MU_PHI_PER_THREAD; ++j) {
    const int r = threadIdx.x + j * MU_THREADS;
    const int rx = r % MU_PX, ry = r / MU_PX;
    src_off[j] = r < MU_PX * MU_PY ? modn(y0 - 2 + ry, g.ny) * g.nx + modn(x0 - 2 + rx, g.nx) : 0;
  }
  // phi planes z0 - 2 .. z1 + 1 into the ring's slots in order; one group per plane (empty past the last)
  int zi = modn(z0 - 2, g.nz), left = z1 - z0 + 4;
  auto issue = [&](int slot) {
    if (left > 0) {
      const float* src = phi + (long long)zi * plane;
      float* dst = &sphi[slot][0][0];
#pragma unroll
      for (int j = 0; j < MU_PHI_PER_THREAD; ++j) {
        const int r = threadIdx.x + j * MU_THREADS;
        if (r < MU_PX * MU_PY) cp_async4(dst + r, src + src_off[j]);
      }
      --left;
      zi = zi + 1 == g.nz ? 0 : zi + 1;
    }
    lbch::cp_async_commit();
  };
  lbch::wait_previous();
#pragma unroll
  for (int k = 0; k < MU_RING - 1; ++k) issue(k);

  PhiPlane P[3] = {};  // phi planes of this column, (Q, w) planes, and the local part of mu_beta:
  QPlane Q[3] = {};    // index K the newest, (K + 2) % 3 and (K + 1) % 3 the one and two below
  float a[3] = {};
  int s3 = 0, buf = 0;                // ring slot of the iteration's first plane; (Q, w) buffer
  unsigned id = (unsigned)((z0 - 3) * plane + gy * g.nx + gx);  // node of plane p - 1 of this column
  auto step = [&](auto kc, int p) {
    constexpr int K = decltype(kc)::value, K1 = (K + 2) % 3, K2 = (K + 1) % 3;
    lbch::cp_async_wait<MU_RING - 2>();  // this thread's copies of plane p have landed
    __syncthreads();                     // and everyone's; so are the (Q, w) of plane p - 2
    issue(K > 0 ? s3 + K - 1 : 5 - s3);
    const int t = p - 1;
    if (p <= z1 + 1) {
      P[K] = phi_plane(sphi[s3 + K], lane + 1, warp + 1);
      if (t >= z0 - 1) {
        const PhiPlane &p0 = P[K], &p1 = P[K1], &p2 = P[K2];
        const float dx = p1.gx + G7 * (p0.X + p2.X);
        const float dy = p1.gy + G7 * (p0.Y + p2.Y);
        const float dz = G1 * (p0.c - p2.c) + G7 * (p0.S - p2.S);
        const float lap = p1.lap + L1 * ((p0.c - p1.c) + (p2.c - p1.c)) +
                          L7 * ((p0.S - 4.0f * p1.c) + (p2.S - 4.0f * p1.c));
        const Aniso r = aniso(c, p1.c, dx, dy, dz, lap);
        sq[buf][0][warp][lane] = r.qx;
        sq[buf][1][warp][lane] = r.qy;
        sq[buf][2][warp][lane] = r.qz;
        sq[buf][3][warp][lane] = r.w;
        if (out && t >= z0 && t < z1) mua[id] = r.mua;
        a[K] = r.a;
      }
    }
    if (t >= z0 && out) {  // (Q, w) of plane t - 1 completes mu_beta of plane t - 2
      Q[K] = q_plane(sq[buf ^ 1], lane, warp);
      if (t - 2 >= z0) {
        const QPlane &q0 = Q[K], &q1 = Q[K1], &q2 = Q[K2];
        const float div = q1.div + G7 * (((q0.X + q2.X) + (q0.Y + q2.Y)) + (q0.Z - q2.Z)) + G1 * (q0.qz - q2.qz);
        const float lapw = q1.lapw + L1 * ((q0.w - q1.w) + (q2.w - q1.w)) +
                           L7 * ((q0.W - 4.0f * q1.w) + (q2.W - 4.0f * q1.w));
        mub[id - 2u * (unsigned)plane] = fmaf(c.eps, lapw, a[K2] - div);  // Eq. 13 minus mu_alpha
      }
    }
    buf ^= 1;
    id += plane;
  };
  for (int p = z0 - 2; p <= z1 + 2; p += 3) {
    step(std::integral_constant<int, 0>{}, p);
    if (p + 1 <= z1 + 2) step(std::integral_constant<int, 1>{}, p + 1);
    if (p + 2 <= z1 + 2) step(std::integral_constant<int, 2>{}, p + 2);
    s3 = 3 - s3;
  }
  lbch::cp_async_wait<0>();
}

// ---------------------------------------------------------------- collide3_kernel

// Moment k of f (row k of Eq. 24 applied to f[0..14]); entries are literals.
template <int K, int I = 0>
__device__ __forceinline__ float moment(const float (&f)[15]) {
  if constexpr (I == 15) {
    return 0.0f;
  } else {
    constexpr int m = MR<K, I>::v;
    const float rest = moment<K, I + 1>(f);
    if constexpr (m == 0) return rest;
    else if constexpr (m == 1) return f[I] + rest;
    else if constexpr (m == -1) return rest - f[I];
    else return fmaf((float)m, f[I], rest);
  }
}

// Population i of M^T n (column i of Eq. 24 against the scaled post-collision moments).
template <int I, int K = 0>
__device__ __forceinline__ float back(const float (&n)[15]) {
  if constexpr (K == 15) {
    return 0.0f;
  } else {
    constexpr int m = MR<K, I>::v;
    const float rest = back<I, K + 1>(n);
    if constexpr (m == 0) return rest;
    else if constexpr (m == 1) return n[K] + rest;
    else if constexpr (m == -1) return rest - n[K];
    else return fmaf((float)m, n[K], rest);
  }
}

template <int K>
__device__ __forceinline__ void relax(const float (&f)[15], float phi, float m_a, float gx, float gy, float gz,
                                      const Consts3& c, float (&nk)[15]) {
  // m^eq = (phi, -2 phi + mu_a, 16 phi - 15 mu_a, 0, ...) (Eq. 18 in the Eq. 24 basis);
  // F_m = M F is nonzero on j (-g/3) and q (7 g/9) only (Eq. 19).
  const float meq = K == 0 ? phi : (K == 1 ? fmaf(-2.0f, phi, m_a) : (K == 2 ? fmaf(16.0f, phi, -15.0f * m_a) : 0.0f));
  const float gk = (K == 3 || K == 4) ? gx : ((K == 5 || K == 6) ? gy : gz);
  const float Fm = (K == 3 || K == 5 || K == 7) ? -gk * (1.0f / 3.0f) : ((K == 4 || K == 6 || K == 8) ? gk * (7.0f / 9.0f) : 0.0f);
  const float m = moment<K>(f);
  const float ms = fmaf(-c.s[K], m - meq, m) + (1.0f - 0.5f * c.s[K]) * Fm;  // Eq. 17 in moments
  nk[K] = ms * (1.0f / (float)MN<K>::v);
  if constexpr (K + 1 < 15) relax<K + 1>(f, phi, m_a, gx, gy, gz, c, nk);
}

template <int I>
__device__ __forceinline__ void unproject(const float (&nk)[15], float (&o)[15]) {
  o[I] = back<I>(nk);
  if constexpr (I + 1 < 15) unproject<I + 1>(nk, o);
}

__global__ void __launch_bounds__(NX3) collide3_kernel(const float* __restrict__ src, const float* __restrict__ mub,
                                                       const float* __restrict__ mua, Grid3 g, Consts3 c,
                                                       float* __restrict__ dst) {
  Site s;
  if (!site_of(g, blockIdx.x, s)) return;
  float f[15];
#pragma unroll
  for (int i = 0; i < 15; ++i) f[i] = ld_pop(src + (long long)i * g.ps + s.at(-cx(i), -cy(i), -cz(i)));
  float gx, gy, gz, unused;
  stencil(mub, s, gx, gy, gz, unused);
  float phi = 0.0f;
#pragma unroll
  for (int i = 0; i < 15; ++i) phi += f[i];
  float nk[15], o[15];
  relax<0>(f, phi, mua[s.id], gx, gy, gz, c, nk);
  unproject<0>(nk, o);
  // Rest population closes the mass exactly (sum_i f* = sum_i f, Eq. 34).
  float d = 0.0f;
#pragma unroll
  for (int i = 1; i < 15; ++i) d += f[i] - o[i];
  o[0] = f[0] + d;
#pragma unroll
  for (int i = 0; i < 15; ++i) dst[(long long)i * g.ps + s.id] = o[i];
}

// ---------------------------------------------------------------- moment form

// Constants of the collision from sums: the factors of j and of g in the axis and the diagonal
// populations, per direction. From n_j = ((1 - s) j - (1 - s/2) g / 3) / 10 and n_q = (7/18) g / 40
// (the j and q rows of Eq. 24 with F_m = M F), axis populations take n_j - 4 n_q and diagonal
// ones n_j + n_q.
struct Sums3 {
  float cj[3], ga[3], gd[3];
};

// Every operation below is one IEEE operation or one fma, spelled out, so that the kernels that
// share them round alike and a run equals its steps bit for bit.
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }

// f* of a node from its sums (o[0] the rest population). As in 2D, the rest population closes the
// mass, and what rounding it drops goes to the eight diagonal populations in equal parts.
__device__ __forceinline__ void collide_sums3(const Sums3& c, float f0, float a, float jx, float jy, float jz,
                                              float mua, float gx, float gy, float gz, float (&o)[15]) {
  const float A0 = mul(1.0f / 9.0f, mua), D0 = mul(1.0f / 72.0f, mua);
  const float Jx = mul(c.cj[0], jx), Jy = mul(c.cj[1], jy), Jz = mul(c.cj[2], jz);
  const float X = __fmaf_rn(c.ga[0], gx, Jx), Y = __fmaf_rn(c.ga[1], gy, Jy), Z = __fmaf_rn(c.ga[2], gz, Jz);
  const float U = __fmaf_rn(c.gd[0], gx, Jx), V = __fmaf_rn(c.gd[1], gy, Jy), W = __fmaf_rn(c.gd[2], gz, Jz);
  o[1] = add(A0, X);
  o[2] = sub(A0, X);
  o[3] = add(A0, Y);
  o[4] = sub(A0, Y);
  o[5] = add(A0, Z);
  o[6] = sub(A0, Z);
  const float P = add(U, V), M = sub(U, V);
  const float p = add(P, W), q = sub(P, W), r = add(M, W), t = sub(M, W);
  o[7] = add(D0, p);    // ( 1,  1,  1)
  o[8] = sub(D0, p);    // (-1, -1, -1)
  o[9] = add(D0, q);    // ( 1,  1, -1)
  o[10] = sub(D0, q);   // (-1, -1,  1)
  o[11] = add(D0, r);   // ( 1, -1,  1)
  o[12] = sub(D0, r);   // (-1,  1, -1)
  o[13] = sub(D0, t);   // (-1,  1,  1)
  o[14] = add(D0, t);   // ( 1, -1, -1)
  const float T = add(add(add(add(o[1], o[2]), add(o[3], o[4])), add(o[5], o[6])),
                      add(add(add(o[7], o[8]), add(o[9], o[10])), add(add(o[11], o[12]), add(o[13], o[14]))));
  const float d = sub(a, T);
  o[0] = add(f0, d);
  const float res = mul(0.125f, sub(d, sub(o[0], f0)));
#pragma unroll
  for (int i = 7; i < 15; ++i) o[i] = add(o[i], res);
}

// The moving populations arriving at a node, by the plane they come from: S is the sum of a group
// and Dx, Dy its c_x- and c_y-weighted sums. v5, v7, .. are the pulled populations.
__device__ __forceinline__ void group_up(float v5, float v7, float v10, float v11, float v13, float& S, float& Dx,
                                         float& Dy) {
  S = add(v5, add(add(v7, v10), add(v11, v13)));
  const float a = sub(v7, v10), b = sub(v11, v13);
  Dx = add(a, b);
  Dy = sub(a, b);
}
__device__ __forceinline__ void group_down(float v6, float v8, float v9, float v12, float v14, float& S, float& Dx,
                                           float& Dy) {
  S = add(v6, add(add(v8, v9), add(v12, v14)));
  const float a = sub(v9, v8), b = sub(v14, v12);
  Dx = add(a, b);
  Dy = sub(a, b);
}

// Populations to moment planes m (f0, a, jx, jy, jz, plane stride g.ps) and phi; one thread per node.
__global__ void __launch_bounds__(NX3) gather3_kernel(const float* f, Grid3 g, float* __restrict__ m,
                                                      float* __restrict__ phi) {
  lbch::begin_dependents();
  lbch::wait_previous();
  Site s;
  if (!site_of(g, blockIdx.x, s)) return;
  float v[15];
#pragma unroll
  for (int i = 0; i < 15; ++i) v[i] = ld_pop_dep(f + (long long)i * g.ps + s.at(-cx(i), -cy(i), -cz(i)));
  float Su, Dux, Duy, Sd, Ddx, Ddy;
  group_up(v[5], v[7], v[10], v[11], v[13], Su, Dux, Duy);
  group_down(v[6], v[8], v[9], v[12], v[14], Sd, Ddx, Ddy);
  const float Sl = add(add(v[1], v[2]), add(v[3], v[4]));
  const float a = add(add(Su, Sl), Sd);
  m[s.id] = v[0];
  m[g.ps + s.id] = a;
  m[2 * g.ps + s.id] = add(add(Dux, sub(v[1], v[2])), Ddx);
  m[3 * g.ps + s.id] = add(add(Duy, sub(v[3], v[4])), Ddy);
  m[4 * g.ps + s.id] = sub(Su, Sd);
  phi[s.id] = add(v[0], a);
}

// What one plane of mu_beta gives the gradient at (x, y), as phi_plane (no Laplacian).
struct MubPlane {
  float c, gx, gy, X, Y, S;
};
__device__ __forceinline__ MubPlane mub_plane(const float (*v)[MU_PX], int rx, int ry) {
  MubPlane r;
  const float e = v[ry][rx + 1], w = v[ry][rx - 1], n = v[ry + 1][rx], s = v[ry - 1][rx];
  const float ne = v[ry + 1][rx + 1], nw = v[ry + 1][rx - 1], se = v[ry - 1][rx + 1], sw = v[ry - 1][rx - 1];
  r.c = v[ry][rx];
  r.gx = mul(G1, sub(e, w));
  r.gy = mul(G1, sub(n, s));
  r.X = add(sub(ne, nw), sub(se, sw));
  r.Y = add(sub(ne, se), sub(nw, sw));
  r.S = add(add(ne, nw), add(se, sw));
  return r;
}

// Shared memory of stream3_kernel: the ring of mu_beta planes and two planes of the ten
// populations that stream across rows (o3, o4 in the plane, the eight diagonal ones).
constexpr int ST_POPS = 10;
constexpr int ST_SMEM = (MU_RING * MU_PY * MU_PX + 2 * ST_POPS * MU_QY * MU_QX) * (int)sizeof(float);

// Sweeps z through a tile as mu3_kernel; thread (lane, warp) owns the column (x0 - 1 + lane,
// y0 - 1 + warp), collides it plane by plane, and streams into its next sums:
//   mu_beta plane p arrives       ->  grad mu_beta and f* on plane t = p - 1, into shared memory
//   one plane (and barrier) later ->  the arrivals from plane t: down to t - 1, which is then
//                                     complete, in the plane to t, and up to t + 1
// so one barrier per plane serves both, and the two halves of an iteration are independent. o1 and
// o2 move along x by shuffles, o5 and o6 stay in the thread. The interior 30 x 14 columns store.
// Bound by instruction issue, like mu3_kernel (78% of the slots): 229 us at 256^3, where 52 bytes per
// node would take about 130 us.
// LAST: stores f* (plane stride g.ps) in `out` instead of the next sums, and no phi.
template <bool LAST>
__global__ void __launch_bounds__(MU_THREADS, 2) stream3_kernel(const float* m, const float* mub, const float* mua,
                                                                Grid3 g, Sums3 c, MuTiles mt, float* __restrict__ out,
                                                                float* __restrict__ phi) {
  lbch::begin_dependents();
  lbch::wait_previous();
  extern __shared__ float smem3[];
  float (*smub)[MU_PY][MU_PX] = reinterpret_cast<float (*)[MU_PY][MU_PX]>(smem3);
  float (*so)[ST_POPS][MU_QY][MU_QX] =
      reinterpret_cast<float (*)[ST_POPS][MU_QY][MU_QX]>(smem3 + MU_RING * MU_PY * MU_PX);
  constexpr int EDGE = LAST ? 0 : 1;  // planes collided beyond each end of the run
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int plane = g.ny * g.nx;
  const int tile = blockIdx.x % mt.tiles, z0 = blockIdx.x / mt.tiles * mt.len, z1 = min(g.nz, z0 + mt.len);
  const int x0 = (tile % mt.tiles_x) * MU_TX, y0 = (tile / mt.tiles_x) * MU_TY;
  {
    const int gx = x0 - 1 + lane, gy = y0 - 1 + warp;  // this column
    const bool store = lane >= 1 && lane <= MU_TX && warp >= 1 && warp <= MU_TY && gx < g.nx && gy < g.ny;
    const int col = modn(gy, g.ny) * g.nx + modn(gx, g.nx);  // its node in a plane

    // mu_beta plane p lands in ring slot (p - first) % MU_RING, as phi in mu3_kernel
    const int first = z0 - 1 - EDGE, last = z1 + EDGE;  // mu_beta planes of the run
    int src_off[MU_PHI_PER_THREAD];
#pragma unroll
    for (int j = 0; j < MU_PHI_PER_THREAD; ++j) {
      const int r = threadIdx.x + j * MU_THREADS;
      const int rx = r % MU_PX, ry = r / MU_PX;
      src_off[j] = r < MU_PX * MU_PY ? modn(y0 - 2 + ry, g.ny) * g.nx + modn(x0 - 2 + rx, g.nx) : 0;
    }
    int zi = modn(first, g.nz), pi = first, si = 0;  // next plane to fetch: wrapped z, plane, slot
    auto issue = [&]() {
      if (pi <= last) {
        const float* src = mub + (long long)zi * plane;
        float* dst = &smub[si][0][0];
#pragma unroll
        for (int j = 0; j < MU_PHI_PER_THREAD; ++j) {
          const int r = threadIdx.x + j * MU_THREADS;
          if (r < MU_PX * MU_PY) cp_async4(dst + r, src + src_off[j]);
        }
        ++pi;
        zi = zi + 1 == g.nz ? 0 : zi + 1;
        si = si + 1 == MU_RING ? 0 : si + 1;
      }
      lbch::cp_async_commit();
    };
    // this column's sums and mu_alpha on the plane collided next, fetched one plane ahead
    int zc = modn(z0 - EDGE, g.nz);
    float nf0, na, njx, njy, njz, nmu;
    auto fetch = [&]() {
      const float* q = m + (long long)zc * plane + col;
      nf0 = q[0];
      na = q[g.ps];
      njx = q[2 * g.ps];
      njy = q[3 * g.ps];
      njz = q[4 * g.ps];
      nmu = mua[(long long)zc * plane + col];
      zc = zc + 1 == g.nz ? 0 : zc + 1;
    };

    MubPlane p1{}, p2{};  // mu_beta planes p - 1 and p - 2 of this column
    float A1 = 0, JX1 = 0, JY1 = 0, SU1 = 0, F1 = 0;  // sums of plane t - 2 but for its down group
    float SU0 = 0, DX0 = 0, DY0 = 0;                   // the up group arriving on plane t - 1
    float o0 = 0, o5 = 0, o6 = 0, lx = 0, ly = 0;      // plane t - 1: rest, up, down; o1 and o2 as pulled
#pragma unroll
    for (int k = 0; k < MU_RING - 1; ++k) issue();
    fetch();
    int slot = 0, buf = 0;
    // Plane t = p - 1 collides for z0 - EDGE <= t < z1 + EDGE; its arrivals are taken at p + 1.
    for (int p = first; p <= last + EDGE; ++p) {
      lbch::cp_async_wait<MU_RING - 2>();
      __syncthreads();  // mu_beta plane p and the populations of plane p - 2 are everyone's
      issue();
      const int t = p - 1;
      if (!LAST && t - 1 >= z0 - EDGE) {  // arrivals from plane t - 1
        if (store) {
          const float (*q)[MU_QY][MU_QX] = so[buf ^ 1];
          float Su, Dux, Duy, Sd, Ddx, Ddy;
          group_up(o5, q[2][warp - 1][lane - 1], q[5][warp + 1][lane + 1], q[6][warp + 1][lane - 1],
                   q[8][warp - 1][lane + 1], Su, Dux, Duy);
          group_down(o6, q[3][warp + 1][lane + 1], q[4][warp - 1][lane - 1], q[7][warp - 1][lane + 1],
                     q[9][warp + 1][lane - 1], Sd, Ddx, Ddy);
          const float v3 = q[0][warp - 1][lane], v4 = q[1][warp + 1][lane];
          const int z = t - 2;  // complete with its down group
          if (z >= z0) {
            const long long id = (long long)z * plane + col;
            const float a = add(A1, Sd);
            out[id] = F1;
            out[g.ps + id] = a;
            out[2 * g.ps + id] = add(JX1, Ddx);
            out[3 * g.ps + id] = add(JY1, Ddy);
            out[4 * g.ps + id] = sub(SU1, Sd);
            phi[id] = add(F1, a);
          }
          A1 = add(SU0, add(add(lx, ly), add(v3, v4)));
          JX1 = add(DX0, sub(lx, ly));
          JY1 = add(DY0, sub(v3, v4));
          SU1 = SU0;
          F1 = o0;
          SU0 = Su;
          DX0 = Dux;
          DY0 = Duy;
        }
      }
      if (p <= last) {
        const MubPlane p0 = mub_plane(smub[slot], lane + 1, warp + 1);
        if (t >= z0 - EDGE) {
          const float f0 = nf0, a = na, jx = njx, jy = njy, jz = njz, mu = nmu;
          if (p < last) fetch();
          const float dx = __fmaf_rn(G7, add(p0.X, p2.X), p1.gx);
          const float dy = __fmaf_rn(G7, add(p0.Y, p2.Y), p1.gy);
          const float dz = __fmaf_rn(G7, sub(p0.S, p2.S), mul(G1, sub(p0.c, p2.c)));
          float o[15];
          collide_sums3(c, f0, a, jx, jy, jz, mu, dx, dy, dz, o);
          if constexpr (LAST) {
            if (store) {
#pragma unroll
              for (int i = 0; i < 15; ++i) out[(long long)i * g.ps + (long long)t * plane + col] = o[i];
            }
          } else {
            float (*q)[MU_QY][MU_QX] = so[buf];
            q[0][warp][lane] = o[3];
            q[1][warp][lane] = o[4];
#pragma unroll
            for (int i = 7; i < 15; ++i) q[i - 5][warp][lane] = o[i];
            lx = __shfl_up_sync(0xffffffffu, o[1], 1);
            ly = __shfl_down_sync(0xffffffffu, o[2], 1);
            o0 = o[0];
            o5 = o[5];
            o6 = o[6];
          }
        }
        p2 = p1;
        p1 = p0;
      }
      slot = slot + 1 == MU_RING ? 0 : slot + 1;
      buf ^= 1;
    }
    lbch::cp_async_wait<0>();
  }
}

// ---------------------------------------------------------------- init and diagnostics

__global__ void __launch_bounds__(NX3) mu_alpha3_kernel(const double* __restrict__ phi, double* __restrict__ mua,
                                                        Grid3 g, double k, double beta4, int* bad) {
  Site s;
  if (!site_of(g, blockIdx.x, s)) return;
  const double c = phi[s.id];
  double lap = 0.0;
#pragma unroll
  for (int i = 1; i < 15; ++i) lap += 2.0 * wgt(i) * (phi[s.at(cx(i), cy(i), cz(i))] - c);
  lap *= 3.0;
  mua[s.id] = beta4 * c * (c * c - 1.0) - k * lap;
  if (!isfinite(c)) atomicOr(bad, 1);
}

// f = f^eq(phi0, mu_alpha) in the pre-streaming form (f*_i(x) streams to f_i(x + c_i)).
__global__ void __launch_bounds__(NX3) init3_kernel(const double* __restrict__ phi0, const double* __restrict__ mua,
                                                    Grid3 g, float* __restrict__ f) {
  Site s;
  if (!site_of(g, blockIdx.x, s)) return;
  f[s.id] = (float)(phi0[s.id] + (wgt(0) - 1.0) * mua[s.id]);
#pragma unroll
  for (int i = 1; i < 15; ++i) f[(long long)i * g.ps + s.id] = (float)(wgt(i) * mua[s.at(cx(i), cy(i), cz(i))]);
}

__global__ void __launch_bounds__(NX3) phi3_f64_kernel(const float* __restrict__ f, Grid3 g, double* __restrict__ phi) {
  Site s;
  if (!site_of(g, blockIdx.x, s)) return;
  double p = 0.0;
#pragma unroll
  for (int i = 0; i < 15; ++i) p += (double)f[(long long)i * g.ps + s.at(-cx(i), -cy(i), -cz(i))];
  phi[s.id] = p;
}

__global__ void mass3_kernel(const float* __restrict__ f, Grid3 g, double* __restrict__ partial) {
  __shared__ double sh[lbch::AUX_THREADS / 32];
  const long long n = (long long)g.nx * g.ny * g.nz;
  lbch::KahanF32 k;
  for (int i = 0; i < 15; ++i)
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
      k.add(f[(long long)i * g.ps + q]);
  const double acc = lbch::block_sum(k.value(), sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// Energy density (reading C11 in 3D) per node; blocks stride over the node-kernel
// blocks with NX3 threads each.
__global__ void __launch_bounds__(NX3) energy3_kernel(const float* __restrict__ phi, Grid3 g, lbch::EnergyConsts c,
                                                      int node_blocks, double* __restrict__ partial) {
  __shared__ double sh[NX3 / 32];
  double acc = 0.0;
  for (int b = blockIdx.x; b < node_blocks; b += gridDim.x) {
    Site s;
    if (!site_of(g, b, s)) continue;
    float dx, dy, dz, lap;
    stencil(phi, s, dx, dy, dz, lap);
    const float p0 = phi[s.id];
    const float g2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    float gamma = 1.0f;
    if (g2 >= 1e-12f) {
      const float rs = rsqrtf(g2);
      const float a = dx * rs, b2 = dy * rs, e = dz * rs;
      gamma = fmaf(c.alpha, fmaf(4.0f, fmaf(a * a, a * a, fmaf(b2 * b2, b2 * b2, e * e * e * e)), -3.0f), 1.0f);
    }
    const float q = p0 * p0 - 1.0f;
    const float F = c.beta * q * q;
    const float wv = fmaf(-c.cw, c.beta4 * p0 * q, lap);
    acc += (double)fmaf(gamma, fmaf(0.5f * c.k, g2, F), c.half_eps * wv * wv);
  }
  acc = lbch::block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

}  // namespace lbch3

struct lbch3_ctx {
  lbch3_params p;
  double k, beta, s[15];
  cudaStream_t stream;
  lbch3::Grid3 g;
  lbch3::Consts3 cs;
  float* buf[2];
  int cur;
  float *phi, *mua, *mub;
  double* stage;
  double* partial;
  double* result;
  int* flags;
  int blocks;      // blocks of the node kernels (NX3 x-nodes each)
  int red_blocks;  // blocks for the reductions
  lbch3::MuTiles mt;
  int mu_blocks;   // blocks of mu3_kernel
  lbch3::Sums3 sums;
  int st_blocks;   // blocks of stream3_kernel (moment form), and their runs
  lbch3::MuTiles st;
  bool fast;       // s_k = 1 except for phi and j: runs of steps in moment form
  bool has_state, failed;
  char err[512];
};

namespace {

const char* check3(const lbch3_params* p) {
  if (!p) return "params is NULL";
  if (p->nx < 1 || p->ny < 1 || p->nz < 1 || p->nx > 4096 || p->ny > 4096 || p->nz > 4096)
    return "nx, ny, nz must be in [1, 4096]";
  if ((long long)p->nx * p->ny * p->nz >= (1LL << 31)) return "nx*ny*nz must be < 2^31";
  if (!(p->M > 0.0) || !std::isfinite(p->M) || !(p->sigma > 0.0) || !(p->D > 0.0) || !(p->eps >= 0.0))
    return "M, sigma, D must be > 0 and eps >= 0";
  if (!(p->alpha >= 0.0 && p->alpha < 1.0)) return "alpha must be in [0, 1)";
  if (p->regularization < LBCH_REG_NONE || p->regularization > LBCH_REG_LINEAR) return "unknown regularization";
  if (p->flags & ~(unsigned)(LBCH_Q_LITERAL | LBCH_MU_NESTED | LBCH_S35_EXPLICIT)) return "unknown flag bits";
  for (int i = 1; i < 15; ++i) {
    if ((i == 3 || i == 5 || i == 7) && !(p->flags & LBCH_S35_EXPLICIT)) continue;
    if (!(p->s[i] > 0.0 && p->s[i] < 2.0)) return "relaxation rates s_1..s_14 must lie in (0, 2)";
  }
  return nullptr;
}

long long ps3(const lbch3_params* p) { return ((long long)p->nx * p->ny * p->nz + 63) / 64 * 64; }

bool cuda3_failed(lbch3_ctx* c, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return false;
  c->failed = true;
  snprintf(c->err, sizeof(c->err), "%s: %s", what, cudaGetErrorString(e));
  return true;
}

lbch_status pre3(lbch3_ctx* c, bool need_state) {
  if (!c) return LBCH_EINVAL;
  if (c->failed) return LBCH_ESTATE;
  if (need_state && !c->has_state) {
    snprintf(c->err, sizeof(c->err), "no state: call lbch3_init_field first");
    return LBCH_EINVAL;
  }
  return LBCH_OK;
}

lbch_status sync3(lbch3_ctx* c, const char* what) {
  if (cuda3_failed(c, cudaGetLastError(), what)) return LBCH_ECUDA;
  if (cuda3_failed(c, cudaStreamSynchronize(c->stream), what)) return LBCH_ECUDA;
  return LBCH_OK;
}

}  // namespace

extern "C" {

size_t lbch3_workspace_bytes(const lbch3_params* p) {
  if (check3(p)) return 0;
  const size_t ps = (size_t)ps3(p);
  return 2 * align_up(ps * 15 * sizeof(float)) + 3 * align_up(ps * sizeof(float)) + align_up(ps * sizeof(double)) +
         align_up(MAX_RED_BLOCKS * sizeof(double)) + align_up(8 * sizeof(double)) + align_up(16 * sizeof(int));
}

lbch_status lbch3_create(const lbch3_params* p, void* d_workspace, size_t bytes, void* cuda_stream, lbch3_ctx** out) {
  if (!out || check3(p)) return LBCH_EINVAL;
  const size_t need = lbch3_workspace_bytes(p);
  if (!d_workspace || bytes < need || ((uintptr_t)d_workspace % ALIGN) != 0) return LBCH_ENOMEM;
  lbch3_ctx* c = new (std::nothrow) lbch3_ctx();
  if (!c) return LBCH_ENOMEM;
  c->p = *p;
  c->beta = 3.0 * p->sigma / (4.0 * p->D);  // Eq. 5
  c->k = 3.0 * p->sigma * p->D / 8.0;
  for (int i = 0; i < 15; ++i) c->s[i] = p->s[i];
  if (!(p->flags & LBCH_S35_EXPLICIT)) c->s[3] = c->s[5] = c->s[7] = 1.0 / (3.0 * p->M + 0.5);
  c->stream = (cudaStream_t)cuda_stream;
  const long long ps = ps3(p);
  const int segs = (p->nx + lbch3::NX3 - 1) / lbch3::NX3;
  c->g = lbch3::Grid3{p->nx, p->ny, p->nz, segs, ps};
  char* q = (char*)d_workspace;
  for (int b = 0; b < 2; ++b) {
    c->buf[b] = (float*)q;
    q += align_up((size_t)ps * 15 * sizeof(float));
  }
  float** planes[3] = {&c->phi, &c->mua, &c->mub};
  for (float** pl : planes) {
    *pl = (float*)q;
    q += align_up((size_t)ps * sizeof(float));
  }
  c->stage = (double*)q;
  q += align_up((size_t)ps * sizeof(double));
  c->partial = (double*)q;
  q += align_up(MAX_RED_BLOCKS * sizeof(double));
  c->result = (double*)q;
  q += align_up(8 * sizeof(double));
  c->flags = (int*)q;
  const bool nested = p->flags & LBCH_MU_NESTED;
  const double eps = p->regularization == LBCH_REG_NONE ? 0.0 : p->eps;
  lbch3::Consts3& k = c->cs;
  k.k = (float)c->k;
  k.kq = (float)((p->flags & LBCH_Q_LITERAL) ? 1.0 : c->k);
  k.kiso = (float)(nested ? c->k : 0.0);
  k.beta4 = (float)(4.0 * c->beta);
  k.beta12 = (float)(12.0 * c->beta);
  k.alpha = (float)p->alpha;
  k.a16 = (float)(16.0 * p->alpha);
  k.eps = (float)eps;
  k.cw = p->regularization == LBCH_REG_LINEAR ? 0.0f : 1.0f;
  k.cfp = p->regularization == LBCH_REG_WILLMORE ? (float)eps : 0.0f;
  k.cnk = (float)(nested ? c->k : 0.0);
  for (int i = 0; i < 15; ++i) k.s[i] = (float)c->s[i];
  c->fast = true;
  for (int i = 1; i < 15; ++i)
    if (i != 3 && i != 5 && i != 7 && c->s[i] != 1.0) c->fast = false;
  c->blocks = segs * p->ny * p->nz;  // < 2^31: segs * nx-rows <= (nx + 127) / 128 * ny * nz
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms < 1) sms = 152;
  auto plan = [&](lbch3::MuTiles& mt, int warm) {
    mt.tiles_x = (p->nx + lbch3::MU_TX - 1) / lbch3::MU_TX;
    mt.tiles = mt.tiles_x * ((p->ny + lbch3::MU_TY - 1) / lbch3::MU_TY);
    return lbch3::plan_segments(mt.tiles, p->nz, warm, sms, &mt.len);
  };
  c->mu_blocks = plan(c->mt, 4);
  c->st_blocks = 0;
  if (c->fast) {
    for (int d = 0; d < 3; ++d) {
      const double sj = c->s[3 + 2 * d], nj = -(1.0 - 0.5 * sj) / 30.0, nq = 7.0 / 18.0 / 40.0;
      c->sums.cj[d] = (float)((1.0 - sj) / 10.0);
      c->sums.ga[d] = (float)(nj - 4.0 * nq);
      c->sums.gd[d] = (float)(nj + nq);
    }
    if (cudaFuncSetAttribute(lbch3::stream3_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             lbch3::ST_SMEM) != cudaSuccess ||
        cudaFuncSetAttribute(lbch3::stream3_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             lbch3::ST_SMEM) != cudaSuccess) {
      delete c;
      return LBCH_ECUDA;
    }
    c->st_blocks = plan(c->st, 5);
  }
  const long long nn = (long long)p->nx * p->ny * p->nz;
  long long rb = (nn + AUX_THREADS - 1) / AUX_THREADS;
  const long long cap = (long long)(sms > 0 ? sms : 152) * 8 < MAX_RED_BLOCKS ? (long long)(sms > 0 ? sms : 152) * 8
                                                                              : MAX_RED_BLOCKS;
  c->red_blocks = (int)(rb < cap ? rb : cap);
  c->cur = 0;
  c->has_state = false;
  c->failed = false;
  c->err[0] = 0;
  *out = c;
  return LBCH_OK;
}

lbch_status lbch3_init_field(lbch3_ctx* c, const double* h_phi0) {
  lbch_status st = pre3(c, false);
  if (st != LBCH_OK) return st;
  if (!h_phi0) return LBCH_EINVAL;
  const size_t n = (size_t)c->p.nx * c->p.ny * c->p.nz;
  c->has_state = false;
  double* mua = reinterpret_cast<double*>(c->buf[1]);  // the second population buffer is free during init
  if (cuda3_failed(c, cudaMemcpyAsync(c->stage, h_phi0, n * sizeof(double), cudaMemcpyHostToDevice, c->stream),
                   "init_field: copy") ||
      cuda3_failed(c, cudaMemsetAsync(c->flags, 0, sizeof(int), c->stream), "init_field: clear"))
    return LBCH_ECUDA;
  lbch3::mu_alpha3_kernel<<<c->blocks, lbch3::NX3, 0, c->stream>>>(c->stage, mua, c->g, c->k, 4.0 * c->beta, c->flags);
  lbch3::init3_kernel<<<c->blocks, lbch3::NX3, 0, c->stream>>>(c->stage, mua, c->g, c->buf[0]);
  int bad = 0;
  if (cuda3_failed(c, cudaMemcpyAsync(&bad, c->flags, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "init_field"))
    return LBCH_ECUDA;
  if ((st = sync3(c, "init_field")) != LBCH_OK) return st;
  if (bad) {
    snprintf(c->err, sizeof(c->err), "init_field: phi0 holds NaN or Inf");
    return LBCH_ENONFINITE;
  }
  c->cur = 0;
  c->has_state = true;
  return LBCH_OK;
}

lbch_status lbch3_step(lbch3_ctx* c, int64_t n) {
  lbch_status st = pre3(c, true);
  if (st != LBCH_OK) return st;
  if (n < 0) return LBCH_EINVAL;
  if (c->fast && n > 0) {
    // Moment planes (5 each, ping-pong) in the population buffer that does not hold the state.
    float* f = c->buf[c->cur];
    float* m[2] = {c->buf[c->cur ^ 1], c->buf[c->cur ^ 1] + 5 * c->g.ps};
    launch_dep(lbch3::gather3_kernel, c->blocks, lbch3::NX3, 0, c->stream, f, c->g, m[0], c->phi);
    for (int64_t t = 0; t < n; ++t) {
      const int k = (int)(t & 1);
      launch_dep(lbch3::mu3_kernel, c->mu_blocks, lbch3::MU_THREADS, 0, c->stream, c->phi, c->g, c->cs, c->mt, c->mua, c->mub);
      if (t + 1 < n)
        launch_dep(lbch3::stream3_kernel<false>, c->st_blocks, lbch3::MU_THREADS, lbch3::ST_SMEM, c->stream, m[k], c->mub, c->mua, c->g, c->sums, c->st, m[k ^ 1], c->phi);
      else
        launch_dep(lbch3::stream3_kernel<true>, c->st_blocks, lbch3::MU_THREADS, lbch3::ST_SMEM, c->stream, m[k], c->mub, c->mua, c->g, c->sums, c->st, f, nullptr);
    }
  }
  for (int64_t t = 0; !c->fast && t < n; ++t) {
    const float* src = c->buf[c->cur];
    float* dst = c->buf[c->cur ^ 1];
    lbch3::phi3_kernel<<<c->blocks, lbch3::NX3, 0, c->stream>>>(src, c->g, c->phi);
    lbch3::mu3_kernel<<<c->mu_blocks, lbch3::MU_THREADS, 0, c->stream>>>(c->phi, c->g, c->cs, c->mt, c->mua, c->mub);
    lbch3::collide3_kernel<<<c->blocks, lbch3::NX3, 0, c->stream>>>(src, c->mub, c->mua, c->g, c->cs, dst);
    c->cur ^= 1;
  }
  if (cuda3_failed(c, cudaGetLastError(), "step: launch")) return LBCH_ECUDA;
  return LBCH_OK;
}

lbch_status lbch3_get_field(lbch3_ctx* c, double* h_phi) {
  lbch_status st = pre3(c, true);
  if (st != LBCH_OK) return st;
  if (!h_phi) return LBCH_EINVAL;
  const size_t n = (size_t)c->p.nx * c->p.ny * c->p.nz;
  lbch3::phi3_f64_kernel<<<c->blocks, lbch3::NX3, 0, c->stream>>>(c->buf[c->cur], c->g, c->stage);
  if (cuda3_failed(c, cudaMemcpyAsync(h_phi, c->stage, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream),
                   "get_field: copy"))
    return LBCH_ECUDA;
  return sync3(c, "get_field");
}

lbch_status lbch3_mass(lbch3_ctx* c, double* out) {
  lbch_status st = pre3(c, true);
  if (st != LBCH_OK) return st;
  if (!out) return LBCH_EINVAL;
  lbch3::mass3_kernel<<<c->red_blocks, AUX_THREADS, 0, c->stream>>>(c->buf[c->cur], c->g, c->partial);
  final_sum_kernel<<<1, 1024, 0, c->stream>>>(c->partial, c->red_blocks, c->result);
  if (cuda3_failed(c, cudaMemcpyAsync(out, c->result, sizeof(double), cudaMemcpyDeviceToHost, c->stream), "mass"))
    return LBCH_ECUDA;
  if ((st = sync3(c, "mass")) != LBCH_OK) return st;
  return std::isfinite(*out) ? LBCH_OK : LBCH_ENONFINITE;
}

lbch_status lbch3_free_energy(lbch3_ctx* c, double* out) {
  lbch_status st = pre3(c, true);
  if (st != LBCH_OK) return st;
  if (!out) return LBCH_EINVAL;
  lbch3::phi3_kernel<<<c->blocks, lbch3::NX3, 0, c->stream>>>(c->buf[c->cur], c->g, c->phi);
  EnergyConsts ec;
  const double eps = c->p.regularization == LBCH_REG_NONE ? 0.0 : c->p.eps;
  ec.k = (float)c->k;
  ec.beta = (float)c->beta;
  ec.beta4 = (float)(4.0 * c->beta);
  ec.alpha = (float)c->p.alpha;
  ec.half_eps = (float)(0.5 * eps);
  ec.cw = c->p.regularization == LBCH_REG_LINEAR ? 0.0f : 1.0f;
  lbch3::energy3_kernel<<<c->red_blocks, lbch3::NX3, 0, c->stream>>>(c->phi, c->g, ec, c->blocks, c->partial);
  final_sum_kernel<<<1, 1024, 0, c->stream>>>(c->partial, c->red_blocks, c->result + 1);
  if (cuda3_failed(c, cudaMemcpyAsync(out, c->result + 1, sizeof(double), cudaMemcpyDeviceToHost, c->stream),
                   "free_energy"))
    return LBCH_ECUDA;
  if ((st = sync3(c, "free_energy")) != LBCH_OK) return st;
  return std::isfinite(*out) ? LBCH_OK : LBCH_ENONFINITE;
}

const char* lbch3_last_error(const lbch3_ctx* c) { return c ? c->err : "context is NULL"; }

void lbch3_destroy(lbch3_ctx* c) { delete c; }

}  // extern "C"
