// Fused time step of the MRT lattice Boltzmann scheme for the anisotropic
// Cahn-Hilliard equation (arXiv 2501.03759, Section 3), one kernel per step.
//
// What one launch computes, for every node x of the periodic grid:
//   f_in,i(x)  = f*_i(x - c_i)                      pull streaming of the previous step
//   phi        = sum_i f_in,i                       Eq. 22
//   grad phi, lap phi                               Eq. 26a, 26b
//   n, gamma(n), P grad_n gamma, Q, f, f', w, mu_a  Eqs. 2, 6, 15, 9, 13, 16
//   mu_beta = (gamma-1) f - div Q + eps(lap w - f' w)   Eqs. 13, 16 (split reading)
//   g = grad mu_beta, F_m = M F                     Eqs. 26a, 19, 25
//   m* = m - S(m - m^eq) + (I - S/2) F_m, f* = M^-1 m*   Eqs. 17, 23, 25
// and stores f* (the state before streaming) in the other buffer.
//
// Work decomposition (GB300): one warp owns a strip of 128 consecutive columns
// (4 per lane, so rows move as 16-byte vectors) and sweeps a segment of rows top to
// bottom. phi is needed up to 3 nodes away from an output node, so each warp keeps
// a rolling three-row window of every stencil in registers: when the phi row r
// arrives it completes grad/lap phi of row r-1, mu_beta of row r-2 and
// grad mu_beta of row r-3, and collides row r-3. Left/right neighbours come from
// warp shuffles; the 4 strip columns at each edge are halo, so a strip yields 120
// output columns. Rows arrive by cp.async into a per-warp shared-memory ring of
// landing slots, fetched PF_DIST rows ahead of use; a row stays in the ring until
// its collision three rows later (each lane reads back only what it copied, so no
// barrier is needed). No tensor cores: the 9x9 moment transform is a handful of
// adds with constant +-1/+-2 entries.
#pragma once

#include <type_traits>

#include "lbch_f2.cuh"
#include "lbch_lattice.cuh"

namespace lbch {

constexpr int STRIP_W = 128;                 // columns per warp strip
constexpr int HALO_W = 4;                    // halo columns on each side
constexpr int OUT_W = STRIP_W - 2 * HALO_W;  // output columns per strip
// A field exactly STRIP_W wide is one strip that covers the whole periodic row: the lane
// neighbour exchanges below rotate (lane 0's left neighbour is lane 31), so every column is
// computed from its true periodic neighbours and all STRIP_W columns are output. In a strip
// of a wider (or narrower) field the rotated-in values reach only halo columns: an output
// column depends on columns at most HALO_W (the stencil depth) away, inside the strip.
__host__ __device__ constexpr int n_strips_for(int nx) { return nx == STRIP_W ? 1 : (nx + OUT_W - 1) / OUT_W; }
constexpr int STEP_WARPS = 4;                // warps per CTA

// Which collision a launch runs. R_ONES and R_SUMS: s_k = 1 for every moment but j_x and j_y, the
// reduced (FAST) collision. R_SUMS is its FP32 form from sums of the populations (collide_sums),
// of contexts that step in moment form; the 16-bit storages have one form, R_ONES.
enum : int { R_GENERAL = 0, R_ONES = 1, R_SUMS = 2 };

// Moment form of the state (relaxation rates of the FAST collision). With s_k = 1 for every
// moment but j_x and j_y, Eq. 17 reads of a node's populations only phi, j_x and j_y (and, to
// close the rest population, the sum of the moving ones). A run of steps therefore need not
// bring the nine populations to memory in between: every step but the last stores the sums its
// own populations stream to, and the last one stores populations again. The planes of a node (FP32) are
//   FP32 storage     f_0, a = sum_{i >= 1} f_i, j_x, j_y   (phi = f_0 + a): 32 B read and written
//                    per node update instead of 72;
//   16-bit storages  phi, j_x, j_y, summed from the rounded deviations the populations would
//                    have been stored as: 24 B instead of 48.
// The sums are formed from the same FP32 values in the same order as the ones a pull of the
// stored populations forms, so a run gives bit for bit what its steps give one by one. A run is
// gather (pull the populations, store the sums), then steps from sums to sums, then one from
// sums to populations.
__host__ __device__ constexpr int m_planes(int st) { return st == ST_F32 ? 4 : 3; }
// Pipeline depth per storage (measured on GB300 at 8192^2): fetch one row ahead and collide
// row r-3 right after its grad mu_beta. The 16-bit storages keep 12 warps per SM (their
// landing slots are smaller); colliding row r-4 first in the iteration with no prefetch
// instead ran 10% slower once their per-row instruction count had come down, and one row
// of prefetch with r-4 needs a sixth slot, which costs a CTA per SM; so does two rows of
// prefetch with r-3 (0.547 -> 0.710 ms per 8192^2 BF16 launch).
template <int ST, bool VEC, bool MI = false>
struct Pipe {
  static constexpr bool DEV16 = ST != ST_F32;
  static constexpr int PF_DIST = MI ? 2 : 1;          // rows fetched ahead of the phi row
  static constexpr int LAG = 3;                         // phi row r collides row r - LAG
  static constexpr int SLOTS = PF_DIST + 1 + LAG;       // rows held per warp: r-LAG .. r+PF_DIST
  // 16-byte units per slot: 9 per lane for FP32 planes (or pulled values on the scalar
  // path); rest + anchor + 8 half-width deviation planes = 6 per lane for vector DEV; the
  // M_PLANES moment planes for moment input.
  static constexpr int SLOT_F4 = (MI ? m_planes(ST) : (DEV16 && VEC ? 6 : 9)) * 32;
  // CTAs per SM the launch bounds plan for. Moment form holds more per thread (the streaming
  // accumulators): FP32 fits 168 registers without a spill, the 16-bit storages take 206 and
  // spill at 168 (8192^2 BF16: 0.526 ms at 3 CTAs, 0.457 ms at 2).
  static constexpr int MIN_CTAS = MI ? (DEV16 ? 2 : 3) : ((DEV16 && VEC) ? 3 : 2);
};
template <int ST, bool VEC, bool MI = false>
constexpr int step_smem() { return STEP_WARPS * Pipe<ST, VEC, MI>::SLOTS * Pipe<ST, VEC, MI>::SLOT_F4 * 16; }

// Constants shared by every field a launch steps.
struct StepArgs {
  // Chemical potential constants.
  float k;     // gradient energy coefficient (Eq. 5)
  float kq;    // factor on |grad phi| P grad_n gamma in Q (k, or 1 for the literal Eq. 15)
  float kiso;  // k times the isotropic part kept in Q (0 split, k nested)
  float beta4, beta12;  // 4 beta and 12 beta (f and f')
  float eps;   // eps on lap w (0 without regularisation)
  float cw;    // w = lap phi - cw f  (1 Willmore, 0 linear)
  float cfp;   // eps on f' w (Willmore only)
  float cnk;   // k lap phi added to mu_beta in nested form
  // Collision: n_k = (m*_k)/|row k of M|^2 in terms of m_k, m^eq_k and g.
  float c1a, c1b, c2a, c2b, c3a, c3g, c4a, c4g, c5a, c5g, c6a, c6g, c7, c8;
  // The constants of pointwise_scaled and collide_sums, where the stencils are left unnormalised.
  float k_s, kq_s, kiso_s, beta4_s, eps_e, eps_c;  // k/12, kq/12, kiso/12, 48 beta, eps/6, 2 eps/3
  float cxg, cug, cyg, cvg;                        // g's in n_3 - 2 n_4, n_3 + n_4 (n_5, n_6), over 144
};

// One periodic field: its buffers, its size and work split, and its anisotropy.
struct Field {
  Buf src, dst;
  long long ps;  // plane stride in elements
  int nx, ny;
  int n_strips, seg_len;
  float alpha, a16;  // alpha and 16 alpha (Eq. 6)
  int mp;  // row pitch of the moment planes (in the population buffers), in elements; a multiple of 8
};

__device__ __forceinline__ int imod(int v, int n) {
  int r = v % n;
  return r < 0 ? r + n : r;
}

// The value of the lane to the left (lane 31 for lane 0) and to the right (lane 0 for 31).
__device__ __forceinline__ float from_lane_left(float v) {
  return __shfl_sync(FULL, v, (threadIdx.x + 31) & 31);
}
__device__ __forceinline__ float from_lane_right(float v) {
  return __shfl_sync(FULL, v, (threadIdx.x + 1) & 31);
}

// How a lane's 4 columns travel as two pairs: plain, (0, 1) and (2, 3), or interleaved (IL),
// (0, 2) and (1, 3). Interleaved, the right neighbours of the first pair are the second pair and
// the left neighbours of the second pair are the first one, as they stand: a neighbour exchange
// builds two new pairs instead of three and a pull shift one instead of two, and a pair whose
// halves lie in different registers costs a move each. The moment planes are stored in
// interleaved order (each aligned group of 4 columns as 0, 2, 1, 3), so their rows load as pairs.
// Left/right neighbour sums and differences of a per-column quantity over the strip:
// s_j = q_{j-1} + q_{j+1}, d_j = q_{j+1} - q_{j-1} for this lane's columns j = 0..3, with the
// outer neighbours from the adjacent lanes.
template <bool IL>
__device__ __forceinline__ void neighbours(const F2 (&q)[2], F2 (&s)[2], F2 (&d)[2]) {
  const float left = from_lane_left(q[1].y);
  const float right = from_lane_right(q[0].x);
  if constexpr (IL) {
    const F2 L = f2(left, q[1].x), R = f2(q[0].y, right);
    s[0] = L + q[1];
    s[1] = q[0] + R;
    d[0] = q[1] - L;
    d[1] = R - q[0];
  } else {
    const F2 A = f2(left, q[0].x), B = f2(q[0].y, q[1].x), C = f2(q[1].y, right);
    s[0] = A + B;
    s[1] = B + C;
    d[0] = B - A;
    d[1] = C - B;
  }
}

// Per-lane addressing of the strip.
struct Cols {
  long long c0;  // aligned first column (vector path)
  int cs[6];     // columns xs + 4 lane + k - 1, k = 0..5 (scalar path), mod nx
};

// Row copies ask L2 to fetch 256-byte blocks (.L2::256B): a warp's row of one plane is 512
// (FP32) or 256 (16-bit) contiguous bytes, so each miss brings in the neighbouring sectors the
// warp reads next. Measured on GB300 at 8192^2: 0.844 -> 0.821 ms per FP32 launch and
// 0.548 -> 0.542 ms per BF16 launch (a 128-byte hint gave no FP32 gain).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global.L2::256B [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// One warp's landing slot for one phi row r, as 16-byte units [q][lane]:
//   vector F32:  q = i holds plane i of row r - c_iy at the strip's aligned columns (raw f*);
//   vector DEV:  q = 0 the rest plane of row r, q = 1 the anchor plane of row r, then (as
//                8-byte units [k][lane]) the deviation plane k+1 of row r - c_(k+1)y;
//   scalar path: q = i holds f_in,i itself (pulled and rebuilt when it was fetched).
// Fetches phi row r (rows ro_m = r-1, ro_0 = r, ro_p = r+1) into a slot; the vector path
// copies asynchronously (cp.async), the scalar path loads and stores synchronously.
template <int ST, bool VEC>
__device__ __forceinline__ void issue_row(const Field& fd, float4* slot, int lane, long long ro_m,
                                          long long ro_0, long long ro_p, const Cols& cl) {
#define LBCH_RO(I) (cy(I) == 1 ? ro_m : (cy(I) == -1 ? ro_p : ro_0))
  if constexpr (VEC) {
    if constexpr (ST == ST_F32) {
#pragma unroll
      for (int i = 0; i < 9; ++i)
        cp_async16(slot + i * 32 + lane, fd.src.f32 + (long long)i * fd.ps + LBCH_RO(i) + cl.c0);
    } else {
      cp_async16(slot + lane, fd.src.f32 + ro_0 + cl.c0);
      cp_async16(slot + 32 + lane, fd.src.f32 + fd.ps + ro_0 + cl.c0);
      uint2* ds = reinterpret_cast<uint2*>(slot + 64);
#pragma unroll
      for (int i = 1; i < 9; ++i)
        cp_async8(ds + (i - 1) * 32 + lane, fd.src.dev + (long long)(i - 1) * fd.ps + LBCH_RO(i) + cl.c0);
    }
  } else {
    float v[9][4];  // every load is issued before the first store to the slot
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const long long ro = LBCH_RO(i);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = cl.cs[j - cx(i) + 1];  // pull: f_in,i(x) = f*_i(x - c_i)
        if constexpr (ST == ST_F32) {
          v[i][j] = fd.src.f32[(long long)i * fd.ps + ro + c];
        } else if (i == 0) {
          v[i][j] = fd.src.f32[ro + c];
        } else {  // w_i times the anchor of this node, plus the deviation from the source node
          v[i][j] = fmaf((float)wgt(i), fd.src.f32[fd.ps + ro_0 + cl.cs[j + 1]],
                         Dev<ST>::load(fd.src.dev[(long long)(i - 1) * fd.ps + ro + c]));
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) slot[i * 32 + lane] = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
  }
#undef LBCH_RO
}

// Pull shift along x of a per-column quantity of the strip: column j takes column j - 1
// (c_x = 1) or column j + 1 (c_x = -1).
template <bool IL>
__device__ __forceinline__ void from_left(F2 (&v)[2]) {
  const float prev = from_lane_left(v[1].y);
  if constexpr (IL) {
    const F2 p = f2(prev, v[1].x);
    v[1] = v[0];
    v[0] = p;
  } else {
    v[1] = f2(v[0].y, v[1].x);
    v[0] = f2(prev, v[0].x);
  }
}
template <bool IL>
__device__ __forceinline__ void from_right(F2 (&v)[2]) {
  const float next = from_lane_right(v[0].x);
  if constexpr (IL) {
    const F2 p = f2(v[0].y, next);
    v[0] = v[1];
    v[1] = p;
  } else {
    v[0] = f2(v[0].y, v[1].x);
    v[1] = f2(v[1].y, next);
  }
}

// Four consecutive columns (a population plane's 16 bytes) to pairs and back.
template <bool IL>
__device__ __forceinline__ void to_pairs(const float4 t, F2 (&v)[2]) {
  v[0] = IL ? f2(t.x, t.z) : f2(t.x, t.y);
  v[1] = IL ? f2(t.y, t.w) : f2(t.z, t.w);
}
template <bool IL>
__device__ __forceinline__ float4 from_pairs(const F2 (&v)[2]) {
  return IL ? make_float4(v[0].x, v[1].x, v[0].y, v[1].y) : make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}
// Two pairs as they stand: a moment plane's 16 bytes in interleaved form, a slot's cached values.
__device__ __forceinline__ void load_pairs(const float4 t, F2 (&v)[2]) {
  v[0] = f2(t.x, t.y);
  v[1] = f2(t.z, t.w);
}
__device__ __forceinline__ float4 store_pairs(const F2 (&v)[2]) { return make_float4(v[0].x, v[0].y, v[1].x, v[1].y); }

// Four consecutive 16-bit deviations to pairs, in storage units, and back (rounded as a pair of
// consecutive columns in one conversion; `scaled`: FP16 values already carry the storage scale).
template <int ST, bool IL>
__device__ __forceinline__ void widen4(const uint2 raw, F2 (&v)[2]) {
  float c[4];
  Dev<ST>::raw2(raw.x, c[0], c[1]);
  Dev<ST>::raw2(raw.y, c[2], c[3]);
  to_pairs<IL>(make_float4(c[0], c[1], c[2], c[3]), v);
}
template <int ST, bool IL>
__device__ __forceinline__ uint2 round4(const F2 (&v)[2]) {
  const float4 c = from_pairs<IL>(v);
  if constexpr (ST == ST_F16) return make_uint2(Dev<ST>::pack2_scaled(c.x, c.y), Dev<ST>::pack2_scaled(c.z, c.w));
  else return make_uint2(Dev<ST>::pack2(c.x, c.y), Dev<ST>::pack2(c.z, c.w));
}

// f_in,I at this lane's 4 columns from a landed slot.
template <int ST, bool VEC, bool IL, int I>
__device__ __forceinline__ void read_row(const float4* slot, int lane, F2 (&v)[2]) {
  constexpr bool REBUILD = VEC && ST != ST_F32 && I != 0;
  if constexpr (!REBUILD) {
    to_pairs<IL>(slot[I * 32 + lane], v);
  } else {  // deviations of the source nodes (row r - c_Iy), shifted below
    const uint2 raw = reinterpret_cast<const uint2*>(slot + 64)[(I - 1) * 32 + lane];
    widen4<ST, IL>(raw, v);
    if constexpr (Dev<ST>::UNSCALE != 1.0f) {
      v[0] = splat(Dev<ST>::UNSCALE) * v[0];
      v[1] = splat(Dev<ST>::UNSCALE) * v[1];
    }
  }
  if constexpr (VEC) {  // the pull shift along x happens here, one shuffle per plane
    if constexpr (cx(I) == 1) {
      from_left<IL>(v);
    } else if constexpr (cx(I) == -1) {
      from_right<IL>(v);
    }
  }
  if constexpr (REBUILD) {  // f*_I(y - c_I) = w_I anchor(y) + d_I(y - c_I)
    const F2 w = splat((float)wgt(I));
    F2 m[2];
    to_pairs<IL>(slot[32 + lane], m);
    v[0] = fma2(w, m[0], v[0]);
    v[1] = fma2(w, m[1], v[1]);
  }
}

// Grouped deviation sums of a landed DEV row at this lane's 4 columns, pulled along x, in
// storage units (FP16 values still carry their scale). The eight moving planes fall into
// three groups by c_x: gp = d1 + d5 + d8 (c_x = 1), gm = d3 + d6 + d7 (c_x = -1) and
// g0 = d2 + d4; with H also their c_y-signed parts hp = d5 - d8, hm = d6 - d7 and
// h0 = d2 - d4. A group shares one pull shift, so it takes one shuffle instead of one per
// plane. Every population arriving at a node is rebuilt on that node's anchor, the weights
// w_1..w_8 sum to 5/9, and the anchor terms cancel in j_x and j_y, so
//   phi = f*_0 + (5/9) anchor + (gp + gm + g0),  j_x = gp - gm,  j_y = hp + hm + h0.
struct DevSums {
  F2 gp[2], gm[2], g0[2], hp[2], hm[2], h0[2];
};
template <int ST, bool IL, bool H>
__device__ __forceinline__ void dev_sums(const float4* slot, int lane, DevSums& s) {
  const uint2* ds = reinterpret_cast<const uint2*>(slot + 64);
  F2 d[9][2];
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    widen4<ST, IL>(ds[(i - 1) * 32 + lane], d[i]);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    s.gp[k] = (d[1][k] + d[5][k]) + d[8][k];
    s.gm[k] = (d[3][k] + d[6][k]) + d[7][k];
    s.g0[k] = d[2][k] + d[4][k];
    if constexpr (H) {
      s.hp[k] = d[5][k] - d[8][k];
      s.hm[k] = d[6][k] - d[7][k];
      s.h0[k] = d[2][k] - d[4][k];
    }
  }
  from_left<IL>(s.gp);
  from_right<IL>(s.gm);
  if constexpr (H) {
    from_left<IL>(s.hp);
    from_right<IL>(s.hm);
  }
}

// phi at this lane's columns of a landed DEV row from its rest population, anchor and
// group sums.
template <int ST, bool IL>
__device__ __forceinline__ void dev_phi(const float4* slot, int lane, const DevSums& s, F2 (&ph)[2]) {
  F2 rest[2], anc[2];
  to_pairs<IL>(slot[lane], rest);
  to_pairs<IL>(slot[32 + lane], anc);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    F2 g = (s.gp[k] + s.gm[k]) + s.g0[k];
    if constexpr (Dev<ST>::UNSCALE != 1.0f) g = splat(Dev<ST>::UNSCALE) * g;
    ph[k] = fma2(splat(5.0f / 9.0f), anc[k], rest[k]) + g;
  }
}

// rsqrt.approx.ftz takes subnormal arguments for zero; the arguments here are at least 1e-12.
__device__ __forceinline__ float rsqrt_normal(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// Pointwise part at two nodes: Q (Eq. 15 reading), w, mu_alpha (Eq. 16) and the local part A
// of mu_beta (Eq. 13 minus Eq. 16's mu_alpha).
__device__ __forceinline__ void pointwise(const StepArgs& a, const Field& fd, F2 phi, F2 dx, F2 dy, F2 lap,
                                          F2& Qx, F2& Qy, F2& w, F2& A, F2& mua) {
  const F2 g2 = fma2(dx, dx, dy * dy);
  const bool okx = g2.x >= 1e-12f, oky = g2.y >= 1e-12f;  // n = 0, gamma = 1 below this
  const F2 rs = f2(rsqrt_normal(okx ? g2.x : 1.0f), rsqrt_normal(oky ? g2.y : 1.0f));
  const F2 n1 = dx * rs, n2 = dy * rs;  // Eq. 2
  const F2 n1s = n1 * n1, n2s = n2 * n2;
  const F2 S4 = fma2(n1s, n1s, n2s * n2s);
  F2 gm1 = splat(fd.alpha) * fma2(splat(4.0f), S4, splat(-3.0f));  // gamma - 1, Eq. 6
  // k_q |grad phi| P grad_n gamma with grad_n gamma = 16 alpha n^3, P = I - n n^T.
  F2 t = splat(a.kq * fd.a16) * (g2 * rs);
  if (!okx) gm1.x = t.x = 0.0f;
  if (!oky) gm1.y = t.y = 0.0f;
  const F2 kg = fma2(splat(a.k), gm1, splat(a.kiso));
  Qx = fma2(kg, dx, t * (n1 * (n1s - S4)));
  Qy = fma2(kg, dy, t * (n2 * (n2s - S4)));
  const F2 phi2 = phi * phi;
  const F2 fb = (splat(a.beta4) * phi) * (phi2 - splat(1.0f));  // f = F'(phi), Eq. 9
  const F2 fp = fma2(splat(a.beta12), phi2, splat(-a.beta4));   // f'(phi), Eq. 13
  w = fma2(splat(-a.cw), fb, lap);
  mua = fma2(splat(-a.k), lap, fb);
  A = fma2(gm1, fb, fma2(splat(-a.cfp) * fp, w, splat(a.cnk) * lap));
}

// The same for R_SUMS, from unnormalised stencils (dx, dy and lap 12 times their values): Q
// itself, and w, mu_alpha and A 12 times theirs. The factors of 1/12 sit
// in the constants, n is the same ratio, and the guard compares 144 |grad phi|^2. The step is
// bound by the FMA pipe (a packed operation holds it two cycles), and unnormalised stencils take
// 9 of about 125 operations per pair off it.
__device__ __forceinline__ void pointwise_scaled(const StepArgs& a, const Field& fd, F2 phi, F2 dx, F2 dy, F2 lap,
                                                 F2& Qx, F2& Qy, F2& w, F2& A, F2& mua) {
  const F2 g2 = fma2(dx, dx, dy * dy);
  const bool okx = g2.x >= 144e-12f, oky = g2.y >= 144e-12f;  // n = 0, gamma = 1 below this
  const F2 rs = f2(rsqrt_normal(okx ? g2.x : 1.0f), rsqrt_normal(oky ? g2.y : 1.0f));
  const F2 n1 = dx * rs, n2 = dy * rs;  // Eq. 2
  const F2 n1s = n1 * n1, n2s = n2 * n2;
  const F2 S4 = fma2(n1s, n1s, n2s * n2s);
  F2 gm1 = splat(fd.alpha) * fma2(splat(4.0f), S4, splat(-3.0f));  // gamma - 1, Eq. 6
  F2 t = splat(a.kq_s * fd.a16) * (g2 * rs);
  if (!okx) gm1.x = t.x = 0.0f;
  if (!oky) gm1.y = t.y = 0.0f;
  const F2 kg = fma2(splat(a.k_s), gm1, splat(a.kiso_s));
  Qx = fma2(kg, dx, t * (n1 * (n1s - S4)));
  Qy = fma2(kg, dy, t * (n2 * (n2s - S4)));
  const F2 phi2 = phi * phi;
  const F2 fb = (splat(a.beta4_s) * phi) * fma2(phi, phi, splat(-1.0f));  // 12 f
  const F2 fp = fma2(splat(a.beta12), phi2, splat(-a.beta4));     // f'(phi), Eq. 13
  w = fma2(splat(-a.cw), fb, lap);
  mua = fma2(splat(-a.k), lap, fb);
  A = fma2(gm1, fb, fma2(splat(-a.cfp) * fp, w, splat(a.cnk) * lap));
}

// Eq. 17 at two nodes in moment space (Eqs. 23, 25) with the closed forms
// m^eq = (phi, -4 phi + 2 mu_a, 4 phi - 3 mu_a, 0, ...) and
// M F = (0, 0, 0, -g_x/3, g_x/3, -g_y/3, g_y/3, 0, 0), and M^-1 = M^T diag(1/|row|^2).
// FAST: s_1 = s_2 = s_4 = s_6 = s_7 = s_8 = 1, so those moments take their (forced)
// equilibrium and need not be formed; the result equals the general path's, whose
// (1 - s_k) m_k terms are then exactly zero.
// FAST collision from the three moments it needs, phi = m_0, j_x = m_3 and j_y = m_5 (the
// others take their equilibrium): o[1..8] of f*; o[0] is left to the caller.
__device__ __forceinline__ void collide_fast(const StepArgs& a, F2 phi, F2 m3, F2 m5, F2 mua, F2 gx, F2 gy,
                                             F2 (&o)[9]) {
  const F2 n0 = phi * splat(1.0f / 9.0f);
  const F2 n1 = splat(a.c1b) * fma2(splat(2.0f), mua, splat(-4.0f) * phi);
  const F2 n2 = splat(a.c2b) * fma2(splat(-3.0f), mua, splat(4.0f) * phi);
  const F2 n4 = splat(a.c4g) * gx, n6 = splat(a.c6g) * gy;
  const F2 n3 = fma2(splat(a.c3a), m3, splat(a.c3g) * gx);
  const F2 n5 = fma2(splat(a.c5a), m5, splat(a.c5g) * gy);
  const F2 A0 = fma2(splat(-2.0f), n2, n0 - n1);
  const F2 X = fma2(splat(-2.0f), n4, n3), Y = fma2(splat(-2.0f), n6, n5);
  o[1] = A0 + X;
  o[3] = A0 - X;
  o[2] = A0 + Y;
  o[4] = A0 - Y;
  const F2 D0 = fma2(splat(2.0f), n1, n0 + n2);
  const F2 U = n3 + n4, V = n5 + n6;
  const F2 P = U + V, Mv = U - V;
  o[5] = D0 + P;
  o[7] = D0 - P;
  o[6] = D0 - Mv;
  o[8] = D0 + Mv;
}

template <bool FAST>
__device__ __forceinline__ void collide(const StepArgs& a, const F2 (&f)[9], F2 mua, F2 gx, F2 gy, F2 (&o)[9],
                                        F2& phi_out) {
  const F2 ab = f[1] + f[3], bb = f[2] + f[4];
  const F2 Sa = ab + bb;
  const F2 e = f[5] + f[7], h = f[6] + f[8];
  const F2 Sd = e + h;
  const F2 phi = (f[0] + Sa) + Sd;
  const F2 x1 = f[1] - f[3], y1 = f[2] - f[4];
  const F2 p = f[5] - f[7], q = f[6] - f[8];
  const F2 pm = p - q, pp = p + q;
  const F2 m3 = x1 + pm, m5 = y1 + pp;
  if constexpr (FAST) {
    collide_fast(a, phi, m3, m5, mua, gx, gy, o);
  } else {
    const F2 n0 = phi * splat(1.0f / 9.0f);
    const F2 m1 = fma2(splat(-4.0f), f[0], fma2(splat(2.0f), Sd, splat(0.0f) - Sa));
    const F2 m2 = fma2(splat(4.0f), f[0], fma2(splat(-2.0f), Sa, Sd));
    const F2 m4 = fma2(splat(-2.0f), x1, pm), m6 = fma2(splat(-2.0f), y1, pp);
    const F2 m7 = ab - bb, m8 = e - h;
    const F2 n1 = fma2(splat(a.c1a), m1, splat(a.c1b) * fma2(splat(2.0f), mua, splat(-4.0f) * phi));
    const F2 n2 = fma2(splat(a.c2a), m2, splat(a.c2b) * fma2(splat(-3.0f), mua, splat(4.0f) * phi));
    const F2 n4 = fma2(splat(a.c4a), m4, splat(a.c4g) * gx);
    const F2 n6 = fma2(splat(a.c6a), m6, splat(a.c6g) * gy);
    const F2 n7 = splat(a.c7) * m7;
    const F2 n8 = splat(a.c8) * m8;
    const F2 n3 = fma2(splat(a.c3a), m3, splat(a.c3g) * gx);
    const F2 n5 = fma2(splat(a.c5a), m5, splat(a.c5g) * gy);
    const F2 A0 = fma2(splat(-2.0f), n2, n0 - n1);
    const F2 B = A0 + n7, C = A0 - n7;
    const F2 X = fma2(splat(-2.0f), n4, n3), Y = fma2(splat(-2.0f), n6, n5);
    o[1] = B + X;
    o[3] = B - X;
    o[2] = C + Y;
    o[4] = C - Y;
    const F2 D0 = fma2(splat(2.0f), n1, n0 + n2);
    const F2 E = D0 + n8, G = D0 - n8;
    const F2 U = n3 + n4, V = n5 + n6;
    const F2 P = U + V, Mv = U - V;
    o[5] = E + P;
    o[7] = E - P;
    o[6] = G - Mv;
    o[8] = G + Mv;
  }
  // Row 0 of M^-1 m* would be n0 - 4 n1 + 4 n2, but FP32 n0 = phi/9 carries a fixed
  // relative bias. Since sum_i f*_i = sum_i f_i (m_0 is conserved, Eq. 34), the rest
  // population takes what the moving ones gave up: f*_0 = f_0 + sum_{i>=1} (f_i - f*_i).
  // The differences of nearby values are exact and small, so the only rounding at the
  // scale of phi is the final add.
  o[0] = f[0] + ((((f[1] - o[1]) + (f[2] - o[2])) + ((f[3] - o[3]) + (f[4] - o[4]))) +
                 (((f[5] - o[5]) + (f[6] - o[6])) + ((f[7] - o[7]) + (f[8] - o[8]))));
  phi_out = phi;
}

template <bool IL>
__device__ __forceinline__ void unpair(const F2 (&v)[2], float (&s)[4]) {
  const float4 t = from_pairs<IL>(v);
  s[0] = t.x;
  s[1] = t.y;
  s[2] = t.z;
  s[3] = t.w;
}

// What R_SUMS needs of a node. phi = f0 + a.
struct Sums {
  F2 f0[2], a[2], jx[2], jy[2];
};

// A node's arriving populations by the row they come from: up (c_y = 1, from the row below),
// level, and down (c_y = -1). S is the sum of a group, D its c_x = 1 member less its c_x = -1
// one; a = (S_up + S_level) + S_down, j_x = (D_up + D_level) + D_down, j_y = S_up - S_down. The
// streaming of the moment form forms the same groups in the same order.
// S = (r + l) + v and D = r - l, r and l pulled along x (v: the group's c_x = 0 member, or null).
template <bool IL, bool PULL>
__device__ __forceinline__ void group(F2 (&r)[2], F2 (&l)[2], const F2 (*v)[2], F2 (&S)[2], F2 (&D)[2]) {
  if constexpr (PULL) {
    from_left<IL>(r);
    from_right<IL>(l);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    S[k] = r[k] + l[k];
    if (v) S[k] = S[k] + (*v)[k];
    D[k] = r[k] - l[k];
  }
}
// The sums of a landed row's populations.
template <bool VEC, bool IL>
__device__ __forceinline__ void f32_sums(const float4* slot, int lane, Sums& s) {
  F2 f[9][2], Su[2], Du[2], Sl[2], Dl[2], Sd[2], Dd[2];
#pragma unroll
  for (int i = 0; i < 9; ++i) to_pairs<IL>(slot[i * 32 + lane], f[i]);
  group<IL, VEC>(f[5], f[6], &f[2], Su, Du);
  group<IL, VEC>(f[1], f[3], nullptr, Sl, Dl);
  group<IL, VEC>(f[8], f[7], &f[4], Sd, Dd);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    s.f0[k] = f[0][k];
    s.a[k] = (Su[k] + Sl[k]) + Sd[k];
    s.jx[k] = (Du[k] + Dl[k]) + Dd[k];
    s.jy[k] = Su[k] - Sd[k];
  }
}

// The R_SUMS collision (mua 12 times mu_alpha, gx and gy 144 times
// grad mu_beta: unnormalised stencils). The terms in phi of m_0, m_1 and m_2 cancel in the moving
// populations, f*_i = w_i mu_alpha plus the flux and forcing parts, and the rest population closes
// the mass: f*_0 = f_0 + d, d = a - sum_{i >= 1} f*_i (a and the sum are of the size of mu_alpha).
// What rounding that add drops (at most half an ulp of f_0, found exactly) goes to the four axis
// populations in equal parts, so that sum_i f*_i = sum_i f_i to rounding at the scale of mu_alpha.
// Dropping it instead loses updates below half an ulp of f_0 with the same sign step after step:
// the 64^2 droplet's mass drifted 5e-6 over 2000 steps.
__device__ __forceinline__ void collide_sums(const StepArgs& a, F2 f0, F2 am, F2 jx, F2 jy, F2 mua, F2 gx, F2 gy,
                                             F2 (&o)[9]) {
  const F2 A0 = splat(1.0f / 108.0f) * mua, D0 = splat(1.0f / 432.0f) * mua;
  const F2 Jx = splat(a.c3a) * jx, Jy = splat(a.c5a) * jy;
  const F2 X = fma2(splat(a.cxg), gx, Jx), U = fma2(splat(a.cug), gx, Jx);
  const F2 Y = fma2(splat(a.cyg), gy, Jy), V = fma2(splat(a.cvg), gy, Jy);
  o[1] = A0 + X;
  o[3] = A0 - X;
  o[2] = A0 + Y;
  o[4] = A0 - Y;
  const F2 P = U + V, Mv = U - V;
  o[5] = D0 + P;
  o[7] = D0 - P;
  o[6] = D0 - Mv;
  o[8] = D0 + Mv;
  const F2 d = am - (((o[1] + o[3]) + (o[2] + o[4])) + ((o[5] + o[7]) + (o[6] + o[8])));
  o[0] = f0 + d;
  const F2 r = d - (o[0] - f0);
#pragma unroll
  for (int i = 1; i <= 4; ++i) o[i] = fma2(splat(0.25f), r, o[i]);
}

// The 16-bit deviations of a collided row at this lane's columns: packed bits (as stored), the
// same values widened in storage units (raw), and the rest population that closes the sum.
template <int ST, bool IL>
__device__ __forceinline__ void quantise(const F2 (&o)[9][2], const F2 (&dmu)[8][2], const F2 (&phi)[2],
                                         uint2 (&pk)[8], F2 (&raw)[8][2], F2 (&rest)[2]) {
  // f*_i as its reader rebuilds it (anchor term plus the stored deviation) closes the rest
  // population.
  F2 sum[2];
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const F2 w = splat((float)wgt(i)), nw = splat(-(float)wgt(i));
    F2 dv[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      dv[k] = fma2(nw, dmu[i - 1][k], o[i][k]);
      if constexpr (ST == ST_F16) dv[k] = splat(F16_SCALE) * dv[k];
    }
    pk[i - 1] = round4<ST, IL>(dv);
    widen4<ST, IL>(pk[i - 1], raw[i - 1]);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      F2 back = raw[i - 1][k];
      if constexpr (Dev<ST>::UNSCALE != 1.0f) back = splat(Dev<ST>::UNSCALE) * back;
      const F2 rb = fma2(w, dmu[i - 1][k], back);
      sum[k] = i == 1 ? rb : sum[k] + rb;
    }
  }
  rest[0] = phi[0] - sum[0];
  rest[1] = phi[1] - sum[1];
}

// Stores one collided row. DEV storage keeps the rest population and this node's
// anchor in FP32 and d_i = f*_i - w_i anchor(x + c_i) in 16 bits; the rest population
// is closed on the values a reader will rebuild, so sum_i f*_i = phi holds (mass is
// conserved to FP32 rounding, not 16-bit rounding). dmu[i-1] is the anchor of the node
// population i streams to, at this lane's columns.
template <int ST, bool IL>
__device__ __forceinline__ void store_row_vec(const Field& fd, long long ro, long long col, const F2 (&o)[9][2],
                                              const F2 (&mua)[2], const F2 (&dmu)[8][2], const F2 (&phi)[2]) {
  if constexpr (ST == ST_F32) {
#pragma unroll
    for (int i = 0; i < 9; ++i)
      *reinterpret_cast<float4*>(fd.dst.f32 + (long long)i * fd.ps + ro + col) =
          from_pairs<IL>(o[i]);
  } else {
    uint2 pk[8];
    F2 raw[8][2], rest[2];
    quantise<ST, IL>(o, dmu, phi, pk, raw, rest);
    // Streaming stores (st.global.cs, evict first in L2): 0.542 -> 0.538 ms per 8192^2 BF16
    // launch on GB300. The FP32 planes keep plain stores: streaming ones ran 0.821 -> 0.834 ms.
    __stcs(reinterpret_cast<float4*>(fd.dst.f32 + ro + col), from_pairs<IL>(rest));
    __stcs(reinterpret_cast<float4*>(fd.dst.f32 + fd.ps + ro + col), from_pairs<IL>(mua));
#pragma unroll
    for (int i = 0; i < 8; ++i)
      __stcs(reinterpret_cast<uint2*>(fd.dst.dev + (long long)i * fd.ps + ro + col), pk[i]);
  }
}

// Scalar-path store for columns that may be partly out of range (grids whose width is not a
// multiple of 4): the first nvalid of the 4 columns at col0.
template <int ST, bool IL>
__device__ __forceinline__ void store_row_masked(const Field& fd, long long ro, int col0, int nvalid,
                                                 const F2 (&o2)[9][2], const F2 (&mua2)[2],
                                                 const F2 (&dmu2)[8][2], const F2 (&phi2)[2]) {
  float o[9][4], mua[4], dmu[8][4], phi[4];
#pragma unroll
  for (int i = 0; i < 9; ++i) unpair<IL>(o2[i], o[i]);
#pragma unroll
  for (int i = 0; i < 8; ++i) unpair<IL>(dmu2[i], dmu[i]);
  unpair<IL>(mua2, mua);
  unpair<IL>(phi2, phi);
  if constexpr (ST == ST_F32) {
    for (int j = 0; j < 4; ++j)
      if (j < nvalid)
#pragma unroll
        for (int i = 0; i < 9; ++i) fd.dst.f32[(long long)i * fd.ps + ro + col0 + j] = o[i][j];
  } else {
    using D = Dev<ST>;
    for (int j = 0; j < 4; ++j) {
      if (j >= nvalid) break;
      float sum = 0.0f;
#pragma unroll
      for (int i = 1; i < 9; ++i) {
        const float w = (float)wgt(i);
        const uint16_t d = D::store(fmaf(-w, dmu[i - 1][j], o[i][j]));
        sum += fmaf(w, dmu[i - 1][j], D::load(d));
        fd.dst.dev[(long long)(i - 1) * fd.ps + ro + col0 + j] = d;
      }
      fd.dst.f32[ro + col0 + j] = phi[j] - sum;
      fd.dst.f32[fd.ps + ro + col0 + j] = mua[j];
    }
  }
}

// A landed row of populations can leave in its slot, when the row's phi is formed, what its collision
// three rows later reads (over values that nothing reads after that, each lane over its own): the
// four sums of a Sums (R_SUMS), or phi, j_x and j_y (16-bit storages with the FAST rates).
template <int ST, bool VEC, int RT>
struct SlotCache {
  static constexpr bool ON = ST == ST_F32 ? RT == R_SUMS : (RT != R_GENERAL && VEC);
};
__device__ __forceinline__ F2* cache_of(float4* slot) { return reinterpret_cast<F2*>(slot + 64); }
__device__ __forceinline__ const F2* cache_of(const float4* slot) { return reinterpret_cast<const F2*>(slot + 64); }

// Interleaved pairs everywhere but where FP32 population rows are read (a load of 4 consecutive
// columns is two plain pairs as it lands, and 9 rows of them would each have to be moved).
template <int ST, bool MI>
struct Pairs {
  static constexpr bool IL = MI || ST != ST_F32;
};

// Position of column c (counted from an aligned one) in a moment row.
__device__ __forceinline__ int moment_pos(int c) { return (c & ~3) | ((c & 1) << 1) | ((c >> 1) & 1); }

// Moment rows: lane's 4 columns c0 .. c0 + 3 (periodic) of every plane of the row at element ro, 16
// bytes at a time where they are an aligned group (plain). On ragged rows (nx % 4 != 0) the columns
// across the seam are not, and go one by one; this costs the warps at the seam a few instructions
// per row. (Rows with periodic copies of the columns at the seam, stored with them, kept every load
// aligned, but their stores took the warps at the seam longer than a row's arithmetic, and a step
// lasts as long as its slowest warp: 1001 x 517 20.2 us a step, 12.6 us this way; 2001 x 800 33 and 20.)
template <int ST>
__device__ __forceinline__ void issue_row_m(const float* base, long long mps, long long ro, int c0, int nx, bool plain,
                                            float4* slot, int lane) {
  if (plain) {
#pragma unroll
    for (int q = 0; q < m_planes(ST); ++q) cp_async16(slot + q * 32 + lane, base + q * mps + ro + c0);
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = c0 + k >= nx ? c0 + k - nx : c0 + k;
      const float* src = base + ro + moment_pos(c);
#pragma unroll
      for (int q = 0; q < m_planes(ST); ++q)
        cp_async4(reinterpret_cast<float*>(slot + q * 32 + lane) + moment_pos(k), src + q * mps);
    }
  }
}

// phi of the landed row in `slot` at this lane's columns; leaves the SlotCache values there.
template <int ST, bool VEC, int RT, bool MI>
__device__ __forceinline__ void land_row(float4* slot, int lane, F2 (&ph)[2]) {
  constexpr bool IL = Pairs<ST, MI>::IL;
  if constexpr (MI) {
    load_pairs(slot[lane], ph);
    if constexpr (ST == ST_F32) {
      F2 a[2];
      load_pairs(slot[32 + lane], a);
      ph[0] = ph[0] + a[0];
      ph[1] = ph[1] + a[1];
    }
  } else if constexpr (SlotCache<ST, VEC, RT>::ON && ST == ST_F32) {
    Sums s;
    f32_sums<VEC, IL>(slot, lane, s);
    slot[32 + lane] = store_pairs(s.a);
    slot[64 + lane] = store_pairs(s.jx);
    slot[96 + lane] = store_pairs(s.jy);
    ph[0] = s.f0[0] + s.a[0];
    ph[1] = s.f0[1] + s.a[1];
  } else if constexpr (VEC && ST != ST_F32) {  // grouped: one shuffle per c_x group
    DevSums ds;
    dev_sums<ST, IL, SlotCache<ST, VEC, RT>::ON>(slot, lane, ds);
    dev_phi<ST, IL>(slot, lane, ds, ph);
    if constexpr (SlotCache<ST, VEC, RT>::ON) {
      F2* cache = cache_of(slot);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        F2 jx = ds.gp[k] - ds.gm[k], jy = (ds.hp[k] + ds.hm[k]) + ds.h0[k];
        if constexpr (Dev<ST>::UNSCALE != 1.0f) {
          jx = splat(Dev<ST>::UNSCALE) * jx;
          jy = splat(Dev<ST>::UNSCALE) * jy;
        }
        cache[k * 32 + lane] = ph[k];
        cache[(2 + k) * 32 + lane] = jx;
        cache[(4 + k) * 32 + lane] = jy;
      }
    }
  } else {
    F2 v[2];
    read_row<ST, VEC, IL, 0>(slot, lane, ph);
#define LBCH_PULL(I)                   \
  read_row<ST, VEC, IL, I>(slot, lane, v); \
  ph[0] = ph[0] + v[0];                \
  ph[1] = ph[1] + v[1];
    LBCH_PULL(1) LBCH_PULL(2) LBCH_PULL(3) LBCH_PULL(4)
    LBCH_PULL(5) LBCH_PULL(6) LBCH_PULL(7) LBCH_PULL(8)
#undef LBCH_PULL
  }
}

// Collides a row from its landing slot: o[i] = f*_i and phic its phi (16-bit storages; o[0] is
// left to the quantisation there when the sums were cached).
template <int ST, bool VEC, int RT, bool MI>
__device__ __forceinline__ void collide_row(const StepArgs& a, const float4* slot, int lane, const F2 (&mu_c)[2],
                                            const F2 (&gx)[2], const F2 (&gy)[2], F2 (&o)[9][2], F2 (&phic)[2]) {
  constexpr bool IL = Pairs<ST, MI>::IL;
  if constexpr (ST == ST_F32 && (MI || SlotCache<ST, VEC, RT>::ON)) {
    Sums s;
    if constexpr (MI)
      load_pairs(slot[lane], s.f0);
    else
      to_pairs<IL>(slot[lane], s.f0);  // the landed plane itself
    load_pairs(slot[32 + lane], s.a);
    load_pairs(slot[64 + lane], s.jx);
    load_pairs(slot[96 + lane], s.jy);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      F2 oj[9];
      collide_sums(a, s.f0[k], s.a[k], s.jx[k], s.jy[k], mu_c[k], gx[k], gy[k], oj);
#pragma unroll
      for (int i = 0; i < 9; ++i) o[i][k] = oj[i];
    }
  } else if constexpr (MI || SlotCache<ST, VEC, RT>::ON) {
    F2 jx[2], jy[2];
    if constexpr (MI) {
      load_pairs(slot[lane], phic);
      load_pairs(slot[32 + lane], jx);
      load_pairs(slot[64 + lane], jy);
    } else {
      const F2* cache = cache_of(slot);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        phic[k] = cache[k * 32 + lane];
        jx[k] = cache[(2 + k) * 32 + lane];
        jy[k] = cache[(4 + k) * 32 + lane];
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      F2 oj[9];
      collide_fast(a, phic[k], jx[k], jy[k], mu_c[k], gx[k], gy[k], oj);
      o[0][k] = splat(0.0f);  // the quantisation closes the rest population from phi
#pragma unroll
      for (int i = 1; i < 9; ++i) o[i][k] = oj[i];
    }
  } else {
    F2 fr[9][2];
    read_row<ST, VEC, IL, 0>(slot, lane, fr[0]);
    read_row<ST, VEC, IL, 1>(slot, lane, fr[1]);
    read_row<ST, VEC, IL, 2>(slot, lane, fr[2]);
    read_row<ST, VEC, IL, 3>(slot, lane, fr[3]);
    read_row<ST, VEC, IL, 4>(slot, lane, fr[4]);
    read_row<ST, VEC, IL, 5>(slot, lane, fr[5]);
    read_row<ST, VEC, IL, 6>(slot, lane, fr[6]);
    read_row<ST, VEC, IL, 7>(slot, lane, fr[7]);
    read_row<ST, VEC, IL, 8>(slot, lane, fr[8]);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      F2 f[9], oj[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) f[i] = fr[i][k];
      collide<RT != R_GENERAL>(a, f, mu_c[k], gx[k], gy[k], oj, phic[k]);
#pragma unroll
      for (int i = 0; i < 9; ++i) o[i][k] = oj[i];
    }
  }
}

// Anchors of the destination nodes x + c_i: dmu[i-1] from mu_alpha of the rows row-1, row, row+1
// (16-bit storages: interleaved pairs).
__device__ __forceinline__ void anchors_of(const F2 (&mu_m)[2], const F2 (&mu_c)[2], const F2 (&mu_p)[2],
                                           F2 (&dmu)[8][2]) {
  F2 l[3][2], r[3][2];  // columns j - 1 and j + 1 of rows row-1, row, row+1
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const F2(&m)[2] = q == 0 ? mu_m : (q == 1 ? mu_c : mu_p);
    l[q][0] = r[q][0] = m[0];
    l[q][1] = r[q][1] = m[1];
    from_left<true>(l[q]);
    from_right<true>(r[q]);
  }
#pragma unroll
  for (int i = 1; i < 9; ++i)
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int q = 1 + cy(i);
      const F2(&m)[2] = q == 0 ? mu_m : (q == 1 ? mu_c : mu_p);
      dmu[i - 1][k] = cx(i) == 1 ? r[q][k] : (cx(i) == -1 ? l[q][k] : m[k]);
    }
}

// Streaming in moment form, one collided row c after another. Row y of the next state takes the
// c_y = 1 populations of row y - 1, the c_y = 0 ones of row y and the c_y = -1 ones of row
// y + 1: after row c is collided, row y = c - 1 is complete.
// FP32 storage: the groups of f32_sums, pulled along x as they are formed.
struct StreamF32 {
  F2 a[2], jx[2], Su[2], f0[2];  // row y: up + level so far, the up sum, the rest population
  F2 Sn[2], Dn[2];               // the up group of row y (for row y + 1)
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 2; ++k) a[k] = jx[k] = Su[k] = f0[k] = Sn[k] = Dn[k] = splat(0.0f);
  }
  // The sums of row c - 1 into m, given the populations o of row c.
  __device__ __forceinline__ void push(F2 (&o)[9][2], Sums& m) {
    F2 Sd[2], Dd[2], Sl[2], Dl[2];
    group<true, true>(o[8], o[7], &o[4], Sd, Dd);
    group<true, true>(o[1], o[3], nullptr, Sl, Dl);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      m.f0[k] = f0[k];
      m.a[k] = a[k] + Sd[k];
      m.jx[k] = jx[k] + Dd[k];
      m.jy[k] = Su[k] - Sd[k];
      f0[k] = o[0][k];
      a[k] = Sn[k] + Sl[k];
      jx[k] = Dn[k] + Dl[k];
      Su[k] = Sn[k];
    }
    group<true, true>(o[5], o[6], &o[2], Sn, Dn);
  }
};
// 16-bit storages: the groups of dev_sums on the rounded deviations v[i - 1] (storage units).
struct StreamDev {
  F2 s15[2], s36[2];       // v1 + v5 and v3 + v6 of row y (v5, v6 streamed from row y - 1)
  F2 rest[2];              // rest population of row y
  F2 p2[2], p5[2], p6[2];  // the upward deviations of row y
  F2 q2[2], q5[2], q6[2];  // and of row y - 1
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < 2; ++k)
      s15[k] = s36[k] = rest[k] = p2[k] = p5[k] = p6[k] = q2[k] = q5[k] = q6[k] = splat(0.0f);
  }
  // phi, j_x and j_y of row c - 1 (whose anchor is anc), given the deviations and rest of row c.
  template <int ST>
  __device__ __forceinline__ void push(const F2 (&v)[8][2], const F2 (&r)[2], const F2 (&anc)[2], F2 (&phi)[2],
                                       F2 (&jx)[2], F2 (&jy)[2]) {
    F2 gp[2], gm[2], g0[2], hp[2], hm[2], h0[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      gp[k] = s15[k] + v[7][k];
      gm[k] = s36[k] + v[6][k];
      g0[k] = q2[k] + v[3][k];
      hp[k] = q5[k] - v[7][k];
      hm[k] = q6[k] - v[6][k];
      h0[k] = q2[k] - v[3][k];
    }
    from_left<true>(gp);
    from_left<true>(hp);
    from_right<true>(gm);
    from_right<true>(hm);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      F2 g = (gp[k] + gm[k]) + g0[k];
      jx[k] = gp[k] - gm[k];
      jy[k] = (hp[k] + hm[k]) + h0[k];
      if constexpr (Dev<ST>::UNSCALE != 1.0f) {
        g = splat(Dev<ST>::UNSCALE) * g;
        jx[k] = splat(Dev<ST>::UNSCALE) * jx[k];
        jy[k] = splat(Dev<ST>::UNSCALE) * jy[k];
      }
      phi[k] = fma2(splat(5.0f / 9.0f), anc[k], rest[k]) + g;
      s15[k] = v[0][k] + p5[k];
      s36[k] = v[2][k] + p6[k];
      rest[k] = r[k];
      q2[k] = p2[k];
      q5[k] = p5[k];
      q6[k] = p6[k];
      p2[k] = v[1][k];
      p5[k] = v[4][k];
      p6[k] = v[5][k];
    }
  }
};

// One plane of a moment row at columns col0 .. col0 + 3 (the last ones may be the row's padding).
template <bool IL>
__device__ __forceinline__ void store_moment(float* row, int col0, const F2 (&v)[2]) {
  *reinterpret_cast<float4*>(row + col0) = IL ? store_pairs(v) : make_float4(v[0].x, v[1].x, v[0].y, v[1].y);
}

// One warp's work: the rows [seg * seg_len, ...) of strip `strip` of field fd. MI: the input is
// in moment form; MO: the output is.
template <int ST, bool VEC, int RT, bool MI, bool MO>
__device__ __forceinline__ void step_warp(const StepArgs& a, const Field& fd, int strip, int seg, float4* slots,
                                          int lane) {
  static_assert(!MI || (ST == ST_F32 ? RT == R_SUMS : RT == R_ONES && VEC), "moment form");
  // The pull, the stencils (3) and the push together reach 5 columns, the strip's halo is 4.
  static_assert(MI || !MO, "moment output needs moment input");
  using PP = Pipe<ST, VEC, MI>;
  constexpr int PF_DIST = PP::PF_DIST, COLLIDE_LAG = PP::LAG, SLOTS = PP::SLOTS, SLOT_F4 = PP::SLOT_F4;
  constexpr int FIRST = MO ? 4 : 3;  // phi rows start at y0 - FIRST (streaming needs one more row)
  const int y0 = seg * fd.seg_len;
  const int y1 = min(y0 + fd.seg_len, fd.ny);
  const bool full_row = fd.nx == STRIP_W;  // one strip over the whole periodic row
  const int xs = full_row ? 0 : strip * OUT_W - HALO_W;  // strip start column (before wrap)

  Cols cl;
  int mcol = 0;
  bool plain = true;
  if constexpr (MI) {
    mcol = imod(xs + 4 * lane, fd.nx);
    plain = (mcol & 3) == 0 && mcol + 4 <= fd.nx;
  } else {
    cl.c0 = imod(xs + 4 * lane, fd.nx);
#pragma unroll
    for (int k = 0; k < 6; ++k) cl.cs[k] = imod(xs + 4 * lane + k - 1, fd.nx);
  }
  const long long mps = (long long)fd.mp * fd.ny;

  // Output columns of this lane: strip columns 4 lane + j in [HALO_W, STRIP_W - HALO_W), or
  // all of them for a full row.
  const int ocol0 = xs + 4 * lane;  // global column of element 0
  const bool lane_out = full_row || (lane >= 1 && lane <= 30 && ocol0 < fd.nx);
  const int nvalid = min(4, fd.nx - ocol0);

  // Rolling accumulators (see the header comment): index 1 = row completing next, 0 = row
  // after; U and V hold the y-difference terms of the last two rows (phi and mu_beta).
  F2 Ax1[2], Al1[2], Ax0[2], U1[2], U0[2], php[2];
  F2 T1[2], T0[2];
  F2 Gx1[2], Gx0[2], V1[2], V0[2];
  F2 mu1[2], mu2[2], mu3[2];  // mu_alpha of rows r-2, r-3, r-4
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    Ax1[k] = Al1[k] = Ax0[k] = U1[k] = U0[k] = php[k] = splat(0.0f);
    T1[k] = T0[k] = Gx1[k] = Gx0[k] = V1[k] = V0[k] = splat(0.0f);
    mu1[k] = mu2[k] = mu3[k] = splat(0.0f);
  }
  constexpr bool IL = Pairs<ST, MI>::IL;
  constexpr bool SC = RT == R_SUMS;  // unnormalised stencils (pointwise_scaled)
  std::conditional_t<ST == ST_F32, StreamF32, StreamDev> st;
  if constexpr (MO) st.clear();

  // phi rows y0 - FIRST .. ; phi row r collides row r - COLLIDE_LAG.
  // Two rows per loop iteration in moment form: the rolling accumulators then change roles instead
  // of registers (8192^2 FP32 0.424 -> 0.404 ms, 2048^2 37.1 -> 35.6 us when it was tried; three
  // rows gave no more). The walk is rounded up to an even number of rows: a separate last row
  // would be compiled without what only a next row uses, and a packed multiply that is left with
  // a single use may be contracted with its add to one fma, which rounds differently. (Seen in a
  // run that then differed from its single steps; the bitwise tests hold even and odd walks.)
  constexpr int UNR = MI && MO ? 2 : 1;
  const int n_it = ((y1 - y0) + 2 * FIRST + UNR - 1) / UNR * UNR;
  const int it_end = (y1 - y0) + 2 * FIRST;  // iterations past it store nothing
  static_assert(COLLIDE_LAG == 3, "row r-3 collides right after its grad mu_beta");
  // Rows r-1, r, r+1 (mod ny) of the next phi row to fetch.
  int fm = imod(y0 - FIRST - 1, fd.ny), f0 = imod(y0 - FIRST, fd.ny), fp = imod(y0 - FIRST + 1, fd.ny);
  auto fetch_next = [&](float4* slot) {
    if constexpr (MI)
      issue_row_m<ST>(fd.src.f32, mps, (long long)f0 * fd.mp, mcol, fd.nx, plain, slot, lane);
    else
      issue_row<ST, VEC>(fd, slot, lane, (long long)fm * fd.nx, (long long)f0 * fd.nx, (long long)fp * fd.nx, cl);
    fm = f0;
    f0 = fp;
    fp = fp + 1 == fd.ny ? 0 : fp + 1;
  };
  wait_previous();
#pragma unroll
  for (int d = 0; d < PF_DIST; ++d) {
    if (d < n_it) fetch_next(slots + d * SLOT_F4);
    cp_async_commit();
  }
  const F2 K12 = splat(1.0f / 12.0f), K6 = splat(1.0f / 6.0f), K3 = splat(1.0f / 3.0f);
  const F2 K23 = splat(2.0f / 3.0f), KM103 = splat(-10.0f / 3.0f), K2 = splat(2.0f), K4 = splat(4.0f), K8 = splat(8.0f);
  const F2 EPS = splat(a.eps);
  int s_cur = 0, s_pf = PF_DIST, s_col = SLOTS - COLLIDE_LAG;  // slots of rows r, r+PF_DIST, r-LAG
  auto row_step = [&](int it) {
    // 1. Fetch row r + PF_DIST.
    if (it + PF_DIST < n_it) fetch_next(slots + s_pf * SLOT_F4);
    cp_async_commit();
    // 2. Wait for row r; pull it and sum phi (Eq. 22).
    cp_async_wait<PF_DIST>();
    F2 ph[2];
    land_row<ST, VEC, RT, MI>(slots + s_cur * SLOT_F4, lane, ph);
    // 3. grad phi and lap phi of row r-1 (Eq. 26a, 26b), rolling over rows.
    F2 dx[2], dy[2], lp[2];
    {
      F2 s[2], d[2];
      neighbours<IL>(ph, s, d);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const F2 e = SC ? d[k] : d[k] * K12;
        const F2 u = SC ? fma2(K4, ph[k], s[k]) : fma2(s[k], K12, ph[k] * K3);
        const F2 c = SC ? fma2(K8, s[k], ph[k] * splat(-40.0f)) : fma2(s[k], K23, ph[k] * KM103);
        dx[k] = Ax1[k] + e;
        dy[k] = u - U1[k];
        lp[k] = fma2(K2, u, Al1[k]);  // the Laplacian's weights for the rows r, r - 2 are twice u's
        Ax1[k] = fma2(K4, e, Ax0[k]);
        U1[k] = U0[k];
        Al1[k] = fma2(K2, U0[k], c);
        Ax0[k] = e;
        U0[k] = u;
      }
    }
    // 4. Pointwise at row r-1.
    F2 Qx[2], Qy[2], w[2], Aq[2], mun[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if constexpr (SC)
        pointwise_scaled(a, fd, php[k], dx[k], dy[k], lp[k], Qx[k], Qy[k], w[k], Aq[k], mun[k]);
      else
        pointwise(a, fd, php[k], dx[k], dy[k], lp[k], Qx[k], Qy[k], w[k], Aq[k], mun[k]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) php[k] = ph[k];
    // 5. mu_beta of row r-2: A - div Q + eps lap w (Eq. 26 on Q and w).
    F2 mub[2];
    {
      F2 sx[2], dqx[2], sqy[2], dqy[2], sw[2], dw[2];
      neighbours<IL>(Qx, sx, dqx);
      neighbours<IL>(Qy, sqy, dqy);
      neighbours<IL>(w, sw, dw);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if constexpr (SC) {  // 12 times mu_beta
          const F2 bb = fma2(K4, Qy[k], sqy[k]), z = fma2(K4, w[k], sw[k]);
          const F2 c = fma2(splat(-5.0f), w[k], sw[k]);
          mub[k] = fma2(splat(a.eps_e), z, T1[k] - (dqx[k] + bb));
          T1[k] = T0[k] + fma2(splat(a.eps_c), c, fma2(splat(-4.0f), dqx[k], Aq[k]));
          T0[k] = fma2(splat(a.eps_e), z, bb - dqx[k]);
          continue;
        }
        const F2 aa = dqx[k] * K12;
        const F2 bb = fma2(sqy[k], K12, Qy[k] * K3);
        const F2 cc = EPS * fma2(sw[k], K6, w[k] * K23);
        mub[k] = T1[k] + ((cc - aa) - bb);
        T1[k] = T0[k] + fma2(EPS, fma2(sw[k], K23, w[k] * KM103), fma2(splat(-4.0f), aa, Aq[k]));
        T0[k] = (bb - aa) + cc;
      }
    }
    // 6. grad mu_beta of row r-3 (Eq. 26a).
    F2 gx[2], gy[2];
    {
      F2 s[2], d[2];
      neighbours<IL>(mub, s, d);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const F2 e = SC ? d[k] : d[k] * K12;
        const F2 u = SC ? fma2(K4, mub[k], s[k]) : fma2(s[k], K12, mub[k] * K3);
        gx[k] = Gx1[k] + e;
        gy[k] = u - V1[k];
        Gx1[k] = fma2(K4, e, Gx0[k]);
        V1[k] = V0[k];
        Gx0[k] = e;
        V0[k] = u;
      }
    }
    // 7. Collide row r-3; store it, or stream it and store row r-4 of the next state.
    if (it >= 6) {
      F2 o[9][2], phic[2], dmu[8][2];
      collide_row<ST, VEC, RT, MI>(a, slots + s_col * SLOT_F4, lane, mu2, gx, gy, o, phic);
      if constexpr (ST != ST_F32) anchors_of(mu3, mu2, mu1, dmu);
      if constexpr (!MO) {
        if (lane_out && (UNR == 1 || it < it_end)) {
          const long long ro = (long long)(y0 + it - 6) * fd.nx;
          if constexpr (VEC) {
            store_row_vec<ST, IL>(fd, ro, ocol0, o, mu2, dmu, phic);
          } else {
            store_row_masked<ST, IL>(fd, ro, ocol0, nvalid, o, mu2, dmu, phic);
          }
        }
      } else {
        const bool out = it >= 8 && it < it_end && lane_out;
        float* row = fd.dst.f32 + (long long)(y0 + it - 8) * fd.mp;
        if constexpr (ST == ST_F32) {
          Sums m;
          st.push(o, m);
          if (out) {
            store_moment<IL>(row, ocol0, m.f0);
            store_moment<IL>(row + mps, ocol0, m.a);
            store_moment<IL>(row + 2 * mps, ocol0, m.jx);
            store_moment<IL>(row + 3 * mps, ocol0, m.jy);
          }
        } else {
          uint2 pk[8];
          F2 raw[8][2], rest[2], m0[2], jx[2], jy[2];
          quantise<ST, IL>(o, dmu, phic, pk, raw, rest);
          st.template push<ST>(raw, rest, mu3, m0, jx, jy);
          if (out) {
            store_moment<IL>(row, ocol0, m0);
            store_moment<IL>(row + mps, ocol0, jx);
            store_moment<IL>(row + 2 * mps, ocol0, jy);
          }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      mu3[k] = mu2[k];
      mu2[k] = mu1[k];
      mu1[k] = mun[k];
    }
    s_cur = s_cur + 1 == SLOTS ? 0 : s_cur + 1;
    s_pf = s_pf + 1 == SLOTS ? 0 : s_pf + 1;
    s_col = s_col + 1 == SLOTS ? 0 : s_col + 1;
  };
  for (int it = 0; it < n_it; it += UNR) {
    row_step(it);
    if constexpr (UNR == 2) row_step(it + 1);
  }
  cp_async_wait<0>();
}

// Populations to moment planes: the rows [seg * seg_len, ...) of strip `strip`, pulled and
// summed as the step's own landing does.
template <int ST, bool VEC>
__device__ __forceinline__ void gather_warp(const Field& fd, int strip, int seg, float4* slots, int lane) {
  using PP = Pipe<ST, VEC, false>;
  constexpr int PF = PP::SLOTS - 1;  // rows in flight: a slot is free once its row is stored
  const int y0 = seg * fd.seg_len;
  const int n_it = min(fd.seg_len, fd.ny - y0);
  const bool full_row = fd.nx == STRIP_W;
  const int xs = full_row ? 0 : strip * OUT_W - HALO_W;
  Cols cl;
  cl.c0 = imod(xs + 4 * lane, fd.nx);
#pragma unroll
  for (int k = 0; k < 6; ++k) cl.cs[k] = imod(xs + 4 * lane + k - 1, fd.nx);
  const long long mps = (long long)fd.mp * fd.ny;
  const int ocol0 = xs + 4 * lane;
  const bool lane_out = full_row || (lane >= 1 && lane <= 30 && ocol0 < fd.nx);
  int fm = imod(y0 - 1, fd.ny), f0 = y0, fp = imod(y0 + 1, fd.ny);
  auto fetch_next = [&](float4* slot) {
    issue_row<ST, VEC>(fd, slot, lane, (long long)fm * fd.nx, (long long)f0 * fd.nx, (long long)fp * fd.nx, cl);
    fm = f0;
    f0 = fp;
    fp = fp + 1 == fd.ny ? 0 : fp + 1;
  };
  wait_previous();
#pragma unroll
  for (int d = 0; d < PF; ++d) {
    if (d < n_it) fetch_next(slots + d * PP::SLOT_F4);
    cp_async_commit();
  }
  int s_cur = 0, s_pf = PF;
  for (int it = 0; it < n_it; ++it) {
    if (it + PF < n_it) fetch_next(slots + s_pf * PP::SLOT_F4);
    cp_async_commit();
    cp_async_wait<PF>();
    float4* slot = slots + s_cur * PP::SLOT_F4;
    constexpr bool IL = Pairs<ST, false>::IL;
    F2 m0[2], am[2], jx[2], jy[2];
    land_row<ST, VEC, ST == ST_F32 ? R_SUMS : R_ONES, false>(slot, lane, m0);
    if constexpr (ST == ST_F32) {
      to_pairs<IL>(slot[lane], m0);
      load_pairs(slot[32 + lane], am);
      load_pairs(slot[64 + lane], jx);
      load_pairs(slot[96 + lane], jy);
    } else {
      const F2* cache = cache_of(slot);
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        jx[k] = cache[(2 + k) * 32 + lane];
        jy[k] = cache[(4 + k) * 32 + lane];
      }
    }
    if (lane_out) {
      float* row = fd.dst.f32 + (long long)(y0 + it) * fd.mp;
      store_moment<IL>(row, ocol0, m0);
      if constexpr (ST == ST_F32) {
        row += mps;
        store_moment<IL>(row, ocol0, am);
      }
      store_moment<IL>(row + mps, ocol0, jx);
      store_moment<IL>(row + 2 * mps, ocol0, jy);
    }
    s_cur = s_cur + 1 == PP::SLOTS ? 0 : s_cur + 1;
    s_pf = s_pf + 1 == PP::SLOTS ? 0 : s_pf + 1;
  }
  cp_async_wait<0>();
}

// A launch of a step, or with MO but not MI of a gather.
template <int ST, bool VEC, int RT, bool MI, bool MO>
__device__ __forceinline__ void launch_warp(const StepArgs& a, const Field& fd, int strip, int seg, float4* slots,
                                            int lane) {
  if constexpr (MO && !MI)
    gather_warp<ST, VEC>(fd, strip, seg, slots, lane);
  else
    step_warp<ST, VEC, RT, MI, MO>(a, fd, strip, seg, slots, lane);
  begin_dependents();
}

// Single field: warp w takes strip w % n_strips of segment w / n_strips.
template <int ST, bool VEC, int RT, bool MI, bool MO>
__global__ void __launch_bounds__(STEP_WARPS * 32, (Pipe<ST, VEC, MI>::MIN_CTAS))
    step_kernel(const __grid_constant__ StepArgs a, const __grid_constant__ Field fd, long long n_warps) {
  extern __shared__ float4 smem_slots[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const long long warp = (long long)blockIdx.x * STEP_WARPS + wib;
  if (warp >= n_warps) return;  // whole warps only: shuffles see all 32 lanes
  float4* slots = smem_slots + wib * (Pipe<ST, VEC, MI>::SLOTS * Pipe<ST, VEC, MI>::SLOT_F4);
  launch_warp<ST, VEC, RT, MI, MO>(a, fd, (int)(warp % fd.n_strips), (int)(warp / fd.n_strips), slots, lane);
}

}  // namespace lbch
