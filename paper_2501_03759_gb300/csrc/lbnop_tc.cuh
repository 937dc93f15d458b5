// The periodic 3 x 3 convolution of lbnop.cu on the 5th-generation tensor cores (tcgen05):
// operands in shared memory in the MMA's canonical K-major layout, FP32 accumulators in
// tensor memory (TMEM), and warps specialised by role, so that loading, the MMAs and the
// epilogue of consecutive tiles overlap.
//
// Scope: rows of a multiple of 128 pixels (W % 128 == 0), H a multiple of 4, c_in and c_out
// in {16, 64, 96}; with X2, c_in = 16 and a second input tensor x2 (the BF16 remainder of
// the first), multiplied by the same weights: the contraction then runs over K = 32, the
// chunks of x followed by those of x2. That covers the finest level of the learned leap on
// 512 x 512 and larger fields, where most of its convolution work is; every other layer keeps
// the mma.sync kernels.
//
// The kernel is persistent: the grid holds as many CTAs per 128-pixel column block as fit on
// the GPU at once, and CTA g takes the g-th of that many equal runs of consecutive output rows
// (flattened over (b, h)), in tiles of up to 2 rows within one sample. Tile k:
//   - loader warps 8-11 copy its input rows (h - 1 .. h + rows, periodic in h) by 16-byte
//     cp.async, consecutive threads reading consecutive bytes, into slots of a ring of six:
//     input row i of tile k in slot (2 k + i) mod 6, as [K / 8 chunks][130 pixel slots]
//     [8 channels], pixel x0 - 1 + s (periodic in x) in pixel slot s. That is the K-major,
//     no-swizzle canonical layout of the MMA's A operand: 16-byte rows (one pixel's 8
//     channels) 16 bytes apart within a chunk block, chunk blocks 131 x 16 bytes apart. The
//     operand of tap (dy, dx) for output row r is input row r + 1 + dy from pixel slot 1 + dx
//     on: a shift of the descriptor's start address, no copy. A 2-row tile that follows a
//     2-row tile of the same sample finds its first two input rows in place (the previous
//     tile's last two) and copies two.
//   - warp 12 (lane 0) issues the 9 taps x K / 16 K-steps of MMAs per row into TMEM
//     accumulator buffer k mod 2 (2 x c_out FP32 columns, lane = pixel), D += A_t B_t^T,
//     while the epilogue still reads buffer (k + 1) mod 2.
//   - warp 13 (lane 0) streams the weight taps of all tiles in order: the weights are kept in
//     global memory already in the B operand's layout (tc_pack_kernel: [K / 8 chunks][c_out]
//     [8], chunk blocks c_out x 16 + 16 bytes apart), so one bulk copy moves a whole tap into
//     a stage of a ring of up to four, once the MMAs that read the stage's previous tap have
//     completed; the copy completes the stage's mbarrier by its byte count.
//   - epilogue warps 0-7: warps w and w + 4 share TMEM lane quarter w (one pixel per thread)
//     and read half of its c_out columns each with tcgen05.ld, add bias and conditioning,
//     scale, and write them out (conv_epilogue's outputs) in whole 32-byte sectors: 8 FP32 or
//     16 BF16 channels of the thread's pixel per store. (Staging rows through shared memory for
//     512-byte stores took two barriers of the 256 threads per row: the four 96 x 96 launches of
//     a training step, 16 samples of 128 x 128 pixels, 346 us that way and 260 us this way.)
// mbarriers order the roles: a_full (rows loaded), mma_done (accumulators complete; input slots
// free), epi_done (accumulator buffer free), and per weight stage b_full / b_empty. Tile k's new
// input rows go where tile k - 2's first two were, so its copies wait for tile k - 2's MMAs.
// Staging the input rows through TMA was measured first: tensor-map boxes whose innermost
// extent is one 8-channel chunk (16 bytes) move each pixel's chunk as a separate request, and
// operand staging then took most of a CTA's time. Coalesced 16-byte copies land the same
// layout at full rate; the weights, whose layout is chosen here, go as whole taps.
// Every wait on an mbarrier is bounded; on timeout the kernel sets an error flag, waits
// (bounded) for its copies and MMAs in flight, frees its TMEM and stops.
#pragma once

namespace nop {

constexpr int TC_SLOTS = 130;                  // pixel slots per chunk block: x0 - 1 .. x0 + 128
constexpr int TC_CHUNK_A = (TC_SLOTS + 1) * 16;  // bytes between chunk blocks of an input row
constexpr int TC_ROWS = 2;                     // output rows per tile at most
constexpr int TC_RING = 6;                     // input-row slots: two tiles in flight
constexpr int TC_EPI = 256;                    // warps 0-7: epilogue
constexpr int TC_LOAD = 128;                   // warps 8-11: input-row loaders
constexpr int TC_MMA_WARP = 12;                // lane 0 issues the MMAs; the warp owns the TMEM
constexpr int TC_PROD_WARP = 13;               // lane 0 streams the weight taps
constexpr int TC_THREADS = 14 * 32;
constexpr int TC_MAX_BSTAGES = 4;
constexpr int TC_BARS = 2 * TC_MAX_BSTAGES + 7;  // b_full, b_empty, a_full[2], mma_done[2], epi_done[2], final
constexpr unsigned TC_SPIN_LIMIT = 1u << 20;   // bounded mbarrier waits (about a second at most)

// Set by a CTA whose wait gave up; every later CTA of the path then returns at once.
__device__ int tc_fault_flag;

// KC = K / 8: 8-channel chunks per pixel of the contraction (c_in / 8, doubled with X2).
template <int KC>
__host__ __device__ constexpr int tc_row_bytes() { return KC * TC_CHUNK_A; }
template <int CO>
__host__ __device__ constexpr int tc_chunk_b() { return CO * 16 + 16; }  // bytes between chunk blocks of a tap
template <int KC, int CO>
__host__ __device__ constexpr int tc_tap_bytes() { return KC * tc_chunk_b<CO>(); }
template <int KC, int CO, int S>
__host__ __device__ constexpr int tc_main_bytes_s() { return TC_RING * tc_row_bytes<KC>() + S * tc_tap_bytes<KC, CO>(); }
// Weight-ring stages: four where they fit in one CTA's shared memory (more taps in flight
// hide the copy latency behind the MMAs), else three, else two.
template <int KC, int CO>
__host__ __device__ constexpr int tc_bstages() {
  return tc_main_bytes_s<KC, CO, 4>() + 512 <= 227 * 1024 ? 4 : (tc_main_bytes_s<KC, CO, 3>() + 512 <= 227 * 1024 ? 3 : 2);
}
// The input slots, the weight ring; then the mbarriers, the TMEM
// address and an abort word (256 bytes), and alignment slack.
template <int KC, int CO>
__host__ __device__ constexpr int tc_main_bytes() { return tc_main_bytes_s<KC, CO, tc_bstages<KC, CO>()>(); }
template <int KC, int CO>
__host__ __device__ constexpr int tc_smem_bytes() { return tc_main_bytes<KC, CO>() + 256 + 128; }
// TMEM columns: a power of two >= 32 that holds two buffers of TC_ROWS accumulators of CO columns.
template <int CO>
__host__ __device__ constexpr int tc_tmem_cols() {
  constexpr int n = 2 * TC_ROWS * CO;
  return n <= 32 ? 32 : (n <= 64 ? 64 : (n <= 128 ? 128 : (n <= 256 ? 256 : 512)));
}
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Waits for the phase with the given parity to complete; false if it did not within the limit.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (unsigned i = 0; i < TC_SPIN_LIMIT; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void tc_cp16(uint32_t smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(gmem) : "memory");
}
// This thread's copies have landed and are visible to the tensor cores (async proxy).
__device__ __forceinline__ void tc_cp_done() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_all;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// This thread's arrival on the mbarrier, raising the phase's expected transaction count by
// `bytes`: the phase completes once the arrivals are in and that many bytes have landed.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// One bulk copy of `bytes` from global to this CTA's shared memory (both addresses 16-byte
// aligned, bytes a multiple of 16) that counts its bytes against the mbarrier's phase.
__device__ __forceinline__ void tc_bulk_copy(uint32_t smem, const void* gmem, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem),
               "l"(gmem), "r"(bytes), "r"(bar)
               : "memory");
}

// Shared-memory matrix descriptor of a K-major operand without swizzling: 8-row x 16-byte
// core matrices, rows 16 bytes apart; lbo = bytes between K-adjacent core matrices, sbo =
// bytes between core matrices adjacent in M (or N); bits 46-47 hold the descriptor version 1.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), BF16 A and B (bits
// 7-9 and 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 in bits 17-22, M >> 4 in bits
// 24-28.
template <int M, int N>
__host__ __device__ constexpr uint32_t umma_idesc_bf16() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
          tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 or 16 consecutive accumulator columns of this thread's TMEM lane, as raw bits; the
// caller waits (tcgen05.wait::ld) before using them.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
      "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// One 32-byte store (a whole sector) of this thread; 32-byte aligned.
__device__ __forceinline__ void st_sector(void* p, const uint32_t (&v)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// The output channels of a pixel that the warps of pair half g (0 or 1) take, in groups of 16, from
// column tc_col(g, j), j < tc_groups: for c_out = 96, 32 columns at 32 g and 16 at 64 + 16 g; for 64,
// 32 at 32 g; for 16, all 16 of every other row.
template <int CO>
__host__ __device__ constexpr int tc_groups() { return CO == 96 ? 3 : (CO == 64 ? 2 : 1); }
template <int CO>
__device__ __forceinline__ int tc_col(int g, int j) { return CO == 16 ? 0 : (j < 2 ? 32 * g + 16 * j : 64 + 16 * g); }

// The accumulators of the groups of half g (TMEM loads of 32 columns start at multiples of 32, of 16
// at multiples of 16; row and buffer offsets are multiples of 16 too).
template <int CO>
__device__ __forceinline__ void tc_read(uint32_t taddr_row, int g, uint32_t (&r)[16 * tc_groups<CO>()]) {
  static_assert(CO == 16 || CO == 64 || CO == 96, "output widths of the network");
  if constexpr (CO == 16) {
    tmem_ld16(taddr_row, r);
  } else {
    tmem_ld32(taddr_row + 32 * g, r);
    if constexpr (CO == 96) tmem_ld16(taddr_row + 64 + 16 * g, r + 32);
  }
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Bias, conditioning (al), scale, SiLU' and the stores of 16 channels n .. n + 15 of a pixel (o: its
// offset) from the accumulators acc (raw bits), as conv_epilogue does. wide: yf is 32-byte aligned.
__device__ __forceinline__ void tc_finish(const ConvArgs& p, const uint32_t* acc, int n, size_t o, float al, float sc,
                                          bool wide, const uint4 (&zg)[2]) {
  float v[16];
#pragma unroll
  for (int e = 0; e < 16; e += 4) {
    float4 b = make_float4(0.0f, 0.0f, 0.0f, 0.0f), f = b;
    if (p.bias) b = make_float4(p.bias[n + e], p.bias[n + e + 1], p.bias[n + e + 2], p.bias[n + e + 3]);
    if (p.film) f = make_float4(p.film[n + e], p.film[n + e + 1], p.film[n + e + 2], p.film[n + e + 3]);
    v[e] = (__uint_as_float(acc[e]) + b.x + __fmul_rn(al, f.x)) * sc;
    v[e + 1] = (__uint_as_float(acc[e + 1]) + b.y + __fmul_rn(al, f.y)) * sc;
    v[e + 2] = (__uint_as_float(acc[e + 2]) + b.z + __fmul_rn(al, f.z)) * sc;
    v[e + 3] = (__uint_as_float(acc[e + 3]) + b.w + __fmul_rn(al, f.w)) * sc;
  }
  if (p.zg) {
    const uint32_t raw[8] = {zg[0].x, zg[0].y, zg[0].z, zg[0].w, zg[1].x, zg[1].y, zg[1].z, zg[1].w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      v[2 * e] *= silu_grad_f(__uint_as_float(raw[e] << 16));
      v[2 * e + 1] *= silu_grad_f(__uint_as_float(raw[e] & 0xffff0000u));
    }
  }
  if (p.yf) {
    float* y = p.yf + o + n;
    if (p.accumulate) {
#pragma unroll
      for (int e = 0; e < 16; e += 4) {
        const float4 old = *reinterpret_cast<const float4*>(y + e);
        v[e] = old.x + v[e];
        v[e + 1] = old.y + v[e + 1];
        v[e + 2] = old.z + v[e + 2];
        v[e + 3] = old.w + v[e + 3];
      }
    }
    if (wide) {
#pragma unroll
      for (int e = 0; e < 16; e += 8) {
        const uint32_t w[8] = {__float_as_uint(v[e]),     __float_as_uint(v[e + 1]), __float_as_uint(v[e + 2]),
                               __float_as_uint(v[e + 3]), __float_as_uint(v[e + 4]), __float_as_uint(v[e + 5]),
                               __float_as_uint(v[e + 6]), __float_as_uint(v[e + 7])};
        st_sector(y + e, w);
      }
    } else {
#pragma unroll
      for (int e = 0; e < 16; e += 4)
        *reinterpret_cast<float4*>(y + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    }
  }
  if (p.z) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack2(__float2bfloat16_rn(v[2 * e]), __float2bfloat16_rn(v[2 * e + 1]));
    st_sector(p.z + o + n, w);
  }
  if (p.a) {
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e)
      w[e] = pack2(__float2bfloat16_rn(silu_f(v[2 * e])), __float2bfloat16_rn(silu_f(v[2 * e + 1])));
    st_sector(p.a + o + n, w);
  }
}

// Output rows of the tile starting at flattened row r: at most TC_ROWS, within the CTA's run
// (which ends before `last`) and within the sample.
__device__ __forceinline__ int tc_tile_rows(int r, int last, int H) {
  const int h = r % H;
  int n = last - r;
  n = n < TC_ROWS ? n : TC_ROWS;
  return n < H - h ? n : H - h;
}

// The tiles of one CTA, in order: rows [r0, r0 + rk), input slot base sk = 2 k mod 6, and
// whether the first two input rows are the previous tile's last two (a full tile of the same
// sample before it). Every role walks the same sequence.
struct TcTiles {
  int first, last, H;
  int k, r0, rk, sk;
  bool reuse;
  __device__ __forceinline__ void start(int f, int l, int h) {
    first = f;
    last = l;
    H = h;
    k = 0;
    r0 = f;
    sk = 0;
    reuse = false;
    rk = r0 < last ? tc_tile_rows(r0, last, H) : 0;
  }
  __device__ __forceinline__ bool more() const { return r0 < last; }
  __device__ __forceinline__ void next() {
    const bool full = rk == TC_ROWS;
    r0 += rk;
    ++k;
    sk = sk + 2 == TC_RING ? 0 : sk + 2;
    reuse = full && r0 < last && r0 % H != 0;
    rk = r0 < last ? tc_tile_rows(r0, last, H) : 0;
  }
};

// Grid: (W / 128) x G CTAs of TC_THREADS; CTA (x, g) takes flattened output rows
// [g N / G, (g + 1) N / G), N = B H, of column block x. p.wpk holds the weights packed by
// tc_pack_kernel for (CI, CO, X2).
template <int CI, int CO, bool X2>
__global__ void __launch_bounds__(TC_THREADS, 1) conv_tc_kernel(const __grid_constant__ ConvArgs p, int* err) {
  constexpr int KC = (X2 ? 2 : 1) * CI / 8;    // 8-channel chunks of the contraction
  constexpr int K = 8 * KC;
  static_assert(K % 16 == 0 && CO % 16 == 0 && CO <= 256, "UMMA shape: K steps of 16, N a multiple of 16");
  static_assert(2 * TC_ROWS * CO <= 512, "two accumulator buffers fit in TMEM");
  static_assert(!X2 || CI == 16, "the second input only on 16-channel layers");
  constexpr int ROW = tc_row_bytes<KC>();       // bytes per staged input row
  constexpr int TAP = tc_tap_bytes<KC, CO>();   // bytes per staged weight tap
  constexpr uint32_t LBO_A = TC_CHUNK_A, LBO_B = tc_chunk_b<CO>(), SBO = 128;
  constexpr int COLS = tc_tmem_cols<CO>();
  constexpr uint32_t IDESC = umma_idesc_bf16<128, CO>();
  constexpr int S = tc_bstages<KC, CO>();
  constexpr int PER_ROW = TC_SLOTS * KC;        // 16-byte copies per input row
  static_assert(PER_ROW >= TC_LOAD, "a loader's copies advance by one row at most");
  extern __shared__ __align__(128) unsigned char tc_smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(tc_smem_raw) + 127) & ~(uintptr_t)127);
  unsigned char* sA = base;
  unsigned char* sB = base + TC_RING * ROW;
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + tc_main_bytes<KC, CO>());
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + TC_BARS);
  volatile int* abort_word = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto b_full = [&](int s) { return smem_u32(&bars[s]); };
  auto b_empty = [&](int s) { return smem_u32(&bars[S + s]); };
  auto a_full = [&](int j) { return smem_u32(&bars[2 * S + j]); };
  auto mma_done = [&](int j) { return smem_u32(&bars[2 * S + 2 + j]); };
  auto epi_done = [&](int j) { return smem_u32(&bars[2 * S + 4 + j]); };
  const uint32_t final_bar = smem_u32(&bars[2 * S + 6]);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int x0 = blockIdx.x * 128;
  const int N = p.B * p.H;
  const int first = (int)((long long)blockIdx.y * N / gridDim.y);
  const int last = (int)((long long)(blockIdx.y + 1) * N / gridDim.y);

  if (tid == 0) {
    *abort_word = *(volatile int*)&tc_fault_flag;  // an earlier CTA's wait gave up: do nothing
    for (int s = 0; s < S; ++s) {
      mbar_init(b_full(s), 1);   // the producer's arrival plus the tap's bytes
      mbar_init(b_empty(s), 1);  // the commit of the MMAs that read the stage
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(a_full(j), TC_LOAD);   // every loader thread, once its copies have landed
      mbar_init(mma_done(j), 1);       // the commit after the tile's MMAs
      mbar_init(epi_done(j), TC_EPI);  // every epilogue thread, once done with the buffer
    }
    mbar_init(final_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (*abort_word || first >= last) return;  // uniform over the CTA: nothing allocated or in flight yet
  if (warp == TC_MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  bool ok = true;
  TcTiles tl;
  tl.start(first, last, p.H);
  if (warp < TC_EPI / 32) {
    // ------------------------------------------------------------ epilogue warps 0-7
    const int quarter = warp & 3, half = warp >> 2;
    const int px = 32 * quarter + lane;  // this thread's TMEM lane: pixel x0 + px
    constexpr int NG = tc_groups<CO>();
    const bool wide = ((uintptr_t)p.yf % 32) == 0;
    for (; tl.more(); tl.next()) {
      const int j = tl.k & 1;
      const bool fin = mbar_wait(mma_done(j), (uint32_t)((tl.k >> 1) & 1));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!__all_sync(0xffffffffu, fin)) {  // uniform over the warp
        ok = false;
        break;
      }
      const int b = tl.r0 / p.H;
      const float al = p.film ? p.alpha[b] : 0.0f;
      const float sc = p.scale_alpha ? p.alpha[b] : 1.0f;
#pragma unroll 1
      for (int r = 0; r < tl.rk; ++r) {
        if (CO == 16 && (r & 1) != half) continue;
        const size_t o = ((size_t)(tl.r0 + r) * p.W + x0 + px) * CO;
        uint4 zg[NG][2];  // loaded ahead of the accumulators
#pragma unroll
        for (int q = 0; q < NG; ++q)
#pragma unroll
          for (int e = 0; e < 2; ++e)
            zg[q][e] = p.zg ? reinterpret_cast<const uint4*>(p.zg + o + tc_col<CO>(half, q))[e] : make_uint4(0u, 0u, 0u, 0u);
        uint32_t acc[16 * NG];
        tc_read<CO>(tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)((j * TC_ROWS + r) * CO), half, acc);
#pragma unroll
        for (int q = 0; q < NG; ++q) tc_finish(p, acc + 16 * q, tc_col<CO>(half, q), o, al, sc, wide, zg[q]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(epi_done(j));  // this thread's accumulator reads are done
    }
  } else if (warp < (TC_EPI + TC_LOAD) / 32) {
    // ------------------------------------------------------------ loader warps 8-11
    const int ltid = tid - TC_EPI;
    const uint32_t sA32 = smem_u32(sA);
    for (; tl.more(); tl.next()) {
      const int j = tl.k & 1;
      // slots of input rows 2, 3: tile k - 2's first two
      if (tl.k >= 2 && !mbar_wait(mma_done(j), (uint32_t)(((tl.k >> 1) + 1) & 1))) {
        ok = false;
        break;
      }
      // slots of input rows 0, 1 when not reused: tile k - 1's last two, read by its MMAs
      if (!tl.reuse && tl.k >= 1 && !mbar_wait(mma_done(j ^ 1), (uint32_t)(((tl.k - 1) >> 1) & 1))) {
        ok = false;
        break;
      }
      const int b = tl.r0 / p.H, h0 = tl.r0 - b * p.H;
      // item (i, pixel slot, chunk), chunk fastest; each loader steps TC_LOAD items at a time
      const int i0 = tl.reuse ? 2 : 0;
      const int n_items = (tl.rk + 2 - i0) * PER_ROW;
      int i = i0, rem = ltid;
      size_t row_px = (size_t)(b * p.H + wrap1(h0 - 1 + i, p.H)) * p.W;  // first pixel of input row i
      int q = tl.sk + i >= TC_RING ? tl.sk + i - TC_RING : tl.sk + i;    // its slot
      for (int idx = ltid; idx < n_items; idx += TC_LOAD) {
        const int sl = rem / KC, c = rem - sl * KC;
        const size_t px = row_px + wrap1(x0 - 1 + sl, p.W);
        const bf16* src = (X2 && c >= CI / 8) ? p.x2 + px * CI + 8 * (c - CI / 8) : p.x + px * CI + 8 * c;
        tc_cp16(sA32 + (uint32_t)(q * ROW + c * TC_CHUNK_A + sl * 16), src);
        rem += TC_LOAD;
        if (rem >= PER_ROW) {
          rem -= PER_ROW;
          ++i;
          row_px = (size_t)(b * p.H + wrap1(h0 - 1 + i, p.H)) * p.W;
          q = q + 1 == TC_RING ? 0 : q + 1;
        }
      }
      tc_cp_done();  // this thread's copies have landed and are visible to the tensor cores
      mbar_arrive(a_full(j));
    }
  } else if (warp == TC_MMA_WARP) {
    // ------------------------------------------------------------ MMA issuer (lane 0)
    if (lane == 0) {
      // Descriptors of input slot 0 and weight stage 0 at their first chunk: every operand
      // start is a 16-byte multiple from them, added to the start-address field (address / 16,
      // 14 bits, which holds every shared-memory address).
      const uint64_t a0 = umma_desc(smem_u32(sA), LBO_A, SBO);
      const uint64_t b0 = umma_desc(smem_u32(sB), LBO_B, SBO);
      for (; tl.more() && ok; tl.next()) {
        const int j = tl.k & 1;
        if (!mbar_wait(a_full(j), (uint32_t)((tl.k >> 1) & 1)) ||
            (tl.k >= 2 && !mbar_wait(epi_done(j), (uint32_t)(((tl.k >> 1) + 1) & 1)))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t dcol = tmem + (uint32_t)(j * TC_ROWS * CO);
        for (int t = 0; t < 9; ++t) {
          const int T = 9 * tl.k + t, s = T % S;
          if (!mbar_wait(b_full(s), (uint32_t)((T / S) & 1))) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int dy = t / 3 - 1, dx = t % 3 - 1;
          const uint64_t bt = b0 + (uint64_t)((s * TAP) >> 4);
#pragma unroll
          for (int r = 0; r < TC_ROWS; ++r) {
            if (r < tl.rk) {
              int q = tl.sk + r + 1 + dy;  // the slot of input row r + 1 + dy
              q = q >= TC_RING ? q - TC_RING : q;
              const uint64_t at = a0 + (uint64_t)((q * ROW + (1 + dx) * 16) >> 4);
#pragma unroll
              for (int kk = 0; kk < K / 16; ++kk)
                umma_bf16(dcol + (uint32_t)(r * CO), at + (uint64_t)((kk * 2 * LBO_A) >> 4),
                          bt + (uint64_t)((kk * 2 * LBO_B) >> 4), IDESC, (t > 0 || kk > 0) ? 1u : 0u);
            }
          }
          umma_commit(b_empty(s));  // the stage is free once these MMAs have read it
        }
        if (!ok) break;
        umma_commit(mma_done(j));  // the tile's accumulators are complete once this arrives
      }
      umma_commit(final_bar);  // every MMA issued above has completed once this arrives
      if (!mbar_wait(final_bar, 0)) ok = false;
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ weight producer (lane 0)
    if (lane == 0) {  // tap T of the run (tile T / 9, tap T % 9) into stage T % S
      int ntiles = 0;
      for (; tl.more(); tl.next()) ++ntiles;
      int last_tap[TC_MAX_BSTAGES] = {-1, -1, -1, -1};
      for (int T = 0; T < 9 * ntiles; ++T) {
        const int s = T % S;
        if (T >= S && !mbar_wait(b_empty(s), (uint32_t)(((T - S) / S) & 1))) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(b_full(s), (uint32_t)TAP);
        tc_bulk_copy(smem_u32(sB + s * TAP), p.wpk + (size_t)(T % 9) * TAP, (uint32_t)TAP, b_full(s));
        last_tap[s] = T;
      }
      // the last copy into each stage has landed before the CTA ends
      for (int s = 0; s < S; ++s)
        if (last_tap[s] >= 0 && !mbar_wait(b_full(s), (uint32_t)((last_tap[s] / S) & 1))) ok = false;
    }
    __syncwarp();
  }
  const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
  if (!all_ok && tid == 0) {
    atomicExch(&tc_fault_flag, 1);
    if (err) atomicExch(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == TC_MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
}

// The weights of a (CI, CO, X2) layer in the layout of the kernel's weight ring:
// out[t][c][n][8] (chunk blocks CO x 16 + 16 bytes apart, the last 16 bytes zero) =
// w[t][n][8 c' .. 8 c' + 7], c' = c mod (CI / 8) (with X2 the chunks repeat: both inputs
// meet the same weights). w is [9][CO][CI] BF16; out holds 9 tc_tap_bytes.
__global__ void tc_pack_kernel(const bf16* __restrict__ w, int CI, int CO, int KC, unsigned char* __restrict__ out) {
  const int per_chunk = CO + 1, n_items = 9 * KC * per_chunk;  // 16-byte items, one pad per chunk block
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n_items; idx += gridDim.x * blockDim.x) {
    const int t = idx / (KC * per_chunk), rem = idx - t * (KC * per_chunk);
    const int c = rem / per_chunk, n = rem - c * per_chunk;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (n < CO) v = *reinterpret_cast<const uint4*>(w + ((size_t)t * CO + n) * CI + 8 * (c % (CI / 8)));
    *reinterpret_cast<uint4*>(out + (size_t)idx * 16) = v;
  }
}

// ---------------------------------------------------------------- weight gradient

// The weight gradient dw[t][o][i] += sum_p dz(p)[o] x(p + d_t)[i] (t = 3 (dy + 1) + dx + 1, the
// data-parallel half of the backward pass of a convolution) on the tensor cores: the pixels are
// the contraction. The staging layout of the convolution above, [chunk][pixel slot][8
// channels], is then the canonical MN-major layout (8 pixels x 8 channels per 128-byte core
// matrix, channel chunks TC_CHUNK_A apart along M or N, 8-pixel groups 128 bytes apart along
// K), so both operands are staged exactly as the convolution stages its input rows and the
// descriptors keep their strides; the instruction descriptor marks A and B MN-major.
// A = dz of one row (M = c_out padded to 128 with zero chunks), B = x of the row dy away (N =
// c_in), shifted by dx through the start address; K = 16 pixels per MMA, 8 per row of 128.
//
// Grid: (W / bw) x 3 (dy) x G CTAs of WG_THREADS. A row is cut into column blocks of bw pixels (the
// largest divisor of W up to 128 that is a multiple of the MMA's 16 pixels), and a stage holds R =
// 128 / bw rows of one column block, row r's x pixels in slots r (bw + 2) .. with its own periodic
// halo and its dz pixels at the same slots: every K-step of 16 pixels lies in one row. CTA (x, dy,
// g) takes the g-th of G equal runs of the groups of R rows (flattened over (b, h)), accumulates
// its three dx taps in TMEM (3 c_in columns, lane = output channel) and adds them into dw at the
// end, four FP32 per atomic. Warps 0-7 stage the groups into a ring (16-byte copies) and warps 0-3
// read TMEM at the end; warp 8 allocates TMEM and its lane 0 issues the MMAs.
//
// The loaders announce a group WG_AHEAD groups after they issued its copies, so that those of the
// next ones are in flight meanwhile: a loader that waited for each group before the next one paid
// the latency of memory per group. 96 x 96 channels, 16 samples of 128 x 128 pixels: 110 -> 88 us;
// at 64 x 64 pixels 64 x 96 channels, where mma.sync ran before, 65 -> 28 us. Bound now
// by the 16-byte copies, about 0.75 of them per cycle and SM.
constexpr int WG_LOAD = 256;
constexpr int WG_MMA_WARP = WG_LOAD / 32;
constexpr int WG_THREADS = WG_LOAD + 32;
constexpr int WG_MCH = 16;                       // chunks of the A operand: M = 128 channels
constexpr int WG_SLOTS = 144;                    // pixel slots per chunk block: R (bw + 2) at most (bw = 16)
constexpr int WG_CHUNK = (WG_SLOTS + 1) * 16;    // bytes between chunk blocks

// With 16 x 16 channels the three dx taps go in one MMA of N = 48: x is staged three times, already
// shifted, and a K-step takes one MMA instead of three (16 samples of 128 x 128 pixels: 47 -> 36 us).
// With c_out = 96 the extra copies cost more than that (53 -> 61 us).
template <int CI, int CO>
__host__ __device__ constexpr bool wg_stacked() { return CI == 16 && CO == 16; }
template <int CI, int CO>
__host__ __device__ constexpr int wg_stage_bytes() { return (WG_MCH + (wg_stacked<CI, CO>() ? 3 : 1) * CI / 8) * WG_CHUNK; }
template <int CI, int CO>
__host__ __device__ constexpr int wg_stages() { return 4 * wg_stage_bytes<CI, CO>() + 512 <= 227 * 1024 ? 4 : 3; }
template <int CI, int CO>
__host__ __device__ constexpr int wg_smem_bytes() { return wg_stages<CI, CO>() * wg_stage_bytes<CI, CO>() + 256 + 128; }
template <int CI>
__host__ __device__ constexpr int wg_tmem_cols() {
  return 3 * CI <= 32 ? 32 : (3 * CI <= 64 ? 64 : (3 * CI <= 128 ? 128 : (3 * CI <= 256 ? 256 : 512)));
}
// Width of a column block of rows of W pixels: the largest divisor of W up to 128 that is a
// multiple of 16, or 0.
__host__ __device__ inline int wg_block_width(int W) {
  for (int bw = 128; bw >= 16; bw -= 16)
    if (W % bw == 0) return bw;
  return 0;
}
// kind::f16, FP32 accumulator, BF16 A and B, both MN-major (bits 15, 16), N >> 3, M >> 4.
template <int M, int N>
__host__ __device__ constexpr uint32_t umma_idesc_bf16_mn() {
  return umma_idesc_bf16<M, N>() | (1u << 15) | (1u << 16);
}

template <int CI, int CO>
__global__ void __launch_bounds__(WG_THREADS, 1) wgrad_tc_kernel(const __grid_constant__ WgradArgs p, int bw,
                                                                 int* err) {
  static_assert(CO <= 128 && CO % 16 == 0 && CI % 16 == 0 && 3 * CI <= 512, "M = 128 channels, 3 taps in TMEM");
  constexpr int ST = wg_stages<CI, CO>(), STG = wg_stage_bytes<CI, CO>();
  constexpr int WG_AHEAD = ST - 2;  // a stage is refilled once its MMAs, a group later, are done
  constexpr int COLS = wg_tmem_cols<CI>();
  constexpr bool STACK = wg_stacked<CI, CO>();
  constexpr uint32_t IDESC = umma_idesc_bf16_mn<128, STACK ? 3 * CI : CI>();
  // MN-major: the leading offset steps along K (8-pixel groups), the stride offset along M / N
  // (channel chunks)
  constexpr uint32_t LBO = 128, SBO = WG_CHUNK;
  constexpr int ZC = CO / 8, XC = CI / 8;  // chunks of dz and of x per pixel
  extern __shared__ __align__(128) unsigned char wg_smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(wg_smem_raw) + 127) & ~(uintptr_t)127);
  // stage s: dz chunk blocks 0..15 (ZC.. zero), then the x chunk blocks
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + ST * STG);  // full[ST], empty[ST], done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * 4 + 1);
  volatile int* abort_word = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto full = [&](int s) { return smem_u32(&bars[s]); };
  auto empty = [&](int s) { return smem_u32(&bars[ST + s]); };
  const uint32_t done_bar = smem_u32(&bars[2 * ST]);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int x0 = blockIdx.x * bw, dy = (int)blockIdx.y - 1;
  const int N = p.B * p.H, R = 128 / bw, NG = (N + R - 1) / R;
  const int first = (int)((long long)blockIdx.z * NG / gridDim.z);
  const int ng = (int)((long long)(blockIdx.z + 1) * NG / gridDim.z) - first;  // groups of this CTA
  auto rows_of = [&](int j) { return min(R, N - (first + j) * R); };           // rows of its j-th group

  if (tid == 0) {
    *abort_word = *(volatile int*)&tc_fault_flag;
    for (int s = 0; s < ST; ++s) {
      mbar_init(full(s), WG_LOAD);
      mbar_init(empty(s), 1);
    }
    mbar_init(done_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the zero chunks of every stage's A operand (M rows CO .. 127), written once
  for (int s = 0; s < ST; ++s)
    for (int k = tid; k < (WG_MCH - ZC) * WG_CHUNK / 16; k += WG_THREADS)
      reinterpret_cast<uint4*>(base + s * STG + ZC * WG_CHUNK)[k] = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (*abort_word || ng <= 0) return;  // uniform: nothing allocated or in flight
  if (warp == WG_MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  bool ok = true;
  if (warp < WG_MMA_WARP) {
    // ------------------------------------------------ loaders: group j of the run into stage j % ST
    const uint32_t base32 = smem_u32(base);
    // q / bw and q / (bw + 2) for q < WG_SLOTS, exactly
    const uint32_t inv_z = 65536u / (uint32_t)bw + 1u, inv_x = 65536u / (uint32_t)(bw + 2) + 1u;
    for (int j = 0; j < ng; ++j) {
      const int s = j % ST;
      if (j >= ST && !mbar_wait(empty(s), (uint32_t)(((j - ST) / ST) & 1))) {
        ok = false;
        break;
      }
      const int row0 = (first + j) * R, rk = rows_of(j), h0 = row0 % p.H;
      // dz: pixel x0 + o of row r in slot r (bw + 2) + 1 + o, chunks 0 .. ZC - 1
      for (int idx = tid; idx < rk * bw * ZC; idx += WG_LOAD) {
        const int q = idx / ZC, c = idx - q * ZC;
        const int r = (int)(((uint32_t)q * inv_z) >> 16), o = q - r * bw;
        tc_cp16(base32 + (uint32_t)(s * STG + c * WG_CHUNK + (q + 2 * r + 1) * 16),
                p.dz + ((size_t)(row0 + r) * p.W + x0 + o) * CO + 8 * c);
      }
      // x: pixel x0 - 1 + o (periodic) of the row dy away in slot r (bw + 2) + o; stacked, pixel
      // x0 + o + dxi - 1 in slot r (bw + 2) + 1 + o of chunks dxi XC ..
      for (int idx = tid; idx < (STACK ? 3 * rk * bw : rk * (bw + 2)) * XC; idx += WG_LOAD) {
        const int q = idx / (STACK ? 3 * XC : XC), c = idx - q * (STACK ? 3 * XC : XC);
        const int r = (int)(((uint32_t)q * (STACK ? inv_z : inv_x)) >> 16);
        const int o = STACK ? q - r * bw + c / XC : q - r * (bw + 2), slot = STACK ? q + 2 * r + 1 : q;
        int h = h0 + r;
        if (h >= p.H) h %= p.H;
        const int row = row0 + r - h + wrap1(h + dy, p.H);
        tc_cp16(base32 + (uint32_t)(s * STG + (WG_MCH + c) * WG_CHUNK + slot * 16),
                p.x + ((size_t)row * p.W + wrap1(x0 - 1 + o, p.W)) * CI + 8 * (c % XC));
      }
      cp_async_commit_group();
      if (j >= WG_AHEAD) {  // group j - WG_AHEAD has landed: visible to the tensor cores
        cp_async_wait_group<WG_AHEAD>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(full((j - WG_AHEAD) % ST));
      }
    }
    cp_async_wait_group<0>();
    if (ok) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      for (int j = max(0, ng - WG_AHEAD); j < ng; ++j) mbar_arrive(full(j % ST));
    }
  } else if (lane == 0) {
    // ------------------------------------------------ MMA issuer: 3 dx taps x bw / 16 K-steps per row
    const uint64_t d0 = umma_desc(smem_u32(base), LBO, SBO);
    for (int j = 0; j < ng; ++j) {
      const int s = j % ST;
      if (!mbar_wait(full(s), (uint32_t)((j / ST) & 1))) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t as = d0 + (uint64_t)((s * STG + 16) >> 4);                  // dz slot 1
      const uint64_t bs = d0 + (uint64_t)((s * STG + WG_MCH * WG_CHUNK) >> 4);   // x slot 0
      const int rk = rows_of(j);
      for (int r = 0; r < rk; ++r)
        for (int kk = 0; kk < bw / 16; ++kk) {
          const uint64_t at = (uint64_t)(r * (bw + 2) + 16 * kk);
#pragma unroll
          for (int dxi = 0; dxi < (STACK ? 1 : 3); ++dxi)
            umma_bf16(tmem + (uint32_t)(dxi * CI), as + at, bs + at + (uint64_t)(STACK ? 1 : dxi), IDESC,
                      (j > 0 || r > 0 || kk > 0) ? 1u : 0u);
        }
      umma_commit(empty(s));
    }
    umma_commit(done_bar);
  }
  __syncwarp();
  // every thread: the accumulators are complete (or the run gave up)
  const bool fin = mbar_wait(done_bar, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const bool good = __syncthreads_and((ok && fin) ? 1 : 0) != 0;
  if (!good && tid == 0) {
    atomicExch(&tc_fault_flag, 1);
    if (err) atomicExch(err, 1);
  }
  if (good && warp < 4) {
    // ------------------------------------------------ epilogue: TMEM lane 32 warp + lane = channel o
    const int o = 32 * warp + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(32 * warp) << 16);
    const bool wide = ((uintptr_t)p.dw % 16) == 0;
#pragma unroll 1
    for (int c0 = 0; c0 < 3 * CI; c0 += 16) {
      uint32_t r[16];
      tmem_ld16(lane_addr + (uint32_t)c0, r);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (o < CO) {
        const int dxi = c0 / CI, i0 = c0 - dxi * CI, t = 3 * (dy + 1) + dxi;
        float* d = p.dw + ((size_t)t * CO + o) * CI + i0;
        if (wide) {
#pragma unroll
          for (int e = 0; e < 16; e += 4)
            atomicAdd(reinterpret_cast<float4*>(d + e),
                      make_float4(__uint_as_float(r[e]), __uint_as_float(r[e + 1]), __uint_as_float(r[e + 2]),
                                  __uint_as_float(r[e + 3])));
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) atomicAdd(d + e, __uint_as_float(r[e]));
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == WG_MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS) : "memory");
}

// ---------------------------------------------------------------- host side

// Whether the tensor-core path takes this convolution: rows of a multiple of 128 pixels, H a
// multiple of 4 (no CTA's rows straddle two samples), one input tensor or, on a 16-channel
// layer, the input and its BF16 remainder x2, no second weight half, and weights packed for
// the path (16-byte aligned operands).
inline bool tc_applies(const ConvArgs& a, int ci, int co) {
  const bool chans = (ci == 16 || ci == 64 || ci == 96) && (co == 16 || co == 64 || co == 96);
  const bool x2ok = a.x2 == nullptr || (ci == 16 && ((uintptr_t)a.x2 % 16) == 0);
  return chans && x2ok && a.w2 == nullptr && a.wpk != nullptr && a.W % 128 == 0 && a.H % 4 == 0 &&
         ((uintptr_t)a.x % 16) == 0 && ((uintptr_t)a.wpk % 16) == 0;
}

// Bytes of a layer's packed weights (tc_pack_kernel) and its 8-channel chunks per pixel.
inline int tc_kc(int ci, bool x2) { return (x2 ? 2 : 1) * ci / 8; }
inline size_t tc_pack_bytes(int ci, int co, bool x2) { return 9 * (size_t)tc_kc(ci, x2) * (co * 16 + 16); }

inline std::atomic<long long>& tc_wgrad_counter() {  // what lbnop_tc_wgrad_launches reports
  static std::atomic<long long> n{0};
  return n;
}
inline std::atomic<long long>& tc_counter() {
  static std::atomic<long long> n{0};
  return n;
}

// One persistent launch: as many CTAs per column block as fit on the GPU at once (never
// more than there are rows), each taking an equal run of rows.
template <int CI, int CO, bool X2>
void launch_tc_x(const ConvArgs& a, int* err, int sms, cudaStream_t s) {
  constexpr int KC = (X2 ? 2 : 1) * CI / 8;
  constexpr int bytes = tc_smem_bytes<KC, CO>();
  static_assert(bytes <= 227 * 1024, "fits in one CTA's shared memory");
  static std::atomic<int> per_sm[64];  // resident CTAs per SM, by device (0: not queried yet)
  int dev = 0;
  cudaGetDevice(&dev);
  int occ = per_sm[dev & 63].load(std::memory_order_relaxed);
  if (occ == 0) {
    cudaFuncSetAttribute(conv_tc_kernel<CI, CO, X2>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, conv_tc_kernel<CI, CO, X2>, TC_THREADS, bytes) !=
            cudaSuccess ||
        occ < 1) {
      cudaGetLastError();
      occ = 1;
    }
    if (occ > 512 / tc_tmem_cols<CO>()) occ = 512 / tc_tmem_cols<CO>();  // co-resident CTAs share TMEM
    per_sm[dev & 63].store(occ, std::memory_order_relaxed);
  }
  const int cols = a.W / 128, rows = a.B * a.H;
  const long long want = ((long long)sms * occ + cols - 1) / cols;
  const int G = (int)(want < rows ? want : rows);
  conv_tc_kernel<CI, CO, X2><<<dim3(cols, G), TC_THREADS, bytes, s>>>(a, err);
}

// The tensor-core weight gradient applies to rows of a multiple of 16 pixels (16-byte aligned
// tensors); every dz row pairs with its own sample's rows, so H is free. Shorter or ragged rows
// keep wgrad_kernel, whose contraction runs over pixels whatever their row.
inline bool wgrad_tc_applies(const WgradArgs& a) {
  return a.W % 16 == 0 && a.B * a.H >= 1 && ((uintptr_t)a.x % 16) == 0 && ((uintptr_t)a.dz % 16) == 0;
}

// One launch: (W / bw) x 3 (dy) x G CTAs, G equal runs of row groups per column block and dy, as
// many CTAs as fit on the GPU at once (never more runs than groups).
template <int CI, int CO>
void launch_wgrad_tc(const WgradArgs& a, int* err, int sms, cudaStream_t s) {
  constexpr int bytes = wg_smem_bytes<CI, CO>();
  static_assert(bytes <= 227 * 1024, "fits in one CTA's shared memory");
  static std::atomic<int> per_sm[64];
  int dev = 0;
  cudaGetDevice(&dev);
  int occ = per_sm[dev & 63].load(std::memory_order_relaxed);
  if (occ == 0) {
    cudaFuncSetAttribute(wgrad_tc_kernel<CI, CO>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, wgrad_tc_kernel<CI, CO>, WG_THREADS, bytes) !=
            cudaSuccess ||
        occ < 1) {
      cudaGetLastError();
      occ = 1;
    }
    if (occ > 512 / wg_tmem_cols<CI>()) occ = 512 / wg_tmem_cols<CI>();  // co-resident CTAs share TMEM
    per_sm[dev & 63].store(occ, std::memory_order_relaxed);
  }
  const int bw = wg_block_width(a.W), cols = a.W / bw, R = 128 / bw, groups = (a.B * a.H + R - 1) / R;
  const long long want = ((long long)sms * occ) / (3LL * cols);
  const int G = (int)(want < 1 ? 1 : (want < groups ? want : groups));
  wgrad_tc_kernel<CI, CO><<<dim3(cols, 3, G), WG_THREADS, bytes, s>>>(a, bw, err);
  tc_wgrad_counter().fetch_add(1, std::memory_order_relaxed);
  if (a.W % 128 == 0) tc_counter().fetch_add(1, std::memory_order_relaxed);  // what lbnop_tc_launches counts
}

// Launches conv_tc_kernel for this convolution (tc_applies holds).
template <int CI, int CO>
bool launch_tc(const ConvArgs& a, int* err, int sms, cudaStream_t s) {
  if constexpr (CI == 16) {
    if (a.x2) {
      launch_tc_x<CI, CO, true>(a, err, sms, s);
      tc_counter().fetch_add(1, std::memory_order_relaxed);
      return true;
    }
  }
  launch_tc_x<CI, CO, false>(a, err, sms, s);
  tc_counter().fetch_add(1, std::memory_order_relaxed);
  return true;
}

}  // namespace nop
