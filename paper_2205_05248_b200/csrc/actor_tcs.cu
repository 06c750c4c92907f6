// Split-operand tensor-core actor kernel for sm_100a: fp32 accuracy from bf16 tcgen05.mma, hidden size 64 or 128.
//
// An fp32 value is the exact sum of three bf16 values (8 + 8 + 8 significand bits, each rounded to nearest), and a
// product of two bf16 values is exact in fp32.  So a matrix product of fp32 operands is the sum of the products of
// their pieces: with x = x0 + x1 + x2 and w = w0 + w1 + w2 the six products of order 2^-16 and above are formed; what
// is left out is below 2^-24 of |x||w|.  The accumulator of tcgen05.mma adds with truncation, so the order matters:
// the five small products go first, while the accumulator is small, and x0 w0 last - few truncations at full
// magnitude.  Measured on 128 x 80 x 64 products of uniform operands: rms error 4.7e-8, largest 3.0e-7; a chain of
// fp32 fused multiply-adds: 9.4e-8 and 6.1e-7 (the six products interleaved K step by K step: 2.9e-7 and 2.1e-6).
// With one piece (NS = 1) the same kernel is the bf16 precision with accurate gate functions.
//
// One thread block owns a tile of whole environments (up to 128 agent rows) and runs all T steps of the launch for it.
// Weights stay in shared memory as far as they fit (hidden 64: all of them); the rest streams from L2 through a ring
// of slices, every step again.  The left operands - observations, fc1 output, hidden state - are written to tensor
// memory and read from there by tcgen05.mma (an A operand in shared memory costs at least 32 clocks a product, one in
// tensor memory 3 at N = 16, 27 at N = 64); only the observations and the fc1 output of the three-piece hidden-128
// variant live in shared memory.  Nothing assumes an alignment beyond that of the element type, and a tile's rows may
// be those of a list (partial steps) or of one unit type (per-type networks: the tiles of all types are dealt to the blocks
// together, those of one type before those of the next, and a block loads a type's network when it comes to its tiles; a
// pass of all blocks per type took 1045 us for 1024 environments of 2 + 3 agents, fp32, 64 steps, this takes 507).
//
// Roles: warps 0-7 epilogue (two groups of 128 threads; a thread owns one row and 16 columns of every block of 32
// hidden columns), warps 8-15 inputs and records (two groups, thread = row), warp 16 issues every tcgen05.mma (from the lane that
// elect.sync picks: 4 products take 325-400 clocks to completion against 577-700 behind "lane == 0"), warp 17 loads weights.
// Per step:
//   E1 (epilogue)  y = relu(fc1 + agent column + last-action column), pieces to the y operand
//   E2 (epilogue)  per block of 32 hidden columns: gates, new hidden state (fp32 in registers); the next block's
//                  products run meanwhile; then its pieces to the hidden operand
//   E3 (group 0)   masked greedy choice
//   inputs (beside E2) of the next step: ring cursor and headers, availability mask, epsilon draw, observation pieces
//                  and record; then this step's Q record
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "gates.cuh"
#include "launch_util.cuh"
#include "tcgen05.cuh"

namespace marl {

constexpr int TS_EPI = 256, TS_PREP = 256, TS_THREADS = 640;
constexpr int TS_UNIT = 2048;       // a staged unit of observations: 32 rows x 16 columns
constexpr int TS_ROWS = 128;
constexpr int TS_BLK = 32;          // hidden columns of a gate block
constexpr uint32_t TS_SMEM_MAX = 232448;
constexpr int TS_MAX_SLOTS = 8;
constexpr int TS_KCHUNK = 96;       // K of one W1 slice: no larger than a gate slice
// Tensor-memory columns.  Two accumulator buffers of a gate block, laid out so that the columns fc1 uses at hidden 64
// (the candidate-input parts of both) are contiguous: HN R Z IN | IN R Z HN.
// Behind them the hidden operand, the y operand, the x operand - with room for all, else x and y share columns - and Q.
constexpr uint32_t TSM_HOP = 256, TSM_COLS = 512;

struct TsLayout {
  int32_t Dk, NQ, nw1, nsl, nres, nslots;   // K of fc1; Q columns; W1 slices; slices; resident ones; ring slots
  int32_t nu;                               // staged units per input warp
  int32_t ept, ntypes;
  int32_t sep;                              // x and y operands have columns of their own
  uint32_t tm_x, tm_q;                      // first columns of x (y follows the hidden operand) and Q
  uint32_t base_bytes, off_b2, off_bias, off_tabA, off_tabL;  // base part of the image: W2 pieces, biases, column tables
  uint32_t img_bytes;
  uint32_t off_sl, off_ring, off_xy, off_scr, off_recp, off_sel, off_pick, off_la, off_close, off_eid, off_row, off_bar, total;
};

struct TsBars {
  uint64_t xrdy, srdy[4], fc1d, hset, yrdy, gd[2], accf[2], hr0, hr1, fc2d, qfree, res[2];
  uint64_t full[TS_MAX_SLOTS], empty[TS_MAX_SLOTS];
  uint32_t tmem_base, abort;
};

__host__ __device__ constexpr uint32_t ts_slice(int H) { return 96u * (uint32_t)H * 2u; }

static uint32_t ts_up(uint32_t v, uint32_t a) { return (v + a - 1) / a * a; }

// Bytes of slice i (order of use: W1, smallest pieces first; then per block the pieces of both gate matrices).
__host__ __device__ inline uint32_t ts_slice_bytes(const TsLayout& L, int H, int ns, int i) {
  if (i >= L.nw1) return ts_slice(H);
  const int c = ns == 3 ? 0 : i;
  const int k = L.Dk - c * TS_KCHUNK;
  return (uint32_t)(k < TS_KCHUNK ? k : TS_KCHUNK) * (uint32_t)H * 2u;
}
__host__ __device__ inline uint32_t ts_slice_off(const TsLayout& L, int H, int ns, int i) {  // within the slices' part
  const int w = i < L.nw1 ? i : L.nw1;
  const uint32_t w1 = ns == 3 ? (uint32_t)w * (uint32_t)L.Dk * (uint32_t)H * 2u
                              : (uint32_t)(w * TS_KCHUNK < L.Dk ? w * TS_KCHUNK : L.Dk) * (uint32_t)H * 2u;
  return w1 + (uint32_t)(i - w) * ts_slice(H);
}

// The image of one network: [W2 pieces | biases and tables (fp32) | slices].
static TsLayout ts_image(int n, int D, int A, int H, int ns) {
  TsLayout L;
  memset(&L, 0, sizeof(L));
  L.Dk = (D + 15) & ~15;
  L.NQ = A <= 16 ? 16 : 32;
  L.nw1 = ns == 3 ? 3 : (L.Dk + TS_KCHUNK - 1) / TS_KCHUNK;
  L.nsl = L.nw1 + (H / TS_BLK) * 2 * ns;
  const uint32_t tm_y = TSM_HOP + (uint32_t)(ns * H / 2);
  L.sep = tm_y + (uint32_t)(ns * (H + L.Dk) / 2 + L.NQ) <= TSM_COLS;
  L.tm_x = L.sep ? tm_y + (uint32_t)(ns * H / 2) : tm_y;
  L.tm_q = TSM_COLS - (uint32_t)L.NQ;
  uint32_t o = (uint32_t)ns * (uint32_t)H * L.NQ * 2;
  L.off_b2 = o; o += 32 * 4;
  L.off_bias = o; o += (H == 128 ? 6u : 4u) * H * 4;  // (hidden 128: reset and update again, for the fast gates)
  L.off_tabA = o; o += (uint32_t)n * (H + 4) * 4;
  L.off_tabL = o; o += (uint32_t)A * (H + 4) * 4;
  L.base_bytes = ts_up(o, 128);
  L.img_bytes = ts_up(L.base_bytes + ts_slice_off(L, H, ns, L.nsl), 256);
  return L;
}

// nt_max: rows of an environment in one tile (the agents, or those of the largest unit type).  ept = 0: does not fit.
static TsLayout ts_layout(int n, int D, int A, int H, int ns, int nt_max, int M, int sms, int ntypes = 1) {
  TsLayout L = ts_image(n, D, A, H, ns);
  int ept = TS_ROWS / nt_max;
  if (M > 0 && sms > 0) {  // even the tiles (of every type) out over the waves they need anyway
    const int tiles = (M + ept - 1) / ept * ntypes, waves = (tiles + sms - 1) / sms;
    const int per_type = waves * sms / ntypes;  // (at least 1: a type has a tile)
    const int e2 = (M + per_type - 1) / per_type;
    if (e2 < ept) ept = e2;
  }
  L.ept = ept;
  L.ntypes = ntypes;
  uint32_t o = L.base_bytes;
  L.off_xy = o;
  if (ns == 3 && H == 128) o += 3u * (uint32_t)(L.Dk > H ? L.Dk : H) * TS_ROWS * 2;
  L.off_bar = o; o += (uint32_t)sizeof(TsBars);
  L.off_recp = o; o += 4u * (uint32_t)ept * 8;
  L.off_sel = o; o += 4u * TS_ROWS * 4;
  L.off_la = o; o += TS_ROWS * 4;
  L.off_close = o; o += 4u * (uint32_t)ept * 4;
  L.off_eid = o; o += (uint32_t)ept * 4;
  L.off_pick = o; o += 4u * TS_ROWS;
  L.off_row = o; o += TS_ROWS * 2;
  o = ts_up(o, 128);
  // observation units in flight: one per input warp at least, a whole step's (up to three) where there is room
  constexpr uint32_t units = (uint32_t)(TS_PREP / 32) * TS_UNIT;
  const int nu_max = (L.Dk / 16 + 1) / 2 < 3 ? (L.Dk / 16 + 1) / 2 : 3;
  L.nu = 1;
  auto more_units = [&]() {  // at the end of shared memory: shifts nothing but the end
    L.off_scr = L.total - units;
    while (L.nu < nu_max && L.total + units <= TS_SMEM_MAX) { L.nu += 1; L.total += units; }
  };
  L.off_sl = o;
  // resident slices: all of them, or what is left beside the ring (three slots where two slices are held at once)
  const uint32_t all = ts_slice_off(L, H, ns, L.nsl);
  if (o + all + units <= TS_SMEM_MAX) {
    L.nres = L.nsl;
    L.nslots = 0;
    L.off_ring = o + all;
    L.total = o + all + units;
    more_units();
    return L;
  }
  L.nslots = ns == 3 ? 3 : 2;
  if (o + units + (uint32_t)L.nslots * ts_slice(H) > TS_SMEM_MAX) {
    L.ept = 0;
    return L;
  }
  const uint32_t room = TS_SMEM_MAX - o - units - (uint32_t)L.nslots * ts_slice(H);
  while (ts_slice_off(L, H, ns, L.nres + 1) <= room) L.nres += 1;
  L.off_ring = o + ts_slice_off(L, H, ns, L.nres);
  while (L.nslots < TS_MAX_SLOTS && L.off_ring + (uint32_t)(L.nslots + 1) * ts_slice(H) + units <= TS_SMEM_MAX) L.nslots += 1;
  L.total = L.off_ring + (uint32_t)L.nslots * ts_slice(H) + units;
  more_units();
  return L;
}

static int ts_pieces(int prec) { return prec == MARL_PRECISION_FP32 ? 3 : 1; }

// Shapes this kernel takes: the operands fit their tensor-memory columns and what must be resident fits shared memory.
// At hidden 64 everything is resident (the products are issued in an order that is not the stream's).
bool tcs_supported(int n, int D, int A, int H, int prec) {
  const int ns = ts_pieces(prec);
  const TsLayout L = ts_layout(n, D, A, H, ns, 1, 0, 0);  // one-row environments: the largest per-tile arrays
  if (L.ept == 0) return false;
  if (H == 64 && L.nres < L.nsl) return false;
  if (ns == 3 && L.Dk > TS_KCHUNK) return false;
  const uint32_t xcols = (uint32_t)(ns * (L.Dk > H ? L.Dk : H) / 2);
  return (ns == 3 && H == 128) || L.sep || TSM_HOP + (uint32_t)(ns * H / 2) + xcols <= L.tm_q;
}

// Dense launches with the hardware's gate functions: bf16 at hidden size 128 on the shapes of the scenarios' teams (the
// domain that the header states for the pipelined kernel at this size).
bool tcs_fast_supported(int n, int D, int A, int H, int prec) {
  return prec == MARL_PRECISION_BF16 && H == 128 && n >= 4 && D <= 256 && D % 8 == 0 && A <= 16 && (n * A) % 16 == 0 &&
         tcs_supported(n, D, A, H, prec);
}

size_t tcs_image_bytes(int n, int D, int A, int H, int prec) {
  return tcs_supported(n, D, A, H, prec) ? ts_image(n, D, A, H, ts_pieces(prec)).img_bytes : 0;
}

static uint16_t ts_bf16(float v) {  // round to nearest even
  uint32_t u;
  memcpy(&u, &v, 4);
  if ((u & 0x7FFFFFFFu) > 0x7F800000u) return (uint16_t)(u >> 16);
  u += 0x7FFFu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}
static float ts_float(uint16_t b) {
  const uint32_t u = (uint32_t)b << 16;
  float v;
  memcpy(&v, &u, 4);
  return v;
}

// One network into its image.  A matrix slice is [K / 8][rows][8] bf16.  Rows of a gate slice follow the accumulator
// columns of the block's buffer: y side R Z IN (buffer 0) or IN R Z, hidden side HN R Z or R Z HN.
void tcs_pack_weights(int n, int D, int A, int H, int prec, const float* W1, const float* b1, const float* Wih,
                      const float* bih, const float* Whh, const float* bhh, const float* W2, const float* b2, uint8_t* dst) {
  const int ns = ts_pieces(prec);
  const TsLayout L = ts_image(n, D, A, H, ns);
  const int I = D + n + A;
  memset(dst, 0, L.img_bytes);
  // Eight consecutive values of a row (n8 of them present) as their pieces, 16 bytes to each of to[piece].
  auto put8 = [&](const float* v, int n8, uint16_t* const (&to)[3]) {
    float r[8];
    for (int k = 0; k < 8; ++k) r[k] = k < n8 ? v[k] : 0.f;
    for (int i = 0; i < ns; ++i)
      for (int k = 0; k < 8; ++k) {
        uint16_t h = ts_bf16(r[k]);
        if (i + 1 < ns && (h & 0x7FFFu) == 0x7F80u) {
          // rounds to infinity: the largest finite piece; an infinity keeps its sign in the smallest one, so that the rest
          // of an infinite operand meets no zero, and stands in the last piece
          const bool inf = r[k] - r[k] != 0.f;
          h = (uint16_t)((h & 0x8000u) | (!inf ? 0x7F7Fu : i == 0 ? 0x0080u : 0u));
          to[i][k] = h;
          if (!inf) r[k] -= ts_float(h);
          continue;
        }
        to[i][k] = h;
        r[k] -= ts_float(h);
      }
  };
  // rows of a K-major matrix: row r of the source's `cols` columns from k0 on to row (r0 + r) of `rows` in base[piece]
  auto put_rows = [&](const float* src, size_t stride, int nrows, int k0, int k1, uint16_t* const (&base)[3], int rows, int r0) {
    for (int r = 0; r < nrows; ++r)
      for (int k = k0; k < k1; k += 8) {
        uint16_t* to[3];
        for (int i = 0; i < ns; ++i) to[i] = base[i] + ((size_t)((k - k0) / 8) * rows + r0 + r) * 8;
        put8(src + r * stride + k, k1 - k < 8 ? k1 - k : 8, to);
      }
  };
  uint16_t* w2 = reinterpret_cast<uint16_t*>(dst);
  {
    uint16_t* const base[3] = {w2, w2 + (size_t)H * L.NQ, w2 + (size_t)2 * H * L.NQ};
    put_rows(W2, H, A, 0, H, base, L.NQ, 0);
  }
  uint8_t* sl = dst + L.base_bytes;
  auto slice = [&](int i) { return reinterpret_cast<uint16_t*>(sl + ts_slice_off(L, H, ns, i)); };
  if (ns == 3) {  // smallest piece first
    uint16_t* const base[3] = {slice(2), slice(1), slice(0)};
    put_rows(W1, I, H, 0, D, base, H, 0);
  } else {
    for (int c = 0; c < L.nw1; ++c) {
      const int k0 = c * TS_KCHUNK, k1 = k0 + TS_KCHUNK > D ? D : k0 + TS_KCHUNK;
      uint16_t* const base[3] = {slice(c), nullptr, nullptr};
      put_rows(W1, I, H, k0, k1, base, H, 0);
    }
  }
  // gate slices of a block: three pieces h2 h1 y2 y1 h0 y0, one piece h0 y0
  for (int b = 0; b < H / TS_BLK; ++b) {
    const int buf = H == 64 ? b : (b + 1) & 1, i0 = L.nw1 + b * 2 * ns;
    // gate blocks of the source are r | z | n
    static const int rows_y[2][3] = {{0, 1, 2}, {2, 0, 1}}, rows_h[2][3] = {{2, 0, 1}, {0, 1, 2}};
    for (int hid = 0; hid < 2; ++hid) {
      uint16_t* base[3] = {slice(i0 + (ns == 3 ? (hid ? 4 : 5) : (hid ? 0 : 1))), nullptr, nullptr};
      if (ns == 3) {
        base[1] = slice(i0 + (hid ? 1 : 3));
        base[2] = slice(i0 + (hid ? 0 : 2));
      }
      uint16_t* const to[3] = {base[0], base[1], base[2]};
      for (int g = 0; g < 3; ++g)
        put_rows((hid ? Whh : Wih) + (size_t)((hid ? rows_h : rows_y)[buf][g] * H + b * TS_BLK) * H, H, TS_BLK, 0, H, to, 96, g * TS_BLK);
    }
  }
  memcpy(dst + L.off_b2, b2, sizeof(float) * A);
  // biases: reset and update as the sigmoid's exponent wants them, candidate input, candidate hidden
  float* bias = reinterpret_cast<float*>(dst + L.off_bias);
  for (int j = 0; j < H; ++j) {
    bias[j] = -TS_LOG2E * (bih[j] + bhh[j]);
    bias[H + j] = -TS_LOG2E * (bih[H + j] + bhh[H + j]);
    bias[2 * H + j] = bih[2 * H + j];
    bias[3 * H + j] = bhh[2 * H + j];
    if (H == 128) {
      bias[4 * H + j] = 0.5f * (bih[j] + bhh[j]);
      bias[5 * H + j] = 0.5f * (bih[H + j] + bhh[H + j]);
    }
  }
  auto col = [&](float v) { return ns == 1 ? ts_float(ts_bf16(v)) : v; };
  float* tabA = reinterpret_cast<float*>(dst + L.off_tabA);
  float* tabL = reinterpret_cast<float*>(dst + L.off_tabL);
  for (int j = 0; j < H; ++j) {
    for (int i = 0; i < n; ++i) tabA[i * (H + 4) + j] = b1[j] + col(W1[(size_t)j * I + D + i]);
    for (int a = 0; a < A; ++a) tabL[a * (H + 4) + j] = col(W1[(size_t)j * I + D + n + a]);
  }
}

// ------------------------------------------------------------------------------------------------
namespace {

__device__ __forceinline__ void ts_arrive(uint64_t* bar, int lane) {  // one arrival per warp
  __syncwarp();
  if (lane == 0) tc::mbar_arrive(bar);
}

// Copies 16 or 4 bytes, of which the first `bytes` are read and the others written as zeros.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ uint32_t ts_pack2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// The same, cut at the largest finite bf16.
__device__ __forceinline__ uint32_t ts_pack2_finite(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}

// The pieces of 16 consecutive values of this thread's row: piece i as 8 packed words to put(i, words).  All but the last are
// cut at the largest finite value: what bf16 would round to infinity splits into finite pieces, and an infinity stands in
// the last piece alone, which meets only the weights' first pieces - infinite pieces against weight pieces of either sign
// would be NaN.  (Finite large pieces stay below an infinite sum for weights up to some 128 in magnitude.)
template <int NS, typename Put>
__device__ __forceinline__ void ts_split16(float (&v)[16], Put put) {
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      w[j] = i + 1 < NS ? ts_pack2_finite(v[2 * j], v[2 * j + 1]) : ts_pack2(v[2 * j], v[2 * j + 1]);
      if (i + 1 < NS) {
        v[2 * j] -= __uint_as_float(w[j] << 16);
        v[2 * j + 1] -= __uint_as_float(w[j] & 0xFFFF0000u);
      }
    }
    put(i, w);
  }
}

// The same with the hardware's tanh (bf16 rollouts at hidden size 128, which have always used it): sigmoid(v) =
// 0.5 tanh(v / 2) + 0.5, b[0] and b[1] halved.  Three special functions per column.
__device__ __forceinline__ float ts_tanh_hw(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void ts_gates2_fast(const float (&v)[4][2], const ts_f2 (&b)[4], float& h0, float& h1) {
  const ts_f2 half = f2(0.5f);
  float r0, r1, z0, z1, u0, u1;
  f2_get(f2_fma(f2(v[0][0], v[0][1]), half, b[0]), r0, r1);
  f2_get(f2_fma(f2(v[1][0], v[1][1]), half, b[1]), z0, z1);
  const ts_f2 rg = f2_fma(f2(ts_tanh_hw(r0), ts_tanh_hw(r1)), half, half);
  const ts_f2 zg = f2_fma(f2(ts_tanh_hw(z0), ts_tanh_hw(z1)), half, half);
  f2_get(f2_fma(rg, f2_add(f2(v[3][0], v[3][1]), b[3]), f2_add(f2(v[2][0], v[2][1]), b[2])), u0, u1);
  const ts_f2 c = f2(ts_tanh_hw(u0), ts_tanh_hw(u1));
  f2_get(f2_fma(zg, f2_fma(c, f2(-1.0f), f2(h0, h1)), c), h0, h1);
}

// D (+)= A B^T, issued by one lane; A in shared memory (AS: descriptor) or in tensor memory (column address).  Descriptors go
// by their low words: the warp that issues has few registers (within 1 % of 64-bit ones either way in every shape timed).
template <bool AS>
__device__ __forceinline__ void ts_mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
  if (AS) tc::mma_bf16_lo(d, a, b, idesc, acc);
  else tc::mma_bf16_ts_lo(d, a, b, idesc, acc);
}
__device__ __forceinline__ uint32_t ts_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | ((lbo >> 4) << 16); }

}  // namespace

template <int NS, int NQ, int H, bool TYPED, bool FAST = false>
__global__ void __launch_bounds__(TS_THREADS, 1)
    actor_tcs_kernel(const __grid_constant__ ActorParams p, const __grid_constant__ TsLayout L) {
  using namespace tc;
  constexpr int NBLK = H / TS_BLK, KH = H / 16;
  // The epilogue's loops over blocks: rolled for one piece at hidden 64 (the shorter code misses the instruction cache
  // less: 353 us against 400 for 4096 x 3 agents x 64 steps), unrolled where the hidden state's registers would have to
  // rotate further (hidden 128: 3394 us against 3997, one launch repeated on the same inputs) or the pieces' arithmetic hides the misses (fp32: 1047
  // against 1064).
  constexpr int UB = NS == 1 && H == 64 ? 1 : NBLK;
  constexpr bool XS = NS == 3 && H == 128;       // x and y pieces in shared memory
  constexpr uint32_t TSM_Y = TSM_HOP + NS * H / 2;
  constexpr uint32_t FC1 = H == 64 ? 96 : 0;     // fc1's accumulator: the candidate-input columns, or buffer 0
  // Registers (setmaxnreg): launched with 96 a thread (640 * 96 = 61440); afterwards
  // 256 * 128 + 256 * 88 + 128 * 48 = 61440, at one piece and hidden 128 256 * 136 + 256 * 72 + 128 * 64: there the epilogue and
  // the issuing warp spill less.  (bf16, accurate gates, narrow -> wide split: 70 environments x 3 agents x 78 steps 595 -> 583 us,
  // 4001 x 5 x 16 steps 320 -> 323.  Per-type networks keep the narrow one: 1024 x 5 agents x 64 steps 653 us, 664.)
  constexpr bool WIDE = NS == 1 && H == 128 && !TYPED;
  constexpr int REGS_EPI = WIDE ? 136 : 128, REGS_PREP = WIDE ? 72 : 88, REGS_SVC = WIDE ? 64 : 48;
  extern __shared__ __align__(1024) uint8_t smem[];
  TsBars* B = reinterpret_cast<TsBars*>(smem + L.off_bar);
  // per-step hand-offs, four buffers each: the input warps run up to two steps ahead of the choice
  unsigned long long* recp_s = reinterpret_cast<unsigned long long*>(smem + L.off_recp);  // [4][ept] record of the step, 0: none
  uint32_t* mask_s = reinterpret_cast<uint32_t*>(smem + L.off_sel);                       // [4][128] availability
  int8_t* pick_s = reinterpret_cast<int8_t*>(smem + L.off_pick);                          // [4][128] random pick or -1
  int32_t* close_s = reinterpret_cast<int32_t*>(smem + L.off_close);                      // [4][ept] the episode ends with the step
  int32_t* la_s = reinterpret_cast<int32_t*>(smem + L.off_la);
  int32_t* eid_s = reinterpret_cast<int32_t*>(smem + L.off_eid);                          // environment's index in the actor
  uint8_t* rowel_s = smem + L.off_row;                                                    // [128] environment of the row, in the tile
  uint8_t* rowag_s = rowel_s + TS_ROWS;                                                   // [128] agent of the row
  const float* b2_s = reinterpret_cast<const float*>(smem + L.off_b2);
  const float* bias_s = reinterpret_cast<const float*>(smem + L.off_bias);
  volatile uint32_t* abortf = &B->abort;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = p.n, D = p.D, A = p.A, T = p.T, ept = L.ept;
  const bool lag = p.lagged != 0;
  const int ntypes = TYPED ? L.ntypes : 1;
  const uint32_t rec_bytes = p.rl.rec_bytes;

  if (tid == 0) {
    mbar_init(&B->xrdy, TS_PREP / 32);
    for (int i = 0; i < 4; ++i) mbar_init(&B->srdy[i], TS_PREP / 32);
    mbar_init(&B->fc1d, 1);
    mbar_init(&B->hset, TS_EPI / 32);
    mbar_init(&B->yrdy, TS_EPI / 32);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&B->gd[i], 1);
      mbar_init(&B->accf[i], TS_EPI / 32);
      mbar_init(&B->res[i], 1);
    }
    mbar_init(&B->hr0, TS_EPI / 32);
    mbar_init(&B->hr1, TS_EPI / 32);
    mbar_init(&B->fc2d, 1);
    mbar_init(&B->qfree, TS_PREP / 64);
    for (int i = 0; i < TS_MAX_SLOTS; ++i) {
      mbar_init(&B->full[i], 1);
      mbar_init(&B->empty[i], 1);
    }
    B->abort = 0;
    mbar_init_fence();
  }
  if (warp == 16) tmem_alloc(&B->tmem_base, 512);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = B->tmem_base;
  // With one network a tile has the rows of all n agents.  The input and epilogue warps of most variants take that n from a register
  // that the compiler does not know to be the parameter: it then keeps fewer of a tile's addresses alive across the steps (bf16,
  // 40001 environments x 3 agents x 16 steps 635 -> 623 us; 4001 x 3 with 20 actions at hidden 128 200 -> 194; fp32 at hidden 128,
  // 2001 x 8, 462 -> 456).  Not with the hardware's gates (2001 x 8 agents x 32 steps 246 -> 253) and in fp32 at hidden 64 (one step of
  // 9001 x 5 agents 52.0 -> 52.4).
  constexpr bool HIDE_NT = !TYPED && !FAST && !(NS == 3 && H == 64);
  auto rows_per_env = [&](int typ) -> int {  // of a pass: the agents of its unit type
    int nt = ntypes > 1 ? 0 : n;
    if (ntypes > 1)
      for (int i = 0; i < n; ++i) nt += (int)((p.agent_type_bits >> (2 * i)) & 3ull) == typ ? 1 : 0;
    return nt;
  };
  // Work units: the tiles of type 0, then those of type 1, ...; a block takes every gridDim.x-th.  With one network nothing of
  // this is left in the kernel: walking types at run time cost shared networks up to 4 % (fp32 at hidden 128, 2001 environments x
  // 8 agents x 16 steps, 481 against 457 us; bf16, 4001 x 5 agents at hidden 128, 339 against 319).
  const int my_tiles = (p.num_tiles * ntypes - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  auto unit_at = [&](int& tile, int& typ) -> bool {  // moves a tile number beyond its type's tiles on to the next type
    if constexpr (TYPED) {
      while (tile >= p.num_tiles) {
        tile -= p.num_tiles;
        if (++typ == ntypes) return false;
      }
      return true;
    } else {
      return tile < p.num_tiles;
    }
  };

  if (warp >= 16) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_SVC));
    if (warp == 16) {
      // =========================== MMA warp ===========================
      grid_wait();  // (no bounded wait may include the run time of the kernel before: its inputs arrive only after that)
      if (my_tiles * T <= 2) grid_release();  // (the input warps would come to it too late to gain from it)
      const uint32_t sb = smem_u32(smem);
      constexpr uint32_t id96 = idesc_bf16_f32(128, 96), id64 = idesc_bf16_f32(128, 64), id32 = idesc_bf16_f32(128, 32),
                         idH = idesc_bf16_f32(128, H), idq = idesc_bf16_f32(128, NQ);
      constexpr uint32_t ks_1 = (2 * H * 16) >> 4, ks_g = (2 * 96 * 16) >> 4, ks_q = (2 * NQ * 16) >> 4, st_q = (H / 16) * ks_q;
      const int nk1 = L.Dk / 16;
      // the left operands and the distance between their pieces and K steps
      const uint32_t a_h = tmem + TSM_HOP;
      constexpr uint32_t h_st = H / 2, h_ks = 8;
      const uint32_t a_x = XS ? ts_lo(sb + L.off_xy, 2048) : tmem + L.tm_x;
      const uint32_t a_y = XS ? a_x : tmem + TSM_Y;
      constexpr uint32_t x_ks = XS ? (2 * 2048) >> 4 : 8;
      const uint32_t x_st = (uint32_t)nk1 * x_ks;
      constexpr uint32_t y_st = KH * x_ks;
      uint32_t g = 0, ri = 0, rpar = 0;  // steps so far; ring slot and its parity
      uint32_t loads = TYPED ? 0 : 1;  // networks loaded so far
      bool first = true;

      // slice i of the step: its address once it is in shared memory
      auto get = [&](int i) -> uint32_t {
        if (i < L.nres) {
          if (first) mbar_wait(&B->res[i < L.nw1 ? 0 : 1], (loads - 1) & 1, abortf);
          return sb + L.off_sl + ts_slice_off(L, H, NS, i);
        }
        mbar_wait(&B->full[ri], rpar, abortf);
        return sb + L.off_ring + ri * ts_slice(H);
      };
      auto next_slot = [&]() {
        if (++ri == (uint32_t)L.nslots) { ri = 0; rpar ^= 1u; }
      };

      // The gate products of one piece pair over all K steps.  (Measured per product
      // of N = 64: 30 clocks in rolled loops around four unrolled ones, 56 in a loop over single ones.)
      // side 1: hidden, side 0: y, whose first product of a step starts the candidate-input columns.
      auto prod = [&](int buf, int hid, uint32_t ai, uint32_t w, uint32_t acc) {
        const uint32_t d = tmem + (hid ? (buf ? 160u : 0u) : (buf ? 128u : 32u));
        if (XS && !hid) {
          const uint32_t a = a_y + ai * y_st;
          if (acc) {
            ts_mma<true>(d, a, w, id96, 1);
          } else {  // buffer 0: R Z at rows 0.., IN at rows 64..; buffer 1: IN at rows 0.., R Z at rows 32..
            ts_mma<true>(d + (buf ? 0u : 64u), a, w + (buf ? 0u : (64u * 16u) >> 4), id32, 0);
            ts_mma<true>(d + (buf ? 32u : 0u), a, w + (buf ? (32u * 16u) >> 4 : 0u), id64, 1);
          }
#pragma unroll
          for (int ks = 1; ks < KH; ++ks) ts_mma<true>(d, a + ks * x_ks, w + ks * ks_g, id96, 1);
        } else {
          const uint32_t a = hid ? a_h + ai * h_st : a_y + ai * y_st;
          if (hid || acc) {
            ts_mma<false>(d, a, w, id96, acc);
          } else {
            ts_mma<false>(d + (buf ? 0u : 64u), a, w + (buf ? 0u : (64u * 16u) >> 4), id32, 0);
            ts_mma<false>(d + (buf ? 32u : 0u), a, w + (buf ? (32u * 16u) >> 4 : 0u), id64, 1);
          }
#pragma unroll
          for (int ks = 1; ks < KH; ++ks) ts_mma<false>(d, a + ks * 8, w + ks * ks_g, id96, 1);
        }
      };

      // fc1 at hidden 64, where all weights are resident: no slices to look up (fp32, one step of 8 environments x 3 agents 11.5 ->
      // 10.6 us, 2001 x 5 agents x 16 steps 147.7 -> 138.6)
      const uint32_t w1_lo = ts_lo(sb + L.off_sl, H * 16), w1_st = (uint32_t)(L.Dk * H * 2) >> 4;
      const uint32_t wg_lo = ts_lo(sb + L.off_sl + ts_slice_off(L, H, NS, L.nw1), 1536);
      auto fc1_resident = [&]() {
        if (elect_one()) {
          // (left piece, slice): (0,0) (1,1) (0,1) (2,2) (1,2) (0,2) - the slices lie smallest piece first
          constexpr uint32_t LA = 0x012010u, SA = 0x222110u;
#pragma unroll 1
          for (int j = 0; j < (NS == 3 ? 6 : 1); ++j) {
            uint32_t a = tmem + L.tm_x, w = w1_lo, acc = j > 0;
            if (NS == 3) {
              a += ((LA >> (4 * j)) & 15u) * (uint32_t)(nk1 * 8);
              w += ((SA >> (4 * j)) & 15u) * w1_st;
            }
            int ks = 0;
#pragma unroll 1
            for (; ks + 2 <= nk1; ks += 2, a += 16, w += 2 * ks_1, acc = 1) {
              ts_mma<false>(tmem + FC1, a, w, idH, acc);
              ts_mma<false>(tmem + FC1, a + 8, w + ks_1, idH, 1);
            }
            if (ks < nk1) ts_mma<false>(tmem + FC1, a, w, idH, acc);
          }
          mma_commit(&B->fc1d);
        }
        __syncwarp();
      };

      // The steps of all tiles of a type are one loop: this warp has few registers, and of tile and step only the number of
      // steps left stays alive (fp32 at hidden 128, 2001 environments x 8 agents x 16 steps: 477 us with a loop over tiles around
      // one over steps, 460 with this one; hidden 128 in bf16, the same rows x 32 steps, 253 and 244).
      for (int typ = 0, tile = blockIdx.x; typ < ntypes; ++typ, tile -= p.num_tiles) {
        if (TYPED && tile >= p.num_tiles) continue;   // no tile of this type is the block's
        if (TYPED && loads++ > 0) __syncthreads();    // every role has left the previous type
        const int tiles = (p.num_tiles - 1 - tile) / (int)gridDim.x + 1;
        if (TYPED) tile += tiles * (int)gridDim.x;
        first = true;
#pragma unroll 1
        for (int left = tiles * T; left > 0; --left, ++g, first = false) {
          const uint32_t par = g & 1;
          // ---- fc1 ----
          if (H == 64) {
            mbar_wait(&B->xrdy, par, abortf);  // (E2 of the previous step has read the columns: hr1)
            if (first) mbar_wait(&B->res[0], (loads - 1) & 1, abortf);
            tc_fence_after_sync();
            fc1_resident();
          } else {
            mbar_wait(&B->xrdy, par, abortf);  // (E2 of the previous step has read the columns: hr1)
            tc_fence_after_sync();
            for (int i = 0; i < L.nw1; ++i) {
              const uint32_t w = ts_lo(get(i), H * 16);
              if (elect_one()) {
                // piece 2 - i against the small products' left pieces, then the main product (one piece: the slice's)
                const int k0 = NS == 3 ? 0 : i * (TS_KCHUNK / 16), nk = min(nk1 - k0, TS_KCHUNK / 16);
#pragma unroll 1
                for (int ai = NS == 3 ? i : 0; ai >= 0; --ai) {
                  uint32_t a = a_x + (uint32_t)ai * x_st + (uint32_t)k0 * x_ks, wk = w;
                  uint32_t acc = i > 0 || (NS == 3 && ai < i);
                  int ks = 0;
#pragma unroll 1
                  for (; ks + 2 <= nk; ks += 2, a += 2 * x_ks, wk += 2 * ks_1, acc = 1) {
                    ts_mma<XS>(tmem + FC1, a, wk, idH, acc);
                    ts_mma<XS>(tmem + FC1, a + x_ks, wk + ks_1, idH, 1);
                  }
                  if (ks < nk) ts_mma<XS>(tmem + FC1, a, wk, idH, acc);
                }
                if (i >= L.nres) mma_commit(&B->empty[ri]);
                if (i == L.nw1 - 1) mma_commit(&B->fc1d);
              }
              __syncwarp();
              if (i >= L.nres) next_slot();
            }
          }
          // ---- gates ----
          if (H == 64) {
            // everything resident: the hidden side's first products run before the fc1 output is there
            mbar_wait(&B->hset, par, abortf);
            if (first) mbar_wait(&B->res[1], (loads - 1) & 1, abortf);
            tc_fence_after_sync();
            constexpr uint32_t SL = ts_slice(64) >> 4;
            // pieces of the small products in order: left, and slice of the hidden and of the y side
            constexpr uint32_t LEFT = 0x10210u, SH = 0x41410u, SY = 0x53532u;
            if (elect_one()) {
#pragma unroll 1
              for (int b = 0; b < NBLK; ++b)
#pragma unroll 1
                for (int j = 0; j < (NS == 3 ? 5 : 1); ++j)
                  prod(b, 1, (LEFT >> (4 * j)) & 15u, wg_lo + (uint32_t)(b * 2 * NS) * SL + (NS == 3 ? (SH >> (4 * j)) & 15u : 0u) * SL, j > 0);
            }
            __syncwarp();
            mbar_wait(&B->yrdy, par, abortf);
            tc_fence_after_sync();
            if (elect_one()) {
#pragma unroll 1
              for (int b = 0; b < NBLK; ++b) {
                const uint32_t wb = wg_lo + (uint32_t)(b * 2 * NS) * SL;
                if (NS == 3) {
#pragma unroll 1
                  for (int j = 0; j < 7; ++j)  // five small ones, then the main products
                    prod(b, j == 5, j < 5 ? (LEFT >> (4 * j)) & 15u : 0u, wb + (j < 5 ? (SY >> (4 * j)) & 15u : (uint32_t)j - 1u) * SL, j > 0);
                } else {
                  prod(b, 0, 0, wb + SL, 0);
                }
                mma_commit(&B->gd[b]);
              }
            }
            __syncwarp();
          } else {
            int i = L.nw1;
#pragma unroll 1
            for (int b = 0; b < NBLK; ++b) {
              const int buf = (b + 1) & 1;
              if (b == 0) {
                mbar_wait(&B->hset, par, abortf);
              } else if (b >= 2) {
                mbar_wait(&B->accf[buf], par, abortf);
              }
              tc_fence_after_sync();
              if (NS == 3) {
                // h2, h1, y2, y1, then h0 and y0 held together: their small products come before both main ones
                uint32_t wh = 0;
                uint32_t rh = 0;
#pragma unroll 1
                for (int k = 0; k < 6; ++k, ++i) {
                  if (b == 0 && k == 2) {
                    mbar_wait(&B->yrdy, par, abortf);
                    tc_fence_after_sync();
                  }
                  const uint32_t w = ts_lo(get(i), 1536);
                  const int hid = k < 2 || k == 4;
                  if (k == 4) { wh = w; rh = ri; }
                  if (elect_one()) {
                    // left pieces: k = 0, 2: 0; 1, 3: 1 0; 4, 5: 2 1; after the last the main products
                    const int first_ai = k >= 4 ? 2 : k & 1, last_ai = k >= 4 ? 1 : 0;
#pragma unroll 1
                    for (int ai = first_ai; ai >= last_ai - (k == 5 ? 2 : 0); --ai) {
                      const bool main = ai < last_ai, mh = main && ai == 0;  // (k == 5: 0 stands for the hidden main, -1 for the y main)
                      prod(buf, main ? mh : hid, main ? 0u : (uint32_t)ai, mh ? wh : w, !((k == 0 || k == 2) && ai == first_ai));
                      if (mh && i - 1 >= L.nres) mma_commit(&B->empty[rh]);
                    }
                    if (i >= L.nres && k != 4) mma_commit(&B->empty[ri]);
                    if (k == 5) mma_commit(&B->gd[buf]);
                  }
                  __syncwarp();
                  if (i >= L.nres) next_slot();
                }
              } else {
                const uint32_t wh = ts_lo(get(i), 1536);
                if (elect_one()) {
                  prod(buf, 1, 0, wh, 0);
                  if (i >= L.nres) mma_commit(&B->empty[ri]);
                }
                __syncwarp();
                if (i >= L.nres) next_slot();
                ++i;
                const uint32_t wy = ts_lo(get(i), 1536);
                if (b == 0) {
                  mbar_wait(&B->yrdy, par, abortf);
                  tc_fence_after_sync();
                }
                if (elect_one()) {
                  prod(buf, 0, 0, wy, 0);
                  if (i >= L.nres) mma_commit(&B->empty[ri]);
                  mma_commit(&B->gd[buf]);
                }
                __syncwarp();
                if (i >= L.nres) next_slot();
                ++i;
              }
            }
          }
          // ---- fc2: the small products of all blocks but the last, then the rest ----
          if (g > 0) mbar_wait(&B->qfree, par ^ 1u, abortf);  // the previous step's Q has been read
          const uint32_t w2 = ts_lo(sb, NQ * 16);
          constexpr int K1 = KH - TS_BLK / 16;  // K steps of the earlier blocks
          auto part_q = [&](auto half_c) {  // K steps [0, K1) or [K1, KH); the second part ends with the main product
            constexpr int half = decltype(half_c)::value, k0 = half ? K1 : 0, k1 = half ? KH : K1;
            mbar_wait(half ? &B->hr1 : &B->hr0, par, abortf);
            tc_fence_after_sync();
            if (elect_one()) {
              if (NS == 3) {  // small products (left, right): (2,0) (1,1) (0,2) (1,0) (0,1)
#pragma unroll 1
                for (int j = 0; j < 5; ++j) {
                  const uint32_t a = a_h + ((0x01012u >> (4 * j)) & 15u) * h_st, w = w2 + ((0x10210u >> (4 * j)) & 15u) * st_q;
#pragma unroll
                  for (int ks = k0; ks < k1; ++ks) ts_mma<false>(tmem + L.tm_q, a + ks * h_ks, w + ks * ks_q, idq, ks > 0 || j > 0);
                }
              }
              if (NS == 1 || half)
#pragma unroll
                for (int ks = NS == 3 ? 0 : k0; ks < k1; ++ks) ts_mma<false>(tmem + L.tm_q, a_h + ks * h_ks, w2 + ks * ks_q, idq, NS == 3 || ks > 0);
              if (half) mma_commit(&B->fc2d);
            }
            __syncwarp();
          };
          part_q(std::integral_constant<int, 0>());
          part_q(std::integral_constant<int, 1>());
        }
      }
    } else if (warp == 17) {
      // =========================== weight warp ===========================
      uint32_t ri = 0, rpar = 1, used = 0;
      for (int tile = blockIdx.x, typ = 0, cur = -1; unit_at(tile, typ); tile += gridDim.x) {
        if (typ == cur) {
          if (!TYPED) break;
          continue;
        }
        if (TYPED && cur >= 0) __syncthreads();
        cur = typ;
        const uint8_t* img = reinterpret_cast<const uint8_t*>(p.wsplit) + (size_t)typ * p.wsplit_stride;
        const uint8_t* sl = img + L.base_bytes;
        if (lane == 0) {
          // resident part: the base and W1 first, then the gate slices
          const int r1 = min(L.nres, L.nw1);
          const uint32_t b1 = ts_slice_off(L, H, NS, r1), b2 = ts_slice_off(L, H, NS, L.nres);
          mbar_arrive_expect_tx(&B->res[0], L.base_bytes + b1);
          bulk_load(smem, img, L.base_bytes, &B->res[0]);
          if (b1) bulk_load(smem + L.off_sl, sl, b1, &B->res[0]);
          mbar_arrive_expect_tx(&B->res[1], b2 - b1);
          for (uint32_t o = b1; o < b2; o += 32768u) bulk_load(smem + L.off_sl + o, sl + o, min(32768u, b2 - o), &B->res[1]);
        }
        __syncwarp();
        if (L.nres < L.nsl) {
          const int steps = ((p.num_tiles - 1 - tile) / (int)gridDim.x + 1) * T;
          for (int g = 0; g < steps; ++g)
            for (int i = L.nres; i < L.nsl; ++i) {
              if (used >= (uint32_t)L.nslots) {
                mbar_wait(&B->empty[ri], rpar, abortf);
              } else if (++used == (uint32_t)L.nslots) {
                grid_wait();  // what is loaded so far was the weights' alone; the ring moves on with the steps
              }
              if (lane == 0) {
                const uint32_t bytes = ts_slice_bytes(L, H, NS, i);
                mbar_arrive_expect_tx(&B->full[ri], bytes);
                bulk_load(smem + L.off_ring + ri * ts_slice(H), sl + ts_slice_off(L, H, NS, i), bytes, &B->full[ri]);
              }
              __syncwarp();
              if (++ri == (uint32_t)L.nslots) {
                ri = 0;
                rpar ^= 1u;
              }
            }
        }
      }
    } else if (TYPED) {
      for (int tile = blockIdx.x, typ = 0, cur = -1; unit_at(tile, typ); tile += gridDim.x) {
        if (typ != cur && cur >= 0) __syncthreads();
        cur = typ;
      }
    }
  } else if (warp >= 8) {
    // =========================== inputs and records ===========================
    // Two groups of four warps share a tile's rows (row = lane of tensor memory): both convert observations, in turn
    // unit by unit (16 columns); group 0 also makes the masks and draws and records the availability, group 1 keeps the
    // ring cursors (of environment `row` of the tile), headers and outcomes and records Q.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_PREP));
    grid_wait();
    auto inputs = [&](auto grp_c) {  // (the group as a constant: each group's code keeps only its own registers)
    constexpr int grp = decltype(grp_c)::value;
    const int row = tid & 127, pw = warp & 3;
    const uint32_t tm = tmem + ((uint32_t)(pw * 32) << 16);
    const int nk = L.Dk / 16, nloc = (nk + 1 - grp) / 2;  // units of a step; this group's (2 k + grp)
    // Units are staged by cp.async: loads that return to registers need a line of L1 each while in flight, and beside
    // 227 KB of shared memory there are too few (a step's requests took 5 k clocks to issue).
    uint8_t* units = smem + L.off_scr + (warp - 8) * L.nu * TS_UNIT;
    const int c4 = lane & 3;  // the unit's columns 4 c4 .. of rows 8 j + lane / 4 are this lane's to copy
    const bool vec = (D & 3) == 0 && (reinterpret_cast<uintptr_t>(p.obs) & 15) == 0;
    uint32_t c_episodes = 0, c_trunc = 0, st_bits = 0, g = 0, loads = TYPED ? 0 : 1;
    int nt = n;
    if constexpr (HIDE_NT) asm volatile("" : "+r"(nt));
    bool fresh = true;
    for (int tile = blockIdx.x, typ = 0, cur = -1; unit_at(tile, typ); tile += gridDim.x) {
      if (TYPED && typ != cur) {
        cur = typ;
        nt = rows_per_env(typ);
        fresh = true;
        if (loads++ > 0) __syncthreads();
      }
      const int e0 = tile * ept;
      const int ne = min(ept, p.M - e0);
      const int R = ne * nt;
      const bool wlive = pw * 32 < R;   // warps without a live row only keep the barriers going
      const bool live = row < R;
      const bool cursor = grp == 1 && row < ne;
      int32_t slot = 0, pos = 0, eok = 0;
      long long epc = 0;
      asm volatile("bar.sync 2, 512;" ::: "memory");  // the previous tile's shared arrays are done with
      if (cursor) {
        const int e = p.env_ids ? __ldg(p.env_ids + e0 + row) : e0 + row;
        slot = p.slot[e];
        pos = p.pos[e];
        epc = p.ep_count[e];
        // (with late outcomes a full slot waits, at pos == L, for its last outcome before it is truncated)
        eok = (slot >= 0 && slot < p.E * p.S && pos >= 0 && pos < p.L + (lag ? 1 : 0)) ? 1 : 0;
        if (!eok) st_bits |= MARL_STATUS_BAD_INDEX;
        int closed = 0;
        if (lag && eok && pos > 0) {
          // the outcome of the previous action completes the record at pos - 1 and may close the episode
          const float r = p.reward[e0 + row];
          const int d = p.done[e0 + row] ? 1 : 0;
          if (typ == 0) {
            uint8_t* rec = p.ring + (size_t)slot * p.slot_stride + (size_t)(pos - 1) * rec_bytes;
            *reinterpret_cast<float*>(rec + p.rl.off_reward) = r;
            rec[p.rl.off_done] = (uint8_t)d;
          }
          if (d || pos == p.L) {
            if (typ == 0) {
              p.slot_len[slot] = pos;
              p.slot_complete[slot] = 1;
              c_episodes += 1;
              if (!d) c_trunc += 1;
            }
            epc += 1;
            slot = e * p.S + (int)(epc % p.S);
            pos = 0;
            closed = 1;
          }
        }
        eid_s[row] = e;
        close_s[((g + 3) & 3) * ept + row] = closed;  // (as if by the step before the first)
      }
      asm volatile("bar.sync 2, 512;" ::: "memory");
      const int el = rowel_s[row], ai = rowag_s[row];
      const int e = eid_s[el];
      int soff[4], poff[4];  // offset of the lane's first column in the tile's observations and in its record (floats)
      uint32_t uel = 0, ulive = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = pw * 32 + 8 * j + (lane >> 2);
        soff[j] = (rowel_s[r] * n + rowag_s[r]) * D + 4 * c4;
        poff[j] = rowag_s[r] * D + 4 * c4;
        uel |= (uint32_t)rowel_s[r] << (8 * j);
        ulive |= (r < R ? 1u : 0u) << j;
      }

      // ---- staging: unit `rq` of the group's sequence over (step, unit) goes to slot rq % nu ----
      int rq_s = 0, rq_k = 0, rq_slot = 0, cv_slot = 0;
      auto request_unit = [&]() {  // one cp.async group per call, empty at the end
        if (wlive && rq_s < T) {
          const int c = (2 * rq_k + grp) * 16 + 4 * c4;  // first column
          const float* obs = p.obs + (size_t)rq_s * p.obs_step_stride + (size_t)e0 * n * D + (c - 4 * c4);
          uint8_t* to = units + rq_slot * TS_UNIT;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int r = 8 * j + (lane >> 2);
            const uint32_t dst = smem_u32(to) + (uint32_t)(r * 64 + ((c4 ^ ((r >> 1) & 3)) * 16));
            const int left = (ulive >> j) & 1u ? D - c : 0;  // columns there are; the others become zeros
            const float* src = left > 0 ? obs + soff[j] : p.obs;
            if (vec) {
              cp_async16(dst, src, left > 0 ? 16u : 0u);
            } else {
#pragma unroll
              for (int k = 0; k < 4; ++k) cp_async4(dst + 4 * k, left > k ? src + k : p.obs, left > k ? 4u : 0u);
            }
          }
          if (++rq_k == nloc) { rq_k = 0; rq_s += 1; }
          if (++rq_slot == L.nu) rq_slot = 0;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
      if (nloc > 0)
        for (int k = 0; k < L.nu; ++k) request_unit();

      float reward_next = 0.f;
      uint32_t done_next = 0;
      constexpr int AW = NQ == 16 ? 5 : 9;
      uint32_t aw[AW], ash = 0;
      // a step's small inputs, requested a step ahead
      auto request_small = [&](int s) {
        if (grp == 0 && live) {  // availability row as aligned words (up to three bytes on either side are read and dropped)
          const uintptr_t a0 = reinterpret_cast<uintptr_t>(p.avail + (size_t)s * p.avail_step_stride + ((size_t)(e0 + el) * n + ai) * A);
          const uint32_t* wp = reinterpret_cast<const uint32_t*>(a0 & ~(uintptr_t)3);
          ash = (uint32_t)(a0 & 3u);
          const uint32_t nw = (ash + (uint32_t)A + 3u) / 4u;
#pragma unroll
          for (int k = 0; k < AW; ++k) aw[k] = (uint32_t)k < nw ? __ldg(wp + k) : 0u;
        }
        if (grp == 1 && live && 2 * L.nu * 16 < D) {  // first touch of the lines whose units wait for a slot
          const float* o1 = p.obs + (size_t)s * p.obs_step_stride + ((size_t)(e0 + el) * n + ai) * D;
          for (int c = 2 * L.nu * 16; c < D; c += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(o1 + c));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(o1 + D - 1));
        }
        if (cursor && !lag) {
          reward_next = p.reward[(size_t)s * p.env_step_stride + e0 + row];
          done_next = p.done[(size_t)s * p.env_step_stride + e0 + row];
        }
      };
      request_small(0);
      unsigned long long myrec = 0, prevrec = 0;  // records of this thread's row: the step prepared, the one before

      auto prepare = [&](int s, uint32_t gk) {
        const uint32_t b = gk & 3;
        if constexpr (grp == 1) {
          if (cursor) {
            // ring cursor, headers, reward and done of this step; the cursor needs only the done flags
            unsigned long long rec = 0;
            int close = 0;
            if (eok) {
              uint8_t* rp = p.ring + (size_t)slot * p.slot_stride + (size_t)pos * rec_bytes;
              rec = reinterpret_cast<unsigned long long>(rp);
              const int done = done_next ? 1 : 0;
              close = (!lag && (done || pos + 1 == p.L)) ? 1 : 0;
              if (typ == 0) {
                if (pos == 0) {  // an episode opens in this slot
                  p.slot_epid[slot] = epc * (long long)p.E + eid_s[row];
                  p.slot_len[slot] = 0;
                  p.slot_complete[slot] = 0;
                }
                *reinterpret_cast<float*>(rp + p.rl.off_reward) = reward_next;
                rp[p.rl.off_done] = (uint8_t)done;
                if (close) {
                  p.slot_len[slot] = pos + 1;
                  p.slot_complete[slot] = 1;
                  c_episodes += 1;
                  if (!done) c_trunc += 1;
                }
              }
              if (close) {
                epc += 1;
                slot = eid_s[row] * p.S + (int)(epc % p.S);
                pos = 0;
              } else {
                pos += 1;
              }
            }
            recp_s[b * ept + row] = rec;
            close_s[b * ept + row] = close;
          }
        } else if (live) {
          unsigned long long bits = 0;
#pragma unroll
          for (int k = 0; k < AW; ++k) {
            const uint32_t v = aw[k];
            const uint32_t nz = ((v | ((v & 0x7F7F7F7Fu) + 0x7F7F7F7Fu)) & 0x80808080u) >> 7;  // 0x01 per non-zero byte
            bits |= (unsigned long long)((nz * 0x01020408u) >> 24 & 0xFu) << (4 * k);
          }
          const uint32_t mask = (uint32_t)(bits >> ash) & (A >= 32 ? 0xFFFFFFFFu : ((1u << A) - 1u));
          const uint32_t t = p.t0 + (uint32_t)s;
          const int pick = mask ? draw_explore(mask, eps_at(p, t), p.seed, t, (uint32_t)e, (uint32_t)ai) : -1;
          mask_s[b * TS_ROWS + row] = mask;
          pick_s[b * TS_ROWS + row] = (int8_t)pick;
        }
        asm volatile("bar.sync 3, 256;" ::: "memory");  // the step's records are known
        ts_arrive(&B->srdy[b], lane);
        prevrec = myrec;
        myrec = live ? recp_s[b * ept + el] : 0ull;
        if (gk > 0) {
          // the operand has been read by the previous step's fc1 or, where y takes its place, the y operand by the
          // gate products (barriers with one phase a step)
          mbar_wait(L.sep ? &B->fc1d : H == 64 ? &B->gd[1] : &B->hr0, (gk - 1) & 1, abortf);
          tc_fence_after_sync();
        }
        if (wlive) {
#pragma unroll 1
          for (int ks = grp; ks < nk; ks += 2) {
            if (L.nu == 1) asm volatile("cp.async.wait_group 0;" ::: "memory");
            else if (L.nu == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
            else asm volatile("cp.async.wait_group 2;" ::: "memory");
            __syncwarp();
            const float4* un = reinterpret_cast<const float4*>(units + cv_slot * TS_UNIT);
            float v[16];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float4 f = un[lane * 4 + (k ^ ((lane >> 1) & 3))];
              v[4 * k] = f.x; v[4 * k + 1] = f.y; v[4 * k + 2] = f.z; v[4 * k + 3] = f.w;
            }
            ts_split16<NS>(v, [&](int i, const uint32_t (&w)[8]) {
              if (XS) {
                uint8_t* to = smem + L.off_xy + (uint32_t)(i * nk + ks) * 4096u + (uint32_t)row * 16u;
                *reinterpret_cast<uint4*>(to) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(to + 2048) = make_uint4(w[4], w[5], w[6], w[7]);
              } else {
                tmem_st8(tm + L.tm_x + (uint32_t)(i * nk + ks) * 8u, w);
              }
            });
            const int c = ks * 16 + 4 * c4;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const unsigned long long rec = (ulive >> j) & 1u ? recp_s[b * ept + ((uel >> (8 * j)) & 0xFFu)] : 0ull;
              const int r = 8 * j + (lane >> 2);
              const float4 f = un[r * 4 + (c4 ^ ((r >> 1) & 3))];
              if (rec) {
                float* to = reinterpret_cast<float*>(rec + p.rl.off_obs) + poff[j] + ks * 16;
                if ((D & 3) == 0) {
                  if (c < D) *reinterpret_cast<float4*>(to) = f;
                } else {
                  if (c < D) to[0] = f.x;
                  if (c + 1 < D) to[1] = f.y;
                  if (c + 2 < D) to[2] = f.z;
                  if (c + 3 < D) to[3] = f.w;
                }
              }
            }
            __syncwarp();  // the slot has been read
            if (++cv_slot == L.nu) cv_slot = 0;
            request_unit();
          }
          if (XS) fence_proxy_async_smem();
          else tmem_st_wait();
        }
        tc_fence_before_sync();
        ts_arrive(&B->xrdy, lane);
        if (grp == 0 && myrec) {
          uint8_t* dst = reinterpret_cast<uint8_t*>(myrec + p.rl.off_avail) + ai * A;
#pragma unroll
          for (int j = 0; j < NQ / 4; ++j) {
            const uint32_t v = __funnelshift_r(aw[j], aw[j + 1], 8u * ash);  // bytes 4 j .. 4 j + 3 of the row
#pragma unroll
            for (int c = 0; c < 4; ++c)
              if (4 * j + c < A) dst[4 * j + c] = (uint8_t)(v >> (8 * c));
          }
        }
        if (s + 1 < T) request_small(s + 1);
      };

      for (int sp = 0; sp <= T; ++sp) {  // prepare step sp, then finish step sp - 1
        if (sp < T) prepare(sp, g + (uint32_t)sp);
        else prevrec = myrec;
        if constexpr (grp == 0) continue;
        if (sp == 0) {
          if (fresh) mbar_wait(&B->res[0], (loads - 1) & 1, abortf);  // the output biases are in place
          continue;
        }
        const int s = sp - 1;
        mbar_wait(&B->fc2d, (g + (uint32_t)s) & 1, abortf);
        tc_fence_after_sync();
        if (wlive) {
          uint32_t qv[NQ];
          tmem_ld16(tm + L.tm_q, *reinterpret_cast<uint32_t(*)[16]>(qv));
          if (NQ == 32) tmem_ld16(tm + L.tm_q + 16, *reinterpret_cast<uint32_t(*)[16]>(qv + NQ - 16));
          tmem_ld_wait();
          tc_fence_before_sync();
          ts_arrive(&B->qfree, lane);
          if (prevrec) {
            float* qrow = reinterpret_cast<float*>(prevrec + p.rl.off_q) + ai * A;
            if ((A & 1) == 0) {  // rows of an even number of floats start on 8-byte boundaries
#pragma unroll
              for (int a = 0; a < NQ; a += 2)
                if (a < A) *reinterpret_cast<float2*>(qrow + a) = make_float2(__uint_as_float(qv[a]) + b2_s[a], __uint_as_float(qv[a + 1]) + b2_s[a + 1]);
            } else {
#pragma unroll
              for (int a = 0; a < NQ; ++a)
                if (a < A) qrow[a] = __uint_as_float(qv[a]) + b2_s[a];
            }
          }
          const int tk = p.trace_first + s;
          if (live && tk < p.trace_cap && p.trace_q) {
            float* tq = p.trace_q + (((size_t)tk * p.E + e) * n + ai) * A;
#pragma unroll
            for (int a = 0; a < NQ; ++a)
              if (a < A) tq[a] = __uint_as_float(qv[a]) + b2_s[a];
          }
        } else {
          ts_arrive(&B->qfree, lane);
        }
      }
      g += (uint32_t)T;
      if (cursor && eok) {
        const int ee = eid_s[row];
        if (typ == 0 && pos > 0) p.slot_len[slot] = pos;
        // The types' tiles of an environment run in any order, on any block: the last one to finish writes the
        // cursor (all have read it by then, and all have come to the same one).
        bool last = true;
        if (ntypes > 1) {
          __threadfence();
          last = atomicAdd(p.type_count + ee, 1) == ntypes - 1;
          if (last) p.type_count[ee] = 0;
        }
        if (last) {
          p.slot[ee] = slot;
          p.pos[ee] = pos;
          p.ep_count[ee] = epc;
        }
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      fresh = false;
    }
    if constexpr (grp == 0) grid_release();  // the last step's inputs are in place
    if (c_episodes) atomicAdd(p.counters + CNT_EPISODES, (unsigned long long)c_episodes);
    if (c_trunc) atomicAdd(p.counters + CNT_TRUNCATED, (unsigned long long)c_trunc);
    if (st_bits) atomicOr(p.status, st_bits);
    };
    if (warp < 12) inputs(std::integral_constant<int, 0>());
    else inputs(std::integral_constant<int, 1>());
  } else {
    // =========================== epilogue ===========================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_EPI));
    grid_wait();
    const int row = tid & 127, grp = warp >> 2;
    const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t c_steps = 0, c_explore = 0, c_noavail = 0;  // (a launch's rows x steps of one thread)
    uint32_t st_bits = 0, g = 0, loads = TYPED ? 0 : 1;
    int nt = n;
    if constexpr (HIDE_NT) asm volatile("" : "+r"(nt));
    bool fresh = true;
    for (int tile = blockIdx.x, typ = 0, cur = -1; unit_at(tile, typ); tile += gridDim.x) {
      if (TYPED && typ != cur) {
        cur = typ;
        nt = rows_per_env(typ);
        fresh = true;
        if (loads++ > 0) __syncthreads();
      }
      const int e0 = tile * ept;
      const int R = min(ept, p.M - e0) * nt;
      const bool wlive = (warp & 3) * 32 < R;   // warps without a live row only keep the barriers going
      const bool live = row < R;
      asm volatile("bar.sync 2, 512;" ::: "memory");  // the previous tile's shared arrays are done with
      if (grp == 0) {
        // row -> (environment, agent): the agents of this pass' unit type, in rising order
        uint8_t el = 0, ag = 0;
        if (live) {
          el = (uint8_t)(row / nt);
          int k = row - el * nt, i = k;
          if (ntypes > 1)
            for (i = 0; i < n; ++i)
              if ((int)((p.agent_type_bits >> (2 * i)) & 3ull) == typ && k-- == 0) break;
          ag = (uint8_t)i;
        }
        rowel_s[row] = el;
        rowag_s[row] = ag;
      }
      asm volatile("bar.sync 2, 512;" ::: "memory");
      const int el = rowel_s[row], ai = rowag_s[row];
      const int e = eid_s[el];
      const size_t grow = (size_t)e * n + ai;
      float h[NBLK][16];
      auto store_h = [&](int b, const float (&hb)[16]) {  // the pieces of block b's hidden state
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = hb[j];
        ts_split16<NS>(v, [&](int i, const uint32_t (&w)[8]) {
          tmem_st8(tm + TSM_HOP + (uint32_t)(i * (H / 2) + b * (TS_BLK / 2) + grp * 8), w);
        });
      };
      {
        const bool carry = live && !close_s[((g + 3) & 3) * ept + el];  // the row continues an episode
#pragma unroll
        for (int b = 0; b < NBLK; ++b) {
          const float4* src = reinterpret_cast<const float4*>(p.h + grow * H + b * TS_BLK + grp * 16);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 v = carry ? src[k] : make_float4(0.f, 0.f, 0.f, 0.f);
            h[b][4 * k] = v.x; h[b][4 * k + 1] = v.y; h[b][4 * k + 2] = v.z; h[b][4 * k + 3] = v.w;
          }
        }
        if (grp == 0) {
          int la = carry ? p.last_action[grow] : -1;
          if (la >= A) la = -1;
          la_s[row] = la;
        }
        if (wlive) {
#pragma unroll
          for (int b = 0; b < NBLK; ++b) store_h(b, h[b]);
          tmem_st_wait();
        }
        tc_fence_before_sync();
        ts_arrive(&B->hset, lane);
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (fresh) mbar_wait(&B->res[0], (loads - 1) & 1, abortf);  // tables and biases are in place
      }
      const float* ta = reinterpret_cast<const float*>(smem + L.off_tabA) + ai * (H + 4) + grp * 16;
      const float* tl0 = reinterpret_cast<const float*>(smem + L.off_tabL) + grp * 16;

      for (int s = 0; s < T; ++s, ++g) {
        const uint32_t par = g & 1u, b4 = g & 3u;
        // ---- E1 ----
        mbar_wait(&B->fc1d, par, abortf);
        tc_fence_after_sync();
        if (wlive) {
          const int last = la_s[row];
          const float* tl = tl0 + (last >= 0 ? last : 0) * (H + 4);
#pragma unroll UB
          for (int b = 0; b < NBLK; ++b) {
            uint32_t a[16];
            tmem_ld16(tm + FC1 + (uint32_t)(b * TS_BLK + grp * 16), a);
            float y[16];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float4 va = *reinterpret_cast<const float4*>(ta + b * TS_BLK + 4 * k);
              float4 vl = *reinterpret_cast<const float4*>(tl + b * TS_BLK + 4 * k);
              if (last < 0) vl = make_float4(0.f, 0.f, 0.f, 0.f);
              y[4 * k] = va.x + vl.x; y[4 * k + 1] = va.y + vl.y; y[4 * k + 2] = va.z + vl.z; y[4 * k + 3] = va.w + vl.w;
            }
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 16; ++k) y[k] = fmaxf(__uint_as_float(a[k]) + y[k], 0.f);
            ts_split16<NS>(y, [&](int i, const uint32_t (&w)[8]) {
              const int k8 = b * (TS_BLK / 8) + grp * 2;  // first 8-column group
              if (XS) {
                uint8_t* to = smem + L.off_xy + (uint32_t)(i * (H / 8) + k8) * 2048u + (uint32_t)row * 16u;
                *reinterpret_cast<uint4*>(to) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(to + 2048) = make_uint4(w[4], w[5], w[6], w[7]);
              } else {
                tmem_st8(tm + TSM_Y + (uint32_t)(i * (H / 2) + k8 * 4), w);
              }
            });
          }
          if (XS) fence_proxy_async_smem();
          else tmem_st_wait();
        }
        tc_fence_before_sync();
        ts_arrive(&B->yrdy, lane);

        // ---- E2 ----
        // one block of 32 hidden columns per pass; the block at work is h[0], the others move up behind it
#pragma unroll UB
        for (int b = 0; b < NBLK; ++b) {
          const int buf = H == 64 ? b : (b + 1) & 1;
          mbar_wait(&B->gd[buf], H == 64 ? par : (uint32_t)(b >> 1), abortf);
          tc_fence_after_sync();
          if (b == NBLK - 1) {  // no product reads the old hidden state any more
            if (wlive) {
#pragma unroll
              for (int k = 0; k < NBLK - 1; ++k) store_h(k, h[k + 1]);
              tmem_st_wait();
            }
            tc_fence_before_sync();
            ts_arrive(&B->hr0, lane);
          }
          if (wlive) {
            // columns of the buffer: HN R Z IN | IN R Z HN
            const uint32_t base = tm + (buf ? 128u : 0u) + (uint32_t)grp * 16u;
            const uint32_t c_in = buf ? 0u : 96u, c_hn = buf ? 96u : 0u;
#pragma unroll
            for (int c8 = 0; c8 < 2; ++c8) {
              uint32_t v[4][8];
              tmem_ld8(base + 32u + c8 * 8, v[0]);
              tmem_ld8(base + 64u + c8 * 8, v[1]);
              tmem_ld8(base + c_in + c8 * 8, v[2]);
              tmem_ld8(base + c_hn + c8 * 8, v[3]);
              tmem_ld_wait();
              if (H == 128 && c8 == 1 && b < NBLK - 2) {
                tc_fence_before_sync();
                ts_arrive(&B->accf[buf], lane);
              }
              const float* bb = bias_s + b * TS_BLK + grp * 16 + c8 * 8;
#pragma unroll
              for (int j = 0; j < 8; j += 4) {
                ulonglong2 bv[4];  // biases of four columns
#pragma unroll
                for (int k = 0; k < 4; ++k) bv[k] = *reinterpret_cast<const ulonglong2*>(bb + (FAST && k < 2 ? k + 4 : k) * H + j);
#pragma unroll
                for (int c = 0; c < 4; c += 2) {
                  float a[4][2];
                  ts_f2 b2[4];
#pragma unroll
                  for (int k = 0; k < 4; ++k) {
                    a[k][0] = __uint_as_float(v[k][j + c]);
                    a[k][1] = __uint_as_float(v[k][j + c + 1]);
                    b2[k] = c == 0 ? bv[k].x : bv[k].y;
                  }
                  if constexpr (FAST) ts_gates2_fast(a, b2, h[0][c8 * 8 + j + c], h[0][c8 * 8 + j + c + 1]);
                  else gates2<false>(a, b2, h[0][c8 * 8 + j + c], h[0][c8 * 8 + j + c + 1]);
                }
              }
            }
          } else if (H == 128 && b < NBLK - 2) {
            ts_arrive(&B->accf[buf], lane);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float x = h[0][j];
#pragma unroll
            for (int k = 0; k + 1 < NBLK; ++k) h[k][j] = h[k + 1][j];
            h[NBLK - 1][j] = x;
          }
        }
        if (wlive) {
          store_h(NBLK - 1, h[NBLK - 1]);
          tmem_st_wait();
        }
        tc_fence_before_sync();
        ts_arrive(&B->hr1, lane);

        // ---- E3 ----
        mbar_wait(&B->srdy[b4], (g >> 2) & 1u, abortf);  // the step's records and draws
        const bool close = live && close_s[b4 * ept + el];
        mbar_wait(&B->fc2d, par, abortf);
        tc_fence_after_sync();
        uint32_t qv[NQ];
        if (grp == 0 && wlive) {
          tmem_ld16(tm + L.tm_q, *reinterpret_cast<uint32_t(*)[16]>(qv));
          if (NQ == 32) tmem_ld16(tm + L.tm_q + 16, *reinterpret_cast<uint32_t(*)[16]>(qv + NQ - 16));
          tmem_ld_wait();
        }
        // a closed episode restarts from a zero hidden state and no last action
        if (wlive && __builtin_expect(__any_sync(0xFFFFFFFFu, close), 0)) {
          if (close) {
#pragma unroll
            for (int b = 0; b < NBLK; ++b)
#pragma unroll
              for (int j = 0; j < 16; ++j) h[b][j] = 0.f;
          }
#pragma unroll
          for (int b = 0; b < NBLK; ++b) store_h(b, h[b]);
          tmem_st_wait();
        }
        tc_fence_before_sync();
        if (s + 1 < T) ts_arrive(&B->hset, lane);
        int act = 0;
        if (grp == 0 && live) {
          const uint32_t mask = mask_s[b4 * TS_ROWS + row];
          const int pick = pick_s[b4 * TS_ROWS + row];
          // greedy rule: m = max over available, thr = m - 1e-4f, lowest available a with Q >= thr (a NaN never
          // compares greater or equal and fmaxf ignores it)
          float qf[NQ];
          float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int a = 0; a < NQ; ++a) {
            qf[a] = __uint_as_float(qv[a]) + b2_s[a];
            m4[a & 3] = fmaxf(m4[a & 3], ((mask >> a) & 1u) ? qf[a] : -INFINITY);
          }
          const float thr = __fsub_rn(fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])), 1e-4f);
          uint32_t ge = 0;
#pragma unroll
          for (int a = 0; a < NQ; ++a) ge |= (qf[a] >= thr ? 1u : 0u) << a;
          ge &= mask;
          const int greedy = ge ? __ffs(ge) - 1 : __ffs(mask) - 1;
          act = mask == 0 ? 0 : (pick >= 0 ? pick : greedy);
          la_s[row] = close ? -1 : act;
          c_steps += 1;
          c_explore += pick >= 0 ? 1u : 0u;
          if (mask == 0) { c_noavail += 1; st_bits |= MARL_STATUS_NO_AVAIL; }
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");  // last actions are in place
        if (grp == 0 && live) {
          const unsigned long long rec = recp_s[b4 * ept + el];
          if (rec) reinterpret_cast<int32_t*>(rec + p.rl.off_action)[ai] = act;
          const int tk = p.trace_first + s;
          if (tk < p.trace_cap && p.trace_actions) p.trace_actions[((size_t)tk * p.E + e) * n + ai] = act;
          if (p.actions_out && s == T - 1) p.actions_out[(size_t)(e0 + el) * n + ai] = act;
        }
      }
      // ---- end of the tile: state back to global memory ----
      if (live) {
#pragma unroll
        for (int b = 0; b < NBLK; ++b) {
          float4* dst = reinterpret_cast<float4*>(p.h + grow * H + b * TS_BLK + grp * 16);
#pragma unroll
          for (int k = 0; k < 4; ++k) dst[k] = make_float4(h[b][4 * k], h[b][4 * k + 1], h[b][4 * k + 2], h[b][4 * k + 3]);
        }
        if (grp == 0) p.last_action[grow] = la_s[row];
      }
      fresh = false;
    }
    if (c_steps) atomicAdd(p.counters + CNT_AGENT_STEPS, (unsigned long long)c_steps);
    if (c_explore) atomicAdd(p.counters + CNT_EXPLORED, (unsigned long long)c_explore);
    if (c_noavail) atomicAdd(p.counters + CNT_NO_AVAIL, (unsigned long long)c_noavail);
    if (st_bits) atomicOr(p.status, st_bits);
  }
  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0 && B->abort) {
    atomicOr(p.status, MARL_STATUS_TIMEOUT);
    atomicCAS(p.status + 1, 0u, ((((B->abort & 0xFFFFFu) - (smem_u32(B) & 0xFFFFFu)) >> 3) & 0xFFu) | (((B->abort >> 20) & 0xFFu) << 8));
  }
  if (warp == 16) tmem_dealloc(tmem, 512);
}

// Returns the number of kernels launched or a negative cudaError.  fast_gates: the hardware tanh (bf16, hidden 128).
int launch_actor_tcs(const ActorParams& p_in, int sms, bool fast_gates, cudaStream_t stream) {
  ActorParams p = p_in;
  int nt_max = p.n, ntypes = 1;
  if (p.n_types > 1) {
    ntypes = p.n_types;
    nt_max = 1;
    for (int k = 0; k < ntypes; ++k) {
      int c = 0;
      for (int i = 0; i < p.n; ++i) c += (int)((p.agent_type_bits >> (2 * i)) & 3ull) == k ? 1 : 0;
      if (c > nt_max) nt_max = c;
    }
  }
  const int ns = ts_pieces(p.prec);
  TsLayout L = ts_layout(p.n, p.D, p.A, p.H, ns, nt_max, p.M, sms, ntypes);
  if (p.H == 128 && !fast_gates) {
    // the accurate gates keep the epilogue so busy that input warps running beside it all step long cost more than the
    // wait for the shared columns (1216 against 1246 us for 4096 x 5 agents x 64 steps; fast gates, 16384 x 8 agents: 3940 against 3410;
    // each one launch repeated on the same inputs)
    L.sep = 0;
    L.tm_x = TSM_HOP + (uint32_t)(ns * p.H / 2);
  }
  p.ept = L.ept;
  p.num_tiles = (p.M + L.ept - 1) / L.ept;
  // One network or one per type, accurate gates: [types][pieces][actions][hidden]; the hardware's gates are the last.  In fp32 at
  // hidden 64 launches of several steps go to the kernel for several types with one network too: there that one is the faster
  // (4096 environments x 8 agents x 64 steps 1028 us against 1039, 1482 x 5 x 28 steps 230.7 against 234.1), in one-step launches it
  // is not (9001 x 5 agents 53.4 against 52.0).
  const bool typed = ntypes > 1 || (ns == 3 && p.H == 64 && L.NQ == 16 && p.T > 1);
  const int v = fast_gates ? 16 : (typed ? 8 : 0) + (ns == 3 ? 0 : 4) + (L.NQ == 16 ? 0 : 2) + (p.H == 64 ? 0 : 1);
  decltype(&actor_tcs_kernel<3, 16, 64, false>) kernels[17] = {
      actor_tcs_kernel<3, 16, 64, false>, actor_tcs_kernel<3, 16, 128, false>, actor_tcs_kernel<3, 32, 64, false>, actor_tcs_kernel<3, 32, 128, false>,
      actor_tcs_kernel<1, 16, 64, false>, actor_tcs_kernel<1, 16, 128, false>, actor_tcs_kernel<1, 32, 64, false>, actor_tcs_kernel<1, 32, 128, false>,
      actor_tcs_kernel<3, 16, 64, true>, actor_tcs_kernel<3, 16, 128, true>, actor_tcs_kernel<3, 32, 64, true>, actor_tcs_kernel<3, 32, 128, true>,
      actor_tcs_kernel<1, 16, 64, true>, actor_tcs_kernel<1, 16, 128, true>, actor_tcs_kernel<1, 32, 64, true>, actor_tcs_kernel<1, 32, 128, true>,
      actor_tcs_kernel<1, 16, 128, false, true>};
  static uint32_t configured[17][SMEM_OPTIN_DEVICES];
  {
    const cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernels[v]), L.total, configured[v]);
    if (e != cudaSuccess) return -(int)e;
  }
  int grid = p.num_tiles * ntypes < sms ? p.num_tiles * ntypes : sms;
  if (grid < 1) grid = 1;
  const cudaError_t err = launch_overlapped(kernels[v], grid, TS_THREADS, L.total, stream, p.early != 0, p, L);
  return err == cudaSuccess ? 1 : -(int)err;
}

}  // namespace marl
