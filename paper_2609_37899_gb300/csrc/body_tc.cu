// body_tc.cu -- the paper's expert body on the tensor cores (tcgen05 / TMEM).
//
// A stream is one (expert, probe) pair, both signs, over a chunk of up to 16
// sequences for all T timesteps, in the mean/difference form of the LSTM
// kernels applied to every linear layer.  With v+- = vbar +- dv (dv the half
// difference), its scaled form dhat = dv / eps, and the perturbed weights
// W +- eps Z:
//   (W +- eps Z)(vbar +- dv) = C +- eps D,  C = W vbar + eps^2 Z dhat,
//   D = W dhat + Z vbar,
// so one MMA of W and one of Z against the operand rows [vbar | dhat] give
// both signs.  dhat is O(1), so its fp16 rounding stays relative (2^-11) at
// any eps, where dv itself would fall into fp16's subnormal range.
// Everything between the linear layers (LayerNorm with perturbed gains, the
// LSTM cell, GELU, the residual stream, the decode's log-sum-exp) runs per
// sign in fp32 on the epilogue warps (the residual stream as fp32 mean and
// half difference), which write the next operand back as [vbar | dhat] in
// fp16.  The tied head E is not perturbed: its logits are E ybar +- eps E dhat_y.
//
// Per timestep and block, for one stream:
//   LN_a -> [u | h] operand -> gates MMA (W_ih|W_hh, gate-major tile) -> cells
//   (state in registers; h and x updated) -> LN_b -> MLP1 MMA -> GELU -> the
//   MLP hidden operand -> MLP2 MMA (the hidden rows as the A operand,
//   [W_2 ; Z_2] as B) -> residual;
// then the final LN, the decode MMA (E, two 128-row tiles) and the NLL.  The
// stream's NLL sums per sign go to partial[(pair, sign)][chunk], which
// body_reduce_kernel (body.cu) turns into L+- and the coefficients.
//
// What bounds it: that chain of about 20 short phases, each of them latency
// (an MMA batch of 4 to 12 instructions, tensor-memory reads, shuffles), so
// what counts is how many chains an SM runs and how many warps share a phase.
// A CTA runs two streams of one expert, which share the expert's tiles: W_hi,
// W_lo and E in shared memory and W_lo of the gates in tensor memory.  Each
// stream has 16 warps (64 registers a thread), its own probe tiles (Z of the
// gates in tensor memory as A operands, Z of the MLP in shared memory),
// operands and 160 accumulator columns, and meets the other stream nowhere.
// Together they take 512 columns of tensor memory and 224 KB of shared memory.
// Where that saves no round of CTAs a CTA runs one (body_streams_per_cta).
// After the barrier that completes an operand, warp 0 of the stream issues the
// phase's MMAs; another merges the decode's partials into the NLL while the next
// gates MMAs run.
// Measured on GB300: the step of 256 bodies, 64 probes, 16 x 512 bytes, 570.7 ms
// with one stream per SM (16 epilogue warps, a CTA barrier per phase), 476 with
// two of 8 epilogue warps and an MMA warp each, 357 with two of 16 warps that
// issue their own MMAs, 331 ms now (offsets and pairs precomputed, LN on half
// of the warps).  Alone on its SM a stream takes about 15,000 cycles per
// timestep: MMA batches 5,000, GELU 2,300 (its erff), LN 2,500, cells and decode
// 2,600 and the rest barriers and tensor-memory reads; two together 24,000,
// 64 % of the issue slots busy.
//
// Precision.  With plain fp16 operands the losses were off by up to ~2e-4
// nats/byte and the coefficients by ~1-2% on small batches: the rounding of
// W and vbar shifts the model both signs see, and the LayerNorms pass the
// shift on.  So, except in the MLP's second layer:
//  - every operand value is split, v = hi + lo (both fp16), as four row
//    groups [vbar_hi | dhat_hi | vbar_lo | dhat_lo], so one W and one Z MMA
//    (N = 64) give both parts of both halves;
//  - W = W_hi + W_lo, W_lo as the A operand of one more MMA (N = 32, the hi rows);
//  - the tied head likewise, E = E_hi + E_lo.
#include <cuda_fp16.h>

#define SOMA_CHECK_FILE 3
#include "checked.cuh"
#include "body_device.cuh"
#include "soma_device.cuh"
#include "soma_launch.h"
#include "tc_primitives.cuh"

namespace soma {

using namespace tc;

namespace {

constexpr int kD = kBodyWidth;  // 32
constexpr int kG = 4 * kD;      // 128
constexpr int kBp = kBodyRows;  // sequences per CTA (16)
constexpr int kN = 2 * kBp;     // operand rows [vbar | dhat] (hi parts; MLP2 operand)
constexpr int kNQ = 4 * kBp;    // operand rows [vbar_hi | dhat_hi | vbar_lo | dhat_lo]
constexpr int kWarps = 16;     // of one stream
constexpr int kIssueWarp = 0;  // issues the MMAs
constexpr int kMergeWarp = 1;  // merges the NLL
constexpr int kLnWarp0 = 4, kLnWarps = 8;  // two warps per scheduler run the LayerNorms
constexpr int kMaxStreams = 2;
constexpr uint32_t kLbo = 128;
constexpr float kLnEps = 1e-5f;

// Shared-memory layout (bytes, from a 1024-aligned base), NS streams.
constexpr uint32_t kGateTile = 128u * 64 * 2;   // [W_ih | W_hh] gate-major, K = 64
constexpr uint32_t kMlp1Tile = 128u * 32 * 2;   // W_1, K = 32
constexpr uint32_t kMlp2Tile = 32u * 128 * 2;   // W_2 or Z_2 as a B operand: 32 rows, K = 128
constexpr uint32_t kHeadTile = 128u * 32 * 2;   // one 128-row tile of E
constexpr uint32_t kOpTile = kNQ * 32 * 2;      // an operand of 32 columns
template <int NS>
struct Smem {
  // per block: W of the gates, W_1, its lo part, then the MLP2 B operands
  // [Z_2 of stream 0 | W_2 | Z_2 of stream 1]: [Z_2 | W_2] and [W_2 | Z_2] are
  // each one 64-row operand
  static constexpr uint32_t blk = kGateTile + 2 * kMlp1Tile + (1 + NS) * kMlp2Tile;
  static constexpr uint32_t w1 = kGateTile, w1lo = w1 + kMlp1Tile, m2 = w1lo + kMlp1Tile;
  static constexpr uint32_t e = kBodyMaxBlocks * blk;  // E_hi, E_lo: [2][2 tiles][128][32]
  static constexpr uint32_t st0 = e + 4 * kHeadTile;
  // per stream.  The MLP2 A operand has 128 rows to the MMA, of which 32 exist;
  // the others' lanes are never read, and the 24 KB after it stand in for them.
  // The LN outputs (4 KB) share its place: each is consumed before the other
  // is written.
  static constexpr uint32_t hid = 0, v = 0;
  static constexpr uint32_t h = hid + 32u * 128 * 2;              // [blocks] h parts
  static constexpr uint32_t z1 = h + kBodyMaxBlocks * kOpTile;    // [blocks] Z_1
  static constexpr uint32_t x = z1 + kBodyMaxBlocks * kMlp1Tile;  // fp32 (mean, half difference) [Bp][d]
  static constexpr uint32_t gain = x + 2u * kBp * kD * 4;         // (+, -) [(2D+1) d]
  static constexpr uint32_t red = gain + 2u * (2 * kBodyMaxBlocks + 1) * kD * 4;  // [2][4][2][Bp] float2
  static constexpr uint32_t ylog = red + 2u * 4 * 2 * kBp * 8;    // [2][Bp]
  static constexpr uint32_t acc = ylog + 2u * kBp * 4;            // [2][Bp] double
  static constexpr uint32_t stream = acc + 2u * kBp * 8;
  static constexpr uint32_t ctl = st0 + NS * stream;
  static constexpr uint32_t bytes = ctl + 256 + 1024;  // + alignment slack
};
static_assert(Smem<2>::bytes <= 227 * 1024, "shared memory");
static_assert(Smem<2>::z1 + kBodyMaxBlocks * kMlp1Tile >= 128u * 128 * 2, "MLP2 A operand");
static_assert(Smem<2>::st0 % 128 == 0 && Smem<2>::stream % 128 == 0 && Smem<2>::acc % 8 == 0,
              "alignment");

// TMEM columns: W_lo of the gates (A operands, 32 columns = K / 2 per block);
// then per stream Z of the gates (32 per block) and the accumulators of the
// current layer (W and Z, 64 each; MLP2: 64), which the decode reuses
// (E_hi x [ybar | dy] of the two halves, 64 each), and E_lo ybar_hi (16 per half).
constexpr uint32_t kTStream0 = 32 * kBodyMaxBlocks, kTZg = 0, kTAcc = 32 * kBodyMaxBlocks,
                   kTZ = 64, kTHeadLo = 128, kTStream = kTAcc + 160, kTmemCols = 512;
static_assert(kTStream0 + kMaxStreams * kTStream <= kTmemCols, "tensor memory");

struct BodyCtl {
  uint64_t mma_bar[kMaxStreams];   // the MMAs of a phase are done
  uint32_t tmem_slot;
  volatile int abort;
};
static_assert(sizeof(BodyCtl) <= 256, "control block");

__device__ __forceinline__ float gelu_b(float a) {
  return 0.5f * a * (1.f + erff(a * 0.70710678118654752f));
}

struct BodyTcArgs {
  const float* params;   // [N][P]
  const float* head;     // [V][d]
  const uint8_t* bytes;  // [N][B][T+1]
  double* partial;       // [N * n * n_sign][chunks]
  int* status;
  int n_experts, n_pert, n_sign, blocks, B, T, chunks;
  int64_t P, goff;
  float eps;
  int sparse;
  uint64_t seed, step;
};

// The weights p0 .. p0 + 7 (p0 % 8 == 0) as fp16, or the rounding residuals
// w - fp16(w) of them.
__device__ __forceinline__ uint4 w_chunk(const float* th, int64_t p0, const BodyTcArgs& a,
                                         bool lo_part) {
  const bool in = SOMA_CHECK(p0 >= 0 && p0 + 8 <= a.P, a.status);  // inside the expert
  __align__(16) __half w[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float x = in ? th[p0 + j] : 0.f;
    const __half hi = __float2half_rn(x);
    w[j] = lo_part ? __float2half_rn(x - __half2float(hi)) : hi;
  }
  return *reinterpret_cast<const uint4*>(w);
}

// Bytes between the row groups [vbar_hi | dhat_hi | vbar_lo | dhat_lo] of a
// 32-column operand.
constexpr uint32_t kRowGroup = (kBp / 8) * (kD * 16);

// Operand rows of one sequence at one column (dst: the first row group's
// element): hi(mean), hi(dif), mean - hi(mean), dif - hi(dif).
__device__ __forceinline__ void store_split(uint8_t* dst, float mean, float dif) {
  const __half mh = __float2half_rn(mean), dh = __float2half_rn(dif);
  *reinterpret_cast<__half*>(dst) = mh;
  *reinterpret_cast<__half*>(dst + kRowGroup) = dh;
  *reinterpret_cast<__half*>(dst + 2 * kRowGroup) = __float2half_rn(mean - __half2float(mh));
  *reinterpret_cast<__half*>(dst + 3 * kRowGroup) = __float2half_rn(dif - __half2float(dh));
}

// fp16 pair word (lo parts of w0, w1): the residual w - fp16(w) of each.
__device__ __forceinline__ uint32_t lo_pair(float w0, float w1) {
  const __half a = __float2half_rn(w0 - __half2float(__float2half_rn(w0)));
  const __half b = __float2half_rn(w1 - __half2float(__float2half_rn(w1)));
  return (uint32_t)__half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
}

// The operand rows (K = 32) of one sequence: mean and scaled half difference
// (times inv_eps = 1 / eps, 0 when eps = 0) of the two signs' LN outputs.  The
// 32 / NF lanes of a sequence hold NF features of both signs each, 32 / NF
// apart, so a sum over the features is NF - 1 additions and log2(32 / NF)
// shuffles, in the order of a 32-lane butterfly (features 16 apart first).
// With NF = 2 half of a stream's warps run a LayerNorm; measured on the
// 256-body step: all sixteen, a lane per (sign, feature pair), 337 ms; eight
// 333 ms; four (NF = 4, the fewest shuffles) 344 ms.
// x: this lane's (mean, half difference) pairs, gain: its first (+, -) pair,
// dst: its first operand element.
constexpr int NF = 16 / kLnWarps, kLnLanes = kD / NF;  // features of a lane, lanes of a sequence
static_assert(NF == 2, "the sums below add two features");
__device__ __forceinline__ void ln_rows(const float2 (&x)[NF], const float2* gain, uint8_t* dst,
                                        float inv_eps) {
  constexpr int L = kLnLanes;
  float c[2][NF], rs[2];
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    c[0][k] = x[k].x + x[k].y;
    c[1][k] = x[k].x - x[k].y;
  }
  float s[2];
#pragma unroll
  for (int g = 0; g < 2; ++g)
    s[g] = c[g][0] + c[g][1];
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
    for (int g = 0; g < 2; ++g) s[g] += __shfl_xor_sync(0xffffffffu, s[g], o);
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const float mean = s[g] * (1.f / kD);
    float q[NF];
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      c[g][k] -= mean;
      q[k] = __fmul_rn(c[g][k], c[g][k]);
    }
    s[g] = __fadd_rn(q[0], q[1]);
  }
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
    for (int g = 0; g < 2; ++g) s[g] += __shfl_xor_sync(0xffffffffu, s[g], o);
#pragma unroll
  for (int g = 0; g < 2; ++g) rs[g] = rsqrtf(fmaf(s[g], 1.f / kD, kLnEps));
#pragma unroll
  for (int k = 0; k < NF; ++k) {
    const float2 g = gain[L * k];
    const float np = __fmul_rn(c[0][k], rs[0]);
    const float um = __fmul_rn(__fmul_rn(c[1][k], rs[1]), g.y);
    // the + sign's product enters exactly, the - sign's rounded
    store_split(dst + 16 * L * k, 0.5f * fmaf(np, g.x, um), 0.5f * fmaf(np, g.x, -um) * inv_eps);
  }
}

// 16x128b view of NG 4-column groups from column taddr: thread l gets column 4
// h + l % 4 of rows l / 4 + 8 k (k = 0..3) of the 32-lane quarter.
template <int NG>
__device__ __forceinline__ void ld_view(uint32_t taddr, uint32_t (&r)[NG][4]) {
  const uint32_t t2 = taddr + (16u << 16);
  if constexpr (NG == 2) {
    tmem_ld_16x128b_x2(taddr, r[0][0], r[0][1], r[1][0], r[1][1]);
    tmem_ld_16x128b_x2(t2, r[0][2], r[0][3], r[1][2], r[1][3]);
  } else {
    tmem_ld_16x128b(taddr, r[0][0], r[0][1]);
    tmem_ld_16x128b(t2, r[0][2], r[0][3]);
  }
}

// C and the half difference D of one layer for this thread's view (rows k):
//   C = W (vbar_hi + vbar_lo) + eps^2 Z (dhat_hi + dhat_lo),
//   D = eps [W (dhat_hi + dhat_lo) + Z (vbar_hi + vbar_lo)],
// from the W accumulator (columns c + {0, 1, 2, 3} Bp; W_lo already added
// to the hi columns) and the Z accumulator.
__device__ __forceinline__ void layer_cd(uint32_t tq, float eps, float (&C)[4], float (&D)[4]) {
  const float eps2 = eps * eps;
  uint32_t w[4][1][4], z[4][1][4];  // [row group]
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    ld_view<1>(tq + g * kBp, w[g]);
    ld_view<1>(tq + kTZ + g * kBp, z[g]);
  }
  tmem_wait_ld();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float wv = __uint_as_float(w[0][0][k]) + __uint_as_float(w[2][0][k]);
    const float wd = __uint_as_float(w[1][0][k]) + __uint_as_float(w[3][0][k]);
    const float zv = __uint_as_float(z[0][0][k]) + __uint_as_float(z[2][0][k]);
    const float zd = __uint_as_float(z[1][0][k]) + __uint_as_float(z[3][0][k]);
    C[k] = fmaf(eps2, zd, wv);
    D[k] = eps * (wd + zv);
  }
}

// fp16 pair words of the 32 coordinates of run q under the body's probe law:
// +-1, or 0 where inactive.
__device__ __forceinline__ void z_row_words(const ProbeKey& pk, int q, const BodyTcArgs& a,
                                            bool do_z, uint32_t (&o)[16]) {
  uint32_t neg = 0, act = 0;
  if (do_z) body_probe_words(pk, q, a.sparse, a.goff, neg, act);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint32_t m = (((act >> (2 * j)) & 1u) ? 0x3C00u : 0u) |
                       (((act >> (2 * j + 1)) & 1u) ? 0x3C000000u : 0u);
    const uint32_t sg = ((neg >> (2 * j)) & 1u) << 15 | ((neg >> (2 * j + 1)) & 1u) << 31;
    o[j] = m | (sg & ((m & 0x04000400u) << 5));  // the sign bit of active coordinates
  }
}

// A wait that runs out records the status and sets the CTA's abort flag;
// every later wait then returns at once.  No warp leaves the loop early, so the
// hardware barriers between the epilogue warps stay matched.
__device__ __forceinline__ bool body_wait(uint64_t* bar, uint32_t parity, volatile int* abort,
                                          int* status) {
  for (uint32_t n = 0; n < (1u << 22); ++n) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((n & 7u) == 7u && *abort) return false;
  }
  *abort = 1;
  atomicCAS(status, 0, kStatusTimeout);
  return false;
}

// NS streams per CTA, of kWarps warps each.  Streams of an expert are numbered
// probe * chunks + chunk; CTA j of an expert runs streams j NS .. j NS + NS - 1.
template <int NS>
__global__ void __launch_bounds__(NS * kWarps * 32, 1) body_tc_kernel(const BodyTcArgs a) {
  using S = Smem<NS>;
  constexpr int kThr = NS * kWarps * 32, kStThr = kWarps * 32;
  extern __shared__ uint8_t dyn_smem[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(dyn_smem) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int streams = a.n_pert * a.chunks;  // of one expert
  const int per_e = (streams + NS - 1) / NS;
  const int64_t cta = blockIdx.x + (int64_t)gridDim.x * blockIdx.y;
  if (cta >= (int64_t)a.n_experts * per_e) return;
  const int e = (int)(cta / per_e), s0 = (int)(cta % per_e) * NS;
  const int st = warp / kWarps, ew = warp % kWarps;  // the warp's stream, its number in it
  const int stid = tid % kStThr;
  const int i = min(s0 + st, streams - 1) / a.chunks, chunk = min(s0 + st, streams - 1) % a.chunks;
  const int64_t pair = (int64_t)e * a.n_pert + i;
  const int b0c = chunk * kBp;
  const int rows = min(kBp, a.B - b0c);
  // the stream's sequences, its expert's parameters and its NLL partials lie inside
  // the caller's buffers
  const bool live = s0 + st < streams &&
                    SOMA_CHECK(chunk < a.chunks && b0c < a.B &&
                                   pair < (int64_t)a.n_experts * a.n_pert,
                               a.status);
  const int D = a.blocks;
  const float eps = a.eps;
  const bool do_z = eps != 0.f;
  const float eps2 = eps * eps;
  const float inv_eps = do_z ? 1.f / eps : 0.f;  // the operand's difference rows are dv / eps
  const float* th = a.params + (int64_t)e * a.P;
  const ProbeKey pk = make_probe_key(a.seed, a.step, (uint32_t)e, (uint32_t)i);
  BodyCtl* ctl = reinterpret_cast<BodyCtl*>(smem + S::ctl);
  volatile int* abort = &ctl->abort;
  uint8_t* sm = smem + S::st0 + st * S::stream;  // this stream's part
  float2* x = reinterpret_cast<float2*>(sm + S::x);         // (mean, half difference) [Bp][d]
  float2* gains = reinterpret_cast<float2*>(sm + S::gain);  // (+, -) [(2D+1) d]
  float2* red = reinterpret_cast<float2*>(sm + S::red);
  float* ylog = reinterpret_cast<float*>(sm + S::ylog);
  double* acc = reinterpret_cast<double*>(sm + S::acc);

  if (tid == 0) {
    for (int k = 0; k < NS; ++k) {
      mbar_init(&ctl->mma_bar[k], 1);
    }
    ctl->abort = 0;
    mbar_fence_init();
  }
  if (warp == 0) tmem_alloc(&ctl->tmem_slot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_slot;
  const uint32_t tst = tmem + kTStream0 + (uint32_t)st * kTStream;
  const int q4 = warp & 3;
  const int r = 32 * q4 + lane;  // TMEM lane of this thread in the set-up

  // ---- A operands in tensor memory (thread = row): Z of the gates by each
  // stream's first eight warps (block = ew / 4), W_lo of the gates by stream 0's
  // last eight
  {
    const int64_t R = (int64_t)tile_gate(r) * kD + tile_unit(r);
    const uint32_t quarter = (uint32_t)(32 * q4) << 16;
    uint32_t pr[16];
    const int zb = ew >> 2;
    if (zb < D) {
      const int q = (int)((zb * 16 * kD * kD + R * kD) >> 5);  // the row's run of W_ih
      z_row_words(pk, q, a, do_z, pr);
      tmem_st16(tst + quarter + kTZg + 32 * zb, pr);
      z_row_words(pk, q + 4 * kD * kD / 32, a, do_z, pr);
      tmem_st16(tst + quarter + kTZg + 32 * zb + 16, pr);
    }
    const int wb = (ew >> 2) - kBodyMaxBlocks;
    if (st == 0 && wb >= 0 && wb < D) {
      const float* wih = th + (int64_t)wb * 16 * kD * kD + R * kD;
      const float* whh = wih + 4 * kD * kD;
#pragma unroll
      for (int c = 0; c < 16; ++c) pr[c] = lo_pair(wih[2 * c], wih[2 * c + 1]);
      tmem_st16(tmem + quarter + 32 * wb, pr);
#pragma unroll
      for (int c = 0; c < 16; ++c) pr[c] = lo_pair(whh[2 * c], whh[2 * c + 1]);
      tmem_st16(tmem + quarter + 32 * wb + 16, pr);
    }
    tmem_wait_st();
  }

  // ---- resident fp16 tiles: W by the whole CTA, Z by each stream's warps ----
  for (int b = 0; b < D; ++b) {
    uint8_t* blk = smem + b * S::blk;
    const int64_t base = (int64_t)b * 16 * kD * kD;
    // gate tile: row r = gate (r / 8) % 4 of unit 8 (r / 32) + r % 8; K = [u | h]
    for (int c = tid; c < 128 * 8; c += kThr) {
      const int rr = c >> 3, k0 = 8 * (c & 7);
      const int64_t R = (int64_t)tile_gate(rr) * kD + tile_unit(rr);
      const int64_t p0 = k0 < kD ? base + R * kD + k0 : base + 4 * kD * kD + R * kD + (k0 - kD);
      *reinterpret_cast<uint4*>(blk + kmajor_offset(rr, k0, 64)) = w_chunk(th, p0, a, false);
    }
    // W_1 [4d][d] and its lo part
    for (int c = tid; c < 128 * 4; c += kThr) {
      const int rr = c >> 2, k0 = 8 * (c & 3);
      const int64_t p0 = base + 8 * kD * kD + (int64_t)rr * kD + k0;
      const uint32_t off = kmajor_offset(rr, k0, 32);
      *reinterpret_cast<uint4*>(blk + S::w1 + off) = w_chunk(th, p0, a, false);
      *reinterpret_cast<uint4*>(blk + S::w1lo + off) = w_chunk(th, p0, a, true);
    }
    // W_2 [d][4d] as a B operand: row j (output feature), K = 128
    for (int c = tid; c < 32 * 16; c += kThr) {
      const int rr = c >> 4, k0 = 8 * (c & 15);
      const int64_t p0 = base + 12 * kD * kD + (int64_t)rr * kG + k0;
      *reinterpret_cast<uint4*>(blk + S::m2 + kMlp2Tile + kmajor_offset(rr, k0, 128)) =
          w_chunk(th, p0, a, false);
    }
    {
      uint8_t* z2 = blk + S::m2 + 2 * st * kMlp2Tile;
      // one run of 32 coordinates per thread and step: Z_1's rows, then Z_2's quarters
      for (int c = stid; c < 128 + 128; c += kStThr) {
        const bool one = c < 128;
        const int rr = one ? c : (c - 128) >> 2, k0 = one ? 0 : 32 * (c & 3);
        const int64_t p0 = base + (one ? 8 * kD * kD + rr * kD : 12 * kD * kD + rr * kG + k0);
        uint32_t w[16];
        z_row_words(pk, (int)(p0 >> 5), a, do_z, w);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint8_t* dst = one ? sm + S::z1 + b * kMlp1Tile + kmajor_offset(rr, 8 * k, 32)
                             : z2 + kmajor_offset(rr, k0 + 8 * k, 128);
          *reinterpret_cast<uint4*>(dst) =
              make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
        }
      }
    }
  }
  for (int c = tid; c < 256 * 4; c += kThr) {  // E [256][32] = E_hi + E_lo, 128-row tiles
    const int v = c >> 2, k0 = 8 * (c & 3);
    __align__(16) __half w[8], wl[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float x = a.head[v * kD + k0 + j];
      w[j] = __float2half_rn(x);
      wl[j] = __float2half_rn(x - __half2float(w[j]));
    }
    const uint32_t off = (v >> 7) * kHeadTile + kmajor_offset(v & 127, k0, 32);
    *reinterpret_cast<uint4*>(smem + S::e + off) = *reinterpret_cast<const uint4*>(w);
    *reinterpret_cast<uint4*>(smem + S::e + 2 * kHeadTile + off) =
        *reinterpret_cast<const uint4*>(wl);
  }
  // perturbed gains per sign (dense probe signs on every gain)
  for (int k = stid; k < (2 * D + 1) * kD; k += kStThr) {
    const int64_t p = a.goff + k;
    float dz = 0.f;
    if (do_z) {
      uint32_t neg, act;
      body_probe_words(pk, (int)(p >> 5), a.sparse, a.goff, neg, act);
      const int j = (int)(p & 31);
      dz = ((act >> j) & 1u) ? (((neg >> j) & 1u) ? -eps : eps) : 0.f;
    }
    gains[k] = make_float2(th[p] + dz, th[p] - dz);
  }
  // operands: zero (the h parts start at h = 0)
  for (uint32_t c = stid; c < S::z1 / 16; c += kStThr)
    reinterpret_cast<uint4*>(sm)[c] = make_uint4(0u, 0u, 0u, 0u);
  for (int c = stid; c < 2 * kBp; c += kStThr) acc[c] = 0.0;

  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  // (an expert's last CTA may have no second stream)
  if (live) {
    uint64_t* mma_bar = &ctl->mma_bar[st];
    const uint32_t tacc = tst + kTAcc, tw = tacc, tz = tacc + kTZ;
    // descriptor words (low word: start address in 16-byte units, the high word
    // depends on the columns of the operand)
    const uint32_t idesc32 = idesc_f16_f32(128, kN), idesc64 = idesc_f16_f32(128, kNQ),
                   idesc16 = idesc_f16_f32(128, kBp);
    const uint64_t d64 = smem_desc(smem_u32(smem), kLbo, 64 * 16);
    const uint32_t hi64 = (uint32_t)(d64 >> 32);
    const uint32_t hi32 = (uint32_t)(smem_desc(smem_u32(smem), kLbo, 32 * 16) >> 32);
    const uint32_t hi128 = (uint32_t)(smem_desc(smem_u32(smem), kLbo, 128 * 16) >> 32);
    const uint32_t lo0 = (uint32_t)d64;  // smem base; same low word for every SBO
    auto lo = [&](uint32_t off) { return lo0 + (off >> 4); };
    const uint32_t so = S::st0 + (uint32_t)st * S::stream;  // this stream's part

    const int sg = ew >> 2;  // the warp's 4 sequences in the layer epilogues
    const int u8 = lane >> 2, bq = lane & 3;
    const int bseq = 4 * sg + bq;
    // this thread's places: in LN (sequence, features f, f + 8, ..), in the cells
    // (sequence bseq, unit) and in the MLP's hidden operand
    const bool ln_warp = ew >= kLnWarp0 && ew < kLnWarp0 + kLnWarps;
    const int lb = ((32 / kLnLanes) * (ew - kLnWarp0) + lane / kLnLanes) & (kBp - 1),
              f0 = lane % kLnLanes;
    const int U = 8 * q4 + u8;
    float2* ln_x = x + lb * kD + f0;
    const float2* ln_g = gains + f0;
    uint8_t* ln_dst = sm + S::v + kmajor_offset(lb, f0, kD);
    float2* cell_x = x + bseq * kD + U;
    uint8_t* h_dst = sm + S::h + kmajor_offset(bseq, U, kD);
    uint8_t* hid_dst = sm + S::hid + kmajor_offset(bseq, 32 * q4 + u8, 128);
    const uint32_t quarter = (uint32_t)(32 * q4) << 16;
    const uint32_t tq = tacc + quarter + (uint32_t)(4 * sg);
    float cst[kBodyMaxBlocks][2];
#pragma unroll
    for (int b = 0; b < kBodyMaxBlocks; ++b) cst[b][0] = cst[b][1] = 0.f;
    // the byte rows (sequences past the batch read row 0)
    const int T1 = a.T + 1;
    const uint8_t* bx = a.bytes + ((int64_t)e * a.B + b0c) * T1;
    const uint8_t* erow = bx + (int64_t)(lb < rows ? lb : 0) * T1;
    // a timestep ahead: the embedding of the next byte of the LN lane's sequence
    float emb[NF];
#pragma unroll
    for (int k = 0; k < NF; ++k) emb[k] = ln_warp ? a.head[(int)erow[0] * kD + f0 + kLnLanes * k] : 0.f;
    uint32_t nph = 0;  // MMA batches so far: the parity of the next wait
    auto mma_wait = [&]() {
      body_wait(mma_bar, nph & 1u, abort, a.status);
      ++nph;
      tc_fence_after();
    };
    auto st_barrier = [&]() {  // the stream's warps
      asm volatile("bar.sync %0, %1;" ::"r"(1 + st), "n"(kStThr) : "memory");
    };
    auto op_barrier = [&]() {  // the operand is written, the accumulators are read
      fence_async_smem();
      tc_fence_before();
      st_barrier();
    };
    // NLL of timestep t: lane = (sign, sequence)
    auto merge = [&]() {
      const int mb = lane & 15, ms = lane >> 4;
      float M = -INFINITY;
      for (int h = 0; h < 8; ++h) M = fmaxf(M, red[(h * 2 + ms) * kBp + mb].x);
      float Ss = 0.f;
      for (int h = 0; h < 8; ++h) {
        const float2 q = red[(h * 2 + ms) * kBp + mb];
        Ss += q.y * __expf(q.x - M);
      }
      acc[ms * kBp + mb] += (double)(M + logf(Ss) - ylog[ms * kBp + mb]);
    };

    for (int t = 0; t < a.T; ++t) {
#pragma unroll
      for (int b = 0; b < kBodyMaxBlocks; ++b) {
        if (b >= D) break;
        const uint32_t blk = b * S::blk;
        // ---- LN_a -> u part of the gate operand
        if (ln_warp) {
          float2 v[NF];
#pragma unroll
          for (int k = 0; k < NF; ++k) {
            // x = E[byte_t] at the first block (E is not perturbed: no difference)
            if (b == 0) ln_x[kLnLanes * k] = make_float2(emb[k], 0.f);
            v[k] = b == 0 ? make_float2(emb[k], 0.f) : ln_x[kLnLanes * k];
          }
          if (b == 0 && t + 1 < a.T) {
            const float* next = a.head + (int)erow[t + 1] * kD + f0;
#pragma unroll
            for (int k = 0; k < NF; ++k) emb[k] = next[kLnLanes * k];
          }
          ln_rows(v, ln_g + 2 * b * kD, ln_dst, inv_eps);
        }
        op_barrier();
        if (ew == kIssueWarp) {
          // gates: W and Z x [u | h], W_lo x the hi rows (added to the hi columns)
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int k16 = 0; k16 < 4; ++k16) {
              const uint32_t ko = 16u * k16, accf = k16 > 0;
              const uint32_t ob =
                  k16 < 2 ? lo(so + S::v) + ko : lo(so + S::h + b * kOpTile) + ko - 32u;
              mma_f16_ss_lohi(tw, lo(blk) + ko, hi64, ob, hi32, idesc64, accf);
              mma_f16_ts_lohi(tz, tst + kTZg + 32 * b + 8 * k16, ob, hi32, idesc64, accf);
              mma_f16_ts_lohi(tw, tmem + 32 * b + 8 * k16, ob, hi32, idesc32, 1u);
            }
            mma_commit(mma_bar);
          }
          __syncwarp();
        }
        // the partials of t - 1 are complete since the barrier
        if (b == 0 && ew == kMergeWarp && t > 0) merge();
        mma_wait();
        // ---- cells: thread = unit 8 q4 + u8, sequence bseq
        {
          float Cg[4], Dg[4];
          layer_cd(tq, eps, Cg, Dg);
          float ap[4], am[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float C = Cg[k], Dd = Dg[k];
            if (k == 2) {
              ap[k] = tanh_f(C + Dd);
              am[k] = tanh_f(C - Dd);
            } else {
              ap[k] = sigmoid_f(C + Dd);
              am[k] = sigmoid_f(C - Dd);
            }
          }
          const float cp = fmaf(ap[1], cst[b][0], ap[0] * ap[2]);
          const float cm = fmaf(am[1], cst[b][1], am[0] * am[2]);
          cst[b][0] = cp;
          cst[b][1] = cm;
          float hsum, hdif;
          h_sum_diff(ap[3], tanh_f(cp), am[3], tanh_f(cm), hsum, hdif);
          const float hb = 0.5f * hsum, hd = 0.5f * hdif;
          store_split(h_dst + b * kOpTile, hb, hd * inv_eps);
          float2 v = *cell_x;
          v.x += hb;
          v.y += hd;
          *cell_x = v;
        }
        st_barrier();
        // ---- LN_b -> MLP1 operand
        if (ln_warp) {
          float2 v[NF];
#pragma unroll
          for (int k = 0; k < NF; ++k) v[k] = ln_x[kLnLanes * k];
          ln_rows(v, ln_g + (2 * b + 1) * kD, ln_dst, inv_eps);
        }
        op_barrier();
        if (ew == kIssueWarp) {
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int k16 = 0; k16 < 2; ++k16) {
              const uint32_t ko = 16u * k16, accf = k16 > 0, ob = lo(so + S::v) + ko;
              mma_f16_ss_lohi(tw, lo(blk + S::w1) + ko, hi32, ob, hi32, idesc64, accf);
              mma_f16_ss_lohi(tz, lo(so + S::z1 + b * kMlp1Tile) + ko, hi32, ob, hi32, idesc64,
                              accf);
              mma_f16_ss_lohi(tw, lo(blk + S::w1lo) + ko, hi32, ob, hi32, idesc32, 1u);
            }
            mma_commit(mma_bar);
          }
          __syncwarp();
        }
        mma_wait();
        // ---- GELU: thread = features 32 q4 + u8 + {0, 8, 16, 24}, sequence bseq
        {
          float Cg[4], Dg[4];
          layer_cd(tq, eps, Cg, Dg);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float C = Cg[k], Dd = Dg[k];
            const float mp = gelu_b(C + Dd), mm = gelu_b(C - Dd);
            // rows bseq and Bp + bseq, 8 features (one core matrix) per k
            *reinterpret_cast<__half*>(hid_dst + 128 * k) = __float2half_rn(0.5f * (mp + mm));
            *reinterpret_cast<__half*>(hid_dst + 128 * k + (kBp / 8) * (128 * 16)) =
                __float2half_rn(0.5f * (mp - mm) * inv_eps);
          }
        }
        op_barrier();
        if (ew == kIssueWarp) {
          // MLP2: [mbar | mhat] (rows) x [Z_2 ; W_2]^T or [W_2 ; Z_2]^T, one MMA
          // of N = 64 per K step
          tc_fence_after();
          if (elect_one()) {
            const uint32_t oa = lo(so + S::hid), wb = lo(blk + S::m2 + (uint32_t)st * kMlp2Tile);
#pragma unroll
            for (int k16 = 0; k16 < 8; ++k16)
              mma_f16_ss_lohi(tw, oa + 16u * k16, hi128, wb + 16u * k16, hi128, idesc64, k16 > 0);
            mma_commit(mma_bar);
          }
          __syncwarp();
        }
        mma_wait();
        // ---- MLP2: lanes 0-15 are the rows mbar of the sequences, 16-31 mhat;
        // columns: Z_2 and W_2 products (stream 0: Z first) of the 32 features,
        // 8 of them for each warp of quarter 0
        if (q4 == 0) {
          const uint32_t cw = st == 0 ? kD : 0u, cz = kD - cw;
          const uint32_t col = (uint32_t)(8 * sg);
          uint32_t wm[2][4], zm[2][4];  // [4-feature group][mbar, mbar, mhat, mhat rows]
          ld_view<2>(tacc + cw + col, wm);
          ld_view<2>(tacc + cz + col, zm);
          tmem_wait_ld();
#pragma unroll
          for (int f = 0; f < 2; ++f) {
            const int j = (int)col + 4 * f + bq;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int sq = u8 + 8 * h;  // sequence
              const float C = fmaf(eps2, __uint_as_float(zm[f][2 + h]), __uint_as_float(wm[f][h]));
              const float Dd = eps * (__uint_as_float(wm[f][2 + h]) + __uint_as_float(zm[f][h]));
              float2 v = x[sq * kD + j];
              v.x += C;
              v.y += Dd;
              x[sq * kD + j] = v;
            }
          }
        }
        st_barrier();
      }

      // ---- y = LN(x) gf -> decode operand; logits = E y ---------------------
      if (ln_warp) {
        float2 v[NF];
#pragma unroll
          for (int k = 0; k < NF; ++k) v[k] = ln_x[kLnLanes * k];
        ln_rows(v, ln_g + 2 * D * kD, ln_dst, inv_eps);
      }
      op_barrier();
      if (ew == kIssueWarp) {
        // E_hi x all rows, E_lo x ybar_hi
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int k16 = 0; k16 < 2; ++k16) {
              const uint32_t ko = 16u * k16, accf = k16 > 0, ob = lo(so + S::v) + ko;
              const uint32_t ea = lo(S::e + h * kHeadTile) + ko;
              mma_f16_ss_lohi(tacc + h * 64, ea, hi32, ob, hi32, idesc64, accf);
              mma_f16_ss_lohi(tacc + kTHeadLo + h * 16, ea + ((2 * kHeadTile) >> 4), hi32, ob, hi32,
                              idesc16, accf);
            }
          }
          mma_commit(mma_bar);
        }
        __syncwarp();
      }
      // warp: vocabulary half sg % 2, quarter q4, sequences 8 (sg / 2) .. + 7;
      // thread l holds rows l / 4 + 8 k (k = 0..3) of the quarter
      const int half = sg & 1, b0 = 8 * (sg >> 1);
      const int vq = 128 * half + 32 * q4;
      const uint32_t th0 = tacc + quarter + half * 64 + b0,
                     tl0 = tacc + quarter + kTHeadLo + half * 16 + b0;
      int tgt[2];  // byte t + 1 of the thread's two sequences (rows past the batch: row 0)
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const int b = b0 + 4 * f + bq;
        tgt[f] = (int)bx[(b < rows ? b : 0) * T1 + t + 1];
      }
      mma_wait();
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        // E_hi times the four row groups, and E_lo ybar_hi
        uint32_t yq[4][1][4], ye[1][4];
#pragma unroll
        for (int g = 0; g < 4; ++g) ld_view<1>(th0 + g * kBp + 4 * f, yq[g]);
        ld_view<1>(tl0 + 4 * f, ye);
        tmem_wait_ld();
        float lp[4], lm[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float C = __uint_as_float(yq[0][0][k]) +
                          (__uint_as_float(yq[2][0][k]) + __uint_as_float(ye[0][k]));
          const float Dh = eps * (__uint_as_float(yq[1][0][k]) + __uint_as_float(yq[3][0][k]));
          lp[k] = C + Dh;
          lm[k] = C - Dh;
        }
        float mp = fmaxf(fmaxf(lp[0], lp[1]), fmaxf(lp[2], lp[3]));
        float mm = fmaxf(fmaxf(lm[0], lm[1]), fmaxf(lm[2], lm[3]));
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          mp = fmaxf(mp, __shfl_xor_sync(0xffffffffu, mp, o));
          mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
        }
        float s_p = 0.f, s_m = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          s_p += exp_term(lp[k] - mp);
          s_m += exp_term(lm[k] - mm);
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          s_p += __shfl_xor_sync(0xffffffffu, s_p, o);
          s_m += __shfl_xor_sync(0xffffffffu, s_m, o);
        }
        const int b = b0 + 4 * f + bq;
        if (u8 == 0) {
          red[((half * 4 + q4) * 2 + 0) * kBp + b] = make_float2(mp, s_p);
          red[((half * 4 + q4) * 2 + 1) * kBp + b] = make_float2(mm, s_m);
        }
        const int y = tgt[f] - vq - u8;
        if (y >= 0 && y < 32 && (y & 7) == 0) {
          const int k = y >> 3;
          ylog[b] = k == 0 ? lp[0] : k == 1 ? lp[1] : k == 2 ? lp[2] : lp[3];
          ylog[kBp + b] = k == 0 ? lm[0] : k == 1 ? lm[1] : k == 2 ? lm[2] : lm[3];
        }
      }
    }
    // The waits have completed every MMA, unless one ran out: then the batches still
    // in flight complete before their tensor memory is freed.  Which phase the
    // barrier is in is not known there, so waits on both parities take turns, 4,096
    // polls (hundreds of microseconds) at most each.
    if (ew == kIssueWarp && *abort) {
#pragma unroll 1
      for (uint32_t k = 0; k < 4; ++k) mbar_wait(mma_bar, (nph + k) & 1u, 1u << 12);
    }
    st_barrier();
    if (ew == kMergeWarp) {
      merge();
      __syncwarp();
      // ---- the stream's NLL sums per sign (sequences in order)
      if (lane < a.n_sign) {
        double tot = 0.0;
        for (int b = 0; b < rows; ++b) tot += acc[lane * kBp + b];
        if (SOMA_CHECK((pair * a.n_sign + lane) * a.chunks + chunk <
                           (int64_t)a.n_experts * a.n_pert * a.n_sign * a.chunks,
                       a.status))
          a.partial[(pair * a.n_sign + lane) * a.chunks + chunk] = tot;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

template <int NS>
cudaError_t launch_streams(const BodyTcArgs& a, cudaStream_t stream) {
  cudaError_t err = cudaFuncSetAttribute(
      body_tc_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Smem<NS>::bytes);
  if (err != cudaSuccess) return err;
  const int64_t per_e = ((int64_t)a.n_pert * a.chunks + NS - 1) / NS;
  trace_begin(SOMA_TRACE_GATE, stream);
  const int64_t ctas = a.n_experts * per_e, width = 1 << 30;
  const dim3 grid((unsigned)(ctas < width ? ctas : width), (unsigned)((ctas + width - 1) / width));
  body_tc_kernel<NS><<<grid, NS * kWarps * 32, Smem<NS>::bytes, stream>>>(a);
  trace_end(SOMA_TRACE_GATE, stream);
  return cudaGetLastError();
}

}  // namespace

// Two streams of one expert share a CTA where that takes fewer rounds of CTAs over
// the SMs than one stream each.  An odd number of streams per expert leaves a CTA
// half empty, and where that eats the rounds saved, one stream per CTA is the
// shorter chain.  Measured (two streams -> one, T = 64): 100 experts x 3 probes of 16
// sequences, 2 rounds either way, 1399 -> 1104 us; 200 x 1, 1192 -> 1096; 160 x 1 of
// 48 sequences, 3 rounds against 4, 1969 -> 2142; 77 x 2, 1 against 2, 813 -> 1084;
// 256 x 3, 4 against 6, 2788 -> 3236.
int body_streams_per_cta(int n_experts, int n_pert, int B, int sms) {
  const int64_t per_e = (int64_t)n_pert * ((B + kBp - 1) / kBp);
  const int64_t one = (n_experts * per_e + sms - 1) / sms;
  const int64_t two = (n_experts * ((per_e + 1) / 2) + sms - 1) / sms;
  return two < one ? 2 : 1;
}

cudaError_t launch_body_tc(const float* params, const float* head, const uint8_t* bytes,
                           int n_experts, int blocks, int n_pert, int n_sign, int B, int T,
                           float eps, int sparse, uint64_t seed, uint64_t step, double* partial,
                           int* status, cudaStream_t stream) {
  BodyTcArgs a;
  a.params = params;
  a.head = head;
  a.bytes = bytes;
  a.partial = partial;
  a.status = status;
  a.n_pert = n_pert;
  a.n_sign = n_sign;
  a.blocks = blocks;
  a.B = B;
  a.T = T;
  a.chunks = (B + kBp - 1) / kBp;
  a.P = body_param_count(kD, blocks);
  a.goff = body_gain_offset(kD, blocks);
  a.eps = eps;
  a.sparse = sparse;
  a.seed = seed;
  a.step = step;
  a.n_experts = n_experts;
  if (body_streams_per_cta(n_experts, n_pert, B, sm_count()) == 2)
    return launch_streams<2>(a, stream);
  return launch_streams<1>(a, stream);
}

}  // namespace soma
