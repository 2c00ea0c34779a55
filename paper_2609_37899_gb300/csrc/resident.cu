// resident.cu -- the SPSA forward of small experts with the whole recurrence
// resident in one CTA (tcgen05 / TMEM).
//
// One CTA runs one (expert, probe) pair, both signs, over all T timesteps in
// the mean/difference form of forward_tc.cu, with the difference operand
// scaled by 1 / eps (dhat = dv / eps, an O(1) quantity):
//   a+- = C +- eps D,  C = W vbar + eps^2 (Z dhat) + b,  D = W dhat + Z vbar + z_b.
// The gate weights W = [W_ih | W_hh] and the head weights W_out are converted
// to fp16 tiles in shared memory once, the probe tiles Z of this pair to fp16
// rows in tensor memory (the A operand of the Z products), and the probes are
// therefore drawn once per step, not once per timestep.
// The operand [vbar | dhat] (rows) x [x | h] (K) also lives in shared memory:
// at timestep t it holds [x_{t+1} | h_t] once the cells of t are done.  Cell
// states stay in registers, and the losses are summed in the CTA.
//
// Roles: EW epilogue warps and one warp that issues the MMAs and, while the
// others work, merges the head's partials into the NLL of the last timestep.
// They meet at mbarriers only (every wait bounded): gate_bar and head_bar (MMAs
// done), op_ready (the operand of the next MMAs is written), acc_free (an
// accumulator has been read), red_full (the head's partials are written).
//
// What bounds it: a timestep is a serial chain (gate MMAs, cells, head MMAs,
// head epilogue) of which no part fills the SM, so two independent chains per
// SM are worth more than a shorter one.  Two forms of the kernel:
//  - more pairs than SMs: two CTAs per SM of 8 epilogue warps, each within half
//    of the shared and tensor memory.  The probe tiles in tensor memory are
//    what makes the pair fit (at E = 32, H = 48, B = 16: 64 KB of weights, 32 KB
//    of embedding tables; 128 columns of probe tiles, 128 of accumulators
//    that the gate and the head use in turn).  One CTA's MMAs and waits run
//    under the other's epilogues.
//  - otherwise: one CTA of 16 epilogue warps with separate accumulators for the
//    gate and, twice, the head: the cells of t, on which everything waits, come
//    first, and the head epilogue of t - 1 runs under the gate MMAs of t + 1.
// Measured on GB300 (a step, update included): 256 experts of E = 32, H = 48, 64
// probes, 16 x 512 bytes: 161.9 ms with one CTA of 16 epilogue warps per SM and
// a CTA barrier per timestep, 105.9 ms now (two per SM with a group of four
// sequences at a time 132 ms; groups in pairs 115; a commit per gate tile 110;
// the MMA loops without a branch on the tile's place 107; the form's own parts
// known at compile time 105.9, at T = 64 15.8 -> 15.1).  One expert of E = 32,
// H = 64, 8 probes, 4 x 64 bytes: 207 -> 156 us (the merge off the epilogue
// warps, no barrier).  One MMA of this size occupies the tensor pipe about 46
// cycles, so the 24 of a gate bound the latter's chain.
// The shape limits are checked by res_supported(); other experts use the
// persistent kernel.
#include <cuda_fp16.h>
#include <type_traits>

#define SOMA_CHECK_FILE 2
#include "checked.cuh"
#include "soma_api.h"
#include "soma_device.cuh"
#include "soma_launch.h"
#include "tc_primitives.cuh"

namespace soma {

using namespace tc;

namespace {

constexpr int kResMaxBp = 32;
constexpr size_t kResMaxSmem = 220 * 1024;
// dynamic shared memory of one CTA when two share an SM (228 KB, 1 KB of it
// reserved per CTA)
constexpr size_t kResHalfSmem = 113 * 1024;
constexpr uint32_t kLboRes = 128;  // bytes between core matrices along K

struct ResGeom {
  int E, H, Ek, Hk, K, MTg, Bp, B, T;
  uint32_t wg, zg, wo, zo, op, opsz, emb, dx, red, ylog, acc, ctl, bytes;  // shared-memory offsets
  uint32_t zcol, hcol;  // TMEM columns: probe tiles, head accumulators (gate accumulators at 0)
  uint32_t tmem_cols;   // allocated
  int z_tmem;           // probe tiles in tensor memory (else in shared memory at zg, zo)
  int sep;              // the gate and the head have accumulators of their own
};

__host__ __device__ inline uint32_t res_align(uint32_t x) { return (x + 1023u) & ~1023u; }

struct ResCtl {
  uint64_t gate_bar[2], head_bar[2], op_ready, acc_free, red_full[2], mma_done;
  uint32_t tmem_slot;
  volatile int abort;
};

void res_dims(ResGeom& r, const Layout& lay, int B, int T) {
  r.E = lay.E;
  r.H = lay.H;
  r.Ek = (lay.E + 15) / 16 * 16;
  r.Hk = (lay.H + 15) / 16 * 16;
  r.K = r.Ek + r.Hk;
  r.MTg = (lay.H + 31) / 32;
  r.Bp = (B + 7) / 8 * 8;
  r.B = B;
  r.T = T;
}

// Shared-memory carve-up; the probe tiles take part unless z_tmem.  The operand
// has two buffers: MMAs still read one (the head's in the one-CTA form, those of
// another gate tile in the two-CTA form) while the cells write the other.
void res_carve(ResGeom& r) {
  uint32_t o = 0;
  const uint32_t gate_tile = 128u * r.K * 2, head_tile = 128u * r.Hk * 2;
  r.wg = o; o = res_align(o + r.MTg * gate_tile);
  r.wo = o; o = res_align(o + 2 * head_tile);
  r.zg = o; if (!r.z_tmem) o = res_align(o + r.MTg * gate_tile);
  r.zo = o; if (!r.z_tmem) o = res_align(o + 2 * head_tile);
  r.opsz = 2u * r.Bp * r.K * 2;  // the operand [vbar | dhat] x K, fp16
  r.op = o; o = res_align(o + 2 * r.opsz);
  r.emb = o; o += 256u * r.Ek * 2;   // fp16 Emb rows [V][Ek]
  r.dx = o; o += 256u * r.Ek * 2;    // fp16 z of the Emb rows (dhat of x = z_emb)
  r.red = o; o += 2u * 2 * 4 * 2 * r.Bp * sizeof(float2);  // [t % 2][half][quarter][sign][Bp]
  r.ylog = o; o += 2u * 2 * r.Bp * sizeof(float);          // [t % 2][sign][Bp]
  o = (o + 7u) & ~7u;
  r.acc = o; o += 3u * r.Bp * sizeof(double);          // per sequence: sum nll+, nll-, diff
  o = (o + 7u) & ~7u;
  r.ctl = o; o += (uint32_t)sizeof(ResCtl);
  r.bytes = o + 1024;  // alignment slack of the dynamic shared-memory base
}

// 4 Bp accumulator columns per 128-row tile: the W and the Z product of
// [vbar | dhat].
uint32_t res_tile_cols(const ResGeom& r) { return 4u * r.Bp; }

// Two CTAs per SM; false if the shape does not fit.
bool make_res_geom_half(ResGeom& r, const Layout& lay, int B, int T) {
  res_dims(r, lay, B, T);
  r.z_tmem = 1;
  const uint32_t gate = r.MTg * res_tile_cols(r), head = 2 * res_tile_cols(r);
  const uint32_t z = r.MTg * r.K / 2 + r.Hk;
  r.sep = gate + head + z <= 256;
  r.hcol = r.sep ? gate : 0;
  r.zcol = r.sep ? gate + head : (gate > head ? gate : head);
  r.tmem_cols = 256;
  res_carve(r);
  return r.zcol + z <= 256 && r.bytes <= kResHalfSmem;
}

// One CTA per SM.
ResGeom make_res_geom(const Layout& lay, int B, int T) {
  ResGeom r;
  res_dims(r, lay, B, T);
  r.sep = 1;
  r.hcol = r.MTg * res_tile_cols(r);
  r.zcol = r.hcol + 4 * res_tile_cols(r);
  const uint32_t z = r.MTg * r.K / 2 + r.Hk;
  r.z_tmem = r.zcol + z <= 512;
  const uint32_t cols = r.zcol + (r.z_tmem ? z : 0);
  r.tmem_cols = 32;
  while (r.tmem_cols < cols) r.tmem_cols <<= 1;
  res_carve(r);
  return r;
}

struct ResArgs {
  Sweep sw;
  ResGeom g;
  int n_sign;         // 2: (L+, L-) per pair; 1: L per expert (eps = 0)
  float* losses_out;  // [N][n][2] or [N]
  float* coef_out;    // [N][n] or null
  float* coef_ws;     // [N][n] or null
  int* status;
  size_t n_params, n_bytes;  // extents for the index checks of the checked build
};

// z of flat parameter p as an fp16 +-1 / 0 (sparse) value.
__device__ __forceinline__ __half z_half(const ProbeBits& b, int j) {
  return ((b.act >> j) & 1u) ? (((b.neg >> j) & 1u) ? __float2half_rn(-1.f) : __float2half_rn(1.f))
                             : __float2half_rn(0.f);
}

// fp16 pair word of z at offsets j, j + 1 of a run (natural bit order).
__device__ __forceinline__ uint32_t z_pair_word(const ProbeBits& b, int j, int valid) {
  const __half lo = j < valid ? z_half(b, j) : __float2half_rn(0.f);
  const __half hi = j + 1 < valid ? z_half(b, j + 1) : __float2half_rn(0.f);
  return (uint32_t)__half_as_ushort(lo) | ((uint32_t)__half_as_ushort(hi) << 16);
}

// EW epilogue warps (8: two CTAs per SM, 16: one) and the MMA warp.
template <int EW>
__global__ void __launch_bounds__((EW + 1) * 32, EW == 8 ? 2 : 1) res_kernel(const ResArgs a) {
  constexpr int kThr = (EW + 1) * 32;
  // timesteps that the head epilogue runs behind (on two accumulators)
  constexpr int kLag = EW == 16 ? 1 : 0;
  constexpr int kSeqSplit = EW / 8;                        // warps that share a row quarter
  constexpr int kGroups = kResMaxBp / 4 / kSeqSplit;       // 4-sequence groups of one warp
  constexpr int kXChunks = 512 / (EW * 32);                // embedding chunks of one thread
  extern __shared__ uint8_t dyn_smem[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(dyn_smem) + 1023) & ~uintptr_t(1023));
  const ResGeom& g = a.g;
  // what the form decides is known here
  const bool z_tmem = EW == 8 || g.z_tmem, sep = EW == 16 || g.sep;
  const Sweep& s = a.sw;
  const Layout& L = s.lay;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int e = blockIdx.x / s.n_pert, i = blockIdx.x % s.n_pert;
  const float* th = s.params + (int64_t)e * L.P;
  const ProbeKey pk = make_probe_key(s.seed, s.step, (uint32_t)e, (uint32_t)i);
  const float eps = s.eps;
  const bool do_z = eps != 0.f;
  const float eps2 = eps * eps;
  // dhat_h = (h+ - h-) / (2 eps); 0 when eps = 0 (both signs coincide)
  const float half_inv_eps = do_z ? 0.5f / eps : 0.f;
  ResCtl* ctl = reinterpret_cast<ResCtl*>(smem + g.ctl);
  volatile int* abort = &ctl->abort;
  float2* red = reinterpret_cast<float2*>(smem + g.red);
  float* ylog = reinterpret_cast<float*>(smem + g.ylog);
  double* acc = reinterpret_cast<double*>(smem + g.acc);

  if (tid == 0) {
    mbar_init(&ctl->gate_bar[0], 1);
    mbar_init(&ctl->gate_bar[1], 1);
    mbar_init(&ctl->head_bar[0], 1);
    mbar_init(&ctl->head_bar[1], 1);
    mbar_init(&ctl->op_ready, EW);
    mbar_init(&ctl->acc_free, EW);
    mbar_init(&ctl->red_full[0], EW);
    mbar_init(&ctl->red_full[1], EW);
    mbar_init(&ctl->mma_done, 1);
    ctl->abort = 0;
    mbar_fence_init();
  }
  if (warp == 0) tmem_alloc(&ctl->tmem_slot, g.tmem_cols);

  // ---- resident tiles: W (and Z without z_tmem) of the gate (gate-major
  // quarters) and the head
  const int gate_chunks = g.MTg * 128 * (g.K / 8);
  for (int c = tid; c < gate_chunks; c += kThr) {
    const int m = c / (128 * (g.K / 8)), rem = c % (128 * (g.K / 8));
    const int r = rem / (g.K / 8), k0 = 8 * (rem % (g.K / 8));
    const int U = 32 * m + tile_unit(r);
    const int64_t R = (int64_t)tile_gate(r) * g.H + U;
    __align__(16) __half w[8], z[8];
    int64_t p0 = -1;
    int kmax = 0;  // valid columns of this chunk
    if (U < g.H) {
      if (k0 < g.Ek) {
        p0 = L.w_ih + R * g.E + k0;
        kmax = min(8, g.E - k0);
      } else {
        p0 = L.w_hh + R * g.H + (k0 - g.Ek);
        kmax = min(8, g.H - (k0 - g.Ek));
      }
    }
    ProbeBits zb = {0u, 0u};
    if (!z_tmem && kmax > 0 && do_z) zb = probe_bits(pk, p0, s.sparse);
    if (kmax > 0 && !SOMA_CHECK((size_t)(e * L.P + p0 + kmax) <= a.n_params, a.status)) kmax = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const bool ok = j < kmax;
      w[j] = __float2half_rn(ok ? th[p0 + j] : 0.f);
      z[j] = ok ? z_half(zb, j) : __float2half_rn(0.f);
    }
    const uint32_t off = m * (128u * g.K * 2) + kmajor_offset(r, k0, g.K);
    if (SOMA_CHECK(off + 16 <= g.MTg * 128u * g.K * 2 && (z_tmem || g.zg + off + 16 <= g.bytes), a.status)) {
      *reinterpret_cast<uint4*>(smem + g.wg + off) = *reinterpret_cast<const uint4*>(w);
      if (!z_tmem)
        *reinterpret_cast<uint4*>(smem + g.zg + off) = *reinterpret_cast<const uint4*>(z);
    }
  }
  const int head_chunks = 2 * 128 * (g.Hk / 8);
  for (int c = tid; c < head_chunks; c += kThr) {
    const int h = c / (128 * (g.Hk / 8)), rem = c % (128 * (g.Hk / 8));
    const int r = rem / (g.Hk / 8), k0 = 8 * (rem % (g.Hk / 8));
    const int64_t p0 = L.w_out + (int64_t)(128 * h + r) * g.H + k0;
    int kmax = min(8, g.H - k0);
    if (kmax > 0 && !SOMA_CHECK((size_t)(e * L.P + p0 + kmax) <= a.n_params, a.status)) kmax = 0;
    ProbeBits zb = {0u, 0u};
    if (!z_tmem && kmax > 0 && do_z) zb = probe_bits(pk, p0, s.sparse);
    __align__(16) __half w[8], z[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const bool ok = j < kmax;
      w[j] = __float2half_rn(ok ? th[p0 + j] : 0.f);
      z[j] = ok ? z_half(zb, j) : __float2half_rn(0.f);
    }
    const uint32_t off = h * (128u * g.Hk * 2) + kmajor_offset(r, k0, g.Hk);
    if (SOMA_CHECK(off + 16 <= 2u * 128u * g.Hk * 2 && (z_tmem || g.zo + off + 16 <= g.bytes), a.status)) {
      *reinterpret_cast<uint4*>(smem + g.wo + off) = *reinterpret_cast<const uint4*>(w);
      if (!z_tmem)
        *reinterpret_cast<uint4*>(smem + g.zo + off) = *reinterpret_cast<const uint4*>(z);
    }
  }
  for (int c = tid; c < (int)(2 * g.opsz / 16); c += kThr)
    reinterpret_cast<uint4*>(smem + g.op)[c] = make_uint4(0u, 0u, 0u, 0u);
  // the embedding table and its probe z (the scaled difference of the two
  // signs' inputs, dhat_x = (x+ - x-) / (2 eps) = z_emb), so that the operand
  // of a timestep is gathered from shared memory
  for (int c = tid; c < 256 * (g.Ek / 8); c += kThr) {
    const int v = c / (g.Ek / 8), k0 = 8 * (c % (g.Ek / 8));
    const int64_t p0 = L.emb + (int64_t)v * g.E + k0;
    const int kmax = min(8, g.E - k0);
    ProbeBits zb = {0u, 0u};
    if (do_z && kmax > 0) zb = probe_bits(pk, p0, s.sparse);
    __align__(16) __half x[8], d[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const bool ok = j < kmax;
      x[j] = __float2half_rn(ok ? th[p0 + j] : 0.f);
      d[j] = ok ? z_half(zb, j) : __float2half_rn(0.f);
    }
    reinterpret_cast<uint4*>(smem + g.emb)[c] = *reinterpret_cast<const uint4*>(x);
    reinterpret_cast<uint4*>(smem + g.dx)[c] = *reinterpret_cast<const uint4*>(d);
  }
  for (int c = tid; c < 3 * g.Bp; c += kThr) acc[c] = 0.0;

  // ---- per-thread constants of the epilogues
  // A warp reads TMEM lane quarter w % 4 of tile (gate) or vocabulary half
  // (head) (w / 4) % 2, and of the 4-sequence groups those j with j % kSeqSplit
  // == w / 8: with 16x128b loads thread l holds rows l / 4 + 8 k (k = 0..3) of
  // the quarter and sequence 4 j + l % 4.
  // gate: the four rows are the four gates of unit 8 (w % 4) + l / 4 of the tile
  const int q4 = warp & 3, tile = (warp >> 2) & 1, sp = kSeqSplit == 1 ? 0 : warp >> 3;
  const int u8 = lane >> 2, bq = lane & 3;
  const int U = 32 * tile + 8 * q4 + u8;
  const bool unit_ok = tile < g.MTg && U < g.H;
  float bias[4] = {0.f, 0.f, 0.f, 0.f}, dbias[4] = {0.f, 0.f, 0.f, 0.f};
  if (unit_ok) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t pb = L.b + (int64_t)k * g.H + U;
      bias[k] = th[pb];
      if (do_z) {
        const ProbeBits zb = probe_bits(pk, pb, s.sparse);
        dbias[k] = eps_z(zb.neg & 1u, zb.act & 1u, eps);
      }
    }
  }
  float cst[kGroups][2];  // [group][sign]
#pragma unroll
  for (int c = 0; c < kGroups; ++c) cst[c][0] = cst[c][1] = 0.f;
  // head
  const int vq = 128 * tile + 32 * q4;
  float bo[4], dbo[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t pb = L.b_out + vq + u8 + 8 * k;
    bo[k] = th[pb];
    dbo[k] = 0.f;
    if (do_z) {
      const ProbeBits zb = probe_bits(pk, pb, s.sparse);
      dbo[k] = eps_z(zb.neg & 1u, zb.act & 1u, eps);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = ctl->tmem_slot;
  // probe tiles in tensor memory: thread = row (lane quarter w % 4), 8 columns
  // (16 k) per store; the warps of a quarter share the k steps.  Columns: the
  // gate tiles (K / 2 each), then the head halves (Hk / 2 each).
  if (z_tmem && warp < EW) {
    const int r = 32 * q4 + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * q4) << 16) + g.zcol;
    const int gsteps = g.K / 16, hsteps = g.Hk / 16;
    for (int st = warp >> 2; st < g.MTg * gsteps + 2 * hsteps; st += EW / 4) {
      int64_t p0;
      int kmax = 0;
      if (st < g.MTg * gsteps) {
        const int m = st / gsteps, k0 = 16 * (st % gsteps);
        const int Ur = 32 * m + tile_unit(r);
        const int64_t R = (int64_t)tile_gate(r) * g.H + Ur;
        p0 = k0 < g.Ek ? L.w_ih + R * g.E + k0 : L.w_hh + R * g.H + (k0 - g.Ek);
        if (Ur < g.H) kmax = k0 < g.Ek ? min(16, g.E - k0) : min(16, g.H - (k0 - g.Ek));
      } else {
        const int hs = st - g.MTg * gsteps, h = hs / hsteps, k0 = 16 * (hs % hsteps);
        p0 = L.w_out + (int64_t)(128 * h + r) * g.H + k0;
        kmax = min(16, g.H - k0);
      }
      ProbeBits zb = {0u, 0u};
      if (do_z && kmax > 0) zb = probe_bits(pk, p0, s.sparse);
      uint32_t v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = z_pair_word(zb, 2 * j, kmax);
      if (SOMA_CHECK(g.zcol + 8u * st + 8u <= g.tmem_cols, a.status)) tmem_st8(trow + 8u * st, v);
    }
    tmem_wait_st();
  }
  // MMA descriptors as 32-bit words: the low word holds the start address in
  // 16-byte units, so a step along K (256 bytes) or to the next tile is an
  // addition; gate tiles and the operand share their high word (SBO = 16 K)
  const uint32_t n2 = (uint32_t)(2 * g.Bp);
  const uint32_t idesc = idesc_f16_f32(128, 2 * g.Bp);
  const uint64_t dg = smem_desc(smem_u32(smem + g.wg), kLboRes, (uint32_t)g.K * 16);
  const uint64_t dh = smem_desc(smem_u32(smem + g.wo), kLboRes, (uint32_t)g.Hk * 16);
  const uint32_t ghi = (uint32_t)(dg >> 32), wg_lo = (uint32_t)dg;
  const uint32_t hhi = (uint32_t)(dh >> 32), wo_lo = (uint32_t)dh;
  const uint32_t zg_lo = wg_lo + ((g.zg - g.wg) >> 4), op_lo = wg_lo + ((g.op - g.wg) >> 4);
  const uint32_t zo_lo = wo_lo + ((g.zo - g.wo) >> 4);
  const uint32_t gstep = 16u * g.K, hstep = 16u * g.Hk;  // one 128-row tile, in 16-byte units
  // the operand chunks this thread gathers every timestep (one row, 8 columns)
  const int nx = 2 * g.Bp * (g.Ek / 8);
  int ynext[kXChunks];
  auto x_chunk = [&](int k, int& row, int& k0, int& b, const uint4*& tab) {
    const int c = tid + k * EW * 32;
    row = c / (g.Ek / 8);
    k0 = 8 * (c % (g.Ek / 8));
    const bool delta = row >= g.Bp;
    b = delta ? row - g.Bp : row;
    tab = reinterpret_cast<const uint4*>(smem + (delta ? g.dx : g.emb));
    return warp < EW && c < nx;
  };
  // the embedding part of the first operand (x_0; h_{-1} = 0)
#pragma unroll
  for (int k = 0; k < kXChunks; ++k) {
    int row, k0, b;
    const uint4* tab;
    ynext[k] = 0;
    if (x_chunk(k, row, k0, b, tab) && b < g.B) {
      const int y0 = s.bytes[seq_offset(s, e, i, b)];
      *reinterpret_cast<uint4*>(smem + g.op + kmajor_offset(row, k0, g.K)) =
          tab[y0 * (g.Ek / 8) + k0 / 8];
      if (g.T > 1) ynext[k] = s.bytes[seq_offset(s, e, i, b) + 1];
    }
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  if (warp == EW) {
    // ------------------------------------------------- MMA issue, NLL merge
    // gate of t: [x_t | h_{t-1}]; head of t: the h part, once h_t is written
    // one 128-row tile: W and Z against the operand at ob, each into its own
    // columns; the descriptors stay in few instructions per MMA
    auto issue_tile = [&](uint32_t d, uint32_t wlo, uint32_t whi, uint32_t zlo, uint32_t zhi,
                          uint32_t zt, uint32_t ob, int steps) {
      if (z_tmem) {
#pragma unroll 4
        for (int k16 = 0; k16 < steps; ++k16) {
          const uint32_t ko = (uint32_t)k16 * 16, af = k16 > 0 ? 1u : 0u;
          mma_f16_ss_lohi(d, wlo + ko, whi, ob + ko, ghi, idesc, af);
          mma_f16_ts_lohi(d + n2, zt + 8u * k16, ob + ko, ghi, idesc, af);
        }
      } else {
#pragma unroll 4
        for (int k16 = 0; k16 < steps; ++k16) {
          const uint32_t ko = (uint32_t)k16 * 16, af = k16 > 0 ? 1u : 0u;
          mma_f16_ss_lohi(d, wlo + ko, whi, ob + ko, ghi, idesc, af);
          mma_f16_ss_lohi(d + n2, zlo + ko, zhi, ob + ko, ghi, idesc, af);
        }
      }
    };
    auto issue_gate = [&](int t) {
      const uint32_t ob = op_lo + ((t & 1) ? g.opsz >> 4 : 0u);
      if (!SOMA_CHECK(g.MTg * 4u * g.Bp <= g.tmem_cols, a.status)) return;
      if (elect_one()) {
#pragma unroll 1
        for (int m = 0; m < g.MTg; ++m) {
          const uint32_t d = tmem + (uint32_t)m * 2 * n2;
          const uint32_t wlo = wg_lo + (uint32_t)m * gstep, zlo = zg_lo + (uint32_t)m * gstep;
          const uint32_t zt = tmem + g.zcol + (uint32_t)(m * g.K / 2);
          issue_tile(d, wlo, ghi, zlo, ghi, zt, ob, g.K / 16);
          if (EW == 8) mma_commit(&ctl->gate_bar[m]);
        }
        if (EW != 8) mma_commit(&ctl->gate_bar[0]);
      }
      __syncwarp();
    };
    auto issue_head = [&](int t) {
      const int buf = kLag ? t & 1 : 0;
      const uint32_t hc = g.hcol + (uint32_t)buf * 4 * n2;
      if (!SOMA_CHECK(hc + 8u * g.Bp <= g.tmem_cols, a.status)) return;
      if (elect_one()) {
        // the operand of t + 1, Ek / 8 core matrices further
        const uint32_t obh = op_lo + (!(t & 1) ? g.opsz >> 4 : 0u) + (uint32_t)g.Ek;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          const uint32_t d = tmem + hc + (uint32_t)h * 2 * n2;
          const uint32_t wlo = wo_lo + (uint32_t)h * hstep, zlo = zo_lo + (uint32_t)h * hstep;
          const uint32_t zt = tmem + g.zcol + (uint32_t)(g.MTg * g.K / 2 + h * g.Hk / 2);
          issue_tile(d, wlo, hhi, zlo, hhi, zt, obh, g.Hk / 16);
        }
        mma_commit(&ctl->head_bar[buf]);
      }
      __syncwarp();
    };
    // NLL of timestep t from the partials: lane = (sequence, sign), two rounds
    // for more than 16 sequences; sums in fp64, the difference exact
    double sum[2] = {0.0, 0.0}, dif[2] = {0.0, 0.0};
    auto merge = [&](int t) {
      const float2* rd = red + (t & 1) * 16 * g.Bp;
      const float* yl = ylog + (t & 1) * 2 * g.Bp;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int idx = lane + 32 * k, b = idx >> 1, sg = idx & 1;
        if (32 * k >= 2 * g.B) break;
        float nll = 0.f;
        if (b < g.B) {
          float M = -INFINITY;
          for (int h = 0; h < 8; ++h) M = fmaxf(M, rd[(h * 2 + sg) * g.Bp + b].x);
          float S = 0.f;
          for (int h = 0; h < 8; ++h) {
            const float2 q = rd[(h * 2 + sg) * g.Bp + b];
            S += q.y * __expf(q.x - M);
          }
          nll = M + logf(S) - yl[sg * g.Bp + b];
        }
        const float other = __shfl_xor_sync(0xffffffffu, nll, 1);
        sum[k] += (double)nll;
        dif[k] += (double)nll - (double)other;  // exact in fp64; the + lane's is used
      }
    };
    issue_gate(0);
    bool alive = true;
    for (int t = 0; t < g.T; ++t) {
      alive = lane_wait_inline(&ctl->op_ready, (uint32_t)t & 1u, abort, a.status);
      if (__any_sync(0xffffffffu, !alive)) break;
      tc_fence_after();
      if (kLag) {
        if (t + 1 < g.T) issue_gate(t + 1);
        issue_head(t);
      } else {
        issue_head(t);
        if (!sep) {
          alive = lane_wait_inline(&ctl->acc_free, (uint32_t)t & 1u, abort, a.status);
          if (__any_sync(0xffffffffu, !alive)) break;
          tc_fence_after();
        }
        if (t + 1 < g.T) issue_gate(t + 1);
      }
      if (t >= kLag) {
        const int tm = t - kLag;
        alive = lane_wait_inline(&ctl->red_full[tm & 1], (uint32_t)(tm >> 1) & 1u, abort, a.status);
        if (__any_sync(0xffffffffu, !alive)) break;
        merge(tm);
      }
    }
    if (__all_sync(0xffffffffu, alive) && kLag) {
      alive = lane_wait_inline(&ctl->red_full[(g.T - 1) & 1], (uint32_t)((g.T - 1) >> 1) & 1u,
                               abort, a.status);
      if (__all_sync(0xffffffffu, alive)) merge(g.T - 1);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int idx = lane + 32 * k, b = idx >> 1, sg = idx & 1;
      if (b < g.B) {
        acc[sg * g.Bp + b] = sum[k];
        if (sg == 0) acc[2 * g.Bp + b] = dif[k];
      }
    }
    // every MMA of this CTA completes before its tensor memory is freed
    if (elect_one()) mma_commit(&ctl->mma_done);
    __syncwarp();
    mbar_wait(&ctl->mma_done, 0);
  } else {
    // ------------------------------------------------------------- epilogues
    const uint32_t tq0 = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)tile * 4 * g.Bp;
    // The accumulator columns of NG 4-sequence groups from sequence b0, in
    // steps of `kStep`: W vbar, W dhat, Z vbar, Z dhat of this thread's four
    // rows.  With one warp per quarter (EW = 8) the groups go in pairs (Bp is a
    // multiple of 8), so one group's dependent chain runs under the other's;
    // with two warps per quarter a group is all the latency there is to hide.
    constexpr int kStep = 4 * kSeqSplit;
    auto load_groups = [&](auto ng, uint32_t tq, int b0, uint32_t (&wv)[2][4],
                           uint32_t (&wd)[2][4], uint32_t (&zv)[2][4], uint32_t (&zd)[2][4]) {
      const uint32_t tq2 = tq + (16u << 16);
#pragma unroll
      for (int h = 0; h < decltype(ng)::value; ++h) {
        const uint32_t cw = (uint32_t)(b0 + h * kStep);
        tmem_ld_16x128b(tq + cw, wv[h][0], wv[h][1]);
        tmem_ld_16x128b(tq2 + cw, wv[h][2], wv[h][3]);
        tmem_ld_16x128b(tq + cw + g.Bp, wd[h][0], wd[h][1]);
        tmem_ld_16x128b(tq2 + cw + g.Bp, wd[h][2], wd[h][3]);
        tmem_ld_16x128b(tq + 2 * g.Bp + cw, zv[h][0], zv[h][1]);
        tmem_ld_16x128b(tq2 + 2 * g.Bp + cw, zv[h][2], zv[h][3]);
        tmem_ld_16x128b(tq + 3 * g.Bp + cw, zd[h][0], zd[h][1]);
        tmem_ld_16x128b(tq2 + 3 * g.Bp + cw, zd[h][2], zd[h][3]);
      }
      tmem_wait_ld();
    };
    // the rows of bytes of this thread's sequences b = bq + 4 sp + k kStep
    const int T1 = g.T + 1;
    const uint8_t* brow = s.bytes + seq_offset(s, e, i, 0) + (int64_t)(bq + 4 * sp) * T1;
    // partials of the warp's quarter and the target logit of NG groups
    auto head_groups = [&](auto ng, int t, int c, uint32_t tq, float2* rd, float* yl, bool last) {
      constexpr int NG = decltype(ng)::value;
      const int b0 = 4 * sp + c * kStep;
      int tgt[NG];  // the target bytes, loaded under the rest
#pragma unroll
      for (int h = 0; h < NG; ++h) {
        tgt[h] = -1;
        if (b0 + h * kStep + bq < g.B &&
            SOMA_CHECK((size_t)(brow - s.bytes) + (size_t)(c + h) * kStep * T1 + t + 1 < a.n_bytes,
                       a.status))
          tgt[h] = brow[(c + h) * kStep * T1 + t + 1];
      }
      uint32_t wv[2][4], wd[2][4], zv[2][4], zd[2][4];
      load_groups(ng, tq, b0, wv, wd, zv, zd);
      if (last && !sep) {  // the last read of the accumulator
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl->acc_free);
      }
      float lp[NG][4], lm[NG][4], mp[NG], mm[NG], s_p[NG], s_m[NG];
#pragma unroll
      for (int h = 0; h < NG; ++h) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float C = fmaf(eps2, __uint_as_float(zd[h][k]), __uint_as_float(wv[h][k])) + bo[k];
          const float D =
              fmaf(eps, __uint_as_float(wd[h][k]) + __uint_as_float(zv[h][k]), dbo[k]);
          lp[h][k] = C + D;
          lm[h][k] = C - D;
        }
        mp[h] = fmaxf(fmaxf(lp[h][0], lp[h][1]), fmaxf(lp[h][2], lp[h][3]));
        mm[h] = fmaxf(fmaxf(lm[h][0], lm[h][1]), fmaxf(lm[h][2], lm[h][3]));
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int h = 0; h < NG; ++h) {
          mp[h] = fmaxf(mp[h], __shfl_xor_sync(0xffffffffu, mp[h], o));
          mm[h] = fmaxf(mm[h], __shfl_xor_sync(0xffffffffu, mm[h], o));
        }
#pragma unroll
      for (int h = 0; h < NG; ++h) {
        s_p[h] = s_m[h] = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          s_p[h] += exp_term(lp[h][k] - mp[h]);
          s_m[h] += exp_term(lm[h][k] - mm[h]);
        }
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1)
#pragma unroll
        for (int h = 0; h < NG; ++h) {
          s_p[h] += __shfl_xor_sync(0xffffffffu, s_p[h], o);
          s_m[h] += __shfl_xor_sync(0xffffffffu, s_m[h], o);
        }
#pragma unroll
      for (int h = 0; h < NG; ++h) {
        const int b = b0 + h * kStep + bq;
        if (u8 == 0) {
          rd[((tile * 4 + q4) * 2 + 0) * g.Bp + b] = make_float2(mp[h], s_p[h]);
          rd[((tile * 4 + q4) * 2 + 1) * g.Bp + b] = make_float2(mm[h], s_m[h]);
        }
        const int y = tgt[h] - vq - u8;
        if (y >= 0 && y < 32 && (y & 7) == 0) {
          const int k = y >> 3;
          yl[b] = k == 0 ? lp[h][0] : k == 1 ? lp[h][1] : k == 2 ? lp[h][2] : lp[h][3];
          yl[g.Bp + b] = k == 0 ? lm[h][0] : k == 1 ? lm[h][1] : k == 2 ? lm[h][2] : lm[h][3];
        }
      }
    };
    // This lane's answer: the caller votes on it.  No lane leaves before the vote,
    // so after a wait that ran out the accumulators are read all the same (in
    // bounds, whatever they hold).
    auto head_epilogue = [&](int t) -> bool {
      const uint32_t hb = kLag ? (uint32_t)t & 1u : 0u;
      const uint32_t par = kLag ? (uint32_t)(t >> 1) & 1u : (uint32_t)t & 1u;
      const bool ok = lane_wait_inline(&ctl->head_bar[hb], par, abort, a.status);
      tc_fence_after();
      const uint32_t tq = tq0 + g.hcol + hb * 8u * g.Bp;
      float2* rd = red + (t & 1) * 16 * g.Bp;
      float* yl = ylog + (t & 1) * 2 * g.Bp;
#pragma unroll
      for (int c = 0; c < kGroups; c += (kSeqSplit == 1 ? 2 : 1)) {
        const int b0 = 4 * sp + c * kStep;
        if (b0 >= g.Bp) break;
        if constexpr (kSeqSplit == 1)
          head_groups(std::integral_constant<int, 2>(), t, c, tq, rd, yl, b0 + 2 * kStep >= g.Bp);
        else
          head_groups(std::integral_constant<int, 1>(), t, c, tq, rd, yl, b0 + kStep >= g.Bp);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->red_full[t & 1]);
      return ok;
    };
    // gates and cells of NG groups; h into the operand of t + 1
    auto gate_groups = [&](auto ng, int c, uint8_t* opn) {
      constexpr int NG = decltype(ng)::value;
      const int b0 = 4 * sp + c * kStep;
      uint32_t wv[2][4], wd[2][4], zv[2][4], zd[2][4];
      load_groups(ng, tq0, b0, wv, wd, zv, zd);
#pragma unroll
      for (int h = 0; h < NG; ++h) {
        float actp[4], actm[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float C =
              fmaf(eps2, __uint_as_float(zd[h][k]), __uint_as_float(wv[h][k])) + bias[k];
          const float D =
              fmaf(eps, __uint_as_float(wd[h][k]) + __uint_as_float(zv[h][k]), dbias[k]);
          if (k == 2) {
            actp[k] = tanh_f(C + D);
            actm[k] = tanh_f(C - D);
          } else {
            actp[k] = sigmoid_f(C + D);
            actm[k] = sigmoid_f(C - D);
          }
        }
        const float cp = fmaf(actp[1], cst[c + h][0], actp[0] * actp[2]);
        const float cm = fmaf(actm[1], cst[c + h][1], actm[0] * actm[2]);
        cst[c + h][0] = cp;
        cst[c + h][1] = cm;
        float hsum, hdif;
        h_sum_diff(actp[3], tanh_f(cp), actm[3], tanh_f(cm), hsum, hdif);
        const int b = b0 + h * kStep + bq;
        if (unit_ok && b < g.B &&
            SOMA_CHECK(kmajor_offset(g.Bp + b, g.Ek + U, g.K) + 2 <= g.opsz, a.status)) {
          *reinterpret_cast<__half*>(opn + kmajor_offset(b, g.Ek + U, g.K)) =
              __float2half_rn(0.5f * hsum);
          *reinterpret_cast<__half*>(opn + kmajor_offset(g.Bp + b, g.Ek + U, g.K)) =
              __float2half_rn(hdif * half_inv_eps);
        }
      }
    };
    bool alive = true;
    for (int t = 0; t < g.T; ++t) {
      // the operand of t + 1: [x_{t+1} | h_t]
      uint8_t* opn = smem + g.op + (!(t & 1) ? g.opsz : 0u);
      alive = lane_wait_inline(&ctl->gate_bar[EW == 8 && tile < g.MTg ? tile : 0], (uint32_t)t & 1u,
                               abort, a.status);
      if (__any_sync(0xffffffffu, !alive)) break;
      tc_fence_after();
      if (32 * tile + 8 * q4 < g.H) {  // the quarter holds units of the expert
#pragma unroll
        for (int c = 0; c < kGroups; c += (kSeqSplit == 1 ? 2 : 1)) {
          const int b0 = 4 * sp + c * kStep;
          if (b0 >= g.Bp) break;
          if constexpr (kSeqSplit == 1)
            gate_groups(std::integral_constant<int, 2>(), c, opn);
          else
            gate_groups(std::integral_constant<int, 1>(), c, opn);
        }
      }
      // the embedding part of t + 1
      if (t + 1 < g.T) {
#pragma unroll
        for (int k = 0; k < kXChunks; ++k) {
          int row, k0, b;
          const uint4* tab;
          if (x_chunk(k, row, k0, b, tab) && b < g.B) {
            *reinterpret_cast<uint4*>(opn + kmajor_offset(row, k0, g.K)) =
                tab[ynext[k] * (g.Ek / 8) + k0 / 8];
            if (t + 2 < g.T) ynext[k] = s.bytes[seq_offset(s, e, i, b) + t + 2];
          }
        }
      }
      fence_async_smem();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->op_ready);
      if (t >= kLag) {
        alive = head_epilogue(t - kLag);
        if (__any_sync(0xffffffffu, !alive)) break;
      }
    }
    if (kLag && __all_sync(0xffffffffu, alive)) head_epilogue(g.T - 1);
  }
  tc_fence_before();
  __syncthreads();

  // ---- losses and coefficient of the pair (fp64 sums, sequences in order)
  if (tid == 0) {
    double sp = 0.0, sm = 0.0, sd = 0.0;
    for (int b = 0; b < g.B; ++b) {
      sp += acc[b];
      sm += acc[g.Bp + b];
      sd += acc[2 * g.Bp + b];
    }
    const double inv = 1.0 / ((double)g.B * (double)g.T);
    const double Lp = sp * inv, Lm = sm * inv, D = sd * inv;
    const double c = (eps == 0.f) ? 0.0 : D / (2.0 * (double)eps);
    const int64_t pair = blockIdx.x;
    if (a.n_sign == 2) {
      a.losses_out[pair * 2] = (float)Lp;
      a.losses_out[pair * 2 + 1] = (float)Lm;
    } else {
      a.losses_out[pair] = (float)Lp;
    }
    if (a.coef_out) a.coef_out[pair] = (float)c;
    if (a.coef_ws) a.coef_ws[pair] = (float)c;
    if (!(isfinite(Lp) && isfinite(Lm) && isfinite(c))) atomicCAS(a.status, 0, kStatusNonFinite);
  }
  if (warp == 0) tmem_dealloc(tmem, g.tmem_cols);
}

}  // namespace

// Which experts run here.  The line is where all tiles of a pair, probe tiles
// included, fit the shared memory of one CTA and the gate and two head
// accumulators the tensor memory; it stays there although the probe tiles now
// sit in tensor memory, because the persistent kernel, which takes the
// others, rounds the eps^2 term differently and a call's results do not move.
bool res_supported(const Layout& lay, int B) {
  if (B < 1 || B > kResMaxBp || lay.H > 64) return false;
  ResGeom g;
  res_dims(g, lay, B, 1);
  const uint32_t gate = g.MTg * 128u * g.K * 2, head = 2u * 128u * g.Hk * 2;
  const uint32_t op = 2u * 2u * g.Bp * g.K * 2;
  uint32_t o = res_align(gate);
  o = res_align(o + gate);
  o = res_align(o + head);
  o = res_align(o + head);
  o = res_align(o + op);
  o += 2u * 256u * g.Ek * 2 + 2u * 4 * 2 * g.Bp * sizeof(float2) + 2u * g.Bp * sizeof(float);
  o += 3u * g.Bp * sizeof(double) + 64 + 1024;
  return o <= kResMaxSmem && 2 * g.Bp * (g.Ek / 8) <= 512 && (g.MTg + 4) * 4 * g.Bp <= 512;
}

template <int EW>
static cudaError_t launch_res(const ResArgs& a, int pairs, cudaStream_t stream) {
  cudaError_t e =
      cudaFuncSetAttribute(res_kernel<EW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           EW == 8 ? (int)kResHalfSmem : kSmemOptIn);
  if (e != cudaSuccess) return e;
  trace_begin(SOMA_TRACE_GATE, stream);
  res_kernel<EW><<<pairs, (EW + 1) * 32, a.g.bytes, stream>>>(a);
  trace_end(SOMA_TRACE_GATE, stream);
  return cudaGetLastError();
}

cudaError_t launch_forward_res(const Sweep& s, int n_sign, float* losses_out, float* coef_out,
                               float* coef_ws, int* status, cudaStream_t stream) {
  ResArgs a;
  a.sw = s;
  a.n_sign = n_sign;
  a.losses_out = losses_out;
  a.coef_out = coef_out;
  a.coef_ws = coef_ws;
  a.status = status;
  a.n_params = (size_t)s.n_experts * s.lay.P;
  a.n_bytes = (size_t)(s.batch_per_probe ? s.n_experts * s.n_pert : s.n_experts) * s.B_mem *
              (size_t)(s.T + 1);
  const int pairs = s.n_experts * s.n_pert;
  if (pairs > sm_count() && make_res_geom_half(a.g, s.lay, s.B, s.T))
    return launch_res<8>(a, pairs, stream);
  a.g = make_res_geom(s.lay, s.B, s.T);
  return launch_res<16>(a, pairs, stream);
}

}  // namespace soma
