// fdd_mac_fp32.cu -- FP32 phase-rotate-and-sum on CUDA cores (Sect. 2.2,
// Eqs. 4 and 7):
//
//   Y[j][k] = sum_nu W(k, nu, j) X[nu][k],   W = exp(+2 pi i k d(nu, DM_j) / L)
//
// for a uniform trial grid DM_j = DM_0 + j dDM.  The phase of W in cycles is
// k DM_0 c_nu / L + k j dDM c_nu / L with c_nu the per-channel delay rate of
// Eq. 1; both terms are held as exact 64-bit fixed-point fractions of a cycle
// (u_nu, v_nu, computed on the host), so the reduction "modulo one cycle" of
// the phase is exact integer wrap-around and needs no FP64 on the device.
//
// Because the phase is linear in j, the phasor factorises over a split of
// the trial index j = a T + b:
//
//   W(k, nu, aT + b) = Q_a(k, nu) P_b(k, nu),
//   Q_a = exp(2 pi i (k u + k aT v) 2^-64),  P_b = exp(2 pi i k b v 2^-64).
//
// Hence for each bin, Y[aT + b] = sum_nu (X Q_a) P_b is a complex
// (A x N_nu)(N_nu x T) matrix product whose operands are generated on the
// fly.  A warp owns one bin (or a few bins) and a block of A*T trials.  For
// every channel, each lane evaluates a few Z_a = X Q_a and P_b directly from
// the exact phase (MUFU sin/cos, no recurrence), the warp swaps them through
// shared memory, and each lane accumulates an AT x BT register tile with four
// FP32 FMAs per complex multiply-accumulate, the FP32-pipe minimum for 8
// flops.
//
// The arithmetic uses Blackwell's paired FMA (__ffma2_rn: two FMAs per issued
// instruction at the single-FMA pipe rate), pairs running along b:
//   re[a][b:b+2] += (zr, zr)(pr_b, pr_b+1) + (-zi, -zi)(pi_b, pi_b+1)
//   im[a][b:b+2] += (zr, zr)(pi_b, pi_b+1) + (zi, zi)(pr_b, pr_b+1)
// with Z swapped as (zr, zi) pairs and P as planes pr, pi; the broadcast
// pairs are formed in registers.  Two schedules share it: the plain one
// (every warp evaluates its phasors, synchronises, loads and accumulates,
// per channel), used by the smaller tiles, and the warp-specialised one
// below, used by the 2048-trial tile.
// Lanes are numbered lane = ga * GB + gb, so each quarter warp reads a single
// Z row (a broadcast) and GB distinct P rows; the P rows are padded so that
// those reads fall in distinct shared-memory banks.
#include <cstdio>

#include "fdd_device.cuh"
#include "fdd_internal.h"

namespace fdd {
namespace {

using dev::top32_mul;
using dev::unit_phasor;

constexpr int kWarps = 8;
constexpr int kUnroll = 4;  // channels per unrolled group (X loads run one group ahead)

template <int AT_, int BT_, int GA_, int GB_>
struct Geom {
  static constexpr int AT = AT_;        // Z_a values per lane
  static constexpr int BT = BT_;        // P_b values per lane
  static constexpr int GA = GA_;        // lanes along a in a bin group
  static constexpr int GB = GB_;        // lanes along b in a bin group
  static constexpr int G = GA * GB;     // lanes per bin group
  static constexpr int NG = 32 / G;     // bin groups per warp
  static constexpr int AW = GA * AT;    // A: super-steps of the trial block
  static constexpr int TW = GB * BT;    // T: sub-steps of the trial block
  static constexpr int DMS = AW * TW;   // trials per block
  static constexpr int ZGEN = (AW + G - 1) / G;  // Z_a evaluated per lane
  static constexpr int PGEN = (TW + G - 1) / G;  // P_b evaluated per lane
  static_assert(32 % G == 0, "bin group must divide a warp");
};

using G8x8 = Geom<8, 8, 4, 8>;  // 32 x 64 = 2048 trials per bin and warp
using G4x8 = Geom<4, 8, 4, 8>;  // 16 x 64 = 1024
using G4x4 = Geom<4, 4, 2, 4>;  //  8 x 16 =  128, four bins per warp
using G8x8q = Geom<8, 8, 2, 4>; // 16 x 32 =  512, four bins per warp

// ------------------------------------------------- paired-FMA tile, compact swap
// Z swapped as (zr, zi) pairs and P as planes pr, pi; the broadcast pairs
// (zr, zr), (zi, zi), (-zi, -zi) are formed in registers.
template <class Gm>
struct PackedCompact {
  static constexpr int AT = Gm::AT, BT = Gm::BT;
  static constexpr int ZROW = 2 * AT + 4;   // padded a-rows of (zr, zi) pairs
  static constexpr int PSTR = BT + 4;       // padded b-rows of a plane
  static constexpr int ZFL = Gm::GA * ZROW;
  static constexpr int PFL = Gm::GB * PSTR;
  static constexpr int GFL = ZFL + 2 * PFL;
  static_assert(AT % 2 == 0 && BT % 4 == 0, "rows are read as float4");

  struct Ops {
    float zr[AT], zi[AT];
    float2 pr[BT / 2], pi[BT / 2];
  };
  struct Acc {
    float2 re[AT][BT / 2], im[AT][BT / 2];
  };
  static __device__ __forceinline__ void zero(Acc& c) {
#pragma unroll
    for (int i = 0; i < AT; ++i)
#pragma unroll
      for (int j = 0; j < BT / 2; ++j) c.re[i][j] = c.im[i][j] = make_float2(0.f, 0.f);
  }
  static __device__ __forceinline__ int z_off(int a) { return (a / AT) * ZROW + 2 * (a % AT); }
  static __device__ __forceinline__ int p_off(int b) { return ZFL + (b / BT) * PSTR + (b % BT); }
  static __device__ __forceinline__ void put_z(float* grp, int off, float zr, float zi) {
    *reinterpret_cast<float2*>(grp + off) = make_float2(zr, zi);
  }
  static __device__ __forceinline__ void put_p(float* grp, int off, float pr, float pi) {
    grp[off] = pr;
    grp[off + PFL] = pi;
  }
  static __device__ __forceinline__ void load(const float* grp, int ga, int gb, Ops& o) {
    const float4* z = reinterpret_cast<const float4*>(grp + ga * ZROW);
#pragma unroll
    for (int h = 0; h < AT / 2; ++h) {
      const float4 v = z[h];
      o.zr[2 * h] = v.x;
      o.zi[2 * h] = v.y;
      o.zr[2 * h + 1] = v.z;
      o.zi[2 * h + 1] = v.w;
    }
    const float* row = grp + ZFL + gb * PSTR;
#pragma unroll
    for (int h = 0; h < BT / 4; ++h) {
      const float4 r = *reinterpret_cast<const float4*>(row + 4 * h);
      const float4 i = *reinterpret_cast<const float4*>(row + PFL + 4 * h);
      o.pr[2 * h] = make_float2(r.x, r.y);
      o.pr[2 * h + 1] = make_float2(r.z, r.w);
      o.pi[2 * h] = make_float2(i.x, i.y);
      o.pi[2 * h + 1] = make_float2(i.z, i.w);
    }
  }
  static __device__ __forceinline__ void mac(Acc& c, const Ops& o) {
#pragma unroll
    for (int i = 0; i < AT; ++i) {
      const float2 zr = make_float2(o.zr[i], o.zr[i]);
      const float2 zi = make_float2(o.zi[i], o.zi[i]);
      const float2 zn = make_float2(-o.zi[i], -o.zi[i]);
#pragma unroll
      for (int j = 0; j < BT / 2; ++j) {
        c.re[i][j] = __ffma2_rn(zr, o.pr[j], c.re[i][j]);
        c.im[i][j] = __ffma2_rn(zr, o.pi[j], c.im[i][j]);
      }
#pragma unroll
      for (int j = 0; j < BT / 2; ++j) {
        c.re[i][j] = __ffma2_rn(zn, o.pi[j], c.re[i][j]);
        c.im[i][j] = __ffma2_rn(zi, o.pr[j], c.im[i][j]);
      }
    }
  }
  static __device__ __forceinline__ float2 get(const Acc& c, int i, int j) {
    const float2 r = c.re[i][j / 2], m = c.im[i][j / 2];
    return (j & 1) ? make_float2(r.y, m.y) : make_float2(r.x, m.x);
  }
};

template <class Gm, class M>
struct Generator {
  uint32_t mz[Gm::ZGEN], mp[Gm::PGEN];
  int zoff[Gm::ZGEN], poff[Gm::PGEN];
  bool zon[Gm::ZGEN], pon[Gm::PGEN];
  uint32_t ku;

  __device__ __forceinline__ void init(uint32_t k, int lg, int j_first) {
    ku = k;
#pragma unroll
    for (int q = 0; q < Gm::ZGEN; ++q) {
      const int ai = lg + q * Gm::G;
      zon[q] = ai < Gm::AW;
      mz[q] = k * static_cast<uint32_t>(j_first + ai * Gm::TW);
      zoff[q] = M::z_off(ai);
    }
#pragma unroll
    for (int q = 0; q < Gm::PGEN; ++q) {
      const int bi = lg + q * Gm::G;
      pon[q] = bi < Gm::TW;
      mp[q] = k * static_cast<uint32_t>(bi);
      poff[q] = M::p_off(bi);
    }
  }
  __device__ __forceinline__ void run(const PhaseConst& p, float2 x, float* grp) const {
    const uint32_t base = top32_mul(ku, p.u_lo, p.u_hi);
#pragma unroll
    for (int q = 0; q < Gm::ZGEN; ++q) {
      if (zon[q]) {
        const float2 w = unit_phasor(base + top32_mul(mz[q], p.v_lo, p.v_hi));
        M::put_z(grp, zoff[q], x.x * w.x - x.y * w.y, x.x * w.y + x.y * w.x);
      }
    }
#pragma unroll
    for (int q = 0; q < Gm::PGEN; ++q) {
      if (pon[q]) {
        const float2 w = unit_phasor(top32_mul(mp[q], p.v_lo, p.v_hi));
        M::put_p(grp, poff[q], w.x, w.y);
      }
    }
  }
};

// One CTA's block of work: bins (bin_tile * W + warp) * NG + g and trials
// dm_block * DMS + .. of one set of spectra, with the phase table already in
// shared memory (pcs) and the swap area behind it.
template <class Gm, class M, int W>
__device__ __forceinline__ void mac_block(const MacArgs& a, const PhaseConst* pcs,
                                          float* swap_all, int bin_tile, int dm_block,
                                          int series) {
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int g = lane / Gm::G;
  const int lg = lane % Gm::G;
  const int ga = lg / Gm::GB;
  const int gb = lg % Gm::GB;
  const int k = (bin_tile * W + warp) * Gm::NG + g;  // local bin
  const bool k_ok = k < a.n_bins;
  const int kl = k_ok ? k : 0;  // idle groups run local bin 0, store nothing
  const uint32_t ku = static_cast<uint32_t>(a.k_begin + kl);
  const int jblk = dm_block * Gm::DMS;
  const int nc = a.n_chan;

  constexpr int kStage = Gm::NG * M::GFL;  // floats per warp per stage
  float* grp0 = swap_all + warp * 2 * kStage + g * M::GFL;

  Generator<Gm, M> gen;
  gen.init(ku, lg, a.j_begin + jblk);

  const float2* xp = a.X + static_cast<int64_t>(series) * a.x_series_stride + kl;
  const int64_t xs = a.x_chan_stride;
  typename M::Acc acc;
  M::zero(acc);

  float2 xcur[kUnroll];
#pragma unroll
  for (int i = 0; i < kUnroll; ++i) xcur[i] = (i < nc) ? __ldg(xp + i * xs) : make_float2(0.f, 0.f);

  // per channel c: generate(c) -> sync -> load(c) -> MAC(c); two swap stages,
  // so generate(c + 1) writes the stage that load(c - 1) read before the sync
  // that closed channel c.
  int stage = 0;
  for (int c0 = 0; c0 < nc; c0 += kUnroll) {
    float2 xnext[kUnroll];
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) {
      const int c = c0 + kUnroll + i;
      xnext[i] = (c < nc) ? __ldg(xp + c * xs) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) {
      const int c = c0 + i;
      if (c < nc) {
        float* cur = grp0 + stage * kStage;
        typename M::Ops ops;
        gen.run(pcs[c], xcur[i], cur);
        __syncwarp();
        M::load(cur, ga, gb, ops);
        M::mac(acc, ops);
        stage ^= 1;
      }
    }
#pragma unroll
    for (int i = 0; i < kUnroll; ++i) xcur[i] = xnext[i];
  }

  if (!k_ok) return;
  const bool real_only = (a.k_begin + k == a.real_bin_a) || (a.k_begin + k == a.real_bin_b);
#pragma unroll
  for (int ii = 0; ii < Gm::AT; ++ii) {
#pragma unroll
    for (int jj = 0; jj < Gm::BT; ++jj) {
      const int jl = jblk + (ga * Gm::AT + ii) * Gm::TW + gb * Gm::BT + jj;
      if (jl < a.n_dm) {
        const float2 v = M::get(acc, ii, jj);
        const float re = v.x * a.scale;
        const float im = real_only ? 0.f : v.y * a.scale;
        const int64_t o = static_cast<int64_t>(series) * a.y_series_stride +
                          static_cast<int64_t>(jl) * a.y_dm_stride + k;
        if (a.out_kind == 2)
          static_cast<float*>(a.Y)[o] = re * re + im * im;
        else
          static_cast<float2*>(a.Y)[o] = make_float2(re, im);
      }
    }
  }
}

template <class Gm, class M, int W = kWarps>
__global__ void __launch_bounds__(W * 32, 1) mac_kernel(const MacArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PhaseConst* pcs = reinterpret_cast<PhaseConst*>(smem_raw);
  float* swap_all = reinterpret_cast<float*>(smem_raw + sizeof(PhaseConst) * a.n_chan);
  for (int i = threadIdx.x; i < a.n_chan; i += W * 32) pcs[i] = a.pc[i];
  __syncthreads();
  mac_block<Gm, M, W>(a, pcs, swap_all, blockIdx.x, blockIdx.y, blockIdx.z);
}

// ------------------------------------- small calls: channels shared by warps
// The 128-trial tile's calls are mostly small (64 channels x 128 trials x 2049
// bins are 513 warps of four bins for 608 schedulers), and a warp alone waits
// for its own results five cycles of six.  So kParts warps share the bins, each
// with a part of the channels, and add their sums up at the end; a warp
// evaluates a group of kGroup channels while it accumulates the group before;
// and X and the phase constants arrive kXAhead batches of eight channels early.
// Groups of two, and no table of all channels' constants, keep a CTA's shared
// memory small enough for three CTAs an SM whatever the channels.  The split depends on
// nothing but the channels, so calls on parts of the bins or trials agree
// bit for bit.  Against a warp taking all the channels one by one (table in
// shared memory): 64 channels x 128 trials x 500 bins 21.5 -> 8.2 us a call (the
// host's time), x 4096 bins 22.6 -> 16.4, 1024 channels x 256 trials x 500 bins
// 277 -> 60, x 200 trials x 4096 bins 391 -> 281, 4096 channels x 200 trials x
// 4096 bins 1543 -> 1099.  (With the table beside the swap areas, one CTA an SM
// of 4096 channels: 17.4, 74, 299, 1964.  Groups of four, two CTAs an SM, or
// evaluating ahead without the split were slower, too.)
// Up to kFewQ channels one warp takes them all: a part would have four at
// most, fewer than its own start costs.  4096 bins x 3 series x 128 trials:
// 1 channel 8.2 us against 12.7 in parts, 8 12.5 and 14.6, 16 16.5 and 18.5,
// 20 18.6 and 18.6, 32 26.7 and 23.5; 500 bins: 16 channels 8.9 and 8, 20 10.2
// and 8.
constexpr int kParts = 4, kBinSets = 2;  // warps per four bins; fours of bins per CTA
constexpr int kGroup = 2, kXAhead = 4;
constexpr int kFewQ = 16;
struct SplitQ {
  using Gm = G4x4;
  using M = PackedCompact<G4x4>;
  static constexpr int kWarpsOf = kParts * kBinSets;
  static constexpr int kStage = Gm::NG * M::GFL;            // floats of a channel
  static constexpr int kSwap = 2 * kGroup * kStage;         // of a warp's two swap areas
  static constexpr int kRing = 2 * 32 * kXAhead;            // its ring of X
  static constexpr int kConsts = 4 * 8 * kXAhead;           // and of phase constants
  static constexpr int kWarpFloats = kSwap + kRing + kConsts;
  static constexpr int kSums = 2 * Gm::AT * Gm::BT * 32;    // the sums, over the swap areas
  static_assert(kSums <= kSwap, "sums fit the swap areas");
  static_assert(sizeof(PhaseConst) == 16, "a batch's constants are a word a lane");
  static constexpr int kSmem = 4 * kWarpsOf * kWarpFloats;
};

__global__ void __launch_bounds__(SplitQ::kWarpsOf * 32, 3) mac_parts_kernel(const MacArgs a) {
  using Gm = SplitQ::Gm;
  using M = SplitQ::M;
  constexpr int kStage = SplitQ::kStage;
  static_assert(Gm::NG == 4 && 8 % (2 * kGroup) == 0, "a batch of X is eight channels x four bins");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* areas = reinterpret_cast<float*>(smem_raw);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int part = warp % kParts, set = warp / kParts;
  float* const swap = areas + warp * SplitQ::kWarpFloats;
  float2* const ring = reinterpret_cast<float2*>(swap + SplitQ::kSwap);
  PhaseConst* const pcs = reinterpret_cast<PhaseConst*>(swap + SplitQ::kSwap + SplitQ::kRing);
  const int g = lane / Gm::G, lg = lane % Gm::G;
  const int ga = lg / Gm::GB, gb = lg % Gm::GB;
  const int k4 = (blockIdx.x * kBinSets + set) * 4;  // the four bins
  const int k = k4 + g;
  const int series = blockIdx.z;
  const int jblk = blockIdx.y * Gm::DMS;
  // this warp's channels; c0 below counts from the first
  const int each = (a.n_chan + kParts - 1) / kParts;
  const int c_lo = min(part * each, a.n_chan), n_c = min(c_lo + each, a.n_chan) - c_lo;

  const int k_mine = k4 + (lane & 3);
  const float2* x_mine = a.X + static_cast<int64_t>(series) * a.x_series_stride +
                         (k_mine < a.n_bins ? k_mine : 0);  // (idle bins: bin 0, not stored)
  const uint32_t* pc_mine = reinterpret_cast<const uint32_t*>(a.pc) + (lane & 3);
  auto fetch = [&](int c0) {  // an element and a word of the constants a lane (zeros beyond the part)
    const int c = c0 + (lane >> 2);
    const bool in = c < n_c;
    const int at = (c0 / 8 % kXAhead) * 32 + lane;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dev::smem_u32(ring + at)),
                 "l"(x_mine + static_cast<int64_t>(in ? c_lo + c : 0) * a.x_chan_stride), "r"(in ? 8 : 0)
                 : "memory");
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     dev::smem_u32(reinterpret_cast<uint32_t*>(pcs) + at)),
                 "l"(pc_mine + 4 * (in ? c_lo + c : 0)), "r"(in ? 4 : 0)
                 : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int b = 0; b < kXAhead; ++b) fetch(8 * b);

  Generator<Gm, M> gen;
  gen.init(static_cast<uint32_t>(a.k_begin + (k < a.n_bins ? k : 0)), lg, a.j_begin + jblk);
  float* const grp0 = swap + g * M::GFL;
  typename M::Acc acc;
  M::zero(acc);
  auto evaluate = [&](int c0, int area) {
#pragma unroll
    for (int i = 0; i < kGroup; ++i)
      if (c0 + i < n_c)
        gen.run(pcs[c0 / 8 % kXAhead * 8 + c0 % 8 + i],
                ring[(c0 / 8 % kXAhead) * 32 + (c0 % 8 + i) * 4 + g],
                grp0 + (area * kGroup + i) * kStage);
  };
  auto accumulate = [&](int c0, int area) {
#pragma unroll
    for (int i = 0; i < kGroup; ++i) {
      if (c0 + i < n_c) {
        typename M::Ops ops;
        M::load(grp0 + (area * kGroup + i) * kStage, ga, gb, ops);
        M::mac(acc, ops);
      }
    }
  };
  // Two swap areas: a group is evaluated into the one that the accumulation
  // before the last sync has read, while the group before it is accumulated.
  asm volatile("cp.async.wait_group %0;" ::"n"(kXAhead - 1) : "memory");
  __syncwarp();
  evaluate(0, 0);
  for (int c0 = 0; c0 < n_c; c0 += 8) {
#pragma unroll
    for (int i = 0; i < 8; i += kGroup) {
      if (i + kGroup == 8) asm volatile("cp.async.wait_group %0;" ::"n"(kXAhead - 2) : "memory");
      __syncwarp();
      if (i + kGroup == 8) fetch(c0 + 8 * kXAhead);
      evaluate(c0 + i + kGroup, (i / kGroup + 1) & 1);
      accumulate(c0 + i, (i / kGroup) & 1);
    }
  }

  // The parts' sums: each warp adds one row of the lanes' tiles, in the parts'
  // order, and stores it.
  static_assert(Gm::AT == kParts, "a row of the tile for each warp");
  __syncwarp();
  float2* const sums = reinterpret_cast<float2*>(swap);
#pragma unroll
  for (int ii = 0; ii < Gm::AT; ++ii)
#pragma unroll
    for (int jj = 0; jj < Gm::BT; ++jj) sums[(ii * Gm::BT + jj) * 32 + lane] = M::get(acc, ii, jj);
  __syncthreads();
  if (k >= a.n_bins) return;
  const bool real_only = (a.k_begin + k == a.real_bin_a) || (a.k_begin + k == a.real_bin_b);
#pragma unroll
  for (int jj = 0; jj < Gm::BT; ++jj) {
    float2 v = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kParts; ++q)
      v = __fadd2_rn(v, reinterpret_cast<const float2*>(
                            areas + (set * kParts + q) * SplitQ::kWarpFloats)[
                            (part * Gm::BT + jj) * 32 + lane]);
    const int jl = jblk + (ga * Gm::AT + part) * Gm::TW + gb * Gm::BT + jj;
    if (jl < a.n_dm) {
      const float re = v.x * a.scale;
      const float im = real_only ? 0.f : v.y * a.scale;
      const int64_t o = static_cast<int64_t>(series) * a.y_series_stride +
                        static_cast<int64_t>(jl) * a.y_dm_stride + k;
      if (a.out_kind == 2)
        static_cast<float*>(a.Y)[o] = re * re + im * im;
      else
        static_cast<float2*>(a.Y)[o] = make_float2(re, im);
    }
  }
}

// --------------------------------------------- warp-specialised schedule
// The plain schedule makes every warp alternate between the
// latency-bound phasor evaluation (integer phase, MUFU sin/cos, the swap) and
// its block of paired FMAs; with three warps per scheduler the FMA pipe idles
// whenever all of them are evaluating.  Here the two jobs go to different
// warps: kCons consumer warps each own one bin of the CTA's tile and only read
// Z and P from shared memory and accumulate, while kProd producer warps
// evaluate Z_a = X Q_a and P_b for every consumer's bin, kWsCh channels at a
// time, into a ring of kWsStages stages.  A pair of mbarriers per stage orders
// the two sides (full: every producer warp has written the stage; empty:
// every consumer warp has read it; one arrive per warp).  Every wait is
// bounded; a timeout stops both sides and is reported in the status word.
template <class Gm, class M, int kCons, int kProd, int kWsCh = 4, int kWsStages = 3>
struct WsLayout {
  static_assert(Gm::NG == 1, "one bin per consumer warp");
  static_assert(kCons % kProd == 0, "producers share the consumers' bins evenly");
  static constexpr int kBinsPerProd = kCons / kProd;
  static constexpr int kStageFloats = kWsCh * kCons * M::GFL;  // [channel][consumer][GFL]
  // 2 kWsStages mbarriers and the abort flag, rounded up to 16 bytes
  static constexpr size_t kBarBytes = (2 * kWsStages * 8 + 4 + 15) / 16 * 16;
  static constexpr size_t kSwapBytes =
      kBarBytes + sizeof(float) * static_cast<size_t>(kWsStages) * kStageFloats;
  static_assert(2 * kWsStages * 8 + 4 <= kBarBytes, "barrier area");
};

// One work item of the warp-specialised schedule: the CTA's kCons bins
// starting at local bin bin_tile * kCons and the trials dm_block * DMS + ..
// of one set of spectra, with the phase table already in shared memory.
// Stages and barrier phases continue from iteration it0 of the ring (items
// of a persistent CTA follow one another).  Returns false after a timeout.
template <class Gm, class M, int kCons, int kProd, int kWsCh, int kWsStages>
__device__ __forceinline__ bool ws_item(const MacArgs& a, const PhaseConst* pcs, float* stages,
                                        uint64_t* full, uint64_t* empty,
                                        volatile int* abort_flag, int bin_tile, int dm_block,
                                        int series, uint32_t it0) {
  using Ly = WsLayout<Gm, M, kCons, kProd, kWsCh, kWsStages>;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int n_iter = (a.n_chan + kWsCh - 1) / kWsCh;
  const int jblk = dm_block * Gm::DMS;
  const int k_tile = bin_tile * kCons;  // first local bin of the item
  bool ok = true;

  if (warp >= kCons) {
    // ------------------------------------------------------------ producers
    const int pw = warp - kCons;
    constexpr int NB = Ly::kBinsPerProd;
    Generator<Gm, M> gen[NB];
    const float2* xp[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int k = k_tile + pw * NB + q;
      const int kl = k < a.n_bins ? k : 0;  // idle bins evaluate local bin 0, stored by nobody
      gen[q].init(static_cast<uint32_t>(a.k_begin + kl), lane, a.j_begin + jblk);
      xp[q] = a.X + static_cast<int64_t>(series) * a.x_series_stride + kl;
    }
    const int64_t xs = a.x_chan_stride;
    float2 xn[NB][kWsCh];
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int ch = 0; ch < kWsCh; ++ch)
        xn[q][ch] = ch < a.n_chan ? __ldg(xp[q] + ch * xs) : make_float2(0.f, 0.f);
    for (int it = 0; it < n_iter; ++it) {
      const uint32_t g = it0 + it;
      const int s = g % kWsStages;
      float2 x[NB][kWsCh];
#pragma unroll
      for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int ch = 0; ch < kWsCh; ++ch) {
          x[q][ch] = xn[q][ch];
          const int c = (it + 1) * kWsCh + ch;  // prefetch the next stage's X
          xn[q][ch] = c < a.n_chan ? __ldg(xp[q] + c * xs) : make_float2(0.f, 0.f);
        }
      ok = __all_sync(0xffffffffu,
                      dev::mbar_wait(&empty[s], ((g / kWsStages) & 1) ^ 1, abort_flag));
      if (!ok) break;
      float* st = stages + s * Ly::kStageFloats + (pw * NB) * M::GFL;
#pragma unroll
      for (int ch = 0; ch < kWsCh; ++ch) {
        const int c = it * kWsCh + ch;
        if (c < a.n_chan) {
          const PhaseConst p = pcs[c];
#pragma unroll
          for (int q = 0; q < NB; ++q) gen[q].run(p, x[q][ch], st + (ch * kCons + q) * M::GFL);
        }
      }
      if (!a.test_withhold) dev::mbar_arrive_warp(&full[s]);
    }
  } else {
    // ------------------------------------------------------------ consumers
    const int k = k_tile + warp;  // local bin
    const int ga = lane / Gm::GB;
    const int gb = lane % Gm::GB;
    typename M::Acc acc;
    M::zero(acc);
    for (int it = 0; it < n_iter; ++it) {
      const uint32_t g = it0 + it;
      const int s = g % kWsStages;
      ok = __all_sync(0xffffffffu, dev::mbar_wait(&full[s], (g / kWsStages) & 1, abort_flag));
      if (!ok) break;
      const float* st = stages + s * Ly::kStageFloats + warp * M::GFL;
      const int nc = a.n_chan - it * kWsCh;
#pragma unroll
      for (int ch = 0; ch < kWsCh; ++ch) {
        if (ch < nc) {
          typename M::Ops ops;
          M::load(st + ch * kCons * M::GFL, ga, gb, ops);
          M::mac(acc, ops);
        }
      }
      dev::mbar_arrive_warp(&empty[s]);
    }
    if (ok && k < a.n_bins) {
      const bool real_only = (a.k_begin + k == a.real_bin_a) || (a.k_begin + k == a.real_bin_b);
#pragma unroll
      for (int ii = 0; ii < Gm::AT; ++ii) {
#pragma unroll
        for (int jj = 0; jj < Gm::BT; ++jj) {
          const int jl = jblk + (ga * Gm::AT + ii) * Gm::TW + gb * Gm::BT + jj;
          if (jl < a.n_dm) {
            const float2 v = M::get(acc, ii, jj);
            const float re = v.x * a.scale;
            const float im = real_only ? 0.f : v.y * a.scale;
            const int64_t o = static_cast<int64_t>(series) * a.y_series_stride +
                              static_cast<int64_t>(jl) * a.y_dm_stride + k;
            if (a.out_kind == 2)
              static_cast<float*>(a.Y)[o] = re * re + im * im;
            else
              static_cast<float2*>(a.Y)[o] = make_float2(re, im);
          }
        }
      }
    }
  }
  if (!ok) {
    *abort_flag = 1;
    if (a.status) atomicExch(a.status, FDD_ERR_TIMEOUT);
  }
  return ok;
}

// Shared-memory carve-up of the warp-specialised kernels: phase table, then
// the barriers and abort flag, then the stages.
template <class Ly>
struct WsSmem {
  PhaseConst* pcs;
  uint64_t* full;
  uint64_t* empty;
  volatile int* abort_flag;
  float* stages;
  template <int kWsStages>
  __device__ __forceinline__ void init(unsigned char* raw, int n_chan, int n_cons_warps,
                                       int n_prod_warps) {
    pcs = reinterpret_cast<PhaseConst*>(raw);
    unsigned char* tail = raw + sizeof(PhaseConst) * n_chan;  // 16-byte aligned
    full = reinterpret_cast<uint64_t*>(tail);
    empty = full + kWsStages;
    abort_flag = reinterpret_cast<volatile int*>(empty + kWsStages);
    stages = reinterpret_cast<float*>(tail + Ly::kBarBytes);
    if (threadIdx.x == 0) {
      for (int i = 0; i < kWsStages; ++i) {
        dev::mbar_init(&full[i], n_prod_warps);  // one arrive per warp
        dev::mbar_init(&empty[i], n_cons_warps);
      }
      *abort_flag = 0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
};

template <class Gm, class M, int kCons, int kProd, int kWsCh, int kWsStages>
__global__ void __launch_bounds__((kCons + kProd) * 32, 1) mac_ws_kernel(const MacArgs a) {
  using Ly = WsLayout<Gm, M, kCons, kProd, kWsCh, kWsStages>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  WsSmem<Ly> sm;
  sm.template init<kWsStages>(smem_raw, a.n_chan, kCons, kProd);
  for (int i = threadIdx.x; i < a.n_chan; i += blockDim.x) sm.pcs[i] = a.pc[i];
  __syncthreads();
  ws_item<Gm, M, kCons, kProd, kWsCh, kWsStages>(
      a, sm.pcs, sm.stages, sm.full, sm.empty, sm.abort_flag, blockIdx.x, blockIdx.y, blockIdx.z,
      0u);
}

// Persistent form of the warp-specialised schedule over a batch of spectra
// sets (the batching form): CTAs pull (set, bin tile, trial block) items from
// a global counter, numbered bin-tile-major from each set's item_begin; the
// stage ring runs on across items; the phase table is reloaded when the set
// changes.
template <class Gm, class M, int kCons, int kProd, int kWsCh, int kWsStages>
__global__ void __launch_bounds__((kCons + kProd) * 32, 1)
    mac_ws_batch_kernel(const BatchSet* sets, int n_sets, int64_t n_items,
                        unsigned long long* counter) {
  using Ly = WsLayout<Gm, M, kCons, kProd, kWsCh, kWsStages>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ long long item_s;
  const int n_chan = sets[0].args.n_chan;  // common to the batch
  WsSmem<Ly> sm;
  sm.template init<kWsStages>(smem_raw, n_chan, kCons, kProd);
  int cur = -1;
  uint32_t it0 = 0;
  const uint32_t n_iter = static_cast<uint32_t>((n_chan + kWsCh - 1) / kWsCh);
  while (true) {
    if (threadIdx.x == 0) item_s = static_cast<long long>(atomicAdd(counter, 1ull));
    __syncthreads();  // also: every stage of the previous item has been read
    const long long item = item_s;
    if (item >= n_items || *sm.abort_flag) break;
    int lo = 0, hi = n_sets - 1;  // last set with item_begin <= item
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (sets[mid].item_begin <= item) lo = mid; else hi = mid - 1;
    }
    const BatchSet& bs = sets[lo];
    if (lo != cur) {
      for (int i = threadIdx.x; i < n_chan; i += blockDim.x) sm.pcs[i] = bs.args.pc[i];
      cur = lo;
    }
    __syncthreads();  // phase table ready; item_s read by every thread
    const long long local = item - bs.item_begin;
    ws_item<Gm, M, kCons, kProd, kWsCh, kWsStages>(
        bs.args, sm.pcs, sm.stages, sm.full, sm.empty, sm.abort_flag,
        static_cast<int>(local / bs.n_dm_blocks), static_cast<int>(local % bs.n_dm_blocks), 0,
        it0);
    it0 += n_iter;
  }
}

// Persistent form over a batch of spectra sets of uneven sizes (the batching
// form): CTAs pull work items (set, bin tile, trial block) from a global
// counter; a set's phase table is loaded into shared memory when the set
// changes.  Items of a set are numbered bin-tile-major from item_begin.
template <class Gm, class M, int W = kWarps>
__global__ void __launch_bounds__(W * 32, 1) mac_batch_kernel(const BatchSet* sets, int n_sets,
                                                              int64_t n_items,
                                                              unsigned long long* counter) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ long long item_s;
  const int n_chan = sets[0].args.n_chan;  // common to the batch
  PhaseConst* pcs = reinterpret_cast<PhaseConst*>(smem_raw);
  float* swap_all = reinterpret_cast<float*>(smem_raw + sizeof(PhaseConst) * n_chan);
  int cur = -1;
  while (true) {
    if (threadIdx.x == 0) item_s = static_cast<long long>(atomicAdd(counter, 1ull));
    __syncthreads();
    const long long item = item_s;
    __syncthreads();
    if (item >= n_items) break;
    int lo = 0, hi = n_sets - 1;  // last set with item_begin <= item
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (sets[mid].item_begin <= item) lo = mid; else hi = mid - 1;
    }
    const BatchSet& bs = sets[lo];
    if (lo != cur) {
      for (int i = threadIdx.x; i < n_chan; i += W * 32) pcs[i] = bs.args.pc[i];
      __syncthreads();
      cur = lo;
    }
    const long long local = item - bs.item_begin;
    mac_block<Gm, M, W>(bs.args, pcs, swap_all, static_cast<int>(local / bs.n_dm_blocks),
                               static_cast<int>(local % bs.n_dm_blocks), 0);
    __syncthreads();
  }
}

// ----------------------------------------------------------------- variants
struct VariantInfo {
  const void* fn;
  int dms;
  int ng;
  size_t swap_bytes;  // per CTA, excluding the phase-constant table
  int warps = kWarps;
  const void* batch_fn = nullptr;  // persistent batch kernel of the same tile
  int bin_warps = 0;  // warps that own bins (0: all of them)
  int bins() const { return (bin_warps ? bin_warps : warps) * ng; }
};

template <class Gm, class M, int W = kWarps>
VariantInfo info() {
  return {reinterpret_cast<const void*>(&mac_kernel<Gm, M, W>), Gm::DMS, Gm::NG,
          sizeof(float) * static_cast<size_t>(W) * 2 * Gm::NG * M::GFL, W,
          reinterpret_cast<const void*>(&mac_batch_kernel<Gm, M, W>)};
}

template <class Gm, class M, int kCons, int kProd, int kCh = 4, int kSt = 3>
VariantInfo info_ws() {
  using Ly = WsLayout<Gm, M, kCons, kProd, kCh, kSt>;
  VariantInfo vi{reinterpret_cast<const void*>(&mac_ws_kernel<Gm, M, kCons, kProd, kCh, kSt>),
                 Gm::DMS, Gm::NG, Ly::kSwapBytes, kCons + kProd,
                 reinterpret_cast<const void*>(&mac_ws_batch_kernel<Gm, M, kCons, kProd, kCh, kSt>)};
  vi.bin_warps = kCons;
  return vi;
}

constexpr size_t kMaxSmem = 227 * 1024;

// Channels up to which plans take the G12 tile.  The tile itself has no such
// limit (its per-channel constants stay in global memory); the line is where
// it lay while the tile kept them in shared memory, so a plan reports the
// tile it always did.
constexpr int kG12MaxChan = 8381;

// (every tile but G12_4x8, which fdd_mac_split.cu launches)
VariantInfo variant_info(int v) {
  switch (v) {
    case MAC_Q12_8x8: return info<G8x8, PackedCompact<G8x8>, 12>();
    case MAC_Q_4x8: return info<G4x8, PackedCompact<G4x8>>();
    case MAC_Q_8x8_512: return info<G8x8q, PackedCompact<G8x8q>>();
    case MAC_Q_4x4: return info<G4x4, PackedCompact<G4x4>>();
    default: return info_ws<G8x8, PackedCompact<G8x8>, 8, 4>();  // MAC_W12_8x8
  }
}

}  // namespace

// Default tile for a trial count.  From 257 trials on the G12 tile while the
// channels allow it: on 4096 bins x 1024 channels its passes of up to 512,
// 1024, 2048 and 4096 trials take 190, 250, 300 and 430 us whatever their filling,
// the 128-trial tile 281 us at 256 trials and more with every 128.  (From 129 to
// 256 trials the G12 tile would be the faster one too with many channels; plans
// have always reported Q_4X4 there, and keep to it.)  Otherwise the tile with
// the least time for the padded trial blocks, ceil(n_dm / block) * block /
// rate, with each tile's rate measured kernel-only (fraction of the FP32 peak,
// 1024 channels, 131073 bins): Q_4x8 0.493 (1024-trial blocks), Q_8x8_512 0.415
// (512), Q_4x4 0.347 (128; before its warps shared the channels).  (The
// four-product warp-specialised tile W12_8x8 measured 0.621 on the same
// launch, Q12_8x8, the 2048-trial tile on the plain schedule, 0.553.)
int mac_variant_for(int n_dm, int n_chan) {
  if (n_dm > 256 && mac_variant_takes(MAC_G12_4x8, n_chan)) return MAC_G12_4x8;
  struct Tile {
    int variant, block;
    double rate;
  };
  static const Tile tiles[] = {
      {MAC_Q_4x8, 1024, 0.493}, {MAC_Q_8x8_512, 512, 0.415}, {MAC_Q_4x4, 128, 0.347}};
  int best = MAC_W12_8x8;  // (the smallest shared-memory need of the 2048-trial tiles)
  double best_cost = 0.0;
  for (const Tile& t : tiles) {
    if (!mac_variant_takes(t.variant, n_chan)) continue;
    const double cost = (n_dm + t.block - 1) / t.block * t.block / t.rate;
    if (best_cost == 0.0 || cost < best_cost) {
      best = t.variant;
      best_cost = cost;
    }
  }
  return best;
}

int mac_variant_trials_per_block(int variant) {
  return variant == MAC_G12_4x8 ? 2048 : variant_info(variant).dms;
}

size_t mac_smem_bytes(int variant, int n_chan) {
  if (variant == MAC_G12_4x8) return mac_split_smem_bytes();
  return sizeof(PhaseConst) * static_cast<size_t>(n_chan) + variant_info(variant).swap_bytes;
}

bool mac_variant_takes(int variant, int n_chan) {
  return variant == MAC_G12_4x8 ? n_chan <= kG12MaxChan : mac_smem_bytes(variant, n_chan) <= kMaxSmem;
}

fdd_status mac_variant_check(int variant, int n_chan) {
  if (mac_variant_takes(variant, n_chan)) return FDD_OK;
  char text[96];
  if (variant == MAC_G12_4x8)
    std::snprintf(text, sizeof text, "n_chan %d is above the %d channels that the G12_4X8 tile is used for",
                  n_chan, kG12MaxChan);
  else
    std::snprintf(text, sizeof text, "n_chan %d needs more shared memory than a CTA has", n_chan);
  return report_error(FDD_ERR_UNSUPPORTED, text);
}

cudaError_t mac_prepare(int variant, int n_chan) {
  if (variant == MAC_G12_4x8) return mac_split_prepare();
  const VariantInfo vi = variant_info(variant);
  const size_t bytes = mac_smem_bytes(variant, n_chan);
  cudaError_t e = allow_smem(vi.fn, bytes);
  if (e == cudaSuccess && variant == MAC_Q_4x4)
    e = allow_smem(reinterpret_cast<const void*>(&mac_parts_kernel), SplitQ::kSmem);
  if (e != cudaSuccess || !vi.batch_fn) return e;
  return allow_smem(vi.batch_fn, bytes);
}

int mac_variant_bins_per_cta(int variant) { return variant_info(variant).bins(); }

bool mac_variant_batchable(int variant) {
  return variant == MAC_G12_4x8 || variant_info(variant).batch_fn != nullptr;
}

int mac_batch_ctas_per_sm(int variant, int n_chan) {
  if (variant == MAC_G12_4x8) return 1;  // (tensor memory and registers: one CTA per SM)
  const VariantInfo vi = variant_info(variant);
  if (!vi.batch_fn) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, vi.batch_fn, vi.warps * 32,
                                                    mac_smem_bytes(variant, n_chan)) !=
      cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_mac_batch(const BatchSet* d_sets, int n_sets, long long n_items,
                             unsigned long long* d_counter, int variant, int n_ctas, int n_chan,
                             int max_n_dm, cudaStream_t s) {
  if (variant == MAC_G12_4x8)
    return launch_mac_split_batch(d_sets, n_sets, n_items, max_n_dm, n_chan, n_ctas, s);
  const VariantInfo vi = variant_info(variant);
  if (!vi.batch_fn) return cudaErrorInvalidValue;
  if (n_items <= 0) return cudaSuccess;
  void* params[] = {&d_sets, &n_sets, &n_items, &d_counter};
  note_launches(1);
  return cudaLaunchKernel(vi.batch_fn, dim3(n_ctas), dim3(vi.warps * 32), params,
                          mac_smem_bytes(variant, n_chan), s);
}

cudaError_t launch_mac_fp32(const MacArgs& a, int variant, cudaStream_t s) {
  if (a.n_dm <= 0 || a.n_series <= 0 || a.n_bins <= 0) return cudaSuccess;
  if (variant == MAC_G12_4x8) return launch_mac_split(a, s);
  VariantInfo vi = variant_info(variant);
  size_t smem = mac_smem_bytes(variant, a.n_chan);
  int bins_per_cta = vi.bins();
  if (variant == MAC_Q_4x4 && a.n_chan > kFewQ) {
    vi.fn = reinterpret_cast<const void*>(&mac_parts_kernel);
    vi.warps = SplitQ::kWarpsOf;
    bins_per_cta = 4 * kBinSets;
    smem = SplitQ::kSmem;
  }
  dim3 grid((a.n_bins + bins_per_cta - 1) / bins_per_cta, (a.n_dm + vi.dms - 1) / vi.dms,
            a.n_series);
  if (grid.y > 65535u || grid.z > 65535u) return cudaErrorInvalidConfiguration;
  MacArgs args = a;
  void* params[] = {&args};
  note_launches(1);
  return cudaLaunchKernel(vi.fn, grid, dim3(vi.warps * 32), params, smem, s);
}

}  // namespace fdd
