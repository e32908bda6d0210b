// fdd_mac_split.cu -- FP32-accurate phase-rotate-and-sum on the tensor cores
// (Sect. 2.2, Eqs. 4 and 7) for one set of spectra: the G12_4X8 tile.
//
//   Y[j][k] = sum_nu W(k, nu, j) X[nu][k],   W = exp(+2 pi i k d(nu, DM_j) / L)
//
// Trials are paired around the centre of their block of at most 2048 (counted
// from the first trial of the call, so that calls on parts made of whole blocks
// agree with a whole call bit for bit).  A block of 256 n_a trials from j_b has
// the centre Jc = j_b + 128 n_a - 1/2 and the trials j = Jc + s (128 al + 64) +
// t (b + 1/2) for s, t = +-1, al < n_a, b < 64.  The phase is linear in j, so
//
//   W = exp(i phi_c) (Ca + i s Sa) (Cb + i t Sb),
//
// with (Ca, Sa) and (Cb, Sb) the cosine and sine of the al and b steps of bin
// k and channel nu.  The sums over channels that all four signs share,
//
//   M = sum Cb {Xr Ca, Xi Ca, Xr Sa, Xi Sa},   N = sum Sb {the same},
//
// (X rotated by exp(i phi_c)) are ONE real matrix product per bin: 128 rows
// (Cb, Sb of 64 b's) x channels times channels x 4 n_a columns, of one block or
// of two that share the rows.  Against the
// complex form this halves both the multiplications (eight real ones for four
// trials' complex products) and the phasors to evaluate (64 for 128 trials).
//
// Each operand is split into two FP16 terms (hi + lo: 22 bits; the columns
// scaled by a power of two per bin and stage of 64 channels) and the product
// formed as hi hi + (hi lo + lo hi) on tcgen05 with FP32 accumulators.  The
// tensor cores round their sums toward zero, so an accumulator only lives for
// one stage; the stages' sums are added in FP32 registers (to nearest).  The
// error of the spectra against FP64 is 2.4e-7 of the result at 64 channels and
// 2.5e-7 at 256 (rows from the hardware sine, columns from a series), 3.4e-7 from 257
// to 512, 3.5e-7 at 1024 and 2048 (both from the hardware sine); the FP32
// multiply-adds this replaces rounded every sum: 3.1e-7 at 64 channels, 4.5e-7
// at 256, 7.7e-7 at 1024, 1.1e-6 at 2048.
//
// Sixty-four channels of a bin are a stage.  Two warps turn the spectra and
// phase constants into a table per stage, thirteen evaluate and split rows and
// columns into shared memory (K-major core matrices), one issues the MMAs,
// four add the stages up and store.  4096 bins x 1024 channels x 2048 trials
// take 300 us, against 1185 us for the FP32 multiply-adds (three real products
// per complex one) at 0.75 of the FP32 peak; 301 bins x 4096 channels x 8192
// trials 212 against 1292 us; 701 trials of 2 x 387 channels 151 against 560 us.
// What bounds it (two series of 2048 trials a pass): writing and reading the
// operands in shared memory (82 % of its cycles, 24 of them the MMAs' reads)
// beside 65 warp instructions per bin and channel (55 % of the issue slots),
// most of them phasors and splits of the 128 rows.  Hence the wide passes: the rows
// serve all columns of a pass, up to 4096 trials of one series.  Several series
// share them too (two, or four up to 1024 trials), each with its own columns
// and scales and the bits it has alone: 4096 (bin, series) x 1024 channels of
// 2048 trials take 300 us each alone and 227 in twos; of 1024 trials 256, 160
// in twos and 130 in fours.  Plans of up to 512 trials fill no wide pass; they
// halve the rows instead, and a stage takes two bins (190 us for 4096 bins x
// 1024 channels x 512 trials, 249 with rows for twice the trials).
// The four adding warps do not take stages while they store an item, so that
// must be short: Cb and Sb of a b are rows of one warp, which exchanges them
// by shuffles (through shared memory and barriers of the four warps: 311 us
// for the first figure, 218, 167, and 267 for two series).
// Measured and dropped: results kept until a whole octet is done in wider
// stores with fewer warps (16 warps of 128 registers: 344 us), four bytes per
// store from registers used at once (317), one octet per task (353), the MMA
// loop unrolled by stage (334: instruction fetch), lo hi as an MMA of its own
// (307), four more warps to store, with the producers at 80 registers (335).
#include <atomic>
#include <climits>

#include <cuda_fp16.h>

#include "fdd_device.cuh"
#include "fdd_internal.h"

namespace fdd {
namespace {

using dev::mbar_arrive;
using dev::mbar_arrive_warp;
using dev::mbar_init;
using dev::smem_u32;
using dev::unit_phasor;

// The warp waits for a phase, bounded: every lane asks (together: a divided
// warp would run what follows twice), suspended in the hardware for up to two
// microseconds at a time, so that waiting takes few shared-memory cycles from
// the operands.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  long long t0 = 0;
  while (true) {
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
                 " selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity), "r"(2000)
                 : "memory");
    if (__all_sync(0xffffffffu, ok)) return true;
    const long long t = clock64();
    if (t0 == 0) t0 = t;
    if (__any_sync(0xffffffffu, *abort_flag != 0 || t - t0 > dev::kWaitCycles)) return false;
  }
}

constexpr int kCh = 64;     // channels per stage (four K steps of 16)
constexpr int kRows = 128;  // Cb, Sb of 64 b's: sixteen b's Cb, then their Sb, and so on
// Up to this many channels the columns' phasors come from the Taylor series,
// too: over so few the FP32 multiply-adds' sums lost little, and the product with
// the hardware's columns would lose more.  Error of the power against FP64,
// FP32 multiply-adds, hardware's columns, series: 64 channels 4.2, 5.0 and
// 3.5e-7, 128 4.8, 5.1 and 3.7, 200 5.3, 5.2 and 3.7, 256 5.7, 5.3 and 3.7, 512
// 7.2, 5.3 and 3.8 (of the spectra the hardware's columns lose more up to some
// 80 channels).  The series costs (911 trials x 1829 bins) nothing at 64 and 128
// channels, 42.0 against 41.0 us at 200, 44.8 against 43.1 at 256, 78.3 against
// 76.6 at 512; the line is the next whole stage above 200.
constexpr int kFewChan = 256;
constexpr int kPairTrials = 256;  // trials per al: s, t = +-1, 64 b's (twin: half)
constexpr int kBlockAls = 8;      // al's of a whole block (2048 trials)

// Warps: 0-3 epilogue (a warp reads the tensor-memory lanes of its quarter),
// the MMA issuer, two that make the stages' tables in turn, and thirteen
// producers of rows and columns: five warps per scheduler, 96 registers each.
constexpr int kEpiWarps = 4;
constexpr int kMmaWarp = kEpiWarps;
constexpr int kPrepFirst = kMmaWarp + 1, kPrepWarps = 2;
constexpr int kProdFirst = kPrepFirst + kPrepWarps, kProdWarps = 13;
constexpr int kThreads = 32 * (kProdFirst + kProdWarps);

// A pass's columns are kBlocks blocks of kAls al's that share its rows: blocks
// of trials of one series (each with its own centre), or the same trials of
// kBlocks series (kSeries).  kNa: al's in all; kBins: bins a CTA works on at a
// time (their accumulators share the epilogue's registers: kNa * kBins = 16).
// For few trials the rows, too, are shared out (kTwin): a stage takes two bins
// (the blocks), rows of 32 b's of each, and the epilogue the quarter of the
// product that has rows and columns of the same bin.
template <int kAls_, int kBlocks_, bool kSeries_, bool kTwin_ = false>
struct Cfg {
  static constexpr int kAls = kAls_, kBlocks = kBlocks_, kNa = kAls * kBlocks;
  static constexpr bool kSeries = kSeries_, kTwin = kTwin_;
  static constexpr int kSeriesSets = kSeries ? kBlocks : 1;       // series of a pass
  static constexpr int kSets = kSeries || kTwin ? kBlocks : 1;    // (series, bin)s of a stage
  static constexpr int kRowBins = kTwin ? 2 : 1;                  // bins of a stage
  static constexpr int kCentres = kSeries || kTwin ? 1 : kBlocks; // centres of a pass
  static constexpr int kCentrePhases = kTwin ? 2 : kCentres;      // of a stage
  static constexpr int kAlTrials = kPairTrials / kRowBins;
  static constexpr int kMostAls = kAls * kCentres;
  static constexpr int kPassTrials = kAlTrials * kMostAls;
  static constexpr int kOwn = kTwin ? kAls : kNa;  // al's a thread of the epilogue adds up
  static constexpr int kBins = 16 / kOwn;          // stages per 64 channels of an item
  static constexpr int kItemBins = kBins * kRowBins;  // stage i: bins i (and kBins + i)
  static constexpr int kN = 4 * kNa;          // columns
  static constexpr int kStages = kNa == 16 ? 4 : 5;
  // (tables run further ahead than operands)
  static constexpr int kTables = 8;
  static constexpr uint32_t kATile = kRows * kCh * 2;  // 16 KB per term
  static constexpr uint32_t kBTile = kN * kCh * 2;
  static constexpr uint32_t kStageBytes = 2 * (kATile + kBTile);
  // tasks of a stage, dealt to the producer warps in turn: the columns (sixteen
  // half octets of channels x kNa al's, two rounds of a warp each), then the
  // rows of each of the four K steps
  static constexpr int kColTasks = kNa / 4;
  static constexpr int kTasks = 4 + kColTasks;
  static_assert((kProdWarps + kTasks - 1) / kTasks < kStages, "a producer's step between tasks");
  // tensor memory: a ring of accumulators, then the sums of the kOutBins
  // bins that are stored together (sixteen (al, bin) units of four a slot; a
  // wide pass of one series stores from registers and keeps the longer ring)
  static constexpr int kSlots = kNa < 16 ? 1 : kSeries ? 2 : 0;
  static constexpr int kOutBins = kSlots > 1 ? kSlots * kBins : kBins;
  static constexpr int kAccs = kSlots > 1 ? 3 : kStages;
  static constexpr uint32_t kPark = kAccs * 2 * kN;
  static_assert(kPark + kSlots * 64 <= 512 && kAccs <= kStages, "tensor memory");
  static constexpr uint32_t kTmemCols = 512;
  static_assert(kSeries || kTwin || kBlocks == 1 || kAls == kBlockAls, "trials in whole blocks");
  static_assert(kAls % 4 == 0, "the epilogue's four al's have one scale");
};

// Per stage: what the producers need of each channel.
template <class C>
struct Table {
  uint32_t hw[C::kRowBins][kCh];   // half the trial step's phase, units of 2^-32 cycle
  uint32_t ha[C::kRowBins][kCh];   // half the step of al's: 64 (32) trial steps
  float fr[C::kRowBins][kCh], fi[C::kRowBins][kCh];  // phasor of 16 trial steps (b -> b + 16)
  float xr[C::kBlocks][kCh], xi[C::kBlocks][kCh];  // X rotated to each block's centre and scaled
  int steps;               // K steps of 16 channels the MMAs read
  int pad[3];
};
template <class C>
struct Smem {
  alignas(128) unsigned char stage[C::kStages][C::kStageBytes];
  alignas(16) Table<C> table[C::kTables];
  float inv[4 * C::kTables][C::kSets];  // undoes a stage's scales (read by the epilogue, well after the table)
  uint64_t pfull[C::kTables], pfree[C::kTables];  // table written; every producer has read it
  uint64_t full[C::kStages], done[C::kStages];   // operands written; MMAs complete
  uint64_t acc_free[C::kAccs];  // accumulators added up
  uint64_t drain;
  uint32_t tmem;
  int abort_flag;
};

// Shared-memory matrix descriptor, K-major without swizzle: 8-row x 16-byte
// core matrices of 128 contiguous bytes, 128 bytes apart along the rows and
// `k_stride` apart along K.
__device__ __forceinline__ uint64_t core_desc(uint32_t addr, uint32_t k_stride) {
  return static_cast<uint64_t>((addr & 0x3FFFF) >> 4) | (static_cast<uint64_t>(k_stride >> 4) << 16) |
         (static_cast<uint64_t>(128 >> 4) << 32) | (static_cast<uint64_t>(1) << 46);
}

// One thread of the (converged) warp, as a value the compiler keeps uniform:
// MMAs issued under it take their descriptors from uniform registers.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(e));
  return e;
}

__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t accum, uint32_t id) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(accum));
}

// Four columns of this warp's 32 lanes from each of four places, waited for:
// one statement, so no use of the values can move before the wait.
__device__ __forceinline__ void tmem_ld4x4(uint32_t t0, uint32_t t1, uint32_t t2, uint32_t t3,
                                           uint32_t (&r)[4][4]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%16];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%17];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8,%9,%10,%11}, [%18];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12,%13,%14,%15}, [%19];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&r"(r[0][0]), "=&r"(r[0][1]), "=&r"(r[0][2]), "=&r"(r[0][3]), "=&r"(r[1][0]),
        "=&r"(r[1][1]), "=&r"(r[1][2]), "=&r"(r[1][3]), "=&r"(r[2][0]), "=&r"(r[2][1]),
        "=&r"(r[2][2]), "=&r"(r[2][3]), "=&r"(r[3][0]), "=&r"(r[3][1]), "=&r"(r[3][2]),
        "=&r"(r[3][3])
      : "r"(t0), "r"(t1), "r"(t2), "r"(t3)
      : "memory");
}

// Sixteen columns of this warp's 32 lanes written; units of four columns read
// from two places, or one to four from one place, and waited for.
__device__ __forceinline__ void tmem_st16(uint32_t t, const float (&v)[4][4]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(t), "f"(v[0][0]), "f"(v[0][1]), "f"(v[0][2]), "f"(v[0][3]), "f"(v[1][0]), "f"(v[1][1]),
      "f"(v[1][2]), "f"(v[1][3]), "f"(v[2][0]), "f"(v[2][1]), "f"(v[2][2]), "f"(v[2][3]),
      "f"(v[3][0]), "f"(v[3][1]), "f"(v[3][2]), "f"(v[3][3])
      : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t t0, uint32_t t1, float (&v)[2][4]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%8];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4,%5,%6,%7}, [%9];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&f"(v[0][0]), "=&f"(v[0][1]), "=&f"(v[0][2]), "=&f"(v[0][3]), "=&f"(v[1][0]),
        "=&f"(v[1][1]), "=&f"(v[1][2]), "=&f"(v[1][3])
      : "r"(t0), "r"(t1)
      : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t t, float (&v)[2][4]) { tmem_ld4(t, t + 4, v); }
__device__ __forceinline__ void tmem_ld4(uint32_t t, float (&v)[4][4]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=&f"(v[0][0]), "=&f"(v[0][1]), "=&f"(v[0][2]), "=&f"(v[0][3]), "=&f"(v[1][0]),
        "=&f"(v[1][1]), "=&f"(v[1][2]), "=&f"(v[1][3]), "=&f"(v[2][0]), "=&f"(v[2][1]),
        "=&f"(v[2][2]), "=&f"(v[2][3]), "=&f"(v[3][0]), "=&f"(v[3][1]), "=&f"(v[3][2]),
        "=&f"(v[3][3])
      : "r"(t)
      : "memory");
}

// v as FP16 hi + lo, both components packed (x in the low half).
__device__ __forceinline__ void split2(float2 v, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(v.x, v.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  float dx, dy;  // hi - v
  asm("sub.rn.f32.f16 %0, %1, %2;" : "=f"(dx) : "h"(__half_as_ushort(__low2half(h))), "f"(v.x));
  asm("sub.rn.f32.f16 %0, %1, %2;" : "=f"(dy) : "h"(__half_as_ushort(__high2half(h))), "f"(v.y));
  const __half2 l = __floats2half2_rn(-dx, -dy);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}

// Cosine and sine of two phases given in units of 2^-32 cycle: the nearest
// quarter cycle taken off exactly in the integers, then the Taylor series to
// x^8 and x^9 on |x| <= pi / 4 (truncation below 3e-8, rounding of the order
// of 2^-24), two phases per instruction.  The stage tables use it: their
// phasors multiply every row and column of a channel, where the hardware
// sine's 2^-21 would be seen twice; and the columns of calls of few channels.
__device__ __forceinline__ void sincos2(uint32_t p0, uint32_t p1, float2& cs, float2& sn) {
  const uint32_t q0 = (p0 + 0x20000000u) >> 30, q1 = (p1 + 0x20000000u) >> 30;
  const float2 r = make_float2(static_cast<float>(static_cast<int>(p0 - (q0 << 30))),
                               static_cast<float>(static_cast<int>(p1 - (q1 << 30))));
  auto two = [](float v) { return make_float2(v, v); };
  const float2 x = __fmul2_rn(r, two(1.46291807926715968e-9f));  // 2 pi / 2^32
  const float2 z = __fmul2_rn(x, x);
  float2 s = __ffma2_rn(z, two(2.7557319e-6f), two(-1.9841270e-4f));
  s = __ffma2_rn(z, s, two(8.3333333e-3f));
  s = __ffma2_rn(z, s, two(-1.6666667e-1f));
  s = __ffma2_rn(__fmul2_rn(x, z), s, x);
  float2 c = __ffma2_rn(z, two(2.4801587e-5f), two(-1.3888889e-3f));
  c = __ffma2_rn(z, c, two(4.1666667e-2f));
  c = __ffma2_rn(z, c, two(-0.5f));
  c = __ffma2_rn(z, c, two(1.0f));
  // (cos, sin)(x + q pi / 2)
  auto turn = [](uint32_t q, float cx, float sx, float& co, float& so) {
    const float a = (q & 1u) ? sx : cx, b = (q & 1u) ? cx : sx;
    co = __uint_as_float(__float_as_uint(a) ^ (((q + 1u) & 2u) << 30));
    so = __uint_as_float(__float_as_uint(b) ^ ((q & 2u) << 30));
  };
  turn(q0, c.x, s.x, cs.x, sn.x);
  turn(q1, c.y, s.y, cs.y, sn.y);
}

// An item of the launch: kItemBins bins from k0 of one set of spectra and
// the pass of up to 256 kNa trials from j_p.
struct Item {
  int set;  // (first) series, or batch set
  int k0, j_p;
  int n_a;  // al's of the pass with trials: whole blocks, then the last one's
};
template <class C>
__host__ __device__ inline int n_passes(int n_dm) {
  return (n_dm + C::kPassTrials - 1) / C::kPassTrials;
}
// al's of block h of a pass with n_a al's (a series')
template <class C>
__device__ __forceinline__ int block_als(int n_a, int h) {
  if (C::kSeries || C::kTwin) return n_a;
  const int left = n_a - h * kBlockAls;
  return left < 0 ? 0 : left < kBlockAls ? left : kBlockAls;
}
template <class C>
__device__ __forceinline__ Item decode(const MacArgs& a, const BatchSet* sets, int n_sets, int item) {
  Item q;
  int local, n_dm, groups;
  if (!C::kSeries && sets) {
    int lo = 0, hi = n_sets - 1;  // last set with item_begin <= item
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (sets[mid].item_begin <= item) lo = mid; else hi = mid - 1;
    }
    q.set = lo;
    local = item - static_cast<int>(sets[lo].item_begin);
    n_dm = sets[lo].args.n_dm;
    groups = sets[lo].n_bin_tiles;
  } else {
    groups = (a.n_bins + C::kItemBins - 1) / C::kItemBins;
    n_dm = a.n_dm;
    const int per_set = groups * n_passes<C>(n_dm);
    q.set = item / per_set;
    local = item - q.set * per_set;
    q.set *= C::kSeriesSets;
  }
  const int p = local / groups;
  q.k0 = (local - p * groups) * C::kItemBins;
  q.j_p = p * C::kPassTrials;
  const int als = (n_dm - q.j_p + C::kAlTrials - 1) / C::kAlTrials;
  q.n_a = als < C::kMostAls ? als : C::kMostAls;
  return q;
}

template <class C>
__global__ void __launch_bounds__(kThreads, 1)
    mac_split_kernel(const MacArgs a, const BatchSet* sets, int n_sets, int n_items) {
  constexpr int kNa = C::kNa;
  constexpr int kBins = C::kBins;
  constexpr int kN = C::kN;
  constexpr int S = C::kStages;
  constexpr int T = C::kTables;
  extern __shared__ unsigned char smem_raw[];
  Smem<C>& sm = *reinterpret_cast<Smem<C>*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  volatile int* abort_flag = &sm.abort_flag;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < C::kTables; ++i) {
      mbar_init(&sm.pfull[i], 1);
      mbar_init(&sm.pfree[i], C::kTasks);
    }
    for (int i = 0; i < S; ++i) {
      mbar_init(&sm.full[i], C::kTasks + (a.test_withhold ? 1 : 0));  // (never all: stalled)
      mbar_init(&sm.done[i], 1);
    }
    for (int i = 0; i < C::kAccs; ++i) mbar_init(&sm.acc_free[i], kEpiWarps);
    mbar_init(&sm.drain, 1);
    sm.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sm.tmem)),
                 "n"(C::kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem;

  const int n_chan = sets ? sets[0].args.n_chan : a.n_chan;  // common to a batch
  const int n_chunks = (n_chan + kCh - 1) / kCh;
  const int per_item = n_chunks * kBins;  // stages of an item: chunk-major, bins inner
  // This CTA's items: every gridDim.x-th; or, where a second bin of the same
  // trials is stored together with a first, every gridDim.x-th two neighbours
  // (CTAs beside each other still work on bins beside each other, which share
  // sectors) and then its part of the rest, so that no CTA has more than one
  // item more than another.
  const int cta = blockIdx.x, n_ctas = gridDim.x;
  const int my_items = n_items / n_ctas + (cta < n_items % n_ctas ? 1 : 0);
  const int rounds = C::kSlots > 1 ? n_items / (2 * n_ctas) : 0;
  const int rest = n_items - rounds * 2 * n_ctas, each = rest / n_ctas, more = rest % n_ctas;
  auto item_at = [&](int i) {
    if (C::kSlots < 2) return cta + i * n_ctas;
    if (i < 2 * rounds) return (i >> 1) * 2 * n_ctas + 2 * cta + (i & 1);
    return rounds * 2 * n_ctas + cta * each + min(cta, more) + i - 2 * rounds;
  };
  const uint32_t total = static_cast<uint32_t>(my_items) * per_item;  // stages of this CTA
  // K steps of 16 channels of an item's last stage (the others have all four)
  const int tail_steps = (n_chan - (n_chunks - 1) * kCh + 15) / 16;
  bool ok = true;
  int* status = sets ? sets[0].args.status : a.status;

  if (warp < kEpiWarps) {
    // ------------------------------------------------------------ epilogue
    // A thread holds sixteen (bin, al) units of four sums each.
    const uint32_t t_lane = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    const bool is_c = lane < 16;  // this lane's row: Cb, or Sb of the same b
    const int b = 16 * (C::kTwin ? warp & 1 : warp) + (lane & 15);
    const int own = C::kTwin ? warp >> 1 : 0;  // this warp's bin of a stage
    uint32_t acc_at = 0;  // the stage's accumulator
    bool held = false;    // the last item's sums wait in slot 0 for this one's
    uint32_t n_item = 0;  // first stage of the item
    for (int i_item = 0; i_item < my_items && ok; ++i_item, n_item += per_item) {
      float2 acc[kBins][4][C::kOwn / 2];
#pragma unroll
      for (int s = 0; s < kBins; ++s)
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int i = 0; i < C::kOwn / 2; ++i) acc[s][t][i] = make_float2(0.f, 0.f);
      for (int c = 0; c < n_chunks && ok; ++c) {
#pragma unroll
        for (int sl = 0; sl < kBins; ++sl) {
          const uint32_t n = n_item + c * kBins + sl;
          const uint32_t s = n % S;
          const uint32_t d = acc_at;
          acc_at = acc_at + 1 == C::kAccs ? 0 : acc_at + 1;
          ok = ok && warp_wait(&sm.done[s], (n / S) & 1, abort_flag);
          if (!ok) break;
          float hv[C::kSeriesSets];
#pragma unroll
          for (int i = 0; i < C::kSeriesSets; ++i) hv[i] = sm.inv[n % (4 * C::kTables)][own + i];
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int h = 0; h < C::kOwn / 4; ++h) {
            const float hs = hv[C::kSeries ? 4 * h / C::kAls : 0];
            const float2 inv = make_float2(hs, hs);
#pragma unroll
            for (int t = 0; t < 4; t += 2) {
              // [type t, t + 1: hi hi; the small products of both][al]
              uint32_t r[4][4];
              const uint32_t col = t_lane + d * 2 * kN + t * kNa + own * C::kAls + 4 * h;
              tmem_ld4x4(col, col + kNa, col + kN, col + kN + kNa, r);
              if (h == C::kOwn / 4 - 1 && t == 2) {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                mbar_arrive_warp(&sm.acc_free[d]);
              }
#pragma unroll
              for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                  float2& to = acc[sl][t + e][2 * h + i];
                  const float2 v = __fadd2_rn(
                      make_float2(__uint_as_float(r[e][2 * i]), __uint_as_float(r[e][2 * i + 1])),
                      make_float2(__uint_as_float(r[2 + e][2 * i]),
                                  __uint_as_float(r[2 + e][2 * i + 1])));
                  to = __ffma2_rn(v, inv, to);
                }
            }
          }
        }
      }
      if (!ok) break;
      // The sums go through tensor memory, whose columns a loop can index.  A
      // wide pass of several series has one bin at a time: it leaves an even
      // bin's there and stores it with the next, sixteen bytes a trial instead
      // of eight (a store touches as many cache lines as lanes, whatever its
      // width).
      const int item = item_at(i_item);
      const Item q = decode<C>(a, sets, n_sets, item);
      const uint32_t park = t_lane + C::kPark + (held ? 64 : 0);
#pragma unroll
      for (int u = 0; u < (C::kSlots > 0 ? 16 : 0); u += 4) {
        float v[4][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int al = (u + e) / kBins, sl = (u + e) % kBins;
#pragma unroll
          for (int t = 0; t < 4; ++t) v[e][t] = (al & 1) ? acc[sl][t][al / 2].y : acc[sl][t][al / 2].x;
        }
        tmem_st16(park + u * 4, v);
      }
      if (C::kSlots > 0) asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      if (C::kSlots > 1 && !held && (q.k0 & 1) == 0 && i_item + 1 < my_items &&
          item_at(i_item + 1) == item + 1) {
        const Item next = decode<C>(a, sets, n_sets, item + 1);
        held = next.set == q.set && next.j_p == q.j_p;
        if (held) continue;
      }
      // Y[s, t] = A_s + i t B_s,  A_s = sum Cb X (Ca + i s Sa), B_s the same
      // with Sb: the lane of a Cb row makes the trials of s = +, that of the
      // Sb row of the same b those of s = -, each with two values of the other.
      constexpr int kOut = C::kOutBins;
      const int k0 = held ? q.k0 - 1 : q.k0 + own * kBins;
      const MacArgs& m = sets ? sets[q.set].args : a;
      const int64_t dm_stride = m.y_dm_stride;
      const int n_dm = m.n_dm, out_kind = m.out_kind;
      const float scale = m.scale;
      const int k_abs = m.k_begin + k0, real_a = m.real_bin_a, real_b = m.real_bin_b;
      const int64_t off = (sets ? 0 : static_cast<int64_t>(q.set) * m.y_series_stride) + k0;
      void* const Yv = m.Y;
      const int n_out = C::kSlots > 1 ? (held ? 2 : 1) : m.n_bins - k0 < kOut ? m.n_bins - k0 : kOut;
      const bool whole = n_out == kOut;
      held = false;
      const float sg = is_c ? 1.f : -1.f;
#pragma unroll (C::kSlots > 0 ? 1 : kNa)
      for (int al = 0; al < C::kOwn; ++al) {
        if (C::kSeries ? al % C::kAls < q.n_a : al < q.n_a) {
          float v[kOut][4];
          if constexpr (C::kSlots > 1)
            tmem_ld4(t_lane + C::kPark + al * 4, t_lane + C::kPark + 64 + al * 4, v);
          else if constexpr (C::kSlots == 1)
            tmem_ld4(t_lane + C::kPark + al * 4 * kBins, v);
          else
#pragma unroll
            for (int t = 0; t < 4; ++t) v[0][t] = (al & 1) ? acc[0][t][al / 2].y : acc[0][t][al / 2].x;
          float2 y[2][kOut];  // t = +, -
#pragma unroll
          for (int sl = 0; sl < kOut; ++sl) {
            const float ox = v[sl][0] - sg * v[sl][3], oy = v[sl][1] + sg * v[sl][2];
            const float rx = __shfl_xor_sync(0xffffffffu, v[sl][0] + sg * v[sl][3], 16);
            const float ry = __shfl_xor_sync(0xffffffffu, v[sl][1] - sg * v[sl][2], 16);
            const float2 A = is_c ? make_float2(ox, oy) : make_float2(rx, ry);
            const float2 B = is_c ? make_float2(rx, ry) : make_float2(ox, oy);
            const bool real_only = k_abs + sl == real_a || k_abs + sl == real_b;
            y[0][sl] = make_float2((A.x - B.y) * scale, real_only ? 0.f : (A.y + B.x) * scale);
            y[1][sl] = make_float2((A.x + B.y) * scale, real_only ? 0.f : (A.y - B.x) * scale);
          }
          // trial of (s, al, t, b)
          const int h = al / C::kAls, step = C::kAlTrials / 2 * (al % C::kAls) + C::kAlTrials / 4;
          const int jc = q.j_p + (C::kSeries ? 0 : kPairTrials * kBlockAls * h) +
                         C::kAlTrials / 2 * block_als<C>(q.n_a, h) + (is_c ? step : -step);
          const int64_t off_h = off + (C::kSeries ? h * m.y_series_stride : 0);
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const int j = t == 0 ? jc + b : jc - 1 - b;
            if (j >= n_dm) continue;
            const int64_t o = off_h + static_cast<int64_t>(j) * dm_stride;
            if (out_kind == 2) {
              float* Y = static_cast<float*>(Yv) + o;
              float pw[kOut];
#pragma unroll
              for (int sl = 0; sl < kOut; ++sl)
                pw[sl] = y[t][sl].x * y[t][sl].x + y[t][sl].y * y[t][sl].y;
              if (kOut == 4 && whole && (reinterpret_cast<uintptr_t>(Y) & 15) == 0) {
                *reinterpret_cast<float4*>(Y) = make_float4(pw[0], pw[1 % kOut], pw[2 % kOut], pw[3 % kOut]);
              } else if (kOut == 2 && whole && (reinterpret_cast<uintptr_t>(Y) & 7) == 0) {
                *reinterpret_cast<float2*>(Y) = make_float2(pw[0], pw[1 % kOut]);
              } else {
#pragma unroll
                for (int sl = 0; sl < kOut; ++sl)
                  if (sl < n_out) Y[sl] = pw[sl];
              }
            } else {
              float2* Y = static_cast<float2*>(Yv) + o;
              if (kOut >= 2 && whole && (reinterpret_cast<uintptr_t>(Y) & 15) == 0) {
#pragma unroll
                for (int sl = 0; sl < kOut; sl += 2)
                  *reinterpret_cast<float4*>(Y + sl) =
                      make_float4(y[t][sl].x, y[t][sl].y, y[t][(sl + 1) % kOut].x, y[t][(sl + 1) % kOut].y);
              } else {
#pragma unroll
                for (int sl = 0; sl < kOut; ++sl)
                  if (sl < n_out) Y[sl] = y[t][sl];
              }
            }
          }
        }
      }
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    const uint32_t el = elect_one();
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t base = __shfl_sync(0xffffffffu, smem_u32(&sm.stage[0][0]), 0);
    constexpr uint32_t id = (1u << 4) | (static_cast<uint32_t>(kN >> 3) << 17) |
                            (static_cast<uint32_t>(kRows >> 4) << 24);  // FP16 x FP16 -> FP32
    constexpr uint32_t id2 = (1u << 4) | (static_cast<uint32_t>(2 * kN >> 3) << 17) |
                             (static_cast<uint32_t>(kRows >> 4) << 24);  // hi and lo columns at once
    bool issued = false;
    uint32_t left = per_item;  // stages of the item still to come
    uint32_t phase = 0, acc_phase = 1;
    int s = 0, acc = 0;
    for (uint32_t n = 0; n < total; ++n) {
      ok = warp_wait(&sm.full[s], phase, abort_flag) &&
           warp_wait(&sm.acc_free[acc], acc_phase, abort_flag);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int steps = left <= kBins ? tail_steps : 4;
      if (el) {
        const uint32_t st = base + s * C::kStageBytes;
        const uint32_t d = tm + acc * 2 * kN;
        const uint64_t a_hi = core_desc(st, kRows * 16);
        const uint64_t a_lo = core_desc(st + C::kATile, kRows * 16);
        const uint64_t b = core_desc(st + 2 * C::kATile, 2 * kN * 16);
        // A K step of 16 channels: two core matrices along K.  The rows' hi
        // term takes both terms of the columns in one MMA of twice the
        // width (the MMAs are bound by reading the rows from shared memory:
        // two reads a K step instead of three); the small products go to
        // the second half of the accumulator.
        constexpr uint32_t ka = 2 * kRows * 16 / 16, kb = 2 * 2 * kN * 16 / 16;
        if (steps == 4) {
#pragma unroll
          for (int i = 0; i < 4; ++i) mma(d, a_hi + i * ka, b + i * kb, i > 0 ? 1u : 0u, id2);
#pragma unroll
          for (int i = 0; i < 4; ++i) mma(d + kN, a_lo + i * ka, b + i * kb, 1u, id);
        } else {
#pragma unroll 1
          for (int i = 0; i < steps; ++i) mma(d, a_hi + i * ka, b + i * kb, i > 0 ? 1u : 0u, id2);
#pragma unroll 1
          for (int i = 0; i < steps; ++i) mma(d + kN, a_lo + i * ka, b + i * kb, 1u, id);
        }
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                smem_u32(&sm.done[s]))
            : "memory");
      }
      issued = true;
      left = left == 1 ? per_item : left - 1;
      if (++s == S) {
        s = 0;
        phase ^= 1;
      }
      if (++acc == C::kAccs) {
        acc = 0;
        acc_phase ^= 1;
      }
      __syncwarp();
    }
    // (the epilogue waits for every stage, so tensor memory is idle at the
    // end; after a timeout the MMAs in flight are drained here)
    if (!ok && issued) {
      if (el)
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                smem_u32(&sm.drain))
            : "memory");
      volatile int never = 0;
      warp_wait(&sm.drain, 0, &never);
    }
  } else if (warp < kProdFirst) {
    // ------------------------------------------------------------ stage tables
    // lane = channels lane and lane + 32 of the stage; the next stage's loads
    // fly while this one's table is made and waits for its place
    struct Fetched {
      float2 x[C::kSets][2];
      uint4 pc[2];      // u_lo, u_hi, v_lo, v_hi
      uint32_t k;       // absolute bin
      uint32_t before[C::kCentres];  // Jc - 1/2: the trial below each block's centre
      int c0;           // this lane's first channel
      int steps;        // K steps of the stage
      bool bin_ok[C::kRowBins];
    };
    const int p = warp - kPrepFirst;
    int i_item = 0, q = p;  // stage within the item
    // the item at hand, in registers: its spectra, constants and phases' origin
    int cur = -1, left_bins = 0, k_abs = 0;
    uint32_t before[C::kCentres] = {};
    const float2* X = nullptr;
    int64_t xs = 0, set_stride = 0;
    const PhaseConst* pcs = nullptr;
    auto fetch = [&](Fetched& f) {
      // The loads are unconditional, from clamped addresses, and idle channels
      // and bins are zeroed where they are used: a load under a condition
      // would be waited for right here, to merge it with the other value.
      while (q >= per_item) {
        q -= per_item;
        ++i_item;
      }
      if (i_item != cur && i_item < my_items) {
        const Item it = decode<C>(a, sets, n_sets, item_at(i_item));
        const MacArgs& m = sets ? sets[it.set].args : a;
        cur = i_item;
        left_bins = m.n_bins - it.k0;
        k_abs = m.k_begin + it.k0;
#pragma unroll
        for (int h = 0; h < C::kCentres; ++h)
          before[h] = static_cast<uint32_t>(m.j_begin + it.j_p + kPairTrials * kBlockAls * h +
                                            C::kAlTrials / 2 * block_als<C>(it.n_a, h) - 1);
        X = m.X + (sets ? 0 : static_cast<int64_t>(it.set) * m.x_series_stride) + it.k0;
        xs = m.x_chan_stride;
        set_stride = m.x_series_stride;
        pcs = m.pc;
      }
      const int slot = q % kBins;
      f.steps = q >= per_item - kBins ? tail_steps : 4;
      f.c0 = q / kBins * kCh + lane;
#pragma unroll
      for (int i = 0; i < C::kRowBins; ++i) f.bin_ok[i] = slot + i * kBins < left_bins;
      f.k = static_cast<uint32_t>(k_abs + slot);
#pragma unroll
      for (int h = 0; h < C::kCentres; ++h) f.before[h] = before[h];
      const float2* xb[C::kRowBins];
#pragma unroll
      for (int i = 0; i < C::kRowBins; ++i) xb[i] = X + (f.bin_ok[i] ? slot + i * kBins : 0);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = min(f.c0 + 32 * h, n_chan - 1);
        asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(f.pc[h].x), "=r"(f.pc[h].y), "=r"(f.pc[h].z), "=r"(f.pc[h].w)
                     : "l"(pcs + c));
#pragma unroll
        for (int i = 0; i < C::kSets; ++i)
          asm volatile("ld.global.nc.v2.f32 {%0,%1}, [%2];"
                       : "=f"(f.x[i][h].x), "=f"(f.x[i][h].y)
                       : "l"(xb[C::kTwin ? i : 0] + (C::kTwin ? 0 : i * set_stride) +
                             static_cast<int64_t>(c) * xs));
      }
      q += kPrepWarps;
    };
    // (Past the CTA's last stage the loads repeat addresses of its last item; a
    // warp without a first stage has no item to load from.)
    Fetched next;
    if (p < total) fetch(next);
    for (uint32_t n = p; n < total; n += kPrepWarps) {
      const uint32_t s = n % T;
      const uint4 pc[2] = {next.pc[0], next.pc[1]};
      const uint32_t k = next.k;
      uint32_t j1[C::kCentres];
#pragma unroll
      for (int h = 0; h < C::kCentres; ++h) j1[h] = next.before[h];
      const int steps = next.steps;
      // power-of-two scale: the stage's largest component to [2^13, 2^14)
      float2 xr[C::kSets], xi[C::kSets];
      int f[C::kSets];
#pragma unroll
      for (int i = 0; i < C::kSets; ++i) {
        float2 x[2];
        uint32_t top = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool use = next.bin_ok[C::kTwin ? i : 0] && next.c0 + 32 * h < n_chan;
          x[h] = use ? next.x[i][h] : make_float2(0.f, 0.f);
          top = max(top, max(__float_as_uint(x[h].x) & 0x7FFFFFFFu, __float_as_uint(x[h].y) & 0x7FFFFFFFu));
        }
        top = __reduce_max_sync(0xffffffffu, top);
        f[i] = 14 + 253 - static_cast<int>(top >> 23);
        f[i] = f[i] < 1 ? 1 : (f[i] > 253 ? 253 : f[i]);
        const float sc = __uint_as_float(static_cast<uint32_t>(f[i]) << 23);
        xr[i] = make_float2(x[0].x * sc, x[1].x * sc);
        xi[i] = make_float2(x[0].y * sc, x[1].y * sc);
      }
      uint32_t hw[C::kRowBins][2], ha[C::kRowBins][2], pf[C::kRowBins][2], pm[C::kCentrePhases][2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint64_t u = (static_cast<uint64_t>(pc[h].y) << 32) | pc[h].x;
        const uint64_t v = (static_cast<uint64_t>(pc[h].w) << 32) | pc[h].z;
        constexpr uint64_t kRound = 0x80000000ull;
        constexpr int kAlShift = C::kTwin ? 6 : 7;
#pragma unroll
        for (int e = 0; e < C::kRowBins; ++e) {
          const uint32_t ke = k + e * kBins;
          const uint64_t half = (v * ke) >> 1;  // half a trial step, mod half a cycle
          hw[e][h] = static_cast<uint32_t>((half + kRound) >> 32);
          ha[e][h] = static_cast<uint32_t>(((half << kAlShift) + kRound) >> 32);
          pf[e][h] = static_cast<uint32_t>(((half << 5) + kRound) >> 32);
#pragma unroll
          for (int i = 0; i < C::kCentres; ++i)  // the blocks' centres
            pm[C::kTwin ? e : i][h] = static_cast<uint32_t>(((u + v * j1[i]) * ke + half) >> 32);
        }
      }
      float2 fc[C::kRowBins], fs[C::kRowBins], zr[C::kBlocks], zi[C::kBlocks];
#pragma unroll
      for (int e = 0; e < C::kRowBins; ++e) sincos2(pf[e][0], pf[e][1], fc[e], fs[e]);
      float2 mc, ms;
#pragma unroll
      for (int i = 0; i < C::kBlocks; ++i) {
        if (i < C::kCentrePhases)
          sincos2(pm[i % C::kCentrePhases][0], pm[i % C::kCentrePhases][1], mc, ms);
        const int e = C::kSets > 1 ? i : 0;
        zr[i] = __ffma2_rn(xr[e], mc, __fmul2_rn(make_float2(-xi[e].x, -xi[e].y), ms));
        zi[i] = __ffma2_rn(xr[e], ms, __fmul2_rn(xi[e], mc));
      }
      fetch(next);
      ok = warp_wait(&sm.pfree[s], ((n / T) & 1) ^ 1, abort_flag);
      if (!ok) break;
      Table<C>& tb = sm.table[s];
#pragma unroll
      for (int e = 0; e < C::kRowBins; ++e) {
        tb.hw[e][lane] = hw[e][0];
        tb.hw[e][lane + 32] = hw[e][1];
        tb.ha[e][lane] = ha[e][0];
        tb.ha[e][lane + 32] = ha[e][1];
        tb.fr[e][lane] = fc[e].x;
        tb.fr[e][lane + 32] = fc[e].y;
        tb.fi[e][lane] = fs[e].x;
        tb.fi[e][lane + 32] = fs[e].y;
      }
#pragma unroll
      for (int i = 0; i < C::kBlocks; ++i) {
        tb.xr[i][lane] = zr[i].x;
        tb.xr[i][lane + 32] = zr[i].y;
        tb.xi[i][lane] = zi[i].x;
        tb.xi[i][lane + 32] = zi[i].y;
      }
      if (lane == 0) tb.steps = steps;
      if (lane == 0) {
#pragma unroll
        for (int i = 0; i < C::kSets; ++i)
          sm.inv[n % (4 * C::kTables)][i] = __uint_as_float(static_cast<uint32_t>(254 - f[i]) << 23);
      }
      // Tables complete in order: a producer steps fewer than T stages at a
      // time, so the table T stages back is then complete when it waits for
      // one (a wait by parity sees only whether the count is odd).
      if (n > 0)
        ok = warp_wait(&sm.pfull[(n - 1) % T], ((n - 1) / T) & 1, abort_flag);
      if (!ok) break;
      mbar_arrive_warp(&sm.pfull[s]);
    }
  } else {
    // ------------------------------------------------------------ producers
    const bool few = n_chan <= kFewChan;
    // Waits by parity see one phase back only.  A producer steps fewer than S
    // stages from task to task and waits for each task's stage to be free, so
    // when it waits for stage n to be free, n - 2 S is (MMAs end in order).
    for (uint32_t task = warp - kProdFirst;; task += kProdWarps) {
      const uint32_t n = task / C::kTasks;
      const int part0 = static_cast<int>(task % C::kTasks);
      const bool rows = part0 >= C::kColTasks;
      const int part = rows ? part0 - C::kColTasks : part0;
      if (n >= total) break;
      const uint32_t s = n % S;
      const uint32_t ts = n % T;
      ok = warp_wait(&sm.pfull[ts], (n / T) & 1, abort_flag);
      if (!ok) break;
      const Table<C>& tb = sm.table[ts];
      const int steps = tb.steps;
      if (rows) {
        // rows: lane = (b < 16, half of an octet of channels): Cb, Sb of four
        // channels for b, b + 16, b + 32 and b + 48, the later ones by the
        // 16-step phasor (both halves of a row's 16 bytes are stored by the
        // same instruction, and only 32 registers hold a lane's results)
        if (part < steps) {
          const int b = lane >> 1, half = lane & 1;  // (16 lanes store 128 contiguous bytes)
          const uint32_t mul = 2u * b + 1u;
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            const int oct = 2 * part + o;
            const int ch = 8 * oct + 4 * half;
            uint32_t hi[8][2], lo[8][2];  // [C, S of b + 16 i][channel pair]
#pragma unroll
            for (int e = 0; e < C::kRowBins; ++e) {  // (twin: i = 0, 1 of each bin)
              const uint4 hv = *reinterpret_cast<const uint4*>(&tb.hw[e][ch]);
              const float4 frv = *reinterpret_cast<const float4*>(&tb.fr[e][ch]);
              const float4 fiv = *reinterpret_cast<const float4*>(&tb.fi[e][ch]);
              constexpr int kSteps = 4 / C::kRowBins;
#pragma unroll
              for (int p = 0; p < 2; ++p) {
                const float2 fr = p ? make_float2(frv.z, frv.w) : make_float2(frv.x, frv.y);
                const float2 fi = p ? make_float2(fiv.z, fiv.w) : make_float2(fiv.x, fiv.y);
                const float2 nfi = make_float2(-fi.x, -fi.y);
                const float2 w0 = unit_phasor(mul * (p ? hv.z : hv.x));
                const float2 w1 = unit_phasor(mul * (p ? hv.w : hv.y));
                float2 cs = make_float2(w0.x, w1.x), sn = make_float2(w0.y, w1.y);
#pragma unroll
                for (int i = 0; i < kSteps; ++i) {
                  split2(cs, hi[e * kSteps + i][p], lo[e * kSteps + i][p]);
                  split2(sn, hi[4 + e * kSteps + i][p], lo[4 + e * kSteps + i][p]);
                  if (i + 1 < kSteps) {
                    const float2 c1 = __ffma2_rn(cs, fr, __fmul2_rn(sn, nfi));
                    sn = __ffma2_rn(cs, fi, __fmul2_rn(sn, fr));
                    cs = c1;
                  }
                }
              }
            }
            if (o == 0) {
              ok = warp_wait(&sm.done[s], ((n / S) & 1) ^ 1, abort_flag);
              if (!ok) break;
            }
            unsigned char* at = &sm.stage[s][oct * kRows * 16 + b * 16 + half * 8];  // (row b)
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              const int row = 32 * (t & 3) + 16 * (t >> 2);
              *reinterpret_cast<uint2*>(at + row * 16) = make_uint2(hi[t][0], hi[t][1]);
              *reinterpret_cast<uint2*>(at + C::kATile + row * 16) = make_uint2(lo[t][0], lo[t][1]);
            }
          }
          if (!ok) break;
        } else {  // (waited for all the same: see the wait by parity)
          ok = warp_wait(&sm.done[s], ((n / S) & 1) ^ 1, abort_flag);
          if (!ok) break;
        }
      } else {
        // columns: lane = (al, half octet): Xr Ca, Xi Ca, Xr Sa, Xi Sa of four
        // channels at a time
        constexpr int kHalves = 32 / kNa;               // half octets at a time: 2, 4, 8
        static_assert(16 / C::kColTasks / kHalves == 2, "two rounds a task");
        const int al = (lane >> 1) % kNa;
        const int blk = al / C::kAls;
        const uint32_t mul = 2u * (al % C::kAls) + 1u;
        const int h0 = part * 2 * kHalves + 2 * (lane / (2 * kNa)) + (lane & 1);
        const bool live = part * 2 * kHalves < 4 * steps;  // (the round's first, so uniform)
        uint32_t hi[2][4][2], lo[2][4][2];  // [round][type][channel pair]
        if (live) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int ch = 4 * (h0 + e * kHalves);
            const uint4 hv = *reinterpret_cast<const uint4*>(&tb.ha[C::kTwin ? blk : 0][ch]);
            const float4 xrv = *reinterpret_cast<const float4*>(&tb.xr[blk][ch]);
            const float4 xiv = *reinterpret_cast<const float4*>(&tb.xi[blk][ch]);
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const float2 xr = p ? make_float2(xrv.z, xrv.w) : make_float2(xrv.x, xrv.y);
              const float2 xi = p ? make_float2(xiv.z, xiv.w) : make_float2(xiv.x, xiv.y);
              const uint32_t p0 = mul * (p ? hv.z : hv.x), p1 = mul * (p ? hv.w : hv.y);
              float2 cs, sn;
              if (few) {
                sincos2(p0, p1, cs, sn);
              } else {
                const float2 w0 = unit_phasor(p0), w1 = unit_phasor(p1);
                cs = make_float2(w0.x, w1.x);
                sn = make_float2(w0.y, w1.y);
              }
              split2(__fmul2_rn(xr, cs), hi[e][0][p], lo[e][0][p]);
              split2(__fmul2_rn(xi, cs), hi[e][1][p], lo[e][1][p]);
              split2(__fmul2_rn(xr, sn), hi[e][2][p], lo[e][2][p]);
              split2(__fmul2_rn(xi, sn), hi[e][3][p], lo[e][3][p]);
            }
          }
        }
        ok = warp_wait(&sm.done[s], ((n / S) & 1) ^ 1, abort_flag);
        if (!ok) break;
        if (live) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int hf = h0 + e * kHalves;
            unsigned char* bt =
                &sm.stage[s][2 * C::kATile + (hf >> 1) * 2 * kN * 16 + al * 16 + (hf & 1) * 8];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              *reinterpret_cast<uint2*>(bt + t * kNa * 16) = make_uint2(hi[e][t][0], hi[e][t][1]);
              *reinterpret_cast<uint2*>(bt + kN * 16 + t * kNa * 16) =
                  make_uint2(lo[e][t][0], lo[e][t][1]);
            }
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&sm.full[s]);
        mbar_arrive(&sm.pfree[ts]);
      }
    }
  }
  if (!ok) {
    *abort_flag = 1;
    if (status && lane == 0) atomicExch(status, FDD_ERR_TIMEOUT);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "n"(C::kTmemCols));
  }
}

// The passes' forms: one series with up to 512 (two bins a stage), 1024, 2048 or
// 4096 trials a pass,
// or two or four series that share the rows of up to 1024, two of up to 2048.
enum Form { kUpTo512, kUpTo1024, kUpTo2048, kUpTo4096, kTwoUpTo1024, kFourUpTo1024, kTwoUpTo2048, kForms };

struct FormInfo {
  const void* fn;
  int smem, sets, bins, pass_trials;
};
template <class C>
FormInfo form_info() {
  return {reinterpret_cast<const void*>(&mac_split_kernel<C>), static_cast<int>(sizeof(Smem<C>)) + 128,
          C::kSeriesSets, C::kItemBins, C::kPassTrials};
}
FormInfo form_info(Form f) {
  switch (f) {
    case kUpTo512: return form_info<Cfg<4, 2, false, true>>();
    case kUpTo1024: return form_info<Cfg<4, 1, false>>();
    case kUpTo2048: return form_info<Cfg<8, 1, false>>();
    case kUpTo4096: return form_info<Cfg<8, 2, false>>();
    case kTwoUpTo1024: return form_info<Cfg<4, 2, true>>();
    case kFourUpTo1024: return form_info<Cfg<4, 4, true>>();
    default: return form_info<Cfg<8, 2, true>>();
  }
}

// The form for n_dm trials of n_series (at least its sets) series.  The rows
// take most of a stage, so the widest pass that the trials or series fill, and
// half the rows where the plan (or batch) has no more than 512 trials (of_n_dm):
// calls on parts of its trials then take the same form as the whole.  The form
// may depend on the series only among those whose results are the same bits.
// 4096 bins x 1024 channels x 512 trials take 190 us in twin stages, 249 in
// those for 1024.
// With few channels the rows cost little and storing the sums is what counts,
// which a pass of more bins does in fewer and longer pieces: there more than
// 2048 trials go through passes of 2048, and series by themselves (in one
// launch), with the same bits.  4096 bins x 8192 trials: 1 channel 159 us in
// passes of 2048 and 378 of 4096, 64 channels 184 and 381, 128 246 and 336
// (3000 trials 119 and 135), 192 340 and 359 (3000 trials 165 and 150).  4096
// bins x 3 series x 700 trials: 1 channel 62 us alone and 72 shared, 32 67 and
// 76, 64 79 and 84 (but 4 series x 600 trials 8 % slower alone); x 2048 trials
// 120 and 169, 124 and 172, 138 and 173, 100 channels 178 and 206 (but 2 series
// x 1100 trials 10 % slower alone).
constexpr int kFewForPass = 128, kFewForTwo2048 = 64, kFewFor1024 = 32;
Form form_for(int n_dm, int n_series, int of_n_dm, int n_chan) {
  const int total = (n_dm + kPairTrials - 1) / kPairTrials;
  if (total > 8) return n_chan > kFewForPass ? kUpTo4096 : kUpTo2048;
  if (of_n_dm > 0 && of_n_dm <= 2 * kPairTrials) return kUpTo512;
  if (total > 4) return n_series >= 2 && n_chan > kFewForTwo2048 ? kTwoUpTo2048 : kUpTo2048;
  if (n_chan <= kFewFor1024) return kUpTo1024;
  return n_series >= 4 ? kFourUpTo1024 : n_series >= 2 ? kTwoUpTo1024 : kUpTo1024;
}

constexpr int kMaxDevices = 64;
std::atomic<int> g_sms[kMaxDevices];

cudaError_t sm_count(int* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int n = dev < kMaxDevices ? g_sms[dev].load(std::memory_order_relaxed) : 0;
  if (n == 0) {
    e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (dev < kMaxDevices) g_sms[dev].store(n, std::memory_order_relaxed);
  }
  *out = n;
  return cudaSuccess;
}

cudaError_t launch_split(const MacArgs& a, const BatchSet* sets, int n_sets, int n_items,
                         const FormInfo& f, int n_ctas, cudaStream_t s) {
  MacArgs args = a;
  void* params[] = {&args, &sets, &n_sets, &n_items};
  const dim3 grid(n_items < n_ctas ? n_items : n_ctas);
  note_launches(1);
  return cudaLaunchKernel(f.fn, grid, dim3(kThreads), params, f.smem, s);
}

constexpr long long kMaxItems = 0x7FFF0000LL;  // item numbers, stepped by the grid, stay in an int

}  // namespace

size_t mac_split_smem_bytes() {
  int most = 0;
  for (int f = 0; f < kForms; ++f) {
    const int b = form_info(static_cast<Form>(f)).smem;
    if (b > most) most = b;
  }
  return most;
}

cudaError_t mac_split_prepare() {
  cudaError_t e = cudaSuccess;
  for (int f = 0; f < kForms && e == cudaSuccess; ++f) {
    const FormInfo i = form_info(static_cast<Form>(f));
    e = cudaFuncSetAttribute(i.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, i.smem);
  }
  return e;
}

bool mac_split_series_share(int n_dm) { return form_info(form_for(n_dm, 2, n_dm, INT_MAX)).sets > 1; }

int mac_split_form(int n_dm, int n_chan) { return form_for(n_dm, 1, n_dm, n_chan); }

void mac_split_batch_shape(int n_dm, int n_chan, long long n_bins, int* bin_groups, int* passes) {
  const FormInfo f = form_info(form_for(n_dm, 1, n_dm, n_chan));
  *bin_groups = static_cast<int>((n_bins + f.bins - 1) / f.bins);
  *passes = (n_dm + f.pass_trials - 1) / f.pass_trials;
}

cudaError_t launch_mac_split_batch(const BatchSet* d_sets, int n_sets, long long n_items,
                                   int max_n_dm, int n_chan, int n_ctas, cudaStream_t s) {
  if (n_items <= 0) return cudaSuccess;
  if (n_items > kMaxItems) return cudaErrorInvalidConfiguration;
  return launch_split(MacArgs{}, d_sets, n_sets, static_cast<int>(n_items),
                      form_info(form_for(max_n_dm, 1, max_n_dm, n_chan)), n_ctas, s);
}

cudaError_t launch_mac_split(const MacArgs& a, cudaStream_t s) {
  int n_sms = 0;
  cudaError_t e = sm_count(&n_sms);
  if (e != cudaSuccess) return e;
  const size_t y_elem = a.out_kind == 2 ? sizeof(float) : sizeof(float2);
  auto items = [&](const FormInfo& f) {
    return static_cast<long long>((a.n_bins + f.bins - 1) / f.bins) *
           ((a.n_dm + f.pass_trials - 1) / f.pass_trials);
  };
  // Series in groups that share passes, then the rest in smaller groups, in
  // launches one after another; or all by themselves in one launch, where that
  // takes no more than one item per SM (of two stages of channels at most, no
  // more than launches saved).  3 series x 600 trials x 48 channels x 200
  // bins: 10 us in one launch, 19 in two; 1024 channels x 64 bins 41 and 70.
  for (int s0 = 0; s0 < a.n_series;) {
    const int left = a.n_series - s0;
    FormInfo f = form_info(form_for(a.n_dm, left, a.of_n_dm, a.n_chan));
    const FormInfo alone = form_info(form_for(a.n_dm, 1, a.of_n_dm, a.n_chan));
    int launches = 0;
    for (int l = left; l > 0; ++launches) l %= form_info(form_for(a.n_dm, l, a.of_n_dm, a.n_chan)).sets;
    if (launches > 1 && left * items(alone) <= (a.n_chan > kFewForPass ? 1 : launches) * n_sms)
      f = alone;
    const long long per_set = items(f);
    if (per_set > kMaxItems) return cudaErrorInvalidConfiguration;
    // (as many as leave item numbers in an int)
    long long sets = left / f.sets;
    if (sets > kMaxItems / per_set) sets = kMaxItems / per_set;
    MacArgs c = a;
    c.n_series = static_cast<int>(sets) * f.sets;
    c.X = a.X + s0 * a.x_series_stride;
    c.Y = static_cast<char*>(a.Y) + y_elem * static_cast<size_t>(s0 * a.y_series_stride);
    e = launch_split(c, nullptr, 0, static_cast<int>(per_set * sets), f, n_sms, s);
    if (e != cudaSuccess) return e;
    s0 += c.n_series;
  }
  return cudaSuccess;
}

}  // namespace fdd
