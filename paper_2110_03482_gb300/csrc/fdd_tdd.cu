// fdd_tdd.cu -- brute-force time-domain dedispersion (Eq. 2; the method the
// paper measures Fourier-domain dedispersion against, Sect. 4):
//
//   y[j][n] = sum_nu x[nu][n + s[j][nu]],   s = delay of Eq. 1 rounded to the
//                                              nearest sample,
//
// for the valid samples n < n_t - D_max (every channel in range).  One CTA
// computes kTdDms trials x kTdSamp samples: for kTdCh channels at a time it
// stages each channel's input window (the samples the block's trials read:
// from t0 + the block's smallest shift, kTdSamp + the shift span wide) in
// shared memory, then every lane adds, for its 4 trials and 8 samples
// (lane + 32 i), one window value per channel: 32 consecutive lanes read 32
// consecutive floats, so each add costs one conflict-free 4-byte shared load.
// Shared-memory bandwidth (128 B per clock per SM) bounds the kernel at 32
// adds per clock per SM.  The stages are double-buffered: the next stage's
// windows and relative shifts stream in with cp.async while the current one
// is summed.  Trial blocks run fastest in the grid, so the blocks that share
// a time window run together and read it from L2.
//
// 8-bit samples (tdd8_kernel): their sums are whole numbers, exact in FP32 up to
// 65793 channels, so they may be added as integers: two 16-bit sums per
// instruction (up to 256 channels, then added to 32-bit ones).  A stage's
// windows arrive as bytes and are laid out four times, shifted by 0 to 3
// bytes, so that every trial reads four samples with one aligned 4-byte load:
// a quarter of the shared-memory traffic per add.  Two byte permutes spread
// a word over two 16-bit pairs, and one three-operand add takes two channels;
// these integer instructions (three for four adds) bound it.  1024 channels x
// 512 trials x 2^17 samples take 4.4 ms, as floats 10.8; that is 54 adds a clock and SM of
// the 79 of the integer pipe.  (Half of the adds as multiply-adds on the other
// pipe, or sixteen channels a stage: the same 4.4.)
#include "fdd_internal.h"

namespace fdd {
namespace {

constexpr int kTdWarps = 8;
constexpr int kTdThreads = kTdWarps * 32;
constexpr int kTdDmsWarp = kTdDms / kTdWarps;  // trials per warp (4)
constexpr int kTdPer = kTdSamp / 32;           // samples per lane (8)

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 4 bytes global -> shared, asynchronously; zeros when !valid (no read).
__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(valid ? 4 : 0)
               : "memory");
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src)
               : "memory");
}

// Stage (channels c0 .. c0 + kTdCh - 1) into buffer (rel, win).
__device__ __forceinline__ void tdd_fill(const TddArgs& a, int blk, int64_t t0, int c0, int* rel,
                                         float* win) {
  // relative shifts: kTdCh x kTdDms ints, contiguous in the table, 16 bytes a thread
  const int nc = a.n_chan - c0 < kTdCh ? a.n_chan - c0 : kTdCh;
  const int* src_rel = a.rel + (static_cast<int64_t>(blk) * a.n_chan + c0) * kTdDms;
  for (int q = threadIdx.x; q < nc * kTdDms / 4; q += kTdThreads)
    cp_async16(rel + 4 * q, src_rel + 4 * q);
#pragma unroll 1
  for (int cc = 0; cc < nc; ++cc) {
    const int c = c0 + cc;
    float* row = win + cc * a.win;
    const int64_t t_first = t0 + a.base[static_cast<int64_t>(blk) * a.n_chan + c];
    const float* src = a.x + static_cast<int64_t>(c) * a.n_t + t_first;
    const int64_t n_in = a.n_t - t_first;
    for (int w = threadIdx.x; w < a.win; w += kTdThreads)
      cp_async4(row + w, w < n_in ? src + w : a.x, w < n_in);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__global__ void __launch_bounds__(kTdThreads) tdd_kernel(const TddArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // two buffers, each [kTdCh][kTdDms] relative shifts then [kTdCh][a.win] window
  const size_t buf_bytes = sizeof(int) * kTdCh * kTdDms + sizeof(float) * size_t(kTdCh) * a.win;
  auto rel_of = [&](int b) { return reinterpret_cast<int*>(smem_raw + b * buf_bytes); };
  auto win_of = [&](int b) {
    return reinterpret_cast<float*>(smem_raw + b * buf_bytes + sizeof(int) * kTdCh * kTdDms);
  };
  const int blk = blockIdx.x;
  const int j0 = blk * kTdDms;
  const int64_t t0 = static_cast<int64_t>(blockIdx.y) * kTdSamp;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  float acc[kTdDmsWarp][kTdPer];
#pragma unroll
  for (int d = 0; d < kTdDmsWarp; ++d)
#pragma unroll
    for (int i = 0; i < kTdPer; ++i) acc[d][i] = 0.f;

  const int n_stages = (a.n_chan + kTdCh - 1) / kTdCh;
  tdd_fill(a, blk, t0, 0, rel_of(0), win_of(0));
  for (int st = 0; st < n_stages; ++st) {
    const int cur = st & 1;
    if (st + 1 < n_stages) {
      tdd_fill(a, blk, t0, (st + 1) * kTdCh, rel_of(cur ^ 1), win_of(cur ^ 1));
      asm volatile("cp.async.wait_group 1;" ::: "memory");  // this stage's copies are done
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();  // ... and every thread's
    const int c0 = st * kTdCh;
    const int nc = a.n_chan - c0 < kTdCh ? a.n_chan - c0 : kTdCh;
    const int* rel = rel_of(cur);
    const float* win = win_of(cur);
#pragma unroll
    for (int cc = 0; cc < kTdCh; ++cc) {
      if (cc < nc) {
        const float* wr = win + cc * a.win + lane;
#pragma unroll
        for (int d = 0; d < kTdDmsWarp; ++d) {
          const int r = rel[cc * kTdDms + warp * kTdDmsWarp + d];
#pragma unroll
          for (int i = 0; i < kTdPer; ++i) acc[d][i] += wr[32 * i + r];
        }
      }
    }
    __syncthreads();  // this buffer is refilled by the next iteration's prefetch
  }

#pragma unroll
  for (int d = 0; d < kTdDmsWarp; ++d) {
    const int j = j0 + warp * kTdDmsWarp + d;
    if (j >= a.n_dm) continue;
#pragma unroll
    for (int i = 0; i < kTdPer; ++i) {
      const int64_t n = t0 + lane + 32 * i;
      if (n < a.out_len) a.y[static_cast<int64_t>(j) * a.out_len + n] = acc[d][i];
    }
  }
}

// ---------------------------------------------------------------- 8-bit samples
constexpr int kPer8 = kTd8Samp / 128;  // words of four samples per lane and trial (4)
constexpr int kFlush = 256 / kTdCh;    // stages whose sums fit 16 bits
static_assert(kTdCh == kTdWarps && kTdDmsWarp == 4, "a warp fills a channel and adds four trials");

__global__ void __launch_bounds__(kTdThreads, 2) tdd8_kernel(const Tdd8Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // offsets of two stages, raw windows of two stages, the shifted copies of one
  int* const off_buf = reinterpret_cast<int*>(smem_raw);
  unsigned char* const raw_buf = smem_raw + 2 * sizeof(int) * kTdCh * kTdDms;
  const int stage_bytes = kTdCh * a.win;
  unsigned char* const copies = raw_buf + 2 * stage_bytes;
  const int blk = blockIdx.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.y) * kTd8Samp;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int n_stages = (a.n_chan + kTdCh - 1) / kTdCh;
  const int chunks = a.win / 16;  // 16-byte pieces of a window

  auto fill = [&](int st) {  // (tables are padded to whole stages)
    const int c0 = st * kTdCh;
    const int64_t row = (static_cast<int64_t>(blk) * n_stages * kTdCh + c0);
    int* off = off_buf + (st & 1) * kTdCh * kTdDms;
    if (threadIdx.x < kTdCh * kTdDms / 4)
      cp_async16(off + 4 * threadIdx.x, a.off + row * kTdDms + 4 * threadIdx.x);
    // warp = channel (base is a multiple of 16; zeros beyond the series and the
    // last channel)
    unsigned char* raw = raw_buf + (st & 1) * stage_bytes + warp * a.win;
    const int c = c0 + warp;
    const int64_t t_first = t0 + a.base[row + warp];
    for (int q = lane; q < chunks; q += 32) {
      const int64_t t = t_first + 16 * q;
      const int64_t left = c < a.n_chan ? a.n_t - t : 0;
      const int n = left >= 16 ? 16 : left > 0 ? static_cast<int>(left) : 0;
      const unsigned char* src = n > 0 ? a.x + static_cast<int64_t>(c) * a.pitch + t : a.x;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(raw + 16 * q)),
                   "l"(src), "r"(n)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  int sum[kTdDmsWarp][4 * kPer8];       // samples 4 (lane + 32 i) + e at [4 i + e]
  uint32_t half[kTdDmsWarp][2 * kPer8];  // their 16-bit sums: e = 0 | 2, then 1 | 3
#pragma unroll
  for (int d = 0; d < kTdDmsWarp; ++d) {
#pragma unroll
    for (int i = 0; i < 4 * kPer8; ++i) sum[d][i] = 0;
#pragma unroll
    for (int i = 0; i < 2 * kPer8; ++i) half[d][i] = 0;
  }
  auto flush = [&]() {
#pragma unroll
    for (int d = 0; d < kTdDmsWarp; ++d)
#pragma unroll
      for (int i = 0; i < kPer8; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          sum[d][4 * i + e] += half[d][2 * i + e] & 0xFFFF;
          sum[d][4 * i + e + 2] += half[d][2 * i + e] >> 16;
          half[d][2 * i + e] = 0;
        }
  };

  fill(0);
  for (int st = 0; st < n_stages; ++st) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the stage has arrived; the copies before it have been read
    if (st + 1 < n_stages) fill(st + 1);
    {
      // word w of copy e: bytes 4 w + e .. + 3 (the window's last word is spare)
      const uint32_t* raw =
          reinterpret_cast<const uint32_t*>(raw_buf + (st & 1) * stage_bytes + warp * a.win);
      uint32_t* out = reinterpret_cast<uint32_t*>(copies + 4 * warp * a.win);
      const int words = a.win / 4;
      for (int w = lane; w < words; w += 32) {
        const uint32_t lo = raw[w], hi = w + 1 < words ? raw[w + 1] : 0u;
        out[w] = lo;
#pragma unroll
        for (int e = 1; e < 4; ++e) out[e * words + w] = __funnelshift_r(lo, hi, 8 * e);
      }
    }
    __syncthreads();
    const int4* off = reinterpret_cast<const int4*>(off_buf + (st & 1) * kTdCh * kTdDms) + warp;
    const unsigned char* mine = copies + 4 * lane;
#pragma unroll
    for (int cc = 0; cc < kTdCh; cc += 2) {
      const int4 o0 = off[cc * (kTdDms / 4)], o1 = off[(cc + 1) * (kTdDms / 4)];
      const int u[kTdDmsWarp] = {o0.x, o0.y, o0.z, o0.w}, v[kTdDmsWarp] = {o1.x, o1.y, o1.z, o1.w};
#pragma unroll
      for (int d = 0; d < kTdDmsWarp; ++d) {
        const uint32_t* p = reinterpret_cast<const uint32_t*>(mine + u[d]);
        const uint32_t* q = reinterpret_cast<const uint32_t*>(mine + v[d]);
#pragma unroll
        for (int i = 0; i < kPer8; ++i) {
          const uint32_t x = p[32 * i], y = q[32 * i];
          half[d][2 * i] += __byte_perm(x, 0, 0x4240) + __byte_perm(y, 0, 0x4240);
          half[d][2 * i + 1] += __byte_perm(x, 0, 0x4341) + __byte_perm(y, 0, 0x4341);
        }
      }
    }
    if ((st + 1) % kFlush == 0) flush();
  }
  flush();

#pragma unroll
  for (int d = 0; d < kTdDmsWarp; ++d) {
    const int j = blk * kTdDms + warp * kTdDmsWarp + d;
    if (j >= a.n_dm) continue;
    float* row = a.y + static_cast<int64_t>(j) * a.out_len;
#pragma unroll
    for (int i = 0; i < kPer8; ++i) {
      const int64_t n = t0 + 4 * (lane + 32 * i);
      if (n + 3 < a.out_len && (reinterpret_cast<uintptr_t>(row + n) & 15) == 0) {
        *reinterpret_cast<float4*>(row + n) =
            make_float4(sum[d][4 * i], sum[d][4 * i + 1], sum[d][4 * i + 2], sum[d][4 * i + 3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (n + e < a.out_len) row[n + e] = static_cast<float>(sum[d][4 * i + e]);
      }
    }
  }
}

}  // namespace

size_t tdd_smem_bytes(int win) {
  return 2 * (sizeof(int) * kTdCh * kTdDms + sizeof(float) * static_cast<size_t>(kTdCh) * win);
}

cudaError_t tdd_prepare(int win) {
  return allow_smem(reinterpret_cast<const void*>(&tdd_kernel), tdd_smem_bytes(win));
}

cudaError_t launch_tdd(const TddArgs& a, cudaStream_t s) {
  if (a.n_dm <= 0 || a.out_len <= 0) return cudaSuccess;
  if (a.win % 4 != 0) return cudaErrorInvalidValue;  // keeps the buffers 16-byte aligned
  const int64_t t_blocks = (a.out_len + kTdSamp - 1) / kTdSamp;
  if (t_blocks > 65535) return cudaErrorInvalidConfiguration;
  dim3 grid((a.n_dm + kTdDms - 1) / kTdDms, static_cast<unsigned>(t_blocks));
  tdd_kernel<<<grid, kTdThreads, tdd_smem_bytes(a.win), s>>>(a);
  note_launches(1);
  return cudaGetLastError();
}

size_t tdd8_smem_bytes(int win) {
  return 2 * sizeof(int) * kTdCh * kTdDms + size_t(6) * kTdCh * win;
}

cudaError_t tdd8_prepare(int win) {
  return allow_smem(reinterpret_cast<const void*>(&tdd8_kernel), tdd8_smem_bytes(win));
}

cudaError_t launch_tdd8(const Tdd8Args& a, cudaStream_t s) {
  if (a.n_dm <= 0 || a.out_len <= 0) return cudaSuccess;
  if (a.win % 16 != 0 || a.pitch % 16 != 0 || (reinterpret_cast<uintptr_t>(a.x) & 15) != 0)
    return cudaErrorInvalidValue;  // (16-byte copies)
  const int64_t t_blocks = (a.out_len + kTd8Samp - 1) / kTd8Samp;
  if (t_blocks > 65535) return cudaErrorInvalidConfiguration;
  dim3 grid((a.n_dm + kTdDms - 1) / kTdDms, static_cast<unsigned>(t_blocks));
  tdd8_kernel<<<grid, kTdThreads, tdd8_smem_bytes(a.win), s>>>(a);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace fdd
