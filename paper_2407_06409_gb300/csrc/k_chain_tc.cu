// Krylov chain step v_{m+1} = D (T_LR W) of Eq. E_k on the fifth-generation tensor cores.
//
// Same sliced arithmetic as the warp-level kernel (ozaki.cuh): T_LR and W = D v_m are cut into
// S signed 7-bit digit planes, digit pairs (k, l) with k + l <= S - 1 are multiplied on the
// tensor cores with FP32 accumulation, one accumulator per digit order, K chunks of at most 256.
// A tile is 128 rows of one central atom's T_LR times all 48 columns of W (M = 128, N = 48).
//
// Reading the digit planes of T_LR bounds a step (9.2 GB at 4096 atoms and 6 digits: 1.4 ms at the
// measured copy rate).  One CTA per SM stays resident and works through a contiguous range of
// tiles with separate roles, so that copies never wait for an epilogue:
//   * warp 9 (one thread) fills the three-slot ring of the tiles one after another;
//   * warp 8 (one thread) issues the MMAs and commits each slot and each K chunk;
//   * warps 0-7 read a finished chunk from tensor memory, add the digit orders up in float-float
//     (warp w: rows 32 (w % 4) .., columns 24 (w / 4) ..), release it, and after the tile's last chunk
//     scale by the row and column exponents and by D while the next tile is under way.
// The digit planes lie in memory as images of the ring's tiles (ozaki.cuh): a stage is one bulk copy for
// T_LR (48 KB) and one for W; the last tile of a centre copies only the rows it has.  With a CTA per tile
// (set-up, ring fill and epilogue in series) a 6-digit step took 0.71 ms per 1024 atoms, now
// 0.545 ms.
// Every wait is bounded (DevParams::tc_wait); a role that gives up stops the others, the block's
// copies and MMAs in flight are waited for (bounded), tensor memory is freed and
// LMBD_FLAG_TIMEOUT set.
#include <algorithm>

#include "ff.cuh"
#include "tc_sliced.cuh"

#define CTC_NB 48

namespace {

__device__ __forceinline__ int ctc_k(int n) { return (n + 31) / 32 * 32; }

#define CTC_THREADS 320

// Barriers and shared state of the roles.
struct ChainShared {
  uint64_t full[TCS_NBUF];    // copies of a slot landed
  uint64_t empty[TCS_NBUF];   // MMAs reading a slot done
  uint64_t acc_full;          // accumulators of a K chunk complete
  uint64_t acc_free;          // ... and read by the eight consumer warps
  uint32_t tmem;
  int stop;                   // a wait ran out
  int issued, committed, chunks;   // stages copied, stages and chunks committed (tear-down)
};

template <int S>
__global__ void __launch_bounds__(CTC_THREADS, 1)
    k_chain_tc(Work w, DevParams p, int m, int c0, int items, int tiles_per_c, int st) {
  using Sh = TcsShape<S, CTC_NB>;
  constexpr int kPerChunk = OZ_KCHUNK / TCS_KS;
  extern __shared__ unsigned char tc_dyn[];
  __shared__ ChainShared sh;
  const uint32_t sbase = (tc_smem_u32(tc_dyn) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {
    tc_alloc(&sh.tmem, TCS_TMEM_COLS);
    tc_relinquish();
  }
  if (threadIdx.x == 32) {
#pragma unroll
    for (int b = 0; b < TCS_NBUF; ++b) {
      tc_mbar_init(&sh.full[b], 1);
      tc_mbar_init(&sh.empty[b], 1);
    }
    tc_mbar_init(&sh.acc_full, 1);
    tc_mbar_init(&sh.acc_free, 8);
    tc_mbar_init_fence();
    sh.stop = 0;
    sh.issued = sh.committed = sh.chunks = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem;
  volatile int* stop = &sh.stop;
  const long long budget = p.tc_wait;
  // this CTA's items (centre, tile): a contiguous range, so that long and short tiles mix
  const int i0 = (int)((long long)items * blockIdx.x / gridDim.x), i1 = (int)((long long)items * (blockIdx.x + 1) / gridDim.x);

  if (warp == 9) {
    if (lane == 0) {
      int g = 0;   // stages copied
      bool ok = true;
      for (int it = i0; it < i1 && ok; ++it) {
        const int c = c0 + it / tiles_per_c, row0 = (it % tiles_per_c) * TCS_M;
        const int N = 3 * w.counts[c].ns, K = ctc_k(N);
        if (row0 >= N) continue;
        const TcsImage A{w.tdig + w.off_tr[c] * st * w.tk + (long long)row0 * K * st, min(TCS_M, N - row0), st};
        const TcsImage B{w.wdig + (long long)c * CTC_NB * S * w.tk, CTC_NB, S};
        const uint32_t bytes = tcs_image_bytes<S>(A) + tcs_image_bytes<S>(B);
        for (int s = 0; s < K / TCS_KS; ++s, ++g) {
          const int slot = g % TCS_NBUF;
          if (g >= TCS_NBUF && !tc_mbar_wait_or_stop(&sh.empty[slot], (g / TCS_NBUF - 1) & 1, budget, stop)) {
            ok = false;
            break;
          }
          const uint32_t sA = sbase + slot * Sh::kSlot;
          tc_mbar_expect_tx(&sh.full[slot], bytes);
          tcs_image_copy<S>(A, s, sA, Sh::kAPlane, &sh.full[slot]);
          tcs_image_copy<S>(B, s, sA + S * Sh::kAPlane, Sh::kBPlane, &sh.full[slot]);
        }
      }
      sh.issued = g;
    }
  } else if (warp == 8) {
    if (lane == 0) {
      int g = 0, ch = 0;   // stages and chunks committed
      bool ok = true;
      for (int it = i0; it < i1 && ok; ++it) {
        const int c = c0 + it / tiles_per_c, row0 = (it % tiles_per_c) * TCS_M;
        const int N = 3 * w.counts[c].ns;
        if (row0 >= N) continue;
        const int nst = ctc_k(N) / TCS_KS;
        for (int s0 = 0; s0 < nst && ok; s0 += kPerChunk) {
          if (ch > 0 && !tc_mbar_wait_or_stop(&sh.acc_free, (ch - 1) & 1, budget, stop)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int s1 = min(nst, s0 + kPerChunk);
          for (int s = s0; s < s1; ++s) {
            const int slot = g % TCS_NBUF;
            if (!tc_mbar_wait_or_stop(&sh.full[slot], (g / TCS_NBUF) & 1, budget, stop)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sA = sbase + slot * Sh::kSlot, sB = sA + S * Sh::kAPlane;
#pragma unroll
            for (int kk = 0; kk < TCS_KS / 16; ++kk)
#pragma unroll
              for (int k = 0; k < S; ++k) {
                const uint64_t ad = tc_desc_k_sw64(sA + k * Sh::kAPlane + kk * 32);
#pragma unroll
                for (int l0 = 0; l0 < S - k; l0 += Sh::kPlanesPerMma) {
                  const int n = (S - k - l0) < Sh::kPlanesPerMma ? (S - k - l0) : Sh::kPlanesPerMma;
                  const uint64_t bd = tc_desc_k_sw64(sB + l0 * Sh::kBPlane + kk * 32);
                  // at the start of a chunk the products of A plane 0 (every order) restart the sums
                  tc_mma_bf16(tmem + (uint32_t)((k + l0) * Sh::kGroupCols), ad, bd, tc_idesc_bf16(TCS_M, n * CTC_NB),
                              (s == s0 && kk == 0 && k == 0) ? 0u : 1u);
                }
              }
            tc_commit(&sh.empty[slot]);
            ++g;
          }
          if (ok) {
            tc_commit(&sh.acc_full);
            ++ch;
          }
        }
      }
      sh.committed = g;
      sh.chunks = ch;
    }
  } else {
    const int cb = (warp >> 2) * 24, rw = 32 * (warp & 3) + lane;
    const int ncv = 3 * p.n_freq;
    int ch = 0;
    bool ok = true;
    for (int it = i0; it < i1 && ok; ++it) {
      const int c = c0 + it / tiles_per_c, row = (it % tiles_per_c) * TCS_M + rw;
      const int N = 3 * w.counts[c].ns;
      if (row - rw >= N) continue;
      const int nst = ctc_k(N) / TCS_KS;
      // sum over the digit orders of acc_g 2^(-7 g), and over the chunks.  The partial sum before
      // order g is a multiple of 2^(-7 (g - 1)), hence of the last place of acc_g 2^(-7 g) (an
      // integer below 2^24 times 2^(-7 g)), so the short two-sum is exact in either order of size.
      float Yh[24], Yl[24];
      for (int s0 = 0; s0 < nst; s0 += kPerChunk, ++ch) {
        // one lane polls for its warp
        int done = 1;
        if (lane == 0) done = tc_mbar_wait_or_stop(&sh.acc_full, ch & 1, budget, stop);
        if (!__shfl_sync(0xffffffffu, done, 0)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int j8 = 0; j8 < 3; ++j8) {
          float h[8], l[8];
#pragma unroll
          for (int g = 0; g < S; ++g) {
            float v[8];
            tc_ld8(tcs_lane_addr(tmem, g * Sh::kGroupCols + cb + j8 * 8), v);
            const float down = __int_as_float((127 - 7 * g) << 23);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if (g == 0) {
                h[i] = v[i];
                l[i] = 0.f;
              } else {
                const float sum = __fmaf_rn(v[i], down, h[i]);
                l[i] = __fadd_rn(l[i], __fmaf_rn(v[i], down, -__fsub_rn(sum, h[i])));
                h[i] = sum;
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int j = j8 * 8 + i;
            ff y = ff_quick_two_sum(h[i], l[i]);
            if (s0 > 0) y = ff_add(y, ff_make(Yh[j], Yl[j]));
            Yh[j] = y.hi;
            Yl[j] = y.lo;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) tc_mbar_arrive(&sh.acc_free);
      }
      if (!ok) break;
      if (row >= N) continue;
      const long long offs = w.off_s[c];
      double* Vout = w.vkr + (long long)m * w.vstride + (offs * 3) * ncv + (long long)row * ncv;
      const double* dsq = w.dsq + (offs + row / 3) * p.nq;
      const int er = w.texp[w.off_tr[c] + row];
      const int* we = w.wexp + (long long)c * 48;
#pragma unroll
      for (int j3 = 0; j3 < 8; ++j3) {   // the three columns of a frequency
        const int col = cb + 3 * j3;
        if (col >= ncv) break;
        const ff d = ff_split(dsq[col / 3 + 1]);
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int j = 3 * j3 + u;
          Vout[col + u] = ff_join(ff_mul(d, ff_make(Yh[j], Yl[j])), er + we[col + u] - 14);
        }
      }
    }
  }
  // tear-down: after an abort, wait (bounded) for the copies and MMAs in flight and their commits, so
  // that nothing lands in shared or tensor memory after the block is gone; then free tensor memory
  tc_fence_before();
  __syncthreads();
  if (sh.stop && threadIdx.x == 0) {
    atomicOr(w.status, LMBD_FLAG_TIMEOUT);
    for (int s = sh.committed; s < sh.issued; ++s)
      tc_mbar_wait(&sh.full[s % TCS_NBUF], (s / TCS_NBUF) & 1, TCS_WAIT_CYCLES);
    if (sh.committed > 0)
      tc_mbar_wait(&sh.empty[(sh.committed - 1) % TCS_NBUF], ((sh.committed - 1) / TCS_NBUF) & 1, TCS_WAIT_CYCLES);
    if (sh.chunks > 0) tc_mbar_wait(&sh.acc_full, (sh.chunks - 1) & 1, TCS_WAIT_CYCLES);
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tc_dealloc(tmem, TCS_TMEM_COLS);
  }
}

static_assert(TcsShape<6, CTC_NB>::kBytes <= 232448, "staging ring exceeds the shared memory of a CTA");

}  // namespace

size_t chain_tc_smem(int digits) { return digits == 6 ? TcsShape<6, CTC_NB>::kBytes : TcsShape<5, CTC_NB>::kBytes; }

bool launch_chain_tc(const Work& w, const DevParams& p, int m, int c0, int c1, int max_ns, int digits, int st,
                     cudaStream_t s) {
  if (c1 <= c0) return true;
  if (digits != 5 && digits != 6) return false;
  launch_slice_w(w, p, m, c0, c1, digits, s);
  const int tiles = (3 * max_ns + TCS_M - 1) / TCS_M;
  const int items = (c1 - c0) * tiles, grid = std::min(items, w.sms);
  if (digits == 6) {
    raise_smem_limit((const void*)k_chain_tc<6>, TcsShape<6, CTC_NB>::kBytes);
    k_chain_tc<6><<<grid, CTC_THREADS, TcsShape<6, CTC_NB>::kBytes, s>>>(w, p, m, c0, items, tiles, st);
  } else {
    raise_smem_limit((const void*)k_chain_tc<5>, TcsShape<5, CTC_NB>::kBytes);
    k_chain_tc<5><<<grid, CTC_THREADS, TcsShape<5, CTC_NB>::kBytes, s>>>(w, p, m, c0, items, tiles, st);
  }
  return true;
}
