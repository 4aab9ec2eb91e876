// Exact check of the tcgen05 products as the library runs them, on digit planes laid out as tile images
// (oz_tile_offset).  Exit status 0 when every value matches.
//
// Pair shape: tcs_mainloop_with<5, 48, 2, 256> with image copies, one block per tile of a matrix with full
// and partial tiles of 126 and 48 rows, K = 16, 0 and 1 chunk boundaries away from a multiple of 32 (columns of
// the image past K hold digits that must not count).  Digits up to 63: every FP32 accumulator of every digit
// order is an exact integer, compared with sum_{k + l = g} A_k B_l^T formed on the host.
//
// Chain kernel: k_chain_tc itself (copy, MMA and consumer roles) on four centres whose matrices have one to
// four row tiles, the last ones partial, one and two K chunks, with 1, 2 and 13 blocks for 16 tiles (slots,
// parities and accumulators carried from tile to tile).  sqrt(alpha) = 1 and random row and column exponents:
//   * one plane of T and one of W at a time with digits up to 127, |sum| < 2^23: the order k + l alone;
//   * all planes with digits -1, 0, 1: the recombined value has at most 45 bits.
// Both results are exact in float-float, so the outputs are compared with equality.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_2407_06409_gb300/csrc/k_chain_tc.cu"

// what the chain's launcher calls; this program launches the kernel itself
void launch_slice_w(const Work&, const DevParams&, int, int, int, int, cudaStream_t) {}
void raise_smem_limit(const void* f, size_t bytes) { cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); }

static unsigned short bf(int v) {
  __nv_bfloat16 h = __float2bfloat16((float)v);
  return *reinterpret_cast<unsigned short*>(&h);
}
template <class T>
static T* device(const std::vector<T>& v) {
  T* d = nullptr;
  cudaMalloc(&d, v.size() * sizeof(T));
  cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return d;
}
static int digit(int top) { return rand() % (2 * top + 1) - top; }

// ---- pair shape ------------------------------------------------------------------------------
constexpr int PS = 5, PN = OZ_W_ROWS, PB = 2, PC = 256;
__global__ void __launch_bounds__(256, 2) pair_shape(const unsigned short* A, const unsigned short* B, int ra, int rb, int K, int tb,
                                                     float* out, int* status) {
  using Sh = TcsShape<PS, PN, PB, PC>;
  extern __shared__ unsigned char dyn[];
  __shared__ TcsBarriers bar;
  const int r0 = blockIdx.x / tb * OZ_P_ROWS, c0 = blockIdx.x % tb * OZ_W_ROWS, KI = (K + 31) / 32 * 32;
  const TcsImage IA{A + (long long)r0 * KI * PS, min(OZ_P_ROWS, ra - r0), PS};
  const TcsImage IB{B + (long long)c0 * KI * PS, min(OZ_W_ROWS, rb - c0), PS};
  const uint32_t sbase = (tc_smem_u32(dyn) + 1023u) & ~1023u;
  const uint32_t tmem = tcs_setup<PB, PC>(bar);
  const int warp = threadIdx.x >> 5, row = 32 * (warp & 3) + (threadIdx.x & 31), cb = (warp >> 2) * 24;
  float* o = out + (long long)blockIdx.x * PS * 128 * PN;
  TcsProgress pr;
  const bool ok = tcs_mainloop_with<PS, PN, PB, PC>(
      [&](int s, uint32_t sA, uint32_t sB, uint64_t* mbar) {
        tc_mbar_expect_tx(mbar, tcs_image_bytes<PS>(IA) + tcs_image_bytes<PS>(IB));
        tcs_image_copy<PS>(IA, s, sA, Sh::kAPlane, mbar);
        tcs_image_copy<PS>(IB, s, sB, Sh::kBPlane, mbar);
      },
      K, sbase, bar, 1LL << 32, pr, [&]() {
        for (int g = 0; g < PS; ++g)
          for (int j8 = 0; j8 < 3; ++j8) {
            float v[8];
            tc_ld8(tcs_lane_addr(tmem, g * PN + cb + j8 * 8), v);
            for (int i = 0; i < 8; ++i) o[(g * 128 + row) * PN + cb + j8 * 8 + i] += v[i];
          }
      });
  tcs_teardown<PB, PC>(bar, !ok, pr, status);
}

static int check_pair(int ra, int rb, int K) {
  const int KI = (K + 31) / 32 * 32, ta = (ra + OZ_P_ROWS - 1) / OZ_P_ROWS, tb = (rb + OZ_W_ROWS - 1) / OZ_W_ROWS;
  std::vector<int> A((size_t)PS * ra * KI), B((size_t)PS * rb * KI);
  std::vector<unsigned short> Ai(A.size()), Bi(B.size());
  for (int k = 0; k < PS; ++k)
    for (int j = 0; j < KI; ++j) {
      for (int r = 0; r < ra; ++r) Ai[oz_tile_offset(r, j, k, PS, OZ_P_ROWS, ra, KI)] = bf(A[((size_t)k * ra + r) * KI + j] = digit(63));
      for (int r = 0; r < rb; ++r) Bi[oz_tile_offset(r, j, k, PS, OZ_W_ROWS, rb, KI)] = bf(B[((size_t)k * rb + r) * KI + j] = digit(63));
    }
  const size_t per = (size_t)PS * 128 * PN;
  std::vector<float> O(per * ta * tb, 0.f);
  std::vector<int> st(1, 0);
  unsigned short *dA = device(Ai), *dB = device(Bi);
  float* dO = device(O);
  int* dS = device(st);
  const int smem = TcsShape<PS, PN, PB, PC>::kBytes;
  raise_smem_limit((const void*)pair_shape, smem);
  const int K16 = (K + 15) / 16 * 16;   // the product stops there: zeros up to it
  for (int k = 0; k < PS; ++k)
    for (int j = K; j < K16; ++j)
      for (int r = 0; r < ra; ++r) {
        A[((size_t)k * ra + r) * KI + j] = 0;
        Ai[oz_tile_offset(r, j, k, PS, OZ_P_ROWS, ra, KI)] = 0;
      }
  cudaMemcpy(dA, Ai.data(), Ai.size() * 2, cudaMemcpyHostToDevice);
  pair_shape<<<ta * tb, 256, smem>>>(dA, dB, ra, rb, K16, tb, dO, dS);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaMemcpy(O.data(), dO, O.size() * 4, cudaMemcpyDeviceToHost);
  cudaMemcpy(st.data(), dS, 4, cudaMemcpyDeviceToHost);
  long bad = 0;
  for (int r = 0; r < ra; ++r)
    for (int c = 0; c < rb; ++c)
      for (int g = 0; g < PS; ++g) {
        long long ref = 0;
        for (int k = 0; k <= g; ++k)
          for (int j = 0; j < K16; ++j) ref += (long long)A[((size_t)k * ra + r) * KI + j] * B[((size_t)(g - k) * rb + c) * KI + j];
        const int tile = r / OZ_P_ROWS * tb + c / OZ_W_ROWS;
        bad += (long long)O[tile * per + (g * 128 + r % OZ_P_ROWS) * PN + c % OZ_W_ROWS] != ref;
      }
  printf("pair shape %d x %d x %d: %s, status %d, %ld wrong\n", ra, rb, K, cudaGetErrorString(e), st[0], bad);
  cudaFree(dA); cudaFree(dB); cudaFree(dO); cudaFree(dS);
  return e != cudaSuccess || st[0] || bad;
}

// ---- chain kernel ----------------------------------------------------------------------------
// plane_t, plane_w: the only planes that are not zero (-1: all of them)
template <int S>
static int check_chain(int grid, int n_freq, int plane_t, int plane_w, int top) {
  const int sites[4] = {5, 43, 160, 107}, nc = 4, st = 6, ncv = 3 * n_freq, nq = n_freq + 1, tiles = 4, tk = 480;
  std::vector<Counts> counts(nc);
  std::vector<long long> off_s(nc + 1, 0), off_tr(nc + 1, 0);
  for (int c = 0; c < nc; ++c) {
    counts[c] = Counts{1, sites[c], sites[c], 0};
    off_s[c + 1] = off_s[c] + sites[c];
    off_tr[c + 1] = off_tr[c] + (3 * sites[c] + 63) / 64 * 64;
  }
  std::vector<unsigned short> tdig((size_t)st * off_tr[nc] * tk, 0), wdig((size_t)nc * 48 * S * tk, 0);
  std::vector<int> texp(off_tr[nc], 0), wexp(nc * 48, 0);
  std::vector<std::vector<int>> T(nc), W(nc);
  for (int c = 0; c < nc; ++c) {
    const int N = 3 * sites[c], K = (N + 31) / 32 * 32;
    T[c].assign((size_t)st * N * K, 0);
    W[c].assign((size_t)S * 48 * K, 0);
    for (int k = 0; k < st; ++k)
      if (plane_t < 0 || k == plane_t)
        for (int r = 0; r < N; ++r)
          for (int j = 0; j < N; ++j)
            tdig[st * off_tr[c] * tk + oz_tile_offset(r, j, k, st, OZ_T_ROWS, N, K)] = bf(T[c][((size_t)k * N + r) * K + j] = digit(top));
    for (int k = 0; k < S; ++k)
      if (plane_w < 0 || k == plane_w)
        for (int r = 0; r < 48; ++r)
          for (int j = 0; j < N; ++j)
            wdig[(size_t)c * 48 * S * tk + oz_tile_offset(r, j, k, S, OZ_W_ROWS, 48, K)] = bf(W[c][((size_t)k * 48 + r) * K + j] = digit(top));
    for (int r = 0; r < N; ++r) texp[off_tr[c] + r] = rand() % 21 - 10;
    for (int r = 0; r < 48; ++r) wexp[c * 48 + r] = rand() % 21 - 10;
  }
  std::vector<double> dsq((size_t)off_s[nc] * nq, 1.0), out((size_t)off_s[nc] * 3 * ncv, 0.0);
  std::vector<int> status(4, 0);
  Work w{};
  DevParams p{};
  w.n_atoms = nc;
  w.counts = device(counts);
  w.off_s = device(off_s);
  w.off_tr = device(off_tr);
  w.tdig = device(tdig);
  w.wdig = device(wdig);
  w.texp = device(texp);
  w.wexp = device(wexp);
  w.dsq = device(dsq);
  w.vkr = device(out);
  w.vstride = 0;
  w.tk = tk;
  w.status = device(status);
  p.n_freq = n_freq;
  p.nq = nq;
  p.tc_wait = 1LL << 32;
  const size_t smem = TcsShape<S, CTC_NB>::kBytes;
  raise_smem_limit((const void*)k_chain_tc<S>, smem);
  k_chain_tc<S><<<grid, CTC_THREADS, smem>>>(w, p, 1, 0, nc * tiles, tiles, st);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaMemcpy(out.data(), w.vkr, out.size() * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(status.data(), w.status, 4, cudaMemcpyDeviceToHost);
  long bad = 0;
  for (int c = 0; c < nc; ++c) {
    const int N = 3 * sites[c], K = (N + 31) / 32 * 32;
    for (int r = 0; r < N; ++r)
      for (int v = 0; v < ncv; ++v) {
        long long Y = 0;   // sum_g acc_g 2^(7 (S - 1 - g))
        for (int k = 0; k < S; ++k)
          for (int l = 0; k + l < S; ++l) {
            if ((plane_t >= 0 && k != plane_t) || (plane_w >= 0 && l != plane_w)) continue;
            long long acc = 0;
            for (int j = 0; j < N; ++j) acc += (long long)T[c][((size_t)k * N + r) * K + j] * W[c][((size_t)l * 48 + v) * K + j];
            Y += acc * (1LL << (7 * (S - 1 - k - l)));
          }
        const double ref = std::ldexp((double)Y, texp[off_tr[c] + r] + wexp[c * 48 + v] - 14 - 7 * (S - 1));
        bad += out[(off_s[c] * 3 + r) * ncv + v] != ref;
      }
  }
  printf("chain S %d, grid %d, %d frequencies, planes %d %d: %s, status %d, %ld wrong\n", S, grid, n_freq, plane_t, plane_w,
         cudaGetErrorString(e), status[0], bad);
  cudaFree(w.counts); cudaFree(w.off_s); cudaFree(w.off_tr); cudaFree(w.tdig); cudaFree(w.wdig); cudaFree(w.texp);
  cudaFree(w.wexp); cudaFree((void*)w.dsq); cudaFree(w.vkr); cudaFree(w.status);
  return e != cudaSuccess || status[0] || bad;
}

int main() {
  srand(11);
  int rc = 0;
  rc |= check_pair(126, 48, 32);
  rc |= check_pair(126 + 3, 48 + 3, 16);
  rc |= check_pair(3, 3, 144);
  rc |= check_pair(2 * 126 + 60, 2 * 48 + 27, 256 + 41);
  rc |= check_pair(126, 96, 9);
  rc |= check_pair(127, 48, 512);
  for (int grid : {1, 2, 13}) {
    rc |= check_chain<6>(grid, 16, -1, -1, 1);
    rc |= check_chain<5>(grid, 11, -1, -1, 1);
  }
  for (int k = 0; k < 6; ++k)
    for (int l = 0; k + l < 6; ++l) rc |= check_chain<6>(3, 12, k, l, 127);
  for (int k = 0; k < 5; ++k)
    for (int l = 0; k + l < 5; ++l) rc |= check_chain<5>(3, 1, k, l, 127);
  printf("%s\n", rc ? "FAILED" : "all exact");
  return rc;
}
