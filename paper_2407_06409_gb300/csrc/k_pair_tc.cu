// Adjoint pair matrix M' = P Q^T on the fifth-generation tensor cores, with the per-pair
// contraction against dT_LR/dr and dT_LR/dS~ (the derivative pieces of Sec. III.D, exact).
//
// P and Q (3 n_s rows, 3 n_freq (n_max - 2) columns per central atom) are cut into 5 digit
// planes.  One CTA owns a tile of 42 row sites (126 rows of P) by 16 column sites (48 rows of Q):
// the tcgen05 main loop (tc_sliced.cuh, M = 128, N = 48) accumulates the digit orders in tensor
// memory while warps 1-7 list the coupled pairs of the tile; the 8 warps then add the orders up in
// float-float (warp w: rows 32 (w % 4) .., columns 24 (w / 4) ..) into a tile in shared memory,
// and every thread runs the pair epilogue on listed pairs; per-site sums go to the force accumulator
// and the SCS-radius seed with one atomic per site and component.
//
// Everything between the accumulators and the atomics is float-float on the FP32 pipe (2^-46,
// against the 2^-35 of the digits), and only coupled pairs are evaluated: with an FP64 tile and
// epilogue over all pairs two thirds of a tile's time was FP64 issue (1024-atom step: 3.55 ms, now 1.22 ms).
// Two CTAs share an SM (256 tensor-memory columns and a two-slot ring each), so that one tile's
// copies and MMAs run under the other's epilogue; the 42 x 32 tile of one CTA per SM re-read less of
// P but left the SM at 24 % of its issue slots (1.77 against 1.33 ms).
// Values are scaled by powers of two to the tile's largest row exponents, so callers' weights of any
// magnitude stay inside the FP32 range.
#include "ff.cuh"
#include "tc_sliced.cuh"

#define PTC_SA 42   // row sites per tile (126 of the 128 MMA rows)
#define PTC_SB 16   // column sites per tile (N = 48)
#define PTC_NB 48
#define PTC_LD 49   // row stride of the float-float tile in shared memory
#define PTC_GL 17   // row-site stride of the per-pair results
#define PTC_BUF 2   // ring slots and tensor-memory columns: two CTAs per SM
#define PTC_COLS 256
#define PTC_PAIRS (PTC_SA * PTC_SB)

namespace {

// Contribution of a coupled pair to dL/dr (out[0..2]: g = dL/dr_t = -dL/dr_s) and the SCS-radius
// seed beta dL/dS~ (out[3]) from its block of the pair matrix and its record (lmbd_internal.cuh).
__device__ __forceinline__ void ptc_epilogue(const float4* rec, const ff (&acc)[3][3], ff (&out)[4]) {
  const float4 r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3];
  const ff x[3] = {ff_make(r0.x, r0.y), ff_make(r0.z, r0.w), ff_make(r1.x, r1.y)};
  const ff k3 = ff_make(r1.z, r1.w), k1 = ff_make(r2.x, r2.y), k2 = ff_make(r2.z, r2.w);
  const ff k4 = ff_make(r3.x, r3.y), k5 = ff_make(r3.z, r3.w);
  ff M[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    M[a][a] = acc[a][a];
#pragma unroll
    for (int b = 0; b < a; ++b) M[a][b] = M[b][a] = ff_scale(ff_add(acc[a][b], acc[b][a]), 0.5f);
  }
  ff Mr[3];
  float h = 0.f, l = 0.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float u = 0.f, v = 0.f;
#pragma unroll
    for (int b = 0; b < 3; ++b) ff_mac(u, v, M[a][b], x[b]);
    Mr[a] = ff_quick_two_sum(u, v);
    ff_mac(h, l, Mr[a], x[a]);
  }
  const ff rMr = ff_quick_two_sum(h, l), tr = ff_add(ff_add(M[0][0], M[1][1]), M[2][2]);
  auto dot2 = [](ff a, ff b, ff c, ff d) {   // a b + c d
    float u = 0.f, v = 0.f;
    ff_mac(u, v, a, b);
    ff_mac(u, v, c, d);
    return ff_quick_two_sum(u, v);
  };
  const ff radial = dot2(k1, rMr, k2, tr);
#pragma unroll
  for (int a = 0; a < 3; ++a) out[a] = dot2(radial, x[a], k3, Mr[a]);
  out[3] = dot2(k4, rMr, k5, tr);
}

__device__ __forceinline__ int ptc_k(int n) { return (n + 31) / 32 * 32; }

template <int S>
__global__ void __launch_bounds__(256, 2)
    k_pair_tc(Work w, DevParams p, int c0, int nb_max, int tiles_per_c) {
  using Sh = TcsShape<S, PTC_NB, PTC_BUF, PTC_COLS>;
  extern __shared__ unsigned char tc_dyn[];
  __shared__ TcsBarriers bar;
  __shared__ unsigned short list[PTC_PAIRS];
  __shared__ int listed, emax[3];
  const int c = c0 + blockIdx.x / tiles_per_c;
  const int tile = blockIdx.x % tiles_per_c;
  if (c >= w.n_atoms) return;
  const int ns = w.counts[c].ns;
  const int s0 = PTC_SA * (tile / nb_max), t0 = PTC_SB * (tile % nb_max);
  // tiles without a site pair s > t inside the sphere have nothing to do
  if (s0 >= ns || t0 >= ns || min(s0 + PTC_SA, ns) - 1 <= t0) return;
  const int K = ptc_k(w.ncol);
  // P and Q tile images of this centre
  const long long dig = w.off_sp[c] * 3LL * K * S;
  const TcsImage A{w.pdig + dig + 3LL * s0 * K * S, min(3 * PTC_SA, 3 * (ns - s0)), S};
  const TcsImage B{w.qdig + dig + 3LL * t0 * K * S, min(PTC_NB, 3 * (ns - t0)), S};
  const uint32_t sraw = tc_smem_u32(tc_dyn);
  const uint32_t sbase = (sraw + 1023u) & ~1023u;
  if (threadIdx.x == 64) {
    listed = 0;
    emax[0] = emax[1] = emax[2] = -1100;
  }
  const uint32_t tmem = tcs_setup<PTC_BUF, PTC_COLS>(bar);   // block barrier inside
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cb = (warp >> 2) * 24;
  const int* pe = w.pexp + w.off_sp[c] * 3 + 3 * s0;
  const int* qe = w.qexp + w.off_sp[c] * 3 + 3 * t0;
  const long long offs = w.off_s[c];
  // while thread 0 feeds the tensor cores, warps 1-7 list the coupled pairs (in any order: every
  // pair has its own result slot) and find the tile's largest row, column and X0 exponents
  if (warp >= 4) {
    const int row = tid - 128;
    int e = -1100;
    if (row < 3 * PTC_SA && 3 * s0 + row < 3 * ns) e = pe[row];
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(&emax[0], e);
  } else if (warp == 1 || warp == 2) {
    const int col = tid - 32;
    int e = -1100;
    if (col < PTC_NB && 3 * t0 + col < 3 * ns) e = qe[col];
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(&emax[1], e);
  }
  if (warp >= 1) {
    for (int k = tid - 32; k < PTC_PAIRS; k += 224) {
      const int sl = k / PTC_SB, s = s0 + sl, t = t0 + k % PTC_SB;
      bool in = false;
      if (s < ns && s > t) {
        in = pair_record(w, c, s, t)[1].z != 0.f;
        if (t == 0 && in) {   // central column: the pair matrix has the further term X0
          int e = 0;
          for (int u = 0; u < 9; ++u) e = max(e, oz_biased_exp(w.x0buf[(offs + s) * 9 + u]));
          atomicMax(&emax[2], e - 1022);
        }
      }
      const unsigned am = __activemask(), m = __ballot_sync(am, in);
      int at = 0;
      if (lane == __ffs(am) - 1) at = atomicAdd(&listed, __popc(m));
      at = __shfl_sync(am, at, __ffs(am) - 1) + __popc(m & ((1u << lane) - 1u));
      if (in) list[at] = (unsigned short)k;
    }
  }
  // sum over the digit orders of acc_g 2^(-7 g) (and over K chunks) as float-float.  The partial sum
  // before order g is a multiple of 2^(-7 (g - 1)), hence of the last place of acc_g 2^(-7 g) (an
  // integer below 2^24 times 2^(-7 g)), so the short two-sum is exact in either order of size.
  float Yh[24], Yl[24];
  bool first = true;
  TcsProgress pr;
  const bool ok = tcs_mainloop_with<S, PTC_NB, PTC_BUF, PTC_COLS>(
      [&](int s, uint32_t sA, uint32_t sB, uint64_t* mbar) {
        tc_mbar_expect_tx(mbar, tcs_image_bytes<S>(A) + tcs_image_bytes<S>(B));
        tcs_image_copy<S>(A, s, sA, Sh::kAPlane, mbar);
        tcs_image_copy<S>(B, s, sB, Sh::kBPlane, mbar);
      },
      (w.ncol + 15) / 16 * 16, sbase, bar, p.tc_wait, pr, [&]() {
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
        if (!first) y = ff_add(y, ff_make(Yh[j], Yl[j]));
        Yh[j] = y.hi;
        Yl[j] = y.lo;
      }
    }
    first = false;
  });
  tcs_teardown<PTC_BUF, PTC_COLS>(bar, !ok, pr, w.status);
  if (!ok) return;

  // scaled tile (126 x 48) and per-pair results (42 x 17 x 4) in the drained staging ring
  float2* Ms = reinterpret_cast<float2*>(tc_dyn + (sbase - sraw));
  float4* gp = reinterpret_cast<float4*>(Ms + 3 * PTC_SA * PTC_LD);
  const int erow = emax[0], ecol = emax[1];
  int scale = erow + ecol - 14;                    // the digits are 2^(er + ec - 14) sum acc_g 2^(-7 g)
  if (t0 == 0) scale = max(scale, emax[2]);
  const int half = scale >> 1;                     // 2^scale in two exact factors: it can pass the FP64 range
  const int row = 32 * (warp & 3) + lane;
  if (row < 3 * PTC_SA) {
    const bool rv = 3 * s0 + row < 3 * ns;
    const float fr = rv ? oz_down(min(pe[row] - erow, 0)) * oz_down(min(erow + ecol - 14 - scale, 0)) : 0.f;
#pragma unroll
    for (int j = 0; j < 24; ++j) {
      const int col = cb + j;
      const float f = rv && 3 * t0 + col < 3 * ns ? fr * oz_down(min(qe[col] - ecol, 0)) : 0.f;
      Ms[row * PTC_LD + col] = make_float2(Yh[j] * f, Yl[j] * f);
    }
  }
  for (int e = tid; e < 2 * PTC_SA * PTC_GL; e += blockDim.x) gp[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  if (t0 == 0) {   // central column: the further term X0
    const double d1 = oz_pow2(-half), d2 = oz_pow2(half - scale);
    for (int e = tid; e < 9 * PTC_SA; e += blockDim.x) {
      const int sl = e / 9, u = e % 9;
      if (s0 + sl >= ns) continue;
      float2& m = Ms[(3 * sl + u / 3) * PTC_LD + u % 3];
      const ff v = ff_add(ff_make(m.x, m.y), ff_from_double(w.x0buf[(offs + s0 + sl) * 9 + u] * d1 * d2));
      m = make_float2(v.hi, v.lo);
    }
    __syncthreads();
  }
  const int count = listed;
  for (int k = tid; k < count; k += blockDim.x) {
    const int e = list[k], sl = e / PTC_SB, tl = e % PTC_SB;
    ff a3[3][3];
#pragma unroll
    for (int al = 0; al < 3; ++al)
#pragma unroll
      for (int be = 0; be < 3; ++be) {
        const float2 v = Ms[(3 * sl + al) * PTC_LD + 3 * tl + be];
        a3[al][be] = ff_make(v.x, v.y);
      }
    ff o[4];
    ptc_epilogue(pair_record(w, c, s0 + sl, t0 + tl), a3, o);
    gp[2 * (sl * PTC_GL + tl)] = make_float4(o[0].hi, o[0].lo, o[1].hi, o[1].lo);
    gp[2 * (sl * PTC_GL + tl) + 1] = make_float4(o[2].hi, o[2].lo, o[3].hi, o[3].lo);
  }
  __syncthreads();
  // deterministic per-site sums, one thread per (site, component): row sites get -g, column sites +g
  const float2* g2 = reinterpret_cast<const float2*>(gp);
  const double u1 = oz_pow2(half), u2 = oz_pow2(scale - half);
  for (int e = tid; e < 4 * (PTC_SA + PTC_SB); e += blockDim.x) {
    const int d = e & 3, sd = e >> 2;
    const bool rs = sd < PTC_SA;
    const int l = rs ? sd : sd - PTC_SA, ss = (rs ? s0 : t0) + l;
    if (ss >= ns) continue;
    const int n = rs ? PTC_SB : PTC_SA, first = rs ? l * PTC_GL : l, step = rs ? 1 : PTC_GL;
    ff s2[2] = {ff_make(0.f, 0.f), ff_make(0.f, 0.f)};   // even and odd terms
#pragma unroll 4
    for (int o = 0; o < n; ++o) {
      const float2 v = g2[4 * (first + o * step) + d];
      s2[o & 1] = ff_add(s2[o & 1], ff_make(v.x, v.y));
    }
    const double sum = ff_to_double(ff_add(s2[0], s2[1])) * u1 * u2;
    if (sum == 0.0) continue;
    if (d == 3) atomicAdd(&w.rbar[offs + ss], sum);
    else atomicAdd(w.gacc + 3 * w.site_atom[(long long)c * w.site_cap + ss] + d, rs ? -sum : sum);
  }
}

static_assert(3 * PTC_SA == OZ_P_ROWS && PTC_NB == OZ_W_ROWS, "tiles of the digit images");
static_assert(TcsShape<5, PTC_NB, PTC_BUF, PTC_COLS>::kBytes <= 113 * 1024, "two staging rings exceed the shared memory of an SM");
static_assert(3 * PTC_SA * PTC_LD * 8 % 16 == 0, "pair results start on a 16-byte boundary");
static_assert((3 * PTC_SA * PTC_LD + 4 * PTC_SA * PTC_GL) * 8 <= TcsShape<5, PTC_NB, PTC_BUF, PTC_COLS>::kBytes - 1024,
              "tile and pair results must fit in the staging ring");

}  // namespace

// The tcgen05 pair kernel on the digit images of P and Q (written by the series adjoint, or here from
// FP64 P, Q).
void launch_pair_tc(const Work& w, const DevParams& p, int c0, int c1, int max_ns, cudaStream_t s) {
  if (c1 <= c0) return;
  launch_slice_pq(w, p, c0, c1, s);
  const int na = (max_ns + PTC_SA - 1) / PTC_SA, nb = (max_ns + PTC_SB - 1) / PTC_SB;
  using Sh = TcsShape<5, PTC_NB, PTC_BUF, PTC_COLS>;
  raise_smem_limit((const void*)k_pair_tc<5>, Sh::kBytes);
  k_pair_tc<5><<<(c1 - c0) * na * nb, 256, Sh::kBytes, s>>>(w, p, c0, nb, na * nb);
}
