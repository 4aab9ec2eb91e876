// Stage 1, mixed precision: local SCS solves (Sec. III.B, Eq. local_pol) for every
// central atom k and frequency omega_q, FP64 results.
//
//   B_K = diag(1/alpha_bar_i) + T_SR,K,ij (i, j in K1),  d_K,i = 1 - sum_{j in K2} T_SR,K,ij alpha_bar_j
//   X = B_K^-1 d_K,  alpha_K,i = Tr(X_i)/3,  alpha_I,k = alpha_K,k
//   T_SR,K,ij = F(r) [A0(r) I + B0(r) r r^T],  F = f_inner f_SR (1 - f(r, S_ij)),
//   A0 = g/r^3, B0 = (h~ - 3 g)/r^5 (Eqs. T_SR, g-func, h-func, written out in lmbd_internal.cuh)
//
// Design for GB300, whose FP64 pipe runs at 1/70 of FP32:
//  * the pairs (i in K1, j in K1 u K2) with r_ij < r_SCS are listed once per central atom
//    with their frequency-independent geometry and damping F, dF/dr (k_scs_count/k_scs_fill);
//  * erf and exp of r/sigma_ij are evaluated once per atom pair and frequency (k_pair_radial,
//    FP64), not once per local system holding the pair; the local systems read the table;
//  * a system is solved by conjugate gradients in FP32 and the FP64 solution recovered by
//    iterative refinement: the residual d - B X is formed in float-float from the sparse pair
//    list, corrections come from further FP32 solves (mixed-precision refinement, Wilkinson/Moler);
//  * the adjoint solve B lambda = dL/dX is the same kernel; the contraction with dB/dr, dd/dr
//    runs pair by pair over all frequencies from the stored radial terms (k_scs_contract).
#include <algorithm>

#include "ff.cuh"
#include "lmbd_internal.cuh"

// pair predicate shared by the counting and filling kernels (identical FP64 arithmetic)
__device__ __forceinline__ bool scs_pair_in(const double* xs, int ld, int i, int j, double rc2, double& rx,
                                            double& ry, double& rz, double& r2) {
  rx = xs[j] - xs[i];
  ry = xs[ld + j] - xs[ld + i];
  rz = xs[2 * ld + j] - xs[2 * ld + i];
  r2 = __dadd_rn(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)), __dmul_rn(rz, rz));
  return r2 < rc2;
}

// FP32 screen of the same predicate: pairs farther than a relative 1e-4 from the radius are
// decided in FP32 (the FP32 error of r^2 is below 1e-5 r_SCS^2 for sites within 27 r_SCS of
// the centre); the others take the FP64 test, so the decision is always the FP64 one.
__device__ __forceinline__ bool scs_pair_in_screened(const float* xf, const double* xs, int ld, int i, int j,
                                                     float lo2, float hi2, double rc2) {
  const float dx = xf[j] - xf[i], dy = xf[ld + j] - xf[ld + i], dz = xf[2 * ld + j] - xf[2 * ld + i];
  const float r2f = dx * dx + dy * dy + dz * dz;
  if (r2f < lo2) return true;
  if (r2f > hi2) return false;
  double rx, ry, rz, r2;
  return scs_pair_in(xs, ld, i, j, rc2, rx, ry, rz, r2);
}

// ---------------------------------------------------------------------------------------
// pair lists: count (before the workspace is sized) and fill
// ---------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_scs_count(Work w, DevParams p, int max_n12) {
  extern __shared__ double smem_d[];
  double* xs = smem_d;                 // 3 x max_n12
  float* xf = (float*)(xs + 3 * max_n12);   // 3 x max_n12, FP32 copies
  __shared__ int cnt_k1k1, cnt_k2;
  const int c = blockIdx.x;
  if (c >= w.n_atoms) return;
  const Counts cn = w.counts[c];
  const int n1 = cn.n1, n12 = cn.n12;
  const long long sbase = (long long)c * w.site_cap;
  const int tid = threadIdx.x;
  for (int s = tid; s < n12; s += blockDim.x)
    for (int d = 0; d < 3; ++d) {
      const double v = w.site_x[3 * (sbase + s) + d];
      xs[d * max_n12 + s] = v;
      xf[d * max_n12 + s] = (float)v;
    }
  if (tid == 0) { cnt_k1k1 = 0; cnt_k2 = 0; }
  __syncthreads();
  const double rc2 = p.r_scs * p.r_scs;
  const float lo2 = (float)(rc2 * (1.0 - 1e-4)), hi2 = (float)(rc2 * (1.0 + 1e-4));
  int a = 0, b = 0;
  const int nkk = n1 * (n1 - 1) / 2;
  for (int e = tid; e < nkk; e += blockDim.x) {
    int i = (int)((sqrtf(8.0f * e + 1.0f) + 1.0f) * 0.5f);
    while (i * (i - 1) / 2 > e) --i;
    while ((i + 1) * i / 2 <= e) ++i;
    int j = e - i * (i - 1) / 2;
    a += scs_pair_in_screened(xf, xs, max_n12, i, j, lo2, hi2, rc2);
  }
  const int n2 = n12 - n1;
  for (int e = tid; e < n1 * n2; e += blockDim.x) {
    int i = e / n2, j = n1 + e % n2;
    b += scs_pair_in_screened(xf, xs, max_n12, i, j, lo2, hi2, rc2);
  }
  atomicAdd(&cnt_k1k1, a);
  atomicAdd(&cnt_k2, b);
  __syncthreads();
  if (tid == 0) {
    w.pcount[2 * c] = cnt_k1k1 + cnt_k2;   // unique pairs
    w.pcount[2 * c + 1] = 2 * cnt_k1k1;    // adjacency entries (both directions of K1-K1 pairs)
  }
}

// One block per central atom.  The K1 pairs of all rows come first (row i: its partners j < i,
// ascending), then the K2 pairs of all rows (partners ascending), so that kernels take one kind
// with whole warps; adjacency rows list every K1 partner j != i (ascending) with the index of the
// shared pair.
__global__ void __launch_bounds__(256) k_scs_fill(Work w, DevParams p, int c0, int max_n12, int max_n1) {
  extern __shared__ double smem_d[];
  double* xs = smem_d;                             // 3 x max_n12
  int* pid = (int*)(xs + 3 * max_n12);             // max_n1 x max_n1 (pair index, -1 = none)
  int* rowk1 = pid + max_n1 * max_n1;              // max_n1
  int* rowcnt = rowk1 + max_n1;                    // max_n1
  int* k1start = rowcnt + max_n1;                  // max_n1 + 1: first K1 pair of each row
  int* k2start = k1start + max_n1 + 1;             // max_n1 + 1: first K2 pair of each row
  int* adjcnt = k2start + max_n1 + 1;              // max_n1
  int* adjstart = adjcnt + max_n1;                 // max_n1 + 1
  int* k2cnt = adjstart + max_n1 + 1;              // max_n12
  float* xf = (float*)(k2cnt + max_n12);           // 3 x max_n12, FP32 copies of xs
  const int c = c0 + blockIdx.x;
  if (c >= w.n_atoms) return;
  const Counts cn = w.counts[c];
  const int n1 = cn.n1, n12 = cn.n12;
  const long long sbase = (long long)c * w.site_cap;
  const long long offp = w.off_p[c], offa = w.off_a[c], rbase = w.off_k1[c] + c;
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32, nw = blockDim.x / 32;
  for (int s = tid; s < n12; s += blockDim.x)
    for (int d = 0; d < 3; ++d) {
      const double v = w.site_x[3 * (sbase + s) + d];
      xs[d * max_n12 + s] = v;
      xf[d * max_n12 + s] = (float)v;
    }
  for (int e = tid; e < n1 * n1; e += blockDim.x) pid[(e / n1) * max_n1 + e % n1] = -1;
  __syncthreads();
  const double rc2 = p.r_scs * p.r_scs;
  const float lo2 = (float)(rc2 * (1.0 - 1e-4)), hi2 = (float)(rc2 * (1.0 + 1e-4));
  // phase 1: per-row counts
  for (int i = warp; i < n1; i += nw) {
    int k1 = 0, k2 = 0;
    for (int j0 = 0; j0 < i; j0 += 32) {
      int j = j0 + lane;
      bool in = j < i && scs_pair_in_screened(xf, xs, max_n12, i, j, lo2, hi2, rc2);
      k1 += __popc(__ballot_sync(0xffffffffu, in));
    }
    for (int j0 = n1; j0 < n12; j0 += 32) {
      int j = j0 + lane;
      bool in = j < n12 && scs_pair_in_screened(xf, xs, max_n12, i, j, lo2, hi2, rc2);
      k2 += __popc(__ballot_sync(0xffffffffu, in));
    }
    if (lane == 0) { rowk1[i] = k1; rowcnt[i] = k2; }
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int i = 0; i < n1; ++i) { k1start[i] = run; run += rowk1[i]; }
    k1start[n1] = run;
    for (int i = 0; i < n1; ++i) { k2start[i] = run; run += rowcnt[i]; }
    k2start[n1] = run;
  }
  __syncthreads();
  // phase 2a: pairs in order (row, partner)
  for (int i = warp; i < n1; i += nw) {
    for (int pass = 0; pass < 2; ++pass) {
      int jb = pass == 0 ? 0 : n1, je = pass == 0 ? i : n12;
      int pos = pass == 0 ? k1start[i] : k2start[i];
      for (int j0 = jb; j0 < je; j0 += 32) {
        int j = j0 + lane;
        bool in = j < je && scs_pair_in_screened(xf, xs, max_n12, i, j, lo2, hi2, rc2);
        unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {
          int slot = pos + __popc(m & ((1u << lane) - 1u));
          long long q = offp + slot;
          w.pr_ij[2 * q] = i;
          w.pr_ij[2 * q + 1] = j;
          if (pass == 0) pid[i * max_n1 + j] = slot;
        }
        pos += __popc(m);
      }
    }
    if (lane == 0) {
      w.prow[rbase + i] = k1start[i];
      w.prow_k2[rbase + i] = k2start[i];
    }
  }
  if (tid == 0) {
    w.prow[rbase + n1] = k1start[n1];
    w.prow_k2[rbase + n1] = k2start[n1];
  }
  __syncthreads();
  // phase 2b, one thread per pair: its entry in the atom-pair radial table, geometry and damping.
  // Searching the table here, with every lane a pair, instead of by the few coupled lanes of phase 2a
  // took three quarters of this kernel's instructions away; distance, exponential and divisions
  // run in FP64, the products of the damping in float-float (1024 atoms: 1.14 -> 0.77 ms).
  const ff d_ff = ff_from_double(p.d), ibuf_ff = ff_from_double(1.0 / p.r_buf), iin_ff = ff_from_double(1.0 / p.r_inner);
  for (int t = tid; t < k2start[n1]; t += blockDim.x) {
    const long long q = offp + t;
    const int2 ij = reinterpret_cast<const int2*>(w.pr_ij)[q];
    const int i = ij.x, j = ij.y;
    const int ai = w.site_atom[sbase + i], aj = w.site_atom[sbase + j];
    double rx, ry, rz, r2;
    scs_pair_in(xs, max_n12, i, j, rc2, rx, ry, rz, r2);
    // the same atom pair in the radial table: the site of atom aj at displacement r = x_j - x_i in
    // atom ai's own K1 list (periodic images of one atom are far apart, so an FP32 match is
    // unambiguous; none only if r ties r_SCS to rounding)
    int gi = -1;
    {
      const long long ab = (long long)ai * w.site_cap;   // site lists start on 16-byte boundaries
      const int na = w.counts[ai].n1;
      const int4* list = reinterpret_cast<const int4*>(w.site_atom + ab);
      const float fx = (float)rx, fy = (float)ry, fz = (float)rz;
      auto match = [&](int u) {
        const double* xt = w.site_x + 3 * (ab + u);
        const float dx = (float)xt[0] - fx, dy = (float)xt[1] - fy, dz = (float)xt[2] - fz;
        if (dx * dx + dy * dy + dz * dz < 1e-4f) gi = (int)(w.off_k1[ai] + u);
      };
#pragma unroll 2
      for (int u = 0; u < na && gi < 0; u += 4) {
        const int4 a = __ldg(list + u / 4);
        if (a.x == aj && u > 0) match(u);
        if (a.y == aj && u + 1 < na && gi < 0) match(u + 1);
        if (a.z == aj && u + 2 < na && gi < 0) match(u + 2);
        if (a.w == aj && u + 3 < na && gi < 0) match(u + 3);
      }
    }
    w.pr_ga[q] = make_int2(gi, aj);
    // 1/r from one reciprocal square root; the Fermi damping (Eq. damping-function) through
    // x = r / S_vdW, its r-derivative f (1 - f) d / S_vdW as f (1 - f) d x / r
    const double ird = rsqrt(r2);
    const double r = r2 * ird;
    const double x = r / (p.beta * (w.rvdw[ai] + w.rvdw[aj]));
    const double f = 1.0 / (1.0 + exp(-p.d * (x - 1.0)));
    const ff ir = ff_split(ird), omf = ff_split(1.0 - f);
    const ff dfr = ff_mul(ff_mul(ff_split(f * (1.0 - f)), d_ff), ff_mul(ff_split(x), ir));
    // F = f_inner f_SR (1 - f); c = f_inner f_SR and its derivative where either differs from 1
    ff F = omf, dF = ff_neg(dfr);
    const double tb = r - (p.r_scs - p.r_buf);
    const bool buffer = tb >= 0.0, inner = j >= n1 && r < p.r_inner;
    if (buffer || inner) {
      ff cs = ff_make(1.f, 0.f), dc = ff_make(0.f, 0.f);
      if (buffer) {
        const ff u = ff_mul(ff_split(tb), ibuf_ff), u2 = ff_mul(u, u);
        cs = ff_add(cs, ff_sub(ff_scale(ff_mul(u2, u), 2.f), ff_scale(u2, 3.f)));
        dc = ff_mul(ff_scale(ff_sub(u2, u), 6.f), ibuf_ff);
        if (!(r < p.r_scs)) cs = dc = ff_make(0.f, 0.f);
      }
      if (inner) {
        const ff u = ff_mul(ff_split(r), iin_ff), u2 = ff_mul(u, u);
        const ff fi = ff_sub(ff_scale(u2, 3.f), ff_scale(ff_mul(u2, u), 2.f));
        const ff di = ff_mul(ff_scale(ff_sub(u, u2), 6.f), iin_ff);
        dc = ff_add(ff_mul(di, cs), ff_mul(fi, dc));
        cs = ff_mul(fi, cs);
      }
      F = ff_mul(cs, omf);
      dF = ff_sub(ff_mul(dc, omf), ff_mul(cs, dfr));
    }
    float4* gf = reinterpret_cast<float4*>(w.pr_gff + 6 * q);
    const ff gx = ff_split(rx), gy = ff_split(ry), gz = ff_split(rz);
    gf[0] = make_float4(gx.hi, gx.lo, gy.hi, gy.lo);
    gf[1] = make_float4(gz.hi, gz.lo, F.hi, F.lo);
    gf[2] = make_float4(dF.hi, dF.lo, ir.hi, ir.lo);
  }
  __syncthreads();
  // phase 3: adjacency rows (K1 partners of every coupled site, both directions)
  for (int i = warp; i < n1; i += nw) {
    int k = 0;
    for (int j0 = 0; j0 < n1; j0 += 32) {
      int j = j0 + lane;
      bool in = j < n1 && j != i && (j < i ? pid[i * max_n1 + j] : pid[j * max_n1 + i]) >= 0;
      k += __popc(__ballot_sync(0xffffffffu, in));
    }
    if (lane == 0) adjcnt[i] = k;
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int i = 0; i < n1; ++i) { adjstart[i] = run; run += adjcnt[i]; }
    adjstart[n1] = run;
  }
  __syncthreads();
  for (int i = warp; i < n1; i += nw) {
    int pos = adjstart[i];
    for (int j0 = 0; j0 < n1; j0 += 32) {
      int j = j0 + lane;
      int pp = -1;
      if (j < n1 && j != i) pp = j < i ? pid[i * max_n1 + j] : pid[j * max_n1 + i];
      unsigned m = __ballot_sync(0xffffffffu, pp >= 0);
      if (pp >= 0) {
        long long q = offa + pos + __popc(m & ((1u << lane) - 1u));
        w.adj[2 * q] = j;
        w.adj[2 * q + 1] = pp;
      }
      pos += __popc(m);
    }
    if (lane == 0) w.arow[rbase + i] = adjstart[i];
  }
  if (tid == 0) w.arow[rbase + n1] = adjstart[n1];
  // phase 4: for every K2 site the pairs in which it is the partner, ascending (rows ascending): a
  // counting sort by the whole block, whose lists (a few entries each) are then put in order.  One warp
  // going through the rows took as long as the rest of the kernel.
  const int kb = k2start[0], ke = k2start[n1];
  for (int j = n1 + tid; j < n12; j += blockDim.x) k2cnt[j] = 0;
  __syncthreads();
  for (int t = kb + tid; t < ke; t += blockDim.x) atomicAdd(&k2cnt[w.pr_ij[2 * (offp + t) + 1]], 1);
  __syncthreads();
  if (warp == 0) {
    int run = 0;
    for (int j0 = n1; j0 < n12; j0 += 32) {
      const int j = j0 + lane, v = j < n12 ? k2cnt[j] : 0;
      int x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (j < n12) w.k2ptr[sbase + j] = k2cnt[j] = run + x - v;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) w.k2ptr[sbase + n12] = run;
  }
  __syncthreads();
  for (int t = kb + tid; t < ke; t += blockDim.x) w.k2rev[offp + atomicAdd(&k2cnt[w.pr_ij[2 * (offp + t) + 1]], 1)] = t;
  __threadfence_block();
  __syncthreads();
  for (int j = n1 + tid; j < n12; j += blockDim.x) {   // k2cnt[j] is the end of list j now
    int* list = w.k2rev + offp;
    const int first = w.k2ptr[sbase + j], end = k2cnt[j];
    for (int u = first + 1; u < end; ++u) {
      const int v = list[u];
      int k = u;
      for (; k > first && list[k - 1] > v; --k) list[k] = list[k - 1];
      list[k] = v;
    }
  }
}

// Radial terms of T_SR (see lmbd_internal.cuh): A0 = g/r^3, B0 = (h~ - 3g)/r^5 and their
// r-derivatives, with x = r / sigma_ij.  For x >= 8, erf(x) = 1 and x^3 exp(-x^2) < 1e-25 in
// double precision, so g = 1 and h~ = 0 exactly; the transcendental calls are skipped there.
__device__ __forceinline__ void tsr_radial_fast(double r, double ir, double s2, double& A0, double& B0,
                                                double& dA0, double& dB0) {
  const double x = r * rsqrt(s2);
  double g = 1.0, ht = 0.0;
  if (x < 8.0) {
    const double two_over_sqrtpi = 1.1283791670955126;
    const double ex = exp(-x * x);
    g = erf(x) - two_over_sqrtpi * x * ex;
    ht = 2.0 * two_over_sqrtpi * x * x * x * ex;
  }
  const double ir2 = ir * ir, ir3 = ir2 * ir, ir4 = ir2 * ir2;
  A0 = g * ir3;
  B0 = (ht - 3.0 * g) * ir4 * ir;
  dA0 = (ht - 3.0 * g) * ir4;
  dB0 = (15.0 * g - 5.0 * ht - 2.0 * x * x * ht) * ir4 * ir2;
}

// Radial terms per atom pair and frequency: for atom a and every site s (1 <= s < n1) of its
// own K1 list, A0, B0 and their r-derivatives at sigma_ab(omega_q).  They depend on |r_ab|
// and sigma_a, sigma_b only, so every central atom whose local system holds the pair reads
// them instead of evaluating erf and exp again (about 50 local systems share each pair).
__global__ void __launch_bounds__(128) k_pair_radial(Work w, DevParams p) {
  const int a = blockIdx.x;
  if (a >= w.n_atoms) return;
  const int n1 = w.counts[a].n1;
  const long long ab = (long long)a * w.site_cap, base = w.off_k1[a];
  // alpha_bar and 1/alpha_bar as float-float, for the solves
  for (int q = threadIdx.x; q < p.nqs; q += blockDim.x) {
    const double v = w.abar[(long long)a * p.nqs + q];
    const ff f = ff_from_double(v), g = ff_from_double(1.0 / v);
    w.abff[(long long)a * p.nqs + q] = make_float2(f.hi, f.lo);
    w.iabff[(long long)a * p.nqs + q] = make_float2(g.hi, g.lo);
  }
  for (int e = threadIdx.x; e < n1 * p.nqs; e += blockDim.x) {
    const int s = e / p.nqs, q = e % p.nqs;
    if (s == 0) continue;
    const double* x = w.site_x + 3 * (ab + s);
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(x[0], x[0]), __dmul_rn(x[1], x[1])), __dmul_rn(x[2], x[2]));
    const double r = sqrt(r2);
    const int b = w.site_atom[ab + s];
    const double sa = w.sig[(long long)a * p.nqs + q], sb = w.sig[(long long)b * p.nqs + q];
    double A0, B0, dA0, dB0;
    tsr_radial_fast(r, 1.0 / r, sa * sa + sb * sb, A0, B0, dA0, dB0);
    const long long o = (base + s) * p.nqs + q;
    w.rad_ab[2 * o] = A0;
    w.rad_ab[2 * o + 1] = B0;
    const double v[4] = {A0, B0, dA0, dB0};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const ff t = ff_split(v[u]);
      w.rad_ff[4 * o + u] = make_float2(t.hi, t.lo);
    }
  }
}

// FP64 geometry and damping of pair pq of centre c (LU fallback, and pairs without a table entry).
struct PairGeo64 {
  double x[3], r, ir, F;
};
__device__ PairGeo64 pair_geo64(const Work& w, const DevParams& p, int c, long long pq) {
  const long long sbase = (long long)c * w.site_cap;
  const int i = w.pr_ij[2 * pq], j = w.pr_ij[2 * pq + 1];
  const double *xi = w.site_x + 3 * (sbase + i), *xj = w.site_x + 3 * (sbase + j);
  PairGeo64 g;
  for (int d = 0; d < 3; ++d) g.x[d] = xj[d] - xi[d];
  const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(g.x[0], g.x[0]), __dmul_rn(g.x[1], g.x[1])), __dmul_rn(g.x[2], g.x[2]));
  g.ir = rsqrt(r2);
  g.r = r2 * g.ir;
  double fsr, dfsr, fin = 1.0, dfin = 0.0;
  cutoff_buf(g.r, p.r_scs, p.r_buf, fsr, dfsr);
  if (j >= w.counts[c].n1) finner(g.r, p.r_inner, fin, dfin);
  const double x = g.r / (p.beta * (w.rvdw[w.site_atom[sbase + i]] + w.rvdw[w.site_atom[sbase + j]]));
  g.F = fin * fsr * (1.0 - 1.0 / (1.0 + exp(-p.d * (x - 1.0))));
  return g;
}

// FP64 damped radial terms F A0, F B0 of the pair at SCS frequency q: from the atom-pair table, or
// evaluated when the pair has no table entry
__device__ __forceinline__ void pair_rad64(const Work& w, const DevParams& p, int c, int q, long long pq,
                                           const PairGeo64& g, double& fa, double& fb) {
  const int gi = w.pr_ga[pq].x;
  double A0, B0;
  if (gi >= 0) {
    const double* ra = w.rad_ab + 2 * ((long long)gi * p.nqs + q);
    A0 = ra[0];
    B0 = ra[1];
  } else {
    const long long sbase = (long long)c * w.site_cap;
    const int i = w.pr_ij[2 * pq], j = w.pr_ij[2 * pq + 1];
    const double si = w.sig[(long long)w.site_atom[sbase + i] * p.nqs + q];
    const double sj = w.sig[(long long)w.site_atom[sbase + j] * p.nqs + q];
    double dA0, dB0;
    tsr_radial_fast(g.r, g.ir, si * si + sj * sj, A0, B0, dA0, dB0);
  }
  fa = g.F * A0;
  fb = g.F * B0;
}

// the right-hand side of Eq. local_pol in FP64 (LU fallback), alpha_bar from global memory
__device__ void scs2_build_rhs64(const Work& w, const DevParams& p, int c, int n1, int q, double* rhs) {
  const long long offp = w.off_p[c], rbase = w.off_k1[c] + c, sbase = (long long)c * w.site_cap;
  for (int e = threadIdx.x; e < 3 * n1; e += blockDim.x) {
    const int i = e / 3, cc = e % 3;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, ad = 0.0;
    const int b = w.prow_k2[rbase + i], en = w.prow_k2[rbase + i + 1];
    for (int t = b; t < en; ++t) {
      const long long pq = offp + t;
      const int j = w.pr_ij[2 * pq + 1];
      const PairGeo64 g = pair_geo64(w, p, c, pq);
      double fa, fb;
      pair_rad64(w, p, c, q, pq, g, fa, fb);
      const double abj = w.abar[(long long)w.site_atom[sbase + j] * p.nqs + q];
      ad += abj * fa;
      const double wb = abj * fb * g.x[cc];
      a0 += wb * g.x[0];
      a1 += wb * g.x[1];
      a2 += wb * g.x[2];
    }
    double* y = rhs + 9 * i;
    y[cc] = (cc == 0 ? 1.0 : 0.0) - a0 - (cc == 0 ? ad : 0.0);
    y[3 + cc] = (cc == 1 ? 1.0 : 0.0) - a1 - (cc == 1 ? ad : 0.0);
    y[6 + cc] = (cc == 2 ? 1.0 : 0.0) - a2 - (cc == 2 ? ad : 0.0);
  }
}

// ---------------------------------------------------------------------------------------
// local screening solves: conjugate gradients in FP32 inside a float-float refinement
// ---------------------------------------------------------------------------------------
// The scaled matrix A^(1/2) B A^(1/2), A = diag(alpha_bar), is I plus the damped dipole coupling:
// its eigenvalues lie in about [0.3, 1.9] at the benchmark density (and tend to 1 at high
// frequency), so conjugate gradients gain a digit in two to three steps: 13 steps to 2e-6 at
// omega = 0, 2 at the highest node.
//
// A thread owns one site: a system is S = 1..3 warps (NC = 3: all three right-hand sides per thread), or three such
// groups (NC = 1: a right-hand side each, independent until the end).  The only large array is the
// packed triangle of pair couplings (11 KB at |K1| = 52 where a packed factor took 49 KB): twelve
// or more systems per SM instead of two or three.
//
// The product B p is dense over the sites: for each partner j its position and p_j are broadcast
// from shared memory (three 16-byte loads, one wavefront each) and a thread reads the scalar
// couplings of its own site from the triangle without bank conflicts (triangular numbers run
// through all residues).  The sparse form (a gather of p_j by adjacency) needs half the FMAs but
// about thirty shared-memory wavefronts per entry.
//
// An FP32 Cholesky factor per system (block-wide, 16-wide blocks, in shared memory) took 32.5 ms
// forward and 22.8 ms for the adjoint solves and their contraction per 4096-atom step, at 40 % of
// the issue slots (two block barriers per block column, serial substitutions, two or three
// systems per SM); this kernel takes 14.0 + 7.7 ms and k_scs_contract 4.1 ms.  It is bound by the
// FP32 issue rate and the latency of the pair loads in the float-float residuals (60 % of the
// issue slots).  A warp per system with packed FP32 pairs (fma.rn.f32x2) measured 17.4 + 10.5 ms:
// the pairs cost as many moves as they save, with half the warps.  The steps grow with the condition
// number, where a factor's time does not: with alpha0 raised until the smallest eigenvalue of B nears zero
// (jittered lattices and chains, 36 to 1000 atoms, all polarisabilities still positive) the forward
// solves of 1000 atoms rise from 4.1 to 5.6 ms (the factors took 10.7) and those of 64 atoms from 0.63 to 0.97 (1.10),
// so no such call is slower than with the factor.  Beyond CG_MAXIT a system goes to LU.
#define CG_MAXIT 250          // steps of one inner solve; systems that need more go to LU
#define CG_OUTER 12           // refinement steps

// What every thread reads of a partner site: position (bohr) and the search direction or correction
// p of the three columns.
struct CgSite {
  float4 a;   // x, y, z, p[2][2]
  float4 b;   // p[0][0..2], p[1][0]
  float4 c;   // p[1][1..2], p[2][0..1]
};
struct CgSmem {
  CgSite* site;
  float2* F;      // packed lower triangle with diagonal: scaled F A0, F B0 of the pair (1, 0 on it)
  float* s;       // sqrt(alpha_bar)
  float* part;    // 4 x 3 x 3 partial sums of the warps of a group
};
__host__ __device__ inline size_t cg_smem_bytes(int ld) {
  return (size_t)ld * (sizeof(CgSite) + sizeof(float)) + (size_t)ld * (ld + 1) / 2 * sizeof(float2) + 36 * sizeof(float);
}
__device__ inline CgSmem cg_carve(unsigned char* base, int ld) {
  CgSmem s;
  s.site = reinterpret_cast<CgSite*>(base);
  s.F = reinterpret_cast<float2*>(s.site + ld);
  s.s = reinterpret_cast<float*>(s.F + ld * (ld + 1) / 2);
  s.part = s.s + ld;
  return s;
}
// component a of column c in a site record, and the same as an address (c, a may be run-time)
__device__ __forceinline__ float* cg_slot(CgSite& t, int c, int a) {
  return reinterpret_cast<float*>(&t) + (3 * c + a == 8 ? 3 : 4 + 3 * c + a);
}

// The S warps that share a system's columns: synchronisation, sums and maxima over them.
template <int S>
struct CgGroup {
  int id, warp;   // group (NC = 1: the column), warp within it
  __device__ __forceinline__ void sync() const {
    if (S == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + id), "n"(32 * S) : "memory");
  }
  // slot: one of four partial-sum areas; the same one may be used again after one more sync()
  template <int NC>
  __device__ __forceinline__ void sum(float (&v)[NC], const CgSmem& sm, int slot) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int c = 0; c < NC; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
    if (S == 1) return;
    float* part = sm.part + 9 * slot;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int c = 0; c < NC; ++c) part[3 * (id + c) + warp] = v[c];
    sync();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      v[c] = part[3 * (id + c)];
#pragma unroll
      for (int k = 1; k < S; ++k) v[c] += part[3 * (id + c) + k];
    }
  }
  template <int NC>
  __device__ __forceinline__ void max(float (&v)[NC], const CgSmem& sm, int slot) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int c = 0; c < NC; ++c) v[c] = fmaxf(v[c], __shfl_xor_sync(0xffffffffu, v[c], o));
    if (S == 1) return;
    float* part = sm.part + 9 * slot;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int c = 0; c < NC; ++c) part[3 * (id + c) + warp] = v[c];
    sync();
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
      for (int k = 0; k < S; ++k) v[c] = fmaxf(v[c], part[3 * (id + c) + k]);
  }
};

// (I + scaled coupling) x = r by conjugate gradients from x = 0 for the NC columns of a group; the
// thread holds the rows of its site i (r = 0 past the last site).  Each column is scaled by a
// power of two to unit size first (its squares stay in range) and stops when its residual has
// fallen by tol.  Returns false (uniformly) when a direction of non-positive curvature shows up
// (matrix not positive definite), on a non-finite value or after CG_MAXIT steps.
template <int S, int NC>
__device__ bool cg_solve(const CgSmem& sm, const CgGroup<S>& grp, int n1, int site, int c0, float tol,
                         float (&r)[NC][3], float (&x)[NC][3]) {
  const bool act = site < n1;
  const int i = act ? site : n1 - 1;
  const float4 own = sm.site[i].a;
  float p[NC][3], rr[NC], thr[NC], unit[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) unit[c] = fmaxf(fabsf(r[c][0]), fmaxf(fabsf(r[c][1]), fabsf(r[c][2])));
  grp.template max<NC>(unit, sm, 0);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    // 2^-e with the largest entry in [2^e, 2^(e+1)), from its biased exponent (0 for a zero column)
    const int eb = min(max((__float_as_int(unit[c]) >> 23) & 0xff, 1), 253);
    unit[c] = __int_as_float(eb << 23);
    const float down = __int_as_float((254 - eb) << 23);
    rr[c] = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      p[c][a] = r[c][a] = r[c][a] * down;
      x[c][a] = 0.f;
      rr[c] += r[c][a] * r[c][a];
    }
  }
  grp.template sum<NC>(rr, sm, 1);
  bool ok = true;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    thr[c] = tol * tol * rr[c];
    ok = ok && rr[c] < 3e38f;   // also false for NaN
  }
  for (int it = 0; ok; ++it) {
    bool more = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) more = more || rr[c] > thr[c];
    if (!more) break;
    if (it == CG_MAXIT) return false;
    // every thread of the group is past the product of the step before (its sums synchronise)
    if (S == 1) __syncwarp();
    if (act) {
      if (NC == 3) {
        sm.site[i].a.w = p[2 % NC][2];
        sm.site[i].b = make_float4(p[0][0], p[0][1], p[0][2], p[1 % NC][0]);
        sm.site[i].c = make_float4(p[1 % NC][1], p[1 % NC][2], p[2 % NC][0], p[2 % NC][1]);
      } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) *cg_slot(sm.site[i], c0, a) = p[0][a];
      }
    }
    grp.sync();
    float q[NC][3];
#pragma unroll
    for (int c = 0; c < NC; ++c) q[c][0] = q[c][1] = q[c][2] = 0.f;
    // q += (3 x 3 coupling of the pair) p_j
    auto partner = [&](int j, const float2 f) {
      CgSite& t = sm.site[j];
      const float4 ta = t.a;
      float pj[NC][3];
      if (NC == 3) {
        const float4 tb = t.b, tc = t.c;
        pj[0][0] = tb.x; pj[0][1] = tb.y; pj[0][2] = tb.z;
        pj[1 % NC][0] = tb.w; pj[1 % NC][1] = tc.x; pj[1 % NC][2] = tc.y;
        pj[2 % NC][0] = tc.z; pj[2 % NC][1] = tc.w; pj[2 % NC][2] = ta.w;
      } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) pj[0][a] = *cg_slot(t, c0, a);
      }
      const float dx = ta.x - own.x, dy = ta.y - own.y, dz = ta.z - own.z;
      const float ux = f.y * dx, uy = f.y * dy, uz = f.y * dz;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float u = fmaf(dz, pj[c][2], fmaf(dy, pj[c][1], dx * pj[c][0]));
        q[c][0] = fmaf(ux, u, fmaf(f.x, pj[c][0], q[c][0]));
        q[c][1] = fmaf(uy, u, fmaf(f.x, pj[c][1], q[c][1]));
        q[c][2] = fmaf(uz, u, fmaf(f.x, pj[c][2], q[c][2]));
      }
    };
    // the row of site i in the triangle is contiguous up to j = i, then the column steps by j + 1;
    // only the 32 partners around the warp's own sites need the choice
    const int row = i * (i + 1) / 2, lo = S == 1 ? 0 : min(32 * grp.warp, n1), hi = S == 1 ? n1 : min(lo + 32, n1);
    int j = 0;
    if (S > 1)
#pragma unroll 4
      for (; j < lo; ++j) partner(j, sm.F[row + j]);
    int col = j * (j + 1) / 2 + i;
#pragma unroll 4
    for (; j < hi; ++j) {
      partner(j, sm.F[j <= i ? row + j : col]);
      col += j + 1;
    }
    if (S > 1)
#pragma unroll 4
      for (; j < n1; ++j) {
        partner(j, sm.F[col]);
        col += j + 1;
      }
    float pq[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
      for (int a = 0; a < 3; ++a) q[c][a] = act ? q[c][a] : 0.f;
      pq[c] = p[c][0] * q[c][0] + p[c][1] * q[c][1] + p[c][2] * q[c][2];
    }
    grp.template sum<NC>(pq, sm, 2);
    float rn[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const bool go = rr[c] > thr[c];
      if (go && !(pq[c] > 0.f)) ok = false;
      const float al = go ? rr[c] / pq[c] : 0.f;
      rn[c] = 0.f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        x[c][a] += al * p[c][a];
        r[c][a] -= al * q[c][a];
        rn[c] += r[c][a] * r[c][a];
      }
    }
    if (!ok) return false;
    grp.template sum<NC>(rn, sm, 3);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const bool go = rr[c] > thr[c];
      const float be = go ? rn[c] / rr[c] : 0.f;
      if (go) rr[c] = rn[c];
      ok = ok && rr[c] < 3e38f;
#pragma unroll
      for (int a = 0; a < 3; ++a) p[c][a] = r[c][a] + be * p[c][a];
    }
  }
#pragma unroll
  for (int c = 0; c < NC; ++c)
#pragma unroll
    for (int a = 0; a < 3; ++a) x[c][a] *= unit[c];
  return ok;
}

// R <- R - B y for the FP32 vector y = p of the site records (the group's columns), in float-float arithmetic on the
// FP32 pipe: F A0 y_j + F B0 r (r . y_j) over the adjacency row of every coupled site, error-free
// products and compensated sums (ff.cuh), 1/alpha_bar on the diagonal.  Called with the FP32
// solution it leaves the residual with an error ~2^-46 |B||x|, called with a correction it
// carries the residual on.  Two lanes per (site, column), each half of the row; the halves are
// combined in a fixed order.
template <int S, int NC>
__device__ void cg_residual_update(const Work& w, const DevParams& p, int c, int q, int n1, int c0, int nk1, int gt,
                                   const CgSmem& sm, double* R) {
  const long long offp = w.off_p[c], offa = w.off_a[c], rbase = w.off_k1[c] + c, sbase = (long long)c * w.site_cap;
  const float4* rad = w.pr_rad4 + offp * p.nqs + (long long)q * nk1;
  const int items = 2 * NC * n1;   // item e: half e % 2 of (site, column)
  for (int base = 0; base < items; base += 32 * S) {
    const int e = base + gt;
    const bool on = e < items;
    const int half = e & 1, cc = c0 + (NC == 1 ? 0 : (e >> 1) % NC), i = on ? (e >> 1) / NC : 0;
    float h0 = 0.f, h1 = 0.f, h2 = 0.f, l0 = 0.f, l1 = 0.f, l2 = 0.f;
    if (on) {
      if (half == 0) {
        const float2 ab = w.iabff[(long long)w.site_atom[sbase + i] * p.nqs + q];
        const ff ia = ff_make(ab.x, ab.y);
        const ff a = ff_scale(ia, *cg_slot(sm.site[i], cc, 0)), b = ff_scale(ia, *cg_slot(sm.site[i], cc, 1)),
                 d = ff_scale(ia, *cg_slot(sm.site[i], cc, 2));
        h0 = a.hi; l0 = a.lo; h1 = b.hi; l1 = b.lo; h2 = d.hi; l2 = d.lo;
      }
      const int b0 = w.arow[rbase + i], e0 = w.arow[rbase + i + 1];
      const int mid = b0 + (e0 - b0 + 1) / 2;
      const int tb = half == 0 ? b0 : mid, te = half == 0 ? mid : e0;
      // the loads of an entry depend on its index pair: the indices run two entries ahead and the
      // data one entry ahead of the arithmetic
      const int2* ap = reinterpret_cast<const int2*>(w.adj) + offa;
      const float4* gp = reinterpret_cast<const float4*>(w.pr_gff) + 3 * offp;
      int2 ad = make_int2(0, 0), an = ad;
      float4 n0, n1v, nf;
      if (tb < te) {
        an = __ldg(ap + tb);
        n0 = __ldg(gp + 3 * an.y); n1v = __ldg(gp + 3 * an.y + 1); nf = rad[an.y];
        ad = __ldg(ap + min(tb + 1, te - 1));
      }
      for (int t = tb; t < te; ++t) {
        const float4 g0 = n0, g1 = n1v, f = nf;     // rx, ry | rz, F (hi, lo each) | F A0, F B0
        CgSite& sj = sm.site[an.x];
        const float3 d = make_float3(*cg_slot(sj, cc, 0), *cg_slot(sj, cc, 1), *cg_slot(sj, cc, 2));
        an = ad;
        n0 = __ldg(gp + 3 * an.y); n1v = __ldg(gp + 3 * an.y + 1); nf = rad[an.y];
        ad = __ldg(ap + min(t + 2, te - 1));
        // s = r . y
        const float p0 = __fmul_rn(g0.x, d.x), p1 = __fmul_rn(g0.z, d.y), p2 = __fmul_rn(g1.x, d.z);
        float s0 = __fmaf_rn(g0.y, d.x, __fmaf_rn(g0.x, d.x, -p0));
        const float s1 = __fmaf_rn(g0.w, d.y, __fmaf_rn(g0.z, d.y, -p1));
        const float s2 = __fmaf_rn(g1.y, d.z, __fmaf_rn(g1.x, d.z, -p2));
        const ff a = ff_two_sum(p0, p1), b = ff_two_sum(a.hi, p2);
        s0 = __fadd_rn(__fadd_rn(s0, s1), __fadd_rn(s2, __fadd_rn(a.lo, b.lo)));
        const ff s = ff_quick_two_sum(b.hi, s0);
        // u = F B0 s
        const float uh = __fmul_rn(f.z, s.hi);
        const float ul = __fmaf_rn(f.w, s.hi, __fmaf_rn(f.z, s.lo, __fmaf_rn(f.z, s.hi, -uh)));
        auto add = [&](float& h, float& l, float dk, float rh, float rl) {
          const float v = __fmul_rn(f.x, dk);
          const float ve = __fmaf_rn(f.y, dk, __fmaf_rn(f.x, dk, -v));
          const float z = __fmul_rn(uh, rh);
          const float ze = __fmaf_rn(ul, rh, __fmaf_rn(uh, rl, __fmaf_rn(uh, rh, -z)));
          const ff m = ff_two_sum(h, v), n = ff_two_sum(m.hi, z);
          h = n.hi;
          l = __fadd_rn(l, __fadd_rn(__fadd_rn(m.lo, n.lo), __fadd_rn(ve, ze)));
        };
        add(h0, l0, d.x, g0.x, g0.y);
        add(h1, l1, d.y, g0.z, g0.w);
        add(h2, l2, d.z, g1.x, g1.y);
      }
    }
    const ff o0 = ff_make(__shfl_xor_sync(0xffffffffu, h0, 1), __shfl_xor_sync(0xffffffffu, l0, 1));
    const ff o1 = ff_make(__shfl_xor_sync(0xffffffffu, h1, 1), __shfl_xor_sync(0xffffffffu, l1, 1));
    const ff o2 = ff_make(__shfl_xor_sync(0xffffffffu, h2, 1), __shfl_xor_sync(0xffffffffu, l2, 1));
    if (on && half == 0) {
      double* Ri = R + 9 * i + cc;
      Ri[0] -= ff_to_double(ff_add(ff_quick_two_sum(h0, l0), ff_quick_two_sum(o0.hi, o0.lo)));
      Ri[3] -= ff_to_double(ff_add(ff_quick_two_sum(h1, l1), ff_quick_two_sum(o1.hi, o1.lo)));
      Ri[6] -= ff_to_double(ff_add(ff_quick_two_sum(h2, l2), ff_quick_two_sum(o2.hi, o2.lo)));
    }
  }
}

// Damped radial terms F A0, F B0 of pair t (of centre c) at SCS frequency q in float-float: F times
// the atom-pair table entry, on the FP32 pipe.
__device__ __noinline__ void pair_rad_slow(const Work& w, const DevParams& p, int c, int q, long long pq, ff& fa,
                                           ff& fb) {
  double da, db;   // no table entry (a distance that ties r_SCS to rounding): evaluate in FP64
  pair_rad64(w, p, c, q, pq, pair_geo64(w, p, c, pq), da, db);
  fa = ff_from_double(da);
  fb = ff_from_double(db);
}
// the table row of entry gi at frequency q: A0, B0 (row 0 where there is no entry)
__device__ __forceinline__ float4 rad_row(const Work& w, const DevParams& p, int gi, int q) {
  return __ldg(reinterpret_cast<const float4*>(w.rad_ff + 4 * ((long long)max(gi, 0) * p.nqs + q)));
}
__device__ __forceinline__ void pair_rad_ff(const Work& w, const DevParams& p, int c, int q, long long pq, int gi,
                                            float4 ra, ff F, ff& fa, ff& fb) {
  if (gi >= 0) {
    fa = ff_mul(F, ff_make(ra.x, ra.y));
    fb = ff_mul(F, ff_make(ra.z, ra.w));
  } else {
    pair_rad_slow(w, p, c, q, pq, fa, fb);
  }
}

// Right-hand side d_i = 1 - sum_{j in K2} T_SR,ij alpha_bar_j (Eq. local_pol) into R: float-float
// sums (fixed order) of the six distinct entries of the symmetric block, four lanes per site.
__device__ void cg_build_rhs(const Work& w, const DevParams& p, int c, int q, int n1, double* R) {
  const long long offp = w.off_p[c], rbase = w.off_k1[c] + c;
  for (int base = 0; base < 4 * n1; base += blockDim.x) {
    const int e = base + threadIdx.x, i = e >> 2;
    const bool on = i < n1;
    float h[7] = {}, l[7] = {};   // xx, yy, zz, xy, xz, yz of F B0 alpha_bar r r^T, then F A0 alpha_bar
    if (on) {
      const int tb = w.prow_k2[rbase + i] + (e & 3), en = w.prow_k2[rbase + i + 1];
      // as in the residual: indices two pairs ahead, data one pair ahead
      const float4* gp = reinterpret_cast<const float4*>(w.pr_gff) + 3 * offp;
      int2 gn = make_int2(-1, 0), ga = gn;
      float4 n0, n1v, nr;
      float2 na;
      if (tb < en) {
        gn = __ldg(w.pr_ga + offp + tb);
        n0 = __ldg(gp + 3 * tb); n1v = __ldg(gp + 3 * tb + 1);
        nr = rad_row(w, p, gn.x, q);
        na = __ldg(w.abff + (long long)gn.y * p.nqs + q);
        ga = __ldg(w.pr_ga + offp + min(tb + 4, en - 1));
      }
      for (int t = tb; t < en; t += 4) {
        const float4 g0 = n0, g1 = n1v, ra = nr;
        const float2 ab = na;
        const int gi = gn.x, tn = min(t + 4, en - 1);
        gn = ga;
        n0 = __ldg(gp + 3 * tn); n1v = __ldg(gp + 3 * tn + 1);
        nr = rad_row(w, p, gn.x, q);
        na = __ldg(w.abff + (long long)gn.y * p.nqs + q);
        ga = __ldg(w.pr_ga + offp + min(t + 8, en - 1));
        ff fa, fb;
        pair_rad_ff(w, p, c, q, offp + t, gi, ra, ff_make(g1.z, g1.w), fa, fb);
        const ff aj = ff_make(ab.x, ab.y);
        const ff rx = ff_make(g0.x, g0.y), ry = ff_make(g0.z, g0.w), rz = ff_make(g1.x, g1.y);
        const ff wb = ff_mul(aj, fb);
        const ff ux = ff_mul(wb, rx), uy = ff_mul(wb, ry), uz = ff_mul(wb, rz);
        ff_mac(h[0], l[0], ux, rx);
        ff_mac(h[1], l[1], uy, ry);
        ff_mac(h[2], l[2], uz, rz);
        ff_mac(h[3], l[3], ux, ry);
        ff_mac(h[4], l[4], ux, rz);
        ff_mac(h[5], l[5], uy, rz);
        ff_mac(h[6], l[6], aj, fa);
      }
    }
    ff s[7];
#pragma unroll
    for (int u = 0; u < 7; ++u) {
      s[u] = ff_quick_two_sum(h[u], l[u]);
#pragma unroll
      for (int o = 1; o < 4; o <<= 1)
        s[u] = ff_add(s[u], ff_make(__shfl_xor_sync(0xffffffffu, s[u].hi, o), __shfl_xor_sync(0xffffffffu, s[u].lo, o)));
    }
    if (on && (e & 3) == 0) {
      double v[6];
#pragma unroll
      for (int u = 0; u < 3; ++u) v[u] = 1.0 - ff_to_double(ff_add(s[u], s[6]));
#pragma unroll
      for (int u = 3; u < 6; ++u) v[u] = -ff_to_double(s[u]);
      double* Ri = R + 9 * i;
      Ri[0] = v[0]; Ri[1] = Ri[3] = v[3]; Ri[2] = Ri[6] = v[4];
      Ri[4] = v[1]; Ri[5] = Ri[7] = v[5]; Ri[8] = v[2];
    }
  }
}

// Systems on the LU list: forward ones and, should the adjoint solve of a system stall, that one.
__device__ __forceinline__ void scs_list_for_lu(const Work& w, int id) {
  w.fb_flag[id] = 1;
  const int e = atomicAdd(w.fb, 1);
  w.fb[1 + e] = id;
}

// dL/dX_i = delta/3 times this: dL/dalpha_K,i, plus dL/dalpha_I,c on the centre's block.
__device__ __forceinline__ double adjoint_seed(const Work& w, const DevParams& p, int c, int q, int i) {
  double v = w.alphaK_bar[(w.off_k1[c] + i) * p.nqs + q];
  if (i == 0) v += w.alphaI_bar[(long long)c * p.nqs + q];
  return v * (1.0 / 3.0);
}
// Biased exponent of the largest seed of a system (every warp by itself), 0x7ff if one is not finite:
// the adjoint systems are solved, and their solutions kept, at unit size (lambda = 2^lexp lsol),
// since a caller's weights may be of any magnitude.
__device__ __forceinline__ int adjoint_exponent(const Work& w, const DevParams& p, int c, int q, int n1) {
  int top = 1;
  for (int i = threadIdx.x & 31; i < n1; i += 32)
    top = max(top, (int)((__double_as_longlong(adjoint_seed(w, p, c, q, i)) >> 52) & 0x7ff));
  top = __reduce_max_sync(0xffffffffu, top);
  return top == 0x7ff ? top : min(top, 2045);
}

// A seed that is not finite (a caller's weight, a negative polarisability) makes the whole solution NaN: the
// gradient it belongs to says so, and the other centres' stay as they are.
__device__ __forceinline__ void adjoint_not_finite(const Work& w, int id, int n1, double* lam) {
  for (int e = threadIdx.x; e < 9 * n1; e += blockDim.x) lam[e] = __longlong_as_double(0x7ff8000000000000LL);
  if (threadIdx.x == 0) w.lexp[id] = 0;
}

// One (centre, frequency) system per block of 32 S (3 / NC) threads.  ADJ = false: X = B^-1 d, refined until
// a correction falls to 2^-52 of it, alpha_K and alpha_I; the couplings and the residuals are float-float, so
// its error is about cond(B) 2^-46.  ADJ = true: lambda = B^-1 dL/dX, to 2^-30 of its largest
// value or better (it feeds the forces only).  The refinement measures its own contraction.
constexpr int cg_min_blocks(int S, int NC) { return NC == 1 ? (S == 1 ? 7 : (S == 2 ? 4 : 2)) : (S == 1 ? 20 : (S == 2 ? 12 : 5)); }
template <int S, int NC, bool ADJ>
__global__ void __launch_bounds__(32 * S * (3 / NC), cg_min_blocks(S, NC))
    k_scs_solve(Work w, DevParams p, const int* order, int b0, int ld) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = order ? order[b0 + blockIdx.x / p.nqs] : b0 + blockIdx.x / p.nqs;
  const int q = blockIdx.x % p.nqs;
  if (c >= w.n_atoms) return;
  const int id = c * p.nqs + q;
  if (ADJ && w.fb_flag[id]) return;   // solved by the LU fallback (k_scs_lu_adjoint)
  const int n1 = w.counts[c].n1;
  const CgSmem sm = cg_carve(smem_raw, ld);
  const int tid = threadIdx.x, gt = tid % (32 * S);   // thread within its group
  const CgGroup<S> grp{tid / (32 * S), gt >> 5};
  const int c0 = grp.id;
  const long long sbase = (long long)c * w.site_cap, offk1 = w.off_k1[c];
  const long long offp = w.off_p[c], rbase = offk1 + c;
  const int nk1 = w.prow[rbase + n1];
  float4* rad = w.pr_rad4 + offp * p.nqs + (long long)q * nk1;
  // the system's slot of the solution array holds its FP64 residual until the solution is known
  double* R = (ADJ ? w.lsol : w.xsol) + offk1 * p.nqs * 9 + (long long)q * n1 * 9;
  for (int s = tid; s < n1; s += blockDim.x) {
    const double* x = w.site_x + 3 * (sbase + s);
    const float ab = w.abff[(long long)w.site_atom[sbase + s] * p.nqs + q].x;
    const float fx = (float)x[0], fy = (float)x[1], fz = (float)x[2];
    sm.site[s].a = make_float4(fx, fy, fz, 0.f);
    sm.s[s] = sqrtf(ab);
  }
  for (int e = tid; e < n1 * (n1 + 1) / 2; e += blockDim.x) sm.F[e] = make_float2(0.f, 0.f);
  __syncthreads();
  for (int s = tid; s < n1; s += blockDim.x) sm.F[s * (s + 1) / 2 + s] = make_float2(1.f, 0.f);
#pragma unroll 2
  for (int t = tid; t < nk1; t += blockDim.x) {
    const int2 ij = __ldg(reinterpret_cast<const int2*>(w.pr_ij) + offp + t);
    float4 f;
    if (ADJ) {
      f = __ldg(rad + t);
    } else {
      const int gi = __ldg(w.pr_ga + offp + t).x;
      const float4 g1 = __ldg(reinterpret_cast<const float4*>(w.pr_gff + 6 * (offp + t)) + 1);
      ff fa, fb;
      pair_rad_ff(w, p, c, q, offp + t, gi, rad_row(w, p, gi, q), ff_make(g1.z, g1.w), fa, fb);
      f = make_float4(fa.hi, fa.lo, fb.hi, fb.lo);
      rad[t] = f;
    }
    const float s = sm.s[ij.x] * sm.s[ij.y];
    sm.F[ij.x * (ij.x + 1) / 2 + ij.y] = make_float2(f.x * s, f.z * s);
  }
  if (!ADJ) {
    cg_build_rhs(w, p, c, q, n1, R);
  } else {
    const int top = adjoint_exponent(w, p, c, q, n1);
    if (top == 0x7ff) {   // uniform over the block
      adjoint_not_finite(w, id, n1, R);
      return;
    }
    if (tid == 0) w.lexp[id] = top - 1023;
    const double up = __longlong_as_double((long long)(2046 - top) << 52);
    const double gv = gt < n1 ? adjoint_seed(w, p, c, q, gt) : 0.0;
    if (gt < n1)
#pragma unroll
      for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int a = 0; a < 3; ++a) R[9 * gt + 3 * a + c0 + k] = a == c0 + k ? gv * up : 0.0;
  }
  __threadfence_block();
  __syncthreads();

  const float rel = ADJ ? 9.313225746154785e-10f : 2.220446049250313e-16f;
  const float inner = ADJ ? 1e-6f : 2e-6f;
  const bool act = gt < n1;
  const float si = act ? sm.s[gt] : 0.f;
  double* const Ri = R + 9 * (act ? gt : 0);
  double xd[NC][3];
#pragma unroll
  for (int k = 0; k < NC; ++k)
#pragma unroll
    for (int a = 0; a < 3; ++a) xd[k][a] = 0.0;
  float lim = 0.f, prev = 0.f, tol = inner;
  bool ok = true;
  for (int it = 0;; ++it) {
    float r[NC][3], x[NC][3], dm[1] = {0.f};
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
      for (int a = 0; a < 3; ++a) r[k][a] = si * (float)Ri[3 * a + c0 + k];
    ok = cg_solve<S, NC>(sm, grp, n1, gt, c0, tol, r, x);
    if (!ok) break;
    grp.sync();
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        x[k][a] *= si;
        xd[k][a] += (double)x[k][a];
        dm[0] = fmaxf(dm[0], fabsf(x[k][a]));
        if (act) *cg_slot(sm.site[gt], c0 + k, a) = x[k][a];
      }
    grp.template max<1>(dm, sm, 2);
    const float dmax = dm[0];
    // contraction estimate rho = |delta_k| / |delta_{k-1}| (delta_0 = the FP32 solution): the error
    // left after correction k is about rho |delta_k|, or tol |delta_k| where its solve was looser
    const float rho = it > 0 ? dmax / prev : 0.f;
    if (it == 0) {
      lim = rel * dmax;
      if (dmax == 0.f) break;
    } else {
      if (dmax <= lim) break;
      if (ADJ && 10.f * rho * dmax <= lim && it == 1) break;
      if (it >= 2 && rho < 0.5f && fmaxf(rho, tol) * dmax <= lim) break;
      if (it == CG_OUTER) { ok = false; break; }
      // the next correction (about rho dmax) only needs the digits down to the limit
      if (!ADJ) tol = fminf(fmaxf(0.25f * lim / (rho * dmax), inner), 1e-2f);
    }
    prev = dmax;
    grp.sync();
    cg_residual_update<S, NC>(w, p, c, q, n1, c0, nk1, gt, sm, R);
    grp.sync();
  }
  // a direction of non-positive curvature (B_K not positive definite: Sec. III.A, polarisation
  // catastrophe) or a refinement that does not converge sends the system to the LU fallback
  if (__syncthreads_or(!ok)) {
    if (tid == 0) scs_list_for_lu(w, id);
    return;
  }
  if (!ADJ && tid == 0) w.fb_flag[id] = 0;
  if (act)
#pragma unroll
    for (int k = 0; k < NC; ++k)
#pragma unroll
      for (int a = 0; a < 3; ++a) Ri[3 * a + c0 + k] = xd[k][a];
  if (!ADJ) {   // alpha_K,i = Tr(X_i) / 3, alpha_I,c = alpha_K,0
    __threadfence_block();
    __syncthreads();
    for (int i = tid; i < n1; i += blockDim.x) {
      const double a = (R[9 * i] + R[9 * i + 4] + R[9 * i + 8]) / 3.0;
      w.alphaK[(offk1 + i) * p.nqs + q] = a;
      if (i == 0) w.alphaI[id] = a;
    }
  }
}

// ---------------------------------------------------------------------------------------
// adjoint contraction: one block per central atom, all frequencies
// ---------------------------------------------------------------------------------------
// Per pair <M, dT_SR/dr> with M = -(lambda_i X_j^T + lambda_j X_i^T) (K1 pairs) or
// M = -alpha_bar_j lambda_i (K2 pairs), symmetrised, T_SR = F (A0 + B0 r r^T):
//   dL/dr_j = r [F dB0 r.M.r + F dA0 Tr M + dF (B0 r.M.r + A0 Tr M)] / |r| + 2 F B0 M r.
// Geometry, F and dF do not depend on the frequency, so a thread runs its pair over all
// frequencies, summing W = sum B0 M, W' = sum dB0 M (six entries each) and the scalars
// sum A0 Tr M, sum dA0 Tr M, and applies geometry once; lambda and X of every frequency are staged
// in shared memory as float-float (97 KB at |K1| = 52 and 13 frequencies, two blocks per SM).
// Float-float throughout (compensated sums, ~2^-46): 4.1 ms per 4096-atom step, bound by its FP32
// instructions; one block per (centre, frequency) with the gradients of each frequency staged in
// global memory took about half of a 22.8 ms adjoint.
// More frequencies than fit in shared memory are taken in chunks, the sums kept in `gstage`; small
// structures split the frequencies of a centre over several blocks (the gradient is linear in the
// sums, so each block finishes its own part).
#define CON_W 14   // 6 + 6 + 2 float-float sums per pair

__device__ __forceinline__ ff ff_ld(const float2* p) {
  const float2 v = *p;
  return ff_make(v.x, v.y);
}

struct ConSum {
  float h[CON_W], l[CON_W];
  __device__ __forceinline__ void add(const ff (&M)[6], ff A0, ff B0, ff dA0, ff dB0) {
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      ff_mac(h[u], l[u], B0, M[u]);
      ff_mac(h[6 + u], l[6 + u], dB0, M[u]);
    }
    const ff tr = ff_add(ff_add(M[0], M[1]), M[2]);
    ff_mac(h[12], l[12], A0, tr);
    ff_mac(h[13], l[13], dA0, tr);
  }
  __device__ __forceinline__ ff get(int u) const { return ff_quick_two_sum(h[u], l[u]); }
};

// A0, B0, dA0, dB0 of pair pq at frequency q (float-float)
__device__ __noinline__ void pair_terms_slow(const Work& w, const DevParams& p, int c, int q, long long pq, ff& A0,
                                             ff& B0, ff& dA0, ff& dB0) {
  const long long sbase = (long long)c * w.site_cap;
  const PairGeo64 g = pair_geo64(w, p, c, pq);
  const double si = w.sig[(long long)w.site_atom[sbase + w.pr_ij[2 * pq]] * p.nqs + q];
  const double sj = w.sig[(long long)w.site_atom[sbase + w.pr_ij[2 * pq + 1]] * p.nqs + q];
  double a, b, da, db;
  tsr_radial_fast(g.r, g.ir, si * si + sj * sj, a, b, da, db);
  A0 = ff_from_double(a); B0 = ff_from_double(b); dA0 = ff_from_double(da); dB0 = ff_from_double(db);
}
__device__ __forceinline__ void pair_terms(const Work& w, const DevParams& p, int c, int q, long long pq, int gi, float4 u,
                                           float4 v, ff& A0, ff& B0, ff& dA0, ff& dB0) {
  if (gi >= 0) {
    A0 = ff_make(u.x, u.y); B0 = ff_make(u.z, u.w); dA0 = ff_make(v.x, v.y); dB0 = ff_make(v.z, v.w);
  } else {
    pair_terms_slow(w, p, c, q, pq, A0, B0, dA0, dB0);
  }
}

// dL/dr_j of the pair from its frequency sums (W carries no minus sign and, for the off-diagonal
// entries, both orders: the symmetrised M is half of them)
__device__ __forceinline__ void con_finish(const Work& w, long long pq, const ConSum& S, ff (&g)[3]) {
  const float4* gf = reinterpret_cast<const float4*>(w.pr_gff + 6 * pq);
  const float4 g0 = gf[0], g1 = gf[1], g2 = gf[2];
  const ff rr[3] = {ff_make(g0.x, g0.y), ff_make(g0.z, g0.w), ff_make(g1.x, g1.y)};
  const ff F = ff_make(g1.z, g1.w), dF = ff_make(g2.x, g2.y), ir = ff_make(g2.z, g2.w);
  ff V[3], rW[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const ff a = S.get(6 * k), b = S.get(6 * k + 1), d = S.get(6 * k + 2);
    const ff xy = ff_scale(S.get(6 * k + 3), 0.5f), xz = ff_scale(S.get(6 * k + 4), 0.5f), yz = ff_scale(S.get(6 * k + 5), 0.5f);
    const ff v0 = ff_fma(xz, rr[2], ff_fma(xy, rr[1], ff_mul(a, rr[0])));
    const ff v1 = ff_fma(yz, rr[2], ff_fma(b, rr[1], ff_mul(xy, rr[0])));
    const ff v2 = ff_fma(d, rr[2], ff_fma(yz, rr[1], ff_mul(xz, rr[0])));
    rW[k] = ff_fma(rr[2], v2, ff_fma(rr[1], v1, ff_mul(rr[0], v0)));
    if (k == 0) { V[0] = v0; V[1] = v1; V[2] = v2; }
  }
  const ff phi = ff_add(rW[0], S.get(12)), inner = ff_add(rW[1], S.get(13));
  const ff radial = ff_mul(ff_fma(F, inner, ff_mul(dF, phi)), ir);
  const ff tang = ff_scale(F, 2.0f);
#pragma unroll
  for (int d = 0; d < 3; ++d) g[d] = ff_neg(ff_fma(tang, V[d], ff_mul(radial, rr[d])));
}

__global__ void __launch_bounds__(256, 2) k_scs_contract(Work w, DevParams p, int c0, int nsplit, int smem, int scratch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = c0 + blockIdx.x / nsplit, split = blockIdx.x % nsplit;
  if (c >= w.n_atoms) return;
  // this block's frequencies
  const int per = (p.nqs + nsplit - 1) / nsplit, qb = split * per, qe = min(p.nqs, qb + per);
  if (qb >= qe) return;
  const int n1 = w.counts[c].n1, n12 = w.counts[c].n12, tid = threadIdx.x;
  const long long sbase = (long long)c * w.site_cap;
  const long long offp = w.off_p[c], offa = w.off_a[c], rbase = w.off_k1[c] + c;
  const int nk1 = w.prow[rbase + n1], np = w.prow_k2[rbase + n1];
  const double* Xg = w.xsol + w.off_k1[c] * p.nqs * 9;
  const double* Lg = w.lsol + w.off_k1[c] * p.nqs * 9;
  int lexp = -2000;   // the block works at the largest scale of its frequencies
  for (int q = qb; q < qe; ++q) lexp = max(lexp, w.lexp[(long long)c * p.nqs + q]);
  const int qc = max(1, min(per, smem / (144 * n1)));   // frequencies staged at once
  float2* Ls = reinterpret_cast<float2*>(smem_raw);   // [qc][9 n1] lambda
  float2* Xs = Ls + qc * 9 * n1;                      // [qc][9 n1] X
  // gradient of each pair, then (frequencies in chunks) its CON_W sums of the chunks so far
  float2* gst = w.gstage + (scratch / nsplit) * (offp * nsplit + (long long)split * np);
  float2* sums = gst + 3LL * np;
  for (int q0 = qb; q0 < qe; q0 += qc) {
    const int nqc = min(qc, qe - q0);
    const bool first = q0 == qb, last = q0 + nqc == qe;
    __syncthreads();
    for (int e = tid; e < nqc * 9 * n1; e += blockDim.x) {
      const int down = w.lexp[(long long)c * p.nqs + q0 + e / (9 * n1)] - lexp;
      const float f = down < -126 ? 0.f : __int_as_float((down + 127) << 23);
      const ff l = ff_split(Lg[(long long)q0 * 9 * n1 + e]), x = ff_split(Xg[(long long)q0 * 9 * n1 + e]);
      Ls[e] = make_float2(l.hi * f, l.lo * f);
      Xs[e] = make_float2(x.hi, x.lo);
    }
    __syncthreads();
    // K1 pairs (whole warps), then K2 pairs
    for (int kind = 0; kind < 2; ++kind) {
      const int tb = kind == 0 ? 0 : nk1, te = kind == 0 ? nk1 : np;
      for (int t = tb + tid; t < te; t += blockDim.x) {
        const long long pq = offp + t;
        const int2 ij = reinterpret_cast<const int2*>(w.pr_ij)[pq];
        const int2 ga = w.pr_ga[pq];
        const int gi = ga.x;
        // table rows of this pair, one frequency ahead of the arithmetic
        const float4* ra = reinterpret_cast<const float4*>(w.rad_ff + 4 * ((long long)max(gi, 0) * p.nqs + q0));
        float4 nu = ra[0], nv = ra[1];
        ConSum S;
#pragma unroll
        for (int u = 0; u < CON_W; ++u) {
          S.h[u] = S.l[u] = 0.f;
          if (!first) {
            const float2 v = sums[(long long)CON_W * t + u];
            S.h[u] = v.x;
            S.l[u] = v.y;
          }
        }
        if (kind == 0) {
          for (int q = 0; q < nqc; ++q) {
            const float4 u4 = nu, v4 = nv;
            const int qn = min(q + 1, nqc - 1);
            nu = ra[2 * qn];
            nv = ra[2 * qn + 1];
            const float2* li = Ls + (q * n1 + ij.x) * 9;
            const float2* lj = Ls + (q * n1 + ij.y) * 9;
            const float2* xi = Xs + (q * n1 + ij.x) * 9;
            const float2* xj = Xs + (q * n1 + ij.y) * 9;
            float h[6] = {}, l[6] = {};
            // row a of lambda times row b of X, summed over the three right-hand sides
            constexpr int idx[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              ff xa[3], xb[3];
#pragma unroll
              for (int b = 0; b < 3; ++b) { xa[b] = ff_ld(xi + 3 * b + k); xb[b] = ff_ld(xj + 3 * b + k); }
#pragma unroll
              for (int a = 0; a < 3; ++a) {
                const ff va = ff_ld(li + 3 * a + k), vb = ff_ld(lj + 3 * a + k);
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                  ff_mac(h[idx[a][b]], l[idx[a][b]], va, xb[b]);
                  ff_mac(h[idx[a][b]], l[idx[a][b]], vb, xa[b]);
                }
              }
            }
            ff M[6];
#pragma unroll
            for (int u = 0; u < 6; ++u) M[u] = ff_quick_two_sum(h[u], l[u]);
            ff A0, B0, dA0, dB0;
            pair_terms(w, p, c, q0 + q, pq, gi, u4, v4, A0, B0, dA0, dB0);
            S.add(M, A0, B0, dA0, dB0);
          }
        } else {
          const float2* abj = w.abff + (long long)ga.y * p.nqs + q0;
          float2 na = abj[0];
          for (int q = 0; q < nqc; ++q) {
            const float4 u4 = nu, v4 = nv;
            const ff a = ff_make(na.x, na.y);
            const int qn = min(q + 1, nqc - 1);
            nu = ra[2 * qn];
            nv = ra[2 * qn + 1];
            na = abj[qn];
            const float2* li = Ls + (q * n1 + ij.x) * 9;
            const ff M[6] = {ff_ld(li), ff_ld(li + 4), ff_ld(li + 8), ff_add(ff_ld(li + 1), ff_ld(li + 3)),
                             ff_add(ff_ld(li + 2), ff_ld(li + 6)), ff_add(ff_ld(li + 5), ff_ld(li + 7))};
            ff A0, B0, dA0, dB0;
            pair_terms(w, p, c, q0 + q, pq, gi, u4, v4, A0, B0, dA0, dB0);
            S.add(M, ff_mul(a, A0), ff_mul(a, B0), ff_mul(a, dA0), ff_mul(a, dB0));
          }
        }
        if (!last) {
#pragma unroll
          for (int u = 0; u < CON_W; ++u) sums[(long long)CON_W * t + u] = make_float2(S.h[u], S.l[u]);
        } else {
          ff g[3];
          con_finish(w, pq, S, g);
#pragma unroll
          for (int d = 0; d < 3; ++d) gst[3LL * t + d] = make_float2(g[d].hi, g[d].lo);
        }
      }
    }
  }
  __threadfence_block();
  __syncthreads();
  const double scale = __longlong_as_double((long long)(min(max(lexp, -1022), 1023) + 1023) << 52);
  // per site (fixed order): owner of its row's pairs (-g), partner of K1 pairs owned by later rows
  // (+g, from the adjacency row) and of K2 pairs (+g, from the reverse list)
  for (int s = tid; s < n12; s += blockDim.x) {
    const int a = w.site_atom[sbase + s];
    if (p.paper && a != c) continue;     // the paper's forces: only atom c's own gradient
    ff gs[3] = {ff_make(0.f, 0.f), ff_make(0.f, 0.f), ff_make(0.f, 0.f)};
    auto acc = [&](int t, bool plus) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const ff v = ff_ld(gst + 3LL * t + d);
        gs[d] = plus ? ff_add(gs[d], v) : ff_sub(gs[d], v);
      }
    };
    if (s < n1) {
      const int e1 = w.prow[rbase + s + 1], e2 = w.prow_k2[rbase + s + 1], e3 = w.arow[rbase + s + 1];
#pragma unroll 4
      for (int t = w.prow[rbase + s]; t < e1; ++t) acc(t, false);
#pragma unroll 4
      for (int t = w.prow_k2[rbase + s]; t < e2; ++t) acc(t, false);
      const int2* ad = reinterpret_cast<const int2*>(w.adj) + offa;
#pragma unroll 4
      for (int t = w.arow[rbase + s]; t < e3; ++t) {
        const int2 v = __ldg(ad + t);
        if (v.x > s) acc(v.y, true);
      }
    } else {
      const int e = w.k2ptr[sbase + s + 1];
#pragma unroll 4
      for (int t = w.k2ptr[sbase + s]; t < e; ++t) acc(__ldg(w.k2rev + offp + t), true);
    }
    const double gx = ff_to_double(gs[0]) * scale, gy = ff_to_double(gs[1]) * scale, gz = ff_to_double(gs[2]) * scale;
    if (gx != 0.0 || gy != 0.0 || gz != 0.0) atomic_add3(w.gacc + 3 * a, gx, gy, gz);
  }
}

// ---------------------------------------------------------------------------------------
// LU fallback for screening matrices that are not positive definite (Sec. III.A: the
// polarisation catastrophe makes B_K indefinite) or on which the refinement does not converge.
// Such systems are rare; each is solved in FP64 by Gaussian elimination with
// partial pivoting (row interchanges), the same factorisation a library dense solve uses, on
// the dense B_K assembled from the pair list into a per-block slot of global memory.  A pivot
// that is exactly zero (B_K singular) sets LMBD_FLAG_NOT_SPD.
// ---------------------------------------------------------------------------------------
struct LuSmem {
  double* x;      // 9 n1: right-hand side, then solution
  double* red;    // 64
  int* piv;       // 3 n1
  int* redi;      // 64
};
__host__ __device__ inline size_t lu_smem_bytes(int max_n1) {
  return (size_t)max_n1 * (9 * sizeof(double) + 3 * sizeof(int)) + 64 * (sizeof(double) + sizeof(int));
}
__device__ inline LuSmem lu_carve(unsigned char* base, int max_n1) {
  LuSmem s;
  s.x = reinterpret_cast<double*>(base);
  s.red = s.x + 9 * max_n1;
  s.piv = reinterpret_cast<int*>(s.red + 64);
  s.redi = s.piv + 3 * max_n1;
  return s;
}

// dense B_K (N1 x N1 row-major, FP64) of one (centre, frequency): diag(1/alpha_bar) plus the
// T_SR blocks of the K1 pairs (symmetric 3 x 3 blocks, F A0 delta + F B0 r r^T)
__device__ void scs2_dense_b(const Work& w, const DevParams& p, int c, int q, int n1, double* A) {
  const int N1 = 3 * n1;
  const long long offp = w.off_p[c], rbase = w.off_k1[c] + c, sbase = (long long)c * w.site_cap;
  const int nk1 = w.prow[rbase + n1];
  for (long long e = threadIdx.x; e < (long long)N1 * N1; e += blockDim.x) A[e] = 0.0;
  __syncthreads();
  for (int i = threadIdx.x; i < n1; i += blockDim.x) {
    const double ia = 1.0 / w.abar[(long long)w.site_atom[sbase + i] * p.nqs + q];
    for (int al = 0; al < 3; ++al) A[(long long)(3 * i + al) * N1 + 3 * i + al] = ia;
  }
  for (int t = threadIdx.x; t < nk1; t += blockDim.x) {
    const long long pq = offp + t;
    const int i = w.pr_ij[2 * pq], j = w.pr_ij[2 * pq + 1];
    const PairGeo64 g = pair_geo64(w, p, c, pq);
    double fa, fb;
    pair_rad64(w, p, c, q, pq, g, fa, fb);
    for (int al = 0; al < 3; ++al)
      for (int be = 0; be < 3; ++be) {
        const double v = fb * g.x[al] * g.x[be] + (al == be ? fa : 0.0);
        A[(long long)(3 * i + al) * N1 + 3 * j + be] = v;
        A[(long long)(3 * j + be) * N1 + 3 * i + al] = v;
      }
  }
  __syncthreads();
}

// In-place LU with partial pivoting of the N1 x N1 matrix A (global memory), whole block:
// P A = L U, L unit lower (below the diagonal), U upper; piv[k] = row swapped with row k.
// Returns (uniformly) false if a pivot is zero or not finite.
__device__ bool lu_factor_dense(double* A, int n, int* piv, double* redv, int* redi) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  __shared__ int ok_s, p_s;
  if (tid == 0) ok_s = 1;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    // pivot: the largest |A[i][k]|, i >= k (ties to the lowest row)
    double best = -1.0;
    int bi = k;
    for (int i = k + tid; i < n; i += blockDim.x) {
      const double v = fabs(A[(long long)i * n + k]);
      if (v > best) { best = v; bi = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (lane == 0) { redv[warp] = best; redi[warp] = bi; }
    __syncthreads();
    if (tid == 0) {
      double b = redv[0];
      int ix = redi[0];
      for (int u = 1; u < nw; ++u)
        if (redv[u] > b || (redv[u] == b && redi[u] < ix)) { b = redv[u]; ix = redi[u]; }
      p_s = ix;
      piv[k] = ix;
      if (!(b > 0.0) || !isfinite(b)) ok_s = 0;
    }
    __syncthreads();
    if (!ok_s) return false;
    const int pr = p_s;
    if (pr != k)
      for (int j = tid; j < n; j += blockDim.x) {
        const double t = A[(long long)k * n + j];
        A[(long long)k * n + j] = A[(long long)pr * n + j];
        A[(long long)pr * n + j] = t;
      }
    __syncthreads();
    const double inv = 1.0 / A[(long long)k * n + k];
    for (int i = k + 1 + tid; i < n; i += blockDim.x) A[(long long)i * n + k] *= inv;
    __syncthreads();
    const int m = n - k - 1;
    for (long long e = tid; e < (long long)m * m; e += blockDim.x) {
      const int i = k + 1 + (int)(e / m), j = k + 1 + (int)(e % m);
      A[(long long)i * n + j] -= A[(long long)i * n + k] * A[(long long)k * n + j];
    }
    __syncthreads();
  }
  return true;
}

// b (n x 3 row-major, shared memory) <- A^-1 b with the factors of lu_factor_dense; warps 0..2
// take one column each (row sums split over the lanes)
__device__ void lu_solve3_dense(const double* A, int n, const int* piv, double* b) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (warp < 3) {
    const int c = warp;
    if (lane == 0)
      for (int k = 0; k < n; ++k)
        if (piv[k] != k) {
          const double t = b[3 * k + c];
          b[3 * k + c] = b[3 * piv[k] + c];
          b[3 * piv[k] + c] = t;
        }
    __syncwarp();
    for (int i = 0; i < n; ++i) {
      double sacc = 0.0;
      for (int j = lane; j < i; j += 32) sacc += A[(long long)i * n + j] * b[3 * j + c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sacc += __shfl_xor_sync(0xffffffffu, sacc, o);
      if (lane == 0) b[3 * i + c] -= sacc;
      __syncwarp();
    }
    for (int i = n - 1; i >= 0; --i) {
      double sacc = 0.0;
      for (int j = i + 1 + lane; j < n; j += 32) sacc += A[(long long)i * n + j] * b[3 * j + c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sacc += __shfl_xor_sync(0xffffffffu, sacc, o);
      if (lane == 0) b[3 * i + c] = (b[3 * i + c] - sacc) / A[(long long)i * n + i];
      __syncwarp();
    }
  }
  __syncthreads();
}

// Forward LU fallback: persistent over the listed (centre, frequency) systems, one dense slot
// of lu_slot doubles per block.
__global__ void __launch_bounds__(256) k_scs_lu_forward(Work w, DevParams p, int max_n1, int tally) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const LuSmem sm = lu_carve(smem_raw, max_n1);
  double* A = w.lu + (long long)blockIdx.x * w.lu_slot;
  const int count = w.fb[0];
  if (tally && blockIdx.x == 0 && threadIdx.x == 0 && count > 0) atomicAdd(w.status + 2, count);
  for (int e = blockIdx.x; e < count; e += gridDim.x) {
    const int id = w.fb[1 + e], c = id / p.nqs, q = id % p.nqs;
    const int n1 = w.counts[c].n1, N1 = 3 * n1;
    const long long offk1 = w.off_k1[c];
    scs2_build_rhs64(w, p, c, n1, q, sm.x);
    scs2_dense_b(w, p, c, q, n1, A);
    if (!lu_factor_dense(A, N1, sm.piv, sm.red, sm.redi)) {
      if (threadIdx.x == 0) atomicOr(w.status, LMBD_FLAG_NOT_SPD);
      __syncthreads();
      continue;
    }
    lu_solve3_dense(A, N1, sm.piv, sm.x);
    double* X = w.xsol + offk1 * p.nqs * 9 + (long long)q * N1 * 3;
    for (int u = threadIdx.x; u < N1 * 3; u += blockDim.x) X[u] = sm.x[u];
    for (int i = threadIdx.x; i < n1; i += blockDim.x) {
      const double a = (sm.x[9 * i] + sm.x[9 * i + 4] + sm.x[9 * i + 8]) / 3.0;
      w.alphaK[(offk1 + i) * p.nqs + q] = a;
      if (i == 0) w.alphaI[id] = a;
    }
    __syncthreads();
  }
}

// Adjoint LU fallback for the listed systems of centres [c0, c1): B_K is factored again (it is
// symmetric, so lambda = B_K^-T dL/dX = B_K^-1 dL/dX).
__global__ void __launch_bounds__(256) k_scs_lu_adjoint(Work w, DevParams p, int c0, int c1, int max_n1) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const LuSmem sm = lu_carve(smem_raw, max_n1);
  double* A = w.lu + (long long)blockIdx.x * w.lu_slot;
  const int count = w.fb[0];
  for (int e = blockIdx.x; e < count; e += gridDim.x) {
    const int id = w.fb[1 + e], c = id / p.nqs, q = id % p.nqs;
    if (c < c0 || c >= c1) continue;
    const int n1 = w.counts[c].n1, N1 = 3 * n1;
    double* lam = w.lsol + w.off_k1[c] * p.nqs * 9 + (long long)q * N1 * 3;
    const int top = adjoint_exponent(w, p, c, q, n1);
    if (top == 0x7ff) {   // uniform over the block
      adjoint_not_finite(w, id, n1, lam);
      continue;
    }
    scs2_dense_b(w, p, c, q, n1, A);
    if (!lu_factor_dense(A, N1, sm.piv, sm.red, sm.redi)) {
      if (threadIdx.x == 0) atomicOr(w.status, LMBD_FLAG_NOT_SPD);
      __syncthreads();
      continue;
    }
    const double up = __longlong_as_double((long long)(2046 - top) << 52);
    if (threadIdx.x == 0) w.lexp[id] = top - 1023;
    for (int u = threadIdx.x; u < 9 * n1; u += blockDim.x)
      sm.x[u] = (u % 9) / 3 == u % 3 ? adjoint_seed(w, p, c, q, u / 9) * up : 0.0;
    __syncthreads();
    lu_solve3_dense(A, N1, sm.piv, sm.x);
    for (int u = threadIdx.x; u < 9 * n1; u += blockDim.x) lam[u] = sm.x[u];
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------
void launch_scs_count(const Work& w, const DevParams& p, int max_n12, cudaStream_t s) {
  if (w.n_atoms == 0) return;
  size_t sm = (sizeof(double) + sizeof(float)) * 3 * (size_t)max_n12;
  raise_smem_limit((const void*)k_scs_count, sm);
  k_scs_count<<<w.n_atoms, 256, sm, s>>>(w, p, max_n12);
}

void launch_scs_fill(const Work& w, const DevParams& p, int c0, int c1, int max_n12, int max_n1, cudaStream_t s) {
  if (c1 <= c0) return;
  size_t sm = sizeof(double) * 3 * (size_t)max_n12 +
              sizeof(int) * ((size_t)max_n1 * max_n1 + 7 * (size_t)max_n1 + 3 + (size_t)max_n12) +
              sizeof(float) * 3 * (size_t)max_n12;
  raise_smem_limit((const void*)k_scs_fill, sm);
  k_scs_fill<<<c1 - c0, 256, sm, s>>>(w, p, c0, max_n12, max_n1);
}

void launch_pair_radial(const Work& w, const DevParams& p, cudaStream_t s) {
  if (w.n_atoms == 0) return;
  k_pair_radial<<<w.n_atoms, 128, 0, s>>>(w, p);
}

// Sites one screening system may hold: |K1| <= 96 (three warps) and, for the largest of them, |K1 u K2| (at most
// 3264 at |K1| = 96).  The second limit is the shared memory of a packed dense factor with its lists; the
// kernels here need less (k_scs_fill 204 KB at 4096 sites), but it stays part of what the entry points accept.
bool scs_capacity(int max_n1, int max_n12) {
  const size_t N1 = 3 * (size_t)max_n1;
  const size_t fl = (N1 * (N1 + 1) / 2 + 7 * N1 + (N1 + 15) / 16 * 136 + 1) & ~size_t(1);
  return max_n1 <= 96 && fl * sizeof(float) + (9 * N1 + (size_t)max_n12 + max_n1 + 64) * sizeof(double) <= 227 * 1024;
}

template <int S, int NC, bool ADJ>
static void run_solve(const Work& w, const DevParams& p, const int* order, int c0, int c1, int ld, cudaStream_t s) {
  const size_t sm = cg_smem_bytes(ld);
  raise_smem_limit((const void*)k_scs_solve<S, NC, ADJ>, sm);
  k_scs_solve<S, NC, ADJ><<<(c1 - c0) * p.nqs, 32 * S * (3 / NC), sm, s>>>(w, p, order, c0, ld);
}

// Centres order[c0..c1) (or c0..c1 when order is NULL), shared memory sized for the largest K1 among
// them.  A structure whose systems are all resident at once is bound by the time of one solve:
// there a group of warps per right-hand side shortens it (64-atom box, forward solves 0.72 ->
// 0.52 ms; 24-atom cluster 82 -> 47 us); larger ones are bound by the issue slots and take the three
// right-hand sides together (4096 atoms: 14.0 against 18.5 ms).  The choice depends on the
// structure, not on the wave, so that energies are the same bits in every partition.
template <bool ADJ>
static void run_solve_any(const Work& w, const DevParams& p, const int* order, int c0, int c1, int max_n1, cudaStream_t s) {
  if (c1 <= c0) return;
  const bool split = (long long)w.n_atoms * p.nqs <= 12LL * w.sms;
  if (split) {
    if (max_n1 <= 32) run_solve<1, 1, ADJ>(w, p, order, c0, c1, max_n1, s);
    else if (max_n1 <= 64) run_solve<2, 1, ADJ>(w, p, order, c0, c1, max_n1, s);
    else run_solve<3, 1, ADJ>(w, p, order, c0, c1, max_n1, s);
  } else {
    if (max_n1 <= 32) run_solve<1, 3, ADJ>(w, p, order, c0, c1, max_n1, s);
    else if (max_n1 <= 64) run_solve<2, 3, ADJ>(w, p, order, c0, c1, max_n1, s);
    else run_solve<3, 3, ADJ>(w, p, order, c0, c1, max_n1, s);
  }
}
void launch_scs_solve(const Work& w, const DevParams& p, const int* order, int c0, int c1, int max_n1, cudaStream_t s) {
  run_solve_any<false>(w, p, order, c0, c1, max_n1, s);
}
void launch_scs_adjoint(const Work& w, const DevParams& p, const int* order, int c0, int c1, int max_n1, cudaStream_t s) {
  run_solve_any<true>(w, p, order, c0, c1, max_n1, s);
}

// Blocks per centre of the contraction: structures of fewer centres than fill the chip twice split
// the frequencies (64-atom box, SCS adjoint phase 0.76 -> 0.57 ms, of which the solves 0.2).
static int scs_contract_split(int n_atoms, int nqs, int sms) {
  const int want = (2 * sms + n_atoms - 1) / (n_atoms > 0 ? n_atoms : 1);
  const int per = (nqs + want - 1) / want;
  return (nqs + per - 1) / per;
}
// Shared memory of its blocks: lambda and X of all a block's frequencies, or two blocks per SM; a centre
// whose |K1| does not fit takes its frequencies in chunks.
static size_t scs_contract_smem(int split, int max_n1, int nqs) {
  const int per = (nqs + split - 1) / split;
  return std::min((size_t)144 * max_n1 * per, (size_t)112 * 1024);
}
// float2 of gradient scratch per pair: 3, and 14 sums when the frequencies go in chunks, per block
int scs_contract_scratch(int n_atoms, int max_n1, int nqs, int sms) {
  const int split = scs_contract_split(n_atoms, nqs, sms), per = (nqs + split - 1) / split;
  return split * (scs_contract_smem(split, max_n1, nqs) < (size_t)144 * max_n1 * per ? 3 + CON_W : 3);
}

void launch_scs_contract(const Work& w, const DevParams& p, int c0, int c1, int max_n1, cudaStream_t s) {
  if (c1 <= c0) return;
  const int split = scs_contract_split(w.n_atoms, p.nqs, w.sms);
  const size_t sm = scs_contract_smem(split, max_n1, p.nqs);
  raise_smem_limit((const void*)k_scs_contract, sm);
  k_scs_contract<<<(c1 - c0) * split, 256, sm, s>>>(w, p, c0, split, (int)sm,
                                                    scs_contract_scratch(w.n_atoms, max_n1, p.nqs, w.sms));
}

// LU fallback launches: a fixed grid of lu_blocks persistent blocks (one dense slot each);
// with an empty list every block exits at once.
void launch_scs_lu_forward(const Work& w, const DevParams& p, int lu_blocks, int max_n1, int tally, cudaStream_t s) {
  k_scs_lu_forward<<<lu_blocks, 256, lu_smem_bytes(max_n1), s>>>(w, p, max_n1, tally);
}

void launch_scs_lu_adjoint(const Work& w, const DevParams& p, int lu_blocks, int c0, int c1, int max_n1, cudaStream_t s) {
  k_scs_lu_adjoint<<<lu_blocks, 256, lu_smem_bytes(max_n1), s>>>(w, p, c0, c1, max_n1);
}
