// Small FP64 kernels of the LAS energy/gradient chain: per-auxiliary-index contractions with the
// block-product RDMs, energy reduction, gradient assembly and layout helpers.
#include <string.h>

#include <algorithm>

#include "las_common.cuh"

namespace lasdf {

// Deterministic block sum of one double per thread, on thread 0 only: the warps' values of a lane
// added in warp order by the first warp, then a butterfly.  FP64 adds are slow on this part (a
// warp's add takes some 18 clocks of the SM), so no thread adds what another one has added.
template <int NT>
__device__ double block_sum0(double v, double* red) {   // red: NT doubles
  red[threadIdx.x] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) t += red[w * 32 + threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

// Cocc[mu][p] = C[mu][p] for p < o, 0 for o <= p < op; and, with dm2, the pair-transposed fragment
// 2-RDMs dm2t_K[wx][uv] = Gamma^K[uv][wx] that k_per_aux reads along uv.
__global__ void k_pack_cocc(const double* __restrict__ C, int n, int nmo, int o, int op,
                            double* __restrict__ Cocc, const double* __restrict__ dm2,
                            FragInfo fi, double* __restrict__ dm2t) {
  pdl_begin();
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const long total = (long)n * op;
  if (i < total) {
    int mu = (int)(i / op), p = (int)(i % op);
    Cocc[i] = (p < o) ? C[(long)mu * nmo + p] : 0.0;
    return;
  }
  if (!dm2) return;
  i -= total;
  for (int K = 0; K < fi.nfrag; ++K) {
    const long m = fi.off[K + 1] - fi.off[K], m2 = m * m;
    if (i < m2 * m2) {
      dm2t[fi.dm2_off[K] + (i % m2) * m2 + i / m2] = dm2[fi.dm2_off[K] + i];
      return;
    }
    i -= m2 * m2;
  }
}

__device__ __forceinline__ int frag_of(const FragInfo& fi, int u) {
  int K = 0;
  while (K + 1 < fi.nfrag && fi.off[K + 1] <= u) ++K;
  return K;
}

// Per auxiliary index L (one CTA each), given T_L = C_occ^T b^L C_occ (op x op):
//   vc = 2 sum_i T(i,i)                     (Coulomb vector of Dc, Eq. J_1 in the MO basis)
//   va = sum_uv D_uv T(u,v)                 (Coulomb vector of the active density)
//   Y(u,v) = sum_wx Gamma_uvwx T(w,x)       (block-product 2-RDM of Eq. las_wfn, applied
//                                            fragment-block by fragment-block)
//   eps_L  = vc^2/2 - sum_ij T(i,j)^2 + vc va - sum_{i,u} Z(i,u) T(i,u) + 1/2 sum_uv T(u,v) Y(u,v)
//            with Z = T(core,act) D  (the L-th term of the two-electron energy)
//   W_L(p,q): the matrix with  dE/dC(two-electron part) = sum_L H_L W_L, H_L = b^L C_occ.
// x * 2^g, and -x * 2^g, in exponent-field and sign-bit arithmetic: an FP64 multiply, comparison or
// negation would each take a slot of the FP64 pipe (and so would those of ldexp, even on a branch
// that no thread takes).  The sign is flipped by the same addition as the exponent: an exclusive or
// with the sign bit is what the compiler takes for a negation and gives to the FP64 pipe (a fifth of
// k_per_aux's FP64 instructions).  Zeros, infinities, NaN and whatever is subnormal before or after
// the scaling (rounded to even) or overflows in it go through scale2_edge.
__device__ __forceinline__ double scale2_edge(unsigned long long b, int g) {
  const unsigned long long sign = b >> 63 << 63, inf = 0x7FF0000000000000ull;
  unsigned long long m = b << 12 >> 12;
  int ex = (int)(b >> 52) & 0x7FF;
  if (ex == 0x7FF || (ex == 0 && m == 0)) return __longlong_as_double((long long)b);
  if (ex == 0) {   // bring the leading one to bit 52
    const int lz = __clzll((long long)m) - 11;
    m <<= lz;
    ex = 1 - lz;
  } else {
    m |= 1ull << 52;
  }
  ex += g;
  if (ex >= 0x7FF) {
    m = inf;
  } else if (ex >= 1) {
    m += (unsigned long long)(ex - 1) << 52;
  } else {
    const int sh = 1 - ex;
    m = sh > 54 ? 0 : (m + (1ull << (sh - 1)) - 1 + ((m >> sh) & 1)) >> sh;
  }
  return __longlong_as_double((long long)(sign | m));
}
template <bool NEG = false>
__device__ __forceinline__ double scale2(double x, int g) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7FF;
  if (min(ex, ex + g) < 1 || max(ex, ex + g) > 2046)
    return scale2_edge(b + (NEG ? 1ull << 63 : 0), g);
  return __longlong_as_double((long long)b + (((long long)(g + (NEG ? 2048 : 0))) << 52));
}
__device__ __forceinline__ double neg_scale2(double x, int g) { return scale2<true>(x, g); }

// FP64 arithmetic is the bound (about 1.75 multiply-adds per clock and SM, a warp's instruction at
// 18 clocks however few of its lanes are live): at 150 core and 5 x 8 active orbitals 1.5e5 of them
// per L, 0.65 ms for 2400 L.  So the loops run over exactly the elements that have work (the
// intra-fragment pairs as one list), signs and powers of two are exponent arithmetic, and sums are
// combined by one warp.  (As one loop over all a x a elements with the fragment test inside, a
// warp's FMAs were four fifths masked: 1.59 ms; now 0.92.)  The rest of the time is the
// phases' latency, overlapped by the other blocks of the SM.
// Element (r, l) of W_L, r the row that is contiguous: FP64 mode W[L][p = r][q = l]; split mode
// (gexp) Wt[q = r][(L, p = l)] * 2^gexp(L, p), in which T(p, q) of the core block is read as
// T(q, p) (T_L is symmetric).
__global__ void __launch_bounds__(256, 5)
k_per_aux(const double* __restrict__ T, int nL, int op, const double* __restrict__ dm1s,
          const double* __restrict__ dm2t, FragInfo fi, double* __restrict__ W,
          double* __restrict__ eps, double* __restrict__ vcv, double* __restrict__ vav,
          int with_grad, const int* __restrict__ gexp, int use_p) {
  pdl_begin();
  extern __shared__ double sm[];
  const int a = fi.nact, c = fi.ncore, o = c + a, nf = fi.nfrag;
  // fragment offsets, offsets of their D blocks (doff[nf] = size of all), fragment of an orbital
  __shared__ int off[LAS_MAX_FRAG + 1], doff[LAS_MAX_FRAG + 1];
  __shared__ unsigned char fk[LAS_MAX_ACT];
  __shared__ double vs[2];                 // vc, va
  double* Taa = sm;               // a*a
  double* Y = Taa + a * a;        // a*a: Y, then Y + vc D^T
  double* red = Y + a * a;        // 256
  double* cK = red + 256;         // nfrag
  double* Ds = cK + LAS_MAX_FRAG; // sum of m_K^2: the blocks of D
  const long Lb = blockIdx.x;
  const double* TL = T + Lb * (long)op * op;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    int s = 0;
    off[0] = 0;
    for (int K = 0; K < nf; ++K) {
      const int o0 = fi.off[K], o1 = fi.off[K + 1];
      doff[K] = s;
      off[K + 1] = o1;
      s += (o1 - o0) * (o1 - o0);
      for (int u = o0; u < o1; ++u) fk[u] = (unsigned char)K;
    }
    doff[nf] = s;
  }
#pragma unroll 4
  for (int i = tid; i < a * a; i += 256) {
    const int u = i / a;
    Taa[i] = TL[(long)(c + u) * op + c + i - u * a];
  }
  __syncthreads();
  const int nd = doff[nf];
  double* P = Ds + nd;            // a*a when the launch provides it (cross-fragment path)
  // fragment of element j of the list of intra-fragment pairs
  auto frag_of_pair = [&](int j) {
    int K = 0;
    while (K + 1 < nf && doff[K + 1] <= j) ++K;
    return K;
  };
  for (int j = tid; j < nd; j += 256) {
    const int K = frag_of_pair(j), m = off[K + 1] - off[K];
    const double* g = dm1s + fi.dm1_off[K] + (j - doff[K]);
    Ds[j] = g[0] + g[m * m];
  }
  __syncthreads();
  // cK = sum of D_K T_KK (one warp per fragment), vc = 2 sum_i T(i,i) (the first warp)
  for (int K = warp - 1; K < nf; K += 8) {
    double t = 0.0;
    if (K < 0) {
      for (int i = lane; i < c; i += 32) t += TL[(long)i * op + i];
    } else {
      const int oK = off[K], m = off[K + 1] - oK;
      for (int j = lane; j < m * m; j += 32) {
        const int u = j / m;
        t += Ds[doff[K] + j] * Taa[(oK + u) * a + oK + j - u * m];
      }
    }
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) t += __shfl_xor_sync(0xffffffffu, t, q);
    if (lane == 0) {
      if (K < 0) vs[0] = 2.0 * t;
      else cK[K] = t;
    }
  }
  __syncthreads();
  if (tid == 0) {
    double va = 0.0;
    for (int K = 0; K < nf; ++K) va += cK[K];
    vs[1] = va;
  }

  // Y = Gamma . T over the active block, fragment structure of Eq. las_wfn; qy += T Y.
  // Cross-fragment blocks: -sum_sigma gK_s (T_KK' gK'_s), P_s = T_aa blockdiag(g_s) first
  double qy = 0.0;
  if (nf > 1 && use_p) {
    for (int sg = 0; sg < 2; ++sg) {
      if (sg) __syncthreads();
      for (int i = tid; i < a * a; i += 256) {
        const int x = i / a, v = i - x * a;
        const int Kp = fk[v], oP = off[Kp], mP = off[Kp + 1] - oP;
        if (x >= oP && x < oP + mP) continue;
        const double* g = dm1s + fi.dm1_off[Kp] + sg * mP * mP + v - oP;
        double t = 0.0;
        for (int w = 0; w < mP; ++w) t += Taa[x * a + oP + w] * g[w * mP];
        P[i] = t;
      }
      __syncthreads();
      for (int i = tid; i < a * a; i += 256) {
        const int u = i / a, v = i - u * a;
        const int K = fk[u], oK = off[K], mK = off[K + 1] - oK;
        if (v >= oK && v < oK + mK) continue;
        const double* g = dm1s + fi.dm1_off[K] + sg * mK * mK + (u - oK) * mK;
        double t = sg ? Y[i] : 0.0;
        for (int x = 0; x < mK; ++x) t -= g[x] * P[(oK + x) * a + v];
        Y[i] = t;
        if (sg) qy += Taa[i] * t;
      }
    }
  } else if (nf > 1) {
    for (int i = tid; i < a * a; i += 256) {
      const int u = i / a, v = i - u * a;
      const int K = fk[u], oK = off[K], mK = off[K + 1] - oK;
      if (v >= oK && v < oK + mK) continue;
      const int Kp = fk[v], oP = off[Kp], mP = off[Kp + 1] - oP;
      double y = 0.0;
      for (int s = 0; s < 2; ++s) {
        const double* gK = dm1s + fi.dm1_off[K] + s * mK * mK + (u - oK) * mK;
        const double* gP = dm1s + fi.dm1_off[Kp] + s * mP * mP + v - oP;
        for (int x = 0; x < mK; ++x) {
          double t = 0.0;
          for (int w = 0; w < mP; ++w) t += Taa[(oK + x) * a + oP + w] * gP[w * mP];
          y -= gK[x] * t;
        }
      }
      Y[i] = y;
      qy += Taa[i] * y;
    }
  }
  __syncthreads();
  const double vc = vs[0], va = vs[1];
  // intra-fragment pairs: Gamma^K . T_KK + D (va - cK)
  for (int j = tid; j < nd; j += 256) {
    const int K = frag_of_pair(j), oK = off[K], m = off[K + 1] - oK, m2 = m * m;
    const int r = j - doff[K], uu = r / m, vv = r - uu * m;
    const double* g2 = dm2t + fi.dm2_off[K] + r;
    double y0 = 0.0, y1 = 0.0;
    for (int w = 0; w < m; ++w) {
      const double* t = Taa + (oK + w) * a + oK;
      const double* g = g2 + (long)w * m * m2;
      int x = 0;
      for (; x + 1 < m; x += 2) {
        y0 += g[(long)x * m2] * t[x];
        y1 += g[(long)(x + 1) * m2] * t[x + 1];
      }
      if (x < m) y0 += g[(long)x * m2] * t[x];
    }
    const double y = y0 + y1 + Ds[j] * (va - cK[K]);
    const int i = (oK + uu) * a + oK + vv;
    qy += Taa[i] * y;
    Y[i] = y + vc * Ds[doff[K] + vv * m + uu];
  }
  __syncthreads();

  // Z(i,u) = sum_v T(i, c+v) D(v,u) over core i and active u; q -= Z T.  W(i,u) = W(u,i) = -2 Z.
  double q = 0.5 * qy;
  double* WL = W + Lb * (long)op * op;
  const long wld = (long)nL * op;
  const int* gL = gexp ? gexp + Lb * (long)op : nullptr;
  if (a > 0) {
    const int du = 256 % a, di = 256 / a;
#pragma unroll 2
    for (int i = tid / a, u = tid % a; i < c;) {
      const int K = fk[u], oK = off[K], m = off[K + 1] - oK;
      const double* Ti = TL + (long)i * op + c;
      const double* d = Ds + doff[K] + u - oK;
      double z = 0.0;
      for (int v = 0; v < m; ++v) z += Ti[oK + v] * d[v * m];
      q -= z * Ti[u];
      if (with_grad) {
        if (gL) {
          W[(long)(c + u) * wld + Lb * (long)op + i] = neg_scale2(z, gL[i] + 1);
          W[(long)i * wld + Lb * (long)op + c + u] = neg_scale2(z, gL[c + u] + 1);
        } else {
          WL[(long)i * op + c + u] = WL[(long)(c + u) * op + i] = neg_scale2(z, 1);
        }
      }
      u += du;
      i += di;
      if (u >= a) {
        u -= a;
        ++i;
      }
    }
  }
  // core-core block (with sum_ij T(i,j)^2), active-active block and zero padding, a warp per row
  const int rows = with_grad ? op : c;
  for (int r = warp; r < rows; r += 8) {
    const double* Tr = TL + (long)r * op;
    double* Wr = gL ? W + (long)r * wld + Lb * (long)op : WL + (long)r * op;
    if (r < c) {
#pragma unroll 4
      for (int l = lane; l < c; l += 32) {
        const double t = Tr[l];
        q -= t * t;
        if (with_grad && l != r) Wr[l] = neg_scale2(t, (gL ? gL[l] : 0) + 2);
      }
      if (with_grad)
        for (int l = o + lane; l < op; l += 32) Wr[l] = 0.0;
    } else if (r < o) {
      const int u = r - c;
      for (int l = lane; l < a; l += 32)
        Wr[c + l] = scale2(gL ? Y[u * a + l] : Y[l * a + u], (gL ? gL[c + l] : 0) + 1);
      for (int l = o + lane; l < op; l += 32) Wr[l] = 0.0;
    } else {
      for (int l = lane; l < op; l += 32) Wr[l] = 0.0;
    }
  }
  if (with_grad)
    for (int r = tid; r < c; r += 256) {
      const double w = scale2(vc + va - TL[(long)r * op + r], (gL ? gL[r] : 0) + 2);
      if (gL) W[(long)r * wld + Lb * (long)op + r] = w;
      else WL[(long)r * op + r] = w;
    }
  const double qs = block_sum0<256>(q, red);
  if (tid == 0) {
    eps[Lb] = 0.5 * vc * vc + vc * va + qs;
    vcv[Lb] = vc;
    vav[Lb] = va;
  }
}

__global__ void __launch_bounds__(256)
k_rescale_w(const double* __restrict__ Wt, long wld, const int* __restrict__ g0,
            const int* __restrict__ g1, double* __restrict__ out) {
  pdl_begin();
  const long k = blockIdx.x * 256L + threadIdx.x;
  if (k >= wld) return;
  const long i = blockIdx.y * wld + k;
  out[i] = scale2(Wt[i], g1[k] - g0[k]);
}

// Columns of each sign of the weights of up to two densities, in order; one warp per density.
__global__ void __launch_bounds__(32)
k_sign_split(const double* __restrict__ w0, int r0, const double* __restrict__ w1, int r1, int o,
             int* __restrict__ idx, int* __restrict__ counts) {
  pdl_begin();
  const int lane = threadIdx.x;
  const double* w = blockIdx.x ? w1 : w0;
  const int r = blockIdx.x ? r1 : r0;
  int* pos = idx + 2 * blockIdx.x * o;
  int* neg = pos + o;
  int np = 0, nn = 0;
  for (int k0 = 0; k0 < r; k0 += 32) {
    const int k = k0 + lane;
    const double v = k < r ? w[k] : 0.0;
    const unsigned mp = __ballot_sync(0xffffffffu, v > 0.0), mn = __ballot_sync(0xffffffffu, v < 0.0);
    const unsigned below = (1u << lane) - 1;
    if (v > 0.0) pos[np + __popc(mp & below)] = k;
    if (v < 0.0) neg[nn + __popc(mn & below)] = k;
    np += __popc(mp);
    nn += __popc(mn);
  }
  if (lane == 0) {
    counts[2 * blockIdx.x] = np;
    counts[2 * blockIdx.x + 1] = nn;
  }
}

// Cocc[mu][j] = Cx[mu][idx[j]] * sqrt(sign * w[idx[j]]) for j < cnt, zero for cnt <= j < op
__global__ void k_pack_weighted(const double* __restrict__ Cx, const double* __restrict__ w,
                                const int* __restrict__ idx, int cnt, double sign, int n, int r,
                                int op, double* __restrict__ Cocc) {
  pdl_begin();
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= (long)n * op) return;
  const int mu = (int)(i / op), j = (int)(i % op);
  double v = 0.0;
  if (j < cnt) {
    const int k = idx[j];
    v = Cx[(long)mu * r + k] * sqrt(sign * w[k]);
  }
  Cocc[i] = v;
}

// K = scale * (its lower triangle, mirrored to the upper)
__global__ void k_mirror_lower(double* __restrict__ K, int n, double scale) {
  pdl_begin();
  long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= (long)n * n) return;
  const int i = (int)(idx / n), j = (int)(idx % n);
  if (i > j) return;   // element (j, i) is handled by its mirror image's thread
  const double v = scale * K[(long)j * n + i];
  K[idx] = v;
  if (scale != 1.0) K[(long)j * n + i] = v;
}

// dT[L][p][q] = X[L][p][q] + X[L][q][p]  (the symmetric tangent of T_L = C^T b^L C)
__global__ void k_sym_add(const double* __restrict__ X, long nL, int op, double* __restrict__ dT) {
  pdl_begin();
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  const long per = (long)op * op;
  if (i >= nL * per) return;
  const long L = i / per, r = i - L * per;
  const int p = (int)(r / op), q = (int)(r - (long)p * op);
  dT[i] = X[i] + X[L * per + (long)q * op + p];
}

// Partials of rows of `cols` values, summed in order into rows `ld` apart.
__global__ void k_reduce_partials(const double* __restrict__ part, int nsplit, long count,
                                  double* __restrict__ out, int accumulate, long cols, long ld,
                                  double scale) {
  pdl_begin();
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= count) return;
  const long o = cols == ld ? i : i / cols * ld + i % cols;
  double s = 0.0;
#pragma unroll 8
  for (int k = 0; k < nsplit; ++k) s += part[(long)k * count + i];
  out[o] = accumulate ? fma(scale, s, out[o]) : scale * s;
}

// One-electron energy sum_mu ( 2 sum_i C(mu,i) hC(mu,i) + sum_u C(mu,u) sum_v D_uv hC(mu,v) ): one
// warp per row mu, one partial per block.  The terms have either sign and n o of them cancel to the
// energy, so each thread carries the rounding errors of its products and sums along (1 to 6 terms of
// 9 FP64 instructions).  Two rows to a block, so that these are shared out over the SMs (48 orbitals:
// 96.7 us; 98.2 with eight rows to a block, 97.7 with eight rows and plain sums).  (Only these elements
// of C_occ^T h C_occ enter the energy; forming the whole matrix took a slicing pass and a product of
// its own, 45 us at 400 orbitals against 4.)
constexpr int E1_WARPS = 2;
__global__ void __launch_bounds__(32 * E1_WARPS)
k_energy_one(const double* __restrict__ Cocc, const double* __restrict__ hC, int n, int op,
             const double* __restrict__ dm1s, FragInfo fi, double* __restrict__ e1) {
  pdl_begin();
  __shared__ double red[32 * E1_WARPS];
  const int lane = threadIdx.x & 31, c = fi.ncore, o = c + fi.nact;
  double s = 0.0, comp = 0.0;
  auto add = [&](double a, double b) {   // s + comp += a b
    const double x = __dmul_rn(a, b), t = s + x, d = t - s;   // (no contraction into s + x)
    comp += fma(a, b, -x);
    comp += (s - (t - d)) + (x - d);
    s = t;
  };
  for (long mu = blockIdx.x * (long)E1_WARPS + (threadIdx.x >> 5); mu < n;
       mu += gridDim.x * (long)E1_WARPS) {
    const double* Cr = Cocc + mu * op;
    const double* hr = hC + mu * op;
    for (int p = lane; p < o; p += 32) {
      if (p < c) {
        add(2.0 * Cr[p], hr[p]);
      } else {
        const int u = p - c, K = frag_of(fi, u), oK = fi.off[K], m = fi.off[K + 1] - oK;
        const double* g = dm1s + fi.dm1_off[K] + (u - oK) * m;
        double t = 0.0;
        for (int v = 0; v < m; ++v) t += (g[v] + g[m * m + v]) * hr[c + oK + v];
        add(Cr[p], t);
      }
    }
  }
  const double t = block_sum0<32 * E1_WARPS>(s + comp, red);
  if (threadIdx.x == 0) e1[blockIdx.x] = t;
}

// E = sum_b e1_b + sum_L eps_L  (one block of 256, fixed order, compensated summation).
struct EnergySum {
  const double* eps;
  int X;
  const double* e1;
  int ne1;
  double* E;
};
__device__ void energy_sum(const EnergySum& a) {
  __shared__ double red[256];
  double s = 0.0, comp = 0.0;
  auto add = [&](double x) {  // Neumaier
    double t = s + x;
    if (fabs(s) >= fabs(x)) comp += (s - t) + x; else comp += (x - t) + s;
    s = t;
  };
#pragma unroll 4
  for (int L = threadIdx.x; L < a.X; L += 256) add(a.eps[L]);
  for (int i = threadIdx.x; i < a.ne1; i += 256) add(a.e1[i]);
  const double tot = block_sum0<256>(s + comp, red);
  if (threadIdx.x == 0) *a.E = tot;
}
__global__ void __launch_bounds__(256) k_energy_final(EnergySum a) {
  pdl_begin();
  energy_sum(a);
}

// dE/dC = [4 h C_core | 2 h C_act D | 0] + Out   (Out = sum_L H_L W_L, n x op); with es.E, the last
// block sums the energy instead.
__global__ void __launch_bounds__(256)
k_assemble_grad(const double* __restrict__ Out, const double* __restrict__ hC,
                const double* __restrict__ dm1s, FragInfo fi, int n, int nmo, int op,
                double* __restrict__ G, EnergySum es) {
  pdl_begin();
  if (es.E && blockIdx.x == gridDim.x - 1) {
    energy_sum(es);
    return;
  }
  long i = blockIdx.x * 256L + threadIdx.x;
  if (i >= (long)n * nmo) return;
  const int mu = (int)(i / nmo), q = (int)(i % nmo);
  const int c = fi.ncore, o = c + fi.nact;
  double g = 0.0;
  if (q < c) {
    g = 4.0 * hC[(long)mu * op + q] + Out[(long)mu * op + q];
  } else if (q < o) {
    const int u = q - c;
    const int K = frag_of(fi, u), oK = fi.off[K], m = fi.off[K + 1] - oK;
    const double* gK = dm1s + fi.dm1_off[K];
    double s = 0.0;
    for (int v = 0; v < m; ++v) {
      double d = gK[v * m + (u - oK)] + gK[m * m + v * m + (u - oK)];
      s += hC[(long)mu * op + c + oK + v] * d;
    }
    g = 2.0 * s + Out[(long)mu * op + q];
  }
  G[i] = g;
}

// g[p][q] = M'[p][q] - M'[q][p],  M'[p][q] = M[p][q] for q < o else 0  (M is nmo x op)
__global__ void k_antisym(const double* __restrict__ M, int nmo, int o, int op,
                          double* __restrict__ g) {
  pdl_begin();
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= (long)nmo * nmo) return;
  const int p = (int)(i / nmo), q = (int)(i % nmo);
  double x = (q < o) ? M[(long)p * op + q] : 0.0;
  double y = (p < o) ? M[(long)q * op + p] : 0.0;
  g[i] = x - y;
}

// Jp[z][pair] = sum_{L in part z} vc[L] Bp[L][pair]  (Eq. J_2 on the packed triangle; coalesced
// along pairs, two per thread, parts of the auxiliary index in grid.y).  One FP64 multiply-add per
// element read is more than the FP64 pipe does in the time of the read (800 orbitals, 1600 L: 0.92 ms
// against 0.61 ms), so the parts are there to fill every SM evenly, some 24 blocks each (one thread
// per pair over all of L: 1.08 ms, and 430 us at 400 orbitals, where it is 228 now).
constexpr int COULOMB_PAIRS = 512;
__global__ void __launch_bounds__(256)
k_coulomb_packed(const double* __restrict__ Bp, const double* __restrict__ vc, int X, int per,
                 long npair, double* __restrict__ Jp) {
  pdl_begin();
  const long i0 = blockIdx.x * (long)COULOMB_PAIRS + threadIdx.x, i1 = i0 + 256;
  const int l0 = blockIdx.y * per, l1 = min(X, l0 + per);
  double s0 = 0.0, s1 = 0.0;
  if (i1 < npair) {
    const double* b = Bp + l0 * npair + i0;
#pragma unroll 8
    for (int L = l0; L < l1; ++L, b += npair) {
      const double v = vc[L];
      s0 += v * b[0];
      s1 += v * b[256];
    }
    Jp[blockIdx.y * npair + i1] = s1;
  } else if (i0 < npair) {
    const double* b = Bp + l0 * npair + i0;
#pragma unroll 8
    for (int L = l0; L < l1; ++L, b += npair) s0 += vc[L] * b[0];
  }
  if (i0 < npair) Jp[blockIdx.y * npair + i0] = s0;
}

__device__ __forceinline__ double coulomb_sum(const double* __restrict__ Jp, int parts, long npair,
                                              long pair) {
  double s = Jp[pair];
  for (int z = 1; z < parts; ++z) s += Jp[z * npair + pair];
  return s;
}

__global__ void k_unpack_sym(const double* __restrict__ Jp, int parts, int n, double scale,
                             double* __restrict__ J) {
  pdl_begin();
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= (long)n * n) return;
  long mu = i / n, nu = i % n;
  long hi = mu > nu ? mu : nu, lo = mu > nu ? nu : mu;
  J[i] = scale * coulomb_sum(Jp, parts, (long)n * (n + 1) / 2, hi * (hi + 1) / 2 + lo);
}

__global__ void k_veff_combine(const double* __restrict__ Jp, int parts,
                               const double* __restrict__ Ka, const double* __restrict__ Kb, int n,
                               double* __restrict__ va, double* __restrict__ vb) {
  pdl_begin();
  long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i >= (long)n * n) return;
  long mu = i / n, nu = i % n;
  long hi = mu > nu ? mu : nu, lo = mu > nu ? nu : mu;
  const double j = coulomb_sum(Jp, parts, (long)n * (n + 1) / 2, hi * (hi + 1) / 2 + lo);
  va[i] = j - Ka[hi * n + lo];
  vb[i] = j - Kb[hi * n + lo];
}

// Lmu[L][mu][u] = Ht[L][u][mu], u < a: 32 values of mu per block through shared memory, so that
// reads and writes are contiguous (element by element, the reads of a warp were n apart: 50 us for
// 1600 x 400 x 16 values, against 27).
__global__ void __launch_bounds__(256)
k_transpose_ht(const double* __restrict__ Ht, int n, int a, double* __restrict__ Lmu) {
  pdl_begin();
  __shared__ double tile[LAS_MAX_ACT][33];
  const long L = blockIdx.y;
  const int mu0 = blockIdx.x * 32, nm = min(32, n - mu0);
  const double* h = Ht + L * (long)a * n + mu0;
  const int lane = threadIdx.x & 31;
  for (int u = threadIdx.x >> 5; u < a; u += 8)
    if (lane < nm) tile[u][lane] = h[(long)u * n + lane];
  __syncthreads();
  double* o = Lmu + (L * n + mu0) * (long)a;
  for (int i = threadIdx.x; i < nm * a; i += 256) o[i] = tile[i % a][i / a];
}

__global__ void k_transpose_cols(const double* __restrict__ C, int n, int op, int r,
                                 double* __restrict__ CT) {
  pdl_begin();
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;   // over r*n, mu fastest
  if (i >= (long)r * n) return;
  const int k = (int)(i / n), mu = (int)(i - (long)k * n);
  CT[i] = C[(long)mu * op + k];
}

// Coulomb traces (fixed summation order) and column maxima of |H|, one block per aux row; a warp
// takes 32 columns x a quarter of the rows k at a time (more items than warps, so that none idles
// long), and a column's maximum reaches memory only where it exceeds what is there.  The FP64
// multiply-adds of the traces are the bound (800 orbitals, 1600 x 100 rows: 0.245 ms of 0.33);
// the maxima of the exchange digits ride along instead of a pass of their own over H (0.18 ms).
__global__ void __launch_bounds__(256)
k_trace_ht(const double* __restrict__ Ht, const double* __restrict__ CT, int r, int n,
           double* __restrict__ vc, double sgn, int accumulate,
           unsigned long long* __restrict__ mx) {
  pdl_begin();
  __shared__ double red[256];
  const long b = blockIdx.x;
  const double* hb = Ht + b * (long)r * n;
  const int lane = threadIdx.x & 31, chunks = (n + 31) / 32, kq = (r + 3) / 4;
  double acc = 0.0;
  for (int it = threadIdx.x >> 5; it < 4 * chunks; it += 8) {
    const int q = it / chunks, mu = (it - q * chunks) * 32 + lane;
    const int k0 = q * kq, k1 = min(r, k0 + kq);
    if (mu >= n) continue;
    unsigned long long m = 0;
    const double* h = hb + mu;
    const double* c = CT + mu;
#pragma unroll 8
    for (int k = k0; k < k1; ++k) {
      const double v = h[(long)k * n];
      const unsigned long long a = (unsigned long long)__double_as_longlong(v) << 1;
      m = a > m ? a : m;
      if (vc) acc = fma(v, c[(long)k * n], acc);
    }
    m >>= 1;
    if (mx && m > *(volatile unsigned long long*)&mx[mu]) atomicMax(&mx[mu], m);
  }
  if (!vc) return;
  const double t = block_sum0<256>(acc, red);
  if (threadIdx.x == 0) vc[b] = accumulate ? fma(sgn, t, vc[b]) : sgn * t;
}

}  // namespace lasdf

using namespace lasdf;

static inline unsigned nblk(long count, int nt) { return (unsigned)((count + nt - 1) / nt); }

void launch_pack_cocc(const double* C, int n, int nmo, int o, int op, double* Cocc,
                      cudaStream_t s, const double* dm2, const FragInfo* fi, double* dm2t) {
  long count = (long)n * op;
  FragInfo f;
  memset(&f, 0, sizeof(f));
  if (dm2) {
    f = *fi;
    for (int K = 0; K < f.nfrag; ++K) {
      const long m = f.off[K + 1] - f.off[K];
      count += m * m * m * m;
    }
  }
  launch_chained(k_pack_cocc, nblk(count, 256), 256, 0, s, C, n, nmo, o, op, Cocc, dm2, f, dm2t);
  las_count_launch();
}

// Dynamic shared memory of k_per_aux (the factored cross-fragment path needs one more a*a buffer)
// and the most that a block may have beside its static 1 KB.
static size_t per_aux_smem(const FragInfo& fi, int use_p) {
  size_t d = 0;
  for (int K = 0; K < fi.nfrag; ++K) {
    const size_t m = fi.off[K + 1] - fi.off[K];
    d += m * m;
  }
  const size_t a2 = (size_t)fi.nact * fi.nact;
  return (2 * a2 + d + (use_p ? a2 : 0) + 256 + LAS_MAX_FRAG) * sizeof(double);
}
constexpr size_t PER_AUX_SMEM_MAX = 226 * 1024;

las_status per_aux_prepare() {
  // always the largest size, so that contexts with different active spaces coexist
  static_assert((3 * (size_t)LAS_MAX_ACT * LAS_MAX_ACT + 256 + LAS_MAX_FRAG) * sizeof(double) <=
                    PER_AUX_SMEM_MAX, "one fragment of every active orbital");
  cudaError_t e = cudaFuncSetAttribute(k_per_aux, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)PER_AUX_SMEM_MAX);
  if (e != cudaSuccess) {
    las_record_cuda_error(e, "cudaFuncSetAttribute(k_per_aux)", __FILE__, __LINE__);
    return LAS_ERR_CUDA;
  }
  return LAS_OK;
}

void launch_per_aux(const double* T, int nL, int op, const double* dm1s, const double* dm2t,
                    const FragInfo& fi, double* W, double* eps, double* vc, double* va,
                    int with_grad, const int* gexp, cudaStream_t s) {
  if (nL <= 0) return;
  const int use_p = fi.nfrag > 1 && per_aux_smem(fi, 1) <= PER_AUX_SMEM_MAX;
  // an ordinary launch, as the FP64 GEMM's: its FP64 work is to be even over the SMs
  k_per_aux<<<nL, 256, per_aux_smem(fi, use_p), s>>>(T, nL, op, dm1s, dm2t, fi, W, eps, vc, va,
                                                     with_grad, gexp, use_p);
  las_count_launch();
}

void launch_rescale_w(const double* Wt, long wld, int rows, const int* g0, const int* g1,
                      double* out, cudaStream_t s) {
  if (wld <= 0 || rows <= 0) return;
  launch_chained(k_rescale_w, dim3(nblk(wld, 256), rows), 256, 0, s, Wt, wld, g0, g1, out);
  las_count_launch();
}

void launch_sign_split(const double* w0, int r0, const double* w1, int r1, int o, int* idx,
                       int* counts, cudaStream_t s) {
  launch_chained(k_sign_split, 2, 32, 0, s, w0, r0, w1, r1, o, idx, counts);
  las_count_launch();
}

void launch_pack_weighted(const double* Cx, const double* w, const int* idx, int cnt,
                          double sign, int n, int r, int op, double* Cocc, cudaStream_t s) {
  launch_chained(k_pack_weighted, nblk((long)n * op, 256), 256, 0, s, Cx, w, idx, cnt, sign, n, r, op,
                                                         Cocc);
  las_count_launch();
}

void launch_mirror_lower(double* K, int n, double scale, cudaStream_t s) {
  launch_chained(k_mirror_lower, nblk((long)n * n, 256), 256, 0, s, K, n, scale);
  las_count_launch();
}

void launch_sym_add(const double* X, int nL, int op, double* dT, cudaStream_t s) {
  const long count = (long)nL * op * op;
  if (count <= 0) return;
  launch_chained(k_sym_add, nblk(count, 256), 256, 0, s, X, nL, op, dT);
  las_count_launch();
}

void launch_transpose_cols(const double* Cocc, int n, int op, int r, double* CT,
                           cudaStream_t s) {
  const long cnt = (long)r * n;
  if (cnt <= 0) return;
  launch_chained(k_transpose_cols, nblk(cnt, 256), 256, 0, s, Cocc, n, op, r, CT);
  las_count_launch();
}

void launch_trace_ht(const double* Ht, const double* CT, int nL, int r, int n, double* vc,
                     double sgn, int accumulate, unsigned long long* mx, cudaStream_t s) {
  if (nL <= 0) return;
  launch_chained(k_trace_ht, nL, 256, 0, s, Ht, CT, r, n, vc, sgn, accumulate, mx);
  las_count_launch();
}

void launch_reduce_partials(const double* part, int nsplit, long count, double* out,
                            int accumulate, cudaStream_t s, long cols, long ld, double scale) {
  launch_chained(k_reduce_partials, nblk(count, 256), 256, 0, s, part, nsplit, count, out, accumulate, cols,
                                                     ld, scale);
  las_count_launch();
}

void launch_assemble_grad(const double* Out, const double* hC, const double* dm1s,
                          const FragInfo& fi, int n, int nmo, int op, double* G,
                          cudaStream_t s) {
  launch_chained(k_assemble_grad, nblk((long)n * nmo, 256), 256, 0, s, Out, hC, dm1s, fi, n, nmo,
                 op, G, EnergySum{});
  las_count_launch();
}

void launch_energy(const double* eps, int X, const double* Cocc, const double* hC, int n, int op,
                   const double* dm1s, const FragInfo& fi, double* e1, double* E,
                   cudaStream_t s, const double* Out, int nmo, double* G) {
  const int nb = (int)std::min<long>(nblk(n, E1_WARPS), E1_BLOCKS);
  launch_chained(k_energy_one, nb, 32 * E1_WARPS, 0, s, Cocc, hC, n, op, dm1s, fi, e1);
  const EnergySum es{eps, X, e1, nb, E};
  if (G)
    launch_chained(k_assemble_grad, nblk((long)n * nmo, 256) + 1, 256, 0, s, Out, hC, dm1s, fi, n,
                   nmo, op, G, es);
  else
    launch_chained(k_energy_final, 1, 256, 0, s, es);
  las_count_launch(2);
}

void launch_antisym(const double* M, int nmo, int o, int op, double* g, cudaStream_t s) {
  launch_chained(k_antisym, nblk((long)nmo * nmo, 256), 256, 0, s, M, nmo, o, op, g);
  las_count_launch();
}

int coulomb_parts(long npair, int X, int sms) {
  const long blocks = (npair + COULOMB_PAIRS - 1) / COULOMB_PAIRS;
  return (int)std::max(1L, std::min({24L, (24L * sms + blocks - 1) / blocks, (long)X / 32}));
}

void launch_coulomb_packed(const double* Bp, const double* vc, int X, long npair, int parts,
                           double* Jp, cudaStream_t s) {
  dim3 grid(nblk(npair, COULOMB_PAIRS), parts);
  launch_chained(k_coulomb_packed, grid, 256, 0, s, Bp, vc, X, (X + parts - 1) / parts, npair, Jp);
  las_count_launch();
}

void launch_unpack_sym(const double* Jp, int parts, int n, double scale, double* J,
                       cudaStream_t s) {
  launch_chained(k_unpack_sym, nblk((long)n * n, 256), 256, 0, s, Jp, parts, n, scale, J);
  las_count_launch();
}

void launch_veff_combine(const double* Jp, int parts, const double* Ka, const double* Kb, int n,
                         double* va, double* vb, cudaStream_t s) {
  launch_chained(k_veff_combine, nblk((long)n * n, 256), 256, 0, s, Jp, parts, Ka, Kb, n, va, vb);
  las_count_launch();
}

void launch_transpose_ht(const double* Ht, int nL, int n, int a, double* Lmu, cudaStream_t s) {
  for (int l0 = 0; l0 < nL; l0 += 32768) {   // the grid's y extent
    const int m = std::min(nL - l0, 32768);
    launch_chained(k_transpose_ht, dim3((n + 31) / 32, m), 256, 0, s, Ht + (size_t)l0 * a * n, n, a,
                                                          Lmu + (size_t)l0 * n * a);
    las_count_launch();
  }
}
