// Observables of a converged C4v environment (arXiv 2410.11596 Sec. III.A):
// the two-site reduced density matrix of a bond and the one-site environment
// eps of Eq. (4), and the adjoint of the density matrix with the environment
// held fixed. Both are evaluated once per environment, in FP64, as a chain
// of permutes and GEMMs over the environment expanded to the plain combined
// basis; they need the individual bra and ket tensors, which carry no Z2
// symmetry (Sec. II.B).
//
// Networks (C corner, T edge, * open site):
//   rho:  C T T C / T * * T / C T T C        eps:  C T C / T * T / C T C
//
// Order of the contractions (chi = c, q = D^2). The half network of a site
// is its ring V[x0, e, k0, k1] (corners and two edges), the site's ket tensor
// over the ket halves of k0 and k1, its bra tensor over the bra halves, and the
// third edge over (e, k2):
//   2 c^2 d D^6 (1 + d) + 2 c^3 d^2 q^2 operations and arrays of at most c^2 d^2 q^2
// entries. Joining the third edge to the ring first and contracting the open
// double layer as one q^3 index took 2 c^3 q^3 + 2 c^2 d^2 q^4 operations and
// two arrays of c^2 q^3 (D = 6, c = 144: 836 against 94 GFLOP for both sites,
// 15.5 against 2.6 GB; 231 -> 10.5 ms with the same GEMM kernels). eps joins two half rings over both of their boundary
// bonds, 4 c^3 q^2 + 2 c^2 q^4 operations instead of 2 c^3 q^3 + 2 c^2 q^4.
#include "hs_ctx.cuh"

using namespace hs;

namespace {

// Open double layer of one site with its physical legs kept:
//   out[(s, s', m) | (c0, u, dd)] = A[s, ...] A[s', ...]
// where m is the open auxiliary leg (right leg r if open_right, else left l)
// and c0 the other horizontal leg; combined index x = ket + D * bra.
__global__ void open_double_layer_kernel(const double* __restrict__ A, int d, int D, bool open_right,
                                         double* __restrict__ out) {
  hs_pdl_enter();
  const int q = D * D;
  const long long total = (long long)d * d * q * q * q * q;
  const long long D4 = (long long)D * D * D * D;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    long long r = e;
    const int xd = (int)(r % q);
    r /= q;
    const int xu = (int)(r % q);
    r /= q;
    const int xc = (int)(r % q);
    r /= q;
    const int xm = (int)(r % q);
    r /= q;
    const int sb = (int)(r % d);
    const int sk = (int)(r / d);
    const int xl = open_right ? xc : xm, xr = open_right ? xm : xc;
    const long long ik = (((long long)(xu % D) * D + xl % D) * D + xd % D) * D + xr % D;
    const long long ib = (((long long)(xu / D) * D + xl / D) * D + xd / D) * D + xr / D;
    out[e] = A[sk * D4 + ik] * A[sb * D4 + ib];
  }
}

// dA from the cotangents of the two open double layers (layouts of
// open_double_layer_kernel: left site open on r, right site open on l). A
// appears in each as the ket factor (index s) and as the bra factor (s'):
//   dA[p, u, l, d, r] = sum over the other factor's indices of dao * A.
__global__ void open_double_layer_vjp_kernel(const double* __restrict__ daoL, const double* __restrict__ daoR,
                                             const double* __restrict__ A, int d, int D, double* __restrict__ dA) {
  hs_pdl_enter();
  const int q = D * D;
  const long long D4 = (long long)D * D * D * D;
  const long long nA = d * D4;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nA;
       e += (long long)gridDim.x * blockDim.x) {
    const int p = (int)(e / D4);
    long long t = e % D4;
    const int ir = (int)(t % D);
    t /= D;
    const int id = (int)(t % D);
    t /= D;
    const int il = (int)(t % D);
    const int iu = (int)(t / D);
    double acc = 0.0;
    for (int s2 = 0; s2 < d; ++s2)
      for (long long o = 0; o < D4; ++o) {
        long long oo = o;
        const int jr = (int)(oo % D);
        oo /= D;
        const int jd = (int)(oo % D);
        oo /= D;
        const int jl = (int)(oo % D);
        const int ju = (int)(oo / D);
        const double a_other = A[s2 * D4 + o];
        // this element as the ket factor: combined index = mine + D * other
        const int ku = iu + D * ju, kl = il + D * jl, kd = id + D * jd, kr = ir + D * jr;
        // this element as the bra factor: combined index = other + D * mine
        const int bu = ju + D * iu, bl = jl + D * il, bd = jd + D * id, br = jr + D * ir;
        // left site: [(s, s', m = r) | (l, u, d)]; right site: [(s, s', m = l) | (r, u, d)]
        const long long kL = ((((((long long)p * d + s2) * q + kr) * q + kl) * q + ku) * q + kd);
        const long long bL = ((((((long long)s2 * d + p) * q + br) * q + bl) * q + bu) * q + bd);
        const long long kR = ((((((long long)p * d + s2) * q + kl) * q + kr) * q + ku) * q + kd);
        const long long bR = ((((((long long)s2 * d + p) * q + bl) * q + br) * q + bu) * q + bd);
        acc += (daoL[kL] + daoL[bL] + daoR[kR] + daoR[bR]) * a_other;
      }
    dA[e] = acc;
  }
}

// Entry (s1, s1', s2, s2') of rho4 from its partial sums, added in order.
__device__ __forceinline__ double rho4_sum(const double* __restrict__ part, int e, int np) {
  double v = 0.0;
  for (int i = 0; i < np; ++i) v += part[(long long)e * np + i];
  return v;
}

// rho[(s1 s2), (s1' s2')] = rho4[s1, s1', s2, s2']; mirror the upper triangle
// when requested; tr[0] = Tr rho, tr[1] = Tr(rho h).
__global__ void finish_rho_kernel(const double* __restrict__ part, int np, int d, bool mirror,
                                  const double* __restrict__ h, double* __restrict__ rho,
                                  double* __restrict__ tr) {
  hs_pdl_enter();
  const int n = d * d;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    int I = e / n, J = e % n;
    if (mirror && I > J) {
      const int t = I;
      I = J;
      J = t;
    }
    const int s1 = I / d, s2 = I % d, t1 = J / d, t2 = J % d;
    rho[e] = rho4_sum(part, ((s1 * d + t1) * d + s2) * d + t2, np);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t0 = 0.0, t1 = 0.0;
    for (int I = 0; I < n; ++I) {
      t0 += rho[I * n + I];
      if (h)
        for (int J = 0; J < n; ++J) t1 += rho[I * n + J] * h[J * n + I];
    }
    tr[0] = t0;
    tr[1] = t1;
  }
}

// One-site reduced density matrix from the one-site environment eps (plain
// combined basis, legs (u, l, d, r), x = ket + D * bra on every leg):
//   rho1[s, s'] = sum_x eps[x_u, x_l, x_d, x_r] A[s, ket(x)] conj(A[s', bra(x)]),
// one CTA per (s, s'); complex eps, A and rho1 interleaved.
__global__ void one_site_rho_kernel(const double* __restrict__ eps, const double* __restrict__ A, int d, int D,
                                    bool cplx, double* __restrict__ rho) {
  hs_pdl_enter();
  const int sk = blockIdx.x / d, sb = blockIdx.x % d;
  const int q = D * D;
  const long long D4 = (long long)D * D * D * D;
  const long long total = (long long)q * q * q * q;
  double re = 0.0, im = 0.0;
  for (long long e = threadIdx.x; e < total; e += blockDim.x) {
    const int xr = (int)(e % q), xd = (int)((e / q) % q), xl = (int)((e / q / q) % q), xu = (int)(e / q / q / q);
    const long long ik = (((long long)(xu % D) * D + xl % D) * D + xd % D) * D + xr % D;
    const long long ib = (((long long)(xu / D) * D + xl / D) * D + xd / D) * D + xr / D;
    if (!cplx) {
      re += eps[e] * A[sk * D4 + ik] * A[sb * D4 + ib];
      continue;
    }
    const double kr = A[2 * (sk * D4 + ik)], ki = A[2 * (sk * D4 + ik) + 1];
    const double br = A[2 * (sb * D4 + ib)], bi = -A[2 * (sb * D4 + ib) + 1];  // conj
    const double pr = kr * br - ki * bi, pi = kr * bi + ki * br;
    const double er = eps[2 * e], ei = eps[2 * e + 1];
    re += er * pr - ei * pi;
    im += er * pi + ei * pr;
  }
  __shared__ double red[2][32];
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x / 32] = re;
    red[1][threadIdx.x / 32] = im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    if (cplx) {
      rho[2 * blockIdx.x] = a;
      rho[2 * blockIdx.x + 1] = b;
    } else {
      rho[blockIdx.x] = a;
    }
  }
}

// tr[0] = Tr rho1, tr[1] = Tr(rho1 h) (h a real d x d matrix, may be null);
// complex: tr = (Re, Im) of each.
__global__ void finish_rho1_kernel(const double* __restrict__ rho, int d, bool cplx, const double* __restrict__ h,
                                   double* __restrict__ tr) {
  hs_pdl_enter();
  if (threadIdx.x != 0) return;
  double t0r = 0.0, t0i = 0.0, t1r = 0.0, t1i = 0.0;
  for (int i = 0; i < d; ++i) {
    t0r += cplx ? rho[2 * (i * d + i)] : rho[i * d + i];
    t0i += cplx ? rho[2 * (i * d + i) + 1] : 0.0;
    if (h)
      for (int j = 0; j < d; ++j) {
        t1r += (cplx ? rho[2 * (i * d + j)] : rho[i * d + j]) * h[j * d + i];
        t1i += cplx ? rho[2 * (i * d + j) + 1] * h[j * d + i] : 0.0;
      }
  }
  if (cplx) {
    tr[0] = t0r;
    tr[1] = t0i;
    tr[2] = t1r;
    tr[3] = t1i;
  } else {
    tr[0] = t0r;
    tr[1] = t1r;
  }
}

// Cotangent of rho for E = Re Tr(rho h) / Tr rho:
//   drho[I, J] = dE (conj(1 / t0) h[J, I] - conj(t1 / t0^2) delta_IJ),
// t0 = Tr rho, t1 = Tr(rho h) as written by the finish kernels (real: tr =
// (t0, t1); complex: tr = (Re t0, Im t0, Re t1, Im t1), drho interleaved).
__global__ void energy_cotangent_kernel(const double* __restrict__ tr, const double* __restrict__ h, int n,
                                        bool cplx, double dE, double* __restrict__ drho) {
  hs_pdl_enter();
  const double t0r = tr[0], t0i = cplx ? tr[1] : 0.0;
  const double t1r = cplx ? tr[2] : tr[1], t1i = cplx ? tr[3] : 0.0;
  // a = 1 / t0, b = t1 / t0^2 (complex division by |t0|^2)
  const double m2 = t0r * t0r + t0i * t0i;
  const double ar = t0r / m2, ai = -t0i / m2;
  const double sr = ar * ar - ai * ai, si = 2.0 * ar * ai;  // 1 / t0^2
  const double br = t1r * sr - t1i * si, bi = t1r * si + t1i * sr;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int I = e / n, J = e % n;
    const double hv = h ? h[J * n + I] : 0.0;
    // conj(a) hv - conj(b) delta
    const double re = ar * hv - (I == J ? br : 0.0);
    const double im = -ai * hv + (I == J ? bi : 0.0);
    if (cplx) {
      drho[2 * e] = dE * re;
      drho[2 * e + 1] = dE * im;
    } else {
      drho[e] = dE * re;
    }
  }
}

unsigned grid_for(long long n) {
  long long g = (n + 255) / 256;
  if (g > 4096) g = 4096;
  if (g < 1) g = 1;
  return (unsigned)g;
}

// A dense tensor with its row and column legs as an all-even Z2 matrix.
Z2Mat dense(std::initializer_list<long long> rows, std::initializer_list<long long> cols) {
  Fused r = fused0(), c = fused0();
  for (long long v : rows) r.leg[r.k++] = make_sect((int)v, 0);
  for (long long v : cols) c.leg[c.k++] = make_sect((int)v, 0);
  return mat(r, c);
}

GemmGroup dense_gemm(long long M, long long N, long long K) {
  GemmGroup g{};
  g.n = 1;
  g.p[0].M = (int)M;
  g.p[0].N = (int)N;
  g.p[0].K = (int)K;
  g.p[0].lda = (int)K;
  g.p[0].ldb = (int)K;
  g.p[0].ldc = (int)N;
  return g;
}

// Complex rho[(s1 s2), (s1' s2')] = rho4[s1, s1', s2, s2'] (planar in,
// interleaved out); tr[0..1] = Tr rho, tr[2..3] = Tr(rho h) for real h.
__global__ void finish_rho_c_kernel(const double* __restrict__ re4, const double* __restrict__ im4, int np, int d,
                                    const double* __restrict__ h, double* __restrict__ rho, double* __restrict__ tr) {
  hs_pdl_enter();
  const int n = d * d;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int I = e / n, J = e % n;
    const int s1 = I / d, s2 = I % d, t1 = J / d, t2 = J % d;
    const int src = ((s1 * d + t1) * d + s2) * d + t2;
    rho[2 * e] = rho4_sum(re4, src, np);
    rho[2 * e + 1] = rho4_sum(im4, src, np);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, c = 0.0, f = 0.0;
    for (int I = 0; I < n; ++I) {
      a += rho[2 * (I * n + I)];
      b += rho[2 * (I * n + I) + 1];
      if (h)
        for (int J = 0; J < n; ++J) {
          c += rho[2 * (I * n + J)] * h[J * n + I];
          f += rho[2 * (I * n + J) + 1] * h[J * n + I];
        }
    }
    tr[0] = a;
    tr[1] = b;
    tr[2] = c;
    tr[3] = f;
  }
}

// ---- kernels of the two-site network ------------------------------------------
//
// A half network L or R is [(x0, s, mk, s', mb) | x4]: boundary bond, ket and
// bra physical index with the ket and bra halves of the bond m between the
// sites, the other boundary bond. Complex ones are planar.

constexpr int kRhoParts = 64;

// Partial sums of rho4[s1, s1', s2, s2'] = sum_{x0, mk, mb, x4} L R: part[pair][i]
// from every kRhoParts-th (x0, mk, mb). The d^4 c^2 q FMAs are 23 us of the FP64
// pipe at D = 6, c = 144; it takes 161 us, waiting for its operands from L2; a 4 x 4 GEMM over
// c^2 q would leave 255 of 256 tile entries idle.
__global__ void __launch_bounds__(128) rho4_kernel(const double* __restrict__ Lr, const double* __restrict__ Li,
                                                   const double* __restrict__ Rr, const double* __restrict__ Ri, int d,
                                                   int D, int chi, double* __restrict__ part_re,
                                                   double* __restrict__ part_im) {
  hs_pdl_enter();
  const int pair = blockIdx.x, s2b = pair % d, s2 = pair / d % d, s1b = pair / d / d % d, s1 = pair / d / d / d;
  double re = 0.0, im = 0.0;
  for (int u = blockIdx.y; u < chi * D * D; u += kRhoParts) {
    const int mb = u % D, mk = u / D % D, x0 = u / D / D;
    const long long lo = (((((long long)x0 * d + s1) * D + mk) * d + s1b) * D + mb) * chi;
    const long long ro = (((((long long)x0 * d + s2) * D + mk) * d + s2b) * D + mb) * chi;
    for (int x = threadIdx.x; x < chi; x += blockDim.x) {
      re += Lr[lo + x] * Rr[ro + x];
      if (Li) {
        re -= Li[lo + x] * Ri[ro + x];
        im += Lr[lo + x] * Ri[ro + x] + Li[lo + x] * Rr[ro + x];
      }
    }
  }
  __shared__ double red[2][4];
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x / 32] = re;
    red[1][threadIdx.x / 32] = im;
  }
  __syncthreads();
  if (threadIdx.x < (Li ? 2 : 1))
    (threadIdx.x ? part_im : part_re)[(long long)pair * kRhoParts + blockIdx.y] =
        (red[threadIdx.x][0] + red[threadIdx.x][1]) + (red[threadIdx.x][2] + red[threadIdx.x][3]);
}

// Cotangent of one half network from that of rho and the other half:
//   out[.., s, .., s', ..] = sum_{o, o'} g conj(in[.., o, .., o', ..]),
// g = drho[(s o), (s' o')] for the left half, drho[(o s), (o' s')] for the right
// one (drho real, or interleaved complex). One thread per (x0, mk, mb, x4).
__global__ void half_adjoint_kernel(const double* __restrict__ drho, const double* __restrict__ in_re,
                                    const double* __restrict__ in_im, int d, int D, int chi, bool left,
                                    double* __restrict__ out_re, double* __restrict__ out_im) {
  hs_pdl_enter();
  const long long total = (long long)chi * D * D * chi;
  const int n = d * d;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int x4 = (int)(e % chi);
    const long long u = e / chi;
    const int mb = (int)(u % D), mk = (int)(u / D % D);
    const long long x0 = u / D / D;
    auto at = [&](int s, int sb) { return (((((x0 * d + s) * D + mk) * d + sb) * D + mb) * chi + x4); };
    for (int s = 0; s < d; ++s)
      for (int sb = 0; sb < d; ++sb) {
        double re = 0.0, im = 0.0;
        for (int o = 0; o < d; ++o)
          for (int ob = 0; ob < d; ++ob) {
            const int I = left ? s * d + o : o * d + s, J = left ? sb * d + ob : ob * d + sb;
            const long long src = at(o, ob);
            if (!in_im) {
              re += drho[I * n + J] * in_re[src];
            } else {
              const double gr = drho[2 * (I * n + J)], gi = drho[2 * (I * n + J) + 1];
              re += gr * in_re[src] + gi * in_im[src];
              im += gi * in_re[src] - gr * in_im[src];
            }
          }
        out_re[at(s, sb)] = re;
        if (in_im) out_im[at(s, sb)] = im;
      }
  }
}

// Which legs of A[s, u, l, d, r] (1..4) are a site's m, k2, k0 and k1.
struct SiteLegs {
  int m, k2, k0, k1;
};

// Position of (s, m, k2, k0, k1) in A[s, u, l, d, r].
__device__ __forceinline__ int a_index(int s, int m, int k2, int k0, int k1, SiteLegs g, int D) {
  int x[5];
  x[0] = s;
  x[g.m] = m;
  x[g.k2] = k2;
  x[g.k0] = k0;
  x[g.k1] = k1;
  return (((x[0] * D + x[1]) * D + x[2]) * D + x[3]) * D + x[4];
}

// The cotangent Q[(s, mk, s', mb, k2k, k2b) | (k0b, k0k, k1b, k1k)] of a site's open
// double layer a = A_ket conj(A_bra), contracted with A row by row (one block
// per row of q^2 contiguous entries, so that Q is read once):
//   pk[row][k0k, k1k] = sum_{k0b, k1b} Q A[s', bra],
//   pb[row][k0b, k1b] = sum_{k0k, k1k} conj(Q) A[s, ket].
// site_sum_kernel adds them up. Bound by reading Q (54 MB at D = 6).
__global__ void __launch_bounds__(64) site_adjoint_kernel(const double* __restrict__ Qr, const double* __restrict__ Qi,
                                                          const double* __restrict__ A, int d, int D, SiteLegs g,
                                                          bool staged, double* __restrict__ pk,
                                                          double* __restrict__ pb) {
  hs_pdl_enter();
  extern __shared__ double sh[];
  const int q = D * D, cx = Qi ? 2 : 1;
  double* ket = sh;  // A[s, ket] over (k0, k1), A[s', bra]
  double* bra = ket + cx * q;
  double* row = bra + cx * q;  // the row's q^2 entries (complex: re, then im), when they fit
  long long r = blockIdx.x;
  const int k2b = (int)(r % D), k2k = (int)(r / D % D), mb = (int)(r / q % D), sb = (int)(r / q / D % d),
            mk = (int)(r / q / D / d % D), s = (int)(r / q / D / d / D);
  const long long base = (long long)blockIdx.x * q * q;
  if (staged)
    for (int i = threadIdx.x; i < q * q; i += blockDim.x) {
      row[i] = Qr[base + i];
      if (cx == 2) row[q * q + i] = Qi[base + i];
    }
  const double* qr = staged ? row : Qr + base;
  const double* qi = staged ? row + q * q : Qi + base;
  for (int i = threadIdx.x; i < q; i += blockDim.x) {
    const int ik = a_index(s, mk, k2k, i / D, i % D, g, D), ib = a_index(sb, mb, k2b, i / D, i % D, g, D);
    for (int c = 0; c < cx; ++c) {
      ket[c * q + i] = A[cx * ik + c];
      bra[c * q + i] = A[cx * ib + c];
    }
  }
  __syncthreads();
  for (int o = threadIdx.x; o < 2 * q; o += blockDim.x) {
    const bool is_ket = o < q;
    const int i0 = o % q / D, i1 = o % D;
    double re = 0.0, im = 0.0;
    for (int j = 0; j < q; ++j) {
      const int j0 = j / D, j1 = j % D;
      const int at = is_ket ? ((j0 * D + i0) * D + j1) * D + i1 : ((i0 * D + j0) * D + i1) * D + j1;
      const double* a = is_ket ? bra : ket;
      if (cx == 1) {
        re += qr[at] * a[j];
      } else {
        const double gr = qr[at], gi = is_ket ? qi[at] : -qi[at];
        re += gr * a[j] - gi * a[q + j];
        im += gr * a[q + j] + gi * a[j];
      }
    }
    double* out = (is_ket ? pk : pb) + ((long long)blockIdx.x * q + o % q) * cx;
    out[0] = re;
    if (cx == 2) out[1] = im;
  }
}

// dA (= or +=) the sums of pk over (s', mb, k2b) and of pb over (s, mk, k2k).
__global__ void site_sum_kernel(const double* __restrict__ pk, const double* __restrict__ pb, int d, int D, int cx,
                                SiteLegs g, bool add, double* __restrict__ dA) {
  hs_pdl_enter();
  const int q = D * D, nS = d * D;
  const long long nA = (long long)d * q * q;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < nA * cx;
       e += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(e % cx);
    const int i = (int)(e / cx);
    const int k1 = i % D, k0 = i / D % D, k2 = i / q % D, m = i / q / D % D, s = i / q / q;
    const int S = s * D + m;
    double v = 0.0;
    for (int T = 0; T < nS; ++T)
      for (int o = 0; o < D; ++o) {
        const long long rk = (((long long)S * nS + T) * D + k2) * D + o;  // this element as the ket
        const long long rb = (((long long)T * nS + S) * D + o) * D + k2;  // as the bra
        v += pk[(rk * q + k0 * D + k1) * cx + c] + pb[(rb * q + k0 * D + k1) * cx + c];
      }
    const long long a = (long long)a_index(s, m, k2, k0, k1, g, D) * cx + c;
    dA[a] = add ? dA[a] + v : v;
  }
}

// ---- the chains -------------------------------------------------------------------

// A real array, or a complex one as planar real and imaginary parts.
struct ZBuf {
  double* re;
  double* im;
  ZBuf at(long long n) const { return {re + n, im ? im + n : nullptr}; }
};

// The largest intermediates, c^2 d^2 q^2 entries, are made a few of their leading
// index's values at a time where they would hold more than this (4 GB a part): at d = 2,
// D = 6, c = 144 they hold 0.9 GB, at d = 16, D = 7, c = 196 two of them were 378 GB.
constexpr long long kObsElems = 1ll << 29;

// One observable's evaluation: real or complex arithmetic on the context's buffers.
struct Obs {
  hs_ctx ctx;
  bool cx;
  hs_gemm_backend be;
  long long c, q, d, D;

  // buffer i (0 <= i < 20), at least n entries
  hs_status buf(int i, long long n, ZBuf* z) const {
    HS_TRY(ctx->zr[2 * i].ensure(n * 8));
    if (cx) HS_TRY(ctx->zr[2 * i + 1].ensure(n * 8));
    *z = {ctx->zr[2 * i].d(), cx ? ctx->zr[2 * i + 1].d() : nullptr};
    return HS_OK;
  }
  // C[M | N] = A[M | K] B[N | K]^T (or conj(B))
  hs_status mul(long long M, long long N, long long K, ZBuf A, ZBuf B, ZBuf C, bool conj_b = false) const {
    const GemmGroup g = dense_gemm(M, N, K);
    if (cx) return zgemm_f64(ctx, g, A.re, A.im, B.re, B.im, C.re, C.im, conj_b);
    return gemm(ctx, be, g, A.re, B.re, C.re);
  }
  hs_status perm(const Z2Mat& in, const Z2Mat& out, std::initializer_list<int> p, ZBuf src, ZBuf dst) const {
    HS_TRY(permute(ctx, in, out, p, src.re, dst.re));
    return cx ? permute(ctx, in, out, p, src.im, dst.im) : HS_OK;
  }
  // interleaved complex -> planar
  hs_status planar(const double* src, long long n, ZBuf dst, DBuf& tmp) const {
    HS_TRY(tmp.ensure(2 * n * 8));
    HS_TRY(permute(ctx, dense({n}, {2}), dense({2}, {n}), {1, 0}, src, tmp.d()));
    HS_CUDA(cudaMemcpyAsync(dst.re, tmp.d(), n * 8, cudaMemcpyDeviceToDevice, ctx->stream));
    HS_CUDA(cudaMemcpyAsync(dst.im, tmp.d() + n, n * 8, cudaMemcpyDeviceToDevice, ctx->stream));
    return HS_OK;
  }
};

// Buffers kept between the steps of a chain; the others are scratch.
enum { bT = 0, bH, bV, bA, bL, bR, bPart, bScratch };

Obs make_obs(hs_ctx ctx, const hs_env* env, int d, int D) {
  return {ctx, env->dtype == HS_C128, env->gemm_backend, (long long)env->chi_even + env->chi_odd, (long long)D * D, d,
          D};
}

// The environment in the plain combined basis: T[(a, x) | b] (bT) and the half
// ring H[(a, x) | b] = C[a, c] T[c, x, e] C[e, b] (bH).
hs_status half_ring(const Obs& o, const hs_env* env, int D) {
  hs_ctx ctx = o.ctx;
  const long long c = o.c, q = o.q, c2 = c * c, cqc = c * q * c;
  ZBuf C, T, Ct, Tq, H1, H;
  HS_TRY(o.buf(bT, cqc, &T));
  HS_TRY(o.buf(bH, cqc, &H));
  HS_TRY(o.buf(bScratch, c2, &C));
  HS_TRY(o.buf(bScratch + 1, c2, &Ct));
  HS_TRY(o.buf(bScratch + 2, cqc, &Tq));
  HS_TRY(o.buf(bScratch + 3, cqc, &H1));
  if (!o.cx) {
    HS_CUDA(launch_env_to_dense(env->C, env->T, D, env->chi_even, env->chi_odd, env->basis == HS_BASIS_HERMITIAN, C.re,
                                T.re, ctx->stream));
  } else if (env->basis == HS_BASIS_DENSE) {
    // a complex environment of the plain basis is stored dense already
    HS_TRY(o.planar(env->C, c2, C, ctx->r[2]));
    HS_TRY(o.planar(env->T, cqc, T, ctx->r[2]));
  } else {
    HS_TRY(ctx->r[0].ensure(2 * c2 * 8));
    HS_TRY(ctx->r[1].ensure(2 * cqc * 8));
    HS_CUDA(launch_env_to_dense_graded(env->C, env->T, D, env->chi_even, env->chi_odd, ctx->r[0].d(), ctx->r[1].d(),
                                       ctx->stream));
    HS_TRY(o.planar(ctx->r[0].d(), c2, C, ctx->r[2]));
    HS_TRY(o.planar(ctx->r[1].d(), cqc, T, ctx->r[2]));
  }
  HS_TRY(o.perm(dense({c}, {c}), dense({c}, {c}), {1, 0}, C, Ct));
  HS_TRY(o.perm(dense({c, q}, {c}), dense({q, c}, {c}), {1, 2, 0}, T, Tq));  // Tq[(x, e) | c]
  // A real corner is diagonal, or nearly: a row's one large entry meets entries of any
  // size, so the digit slices would leave a tenth of the products' entries to FMAs
  // (c = 100, q = 25: 107 us a product against the FP64 kernel's 55).
  const NoSlices keep(ctx, !o.cx);
  HS_TRY(o.mul(c, q * c, c, C, Tq, H1));                                      // H1[a | (x, e)]
  return o.mul(c * q, c, c, H1, Ct, H);                                       // H[(a, x) | b]
}

// eps[u, l, d, r] (Eq. (4)) from two half rings joined over both boundary bonds.
//   real:    up[t, u, l, t'..] E[t, u, b] T[t, l, t'] and T[b, r, b'] E[t', d, b'] over (b, t')
//   complex: H[a, u, b] T[b, r, b'] and H[b', d, a'] T[a', l, a] over (a, b') (clockwise ring)
hs_status one_site_chain(hs_ctx ctx, const hs_env* env, int d, int D, double* eps) {
  const Obs o = make_obs(ctx, env, d, D);
  HS_TRY(half_ring(o, env, D));
  const long long c = o.c, q = o.q, n = c * c * q * q, q4 = q * q * q * q;
  ZBuf T, H, W1, W2, U, W, E, x1, x2;
  HS_TRY(o.buf(bT, c * q * c, &T));
  HS_TRY(o.buf(bH, c * q * c, &H));
  HS_TRY(o.buf(bScratch, n, &W1));
  HS_TRY(o.buf(bScratch + 1, n, &U));
  HS_TRY(o.buf(bScratch + 2, n, &W2));
  HS_TRY(o.buf(bScratch + 3, n, &W));
  HS_TRY(o.buf(bScratch + 4, c * q * c, &x1));
  HS_TRY(o.buf(bScratch + 5, c * q * c, &x2));
  HS_TRY(o.buf(bScratch + 6, q4, &E));
  const Z2Mat edge = dense({c, q}, {c}), rev = dense({c, q}, {c});
  if (!o.cx) {
    HS_TRY(o.perm(edge, rev, {2, 1, 0}, H, x1));                                                    // [(b, u) | t]
    HS_TRY(o.perm(edge, rev, {2, 1, 0}, T, x2));                                                    // [(t', l) | t]
    HS_TRY(o.mul(c * q, c * q, c, x1, x2, W1));                                                     // [(b, u) | (t', l)]
    HS_TRY(o.perm(dense({c, q}, {c, q}), dense({q, q}, {c, c}), {1, 3, 0, 2}, W1, U));              // [(u, l) | (b, t')]
    HS_TRY(o.mul(c * q, c * q, c, T, H, W2));                                                       // [(b, r) | (t', d)]
    HS_TRY(o.perm(dense({c, q}, {c, q}), dense({q, q}, {c, c}), {3, 1, 0, 2}, W2, W));              // [(d, r) | (b, t')]
    return gemm(ctx, o.be, dense_gemm(q * q, q * q, c * c), U.re, W.re, eps);                       // [(u, l) | (d, r)]
  }
  HS_TRY(o.perm(edge, rev, {2, 1, 0}, T, x1));                                                      // [(b', r) | b]
  HS_TRY(o.mul(c * q, c * q, c, H, x1, W1));                                                        // [(a, u) | (b', r)]
  HS_TRY(o.perm(dense({c, q}, {c, q}), dense({q, q}, {c, c}), {1, 3, 0, 2}, W1, U));                // [(u, r) | (a, b')]
  HS_TRY(o.perm(edge, rev, {2, 1, 0}, T, x1));                                                      // [(a, l) | a']
  HS_TRY(o.mul(c * q, c * q, c, x1, H, W2));                                                        // [(a, l) | (b', d)]
  HS_TRY(o.perm(dense({c, q}, {c, q}), dense({q, q}, {c, c}), {1, 3, 0, 2}, W2, W));                // [(l, d) | (a, b')]
  HS_TRY(o.mul(q * q, q * q, c * c, U, W, E));                                                      // [(u, r) | (l, d)]
  ZBuf Eo;
  HS_TRY(ctx->r[2].ensure(2 * q4 * 8));
  Eo = {ctx->r[2].d(), ctx->r[2].d() + q4};
  HS_TRY(o.perm(dense({q, q}, {q, q}), dense({q, q}, {q, q}), {0, 2, 3, 1}, E, Eo));                // u, l, d, r
  return permute(ctx, dense({2}, {q4}), dense({q4}, {2}), {1, 0}, ctx->r[2].d(), eps);
}

// The legs of the two sites (index into A[s, u, l, d, r]); m joins the sites.
//   real:    V over the site's outer leg, then up; the bottom edge closes k2 = down
//   complex: left chain down, outer, up; right chain up, outer, down (clockwise)
SiteLegs site_legs(bool cx, bool left) {
  if (!cx) return left ? SiteLegs{4, 3, 2, 1} : SiteLegs{2, 3, 4, 1};
  return left ? SiteLegs{4, 1, 3, 2} : SiteLegs{2, 3, 1, 4};
}

// A site's half network out[(x0, S, S') | x4], S = (s, m): Xp[(x0, e, k0b, k1b) | (k0k, k1k)]
// with the ket tensor, the bra tensor and the edge T[e, k2, x4]. Every step keeps x0
// outermost, so that it runs on ranges of x0 (kObsElems).
hs_status site_half(const Obs& o, ZBuf Xp, const SiteLegs& g, ZBuf out) {
  const long long c = o.c, D = o.D, q = o.q, S = o.d * D;
  ZBuf A, AP, T, TB, Y1, Y1p, Y2, Xf;
  const long long per = c * S * D * (q > S * D ? q : S * D);  // entries a value of x0
  const long long cb = kObsElems / per > c ? c : kObsElems / per > 0 ? kObsElems / per : 1;
  HS_TRY(o.buf(bA, S * D * q, &A));
  HS_TRY(o.buf(bT, c * q * c, &T));
  HS_TRY(o.buf(bScratch + 1, S * D * q, &AP));
  HS_TRY(o.buf(bScratch + 2, c * q * c, &TB));
  HS_TRY(o.buf(bScratch + 3, cb * per, &Y1));
  HS_TRY(o.buf(bScratch + 4, cb * per, &Y1p));
  Y2 = Y1;
  Xf = Y1p;
  HS_TRY(o.perm(dense({o.d, D, D, D}, {D}), dense({o.d, D, D}, {D, D}), {0, g.m, g.k2, g.k0, g.k1}, A, AP));
  HS_TRY(o.perm(dense({c, D, D}, {c}), dense({c}, {c, D, D}), {3, 0, 2, 1}, T, TB));              // [x4 | (e, k2k, k2b)]
  for (long long x0 = 0; x0 < c; x0 += cb) {
    const long long b = c - x0 < cb ? c - x0 : cb;
    HS_TRY(o.mul(b * c * q, S * D, q, Xp.at(x0 * c * q * q), AP, Y1));                               // [(x0, e, k0b, k1b) | (S, k2k)]
    HS_TRY(o.perm(dense({b * c, q}, {S * D}), dense({b * c, S * D}, {q}), {0, 2, 1}, Y1, Y1p));      // [(x0, e, S, k2k) | (k0b, k1b)]
    HS_TRY(o.mul(b * c * S * D, S * D, q, Y1p, AP, Y2, true));                                       // [(x0, e, S, k2k) | (S', k2b)]
    HS_TRY(o.perm(dense({b, c, S, D}, {S, D}), dense({b, S, S}, {c, D, D}), {0, 2, 4, 1, 3, 5}, Y2, Xf));
    HS_TRY(o.mul(b * S * S, c, c * q, Xf, TB, out.at(x0 * S * S * c)));
  }
  return HS_OK;
}

// Forward chain of the two-site network: leaves T (bT), the ring V (bV, [(e, k0) | (x0, k1)]
// real, [(x0, k0) | (e, k1)] complex), the tensor A (bA), the half networks of
// the left site L[(x0, S, S') | x4] (bL) and the right one (bR, x0 and x4 those of
// L), and the partial sums of rho4 (bPart).
hs_status rdm_chain(hs_ctx ctx, const hs_env* env, const double* A, int d, int D) {
  const Obs o = make_obs(ctx, env, d, D);
  HS_TRY(half_ring(o, env, D));
  const long long c = o.c, q = o.q, nA = (long long)d * q * q, nh = c * c * d * d * q, nx = c * c * q * q;
  ZBuf T, H, V, Az, L, R, part, Xp, x1, x2;
  HS_TRY(o.buf(bT, c * q * c, &T));
  HS_TRY(o.buf(bH, c * q * c, &H));
  HS_TRY(o.buf(bV, nx, &V));
  HS_TRY(o.buf(bA, nA, &Az));
  HS_TRY(o.buf(bL, nh, &L));
  HS_TRY(o.buf(bR, nh, &R));
  HS_TRY(o.buf(bPart, (long long)d * d * d * d * kRhoParts, &part));
  HS_TRY(o.buf(bScratch, nx, &Xp));
  HS_TRY(o.buf(bScratch + 1, c * q * c, &x1));
  HS_TRY(o.buf(bScratch + 2, c * q * c, &x2));
  if (o.cx)
    HS_TRY(o.planar(A, nA, Az, ctx->r[2]));
  else
    HS_CUDA(cudaMemcpyAsync(Az.re, A, nA * 8, cudaMemcpyDeviceToDevice, ctx->stream));
  const Z2Mat edge = dense({c, q}, {c});
  const Z2Mat vl = dense({c, D, D}, {c, D, D}), xl = dense({c, c, D, D}, {D, D});
  if (!o.cx) {
    // V[b, l, t', u] = E[t, l, b] T[t, u, t']: x0 = t', e = b, k0 = l (r on the right), k1 = u
    HS_TRY(o.perm(edge, edge, {2, 1, 0}, H, x1));
    HS_TRY(o.perm(edge, edge, {2, 1, 0}, T, x2));
    HS_TRY(o.mul(c * q, c * q, c, x1, x2, V));
    HS_TRY(o.perm(vl, xl, {3, 0, 1, 4, 2, 5}, V, Xp));
  } else {
    // V[x0, k0, e, k1] = T[x0, k0, a] H[a, k1, e]
    HS_TRY(o.perm(edge, edge, {2, 1, 0}, H, x1));
    HS_TRY(o.mul(c * q, c * q, c, T, x1, V));
    HS_TRY(o.perm(vl, xl, {0, 3, 1, 4, 2, 5}, V, Xp));
  }
  HS_TRY(site_half(o, Xp, site_legs(o.cx, true), L));
  if (!o.cx) {
    HS_TRY(site_half(o, Xp, site_legs(false, false), R));
  } else {
    // the right chain runs from t to b: exchanged to the left one's bonds
    ZBuf Rt;
    HS_TRY(o.buf(bScratch + 5, nh, &Rt));
    HS_TRY(site_half(o, Xp, site_legs(true, false), Rt));
    HS_TRY(o.perm(dense({c, (long long)d * d * q}, {c}), dense({c, (long long)d * d * q}, {c}), {2, 1, 0}, Rt, R));
  }
  hs_launch(rho4_kernel, dim3((unsigned)(d * d * d * d), kRhoParts), 128, 0, ctx->stream, (const double*)L.re,
            (const double*)L.im, (const double*)R.re, (const double*)R.im, d, D, (int)c, part.re, part.im);
  HS_CUDA(cudaGetLastError());
  ctx->launches += 1;
  return HS_OK;
}

// rho and its traces from rdm_chain's partial sums.
hs_status finish_rdm(hs_ctx ctx, const hs_env* env, int d, int D, const double* h, double* rho, double* tr) {
  const Obs o = make_obs(ctx, env, d, D);
  ZBuf part;
  HS_TRY(o.buf(bPart, (long long)d * d * d * d * kRhoParts, &part));
  if (o.cx)
    hs_launch(finish_rho_c_kernel, 1, 256, 0, ctx->stream, (const double*)part.re, (const double*)part.im, kRhoParts, d,
              h, rho, tr);
  else
    hs_launch(finish_rho_kernel, 1, 256, 0, ctx->stream, (const double*)part.re, kRhoParts, d,
              env->basis == HS_BASIS_HERMITIAN, h, rho, tr);
  HS_CUDA(cudaGetLastError());
  ctx->launches += 1;
  return HS_OK;
}

// Reverse pass of rdm_chain, which must have run on the same environment and A
// just before: drho (d^4, real or interleaved complex) -> dA. Per site: the
// half network's cotangent, through the edge to the ring and the open double
// layer, Q = dXf conj(V) over the boundary bonds, then A (site_adjoint_kernel).
hs_status rdm_vjp_after_chain(hs_ctx ctx, const hs_env* env, int d, int D, const double* A, const double* drho,
                              double* dA_out) {
  const Obs o = make_obs(ctx, env, d, D);
  const long long c = o.c, q = o.q, S = (long long)d * D, nh = c * c * S * S, nx = c * c * q * q, per = c * S * c * q,
                  nq = S * S * q * q * q;
  const long long sb = kObsElems / per > S ? S : kObsElems / per > 0 ? kObsElems / per : 1;  // values of S at a time
  const long long nf = sb * per;
  ZBuf T, V, half[2], dh, dht, dS, TT, Vt, F, Fp, Q;
  HS_TRY(o.buf(bT, c * q * c, &T));
  HS_TRY(o.buf(bV, nx, &V));
  HS_TRY(o.buf(bL, nh, &half[0]));
  HS_TRY(o.buf(bR, nh, &half[1]));
  HS_TRY(o.buf(bScratch, nx, &Vt));
  HS_TRY(o.buf(bScratch + 2, c * q * c, &TT));
  HS_TRY(o.buf(bScratch + 3, nf, &F));
  HS_TRY(o.buf(bScratch + 4, nf, &Fp));
  HS_TRY(o.buf(bScratch + 5, nh, &dh));
  HS_TRY(o.buf(bScratch + 6, nq, &Q));
  HS_TRY(o.buf(bScratch + 7, nh, &dht));
  if (sb < S) HS_TRY(o.buf(bScratch + 8, nh, &dS));
  const int cx = o.cx ? 2 : 1;
  const long long rows = S * S * q, npart = rows * q * cx;
  HS_TRY(ctx->hb[0].ensure(2 * npart * 8));
  double *pk = ctx->hb[0].d(), *pb = pk + npart;
  HS_TRY(o.perm(dense({c, D, D}, {c}), dense({c, D, D}, {c}), {0, 2, 1, 3}, T, TT));  // [(e, k2k, k2b) | x4]
  if (!o.cx)
    HS_TRY(o.perm(dense({c, q}, {c, q}), dense({q, q}, {c, c}), {1, 3, 2, 0}, V, Vt));  // [(k0, k1) | (x0, e)]
  else
    HS_TRY(o.perm(dense({c, q}, {c, q}), dense({q, q}, {c, c}), {1, 3, 0, 2}, V, Vt));
  size_t sm = (size_t)(cx * (q * q + 2 * q)) * sizeof(double);
  constexpr size_t kMaxRow = 200 * 1024;
  const bool staged = sm <= kMaxRow;
  if (!staged) sm = (size_t)(cx * 2 * q) * sizeof(double);
  HS_CUDA(ensure_smem_attr(reinterpret_cast<const void*>(site_adjoint_kernel), (int)kMaxRow));
  for (int site = 0; site < 2; ++site) {
    const bool left = site == 0;
    const SiteLegs g = site_legs(o.cx, left);
    hs_launch(half_adjoint_kernel, grid_for(c * q * c), 256, 0, ctx->stream, drho, (const double*)half[1 - site].re,
              (const double*)half[1 - site].im, d, D, (int)c, left, dh.re, dh.im);
    HS_CUDA(cudaGetLastError());
    ZBuf din = dh;
    if (o.cx && !left) {  // back to the right chain's own bonds
      HS_TRY(o.perm(dense({c, S * S}, {c}), dense({c, S * S}, {c}), {2, 1, 0}, dh, dht));
      din = dht;
    }
    if (sb >= S) {
      HS_TRY(o.mul(c * S * S, c * q, c, din, TT, F, true));  // [(x0, S, S') | (e, k2k, k2b)]
      HS_TRY(o.perm(dense({c, S, S}, {c, D, D}), dense({S, S, D, D}, {c, c}), {1, 2, 4, 5, 0, 3}, F, Fp));
      HS_TRY(o.mul(rows, q * q, c * c, Fp, Vt, Q, true));  // [(S, S', k2k, k2b) | (k0, k1)]
    } else {  // the same with S outermost, on ranges of it
      HS_TRY(o.perm(dense({c, S, S}, {c}), dense({S, c, S}, {c}), {1, 0, 2, 3}, din, dS));
      for (long long s0 = 0; s0 < S; s0 += sb) {
        const long long b = S - s0 < sb ? S - s0 : sb;
        HS_TRY(o.mul(b * c * S, c * q, c, dS.at(s0 * c * S * c), TT, F, true));
        HS_TRY(o.perm(dense({b, c, S}, {c, D, D}), dense({b, S, D, D}, {c, c}), {0, 2, 4, 5, 1, 3}, F, Fp));
        HS_TRY(o.mul(b * S * q, q * q, c * c, Fp, Vt, Q.at(s0 * S * q * q * q), true));
      }
    }
    hs_launch(site_adjoint_kernel, (unsigned)rows, 64, sm, ctx->stream, (const double*)Q.re, (const double*)Q.im, A, d,
              D, g, staged, pk, pb);
    HS_CUDA(cudaGetLastError());
    hs_launch(site_sum_kernel, grid_for((long long)d * q * q * cx), 256, 0, ctx->stream, (const double*)pk,
              (const double*)pb, d, D, cx, g, !left, dA_out);
    HS_CUDA(cudaGetLastError());
    ctx->launches += 3;
  }
  return HS_OK;
}

}  // namespace

namespace hs {
// The open double layers of the two-site network (left site open on r, right
// site open on l) and their adjoint, for the gradient through the iterations.
cudaError_t launch_open_double_layers(const double* A, int d, int D, double* aoL, double* aoR, cudaStream_t s) {
  const long long q = (long long)D * D, nao = (long long)d * d * q * q * q * q;
  hs_launch(open_double_layer_kernel, grid_for(nao), 256, 0, s, A, d, D, true, aoL);
  hs_launch(open_double_layer_kernel, grid_for(nao), 256, 0, s, A, d, D, false, aoR);
  return cudaGetLastError();
}
cudaError_t launch_open_double_layers_vjp(const double* daoL, const double* daoR, const double* A, int d, int D,
                                          double* dA, cudaStream_t s) {
  const long long nA = (long long)d * D * D * D * D;
  hs_launch(open_double_layer_vjp_kernel, grid_for(nA), 256, 0, s, daoL, daoR, A, d, D, dA);
  return cudaGetLastError();
}
}  // namespace hs

extern "C" hs_status hs_rdm(hs_ctx ctx, const hs_env* env, const double* A, int d, int D,
                            hs_dtype dtype, hs_rdm_kind kind, const double* h, double* out,
                            double* tr_out) {
  HS_TRY(check_ctx(ctx));
  if (!env || !A || !out || d <= 0 || D != env->D) return fail(HS_ERR_INVALID_ARG, "bad arguments");
  if (dtype != HS_F64 && dtype != HS_C128) return fail(HS_ERR_DTYPE, "unknown dtype");
  if (kind != HS_RDM_TWO_SITE && kind != HS_RDM_ENV_ONE_SITE && kind != HS_RDM_ONE_SITE)
    return fail(HS_ERR_INVALID_ARG, "unknown rdm kind");
  if (kind != HS_RDM_ENV_ONE_SITE && !tr_out) return fail(HS_ERR_INVALID_ARG, "tr_out is required");
  if ((dtype == HS_C128) != (env->dtype == HS_C128)) return fail(HS_ERR_DTYPE, "A and environment disagree on dtype");
  if (kind == HS_RDM_ONE_SITE) {
    // eps first (workspace), then the contraction with A and conj(A)
    const bool cplx = dtype == HS_C128;
    const long long q = (long long)D * D, n4 = q * q * q * q;
    DBuf& eps = ctx->hb[11];
    HS_TRY(eps.ensure((size_t)n4 * (cplx ? 2 : 1) * sizeof(double)));
    HS_TRY(one_site_chain(ctx, env, d, D, eps.d()));
    hs_launch(one_site_rho_kernel, d * d, 256, 0, ctx->stream, eps.d(), A, d, D, cplx, out);
    HS_CUDA(cudaGetLastError());
    hs_launch(finish_rho1_kernel, 1, 32, 0, ctx->stream, out, d, cplx, h, tr_out);
    HS_CUDA(cudaGetLastError());
    ctx->launches += 2;
    return HS_OK;
  }
  if (kind == HS_RDM_ENV_ONE_SITE) return one_site_chain(ctx, env, d, D, out);
  HS_TRY(rdm_chain(ctx, env, A, d, D));
  return finish_rdm(ctx, env, d, D, h, out, tr_out);
}

extern "C" hs_status hs_rdm_vjp(hs_ctx ctx, const hs_env* env, const double* A, int d, int D, hs_dtype dtype,
                                const double* drho, double* dA_out) {
  HS_TRY(check_ctx(ctx));
  if (!env || !A || !drho || !dA_out || d <= 0 || D != env->D) return fail(HS_ERR_INVALID_ARG, "bad arguments");
  if (dtype != HS_F64 && dtype != HS_C128) return fail(HS_ERR_DTYPE, "unknown dtype");
  if ((dtype == HS_C128) != (env->dtype == HS_C128)) return fail(HS_ERR_DTYPE, "A and environment disagree on dtype");
  HS_TRY(rdm_chain(ctx, env, A, d, D));
  return rdm_vjp_after_chain(ctx, env, d, D, A, drho, dA_out);
}

extern "C" hs_status hs_energy_vjp(hs_ctx ctx, const hs_env* env, const double* A, int d, int D, hs_dtype dtype,
                                   const double* h, double dE, double* dA_out) {
  HS_TRY(check_ctx(ctx));
  if (!env || !A || !h || !dA_out || d <= 0 || D != env->D) return fail(HS_ERR_INVALID_ARG, "bad arguments");
  if (dtype != HS_F64 && dtype != HS_C128) return fail(HS_ERR_DTYPE, "unknown dtype");
  if ((dtype == HS_C128) != (env->dtype == HS_C128)) return fail(HS_ERR_DTYPE, "A and environment disagree on dtype");
  const bool cplx = dtype == HS_C128;
  const int n = d * d;
  // rho (scratch), its traces, the cotangent
  DBuf& w = ctx->hb[12];
  HS_TRY(w.ensure((size_t)(2 * n * n * (cplx ? 2 : 1) + 8) * sizeof(double)));
  double* rho = w.d();
  double* drho = rho + (long long)n * n * (cplx ? 2 : 1);
  double* tr = drho + (long long)n * n * (cplx ? 2 : 1);
  HS_TRY(rdm_chain(ctx, env, A, d, D));
  HS_TRY(finish_rdm(ctx, env, d, D, h, rho, tr));
  hs_launch(energy_cotangent_kernel, 1, 256, 0, ctx->stream, (const double*)tr, h, n, cplx, dE, drho);
  HS_CUDA(cudaGetLastError());
  ctx->launches += 1;
  return rdm_vjp_after_chain(ctx, env, d, D, A, drho, dA_out);
}

