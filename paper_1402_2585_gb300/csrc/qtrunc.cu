// High-mode preconditioner of the little Dirac operator (Sec. 5.2, "Truncated
// little Dirac operator as preconditioner"; Table hierarchy: order 16 on
// [0.5, 45]).
//
// Q_trunc keeps the couplings of A within one block hop (the self block and
// the eight nearest neighbours, taxicab distance <= 1; pairs l, -l together,
// so it stays Hermitian), i.e. 9 of the 81 blocks.  M = p(Q_trunc + shift)
// with p the Chebyshev-acceleration polynomial of degree order - 1 on
// [lo, hi]:  1 - x p(x) = T_order((theta - x)/delta) / T_order(theta/delta),
// theta, delta the interval's midpoint and half-width.  p is positive below
// hi, so M is Hermitian positive definite when the spectrum of Q_trunc + shift
// lies below hi; hi defaults to 1.1 times a power-iteration estimate of its
// largest eigenvalue and lo to hi / 90 (the ratio of the paper's interval).
// Evaluated by the three-term recurrence of Chebyshev acceleration:
//   y_0 = 0, s_0 = r, d_0 = r / theta, rho_0 = delta / theta;
//   y_{k+1} = y_k + d_k, s_{k+1} = s_k - Q d_k,
//   rho_{k+1} = 1 / (2 theta / delta - rho_k),
//   d_{k+1} = rho_{k+1} rho_k d_k + (2 rho_{k+1} / delta) s_{k+1},
// order - 1 products with Q_trunc.  Vectors FP32 [e][r] (e = a Nvec + j).
#include <cmath>
#include <vector>

#include "coarse.cuh"

namespace hdcg {

namespace {

unsigned nblk(size_t n) { return (unsigned)((n + 255) / 256); }

// One CTA per coarse site: the site's kept blocks are one (nq n) x n matrix
// [row = (q, k)][j], read once in 16-byte pieces (VJ 2; odd n: VJ 1, rows start
// on 8 bytes only).  Thread (ks, jp) takes VJ columns jp of the rows ks, ks + KS,
// ... for RB right-hand sides at a time; the neighbours' vectors sit in shared
// memory and the KS partial sums are added there in a fixed order.  Bound by the
// blocks' stream (L2 between the products of one polynomial, when they fit).
// One warp per site instead leaves 512 sites on 152 SMs to the latency of a serial
// loop over all rows: 16^3 x 32, Nvec 40, 4 right-hand sides, order 8 took 2451 us
// a call that way (345 us a product), 171 us this way, calls and copies included;
// the blocks (59 MB) need 9 us a product from HBM.
//
// STEP 0: y = Q x + shift x.  STEP 1, 2: the Chebyshev step on d = x fused in:
// y += d, s -= Q d, d' = c1 d + c2 s (d' to its own array: other sites still
// read d); STEP 2, the last one, also adds d' to y and leaves max(|Re y|, |Im y|)
// of each right-hand side in xm (cleared beforehand; may be null).
struct QtArgs {
  const float2* A9;
  const int* nb9;
  const float2* x;
  float2* y;
  float2* s;
  float2* dn;
  const int* skip;
  unsigned* xm;
  int nq, n, R;
  float shift, c1, c2;
};
constexpr int QT_THREADS = 288;
__host__ __device__ constexpr int qt_ks(int n, int VJ) { return QT_THREADS / ((n + VJ - 1) / VJ); }

template <int VJ, int RB, int STEP>
__global__ void __launch_bounds__(QT_THREADS) k_qtrunc_apply(const QtArgs g) {
  extern __shared__ float2 qsm[];
  if (g.skip && *g.skip) return;
  const size_t a = blockIdx.x;
  const int n = g.n, R = g.R, rows = g.nq * n;
  const int NJ = (n + VJ - 1) / VJ, KS = qt_ks(n, VJ);
  const int jp = threadIdx.x % NJ, ks = threadIdx.x / NJ;
  float2* xs = qsm;                       // [row][RB]
  float2* part = qsm + (size_t)rows * RB;   // [ks][j][RB]
  const float2* A = g.A9 + a * 9 * (size_t)n * n;
  for (int r0 = 0; r0 < R; r0 += RB) {
    const int rb = min(RB, R - r0);
    __syncthreads();
    for (int i = threadIdx.x; i < rows * RB; i += QT_THREADS) {
      const int row = i / RB, r = i % RB;
      const size_t b = (size_t)__ldg(g.nb9 + a * 9 + row / n);
      xs[i] = r < rb ? __ldg(g.x + (b * n + row % n) * R + r0 + r) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    float2 acc[VJ][RB];
#pragma unroll
    for (int v = 0; v < VJ; ++v)
#pragma unroll
      for (int r = 0; r < RB; ++r) acc[v][r] = make_float2(0.f, 0.f);
    if (ks < KS) {
      constexpr int U = 4;
      for (int row = ks; row < rows; row += U * KS) {
        float m[U][2 * VJ];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = row + u * KS;
          const bool on = k < rows;
          if constexpr (VJ == 2) {
            const float4 q = on ? __ldg(reinterpret_cast<const float4*>(A + (size_t)k * n) + jp) : make_float4(0.f, 0.f, 0.f, 0.f);
            m[u][0] = q.x; m[u][1] = q.y; m[u][2] = q.z; m[u][3] = q.w;
          } else {
            const float2 q = on ? __ldg(A + (size_t)k * n + jp) : make_float2(0.f, 0.f);
            m[u][0] = q.x; m[u][1] = q.y;
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = min(row + u * KS, rows - 1);
#pragma unroll
          for (int r = 0; r < RB; ++r) {
            const float2 x = xs[k * RB + r];
#pragma unroll
            for (int v = 0; v < VJ; ++v) {
              acc[v][r].x = fmaf(m[u][2 * v], x.x, acc[v][r].x);
              acc[v][r].y = fmaf(m[u][2 * v], x.y, acc[v][r].y);
              acc[v][r].x = fmaf(-m[u][2 * v + 1], x.y, acc[v][r].x);
              acc[v][r].y = fmaf(m[u][2 * v + 1], x.x, acc[v][r].y);
            }
          }
        }
      }
#pragma unroll
      for (int v = 0; v < VJ; ++v)
#pragma unroll
        for (int r = 0; r < RB; ++r) part[((size_t)ks * n + jp * VJ + v) * RB + r] = acc[v][r];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n * RB; i += QT_THREADS) {
      const int j = i / RB, r = i % RB;
      float2 q = make_float2(0.f, 0.f);
      for (int k = 0; k < KS; ++k) {
        const float2 p = part[(size_t)k * n * RB + i];
        q.x += p.x;
        q.y += p.y;
      }
      float mx = 0.f;
      if (r < rb) {
        const size_t o = (a * n + j) * R + r0 + r;
        const float2 d = g.x[o];
        q.x += g.shift * d.x;
        q.y += g.shift * d.y;
        if (STEP == 0) {
          g.y[o] = q;
        } else {
          float2 y = g.y[o], s = g.s[o], e;
          y.x += d.x;
          y.y += d.y;
          s.x -= q.x;
          s.y -= q.y;
          e.x = g.c1 * d.x + g.c2 * s.x;
          e.y = g.c1 * d.y + g.c2 * s.y;
          if (STEP == 2) {
            y.x += e.x;
            y.y += e.y;
            mx = fmaxf(fabsf(y.x), fabsf(y.y));
          } else {
            g.s[o] = s;
            g.dn[o] = e;
          }
          g.y[o] = y;
        }
      }
      if (STEP == 2 && g.xm && mx > 0.f) atomicMax(g.xm + r0 + r, __float_as_uint(mx));
    }
  }
}

// d = r / theta, s = r, y = 0
__global__ void k_cheb_init(const float2* __restrict__ r, float2* d, float2* s, float2* y, size_t n, float itheta,
                            const int* skip) {
  if (skip && *skip) return;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float2 v = r[t];
  d[t] = make_float2(itheta * v.x, itheta * v.y);
  s[t] = v;
  y[t] = make_float2(0.f, 0.f);
}

// y += d; with xm != null, max(|Re y|, |Im y|) of each right-hand side into xm
// (cleared beforehand): the tensor-core operand scale of y
__global__ void k_cheb_last(float2* y, const float2* __restrict__ d, size_t ne, int R, unsigned* xm, const int* skip) {
  if (skip && *skip) return;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  float m[RMAX];
#pragma unroll
  for (int q = 0; q < RMAX; ++q) m[q] = 0.f;
  if (t < ne) {
#pragma unroll
    for (int q = 0; q < RMAX; ++q)
      if (q < R) {
        const size_t o = t * R + q;
        float2 yv = y[o];
        const float2 dv = d[o];
        yv.x += dv.x;
        yv.y += dv.y;
        y[o] = yv;
        m[q] = fmaxf(fabsf(yv.x), fabsf(yv.y));
      }
  }
  if (!xm) return;
#pragma unroll
  for (int q = 0; q < RMAX; ++q) {
    if (q >= R) break;
    float u = m[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u = fmaxf(u, __shfl_xor_sync(FULL_MASK, u, o));
    if ((threadIdx.x & 31) == 0 && u > 0.f) atomicMax(xm + q, __float_as_uint(u));
  }
}

template <typename AT>
__global__ void k_qtrunc_extract(const AT* __restrict__ A, const int* __restrict__ lsel, int nq, int n, size_t Vc,
                                 float2* A9) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t per = (size_t)nq * n * n;
  if (t >= Vc * per) return;
  const size_t a = t / per;
  const int rem = (int)(t % per);
  const int q = rem / (n * n), e = rem % (n * n);
  const size_t src = ((a * 81 + lsel[q]) * n) * (size_t)n + e;
  if constexpr (sizeof(AT) == 16) {
    const double2 v = ((const double2*)A)[src];
    A9[(a * 9 + q) * (size_t)n * n + e] = make_float2((float)v.x, (float)v.y);
  } else {
    A9[(a * 9 + q) * (size_t)n * n + e] = ((const float2*)A)[src];
  }
}

__global__ void k_qtrunc_nb(const int* __restrict__ cnbr, const int* __restrict__ lsel, int nq, size_t Vc, int* nb9) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Vc * 9) return;
  const size_t a = t / 9;
  const int q = (int)(t % 9);
  nb9[t] = q < nq ? cnbr[a * 81 + lsel[q]] : 0;
}

// |v|^2 and Re<v, w> over n complex, one block (power iteration, setup only)
__global__ void k_pow_dots(const float2* __restrict__ v, const float2* __restrict__ w, size_t n, double* out) {
  double s[2] = {0.0, 0.0};
  for (size_t t = threadIdx.x; t < n; t += blockDim.x) {
    const float2 a = v[t], b = w[t];
    s[0] += (double)a.x * a.x + (double)a.y * a.y;
    s[1] += (double)a.x * b.x + (double)a.y * b.y;
  }
  block_sum<2>(s);
  if (threadIdx.x == 0) {
    out[0] = s[0];
    out[1] = s[1];
  }
}

// v = w / sqrt(nrm[0]) (nrm[0] = |w|^2)
__global__ void k_pow_norm(const float2* __restrict__ w, float2* v, size_t n, const double* nrm) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float f = (float)(1.0 / sqrt(nrm[0]));
  v[t] = make_float2(f * w[t].x, f * w[t].y);
}

}  // namespace

template <int VJ, int RB, int STEP>
static void launch_qtrunc(Ctx& c, const Coarse& A, const QtArgs& g) {
  const size_t sm = ((size_t)g.nq * g.n + (size_t)qt_ks(g.n, VJ) * g.n) * RB * sizeof(float2);
  auto fn = k_qtrunc_apply<VJ, RB, STEP>;
  if (sm > 48 * 1024)
    HDCG_CUDA(cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  fn<<<(unsigned)A.Vc, QT_THREADS, sm, c.stream>>>(g);
  HDCG_CUDA(cudaGetLastError());
  ++c.launches;
}

// Right-hand sides per pass over the blocks: 1, 4 or 8.  A second pass re-reads a
// site's blocks from L1 / L2; 16 accumulator sets would halve the resident warps.
template <int STEP>
static void dispatch_qtrunc(Ctx& c, const Coarse& A, QtArgs g) {
  const bool vec = g.n % 2 == 0;
  if (g.R == 1) vec ? launch_qtrunc<2, 1, STEP>(c, A, g) : launch_qtrunc<1, 1, STEP>(c, A, g);
  else if (g.R <= 4) vec ? launch_qtrunc<2, 4, STEP>(c, A, g) : launch_qtrunc<1, 4, STEP>(c, A, g);
  else vec ? launch_qtrunc<2, 8, STEP>(c, A, g) : launch_qtrunc<1, 8, STEP>(c, A, g);
}

static QtArgs qtrunc_args(const Coarse& A, int R, const float2* x, float2* y, double shift, const int* skip) {
  QtArgs g{};
  g.A9 = A.qt.A9.as<float2>();
  g.nb9 = A.qt.nb9.as<int>();
  g.x = x;
  g.y = y;
  g.skip = skip;
  g.nq = A.qt.nq;
  g.n = A.nvec;
  g.R = R;
  g.shift = (float)shift;
  return g;
}

void qtrunc_apply(Ctx& c, const Coarse& A, int R, const float2* x, float2* y, double shift, const int* skip) {
  dispatch_qtrunc<0>(c, A, qtrunc_args(A, R, x, y, shift, skip));
}

// y = M r for R right-hand sides (FP32 [e][r]); xm (nullable, cleared here)
// receives the per-rhs max |y| for a following tensor-core apply
void qtrunc_precondition(Ctx& c, Coarse& A, int R, const float2* r, float2* y, unsigned* xm, const int* skip) {
  QTrunc& Q = A.qt;
  const size_t ne = A.Vc * A.nvec, nc = ne * R;
  Q.work.ensure(3 * nc * sizeof(float2));
  float2* s = Q.work.as<float2>();
  float2* d[2] = {s + nc, s + 2 * nc};   // the direction and the next one
  const double theta = 0.5 * (Q.hi + Q.lo), delta = 0.5 * (Q.hi - Q.lo);
  if (xm) HDCG_CUDA(cudaMemsetAsync(xm, 0, RMAX * sizeof(unsigned), c.stream));
  k_cheb_init<<<nblk(nc), 256, 0, c.stream>>>(r, d[0], s, y, nc, (float)(1.0 / theta), skip);
  ++c.launches;
  double rho = delta / theta;
  for (int k = 0; k + 1 < Q.order; ++k) {
    const double rn = 1.0 / (2.0 * theta / delta - rho);
    QtArgs g = qtrunc_args(A, R, d[k & 1], y, Q.shift, skip);
    g.s = s;
    g.dn = d[(k & 1) ^ 1];
    g.c1 = (float)(rn * rho);
    g.c2 = (float)(2.0 * rn / delta);
    g.xm = xm;
    if (k + 2 < Q.order) dispatch_qtrunc<1>(c, A, g);
    else dispatch_qtrunc<2>(c, A, g);
    rho = rn;
  }
  if (Q.order == 1) {   // no product: y = d
    k_cheb_last<<<nblk(ne), 256, 0, c.stream>>>(y, d[0], ne, R, xm, skip);
    ++c.launches;
  }
  HDCG_CUDA(cudaGetLastError());
}

void qtrunc_setup(Ctx& c, Coarse& A, int order, double lo, double hi, double shift) {
  QTrunc& Q = A.qt;
  Q.order = 0;
  if (order <= 0) return;
  HDCG_REQUIRE(A.vec_prec() == HDCG_F32, HDCG_ERR_ARG, "the Q_trunc preconditioner needs an FP32 or FP16 operator");
  HDCG_REQUIRE(A.nvec <= 64, HDCG_ERR_ARG, "Nvec <= 64");
  // the stored offsets within one block hop
  int cd[4] = {0, 0, 0, 0};
  {
    // coarse extents from the neighbour table's reach: recover them from Vc's factorisation
    // through the subspace (the only owner of the geometry)
    const Subspace* s = c.sub;
    HDCG_REQUIRE(s, HDCG_ERR_STATE, "no subspace");
    for (int mu = 0; mu < 4; ++mu) cd[mu] = s->cdims[mu];
  }
  std::vector<int> lsel;
  for (int l = 0; l < 81; ++l) {
    int q = l, hops = 0;
    bool ok = true;
    for (int mu = 0; mu < 4; ++mu) {
      const int d = q % 3 - 1;
      q /= 3;
      hops += d != 0;
      const int L = cd[mu];
      ok = ok && (L >= 3 || (L == 2 ? d >= 0 : d == 0));
    }
    if (ok && hops <= 1) lsel.push_back(l);
  }
  Q.nq = (int)lsel.size();
  const int n = A.nvec;
  DevMem dl;
  dl.ensure(lsel.size() * sizeof(int));
  HDCG_CUDA(cudaMemcpyAsync(dl.p, lsel.data(), lsel.size() * sizeof(int), cudaMemcpyHostToDevice, c.stream));
  Q.A9.ensure(A.Vc * 9 * (size_t)n * n * sizeof(float2));
  Q.nb9.ensure(A.Vc * 9 * sizeof(int));
  const size_t tot = A.Vc * (size_t)Q.nq * n * n;
  const void* src = A.prec == HDCG_F16 ? A.Aacc.p : A.A.p;
  HDCG_REQUIRE(src, HDCG_ERR_STATE, "no FP32 copy of the FP16 little Dirac operator");
  if (A.prec == HDCG_F64)
    k_qtrunc_extract<double2><<<nblk(tot), 256, 0, c.stream>>>((const double2*)src, dl.as<int>(), Q.nq, n, A.Vc,
                                                               Q.A9.as<float2>());
  else
    k_qtrunc_extract<float2><<<nblk(tot), 256, 0, c.stream>>>((const float2*)src, dl.as<int>(), Q.nq, n, A.Vc,
                                                              Q.A9.as<float2>());
  k_qtrunc_nb<<<nblk(A.Vc * 9), 256, 0, c.stream>>>(A.cnbr.as<int>(), dl.as<int>(), Q.nq, A.Vc, Q.nb9.as<int>());
  HDCG_CUDA(cudaGetLastError());
  c.launches += 2;
  Q.shift = shift;
  if (!(hi > 0)) {
    // largest eigenvalue of Q_trunc + shift: power iteration from a Gaussian
    // vector (the coarse noise stream, seed 0x5157), Rayleigh quotient
    const size_t ne = A.Vc * n;
    DevMem v, w, dots;
    v.ensure(ne * sizeof(float2));
    w.ensure(ne * sizeof(float2));
    dots.ensure(2 * sizeof(double));
    coarse_noise(c, v.as<float2>(), ne, 0x5157ull);
    double h[2] = {1.0, 0.0};
    for (int it = 0; it < 100; ++it) {
      qtrunc_apply(c, A, 1, v.as<float2>(), w.as<float2>(), shift, nullptr);
      k_pow_dots<<<1, 1024, 0, c.stream>>>(v.as<float2>(), w.as<float2>(), ne, dots.as<double>());
      k_pow_dots<<<1, 1024, 0, c.stream>>>(w.as<float2>(), w.as<float2>(), ne, dots.as<double>() + 0);
      k_pow_norm<<<nblk(ne), 256, 0, c.stream>>>(w.as<float2>(), v.as<float2>(), ne, dots.as<double>());
      c.launches += 4;
    }
    // Rayleigh quotient of the last normalised vector
    qtrunc_apply(c, A, 1, v.as<float2>(), w.as<float2>(), shift, nullptr);
    k_pow_dots<<<1, 1024, 0, c.stream>>>(v.as<float2>(), w.as<float2>(), ne, dots.as<double>());
    c.launches += 2;
    HDCG_CUDA(cudaMemcpyAsync(h, dots.p, 2 * sizeof(double), cudaMemcpyDeviceToHost, c.stream));
    HDCG_CUDA(cudaStreamSynchronize(c.stream));
    HDCG_REQUIRE(h[0] > 0 && std::isfinite(h[1]), HDCG_ERR_NONFINITE, "Q_trunc power iteration failed");
    hi = 1.1 * h[1] / h[0];
  }
  if (!(lo > 0)) lo = hi * (lo < 0 ? -lo : 1.0 / 90.0);
  HDCG_REQUIRE(lo > 0 && hi > lo, HDCG_ERR_ARG, "the Chebyshev interval needs 0 < lo < hi");
  Q.lo = lo;
  Q.hi = hi;
  Q.order = order;
  HDCG_CUDA(cudaStreamSynchronize(c.stream));
}

// canonical [R][Vc][Nvec] complex double in and out (device): y = M x
void qtrunc_precondition_canon(Ctx& c, Coarse& A, int R, const void* x64, void* y64) {
  HDCG_REQUIRE(A.qt.order > 0, HDCG_ERR_STATE, "no coarse preconditioner");
  HDCG_REQUIRE(R >= 1 && R <= RMAX, HDCG_ERR_ARG, "1..16 right-hand sides");
  const size_t ne = A.Vc * A.nvec;
  DevMem &x = c.coarse_io[0], &y = c.coarse_io[1];
  x.ensure(ne * R * sizeof(float2));
  y.ensure(ne * R * sizeof(float2));
  coarse_canon_to_multi(c, x64, x.as<float2>(), ne, R);
  qtrunc_precondition(c, A, R, x.as<float2>(), y.as<float2>(), nullptr, nullptr);
  coarse_multi_to_canon(c, y.as<float2>(), y64, ne, R);
  HDCG_CUDA(cudaStreamSynchronize(c.stream));
}

}  // namespace hdcg
