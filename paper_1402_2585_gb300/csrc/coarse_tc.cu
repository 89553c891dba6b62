// Little Dirac operator on the tensor cores (tcgen05), for 1..16 right-hand
// sides at once:  Y_a = sum_{l in {-1,0,1}^4} A^{a,a+l} X_{a+l}  (Sec. 5.1).
//
// The complex Nvec x Nvec block A^{a,l} enters the MMA as a real matrix with
// interleaved rows m = 2j + ri (ri = 0: Re A_jk, ri = 1: Im A_jk), so
//   D[2j+0][c] = sum_k Re A_jk B[k][c],   D[2j+1][c] = sum_k Im A_jk B[k][c]
// and the complex product follows in the epilogue from the columns of B,
// which hold, per right-hand side r, the four real vectors
//   c = 4r + {0: Re X_hi, 1: Im X_hi, 2: Re X_lo, 3: Im X_lo}.
// X_hi + X_lo is the FP32 vector scaled by a power of two per right-hand side
// (largest entry in [2^13, 2^14)) and split into two FP16 parts, so the
// product carries about 22 significant bits of X, with A in FP16 and FP32
// accumulation.  Re Y = P_even - Q_odd, Im Y = Q_even + P_odd, where P = D[.,
// Re X_hi] + D[., Re X_lo] and Q = D[., Im X_hi] + D[., Im X_lo] of the two
// rows of coefficient j (adjacent TMEM lanes, exchanged by one shuffle).
//
// Every coarse site's 81 blocks carry one power-of-two scale (largest entry in
// [2^13, 2^14)), so the far couplings, many orders of magnitude below the
// diagonal block, stay in FP16's normal range; the epilogue removes it.  An FP32
// operator is split into FP16 hi + lo parts (about 22 significant bits) that
// enter as two MMAs against the same B tile; an FP16 operator is one part.
//
// With Nvec <= 32 a block has at most 64 rows, so two coarse sites share one
// M = 128 MMA (rows 0..63 site a0, 64..127 site a1) against B = [B_{a0+l} |
// B_{a1+l}]; the two off-diagonal quadrants of D are discarded.  Above 32 one
// site per MMA: its 2 Nvec rows are stored and the MMA's remaining rows are
// discarded.
// K = Nvec padded to a multiple of 16.  Both operands are pre-tiled in global
// memory in the no-swizzle K-major core-matrix layout, so every stage of the
// pipeline is filled by plain bulk copies: the A blocks of the sites (the HBM
// stream, exactly the operator's bytes) and the B tiles of their neighbours
// (L2-resident).
//
// Pipeline per CTA (persistent, up to two CTAs per SM): warp 0 issues the
// copies into a ring of stages, warp 1 issues the MMAs (one accumulator in
// tensor memory per site pair) and releases stages through tcgen05.commit,
// warps 2..5 read the accumulator (one TMEM lane quarter each), combine,
// unscale and store Y and the per-right-hand-side <X, Y>.
#include <algorithm>
#include <cstring>

#include "coarse.cuh"
#include "tc.cuh"

namespace hdcg {

namespace {

constexpr int TC_THREADS = 192;
constexpr int TC_RPMAX = RMAX;                 // right-hand sides per launch
constexpr uint32_t TC_RING_BYTES = 96 * 1024;  // two CTAs per SM
constexpr uint32_t TC_RING_BYTES_1 = 192 * 1024;  // one CTA per SM

void set_smem(const void* fn, size_t bytes) {
  HDCG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

// power-of-two scale that brings max|x| into [2^13, 2^14): exponent e, clamped
__device__ __forceinline__ int scale_exp(unsigned maxbits) {
  if (maxbits == 0) return 0;
  const int E = (int)((maxbits >> 23) & 0xffu);
  return min(126, max(-126, 140 - E));
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }

}  // namespace

TcGeom tc_geom(int nvec, int R, int parts, uint32_t ring_bytes) {
  HDCG_REQUIRE(nvec >= 1 && nvec <= 64, HDCG_ERR_ARG, "tensor-core coarse operator needs Nvec <= 64");
  HDCG_REQUIRE(R >= 1 && R <= TC_RPMAX, HDCG_ERR_ARG, "1..16 right-hand sides");
  TcGeom g;
  // two sites share an MMA for Nvec <= 32 (exactly its 128 rows at Nvec 32);
  // one site per MMA above that, with the compact layout below, which copies
  // only the operator's bytes
  g.sites = nvec <= 32 ? 2 : 1;
  g.MS = 128 / g.sites;
  g.Kp = (nvec + 15) / 16 * 16;
  const int q = g.sites == 2 ? 2 : 4;   // keeps N = sites * 4 Rp a multiple of 16
  g.Rp = (R + q - 1) / q * q;
  g.NS = 4 * g.Rp;
  g.NMMA = g.sites * g.NS;
  g.ncols = 32;
  while (g.ncols < g.NMMA) g.ncols *= 2;
  g.b_bytes = (uint32_t)g.NS * g.Kp * 2;
  g.parts = parts;
  if (g.sites == 2) {
    // two sites share the M = 128 rows: each block stored whole (MS x Kp),
    // core matrices K-adjacent 128 B apart and M-adjacent 16 Kp B apart
    g.rows = g.MS;
    g.kgs = g.Kp / 8;
    g.a_gbytes = (uint32_t)g.MS * g.Kp * 2;
    g.a_sbytes = g.a_gbytes;
    g.lbo_a = 128;
    g.sbo_a = (uint32_t)g.Kp * 16;
  } else {
    // one site: only the 2 Nvec rows (in 8-row groups) and the Nvec columns
    // (in 8-wide K groups) are stored, K group by K group (M-adjacent core
    // matrices 128 B apart, K-adjacent RG 128 B apart), so a stage copies
    // exactly the operator's bytes.  The MMA reads 16 row groups and Kp / 8
    // K groups: rows past 2 Nvec come from the next K group (finite values;
    // their output rows are discarded), and the K groups past Nvec from the
    // slot's tail, which no copy writes and which stays zero (the kernel
    // clears the ring once).
    const int RG = (2 * nvec + 7) / 8;
    g.rows = 8 * RG;
    g.kgs = (nvec + 7) / 8;
    g.a_gbytes = (uint32_t)(g.kgs * RG * 128);
    g.a_sbytes = (uint32_t)(((g.Kp / 8 - 1) * RG + 16) * 128);
    g.lbo_a = (uint32_t)RG * 128u;
    g.sbo_a = 128;
  }
  g.stage_bytes = g.sites * (parts * g.a_sbytes + g.b_bytes);
  g.copy_bytes = g.sites * (parts * g.a_gbytes + g.b_bytes);
  g.stages = (int)std::min<uint32_t>(16, ring_bytes / g.stage_bytes);
  g.stages = std::max(g.stages, 2);
  return g;
}

__device__ __forceinline__ float2 a_value(const __half2* A, size_t i) { return __half22float2(A[i]); }
__device__ __forceinline__ float2 a_value(const float2* A, size_t i) { return A[i]; }

// per coarse site: scale exponent bringing the largest |Re|, |Im| of its 81 blocks into [2^13, 2^14)
template <typename AT>
__global__ void k_site_scale(const AT* __restrict__ A, int n, int* sexp) {
  const size_t a = blockIdx.x;
  const size_t per = (size_t)81 * n * n;
  float m = 0.f;
  for (size_t i = threadIdx.x; i < per; i += blockDim.x) {
    const float2 v = a_value(A, a * per + i);
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
  __shared__ float sm[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL_MASK, m, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sm[w]);
    sexp[a] = scale_exp(__float_as_uint(fmaxf(m, sm[0])));
  }
}

// A ([a][l][k][j] complex, FP16 or FP32) -> tiled operand, one 16-byte row segment per
// thread: element (m, k) (m < rows, k < 8 kgs) of part p of block (a, l) at byte
// tc_block(a, l, p) a_gbytes + (m/8) sbo + (k/8) lbo + (m%8) 16 + (k%8) 2; part 0 = hi,
// part 1 = lo.  The sites of an MMA lie side by side, part by part, coupling by
// coupling: a stage's A is one contiguous run.
__device__ __forceinline__ size_t tc_block(size_t a, int l, int p, int sites, int parts) {
  return ((a / sites * 81 + l) * parts + p) * sites + a % sites;
}
template <typename AT>
__global__ void k_a_to_tc(const AT* __restrict__ A, uint4* __restrict__ Atc, size_t nblk, int n, int rows, int kgs,
                          uint32_t a_gbytes, uint32_t lbo, uint32_t sbo, int sites, int parts,
                          const int* __restrict__ sexp) {
  const int KG = kgs;
  const size_t per = (size_t)rows * KG;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nblk * per) return;
  const size_t blk = t / per;
  const int rem = (int)(t % per);
  const int m = rem / KG, kg = rem % KG;
  const int j = m >> 1, ri = m & 1;
  const float s = pow2f(sexp[blk / 81]);
  __align__(16) __half hi[8];
  __align__(16) __half lo[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = kg * 8 + q;
    float x = 0.f;
    if (j < n && k < n) {
      const float2 e = a_value(A, (blk * n + k) * n + j);
      x = (ri ? e.y : e.x) * s;
    }
    hi[q] = __float2half_rn(x);
    lo[q] = __float2half_rn(x - __half2float(hi[q]));
  }
  const size_t a = blk / 81;
  const int l = (int)(blk % 81);
  char* dst = reinterpret_cast<char*>(Atc) + (size_t)(m / 8) * sbo + (size_t)kg * lbo + (m % 8) * 16;
  *reinterpret_cast<uint4*>(dst + tc_block(a, l, 0, sites, parts) * a_gbytes) = *reinterpret_cast<const uint4*>(hi);
  if (parts == 2)
    *reinterpret_cast<uint4*>(dst + tc_block(a, l, 1, sites, parts) * a_gbytes) = *reinterpret_cast<const uint4*>(lo);
}

// X (FP32 complex [a][k][r]) -> tiled B operand of every coarse site: thread
// (a, kg, r) writes the four 16-byte rows c = 4r + part for k = 8 kg .. 8 kg + 7.
// Rows r >= R and k >= n are written as zeros, so the whole tile is defined.
__global__ void k_x_to_tc(const float2* __restrict__ x, uint4* __restrict__ xtc, size_t Vc, int n, int R, int Rp,
                          int Kp, const unsigned* __restrict__ xmax, const int* skip) {
  if (skip && *skip) return;
  const int KG = Kp / 8;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Vc * KG * Rp) return;
  const int r = (int)(t % Rp);
  const int kg = (int)((t / Rp) % KG);
  const size_t a = t / ((size_t)Rp * KG);
  const float s = r < R ? pow2f(scale_exp(xmax[r])) : 0.f;
  __align__(16) __half v[4][8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = kg * 8 + q;
    float2 xv = make_float2(0.f, 0.f);
    if (r < R && k < n) xv = x[(a * n + k) * R + r];
    const float re = xv.x * s, im = xv.y * s;
    const __half rh = __float2half_rn(re), ih = __float2half_rn(im);
    v[0][q] = rh;
    v[1][q] = ih;
    v[2][q] = __float2half_rn(re - __half2float(rh));
    v[3][q] = __float2half_rn(im - __half2float(ih));
  }
  const int NS = 4 * Rp;
  char* tile = reinterpret_cast<char*>(xtc) + a * (size_t)NS * Kp * 2;
#pragma unroll
  for (int part = 0; part < 4; ++part) {
    const int c = 4 * r + part;
    *reinterpret_cast<uint4*>(tile + (size_t)(c / 8) * (Kp * 16) + kg * 128 + (c % 8) * 16) =
        *reinterpret_cast<const uint4*>(v[part]);
  }
}

// The same from canonical vectors [r][a][k] (complex double): consecutive threads
// take consecutive k groups of a right-hand side, 128 contiguous bytes each.
__global__ void k_canon_to_tc(const double2* __restrict__ x, uint4* __restrict__ xtc, size_t Vc, int n, int R, int Rp,
                              int Kp, const unsigned* __restrict__ xmax) {
  const int KG = Kp / 8;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Vc * KG * Rp) return;
  const int kg = (int)(t % KG);
  const size_t a = (t / KG) % Vc;
  const int r = (int)(t / ((size_t)KG * Vc));
  const float s = r < R ? pow2f(scale_exp(xmax[r])) : 0.f;
  __align__(16) __half v[4][8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = kg * 8 + q;
    double2 xv = make_double2(0., 0.);
    if (r < R && k < n) xv = x[((size_t)r * Vc + a) * n + k];
    const float re = (float)xv.x * s, im = (float)xv.y * s;
    const __half rh = __float2half_rn(re), ih = __float2half_rn(im);
    v[0][q] = rh;
    v[1][q] = ih;
    v[2][q] = __float2half_rn(re - __half2float(rh));
    v[3][q] = __float2half_rn(im - __half2float(ih));
  }
  char* tile = reinterpret_cast<char*>(xtc) + a * (size_t)(4 * Rp) * Kp * 2;
#pragma unroll
  for (int part = 0; part < 4; ++part) {
    const int c = 4 * r + part;
    *reinterpret_cast<uint4*>(tile + (size_t)(c / 8) * (Kp * 16) + kg * 128 + (c % 8) * 16) =
        *reinterpret_cast<const uint4*>(v[part]);
  }
}

// xmax[r] of canonical vectors (grid y: right-hand side)
__global__ void k_canon_max(const double2* __restrict__ x, size_t ne, unsigned* xmax) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  float m = 0.f;
  if (t < ne) {
    const double2 v = x[blockIdx.y * ne + t];
    m = fmaxf(fabsf((float)v.x), fabsf((float)v.y));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL_MASK, m, o));
  if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(xmax + blockIdx.y, __float_as_uint(m));
}

// per-right-hand-side max(|Re x|, |Im x|) as float bits (atomicMax on non-negative floats)
__global__ void k_cmax(const float2* __restrict__ x, size_t ne, int R, unsigned* xmax) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  float m[RMAX];
#pragma unroll
  for (int r = 0; r < RMAX; ++r) m[r] = 0.f;
  if (t < ne)
#pragma unroll
    for (int r = 0; r < RMAX; ++r)
      if (r < R) {
        const float2 v = x[t * R + r];
        m[r] = fmaxf(fabsf(v.x), fabsf(v.y));
      }
#pragma unroll
  for (int r = 0; r < RMAX; ++r) {
    if (r >= R) break;
    float v = m[r];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL_MASK, v, o));
    if ((threadIdx.x & 31) == 0 && v > 0.f) atomicMax(xmax + r, __float_as_uint(v));
  }
}

struct TcArgs {
  const uint4* Atc;
  const int* cnbr;
  const uint4* xtc;
  const unsigned* xmax;
  const float2* x;     // FP32 X for <X, Y> (nullable)
  float2* y;
  double2* y64;        // not null: Y canonical, [r][site][j] complex double, instead of y
  const int* skip;     // nonzero: the launch has nothing to do (nullable)
  unsigned* err;       // bit flags of expired waits
  int Vc, n, R, sites, MS, Kp, NS, stages, ncols;
  uint32_t a_gbytes, a_sbytes, lbo_a, sbo_a, b_bytes, copy_bytes, idesc;
  float shift;         // Y = (A + shift) X (needs x)
  int parts;           // 1: FP16 operator, 2: FP32 operator as FP16 hi + lo
  const int* sexp;     // per-site scale exponents of the tiled operator
  // The 81 couplings of a pair split over nsplit work items (items of one pair add
  // up: part s goes to y + s part; the shift joins part 0).  1 for operators with
  // enough pairs to fill the chip.
  int nsplit;
  size_t part;
  uint64_t wait_ns;    // limit of a wait for another role; waits for what was issued have WAIT_LIMIT_NS
};
__device__ __forceinline__ int split_begin(int s, int nsplit) { return s * 81 / nsplit; }

__global__ void __launch_bounds__(TC_THREADS, 2) k_capply_tc(TcArgs g, Reduction red) {
  extern __shared__ __align__(128) unsigned char smem[];
  if (g.skip && *g.skip) return;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t stage_bytes = g.sites * (g.parts * g.a_sbytes + g.b_bytes);
  const uint32_t ring = tc::smem_u32(smem);
  // clear the ring once: the tails of the A slots that no copy writes are read
  // by the MMAs as K padding and must be zero
  for (uint32_t i = threadIdx.x; i < (uint32_t)g.stages * stage_bytes / 16u; i += blockDim.x)
    reinterpret_cast<uint4*>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
  tc::fence_proxy_async_smem();
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)g.stages * stage_bytes);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2 * g.stages + 3);
  const uint32_t bar0 = tc::smem_u32(bars);
  const uint32_t ACC_FULL = bar0 + 8u * (2 * g.stages), ACC_EMPTY = ACC_FULL + 8u, DRAIN = ACC_FULL + 16u;
#define TC_FULL(s) (bar0 + 8u * (uint32_t)(s))
#define TC_EMPTY(s) (bar0 + 8u * (uint32_t)(g.stages + (s)))
  if (threadIdx.x == 0) {
    for (int s = 0; s < g.stages; ++s) {
      tc::mbar_init(TC_FULL(s), 1);
      tc::mbar_init(TC_EMPTY(s), 1);
    }
    tc::mbar_init(ACC_FULL, 1);
    tc::mbar_init(ACC_EMPTY, 4);
    tc::mbar_init(DRAIN, 1);
    tc::fence_mbar_init();
  }
  if (w == 1) {
    tc::tmem_alloc(tc::smem_u32(tslot), (uint32_t)g.ncols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tslot;
  const int items = (g.Vc + g.sites - 1) / g.sites * g.nsplit;   // (pair, part), part fastest
  double dot[RMAX];
#pragma unroll
  for (int r = 0; r < RMAX; ++r) dot[r] = 0.0;

  if (w == 0) {
    // ---- producer: bulk copies of A blocks and neighbour B tiles --------------------
    // The whole warp first fetches the pair's 81 (or 162) neighbour indices into
    // shared memory in one round trip.  Then every lane of the first few issues one
    // copy of a stage, its source advancing by itself: lane 0 the A run of both sites
    // (one site with K padding: one lane per part), the next lanes the B tiles.  With
    // one lane issuing all four to six copies and dividing for its ring position, a
    // stage took 0.65 to 0.82 us whatever its size (24^3 x 48, FP16: 244 us an apply).
    __shared__ int snb[2 * 81];
    const int nA = g.sites == 2 ? 1 : g.parts, ncopy = nA + g.sites;
    const uint32_t abytes = g.sites == 2 ? 2u * g.parts * g.a_gbytes : g.a_gbytes;
    const size_t astep = (size_t)g.sites * g.parts * g.a_gbytes;     // one coupling of a pair
    const uint32_t doff = lane < nA ? (uint32_t)lane * g.a_sbytes
                                    : (uint32_t)(g.sites * g.parts) * g.a_sbytes + (uint32_t)(lane - nA) * g.b_bytes;
    const uint32_t bytes = lane < nA ? abytes : g.b_bytes;
    uint32_t it = 0, s = 0, ph = 0;
    bool ok = true;
    for (int p = blockIdx.x; ok && p < items; p += gridDim.x) {
      const int pair = p / g.nsplit, s0 = pair * g.sites;
      const int l0 = split_begin(p % g.nsplit, g.nsplit), l1 = split_begin(p % g.nsplit + 1, g.nsplit);
      const int s1 = min(s0 + 1, g.Vc - 1);
      for (int q = lane; q < g.sites * 81; q += 32)
        snb[q] = __ldg(g.cnbr + (size_t)(q < 81 ? s0 : s1) * 81 + q % 81);
      __syncwarp();
      const char* src = reinterpret_cast<const char*>(g.Atc) + ((size_t)pair * 81 + l0) * astep + (size_t)lane * g.a_gbytes;
      const int* nb = snb + (lane >= nA && lane < ncopy ? (lane - nA) * 81 : 0);
      for (int l = l0; l < l1; ++l, ++it) {
        // All lanes issue or none: a stage that only some of them saw empty in time would
        // get a part of its copies, which FULL and the wait before the exit do not cover.
        const bool empty = lane >= ncopy || tc::mbar_wait(TC_EMPTY(s), ph ^ 1u, g.wait_ns);
        ok = __all_sync(FULL_MASK, empty);
        if (!ok) {
          if (lane == 0) atomicOr(g.err, 1u);
          break;
        }
        if (lane == 0) tc::mbar_arrive_expect_tx(TC_FULL(s), g.copy_bytes);
        // stage: [part 0: site 0, site 1][part 1: site 0, site 1][B site 0][B site 1]
        if (lane < ncopy)
          tc::bulk_g2s(ring + s * stage_bytes + doff,
                       lane < nA ? src : reinterpret_cast<const char*>(g.xtc) + (size_t)nb[l] * g.b_bytes, bytes,
                       TC_FULL(s));
        src += astep;
        if (++s == (uint32_t)g.stages) {
          s = 0;
          ph ^= 1u;
        }
      }
      __syncwarp();   // every lane is done with snb before the next pair overwrites it
    }
    if (lane == 0) {
      // every copy issued has to land before the CTA exits
      const uint32_t first = it > (uint32_t)g.stages ? it - (uint32_t)g.stages : 0u;
      for (uint32_t j = first; j < it; ++j)
        if (!tc::mbar_wait(TC_FULL(j % (uint32_t)g.stages), (j / (uint32_t)g.stages) & 1u)) atomicOr(g.err, 2u);
    }
  } else if (w == 1) {
    // ---- MMA issuer ------------------------------------------------------------------
    if (lane == 0) {
      uint32_t s = 0, ph = 0;
      int np = 0;
      bool ok = true;
      const uint64_t bdesc = tc::smem_desc(0, 128u, (uint32_t)g.Kp * 16u), adesc = tc::smem_desc(0, g.lbo_a, g.sbo_a);
      const int ksteps = g.Kp / 16;
      const uint32_t pstep = g.sites * g.a_sbytes;
      for (int p = blockIdx.x; ok && p < items; p += gridDim.x, ++np) {
        const int l0 = split_begin(p % g.nsplit, g.nsplit), l1 = split_begin(p % g.nsplit + 1, g.nsplit);
        if (np > 0 && !tc::mbar_wait(ACC_EMPTY, (uint32_t)(np - 1) & 1u, g.wait_ns)) {
          ok = false;
          atomicOr(g.err, 4u);
          break;
        }
        tc::fence_after_sync();
        for (int l = l0; l < l1; ++l) {
          if (!tc::mbar_wait(TC_FULL(s), ph, g.wait_ns)) {
            ok = false;
            atomicOr(g.err, 8u);
            break;
          }
          tc::fence_after_sync();
          const uint32_t abase = ring + s * stage_bytes;
          const uint32_t bbase = abase + g.sites * g.parts * g.a_sbytes;
          // addresses below 256 KB: a step is an addition to the descriptor's low word
          const uint64_t bd0 = bdesc | (bbase >> 4), ad0 = adesc | (abase >> 4);
          for (int ks = 0; ks < ksteps; ++ks) {
            const uint64_t bd = bd0 + 16u * ks;
            for (int p = 0; p < g.parts; ++p) {
              const uint64_t ad = ad0 + ((p * pstep + 2u * g.lbo_a * ks) >> 4);
              tc::mma_f16(tmem, ad, bd, g.idesc, (l != l0 || (ks | p) != 0) ? 1u : 0u);
            }
          }
          tc::mma_commit(TC_EMPTY(s));
          if (++s == (uint32_t)g.stages) {
            s = 0;
            ph ^= 1u;
          }
        }
        if (ok) tc::mma_commit(ACC_FULL);
      }
      // all MMAs issued by this thread complete before the accumulator is freed
      tc::mma_commit(DRAIN);
      if (!tc::mbar_wait(DRAIN, 0u)) atomicOr(g.err, 16u);
    }
  } else {
    // ---- epilogue: TMEM lane quarter (w % 4) --------------------------------------------
    const int q = w & 3;
    const int row = 32 * q + lane;
    const int si = row / g.MS, mrow = row % g.MS;
    const int j = mrow >> 1, ri = mrow & 1;
    const uint32_t taddr = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(si * g.NS);
    float inv[RMAX];
#pragma unroll
    for (int r = 0; r < RMAX; ++r) inv[r] = r < g.R ? pow2f(-scale_exp(g.xmax[r])) : 0.f;
    int np = 0;
    for (int p = blockIdx.x; p < items; p += gridDim.x, ++np) {
      const bool ok = tc::mbar_wait(ACC_FULL, (uint32_t)np & 1u, g.wait_ns);
      if (!__all_sync(FULL_MASK, ok)) {
        if (lane == 0) atomicOr(g.err, 32u);
        break;
      }
      tc::fence_after_sync();
      float d[4 * TC_RPMAX];
#pragma unroll
      for (int c8 = 0; c8 < TC_RPMAX / 2; ++c8)
        if (8 * c8 < g.NS) tc::tmem_ld8(taddr + 8u * c8, d + 8 * c8);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(ACC_EMPTY);
      const int part = p % g.nsplit, site = p / g.nsplit * g.sites + si;
      const bool valid = site < g.Vc && j < g.n;
      const float sinv = valid ? pow2f(-__ldg(g.sexp + site)) : 0.f;
#pragma unroll
      for (int r = 0; r < TC_RPMAX; ++r) {
        if (r < g.R) {
          const float P = d[4 * r] + d[4 * r + 2];
          const float Q = d[4 * r + 1] + d[4 * r + 3];
          const float t = __shfl_xor_sync(FULL_MASK, Q, 1);
          float v = (ri ? t + P : P - t) * (inv[r] * sinv);
          if (valid) {
            if (g.y64) {   // lanes run over (j, ri): 256 contiguous bytes per right-hand side
              reinterpret_cast<double*>(g.y64)[2 * (((size_t)r * g.Vc + site) * g.n + j) + ri] = (double)v;
              continue;
            }
            const size_t e = ((size_t)site * g.n + j) * g.R + r;
            if (g.x) {
              const float xv = reinterpret_cast<const float*>(g.x)[2 * e + ri];
              if (part == 0) v += g.shift * xv;
              dot[r] += (double)xv * (double)v;
            }
            reinterpret_cast<float*>(g.y + part * g.part)[2 * e + ri] = v;
          }
        }
      }
    }
  }
#undef TC_FULL
#undef TC_EMPTY
  __syncthreads();
  if (w == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, (uint32_t)g.ncols);
  }
  if (red.result) grid_reduce<RMAX>(dot, red, g.R);
}

// ---------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------

bool coarse_tc_supported(const Coarse& A) {
  return (A.prec == HDCG_F16 || A.prec == HDCG_F32) && A.nvec >= 1 && A.nvec <= 64;
}
static int tc_parts(const Coarse& A) { return A.prec == HDCG_F32 ? 2 : 1; }

void coarse_tc_prepare(Ctx& c, Coarse& A) {
  HDCG_REQUIRE(coarse_tc_supported(A), HDCG_ERR_ARG,
               "tensor-core coarse operator needs an FP16 or FP32 A and Nvec <= 64");
  if (A.tc_ready) return;
  const int parts = tc_parts(A);
  const TcGeom g = tc_geom(A.nvec, 1, parts);
  const size_t nblk = A.Vc * 81;
  const size_t abytes = (A.Vc + g.sites - 1) / g.sites * g.sites * 81 * parts * (size_t)g.a_gbytes;
  A.Atc.ensure(abytes);
  if (A.Vc % g.sites) HDCG_CUDA(cudaMemsetAsync(A.Atc.p, 0, abytes, c.stream));   // the last pair's missing site
  A.sexp.ensure(A.Vc * sizeof(int));
  A.tcs.ensure(sizeof(TcState));
  HDCG_CUDA(cudaMemsetAsync(A.tcs.p, 0, sizeof(TcState), c.stream));
  const size_t nt = nblk * g.rows * g.kgs;
  if (A.prec == HDCG_F32) {
    k_site_scale<float2><<<(unsigned)A.Vc, 256, 0, c.stream>>>(A.A.as<float2>(), A.nvec, A.sexp.as<int>());
    k_a_to_tc<float2><<<(unsigned)((nt + 255) / 256), 256, 0, c.stream>>>(
        A.A.as<float2>(), A.Atc.as<uint4>(), nblk, A.nvec, g.rows, g.kgs, g.a_gbytes, g.lbo_a, g.sbo_a, g.sites, parts,
        A.sexp.as<int>());
  } else {
    k_site_scale<__half2><<<(unsigned)A.Vc, 256, 0, c.stream>>>(A.A.as<__half2>(), A.nvec, A.sexp.as<int>());
    k_a_to_tc<__half2><<<(unsigned)((nt + 255) / 256), 256, 0, c.stream>>>(
        A.A.as<__half2>(), A.Atc.as<uint4>(), nblk, A.nvec, g.rows, g.kgs, g.a_gbytes, g.lbo_a, g.sbo_a, g.sites, parts,
        A.sexp.as<int>());
  }
  HDCG_CUDA(cudaGetLastError());
  c.launches += 2;
  A.tc_ready = true;
}

void coarse_tc_check(Ctx& c, Coarse& A) {
  unsigned* flags = c.pinned.at<unsigned>(8064);
  HDCG_CUDA(cudaMemcpyAsync(flags, &A.tcs.as<TcState>()->err, sizeof(unsigned), cudaMemcpyDeviceToHost, c.stream));
  HDCG_CUDA(cudaStreamSynchronize(c.stream));
  const unsigned err = *flags;
  if (err) {
    HDCG_CUDA(cudaMemsetAsync(A.tcs.p, 0, sizeof(unsigned), c.stream));
    throw Error{HDCG_ERR_TIMEOUT, "tensor-core coarse apply: a pipeline wait expired (flags " +
                                      std::to_string(err) + ")"};
  }
}

void coarse_tc_max(Ctx& c, const float2* x, size_t ne, int R, unsigned* xmax) {
  HDCG_CUDA(cudaMemsetAsync(xmax, 0, RMAX * sizeof(unsigned), c.stream));
  k_cmax<<<(unsigned)((ne + 255) / 256), 256, 0, c.stream>>>(x, ne, R, xmax);
  HDCG_CUDA(cudaGetLastError());
  c.launches += 1;
}

void coarse_tc_to_b(Ctx& c, Coarse& A, int R, const float2* x, const unsigned* xmax, const int* skip) {
  const TcGeom g = tc_geom(A.nvec, R, tc_parts(A));
  A.xtc.ensure(A.Vc * (size_t)g.b_bytes);
  const size_t nt = A.Vc * (size_t)(g.Kp / 8) * g.Rp;
  k_x_to_tc<<<(unsigned)((nt + 255) / 256), 256, 0, c.stream>>>(x, A.xtc.as<uint4>(), A.Vc, A.nvec, R, g.Rp, g.Kp,
                                                                 xmax, skip);
  HDCG_CUDA(cudaGetLastError());
  ++c.launches;
}

// one launch with cpsm (1 or 2) persistent CTAs per SM and the matching ring
static void launch_tc(Ctx& c, Coarse& A, int R, const float2* x, float2* y, const unsigned* xmax, const int* skip,
                      double* dot_result, double shift, int cpsm, double2* y64, int nsplit = 1) {
  const TcGeom g = tc_geom(A.nvec, R, tc_parts(A), cpsm == 1 ? TC_RING_BYTES_1 : TC_RING_BYTES);
  TcArgs a;
  a.Atc = A.Atc.as<uint4>();
  a.cnbr = A.cnbr.as<int>();
  a.xtc = A.xtc.as<uint4>();
  a.xmax = xmax;
  a.x = x;
  a.y = y;
  a.y64 = y64;
  a.skip = skip;
  a.err = &A.tcs.as<TcState>()->err;
  a.Vc = (int)A.Vc;
  a.n = A.nvec;
  a.R = R;
  a.sites = g.sites;
  a.MS = g.MS;
  a.Kp = g.Kp;
  a.NS = g.NS;
  a.stages = g.stages;
  a.ncols = g.ncols;
  a.a_gbytes = g.a_gbytes;
  a.a_sbytes = g.a_sbytes;
  a.lbo_a = g.lbo_a;
  a.sbo_a = g.sbo_a;
  a.copy_bytes = g.copy_bytes;
  a.b_bytes = g.b_bytes;
  a.idesc = tc::idesc_f16_f32(128, g.NMMA);
  a.shift = (float)shift;
  a.parts = g.parts;
  a.nsplit = nsplit;
  a.part = A.Vc * A.nvec * (size_t)R;
  a.wait_ns = c.tc_wait_ns;
  a.sexp = A.sexp.as<int>();
  const size_t smem = (size_t)g.stages * g.stage_bytes + (2 * g.stages + 3) * 8 + 16;
  static size_t smem_set = 0;
  if (smem > smem_set) {
    set_smem((const void*)k_capply_tc, std::max<size_t>(smem, 100 * 1024));
    smem_set = std::max<size_t>(smem, 100 * 1024);
  }
  const int npairs = (int)((A.Vc + g.sites - 1) / g.sites);
  const unsigned grid = (unsigned)std::min(npairs * nsplit, cpsm * device_sms());
  const Reduction red = dot_result ? make_reduction(c, grid, RMAX, dot_result, 0) : Reduction{};
  k_capply_tc<<<grid, TC_THREADS, smem, c.stream>>>(a, red);
  HDCG_CUDA(cudaGetLastError());
  ++c.launches;
}

// The first apply to R vectors of an operator times two persistent shapes, two
// CTAs per SM with a 96 KB ring and one CTA per SM with a 192 KB ring (twice
// the stages in flight), and keeps the faster.  Both run the same MMAs in the
// same order, so the choice never changes a result.  Inside a stream capture
// the two-CTA shape runs untimed.
static void tc_apply(Ctx& c, Coarse& A, int R, const float2* x, float2* y, const unsigned* xmax, const int* skip,
                     double* dot_result, double shift, double2* y64) {
  int cfg = c.tc_force ? c.tc_force : A.tc_cfg[R];
  if (cfg == 0) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    HDCG_CUDA(cudaStreamIsCapturing(c.stream, &cs));
    if (cs != cudaStreamCaptureStatusNone) {
      cfg = 2;
    } else {
      cudaEvent_t e0, e1;
      HDCG_CUDA(cudaEventCreate(&e0));
      HDCG_CUDA(cudaEventCreate(&e1));
      float best = 1e30f;
      for (int cand : {2, 1}) {
        launch_tc(c, A, R, x, y, xmax, skip, dot_result, shift, cand, y64);
        HDCG_CUDA(cudaEventRecord(e0, c.stream));
        for (int i = 0; i < 3; ++i) launch_tc(c, A, R, x, y, xmax, skip, dot_result, shift, cand, y64);
        HDCG_CUDA(cudaEventRecord(e1, c.stream));
        HDCG_CUDA(cudaEventSynchronize(e1));
        float ms = 0.f;
        HDCG_CUDA(cudaEventElapsedTime(&ms, e0, e1));
        if (ms < best) {
          best = ms;
          cfg = cand;
        }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      A.tc_cfg[R] = cfg;
    }
  }
  launch_tc(c, A, R, x, y, xmax, skip, dot_result, shift, cfg, y64);
}
void coarse_tc_apply(Ctx& c, Coarse& A, int R, const float2* x, float2* y, const unsigned* xmax, const int* skip,
                     double* dot_result, double shift) {
  tc_apply(c, A, R, x, y, xmax, skip, dot_result, shift, nullptr);
}

// ---------------------------------------------------------------------------------
// coarse CG for R right-hand sides on the tensor-core operator (vectors FP32 [a][k][r])
// ---------------------------------------------------------------------------------

struct CCtlT {
  double rr[2][RMAX];
  double pAp[RMAX];
  double stop[RMAX];
  int done[RMAX];
  int iter;
  int all_done;
};

__global__ void k_cgt_init(const float2* __restrict__ rhs, float2* x, float2* r, float2* p, size_t ne, int R,
                           unsigned* xmax, Reduction red) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  double v[RMAX];
  float m[RMAX];
#pragma unroll
  for (int q = 0; q < RMAX; ++q) {
    v[q] = 0.0;
    m[q] = 0.f;
  }
  if (t < ne) {
#pragma unroll
    for (int q = 0; q < RMAX; ++q)
      if (q < R) {
        const float2 b = rhs[t * R + q];
        x[t * R + q] = make_float2(0.f, 0.f);
        r[t * R + q] = b;
        p[t * R + q] = b;
        v[q] = (double)b.x * b.x + (double)b.y * b.y;
        m[q] = fmaxf(fabsf(b.x), fabsf(b.y));
      }
  }
#pragma unroll
  for (int q = 0; q < RMAX; ++q) {
    if (q >= R) break;
    float u = m[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u = fmaxf(u, __shfl_xor_sync(FULL_MASK, u, o));
    if ((threadIdx.x & 31) == 0 && u > 0.f) atomicMax(xmax + q, __float_as_uint(u));
  }
  grid_reduce<RMAX>(v, red, R);
}

__global__ void k_cgt_start(CCtlT* ctl, int R, double tol, int maxiter) {
  int all = 1;
  for (int q = 0; q < R; ++q) {
    ctl->stop[q] = tol * tol * ctl->rr[0][q];
    ctl->done[q] = (ctl->rr[0][q] == 0.0 || maxiter <= 0) ? 1 : 0;
    all &= ctl->done[q];
  }
  ctl->iter = 0;
  ctl->all_done = all;
}

// x += alpha p, r -= alpha w for the right-hand sides still running; |r|^2; clears xmax
__global__ void k_cgt_update(float2* x, float2* r, const float2* __restrict__ p, const float2* __restrict__ w,
                             size_t ne, int R, const CCtlT* ctl, int par, unsigned* xmax, Reduction red) {
  if (ctl->all_done) return;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t == 0)
    for (int q = 0; q < RMAX; ++q) xmax[q] = 0u;
  __shared__ float s_al[RMAX];   // one FP64 division per right-hand side and CTA
  if (threadIdx.x < R) {
    const double pap = ctl->pAp[threadIdx.x];
    s_al[threadIdx.x] = (float)(pap > 0 ? ctl->rr[par][threadIdx.x] / pap : 0.0);
  }
  __syncthreads();
  double v[RMAX];
#pragma unroll
  for (int q = 0; q < RMAX; ++q) v[q] = 0.0;
  if (t < ne) {
#pragma unroll
    for (int q = 0; q < RMAX; ++q) {
      if (q < R) {
        const size_t e = t * R + q;
        float2 rv = r[e];
        if (!ctl->done[q]) {
          const float al = s_al[q];
          const float2 pv = p[e], wv = w[e];
          float2 xv = x[e];
          xv.x += al * pv.x;
          xv.y += al * pv.y;
          rv.x -= al * wv.x;
          rv.y -= al * wv.y;
          x[e] = xv;
          r[e] = rv;
        }
        const double re = widen(rv.x), im = widen(rv.y);
        v[q] = fma(re, re, im * im);
      }
    }
  }
  grid_reduce_shared<RMAX>(v, red, R);
}

// p = r + beta p for the right-hand sides still running; max|p| of every right-hand side
__global__ void k_cgt_p(float2* p, const float2* __restrict__ r, size_t ne, int R, const CCtlT* ctl, int par,
                        unsigned* xmax) {
  if (ctl->all_done) return;
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  __shared__ float s_be[RMAX];
  if (threadIdx.x < R) {
    const double ro = ctl->rr[par][threadIdx.x], rn = ctl->rr[par ^ 1][threadIdx.x];
    s_be[threadIdx.x] = (float)(ro > 0 ? rn / ro : 0.0);
  }
  __syncthreads();
  float m[RMAX];
#pragma unroll
  for (int q = 0; q < RMAX; ++q) m[q] = 0.f;
  if (t < ne) {
#pragma unroll
    for (int q = 0; q < RMAX; ++q) {
      if (q < R) {
        const size_t e = t * R + q;
        float2 pv = p[e];
        if (!ctl->done[q]) {
          const float beta = s_be[q];
          const float2 rv = r[e];
          pv.x = rv.x + beta * pv.x;
          pv.y = rv.y + beta * pv.y;
          p[e] = pv;
        }
        m[q] = fmaxf(fabsf(pv.x), fabsf(pv.y));
      }
    }
  }
#pragma unroll
  for (int q = 0; q < RMAX; ++q) {
    if (q >= R) break;
    float u = m[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) u = fmaxf(u, __shfl_xor_sync(FULL_MASK, u, o));
    if ((threadIdx.x & 31) == 0 && u > 0.f) atomicMax(xmax + q, __float_as_uint(u));
  }
}

__global__ void k_cgt_check(CCtlT* ctl, int R, int par, int maxiter) {
  if (ctl->all_done) return;
  const int it = ctl->iter + 1;
  ctl->iter = it;
  int all = 1;
  for (int q = 0; q < R; ++q) {
    const double rn = ctl->rr[par ^ 1][q];
    if (!ctl->done[q] && (rn <= ctl->stop[q] || it >= maxiter || !(rn == rn))) ctl->done[q] = 1;
    all &= ctl->done[q];
  }
  ctl->all_done = all;
}

// ---------------------------------------------------------------------------------
// Small coarse grids: everything of a CG iteration but the stencil in one launch.
// The vectors of a 4^4 coarse grid (24 vectors, 4 right-hand sides: 196 KB) are a
// few microseconds of work, but the update, the new direction, its largest entry,
// the operand and the bookkeeping need each other's results over the whole grid:
// as four launches of 16 to 24 CTAs they took 33 us of an iteration, k_cgt_update
// 18 of them.  One cluster of eight CTAs meets at two cluster barriers instead:
// 14.8 us, with the scalars computed by one thread of a CTA; 18 with |r|^2 in FP64
// (an iteration 62.5 -> 66 us for 4 right-hand sides, 93 -> 105 for 16).
// With the split couplings (78 us a product on 128 of 152 SMs before, for 170 MB:
// the 95 MB of the operator, its 48 x 24 blocks padded to 64 x 32)
// the batched solve of four sources on 16^4 x 16 went from 217 to 202 ms.
// A thread owns the same (site, eight coefficients, right-hand side) items in every
// phase.  |r|^2 in FP64, squares and sums: entries of FP32's whole range.
// ---------------------------------------------------------------------------------
constexpr int CS_CTAS = 8, CS_THREADS = 512, CS_ITEMS = 4;   // at most CS_ITEMS items a thread
struct CgStepScratch {
  double rr[CS_CTAS][RMAX];
  unsigned xm[CS_CTAS][RMAX];
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __cluster_dims__(CS_CTAS, 1, 1) __launch_bounds__(CS_THREADS)
    k_cgt_step(float2* x, float2* r, float2* p, const float2* w, int nsplit, size_t part, int Vc, int n, int R, int Rp,
               int Kp, char* xtc, CCtlT* ctl, CgStepScratch* sc, int par, int maxiter, unsigned* xmax) {
  if (ctl->all_done) return;   // written by CTA 0 behind the last barrier only
  __shared__ double srr[CS_THREADS];
  __shared__ unsigned sxm[RMAX];
  __shared__ double s_rn[RMAX];
  __shared__ float s_al[RMAX], s_be[RMAX];
  const int cta = blockIdx.x, tid = threadIdx.x, gid = cta * CS_THREADS + tid;
  const int stride = CS_CTAS * CS_THREADS / Rp * Rp;    // whole groups of Rp: a thread keeps its right-hand side
  const int q = gid % Rp, KG = Kp / 8, N = Vc * KG * Rp;
  const bool live = gid < stride && q < R;
  const bool run = live && !ctl->done[q];
  if (tid < RMAX) sxm[tid] = 0u;
  // FP64 divisions and sums once per right-hand side and CTA: by every thread they
  // were most of the kernel (FP64 does two lanes per clock and SM)
  if (tid < R) {
    const double pap = ctl->pAp[tid];
    s_al[tid] = (float)(pap > 0 ? ctl->rr[par][tid] / pap : 0.0);
  }
  __syncthreads();
  // x += alpha p, r -= alpha w, |r|^2
  double s = 0.0;
  if (live) {
    const float al = s_al[q];
    for (int j = gid; j < N; j += stride) {
      const int it = j / Rp, a = it / KG, k0 = 8 * (it % KG), kc = min(8, n - k0);
      const size_t o0 = ((size_t)a * n + k0) * R + q;
      // every load of the item in flight before the first use
      float2 rv[8], pv[8], wv[8], xv[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const size_t o = o0 + (size_t)min(k, kc - 1) * R;
        rv[k] = r[o];
        pv[k] = p[o];
        wv[k] = w[o];
        xv[k] = x[o];
      }
      for (int t = 1; t < nsplit; ++t)
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float2 u = w[t * part + o0 + (size_t)min(k, kc - 1) * R];
          wv[k].x += u.x;
          wv[k].y += u.y;
        }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (k < kc) {
          if (run) {
            const size_t o = o0 + (size_t)k * R;
            xv[k].x += al * pv[k].x;
            xv[k].y += al * pv[k].y;
            rv[k].x -= al * wv[k].x;
            rv[k].y -= al * wv[k].y;
            x[o] = xv[k];
            r[o] = rv[k];
          }
          const double re = widen(rv[k].x), im = widen(rv[k].y);
          s = fma(re, re, s);
          s = fma(im, im, s);
        }
      }
    }
  }
  srr[tid] = s;
  __syncthreads();
  {
    // warp w sums right-hand side w over the CTA's threads
    const int wq = tid >> 5;
    if (wq < R) {
      double v = 0.0;
      int i = (wq - cta * CS_THREADS % Rp + Rp) % Rp;      // the CTA's first thread of this right-hand side
      for (i += (tid & 31) * Rp; i < CS_THREADS; i += 32 * Rp) v += srr[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
      if ((tid & 31) == 0) sc->rr[cta][wq] = v;
    }
  }
  cluster_sync();
  // p = r + beta p, max |p|
  if (tid < R) {
    double rn = 0.0;
    for (int c = 0; c < CS_CTAS; ++c) rn += __ldcg(&sc->rr[c][tid]);
    const double ro = ctl->rr[par][tid];
    s_rn[tid] = rn;
    s_be[tid] = (float)(ro > 0 ? rn / ro : 0.0);
  }
  __syncthreads();
  if (live) {
    const float be = s_be[q];
    float m = 0.f;
    for (int j = gid; j < N; j += stride) {
      const int it = j / Rp, a = it / KG, k0 = 8 * (it % KG), kc = min(8, n - k0);
      const size_t o0 = ((size_t)a * n + k0) * R + q;
      float2 rv[8], pv[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const size_t o = o0 + (size_t)min(k, kc - 1) * R;
        rv[k] = r[o];
        pv[k] = p[o];
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (k < kc) {
          if (run) {
            pv[k].x = rv[k].x + be * pv[k].x;
            pv[k].y = rv[k].y + be * pv[k].y;
            p[o0 + (size_t)k * R] = pv[k];
          }
          m = fmaxf(m, fmaxf(fabsf(pv[k].x), fabsf(pv[k].y)));
        }
      }
    }
    if (m > 0.f) atomicMax(&sxm[q], __float_as_uint(m));
  }
  __syncthreads();
  if (tid < R) sc->xm[cta][tid] = sxm[tid];
  cluster_sync();
  // the operand rows 4 q + {Re hi, Im hi, Re lo, Im lo} (zero for q >= R), as k_x_to_tc
  unsigned xm = 0u;
  if (live)
    for (int c = 0; c < CS_CTAS; ++c) xm = max(xm, __ldcg(&sc->xm[c][q]));
  const float scale = live ? pow2f(scale_exp(xm)) : 0.f;
  if (gid < stride) {
    for (int j = gid; j < N; j += stride) {
      const int it = j / Rp, a = it / KG, kg = it % KG;
      __align__(16) __half v[4][8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        float2 pv = make_float2(0.f, 0.f);
        if (live && 8 * kg + k < n) pv = p[((size_t)a * n + 8 * kg + k) * R + q];
        const float re = pv.x * scale, im = pv.y * scale;
        const __half rh = __float2half_rn(re), ih = __float2half_rn(im);
        v[0][k] = rh;
        v[1][k] = ih;
        v[2][k] = __float2half_rn(re - __half2float(rh));
        v[3][k] = __float2half_rn(im - __half2float(ih));
      }
      char* tile = xtc + (size_t)a * (4 * Rp) * Kp * 2;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int row = 4 * q + h;
        *reinterpret_cast<uint4*>(tile + (size_t)(row / 8) * (Kp * 16) + kg * 128 + (row % 8) * 16) =
            *reinterpret_cast<const uint4*>(v[h]);
      }
    }
  }
  // bookkeeping (nobody reads it in this launch any more)
  if (gid < R) {
    ctl->rr[par ^ 1][gid] = s_rn[gid];
    xmax[gid] = xm;
  }
  if (cta == 0) {
    __syncthreads();
    if (tid == 0) {
      const int it = ctl->iter + 1;
      ctl->iter = it;
      int all = 1;
      for (int i = 0; i < R; ++i) {
        const double v = ctl->rr[par ^ 1][i];
        if (!ctl->done[i] && (v <= ctl->stop[i] || it >= maxiter || !(v == v))) ctl->done[i] = 1;
        all &= ctl->done[i];
      }
      ctl->all_done = all;
    }
  }
}

// Couplings split and one-launch step for grids whose pairs leave SMs idle and whose
// vectors fit the cluster's items.
static bool small_grid(const Coarse& A, const TcGeom& g, int& nsplit) {
  const int npairs = (int)((A.Vc + g.sites - 1) / g.sites), slots = 2 * device_sms();
  nsplit = std::max(1, std::min(8, slots / npairs));
  const int threads = CS_CTAS * CS_THREADS / g.Rp * g.Rp;
  return A.Vc * (g.Kp / 8) * g.Rp <= (size_t)threads * CS_ITEMS;
}

int coarse_cg_tc(Ctx& c, Coarse& A, int R, const void* rhs, void* sol, double tol, int maxiter, double shift) {
  coarse_tc_prepare(c, A);
  const size_t ne = A.Vc * A.nvec;
  const size_t nc = ne * R;
  const TcGeom g = tc_geom(A.nvec, R, tc_parts(A));
  int nsplit = 1;
  const bool small = small_grid(A, g, nsplit);
  if (!small) nsplit = 1;
  A.work.ensure((2 + nsplit) * nc * sizeof(float2));
  A.ctl.ensure(sizeof(CCtlT) + sizeof(CgStepScratch));
  float2* r = A.work.as<float2>();
  float2* p = r + nc;
  float2* w = p + nc;
  CCtlT* ctl = A.ctl.as<CCtlT>();
  CgStepScratch* sc = reinterpret_cast<CgStepScratch*>(ctl + 1);
  unsigned* xmax = A.tcs.as<TcState>()->xmax;
  const int* skip = &ctl->all_done;
  const unsigned ge = (unsigned)((ne + 255) / 256);
  HDCG_CUDA(cudaMemsetAsync(xmax, 0, RMAX * sizeof(unsigned), c.stream));
  k_cgt_init<<<ge, 256, 0, c.stream>>>((const float2*)rhs, (float2*)sol, r, p, ne, R, xmax,
                                       make_reduction(c, ge, RMAX, &ctl->rr[0][0], 0));
  k_cgt_start<<<1, 1, 0, c.stream>>>(ctl, R, tol, maxiter);
  c.launches += 2;
  if (small) coarse_tc_to_b(c, A, R, p, xmax, skip);   // afterwards the step kernel writes the operand
  auto iteration = [&](int par) {
    if (small) {
      launch_tc(c, A, R, p, w, xmax, skip, &ctl->pAp[0], shift, c.tc_force ? c.tc_force : 2, nullptr, nsplit);
      k_cgt_step<<<CS_CTAS, CS_THREADS, 0, c.stream>>>((float2*)sol, r, p, w, nsplit, nc, (int)A.Vc, A.nvec, R, g.Rp, g.Kp,
                                                       A.xtc.as<char>(), ctl, sc, par, maxiter, xmax);
      ++c.launches;
      return;
    }
    coarse_tc_to_b(c, A, R, p, xmax, skip);
    coarse_tc_apply(c, A, R, p, w, xmax, skip, &ctl->pAp[0], shift);
    k_cgt_update<<<ge, 256, 0, c.stream>>>((float2*)sol, r, p, w, ne, R, ctl, par, xmax,
                                           make_reduction(c, ge, RMAX, &ctl->rr[par ^ 1][0], 0));
    k_cgt_p<<<ge, 256, 0, c.stream>>>(p, r, ne, R, ctl, par, xmax);
    k_cgt_check<<<1, 1, 0, c.stream>>>(ctl, R, par, maxiter);
    c.launches += 3;
  };
  // pairs of iterations (parities 0, 1): the first directly, later ones as a replayed graph
  uint64_t shift_bits;
  std::memcpy(&shift_bits, &shift, sizeof(shift_bits));
  const std::vector<uintptr_t> key = {(uintptr_t)A.work.p, (uintptr_t)A.ctl.p, (uintptr_t)sol, (uintptr_t)A.Atc.p,
                                      (uintptr_t)A.xtc.p, (uintptr_t)A.tcs.p, (uintptr_t)c.red_partials.p,
                                      (uintptr_t)c.red_ticket.p, (uintptr_t)R, (uintptr_t)maxiter,
                                      (uintptr_t)shift_bits, (uintptr_t)nsplit};
  int queued = 0;
  int batch = std::max(2, A.last_iters);
  CCtlT& h = *c.pinned.at<CCtlT>(4096);
  while (true) {
    for (int bq = 0; bq < batch && queued < maxiter; bq += 2, queued += 2) {
      if (queued == 0) {
        iteration(0);
        iteration(1);
      } else {
        run_captured(c, A.graph_cg, key, [&] {
          iteration(0);
          iteration(1);
        });
      }
    }
    HDCG_CUDA(cudaGetLastError());
    HDCG_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(CCtlT), cudaMemcpyDeviceToHost, c.stream));
    coarse_tc_check(c, A);   // synchronises the stream
    if (h.all_done || queued >= maxiter) break;
    batch = 2;
  }
  A.last_iters = std::max(1, h.iter);
  return h.iter;
}

// ---------------------------------------------------------------------------------
// canonical multi-right-hand-side apply: x, y [R][Vc][Nvec] complex double (device)
// ---------------------------------------------------------------------------------

// [r][e] complex double <-> [e][r] complex float or double
template <typename V>
__global__ void k_canon_to_multi(const double2* __restrict__ in, V* out, size_t ne, int R) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ne * R) return;
  const size_t e = t / R;
  const int r = (int)(t % R);
  const double2 v = in[(size_t)r * ne + e];
  out[t] = {(decltype(out[t].x))v.x, (decltype(out[t].y))v.y};
}
template <typename V>
__global__ void k_multi_to_canon(const V* __restrict__ in, double2* out, size_t ne, int R) {
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ne * R) return;
  const size_t e = t / R;
  const int r = (int)(t % R);
  out[(size_t)r * ne + e] = make_double2((double)in[t].x, (double)in[t].y);
}

void coarse_canon_to_multi(Ctx& c, const void* in64, float2* out, size_t ne, int R) {
  k_canon_to_multi<float2><<<(unsigned)((ne * R + 255) / 256), 256, 0, c.stream>>>((const double2*)in64, out, ne, R);
  HDCG_CUDA(cudaGetLastError());
  ++c.launches;
}
void coarse_multi_to_canon(Ctx& c, const float2* in, void* out64, size_t ne, int R) {
  k_multi_to_canon<float2><<<(unsigned)((ne * R + 255) / 256), 256, 0, c.stream>>>(in, (double2*)out64, ne, R);
  HDCG_CUDA(cudaGetLastError());
  ++c.launches;
}

int coarse_solve_canon(Ctx& c, Coarse& A, int R, const void* b64, void* x64, double tol, int maxiter) {
  HDCG_REQUIRE(R >= 1 && R <= RMAX, HDCG_ERR_ARG, "1..16 right-hand sides");
  const size_t ne = A.Vc * A.nvec, nc = ne * R;
  const unsigned gt = (unsigned)((nc + 255) / 256);
  DevMem& tmp = c.coarse_io[0];
  int it;
  if (A.l2) A.l2->last_broke = 0;
  if (A.vec_prec() == HDCG_F32) {
    tmp.ensure(2 * nc * sizeof(float2));
    float2* bi = tmp.as<float2>();
    float2* xi = bi + nc;
    k_canon_to_multi<float2><<<gt, 256, 0, c.stream>>>((const double2*)b64, bi, ne, R);
    it = coarse_cg_multi(c, A, R, bi, xi, tol, maxiter);
    k_multi_to_canon<float2><<<gt, 256, 0, c.stream>>>(xi, (double2*)x64, ne, R);
    HDCG_REQUIRE(!(A.l2 && A.l2->last_broke), HDCG_ERR_BREAKDOWN,
                 "level-1 solve: (p, A p) <= 0 or a non-finite residual before the tolerance");
  } else {
    tmp.ensure(2 * nc * sizeof(double2));
    double2* bi = tmp.as<double2>();
    double2* xi = bi + nc;
    k_canon_to_multi<double2><<<gt, 256, 0, c.stream>>>((const double2*)b64, bi, ne, R);
    it = coarse_cg_multi(c, A, R, bi, xi, tol, maxiter);
    k_multi_to_canon<double2><<<gt, 256, 0, c.stream>>>(xi, (double2*)x64, ne, R);
  }
  c.launches += 2;
  HDCG_CUDA(cudaGetLastError());
  HDCG_CUDA(cudaStreamSynchronize(c.stream));
  return it;
}

// Mean device time of one tensor-core stencil apply (k_capply_tc alone) to R
// Gaussian coarse vectors: 3 warm-up launches, then reps launches between two
// CUDA events on the handle's stream (the B operand is prepared once).
double coarse_tc_time_us(Ctx& c, Coarse& A, int R, int reps) {
  HDCG_REQUIRE(coarse_tc_supported(A), HDCG_ERR_ARG, "the tensor-core apply needs an FP16 or FP32 A, Nvec <= 64");
  HDCG_REQUIRE(R >= 1 && R <= RMAX && reps >= 1, HDCG_ERR_ARG, "1..16 right-hand sides, reps >= 1");
  coarse_tc_prepare(c, A);
  const size_t ne = A.Vc * A.nvec, nc = ne * R;
  DevMem tmp;
  tmp.ensure(2 * nc * sizeof(float2));
  float2* xi = tmp.as<float2>();
  float2* yi = xi + nc;
  coarse_noise(c, xi, nc, 0x7e57);
  unsigned* xmax = A.tcs.as<TcState>()->xmax;
  coarse_tc_max(c, xi, ne, R, xmax);
  coarse_tc_to_b(c, A, R, xi, xmax, nullptr);
  for (int i = 0; i < 3; ++i) coarse_tc_apply(c, A, R, xi, yi, xmax, nullptr, nullptr, 0.0);
  cudaEvent_t e0, e1;
  HDCG_CUDA(cudaEventCreate(&e0));
  HDCG_CUDA(cudaEventCreate(&e1));
  HDCG_CUDA(cudaEventRecord(e0, c.stream));
  for (int i = 0; i < reps; ++i) coarse_tc_apply(c, A, R, xi, yi, xmax, nullptr, nullptr, 0.0);
  HDCG_CUDA(cudaEventRecord(e1, c.stream));
  HDCG_CUDA(cudaEventSynchronize(e1));
  float ms = 0.f;
  HDCG_CUDA(cudaEventElapsedTime(&ms, e0, e1));
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  coarse_tc_check(c, A);
  return 1e3 * ms / reps;
}

void coarse_apply_multi_canon(Ctx& c, Coarse& A, int R, const void* x64, void* y64) {
  HDCG_REQUIRE(R >= 1 && R <= RMAX, HDCG_ERR_ARG, "1..16 right-hand sides");
  const size_t ne = A.Vc * A.nvec, nc = ne * R;
  const unsigned gt = (unsigned)((nc + 255) / 256);
  if (coarse_tc_supported(A)) {
    // the operand straight from x, the result straight into y: no staging
    coarse_tc_prepare(c, A);
    const double2* x = (const double2*)x64;
    unsigned* xmax = A.tcs.as<TcState>()->xmax;
    HDCG_CUDA(cudaMemsetAsync(xmax, 0, RMAX * sizeof(unsigned), c.stream));
    k_canon_max<<<dim3((unsigned)((ne + 255) / 256), (unsigned)R), 256, 0, c.stream>>>(x, ne, xmax);
    const TcGeom g = tc_geom(A.nvec, R, tc_parts(A));
    A.xtc.ensure(A.Vc * (size_t)g.b_bytes);
    const size_t nt = A.Vc * (size_t)(g.Kp / 8) * g.Rp;
    k_canon_to_tc<<<(unsigned)((nt + 255) / 256), 256, 0, c.stream>>>(x, A.xtc.as<uint4>(), A.Vc, A.nvec, R, g.Rp,
                                                                      g.Kp, xmax);
    HDCG_CUDA(cudaGetLastError());
    c.launches += 2;
    tc_apply(c, A, R, nullptr, nullptr, xmax, nullptr, nullptr, 0.0, (double2*)y64);
    coarse_tc_check(c, A);
    return;
  }
  // FP32 / FP64 operator: the CUDA-core kernel on [a][k][r] complex double
  DevMem& tmp = c.coarse_io[0];
  tmp.ensure(2 * nc * sizeof(double2));
  double2* xi = tmp.as<double2>();
  double2* yi = xi + nc;
  k_canon_to_multi<double2><<<gt, 256, 0, c.stream>>>((const double2*)x64, xi, ne, R);
  coarse_apply_multi(c, A, R, xi, yi);
  k_multi_to_canon<double2><<<gt, 256, 0, c.stream>>>(yi, (double2*)y64, ne, R);
  c.launches += 2;
  HDCG_CUDA(cudaGetLastError());
  HDCG_CUDA(cudaStreamSynchronize(c.stream));
}

}  // namespace hdcg
