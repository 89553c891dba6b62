// Fine-operator hop passes of 16-bit storage on the tensor cores (Ls 8, 16, 32).
//
// One hop is, per output site, a contraction with the Ls fifth-dimension slices
// as rows: D[s][out] = sum_k psi[s][k] M[k][out], k over the 8 neighbours' 24
// reals and out over the site's 24 reals, M built from the eight links and the
// spin projectors.  The entries of (1 -+ gamma_mu) are 0, +-1 and +-i, so M holds
// link components with a sign or with real and imaginary part exchanged: the
// 16-bit links and the 16-bit fields enter mma.m16n8k16 exactly as stored and every
// product is exact.  The FP32 sums are truncated towards zero (mma.cuh) where the
// scalar pass rounds u -+ A l and its sums to nearest: against 64 bits both are as
// far off as the 16-bit storage makes them (H of FP16 fields 3.16e-4 Shamir, 3.46e-4
// Moebius, BF16 2.53e-3 and 2.77e-3, either pass within 0.1 %), and <psi, H psi> moves by
// 1e-7 of itself on average, towards zero.  M differs from site to site and is 24 columns wide, which
// rules out tcgen05: its M = 128 rows would share one shared-memory operand.
//
// Shape: m16 are 16 slices of one 4D site (Ls 32: two tiles, Ls 8: half a tile),
// n8 is one output spin (3 colours x re, im; 2 columns idle).  k may be permuted
// freely as long as both operands agree, so lane (g, t) = (lane / 4, lane % 4)
// supplies colour t of row g (t = 3 is idle: zeros), and one k8 is one neighbour
// and one of its spins: of each neighbour an output spin takes its own spin and
// the one that gamma_mu pairs it with, 16 k8 = 8 MMAs per output spin, 32 per
// site (for 16 x 1440 scalar flops).
//
// Fragments come straight from memory: with the 16-bit layout (common.cuh) a
// granule is colour t of one slice with its four spins, i.e. four A registers,
// and 8 lanes (two slices, three colours) read 96 contiguous bytes.  What bounds
// the pass is this load path: with the chunks of a site apart (and each lane
// taking other directions) a quarter warp touched four lines per load and the L1
// data pipe was 85 to 91 % busy with 270 wavefronts per site.  Loads run a site
// ahead (see load_tile), and 12 warps with their loads in flight hide more than 16
// that wait.  The B register of
// output column g = 2 colour + {re, im} is the one link entry U[colour][t] with a
// byte permutation and a sign mask that depend on the lane only.
//
// The s-direction operators act on the FP32 accumulators (lane t < 3: colour t,
// all four spins, slices g + 8 q).  K on the input of pass A (Moebius) is linear
// in s and acts per chirality of the input, so the sums over the own and over the
// partner spins are kept apart and K is applied to the two sums, not to the eight
// neighbours.  A lane's results are whole granules; P_s of the self term in
// passes B and D is a load of the neighbouring slice.
//
// Per pass (mean of the four, FP16, 24^3 x 48 x 16; the field's own bytes need 129
// us at the copy rate): Moebius 399 us with the scalar kernel, 277 us here; Shamir
// 360 and 247; Ls 8 204 and 184; BF16 Ls 32 on 16^3 x 32 164 and 139; 8^4 x 16 9.0
// and 7.9.  Now the L1 data pipe is 57 to 74 % busy, the issue slots 42 to 62 %, HBM
// 30 to 47 %.
#pragma once

namespace hdcg {
namespace tch {

template <typename St> __device__ __forceinline__ float2 unpack2(unsigned v) {
  if constexpr (std::is_same<St, f16_t>::value) return h2f(v);
  else return b2f(v);
}

// The slices s = g + 8 q, q < S, of one column over the eight lanes g; values of
// slice s - d (DOWN) or s + d, s taken modulo Ls = 8 S.  d < 8: one shuffle per
// value, lanes that wrap take the one of the next group of eight; d >= 8: own registers.
template <int S, bool DOWN>
__device__ __forceinline__ void shift(const float (&v)[S], float (&o)[S], int d, int lane) {
  if (d >= 8) {
#pragma unroll
    for (int q = 0; q < S; ++q) o[q] = v[(DOWN ? q + S - d / 8 : q + d / 8) & (S - 1)];
  } else {
    float x[S];
#pragma unroll
    for (int q = 0; q < S; ++q) x[q] = __shfl_sync(FULL_MASK, v[q], DOWN ? lane - 4 * d : lane + 4 * d);
    const int g = lane >> 2;
    const bool wrap = DOWN ? g < d : g + d >= 8;
#pragma unroll
    for (int q = 0; q < S; ++q) o[q] = wrap ? x[(DOWN ? q + S - 1 : q + 1) & (S - 1)] : x[q];
  }
}

// v[spin][q][ri] <- a v + b P v (ADD: v + b P v); spins 0, 1 are chirality +
template <int S, bool DAG, bool ADD>
__device__ __forceinline__ void s_step(float (&v)[4][S][2], float a, float b, int d, int lane, float m) {
  const int g = lane >> 2;
#pragma unroll
  for (int sp = 0; sp < 4; ++sp)
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      float c[S], o[S];
#pragma unroll
      for (int q = 0; q < S; ++q) c[q] = v[sp][q][ri];
      if ((sp < 2) != DAG) shift<S, true>(c, o, d, lane);
      else shift<S, false>(c, o, d, lane);
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const bool wall = (sp < 2) != DAG ? g + 8 * q < d : g + 8 * q + d >= 8 * S;
        const float f = wall ? -m * b : b;
        v[sp][q][ri] = ADD ? f * o[q] + c[q] : a * c[q] + f * o[q];
      }
    }
}

template <int S, bool DAG>
__device__ __forceinline__ void minv(float (&v)[4][S][2], int lane, const HopArgs& a) {
#pragma unroll
  for (int j = 0; j < (S == 1 ? 3 : S == 2 ? 4 : 5); ++j)
    s_step<S, DAG, true>(v, 1.f, a.frpow[j], 1 << j, lane, a.fmass);
#pragma unroll
  for (int sp = 0; sp < 4; ++sp)
#pragma unroll
    for (int q = 0; q < S; ++q) {
      v[sp][q][0] *= a.fminv_norm;
      v[sp][q][1] *= a.fminv_norm;
    }
}

// spin paired with sp by gamma_mu, and the sign of its phase for SG = +1 (the
// phase itself: i along x and z, 1 along y and t), from (1 - SG gamma_mu)
__host__ __device__ constexpr int partner(int mu, int sp) { return mu < 2 ? 3 - sp : sp ^ 2; }
__host__ __device__ constexpr bool partner_neg(int mu, int sp) {
  return mu == 0 ? sp >= 2 : mu == 3 ? true : sp == 1 || sp == 2;
}

constexpr int TC_WARPS = 4;   // warps (one 4D site each at a time) per CTA
// CTAs per SM: 128 registers at Ls 8, else 168 (at 128, Ls 16 spills in two of
// the passes)
__host__ __device__ constexpr int tc_ctas(int S) { return S == 1 ? 4 : 3; }

template <typename St, int PASS, bool MOB, int S>
__global__ void __launch_bounds__(32 * TC_WARPS, tc_ctas(S)) hop_tc_kernel(const HopArgs a) {
  constexpr int LS = 8 * S, NT = (S + 1) / 2, SQ = S == 1 ? 1 : 2;   // tiles of 16 rows, slices per tile and lane
  constexpr bool DAG = (PASS == PASS_C || PASS == PASS_D);
  constexpr bool SPLIT = PASS == PASS_A && MOB;
  constexpr bool EPI = (PASS == PASS_B || PASS == PASS_D);
  constexpr bool EARLY = S < 4;   // the epilogue's operands before the contraction (Ls 32 would spill)
  __shared__ double s_alpha;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int n4 = (int)(a.n5 / LS);
  const size_t roff = (size_t)blockIdx.y * a.fstride;
  const bool cg = PASS == PASS_D && a.cg_r != nullptr;
  if (cg) {
    if (threadIdx.x == 0) {
      const int rhs = blockIdx.y;
      double den = a.al_den0[rhs];
      if (a.al_den1) den += a.al_lam * a.al_den1[rhs];
      const bool live = a.al_mask == nullptr || a.al_mask[rhs] != 0;
      s_alpha = (den != 0.0 && live) ? a.al_num[rhs] / den : 0.0;
    }
    __syncthreads();
  }
  // column g: Re (even g) or Im of colour g / 2; U psi and i U psi from (Re U, Im U)
  constexpr unsigned NEG = 0x80008000u, NHI = 0x80000000u;
  const bool im = g & 1;
  const unsigned sel1 = im ? 0x1032u : 0x3210u, mask1 = im ? 0u : NHI;
  const unsigned seli = im ? 0x3210u : 0x1032u, maski = im ? NHI : NEG;
  // link entry U[g / 2][t]; idle lanes and columns take the zero that pads row 0
  const int lk = (g < 6 && t < 3) ? (g >> 1) * 4 + t : 3;
  float nhi = 0.f, nlo = 0.f;   // |out|^2 of this lane: double-float over its sites
  const int step = (int)gridDim.x * TC_WARPS;
  int x4 = (int)blockIdx.x * TC_WARPS + w;                 // the same for the whole warp
  int nb[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  auto neighbours = [&](int x) {
    const int4 n0 = __ldg(reinterpret_cast<const int4*>(a.nbr) + (size_t)x * 2);
    const int4 n1 = __ldg(reinterpret_cast<const int4*>(a.nbr) + (size_t)x * 2 + 1);
    nb[0] = n0.x; nb[1] = n0.y; nb[2] = n0.z; nb[3] = n0.w;
    nb[4] = n1.x; nb[5] = n1.y; nb[6] = n1.z; nb[7] = n1.w;
  };
  unsigned L[8];
  uint4 W[8][SQ];
  // colour t (idle lanes: colour 2 again, against zero link entries), slices
  // g + 8 (2 j + q) of the eight neighbours
  const uint4* in = a.in + roff + 3 * g + min(t, 2);
  auto load_tile = [&](int j) {
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const uint4* p = in + (size_t)(unsigned)nb[d] * (LS * 3) + 48 * j;
#pragma unroll
      for (int q = 0; q < SQ; ++q) W[d][q] = __ldg(p + 24 * q);
    }
  };
  auto load_links = [&](int x) {
    const unsigned* links = reinterpret_cast<const unsigned*>(a.links) + (size_t)(unsigned)x * 96 + lk;
#pragma unroll
    for (int d = 0; d < 8; ++d) L[d] = __ldg(links + 12 * d);
  };
  // A site's tile is on its way while the site before it goes through its
  // s-direction operators and stores; its neighbour indices one site earlier still.
  if (x4 < n4) {
    neighbours(x4);
    load_tile(0);
    load_links(x4);
    if (NT == 1 && x4 + step < n4) neighbours(x4 + step);
  }
  for (; x4 < n4; x4 += step) {
    // the self term's granules (slice s, and the halves of s - 1 and s + 1), early
    const size_t o0 = roff + (size_t)x4 * (LS * 3) + min(t, 2);
    uint4 self[S];
    uint2 side[S][2];
    auto load_self = [&] {
      const uint4* f2 = a.in2 + o0;
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const int s = g + 8 * q;
        self[q] = __ldg(f2 + 3 * s);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int ss = ((h == 0) != DAG ? s + LS - 1 : s + 1) & (LS - 1);
          side[q][h] = __ldg(reinterpret_cast<const uint2*>(f2 + 3 * ss) + h);
        }
      }
    };
    if (EPI && EARLY) load_self();
    float acc[SPLIT ? 2 : 1][4][NT][4];
#pragma unroll
    for (int h = 0; h < (SPLIT ? 2 : 1); ++h)
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[h][sp][j][i] = 0.f;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      if (j > 0) load_tile(j);
      // ---- the contraction: directions mu and mu + 4 share an MMA -----------------------------
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        unsigned BO[2], BP[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const unsigned l = L[mu + 4 * b];
          BO[b] = __byte_perm(l, 0u, sel1) ^ mask1;
          BP[b] = mu == 0 || mu == 2 ? __byte_perm(l, 0u, seli) ^ maski : BO[b];
        }
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) {
          const int pa = partner(mu, sp);
          auto word = [&](int b, int q, int s) {
            const uint4& v = W[mu + 4 * b][q < SQ ? q : 0];
            return q >= SQ ? 0u : s == 0 ? v.x : s == 1 ? v.y : s == 2 ? v.z : v.w;
          };
          mma<St>(acc[0][sp][j], word(0, 0, sp), word(0, 1, sp), word(1, 0, sp), word(1, 1, sp), BO[0], BO[1]);
          // forward SG = 1 (DAG: -1), backward the reverse
          const unsigned m0 = partner_neg(mu, sp) != DAG ? NEG : 0u, m1 = m0 ^ NEG;
          mma<St>(acc[SPLIT ? 1 : 0][sp][j], word(0, 0, pa), word(0, 1, pa), word(1, 0, pa), word(1, 1, pa),
                  BP[0] ^ m0, BP[1] ^ m1);
        }
      }
    }
    if (x4 + step < n4) {
      if (NT > 1) neighbours(x4 + step);
      load_tile(0);
      load_links(x4 + step);
      if (NT == 1 && x4 + 2 * step < n4) neighbours(x4 + 2 * step);
    }
    uint4 cr[S], cx[S], cp[S];
    auto load_cg = [&] {
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const size_t at = o0 + 3 * (g + 8 * q);
        cr[q] = a.cg_r[at];
        cx[q] = a.cg_x[at];
        cp[q] = __ldg(a.cg_p + at);
      }
    };
    if (EARLY && cg) load_cg();
    // ---- s-direction operators on v[spin][q][re, im] (lane t < 3: colour t) -----------------
    float v[4][S][2];
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)
#pragma unroll
      for (int q = 0; q < S; ++q)
#pragma unroll
        for (int ri = 0; ri < 2; ++ri) v[sp][q][ri] = acc[0][sp][q / 2][2 * (q & 1) + ri];
    if constexpr (SPLIT) {
      // K of the input: own spins have the output's chirality, partner spins the other
      float o[4][S][2];
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int q = 0; q < S; ++q)
#pragma unroll
          for (int ri = 0; ri < 2; ++ri) o[sp][q][ri] = acc[1][sp][q / 2][2 * (q & 1) + ri];
      s_step<S, false, false>(v, a.fb, a.fc, 1, lane, a.fmass);
      s_step<S, true, false>(o, a.fb, a.fc, 1, lane, a.fmass);
#pragma unroll
      for (int sp = 0; sp < 4; ++sp)
#pragma unroll
        for (int q = 0; q < S; ++q) {
          v[sp][q][0] += o[sp][q][0];
          v[sp][q][1] += o[sp][q][1];
        }
    }
    if (PASS == PASS_A) minv<S, false>(v, lane, a);
    if (PASS != PASS_B) {
      if (MOB) {
        s_step<S, DAG, false>(v, a.fb, a.fc, 1, lane, a.fmass);
      } else {
        const float k = PASS == PASS_A ? a.fb * a.fb : a.fb;
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
          for (int q = 0; q < S; ++q) {
            v[sp][q][0] *= k;
            v[sp][q][1] *= k;
          }
      }
    }
    if (PASS == PASS_C) minv<S, true>(v, lane, a);
    // ---- whole granules: slice g + 8 q, colour t -----------------------------------------------
    float nrm = 0.f;
    if (EPI && !EARLY) load_self();
    if (!EARLY && cg) load_cg();
    if (t < 3) {
#pragma unroll
      for (int q = 0; q < S; ++q) {
        const int s = g + 8 * q;
        const size_t at = o0 + 3 * s;
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = v[i / 2][q][i & 1];
        if constexpr (EPI) {
          // M_oo self: spins 0, 1 take slice s - 1, spins 2, 3 slice s + 1, DAG the reverse
          float f[8];
          unpack(St{}, self[q], f);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const bool dn = (h == 0) != DAG;
            const float2 y0 = unpack2<St>(side[q][h].x), y1 = unpack2<St>(side[q][h].y);
            const float bf = (dn ? s == 0 : s == LS - 1) ? a.fbeta * -a.fmass : a.fbeta;
            const float y[4] = {y0.x, y0.y, y1.x, y1.y};
#pragma unroll
            for (int i = 0; i < 4; ++i) x[4 * h + i] = (a.falpha * f[4 * h + i] + bf * y[i]) - 0.25f * x[4 * h + i];
          }
          if (PASS == PASS_D) {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] *= a.fsD;
            if (a.extra) {
              unpack(St{}, __ldg(a.extra + at), f);
#pragma unroll
              for (int i = 0; i < 8; ++i) x[i] += a.flam * f[i];
            }
          }
        }
        if (cg) {
          const float alpha = (float)s_alpha;
          float r[8], xv[8], p[8];
          unpack(St{}, cr[q], r);
          unpack(St{}, cx[q], xv);
          unpack(St{}, cp[q], p);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            r[i] -= alpha * x[i];
            xv[i] += alpha * p[i];
            x[i] = r[i];
          }
          a.cg_r[at] = pack(St{}, r);
          a.cg_x[at] = pack(St{}, xv);
        } else {
          a.out[at] = pack(St{}, x);
        }
        if (EPI && a.do_red) {
#pragma unroll
          for (int i = 0; i < 8; ++i) nrm = fmaf(x[i], x[i], nrm);
        }
      }
    }
    if (EPI && a.do_red) {
      float s, e;
      two_sum(nhi, nrm, s, e);
      nhi = s;
      nlo = __fadd_rn(nlo, e);
    }
  }
  if constexpr (EPI)
    if (a.do_red) norm2_reduce(nhi, nlo, a.red);
}

}  // namespace tch

// one hop pass, Ls 8, 16 or 32 (16-bit storage)
template <typename St>
void launch_hop_tc(int pass, bool mob, const HopArgs& a, dim3 grid, cudaStream_t st) {
#define HDCG_HOP_TC_S(P, S)                                                                     \
  if (mob) tch::hop_tc_kernel<St, P, true, S><<<grid, 32 * tch::TC_WARPS, 0, st>>>(a);          \
  else tch::hop_tc_kernel<St, P, false, S><<<grid, 32 * tch::TC_WARPS, 0, st>>>(a);
#define HDCG_HOP_TC(P)                                                                          \
  if (pass == P) {                                                                              \
    if (a.Ls == 8) { HDCG_HOP_TC_S(P, 1) }                                                      \
    else if (a.Ls == 16) { HDCG_HOP_TC_S(P, 2) }                                                \
    else { HDCG_HOP_TC_S(P, 4) }                                                                \
    return;                                                                                     \
  }
  HDCG_HOP_TC(PASS_A) HDCG_HOP_TC(PASS_B) HDCG_HOP_TC(PASS_C) HDCG_HOP_TC(PASS_D)
#undef HDCG_HOP_TC
#undef HDCG_HOP_TC_S
}

}  // namespace hdcg
