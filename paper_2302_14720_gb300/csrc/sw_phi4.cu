// sw_phi4.cu -- the multicluster update of the O(4) phi^4 theory in four
// dimensions (the paper's §3, Eqs. 2 and 3), conventions O1-O5 of
// include/sw.h.
//
// One update at counter t:
//   host      the direction r, uniform on the 3-sphere (O3), by rejection
//             from Philox blocks, computed on the host;
//   project   a thread per site: a_x = phi_x . r;
//   brick     a CTA per brick of sites draws the words of block (x, t, 4, 0)
//             and bonds the forward edges (Eq. 2): none unless the two
//             projections have the same sign, else iff w < (1 - e^{-z}) 2^32
//             with z = 4 kappa a_x a_y; the exponential is this file's own
//             (range reduction and a Taylor polynomial with fused
//             multiply-adds), so the decisions are reproducible bit for bit.
//             The brick's clusters are labelled in shared memory;
//   unite     lock-free union-find over int32 parents (larger root under the
//             smaller) of the bonds that leave a brick, so roots are the
//             clusters' smallest sites;
//   roots     every local root gets its cluster's root and the flip drawn for
//             it (bit 31 of word 0 of block (root, t, 6, 0));
//   reflect   every site of a flipped cluster is reflected in the hyperplane
//             orthogonal to r (Eq. 3): phi <- phi - 2 (phi . r) r;
//   observe   E = sum over the 4N edges of phi_x . phi_{x+mu} and M = sum of
//             phi, in fixed point or binary64 (the summation order differs
//             from a serial sum, so these agree with one to rounding only).
// Every operation that feeds a bond decision or a new field value is an
// explicitly rounded intrinsic, so nothing is contracted differently from a
// serial restatement compiled without contraction.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>

#include <cmath>
#include <limits>
#include <new>

#include "sw.h"
#include "sw_internal.h"

namespace {

constexpr int kFindCap = 1 << 24;
constexpr int kUnionCap = 1 << 16;

struct Dir {
  double r[4];
  double m2r[4];  // -2 r, exactly
};

// One site's field, binary64 x 4 (O1), 32-byte aligned.
struct __align__(32) F4 {
  double x, y, z, w;
};

// e^{-z} for 0 <= z <= 40 (0 beyond, where 1 - e^{-z} rounds to 1): z =
// n ln2 + r with a 32-bit head of ln2 (n * head exact) and its tail (Cody
// and Waite), e^{-r} by the Taylor series to degree 14 with fused
// multiply-adds (remainder below 2^-60 for |r| <= 0.35), then 2^-n.
__device__ double exp_neg(double z) {
  constexpr double kLn2Head = 0x1.62e42feep-1;
  constexpr double kLn2Tail = 0x1.a39ef35793c76p-33;
  constexpr double kInvLn2 = 0x1.71547652b82fep+0;
  constexpr double kInvFact[15] = {0x1p+0,
                                   0x1p+0,
                                   0x1p-1,
                                   0x1.5555555555555p-3,
                                   0x1.5555555555555p-5,
                                   0x1.1111111111111p-7,
                                   0x1.6c16c16c16c17p-10,
                                   0x1.a01a01a01a01ap-13,
                                   0x1.a01a01a01a01ap-16,
                                   0x1.71de3a556c734p-19,
                                   0x1.27e4fb7789f5cp-22,
                                   0x1.ae64567f544e4p-26,
                                   0x1.1eed8eff8d898p-29,
                                   0x1.6124613a86d09p-33,
                                   0x1.93974a8c07c9dp-37};
  if (z > 40.0) return 0.0;
  const double n = floor(__dadd_rn(__dmul_rn(z, kInvLn2), 0.5));
  const double r = __fma_rn(-n, kLn2Tail, __fma_rn(-n, kLn2Head, z));
  double p = kInvFact[14];
#pragma unroll
  for (int k = 13; k >= 0; --k) p = __fma_rn(p, -r, kInvFact[k]);
  return ldexp(p, -(int)n);
}

__device__ __forceinline__ double proj(const F4 f, const Dir& d) {
  return __fma_rn(f.w, d.r[3], __fma_rn(f.z, d.r[2], __fma_rn(f.y, d.r[1], __dmul_rn(f.x, d.r[0]))));
}

// The coordinates of site x = c0 + L c1 + L^2 c2 + L^3 c3 (O2); L^4 < 2^31,
// so 32-bit arithmetic holds every index.
struct Coords {
  uint32_t c[4];
};
__device__ __forceinline__ Coords coords_of(uint32_t x, uint32_t L) {
  Coords k;
#pragma unroll
  for (int mu = 0; mu < 3; ++mu) {
    const uint32_t q = x / L;
    k.c[mu] = x - q * L;
    x = q;
  }
  k.c[3] = x;
  return k;
}

// The forward neighbour of x in direction mu (periodic), stride = L^mu.
__device__ __forceinline__ uint32_t nb(uint32_t x, int mu, const Coords& k, uint32_t L, uint32_t stride) {
  return k.c[mu] == L - 1 ? x - (L - 1) * stride : x + stride;
}

// The bond decision of Eq. 2 for the edge (x, y): bonded iff q = a_x a_y > 0
// and w < (1 - e^{-z}) 2^32 with z = k4 q, all in binary64 with exp_neg.
// GB300 runs binary64 at a small fraction of its binary32 rate, so a
// binary32 estimate decides first, from the projections rounded to binary32
// (af, each within 2^-24 relative): with both |af| >= 2^-60 and k4 >= 2^-66
// (k4 af is then a normal number; smaller couplings come as NaN) the estimate
// of z (three roundings of 2^-24 and two products) is within 5 * 2^-24 relative,
// or below 2^-126 with z, and has the sign of q, so for 0 < z <= 40 e^{-z} from expf (2 ulp) is within
// 40 * 5 * 2^-24 + 2^-22 of the binary64 value and (1 - e) 2^32 within 2^16 of
// the binary64 threshold; beyond 40 both thresholds are 2^32 to binary32
// precision, and for z < 0 the estimate is not positive. A word more than 2^18
// from the estimate (words round to binary32 within 2^8) takes the same
// decision as the binary64 test; the others (about 1e-4 of the edges), edges
// with a tiny projection and estimates that are not a number take the
// binary64 test itself.
__device__ __forceinline__ bool bonded_exact(double ax, double ay, double k4, uint32_t w) {
  const double q = __dmul_rn(ax, ay);
  if (!(q > 0.0)) return false;
  const double e = exp_neg(__dmul_rn(k4, q));
  return __uint2double_rn(w) < __dmul_rn(__dsub_rn(1.0, e), 0x1p32);
}

__device__ __forceinline__ bool bonded(const double* a, uint32_t x, uint32_t y, float fx, float fy, float k4f,
                                       double k4, uint32_t w) {
  const float z = __fmul_rn(__fmul_rn(k4f, fx), fy);
  const float d = __fsub_rn((float)w, __fmaf_rn(-expf(-z), 0x1p32f, 0x1p32f));  // w - (1 - e) 2^32
  if (fabsf(d) > 0x1p18f && fminf(fabsf(fx), fabsf(fy)) >= 0x1p-60f) return d < 0.0f;
  return bonded_exact(a[x], a[y], k4, w);
}

__device__ __forceinline__ double unit_interval(uint32_t w) {
  return __dsub_rn(__dmul_rn(__dadd_rn(__uint2double_rn(w), 0.5), 0x1p-31), 1.0);
}

// Union-find over parents in global or shared memory: a link is one
// compare-and-swap of a root's own entry, so only entries of non-roots change
// otherwise, and halving a path is a plain store of an ancestor. G: global
// memory (loads and stores past L1, which is not kept coherent).
template <bool G>
__device__ __forceinline__ int ld_par(const int* p) {
  return G ? __ldcg(p) : *(const volatile int*)p;
}
template <bool G>
__device__ __forceinline__ void st_par(int* p, int v) {
  if (G) __stcg(p, v);
  else *(volatile int*)p = v;
}

// The unions of a warp's list of n pairs, pair(k, a, b) giving the k-th. One
// state machine per lane: a lane takes its next pair when its union is done,
// and every warp-wide trip moves each busy lane one step (both nodes to their
// grandparents, or at two distinct roots the larger hung under the smaller),
// so lanes with long walks do not idle the others. Every lane of the warp
// calls this.
template <bool G, typename Pair>
__device__ __forceinline__ void unite_list(int* par, int n, Pair pair, int* err) {
  int k = threadIdx.x & 31, a = 0, b = 0;
  bool busy = false;
  for (int it = 0;; ++it) {
    if (!busy && k < n) {
      pair(k, a, b);
      k += 32;
      busy = true;
    }
    if (!__any_sync(0xffffffffu, busy)) return;
    if (it >= kUnionCap) {
      if (busy) atomicCAS(err, 0, 1);
      return;
    }
    if (!busy) continue;
    const int pa = ld_par<G>(par + a), pb = ld_par<G>(par + b);
    if (pa == a && pb == b) {
      if (a == b) {
        busy = false;
      } else {
        const int hi = max(a, b), lo = min(a, b), old = atomicCAS(par + hi, hi, lo);
        busy = old != hi;  // another lane hung that root first: go on from its parent
        a = old;
        b = lo;
      }
    } else {
      const int ga = pa == a ? a : ld_par<G>(par + pa), gb = pb == b ? b : ld_par<G>(par + pb);
      if (ga != pa) st_par<G>(par + a, ga);
      if (gb != pb) st_par<G>(par + b, gb);
      a = ga;
      b = gb;
    }
  }
}

#define GRID_LOOP(i, n) \
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

__global__ void phi4_init_kernel(F4* phi, int64_t n, sw::KeySchedule ks, int cold) {
  GRID_LOOP(x, n) {
    if (cold) {
      phi[x] = F4{1.0, 0.0, 0.0, 0.0};
    } else {
      const uint4 w = sw::philox4x32_10(make_uint4((uint32_t)x, 0u, 7u, 0u), ks);
      phi[x] = F4{unit_interval(w.x), unit_interval(w.y), unit_interval(w.z), unit_interval(w.w)};
    }
  }
}

__device__ __forceinline__ uint32_t abs_high(double d) { return (uint32_t)__double2hiint(d) & 0x7fffffffu; }

// v rounded to binary32, by integer operations where the result is a normal
// number: the conversion instruction runs in the binary64 pipe, which bounds the
// projection (four operations a site; 164 -> 156 us at L = 64 without it).
__device__ __forceinline__ float to_binary32(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  if (((hi >> 20) & 0x7ffu) - 897u > 253u) return __double2float_rn(v);
  const uint32_t m = __funnelshift_l(lo, hi, 3);  // low bits of the exponent, 23 bits of the mantissa
  const uint32_t up = ((lo & 0x1fffffffu) + 0x0fffffffu + (m & 1u)) >> 29;  // to nearest, ties to even
  return __uint_as_float((hi & 0x80000000u) | ((m - (896u << 23) + up) & 0x7fffffffu));
}

// The projections in binary64 and, for the bond kernel's first test, rounded
// to binary32.
__global__ void phi4_project_kernel(const F4* phi, double* a, float* af, int64_t n, Dir d, uint32_t* top) {
  sw::start_next();
  sw::after_previous();
  uint32_t big = 0u;  // high word of the largest |component|
  GRID_LOOP(x, n) {
    const F4 f = phi[x];
    const double v = proj(f, d);
    a[x] = v;
    af[x] = to_binary32(v);
    big = max(max(max(big, abs_high(f.x)), abs_high(f.y)), max(abs_high(f.z), abs_high(f.w)));
  }
  if (top) {
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0) atomicMax(top, big);
  }
}

// ------------------------------------------------------------ clusters
//
// Bonds and clusters brick by brick: a CTA takes a brick of B0 x B1 x B2 x B3
// sites, decides the forward bonds of its sites and labels the brick's
// clusters in shared memory; only the bonds that leave a brick (14 % of the
// edges for 16 x 8 x 8 x 4) go to the union-find in global memory. With every
// edge united in global memory (L = 64) the bonds ran 180 us, the unions 960
// and the pass that points every site at its root 315, both waiting for
// dependent L2 loads with 4 of 32 lanes active; the brick kernel runs 275 us,
// bound by instruction issue (the Philox draws, expf and the walks), the unions
// that are left 122 and the local roots' pass 75 to 97.
//
// Within a brick the local site order is the global one, so a component's
// smallest local site is its smallest site. Results: par[x] = the smallest
// site of x's brick component (its local root; itself for a local root), and
// in bonds[x] the forward bonds that leave the brick (bits 0-3) and kLocalRoot
// for a local root.
constexpr uint32_t kLocalRoot = 16u;
constexpr int kSiteMask = 0x7fffffff;  // a parent entry without its decision bit

template <int B0, int B1, int B2, int B3, int NT>
__global__ void __launch_bounds__(NT)
    phi4_brick_kernel(const double* a, const float* af, uint8_t* bonds, int* par, int L, double k4, float k4f, uint32_t t,
                      sw::KeySchedule ks, int* err) {
  sw::start_next();
  sw::after_previous();
  constexpr int V = B0 * B1 * B2 * B3, S1 = B0, S2 = B0 * B1, S3 = B0 * B1 * B2;
  // a warp's list of unions: a round over 32 sites may append one entry per
  // site and direction, 96, so no list is shorter and none is left longer
  // than CAP - 96 between rounds
  constexpr int kRound = 3 * 32, NW = NT / 32, CAP = 2 * V / NW > kRound ? 2 * V / NW : kRound;
  __shared__ __align__(4) uint8_t s_buf[NW * CAP * 2 > 4 * V ? NW * CAP * 2 : 4 * V];
  float* const s_af = reinterpret_cast<float*>(s_buf);  // [V] projections, then the warps' lists
  __shared__ int s_par[V];
  __shared__ uint8_t s_b[V];  // bits 0-3: bonds inside the brick, 4-7: bonds that leave it
  const uint32_t uL = (uint32_t)L, L2 = uL * uL, L3 = L2 * uL;
  uint32_t q = blockIdx.x;
  const uint32_t g0 = (uL + B0 - 1) / B0, g1 = (uL + B1 - 1) / B1, g2 = (uL + B2 - 1) / B2;
  const uint32_t o0 = q % g0 * B0;
  q /= g0;
  const uint32_t o1 = q % g1 * B1;
  q /= g1;
  const uint32_t o2 = q % g2 * B2, o3 = q / g2 * B3;
  const uint32_t base = o0 + uL * o1 + L2 * o2 + L3 * o3;
  // the global site of local site l, and whether the lattice has it
  auto site = [&](int l) {
    return base + (uint32_t)(l % B0) + uL * (uint32_t)(l / S1 % B1) + L2 * (uint32_t)(l / S2 % B2) +
           L3 * (uint32_t)(l / S3);
  };
  auto valid = [&](int l) {
    return o0 + l % B0 < uL && o1 + l / S1 % B1 < uL && o2 + l / S2 % B2 < uL && o3 + l / S3 < uL;
  };
#pragma unroll 4
  for (int l = threadIdx.x; l < V; l += NT) s_af[l] = valid(l) ? af[site(l)] : 0.0f;
  __syncthreads();

  for (int l = threadIdx.x; l < V; l += NT) {
    uint32_t bits = 0u;
    if (valid(l)) {
      const uint32_t x = site(l);
      const uint4 w4 = sw::philox4x32_10(make_uint4(x, t, 4u, 0u), ks);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
      const uint32_t i[4] = {(uint32_t)(l % B0), (uint32_t)(l / S1 % B1), (uint32_t)(l / S2 % B2), (uint32_t)(l / S3)};
      const uint32_t o[4] = {o0, o1, o2, o3}, gs[4] = {1u, uL, L2, L3};
      constexpr uint32_t B[4] = {B0, B1, B2, B3}, S[4] = {1, S1, S2, S3};
      const float fx = s_af[l];
#pragma unroll
      for (int mu = 0; mu < 4; ++mu) {
        const bool last = o[mu] + i[mu] + 1 == uL, inside = i[mu] + 1 < B[mu] && !last;
        const uint32_t y = last ? x - (uL - 1) * gs[mu] : x + gs[mu];
        const float fy = inside ? s_af[l + S[mu]] : af[y];
        if (bonded(a, x, y, fx, fy, k4f, k4, w[mu])) bits |= (inside ? 1u : 16u) << mu;
      }
    }
    s_b[l] = (uint8_t)bits;
  }
  __syncthreads();

  // every site starts under the first site of its run of x0 bonds, and a bond
  // in another direction is skipped when the one to its left joins the same
  // two runs
  for (int l = threadIdx.x; l < V; l += NT) {
    int r = l;
    while (r % B0 != 0 && (s_b[r - 1] & 1u)) --r;
    s_par[l] = r;
  }
  __syncthreads();
  {
    // the warp's bonds to unite, as l + V (mu - 1)
    constexpr int J = V / NT;
    static_assert(V % NT == 0 && 3 * V <= 65536, "list entries");
    static_assert(CAP >= kRound && NW * CAP * sizeof(uint16_t) <= sizeof s_buf, "a round's entries fit the list");
    uint16_t* const list = reinterpret_cast<uint16_t*>(s_buf) + (threadIdx.x >> 5) * CAP;
    const int lane = threadIdx.x & 31;
    int n = 0;
    auto drain = [&] {
      __syncwarp();
      unite_list<false>(
          s_par, n,
          [&](int k, int& x, int& y) {
            const int e = list[k], mu = e / V;
            x = e - mu * V;
            y = x + (mu == 0 ? S1 : mu == 1 ? S2 : S3);
          },
          err);
      __syncwarp();
      n = 0;
    };
#pragma unroll 1
    for (int j = 0; j < J; ++j) {
      const int l = threadIdx.x + j * NT;
      const uint32_t b = s_b[l], left = l % B0 != 0 && (s_b[l - 1] & 1u) ? s_b[l - 1] : 0u;
      constexpr int S[4] = {1, S1, S2, S3};
#pragma unroll
      for (int mu = 1; mu < 4; ++mu) {
        const bool need = ((b >> mu) & 1u) && !(((left >> mu) & 1u) && (s_b[l - 1 + S[mu]] & 1u));
        const uint32_t m = __ballot_sync(0xffffffffu, need);
        if (need) list[n + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(l + V * (mu - 1));
        n += __popc(m);
      }
      if (n > CAP - kRound) drain();
    }
    if (n) drain();
  }
  __syncthreads();
  for (int l = threadIdx.x; l < V; l += NT) {
    if (!valid(l)) continue;
    int r = l, p = s_par[r];
    while (p != r) {
      r = p;
      p = s_par[r];
    }
    const uint32_t x = site(l);
    par[x] = (int)site(r);
    bonds[x] = (uint8_t)((s_b[l] >> 4) | (r == l ? kLocalRoot : 0u));
  }
}

// Unions across brick borders, from the local roots of a bond's two sites;
// consecutive sites whose bonds join the same two local roots unite once. A
// warp lists the pairs of ROWS * 32 sites and unites them together: one site
// in two has no bond that leaves its brick, and a union is a chain of
// dependent L2 loads, so the lanes in flight set the rate. At L = 64 (bricks
// of 16 x 8 x 8 x 4) eight rows take 122 us, four 130, two 134, one 177 and a
// thread per site without lists 255; at L = 16 one row takes 12 us, two 12,
// four 17 and eight 21 (fewer warps than the chip holds).
constexpr int kUniteWarps = 4, kUniteCap = 2 * 128;
template <int ROWS>
__global__ void __launch_bounds__(32 * kUniteWarps)
    phi4_unite_kernel(const uint8_t* bonds, int* par, int L, int64_t n, int* err) {
  sw::start_next();
  sw::after_previous();
  __shared__ int2 s_list[kUniteWarps][kUniteCap];
  const int lane = threadIdx.x & 31;
  int2* const list = s_list[threadIdx.x >> 5];
  const int64_t x0 = ((int64_t)blockIdx.x * kUniteWarps + (threadIdx.x >> 5)) * (32 * ROWS);
  uint32_t b[ROWS];
#pragma unroll
  for (int j = 0; j < ROWS; ++j) b[j] = x0 + 32 * j + lane < n ? bonds[x0 + 32 * j + lane] & 15u : 0u;
  int cnt = 0;
  auto drain = [&] {
    __syncwarp();
    unite_list<true>(
        par, cnt,
        [&](int k, int& u, int& v) {
          u = list[k].x;
          v = list[k].y;
        },
        err);
    __syncwarp();
    cnt = 0;
  };
#pragma unroll
  for (int j = 0; j < ROWS; ++j) {
    if (!__any_sync(0xffffffffu, b[j] != 0u)) continue;
    const uint32_t x = (uint32_t)(x0 + 32 * j + lane);
    const Coords k = coords_of(x, (uint32_t)L);
    const int ra = b[j] ? __ldcg(par + x) : -1;
    int rb[4];
    uint32_t stride = 1;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu, stride *= (uint32_t)L)
      rb[mu] = (b[j] >> mu) & 1u ? __ldcg(par + nb(x, mu, k, (uint32_t)L, stride)) : -1;
    const int la = __shfl_up_sync(0xffffffffu, ra, 1);
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int lb = __shfl_up_sync(0xffffffffu, rb[mu], 1);
      const bool need = rb[mu] >= 0 && ra != rb[mu] && !(lane > 0 && la == ra && lb == rb[mu]);
      const uint32_t m = __ballot_sync(0xffffffffu, need);
      if (need) list[cnt + __popc(m & ((1u << lane) - 1u))] = make_int2(ra, rb[mu]);
      cnt += __popc(m);
    }
    if (cnt > kUniteCap - 128) drain();
  }
  if (cnt) drain();
}

// Every local root gets its cluster's root and the decision drawn for it:
// par[x] = root | decision << 31. Walks of other threads that meet a rewritten
// entry still end at the same root. A warp lists the local roots of its
// ROWS * 32 sites and takes them 32 at a time: four rows take 75 to 97 us at
// L = 64 (eight 82 to 106, a thread per site 104 to 116); at L = 16 one row
// takes 4.7 us and four 8.
constexpr int kRootWarps = 4;
template <int ROWS>
__global__ void __launch_bounds__(32 * kRootWarps)
    phi4_roots_kernel(const uint8_t* bonds, int* par, int64_t n, uint32_t t, sw::KeySchedule ks, int* err) {
  sw::start_next();
  sw::after_previous();
  __shared__ uint8_t s_list[kRootWarps][32 * ROWS];
  static_assert(32 * ROWS <= 256, "8-bit entries");
  const int lane = threadIdx.x & 31;
  uint8_t* const list = s_list[threadIdx.x >> 5];
  const int64_t x0 = ((int64_t)blockIdx.x * kRootWarps + (threadIdx.x >> 5)) * (32 * ROWS);
  uint32_t b[ROWS];
#pragma unroll
  for (int j = 0; j < ROWS; ++j) b[j] = x0 + 32 * j + lane < n ? bonds[x0 + 32 * j + lane] : 0u;
  int cnt = 0;
#pragma unroll
  for (int j = 0; j < ROWS; ++j) {
    const bool is = (b[j] & kLocalRoot) != 0u;
    const uint32_t m = __ballot_sync(0xffffffffu, is);
    if (is) list[cnt + __popc(m & ((1u << lane) - 1u))] = (uint8_t)(32 * j + lane);
    cnt += __popc(m);
  }
  __syncwarp();
  for (int k = lane; k < cnt; k += 32) {
    const int x = (int)x0 + list[k];
    int r = x, p = __ldcg(par + r) & kSiteMask;
    for (int it = 0; p != r; ++it) {
      if (it >= kFindCap) {
        atomicCAS(err, 0, 1);
        break;
      }
      r = p;
      p = __ldcg(par + r) & kSiteMask;
    }
    const uint32_t f = sw::philox4x32_10(make_uint4((uint32_t)r, t, 6u, 0u), ks).x & 0x80000000u;
    par[x] = (int)((uint32_t)r | f);
  }
}

__global__ void phi4_labels_kernel(const int* par, int* out, int64_t n) {
  sw::start_next();
  sw::after_previous();
  GRID_LOOP(x, n) out[x] = par[par[x] & kSiteMask] & kSiteMask;
}

// v, or infinity of its sign where v is finite and 2 v is not.
__device__ __forceinline__ double overflow_if_doubled(double v) {
  const bool over = abs_high(v) - 0x7fe00000u < 0x00100000u;
  const int hi = __double2hiint(v);
  return __hiloint2double(over ? (hi | 0x7ff00000) & ~0xfffff : hi, over ? 0 : __double2loint(v));
}

__global__ void phi4_reflect_kernel(F4* phi, const double* a, const int* par, int64_t n, Dir d) {
  sw::start_next();
  sw::after_previous();
  GRID_LOOP(x, n) {
    if (par[par[x] & kSiteMask] >= 0) continue;  // the cluster's decision: not flipped
    // a (-2 r_c) is the same product as (-2 a) r_c, both factors exact, and
    // saves one of five binary64 operations (171 -> 162 us at L = 64); where
    // -2 a overflows, an infinite a gives what it would
    const double ax = overflow_if_doubled(a[x]);
    F4 f = phi[x];
    f.x = __fma_rn(ax, d.m2r[0], f.x);
    f.y = __fma_rn(ax, d.m2r[1], f.y);
    f.z = __fma_rn(ax, d.m2r[2], f.z);
    f.w = __fma_rn(ax, d.m2r[3], f.w);
    phi[x] = f;
  }
}

// ------------------------------------------------------------ E and M
//
// E and M of the new field. GB300's binary64 rate is about 1/60 of its
// integer rate, and E takes 24 binary64 operations a site: at L = 64 the
// binary64 kernel below ran 739 us, all of it in that pipe; the fixed-point one
// runs about 225 us (16.8M sites, 0.54 GB of field), bound by instruction
// issue, its check of the field's range (below) included.
// Large lattices therefore sum in 64-bit fixed point: with 2^T above every
// |phi| (T from the largest component, which the projection kernel leaves in
// *top; a reflection keeps the length of phi), a component c becomes the
// integer nearest to c 2^(58-T): exact for components down to 2^-5 of 2^T,
// else off by at most half a unit. From there on neighbour sums, M and the
// products phi . S (S the sum of the four forward neighbours) are integers:
// the products from 30-bit low and signed high parts, a site's rounded once to
// a multiple of 2^60 (2^-56 of 2^2T). |phi| <= 2^58 and |S| <= 2^60 in these
// units, so a site adds at most 2^58 to the sum of phi . S 2^-60, its mixed
// products stay below 2^62.4 and the low ones below 2^62, and sixteen sites fit.
//
// One grid for the whole field serves fields whose components lie within a few
// orders of magnitude. Each block checks that on its own sites (kMeanBits,
// kProductBits) and takes binary64 sums where it does not hold: a few large
// sites among ordinary ones, a component that is small everywhere, large and
// tiny sites in turn.

struct Fix4 {
  int64_t v[4];
};

// d 2^(58-T) rounded to the nearest integer, ties away from zero; shift0 = T +
// 1027. A double is m 2^(e - 1086) with m its mantissa from bit 63 down, so the
// result is m >> (T + 1028 - e), taken with one more bit. (Ties are common just
// below the exact range, where a component loses a bit or two: about 1 % of
// components, so that their fixed direction adds some 2^-62 a site to M. On a
// grid of 54 bits half of the components had them, and M was 1e-14 off.)
__device__ __forceinline__ int64_t to_fixed(double d, int shift0) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint64_t m = ((uint64_t)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11);
  const uint32_t sh = (uint32_t)(shift0 - (int)((hi >> 20) & 0x7ffu));
  uint64_t x;
  asm("shr.b64 %0, %1, %2;" : "=l"(x) : "l"(m), "r"(sh));  // shifts past 63 give 0
  const int64_t s = (int32_t)hi >> 31;
  return ((int64_t)((x + 1u) >> 1) ^ s) - s;
}
__device__ __forceinline__ Fix4 to_fixed(const F4& f, int shift0) {
  return Fix4{{to_fixed(f.x, shift0), to_fixed(f.y, shift0), to_fixed(f.z, shift0), to_fixed(f.w, shift0)}};
}

// Whether d 2^(58-T) is no integer: the T + 1028 - e lowest bits of m (all of
// them from 64 on) are not all 0. A zero has no leading bit to lose.
__device__ __forceinline__ bool off_grid(double d, int shift0) {
  const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
  const uint64_t m = ((uint64_t)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (lo << 11);
  const int above = max(63 - shift0 + (int)((hi >> 20) & 0x7ffu), 0);
  uint64_t below;
  asm("shl.b64 %0, %1, %2;" : "=l"(below) : "l"(m), "r"(above));
  return below != 0u && ((hi << 1) | lo) != 0u;
}
// The components of f off the grid, counted in the bytes.
__device__ __forceinline__ uint32_t off_grid(const F4& f, int shift0) {
  return (off_grid(f.x, shift0) ? 1u : 0u) | (off_grid(f.y, shift0) ? 1u << 8 : 0u) |
         (off_grid(f.z, shift0) ? 1u << 16 : 0u) | (off_grid(f.w, shift0) ? 1u << 24 : 0u);
}

// The block's sums of v[0..4], in threads 0..4. The five values are reduced
// together: two of them share each of the first three exchange steps (a lane
// keeps one and passes the other on), so a warp takes 8 binary64 additions
// instead of 25 (this pipe bounds the kernels that end here).
__device__ __forceinline__ double block_sum5(const double v[5]) {
  __shared__ double red[5][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  auto pass = [&](double keep0, double keep1, int bit) {  // lanes with the bit keep the second value
    const bool up = (lane & bit) != 0;
    return (up ? keep1 : keep0) + __shfl_xor_sync(0xffffffffu, up ? keep0 : keep1, bit);
  };
  const double p = pass(v[0], v[1], 1), q = pass(v[2], v[3], 1), r = v[4] + __shfl_xor_sync(0xffffffffu, v[4], 1);
  const double pq = pass(p, q, 2), rr = r + __shfl_xor_sync(0xffffffffu, r, 2);
  double w = pass(pq, rr, 4);  // lane bits 2..0: 000 v0, 001 v1, 010 v2, 011 v3, 1xx v4
  w += __shfl_xor_sync(0xffffffffu, w, 8);
  w += __shfl_xor_sync(0xffffffffu, w, 16);
  if (lane < 5) red[lane][warp] = w;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 5)
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[threadIdx.x][k];
  return s;
}

// Adds site x's terms to the binary64 sums v.
__device__ __forceinline__ void observe_site(const F4* phi, uint32_t L, uint32_t x, double v[5]) {
  const Coords k = coords_of(x, L);
  const F4 f = phi[x];
  uint32_t stride = 1;
  for (int mu = 0; mu < 4; ++mu) {
    const F4 g = phi[nb(x, mu, k, L, stride)];
    v[0] += f.x * g.x + f.y * g.y + f.z * g.z + f.w * g.w;
    stride *= L;
  }
  v[1] += f.x;
  v[2] += f.y;
  v[3] += f.z;
  v[4] += f.w;
}

__global__ void phi4_observe_kernel(const F4* phi, int L, int64_t n, double* out /* E, M0..M3 */) {
  sw::start_next();
  sw::after_previous();
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
    observe_site(phi, (uint32_t)L, (uint32_t)x, v);
  const double s = block_sum5(v);
  if (threadIdx.x < 5) atomicAdd(out + threadIdx.x, s);
}

// The grid's sums of v[0..4] into out[0..4]: every block leaves its own in
// part[block][5], and the one that finds it is the last (*done counts them,
// and is 0 again afterwards) adds them up in a fixed order, the same in every
// run. With an addition into out for each of the 4096 blocks of L = 64 that sum
// rounded as often: E and M were 1.3e-15 to 2.6e-15 off there (rms of nine
// fields; the binary64 sums of 2432 blocks 0.8e-15 to 1.8e-15), 1.0e-16 to
// 1.3e-16 so.
__device__ __forceinline__ void grid_sum5(double v[5], double* part, uint32_t* done, double* out) {
  __shared__ bool s_last;
  const uint32_t b = blockIdx.y * gridDim.x + blockIdx.x, nb = gridDim.x * gridDim.y;
  double s = block_sum5(v);
  if (threadIdx.x < 5) __stcg(part + (size_t)5 * b + threadIdx.x, s);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == nb - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
#pragma unroll
  for (int c = 0; c < 5; ++c) v[c] = 0.0;
#pragma unroll 2
  for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x)
#pragma unroll
    for (int c = 0; c < 5; ++c) v[c] += __ldcg(part + (size_t)5 * i + c);
  s = block_sum5(v);  // (the barriers above lie between its two uses)
  if (threadIdx.x < 5) out[threadIdx.x] = s;
  if (threadIdx.x == 0) *done = 0u;
}

// A block takes kObserveThreads consecutive sites of the (x0, x1, x2) volume
// and marches `steps` slices up x3: a thread's next slice is the x3 neighbour
// of its current one, and the x0 and x1 neighbours are mostly other threads'
// sites, passed as integers in shared memory (two slices' buffers, so one
// barrier a slice). Only the x2 neighbour, and those past the block's range,
// are loaded and converted again: 2.25 conversions a site at L = 64.
constexpr int kObserveThreads = 256;
constexpr int kObserveSteps = 16;
// What a block's sites must show for its fixed-point sums to stand, in units
// of the grid (2^58 and 2^56 are 2^T and 2^2T there):
//   M_c  sum |phi_c| >= 2^kMeanBits for every component c that lost bits: the
//        half units lost add up to at most 2^-53 of that sum, half an ulp;
//   E    sum |phi . S| >= 2^kProductBits for every site, 2^-8 of the bound. A
//        site's phi . S is off by about 2^-59 of the bound, at random, so the
//        sum of a block by less than 2^-56 of the sum of |phi . S|; binary64
//        rounds the running sum 16 times a site.
// A field of directions (|phi| about 1) has 2^55 and 2^53, a Gaussian one of
// 2^24 sites 2^54 and 2^50.
constexpr int kMeanBits = 52, kProductBits = 48;
// From 2^20 sites the large bricks (4096 sites: fewer bonds leave them) and the
// merge with several rows a warp; below, one site a thread and small bricks, so
// that L = 16 still has 256 CTAs: 8 us against 20 with 8 x 4 x 4 x 4 bricks of
// 128 threads. E and M take the fixed-point kernel from there too: below, the
// binary64 kernel takes 10 us or less (L = 16), most of it latency, and the
// fixed-point one has too few blocks of sixteen slices.
constexpr int64_t kLargeSites = 1 << 20;

//
// PROJECT: the same pass takes the projections of the next update, which read
// the same field and are bound by the binary64 pipe while the sums are bound
// by integer issue: 303 us together, 222 + 156 apart (L = 64).
template <bool PROJECT>
__global__ void __launch_bounds__(kObserveThreads)
    phi4_observe_fixed_kernel(const F4* phi, int L, int64_t n, const uint32_t* top, int steps, double* part,
                              uint32_t* done, double* out, double* a, float* af, Dir d, uint32_t* next_top) {
  sw::start_next();
  sw::after_previous();
  uint32_t big = 0u;
  auto project = [&](const F4& f, size_t x) {
    const double v = proj(f, d);
    a[x] = v;
    af[x] = __double2float_rn(v);
    big = max(max(max(big, abs_high(f.x)), abs_high(f.y)), max(abs_high(f.z), abs_high(f.w)));
  };
  auto leave_top = [&] {
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0) atomicMax(next_top, big);
  };
  double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  const int et = (int)(*top >> 20);  // biased exponent of the largest component before the reflection
  if (et < 1023 - 400 || et > 1023 + 400) {
    // zero, subnormal, huge, infinite or NaN components: the binary64 sums
    const int64_t b = (int64_t)blockIdx.y * gridDim.x + blockIdx.x,
                  step = (int64_t)gridDim.x * gridDim.y * blockDim.x;
    for (int64_t x = b * blockDim.x + threadIdx.x; x < n; x += step) {
      observe_site(phi, (uint32_t)L, (uint32_t)x, v);
      if (PROJECT) project(phi[x], x);
    }
    if (PROJECT) leave_top();
    grid_sum5(v, part, done, out);
    return;
  }
  const int T = et - 1023 + 2;        // |phi| <= 2 max component < 2^T
  const int shift0 = T + 1027;
  __shared__ longlong2 s_x[2][2][kObserveThreads];
  __shared__ uint32_t s_chk[7];  // sums of |phi_c| and |phi . S| (2^-40), counts of components that lost bits
  if (threadIdx.x < 7) s_chk[threadIdx.x] = 0u;  // (the loop's barriers follow)
  const uint32_t V = (uint32_t)L * L * L, s0 = blockIdx.x * kObserveThreads, s = s0 + threadIdx.x;
  const bool have = s < V;
  const uint32_t sc = have ? s : V - 1;
  const Coords k = coords_of(sc, (uint32_t)L);
  const uint32_t n0 = nb(sc, 0, k, L, 1), n1 = nb(sc, 1, k, L, L), n2 = sc + (k.c[2] + 1 == (uint32_t)L ? L * L - V : L * L);
  const bool in0 = n0 - s0 < kObserveThreads, in1 = n1 - s0 < kObserveThreads;
  const int z0 = blockIdx.y * steps, z1 = min(z0 + steps, L);
  int64_t E = 0, m[4] = {0, 0, 0, 0};
  uint32_t am[4] = {0u, 0u, 0u, 0u}, ae = 0u, own_lost, up_lost, nlost = 0u;  // high words of |.|; counts by byte
  const F4 first = phi[(size_t)z0 * V + sc];
  if (PROJECT && have) project(first, (size_t)z0 * V + sc);
  Fix4 own = to_fixed(first, shift0);
  own_lost = off_grid(first, shift0);
  for (int z = z0; z < z1; ++z) {
    const F4* slice = phi + (size_t)z * V;
    const F4 fu = phi[(size_t)(z + 1 == L ? 0 : z + 1) * V + sc];
    if (PROJECT && have && z + 1 < z1) project(fu, (size_t)(z + 1) * V + sc);
    const Fix4 up = to_fixed(fu, shift0);
    up_lost = off_grid(fu, shift0);
    const F4 g2 = slice[n2];
    longlong2(&buf)[2][kObserveThreads] = s_x[z & 1];
    buf[0][threadIdx.x] = make_longlong2(own.v[0], own.v[1]);
    buf[1][threadIdx.x] = make_longlong2(own.v[2], own.v[3]);
    Fix4 S = to_fixed(g2, shift0);
#pragma unroll
    for (int c = 0; c < 4; ++c) S.v[c] += up.v[c];
    __syncthreads();
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const uint32_t nbr = d ? n1 : n0;
      Fix4 g;
      if (d ? in1 : in0) {
        const longlong2 u = buf[0][nbr - s0], w = buf[1][nbr - s0];
        g = Fix4{{u.x, u.y, w.x, w.y}};
      } else {
        g = to_fixed(slice[nbr], shift0);
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) S.v[c] += g.v[c];
    }
    int64_t hh = 0, cr = 0, ll = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int xh = (int)(own.v[c] >> 30), Sh = (int)(S.v[c] >> 30);
      const int xl = (int)own.v[c] & 0x3fffffff, Sl = (int)S.v[c] & 0x3fffffff;
      hh += (int64_t)xh * Sh;
      cr += (int64_t)xh * Sl + (int64_t)xl * Sh;
      ll += (int64_t)xl * Sl;
      m[c] += own.v[c];
      am[c] += (uint32_t)abs((int)(own.v[c] >> 32));
    }
    // phi . S = hh 2^60 + cr 2^30 + ll, to the nearest multiple of 2^60
    const int64_t e = hh + ((cr + (ll >> 30) + (1 << 29)) >> 30);
    E += e;
    ae += (uint32_t)abs((int)(e >> 32));
    nlost += own_lost;
    own = up;
    own_lost = up_lost;
  }
  {
    const uint32_t w[7] = {am[0] >> 8, am[1] >> 8, am[2] >> 8, am[3] >> 8,
                           ae >> 8,    nlost & 0x00ff00ffu, (nlost >> 8) & 0x00ff00ffu};
#pragma unroll
    for (int c = 0; c < 7; ++c) {
      const uint32_t sum = __reduce_add_sync(0xffffffffu, have ? w[c] : 0u);
      if ((threadIdx.x & 31) == 0) atomicAdd(&s_chk[c], sum);
    }
  }
  __syncthreads();
  const uint32_t sites = min((uint32_t)kObserveThreads, V - s0) * (uint32_t)(z1 - z0);
  const bool fixed = s_chk[4] >= sites << (kProductBits - 40) &&
                     s_chk[0] >= (s_chk[5] & 0xffffu) << (kMeanBits - 40) &&
                     s_chk[1] >= (s_chk[6] & 0xffffu) << (kMeanBits - 40) &&
                     s_chk[2] >= (s_chk[5] >> 16) << (kMeanBits - 40) &&
                     s_chk[3] >= (s_chk[6] >> 16) << (kMeanBits - 40);  // the same in every thread
  if (have && fixed) {
    v[0] = (double)E * scalbn(1.0, 2 * T - 56);
    const double u = scalbn(1.0, T - 58);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[1 + c] = (double)m[c] * u;
  } else if (have) {
    for (int z = z0; z < z1; ++z) observe_site(phi, (uint32_t)L, (uint32_t)z * V + s, v);
  }
  if (PROJECT) leave_top();
  grid_sum5(v, part, done, out);
}

int grid_of(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152LL * 16) g = 152LL * 16;
  return (int)(g < 1 ? 1 : g);
}

thread_local char g_msg[256];

int ffail(int code, const char* what) { return sw::record_error(code, what); }

double unit_interval_host(uint32_t w) { return ((double)w + 0.5) * 0x1p-31 - 1.0; }

}  // namespace

struct sw_phi4 {
  int L = 0;
  int64_t n = 0;
  double kappa = 0.0;
  uint64_t seed = 0;
  sw::KeySchedule ks{};
  int64_t t = 0, t_base = 0, cap = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  F4* phi = nullptr;
  double* a = nullptr;
  float* af = nullptr;  // the projections rounded to binary32 (the bond kernel's first test)
  int* par = nullptr;
  uint8_t* bonds = nullptr;
  double* obs = nullptr;  // [cap][5]: E, M0..M3
  uint32_t* top = nullptr;  // [2], by update parity: high word of the field's largest |component| (projection -> E and M)
  double* part = nullptr;   // large lattices: the blocks' E and M, [blocks][5]
  uint32_t* done = nullptr;  // and the count of those that are in
  int* err = nullptr;
  sw::ReadBack read;
};

namespace {

#define F_CUDA(call, what)                                                          \
  do {                                                                              \
    cudaError_t e_ = (call);                                                        \
    if (e_ != cudaSuccess) {                                                        \
      snprintf(g_msg, sizeof g_msg, "%s: %s", what, cudaGetErrorString(e_));        \
      return ffail(e_ == cudaErrorMemoryAllocation ? SW_ENOMEM : SW_ECUDA, g_msg); \
    }                                                                               \
  } while (0)

void free_phi4(sw_phi4* h) {
  void* ptrs[] = {h->phi, h->a, h->af, h->par, h->bonds, h->obs, h->top, h->part, h->done, h->err};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
}

// As sync_and_check of an Ising lattice.
int check_phi4(sw_phi4* h, const void* src = nullptr, size_t words = 0, void* out = nullptr) {
  int flag = 0;
  F_CUDA(h->read(h->stream, h->err, src, words, &flag, out), "stream synchronize and read");
  if (flag == 1) return ffail(SW_ETIMEOUT, "a capped union-find loop gave up");
  if (flag != 0) return ffail(SW_EDEVICE, "device error flag set");
  return SW_OK;
}

int grow(sw_phi4* h, int64_t need) {
  if (need <= h->cap) return SW_OK;
  int64_t ncap = h->cap ? h->cap : 1024;
  while (ncap < need) ncap *= 2;
  double* obs = nullptr;
  F_CUDA(cudaMalloc(&obs, (size_t)ncap * 5 * sizeof(double)), "trace growth");
  if (h->cap) {
    cudaError_t e = cudaMemcpyAsync(obs, h->obs, (size_t)h->cap * 5 * sizeof(double), cudaMemcpyDeviceToDevice,
                                    h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) {
      cudaFree(obs);
      F_CUDA(e, "trace growth");
    }
    cudaFree(h->obs);
  }
  h->obs = obs;
  h->cap = ncap;
  return SW_OK;
}

// O3 on the host: the first attempt k with 2^-20 < |v|^2 <= 1.
int direction(uint64_t seed, uint32_t t, Dir& d) {
  const sw::KeySchedule ks = sw::make_key_schedule(seed);
  for (uint32_t k = 0; k < 1000; ++k) {
    const uint4 w = sw::philox4x32_10(make_uint4(k, t, 5u, 0u), ks);
    const double v[4] = {unit_interval_host(w.x), unit_interval_host(w.y), unit_interval_host(w.z),
                         unit_interval_host(w.w)};
    const double s = std::fma(v[3], v[3], std::fma(v[2], v[2], std::fma(v[1], v[1], v[0] * v[0])));
    if (s <= 1.0 && s > 0x1p-20) {
      const double nrm = std::sqrt(s);
      for (int a = 0; a < 4; ++a) {
        d.r[a] = v[a] / nrm;
        d.m2r[a] = -2.0 * d.r[a];
      }
      return 0;
    }
  }
  return -1;
}

template <int B0, int B1, int B2, int B3, int NT>
void launch_brick(sw_phi4* h) {
  const int L = h->L;
  const double k4 = 4.0 * h->kappa;
  // (k4 f) f stays in binary32's normal range, or vanishes, for |f| >= 2^-60
  // unless k4 is below 2^-66: with NaN every edge takes the binary64 test.
  // (Taken on the host: every thread's binary64 comparisons cost 2 us an update
  // at L = 64.)
  const float k4f = k4 == 0.0 || k4 >= 0x1p-66 ? (float)k4 : std::numeric_limits<float>::quiet_NaN();
  const unsigned g = (unsigned)((L + B0 - 1) / B0) * ((L + B1 - 1) / B1) * ((L + B2 - 1) / B2) * ((L + B3 - 1) / B3);
  sw::launch_after(phi4_brick_kernel<B0, B1, B2, B3, NT>, g, NT, 0, h->stream, h->a, h->af, h->bonds, h->par, L,
                   k4, k4f, (uint32_t)h->t, h->ks, h->err);
}

template <int UNITE_ROWS, int ROOT_ROWS>
void launch_merge(sw_phi4* h) {
  const int64_t u = 32 * kUniteWarps * UNITE_ROWS, r = 32 * kRootWarps * ROOT_ROWS;
  sw::launch_after(phi4_unite_kernel<UNITE_ROWS>, (unsigned)((h->n + u - 1) / u), 32 * kUniteWarps, 0, h->stream,
                   h->bonds, h->par, h->L, h->n, h->err);
  sw::launch_after(phi4_roots_kernel<ROOT_ROWS>, (unsigned)((h->n + r - 1) / r), 32 * kRootWarps, 0, h->stream,
                   h->bonds, h->par, h->n, (uint32_t)h->t, h->ks, h->err);
}

dim3 observe_grid(int L) {
  return dim3((unsigned)(((int64_t)L * L * L + kObserveThreads - 1) / kObserveThreads),
              (unsigned)((L + kObserveSteps - 1) / kObserveSteps));
}

// The direction of update t and, on large lattices, its cleared range word.
int begin_update(sw_phi4* h, int64_t t, Dir& d) {
  if (direction(h->seed, (uint32_t)t, d) != 0) return ffail(SW_EDEVICE, "no direction found");
  if (h->n >= kLargeSites) F_CUDA(cudaMemsetAsync(h->top + (t & 1), 0, sizeof(uint32_t), h->stream), "range word");
  return SW_OK;
}

// Projections of update t on direction d.
void project(sw_phi4* h, const Dir& d) {
  sw::launch_after(phi4_project_kernel, grid_of(h->n), 256, 0, h->stream, h->phi, h->a, h->af, h->n, d,
                   h->n >= kLargeSites ? h->top + (h->t & 1) : nullptr);
}

// Bonds, clusters and flips of update t from its projections.
int clusters(sw_phi4* h) {
  if (h->n >= kLargeSites) {
    launch_brick<16, 8, 8, 4, 1024>(h);
    launch_merge<8, 4>(h);
  } else {
    launch_brick<8, 4, 4, 2, 256>(h);
    launch_merge<1, 1>(h);
  }
  F_CUDA(cudaGetLastError(), "phi4 update launch");
  return SW_OK;
}

}  // namespace

extern "C" {

int sw_phi4_direction(uint64_t seed, uint32_t t, double* r_out) {
  if (!r_out) return ffail(SW_EINVAL, "NULL argument");
  Dir d;
  if (direction(seed, t, d) != 0) return ffail(SW_EDEVICE, "no direction found");
  for (int a = 0; a < 4; ++a) r_out[a] = d.r[a];
  return SW_OK;
}

int sw_phi4_create(int32_t L, double kappa, uint64_t seed, int32_t init, void* stream, sw_phi4** out) {
  if (!out) return ffail(SW_EINVAL, "out is NULL");
  *out = nullptr;
  if (L < 2 || (int64_t)L * L * L * L >= ((int64_t)1 << 31)) return ffail(SW_EINVAL, "L outside 2 <= L, L^4 < 2^31");
  if (!(kappa >= 0.0) || std::isinf(kappa)) return ffail(SW_EINVAL, "kappa must be finite and >= 0");
  if (init != SW_INIT_HOT && init != SW_INIT_COLD) return ffail(SW_EINVAL, "init must be SW_INIT_HOT or SW_INIT_COLD");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
    cudaGetLastError();
    return ffail(SW_ECUDA, "no CUDA device available (libsw has no CPU fallback)");
  }
  sw_phi4* h = new (std::nothrow) sw_phi4();
  if (!h) return ffail(SW_ENOMEM, "host allocation failed");
  h->L = L;
  h->n = (int64_t)L * L * L * L;
  h->kappa = kappa;
  h->seed = seed;
  h->ks = sw::make_key_schedule(seed);
  const size_t n = (size_t)h->n;
  cudaError_t e = cudaSuccess;
  if (stream) {
    h->stream = (cudaStream_t)stream;
  } else {
    e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
    h->own_stream = e == cudaSuccess;
  }
  if (e == cudaSuccess) e = cudaMalloc(&h->phi, n * sizeof(F4));
  if (e == cudaSuccess) e = cudaMalloc(&h->a, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&h->af, n * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&h->par, n * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&h->bonds, n);
  if (e == cudaSuccess) e = cudaMalloc(&h->top, 2 * sizeof(uint32_t));
  if (e == cudaSuccess && h->n >= kLargeSites) {
    const dim3 g = observe_grid(L);
    e = cudaMalloc(&h->part, (size_t)g.x * g.y * 5 * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc(&h->done, sizeof(uint32_t));
    if (e == cudaSuccess) e = cudaMemsetAsync(h->done, 0, sizeof(uint32_t), h->stream);
  }
  if (e == cudaSuccess) e = cudaMalloc(&h->err, sizeof(int));
  if (e == cudaSuccess) e = cudaMemsetAsync(h->err, 0, sizeof(int), h->stream);
  if (e == cudaSuccess) {
    phi4_init_kernel<<<grid_of(h->n), 256, 0, h->stream>>>(h->phi, h->n, h->ks, init == SW_INIT_COLD);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    snprintf(g_msg, sizeof g_msg, "sw_phi4_create: %s", cudaGetErrorString(e));
    free_phi4(h);
    delete h;
    return ffail(e == cudaErrorMemoryAllocation ? SW_ENOMEM : SW_ECUDA, g_msg);
  }
  const int rc = grow(h, 1024);
  if (rc != SW_OK) {
    free_phi4(h);
    delete h;
    return rc;
  }
  *out = h;
  return SW_OK;
}

int sw_phi4_sweep(sw_phi4* h, int32_t n) {
  if (!h) return ffail(SW_EINVAL, "handle is NULL");
  if (n < 0) return ffail(SW_EINVAL, "n must be >= 0");
  int rc = grow(h, h->t - h->t_base + n);
  if (rc != SW_OK) return rc;
  if (n == 0) return SW_OK;
  const int g = grid_of(h->n), L = h->L;
  const bool large = h->n >= kLargeSites;
  const dim3 og = observe_grid(L);
  Dir d, next{};
  rc = begin_update(h, h->t, d);
  if (rc != SW_OK) return rc;
  F_CUDA(cudaMemsetAsync(h->obs + 5 * (h->t - h->t_base), 0, (size_t)n * 5 * sizeof(double), h->stream), "trace rows");
  project(h, d);
  for (int32_t k = 0; k < n; ++k) {
    rc = clusters(h);
    if (rc != SW_OK) return rc;
    double* o = h->obs + 5 * (h->t - h->t_base);
    uint32_t* const top = h->top + (h->t & 1);
    sw::launch_after(phi4_reflect_kernel, g, 256, 0, h->stream, h->phi, h->a, h->par, h->n, d);
    // E and M, with the next update's projections unless the call ends here
    // (the caller may change the field before the next one)
    const bool more = k + 1 < n;
    if (more) {
      rc = begin_update(h, h->t + 1, next);
      if (rc != SW_OK) return rc;
    }
    if (large && more)
      sw::launch_after(phi4_observe_fixed_kernel<true>, og, kObserveThreads, 0, h->stream, h->phi, L, h->n, top,
                       kObserveSteps, h->part, h->done, o, h->a, h->af, next, h->top + ((h->t + 1) & 1));
    else if (large)
      sw::launch_after(phi4_observe_fixed_kernel<false>, og, kObserveThreads, 0, h->stream, h->phi, L, h->n, top,
                       kObserveSteps, h->part, h->done, o, nullptr, nullptr, d, nullptr);
    else
      sw::launch_after(phi4_observe_kernel, g, 256, 0, h->stream, h->phi, L, h->n, o);
    F_CUDA(cudaGetLastError(), "phi4 reflect launch");
    h->t += 1;
    if (more && !large) project(h, next);
    d = next;
  }
  return SW_OK;
}

int sw_phi4_observables(sw_phi4* h, int64_t first, int64_t count, double* E_host, double* M_host) {
  if (!h) return ffail(SW_EINVAL, "handle is NULL");
  if (count < 0 || first < h->t_base || first + count > h->t) return ffail(SW_EINVAL, "update range outside the trace");
  double* buf = count ? (double*)malloc((size_t)count * 5 * sizeof(double)) : nullptr;
  if (count && !buf) return ffail(SW_ENOMEM, "host allocation failed");
  const int rc = check_phi4(h, h->obs + 5 * (first - h->t_base), (size_t)count * 5, buf);
  for (int64_t k = 0; rc == SW_OK && k < count; ++k) {
    if (E_host) E_host[k] = buf[5 * k];
    if (M_host)
      for (int a = 0; a < 4; ++a) M_host[4 * k + a] = buf[5 * k + 1 + a];
  }
  free(buf);
  return rc;
}

int sw_phi4_field(sw_phi4* h, double* out, int32_t out_is_device) {
  if (!h || !out) return ffail(SW_EINVAL, "NULL argument");
  F_CUDA(cudaMemcpyAsync(out, h->phi, (size_t)h->n * sizeof(F4),
                         out_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, h->stream),
         "field copy");
  if (out_is_device) return SW_OK;
  return check_phi4(h);
}

int sw_phi4_set_field(sw_phi4* h, const double* in, uint32_t t, int32_t in_is_device) {
  if (!h || !in) return ffail(SW_EINVAL, "NULL argument");
  int rc = check_phi4(h);
  if (rc != SW_OK) return rc;
  F_CUDA(cudaMemcpyAsync(h->phi, in, (size_t)h->n * sizeof(F4),
                         in_is_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, h->stream),
         "field copy");
  rc = check_phi4(h);
  if (rc != SW_OK) return rc;
  h->t = t;
  h->t_base = t;
  return SW_OK;
}

int sw_phi4_labels(sw_phi4* h, int32_t* out, int32_t out_is_device) {
  if (!h || !out) return ffail(SW_EINVAL, "NULL argument");
  Dir d;
  int rc = begin_update(h, h->t, d);
  if (rc != SW_OK) return rc;
  project(h, d);
  rc = clusters(h);
  if (rc != SW_OK) return rc;
  // host labels pass through the projections' buffer (8 bytes a site), done with here
  int32_t* const dst = out_is_device ? out : reinterpret_cast<int32_t*>(h->a);
  F_CUDA(sw::launch_after(phi4_labels_kernel, grid_of(h->n), 256, 0, h->stream, h->par, dst, h->n),
         "phi4 labels launch");
  if (out_is_device) return SW_OK;
  F_CUDA(cudaMemcpyAsync(out, dst, (size_t)h->n * sizeof(int32_t), cudaMemcpyDeviceToHost, h->stream), "labels copy");
  return check_phi4(h);
}

int sw_phi4_get_sweep(sw_phi4* h, uint32_t* t_out) {
  if (!h || !t_out) return ffail(SW_EINVAL, "NULL argument");
  *t_out = (uint32_t)h->t;
  return SW_OK;
}

int sw_phi4_destroy(sw_phi4* h) {
  if (!h) return SW_OK;
  if (h->stream) cudaStreamSynchronize(h->stream);
  free_phi4(h);
  delete h;
  return SW_OK;
}

}  // extern "C"
