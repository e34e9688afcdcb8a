// sw_small.cu -- whole sweeps of a small lattice in one CTA.
//
// A lattice of at most 256 x 256 sites would fit one CTA's shared memory whole
// (spins and bonds as bit masks, and a 16-bit label per site); the launchers
// take sides up to kSmallMaxL, past which the tiles are faster. One launch runs
// n sweeps back to back with block barriers between the steps, so a small
// lattice costs no cross-tile merge and no launch per phase. The steps and
// their results are those of the tiled path:
//   draws (C5)        a Philox block per pair of consecutive site indices,
//                     straight through the lattice (pairs straddle rows of
//                     an odd side), into flat bit strings;
//   bonds (§2.1)      a thread per row word, which shifts its draws out of
//                     the strings; E and M (C10) of the state fall out of the
//                     same words, so they are summed here, one sweep late;
//   clusters (§2.3)   a warp per segment (a 32-column band of a few rows): a
//                     Hoshen-Kopelman scan down the segment (row_masks)
//                     labels its runs, a warp-private union-find joins the
//                     runs that meet, and the bonds out of the segment (east,
//                     south, the periodic wraps) are united across warps by
//                     compare-and-swap; the larger root is hung under the
//                     smaller, so every root is its cluster's smallest site;
//   new spins (§2.4)  a lane per site walks its label to the root, four rows
//                     at a time, and takes the root's flip bit (C6; the bits
//                     of all site indices are filled from their blocks) or
//                     the fresh spin drawn for it (C6b).
// Spins are read at the start and written back after the last sweep.
//
// What bounds it: one SM. Up to about L = 64 a sweep is a chain of four
// barriers with dependent shared-memory loads between them, so the work is
// cut into 32 segments (one a warp) rather than into few tall ones; above,
// the instructions of the Philox blocks and of the scan. Cycles of a sweep at
// L = 64 (18.6 k): draws 2.4 k, bonds 0.6 k, scan 2.0 k, unions inside a
// segment 3.0 k, across segments 4.6 k, walks and new spins 5.4 k. Measured
// and not kept: half the warps drawing the next sweep's blocks while the
// others label (9.3 us against 9.0 at L = 64, 27 against 21 at 144), and
// pointing every label at its root before the sites look (10.9 from work
// lists, 9.7 in step).
#include <cuda_runtime.h>
#include <stdint.h>

#include "sw_band.cuh"
#include "sw_internal.h"
#include "sw_philox.cuh"

namespace sw {
namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSmallUnionCap = 1 << 20;
constexpr int kSmallMinRows = 4;    // rows of a segment at least
constexpr int kSmallListCap = 128;  // entries of a warp's work list

// Sizes of a lattice's pieces in shared memory.
struct SmallShape {
  int N, WPL, RWN, DW;   // sites, words a row, row words, flat words
  int S, nseg;           // rows of a segment, segments
  __host__ __device__ explicit SmallShape(int L) {
    N = L * L;
    WPL = (L + 31) >> 5;
    RWN = L * WPL;
    DW = (N + 31) >> 5;
    // as many segments a warp as keep a segment within 32 rows (a lane holds
    // a row's masks), the rows spread evenly over them
    for (int per_warp = 1;; ++per_warp) {
      const int bands = per_warp * (kSmallThreads / 32) / WPL;
      S = (L + bands - 1) / bands;
      if (S <= 32) break;
    }
    if (S < kSmallMinRows) S = kSmallMinRows;
    nseg = WPL * ((L + S - 1) / S);
  }
};

// The draws of sweep t by the whole block: the C5 bits by site index into rawE / rawS, lane p taking the block of sites 2p and 2p + 1
// (four lanes' bits make a byte of each string), and under the flip rule the
// C6 bits of all site indices into dec (word k of it is word k & 3 of block
// k >> 2).
__device__ __forceinline__ void small_draws(const SmallArgs& a, int N, int DW, uint32_t t, uint32_t* rawE,
                                            uint32_t* rawS, uint32_t* dec) {
  constexpr int nw = kSmallThreads / 32;
  const int lane = threadIdx.x & 31, i = threadIdx.x >> 5;
  const int np = (((N + 1) >> 1) + 3) & ~3;
  uint8_t* rawE8 = reinterpret_cast<uint8_t*>(rawE);
  uint8_t* rawS8 = reinterpret_cast<uint8_t*>(rawS);
  for (int p0 = 32 * i; p0 < np; p0 += 32 * nw) {
    const int p = p0 + lane, sh = 2 * (p & 3);
    const uint4 q = philox4x32_10(make_uint4((uint32_t)p, t, 0u, 0u), a.ks);
    uint32_t v = (((uint32_t)(q.x < a.thr) | ((uint32_t)(q.z < a.thr) << 1)) << sh) |
                 (((uint32_t)(q.y < a.thr) | ((uint32_t)(q.w < a.thr) << 1)) << (8 + sh));
    v |= __shfl_xor_sync(0xffffffffu, v, 1);
    v |= __shfl_xor_sync(0xffffffffu, v, 2);
    if ((lane & 3) == 0 && p < np) {
      rawE8[p >> 2] = (uint8_t)v;
      rawS8[p >> 2] = (uint8_t)(v >> 8);
    }
  }
  if (a.rule == 0) {
    for (int b = 32 * (nw - 1 - i) + lane; 4 * b < DW; b += 32 * nw) {
      const uint4 q = philox4x32_10(make_uint4((uint32_t)b, t, 1u, 0u), a.ks);
      dec[4 * b] = q.x;
      if (4 * b + 1 < DW) dec[4 * b + 1] = q.y;
      if (4 * b + 2 < DW) dec[4 * b + 2] = q.z;
      if (4 * b + 3 < DW) dec[4 * b + 3] = q.w;
    }
  }
}

// The n sweeps of one lattice by the whole CTA (smem: small_smem_bytes(L)).
__device__ __forceinline__ void small_body(const SmallArgs& a, uint32_t* smem) {
  constexpr int NT = kSmallThreads, NW = NT / 32;
  __shared__ uint16_t s_list[NW][kSmallListCap];  // a warp's unions, its labels, roots waiting for their draw
  __shared__ int s_em[2];
  const SmallShape Z(a.L);
  const int L = a.L, N = Z.N, WPL = Z.WPL, RWN = Z.RWN, DW = Z.DW;
  uint32_t* s_spin = smem;        // [RWN] sign bits (1 = -1)
  uint32_t* s_e = s_spin + RWN;   // [RWN] east bonds
  uint32_t* s_s = s_e + RWN;      // [RWN] south bonds
  uint32_t* s_new = s_s + RWN;    // [RWN] sites that name a label of their own
  uint32_t* s_dec = s_new + RWN;  // [2][DW] decision bit of every root, by sweep parity
  uint32_t* rawE = s_dec + 2 * DW;   // [DW + 1] draws by site index, east
  uint32_t* rawS = rawE + DW + 1;    // [DW + 1] south
  uint16_t* par = reinterpret_cast<uint16_t*>(rawS + DW + 1);  // [N] labels; a label's entry is its parent
  volatile uint16_t* vpar = par;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool flip_rule = a.rule == 0;
  // this thread's first row word, and the step to its next
  const int ry0 = tid / WPL, rw0 = tid - ry0 * WPL, rdy = NT / WPL, rdw = NT - rdy * WPL;
  // this warp's first segment (band sw0, rows from sj0 * S on), and the step to its next
  const int sj0 = warp / WPL, sw0 = warp - sj0 * WPL, sdj = NW / WPL, sdw = NW - sdj * WPL;

  for (int rw = warp; rw < RWN; rw += NW) {
    const int y = rw / WPL, x = (rw % WPL) * 32 + lane;
    const bool minus = x < L && a.spins[(size_t)y * L + x] < 0;
    const uint32_t m = __ballot_sync(0xffffffffu, minus);
    if (lane == 0) s_spin[rw] = m;
  }
  if (tid < 2) s_em[tid] = 0;
  for (int k = 0;; ++k) {
    const uint32_t t = a.t0 + (uint32_t)k;
    uint32_t* dec = s_dec + (k & 1) * DW;  // (the sweep before's may still be read)
    if (k < a.n) small_draws(a, N, DW, t, rawE, rawS, dec);
    __syncthreads();

    // ---- E and M (C10) of the state, that of the sweep before, and the bonds
    // (§2.1) of this sweep
    for (int rw = tid, y = ry0, w = rw0, r0 = tid & ~31; r0 < RWN; r0 += NT, rw += NT) {
      int e = 0, m = 0;
      if (rw < RWN) {
        const int nb = min(32, L - 32 * w);
        const uint32_t vm = 0xffffffffu >> (32 - nb);
        const uint32_t sp = s_spin[rw];
        // east neighbours: the next site in the word; the word's last site
        // meets the next word's first, or column 0 of its row (periodic)
        const uint32_t nxt = s_spin[w + 1 < WPL ? rw + 1 : y * WPL];
        const uint32_t dE = (sp ^ (((sp >> 1) & (vm >> 1)) | ((nxt & 1u) << (nb - 1)))) & vm;
        const uint32_t dS = (sp ^ s_spin[y + 1 == L ? w : rw + WPL]) & vm;
        e = 2 * (__popc(dE) + __popc(dS)) - 2 * nb;
        m = nb - 2 * __popc(sp & vm);
        const int i0 = y * L + 32 * w, q = i0 >> 5, o = i0 & 31;
        s_e[rw] = __funnelshift_r(rawE[q], rawE[q + 1], o) & ~dE & vm;
        s_s[rw] = __funnelshift_r(rawS[q], rawS[q + 1], o) & ~dS & vm;
      }
      e = __reduce_add_sync(0xffffffffu, e);
      m = __reduce_add_sync(0xffffffffu, m);
      if (lane == 0) {
        atomicAdd(&s_em[0], e);
        atomicAdd(&s_em[1], m);
      }
      y += rdy;
      w += rdw;
      if (w >= WPL) {
        w -= WPL;
        ++y;
      }
    }
    if (!flip_rule)
      for (int i = tid; i < DW; i += NT) dec[i] = 0u;
    __syncthreads();
    if (tid < 2) {
      if (k > 0) a.em[2 * (k - 1) + tid] = s_em[tid];
      s_em[tid] = 0;
    }
    if (k == a.n) break;

    // ---- clusters (§2.3) inside each segment: lane l holds the masks of
    // the segment's row l; the warp scans the rows top to bottom, lane l
    // holding column l (see phase 1 of the tiled path)
    uint16_t* list = s_list[warp];
    for (int seg = warp, j = sj0, w = sw0; seg < Z.nseg; seg += NW) {
      const int y0 = j * Z.S, n = min(Z.S, L - y0), nb = min(32, L - 32 * w);
      const int org = y0 * L + 32 * w;  // the segment's first site
      const uint32_t vm = 0xffffffffu >> (32 - nb);
      RowMasks m{0u, 0u, 0u, 0u};
      if (lane < n) {
        const int rw = (y0 + lane) * WPL + w;
        const bool up = lane > 0;
        m = row_masks(s_e[rw] & (vm >> 1), vm, up ? s_e[rw - WPL] & (vm >> 1) : 0u, up ? vm : 0u,
                      up ? s_s[rw - WPL] : 0u);
        s_new[rw] = m.S & ~m.F;
      }
      {
        const uint32_t le = 0xffffffffu >> (31 - lane);
        uint32_t lab = 0u;
        int own = org + lane;
#pragma unroll 4
        for (int r = 0; r < n; ++r) {
          const uint32_t R = __shfl_sync(0xffffffffu, m.R, r);
          const uint32_t S = __shfl_sync(0xffffffffu, m.S, r);
          const uint32_t F = __shfl_sync(0xffffffffu, m.F, r);
          const int s = 31 - __clz(R & le);
          const int src = __ffs(S & (0xffffffffu << s)) - 1;
          const uint32_t v = ((F >> lane) & 1u) ? lab : (uint32_t)own;
          lab = __shfl_sync(0xffffffffu, v, src & 31);
          if (lane < nb) par[own] = (uint16_t)lab;
          own += L;
        }
      }
      __syncwarp();
      // the unions M asks for, from a list, one state machine a lane. Only
      // this warp touches the segment's labels, so a link is a plain store
      // checked after __syncwarp.
      const int cnt = __popc(m.M), first = warp_exclusive_sum(cnt, lane);
      const int total = __shfl_sync(0xffffffffu, first + cnt, 31);
      for (int r0 = 0; r0 < total; r0 += kSmallListCap) {
        int idx = first;
        for (uint32_t mm = m.M; mm; mm &= mm - 1, ++idx)
          if (idx >= r0 && idx < r0 + kSmallListCap) list[idx - r0] = (uint16_t)(org + lane * L + __ffs(mm) - 1);
        __syncwarp();
        const int nu = min(kSmallListCap, total - r0);
        int q = lane, xa = 0, xb = 0;
        bool busy = false;
        for (int it = 0;; ++it) {
          if (!busy && q < nu) {
            xb = list[q];
            xa = xb - L;
            q += 32;
            busy = true;
          }
          if (!__any_sync(0xffffffffu, busy)) break;
          if (it >= kSmallUnionCap) {
            if (busy) atomicCAS(a.err, 0, kErrUnionCap);
            break;
          }
          int hi = -1, lo = 0;
          if (busy) {
            const int pa = vpar[xa], pb = vpar[xb];
            if (pa == xa && pb == xb) {
              if (xa == xb) {
                busy = false;
              } else {
                hi = max(xa, xb);
                lo = min(xa, xb);
                vpar[hi] = (uint16_t)lo;
              }
            } else {
              const int ga = vpar[pa], gb = vpar[pb];
              if (ga != pa) vpar[xa] = (uint16_t)ga;
              if (gb != pb) vpar[xb] = (uint16_t)gb;
              xa = ga;
              xb = gb;
            }
          }
          __syncwarp();
          if (hi >= 0) {
            const int now = vpar[hi];
            busy = now != lo;
            xa = now;
            xb = lo;
          }
        }
        __syncwarp();
      }
      j += sdj;
      w += sdw;
      if (w >= WPL) {
        w -= WPL;
        ++j;
      }
    }
    __syncthreads();

    // ---- the bonds out of each segment, united by compare-and-swap: lane l
    // has the south bond of column l of its last row (unless the one left of
    // it joins the same two runs), then the east bond out of its row l
    // (unless the row above has one and both ends hang on it). The lanes
    // walk to their roots first, and lanes with the same pair of roots leave
    // it to the lowest of them: most bonds join the same few clusters.
    for (int seg = warp, j = sj0, w = sw0; seg < Z.nseg; seg += NW) {
      const int y0 = j * Z.S, n = min(Z.S, L - y0), nb = min(32, L - 32 * w);
      const uint32_t vm = 0xffffffffu >> (32 - nb), lastb = 1u << (nb - 1);
      const int yl = y0 + n - 1, yn = yl + 1 == L ? 0 : yl + 1, wn = w + 1 < WPL ? w + 1 : 0;
      const uint32_t d = s_s[yl * WPL + w];
      const uint32_t need = d & ~((d & s_e[yl * WPL + w] & s_e[yn * WPL + w] & (vm >> 1)) << 1);
      bool east = false;
      if (lane < n) {
        const int rw = (y0 + lane) * WPL + w, rn = (y0 + lane) * WPL + wn;
        east = (s_e[rw] & lastb) != 0u;
        if (lane > 0 && (s_e[rw - WPL] & s_s[rw - WPL] & lastb) && (s_s[rn - WPL] & 1u)) east = false;
      }
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        bool busy = pass == 0 ? ((need >> lane) & 1u) != 0u : east;
        int xa = 0, xb = 0;
        if (busy) {
          xa = vpar[pass == 0 ? yl * L + 32 * w + lane : (y0 + lane) * L + 32 * w + nb - 1];
          xb = vpar[pass == 0 ? yn * L + 32 * w + lane : (y0 + lane) * L + 32 * wn];
        }
        for (bool more = true; __any_sync(0xffffffffu, more);) {
          const int pa = vpar[xa], pb = vpar[xb];
          more = busy && (pa != xa || pb != xb);
          xa = pa;
          xb = pb;
        }
        busy = busy && xa != xb;
        {
          const uint32_t key = busy ? (uint32_t)(xa > xb ? xa << 16 | xb : xb << 16 | xa) : 0u;
          const uint32_t peers = __match_any_sync(0xffffffffu, key);
          busy = busy && lane == __ffs(peers) - 1;
        }
        for (int it = 0; __any_sync(0xffffffffu, busy); ++it) {
          if (it >= kSmallUnionCap) {
            if (busy) atomicCAS(a.err, 0, kErrUnionCap);
            break;
          }
          if (busy) {
            const int pa = vpar[xa], pb = vpar[xb];
            if (pa == xa && pb == xb) {
              if (xa == xb) {
                busy = false;
              } else {
                const int hi = max(xa, xb), lo = min(xa, xb);
                const int old = (int)atomicCAS(par + hi, (uint16_t)hi, (uint16_t)lo);
                busy = old != hi;
                xa = old;  // on failure: the root's new parent
                xb = lo;
              }
            } else {
              const int ga = vpar[pa], gb = vpar[pb];
              if (ga != pa) vpar[xa] = (uint16_t)ga;
              if (gb != pb) vpar[xb] = (uint16_t)gb;
              xa = ga;
              xb = gb;
            }
          }
        }
      }
      j += sdj;
      w += sdw;
      if (w >= WPL) {
        w -= WPL;
        ++j;
      }
    }
    __syncthreads();

    // ---- assignment rule (C6b): the roots are queued per warp and drawn 32
    // at a time so that every lane draws
    if (!flip_rule) {
      int qh = 0, qn = 0;  // the same in every lane of the warp
      auto draw = [&](int x) {
        if (decision_bit((uint32_t)x, t, a.ks, a.rule)) atomicOr(&dec[x >> 5], 1u << (x & 31));
      };
      for (int rw = warp; rw < RWN; rw += NW) {
        const int y = rw / WPL, x = y * L + 32 * (rw - y * WPL) + lane;
        const bool isroot = ((s_new[rw] >> lane) & 1u) && par[x] == x;
        const uint32_t mr = __ballot_sync(0xffffffffu, isroot);
        if (isroot) list[(qh + qn + __popc(mr & ((1u << lane) - 1u))) & 63] = (uint16_t)x;
        qn += __popc(mr);
        __syncwarp();
        if (qn >= 32) {
          draw(list[(qh + lane) & 63]);
          qh += 32;
          qn -= 32;
          __syncwarp();
        }
      }
      if (lane < qn) draw(list[(qh + lane) & 63]);
      __syncthreads();
    }

    // ---- new spins (§2.4): every site walks from its label to the root, four
    // rows of the warp's segment in step, and takes the root's decision
    for (int seg = warp, j = sj0, w = sw0; seg < Z.nseg; seg += NW) {
      const int y0 = j * Z.S, n = min(Z.S, L - y0), nb = min(32, L - 32 * w);
      const int org = y0 * L + 32 * w + min(lane, nb - 1);
      for (int r0 = 0; r0 < n; r0 += 4) {
        int x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = par[org + min(r0 + i, n - 1) * L];  // past the end: the last row again
        bool more = true;
        while (__any_sync(0xffffffffu, more)) {
          more = false;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int p = par[x[i]];
            more |= p != x[i];
            x[i] = p;
          }
        }
        uint32_t mine = 0u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t dm = __ballot_sync(0xffffffffu, lane < nb && ((dec[x[i] >> 5] >> (x[i] & 31)) & 1u));
          if (lane == i) mine = dm;
        }
        if (lane < 4 && r0 + lane < n) {  // lane i has row r0 + i
          uint32_t* p = s_spin + (y0 + r0 + lane) * WPL + w;
          *p = (flip_rule ? *p : 0u) ^ mine;
        }
      }
      j += sdj;
      w += sdw;
      if (w >= WPL) {
        w -= WPL;
        ++j;
      }
    }
    // the next sweep's draws touch nothing that is still read here
  }

  for (int rw = warp; rw < RWN; rw += NW) {
    const int y = rw / WPL, x = (rw % WPL) * 32 + lane;
    if (x < L) a.spins[(size_t)y * L + x] = ((s_spin[rw] >> lane) & 1u) ? (int8_t)-1 : (int8_t)1;
  }
}

__global__ void __launch_bounds__(kSmallThreads, 1) small_sweep_kernel(const SmallArgs a) {
  extern __shared__ __align__(16) uint32_t smem[];
  small_body(a, smem);
}

// Batch replicas on the one-CTA path: CTA i runs replica small[i] for the
// sweeps of this chunk it has left (at most n), writes its trace rows and
// then advances its counter, trace row and sweeps left itself (the tiled
// schedule's counter advance skips these replicas).
__global__ void __launch_bounds__(kSmallThreads, 1)
    small_batch_kernel(const BatchArgs b, const int* small, int n) {
  extern __shared__ __align__(16) uint32_t smem[];
  ReplicaDesc* D = b.descs + small[blockIdx.x];
  if (!D->active || D->t_left <= 0) return;
  const int m = D->t_left < n ? (int)D->t_left : n;
  SmallArgs a;
  a.L = D->a.g.L;
  a.thr = D->a.thr;
  a.rule = D->a.rule;
  a.t0 = D->t;
  a.n = m;
  a.ks = D->a.ks;
  a.spins = D->a.spins_out;
  a.em = D->em_base + 2 * D->em_next;
  a.err = D->a.tb.err;
  small_body(a, smem);
  __syncthreads();
  if (threadIdx.x == 0) {
    D->t += (uint32_t)m;
    D->em_next += m;
    D->t_left -= m;
  }
}

size_t small_smem_bytes(int L) {
  const SmallShape Z(L);
  return (4 * (size_t)Z.RWN + 4 * (size_t)Z.DW + 2) * sizeof(uint32_t) + (size_t)Z.N * sizeof(uint16_t);
}

}  // namespace

cudaError_t launch_small(const SmallArgs& a, cudaStream_t st) {
  if (a.L < 2 || a.L > kSmallMaxL) return cudaErrorInvalidValue;
  if (a.n <= 0) return cudaSuccess;
  const size_t dyn = small_smem_bytes(kSmallMaxL);
  static bool attr_done = false;  // set once per process; the attribute is per function
  if (!attr_done) {
    const cudaError_t e =
        cudaFuncSetAttribute(small_sweep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  small_sweep_kernel<<<1, kSmallThreads, small_smem_bytes(a.L), st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_small_batch(const BatchArgs& b, const int* small, int nsmall, int max_L, int n, cudaStream_t st) {
  if (nsmall <= 0 || n <= 0) return cudaSuccess;
  if (max_L < 2 || max_L > kSmallMaxL) return cudaErrorInvalidValue;
  static bool attr_done = false;
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(small_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)small_smem_bytes(kSmallMaxL));
    if (e != cudaSuccess) return e;
    attr_done = true;
  }
  small_batch_kernel<<<nsmall, kSmallThreads, small_smem_bytes(max_L), st>>>(b, small, n);
  return cudaGetLastError();
}

}  // namespace sw
