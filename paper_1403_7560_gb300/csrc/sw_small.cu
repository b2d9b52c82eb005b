// Small Ising/Potts lattices (small_lattice in this file): whole sweeps by
// one CTA with the lattice in shared memory, n sweeps per launch.
//
// The tiled path pays four kernel launches and a global merge per sweep,
// which for a lattice of a few thousand sites is nearly all of the time.
// Here one CTA keeps the state, the bond planes and a union-find forest in
// shared memory and loops over the sweeps.  One SM runs every phase, so both
// its issue slots and the barriers count; the phases therefore work on whole
// row words where the arithmetic allows and on four sites a thread where it
// does not, with four barriers a sweep:
//   state: bit-planes of the row words (one plane for two-state lattices,
//     ceil(log2 q) for Potts), so that equality with the +x/+y/+z neighbours
//     is a few XORs a word and the measurement (popcounts of the planes and
//     of the same equality masks) rides on the next sweep's bonds;
//   phase 1: bond words, up to four threads per (row word, direction), one
//     Philox call of the bit-sliced comparison each (a word's uniforms are
//     compared most significant first; the partial results (less, equal)
//     combine in order), the cluster draws, every site its own parent;
//   phase 2a: the lowest bond of every x-run to the rows before it hooks the
//     run's start with a plain store (one parent, a smaller index);
//   phase 2b: unions for the other bonds (a fifth, plus those along x between
//     row words and around the torus), listed by phase 2a, a thread each;
//   phase 3: four sites a thread walk to their roots together and take the
//     roots' draws (the same draw definitions as the tiled path); eight
//     threads assemble a row word's planes.
// Forest nodes are (row word, bit), an order that agrees with the site order,
// so a cluster's root is its smallest site index.  Records are gathered in
// shared memory and written (with the FP64 accumulators, in sweep order)
// every kRing sweeps by one warp.
//   What bounds it is one warp's chain of instructions and the barriers (8
// cycles from one instruction of a warp to its next, 52% of the SM's issue
// slots at L = 64), so work per phase was cut rather than spread.  us per
// sweep, this kernel against a thread per site with byte states: 2D Ising L =
// 64 13.3 -> 7.4, L = 90 21.5 -> 12.9, 3D L = 16 24.3 -> 11.4.  Listing the
// unions for all threads (instead of a loop over a thread's own) took L = 64
// from 8.8 to 7.4.
//   After the last sweep the spins, that
// sweep's bond planes and a forest of (root, marker, draw) words are written
// back, so every readout call sees the same state as after tiled sweeps.
#include <string>

#include "../../include/sw.h"
#include "sw_device.cuh"

namespace swgb {
namespace {

using namespace dev;

constexpr int kSmallThreads = 1024, kRing = 64;

struct SmallLayout {
  size_t par, planes, state, draws, info, list, pdraw, total;
};

// Shared memory of a lattice of `rw` row words in state planes `nb`.
__host__ __device__ SmallLayout small_layout(const Lattice& lat, bool potts) {
  const size_t rw = (size_t)lat.R * (size_t)lat.W;
  const size_t nb = potts ? (size_t)lat.sbits : 1;
  SmallLayout s;
  s.par = 0;
  s.planes = s.par + 128 * rw;                       // a node per bit of a row word
  s.state = s.planes + 4 * (size_t)lat.dim * rw;
  s.draws = s.state + 4 * nb * rw;                   // two-state draw words
  s.info = s.draws + 4 * rw;                         // a row word's place (WordInfo)
  // unions, node << 16 | node: at most every +y and +z bond and one bond
  // along x per row word
  s.list = s.info + 4 * rw;
  s.pdraw = s.list + 4 * ((size_t)(lat.dim - 1) * lat.N + rw);
  s.total = s.pdraw + (potts && lat.dq != 2 ? 32 * rw : 0);
  s.total = (s.total + 15) & ~(size_t)15;
  return s;
}

// Shared memory of a small sweep besides the dynamic lattice block: the
// records' integer sums of the last kRing sweeps and what is derived of them.
struct SmallScratch {
  int M[kRing], E[kRing], ncl[kRing];
  unsigned int S2[kRing];
  double M2[kRing], Ed[kRing];
  unsigned int hist[256];
  uint32_t listed;                             // pairs counted into the list this sweep
};

// Division by an invariant divisor d (Granlund & Montgomery, "Division by
// invariant integers using multiplication", 1994): with m = floor((2^32 -
// 1) / d) + 1, floor(n / d) = umulhi(n, m) whenever n * d < 2^32 (the
// product overshoots n / d by less than n / 2^32 < 1 / d, which cannot
// carry the quotient past the next integer); d = 1 takes n itself.  The
// small lattices' indices (n < 2^16, d < 2^13) are far inside.
struct InvDiv {
  uint32_t d, m;
  __device__ explicit InvDiv(uint32_t dv) : d(dv), m(dv > 1u ? 0xffffffffu / dv + 1u : 0u) {}
  __device__ __forceinline__ uint32_t div(uint32_t n) const { return d > 1u ? __umulhi(n, m) : n; }
  __device__ __forceinline__ uint32_t mod(uint32_t n) const { return n - div(n) * d; }
};

// Place of a row word, packed once per launch: its highest valid bit, whether
// it has a row before it and is the last one along y and z, whether it ends
// its row, and its position in the row.
struct WordInfo {
  static constexpr uint32_t kYBefore = 1u << 5, kYLast = 1u << 6, kZBefore = 1u << 7, kZLast = 1u << 8,
                            kRowEnd = 1u << 9;
  static constexpr int kXWord = 10;
  static __device__ __forceinline__ uint32_t top(uint32_t w) { return w & 31u; }
  static __device__ __forceinline__ uint32_t valid(uint32_t w) { return kFull >> (31u - (w & 31u)); }
  static __device__ __forceinline__ uint32_t xword(uint32_t w) { return w >> kXWord; }
};

// The record's states up to this q are counted from the state planes.
constexpr int kPlaneHistQ = 16;

// Writes the records of the `cnt` (<= kRing) sweeps up to `last` from the
// ring, adds them to acc (global) in sweep order and clears their slots;
// called by one whole warp, slots indexed by sweep % kRing.
__device__ __forceinline__ void flush_records(const Lattice& lat, const Measure& mb, SmallScratch& sc,
                                              uint32_t last, int cnt) {
  const int lane = (int)(threadIdx.x & 31u);
  __syncwarp();
  for (int k = lane; k < cnt; k += 32) {
    const uint32_t sweep = last - (uint32_t)(cnt - 1 - k), slot = sweep % kRing;
    store_record(lat, mb, sweep, (long long)sc.M[slot], (long long)sc.E[slot], (long long)sc.S2[slot], 0.0, 0.0,
                 0.0, (long long)sc.ncl[slot], sc.M2[slot], sc.Ed[slot]);
  }
  __syncwarp();
  if (lane < 6) {
    double a = mb.acc[lane];
    for (int k = 0; k < cnt; ++k) {
      const uint32_t slot = (last - (uint32_t)(cnt - 1 - k)) % kRing;
      const double m2 = sc.M2[slot], ed = sc.Ed[slot];
      const double v = lane == 0   ? 1.0
                       : lane == 1 ? m2
                       : lane == 2 ? __dmul_rn(m2, m2)
                       : lane == 3 ? ed
                       : lane == 4 ? __dmul_rn(ed, ed)
                                   : (double)sc.ncl[slot];
      a = __dadd_rn(a, v);
    }
    mb.acc[lane] = a;
  }
  __syncwarp();
  for (int k = lane; k < cnt; k += 32) {
    const uint32_t slot = (last - (uint32_t)k) % kRing;
    sc.M[slot] = sc.E[slot] = sc.ncl[slot] = 0;
    sc.S2[slot] = 0u;
  }
  __syncwarp();
}

// Joins the trees of a and b: both walks advance together, each step on a
// non-root halving its path (one walk's loads hide the other's; without the
// halving 2D L = 64 took 10.0 us a sweep, with it 7.4, and two walks one
// after the other 7.5), then the larger root hooks under the smaller.
// sunion's contract (bounded, an error past cap).
__device__ __forceinline__ void join_pair(uint32_t* par, uint32_t a, uint32_t b, int* err, uint32_t cap) {
  volatile uint32_t* vp = par;
  for (uint32_t it = 0; it < cap; ++it) {
    for (int k = 0; k < 65536; ++k) {
      const uint32_t a2 = vp[a], b2 = vp[b];
      if (a2 == a && b2 == b) break;
      const uint32_t a3 = vp[a2], b3 = vp[b2];
      if (a3 != a2) vp[a] = a3;
      if (b3 != b2) vp[b] = b3;
      a = a3;
      b = b3;
      if (a == b) break;
    }
    if (a == b) return;
    const uint32_t hi = max(a, b), lo = min(a, b);
    const uint32_t old = atomicMin(&par[hi], lo);
    if (old == hi) return;
    a = old;
    b = lo;
  }
  atomicExch(err, kErrTimeout);
}

// n sweeps after sweep0 of one small lattice by the whole CTA (whole warps).
template <int D, bool POTTS>
__device__ __forceinline__ void sweep_small(const Lattice& lat, const Measure& mb, uint32_t sweep0, int n,
                                            bool measure, const SmallLayout& lay, unsigned char* smem,
                                            SmallScratch& sc) {
  uint32_t* par = reinterpret_cast<uint32_t*>(smem + lay.par);
  uint32_t* pl = reinterpret_cast<uint32_t*>(smem + lay.planes);
  uint32_t* st = reinterpret_cast<uint32_t*>(smem + lay.state);
  uint32_t* dw = reinterpret_cast<uint32_t*>(smem + lay.draws);
  uint32_t* info = reinterpret_cast<uint32_t*>(smem + lay.info);
  uint32_t* list = reinterpret_cast<uint32_t*>(smem + lay.list);
  uint8_t* pd = smem + lay.pdraw;
  const uint32_t N = lat.N, L = (uint32_t)lat.L, W = (uint32_t)lat.W, RW = lat.R * W, LW = L * W;
  const InvDiv byL(L), byW(W), byRW(RW);
  const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u, warp = tid >> 5, nwarps = nt >> 5;
  const int sb = lat.sbits, shift = sb + 1;
  const int nb = POTTS ? sb : 1;
  const bool two_state = !POTTS || lat.dq == 2;
  const uint32_t lr_bit = 1u << sb;
  const uint32_t t_bond = lat.t_bond;
  // threads per bond word: as many of a word's first Philox calls in parallel
  // as the CTA has threads for
  const uint32_t ndraw = two_state ? RW : 0u;
  const uint32_t ksh = 4u * D * RW + ndraw <= nt ? 2u : (2u * D * RW + ndraw <= nt ? 1u : 0u);
  const uint32_t nbond = (D * RW) << ksh, nbond32 = (nbond + 31u) & ~31u;
  const uint32_t nquads = 8u * RW;
  uint8_t* gs = static_cast<uint8_t*>(lat.spins);

  // equality of row word g with its neighbour along d, from the state planes
  auto equal_word = [&](uint32_t d, uint32_t g) {
    const uint32_t wi = info[g];
    uint32_t diff = 0u;
    if (d == 0) {
      // the word of the next x (the row's first after the last)
      const uint32_t gn = (wi & WordInfo::kRowEnd) ? g - WordInfo::xword(wi) : g + 1u;
      for (int k = 0; k < nb; ++k) {
        const uint32_t w = st[k * RW + g];
        diff |= w ^ ((w >> 1) | ((st[k * RW + gn] & 1u) << WordInfo::top(wi)));
      }
    } else {
      const uint32_t gn = d == 1 ? ((wi & WordInfo::kYLast) ? g - (L - 1u) * W : g + W)
                                 : ((wi & WordInfo::kZLast) ? g - (L - 1u) * LW : g + LW);
      for (int k = 0; k < nb; ++k) diff |= st[k * RW + g] ^ st[k * RW + gn];
    }
    return ~diff & WordInfo::valid(wi);
  };
  // M (Ising) or the histogram (Potts) of the state in the planes; the warp's
  // share is added to the slot
  auto add_state = [&](uint32_t slot) {
    if (!POTTS) {
      int m = 0;
      for (uint32_t g = tid; g < RW; g += nt) m -= 2 * __popc(st[g]);
      if (warp * 32u < RW) {
        m = __reduce_add_sync(kFull, m);
        if (lane == 0) atomicAdd(&sc.M[slot], m);
      }
      if (tid == 0) atomicAdd(&sc.M[slot], (int)N);
    } else if (lat.q <= kPlaneHistQ) {
      const uint32_t padded = (RW + 31u) & ~31u;  // whole warps per state
      for (uint32_t c = tid; c < padded * (uint32_t)lat.q; c += nt) {
        const uint32_t k = c / padded, g = c - k * padded;
        int m = 0;
        if (g < RW) {
          uint32_t is = WordInfo::valid(info[g]);
          for (int b = 0; b < nb; ++b) is &= st[b * RW + g] ^ ((k >> b) & 1u ? 0u : kFull);
          m = __popc(is);
        }
        m = __reduce_add_sync(kFull, m);
        if (lane == 0 && m) atomicAdd(&sc.hist[k], (unsigned)m);
      }
    }
  };
  // sum of the squared histogram of the state, by one warp; clears it
  auto take_histogram = [&](uint32_t slot) {
    unsigned s2 = 0u;
    for (int k = (int)lane; k < 256; k += 32) {
      const unsigned h = sc.hist[k];
      if (k < lat.q) s2 += h * h;  // at most N^2 < 2^32 in all
      sc.hist[k] = 0u;
    }
    s2 = __reduce_add_sync(kFull, s2);
    if (lane == 0) sc.S2[slot] = s2;
  };

  for (uint32_t k = tid; k < (uint32_t)kRing; k += nt) {
    sc.M[k] = sc.E[k] = sc.ncl[k] = 0;
    sc.S2[k] = 0u;
  }
  for (uint32_t k = tid; k < 256u; k += nt) sc.hist[k] = 0u;
  // equality masks of the incoming state, from its bytes (a warp per row word)
  for (uint32_t g = warp; g < RW; g += nwarps) {
    const uint32_t row = byW.div(g), x = 32u * (g - row * W) + lane;
    const uint32_t z = byL.div(row), y = row - z * L;
    bool q0 = false, q1 = false, q2 = false;
    if (x < L) {
      const uint8_t si = gs[row * L + x];
      q0 = gs[row * L + (x + 1u == L ? 0u : x + 1u)] == si;
      q1 = gs[((y + 1u == L ? 0u : y + 1u) + L * z) * L + x] == si;
      if (D == 3) q2 = gs[(y + L * (z + 1u == L ? 0u : z + 1u)) * L + x] == si;
    }
    const uint32_t b0 = __ballot_sync(kFull, q0), b1 = __ballot_sync(kFull, q1), b2 = __ballot_sync(kFull, q2);
    if (lane < (uint32_t)D) pl[lane * RW + g] = lane == 0 ? b0 : lane == 1 ? b1 : b2;
    if (lane == 0) {
      const uint32_t xw = g - row * W;
      info[g] = (xw + 1u < W ? 31u : (L - 1u) & 31u) | (y > 0u ? WordInfo::kYBefore : 0u) |
                (y + 1u == L ? WordInfo::kYLast : 0u) | (z > 0u ? WordInfo::kZBefore : 0u) |
                (z + 1u == L ? WordInfo::kZLast : 0u) | (xw + 1u == W ? WordInfo::kRowEnd : 0u) |
                (xw << WordInfo::kXWord);
    }
  }

  for (int s = 0; s < n; ++s) {
    const uint32_t sweep = sweep0 + (uint32_t)s + 1u;
    const bool last = s + 1 == n;
    const bool take = measure && s > 0;  // this sweep's bonds also measure the previous sweep's state
    const uint32_t prev = (sweep - 1u) % kRing;
    __syncthreads();
    // ---- phase 1
    if (tid == 0) sc.listed = 0u;
    int same = 0;
    for (uint32_t c0 = 0; c0 < nbond32 + ndraw; c0 += nt) {
      if (c0 + tid - lane >= nbond32) {  // whole warps: the two-state draw words
        const uint32_t g = c0 + tid - nbond32;
        if (g < ndraw) dw[g] = philox(g, sweep, kDraw, 1u, lat.rk).x;
        continue;
      }
      const uint32_t t = c0 + tid, c = t >> ksh, sub = t & ((1u << ksh) - 1u);
      uint32_t lt = 0u, eq = 0u, d = 0u, g = 0u;
      if (c < D * RW) {
        d = byRW.div(c);
        g = c - d * RW;
        eq = s > 0 ? equal_word(d, g) : pl[c];
        if (sub == 0) same += __popc(eq);
        if (eq) {
          const uint4 w = philox(g, sweep, kBond, 8u * d + sub, lat.rk);
          const uint32_t tb = t_bond << (4u * sub);  // the call's four threshold bits on top
          cmp_step_lane(lt, eq, w.x, (int)tb >> 31);
          cmp_step_lane(lt, eq, w.y, (int)(tb << 1) >> 31);
          cmp_step_lane(lt, eq, w.z, (int)(tb << 2) >> 31);
          cmp_step_lane(lt, eq, w.w, (int)(tb << 3) >> 31);
        }
      }
      for (uint32_t o = 1; o < (1u << ksh); o <<= 1) {
        const uint32_t l2 = __shfl_down_sync(kFull, lt, o), e2 = __shfl_down_sync(kFull, eq, o);
        lt |= eq & l2;
        eq &= e2;
      }
      if (sub == 0 && c < D * RW) {
        if (eq) lt |= bernoulli_tail(g, sweep, (int)d, t_bond, eq, lat.rk, 1 << ksh);
        pl[c] = lt;
      }
    }
    if (take) {
      if (warp * 32u < nbond) {
        same = __reduce_add_sync(kFull, same);
        // E: Ising -(parallel - antiparallel), Potts the unequal bonds
        if (lane == 0) atomicAdd(&sc.E[prev], POTTS ? -same : -2 * same);
      }
      if (tid == 0) atomicAdd(&sc.E[prev], D * (int)N);
      add_state(prev);
    }
    if (POTTS && !two_state) {
      // Potts draw of every site: word (i & 3) of Philox(i >> 2, sweep, DRAW, 0)
      for (uint32_t c = tid; 4u * c < N; c += nt) {
        const uint4 w = philox(c, sweep, kDraw, 0u, lat.rk);
        uint32_t row = byL.div(4u * c), x = 4u * c - row * L;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (4u * c + (uint32_t)k < N)
            pd[32u * (row * W + (x >> 5)) + (x & 31u)] = (uint8_t)draw_value(word_of(w, k), (uint32_t)lat.dq);
          if (++x == L) {
            x = 0u;
            ++row;
          }
        }
      }
    }
    for (uint32_t c = tid; c < nquads; c += nt)
      reinterpret_cast<uint4*>(par)[c] = make_uint4(4u * c, 4u * c + 1u, 4u * c + 2u, 4u * c + 3u);
    __syncthreads();

    // ---- phase 2a: hooks, eight threads per row word, each its four bits
    if (take && warp == nwarps - 1u) {
      if (POTTS) take_histogram(prev);
      if ((uint32_t)s % kRing == 0u) flush_records(lat, mb, sc, sweep - 1u, kRing);
    }
    for (uint32_t c0 = 0; c0 < nquads; c0 += nt) {
      if (c0 + tid - lane >= nquads) break;  // whole warps
      const uint32_t c = c0 + tid, g = c >> 3, sh4 = 4u * (c & 7u);
      uint32_t wi = 0u, vmask = 0u, S = 0u, Sy = 0u, Sz = 0u, ny = 0u, nz = 0u, wy = 0u, wz = 0u, nx = 0u;
      if (c < nquads) {
        wi = info[g];
        vmask = WordInfo::valid(wi);
        const bool has_y = (wi & WordInfo::kYBefore) != 0u, has_z = D == 3 && (wi & WordInfo::kZBefore) != 0u;
        const uint32_t A0 = pl[g], X = A0 & (vmask >> 1), joined = X << 1;
        S = ~joined;
        const uint32_t Yp = has_y ? pl[RW + g - W] : 0u, Xy = has_y ? pl[g - W] & (vmask >> 1) : 0u;
        const uint32_t Zp = has_z ? pl[2u * RW + g - LW] : 0u, Xz = has_z ? pl[g - LW] & (vmask >> 1) : 0u;
        // bonds whose runs the previous bit has not joined already
        uint32_t Y2 = Yp & ~((Yp & X & Xy) << 1), Z2 = Zp & ~((Zp & X & Xz) << 1);
        const uint32_t both = Y2 | Z2;
        // bits above the first one of their run: a carry from each bit runs up
        // the joined bits and stops at the end of the run
        const uint32_t seed = (both << 1) & joined;
        const uint32_t F = both & ~((((seed + joined) ^ joined) | seed) & joined);
        const uint32_t FY = F & Y2;
        Z2 &= ~(F & ~Y2);
        Y2 &= ~F;
        Sy = ~(Xy << 1);
        Sz = ~(Xz << 1);
        for (uint32_t f = (F >> sh4) & 15u; f; f &= f - 1u) {
          const int b = (int)sh4 + __ffs(f) - 1;
          const bool y_bond = D == 2 || ((FY >> b) & 1u);
          par[32u * g + run_start(S, b)] =
              y_bond ? 32u * (g - W) + run_start(Sy, b) : 32u * (g - LW) + run_start(Sz, b);
        }
        ny = (Y2 >> sh4) & 15u;
        if (D == 3) nz = (Z2 >> sh4) & 15u;
        // around the torus
        if (wi & WordInfo::kYLast) wy = (pl[RW + g] >> sh4) & 15u;
        if (D == 3 && (wi & WordInfo::kZLast)) wz = (pl[2u * RW + g] >> sh4) & 15u;
        // to the next row word along x, or around
        const uint32_t top = WordInfo::top(wi);
        nx = (top & ~3u) == sh4 ? (A0 >> top) & 1u : 0u;
      }
      // the other bonds go to the lattice's list of unions (most threads have
      // none, a few have several: from the list each thread takes one)
      const uint32_t mine = (uint32_t)(__popc(ny) + __popc(nz) + __popc(wy) + __popc(wz)) + nx;
      uint32_t upto = mine;
#pragma unroll
      for (uint32_t o = 1; o < 32u; o <<= 1) {
        const uint32_t u = __shfl_up_sync(kFull, upto, o);
        if (lane >= o) upto += u;
      }
      uint32_t base = 0u;
      if (lane == 31u && upto) base = atomicAdd(&sc.listed, upto);
      base = __shfl_sync(kFull, base, 31);
      if (mine) {
        uint32_t at = base + upto - mine;
        auto put = [&](uint32_t bits, uint32_t gn, uint32_t Sn) {
          for (uint32_t u = bits; u; u &= u - 1u) {
            const int b = (int)sh4 + __ffs(u) - 1;
            list[at++] = (32u * g + run_start(S, b)) << 16 | (32u * gn + run_start(Sn, b));
          }
        };
        put(ny, g - W, Sy);
        if (D == 3) put(nz, g - LW, Sz);
        if (wy) put(wy, g - (L - 1u) * W, ~((pl[g - (L - 1u) * W] & (vmask >> 1)) << 1));
        if (D == 3 && wz) put(wz, g - (L - 1u) * LW, ~((pl[g - (L - 1u) * LW] & (vmask >> 1)) << 1));
        if (nx)
          list[at] = (32u * g + run_start(S, (int)WordInfo::top(wi))) << 16 |
                     32u * ((wi & WordInfo::kRowEnd) ? g - WordInfo::xword(wi) : g + 1u);
      }
    }
    __syncthreads();

    // ---- phase 2b: the listed unions
    for (uint32_t e = tid; e < sc.listed; e += nt)
      join_pair(par, list[e] >> 16, list[e] & 0xffffu, lat.err, lat.cap);
    __syncthreads();

    // ---- phase 3: roots, new states; a row word per eight lanes
    int roots = 0;
    for (uint32_t c0 = 0; c0 < nquads; c0 += nt) {
      if (c0 + tid - lane >= nquads) break;  // whole warps
      const uint32_t c = c0 + tid, g = c >> 3, sh4 = 4u * (c & 7u), t0 = 4u * c;
      uint32_t bits = 0u, v[4] = {0u, 0u, 0u, 0u}, p[4] = {0u, 0u, 0u, 0u};
      if (c < nquads) {
        const uint32_t vmask = WordInfo::valid(info[g]);
        bits = (vmask >> sh4) & 15u;
        if (bits) {
          const uint32_t S = ~((pl[g] & (vmask >> 1)) << 1);
          const uint4 own = reinterpret_cast<const uint4*>(par)[c];
          p[0] = ((S >> sh4) & 1u) ? own.x : par[32u * g + run_start(S, (int)sh4)];
          p[1] = ((S >> sh4) & 2u) ? own.y : p[0];
          p[2] = ((S >> sh4) & 4u) ? own.z : p[1];
          p[3] = ((S >> sh4) & 8u) ? own.w : p[2];
          uint32_t moved = 1u;  // parents only decrease: at most a walk per node
          for (uint32_t it = 0; it < 32u * RW && moved; ++it) {
            moved = 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t up = par[p[j]];
              moved |= up ^ p[j];
              p[j] = up;
            }
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            v[j] = two_state ? (dw[p[j] >> 5] >> (p[j] & 31u)) & 1u : (uint32_t)pd[p[j]];
            if (((bits >> j) & 1u) && p[j] == t0 + (uint32_t)j) ++roots;
          }
        }
      }
      for (int k = 0; k < nb; ++k) {
        uint32_t w = ((v[0] >> k) & 1u) | (((v[1] >> k) & 1u) << 1) | (((v[2] >> k) & 1u) << 2) |
                     (((v[3] >> k) & 1u) << 3);
        w = (w & bits) << sh4;
        w |= __shfl_xor_sync(kFull, w, 1);
        w |= __shfl_xor_sync(kFull, w, 2);
        w |= __shfl_xor_sync(kFull, w, 4);
        if (sh4 == 0u && c < nquads) st[k * RW + g] = w;
      }
      if (POTTS && measure && lat.q > kPlaneHistQ)
        for (int j = 0; j < 4; ++j)
          if ((bits >> j) & 1u) atomicAdd(&sc.hist[v[j]], 1u);
      if (last) {
        const uint32_t row = byW.div(g), xw = g - row * W;
        for (int j = 0; j < 4; ++j) {
          if (!((bits >> j) & 1u)) continue;
          const uint32_t i = row * L + 32u * xw + sh4 + (uint32_t)j, t = t0 + (uint32_t)j;
          const uint32_t gr = p[j] >> 5, rr = byW.div(gr), r = rr * L + 32u * (gr - rr * W) + (p[j] & 31u);
          const uint32_t own = two_state ? (dw[g] >> (t & 31u)) & 1u : (uint32_t)pd[t];
          lat.forest[i] = (r << shift) | (p[j] == t ? lr_bit : 0u) | own;
          gs[i] = POTTS ? (uint8_t)v[j] : (uint8_t)(v[j] ? (int8_t)-1 : (int8_t)1);
        }
      }
    }
    if (measure) {
      if (warp * 32u < nquads) {
        roots = __reduce_add_sync(kFull, roots);
        if (lane == 0 && roots) atomicAdd(&sc.ncl[sweep % kRing], roots);
      }
    }
  }
  __syncthreads();
  if (measure) {
    // the last sweep's state
    const uint32_t slot = (sweep0 + (uint32_t)n) % kRing;
    int same = 0;
    for (uint32_t c = tid; c < D * RW; c += nt) {
      const uint32_t d = byRW.div(c);
      same += __popc(equal_word(d, c - d * RW));
    }
    if (warp * 32u < D * RW) {
      same = __reduce_add_sync(kFull, same);
      if (lane == 0) atomicAdd(&sc.E[slot], POTTS ? -same : -2 * same);
    }
    if (tid == 0) atomicAdd(&sc.E[slot], D * (int)N);
    add_state(slot);
    __syncthreads();
    if (warp == 0) {
      if (POTTS) take_histogram(slot);
      flush_records(lat, mb, sc, sweep0 + (uint32_t)n, (n - 1) % kRing + 1);
    }
  }
  for (uint32_t w = tid; w < (uint32_t)D * RW; w += nt) lat.planes[w] = pl[w];
}

template <int D, bool POTTS>
__global__ void __launch_bounds__(kSmallThreads, 1)
    k_sweep_small(const __grid_constant__ Lattice lat, const __grid_constant__ Measure mb, uint32_t sweep0,
                  int n, int measure, SmallLayout lay) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SmallScratch sc;
  sweep_small<D, POTTS>(lat, mb, sweep0, n, measure != 0, lay, smem, sc);
}

// Small members of a batch, one CTA per member (list[blockIdx.x]): up to n
// measured sweeps from sweep `first` (0-based) of the member's sweeps of the
// current call.
template <int D>
__global__ void __launch_bounds__(kSmallThreads, 1)
    k_sweep_small_batch(const BatchMember* members, const uint32_t* list, uint32_t first, uint32_t n) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ SmallScratch sc;
  __shared__ Lattice s_lat;  // read on every Philox round
  static_assert(sizeof(Lattice) % 4 == 0, "lattice copy");
  const BatchMember& m = members[__ldg(&list[blockIdx.x])];
  if (first >= m.nsweeps) return;  // the member has had its sweeps this call
  for (uint32_t k = threadIdx.x; k < sizeof(Lattice) / 4; k += blockDim.x)
    reinterpret_cast<uint32_t*>(&s_lat)[k] = reinterpret_cast<const uint32_t*>(&m.lat)[k];
  __syncthreads();
  const uint32_t left = m.nsweeps - first;
  const int k = (int)(left < n ? left : n);
  if (s_lat.model == kPotts)
    sweep_small<D, true>(s_lat, m.meas, m.sweep0 + first, k, true, small_layout(s_lat, true), smem, sc);
  else
    sweep_small<D, false>(s_lat, m.meas, m.sweep0 + first, k, true, small_layout(s_lat, false), smem, sc);
}

// Threads for a lattice: one per four sites, whole warps.
unsigned small_threads(const Lattice& lat) {
  const uint32_t quads = 8u * lat.R * (uint32_t)lat.W;
  const uint32_t t = (quads + 31u) & ~31u;
  return t < (uint32_t)kSmallThreads ? t : (unsigned)kSmallThreads;
}

// The shared-memory limit of a kernel on the current device, raised once per
// device.
template <class K>
cudaError_t allow_small_smem(K* k, int& configured_device) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || configured_device == dev) return e;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_layout_bytes_max());
  if (e == cudaSuccess) configured_device = dev;
  return e;
}

template <int D, bool POTTS>
cudaError_t launch_small_t(const Lattice& lat, const Measure& m, uint32_t sweep0, int n, bool measure,
                           cudaStream_t st) {
  const SmallLayout lay = small_layout(lat, POTTS);
  static thread_local int configured_device = -1;
  const cudaError_t e = allow_small_smem(k_sweep_small<D, POTTS>, configured_device);
  if (e != cudaSuccess) return e;
  k_sweep_small<D, POTTS><<<1, small_threads(lat), lay.total, st>>>(lat, m, sweep0, n, measure ? 1 : 0, lay);
  return cudaGetLastError();
}

// Two CTAs of `smem` bytes of dynamic shared memory on one SM (228 KB, of which
// each CTA takes its static part and 1 KB besides, in units of 128 bytes).
bool two_fit(size_t smem) {
  const size_t cta = ((smem + sizeof(SmallScratch) + sizeof(Lattice) + 127) & ~(size_t)127) + 1024;
  return 2 * cta <= 228 * 1024;
}

template <int D>
cudaError_t launch_small_batch_t(const BatchMember* members, const uint32_t* list, uint32_t count, size_t smem,
                                 uint32_t first, uint32_t n, cudaStream_t st) {
  static thread_local int configured_device = -1;
  const cudaError_t e = allow_small_smem(k_sweep_small_batch<D>, configured_device);
  if (e != cudaSuccess) return e;
  // members beyond one CTA per SM share SMs in pairs of half-size CTAs, where
  // an SM's shared memory holds two of the largest; else each has an SM to
  // itself and all of its threads.  us per batch sweep of 300 members, 512 /
  // 1024 threads: pairs fit, 2D Ising L = 64 18.9 / 23.5, 104 36.4 / 43.1, 3D
  // 18 39.0 / 43.5; they do not, 2D 112 49.6 / 44.2, Potts q = 3 L = 100 60.6
  // / 53.8, 3D 20 56.6 / 50.6, 300 of L = 64 and one of 112 37.0 / 34.0
  const bool pairs = count > (uint32_t)sm_count() && two_fit(smem);
  const unsigned threads = pairs ? kSmallThreads / 2 : kSmallThreads;
  k_sweep_small_batch<D><<<count, threads, smem, st>>>(members, list, first, n);
  return cudaGetLastError();
}

}  // namespace

size_t small_layout_bytes_max() { return kSmallSharedBytes; }

bool small_lattice(const Lattice& lat) {
  if (lat.model != kIsing && lat.model != kPotts) return false;
  if (lat.N > (lat.dim == 2 ? kSmallSites2D : kSmallSites3D)) return false;
  return small_layout(lat, lat.model == kPotts).total <= small_layout_bytes_max();
}

size_t small_layout_bytes(const Lattice& lat) { return small_layout(lat, lat.model == kPotts).total; }

cudaError_t launch_small_batch(const BatchMember* members, int dim, const uint32_t* list, uint32_t count,
                               size_t smem, uint32_t first, uint32_t n, cudaStream_t st) {
  return dim == 2 ? launch_small_batch_t<2>(members, list, count, smem, first, n, st)
                  : launch_small_batch_t<3>(members, list, count, smem, first, n, st);
}

cudaError_t launch_sweeps_small(const Lattice& lat, const Measure& m, uint32_t sweep0, int n, bool measure,
                                cudaStream_t st) {
  const bool potts = lat.model == kPotts;
  if (lat.dim == 2) return potts ? launch_small_t<2, true>(lat, m, sweep0, n, measure, st)
                                 : launch_small_t<2, false>(lat, m, sweep0, n, measure, st);
  return potts ? launch_small_t<3, true>(lat, m, sweep0, n, measure, st)
               : launch_small_t<3, false>(lat, m, sweep0, n, measure, st);
}

}  // namespace swgb
