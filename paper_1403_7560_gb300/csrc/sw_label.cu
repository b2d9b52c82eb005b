// Steps (1) and (2) of the SW sweep (Komura & Okabe, Sec. 2): active bond
// generation and the tile-local half of the cluster labeling.
//
// k_label: one CTA per 32 x TY (x TZ) tile, one thread per 32-site row word.
//   phase 1 (thread per row word): Ising/Potts bonds from the int8/uint8
//     spins -- equality of the row with its +x/+y/+z neighbour rows from
//     byte-lane compares, AND a bit-sliced Bernoulli word per direction
//     (u < t decided for 32 sites at once from whole Philox words) -- and
//     the row's cluster draws (one Philox word per row word for two-state
//     draws, one per four sites for Potts); or the bonds read from the
//     bit-planes.
//   Before it, every site is its own parent in the shared-memory forest; an
//   x-run is represented by its start, the only site of it ever looked up.
//   phase 2 (thread per row word): the lowest bond of every run to the rows
//     before it (-y, -z) hooks the run's start there with a plain store: a
//     start has one parent and every parent a smaller index, so no find and
//     no atomic is needed.  The other in-tile bonds (a fifth of them at the
//     critical point) are shared-memory unions (runs already joined through
//     the previous bit are skipped).
//   phase 3 (thread per four sites, or lane per site where L is not a
//     multiple of 4): find the tile-local root of the site's run start and
//     write the forest word (root as a global index, local-root marker,
//     cluster draw).
//   The kernel is issue-bound (71% of issue slots, 20 of 32 lanes): what
//   counts is instructions.  A union is two walks and an atomic in a loop the
//   warp leaves with its slowest thread, so the hooks took the loop from 21 to
//   8 trips a warp; four sites per thread share the row's loads, address
//   arithmetic and one 16-byte store.  3D Ising L = 256 at T_c: 85.0 M -> 67.4
//   M warp instructions, 108.9 -> 85.4 us; from bond planes (XY) 76.2 -> 59.3
//   us; 2D L = 4096 94.8 -> 76.2 us (ncu, cold L2).
//   With MEASURE the row threads also measure the incoming spins (the state
//   after the previous sweep) from the same bytes and equality masks.
// k_bonds_xy: XY bonds: project on the sweep's mirror axis (once per site,
//   through a shared-memory block with halo) and test the embedded-Ising
//   probability; ballot into the bit-planes; optionally measure the
//   incoming state from the same projections.
#include "sw_device.cuh"

namespace swgb {
namespace {

using namespace dev;

constexpr int kSmallQ = 16;  // Potts histograms up to this q are counted per thread

// The 32 spin bytes of a row word and of its +x, +y, +z neighbour words.
struct RowBytes {
  uint32_t a[9], ax[8], ay[8], az[8];
};

// The 32 bytes from s[base] on as 8 words (and w[8], whose low byte is byte
// 32), whatever the alignment: two 16-byte loads where every row is 16-byte
// aligned (L a multiple of 16), else aligned words shifted into place (against
// a byte load per site: 2D L = 515 sweeps 39.7 -> 32.2 us, 3D L = 100 46.3 ->
// 41.5, the labeling unsplit).  Up to 36 bytes from s[base] are read: past the row's end they belong to the next row, past
// the lattice's to the buffer's padding (kSpinPad), and the caller masks them.
template <bool NEXT>
__device__ __forceinline__ void load32(const uint8_t* s, uint32_t base, bool vec16, uint32_t* w) {
  if (vec16) {
    const uint4* p = reinterpret_cast<const uint4*>(s + base);
    const uint4 v0 = __ldg(p), v1 = __ldg(p + 1);
    w[0] = v0.x; w[1] = v0.y; w[2] = v0.z; w[3] = v0.w;
    w[4] = v1.x; w[5] = v1.y; w[6] = v1.z; w[7] = v1.w;
    if (NEXT) w[8] = __ldg(s + base + 32);
  } else {
    const uint32_t* p = reinterpret_cast<const uint32_t*>(s + (base & ~3u));
    const uint32_t sh = 8u * (base & 3u);
    uint32_t v = __ldg(p);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t v1 = __ldg(p + k + 1);
      w[k] = __funnelshift_r(v, v1, sh);
      v = v1;
    }
    if (NEXT) w[8] = v >> sh;
  }
}

// A row word's bytes moved by one site along +x; w[8] holds byte 32.  The last
// site of the row has the row's first one as its neighbour.
__device__ __forceinline__ void shift_row(const uint8_t* s, uint32_t* w, uint32_t row_start, int L, int x0,
                                          int nvalid, uint32_t* ax) {
  const bool row_end = x0 + 32 >= L;
  const uint32_t first = row_end ? (uint32_t)__ldg(s + row_start) : 0u;
  if (row_end && nvalid == 32) w[8] = first;
#pragma unroll
  for (int k = 0; k < 8; ++k) ax[k] = __byte_perm(w[k], w[k + 1], 0x4321);
  if (row_end && nvalid < 32) {
    const int at = nvalid - 1;
    const uint32_t byte = 0xffu << (8 * (at & 3)), rep = first * 0x01010101u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t m = (at >> 2) == k ? byte : 0u;
      ax[k] = (ax[k] & ~m) | (rep & m);
    }
  }
}

template <int D>
__device__ __forceinline__ void load_rows(const uint8_t* s, int L, int x0, int nvalid, uint32_t row,
                                          uint32_t row_y, uint32_t row_z, RowBytes& rb) {
  const bool vec16 = (L & 15) == 0;
  const uint32_t rowL = row * (uint32_t)L;
  load32<true>(s, rowL + (uint32_t)x0, vec16, rb.a);
  load32<false>(s, row_y * (uint32_t)L + (uint32_t)x0, vec16, rb.ay);
  if (D == 3) load32<false>(s, row_z * (uint32_t)L + (uint32_t)x0, vec16, rb.az);
  shift_row(s, rb.a, rowL, L, x0, nvalid, rb.ax);
}

// Measurement of one 32-site row word from its bytes and the equality masks
// e0..e2 with its +x/+y/+z neighbours.  MM 1 (Ising): M = #(+1) - #(-1) and
// E = -(#parallel - #antiparallel) over the +d bonds.  MM 2 (Potts): E = the
// number of unequal +d bonds, and the histogram n[k] of the states (per-warp
// bins for q <= kSmallQ, shared bins above).
template <int MM>
__device__ __forceinline__ void measure_state(const uint32_t* a, uint32_t vmask, int nvalid, int q, int& m_acc,
                                              unsigned int* warp_hist, unsigned int* s_hist) {
  if (MM == 1) {
    uint32_t ones[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) ones[k] = 0x01010101u;
    m_acc += 2 * __popc(eq_bits(a, ones) & vmask) - nvalid;
  } else if (MM == 2) {
    if (q <= kSmallQ) {
      for (int k = 0; k < q; ++k) {
        uint32_t kk[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) kk[j] = 0x01010101u * (uint32_t)k;
        const unsigned c = (unsigned)__popc(eq_bits(a, kk) & vmask);
        if (c) atomicAdd(&warp_hist[k], c);
      }
    } else {
#pragma unroll
      for (int b = 0; b < 32; ++b)
        if (b < nvalid) atomicAdd(&s_hist[(a[b >> 2] >> (8 * (b & 3))) & 0xffu], 1u);
    }
  }
}

template <int D, int MM>
__device__ __forceinline__ void measure_row(const RowBytes& rb, uint32_t e0, uint32_t e1, uint32_t e2,
                                            uint32_t vmask, int nvalid, int q, int& m_acc, int& e_acc,
                                            unsigned int* warp_hist, unsigned int* s_hist) {
  const int par_bonds = __popc(e0) + __popc(e1) + (D == 3 ? __popc(e2) : 0);
  e_acc += D * nvalid - (MM == 1 ? 2 : 1) * par_bonds;
  measure_state<MM>(rb.a, vmask, nvalid, q, m_acc, warp_hist, s_hist);
}

// MM (measurement mode) 1 = Ising, 2 = Potts: also measure the incoming
// spins (the state after sweep - 1): M and E from the row words' equality
// masks and the Potts histogram, added to the measurement slots (the flip
// kernel of this sweep writes the record of sweep - 1).  MM 0 and 3: no
// measurement, two-state (0: Ising, and XY / clock from their bond planes)
// or Potts (3) cluster draws.
// Shared memory of one tile's labeling in measurement mode MM (the Potts
// draw words and histograms only where Potts lattices can run).
template <class S, int MM, int K = 1>
struct LabelSmem {
  static constexpr int ROWS = S::ROWS, NW = K * S::THREADS / 32;
  static constexpr bool kPottsDraws = MM >= 2;  // MM 0 and 1: two-state draws only
  static constexpr int kDrawWords = (kPottsDraws ? 8 : 1) * (ROWS + 1);
  static constexpr int kHist = MM == 2 ? 256 : 1, kWHist = MM == 2 ? NW * kSmallQ : 1;
  alignas(16) uint32_t par[ROWS * 32];
  uint32_t srow[ROWS];  // global index of each row word's first site
  // cluster draws of the tile: two-state draws, row r's 32 bits in word r;
  // Potts, row r's bytes 4j..4j+3 in word j*(ROWS+1)+r (row-thread stores
  // and lane reads both bank-conflict free)
  uint32_t sdraw[kDrawWords];
  uint32_t sX[ROWS], sY[ROWS];      // bonds along +x inside the word, +y inside the tile
  uint32_t sZ[S::D == 3 ? ROWS : 1];      // bonds along +z inside the tile
  // Potts histogram: per-warp bins for q <= kSmallQ, shared bins above
  unsigned int s_hist[kHist];
  unsigned int s_whist[kWHist];
  long long s_red[NW];
};

template <class Sh, int K, bool FROM_MASK, int MM, class Smem>
__device__ __forceinline__ void label_tile(const Lattice& lat, uint32_t tile, uint32_t sweep,
                                           const Measure& mb, Smem& sm) {
  constexpr bool MEASURE = MM == 1 || MM == 2;
  constexpr int D = Sh::D, TY = Sh::TY, TZ = Sh::TZ, ROWS = Sh::ROWS, NT = K * Sh::THREADS;
  constexpr int NW = NT / 32, RPW = ROWS / NW;
  static_assert(ROWS == Sh::THREADS && ROWS % 32 == 0, "K threads per row word, whole warps");
  static_assert(!(MEASURE && FROM_MASK), "measurement needs the spins");
  uint32_t* par = sm.par;
  uint32_t* sdraw = sm.sdraw;
  uint32_t* sX = sm.sX;
  uint32_t* sY = sm.sY;
  unsigned int* s_hist = sm.s_hist;
  unsigned int* s_whist = sm.s_whist;
  long long* s_red = sm.s_red;
  int m_acc = 0, e_acc = 0;
  if (MM == 2) {
    for (int k = threadIdx.x; k < 256; k += NT) s_hist[k] = 0u;
    for (int k = threadIdx.x; k < NW * kSmallQ; k += NT) s_whist[k] = 0u;
    __syncthreads();
  }

  const TileCoord tc = tile_coord<Sh>(lat, tile);
  const int L = lat.L;
  const uint32_t plane = lat.R * (uint32_t)lat.W;
  const int nvalid = min(32, L - tc.x0);
  const uint32_t vmask = (nvalid >= 32) ? kFull : ((1u << nvalid) - 1u);
  const bool draws = (sweep != 0u);
  const bool two_state = lat.dq == 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  // every run start is its own parent until the unions (other sites are
  // never looked up: a site's root is the root of its run start)
  {
    uint4* p4 = reinterpret_cast<uint4*>(par);
#pragma unroll
    for (int k = 0; k < ROWS * 32 / 4 / NT; ++k) {
      const uint32_t t = 4u * (uint32_t)(threadIdx.x + k * NT);
      p4[threadIdx.x + k * NT] = make_uint4(t, t + 1u, t + 2u, t + 3u);
    }
  }

  // global memory only after the preceding kernel of the sweep is done
  pdl_wait();

  // ---- phase 1: bonds, runs and draws of this thread's row word; with K > 1
  // the word's tasks (a bond direction each, then the draws) are dealt to its
  // K threads, which lie in different warps
  const int r = threadIdx.x & (ROWS - 1), part = K == 1 ? 0 : (int)threadIdx.x / ROWS;
  static_assert((ROWS & (ROWS - 1)) == 0, "rows by mask");
  const int ry = r % TY, rz = r / TY;
  const int y = tc.y0 + ry, z = tc.z0 + rz;
  const bool rowv = (y < L) && (D == 2 || z < L);
  const int y1 = (y + 1 == L) ? 0 : y + 1;
  const int z1 = (D == 3) ? ((z + 1 == L) ? 0 : z + 1) : 0;
  const bool in_y = y1 - tc.y0 >= 0 && y1 - tc.y0 < TY, in_z = D == 3 && z1 - tc.z0 >= 0 && z1 - tc.z0 < TZ;
  auto task = [&](int t) { return K == 1 || t % K == part; };
  uint32_t A0 = 0u, A1 = 0u, A2 = 0u;
  if (rowv) {
    const uint32_t row = (uint32_t)y + (uint32_t)L * (uint32_t)z;
    if (task(0)) sm.srow[r] = row * (uint32_t)L + (uint32_t)tc.x0;
    const uint32_t g = row * (uint32_t)lat.W + (uint32_t)tc.tx;
    if (FROM_MASK) {
      if (task(0)) A0 = __ldg(&lat.planes[g]) & vmask;
      if (task(1)) A1 = __ldg(&lat.planes[plane + g]) & vmask;
      if (D == 3 && task(2)) A2 = __ldg(&lat.planes[2 * plane + g]) & vmask;
    } else {
      const uint8_t* s = static_cast<const uint8_t*>(lat.spins);
      const bool vec16 = (L & 15) == 0;
      const uint32_t rowL = row * (uint32_t)L;
      const uint32_t row_y = (uint32_t)y1 + (uint32_t)L * (uint32_t)z;
      const uint32_t row_z = (uint32_t)y + (uint32_t)L * (uint32_t)z1;
      // equality masks (and the measurement) first, so the row bytes are
      // dead before the Bernoulli words are drawn
      uint32_t e0 = 0u, e1 = 0u, e2 = 0u;
      {
        uint32_t w[9];
        load32<true>(s, rowL + (uint32_t)tc.x0, vec16, w);
        if (MEASURE && task(D)) measure_state<MM>(w, vmask, nvalid, lat.q, m_acc, s_whist + warp * kSmallQ, s_hist);
        uint32_t n[8];
        if (task(1)) {
          load32<false>(s, row_y * (uint32_t)L + (uint32_t)tc.x0, vec16, n);
          e1 = eq_bits(w, n) & vmask;
        }
        if (D == 3 && task(2)) {
          load32<false>(s, row_z * (uint32_t)L + (uint32_t)tc.x0, vec16, n);
          e2 = eq_bits(w, n) & vmask;
        }
        if (task(0)) {
          shift_row(s, w, rowL, L, tc.x0, nvalid, n);
          e0 = eq_bits(w, n) & vmask;
        }
      }
      if (MEASURE) {
        const int par_bonds = __popc(e0) + __popc(e1) + (D == 3 ? __popc(e2) : 0);
        const int nbonds = (task(D) ? D : 0) * nvalid;  // counted once a row word
        e_acc += MM == 1 ? nbonds - 2 * par_bonds : nbonds - par_bonds;
      }
      if (e0) A0 = e0 & bernoulli_word(g, sweep, 0, lat.t_bond, e0, lat.rk);
      if (e1) A1 = e1 & bernoulli_word(g, sweep, 1, lat.t_bond, e1, lat.rk);
      if (D == 3 && e2) A2 = e2 & bernoulli_word(g, sweep, 2, lat.t_bond, e2, lat.rk);
      if (task(0)) lat.planes[g] = A0;
      if (task(1)) lat.planes[plane + g] = A1;
      if (D == 3 && task(2)) lat.planes[2 * plane + g] = A2;
    }
    if (draws && two_state) {
      // two-state cluster draws: bit (x & 31) of word 0 of Philox(g, sweep, DRAW, 1)
      if (task(D)) sdraw[r] = philox(g, sweep, kDraw, 1u, lat.rk).x;
    } else if (draws && Smem::kPottsDraws) {
      // Potts cluster draw of every site: word (i & 3) of Philox(i >> 2, sweep, DRAW, 0)
      const uint32_t i0 = row * (uint32_t)L + (uint32_t)tc.x0;
      const uint32_t dq = (uint32_t)lat.dq;
      if ((L & 3) == 0) {
        // L a multiple of 4 (the same branch for the whole lattice): the row
        // word starts a Philox group, and group j holds the draws of its
        // sites 4j..4j+3 (those past the end of the row go unused)
#pragma unroll 1
        for (int j = part; j < 8; j += K) {
          const uint4 w = philox((i0 >> 2) + (uint32_t)j, sweep, kDraw, 0u, lat.rk);
          sdraw[j * (ROWS + 1) + r] = draw_value(w.x, dq) | (draw_value(w.y, dq) << 8) |
                                      (draw_value(w.z, dq) << 16) | (draw_value(w.w, dq) << 24);
        }
      } else {
        uint32_t cached = 0xffffffffu;
        uint4 w = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
        for (int j = part * (8 / K); j < (part + 1) * (8 / K); ++j) {
          uint32_t packed = 0u;
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int b = 4 * j + t;
            if (b < nvalid) {
              const uint32_t i = i0 + (uint32_t)b;
              if ((i >> 2) != cached) {
                cached = i >> 2;
                w = philox(cached, sweep, kDraw, 0u, lat.rk);
              }
              packed |= draw_value(word_of(w, (int)(i & 3u)), dq) << (8 * t);
            }
          }
          sdraw[j * (ROWS + 1) + r] = packed;
        }
      }
    }
  }
  // x-bonds whose +x site is in the same word (and, for a one-word row, the
  // bond around it in bit 31: no bond inside the word has that bit), y- and
  // z-bonds inside the tile
  if (task(0)) {
    const bool around = tc.x0 == 0 && L <= 32 && ((A0 >> (L - 1)) & 1u);
    sX[r] = (A0 & (vmask >> 1)) | (around ? 0x80000000u : 0u);
  }
  if (task(1)) sY[r] = in_y ? A1 : 0u;
  if (D == 3 && task(2)) sm.sZ[r] = in_z ? A2 : 0u;
  __syncthreads();

  // ---- phase 2a: the first bond of every x-run to the rows before it hooks
  // the run's start there (a plain store: each start is written by its own
  // row's thread only, and its new parent has a smaller index)
  const uint32_t cap = lat.cap;
  uint32_t Y2 = 0u, Z2 = 0u, Sy = 0u, Sz = 0u, S = 0u, XW = 0u;
  constexpr uint32_t kInWord = 0x7fffffffu;
  // this thread's bits of the row word
  const uint32_t own_bits = K == 1 ? kFull : ((1u << (32 / K % 32)) - 1u) << (32 / K * part);
  if (rowv) {
    const uint32_t XX = sX[r], X = XX & kInWord;
    S = ~(X << 1) & vmask;  // x-run starts
    XW = XX >> 31;
    const uint32_t Yp = ry > 0 ? sY[r - 1] : 0u;
    const uint32_t Zp = (D == 3 && rz > 0) ? sm.sZ[r - TY] : 0u;
    const uint32_t joined = X << 1;  // bit b: site b is bonded to site b - 1
    uint32_t both = 0u;
    if (Yp) {
      const uint32_t Xn = sX[r - 1] & kInWord;
      Sy = ~(Xn << 1) & vmask;
      Y2 = Yp & ~((Yp & X & Xn) << 1);
    }
    if (D == 3 && Zp) {
      const uint32_t Xn = sX[r - TY] & kInWord;
      Sz = ~(Xn << 1) & vmask;
      Z2 = Zp & ~((Zp & X & Xn) << 1);
    }
    both = Y2 | Z2;
    // bits above the first one of their run: a carry from each bit runs up
    // the joined bits and stops at the end of the run
    const uint32_t seed = (both << 1) & joined;
    uint32_t F = both & ~((((seed + joined) ^ joined) | seed) & joined);
    Z2 &= ~(F & ~Y2);
    const uint32_t FY = F & Y2;
    Y2 &= ~F & own_bits;
    Z2 &= own_bits;
    F &= own_bits;
    while (F) {
      const int b = __ffs(F) - 1;
      F &= F - 1u;
      const bool y_bond = D == 2 || ((FY >> b) & 1u);
      par[32 * r + run_start(S, b)] =
          y_bond ? (uint32_t)(32 * (r - 1)) + run_start(Sy, b) : (uint32_t)(32 * (r - TY)) + run_start(Sz, b);
    }
  }
  __syncthreads();

  // ---- phase 2b: unions for the other in-tile bonds
  if (rowv) {
    while (Y2 | Z2) {
      const bool y_bond = D == 2 || Y2 != 0u;
      const uint32_t U = y_bond ? Y2 : Z2;
      const int b = __ffs(U) - 1;
      if (y_bond) Y2 &= Y2 - 1u;
      else Z2 &= Z2 - 1u;
      sunion(par, (uint32_t)(32 * r) + run_start(S, b),
             y_bond ? (uint32_t)(32 * (r - 1)) + run_start(Sy, b) : (uint32_t)(32 * (r - TY)) + run_start(Sz, b),
             lat.err, cap);
    }
    // bonds around the torus inside the tile (a lattice no longer than it)
    if (y1 < y && in_y) {
      const int rn = r + (y1 - y);
      const uint32_t Sn = ~(sX[rn] << 1) & vmask;
      for (uint32_t U = sY[r] & own_bits; U; U &= U - 1u) {
        const int b = __ffs(U) - 1;
        sunion(par, (uint32_t)(32 * r) + run_start(S, b), (uint32_t)(32 * rn) + run_start(Sn, b), lat.err, cap);
      }
    }
    if (D == 3 && z1 < z && in_z) {
      const int rn = r + TY * (z1 - z);
      const uint32_t Sn = ~(sX[rn] << 1) & vmask;
      for (uint32_t U = sm.sZ[r] & own_bits; U; U &= U - 1u) {
        const int b = __ffs(U) - 1;
        sunion(par, (uint32_t)(32 * r) + run_start(S, b), (uint32_t)(32 * rn) + run_start(Sn, b), lat.err, cap);
      }
    }
    if (XW && part == 0) sunion(par, (uint32_t)(32 * r) + run_start(S, L - 1), (uint32_t)(32 * r), lat.err, cap);
  }
  __syncthreads();

  // ---- phase 3: forest word of every site
  const uint32_t lr_bit = 1u << lat.sbits;
  const int shift = lat.sbits + 1;
  const int nrows_y = L - tc.y0, nrows_z = (D == 3) ? L - tc.z0 : 1;  // valid rows (at least)
  if ((L & 3) == 0) {
    // a thread per four consecutive sites: their walks advance together, one
    // 16-byte store.  Walked sites are stored at their roots while other
    // threads walk, without a barrier: a thread stores only to its own four
    // words, and whether a read gives the old word, the new one or one read
    // before, it is an ancestor of the same tree; roots store themselves.  So
    // every walk ends at the same root.  The reads are plain: volatile ones
    // keep the four walks' loads in program order (3D L = 256 146.7 -> 152.8 us
    // a sweep, 2D L = 4096 117.2 -> 128.5).
    const int b0 = 4 * (lane & 7);
#pragma unroll 1
    for (int k = 0; k < RPW / 4; ++k) {
      const int rr = 4 * (warp + NW * k) + (lane >> 3);
      if (b0 >= nvalid || rr % TY >= nrows_y || rr / TY >= nrows_z) continue;
      const uint32_t st = ~(sX[rr] << 1);
      const uint32_t t0 = (uint32_t)(32 * rr + b0);
      const uint4 own = *reinterpret_cast<const uint4*>(par + t0);
      uint32_t p[4];
      p[0] = ((st >> b0) & 1u) ? own.x : par[32 * rr + run_start(st, b0)];
      p[1] = ((st >> b0) & 2u) ? own.y : p[0];
      p[2] = ((st >> b0) & 4u) ? own.z : p[1];
      p[3] = ((st >> b0) & 8u) ? own.w : p[2];
      uint32_t moved = 1u;  // parents only decrease: at most a walk per site of the tile
      for (int it = 0; it < ROWS * 32 && moved; ++it) {
        moved = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t up = par[p[j]];
          moved |= up ^ p[j];
          p[j] = up;
        }
      }
      // the starts now point at their roots: rows are taken in rising order
      // and parents lie in earlier rows, so later walks are short (3D L = 256:
      // 70.8 M -> 67.3 M warp instructions, 88.5 -> 85.4 us)
      *reinterpret_cast<uint4*>(par + t0) = make_uint4(p[0], p[1], p[2], p[3]);
      const uint32_t dr = !draws ? 0u
                          : (two_state || !Smem::kPottsDraws) ? sdraw[rr] >> b0
                                                              : sdraw[(lane & 7) * (ROWS + 1) + rr];
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t draw = (two_state || !Smem::kPottsDraws) ? (dr >> j) & 1u : (dr >> (8 * j)) & 0xffu;
        const uint32_t gidx = sm.srow[p[j] >> 5] + (p[j] & 31u);
        w[j] = (gidx << shift) | (p[j] == t0 + (uint32_t)j ? lr_bit : 0u) | draw;
      }
      *reinterpret_cast<uint4*>(lat.forest + sm.srow[rr] + (uint32_t)b0) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  } else {
#pragma unroll 2
    for (int k = 0; k < RPW; ++k) {
      const int rr = warp + NW * k;
      if (lane >= nvalid || rr % TY >= nrows_y || rr / TY >= nrows_z) continue;
      const uint32_t st = ~(sX[rr] << 1);
      const uint32_t t = (uint32_t)(32 * rr + lane);
      const uint32_t lr = sfind(par, (uint32_t)(32 * rr) + run_start(st, lane));
      const uint32_t gidx = sm.srow[lr >> 5] + (lr & 31u);
      const uint32_t i = sm.srow[rr] + (uint32_t)lane;
      const uint32_t draw = !draws ? 0u
                            : (two_state || !Smem::kPottsDraws)
                                ? (sdraw[rr] >> lane) & 1u
                                : (sdraw[(lane >> 2) * (ROWS + 1) + rr] >> (8 * (lane & 3))) & 0xffu;
      lat.forest[i] = (gidx << shift) | (lr == t ? lr_bit : 0u) | draw;
    }
  }
  if (MEASURE) {
    if (MM == 2) {
      __syncthreads();
      for (int k = threadIdx.x; k < kSmallQ; k += NT)
        for (int w = 0; w < NW; ++w) s_hist[k] += s_whist[w * kSmallQ + k];
      __syncthreads();
      add_histogram(lat, mb, tile, s_hist);
    }
    add_integer_sums<NW>(mb, tile, (long long)m_acc, (long long)e_acc, s_red);
  }
}

// Threads of an SM the split labeling counts on (64 registers a thread).
constexpr int kLabelSplitThreads = 1024;

// K threads per row word (label_split).  K = 1: five 256-thread CTAs per SM,
// proportionally more of smaller tiles.
template <int D, int K, bool FROM_MASK, int MM>
__global__ void __launch_bounds__(K* Tile<D>::THREADS, K == 1 ? 5 * 256 / Tile<D>::THREADS : kLabelSplitThreads / (K * Tile<D>::THREADS))
    k_label(const __grid_constant__ Lattice lat, uint32_t sweep, const __grid_constant__ Measure mb) {
  __shared__ LabelSmem<Tile<D>, MM, K> sm;
  label_tile<Tile<D>, K, FROM_MASK, MM>(lat, blockIdx.x, sweep, mb, sm);
}

// Ising/Potts lattices of a batch, one tile of shape S per CTA; sweep
// numbers come from the batch step counter, and every step after the first
// (the first too when the member's last record is pending) also measures
// the incoming state of its lattice (the record of the previous sweep).  A
// member stops after its own number of sweeps.  The tile map lists the
// Ising members' tiles first.
// LAYOUT 1: Ising tiles only, two-state layout; LAYOUT 2: Potts tiles only;
// LAYOUT 3: any tile, Potts layout, the member's model picked per tile.
// Resident CTAs per SM: five 256-thread CTAs (two-state layout) or four
// (Potts layout), and proportionally more of smaller tiles.
constexpr int label_blocks(int threads, int layout) {
  return (layout == 1 ? 5 : 4) * 256 / threads > 32 ? 32 : (layout == 1 ? 5 : 4) * 256 / threads;
}

// One tile-map entry of a batch label launch: the member's lattice view is
// copied to shared memory (the Philox round keys are read on every round).
template <class S, int LAYOUT, class Smem>
__device__ __forceinline__ void label_batch_entry(const BatchView& bv, uint32_t e, uint32_t step, Smem& sm,
                                                  Lattice& s_lat) {
  static_assert(sizeof(Lattice) % 4 == 0, "lattice copy");
  const uint32_t b = __ldg(&bv.tile_lattice[e]);
  const uint32_t tile = __ldg(&bv.tile_index[e]);
  const BatchMember& m = bv.members[b];
  for (uint32_t k = threadIdx.x; k < sizeof(Lattice) / 4; k += S::THREADS)
    reinterpret_cast<uint32_t*>(&s_lat)[k] = reinterpret_cast<const uint32_t*>(&m.lat)[k];
  __syncthreads();
  if (step >= m.nsweeps) return;  // the member has had its sweeps this call
  const uint32_t sweep = m.sweep0 + step + 1u;
  const bool potts = LAYOUT == 2 || (LAYOUT == 3 && s_lat.model == kPotts);
  if (step == 0u && !m.measure0) label_tile<S, 1, false, 0>(s_lat, tile, sweep, m.meas, sm);
  else if (LAYOUT != 1 && potts) label_tile<S, 1, false, 2>(s_lat, tile, sweep, m.meas, sm);
  else if (LAYOUT != 2) label_tile<S, 1, false, 1>(s_lat, tile, sweep, m.meas, sm);
}

// PERSISTENT false: CTA k labels tile-map entry first + k (the grid covers
// the map).  PERSISTENT true: a grid of resident CTAs, each taking entries
// first + t for t = blockIdx.x, blockIdx.x + gridDim.x, ... below first + n.
// Separate instantiations, so that the loop costs the one-entry kernel no
// registers; the persistent one allows a quarter fewer CTAs per SM (its
// grid is sized by the occupancy it gets), so that its loop does not spill.
constexpr int persistent_blocks(int blocks) { return blocks * 3 / 4 > 1 ? blocks * 3 / 4 : 1; }

template <class S, int LAYOUT, bool PERSISTENT>
__global__ void __launch_bounds__(S::THREADS, PERSISTENT ? persistent_blocks(label_blocks(S::THREADS, LAYOUT))
                                                         : label_blocks(S::THREADS, LAYOUT))
    k_label_batch(BatchView bv, uint32_t first, uint32_t n) {
  __shared__ LabelSmem<S, LAYOUT == 1 ? 1 : 2> sm;
  __shared__ Lattice s_lat;
  pdl_wait();
  const uint32_t step = *bv.step;
  if constexpr (PERSISTENT) {
    for (uint32_t t = blockIdx.x; t < n; t += gridDim.x) {
      __syncthreads();  // the previous entry's readers of s_lat and sm are done
      label_batch_entry<S, LAYOUT>(bv, first + t, step, sm, s_lat);
    }
  } else {
    label_batch_entry<S, LAYOUT>(bv, first + blockIdx.x, step, sm, s_lat);
  }
}

// Stand-alone measurement of an Ising (MM 1) or Potts (MM 2) state as the
// record of `sweep`: a thread per 32-site row word (grid-stride), the
// labeling kernel's row loads and equality masks, sums added to the
// measurement slots by block; the last block to finish (a counter) writes
// the record and the FP64 accumulators from the complete slots.
template <int D, int MM>
__global__ void __launch_bounds__(256) k_measure_rows(const __grid_constant__ Lattice lat,
                                                      const __grid_constant__ Measure mb, uint32_t sweep) {
  constexpr int NW = 256 / 32;
  __shared__ unsigned int s_hist[MM == 2 ? 256 : 1];
  __shared__ unsigned int s_whist[MM == 2 ? NW * kSmallQ : 1];
  __shared__ long long s_red[NW];
  __shared__ double s_rd[NW];
  __shared__ bool s_last;
  const int warp = threadIdx.x >> 5;
  if (MM == 2) {
    for (int k = threadIdx.x; k < 256; k += 256) s_hist[k] = 0u;
    for (int k = threadIdx.x; k < NW * kSmallQ; k += 256) s_whist[k] = 0u;
    __syncthreads();
  }
  const int L = lat.L;
  const uint32_t words = lat.R * (uint32_t)lat.W;
  int m_acc = 0, e_acc = 0;
  // L a power of two (then so is W): indices by shifts and masks
  const bool pow2 = (L & (L - 1)) == 0;
  const int lsh = __ffs(L) - 1, wsh = __ffs(lat.W) - 1;
  for (uint32_t g = blockIdx.x * 256u + threadIdx.x; g < words; g += gridDim.x * 256u) {
    uint32_t row, tx, y, z;
    if (pow2) {
      row = g >> wsh;
      tx = g & (uint32_t)(lat.W - 1);
      y = row & (uint32_t)(L - 1);
      z = row >> lsh;
    } else {
      row = g / (uint32_t)lat.W;
      tx = g % (uint32_t)lat.W;
      y = row % (uint32_t)L;
      z = row / (uint32_t)L;
    }
    const int x0 = 32 * (int)tx;
    const int nvalid = min(32, L - x0);
    const uint32_t vmask = (nvalid >= 32) ? kFull : ((1u << nvalid) - 1u);
    const uint32_t y1 = (y + 1u == (uint32_t)L) ? 0u : y + 1u;
    const uint32_t z1 = (D == 3) ? ((z + 1u == (uint32_t)L) ? 0u : z + 1u) : 0u;
    RowBytes rb;
    load_rows<D>(static_cast<const uint8_t*>(lat.spins), L, x0, nvalid, row, y1 + (uint32_t)L * z, y + (uint32_t)L * z1, rb);
    const uint32_t e0 = eq_bits(rb.a, rb.ax) & vmask;
    const uint32_t e1 = eq_bits(rb.a, rb.ay) & vmask;
    const uint32_t e2 = (D == 3) ? (eq_bits(rb.a, rb.az) & vmask) : 0u;
    measure_row<D, MM>(rb, e0, e1, e2, vmask, nvalid, lat.q, m_acc, e_acc, s_whist + warp * kSmallQ, s_hist);
  }
  if (MM == 2) {
    __syncthreads();
    for (int k = threadIdx.x; k < kSmallQ; k += 256)
      for (int w = 0; w < NW; ++w) s_hist[k] += s_whist[w * kSmallQ + k];
    __syncthreads();
    add_histogram(lat, mb, blockIdx.x, s_hist);
  }
  add_integer_sums<NW>(mb, blockIdx.x, (long long)m_acc, (long long)e_acc, s_red);
  // this block's slot additions are visible before it counts itself done
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(mb.done, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  finalize_record<NW>(lat, mb, sweep, s_red, s_rd);
  if (threadIdx.x == 0) *mb.done = 0u;
}

// Stand-alone measurement of every tiled member of a batch that had sweeps in
// the current call, as the record of its last one: a CTA per tile-map entry,
// k_measure_rows' work on the tile's rows; the last of a member's CTAs to
// finish writes its record.
template <class S>
__global__ void __launch_bounds__(S::THREADS) k_measure_batch(BatchView bv) {
  constexpr int D = S::D, NT = S::THREADS, NW = NT / 32;
  __shared__ unsigned int s_hist[256];
  __shared__ unsigned int s_whist[NW * kSmallQ];
  __shared__ long long s_red[NW];
  __shared__ double s_rd[NW];
  __shared__ bool s_last;
  const BatchMember& m = bv.members[__ldg(&bv.tile_lattice[blockIdx.x])];
  if (m.nsweeps == 0u) return;  // its record is written, or was pending before the call
  const Lattice lat = m.lat;    // a private copy: global stores cannot alias it
  const Measure mb = m.meas;
  const uint32_t tile = __ldg(&bv.tile_index[blockIdx.x]);
  const TileCoord tc = tile_coord<S>(lat, tile);
  const bool potts = lat.model == kPotts;
  const int L = lat.L, warp = threadIdx.x >> 5;
  for (int k = threadIdx.x; k < 256; k += NT) s_hist[k] = 0u;
  for (int k = threadIdx.x; k < NW * kSmallQ; k += NT) s_whist[k] = 0u;
  __syncthreads();
  const int r = threadIdx.x, y = tc.y0 + r % S::TY, z = tc.z0 + r / S::TY;
  int m_acc = 0, e_acc = 0;
  if (y < L && (D == 2 || z < L)) {
    const int nvalid = min(32, L - tc.x0);
    const uint32_t vmask = (nvalid >= 32) ? kFull : ((1u << nvalid) - 1u);
    const int y1 = (y + 1 == L) ? 0 : y + 1, z1 = (D == 3) ? ((z + 1 == L) ? 0 : z + 1) : 0;
    RowBytes rb;
    load_rows<D>(static_cast<const uint8_t*>(lat.spins), L, tc.x0, nvalid, (uint32_t)y + (uint32_t)L * (uint32_t)z,
                 (uint32_t)y1 + (uint32_t)L * (uint32_t)z, (uint32_t)y + (uint32_t)L * (uint32_t)z1, rb);
    const uint32_t e0 = eq_bits(rb.a, rb.ax) & vmask;
    const uint32_t e1 = eq_bits(rb.a, rb.ay) & vmask;
    const uint32_t e2 = (D == 3) ? (eq_bits(rb.a, rb.az) & vmask) : 0u;
    if (potts) measure_row<D, 2>(rb, e0, e1, e2, vmask, nvalid, lat.q, m_acc, e_acc, s_whist + warp * kSmallQ, s_hist);
    else measure_row<D, 1>(rb, e0, e1, e2, vmask, nvalid, lat.q, m_acc, e_acc, s_whist + warp * kSmallQ, s_hist);
  }
  if (potts) {
    __syncthreads();
    for (int k = threadIdx.x; k < kSmallQ; k += NT)
      for (int w = 0; w < NW; ++w) s_hist[k] += s_whist[w * kSmallQ + k];
    __syncthreads();
    add_histogram(lat, mb, tile, s_hist);
  }
  add_integer_sums<NW>(mb, tile, (long long)m_acc, (long long)e_acc, s_red);
  // this CTA's slot additions are visible before it counts itself done
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(mb.done, 1u) == (uint32_t)(lat.ntx * lat.nty * lat.ntz) - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  finalize_record<NW>(lat, mb, m.sweep0 + m.nsweeps, s_red, s_rd);
  if (threadIdx.x == 0) *mb.done = 0u;
}

// ---------------------------------------------------------------- XY bonds
// 1 + the top 23 bits of w as a fraction (a bit pattern: no conversion, which
// would share the exp's pipe).
__device__ __forceinline__ float unit_bits(uint32_t w) { return __uint_as_float(0x3f800000u | (w >> 9)); }

// 2^x, within 2^-22 relative (the hardware approximation).
__device__ __forceinline__ float fast_exp2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// One CTA per 32 x BY (x BZ) block of sites, grid-strided over the blocks.
// The projections (x, y) = (cos, sin)(theta - phi) on the sweep's mirror
// axis are computed once per site of the block and its +x/+y/+z halo into
// shared memory; bond (i,d) is active iff x_i x_j > 0 and the uniform of
// word d of Philox(i, sweep, BOND, 0) is below 1 - exp(-2K x_i x_j); warps
// ballot their rows into the bit-planes.  With MEASURE the same values
// measure the incoming state (the state after sweep - 1): sum x, sum y and
// the bond energies x_i x_j + y_i y_j (cos(theta_i - theta_j), invariant
// under the rotation by phi) in float per thread, then double per block;
// the block's (sum cos theta, sum sin theta, E) partial, rotated back by
// phi, goes to slot blockIdx of the XY partials.
template <int D>
struct XYBlock;
template <>
struct XYBlock<2> {
  static constexpr int BY = 128, BZ = 1;
};
template <>
struct XYBlock<3> {
  static constexpr int BY = 16, BZ = 8;
};

//
// The kernel is issue-bound (65% of issue slots): a lane's Philox word and its
// sincosf are about half of its instructions, so the rest was cut -- the bond
// decision without an integer conversion, a warp's row coordinates by
// constants, and its bond words kept a lane per row and stored once per block
// instead of a predicated store per row and direction.  3D L = 256: 145.1 M ->
// 117.0 M warp instructions, 183.1 -> 150.6 us measured, 173.8 -> 139.9 not;
// the sweep 307 -> 273 us.
//
// CTAs per SM of the one-wave grid.  Fixed, not asked of the occupancy
// calculator: the partial sums of the measurement are added in an order that
// depends on the grid.
constexpr int kXYBlocksPerSM[2] = {6, 5};

// K > 1: K times the threads for lattices with fewer blocks than SMs, where
// the kernel is one warp's chain of rows.  A block's rows are dealt to the K
// sets of warps; the first set then adds the moments alone, in K = 1's order,
// so the sums are the same bits.  3D L = 16 (two blocks): 18.0 -> 10.5 us, 22.4
// -> 16.5 with the moments.
template <int D, int K, bool MEASURE>
__global__ void __launch_bounds__(256 * K, K == 1 ? kXYBlocksPerSM[D - 2] : 1)
    k_bonds_xy(const __grid_constant__ Lattice lat, uint32_t sweep, const __grid_constant__ Measure mb) {
  constexpr int BY = XYBlock<D>::BY, BZ = XYBlock<D>::BZ;
  constexpr int HX = 33, HY = BY + 1, HZ = (D == 3) ? BZ + 1 : 1, NBOX = HX * HY * HZ;
  constexpr int NW = 256 / 32, RW = BY * BZ / NW;  // rows per warp
  static_assert(BY % NW == 0 && RW <= 32 && RW % K == 0, "a lane per row of the warp");
  __shared__ float2 sv[NBOX];
  __shared__ float s_phi;
  __shared__ double s_rd[K * NW];
  if (threadIdx.x == 0) s_phi = xy_phi(lat, sweep);
  pdl_wait();
  __syncthreads();
  const float phi = s_phi;
  const float kexp = -__fmul_rn(lat.twoK, 0x1.715476p+0f);  // -2K log2 e
  const int L = lat.L, lane = threadIdx.x & 31, warp = K == 1 ? threadIdx.x >> 5 : (threadIdx.x >> 5) & (NW - 1);
  const int set = K == 1 ? 0 : threadIdx.x / (32 * NW);
  const uint32_t plane = lat.R * (uint32_t)lat.W;
  const float* th = static_cast<const float*>(lat.spins);
  const uint32_t nbx = (uint32_t)lat.W, nby = (uint32_t)((L + BY - 1) / BY);
  const uint32_t nbz = (D == 3) ? (uint32_t)((L + BZ - 1) / BZ) : 1u;
  const uint32_t nblocks = nbx * nby * nbz;
  float fx = 0.f, fy = 0.f, fe = 0.f;
  for (uint32_t t = blockIdx.x; t < nblocks; t += gridDim.x) {
    const int x0 = 32 * (int)(t % nbx), y0 = BY * (int)((t / nbx) % nby), z0 = BZ * (int)(t / (nbx * nby));
    const int nx = min(32, L - x0), ny = min(BY, L - y0), nz = (D == 3) ? min(BZ, L - z0) : 1;
    __syncthreads();  // the previous block's values are no longer read
    auto project = [&](int yy, int zz, int xx) {
      int gx = x0 + xx, gy = y0 + yy, gz = (D == 3) ? z0 + zz : 0;
      if (gx >= L) gx -= L;
      if (gy >= L) gy -= L;
      if (D == 3 && gz >= L) gz -= L;
      float sn, cs;
      sincosf(__fsub_rn(__ldg(&th[(uint32_t)gx + (uint32_t)L * ((uint32_t)gy + (uint32_t)L * (uint32_t)gz)]),
                        phi), &sn, &cs);
      sv[(yy + HY * zz) * HX + xx] = make_float2(cs, sn);
    };
    // a warp per halo row (yy, zz), lanes along x; then the +x halo column
    // (entry 32 of every row) a thread per row
    if (lane <= nx)
      for (int yy = K == 1 ? warp : (warp + NW * set) % HY, zz = K == 1 ? 0 : (warp + NW * set) / HY;
           zz < HZ && zz <= nz;) {
        if (yy <= ny) project(yy, zz, lane);
        yy += K * NW;
        if (K == 1) {
          if (yy >= HY) {
            yy -= HY;
            ++zz;
          }
        } else {
          while (yy >= HY) {
            yy -= HY;
            ++zz;
          }
        }
      }
    if (nx == 32)
      for (int hr = threadIdx.x; hr < HY * HZ; hr += 256 * K) {
        const int yy = hr % HY, zz = hr / HY;
        if (yy <= ny && zz <= nz) project(yy, zz, 32);
      }
    __syncthreads();
    // a warp's rows in turn, row k = (warp + 8 (k mod BY / 8), k / (BY / 8));
    // lane k keeps row k's bond words
    uint32_t m[D];
#pragma unroll
    for (int d = 0; d < D; ++d) m[d] = 0u;
    const uint32_t i0 = (uint32_t)(x0 + lane) + (uint32_t)L * ((uint32_t)(y0 + warp) + (uint32_t)L * (uint32_t)z0);
    constexpr int RY = BY / NW;  // rows of the warp per z
#pragma unroll 2
    for (int k = set; k < RW; k += K) {
      const int yy = warp + NW * (k % RY), zz = k / RY;
      bool act[D];
#pragma unroll
      for (int d = 0; d < D; ++d) act[d] = false;
      if (yy < ny && zz < nz && lane < nx) {
        const uint32_t i = i0 + (uint32_t)L * ((uint32_t)(NW * (k % RY)) + (uint32_t)L * (uint32_t)zz);
        const uint4 w = philox(i, sweep, kBond, 0u, lat.rk);
        const int c = lane + HX * (yy + HY * zz);
        const float2 si = sv[c];
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const float2 sj = sv[c + (d == 0 ? 1 : d == 1 ? HX : HX * HY)];
          const float prod = __fmul_rn(si.x, sj.x);
          // u < p with p = -expm1f(-2K prod), u = (w >> 8) 2^-24: the sign
          // of (1 + u) + exp(-2K prod) - 2 decides, with u cut to 23 bits
          // and the hardware's 2^x, unless it lies within a margin far above
          // their error (below 5.5e-7, as for the clock bonds), where expm1f
          // decides
          const float near = __fsub_rn(
              __fadd_rn(unit_bits(word_of(w, d)), fast_exp2(__fmul_rn(kexp, prod))), 2.0f);
          act[d] = prod > 0.0f && near < 0.0f;
          if (prod > 0.0f && fabsf(near) <= 0x1p-16f) {
            const float u = __fmul_rn((float)(word_of(w, d) >> 8), 0x1p-24f);
            act[d] = u < -expm1f(-__fmul_rn(lat.twoK, prod));
          }
          if (MEASURE && K == 1) fe = __fadd_rn(fe, __fadd_rn(prod, __fmul_rn(si.y, sj.y)));
        }
        if (MEASURE && K == 1) {
          fx = __fadd_rn(fx, si.x);
          fy = __fadd_rn(fy, si.y);
        }
      }
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const uint32_t bal = __ballot_sync(kFull, act[d]);
        if (lane == k) m[d] = bal;
      }
    }
    {
      const int yy = warp + NW * (lane % RY), zz = lane / RY;
      if (lane < RW && (K == 1 || lane % K == set) && yy < ny && zz < nz) {
        const uint32_t g = ((uint32_t)(y0 + yy) + (uint32_t)L * (uint32_t)(z0 + zz)) * (uint32_t)lat.W + (uint32_t)(x0 >> 5);
#pragma unroll
        for (int d = 0; d < D; ++d) lat.planes[d * plane + g] = m[d];
      }
    }
    if (MEASURE && K > 1 && set == 0 && lane < nx) {
#pragma unroll 2
      for (int k = 0; k < RW; ++k) {
        const int yy = warp + NW * (k % RY), zz = k / RY;
        if (yy >= ny || zz >= nz) continue;
        const int c = lane + HX * (yy + HY * zz);
        const float2 si = sv[c];
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const float2 sj = sv[c + (d == 0 ? 1 : d == 1 ? HX : HX * HY)];
          fe = __fadd_rn(fe, __fadd_rn(__fmul_rn(si.x, sj.x), __fmul_rn(si.y, sj.y)));
        }
        fx = __fadd_rn(fx, si.x);
        fy = __fadd_rn(fy, si.y);
      }
    }
  }
  if (MEASURE) {
    const double sx = block_combine<NW>((double)warp_sum(fx), s_rd);
    const double sy = block_combine<NW>((double)warp_sum(fy), s_rd);
    const double se = block_combine<NW>((double)warp_sum(fe), s_rd);
    if (threadIdx.x == 0) {
      const double c = cos((double)phi), sn = sin((double)phi);
      mb.part_d[3 * blockIdx.x + 0] = __dsub_rn(__dmul_rn(c, sx), __dmul_rn(sn, sy));
      mb.part_d[3 * blockIdx.x + 1] = __dadd_rn(__dmul_rn(sn, sx), __dmul_rn(c, sy));
      mb.part_d[3 * blockIdx.x + 2] = -se;
    }
  }
}

// ---------------------------------------------------------------- clock bonds
// q-state clock: x_i = sin(pi k_i / q), k_i = (2 p_i - s) mod 2q for the
// sweep's mirror index s; bond (i,d) active iff u(i,d) < t[k_i][k_j] (the
// table is 0 where x_i x_j <= 0); u(i,d) = word d of Philox(i, sweep, BOND, 0).
// The comparison is decided from a float estimate of u - t (the projections in
// shared memory, the hardware's 2^x) unless it lies within a margin far above
// the estimate's error, where the exact table entry decides: the result is
// the table's, without a table gather per bond.
// With MEASURE the same loads measure the incoming state: integer sums of
// the fixed-point tables C[p_i], S[p_i] and C[(p_i - p_j) mod q], added to
// the clock slots per block.
//
// CTAs per SM of the one-wave grid, update only and measured: what registers
// (32 and 40) and shared memory (8 and 24 KB) allow.  Fixed, not asked of the
// occupancy calculator, which every sweep's launch would wait for.
constexpr int kClockBlocksPerSM[2] = {8, 6};

template <int D, bool MEASURE>
__global__ void __launch_bounds__(256, kClockBlocksPerSM[MEASURE]) k_bonds_clock(const __grid_constant__ Lattice lat, uint32_t sweep,
                                                      const __grid_constant__ Measure mb) {
  __shared__ uint32_t s_mirror;
  __shared__ long long s_red[256 / 32];
  __shared__ float s_x[2 * kMaxClockQ];
  // the fixed-point cos / sin tables of the measurement (gathered per site)
  __shared__ long long s_fix[MEASURE ? 2 * kMaxClockQ : 1];
  if (threadIdx.x == 0) s_mirror = clock_mirror(lat, sweep);
  pdl_wait();
  const int L = lat.L, lane = threadIdx.x & 31;
  const int q = lat.q, q2 = 2 * q;
  for (int k = threadIdx.x; k < q2; k += 256) {
    s_x[k] = __ldg(&lat.cproj[k]);
    if (MEASURE) s_fix[k] = __ldg(&mb.cfix[k]);
  }
  __syncthreads();
  // Error of the estimate below of u - t/2^32: 2^-23 for the draw cut to 23
  // bits, 2^-22 for the hardware's 2^x, 2^-23 for the addition, and seven
  // roundings of the exponent (2K, log2 e, two projections, three products),
  // 2^-24 of a each, which e^-a turns into at most 2^-24 / e each: below
  // 6.4e-7.  The margin is 24 times that and more, and draws inside it read
  // the exact entry.
  const float margin = __fadd_rn(0x1p-16f, __fmul_rn(lat.twoK, 0x1p-20f));
  const float kexp = -__fmul_rn(lat.twoK, 0x1.715476p+0f);  // -2K log2 e
  const int mirror = (int)s_mirror;
  const uint32_t nwords = lat.R * (uint32_t)lat.W;
  const uint32_t plane = nwords;
  const uint16_t* sp = static_cast<const uint16_t*>(lat.spins);
  const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
  long long cx = 0, sy = 0, eb = 0;
  // L a power of two (then so is W): a row word's indices by shifts and
  // masks instead of four divisions (the same branch for the whole lattice)
  const bool pow2 = (L & (L - 1)) == 0;
  const int lsh = __ffs(L) - 1, wsh = __ffs(lat.W) - 1;
  for (uint32_t g = gw; g < nwords; g += nw) {
    uint32_t row, xw, y, z;
    if (pow2) {
      row = g >> wsh;
      xw = g & (uint32_t)(lat.W - 1);
      y = row & (uint32_t)(L - 1);
      z = row >> lsh;
    } else {
      row = g / (uint32_t)lat.W;
      xw = g % (uint32_t)lat.W;
      y = row % (uint32_t)L;
      z = row / (uint32_t)L;
    }
    const int x = (int)(32 * xw) + lane;
    uint32_t a = 0u;
    if (x < L) {
      const uint32_t i = (uint32_t)x + (uint32_t)L * row;
      const uint4 w = philox(i, sweep, kBond, 0u, lat.rk);
      uint32_t jn[3];
      jn[0] = (x + 1 == L) ? i - (uint32_t)x : i + 1u;
      jn[1] = (y + 1 == (uint32_t)L) ? i - y * L : i + (uint32_t)L;
      jn[2] = (D == 3) ? ((z + 1 == (uint32_t)L) ? i - z * L * L : i + (uint32_t)L * L) : 0u;
      const int pi = clock_state(sp[i], q);
      const int ki = wrap_mod(2 * pi - mirror, q2);
      if (MEASURE) {
        cx += s_fix[pi];
        sy += s_fix[q + pi];
      }
      const float xi = s_x[ki];
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const int pj = clock_state(sp[jn[d]], q);
        const int kj = wrap_mod(2 * pj - mirror, q2);
        // the table entry is 0 where x_i x_j <= 0 (the sign of a float
        // product is the exact one; |x| >= sin(pi/q) off k = 0, q)
        const float prod = __fmul_rn(xi, s_x[kj]);
        bool act = false;
        if (prod > 0.0f) {
          const uint32_t wd = word_of(w, d);
          const float near = __fsub_rn(__fadd_rn(unit_bits(wd), fast_exp2(__fmul_rn(kexp, prod))), 2.0f);
          act = (fabsf(near) > margin) ? near < 0.0f
                                       : wd < __ldg(&lat.ctab[(size_t)ki * (size_t)q2 + (size_t)kj]);
        }
        a |= (uint32_t)act << d;
        if (MEASURE) eb += s_fix[wrap_mod(pi - pj, q)];
      }
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const uint32_t bal = __ballot_sync(kFull, (a >> d) & 1u);
      if (lane == d) lat.planes[d * plane + g] = bal;
    }
  }
  if (MEASURE) add_clock_sums<256 / 32>(mb, blockIdx.x, cx, sy, eb, s_red);
}

}  // namespace

cudaError_t launch_bonds_clock(const Lattice& lat, uint32_t sweep, const Measure* m, cudaStream_t st) {
  const uint32_t words = lat.R * (uint32_t)lat.W;
  // a warp per row word, striding over them; the sums are exact integers, so
  // the grid changes no result.  Few row words: one wave of CTAs, each filling
  // its tables (12 KB at q = 512) once; many: up to 4096 CTAs, whose unequal
  // ends the next ones fill.  us per measured sweep, one wave / 4096: 3D L = 64
  // q = 512 (8192 row words) 28.1 / 29.3, 128 (65536) 58.5 / 60.5, 2D L = 1448
  // (66608) 53.3 / 56.5, 3D q = 6 L = 129 (83205) 74.9 / 75.5, 144 (103680) 82.5
  // / 81.6, 160 (128000) 97.7 / 95.1, 200 (280000) 179.1 / 170.6, 400 1177 /
  // 1100; 2D L = 8000 974 / 892.
  constexpr uint32_t kWaveWords = 3u << 15;
  const uint32_t ctas = (words + 7u) / 8u;
  const uint32_t most = words <= kWaveWords ? (uint32_t)(sm_count() * kClockBlocksPerSM[m != nullptr]) : 4096u;
  const unsigned g = ctas < most ? ctas : most;
  auto launch = [&](auto kernel, const Measure& mm) { return launch_pdl(kernel, g, 256, st, lat, sweep, mm); };
  const Measure none{};
  if (lat.dim == 2) return m ? launch(k_bonds_clock<2, true>, *m) : launch(k_bonds_clock<2, false>, none);
  return m ? launch(k_bonds_clock<3, true>, *m) : launch(k_bonds_clock<3, false>, none);
}

void tiles_for(int dim, int L, int* ntx, int* nty, int* ntz, int shape) {
  if (shape < 0) shape = kSingleShape[dim - 2];
  const int ty = kShapeTY[dim - 2][shape], tz = kShapeTZ[dim - 2][shape];
  *ntx = (L + 31) / 32;
  *nty = (L + ty - 1) / ty;
  *ntz = (dim == 2) ? 1 : (L + tz - 1) / tz;
}

// Threads per row word of a lattice's labeling: the most (4, 2 or 1) with
// which the GPU holds all tiles at once.  With few tiles the kernel is a chain
// of latencies -- a thread's three Bernoulli words, its hooks and unions, its
// rows' walks -- and the threads added shorten every link; once the tiles
// come in waves the extra row-word arithmetic only costs.  us per sweep with
// 1, 2 and 4 threads: 2D L = 128 27.9 / 22.5 / 20.4, 515 32.2 / 26.6 / 24.1,
// 1024 (256 tiles) 31.1 / 27.7 / 27.4, 1448 (552) 36.7 / 33.9 / 38.9; 3D L =
// 32 29.8 / 27.1 / 26.9, 100 (196 tiles of twice the size) 41.5 / 40.1 /
// 43.2, 128 (256) 44.2 / 43.1 / 50.1, 161 (726) 68.9 / 71.7 / 84.3.
int tile_split(const Lattice& lat) {
  const int tiles = lat.ntx * lat.nty * lat.ntz;
  const int threads = kShapeTY[lat.dim - 2][kSingleShape[lat.dim - 2]] * kShapeTZ[lat.dim - 2][kSingleShape[lat.dim - 2]];
  const int whole = sm_count() * (kLabelSplitThreads / threads);  // tiles held at one thread a row word
  return 4 * tiles <= whole ? 4 : 2 * tiles <= whole ? 2 : 1;
}

namespace {

template <int D, bool FROM_MASK, int MM>
cudaError_t launch_label_kernel(const Lattice& lat, uint32_t sweep, const Measure& m, cudaStream_t st) {
  const unsigned g = (unsigned)(lat.ntx * lat.nty * lat.ntz), t = (unsigned)Tile<D>::THREADS;
  switch (tile_split(lat)) {
    case 4: return launch_pdl(k_label<D, 4, FROM_MASK, MM>, g, 4 * t, st, lat, sweep, m);
    case 2: return launch_pdl(k_label<D, 2, FROM_MASK, MM>, g, 2 * t, st, lat, sweep, m);
    default: return launch_pdl(k_label<D, 1, FROM_MASK, MM>, g, t, st, lat, sweep, m);
  }
}

template <int D>
cudaError_t launch_label_dim(const Lattice& lat, uint32_t sweep, bool from_mask, bool potts_draws,
                             cudaStream_t st) {
  const Measure none{};
  if (from_mask) {
    if (potts_draws) return launch_label_kernel<D, true, 3>(lat, sweep, none, st);
    return launch_label_kernel<D, true, 0>(lat, sweep, none, st);
  }
  if (potts_draws) return launch_label_kernel<D, false, 3>(lat, sweep, none, st);
  return launch_label_kernel<D, false, 0>(lat, sweep, none, st);
}
}  // namespace

cudaError_t launch_label(const Lattice& lat, uint32_t sweep, bool from_mask, cudaStream_t st) {
  // the Potts layout (a draw byte per site in shared memory) only where
  // Potts draws are made; two-state draws or none take the smaller layout
  const bool potts_draws = sweep != 0u && lat.dq != 2;
  if (lat.dim == 2) return launch_label_dim<2>(lat, sweep, from_mask, potts_draws, st);
  return launch_label_dim<3>(lat, sweep, from_mask, potts_draws, st);
}

namespace {

// Schedule bit 0: Ising and Potts tiles in one launch (Potts layout) or
// two; bit 1: persistent grids (batch_grid).
template <class S, int LAYOUT>
cudaError_t label_batch_launch(const BatchView& bv, uint32_t first, uint32_t n, bool persistent,
                               cudaStream_t st) {
  if (!persistent) return launch_pdl(k_label_batch<S, LAYOUT, false>, n, (unsigned)S::THREADS, st, bv, first, n);
  const unsigned g = batch_grid(k_label_batch<S, LAYOUT, true>, S::THREADS, n);
  return launch_pdl(k_label_batch<S, LAYOUT, true>, g, (unsigned)S::THREADS, st, bv, first, n);
}

template <int D, int SH>
cudaError_t label_batch_shape(const BatchView& bv, int schedule, uint32_t ising_tiles, uint32_t potts_tiles,
                              cudaStream_t st) {
  using S = ShapeOf<D, SH>;
  const bool persistent = (schedule & 2) != 0;
  if ((schedule & 1) && ising_tiles && potts_tiles)
    return label_batch_launch<S, 3>(bv, 0u, ising_tiles + potts_tiles, persistent, st);
  cudaError_t e = cudaSuccess;
  if (ising_tiles) e = label_batch_launch<S, 1>(bv, 0u, ising_tiles, persistent, st);
  if (e == cudaSuccess && potts_tiles) e = label_batch_launch<S, 2>(bv, ising_tiles, potts_tiles, persistent, st);
  return e;
}

template <int D>
cudaError_t label_batch_dim(const BatchView& bv, int shape, int schedule, uint32_t ising_tiles,
                            uint32_t potts_tiles, cudaStream_t st) {
  if (shape == 1) return label_batch_shape<D, 1>(bv, schedule, ising_tiles, potts_tiles, st);
  if (shape == 2) return label_batch_shape<D, 2>(bv, schedule, ising_tiles, potts_tiles, st);
  return label_batch_shape<D, 0>(bv, schedule, ising_tiles, potts_tiles, st);
}

}  // namespace

cudaError_t launch_label_batch(const BatchView& bv, int dim, int shape, int schedule, uint32_t ising_tiles,
                               uint32_t potts_tiles, cudaStream_t st) {
  static_assert(kTileShapes == 3, "one instantiation per shape");
  if (dim == 2) return label_batch_dim<2>(bv, shape, schedule, ising_tiles, potts_tiles, st);
  return label_batch_dim<3>(bv, shape, schedule, ising_tiles, potts_tiles, st);
}

cudaError_t launch_measure_batch(const BatchView& bv, int dim, int shape, uint32_t ntiles, cudaStream_t st) {
  static_assert(kTileShapes == 3, "one instantiation per shape");
  auto one = [&](auto kernel, int threads) {
    kernel<<<ntiles, (unsigned)threads, 0, st>>>(bv);
    return cudaGetLastError();
  };
  if (dim == 2) {
    if (shape == 1) return one(k_measure_batch<ShapeOf<2, 1>>, ShapeOf<2, 1>::THREADS);
    if (shape == 2) return one(k_measure_batch<ShapeOf<2, 2>>, ShapeOf<2, 2>::THREADS);
    return one(k_measure_batch<ShapeOf<2, 0>>, ShapeOf<2, 0>::THREADS);
  }
  if (shape == 1) return one(k_measure_batch<ShapeOf<3, 1>>, ShapeOf<3, 1>::THREADS);
  if (shape == 2) return one(k_measure_batch<ShapeOf<3, 2>>, ShapeOf<3, 2>::THREADS);
  return one(k_measure_batch<ShapeOf<3, 0>>, ShapeOf<3, 0>::THREADS);
}

cudaError_t launch_measure_rows(const Lattice& lat, uint32_t sweep, const Measure& m, cudaStream_t st) {
  const uint32_t words = lat.R * (uint32_t)lat.W;
  unsigned g = (words + 255u) / 256u;
  if (g > (unsigned)kMeasureBlocks) g = (unsigned)kMeasureBlocks;
  if (g == 0) g = 1;
  const bool potts = lat.model == kPotts;
  if (lat.dim == 2) {
    if (potts) k_measure_rows<2, 2><<<g, 256, 0, st>>>(lat, m, sweep);
    else k_measure_rows<2, 1><<<g, 256, 0, st>>>(lat, m, sweep);
  } else {
    if (potts) k_measure_rows<3, 2><<<g, 256, 0, st>>>(lat, m, sweep);
    else k_measure_rows<3, 1><<<g, 256, 0, st>>>(lat, m, sweep);
  }
  return cudaGetLastError();
}

cudaError_t launch_label_measured(const Lattice& lat, uint32_t sweep, const Measure& m,
                                  cudaStream_t st) {
  const bool potts = lat.model == kPotts;
  if (lat.dim == 2)
    return potts ? launch_label_kernel<2, false, 2>(lat, sweep, m, st)
                 : launch_label_kernel<2, false, 1>(lat, sweep, m, st);
  return potts ? launch_label_kernel<3, false, 2>(lat, sweep, m, st)
               : launch_label_kernel<3, false, 1>(lat, sweep, m, st);
}

cudaError_t launch_bonds_xy(const Lattice& lat, uint32_t sweep, const Measure* m, int* blocks,
                            cudaStream_t st) {
  const uint32_t ny = (uint32_t)((lat.L + XYBlock<3>::BY - 1) / XYBlock<3>::BY);
  const uint32_t nb = (lat.dim == 2)
                          ? (uint32_t)lat.W * (uint32_t)((lat.L + XYBlock<2>::BY - 1) / XYBlock<2>::BY)
                          : (uint32_t)lat.W * ny * (uint32_t)((lat.L + XYBlock<3>::BZ - 1) / XYBlock<3>::BZ);
  // one wave: the CTAs the GPU holds at once, each striding over the blocks;
  // at most kMeasureBlocks (the slots of the XY partials)
  unsigned g = 0;
  g = (unsigned)(sm_count() * kXYBlocksPerSM[lat.dim - 2]);
  if (g > nb) g = nb;
  if (g > (unsigned)kMeasureBlocks) g = (unsigned)kMeasureBlocks;
  // the threads of four blocks for each where every block has an SM of its own
  const bool split = nb <= (uint32_t)sm_count();
  auto launch = [&](auto kernel, auto wide, const Measure& mm) {
    return split ? launch_pdl(wide, g, 1024, st, lat, sweep, mm) : launch_pdl(kernel, g, 256, st, lat, sweep, mm);
  };
  cudaError_t e = cudaSuccess;
  const Measure none{};
  if (lat.dim == 2) {
    if (m) e = launch(k_bonds_xy<2, 1, true>, k_bonds_xy<2, 4, true>, *m);
    else e = launch(k_bonds_xy<2, 1, false>, k_bonds_xy<2, 4, false>, none);
  } else {
    if (m) e = launch(k_bonds_xy<3, 1, true>, k_bonds_xy<3, 4, true>, *m);
    else e = launch(k_bonds_xy<3, 1, false>, k_bonds_xy<3, 4, false>, none);
  }
  if (blocks) *blocks = (int)g;
  return e;
}

}  // namespace swgb
