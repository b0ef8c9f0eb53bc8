// kite_resident.cuh -- the 1D moment sweep of a mid-size lattice held on chip by the whole
// GPU: one cooperative launch runs every recursion step of a batch (Eqs. e6-e8).
//
// The lattice is cut as the streaming kernels cut it: strips of TX cells, row segments as
// work units in strip order, and a range of units per (virtual) CTA of the streaming grid.
// One SM owns the units of a few consecutive virtual CTAs, its region: a block of rows of
// one strip, or the end of one strip and the beginning of the next.  It keeps r_n and
// r_{n-1} of the region in shared memory, each with a frame of one halo cell, and the
// on-site terms beside them; r_0 as far as it fits, the rest of it is read from L2.  r_{n+1}
// overwrites r_{n-1} in place.
//
// Per step the compute threads (one per column of a virtual CTA, sublattice and unit of a
// sweep's vectors) march down their rows with the next row's operands in flight, while 256 exchange
// threads (1) compute the region's edge sites once more, with their r_{n-1} in registers, and
// send them at once, (2) add up the moment partials of the step before, (3) receive the
// neighbours' edge sites into the frame.  The exchange's latency thus lies beside the march.
// No grid-wide barrier and no fence: a unit travels as 8-byte words of 32 data bits and the
// 32-bit step number, so a word that carries the step's number carries its data (8-byte
// accesses are single copies).
// The records are double-buffered by step parity: a region sends r_{n+1} only after it has
// received all of its neighbours' r_n, which they sent after they had received r_{n-1}, so
// the record that r_{n+1} overwrites has been read.  (A flag per region behind a release
// fence, with the halo read after an acquire, took 9.5 us per step whatever the size.)
//
// Results: the site update is the streaming kernels' rounding sequence, so the iterates are
// the same bits; and each FP32 moment sum runs over the same sites in the same order as in
// the streaming launch it stands in for (a virtual CTA's rows of one column, promoted to
// FP64 every kRFlush rows), so the moments agree with that launch's to the rounding of FP64
// sums.  As there, the FP32 sweeps form the imaginary part too and the FP64 sweeps do not.
//
// What bounds it: the march, by shared-memory wavefronts and issue slots (five 16-byte loads
// and a store per chunk), with the exchange (1.4-1.7 us: edge sites, one flight through L2, a
// poll) beside it.  Per recursion step of the batch, against the streaming kernels' launch,
// ring fill and CTA reduction per step: honeycomb 257 x 510, R = 8 FP32 14.6 -> 5.0 us (two
// sweeps of four vectors), 512 x 601 in a field, R = 4 17.4 -> 5.9 us, 300 x 300, R = 8
// 11.4 -> 3.8 us; 64 x 64, R = 4 FP64 1.6-1.9 us against the cluster sweep's 2.2 us.  In units
// of one complex FP32 vector, orbital updates per second: square 1024 x 1024, R = 4
// 1.94e11 -> 4.65e11, R = 8 2.36e11 -> 3.77e11, 957 x 957, R = 4 1.78e11 -> 4.31e11, 1200 x 1200
// 1.95e11 -> 2.55e11 (r_0 from L2), honeycomb 800 x 800 2.04e11 -> 2.45e11.  Which runs is
// measured (resident_choice in kite_kpm1d.cu).
//
// The plans and the launches are kite_resident.cu's, with the FP32 kernels; the FP64 kernels are
// kite_resident64.cu's: a program loads a translation unit's kernels together, and all of them in
// one took 16 ms of the first on-chip sweep, 2 ms in two.
#pragma once
#include <math.h>

#include "kite_device.cuh"
#include "kite_internal.h"

namespace kite {
namespace {

constexpr int kRMax = 256;     // most compute threads of a CTA (512 threads: 128 registers each)
constexpr int kRComm = 256;    // exchange threads
// Most edge sites, and most halo chunks, of one exchange thread: kRSites, or kRFew where a plan's
// lists are short enough.  Fewer of them leave the exchange warps less to carry along: 64 x 64
// honeycomb cells, FP64, R = 4, M = 256 578 -> 562 us a call, 200 x 200, FP32, R = 4 589 -> 577.
constexpr int kRSites = 3, kRFew = 2;
constexpr int kRMaxV = 64;     // most virtual CTAs of a region
constexpr int kRFlush = 32;    // rows of one FP32 moment sum (the streaming kernels' kFlushRows)
constexpr int kResSmem = 227 * 1024 - 512;  // (the rest: static shared memory)

// The unit of a sweep's vectors: a 16-byte chunk of the batch layout (two complex FP32 or one
// complex FP64 vector), or half of one in FP32.  Half chunks let lattices of twice the size
// stay on chip, one complex vector per sweep.
struct alignas(8) HalfChunk {
  static constexpr int kReals = 2;
  static constexpr int kVecs = 1;
  float v[2];
  __device__ __forceinline__ static HalfChunk ldg(const void* base, size_t idx) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(base) + idx);
    HalfChunk c;
    c.v[0] = t.x;
    c.v[1] = t.y;
    return c;
  }
  __device__ __forceinline__ void st(void* base, size_t idx) const {
    reinterpret_cast<float2*>(base)[idx] = make_float2(v[0], v[1]);
  }
};
template <typename Real, int CBY>
struct ResUnit {
  using T = Chunk<Real>;
};
template <>
struct ResUnit<float, 8> {
  using T = HalfChunk;
};

// One record: a unit's data as 8-byte words of (32 data bits, step number), moved by one
// 32-byte (half chunks: 16-byte) access.
template <int W>
struct alignas(8 * W) Rec {
  unsigned long long w[W];
};
template <int W>
__device__ __forceinline__ void send_rec(Rec<W>* p, const uint32_t (&d)[W], uint32_t step) {
  const unsigned long long h = (unsigned long long)step << 32;
  if constexpr (W == 4)
    asm volatile("st.relaxed.gpu.global.v4.u64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(h | d[0]), "l"(h | d[1]),
                 "l"(h | d[2]), "l"(h | d[3])
                 : "memory");
  else
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(h | d[0]), "l"(h | d[1]) : "memory");
}
template <int W>
__device__ __forceinline__ Rec<W> load_rec(const Rec<W>* p) {
  Rec<W> r;
  if constexpr (W == 4)
    asm volatile("ld.relaxed.gpu.global.v4.u64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(r.w[0]), "=l"(r.w[1]), "=l"(r.w[2]), "=l"(r.w[3])
                 : "l"(p)
                 : "memory");
  else
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(r.w[0]), "=l"(r.w[1]) : "l"(p) : "memory");
  return r;
}
template <int W>
__device__ __forceinline__ bool rec_ready(const Rec<W>& r, uint32_t step) {
  bool ok = true;
#pragma unroll
  for (int i = 0; i < W; ++i) ok = ok && (uint32_t)(r.w[i] >> 32) == step;
  return ok;
}

template <typename Real>
struct ResArgs {
  const void* r0;     // batch layout [cell][sublattice][C units]
  const Real* vt;     // 2 V~ per orbital, NaN on vacancies
  const Real* phase;  // [Ly][sublattice][2][2] (cos, sin), field only
  void* last[2];      // r_last: the last two iterates in the batch layout, r_n in last[n & 1]
  double* part;       // moment partials [slot n][CTA][exchange warps][32 >> levels]
  void* rec;          // edge records [parity][cell][sublattice][CR units]
  volatile int* err;  // host memory: 1 when a wait gave up
  Real tt;
  int Lx, Ly, TX, G;  // strip width, virtual CTAs
  int rows_max, nv_max, nfl, r0_rows, levels;
  int C, c0, CR;      // units per orbital of the batch, first unit and units of this sweep
  int steps, open_x, open_y, stall;
  int write_last;
};

// Shared-memory carve, the same on host and device: offsets in bytes.
struct ResSmem {
  int x0, x1, r0, vt, phase, sums, total;
};
__host__ __device__ inline ResSmem res_smem(int cby, int sorb, int CR, int TX, int rows, int nv, int nfl, int real_bytes,
                                            int nsums, int dbl, int r0_rows, int field) {
  ResSmem s;
  const int cellb = sorb * CR * cby, frame = (rows + 4) * (TX + 2);
  int off = 0;
  auto take = [&](int bytes) {
    const int at = off;
    off += (bytes + 127) & ~127;
    return at;
  };
  s.x0 = take(frame * cellb);
  s.x1 = take(frame * cellb);
  s.vt = take(rows * TX * sorb * real_bytes);
  s.phase = take(field ? rows * sorb * 4 * real_bytes : 0);
  s.sums = take((dbl ? 4 : 2) * nv * nfl * TX * sorb * CR * nsums * real_bytes);  // of two steps
  s.r0 = take(r0_rows * TX * cellb);
  s.total = off;
  return s;
}

// VAR 0: complex vectors, 1: complex vectors in a magnetic field, 2: real vectors.
template <typename Real, int CBY, int LAT, bool DBL, int VAR, int SITES>
__global__ void __launch_bounds__(kRMax + kRComm, 1) k_resident(const ResArgs<Real> a) {
  using Ch = typename ResUnit<Real, CBY>::T;
  constexpr int W = CBY / 4;  // words of a record
  constexpr int SORB = LAT == KITE_HONEYCOMB ? 2 : 1;
  constexpr int NR = Ch::kReals, VPC = Ch::kVecs;
  constexpr bool IM = sizeof(Real) == 4 && VAR != 2;          // real and imaginary parts
  constexpr int NV = VAR == 2 ? NR : (IM ? 2 * VPC : VPC);    // moment sums per chunk
  constexpr int SETS = DBL ? 2 : 1;        // <.|r_{n+1}>, and <r_n|r_n> with doubling
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int s_abort, s_vrow[kRMaxV + 1];  // first local row of each virtual CTA
  const int T = (int)blockDim.x - kRComm;  // compute threads
  const int tid = threadIdx.x, cta = blockIdx.x;
  const int CR = a.CR, TPC = SORB * CR, TX = a.TX, colT = TX * TPC;
  const ResSmem sm = res_smem(CBY, SORB, CR, TX, a.rows_max, a.nv_max, a.nfl, (int)sizeof(Real), NV, DBL, a.r0_rows,
                              VAR == 1);
  // r_n and r_{n-1} are kept by sublattice, [sublattice][framed cell][chunk]: a warp's lanes
  // hold one sublattice of a row (where a row of TX * CR chunks fills whole warps)
  const int P = TX + 2, CB = CR * CBY, PB = P * CB;   // framed row; bytes of a cell, of a framed row
  const int PS = (a.rows_max + 4) * PB;              // bytes of a sublattice
  // the region: virtual CTAs v0 .. v1-1, units U0 .. U0+nrows-1, in one or two segments
  const long long units = (long long)((a.Lx + TX - 1) / TX) * a.Ly;
  const int v0 = (int)((long long)a.G * cta / gridDim.x), v1 = (int)((long long)a.G * (cta + 1) / gridDim.x);
  const long long U0 = units * v0 / a.G;
  const int nrows = (int)(units * v1 / a.G - U0);
  const int sx = (int)(U0 / a.Ly), yb = (int)(U0 - (long long)sx * a.Ly);
  const int nr0 = min(nrows, a.Ly - yb), nr1 = nrows - nr0;
  // segment g: strip sx + g, first row (g ? 0 : yb), owned rows local 0 .. and frame row base
  auto seg_tx = [&](int g) { return min(TX, a.Lx - (sx + g) * TX); };
  auto row_y = [&](int r) { return r < nr0 ? yb + r : r - nr0; };
  auto frame_row = [&](int r) { return r < nr0 ? r + 1 : r + 3; };
  Real* vts = reinterpret_cast<Real*>(smem + sm.vt);
  Real* phs = reinterpret_cast<Real*>(smem + sm.phase);
  Real* sums = reinterpret_cast<Real*>(smem + sm.sums);  // [parity][set][(j, flush, column)][NV]
  const int nsum = a.nv_max * a.nfl * colT * NV;          // of one set

  auto wrap = [](int v, int L) { return v < 0 ? v + L : (v >= L ? v - L : v); };
  // lattice cell of segment g's local (lx, ly), -1 across an open boundary
  auto lattice_cell = [&](int g, int lx, int ly) -> int {
    const int x = (sx + g) * TX + lx, y = (g ? 0 : yb) + ly;
    if ((a.open_x && (x < 0 || x >= a.Lx)) || (a.open_y && (y < 0 || y >= a.Ly))) return -1;
    return wrap(y, a.Ly) * a.Lx + wrap(x, a.Lx);
  };
  auto frame_cell = [&](int g, int lx, int ly) { return ((g ? nr0 + 2 : 0) + ly + 1) * P + lx + 1; };

  for (int i = tid; i < nrows * TX * SORB; i += blockDim.x) {
    const int r = i / (TX * SORB), k = i - r * TX * SORB, lx = k / SORB, s = k - lx * SORB;
    const int g = r < nr0 ? 0 : 1;
    if (lx < seg_tx(g))
      vts[(s * a.rows_max + r) * TX + lx] = a.vt[((size_t)row_y(r) * a.Lx + (sx + g) * TX + lx) * SORB + s];
  }
  if (VAR == 1)
    for (int i = tid; i < nrows * SORB * 4; i += blockDim.x) {
      const int r = i / (SORB * 4);
      phs[i] = a.phase[(size_t)row_y(r) * SORB * 4 + (i - r * SORB * 4)];
    }
  for (int i = tid; i < SETS * 2 * nsum; i += blockDim.x) sums[i] = Real(0);
  if (tid == 0) s_abort = 0;
  if (tid <= v1 - v0) s_vrow[tid] = (int)(units * (v0 + tid) / a.G - U0);
  // r_0 with its frame; the other buffer starts at zero (open boundaries keep it so)
  for (int g = 0; g < (nr1 ? 2 : 1); ++g) {
    const int w = seg_tx(g) + 2, h = (g ? nr1 : nr0) + 2;
    for (int i = tid; i < w * h * TPC; i += blockDim.x) {
      const int f = i / TPC, k = i - f * TPC;
      const int ly = f / w - 1, lx = f - (ly + 1) * w - 1;
      const int s = k / CR, c = k - s * CR;
      const int at = s * PS + frame_cell(g, lx, ly) * CB + c * CBY;
      const int q = lattice_cell(g, lx, ly);
      Ch z, r;
#pragma unroll
      for (int e = 0; e < NR; ++e) z.v[e] = r.v[e] = Real(0);
      if (q >= 0) r = Ch::ldg(a.r0, ((size_t)q * SORB + s) * a.C + a.c0 + c);
      *reinterpret_cast<Ch*>(smem + sm.x0 + at) = r;
      *reinterpret_cast<Ch*>(smem + sm.x1 + at) = z;
      if (!DBL && lx >= 0 && lx < w - 2 && ly >= 0 && ly < h - 2) {
        const int row = (g ? nr0 : 0) + ly;
        if (row < a.r0_rows) reinterpret_cast<Ch*>(smem + sm.r0)[((s * a.r0_rows + row) * TX + lx) * CR + c] = r;
      }
    }
  }
  unsigned char* const xb = smem + sm.x0;
  const int xd = sm.x1 - sm.x0;
  const Real tt = a.tt, tt2 = a.tt + a.tt;

  // byte offsets of the neighbours of a site of sublattice s from its own chunk
  struct Nb {
    int o1, o2, o3, o4;
  };
  auto offsets = [&](int s) {
    Nb b;
    if (LAT == KITE_HONEYCOMB) {
      b.o1 = s == 0 ? PS : -PS;
      b.o3 = b.o1 + (s == 0 ? -PB : PB);
      b.o2 = b.o3 + (s == 0 ? CB : -CB);
      b.o4 = 0;
    } else {
      b.o1 = -CB;
      b.o2 = CB;
      b.o3 = -PB;
      b.o4 = PB;
    }
    return b;
  };
  auto ld = [](const unsigned char* p) { return *reinterpret_cast<const Ch*>(p); };
  // the streaming kernels' site update; ph: the site's two bond rotations (field)
  auto update = [&](auto first_tag, Ch n1, Ch n2, Ch n3, const Ch& n4, const Ch& me, const Ch& pv, Real v,
                    const Real* ph) -> Ch {
    constexpr bool FIRST = decltype(first_tag)::value;
    if constexpr (VAR == 1) {
      auto rot = [&](Ch& x, Real cph, Real sph) {
#pragma unroll
        for (int q = 0; q < VPC; ++q) {
          const Real re = x.v[2 * q], im = x.v[2 * q + 1];
          x.v[2 * q] = rfma(cph, re, -rmul(sph, im));
          x.v[2 * q + 1] = rfma(sph, re, rmul(cph, im));
        }
      };
      if (LAT == KITE_HONEYCOMB) {
        rot(n2, ph[0], ph[1]);
        rot(n3, ph[2], ph[3]);
      } else {
        rot(n1, ph[0], ph[1]);
        rot(n2, ph[2], ph[3]);
      }
    }
    const bool vacant = is_vacancy(v);
    Ch out;
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      Real sum = radd(n1.v[q], n2.v[q]);
      sum = radd(sum, n3.v[q]);
      if (LAT == KITE_SQUARE) sum = radd(sum, n4.v[q]);
      const Real o = FIRST ? rfma(tt, sum, rmul(Real(0.5) * v, me.v[q])) : rfma(tt2, sum, rfma(v, me.v[q], -pv.v[q]));
      out.v[q] = vacant ? Real(0) : o;
    }
    return out;
  };
  __syncthreads();

  if (tid >= T) {  // ---- exchange threads
    const int ct = tid - T, lane = ct & 31, warp = ct >> 5;
    const size_t half = (size_t)a.Lx * a.Ly * TPC;  // records per parity
    // edge sites (sent) and halo chunks (received) of this thread: smem offset, record
    int e_off[SITES], h_off[SITES], e_row[SITES];
    unsigned e_rec[SITES], h_rec[SITES];
    Real e_v[SITES];
    Ch e_prev[SITES];
    unsigned e_on = 0, h_on = 0, e_s = 0;
    {
      int off = 0, hoff = 0;  // list positions of the segment's first entry
      for (int g = 0; g < (nr1 ? 2 : 1); ++g) {
        const int w = seg_tx(g), h = g ? nr1 : nr0, base = g ? nr0 : 0;
        // honeycomb: A along the first row and the last column, B along the last row and the
        // first column; square: the four sides
        const int len = LAT == KITE_HONEYCOMB ? 2 * (w + h - 1) : 2 * (w + h);
#pragma unroll
        for (int u = 0; u < SITES; ++u) {
          const int j = ct + u * kRComm, e = j / CR - off, c = j - (j / CR) * CR;
          if (e < 0 || e >= len) continue;
          int lx, ly, s = 0;
          if (LAT == KITE_HONEYCOMB) {
            const int hl = w + h - 1, k = e < hl ? e : e - hl;
            s = e < hl ? 0 : 1;
            if (s == 0) lx = k < w ? k : w - 1, ly = k < w ? 0 : k - w + 1;
            else lx = k < w ? k : 0, ly = k < w ? h - 1 : k - w;
          } else {
            if (e < 2 * w) lx = e >> 1, ly = (e & 1) ? h - 1 : 0;
            else lx = (e & 1) ? w - 1 : 0, ly = (e - 2 * w) >> 1;
          }
          e_on |= 1u << u;
          e_s |= (unsigned)s << u;
          e_off[u] = s * PS + frame_cell(g, lx, ly) * CB + c * CBY;
          e_row[u] = base + ly;
          e_v[u] = vts[(s * a.rows_max + base + ly) * TX + lx];
          e_rec[u] = (unsigned)((lattice_cell(g, lx, ly) * SORB + s) * CR + c);
        }
        off += len;
        const int hlen = 2 * (w + h);
#pragma unroll
        for (int u = 0; u < SITES; ++u) {
          const int j = ct + u * kRComm, e = j / CR - hoff, c = j - (j / CR) * CR;
          if (e < 0 || e >= hlen) continue;
          int lx, ly, s = 0;
          if (LAT == KITE_HONEYCOMB) {
            const int k = e < w + h ? e : e - (w + h);
            if (e < w + h) {  // B above (and above right), then B right
              s = 1;
              lx = k <= w ? k : w;
              ly = k <= w ? -1 : k - w - 1;
            } else {  // A below (and below left), then A left
              lx = k <= w ? k - 1 : -1;
              ly = k <= w ? h : k - w;
            }
          } else {
            if (e < 2 * w) lx = e >> 1, ly = (e & 1) ? h : -1;
            else lx = (e & 1) ? w : -1, ly = (e - 2 * w) >> 1;
          }
          const int q = lattice_cell(g, lx, ly);
          if (q < 0) continue;
          h_on |= 1u << u;
          h_off[u] = s * PS + frame_cell(g, lx, ly) * CB + c * CBY;
          h_rec[u] = (unsigned)((q * SORB + s) * CR + c);
        }
        hoff += hlen;
      }
    }
    const Nb nb0 = offsets(0), nb1 = offsets(1);
    const bool mute = a.stall && cta == 0;
    auto send_edges = [&](int n, auto first_tag) {
      const unsigned char* cur = xb + (n & 1) * xd;
      Rec<W>* dst = static_cast<Rec<W>*>(a.rec) + ((n + 1) & 1) * half;
#pragma unroll
      for (int u = 0; u < SITES; ++u) {
        if (!(e_on >> u & 1)) continue;
        const Nb nb = (e_s >> u & 1) ? nb1 : nb0;
        const unsigned char* p = cur + e_off[u];
        const Ch me = ld(p);
        Ch n4 = me;
        if (LAT == KITE_SQUARE) n4 = ld(p + nb.o4);
        const Ch out = update(first_tag, ld(p + nb.o1), ld(p + nb.o2), ld(p + nb.o3), n4, me, e_prev[u], e_v[u],
                              phs + (e_row[u] * SORB + (int)(e_s >> u & 1)) * 4);
        e_prev[u] = me;
        if (!mute) send_rec<W>(dst + e_rec[u], *reinterpret_cast<const uint32_t(*)[W]>(&out), (uint32_t)(n + 1));
      }
    };
    // FP64 sums of step n's partials: each thread every kRComm-th entry (its own (chunk, sum)
    // class), then `levels` folds inside the warp
    const int keep = 32 >> a.levels;
    const size_t pstep = (size_t)gridDim.x * (kRComm / 32) * keep;
    double* pp = a.part + ((size_t)cta * (kRComm / 32) + warp) * keep + lane;
    auto add_sums = [&](int n) {  // (plain: n = -1 is <r_0|r_0>)
      const Real* src = sums + (size_t)(n & 1) * SETS * nsum;
#pragma unroll
      for (int set = 0; set < SETS; ++set) {
        double d = 0.0;
        for (int e = ct; e < nsum; e += kRComm) d += (double)src[set * nsum + e];
        for (int l = 0, o = 16; l < a.levels; ++l, o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane < keep) pp[(size_t)(DBL ? 2 * n + 1 - set : n + 1) * pstep] = d;
      }
    };
    __syncthreads();  // <r_0|r_0> is in the sums of step -1
    for (int n = 0; n < a.steps; ++n) {
      bool ok = true;
      if (n + 1 < a.steps) {
        if (n == 0) send_edges(n, std::true_type{});
        else send_edges(n, std::false_type{});
      }
      if (n > 0 || !DBL) add_sums(n - 1);
      if (n + 1 < a.steps) {
        const uint32_t step = (uint32_t)(n + 1);
        unsigned char* nxt = xb + ((n + 1) & 1) * xd;
        const Rec<W>* src = static_cast<const Rec<W>*>(a.rec) + ((n + 1) & 1) * half;
        unsigned want = h_on;
        const long long t0 = clock64();
        while (want) {
          Rec<W> d[SITES];
#pragma unroll
          for (int u = 0; u < SITES; ++u)
            if (want >> u & 1) d[u] = load_rec(src + h_rec[u]);
#pragma unroll
          for (int u = 0; u < SITES; ++u)
            if ((want >> u & 1) && rec_ready(d[u], step)) {
              Ch x;
              uint32_t(&xw)[W] = *reinterpret_cast<uint32_t(*)[W]>(&x);
#pragma unroll
              for (int i = 0; i < W; ++i) xw[i] = (uint32_t)d[u].w[i];
              *reinterpret_cast<Ch*>(nxt + h_off[u]) = x;
              want &= ~(1u << u);
            }
          if (want && clock64() - t0 > kWaitCycles) {
            ok = false;
            break;
          }
        }
      }
      if (!ok) s_abort = 1;
      __syncthreads();  // r_{n+1} complete in the region and its frame
      if (s_abort) {
        if (ct == 0) *a.err = 1;
        return;
      }
    }
    add_sums(a.steps - 1);
    return;
  }

  // ---- compute threads
  const int col = tid % colT, s = col / (TX * CR), xc = col - s * TX * CR, xl = xc / CR, c = xc - xl * CR;
  const int jstep = T / colT, jfirst = tid < jstep * colT ? tid / colT : v1 - v0;
  const Nb nb = offsets(s);
  const bool tx_on0 = xl < seg_tx(0), tx_on1 = nr1 && xl < seg_tx(1);
  const size_t gstep = (size_t)a.Lx * SORB * a.C;

  if constexpr (!DBL) {  // <r_0|r_0>, grouped as the other moments (real part)
    Real* out_sums = sums + nsum;
    for (int j = jfirst; j < v1 - v0; j += jstep) {
      const int re = s_vrow[j + 1];
      Real f[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) f[q] = Real(0);
      int rows = 0, fl = 0;
      auto flush = [&]() {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          out_sums[((size_t)(j * a.nfl + fl) * colT + col) * NV + q] = f[q];
          f[q] = Real(0);
        }
        rows = 0;
        ++fl;
      };
      for (int r = s_vrow[j]; r < re; ++r) {
        if (!(r < nr0 ? tx_on0 : tx_on1)) continue;
        const Ch me = ld(xb + s * PS + (frame_row(r) * P + xl + 1) * CB + c * CBY);
#pragma unroll
        for (int q = 0; q < NV; ++q) {
          const int v = IM ? q >> 1 : q;
          if (VAR == 2) f[q] = rfma(me.v[q], me.v[q], f[q]);
          else if (!IM || !(q & 1)) f[q] = rfma(me.v[2 * v + 1], me.v[2 * v + 1], rfma(me.v[2 * v], me.v[2 * v], f[q]));
        }
        if (++rows == kRFlush) flush();
      }
      if (rows) flush();
    }
  }
  __syncthreads();

  // rows [r, rend) of segment g in one column, S the sublattice (a template argument: the
  // carried neighbour is the first or the third of the sum)
  Real f0[NV], f1[NV];       // FP32 (FP64) sums since the last flush, over `rows` rows
  int rows = 0;
  Real* sum_at = nullptr;    // where the next flush goes
  auto flush = [&]() {
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      sum_at[q] = f0[q];
      if (DBL) sum_at[(SETS - 1) * nsum + q] = f1[q];
      f0[q] = f1[q] = Real(0);
    }
    rows = 0;
    sum_at += colT * NV;
  };
  auto march = [&](auto first_tag, auto s_tag, const unsigned char* cur, unsigned char* nxt, int g, int r, int rend) {
    constexpr bool FIRST = decltype(first_tag)::value;
    constexpr int S = decltype(s_tag)::value;
    int at = s * PS + (frame_row(r) * P + xl + 1) * CB + c * CBY;
    const Real* pv_v = vts + (s * a.rows_max + r) * TX + xl;
    const Ch* pr = reinterpret_cast<const Ch*>(smem + sm.r0) + ((s * a.r0_rows + r) * TX + xl) * CR + c;
    size_t gq = (((size_t)row_y(r) * a.Lx + (sx + g) * TX + xl) * SORB + s) * a.C + a.c0 + c;
    const Real* ph = phs + (r * SORB + s) * 4;
    // honeycomb: B(x,y-1) for A, A(x,y) for B; square: the upper and the own value
    Ch up, mid;
    if (LAT == KITE_HONEYCOMB) up = ld(cur + at + (S == 0 ? nb.o3 : nb.o1));
    else up = ld(cur + at + nb.o3), mid = ld(cur + at);
    auto row = [&](Ch na, Ch nbv, Ch nc, const Ch& pv, Ch z0, Real v, int at_, const Real* ph_) {
      Ch n1, n2, n3, n4, me;
      if (LAT == KITE_HONEYCOMB) {  // na: B(x,y) for A, A(x,y+1) for B
        n1 = S == 0 ? na : up;
        n3 = S == 0 ? up : na;
        up = na;
        n2 = nbv;
        me = n4 = nc;
      } else {  // left, right, below
        n1 = na;
        n2 = nbv;
        n3 = up;
        me = mid;
        n4 = nc;
        up = mid;
        mid = nc;
      }
      const Ch out = update(first_tag, n1, n2, n3, n4, me, pv, v, ph_);
      *reinterpret_cast<Ch*>(nxt + at_) = out;
      const Ch& l = (DBL || FIRST) ? me : z0;  // the bra: <r_n| with doubling, else <r_0|
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        if (VAR == 2) {
          f0[q] = rfma(l.v[q], out.v[q], f0[q]);
          if (DBL) f1[q] = rfma(l.v[q], l.v[q], f1[q]);
        } else {
          const int w = IM ? q >> 1 : q;  // conj(bra) ket, as in the streaming kernels' cacc
          const Real br = l.v[2 * w], bi = l.v[2 * w + 1], kr = out.v[2 * w], ki = out.v[2 * w + 1];
          if (!IM || !(q & 1)) {
            f0[q] = rfma(bi, ki, rfma(br, kr, f0[q]));
            if (DBL) f1[q] = rfma(bi, bi, rfma(br, br, f1[q]));
          } else {
            f0[q] = rfma(-bi, kr, rfma(br, ki, f0[q]));
          }
        }
      }
      if (++rows == kRFlush) flush();
    };
    auto oa = (LAT == KITE_HONEYCOMB && S == 1) ? nb.o3 : nb.o1;
    auto oc = LAT == KITE_HONEYCOMB ? 0 : nb.o4;
    // two rows' operands in flight; the rows whose r_0 is off chip apart (their loads take an
    // L2 round trip)
    auto run = [&](const int end, const bool on_chip) {
      for (; r + 1 < end; r += 2) {
        const unsigned char *p = cur + at, *p1 = p + PB;
        const Ch a0 = ld(p + oa), b0 = ld(p + nb.o2), c0_ = ld(p + oc), a1 = ld(p1 + oa), b1 = ld(p1 + nb.o2),
                 c1 = ld(p1 + oc);
        Ch q0, q1;
        if (!FIRST) q0 = ld(nxt + at), q1 = ld(nxt + at + PB);
        Ch z0, z1;
        if (!FIRST && !DBL) {
          z0 = on_chip ? pr[0] : Ch::ldg(a.r0, gq);
          z1 = on_chip ? pr[TX * CR] : Ch::ldg(a.r0, gq + gstep);
        }
        const Real va = pv_v[0], vb = pv_v[TX];
        row(a0, b0, c0_, q0, z0, va, at, ph);
        row(a1, b1, c1, q1, z1, vb, at + PB, ph + SORB * 4);
        at += 2 * PB;
        pv_v += 2 * TX;
        pr += 2 * TX * CR;
        gq += 2 * gstep;
        ph += 2 * SORB * 4;
      }
      if (r < end) {
        const unsigned char* p = cur + at;
        Ch q0, z0;
        if (!FIRST) q0 = ld(nxt + at);
        if (!FIRST && !DBL) z0 = on_chip ? pr[0] : Ch::ldg(a.r0, gq);
        row(ld(p + oa), ld(p + nb.o2), ld(p + oc), q0, z0, *pv_v, at, ph);
        ++r;
        at += PB;
        pv_v += TX;
        pr += TX * CR;
        gq += gstep;
        ph += SORB * 4;
      }
    };
    if (FIRST || DBL) {
      run(rend, true);
    } else {
      if (r < a.r0_rows) run(min(rend, a.r0_rows), true);
      if (r < rend) run(rend, false);
    }
  };
  auto run_step = [&](int n, auto first_tag) {
    const unsigned char* cur = xb + (n & 1) * xd;
    unsigned char* nxt = xb + ((n + 1) & 1) * xd;
    Real* out_sums = sums + (size_t)(n & 1) * SETS * nsum;
    for (int j = jfirst; j < v1 - v0; j += jstep) {
      const int r = s_vrow[j], re = s_vrow[j + 1];
#pragma unroll
      for (int q = 0; q < NV; ++q) f0[q] = f1[q] = Real(0);
      rows = 0;
      sum_at = out_sums + ((size_t)j * a.nfl * colT + col) * NV;
      // the virtual CTA's rows of segment 0, then of segment 1
      for (int g = 0; g < 2; ++g) {
        const int ra = g ? max(r, nr0) : r, rb = g ? re : min(re, nr0);
        if (ra >= rb || !(g ? tx_on1 : tx_on0)) continue;
        if (SORB == 1 || s == 0)
          march(first_tag, std::integral_constant<int, 0>{}, cur, nxt, g, ra, rb);
        else
          march(first_tag, std::integral_constant<int, 1>{}, cur, nxt, g, ra, rb);
      }
      if (rows) flush();
    }
  };
  run_step(0, std::true_type{});
  __syncthreads();
  for (int n = 1; n < a.steps; ++n) {
    if (s_abort) return;
    run_step(n, std::false_type{});
    __syncthreads();
  }
  if (a.write_last && !s_abort) {  // r_{steps-1} and r_steps
    for (int i = tid; i < nrows * colT; i += T) {
      const int r = i / colT, kk = i - r * colT, ss = kk / (TX * CR), lx = (kk - ss * TX * CR) / CR, q = kk % CR;
      const int g = r < nr0 ? 0 : 1;
      if (lx >= seg_tx(g)) continue;
      const int at = ss * PS + (frame_row(r) * P + lx + 1) * CB + q * CBY;
      const size_t o = (((size_t)row_y(r) * a.Lx + (sx + g) * TX + lx) * SORB + ss) * a.C + a.c0 + q;
      for (int b = 0; b < 2; ++b) ld(xb + b * xd + at).st(a.last[b], o);
    }
  }
}

template <typename Real, int CBY, int LAT, bool DBL, int SITES>
const void* res_kernel_var(int var) {
  return var == 0   ? reinterpret_cast<const void*>(&k_resident<Real, CBY, LAT, DBL, 0, SITES>)
         : var == 1 ? reinterpret_cast<const void*>(&k_resident<Real, CBY, LAT, DBL, 1, SITES>)
                    : reinterpret_cast<const void*>(&k_resident<Real, CBY, LAT, DBL, 2, SITES>);
}
template <typename Real, int CBY, int SITES>
const void* res_kernel_sites(int lattice, int dbl, int var) {
  if (lattice == KITE_HONEYCOMB)
    return dbl ? res_kernel_var<Real, CBY, KITE_HONEYCOMB, true, SITES>(var)
               : res_kernel_var<Real, CBY, KITE_HONEYCOMB, false, SITES>(var);
  return dbl ? res_kernel_var<Real, CBY, KITE_SQUARE, true, SITES>(var)
             : res_kernel_var<Real, CBY, KITE_SQUARE, false, SITES>(var);
}
template <typename Real, int CBY>
const void* res_kernel(int lattice, int dbl, int var, int sites) {
  if constexpr (CBY == 16)  // (half chunks: lattices with long lists)
    if (sites <= kRFew) return res_kernel_sites<Real, CBY, kRFew>(lattice, dbl, var);
  return res_kernel_sites<Real, CBY, kRSites>(lattice, dbl, var);
}

}  // namespace
}  // namespace kite
