// kite_resident.cu -- plans and launches of the on-chip sweep of mid-size lattices
// (kite_resident.cuh), and its FP32 kernels.
#include <math.h>

#include <algorithm>
#include <mutex>
#include <set>
#include <utility>

#include "kite_resident.cuh"

namespace kite {

const void* resident_kernel64(int lattice, int dbl, int var, int sites);  // kite_resident64.cu

namespace {

// mu_vec[vec_base + vector][n]: the sum of slot n's partials in a fixed order (a class of
// entries per thread, then a tree), over N_eff.  One block per moment; entry e belongs to the
// lane e % lanes of the sweep: a vector, or its real and imaginary part (im).
__global__ void __launch_bounds__(256) k_resident_reduce(const double* __restrict__ part, int M, int count, int lanes,
                                                         int im, int nvec, int vec_base,
                                                         const unsigned long long* __restrict__ n_eff,
                                                         double* __restrict__ mu_vec) {
  const int n = blockIdx.x;
  const double* p = part + (size_t)n * count;
  double s = 0.0;
  for (int e = threadIdx.x; e < count; e += 256) s += p[e];  // 256 is a multiple of lanes
  __shared__ double red[256];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int st = 128; st >= lanes; st >>= 1) {
    if ((int)threadIdx.x < st) red[threadIdx.x] += red[threadIdx.x + st];
    __syncthreads();
  }
  const int l = (int)threadIdx.x, v = im ? l >> 1 : l;
  if (l < lanes && v < nvec) {
    const double ne = (double)*n_eff;
    double* out = mu_vec + ((size_t)(vec_base + v) * M + n) * 2;
    out[im ? l & 1 : 0] = ne > 0.0 ? red[l] / ne : 0.0;
    if (!im) out[1] = 0.0;
  }
}

// Vectors and moment sums (real and imaginary part in FP32) of a unit of cby bytes.
int vectors_of(int fp64, int realv, int cby) { return (fp64 ? 1 : cby / 8) * (realv ? 2 : 1); }
int sums_of(int fp64, int realv, int cby) { return fp64 ? (realv ? 2 : 1) : cby / 4; }

}  // namespace

// The regions for strips of TX cells and G virtual CTAs, and the units per sweep of a batch of
// C 16-byte chunks: as many as fit on chip (fewer sweeps), with as many rows of r_0 as fit
// beside them; half chunks only where no whole one fits.  CR = 0: no fit.
ResidentPlan resident_plan(kite_ctx* ctx, int fp64, int lattice, int doubling, int realv, int field, int Lx, int Ly,
                           int C, int M, int TX, long long G, int cby) {
  ResidentPlan p{};
  C *= 16 / cby;
  const int sorb = lattice == KITE_HONEYCOMB ? 2 : 1, real = fp64 ? 8 : 4;
  const int nstrips = (Lx + TX - 1) / TX;
  const long long units = (long long)nstrips * Ly;
  // (records are indexed in 32 bits)
  if (Lx < 3 || Ly < 3 || M < 4 || G < 1 || G > units || (double)Lx * Ly * sorb * C > 4e8) return p;
  const int regions = (int)std::min<long long>(ctx->num_sms, G);
  int rows = 0, nv = 0, edge = 0;
  const int vrows = (int)((units + G - 1) / G);
  for (int i = 0; i < regions; ++i) {
    const long long v0 = G * i / regions, v1 = G * (i + 1) / regions, u0 = units * v0 / G, u1 = units * v1 / G;
    if (u1 - u0 > Ly) return p;  // more than two segments
    rows = std::max(rows, (int)(u1 - u0));
    nv = std::max(nv, (int)(v1 - v0));
    const bool two = u0 / Ly != (u1 - 1) / Ly;
    edge = std::max(edge, 2 * ((int)(u1 - u0) + (two ? 2 : 1) * TX));
  }
  if (nv > kRMaxV) return ResidentPlan{};
  p.nfl = (vrows + kRFlush - 1) / kRFlush;
  for (int cr = C; cr >= 1; cr >>= 1) {
    const int colT = TX * sorb * cr;
    if (colT > kRMax || edge * cr > kRSites * kRComm) continue;
    const int per = sums_of(fp64, realv, cby);
    auto need = [&](int r0_rows) {
      return res_smem(cby, sorb, cr, TX, rows, nv, p.nfl, real, per, doubling, r0_rows, field).total;
    };
    if (need(0) > kResSmem) continue;
    int r0_rows = doubling ? 0 : rows;
    while (r0_rows > 0 && need(r0_rows) > kResSmem) --r0_rows;
    p.cby = cby;
    p.vecs = vectors_of(fp64, realv, cby);
    p.regions = regions;
    p.TX = TX;
    p.G = (int)G;
    p.rows = rows;
    p.nv = nv;
    p.r0_rows = r0_rows;
    p.CR = cr;
    p.sites = edge * cr <= kRFew * kRComm ? kRFew : kRSites;
    p.T = std::min(nv, kRMax / colT) * colT;
    p.T = (p.T + 31) / 32 * 32;
    p.smem = need(r0_rows);
    int lv = 0;
    while ((32 >> (lv + 1)) >= cr * per && (!fp64 || lv < 2)) ++lv;
    p.levels = lv;
    return p;
  }
  return cby == 16 && !fp64 ? resident_plan(ctx, fp64, lattice, doubling, realv, field, Lx, Ly, C, M, TX, G, 8) : p;
}

// FP64 sums may be grouped freely: strips and virtual CTAs that give every SM a compact
// region and its threads one column of few rows each.
ResidentPlan resident_plan_free(kite_ctx* ctx, int lattice, int doubling, int realv, int field, int Lx, int Ly, int C,
                                int M) {
  ResidentPlan best{};
  long long best_cost = -1;
  const int sorb = lattice == KITE_HONEYCOMB ? 2 : 1;
  for (int TX = 4; TX <= 128; TX += TX < 16 ? 1 : (TX < 32 ? 2 : 8)) {
    const int nstrips = (Lx + TX - 1) / TX;
    const long long units = (long long)nstrips * Ly;
    const int regions = (int)std::min<long long>(ctx->num_sms, units);
    const int rows = (int)((units + regions - 1) / regions);
    // sub-columns: as many virtual CTAs per region as fill the compute threads
    const int colT = TX * sorb * C;
    const int nv = std::max(1, std::min(rows, kRMax / std::max(1, colT)));
    const ResidentPlan p = resident_plan(ctx, 1, lattice, doubling, realv, field, Lx, Ly, C, M, TX,
                                         std::min<long long>((long long)regions * nv, units), 16);
    if (p.CR == 0) continue;
    // a step: the rows of the longest column in sites of the whole SM, plus the edge
    const long long sweeps = C / p.CR;
    // (a warp with both sublattices runs the march twice)
    const int twice = sorb == 2 && (p.TX * p.CR) % 32 ? 2 : 1;
    const long long cost = sweeps * (4LL * twice * p.rows * p.TX * sorb * p.CR + 2LL * (p.rows + p.TX) * p.CR + 400);
    if (best_cost < 0 || cost < best_cost) best_cost = cost, best = p;
  }
  return best;
}

size_t rec_bytes_of(int lattice, int Lx, int Ly, int CR, int cby) {
  return (size_t)2 * Lx * Ly * (lattice == KITE_HONEYCOMB ? 2 : 1) * CR * 2 * cby;
}

void resident_space(kite_ctx* ctx, int fp64, int lattice, int realv, int Lx, int Ly, int C, int slots, size_t* rec,
                    size_t* part) {
  *rec = *part = 0;
  const double orb = (double)Lx * Ly * (lattice == KITE_HONEYCOMB ? 2 : 1);
  for (int cby = 16; cby >= (fp64 ? 16 : 8); cby >>= 1) {
    int cr = C * 16 / cby;  // two iterates of cr units must fit the SMs together
    while (cr >= 1 && orb * cr * 2.0 * cby > (double)ctx->num_sms * kResSmem) cr >>= 1;
    if (cr < 1) continue;
    const int lanes = cr * sums_of(fp64, realv, cby);
    *rec = std::max(*rec, rec_bytes_of(lattice, Lx, Ly, cr, cby));
    *part = std::max(*part, (size_t)slots * ctx->num_sms * (kRComm / 32) * (fp64 ? std::max(8, lanes) : lanes) *
                                sizeof(double));
  }
}

int resident_sweep(kite_ctx* ctx, ResidentSweep* a, int timing_steps) {
  const ResidentPlan& p = a->plan;
  if (ctx->fail_count > 0) {  // test hook
    if (ctx->fail_skip > 0) {
      --ctx->fail_skip;
    } else {
      --ctx->fail_count;
      if (ctx->fail_kind == KITE_FAIL_LAUNCH)
        return cuda_fail(ctx, cudaErrorCooperativeLaunchTooLarge, "on-chip sweep");
      a->stall = 1;
    }
  }
  const int var = a->phase ? 1 : (a->realv ? 2 : 0);
  const void* fn = a->fp64        ? resident_kernel64(a->lattice, a->doubling, var, p.sites)
                   : p.cby == 16 ? res_kernel<float, 16>(a->lattice, a->doubling, var, p.sites)
                                 : res_kernel<float, 8>(a->lattice, a->doubling, var, p.sites);
  {
    static std::mutex mu;
    static std::set<std::pair<const void*, int>> done;
    std::lock_guard<std::mutex> lock(mu);
    if (!done.count({fn, ctx->device})) {
      KITE_CUDA_TRY(ctx, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem));
      done.insert({fn, ctx->device});
    }
  }
  if (!ctx->sweep_status) {
    void* word = nullptr;
    KITE_CUDA_TRY(ctx, cudaHostAlloc(&word, 64, cudaHostAllocMapped));  // (unified addressing: one address)
    ctx->sweep_status = static_cast<volatile int*>(word);
  }
  *ctx->sweep_status = 0;  // (no sweep of this context is in flight: each one is waited for)
  const int steps = timing_steps > 0 ? timing_steps : (a->doubling ? (a->M + 1) / 2 : a->M - 1);
  const int per = p.vecs, C = a->C * (16 / p.cby);  // vectors per unit, units per orbital
  const size_t rec_bytes = rec_bytes_of(a->lattice, a->Lx, a->Ly, p.CR, p.cby);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.regions);
  cfg.blockDim = dim3((unsigned)(p.T + kRComm));
  cfg.dynamicSmemBytes = (size_t)p.smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // neighbouring CTAs wait on one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  KITE_CUDA_TRY(ctx, cudaEventRecord(ctx->ev2, ctx->stream));
  for (int c0 = 0; c0 < C && c0 * per < a->nvec; c0 += p.CR) {
    // no record may carry a step number of an earlier sweep
    KITE_CUDA_TRY(ctx, cudaMemsetAsync(a->rec, 0, rec_bytes, ctx->stream));
    auto launch = [&](auto tag) -> cudaError_t {
      using Real = decltype(tag);
      ResArgs<Real> r{};
      r.r0 = a->r0;
      r.vt = static_cast<const Real*>(a->vt);
      r.phase = static_cast<const Real*>(a->phase);
      r.last[1] = a->bA;  // odd iterates
      r.last[0] = a->bB;
      r.part = a->part;
      r.rec = a->rec;
      r.err = ctx->sweep_status;
      r.tt = (Real)a->tt;
      r.Lx = a->Lx;
      r.Ly = a->Ly;
      r.TX = p.TX;
      r.G = p.G;
      r.rows_max = p.rows;
      r.nv_max = p.nv;
      r.nfl = p.nfl;
      r.r0_rows = p.r0_rows;
      r.levels = p.levels;
      r.C = C;
      r.c0 = c0;
      r.CR = p.CR;
      r.steps = steps;
      r.open_x = a->open_x;
      r.open_y = a->open_y;
      r.stall = a->stall;
      r.write_last = timing_steps > 0 ? 0 : a->want_last;
      void* kargs[] = {&r};
      return cudaLaunchKernelExC(&cfg, fn, kargs);
    };
    KITE_CUDA_TRY(ctx, a->fp64 ? launch(double()) : launch(float()));
    a->stall = 0;
    if (timing_steps > 0) break;
    const int nvec = std::min(a->nvec - c0 * per, p.CR * per);
    k_resident_reduce<<<a->M, 256, 0, ctx->stream>>>(a->part, a->M, p.regions * (kRComm / 32) * (32 >> p.levels),
                                                     p.CR * sums_of(a->fp64, a->realv, p.cby),
                                                     !a->fp64 && !a->realv, nvec, a->vec_base + c0 * per, a->n_eff,
                                                     a->mu_vec);
    KITE_CUDA_TRY(ctx, cudaGetLastError());
  }
  KITE_CUDA_TRY(ctx, cudaEventRecord(ctx->ev3, ctx->stream));
  float ms = 0.f;
  KITE_CUDA_TRY(ctx, cudaEventSynchronize(ctx->ev3));
  KITE_CUDA_TRY(ctx, cudaEventElapsedTime(&ms, ctx->ev2, ctx->ev3));
  if (*ctx->sweep_status) return fail(ctx, KITE_ERR_TIMEOUT, "a bounded wait of the on-chip sweep gave up");
  a->seconds = 1e-3 * ms;
  a->grid = p.regions;
  a->block = p.T + kRComm;
  const int sorb = a->lattice == KITE_HONEYCOMB ? 2 : 1;
  // bytes to and from device memory: r_0 and the on-site terms in (the rows of r_0 that are
  // not kept on chip once per step), the moment partials out
  const double n_orb = (double)a->Lx * a->Ly * sorb;
  const double off_chip = a->doubling ? 0.0 : 1.0 - (double)p.r0_rows / p.rows;
  a->bytes = n_orb * a->C * 16.0 * (1.0 + off_chip * steps) + n_orb * (a->fp64 ? 8.0 : 4.0) +
             8.0 * a->M * p.regions * (kRComm / 32) * (32 >> p.levels) * ((C + p.CR - 1) / p.CR);
  return KITE_OK;
}

}  // namespace kite
