// Register-tile 2D stencil: kernel variants, the rule that picks one for a
// grid, and the launch.
#include "block2d.cuh"
#include "block2d_fx.cuh"

namespace ac {

namespace {

// The variants and their measured costs on GB300 (graph-replayed launches,
// microseconds): a launch of k steps over n tiles takes about
//   t0 + sum over an SM's rounds of (load + k * max(lat, tiles * warps * busy))
// with t0 the launch, load one tile's load and store, lat one step's latency
// and busy the time a warp's step keeps the SM busy.  Fitted to sweeps over
// 64^2 .. 8192^2, warps and k; on those grids the variant, warps and k that
// the fit picks run within 2 % of the best measured (FP16 storage at 8192^2:
// 7 %).  Which wins where: 4 x 4 cells a lane up to 512^2 (400x200: 0.371 us a
// step against 0.405 and 0.486), 8 rows near 1024^2 (0.78 against 0.87 and
// 0.98), 7 rows in 64 registers (two CTAs to an SM) from 2048^2 (4096^2: 8.0 us
// against 9.4 and 10.9), and for FP16 storage 9 rows there (4096^2: 7.3; 7.7
// with 8 x 8 cells).
struct B2Variant {
  int E, R, regs;  // E: cells a lane and row (FP64: 1)
  double t0, load, lat, busy;
};
constexpr B2Variant kB2[] = {
    {4, 4, 72, 1.06, 1.55, 0.069, 0.0202},
    {4, 7, 64, 1.49, 1.81, 0.131, 0.0363},
    {4, 8, 112, 1.13, 2.15, 0.005, 0.0404},
    {4, 9, 64, 2.18, 1.41, 0.207, 0.0476},  // FP16 storage
    // FP64 (block2d_fx.cuh): two rows a lane (200^2 1.61 us a step against 1.79 with
    // four)
    {1, 2, 40, 2.67, 0.0, 0.036, 0.0627},
};
constexpr int kB2Count = sizeof(kB2) / sizeof(kB2[0]);

bool offered(const B2Variant &b, int dtype) {
  return dtype == AC_F64 ? b.E == 1 : b.E == 4 && (b.R != 9 || dtype == AC_F16S);
}

// Halo columns: whole memory vectors of 4 cells (FP64: single cells).
int halo_x(int E, int k) { return (k + E - 1) / E * E; }

double launch_cost(const B2Variant &b, int64_t nx, int64_t ny, int warps, int k, int num_sms) {
  const int ow = 32 * b.E - 2 * halo_x(b.E, k), oh = warps * b.R - 2 * k;
  const double tiles = std::ceil((double)nx / ow) * std::ceil((double)ny / oh);
  const int occ = std::max(1, std::min(65536 / (b.regs * warps * 32), 64 / warps));
  const double per_sm = std::ceil(tiles / num_sms);
  const double full = std::floor(per_sm / occ), rest = per_sm - full * occ;
  auto step = [&](double c) { return std::max(b.lat, c * warps * b.busy); };
  return b.t0 + full * (b.load + k * step(occ)) + (rest > 0 ? b.load + k * step(rest) : 0.0);
}

// The same for FP32 and FP16 storage beyond L2 (two fields of more than 100 MB),
// with the time that the field's bytes take, read with the halos, as a p-norm.
// Without it six launches of 4 steps at 8192^2 (881 us) came out cheaper than
// four of 6 (744).
struct B2Memory {
  double p, rate;  // bytes per microsecond
};
constexpr B2Memory kB2MemF32 = {4.0, 6.5e6}, kB2MemF16 = {2.0, 5.5e6};

double tiled_cost(const B2Variant &b, int dtype, int64_t nx, int64_t ny, int warps, int k, int num_sms) {
  const double c = launch_cost(b, nx, ny, warps, k, num_sms);
  const double bytes = (dtype == AC_F32 ? 4.0 : 2.0) * (double)nx * (double)ny;
  if (dtype == AC_F64 || 2.0 * bytes < 100e6) return c;
  const B2Memory &m = dtype == AC_F32 ? kB2MemF32 : kB2MemF16;
  const int ow = 32 * b.E - 2 * halo_x(b.E, k), oh = warps * b.R - 2 * k;
  const double read = 32.0 * b.E / ow * (double)std::min<int64_t>(ny, warps * b.R) / (double)std::min<int64_t>(ny, oh);
  return std::pow(std::pow(c, m.p) + std::pow(bytes * (1.0 + read) / m.rate, m.p), 1.0 / m.p);
}

template <typename T, int E, int R, int MINB>
cudaError_t launch_t(const GridParams &g, const void *src, void *dst, int warps, int k, uint32_t mask,
                     cudaStream_t s) {
  static KernelSetup ks;
  int occ = 1;
  cudaError_t e = kernel_setup(ks, (const void *)block2d_k<T, E, R, MINB>, kB2MaxWarps * 32,
                               b2_smem_bytes(E, kB2MaxWarps), &occ);
  if (e != cudaSuccess) return e;
  const int hx = halo_x(E, k);
  const int ow = 32 * E - 2 * hx, oh = warps * R - 2 * k;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((g.nx + ow - 1) / ow), (unsigned)((g.ny + oh - 1) / oh));
  cfg.blockDim = dim3(warps * 32);
  cfg.dynamicSmemBytes = b2_smem_bytes(E, warps);
  cfg.stream = s;
  // programmatic stream serialization: the launch overlaps the previous
  // one's tail (0.39 against 0.42 us a step at 64^2, nothing at 4096^2)
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, block2d_k<T, E, R, MINB>, (const T *)src, (T *)dst, g, k, hx, mask);
}

template <int R>
cudaError_t launch_fx_t(const GridParams &g, const void *src, void *dst, int warps, int k, cudaStream_t s) {
  static KernelSetup ks;
  int occ = 1;
  cudaError_t e = kernel_setup(ks, (const void *)block2d_fx_k<R>, kB2FxMaxWarps * 32,
                               b2fx_smem_bytes(kB2FxMaxWarps), &occ);
  if (e != cudaSuccess) return e;
  const int ow = 32 - 2 * k, oh = warps * R - 2 * k;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((g.nx + ow - 1) / ow), (unsigned)((g.ny + oh - 1) / oh));
  cfg.blockDim = dim3(warps * 32);
  cfg.dynamicSmemBytes = b2fx_smem_bytes(warps);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, block2d_fx_k<R>, (const double *)src, (double *)dst, g, k);
}

}  // namespace

// A step of the FP64 kernels that take one step a launch (k_direct.cu): 1.5, 1.6,
// 1.8, 2.8 and 3.6 us on GB300 at 64^2, 200^2, 256^2, 400^2 and 512^2, where the best
// tiles take 1.1, 1.6, 1.7, 2.6 and 3.5 on smooth fields.  From 50000 cells on
// tiles are not tried: their fit is up to a third short where they fill the SMs'
// last round exactly (400^2: 3.4), and rough fields cost them more (256^2 2.7
// against 2.2 for the heat equation from noise).
constexpr int64_t kB2FxCells = 50000;
static double single_cost(int64_t nx, int64_t ny) { return 1.45 + 8.4e-6 * (double)nx * (double)ny; }

// A pass of k steps of the streaming kernel (stream2d.cuh): t0, a row of a warp's
// chunk (l0 + l1 k if its chain of dependences bounds it, p0 + p1 k for each
// vector of 8 cells and warp of the SM if its instructions do), the field's bytes.
// Fitted to passes of every depth over 1 x 2048 .. 16384^2 (6 to 10 % rms).
struct S2Cost {
  int vec, cells;  // of a lane
  double t0, l0, l1, p0, p1, mem;
};
constexpr S2Cost kS2F32 = {4, 4, 1.00, 0.226, 0.0491, 0.0444, 0.0104, 14.0e6},
                 kS2F32Wide = {4, 8, 0.0, 0.278, 0.204, 0.0, 0.0, 6.0e6},
                 kS2F16 = {8, 8, 1.18, 0.245, 0.0899, 0.0159, 0.0139, 16.7e6};

static double stream_cost(int dtype, int tile, int64_t nx, int64_t ny, int k, int num_sms) {
  const S2Cost &c = dtype == AC_F16S ? kS2F16 : tile == 1 ? kS2F32Wide : kS2F32;
  const int ow = 32 * c.cells - 2 * ((k + c.vec - 1) / c.vec * c.vec);
  const double strips = std::ceil((double)nx / ow);
  double chunks = std::max(1.0, std::floor(16.0 * num_sms / strips));  // two CTAs of 8 warps an SM
  chunks = std::min(chunks, std::max(1.0, std::floor((double)ny / std::max(16, 3 * k))));
  const double chunk = std::ceil((double)ny / chunks);
  const double warps = strips * std::ceil((double)ny / chunk) / num_sms;
  const double rows = chunk < (double)ny ? chunk + 2 * k : (double)ny + k;
  const double lat = c.t0 + rows * (c.l0 + c.l1 * k);
  const double issue = c.t0 + rows * std::max(1.0, warps) * (c.p0 + c.p1 * k) * c.cells / 8;
  const double mem = c.t0 + 2.0 * (dtype == AC_F16S ? 2 : 4) * (double)nx * (double)ny / c.mem;
  return std::pow(lat * lat * lat * lat + issue * issue * issue * issue + mem * mem * mem * mem, 0.25);
}

double block2d_other(int dtype, int tile, int64_t nx, int64_t ny, const int64_t *passes, int kmax, int num_sms) {
  if (dtype == AC_F64) return (double)passes[1] * single_cost(nx, ny);
  double t = 0.0;
  int64_t steps = 0;
  for (int k = 1; k <= kmax; ++k)
    if (passes[k]) {
      t += (double)passes[k] * stream_cost(dtype, tile, nx, ny, k, num_sms);
      steps += passes[k] * k;
    }
  // The fits' error: for calls of a few steps on large grids the tiles' is too
  // cheap (4096^2, 3 steps: 60 us, against 51 streaming), with many steps too dear.
  return (steps <= 4 && nx * ny >= 4000000 ? 0.87 : 1.02) * t;
}

bool block2d_plan(int dtype, int64_t nx, int64_t ny, int64_t passes, int depth, const int *depths, double other,
                  int num_sms, Block2DPlan *out) {
  if (passes < 1 || (dtype == AC_F64 && nx * ny > kB2FxCells)) return false;
  double best = other;
  bool found = false;
  for (int v = 0; v < kB2Count; ++v) {
    if (!offered(kB2[v], dtype)) continue;
    for (int warps = 4; warps <= kB2MaxWarps; warps += 4)
      for (int kmax = dtype == AC_F64 ? 2 : 4; kmax <= (dtype == AC_F64 ? 8 : kB2MaxDepth);
           kmax += dtype == AC_F64 ? 1 : 4) {
        const int per = kmax / depth;  // passes per launch
        if (per < 1 || warps * kB2[v].R - 2 * per * depth < 4) continue;
        int64_t launches = (passes + per - 1) / per;
        if (launches % 2 && passes > 1) ++launches;  // an even count ends in the source buffer
        const int64_t few = passes / launches, more = passes % launches;  // launches of few + 1 passes
        const int k = (int)(few + (more > 0)) * depth;
        const int oh = warps * kB2[v].R - 2 * k;
        if ((ny + oh - 1) / oh > 65535) continue;  // CUDA's grid limit in y
        auto cost_of = [&](int q) { return tiled_cost(kB2[v], dtype, nx, ny, warps, q, num_sms); };
        double cost = 0.0;
        if (depths && passes <= 16) {  // the last passes may be shorter than depth
          for (int64_t i = 0; i < launches; ++i) {
            int q = 0;
            for (int64_t p = passes * i / launches; p < passes * (i + 1) / launches; ++p) q += depths[p];
            cost += cost_of(q);
          }
        } else {
          cost = (double)(launches - more) * cost_of((int)few * depth);
          if (more) cost += (double)more * cost_of((int)(few + 1) * depth);
        }
        if (cost < best) {
          best = cost;
          found = true;
          *out = Block2DPlan{v, warps, launches};
        }
      }
  }
  return found;
}

cudaError_t launch_block2d(int dtype, const Block2DPlan &p, const GridParams &g, const void *src, void *dst,
                           int k, uint32_t round_mask, cudaStream_t s) {
  if (dtype == AC_F32) {
    switch (p.variant) {
      case 0: return launch_t<float, 4, 4, 1>(g, src, dst, p.warps, k, 0u, s);
      case 1: return launch_t<float, 4, 7, 2>(g, src, dst, p.warps, k, 0u, s);
      case 2: return launch_t<float, 4, 8, 1>(g, src, dst, p.warps, k, 0u, s);
    }
  } else if (dtype == AC_F64) {
    switch (p.variant) {
      case 4: return launch_fx_t<2>(g, src, dst, p.warps, k, s);
    }
  } else if (dtype == AC_F16S) {
    switch (p.variant) {
      case 0: return launch_t<__half, 4, 4, 1>(g, src, dst, p.warps, k, round_mask, s);
      case 1: return launch_t<__half, 4, 7, 2>(g, src, dst, p.warps, k, round_mask, s);
      case 2: return launch_t<__half, 4, 8, 1>(g, src, dst, p.warps, k, round_mask, s);
      case 3: return launch_t<__half, 4, 9, 2>(g, src, dst, p.warps, k, round_mask, s);
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace ac
