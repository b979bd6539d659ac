// Plan and launch of the resident-brick kernel (lbm_brick.cuh).
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

const void* brick_kernel_f32(int mode, int var, bool pair, bool in_place);
cudaError_t state_sums_f32(const float* state, const float* phi, const Geometry& geo, double* partial,
                        double* out, const double* word, int* count, cudaStream_t st);
const void* brick_kernel_f16(int mode, int var, bool pair, bool in_place);
cudaError_t state_sums_f16(const float* state, const float* phi, const Geometry& geo, double* partial,
                        double* out, const double* word, int* count, cudaStream_t st);
const void* brick_kernel_bf16(int mode, int var, bool pair, bool in_place);
cudaError_t state_sums_bf16(const float* state, const float* phi, const Geometry& geo, double* partial,
                        double* out, const double* word, int* count, cudaStream_t st);

namespace {

constexpr int kBrickTwoLeast = 54000;      // bytes a block from which a third one matters
constexpr int kBrickTwoSmem = 77 * 1024;   // more than a third of an SM's 228 KB

// ceil(2^kBrickDivShift / d), and whether k * it >> kBrickDivShift = k / d for every k up to
// `most`.
unsigned brick_div(int d) { return ((1u << kBrickDivShift) + d - 1) / d; }

bool brick_div_ok(int d, long long most) {
  const unsigned long long m = brick_div(d), over = m * d - (1ull << kBrickDivShift);
  return most * m < (1ull << 32) && most * over < (1ull << kBrickDivShift);
}

const void* kernel_of(const Geometry& geo, const Physics& ph, int mode, bool pair, bool in_place) {
  const int var = mode == kBrickTracking
                      ? 0
                      : (ph.srt_flow ? kVarSrtFlow : 0) | (ph.d3q7_stencil ? kVarD3Q7 : 0);
  return geo.storage == kF16    ? brick_kernel_f16(mode, var, pair, in_place)
         : geo.storage == kBF16 ? brick_kernel_bf16(mode, var, pair, in_place)
                                : brick_kernel_f32(mode, var, pair, in_place);
}

// One way to cut an axis: bricks, cells of the largest, bricks within the cells a step reads.
struct AxisCut {
  int nb, b, reach;
};

AxisCut cut_axis(int n, int want, int halo) {
  AxisCut c;
  c.nb = (n + want - 1) / want;
  c.b = (n + c.nb - 1) / c.nb;
  const int least = n / c.nb;
  c.reach = (halo + 1 + least - 1) / least;
  return c;
}

// Whether the kernel's small divisions are exact for bricks of these sizes (cell numbers run
// up to two rounds of threads beyond a brick's cells).
bool divisions_ok(const AxisCut c[3], int halo) {
  const long long cells = static_cast<long long>(c[0].b) * c[1].b * c[2].b + 2 * kBrickThreads;
  if (!brick_div_ok(c[0].b, cells) || !brick_div_ok(c[1].b, cells / c[0].b + 1)) return false;
  for (int add : {2, 2 * halo, 2 * halo + 2}) {
    const long long x = c[0].b + add, y = c[1].b + add, z = c[2].b + add;
    if (!brick_div_ok(static_cast<int>(x), x * y * z) || !brick_div_ok(static_cast<int>(y), y * z + 1))
      return false;
  }
  return true;
}

}  // namespace

// The line lies where the two state arrays outgrow the L2 cache (129 MB): 640,000 cells of
// 2 x 100 B coupled in FP32, 1.6M of 2 x 40 B in tracking mode, where f and phi u are all
// that moves.  Measured just inside it, three passes (one in tracking mode) -> bricks:
// 96x96x64 (590k cells) 32.6 -> 27.6 us a step, 80^3 27.7 -> 27.6, tracking at 116^3 (1.56M)
// 41.9 -> 32.8; beyond it (64x64x256, 1.05M cells) the bricks' halos come from DRAM: 57-63 us
// against 48.  With 16-bit populations the coupled kernel gains less (its 2-byte loads bring
// half as much each): 56x57x55 (176k cells) 14.4 -> 13.9 us, 64^3 (262k) 18.4 -> 18.5.  In
// place a step has two waits and the bricks pay for the smallest boxes only: 32^3 9.2 -> 8.8
// us, 48^3 11.3 -> 11.7; tracking 64^3 19.2 -> 12.4, 80^3 20.5 -> 21.0.
// Boxes of any shape below the lines, part of the three-kernel step's time (geometric mean;
// worst): FP32 0.87 (1.10 at 317x1049x1) over 110, FP16 0.77 (1.17 at 35x59x72) over 105; in
// place FP32 0.86 (1.18 at 1x75x363) over 119, BF16 0.84 (1.14 at 33x29x22) over 109; tracking
// in place 0.58 (0.88) over 81.
long long brick_most_cells(int mode, int storage, bool in_place) {
  if (in_place) return mode == kBrickTracking ? 270000 : 36000;
  if (mode == kBrickTracking) return 1600000;
  return storage == kF32 ? 640000 : 180000;
}

// The cut with the least modelled step time among those that keep every block resident.  The
// model, fitted to 190 measured cuts of 16^3 to 96x96x64 (within 20 % of them): 3.65 us for
// the wait, the loads' latency and the stores, and per block of an SM 0.44 ns for each place
// of its phi and mu regions and 2.7 ns (tracking: 1.2) for each of its cells in whole rounds
// of threads, more for short rows (a region row of 20 touches as many lines as one of 36) and
// for rows that do not start on tiles; a lone block with several rounds per SM waits more.
// Two cells per thread pay from about 1024 cells a block (64x64x128, 256 bricks of 32x8x8:
// 24.9 us, one cell per thread 26.3); they leave room for 2 blocks an SM instead of 3.  Boxes
// with 16-bit populations are too small for that: none of 19,671 sampled ones took it.
// Measured per step, three passes -> bricks: 16^3 9.2 -> 4.2 us, 32^3 9.2 -> 4.9, 48^3
// 11.5 -> 7.9, 64^3 18.5 -> 13.7, 64x64x128 29.6 -> 25.1, 37x41x45 10.3 -> 8.5; tracking 48^3
// 12.3 -> 5.6, 100^3 30.6 -> 21.3; FP16 32^3 10.2 -> 6.2.
BrickPlan brick_plan(const Geometry& geo, const Physics& ph, int mode, bool in_place, int sms) {
  BrickPlan p{};
  p.in_place = in_place ? 1 : 0;
  if (geo.n > brick_most_cells(mode, geo.storage, in_place) || sms < 1) return p;
  const int halo = mode == kBrickTracking ? 1 : 2;
  constexpr int kWant = 9;
  static const int want[2][kWant] = {{8, 12, 16, 24, 32, 48, 64, 96, 128}, {2, 3, 4, 5, 6, 8, 10, 12, 16}};
  AxisCut axis[3][kWant];
  for (int i = 0; i < kWant; ++i) {
    axis[0][i] = cut_axis(geo.nx, want[0][i], halo);
    axis[1][i] = cut_axis(geo.ny, want[1][i], halo);
    axis[2][i] = cut_axis(geo.nz, want[1][i], halo);
  }
  double cost = 0.0;
  for (int i = 0; i < kWant; ++i)
    for (int j = 0; j < kWant; ++j)
      for (int k = 0; k < kWant; ++k) {
        const AxisCut c[3] = {axis[0][i], axis[1][j], axis[2][k]};
        const long long bricks = static_cast<long long>(c[0].nb) * c[1].nb * c[2].nb;
        if (bricks > 3LL * sms || bricks > kBrickMax) continue;
        long long cells = 1, phi = 1, mu = 1, offsets = 1, around = 1;
        for (const AxisCut& a : c) {
          cells *= a.b;
          phi *= a.b + 2 * halo;
          mu *= a.b + 2;
          offsets *= a.b + 2 * halo + 2;
          around *= std::min(a.nb, 2 * a.reach + 1);
        }
        if (mode == kBrickTracking) mu = 0;
        const long long smem = 4 * (phi + mu + (in_place ? 0 : offsets));
        const int per = static_cast<int>((bricks + sms - 1) / sms);
        if (around > kBrickThreads || smem > kBrickSmem || per * (smem + 1024) > 226 * 1024) continue;
        for (int pair = 0; pair < 2; ++pair) {
          if (pair && (mode == kBrickTracking || in_place || geo.storage != kF32 || cells < 1024 || per > 2))
            continue;
          const long long round = pair ? 2 * kBrickThreads : kBrickThreads;
          const double cell = mode == kBrickTracking ? 1.2e-3 : (cells >= 1024 && !pair ? 2.9e-3 : 2.7e-3);
          double work = 4.4e-4 * ((in_place ? phi / 3 : phi) + mu) + cell * ((cells + round - 1) / round * round);
          work *= 1.0 + 4.0 / c[0].b;
          if (geo.row_tiles && c[0].b % 16 != 0) work *= 1.08;
          const double est = 3.65 + per * work * (per == 1 && cells > 512 ? 1.3 : 1.0);
          if ((p.nbricks && est >= cost) || !divisions_ok(c, halo)) continue;
          cost = est;
          p.nbricks = static_cast<int>(bricks);
          p.mode = mode;
          p.pair = pair;
          p.around = static_cast<int>(around);
          p.smem = static_cast<int>(smem);
          for (int a = 0; a < 3; ++a) {
            p.nb[a] = c[a].nb;
            p.b[a] = c[a].b;
            p.reach[a] = c[a].reach;
          }
        }
      }
  if (p.nbricks == 0) return p;
  // Two blocks an SM that leave shared memory for a third may be placed three on some SMs, and
  // the L1 cache, which the pulled f comes from several times, shrinks to what three leave: ask
  // for as much as lets no third in (97x105x57 52.2 -> 34.1 us a step, 83x117x63 48.2 -> 33.3,
  // 128x110x43 40.6 -> 31.5; tracking 68x98x187 30.4 -> 24.9).  It counts from 54 KB a block (0.97
  // of the time at 55 KB, 0.65 to 0.82 at 67 to 76; below it 0.99 to 1.01); with two cells per
  // thread the registers keep a third out.
  if (p.nbricks > sms && p.nbricks <= 2 * sms && !p.pair && p.smem > kBrickTwoLeast)
    p.smem = std::max(p.smem, kBrickTwoSmem);
  const void* k = kernel_of(geo, ph, mode, p.pair != 0, in_place);
  int per = 0;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kBrickSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, kBrickThreads, p.smem) != cudaSuccess ||
      static_cast<long long>(per) * sms < p.nbricks) {
    cudaGetLastError();
    return BrickPlan{};
  }
  p.slots = per * sms;
  p.m_qx = brick_div(p.b[0] + 2 * halo + 2);
  p.m_qy = brick_div(p.b[1] + 2 * halo + 2);
  p.m_px = brick_div(p.b[0] + 2 * halo);
  p.m_py = brick_div(p.b[1] + 2 * halo);
  p.m_mx = brick_div(p.b[0] + 2);
  p.m_my = brick_div(p.b[1] + 2);
  p.m_bx = brick_div(p.b[0]);
  p.m_by = brick_div(p.b[1]);
  return p;
}

cudaError_t launch_brick(float* state0, float* state1, float* phi, const Geometry& geo,
                         const Physics& ph, const BrickPlan& plan, const BrickTimes& times, int steps,
                         int* flags, int base, bool have_prev, bool odd, int* err, long long polls,
                         cudaStream_t st) {
  BrickPlan bp = plan;
  bp.steps = steps;
  int hp = have_prev ? 1 : 0;
  int od = odd ? 1 : 0;
  if (plan.in_place) {
    void* args[] = {&state0, &phi, const_cast<Geometry*>(&geo), const_cast<Physics*>(&ph), &bp,
                    const_cast<BrickTimes*>(&times), &flags, &base, &hp, &od, &err, &polls};
    return cudaLaunchCooperativeKernel(kernel_of(geo, ph, plan.mode, false, true), dim3(plan.nbricks),
                                       dim3(kBrickThreads), args, plan.smem, st);
  }
  void* args[] = {&state0, &state1, &phi, const_cast<Geometry*>(&geo), const_cast<Physics*>(&ph), &bp,
                  const_cast<BrickTimes*>(&times), &flags, &base, &hp, &err, &polls};
  const void* k = kernel_of(geo, ph, plan.mode, plan.pair != 0, plan.in_place != 0);
  // in a single step no block waits for another, so they need not be resident together
  return steps == 1
             ? cudaLaunchKernel(k, dim3(plan.nbricks), dim3(kBrickThreads), args, plan.smem, st)
             : cudaLaunchCooperativeKernel(k, dim3(plan.nbricks), dim3(kBrickThreads), args, plan.smem, st);
}

cudaError_t launch_state_sums(const float* state, const float* phi, const Geometry& geo, double* partial,
                              double* out, const double* word, int* count, cudaStream_t st) {
  return geo.storage == kF16    ? state_sums_f16(state, phi, geo, partial, out, word, count, st)
         : geo.storage == kBF16 ? state_sums_bf16(state, phi, geo, partial, out, word, count, st)
                                : state_sums_f32(state, phi, geo, partial, out, word, count, st);
}

}  // namespace lbm
