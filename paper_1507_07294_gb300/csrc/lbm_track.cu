// One-pass time step of the interface-tracking mode (prescribed velocity; pattern AB, FP32) on
// grids beyond the resident bricks: the order parameter (Eqs. 13, 16), the chemical potential
// (Eq. 2) and the D3Q7 collision (Eqs. 15, 17, 18, 34) in one kernel, phi in shared memory
// only.  The three passes move 128 B a cell (f twice, phi and mu written and read); this one
// reads f and phi u once and writes them once, 80 B (78.6 by ncu at 192^3).  It is bound by
// instruction issue and the barriers between planes, not by that traffic: 67 % of the issue
// slots at 62 % of the DRAM rate, 395 instructions a cell.  Every value is formed
// by the operations of the three passes in their order, so the state is the same bit for bit.
// Measured per step, three passes -> one: 256^3 335 -> 282 us, 192^3 155 -> 128, 128^3
// 55.4 -> 45.1 (k_track_rows); 150^3 91.8 -> 75.9, 200^3 193 -> 166 (k_track).
#include <cuda_runtime.h>

#include "lbm_brick.cuh"

namespace lbm {

namespace {

constexpr int kTrackThreads = 256;

struct TrackPlan {
  int b[3], nb[3];
  unsigned m_px, m_py, m_bx, m_by;
};

// Grids of other shapes (columns_suit): a block takes a brick of at most 32 x 8 x 8 cells, phi on it and one cell
// around it from the pulled f, then mu and the collision of its cells, whose f it pulls again
// (from L1 and L2).
__global__ void __launch_bounds__(kTrackThreads, 4)
    k_track(const float* __restrict__ src, float* __restrict__ dst,
            const __grid_constant__ Geometry geo, const __grid_constant__ Physics ph,
            const __grid_constant__ TrackPlan tp, int have_prev, float tf) {
  extern __shared__ float smem[];
  constexpr int S = kF32, T = kTrackThreads, SL = kTile * 4;
  const int tid = threadIdx.x;
  const int px = tp.b[0] + 2, py = tp.b[1] + 2, pz = tp.b[2] + 2;
  float* sphi = smem;
  // the cell index that each x, y and z of the region and one cell around it adds
  int* xo = reinterpret_cast<int*>(smem + px * py * pz);
  int* yo = xo + px + 2;
  int* zs = yo + py + 2;
  float* sn = reinterpret_cast<float*>(zs + pz + 2);  // sin(pi x / L), sin(2 pi x / L) of x, y, z
  const int sny = 2 * tp.b[0], snz = sny + 2 * tp.b[1];
  const int bxy = tp.nb[0] * tp.nb[1], br = blockIdx.x;
  const int bk = br / bxy, bj = (br - bk * bxy) / tp.nb[0], bi = br - bk * bxy - bj * tp.nb[0];
  const int x0 = brick_first(bi, geo.nx, tp.nb[0]), y0 = brick_first(bj, geo.ny, tp.nb[1]),
            z0 = brick_first(bk, geo.nz, tp.nb[2]);
  const int dx = brick_first(bi + 1, geo.nx, tp.nb[0]) - x0,
            dy = brick_first(bj + 1, geo.ny, tp.nb[1]) - y0,
            dz = brick_first(bk + 1, geo.nz, tp.nb[2]) - z0;
  // tables
  for (int k = tid; k < px + 2; k += T) {
    const int x = wrap_near(x0 - 2 + min(k, dx + 3), geo.nx);
    xo[k] = x;
  }
  for (int k = tid; k < py + 2; k += T) {
    const int y = wrap_near(y0 - 2 + min(k, dy + 3), geo.ny);
    yo[k] = y * geo.nx;
  }
  for (int k = tid; k < pz + 2; k += T) {
    const int zz = z0 - 2 + min(k, dz + 3);
    zs[k] = geo.walls ? min(max(zz, 0), geo.nz - 1) : wrap_near(zz, geo.nz);
  }
  if (ph.vel_kind == kVelDeformation) {
    const float inv_l = 1.0f / static_cast<float>(geo.nx);
    for (int k = tid; k < tp.b[0] + tp.b[1] + tp.b[2]; k += T) {
      const int axis = k < tp.b[0] ? 0 : (k < tp.b[0] + tp.b[1] ? 1 : 2);
      const int i = axis == 0 ? k : (axis == 1 ? k - tp.b[0] : k - tp.b[0] - tp.b[1]);
      const float a = static_cast<float>((axis == 0 ? x0 : (axis == 1 ? y0 : z0)) + i) * inv_l;
      float* s = sn + (axis == 0 ? 0 : (axis == 1 ? sny : snz)) + 2 * i;
      s[0] = sinpif(a);
      s[1] = sinpif(2.0f * a);
    }
  }
  __syncthreads();
  const char* state = reinterpret_cast<const char*>(src);
  auto value = [&](int c, int slot) {
    return *reinterpret_cast<const float*>(
        state + static_cast<long long>(c >> kTileShift) * tile_bytes<S>() + (c & (kTile - 1)) * 4 + slot * SL);
  };
  auto pull = [&](int i, int j, int l, float q[7]) {  // places in the tables (region + 1)
    const int z = zs[l], xc = xo[i], yc = yo[j], c = z * geo.plane;
    // across a wall f_5 (f_6) is the cell's own slot 6 (5)
    const bool lo = geo.walls && z == 0, hi = geo.walls && z == geo.nz - 1;
    q[0] = value(c + xc + yc, 0);
    q[1] = value(c + xo[i - 1] + yc, 1);
    q[2] = value(c + xo[i + 1] + yc, 2);
    q[3] = value(c + xc + yo[j - 1], 3);
    q[4] = value(c + xc + yo[j + 1], 4);
    q[5] = value(zs[l - 1] * geo.plane + xc + yc, lo ? 6 : 5);
    q[6] = value(zs[l + 1] * geo.plane + xc + yc, hi ? 5 : 6);
  };
  const int nphi = px * py * (dz + 2);
  constexpr int U = 4;
  for (int k0 = tid; k0 < nphi; k0 += U * T) {
    float q[U][7];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = min(k0 + u * T, nphi - 1);
      const int r = small_div(k, tp.m_px), i = k - r * px;
      const int l = small_div(r, tp.m_py), j = r - l * py;
      int lc = l;
      if (geo.walls) lc = min(max(z0 - 1 + l, 0), geo.nz - 1) - (z0 - 1);
      pull(i + 1, j + 1, lc + 1, q[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (k0 + u * T < nphi)
        sphi[k0 + u * T] =
            q[u][0] + ((q[u][1] + q[u][2]) + (q[u][3] + q[u][4]) + (q[u][5] + q[u][6]));
  }
  __syncthreads();
  const int ncell = tp.b[0] * tp.b[1] * dz;
#pragma unroll 2
  for (int k = tid; k < ncell; k += T) {
    const int r = small_div(k, tp.m_bx), i = k - r * tp.b[0];
    const int l = small_div(r, tp.m_by), j = r - l * tp.b[1];
    if (i >= dx || j >= dy) continue;
    const int x = x0 + i, y = y0 + j, z = z0 + l;
    const int idx = (z * geo.ny + y) * geo.nx + x;
    float f[7], prev[3];
    pull(i + 2, j + 2, l + 2, f);
#pragma unroll
    for (int a = 0; a < 3; ++a) prev[a] = src[phiu_index<S>(idx, a)];
    const float* c = sphi + ((l + 1) * py + j + 1) * px + i + 1;
    const float phi_c = c[0];
    const float mu_c = ph.d3q7_stencil ? region_mu<true>(c, px, px * py, ph)
                                       : region_mu<false>(c, px, px * py, ph);
    float u[3], dphiu[3];
    if (ph.vel_kind == kVelDeformation) {
      const float *sx = sn + 2 * i, *sy = sn + sny + 2 * j, *sz = sn + snz + 2 * l;
      deformation_velocity(ph.vel_U, tf, sx[0], sx[1], sy[0], sy[1], sz[0], sz[1], u);
    } else {
      prescribed_velocity(ph, geo, x, y, z, tf, u);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float cur = __fmul_rn(phi_c, u[a]);
      dphiu[a] = have_prev ? __fsub_rn(cur, prev[a]) : 0.0f;
      dst[phiu_index<S>(idx, a)] = cur;
    }
    collide_d3q7<false>(ph, f, phi_c, mu_c, u, dphiu);
    store_f<kAB, S>(dst, idx, Nbr{}, f);
  }
}

// The same step for grids whose rows are whole tiles, where columns_suit: a block marches up z through a column of
// 32 x 8 cells, one warp per row, two more for the rows beside the column and one for the
// cells beside each row.  In iteration z the
// loads of plane z + 2 are issued, phi of plane z + 1 goes to a ring in shared memory and plane
// z is collided with the f and phi u that were loaded two planes ago: one barrier a plane,
// loads always in flight.  Where a lane's cells lie within a plane does not change from plane
// to plane, so the offsets are worked out once and a load is the plane's address and a
// constant of the lane.
constexpr int kColY = 8;
constexpr int kColThreads = kTile * (kColY + 3);
constexpr int kRing = 4;      // planes of phi: z - 1, z, z + 1, and one that slower warps still read
constexpr int kColSeg = 32;   // planes of a block
constexpr int kColAhead = 5;  // planes ahead of which f and phi u are prefetched into L2

struct Pull {  // byte offsets within a plane of a cell's pulled f: own, x -/+ 1, y -/+ 1
  unsigned c, xm, xp, ym, yp;
};

__device__ __forceinline__ Pull pull_at(const Geometry& geo, int x, int y) {
  const int xm = x ? x - 1 : geo.nx - 1, xp = x != geo.nx - 1 ? x + 1 : 0;
  const int ym = y ? y - 1 : geo.ny - 1, yp = y != geo.ny - 1 ? y + 1 : 0;
  Pull p;
  p.c = cell_bytes<kF32>(y * geo.nx + x);
  p.xm = cell_bytes<kF32>(y * geo.nx + xm);
  p.xp = cell_bytes<kF32>(y * geo.nx + xp);
  p.ym = cell_bytes<kF32>(ym * geo.nx + x);
  p.yp = cell_bytes<kF32>(yp * geo.nx + x);
  return p;
}

__global__ void __launch_bounds__(kColThreads, 2)
    k_track_rows(const float* __restrict__ src, float* __restrict__ dst,
                 const __grid_constant__ Geometry geo, const __grid_constant__ Physics ph,
                 int nbx, int have_prev, float tf) {
  constexpr int TB = tile_bytes<kF32>(), SL = kTile * 4, PX = kTile + 2, PP = (kColY + 2) * PX;
  __shared__ float ring[kRing][PP];
  __shared__ float2 sz[kColSeg];  // sin(pi z / L), sin(2 pi z / L)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bi = blockIdx.x % nbx, bj = blockIdx.x / nbx;
  const int y0 = bj * kColY, z0 = blockIdx.y * kColSeg, z1 = min(z0 + kColSeg, geo.nz);
  const int dy = min(kColY, geo.ny - y0);
  // the thread's cell of each plane: region row j (y0 + j - 1), column i (32 bi + i - 1)
  const bool beside = warp == kColY + 2;
  const int side = lane >= kColY + 2 ? 1 : 0;
  const int j = beside ? lane - side * (kColY + 2) : warp, i = beside ? side * (PX - 1) : lane + 1;
  const bool in = j < dy + 2 && (!beside || lane < 2 * (kColY + 2));
  const bool mine = !beside && j >= 1 && j <= dy;
  const int xx = bi * kTile + i - 1, yy = y0 + j - 1;
  const int x = xx < 0 ? geo.nx - 1 : (xx >= geo.nx ? 0 : xx);
  const int y = yy < 0 ? geo.ny - 1 : (yy >= geo.ny ? 0 : yy);
  const long long plane_b = static_cast<long long>(geo.ny) * nbx * TB;
  const Pull p = pull_at(geo, x, in ? y : 0);
  const int place = j * PX + i;
  const bool deform = ph.vel_kind == kVelDeformation;
  const float inv_l = 1.0f / static_cast<float>(geo.nx);
  float sx = 0, s2x = 0, sy = 0, s2y = 0;
  if (deform) {
    const float ax = static_cast<float>(x) * inv_l, ay = static_cast<float>(y) * inv_l;
    sx = sinpif(ax);
    s2x = sinpif(2.0f * ax);
    sy = sinpif(ay);
    s2y = sinpif(2.0f * ay);
    for (int k = threadIdx.x; k < z1 - z0; k += kColThreads) {
      const float az = static_cast<float>(z0 + k) * inv_l;
      sz[k] = make_float2(sinpif(az), sinpif(2.0f * az));
    }
  }
  auto at = [](const char* plane, unsigned off) { return *reinterpret_cast<const float*>(plane + off); };
  struct Plane {
    float f[7], prev[3];
  };
  auto load = [&](int zz, Plane& v) {
    const int z = geo.walls ? min(max(zz, 0), geo.nz - 1) : (zz < 0 ? geo.nz - 1 : (zz >= geo.nz ? 0 : zz));
    const char* P = reinterpret_cast<const char*>(src) + z * plane_b;
    // across a wall f_5 (f_6) is the cell's own slot 6 (5)
    const char* M = z ? P - plane_b : (geo.walls ? P + SL : P + (geo.nz - 1) * plane_b);
    const char* N = z != geo.nz - 1 ? P + plane_b : (geo.walls ? P - SL : P - (geo.nz - 1) * plane_b);
    if (in) {
      v.f[0] = at(P, p.c);
      v.f[1] = at(P, p.xm + 1 * SL);
      v.f[2] = at(P, p.xp + 2 * SL);
      v.f[3] = at(P, p.ym + 3 * SL);
      v.f[4] = at(P, p.yp + 4 * SL);
      v.f[5] = at(M, p.c + 5 * SL);
      v.f[6] = at(N, p.c + 6 * SL);
    }
    if (mine) {
#pragma unroll
      for (int a = 0; a < 3; ++a) v.prev[a] = at(P, p.c + (kSlotPhiu + a) * SL);
    }
  };
  auto sum = [](const float f[7]) { return f[0] + ((f[1] + f[2]) + (f[3] + f[4]) + (f[5] + f[6])); };
  auto put = [&](int zz, const Plane& v) {
    if (in) ring[(zz + 4) & (kRing - 1)][place] = sum(v.f);
  };
  auto sums = [&](int zz, float& c, float& fs, float& d) {
    const float* r = ring[(zz + 4) & (kRing - 1)] + place;
    c = r[0];
    fs = (r[-1] + r[1]) + (r[-PX] + r[PX]);
    d = (r[-PX - 1] + r[-PX + 1]) + (r[PX - 1] + r[PX + 1]);
  };
  float c0, c1, c2, f1, f2, d0, d1, d2;
  Plane a, b, n;
  load(z0 - 1, n);
  load(z0, a);
  load(z0 + 1, b);
  put(z0 - 1, n);
  put(z0, a);
  __syncthreads();
  if (mine) {
    float unused;
    sums(z0 - 1, c0, unused, d0);
    sums(z0, c1, f1, d1);
  }
#pragma unroll 3
  for (int z = z0; z < z1; ++z) {
    // f and prev: a plane z, b plane z + 1 (in flight)
    if (lane == 0 && mine && z + kColAhead < geo.nz) {
      const char* t = reinterpret_cast<const char*>(src) + (z + kColAhead) * plane_b + p.c;
      prefetch_l2(t, kQ7 * SL);
      prefetch_l2(t + kSlotPhiu * SL, 3 * SL);
    }
    put(z + 1, b);
    if (z + 1 < z1) load(z + 2, n);
    __syncthreads();
    if (mine) {
      sums(z + 1, c2, f2, d2);
      const float lap = ph.d3q7_stencil ? lap7_columns(c0, c1, c2, f1) : lap15_columns(c0, c1, c2, f1, d0, d2);
      const float mu_c = chemical_potential(ph, c1, lap);
      float u[3], dphiu[3];
      if (deform)
        deformation_velocity(ph.vel_U, tf, sx, s2x, sy, s2y, sz[z - z0].x, sz[z - z0].y, u);
      else
        prescribed_velocity(ph, geo, x, y, z, tf, u);
      char* D = reinterpret_cast<char*>(dst) + z * plane_b;
      auto store = [&](unsigned off, float v) { *reinterpret_cast<float*>(D + off) = v; };
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float cur = __fmul_rn(c1, u[k]);
        dphiu[k] = have_prev ? __fsub_rn(cur, a.prev[k]) : 0.0f;
        store(p.c + (kSlotPhiu + k) * SL, cur);
      }
      collide_d3q7<false>(ph, a.f, c1, mu_c, u, dphiu);
#pragma unroll
      for (int i = 0; i < 7; ++i) store(p.c + i * SL, a.f[i]);
      c0 = c1;
      d0 = d1;
      c1 = c2;
      f1 = f2;
      d1 = d2;
    }
    a = b;
    b = n;
  }
}

// How k_track cuts an axis of n cells into bricks of at most `want`.
void cut(int n, int want, int& nb, int& b) {
  nb = (n + want - 1) / want;
  b = (n + nb - 1) / nb;
}

// Whether the columns of k_track_rows suit the grid.  A block marches through its 32 planes one
// after the other, so there have to be as many blocks as SMs, or few planes; columns that hang
// over the grid's last row waste their warps.  Measured, us a step, columns (bricks): 32^3 24.6
// (8.3), 64x33x64 26.8 (14.4), 64x64x400 62 (68); with 5 of 8 rows used 96x5x3541, 333 blocks,
// 56 (45), 96x5x8333 94 (92), 96x5x25000 241 (258); 4 of 8 92.4 (98.3) at 32x4x31250.
bool columns_suit(const Geometry& geo, int sms) {
  const long long segments = (geo.nz + kColSeg - 1) / kColSeg;
  if (geo.row_tiles == 0 || segments > 65535) return false;
  if (geo.nz <= 8) return true;
  const int across = (geo.ny + kColY - 1) / kColY;
  const long long blocks = segments * across * geo.row_tiles;
  if (geo.ny <= kColY / 2 || blocks < sms) return false;
  // two blocks an SM: between one wave and 1.4 a mostly empty second one is worth it only for
  // columns that are nearly full
  return 4 * geo.ny >= 3 * kColY * across || blocks <= 2 * sms || 5 * blocks >= 14 * sms;
}

}  // namespace

// Bricks of few cells (grids thin in two directions) cost more than three passes, whose
// order-parameter and collision passes do not care about the shape, unless the grid fills less
// than half a dozen blocks an SM.  The line is the crossing of two fitted costs in ns a cell:
// bricks 6.5 / (cells of a brick) + 0.019, three passes 8.5 / (cells of a chemical-potential
// block) + 0.0225.  Measured, us a step, three passes (bricks): 8x1x750000 500 (923), 5x2x170000
// 134 (193), 500x2x6000 170 (200), 256x1x15625 146 (164), 8x1x12500 21 (18), 8x53125x4 120 (72),
// 100x4x15000 156 (160), 500x4x3000 148 (138).
bool track_shape_ok(const Geometry& geo, int sms) {
  if (geo.storage != kF32) return false;
  if (columns_suit(geo, sms)) return true;
  const int n[3] = {geo.nx, geo.ny, geo.nz}, want[3] = {32, 8, 8}, mu[3] = {32, 8, 16};
  double brick = 1.0, block = geo.n;
  for (int a = 0; a < 3; ++a) {
    int nb, b;
    cut(n[a], want[a], nb, b);
    brick *= b;
    block /= (n[a] + mu[a] - 1) / mu[a];
  }
  return geo.n <= 21.0 * sms * brick || 6.5 / brick < 8.5 / block + 0.0035;
}

// Rows of whole tiles march up columns in segments of 32 planes (a segment forms phi on one
// plane beyond each end; 256^3: 16 planes 287 us, 32 282, 64 289) and prefetch 5 planes ahead
// (0: 322, 3: 291, 8: 293); other grids take bricks (150^3: 32x8x8 75.9 us, 64x8x4 78.5,
// 32x16x8 81.4).
cudaError_t launch_track(const float* src, float* dst, const Geometry& geo, const Physics& ph,
                         bool have_prev, float tf, int sms, cudaStream_t st) {
  const int prev = have_prev ? 1 : 0;
  if (columns_suit(geo, sms)) {
    const dim3 grid(geo.row_tiles * ((geo.ny + kColY - 1) / kColY), (geo.nz + kColSeg - 1) / kColSeg);
    k_track_rows<<<grid, kColThreads, 0, st>>>(src, dst, geo, ph, geo.row_tiles, prev, tf);
    return cudaGetLastError();
  }
  TrackPlan p{};
  const int n[3] = {geo.nx, geo.ny, geo.nz}, want[3] = {32, 8, 8};
  long long bricks = 1;
  for (int a = 0; a < 3; ++a) {
    cut(n[a], want[a], p.nb[a], p.b[a]);
    bricks *= p.nb[a];
  }
  // exact for the numbers of a brick: k (m d - 2^kBrickDivShift) < 3400 * 34 < 2^kBrickDivShift
  auto small_div_of = [](int d) { return ((1u << kBrickDivShift) + d - 1) / d; };
  p.m_px = small_div_of(p.b[0] + 2);
  p.m_py = small_div_of(p.b[1] + 2);
  p.m_bx = small_div_of(p.b[0]);
  p.m_by = small_div_of(p.b[1]);
  const int smem = 4 * ((p.b[0] + 2) * (p.b[1] + 2) * (p.b[2] + 2) + 3 * (p.b[0] + p.b[1] + p.b[2]) + 12);
  k_track<<<static_cast<unsigned>(bricks), kTrackThreads, smem, st>>>(src, dst, geo, ph, p, prev, tf);
  return cudaGetLastError();
}

}  // namespace lbm
