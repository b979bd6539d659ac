// Many time steps of a small grid in one launch (lbm_brick_*.cu instantiate it, one storage
// type each): the passes of lbm_kernels.cu -- order parameter (Eqs. 13, 16), chemical
// potential (Eq. 2), stream-collide (Eqs. 14-34) -- for boxes whose two state arrays stay in
// the L2 cache (n up to brick_most_cells).
//
// What bounds such a box is not bandwidth but latency: three launches a step, each with a
// ramp, a tail and one round of loads, take 9.2 us at 32^3 and 18.5 us at 64^3, of which the
// arithmetic is 1-3 us.  Here every block keeps one brick of cells for the whole launch
// (all blocks are resident: a cooperative launch) and a step costs one wait: the block
// forms phi on its brick and two cells around it from the streamed f, mu on one cell
// around it, both in shared memory, collides its cells and tells the blocks around it.
// The halo is computed twice or more (2 to 5 times the brick's cells, 40 instructions
// each) to save the two exchanges that passing phi and mu between blocks would take, about
// 2 us each.  Where everything lies -- the byte offset in the state of each cell of the
// brick and of those around it -- is worked out once per launch and kept in shared memory.
// Every value is formed by the operations of the three passes in their order, so the state
// is the same bit for bit.
//
// At 32^3, when a step took 5.1 us (4.9 now), these were the wait (0.6), the loads' issue (0.5), phi
// (0.9), mu (0.5), the collision (1.4) and the release of the stores (0.6), as clocks read
// in the kernel say: latency throughout.  At 64^3 (13.7 us) the collision's
// arithmetic is the largest part.  brick_plan has the times over the sizes.
#pragma once

#include <cuda_runtime.h>

#include "lbm_cells.cuh"
#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

__device__ __forceinline__ int flag_load(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void flag_store(int* p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// First cell of brick i of nb along an axis of n cells (sizes differ by at most one).
__device__ __forceinline__ int brick_first(int i, int n, int nb) {
  return static_cast<int>(static_cast<long long>(i) * n / nb);
}

// v mod n for a v a few cells outside [0, n).
__device__ __forceinline__ int wrap_near(int v, int n) {
  if (v < 0) v += n;
  if (v >= n) v -= n;
  return (v < 0 || v >= n) ? ((v % n) + n) % n : v;
}

// k / d for the numbers of a brick's region, with m = brick_div(d).
__device__ __forceinline__ int small_div(int k, unsigned m) {
  return static_cast<int>((static_cast<unsigned>(k) * m) >> kBrickDivShift);
}

// Byte offset of slot 0 of a cell in the state: 32 bits, the grids of this kernel are small.
template <int S>
__device__ __forceinline__ int cell_bytes(int c) {
  constexpr int EB = static_cast<int>(sizeof(typename Elem<S>::T));
  return (c >> kTileShift) * tile_bytes<S>() + (c & (kTile - 1)) * EB;
}

template <int S>
__device__ __forceinline__ float state_at(const float* state, int bytes) {
  typedef typename Elem<S>::T T;
  return Elem<S>::get(*reinterpret_cast<const T*>(reinterpret_cast<const char*>(state) + bytes));
}

// The 15 values around a place of a region whose rows and planes lie sy and sz apart.
__device__ __forceinline__ void region_stencil(const float* c, int sy, int sz, Stencil& s) {
  s.c = c[0];
  s.xm = c[-1];
  s.xp = c[1];
  s.ym = c[-sy];
  s.yp = c[sy];
  s.zm = c[-sz];
  s.zp = c[sz];
#pragma unroll
  for (int b = 0; b < 8; ++b)
    s.k[b] = c[((b & 1) ? 1 : -1) + ((b & 2) ? sy : -sy) + ((b & 4) ? sz : -sz)];
}

__device__ __forceinline__ StencilV<float2> region_stencil2(const float* c0, const float* c1,
                                                            int sy, int sz) {
  Stencil a, b;
  region_stencil(c0, sy, sz, a);
  region_stencil(c1, sy, sz, b);
  StencilV<float2> v;
  v.c = make_float2(a.c, b.c);
  v.xm = make_float2(a.xm, b.xm);
  v.xp = make_float2(a.xp, b.xp);
  v.ym = make_float2(a.ym, b.ym);
  v.yp = make_float2(a.yp, b.yp);
  v.zm = make_float2(a.zm, b.zm);
  v.zp = make_float2(a.zp, b.zp);
#pragma unroll
  for (int i = 0; i < 8; ++i) v.k[i] = make_float2(a.k[i], b.k[i]);
  return v;
}

// mu at a place of the phi region (the sums of mu_columns in their order).
template <bool D3Q7>
__device__ __forceinline__ float region_mu(const float* c, int sy, int sz, const Physics& ph) {
  const float* a = c - sz;
  const float* b = c + sz;
  const float c0 = a[0], c1 = c[0], c2 = b[0];
  const float f1 = (c[-1] + c[1]) + (c[-sy] + c[sy]);
  float lap;
  if (D3Q7) {
    lap = lap7_columns(c0, c1, c2, f1);
  } else {
    const float d0 = (a[-sy - 1] + a[-sy + 1]) + (a[sy - 1] + a[sy + 1]);
    const float d2 = (b[-sy - 1] + b[-sy + 1]) + (b[sy - 1] + b[sy + 1]);
    lap = lap15_columns(c0, c1, c2, f1, d0, d2);
  }
  return chemical_potential(ph, c1, lap);
}

// Counter of the brick that this thread waits for, of those around brick (bi, bj, bk) that lie
// within the cells a step reads; null for the threads beyond their number.
__device__ __forceinline__ const int* brick_neighbour(const BrickPlan& bp, const int* flags, int bi,
                                                      int bj, int bk) {
  const int tid = threadIdx.x;
  if (tid >= bp.around) return nullptr;
  const int ax = min(bp.nb[0], 2 * bp.reach[0] + 1), ay = min(bp.nb[1], 2 * bp.reach[1] + 1);
  const int k = tid / (ax * ay), j = (tid - k * ax * ay) / ax, i = tid - (k * ay + j) * ax;
  const int ni = wrap_near(bi - bp.reach[0] + i, bp.nb[0]);
  const int nj = wrap_near(bj - bp.reach[1] + j, bp.nb[1]);
  const int nk = wrap_near(bk - bp.reach[2] + k, bp.nb[2]);
  return flags + ((nk * bp.nb[1] + nj) * bp.nb[0] + ni) * kBrickFlag;
}

// MODE: kBrickCoupled, or kBrickTracking (prescribed velocity: only f evolves, mu is needed
// at the brick's own cells only, so the halo is one cell narrower and there is no mu region).
// NC cells per thread at a time in the coupled collision: 1, or 2 in the lanes of paired
// arithmetic (bricks of many cells, where issue counts more than the spare warps).
template <int MODE, int VAR, int S, int NC>
__global__ void __launch_bounds__(kBrickThreads, NC == 1 ? 3 : 2)
    k_brick(float* state0, float* state1, float* phi, const __grid_constant__ Geometry geo,
            const __grid_constant__ Physics ph, const __grid_constant__ BrickPlan bp,
            const __grid_constant__ BrickTimes times, int* flags, int base, int have_prev, int* err,
            long long polls) {
  extern __shared__ float smem[];
  constexpr bool TRACK = MODE == kBrickTracking;
  constexpr bool D3Q7 = (VAR & kVarD3Q7) != 0;
  constexpr int H = TRACK ? 1 : 2;                // halo of phi
  constexpr int SL = kTile * static_cast<int>(sizeof(typename Elem<S>::T));  // bytes of a slot
  constexpr int T = kBrickThreads;
  const int tid = threadIdx.x;
  const int px = bp.b[0] + 2 * H, py = bp.b[1] + 2 * H;          // phi region
  const int mx = bp.b[0] + 2, my = bp.b[1] + 2;                  // mu region (coupled)
  const int qx = bp.b[0] + 2 * H + 2, qy = bp.b[1] + 2 * H + 2;  // where pulled values lie
  float* sphi = smem;
  float* smu = smem + px * py * (bp.b[2] + 2 * H);
  int* sat = reinterpret_cast<int*>(TRACK ? smu : smu + mx * my * (bp.b[2] + 2));

  // this block's brick and the blocks around it
  const int br = blockIdx.x, bxy = bp.nb[0] * bp.nb[1];
  const int bk = br / bxy, bj = (br - bk * bxy) / bp.nb[0], bi = br - bk * bxy - bj * bp.nb[0];
  const int x0 = brick_first(bi, geo.nx, bp.nb[0]), y0 = brick_first(bj, geo.ny, bp.nb[1]),
            z0 = brick_first(bk, geo.nz, bp.nb[2]);
  const int dx = brick_first(bi + 1, geo.nx, bp.nb[0]) - x0,
            dy = brick_first(bj + 1, geo.ny, bp.nb[1]) - y0,
            dz = brick_first(bk + 1, geo.nz, bp.nb[2]) - z0;
  const int* neighbour = brick_neighbour(bp, flags, bi, bj, bk);

  // byte offsets of the brick's cells and of those around it (beyond the brick's last row or
  // column, where bricks differ in size, those of the last one: never used)
  for (int k = tid; k < qx * qy * (dz + 2 * H + 2); k += T) {
    const int r = small_div(k, bp.m_qx), i = k - r * qx;
    const int l = small_div(r, bp.m_qy), j = r - l * qy;
    const int x = wrap_near(x0 - H - 1 + min(i, dx + 2 * H + 1), geo.nx);
    const int y = wrap_near(y0 - H - 1 + min(j, dy + 2 * H + 1), geo.ny);
    const int zz = z0 - H - 1 + l;
    // across a wall f_5 (f_6) is the cell's own slot 6 (5), one slot further (back)
    int z, slot = 0;
    if (geo.walls) {
      z = min(max(zz, 0), geo.nz - 1);
      slot = zz < 0 ? SL : (zz >= geo.nz ? -SL : 0);
    } else {
      z = wrap_near(zz, geo.nz);
    }
    sat[k] = cell_bytes<S>((z * geo.ny + y) * geo.nx + x) + slot;
  }
  const int nphi = px * py * (dz + 2 * H);
  // The plane of the region that stands for plane l: beyond a wall the wall's own cells.
  auto real_plane = [&](int l, int first) {
    return geo.walls ? min(max(first + l, 0), geo.nz - 1) - first : l;
  };
  if (S != kF32) {
    // slot 0 holds f_0 - phi of the step that wrote it: from the phi array for the first
    // step, after it the region's own values of the step before
    for (int k = tid; k < nphi; k += T) {
      const int r = small_div(k, bp.m_px), i = k - r * px;
      const int l = small_div(r, bp.m_py), j = r - l * py;
      const int x = wrap_near(x0 - H + min(i, dx + 2 * H - 1), geo.nx);
      const int y = wrap_near(y0 - H + min(j, dy + 2 * H - 1), geo.ny);
      const int z = wrap_near(z0 - H + real_plane(l, z0 - H), geo.nz);
      sphi[k] = phi[(z * geo.ny + y) * geo.nx + x];
    }
  }
  __syncthreads();

  const int ncell = bp.b[0] * bp.b[1] * dz;
  struct At {
    int idx, x, y, z;
    int ci, cm, ca;  // its places in the phi, mu and offset regions
    bool in, wlo, whi;
  };
  auto place = [&](int k) {
    At a;
    const int r = small_div(k, bp.m_bx), i = k - r * bp.b[0];
    const int l = small_div(r, bp.m_by), j = r - l * bp.b[1];
    a.in = k < ncell && i < dx && j < dy;
    const int ii = min(i, dx - 1), jj = min(j, dy - 1), ll = min(l, dz - 1);
    a.x = x0 + ii;
    a.y = y0 + jj;
    a.z = z0 + ll;
    a.idx = (a.z * geo.ny + a.y) * geo.nx + a.x;
    a.wlo = geo.walls && a.z == 0;
    a.whi = geo.walls && a.z == geo.nz - 1;
    a.ci = ((ll + H) * py + jj + H) * px + ii + H;
    a.cm = ((ll + 1) * my + jj + 1) * mx + ii + 1;
    a.ca = ((ll + H + 1) * qy + jj + H + 1) * qx + ii + H + 1;
    return a;
  };
  for (int t = 0; t < bp.steps; ++t) {
    const float* src = (t & 1) ? state1 : state0;
    float* dst = (t & 1) ? state0 : state1;
    const int hp = t > 0 ? 1 : have_prev;
    const bool last = t == bp.steps - 1;
    if (t > 0) {
      // Every block around has taken step t - 1: what it wrote is here, and what it read
      // may be overwritten.
      bool ok = true;
      if (neighbour) {
        ok = false;
        for (long long q = 0; q < polls; ++q) {
          if (flag_load(neighbour) - base >= t) {
            ok = true;
            break;
          }
          if ((q & 63) == 63 && flag_load(err) != 0) break;
        }
      }
      if (!__syncthreads_and(ok)) {
        if (tid == 0) atomicMax(err, 1);
        return;
      }
    }
    // The first cells' populations, loaded now so that they arrive while phi and mu form.
    At at[NC];
    float g[NC][15], f[NC][7], prev[NC][3];
    auto load = [&](int k) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        at[c] = place(k + c * T);
        const At& a = at[c];
        const int* o = sat + a.ca;
#define X(I, O, CX, CY, CZ) f[c][I] = state_at<S>(src, o[-CX - CY * qx - CZ * qx * qy] + I * SL);
        LBM_D3Q7_LIST(X)
#undef X
        if (!TRACK) {
          if (a.wlo || a.whi) {
            load_g<kAB, S>(src, a.idx, make_nbr(geo, a.x, a.y, a.z), g[c]);
          } else {
#define X(I, O, CX, CY, CZ) g[c][I] = state_at<S>(src, o[-CX - CY * qx - CZ * qx * qy] + (7 + I) * SL);
            LBM_D3Q15_LIST(X)
#undef X
          }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) prev[c][i] = src[phiu_index<S>(a.idx, i)];
      }
    };
    load(tid);
    // phi on the region
    constexpr int U = NC == 1 && S == kF32 ? 5 : 4;
    for (int k0 = tid; k0 < nphi; k0 += U * T) {
      float q[U][7];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = min(k0 + u * T, nphi - 1);
        const int r = small_div(k, bp.m_px), i = k - r * px;
        const int l = small_div(r, bp.m_py), j = r - l * py;
        const int* o = sat + ((real_plane(l, z0 - H) + 1) * qy + j + 1) * qx + i + 1;
#define X(I, O, CX, CY, CZ) q[u][I] = state_at<S>(src, o[-CX - CY * qx - CZ * qx * qy] + I * SL);
        LBM_D3Q7_LIST(X)
#undef X
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u * T;
        if (k < nphi) {
          const float f0 = S != kF32 ? q[u][0] + sphi[k] : q[u][0];
          sphi[k] = f0 + ((q[u][1] + q[u][2]) + (q[u][3] + q[u][4]) + (q[u][5] + q[u][6]));
        }
      }
    }
    __syncthreads();
    if (!TRACK) {
      // mu on the brick and one cell around it; beyond a wall, of the wall's own cells
      const int nmu = mx * my * (dz + 2);
#pragma unroll 3
      for (int k = tid; k < nmu; k += T) {
        const int r = small_div(k, bp.m_mx), i = k - r * mx;
        const int l = small_div(r, bp.m_my), j = r - l * my;
        const float* c = sphi + ((real_plane(l, z0 - 1) + 1) * py + j + 1) * px + i + 1;
        smu[k] = region_mu<D3Q7>(c, px, px * py, ph);
      }
      __syncthreads();
    }
    for (int k = tid; k - tid < ncell; k += NC * T) {
      if (k != tid) load(k);
      if (TRACK) {
        const At& a = at[0];
        if (a.in) {
          const float* c = sphi + a.ci;
          const float phi_c = c[0];
          const float mu_c = ph.d3q7_stencil ? region_mu<true>(c, px, px * py, ph)
                                             : region_mu<false>(c, px, px * py, ph);
          float u[3], dphiu[3];
          prescribed_velocity(ph, geo, a.x, a.y, a.z, times.tf[t], u);
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const float cur = __fmul_rn(phi_c, u[i]);
            dphiu[i] = hp ? __fsub_rn(cur, prev[0][i]) : 0.0f;
            dst[phiu_index<S>(a.idx, i)] = cur;
          }
          collide_d3q7<S != kF32>(ph, f[0], phi_c, mu_c, u, dphiu);
          store_f<kAB, S>(dst, a.idx, Nbr{}, f[0]);
          if (S != kF32 && last) phi[a.idx] = phi_c;
        }
      } else if (NC == 1) {
        const At& a = at[0];
        if (a.in) {
          Nbr nb{};
          nb.wlo = a.wlo;
          nb.whi = a.whi;
          collide_loaded<kAB, VAR, S, false>(
              dst, geo, ph, hp, a.idx, nb, g[0], f[0], prev[0],
              [&] {
                CellStencils cs;
                Stencil st;
                region_stencil(sphi + a.ci, px, px * py, st);
                if (D3Q7)
                  stencil_grad7(st, cs.grad_phi);
                else
                  stencil_grad(st, cs.grad_phi);
                cs.phi = st.c;
                region_stencil(smu + a.cm, mx, mx * my, st);
                cs.lap_mu = D3Q7 ? stencil_lap7(st) : stencil_lap(st);
                cs.mu = st.c;
                return cs;
              },
              nullptr);
          if (S != kF32 && last) phi[a.idx] = sphi[a.ci];
        }
      } else {
        constexpr int B = NC - 1;  // the second cell
        const bool in0 = at[0].in, in1 = at[B].in;
        if (in0 || in1) {
          // a cell beyond the brick: the other one's stencils, its result not stored
          const int c0 = in0 ? at[0].ci : at[B].ci, c1 = in1 ? at[B].ci : at[0].ci;
          const int m0 = in0 ? at[0].cm : at[B].cm, m1 = in1 ? at[B].cm : at[0].cm;
          const StencilV<float2> sp = region_stencil2(sphi + c0, sphi + c1, px, px * py);
          const StencilV<float2> sm = region_stencil2(smu + m0, smu + m1, mx, mx * my);
          float2 g2[15], f2[7], p2[3], cur[3];
#pragma unroll
          for (int i = 0; i < 15; ++i) g2[i] = make_float2(g[0][i], g[B][i]);
#pragma unroll
          for (int i = 0; i < 7; ++i) f2[i] = make_float2(f[0][i], f[B][i]);
#pragma unroll
          for (int i = 0; i < 3; ++i) p2[i] = make_float2(prev[0][i], prev[B][i]);
          pair_compute<VAR, S>(ph, hp, g2, f2, p2, sp, sm, cur);
          auto put = [&](const At& a, int lane2) {
            const Nbr nb{};
            float v[15];
#pragma unroll
            for (int i = 0; i < 15; ++i) v[i] = lane2 ? g2[i].y : g2[i].x;
            store_g<kAB, S>(dst, a.idx, nb, v);
#pragma unroll
            for (int i = 0; i < 3; ++i)
              dst[phiu_index<S>(a.idx, i)] = lane2 ? cur[i].y : cur[i].x;
#pragma unroll
            for (int i = 0; i < 7; ++i) v[i] = lane2 ? f2[i].y : f2[i].x;
            store_f<kAB, S>(dst, a.idx, nb, v);
            if (S != kF32 && last) phi[a.idx] = sphi[a.ci];
          };
          if (in0) put(at[0], 0);
          if (in1) put(at[B], 1);
        }
      }
    }
    __syncthreads();
    if (tid == 0) flag_store(flags + br * kBrickFlag, base + t + 1);
  }
}

// The same for the in-place pattern.  A neighbour's f may already be overwritten when a halo
// would be formed from it, so phi is passed between blocks instead of computed twice: a block
// forms phi of its own cells, writes it and tells the blocks around it, waits for theirs, reads
// the halo of phi, forms mu and collides -- two waits a step.  `odd`: parity of the stored
// populations at the first step.  phi holds the order parameter of the step before (16-bit
// storage) and of each step in turn.
// Measured per step, three passes -> bricks: 16^3 9.2 -> 6.1 us, 32^3 9.2 -> 8.8; tracking 32^3
// 14.4 -> 6.9, 64^3 19.2 -> 12.4.
template <int MODE, int VAR, int S>
__global__ void __launch_bounds__(kBrickThreads, 3)
    k_brick_aa(float* state, float* phi, const __grid_constant__ Geometry geo,
               const __grid_constant__ Physics ph, const __grid_constant__ BrickPlan bp,
               const __grid_constant__ BrickTimes times, int* flags, int base, int have_prev, int odd,
               int* err, long long polls) {
  extern __shared__ float smem[];
  constexpr bool TRACK = MODE == kBrickTracking;
  constexpr bool D3Q7 = (VAR & kVarD3Q7) != 0;
  constexpr int H = TRACK ? 1 : 2, T = kBrickThreads;
  const int tid = threadIdx.x;
  const int px = bp.b[0] + 2 * H, py = bp.b[1] + 2 * H;
  const int mx = bp.b[0] + 2, my = bp.b[1] + 2;
  float* sphi = smem;
  float* smu = smem + px * py * (bp.b[2] + 2 * H);
  const int br = blockIdx.x, bxy = bp.nb[0] * bp.nb[1];
  const int bk = br / bxy, bj = (br - bk * bxy) / bp.nb[0], bi = br - bk * bxy - bj * bp.nb[0];
  const int x0 = brick_first(bi, geo.nx, bp.nb[0]), y0 = brick_first(bj, geo.ny, bp.nb[1]),
            z0 = brick_first(bk, geo.nz, bp.nb[2]);
  const int dx = brick_first(bi + 1, geo.nx, bp.nb[0]) - x0,
            dy = brick_first(bj + 1, geo.ny, bp.nb[1]) - y0,
            dz = brick_first(bk + 1, geo.nz, bp.nb[2]) - z0;
  const int* neighbour = brick_neighbour(bp, flags, bi, bj, bk);
  const int nphi = px * py * (dz + 2 * H);
  auto real_plane = [&](int l, int first) {
    return geo.walls ? min(max(first + l, 0), geo.nz - 1) - first : l;
  };
  // one wait for every block around to have reached `step` (in half steps)
  auto wait = [&](int step) {
    bool ok = true;
    if (neighbour) {
      ok = false;
      for (long long q = 0; q < polls; ++q) {
        if (flag_load(neighbour) - base >= step) {
          ok = true;
          break;
        }
        if ((q & 63) == 63 && flag_load(err) != 0) break;
      }
    }
    if (__syncthreads_and(ok)) return true;
    if (tid == 0) atomicMax(err, 1);
    return false;
  };
  const int ncell = bp.b[0] * bp.b[1] * dz;
  struct At {
    int idx, x, y, z, ci, cm;
    bool in;
  };
  auto place = [&](int k) {
    At a;
    const int r = small_div(k, bp.m_bx), i = k - r * bp.b[0];
    const int l = small_div(r, bp.m_by), j = r - l * bp.b[1];
    a.in = k < ncell && i < dx && j < dy;
    const int ii = min(i, dx - 1), jj = min(j, dy - 1), ll = min(l, dz - 1);
    a.x = x0 + ii;
    a.y = y0 + jj;
    a.z = z0 + ll;
    a.idx = (a.z * geo.ny + a.y) * geo.nx + a.x;
    a.ci = ((ll + H) * py + jj + H) * px + ii + H;
    a.cm = ((ll + 1) * my + jj + 1) * mx + ii + 1;
    return a;
  };
  for (int t = 0; t < bp.steps; ++t) {
    const bool odd_step = ((odd + t) & 1) != 0;
    const int hp = t > 0 ? 1 : have_prev;
    if (t > 0 && !wait(2 * t)) return;
    // the first cells' populations are kept for their collision
    At at = place(tid);
    Nbr nb = make_nbr(geo, at.x, at.y, at.z);
    float g[15], f[7], prev[3];
    auto load = [&](const At& a, const Nbr& n) {
      if (TRACK) {
        odd_step ? load_f<kAAOdd, S>(state, a.idx, n, f) : load_f<kAAEven, S>(state, a.idx, n, f);
#pragma unroll
        for (int i = 0; i < 3; ++i) prev[i] = state[phiu_index<S>(a.idx, i)];
      } else if (odd_step) {
        load_cell<kAAOdd, S, true>(state, geo, a.idx, n, g, f, prev);
      } else {
        load_cell<kAAEven, S, true>(state, geo, a.idx, n, g, f, prev);
      }
    };
    auto own_phi = [&](const At& a, const float* v) {
      const float f0 = S != kF32 ? v[0] + phi[a.idx] : v[0];
      const float p = f0 + ((v[1] + v[2]) + (v[3] + v[4]) + (v[5] + v[6]));
      if (a.in) {
        sphi[a.ci] = p;
        phi[a.idx] = p;
      }
    };
    load(at, nb);
    for (int k = tid + T; k - tid < ncell; k += T) {
      const At a = place(k);
      const Nbr n = make_nbr(geo, a.x, a.y, a.z);
      float q[7];
      odd_step ? load_f<kAAOdd, S>(state, a.idx, n, q) : load_f<kAAEven, S>(state, a.idx, n, q);
      own_phi(a, q);
    }
    own_phi(at, f);
    __syncthreads();
    if (tid == 0) flag_store(flags + br * kBrickFlag, base + 2 * t + 1);
    if (!wait(2 * t + 1)) return;
#pragma unroll 4
    for (int k = tid; k < nphi; k += T) {
      const int r = small_div(k, bp.m_px), i = k - r * px;
      const int l = small_div(r, bp.m_py), j = r - l * py;
      if (i >= H && i < dx + H && j >= H && j < dy + H && l >= H && l < dz + H) continue;
      const int x = wrap_near(x0 - H + min(i, dx + 2 * H - 1), geo.nx);
      const int y = wrap_near(y0 - H + min(j, dy + 2 * H - 1), geo.ny);
      const int z = wrap_near(z0 - H + real_plane(l, z0 - H), geo.nz);
      sphi[k] = phi[(z * geo.ny + y) * geo.nx + x];
    }
    __syncthreads();
    if (!TRACK) {
      const int nmu = mx * my * (dz + 2);
#pragma unroll 3
      for (int k = tid; k < nmu; k += T) {
        const int r = small_div(k, bp.m_mx), i = k - r * mx;
        const int l = small_div(r, bp.m_my), j = r - l * my;
        const float* c = sphi + ((real_plane(l, z0 - 1) + 1) * py + j + 1) * px + i + 1;
        smu[k] = region_mu<D3Q7>(c, px, px * py, ph);
      }
      __syncthreads();
    }
    for (int k = tid; k - tid < ncell; k += T) {
      if (k != tid) {
        at = place(k);
        nb = make_nbr(geo, at.x, at.y, at.z);
        load(at, nb);
      }
      if (!at.in) continue;
      if (TRACK) {
        const float* c = sphi + at.ci;
        const float phi_c = c[0];
        const float mu_c = ph.d3q7_stencil ? region_mu<true>(c, px, px * py, ph)
                                           : region_mu<false>(c, px, px * py, ph);
        float u[3], dphiu[3];
        prescribed_velocity(ph, geo, at.x, at.y, at.z, times.tf[t], u);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const float cur = __fmul_rn(phi_c, u[i]);
          dphiu[i] = hp ? __fsub_rn(cur, prev[i]) : 0.0f;
          state[phiu_index<S>(at.idx, i)] = cur;
        }
        collide_d3q7<S != kF32>(ph, f, phi_c, mu_c, u, dphiu);
        odd_step ? store_f<kAAOdd, S>(state, at.idx, nb, f) : store_f<kAAEven, S>(state, at.idx, nb, f);
      } else {
        auto stencils = [&] {
          CellStencils cs;
          Stencil st;
          region_stencil(sphi + at.ci, px, px * py, st);
          if (D3Q7)
            stencil_grad7(st, cs.grad_phi);
          else
            stencil_grad(st, cs.grad_phi);
          cs.phi = st.c;
          region_stencil(smu + at.cm, mx, mx * my, st);
          cs.lap_mu = D3Q7 ? stencil_lap7(st) : stencil_lap(st);
          cs.mu = st.c;
          return cs;
        };
        if (odd_step)
          collide_loaded<kAAOdd, VAR, S, false>(state, geo, ph, hp, at.idx, nb, g, f, prev, stencils, nullptr);
        else
          collide_loaded<kAAEven, VAR, S, false>(state, geo, ph, hp, at.idx, nb, g, f, prev, stencils, nullptr);
      }
    }
    __syncthreads();
    if (tid == 0) flag_store(flags + br * kBrickFlag, base + 2 * t + 2);
  }
}

// Sums of the state as launch_collide_sums forms them, from the post-collision values the
// last step stored (pattern AB; with 16-bit storage phi of that step), in one launch: block b
// sums the warps' tiles [b chunk, (b + 1) chunk) of launch_step_sums_final's first pass, the
// last block to finish its second.  Same values in the same order, so the same bits.
constexpr int kSumTiles = 64;  // most tiles of a block
template <int S>
__global__ void __launch_bounds__(kBlock) k_state_sums(const float* __restrict__ state,
                                                       const float* __restrict__ phi,
                                                       const __grid_constant__ Geometry geo,
                                                       int ntiles, int chunk,
                                                       double* __restrict__ partial, double* out,
                                                       const double* word, int* count) {
  __shared__ float parts[kSumTiles * 5];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t0 = blockIdx.x * chunk, nt = min(ntiles, t0 + chunk) - t0;
  for (int k = warp; k < nt; k += kBlock / 32) {
    const int idx = (t0 + k) * kTile + lane;
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    bool bad = false;
    if (idx < geo.n) {
      float f[7], g[15];
      load_f<kAAEven, S>(state, idx, Nbr{}, f);  // the cell's own slots
      load_g<kAAEven, S>(state, idx, Nbr{}, g);
      int x, y, z;
      cell_coords(geo, idx, x, y, z);
      const Nbr nb = make_nbr(geo, x, y, z);
      if (S != kF32) f[0] += phi[idx];
      s[0] = f[0] + ((f[1] + f[2]) + (f[3] + f[4]) + (f[5] + f[6]));
      momentum_sums(g, nb, s + 1);
      bad = !(isfinite(s[0]) && isfinite(s[1]) && isfinite(s[2]) && isfinite(s[3]));
    }
    warp_sums_store(s, bad, parts, static_cast<long long>(k) * kTile);
  }
  __syncthreads();
  // k_reduce_chunks' tree over 256 threads, of which only the first nt <= 64 hold values
  if (warp < 5) {
    double v = lane < nt ? parts[lane * 5 + warp] : 0.0;
    if (lane + 32 < nt) v += parts[(lane + 32) * 5 + warp];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) {
      partial[blockIdx.x * 5 + warp] = v;
      __threadfence();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(count, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // k_reduce_final: thread t of 256 takes partials t, t + 256, ...; here lane l of one warp
  // stands for the threads l, l + 32, ..., l + 224
  if (warp < 5) {
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[j] = 0.0;
      for (int b = lane + 32 * j; b < static_cast<int>(gridDim.x); b += 256)
        v[j] += __ldcg(partial + b * 5 + warp);
    }
#pragma unroll
    for (int w = 4; w > 0; w >>= 1)
#pragma unroll
      for (int j = 0; j < w; ++j) v[j] += v[j + w];
    double r = v[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
    if (lane == 0) out[warp] = r;
  }
  if (threadIdx.x == 0) {
    *count = 0;
    if (word) out[7] = *word;
  }
}

template <int S>
cudaError_t state_sums(const float* state, const float* phi, const Geometry& geo, double* partial,
                       double* out, const double* word, int* count, cudaStream_t st) {
  const int ntiles = cell_warps(geo.n);
  const int groups = ntiles < kReduceMaxParts ? ntiles : kReduceMaxParts;
  const int chunk = (ntiles + groups - 1) / groups;
  if (chunk > kSumTiles) return cudaErrorInvalidValue;
  k_state_sums<S><<<groups, kBlock, 0, st>>>(state, phi, geo, ntiles, chunk, partial, out, word, count);
  return cudaGetLastError();
}

// The instance for (mode, variant, cells per thread; in place) of storage S.
template <int S>
const void* brick_kernel(int mode, int var, bool pair, bool in_place) {
#define LBM_BRICK_AA(MODE, VAR) reinterpret_cast<const void*>(&k_brick_aa<MODE, VAR, S>)
  if (in_place) {
    if (mode == kBrickTracking) return LBM_BRICK_AA(kBrickTracking, 0);
    return var == 0               ? LBM_BRICK_AA(kBrickCoupled, 0)
           : var == kVarSrtFlow   ? LBM_BRICK_AA(kBrickCoupled, kVarSrtFlow)
           : var == kVarD3Q7      ? LBM_BRICK_AA(kBrickCoupled, kVarD3Q7)
                                  : LBM_BRICK_AA(kBrickCoupled, kVarSrtFlow | kVarD3Q7);
  }
#undef LBM_BRICK_AA
// two cells per thread with FP32 populations only (brick_plan)
#define LBM_BRICK(MODE, VAR)                                                       \
  (pair && S == kF32 ? reinterpret_cast<const void*>(&k_brick<MODE, VAR, S, kPair>) \
                     : reinterpret_cast<const void*>(&k_brick<MODE, VAR, S, 1>))
  constexpr int kPair = S == kF32 ? 2 : 1;
  if (mode == kBrickTracking)
    return reinterpret_cast<const void*>(&k_brick<kBrickTracking, 0, S, 1>);
  switch (var) {
    case 0: return LBM_BRICK(kBrickCoupled, 0);
    case kVarSrtFlow: return LBM_BRICK(kBrickCoupled, kVarSrtFlow);
    case kVarD3Q7: return LBM_BRICK(kBrickCoupled, kVarD3Q7);
    default: return LBM_BRICK(kBrickCoupled, kVarSrtFlow | kVarD3Q7);
  }
#undef LBM_BRICK
}

}  // namespace lbm
