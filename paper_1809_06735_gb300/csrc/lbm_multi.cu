// Several time steps per pass over memory (temporal blocking) of the batched
// FP32 stream-collide: eq. (1) advanced by T = 2..4 steps between one read
// and one write of the populations, for double-buffer storage.
//
// The single-step kernel moves 72 B per lattice update and runs at 92-97% of
// the copy bandwidth, so only fewer bytes per update make it faster.  Here a
// group of warps sweeps a block of rows upwards.  Per row it pulls the state
// n from memory and collides it (stage 1); stage s + 1 pulls from stage s's
// post-collision rows, which never leave the SM:
//   - along x the one-cell shift is a warp shuffle, and between the warps of
//     a group an exchange of the edge cells through shared memory;
//   - along y the rows y - 1 and y of stage s wait in shared memory slots
//     private to each thread (c_y = 0 populations one row, c_y = +1 two rows,
//     c_y = -1 none): 144 B per thread and stage, no bank conflicts and no
//     barrier.
// Stage T's rows go to the other population buffer: 72 / T bytes per update
// plus the T - 1 extra rows on each side of a block.
//
// A group is the G = ceil(nx / 128) warps of a whole periodic row where that
// is at most 8 (no column is computed twice, a barrier per stage), or a strip
// of one warp whose first and last lane hold a halo of four columns (T <= 4
// needs three; no barrier).
//
// Two cells per packed FP32 instruction (collide2_f32): with collide_f32 the
// kernel ran 6.1 warp instructions per update and was bound by the issue
// slots (64 x 512^2, T = 3: 162 us per step, single-step kernel 183 us); with
// 2.5 it is bound by memory at T = 2 and 3 and by latency and issue at T = 4.
// Measured, us per step, single-step kernel / T = 2 / 3 / 4: decaying 64 x
// 512^2 183 / 98 / 68.5 / 77 (T = 3: 245 GLUPS, 87% of the copy bandwidth at
// 24 B), forced 8192^2 755 / 444 / 351 / 383, 15 forced members of 256^2 ..
// 1024^2 79 / 52 / 45 / 50 (strips; whole rows 55 at T = 3: the barrier of 8
// warps costs more than the halo lanes).
#include <algorithm>

#include "lbm_collide.cuh"

namespace lbm {

namespace {

// The delay slots of one stage boundary: populations 0, 1, 3 (c_y = 0) of the
// last row, 2, 5, 6 (c_y = +1) of the last two rows.
constexpr int kDelaySlots = 9;

template <int T>
constexpr size_t multi_smem() {
  return (size_t)(T - 1) * (kDelaySlots * 32 * kMultiWarps * sizeof(float4) +
                            2 * kMultiWarps * 8 * sizeof(float)) +
         kMultiWarps * 2 * kQ * sizeof(float);
}

__device__ __forceinline__ void group_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void copy_async4(float *s, const float *g) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(s)),
               "l"(g)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// One row's loads of the pull (double-buffer layout): four cells per
// population and lane, and the cell beyond the warp's columns that the x-shift
// needs, by the warp's first and last lane into their slots e[l] of shared
// memory (read by the same lane; a register per population less).
__device__ __forceinline__ void multi_load(const float *__restrict__ src, size_t plane, int pitch,
                                           int y, int ny, int x, int xprev, int xnext, bool first,
                                           bool last, ulonglong2 (&o)[kQ], float *e) {
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y + 1 == ny ? 0 : y + 1;
  const size_t r[3] = {(size_t)yp * pitch, (size_t)y * pitch, (size_t)ym * pitch};
#pragma unroll
  for (int l = 0; l < kQ; ++l) {
    const float *row = src + (size_t)l * plane + r[1 + cy_of(l)];
    o[l] = __ldg(reinterpret_cast<const ulonglong2 *>(row + x));
    if (cx_of(l) > 0 && first) copy_async4(e + l, row + xprev);
    if (cx_of(l) < 0 && last) copy_async4(e + l, row + xnext);
  }
}

// A lane's four cells as two pairs, moved one cell to the right (prev enters)
// or to the left (next enters).
__device__ __forceinline__ void shift_right(f32x2 (&v)[2], float prev) {
  float a, b, c, d;
  unpack2(v[0], a, b);
  unpack2(v[1], c, d);
  v[0] = pack2(prev, a);
  v[1] = pack2(b, c);
}
__device__ __forceinline__ void shift_left(f32x2 (&v)[2], float next) {
  float a, b, c, d;
  unpack2(v[0], a, b);
  unpack2(v[1], c, d);
  v[0] = pack2(b, c);
  v[1] = pack2(d, next);
}
__device__ __forceinline__ float first_of(const f32x2 (&v)[2]) {
  float a, b;
  unpack2(v[0], a, b);
  return a;
}
__device__ __forceinline__ float last_of(const f32x2 (&v)[2]) {
  float a, b;
  unpack2(v[1], a, b);
  return b;
}

// T steps of the members' rows (BGK, or ELBM: the entropic collision; FORCED:
// some member has a force or drag).
template <int T, bool FORCED, bool ELBM>
__global__ void __launch_bounds__(32 * kMultiWarps, 2)
    k_multi(const Member *__restrict__ members, const MultiWarp *__restrict__ tab, int ctas, int cur,
            int flip) {
  extern __shared__ ulonglong2 delay[];  // [T - 1][kDelaySlots][256], then the edge cells
  constexpr int kS = 32 * kMultiWarps;
  float *edges = reinterpret_cast<float *>(delay + (T - 1) * kDelaySlots * kS);
  const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
  const int cta = flip ? ctas - 1 - (int)blockIdx.x : (int)blockIdx.x;
  const MultiWarp W = tab[(size_t)cta * kMultiWarps + warp];
  if (W.member < 0) return;  // whole groups
  const Member &M = members[W.member];
  const int nx = M.nx, ny = M.ny, pitch = M.pitch;
  const size_t plane = M.plane;
  const float *__restrict__ src = static_cast<const float *>(M.pop[cur]);
  float *__restrict__ dst = static_cast<float *>(M.pop[cur ^ 1]);
  const float *__restrict__ fxt = static_cast<const float *>(M.fx_tab);
  const float rho0 = M.rho0_f, om = M.omega_f, alpha = FORCED ? M.alpha_f : 0.f;
  // columns: xu unwrapped (a strip's halo may lie past the grid's edges); a
  // lane past the last column works on column 0 and stores nothing
  const int xu = W.x0 + 4 * lane;
  const bool active = xu < W.xend;
  const int x = !active ? 0 : (xu < 0 ? xu + nx : (xu >= nx ? xu - nx : xu));
  const bool first = lane == 0, last = active && (lane == 31 || xu + 4 >= W.xend);
  const int lastlane = min(31, (W.xend - W.x0) / 4 - 1);
  const int xprev = x == 0 ? nx - 1 : x - 1, xnext = x + 4 >= nx ? 0 : x + 4;
  const bool out = active && xu >= W.out0 && xu < W.out1;
  const int lprev = lane == 0 ? lastlane : lane - 1, lnext = lane == lastlane ? 0 : lane + 1;
  // the group's warps in the CTA and the neighbours' slots in the edge table
  const int base = warp - W.w, wp = base + (W.w == 0 ? W.g - 1 : W.w - 1),
            wn = base + (W.w + 1 == W.g ? 0 : W.w + 1);
  f32x2 fy[2] = {0, 0};
  if (FORCED) {
    const ulonglong2 q =
        __ldg(reinterpret_cast<const ulonglong2 *>(static_cast<const float *>(M.fy_tab) + x));
    fy[0] = q.x;
    fy[1] = q.y;
  }

  const int R = W.rows + 2 * (T - 1);
  int ya = wrapi(W.y0 - (T - 1), ny);
  ulonglong2 o[kQ];
  float fx[T], fxn = 0.f;  // fx[s]: the force of stage s's row
  float *e = edges + 2 * (T - 1) * kMultiWarps * 8 + (warp * 2 + (first ? 0 : 1)) * kQ;
#pragma unroll
  for (int s = 0; s < T; ++s) fx[s] = 0.f;
  multi_load(src, plane, pitch, ya, ny, x, xprev, xnext, first, last, o, e);
  if (FORCED) fxn = __ldg(fxt + ya);
#pragma unroll 1
  for (int r = 0; r < R; ++r) {
    f32x2 v[kQ][2];
    copy_async_wait();
#pragma unroll
    for (int l = 0; l < kQ; ++l) {  // stage 1: the pull's x-shift
      v[l][0] = o[l].x;
      v[l][1] = o[l].y;
      if (cx_of(l) > 0) {
        float prev = __shfl_up_sync(0xffffffffu, last_of(v[l]), 1);
        if (first) prev = e[l];
        shift_right(v[l], prev);
      } else if (cx_of(l) < 0) {
        float next = __shfl_down_sync(0xffffffffu, first_of(v[l]), 1);
        if (last) next = e[l];
        shift_left(v[l], next);
      }
    }
    if (FORCED) {
#pragma unroll
      for (int s = T - 1; s > 0; --s) fx[s] = fx[s - 1];
      fx[0] = fxn;
    }
    const int y1 = ya + 1 == ny ? 0 : ya + 1;
    // the next row's loads are in flight during this row's stages
    if (r + 1 < R) {
      multi_load(src, plane, pitch, y1, ny, x, xprev, xnext, first, last, o, e);
      if (FORCED) fxn = __ldg(fxt + y1);
    }
    bool done = false;
#pragma unroll
    for (int s = 0; s < T; ++s) {
      if (s > 0) {
        // pull from stage s - 1: its row y + 1 is in v, rows y and y - 1 in
        // the delay slots (already x-shifted when they were stored)
        float *ed = edges + (((r & 1) * (T - 1) + s - 1) * kMultiWarps) * 8;
        if (W.g > 1) {
          if (last) {
            ed[warp * 8 + 0] = last_of(v[1]);
            ed[warp * 8 + 1] = last_of(v[5]);
            ed[warp * 8 + 2] = last_of(v[8]);
          }
          if (first) {
            ed[warp * 8 + 3] = first_of(v[3]);
            ed[warp * 8 + 4] = first_of(v[6]);
            ed[warp * 8 + 5] = first_of(v[7]);
          }
          group_sync(base + 1, 32 * W.g);
        }
#pragma unroll
        for (int l = 0; l < kQ; ++l) {
          if (cx_of(l) > 0) {
            float prev = __shfl_sync(0xffffffffu, last_of(v[l]), lprev);
            if (W.g > 1 && first) prev = ed[wp * 8 + (l == 1 ? 0 : (l == 5 ? 1 : 2))];
            shift_right(v[l], prev);
          } else if (cx_of(l) < 0) {
            float next = __shfl_sync(0xffffffffu, first_of(v[l]), lnext);
            if (W.g > 1 && last) next = ed[wn * 8 + (l == 3 ? 3 : (l == 6 ? 4 : 5))];
            shift_left(v[l], next);
          }
        }
        ulonglong2 *dl = delay + (size_t)(s - 1) * kDelaySlots * kS + tid;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          const int l = k == 0 ? 0 : (k == 1 ? 1 : (k == 2 ? 3 : (k == 3 ? 2 : (k == 4 ? 5 : 6))));
          ulonglong2 *p = dl + (k < 3 ? k : 3 + 2 * (k - 3) + (r & 1)) * kS;
          const ulonglong2 old = *p;
          *p = make_ulonglong2(v[l][0], v[l][1]);
          v[l][0] = old.x;
          v[l][1] = old.y;
        }
        if (r < 2 * s) break;  // the block's first rows: not enough below them yet
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        f32x2 g[kQ];
#pragma unroll
        for (int l = 0; l < kQ; ++l) g[l] = v[l][c];
        if constexpr (ELBM) {
          // lanes past the row and the rim of a strip hold values that reach no
          // output (mixed from cells that are not neighbours): no iterations
          // for them.  23 members of 392 x 665, T = 3, no cell outside the
          // series: 651 us per step with them, single steps 97
          const int reach = T - 1 - s, xc = xu + 2 * c;
          const bool used = active && xc + 1 >= W.out0 - reach && xc < W.out1 + reach;
          if (!collide2_elbm<FORCED>(g, rho0, 2.0f * M.tau_f, both2(fx[s]), fy[c], alpha) && used) {
            float ga[kQ], gb[kQ], fya, fyb;  // a cell whose root needs iterations
#pragma unroll
            for (int l = 0; l < kQ; ++l) unpack2(g[l], ga[l], gb[l]);
            unpack2(fy[c], fya, fyb);
            collide_elbm_call(ga, rho0, M.tau_f, fx[s], fya, alpha);
            collide_elbm_call(gb, rho0, M.tau_f, fx[s], fyb, alpha);
#pragma unroll
            for (int l = 0; l < kQ; ++l) g[l] = pack2(ga[l], gb[l]);
          }
        } else {
          collide2_f32<FORCED>(g, rho0, om, both2(fx[s]), fy[c], alpha);
        }
#pragma unroll
        for (int l = 0; l < kQ; ++l) v[l][c] = g[l];
      }
      done = s == T - 1;
    }
    if (done && out) {
      int ys = ya - (T - 1);
      if (ys < 0) ys += ny;
      float *drow = dst + (size_t)ys * pitch + x;
#pragma unroll
      for (int l = 0; l < kQ; ++l) {
        float4 q;
        unpack2(v[l][0], q.x, q.y);
        unpack2(v[l][1], q.z, q.w);
        __stcs(reinterpret_cast<float4 *>(drow + (size_t)l * plane), q);
      }
    }
    ya = y1;
  }
}

template <int T, bool FORCED, bool ELBM>
cudaError_t launch(const Member *d_members, const MultiWarp *tab, int ctas, int state, int flip,
                   cudaStream_t s) {
  constexpr size_t smem = multi_smem<T>();
  const cudaError_t e = cudaFuncSetAttribute(
      k_multi<T, FORCED, ELBM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_multi<T, FORCED, ELBM><<<ctas, dim3(32, kMultiWarps), smem, s>>>(d_members, tab, ctas, state, flip);
  return cudaGetLastError();
}

}  // namespace

// How the columns of a member are split: whole rows as one group of g warps
// where that takes at most gmax warps and no more of a CTA than strips would
// (whole rows keep floor(8 / g) g of its 8 warps busy, a strip of one warp
// loses its halo lanes), else strips of `width` columns.
struct Split {
  int g, strips, width;
};
static Split split_columns(int nx, int gmax) {
  const int full = (nx + 127) / 128, ns = (nx + 119) / 120;
  if (full == 1 || (full <= gmax && kMultiWarps / (kMultiWarps / full) <= ns))
    return Split{full, 1, nx};
  return Split{1, ns, ((nx + ns - 1) / ns + 3) / 4 * 4};
}
static int block_rows(int ny, int rows) {
  rows = std::min(rows, ny);  // any larger asks for whole columns
  const int nb = (ny + rows - 1) / rows;
  return (ny + nb - 1) / nb;
}

double multi_ctas(int nx, int ny, int rows, int gmax) {
  const Split S = split_columns(nx, gmax);
  const int h = block_rows(ny, rows);
  return (double)((ny + h - 1) / h) * S.strips / (kMultiWarps / S.g);
}

void multi_member(int member, int nx, int ny, int rows, int gmax, std::vector<MultiWarp> *tab) {
  const Split S = split_columns(nx, gmax);
  const int h = block_rows(ny, rows);
  for (int y0 = 0; y0 < ny; y0 += h)
    for (int i = 0; i < S.strips; ++i) {
      const int o0 = i * S.width, o1 = o0 + S.width < nx ? o0 + S.width : nx;
      if (o0 >= nx) continue;
      const int used = (int)(tab->size() % kMultiWarps);
      if (used + S.g > kMultiWarps)  // a group does not straddle CTAs
        for (int k = used; k < kMultiWarps; ++k) tab->push_back(MultiWarp{-1});
      for (int w = 0; w < S.g; ++w) {
        MultiWarp W{};
        W.member = member;
        W.x0 = S.strips == 1 ? 128 * w : o0 - 4;
        W.xend = S.strips == 1 ? nx : o1 + 4;
        W.out0 = o0;
        W.out1 = o1;
        W.y0 = y0;
        W.rows = y0 + h < ny ? h : ny - y0;
        W.g = S.g;
        W.w = w;
        tab->push_back(W);
      }
    }
}

size_t multi_capacity(int nx, int ny) {
  // at most one warp per 60 columns and kMultiMinRows rows, and a CTA's padding
  return ((size_t)nx / 60 + 2) * ((size_t)ny / kMultiMinRows + 2) * 2 + kMultiWarps;
}

cudaError_t launch_multi(int T, bool forced, bool elbm, const Member *d_members, const MultiWarp *tab, int ctas,
                         int state, int flip, cudaStream_t s) {
  if (state > 1 || ctas < 1) return cudaErrorInvalidValue;
#define LBM_MULTI(T_)                                                                 \
  if (T == T_ && elbm)                                                                \
    return forced ? launch<T_, true, true>(d_members, tab, ctas, state, flip, s)      \
                  : launch<T_, false, true>(d_members, tab, ctas, state, flip, s);    \
  if (T == T_)                                                                        \
    return forced ? launch<T_, true, false>(d_members, tab, ctas, state, flip, s)     \
                  : launch<T_, false, false>(d_members, tab, ctas, state, flip, s)
  LBM_MULTI(2);
  LBM_MULTI(3);
  LBM_MULTI(4);
#undef LBM_MULTI
  return cudaErrorInvalidValue;
}

}  // namespace lbm
