// exchange.cuh -- device pieces of the momentum exchange (Eq. hlbm:mea,
// Sec. 3.2) of one particle from the populations alone, on the library's
// blocked storage.
#pragma once
#include "lbm_common.cuh"

namespace hlbm {

constexpr int XCH_MAX_T = 256;  // threads per block: 128 or 256

// The bounding box [floor(X - r_c), ceil(X + r_c)] of a particle (clipped at
// walls and to a slab's owned planes) and, per plane of the block, its rows
// that meet the circumscribed sphere (+-1 cell of margin), flattened: row r
// of plane j covers the flat cells [start[j][r], start[j][r + 1]) from
// unwrapped x = lo[0] + xa[j][r] on.
struct ExchangeBox {
  int lo[3], ext[3];
  float x0, rc2;
  float dy[MAX_PLANES], dz[MAX_PLANES];
  unsigned short start[MAX_PLANES][MAX_PLANES + 2];
  signed char xa[MAX_PLANES][MAX_PLANES];
};

// Fills the box for planes [q0, q0 + nq); called by all threads of the block
// (it synchronises).  The only FP64 arithmetic of the walk, and done once
// per block, a lane per axis, row or plane: an FP64 instruction holds a
// GB300 SM's narrow pipe for 16 cycles per warp however few lanes run.
__device__ __forceinline__ void exchange_box(const PartArgs& a, int p, const BoxDesc& bd, int q0, int nq,
                                             ExchangeBox& b) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* Xp = a.P + (long long)PF_X * a.cap + p;
  if (tid < 3) {
    const int n = tid == 0 ? bd.nx : (tid == 1 ? bd.ny : bd.nz);
    const double X = Xp[(long long)tid * a.cap], rc = a.P[(long long)PF_RC * a.cap + p];
    int l = 0, h = -1;
    if (X > -1.0e6 && X < 1.0e6) {  // no interior cells otherwise (the update flags it)
      l = (int)floor(X - rc);
      h = (int)ceil(X + rc);
      if ((bd.bc >> tid) & 1) {
        const bool cut = tid == 2 && (bd.bc & BC_CUT_Z);  // owned planes only
        l = max(l, cut ? bd.own_lo : 0);
        h = min(h, cut ? bd.own_hi - 1 : n - 1);
      }
    } else {
      atomicOr(a.status, ST_UNSTABLE);
    }
    b.lo[tid] = l;
    b.ext[tid] = min(max(h - l + 1, 0), MAX_PLANES);
    if (tid == 0) {
      b.x0 = (float)X;
      b.rc2 = (float)(rc * rc) * 1.0001f + 1e-3f;
    }
  }
  __syncthreads();
  {
    const int j = tid & (MAX_PLANES - 1);  // warps 0, 1: rows; 2, 3: planes
    if (tid < 2 * MAX_PLANES) {
      const int ax = tid < MAX_PLANES ? 1 : 2;
      const float d = (float)((double)(b.lo[ax] + j) - Xp[(long long)ax * a.cap]);
      (ax == 1 ? b.dy : b.dz)[j] = d;
    }
  }
  __syncthreads();
  for (int j = warp; j < nq; j += blockDim.x >> 5) {
    if (q0 + j >= b.ext[2]) break;
    int len[2], xa[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int iy = lane + 32 * u;
      const float dy = b.dy[iy], dz = b.dz[q0 + j];
      len[u] = xa[u] = 0;
      const float d2 = __fmaf_rn(dz, dz, __fmul_rn(dy, dy));
      if (iy < b.ext[1] && d2 < b.rc2) {
        const float s = sqrtf(b.rc2 - d2);
        const int x = max(b.lo[0], (int)floorf(b.x0 - s) - 1);
        const int xb = min(b.lo[0] + b.ext[0] - 1, (int)ceilf(b.x0 + s) + 1);
        len[u] = max(xb - x + 1, 0);
        xa[u] = min(max(x - b.lo[0], 0), MAX_PLANES - 1);
      }
    }
    int s0 = len[0], s1 = len[1];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t0 = __shfl_up_sync(0xffffffffu, s0, off);
      const int t1 = __shfl_up_sync(0xffffffffu, s1, off);
      if (lane >= off) { s0 += t0; s1 += t1; }
    }
    s1 += __shfl_sync(0xffffffffu, s0, 31);
    b.start[j][lane] = (unsigned short)(s0 - len[0]);
    b.start[j][lane + 32] = (unsigned short)(s1 - len[1]);
    b.xa[j][lane] = (signed char)xa[0];
    b.xa[j][lane + 32] = (signed char)xa[1];
    if (lane == 31) b.start[j][MAX_PLANES] = (unsigned short)s1;
  }
  __syncthreads();
}

// Sum over the links of an interior cell (used form of Eq. hlbm:mea):
//   sum_i (c_i - u_p) f_i(x) + (c_i + u_p) f_ibar(x - c_i)
// = sum_i c_i (in_i + out_i) - u_p sum_i (in_i - out_i), in_i = f_i(x), out_i
// = f_ibar(x - c_i).  This is the printed per-cell sum with the opposite
// sign: on post-streaming populations the printed sum is what the cell hands
// to the fluid, and the particle feels the reverse.  In both AA parities the
// pair of slots is {slot i of x, slot ibar of x - c_i}; only which of the two
// is the arrival differs.  A link to a node beyond a wall carries no fluid
// and is left out; on deviations d = f - w that leaves -2 c_i w_i per omitted
// link, because the weights of all 18 links sum to zero.  All 36 loads are
// independent of one another and of any branch.
template <typename S, int PAR, bool W>
__device__ __forceinline__ void exchange_links(const S* f, const BoxDesc& bd, int x, int y, int z, float scale,
                                               float inv_s, float (&F)[3], float& mgain) {
  const RowBlocks rb = row_blocks<W>(bd, x, y, 1);
  int zb[3];
  slice_blocks<W>(bd, z, zb);
  const S* own = cell_ptr(f, zb[1] + rb.yb[1] + rb.xb, rb.xin);
  float va[Q], vb[Q];
  unsigned walls = 0;  // bit i: x - c_i lies beyond a wall
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int by = rb.yb[1 - cy(i)], bz = zb[1 - cz(i)];
    const bool wall = W && (by < 0 || bz < 0 || (cx(i) > 0 && rb.wl) || (cx(i) < 0 && rb.wr));
    const int dx = cx(i) > 0 ? rb.dl : (cx(i) < 0 ? rb.dr : 0);
    const S* nb = wall ? own : cell_ptr(f, bz + by + rb.xb, rb.xin) + dx;
    if (wall) walls |= 1u << i;
    va[i] = Pop<S>::ld_raw(own + i * VB);
    vb[i] = Pop<S>::ld_raw(nb + opp(i) * VB);
  }
  // in stored units; the scale is a power of two
  F[0] = F[1] = F[2] = 0.0f;
  mgain = 0.0f;
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const float in = PAR == 0 ? va[i] : vb[i], out = PAR == 0 ? vb[i] : va[i];
    float sum = in + out, dif = in - out;
    if (W && ((walls >> i) & 1u)) {
      sum = Pop<S>::SCALED ? -2.0f * (float)wq(i) * scale : -2.0f * (float)wq(i);
      dif = 0.0f;
    }
    if (cx(i)) F[0] += (float)cx(i) * sum;
    if (cy(i)) F[1] += (float)cy(i) * sum;
    if (cz(i)) F[2] += (float)cz(i) * sum;
    mgain += dif;
  }
  if (Pop<S>::SCALED) {
#pragma unroll
    for (int j = 0; j < 3; ++j) F[j] = __fmul_rn(F[j], inv_s);
    mgain = __fmul_rn(mgain, inv_s);
  }
}

// One warp's share of one group of planes [j0, j1) of the block's box: flat
// cells 32 vw + lane, + 128, ... of each plane, as if four warps (vw = 0 .. 3)
// walked the group together; per-thread sums (F, T) in FP32 over the cells
// and then the planes, added over the warp by shuffles.  The split and the
// order are part of the result (a force to the last bit): warps may take the
// shares in any order.
template <typename S, int PAR, bool WALLS, bool GRIDS>
__device__ __forceinline__ void exchange_share(const PartArgs& a, const Rec& R, const BoxDesc& bd,
                                               const ExchangeBox& b, int q0, int j0, int j1, int vw, float (&v)[6]) {
  const S* f = reinterpret_cast<const S*>(a.f);
  const int lane = threadIdx.x & 31;
  const GridSet gs = GRIDS ? a.grids : GridSet{};
  bool any = false;
#pragma unroll
  for (int k = 0; k < 6; ++k) v[k] = 0.0f;
  for (int j = j0; j < j1; ++j) {
    const int zu = b.lo[2] + q0 + j;
    const int z = zu < 0 ? zu + bd.nz : (zu >= bd.nz ? zu - bd.nz : zu);
    const int total = b.start[j][MAX_PLANES];
    float s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int q = 32 * vw + lane; q < total; q += 128) {
      int r = 0;  // the row holding flat index q: the last one starting at or before it
#pragma unroll
      for (int step = 32; step > 0; step >>= 1)
        if (b.start[j][r + step] <= q) r += step;
      const int xu = b.lo[0] + b.xa[j][r] + (q - b.start[j][r]);
      const int yu = b.lo[1] + r;
      const int x = xu < 0 ? xu + bd.nx : (xu >= bd.nx ? xu - bd.nx : xu);
      const int y = yu < 0 ? yu + bd.ny : (yu >= bd.ny ? yu - bd.ny : yu);
      float rr[3];
      const bool in = (unsigned)x < (unsigned)bd.nx && (unsigned)y < (unsigned)bd.ny &&
                      (unsigned)z < (unsigned)bd.nz && inside_fp32(R, bd, x, y, z, rr, gs);
      auto cell = [&](auto wtag) {
        float Fc[3], mg;
        exchange_links<S, PAR, decltype(wtag)::value>(f, bd, x, y, z, a.scale, a.inv_scale, Fc, mg);
        const float upx = R.u[0] + (R.w[1] * rr[2] - R.w[2] * rr[1]);
        const float upy = R.u[1] + (R.w[2] * rr[0] - R.w[0] * rr[2]);
        const float upz = R.u[2] + (R.w[0] * rr[1] - R.w[1] * rr[0]);
        Fc[0] -= upx * mg;
        Fc[1] -= upy * mg;
        Fc[2] -= upz * mg;
        s[0] += Fc[0];
        s[1] += Fc[1];
        s[2] += Fc[2];
        s[3] += rr[1] * Fc[2] - rr[2] * Fc[1];
        s[4] += rr[2] * Fc[0] - rr[0] * Fc[2];
        s[5] += rr[0] * Fc[1] - rr[1] * Fc[0];
      };
      if (WALLS) {
        // only cells next to a wall take the wall selects
        const bool edge = ((bd.bc & 1) && (x == 0 || x == bd.nx - 1)) || ((bd.bc & 2) && (y == 0 || y == bd.ny - 1)) ||
                          ((bd.bc & 4) && (z == 0 || z == bd.nz - 1));
        if (in && edge) cell(std::integral_constant<bool, WALLS>{});
        if (in && !edge) cell(std::integral_constant<bool, false>{});
      } else if (in) {
        cell(std::integral_constant<bool, false>{});
      }
      any = any || in;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] += s[k];
  }
  if (__any_sync(0xffffffffu, any)) {
#pragma unroll
    for (int k = 0; k < 6; ++k)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
}

// ------------------------------------------------- the moments form
// Per interior cell x the used-sign sum is the momentum the cell gained by
// the last streaming, minus u_p times the mass it gained:
//   F(x) = (j - j*) - u_p(x) (rho - rho*)  [links into a wall: - 2 c_i f_i(x)]
// j, rho the moments of the arrivals f_i(x), j*, rho* those of the cell's own
// post-collision values f*_i(x), which the populations still hold (as the
// departures).  Each cell's terms are rounded to fixed point (ACC_FRAC_BITS)
// and added as integers: the sums depend on no order, so the cells may be
// spread over threads, warps and blocks in any way.

// FP32 radius about the centre that holds the particle (rounded up; grid
// particles carry theirs in a[0])
__device__ __forceinline__ float exchange_reach(const Rec& R) {
  float rc;
  if (R.shape == 0 || R.shape == 4) rc = R.a[0];
  else if (R.shape == 1) rc = fmaxf(R.a[0], fmaxf(R.a[1], R.a[2]));
  else if (R.shape == 3) rc = R.a[0] + R.a[2];
  else rc = sqrtf(R.a[0] * R.a[0] + R.a[1] * R.a[1] + R.a[2] * R.a[2]);
  return rc * 1.00001f + 0.01f;
}

// cells [lo, lo + ext) of one axis whose centre can lie within rc of the
// particle's centre, unwrapped; clipped at walls
__device__ __forceinline__ void exchange_extent(float xh, float rc, bool wall, int w_lo, int w_hi, int& lo, int& ext) {
  const float m = rc + fabsf(xh) * 2.4e-7f;  // the centre's rounding in FP32
  int l = (int)ceilf(xh - m), h = (int)floorf(xh + m);
  if (wall) {
    l = max(l, w_lo);
    h = min(h, w_hi);
  }
  lo = l;
  ext = min(max(h - l + 1, 0), MAX_PLANES);
}

// Offsets [t0, t1] along x from the centre that can lie inside the particle,
// on the x-parallel line at offset (ry, rz): the chord of the circumscribed
// sphere, for elongated shapes cut to their enclosing capsule (to the
// infinite cylinder about its axis and to its ends).  False: none.
__device__ __forceinline__ bool exchange_chord(const Rec& R, const Capsule& cap, float rc, float ry, float rz,
                                               float& t0, float& t1) {
  const float d2 = ry * ry + rz * rz;
  const float h2 = rc * rc - d2;
  if (!(h2 >= 0.0f)) return false;
  const float s = sqrtf(h2);
  t0 = -s;
  t1 = s;
  if (R.shape == 0) return true;
  if (capsule_row_dist2(cap, ry, rz) >= cap.r2) return false;
  const float w = ry * cap.u[1] + rz * cap.u[2];
  const float A = 1.0f - cap.u[0] * cap.u[0];
  if (A > 1e-2f) {
    // |(x, ry, rz)|^2 - ((x, ry, rz) . u)^2 < r^2
    const float b = cap.u[0] * w;
    const float disc = b * b - A * (d2 - w * w - cap.r2);
    if (!(disc >= 0.0f)) return false;
    const float q = sqrtf(disc);
    t0 = fmaxf(t0, (b - q) / A);
    t1 = fminf(t1, (b + q) / A);
  }
  if (fabsf(cap.u[0]) > 1e-2f) {
    const float e = cap.h + sqrtf(cap.r2), iu = 1.0f / fabsf(cap.u[0]);
    const float c = cap.u[0] > 0.0f ? -w : w;
    t0 = fmaxf(t0, (c - e) * iu);
    t1 = fminf(t1, (c + e) * iu);
  }
  return t1 >= t0;
}

// Rows of the bounding box that can hold interior cells, flattened: row r
// covers the cells [start[r], start[r + 1]) of the flat index; xa is the
// unwrapped x of its first cell, y and z are wrapped.
struct ExchangeRows {
  int start[XCH_MAX_T];
  int xa[XCH_MAX_T], y[XCH_MAX_T], z[XCH_MAX_T];
  int wtot[XCH_MAX_T / 32];
  unsigned found[XCH_MAX_T / 32][64];  // grid particles: a warp's interior cells, row << 8 | x - xa[row]
};
static_assert(MAX_PLANES <= 256 && XCH_MAX_T <= 1 << 24, "packing of ExchangeRows::found");

// Calls cell(x, y, z, rr) for every interior cell of the planes of the
// particle's bounding box from q0 on, and of the rows of each, that a block
// takes (part is .z of its entry of PartArgs::chunks; rr the cell's offset from
// the centre), spread over the block's threads (blockDim.x a power of two; all
// of them call, it synchronises).  One thread finds the x-range of one row; the
// rows' cells are then flattened, so that lanes stay busy whatever the shape.
template <bool GRIDS, typename Cell>
__device__ __forceinline__ void for_interior(const Rec& R, const BoxDesc& bd, int q0, int part, GridSet grids,
                                             ExchangeRows& sh, Cell cell) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const GridSet gs = GRIDS ? grids : GridSet{};
  const float rc = exchange_reach(R);
  const bool cutz = bd.bc & BC_CUT_Z;  // a slab: owned planes only
  int lox, extx, loy, exty, loz, extz;
  exchange_extent(R.xh[0], rc, bd.bc & 1, 0, bd.nx - 1, lox, extx);
  exchange_extent(R.xh[1], rc, bd.bc & 2, 0, bd.ny - 1, loy, exty);
  exchange_extent(R.xh[2], rc, bd.bc & 4, cutz ? bd.own_lo : 0, cutz ? bd.own_hi - 1 : bd.nz - 1, loz, extz);
  loy += (part >> 8) & 0xff;
  exty = max(min(exty - ((part >> 8) & 0xff), part >> 16), 0);
  const int planes = min(part & 0xff, extz - q0);
  const int rows = planes > 0 ? planes * exty : 0;
  Capsule cap = capsule_of(R, 0.0f);
  if (GRIDS && R.shape == 4 && gs.desc) {  // the interior only
    cap.h = gs.desc[__float_as_int(R.in2)].out_h;
    cap.r2 = gs.desc[__float_as_int(R.in2)].out_r2;
  }
  for (int row0 = 0; row0 < rows; row0 += nt) {
    const int row = row0 + tid;
    int len = 0, xa = 0, y = 0, z = 0;
    if (row < rows) {
      const int iz = row / exty;
      y = loy + (row - iz * exty);
      z = loz + q0 + iz;
      const float ry = ((float)y - R.xh[1]) - R.xl[1], rz = ((float)z - R.xh[2]) - R.xl[2];
      float t0, t1;
      if (exchange_chord(R, cap, rc, ry, rz, t0, t1)) {
        const float m = 0.02f + fabsf(R.xh[0]) * 2.4e-7f;
        xa = max((int)ceilf(R.xh[0] + t0 - m), lox);
        const int xb = min((int)floorf(R.xh[0] + t1 + m), lox + extx - 1);
        len = max(xb - xa + 1, 0);
      }
      y = y < 0 ? y + bd.ny : (y >= bd.ny ? y - bd.ny : y);
      z = z < 0 ? z + bd.nz : (z >= bd.nz ? z - bd.nz : z);
      if ((unsigned)y >= (unsigned)bd.ny || (unsigned)z >= (unsigned)bd.nz) len = 0;
    }
    int sum = len;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, sum, off);
      if (lane >= off) sum += t;
    }
    if (lane == 31) sh.wtot[warp] = sum;
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < (nt >> 5); ++w) {
      const int t = sh.wtot[w];
      if (w < warp) before += t;
      total += t;
    }
    sh.start[tid] = before + sum - len;
    sh.xa[tid] = xa;
    sh.y[tid] = y;
    sh.z[tid] = z;
    __syncthreads();
    if (GRIDS && R.shape == 4) {
      // Half the candidate cells or more lie outside: the warp collects the
      // inside ones and takes 32 at a time (the sums depend on no order).
      // 1300 rounded boxes in 224^3: exchange 117 -> 104 us FP32, 108 -> 89
      // FP16, with the candidates from the interior's capsule.
      // Ellipsoids, cuboids and capsules fill their chords better and lose by
      // it (2000 of them: 113 -> 117 us FP32, 91 -> 95 FP16).
      int held = 0;  // of found[warp], the same in every lane
      auto take = [&](int n) {
        __syncwarp();
        if (lane < n) {
          const unsigned e = sh.found[warp][lane];
          const int r = (int)(e >> 8), xu = sh.xa[r] + (int)(e & 255u);
          const int x = xu < 0 ? xu + bd.nx : (xu >= bd.nx ? xu - bd.nx : xu);
          const float rr[3] = {offset_fp32(x, bd.nx, bd.bc & 1, R.xh[0], R.xl[0]),
                               offset_fp32(sh.y[r], bd.ny, bd.bc & 2, R.xh[1], R.xl[1]),
                               offset_fp32(sh.z[r], bd.nz, bd.bc & 4, R.xh[2], R.xl[2])};
          cell(x, sh.y[r], sh.z[r], rr);
        }
        __syncwarp();
      };
      for (int q0w = 32 * warp; q0w < total; q0w += nt) {
        const int q = q0w + lane;
        bool in = false;
        unsigned e = 0;
        if (q < total) {
          int r = 0;
          for (int step = nt >> 1; step > 0; step >>= 1)
            if (sh.start[r + step] <= q) r += step;
          e = ((unsigned)r << 8) | (unsigned)(q - sh.start[r]);
          const int xu = sh.xa[r] + (q - sh.start[r]);
          const int x = xu < 0 ? xu + bd.nx : (xu >= bd.nx ? xu - bd.nx : xu);
          float rr[3];
          in = (unsigned)x < (unsigned)bd.nx && inside_fp32(R, bd, x, sh.y[r], sh.z[r], rr, gs);
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) sh.found[warp][held + __popc(m & ((1u << lane) - 1u))] = e;
        held += __popc(m);
        if (held >= 32) {
          take(32);
          const unsigned rest = lane + 32 < held ? sh.found[warp][lane + 32] : 0u;
          held -= 32;
          if (lane < held) sh.found[warp][lane] = rest;
          __syncwarp();
        }
      }
      if (held) take(held);
      __syncthreads();
      continue;
    }
    for (int q = tid; q < total; q += nt) {
      int r = 0;  // the row holding flat index q: the last one starting at or before it
      for (int step = nt >> 1; step > 0; step >>= 1)
        if (sh.start[r + step] <= q) r += step;
      const int xu = sh.xa[r] + (q - sh.start[r]);
      const int x = xu < 0 ? xu + bd.nx : (xu >= bd.nx ? xu - bd.nx : xu);
      float rr[3];
      if ((unsigned)x < (unsigned)bd.nx && inside_fp32(R, bd, x, sh.y[r], sh.z[r], rr, gs)) cell(x, sh.y[r], sh.z[r], rr);
    }
    __syncthreads();  // the rows are rewritten by the next chunk
  }
}

// force and torque terms of one interior cell; PAIRS: the departures summed
// by opposite pairs, as the two-cell collision does, otherwise one by one, as
// the one-cell collision (the sums agree to rounding)
template <typename S, int PAR, bool W>
__device__ __forceinline__ void exchange_moments(const S* f, const Rec& R, const BoxDesc& bd, int x, int y, int z,
                                                 const float (&r)[3], float inv_s, bool pairs, float (&F)[3],
                                                 float (&T)[3]) {
  const RowBlocks rb = row_blocks<W>(bd, x, y, 1);
  int zb[3];
  slice_blocks<W>(bd, z, zb);
  const S* own = cell_ptr(f, zb[1] + rb.yb[1] + rb.xb, rb.xin);
  float va[Q], vb[Q];  // slot i of x; slot ibar of x - c_i (slot i of x when that lies beyond a wall)
  unsigned walls = 0;  // bit i: x - c_i lies beyond a wall
  va[0] = vb[0] = Pop<S>::ld_raw(own);
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int by = rb.yb[1 - cy(i)], bz = zb[1 - cz(i)];
    const bool wall = W && (by < 0 || bz < 0 || (cx(i) > 0 && rb.wl) || (cx(i) < 0 && rb.wr));
    const int dx = cx(i) > 0 ? rb.dl : (cx(i) < 0 ? rb.dr : 0);
    const S* nb = wall ? own + i * VB : cell_ptr(f, bz + by + rb.xb, rb.xin) + (dx + opp(i) * VB);
    if (wall) walls |= 1u << i;
    va[i] = Pop<S>::ld_raw(own + i * VB);
    vb[i] = Pop<S>::ld_raw(nb);
  }
  // arrivals f_i(x) are slot i of x (even parity) or slot ibar of x - c_i
  // (odd parity); the departure f*_i(x) is the other kind for ibar.  Sums in
  // stored units (the scale is a power of two).
  float ms = 0.f, px = 0.f, py = 0.f, pz = 0.f;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const float d = PAR == 0 ? va[i] : vb[i];
    ms += d;
    if (cx(i)) px += (float)cx(i) * d;
    if (cy(i)) py += (float)cy(i) * d;
    if (cz(i)) pz += (float)cz(i) * d;
  }
  float m0, jx, jy, jz;
  auto dep = [&](int i) { return PAR == 0 ? vb[opp(i)] : va[opp(i)]; };
  if (pairs) {
    float m[Q];
    m0 = dep(0);
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      m0 = m0 + (dep(i) + dep(i + 1));
      m[i] = dep(i) - dep(i + 1);
    }
    jx = ((m[1] + m[7]) + (m[9] + m[11])) + m[13];
    jy = (((m[3] + m[7]) - m[9]) + m[15]) + m[17];
    jz = (((m[5] + m[11]) - m[13]) + m[15]) - m[17];
  } else {
    m0 = jx = jy = jz = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      m0 += dep(i);
      if (cx(i)) jx += (float)cx(i) * dep(i);
      if (cy(i)) jy += (float)cy(i) * dep(i);
      if (cz(i)) jz += (float)cz(i) * dep(i);
    }
  }
  const float dm = Pop<S>::SCALED ? __fmul_rn(ms - m0, inv_s) : ms - m0;
  const float dx = Pop<S>::SCALED ? __fmul_rn(px - jx, inv_s) : px - jx;
  const float dy = Pop<S>::SCALED ? __fmul_rn(py - jy, inv_s) : py - jy;
  const float dz = Pop<S>::SCALED ? __fmul_rn(pz - jz, inv_s) : pz - jz;
  const float upx = R.u[0] + (R.w[1] * r[2] - R.w[2] * r[1]);
  const float upy = R.u[1] + (R.w[2] * r[0] - R.w[0] * r[2]);
  const float upz = R.u[2] + (R.w[0] * r[1] - R.w[1] * r[0]);
  F[0] = dx - upx * dm;
  F[1] = dy - upy * dm;
  F[2] = dz - upz * dm;
  if (W) {
#pragma unroll
    for (int i = 1; i < Q; ++i)
      if ((walls >> i) & 1u) {
        const float d = PAR == 0 ? va[i] : vb[i];
        const float v = 2.0f * ((float)wq(i) + (Pop<S>::SCALED ? __fmul_rn(d, inv_s) : d));
        if (cx(i)) F[0] -= (float)cx(i) * v;
        if (cy(i)) F[1] -= (float)cy(i) * v;
        if (cz(i)) F[2] -= (float)cz(i) * v;
      }
  }
  T[0] = r[1] * F[2] - r[2] * F[1];
  T[1] = r[2] * F[0] - r[0] * F[2];
  T[2] = r[0] * F[1] - r[1] * F[0];
}

// Exact warp sum of 64-bit values, from three limbs with single-instruction
// warp reductions: v = a 2^42 + b 2^21 + c with c, b in [0, 2^21) and
// a = v >> 42 in [-2^21, 2^21), so 32 lanes' limb sums stay within 32 bits.
__device__ __forceinline__ long long warp_sum_i64(long long v) {
  const unsigned c = (unsigned)v & 0x1fffffu;
  const unsigned b = (unsigned)(v >> 21) & 0x1fffffu;
  const int hi = (int)(v >> 42);
  const unsigned sc = __reduce_add_sync(0xffffffffu, c);
  const unsigned sb = __reduce_add_sync(0xffffffffu, b);
  const int sa = __reduce_add_sync(0xffffffffu, hi);
  return (long long)(((unsigned long long)(long long)sa << 42) + ((unsigned long long)sb << 21) + sc);
}

}  // namespace hlbm
