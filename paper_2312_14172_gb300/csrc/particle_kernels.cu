// particle_kernels.cu -- fluid -> particle coupling and particle motion.
//
//   mea_kernel, mea_moments_kernel
//                   momentum exchange (Eq. hlbm:mea) summed over the cells
//                   whose centre lies inside each particle (Eqs.
//                   hydrodynamicforce, hydrodynamictorque); one or more
//                   thread blocks per particle, each on a run of z-planes
//                   of its bounding box; per-cell sums and warp shuffles in
//                   FP32, block sums in FP64, in a fixed order; or, in the
//                   moments form, per-cell terms added as integers (both
//                   deterministic).
//   update_kernel   weight minus buoyancy (Sec. 5.1), Newton-Euler update
//                   (Eqs. particlemotiontrans, motionrot) in FP64, the FP32
//                   coupling record of the new state, and the per-tile particle
//                   lists (the single-GPU form of the paper's particle
//                   assignment, Sec. 4.2.3) that the collision kernel reads.
//   records_kernel  coupling records only (after particles are added or set).
#include <type_traits>

#include "exchange.cuh"
#include "mea_common.cuh"

namespace hlbm {

__device__ __forceinline__ double pget(const double* P, int cap, int field, int p) {
  return P[(long long)field * cap + p];
}
__device__ __forceinline__ void pset(double* P, int cap, int field, int p, double v) {
  P[(long long)field * cap + p] = v;
}

// FP32 coupling record of a particle state (X, U, W, q; semi-axes A, their
// FP32 inverses iA, radius r_inf beyond which B = 0; interface width eps)
__device__ __forceinline__ void make_record(const double X[3], const double U[3], const double W[3],
                                            const double q[4], const double A[3], const double iA[3],
                                            double rinf, float eps, int p, int shape, int box, Rec& R) {
  double Rm[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};  // a sphere needs no orientation
  if (shape != 0) rotation_rn(q, Rm);
  for (int j = 0; j < 3; ++j) {
    const float xh = __double2float_rn(X[j]);
    R.xh[j] = xh;
    R.xl[j] = __double2float_rn(X[j] - (double)xh);
    R.u[j] = (float)U[j];
    R.w[j] = (float)W[j];
    R.a[j] = __double2float_rn(A[j]);
    R.ia[j] = (float)iA[j];
  }
  for (int k = 0; k < 9; ++k) R.M[k] = __double2float_rn(Rm[k]);
  R.in2 = __double2float_rn(A[0] * A[0]);
  if (shape == 4) R.in2 = __int_as_float((int)iA[0]);  // a grid particle: its grid id
  if (shape == 0) {
    // a sphere needs no rotation: its slots hold the FP32 bounds of the
    // collision's per-cell tests (the same roundings as computed there)
    const float a_in = __fsub_rn(R.a[0], __fmul_rn(0.5f, eps));
    const float a_out = __fadd_rn(R.a[0], __fmul_rn(0.5f, eps));
    R.M[SPH_R2_IN] = a_in > 0.0f ? __fmul_rn(a_in, a_in) : -1.0f;
    R.M[SPH_R2_OUT] = __fmul_rn(a_out, a_out);
  }
  // B vanishes beyond r_inf; a slightly larger FP32 bound keeps the test safe
  const double rb = rinf + 0.01;
  R.rinf2 = (float)(rb * rb);
  R.shape = shape;
  R.box = box;
  R.pid = p;
}

__device__ void build_record(const double* P, int cap, int p, int shape, int box, float eps, Rec& R) {
  double X[3], U[3], W[3], q[4], A[3], iA[3];
  for (int j = 0; j < 3; ++j) {
    X[j] = pget(P, cap, PF_X + j, p);
    U[j] = pget(P, cap, PF_U + j, p);
    W[j] = pget(P, cap, PF_W + j, p);
    A[j] = pget(P, cap, PF_A + j, p);
    iA[j] = pget(P, cap, PF_IA + j, p);
  }
  for (int j = 0; j < 4; ++j) q[j] = pget(P, cap, PF_Q + j, p);
  make_record(X, U, W, q, A, iA, pget(P, cap, PF_RINF, p), eps, p, shape, box, R);
}

// the bin tiles along one axis touched by cells [lo, hi]: one range
// [a0, a1], plus a second range [b0, b1] (empty when b1 < b0) where the cell
// range wraps around a periodic axis
struct AxisTiles {
  int a0, a1, b0, b1;
  __device__ __forceinline__ int count() const { return (a1 - a0 + 1) + max(b1 - b0 + 1, 0); }
  __device__ __forceinline__ int at(int t) const {
    const int na = a1 - a0 + 1;
    return t < na ? a0 + t : b0 + (t - na);
  }
};

__device__ AxisTiles axis_tiles(int lo, int hi, int n, int T, bool wall) {
  AxisTiles r{0, -1, 0, -1};
  if (wall) {
    lo = max(lo, 0);
    hi = min(hi, n - 1);
    if (lo <= hi) { r.a0 = lo / T; r.a1 = hi / T; }
    return r;
  }
  if (hi - lo + 1 >= n) {  // the whole periodic axis
    r.a0 = 0; r.a1 = (n - 1) / T;
    return r;
  }
  if (lo < 0) {            // [lo + n, n - 1] and [0, hi]
    r.a0 = (lo + n) / T; r.a1 = (n - 1) / T;
    r.b0 = 0; r.b1 = hi / T;
  } else if (hi >= n) {    // [lo, n - 1] and [0, hi - n]
    r.a0 = lo / T; r.a1 = (n - 1) / T;
    r.b0 = 0; r.b1 = (hi - n) / T;
  } else {
    r.a0 = lo / T; r.a1 = hi / T;
  }
  // both ends in the same tiles (an axis of one or two tiles): merge
  if (r.b1 >= r.b0 && r.b1 >= r.a0) {
    r.a0 = 0; r.a1 = max(r.a1, r.b1);
    r.b0 = 0; r.b1 = -1;
  }
  return r;
}

// Tiles of one particle's bin range, kept in shared memory between the
// Newton-Euler step and the binning.
struct BinRange {
  AxisTiles at[3];
  long long tile_off;
  int ntx, nty;
  int count;  // tiles; 0 when the particle is not binned
};

// cells [lo, hi] along one axis of the bin range of a particle at X: its
// influence sphere, widened so that the cells next to the interior (which
// feed its momentum exchange) see it too, rounded outwards in FP32
__device__ __forceinline__ AxisTiles bin_axis(double X, float rb, int n, int T, bool wall) {
  const int lo = (int)floorf(__fsub_rd(__double2float_rd(X), rb)) - 1;
  const int hi = (int)ceilf(__fadd_ru(__double2float_ru(X), rb)) + 1;
  return axis_tiles(lo, hi, n, T, wall);
}

// adds particle p to the lists of the tiles of its bin range: threads sub,
// sub + step, ... take the tiles in turn
__device__ __forceinline__ void bin_particle(const PartArgs& a, const BinRange& br, int p, int sub, int step) {
  const int cx_ = br.at[0].count(), cy_ = br.at[1].count();
  for (int t = sub; t < br.count; t += step) {
    const int ix = t % cx_, r = t / cx_, iy = r % cy_, iz = r / cy_;
    const long long tile = br.tile_off + ((long long)br.at[2].at(iz) * br.nty + br.at[1].at(iy)) * br.ntx +
                           br.at[0].at(ix);
    const int slot = atomicAdd(&a.bin_count[tile], 1);
    if (slot < a.bin_cap) a.bin_ids[tile * a.bin_cap + slot] = p;
    else atomicOr(a.status, ST_CAPACITY);
  }
}

// clears the tile counts the next step will fill
__device__ __forceinline__ void clear_bins(const PartArgs& a) {
  const long long nthr = (long long)gridDim.x * blockDim.x;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < a.ntiles; t += nthr) a.bin_count_clear[t] = 0;
}

// ------------------------------------------- one particle moved by one block
// The Newton-Euler step of the update kernel (below) for the particle whose
// momentum exchange this block has just summed, with the vector components
// and the quaternion's on lanes of their own: an FP64 instruction costs a
// GB300 SM 16 cycles per warp whether one lane runs it or 32, so a particle
// takes a third of the instructions that it takes on one lane.  Translation
// on warp 0, rotation on warp 1.  Every operation is the one of the update
// kernel, in its order (contractions written out), so that both move a
// particle to the same bits.
struct MoveScratch {
  double P[PF_COUNT];  // the particle's row of the table before the step
  double F[6];         // force and torque of the momentum exchange
  double v[7];         // w x y z and the angular velocity of the quaternion step
  double R[9], wb[3], Lb[3];
  BinRange br;
};

__device__ __forceinline__ double sum2(double a, double b, double c, double d) {  // a b + c d
  return __fma_rn(a, b, __dmul_rn(c, d));
}
__device__ __forceinline__ double dif2(double a, double b, double c, double d) {  // a b - c d
  return __fma_rn(a, b, -__dmul_rn(c, d));
}

// entry e of the rotation matrix of the quaternion v[0..3] (as rotation_rn):
// v[a] v[b] +- v[c] v[d], doubled, on the diagonal taken from 1
__device__ __forceinline__ double rotation_entry(const double* v, int e) {
  // w x y z = 0 1 2 3; per entry a, b, c, d as digits of base 4
  const unsigned tab[9] = {0xAF, 0x63, 0x72, 0x63, 0x5F, 0xB1, 0x72, 0xB1, 0x5A};
  const unsigned t = tab[e];
  const double p = __dmul_rn(v[(t >> 6) & 3], v[(t >> 4) & 3]), q = __dmul_rn(v[(t >> 2) & 3], v[t & 3]);
  const bool minus = e == 1 || e == 5 || e == 6;
  const double s = __dmul_rn(2.0, minus ? __dsub_rn(p, q) : __dadd_rn(p, q));
  return e % 4 == 0 ? __dsub_rn(1.0, s) : s;
}

// called by all threads of the block; m.P, m.F are filled (and synchronised);
// R holds the particle's record before the step
__device__ __forceinline__ void move_particle(const PartArgs& a, int p, const BoxDesc& bd, Rec& R, MoveScratch& m) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cap = a.cap;
  if (warp == 0) {
    if (lane < 3) {
      const int j = lane;
      double Fh = m.F[j];
      if (a.contact_k > 0.0) Fh += m.P[PF_FC + j];
      const double F = __fma_rn(__dmul_rn(__dsub_rn(m.P[PF_RHO], 1.0), m.P[PF_V]), a.g[j], Fh);
      const double U = __fma_rn(F, m.P[PF_IM], m.P[PF_U + j]);
      double X = __dadd_rn(m.P[PF_X + j], U);
      if (!(isfinite(X) && isfinite(U))) atomicOr(a.status, ST_UNSTABLE);
      const int n = j == 0 ? bd.nx : (j == 1 ? bd.ny : bd.nz);
      const bool wall = (bd.bc >> j) & 1;
      if (wall) {
        const bool cut = j == 2 && (bd.bc & BC_CUT_Z);
        if (!cut && !(X > -0.5 && X < n - 0.5)) atomicOr(a.status, ST_LEFT_DOMAIN);
      } else {
        const double L = (double)n;
        if (X >= L) X -= L;
        else if (X < 0.0) X += L;
      }
      pset(a.P, cap, PF_X + j, p, X);
      pset(a.P, cap, PF_U + j, p, U);
      const float xh = __double2float_rn(X);
      R.xh[j] = xh;
      R.xl[j] = __double2float_rn(X - (double)xh);
      R.u[j] = (float)U;
      const bool binned = X > -1.0e6 && X < 1.0e6;  // flagged above otherwise
      const float rb = __double2float_ru(fmax(m.P[PF_RINF], __dadd_rn(m.P[PF_RC], 1.5)));
      m.br.at[j] = binned ? bin_axis(X, rb, n, j == 0 ? TILE_X : (j == 1 ? TILE_Y : TILE_Z), wall) : AxisTiles{0, -1, 0, -1};
    }
    __syncwarp();
    if (lane == 0) {
      m.br.tile_off = bd.tile_off;
      m.br.ntx = bd.ntx;
      m.br.nty = bd.nty;
      m.br.count = m.br.at[0].count() * m.br.at[1].count() * m.br.at[2].count();
    }
  } else if (warp == 1) {
    const bool sphere = R.shape == 0;
    const int j = lane < 3 ? lane : 0, j1 = j == 2 ? 0 : j + 1, j2 = j == 0 ? 2 : j - 1;
    if (lane < 4) m.v[lane] = m.P[PF_Q + lane];
    __syncwarp();
    double W = m.P[PF_W + j], Th = m.F[3 + j];
    if (a.contact_k > 0.0) Th += m.P[PF_TC + j];
    if (sphere) {
      W = __fma_rn(Th, m.P[PF_II + j], W);
      if (lane < 3) m.v[4 + lane] = W;
    } else {
      if (lane < 9) m.R[lane] = rotation_entry(m.v, lane);
      if (lane < 3) {
        m.wb[lane] = W;
        m.Lb[lane] = Th;
      }
      __syncwarp();
      // into the body frame
      double wb = __fma_rn(m.R[6 + j], m.wb[2], sum2(m.R[j], m.wb[0], m.R[3 + j], m.wb[1]));
      const double Tb = __fma_rn(m.R[6 + j], m.Lb[2], sum2(m.R[j], m.Lb[0], m.R[3 + j], m.Lb[1]));
      __syncwarp();
      if (lane < 3) {
        m.wb[lane] = wb;
        m.Lb[lane] = __dmul_rn(m.P[PF_I + j], wb);
      }
      __syncwarp();
      const double gy = dif2(m.wb[j1], m.Lb[j2], m.wb[j2], m.Lb[j1]);
      wb = __fma_rn(__dsub_rn(Tb, gy), m.P[PF_II + j], wb);
      if (lane < 3) m.v[4 + lane] = wb;
      __syncwarp();
      W = __fma_rn(m.R[3 * j + 2], m.v[6], sum2(m.R[3 * j], m.v[4], m.R[3 * j + 1], m.v[5]));
    }
    __syncwarp();
    // q += q (x) (0, omega_b) / 2, for a sphere in the equal form (0, omega)
    // (x) q / 2: per component s (v[a] v[b] + v[c] v[d] -+ v[e] v[f])
    double q = 0.0, nq;
    if (lane < 4) {
      const double* v = m.v;
      const int l = lane;
      double t;
      if (l == 0) {
        t = sphere ? -__fma_rn(v[6], v[3], sum2(v[4], v[1], v[5], v[2]))
                   : __fma_rn(-v[3], v[6], dif2(-v[1], v[4], v[2], v[5]));
      } else if (sphere) {
        // w W_l-1 + W_l y_l+1 - W_l+1 y_l, y = x y z
        const int b = l - 1, c = l % 3, d = (l + 1) % 3;
        t = __fma_rn(-v[4 + d], v[1 + c], sum2(v[0], v[4 + b], v[4 + c], v[1 + d]));
      } else {
        const int b = l - 1, c = l % 3, d = (l + 1) % 3;
        t = __fma_rn(-v[1 + d], v[4 + c], sum2(v[0], v[4 + b], v[1 + c], v[4 + d]));
      }
      q = __fma_rn(0.5, t, v[l]);
    }
    {
      const double q0 = __shfl_sync(0xffffffffu, q, 0), q1 = __shfl_sync(0xffffffffu, q, 1);
      const double q2 = __shfl_sync(0xffffffffu, q, 2), q3 = __shfl_sync(0xffffffffu, q, 3);
      nq = __fma_rn(q3, q3, __fma_rn(q2, q2, sum2(q0, q0, q1, q1)));
    }
    q = __dmul_rn(q, rsqrt(nq));
    __syncwarp();
    if (lane < 4) {
      m.v[lane] = q;
      pset(a.P, cap, PF_Q + lane, p, q);
    }
    if (lane < 3) {
      if (!isfinite(W)) atomicOr(a.status, ST_UNSTABLE);
      pset(a.P, cap, PF_W + lane, p, W);
      R.w[lane] = (float)W;
    }
    __syncwarp();
    if (!sphere && lane < 9) R.M[lane] = __double2float_rn(rotation_entry(m.v, lane));
  } else if (warp == 2 && lane < 6) {
    pset(a.P, cap, (lane < 3 ? PF_F : PF_T - 3) + lane, p, m.F[lane]);
  }
  __syncthreads();
  if (threadIdx.x < 32)
    reinterpret_cast<int*>(&a.rec[p])[threadIdx.x] = reinterpret_cast<const int*>(&R)[threadIdx.x];
  bin_particle(a, m.br, p, threadIdx.x, blockDim.x);
}

// Momentum exchange of every particle from the populations alone: block
// `chunk` walks p_planes planes of the bounding box of particle
// chunk_p[chunk] from plane chunk_q[chunk] on, in groups of mea_group planes.
// A group's sum is that of four warps in FP64; a particle's force and torque
// are its groups' sums added in plane order, by the block that finishes last
// when it has several.  Bound by the latency and the L1 wavefronts of the 36
// scattered loads per cell, which 128 registers a thread keep all in flight.
// Before (FP64 bounding-box arithmetic in every thread, a wall branch
// between the loads, a block per plane): 200 spheres in 128^3 FP32 51 us, now
// 35; 2000 ellipsoids and cuboids in 256^3 355 -> 170; 50 000 spheres FP16
// 3312 -> 1470.
template <typename S, int PAR, bool WALLS, bool GRIDS>
__global__ void __launch_bounds__(XCH_MAX_T, 2) mea_kernel(PartArgs a) {
  // what no step changes is read before the wait for the kernel before
  const int4 chunk = a.chunks[blockIdx.x];
  const int p = chunk.x, q0 = chunk.y, planes = chunk.z, parts = chunk.w;
  const BoxDesc bd = a.boxes[a.box[p]];
  pdl_trigger();
  pdl_wait();
  __shared__ Rec R;
  __shared__ ExchangeBox box;
  __shared__ float wsum[MAX_PLANES][4][6];
  __shared__ double gsum[MAX_PLANES][6];
  __shared__ MoveScratch mv;
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 32) reinterpret_cast<int*>(&R)[tid] = reinterpret_cast<const int*>(&a.rec[p])[tid];
  if (a.move) {
    clear_bins(a);
    if (tid >= 64 && tid < 64 + PF_COUNT) mv.P[tid - 64] = pget(a.P, a.cap, tid - 64, p);
  }
  exchange_box(a, p, bd, q0, planes, box);
  const int G = a.mea_group;
  const int here = max(min(planes, box.ext[2] - q0), 0);  // planes that hold cells
  const int groups = (here + G - 1) / G;
  for (int item = warp; item < 4 * groups; item += blockDim.x >> 5) {
    const int g = item >> 2, vw = item & 3;
    float v[6];
    exchange_share<S, PAR, WALLS, GRIDS>(a, R, bd, box, q0, g * G, min((g + 1) * G, here), vw, v);
    if (lane == 0)
      for (int k = 0; k < 6; ++k) wsum[g][vw][k] = v[k];
  }
  __syncthreads();
  double* part = a.partial + ((long long)p * MAX_PLANES + q0 / G) * 6;
  // the groups past the box add nothing
  const int slots = min((planes + G - 1) / G, MAX_PLANES - q0 / G);
  for (int e = tid; e < 6 * slots; e += blockDim.x) {
    const int g = e / 6, k = e - 6 * g;
    double t = 0.0;
    if (g < groups)
      for (int w = 0; w < 4; ++w) t += (double)wsum[g][w][k];
    if (parts > 1) part[e] = t;
    else gsum[g][k] = t;
  }
  int total = slots;
  if (parts > 1) {
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(&a.done[p], 1) == parts - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    total = min(parts * ((planes + G - 1) / G), MAX_PLANES);
    for (int e = tid; e < 6 * total; e += blockDim.x)
      gsum[e / 6][e % 6] = __ldcg(a.partial + (long long)p * MAX_PLANES * 6 + e);
    if (tid == 0) a.done[p] = 0;
  }
  __syncthreads();
  if (tid < 6) {
    double t = 0.0;
    for (int g = 0; g < total; ++g) t += gsum[g][tid];
    if (a.move) mv.F[tid] = t;
    else pset(a.P, a.cap, (tid < 3 ? PF_F : PF_T - 3) + tid, p, t);
  }
  if (!a.move) return;
  __syncthreads();
  move_particle(a, p, bd, R, mv);
}

// Momentum exchange of every particle in the moments form: blocks of whole
// planes as above, sums in fixed point.  It took the place of a list of interior cells that the collision
// wrote (cell, particle and departing moments, 24 bytes a cell) and a kernel
// that walked it: the populations hold the departures too, the particle's
// geometry gives the cells, and the collision is rid of the appends (us,
// collision + exchange, before and now: 2000 ellipsoids and cuboids FP32
// 483 + 105, now 439 + 118; 64 boxes FP32 979 + 243, now 896 + 230; 50 000
// spheres FP16 4695 + 905, now 4547 + 958; 200 spheres 128^3 FP16 51.6 + 17.8,
// now 44.9 + 21.7).
template <typename S, int PAR, bool WALLS, bool GRIDS>
__global__ void __launch_bounds__(XCH_MAX_T, 2) mea_moments_kernel(PartArgs a) {
  const int4 chunk = a.chunks[blockIdx.x];
  const int p = chunk.x, parts = chunk.w;
  const BoxDesc bd = a.boxes[a.box[p]];
  pdl_trigger();
  pdl_wait();
  __shared__ Rec R;
  __shared__ ExchangeRows rows;
  __shared__ long long wsum[XCH_MAX_T / 32][6];
  __shared__ MoveScratch mv;
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < 32) reinterpret_cast<int*>(&R)[tid] = reinterpret_cast<const int*>(&a.rec[p])[tid];
  if (a.move) {
    clear_bins(a);
    if (tid >= 64 && tid < 64 + PF_COUNT) mv.P[tid - 64] = pget(a.P, a.cap, tid - 64, p);
  }
  __syncthreads();
  long long s[6] = {0, 0, 0, 0, 0, 0};
  const S* f = reinterpret_cast<const S*>(a.f);
  const bool pairs = a.cells_x == 2;
  // a particle whose centre is not finite or far outside the box has no
  // interior cells (the update flags it)
  if (fabsf(R.xh[0]) < 1.0e6f && fabsf(R.xh[1]) < 1.0e6f && fabsf(R.xh[2]) < 1.0e6f) {
    for_interior<GRIDS>(R, bd, chunk.y, chunk.z, a.grids, rows, [&](int x, int y, int z, const float (&r)[3]) {
      float F[3], T[3];
      // cells next to a wall take the wall selects
      if (WALLS && (((bd.bc & 1) && (x == 0 || x == bd.nx - 1)) || ((bd.bc & 2) && (y == 0 || y == bd.ny - 1)) ||
                    ((bd.bc & 4) && (z == 0 || z == bd.nz - 1))))
        exchange_moments<S, PAR, WALLS>(f, R, bd, x, y, z, r, a.inv_scale, pairs, F, T);
      else
        exchange_moments<S, PAR, false>(f, R, bd, x, y, z, r, a.inv_scale, pairs, F, T);
#pragma unroll
      for (int k = 0; k < 6; ++k)
        s[k] += __float2ll_rn(__fmul_rn(k < 3 ? F[k % 3] : T[k % 3], (float)(1LL << ACC_FRAC_BITS)));
    });
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const long long v = warp_sum_i64(s[k]);
    if (lane == 0) wsum[tid >> 5][k] = v;
  }
  __syncthreads();
  long long sum = 0;
  if (tid < 6)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) sum += wsum[w][tid];
  unsigned long long* acc = reinterpret_cast<unsigned long long*>(a.acc) + (long long)p * 6;
  if (parts > 1) {
    if (tid < 6) {
      atomicAdd(&acc[tid], (unsigned long long)sum);
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) s_last = (atomicAdd(&a.done[p], 1) == parts - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid < 6) {
      sum = (long long)__ldcg(&acc[tid]);
      acc[tid] = 0;
    }
    if (tid == 0) a.done[p] = 0;
  }
  if (tid < 6) {
    const double t = (double)sum * (1.0 / (double)(1LL << ACC_FRAC_BITS));
    if (a.move) mv.F[tid] = t;
    else pset(a.P, a.cap, (tid < 3 ? PF_F : PF_T - 3) + tid, p, t);
  }
  if (!a.move) return;
  __syncthreads();
  move_particle(a, p, bd, R, mv);
}

// interior cells of every particle, added to *count
__global__ void __launch_bounds__(XCH_MAX_T) count_interior_kernel(PartArgs a, unsigned long long* count) {
  const int4 chunk = a.chunks[blockIdx.x];
  __shared__ Rec R;
  __shared__ ExchangeRows rows;
  if (threadIdx.x < 32)
    reinterpret_cast<int*>(&R)[threadIdx.x] = reinterpret_cast<const int*>(&a.rec[chunk.x])[threadIdx.x];
  const BoxDesc bd = a.boxes[a.box[chunk.x]];
  __syncthreads();
  unsigned n = 0;
  if (fabsf(R.xh[0]) < 1.0e6f && fabsf(R.xh[1]) < 1.0e6f && fabsf(R.xh[2]) < 1.0e6f)
    for_interior<true>(R, bd, chunk.y, chunk.z, a.grids, rows, [&](int, int, int, const float (&)[3]) { ++n; });
  n = __reduce_add_sync(0xffffffffu, n);
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(count, (unsigned long long)n);
}

__device__ __forceinline__ void cross3(const double a[3], const double b[3], double o[3]) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// Newton-Euler step (Eqs. particlemotiontrans, motionrot), symplectic Euler:
// U += F / m with F = F_h + (rho_p - rho_f) V g, X += U; spheres:
// omega += T / I; other shapes: body-frame Euler equations
// omega_b += (T_b - omega_b x (I omega_b)) / I with the rotation of the old
// quaternion; q += q (x) (0, omega_b) / 2, normalised (for a sphere in the
// equal form (0, omega) (x) q / 2, which needs no rotation).  GB300's FP64
// pipe is narrow: a warp's FP64 instruction takes it for many cycles however
// few lanes are active, so the translation and the rotation of a block's
// particles run on two warps (two SM sub-partitions) at once, each lane one
// particle, and meet in shared memory for the record and the binning.

// force of the momentum exchange (row base PF_F) or torque (PF_T) of particle
// p, as the exchange left it in the table, with the contact force or torque
// as an acting one beside it
__device__ __forceinline__ void exchange_force(const PartArgs& a, int p, int row, int crow, double Fo[3]) {
  for (int j = 0; j < 3; ++j) Fo[j] = pget(a.P, a.cap, row + j, p);
  if (a.contact_k > 0.0)
    for (int j = 0; j < 3; ++j) Fo[j] += pget(a.P, a.cap, crow + j, p);
}

// translation of particle p: force, U, X (wrapped on periodic axes), the
// record's position and velocity, and the tiles its bins cover
__device__ __forceinline__ void translate_particle(const PartArgs& a, int p, Rec& R, BinRange& br) {
  const double* __restrict__ P = a.P;
  const int cap = a.cap;
  const BoxDesc bd = a.boxes[a.box[p]];
  double X[3], U[3], Fh[3];
  for (int j = 0; j < 3; ++j) {
    X[j] = pget(P, cap, PF_X + j, p);
    U[j] = pget(P, cap, PF_U + j, p);
  }
  const double im = pget(P, cap, PF_IM, p), V = pget(P, cap, PF_V, p), rho = pget(P, cap, PF_RHO, p);
  const double rinf = pget(P, cap, PF_RINF, p), rc = pget(P, cap, PF_RC, p);
  exchange_force(a, p, PF_F, PF_FC, Fh);
  bool ok = true;
  for (int j = 0; j < 3; ++j) {
    const double F = Fh[j] + (rho - 1.0) * V * a.g[j];  // Fh: hydrodynamic (and contact) force
    U[j] += F * im;
    X[j] += U[j];
    ok = ok && isfinite(X[j]) && isfinite(U[j]);
  }
  if (!ok) atomicOr(a.status, ST_UNSTABLE);
  const int n[3] = {bd.nx, bd.ny, bd.nz};
  for (int j = 0; j < 3; ++j) {
    if ((bd.bc >> j) & 1) {
      // a slab's cut z faces are not walls: centres may lie beyond them
      const bool cut = j == 2 && (bd.bc & BC_CUT_Z);
      if (!cut && !(X[j] > -0.5 && X[j] < n[j] - 0.5)) atomicOr(a.status, ST_LEFT_DOMAIN);
    } else {
      // a particle moves far less than a box length per step
      const double L = (double)n[j];
      if (X[j] >= L) X[j] -= L;
      else if (X[j] < 0.0) X[j] += L;
    }
  }
  for (int j = 0; j < 3; ++j) {
    pset(a.P, cap, PF_X + j, p, X[j]);
    pset(a.P, cap, PF_U + j, p, U[j]);
    const float xh = __double2float_rn(X[j]);
    R.xh[j] = xh;
    R.xl[j] = __double2float_rn(X[j] - (double)xh);
    R.u[j] = (float)U[j];
  }
  br.tile_off = bd.tile_off;
  br.ntx = bd.ntx;
  br.nty = bd.nty;
  br.count = 0;
  const float rb = __double2float_ru(fmax(rinf, rc + 1.5));
  const int T[3] = {TILE_X, TILE_Y, TILE_Z};
  for (int j = 0; j < 3; ++j) {
    if (!(X[j] > -1.0e6 && X[j] < 1.0e6)) return;  // flagged above; not binned
    br.at[j] = bin_axis(X[j], rb, n[j], T[j], (bd.bc >> j) & 1);
  }
  br.count = br.at[0].count() * br.at[1].count() * br.at[2].count();
}

// rotation of particle p: torque, omega, quaternion, the record's angular
// velocity and orientation; the record's fixed fields (shape, box, id, sizes
// and the bounds derived from them) come from its previous record
__device__ __forceinline__ void rotate_particle(const PartArgs& a, int p, Rec& R) {
  const double* __restrict__ P = a.P;
  const int cap = a.cap;
  const int shape = a.shape[p];
  double W[3], q[4], I[3], iI[3], Th[3];
  for (int j = 0; j < 3; ++j) {
    W[j] = pget(P, cap, PF_W + j, p);
    iI[j] = pget(P, cap, PF_II + j, p);
    I[j] = shape == 0 ? 0.0 : pget(P, cap, PF_I + j, p);
  }
  for (int j = 0; j < 4; ++j) q[j] = pget(P, cap, PF_Q + j, p);
  const Rec& old = a.rec[p];
  for (int j = 0; j < 3; ++j) {
    R.a[j] = old.a[j];
    R.ia[j] = old.ia[j];
  }
  R.in2 = old.in2;
  R.rinf2 = old.rinf2;
  R.shape = old.shape;
  R.box = old.box;
  R.pid = old.pid;
  if (shape == 0)
    for (int k = 0; k < 9; ++k) R.M[k] = old.M[k];  // a sphere's collision bounds
  exchange_force(a, p, PF_T, PF_TC, Th);
  const double w = q[0], x = q[1], y = q[2], z = q[3];
  double dq[4];
  if (shape == 0) {
    // q (x) (0, omega_b) equals (0, omega) (x) q: no rotation needed
    for (int j = 0; j < 3; ++j) W[j] += Th[j] * iI[j];
    dq[0] = -0.5 * (W[0] * x + W[1] * y + W[2] * z);
    dq[1] = 0.5 * (w * W[0] + W[1] * z - W[2] * y);
    dq[2] = 0.5 * (w * W[1] + W[2] * x - W[0] * z);
    dq[3] = 0.5 * (w * W[2] + W[0] * y - W[1] * x);
  } else {
    double Rm[9], wb[3], Tb[3], Lb[3], gy[3];
    rotation_rn(q, Rm);
    for (int j = 0; j < 3; ++j) {
      wb[j] = Rm[0 * 3 + j] * W[0] + Rm[1 * 3 + j] * W[1] + Rm[2 * 3 + j] * W[2];
      Tb[j] = Rm[0 * 3 + j] * Th[0] + Rm[1 * 3 + j] * Th[1] + Rm[2 * 3 + j] * Th[2];
    }
    for (int j = 0; j < 3; ++j) Lb[j] = I[j] * wb[j];
    cross3(wb, Lb, gy);
    for (int j = 0; j < 3; ++j) wb[j] += (Tb[j] - gy[j]) * iI[j];
    for (int j = 0; j < 3; ++j) W[j] = Rm[j * 3 + 0] * wb[0] + Rm[j * 3 + 1] * wb[1] + Rm[j * 3 + 2] * wb[2];
    dq[0] = 0.5 * (-x * wb[0] - y * wb[1] - z * wb[2]);
    dq[1] = 0.5 * (w * wb[0] + y * wb[2] - z * wb[1]);
    dq[2] = 0.5 * (w * wb[1] + z * wb[0] - x * wb[2]);
    dq[3] = 0.5 * (w * wb[2] + x * wb[1] - y * wb[0]);
  }
  double nq = 0.0;
  for (int j = 0; j < 4; ++j) {
    q[j] += dq[j];
    nq += q[j] * q[j];
  }
  const double inq = rsqrt(nq);
  for (int j = 0; j < 4; ++j) q[j] *= inq;
  if (!(isfinite(W[0]) && isfinite(W[1]) && isfinite(W[2]))) atomicOr(a.status, ST_UNSTABLE);
  for (int j = 0; j < 3; ++j) {
    pset(a.P, cap, PF_W + j, p, W[j]);
    R.w[j] = (float)W[j];
  }
  for (int j = 0; j < 4; ++j) pset(a.P, cap, PF_Q + j, p, q[j]);
  if (shape != 0) {
    double Rn[9];
    rotation_rn(q, Rn);
    for (int k = 0; k < 9; ++k) R.M[k] = __double2float_rn(Rn[k]);
  }
}

// a.ppb particles per block of UPD_T threads (ppb a power of two up to
// UPD_P): lane k of warp 0 moves particle k of the block, lane k of warp 1
// turns it; then all threads store the records and add the block's
// particles to the per-tile lists, UPD_T / ppb threads per particle taking
// its tiles in turn.  Few particles get small groups, so that the blocks
// spread over the GPU and each particle's tiles take one round of atomics.
constexpr int UPD_P = 32, UPD_T = 256;

__global__ void __launch_bounds__(UPD_T) update_kernel(PartArgs a) {
  __shared__ BinRange s_br[UPD_P];
  __shared__ Rec s_rec[UPD_P];
  pdl_trigger();
  pdl_wait();
  clear_bins(a);
  const int ppb = a.ppb;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (long long base = blockIdx.x * (long long)ppb; base < a.np; base += (long long)gridDim.x * ppb) {
    if (warp < 2 && lane < ppb) {
      const long long p = base + lane;
      if (p < a.np) {
        if (warp == 0) translate_particle(a, (int)p, s_rec[lane], s_br[lane]);
        else rotate_particle(a, (int)p, s_rec[lane]);
      } else if (warp == 0) {
        s_br[lane].count = 0;
      }
    }
    __syncthreads();
    const long long nrec = min((long long)ppb, a.np - base);
    for (int e = threadIdx.x; e < nrec * 32; e += UPD_T)
      reinterpret_cast<int*>(&a.rec[base + (e >> 5)])[e & 31] = reinterpret_cast<const int*>(&s_rec[e >> 5])[e & 31];
    const int k = threadIdx.x % ppb, sub = threadIdx.x / ppb;
    bin_particle(a, s_br[k], (int)(base + k), sub, UPD_T / ppb);
    __syncthreads();
  }
}

// ---------------------------------------------------------------- contact
// Contact between particles (an extension: the paper counts contact among
// the acting forces of Sec. 2.2 without stating a model, and its runs have
// none).  Each particle is enclosed by a capsule, the points within r_c of
// the segment X +- h_c e: a sphere by itself (h_c = 0), a capsule by itself,
// an ellipsoid by the capsule along its longest semi-axis a_k with r_c the
// larger other semi-axis and h_c = a_k - r_c, a cuboid by the capsule along
// its longest half-extent h_k with r_c = |(h_i, h_j)| and h_c = h_k.  Two
// capsules whose segments come closest at p_i, p_j (minimum image) with gap
// delta = |p_i - p_j| - r_i - r_j < zeta repel along n = (p_i - p_j) / |.|
// with k ((zeta - delta) / zeta)^2, and particle i takes the torque
// (p_i - X_i) x F_i; a wall pushes the segment end nearest to it the same
// way.  All in FP64 from the particle table at the state before the update.

// enclosing capsule of particle p: unit axis e, half-length h, radius r
__device__ __forceinline__ void contact_capsule(const double* P, int cap, int p, int shape, double e[3],
                                                double& h, double& r) {
  double A[3], q[4];
  for (int j = 0; j < 3; ++j) A[j] = pget(P, cap, PF_A + j, p);
  for (int j = 0; j < 4; ++j) q[j] = pget(P, cap, PF_Q + j, p);
  int k = 2;
  if (shape == 0 || shape == 4) {  // a grid particle: the sphere of its circumscribed radius
    h = 0.0;
    r = A[0];
  } else if (shape == 3) {
    h = A[2];
    r = A[0];
  } else {
    k = A[1] > A[0] ? 1 : 0;
    if (A[2] > A[k]) k = 2;
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    if (shape == 1) {
      r = fmax(A[i], A[j]);
      h = A[k] - r;
    } else {
      r = sqrt(A[i] * A[i] + A[j] * A[j]);
      h = A[k];
    }
  }
  if (shape == 0 || shape == 4) {
    e[0] = 0.0; e[1] = 0.0; e[2] = 1.0;
    return;
  }
  double R[9];
  rotation_rn(q, R);
  for (int j = 0; j < 3; ++j) e[j] = R[j * 3 + k];
}

// FP32 bound on the reach of a particle's contact capsule from its centre
__device__ __forceinline__ float contact_reach(const Rec& R) {
  if (R.shape == 0 || R.shape == 4) return R.a[0];
  if (R.shape == 3) return R.a[0] + R.a[2];
  const float amax = fmaxf(R.a[0], fmaxf(R.a[1], R.a[2]));
  if (R.shape == 1) return amax;
  return sqrtf(R.a[0] * R.a[0] + R.a[1] * R.a[1] + R.a[2] * R.a[2]) + amax;  // >= h_k + |(h_i, h_j)|
}

// closest points P + s u, Q + t v of two segments (|s| <= hu, |t| <= hv,
// unit u, v): the points of closest approach of the two lines, s clamped,
// t taken from s and clamped, s taken again from t and clamped
__device__ __forceinline__ void segment_closest(const double P[3], const double u[3], double hu,
                                                const double Q[3], const double v[3], double hv,
                                                double& s, double& t) {
  double b = 0.0, d = 0.0, f = 0.0;
  for (int j = 0; j < 3; ++j) {
    const double w = P[j] - Q[j];
    b += u[j] * v[j];
    d += u[j] * w;
    f += v[j] * w;
  }
  const double den = 1.0 - b * b;
  s = den > 1e-12 ? fmin(fmax((b * f - d) / den, -hu), hu) : 0.0;
  t = fmin(fmax(b * s + f, -hv), hv);
  s = fmin(fmax(b * t - d, -hu), hu);
}

__device__ __forceinline__ double contact_ramp(double k, double zeta, double gap) {
  const double x = (zeta - gap) / zeta;
  return k * x * x;
}

// One warp per particle.  The block stages the others' centres and reaches
// in shared memory, CT_CHUNK at a time; the lanes test them in FP32 (centre
// distance against the capsules' reach) and list those near enough, which
// then take the FP64 arithmetic together, a lane each: its long dependent
// chains cost the same for one lane and for 32, and a warp that ran them at
// every group of 32 with a near particle spent its time there (495 spheres 33
// us before).  Lane 0 takes the walls; the warp's FP64 sums are added in a
// fixed order.
constexpr int CT_WARPS = 4, CT_CHUNK = 256, CT_NEAR = 64;

__global__ void __launch_bounds__(CT_WARPS * 32) contact_kernel(PartArgs a) {
  __shared__ float4 s_pos[CT_CHUNK];  // centre, reach of the contact capsule
  __shared__ int s_box[CT_CHUNK];
  __shared__ int s_near[CT_WARPS][CT_NEAR];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * CT_WARPS + warp;
  const bool active = i < a.np;  // whole warps; all threads stage
  const double* P = a.P;
  const int cap = a.cap;
  // what no step changes is read before the wait for the kernel before
  const int box = active ? a.box[i] : 0, shape = active ? a.shape[i] : 0;
  const BoxDesc bd = a.boxes[box];
  pdl_trigger();
  pdl_wait();
  const int n[3] = {bd.nx, bd.ny, bd.nz};
  const float L[3] = {(float)bd.nx, (float)bd.ny, (float)bd.nz};
  float xi[3] = {0.f, 0.f, 0.f}, reach_i = 0.f;
  double Xi[3] = {0.0, 0.0, 0.0}, ei[3] = {0.0, 0.0, 1.0}, hi = 0.0, ri = 0.0;
  if (active) {
    const Rec& Ri = a.rec[i];
    for (int c = 0; c < 3; ++c) {
      xi[c] = Ri.xh[c];
      Xi[c] = pget(P, cap, PF_X + c, i);
    }
    reach_i = contact_reach(Ri);
    contact_capsule(P, cap, i, shape, ei, hi, ri);
  }
  const double k = a.contact_k, zeta = a.contact_zeta;
  double F[3] = {0.0, 0.0, 0.0}, T[3] = {0.0, 0.0, 0.0};
  auto add = [&](const double pt[3], const double f[3]) {
    const double arm[3] = {pt[0] - Xi[0], pt[1] - Xi[1], pt[2] - Xi[2]};
    double tq[3];
    cross3(arm, f, tq);
    for (int c = 0; c < 3; ++c) {
      F[c] += f[c];
      T[c] += tq[c];
    }
  };
  auto pair = [&](int j) {
    double Xj[3], ej[3], hj, rj;
    for (int c = 0; c < 3; ++c) {
      double dc = pget(P, cap, PF_X + c, j) - Xi[c];
      if (!((bd.bc >> c) & 1)) {
        const double Ld = (double)n[c];
        if (dc > Ld / 2.0) dc -= Ld;
        else if (dc < -Ld / 2.0) dc += Ld;
      }
      Xj[c] = Xi[c] + dc;
    }
    contact_capsule(P, cap, j, a.shape[j], ej, hj, rj);
    double s = 0.0, t = 0.0;
    if (hi > 0.0 || hj > 0.0) segment_closest(Xi, ei, hi, Xj, ej, hj, s, t);  // two spheres: the centres
    double pi[3], dv[3], dist = 0.0;
    for (int c = 0; c < 3; ++c) {
      pi[c] = Xi[c] + s * ei[c];
      dv[c] = pi[c] - (Xj[c] + t * ej[c]);
      dist += dv[c] * dv[c];
    }
    dist = sqrt(dist);
    const double gap = dist - ri - rj;
    if (gap >= zeta || !(dist > 0.0)) return;
    const double fm = contact_ramp(k, zeta, gap);
    const double f[3] = {fm * dv[0] / dist, fm * dv[1] / dist, fm * dv[2] / dist};
    add(pi, f);
  };
  int near = 0;
  auto flush = [&]() {
    __syncwarp();
    for (int c = lane; c < near; c += 32) pair(s_near[warp][c]);
    __syncwarp();
    near = 0;
  };
  const float far = (float)zeta + 0.05f;
  for (int j0 = 0; j0 < a.np; j0 += CT_CHUNK) {
    __syncthreads();
    for (int e = threadIdx.x; e < CT_CHUNK && j0 + e < a.np; e += CT_WARPS * 32) {
      const Rec& Rj = a.rec[j0 + e];
      s_pos[e] = make_float4(Rj.xh[0], Rj.xh[1], Rj.xh[2], contact_reach(Rj));
      s_box[e] = Rj.box;
    }
    __syncthreads();
    if (!active) continue;
    const int m = min(CT_CHUNK, a.np - j0);
    for (int e0 = 0; e0 < m; e0 += 32) {
      const int e = e0 + lane;
      bool hit = false;
      if (e < m && j0 + e != i && s_box[e] == box) {
        const float4 q = s_pos[e];
        float d2 = 0.0f;
        const float xj[3] = {q.x, q.y, q.z};
        for (int c = 0; c < 3; ++c) {
          float dc = xj[c] - xi[c];
          if (!((bd.bc >> c) & 1)) {
            if (dc > 0.5f * L[c]) dc -= L[c];
            else if (dc < -0.5f * L[c]) dc += L[c];
          }
          d2 += dc * dc;
        }
        const float lim = reach_i + q.w + far;
        hit = d2 < lim * lim;
      }
      const unsigned h = __ballot_sync(0xffffffffu, hit);
      if (!h) continue;
      if (near + __popc(h) > CT_NEAR) flush();
      if (hit) s_near[warp][near + __popc(h & ((1u << lane) - 1u))] = j0 + e;
      near += __popc(h);
    }
  }
  if (!active) return;
  flush();
  if (lane == 0)
    for (int c = 0; c < 3; ++c) {
      if (!((bd.bc >> c) & 1) || (c == 2 && (bd.bc & BC_CUT_Z))) continue;
      for (int side = 0; side < 2; ++side) {
        const double dir = side == 0 ? -1.0 : 1.0;
        const double t = ei[c] * dir > 0.0 ? hi : (ei[c] * dir < 0.0 ? -hi : 0.0);
        const double pt[3] = {Xi[0] + t * ei[0], Xi[1] + t * ei[1], Xi[2] + t * ei[2]};
        const double gap = (side == 0 ? pt[c] + 0.5 : (n[c] - 0.5) - pt[c]) - ri;
        if (gap >= zeta) continue;
        double f[3] = {0.0, 0.0, 0.0};
        f[c] = -dir * contact_ramp(k, zeta, gap);
        add(pt, f);
      }
    }
  if (__any_sync(0xffffffffu, F[0] != 0.0 || F[1] != 0.0 || F[2] != 0.0))
    for (int c = 0; c < 3; ++c)
      for (int o = 16; o > 0; o >>= 1) {
        F[c] += __shfl_xor_sync(0xffffffffu, F[c], o);
        T[c] += __shfl_xor_sync(0xffffffffu, T[c], o);
      }
  if (lane == 0)
    for (int c = 0; c < 3; ++c) {
      pset(a.P, cap, PF_FC + c, i, F[c]);
      pset(a.P, cap, PF_TC + c, i, T[c]);
    }
}

__global__ void records_kernel(PartArgs a) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.np) return;
  Rec R;
  build_record(a.P, a.cap, p, a.shape[p], a.box[p], (float)a.eps, R);
  a.rec[p] = R;
}

template <typename S, int PAR>
static cudaError_t launch_mea_sp(const PartArgs& a, bool walls, bool moments, cudaStream_t s) {
  const bool g = a.grids.desc != nullptr;
  auto go = [&](auto kern) {
    return launch_k(kern, dim3((unsigned)a.nchunks), dim3((unsigned)a.mea_threads), 0, s, a.pdl != 0, a);
  };
  if (moments) {
    if (walls) return g ? go(mea_moments_kernel<S, PAR, true, true>) : go(mea_moments_kernel<S, PAR, true, false>);
    return g ? go(mea_moments_kernel<S, PAR, false, true>) : go(mea_moments_kernel<S, PAR, false, false>);
  }
  if (walls) return g ? go(mea_kernel<S, PAR, true, true>) : go(mea_kernel<S, PAR, true, false>);
  return g ? go(mea_kernel<S, PAR, false, true>) : go(mea_kernel<S, PAR, false, false>);
}

cudaError_t launch_mea(const PartArgs& a, int precision, int parity, bool walls, bool moments, cudaStream_t s) {
  if (a.np <= 0 || a.nchunks <= 0) return cudaSuccess;
  if (precision == 0)
    return parity == 0 ? launch_mea_sp<float, 0>(a, walls, moments, s) : launch_mea_sp<float, 1>(a, walls, moments, s);
  return parity == 0 ? launch_mea_sp<__half, 0>(a, walls, moments, s) : launch_mea_sp<__half, 1>(a, walls, moments, s);
}

cudaError_t launch_count_interior(const PartArgs& a, unsigned long long* count, cudaStream_t s) {
  if (a.np <= 0 || a.nchunks <= 0) return cudaSuccess;
  count_interior_kernel<<<(unsigned)a.nchunks, (unsigned)a.mea_threads, 0, s>>>(a, count);
  return cudaGetLastError();
}

cudaError_t launch_update(const PartArgs& a_in, cudaStream_t s) {
  PartArgs a = a_in;
  // particles per block: the smallest power of two that keeps the blocks
  // within about one per SM, at most UPD_P
  const long long target = a.nsm > 0 ? a.nsm : 152;
  a.ppb = 1;
  while (a.ppb < UPD_P && (long long)a.ppb * target < a.np) a.ppb *= 2;
  long long blocks = (a.np + a.ppb - 1) / a.ppb;
  long long clear_blocks = (a.ntiles + UPD_T - 1) / UPD_T;
  if (clear_blocks > blocks) blocks = clear_blocks;
  if (blocks > 65535) blocks = 65535;
  if (blocks < 1) blocks = 1;
  return launch_k(update_kernel, dim3((unsigned)blocks), dim3(UPD_T), 0, s, a.pdl != 0, a);
}

cudaError_t launch_contact(const PartArgs& a, cudaStream_t s) {
  if (a.np <= 0 || !(a.contact_k > 0.0)) return cudaSuccess;
  return launch_k(contact_kernel, dim3((unsigned)((a.np + CT_WARPS - 1) / CT_WARPS)), dim3(CT_WARPS * 32), 0, s,
                  a.pdl != 0, a);
}

cudaError_t launch_records(const PartArgs& a, cudaStream_t s) {
  if (a.np <= 0) return cudaSuccess;
  records_kernel<<<(a.np + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace hlbm
