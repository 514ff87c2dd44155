// The truncation of one bond (OpTrunc of pv_batch.cuh: one-sided Jacobi, the leading left
// singular vectors, the normalised environment tensor) as a device kernel that computes the
// same bits as OpTrunc::run with the pairing of a `gthr`-thread block.
//
// What bounds it: a sweep visits nc (nc - 1) / 2 column pairs, each a dot product, a test and,
// where it rotates, an update of both columns and their norms; the matrix stays in shared
// memory, so the costs are FMA issue, shared-memory accesses and the scalar arithmetic of a
// rotation (two square roots and three divisions), which in float64 (2 FMAs per clock and SM on
// GB300) outweighs the columns' own work.  Measured in float32 (ncu): eight matrices of an 8x8
// D=4 chi=16 bond an SM issue in 53 % of the cycles with the shared-memory pipe at 31 to 36 %, one
// 216 x 216 matrix an SM in 45 % at 20 to 35 %: the 14 to 16 warps that 118 to 127 registers a thread
// leave an SM do not cover the latency of dependent arithmetic and shared-memory loads (1.5 and
// 1.4 stalled warps an issue) and, at 216 columns, of a round's barrier (1.4).
//
// Layout: G lanes own a pair; lane gl holds the elements i = gl + G e of both columns (the
// summation order of jacobi()), stored so that VW = 16 / sizeof(T) consecutive e of one lane are
// one 16-byte vector and the G lanes of a vector index are contiguous (no bank conflicts, one
// load per VW elements instead of VW).  A warp takes TT pairs per lane group at a time in
// registers:
//  - the squared norms of the columns (and their roots) are kept per column and recomputed, in
//    the order jacobi() sums them, only when a rotation changes the column: a visit that does
//    not rotate costs one dot product instead of three and no square root;
//  - the TT dot products of a group are reduced by recursive halving (each level exchanges
//    half of the values), which leaves each pair's sum in its own lanes, so the scalar
//    arithmetic of all pairs of the warp's step is done once, one pair per lane, instead of once
//    per lane group and step;
//  - c and s are broadcast back to the lane group; a step in which no pair rotates stores
//    nothing.
// Sums are the same trees as the butterfly's (addition commutes) and every product that enters one
// is fused as there (jac_fma, jac_rot), so every bit is that of jacobi(), in float32 and float64.
//
// Measured (mean per launch over one evaluation, the former kernel in brackets): float32 8x8
// D=4 chi=16, 2048 chains 0.51 ms (1.73); 6x6 D=4 chi=16, 128 chains 63 us (347); 10x10 D=6
// chi=36 (up to 216 x 216), 192 chains 4.4 ms (7.6); float64 8x8 D=4 chi=16, 128 chains 2.9 ms
// (7.2).
#ifndef PV_JACOBI_CUH
#define PV_JACOBI_CUH

#if defined(__CUDACC__)
namespace pv {

// Work shape of a truncation in shared memory: lanes per pair (as jacobi() picks them for a
// block of gthr threads), 16-byte vectors per lane of a column of Y and of V, and the bytes.
struct JacShape {
  int G, lg, chY, chV;
  size_t bytes;
};

template <typename T>
inline JacShape jac_shape(int nc, int len, int m, bool tall, int gthr) {
  JacShape s;
  const int npair = (nc + (nc & 1)) / 2, VW = 16 / (int)sizeof(T);
  s.G = 1;
  s.lg = 0;
  while (s.G < 32 && s.G * 2 * npair <= gthr) {
    s.G *= 2;
    ++s.lg;
  }
  const int q = VW * s.G;
  s.chY = (len + q - 1) / q;
  s.chV = tall ? 0 : (m + q - 1) / q;
  const size_t elems = (size_t)nc * s.chY * q + (size_t)m * s.chV * q + 3 * ((size_t)nc + 4);
  s.bytes = elems * sizeof(T) + ((size_t)nc + 4) * sizeof(int) + 16;
  return s;
}

template <typename T>
struct JacVec;
template <>
struct JacVec<float> {
  typedef float4 V;
};
template <>
struct JacVec<double> {
  typedef double2 V;
};

template <typename T, int VW>
__device__ __forceinline__ void jac_ld(T* r, const T* p) {
  typedef typename JacVec<T>::V V;
  const V v = *(const V*)p;
  r[0] = v.x;
  r[1] = v.y;
  if constexpr (VW == 4) {
    r[2] = v.z;
    r[3] = v.w;
  }
}
template <typename T, int VW>
__device__ __forceinline__ void jac_st(T* p, const T* r) {
  typedef typename JacVec<T>::V V;
  V v;
  v.x = r[0];
  v.y = r[1];
  if constexpr (VW == 4) {
    v.z = r[2];
    v.w = r[3];
  }
  *(V*)p = v;
}

// Sums v[t] over the G lanes of a group; returns the sum of the value t that this lane owns
// (jac_own): the first log2(TT) levels exchange halves, the rest are a butterfly.
template <typename T, int TT>
__device__ __forceinline__ T jac_reduce(T (&v)[TT], int G, int gl) {
  int o = G >> 1;
  if constexpr (TT == 4) {
    const bool h = gl & o;
    const T k0 = h ? v[2] : v[0], k1 = h ? v[3] : v[1];
    const T s0 = h ? v[0] : v[2], s1 = h ? v[1] : v[3];
    const T r0 = k0 + __shfl_xor_sync(0xffffffffu, s0, o), r1 = k1 + __shfl_xor_sync(0xffffffffu, s1, o);
    o >>= 1;
    const bool h2 = gl & o;
    T r = (h2 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, h2 ? r0 : r1, o);
    for (o >>= 1; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
  } else if constexpr (TT == 2) {
    const bool h = gl & o;
    T r = (h ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, h ? v[0] : v[1], o);
    for (o >>= 1; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
  } else {
    T r = v[0];
    for (; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
  }
}

// One term of a dot product or norm, and the rotation of one element of a pair, their rounding
// pinned to that of jacobi().  Left to the compiler, which products of an unrolled sum are fused depends
// on the variant below: in float64 the variants then differed from each other in the last bits
// (2e-14 in the kept vectors of 64 x 64 matrices).
__device__ __forceinline__ float jac_fma(float x, float y, float a) { return __fmaf_rn(x, y, a); }
__device__ __forceinline__ double jac_fma(double x, double y, double a) { return __fma_rn(x, y, a); }
__device__ __forceinline__ float jac_mul(float x, float y) { return __fmul_rn(x, y); }
__device__ __forceinline__ double jac_mul(double x, double y) { return __dmul_rn(x, y); }
template <typename T>
__device__ __forceinline__ void jac_rot(T c, T s, T x, T y, T& u, T& w) {
  u = jac_fma(c, x, -jac_mul(s, y));
  w = jac_fma(s, x, jac_mul(c, y));
}

// Column pair of slot pr in round rnd of the round-robin order (p < q); false when the slot is
// past the end or holds the empty position of an odd column count.
__device__ __forceinline__ bool jac_pair(int rnd, int pr, int np, int nc, int& p, int& q) {
  const int w = np - 1;
  int a = rnd + pr, b = rnd - pr;
  if (a >= w) a -= w;
  if (b < 0) b += w;
  if (pr == 0) {
    a = w;
    b = rnd;
  }
  p = a < b ? a : b;
  q = a < b ? b : a;
  if (pr >= (np >> 1) || q >= nc) {
    p = q = 0;
    return false;
  }
  return true;
}

// T: working type; ST: storage type of Y, U and the environment.  CH: 16-byte vectors per lane
// and column held in registers (at least chY), or 0 to read the columns again for the rotation
// (columns too long for registers).
// The whole block works on matrix s; `dyn` is its shared work area (JacShape::bytes), `red` 32
// shared entries.
template <typename T, typename ST, int CH, int TT>
__device__ __forceinline__ void jac_matrix(const OpTrunc<ST>& op, int s, unsigned char* dyn, T* red, int G,
                                           int lg, int chY, int chV, T tol) {
  constexpr int VW = 16 / sizeof(T);
  constexpr int R = CH > 0 ? CH * VW : 1;
  const int nc = op.nc, len = op.len, m = op.m, kk = op.kk;
  const bool tall = op.tall;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  const int ldy = chY * VW * G, ldv = chV * VW * G;
  T* Y = (T*)dyn;
  T* V = Y + (size_t)nc * ldy;
  T* nrm = V + (tall ? (size_t)0 : (size_t)m * ldv);
  T* rt = nrm + nc + 4;    // square roots of nrm
  T* sig = rt + nc + 4;
  int* order = (int*)(sig + nc + 4);
  const int gl = lane & (G - 1), grpw = lane >> lg, gpw = 32 >> lg;
  const int np = nc + (nc & 1), npair = np >> 1;
  const T eps = sizeof(T) == 4 ? (T)1.1920929e-7 : (T)2.220446049250313e-16;
  const T tol_eff = tol > (T)4 * len * eps ? tol : (T)4 * len * eps;
  // position of element i of a column
  auto pos = [&](int i) {
    const int e = i >> lg, g = i & (G - 1);
    return ((e / VW) * G + g) * VW + (e & (VW - 1));
  };
  // the pair whose sums this lane owns after jac_reduce
  const int own = TT == 4 ? ((gl & (G >> 1)) ? 2 : 0) + ((gl & (G >> 2)) ? 1 : 0)
                          : (TT == 2 ? ((gl & (G >> 1)) ? 1 : 0) : 0);
  const bool writer = (gl & ((TT == 4 ? G >> 2 : (TT == 2 ? G >> 1 : G)) - 1)) == 0;

  {
    const ST* Ys = op.Y + (long long)s * op.ys;
    for (int j = warp; j < nc; j += nwarp)
      for (int i = lane; i < ldy; i += 32) Y[j * ldy + pos(i)] = i < len ? (T)Ys[(long long)j * len + i] : (T)0;
    if (!tall)
      for (int j = warp; j < m; j += nwarp)
        for (int i = lane; i < ldv; i += 32) V[j * ldv + pos(i)] = i == j ? (T)1 : (T)0;
    __syncthreads();
    int sw = 0;
    if (nc >= 2) {
      // squared norm of the matrix in jacobi()'s order
      T nf2 = 0;
      if (warp == 0) {
        for (int j = 0; j < nc; ++j)
          for (int i = lane; i < len; i += 32) {
            const T y = Y[j * ldy + pos(i)];
            nf2 = jac_fma(y, y, nf2);
          }
        nf2 = warp_sum(nf2);
        if (lane == 0) red[0] = nf2;
      }
      // squared norms of the columns
      for (int j0 = warp * gpw; j0 < nc; j0 += nwarp * gpw) {
        const int j = j0 + grpw;
        T a = 0;
        if (j < nc)
          for (int c = 0; c < chY; ++c) {
            T u[VW];
            jac_ld<T, VW>(u, Y + (size_t)j * ldy + (c * G + gl) * VW);
#pragma unroll
            for (int k = 0; k < VW; ++k) a = jac_fma(u[k], u[k], a);
          }
        for (int o = G >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (j < nc && gl == 0) {
          nrm[j] = a;
          rt[j] = sqrt(a);
        }
      }
      __syncthreads();
      nf2 = red[0];
      const T tiny = (eps * len) * (eps * len) * nf2;
      int sweep = 0;
      for (; sweep < op.max_sweeps; ++sweep) {
        bool any = false;
        for (int rnd = 0; rnd < np - 1; ++rnd) {
          for (int base = warp * (gpw * TT); base < npair; base += nwarp * (gpw * TT)) {
            T x[TT][R], y[TT][R], g[TT];
            int xp[TT], xq[TT];   // element offsets of this lane's first vectors in Y
            bool act[TT];
#pragma unroll
            for (int t = 0; t < TT; ++t) {
              int p, q;
              act[t] = jac_pair(rnd, base + t * gpw + grpw, np, nc, p, q);
              xp[t] = p * ldy + gl * VW;
              xq[t] = q * ldy + gl * VW;
              g[t] = 0;
              if constexpr (CH > 0) {
#pragma unroll
                for (int c = 0; c < CH; ++c)
                  if (c < chY) {
                    jac_ld<T, VW>(x[t] + c * VW, Y + xp[t] + c * G * VW);
                    jac_ld<T, VW>(y[t] + c * VW, Y + xq[t] + c * G * VW);
                  }
              }
            }
#pragma unroll
            for (int t = 0; t < TT; ++t) {
              if constexpr (CH > 0) {
#pragma unroll
                for (int c = 0; c < CH; ++c)
                  if (c < chY)
#pragma unroll
                    for (int k = 0; k < VW; ++k) g[t] = jac_fma(x[t][c * VW + k], y[t][c * VW + k], g[t]);
              } else {
                for (int c = 0; c < chY; ++c) {
                  T u[VW], w[VW];
                  jac_ld<T, VW>(u, Y + xp[t] + c * G * VW);
                  jac_ld<T, VW>(w, Y + xq[t] + c * G * VW);
#pragma unroll
                  for (int k = 0; k < VW; ++k) g[t] = jac_fma(u[k], w[k], g[t]);
                }
              }
            }
            const T gv = jac_reduce<T, TT>(g, G, gl);
            // this lane's own pair
            int p, q;
            const bool a_own = jac_pair(rnd, base + own * gpw + grpw, np, nc, p, q);
            const T a = nrm[p], b = nrm[q];
            const T ag = gv < 0 ? -gv : gv;
            const bool rot = a_own && ag > tol_eff * rt[p] * rt[q] && a > tiny && b > tiny;
            const unsigned mask = __ballot_sync(0xffffffffu, rot);
            if (!mask) continue;
            any = true;
            T cs = 1, sn = 0;
            if (rot) {
              const T zeta = (b - a) / ((T)2 * gv);
              const T az = zeta < 0 ? -zeta : zeta;
              T t = (T)1 / (az + sqrt((T)1 + az * az));
              if (zeta < 0) t = -t;
              cs = (T)1 / sqrt((T)1 + t * t);
              sn = cs * t;
            }
            T na[TT], nb[TT];
#pragma unroll
            for (int t = 0; t < TT; ++t) {
              int src = lane & ~(G - 1);   // a lane of this group that owns pair t
              if (TT == 4) src += (t & 2 ? G >> 1 : 0) + (t & 1 ? G >> 2 : 0);
              if (TT == 2) src += t ? G >> 1 : 0;
              const T c0 = __shfl_sync(0xffffffffu, cs, src), s0 = __shfl_sync(0xffffffffu, sn, src);
              na[t] = nb[t] = 0;
              if (act[t] && ((mask >> src) & 1u)) {
                if constexpr (CH > 0) {
#pragma unroll
                  for (int c = 0; c < CH; ++c)
                    if (c < chY) {
                      T u[VW], w[VW];
#pragma unroll
                      for (int k = 0; k < VW; ++k) {
                        const T x0 = x[t][c * VW + k], y0 = y[t][c * VW + k];
                        jac_rot(c0, s0, x0, y0, u[k], w[k]);
                        na[t] = jac_fma(u[k], u[k], na[t]);
                        nb[t] = jac_fma(w[k], w[k], nb[t]);
                      }
                      jac_st<T, VW>(Y + xp[t] + c * G * VW, u);
                      jac_st<T, VW>(Y + xq[t] + c * G * VW, w);
                    }
                } else {
                  for (int c = 0; c < chY; ++c) {
                    T u[VW], w[VW];
                    jac_ld<T, VW>(u, Y + xp[t] + c * G * VW);
                    jac_ld<T, VW>(w, Y + xq[t] + c * G * VW);
#pragma unroll
                    for (int k = 0; k < VW; ++k) {
                      const T x0 = u[k], y0 = w[k];
                      jac_rot(c0, s0, x0, y0, u[k], w[k]);
                      na[t] = jac_fma(u[k], u[k], na[t]);
                      nb[t] = jac_fma(w[k], w[k], nb[t]);
                    }
                    jac_st<T, VW>(Y + xp[t] + c * G * VW, u);
                    jac_st<T, VW>(Y + xq[t] + c * G * VW, w);
                  }
                }
                if (!tall) {
                  T* vp = V + xp[t] / ldy * ldv + gl * VW;
                  T* vq = V + xq[t] / ldy * ldv + gl * VW;
                  for (int c = 0; c < chV; ++c) {
                    T u[VW], w[VW];
                    jac_ld<T, VW>(u, vp + c * G * VW);
                    jac_ld<T, VW>(w, vq + c * G * VW);
#pragma unroll
                    for (int k = 0; k < VW; ++k) {
                      const T x0 = u[k], y0 = w[k];
                      jac_rot(c0, s0, x0, y0, u[k], w[k]);
                    }
                    jac_st<T, VW>(vp + c * G * VW, u);
                    jac_st<T, VW>(vq + c * G * VW, w);
                  }
                }
              }
            }
            const T a1 = jac_reduce<T, TT>(na, G, gl);
            const T b1 = jac_reduce<T, TT>(nb, G, gl);
            if (rot && writer) {
              nrm[p] = a1;
              rt[p] = sqrt(a1);
              nrm[q] = b1;
              rt[q] = sqrt(b1);
            }
          }
          __syncthreads();
        }
        if (!__syncthreads_or(any)) break;
      }
      sw = sweep + 1;
    }
    // singular values, their order, the kept vectors (as OpTrunc::run)
    for (int j = warp; j < nc; j += nwarp) {
      T s2 = 0;
      for (int i = lane; i < len; i += 32) {
        const T y = Y[j * ldy + pos(i)];
        s2 += y * y;
      }
      s2 = warp_sum(s2);
      if (lane == 0) sig[j] = sqrt(s2);
    }
    __syncthreads();
    for (int j = tid; j < nc; j += nthr) {
      int rank = 0;
      const T sj = sig[j];
      for (int i = 0; i < nc; ++i) {
        const T si = sig[i];
        rank += sv_before(si, i, sj, j) ? 1 : 0;
      }
      order[rank] = j;
    }
    T zero2 = 0;
    if (tall) {
      T nf2 = 0;
      for (int j = 0; j < nc; ++j) nf2 += sig[j] * sig[j];
      zero2 = (eps * len) * (eps * len) * nf2;
    }
    __syncthreads();
    ST* U = op.Uk + (long long)s * op.uks;
    ST* o = op.out + (long long)s * op.outs;
    ST mx = 0;
    for (int idx = tid; idx < m * kk; idx += nthr) {
      const int q = idx / kk, j = order[idx - q * kk];
      T v;
      if (tall) {
        const T sg = sig[j];
        v = sg * sg > zero2 ? Y[j * ldy + pos(q)] / sg : (T)0;
      } else {
        v = V[j * ldv + pos(q)];
      }
      const ST u = (ST)v;
      U[idx] = u;
      o[idx] = u;
      const ST au = u < 0 ? -u : u;
      mx = au > mx ? au : mx;
    }
    mx = cta_max(mx, (ST*)red);
    double l = 0.0;
    if (mx > 0) {
      const ST inv = (ST)1 / mx;
      for (int idx = tid; idx < m * kk; idx += nthr) o[idx] *= inv;
      l = log((double)mx);
    }
    if (tid == 0) {
      op.lsv[(long long)s * op.lstride] += l;
      const double jf = (double)sw * 0.5 * nc * (nc - 1) * (12.0 * len + (tall ? 0.0 : 6.0 * m));
      atomicAdd(op.sweeps, (unsigned long long)sw);
      if (op.jflops) atomicAdd(op.jflops, jf);
    }
    __syncthreads();
  }
}

template <typename T, typename ST, int CH, int TT, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 2 : 1) kb_jac(OpTrunc<ST> op, int n, int G, int lg,
                                                                    int chY, int chV, T tol) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ T red[32];
  for (int s = blockIdx.x; s < n; s += gridDim.x) jac_matrix<T, ST, CH, TT>(op, s, dyn, red, G, lg, chY, chV, tol);
}

constexpr int JAC_SMEM_MAX = 220 * 1024;   // most dynamic shared memory of the kernels

// Launches the truncation of n chains; `threads`: 0 chooses the block, else its size.  Blocks
// of few warps that take TT pairs per lane group keep the scalar arithmetic and the barriers of
// a round cheap and are the choice when enough matrices are resident on an SM (at least eight
// warps); fewer matrices than that get one pair per lane group and more warps each, since a
// round's latency then bounds the sweep.
template <typename T, typename ST>
inline void jac_launch(const OpTrunc<ST>& op, int n, const JacShape& s, T tol, int sms, int threads,
                       cudaStream_t st) {
  const int npair = (op.nc + 1) / 2, gpw = 32 / s.G;
  int res = (int)((size_t)(227 * 1024) / (s.bytes + 1280));
  res = res < 1 ? 1 : (res > 32 ? 32 : res);
  const int per_sm = (n + sms - 1) / sms;
  const int mats = per_sm < res ? per_sm : res;
  int TT = s.chY <= 2 ? 4 : (s.chY <= 4 ? 2 : 1);
  while (TT > s.G) TT >>= 1;
  auto steps = [&](int tt) { return (npair + gpw * tt - 1) / (gpw * tt); };   // warp steps of a round
  if (s.G < 4 || mats * steps(TT) < 8) TT = 1;
  const int maxw = s.chY > 4 ? 16 : 8;
  int W = threads > 0 ? threads / 32 : (mats >= 16 ? 1 : (16 + mats - 1) / mats);
  const int need = steps(TT);
  W = W < need ? W : need;
  W = W < maxw ? W : maxw;
  W = W < 1 ? 1 : W;
  const int iters = (need + W - 1) / W;
  W = (need + iters - 1) / iters;   // no warp without work in the last step
  int grid = sms * res;
  grid = n < grid ? n : grid;
  const int nt = 32 * W;
  auto go = [&](auto kern) {
    smem_cap(kern, s.bytes, JAC_SMEM_MAX);
    kern<<<grid, nt, s.bytes, st>>>(op, n, s.G, s.lg, s.chY, s.chV, tol);
  };
  if (s.chY <= 1) {
    if (TT == 4) go(kb_jac<T, ST, 1, 4, 256>); else go(kb_jac<T, ST, 1, 1, 256>);
  } else if (s.chY <= 2) {
    if (TT == 4) go(kb_jac<T, ST, 2, 4, 256>); else go(kb_jac<T, ST, 2, 1, 256>);
  } else if (s.chY <= 4) {
    if (TT == 2) go(kb_jac<T, ST, 4, 2, 256>); else go(kb_jac<T, ST, 4, 1, 256>);
  } else if (s.chY <= 8) {
    go(kb_jac<T, ST, 8, 1, 512>);
  } else {
    go(kb_jac<T, ST, 0, 1, 512>);
  }
}

}  // namespace pv
#endif  // __CUDACC__
#endif
