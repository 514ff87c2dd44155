// Executor of chain programs (pv_prog.cuh).
#include <cuda_runtime.h>

#include "pv_batch.cuh"
#include "pv_direct.cuh"

namespace pv {
namespace {

template <typename T>
struct PgShared {
  PgOp op[2][PG_BLOCK];
  T red[32];
  T alpha[2], vn2[2], piv[2];
  T sc[4];               // val, num, den, val2
  int8_t i8[4];          // si, sj, valid, accepted
  int abort, stuck;
  uint64_t bar[2];
  uint32_t tslot;
  uint8_t S[256];
};

// Dynamic shared memory: PgShared, then the operations' work area.  Functions name the array itself
// (not a pointer to it), which keeps their accesses shared-memory instructions.
extern __shared__ __align__(16) unsigned char pg_smem[];
template <typename T>
PV_HD constexpr int pg_arena_off() {
  return (int)((sizeof(PgShared<T>) + 127) & ~(size_t)127);
}

// Tensor-core state of a block across operations.
struct PgTcState {
  uint32_t tmem, bar[2];
  uint32_t ph, outst;    // barrier phases; commits not yet waited for
  int next;              // stage of the next chunk
  bool dead;             // a wait ran out: skip the others
};

__device__ __forceinline__ char* pg_global(pgptr p, const PgArgs& a) { return a.gbase + (long long)(p - a.gint); }

__device__ __forceinline__ char* pg_dec(pgptr p, const PgArgs& a) {
  const unsigned tag = (unsigned)(p >> PG_TAG);
  return pg_global(tag ? (pgptr)a.slot[tag - 1] + (p & PG_OFF) : p, a);
}

// A scalar of the first thread: a shared one, or an element of an array.
template <typename T>
__device__ __forceinline__ T pg_get(pgptr p, long long off, const PgArgs& a, const PgShared<T>& sh) {
  const unsigned tag = (unsigned)(p >> PG_TAG);
  if (tag >= (unsigned)PG_SC) return sh.sc[tag - PG_SC];
  return ((const T*)pg_dec(p, a))[off];
}

template <typename T>
__device__ __forceinline__ const T* pg_at(const PgOpnd& o, int s, const PgArgs& a, const PgShared<T>& sh) {
  const T* b = (const T*)pg_global(o.base, a);
  if (o.mode == OP_BATCH) return b + (long long)s * o.stride;
  const int v = o.mode == OP_SITE_S ? (int)sh.S[o.site] : (int)sh.i8[o.sel];
  return b + (long long)v * o.stride;
}

// TM x TN outputs per thread (rows tm + i * nm, columns tn + j * nn, so that neighbouring threads
// read and write neighbouring columns), each one chain of fused multiply-adds in index order.
template <typename T, int TM, int TN>
__device__ __forceinline__ void pg_fma_tiles(const PgFma& f, const T* A, const T* B, T* C,
                                             const int* __restrict__ tab) {
  const int nm = (f.M + TM - 1) / TM, nn = (f.N + TN - 1) / TN, total = nm * nn;
  const int *ra = tab + f.rowA, *rc = tab + f.rowC, *cb = tab + f.colB, *cc = tab + f.colC;
  const int K0 = f.ks[0], K1 = f.ks[1], K2 = f.ks[2], a0 = f.ka[0], b0 = f.kb[0];
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int tm = t / nn, tn = t - tm * nn;
    const T *pa[TM], *pb[TN];
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i) pa[i] = A + __ldg(ra + min(tm + i * nm, f.M - 1));
#pragma unroll
    for (int j = 0; j < TN; ++j) pb[j] = B + __ldg(cb + min(tn + j * nn, f.N - 1));
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = 0;
    for (int k2 = 0; k2 < K2; ++k2)
      for (int k1 = 0; k1 < K1; ++k1) {
        int oa = k2 * f.ka[2] + k1 * f.ka[1], ob = k2 * f.kb[2] + k1 * f.kb[1];
#pragma unroll 4
        for (int k0 = 0; k0 < K0; ++k0) {
          T av[TM], bv[TN];
#pragma unroll
          for (int i = 0; i < TM; ++i) av[i] = pa[i][oa];
#pragma unroll
          for (int j = 0; j < TN; ++j) bv[j] = pb[j][ob];
#pragma unroll
          for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] += av[i] * bv[j];
          oa += a0;
          ob += b0;
        }
      }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int r = tm + i * nm;
      if (r < f.M) {
        T* pc = C + __ldg(rc + r);
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int c = tn + j * nn;
          if (c < f.N) pc[__ldg(cc + c)] = acc[i][j];
        }
      }
    }
  }
}

// ------------------------------------------------------------------ tensor-core contraction

// Operand chunk (rows row0 .. row0 + rows - 1 of `lim`, Kc = 4 << lq indices from k0 of K) into the
// canonical K-major layout without swizzle, rounded to TF32; the operand was written by this block,
// so its loads are plain ones.  Index tables `roff` (rows) and `koff`.
__device__ __forceinline__ void pg_gather(float* dst, float* dlo, const float* src, int mode, int rows, int row0,
                                          int lim, int lq, int k0, int K, const int* __restrict__ roff,
                                          const int* __restrict__ koff) {
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int qn = 1 << lq;
  if (mode == TC_VEC_K) {
    const int total = rows << lq;   // 16-byte pieces
    for (int e0 = tid; e0 < total; e0 += nthr * TC_UNROLL) {
      float4 v[TC_UNROLL];
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int e = e0 + u * nthr;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < total) {
          const int cm = e >> 3, g = cm >> lq, q = cm & (qn - 1);
          const int r = row0 + g * 8 + (e & 7), k = k0 + q * 4;
          if (r < lim && k < K) v[u] = *(const float4*)(src + __ldg(roff + r) + __ldg(koff + k));
        }
      }
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int e = e0 + u * nthr;
        if (e < total) tc_st4(dst, dlo, e, v[u]);
      }
    }
  } else if (mode == TC_VEC_T) {
    // blocks of 4 rows x 4 indices; lane j of a quad loads index 4 kq + j of four rows, and the
    // quad transposes the block
    int lr = 1;
    while ((4 << lr) < rows) ++lr;
    const int nrb = rows >> 2, total = 1 << (lr + lq);
    const int lane = tid & 31, j = lane & 3;
    for (int b0 = tid >> 2; b0 - (lane >> 2) < total; b0 += (nthr >> 2) * TC_UNROLL) {
      float4 v[TC_UNROLL];
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int blk = b0 + u * (nthr >> 2), rb = blk & ((1 << lr) - 1), kq = blk >> lr;
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int r = row0 + rb * 4, k = k0 + kq * 4 + j;
        if (blk < total && r < lim && k < K) v[u] = *(const float4*)(src + __ldg(roff + r) + __ldg(koff + k));
      }
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int blk = b0 + u * (nthr >> 2), rb = blk & ((1 << lr) - 1), kq = blk >> lr;
        float o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int c = (j - r) & 3;
          const float send = c == 0 ? v[u].x : (c == 1 ? v[u].y : (c == 2 ? v[u].z : v[u].w));
          const float got = __shfl_sync(0xffffffffu, send, (lane & ~3) | ((j + r) & 3));
          const int idx = (j + r) & 3;
          o0 = idx == 0 ? got : o0;
          o1 = idx == 1 ? got : o1;
          o2 = idx == 2 ? got : o2;
          o3 = idx == 3 ? got : o3;
        }
        if (blk < total && rb < nrb) {
          const int r = rb * 4 + j;
          tc_st4(dst, dlo, (((r >> 3) << lq) + kq) * 8 + (r & 7), make_float4(o0, o1, o2, o3));
        }
      }
    }
  } else {
    const int total = rows << (lq + 2);
    for (int e0 = tid; e0 < total; e0 += nthr * TC_UNROLL) {
      float v[TC_UNROLL];
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int e = e0 + u * nthr;
        v[u] = 0.f;
        if (e < total) {
          const int cm = e >> 5, j = e & 31, g = cm >> lq, q = cm & (qn - 1);
          const int r = row0 + g * 8 + (j >> 2), k = k0 + q * 4 + (j & 3);
          if (r < lim && k < K) v[u] = src[__ldg(roff + r) + __ldg(koff + k)];
        }
      }
#pragma unroll
      for (int u = 0; u < TC_UNROLL; ++u) {
        const int e = e0 + u * nthr;
        if (e < total) tc_st(dst, dlo, e, v[u]);
      }
    }
  }
}

// One chain's contraction C[m][n] = sum_k P[m][k] Q[n][k] on the tensor cores: the 128-row x TN
// tiles in turn, the chunks of Kc indices of a tile through two operand stages, a tile's
// accumulator read back while the next tile's first chunk is multiplied into the other one.
__device__ __forceinline__ void pg_tc(const PgTc& t, const float* P, const float* Q, float* C, float* arena,
                                      const int* __restrict__ tab, PgTcState& ts, int* sh_abort, int* sh_stuck) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwq = blockDim.x >> 7;
  const int Kc = t.Kc, TN = t.TN;
  const int sa = TC_ROWS * Kc, sb = t.sym ? 0 : TN * Kc, sst = (sa + sb) * (t.split ? 2 : 1);
  const int Kp = ((t.K + 7) >> 3) << 3;
  const uint32_t idesc = tc_idesc(TC_ROWS, TN);
  const int tilesM = (t.M + TC_ROWS - 1) / TC_ROWS, tilesN = (t.N + TN - 1) / TN;
  auto wait = [&](int st) {
    if (!((ts.outst >> st) & 1u)) return;
    ts.outst &= ~(1u << st);
    if (!ts.dead) {
      const uint32_t par = (ts.ph >> st) & 1u;
      if (!tc_wait(ts.bar[st], par)) {
        if (!tc_wait(ts.bar[st], par)) *sh_stuck = 1;
        *sh_abort = 1;
        ts.dead = true;
      }
    }
    ts.ph ^= 1u << st;
  };
  int tile = 0, pend = -1, pend_st = 0;
  auto epilogue = [&](int id) {   // tile id's accumulator to C
    wait(pend_st);
    __syncwarp();
    tc_fence_after();
    const int tm = id / tilesN, n0 = (id - tm * tilesN) * TN, acc = id & (t.nacc - 1);
    const int r = tm * TC_ROWS + (warp & 3) * 32 + lane;
    float* pc = C + (r < t.M ? __ldg(tab + t.rowC + r) : 0);
    const int* __restrict__ cc = tab + t.colC + n0;
    const int nlim = min(TN, t.N - n0);
    for (int c0 = (warp >> 2) * 16; c0 < nlim; c0 += nwq * 16) {
      uint32_t v[16];
      tc_ld16(ts.tmem + (uint32_t)(acc * TN) + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
      if (r < t.M) {
        if (t.vecC) {
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            if (c0 + j < nlim)
              *(float4*)(pc + __ldg(cc + c0 + j)) = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                                                __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < nlim) pc[__ldg(cc + c0 + j)] = __uint_as_float(v[j]);
        }
      }
    }
    tc_fence_before();
  };
  for (int tm = 0; tm < tilesM; ++tm) {
    const int m0 = tm * TC_ROWS;
    const int rowsA = min(TC_ROWS, ((t.M - m0 + 7) >> 3) << 3);
    for (int tn = 0; tn < tilesN; ++tn, ++tile) {
      const int n0 = tn * TN;
      const int rowsB = min(TN, ((t.N - n0 + 7) >> 3) << 3);
      const uint32_t acc = ts.tmem + (uint32_t)((tile & (t.nacc - 1)) * TN);
      for (int k0 = 0; k0 < t.K; k0 += Kc) {
        const int st = t.nst == 2 ? ts.next : 0;
        float* As = arena + st * sst;
        float* Bs = t.sym ? As : As + sa;
        float* Al = t.split ? As + sa + sb : nullptr;
        float* Bl = t.split ? (t.sym ? Al : Al + sa) : nullptr;
        wait(st);
        pg_gather(As, Al, P, t.modeP, rowsA, m0, t.M, t.lq, k0, t.K, tab + t.rowP, tab + t.kP);
        if (!t.sym) pg_gather(Bs, Bl, Q, t.modeQ, rowsB, n0, t.N, t.lq, k0, t.K, tab + t.colQ, tab + t.kQ);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        if (tid == 0) {
          tc_fence_after();
          const uint32_t a = tc_smem_addr(As), b = tc_smem_addr(Bs);
          const uint32_t al = t.split ? tc_smem_addr(Al) : 0, bl = t.split ? tc_smem_addr(Bl) : 0;
          const int nkb = (Kp - k0 < Kc ? Kp - k0 : Kc) >> 3;
          for (int kb = 0; kb < nkb; ++kb) tc_mma_k(t.split, acc, a, b, al, bl, Kc, kb, idesc, k0 > 0 || kb > 0);
          tc_commit(ts.bar[st]);
        }
        __syncwarp();
        ts.outst |= 1u << st;
        if (pend >= 0) {
          epilogue(pend);
          pend = -1;
        }
        pend_st = st;
        ts.next = st ^ 1;
      }
      pend = tile;
    }
  }
  epilogue(pend);
  wait(0);
  wait(1);
  __syncwarp();
}

// ------------------------------------------------------------------ factorisations

// lq_factor() with the partial sums of its 256-thread block (eight warps of the norm) for any
// block size: thread v of that block is thread v mod blockDim of this one.
template <typename T>
__device__ __forceinline__ void pg_lq(T* Lout, T* W, int m, int n, T* red) {
  const int K = m < n ? m : n, tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
  for (int i = tid; i < m * K; i += nthr) Lout[i] = 0;
  __syncthreads();
  for (int j = 0; j < K; ++j) {
    T* x = W + (long long)j * n;
    __syncthreads();
    for (int v = tid; v < 256; v += nthr) {
      T part = 0;
      for (int i = j + v; i < n; i += 256) part += x[i] * x[i];
      part = warp_sum(part);
      if (lane == 0) red[v >> 5] = part;
    }
    __syncthreads();
    T nrm2 = 0;
    for (int i = 0; i < 8; ++i) nrm2 += red[i];
    const T x0 = x[j];
    const T nrm = sqrt(nrm2);
    const T alpha = x0 >= 0 ? -nrm : nrm;
    const T v0 = x0 - alpha;
    const T ax0 = x0 < 0 ? -x0 : x0;
    const T vn2 = (T)2 * (nrm2 + nrm * ax0);
    __syncthreads();
    if (tid == 0) {
      x[j] = v0;
      Lout[(long long)j * K + j] = alpha;
    }
    __syncthreads();
    const bool active = nrm2 > 0 && vn2 > 0;
    for (int jj = j + 1 + (tid >> 5); jj < m; jj += nthr >> 5) {
      T* a = W + (long long)jj * n;
      if (active) {
        T p = 0;
        for (int i = j + lane; i < n; i += 32) p += x[i] * a[i];
        p = warp_sum(p);
        const T g = (T)2 * p / vn2;
        for (int i = j + lane; i < n; i += 32) a[i] -= g * x[i];
      }
      __syncwarp();
      if (lane == 0) Lout[(long long)jj * K + j] = a[j];
    }
  }
  __syncthreads();
}

// ------------------------------------------------------------------ the executor

template <typename T>
__device__ __forceinline__ OpTrunc<T> pg_optrunc(const PgOp& o, const PgArgs& a, T jtol, int max_sweeps,
                                                 unsigned long long* sweeps) {
  OpTrunc<T> t;
  t.Y = (const T*)pg_global(o.g.p[0], a);
  t.ys = o.g.l[0];
  t.tall = o.g.i[3] != 0;
  t.nc = o.g.i[0];
  t.len = o.g.i[1];
  t.m = o.g.i[2];
  t.kk = o.g.i[4];
  t.Uk = (T*)pg_global(o.g.p[1], a);
  t.uks = o.g.l[1];
  t.out = (T*)pg_global(o.g.p[2], a);
  t.outs = o.g.l[2];
  t.lsv = (double*)pg_global(o.g.p[3], a);
  t.lstride = o.g.i[5];
  t.jtol = jtol;
  t.max_sweeps = max_sweeps;
  t.sweeps = sweeps;
  t.jflops = a.jflops;
  return t;
}

// Operations of the first thread (PG_DOT: the first warp).
template <typename T>
__device__ __noinline__ void pg_op0(int buf, int q, int s, const PgArgs& a) {
  PgShared<T>& sh = *(PgShared<T>*)pg_smem;
  const PgOp& o = sh.op[buf][q];
  const int tid = threadIdx.x;
  if (o.kind == PG_DOT) {
    const T* x = (const T*)pg_dec(o.g.p[0], a) + (long long)s * o.g.l[0];
    const T* y = (const T*)pg_dec(o.g.p[1], a) + (long long)s * o.g.l[1];
    const int len = (int)o.g.l[2];
    T acc = 0;
    int k = tid;
    constexpr int U = sizeof(T) == 4 ? 16 : 8;
    for (; k + 32 * (U - 1) < len; k += 32 * U) {
      T u[U], v[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        u[i] = x[k + 32 * i];
        v[i] = y[k + 32 * i];
      }
#pragma unroll
      for (int i = 0; i < U; ++i) acc += u[i] * v[i];
    }
    for (; k < len; k += 32) acc += x[k] * y[k];
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    if (tid == 0) sh.sc[(unsigned)(o.g.p[2] >> PG_TAG) - PG_SC] = acc;
    return;
  }
  if (tid != 0) return;
  switch (o.kind) {
    case PG_SET: ((T*)pg_dec(o.g.p[0], a))[(long long)s * o.g.l[0] + o.g.l[1]] = (T)o.g.d; break;
    case PG_SETD: ((double*)pg_dec(o.g.p[0], a))[(long long)s * o.g.l[0] + o.g.l[1]] = o.g.d; break;
    case PG_COPYD: {
      double* x = (double*)pg_dec(o.g.p[0], a) + (long long)s * o.g.l[0];
      x[o.g.i[0]] = x[o.g.i[1]];
      break;
    }
    case PG_SETI8: sh.i8[o.g.i[0]] = (int8_t)o.g.i[1]; break;
    case PG_SEL: {
      ElemSel f{sh.S, 0, o.g.i[0], o.g.i[1], o.g.i[2], &sh.i8[0], &sh.i8[1], &sh.i8[2]};
      f(0);
      break;
    }
    case PG_RATIO:
      if (sh.i8[2]) {
        double* e = (double*)pg_dec(o.g.p[2], a) + s;
        *e += o.g.d * (double)pg_get(o.g.p[0], s, a, sh) / (double)pg_get(o.g.p[1], (long long)s * o.g.l[0], a, sh);
      }
      break;
    case PG_ACCEPT: {
      sh.i8[3] = 0;
      if (!sh.i8[2]) break;
      const int i = o.g.i[0], j = o.g.i[1];
      T* num = &sh.sc[(unsigned)(o.g.p[0] >> PG_TAG) - PG_SC];
      T* den = &sh.sc[(unsigned)(o.g.p[1] >> PG_TAG) - PG_SC];
      const double u = philox_uniform(a.seed, (uint32_t)(a.chain0 + s), *a.sweep_dev, (uint32_t)o.g.i[2], TAG_MC);
      const double ratio = (double)*num / (double)*den;
      const double q = a.p == 2 ? ratio * ratio : (ratio < 0 ? -ratio : ratio);
      ((int*)a.slot[PS_PROP])[s] += 1;
      if (u < q) {
        ((int*)a.slot[PS_ACC])[s] += 1;
        sh.i8[3] = 1;
        uint8_t* S = (uint8_t*)a.slot[PS_S] + (long long)s * a.N;
        S[i] = sh.S[i] = (uint8_t)sh.i8[0];
        if (j >= 0) S[j] = sh.S[j] = (uint8_t)sh.i8[1];
        *den = *num;
      }
      break;
    }
    case PG_AMP: {
      ElemAmp<T> f{(const T*)pg_dec(o.g.p[0], a), o.g.l[0], (const double*)pg_dec(o.g.p[1], a), o.g.i[0],
                   (double*)a.slot[PS_LA], (int8_t*)a.slot[PS_SG]};
      f(s);
      break;
    }
    case PG_DRAW: {
      // the chain's uniforms and configuration rows, its candidates in shared memory
      uint8_t* S = (uint8_t*)a.slot[PS_S] + (long long)s * a.N;
      ElemDraw<T> f{S, 0, o.g.i[0], &sh.sc[0], &sh.sc[1], &sh.sc[2], &sh.sc[3], a.b_d, a.expo,
                    (const double*)a.slot[PS_U] + (long long)s * a.N, (double*)a.slot[PS_LOGQ] + s};
      f(0);
      sh.S[o.g.i[0]] = S[o.g.i[0]];
      break;
    }
  }
}

// One function per kind of operation, not inlined: the kernel's own loop stays small and an
// operation's code contiguous, which the instruction cache needs with several blocks at
// different operations (inlining everything made an 8x8 evaluation 30 % slower).
template <typename T>
__device__ __noinline__ void pg_do_fma(int buf, int q, int s, const PgArgs& a, const int* __restrict__ tab) {
  const PgShared<T>& sh = *(const PgShared<T>*)pg_smem;
  const PgOp& o = sh.op[buf][q];
  const T *A = pg_at(o.e.A, s, a, sh), *B = pg_at(o.e.B, s, a, sh);
  T* C = (T*)pg_global(o.e.out, a) + (long long)s * o.e.os;
  const PgFma f = o.e.f;
  if (f.tm == 4 && f.tn == 4) pg_fma_tiles<T, 4, 4>(f, A, B, C, tab);
  else if (f.tm == 2) pg_fma_tiles<T, 2, 2>(f, A, B, C, tab);
  else if (f.tm == 4) pg_fma_tiles<T, 4, 1>(f, A, B, C, tab);
  else if (f.tn == 4) pg_fma_tiles<T, 1, 4>(f, A, B, C, tab);
  else pg_fma_tiles<T, 1, 1>(f, A, B, C, tab);
}

__device__ __noinline__ void pg_do_tc(int buf, int q, int s, const PgArgs& a, const int* __restrict__ tab,
                                      PgTcState& ts) {
  PgShared<float>& sh = *(PgShared<float>*)pg_smem;
  const PgOp& o = sh.op[buf][q];
  const float *x = pg_at(o.e.A, s, a, sh), *y = pg_at(o.e.B, s, a, sh);
  const PgTc t = o.e.t;
  PgTcState l = ts;
  pg_tc(t, t.swap ? y : x, t.swap ? x : y, (float*)pg_global(o.e.out, a) + (long long)s * o.e.os,
        (float*)(pg_smem + pg_arena_off<float>()), tab, l, &sh.abort, &sh.stuck);
  ts = l;
}

template <typename T>
__device__ __noinline__ void pg_do_factor(int buf, int q, int s, const PgArgs& a) {
  PgShared<T>& sh = *(PgShared<T>*)pg_smem;
  const PgOp& o = sh.op[buf][q];
  T* arena = (T*)(pg_smem + pg_arena_off<T>());
  T *p0 = (T*)pg_global(o.g.p[0], a), *p1 = (T*)pg_global(o.g.p[1], a);
  const int m = o.g.i[0], nn = o.g.i[1], nthr = blockDim.x;
  if (o.kind == PG_CHOL) {
    const OpChol<T> f{p0, o.g.l[0], p1, o.g.l[1], m};
    if (m > 64 || nthr < 128) chol_matrix(f, s, arena, sh.red, sh.piv);
    else if (nthr == 128) chol64<T, 8>(f, s, arena, sh.red);
    else if (nthr == 256) chol64<T, 16>(f, s, arena, sh.red);
    else chol64<T, 32>(f, s, arena, sh.red);
  } else if (o.kind == PG_LQ2) {
    const OpLq<T> f{p0, o.g.l[0], p1, o.g.l[1], m, nn, nullptr};
    lq2_matrix(f, s, arena, sh.alpha, sh.vn2, o.g.i[2], o.g.i[3]);
  } else {
    T* W = p1 + (long long)s * o.g.l[1];
    T* Lo = p0 + (long long)s * o.g.l[0];
    if (o.g.i[2]) {   // the matrix fits the shared work area
      for (int i = threadIdx.x; i < m * nn; i += nthr) arena[i] = W[i];
      __syncthreads();
      pg_lq<T>(Lo, arena, m, nn, sh.red);
    } else {
      pg_lq<T>(Lo, W, m, nn, sh.red);
    }
  }
}

struct PgJac {
  int buf, q, s, max_sweeps;
  unsigned long long* sweeps;
};
template <typename T, typename W, int CH, int TT>
__device__ __noinline__ void pg_jac(const PgJac j, const PgArgs& a, T jtol, W tol) {
  PgShared<T>& sh = *(PgShared<T>*)pg_smem;
  const PgOp& o = sh.op[j.buf][j.q];
  unsigned char* arena = pg_smem + pg_arena_off<T>();
  jac_matrix<W, T, CH, TT>(pg_optrunc<T>(o, a, jtol, j.max_sweeps, j.sweeps), j.s, arena + 256, (W*)arena, o.g.i[6],
                           o.g.i[7], o.g.i[8], o.g.i[9], tol);
}

// The variant of a truncation: columns in registers where they fit, and several pairs per lane
// group as long as every warp has work (fewer scalar instructions).
template <typename T, typename W>
__device__ __forceinline__ void pg_do_trunc(const PgJac& j, const PgArgs& a, T jtol, W tol) {
  const PgOp& o = ((PgShared<T>*)pg_smem)->op[j.buf][j.q];
  const int G = o.g.i[6], chY = o.g.i[8];
  const int tt = ((o.g.i[0] + 1) >> 1) / ((32 >> o.g.i[7]) * (int)(blockDim.x >> 5));
  if (chY <= 1) {
    if (tt >= 4 && G >= 4) pg_jac<T, W, 1, 4>(j, a, jtol, tol);
    else pg_jac<T, W, 1, 1>(j, a, jtol, tol);
  } else if (chY <= 2) {
    if (tt >= 2 && G >= 2) pg_jac<T, W, 2, 2>(j, a, jtol, tol);
    else pg_jac<T, W, 2, 1>(j, a, jtol, tol);
  } else if (chY <= 4) {
    if ((tt >= 2 || sizeof(W) == 8) && G >= 2) pg_jac<T, W, 4, 2>(j, a, jtol, tol);
    else pg_jac<T, W, 4, 1>(j, a, jtol, tol);
  } else {
    pg_jac<T, W, 0, 1>(j, a, jtol, tol);
  }
}

template <typename T>
__global__ void __launch_bounds__(512, 1) kb_prog(const PgOp* __restrict__ ops, int nblk, const int* __restrict__ tab,
                                                  const __grid_constant__ PgArgs a, int tmem_cols, T jtol, double jtol64, int max_sweeps,
                                                  unsigned long long* sweeps, int* err) {
  PgShared<T>& sh = *(PgShared<T>*)pg_smem;
  const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5;
  PgTcState ts;
  ts.tmem = 0;
  ts.ph = ts.outst = 0;
  ts.next = 0;
  ts.dead = false;
  if (tid == 0) sh.abort = sh.stuck = 0;
  if constexpr (sizeof(T) == 4) {
    ts.bar[0] = tc_smem_addr(&sh.bar[0]);
    ts.bar[1] = tc_smem_addr(&sh.bar[1]);
    // allocated even where no operation uses it: a block of this kernel that neither allocates nor
    // gives up the right to allocate keeps further blocks off its SM (measured: one block per SM)
    if (warp == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       tc_smem_addr(&sh.tslot)),
                   "r"((uint32_t)tmem_cols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(ts.bar[0]), "r"(1) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(ts.bar[1]), "r"(1) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    ts.tmem = sh.tslot;
  }
  constexpr int REC = (int)(sizeof(PgOp) * PG_BLOCK / 16);   // 16-byte pieces of a block of records
  auto fetch = [&](int b) {
    const char* src = (const char*)(ops + (long long)b * PG_BLOCK);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sh.op[b & 1][0]);
    for (int i = tid; i < REC; i += nthr)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 16), "l"(src + i * 16) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  bool stop = false;
  int skip = 0;   // operations still to leave out (the same in every thread)
  for (int s = blockIdx.x; s < a.n && !stop; s += gridDim.x) {
    const uint8_t* S = (const uint8_t*)a.slot[PS_S] + (long long)s * a.N;
    for (int i = tid; i < a.N; i += nthr) sh.S[i] = S[i];
    fetch(0);
    for (int b = 0; b < nblk && !stop; ++b) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      if (b + 1 < nblk) fetch(b + 1);
      for (int q = 0; q < PG_BLOCK; ++q) {
        const PgOp& o = sh.op[b & 1][q];
        if (o.kind < 0) break;
        if (skip > 0) {
          --skip;
          continue;
        }
        if (o.kind >= PG_T0) {
          if (warp == 0) pg_op0<T>(b & 1, q, s, a);
        } else {
          switch (o.kind) {
            case PG_SKIP: skip = sh.i8[2] ? 0 : o.g.i[0]; break;
            case PG_FMA: pg_do_fma<T>(b & 1, q, s, a, tab); break;
            case PG_TC:
              if constexpr (sizeof(T) == 4) pg_do_tc(b & 1, q, s, a, tab, ts);
              break;
            case PG_EIN: {
              const MSpec& m = *(const MSpec*)(tab + o.e.mspec);
              const T *x = pg_at(o.e.A, s, a, sh), *y = pg_at(o.e.B, s, a, sh);
              T* z = (T*)pg_global(o.e.out, a) + (long long)s * o.e.os;
              for (int i = tid; i < m.total; i += nthr) ein_one(m, z, x, y, i);
              break;
            }
            case PG_COPY: {   // masked by a shared selection (i[0] >= 0)
              if (o.g.i[0] >= 0 && !sh.i8[o.g.i[0]]) break;
              T* d = (T*)pg_global(o.g.p[0], a) + (long long)s * o.g.l[0];
              const T* c = (const T*)pg_global(o.g.p[1], a) + (long long)s * o.g.l[1];
              for (int i = tid; i < (int)o.g.l[2]; i += nthr) d[i] = c[i];
              break;
            }
            case PG_NORM: {
              const double l = normalize_maxabs((T*)pg_global(o.g.p[0], a) + (long long)s * o.g.l[0], o.g.l[1], sh.red);
              if (tid == 0) ((double*)pg_global(o.g.p[1], a))[(long long)s * o.g.i[0]] += l;
              break;
            }
            case PG_LQ:
            case PG_LQ2:
            case PG_CHOL: pg_do_factor<T>(b & 1, q, s, a); break;
            case PG_TRUNC: pg_do_trunc<T, T>(PgJac{b & 1, q, s, max_sweeps, sweeps}, a, jtol, jtol); break;
            case PG_TRUNC64:
              if constexpr (sizeof(T) == 4) pg_do_trunc<T, double>(PgJac{b & 1, q, s, max_sweeps, sweeps}, a, jtol, jtol64);
              break;
            case PG_O: {
              T* O = (T*)pg_global((pgptr)a.slot[PS_O], a) + (long long)s * o.g.l[0] + o.g.l[1];
              const T* e = (const T*)pg_global(o.g.p[0], a) + (long long)s * o.g.l[2];
              const T v = ((const T*)pg_global(o.g.p[1], a))[(long long)s * o.g.l[3]];
              for (int i = tid; i < (int)o.g.l[4]; i += nthr) {
                T x = e[i] / v;
                if constexpr (sizeof(T) == 4) {
                  // the float64 quotient rounded to float32 is the float32 quotient except where
                  // that is subnormal
                  const T ax = x < 0 ? -x : x;
                  if (!(ax >= 2.4e-38f)) x = (T)((double)e[i] / (double)v);
                }
                O[i] = x;
              }
              break;
            }
            case PG_DIAG: {
              // system energy on the first thread, ancilla energy on the second
              if (tid < 2) {
                const int sh_bit = tid == 0 ? 1 : 0;
                const int *bi = (const int*)pg_global(o.g.p[0], a), *bj = (const int*)pg_global(o.g.p[1], a);
                const double* bJ = (const double*)pg_global(o.g.p[2], a);
                double e = 0;
#pragma unroll 4
                for (int k = 0; k < o.g.i[0]; ++k) {
                  const int x = sh.S[__ldg(bi + k)] >> sh_bit, y = sh.S[__ldg(bj + k)] >> sh_bit;
                  const double z = ((x & 1) ? -0.5 : 0.5) * ((y & 1) ? -0.5 : 0.5);
                  e += __ldg(bJ + k) * z;
                }
                ((double*)a.slot[tid == 0 ? PS_ES : PS_EA])[s] = e;
              }
              break;
            }
          }
        }
        if (o.bar) __syncthreads();
      }
      if constexpr (sizeof(T) == 4) stop = *(volatile int*)&sh.abort != 0;
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if constexpr (sizeof(T) == 4) {
    __syncthreads();
    if (warp == 0) {
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ts.tmem), "r"((uint32_t)tmem_cols)
                   : "memory");
    }
    if (tid == 0 && sh.abort) atomicOr(err, sh.stuck ? 3 : 1);
  }
}

}  // namespace

template <typename T>
void pg_launch(const PgProgram& p, const PgArgs& a, T jtol, double jtol64, int max_sweeps, unsigned long long* sweeps,
               int* err, int sms, cudaStream_t st) {
  const int grid = a.n < sms * p.per_sm ? a.n : sms * p.per_sm;
  const size_t smem = pg_arena_off<T>() + p.arena;
  smem_cap(kb_prog<T>, smem, (int)(PG_SMEM - 1024));
  kb_prog<T><<<grid, p.threads, smem, st>>>(p.d_ops, (p.nops + PG_BLOCK - 1) / PG_BLOCK, p.d_tab, a, p.tmem_cols,
                                               jtol, jtol64, max_sweeps, sweeps, err);
}

template void pg_launch<float>(const PgProgram&, const PgArgs&, float, double, int, unsigned long long*, int*, int,
                               cudaStream_t);
template void pg_launch<double>(const PgProgram&, const PgArgs&, double, double, int, unsigned long long*, int*, int,
                                cudaStream_t);

}  // namespace pv
