// Tensor-core contraction of the batched engine: the strided GEMM per chain of pv_tc.cuh
// (C[m][n] = sum_k P[m][k] Q[n][k], multi-indices of arbitrary strides, TF32 or split operands,
// FP32 accumulation), for every chain or for a list of them.
//
// A CTA of four warps owns one 128-row x TN tile and walks the chains assigned to it.  A thread
// loads its part of a contraction chunk of both operands into registers, rounds it and stores it
// to the one operand stage; one thread issues the chunk's MMAs; the loads of the next chunk (or
// chain) are then in flight while the MMAs run and the accumulator is read and stored.  Every wait
// on the mbarrier is bounded: when it runs out the kernel raises `err`, waits once more, frees its
// tensor memory and returns (err bit 2 when that second wait ran out too).
//
// What bounds it: the operands and results of most contractions are 4 to 64 KB a chain, so the
// instructions that gather an element and the latency of a chain's round trip cost more than its
// bytes (8x8 D=4 chi=16, 8192 chains: 2.5 to 3 TB/s of the operands' and results') or its MMAs.  Hence
//  - every lane moves 16 bytes at a time, contiguous rows included (4 x 4 blocks transposed in
//    registers; the former kernels copied those 4 bytes at a time), index arithmetic is shifts
//    (chunks are powers of two) and offsets come from tables;
//  - one stage and one accumulator: with chunks this small more CTAs on an SM (four to five)
//    overlap a round trip better than a second stage in each.
// Measured against the kernels this one replaced (a register-staged one and a cp.async ring of 4-
// and 16-byte copies): 8x8 D=4 chi=16 step of 8192 chains 864 -> 668 ms, 10x10 D=6 chi=36 evaluation
// of 192 chains 1330 -> 1176, 6x6 direct draw of 8192 chains 91 -> 77.  The operand forms compiled
// apart then took the 1555 contractions of an 8x8 evaluation of 2048 chains from 61 to 52 ms, and
// merged contiguous dims with pairs the 10x10 evaluation from 940 to 845 ms.
#ifndef PV_GEMM_CUH
#define PV_GEMM_CUH
#include <cstdint>

namespace pv {

// Floats of an operand chunk: groups of 8 rows hold qn core matrices (8 rows x 16 bytes, 128
// contiguous bytes each) and 16 bytes of padding, so that the rows a warp stores at once fall on
// different banks also where its lanes hold whole groups of four rows.
PV_HD int tc_group(int Kc) { return Kc * 8 + 4; }
inline size_t tc_smem_bytes(const TcSpec& t) {
  const size_t stage = (size_t)(TC_ROWS + (t.sym ? 0 : t.TN)) / 8 * tc_group(t.Kc) * sizeof(float);
  return stage * (t.split ? 2 : 1) + (size_t)(2 * TC_ROWS + 2 * t.TN + 2 * t.K) * sizeof(int);
}

// Contraction chunk: the 16-byte vectors of one chunk are held in registers (NA of P and NB of Q
// per thread), so chunks of 32 are taken only with at most 64 columns.
inline void tc_shape(TcSpec& t, int kc_max) {
  int kc = t.K <= 8 ? 8 : (t.K > 16 && (t.TN <= 64 || t.sym) ? 32 : 16);
  while (kc > kc_max && kc > 8) kc >>= 1;
  t.Kc = kc;
}

#if defined(__CUDACC__)

// One chunk of an operand (`rows` rows, contraction indices k0..k0+Kc) to registers.  lq: log2 of
// the quads of contraction indices (Kc / 4).  Every lane's vector is four contraction indices of
// a row or, in a 4 x 4 block of an operand that is contiguous in its rows (TC_VEC_T), four rows
// at four indices: transposed by naming, when it is stored.
template <int mode, int NU>
__device__ __forceinline__ void tc_load(float4 (&r)[NU], const float* __restrict__ src, bool kfast, bool pair,
                                         int rows, int lq, int k0, int K, const int* roff, const int* koff,
                                         int tid) {
  const int qn = 1 << lq;
  if constexpr (mode == TC_VEC_K) {
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int e = tid + u * TC_THREADS;
      const int rr = (e & 7) | ((e >> (3 + lq)) << 3), k = k0 + (((e >> 3) & (qn - 1)) << 2);
      r[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (rr < rows && k < K) {
        const int ro = roff[rr];
        if (ro >= 0) r[u] = *(const float4*)(src + ro + koff[k]);
      }
    }
  } else if constexpr (mode == TC_VEC_T) {
#pragma unroll
    for (int b = 0; b < NU / 4; ++b) {
      const int e = tid + b * TC_THREADS;
      const int rr = ((e & 7) | ((e >> (3 + lq)) << 3)) << 2, kb = k0 + (((e >> 3) & (qn - 1)) << 2);
      const int ro = rr < rows ? roff[rr] : -1;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        r[4 * b + i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (ro >= 0 && kb + i < K) r[4 * b + i] = *(const float4*)(src + ro + koff[kb + i]);
      }
    }
  } else {
    // single elements, neighbouring lanes along the operand's contiguous side
    const int sh = kfast ? 3 : 4;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int e = tid + u * TC_THREADS;
      const int rr = (e & ((1 << sh) - 1)) | ((e >> (sh + lq)) << sh), kb = k0 + (((e >> sh) & (qn - 1)) << 2);
      const int ro = rr < rows ? roff[rr] : -1;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (ro >= 0) {
        if (pair) {
#pragma unroll
          for (int i = 0; i < 4; i += 2)
            if (kb + i < K) {
              const float2 w = *(const float2*)(src + ro + koff[kb + i]);
              v[i] = w.x;
              v[i + 1] = w.y;
            }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (kb + i < K) v[i] = src[ro + koff[kb + i]];
        }
      }
      r[u] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// Rounds the registers of tc_load to TF32 and stores them in the K-major layout without swizzle
// (and the rounding of the remainders to `lo` where it is given).
template <int mode, int NU>
__device__ __forceinline__ void tc_store(const float4 (&r)[NU], float* hi, float* lo, bool kfast, int rows, int lq,
                                         int tid) {
  const int qn = 1 << lq, gs = (qn << 5) + 4;
  auto put = [&](int rr, int q, float4 v) {
    const int e = (rr >> 3) * gs + (q << 5) + ((rr & 7) << 2);
    const float4 h = tc_round4(v);
    *(float4*)(hi + e) = h;
    if (lo) *(float4*)(lo + e) = tc_round4(make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w));
  };
  if constexpr (mode == TC_VEC_T) {
#pragma unroll
    for (int b = 0; b < NU / 4; ++b) {
      const int e = tid + b * TC_THREADS;
      const int rr = ((e & 7) | ((e >> (3 + lq)) << 3)) << 2, q = (e >> 3) & (qn - 1);
      if (rr < rows) {
        put(rr, q, make_float4(r[4 * b].x, r[4 * b + 1].x, r[4 * b + 2].x, r[4 * b + 3].x));
        put(rr + 1, q, make_float4(r[4 * b].y, r[4 * b + 1].y, r[4 * b + 2].y, r[4 * b + 3].y));
        put(rr + 2, q, make_float4(r[4 * b].z, r[4 * b + 1].z, r[4 * b + 2].z, r[4 * b + 3].z));
        put(rr + 3, q, make_float4(r[4 * b].w, r[4 * b + 1].w, r[4 * b + 2].w, r[4 * b + 3].w));
      }
    }
  } else {
    const int sh = mode == TC_VEC_K || kfast ? 3 : 4;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const int e = tid + u * TC_THREADS;
      const int rr = (e & ((1 << sh) - 1)) | ((e >> (sh + lq)) << sh);
      if (rr < rows) put(rr, (e >> sh) & (qn - 1), r[u]);
    }
  }
}

// MP, MQ: the operands' gather forms (compiled apart: an item is some 350 instructions, and the
// instruction cache pays for every path that lies between them).
template <int NA, int NB, int MINB, int MP, int MQ>
__global__ void __launch_bounds__(TC_THREADS, MINB) kb_gemm_tc(TcSpec t, float* C, long long cs, Operand<float> P,
                                                               Operand<float> Q, int n, int tilesN, int* err,
                                                               ChainList cl) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tslot;
  __shared__ int abort_flag;
  __shared__ int stuck;   // a grace wait ran out too: an MMA may still be writing tensor memory
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tm = blockIdx.x / tilesN, tn = blockIdx.x - tm * tilesN;
  const int TN = t.TN, Kc = t.Kc, lq = Kc == 8 ? 1 : (Kc == 16 ? 2 : 3);
  const int m0 = tm * TC_ROWS, n0 = tn * TN, gs = tc_group(Kc);
  const int sa = TC_ROWS / 8 * gs, sb = t.sym ? 0 : TN / 8 * gs;
  const int rowsA = min(TC_ROWS, ((t.M - m0 + 7) >> 3) << 3);
  const int rowsB = min(TN, ((t.N - n0 + 7) >> 3) << 3);
  const bool kfP = t.nk > 0 && t.kP[t.nk - 1] == 1, kfQ = t.nk > 0 && t.kQ[t.nk - 1] == 1;
  float* As = (float*)dyn;
  float* Bs = t.sym ? As : As + sa;
  float* Al = t.split ? As + sa + sb : nullptr;
  float* Bl = t.split ? (t.sym ? Al : Al + sa) : nullptr;
  int* rowP = (int*)(As + (long long)(sa + sb) * (t.split ? 2 : 1));
  int* rowC = rowP + TC_ROWS;
  int* colQ = rowC + TC_ROWS;
  int* colC = colQ + TN;
  int* kPo = colC + TN;
  int* kQo = kPo + t.K;
  for (int i = tid; i < TC_ROWS; i += TC_THREADS) {
    const int m = m0 + i;
    if (m < t.M) gemm_offsets(m, t.nr, t.rs, t.rP, t.rC, rowP[i], rowC[i]);
    else rowP[i] = rowC[i] = -1;
  }
  for (int i = tid; i < TN; i += TC_THREADS) {
    const int c = n0 + i;
    if (c < t.N) gemm_offsets(c, t.nc, t.cs, t.cQ, t.cC, colQ[i], colC[i]);
    else colQ[i] = colC[i] = -1;
  }
  for (int k = tid; k < t.K; k += TC_THREADS) gemm_offsets(k, t.nk, t.ks, t.kP, t.kQ, kPo[k], kQo[k]);
  const uint32_t ncols = (uint32_t)tc_cols(TN), bar = tc_smem_addr(&mbar);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_addr(&tslot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    abort_flag = 0;
    stuck = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(1) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_go();
  pdl_wait();
  const uint32_t tmem = tslot, idesc = tc_idesc(TC_ROWS, TN);
  const uint32_t a = tc_smem_addr(As), b = tc_smem_addr(Bs);
  const uint32_t al = t.split ? tc_smem_addr(Al) : 0, bl = t.split ? tc_smem_addr(Bl) : 0;
  const int Kp = ((t.K + 7) >> 3) << 3, gy = gridDim.y;
  n = cl.count(n);
  uint32_t ph = 0u;
  float4 ra[NA], rb[NB];
  auto load = [&](const float* p, const float* q, int k0) {
    tc_load<MP>(ra, p, kfP, t.pairP, rowsA, lq, k0, t.K, rowP, kPo, tid);
    if (!t.sym) tc_load<MQ>(rb, q, kfQ, t.pairQ, rowsB, lq, k0, t.K, colQ, kQo, tid);
  };
  auto desc = [&](uint32_t base, int kb) { return tc_desc(base + kb * 256, 128, (uint32_t)gs * 4u); };
  const float *pn = nullptr, *qn = nullptr;   // operands of the next chain: their addresses are formed
                                              // a chain ahead (a site's slice depends on a load)
  int s = 0, sn = 0;
  if ((int)blockIdx.y < n) {
    s = cl.chain(blockIdx.y);
    load(P.at(s), Q.at(s), 0);
  }
  const float *pc = nullptr, *qc = nullptr;
  if ((int)blockIdx.y < n) {
    pc = P.at(s);
    qc = Q.at(s);
  }
  if ((int)blockIdx.y + gy < n) {
    sn = cl.chain(blockIdx.y + gy);
    pn = P.at(sn);
    qn = Q.at(sn);
  }
  bool stop = false;
  for (int k = blockIdx.y; k < n && !stop; k += gy) {
    bool good = true;
    for (int k0 = 0; k0 < t.K; k0 += Kc) {
      tc_store<MP>(ra, As, Al, kfP, rowsA, lq, tid);
      if (!t.sym) tc_store<MQ>(rb, Bs, Bl, kfQ, rowsB, lq, tid);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncthreads();
      if (abort_flag) {
        stop = true;
        break;
      }
      if (tid == 0 && !t.no_mma) {
        tc_fence_after();
        const int nkb = (Kp - k0 < Kc ? Kp - k0 : Kc) >> 3;
        for (int kb = 0; kb < nkb; ++kb) {
          tc_mma(tmem, desc(a, kb), desc(b, kb), idesc, k0 > 0 || kb > 0 ? 1 : 0);
          if (t.split) {
            tc_mma(tmem, desc(a, kb), desc(bl, kb), idesc, 1);
            tc_mma(tmem, desc(al, kb), desc(b, kb), idesc, 1);
          }
        }
        tc_commit(bar);
      }
      // the next chunk's operands, in flight during the MMAs and the epilogue
      if (k0 + Kc < t.K) {
        load(pc, qc, k0 + Kc);
      } else if (k + gy < n) {
        pc = pn;
        qc = qn;
        load(pc, qc, 0);
      }
      bool ok = tc_wait(bar, ph);
      if (!ok) {
        if (!tc_wait(bar, ph)) stuck = 1;
        abort_flag = 1;
      }
      ph ^= 1u;
      good = good && ok;
    }
    if (stop) break;
    if (__all_sync(0xffffffffu, good)) {   // tcgen05.ld is warp-collective
      tc_fence_after();
      tc_epilogue(t, tmem, C + (long long)s * cs, rowC, colC, warp, lane);
    }
    s = sn;
    if (k + 2 * gy < n) {
      sn = cl.chain(k + 2 * gy);
      pn = P.at(sn);
      qn = Q.at(sn);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
  }
  if (tid == 0 && abort_flag) atomicOr(err, stuck ? 3 : 1);
}

// f(kernel, resident CTAs per SM that its registers allow) for the variant of a spec.
constexpr int TC_SMEM_MAX = 200 * 1024;   // most dynamic shared memory of the kernels
template <int NA, int NB, int MINB, typename F>
void tc_modes(int mp, int mq, F&& f) {
  auto q = [&](auto MP) {
    if (mq == TC_VEC_K) f(kb_gemm_tc<NA, NB, MINB, MP.value, TC_VEC_K>, MINB);
    else if (mq == TC_VEC_T) f(kb_gemm_tc<NA, NB, MINB, MP.value, TC_VEC_T>, MINB);
    else f(kb_gemm_tc<NA, NB, MINB, MP.value, TC_SCALAR>, MINB);
  };
  if (mp == TC_VEC_K) q(std::integral_constant<int, TC_VEC_K>());
  else if (mp == TC_VEC_T) q(std::integral_constant<int, TC_VEC_T>());
  else q(std::integral_constant<int, TC_SCALAR>());
}
template <typename F>
void tc_kernel(const TcSpec& t, F&& f) {
  if (t.Kc == 32) tc_modes<8, 4, 4>(t.modeP, t.modeQ, f);
  else if (t.TN <= 128) tc_modes<4, 4, 5>(t.modeP, t.modeQ, f);
  else tc_modes<4, 8, 4>(t.modeP, t.modeQ, f);
}
#endif  // __CUDACC__

}  // namespace pv
#endif
