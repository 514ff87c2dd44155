// Tensor-core contractions of the batched engine (float32 storage, TF32 multiplies, FP32
// accumulation): one strided GEMM per chain, C[m][n] = sum_k P[m][k] Q[n][k], where the row,
// column and contraction indices are multi-indices with arbitrary strides (the transfer
// contractions of the boundary-MPS environments and strips, Sec. II).
//
// Operand chunks are rounded to TF32 and written to shared memory in the canonical K-major layout
// without swizzle (core matrices of 8 rows x 16 bytes stored as 128 contiguous bytes); one thread
// issues `tcgen05.mma.kind::tf32` (M = 128, N = the tile width, K = 8 an instruction) into an
// accumulator in tensor memory and commits them to an mbarrier; each warp reads its 32 accumulator
// lanes with `tcgen05.ld` and scatters them to C.  The kernel of the batched launches is in
// pv_gemm.cuh, the form that the chain programs use in pv_prog.cu.
#ifndef PV_TC_CUH
#define PV_TC_CUH
#include <cstdint>

namespace pv {

// Index plan of one tensor-core contraction; rows are the larger of the two free sides.
struct TcSpec {
  int nr, nc, nk;
  int rs[4], rP[4], rC[4];   // row dims: sizes, strides in P, strides in C
  int cs[4], cQ[4], cC[4];   // column dims: sizes, strides in Q, strides in C
  int ks[4], kP[4], kQ[4];   // contraction dims: sizes, strides in P and in Q
  int M, N, K;
  int TN;                    // tile width: a multiple of 16, at most 256
  int Kc;                    // contraction chunk: 8, 16 or 32 (tc_shape)
  int modeP, modeQ;          // operand gather forms (TC_SCALAR, TC_VEC_K, TC_VEC_T)
  int pairP, pairQ;          // TC_SCALAR: pairs of contraction indices are adjacent and 8-byte aligned
  int vecC;                  // 16-byte stores of four consecutive columns of C
  int split;                 // 3xTF32: operands as hi + lo TF32 parts, products hi.hi + hi.lo + lo.hi
  int sym;                   // Q is P with the same index maps (C = P P^T, one tile): the B
                             // operand is read from the A stage instead of being gathered
  int no_mma;                // self-test only: issue no MMA and no commit, so every wait runs out
};

constexpr int TC_ROWS = 128;
constexpr int TC_THREADS = 128;
constexpr unsigned long long TC_WAIT_NS = 1000000000ull;   // bound of one completion wait (1 s)
constexpr int TC_SCALAR = 0, TC_VEC_K = 1, TC_VEC_T = 2;

// Plans C = A.B of a GEMM-shaped contraction for the tensor cores; false when the shape
// does not suit them (no contraction worth the name, or both free sides small).
inline bool tc_plan(const GSpec& g, TcSpec& t, bool& swap, int tc_min_rows = 64) {
  if (!g.ok || g.K < 4 || g.K > 4096) return false;
  swap = g.N > g.M;
  const int M = swap ? g.N : g.M, N = swap ? g.M : g.N;
  if (M < tc_min_rows) return false;
  t.M = M;
  t.N = N;
  t.K = g.K;
  t.nr = swap ? g.nn : g.nm;
  t.nc = swap ? g.nm : g.nn;
  t.nk = g.nk;
  for (int d = 0; d < 4; ++d) {
    t.rs[d] = swap ? g.ns[d] : g.ms[d];
    t.rP[d] = swap ? g.nB[d] : g.mA[d];
    t.rC[d] = swap ? g.nC[d] : g.mC[d];
    t.cs[d] = swap ? g.ms[d] : g.ns[d];
    t.cQ[d] = swap ? g.mA[d] : g.nB[d];
    t.cC[d] = swap ? g.mC[d] : g.nC[d];
    t.ks[d] = g.ks[d];
    t.kP[d] = swap ? g.kB[d] : g.kA[d];
    t.kQ[d] = swap ? g.kA[d] : g.kB[d];
  }
  int n16 = ((N + 15) / 16) * 16;
  t.TN = n16 < 256 ? n16 : 256;
  t.Kc = 8;
  t.modeP = t.modeQ = TC_SCALAR;
  t.vecC = t.pairP = t.pairQ = 0;
  t.split = 0;
  t.sym = 0;
  t.no_mma = 0;
  return true;
}

// Whether C = P Q^T is a Gram product P P^T that one tile covers: the column side and its
// strides in Q are the row side and its strides in P, the contraction strides agree, and the
// caller passes the same operand twice (`same`).
inline bool tc_symmetric(const TcSpec& t, bool same) {
  if (!same || t.M != t.N || t.M > TC_ROWS || t.TN < t.N || t.nr != t.nc) return false;
  for (int d = 0; d < t.nr; ++d)
    if (t.rs[d] != t.cs[d] || t.rP[d] != t.cQ[d]) return false;
  for (int d = 0; d < t.nk; ++d)
    if (t.kP[d] != t.kQ[d]) return false;
  return t.modeP == t.modeQ;
}

inline bool tc_all4(const int* st, int n) {
  for (int d = 0; d < n; ++d)
    if (st[d] % 4) return false;
  return true;
}

// Operand form: 16-byte loads along the contraction index or along the rows when the
// operand is unit-stride there in blocks of four and every other stride keeps 16-byte
// alignment (`al`: the operand's base and per-chain offsets are multiples of 16 bytes).
// Length of the contiguous run of the trailing dims (0 unless the last is unit-stride); d: its first dim.
inline int tc_run(int n, const int* sz, const int* st, int& d) {
  d = n - 1;
  if (n == 0 || st[n - 1] != 1) return 0;
  int run = sz[d];
  while (d > 0 && st[d - 1] == st[d] * sz[d]) run *= sz[--d];
  return run;
}

inline int tc_mode(bool al, int nr, const int* rsz, const int* rst, int nk, const int* ksz,
                   const int* kst) {
  if (!al) return TC_SCALAR;
  int d = 0, run = tc_run(nk, ksz, kst, d);
  if (run && run % 4 == 0 && tc_all4(kst, d) && tc_all4(rst, nr)) return TC_VEC_K;
  run = tc_run(nr, rsz, rst, d);
  if (run && run % 4 == 0 && tc_all4(rst, d) && tc_all4(kst, nk)) return TC_VEC_T;
  return TC_SCALAR;
}

// Whether an element-wise operand can be loaded two contraction indices at a time (`al8`: base and
// per-chain offsets are multiples of 8 bytes): contiguous in runs of even length, as the bonds of
// D = 6 are.
inline int tc_pairs(bool al8, int nr, const int* rst, int nk, const int* ksz, const int* kst) {
  if (!al8 || nk == 0 || kst[nk - 1] != 1 || ksz[nk - 1] % 2) return 0;
  for (int d = 0; d < nr; ++d)
    if (rst[d] % 2) return 0;
  for (int d = 0; d < nk - 1; ++d)
    if (kst[d] % 2) return 0;
  return 1;
}

inline void tc_forms(TcSpec& t, bool p_al, bool q_al, bool c_al, bool p_al8 = false, bool q_al8 = false) {
  t.modeP = tc_mode(p_al, t.nr, t.rs, t.rP, t.nk, t.ks, t.kP);
  t.modeQ = tc_mode(q_al, t.nc, t.cs, t.cQ, t.nk, t.ks, t.kQ);
  t.pairP = t.modeP == TC_SCALAR && tc_pairs(p_al8, t.nr, t.rP, t.nk, t.ks, t.kP);
  t.pairQ = t.modeQ == TC_SCALAR && tc_pairs(q_al8, t.nc, t.cQ, t.nk, t.ks, t.kQ);
  // four consecutive columns are adjacent in C when the trailing column dims that are contiguous
  // there together hold a multiple of four (6 x 6 bond pairs at D = 6)
  int d = 0;
  const int run = tc_run(t.nc, t.cs, t.cC, d);
  t.vecC = c_al && run && run % 4 == 0 && tc_all4(t.cC, d) && tc_all4(t.rC, t.nr) ? 1 : 0;
}

PV_HD int tc_cols(int TN) {
  int c = 32;
  while (c < TN) c <<= 1;
  return c;
}

#if defined(__CUDACC__)

__device__ __forceinline__ uint32_t tc_smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: start address, leading-dimension byte offset (between
// core matrices along K), stride-dimension byte offset (between 8-row groups), descriptor
// version 1 (bits 46-47), base offset 0, no swizzle.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of kind::tf32: D float32 (bits 4-5 = 1), A and B TF32 (bits 7-9 and
// 10-12 = 2), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ float tc_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                       int accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

__device__ __forceinline__ unsigned long long tc_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool tc_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}

// Waits for the phase `parity` of an mbarrier to complete; false after TC_WAIT_NS.  The timer is
// read only when the first attempts have failed: reading it costs more than a tile's MMAs.
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < 1024; ++i)
    if (tc_try_wait(bar, parity)) return true;
  const unsigned long long t0 = tc_now();
  for (;;) {
    for (int i = 0; i < 64; ++i)
      if (tc_try_wait(bar, parity)) return true;
    if (tc_now() - t0 > TC_WAIT_NS) return false;
  }
}

// 16 consecutive accumulator columns of this thread's lane.
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

constexpr int TC_UNROLL = 4;

__device__ __forceinline__ float4 tc_round4(float4 v) {
  return make_float4(tc_round(v.x), tc_round(v.y), tc_round(v.z), tc_round(v.w));
}

// Stores the TF32 rounding of v, and, for split operands, the rounding of the remainder.
__device__ __forceinline__ void tc_st(float* hi, float* lo, int e, float v) {
  const float h = tc_round(v);
  hi[e] = h;
  if (lo) lo[e] = tc_round(v - h);
}
__device__ __forceinline__ void tc_st4(float* hi, float* lo, int e, float4 v) {
  const float4 h = tc_round4(v);
  ((float4*)hi)[e] = h;
  if (lo) ((float4*)lo)[e] = tc_round4(make_float4(v.x - h.x, v.y - h.y, v.z - h.z, v.w - h.w));
}

// Descriptor of k-block kb (8 contraction indices = two core matrices along K).
__device__ __forceinline__ uint64_t tc_kdesc(uint32_t base, int Kc, int kb) {
  return tc_desc(base + kb * 256, 128, (uint32_t)Kc * 32u);
}

// The MMAs of k-block kb: hi.hi, and for split operands also hi.lo and lo.hi.
__device__ __forceinline__ void tc_mma_k(int split, uint32_t tmem, uint32_t a, uint32_t b,
                                         uint32_t al, uint32_t bl, int Kc, int kb,
                                         uint32_t idesc, bool accumulate) {
  tc_mma(tmem, tc_kdesc(a, Kc, kb), tc_kdesc(b, Kc, kb), idesc, accumulate ? 1 : 0);
  if (split) {
    tc_mma(tmem, tc_kdesc(a, Kc, kb), tc_kdesc(bl, Kc, kb), idesc, 1);
    tc_mma(tmem, tc_kdesc(al, Kc, kb), tc_kdesc(b, Kc, kb), idesc, 1);
  }
}

// Accumulator rows of this warp's lane quarter to C (16-byte stores when C is unit-stride
// in its columns).
__device__ __forceinline__ void tc_epilogue(const TcSpec& t, uint32_t tmem, float* pc,
                                            const int* rowC, const int* colC, int warp, int lane) {
  const int oc = rowC[warp * 32 + lane];
  for (int c0 = 0; c0 < t.TN; c0 += 16) {
    uint32_t v[16];
    tc_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
    if (oc >= 0) {
      if (t.vecC) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
          const int cc = colC[c0 + j];
          if (cc >= 0)
            *(float4*)(pc + oc + cc) = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                                   __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int cc = colC[c0 + j];
          if (cc >= 0) pc[oc + cc] = __uint_as_float(v[j]);
        }
      }
    }
  }
}

#endif  // __CUDACC__

}  // namespace pv
#endif
