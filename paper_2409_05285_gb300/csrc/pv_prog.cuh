// Chain programs: the operations of a whole evaluation, sweep, draw or amplitude as one launch.
//
// No operation of the batched runner reads another chain's data, so a sequence of them can run
// chain by chain: a thread block takes a chain and executes the recorded list of operations
// with a block barrier between them, while other blocks do the same for other chains.  Against
// one launch per operation over all chains this removes the launches (thousands per call, about
// 5 us each, which bound small problems) and keeps a chain's intermediates in the caches of
// the SM that made them instead of streaming every one through device memory (which bounds
// large ones).  Every operation computes the bits of its batched kernel: contractions sum in
// the same order (the same tcgen05 instructions over the same blocks of eight indices on the
// tensor cores, one fused multiply-add per index elsewhere), and the factorisations,
// truncations and dot products run the same per-matrix routines.
//
// A program is a list of PgOp records plus a pool of index tables in device memory, made once
// per (sequence, block shape) and kept with the runner's work buffers, up to pg_pool_bytes().  Pointers to those
// buffers are absolute; the caller's arrays (configurations, outputs) are slots that every
// launch binds anew.  Per-chain scalars and selections (val, num, den, val2; si, sj, valid,
// accepted) and the chain's configuration live in shared memory.
#ifndef PV_PROG_CUH
#define PV_PROG_CUH

#if defined(__CUDACC__)
#include <array>
#include <cstring>
#include <map>
#include <tuple>
#include <vector>

namespace pv {

enum PgKind : int {
  PG_FMA, PG_TC, PG_EIN, PG_COPY, PG_NORM, PG_LQ, PG_LQ2, PG_CHOL, PG_TRUNC, PG_TRUNC64, PG_O, PG_DIAG,
  PG_SKIP,   // the next i[0] operations are left out where the proposal changes nothing
  // executed by the first thread (PG_DOT: the first warp): no barrier between two of them
  PG_T0, PG_SET = PG_T0, PG_SETD, PG_COPYD, PG_SETI8, PG_SEL, PG_DOT, PG_RATIO, PG_ACCEPT, PG_AMP, PG_DRAW
};

// Slots of the caller's arrays.
enum PgSlot : int { PS_S, PS_LA, PS_SG, PS_ES, PS_EA, PS_O, PS_ACC, PS_PROP, PS_U, PS_LOGQ, PS_N };

// Encoded pointer: absolute, or (tag << 56) + byte offset with tag 1 + slot, or a shared scalar.
typedef unsigned long long pgptr;
constexpr int PG_TAG = 56;
constexpr pgptr PG_OFF = (1ull << PG_TAG) - 1;
constexpr int PG_SC = 64;   // tag of shared scalar i: PG_SC + i (0 val, 1 num, 2 den, 3 val2)

struct PgArgs {
  char* gbase;           // a device allocation, and its address again as an integer: pointers read
  pgptr gint;            // from memory are formed from the two, which marks them as global memory
  void* slot[PS_N];
  int n, N, chain0, p;
  uint64_t seed;
  const uint32_t* sweep_dev;
  double b_d, expo;
  double* jflops;
};

struct PgOpnd {   // a contraction operand: base + (chain | local index) * stride elements
  pgptr base;
  long long stride;
  int mode, site, sel;   // OP_BATCH, OP_SITE_S (site) or OP_SITE_SEL (sel: shared selection)
  int pad;
};

struct PgFma {
  int M, N, ks[3], ka[3], kb[3];     // contraction dims, innermost first
  int tm, tn;                        // outputs per thread
  int rowA, rowC, colB, colC;        // index tables
};
struct PgTc {
  int M, N, K, TN, Kc, lq;           // lq: log2(Kc / 4)
  int modeP, modeQ, vecC, split, sym, nst, nacc, swap;
  int rowP, rowC, colQ, colC, kP, kQ;
};
struct alignas(16) PgOp {
  int kind, bar;                     // bar: block barrier after this operation
  union {
    struct {
      PgOpnd A, B;
      pgptr out;
      long long os;
      union {
        PgFma f;
        PgTc t;
        int mspec;
      };
    } e;
    struct {
      pgptr p[6];
      long long l[6];
      int i[10];
      double d;
    } g;
  };
};
static_assert(sizeof(PgOp) % 16 == 0, "16-byte copies");

constexpr int PG_BLOCK = 8;          // operations fetched at a time

struct PgProgram {
  PgOp* d_ops = nullptr;             // device: nblk * PG_BLOCK records, then ...
  int* d_tab = nullptr;              // ... the tables, `size` bytes together
  size_t size = 0;
  long long used = 0;                // the last call that ran it
  int nops = 0, threads = 0, per_sm = 0, tmem_cols = 0;
  size_t arena = 0;                  // dynamic shared memory of a block
  double flops = 0, bytes = 0;       // per chain
  bool bad = false;                  // an operation has no program form: use the batched launches
};

template <typename T>
void pg_launch(const PgProgram& p, const PgArgs& a, T jtol, double jtol64, int max_sweeps, unsigned long long* sweeps,
               int* err, int sms, cudaStream_t st);

constexpr size_t PG_STATIC = 5 * 1024;        // PgShared and the system's share
constexpr size_t PG_SMEM = 227 * 1024;
constexpr int PG_PER_SM = 16;                 // most chains an SM holds: a warp each

// Device bytes that the programs of one engine may take on a lattice of N sites.  The longest
// sequence (an evaluation with J2) is 99 records of 176 bytes a site and up to 55 KB of tables, 17 KB
// a site at 8x8 D=4 chi=16: room for fifteen of them.
inline size_t pg_pool_bytes(int N) { return (size_t)N * 256 * 1024; }

// Threads per block for n chains on `sms` SMs (one chain per block): the 512 threads that 128
// registers allow an SM are shared among the chains it has, down to one warp each, but a chain
// gets no more than half the outputs of its largest contraction, and at least the four warps
// that read tensor memory where it uses the tensor cores.
inline int pg_threads(int n, int sms, long long largest, bool tc) {
  const int q = (n + sms - 1) / sms;
  int share = 512;
  while (share > 32 && 512 / share < q) share >>= 1;
  int want = 32;
  while (want < 512 && want * 2 < largest) want <<= 1;
  int t = share < want ? share : want;
  if (tc && t < 128) t = share < 128 ? 128 : (want < 128 ? 128 : t);
  return t;
}

// Whether a sequence of `ops` operations and `flops` per chain runs as a program for n chains:
// where the launches bound it.  Measured, a sweep as a program / launched (ms):
//   float64 4x4 D=2 chi=4 (55 flops per operation): 64 chains 1.2 / 7.2, 16384 chains 18.6 / 41.8;
//   TF32 8x8 D=2 chi=4 (180): 64 chains 6.5 / 36, 4096 chains 45 / 65, 16384 chains 200 / 126;
//   TF32 5x5 D=3 chi=5 (640): 1024 chains 4.7 / 19.3, 4096 chains 37 / 28;
//   TF32 6x6 D=3 chi=9 (3e3): 1024 chains 18.4 / 33.3, 4096 chains 74 / 55;
//   TF32 4x4 D=4 chi=16 (7e3): 1024 chains 8.0 / 16.8, 4096 chains 35 / 27;
//   TF32 8x8 D=4 chi=16 (7e4): 256 chains 40 / 73, 1024 chains 134 / 123;
//   TF32 4x4 D=6 chi=36 (1.6e5): 64 chains 11.6 / 17.3, 256 chains 24 / 26, 1024 chains 110 / 51;
//   float64 6x6 D=4 chi=16 (4e4): 256 chains 140 / 164, 1024 chains 865 / 426.
// One block per chain is too slow for larger operations at any chain count (10x10 D=6 chi=36,
// 3.8e6 flops per operation).
inline bool pg_wins(int n, double ops, double flops, bool fp64) {
  const double per = flops / (ops > 1 ? ops : 1);
  return per <= 2.5e5 && n * (per > 1 ? per : 1) <= (fp64 ? 1.5e7 : 4e7) &&
         (n <= 3000 || n * per <= (fp64 ? 3e6 : 2e6));
}

// Records operations.  The runner's back end hands each one over instead of launching it.
template <typename T>
struct PgBuild {
  std::vector<PgOp> ops;
  std::vector<int> tab;
  std::map<std::vector<int>, int> tables;
  struct Ext {
    const char* base;
    size_t bytes;
    int slot;
  };
  std::vector<Ext> ext;
  const void* sc[4] = {nullptr, nullptr, nullptr, nullptr};    // val, num, den, val2
  const void* i8[4] = {nullptr, nullptr, nullptr, nullptr};    // si, sj, valid, accepted
  bool bad = false;
  int per_sm = 1, threads = 512, tmem = 0;
  size_t budget = 0;      // bytes a block may take
  size_t need = 0;        // bytes its largest operation takes
  double bytes = 0;
  long long largest = 0;  // outputs of its largest contraction
  bool tc_used = false;

  pgptr enc(const void* p) {
    if (!p) return 0;
    for (int i = 0; i < 4; ++i) {
      if (p == sc[i]) return (pgptr)(PG_SC + i) << PG_TAG;
      if (p == i8[i]) {
        bad = true;   // a selection array where a data pointer is expected
        return 0;
      }
    }
    for (const Ext& e : ext)
      if ((const char*)p >= e.base && (const char*)p < e.base + e.bytes)
        return ((pgptr)(1 + e.slot) << PG_TAG) + (pgptr)((const char*)p - e.base);
    return (pgptr)p;
  }
  int sel(const int8_t* p) {
    for (int i = 0; i < 4; ++i)
      if (p == i8[i]) return i;
    bad = true;
    return 0;
  }
  PgOp& add(int kind) {
    PgOp o;
    memset(&o, 0, sizeof(o));
    o.kind = kind;
    o.bar = 1;
    if (!ops.empty() && ops.back().kind >= PG_T0 && kind >= PG_T0) ops.back().bar = 0;
    ops.push_back(o);
    return ops.back();
  }
  int table(const std::vector<int>& v) {
    auto it = tables.find(v);
    if (it != tables.end()) return it->second;
    const int off = (int)tab.size();
    tab.insert(tab.end(), v.begin(), v.end());
    while (tab.size() & 3) tab.push_back(0);
    tables.emplace(v, off);
    return off;
  }
  // offsets of every row-major multi-index over n dims (at most four), one table per index map
  std::map<std::array<int, 10>, int> maps;
  int offsets(int n, const int* sz, const int* st, int total) {
    std::array<int, 10> key{};
    key[0] = n;
    key[1] = total;
    for (int d = 0; d < n; ++d) {
      key[2 + d] = sz[d];
      key[6 + d] = st[d];
    }
    auto it = maps.find(key);
    if (it != maps.end()) return it->second;
    std::vector<int> v(total);
    for (int i = 0; i < total; ++i) {
      int idx = i, o = 0;
      for (int d = n - 1; d >= 0; --d) {
        o += (idx % sz[d]) * st[d];
        idx /= sz[d];
      }
      v[i] = o;
    }
    const int off = table(v);
    maps.emplace(key, off);
    return off;
  }
  PgOpnd opnd(const Operand<T>& o) {
    PgOpnd q;
    memset(&q, 0, sizeof(q));
    q.mode = o.mode;
    if (o.mode == OP_BATCH) {
      q.base = enc(o.base);
      q.stride = o.stride;
    } else {
      q.base = enc(o.base + o.site_off);
      q.stride = o.site_sz;
      q.site = o.site;
      if (o.mode == OP_SITE_S) {
        const pgptr s = enc(o.S);
        if (s != ((pgptr)(1 + PS_S) << PG_TAG)) bad = true;
      } else {
        q.sel = sel(o.sel);
      }
    }
    if (q.base >> PG_TAG) bad = true;
    return q;
  }
  // tensor-core contraction (tc_plan and tc_forms done; t.split, t.sym set)
  void tc(const TcSpec& t, bool swap, T* out, long long os, const Operand<T>& A, const Operand<T>& B) {
    PgTc q;
    memset(&q, 0, sizeof(q));
    q.M = t.M;
    q.N = t.N;
    q.K = t.K;
    q.modeP = t.modeP;
    q.modeQ = t.modeQ;
    q.vecC = t.vecC;
    q.split = t.split;
    q.swap = swap ? 1 : 0;
    const int n16 = (t.N + 15) / 16 * 16, cols = 512 / (per_sm <= 1 ? 1 : (per_sm <= 2 ? 2 : 4));
    const int cap = cols / 2;   // two accumulators
    const int tiles = (n16 + cap - 1) / cap;
    q.TN = ((t.N + tiles - 1) / tiles + 15) / 16 * 16;
    q.nacc = 2;
    q.sym = t.sym && t.M <= TC_ROWS && q.TN >= t.N;
    int Kc = 8;
    while (Kc < 32 && Kc < t.K) Kc *= 2;
    q.nst = 2;
    auto bytes_of = [&]() {
      return (size_t)(TC_ROWS + (q.sym ? 0 : q.TN)) * Kc * sizeof(float) * (t.split ? 2 : 1) * q.nst;
    };
    while (bytes_of() > budget && Kc > 8) Kc >>= 1;
    if (bytes_of() > budget) q.nst = 1;
    if (bytes_of() > budget) bad = true;
    need = need > bytes_of() ? need : bytes_of();
    q.Kc = Kc;
    q.lq = Kc == 8 ? 1 : (Kc == 16 ? 2 : 3);
    int c = tc_cols(q.TN * q.nacc);
    tmem = tmem > c ? tmem : c;
    q.rowP = offsets(t.nr, t.rs, t.rP, t.M);
    q.rowC = offsets(t.nr, t.rs, t.rC, t.M);
    q.colQ = offsets(t.nc, t.cs, t.cQ, t.N);
    q.colC = offsets(t.nc, t.cs, t.cC, t.N);
    q.kP = offsets(t.nk, t.ks, t.kP, t.K);
    q.kQ = offsets(t.nk, t.ks, t.kQ, t.K);
    tc_used = true;
    largest = largest > (long long)t.M * t.N ? largest : (long long)t.M * t.N;
    PgOp& o = add(PG_TC);
    o.e.A = opnd(A);
    o.e.B = opnd(B);
    o.e.out = enc(out);
    o.e.os = os;
    o.e.t = q;
  }
  // every other GEMM-shaped contraction: one fused multiply-add per index, in index order
  void fma(const GSpec& g, T* out, long long os, const Operand<T>& A, const Operand<T>& B) {
    PgFma f;
    memset(&f, 0, sizeof(f));
    f.M = g.M;
    f.N = g.N;
    int nk = 0, ks[4], ka[4], kb[4];
    for (int d = 0; d < g.nk; ++d) {
      if (nk > 0 && ka[nk - 1] == g.kA[d] * g.ks[d] && kb[nk - 1] == g.kB[d] * g.ks[d]) {
        ks[nk - 1] *= g.ks[d];
        ka[nk - 1] = g.kA[d];
        kb[nk - 1] = g.kB[d];
      } else {
        ks[nk] = g.ks[d];
        ka[nk] = g.kA[d];
        kb[nk] = g.kB[d];
        ++nk;
      }
    }
    if (nk > 3) bad = true;
    for (int d = 0; d < 3; ++d) {
      const int s = nk - 1 - d;
      f.ks[d] = s >= 0 ? ks[s] : 1;
      f.ka[d] = s >= 0 ? ka[s] : 0;
      f.kb[d] = s >= 0 ? kb[s] : 0;
    }
    // outputs per thread: as many as keep every thread busy, at most 4 x 4
    const long long tot = (long long)g.M * g.N;
    largest = largest > tot ? largest : tot;
    f.tm = f.tn = 1;
    if (tot >= 16LL * threads && g.M >= 4 && g.N >= 4) f.tm = f.tn = 4;
    else if (tot >= 4LL * threads && g.M >= 2 && g.N >= 2) f.tm = f.tn = 2;
    else if (tot >= 4LL * threads && g.M >= 4) f.tm = 4;
    else if (tot >= 4LL * threads && g.N >= 4) f.tn = 4;
    f.rowA = offsets(g.nm, g.ms, g.mA, g.M);
    f.rowC = offsets(g.nm, g.ms, g.mC, g.M);
    f.colB = offsets(g.nn, g.ns, g.nB, g.N);
    f.colC = offsets(g.nn, g.ns, g.nC, g.N);
    PgOp& o = add(PG_FMA);
    o.e.A = opnd(A);
    o.e.B = opnd(B);
    o.e.out = enc(out);
    o.e.os = os;
    o.e.f = f;
  }
  void ein(const MSpec& m, T* out, long long os, const Operand<T>& A, const Operand<T>& B) {
    std::vector<int> v(sizeof(MSpec) / sizeof(int));
    memcpy(v.data(), &m, sizeof(MSpec));
    const int off = table(v);
    PgOp& o = add(PG_EIN);
    o.e.A = opnd(A);
    o.e.B = opnd(B);
    o.e.out = enc(out);
    o.e.os = os;
    o.e.mspec = off;
  }
  void fits(size_t b) {
    if (b > budget) bad = true;
    need = need > b ? need : b;
  }
};

}  // namespace pv
#endif  // __CUDACC__
#endif
