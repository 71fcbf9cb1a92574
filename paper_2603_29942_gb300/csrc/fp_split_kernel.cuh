// fp_split_kernel.cuh -- tensor-core enumeration kernel for one code (p = 3,
// 5, 7): the passes of the Brouwer-Zimmermann search as class comparisons of
// stems with tails (fp_split.cuh) on the fifth-generation tensor cores.
//
// One persistent CTA per SM: 512 working threads and a warpgroup of which
// one warp claims tasks ahead, counts finished ones off and polls the best
// weight, so that no working warp waits for L2 (F_3 [80,40] 161 -> 118 us,
// F_7 [50,25] 454 -> 328 us).  A CTA holds one block of tails
// of one information set in shared memory, each tail's class values as one
// row of K fp8 bytes (the B operand, 96 rows to a tile).  Its four
// warpgroups work on their own: each lane walks its own stems (one exact
// bit-sliced add per step), writes the current stem's class values as its
// row of the A operand in tensor memory, and the 128 stems are compared
// with a tile of tails by tcgen05.mma (M = 128, N = 96, K / 32 steps).  The
// threshold rides along as three more values of each row, so a result is
// negative exactly where the bound says that neither S + B nor S - B can
// matter.  Each lane reads its row of results as packed f16, ANDs the sign
// bits (one LOP3 for four codewords), and only results of sign 0 go on to
// the exact weights.
//
// What bounds it: the read and the AND of the results and the tensor pipe
// are balanced at K = 64 (109 results, 218 codewords, a clock and SM
// measured with nothing else; 85 at K = 96 and 64 at K = 128, where the
// tensor pipe is full), so what is left is the stems: the walk, the
// exact add and the class values, paid once per stem and block of tails,
// and the latency of a step (1 to 1.6 us a step of 128 stems a warpgroup,
// 0.5 to 0.7 us a tile).  That is why tails
// have two or three rows, whichever costs less over the pass (plan_split):
// the pair table of the popcount kernel serves a stem of a deep pass only
// 36 to 104 entries.  M = 128 with the A operand in tensor memory keeps the
// stems out of shared memory, whose read port the B operand needs; N = 96
// is what four warpgroups of up to 32 + 96 columns leave room for, and
// setmaxnreg moves the claiming warpgroup's registers to the working ones
// (96 at launch, then 112 and 32: F_7 [52,19] 2534 -> 1965 us, fewer spills in
// the steps).  Three warpgroups of N = 128, or of two N = 64 accumulators,
// and two half-size table buffers were slower.
//
// Against the popcount kernels (whole search): F_3 [80,40] 174 -> 120 us,
// F_7 [50,25] 845 -> 301, F_7 [52,19] 17389 -> 1940, F_3 [74,50] 1254 ->
// 375, F_5 [51,24] 431 -> 126.  ncu, F_7 [50,25]: tensor pipe 24 %, ALU 41 %,
// issue slots 38 %: bound by latency within a step, not by a pipe.
#pragma once
#include "fp_kernel.cuh"
#include "fp_split.cuh"

namespace fpk {

constexpr int kSplitWarps = kSplitThreads / 32;
constexpr uint32_t kTmemCols = 512;    // all of the SM's tensor memory: one such CTA per SM
constexpr uint32_t kTmemGroup = 128;   // a warpgroup's columns: the A tile (up to 32), then the results
constexpr uint32_t kTmemD = 32;

// ------------------------------------------------------------- tcgen05 ----
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(e));
  return e != 0;
}
__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void group_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
constexpr int kCloseBar = 6;  // named barriers: 1 .. 4 the warpgroups' products, 5 the working warps, 6 .. 9 the warpgroups' closes
constexpr int kLost = 2;
__device__ __forceinline__ void group_arrive(int id) { asm volatile("bar.arrive %0, 128;" ::"r"(id) : "memory"); }

// D (f16, 128 x N, tensor memory) = (accumulate ? D : 0) + A (e4m3, tensor memory) B^T (e4m3, shared memory)
template <bool ACC>
__device__ __forceinline__ void mma_step(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc) {
  if constexpr (ACC)
    asm volatile("tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, 1;" ::"r"(d), "r"(a), "l"(b), "r"(idesc)
                 : "memory");
  else
    asm volatile("tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, 0;" ::"r"(d), "r"(a), "l"(b), "r"(idesc)
                 : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok)
               : "r"(bar), "r"(parity)
               : "memory");
  return ok != 0;
}
// Bounded: false if the barrier's phase has not completed after 2^18 tries (about a second).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < (1 << 18); ++i)
    if (mbar_test(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ void tmem_store8(uint32_t addr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// 32 f16 results of the lane's row, two to a register.
__device__ __forceinline__ void tmem_load16(uint32_t addr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.pack::16b.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
      "%14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(addr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait_store() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_load(uint32_t (&a)[16], uint32_t (&b)[16], uint32_t (&c)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(a[i]), "+r"(b[i]), "+r"(c[i])::);  // no use before the wait
}
// Instruction descriptor: f16 results, e4m3 operands, both K-major, M = 128.
constexpr uint32_t kSplitIdesc = ((uint32_t)kSplitN >> 3) << 17 | (128u >> 4) << 24;
// Shared-memory descriptor of the B tile whose first row group is at `addr`:
// no swizzle, 8-row x 16-byte core matrices, the K / 16 matrices of a row
// group one after another (128 bytes apart), row groups 8 K bytes apart.
__device__ __forceinline__ uint64_t tile_desc(uint32_t addr, uint32_t K) {
  return (uint64_t)(addr >> 4 & 0x3FFFu) | (uint64_t)(128u >> 4) << 16 | (uint64_t)((8u * K) >> 4) << 32 | 1ull << 46;
}
__device__ __forceinline__ uint32_t and3(uint32_t a, uint32_t b, uint32_t c) { return a & b & c; }

// --------------------------------------------------------- class values ----
// Class bits of a vector over its first nu positions, values one after
// another (p = 3: one bit a position; p = 5, 7: the three character bits),
// as four 32-bit words (unused ones zero).
template <int P, int R, int W>
__device__ __forceinline__ void class_bits(const uint32_t (&s)[R * W], int nu, uint32_t (&o)[4]) {
  if constexpr (P == 3) {
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      if (w < W) {
        const int left = nu - 32 * w;
        const uint32_t x = s[w * R] ^ s[w * R + 1];
        o[w] = left >= 32 ? x : left > 0 ? x & ((1u << left) - 1u) : 0u;
      } else {
        o[w] = 0u;
      }
    }
  } else {
    uint64_t u = 0, v = 0;
#pragma unroll
    for (int w = 0; w < W && w < 2; ++w) {
      uint32_t a, c;
      if constexpr (P == 7) {  // -x is the complement of x != 0: neighbouring slices' differences tell the class
        a = s[w * R] ^ s[w * R + 1];
        c = s[w * R + 1] ^ s[w * R + 2];
      } else {  // p = 5: {1, 4} and {2, 3}
        a = s[w * R + 2] | (s[w * R] & ~s[w * R + 1]);
        c = s[w * R + 1];
      }
      u |= (uint64_t)a << (32 * w);
      v |= (uint64_t)c << (32 * w);
    }
    const uint64_t m = (1ull << nu) - 1ull;  // nu <= 41 here
    u &= m;
    v &= m;
    const uint64_t x = u ^ v;
    const int s2 = 2 * nu;
    const uint64_t lo = u | v << nu | (s2 < 64 ? x << s2 : 0ull);
    const uint64_t hi = v >> (64 - nu) | (s2 < 64 ? x >> (64 - s2) : x << (s2 - 64));
    o[0] = (uint32_t)lo;
    o[1] = (uint32_t)(lo >> 32);
    o[2] = (uint32_t)hi;
    o[3] = (uint32_t)(hi >> 32);
  }
}
// 32 class bits -> 32 fp8 values (bit 0: 1.0, bit 1: -1.0), four to a word:
// a nibble times 0x10204080 has bit i at bit 8 i + 7.
__device__ __forceinline__ void class_bytes(uint32_t bits, uint32_t (&w)[8]) {
  const uint32_t t = bits & 0x0F0F0F0Fu, u = bits >> 4 & 0x0F0F0F0Fu;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    w[2 * j] = (__byte_perm(t, 0u, 0x4440u | j) * 0x10204080u & 0x80808080u) | 0x38383838u;
    w[2 * j + 1] = (__byte_perm(u, 0u, 0x4440u | j) * 0x10204080u & 0x80808080u) | 0x38383838u;
  }
}
constexpr uint32_t kTailMarks = 0x00383800u;     // last word of a tail: unused, 1, 1, 0
constexpr uint32_t kTailPadding = 0xFE000000u;   // of a row past the block's tails: 0, 0, 0, -448
constexpr uint32_t kStemNone = 0x38FEFE00u;      // last word of a lane without a stem: unused, -448, -448, 1
// Last word of a stem: minus the value that the result must exceed, as a
// multiple of 16 and a rest, and the 1 that the padding rows' mark meets.
// <S, B> = same nu - (same + 1) lb, and lb < thr is asked, so the value is
// same nu - (same + 1) thr + 1: results are odd multiples apart from zero.
template <int P>
__device__ __forceinline__ uint32_t stem_marks(int nu, int thr) {
  constexpr int same = ClassCode<P>::kSame;
  int v = (same + 1) * thr - 1 - same * nu;
  v = min(max(v, -255), 255);  // outside, no bound of a real row changes sign
  const int coarse = v / 16 * 16, fine = v - coarse;
  uint16_t h;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(h) : "f"((float)fine), "f"((float)coarse));
  return (uint32_t)h << 8 | 0x38000000u;
}

// ------------------------------------------------------------- the CTA ----
// Tails [first, first + n) of a set into shared memory: packed rows and
// coefficients, and (table) the class values as rows of the B operand,
// rows n .. padded to whole tiles marked as padding.  A thread takes a run
// of consecutive tails (one exact add each; the run's length is odd, so the
// threads' 16-byte stores fall into different banks).
template <int P, int R, int W>
__device__ __noinline__ void build_tails(uint32_t *tails, char *table, const uint32_t *mult, const fpenum::BinomCols B,
                                         int k, int t, uint32_t first, uint32_t n, int K, int nu, bool with_table) {
  constexpr int b = P - 1, RW = R * W;
  const uint32_t rows = with_table ? (n + kSplitN - 1) / kSplitN * kSplitN : n;
  const uint32_t run = ((rows + kSplitThreads - 1) / kSplitThreads) | 1u;
  const uint32_t e0 = threadIdx.x * run, e1 = min(e0 + run, rows);
  const int vals = nu * ClassCode<P>::kVals;
  if (e0 >= e1) return;
  Tail a{};
  uint32_t part[RW];
  bool fresh = true;
  if (e0 < n) a = tail_unrank(B, first + e0, k, t, b);
  for (uint32_t e = e0; e < e1; ++e) {
    uint32_t o[4] = {0u, 0u, 0u, 0u};
    if (e < n) {
      tails[e] = tail_pack(a);
      if (with_table) {
        if (fresh) {
          set_row<P, R, W>(part, mult, a.z, 1, P);
          if (a.cy) add_row<P, R, W>(part, mult, a.y, a.cy, P);
        }
        uint32_t sum[RW];
#pragma unroll
        for (int q = 0; q < RW; ++q) sum[q] = part[q];
        add_row<P, R, W>(sum, mult, a.x, a.cx, P);
        class_bits<P, R, W>(sum, nu, o);
      }
      if (e + 1 < n) fresh = tail_next(a, k, t, b);
    }
    if (with_table) {
      char *row = table + (size_t)(e >> 3) * (8 * K) + (e & 7) * 16;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        if (32 * s >= K) break;
        uint32_t w[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
        const int left = vals - 32 * s;  // the same for all tails
        if (e < n && left > 0) {
          class_bytes(o[s], w);
          if (left < 32) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              w[i] = left >= 4 * i + 4 ? w[i] : left > 4 * i ? w[i] & ((1u << (8 * (left - 4 * i))) - 1u) : 0u;
          }
        }
        if (32 * (s + 1) == K) w[7] = e < n ? kTailMarks : kTailPadding;
        *reinterpret_cast<uint4 *>(row + s * 256) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4 *>(row + s * 256 + 128) = make_uint4(w[4], w[5], w[6], w[7]);
      }
    }
  }
}

// A warp's candidates: (tail of the block) << 5 | lane.
struct SplitQueue {
  uint32_t item[64];  // fewer than 32 left over, then at most one per lane
};

// A task as the scheduler warp hands it to the warpgroups.
struct SplitTask {
  Claim cl;
  PassDesc pd;
  int cmd;                   // kCmdRun or kCmdExit
  int stage, build;          // stage the set's multiples; build its tail block: 1 packed tails, 2 also the B operand
  int drop;                  // the code finished before the task began
  unsigned long long count;  // codewords evaluated
};

// What the threads of a CTA share.
struct SplitShared {
  int32_t stop[kSplitGroups][2];  // by the parity of the product: the code has finished, the warpgroup drops the rest
                                  // of its task (two, since the first warp may be a product ahead of the last)
  unsigned long long best_key;    // the code's best key (inverted) and finished flag, as the scheduler last read them
  int32_t finished;
  int32_t over;                   // the scheduler has given up a running task: nothing more is handed out
  int32_t lost_any;               // ... or a warpgroup has lost a product
  int32_t lost[kSplitGroups];     // a product of the warpgroup never came: it issues no more
  SlotState *states;              // of the launch
  SlotAux *aux;
  CtlDyn *cdyn;
  SplitQueue queue[kSplitWarps];
  SplitTask task[2];              // the one that runs and the next one
  // mbarriers: of each task buffer, full (1 arrival), near its end (one per
  // warpgroup) and done (one per warp); of each warpgroup, its products
  // (the commit's arrival and the issuing warp's)
  unsigned long long full[2], near[2], done[2], product[kSplitGroups];
};

// The stem a lane holds: its exact sum, its rows and coefficients.
template <int RW>
struct Stem {
  uint32_t s[RW];
  StemPos pos;
};

template <int P, int R, int W, int DB>
__device__ __forceinline__ void stem_sum(Stem<R * W> &x, const uint32_t *mult, int l) {
  constexpr int b = P - 1;
  set_row<P, R, W>(x.s, mult, x.pos.m, fpenum::gray_digit<DB>(x.pos.d, l - 1, b, l) + 1, P);
  uint64_t Q = x.pos.Q;
  for (int s = 0; s + 1 < l; ++s) {
    const int q = fpenum::ctz64(Q);
    Q &= Q - 1;
    add_row<P, R, W>(x.s, mult, q, fpenum::gray_digit<DB>(x.pos.d, s, b, l) + 1, P);
  }
}

template <int P, int R, int W, int DB>
__device__ __forceinline__ void stem_start(Stem<R * W> &x, const uint32_t *mult, const fpenum::BinomCols &B,
                                           uint64_t J, int k, int t, int l, uint64_t ncl) {
  x.pos = stem_unrank<DB>(B, J, k, t, l, P - 1, ncl);
  stem_sum<P, R, W, DB>(x, mult, l);
}

template <int P, int R, int W, int DB>
__device__ __forceinline__ void stem_next(Stem<R * W> &x, const uint32_t *mult, int l) {
  int dir = 1;
  const int slot = stem_advance<DB>(x.pos, P - 1, l, &dir);
  if (slot >= 0) {
    const int q = slot == l - 1 ? x.pos.m : fpenum::nth_member(x.pos.Q, slot);
    add_row<P, R, W>(x.s, mult, q, dir > 0 ? 1 : P - 1, P);  // c -> c+1: +A; c -> c-1: +(p-1)A
  } else {
    stem_sum<P, R, W, DB>(x, mult, l);
  }
}

// Exact redundant weights of S + B and S - B for the packed tail.
template <int P, int R, int W>
__device__ __forceinline__ void split_weights(const uint32_t (&s)[R * W], const Tail &a, const uint32_t *mult, int &wp,
                                              int &wm) {
  uint32_t v[R * W];
  set_row<P, R, W>(v, mult, a.z, 1, P);
  if (a.cy) add_row<P, R, W>(v, mult, a.y, a.cy, P);
  add_row<P, R, W>(v, mult, a.x, a.cx, P);
  wp = 0;
  wm = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    uint32_t sum[R];
    fpbs::add_exact<P, R>(&s[w * R], &v[w * R], sum, P);
    wp += __popc(fpbs::nz<R>(sum));
    wm += __popc(fpbs::nz_sub<R>(&s[w * R], &v[w * R]));
  }
}

// The least key of a lane's hits: out of line, it runs for codewords at or
// under the bound only.
template <int DB>
__device__ __noinline__ uint64_t hit_key(const fpenum::BinomCols B, bool pair, int k, int p, int g, int pass, int wp,
                                         int wm, int thr, StemPos pf, int l, uint32_t tail) {
  const Tail a = tail_unpack(tail);
  uint64_t best = kNoKey;
  if (wp < thr) best = split_key<DB>(B, pair, k, p, g, (uint32_t)pass, (uint32_t)(g + wp), pf, l, a, 0);
  if (l > 0 && wm < thr) best = min(best, split_key<DB>(B, pair, k, p, g, (uint32_t)pass, (uint32_t)(g + wm), pf, l, a, 1));
  return best;
}

// One task of a pass with g >= 2: units [ulo, uhi) of one tail block, a
// unit being 128 stems (tensor-core passes) or one stem (direct passes).
// Every warpgroup takes an equal run of them (esplit 0), or a run and one of
// 2 or 4 interleaved slices of the tails, so nothing is handed out inside a
// task; `near` is told when its last step begins.
template <int P, int R, int W>
__device__ __forceinline__ unsigned long long task_split(const SlotDesc &sd, SplitShared &sh, int buf, const uint32_t *mult,
                                                         const uint32_t *tails, uint32_t table, uint32_t tmem,
                                                         uint32_t &parity, const fpenum::BinomCols &B) {
  const PassDesc &pd = sh.task[buf].pd;
  const Claim &cl = sh.task[buf].cl;
  constexpr int DB = P == 3 ? 1 : 4, RW = R * W, b = P - 1;
  constexpr unsigned FULL = 0xffffffffu;
  const int k = sd.k, g = pd.g, t = pd.tail_rows(), l = g - t;
  const int lane = threadIdx.x & 31, row = threadIdx.x & (kSplitGroup - 1);
  const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0), grp = warp / (kSplitGroup / 32);
  const uint32_t mbar = smem_u32(&sh.product[grp]), near = smem_u32(&sh.near[buf]);
  const bool pair = sd.pair_sigp > 0;
  const uint64_t ncl = pd.ncl();
  const uint32_t etot = tails_above(B, k, t, b, -1);
  const uint32_t first = cl.block * pd.block(), nb = min(pd.block(), etot - first);
  const uint64_t ns = l > 0 ? B(cl.zhi, l) * ncl : 1ull;
  const int K = sd.split_k(), nu = sd.split_nu();
  uint32_t seen = 0;  // this lane's stem-tail pairs (a task's fit 32 bits): two codewords each, or one (l = 0)
  // the warpgroup's units [u0, u0 + steps) and its slice of the tails
  const uint32_t parts = pd.esplit() ? 1u : (uint32_t)kSplitGroups, part = pd.esplit() ? 0u : (uint32_t)grp;
  const uint32_t slices = pd.esplit() ? (uint32_t)kSplitGroups : 1u, slice = pd.esplit() ? (uint32_t)grp : 0u;
  const uint32_t share = ((uint32_t)(cl.uhi - cl.ulo) + parts - 1) / parts;
  const uint64_t u0 = min(cl.ulo + (uint64_t)part * share, cl.uhi);
  const uint32_t steps = (uint32_t)(min(u0 + share, cl.uhi) - u0);
  auto nearly = [&]() {
    if (row == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(near) : "memory");
  };
  int thr = cl.U - g + 1;  // record weights <= U: redundant weight < U - g + 1
  SplitQueue &wq = sh.queue[warp];

  // Up to date with the records of other warps and CTAs: the scheduler warp
  // keeps reading the best key and the finished flag into shared memory.  (A
  // load by each warp cost it 2 us a step: the value's first use waits for
  // the L2, which serves the one line to every warp of the grid.)
  auto take_up = [&]() {
    const uint64_t key = ~(uint64_t)*(volatile unsigned long long *)&sh.best_key;
    if (key != kNoKey) thr = min(thr, (int)key_weight(key) - g + 1);
    thr = (int)__reduce_min_sync(FULL, (unsigned)max(thr, 0));  // one value for the warp
  };
  auto finished = [&]() { return *(volatile int32_t *)&sh.finished; };
  auto note = [&](uint64_t best) {  // the warp's best key, if any lane has one
    if (__any_sync(FULL, best != kNoKey)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) best = min(best, (uint64_t)__shfl_xor_sync(FULL, (unsigned long long)best, o));
      if (lane == 0) record(sh.states, sh.aux, cl.pass, best);
      thr = min(thr, (int)key_weight(best) - g + 1);
    }
  };
  Stem<RW> x;
#pragma unroll
  for (int q = 0; q < RW; ++q) x.s[q] = 0;
  x.pos = StemPos{-1, 0, 0};

  if (pd.direct()) {
    // few codewords: one stem per warpgroup at a time, its tails over the 128
    // lanes, every weight exact (no table; before the first records most bounds would
    // pass the threshold anyway)
    nearly();
    if (l > 0 && steps) stem_start<P, R, W, DB>(x, mult, B, u0, k, t, l, ncl);
    // (one lane's read of the flag for the warp: it changes meanwhile, and the body's collectives take all lanes)
    for (uint32_t i = 0; i < steps && !__shfl_sync(FULL, finished(), 0); ++i) {
      if (l > 0 && i) stem_next<P, R, W, DB>(x, mult, l);
      const uint32_t E = min(nb, tails_above(B, k, t, b, x.pos.m) - first);
      take_up();
      for (uint32_t e0 = slice * kSplitGroup; e0 < E; e0 += kSplitGroup * slices) {
        const uint32_t e = e0 + row;
        uint64_t best = kNoKey;
        if (e < E) {
          const uint32_t tl = tails[e];
          int wp, wm;
          split_weights<P, R, W>(x.s, tail_unpack(tl), mult, wp, wm);
          if (wp < thr || (l > 0 && wm < thr))
            best = hit_key<DB>(B, pair, k, P, g, cl.pass, wp, wm, thr, x.pos, l, tl);
          ++seen;
        }
        note(best);
      }
    }
    return (unsigned long long)seen << (l > 0 ? 1 : 0);
  }

  const uint32_t tA = tmem + (uint32_t)grp * kTmemGroup, tD = tA + kTmemD;
  const uint32_t my_lanes = (uint32_t)(warp & 3) << 21;  // 32 lanes a warp, in the address's upper half
  const uint64_t J0 = u0 * kSplitGroup, J = J0 + (uint64_t)row * steps;  // a lane's run of stems
  const uint32_t nst = J < ns ? (uint32_t)min((uint64_t)steps, ns - J) : 0u;
  if (l > 0 && nst) stem_start<P, R, W, DB>(x, mult, B, J, k, t, l, ncl);
  // tails of the block above the run's first stem: as many tiles as any lane needs
  const int q0 = l > 0 && steps ? comb_floor(B, l - 1, k - t - 1, l, ncl, J0) : -1;
  const uint32_t tiles = (min(nb, tails_above(B, k, t, b, q0) - first) + kSplitN - 1) / kSplitN;
  // the same for the whole warpgroup: `lost` as of the close of an earlier task
  if (steps == 0 || slice >= tiles || *(volatile int32_t *)&sh.lost[grp]) {
    nearly();
    return 0;
  }
  int stop = 0;  // the code has finished, or (kLost) a product never came
  for (uint32_t i = 0; i < steps; ++i) {
    if (i + 1 == steps) nearly();
    const bool act = i < nst;
    take_up();
    {
      __syncwarp();
      uint32_t o[4], w[8];
      class_bits<P, R, W>(x.s, nu, o);
      const uint32_t marks = act ? stem_marks<P>(nu, thr) : kStemNone;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        if (32 * s >= K) break;
        class_bytes(o[s], w);
        if (32 * (s + 1) == K) w[7] = marks;
        tmem_store8(tA + my_lanes + 8 * s, w);
      }
      tmem_wait_store();
    }
    uint32_t n = 0;  // candidates in the warp's queue
    int thr_set = thr;  // the threshold in the rows' last words
    // exact weights of `cnt` candidates from `at`: a lane takes one and fetches the owner's stem
    auto check = [&](uint32_t at, uint32_t cnt) {
      __syncwarp();
      const bool have = (uint32_t)lane < cnt;
      const uint32_t item_ = have ? wq.item[at + lane] : 0u;
      const int src = (int)(item_ & 31u);
      uint32_t so[RW];
#pragma unroll
      for (int q = 0; q < RW; ++q) so[q] = __shfl_sync(FULL, x.s[q], src);
      const int qo = __shfl_sync(FULL, x.pos.m, src);
      const uint32_t tl = tails[item_ >> 5];
      const Tail a = tail_unpack(tl);
      int wp = 1 << 20, wm = 1 << 20;
      if (have && a.z > qo) split_weights<P, R, W>(so, a, mult, wp, wm);
      const bool hit = wp < thr || (l > 0 && wm < thr);
      if (__any_sync(FULL, hit)) {
        StemPos po;
        po.m = qo;
        po.Q = __shfl_sync(FULL, (unsigned long long)x.pos.Q, src);
        po.d = __shfl_sync(FULL, (unsigned long long)x.pos.d, src);
        note(hit ? hit_key<DB>(B, pair, k, P, g, cl.pass, wp, wm, thr, po, l, tl) : kNoKey);
      }
      __syncwarp();
    };
    // candidates of the lane's 96 results, those of sign 0, onto the queue:
    // a word of 32 bits per 32 results (low half: even columns), then one
    // candidate per lane and round
    auto scan = [&](const uint32_t (&v0)[16], const uint32_t (&v1)[16], const uint32_t (&v2)[16], uint32_t col0) {
      uint32_t m0 = 0, m1 = 0, m2 = 0;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        m0 = (m0 >> 1) | (~v0[q] & 0x80008000u);
        m1 = (m1 >> 1) | (~v1[q] & 0x80008000u);
        m2 = (m2 >> 1) | (~v2[q] & 0x80008000u);
      }
      unsigned any = __ballot_sync(FULL, (m0 | m1 | m2) != 0);
      do {
        if (m0 | m1 | m2) {
          const uint32_t m = m0 ? m0 : m1 ? m1 : m2, col = m0 ? 0u : m1 ? 32u : 64u;
          const int bit = fpenum::ctz32(m);
          const uint32_t less = m & (m - 1);
          if (m0) m0 = less;
          else if (m1) m1 = less;
          else m2 = less;
          wq.item[n + __popc(any & ((1u << lane) - 1u))] =
              (col0 + col + 2u * (uint32_t)(bit & 15) + (uint32_t)(bit >> 4)) << 5 | (uint32_t)lane;
        }
        n += __popc(any);
        any = __ballot_sync(FULL, (m0 | m1 | m2) != 0);
        if (n >= 32) {
          n -= 32;
          check(n, 32);
        }
      } while (any);
    };
    for (uint32_t c = slice; c < tiles && !stop; c += slices) {
      tc_before_sync();
      if ((warp & 3) == 0) {
        group_sync(1 + grp);
        tc_after_sync();
        if (elect_one()) {
          const uint64_t d0 = tile_desc(table + c * (uint32_t)(kSplitN * K), (uint32_t)K);
          mma_step<false>(tD, tA, d0, kSplitIdesc);
          if (K > 32) mma_step<true>(tD, tA + 8, d0 + 16, kSplitIdesc);
          if (K > 64) mma_step<true>(tD, tA + 16, d0 + 32, kSplitIdesc);
          if (K > 96) mma_step<true>(tD, tA + 24, d0 + 48, kSplitIdesc);
          mma_commit(mbar);
          // the product's barrier takes the commit and this release: who sees its
          // phase sees `stop` (written after the group's barrier, so of a warp
          // that has given up an earlier product too; ahead of that barrier the
          // release cost F_3 [74,50] 12 %)
          *(volatile int32_t *)&sh.stop[grp][parity] = finished() | *(volatile int32_t *)&sh.lost[grp];
          mbar_arrive(mbar);
        }
        __syncwarp();
      } else {
        group_arrive(1 + grp);
      }
      if (!__all_sync(FULL, mbar_wait(mbar, parity))) {
        stop = kLost;
        break;
      }
      stop = *(volatile int32_t *)&sh.stop[grp][parity];
      parity ^= 1u;
      tc_after_sync();
      uint32_t v0[16], v1[16], v2[16];
      tmem_load16(tD + my_lanes, v0);
      tmem_load16(tD + my_lanes + 32, v1);
      tmem_load16(tD + my_lanes + 64, v2);
      tmem_wait_load(v0, v1, v2);
      uint32_t a0 = ~0u, a1 = ~0u, a2 = ~0u;
#pragma unroll
      for (int q = 0; q < 16; q += 2) {
        a0 = and3(a0, v0[q], v0[q + 1]);
        a1 = and3(a1, v1[q], v1[q + 1]);
        a2 = and3(a2, v2[q], v2[q + 1]);
      }
      if (__any_sync(FULL, (~and3(a0, a1, a2) & 0x80008000u) != 0)) {
        scan(v0, v1, v2, c * kSplitN);
        take_up();
        if (thr < thr_set && c + slices < tiles) {  // a lower bound since: into the rows, for the step's other tiles
          thr_set = thr;
          const uint32_t marks = act ? stem_marks<P>(nu, thr) : kStemNone;
          __syncwarp();
          asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(tA + my_lanes + (uint32_t)(K / 4 - 1)), "r"(marks)
                       : "memory");
          tmem_wait_store();
        }
      }
    }
    if (n) check(0, n);
    if (act) {
      // this lane's tails, in the slice's tiles
      const uint32_t above = tails_above(B, k, t, b, x.pos.m);
      const uint32_t E = above > first ? min(nb, above - first) : 0u;
      const uint32_t full = E / kSplitN, rest = E - full * kSplitN;  // whole tiles, then part of one
      const uint32_t mine = full > slice ? (full - slice + slices - 1) / slices : 0u;
      const uint32_t tailn = mine * kSplitN + (full % slices == slice ? rest : 0u);
      seen += tailn;
    }
    if (stop) {
      if (i + 1 < steps) nearly();
      break;
    }
    if (i + 1 < nst) stem_next<P, R, W, DB>(x, mult, l);
  }
  if (stop == kLost) {
    // This warp gives the product up.  The others of its group may have seen
    // it in time: they get this warp's part in one more product (the named
    // barrier's arrival; from the issuing warp the end of the product's phase)
    // and leave by `stop` at the latest then.  No warp waits for this one but
    // at the close, which all four come to whichever way.
    if (lane == 0) {
      *(volatile int32_t *)&sh.lost[grp] = 1;
      *(volatile int32_t *)&sh.lost_any = 1;
      atomicExch(&sh.cdyn->err, 1);
      if ((warp & 3) == 0) {
        *(volatile int32_t *)&sh.stop[grp][0] = 1;
        *(volatile int32_t *)&sh.stop[grp][1] = 1;
        mbar_arrive(mbar);
        mbar_arrive(mbar);
      }
    }
    __syncwarp();
    if ((warp & 3) != 0) group_arrive(1 + grp);
  }
  group_sync(kCloseBar + grp);  // the close: after it, all four warps know of a loss (`lost`)
  return (unsigned long long)seen << (l > 0 ? 1 : 0);
}

__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 5, %0;" ::"n"(kSplitThreads) : "memory"); }

// The kernel: claims, counts and termination tests follow bz_kernel's
// protocol on the same state.  One code per launch.  Sixteen warps work; one
// more claims: it hands out the next task when the running one
// nears its end and counts the finished one off while the next runs (in
// bz_kernel, where thread 0 does both between tasks, a hand-off holds the
// CTA for about 4 us, a tenth to a third of these searches).  Claiming only
// near the end keeps the tasks of a pass's end with the CTAs that are free.
template <int P, int R, int W>
__global__ void __launch_bounds__(kSplitLaunch, 1)
    split_kernel(const SlotDesc *__restrict__ slots, SlotState *states, const CtlStatic *__restrict__ ctl, CtlDyn *cdyn,
                 KParams kp) {
  extern __shared__ uint4 smem_raw[];
  char *smem = reinterpret_cast<char *>(smem_raw);
  uint64_t *bcols = reinterpret_cast<uint64_t *>(smem_raw);
  __shared__ ClaimCache s_cc;
  __shared__ SegCache<kSplitSegCache, SplitSeg> s_sc;
  __shared__ __align__(16) PassDesc s_pc[kSplitPassCache];
  __shared__ SplitShared s_sh;
  __shared__ uint32_t s_tmem;

  const CtlStatic cs = *ctl;
  const int tid = threadIdx.x, threads = kSplitLaunch;
  const unsigned long long t_start = globaltimer();
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  // longest wait for another warp: past every bounded wait of the claims
  const unsigned long long wait_ns = 2 * kp.wait_limit_ns + 60000000000ull;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    // (a test has the first warpgroup wait for an arrival that nobody makes)
    for (int i = 0; i < kSplitGroups; ++i) mbar_init(smem_u32(&s_sh.product[i]), kp.lose && i == 0 ? 3 : 2);
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&s_sh.full[i]), 1);
      mbar_init(smem_u32(&s_sh.near[i]), kSplitGroups);
      mbar_init(smem_u32(&s_sh.done[i]), kSplitWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_sh.over = s_sh.lost_any = 0;
    for (int i = 0; i < kSplitGroups; ++i) s_sh.lost[i] = 0;
    s_sh.best_key = 0;
    s_sh.finished = 0;
    s_sh.states = states;
    s_sh.aux = cs.aux;
    s_sh.cdyn = cdyn;
    s_cc.sd = load_nc(&slots[0]);  // one thread per CTA, through L1: every CTA reads the same bytes at once
    s_cc.slot = 0;
    s_cc.gen = s_cc.sd.seq & kGenMask;
    s_cc.P = -1;
    s_cc.sleep_ns = 128;
    s_cc.busy_note = 0;
    s_sc.slot = -1;
    s_sc.pass = -1;
    s_sc.gen = 0;
  }
  {
    const uint4 *bsrc = reinterpret_cast<const uint4 *>(cs.binom->cols);
    for (int i = tid; i < kBinomBytes / 16; i += threads) smem_raw[i] = __ldg(bsrc + i);
  }
  const fpenum::BinomCols binom{bcols};
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = s_tmem;
  if (blockIdx.x == 0 && tid == 0 && s_cc.sd.pass_times) s_cc.sd.pass_times[kMaxPasses] = t_start;  // launch start
  const int np = s_cc.sd.npasses;
  const int npc = np < kSplitPassCache ? np : kSplitPassCache;
  {
    // pass descriptors and segments: nothing in the launch writes them
    const uint4 *src = reinterpret_cast<const uint4 *>(s_cc.sd.passes);
    for (int i = tid; i < npc * (int)(sizeof(PassDesc) / 16); i += threads) reinterpret_cast<uint4 *>(s_pc)[i] = __ldg(src + i);
    const int nsegs = s_cc.sd.nsegs;
    if (nsegs > 0 && nsegs <= kSplitSegCache) {
      const uint4 *ssrc = reinterpret_cast<const uint4 *>(s_cc.sd.passes + np);
      for (int i = tid; i < nsegs; i += threads) reinterpret_cast<uint4 *>(s_sc.seg)[i] = __ldg(ssrc + i);
      if (tid == 0) {
        s_sc.slot = 0;
        s_sc.gen = s_cc.sd.seq & kGenMask;
        s_sc.pass = -2;
      }
    }
  }
  __syncthreads();
  if (warp >= kSplitWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (tid == kSplitThreads) {
      // what the tables hold: the set, the block (tail length and size, index) and how much of it
      int rr = 0, staged_j = -1, built = -1, built_n = 0;
      unsigned int built_block = 0;
      unsigned long long wait_t0 = 0;
      if (np > 0) {
        s_cc.pd = s_pc[0];
        s_cc.P = 0;
      }
      uint32_t head = 0, tail = 0;  // tasks handed out, tasks counted off
      unsigned long long since = 0;  // when the scheduler began to wait for a running task
      bool over = false, stuck = false;
      for (;;) {
        if (!over && head - tail < 2) {
          // one task runs: the next is claimed once its warpgroups are in their last steps
          const uint32_t r = (head - 1) & 1u, rp = ((head - 1) >> 1) & 1u;
          if (head == tail || mbar_test(smem_u32(&s_sh.near[r]), rp) || mbar_test(smem_u32(&s_sh.done[r]), rp)) {
            SplitTask &tk = s_sh.task[head & 1u];
            if (head != tail) s_cc.sleep_ns = 128;  // a finished task must not wait for the back-off
            const int cmd = claim(slots, states, cs, kp, cdyn, rr, wait_t0, t_start, &tk.cl, s_cc, s_sc, s_pc, npc, binom);
            if (cmd == kCmdExit) {
              over = true;
            } else if (cmd == kCmdRun) {
              tk.pd = s_cc.pd;
              tk.cmd = kCmdRun;
              tk.count = 0;
              tk.stage = tk.build = tk.drop = 0;
              if (!tk.cl.skip) {
                // a direct pass needs the packed tails only, which a built table of the same block has too
                const int need = tk.pd.g < 2 ? 0 : tk.pd.direct() ? 1 : 2, bt = tk.pd.tail_rows() << 16 | (int)tk.pd.block();
                tk.stage = staged_j != tk.pd.j;
                if (need && (tk.stage || built != bt || built_block != tk.cl.block || built_n < need)) {
                  tk.build = need;
                  built = bt;
                  built_block = tk.cl.block;
                  built_n = need;
                } else if (tk.stage) {
                  built = -1;
                }
                staged_j = tk.pd.j;
              }
              mbar_arrive(smem_u32(&s_sh.full[head & 1u]));
              ++head;
              continue;
            }
          }
        }
        if (head == tail) {
          if (over) break;
          continue;
        }
        const uint32_t o = tail & 1u, op = (tail >> 1) & 1u;
        {  // pass on the best key and the finished flag (the loads pace this loop)
          const unsigned long long key = ld_vol(&states[0].best_key);
          const int fin = ld_vol(&states[0].finished);
          *(volatile unsigned long long *)&s_sh.best_key = key;
          *(volatile int32_t *)&s_sh.finished = fin;
        }
        if (mbar_test(smem_u32(&s_sh.done[o]), op)) {
          const SplitTask &tk = s_sh.task[o];
          // A lost product: some of the task's codewords were never compared.
          // It is not counted off, so its pass never counts as complete and
          // the search ends as a timeout, unless an earlier pass certifies.
          if (*(volatile int32_t *)&s_sh.lost_any) break;
          if (tk.count) {
            atomicAdd(&states[0].enumerated, tk.count);
            atomicAdd(&cs.aux->pass_count[tk.cl.pass], tk.count);
          }
          if (finish_task(cs, kp, cdyn, s_cc.sd, &states[0], cs.aux, 0, tk.cl.pass, tk.pd, tk.cl.ndone, s_pc, npc))
            over = true;
          ++tail;
          since = 0;
        } else if (since == 0) {
          since = globaltimer();
        } else if (globaltimer() - since > wait_ns) {
          atomicExch(&cdyn->err, 1);  // a warp never finished: report a timeout
          stuck = true;
          break;
        } else {
          __nanosleep(200);  // the issue slots belong to the warps that work
        }
      }
      if (stuck && head - tail == 2) {  // both buffers hold tasks that are not counted off
        *(volatile int32_t *)&s_sh.over = 1;
      } else {
        s_sh.task[head & 1u].cmd = kCmdExit;
        mbar_arrive(smem_u32(&s_sh.full[head & 1u]));
      }
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const SlotDesc &sd = s_cc.sd;
    uint32_t *mult = reinterpret_cast<uint32_t *>(smem + kBinomBytes);
    uint32_t *tails = reinterpret_cast<uint32_t *>(smem + split_off_tails(sd.k, P, sd.rwpad));
    char *table = smem + split_off_table(sd.k, P, sd.rwpad, sd.split_cap());
    uint32_t parity = 0;
    for (uint32_t n = 0;; ++n) {
      const int b = (int)(n & 1u);
      SplitTask &tk = s_sh.task[b];
      // the next task: the scheduler's waits are bounded, and it ends by an exit
      // command or, where no buffer is free for one, by `over` (with nothing
      // handed out after it: the warps leave at the same task)
      bool have = false;
      for (uint32_t r = 0; !have && r < (1u << 31); ++r) {
        const bool over = *(volatile int32_t *)&s_sh.over;
        have = __all_sync(0xffffffffu, mbar_test(smem_u32(&s_sh.full[n & 1u]), (n >> 1) & 1u));
        if (__any_sync(0xffffffffu, over)) break;
      }
      if (!have) break;
      if (tk.cmd == kCmdExit) break;
      if (tk.stage || tk.build) {
        if (tid == 0) tk.drop = *(volatile int32_t *)&s_sh.finished;
        workers_sync();  // every warp has left the previous task: its tables may go
        if (tk.stage && !tk.drop) {
          const int nv = split_mult_words(sd.k, P, sd.rwpad) / 4;
          const uint4 *src = reinterpret_cast<const uint4 *>(sd.table + (size_t)tk.pd.j * (size_t)table_words(sd));
          for (int i = tid; i < nv; i += kSplitThreads) reinterpret_cast<uint4 *>(mult)[i] = __ldg(src + i);
          workers_sync();
        }
        if (tk.build && !tk.drop) {
          const uint32_t etot = tails_above(binom, sd.k, tk.pd.tail_rows(), P - 1, -1), first = tk.cl.block * tk.pd.block();
          build_tails<P, R, W>(tails, table, mult, binom, sd.k, tk.pd.tail_rows(), first, min(tk.pd.block(), etot - first),
                               sd.split_k(), sd.split_nu(), tk.build == 2);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tensor cores read the table
          workers_sync();
        }
      }
      unsigned long long count = 0;
      if (tk.cl.skip || tk.drop || tk.pd.g == 1) {
        if ((tid & (kSplitGroup - 1)) == 0) mbar_arrive(smem_u32(&s_sh.near[b]));
        if (!tk.cl.skip && !tk.drop && tk.cl.ulo == 0) task_rows<P, R, W>(sd, tk.cl.pass, mult, tk.cl.U, &states[0], cs.aux, count);
      } else {
        count = task_split<P, R, W>(sd, s_sh, b, mult, tails, smem_u32(table), tmem, parity, binom);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
      __syncwarp();  // lane 0 arrives for the records of all lanes
      if ((tid & 31) == 0) {
        if (count) atomicAdd(&tk.count, count);
        mbar_arrive(smem_u32(&s_sh.done[b]));
      }
    }
  }
  if (*(volatile int32_t *)&s_sh.lost_any)  // a product may still be under way: a millisecond for it before the tensor memory goes
    for (int i = 0; i < 1000; ++i) __nanosleep(1000);
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  leave_launch(states, cs, cdyn);
}

}  // namespace fpk
