// fp_split.cuh -- split enumeration of a pass for the tensor-core kernel.
//
// A codeword of pass g with rows T splits into its t largest rows (the
// tail, z < y < x or z < x, coefficient of z fixed to 1) and the others
// (the stem, l = g - t rows, largest row q < z, coefficient of q in
// [1, (p-1)/2]).  Every projective class is met once as stem + tail or
// stem - tail (l = 0: one empty stem, tails alone).
//
// Tails are numbered by z descending, so the tails with z > q come first:
//   t = 2: z descending, x ascending, c_x ascending;
//   t = 3: z descending, y descending, c_y ascending, x ascending, c_x.
// They are cut into blocks of PassDesc::block() entries, one block of which a
// CTA holds in shared memory at a time.  Stems of a block are those with q
// below the z of its first tail, numbered by q ascending, then by the
// revolving-door rank of the other rows, then by the reflected Gray code of
// the coefficients (q's the most significant digit), so that the stems of
// any block are a prefix of one sequence.
//
// The recorded keys are those of the code's leaf form (fp_types.h): the
// split is how a pass is walked, not what it reports.
#pragma once
#include "fp_enum.cuh"
#include "fp_types.h"

namespace fpk {

// One run of tasks of a split pass: units [item0, item1) of one tail block,
// `per` to a task.  A unit is 128 stems (tensor-core passes) or one stem
// (direct passes).  The four warpgroups of a CTA share a task's units
// evenly, or (esplit) all take the same units and interleaved slices of the
// block's tails.
struct SplitSeg {
  uint32_t task_end;  // tasks of the pass up to the end of this run
  uint32_t item0, item1;
  uint16_t per;
  uint8_t block;
  uint8_t zhi;        // z of the block's first tail (l >= 1: stems have q < zhi)
};
static_assert(sizeof(SplitSeg) == 16, "SplitSeg layout");

// Runs of one pass at most (the kernel's copy of the runs of the pass it
// claims from, when a code has too many to keep them all).
constexpr int kSplitPassSegs = 192;

// Units [lo, hi) of task t of a split pass whose runs are seg[0 .. nseg);
// returns the run.
FPK_HD SplitSeg split_task(const SplitSeg *seg, int nseg, uint64_t t, uint64_t *lo, uint64_t *hi) {
  int a = 0, z = nseg - 1;
  while (a < z) {
    const int mid = (a + z) >> 1;
    if (seg[mid].task_end > t) z = mid;
    else a = mid + 1;
  }
  const SplitSeg g = seg[a];
  const uint32_t i = (uint32_t)t - (a > 0 ? seg[a - 1].task_end : 0u);
  const uint32_t l = g.item0 + i * g.per;
  *lo = l;
  *hi = l + g.per < g.item1 ? l + g.per : g.item1;
  return g;
}

constexpr int kSplitGroups = 4;     // warpgroups that work in a CTA (one more warp claims)
constexpr int kSplitGroup = 128;    // their lanes: rows of one accumulator tile
constexpr int kSplitThreads = kSplitGroups * kSplitGroup;
constexpr int kSplitLaunch = kSplitThreads + 128;  // with the claiming warp's warpgroup
constexpr int kSplitN = 96;         // tails per accumulator tile

// (p-1)^(t-1) coefficient vectors per tail subset.
FPK_HD uint32_t tail_coefs(int t, int b) { return t == 3 ? (uint32_t)(b * b) : (uint32_t)b; }

// Tails whose smallest row lies above q (q = -1: all).
template <class BT>
FPK_HD uint32_t tails_above(const BT &B, int k, int t, int b, int q) {
  return tail_coefs(t, b) * (uint32_t)B(k - 1 - q, t);
}

struct Tail {
  int z, y, x, cy, cx;  // t = 2: y = z, cy = 0
};

// Tail <-> 24 bits: rows of 6 bits, coefficients of 3 (p <= 7).
FPK_HD uint32_t tail_pack(const Tail &a) {
  return (uint32_t)a.z | (uint32_t)a.y << 6 | (uint32_t)a.x << 12 | (uint32_t)a.cy << 18 | (uint32_t)a.cx << 21;
}
FPK_HD Tail tail_unpack(uint32_t v) {
  return Tail{(int)(v & 63u), (int)(v >> 6 & 63u), (int)(v >> 12 & 63u), (int)(v >> 18 & 7u), (int)(v >> 21 & 7u)};
}

// Largest m in [lo, hi] with f C(m, t) <= e (C(lo, t) = 0).
template <class BT>
FPK_HD int comb_floor(const BT &B, int lo, int hi, int t, uint64_t f, uint64_t e) {
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (f * B(mid, t) <= e) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <class BT>
FPK_HD Tail tail_unrank(const BT &B, uint32_t e, int k, int t, int b) {
  Tail a;
  const uint32_t bt = tail_coefs(t, b);
  const int m = comb_floor(B, t - 1, k - 1, t, bt, e);  // rows above z
  uint32_t s = e - bt * (uint32_t)B(m, t);
  a.z = k - 1 - m;
  if (t == 2) {
    const uint32_t xi = s / (uint32_t)b;
    a.y = a.z;
    a.cy = 0;
    a.x = a.z + 1 + (int)xi;
    a.cx = (int)(s - xi * (uint32_t)b) + 1;
    return a;
  }
  const int my = comb_floor(B, 1, m - 1, 2, bt, s);  // rows above y
  s -= bt * (uint32_t)B(my, 2);
  a.y = k - 1 - my;
  const uint32_t w = (uint32_t)(my * b), c = s / w;
  s -= c * w;
  a.cy = (int)c + 1;
  const uint32_t xi = s / (uint32_t)b;
  a.x = a.y + 1 + (int)xi;
  a.cx = (int)(s - xi * (uint32_t)b) + 1;
  return a;
}

// The next tail; returns true when the part without x (z, y, c_y) changed.
FPK_HD bool tail_next(Tail &a, int k, int t, int b) {
  if (a.cx < b) {
    ++a.cx;
    return false;
  }
  a.cx = 1;
  if (a.x < k - 1) {
    ++a.x;
    return false;
  }
  if (t == 2) {
    --a.z;
    a.y = a.z;
    a.x = a.z + 1;
    return true;
  }
  if (a.cy < b) {
    ++a.cy;
  } else {
    a.cy = 1;
    if (a.y > a.z + 1) {
      --a.y;
    } else {
      --a.z;
      a.y = k - 2;
    }
  }
  a.x = a.y + 1;
  return true;
}

// A stem: its largest row, the mask of the other l - 1 rows, and the packed
// counter digits of all l coefficients (slot l - 1: the largest row).  The
// next stem follows from these alone (no ranks are kept: a lane of the
// kernel holds its stem in few registers).
struct StemPos {
  int m;
  uint64_t Q, d;
};

// Stem of index J; ncl = (b/2) b^(l-1) coefficient vectors per row subset.
template <int DB, class BT>
FPK_HD StemPos stem_unrank(const BT &B, uint64_t J, int k, int t, int l, int b, uint64_t ncl) {
  StemPos P;
  P.m = comb_floor(B, l - 1, k - t - 1, l, ncl, J);
  const uint64_t rem = J - ncl * B(P.m, l);
  uint64_t qi, ci;
  if constexpr (DB == 1) {
    qi = rem >> (l - 1);
    ci = rem & (ncl - 1);
  } else if ((rem | ncl) >> 32) {
    qi = rem / ncl;
    ci = rem - qi * ncl;
  } else {
    qi = (uint32_t)rem / (uint32_t)ncl;
    ci = (uint32_t)rem - (uint32_t)qi * (uint32_t)ncl;
  }
  P.Q = fpenum::rd_unrank(B, qi, P.m, l - 1);
  if constexpr (DB == 1) {
    P.d = ci;
  } else if (ci >> 32) {
    P.d = fpenum::counter_digits<DB>(ci, b, l);
  } else {
    P.d = 0;
    uint32_t c = (uint32_t)ci;
    for (int s = 0; s < l; ++s) {
      P.d |= (uint64_t)(c % (uint32_t)b) << (s * DB);
      c /= (uint32_t)b;
    }
  }
  return P;
}

// The last counter value of a row subset: digits b - 1, the top one b/2 - 1.
template <int DB>
FPK_HD uint64_t stem_last(int b, int l) {
  const int top = DB * (l - 1);
  const uint64_t all = DB == 1 ? ~0ull : 0x1111111111111111ull * (uint64_t)(b - 1);
  return (all & fpenum::low_mask(top)) | (uint64_t)(b / 2 - 1) << top;
}

// Next stem: the slot whose coefficient changed by *dir, or -1 when the row
// subset changed (all coefficients back to 1).
template <int DB>
FPK_HD int stem_advance(StemPos &P, int b, int l, int *dir) {
  if (P.d != stem_last<DB>(b, l)) return fpenum::gray_step<DB>(&P.d, b, l, dir);
  P.d = 0;
  uint64_t nQ = P.Q;
  int rm = 0, ad = 0;
  if (fpenum::rd_next(P.Q, P.m, l - 1, &nQ, &rm, &ad)) {
    P.Q = nQ;
  } else {
    ++P.m;
    P.Q = fpenum::low_mask(l - 1);
  }
  return -1;
}

// Packed key, in the code's leaf form, of the codeword stem + tail (sign 0)
// or stem - tail (sign 1) of pass `pass`: `pair` is the form (true: stem
// index and pair entry; false: prefix index, leaf row and coefficient).
template <int DB, class BT>
FPK_HD uint64_t split_key(const BT &B, bool pair, int k, int p, int g, uint32_t pass, uint32_t weight,
                          const StemPos &P, int l, const Tail &a, int sign) {
  const int b = p - 1;
  int row[fpenum::kBinomCols], c[fpenum::kBinomCols];
  int n = 0;
  uint64_t Q = P.Q;
  for (int s = 0; s + 1 < l; ++s) {
    row[n] = fpenum::ctz64(Q);
    Q &= Q - 1;
    c[n++] = fpenum::gray_digit<DB>(P.d, s, b, l) + 1;
  }
  if (l > 0) {
    row[n] = P.m;
    c[n++] = fpenum::gray_digit<DB>(P.d, l - 1, b, l) + 1;
  }
  row[n] = a.z;
  c[n++] = sign ? b : 1;
  if (a.cy) {
    row[n] = a.y;
    c[n++] = sign ? p - a.cy : a.cy;
  }
  row[n] = a.x;
  c[n++] = sign ? p - a.cx : a.cx;
  // scale so that the second-largest row has coefficient 1
  int inv = 1;
  while (c[g - 2] * inv % p != 1) ++inv;
  for (int i = 0; i < g; ++i) c[i] = c[i] * inv % p;
  const int cx = c[g - 1];
  int neg = 0;
  const int L = pair ? g - 3 : g - 2;  // rows with a digit of the coefficient counter
  if (pair && g >= 3 && c[g - 3] > b / 2) {  // the stem's largest row has its coefficient in [1, (p-1)/2]
    neg = 1;
    for (int i = 0; i < g; ++i) c[i] = p - c[i];
  }
  uint64_t ci = 0, R = 0, NC = 1;
  int up = 0;
  for (int s = L - 1; s >= 0; --s) {
    const int e = c[s] - 1, d = (up & 1) ? b - 1 - e : e;
    ci = ci * (uint64_t)b + (uint64_t)d;
    up = d;
    R |= 1ull << row[s];
    NC *= (uint64_t)b;
  }
  if (pair) {
    const int y = row[g - 2], x = row[g - 1], ty = k - 1 - y;
    const uint32_t e = (uint32_t)b * (uint32_t)(ty * (ty - 1) / 2 + (x - y - 1)) + (uint32_t)(cx - 1);
    uint64_t J = 0;
    if (g >= 3) {
      const int q = row[g - 3];
      J = (uint64_t)(c[g - 3] - 1) * B(k - 2, g - 2) * NC + B(q, g - 2) * NC + fpenum::rd_rank(B, R, q, L) * NC + ci;
    }
    return make_pair_key(weight, pass, J, e, (uint32_t)neg);
  }
  const int m = row[g - 2];
  const uint64_t I = B(m, g - 1) * NC + fpenum::rd_rank(B, R, m, L) * NC + ci;
  return make_key(weight, pass, I, (uint32_t)row[g - 1], (uint32_t)cx);
}

// ---------------------------------------------------------------------------
// Class comparison on the tensor cores.  The symbols of F_p fall into the
// classes {c, -c}: S + B and S - B are both nonzero at a position exactly
// where S and B are of different classes, so the positions that differ
// bound both weights from below (the pair bound of the isometric last
// addition, Sec. 4.3).  With a class written as +-1 values whose inner
// product is `kSame` for equal classes and -1 otherwise (p = 3: one value;
// p = 5, 7: three, the characters of a group of four), the bound lb over nu
// positions is (kSame nu - <S, B>) / (kSame + 1).
// ---------------------------------------------------------------------------
template <int P>
struct ClassCode {
  static constexpr int kVals = P == 3 ? 1 : 3;
  static constexpr int kSame = kVals;
};
FPK_HD int class_vals(int p) { return p == 3 ? 1 : 3; }

// K (values per row, a multiple of 32) and positions compared for n - k = N
// redundant symbols; K = 0: the code does not fit.  Four values of the last
// word hold the threshold and the padding mark.  A comparison of fewer
// positions is a weaker bound: one position in 32 is left out where that
// saves 32 values a row, no more (F_7 [52,19] at 30 of 33 positions: 43 % of
// a warp's tiles held a candidate, and their exact checks cost more than the
// shorter rows saved).
FPK_HD int split_k(int p, int N, int *nu) {
  const int v = class_vals(p);
  int K = (v * N + 4 + 31) / 32 * 32;
  *nu = N;
  const int fit = (K - 32 - 4) / v;  // positions that 32 values fewer hold
  if (K > 32 && fit < N && (N - fit) * 32 <= N) {
    K -= 32;
    *nu = fit;
  }
  return K <= 128 ? K : 0;
}

// Shared memory of a CTA: the binomial columns, one set's multiples, the
// packed tails of a block, then (128-byte aligned) their K class values.
constexpr int kSplitBinomBytes = fpenum::kBinomCols * (fpenum::kMaxK + 1) * 8;
FPK_HD int split_mult_words(int k, int p, int rwpad) { return k * (p - 1) * rwpad; }
FPK_HD int split_off_tails(int k, int p, int rwpad) {
  return kSplitBinomBytes + (split_mult_words(k, p, rwpad) * 4 + 15) / 16 * 16;
}
FPK_HD int split_off_table(int k, int p, int rwpad, int cap) {
  return (split_off_tails(k, p, rwpad) + cap * 4 + 127) / 128 * 128;
}
FPK_HD int split_smem(int k, int p, int rwpad, int cap, int K) {
  const int block = split_off_table(k, p, rwpad, cap) + cap * K;
  const int direct = split_off_tails(k, p, rwpad) + (p - 1) * (k * (k - 1) / 2) * 4;  // packed tails of two rows alone
  return block > direct ? block : direct;
}

}  // namespace fpk
