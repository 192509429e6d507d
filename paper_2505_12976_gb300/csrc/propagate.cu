// Winners only, by the paper's vertex-centric algorithm (Sect. 4, Alg. 1-4),
// restated on the dense tally for one GPU: a comparator for the closure
// path. Every candidate c keeps a status (unknown / loser / winner); each
// iteration of the while-loop
//   * preprocessing (Alg. 2): unknown c starts as its own source and target
//     (s = t = c, widths "infinite"), decided ones as relays (s = t = none);
//   * forward-backward propagation (Alg. 3), in synchronous rounds until
//     nothing changes: c keeps the smallest source id reaching it and, for
//     that id, the widest width over its incoming edges (u, c) of
//     min(width at u, w(u, c)); likewise the smallest target id it reaches
//     and the widest width, against the edges;
//   * postprocessing (Alg. 4): loser marks from s < t, s > t, the widths of a
//     found SCC, and incoming edges from another SCC; then the unknown c with
//     s = t = c become winners.
// Readings: a decided status never changes (marks only turn unknown into
// loser); the optional zeroing of edges into dominated SCCs is left out.
//
// Edge weights come from d on the fly: with a = d[c][u] and b = d[u][c],
// the outgoing edge (c, u) weighs a if a > b (a - b with margins) and the
// incoming edge (u, c) weighs b if b > a. A pass takes pairs of 64 x 64
// blocks (A, B) and (B, A) of d, each read once, and serves the candidates of
// both; a side of a pair whose sources cannot give anything new (propagation:
// nothing changed in the round before) or whose targets nobody asks about
// (marks) is left out, and a pair without a side is not read. So a round that
// starts at a few unknown candidates touches their rows and columns only, and
// one in which everything changed reads d once. On m = 18407 (top-200 lists)
// the two iterations took 6.3 ms with a transposed copy of d and two rows
// per candidate read in every pass, 1.2 ms in this form.
#include <algorithm>

#include "internal.cuh"

namespace schulze {
namespace {

constexpr int32_t kNone = 0x7fffffff;  // no id / infinite width
constexpr int32_t kUnknown = 0, kLoser = 1, kWinner = 2;
constexpr int kPT = 64;  // block size

__device__ __forceinline__ int32_t edge(int32_t x, int32_t y, int margin) {
  return x > y ? (margin ? x - y : x) : 0;
}

// (id, width) with the smallest id first and, for equal ids, the widest
// width first, as one 64-bit key (smaller is better): a candidate's source
// (f) and target (b). No id: key(kNone, 0), above every other key.
using Key = unsigned long long;
__device__ __forceinline__ Key key(int32_t id, int32_t width) {
  return (Key(uint32_t(id)) << 32) | Key(0xFFFFFFFFu - uint32_t(width));
}
__device__ __forceinline__ int32_t key_id(Key k) { return int32_t(k >> 32); }
// the key carried along an edge of weight w: the same id, the smaller width
__device__ __forceinline__ Key along(Key k, int32_t w) {
  return (k & 0xFFFFFFFF00000000ull) | Key(max(uint32_t(k), 0xFFFFFFFFu - uint32_t(w)));
}

enum Pass : int { kInit = 0, kPropagate = 1, kMarks = 2 };
struct PassArgs {
  const int32_t* d;
  int32_t m, margin;
  int32_t *in, *out;        // kInit: heaviest incoming / outgoing edge (zeroed before)
  const int32_t* flag;      // per block of 64: kPropagate: a key changed; kMarks: asked about
  const Key *f, *b;         // keys
  Key *fn, *bn;             // kPropagate: the next round's (start as f and b)
  int32_t* changed;         // kPropagate: cleared here, set by commit_kernel
  const int32_t* asked;     // kMarks: candidates asked about
  const int4* label;        // kMarks: per block its first candidate's ids (x, y), z: all share them
  int32_t *lose, *scc_lose;  // kMarks
  int32_t* status;          // rows_kernel: kInit sets it, kMarks reads it
};

// One pass over the pairs of blocks; a thread holds four columns of four rows
// of d[A..][B..] and of d[B..][A..], their transposed partners are in shared
// memory. kVec (rows on 16-byte boundaries): the columns are neighbours, one
// 16-byte load. Else they lie 16 apart, so that each 4-byte load of a
// half-warp covers 64 neighbouring bytes: with neighbours there too, every
// sector went through L1 four times (m = 18407, a full round 318 -> 309 us).
// A round is bound by its compares as much as by d: one 64-bit compare per
// entry instead of two 309 -> 276 us, four CTAs per SM instead of three (at
// the price of a few spilled words) 256 us.
template <int kPass, bool kVec>
__global__ void __launch_bounds__(256, 4) pair_kernel(PassArgs g) {
  if (kPass == kPropagate && blockIdx.x == 0 && threadIdx.x == 0) *g.changed = 0;
  const int32_t m = g.m, nbt = (m + kPT - 1) / kPT;
  int32_t a = 0;
  int64_t rem = blockIdx.x;  // pair (a, a + rem), numbered row by row
  {
    const float x = float(nbt) + 0.5f;  // a from the triangular numbering, then corrected (FP64 is slow here)
    a = max(0, min(nbt - 1, int32_t(x - sqrtf(max(0.f, x * x - 2.f * float(rem))))));
    auto first = [&](int64_t r) { return r * nbt - r * (r - 1) / 2; };
    while (a > 0 && first(a) > rem) --a;
    while (a + 1 < nbt && first(a + 1) <= rem) ++a;
    rem -= first(a);
  }
  const int32_t bt = a + int32_t(rem), A = a * kPT, B = bt * kPT;
  // side 0: targets in A, sources in B; side 1: the other way round
  bool s0 = true, s1 = A != B;
  if (kPass == kPropagate) s0 = g.flag[bt] != 0, s1 = s1 && g.flag[a] != 0;
  if (kPass == kMarks) {
    // blocks of one and the same label hold no edge from another SCC
    const bool same = g.label[a].z && g.label[bt].z && g.label[a].x == g.label[bt].x && g.label[a].y == g.label[bt].y;
    s0 = g.flag[a] != 0 && !same, s1 = s1 && g.flag[bt] != 0 && !same;
  }
  if (!s0 && !s1) return;
  __shared__ int32_t t1[kPT][kPT + 1], t2[kPT][kPT + 1];  // t1 = d[A.., B..], t2 = d[B.., A..]
  __shared__ Key sf[2][kPT], sb[2][kPT];                  // keys of A, of B
  const int lane = threadIdx.x & 31;
  constexpr int kCs = kVec ? 1 : 16;
  const int rq = threadIdx.x >> 4, c0 = (threadIdx.x & 15) * (kVec ? 4 : 1);  // rows rq + 16 q, columns c0 + kCs e
  int32_t x1[4][4], x2[4][4];
  auto load = [&](int32_t R, int32_t C, int32_t (&x)[4][4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int32_t i = R + rq + 16 * q, j = C + c0;
      if (kVec) {
        int4 v = make_int4(0, 0, 0, 0);
        if (i < m && j < m) v = __ldcs(reinterpret_cast<const int4*>(g.d + int64_t(i) * m + j));
        x[q][0] = v.x, x[q][1] = v.y, x[q][2] = v.z, x[q][3] = v.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) x[q][e] = (i < m && j + kCs * e < m) ? __ldcs(g.d + int64_t(i) * m + j + kCs * e) : 0;
      }
    }
  };
  load(A, B, x1);
  if (A != B) load(B, A, x2);
  if (kPass == kInit && threadIdx.x < 2 * kPT) {  // what the candidates have by now (it only grows)
    const int side = threadIdx.x / kPT, t = threadIdx.x % kPT;
    const int32_t c = (side ? B : A) + t;
    sf[side][t] = c < m ? Key(__ldcg(g.in + c)) : 0, sb[side][t] = c < m ? Key(__ldcg(g.out + c)) : 0;
  }
  if (kPass != kInit && threadIdx.x < 2 * kPT) {
    const int side = threadIdx.x / kPT, t = threadIdx.x % kPT;
    const int32_t c = (side ? B : A) + t;
    sf[side][t] = c < m ? g.f[c] : key(kNone, 0), sb[side][t] = c < m ? g.b[c] : key(kNone, 0);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      t1[rq + 16 * q][c0 + kCs * e] = x1[q][e];
      if (A != B) t2[rq + 16 * q][c0 + kCs * e] = x2[q][e];
    }
  __syncthreads();
  // targets T + r of tile side ts (their d rows in x), sources S + c (their d rows in `other`)
  auto serve = [&](int32_t T, int ts, int ss, const int32_t (&x)[4][4], const int32_t(*other)[kPT + 1]) {
    Key uf[4], ub[4];  // the keys of this thread's sources
    if (kPass != kInit) {
#pragma unroll
      for (int e = 0; e < 4; ++e) uf[e] = sf[ss][c0 + kCs * e], ub[e] = sb[ss][c0 + kCs * e];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = rq + 16 * q;
      const int32_t c = T + r;
      if (kPass == kInit) {
        int32_t in = 0, out = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int32_t o = other[c0 + kCs * e][r];
          out = max(out, edge(x[q][e], o, g.margin)), in = max(in, edge(o, x[q][e], g.margin));
        }
        const int32_t had_in = int32_t(sf[ts][r]), had_out = int32_t(sb[ts][r]);
        // seldom, once the heavy edges were met (m = 18407: 494 -> 320 us for
        // the pass, which every pair's shuffles and atomics bounded)
        if (__any_sync(0xFFFFFFFFu, in > had_in || out > had_out)) {
#pragma unroll
          for (int o = 8; o; o >>= 1) {
            in = max(in, __shfl_xor_sync(0xFFFFFFFFu, in, o));
            out = max(out, __shfl_xor_sync(0xFFFFFFFFu, out, o));
          }
          if ((lane & 15) == 0 && c < m) {
            if (in > had_in) atomicMax(&g.in[c], in);
            if (out > had_out) atomicMax(&g.out[c], out);
          }
        }
      } else if (kPass == kPropagate) {
        const Key mf = sf[ts][r], mb = sb[ts][r];
        // along (u, c) from u's source, against (c, u) from u's target; most
        // of the pass finds nothing better, so that is all that it asks first
        // (of the two edges between them one at most is there: its side's keys
        // are picked first, then compared once)
        bool better = false;
        int32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          o[e] = other[c0 + kCs * e][r];
          const bool in = o[e] > x[q][e];
          const int32_t w = g.margin ? abs(o[e] - x[q][e]) : max(o[e], x[q][e]);
          better |= o[e] != x[q][e] && along(in ? uf[e] : ub[e], w) < (in ? mf : mb);
        }
        if (__any_sync(0xFFFFFFFFu, better)) {
          Key bf = mf, bb = mb;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int32_t wi = edge(o[e], x[q][e], g.margin), wo = edge(x[q][e], o[e], g.margin);
            if (wi) bf = min(bf, along(uf[e], wi));
            if (wo) bb = min(bb, along(ub[e], wo));
          }
#pragma unroll
          for (int h = 8; h; h >>= 1) {
            bf = min(bf, __shfl_xor_sync(0xFFFFFFFFu, bf, h));
            bb = min(bb, __shfl_xor_sync(0xFFFFFFFFu, bb, h));
          }
          if ((lane & 15) == 0 && c < m) {
            if (bf < mf) atomicMin(&g.fn[c], bf);
            if (bb < mb) atomicMin(&g.bn[c], bb);
          }
        }
      } else {
        // an incoming edge (u, c) from another SCC
        const int32_t ms = key_id(sf[ts][r]), mt = key_id(sb[ts][r]);
        bool other_scc = false;
#pragma unroll
        for (int e = 0; e < 4; ++e)
          other_scc |= other[c0 + kCs * e][r] > x[q][e] && (key_id(uf[e]) != ms || key_id(ub[e]) != mt);
        const uint32_t any = __ballot_sync(0xFFFFFFFFu, other_scc) >> (lane & 16) & 0xFFFFu;
        if ((lane & 15) == 0 && any && c < m && g.asked[c]) {
          if (ms == mt) g.scc_lose[ms == kNone ? m : ms] = 1;
          else g.lose[c] = 1;
        }
      }
    }
  };
  if (s0) serve(A, 0, A == B ? 0 : 1, x1, A == B ? t1 : t2);
  if (s1) serve(B, 1, 0, x2, t1);
}

// Postprocessing (Alg. 4) without edges: the loser among c, its source and its
// target, and whether c's incoming edges matter: those of the unknown
// candidates, and of those with an SCC's label (s = t), which may be an unknown
// candidate's.
__device__ __forceinline__ void mark_by_keys(Key f, Key b, int32_t c, int32_t* lose) {
  const int32_t s = key_id(f), t = key_id(b);
  if (s < t) {
    lose[c] = 1;
  } else if (s > t) {
    lose[t] = 1;  // an id: t < s
  } else if (s != kNone) {
    // smaller low words are wider
    if (uint32_t(f) < uint32_t(b)) lose[c] = 1;
    else if (uint32_t(f) > uint32_t(b)) lose[s] = 1;
  }
}
__device__ __forceinline__ bool asks(int32_t status, int32_t s, int32_t t) {
  return status == kUnknown || (s == t && s != kNone);
}

// The same passes for few candidates, a warp per candidate on its row of d and
// of dT (d transposed): a round is one launch that no atomics and no commit
// follow, and a square of few blocks still gives every SM a warp. Bound by
// latency and by the host's look at *set after every round (20 to 27 us each).
// Uniform random d, the whole call, against pairs of blocks: m = 64 740 and 1144
// us, m = 300 2740 and 4290, m = 700 3550 and 4110, m = 1024 7270 and 7690.
// *clear is the word that the next round sets when a key changes.
constexpr int kRowWarps = 4;
template <int kPass>
__global__ void __launch_bounds__(32 * kRowWarps) rows_kernel(PassArgs g, const int32_t* __restrict__ dT,
                                                              int32_t* __restrict__ set, int32_t* __restrict__ clear) {
  if (kPass == kPropagate && blockIdx.x == 0 && threadIdx.x == 0) *clear = 0;
  const int lane = threadIdx.x & 31;
  const int32_t c = blockIdx.x * kRowWarps + (threadIdx.x >> 5), m = g.m;
  if (c >= m) return;
  const int32_t *dr = g.d + int64_t(c) * m, *tr = dT + int64_t(c) * m;
  if (kPass == kInit) {
    int32_t in = 0, out = 0;
    for (int32_t u = lane; u < m; u += 32) {
      const int32_t x = dr[u], o = tr[u];
      out = max(out, edge(x, o, g.margin)), in = max(in, edge(o, x, g.margin));
    }
    in = __reduce_max_sync(0xFFFFFFFFu, in), out = __reduce_max_sync(0xFFFFFFFFu, out);
    if (lane == 0) g.status[c] = in > out ? kLoser : kUnknown;
    return;
  }
  const Key mf = g.f[c], mb = g.b[c];
  if (kPass == kPropagate) {
    Key bf = mf, bb = mb;
    constexpr int kU = 4;  // loads in flight, also in a last step that not all lanes need
    for (int32_t u0 = lane; u0 < m; u0 += 32 * kU) {
      int32_t x[kU], o[kU];
      Key uf[kU], ub[kU];
#pragma unroll
      for (int e = 0; e < kU; ++e) {
        const int32_t u = u0 + 32 * e;
        const bool in = u < m;
        x[e] = in ? dr[u] : 0, o[e] = in ? tr[u] : 0;
        uf[e] = in ? g.f[u] : 0, ub[e] = in ? g.b[u] : 0;
      }
#pragma unroll
      for (int e = 0; e < kU; ++e) {
        const int32_t w = g.margin ? abs(o[e] - x[e]) : max(o[e], x[e]);
        if (o[e] > x[e]) bf = min(bf, along(uf[e], w));  // along (u, c) from u's source
        if (x[e] > o[e]) bb = min(bb, along(ub[e], w));  // against (c, u) from u's target
      }
    }
#pragma unroll
    for (int h = 16; h; h >>= 1) {
      bf = min(bf, __shfl_xor_sync(0xFFFFFFFFu, bf, h));
      bb = min(bb, __shfl_xor_sync(0xFFFFFFFFu, bb, h));
    }
    if (lane == 0) {
      g.fn[c] = bf, g.bn[c] = bb;
      if (bf != mf || bb != mb) *set = 1;
    }
  } else {
    const int32_t ms = key_id(mf), mt = key_id(mb);
    if (lane == 0) mark_by_keys(mf, mb, c, g.lose);
    if (!asks(g.status[c], ms, mt)) return;
    bool other = false;  // an incoming edge (u, c) from another SCC
    for (int32_t u = lane; u < m; u += 32)
      other |= tr[u] > dr[u] && (key_id(g.f[u]) != ms || key_id(g.b[u]) != mt);
    if (__any_sync(0xFFFFFFFFu, other) && lane == 0) {
      if (ms == mt) g.scc_lose[ms == kNone ? m : ms] = 1;
      else g.lose[c] = 1;
    }
  }
}

// dT = d transposed, through 32 x 32 shared-memory tiles.
__global__ void __launch_bounds__(256) transpose_kernel(const int32_t* __restrict__ d, int32_t m,
                                                        int32_t* __restrict__ dT) {
  __shared__ int32_t tile[32][33];
  const int32_t j0 = blockIdx.x * 32, i0 = blockIdx.y * 32, x = threadIdx.x & 31;
  for (int r = threadIdx.x >> 5; r < 32; r += 8) tile[r][x] = i0 + r < m && j0 + x < m ? d[int64_t(i0 + r) * m + j0 + x] : 0;
  __syncthreads();
  for (int r = threadIdx.x >> 5; r < 32; r += 8)
    if (j0 + r < m && i0 + x < m) dT[int64_t(j0 + r) * m + i0 + x] = tile[x][r];
}

// Initialisation-of-vertices (Alg. 1): c is a loser when its heaviest
// incoming edge outweighs its heaviest outgoing one.
__global__ void init_status_kernel(const int32_t* __restrict__ in, const int32_t* __restrict__ out, int32_t m,
                                   int32_t* __restrict__ status) {
  for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x)
    status[c] = in[c] > out[c] ? kLoser : kUnknown;
}

// Preprocessing (Alg. 2), a CTA per block of 64: the keys, and the blocks
// whose candidates start a propagation; also clears the marks (slot m too).
__global__ void __launch_bounds__(kPT) preprocess_kernel(const int32_t* __restrict__ status, int32_t m,
                                                         Key* __restrict__ f, Key* __restrict__ b,
                                                         Key* __restrict__ fn, Key* __restrict__ bn,
                                                         int32_t* __restrict__ flag, int32_t* __restrict__ lose,
                                                         int32_t* __restrict__ scc_lose) {
  const int32_t c = blockIdx.x * kPT + threadIdx.x;
  const bool unknown = c < m && status[c] == kUnknown;
  if (c < m) {
    const Key k = unknown ? key(c, kNone) : key(kNone, 0);
    f[c] = b[c] = fn[c] = bn[c] = k;
    lose[c] = scc_lose[c] = 0;
  }
  if (c == 0) scc_lose[m] = 0;
  const int any = __syncthreads_or(unknown);
  if (threadIdx.x == 0) flag[blockIdx.x] = any;
}

// The end of a round, a CTA per block of 64: the next keys become the
// current ones; the block's flag and *changed say whether any differ.
__global__ void __launch_bounds__(kPT) commit_kernel(int32_t m, Key* __restrict__ f, Key* __restrict__ b,
                                                     const Key* __restrict__ fn, const Key* __restrict__ bn,
                                                     int32_t* __restrict__ flag, int32_t* __restrict__ changed) {
  const int32_t c = blockIdx.x * kPT + threadIdx.x;
  bool ch = false;
  if (c < m) {
    ch = fn[c] != f[c] || bn[c] != b[c];
    f[c] = fn[c], b[c] = bn[c];
  }
  const int any = __syncthreads_or(ch);
  if (threadIdx.x == 0) {
    flag[blockIdx.x] = any;
    if (any) *changed = 1;
  }
}

// Postprocessing (Alg. 4), the marks that need no edges, the candidates whose
// incoming edges matter (the marks pass), and what the blocks have in common. A
// CTA per block of 64.
__global__ void __launch_bounds__(kPT) label_kernel(const Key* __restrict__ f, const Key* __restrict__ b, int32_t m,
                                                    const int32_t* __restrict__ status, int32_t* __restrict__ lose,
                                                    int32_t* __restrict__ asked, int32_t* __restrict__ flag,
                                                    int4* __restrict__ label) {
  const int32_t c = blockIdx.x * kPT + threadIdx.x;
  const int32_t s0 = key_id(f[blockIdx.x * kPT]), t0 = key_id(b[blockIdx.x * kPT]);
  bool ask = false, same = true;
  if (c < m) {
    const int32_t s = key_id(f[c]), t = key_id(b[c]);
    same = s == s0 && t == t0;
    mark_by_keys(f[c], b[c], c, lose);
    ask = asks(status[c], s, t);
    asked[c] = ask;
  }
  const int any = __syncthreads_or(ask), one = __syncthreads_and(same);
  if (threadIdx.x == 0) flag[blockIdx.x] = any, label[blockIdx.x] = make_int4(s0, t0, one, 0);
}

// Postprocessing, applied: unknown candidates marked (or in a marked SCC)
// become losers; then unknown c with s = t = c become winners. decided[0]
// counts the changes.
__global__ void apply_kernel(const Key* __restrict__ f, const Key* __restrict__ b, int32_t m,
                             const int32_t* __restrict__ lose, const int32_t* __restrict__ scc_lose,
                             int32_t* __restrict__ status, int32_t* __restrict__ decided) {
  for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x) {
    if (status[c] != kUnknown) continue;
    const int32_t s = key_id(f[c]), t = key_id(b[c]);
    const bool in_lost = s == t && scc_lose[s == kNone ? m : s];
    if (lose[c] || in_lost) {
      status[c] = kLoser;
      atomicAdd(decided, 1);
    } else if (s == c && t == c) {
      status[c] = kWinner;
      atomicAdd(decided, 1);
    }
  }
}

__global__ void winners_out_kernel(const int32_t* __restrict__ status, int32_t m, int32_t* __restrict__ winners,
                                   int32_t* __restrict__ unknown) {
  for (int32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x) {
    winners[c] = status[c] == kWinner;
    if (status[c] == kUnknown) atomicAdd(unknown, 1);
  }
}

}  // namespace

// Candidates up to which rows_kernel does the passes (from there on the pairs of
// blocks, which read d once a round and leave blocks out, are as fast).
constexpr int32_t kRowsMax = 1024;

size_t propagation_workspace_bytes(int32_t m) {
  const size_t mv = align_up((size_t(m) + 1) * 4, 256);
  return 4 * align_up(size_t(m) * 8, 256) + 8 * mv + (m <= kRowsMax ? align_up(size_t(m) * size_t(m) * 4, 256) : 0) + 4096;
}

int winners_propagation_launch(schulze_ctx* ctx, const int32_t* d, int32_t m, bool margin, int32_t* winners,
                               int32_t* stats, void* ws, cudaStream_t stream, const int32_t* max_in,
                               const int32_t* max_out) {
  Carver cv(ws);
  Key* f = cv.take<Key>(size_t(m));
  Key* b = cv.take<Key>(size_t(m));
  Key* fn = cv.take<Key>(size_t(m));
  Key* bn = cv.take<Key>(size_t(m));
  int32_t* status = cv.take<int32_t>(size_t(m) + 1);
  int32_t* lose = cv.take<int32_t>(size_t(m) + 1);
  int32_t* scc_lose = cv.take<int32_t>(size_t(m) + 1);
  int32_t* asked = cv.take<int32_t>(size_t(m) + 1);
  int32_t* inout = cv.take<int32_t>(2 * size_t(m) + 1);  // heaviest incoming, outgoing edges
  int32_t* words = cv.take<int32_t>(4);                  // [0] changed, [1] decided, [2] unknown, [3] changed (in turn)
  const int32_t nbt = (m + kPT - 1) / kPT;
  int32_t* flag = cv.take<int32_t>(size_t(nbt));
  int4* label = cv.take<int4>(size_t(nbt));
  const bool rows = m <= kRowsMax && !max_in;
  int32_t* dT = rows ? cv.take<int32_t>(size_t(m) * size_t(m)) : nullptr;
  const unsigned row_grid = unsigned((m + kRowWarps - 1) / kRowWarps);
  const unsigned pairs = unsigned(int64_t(nbt) * (nbt + 1) / 2);
  const int g = std::max(1, std::min((m + 255) / 256, 1024));
  PassArgs pa{};
  pa.d = d, pa.m = m, pa.margin = margin ? 1 : 0;
  const bool vec = rows_vec16(d, m);
  pa.in = inout, pa.out = inout + m, pa.flag = flag, pa.f = f, pa.b = b, pa.fn = fn, pa.bn = bn, pa.changed = words;
  pa.asked = asked, pa.label = label, pa.lose = lose, pa.scc_lose = scc_lose, pa.status = status;
  {
    Launch L(ctx, stream, "propagation_init", double(m) * double(m) * 4.0);
    if (rows) {
      const unsigned t = unsigned((m + 31) / 32);
      transpose_kernel<<<dim3(t, t), 256, 0, stream>>>(d, m, dT);
      rows_kernel<kInit><<<row_grid, 32 * kRowWarps, 0, stream>>>(pa, dT, nullptr, nullptr);
    } else if (!max_in) {
      if (cudaMemsetAsync(inout, 0, 2 * size_t(m) * 4, stream) != cudaSuccess) return SCHULZE_ECUDA;
      (vec ? pair_kernel<kInit, true> : pair_kernel<kInit, false>)<<<pairs, 256, 0, stream>>>(pa);
    }
    if (!rows) init_status_kernel<<<g, 256, 0, stream>>>(max_in ? max_in : pa.in, max_in ? max_out : pa.out, m, status);
  }
  if (int rc = check_launch()) return rc;
  int32_t iterations = 0, rounds = 0;
  for (;;) {
    int32_t host[3] = {0, 0, 0};
    if (cudaMemsetAsync(words, 0, 4 * sizeof(int32_t), stream) != cudaSuccess) return SCHULZE_ECUDA;
    winners_out_kernel<<<g, 256, 0, stream>>>(status, m, winners, words + 2);
    if (cudaMemcpyAsync(host, words, sizeof(host), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
      return SCHULZE_ECUDA;
    if (host[2] == 0) break;  // no unknown candidate left
    if (iterations >= m) return SCHULZE_EDATA;  // every iteration decides one at least
    ++iterations;
    preprocess_kernel<<<nbt, kPT, 0, stream>>>(status, m, f, b, fn, bn, flag, lose, scc_lose);
    // rounds until nothing changes; a chain of m candidates settles in m rounds
    for (int32_t r = 0; r <= m; ++r) {
      int32_t changed = 0, *word = words;
      if (rows) {
        Launch L(ctx, stream, "propagation_round", double(m) * double(m) * 8.0);
        word = words + (r & 1 ? 3 : 0);
        pa.f = f, pa.b = b, pa.fn = fn, pa.bn = bn;
        rows_kernel<kPropagate><<<row_grid, 32 * kRowWarps, 0, stream>>>(pa, dT, word, words + (r & 1 ? 0 : 3));
        std::swap(f, fn), std::swap(b, bn);
      } else {
        Launch L(ctx, stream, "propagation_round", double(m) * double(m) * 4.0);
        (vec ? pair_kernel<kPropagate, true> : pair_kernel<kPropagate, false>)<<<pairs, 256, 0, stream>>>(pa);
        commit_kernel<<<nbt, kPT, 0, stream>>>(m, f, b, fn, bn, flag, words);
      }
      ++rounds;
      if (cudaMemcpyAsync(&changed, word, sizeof(int32_t), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
          cudaStreamSynchronize(stream) != cudaSuccess)
        return SCHULZE_ECUDA;
      if (!changed) break;
    }
    {
      Launch L(ctx, stream, "propagation_marks", double(m) * double(m) * 4.0);
      if (rows) {
        pa.f = f, pa.b = b;
        rows_kernel<kMarks><<<row_grid, 32 * kRowWarps, 0, stream>>>(pa, dT, nullptr, nullptr);
      } else {
        label_kernel<<<nbt, kPT, 0, stream>>>(f, b, m, status, lose, asked, flag, label);
        (vec ? pair_kernel<kMarks, true> : pair_kernel<kMarks, false>)<<<pairs, 256, 0, stream>>>(pa);
      }
    }
    apply_kernel<<<g, 256, 0, stream>>>(f, b, m, lose, scc_lose, status, words + 1);
    int32_t decided = 0;
    if (cudaMemcpyAsync(&decided, words + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
      return SCHULZE_ECUDA;
    if (decided == 0) return SCHULZE_EDATA;  // never expected: Alg. 4 decides one candidate at least
  }
  if (stats) stats[0] = iterations, stats[1] = rounds;
  return check_launch();
}

}  // namespace schulze
