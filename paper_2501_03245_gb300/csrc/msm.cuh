// Pippenger multi-scalar multiplication on top of the batched affine PADD.
//
// The paper's text has no MSM section; the method is the standard bucket
// method built from the paper's primitives:
//   1. digits: scalar k_i (reduced mod r) in signed c-bit windows
//      d_w in [-2^(c-1) + 1, 2^(c-1)], W = ceil((bits(r) + 1) / c) windows, or of
//      both halves of a split scalar (glv.cuh), half as many windows of twice the
//      points: as many additions, half the buckets and half the doublings at the end;
//   2. counting (one-digit radix) sort of the (bucket id, point) pairs by bucket
//      id: histogram with atomics, exclusive scan, scatter with atomic cursors;
//   3. bucket accumulation with batched affine additions (Section 3.3): the
//      sorted array is cut into chunks of CH consecutive entries and each chunk
//      keeps one running sum; round j adds entry j of every chunk to its running
//      sum, all chunks of a CTA sharing one inversion per round (Montgomery's
//      trick with GAS, Section 3.2).  A chunk entry that starts a new bucket
//      flushes the running sum as a partial bucket sum and restarts it (a copy,
//      no inversion needed).  CH rounds finish the whole array in one launch;
//      (calls with few entries: one thread per chunk in Jacobian coordinates);
//   4. bucket reduction sum_k k B_k per window: running sums over chunks of
//      buckets, then a binary tree that keeps the sums of the chunks whose index
//      has bit j set, for every j;
//   5. window combination sum_w 2^(c w) S_w in Jacobian coordinates, four lanes per
//      chain.
// Several independent MSM instances (different sizes, windows and bases) run
// through the same launches: every instance owns a disjoint range of bucket ids.
#pragma once
#include "glv.cuh"
#include "jac.cuh"

namespace ecc {

constexpr int kAccLog = 5;
constexpr int kAccChunk = 1 << kAccLog;  // entries per running-sum chunk (rounds of step 3)

struct MsmInst {
  uint32_t n;            // points of the instance
  uint32_t c;            // window bits
  uint32_t W;            // windows (digits per scalar)
  uint32_t bucket_base;  // first global bucket id
  uint64_t point_off;    // first point in the global bases array
  uint64_t scalar_off;   // first scalar in the global scalar array
  // Bases with precomputed window multiples: window w of point i is the point
  // 2^(c w) P_i at index w * pre_stride + i, all windows share one set of
  // buckets (Wr = 1) and need no combination.  pre_stride = 0: Wr = W rows of
  // buckets, one per window.
  uint64_t pre_stride;
  uint32_t Wr;           // bucket rows (windows reduced separately)
  uint32_t red_log;      // log2 of the buckets per reduction chunk (element)
  uint64_t elem_off;     // first reduction element; 2^(c - 1 - red_log) per bucket row
  uint32_t row_off;      // first bucket row
  uint32_t cta_off;      // first CTA of the reduction tree's first pass
  // Split scalars: the image of the point at index i under the endomorphism is at
  // i + phi, and both halves' digits of a window go to its buckets.  0: not split.
  uint64_t phi;
};

// log2 of the reduction elements per bucket row
__host__ __device__ inline uint32_t elem_log(const MsmInst& in) { return in.c - 1 - in.red_log; }

// ------------------------------------------------------------------ digits

// k mod r for a 256-bit k (at most a few subtractions: r > 2^253)
template <class C>
ECC_DEV void scalar_mod_r(uint32_t* k) {
  uint32_t rr[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) rr[q] = C::n(q);
  for (int it = 0; it < 8; ++it) {
    uint32_t t[8];
    t[0] = ptx::sub_cc(k[0], rr[0]);
#pragma unroll
    for (int q = 1; q < 8; ++q) t[q] = ptx::subc_cc(k[q], rr[q]);
    const uint32_t borrow = ptx::subc(0, 0);
    if (borrow) break;
#pragma unroll
    for (int q = 0; q < 8; ++q) k[q] = t[q];
  }
}

// Calls fn(w, d) for every window with signed digit d != 0 of the K-word k, or of -k.
// The words shift down by a window at a time, which keeps them in registers.
template <int K, class Fn>
ECC_DEV void for_each_digit(const uint32_t* src, bool neg, int c, int W, Fn fn) {
  uint32_t k[K + 1], carry = 0;
#pragma unroll
  for (int q = 0; q < K; ++q) k[q] = src[q];
  k[K] = 0;
  const uint32_t half = 1u << (c - 1);
#pragma unroll 1
  for (int w = 0; w < W; ++w) {
    const uint32_t v = (k[0] & ((1u << c) - 1u)) + carry;
#pragma unroll
    for (int q = 0; q < K; ++q) k[q] = __funnelshift_r(k[q], k[q + 1], c);
    carry = v > half ? 1u : 0u;
    const int d = carry ? (int)v - (int)(1u << c) : (int)v;
    if (d != 0) fn(w, neg ? -d : d);
  }
}

// Calls fn(w, d, shift) for the nonzero digits of the scalar at `src` of instance
// `in`: bucket row w, and the point at `shift` from the scalar's own.
template <class C, class Fn>
ECC_DEV void for_each_entry(const MsmInst& in, const uint32_t* __restrict__ src, Fn fn) {
  uint32_t k[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) k[q] = src[q];
  scalar_mod_r<C>(k);
  if constexpr (C::GLV) {
    if (in.phi) {
      uint32_t m[2][5];
      bool neg[2];
      glv_split<C>(k, m[0], neg[0], m[1], neg[1]);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        for_each_digit<4>(m[h], neg[h], in.c, in.W, [&](int w, int d) { fn(w, d, h ? in.phi : 0ull); });
      return;
    }
  }
  for_each_digit<8>(k, false, in.c, in.W, [&](int w, int d) { fn(w, d, (uint64_t)w * in.pre_stride); });
}

ECC_DEV int find_inst(const MsmInst* inst, int num, uint64_t g) {
  int lo = 0, hi = num - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (inst[mid].scalar_off <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// A ragged batch whose instance sizes live in device memory: the scalar rows
// of all instances (rows [0, total)) and whether the sizes were refused.
struct MsmDevHdr {
  uint64_t total;
  uint32_t failed;
  uint32_t pad;
};

// Levels of the reduction tree that its first pass does inside one CTA, and that
// pass's CTAs for an instance.
constexpr uint32_t kTreeLog = 8;
__host__ __device__ inline uint32_t tree_ctas(const MsmInst& in) {
  const uint32_t m = elem_log(in);
  return in.Wr << (m > kTreeLog ? m - kTreeLog : 0);
}

// Rows of the batch: the host's count, or the device header's when present.
ECC_DEV uint64_t batch_rows(uint64_t host_total, const MsmDevHdr* hdr) {
  return hdr ? hdr->total : host_total;
}

// Instance table of a ragged batch whose sizes are in device memory.  Every
// instance has the window width, bucket rows and reduction chunk of `proto`, so
// instance i's buckets start at i Wr 2^(c-1) and nothing else about the launch
// sequence depends on the sizes.  rows: sizes[num] (resident bases, scalar rows
// back to back, each size at most n_bases) or offsets[num + 1] (offsets[0] = 0,
// point and scalar rows of instance i from offsets[i]).  Sizes that break these
// rules or a total above `cap` leave an empty batch (total 0, failed = 1: every
// output is O) and record ECC_EINVAL (-1) in the status word.  One CTA.
static __global__ void k_msm_inst_dev(const uint64_t* __restrict__ rows, uint32_t num, int sizes_mode,
                               uint64_t n_bases, uint64_t cap, MsmInst proto, MsmInst* __restrict__ inst,
                               MsmDevHdr* hdr, int* status) {
  __shared__ uint64_t warp_sum[32];
  __shared__ uint64_t carry;
  __shared__ int bad;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) {
    carry = 0;
    bad = !sizes_mode && rows[0] != 0;
  }
  __syncthreads();
  const uint64_t per_bucket_row = (uint64_t)proto.Wr << (proto.c - 1);
  for (uint32_t base = 0; base < num; base += blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    uint64_t n = 0, off = 0;
    if (i < num) {
      if (sizes_mode) {
        n = rows[i];
        if (n > n_bases) bad = 1;
      } else {
        off = rows[i];
        const uint64_t hi = rows[i + 1];
        if (hi < off) bad = 1;
        n = hi >= off ? hi - off : 0;
      }
    }
    // block-wide exclusive prefix of n (scalar rows before instance i)
    uint64_t x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint64_t w = lane < nw ? warp_sum[lane] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, w, o);
        if (lane >= o) w += y;
      }
      if (lane < nw) warp_sum[lane] = w;
    }
    __syncthreads();
    const uint64_t before = carry + (warp > 0 ? warp_sum[warp - 1] : 0) + x - n;
    if (i < num) {
      MsmInst m = proto;
      m.n = (uint32_t)n;
      m.bucket_base = (uint32_t)(i * per_bucket_row);
      m.elem_off = i * ((uint64_t)proto.Wr << elem_log(proto));
      m.row_off = i * proto.Wr;
      m.cta_off = i * tree_ctas(proto);
      m.scalar_off = sizes_mode ? before : off;
      m.point_off = sizes_mode ? 0 : off;
      inst[i] = m;
    }
    __syncthreads();
    if (threadIdx.x == 0) carry += warp_sum[nw - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const uint64_t total = sizes_mode ? carry : rows[num];
    const bool fail = bad || total > cap;
    hdr->total = fail ? 0 : total;
    hdr->failed = fail ? 1u : 0u;
    if (fail) atomicCAS(status, 0, -1);
  }
}

// Histogram of the bucket ids (fire-and-forget atomic increments).
template <class C>
__global__ void k_msm_count(const MsmInst* inst, int num, const uint32_t* __restrict__ scalars,
                            uint64_t total, const MsmDevHdr* hdr, uint32_t* __restrict__ count) {
  const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (g >= batch_rows(total, hdr)) return;
  const MsmInst in = inst[find_inst(inst, num, g)];
  const uint32_t row = in.pre_stride ? 0u : 1u << (in.c - 1);
  for_each_entry<C>(in, scalars + 8 * g, [&](int w, int d, uint64_t) {
    atomicAdd(count + in.bucket_base + w * row + (uint32_t)(d < 0 ? -d : d) - 1, 1u);
  });
}

// Entries are written chunk-transposed: entry p goes to [p % CH][p / CH], CH =
// 2^ch_log.  Only
// the point index is stored; the bucket of position p follows from the offsets.
// The bucket of each chunk's first entry is recorded in cur (the accumulation's
// per-chunk bucket cursor starts there).
template <class C>
__global__ void k_msm_scatter(const MsmInst* inst, int num, const uint32_t* __restrict__ scalars,
                              uint64_t total, const MsmDevHdr* hdr, uint32_t* __restrict__ cursor,
                              uint32_t* __restrict__ vals, uint64_t n_chunks, int ch_log,
                              uint32_t* __restrict__ cur) {
  const uint64_t g = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (g >= batch_rows(total, hdr)) return;
  const MsmInst in = inst[find_inst(inst, num, g)];
  const uint32_t row = in.pre_stride ? 0u : 1u << (in.c - 1);
  const uint64_t pidx = in.point_off + (g - in.scalar_off);
  for_each_entry<C>(in, scalars + 8 * g, [&](int w, int d, uint64_t shift) {
    const uint32_t b = in.bucket_base + w * row + (uint32_t)(d < 0 ? -d : d) - 1;
    const uint32_t p = atomicAdd(cursor + b, 1u);
    const uint32_t idx = (uint32_t)(pidx + shift);  // < 2^31 (host check)
    const uint32_t j = p & ((1u << ch_log) - 1u), chunk = p >> ch_log;
    vals[(uint64_t)j * n_chunks + chunk] = idx | (d < 0 ? 0x80000000u : 0u);
    if (j == 0) cur[chunk] = b;
  });
}

// Partial-sum slots per bucket: one per chunk the bucket's entries touch.
static __global__ void k_msm_npart(const uint32_t* __restrict__ off, uint32_t n_buckets, int ch_log,
                                   uint32_t* __restrict__ npart) {
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n_buckets) return;
  const uint32_t lo = off[b], hi = off[b + 1];
  npart[b] = hi > lo ? ((hi - 1) >> ch_log) - (lo >> ch_log) + 1 : 0;
}

// ------------------------------------------------------------------ accumulation

template <class C>
struct AccArgs {
  using F = typename C::Fp;
  const uint32_t* vals;   // sorted (point index | sign bit), [CH][n_chunks]
  const uint32_t* off;    // bucket offsets (exclusive scan), off[n_buckets] = entries
  const uint32_t* poff;   // partial-slot offsets per bucket
  uint32_t n_buckets;
  uint64_t n_chunks;
  const uint32_t* bases;  // AoS Montgomery affine points, 2N words each
  uint32_t* cur;          // bucket of the chunk's current entry
  PtSoA<F> S;             // running sum per chunk
  PtSoA<F> partial;       // partial bucket sums
  SoA<F> M;               // GAS prefix products
};

template <class C>
ECC_DEV const uint4* base_ptr(const AccArgs<C>& a, uint32_t v) {
  return reinterpret_cast<const uint4*>(a.bases + (uint64_t)(v & 0x7fffffffu) * 2 * C::Fp::N);
}

// x of the base a digit names (the sign only touches y)
template <class C>
ECC_DEV void load_base_x(const AccArgs<C>& a, uint32_t v, uint32_t* x) {
  constexpr int N = C::Fp::N;
  const uint4* p = base_ptr(a, v);
#pragma unroll
  for (int g = 0; g < N / 4; ++g) {
    const uint4 t = p[g];
    x[4 * g] = t.x; x[4 * g + 1] = t.y; x[4 * g + 2] = t.z; x[4 * g + 3] = t.w;
  }
}

// y of the base a digit names, negated for a negative digit
template <class C>
ECC_DEV void load_base_y(const AccArgs<C>& a, uint32_t v, uint32_t* y) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint4* p = base_ptr(a, v);
#pragma unroll
  for (int g = 0; g < N / 4; ++g) {
    const uint4 t = p[N / 4 + g];
    y[4 * g] = t.x; y[4 * g + 1] = t.y; y[4 * g + 2] = t.z; y[4 * g + 3] = t.w;
  }
  if (v & 0x80000000u) fe_neg<F>(y, y);
}

template <class C>
ECC_DEV void load_base(const AccArgs<C>& a, uint32_t v, uint32_t* x, uint32_t* y) {
  load_base_x<C>(a, v, x);
  load_base_y<C>(a, v, y);
}

template <class C>
ECC_DEV uint64_t partial_slot(const AccArgs<C>& a, uint32_t b, uint64_t chunk) {
  return a.poff[b] + (chunk - a.off[b] / kAccChunk);
}

// The bucket holding sorted position p: the last b in [lo, n) with off[b] <= p
// (requires off[lo] <= p < off[n]).
ECC_DEV uint32_t bucket_of(const uint32_t* off, uint32_t lo, uint32_t n, uint32_t p) {
  uint32_t hi = n;
  while (hi - lo > 1) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (off[mid] <= p) lo = mid; else hi = mid;
  }
  return lo;
}

// Entry j of chunk c: whether it exists, its bucket, and whether it starts a
// new running sum.  pb = the chunk's bucket before this entry (for j = 0 the
// bucket of the entry itself, recorded by the scatter); off1 = off[pb + 1],
// the end of that bucket (unused for j = 0).
struct AccCls {
  bool live, start;
  uint32_t bucket, prev;
};

template <class C>
ECC_DEV AccCls acc_classify(const AccArgs<C>& a, uint64_t c, int j, uint32_t entries, uint32_t pb,
                            uint32_t off1) {
  AccCls k{false, false, pb, pb};
  const uint32_t p = (uint32_t)(c * kAccChunk + j);
  if (p >= entries) return k;
  k.live = true;
  if (j == 0 || p >= off1) k.start = true;
  if (j == 0 || p < off1) return k;
  k.bucket = pb + 1;  // usually the next bucket; skip empty ones otherwise
  if (a.off[k.bucket + 1] <= p) k.bucket = bucket_of(a.off, k.bucket + 1, a.n_buckets, p);
  return k;
}

// ---- One round with every operand staged in shared memory (cp.async).
// Entry j of every chunk is added to the chunk's running sum S (or starts a
// new one at a bucket boundary).  Each thread owns 5 G 16-byte vectors of
// shared memory (G = N / 4 vectors per field element; layout [vector][thread],
// so a warp's copies of one vector are 512 contiguous bytes).  They are the
// thread's own column of the GAS tree, which is dead outside cta_invert: the
// staging costs no shared memory of its own.  While a thread computes on its
// item k, the copies of item k+1's operands and the first-level loads of item
// k+2 (its sorted entry and its chunk's bucket cursor, into registers) are in
// flight, and so is item k+1's bucket end off[pb + 1], so the gathers behind
// the sorted entries do not stall the arithmetic.  Compress stages only x of S
// and of the base (the compress step of Section 3.3); y is read, directly, only
// when an operand may be O (x = 0) or the two x agree (doubling or P = -T),
// which random inputs almost never hit.  DCWPA stages S, the base and the prefix
// product.  With 8 limbs it holds all of them in registers from the top of the
// item, so the next item's copies start at once; with 12 limbs (no registers to
// spare) it computes the item's two DCWPA products from the staged values first,
// then loads the finish operands and only then starts the next item's copies.
// No denominator array exists for either width.
template <int N, int BLOCK>
struct Stage {
  static constexpr int G = N / 4;
  // vector bases: S.x, S.y, base.x, base.y, prefix product
  static constexpr int SX = 0, SY = G, BX = 2 * G, BY = 3 * G, PRE = 4 * G;
  uint4* v;  // [5 G][BLOCK]
  ECC_DEV uint4* at(int k) const { return v + k * BLOCK + threadIdx.x; }
  ECC_DEV void get(int k0, uint32_t* r) const {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint4 p = *at(k0 + g);
      r[4 * g] = p.x;
      r[4 * g + 1] = p.y;
      r[4 * g + 2] = p.z;
      r[4 * g + 3] = p.w;
    }
  }
};

// Issues the copies of chunk c's operands (entry v): x of S and of the base,
// and with `full` also y of both and the prefix product.  The base is touched
// only for an existing entry (v is meaningful only then).
template <class C, int BLOCK>
ECC_DEV void acc_stage(const Stage<C::Fp::N, BLOCK>& sg, const AccArgs<C>& a, uint64_t c, uint32_t v,
                       bool live, bool full) {
  using S = Stage<C::Fp::N, BLOCK>;
#pragma unroll
  for (int g = 0; g < S::G; ++g) ptx::cp_async16(sg.at(S::SX + g), a.S.x.vec + g * a.S.x.stride + c);
  if (full) {
#pragma unroll
    for (int g = 0; g < S::G; ++g) {
      ptx::cp_async16(sg.at(S::SY + g), a.S.y.vec + g * a.S.y.stride + c);
      ptx::cp_async16(sg.at(S::PRE + g), a.M.vec + g * a.M.stride + c);
    }
  }
  if (live) {
    const uint4* p = base_ptr(a, v);
#pragma unroll
    for (int g = 0; g < S::G; ++g) ptx::cp_async16(sg.at(S::BX + g), p + g);
    if (full) {
#pragma unroll
      for (int g = 0; g < S::G; ++g) ptx::cp_async16(sg.at(S::BY + g), p + S::G + g);
    }
  }
  ptx::cp_async_commit();
}

template <class C, int BLOCK>
__device__ void acc_round_staged(const AccArgs<C>& a, int j, uint32_t entries, uint64_t begin,
                                 uint64_t end, GasSmem<C::Fp::N, BLOCK>& sm) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  using S = Stage<N, BLOCK>;
  constexpr bool kEarly = N <= 8;
  static_assert(sizeof(sm.tree) >= 5 * S::G * BLOCK * sizeof(uint4), "staging fits the GAS tree");
  const S sg{&sm.tree[0][0][0]};
  const uint64_t i0 = begin + threadIdx.x;
  const uint64_t row = (uint64_t)j * a.n_chunks;
  auto is_live = [&](uint64_t c) { return (uint32_t)(c * kAccChunk + j) < entries; };
  // pipeline registers: item k (v0, pb0, o0), item k+1 (v1, pb1), item k+2 (v2, pb2)
  uint32_t v0 = 0, pb0 = 0, o0 = 0, v1 = 0, pb1 = 0;
  // ---- compress, ascending
  uint32_t run[N];
  fe_set_one<F>(run);
  if (i0 < end) {
    v0 = a.vals[row + i0];
    pb0 = a.cur[i0];
    acc_stage<C, BLOCK>(sg, a, i0, v0, is_live(i0), false);
    if (j > 0) o0 = a.off[pb0 + 1];
    if (i0 + BLOCK < end) {
      v1 = a.vals[row + i0 + BLOCK];
      pb1 = a.cur[i0 + BLOCK];
    }
  }
  for (uint64_t c = i0; c < end; c += BLOCK) {
    ptx::cp_async_wait_all();
    uint32_t x1[N], x2[N];
    sg.get(S::SX, x1);
    sg.get(S::BX, x2);
    const uint64_t cn = c + BLOCK;
    uint32_t o1 = 0, v2 = 0, pb2 = 0;
    if (cn < end) {
      acc_stage<C, BLOCK>(sg, a, cn, v1, is_live(cn), false);
      if (j > 0) o1 = a.off[pb1 + 1];
      if (cn + BLOCK < end) {
        v2 = a.vals[row + cn + BLOCK];
        pb2 = a.cur[cn + BLOCK];
      }
    }
    a.M.store(c, run);
    const AccCls k = acc_classify(a, c, j, entries, pb0, o0);
    uint32_t d[N];
    if (!k.live || k.start) {
      fe_set_one<F>(d);
    } else if (fe_is_zero<F>(x1) || fe_is_zero<F>(x2) || fe_eq<F>(x1, x2)) {
      uint32_t y1[N], y2[N];
      a.S.y.load(c, y1);
      load_base_y<C>(a, v0, y2);
      add_den<C>(d, x1, y1, x2, y2);
    } else {
      fe_sub<F>(d, x2, x1);
    }
    mont_mul<F>(run, run, d);
    v0 = v1; pb0 = pb1; o0 = o1;
    v1 = v2; pb1 = pb2;
  }
  // ---- inverse of the CTA's product (GAS, Section 3.2); the staging area is
  // the tree inside, so every copy of this thread has landed (waited above)
  uint32_t inv[N];
  cta_invert<F, BLOCK>(inv, run, sm);
  if (i0 >= end) return;
  // ---- DCWPA, descending
  const uint64_t last = i0 + ((end - 1 - i0) / BLOCK) * BLOCK;
  v0 = a.vals[row + last];
  pb0 = a.cur[last];
  acc_stage<C, BLOCK>(sg, a, last, v0, is_live(last), true);
  o0 = j > 0 ? a.off[pb0 + 1] : 0u;
  if (last >= i0 + BLOCK) {
    v1 = a.vals[row + last - BLOCK];
    pb1 = a.cur[last - BLOCK];
  }
  for (uint64_t c = last;; c -= BLOCK) {
    ptx::cp_async_wait_all();
    const bool more = c >= i0 + BLOCK;
    uint32_t o1 = 0, v2 = 0, pb2 = 0;
    // next item's copies and bucket end, first-level loads of the one after
    auto ahead = [&]() {
      if (!more) return;
      const uint64_t cn = c - BLOCK;
      acc_stage<C, BLOCK>(sg, a, cn, v1, is_live(cn), true);
      if (j > 0) o1 = a.off[pb1 + 1];
      if (cn >= i0 + BLOCK) {
        v2 = a.vals[row + cn - BLOCK];
        pb2 = a.cur[cn - BLOCK];
      }
    };
    const AccCls k = acc_classify(a, c, j, entries, pb0, o0);
    const bool neg = (v0 & 0x80000000u) != 0;
    uint32_t xs[N], ys[N], xp[N], yp[N], d[N], mine[N];
    int kind = ADD_RET_T;
    if constexpr (kEarly) {
      uint32_t pre[N];
      sg.get(S::SX, xs);
      sg.get(S::SY, ys);
      sg.get(S::BX, xp);
      sg.get(S::BY, yp);
      sg.get(S::PRE, pre);
      ahead();
      if (neg) fe_neg<F>(yp, yp);
      if (!k.live || k.start) {
        fe_set_one<F>(d);
      } else {
        kind = add_den<C>(d, xs, ys, xp, yp);
      }
      mont_mul<F>(mine, inv, pre);
      mont_mul<F>(inv, inv, d);
    } else {
      if (!k.live || k.start) {
        fe_set_one<F>(d);
      } else {
        sg.get(S::SX, xs);
        sg.get(S::BX, xp);
        if (fe_is_zero<F>(xs) || fe_is_zero<F>(xp) || fe_eq<F>(xs, xp)) {
          sg.get(S::SY, ys);
          sg.get(S::BY, yp);
          if (neg) fe_neg<F>(yp, yp);
          kind = add_den<C>(d, xs, ys, xp, yp);
        } else {
          kind = ADD_REGULAR;
          fe_sub<F>(d, xp, xs);
        }
      }
      {
        uint32_t pre[N];
        sg.get(S::PRE, pre);
        mont_mul<F>(mine, inv, pre);
      }
      mont_mul<F>(inv, inv, d);
      sg.get(S::SX, xs);
      sg.get(S::SY, ys);
      sg.get(S::BX, xp);
      sg.get(S::BY, yp);
      ahead();
      if (neg) fe_neg<F>(yp, yp);
    }
    if (k.live) {
      if (k.start) {
        if (j > 0) {
          a.partial.store(partial_slot(a, k.prev, c), xs, ys);
          a.cur[c] = k.bucket;
        }
        a.S.store(c, xp, yp);
      } else {
        add_finish<C>(xs, ys, kind, mine, xs, ys, xp, yp);
        a.S.store(c, xs, ys);
      }
    }
    if (!more) break;
    v0 = v1; pb0 = pb1; o0 = o1;
    v1 = v2; pb1 = pb2;
  }
}

template <class C, int BLOCK>
__global__ void __launch_bounds__(BLOCK, kGasResidentThreads / BLOCK) k_msm_accumulate(AccArgs<C> a) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  auto& sm = gas_smem<N, BLOCK>();
  const uint32_t entries = a.off[a.n_buckets];
  const uint64_t used = (entries + kAccChunk - 1) / kAccChunk;
  // equal shares of the chunks actually used (at least 32 per CTA)
  uint64_t per = (used + gridDim.x - 1) / gridDim.x;
  if (per < 32) per = 32;
  const uint64_t begin = blockIdx.x * per;
  uint64_t end = begin + per;
  if (end > used) end = used;
  if (end < begin) end = begin;
  for (int j = 0; j < kAccChunk; ++j) acc_round_staged<C, BLOCK>(a, j, entries, begin, end, sm);
  // flush the last running sum of every chunk
  for (uint64_t c = begin + threadIdx.x; c < end; c += BLOCK) {
    uint32_t xs[N], ys[N];
    a.S.load(c, xs, ys);
    a.partial.store(partial_slot(a, a.cur[c], c), xs, ys);
  }
}

// ------------------------------------------------------------------ few entries
//
// A batched affine round costs a CTA-wide inversion whatever it holds (about 25 us
// with 8 limbs, 40 with 12), and an accumulation has 32 of them.  Below
// kDirectEntries entries (msm_host.cuh) a mixed Jacobian addition (11 products
// instead of 6) by one thread per chunk, which waits for nobody, is faster.

template <class F>
struct JacSoA {
  SoA<F> x, y, z;
  ECC_DEV void load(size_t i, uint32_t* X, uint32_t* Y, uint32_t* Z) const {
    x.load(i, X);
    y.load(i, Y);
    z.load(i, Z);
  }
  ECC_DEV void store(size_t i, const uint32_t* X, const uint32_t* Y, const uint32_t* Z) const {
    x.store(i, X);
    y.store(i, Y);
    z.store(i, Z);
  }
};

// Threads of the Jacobian kernels: 128 registers a thread hold the additions of 8
// limbs, 168 those of 12.
constexpr int kJacThreads = 128;
template <int N>
constexpr int kJacCtas = N <= 8 ? 4 : 3;

// Running sums of the chunks as in the affine rounds, with partial sums in
// Jacobian coordinates.
template <class C>
__global__ void __launch_bounds__(kJacThreads, kJacCtas<C::Fp::N>)
    k_msm_accumulate_jac(AccArgs<C> a, JacSoA<typename C::Fp> partial, int ch_log) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint32_t entries = a.off[a.n_buckets];
  const uint64_t c = blockIdx.x * (uint64_t)kJacThreads + threadIdx.x;
  const uint32_t p0 = (uint32_t)(c << ch_log);
  if ((c << ch_log) >= entries) return;
  const uint32_t ch = entries - p0 < (1u << ch_log) ? entries - p0 : 1u << ch_log;
  uint32_t b = a.cur[c], end = a.off[b + 1];
  uint32_t X[N], Y[N], Z[N], H[N];
  jac_set_inf<F>(X, Y, Z);
  auto flush = [&]() { partial.store(a.poff[b] + (c - (a.off[b] >> ch_log)), X, Y, Z); };
#pragma unroll 1
  for (uint32_t j = 0; j < ch; ++j) {
    const uint32_t p = p0 + j;
    if (p >= end) {
      flush();
      jac_set_inf<F>(X, Y, Z);
      ++b;  // usually the next bucket; skip empty ones otherwise
      if (a.off[b + 1] <= p) b = bucket_of(a.off, b + 1, a.n_buckets, p);
      end = a.off[b + 1];
    }
    uint32_t x[N], y[N];
    load_base<C>(a, a.vals[(uint64_t)j * a.n_chunks + c], x, y);
    if (!pt_is_inf<F>(x, y)) jac_madd<C>(X, Y, Z, x, y, H);
  }
  flush();
}

// ------------------------------------------------------------------ reduction
//
// Window sum sum_b b E_b (E_b the bucket sums, b = 1 .. 2^(c-1)).  Before it the
// partial sums of every bucket are folded into the first one (a pairwise tree,
// ceil(log2 k) rounds for k partials; CTAs take equal shares of the partial slots and
// buckets, so a bucket holding many entries costs rounds only in the CTA that owns it).
//
// A window row is cut into elements of K = 2^red_log consecutive buckets: element u
// has R_u, the plain sum, and S_u = sum_i i E_(K u + i), i = 1 .. K, from two running
// sums by one thread (k_msm_elems).  The window sum is sum_u S_u + K sum_u u R_u, and
// sum_u u R_u = sum_j 2^j Q_j with Q_j the sum of the R_u whose u has bit j set.  A
// binary tree computes all Q_j at once, in place (k_msm_tree): when the block of
// 2^(l+1) elements at e joins its halves, R[e] += R[e + 2^l] is the block's sum,
// the old R[e + 2^l] stays behind as the block's Q_l, and Q_j of the halves, at
// R[e + 2^j] and R[e + 2^l + 2^j], are added for j < l.  That is two additions an
// element in all, log2 of the elements deep.  k_msm_combine then forms the window
// sums and the windows' combination.
//
// This replaced batched affine rounds (12 products a bucket instead of 27, but a
// walk of 2^red_log + 1 + red_log rounds of about 25 us or more, then levels of four
// elements by one thread): 4096 BN254 points 0.9 -> 0.06 ms, 256 BN254 MSMs of 2^10 to
// 2^18 points 8.9 -> 5.3, 16 x 2^20 BLS12-381 points 12.4 -> 7.6; bound by the products
// of k_msm_elems where there are many buckets.  The combination below took 1.1 ms for
// one BN254 result by one thread and takes 0.28 (half the doublings, by a quad); for
// 65536 results of whole scalars it takes as long either way.

constexpr int kRedLog1Default = 5;      // log2 buckets per element, at most, by default
constexpr int kRedLog1Max = 10;

// ---- fold: the partial sums of every bucket into its first partial slot
template <class C>
struct FoldArgs {
  using F = typename C::Fp;
  const uint32_t* poff;         // partial-slot offsets per bucket (n_buckets + 1)
  uint32_t n_buckets;
  PtSoA<F> partial;
  SoA<F> M;                     // GAS prefix products, one per slot
  uint32_t* ops;                // per-round list of additions, one word per slot
  JacSoA<F> jac;                // the partial sums when they are in Jacobian coordinates
};

// Buckets are shared out among the fold's CTAs by kFoldSlot for each partial slot before
// them and one for each bucket.  By slots alone one CTA gets all empty buckets between
// two full ones and walks them in every round: 4 vectors of 4096 zeros and ones on a
// table of 22-bit windows 33 ms, now 0.2; 65536 BN254 points with 20-bit windows, whose
// top window fills 2^6 of 2^19 buckets, 8.1 ms, now 0.5.  By slots and buckets alike a top
// window of many partial sums comes to too few CTAs (2^20 points, 24 bits: 0.65, 1.33 ms).
constexpr uint64_t kFoldSlot = 8;

ECC_DEV uint64_t fold_key(const uint32_t* poff, uint32_t b) { return kFoldSlot * poff[b] + b; }

// first b in [0, n] with fold_key(b) >= x
ECC_DEV uint32_t fold_bound(const uint32_t* poff, uint32_t n, uint64_t x) {
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (fold_key(poff, mid) < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Round with stride h: slot l of a bucket with k partials adds slot l + h for
// every l that is a multiple of 2h with l + h < k (fold_round_staged below).

// Exclusive prefix sum of v over the CTA (warp shuffles, then the warp
// totals); total gets the CTA sum.  wsum: BLOCK / 32 shared words.
template <int BLOCK>
ECC_DEV uint32_t cta_exclusive_sum(uint32_t v, uint32_t* wsum, uint32_t& total) {
  constexpr int NW = BLOCK / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < NW ? wsum[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < NW) wsum[lane] = w;
  }
  __syncthreads();
  const uint32_t before = warp > 0 ? wsum[warp - 1] : 0u;
  total = wsum[NW - 1];
  __syncthreads();  // wsum is reused
  return before + x - v;
}

// One fold round over the listed additions (slot s += slot s + h) with the
// operands staged in shared memory: the two partial sums and the prefix
// product of each addition (5 G 16-byte vectors, G = N / 4), the thread's own
// column of the GAS tree (dead outside cta_invert).  The slot list is read two
// additions ahead and the copies run one addition ahead.  With 8 limbs DCWPA
// holds every operand in registers from the top of an addition, so the next
// copies start at once; with 12 limbs it forms the two DCWPA products first
// and starts the next copies once the finish operands are in registers.
template <class C, int BLOCK>
__device__ void fold_round_staged(const FoldArgs<C>& a, uint32_t h, uint64_t s0, uint32_t n_ops,
                                  GasSmem<C::Fp::N, BLOCK>& sm) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  constexpr int G = N / 4;
  constexpr int X0 = 0, Y0 = G, X1 = 2 * G, Y1 = 3 * G, PRE = 4 * G;
  constexpr bool kEarly = N <= 8;
  static_assert(sizeof(sm.tree) >= 5 * G * BLOCK * sizeof(uint4), "staging fits the GAS tree");
  uint4* const base = &sm.tree[0][0][0] + threadIdx.x;
  auto at = [&](int k) { return base + k * BLOCK; };
  auto get = [&](int k0, uint32_t* r) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint4 q = *at(k0 + g);
      r[4 * g] = q.x;
      r[4 * g + 1] = q.y;
      r[4 * g + 2] = q.z;
      r[4 * g + 3] = q.w;
    }
  };
  auto stage = [&](uint32_t sl, bool full) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      ptx::cp_async16(at(X0 + g), a.partial.x.vec + g * a.partial.x.stride + sl);
      ptx::cp_async16(at(Y0 + g), a.partial.y.vec + g * a.partial.y.stride + sl);
      ptx::cp_async16(at(X1 + g), a.partial.x.vec + g * a.partial.x.stride + sl + h);
      ptx::cp_async16(at(Y1 + g), a.partial.y.vec + g * a.partial.y.stride + sl + h);
      if (full) ptx::cp_async16(at(PRE + g), a.M.vec + g * a.M.stride + sl);
    }
    ptx::cp_async_commit();
  };
  const uint32_t t = threadIdx.x;
  // ---- compress, ascending
  uint32_t run[N];
  fe_set_one<F>(run);
  uint32_t sA = 0, sB = 0;
  if (t < n_ops) {
    sA = a.ops[s0 + t];
    stage(sA, false);
    if (t + BLOCK < n_ops) sB = a.ops[s0 + t + BLOCK];
  }
  for (uint32_t e = t; e < n_ops; e += BLOCK) {
    ptx::cp_async_wait_all();
    uint32_t x0[N], y0[N], x1[N], y1[N], d[N];
    get(X0, x0);
    get(Y0, y0);
    get(X1, x1);
    get(Y1, y1);
    uint32_t sC = 0;
    if (e + BLOCK < n_ops) {
      stage(sB, false);
      if (e + 2 * BLOCK < n_ops) sC = a.ops[s0 + e + 2 * BLOCK];
    }
    a.M.store(sA, run);
    add_den<C>(d, x0, y0, x1, y1);
    mont_mul<F>(run, run, d);
    sA = sB;
    sB = sC;
  }
  // ---- inverse of the CTA's product (GAS, Section 3.2)
  uint32_t inv[N];
  cta_invert<F, BLOCK>(inv, run, sm);
  if (t >= n_ops) return;
  // ---- DCWPA, descending
  const uint32_t last = t + ((n_ops - 1 - t) / BLOCK) * BLOCK;
  sA = a.ops[s0 + last];
  stage(sA, true);
  sB = last >= t + BLOCK ? a.ops[s0 + last - BLOCK] : 0u;
  for (uint32_t e = last;; e -= BLOCK) {
    ptx::cp_async_wait_all();
    const bool more = e >= t + BLOCK;
    uint32_t sC = 0;
    auto ahead = [&]() {
      if (!more) return;
      stage(sB, true);
      if (e >= t + 2 * BLOCK) sC = a.ops[s0 + e - 2 * BLOCK];
    };
    uint32_t x0[N], y0[N], x1[N], y1[N], d[N], mine[N];
    int kind;
    if constexpr (kEarly) {
      uint32_t pre[N];
      get(X0, x0);
      get(Y0, y0);
      get(X1, x1);
      get(Y1, y1);
      get(PRE, pre);
      ahead();
      kind = add_den<C>(d, x0, y0, x1, y1);
      mont_mul<F>(mine, inv, pre);
    } else {
      get(X0, x0);
      get(X1, x1);
      if (fe_is_zero<F>(x0) || fe_is_zero<F>(x1) || fe_eq<F>(x0, x1)) {
        get(Y0, y0);
        get(Y1, y1);
        kind = add_den<C>(d, x0, y0, x1, y1);
      } else {
        kind = ADD_REGULAR;
        fe_sub<F>(d, x1, x0);
      }
      {
        uint32_t pre[N];
        get(PRE, pre);
        mont_mul<F>(mine, inv, pre);
      }
      get(Y0, y0);
      get(Y1, y1);
      ahead();
    }
    mont_mul<F>(inv, inv, d);
    add_finish<C>(x0, y0, kind, mine, x0, y0, x1, y1);
    a.partial.store(sA, x0, y0);
    if (!more) break;
    sA = sB;
    sB = sC;
  }
}

// Each round first lists the CTA's pair additions (slot of the left operand)
// in ops[s0 ..), then runs the batched additions over that list, so the work
// of a bucket with many partial sums (the top window often puts most entries
// into a few buckets) is shared by the whole CTA and lanes never idle on
// inactive slots.
// JAC: partial sums in Jacobian coordinates, added one by one.
template <class C, int BLOCK, bool JAC>
__global__ void __launch_bounds__(BLOCK, JAC && C::Fp::N > 8 ? 1 : kGasResidentThreads / BLOCK)
    k_msm_fold(FoldArgs<C> a) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  __shared__ uint32_t wsum[BLOCK / 32];
  const uint64_t total_slots = a.poff[a.n_buckets];
  if (total_slots == 0) return;  // uniform over the grid
  // this CTA owns the buckets that begin in its equal share
  const uint64_t share = (fold_key(a.poff, a.n_buckets) + gridDim.x - 1) / gridDim.x;
  const uint32_t b0 = fold_bound(a.poff, a.n_buckets, blockIdx.x * share);
  const uint32_t b1 = blockIdx.x + 1 == gridDim.x
                          ? a.n_buckets
                          : fold_bound(a.poff, a.n_buckets, (blockIdx.x + 1) * share);
  const uint64_t s0 = a.poff[b0];
  uint32_t kmax = 0;
  for (uint32_t b = b0 + threadIdx.x; b < b1; b += BLOCK) {
    const uint32_t k = a.poff[b + 1] - a.poff[b];
    kmax = k > kmax ? k : kmax;
  }
  // ceil(log2 kmax) rounds; each halves the partials of every bucket
  for (uint32_t h = 1; __syncthreads_or(h < kmax); h *= 2) {
    // list the round's additions: l = 0, 2h, 4h, .. with l + h < k
    uint32_t cnt = 0;
    for (uint32_t b = b0 + threadIdx.x; b < b1; b += BLOCK) {
      const uint32_t k = a.poff[b + 1] - a.poff[b];
      if (k > h) cnt += (k - h - 1) / (2 * h) + 1;
    }
    uint32_t n_ops;
    uint32_t pos = cta_exclusive_sum<BLOCK>(cnt, wsum, n_ops);
    for (uint32_t b = b0 + threadIdx.x; b < b1; b += BLOCK) {
      const uint32_t p = a.poff[b];
      const uint32_t k = a.poff[b + 1] - p;
      for (uint32_t l = 0; l + h < k; l += 2 * h) a.ops[s0 + pos++] = p + l;
    }
    __syncthreads();  // the list is complete
    if constexpr (JAC) {
#pragma unroll 1
      for (uint32_t e = threadIdx.x; e < n_ops; e += BLOCK) {
        const uint32_t sl = a.ops[s0 + e];
        uint32_t X[N], Y[N], Z[N], X2[N], Y2[N], Z2[N];
        a.jac.load(sl, X, Y, Z);
        a.jac.load(sl + h, X2, Y2, Z2);
        jac_addto<C>(X, Y, Z, X2, Y2, Z2);
        a.jac.store(sl, X, Y, Z);
      }
      __syncthreads();  // the sums are in place, the list is free
    } else {
      fold_round_staged<C, BLOCK>(a, h, s0, n_ops, gas_smem<N, BLOCK>());
    }
  }
}

// ---- elements
template <class C>
struct RedArgs {
  using F = typename C::Fp;
  const MsmInst* inst;
  uint32_t num;
  uint64_t elems;
  const uint32_t* poff;   // partial-slot offsets per bucket: its sum is in the first
  PtSoA<F> partial;
  JacSoA<F> jac;
  Jac<F>* R;              // per element
  Jac<F>* S;
  Jac<F>* row;            // window sums
};

// the instance whose range (starting at inst[i].*field) holds t
template <class T>
ECC_DEV uint32_t find_by(const MsmInst* inst, uint32_t num, T MsmInst::*field, uint64_t t) {
  uint32_t lo = 0, hi = num - 1;
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (inst[mid].*field <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <class C, bool JAC>
__global__ void __launch_bounds__(kJacThreads, kJacCtas<C::Fp::N>) k_msm_elems(RedArgs<C> a) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint64_t t = blockIdx.x * (uint64_t)kJacThreads + threadIdx.x;
  if (t >= a.elems) return;
  const MsmInst in = a.inst[find_by(a.inst, a.num, &MsmInst::elem_off, t)];
  const uint64_t b0 = in.bucket_base + ((t - in.elem_off) << in.red_log);  // rows follow each other
  uint32_t X[N], Y[N], Z[N], SX[N], SY[N], SZ[N];
  jac_set_inf<F>(X, Y, Z);
  jac_set_inf<F>(SX, SY, SZ);
  uint32_t hi = a.poff[b0 + (1ull << in.red_log)];
#pragma unroll 1
  for (uint32_t i = 1u << in.red_log; i-- > 0;) {
    const uint32_t slot = a.poff[b0 + i];
    if (hi > slot) {
      if constexpr (JAC) {
        uint32_t X2[N], Y2[N], Z2[N];
        a.jac.load(slot, X2, Y2, Z2);
        jac_addto<C>(X, Y, Z, X2, Y2, Z2);
      } else {
        uint32_t x[N], y[N], H[N];
        a.partial.load(slot, x, y);
        if (!pt_is_inf<F>(x, y)) jac_madd<C>(X, Y, Z, x, y, H);
      }
    }
    hi = slot;
    jac_addto<C>(SX, SY, SZ, X, Y, Z);
  }
  jac_store<F>(a.R + t, X, Y, Z);
  jac_store<F>(a.S + t, SX, SY, SZ);
}

// Levels [l0, l1) of the tree over the blocks of 2^l1 elements: pass 0 does the
// first kTreeLog levels of every row, a CTA per block; pass 1 the others, a CTA per
// row.  While a level has a quad for each of its additions the quads do them.
template <class C>
__global__ void __launch_bounds__(kJacThreads, kJacCtas<C::Fp::N>) k_msm_tree(RedArgs<C> a, int pass) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint32_t blk = blockIdx.x;
  const MsmInst in = a.inst[pass ? find_by(a.inst, a.num, &MsmInst::row_off, blk)
                                 : find_by(a.inst, a.num, &MsmInst::cta_off, blk)];
  const uint32_t m = elem_log(in), first = m < kTreeLog ? m : kTreeLog;
  const uint32_t l0 = pass ? kTreeLog : 0u, l1 = pass ? m : first;
  if (l0 >= l1) return;
  const uint64_t e0 = in.elem_off + ((uint64_t)(blk - (pass ? in.row_off : in.cta_off)) << l1);
#pragma unroll 1
  for (uint32_t l = l0; l < l1; ++l) {
    const uint32_t per = l + 2, n_ops = per << (l1 - 1 - l), half = 1u << l;
    const bool quads = 4 * n_ops <= kJacThreads;
#pragma unroll 1
    for (uint32_t o = quads ? threadIdx.x / 4 : threadIdx.x; o < n_ops; o += kJacThreads) {
      const uint32_t pair = o / per, i = o - pair * per;
      const uint64_t e = e0 + ((uint64_t)pair << (l + 1)) + (i == 0 || i > l ? 0u : 1u << (i - 1));
      Jac<F>* dst = (i > l ? a.S : a.R) + e;
      if (quads) {
        JacReg<F> P = quad_load(dst);
        const JacReg<F> Q = quad_load(dst + half);
        __syncwarp(quad_mask());  // all four have dst before one stores it: O + Q exchanges nothing
        quad_add<C>(P, Q);
        if ((threadIdx.x & 3u) == 0) jac_store<F>(dst, P.X.v, P.Y.v, P.Z.v);
      } else {
        uint32_t X[N], Y[N], Z[N], X2[N], Y2[N], Z2[N];
        jac_load<F>(dst, X, Y, Z);
        jac_load<F>(dst + half, X2, Y2, Z2);
        jac_addto<C>(X, Y, Z, X2, Y2, Z2);
        jac_store<F>(dst, X, Y, Z);
      }
    }
    __syncthreads();
  }
}

// Window sum of a row by one quad: S + 2^red_log sum_j 2^j Q_j.
template <class C>
__global__ void __launch_bounds__(64) k_msm_rows(RedArgs<C> a, uint32_t rows) {
  using F = typename C::Fp;
  const uint32_t row = (blockIdx.x * 64 + threadIdx.x) / 4;
  if (row >= rows) return;
  const MsmInst in = a.inst[find_by(a.inst, a.num, &MsmInst::row_off, row)];
  const uint32_t m = elem_log(in);
  const uint64_t e0 = in.elem_off + ((uint64_t)(row - in.row_off) << m);
  JacReg<F> P;
  jac_set_inf<F>(P.X.v, P.Y.v, P.Z.v);
#pragma unroll 1
  for (uint32_t j = m + 1; j-- > 0;) {  // add Q_(j-1), double; at last add S
    quad_add<C>(P, quad_load(j > 0 ? a.R + e0 + (1ull << (j - 1)) : a.S + e0));
#pragma unroll 1
    for (uint32_t s = j > 1 ? 1u : j * in.red_log; s > 0; --s) quad_dbl<C>(P);
  }
  if ((threadIdx.x & 3u) == 0) jac_store<F>(a.row + row, P.X.v, P.Y.v, P.Z.v);
}

// result_i = sum_w 2^(c w) S_w (Horner) by one quad, converted to canonical affine
// limbs.  Quad t takes instance order[t]: the host lists the instances grouped by
// window width, so the quads of a warp run chains of one length.
template <class C>
__global__ void __launch_bounds__(32) k_msm_combine(RedArgs<C> a, const uint32_t* order, const MsmDevHdr* hdr,
                                                    uint32_t* out_all) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint32_t t = (blockIdx.x * 32 + threadIdx.x) / 4;
  if (t >= a.num) return;
  const uint32_t id = order[t];
  const bool write = (threadIdx.x & 3u) == 0;
  uint32_t* o = out_all + (uint64_t)id * 2 * N;
  if (hdr && hdr->failed) {  // refused sizes: O, written (0, 0)
    for (int q = 0; q < 2 * N && write; ++q) o[q] = 0;
    return;
  }
  const MsmInst in = a.inst[id];
  JacReg<F> P;
  jac_set_inf<F>(P.X.v, P.Y.v, P.Z.v);
#pragma unroll 1
  for (uint32_t w = in.Wr; w-- > 0;) {
#pragma unroll 1
    for (uint32_t s = w + 1 < in.Wr ? in.c : 0u; s > 0; --s) quad_dbl<C>(P);
    quad_add<C>(P, quad_load(a.row + in.row_off + w));
  }
  uint32_t x[N], y[N];
  jac_to_affine<F>(x, y, P);
  from_mont<F>(x, x);
  from_mont<F>(y, y);
  if (!write) return;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    o[q] = x[q];
    o[N + q] = y[q];
  }
}

// canonical AoS points -> Montgomery AoS points (gather layout of the bases), and
// with phi > 0 their images (beta x, y) at rows phi, phi + 1, ..
template <class C>
__global__ void k_points_to_mont(const uint32_t* __restrict__ in, uint64_t n, const MsmDevHdr* hdr,
                                 uint32_t* __restrict__ out, uint64_t phi) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (i >= batch_rows(n, hdr)) return;
  uint32_t x[N], y[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    x[q] = in[2 * N * i + q];
    y[q] = in[2 * N * i + N + q];
  }
  to_mont<F>(x, x);
  to_mont<F>(y, y);
  store_affine<F>(out, i, x, y);
  if constexpr (C::GLV) {
    if (phi) {
      uint32_t beta[N];
#pragma unroll
      for (int q = 0; q < N; ++q) beta[q] = C::glv_beta(q);
      mont_mul<F>(x, x, beta);
      store_affine<F>(out, phi + i, x, y);
    }
  }
}

// ------------------------------------------------------------------ window multiples
// For bases reused across calls: window w of base i becomes 2^(c w) P_i
// (window-major AoS, Montgomery form), so one set of buckets serves every
// window.  Window w is window w-1 doubled c times: c batched PDBL rounds per
// window, every item an independent base.
template <class C>
struct ShiftArgs {
  using F = typename C::Fp;
  uint32_t* pre;     // W windows of n points, 2N words each; window 0 filled in
  uint64_t n;
  uint32_t W, c;
  SoA<F> M;
  uint64_t per_cta;
};

template <class C>
struct ShiftRound {
  using F = typename C::Fp;
  static constexpr int N = F::N;
  const uint32_t* src;
  uint32_t* dst;
  bool live;
  ECC_DEV void den(size_t i, uint32_t* d) {
    uint32_t x[N], y[N];
    load_affine<F>(src, i, x, y);
    live = dbl_den<C>(d, y);
  }
  ECC_DEV void finish(size_t i, const uint32_t* inv) {
    uint32_t x[N], y[N];
    load_affine<F>(src, i, x, y);
    dbl_finish<C>(x, y, live, inv, x, y);
    store_affine<F>(dst, i, x, y);
  }
};

template <class C, int BLOCK>
__global__ void __launch_bounds__(BLOCK, kGasResidentThreads / BLOCK) k_bases_shift(ShiftArgs<C> a) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  auto& sm = gas_smem<N, BLOCK>();
  const uint64_t begin = blockIdx.x * a.per_cta;
  uint64_t end = begin + a.per_cta;
  if (end > a.n) end = a.n;
  if (end < begin) end = begin;
  for (uint32_t w = 1; w < a.W; ++w) {
    uint32_t* dst = a.pre + (uint64_t)w * a.n * 2 * N;
    for (uint32_t r = 0; r < a.c; ++r) {
      ShiftRound<C> rd{r == 0 ? dst - a.n * 2 * N : dst, dst};
      batch_round<F, BLOCK>(rd, begin, end, a.M, sm);
    }
  }
}

}  // namespace ecc
