// Host side of the Pippenger MSM (included once per curve): planning (window
// width per instance, bucket id ranges), workspace layout and the launch
// sequence.  Every launch is stream-ordered and the call performs no host
// synchronisation, so a whole ragged batch can be captured once in a CUDA graph
// and replayed.
#pragma once
#include <algorithm>
#include <vector>

#include "internal.h"
#include "msm.cuh"
#include "scan.cuh"
#include "upload.cuh"

namespace ecc {

namespace msm_detail {

constexpr int kAccBlock = kGasThreads;
static_assert(kRedLog1Max == kMsmReduceLogMax, "one bound for the first-level reduction chunk");

inline int scalar_bits(int curve) {
  switch (curve) {
    case 0: return Secp256k1::SCALAR_BITS;
    case 1: return P256::SCALAR_BITS;
    case 2: return BN254::SCALAR_BITS;
    case 4: return SM2::SCALAR_BITS;
    default: return BLS12_381::SCALAR_BITS;
  }
}

inline int windows_for(int curve, int c) { return (scalar_bits(curve) + 1 + c - 1) / c; }

// Windows of the halves of a split scalar (below 2^GLV_BITS in magnitude).
template <class C>
int half_windows(int c) {
  if constexpr (C::GLV) {
    static_assert(C::GLV_BITS < 128, "magnitudes and their top carry fit four words");
    return (C::GLV_BITS + 1 + c - 1) / c;
  }
  return 0;
}

struct Layout {
  std::vector<MsmInst> inst;
  uint64_t buckets = 0, entries_max = 0, n_chunks = 0, total_points = 0;
  uint64_t elems = 0;          // reduction elements
  uint32_t rows = 0, ctas = 0; // bucket rows, CTAs of the reduction tree's first pass
  uint64_t phi = 0;            // split scalars: rows between the points and their images
  bool direct = false;         // Jacobian accumulation
  int ch_log = kAccLog;        // log2 of the entries per chunk
};

// Entries up to which one Jacobian thread per chunk accumulates faster than batched
// affine rounds.  Whole calls of n points, rounds / threads: BN254 n = 2^15 1.90 /
// 1.07 ms, 2^18 2.37 / 1.82, 2^19 (8.9 M entries) 3.04 / 2.63, 2^20 (16.8 M) 4.34 /
// 4.32; BLS12-381 2^15 3.58 / 1.91, 2^18 5.09 / 3.86, 2^19 6.14 / 5.47, 2^20 8.69 / 8.63.
constexpr uint64_t kDirectEntries = 12u << 20;

// log2 of the buckets per reduction element: the caller's override, or the most (up
// to kRedLog1Default) that leaves two CTAs of elements per SM: fewer elements are
// longer serial sums, more of them are work for the tree (2^18 BN254 points, 278000
// buckets: 1.95, 1.86, 1.82, 1.82, 1.90, 2.15 ms a call for 0 .. 5).
inline int red_log(int curve, uint64_t n, uint64_t buckets) {
  int k = msm_reduce_override(curve, n);
  if (k <= 0) {
    const uint64_t threads = (uint64_t)device_sm_count() * kJacThreads * 2;
    for (k = 0; k < kRedLog1Default && (buckets >> (k + 1)) >= threads;) ++k;
  }
  return k;
}

// Chunks, accumulation form and reduction layout of the planned instances.  lean: the
// longest chunks and elements, which take the least workspace.
template <int N>
void finish_plan(int curve, Layout& L, const uint64_t* sizes, uint64_t size_all, bool lean) {
  BySize<int> log;
  for (size_t i = 0; i < L.inst.size(); ++i) {
    MsmInst& m = L.inst[i];
    const uint64_t n = sizes ? sizes[i] : size_all;
    const int k = log.get(n, [&] { return lean ? msm_reduce_log(curve, n) : red_log(curve, n, L.buckets); });
    m.red_log = (uint32_t)std::min(k, (int)m.c - 1);
    m.elem_off = L.elems;
    m.row_off = L.rows;
    m.cta_off = L.ctas;
    L.elems += (uint64_t)m.Wr << elem_log(m);
    L.rows += m.Wr;
    L.ctas += tree_ctas(m);
  }
  L.direct = L.entries_max < kDirectEntries;
  if (L.direct && !lean) {  // chunks of 8 to 32 entries, about four for each resident thread
    constexpr uint32_t chunks = N <= 8 ? 1u << 18 : 1u << 17;
    for (L.ch_log = 3; L.ch_log < kAccLog && (L.entries_max >> (L.ch_log + 1)) >= chunks;) ++L.ch_log;
  }
  L.n_chunks = (L.entries_max + (1u << L.ch_log) - 1) >> L.ch_log;
}

// Instance sizes held in device memory (capture-time capacity): rows are
// sizes[num] (sizes_mode, resident bases) or offsets[num + 1]; every instance
// has the layout of L.inst[0], and L's totals are the capacity.
struct DevRows {
  const uint64_t* rows;
  int sizes_mode;
  uint64_t n_bases;
  uint64_t cap;
};

// raw_points (optional): canonical caller points to convert into the gather
// layout first (rows [0, total) of the batch); otherwise bases_mont is used.
template <class C>
cudaError_t run_set(int curve, const Layout& L, const uint32_t* bases_mont, const uint32_t* scalars,
                    uint32_t* out, cudaStream_t st, const DevRows* dev = nullptr,
                    const uint32_t* raw_points = nullptr) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const int num = (int)L.inst.size();
  const uint64_t B = L.buckets, NC = std::max<uint64_t>(L.n_chunks, 1);
  const uint64_t n_part = B + NC;
  // ---- workspace
  auto up = [](uint64_t b) { return (b + 255) / 256 * 256; };
  const uint64_t sz_inst = up(num * sizeof(MsmInst));
  const uint64_t sz_b1 = up((B + 1) * 4);
  const uint64_t sz_kv = up((NC << L.ch_log) * 4), sz_cur = up(NC * 4);
  const uint64_t sz_S = soa_bytes<F>(NC), sz_P = soa_bytes<F>(n_part);
  const uint64_t sz_ops = up(n_part * 4);
  // per chunk: running sum (x, y) and prefix product; per partial sum: x, y and
  // prefix product, or X, Y and Z
  const uint64_t kChunkArrays = L.direct ? 0 : 3;
  const uint64_t sz_hdr = up(sizeof(MsmDevHdr));
  const uint64_t sz_pts = raw_points ? up(std::max<uint64_t>(L.phi + L.total_points, 1) * 2 * N * 4) : 0;
  const uint64_t bytes = sz_inst + sz_hdr + sz_pts + 5 * sz_b1 + sz_kv + sz_cur + kChunkArrays * sz_S +
                         3 * sz_P + sz_ops + 256;
  Scratch ws;
  cudaError_t e = ws.alloc(bytes, st);
  if (e != cudaSuccess) return e;
  char* p = ws.as<char>();
  auto take = [&](uint64_t b) { char* r = p; p += b; return r; };
  MsmInst* d_inst = reinterpret_cast<MsmInst*>(take(sz_inst));
  MsmDevHdr* hdr = dev ? reinterpret_cast<MsmDevHdr*>(take(sz_hdr)) : nullptr;
  uint32_t* pts_mont = raw_points ? reinterpret_cast<uint32_t*>(take(sz_pts)) : nullptr;
  uint32_t* count = reinterpret_cast<uint32_t*>(take(sz_b1));
  uint32_t* off = reinterpret_cast<uint32_t*>(take(sz_b1));
  uint32_t* cursor = reinterpret_cast<uint32_t*>(take(sz_b1));
  uint32_t* npart = reinterpret_cast<uint32_t*>(take(sz_b1));
  uint32_t* poff = reinterpret_cast<uint32_t*>(take(sz_b1));
  uint32_t* vals = reinterpret_cast<uint32_t*>(take(sz_kv));
  uint32_t* cur = reinterpret_cast<uint32_t*>(take(sz_cur));
  uint4* sbuf = reinterpret_cast<uint4*>(take(kChunkArrays * sz_S));
  uint4* pbuf = reinterpret_cast<uint4*>(take(3 * sz_P));
  uint32_t* fold_ops = reinterpret_cast<uint32_t*>(take(sz_ops));
  if (dev) {
    k_msm_inst_dev<<<1, 1024, 0, st>>>(dev->rows, (uint32_t)num, dev->sizes_mode, dev->n_bases, dev->cap,
                                       L.inst[0], d_inst, hdr, status_word());
    e = cudaGetLastError();
  } else {
    e = upload_words(d_inst, L.inst.data(), num * sizeof(MsmInst), st);
  }
  if (e != cudaSuccess) return e;
  if (raw_points && L.total_points) {
    k_points_to_mont<C><<<(unsigned)((L.total_points + 255) / 256), 256, 0, st>>>(raw_points, L.total_points,
                                                                                 hdr, pts_mont, L.phi);
    bases_mont = pts_mont;
  }
  phase_mark(0, st);
  // ---- 1-2: digits, counting sort by bucket id
  e = cudaMemsetAsync(count, 0, (B + 1) * 4, st);
  if (e != cudaSuccess) return e;
  const unsigned pb = (unsigned)((L.total_points + 255) / 256);
  if (L.total_points)
    k_msm_count<C><<<pb, 256, 0, st>>>(d_inst, num, scalars, L.total_points, hdr, count);
  e = exclusive_scan(count, B, off, st);
  if (e != cudaSuccess) return e;
  e = cudaMemcpyAsync(cursor, off, B * 4, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  if (B) k_msm_npart<<<(unsigned)((B + 255) / 256), 256, 0, st>>>(off, (uint32_t)B, L.ch_log, npart);
  e = exclusive_scan(npart, B, poff, st);
  if (e != cudaSuccess) return e;
  if (L.total_points)
    k_msm_scatter<C><<<pb, 256, 0, st>>>(d_inst, num, scalars, L.total_points, hdr, cursor, vals, NC,
                                          L.ch_log, cur);
  phase_mark(1, st);
  // ---- 3: bucket accumulation (batched affine, one launch)
  AccArgs<C> a;
  a.vals = vals;
  a.cur = cur;
  a.off = off;
  a.poff = poff;
  a.n_buckets = (uint32_t)B;
  a.n_chunks = NC;
  a.bases = bases_mont;
  a.S = PtSoA<F>{SoA<F>{sbuf, NC}, SoA<F>{sbuf + sz_S / 16, NC}};
  a.M = SoA<F>{sbuf + 2 * sz_S / 16, NC};
  a.partial = PtSoA<F>{SoA<F>{pbuf, n_part}, SoA<F>{pbuf + sz_P / 16, n_part}};
  const size_t smem = sizeof(GasSmem<N, kAccBlock>);
  const JacSoA<F> jac{SoA<F>{pbuf, n_part}, SoA<F>{pbuf + sz_P / 16, n_part}, SoA<F>{pbuf + 2 * sz_P / 16, n_part}};
  if (L.direct) {
    k_msm_accumulate_jac<C><<<(unsigned)((NC + kJacThreads - 1) / kJacThreads), kJacThreads, 0, st>>>(a, jac, L.ch_log);
  } else {
    // persistent CTAs; each takes an equal share of the chunks the sort filled
    uint64_t ctas = (uint64_t)device_sm_count() * kGasCtasPerSm;
    ctas = std::max<uint64_t>(1, std::min<uint64_t>(ctas, (NC + 31) / 32));
    e = cudaFuncSetAttribute(k_msm_accumulate<C, kAccBlock>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_msm_accumulate<C, kAccBlock><<<(unsigned)ctas, kAccBlock, smem, st>>>(a);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  phase_mark(2, st);
  // ---- fold the partial sums of every bucket into its first slot
  if (B) {
    FoldArgs<C> f;
    f.poff = poff;
    f.n_buckets = (uint32_t)B;
    f.partial = a.partial;
    f.M = SoA<F>{pbuf + 2 * sz_P / 16, n_part};
    f.ops = fold_ops;
    f.jac = jac;
    if (L.direct) {
      const unsigned ctas = (unsigned)std::min<uint64_t>((uint64_t)device_sm_count() * 4, (n_part + 63) / 64);
      k_msm_fold<C, kJacThreads, true><<<ctas, kJacThreads, 0, st>>>(f);
    } else {
      e = cudaFuncSetAttribute(k_msm_fold<C, kAccBlock, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem);
      if (e != cudaSuccess) return e;
      k_msm_fold<C, kAccBlock, false>
          <<<(unsigned)(device_sm_count() * kGasCtasPerSm), kAccBlock, smem, st>>>(f);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  phase_mark(3, st);
  // ---- 4: bucket reduction
  // combination order: instances grouped by (rows, window width), so a warp's
  // Horner chains have one length
  std::vector<uint32_t> order(num);
  for (int i = 0; i < num; ++i) order[i] = (uint32_t)i;
  std::stable_sort(order.begin(), order.end(), [&](uint32_t x, uint32_t y) {
    return std::make_pair(L.inst[x].Wr, L.inst[x].c) < std::make_pair(L.inst[y].Wr, L.inst[y].c);
  });
  Scratch rs;
  e = rs.alloc(up(num * 4ull) + 2 * up(L.elems * sizeof(Jac<F>)) + up(L.rows * sizeof(Jac<F>)), st);
  if (e != cudaSuccess) return e;
  char* q = rs.as<char>();
  auto take_r = [&](uint64_t b) { char* r = q; q += up(b); return r; };
  uint32_t* d_order = reinterpret_cast<uint32_t*>(take_r(num * 4ull));
  e = upload_words(d_order, order.data(), num * 4ull, st);
  if (e != cudaSuccess) return e;
  RedArgs<C> r;
  r.inst = d_inst;
  r.num = (uint32_t)num;
  r.elems = L.elems;
  r.poff = poff;
  r.partial = a.partial;
  r.jac = jac;
  r.R = reinterpret_cast<Jac<F>*>(take_r(L.elems * sizeof(Jac<F>)));
  r.S = reinterpret_cast<Jac<F>*>(take_r(L.elems * sizeof(Jac<F>)));
  r.row = reinterpret_cast<Jac<F>*>(take_r(L.rows * sizeof(Jac<F>)));
  if (L.elems) {
    const unsigned eb = (unsigned)((L.elems + kJacThreads - 1) / kJacThreads);
    if (L.direct) {
      k_msm_elems<C, true><<<eb, kJacThreads, 0, st>>>(r);
    } else {
      k_msm_elems<C, false><<<eb, kJacThreads, 0, st>>>(r);
    }
    uint32_t m = 0;
    for (const MsmInst& in : L.inst) m = std::max(m, elem_log(in));
    if (m > 0) k_msm_tree<C><<<L.ctas, kJacThreads, 0, st>>>(r, 0);
    if (m > kTreeLog) k_msm_tree<C><<<L.rows, kJacThreads, 0, st>>>(r, 1);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  phase_mark(4, st);
  // ---- 5: window sums and their combination, every instance in one launch
  if (num) {
    k_msm_rows<C><<<(L.rows + 15) / 16, 64, 0, st>>>(r, L.rows);
    k_msm_combine<C><<<(num + 7) / 8, 32, 0, st>>>(r, d_order, hdr, out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  phase_mark(5, st);
  return cudaSuccess;
}

// pre_c > 0: the bases hold precomputed window multiples for width pre_c,
// pre_stride points apart.  phi > 0: the points' images are phi rows after them, and
// scalars are split.  lean: the plan of least workspace, with whole scalars and the widths
// by which sizes are admitted (msm_counts): also that of a batch whose digits, buckets or
// rows would not fit their 31-bit indices.
template <class C>
Layout plan(int curve, uint32_t num, const uint64_t* sizes, const uint64_t* point_off,
            const uint64_t* scalar_off, int pre_c, uint64_t pre_stride, uint64_t phi, bool lean) {
  Layout L;
  if (phi) {  // split where that is the better half of the work
    BySize<double> gain;
    double sum = 0;
    for (uint32_t i = 0; i < num && !lean; ++i)
      sum += gain.get(sizes[i], [&] { return msm_split_gain(sizes[i], num, 0); });
    if (lean || sum < 0) phi = 0;
  }
  L.inst.resize(num);
  L.phi = phi;
  BySize<int> width;
  for (uint32_t i = 0; i < num; ++i) {
    MsmInst& m = L.inst[i];
    m.n = (uint32_t)sizes[i];
    m.c = (uint32_t)(pre_c > 0 ? pre_c : width.get(sizes[i], [&] {
      return lean ? msm_admitted_window(curve, sizes[i]) : msm_window(curve, sizes[i], num, phi > 0);
    }));
    m.W = (uint32_t)(phi ? half_windows<C>((int)m.c) : windows_for(curve, (int)m.c));
    m.bucket_base = (uint32_t)L.buckets;
    m.point_off = point_off[i];
    m.scalar_off = scalar_off[i];
    m.pre_stride = pre_c > 0 ? pre_stride : 0;
    m.phi = phi;
    m.Wr = pre_c > 0 ? 1u : m.W;
    L.buckets += (uint64_t)m.Wr << (m.c - 1);
    L.entries_max += (uint64_t)m.W * m.n * (phi ? 2 : 1);
    L.total_points += m.n;
    if (!lean && (L.entries_max >= kMsmMaxDigits || L.buckets >= kMsmMaxDigits || 2 * phi >= kMsmMaxDigits))
      return plan<C>(curve, num, sizes, point_off, scalar_off, pre_c, pre_stride, 0, true);
  }
  finish_plan<C::Fp::N>(curve, L, sizes, 0, lean);
  return L;
}

// run(false), or, where its workspace is refused, run(true) with the lean plan: chunks of 8
// entries, short elements, wider windows and the points' images take up to 3 times (and a
// few MB for the smallest calls) the workspace that the call needs.
template <class Run>
cudaError_t run_or_lean(Run run) {
  cudaError_t e = run(false);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    e = run(true);
  }
  return e;
}

template <class C>
cudaError_t msm_points(int curve, uint32_t num, const uint64_t* offsets, const uint32_t* points,
                       const uint32_t* scalars, uint32_t* out, cudaStream_t st) {
  using F = typename C::Fp;
  const uint64_t total = offsets[num] - offsets[0];
  std::vector<uint64_t> sizes(num), poff(num);
  for (uint32_t i = 0; i < num; ++i) {
    sizes[i] = offsets[i + 1] - offsets[i];
    poff[i] = offsets[i] - offsets[0];
  }
  return run_or_lean([&](bool lean) {
    const Layout L = plan<C>(curve, num, sizes.data(), poff.data(), poff.data(), 0, 0, C::GLV ? total : 0, lean);
    return run_set<C>(curve, L, nullptr, scalars + offsets[0] * 8, out, st, nullptr, points + offsets[0] * 2 * F::N);
  });
}

// The uniform per-instance layout of a device-sized batch (window width c, or
// the library's width for bases with window multiples of width pre_c) with the
// capacity totals: cap scalar rows in num instances.  phi, lean and the indices as in
// plan; c = 0: the library's width for the mean size.
template <class C>
Layout plan_uniform(int curve, uint32_t num, int c, uint64_t cap, int pre_c, uint64_t pre_stride, uint64_t phi,
                    bool lean) {
  Layout L;
  MsmInst m{};
  const uint64_t mean = num ? std::max<uint64_t>(cap / num, 2) : 2;
  if (phi && (lean || msm_split_gain(mean, num, c) < 0)) phi = 0;
  if (pre_c <= 0 && c <= 0) {
    c = lean ? msm_admitted_window(curve, mean) : msm_window(curve, mean, num, phi > 0);
    const uint64_t W = (uint64_t)windows_for(curve, c);
    if (W * cap >= kMsmMaxDigits || (num * W) << (c - 1) >= kMsmMaxDigits) c = msm_admitted_window(curve, mean);
  }
  m.c = (uint32_t)(pre_c > 0 ? pre_c : c);
  if (phi && ((uint64_t)half_windows<C>((int)m.c) * cap * 2 >= kMsmMaxDigits || 2 * phi >= kMsmMaxDigits)) phi = 0;
  m.W = (uint32_t)(phi ? half_windows<C>((int)m.c) : windows_for(curve, (int)m.c));
  m.Wr = pre_c > 0 ? 1u : m.W;
  m.pre_stride = pre_c > 0 ? pre_stride : 0;
  m.phi = phi;
  L.phi = phi;
  L.inst.assign(num, m);
  for (uint32_t i = 0; i < num; ++i) L.inst[i].bucket_base = (uint32_t)(i * ((uint64_t)m.Wr << (m.c - 1)));
  L.buckets = (uint64_t)num * ((uint64_t)m.Wr << (m.c - 1));
  L.entries_max = cap * m.W * (phi ? 2 : 1);
  L.total_points = cap;
  finish_plan<C::Fp::N>(curve, L, nullptr, mean, lean);
  return L;
}

// Ragged MSMs over caller points with device offsets[num + 1] (offsets[0] = 0),
// at most cap rows, one window width c for every instance.
template <class C>
cudaError_t msm_points_dev(int curve, uint32_t num, uint64_t cap, const uint64_t* offsets, int c,
                           const uint32_t* points, const uint32_t* scalars, uint32_t* out, cudaStream_t st) {
  DevRows dev{offsets, 0, 0, cap};
  return run_or_lean([&](bool lean) {
    const Layout L = plan_uniform<C>(curve, num, c, cap, 0, 0, C::GLV ? cap : 0, lean);
    return run_set<C>(curve, L, nullptr, scalars, out, st, &dev, points);
  });
}

struct Bases {
  int curve;
  uint64_t n;
  uint32_t* mont;          // AoS Montgomery affine, owned
  uint64_t phi = 0;        // rows to the points' images under the endomorphism (0: none)
  uint32_t* pre = nullptr; // window multiples (window-major, window 0 = mont copy), owned
  int pre_c = 0;           // window width of pre (0: none)
};

// Fills bs->pre with 2^(c w) P_i for w < W (W windows of width c).
template <class C>
cudaError_t precompute_t(Bases* bs, int c, cudaStream_t st) {
  using F = typename C::Fp;
  constexpr int N = F::N;
  const uint32_t W = (uint32_t)windows_for(bs->curve, c);
  const uint64_t n = bs->n;
  if ((uint64_t)W * n >= (1ull << 31)) return cudaErrorInvalidValue;  // 31-bit point indices
  uint32_t* pre = nullptr;
  cudaError_t e = cudaMalloc(&pre, std::max<uint64_t>(W * n, 1) * 2 * N * 4);
  if (e != cudaSuccess) return e;
  if (n) e = cudaMemcpyAsync(pre, bs->mont, n * 2 * N * 4, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess && n && W > 1) {
    Scratch m;
    e = m.alloc(soa_bytes<F>(n), st);
    if (e == cudaSuccess) {
      ShiftArgs<C> a;
      a.pre = pre;
      a.n = n;
      a.W = W;
      a.c = (uint32_t)c;
      a.M = SoA<F>{m.as<uint4>(), n};
      uint64_t ctas = (uint64_t)device_sm_count() * kGasCtasPerSm;
      uint64_t per = (n + ctas - 1) / ctas;
      if (per < 32) per = 32;
      ctas = (n + per - 1) / per;
      a.per_cta = per;
      const size_t smem = sizeof(GasSmem<N, kAccBlock>);
      e = cudaFuncSetAttribute(k_bases_shift<C, kAccBlock>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e == cudaSuccess) {
        k_bases_shift<C, kAccBlock><<<(unsigned)ctas, kAccBlock, smem, st>>>(a);
        e = cudaGetLastError();
      }
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the old table may be in use until here
  if (e != cudaSuccess) {
    cudaFree(pre);
    return e;
  }
  if (bs->pre) cudaFree(bs->pre);
  bs->pre = pre;
  bs->pre_c = c;
  return cudaSuccess;
}

// Ragged MSMs over resident bases with device sizes[num] (scalar rows back to
// back, at most cap in all), one window width for every instance (the table's
// when the handle has window multiples, else c).
template <class C>
cudaError_t msm_bases_dev_t(Bases* bs, uint32_t num, uint64_t cap, const uint64_t* sizes, int c,
                            const uint32_t* scalars, uint32_t* out, cudaStream_t st) {
  DevRows dev{sizes, 1, bs->n, cap};
  return run_or_lean([&](bool lean) {
    const Layout L =
        plan_uniform<C>(bs->curve, num, c, cap, bs->pre ? bs->pre_c : 0, bs->n, bs->pre ? 0 : bs->phi, lean);
    return run_set<C>(bs->curve, L, bs->pre ? bs->pre : bs->mont, scalars, out, st, &dev);
  });
}

template <class C>
cudaError_t msm_bases_t(Bases* bs, uint32_t num_vectors, const uint64_t* vec_sizes,
                        const uint32_t* scalars, uint32_t* out, cudaStream_t st) {
  // instance v uses bases [0, size_v) and the scalar rows that follow the
  // previous instances' (all n bases each when vec_sizes is null)
  std::vector<uint64_t> sizes(num_vectors, bs->n), poff(num_vectors, 0), soff(num_vectors);
  uint64_t acc = 0;
  for (uint32_t v = 0; v < num_vectors; ++v) {
    if (vec_sizes) sizes[v] = vec_sizes[v];
    soff[v] = acc;
    acc += sizes[v];
  }
  return run_or_lean([&](bool lean) {
    const Layout L = plan<C>(bs->curve, num_vectors, sizes.data(), poff.data(), soff.data(), bs->pre ? bs->pre_c : 0,
                             bs->n, bs->pre ? 0 : bs->phi, lean);
    return run_set<C>(bs->curve, L, bs->pre ? bs->pre : bs->mont, scalars, out, st);
  });
}

}  // namespace msm_detail
}  // namespace ecc
