// Exact top-k (Definition "SMIPS", Section 2) on the device: the recall
// judge, and the exact kappa-NN graph (Eq. "knn-graph") for small
// collections.
//
// The collection is cut into tiles of up to ex_tile documents whose fp32
// accumulators fit shared memory.  A CTA takes a query (or, when there are
// fewer queries than CTAs, a share of its tiles) and, tile by tile, adds the
// query's terms in ascending order: the postings of a term inside the tile are
// one contiguous piece of its (document-ascending) list, distinct documents, so
// a barrier between terms makes every sum deterministic.  k_exact_bounds finds
// the pieces of the terms a batch uses.  Then the tile's documents, untouched
// ones with score 0 among them, are compared with the k-th best so far; the few
// that pass are merged by a bitonic sort of packed (score desc, id asc) keys.
// A first tile has no k-th best yet: the k-th largest of 1024 group maxima (of
// distinct documents) is a bound below it, and keeps nearly all documents out.
//
// Bound by the latency of a term's step (a posting load, a shared-memory
// update, a barrier), so the next two terms' postings are loaded ahead.  With
// the accumulators in global memory (n_docs floats per CTA, cleared before and
// after each query, every posting a scattered read-modify-write in L2 or DRAM)
// 1000 queries over 100,000 documents took 5.35 ms; here 0.71 ms (one query of 40 entries over 1M documents: 4.1 ms, here 0.12).
#include <cmath>

#include "search_impl.h"

namespace seismic {

namespace {

constexpr uint32_t kExNT = 512;
// Two CTAs per SM: 64 registers per thread, and tiles as large as leave room for two beside the sort area (k <= 256:
// 24,576 documents, 96 KB; more: 16,384 and a sort area four times as large).  1000 queries of 10..150 entries, 1M
// documents: 10.3 ms; with 16,384 documents 13.7, with three CTAs (40 registers, 14,848 documents) 11.4.
constexpr uint32_t kExCtas = 2;
constexpr uint32_t ex_area(uint32_t k) { return k <= 256u ? 1024u : 4096u; }
constexpr uint32_t ex_tile(uint32_t k) { return k <= 256u ? 24576u : 16384u; }
constexpr size_t ex_smem(uint32_t k, uint32_t tile) { return (size_t)ex_area(k) * 8 + (size_t)k * 8 + (size_t)tile * 4; }

__device__ __forceinline__ uint32_t f2ord(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t o) {
  uint32_t u = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
  return __uint_as_float(u);
}
// ascending key order = (score desc, id asc)
__device__ __forceinline__ unsigned long long mkkey(float s, uint32_t id) {
  return ((unsigned long long)(~f2ord(s)) << 32) | id;
}

constexpr uint32_t kExGroups = 1024;  // group maxima that bound a first tile's k-th best; at least kExactMaxK
constexpr size_t kExSmem = std::max(ex_smem(256, ex_tile(256)), ex_smem(kExactMaxK, ex_tile(kExactMaxK)));
static_assert(kExCtas * (kExSmem + 7u * 1024u + 1024u) <= 228u * 1024u, "two CTAs, their ExShared and what each reserves");
static_assert(kExGroups >= kExactMaxK && kExGroups % kExNT == 0, "a group maximum per result, whole groups per thread");

struct ExShared {
  uint32_t cbn, count, pass;
  unsigned long long theta;
  uint32_t lo[kExNT], hi[kExNT];
  float v[kExNT];
  uint32_t posts[kExNT / 32];
};

__device__ void ex_sort(unsigned long long *cb, uint32_t P2) {
  for (uint32_t k2 = 2; k2 <= P2; k2 <<= 1)
    for (uint32_t j = k2 >> 1; j > 0; j >>= 1) {
      for (uint32_t x = threadIdx.x; x < P2 / 2; x += kExNT) {
        const uint32_t i = ((x & ~(j - 1u)) << 1) | (x & (j - 1u)), l = i | j;
        const unsigned long long a = cb[i], b = cb[l];
        if ((a > b) == ((i & k2) == 0)) { cb[i] = b; cb[l] = a; }
      }
      __syncthreads();
    }
}

// Merges the sh.cbn buffered keys with the top-k; every thread calls it after a barrier.
__device__ void ex_merge(unsigned long long *cb, unsigned long long *tk, ExShared &sh, uint32_t k) {
  const uint32_t tid = threadIdx.x, cbn = sh.cbn, cnt = sh.count, n = cbn + cnt;
  for (uint32_t i = tid; i < cnt; i += kExNT) cb[cbn + i] = tk[i];
  uint32_t P2 = 1;
  while (P2 < n) P2 <<= 1;
  for (uint32_t i = n + tid; i < P2; i += kExNT) cb[i] = ~0ull;
  __syncthreads();
  ex_sort(cb, P2);
  const uint32_t nc = min(k, n);
  for (uint32_t i = tid; i < nc; i += kExNT) tk[i] = cb[i];
  __syncthreads();
  if (tid == 0) {
    sh.count = nc;
    sh.cbn = 0;
    sh.theta = nc == k ? tk[k - 1] : ~0ull;
  }
  __syncthreads();
}

__device__ void ex_write(const ExactArgs &a, uint32_t q, const unsigned long long *tk, uint32_t count) {
  for (uint32_t i = threadIdx.x; i < a.k; i += kExNT) {
    const bool ok = i < count;
    a.ids[(size_t)q * a.k + i] = ok ? (uint32_t)(tk[i] & 0xFFFFFFFFu) : SEISMIC_NONE_ID;
    a.scores[(size_t)q * a.k + i] = ok ? ord2f(~(uint32_t)(tk[i] >> 32)) : -INFINITY;
  }
}

// bounds[t][x] = first posting of list t whose document is in tile x or a
// later one, for every term t of the queries (the first entry to claim a term
// does its list).
__global__ void __launch_bounds__(kExNT) k_exact_bounds(const ExactArgs a) {
  __shared__ uint32_t claimed;
  const uint32_t q = blockIdx.x;
  for (uint64_t e = a.q_indptr[q] + blockIdx.y; e < a.q_indptr[q + 1]; e += gridDim.y) {
    const uint32_t t = a.q_terms[e];
    if (a.q_vals[e] == 0.0f || t >= a.dim) continue;  // uniform
    if (threadIdx.x == 0) claimed = atomicExch(a.claim + t, 1u);
    __syncthreads();
    const uint32_t done = claimed;
    __syncthreads();
    if (done) continue;
    const uint32_t p0 = a.full_ptr[t], p1 = a.full_ptr[t + 1];
    uint32_t *b = a.bounds + (size_t)t * (a.tiles + 1);
    for (uint64_t p = (uint64_t)p0 + threadIdx.x; p <= p1; p += kExNT) {
      const uint32_t from = p == p0 ? 0u : a.full_doc[p - 1] / a.tile + 1u;
      const uint32_t to = p == p1 ? a.tiles : a.full_doc[p] / a.tile;
      for (uint32_t x = from; x <= to; x++) b[x] = (uint32_t)p;
    }
  }
}

__global__ void __launch_bounds__(kExNT, kExCtas) k_exact(const ExactArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ ExShared sh;
  unsigned long long *cb = reinterpret_cast<unsigned long long *>(sm);  // sort area: buffer + top-k
  unsigned long long *tk = cb + a.area;
  float *acc = reinterpret_cast<float *>(tk + a.k);
  const uint32_t tid = threadIdx.x;
  const uint64_t items = (uint64_t)a.nq * a.splits;
  bool dirty = true;  // the accumulators are not all 0
  for (uint64_t it = blockIdx.x; it < items; it += gridDim.x) {
    const uint32_t q = (uint32_t)(it / a.splits), part = (uint32_t)(it % a.splits);
    const uint64_t qb = a.q_indptr[q], qe = a.q_indptr[q + 1];
    if (tid == 0) { sh.cbn = 0; sh.count = 0; sh.theta = ~0ull; }
    for (uint32_t x = (uint32_t)((uint64_t)a.tiles * part / a.splits);
         x < (uint32_t)((uint64_t)a.tiles * (part + 1) / a.splits); x++) {
      if ((uint64_t)x * a.tile >= a.n_docs) break;  // uniform
      const uint32_t d0 = x * a.tile, nd = min(a.tile, a.n_docs - d0);
      // Where a document without a posting (score 0) cannot enter any more, a tile costs what its postings cost:
      // nothing without any, and with few of them only they are offered.  (4000 queries of one rare term, 1M
      // documents: 1.29 ms; with every tile cleared and compared whole 3.77, and 1.53 with accumulators in global memory.)
      enum { kNone, kFew, kAll } mode = kAll;
      for (uint64_t e0 = qb; e0 == qb || e0 < qe; e0 += kExNT) {  // the query's entries, kExNT at a time
        const uint32_t ne = (uint32_t)min((uint64_t)kExNT, qe - e0);
        __syncthreads();  // the entries before these are no longer read
        uint32_t len = 0u;
        if (tid < ne) {
          const uint32_t t = a.q_terms[e0 + tid];
          const float v = a.q_vals[e0 + tid];
          const bool on = v != 0.0f && t < a.dim;
          const uint32_t *b = a.bounds + (size_t)(on ? t : 0u) * (a.tiles + 1) + x;
          const uint32_t lo = on ? b[0] : 0u, hi = on ? b[1] : 0u;
          sh.v[tid] = v;
          sh.lo[tid] = lo;
          sh.hi[tid] = hi;
          len = hi - lo;
        }
        len = __reduce_add_sync(0xffffffffu, len);
        if ((tid & 31u) == 0) sh.posts[tid >> 5] = len;
        __syncthreads();
        if (e0 == qb) {
          const bool zeros = sh.count < a.k || mkkey(0.0f, d0) <= sh.theta;
          uint32_t posts = 0u;
          if (qe - qb <= kExNT && !zeros) {
            for (uint32_t w = 0; w < kExNT / 32; w++) posts += sh.posts[w];
            mode = posts == 0u ? kNone : posts + a.k <= a.area ? kFew : kAll;
          }
          if (mode == kNone) break;
          const uint32_t waiting = sh.cbn;  // offers of tiles before (then the top-k is full)
          if (waiting && (mode == kAll || waiting + posts + a.k > a.area)) ex_merge(cb, tk, sh, a.k);
          if (dirty) {
            for (uint32_t i = tid; i < a.tile; i += kExNT) acc[i] = 0.0f;
            __syncthreads();
          }
          dirty = mode == kAll;
        }
        // postings of the terms e and e + 1 are in registers while e is added
        uint32_t dn[2] = {0u, 0u};
        float xn[2] = {0.0f, 0.0f};
        auto fetch = [&](uint32_t e, uint32_t &d, float &v) {
          if (e < ne && sh.lo[e] + tid < sh.hi[e]) {
            d = a.full_doc[sh.lo[e] + tid];
            v = a.full_val[sh.lo[e] + tid];
          }
        };
        fetch(0, dn[0], xn[0]);
        fetch(1, dn[1], xn[1]);
        for (uint32_t e = 0; e < ne; e++) {
          const uint32_t lo = sh.lo[e], hi = sh.hi[e], d = dn[0];
          const float v = sh.v[e], xv = xn[0];
          dn[0] = dn[1];
          xn[0] = xn[1];
          fetch(e + 2, dn[1], xn[1]);
          if (lo >= hi) continue;  // uniform
          if (lo + tid < hi) acc[d - d0] = fmaf(v, xv, acc[d - d0]);
          for (uint64_t p = (uint64_t)lo + tid + kExNT; p < hi; p += kExNT) {
            const uint32_t dd = a.full_doc[p] - d0;
            acc[dd] = fmaf(v, a.full_val[p], acc[dd]);
          }
          __syncthreads();
        }
      }
      if (mode == kNone) continue;
      if (mode == kFew) {
        const unsigned long long theta = sh.theta;
        for (uint32_t e = tid >> 5; e < (uint32_t)(qe - qb); e += kExNT / 32)
          for (uint64_t p = (uint64_t)sh.lo[e] + (tid & 31u); p < sh.hi[e]; p += 32u) {
            const uint32_t d = a.full_doc[p];
            // a document of several terms is offered once: what is left of it, 0, does not enter (and is clear again)
            const unsigned long long key = mkkey(atomicExch(acc + (d - d0), 0.0f), d);
            if (key <= theta) cb[atomicAdd(&sh.cbn, 1u)] = key;
          }
        continue;
      }
      __syncthreads();
      // what has to be beaten: the k-th best, or a bound below it
      unsigned long long theta = sh.theta;
      if (sh.count < a.k && nd > kExGroups) {
        for (uint32_t g = tid; g < kExGroups; g += kExNT) {
          unsigned long long best = ~0ull;
          for (uint32_t i = g; i < nd; i += kExGroups) best = min(best, mkkey(acc[i], d0 + i));
          cb[g] = best;
        }
        __syncthreads();
        ex_sort(cb, kExGroups);
        theta = min(theta, cb[a.k - 1]);  // at least k documents of this tile reach it
        __syncthreads();
      }
      uint32_t n = 0;
      for (uint32_t i = tid; i < nd; i += kExNT) n += mkkey(acc[i], d0 + i) <= theta ? 1u : 0u;
      if (tid == 0) sh.pass = 0u;
      __syncthreads();
      n = __reduce_add_sync(0xffffffffu, n);
      if ((tid & 31u) == 0 && n) atomicAdd(&sh.pass, n);
      __syncthreads();
      if (sh.pass == 0) continue;
      if (sh.pass + a.k <= a.area) {
        for (uint32_t i = tid; i < nd; i += kExNT) {
          const unsigned long long key = mkkey(acc[i], d0 + i);
          if (key <= theta) cb[atomicAdd(&sh.cbn, 1u)] = key;
        }
        __syncthreads();
        ex_merge(cb, tk, sh, a.k);
      } else {  // many documents pass (ties, large k): a row of kExNT at a time, merged when the buffer fills
        for (uint32_t i0 = 0; i0 < nd; i0 += kExNT) {
          const uint32_t i = i0 + tid;
          if (i < nd) {
            const unsigned long long key = mkkey(acc[i], d0 + i);
            if (key <= theta && key <= sh.theta) cb[atomicAdd(&sh.cbn, 1u)] = key;
          }
          __syncthreads();
          const uint32_t filled = sh.cbn;
          __syncthreads();  // nobody adds to it before everybody has read it
          if (filled + kExNT + a.k > a.area) ex_merge(cb, tk, sh, a.k);
        }
        if (sh.cbn) ex_merge(cb, tk, sh, a.k);
      }
    }
    __syncthreads();
    if (sh.cbn) ex_merge(cb, tk, sh, a.k);
    if (a.splits == 1) {
      ex_write(a, q, tk, sh.count);
    } else {
      for (uint32_t i = tid; i < a.k; i += kExNT) a.part[it * a.k + i] = i < sh.count ? tk[i] : ~0ull;
    }
    __syncthreads();
  }
}

// The top-k of a query's splits.
__global__ void __launch_bounds__(kExNT) k_exact_join(const ExactArgs a) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ ExShared sh;
  unsigned long long *cb = reinterpret_cast<unsigned long long *>(sm), *tk = cb + a.area;
  const uint32_t q = blockIdx.x, n = a.splits * a.k;
  if (threadIdx.x == 0) { sh.cbn = 0; sh.count = 0; sh.theta = ~0ull; }
  __syncthreads();
  for (uint32_t i0 = 0; i0 < n; i0 += kExNT) {
    const uint32_t i = i0 + threadIdx.x;
    const unsigned long long key = i < n ? a.part[(size_t)q * n + i] : ~0ull;
    if (key < sh.theta) cb[atomicAdd(&sh.cbn, 1u)] = key;
    __syncthreads();
    const uint32_t filled = sh.cbn;
    __syncthreads();
    if (filled + kExNT + a.k > a.area) ex_merge(cb, tk, sh, a.k);
  }
  if (sh.cbn) ex_merge(cb, tk, sh, a.k);
  ex_write(a, q, tk, sh.count);
}

}  // namespace

// Fewer queries than about one and a half times the CTAs that run at once (slots): several CTAs share a query's tiles.
// Least of the rounds of CTAs times a CTA's documents; a tile's barriers count as 13,000 more (152 queries, 100,000
// documents: 3 tiles of 20,000 each 191 us, 4 of 14,286 210), a CTA's first bound on the k-th best as 4000; the
// smaller tiles only where they win.  100,000 documents, queries of 10..150 entries, with tiles of 24,576
// and as many splits as all run at once, and here: 10 queries 103 and 96 us, 67 queries 177 and 141, 200 queries 378 and 287,
// 400 queries 555 and 484.
static void ex_split(ExactArgs &a, uint32_t least, uint32_t most, uint32_t slots) {
  a.tiles = least;
  a.splits = 1;
  if (2ull * a.nq >= 3ull * slots) return;
  double best = 1e300;
  for (uint32_t tiles : {least, most}) {
    const double docs = (double)((a.n_docs + tiles - 1) / tiles);
    for (uint32_t s = 1; s <= std::min(tiles, std::max(1u, 4u * slots / a.nq)); s++) {
      if (s > 1 && (uint64_t)a.nq * s * a.k > (uint64_t)slots * kExactMaxK) break;  // the splits' results
      // rounds: a last one that is not full costs its part and a third of the rest; past one they have to win by a tenth
      // (50 queries of 40 entries, 1M documents: 6 parts 0.455 ms, 12 in two rounds 0.510)
      const double x = (double)a.nq * s / slots;
      const double rounds = x <= 1.0 ? 1.0 : x + (std::ceil(x) - x) / 3.0, per = x <= 1.0 ? (tiles + s - 1) / s : (double)tiles / s;
      const double cost = (x <= 1.0 ? 1.0 : 1.1) * rounds * (per * (docs + 13000.0) + 4000.0);
      if (cost < best) {
        best = cost;
        a.tiles = tiles;
        a.splits = s;
      }
    }
  }
}

// Working memory: the bounds table, the claim words and the splits' results; it
// depends on the index only, so it is allocated once.
size_t exact_layout(ExactArgs &a, uint32_t sms, void *base) {
  const uint32_t least = (a.n_docs + ex_tile(a.k) - 1) / ex_tile(a.k);
  const uint32_t most = (a.n_docs + ex_tile(kExactMaxK) - 1) / ex_tile(kExactMaxK);
  ex_split(a, least, most, kExCtas * sms);
  a.tile = (a.n_docs + a.tiles - 1) / a.tiles;
  a.area = ex_area(a.k);
  a.sms = sms;
  const size_t claim = ((size_t)a.dim * 4 + 255) & ~(size_t)255;
  const size_t bounds = ((size_t)a.dim * (most + 1) * 4 + 255) & ~(size_t)255;
  unsigned char *p = reinterpret_cast<unsigned char *>(base);
  a.claim = reinterpret_cast<uint32_t *>(p);
  a.bounds = reinterpret_cast<uint32_t *>(p + claim);
  a.part = reinterpret_cast<unsigned long long *>(p + claim + bounds);
  return claim + bounds + (size_t)kExCtas * sms * kExactMaxK * 8;
}

int launch_exact(ExactArgs a, cudaStream_t st) {
  if (a.k == 0 || a.k > kExactMaxK) return fail(SEISMIC_EINVAL, "exact search: k must be in 1..1024");
  const size_t smem = ex_smem(a.k, a.tile);
  static std::atomic<uint64_t> configured{0}, configured2{0};
  int rc;
  if ((rc = set_smem_limit_once(configured, (const void *)k_exact, (int)kExSmem)) ||
      (rc = set_smem_limit_once(configured2, (const void *)k_exact_join, (int)(4096 * 8 + kExactMaxK * 8))))
    return rc;
  SZ_CUDA(cudaMemsetAsync(a.claim, 0, (size_t)a.dim * 4, st));
  const uint32_t per_query = std::min<uint32_t>(64u, std::max<uint32_t>(1u, 8u * a.sms / a.nq));
  k_exact_bounds<<<dim3(a.nq, per_query), kExNT, 0, st>>>(a);
  SZ_CUDA(cudaGetLastError());
  const uint64_t items = (uint64_t)a.nq * a.splits;
  k_exact<<<(uint32_t)std::min<uint64_t>(items, 8ull * a.sms), kExNT, smem, st>>>(a);
  SZ_CUDA(cudaGetLastError());
  if (a.splits > 1) {
    k_exact_join<<<a.nq, kExNT, (size_t)(a.area + a.k) * 8, st>>>(a);
    SZ_CUDA(cudaGetLastError());
  }
  return SEISMIC_OK;
}

}  // namespace seismic
