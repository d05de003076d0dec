// Query processing: Algorithm "Query processing with Seismic" (Section 4.5),
// one CTA per query.
//
//  H0  the query is held in shared memory as a vocabulary bitmap plus a
//      popcount rank per 32-term word and its values in term order: a lookup
//      is one 4-byte shared load when the term is absent (the common case)
//      and two more when present.  About 8 KB per query instead of a 122 KB
//      dense vector, so several queries share an SM.
//  H1  list terms: the top-`cut` query terms by (value desc, term asc), or
//      the alpha_q-MSS of q (Section 3.2 applied to the query).
//  H2  r_b = <q, S_b> for every block of the list with the full query.  The
//      summaries are stored term-major per list (a column per term, blocks
//      ascending), so only the query's columns are read; each warp owns a
//      partial-score array and the partials are added in warp order, which
//      makes r_b deterministic.
//  H3  blocks are ordered by (r desc, block asc) with a bitonic sort.
//  H4  a block is skipped iff the top-k is full and r < hf * theta (or
//      r < theta / hf); r is non-increasing and theta non-decreasing along
//      the order, so the first skipped block ends the list.
//  H5  forward rows: each warp takes some of a wave's documents and goes over
//      their rows laid end to end (group 1), or groups of G lanes score one
//      document each; a row is a record of 8-entry chunks read with 16- and
//      32-byte vector loads.  With lane groups every row of a wave is
//      prefetched into L2 at its start, one TMA bulk prefetch per document; the
//      member lists of the next blocks are always.  Each document is scored at
//      most once per query (a global bitmap per persistent CTA, a bitmap in
//      shared memory for a small collection, or a bounded shared-memory hash set).
//  H6  top-k by (score desc, id asc): candidates that beat the k-th score are
//      collected per wave and merged by rank.
//  H7  kappa-NN expansion of the top-k after the lists (S fixed first).
//
// Waves: with wave = 1 every block is evaluated before the next skip test,
// which is exactly the sequential order of the algorithm (the final heap
// after a block does not depend on the order of its documents).  With wave =
// W the next W blocks that pass the test against the threshold at the wave's
// start are evaluated together (batch-synchronous).
#include <algorithm>

#include "search_common.cuh"

namespace seismic {

namespace {

using namespace dev;

// Insert d into the per-query seen set; true when d was not there before (or
// the set cannot tell, in which case d is scored again).  A set that is three
// quarters full stops probing: a document takes its slot whatever is there, so a lookup
// stays one atomic, and what was there is forgotten.  (Few documents are met
// twice -- 3 % of a search of 34,000 -- so forgetting costs little, while 16 probes
// per document make one query over 1M documents take 2.7 ms instead of 1.5.)
__device__ __forceinline__ bool seen_insert(uint32_t *tab, uint32_t hs_mask, uint32_t d, bool crowded, uint32_t *full) {
  const uint32_t key = d + 1u;
  uint32_t h = (d * 0x9E3779B1u) & hs_mask;
  if (!crowded) {
#pragma unroll 1
    for (int p = 0; p < 16; p++) {
      uint32_t old = atomicCAS(&tab[h], 0u, key);
      if (old == 0u) return true;
      if (old == key) return false;
      h = (h + 1u) & hs_mask;
    }
  } else if (atomicExch(&tab[h], key) == key) {
    return false;
  }
  *full = 1u;
  return true;
}

template <int NT>
__device__ uint32_t block_rank_scan(const uint32_t *bits, uint16_t *rank, uint32_t W, uint32_t *wtmp) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nw = NT / 32;
  const uint32_t per = (W + NT - 1) / NT, lo = min(W, tid * per), hi = min(W, lo + per);
  uint32_t s = 0;
  for (uint32_t i = lo; i < hi; i++) s += __popc(bits[i]);
  uint32_t x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wtmp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t v = lane < nw ? wtmp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane < nw) wtmp[lane] = v;
  }
  __syncthreads();
  uint32_t base = (warp ? wtmp[warp - 1] : 0) + x - s;
  for (uint32_t i = lo; i < hi; i++) {
    rank[i] = (uint16_t)min(base, 65535u);
    base += __popc(bits[i]);
  }
  const uint32_t total = wtmp[nw - 1];
  __syncthreads();
  return total;
}

// The query's shared-memory arrays.  Each is addressed from the dynamic
// shared-memory base and its offset in the launch arguments (constant bank)
// when used, so no pointer to them stays live in a register.
extern __shared__ __align__(16) unsigned char g_sm[];

struct WarpDocs;

struct Smem {
  const SearchArgs &a;
  uint32_t *seen;  // this CTA's seen bitmap (global memory, or shared for a small collection), or NULL: the hash set
  uint32_t turn;   // the wave's candidate counter
  __device__ __forceinline__ uint32_t *qbits() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_qbits); }
  __device__ __forceinline__ uint16_t *qrank() const { return reinterpret_cast<uint16_t *>(g_sm + a.off_qrank); }
  __device__ __forceinline__ float *qval() const { return reinterpret_cast<float *>(g_sm + a.off_qval); }
  __device__ __forceinline__ uint16_t *qterm() const { return reinterpret_cast<uint16_t *>(g_sm + a.off_qterm); }
  __device__ __forceinline__ uint16_t *cutT() const { return reinterpret_cast<uint16_t *>(g_sm + a.off_cut); }
  __device__ __forceinline__ float *aq() const { return reinterpret_cast<float *>(g_sm + a.off_aq); }
  __device__ __forceinline__ float *part() const { return reinterpret_cast<float *>(g_sm + a.off_part); }
  __device__ __forceinline__ unsigned long long *keys() const { return reinterpret_cast<unsigned long long *>(g_sm + a.off_keys); }
  __device__ __forceinline__ uint32_t *clo() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_clo); }
  __device__ __forceinline__ uint32_t *chi() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_chi); }
  __device__ __forceinline__ uint32_t *hash() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_hash); }
  __device__ __forceinline__ float *tk_s() const { return reinterpret_cast<float *>(g_sm + a.off_tk_s); }
  __device__ __forceinline__ float *tmp_s() const { return reinterpret_cast<float *>(g_sm + a.off_tmp_s); }
  __device__ __forceinline__ float *cand_s() const { return reinterpret_cast<float *>(g_sm + a.off_cand_s); }
  __device__ __forceinline__ uint32_t *tk_id() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_tk_id); }
  __device__ __forceinline__ uint32_t *tmp_id() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_tmp_id); }
  __device__ __forceinline__ uint32_t *cand_id() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_cand_id); }
  __device__ __forceinline__ uint8_t *cand_ok() const { return reinterpret_cast<uint8_t *>(g_sm + a.off_cand_ok); }
  __device__ __forceinline__ uint32_t *bptr() const { return reinterpret_cast<uint32_t *>(g_sm + a.off_bptr); }
  __device__ __forceinline__ WarpDocs *wdocs() const { return reinterpret_cast<WarpDocs *>(g_sm + a.off_wdocs); }
  __device__ __forceinline__ unsigned char *wqueue() const { return g_sm + a.off_wqueue; }
  __device__ __forceinline__ uint16_t *cand_i() const { return reinterpret_cast<uint16_t *>(g_sm + a.off_cand_i); }
  __device__ __forceinline__ uint8_t *fresh() const { return reinterpret_cast<uint8_t *>(g_sm + a.off_fresh); }
  __device__ __forceinline__ uint8_t *qfilt() const { return reinterpret_cast<uint8_t *>(g_sm + a.off_qfilt); }
};

struct Shared {
  uint32_t q, nzq, ncut, count, nvalid, hash_full, hash_n, crowded, bad;
  uint32_t ncand[2];  // candidates of a wave; waves take turns, so one may begin while another's count is still read
  float hf;
  uint32_t cut;
  uint32_t wtmp[32];
  unsigned long long st[SEISMIC_STATS_N];
};

// Members of the current list: of the blocks keys[0 .. nw) (sorted positions),
// as one run -- member i is found by walking the blocks' sizes in shared memory,
// so forming a wave needs no barrier -- or, with nw = 0, the list's own order.
// Either way starting with member i0.
struct ListSrc {
  const unsigned long long *keys;
  const uint32_t *bptr;
  uint32_t nw, i0;
  const uint32_t *ids;
  const unsigned long long *rows;
  __device__ __forceinline__ uint32_t at(uint32_t i) const {
    i += i0;
    if (nw == 0) return i;
    uint32_t b = (uint32_t)(keys[0] & 0xFFFFFFFFu), lo = bptr[b], nd = bptr[b + 1] - lo;
    for (uint32_t w = 1; w < nw && i >= nd; w++) {
      i -= nd;
      b = (uint32_t)(keys[w] & 0xFFFFFFFFu);
      lo = bptr[b];
      nd = bptr[b + 1] - lo;
    }
    return lo + i;
  }
  __device__ __forceinline__ void fetch(uint32_t i, uint32_t &d, unsigned long long &r) const {
    const uint32_t m = at(i);
    d = __ldg(ids + m);
    r = __ldg(rows + m);
  }
};

// Documents by the graph: a seed document and its neighbours (ids = NULL), or
// the neighbours of the documents ids[..], starting with the i0-th.
struct NeighbourSrc {
  const uint32_t *ids, *knn;
  const unsigned long long *frow;
  uint32_t doc, kappa, bits, i0;
  __device__ __forceinline__ void fetch(uint32_t i, uint32_t &d, unsigned long long &r) const {
    i += i0;
    if (ids) d = knn_entry(knn, bits, (uint64_t)ids[i / kappa] * kappa + (i % kappa));
    else d = i == 0 ? doc : knn_entry(knn, bits, (uint64_t)doc * kappa + (i - 1));
    r = d == SEISMIC_NONE_ID ? 0ull : __ldg(frow + d);
  }
};

// Ranks m candidates -- with `part`, those of the wave's members from .. to --
// among the cnt entries of the top-k, into tmp; returns the new count.  Ends
// with a barrier; sh.nvalid is used and has to be 0 (merge_commit clears it).
template <int NT>
__device__ uint32_t merge_rank(const SearchArgs &a, Smem &s, Shared &sh, uint32_t m, bool part, uint32_t from,
                               uint32_t to) {
  const int tid = threadIdx.x;
  const uint32_t cnt = sh.count, k = a.k;
  // With the global seen bitmap a document becomes fresh once per query, so no
  // candidate repeats a heap entry or another candidate.  The bounded hash set
  // may score a document again when it is crowded: there repeats are dropped.
  const bool repeats = s.seen == nullptr, check = repeats || part;
  uint32_t nvalid = m;
  if (check) {
    const bool dupcheck = repeats && sh.hash_full != 0u;
    auto in = [&](uint32_t i) { return !part || (s.cand_i()[i] >= from && s.cand_i()[i] < to); };
    for (uint32_t i = tid; i < m; i += NT) {
      const uint32_t id = s.cand_id()[i];
      uint8_t ok = in(i) ? 1 : 0;
      if (ok && repeats)
        for (uint32_t j = 0; j < cnt; j++)
          if (s.tk_id()[j] == id) { ok = 0; break; }
      if (ok && dupcheck)
        for (uint32_t j = 0; j < i; j++)
          if (s.cand_id()[j] == id && in(j)) { ok = 0; break; }
      s.cand_ok()[i] = ok;
      if (ok) atomicAdd(&sh.nvalid, 1u);
    }
    __syncthreads();
    nvalid = sh.nvalid;
  }
  for (uint32_t i = tid; i < m; i += NT) {
    if (check && !s.cand_ok()[i]) continue;
    const float sc = s.cand_s()[i];
    const uint32_t id = s.cand_id()[i];
    uint32_t lo = 0, hi = cnt;  // topk entries better than (sc, id)
    while (lo < hi) {
      uint32_t mid = (lo + hi) >> 1;
      if (better(s.tk_s()[mid], s.tk_id()[mid], sc, id)) lo = mid + 1; else hi = mid;
    }
    uint32_t r = lo;
    for (uint32_t j = 0; j < m; j++)
      if ((!check || s.cand_ok()[j]) && better(s.cand_s()[j], s.cand_id()[j], sc, id)) r++;
    if (r < k) { s.tmp_s()[r] = sc; s.tmp_id()[r] = id; }
  }
  for (uint32_t i = tid; i < cnt; i += NT) {
    const float sc = s.tk_s()[i];
    const uint32_t id = s.tk_id()[i];
    uint32_t r = i;
    for (uint32_t j = 0; j < m; j++)
      if ((!check || s.cand_ok()[j]) && better(s.cand_s()[j], s.cand_id()[j], sc, id)) r++;
    if (r < k) { s.tmp_s()[r] = sc; s.tmp_id()[r] = id; }
  }
  __syncthreads();
  return min(k, cnt + nvalid);
}

// Sets sh.crowded once the hash set is three quarters full: by one thread, between a
// wave's last barrier and the next one, so that it is the same for all of a wave's documents.
__device__ __forceinline__ void note_crowded(const SearchArgs &a, const Smem &s, Shared &sh) {
  if (!s.seen && sh.hash_n > a.HS / 4 * 3) sh.crowded = 1u;
}

// Makes the nc ranked entries the top-k; `done` also drops the wave's candidates.
template <int NT>
__device__ void merge_commit(const SearchArgs &a, Smem &s, Shared &sh, uint32_t nc, bool done) {
  const int tid = threadIdx.x;
  for (uint32_t i = tid; i < nc; i += NT) { s.tk_s()[i] = s.tmp_s()[i]; s.tk_id()[i] = s.tmp_id()[i]; }
  if (tid == 0) {
    sh.count = nc;
    sh.nvalid = 0;
    if (done) sh.ncand[s.turn ^ 1u] = 0;
    note_crowded(a, s, sh);
  }
  __syncthreads();
}

// Scores up to CAND documents of a source; ends with a barrier.
template <int G, int NT, class Src>
__device__ void eval_wave(const SearchArgs &a, Smem &s, Shared &sh, uint32_t n, const Src &src, int knn_stage) {
  constexpr int NG = NT / G;
  const int tid = threadIdx.x, grp = tid / G, gl = tid % G;
  const uint32_t lane = tid & 31;
  const uint32_t gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(uint32_t)(G - 1)));
  const bool full = sh.count == a.k;
  const float th = full ? s.tk_s()[a.k - 1] : -INFINITY;
  const uint32_t thid = full ? s.tk_id()[a.k - 1] : 0u;
  if (a.prefetch && n > (uint32_t)NG) {  // every row of the wave into L2, one bulk prefetch each
    for (uint32_t i = tid; i < n; i += NT) {
      uint32_t d;
      unsigned long long row;
      src.fetch(i, d, row);
      if (d != SEISMIC_NONE_ID) prefetch_row(a.fwd_data, row, a.fp16);
    }
  }
  // Software pipeline per lane group: the next document's (id, row) are loaded
  // while the current one is scored, and the seen-bitmap test is issued with
  // the row's loads and read after the dot (a seen document's score is dropped).
  const bool crowded = sh.crowded != 0u;
  uint32_t dn = SEISMIC_NONE_ID;
  unsigned long long rn = 0ull;
  if ((uint32_t)grp < n) src.fetch(grp, dn, rn);
  for (uint32_t i = grp; i < n; i += NG) {
    const uint32_t d = dn;
    const unsigned long long row = rn;
    if (i + NG < n) src.fetch(i + NG, dn, rn);
    if (d == SEISMIC_NONE_ID) continue;
    uint32_t old = 0u, fresh = 0u;
    const uint32_t bit = 1u << (d & 31);
    if (gl == 0) {
      if (s.seen) old = atomicOr(s.seen + (d >> 5), bit);
      else if (seen_insert(s.hash(), a.HS - 1u, d, crowded, &sh.hash_full)) { fresh = 1u; atomicAdd(&sh.hash_n, 1u); }
    }
    const float p = row_dot<G>(a.fwd_data, row, a.fp16, gl, gmask, s.qbits(), s.qrank(), s.qval());
    if (s.seen) fresh = (old & bit) ? 0u : 1u;
    fresh = __shfl_sync(gmask, fresh, 0, G);
    if (!fresh) continue;
    if (gl == 0) {
      if (a.stats) {
        atomicAdd(&sh.st[knn_stage ? SEISMIC_ST_KNN_DOCS : SEISMIC_ST_DOCS], 1ull);
        atomicAdd(&sh.st[knn_stage ? SEISMIC_ST_KNN_NNZ : SEISMIC_ST_DOC_NNZ], (unsigned long long)a.fwd_nnz[d]);
      }
      if (!full || better(p, d, th, thid)) {
        uint32_t pos = atomicAdd(&sh.ncand[s.turn], 1u);
        s.cand_s()[pos] = p;
        s.cand_id()[pos] = d;
      }
    }
  }
  __syncthreads();
}

// Which of 8 terms (two per word) may be in the query: bit e for term e.
__device__ __forceinline__ uint32_t probe8(const uint4 &t, const uint8_t *__restrict__ filter) {
  const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
  uint32_t m = 0;
#pragma unroll
  for (int e = 0; e < 8; e++)
    m += (uint32_t)filter[((e & 1) ? (tw[e >> 1] >> 16) : tw[e >> 1]) & (kFilter - 1u)] << e;
  return m;
}

// 16-bit value e (0 .. 7) of 8 in four words.
__device__ __forceinline__ uint32_t pick8(const uint4 &t, uint32_t e) {
  const uint32_t lo = (e & 2u) ? t.y : t.x, hi = (e & 2u) ? t.w : t.z;
  return (((e & 4u) ? hi : lo) >> ((e & 1u) * 16u)) & 0xFFFFu;
}

__device__ __forceinline__ uint32_t pick16(const uint4 &t, const uint4 &t2, uint32_t e) {
  return pick8(make_uint4((e & 8u) ? t2.x : t.x, (e & 8u) ? t2.y : t.y, (e & 8u) ? t2.z : t.z, (e & 8u) ? t2.w : t.w),
               e & 7u);
}

// Queues a unit's candidates (the bits of m): document x, position pos0 + e,
// terms t and t2.
__device__ __forceinline__ void push_candidates(uint32_t *q, uint32_t m, const uint4 &t, const uint4 &t2, uint32_t x,
                                                uint32_t pos0) {
  const uint32_t base = (x << 27) | (pos0 << 16);
  while (m) {
    const uint32_t e = __ffs(m) - 1u;
    m &= m - 1u;
    *q++ = (base + (e << 16)) | pick16(t, t2, e);
  }
}

// The warp's own arrays while it scores documents (group 1).  The queue holds,
// in document, row order, the candidates of some documents -- document (5 bits)
// | position in the row (11) | term (16); the second pass replaces an entry by
// its chunk's partial score (the chunk's first entry) or 0 -- or, for fp16 rows,
// the two partials of each unit with a hit.
struct WarpDocs {
  unsigned long long unit0[32];  // address of the document's first unit, less 32 bytes per unit of the documents before it
  unsigned long long val[32];    // fp32 rows: address of its first value
  uint32_t p0[32];               // units of the documents before it
  uint32_t doc[32];
  uint16_t nch[32];              // its 8-entry chunks
  uint16_t start[32];            // its first queue entry
  uint16_t member[32];           // its place in the wave
};
static_assert(sizeof(WarpDocs) == kWarpDocsBytes, "search_layout reserves it");

// <q, row> of one row by a whole warp, a chunk per lane: chunk partials in
// entry order, added in chunk order (every lane returns the sum).
template <bool FP16>
__device__ float warp_row(const SearchArgs &a, const Smem &s, unsigned long long row, uint32_t lane) {
  const uint8_t *rec = row_base(a.fwd_data, row);
  const uint32_t nch = (uint32_t)(row >> 32);
  float p = 0.0f;
  for (uint32_t c0 = 0; c0 < nch; c0 += 32) {
    const uint32_t c = c0 + lane;
    float acc = 0.0f;
    if (c < nch) {
      const uint4 t = ldg_na(chunk_terms(rec, c, FP16));
      const uint8_t *vp = chunk_vals(rec, nch, c, FP16);
      const uint32_t tw[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
      for (int e = 0; e < 8; e++) {
        const float q = qlookup(s.qbits(), s.qrank(), s.qval(), (e & 1) ? (tw[e >> 1] >> 16) : (tw[e >> 1] & 0xFFFFu));
        if (q != 0.0f)
          acc = fmaf(q, FP16 ? __half2float(reinterpret_cast<const __half *>(vp)[e]) : reinterpret_cast<const float *>(vp)[e], acc);
      }
    }
    for (uint32_t l = 0; l < 32; l++) p += __shfl_sync(0xffffffffu, acc, l);
  }
  return p;
}

// Group 1.  A wave's documents are dealt to the warps in runs of up to 32, one
// per lane, and from there on a warp works by itself, without CTA barriers: it
// drops the documents seen before, lays the others' rows end to end as units of
// two 8-entry chunks (fp32 rows: 32 bytes of terms; fp16 rows: 64 bytes of terms
// and values) and goes over them 32 units at a time, U such groups in flight.
// Each term is tested against a byte filter of the query, which about 2.8 % of
// them pass, three quarters of those being hits.
//   fp32 rows: the candidates are queued, and a second pass takes the queue one
//   candidate per lane: it looks the term up in the query and reads the value of
//   a hit, so the value reads of 32 entries are in flight together and chunks
//   without hits read no values.
//   fp16 rows: the values came with the terms, so each lane adds its own unit's
//   hits (queued and looked up as above: 16.2 ms where this takes 14.6; fp32 rows
//   this way, a value read behind the other: 65.6 ms where the queue takes 63.5).
// The products of a chunk are added in entry order, a document's chunk partials
// in chunk order, so a score is deterministic and independent of the launch shape.
//
// What bounds it: issue slots and shared-memory probes, then latency -- not DRAM.
// With every thread of the CTA on the wave's chunks, eight exact lookups per chunk
// and 7 barriers per wave, 32 chunks took 259 warp instructions and 69 shared-
// memory wavefronts, an L1 pipe at 77 %; a filter byte costs 3 instructions where
// a bit of the query's bitmap and the predicated lookup cost 20.  1M documents,
// 10k queries: cut 10, wave 8: 70.0 to 63.5 ms; cut 30 with the graph, wave 4: 149.5
// to 137.8 ms.  300k documents, fp16 rows: 14.9 to 14.6 ms.  100k documents, every
// block visited: 2.94 to 1.93 ms.  A filter of 4096 bytes (4.6 candidates per
// document instead of 3.6): 67.6 ms; of 16,384 bytes (3 CTAs per SM): 65.9 ms.
// Prefetching the rows into L2 no longer pays (64.3 ms) and is gone here.
template <int NT, bool FP16, bool SMALL, class Src>
__device__ __forceinline__ void eval_wave_flat(const SearchArgs &a, Smem &s, Shared &sh, uint32_t n, const Src &src,
                                               int knn_stage) {
  constexpr int U = FP16 || SMALL ? 1 : 2, NW = NT / 32;
  constexpr uint32_t kUnit = FP16 ? 2u * kUnitBytes : kUnitBytes;  // bytes of two chunks: their terms (fp16 rows: and values)
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, below = (1u << lane) - 1u;
  const bool full = sh.count == a.k;
  const float th = full ? s.tk_s()[a.k - 1] : -INFINITY;
  const uint32_t thid = full ? s.tk_id()[a.k - 1] : 0u;
  uint32_t *ncand = &sh.ncand[s.turn];
  auto offer = [&](float p, uint32_t d, uint32_t i) {
    if (!full || better(p, d, th, thid)) {
      const uint32_t pos = atomicAdd(ncand, 1u);
      s.cand_s()[pos] = p;
      s.cand_id()[pos] = d;
      s.cand_i()[pos] = (uint16_t)i;
    }
  };
  WarpDocs &wd = s.wdocs()[warp];
  // a warp's queue holds the candidates of 24 units at least, or the partials of 192 units (fp16 rows)
  constexpr uint32_t kQueue = kWarpQueueBytes / 4, kSums = kWarpQueueBytes / 8;
  uint32_t *queue = reinterpret_cast<uint32_t *>(s.wqueue() + warp * kWarpQueueBytes);
  float2 *sums = reinterpret_cast<float2 *>(queue);
  const uint8_t *qf = s.qfilt();
  const uint32_t per = (n + NW - 1) / NW, rounds = (per + 31u) / 32u, dpw = (per + rounds - 1) / rounds;
  const bool crowded = sh.crowded != 0u;
  const uint32_t mine = min(n, (warp + 1) * per);  // the warp's members: warp * per .. mine
  for (uint32_t r0 = warp * per; r0 < mine; r0 += dpw) {
    const uint32_t i = r0 + lane;
    uint32_t d = SEISMIC_NONE_ID, nch = 0;
    unsigned long long row = 0ull;
    if (lane < dpw && i < mine) {
      src.fetch(i, d, row);
      bool fresh = false;
      if (d != SEISMIC_NONE_ID) {
        if (s.seen) {
          const uint32_t bit = 1u << (d & 31);
          fresh = !(atomicOr(s.seen + (d >> 5), bit) & bit);
        } else {
          fresh = seen_insert(s.hash(), a.HS - 1u, d, crowded, &sh.hash_full);
        }
        if (fresh) {
          nch = (uint32_t)(row >> 32);
          if (a.stats) {
            atomicAdd(&sh.st[knn_stage ? SEISMIC_ST_KNN_DOCS : SEISMIC_ST_DOCS], 1ull);
            atomicAdd(&sh.st[knn_stage ? SEISMIC_ST_KNN_NNZ : SEISMIC_ST_DOC_NNZ], (unsigned long long)a.fwd_nnz[d]);
          }
          if (!nch) offer(0.0f, d, i);  // an empty row
        }
      }
      s.fresh()[i] = fresh ? 1 : 0;
      if (!s.seen && fresh) atomicAdd(&sh.hash_n, 1u);
    }
    // rows beyond the queue's 11-bit positions go one at a time
    uint32_t longs = __ballot_sync(0xffffffffu, nch > kShortChunks);
    while (longs) {
      const int l = __ffs(longs) - 1;
      longs &= longs - 1u;
      const unsigned long long r = __shfl_sync(0xffffffffu, row, l);
      const float p = warp_row<FP16>(a, s, r, lane);
      if ((int)lane == l) offer(p, d, i);
    }
    const uint32_t nu = nch > kShortChunks ? 0u : (nch + 1u) / 2u;
    uint32_t end = nu;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, end, 31);
    if (total == 0) continue;  // uniform over the warp
    const uint32_t kept = __ballot_sync(0xffffffffu, nu != 0u), nd = __popc(kept);
    if (nu) {
      const uint32_t x = __popc(kept & below), p0 = end - nu;
      const unsigned long long rec = reinterpret_cast<unsigned long long>(row_base(a.fwd_data, row));
      wd.unit0[x] = rec - (unsigned long long)kUnit * p0;
      if (!FP16) wd.val[x] = rec + (unsigned long long)kUnitBytes * nu;
      wd.p0[x] = p0;
      wd.doc[x] = d;
      wd.nch[x] = (uint16_t)nch;
      wd.member[x] = (uint16_t)i;
    }
    __syncwarp();
    // from here on lane x stands for document x of the nd kept ones
    const uint32_t myp0 = lane < nd ? wd.p0[lane] : total;
    float p = 0.0f;
    uint32_t nq = 0, wbeg = 0;  // queue entries, and the first unit they may come from

    // Scores the queue's entries, which come from the units wbeg .. wend.
    auto flush = [&](uint32_t wend) {
      __syncwarp();
      for (uint32_t r = 0; !FP16 && r < nq;) {
        uint32_t cnt = min(32u, nq - r);
        const uint32_t ent = lane < cnt ? queue[r + lane] : 0u, key = ent >> 19;  // document, chunk
        const uint32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
        const bool first = lane == 0 || key != prev;
        uint32_t firsts = __ballot_sync(0xffffffffu, first && lane < cnt);
        if (r + cnt < nq && (queue[r + cnt] >> 19) == __shfl_sync(0xffffffffu, key, 31)) {
          cnt = 31u - __clz(firsts);  // the last chunk's entries go on: it waits for the next 32 (a chunk has at most 8)
          firsts &= (1u << cnt) - 1u;
        }
        const uint32_t t = ent & 0xFFFFu, w = s.qbits()[t >> 5], bit = 1u << (t & 31u);
        const uint32_t x = ent >> 27, pos = (ent >> 16) & 0x7FFu;
        // a row of an odd number of chunks ends in half a unit that is not its own
        const bool hit = lane < cnt && (w & bit) && pos < 8u * wd.nch[x];
        float q = 0.0f, v = 0.0f;
        if (hit) {
          q = s.qval()[s.qrank()[t >> 5] + __popc(w & (bit - 1u))];
          v = ldg_na_f32(wd.val[x] + 4u * pos);
        }
        const uint32_t hits = __ballot_sync(0xffffffffu, hit);
        float acc = hit ? fmaf(q, v, 0.0f) : 0.0f;
        // hits behind another one of their chunk: chained in entry order onto the chunk's first entry
        const uint32_t self = firsts & (below | (1u << lane)), run = self ? 31u - __clz(self) : 0u;
        const bool again = hit && (hits & below & (~0u << run));
        if (__any_sync(0xffffffffu, again)) {
          const uint32_t later = lane < 31u ? firsts & (~0u << (lane + 1u)) : 0u;
          const uint32_t len = (firsts >> lane) & 1u ? (later ? __ffs(later) - 1u : cnt) - lane : 0u;  // a first entry's chunk
          const uint32_t longest = __reduce_max_sync(0xffffffffu, len);
          for (uint32_t o = 1; o < longest; o++) {
            const float q2 = __shfl_down_sync(0xffffffffu, q, o), v2 = __shfl_down_sync(0xffffffffu, v, o);
            if (o < len && ((hits >> (lane + o)) & 1u)) acc = fmaf(q2, v2, acc);
          }
          if (len == 0) acc = 0.0f;
        }
        if (lane < cnt) queue[r + lane] = __float_as_uint(acc);
        r += cnt;
      }
      __syncwarp();
      const uint32_t from = myp0 < wbeg ? 0u : myp0 < wend ? wd.start[lane] : nq;
      uint32_t to = __shfl_down_sync(0xffffffffu, from, 1);
      if (lane == 31) to = nq;
      for (uint32_t e = from; e < to; e++) {
        if constexpr (FP16) {
          const float2 x = sums[e];
          p += x.x;
          p += x.y;
        } else {
          p += __uint_as_float(queue[e]);
        }
      }
      __syncwarp();
    };

#pragma unroll 1
    for (uint32_t j0 = 0; j0 < total; j0 += 32 * U) {
      uint4 t[U], t2[U], h[U], h2[U];  // the two chunks' terms, fp16 rows: and values
      uint32_t head[U], dx[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        // group of units gb .. gb + 31 (past the end: the last one again, and the last unit in lanes past the
        // end); its first unit's document, and a bit for each document that starts in it
        const uint32_t gb = min(j0 + 32u * u, (total - 1u) & ~31u), jj = min(gb + lane, total - 1u);
        const uint32_t x0 = __popc(__ballot_sync(0xffffffffu, myp0 <= gb)) - 1u;
        head[u] = __reduce_or_sync(0xffffffffu, lane < nd && (myp0 & ~31u) == gb ? 1u << (myp0 & 31u) : 0u);
        dx[u] = x0 + __popc(head[u] & ((2u << (jj & 31u)) - 2u));
        const unsigned long long tp = wd.unit0[dx[u]] + (unsigned long long)kUnit * jj;
        if (FP16) {  // an odd row's last unit reads 32 bytes behind the row; its candidates are dropped below
          ldg_na_v8(reinterpret_cast<const void *>(tp), t[u], h[u]);
          ldg_na_v8(reinterpret_cast<const void *>(tp + kUnitBytes), t2[u], h2[u]);
        } else {
          ldg_na_v8(reinterpret_cast<const void *>(tp), t[u], t2[u]);
        }
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        const uint32_t gb = j0 + 32u * u;
        if (gb >= total) break;
        uint32_t m = probe8(t[u], qf) | probe8(t2[u], qf) << 8;
        if (gb + lane >= total) m = 0u;
        if constexpr (FP16) {
          float s0 = 0.0f, s1 = 0.0f;
          bool some = false;
          if (m) {
            const uint32_t x = dx[u], pos0 = 16u * (gb + lane - wd.p0[x]);
            if (pos0 + 8u >= 8u * wd.nch[x]) m &= 0xFFu;  // a row of an odd number of chunks ends in half a unit
            while (m) {
              const uint32_t e = __ffs(m) - 1u;
              m &= m - 1u;
              const uint32_t tt = pick16(t[u], t2[u], e), w = s.qbits()[tt >> 5], bit = 1u << (tt & 31u);
              if (w & bit) {
                const float q = s.qval()[s.qrank()[tt >> 5] + __popc(w & (bit - 1u))];
                const float v = __half2float(__ushort_as_half((unsigned short)pick16(h[u], h2[u], e)));
                if (e < 8u) s0 = fmaf(q, v, s0); else s1 = fmaf(q, v, s1);
                some = true;
              }
            }
          }
          const uint32_t ball = __ballot_sync(0xffffffffu, some);
          if (nq + __popc(ball) > kSums) {
            flush(gb);
            nq = 0;
            wbeg = gb;
          }
          const uint32_t at = nq + __popc(ball & below);
          if ((head[u] >> lane) & 1u) wd.start[dx[u]] = (uint16_t)at;
          if (some) sums[at] = make_float2(s0, s1);
          nq += __popc(ball);
          continue;
        }
        const uint32_t c = __popc(m);
        uint32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += y;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
        if (nq + tot > kQueue) {
          flush(gb);
          nq = 0;
          wbeg = gb;
        }
        // a group with more candidates than the queue holds goes in two halves of 16 units
        const bool halves = tot > kQueue;
        uint32_t at = nq + inc - c, mid = 0;
        if (halves) {
          mid = __shfl_sync(0xffffffffu, inc, 15);
          if (lane >= 16) at -= mid;
          if (lane < 16) {
            if ((head[u] >> lane) & 1u) wd.start[dx[u]] = (uint16_t)at;
            push_candidates(queue + at, m, t[u], t2[u], dx[u], 16u * (gb + lane - wd.p0[dx[u]]));
          }
          nq = mid;
          flush(gb + 16u);
          nq = 0;
          wbeg = gb + 16u;
        }
        if (!halves || lane >= 16) {
          if ((head[u] >> lane) & 1u) wd.start[dx[u]] = (uint16_t)at;
          if (m) push_candidates(queue + at, m, t[u], t2[u], dx[u], 16u * (gb + lane - wd.p0[dx[u]]));
        }
        nq += halves ? tot - mid : tot;
      }
    }
    flush(total);
    if (lane < nd) offer(p, wd.doc[lane], wd.member[lane]);
    __syncwarp();
  }
  __syncthreads();
}

// Scores n documents of a source; returns the number of candidates (the same in every thread).
template <int G, int NT, bool SMALL, class Src>
__device__ __forceinline__ uint32_t score(const SearchArgs &a, Smem &s, Shared &sh, uint32_t n, const Src &src,
                                          int knn_stage) {
  if constexpr (G == 1) {
    if (a.fp16) eval_wave_flat<NT, true, SMALL>(a, s, sh, n, src, knn_stage);
    else eval_wave_flat<NT, false, SMALL>(a, s, sh, n, src, knn_stage);
  } else {
    eval_wave<G, NT>(a, s, sh, n, src, knn_stage);
  }
  const uint32_t m = sh.ncand[s.turn];
  s.turn ^= 1u;
  if (!s.seen && m == 0) {  // no merge follows
    if (threadIdx.x == 0) note_crowded(a, s, sh);
    __syncthreads();
  }
  return m;
}

// Takes a document of a wave back out of the seen set (its block turned out to be skipped).
__device__ __forceinline__ void unsee(const SearchArgs &a, const Smem &s, uint32_t d) {
  if (s.seen) {
    atomicAnd(s.seen + (d >> 5), ~(1u << (d & 31)));
    return;
  }
  uint32_t h = (d * 0x9E3779B1u) & (a.HS - 1u);
  for (int p = 0; p < 16; p++) {
    if (s.hash()[h] == d + 1u) {
      s.hash()[h] = 0xFFFFFFFFu;  // no document's key, and not free: the probes behind it still find theirs
      return;
    }
    h = (h + 1u) & (a.HS - 1u);
  }
}

template <int NT>
__device__ void bitonic_sort_u64(unsigned long long *keys, uint32_t P2) {
  const int tid = threadIdx.x;
  for (uint32_t k2 = 2; k2 <= P2; k2 <<= 1)
    for (uint32_t j = k2 >> 1; j > 0; j >>= 1) {
      for (uint32_t i = tid; i < P2; i += NT) {
        uint32_t ixj = i ^ j;
        if (ixj > i) {
          unsigned long long x = keys[i], y = keys[ixj];
          bool up = (i & k2) == 0;
          if ((x > y) == up) { keys[i] = y; keys[ixj] = x; }
        }
      }
      __syncthreads();
    }
}

// Lane groups: 5 CTAs of 256 threads per SM (48 registers).  Group 1: 4 CTAs (64
// registers, two groups of units in flight, 46 KB of shared memory each).  SMALL:
// 5 CTAs (48 registers, one group in flight), which took 69 ms where 4 take 64 (1M documents,
// 10k queries, cut 10), but win in small collections, where most of a query is the
// latency of its lists' block scores and first waves (search_fit).
template <int G, int NW, bool SMALL>
__global__ void __launch_bounds__(NW * 32, (G == 1 && !SMALL ? 1024 : 1280) / (NW * 32))
    k_search(const __grid_constant__ SearchArgs a) {
  constexpr int NT = NW * 32;
  __shared__ Shared sh;
  Smem s{a, a.seen_bm ? a.seen_bm + (size_t)blockIdx.x * a.seen_words
                      : a.seen_words ? reinterpret_cast<uint32_t *>(g_sm + a.off_hash) : nullptr, 0u};
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  bool first = true;

  for (;;) {
    if (tid == 0) {
      if (a.persistent) {
        const uint32_t slot = atomicAdd(a.queue, 1u);
        sh.q = (a.perm && slot < a.nq) ? a.perm[slot] : slot;
      }
      else sh.q = first ? blockIdx.x : a.nq;
    }
    first = false;
    __syncthreads();
    const uint32_t q = sh.q;
    if (q >= a.nq) break;

    // ---------------------------------------------------------- H0: ingest
    const uint64_t qb = a.q_indptr[q], qe = a.q_indptr[q + 1];
    const uint32_t nnz = (uint32_t)(qe - qb);
    for (uint32_t i = tid; i < a.W; i += NT) s.qbits()[i] = 0u;
    if (G == 1)
      for (uint32_t i = tid; i < kFilter / 4; i += NT) reinterpret_cast<uint32_t *>(s.qfilt())[i] = 0u;
    if (s.seen) {  // seen_words is a multiple of 4 and the slot is 16-byte aligned
      uint4 *z = reinterpret_cast<uint4 *>(s.seen);
      for (uint32_t i = tid; i < a.seen_words / 4; i += NT) z[i] = make_uint4(0u, 0u, 0u, 0u);
    } else {
      for (uint32_t i = tid; i < a.HS; i += NT) s.hash()[i] = 0u;
    }
    if (tid < SEISMIC_STATS_N) sh.st[tid] = tid == SEISMIC_ST_T_START && a.stats ? globaltimer_ns() : 0ull;
    if (tid == 0) {
      sh.count = 0; sh.ncand[0] = 0; sh.ncand[1] = 0; sh.nvalid = 0; sh.hash_full = 0; sh.hash_n = 0; sh.crowded = 0; sh.bad = 0;
      sh.cut = a.cut;
      sh.hf = a.hf;
      if (a.q_cut) {  // learned per-query parameters (already validated by their producer)
        sh.cut = a.q_cut[q];
        sh.hf = a.q_hf[q];
      }
    }
    __syncthreads();
    for (uint32_t i = tid; i < nnz; i += NT) {
      const float v = a.q_vals[qb + i];
      if (v != 0.0f) {
        const uint32_t t = a.q_terms[qb + i];
        if (t < a.dim) atomicOr(&s.qbits()[t >> 5], 1u << (t & 31));
        else sh.bad = 1u;
      }
    }
    __syncthreads();
    const uint32_t nzq = block_rank_scan<NT>(s.qbits(), s.qrank(), a.W, sh.wtmp);
    if (nzq > a.QN || sh.bad) {  // more nonzeros than the launch was sized for, or a bad term
      if (tid == 0) atomicOr(a.queue + 1, 1u);
      for (uint32_t i = tid; i < a.k; i += NT) {
        a.ids[(size_t)q * a.k + i] = SEISMIC_NONE_ID;
        a.scores[(size_t)q * a.k + i] = -INFINITY;
      }
      __syncthreads();
      if (!a.persistent) break;
      continue;
    }
    for (uint32_t i = tid; i < nnz; i += NT) {
      const float v = a.q_vals[qb + i];
      if (v != 0.0f) {
        const uint32_t t = a.q_terms[qb + i];
        const uint32_t w = s.qbits()[t >> 5];
        const uint32_t pos = s.qrank()[t >> 5] + __popc(w & ((1u << (t & 31)) - 1u));
        s.qval()[pos] = v;
        s.qterm()[pos] = (uint16_t)t;
        if (G == 1) s.qfilt()[t & (kFilter - 1u)] = 1;
      }
    }
    __syncthreads();
    // ---------------------------------------------------------- H1: list terms
    if (a.seed) {
      if (tid == 0) sh.ncut = 0;  // graph refinement: no lists
    } else if (a.alpha_q > 0.0f) {
      for (uint32_t i = tid; i < nzq; i += NT) {
        const float av = fabsf(s.qval()[i]);
        const uint32_t t = s.qterm()[i];
        uint32_t r = 0;
        for (uint32_t j = 0; j < nzq; j++) {
          const float aj = fabsf(s.qval()[j]);
          r += (aj > av || (aj == av && s.qterm()[j] < t)) ? 1u : 0u;
        }
        s.aq()[r] = av;
        s.cutT()[r] = (uint16_t)t;
      }
      __syncthreads();
      if (tid == 0) {  // alpha_q-MSS: fp64 prefix mass in sketch order
        double tot = 0.0;
        for (uint32_t i = 0; i < nzq; i++) tot += (double)s.aq()[i];
        const double target = (double)a.alpha_q * tot;
        double c = 0.0;
        uint32_t keep = nzq;
        for (uint32_t i = 0; i < nzq; i++) {
          c += (double)s.aq()[i];
          if (c >= target) { keep = i + 1; break; }
        }
        sh.ncut = keep;
      }
    } else {
      const uint32_t cut = sh.cut;
      for (uint32_t i = tid; i < nzq; i += NT) {
        const float v = s.qval()[i];
        const uint32_t t = s.qterm()[i];
        uint32_t r = 0;
        for (uint32_t j = 0; j < nzq; j++) {
          const float vj = s.qval()[j];
          r += (vj > v || (vj == v && s.qterm()[j] < t)) ? 1u : 0u;
        }
        if (r < cut) s.cutT()[r] = (uint16_t)t;
      }
      if (tid == 0) sh.ncut = min(cut, nzq);
    }
    __syncthreads();
    const uint32_t ncut = sh.ncut;
    const float hf = sh.hf;
    if (a.stats && tid == 0) sh.st[SEISMIC_ST_QUERY_NNZ] = nnz;

    // ---------------------------------------------------------- lists
    for (uint32_t li = 0; li < ncut; li++) {
      const uint32_t t = s.cutT()[li];
      const uint32_t g0 = a.blk_ptr[t], nb = a.blk_ptr[t + 1] - g0;
      if (a.stats && tid == 0) sh.st[SEISMIC_ST_LISTS]++;
      if (nb == 0) continue;
      if (a.exhaustive) {
        const uint32_t d0 = a.bdoc_ptr[g0], d1 = a.bdoc_ptr[g0 + nb];
        if (a.stats && tid == 0) {
          sh.st[SEISMIC_ST_BLOCKS_EVALUATED] += nb;
          sh.st[SEISMIC_ST_BLOCK_DOCS] += d1 - d0;
        }
        for (uint32_t c0 = d0; c0 < d1; c0 += a.CAND) {
          const ListSrc src{nullptr, nullptr, 0u, c0, a.bdoc, a.bdoc_row};
          const uint32_t m = score<G, NT, SMALL>(a, s, sh, min(a.CAND, d1 - c0), src, 0);
          if (m) merge_commit<NT>(a, s, sh, merge_rank<NT>(a, s, sh, m, false, 0, 0), true);
        }
        continue;
      }
      // ---- H2: summary scores of every block of the list
      {
        uint32_t words = 0;
        for (uint32_t i = tid; i < nzq; i += NT)
          words += summary_column(a.sbm, a.scptr, a.W, t, s.qterm()[i], s.clo() + i, s.chi() + i);
        if (a.stats && words) atomicAdd(&sh.st[SEISMIC_ST_DIR_LOOKUPS], (unsigned long long)words);
      }
      for (uint32_t i = tid; i < a.NP * a.BMAX; i += NT) s.part()[i] = 0.0f;
      for (uint32_t b = tid; b <= nb; b += NT) s.bptr()[b] = __ldg(a.bdoc_ptr + g0 + b);  // block member ranges
      __syncthreads();
      if ((uint32_t)warp < a.NP) {
        float *pw = s.part() + warp * a.BMAX;
        const float *bm = a.blk_m + g0;
        const float *bs = a.blk_size + g0;
        uint32_t ent = 0;
        for (uint32_t i = warp; i < nzq; i += a.NP) {
          const uint32_t lo = s.clo()[i], hi = s.chi()[i];
          const float qv = s.qval()[i];
          ent += hi - lo;
          for (uint32_t e = lo + lane; e < hi; e += 32) {
            const uint32_t b = __ldg(a.scol_blk + e);
            float sv;
            if (a.quant) sv = fmaf((float)__ldg(a.scol_code + e), __ldg(bs + b), __ldg(bm + b));
            else sv = __ldg(a.scol_val + e);
            pw[b] = fmaf(qv, sv, pw[b]);
          }
          __syncwarp();
        }
        if (a.stats && lane == 0) atomicAdd(&sh.st[SEISMIC_ST_SUMMARY_ENTRIES], (unsigned long long)ent);
      }
      __syncthreads();
      uint32_t P2 = 1;
      while (P2 < nb) P2 <<= 1;
      for (uint32_t b = tid; b < P2; b += NT) {
        if (b < nb) {
          float r = 0.0f;
          for (uint32_t w = 0; w < a.NP; w++) r += s.part()[w * a.BMAX + b];
          s.keys()[b] = ((unsigned long long)(~f2ord(r)) << 32) | b;
        } else {
          s.keys()[b] = ~0ull;
        }
      }
      if (a.stats && tid == 0) sh.st[SEISMIC_ST_BLOCKS_SCORED] += nb;
      __syncthreads();
      // ---- H3: order blocks by (r desc, block asc)
      bitonic_sort_u64<NT>(s.keys(), P2);
      // ---- H4/H5/H6: visit blocks in order.  A wave is the next W blocks that
      // pass the test against theta (fewer past kCand documents; a larger block
      // goes alone, in pieces).  With a full top-k, group 1 scores as many whole waves at
      // once as fit CAND documents, as if theta stayed; when it rose so far that a
      // later wave would have tested otherwise, the waves are merged one by one and
      // what lies behind the first skip is undone.  So small waves cost a
      // barrier and a round of memory latency per CAND documents, not per wave
      // (300k documents, 2000 queries, wave 1: 21.1 ms; here 11.6).  While the top-k
      // fills theta does not stay: waves scored together then were mostly undone
      // (one query, 20k documents, lists of 500: 0.207 ms; here 0.150).
      const uint32_t W = min(a.wave, kMaxWave);
      const unsigned long long *keys = s.keys();
      auto bscore = [&](uint32_t i) { return ord2f(~(uint32_t)(keys[i] >> 32)); };
      auto limit = [&](float theta) { return a.hf_mode == 0 ? hf * theta : theta / hf; };
      // the wave from block p on: its end, and its documents in nd
      auto wave_end = [&](uint32_t p, uint32_t last, bool full, float thr, uint32_t &nd) {
        uint32_t e = p;
        nd = 0;
        while (e < last && e - p < W) {
          const uint32_t b = (uint32_t)(keys[e] & 0xFFFFFFFFu), bn = s.bptr()[b + 1] - s.bptr()[b];
          if (e > p && ((full && bscore(e) < thr) || nd + bn > kCand)) break;
          nd += bn;
          e++;
        }
        return e;
      };
      uint32_t bi = 0;
      while (bi < nb) {
        // skip test at the head of the wave (uniform: shared state after a barrier)
        const bool fullk = sh.count == a.k;
        const float thr = fullk ? limit(s.tk_s()[a.k - 1]) : -INFINITY;
        if (fullk && bscore(bi) < thr) {
          if (a.stats && tid == 0) sh.st[SEISMIC_ST_BLOCKS_SKIPPED] += nb - bi;
          break;
        }
        uint32_t ndocs = 0;
        const uint32_t first_end = wave_end(bi, nb, fullk, thr, ndocs);
        uint32_t be = first_end;
        while (G == 1 && fullk && be < nb && bscore(be) >= thr) {
          uint32_t nd;
          const uint32_t e = wave_end(be, nb, fullk, thr, nd);
          if (ndocs + nd > a.CAND || e - bi > kMaxWave) break;
          ndocs += nd;
          be = e;
        }
        if (a.prefetch && tid < (G == 1 ? max(W, 8u) : W) && be + tid < nb) {  // member lists of the next blocks
          const uint32_t b = (uint32_t)(keys[be + tid] & 0xFFFFFFFFu);
          const uint32_t e0 = s.bptr()[b], e1 = s.bptr()[b + 1];
          prefetch_l2(a.bdoc + e0, 4 * (e1 - e0));
          prefetch_l2(a.bdoc_row + e0, 8 * (e1 - e0));
        }
        uint32_t done = be, taken = ndocs;  // blocks up to here, and their documents, count
        for (uint32_t c0 = 0; c0 < ndocs; c0 += a.CAND) {  // one round, unless a single block is larger
          // (lane groups: one block's members lie side by side, no walk over the blocks' sizes)
          const bool single = G != 1 && be - bi == 1;
          const ListSrc src{keys + bi, s.bptr(), single ? 0u : be - bi,
                            single ? s.bptr()[(uint32_t)(keys[bi] & 0xFFFFFFFFu)] + c0 : c0, a.bdoc, a.bdoc_row};
          const uint32_t m = score<G, NT, SMALL>(a, s, sh, min(a.CAND, ndocs - c0), src, 0);
          if (m == 0) continue;
          const uint32_t nc = merge_rank<NT>(a, s, sh, m, false, 0, 0);
          if (G != 1 || be == first_end || nc < a.k || bscore(be - 1) >= limit(s.tmp_s()[a.k - 1])) {
            merge_commit<NT>(a, s, sh, nc, true);
            continue;
          }
          __syncthreads();  // everybody has read tmp
          if (tid == 0) sh.nvalid = 0;
          __syncthreads();
          done = bi;
          taken = 0;
          while (done < be) {
            const bool fk = sh.count == a.k;
            const float th = fk ? limit(s.tk_s()[a.k - 1]) : -INFINITY;
            if (fk && bscore(done) < th) break;
            uint32_t nd;
            const uint32_t e = wave_end(done, be, fk, th, nd);
            merge_commit<NT>(a, s, sh, merge_rank<NT>(a, s, sh, m, true, taken, taken + nd), false);
            taken += nd;
            done = e;
          }
          for (uint32_t i = taken + tid; i < ndocs; i += NT)
            if (s.fresh()[i]) {
              uint32_t d;
              unsigned long long row;
              src.fetch(i, d, row);
              unsee(a, s, d);
              if (a.stats) {
                atomicAdd(&sh.st[SEISMIC_ST_DOCS], ~0ull);
                atomicAdd(&sh.st[SEISMIC_ST_DOC_NNZ], 0ull - (unsigned long long)a.fwd_nnz[d]);
              }
            }
          if (tid == 0) sh.ncand[s.turn ^ 1u] = 0;
          __syncthreads();
        }
        if (a.stats && tid == 0) {
          sh.st[SEISMIC_ST_BLOCKS_EVALUATED] += done - bi;
          sh.st[SEISMIC_ST_BLOCK_DOCS] += taken;
        }
        bi = done;
      }
      __syncthreads();
    }

    // graph refinement starts the heap from the document and its neighbours; then
    // ---------------------------------------------------------- H7: kappa-NN expansion
    for (int stage = a.seed ? 0 : 1; stage < 2; stage++) {
      uint32_t total = 1 + a.kappa;
      if (stage == 1) {
        const uint32_t ns = sh.count;
        if (!(a.use_knn && a.kappa > 0 && ns > 0)) break;
        for (uint32_t i = tid; i < ns; i += NT) s.clo()[i] = s.tk_id()[i];  // S, fixed before expanding
        __syncthreads();
        total = ns * a.kappa;
      }
      for (uint32_t c0 = 0; c0 < total; c0 += a.CAND) {
        const NeighbourSrc src{stage ? s.clo() : nullptr, a.knn, a.fwd_row, stage ? 0u : a.seed[q], a.kappa, a.knn_bits, c0};
        const uint32_t m = score<G, NT, SMALL>(a, s, sh, min(a.CAND, total - c0), src, stage);
        if (m) merge_commit<NT>(a, s, sh, merge_rank<NT>(a, s, sh, m, false, 0, 0), true);
      }
    }

    // ---------------------------------------------------------- output
    for (uint32_t i = tid; i < a.k; i += NT) {
      const bool ok = i < sh.count;
      a.ids[(size_t)q * a.k + i] = ok ? s.tk_id()[i] : SEISMIC_NONE_ID;
      a.scores[(size_t)q * a.k + i] = ok ? s.tk_s()[i] : -INFINITY;
    }
    if (a.stats && tid == SEISMIC_ST_T_END) sh.st[tid] = globaltimer_ns();
    if (a.stats && tid < SEISMIC_STATS_N) a.stats[(size_t)q * SEISMIC_STATS_N + tid] = sh.st[tid];
    __syncthreads();
    if (!a.persistent) break;
  }
}

template <int G, int NW, bool SMALL = false>
int launch_t(const SearchArgs &a, size_t smem, uint32_t grid, cudaStream_t st) {
  static std::atomic<uint64_t> configured{0};
  int rc = set_smem_limit_once(configured, (const void *)k_search<G, NW, SMALL>, (int)kMaxSmem);
  if (rc) return rc;
  k_search<G, NW, SMALL><<<grid, NW * 32, smem, st>>>(a);
  SZ_CUDA(cudaGetLastError());
  return SEISMIC_OK;
}

template <int G, int NW, bool SMALL = false>
int occupancy_t(size_t smem, int *blocks) {
  SZ_CUDA(cudaFuncSetAttribute(k_search<G, NW, SMALL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem));
  SZ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, k_search<G, NW, SMALL>, NW * 32, smem));
  return SEISMIC_OK;
}

}  // namespace

static inline uint32_t al16(uint32_t x) { return (x + 15u) & ~15u; }

size_t search_layout(SearchArgs &a, uint32_t nw) {
  uint32_t o = 0;
  auto take = [&](uint32_t bytes) {
    uint32_t r = o;
    o = al16(o + bytes);
    return r;
  };
  a.off_qbits = take(a.W * 4);
  a.off_qrank = take(a.W * 2);
  a.off_qval = take(a.QN * 4);
  a.off_qterm = take(a.QN * 2);
  a.off_cut = take(a.QN * 2);
  a.off_aq = take(a.alpha_q > 0.0f ? a.QN * 4 : 4);
  // Block-score partials and, while documents are scored (the partials are dead then), the warps' candidate
  // queues.  One behind the other where the queues are the larger, they left room for three CTAs per SM, not four:
  // 4000 documents as queries, 100,000 documents, 300 blocks a list: 15.5 ms, here 13.1.
  const uint32_t partials = a.exhaustive ? 4u : a.NP * a.BMAX * 4u, queues = a.flat ? nw * kWarpQueueBytes : 0u;
  a.off_part = a.off_wqueue = take(std::max(partials, queues));
  a.off_keys = take(a.exhaustive ? 8 : a.BPOW2 * 8);
  const uint32_t nclo = std::max(a.QN, a.k);  // clo also holds S during the expansion
  a.off_clo = take(nclo * 4);
  a.off_chi = take(a.QN * 4);
  a.off_hash = take(a.HS * 4);
  a.off_tk_s = take(a.k * 4);
  a.off_tk_id = take(a.k * 4);
  a.off_tmp_s = take(a.k * 4);
  a.off_tmp_id = take(a.k * 4);
  a.off_cand_s = take(a.CAND * 4);
  a.off_cand_id = take(a.CAND * 4);
  a.off_cand_ok = take(a.CAND);
  a.off_cand_i = take(a.flat ? a.CAND * 2 : 0);
  a.off_fresh = take(a.flat ? a.CAND : 0);
  a.off_bptr = take(a.exhaustive ? 4 : (a.BMAX + 1) * 4);
  a.off_qfilt = take(a.flat ? kFilter : 0);
  a.off_wdocs = take(a.flat ? nw * kWarpDocsBytes : 0);
  return o;
}

// What a call is refused by (200 KB): the query, the block scores of a list, the seen set, the top-k and a wave's
// candidates in a CTA of nw warps, and for group 1 what its documents' rows were once laid out in (12 bytes a
// document, and one a block score or five for each of 2048).  A property of the call, not of the arrays above, so that a change of these
// refuses no call that was accepted.
static size_t search_budget(const SearchArgs &a, uint32_t nw) {
  const uint32_t scores = a.exhaustive ? 0u : nw * a.BMAX;  // block-score partials
  size_t b = 0;
  for (size_t bytes : {a.W * 4u, a.W * 2u, a.QN * 4u, a.QN * 2u, a.QN * 2u, a.alpha_q > 0.0f ? a.QN * 4u : 4u,
                       std::max(scores * 4u, 4u), a.exhaustive ? 8u : a.BPOW2 * 8u, std::max(a.QN, a.k) * 4u, a.QN * 4u,
                       a.HS * 4u, a.k * 4u, a.k * 4u, a.k * 4u, a.k * 4u, kCand * 9u,
                       a.exhaustive ? 4u : (a.BMAX + 1u) * 4u})
    b += al16((uint32_t)bytes);
  if (a.flat) b += kCand * 12u + 16u + std::max(2048u, scores) + (scores < 2048u ? 8192u : 0u);
  return b;
}

// A query alone on its SM is bound by latency: the more warps share a wave's
// documents, the fewer loads follow one another.  One CTA of 32 warps per SM up
// to as many queries as SMs, 16 warps up to four times that (two CTAs per SM, in
// up to two rounds), else 8.  1M documents, cut 10: one query 2.6 ms with 8 warps,
// 1.5 with 32; 305 queries 4.95 with 8, 3.35 with 16; 450: 6.2, 5.2; 608: 6.6, 6.2; 700: 6.9,
// 7.6.  The block scores are added up as by 8 warps in each (SearchArgs::NP), so the results do
// not depend on the choice.
//
// Beside queries of other calls (a server's batches) 16 warps hold up to eight queries per SM: new batches find the
// GPU partly idle, and a batch that ends sooner frees its slots sooner.  8.8M documents, cut 30, graph, 40k requests
// a second, p50 / p99: 22.9 / 50.7 ms, with the line at four 37.2 / 64.2, with 16 warps at any load 23.5 / 44.2; all
// requests at once 46.5k, 46.3k and 46.7k q/s, and over 1M documents 259k with the line at four, 248k with 16 warps.
static uint32_t search_warps(uint32_t nq, uint32_t beside, uint32_t sms) {
  const uint32_t n = nq + beside;
  return n > (beside ? 8u : 4u) * sms ? 8u : n > sms ? 16u : 32u;
}

size_t search_fit(SearchArgs &a, uint32_t &group, uint32_t asked, uint32_t beside, uint32_t sms, uint32_t bitmap_words,
                  uint32_t &nw) {
  nw = asked ? asked : 8u;
  a.NP = nw;
  a.flat = group == 1 ? 1u : 0u;
  a.CAND = kCand;
  a.budget = (uint32_t)std::min<size_t>(search_budget(a, nw), 0xFFFFFFFFu);
  if (a.budget > 200u * 1024u) return 0;
  size_t smem = 0;
  if (a.persistent) a.HS = 16;  // the seen set is a bitmap in global memory
  if (!a.flat) return search_layout(a, nw);
  const uint32_t slots = a.HS, wide = asked ? asked : search_warps(a.nq, beside, sms);
  for (int form = bitmap_words ? 0 : 1; form < 2; form++) {
    a.seen_words = form == 0 ? bitmap_words : 0u;
    a.HS = form == 0 ? bitmap_words : slots;
    for (uint32_t w : {wide, nw}) {
      // wide CTAs score more documents at once: one query 1.49 ms instead of 1.82, but batches of 8-warp
      // CTAs 65.9 instead of 63.7
      a.CAND = w > nw ? kWideCand : kCand;
      if ((smem = search_layout(a, w)) <= kMaxSmem) {
        // 8000 queries of 10..150 entries with 4 and with 5 CTAs per SM: 2000 documents 1.91 and 1.71 ms, 20,000 4.44 and
        // 4.02, 50,000 (lists of 1000) 8.02 and 7.41; 1000 queries of 20,000 0.850 and 0.847.  Batches that
        // 4 CTAs hold in two rounds gain nothing
        a.small = w == 8 && smem <= kSmallSmem && a.n_docs <= kSmallDocs && a.nq + beside > 8 * sms;
        nw = w;
        return smem;
      }
    }
  }
  // very long queries: the lane groups need less besides the query
  group = 8;
  a.flat = 0;
  a.CAND = kCand;
  return search_layout(a, nw);
}

int launch_search(const SearchArgs &a, uint32_t group, uint32_t nw, size_t smem, uint32_t grid, cudaStream_t st) {
#define SZ_CASE(G_, NW_) \
  if (group == G_ && nw == NW_) return launch_t<G_, NW_>(a, smem, grid, st);
  if (a.small && group == 1 && nw == 8) return launch_t<1, 8, true>(a, smem, grid, st);
  SZ_CASE(1, 4) SZ_CASE(1, 8) SZ_CASE(1, 16) SZ_CASE(1, 32)
  SZ_CASE(8, 4) SZ_CASE(8, 8) SZ_CASE(8, 16)
  SZ_CASE(16, 4) SZ_CASE(16, 8) SZ_CASE(16, 16)
  SZ_CASE(32, 4) SZ_CASE(32, 8) SZ_CASE(32, 16)
#undef SZ_CASE
  return fail(SEISMIC_EINVAL, "group must be 1/8/16/32 and cta_warps 4/8/16");
}

int search_occupancy(const SearchArgs &a, uint32_t group, uint32_t nw, size_t smem, int *blocks) {
#define SZ_CASE(G_, NW_) \
  if (group == G_ && nw == NW_) return occupancy_t<G_, NW_>(smem, blocks);
  if (a.small && group == 1 && nw == 8) return occupancy_t<1, 8, true>(smem, blocks);
  SZ_CASE(1, 4) SZ_CASE(1, 8) SZ_CASE(1, 16) SZ_CASE(1, 32)
  SZ_CASE(8, 4) SZ_CASE(8, 8) SZ_CASE(8, 16)
  SZ_CASE(16, 4) SZ_CASE(16, 8) SZ_CASE(16, 16)
  SZ_CASE(32, 4) SZ_CASE(32, 8) SZ_CASE(32, 16)
#undef SZ_CASE
  return fail(SEISMIC_EINVAL, "group must be 1/8/16/32 and cta_warps 4/8/16");
}

}  // namespace seismic
