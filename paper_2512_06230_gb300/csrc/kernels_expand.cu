// Child expansion, scoring and per-parent deduplication (arXiv 2512.06230,
// Section 3: two-stage sampling of H_up children per hypothesis, weight =
// parent weight x joint likelihood of the sampled deaths and associations,
// retention of unique children), and the regeneration of the retained
// children for the batched track update.
//
// Four kernels share one per-parent image in global memory:
//   stage     one CTA per parent builds the parent's tables (in shared memory
//             when they fit, then copied out; else in place): its gated pairs
//             re-indexed by detection row (slots ascending within a row), per
//             row integer thresholds of the categorical draw under "all slots
//             alive", a reference association (each row's most likely option)
//             with its exact score, and per slot the m-only part of the track
//             term for m_ref - 2 .. m_ref + 2 detections, and the exact score
//             change of each slot dying.  What only deviating children read
//             (innovations, covariances) stays in the pair and component
//             tables: the images of the 3-D N = 200 scene shrink by 28 %, and
//             the staging's reads go out together instead of each waiting for
//             the write before it (with the follow-up below, expansion of the
//             scene 577 -> 519 us per frame, gated 311 -> 266);
//   draw      one thread per child: Philox words for the slots that can die
//             (stage 1) and one per detection row (stage 2); the row's option
//             is the first whose threshold exceeds the 24-bit uniform (rows
//             with a dead candidate fall back to the FP32 normalised row of
//             C'_k); deaths and rows that leave the reference are listed in
//             shared memory; the child's log-weight is the reference score
//             plus its deviations' changes (finish_notes, in the warp
//             kernel's launch, for the few children that have any), or, when
//             a slot is met twice, the exact rescoring of every met slot
//             (stage 3), in fixed point;
//   warp      one warp per child, rows split over the lanes and per-slot sums
//             in shared memory: children whose lists overflow the draw
//             kernel's, every child when parents are too few to fill
//             the GPU with threads, and the regeneration of retained children
//             (association rows, track lists, updated-component requests);
//   mat_prep  the updated components of each retained parent's reference
//             association, requested once per parent.
// The duplicate test keys a child by the order-free sum of mix64 keys of its
// deviations and deaths.
#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "glmb_kernels.h"

namespace glmb {

// ---- per-parent image ----

struct Lay {
  int scal;
  int row, rowbl, seref, sqref, termref, hwref, deadd;
  int rowrk, rch, rowoff, rowfill, roww0, rowthr0;
  int comp, dthr, mref, refnew, dpc, dth;
  int cthr, ceidx, cw, cslot;
  int ninfref, dninf, srow;
  int total;
};

// Chunk of four detection rows with candidates, as the thread-per-child
// draw reads it: head = (chunk index, bit b set when row 4 cc + b has a
// candidate slot that can die, low and high words of the bloom of those
// slots over the four rows), then the four rows' reference intervals
// [lo, hi) of the 24-bit uniform u = word >> 8 (rows without candidates, or
// beyond the detections: [0, 2^24)), held as base = lo << 8 and
// span = ((hi - lo) << 8) - 1 (mod 2^32): u is in [lo, hi) exactly when
// word - base <= span, as unsigned 32-bit arithmetic (hi - lo >= 1).
struct RowChunk {
  uint4 head;
  uint4 base;
  uint4 span;
};

struct Bump {
  int off = 0;
  __host__ __device__ int take(long long bytes) {
    const int o = off;
    off += (int)((bytes + 15) & ~15LL);
    return o;
  }
};

struct Scal {
  long long ref_score;
  unsigned long long uid;
  double logw;
  int ninf_ref, nclut_ref, T, Town, K, ndpc, nrca, bad;
};

// T, K, M: the plan's slots, gated pairs and detection rows per parent.
// Per-slot arrays are indexed with the parent's own slot count as stride,
// per-pair arrays with K.
__host__ __device__ inline Lay make_lay(int dz, int T, int K, int M) {
  Lay L;
  Bump b;
  L.scal = b.take(sizeof(Scal));
  L.row = b.take(16LL * M);                 // packed row descriptors (uint4)
  L.rowbl = b.take(8LL * M);                // bit (slot mod 64) of each candidate slot
  L.seref = b.take(8LL * dz * T);           // reference sums of innovations (fixed point)
  L.sqref = b.take(8LL * T);                // reference sums of e^T R^-1 e
  L.termref = b.take(8LL * T);              // reference track terms
  L.hwref = b.take(8LL * T);                // reference detection-set keys
  // exact score change of a slot dying (deadd[t]) and of its infinite-term
  // count (dninf); a row's deviations are scored by the child that makes them
  L.deadd = b.take(8LL * T);
  L.rowrk = b.take(4LL * M);                // reference option's slot and pair
  L.rch = b.take(48LL * ((M + 3) / 4 + 1)); // chunks of 4 rows with candidates (RowChunk)
  L.rowoff = b.take(4LL * (M + 1));
  L.rowfill = b.take(4LL * (M + 1));
  L.roww0 = b.take(4LL * M);
  L.rowthr0 = b.take(4LL * M);              // clutter option's threshold
  L.comp = b.take(4LL * T);
  L.dthr = b.take(4LL * T);
  L.mref = b.take(4LL * T);
  L.refnew = b.take(4LL * T);
  L.dpc = b.take(4LL * (T / 4 + 2));        // chunks of 4 slots that can die
  L.dth = b.take(16LL * (T / 4 + 2));       // their slots' largest dying words (see the chunk lists)
  L.cthr = b.take(4LL * K);
  L.ceidx = b.take(4LL * K);                // the pair's place in the table (innovation, q, log C)
  L.cw = b.take(4LL * K);
  L.cslot = b.take(2LL * K);
  L.ninfref = b.take(T);
  L.dninf = b.take(T);
  L.srow = b.take(T);                       // slot can die and is a candidate of some row
  L.total = b.off;
  return L;
}

// The staging kernel's shared scratch beside the image: the next-parent
// word (16 B) and the scan's warp sums (32 B); then, when the image is
// built in global memory, the arrays the staging reads back many times:
// mode >= 1 the row offsets and fill cursors, mode 2 also the candidates'
// slots and pair indices and the per-slot reference counts, sums, terms
// and infinite-term counts (copied to the image at the end of the parent).
// Offsets from its base.
struct StageTail {
  int rowoff, rowfill, cslot, ceidx, mref, seref, sqref, hwref, termref, ninfref, dthr, total;
};
__host__ __device__ inline StageTail make_stage_tail(int dz, int T, int K, int M, int mode) {
  StageTail S{};
  Bump b;
  b.take(16);   // next-parent word
  b.take(32);   // the parent's sizes, counts and flags
  b.take(128);  // warp sums of the row-count scan
  if (mode >= 1) {
    S.rowoff = b.take(4LL * (M + 1));
    S.rowfill = b.take(4LL * (M + 1));
  }
  if (mode >= 2) {
    S.cslot = b.take(2LL * K);
    S.ceidx = b.take(4LL * K);
    S.mref = b.take(4LL * T);
    S.seref = b.take(8LL * dz * T);
    S.sqref = b.take(8LL * T);
    S.hwref = b.take(8LL * T);
    S.termref = b.take(8LL * T);
    S.ninfref = b.take(T);
    S.dthr = b.take(4LL * T);
  }
  S.total = b.off;
  return S;
}

int expand_image_bytes(int dz, int T, int K, int M) {
  return (make_lay(dz, T, K, M).total + 127) & ~127;
}

// per-warp work area of the warp kernel
struct WLay {
  int se, sq, hw, cnt, newval, tmask, dmask, dpre, nt, tlist, red, total;
};

__host__ __device__ inline WLay make_wlay(int dz, int mat, int T, int grp = 0) {
  WLay L;
  Bump b;
  const int W = (T + 31) / 32 + 1;
  L.se = b.take(8LL * dz * T);
  L.sq = b.take(8LL * T);
  L.hw = mat ? b.take(8LL * T) : 0;
  L.cnt = b.take(4LL * T);
  L.newval = mat ? b.take(4LL * T) : 0;
  L.tmask = b.take(4LL * W);
  L.dmask = b.take(4LL * W);
  L.dpre = b.take(4LL * W);
  L.nt = b.take(16);
  L.tlist = b.take(2LL * T);
  L.red = grp ? b.take(64) : 0;   // a multi-warp group's reductions
  L.total = b.off;
  return L;
}

int expand_warp_smem(int dz, int materialize, int T, int warps, int grp) {
  return warps * make_wlay(dz, materialize, T, grp).total;
}

template <typename T>
__device__ __forceinline__ T* at(unsigned char* base, int off) {
  return reinterpret_cast<T*>(base + off);
}
template <typename T>
__device__ __forceinline__ const T* at(const unsigned char* base, int off) {
  return reinterpret_cast<const T*>(base + off);
}

__device__ __forceinline__ uint32_t thr_of(float frac) {
  // smallest integer k0 with k0 >= frac * 2^24, clamped to [0, 2^24]
  if (!(frac > 0.f)) return 0u;
  if (frac >= 1.f) return kOne24;
  return (uint32_t)ceilf(frac * 16777216.f);
}

// A child of the warp path is handled by a group of gsz threads (one warp,
// or several consecutive warps of the CTA that share one work area and
// synchronise on named barrier gid + 1).
__device__ __forceinline__ void group_sync(int gsz, int gid) {
  if (gsz == 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(gid + 1), "r"(gsz) : "memory");
}

__device__ __forceinline__ void touch(uint32_t* tmask, uint16_t* tlist, int* nt, int t) {
  const uint32_t bit = 1u << (t & 31);
  const uint32_t old = atomicOr(&tmask[t >> 5], bit);
  if (!(old & bit)) tlist[atomicAdd(nt, 1)] = (uint16_t)t;
}

// H P H^T of component c
template <int DZ>
__device__ __forceinline__ void slot_HPH(const CompTable& ct, int dx, uint32_t c, float (&HPH)[DZ][DZ]) {
#pragma unroll
  for (int x = 0; x < DZ; ++x)
#pragma unroll
    for (int y = x; y < DZ; ++y) {
      const float v = ct.cov[(size_t)pidx(dx, x, y) * ct.cap + c];
      HPH[x][y] = v;
      HPH[y][x] = v;
    }
}

// The m-only parts of component c's alive term with m detections, from the
// frame's per-component table (built by the table kernel).
template <int DZ>
__device__ __forceinline__ SlotM<DZ> load_cslm(const float* slm, const int8_t* sln, int cap, int m, uint32_t c) {
  constexpr int NP = DZ * (DZ + 1) / 2;
  SlotM<DZ> s;
  const size_t base = (size_t)(m - 1) * (NP + 1);
#pragma unroll
  for (int k = 0; k < NP; ++k) s.Sinv[k] = slm[(base + k) * cap + c];
  s.c = slm[(base + NP) * cap + c];
  s.ninf = sln[(size_t)(m - 1) * cap + c];
  return s;
}

// Term of slot t alive with m detections, built from H P H^T (kept out of
// line: it is rare and needs many registers)
struct TermOut {
  long long term;
  int ninf;
};
template <int DZ>
struct SeVec {
  long long v[DZ];
};

template <int DZ>
__device__ __noinline__ TermOut slot_term_full(const Model& md, const CompTable& ct, uint32_t c, int m,
                                               const SeVec<DZ> se, long long sq) {
  // the sums come and the result goes by value, so a caller keeps them in
  // registers (an array passed by reference would live in local memory)
  float HPH[DZ][DZ];
  slot_HPH<DZ>(ct, md.dx, c, HPH);
  TermOut o;
  o.term = alive_term<DZ>(md, HPH, ct.logp[c], m, se.v, sq, o.ninf);
  return o;
}

// read-only view of a staged parent
struct View {
  const Scal* sc;
  const uint4* row;
  const unsigned long long* rowbl;
  const long long *seref, *sqref, *termref, *deadd;
  const unsigned long long* hwref;
  const RowChunk* rch;
  const uint4* dth;
  const uint32_t *rowrk, *rowthr0, *comp, *dthr, *refnew, *dpc, *cthr, *ceidx;
  const float *roww0, *cw;
  const PairTable* pt;    // the pairs, and the per-component m-only term parts (slm)
  const CompTable* ct;
  const int* mref;
  const uint16_t* cslot;
  const uint8_t* ninfref;
  const int8_t* dninf;
  const uint8_t* srow;
};

__device__ __forceinline__ View make_view(const unsigned char* b, const Lay& L, const PairTable& pt, const CompTable& ct) {
  View v;
  v.sc = at<Scal>(b, L.scal);
  v.row = at<uint4>(b, L.row);
  v.rowbl = at<unsigned long long>(b, L.rowbl);
  v.seref = at<long long>(b, L.seref);
  v.sqref = at<long long>(b, L.sqref);
  v.termref = at<long long>(b, L.termref);
  v.deadd = at<long long>(b, L.deadd);
  v.dninf = at<int8_t>(b, L.dninf);
  v.hwref = at<unsigned long long>(b, L.hwref);
  v.rowrk = at<uint32_t>(b, L.rowrk);
  v.rch = at<RowChunk>(b, L.rch);
  v.dth = at<uint4>(b, L.dth);
  v.srow = at<uint8_t>(b, L.srow);
  v.rowthr0 = at<uint32_t>(b, L.rowthr0);
  v.comp = at<uint32_t>(b, L.comp);
  v.dthr = at<uint32_t>(b, L.dthr);
  v.refnew = at<uint32_t>(b, L.refnew);
  v.dpc = at<uint32_t>(b, L.dpc);
  v.cthr = at<uint32_t>(b, L.cthr);
  v.roww0 = at<float>(b, L.roww0);
  v.ceidx = at<uint32_t>(b, L.ceidx);
  v.pt = &pt;
  v.ct = &ct;
  v.cw = at<float>(b, L.cw);
  v.mref = at<int>(b, L.mref);
  v.cslot = at<uint16_t>(b, L.cslot);
  v.ninfref = at<uint8_t>(b, L.ninfref);
  return v;
}

// A candidate pair's innovation and e^T R^-1 e (the factorised mode sums log C
// instead), in fixed point, from the table: few children need one, so the
// images do not repeat them.
template <int DZ>
__device__ __forceinline__ void pair_sums(const Model& md, const View& v, uint32_t pos, long long (&e)[DZ],
                                          long long& q) {
  const uint32_t j = v.ceidx[pos];
#pragma unroll
  for (int d = 0; d < DZ; ++d) e[d] = fx_of(v.pt->e[(size_t)d * v.pt->cap_pairs + j]);
  q = fx_of(md.score_mode == 1 ? v.pt->logC[j] : v.pt->q[j]);
}

// Term of slot t alive with m detections whose sums are (se, sq): the m-only
// parts from the per-component table when it holds (component, m), else
// built from H P H^T (the same function, so the same values).
template <int DZ>
__device__ __forceinline__ long long slot_term(const Model& md, const View& v, int t, int m,
                                               const long long (&se)[DZ], long long sq, int& ninf) {
  const uint32_t c = v.comp[t];
  if (md.score_mode == 1) return factor_term(md, v.ct->logp[c], m, sq, ninf);
  if (m >= 1 && m <= kSlmM && c < (uint32_t)v.pt->slm_cap)
    return term_from<DZ>(md, load_cslm<DZ>(v.pt->slm, v.pt->sln, v.pt->slm_cap, m, c), m, se, sq, ninf);
  SeVec<DZ> sv;
#pragma unroll
  for (int d = 0; d < DZ; ++d) sv.v[d] = se[d];
  const TermOut o = slot_term_full<DZ>(md, *v.ct, c, m, sv, sq);
  ninf = o.ninf;
  return o.term;
}

__device__ __forceinline__ bool bit_of(const uint32_t* m, int t) {
  return (m[t >> 5] >> (t & 31)) & 1u;
}

// insert (component, detection-set key) into the update table; returns the
// tagged hash slot to be resolved to a component index after the kernel
template <int DZ>
__device__ uint32_t upd_insert(const ExpandArgs& a, uint32_t comp, unsigned long long hw, int m,
                               const long long (&se)[DZ]) {
  unsigned long long key = mix64(hw + 0x9E3779B97F4A7C15ULL * ((unsigned long long)comp + 1ULL));
  if (key == 0ULL) key = 1ULL;
  uint32_t slot = (uint32_t)key & a.hmask;
  for (uint32_t probe = 0; probe <= a.hmask; ++probe) {
    // most requests repeat one already made (hypotheses share their
    // updates): a cached read finds it without an atomic on the shared
    // address.  Slots only go from empty to a key while requests are made,
    // so a stale read can only be empty, and then the atomic decides
    unsigned long long prev;
    asm volatile("ld.global.ca.u64 %0, [%1];" : "=l"(prev) : "l"(a.hkeys + slot) : "memory");
    if (prev == 0ULL) prev = atomicCAS(&a.hkeys[slot], 0ULL, key);
    else if (prev != key) {
      slot = (slot + 1u) & a.hmask;
      continue;
    }
    if (prev == 0ULL) {
      const uint32_t id = atomicAdd(a.upd_count, 1u);
      if (id < (uint32_t)a.cap_upd) {
        a.upd_src[id] = comp;
        a.upd_m[id] = (uint32_t)m;
#pragma unroll
        for (int d = 0; d < DZ; ++d) a.upd_se[(size_t)d * a.cap_upd + id] = se[d];
        a.hvals[slot] = id;
        a.upd_slot[id] = slot;
      } else {
        atomicOr(a.err, kErrUpdates);
        a.hvals[slot] = 0u;
      }
      return kNewTag | slot;
    }
    if (prev == key) return kNewTag | slot;
    slot = (slot + 1u) & a.hmask;
  }
  atomicOr(a.err, kErrHash);
  return kNewTag;
}

// ====================== stage: one CTA per parent ======================
// Detection rows with at most this many candidate slots are sorted and
// weighed in registers (nearly all rows: a detection gates to one track or
// a few).
constexpr int kRowReg = 4;
template <int N>
struct FVec {
  float v[N];
};
// Builds parent h's image at `sm` (shared memory, or the image itself).
// `tb`: the shared scratch beside the image (StageTail).  With the image in
// global memory (in_tail) the arrays it lists live there while the parent
// is staged, so that their atomics and read-backs stay on chip, and are
// copied to the image at the end.
template <int DZ>
__device__ void stage_parent(const ExpandArgs& a, const int h, const Lay& L, unsigned char* sm, unsigned char* tb,
                             int mode) {
  const StageTail TS = make_stage_tail(DZ, a.T_max, a.K_max, a.M_plan, mode);
  const bool in_tail = mode >= 2;
  const Model& md = a.md;
  const int M = a.fs->M;
  const int birth_base = a.fs->n_comp, nb = a.fs->nb;
  Scal& sc = *at<Scal>(sm, L.scal);
  uint4* s_row = at<uint4>(sm, L.row);
  unsigned long long* s_rowbl = at<unsigned long long>(sm, L.rowbl);
  long long* s_seref = in_tail ? at<long long>(tb, TS.seref) : at<long long>(sm, L.seref);
  long long* s_sqref = in_tail ? at<long long>(tb, TS.sqref) : at<long long>(sm, L.sqref);
  long long* s_termref = in_tail ? at<long long>(tb, TS.termref) : at<long long>(sm, L.termref);
  unsigned long long* s_hwref = in_tail ? at<unsigned long long>(tb, TS.hwref) : at<unsigned long long>(sm, L.hwref);
  uint32_t* s_rowrk = at<uint32_t>(sm, L.rowrk);
  RowChunk* s_rch = at<RowChunk>(sm, L.rch);
  uint8_t* s_srow = at<uint8_t>(sm, L.srow);
  uint32_t* s_rowthr0 = at<uint32_t>(sm, L.rowthr0);
  uint32_t* s_wsum = at<uint32_t>(tb, 16), *s_scan = at<uint32_t>(tb, 48);
  uint32_t* s_rowoff = mode >= 1 ? at<uint32_t>(tb, TS.rowoff) : at<uint32_t>(sm, L.rowoff);
  uint32_t* s_rowfill = mode >= 1 ? at<uint32_t>(tb, TS.rowfill) : at<uint32_t>(sm, L.rowfill);
  float* s_roww0 = at<float>(sm, L.roww0);
  uint32_t* s_comp = at<uint32_t>(sm, L.comp);
  // death thresholds: written to the image, read back on chip
  uint32_t* g_dthr = at<uint32_t>(sm, L.dthr);
  uint32_t* s_dthr = in_tail ? at<uint32_t>(tb, TS.dthr) : g_dthr;
  int* s_mref = in_tail ? at<int>(tb, TS.mref) : at<int>(sm, L.mref);
  uint32_t* s_dpc = at<uint32_t>(sm, L.dpc);
  uint4* s_dth = at<uint4>(sm, L.dth);
  uint32_t* s_cthr = at<uint32_t>(sm, L.cthr);
  uint32_t* s_ceidx = in_tail ? at<uint32_t>(tb, TS.ceidx) : at<uint32_t>(sm, L.ceidx);
  float* s_cw = at<float>(sm, L.cw);
  uint16_t* s_cslot = in_tail ? at<uint16_t>(tb, TS.cslot) : at<uint16_t>(sm, L.cslot);
  uint8_t* s_ninfref = in_tail ? at<uint8_t>(tb, TS.ninfref) : at<uint8_t>(sm, L.ninfref);
  const CompTable& ct = a.ct;
  const PairTable& pt = a.pt;
  const size_t capp = (size_t)pt.cap_pairs;
  const int tid = threadIdx.x, nthr = blockDim.x;

  // ---- parent header ----
  if (tid == 0) {
    const uint32_t lo = a.parents.ptr[h], hi = a.parents.ptr[h + 1];
    sc.Town = (int)(hi - lo);
    sc.T = sc.Town + nb;
    sc.ref_score = 0;
    sc.ninf_ref = 0;
    sc.nclut_ref = 0;
    sc.ndpc = 0;
    sc.nrca = 0;
    sc.bad = 0;
    sc.K = 0;
    sc.uid = a.parents.uid[h];
    sc.logw = a.parents.logw[h];
    // the block reads its sizes and counts on chip (the scan's words are
    // free until the scan)
    s_wsum[2] = (uint32_t)sc.T;
    s_wsum[3] = (uint32_t)sc.Town;
    s_wsum[4] = 0u;   // gated pairs
    s_wsum[5] = 0u;   // bad
  }
  __syncthreads();
  const int T = (int)s_wsum[2], Town = (int)s_wsum[3];
  const uint32_t plo = a.parents.ptr[h];
  // the parent's gated pairs, counted for every parent (also one beyond the
  // plan): the frame's maxima plan the next frame, or this frame's redo
  {
    unsigned kp = 0;
    for (int t = tid; t < T; t += nthr) {
      const uint32_t c = t < Town ? a.parents.comp[plo + t] : (uint32_t)(birth_base + (t - Town));
      if (c >= (uint32_t)(birth_base + nb)) {   // invariant: slots name the working table
        atomicOr(a.err, kErrChkComp);
        continue;
      }
      kp += pt.cnt[c];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kp += __shfl_xor_sync(0xFFFFFFFFu, kp, o);
    if ((tid & 31) == 0 && kp) atomicAdd(&s_wsum[4], kp);
  }
  __syncthreads();
  if (tid == 0) {
    const int K = (int)s_wsum[4];
    sc.K = K;
    int bad = (*(volatile const unsigned*)a.err & kErrChkComp) ? 1 : 0;
    if (a.max_T) atomicMax(a.max_T, (unsigned)T);
    if (a.max_K) atomicMax(a.max_K, (unsigned)K);
    if (T > a.T_max || M > a.M_plan || K > a.K_max) {
      bad = 1;
      atomicOr(a.err, kErrSlots);
    }
    sc.bad = bad;
    s_wsum[5] = (uint32_t)bad;
  }
  __syncthreads();
  if (s_wsum[5]) return;

  // ---- slots ----
  for (int t = tid; t < T; t += nthr) {
    const uint32_t c = t < Town ? a.parents.comp[plo + t] : (uint32_t)(birth_base + (t - Town));
    s_comp[t] = c;
    const uint32_t dt = pt.dthr[c];
    s_dthr[t] = dt;
    if (in_tail) g_dthr[t] = dt;
    s_mref[t] = 0;
#pragma unroll
    for (int d = 0; d < DZ; ++d) s_seref[d * T + t] = 0;
    s_sqref[t] = 0;
    s_hwref[t] = 0;
  }
  for (int i = tid; i <= M; i += nthr) s_rowfill[i] = 0;
  __syncthreads();
  for (int t = tid; t < T; t += nthr) {
    const uint32_t c = s_comp[t];
    const uint32_t n = pt.cnt[c], j0 = pt.ptr[c];
    for (uint32_t x = 0; x < n; x += 4) {   // four reads in flight
      uint32_t i4[4];
#pragma unroll
      for (uint32_t y = 0; y < 4; ++y) i4[y] = x + y < n ? pt.meas[j0 + x + y] : 0u;
#pragma unroll
      for (uint32_t y = 0; y < 4; ++y)
        if (x + y < n) atomicAdd(&s_rowfill[i4[y]], 1u);
    }
    s_srow[t] = (n && s_dthr[t] > 0u) ? 1 : 0;
  }
  __syncthreads();
  // exclusive scan of the row counts over the block: each thread a
  // contiguous run of rows, a scan of the runs' totals across the warps;
  // the offsets are also the fill cursors
  {
    const int per = (M + nthr - 1) / nthr;
    const int b0 = min(M, tid * per), b1 = min(M, b0 + per);
    uint32_t run = 0;
    for (int i = b0; i < b1; ++i) run += s_rowfill[i];
    const int lane = tid & 31, wp = tid >> 5;
    uint32_t x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_scan[wp] = x;
    __syncthreads();
    uint32_t base = x - run;
    for (int w = 0; w < wp; ++w) base += s_scan[w];
    for (int i = b0; i < b1; ++i) {
      const uint32_t v = s_rowfill[i];
      s_rowoff[i] = base;
      s_rowfill[i] = base;
      base += v;
    }
    if (tid == nthr - 1) {
      // the last thread's run ends at M (or is empty, with base the total)
      s_rowoff[M] = base;
      sc.K = (int)base;
      const bool over = (int)base > a.K_max;
      if (over) {
        sc.bad = 1;
        atomicOr(a.err, kErrSlots);
      }
      s_wsum[7] = over ? 1u : 0u;
    }
  }
  __syncthreads();
  if (s_wsum[7]) return;
  for (int t = tid; t < T; t += nthr) {
    const uint32_t c = s_comp[t];
    const uint32_t n = pt.cnt[c], j0 = pt.ptr[c];
    for (uint32_t x = 0; x < n; x += 4) {
      uint32_t i4[4];
#pragma unroll
      for (uint32_t y = 0; y < 4; ++y) i4[y] = x + y < n ? pt.meas[j0 + x + y] : 0u;
#pragma unroll
      for (uint32_t y = 0; y < 4; ++y)
        if (x + y < n) {
          const uint32_t pos = atomicAdd(&s_rowfill[i4[y]], 1u);
          s_cslot[pos] = (uint16_t)t;
          s_ceidx[pos] = j0 + x + y;
        }
    }
  }
  __syncthreads();

  // ---- rows: order, weights, thresholds, reference option ----
  // (the scan's sums are read; their words count the chunk lists next)
  if (tid == 0) {
    s_wsum[0] = 0u;
    s_wsum[1] = 0u;
  }
  {
    int my_clut = 0;
    // every thread runs the same rounds, so that the four rows of a chunk
    // (four neighbouring lanes: nthr is a multiple of 32) can pass their
    // parts of the chunk's record to its first lane
    for (int rb = 0; rb < M; rb += nthr) {
    const int i = rb + tid;
    bool r_has = false, r_flag = false;
    uint32_t r_lo = 0u, r_hi = kOne24;
    unsigned long long r_bl = 0ull;
    auto row_body = [&]() {
      if (i >= M) return;
      const uint32_t off = s_rowoff[i];
      const int nc = (int)(s_rowoff[i + 1] - off);
      if (nc == 0) {
        s_row[i] = make_uint4(off, 0u, 0u, kOne24);
        s_rowthr0[i] = kOne24;
        s_rowbl[i] = 0ull;
        s_rowrk[i] = 0u;
        s_roww0[i] = 1.f;
        ++my_clut;
        return;
      }
      // row i: x = first candidate, y = count | may-die flag << 15 |
      // reference option << 16, [z, w) = the uniforms that pick the reference
      // option when every candidate is alive; the reference slot's sums
      auto finish_row = [&](int ref, bool flag, uint32_t thr0, uint32_t lo, uint32_t hi, unsigned long long bl,
                            float w0, int r, const FVec<DZ> e_ref, float q_ref) {
        s_row[i] = make_uint4(off, (uint32_t)nc | (flag ? 0x8000u : 0u) | ((uint32_t)ref << 16), lo, hi);
        s_rowthr0[i] = thr0;
        s_rowbl[i] = bl;
        s_rowrk[i] = ref > 0 ? (((uint32_t)r + 1u) << 16) | (off + ref - 1) : 0u;
        s_roww0[i] = w0;
        r_has = true;
        r_flag = flag;
        r_lo = lo;
        r_hi = hi;
        r_bl = bl;
        if (ref == 0) {
          ++my_clut;
        } else {
          atomicAdd(&s_mref[r], 1);
#pragma unroll
          for (int d = 0; d < DZ; ++d)
            atomicAdd((unsigned long long*)&s_seref[d * T + r], (unsigned long long)fx_of(e_ref.v[d]));
          atomicAdd((unsigned long long*)&s_sqref[r], (unsigned long long)fx_of(q_ref));
          atomicAdd(&s_hwref[r], wset_key(i));
        }
      };
      if (nc <= kRowReg) {
        // the candidates in registers: sorted, weighed and thresholded with
        // the same operations in the same order as the general path below
        uint32_t cs[kRowReg], ce[kRowReg];
#pragma unroll
        for (int x = 0; x < kRowReg; ++x) {
          cs[x] = x < nc ? s_cslot[off + x] : 0xFFFFu;
          ce[x] = x < nc ? s_ceidx[off + x] : 0u;
        }
#pragma unroll
        for (int x = 1; x < kRowReg; ++x)
#pragma unroll
          for (int y = x; y > 0; --y)
            if (cs[y - 1] > cs[y]) {   // unused entries (0xFFFF) stay last
              const uint32_t ts = cs[y - 1], te = ce[y - 1];
              cs[y - 1] = cs[y];
              ce[y - 1] = ce[y];
              cs[y] = ts;
              ce[y] = te;
            }
        float lc[kRowReg];
        float smax = md.kappa_zero ? -INFINITY : md.log_kappa;
        // (reads before the writes, which might otherwise be the same memory
        // to the compiler and hold each read back for the write before it)
#pragma unroll
        for (int x = 0; x < kRowReg; ++x) lc[x] = x < nc ? pt.logC[ce[x]] : 0.f;
#pragma unroll
        for (int x = 0; x < kRowReg; ++x) {
          if (x >= nc) break;
          s_cslot[off + x] = (uint16_t)cs[x];
          s_ceidx[off + x] = ce[x];
          smax = fmaxf(smax, lc[x]);
        }
        const float w0 = md.kappa_zero ? 0.f : expf(md.log_kappa - smax);
        float wv[kRowReg];
        float sum = w0;
#pragma unroll
        for (int x = 0; x < kRowReg; ++x) {
          if (x >= nc) break;
          wv[x] = expf(lc[x] - smax);
          s_cw[off + x] = wv[x];
          sum += wv[x];
        }
        float cum = w0, best = w0;
        int ref = 0;
        bool flag = false;
        const uint32_t thr0 = thr_of(cum / sum);
        uint32_t lo = 0u, hi = thr0, prev = thr0;
        unsigned long long bl = 0ull;
        int r = 0;
        uint32_t rce = 0u;
        float rlc = 0.f;
#pragma unroll
        for (int x = 0; x < kRowReg; ++x) {
          if (x >= nc) break;
          const bool can_die = s_dthr[cs[x]] > 0u;
          if (can_die) bl |= 1ull << (cs[x] & 63);
          cum += wv[x];
          const uint32_t th = (x == nc - 1) ? kOne24 : thr_of(cum / sum);
          s_cthr[off + x] = th;
          if (wv[x] > best) {
            best = wv[x];
            ref = x + 1;
            lo = prev;
            hi = th;
            r = (int)cs[x];
            rce = ce[x];
            rlc = lc[x];
          }
          prev = th;
          flag |= can_die;
        }
        // the reference pair's innovation and q
        FVec<DZ> e_ref;
        float q_ref = 0.f;
#pragma unroll
        for (int d = 0; d < DZ; ++d) e_ref.v[d] = ref > 0 ? pt.e[d * capp + rce] : 0.f;
        if (ref > 0) q_ref = md.score_mode == 1 ? rlc : pt.q[rce];
        finish_row(ref, flag, thr0, lo, hi, bl, w0, r, e_ref, q_ref);
        return;
      }
      for (int x = 1; x < nc; ++x) {   // insertion sort by slot
        const uint16_t ks = s_cslot[off + x];
        const uint32_t ke = s_ceidx[off + x];
        int y = x - 1;
        while (y >= 0 && s_cslot[off + y] > ks) {
          s_cslot[off + y + 1] = s_cslot[off + y];
          s_ceidx[off + y + 1] = s_ceidx[off + y];
          --y;
        }
        s_cslot[off + y + 1] = ks;
        s_ceidx[off + y + 1] = ke;
      }
      float smax = md.kappa_zero ? -INFINITY : md.log_kappa;
      for (int j = 0; j < nc; ++j) {
        const uint32_t ei = s_ceidx[off + j];
        smax = fmaxf(smax, pt.logC[ei]);
      }
      const float w0 = md.kappa_zero ? 0.f : expf(md.log_kappa - smax);
      float sum = w0;
      for (int j = 0; j < nc; ++j) {
        const float w = expf(pt.logC[s_ceidx[off + j]] - smax);
        s_cw[off + j] = w;
        sum += w;
      }
      float cum = w0, best = w0;
      int ref = 0;
      bool flag = false;
      const uint32_t thr0 = thr_of(cum / sum);
      unsigned long long bl = 0ull;
      for (int j = 0; j < nc; ++j) {
        const float w = s_cw[off + j];
        const bool can_die = s_dthr[s_cslot[off + j]] > 0u;
        if (can_die) bl |= 1ull << (s_cslot[off + j] & 63);
        cum += w;
        s_cthr[off + j] = (j == nc - 1) ? kOne24 : thr_of(cum / sum);
        if (w > best) { best = w; ref = j + 1; }
        flag |= can_die;
      }
      const uint32_t lo = ref == 0 ? 0u : (ref == 1 ? thr0 : s_cthr[off + ref - 2]);
      const uint32_t hi = ref == 0 ? thr0 : s_cthr[off + ref - 1];
      FVec<DZ> e_ref;
      float q_ref = 0.f;
      int r = 0;
#pragma unroll
      for (int d = 0; d < DZ; ++d) e_ref.v[d] = 0.f;
      if (ref > 0) {
        const uint32_t pos = off + ref - 1;
        r = s_cslot[pos];
        const uint32_t ei = s_ceidx[pos];
#pragma unroll
        for (int d = 0; d < DZ; ++d) e_ref.v[d] = pt.e[d * capp + ei];
        // e^T R^-1 e of the pair; the factorised mode sums log C instead
        q_ref = md.score_mode == 1 ? pt.logC[ei] : pt.q[ei];
      }
      finish_row(ref, flag, thr0, lo, hi, bl, w0, r, e_ref, q_ref);
    };
    row_body();
    // the chunk's record, at its first lane
    {
      const int lane = tid & 31, lead = lane & ~3;
      uint32_t cmask = 0u, cdmask = 0u, blo = 0u, bhi = 0u, lo4[4], hi4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t has = __shfl_sync(0xFFFFFFFFu, r_has ? 1u : 0u, lead + q);
        const uint32_t fl = __shfl_sync(0xFFFFFFFFu, r_flag ? 1u : 0u, lead + q);
        const uint32_t bl0 = __shfl_sync(0xFFFFFFFFu, (uint32_t)r_bl, lead + q);
        const uint32_t bl1 = __shfl_sync(0xFFFFFFFFu, (uint32_t)(r_bl >> 32), lead + q);
        lo4[q] = __shfl_sync(0xFFFFFFFFu, r_lo, lead + q);
        hi4[q] = __shfl_sync(0xFFFFFFFFu, r_hi, lead + q);
        cmask |= has << q;
        if (fl) {
          cdmask |= 1u << q;
          blo |= bl0;
          bhi |= bl1;
        }
      }
      if (lane == lead && cmask) {
        RowChunk rc;
        rc.head = make_uint4((uint32_t)(i >> 2), cdmask, blo, bhi);
        rc.base = make_uint4(lo4[0] << 8, lo4[1] << 8, lo4[2] << 8, lo4[3] << 8);
        rc.span = make_uint4(((hi4[0] - lo4[0]) << 8) - 1u, ((hi4[1] - lo4[1]) << 8) - 1u,
                             ((hi4[2] - lo4[2]) << 8) - 1u, ((hi4[3] - lo4[3]) << 8) - 1u);
        s_rch[atomicAdd(&s_wsum[1], 1u)] = rc;
      }
    }
    }
    if (my_clut) atomicAdd(&sc.nclut_ref, my_clut);
  }
  __syncthreads();

  // ---- chunk lists ----
  {
    const int nch = (T + 3) >> 2;
    for (int cc = tid; cc < nch; cc += nthr) {
      // u < threshold, on the whole word: word <= (threshold << 8) - 1 (a
      // slot that cannot die keeps 0, which the mask bit sorts out)
      uint32_t mask = 0, top[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int t = 4 * cc + b;
        const uint32_t dt = t < T ? s_dthr[t] : 0u;
        if (dt > 0u) mask |= 1u << b;
        top[b] = dt > 0u ? (dt << 8) - 1u : 0u;
      }
      if (mask) {
        const uint32_t x = atomicAdd(&s_wsum[0], 1u);
        s_dpc[x] = ((uint32_t)cc << 4) | mask;
        s_dth[x] = make_uint4(top[0], top[1], top[2], top[3]);
      }
    }
  }
  __syncthreads();
  if (tid == 0) {
    sc.ndpc = (int)s_wsum[0];
    sc.nrca = (int)s_wsum[1];
  }

  // ---- reference terms ----
  {
    long long my_term = 0;
    int my_ninf = 0;
    for (int t = tid; t < T; t += nthr) {
      long long se[DZ];
#pragma unroll
      for (int d = 0; d < DZ; ++d) se[d] = s_seref[d * T + t];
      const int mr = s_mref[t];
      int ninf;
      long long term;
      if (md.score_mode == 0 && mr >= 1 && mr <= kSlmM && s_comp[t] < (uint32_t)a.pt.slm_cap) {
        term = term_from<DZ>(md, load_cslm<DZ>(a.pt.slm, a.pt.sln, a.pt.slm_cap, mr, s_comp[t]), mr, se, s_sqref[t],
                             ninf);
      } else {
        float HPH[DZ][DZ];
        slot_HPH<DZ>(ct, md.dx, s_comp[t], HPH);
        term = alive_term<DZ>(md, HPH, ct.logp[s_comp[t]], mr, se, s_sqref[t], ninf);
      }
      s_termref[t] = term;
      s_ninfref[t] = (uint8_t)ninf;
      my_term += term;
      my_ninf += ninf;
    }
    if (my_term) atomicAdd((unsigned long long*)&sc.ref_score, (unsigned long long)my_term);
    if (my_ninf) atomicAdd(&sc.ninf_ref, my_ninf);
  }
  __syncthreads();

  // ---- death deltas: a slot dying changes its term to the dead term (the
  // rows' single deviations are scored by the children that make them) ----
  {
    long long* s_deadd = at<long long>(sm, L.deadd);
    int8_t* s_dninf = at<int8_t>(sm, L.dninf);
    for (int t = tid; t < T; t += nthr) {
      int ninf;
      const long long term = dead_term(ct.log1mp[s_comp[t]], ninf);
      s_deadd[t] = term - s_termref[t];
      s_dninf[t] = (int8_t)(ninf - (int)s_ninfref[t]);
    }
  }
  if (in_tail) {
    // the arrays staged on chip go to the image
    __syncthreads();
    const int K = sc.K;
    uint16_t* g_cslot = at<uint16_t>(sm, L.cslot);
    uint32_t* g_ceidx = at<uint32_t>(sm, L.ceidx);
    for (int i = tid; i < K; i += nthr) {
      g_cslot[i] = s_cslot[i];
      g_ceidx[i] = s_ceidx[i];
    }
    int* g_mref = at<int>(sm, L.mref);
    long long* g_seref = at<long long>(sm, L.seref);
    long long* g_sqref = at<long long>(sm, L.sqref);
    unsigned long long* g_hwref = at<unsigned long long>(sm, L.hwref);
    long long* g_termref = at<long long>(sm, L.termref);
    uint8_t* g_ninfref = at<uint8_t>(sm, L.ninfref);
    for (int t = tid; t < T; t += nthr) {
      g_mref[t] = s_mref[t];
#pragma unroll
      for (int d = 0; d < DZ; ++d) g_seref[d * T + t] = s_seref[d * T + t];
      g_sqref[t] = s_sqref[t];
      g_hwref[t] = s_hwref[t];
      g_termref[t] = s_termref[t];
      g_ninfref[t] = s_ninfref[t];
    }
  }
  if (tid == 0) {
    sc.ref_score += __double2ll_rn(sc.logw * 4294967296.0);
    if (md.kappa_zero) sc.ninf_ref += sc.nclut_ref;
    else sc.ref_score += (long long)sc.nclut_ref * md.fx_log_kappa;
  }
}

// Persistent: CTA b stages parent b first (the launch spreads CTAs over the
// SMs, so a frame with few parents gets one SM each), then takes the next
// parent from a counter until none is left (parents differ in slots and
// pairs, so a fixed share per CTA would leave SMs idle at the end).
// SMEM: staged in shared memory and copied to the image (16-byte words).
// WIDE: CTAs of kStageWide threads, for a few parents of many slots and rows.
template <int DZ, bool SMEM, bool WIDE>
__global__ void __launch_bounds__(WIDE ? kStageWide : 256, WIDE ? 1 : 3) stage_kernel(const __grid_constant__ ExpandArgs a) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char sm[];
  const Lay L = make_lay(DZ, a.T_max, a.K_max, a.M_plan);
  // after the staged image (SMEM) or alone: the next-parent word, then the
  // staging's shared scratch (expand_stage_tail_bytes)
  unsigned char* tb = sm + (SMEM ? L.total : 0);
  int& s_next = *reinterpret_cast<int*>(tb);
  const int H = a.fs->H;
  // a table that failed (e.g. pairs beyond capacity, whose offsets then run
  // past the pair arrays) is not staged; the frame is abandoned.  The flags
  // this kernel raises itself (a parent beyond the plan, a bad slot index)
  // are set by its CTAs while others start, so they must not stop a CTA:
  // every parent's counts are recorded
  if (*(volatile const unsigned*)a.err & (kErrFatal & ~(kErrSlots | kErrChkComp))) return;
  for (int h = blockIdx.x; h < H;) {
    unsigned char* img = a.img + (size_t)h * a.img_stride;
    stage_parent<DZ>(a, h, L, SMEM ? sm : img, tb, SMEM ? 0 : a.stage_tail);
    __syncthreads();
    if (SMEM) {
      // a parent whose staging failed copies only its header
      const int bytes = at<Scal>(sm, L.scal)->bad ? (int)sizeof(Scal) : L.total;
      const uint4* src = reinterpret_cast<const uint4*>(sm);
      uint4* dst = reinterpret_cast<uint4*>(img);
      for (int w = threadIdx.x; w < (bytes + 15) / 16; w += blockDim.x) dst[w] = src[w];
    }
    __syncthreads();   // the copy-out has read shared memory, s_next is free
    if (threadIdx.x == 0) s_next = (int)gridDim.x + (int)atomicAdd(a.stage_next, 1u);
    __syncthreads();
    h = s_next;
  }
}

// ====================== draw: one thread per child ======================
// A child's deaths come first: one Philox4x32-10 call per chunk of four
// slots that can die.  Then one categorical draw per detection row with
// candidates, one call per chunk of four rows.  A row keeps its reference
// option when its 24-bit uniform falls in the reference interval and none
// of its candidates died -- nearly always -- so the common path reads one
// 48-byte chunk record and tests four intervals per call, and holds only
// the chunk loop's state in registers.  Everything else about a row is left
// to finish_notes: a row with a candidate that may have died is drawn
// among the living, and a row that leaves the reference adds the change of
// a single deviation.  Whether a slot died is answered by its
// bloom bit and, when that is set, by regenerating the slot's death draw,
// so a thread keeps no lists.  The slots a child's deviations meet are
// kept as a 64-bit mask (bit slot mod 64): when a bit is met again (a slot
// met twice, or two slots sharing a bit), the slots met more than once are
// rescored exactly after the rows.

// Whether slot t of the child whose death stream is pd died.
__device__ __forceinline__ bool slot_died(const uint32_t* __restrict__ dthr, const PhiloxRun& pd, uint2 key,
                                          uint32_t t) {
  const uint4 r = philox_at_rk(pd, t >> 2, key);
  return (word_of(r, (int)(t & 3u)) >> 8) < dthr[t];
}

// Rows a child's chunk loop sets aside for finish_notes (per-thread list in
// shared memory, entry q at [q * blockDim.x]); a child with more goes to
// the warp kernel.
constexpr int kDrawSlow = 24;
// Dead slots the first death pass records for the score pass (the same
// kind of per-thread list, after the noted rows); a child with more
// regenerates its death draws instead.
constexpr int kDrawDead = 8;
// Chunks per iteration of the draw loops: independent Philox chains in
// flight (rows: 2 or 4 measured the same as 3 within 1 %).
constexpr int kDrawDeaths = 2, kDrawRows = 3;

// What the chunk loops read of a parent, staged in shared memory beside the
// other parents of a CTA's children: offsets from the parent's part.
struct DrawRec {
  int rch, dth, dpc, total;
};
__host__ __device__ inline DrawRec make_draw_rec(int T, int M) {
  DrawRec R;
  Bump b;
  R.rch = b.take(48LL * ((M + 3) / 4 + 1));
  R.dth = b.take(16LL * (T / 4 + 2));
  R.dpc = b.take(4LL * (T / 4 + 2));
  R.total = b.off;
  return R;
}
// A child whose chunk loop noted rows: what finish_notes needs beside the
// child's partial sums (child_key, child_hash, child_alive).
struct DrawNote {
  uint32_t child;
  uint16_t n_rows;
  int16_t dninf;
  unsigned long long bloom;
  uint16_t rows[kDrawSlow];
};
size_t expand_note_bytes() { return sizeof(DrawNote); }
// parents that `threads` consecutive children can belong to
__host__ __device__ inline int draw_parents(int threads, int h_up) { return (threads - 1) / h_up + 2; }

template <int N>
struct Int {
  static constexpr int value = N;
};

// Draws child n of the parent staged at img; rch, dth and dpc are the
// parent's arrays of these names (in shared memory, or the image's).  The
// chunk loops only test the thresholds and intervals and note the slots that
// die and the rows that need more (their uniform is regenerated afterwards),
// so they hold nothing but their own state in registers.  Slots its
// deviations meet more than once are rescored exactly (finish_notes).  A child
// with more noted rows than the list holds is left to the warp kernel (the
// redo list).
template <int DZ>
__device__ __forceinline__ void thread_child(const ExpandArgs& a, const unsigned char* img, const Lay& L, const int h,
                                             const int n, const uint2 key, uint16_t* s_slow, uint16_t* s_dead,
                                             const RowChunk* rch, const uint4* dth, const uint32_t* dpc) {
  const Model& md = a.md;
  const Scal& sc = *at<Scal>(img, L.scal);
  const int bd = (int)blockDim.x;
  unsigned long long bloom = 0ull;
  int nd = 0;
  {
    // stage 1: deaths; only their bloom (slots with candidate rows) is kept
    // through the chunk loop, their score and key changes are summed after
    const uint8_t* srow = at<uint8_t>(img, L.srow);
    const PhiloxRun pd = philox_run((uint32_t)sc.uid, (uint32_t)(sc.uid >> 32), 2u * (uint32_t)n, key);
    const int ndpc = sc.ndpc;
    // N chunks: N independent Philox chains in flight
    auto chunks = [&](int x, auto nn) {
      constexpr int N = decltype(nn)::value;
      uint32_t e[N];
      uint4 r[N];
#pragma unroll
      for (int u = 0; u < N; ++u) e[u] = dpc[x + u];
#pragma unroll
      for (int u = 0; u < N; ++u) r[u] = philox_at(pd, e[u] >> 4, key);
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const uint4 th = dth[x + u];
        if (r[u].x <= th.x || r[u].y <= th.y || r[u].z <= th.z || r[u].w <= th.w) {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (word_of(r[u], b) <= word_of(th, b) && ((e[u] >> b) & 1u)) {
              const uint32_t t = 4u * (e[u] >> 4) + (uint32_t)b;
              if (nd < kDrawDead) s_dead[nd * bd] = (uint16_t)t;
              ++nd;
              if (srow[t]) bloom |= 1ull << (t & 63u);
            }
        }
      }
    };
    int x = 0;
    for (; x + kDrawDeaths <= ndpc; x += kDrawDeaths) chunks(x, Int<kDrawDeaths>());
    for (; x < ndpc; ++x) chunks(x, Int<1>());
  }
  // stage 2: one categorical draw per detection row with candidates; rows
  // outside their reference interval, or whose candidates' bloom meets the
  // dead slots', are noted
  int nslow = 0;
  {
    const PhiloxRun pr = philox_run((uint32_t)sc.uid, (uint32_t)(sc.uid >> 32), 2u * (uint32_t)n + 1u, key);
    const unsigned long long* rowbl = at<unsigned long long>(img, L.rowbl);
    const uint32_t blo = (uint32_t)bloom, bhi = (uint32_t)(bloom >> 32);
    const int nrca = sc.nrca;
    auto chunks = [&](int x, auto nn) {
      constexpr int N = decltype(nn)::value;
      uint4 r[N];
#pragma unroll
      for (int u = 0; u < N; ++u) r[u] = philox_at(pr, rch[x + u].head.x, key);
#pragma unroll
      for (int u = 0; u < N; ++u) {
        const uint4 hd = rch[x + u].head, base = rch[x + u].base, span = rch[x + u].span;
        const uint32_t hit = (hd.z & blo) | (hd.w & bhi);
        // nearly always false: all four rows keep their reference
        if (r[u].x - base.x > span.x || r[u].y - base.y > span.y || r[u].z - base.z > span.z ||
            r[u].w - base.w > span.w || hit) {
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const uint32_t i = 4u * hd.x + (uint32_t)b;
            bool look = word_of(r[u], b) - word_of(base, b) > word_of(span, b);
            // a row of a chunk whose bloom meets the dead slots', still in
            // its reference interval: noted only if its own bloom does
            if (!look && hit && ((hd.y >> b) & 1u)) look = (rowbl[i] & bloom) != 0ull;
            if (look) {
              if (nslow < kDrawSlow) s_slow[nslow * bd] = (uint16_t)i;
              ++nslow;
            }
          }
        }
      }
    };
    int x = 0;
    for (; x + kDrawRows <= nrca; x += kDrawRows) chunks(x, Int<kDrawRows>());
    for (; x < nrca; ++x) chunks(x, Int<1>());
  }
  const size_t j = (size_t)h * md.h_up + n;
  if (nslow > kDrawSlow) {
    a.redo_list[atomicAdd(a.redo_count, 1u)] = (uint32_t)j;
    return;
  }
  // the deaths' score and key changes (a dead slot's change is its dead term)
  unsigned long long hsh = 0ull;
  long long delta = 0;
  int dninf = 0;
  const long long* deadd = at<long long>(img, L.deadd);
  const int8_t* dninf8 = at<int8_t>(img, L.dninf);
  if (nd <= kDrawDead) {
    // four deaths' loads in flight (the image's tables come from L2 or HBM)
    for (int q0 = 0; q0 < nd; q0 += 4) {
#pragma unroll
      for (int q = q0; q < q0 + 4; ++q)
        if (q < nd) {
          const int t = s_dead[q * bd];
          hsh += dead_key(t);
          delta += deadd[t];
          dninf += dninf8[t];
        }
    }
  } else {
    // more deaths than the list holds: their draws again
    const PhiloxRun pd = philox_run((uint32_t)sc.uid, (uint32_t)(sc.uid >> 32), 2u * (uint32_t)n, key);
    const int ndpc = sc.ndpc;
    for (int x = 0, left = nd; x < ndpc && left; ++x) {
      const uint32_t ent = dpc[x];
      const uint4 r = philox_at(pd, ent >> 4, key), th = dth[x];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint32_t t = 4u * (ent >> 4) + (uint32_t)b;
        if (word_of(r, b) <= word_of(th, b) && ((ent >> b) & 1u)) {
          --left;
          hsh += dead_key((int)t);
          delta += deadd[t];
          dninf += dninf8[t];
        }
      }
    }
  }
  a.child_hash[j] = hsh;
  a.child_alive[j] = (uint16_t)(sc.T - nd);
  if (nslow) {
    // the noted rows are left to finish_notes, with the deaths' sums
    const unsigned act = __activemask();
    const int lane = (int)threadIdx.x & 31, lead = __ffs(act) - 1;
    unsigned k = 0;
    if (lane == lead) k = atomicAdd(a.note_count, (unsigned)__popc(act));
    k = __shfl_sync(act, k, lead) + __popc(act & ((1u << lane) - 1u));
    if (k >= a.note_cap) {
      a.redo_list[atomicAdd(a.redo_count, 1u)] = (uint32_t)j;
      return;
    }
    DrawNote* o = reinterpret_cast<DrawNote*>(a.notes) + k;
    o->child = (uint32_t)j;
    o->n_rows = (uint16_t)nslow;
    o->dninf = (int16_t)dninf;
    o->bloom = bloom;
    for (int q = 0; q < nslow; ++q) o->rows[q] = s_slow[q * bd];
    a.child_key[j] = delta;
    return;
  }
  const int ninf = sc.ninf_ref + dninf;
  a.child_key[j] = ninf == 0 ? sc.ref_score + delta : kKeyInvalid;
  a.child_status[j] = ninf == 0 ? 1 : 0;
}

// The noted children, kNoteLanes lanes each, a row to a lane at a time.  In
// the draw kernel itself the few lanes with noted rows would hold their warps
// through the rows' chains of dependent loads (row, candidate, pair, slot,
// term); here the lanes are dense and a child's chains run side by side
// (the launch with a lane per child and its images' own copies of the pairs:
// 25 us at 3-D N = 50, 51 at N = 200; now 14.6 and about 20).
// Each row's uniform is regenerated; a row whose candidates' bloom meets the
// child's dead slots is drawn among the living candidates in proportion to
// their weights (clutter first), in the FP32 arithmetic of the warp kernel;
// otherwise its option is the first whose cumulative threshold exceeds the
// uniform.  A row that leaves its reference option adds the changes of the
// slots it leaves and joins, each scored alone (a dead reference slot is not
// met: its change is the death's).  When the deviations meet a slot more than
// once, that slot's change is not the sum of the single changes but the exact
// rescoring of the slot with every detection that joins and leaves it: such
// slots are rescored with the warp kernel's functions and inputs, so the keys
// are bit-identical.
constexpr int kNoteLanes = 8, kNoteEnt = 2 * (kDrawSlow / kNoteLanes);
static_assert(kDrawSlow % kNoteLanes == 0, "rows of a note over its lanes");

template <int DZ>
__device__ __noinline__ void finish_notes(const ExpandArgs& a, const Lay& L, const uint2 key) {
  const Model& md = a.md;
  const uint32_t count = min(*a.note_count, a.note_cap), HU = (uint32_t)md.h_up;
  const int lane = (int)threadIdx.x & 31, gl = lane & (kNoteLanes - 1);
  const unsigned gm = ((1u << kNoteLanes) - 1u) << (lane - gl);
  const uint32_t step = gridDim.x * blockDim.x / kNoteLanes;
  for (uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) / kNoteLanes; k < count; k += step) {
    const DrawNote* o = reinterpret_cast<const DrawNote*>(a.notes) + k;
    const uint32_t j = o->child, h = j / HU, n = j - h * HU;
    const int n_rows = o->n_rows;
    const unsigned long long bloom = o->bloom;
    const View v = make_view(a.img + (size_t)h * a.img_stride, L, a.pt, a.ct);
    const Scal& sc = *v.sc;
    const int T = sc.T;
    const PhiloxRun pd = philox_run((uint32_t)sc.uid, (uint32_t)(sc.uid >> 32), 2u * n, key);
    const PhiloxRun pr = philox_run((uint32_t)sc.uid, (uint32_t)(sc.uid >> 32), 2u * n + 1u, key);
    long long dsum = 0;
    unsigned long long hw = 0ull, metm = 0ull;
    int ninf = 0, clut = 0, ne = 0;
    unsigned flags = 0u;   // 1: a row without a weight, 2: a slot met twice
    // this lane's single deviations: slot + 1, leaving << 16, (infinite-term
    // change + 128) << 17; the pair; the score change
    uint32_t e_tag[kNoteEnt], e_pos[kNoteEnt];
    long long e_d[kNoteEnt];
    auto deviation = [&](uint32_t s1, uint32_t pos, int sg) {   // alone: joining (1) or leaving (-1) slot s1 - 1
      const int t = (int)s1 - 1;
      long long e[DZ], q, se[DZ];
      pair_sums<DZ>(md, v, pos, e, q);
#pragma unroll
      for (int d = 0; d < DZ; ++d) se[d] = v.seref[d * T + t] + (long long)sg * e[d];
      int ni;
      const long long term = slot_term<DZ>(md, v, t, v.mref[t] + sg, se, v.sqref[t] + (long long)sg * q, ni);
      const long long d = term - v.termref[t];
      const int dn = ni - (int)v.ninfref[t];
      dsum += d;
      ninf += dn;
      const unsigned long long m = 1ull << ((uint32_t)t & 63u);
      if (metm & m) flags |= 2u;
      metm |= m;
      e_tag[ne] = s1 | (sg < 0 ? 1u << 16 : 0u) | ((uint32_t)(dn + 128) << 17);
      e_pos[ne] = pos;
      e_d[ne] = d;
      ++ne;
    };
    for (int r = gl; r < n_rows; r += kNoteLanes) {
      const int i = o->rows[r];
      const uint4 rr = philox_at_rk(pr, (uint32_t)i >> 2, key);
      const uint32_t u = word_of(rr, i & 3) >> 8;
      const uint4 R = v.row[i];
      const uint32_t off = R.x;
      const int nc = (int)(R.y & 0x7FFFu);
      const int ref = (int)(R.y >> 16);
      int opt = -1;
      if (v.rowbl[i] & bloom) {
        auto is_dead = [&](int x) -> bool {
          const uint32_t t = v.cslot[off + x];
          return ((bloom >> (t & 63u)) & 1ull) && slot_died(v.dthr, pd, key, t);
        };
        uint32_t dm = 0u;
        bool any = false;
        for (int x = 0; x < nc; ++x)
          if (is_dead(x)) {
            any = true;
            if (x < 32) dm |= 1u << x;
          }
        if (any) {
          auto dead_x = [&](int x) -> bool { return x < 32 ? ((dm >> x) & 1u) != 0u : is_dead(x); };
          const float w0 = md.kappa_zero ? 0.f : v.roww0[i];
          float sum = w0;
          for (int x = 0; x < nc; ++x)
            if (!dead_x(x)) sum += v.cw[off + x];
          if (!(sum > 0.f)) {
            flags |= 1u;
            opt = 0;
          } else {
            const float xk = (float)u * 5.9604644775390625e-8f * sum;
            float cum = w0;
            int last = w0 > 0.f ? 0 : -1;
            if (w0 > 0.f && xk < cum) opt = 0;
            for (int x = 0; x < nc; ++x) {
              if (dead_x(x)) continue;
              const float w = v.cw[off + x];
              if (!(w > 0.f)) continue;
              cum += w;
              last = x + 1;
              if (opt < 0 && xk < cum) opt = x + 1;
            }
            if (opt < 0) opt = last < 0 ? 0 : last;
          }
        }
      }
      if (opt < 0) {
        if (u - R.z < R.w - R.z) continue;   // the reference option
        if (u < v.rowthr0[i]) {
          opt = 0;
        } else {
          int x = 0;
          while (x < nc - 1 && u >= v.cthr[off + x]) ++x;
          opt = x + 1;
        }
      }
      if (opt == ref) continue;
      uint32_t rs1 = ref > 0 ? (uint32_t)v.cslot[off + ref - 1] + 1u : 0u;
      const uint32_t ns1 = opt > 0 ? (uint32_t)v.cslot[off + opt - 1] + 1u : 0u;
      hw += row_key(i, (int)ns1) - row_key(i, (int)rs1);
      clut += (opt == 0) - (ref == 0);
      if (rs1 && ((bloom >> ((rs1 - 1u) & 63u)) & 1ull) && slot_died(v.dthr, pd, key, rs1 - 1u)) rs1 = 0u;
      if (rs1) deviation(rs1, off + (uint32_t)ref - 1u, -1);
      if (ns1) deviation(ns1, off + (uint32_t)opt - 1u, 1);
    }
    __syncwarp(gm);
    // two lanes that met the same slot (or slots that share a bit)
#pragma unroll
    for (int x = 1; x < kNoteLanes; x <<= 1) {
      const unsigned long long other = __shfl_xor_sync(gm, metm, x);
      if (metm & other) flags |= 2u;
      metm |= other;
    }
    flags = __reduce_or_sync(gm, flags);
    if (flags & 2u) {
      // slots met more than once, each by the lane of its first deviation:
      // exact term minus reference term minus the single changes added above
      const int most = (int)__reduce_max_sync(gm, (unsigned)ne);
      for (int w = 0; w < most; ++w) {
        const uint32_t mine = w < ne ? e_tag[w] & 0xFFFFu : 0u;
        bool first = mine != 0u;
        int cnt = 0, dcnt = 0, sninf = 0;
        long long dse[DZ], dsq = 0, single = 0;
#pragma unroll
        for (int d = 0; d < DZ; ++d) dse[d] = 0;
        for (int src = 0; src < kNoteLanes; ++src) {
          const int from = lane - gl + src;
          const int n_src = __shfl_sync(gm, ne, from);
          for (int x = 0; x < n_src; ++x) {
            const int y = min(x, kNoteEnt - 1);
            const uint32_t tag = __shfl_sync(gm, e_tag[y], from), pos = __shfl_sync(gm, e_pos[y], from);
            const long long d1 = __shfl_sync(gm, e_d[y], from);
            if ((tag & 0xFFFFu) != mine) continue;
            if (src < gl || (src == gl && x < w)) first = false;
            if (!first) continue;
            ++cnt;
            const int sg = (tag >> 16) & 1u ? -1 : 1;
            single += d1;
            sninf += (int)(tag >> 17) - 128;
            dcnt += sg;
            long long e[DZ], q;
            pair_sums<DZ>(md, v, pos, e, q);
#pragma unroll
            for (int d = 0; d < DZ; ++d) dse[d] += sg * e[d];
            dsq += sg * q;
          }
        }
        if (first && cnt >= 2) {
          const int t = (int)mine - 1;
          long long se[DZ];
#pragma unroll
          for (int d = 0; d < DZ; ++d) se[d] = v.seref[d * T + t] + dse[d];
          int ni;
          const long long term = slot_term<DZ>(md, v, t, v.mref[t] + dcnt, se, v.sqref[t] + dsq, ni);
          dsum += term - v.termref[t] - single;
          ninf += ni - (int)v.ninfref[t] - sninf;
        }
        __syncwarp(gm);
      }
    }
#pragma unroll
    for (int x = 1; x < kNoteLanes; x <<= 1) {
      dsum += __shfl_xor_sync(gm, dsum, x);
      hw += __shfl_xor_sync(gm, hw, x);
      ninf += __shfl_xor_sync(gm, ninf, x);
      clut += __shfl_xor_sync(gm, clut, x);
    }
    if (gl == 0) {
      const long long score =
          sc.ref_score + a.child_key[j] + dsum + (md.kappa_zero ? 0LL : (long long)clut * md.fx_log_kappa);
      const bool valid = !(flags & 1u) && sc.ninf_ref + o->dninf + ninf + (md.kappa_zero ? clut : 0) == 0;
      a.child_key[j] = valid ? score : kKeyInvalid;
      a.child_hash[j] += hw;
      a.child_status[j] = valid ? 1 : 0;
    }
  }
}

int expand_stage_tail_bytes(int dz, int T_plan, int K_plan, int M_plan, int mode) {
  return make_stage_tail(dz, T_plan, K_plan, M_plan, mode).total;
}

// lists of the threads, then (staged) the parents' records
int expand_draw_smem(int threads, int h_up, int T, int M, bool staged) {
  return threads * (kDrawSlow + kDrawDead) * (int)sizeof(uint16_t) +
         (staged ? draw_parents(threads, h_up) * make_draw_rec(T, M).total : 0);
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Persistent over the children of the frame, one thread per child in the
// order parent * h_up + draw (a warp holds 32 consecutive children, of at
// most two parents when h_up >= 32).  STAGED: the CTA first copies what the
// chunk loops read of its children's parents to shared memory, so that the
// loops wait for no cache miss (a parent's records are read by three or four
// warps only: from the image one load in four missed L1, half of those L2).
// What bounds the loops is the integer pipes: 41 instructions per Philox call
// (16 wide multiplications at half rate), issued on 57 % of the cycles.
// Measured with the rows' follow-up moved to finish_notes, one launch of the
// 3-D N = 200 scene at H_max = 5000: 295 -> 226 us (161 -> 127 M warp
// instructions); two children per thread sharing the records' loads: 3-9 %
// slower, 64 registers (four CTAs per SM, spilled): 4 % slower, 128 registers
// (two CTAs): 4 % slower.
template <int DZ, bool STAGED>
__global__ void __launch_bounds__(256, 3) draw_kernel(const __grid_constant__ ExpandArgs a) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char sm[];
  const int bd = (int)blockDim.x, tid = (int)threadIdx.x;
  uint16_t* s_slow = reinterpret_cast<uint16_t*>(sm) + tid;
  uint16_t* s_dead = s_slow + kDrawSlow * bd;
  unsigned char* s_rec = sm + bd * (kDrawSlow + kDrawDead) * (int)sizeof(uint16_t);
  const Lay L = make_lay(DZ, a.T_max, a.K_max, a.M_plan);
  const DrawRec R = make_draw_rec(a.T_max, a.M_plan);
  const int H = a.fs->H, HU = a.md.h_up;
  const uint2 key = make_uint2(a.key_x, a.key_y);
  // a failed table or staging (the frame is redone or abandoned): the
  // images may be stale, so nothing is drawn
  if (*(volatile const unsigned*)a.err & kErrFatal) return;
  const long long total = (long long)H * HU;
  // children a CTA takes at a time: one per thread, or fewer (whole warps)
  // when the children would leave CTAs without any
  const int q = (int)min((long long)bd, ((total + gridDim.x - 1) / gridDim.x + 31) / 32 * 32);
  for (long long j0 = (long long)blockIdx.x * q; j0 < total; j0 += (long long)gridDim.x * q) {
    const int nk = (int)min((long long)q, total - j0);
    const int h0 = (int)(j0 / HU);
    const int n0 = (int)(j0 - (long long)h0 * HU);   // the first child's draw
    if (STAGED) {
      const int np = (n0 + nk - 1) / HU + 1;
      __syncthreads();   // the last round's records are read
      for (int p = 0; p < np; ++p) {
        const unsigned char* img = a.img + (size_t)(h0 + p) * a.img_stride;
        const Scal& sc = *at<Scal>(img, L.scal);
        if (sc.bad) continue;
        unsigned char* rec = s_rec + p * R.total;
        const int nr = 3 * sc.nrca, nt = sc.ndpc, nc = (sc.ndpc + 3) >> 2;
        for (int w = tid; w < nr; w += bd) cp_async16(rec + R.rch + 16 * w, img + L.rch + 16 * w);
        for (int w = tid; w < nt; w += bd) cp_async16(rec + R.dth + 16 * w, img + L.dth + 16 * w);
        for (int w = tid; w < nc; w += bd) cp_async16(rec + R.dpc + 16 * w, img + L.dpc + 16 * w);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
    }
    if (tid < nk) {
      const int h = h0 + (n0 + tid) / HU;
      const unsigned char* img = a.img + (size_t)h * a.img_stride;
      if (!at<Scal>(img, L.scal)->bad) {
        const unsigned char* rec = s_rec + (h - h0) * R.total;
        thread_child<DZ>(a, img, L, h, n0 + tid - (h - h0) * HU, key, s_slow, s_dead,
                         STAGED ? at<RowChunk>(rec, R.rch) : at<RowChunk>(img, L.rch),
                         STAGED ? at<uint4>(rec, R.dth) : at<uint4>(img, L.dth),
                         STAGED ? at<uint32_t>(rec, R.dpc) : at<uint32_t>(img, L.dpc));
      }
    }
  }
}

// ====================== warp: one warp per child ======================
// The work area's sums, masks and touched list are zero on entry and are
// left zero on return.
template <int DZ, bool MAT, bool GRP>
__device__ void warp_child(const ExpandArgs& a, const View& v, const int T, const int M,
                           const int h, const int n, const int s_out, const uint2 key, unsigned char* gb,
                           const WLay& WL, const int gsz_in, const int gid) {
  const int gsz = GRP ? gsz_in : 32;   // one warp: the group code folds away
  const Model& md = a.md;
  const Scal& sc = *v.sc;
  const int HU = md.h_up;
  const int lane = threadIdx.x & 31;
  const int gl = (int)threadIdx.x % gsz;   // the thread's index in its group
  unsigned long long* red = at<unsigned long long>(gb, WL.red);
  const int W = (T + 31) >> 5;
  const int nrc = (M + 3) >> 2;
  const uint32_t uid_lo = (uint32_t)sc.uid, uid_hi = (uint32_t)(sc.uid >> 32);
  const int ndpc = sc.ndpc;
  int* acc_cnt = at<int>(gb, WL.cnt);
  long long* acc_se = at<long long>(gb, WL.se);
  long long* acc_sq = at<long long>(gb, WL.sq);
  unsigned long long* acc_hw = at<unsigned long long>(gb, WL.hw);
  uint32_t* newval = at<uint32_t>(gb, WL.newval);
  uint32_t* tmask = at<uint32_t>(gb, WL.tmask);
  uint32_t* dmask = at<uint32_t>(gb, WL.dmask);
  uint32_t* dpre = at<uint32_t>(gb, WL.dpre);
  uint16_t* tlist = at<uint16_t>(gb, WL.tlist);
  int* ntp = at<int>(gb, WL.nt);

  // phase 1: deaths
  int my_dead = 0;
  unsigned long long hsh = 0;
  for (int x = gl; x < ndpc; x += gsz) {
    const uint32_t ent = v.dpc[x];
    const uint4 th = v.dth[x];
    const uint32_t cc = ent >> 4;
    const uint4 r = philox10(make_uint4(uid_lo, uid_hi, 2u * (uint32_t)n, cc), key);
    if (r.x <= th.x || r.y <= th.y || r.z <= th.z || r.w <= th.w) {
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (word_of(r, b) <= word_of(th, b) && ((ent >> b) & 1u)) {
          const int t = 4 * (int)cc + b;
          atomicOr(&dmask[t >> 5], 1u << (t & 31));
          touch(tmask, tlist, ntp, t);
          ++my_dead;
          hsh += dead_key(t);
        }
    }
  }
  group_sync(gsz, gid);
  if (MAT) {
    if (gl < 32) {   // the group's first warp
      uint32_t carry = 0;
      for (int base = 0; base < W; base += 32) {
        const int w = base + lane;
        const uint32_t val = w < W ? (uint32_t)__popc(dmask[w]) : 0u;
        uint32_t x = val;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
          if (lane >= o) x += y;
        }
        if (w < W) dpre[w] = carry + x - val;
        carry += __shfl_sync(0xFFFFFFFFu, x, 31);
      }
    }
    group_sync(gsz, gid);
  }
  // phase 2: one categorical draw per detection row.  The dead slots'
  // bloom (slot mod 64) screens a row's candidates before the exact check;
  // a row none of whose candidates died whose uniform is in its reference
  // interval keeps its reference option without its thresholds
  int my_dclut = 0;
  bool bad_row = false;
  unsigned long long dbl = 0ull;
  for (int w = gl; w < W; w += gsz)
    for (uint32_t m = dmask[w]; m; m &= m - 1u) dbl |= 1ull << ((32 * w + __ffs(m) - 1) & 63);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dbl |= __shfl_xor_sync(0xFFFFFFFFu, dbl, o);
  if (gsz > 32) {
    if (lane == 0 && dbl) atomicOr(&red[0], dbl);
    group_sync(gsz, gid);
    dbl = red[0];
  }
  const PhiloxRun pr = philox_run(uid_lo, uid_hi, 2u * (uint32_t)n + 1u, key);
  // detection i takes slot ns (-1: clutter): its place among the survivors
  auto put_theta = [&](int i, int ns) {
    uint16_t th = 0;
    if (ns >= 0) {
      const uint32_t below = dpre[ns >> 5] + __popc(dmask[ns >> 5] & ((1u << (ns & 31)) - 1u));
      th = (uint16_t)(ns - (int)below + 1);
    }
    a.out_theta[(size_t)s_out * M + i] = th;
  };
  for (int cc = gl; cc < nrc; cc += gsz) {
    const int i0 = 4 * cc;
    const int nr = min(4, M - i0);
    // the chunk's rows, all loads in flight before the first test: row by
    // row (and the option's slot after the row) the chunk was a chain of
    // eight dependent reads of the image (expansion of 40 particle tracks
    // with 10 000 children 38.5 -> 35.5 us; regeneration of the 3-D N = 200
    // scene's retained children 105 -> 98 us, 2-D N = 100 27 -> 24 us)
    uint4 R4[4];
    unsigned long long bl4[4];
    uint32_t rk4[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      R4[b] = b < nr ? v.row[i0 + b] : make_uint4(0u, 0u, 0u, kOne24);
      bl4[b] = b < nr ? v.rowbl[i0 + b] : 0ull;
      if (MAT) rk4[b] = b < nr ? v.rowrk[i0 + b] : 0u;
    }
    const uint4 r = philox_at(pr, (uint32_t)cc, key);
    uint32_t look = 0u;   // rows that left their reference interval, or whose candidates may have died
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const uint32_t k = word_of(r, b) >> 8;
      if (!(k - R4[b].z < R4[b].w - R4[b].z) || ((R4[b].y & 0x8000u) && (bl4[b] & dbl))) look |= 1u << b;
      else if (MAT && b < nr) put_theta(i0 + b, (int)(rk4[b] >> 16) - 1);   // the reference option's slot
    }
    while (look) {
      const int b = __ffs(look) - 1;
      look &= look - 1u;
      const int i = i0 + b;
      const uint4 R = v.row[i];
      const uint32_t off = R.x;
      const int nc = (int)(R.y & 0x7FFFu);
      const uint32_t k = word_of(r, b) >> 8;
      bool fast = true;
      if ((R.y & 0x8000u) && (v.rowbl[i] & dbl))
        for (int j = 0; j < nc; ++j)
          if (bit_of(dmask, v.cslot[off + j])) { fast = false; break; }
      const int ref = (int)(R.y >> 16);
      int opt;
      if (fast && k - R.z < R.w - R.z) {
        opt = ref;
      } else if (fast) {
        if (k < v.rowthr0[i]) {
          opt = 0;
        } else {
          int j = 0;
          while (j < nc - 1 && k >= v.cthr[off + j]) ++j;
          opt = j + 1;
        }
      } else {
        const float w0 = md.kappa_zero ? 0.f : v.roww0[i];
        float sum = w0;
        for (int j = 0; j < nc; ++j)
          if (!bit_of(dmask, v.cslot[off + j])) sum += v.cw[off + j];
        if (!(sum > 0.f)) {
          bad_row = true;
          opt = 0;
        } else {
          const float xk = (float)k * 5.9604644775390625e-8f * sum;
          float cum = w0;
          int last = w0 > 0.f ? 0 : -1;
          opt = -1;
          if (w0 > 0.f && xk < cum) opt = 0;
          for (int j = 0; j < nc; ++j) {
            if (bit_of(dmask, v.cslot[off + j])) continue;
            const float w = v.cw[off + j];
            if (!(w > 0.f)) continue;
            cum += w;
            last = j + 1;
            if (opt < 0 && xk < cum) opt = j + 1;
          }
          if (opt < 0) opt = last < 0 ? 0 : last;
        }
      }
      int ns = -1;
      if (opt > 0) ns = v.cslot[off + opt - 1];
      if (opt != ref) {
        int rs = -1;
        if (ref > 0) {
          rs = v.cslot[off + ref - 1];
          long long e[DZ], q;
          pair_sums<DZ>(md, v, off + ref - 1, e, q);
          atomicSub(&acc_cnt[rs], 1);
#pragma unroll
          for (int d = 0; d < DZ; ++d)
            atomicAdd((unsigned long long*)&acc_se[d * T + rs], (unsigned long long)(-e[d]));
          atomicAdd((unsigned long long*)&acc_sq[rs], (unsigned long long)(-q));
          if (MAT) atomicAdd(&acc_hw[rs], (unsigned long long)(0ULL - wset_key(i)));
          touch(tmask, tlist, ntp, rs);
        } else {
          --my_dclut;
        }
        if (opt > 0) {
          long long e[DZ], q;
          pair_sums<DZ>(md, v, off + opt - 1, e, q);
          atomicAdd(&acc_cnt[ns], 1);
#pragma unroll
          for (int d = 0; d < DZ; ++d) atomicAdd((unsigned long long*)&acc_se[d * T + ns], (unsigned long long)e[d]);
          atomicAdd((unsigned long long*)&acc_sq[ns], (unsigned long long)q);
          if (MAT) atomicAdd(&acc_hw[ns], wset_key(i));
          touch(tmask, tlist, ntp, ns);
        } else {
          ++my_dclut;
        }
        hsh += row_key(i, opt > 0 ? ns + 1 : 0) - row_key(i, ref > 0 ? rs + 1 : 0);
      }
      if (MAT) put_theta(i, ns);
    }
  }
  group_sync(gsz, gid);
  // phase 3: rescore touched slots
  const int nt = *((volatile int*)ntp);
  long long my_delta = 0;
  int my_dninf = 0;
  for (int x = gl; x < nt; x += gsz) {
    const int t = tlist[x];
    int ninf;
    long long term;
    long long se[DZ];
    int m = 0;
    const bool is_dead = bit_of(dmask, t);
    if (is_dead) {
      term = dead_term(v.ct->log1mp[v.comp[t]], ninf);
    } else {
      m = v.mref[t] + acc_cnt[t];
#pragma unroll
      for (int d = 0; d < DZ; ++d) se[d] = v.seref[d * T + t] + acc_se[d * T + t];
      term = slot_term<DZ>(md, v, t, m, se, v.sqref[t] + acc_sq[t], ninf);
    }
    my_delta += term - v.termref[t];
    my_dninf += ninf - (int)v.ninfref[t];
    if (MAT && !is_dead)
      newval[t] = m >= 1 ? upd_insert<DZ>(a, v.comp[t], v.hwref[t] + acc_hw[t], m, se) : v.comp[t];
    acc_cnt[t] = 0;
#pragma unroll
    for (int d = 0; d < DZ; ++d) acc_se[d * T + t] = 0;
    acc_sq[t] = 0;
    if (MAT) acc_hw[t] = 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    my_delta += __shfl_xor_sync(0xFFFFFFFFu, my_delta, o);
    my_dninf += __shfl_xor_sync(0xFFFFFFFFu, my_dninf, o);
    my_dclut += __shfl_xor_sync(0xFFFFFFFFu, my_dclut, o);
    my_dead += __shfl_xor_sync(0xFFFFFFFFu, my_dead, o);
    hsh += __shfl_xor_sync(0xFFFFFFFFu, hsh, o);
  }
  bool any_bad = __any_sync(0xFFFFFFFFu, bad_row);
  if (gsz > 32 && !MAT) {
    // the group's totals (integers: the same whatever the order)
    if (lane == 0) {
      atomicAdd(&red[1], (unsigned long long)my_delta);
      atomicAdd(&red[2], (unsigned long long)(long long)my_dninf);
      atomicAdd(&red[3], (unsigned long long)(long long)my_dclut);
      atomicAdd(&red[4], (unsigned long long)(long long)my_dead);
      atomicAdd(&red[5], hsh);
      if (any_bad) atomicOr(&red[6], 1ull);
    }
    group_sync(gsz, gid);
    my_delta = (long long)red[1];
    my_dninf = (int)(long long)red[2];
    my_dclut = (int)(long long)red[3];
    my_dead = (int)(long long)red[4];
    hsh = red[5];
    any_bad = red[6] != 0ull;
  }
  group_sync(gsz, gid);
  if (MAT) {
    const uint32_t base = a.out_ptr[s_out];
    // four slots' reference components in flight
    for (int t0 = gl; t0 < T; t0 += 4 * gsz) {
      uint32_t ref4[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) ref4[u] = t0 + u * gsz < T ? v.refnew[t0 + u * gsz] : 0u;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int t = t0 + u * gsz;
        if (t >= T || bit_of(dmask, t)) continue;
        const uint32_t below = dpre[t >> 5] + __popc(dmask[t >> 5] & ((1u << (t & 31)) - 1u));
        const uint32_t val = bit_of(tmask, t) ? newval[t] : ref4[u];
        a.out_comp[base + (uint32_t)t - below] = val;
        if (!(val & kNewTag)) {   // an old component stays
          if (val < (uint32_t)a.fs->T) a.gc_flag[val] = 1u;
          else atomicOr(a.err, kErrChkRemap);
        }
      }
    }
    group_sync(gsz, gid);
  }
  for (int w = gl; w < W; w += gsz) { tmask[w] = 0; dmask[w] = 0; }
  if (GRP && gl < 8) red[gl] = 0ull;   // every reader has passed a barrier since
  if (gl == 0) {
    *ntp = 0;
    if (!MAT) {
      const long long score = sc.ref_score + my_delta + (md.kappa_zero ? 0LL : (long long)my_dclut * md.fx_log_kappa);
      const int ninf = sc.ninf_ref + my_dninf + (md.kappa_zero ? my_dclut : 0);
      const bool valid = !any_bad && ninf == 0;
      const size_t j = (size_t)h * HU + n;
      a.child_key[j] = valid ? score : kKeyInvalid;
      a.child_hash[j] = hsh;
      a.child_status[j] = valid ? 1 : 0;
      a.child_alive[j] = (uint16_t)(T - my_dead);
    }
  }
  group_sync(gsz, gid);
}

// Persistent over a list of children, one group of a.warp_group warps each
// (several when the children are few and long): the survivors (MAT), every
// child of every parent (a.warp_all), or the draw kernel's overflow (NOTES:
// after its noted children; an instantiation of its own, because the calls'
// stack costs the others 2 us a launch).
template <int DZ, bool MAT, bool GRP, bool NOTES>
__global__ void __launch_bounds__(512) warp_kernel(const __grid_constant__ ExpandArgs a) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char sm[];
  const Lay L = make_lay(DZ, a.T_max, a.K_max, a.M_plan);
  const WLay WL = make_wlay(DZ, MAT, a.T_max, GRP ? 1 : 0);
  // groups of a.warp_group warps per child, one work area each
  const int gsz = GRP ? 32 * a.warp_group : 32, groups = (int)blockDim.x / gsz;
  const int g = (int)threadIdx.x / gsz, gl = (int)threadIdx.x % gsz;
  const int HU = a.md.h_up, M = a.fs->M;
  const uint2 key = make_uint2(a.key_x, a.key_y);
  // a frame already abandoned (e.g. entries beyond capacity) writes
  // nothing; a failed table or staging leaves the images stale
  if (MAT && (*(volatile unsigned*)a.err & (kErrEntries | kErrSlots | kErrPairs))) return;
  if (!MAT && (*(volatile const unsigned*)a.err & kErrFatal)) return;
  const long long count = MAT ? (long long)*a.n_surv
                              : (a.warp_all ? (long long)a.fs->H * HU : (long long)*a.redo_count);
  if (NOTES) finish_notes<DZ>(a, L, key);
  // an empty list (the usual overflow case) costs no work-area set-up
  if ((long long)blockIdx.x * groups >= count) return;
  unsigned char* gb = sm + g * WL.total;
  {
    // the sums are indexed d * T + t with each parent's own T <= T_max
    const int Wm = (a.T_max + 31) / 32 + 1;
    int* acc_cnt = at<int>(gb, WL.cnt);
    long long* acc_se = at<long long>(gb, WL.se);
    long long* acc_sq = at<long long>(gb, WL.sq);
    unsigned long long* acc_hw = at<unsigned long long>(gb, WL.hw);
    for (int t = gl; t < a.T_max; t += gsz) {
      acc_cnt[t] = 0;
#pragma unroll
      for (int d = 0; d < DZ; ++d) acc_se[d * a.T_max + t] = 0;
      acc_sq[t] = 0;
      if (MAT) acc_hw[t] = 0;
    }
    for (int w = gl; w < Wm; w += gsz) {
      at<uint32_t>(gb, WL.tmask)[w] = 0;
      at<uint32_t>(gb, WL.dmask)[w] = 0;
    }
    if (gl == 0) *at<int>(gb, WL.nt) = 0;
    if (GRP && gl < 8) at<unsigned long long>(gb, WL.red)[gl] = 0ull;
    group_sync(gsz, g);
  }
  const long long nw = (long long)gridDim.x * groups;
  for (long long c = (long long)blockIdx.x * groups + g; c < count; c += nw) {
    const long long ci = MAT ? a.surv_idx[c] : (a.warp_all ? c : (long long)a.redo_list[c]);
    const int h = (int)(ci / HU), n = (int)(ci % HU);
    const View v = make_view(a.img + (size_t)h * a.img_stride, L, a.pt, a.ct);
    if (v.sc->bad) continue;
    warp_child<DZ, MAT, GRP>(a, v, v.sc->T, M, h, n, (int)c, key, gb, WL, gsz, g);
  }
}

// The reference association's updated components of every retained parent,
// requested once per parent: by one warp per first survivor of a parent, or,
// when the survivors are few, by as many warps as the launch has for each
// (a scene of 1000 objects keeps about 15 hypotheses of 1400 slots: 59 us
// with a warp per parent, a chain of 44 rounds of table requests; the
// regeneration stage with it and the cached reads went from 68 to 38 us).
template <int DZ>
__global__ void __launch_bounds__(256) mat_prep_kernel(const __grid_constant__ ExpandArgs a) {
  pdl_enter();
  const Lay L = make_lay(DZ, a.T_max, a.K_max, a.M_plan);
  const int lane = threadIdx.x & 31;
  const uint32_t HU = (uint32_t)a.md.h_up;
  // the kept-component flags the materialisation sets: cleared here over
  // the working table only (the next kernel waits for this one)
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < a.fs->T; c += gridDim.x * blockDim.x) a.gc_flag[c] = 0u;
  if (*(volatile unsigned*)a.err & (kErrEntries | kErrSlots | kErrPairs)) return;
  const uint32_t count = *a.n_surv;
  if (count == 0) return;
  const uint32_t nw = gridDim.x * (blockDim.x >> 5), w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  // warps per survivor, at most one per 32 slots
  const uint32_t parts = max(1u, min(nw / count, ((uint32_t)a.T_max + 31u) >> 5));
  auto parent_of = [&](uint32_t c) {
    const long long i = a.surv_idx[c];
    return (i >> 32) ? (uint32_t)(i / HU) : (uint32_t)i / HU;
  };
  for (uint32_t w = w0; w < count * parts; w += nw) {   // (parts > 1 only while count * parts <= nw)
    const uint32_t c = w / parts, part = w - c * parts;
    const uint32_t h = parent_of(c);
    if (c > 0 && parent_of(c - 1) == h) continue;
    unsigned char* img = a.img + (size_t)h * a.img_stride;
    const Scal& sc = *at<Scal>(img, L.scal);
    if (sc.bad) continue;
    const int T = sc.T;
    const int* mref = at<int>(img, L.mref);
    const uint32_t* comp = at<uint32_t>(img, L.comp);
    const long long* seref = at<long long>(img, L.seref);
    const unsigned long long* hwref = at<unsigned long long>(img, L.hwref);
    uint32_t* refnew = at<uint32_t>(img, L.refnew);
    for (int t = (int)part * 32 + lane; t < T; t += 32 * (int)parts) {
      long long se[DZ];
#pragma unroll
      for (int d = 0; d < DZ; ++d) se[d] = seref[d * T + t];
      refnew[t] = mref[t] >= 1 ? upd_insert<DZ>(a, comp[t], hwref[t], mref[t], se) : comp[t];
    }
  }
}

// Unique children of each parent (Section 3: only unique hypotheses are
// retained): a valid child whose key equals a lower valid draw's is a
// duplicate; its weight is dropped.  One block per parent: every valid child
// enters an open-addressing table in shared memory (key -> lowest draw).
// What bounds it is latency, one parent after another in a block: the next
// parent's children are read while this one's are entered, and two tables
// take turns, one cleared while the other is looked up (13 000 parents of
// 100 draws: 64 -> 29 us; 5000: 17 -> 11; 25: 6.2 -> 5.3).
__device__ __forceinline__ int dedup_table_size(int HU) {
  int ts = 64;
  while (ts < 2 * HU) ts <<= 1;
  return ts;
}

constexpr int kDedupThreads = 128;

__global__ void __launch_bounds__(kDedupThreads) dedup_kernel(const FrameDev* __restrict__ fs, int HU,
                                                              long long* child_key,
                                                              const unsigned long long* __restrict__ child_hash,
                                                              int8_t* child_status, const unsigned* err,
                                                              long long* part_max, double* part_sum,
                                                              unsigned* part_cnt, int tables) {
  pdl_enter();
  extern __shared__ unsigned long long s_k[];   // one or two tables: [ts] keys, 0 = empty, and [ts] lowest draws
  const int ts = dedup_table_size(HU);
  uint32_t* s_n = reinterpret_cast<uint32_t*>(s_k + tables * ts);
  __shared__ uint32_t s_zero[2];                             // lowest draw whose key is 0
  __shared__ long long s_pm[4];
  __shared__ double s_ps[4];
  __shared__ unsigned s_pc[4];
  const int tid = (int)threadIdx.x;
  auto clear = [&](int t) {
    for (int i = tid; i < ts; i += kDedupThreads) {
      s_k[t * ts + i] = 0ull;
      s_n[t * ts + i] = 0xFFFFFFFFu;
    }
    if (tid == 0) s_zero[t] = 0xFFFFFFFFu;
  };
  clear(0);
  const int H = fs->H;
  if (*(volatile const unsigned*)err & kErrFatal) return;   // the draws were skipped
  // a block beyond the parents (fixed launches are sized for the most
  // parents a frame can have) holds an empty partial; the selection reads
  // only the first H partials
  if (blockIdx.x >= H) return;
  LseAcc acc;   // this thread's unique children
  // a thread's first child of the parent at hand
  int8_t st = 0;
  unsigned long long hv = 0ull;
  long long key = 0;
  auto load = [&](int h) {
    st = 0;
    if (h < H && tid < HU) {
      const size_t j = (size_t)h * HU + tid;
      st = child_status[j];
      hv = child_hash[j];
      key = child_key[j];
    }
  };
  load(blockIdx.x);
  for (int h = blockIdx.x, t = 0; h < H; h += gridDim.x, t ^= tables - 1) {
    const size_t base = (size_t)h * HU;
    unsigned long long* tk = s_k + t * ts;
    uint32_t* tn = s_n + t * ts;
    const int8_t st0 = st;
    const unsigned long long hv0 = hv;
    const long long key0 = key;
    __syncthreads();   // this table is clear, the other one looked up
    if (tables == 1 && h != (int)blockIdx.x) {   // (very many draws: one table)
      clear(0);
      __syncthreads();
    }
    load(h + (int)gridDim.x);
    auto enter = [&](int n, unsigned long long v) -> uint32_t {   // the entry's place
      if (v == 0ull) {
        atomicMin(&s_zero[t], (uint32_t)n);
        return 0u;
      }
      uint32_t slot = (uint32_t)(v ^ (v >> 32)) & (uint32_t)(ts - 1);
      for (int probe = 0; probe < ts; ++probe) {   // ts > entries: a slot is found
        const unsigned long long prev = atomicCAS(&tk[slot], 0ull, v);
        if (prev == 0ull || prev == v) {
          atomicMin(&tn[slot], (uint32_t)n);
          break;
        }
        slot = (slot + 1u) & (uint32_t)(ts - 1);
      }
      return slot;
    };
    uint32_t slot0 = 0u;
    if (st0) slot0 = enter(tid, hv0);
    for (int n = tid + kDedupThreads; n < HU; n += kDedupThreads)
      if (child_status[base + n]) enter(n, child_hash[base + n]);
    __syncthreads();
    if (tables == 2) clear(t ^ 1);
    auto settle = [&](int n, uint32_t low, long long k) {
      if (low < (uint32_t)n) {
        child_status[base + n] = 2;
        child_key[base + n] = kKeyInvalid;
      } else {
        acc.add(k);
      }
    };
    if (st0) settle(tid, hv0 == 0ull ? s_zero[t] : tn[slot0], key0);
    for (int n = tid + kDedupThreads; n < HU; n += kDedupThreads) {
      if (child_status[base + n] == 0) continue;
      const unsigned long long v = child_hash[base + n];
      uint32_t low = s_zero[t];
      if (v != 0ull) {
        uint32_t slot = (uint32_t)(v ^ (v >> 32)) & (uint32_t)(ts - 1);
        for (int probe = 0; probe < ts && tk[slot] != v; ++probe) slot = (slot + 1u) & (uint32_t)(ts - 1);
        low = tn[slot];
      }
      settle(n, low, child_key[base + n]);
    }
  }
  // the block's partial: maximum, sum rescaled to it (FP64), count
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  long long M = acc.m;
  unsigned c = acc.n;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    M = max(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
    c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
  }
  if (lane == 0) {
    s_pm[wp] = M;
    s_pc[wp] = c;
  }
  __syncthreads();
  M = s_pm[0];
  c = s_pc[0];
  for (int w = 1; w < nw; ++w) {
    M = max(M, s_pm[w]);
    c += s_pc[w];
  }
  double r = lse_rescale(acc.m, acc.sum(), M);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, o);
  if (lane == 0) s_ps[wp] = r;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += s_ps[w];
    part_max[blockIdx.x] = M;
    part_sum[blockIdx.x] = t;
    part_cnt[blockIdx.x] = c;
  }
}

void launch_dedup(const FrameDev* fs, int HU, long long* child_key, const unsigned long long* child_hash,
                  int8_t* child_status, const unsigned* err, const PruneWork& w, int grid, cudaStream_t s) {
  int ts = 64;
  while (ts < 2 * HU) ts <<= 1;
  const int tables = 2 * ts * 12 <= 96 * 1024 ? 2 : 1;   // (8192 draws: 196 KB a table)
  const int smem = tables * ts * 12;
  launch_k(dedup_kernel, std::min(grid, kMaxLseParts), kDedupThreads, smem, s, fs, HU, child_key, child_hash, child_status,
           err, w.part_max, w.part_sum, w.part_cnt, tables);
}

// ---- host side ----
using KernelFn = void (*)(const ExpandArgs);

static KernelFn stage_fn(int dz, bool smem, bool wide) {
  if (wide) return dz == 2 ? stage_kernel<2, false, true> : stage_kernel<3, false, true>;
  if (dz == 2) return smem ? stage_kernel<2, true, false> : stage_kernel<2, false, false>;
  return smem ? stage_kernel<3, true, false> : stage_kernel<3, false, false>;
}
static KernelFn draw_fn(int dz, bool staged) {
  if (dz == 2) return staged ? draw_kernel<2, true> : draw_kernel<2, false>;
  return staged ? draw_kernel<3, true> : draw_kernel<3, false>;
}
static KernelFn warp_fn(int dz, bool mat, bool grp = false, bool notes = false) {
  if (notes) return dz == 2 ? warp_kernel<2, false, false, true> : warp_kernel<3, false, false, true>;
  if (grp) {
    if (dz == 2) return mat ? warp_kernel<2, true, true, false> : warp_kernel<2, false, true, false>;
    return mat ? warp_kernel<3, true, true, false> : warp_kernel<3, false, true, false>;
  }
  if (dz == 2) return mat ? warp_kernel<2, true, false, false> : warp_kernel<2, false, false, false>;
  return mat ? warp_kernel<3, true, false, false> : warp_kernel<3, false, false, false>;
}
static KernelFn prep_fn(int dz) { return dz == 2 ? mat_prep_kernel<2> : mat_prep_kernel<3>; }

void expand_init(int smem_limit) {
  opt_in_smem(dedup_kernel, smem_limit);
  for (int dz = 2; dz <= 3; ++dz) {
    cudaFuncSetAttribute(stage_fn(dz, true, false), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    for (int wide = 0; wide < 2; ++wide)
      cudaFuncSetAttribute(stage_fn(dz, false, wide), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    for (int st = 0; st < 2; ++st)
      cudaFuncSetAttribute(draw_fn(dz, st), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    cudaFuncSetAttribute(warp_fn(dz, false, false, true), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    for (int grp = 0; grp < 2; ++grp) {
      cudaFuncSetAttribute(warp_fn(dz, false, grp), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
      cudaFuncSetAttribute(warp_fn(dz, true, grp), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit);
    }
  }
}

static KernelFn kernel_of(const ExpandArgs& a, ExpandKernel k) {
  switch (k) {
    case ExpandKernel::kStage: return stage_fn(a.md.dz, a.stage_smem != 0, a.stage_wide != 0);
    case ExpandKernel::kDraw: return draw_fn(a.md.dz, a.draw_staged != 0);
    case ExpandKernel::kWarp: return warp_fn(a.md.dz, a.materialize != 0, a.warp_group > 1, !a.materialize && !a.warp_all);
    default: return prep_fn(a.md.dz);
  }
}

int expand_occupancy(const ExpandArgs& a, ExpandKernel k, int threads, int smem) {
  int per_sm = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel_of(a, k), threads, smem);
  return e == cudaSuccess ? per_sm : 0;
}

void launch_expand_kernel(const ExpandArgs& a, ExpandKernel k, int grid, int threads, int smem,
                          cudaStream_t s) {
  if (grid <= 0) return;
  launch_k(kernel_of(a, k), grid, threads, smem, s, a);
}

int expand_warp_best_cta(int dz, int materialize, int T, int max_warps, int smem_limit) {
  static std::mutex mu;
  static std::map<std::tuple<int, int, int, int, int>, int> memo;
  const auto key = std::make_tuple(dz, materialize, T, max_warps, smem_limit);
  std::lock_guard<std::mutex> lock(mu);
  auto it = memo.find(key);
  if (it != memo.end()) return it->second;
  int best = 0, best_res = 0;
  for (int g = 1; g <= max_warps; ++g) {
    const int smem = expand_warp_smem(dz, materialize, T, g, 0);
    if (smem > smem_limit) break;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, warp_fn(dz, materialize != 0), 32 * g, smem) !=
        cudaSuccess)
      per_sm = 0;
    if (per_sm * g >= best_res && per_sm > 0) {   // ties: the larger CTA
      best_res = per_sm * g;
      best = g;
    }
  }
  cudaGetLastError();
  memo[key] = best;
  return best;
}

bool expand_kernel_takes_key(const void* fn) {
  for (int dz = 2; dz <= 3; ++dz)
    if (fn == (const void*)draw_fn(dz, false) || fn == (const void*)draw_fn(dz, true) ||
         fn == (const void*)warp_fn(dz, false, false, true) || fn == (const void*)warp_fn(dz, false) ||
         fn == (const void*)warp_fn(dz, true) ||
        fn == (const void*)warp_fn(dz, false, true) || fn == (const void*)warp_fn(dz, true, true))
      return true;
  return false;
}

}  // namespace glmb
