// The cell test of the bucket path for models without warp or grid barriers:
// every bucket's cells are decided in shared memory, without sorting the
// bucket's keys.
//
// A cell is racy iff it has a write and either two blocks meet in it or, inside
// one block, some barrier interval holds two threads and a write (the
// cell-level form of the pair rule in include/rc.h).  Every cell of a bucket has
// its own slot of a table in shared memory (the slot is the rest of the cell
// hash below the bucket bits, so equal slots are equal cells), and a key's low
// word holds its interval, block, thread and kind:
//   1. every write stores its low word in its cell's slot; whichever store wins
//      is the cell's representative write;
//   2. every key compares itself with the representative.  Another block, or
//      another thread in the representative's interval: the cell is racy.
//      Another thread in another interval: the cell has two threads.  A write in
//      another interval: the cell has writes in two intervals.
//      A cell that is not racy by now races only if both marks are there (with
//      one write interval the representative stands for it, and every key was
//      compared with it): few cells in practice;
//   3. these candidate cells are numbered, and 1 and 2 are done again per
//      (candidate cell, barrier interval): a key that finds another thread's
//      write in its own interval makes the cell racy.
// A representative decides exactly: if an interval (or cell) has a write and two
// threads (or blocks), at least one of its keys differs from whichever write
// was kept.  Which store wins does not matter, so the stores need no order.
//
// With atomics (AT; a 2-bit kind field) a conflict is a write, or an atomic and a
// plain read.  The representative is then any write or atomic of the cell, and
// beside the marks for blocks, threads and intervals the cell keeps whether it
// has a write and a plain read, in all and in the representative's interval: two
// blocks or threads meet in a conflict iff there is a write, or a read beside the
// atomic (two threads among the atomics and reads of a group that holds both
// always make an atomic and a read of different threads).
//
// What bounds it: one read of every key (8 bytes); about 78 warp instructions per
// 32 keys keep the issue slots 76 % busy.  On the 4096 x 256 random affine model
// with a key per point (578 M keys, 2^17 buckets of 4,400 keys) 1.35 ms, where the
// counting sort of every bucket and the cell scan that it replaces there took
// 3.52 + 1.66 ms; on 49 M keys with hot cells 0.26 ms against 1.63 + 0.22 ms.  (With
// a key per distinct point: 303 M keys in 0.94 ms.)  Blocks of 256 threads with 20
// keys each in registers, 4 per SM, were the fastest split without spills (512
// threads, 2 per SM: 1.95 ms; 384 threads with 16 keys, 3 per SM: 1.51 ms): the
// barriers between the steps stall fewer warps.  The hashed table (HT) takes 3
// blocks per SM; on 2,000 small models in one batch (34 cell bits, some 28 M kept
// keys) the check takes 1.99 ms with it, 2.62 ms with the local sort and scan.
#include <cuda_runtime.h>

#include "fold.cuh"
#include "kernels.h"

namespace rc {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kFltThreads = 256;
constexpr int kFltBlocks = 4;                      // blocks per SM
constexpr int kFltKPT = 20;                        // keys per thread held in registers
constexpr int kFltStreamKPT = 12;                  // keys per thread and step of a larger bucket
constexpr unsigned kFltCap = kFltThreads * kFltKPT;
static_assert((1 << kFilterMaxSlotBits) / 32 <= kFltThreads, "a word of a bit mask per thread");
static_assert(kFltCap < (1 << kFilterMaxSlotBits), "a bucket in registers leaves free slots in a hashed table");
constexpr unsigned kNoTag = 0xffffffffu;           // (tags have at most 31 bits)
constexpr unsigned kTagMul = 0x9E3779B1u;          // home slot of a tag (Fibonacci hashing: its low bits alone
                                                   // are those of the cell's low bits, equal for equal strides)
constexpr unsigned kPartMul = 0x85EBCA77u;         // part of a tag (odd: 32 part bits tell all tags apart)

// inverse of the odd hash multiplier modulo 2^64 (Newton's iteration: each step
// doubles the number of correct low bits)
constexpr uint64_t hash_inverse() {
  uint64_t x = kCellHashMul;   // correct to 3 bits
  for (int i = 0; i < 5; ++i) x *= 2ull - kCellHashMul * x;
  return x;
}
static_assert(hash_inverse() * kCellHashMul == 1ull, "inverse of the cell hash multiplier");

// Words of a table.  Direct (r <= kFilterMaxSlotBits): the slot is the cell's r
// hash bits.  At least 4096, and up to 2^kFilterMaxSlotBits where every cell's
// intervals (two 16-bit entries of step 3 a word) would fill them: with half as many
// a tile buffer of 42 M keys in one-pass buckets took 0.38 ms instead of 0.33.
// Hashed (HT, larger r): 2^kFilterMaxSlotBits slots with a tag.
unsigned table_words(uint32_t r, uint32_t phase_bits) {
  const uint32_t bits = r + phase_bits > 13u ? r + phase_bits - 1u : 12u;
  return 1u << (bits > kFilterMaxSlotBits || r > kFilterMaxSlotBits ? kFilterMaxSlotBits : bits > r ? bits : r);
}
__host__ __device__ __forceinline__ unsigned mask_words(uint32_t r) {
  return r < 5 ? 1u : r > kFilterMaxSlotBits ? 1u << (kFilterMaxSlotBits - 5) : 1u << (r - 5);
}
// (four words behind the table: the slot of padding keys and of cells without a write)
size_t filter_smem(uint32_t r, uint32_t phase_bits, bool at) {
  const size_t tw = table_words(r, phase_bits), mw = mask_words(r);
  return (tw + 4 + (r > kFilterMaxSlotBits ? tw : 0) + (at ? 10 : 5) * mw + 1 + (at ? 3 * (2 * tw / 32) : 0)) *
         sizeof(unsigned);
}

// One block per bucket.  A bucket of at most kFltCap keys is held in registers
// as (low word, slot); a larger one is read again in every step.  Key slots of
// a thread past the bucket's end repeat its first key (the same instance, which
// changes nothing), so no step tests for them; PAD: the bucket holds padding
// keys (the unpartitioned single bucket), held as reads of the word behind the table.
// HT: the cell space is too sparse for a slot per cell.  The written cells take
// slots of an open-addressed table (the cell's r hash bits are its tag), and
// every key looks its cell up: not found, it has no write and cannot race.  A
// bucket in registers has fewer keys than the table has slots.  A larger one may
// hold more written cells: where the table runs out, its cells are taken in
// halves, quarters and so on by another hash of the tag.
template <bool PAD, bool REGS, bool AT, bool HT>
__device__ __forceinline__ void filter_bucket(const FilterArgs& a, const uint64_t* src, uint64_t len) {
  extern __shared__ __align__(16) unsigned s_tab[];
  const unsigned tw = a.tw, mw = mask_words(a.r);
  unsigned* s_tag = s_tab + tw + 4;     // (HT) the cell of every slot
  unsigned* s_two = s_tag + (HT ? tw : 0u);   // cells with two threads of a block, a bit per slot
  unsigned* s_wi = s_two + mw;          // cells with writes in two intervals, then the candidate cells
  unsigned* s_racy = s_wi + mw;         // racy cells
  unsigned* s_hot = s_racy + mw;        // racy candidate cells, a bit per candidate
  unsigned* s_rank = s_hot + mw + 1;    // candidate cells before each word of s_wi
  // with atomics: cells with two threads in the representative's interval, with a
  // write, with a read, and with those in its interval; the same three per entry
  unsigned* s_g = s_rank + mw;
  unsigned* s_w = s_g + mw;
  unsigned* s_r = s_w + mw;
  unsigned* s_wp = s_r + mw;
  unsigned* s_rp = s_wp + mw;
  unsigned* s_e2 = s_rp + mw;
  unsigned* s_ew = s_e2 + 2 * tw / 32;
  unsigned* s_er = s_ew + 2 * tw / 32;
  __shared__ unsigned s_wsum[kFltThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t pb = a.s.phase_bits, bb = a.s.block_bits, tb = a.s.thread_bits;
  // a low word's fields: kind (R = 0, W = 1, A = 2), (block, thread), block, interval
  constexpr unsigned kb = AT ? 2u : 1u, kmask = AT ? 3u : 1u;
  const unsigned m_bt = (unsigned)(((1ull << (bb + tb)) - 1ull) << kb),
                 m_b = (unsigned)(((1ull << bb) - 1ull) << (kb + tb)),
                 m_p = (unsigned)(((1ull << pb) - 1ull) << (kb + tb + bb));
  const uint32_t cs = a.s.cell_shift;
  const unsigned smask = (1u << a.r) - 1u;   // (r <= 31)
  uint32_t part_bits = 0, part = 0;          // (HT, not REGS) the part of the bucket's cells in hand
  const unsigned lmask = cs < 32 ? (1u << cs) - 1u : ~0u;
  // low word and slot (HT: tag) of a key (the low r bits of the hash depend on the
  // low bits of the cell alone)
  auto unpack = [&](uint64_t k, unsigned& kl, unsigned& sl) {
    kl = (uint32_t)k & lmask;
    sl = (__funnelshift_rc((uint32_t)k, (uint32_t)(k >> 32), cs) * (uint32_t)kCellHashMul) & smask;
    if (PAD && k == kSentinel) {
      sl = HT ? kNoTag : tw;
      kl = 0;
    }
  };
  // the slot of a cell, or tw if it has none
  constexpr unsigned kProbes = REGS ? (1u << kFilterMaxSlotBits) : 512u;
  auto find = [&](unsigned tag) -> unsigned {
    unsigned i = (tag * kTagMul) >> (32 - kFilterMaxSlotBits);
    for (unsigned n = 0; n < kProbes; ++n, i = (i + 1u) & (tw - 1u)) {
      const unsigned t = s_tag[i];
      if (t == tag) return i;
      if (t == kNoTag) break;
    }
    return tw;
  };
  auto in_part = [&](unsigned tag) { return part_bits == 0u || (tag * kPartMul) >> (32u - part_bits) == part; };
  unsigned rl[kFltKPT], rs[kFltKPT];   // (REGS) the bucket
  const int nq = REGS ? (int)((len + kFltThreads - 1) / kFltThreads) : 0;
  if constexpr (REGS) {
    const uint64_t* p = src + tid;
    uint64_t k[kFltKPT];
    const uint64_t k0 = __ldg(src);
#pragma unroll
    for (int q = 0; q < kFltKPT; ++q) {
      if (q >= nq) break;
      k[q] = k0;
      if (q < nq - 1 || (unsigned)(q * kFltThreads + tid) < (unsigned)len) k[q] = __ldg(p + q * kFltThreads);
    }
#pragma unroll
    for (int q = 0; q < kFltKPT; ++q) {
      if (q >= nq) break;
      unpack(k[q], rl[q], rs[q]);
    }
  }
  bool resolve = false;   // (HT, not REGS) whether the written cells have their slots
  // f(low word, slot) for the keys of the bucket
  auto each = [&](auto&& f) {
    if constexpr (REGS) {
#pragma unroll
      for (int q = 0; q < kFltKPT; ++q) {
        if (q >= nq) break;
        // (opaque to the compiler, which would keep what it derives from the pair in
        // one step for the next one and run out of registers)
        asm volatile("" : "+r"(rl[q]), "+r"(rs[q]));
        f(rl[q], rs[q]);
      }
    } else {
      const uint64_t k0 = __ldg(src);
      for (uint64_t i = tid; i < len; i += kFltStreamKPT * kFltThreads) {
        uint64_t k[kFltStreamKPT];
#pragma unroll
        for (int u = 0; u < kFltStreamKPT; ++u)
          k[u] = i + u * kFltThreads < len ? __ldg(src + i + u * kFltThreads) : k0;
#pragma unroll
        for (int u = 0; u < kFltStreamKPT; ++u) {
          unsigned kl, sl;
          unpack(k[u], kl, sl);
          if constexpr (HT) {
            if (!in_part(sl)) continue;
            if (resolve) sl = find(sl);
          }
          f(kl, sl);
        }
      }
    }
  };
  auto clear_table = [&](unsigned words) {
    for (unsigned i = 4 * tid; i < words; i += 4 * kFltThreads)
      *reinterpret_cast<uint4*>(s_tab + i) = make_uint4(0, 0, 0, 0);
  };
  auto mark = [&](unsigned* bits, unsigned i) {
    const unsigned bit = 1u << (i & 31u);
    if (!(bits[i >> 5] & bit)) atomicOr(&bits[i >> 5], bit);
  };
  // one test of the bucket's cells (HT: of those in hand); false: the table ran out
  auto test = [&]() -> bool {
  resolve = false;
  // (the slots rounded up to whole 16-byte stores lie inside the table)
  clear_table(PAD || HT ? tw + 4u : ((1u << a.r) + 3u) & ~3u);
  if constexpr (HT)
    for (unsigned i = 4 * tid; i < tw; i += 4 * kFltThreads)
      *reinterpret_cast<uint4*>(s_tag + i) = make_uint4(kNoTag, kNoTag, kNoTag, kNoTag);
  for (unsigned i = tid; i < (AT ? 10 : 4) * mw + 1; i += kFltThreads) s_two[i] = 0;
  __syncthreads();
  bool any = false;
  if constexpr (HT) {
    // 1. a slot for every written cell and its representative (in one reading of a
    // larger bucket), then, when all have one, every key's slot
    bool full = false;
    each([&](unsigned k, unsigned tag) {
      if ((k & kmask) == 0u) return;
      unsigned i = (tag * kTagMul) >> (32 - kFilterMaxSlotBits), n = 0;
      for (; n < kProbes; ++n, i = (i + 1u) & (tw - 1u)) {
        unsigned t = s_tag[i];
        if (t == kNoTag) t = atomicCAS(&s_tag[i], kNoTag, tag);
        if (t == kNoTag || t == tag) break;
      }
      if (n == kProbes) {
        full = true;
        return;
      }
      s_tab[i] = k;
      any = true;
    });
    if constexpr (!REGS)
      if (__syncthreads_or(full)) return false;
    resolve = true;
  } else {
    // 1. the representative of every written cell (its low word is not 0)
    each([&](unsigned k, unsigned s) {
      if (k & kmask) {
        s_tab[s] = k;
        any = true;
      }
    });
  }
  if (!__syncthreads_or(any)) return true;   // no write: nothing can race
  if constexpr (HT && REGS) {
#pragma unroll
    for (int q = 0; q < kFltKPT; ++q) {
      if (q >= nq) break;
      rs[q] = find(rs[q]);
    }
  }
  // 2. every key against its cell's representative
  any = false;
  each([&](unsigned k, unsigned s) {
    const unsigned rep = s_tab[s];
    const unsigned d = rep ^ k;
    if constexpr (AT) {
      if (rep == 0u) return;
      const unsigned kind = k & kmask;
      if (kind != 2u) mark(kind ? s_w : s_r, s);
      any = any || (d & m_bt) != 0u;
      if (d & m_b) {
        mark(s_racy, s);   // (two blocks: racy if the cell has a conflict)
      } else if (d & m_p) {
        if (d & m_bt) mark(s_two, s);
        if (kind) mark(s_wi, s);
      } else {
        if (d & m_bt) mark(s_g, s);
        if (kind != 2u) mark(kind ? s_wp : s_rp, s);
      }
    } else if (rep != 0u && (d & ((k & 1u) ? m_bt | m_p : m_bt)) != 0u) {
      any = true;
      if (d & m_bt) mark((d & m_b) || !(d & m_p) ? s_racy : s_two, s);
      if ((k & 1u) && (d & m_p)) mark(s_wi, s);
    }
  });
  if (!__syncthreads_or(any)) return true;   // every written cell has one thread and interval
  // 3. the candidate cells numbered in slot order; at most one word of a bit
  // mask per thread
  unsigned cand = 0;
  if (tid < (int)mw) {
    if constexpr (AT) {
      const unsigned conf = s_w[tid] | s_r[tid];
      const unsigned racy = (s_racy[tid] & conf) | (s_g[tid] & (s_wp[tid] | s_rp[tid]));
      s_racy[tid] = racy;
      cand = s_wi[tid] & (s_two[tid] | s_g[tid]) & conf & ~racy;
    } else {
      cand = s_two[tid] & s_wi[tid] & ~s_racy[tid];
    }
    s_wi[tid] = cand;
  }
  if (__syncthreads_or(cand != 0u)) {
    const unsigned c = __popc(cand);
    unsigned x = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(FULL, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_wsum[w] = x;
    __syncthreads();
    unsigned before = 0, ncand = 0;
#pragma unroll 4
    for (int i = 0; i < kFltThreads / 32; ++i) {
      if (i < w) before += s_wsum[i];
      ncand += s_wsum[i];
    }
    if (tid < (int)mw) s_rank[tid] = before + x - c;
    __syncthreads();
    // the entry (candidate << pb | interval) of a key, ~0 if its cell is no candidate
    auto entry = [&](unsigned k, unsigned s) -> unsigned {
      if ((PAD || HT) && s == tw) return ~0u;
      const unsigned m = s_wi[s >> 5];
      if (!((m >> (s & 31u)) & 1u)) return ~0u;
      return ((s_rank[s >> 5] + __popc(m & ((1u << (s & 31u)) - 1u))) << pb) | (unsigned)((uint64_t)k >> (kb + bb + tb));
    };
    // Windows of the table; the bucket is read twice for each.  All keys of a candidate
    // lie in one block (a key of another block has decided its cell), so where a larger
    // bucket is read from memory an entry holds the thread of a write alone, in 16 bits
    // if it fits: half as many windows.  (A bucket in registers costs no reads.)
    const bool half = !REGS && tb <= kFilterHalfThreadBits;
    unsigned short* s_tab16 = reinterpret_cast<unsigned short*>(s_tab);
    const unsigned tmask = (1u << tb) - 1u;   // (a block has at most 2^20 threads)
    auto thread_of = [&](unsigned k) { return (((k >> kb) & tmask) << 1) | 1u; };
    const unsigned room = half ? 2u * tw : tw;
    for (unsigned e0 = 0; e0 < (ncand << pb); e0 += room) {
      const unsigned used = min(room, (ncand << pb) - e0);
      clear_table(((half ? (used + 1u) / 2u : used) + 3u) & ~3u);
      if constexpr (AT)
        for (unsigned i = tid; i < 3 * (2 * tw / 32); i += kFltThreads) s_e2[i] = 0;
      __syncthreads();
      each([&](unsigned k, unsigned s) {
        if (k & kmask) {
          const unsigned e = entry(k, s) - e0;
          if (e < used) {
            if (half) s_tab16[e] = (unsigned short)thread_of(k);
            else s_tab[e] = k;
          }
        }
      });
      __syncthreads();
      each([&](unsigned k, unsigned s) {
        const unsigned e = entry(k, s) - e0;
        if (e < used) {
          const unsigned rep = half ? s_tab16[e] : s_tab[e];
          const bool other = half ? rep != thread_of(k) : ((rep ^ k) & m_bt) != 0u;
          if constexpr (AT) {
            if (rep == 0u) return;
            if (other) mark(s_e2, e);
            if ((k & kmask) != 2u) mark(k & kmask ? s_ew : s_er, e);
          } else {
            if (rep != 0u && other) mark(s_hot, (e + e0) >> pb);
          }
        }
      });
      __syncthreads();
      if constexpr (AT) {
        for (unsigned i = tid; 32 * i < used; i += kFltThreads)
          for (unsigned m = s_e2[i] & (s_ew[i] | s_er[i]); m; m &= m - 1u)
            mark(s_hot, (32 * i + (unsigned)__ffs(m) - 1u + e0) >> pb);
        __syncthreads();
      }
    }
  }
  // the racy cells: counted, and the smallest by value kept.  Slot s of bucket b
  // (HT: its tag) has hash (part | b | s), whose cell is hash * inverse mod 2^(cell bits).
  const uint64_t inv = hash_inverse();
  unsigned count = 0;
  unsigned long long first = ~0ull;
  if (tid < (int)mw) {
    unsigned m = s_racy[tid];
    if (cand) {
      // the racing candidates of this word back to their slots
      const unsigned r0 = s_rank[tid];
      unsigned hot = __funnelshift_r(s_hot[r0 >> 5], s_hot[(r0 >> 5) + 1], r0 & 31u);
      for (unsigned c = cand; c && hot; c &= c - 1u, hot >>= 1)
        if (hot & 1u) m |= c & (0u - c);
    }
    count = __popc(m);
    while (m) {
      const unsigned slot = 32u * tid + (unsigned)__ffs(m) - 1u;
      m &= m - 1u;
      const uint64_t h = a.part_hash | ((uint64_t)blockIdx.x << a.r) | (HT ? s_tag[slot] : slot);
      const uint64_t cell = (h * inv) & a.hmask;
      if (a.s.n_models) {
        DevResult* r = result_of(a.s, cell);
        atomicAdd(&r->racy_cells, 1ull);
        atomicMin(&r->hash_cell, (unsigned long long)cell);
      } else {
        first = min(first, (unsigned long long)cell);
      }
    }
  }
  if (a.s.n_models) return true;
  count = __reduce_add_sync(FULL, count);
  if (count == 0) return true;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) first = min(first, __shfl_xor_sync(FULL, first, o));
  if (lane == 0) {
    atomicAdd(&a.s.res->racy_cells, (unsigned long long)count);
    atomicMin(&a.s.res->hash_cell, first);
  }
  return true;
  };
  if constexpr (REGS || !HT) {
    test();
  } else {
    // the parts (part_bits, part) in order; one that is too large is halved
    do {
      if (!test()) {
        ++part_bits;
        part *= 2u;
      } else {
        ++part;
        while (part_bits != 0u && (part & 1u) == 0u) {
          part >>= 1;
          --part_bits;
        }
      }
      __syncthreads();
    } while (part_bits != 0u || part == 0u);
  }
}

template <bool PAD, bool AT, bool HT>
__global__ void __launch_bounds__(kFltThreads, HT ? 3 : kFltBlocks) bucket_filter_kernel(FilterArgs a) {
  const uint64_t lo = a.boff[blockIdx.x], hi = a.boff[blockIdx.x + 1];
  if (hi < lo + 2) return;              // a race needs two keys
  if (hi - lo <= (uint64_t)kFltCap) filter_bucket<PAD, true, AT, HT>(a, a.keys_in + lo, hi - lo);
  else filter_bucket<PAD, false, AT, HT>(a, a.keys_in + lo, hi - lo);
}

template <bool PAD, bool AT, bool HT>
cudaError_t launch_filter(const FilterArgs& a, uint32_t D, cudaStream_t st) {
  const cudaError_t e = ensure_kernel_smem(reinterpret_cast<const void*>(bucket_filter_kernel<PAD, AT, HT>),
                                           filter_smem(HT ? 31 : kFilterMaxSlotBits, 0, AT));
  if (e != cudaSuccess) return e;
  bucket_filter_kernel<PAD, AT, HT><<<1u << D, kFltThreads, filter_smem(a.r, a.s.phase_bits, AT), st>>>(a);
  return cudaGetLastError();
}
template <bool PAD>
cudaError_t launch_filter(const FilterArgs& a, uint32_t D, cudaStream_t st) {
  const bool at = a.s.thread_shift == 2;
  if (a.r > kFilterMaxSlotBits)
    return at ? launch_filter<PAD, true, true>(a, D, st) : launch_filter<PAD, false, true>(a, D, st);
  return at ? launch_filter<PAD, true, false>(a, D, st) : launch_filter<PAD, false, false>(a, D, st);
}

}  // namespace

cudaError_t launch_bucket_filter(const FilterArgs& args, uint32_t D, cudaStream_t st) {
  FilterArgs a = args;
  a.tw = table_words(a.r, a.s.phase_bits);
  if (a.r > kFilterMaxTagBits || a.s.cell_shift > kFilterMaxLowBits) return cudaErrorInvalidValue;
  // an unpartitioned bucket holds padding keys, which take the word behind the table
  return D == 0 ? launch_filter<true>(a, D, st) : launch_filter<false>(a, D, st);
}

}  // namespace rc
