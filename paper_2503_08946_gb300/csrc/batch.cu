// Batched check: many models in one pipeline.
//
// The models of a batch are checked together instead of one pipeline per
// model.  Every model keeps its own lowered program; the batch gives each model
// its own range of cells, so that the keys of all models can be sorted and
// scanned as one array:
//
//   batch key = [model's first batch cell + cell | phase | block | thread | kind]
//
// with the phase, block and thread fields as wide as the widest model's.  A
// racy cell of the shared scan is charged to the model whose cell range holds
// it, and the witness kernels run once per model (blockIdx.y), on the first
// racy cell of that model.  Models whose combined fields would not fit in 63
// bits go to separate packs, each checked by its own pipeline in turn.
//
// Expansion is one persistent kernel over a work queue: a unit is (model,
// chunk of kExpandThreads threads) with all the model's statements, and blocks
// take units in groups from an atomic counter until the queue is empty.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>

#include "expand_core.cuh"
#include "kernels.h"

namespace rc {

namespace {

constexpr int kUnitsPerGrab = 16;
static_assert(kExpandThreadsHost == kExpandThreads, "host and device chunk sizes agree");

// Keys are re-packed from the model's layout into the batch layout.
struct BatchSink {
  uint64_t* keys;
  uint64_t cell_base;
  uint32_t mcs, mps, mbs, mts;       // model field shifts (thread field at mts = its kind bits)
  uint64_t pm, bm, tm;               // model field masks
  uint32_t bcs, bps, bbs, bts;       // batch field shifts
  __device__ __forceinline__ void put(uint64_t i, uint64_t key, uint64_t) {
    if (key != kSentinel) {
      const uint64_t cell = key >> mcs;
      const uint64_t ph = (key >> mps) & pm, b = (key >> mbs) & bm, t = (key >> mts) & tm;
      key = ((cell_base + cell) << bcs) | (ph << bps) | (b << bbs) | (t << bts) | (key & ((1ull << mts) - 1ull));
    }
    keys[i] = key;
  }
  __device__ __forceinline__ void pad(uint64_t i) { keys[i] = kSentinel; }
};

// LF: every statement of the pack is loop-free -- only the one-point
// expansion is compiled (fewer registers, no row cache: more resident warps)
template <bool LF>
__global__ void __launch_bounds__(kExpandThreads, LF ? 6 : 4) batch_expand_kernel(BatchArgs a) {
  __shared__ int64_t s_tval[kMaxTerms * kExpandThreads];
  __shared__ int64_t s_cache[LF ? 1 : kFastCache * kExpandThreads];
  __shared__ unsigned long long s_u;
  __shared__ uint32_t s_model;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      s_u = atomicAdd(a.queue, (unsigned long long)a.grab);
      // the model of the grab's first unit (binary search once per grab)
      uint32_t lo = 0, hi = a.n_models;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.models[mid].unit_base <= s_u) lo = mid;
        else hi = mid;
      }
      s_model = lo;
    }
    __syncthreads();
    const uint64_t u0 = s_u;
    if (u0 >= a.n_units) break;
    const uint64_t u1 = min(a.n_units, u0 + a.grab);
    for (uint64_t u = u0; u < u1; ++u) {
      // the model of unit u: the grab's units are consecutive, so step forward
      if (threadIdx.x == 0) {
        uint32_t m = s_model;
        while (m + 1 < a.n_models && a.models[m + 1].unit_base <= u) ++m;
        s_model = m;
      }
      __syncthreads();
      const uint32_t lo = s_model;
      const BatchModel& B = a.models[lo];
      // one unit = one chunk of kExpandThreads threads of the model, all its statements
      const uint64_t g = (u - B.unit_base) * kExpandThreads + threadIdx.x;
      const DevModel& M = *B.dm;
      DevResult* res = a.res + lo;
      unsigned long long count = 0;
      if (g < B.n_threads) {
        BatchSink sink;
        sink.keys = a.keys + B.key_base;
        sink.cell_base = B.cell_base;
        sink.mcs = B.cell_shift;
        sink.mps = B.phase_shift;
        sink.mbs = B.block_shift;
        sink.mts = B.thread_shift;
        sink.pm = (1ull << B.phase_bits) - 1;
        sink.bm = (1ull << B.block_bits) - 1;
        sink.tm = (1ull << B.thread_bits) - 1;
        sink.bcs = a.cell_shift;
        sink.bps = a.phase_shift;
        sink.bbs = a.block_shift;
        sink.bts = a.thread_shift;
        const ThreadVars tv = thread_vars(M, g);
        for (uint32_t s = 0; s < B.n_stmts; ++s) {
          const DevStmt& S = M.stmts[s];
          if (LF) {
            FastCtx c;
            c.M = B.dm;
            c.S = &S;
            c.tv = tv;
            c.tval = s_tval + threadIdx.x;
            c.cache = s_cache;   // not read: a loop-free statement evaluates its rows where used
            expand_unit_fast<0>(c, s, g, res, count, sink);
          } else if (S.n_loops > kFastLoops) {
            expand_unit_generic(M, s, g, res, count, sink);
          } else {
            FastCtx c;
            c.M = B.dm;
            c.S = &S;
            c.tv = tv;
            c.tval = s_tval + threadIdx.x;
            c.cache = s_cache + threadIdx.x;
            expand_unit_dispatch(c, s, g, res, count, sink);
          }
        }
      }
      count = warp_sum(count);
      if ((threadIdx.x & 31) == 0 && count) atomicAdd(&res->instances, count);
      __syncthreads();   // s_model is rewritten for the next unit
    }
  }
}

// ---------------------------------------------------------------------------
// Expansion of packs whose models are all loop-free with one-dimensional grids
// and blocks: every thread expands J model threads at once.
//
// The interpreted expansion is a chain of dependent loads of the lowered program
// (the same for all lanes) with a few integer operations between them, so it is
// bound by their latency and by the instructions that decode the program.  J
// model threads per lane share every load and every decision: a row is three
// coefficients (constant, thread, block) and its terms, read once for J values.
// ---------------------------------------------------------------------------
template <int J>
struct FlatCtx {
  const DevModel* M;
  uint32_t t[J], b[J];   // thread in block, block
  int64_t* tval;         // term q of model thread j: tval[(q * J + j) * kExpandThreads]
};

template <int J>
__device__ __forceinline__ void flat_row(const FlatCtx<J>& c, int r, int64_t (&x)[J]) {
  const Row* R = c.M->rows + r;
  const int64_t c0 = __ldg(&R->c0), kt = __ldg(&R->ct[0]), kbl = __ldg(&R->ct[3]);
  const int2 on = __ldg(reinterpret_cast<const int2*>(&R->off));   // off, nnz
#pragma unroll
  for (int j = 0; j < J; ++j) x[j] = wadd(c0, wadd(wmul(kt, (int64_t)c.t[j]), wmul(kbl, (int64_t)c.b[j])));
  for (int k = 0; k < on.y; ++k) {   // (no iterators: every variable is a term)
    const LinTerm* lt = c.M->lin + on.x + k;
    const int64_t* tv = c.tval + (size_t)(__ldg(&lt->var) - kMaxLoops) * J * kExpandThreads;
    const int64_t coef = __ldg(&lt->coef);
#pragma unroll
    for (int j = 0; j < J; ++j) x[j] = wadd(x[j], wmul(coef, tv[j * kExpandThreads]));
  }
}
static_assert(offsetof(Row, off) % 8 == 0 && offsetof(Row, nnz) == offsetof(Row, off) + 4, "off and nnz are read together");

template <int J>
__device__ __forceinline__ void flat_statement(const FlatCtx<J>& c, const BatchArgs& a, const BatchModel& B, uint32_t s,
                                               uint64_t g0, unsigned valid, DevResult* res,
                                               unsigned long long& count) {
  const DevModel& M = *c.M;
  const DevStmt& S = M.stmts[s];
  int64_t x[J];
  const int n_terms = S.n_terms;
  for (int q = 0; q < n_terms; ++q) {
    const Term* T = M.terms + S.term0 + q;
    flat_row<J>(c, __ldg(&T->row), x);
    const int64_t d = __ldg(&T->d);
    const uint64_t mg = __ldg(&T->magic);
    const int32_t op = __ldg(&T->op);
#pragma unroll
    for (int j = 0; j < J; ++j)
      c.tval[(q * J + j) * kExpandThreads] = op == kFdiv   ? fast_floor_div(x[j], d, mg)
                                             : op == kMod ? fast_euclid_mod(x[j], d, mg)
                                                          : table_load(M, d, x[j]);
  }
  unsigned ok = valid;   // model threads whose guards hold
  for (int g = 0; g < S.n_guards; ++g) {
    flat_row<J>(c, S.guard_row0 + g, x);
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (x[j] < 0) ok &= ~(1u << j);
  }
  count += (unsigned long long)(__popc(ok) * S.n_acc);
  // the fine interval of every model thread, ~0 if it is out of range
  int64_t ph[J];
  flat_row<J>(c, S.row_phase, ph);
  unsigned bad_phase = 0;
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (ph[j] < 0 || ph[j] >= M.n_phases) bad_phase |= 1u << j;
  if (S.row_wphase >= 0) {
    flat_row<J>(c, S.row_wphase, x);
#pragma unroll
    for (int j = 0; j < J; ++j) {
      if (x[j] < 0 || x[j] >= M.n_wphases) bad_phase |= 1u << j;
      ph[j] = ph[j] * M.n_wphases + x[j];
    }
  } else {
#pragma unroll
    for (int j = 0; j < J; ++j) ph[j] *= M.n_wphases;
  }
  uint64_t* keys = a.keys + B.key_base + S.slot_base + g0;
  const uint64_t T = M.n_threads;
  for (int ai = 0; ai < S.n_acc; ++ai) {
    const DevAccess* A = M.accs + S.acc0 + ai;
    const DevArray* arr = M.arrays + __ldg(&A->array);
    const int nd = __ldg(&A->ndims), row0 = __ldg(&A->row0), kidx = __ldg(&A->key_idx);
    uint64_t e[J];
#pragma unroll
    for (int j = 0; j < J; ++j) e[j] = 0;
    unsigned bad = bad_phase & ok;
    if (bad) {
#pragma unroll
      for (int j = 0; j < J; ++j)
        if ((bad >> j) & 1u)
          atomicMin(&res->oob_code, oob_pack(s, (uint32_t)ai, g0 + (uint64_t)j * kExpandThreads, 0));
    }
    for (int d = 0; d < nd; ++d) {
      flat_row<J>(c, row0 + d, x);
      const int64_t ext = __ldg(&arr->ext[d]);
#pragma unroll
      for (int j = 0; j < J; ++j) {
        if ((x[j] < 0 || x[j] >= ext) && ((ok >> j) & 1u)) {
          atomicMin(&res->oob_code, oob_pack(s, (uint32_t)ai, g0 + (uint64_t)j * kExpandThreads, (uint32_t)d + 1));
          bad |= 1u << j;
        }
        e[j] = e[j] * (uint64_t)ext + (uint64_t)x[j];
      }
    }
    if (kidx < 0) continue;   // array never written: bounds-checked and counted, no key
    const uint64_t base = B.cell_base + __ldg(&arr->base);
    const uint64_t per_block = __ldg(&arr->shared) ? __ldg(&arr->cells) : 0ull;
    const uint64_t kind = (uint64_t)__ldg(&A->kind);
#pragma unroll
    for (int j = 0; j < J; ++j)
      if ((valid >> j) & 1u) {
        const uint64_t cell = base + per_block * c.b[j] + e[j];
        const uint64_t key = (cell << a.cell_shift) | ((uint64_t)ph[j] << a.phase_shift) |
                             ((uint64_t)c.b[j] << a.block_shift) | ((uint64_t)c.t[j] << a.thread_shift) | kind;
        keys[(uint64_t)kidx * T + (uint64_t)j * kExpandThreads] = ((ok & ~bad) >> j) & 1u ? key : kSentinel;
      }
  }
}

template <int J>
__global__ void __launch_bounds__(kExpandThreads, J > 1 ? 4 : 7) batch_expand_flat_kernel(BatchArgs a) {
  extern __shared__ int64_t s_terms[];
  __shared__ unsigned long long s_u;
  __shared__ uint32_t s_model;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      s_u = atomicAdd(a.queue, (unsigned long long)a.grab);
      uint32_t lo = 0, hi = a.n_models;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a.models[mid].unit_base <= s_u) lo = mid;
        else hi = mid;
      }
      s_model = lo;
    }
    __syncthreads();
    const uint64_t u0 = s_u;
    if (u0 >= a.n_units) break;
    const uint64_t u1 = min(a.n_units, u0 + a.grab);
    uint32_t mi = s_model;   // (every thread steps forward by itself: the table entries are broadcast loads)
    for (uint64_t u = u0; u < u1; ++u) {
      while (mi + 1 < a.n_models && a.models[mi + 1].unit_base <= u) ++mi;
      const BatchModel& B = a.models[mi];
      const DevModel& M = *B.dm;
      const uint64_t g0 = (u - B.unit_base) * (uint64_t)(kExpandThreads * J) + threadIdx.x;
      DevResult* res = a.res + mi;
      FlatCtx<J> c;
      c.M = B.dm;
      c.tval = s_terms + threadIdx.x;
      unsigned valid = 0;
      const uint64_t mg = M.div_magic[0];
      const uint32_t bs = M.bs;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const uint64_t g = g0 + (uint64_t)j * kExpandThreads;
        if (g < B.n_threads) valid |= 1u << j;
        c.b[j] = (uint32_t)div_small(g, mg);
        c.t[j] = (uint32_t)g - c.b[j] * bs;
      }
      unsigned long long count = 0;
      for (uint32_t s = 0; s < B.n_stmts; ++s) flat_statement<J>(c, a, B, s, g0, valid, res, count);
      count = warp_sum(count);
      if ((threadIdx.x & 31) == 0 && count) atomicAdd(&res->instances, count);
    }
  }
}

// Errors of a pack's shared stages (sort look-back, scan) reach every model.
__global__ void batch_errors_kernel(const DevResult* pack, DevResult* res, uint32_t n) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned e = pack->err;
  if (i < n && e) res[i].err |= e;
}

}  // namespace

cudaError_t launch_batch_errors(const DevResult* pack, DevResult* res, uint32_t n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  batch_errors_kernel<<<(n + 127) / 128, 128, 0, st>>>(pack, res, n);
  return cudaGetLastError();
}

template <int J>
static cudaError_t launch_flat(BatchArgs a, uint32_t max_terms, int sms, cudaStream_t st) {
  const size_t smem = (size_t)(max_terms ? max_terms : 1) * J * kExpandThreads * 8;
  const void* fn = reinterpret_cast<const void*>(batch_expand_flat_kernel<J>);
  const cudaError_t e = ensure_kernel_smem(fn, (size_t)kMaxTerms * J * kExpandThreads * 8, false);
  if (e != cudaSuccess) return e;
  int per_sm = 4;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_expand_flat_kernel<J>, kExpandThreads, smem);
  if (per_sm < 1) per_sm = 1;
  const uint64_t full = (uint64_t)sms * per_sm;
  // several grabs per block, so that the blocks end together
  a.grab = (uint32_t)std::min<uint64_t>(kUnitsPerGrab, std::max<uint64_t>(1, a.n_units / (full * 8)));
  const uint64_t grid = std::min(full, (a.n_units + a.grab - 1) / a.grab);
  batch_expand_flat_kernel<J><<<(unsigned)grid, kExpandThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_batch_expand(const BatchArgs& a, bool loop_free, uint32_t flat, uint32_t max_terms,
                                cudaStream_t st) {
  if (a.n_units == 0) return cudaSuccess;
  int dev = 0, sms = 152, per_sm = 4;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (flat == kBatchFlatThreads) return launch_flat<kBatchFlatThreads>(a, max_terms, sms, st);
  if (flat == 1) return launch_flat<1>(a, max_terms, sms, st);
  if (loop_free) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_expand_kernel<true>, kExpandThreads, 0);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_expand_kernel<false>, kExpandThreads, 0);
  if (per_sm < 1) per_sm = 1;
  BatchArgs b = a;
  const uint64_t full = (uint64_t)sms * per_sm;
  b.grab = (uint32_t)std::min<uint64_t>(kUnitsPerGrab, std::max<uint64_t>(1, a.n_units / (full * 8)));
  const uint64_t grid = std::min(full, (a.n_units + b.grab - 1) / b.grab);
  if (loop_free) batch_expand_kernel<true><<<(unsigned)grid, kExpandThreads, 0, st>>>(b);
  else batch_expand_kernel<false><<<(unsigned)grid, kExpandThreads, 0, st>>>(b);
  return cudaGetLastError();
}

}  // namespace rc
