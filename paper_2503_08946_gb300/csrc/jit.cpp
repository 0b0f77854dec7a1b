// Per-model expansion kernel generated as CUDA C and compiled at run time with
// NVRTC for sm_103a.
//
// The interpreted expansion (expand.cu) reads every coefficient, divisor and
// array constant from the lowered program at every access instance.  For a
// large model the same lowered rows are instead written out as source code:
// each statement becomes a real loop nest with its coefficients, extents and
// divisors as literals, so the compiler folds constants, hoists the
// thread-constant expressions out of the loops and turns floor division and
// modulo by constants into multiply-shift sequences (or masks and shifts for
// powers of two).  With all points (rc_expand_keys) the generated kernel writes
// exactly the keys of the interpreted one (same slots, same padding, same
// out-of-bounds report).
//
// NVRTC and the CUDA driver entry points are resolved at run time (dlopen and
// cudaGetDriverEntryPointByVersion), so the library loads on machines without
// them; rc_model_create then keeps the interpreted expansion.  Compiled
// kernels are cached per device by their source text.
//
// A check expands each statement's distinct points only (find_distinct_points), in
// slots of their own (Model.check_slots instead of key_slots), and writes padding for
// an access that repeats its instance in the innermost loop.  Random affine models of
// 4096 x 256 threads keep 29 to 52 % of their keys, and every later stage moves that
// much less.  Measured on one of them (303 of 578 M keys): the expansion 0.89 -> 0.71
// ms (it evaluates a point from its number instead of stepping a loop), the check
// 7.2 -> 4.3 ms.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <nvrtc.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "rc_internal.h"

namespace rc {

namespace {

// ---------------------------------------------------------------------------
// run-time loaded NVRTC and driver entry points
// ---------------------------------------------------------------------------
struct Nvrtc {
  bool ok = false;
  nvrtcResult (*create)(nvrtcProgram*, const char*, const char*, int, const char* const*, const char* const*);
  nvrtcResult (*compile)(nvrtcProgram, int, const char* const*);
  nvrtcResult (*cubin_size)(nvrtcProgram, size_t*);
  nvrtcResult (*cubin)(nvrtcProgram, char*);
  nvrtcResult (*destroy)(nvrtcProgram*);
};

struct Driver {
  bool ok = false;
  CUresult (*load)(CUmodule*, const void*);
  CUresult (*get)(CUfunction*, CUmodule, const char*);
  CUresult (*launch)(CUfunction, unsigned, unsigned, unsigned, unsigned, unsigned, unsigned, unsigned, CUstream,
                     void**, void**);
};

std::mutex g_jit_mu;

// The NVRTC entry points, looked up once per process (a function-local static
// is initialised once even when several host threads get here together).
Nvrtc load_nvrtc() {
  Nvrtc n;
  const char* names[] = {"libnvrtc.so.13", "libnvrtc.so", "/usr/local/cuda/lib64/libnvrtc.so.13",
                         "/usr/local/cuda/lib64/libnvrtc.so"};
  void* h = nullptr;
  for (const char* nm : names)
    if ((h = dlopen(nm, RTLD_NOW | RTLD_LOCAL)) != nullptr) break;
  if (!h) return n;
  n.create = reinterpret_cast<decltype(n.create)>(dlsym(h, "nvrtcCreateProgram"));
  n.compile = reinterpret_cast<decltype(n.compile)>(dlsym(h, "nvrtcCompileProgram"));
  n.cubin_size = reinterpret_cast<decltype(n.cubin_size)>(dlsym(h, "nvrtcGetCUBINSize"));
  n.cubin = reinterpret_cast<decltype(n.cubin)>(dlsym(h, "nvrtcGetCUBIN"));
  n.destroy = reinterpret_cast<decltype(n.destroy)>(dlsym(h, "nvrtcDestroyProgram"));
  n.ok = n.create && n.compile && n.cubin_size && n.cubin && n.destroy;
  return n;
}
Nvrtc& nvrtc() {
  static Nvrtc n = load_nvrtc();
  return n;
}

Driver load_driver() {
  Driver d;
  auto get = [](const char* sym, void** fn) {
    cudaDriverEntryPointQueryResult q;
    return cudaGetDriverEntryPointByVersion(sym, fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
           q == cudaDriverEntryPointSuccess && *fn != nullptr;
  };
  void *a = nullptr, *b = nullptr, *c = nullptr;
  d.ok = get("cuModuleLoadData", &a) && get("cuModuleGetFunction", &b) && get("cuLaunchKernel", &c);
  d.load = reinterpret_cast<decltype(d.load)>(a);
  d.get = reinterpret_cast<decltype(d.get)>(b);
  d.launch = reinterpret_cast<decltype(d.launch)>(c);
  return d;
}
Driver& driver() {
  static Driver d = load_driver();
  return d;
}

std::map<std::string, void*> g_cache;   // (device, source) -> CUfunction

// ---------------------------------------------------------------------------
// code generation
// ---------------------------------------------------------------------------
std::string lit(int64_t v) {
  if (v == INT64_MIN) return "((long long)0x8000000000000000ull)";
  return "(" + std::to_string(v) + "LL)";
}
std::string ulit(uint64_t v) { return std::to_string(v) + "ull"; }

bool is_pow2(int64_t d) { return d > 0 && (d & (d - 1)) == 0; }
int log2i(int64_t d) {
  int k = 0;
  while ((1ll << k) < d) ++k;
  return k;
}

// The distinct points of a statement's loop nest: flat iteration numbers, and
// how many points each stands for.
struct DistinctPoints {
  std::vector<uint32_t> point, times;
};
constexpr unsigned kRouteChunks = 1024;            // chunks of a wave routed in two sweeps
constexpr uint64_t kDistinctMaxPoints = 4096;      // points of a nest that are compared
constexpr size_t kConstantBytes = 60 << 10;
constexpr size_t kDistinctTableBytes = 48 << 10;   // constant memory for the points of all statements

struct Gen {
  const Model& m;
  bool chunked = false;   // count / route kernel of chunked checks instead of the slot kernel
  const uint8_t* img;
  const DevStmt* stmts;
  const DevAccess* accs;
  const DevArray* arrays;
  const Row* rows;
  const LinTerm* lin;
  const Term* terms;
  std::ostringstream o;
  std::vector<DistinctPoints> dp;   // per statement (empty: every point is expanded)
  std::vector<uint64_t> check_base; // first key slot of each dense statement's distinct points
  uint64_t check_dense = 0;         // key slots of all dense statements' distinct points

  explicit Gen(const Model& mm) : m(mm), img(mm.program.data()) {
    stmts = reinterpret_cast<const DevStmt*>(img + m.sec_stmts);
    accs = reinterpret_cast<const DevAccess*>(img + m.sec_accs);
    arrays = reinterpret_cast<const DevArray*>(img + m.sec_arrays);
    rows = reinterpret_cast<const Row*>(img + m.sec_rows);
    lin = reinterpret_cast<const LinTerm*>(img + m.sec_lin);
    terms = reinterpret_cast<const Term*>(img + m.sec_terms);
    find_distinct_points();
    plan_blocks();
  }

  // The slot kernel's blocks.  Every block counts the pass-A histogram of its keys
  // in shared memory and adds it to the global one, whose few cache lines all
  // blocks share: with a block per 128 threads and statement those additions took
  // most of the time of statements with few keys per thread (the transposition,
  // 12.6 M key slots: 77 us with 768 slots per block, 23 us with 7,000).  So a
  // block takes as many 128-thread units of its statement as make about an equal
  // share of the model's work: 10,000 keys (4,000 measured slower on models of 10
  // to 50 M keys), in 12 to 64 blocks per SM (fewer leave SMs idle at the end;
  // 4096 x 256: 0.60 ms with 16, 0.46 ms with 64), heavy statements first.
  std::vector<uint32_t> blk_stmt, blk_first, blk_units;   // per statement, in launch order
  uint64_t blocks = 0;
  void plan_blocks() {
    const uint32_t ns = m.host.n_stmts;
    const uint64_t T = m.host.n_threads, units = (T + 127) / 128;
    uint64_t general_keys = 0;
    for (uint32_t s = 0; s < ns; ++s)
      if (!stmts[s].dense) general_keys += stmts[s].n_key;
    // keys per thread, an access without a key as half of one (points of
    // statements with thread-dependent trips: their average)
    std::vector<double> w(ns);
    double total = 0;
    for (uint32_t s = 0; s < ns; ++s) {
      const DevStmt& S = stmts[s];
      double pts = 16;
      if (S.dense) pts = dp[s].point.empty() ? (double)S.n_iter : (double)dp[s].point.size();
      else if (general_keys) pts = std::max(1.0, (double)m.host.general_slots / (double)(general_keys * T));
      w[s] = pts * (S.n_key + 0.5 * (S.n_acc - S.n_key)) + 0.5;
      total += w[s] * (double)units;
    }
    const double per_sm = std::min(64.0, std::max(12.0, total * 128.0 / (10000.0 * 152.0)));
    double share = std::max(total / (152.0 * per_sm), 8.0);
    std::vector<uint32_t> u(ns);
    for (;; share *= 2) {
      blocks = 0;
      for (uint32_t s = 0; s < ns; ++s) {
        const double n = share / w[s];
        u[s] = n < 1 ? 1u : n > (double)units ? (uint32_t)std::min<uint64_t>(units, 1u << 30) : (uint32_t)n;
        if (u[s] == 0) u[s] = 1;
        blocks += (units + u[s] - 1) / u[s];
      }
      if (blocks <= 0x7fffffffull || units == 0) break;
    }
    blk_stmt.resize(ns);
    for (uint32_t s = 0; s < ns; ++s) blk_stmt[s] = s;
    std::stable_sort(blk_stmt.begin(), blk_stmt.end(), [&](uint32_t a, uint32_t b) { return w[a] * u[a] > w[b] * u[b]; });
    uint64_t first = 0;
    for (uint32_t s : blk_stmt) {
      blk_first.push_back((uint32_t)first);
      blk_units.push_back(u[s]);
      first += (units + u[s] - 1) / u[s];
    }
  }

  // Whether every point differs from all others in some row, shown without looking
  // at the points: a row whose coefficients grow faster than what the smaller ones
  // can add up to tells the numbers of its loops (a mixed radix), and what is known
  // leaves the other rows with fewer loops.  (False: not shown.)
  static bool all_points_differ(const DevStmt& S, const std::vector<std::vector<uint64_t>>& co) {
    uint32_t known = 0;
    for (int l = 0; l < S.n_loops; ++l)
      if (S.trips[l] <= 1) known |= 1u << l;
    for (bool more = true; more;) {
      more = false;
      for (const std::vector<uint64_t>& c : co) {
        std::vector<std::pair<unsigned __int128, int>> a;   // (magnitude, loop)
        for (int l = 0; l < S.n_loops; ++l) {
          const int64_t v = (int64_t)c[l];
          if (v != 0 && !((known >> l) & 1u)) a.emplace_back(v < 0 ? -(__int128)v : (__int128)v, l);
        }
        if (a.empty()) continue;
        std::sort(a.begin(), a.end());
        unsigned __int128 sum = 0;   // (trips are at most kDistinctMaxPoints)
        bool radix = true;
        for (const auto& x : a) {
          radix = radix && x.first > sum;
          sum += x.first * (unsigned __int128)(S.trips[x.second] - 1);
        }
        if (!radix || sum >> 63) continue;   // (rows are evaluated modulo 2^64)
        for (const auto& x : a) known |= 1u << x.second;
        more = true;
      }
    }
    return known == (1u << S.n_loops) - 1u;
  }

  // The distinct points in order of their first, if they are at most `most`: the
  // loops that move some row are run through, the others multiply.
  bool enumerate_points(const DevStmt& S, const std::vector<std::vector<uint64_t>>& co, size_t most, DistinctPoints* p) {
    const size_t nr = co.size();
    std::vector<int> moving;
    std::vector<uint64_t> stride(S.n_loops);
    uint64_t n = 1, times = 1, at = 1;
    for (int l = S.n_loops - 1; l >= 0; --l) {
      stride[l] = at;
      at *= (uint64_t)S.trips[l];
      bool moves = false;
      for (size_t r = 0; r < nr; ++r) moves = moves || co[r][l] != 0;
      if (moves) {
        moving.insert(moving.begin(), l);
        n *= (uint64_t)S.trips[l];
      } else {
        times *= (uint64_t)S.trips[l];
      }
    }
    // an open-addressed table of the points found (1 + their number) and their images
    size_t cap = 64;
    while (cap < 2 * n) cap *= 2;
    point_table.assign(cap, 0u);
    point_images.clear();
    std::vector<uint64_t> im(nr, 0);
    std::vector<int64_t> k(moving.size(), 0);
    uint64_t e = 0;
    for (uint64_t x = 0; x < n; ++x) {
      uint64_t h = 0;
      for (uint64_t v : im) h = (h ^ v) * 0x9E3779B97F4A7C15ull, h ^= h >> 29;
      size_t i = (size_t)h & (cap - 1);
      for (; point_table[i] != 0u; i = (i + 1) & (cap - 1))
        if (std::equal(im.begin(), im.end(), point_images.begin() + (size_t)(point_table[i] - 1u) * nr)) break;
      if (point_table[i] == 0u) {
        if (p->point.size() >= most) return false;
        p->point.push_back((uint32_t)e);
        p->times.push_back(0);
        point_images.insert(point_images.end(), im.begin(), im.end());
        point_table[i] = (uint32_t)p->point.size();
      }
      p->times[point_table[i] - 1u] += (uint32_t)times;
      for (size_t q = moving.size(); q-- > 0;) {   // the next point
        const int l = moving[q];
        if (++k[q] < S.trips[l]) {
          e += stride[l];
          for (size_t r = 0; r < nr; ++r) im[r] += co[r][l];
          break;
        }
        k[q] = 0;
        e -= stride[l] * (uint64_t)(S.trips[l] - 1);
        for (size_t r = 0; r < nr; ++r) im[r] -= co[r][l] * (uint64_t)(S.trips[l] - 1);
      }
    }
    return true;
  }
  std::vector<uint32_t> point_table;   // scratch of enumerate_points
  std::vector<uint64_t> point_images;

  // The points of a dense statement's loop nest that differ in some row.  A
  // point enters an instance only through the rows of the statement (guards,
  // intervals, indices, operands of its terms), each linear in the iterators, so
  // two points at which the iterators add the same to every row give every
  // thread the same instances: equal tuples, which are one instance of the race
  // question (all of them are counted).  A loop over which an access does not
  // move, or moves along with another loop, is the usual case.  Statements whose
  // loop bounds move with an outer iterator keep all their points.
  void find_distinct_points() {
    const uint32_t ns = m.host.n_stmts;
    dp.resize(ns);
    check_base.assign(ns, 0);
    // (constant memory holds 64 KB, of which the block table takes 12 bytes a statement)
    const size_t blk_bytes = 12 * ((size_t)ns + 1);
    size_t budget = blk_bytes + kDistinctTableBytes <= kConstantBytes ? kDistinctTableBytes
                    : blk_bytes < kConstantBytes                      ? kConstantBytes - blk_bytes
                                                                      : 0;
    for (uint32_t s = 0; s < ns; ++s) {
      const DevStmt& S = stmts[s];
      if (!S.dense) continue;
      check_base[s] = check_dense;
      uint64_t n_pts = S.n_iter;
      bool ok = S.n_loops > 0 && S.n_iter > 1 && S.n_iter <= kDistinctMaxPoints;
      for (int l = 0; l < S.n_loops; ++l) ok = ok && rows[S.row_lower[l]].nnz == 0;
      if (ok) {
        std::vector<int> rr;
        for (int g = 0; g < S.n_guards; ++g) rr.push_back(S.guard_row0 + g);
        rr.push_back(S.row_phase);
        if (S.row_wphase >= 0) rr.push_back(S.row_wphase);
        for (int a = 0; a < S.n_acc; ++a)
          for (int d = 0; d < accs[S.acc0 + a].ndims; ++d) rr.push_back(accs[S.acc0 + a].row0 + d);
        for (int q = 0; q < S.n_terms; ++q) rr.push_back(terms[S.term0 + q].row);
        // what one step of each loop adds to each row (modulo 2^64, as the rows
        // are evaluated); equal and all-zero rows tell nothing more
        std::vector<std::vector<uint64_t>> co;
        for (int r : rr) {
          std::vector<uint64_t> c(S.n_loops, 0);
          for (int k = 0; k < rows[r].nnz; ++k) {
            const LinTerm& t = lin[rows[r].off + k];
            if (t.var < kMaxLoops) c[t.var] += (uint64_t)t.coef * (uint64_t)S.step[t.var];
          }
          bool zero = true;
          for (uint64_t v : c) zero = zero && v == 0;
          if (!zero && std::find(co.begin(), co.end(), c) == co.end()) co.push_back(c);
        }
        DistinctPoints p;
        // (a table and a division per point: worth it from a tenth of the points on)
        const size_t most = std::min<size_t>(budget / 4, (size_t)(S.n_iter * 9 / 10));
        if (!all_points_differ(S, co) && enumerate_points(S, co, most, &p)) {
          budget -= 4 * p.point.size();
          n_pts = p.point.size();
          dp[s] = std::move(p);
        }
      }
      check_dense += n_pts * (uint64_t)S.n_key * m.host.n_threads;
    }
  }

  // -------------------------------------------------------------------------
  // Value ranges.  Every row of a statement is bounded from the grid, the loop
  // bounds, the divisors and the table values.  Rows whose values fit 32 bits are
  // evaluated in 32-bit arithmetic (modulo 2^32 every partial result may wrap, the
  // value itself does not), and checks that a range decides are left out.  A row
  // without a bound (or one that might leave 64 bits) is evaluated as it is
  // written, in 64 bits.
  // -------------------------------------------------------------------------
  struct Range {
    __int128 lo = 0, hi = 0;
    bool known = false;
    bool narrow() const { return known && lo >= -2147483647 && hi <= 2147483647; }
    bool inside(__int128 a, __int128 b) const { return known && lo >= a && hi < b; }   // [a, b)
  };
  std::vector<Range> r_it, r_term;   // the statement's iterators and terms
  std::vector<bool> n_it, n_term;    // ... that are 32-bit variables

  static Range bounded(__int128 lo, __int128 hi) {
    Range r;
    r.lo = lo;
    r.hi = hi;
    const __int128 lim = (__int128)1 << 62;
    r.known = lo >= -lim && hi <= lim;
    return r;
  }
  Range range(int r) const {
    const Row& R = rows[r];
    __int128 lo = R.c0, hi = R.c0;
    const __int128 lim = (__int128)1 << 62;
    auto add = [&](int64_t c, __int128 l, __int128 h) {   // (|c| < 2^64, |l|, |h| <= 2^62: no overflow)
      lo += c >= 0 ? c * l : c * h;
      hi += c >= 0 ? c * h : c * l;
    };
    for (int i = 0; i < 6; ++i) {
      if (!R.ct[i]) continue;
      const uint32_t n = i < 3 ? m.host.block[i] : m.host.grid[i - 3];
      add(R.ct[i], 0, (__int128)n - 1);
      if (lo < -lim || hi > lim) return Range();
    }
    for (int k = 0; k < R.nnz; ++k) {
      const LinTerm& t = lin[R.off + k];
      const Range& v = t.var < kMaxLoops ? r_it[t.var] : r_term[t.var - kMaxLoops];
      if (!v.known) return Range();
      add(t.coef, v.lo, v.hi);
      if (lo < -lim || hi > lim) return Range();
    }
    return bounded(lo, hi);
  }
  static __int128 fdiv128(__int128 a, int64_t d) { return a >= 0 ? a / d : -((-a + d - 1) / d); }
  Range term_range(const Term& T) const {
    const Range a = range(T.row);
    if (T.op == kLoad) {
      const uint64_t* tidx = reinterpret_cast<const uint64_t*>(img + m.sec_tabidx);
      const int64_t* data = reinterpret_cast<const int64_t*>(img + m.sec_tdata) + tidx[2 * T.d];
      const uint64_t n = tidx[2 * T.d + 1];
      int64_t lo = 0, hi = 0;   // (a load outside the table is 0)
      for (uint64_t i = 0; i < n; ++i) {
        lo = std::min(lo, data[i]);
        hi = std::max(hi, data[i]);
      }
      return bounded(lo, hi);
    }
    if (T.op == kFdiv) return a.known ? bounded(fdiv128(a.lo, T.d), fdiv128(a.hi, T.d)) : Range();
    return a.inside(0, T.d) ? a : bounded(0, (__int128)T.d - 1);
  }
  // the ranges of a statement's iterators and terms, outer levels first
  void find_ranges(const DevStmt& S) {
    r_it.assign(kMaxLoops, Range());
    r_term.assign(kMaxTerms, Range());
    n_it.assign(kMaxLoops, false);
    n_term.assign(kMaxTerms, false);
    for (int l = 0; l <= S.n_loops; ++l) {
      for (int q = 0; q < S.n_terms; ++q)
        if (terms[S.term0 + q].level == l) {
          r_term[q] = term_range(terms[S.term0 + q]);
          n_term[q] = r_term[q].narrow();
        }
      if (l == S.n_loops) break;
      const Range lo = range(S.row_lower[l]), hi = range(S.row_upper[l]);
      if (!lo.known || !hi.known) continue;
      r_it[l] = bounded(lo.lo, std::max(hi.hi - 1, lo.lo));
      // (the variable itself runs past the upper bound by a step at most)
      n_it[l] = lo.narrow() && hi.narrow() && S.step[l] < (1ll << 30) && hi.hi + S.step[l] <= 2147483647 && r_it[l].narrow();
    }
  }

  // a row in 64 bits, wrapping (so in unsigned arithmetic: the compiler may take
  // signed values for bounded)
  std::string row64(int r) {
    static const char* tv[6] = {"tx", "ty", "tz", "bx", "by", "bz"};
    const Row& R = rows[r];
    std::string e = ulit((uint64_t)R.c0);
    for (int i = 0; i < 6; ++i)
      if (R.ct[i]) e += " + " + ulit((uint64_t)R.ct[i]) + " * (unsigned long long)" + tv[i];
    for (int k = 0; k < R.nnz; ++k) {
      const LinTerm& t = lin[R.off + k];
      const std::string v = t.var < kMaxLoops ? "i" + std::to_string(t.var) : "q" + std::to_string(t.var - kMaxLoops);
      e += " + " + ulit((uint64_t)t.coef) + " * (unsigned long long)" + v;
    }
    return "((long long)(" + e + "))";
  }
  // its value modulo 2^32
  std::string row32(int r) {
    static const char* tv[6] = {"tx", "ty", "tz", "bx", "by", "bz"};
    const Row& R = rows[r];
    auto u = [](int64_t v) { return std::to_string((uint32_t)(uint64_t)v) + "u"; };
    std::string e = u(R.c0);
    for (int i = 0; i < 6; ++i)
      if (R.ct[i]) e += " + " + u(R.ct[i]) + " * (unsigned)" + tv[i];
    for (int k = 0; k < R.nnz; ++k) {
      const LinTerm& t = lin[R.off + k];
      const std::string v = t.var < kMaxLoops ? "i" + std::to_string(t.var) : "q" + std::to_string(t.var - kMaxLoops);
      e += " + " + u(t.coef) + " * (unsigned)" + v;
    }
    return "((int)(" + e + "))";
  }
  std::string row(int r) { return range(r).narrow() ? row32(r) : row64(r); }
  std::string row_type(int r) { return range(r).narrow() ? "int" : "long long"; }

  void emit_terms(const DevStmt& S, int level, const std::string& ind) {
    for (int q = 0; q < S.n_terms; ++q) {
      const Term& T = terms[S.term0 + q];
      if (T.level != level) continue;
      const Range a = range(T.row);
      const bool small_d = T.d < (1ll << 31);
      std::string v;
      if (T.op == kLoad) {
        const uint64_t* tidx = reinterpret_cast<const uint64_t*>(img + m.sec_tabidx);
        v = "tload_c(tdata, " + ulit(tidx[2 * T.d]) + ", " + ulit(tidx[2 * T.d + 1]) + ", (long long)" + row(T.row) + ")";
      } else if (T.op == kMod && a.inside(0, T.d)) {
        v = row(T.row);
      } else if (is_pow2(T.d) && (!a.narrow() || small_d)) {
        v = T.op == kFdiv ? "(" + row(T.row) + " >> " + std::to_string(log2i(T.d)) + ")"
                          : "(" + row(T.row) + " & " + (a.narrow() ? std::to_string(T.d - 1) : lit(T.d - 1)) + ")";
      } else if (a.narrow() && small_d) {
        const std::string d = std::to_string(T.d);
        if (a.lo >= 0) v = "(int)((unsigned)" + row32(T.row) + (T.op == kFdiv ? " / " : " % ") + d + "u)";
        else v = (T.op == kFdiv ? "fdiv_n(" : "mod_n(") + row32(T.row) + ", " + d + ")";
      } else {
        v = (T.op == kFdiv ? "fdiv_c(" : "mod_c(") + row64(T.row) + ", " + lit(T.d) + ")";
      }
      o << ind << "const " << (n_term[q] ? "int" : "long long") << " q" << q << " = "
        << (n_term[q] ? "(int)" : "(long long)") << v << ";\n";
    }
  }

  // whether a row keeps its value while only the innermost iterator moves
  bool fixed_inside(const DevStmt& S, int r) const {
    for (int k = 0; k < rows[r].nnz; ++k) {
      const LinTerm& t = lin[rows[r].off + k];
      if (t.var < kMaxLoops ? t.var == S.n_loops - 1 : terms[S.term0 + t.var - kMaxLoops].level == S.n_loops) return false;
    }
    return true;
  }

  void emit_stmt(uint32_t s) {
    const DevStmt& S = stmts[s];
    const DevModel& h = m.host;
    const uint64_t T = h.n_threads;
    find_ranges(S);
    o << "    case " << s << ": {\n";
    const bool distinct = !dp[s].point.empty();
    if (chunked) {
      // keys go to chunk_put; no slots
    } else if (S.dense) {
      o << "      unsigned long long* out = keys + (all_points ? " << ulit(S.slot_base) << " : " << ulit(check_base[s])
        << ") + g;\n";
    } else {
      o << "      unsigned long long* out = keys + unit_offset[" << ulit(S.slot_base) << " + g]"
        << (check_dense != h_dense() ? " - (all_points ? 0ull : " + ulit(h_dense() - check_dense) + ")" : std::string())
        << ";\n";
    }
    // An access that stays where it is while the innermost loop runs repeats its
    // last key there (the same instance again): only the first is kept.
    std::vector<bool> repeats(S.n_acc, false);
    for (int a = 0; a < S.n_acc && S.n_loops > 0 && !distinct; ++a) {
      const DevAccess& A = accs[S.acc0 + a];
      if (A.key_idx < 0) continue;
      bool fixed = fixed_inside(S, S.row_phase) && (S.row_wphase < 0 || fixed_inside(S, S.row_wphase));
      for (int d = 0; d < A.ndims; ++d) fixed = fixed && fixed_inside(S, A.row0 + d);
      repeats[a] = fixed;
      if (fixed) o << "      unsigned long long last" << a << " = ~0ull" << (chunked ? ", lastc" + std::to_string(a) + " = ~0ull" : std::string()) << ";\n";
    }
    emit_terms(S, 0, "      ");
    std::string ind = "      ";
    if (distinct) {
      // one loop over the statement's distinct points (or over all of them)
      o << ind << "for (unsigned p = 0; p < " << (chunked ? "" : "(all_points ? " + std::to_string(S.n_iter) + "u : ")
        << dp[s].point.size() << (chunked ? "u" : "u)") << "; ++p) {\n";
      ind += "  ";
      o << ind << "unsigned e = " << (chunked ? "" : "all_points ? p : ") << "(unsigned)pts" << s << "[p].x;\n";
      for (int l = S.n_loops - 1; l >= 0; --l) {
        const std::string k = "(e" + (l ? " % " + std::to_string(S.trips[l]) + "u" : std::string()) + ")";
        // (the iterator fits its type, the step times the point's number may not: it wraps)
        if (n_it[l])
          o << ind << "const int i" << l << " = (int)((unsigned)" << row32(S.row_lower[l]) << " + " << S.step[l]
            << "u * (unsigned)" << k << ");\n";
        else
          o << ind << "const long long i" << l << " = (long long)((unsigned long long)" << row64(S.row_lower[l]) << " + "
            << ulit((uint64_t)S.step[l]) << " * (unsigned long long)" << k << ");\n";
        if (l) o << ind << "e /= " << S.trips[l] << "u;\n";
      }
      for (int l = 0; l < S.n_loops; ++l) emit_terms(S, l + 1, ind);
    }
    for (int l = 0; l < S.n_loops && !distinct; ++l) {
      if (n_it[l])
        o << ind << "for (int i" << l << " = " << row32(S.row_lower[l]) << "; i" << l << " < " << row32(S.row_upper[l])
          << "; i" << l << " += " << S.step[l] << ") {\n";
      else
        o << ind << "for (long long i" << l << " = " << row64(S.row_lower[l]) << "; i" << l << " < "
          << row64(S.row_upper[l]) << "; i" << l << " += " << lit(S.step[l]) << ") {\n";
      ind += "  ";
      emit_terms(S, l + 1, ind);
    }
    // guards (those that the ranges decide left out)
    std::string gcond = "true";
    for (int gi = 0; gi < S.n_guards; ++gi) {
      const Range r = range(S.guard_row0 + gi);
      if (r.known && r.lo >= 0) continue;
      gcond += " && " + row(S.guard_row0 + gi) + " >= 0";
    }
    o << ind << "if (" << gcond << ") {\n";
    const std::string in2 = ind + "  ";
    const bool fine = S.row_wphase >= 0 || h.n_wphases > 1;
    // the (fine) interval; ph_ok: the ranges show that it is one
    bool ph_ok = range(S.row_phase).inside(0, h.n_phases);
    if (S.row_wphase >= 0) ph_ok = ph_ok && range(S.row_wphase).inside(0, h.n_wphases);
    if (fine) {
      // the fine interval phase * n_wphases + warp phase; -1 if either is out of range
      o << in2 << "const long long ph0 = " << row(S.row_phase) << ";\n";
      o << in2 << "const long long wph = " << (S.row_wphase >= 0 ? row(S.row_wphase) : std::string("0LL")) << ";\n";
      o << in2 << "const long long ph = (ph0 < 0 || ph0 >= " << lit(h.n_phases) << " || wph < 0 || wph >= "
        << lit(h.n_wphases) << ") ? -1LL : ph0 * " << lit(h.n_wphases) << " + wph;\n";
    } else {
      o << in2 << "const " << row_type(S.row_phase) << " ph = " << row(S.row_phase) << ";\n";
    }
    o << in2 << "(void)ph;\n";
    // Statements with thread-dependent trips: every thread writes its own run, so
    // each 8-byte store of a warp is 32 sectors; the keys of a point are stored in
    // pairs where the run is 16-byte aligned.
    const bool pairs = !chunked && !S.dense && S.n_key > 1;
    if (pairs)
      for (int kq = 0; kq < S.n_key; ++kq) o << in2 << "unsigned long long k" << kq << " = ~0ull;\n";
    const bool cl32 = m.total_cells < (1ull << 32);
    for (int a = 0; a < S.n_acc; ++a) {
      const DevAccess& A = accs[S.acc0 + a];
      const DevArray& arr = arrays[A.array];
      bool sure = ph_ok, dims32 = true;   // every check decided; every index in 32 bits
      for (int d = 0; d < A.ndims; ++d) {
        const Range r = range(A.row0 + d);
        sure = sure && r.inside(0, arr.ext[d]);
        dims32 = dims32 && r.narrow();
      }
      if (sure && A.key_idx < 0) continue;   // an array never written, always in bounds: counted below
      o << in2 << "{\n";
      const std::string in3 = in2 + "  ";
      for (int d = 0; d < A.ndims; ++d)
        o << in3 << "const " << row_type(A.row0 + d) << " v" << d << " = " << row(A.row0 + d) << ";\n";
      if (!sure) {
        o << in3 << "unsigned dc = 0xFFFFFFFFu;\n";
        if (!ph_ok) o << in3 << "if (ph < 0 || ph >= " << lit(h.n_phases * h.n_wphases) << ") dc = 0u;\n" << in3 << "else\n";
        for (int d = 0; d < A.ndims; ++d) {
          const Range r = range(A.row0 + d);
          if (r.inside(0, arr.ext[d])) continue;
          if (r.narrow() && arr.ext[d] < (1ll << 31))
            o << in3 << "if ((unsigned)v" << d << " >= " << arr.ext[d] << "u) dc = " << d + 1 << "u;\n" << in3 << "else\n";
          else
            o << in3 << "if (v" << d << " < 0 || v" << d << " >= " << lit(arr.ext[d]) << ") dc = " << d + 1 << "u;\n"
              << in3 << "else\n";
        }
        o << in3 << "{ }\n";
      }
      // the linear cell, row-major (32-bit where every cell number is)
      const bool c32 = cl32 && dims32;
      std::string e = c32 ? std::to_string((uint32_t)arr.base) + "u" : ulit(arr.base);
      for (int d = 0; d < A.ndims; ++d) {
        int64_t stride = 1;
        for (int d2 = d + 1; d2 < A.ndims; ++d2) stride *= arr.ext[d2];
        if (c32) e += " + (unsigned)v" + std::to_string(d) + " * " + std::to_string((uint32_t)stride) + "u";
        else e += " + (unsigned long long)((long long)v" + std::to_string(d) + " * " + lit(stride) + ")";
      }
      if (arr.shared) e += c32 ? " + (unsigned)b * " + std::to_string((uint32_t)arr.cells) + "u" : " + b * " + ulit(arr.cells);
      const std::string cell_t = c32 ? "unsigned" : "unsigned long long";
      // the key's fields below the cell in one 32-bit word where they fit
      const bool low32 = h.cell_shift <= 32 && ph_ok && !fine;
      auto make = [&](const std::string& cl) {
        const std::string c64 = "((unsigned long long)" + cl + " << " + std::to_string(h.cell_shift) + ")";
        if (low32)
          return c64 + " | (((unsigned)ph << " + std::to_string(h.phase_shift & 31u) + ") | (unsigned)low | " +
                 std::to_string(A.kind) + "u)";
        return c64 + " | ((unsigned long long)ph << " + std::to_string(h.phase_shift) + ") | low | " +
               ulit((uint64_t)A.kind);
      };
      const uint64_t pack = ((unsigned long long)s << 51) | ((unsigned long long)a << 45);
      const std::string report = "atomicMin(oob, " + ulit(pack) + " | ((g & 0x3FFFFFFFFFFull) << 3) | dc);";
      if (chunked) {
        // the whole cell goes to the sink beside the key, whose cell field may not hold it
        o << in3 << "unsigned long long key = ~0ull, cl = ~0ull;\n";
        if (!sure) o << in3 << "if (dc != 0xFFFFFFFFu) " << report << "\n" << in3 << "else\n";
        o << in3 << "{ cl = " << e << "; key = " << make("cl") << "; }\n";
        if (A.key_idx < 0) o << in3 << "(void)key; (void)cl;\n";
        else if (repeats[a])
          // the same instance again: the same cell (a wide model's key may not hold all of it)
          // and the same fields below it, the interval among them, which an outer loop may move
          o << in3 << "if (cl != lastc" << a << " || key != last" << a << ") chunk_put(a, key, cl, sweep);\n"
            << in3 << "lastc" << a << " = cl;\n" << in3 << "last" << a << " = key;\n";
        else o << in3 << "chunk_put(a, key, cl, sweep);\n";
        o << in2 << "}\n";
        continue;
      }
      if (A.key_idx < 0) {
        o << in3 << "if (dc != 0xFFFFFFFFu) " << report << "\n" << in2 << "}\n";   // checked, no key
        continue;
      }
      o << in3 << "unsigned long long key = ~0ull;\n";
      if (!sure) o << in3 << "if (dc != 0xFFFFFFFFu) " << report << "\n" << in3 << "else\n";
      o << in3 << "{\n" << in3 << "  const " << cell_t << " cl = " << e << ";\n";
      o << in3 << "  if (!part_check || (cl >= cell_lo && cl < cell_hi && ((cl * " << ulit(kCellHashMul)
        << ") & part_mask) == part_val)) key = " << make("cl") << ";\n";
      if (repeats[a]) {
        o << in3 << "  const unsigned long long now = key;\n";
        o << in3 << "  if (!all_points && key == last" << a << ") key = ~0ull;\n" << in3 << "  last" << a << " = now;\n";
      }
      // the pass-A histogram of the bucket path, counted as the keys are written
      o << in3 << "  if (hist_a != nullptr && key != ~0ull) atomicAdd(&hA["
        << (c32 ? "((cl * " + std::to_string((uint32_t)kCellHashMul) + "u) & (unsigned)hmask) >> hsh"
                : "(unsigned)(((cl * " + ulit(kCellHashMul) + ") & hmask) >> hsh)")
        << "], 1u);\n" << in3 << "}\n";
      if (S.dense) o << in3 << "out[" << ulit((uint64_t)A.key_idx * T) << "] = key;\n";
      else if (pairs) o << in3 << "k" << A.key_idx << " = key;\n";
      else o << in3 << "out[" << A.key_idx << "] = key;\n";
      o << in2 << "}\n";
    }
    if (!distinct) o << in2 << "cnt += " << S.n_acc << ";\n";
    else
      o << in2 << "cnt += " << S.n_acc << "u * (" << (chunked ? "" : "all_points ? 1u : ") << "(unsigned)pts" << s
        << "[p].y);\n";
    if (pairs) {
      o << in2 << "if (((unsigned long long)out & 15ull) == 0ull) {\n";
      for (int kq = 0; kq + 1 < S.n_key; kq += 2)
        o << in2 << "  *reinterpret_cast<ulonglong2*>(out + " << kq << ") = make_ulonglong2(k" << kq << ", k" << kq + 1 << ");\n";
      if (S.n_key & 1) o << in2 << "  out[" << S.n_key - 1 << "] = k" << S.n_key - 1 << ";\n";
      o << in2 << "} else {\n";
      for (int kq = 0; kq < S.n_key; ++kq) o << in2 << "  out[" << kq << "] = k" << kq << ";\n";
      o << in2 << "}\n";
    }
    if (!S.dense && !chunked) o << in2 << "out += " << S.n_key << ";\n";
    o << ind << "}";
    if (chunked) {
      o << "\n";
    } else if (S.dense) {
      o << " else {\n";
      for (int kq = 0; kq < S.n_key; ++kq) o << in2 << "out[" << ulit((uint64_t)kq * T) << "] = ~0ull;\n";
      o << ind << "}\n";
      o << ind << "out += " << ulit((uint64_t)S.n_key * T) << ";\n";
    } else {
      o << "\n";
    }
    for (int l = distinct ? 0 : S.n_loops - 1; l >= 0; --l) {
      ind.resize(ind.size() - 2);
      o << ind << "}\n";
    }
    o << "    } break;\n";
  }
  uint64_t h_dense() const { return m.host.dense_slots; }

  std::string source() {
    const DevModel& h = m.host;
    o << "// generated expansion kernel\n";
    o << "__device__ __forceinline__ long long fdiv_c(long long a, long long d) {\n"
         "  return a >= 0 ? a / d : -1 - (-(a + 1)) / d;\n}\n";
    o << "__device__ __forceinline__ long long mod_c(long long a, long long d) { return a - fdiv_c(a, d) * d; }\n";
    o << "__device__ __forceinline__ int fdiv_n(int a, int d) {\n"
         "  return a >= 0 ? (int)((unsigned)a / (unsigned)d) : -1 - (int)((unsigned)(-(a + 1)) / (unsigned)d);\n}\n"
         "__device__ __forceinline__ int mod_n(int a, int d) { return a - fdiv_n(a, d) * d; }\n";
    o << "__device__ __forceinline__ long long tload_c(const long long* t, unsigned long long off, "
         "unsigned long long len, long long i) {\n"
         "  return (i < 0 || (unsigned long long)i >= len) ? 0LL : t[off + (unsigned long long)i];\n}\n";
    // the distinct points of a statement: (flat iteration number, points it stands for)
    for (uint32_t s = 0; s < h.n_stmts; ++s) {
      const DistinctPoints& p = dp[s];
      if (p.point.empty()) continue;
      o << "__constant__ ushort2 pts" << s << "[" << p.point.size() << "] = {";
      for (size_t i = 0; i < p.point.size(); ++i) o << "{" << p.point[i] << "," << p.times[i] << "},";
      o << "};\n";
    }
    if (chunked) {
      // same layout as rc::ChunkJitArgs
      o << "struct ChunkJitArgs {\n"
           "  unsigned long long* oob; unsigned long long* inst; const long long* tdata;\n"
           "  int mode; int pad;\n"
           "  unsigned long long* counts; unsigned long long lo, span; unsigned bshift, cell_shift;\n"
           "  unsigned long long* keys; const unsigned* chunk_of; const unsigned long long* c_lo;\n"
           "  const unsigned long long* c_base; const unsigned long long* c_end; unsigned long long* c_ctr;\n"
           "  unsigned long long b0, n_buckets, low_mask; unsigned* err; unsigned k0, nk;\n};\n";
      // mode 0: count keys per bucket; mode 1: route keys to their chunk's segment.
      // A wave of at most kRouteChunks chunks is routed in two sweeps over the
      // block's points: the first counts the block's keys per chunk (so that a
      // block reserves once per chunk instead of every warp for every key: those
      // atomics on a few addresses took most of the pass), the second places them.
      o << "__shared__ unsigned sC[" << kRouteChunks << "];\n"
           "__shared__ unsigned long long sB[" << kRouteChunks << "];\n"
           "__device__ __forceinline__ void chunk_put(const ChunkJitArgs& a, unsigned long long key, "
           "unsigned long long cell, int sweep) {\n"
           "  if (key == ~0ull) return;\n"
           "  const unsigned long long rel = cell - a.lo;\n"
           "  if (rel >= a.span) return;\n"
           "  const unsigned long long bucket = rel >> a.bshift;\n"
           "  const unsigned lane = threadIdx.x & 31u;\n"
           "  if (a.mode == 0) {\n"
           "    const unsigned act = __activemask();\n"
           "    const int leader = __ffs(act) - 1;\n"
           "    const unsigned long long b0 = __shfl_sync(act, bucket, leader);\n"
           "    if (__all_sync(act, bucket == b0)) {\n"
           "      if ((int)lane == leader) atomicAdd(a.counts + b0, (unsigned long long)__popc(act));\n"
           "    } else {\n"
           "      atomicAdd(a.counts + bucket, 1ull);\n"
           "    }\n"
           "    return;\n"
           "  }\n"
           "  const unsigned long long bk = bucket - a.b0;\n"
           "  if (bk >= a.n_buckets) return;\n"
           "  const unsigned k = a.chunk_of[bk];\n"
           "  if (k == 0xffffffffu) return;\n"
           "  const unsigned long long out = ((cell - a.c_lo[k]) << a.cell_shift) | (key & a.low_mask);\n"
           "  // one reservation per chunk among the lanes here together (a warp's keys lie in\n"
           "  // few chunks, and all warps add to the same counters)\n"
           "  const unsigned act = __activemask();\n"
           "  const unsigned peers = __match_any_sync(act, k);\n"
           "  const int leader = __ffs(peers) - 1;\n"
           "  unsigned long long pos = 0;\n"
           "  const unsigned np = __popc(peers);\n"
           "  if (sweep == 0) {\n"
           "    if ((int)lane == leader) atomicAdd(&sC[k - a.k0], np);\n"
           "    return;\n"
           "  }\n"
           "  if ((int)lane == leader)\n"
           "    pos = sweep == 1 ? sB[k - a.k0] + atomicAdd(&sC[k - a.k0], np)\n"
           "                     : atomicAdd(a.c_ctr + k, (unsigned long long)np);\n"
           "  pos = __shfl_sync(peers, pos, leader) + __popc(peers & ((1u << lane) - 1u));\n"
           "  pos += a.c_base[k];\n"
           "  if (pos < a.c_end[k]) a.keys[pos] = out;\n"
           "  else atomicOr(a.err, " + std::to_string((unsigned)kErrChunkOverflow) + "u);\n"
           "}\n";
      o << "extern \"C\" __global__ void __launch_bounds__(128) rc_chunk_jit(const ChunkJitArgs a) {\n";
      o << "  unsigned long long* oob = a.oob;\n  const long long* tdata = a.tdata;\n  (void)tdata;\n";
    } else {
      // hist_a: the bucket path's pass-A digit counts (null: not counted here).  The
      // blocks of launch position i are [blk[i].x, blk[i + 1].x), each of blk[i].z
      // consecutive 128-thread units of statement blk[i].y.
      o << "__constant__ uint3 blk[" << h.n_stmts + 1 << "] = {";
      for (uint32_t i = 0; i < h.n_stmts; ++i) o << "{" << blk_first[i] << "," << blk_stmt[i] << "," << blk_units[i] << "},";
      o << "{" << blocks << ",0,1}};\n";
      o << "extern \"C\" __global__ void __launch_bounds__(128) rc_expand_jit(unsigned long long* __restrict__ keys, "
           "unsigned long long* oob, unsigned long long* inst, const unsigned long long* __restrict__ unit_offset, "
           "unsigned long long cell_lo, unsigned long long cell_hi, unsigned long long part_mask, unsigned long long part_val, "
           "const long long* __restrict__ tdata, "
           "unsigned long long* hist_a, unsigned long long hmask, unsigned hsh, unsigned hbins, unsigned all_points) {\n";
      // a partial check (cell range or hash part); uniform
      o << "  const bool part_check = cell_lo != 0ull || cell_hi != ~0ull || part_mask != 0ull;\n  (void)part_check;\n";
      o << "  __shared__ unsigned hA[" << kBucketMaxHistBins << "];\n";
      o << "  if (hist_a != nullptr) {\n"
           "    for (unsigned i = threadIdx.x; i < hbins; i += 128u) hA[i] = 0u;\n"
           "    __syncthreads();\n  }\n";
    }
    o << "  unsigned long long cnt = 0;\n";
    if (chunked)
      // sweep 0 counts, 1 places from the block's reservations, 2 places one by one (or mode 0)
      o << "  const bool two = a.mode == 1 && a.nk != 0u;\n"
           "  for (int sweep = two ? 0 : 2; sweep != 3; sweep = sweep == 0 ? 1 : 3) {\n"
           "  if (two) {\n"
           "    __syncthreads();\n"
           "    for (unsigned k = threadIdx.x; k < a.nk; k += 128u) {\n"
           "      if (sweep == 1) {\n"
           "        const unsigned n = sC[k];\n"
           "        if (n) sB[k] = atomicAdd(a.c_ctr + a.k0 + k, (unsigned long long)n);\n"
           "      }\n"
           "      sC[k] = 0u;\n"
           "    }\n"
           "    __syncthreads();\n"
           "  }\n"
           "  if (sweep == 1) cnt = 0;\n";
    if (!chunked)
      o << "  unsigned bi = 0;\n  for (unsigned hi = " << h.n_stmts << "u; hi - bi > 1u;) {\n"
           "    const unsigned mid = (bi + hi) >> 1;\n"
           "    if (blk[mid].x <= blockIdx.x) bi = mid; else hi = mid;\n  }\n"
           "  const unsigned stmt = blk[bi].y, units = blk[bi].z;\n"
           "  for (unsigned u = 0; u < units; ++u) {\n";
    o << "  const unsigned long long g = " << (chunked ? "(unsigned long long)blockIdx.x" :
                                                   "((unsigned long long)(blockIdx.x - blk[bi].x) * units + u)")
      << " * 128ull + threadIdx.x;\n";
    o << "  if (g < " << ulit(h.n_threads) << ") {\n";
    if (h.n_threads < (1ull << 31)) {
      // (every dimension is below 2^31 too)
      o << "    const unsigned g32 = (unsigned)g, b32 = g32 / " << h.bs << "u, t = g32 - b32 * " << h.bs << "u;\n";
      o << "    const int tx = t % " << h.block[0] << "u, ty = (t / " << h.block[0] << "u) % " << h.block[1]
        << "u, tz = t / " << h.block[0] * h.block[1] << "u;\n";
      o << "    const int bx = b32 % " << h.grid[0] << "u, by = (b32 / " << h.grid[0] << "u) % " << h.grid[1]
        << "u, bz = b32 / " << h.grid[0] * h.grid[1] << "u;\n";
      o << "    const unsigned long long b = b32;\n";
    } else {
      o << "    const unsigned long long b = g / " << ulit(h.bs) << ";\n";
      o << "    const unsigned t = (unsigned)(g - b * " << ulit(h.bs) << ");\n";
      o << "    const long long tx = t % " << h.block[0] << "u, ty = (t / " << h.block[0] << "u) % " << h.block[1]
        << "u, tz = t / " << (uint64_t)h.block[0] * h.block[1] << "u;\n";
      o << "    const long long bx = (long long)(b % " << ulit(h.grid[0]) << "), by = (long long)((b / " << ulit(h.grid[0])
        << ") % " << ulit(h.grid[1]) << "), bz = (long long)(b / " << ulit((uint64_t)h.grid[0] * h.grid[1]) << ");\n";
    }
    o << "    (void)tx; (void)ty; (void)tz; (void)bx; (void)by; (void)bz; (void)b;\n";
    o << "    const unsigned long long low = (b << " << h.block_shift << ") | ((unsigned long long)t << "
      << h.thread_shift << ");\n    (void)low;\n";
    o << "    switch (" << (chunked ? "blockIdx.y" : "stmt") << ") {\n";
    for (uint32_t s = 0; s < h.n_stmts; ++s) emit_stmt(s);
    o << "    default: break;\n    }\n  }\n";
    o << "  }\n";
    o << "  for (int d = 16; d > 0; d >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, d);\n";
    o << "  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(" << (chunked ? "a.inst" : "inst") << ", cnt);\n";
    if (!chunked)
      o << "  if (hist_a != nullptr) {\n"
           "    __syncthreads();\n"
           "    for (unsigned i = threadIdx.x; i < hbins; i += 128u)\n"
           "      if (hA[i]) atomicAdd(&hist_a[i], (unsigned long long)hA[i]);\n  }\n";
    o << "}\n";
    return o.str();
  }
};

}  // namespace

std::string jit_expand_source(const Model& m) {
  Gen g(m);
  return g.source();
}

std::string jit_chunk_source(const Model& m) {
  Gen g(m);
  g.chunked = true;
  return g.source();
}

namespace {

// Compile `src` for the current device (or fetch it from the cache) and return
// its kernel `name`, or null if NVRTC, the driver or the compile fails.
void* jit_compile(const std::string& src, const char* name) {
  std::lock_guard<std::mutex> lk(g_jit_mu);
  Nvrtc& nv = nvrtc();
  Driver& dr = driver();
  if (!nv.ok || !dr.ok) return nullptr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  const std::string key = std::to_string(dev) + "\n" + name + "\n" + src;
  auto it = g_cache.find(key);
  if (it != g_cache.end()) return it->second;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return nullptr;
  const std::string arch = "--gpu-architecture=sm_" + std::to_string(prop.major) + std::to_string(prop.minor) + "a";
  nvrtcProgram prog;
  if (nv.create(&prog, src.c_str(), "rc_expand_jit.cu", 0, nullptr, nullptr) != NVRTC_SUCCESS) return nullptr;
  const char* opts[] = {arch.c_str(), "--std=c++17"};
  bool ok = nv.compile(prog, 2, opts) == NVRTC_SUCCESS;
  std::vector<char> cubin;
  if (ok) {
    size_t n = 0;
    ok = nv.cubin_size(prog, &n) == NVRTC_SUCCESS && n > 0;
    if (ok) {
      cubin.resize(n);
      ok = nv.cubin(prog, cubin.data()) == NVRTC_SUCCESS;
    }
  }
  nv.destroy(&prog);
  if (!ok) return nullptr;
  CUmodule mod;
  CUfunction fn;
  if (dr.load(&mod, cubin.data()) != CUDA_SUCCESS) return nullptr;
  if (dr.get(&fn, mod, name) != CUDA_SUCCESS) return nullptr;
  g_cache[key] = reinterpret_cast<void*>(fn);
  return reinterpret_cast<void*>(fn);
}

// RC_JIT=0 disables generated kernels, RC_JIT=1 forces them for every model
bool jit_wanted(const Model& m) {
  const char* env = std::getenv("RC_JIT");
  if (env && env[0] == '0') return false;
  const bool force = env && env[0] == '1';
  if (!force && m.key_slots < kJitMinKeys) return false;
  return m.host.n_stmts != 0 && m.host.n_threads != 0;
}

}  // namespace

// The model's generated kernel: the slot kernel of the ordinary check, or for
// a wide model the count / route kernel of its chunked checks.  Returns false
// (the interpreted kernels stay in use) if NVRTC, the driver or the compile fails.
bool jit_expand_build(Model* m) {
  if (!jit_wanted(*m)) return false;
  if (m->wide) {
    m->jit_chunk_fn = jit_compile(jit_chunk_source(*m), "rc_chunk_jit");
    return m->jit_chunk_fn != nullptr;
  }
  Gen g(*m);
  m->jit_fn = jit_compile(g.source(), "rc_expand_jit");
  if (m->jit_fn) {
    m->check_slots = g.check_dense + m->host.general_slots;
    m->jit_blocks = (uint32_t)g.blocks;
  }
  return m->jit_fn != nullptr;
}

cudaError_t jit_chunk_launch(const Model& m, const ChunkJitArgs& a, cudaStream_t st) {
  Driver& dr = driver();
  CUfunction fn = reinterpret_cast<CUfunction>(m.jit_chunk_fn);
  ChunkJitArgs args = a;
  if (args.nk > kRouteChunks) args.nk = 0;   // (too many for the block's counters)
  void* params[] = {&args};
  const unsigned gx = (unsigned)((m.host.n_threads + 127) / 128);
  const CUresult r = dr.launch(fn, gx, m.host.n_stmts, 1, 128, 1, 1, 0, reinterpret_cast<CUstream>(st), params, nullptr);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorLaunchFailure;
}

cudaError_t jit_expand_launch(const Model& m, uint64_t* keys, DevResult* res, cudaStream_t st, const CellFilter& cf,
                              const ExpandHist* eh, bool all_points) {
  Driver& dr = driver();
  CUfunction fn = reinterpret_cast<CUfunction>(m.jit_fn);
  unsigned long long* oob = &res->oob_code;
  unsigned long long* inst = &res->instances;
  const uint64_t* uo = m.host.unit_offset;
  unsigned long long lo = cf.lo, hi = cf.hi;
  unsigned long long pmask = cf.pmask, pval = cf.pval;
  const int64_t* td = m.host.tdata;
  unsigned long long* hist = eh ? eh->hist : nullptr;
  unsigned long long hmask = eh ? eh->cmask : 0ull;
  unsigned hsh = eh ? eh->shift : 0u, hbins = eh ? eh->bins : 0u;
  if (hbins > (unsigned)kBucketMaxHistBins) return cudaErrorInvalidValue;
  unsigned all32 = all_points ? 1u : 0u;
  void* params[] = {&keys, &oob, &inst, &uo, &lo, &hi, &pmask, &pval, &td, &hist, &hmask, &hsh, &hbins, &all32};
  const CUresult r = dr.launch(fn, m.jit_blocks, 1, 1, 128, 1, 1, 0, reinterpret_cast<CUstream>(st), params, nullptr);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorLaunchFailure;
}

}  // namespace rc
