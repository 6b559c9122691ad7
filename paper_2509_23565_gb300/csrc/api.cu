// C-ABI entry points: handle management, slicing, level sums and the emulated
// DGEMM (arXiv 2509.23565, Section 2, Eq. 1-4; Section 4, Eq. 7).
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include <mutex>
#include <set>
#include <utility>

#include <cudaTypedefs.h>

#include "handle.h"

namespace emul {

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }
inline long kpad_of(int k) { return (static_cast<long>(k) + 7) / 8 * 8; }

// The slice pairs kept: p <= sa slices of A, q <= sb slices of B (sa = sb = s
// for the method itself; unequal counts keep a subset of the pairs of the
// max(sa, sb)-slice split, whose leading slices are those of a shorter split).
struct PairSet {
  int sa, sb;
  int lo(int L) const { return L - sb > 1 ? L - sb : 1; }          // first p of level L
  int hi(int L) const { return L - 1 < sa ? L - 1 : sa; }          // last p of level L
  int count(int L) const { return hi(L) >= lo(L) ? hi(L) - lo(L) + 1 : 0; }
  // highest slice index of A or B a pair of level L uses
  int planes(int L) const { return hi(L) > L - lo(L) ? hi(L) : L - lo(L); }
};

// Sum over the levels L = 2..last of n_L 2^(7(last-L)) times 127^2: the
// worst-case magnitude per unit of k of T = sum_L I_L 2^(7(last-L)) (the
// wide variant's state after all its jobs, last = t).
long double exact_sum_bound_per_k(const PairSet& ps, int last) {
  long double acc = 0.0L;
  for (int L = 2; L <= last; ++L) acc = acc * 128.0L + ps.count(L);
  return acc * 127.0L * 127.0L;
}

// K chunks per accumulator job of n slice pairs under the exactness budget.
int seg_chunks(int n) { return n > 0 ? kExactBudget / (n * kBK) : 0; }

struct Job {
  int L, pb, pe, c0, c1;
  bool fin;   // completes and rounds the sum
};

Job make_job(const PairSet& ps, int L, int c0, int c1, bool fin) {
  return Job{L, ps.lo(L), ps.hi(L), c0, c1, fin};
}

// A sweep of jobs over one K range, in the order given.
void push_sweep(std::vector<Sweep>& out, const std::vector<Job>& jobs) {
  Sweep sw{};
  sw.k0c = static_cast<int16_t>(jobs[0].c0);
  sw.k1c = static_cast<int16_t>(jobs[0].c1);
  sw.njobs = static_cast<int8_t>(jobs.size());
  int np = 0;
  for (size_t j = 0; j < jobs.size(); ++j) {
    const Job& q = jobs[j];
    sw.L[j] = static_cast<int8_t>(q.L);
    sw.pp[j] = static_cast<uint8_t>(q.pb | (q.pe << 4));
    if (q.fin) sw.final_mask = static_cast<int8_t>(sw.final_mask | (1 << j));
    const int pj = q.pe > q.L - q.pb ? q.pe : q.L - q.pb;
    np = np > pj ? np : pj;
  }
  sw.nplanes = static_cast<int8_t>(np);
  out.push_back(sw);
}

// Banded schedule: the levels are covered by bands of one level or of two
// adjacent levels.  A two-level band (L, L+1) shares every staged chunk
// between both levels (the planes of L are a subset of those of L+1); a band
// that does not fit the exactness budget over the whole K runs in K groups.  The bands minimise the staged planes per K chunk (dynamic
// programme over the levels).  The epilogue adds every job's level sum with
// its weight, R += I_L 2^(7(t-L)), so the jobs may come in any order: the
// bands are issued from the highest level down, each tile starting with its
// longest MMA jobs (they keep the tensor cores busy while the epilogue rounds
// the previous tile) and ending, in the 64-bit variant, with level 2 as one
// single job: the final job, whose term 2^(7(t-2)) I_2 is added and rounded
// last.
bool build_banded(const PairSet& ps, int t, int nch, bool wide, std::vector<Sweep>& out) {
  out.clear();
  const int kInf = 1 << 28;
  std::vector<int> cost(t + 3, 0), choice(t + 3, 0);
  auto groups = [&](int seg) { return (nch + seg - 1) / seg; };
  for (int L = t; L >= 2; --L) {
    cost[L] = kInf;
    const int sg1 = seg_chunks(ps.count(L));
    // the final job (level 2 in the 64-bit variant) must be one job alone
    if (sg1 >= 1 && cost[L + 1] < kInf && (wide || L > 2 || groups(sg1) == 1)) {
      cost[L] = ps.planes(L) + cost[L + 1];
      choice[L] = 1;
    }
    if (L + 1 <= t && cost[L + 2] < kInf && (wide || L > 2)) {
      const int a = seg_chunks(ps.count(L)), b = seg_chunks(ps.count(L + 1));
      const int sg2 = a < b ? a : b;
      if (sg2 >= 1 && ps.planes(L + 1) + cost[L + 2] < cost[L]) {
        cost[L] = ps.planes(L + 1) + cost[L + 2];
        choice[L] = 2;
      }
    }
  }
  if (cost[2] >= kInf) return false;
  std::vector<std::pair<int, int>> bands;   // (first level, levels)
  for (int L = 2; L <= t; L += choice[L]) bands.push_back({L, choice[L]});
  for (auto it = bands.rbegin(); it != bands.rend(); ++it) {
    const int L = it->first;
    if (it->second == 1) {
      const int G = groups(seg_chunks(ps.count(L)));
      const int size = (nch + G - 1) / G;
      for (int g = 0; g < G; ++g) {
        const int c0 = g * size, c1 = c0 + size < nch ? c0 + size : nch;
        push_sweep(out, {make_job(ps, L, c0, c1, !wide && L == 2)});
      }
    } else {
      const int a = seg_chunks(ps.count(L)), b = seg_chunks(ps.count(L + 1));
      const int G = groups(a < b ? a : b);
      const int size = (nch + G - 1) / G;
      for (int g = 0; g < G; ++g) {
        const int c0 = g * size, c1 = c0 + size < nch ? c0 + size : nch;
        push_sweep(out, {make_job(ps, L, c0, c1, false), make_job(ps, L + 1, c0, c1, false)});
      }
    }
  }
  return true;
}

// Level-ordered schedule, the fallback: from the highest level down, a level
// whose n_L pairs fit the budget over the whole K is one job; otherwise its
// pairs are split into groups that fit (64-bit variant) or its K range into
// segments (128-bit variant).  Consecutive jobs of one K range share a sweep.
// In the 64-bit variant level 2 comes last as one job (the final job).
bool build_levelwise(const PairSet& ps, int t, int nch, bool wide, std::vector<Sweep>& out) {
  out.clear();
  std::vector<Job> jobs;
  const int kc = nch * kBK;
  for (int L = t; L >= 2; --L) {
    const int pb = ps.lo(L);
    const int pe = ps.hi(L);
    const int n = pe - pb + 1;
    const bool fin = !wide && L == 2;
    if (n * kc <= kExactBudget) {
      jobs.push_back(Job{L, pb, pe, 0, nch, fin});
    } else if (!wide) {
      if (fin) return false;
      const int per = kExactBudget / kc;          // pairs per job
      if (per < 1) return false;
      for (int p = pb; p <= pe; p += per)
        jobs.push_back(Job{L, p, p + per - 1 < pe ? p + per - 1 : pe, 0, nch, false});
    } else {
      int cm = kExactBudget / (kBK * n);
      if (cm < 1) cm = 1;
      for (int c0 = 0; c0 < nch; c0 += cm) jobs.push_back(Job{L, pb, pe, c0, c0 + cm < nch ? c0 + cm : nch, false});
    }
  }
  for (size_t i = 0; i < jobs.size();) {
    // the final job stays alone in its sweep
    if (i + 1 < jobs.size() && !jobs[i + 1].fin && jobs[i + 1].c0 == jobs[i].c0 &&
        jobs[i + 1].c1 == jobs[i].c1) {
      push_sweep(out, {jobs[i], jobs[i + 1]});
      i += 2;
    } else {
      push_sweep(out, {jobs[i]});
      i += 1;
    }
  }
  return true;
}

// K chunks per stage: a stage holds s tiles of A and s of B, so a sweep that
// stages fewer planes packs several chunks into one stage (one barrier phase
// for more bytes; the copy engine's rate grows with the bytes per phase).
void set_chunks_per_stage(int s, std::vector<Sweep>& out) {
  for (Sweep& w : out) {
    const int nc = w.k1c - w.k0c;
    const int kmax = w.nplanes > 0 && s / w.nplanes > 1 ? s / w.nplanes : 1;
    const int nst = (nc + kmax - 1) / kmax;
    w.kcs = static_cast<int8_t>(nst > 0 ? (nc + nst - 1) / nst : 1);
  }
}

// Schedule of the one-CTA variants for the levels 2..t (t = 0: the default
// threshold s + 1 of the method): the banded one when it exists, else the
// level-ordered one.  The level-sum mode drains every job the same way and uses the
// same schedule.
// sa, sb: slices of A and of B whose pairs are kept (0: s); s = max(sa, sb)
// is the split both operands get and the number of planes a stage holds.
bool build_schedule(int s, int nch, bool wide, std::vector<Sweep>& out, int t = 0, int sa = 0, int sb = 0) {
  if (sa == 0) sa = s;
  if (sb == 0) sb = s;
  if (t == 0) t = s + 1;
  if (t < 2 || t > sa + sb || (sa > sb ? sa : sb) != s) return false;
  const PairSet ps{sa, sb};
  if (!build_banded(ps, t, nch, wide, out) && !build_levelwise(ps, t, nch, wide, out)) return false;
  set_chunks_per_stage(s, out);
  return !out.empty();
}

// Schedule of the CTA-pair kernel: bands of up to four adjacent levels share every
// staged chunk.  A sweep may hold as many jobs as there are slots: the two issuing
// warps take its jobs alternately, each waits for a job's slot only before that
// job's own first MMA, and the slot's job before it belongs to an earlier sweep,
// whose MMAs are all issued; both warps commit every stage, so a stage is freed also
// when one of them has no job in the sweep.  At s = 7 the bands {8,7,6,5} and {4,3,2} stage 10 planes per chunk,
// bands of two levels 16, and the staged bytes set the pace (12 KB per plane
// and chunk against 64 cycles per MMA: with 16 planes the copies alone need
// 1.0 of the MMAs' time at 54 bytes per clock, with 10 planes 0.65).  The bands
// minimise the staged planes (dynamic programme over the levels), then the
// jobs; they are issued from the highest level down, and so are the jobs of a
// sweep, each sweep's longest MMA job first.  A band runs in K groups that
// keep every job inside the exactness budget; the last job of all, level 2's
// last group, completes the sum.
bool build_pair(const PairSet& ps, int t, int nch, std::vector<Sweep>& out) {
  out.clear();
  constexpr long kInf = 1l << 40;
  std::vector<long> cost(t + 6, kInf);
  std::vector<int> choice(t + 6, 0);
  cost[t + 1] = 0;
  auto seg_of = [&](int L, int b) {   // chunks per group of the band L .. L+b-1
    int seg = nch;
    for (int l = L; l < L + b; ++l) {
      const int n = ps.count(l);
      if (n > 0 && seg_chunks(n) < seg) seg = seg_chunks(n);
    }
    return seg;
  };
  auto planes_of = [&](int L, int b) {
    int np = 0;
    for (int l = L; l < L + b; ++l) np = ps.planes(l) > np ? ps.planes(l) : np;
    return np;
  };
  for (int L = t; L >= 2; --L)
    for (int b = 1; b <= kSweepJobs && L + b <= t + 1; ++b) {
      const int seg = seg_of(L, b);
      if (seg < 1 || cost[L + b] >= kInf) continue;
      const long jobs = static_cast<long>((nch + seg - 1) / seg) * b;
      const long c = cost[L + b] + static_cast<long>(planes_of(L, b)) * nch * 64 + jobs;
      if (c < cost[L]) {
        cost[L] = c;
        choice[L] = b;
      }
    }
  if (cost[2] >= kInf) return false;
  std::vector<std::pair<int, int>> bands;
  for (int L = 2; L <= t; L += choice[L]) bands.push_back({L, choice[L]});
  for (auto it = bands.rbegin(); it != bands.rend(); ++it) {
    const int seg = seg_of(it->first, it->second);
    const int G = (nch + seg - 1) / seg, size = (nch + G - 1) / G;
    for (int c0 = 0; c0 < nch; c0 += size) {
      const int c1 = c0 + size < nch ? c0 + size : nch;
      std::vector<Job> jobs;
      for (int L = it->first + it->second - 1; L >= it->first; --L)
        if (ps.count(L) > 0) jobs.push_back(make_job(ps, L, c0, c1, L == 2 && c1 == nch));
      push_sweep(out, jobs);
    }
  }
  return true;
}

// Which CTA-pair variant sums the levels 2..t exactly: 0 none, 1 the 64-bit
// state, 2 the 64-bit state with the 16 low bits put aside.  R is the state
// before the final job's term; it must stay below 2^61 (the term is tested in
// the kernel).  The low bits are put aside after the first band: what follows
// has to weigh at least 2^16 (levels t-3 and down: 2^21 after a band of three),
// and what came before has to fit in 64 bits.
int pair_plan(int s, int t, int nch, int sa, int sb, std::vector<Sweep>* sweeps, int* stash_job) {
  const PairSet ps{sa, sb};
  std::vector<Sweep> sw;
  if (!build_pair(ps, t, nch, sw)) return 0;
  set_chunks_per_stage(s, sw);
  const long double kk = static_cast<long double>(nch * kBK) * 127.0L * 127.0L;
  const long double lim = 2305843009213693952.0L;   // 2^61
  // everything but the final job's term, which is the last group of level 2
  const Sweep& last = sw.back();
  long double all = 0.0L;
  for (int L = 2; L <= t; ++L) all += ps.count(L) * kk * powl(2.0L, 7.0L * (t - L));
  const long double fin =
      static_cast<long double>((last.k1c - last.k0c) * kBK) * 127.0L * 127.0L * powl(2.0L, 7.0L * (t - 2));
  const long double r = all - fin;
  int kind = 0, stash = -1;
  if (r < lim) {
    kind = 1;
  } else {
    // jobs of the first band
    const int top = sw[0].L[0], bottom = sw[0].L[sw[0].njobs - 1];
    int jobs = 0;
    size_t i = 0;
    for (; i < sw.size() && sw[i].L[0] == top; ++i) jobs += sw[i].njobs;
    long double before = 0.0L;
    for (int L = bottom; L <= t; ++L) before += ps.count(L) * kk * powl(2.0L, 7.0L * (t - L));
    if (i < sw.size() && bottom > 2 && 7 * (t - bottom + 1) >= 16 && before < lim && r / 65536.0L < lim &&
        fin / 65536.0L < 2.0L * lim) {
      kind = 2;
      stash = jobs - 1;
    }
  }
  if (kind && sweeps) {
    *sweeps = sw;
    *stash_job = stash;
  }
  return kind;
}

// The constants that the kernel's drains leave in the 64-bit state, negated:
// kMagicPair per unit of weight for two adjacent levels drained together,
// kMagicBits for a job drained alone, in the units of the state before and
// after the low bits were put aside.
DrainConstants drained_constants(const std::vector<Sweep>& sw, int t, int stash_job) {
  DrainConstants d{stash_job, 0, 0};
  uint64_t sum[2] = {0, 0};
  int jj = 0;
  for (const Sweep& w : sw)
    for (int j = 0; j < w.njobs;) {
      const bool after = stash_job >= 0 && jj > stash_job;
      const int units = after ? 16 : 0;
      const int d1 = j + 1 < w.njobs ? w.L[j + 1] - w.L[j] : 0;
      if ((d1 == 1 || d1 == -1) && !((w.final_mask >> j) & 1) && !((w.final_mask >> (j + 1)) & 1)) {
        const int L = w.L[j] > w.L[j + 1] ? w.L[j] : w.L[j + 1];
        sum[after] += static_cast<uint64_t>(static_cast<int64_t>(kMagicPair)) << (7 * (t - L) - units);
        j += 2;
        jj += 2;
      } else {
        sum[after] += static_cast<uint64_t>(kMagicBits) << (7 * (t - w.L[j]) - units);
        j += 1;
        jj += 1;
      }
    }
  d.r_init = static_cast<long long>(0 - sum[0]);
  d.r_init2 = static_cast<long long>(0 - sum[1]);
  return d;
}

// The narrow variant keeps the state R in int64 and completes T = R + I_2 2^(7(t-2))
// in its final job (in 64 bits when the warp's terms allow, else in 128): it
// needs level 2 in one job and the sum of the other levels inside int64.
bool narrow_ok(int s, int k, int t = 0, int sa = 0, int sb = 0) {
  if (sa == 0) sa = s;
  if (sb == 0) sb = s;
  if (t == 0) t = s + 1;
  if (s > 7) return false;
  const int nch = (k + kBK - 1) / kBK;
  std::vector<Sweep> tmp;
  if (!build_schedule(s, nch, false, tmp, t, sa, sb)) return false;
  // R, the sum of the levels 3..t with their weights, stays below 2^61, so
  // that R + I_2 2^(7(t-2)) fits in 64 bits whenever |I_2| 2^(7(t-2)) <= 2^62
  // (the epilogue's test; otherwise it adds the term in 128 bits).
  const PairSet ps{sa, sb};
  const long double kk = static_cast<long double>(nch * kBK);
  long double r = 0.0L;
  for (int L = 3; L <= t; ++L) r += ps.count(L) * 127.0L * 127.0L * kk * powl(2.0L, 7.0L * (t - L));
  return r < 2305843009213693952.0L;   // 2^61
}

// The wide variant's 128-bit exact sum T must stay below 2^126.
bool wide_ok(int s, int t, int k, int sa = 0, int sb = 0) {
  const int nch = (k + kBK - 1) / kBK;
  return exact_sum_bound_per_k(PairSet{sa ? sa : s, sb ? sb : s}, t) * static_cast<long double>(nch * kBK) < 8.5e37L;
}

int get_schedule(emul_handle_t h, int s, int t, int nch, bool wide, bool pair, Sweep** dptr, int* count,
                 DrainConstants* drains, int sa, int sb) {
  const uint64_t key = (static_cast<uint64_t>(pair) << 48) | (static_cast<uint64_t>(sa) << 40) |
                       (static_cast<uint64_t>(sb) << 32) | (static_cast<uint64_t>(s) << 24) |
                       (static_cast<uint64_t>(wide) << 23) | (static_cast<uint64_t>(t) << 13) |
                       static_cast<uint64_t>(nch);   // nch < 2^13 (k <= 65536)
  auto it = h->sched_cache.find(key);
  if (it != h->sched_cache.end()) {
    *dptr = it->second.sched;
    *count = it->second.nsweeps;
    *drains = it->second.drains;
    return EMUL_OK;
  }
  std::vector<Sweep> v;
  int stash = -1;
  if (pair ? pair_plan(s, t, nch, sa, sb, &v, &stash) == 0 : !build_schedule(s, nch, wide, v, t, sa, sb))
    return set_error(h, EMUL_INVALID_ARG, "no schedule for this slice count / k");
  const DrainConstants dc = drained_constants(v, t, stash);
  Sweep* d = nullptr;
  if (cudaMalloc(&d, v.size() * sizeof(Sweep)) != cudaSuccess)
    return set_error(h, EMUL_NO_WORKSPACE, "schedule allocation failed");
  if (cudaMemcpy(d, v.data(), v.size() * sizeof(Sweep), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaFree(d);
    return set_error(h, EMUL_CUDA_ERROR, "schedule upload failed");
  }
  h->sched_cache[key] = emul_handle_s::SchedEntry{d, static_cast<int>(v.size()), dc};
  *dptr = d;
  *count = static_cast<int>(v.size());
  *drains = dc;
  return EMUL_OK;
}

int encode_slices_map(emul_handle_t h, CUtensorMap* map, const uint16_t* base, int rows, int k, long kpad, int s,
                      int box_rows) {
  auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(h->encode_fn);
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(k), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(s)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(kpad) * 2, static_cast<cuuint64_t>(kpad) * 2 * rows};
  cuuint32_t box[3] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows), 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(h, EMUL_CUDA_ERROR, "cuTensorMapEncodeTiled failed");
  return EMUL_OK;
}

__global__ void scale_c_kernel(int m, int n, double alpha, double beta, double* C, long ldc) {
  const long total = static_cast<long>(m) * n;
  for (long i = blockIdx.x * static_cast<long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long>(gridDim.x) * blockDim.x) {
    const int r = static_cast<int>(i % m);
    const long c = i / m;
    double* p = C + r + c * ldc;
    const double ad = __dmul_rn(alpha, 0.0);
    *p = (beta == 0.0) ? ad : __dadd_rn(ad, __dmul_rn(beta, *p));
  }
}

__global__ void zero_levels_kernel(int m, int n, int planes, int32_t* lv, long ldl, long ldp) {
  const long total = static_cast<long>(m) * n * planes;
  for (long i = blockIdx.x * static_cast<long>(blockDim.x) + threadIdx.x; i < total;
       i += static_cast<long>(gridDim.x) * blockDim.x) {
    const int r = static_cast<int>(i % m);
    const long rest = i / m;
    const long c = rest % n;
    const long p = rest / n;
    lv[p * ldp + r + c * ldl] = 0;
  }
}

}  // namespace

// The attribute belongs to the device, and one process may drive several GPUs.
void smem_attr(const void* fn, int bytes) {
  static std::mutex mu;
  static std::set<std::pair<int, const void*>> done;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  if (done.insert({dev, fn}).second) cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

void prefer_l1(const void* fn) {
  static std::mutex mu;
  static std::set<std::pair<int, const void*>> done;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  if (done.insert({dev, fn}).second)
    cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxL1);
}

int set_error(emul_handle_t h, int code, const std::string& msg) {
  if (h) h->last_error = msg;
  return code;
}

int check_cuda(emul_handle_t h, cudaError_t e, const char* what) {
  if (e == cudaSuccess) return EMUL_OK;
  return set_error(h, EMUL_CUDA_ERROR, std::string(what) + ": " + cudaGetErrorString(e));
}

int reserve_workspace(emul_handle_t h, size_t bytes) {
  if (bytes <= h->ws_bytes) return EMUL_OK;
  if (h->ws) {
    cudaStreamSynchronize(h->stream);
    cudaFree(h->ws);
    h->ws = nullptr;
    h->ws_bytes = 0;
  }
  const size_t want = align_up(bytes + bytes / 8);
  if (cudaMalloc(&h->ws, want) != cudaSuccess) {
    cudaGetLastError();
    return set_error(h, EMUL_NO_WORKSPACE, "workspace allocation failed");
  }
  h->ws_bytes = want;
  return EMUL_OK;
}

size_t gemm_workspace_bytes(int m, int n, int k, int s, bool same_operand) {
  const size_t kp = static_cast<size_t>(kpad_of(k));
  size_t b = align_up(static_cast<size_t>(s) * m * kp * 2) + align_up(static_cast<size_t>(m) * 4);
  if (!same_operand) b += align_up(static_cast<size_t>(s) * n * kp * 2) + align_up(static_cast<size_t>(n) * 4);
  return b + kAlign;
}

namespace {

// Event bracket of one product launch while profiling is enabled.
int prof_begin(emul_handle_t h, emul_handle_s::ProfRec* rec, int m, int n, int k, int s, int t, int s_a, int s_b,
               bool lower, double beta, bool same) {
  if (!h->prof) return EMUL_OK;
  for (int i = 0; i < 2; ++i) {
    cudaEvent_t ev;
    if (!h->event_pool.empty()) {
      ev = h->event_pool.back();
      h->event_pool.pop_back();
    } else if (cudaEventCreate(&ev) != cudaSuccess) {
      return set_error(h, EMUL_CUDA_ERROR, "event creation failed");
    }
    (i == 0 ? rec->e0 : rec->e1) = ev;
  }
  // slice pairs kept: those of the levels L = 2..t (s(s+1)/2 at t = s + 1)
  double P = 0.0;
  for (int L = 2; L <= t; ++L) P += PairSet{s_a, s_b}.count(L);
  const double cells = lower ? 0.5 * m * (double)n : static_cast<double>(m) * n;
  rec->flops = 2.0 * cells * k * P;
  rec->bytes = cells * (beta != 0.0 ? 16.0 : 8.0) + static_cast<double>(s) * 2.0 * k * (m + (same ? 0 : n));
  cudaEventRecord(rec->e0, h->stream);
  return EMUL_OK;
}

void prof_end(emul_handle_t h, const emul_handle_s::ProfRec& rec) {
  if (!h->prof) return;
  cudaEventRecord(rec.e1, h->stream);
  h->recs.push_back(rec);
}

// Whether the m x n block C (ldc) and the rows x k operand X share an entry.
// Blocks of different leading dimensions whose address ranges meet count as
// sharing one.
bool blocks_meet(const double* C, long ldc, int m, int n, const Operand& X, int rows, int k) {
  const bool by_rows = X.rs == 1;
  const long ld = by_rows ? X.cs : X.rs, xr = by_rows ? rows : k, xc = by_rows ? k : rows;
  const long c_len = (n - 1) * ldc + m, x_len = (xc - 1) * ld + xr;
  const long d = X.ptr - C;                 // of X's first entry from C's
  if (d >= c_len || -d >= x_len) return false;
  if (ld != ldc || xr > ld || m > ldc) return true;
  // position of X's first entry in C's columns: row r0 in (-ld, ld), for both columns it may be counted in
  const long q = d >= 0 ? d / ld : -((-d + ld - 1) / ld);
  const long r = d - q * ld;                // 0 <= r < ld
  auto meet = [&](long r0, long c0) { return r0 < m && r0 + xr > 0 && c0 < n && c0 + xc > 0; };
  return meet(r, q) || meet(r - ld, q + 1);
}

// The one-launch product reads its operands while other blocks write C, where
// the sliced product reads all of both first.  C may lie over an operand only
// when each block alone reads what it overwrites: over B with one row of tiles,
// entry for entry, or over A with one column of tiles.
bool small_product_alias_ok(int m, int n, int k, const Operand& A, const Operand& B, const double* C, long ldc) {
  const bool one_row = m <= 128, one_col = n <= 32;
  if (blocks_meet(C, ldc, m, n, A, m, k) && !(one_col && (one_row || (A.ptr == C && A.rs == 1 && A.cs == ldc)))) return false;
  if (blocks_meet(C, ldc, m, n, B, n, k) && !(one_row && (one_col || (B.ptr == C && B.cs == 1 && B.rs == ldc)))) return false;
  return true;
}

}  // namespace

int gemm_run(emul_handle_t h, int m, int n, int k, double alpha, Operand A, Operand B, double beta, double* C,
             long ldc, int s, bool lower, int mode, int32_t* levels, long ldl, long ldl_plane, size_t ws_offset,
             int t, int s_a, int s_b) {
  if (s_a == 0) s_a = s;
  if (s_b == 0) s_b = s;
  if (t == 0) t = s + 1;
  if (m <= 0 || n <= 0) return EMUL_OK;
  if (k <= 0) {
    if (mode == 1) {
      zero_levels_kernel<<<256, 256, 0, h->stream>>>(m, n, s, levels, ldl, ldl_plane);
      h->launches++;
      return check_cuda(h, cudaGetLastError(), "zero levels");
    }
    scale_c_kernel<<<1024, 256, 0, h->stream>>>(m, n, alpha, beta, C, ldc);
    h->launches++;
    return check_cuda(h, cudaGetLastError(), "scale C");
  }
  const bool same = (A.ptr == B.ptr && A.rs == B.rs && A.cs == B.cs && m == n);
  if (mode == 0 && !lower && t == s + 1 && s_a == s_b && small_product_fits(m, n, k, s, h->nsm) &&
      small_product_alias_ok(m, n, k, A, B, C, ldc)) {
    emul_handle_s::ProfRec rec{};
    if (int pe = prof_begin(h, &rec, m, n, k, s, t, s_a, s_b, false, beta, same)) return pe;
    const int rc_small = check_cuda(h, launch_small_product(h->stream, m, n, k, alpha, A.ptr, A.rs, A.cs, B.ptr, B.rs, B.cs, beta,
                                                  C, ldc, s, h->d_status, h->wait_limit), "small product");
    h->launches++;
    prof_end(h, rec);
    return rc_small;
  }
  const size_t need = ws_offset + gemm_workspace_bytes(m, n, k, s, same);
  int rc = reserve_workspace(h, need);
  if (rc) return rc;
  const long kp = kpad_of(k);
  uint8_t* w = static_cast<uint8_t*>(h->ws) + ws_offset;
  uint16_t* sa = reinterpret_cast<uint16_t*>(w);
  w += align_up(static_cast<size_t>(s) * m * kp * 2);
  int32_t* ea = reinterpret_cast<int32_t*>(w);
  w += align_up(static_cast<size_t>(m) * 4);
  uint16_t* sb = sa;
  int32_t* fb = ea;
  if (!same) {
    sb = reinterpret_cast<uint16_t*>(w);
    w += align_up(static_cast<size_t>(s) * n * kp * 2);
    fb = reinterpret_cast<int32_t*>(w);
  }
  rc = check_cuda(h, same ? launch_split(h->stream, m, k, A.ptr, A.rs, A.cs, s, ea, sa, kp)
                          : launch_split2(h->stream, k, s, kp, m, A.ptr, A.rs, A.cs, ea, sa, n, B.ptr, B.rs, B.cs, fb, sb),
                  "split");
  if (rc) return rc;
  h->launches++;
  if (mode == 1) {
    h->launches++;
    zero_levels_kernel<<<256, 256, 0, h->stream>>>(m, n, s, levels, ldl, ldl_plane);
    rc = check_cuda(h, cudaGetLastError(), "zero levels");
    if (rc) return rc;
  }
  const int nch = (k + kBK - 1) / kBK;
  // the variant tests plan a schedule; they are made once per (s, t, K chunks)
  const uint64_t nkey = (static_cast<uint64_t>(s_a) << 48) | (static_cast<uint64_t>(s_b) << 40) |
                        (static_cast<uint64_t>(s) << 32) | (static_cast<uint64_t>(t) << 16) | static_cast<uint64_t>(nch);
  Sweep* sched = nullptr;
  int nsweeps = 0;
  DrainConstants drains{};
  auto nit = h->narrow_cache.find(nkey);
  if (nit == h->narrow_cache.end()) {
    const int kinds = (narrow_ok(s, k, t, s_a, s_b) ? 4 : 0) |
                      pair_plan(s, t, nch, s_a, s_b, nullptr, nullptr);
    nit = h->narrow_cache.emplace(nkey, kinds).first;
    // the schedules of both shapes of tile now: the first product with this k and
    // slice count is then the only one that allocates, whatever the others' m and n
    // (a later one may be captured); one that this call needs is asked for again below
    get_schedule(h, s, t, nch, !(kinds & 4), false, &sched, &nsweeps, &drains, s_a, s_b);
    if (kinds & 3) get_schedule(h, s, t, nch, false, true, &sched, &nsweeps, &drains, s_a, s_b);
  }
  // CTA pairs (cta_group::2) once there are two 128-row tiles: each SM stages
  // half of B, a quarter less than alone.  64-column tiles where the pairs take them
  // all at once: a wave of them costs 0.7 of a wave of 128-column tiles, so they gain
  // only while they are one wave too.  us, 64 / 128 columns, s = 7, 76 pairs: 1024 x
  // 1024 x 256 (64 tiles of 64 columns) 31 / 38, 4864 x 256 x 256 (76) 34 / 41, with k
  // = 1024 120 / 152, at s = 8 37 / 50, at s = 3 28 / 30; just past the line 2560 x
  // 512 x 256 (80) 49 / 39, k = 1024 167 / 130, s = 8 55 / 49, s = 3 38 / 31, and
  // 2048 x 1152 x 256 (144) 49 / 40.  With a short K what a wave waits for is a ragged
  // tile's rounding with its checks, half as long with 64 columns: up to short_k they
  // gain as long as 128-column tiles are one wave.  2262 x 691, s = 7: k = 79 30.1 / 33.3,
  // 128 32.9 / 34.7, 256 50.8 / 46.9; s = 8: 128 38.5 / 43.0, 256 57.3 / 56.9; s = 3: 128
  // 23.7 / 27.5, 256 32.3 / 32.7; whole tiles, 2304 x 1024 x 64 at s = 7: 25.0 / 23.1
  GemmConfig cfg{Variant::kWide, 64, false};
  const int pair_kind = nit->second & 3;
  if (pair_kind && m > 128 && h->nsm >= 2) {
    GemmConfig c{Variant::kPair, 128, pair_kind == 2};
    const long rows = (m + 255) / 256, tiles64 = rows * ((n + 63) / 64), tiles128 = rows * ((n + 127) / 128);
    const int pairs = (h->nsm - h->sm_spare) / 2, short_k = s == 8 ? 224 : s <= 3 ? 256 : 160;
    const bool ragged = m % 256 != 0 || n % 128 != 0;
    if (!lower && (tiles64 <= pairs || (ragged && k <= short_k && tiles128 < pairs))) c.bn = 64;
    // level sums read and write their planes once per job, and bands of two levels
    // have fewer jobs: one CTA per tile, and 128-column pair tiles (us): 2000 x 2500 x 200,
    // s = 8 572 / 698, with k = 1000 1238 / 1823, at s = 7 1235 / 1565; 5000 x 5000 x 256, s =
    // 7 2427 / 2531.  In one wave of small tiles pairs gain (512 x 512 x 256 79, 105 before)
    const bool fewer_jobs = mode == 1 && c.bn == 128;
    size_t smem_pair = 0;
    if (!fewer_jobs && gemm_stages(c, s, &smem_pair) >= 2 && gemm_pair_capacity(smem_pair) >= 1)
      cfg = c;   // else one CTA per tile
  }
  const bool pair = cfg.var == Variant::kPair;
  if (!pair && (nit->second & 4)) cfg = GemmConfig{Variant::kNarrow, 128, false};
  const bool wide = cfg.var == Variant::kWide;
  if (wide && mode == 0 && !wide_ok(s, t, k, s_a, s_b))
    return set_error(h, EMUL_NOT_SUPPORTED, "threshold too high for this k: the 128-bit exact sum could overflow");
  rc = get_schedule(h, s, t, nch, wide, pair, &sched, &nsweeps, &drains, s_a, s_b);
  if (rc) return rc;
  const int BN = cfg.bn;
  CUtensorMap tmA, tmB;
  rc = encode_slices_map(h, &tmA, sa, m, k, kp, s, 128);
  if (rc) return rc;
  rc = encode_slices_map(h, &tmB, sb, n, k, kp, s, pair ? BN / 2 : BN);
  if (rc) return rc;

  GemmArgs a{};
  a.M = m;
  a.N = n;
  a.K = k;
  a.s = s;
  a.t = t;
  a.alpha = alpha;
  a.beta = beta;
  a.C = C;
  a.ldc = ldc;
  a.ea = ea;
  a.fb = fb;
  a.sched = sched;
  a.nsweeps = nsweeps;
  a.stash_job = drains.stash_job;
  a.r_init = drains.r_init;
  a.r_init2 = drains.r_init2;
  a.tiles_m = pair ? (m + 255) / 256 : (m + 127) / 128;
  a.tiles_n = (n + BN - 1) / BN;
  a.lower = lower ? 1 : 0;
  a.tri = (lower && !wide && m == n) ? 1 : 0;
  if (!a.tri)
    a.ntiles = a.tiles_m * a.tiles_n;
  else if (!pair)
    a.ntiles = a.tiles_m * (a.tiles_m + 1) / 2;
  else   // row pair r < tiles_m - 1 holds 2r + 2 tiles reaching the diagonal, the last one tiles_n
    a.ntiles = (a.tiles_m - 1) * a.tiles_m + a.tiles_n;
  a.mode = mode;
  a.levels = levels;
  a.ldl = ldl;
  a.ldl_plane = ldl_plane;
  a.status = h->d_status;
  a.wait_limit = h->wait_limit;

  size_t smem = 0;
  const int stages = gemm_stages(cfg, s, &smem);
  if (stages < 2) return set_error(h, EMUL_NOT_SUPPORTED, "slice tiles do not fit in shared memory");
  const int sms = h->nsm - h->sm_spare;
  const int units = pair ? sms / 2 : sms;   // CTAs, or CTA pairs
  const int grid = (a.ntiles < units ? a.ntiles : units) * (pair ? 2 : 1);
  emul_handle_s::ProfRec rec{};
  rc = prof_begin(h, &rec, m, n, k, s, t, s_a, s_b, lower, beta, same);
  if (rc) return rc;
  rc = check_cuda(h, launch_gemm(h->stream, cfg, tmA, tmB, a, grid, stages, smem), "gemm kernel");
  h->launches++;
  prof_end(h, rec);
  return rc;
}

}  // namespace emul

using emul::Operand;

namespace emul {

namespace {
bool pool_event(emul_handle_t h, cudaEvent_t* ev) {
  if (!h->event_pool.empty()) {
    *ev = h->event_pool.back();
    h->event_pool.pop_back();
    return true;
  }
  return cudaEventCreate(ev) == cudaSuccess;
}
}  // namespace

int phase_begin(emul_handle_t h, int kind, cudaStream_t st) {
  if (!h->prof) return -1;
  emul_handle_s::PhaseRec r{kind, nullptr, nullptr};
  if (!pool_event(h, &r.e0)) return -1;
  if (!pool_event(h, &r.e1)) {
    h->event_pool.push_back(r.e0);
    return -1;
  }
  cudaEventRecord(r.e0, st);
  h->phases.push_back(r);
  return static_cast<int>(h->phases.size()) - 1;
}

void phase_end(emul_handle_t h, int idx, cudaStream_t st) {
  if (idx >= 0 && idx < static_cast<int>(h->phases.size())) cudaEventRecord(h->phases[idx].e1, st);
}

int phase_begin(emul_handle_t h, int kind) { return phase_begin(h, kind, h->stream); }

void phase_end(emul_handle_t h, int idx) { phase_end(h, idx, h->stream); }

}  // namespace emul

extern "C" {

int emul_create(emul_handle_t* handle, void* stream) {
  if (!handle) return EMUL_INVALID_ARG;
  *handle = nullptr;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return EMUL_CUDA_ERROR;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return EMUL_CUDA_ERROR;
  if (prop.major != 10 || prop.minor != 3) return EMUL_NOT_SUPPORTED;
  auto* h = new emul_handle_s();
  h->stream = static_cast<cudaStream_t>(stream);
  h->device = dev;
  h->nsm = prop.multiProcessorCount;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &h->encode_fn, 12000, cudaEnableDefault, &q) !=
          cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !h->encode_fn) {
    delete h;
    return EMUL_CUDA_ERROR;
  }
  if (cudaMalloc(&h->d_status, sizeof(int)) != cudaSuccess) {
    delete h;
    return EMUL_NO_WORKSPACE;
  }
  cudaMemset(h->d_status, 0, sizeof(int));
  *handle = h;
  return EMUL_OK;
}

int emul_destroy(emul_handle_t h) {
  if (!h) return EMUL_INVALID_ARG;
  cudaStreamSynchronize(h->stream);
  for (auto& kv : h->sched_cache) cudaFree(kv.second.sched);
  for (auto& r : h->recs) {
    cudaEventDestroy(r.e0);
    cudaEventDestroy(r.e1);
  }
  for (auto& r : h->phases) {
    cudaEventDestroy(r.e0);
    cudaEventDestroy(r.e1);
  }
  for (auto ev : h->event_pool) cudaEventDestroy(ev);
  if (h->aux) {
    cudaStreamSynchronize(h->aux);
    cudaStreamDestroy(h->aux);
  }
  if (h->aux_start) cudaEventDestroy(h->aux_start);
  if (h->aux_done) cudaEventDestroy(h->aux_done);
  emul::selector_free(h);
  emul::batched_free(h);
  if (h->ws) cudaFree(h->ws);
  if (h->d_status) cudaFree(h->d_status);
  delete h;
  return EMUL_OK;
}

int emul_set_stream(emul_handle_t h, void* stream) {
  if (!h) return EMUL_INVALID_ARG;
  h->stream = static_cast<cudaStream_t>(stream);
  return EMUL_OK;
}

const char* emul_last_error(emul_handle_t h) { return h ? h->last_error.c_str() : "null handle"; }

int emul_sync_status(emul_handle_t h) {
  if (!h) return EMUL_INVALID_ARG;
  int rc = emul::check_cuda(h, cudaStreamSynchronize(h->stream), "stream synchronize");
  if (rc) return rc;
  int st = 0;
  rc = emul::check_cuda(h, cudaMemcpy(&st, h->d_status, sizeof(int), cudaMemcpyDeviceToHost), "status read");
  if (rc) return rc;
  cudaMemset(h->d_status, 0, sizeof(int));
  if (st != 0) return emul::set_error(h, st, "a device-side wait gave up");
  return EMUL_OK;
}

size_t emul_workspace_bytes(emul_handle_t h) { return h ? h->ws_bytes : 0; }

int emul_profile_enable(emul_handle_t h, int enable) {
  if (!h) return EMUL_INVALID_ARG;
  h->prof = enable != 0;
  return EMUL_OK;
}

int emul_profile_read(emul_handle_t h, emul_profile* out) {
  if (!h || !out) return EMUL_INVALID_ARG;
  int rc = emul::check_cuda(h, cudaStreamSynchronize(h->stream), "stream synchronize");
  if (rc) return rc;
  emul_profile p{};
  p.kernel_launches = h->launches;
  for (auto& r : h->recs) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, r.e0, r.e1);
    p.product_launches++;
    p.product_ms += ms;
    p.product_tensor_flops += r.flops;
    p.product_bytes += r.bytes;
    h->event_pool.push_back(r.e0);
    h->event_pool.push_back(r.e1);
  }
  h->recs.clear();
  for (auto& r : h->phases) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.e0, r.e1) == cudaSuccess && r.kind >= 0 && r.kind < 5) p.phase_ms[r.kind] += ms;
    h->event_pool.push_back(r.e0);
    h->event_pool.push_back(r.e1);
  }
  h->phases.clear();
  h->launches = 0;
  *out = p;
  return EMUL_OK;
}

int emul_schedule(int slices, int k, int wide, int level_sums, int threshold, int* sweeps, int cap_sweeps,
                  unsigned char* table, int cap_table, int* meta) {
  using namespace emul;
  if (slices < 1 || slices > kMaxSlices || k < 1 || !meta) return EMUL_INVALID_ARG;
  if (threshold != 0 && (threshold < 2 || threshold > 2 * slices)) return EMUL_INVALID_ARG;
  (void)level_sums;                  // both modes take the same schedule
  const int nch = (k + kBK - 1) / kBK;
  std::vector<Sweep> v;
  if (!build_schedule(slices, nch, wide != 0, v, threshold)) return EMUL_INVALID_ARG;
  int njobs = 0, period = 1;
  for (const Sweep& w : v) njobs += w.njobs;
  // jobs counted over all tiles take the slots in turn: 8 jobs until slot and parity repeat
  while (period * njobs % (2 * kTmemSlots) != 0) ++period;
  std::vector<uint8_t> tab(static_cast<size_t>(period) * njobs);
  for (size_t j = 0; j < tab.size(); ++j) tab[j] = static_cast<uint8_t>(j % kTmemSlots | (j / kTmemSlots & 1) << 2);
  meta[0] = static_cast<int>(v.size());
  meta[1] = njobs;
  meta[2] = 0;
  meta[3] = period;
  meta[4] = static_cast<int>(tab.size());
  if (!sweeps || !table || cap_sweeps < static_cast<int>(v.size()) || cap_table < static_cast<int>(tab.size()))
    return EMUL_INVALID_ARG;
  for (size_t i = 0; i < v.size(); ++i) {
    const Sweep& w = v[i];
    const int row[EMUL_SWEEP_INTS] = {w.k0c,        w.k1c,        w.L[0],           w.L[1],
                                      w.pp[0] & 15, w.pp[1] & 15, w.pp[0] >> 4,     w.pp[1] >> 4,
                                      w.final_mask & 1, w.final_mask >> 1, w.nplanes, w.kcs};
    for (int j = 0; j < EMUL_SWEEP_INTS; ++j) sweeps[i * EMUL_SWEEP_INTS + j] = row[j];
  }
  std::memcpy(table, tab.data(), tab.size());
  return EMUL_OK;
}

int emul_schedule_pair(int slices_a, int slices_b, int k, int threshold, int* sweeps, int cap_sweeps, int* meta) {
  using namespace emul;
  if (!meta) return EMUL_INVALID_ARG;
  meta[0] = meta[1] = 0;
  meta[2] = -1;
  const int s = slices_a > slices_b ? slices_a : slices_b;
  if (slices_a < 1 || slices_b < 1 || s > kMaxSlices || k < 1 || k > 16384 * 4 ||
      (threshold != 0 && (threshold < 2 || threshold > slices_a + slices_b)))
    return EMUL_INVALID_ARG;
  std::vector<Sweep> v;
  int stash = -1;
  const int kind = pair_plan(s, threshold ? threshold : s + 1, (k + kBK - 1) / kBK, slices_a, slices_b, &v, &stash);
  if (!kind) return EMUL_INVALID_ARG;
  meta[0] = static_cast<int>(v.size());
  meta[1] = kind;
  meta[2] = stash;
  if (!sweeps || cap_sweeps < static_cast<int>(v.size())) return EMUL_INVALID_ARG;
  for (size_t i = 0; i < v.size(); ++i) {
    const Sweep& w = v[i];
    int* r = sweeps + i * EMUL_PAIR_SWEEP_INTS;
    int fin = -1;
    for (int j = 0; j < w.njobs; ++j)
      if ((w.final_mask >> j) & 1) fin = j;
    r[0] = w.k0c;
    r[1] = w.k1c;
    r[2] = w.njobs;
    r[3] = fin;
    r[4] = w.nplanes;
    r[5] = w.kcs;
    for (int j = 0; j < kSweepJobs; ++j) {
      r[6 + 3 * j] = w.L[j];
      r[7 + 3 * j] = w.pp[j] & 15;
      r[8 + 3 * j] = w.pp[j] >> 4;
    }
  }
  return EMUL_OK;
}

int emul_split(emul_handle_t h, int rows, int k, const double* X, long rs, long cs, int slices, int32_t* exps,
               uint16_t* slice_out, long ldk) {
  if (!h) return EMUL_INVALID_ARG;
  if (rows < 0 || k < 0 || slices < 1 || slices > emul::kMaxSlices || ldk < k || ldk % 8 != 0 ||
      (rs != 1 && cs != 1) || (rows > 0 && (!X || !exps || !slice_out)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_split: invalid argument");
  h->launches++;
  return emul::check_cuda(h, emul::launch_split(h->stream, rows, k, X, rs, cs, slices, exps, slice_out, ldk),
                          "split");
}

int emul_level_sums(emul_handle_t h, int m, int n, int k, const double* A, int lda, const double* B, int ldb,
                    int slices, int32_t* levels, int ldl, long ldl_plane) {
  if (!h) return EMUL_INVALID_ARG;
  if (m < 0 || n < 0 || k < 0 || slices < 1 || slices > emul::kMaxSlices || lda < (m > 1 ? m : 1) ||
      ldb < (k > 1 ? k : 1) || ldl < (m > 1 ? m : 1) || ldl_plane < static_cast<long>(ldl) * n || !levels ||
      k > 16384 * 4)
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_level_sums: invalid argument");
  return emul::gemm_run(h, m, n, k, 1.0, Operand{A, 1, lda}, Operand{B, ldb, 1}, 0.0, nullptr, 0, slices, false, 1,
                        levels, ldl, ldl_plane);
}

int emul_dgemm_threshold(emul_handle_t h, int m, int n, int k, double alpha, const double* A, int lda,
                         const double* B, int ldb, double beta, double* C, int ldc, int slices, int threshold) {
  if (!h) return EMUL_INVALID_ARG;
  if (m < 0 || n < 0 || k < 0 || slices < 1 || slices > emul::kMaxSlices || lda < (m > 1 ? m : 1) ||
      ldb < (k > 1 ? k : 1) || ldc < (m > 1 ? m : 1) || (m > 0 && n > 0 && !C) ||
      (m > 0 && n > 0 && k > 0 && (!A || !B)) || k > 16384 * 4 ||
      (threshold != 0 && (threshold < 2 || threshold > 2 * slices)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dgemm: invalid argument");
  return emul::gemm_run(h, m, n, k, alpha, Operand{A, 1, lda}, Operand{B, ldb, 1}, beta, C, ldc, slices, false, 0,
                        nullptr, 0, 0, 0, threshold);
}

int emul_dgemm(emul_handle_t h, int m, int n, int k, double alpha, const double* A, int lda, const double* B,
               int ldb, double beta, double* C, int ldc, int slices) {
  return emul_dgemm_threshold(h, m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, slices, 0);
}

int emul_dgemm_unequal(emul_handle_t h, int m, int n, int k, double alpha, const double* A, int lda,
                       const double* B, int ldb, double beta, double* C, int ldc, int slices_a, int slices_b,
                       int threshold) {
  if (!h) return EMUL_INVALID_ARG;
  const int s = slices_a > slices_b ? slices_a : slices_b;
  if (m < 0 || n < 0 || k < 0 || slices_a < 1 || slices_b < 1 || s > emul::kMaxSlices || lda < (m > 1 ? m : 1) ||
      ldb < (k > 1 ? k : 1) || ldc < (m > 1 ? m : 1) || (m > 0 && n > 0 && !C) ||
      (m > 0 && n > 0 && k > 0 && (!A || !B)) || k > 16384 * 4 ||
      (threshold != 0 && (threshold < 2 || threshold > slices_a + slices_b)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dgemm_unequal: invalid argument");
  return emul::gemm_run(h, m, n, k, alpha, Operand{A, 1, lda}, Operand{B, ldb, 1}, beta, C, ldc, s, false, 0, nullptr,
                        0, 0, 0, threshold, slices_a, slices_b);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// emul_dgemm_noalloc: the emulated DGEMM for callers that cannot allocate
// device memory: a host library whose device memory belongs to another
// allocator (a framework's caching allocator, a pool sized at start-up), or a
// latency-bound loop that must not call cudaMalloc / cudaFree (both can
// synchronise the whole device).  All scratch lives in one file-scope device
// array of kNoAllocScratchBytes that every GPU which loads this library keeps
// until the process exits.
namespace emul {
namespace {

constexpr size_t kNoAllocScratchBytes = size_t(16) << 20;   // 16 MiB
constexpr size_t kNoAllocSchedBytes = 16384;                // 1024 sweeps
constexpr int kNoAllocMaxDevices = 64;

__device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

struct NoAllocDevice {
  unsigned char* base = nullptr;   // device address of g_noalloc_scratch on this device
  int nsm = 0;
};
NoAllocDevice g_noalloc_dev[kNoAllocMaxDevices];
void* g_noalloc_encode = nullptr;
std::mutex g_noalloc_mu;

// One-time set-up per device, with that device current: the device address of
// the static scratch (host code must not use the symbol itself) and the
// tensor-map encoder.
int noalloc_setup(int dev, NoAllocDevice** out) {
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  NoAllocDevice& d = g_noalloc_dev[dev];
  if (!d.base) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return EMUL_CUDA_ERROR;
    int nsm = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return EMUL_CUDA_ERROR;
    if (!g_noalloc_encode) {
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &g_noalloc_encode, 12000, cudaEnableDefault,
                                           &q) != cudaSuccess ||
          q != cudaDriverEntryPointSuccess || !g_noalloc_encode)
        return EMUL_CUDA_ERROR;
    }
    d.base = static_cast<unsigned char*>(ptr);
    d.nsm = nsm;
  }
  *out = &d;
  return EMUL_OK;
}

int noalloc_map(CUtensorMap* map, const uint16_t* base, int rows, int k, long kpad, int s, int box_rows) {
  auto fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(g_noalloc_encode);
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(k), static_cast<cuuint64_t>(rows), static_cast<cuuint64_t>(s)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(kpad) * 2, static_cast<cuuint64_t>(kpad) * 2 * rows};
  cuuint32_t box[3] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows), 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<uint16_t*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? EMUL_OK
             : EMUL_CUDA_ERROR;
}

}  // namespace
}  // namespace emul

extern "C" int emul_dgemm_noalloc(void* stream, int m, int n, int k, double alpha, const double* A, int lda,
                                  const double* B, int ldb, double beta, double* C, int ldc, int slices) {
  using namespace emul;
  if (m < 0 || n < 0 || k < 0 || slices < 1 || slices > kMaxSlices || lda < (m > 1 ? m : 1) ||
      ldb < (k > 1 ? k : 1) || ldc < (m > 1 ? m : 1) || (m > 0 && n > 0 && !C) ||
      (m > 0 && n > 0 && k > 0 && (!A || !B)) || k > 16384 * 4)
    return EMUL_INVALID_ARG;
  if (m == 0 || n == 0) return EMUL_OK;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return EMUL_CUDA_ERROR;
  NoAllocDevice* d = nullptr;
  int rc = noalloc_setup(dev, &d);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (k == 0) {
    scale_c_kernel<<<1024, 256, 0, st>>>(m, n, alpha, beta, C, ldc);
    return cudaGetLastError() == cudaSuccess ? EMUL_OK : EMUL_CUDA_ERROR;
  }
  // scratch layout: status word | schedule | row scales | column scales | slices of A | slices of B
  const long kp = kpad_of(k);
  const size_t off_sched = kAlign;
  const size_t off_ea = off_sched + kNoAllocSchedBytes;
  const size_t off_fb = off_ea + align_up(static_cast<size_t>(m) * 4);
  const size_t off_sa = off_fb + align_up(static_cast<size_t>(n) * 4);
  const size_t off_sb = off_sa + align_up(static_cast<size_t>(slices) * m * kp * 2);
  const size_t need = off_sb + align_up(static_cast<size_t>(slices) * n * kp * 2);
  if (need > kNoAllocScratchBytes) return EMUL_NO_WORKSPACE;   // operands exceed the 16 MiB static scratch

  unsigned char* base = d->base;
  int* status = reinterpret_cast<int*>(base);
  Sweep* sched = reinterpret_cast<Sweep*>(base + off_sched);
  int32_t* ea = reinterpret_cast<int32_t*>(base + off_ea);
  int32_t* fb = reinterpret_cast<int32_t*>(base + off_fb);
  uint16_t* sa = reinterpret_cast<uint16_t*>(base + off_sa);
  uint16_t* sb = reinterpret_cast<uint16_t*>(base + off_sb);

  const bool wide = !narrow_ok(slices, k);
  const int nch = (k + kBK - 1) / kBK;
  std::vector<Sweep> v;
  if (!build_schedule(slices, nch, wide, v)) return EMUL_INVALID_ARG;
  if (v.size() * sizeof(Sweep) > kNoAllocSchedBytes) return EMUL_NO_WORKSPACE;
  const DrainConstants drains = drained_constants(v, slices + 1, -1);
  // the status word must start at zero; the rest is fully rewritten by this call
  if (cudaMemsetAsync(status, 0, sizeof(int), st) != cudaSuccess) return EMUL_CUDA_ERROR;
  if (cudaMemcpyAsync(sched, v.data(), v.size() * sizeof(Sweep), cudaMemcpyHostToDevice, st) != cudaSuccess)
    return EMUL_CUDA_ERROR;
  if (launch_split2(st, k, slices, kp, m, A, 1, lda, ea, sa, n, B, ldb, 1, fb, sb) != cudaSuccess)
    return EMUL_CUDA_ERROR;
  const int BN = wide ? 64 : 128;
  CUtensorMap tmA, tmB;
  rc = noalloc_map(&tmA, sa, m, k, kp, slices, 128);
  if (rc) return rc;
  rc = noalloc_map(&tmB, sb, n, k, kp, slices, BN);
  if (rc) return rc;
  GemmArgs a{};
  a.M = m;
  a.N = n;
  a.K = k;
  a.s = slices;
  a.t = slices + 1;
  a.alpha = alpha;
  a.beta = beta;
  a.C = C;
  a.ldc = ldc;
  a.ea = ea;
  a.fb = fb;
  a.sched = sched;
  a.nsweeps = static_cast<int>(v.size());
  a.stash_job = drains.stash_job;
  a.r_init = drains.r_init;
  a.r_init2 = drains.r_init2;
  a.tiles_m = (m + 127) / 128;
  a.tiles_n = (n + BN - 1) / BN;
  a.ntiles = a.tiles_m * a.tiles_n;
  a.status = status;
  a.wait_limit = 2000000000LL;
  const GemmConfig cfg = wide ? GemmConfig{Variant::kWide, 64, false} : GemmConfig{Variant::kNarrow, 128, false};
  size_t smem = 0;
  const int stages = gemm_stages(cfg, slices, &smem);
  if (stages < 2) return EMUL_NOT_SUPPORTED;
  const int grid = a.ntiles < d->nsm ? a.ntiles : d->nsm;
  return launch_gemm(st, cfg, tmA, tmB, a, grid, stages, smem) == cudaSuccess ? EMUL_OK : EMUL_CUDA_ERROR;
}
