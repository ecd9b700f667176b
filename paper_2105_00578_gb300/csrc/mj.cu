// mj.cu -- multi-jagged multisection of the spectral coordinates (Sec. 4).
//
// Rule (exact, integer): a section owning parts [lo, lo + k) splits into
// k_L = ceil(k/2) and k_R = floor(k/2) parts along dimension level mod dims.
// Its points are ordered by the composite key (coordinate, vertex id), the
// coordinate compared as an IEEE value (-0 == +0); the left side is the
// shortest prefix p minimising |k cumW(p) - k_L W| (cumW strictly increasing
// because vertex weights are >= 1).
//
// GPU schedule, one level at a time for all sections at once:
//  * sections are contiguous ranges of a permutation array `perm`; where the
//    scratch allows it the level's ordered keys lie beside it, so that the passes
//    stream them instead of gathering a coordinate per point;
//  * the split element e (the first point with k cumW >= k_L W) is found by
//    a most-significant-digit radix select over the composite key, 11 bits per
//    pass (8 where thousands of sections would need large bins): a histogram
//    kernel adds the weight and count of every candidate point into the bins of
//    its section (in shared memory where a CTA's chunk touches at most two), a
//    select kernel scans the bins and fixes one digit.  A section whose
//    candidates are down to one is done: the later passes skip it, and
//    comparisons use the digits fixed so far;
//  * a decide kernel compares the prefixes ending just before and just after e,
//    and a scatter kernel moves every point to its child range, a CTA counting
//    its 4096 points first so that it takes one global ticket a side; the last
//    level writes the part ids instead.  The resulting sets (hence part ids) are
//    exact and independent of scheduling.
// 2,097,152 points, K = 64, six float dimensions, with the evaluation of the cut
// that follows: 2893 -> 976 us a call (707 us with the scratch kept in a pool).
// Before, every pass gathered its coordinates, 8-bit digits put nearly all points
// in a few bins (a float's top eight bits are sign and exponent), and a warp took
// each scatter ticket.
#include "internal.cuh"

#include <cstring>
#include <memory>
#include <mutex>

namespace sphynx {

namespace {

constexpr int kMjThreads = 256;
constexpr int kMjChunk = 4096;

struct MjSec {             // per-section select state (device)
  unsigned long long phi, plo, mhi, mlo;
  long long before, beforecnt, ew, ec;
  long long nleft, wleft;
  int incl, pad;
  unsigned curl, curr;
};

__device__ __forceinline__ unsigned long long ordered_key(const void *coords, int dt, int64_t v, int ldc,
                                                          int dim) {
  if (dt == SPHYNX_DT_F64) {
    double x = static_cast<const double *>(coords)[v * ldc + dim];
    unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(x));
    if (x == 0.0) u = 0ull;
    return (u >> 63) ? ~u : (u | (1ull << 63));
  }
  float x = static_cast<const float *>(coords)[v * ldc + dim];
  unsigned u = __float_as_uint(x);
  if (x == 0.0f) u = 0u;
  return static_cast<unsigned long long>((u >> 31) ? ~u : (u | 0x80000000u));
}

// one digit of the composite key (coordinate key hi, vertex id lo)
struct Digit {
  int lo;      // taken from the id
  int shift;
  int bits;
  int first;   // the level's first pass
};

__device__ __forceinline__ int digit_of(unsigned long long hi, unsigned long long lo, Digit d) {
  return static_cast<int>(((d.lo ? lo : hi) >> d.shift) & ((1ull << d.bits) - 1ull));
}

// does the section still have several candidates for its split element?
__device__ __forceinline__ bool selecting(const int *split, const MjSec *sec, int s, Digit d) {
  return split[s] && (d.first || sec[s].ec > 1);
}

// where a level's ordered keys come from: the array beside perm, or the coordinates
struct KeySrc {
  const void *keys;     // uint32 (float coordinates) or uint64 by position; NULL: gather
  const void *coords;
  int dt, ldc, dim;
};
__device__ __forceinline__ unsigned long long key_at(const KeySrc &k, int64_t pos, int32_t v) {
  if (!k.keys) return ordered_key(k.coords, k.dt, v, k.ldc, k.dim);
  return k.dt == SPHYNX_DT_F64 ? static_cast<const unsigned long long *>(k.keys)[pos]
                               : static_cast<unsigned long long>(static_cast<const unsigned *>(k.keys)[pos]);
}
__device__ __forceinline__ void key_store(void *keys, int dt, int64_t pos, unsigned long long key) {
  if (dt == SPHYNX_DT_F64) static_cast<unsigned long long *>(keys)[pos] = key;
  else static_cast<unsigned *>(keys)[pos] = static_cast<unsigned>(key);
}

// the side of a point of section state q: left of the split, or the split
// element itself when it belongs to the left
__device__ __forceinline__ bool goes_left(const MjSec &q, unsigned long long hi, unsigned long long lo) {
  hi &= q.mhi;
  lo &= q.mlo;
  return hi < q.phi || (hi == q.phi && (lo < q.plo || (q.incl && lo == q.plo)));
}

__device__ __forceinline__ int section_of(const long long *start, int S, int64_t pos) {
  int lo = 0, hi = S - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= pos) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// perm = identity, the first level's keys, NaN and weight checks, total weight
__global__ void k_mj_init(int32_t *perm, void *keys, int64_t n, const void *coords, int dt, int ldc, int dims,
                          const int64_t *vw, unsigned long long *wsum, unsigned *bad) {
  unsigned long long s = 0;
  unsigned b = 0;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    perm[i] = static_cast<int32_t>(i);
    for (int d = 0; d < dims; ++d) {
      if (dt == SPHYNX_DT_F64) {
        if (isnan(static_cast<const double *>(coords)[i * ldc + d])) b |= 1;
      } else {
        if (isnan(static_cast<const float *>(coords)[i * ldc + d])) b |= 1;
      }
    }
    if (keys) key_store(keys, dt, i, ordered_key(coords, dt, i, ldc, 0));
    const long long w = vw ? vw[i] : 1;
    if (w < 1) b |= 2;
    s += static_cast<unsigned long long>(w);
  }
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) atomicAdd(wsum, s);
  if (b) atomicOr(bad, b);
}

__global__ void k_mj_level0(long long *start, long long *end, long long *W, int64_t n, const unsigned long long *wsum,
                            MjSec *sec) {
  sec[0] = MjSec{};
  start[0] = 0;
  end[0] = n;
  W[0] = static_cast<long long>(*wsum);
}

// W[g] = total vertex weight of graph g, vertices [gptr[g], gptr[g+1]); one CTA per graph
__global__ void k_mj_graph_weights(const int64_t *vw, const int64_t *gptr, long long *W) {
  __shared__ unsigned long long red[8];
  const int g = blockIdx.x;
  unsigned long long s = 0;
  for (int64_t i = gptr[g] + threadIdx.x; i < gptr[g + 1]; i += blockDim.x) s += static_cast<unsigned long long>(vw[i]);
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int k = 0; k < 8; ++k) t += red[k];
    W[g] = static_cast<long long>(t);
  }
}

// candidates' (weight, count) per digit value: hist [section][2^bits][2]
// (weight slot unused with unit weights)
__global__ void __launch_bounds__(kMjThreads)
k_mj_hist(const int32_t *perm, int64_t n, KeySrc ks, const int64_t *vw, const long long *start, int S,
          const int *split, const MjSec *sec, Digit d, int bins, unsigned long long *hist) {
  extern __shared__ unsigned long long mj_sh[];   // [bins] weights (with vw), then [bins] counts
  unsigned long long *shw = mj_sh;
  unsigned *shc = reinterpret_cast<unsigned *>(vw ? mj_sh + bins : mj_sh);
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * kMjChunk;
  if (c0 >= n) return;
  const int64_t c1 = c0 + kMjChunk < n ? c0 + kMjChunk : n;
  const int s0 = section_of(start, S, c0), s1 = section_of(start, S, c1 - 1);
  if (s1 - s0 > 1) {   // many sections: straight to their bins
    for (int64_t pos = c0 + threadIdx.x; pos < c1; pos += blockDim.x) {
      const int s = section_of(start, S, pos);
      if (!selecting(split, sec, s, d)) continue;
      const int32_t v = perm[pos];
      const unsigned long long hi = key_at(ks, pos, v), lo = static_cast<unsigned long long>(v);
      const MjSec &q = sec[s];
      if ((hi & q.mhi) != q.phi || (lo & q.mlo) != q.plo) continue;
      unsigned long long *h = hist + (static_cast<int64_t>(s) * bins + digit_of(hi, lo, d)) * 2;
      if (vw) atomicAdd(h, static_cast<unsigned long long>(vw[v]));
      atomicAdd(h + 1, 1ull);
    }
    return;
  }
  for (int s = s0; s <= s1; ++s) {
    if (!selecting(split, sec, s, d)) continue;   // uniform
    const int64_t b0 = s == s0 ? c0 : start[s], b1 = s == s1 ? c1 : start[s + 1];
    for (int k = threadIdx.x; k < bins; k += blockDim.x) {
      shc[k] = 0;
      if (vw) shw[k] = 0;
    }
    __syncthreads();
    const unsigned long long phi = sec[s].phi, plo = sec[s].plo, mhi = sec[s].mhi, mlo = sec[s].mlo;
    for (int64_t pos = b0 + threadIdx.x; pos < b1; pos += blockDim.x) {
      const int32_t v = ks.keys && !vw && !d.lo && !mlo ? 0 : perm[pos];   // the id only where it is needed
      const unsigned long long hi = key_at(ks, pos, v), lo = static_cast<unsigned long long>(v);
      if ((hi & mhi) != phi || (lo & mlo) != plo) continue;
      const int dg = digit_of(hi, lo, d);
      atomicAdd(&shc[dg], 1u);
      if (vw) atomicAdd(&shw[dg], static_cast<unsigned long long>(vw[v]));
    }
    __syncthreads();
    for (int k = threadIdx.x; k < bins; k += blockDim.x) {
      if (!shc[k]) continue;
      unsigned long long *h = hist + (static_cast<int64_t>(s) * bins + k) * 2;
      if (vw) atomicAdd(h, shw[k]);
      atomicAdd(h + 1, static_cast<unsigned long long>(shc[k]));
    }
    __syncthreads();
  }
}

// one CTA of 256 threads per section: find the bin holding the first point
// with k (before + cum) >= k_L W, fix that digit, clear the bins
__global__ void __launch_bounds__(256)
k_mj_select(unsigned long long *hist, int bins, int unit, const int *split, const int *ks, const long long *W,
            MjSec *sec, Digit d) {
  constexpr int kPer = 8;            // bins a thread owns: 2048 bins, or 256 of one each
  __shared__ long long sw[8], sc[8];
  __shared__ int first;
  const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (!selecting(split, sec, s, d)) return;   // uniform
  const int per = bins / 256;
  unsigned long long *h = hist + (static_cast<int64_t>(s) * bins + tid * per) * 2;
  long long wb[kPer], cb[kPer];
  long long lw = 0, lc = 0;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    wb[u] = cb[u] = 0;
    if (u < per) {
      cb[u] = static_cast<long long>(h[2 * u + 1]);
      wb[u] = unit ? cb[u] : static_cast<long long>(h[2 * u]);
      if (cb[u]) h[2 * u] = h[2 * u + 1] = 0;
    }
    lw += wb[u];
    lc += cb[u];
  }
  long long pw = lw, pc = lc;        // inclusive scans over the warp, then the warps
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const long long tw = __shfl_up_sync(0xffffffffu, pw, off);
    const long long tc = __shfl_up_sync(0xffffffffu, pc, off);
    if (lane >= off) { pw += tw; pc += tc; }
  }
  if (lane == 31) {
    sw[warp] = pw;
    sc[warp] = pc;
  }
  if (tid == 0) first = bins;
  MjSec &q = sec[s];
  const long long k = ks[s], T = (k + 1) / 2 * W[s];
  long long cw = q.before + pw - lw, cc = q.beforecnt + pc - lc;
  __syncthreads();
  for (int w = 0; w < warp; ++w) {
    cw += sw[w];
    cc += sc[w];
  }
  int found = -1;
  long long fw = 0, fc = 0, ew = 0, ec = 0;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    if (found < 0 && cb[u] > 0 && k * (cw + wb[u]) >= T) {
      found = tid * per + u;
      fw = cw;
      fc = cc;
      ew = wb[u];
      ec = cb[u];
    }
    cw += wb[u];
    cc += cb[u];
  }
  if (found >= 0) atomicMin(&first, found);
  __syncthreads();
  if (found >= 0 && found == first) {
    q.before = fw;
    q.beforecnt = fc;
    q.ew = ew;
    q.ec = ec;
    const unsigned long long dm = ((1ull << d.bits) - 1ull) << d.shift, dv = static_cast<unsigned long long>(found)
                                                                            << d.shift;
    if (d.lo) {
      q.plo |= dv;
      q.mlo |= dm;
    } else {
      q.phi |= dv;
      q.mhi |= dm;
    }
  }
}

// choose the prefix ending just before or just after e; build the next level
__global__ void k_mj_decide(int S, const int *split, const int *ks, const int *child, const long long *start,
                            const long long *end, const long long *W, MjSec *sec, long long *nstart,
                            long long *nend, long long *nW, MjSec *nsec) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const int cb = child[s];
  nsec[cb] = MjSec{};
  if (split[s]) nsec[cb + 1] = MjSec{};
  if (!split[s]) {
    nstart[cb] = start[s];
    nend[cb] = end[s];
    nW[cb] = W[s];
    return;
  }
  MjSec &q = sec[s];
  const long long k = ks[s], kl = (k + 1) / 2, w = W[s], T = kl * w;
  long long nl = 0, wl = 0;
  int incl = 0;
  if (w > 0) {
    long long flo = k * q.before - T, fhi = k * (q.before + q.ew) - T;
    flo = flo < 0 ? -flo : flo;
    fhi = fhi < 0 ? -fhi : fhi;
    if (flo <= fhi) {
      nl = q.beforecnt;
      wl = q.before;
    } else {
      nl = q.beforecnt + 1;
      wl = q.before + q.ew;
      incl = 1;
    }
  }
  q.nleft = nl;
  q.wleft = wl;
  q.incl = incl;
  q.curl = 0;
  q.curr = 0;
  nstart[cb] = start[s];
  nend[cb] = start[s] + nl;
  nW[cb] = wl;
  nstart[cb + 1] = start[s] + nl;
  nend[cb + 1] = end[s];
  nW[cb + 1] = w - wl;
}

// moves every point of a 4096-point chunk to its child's range, with the next
// level's key where keys are kept
__global__ void __launch_bounds__(kMjThreads)
k_mj_scatter(const int32_t *perm, int32_t *perm2, int64_t n, KeySrc ks, void *keys2, int next_dim,
             const long long *start, int S, const int *split, MjSec *sec) {
  constexpr int kItems = kMjChunk / kMjThreads;
  __shared__ unsigned wl[kMjThreads / 32], wr[kMjThreads / 32];
  __shared__ unsigned base[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * kMjChunk;
  const int64_t c1 = c0 + kMjChunk < n ? c0 + kMjChunk : n;
  const int s0 = section_of(start, S, c0), s1 = section_of(start, S, c1 - 1);
  if (s0 == s1 && split[s0]) {
    const MjSec q = sec[s0];
    int32_t v[kItems];
    unsigned left[kItems];           // the warp's left lanes, per item
    unsigned nl = 0, nr = 0;
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      const int64_t pos = c0 + u * kMjThreads + tid;
      const bool in = pos < c1;
      v[u] = in ? perm[pos] : -1;
      const bool l = in && goes_left(q, key_at(ks, in ? pos : c0, in ? v[u] : perm[c0]),
                                     static_cast<unsigned long long>(static_cast<unsigned>(v[u])));
      left[u] = __ballot_sync(0xffffffffu, l);
      nl += __popc(left[u]);
      nr += __popc(__ballot_sync(0xffffffffu, in)) - __popc(left[u]);
    }
    if (lane == 0) {
      wl[warp] = nl;
      wr[warp] = nr;
    }
    __syncthreads();
    unsigned bl = 0, br = 0, tl = 0, tr = 0;
    for (int w = 0; w < kMjThreads / 32; ++w) {
      bl += w < warp ? wl[w] : 0;
      br += w < warp ? wr[w] : 0;
      tl += wl[w];
      tr += wr[w];
    }
    if (tid == 0) {
      base[0] = atomicAdd(&sec[s0].curl, tl);
      base[1] = atomicAdd(&sec[s0].curr, tr);
    }
    __syncthreads();
    int64_t pl = start[s0] + base[0] + bl, pr = start[s0] + q.nleft + base[1] + br;
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      const unsigned in = __ballot_sync(0xffffffffu, v[u] >= 0), right = in & ~left[u];
      if (v[u] >= 0) {
        const bool l = (left[u] >> lane) & 1u;
        const int64_t to = l ? pl + __popc(left[u] & below) : pr + __popc(right & below);
        perm2[to] = v[u];
        if (keys2) key_store(keys2, ks.dt, to, ordered_key(ks.coords, ks.dt, v[u], ks.ldc, next_dim));
      }
      pl += __popc(left[u]);
      pr += __popc(right);
    }
    return;
  }
  for (int64_t b = c0 + (tid & ~31); b < c1; b += kMjThreads) {   // several sections, or one that stays
    const int64_t pos = b + lane;
    int s = 0;
    int32_t v = 0;
    int64_t to = -1;
    long long key = -1;  // group key: section * 2 + side, -1 for lanes with nothing to place
    if (pos < c1) {
      s = section_of(start, S, pos);
      v = perm[pos];
      if (!split[s]) {
        to = pos;
      } else {
        const bool left = goes_left(sec[s], key_at(ks, pos, v), static_cast<unsigned long long>(v));
        key = static_cast<long long>(s) * 2 + (left ? 0 : 1);
      }
    }
    const unsigned grp = __match_any_sync(0xffffffffu, key);
    if (key >= 0) {
      const int leader = __ffs(grp) - 1;
      const unsigned rank = __popc(grp & ((1u << lane) - 1u));
      unsigned ticket = 0;
      const bool left = (key & 1) == 0;
      if (lane == leader) ticket = atomicAdd(left ? &sec[s].curl : &sec[s].curr, static_cast<unsigned>(__popc(grp)));
      ticket = __shfl_sync(grp, ticket, leader);
      to = (left ? start[s] : start[s] + sec[s].nleft) + ticket + rank;
    }
    if (to >= 0) {
      perm2[to] = v;
      if (keys2) key_store(keys2, ks.dt, to, ordered_key(ks.coords, ks.dt, v, ks.ldc, next_dim));
    }
  }
}

// the last level: part ids instead of a new order; lo[c] is the part of child c
__global__ void __launch_bounds__(kMjThreads)
k_mj_parts(const int32_t *perm, int64_t n, KeySrc ks, const long long *start, int S, const int *split,
           const int *child, const MjSec *sec, const int *lo, int32_t *part) {
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * kMjChunk;
  const int64_t c1 = c0 + kMjChunk < n ? c0 + kMjChunk : n;
  const int s0 = section_of(start, S, c0), s1 = section_of(start, S, c1 - 1);
  for (int64_t pos = c0 + threadIdx.x; pos < c1; pos += blockDim.x) {
    const int s = s0 == s1 ? s0 : section_of(start, S, pos);
    const int32_t v = perm[pos];
    int c = child[s];
    if (split[s] && !goes_left(sec[s], key_at(ks, pos, v), static_cast<unsigned long long>(v))) c += 1;
    part[v] = lo[c];
  }
}

int mj_grid(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 8 * kSmCount) g = 8 * kSmCount;
  return static_cast<int>(g < 1 ? 1 : g);
}

struct Level {
  std::vector<int> lo, k, split, child;
};

}  // namespace

namespace {

// The least scratch a call runs in: 8-bit digits, keys gathered.  The level
// tables take at most 64 bytes a part; the rest of their 1024 holds the second
// set of section states.
size_t mj_least_bytes(int64_t n, int K, int count) {
  const size_t Ks = static_cast<size_t>(K);
  return static_cast<size_t>(n) * 8 + Ks * 512 * 8 + Ks * sizeof(MjSec) + Ks * 8 * 6 + 64 +
         Ks * 4 * 4 * 64 /* level tables, up to 64 levels */ + 16 * 256 + 4096 +
         (count > 1 ? static_cast<size_t>(count + 1) * 8 + 256 : 0);
}
static_assert(sizeof(MjSec) <= 512, "the tables' slack holds the second section states");

// What a scratch of `bytes` allows.  11-bit digits for at most 2048 parts (64 MB
// of bins), and keys beside the permutation while they take at most 1 GiB.
struct MjPlan {
  int bits = 8;
  bool keys = false;
  size_t bytes = 0;
};
MjPlan mj_plan(int64_t n, int K, int count, DT dt, size_t limit) {
  MjPlan p;
  p.bytes = mj_least_bytes(n, K, count);
  const size_t wide = static_cast<size_t>(K) * (2048 - 256) * 16;
  if (K <= 2048 && p.bytes + wide <= limit) {
    p.bits = 11;
    p.bytes += wide;
  }
  const size_t keys = 2 * (static_cast<size_t>(n) * dt_size(dt) + 256);
  if (keys <= (size_t{1} << 30) && p.bytes + keys <= limit) {
    p.keys = true;
    p.bytes += keys;
  }
  return p;
}

}  // namespace

size_t mj_scratch_bytes(int64_t n, int K, int count, DT dt) { return mj_plan(n, K, count, dt, SIZE_MAX).bytes; }

namespace {
// alloc() of `bytes`; where the memory is short, of the least that serves
template <class F> void or_least(size_t &bytes, size_t least, F alloc) {
  try {
    alloc();
  } catch (const Error &e) {
    if (e.code != SPHYNX_ERR_OOM || bytes <= least) throw;
    clear_error();
    bytes = least;
    alloc();
  }
}
}  // namespace

void *mj_workspace(sphynx_graph *g, int64_t n, int K, int count, DT dt, size_t *bytes) {
  void *p = nullptr;
  *bytes = mj_scratch_bytes(n, K, count, dt);
  or_least(*bytes, mj_least_bytes(n, K, count), [&] { p = g->workspace("mj", *bytes, false); });
  return p;
}

void run_mj_scratch(cudaStream_t st, DT dt, const void *coords, int ldc, int dims, int64_t n, const int64_t *vw,
                    int K, int32_t *part, Counters *ctr, void *scratch, size_t scratch_bytes, const int64_t *h_gptr,
                    int count) {
  if (K < 1) fail(SPHYNX_ERR_INVALID_ARG, "K must be >= 1");
  if (K > (1 << 20)) fail(SPHYNX_ERR_UNSUPPORTED, "K > 2^20");
  if (n < 0) fail(SPHYNX_ERR_INVALID_ARG, "n < 0");
  if (count < 1 || (count > 1 && (!h_gptr || K % count != 0)))
    fail(SPHYNX_ERR_INVALID_ARG, "multi-jagged over %d graphs needs their offsets and K a multiple of the count",
         count);
  if (n == 0) return;
  const int k_each = K / count;   // parts of every graph; graph g owns parts [g k_each, (g + 1) k_each)
  if (K == 1) {
    SPX_CUDA(cudaMemsetAsync(part, 0, n * sizeof(int32_t), st));
    return;
  }
  if (dims < 1) fail(SPHYNX_ERR_INVALID_ARG, "multi-jagged needs at least one coordinate");
  if (dt != DT::F32 && dt != DT::F64) fail(SPHYNX_ERR_INVALID_ARG, "coordinates must be float or double");
  const int dti = dt == DT::F64 ? SPHYNX_DT_F64 : SPHYNX_DT_F32;

  // host section tree: (lo, k) per level until every section has k == 1
  std::vector<Level> levels;
  {
    Level l0;
    for (int gi = 0; gi < count; ++gi) {   // one first-level section per graph
      l0.lo.push_back(gi * k_each);
      l0.k.push_back(k_each);
    }
    levels.push_back(l0);
    for (;;) {
      Level &cur = levels.back();
      bool any = false;
      Level nx;
      cur.split.assign(cur.k.size(), 0);
      cur.child.assign(cur.k.size(), 0);
      for (size_t s = 0; s < cur.k.size(); ++s) {
        cur.child[s] = static_cast<int>(nx.k.size());
        if (cur.k[s] >= 2) {
          any = true;
          cur.split[s] = 1;
          const int kl = (cur.k[s] + 1) / 2;
          nx.lo.push_back(cur.lo[s]);
          nx.k.push_back(kl);
          nx.lo.push_back(cur.lo[s] + kl);
          nx.k.push_back(cur.k[s] - kl);
        } else {
          nx.lo.push_back(cur.lo[s]);
          nx.k.push_back(cur.k[s]);
        }
      }
      if (!any) break;
      levels.push_back(nx);
    }
  }
  const int nlev = static_cast<int>(levels.size());
  if (nlev > 64) fail(SPHYNX_ERR_UNSUPPORTED, "too many levels");

  // scratch layout
  char *p = static_cast<char *>(scratch);
  auto take = [&](size_t bytes) {
    char *r = p;
    p += (bytes + 255) & ~static_cast<size_t>(255);
    return r;
  };
  const MjPlan plan = mj_plan(n, K, count, dt, scratch_bytes);
  const int bins = 1 << plan.bits;
  int32_t *perm = reinterpret_cast<int32_t *>(take(n * 4));
  int32_t *perm2 = reinterpret_cast<int32_t *>(take(n * 4));
  unsigned long long *hist = reinterpret_cast<unsigned long long *>(take(static_cast<size_t>(K) * bins * 16));
  MjSec *sec = reinterpret_cast<MjSec *>(take(static_cast<size_t>(K) * sizeof(MjSec)));
  MjSec *sec2 = reinterpret_cast<MjSec *>(take(static_cast<size_t>(K) * sizeof(MjSec)));
  void *keys = plan.keys ? take(static_cast<size_t>(n) * dt_size(dt)) : nullptr;
  void *keys2 = plan.keys ? take(static_cast<size_t>(n) * dt_size(dt)) : nullptr;
  long long *tab[2][3];
  for (int a = 0; a < 2; ++a)
    for (int b = 0; b < 3; ++b) tab[a][b] = reinterpret_cast<long long *>(take(static_cast<size_t>(K) * 8));
  unsigned long long *misc = reinterpret_cast<unsigned long long *>(take(64));
  // all levels' (k, split, child, lo) tables in one upload
  std::vector<int> host_tab;
  std::vector<size_t> off(nlev);
  for (int l = 0; l < nlev; ++l) {
    off[l] = host_tab.size();
    const Level &L = levels[l];
    const size_t S = L.k.size();
    host_tab.insert(host_tab.end(), L.k.begin(), L.k.end());
    if (L.split.size() == S) host_tab.insert(host_tab.end(), L.split.begin(), L.split.end());
    else host_tab.insert(host_tab.end(), S, 0);
    if (L.child.size() == S) host_tab.insert(host_tab.end(), L.child.begin(), L.child.end());
    else host_tab.insert(host_tab.end(), S, 0);
    host_tab.insert(host_tab.end(), L.lo.begin(), L.lo.end());
  }
  int *dtab = reinterpret_cast<int *>(take(host_tab.size() * 4));
  SPX_CUDA(cudaMemcpyAsync(dtab, host_tab.data(), host_tab.size() * 4, cudaMemcpyHostToDevice, st));
  int64_t *dgptr = count > 1 ? reinterpret_cast<int64_t *>(take(static_cast<size_t>(count + 1) * 8)) : nullptr;
  if (dgptr) {
    if (h_gptr[0] != 0 || h_gptr[count] != n) fail(SPHYNX_ERR_INVALID_ARG, "graph offsets must span [0, n)");
    for (int gi = 0; gi < count; ++gi)
      if (h_gptr[gi + 1] < h_gptr[gi]) fail(SPHYNX_ERR_INVALID_ARG, "graph offsets must not decrease");
    SPX_CUDA(cudaMemcpyAsync(dgptr, h_gptr, static_cast<size_t>(count + 1) * 8, cudaMemcpyHostToDevice, st));
  }
  SPX_CUDA(cudaMemsetAsync(hist, 0, static_cast<size_t>(K) * bins * 16, st));
  SPX_CUDA(cudaMemsetAsync(misc, 0, 64, st));

  k_mj_init<<<mj_grid(n), 256, 0, st>>>(perm, keys, n, coords, dti, ldc, dims, vw, misc,
                                        reinterpret_cast<unsigned *>(misc + 1));
  SPX_LAUNCHED();
  unsigned long long head[2] = {0, 0};   // total weight, bad flags
  SPX_CUDA(cudaMemcpyAsync(head, misc, sizeof(head), cudaMemcpyDeviceToHost, st));
  SPX_CUDA(cudaStreamSynchronize(st));
  const unsigned long long wtot = head[0];
  if (head[1] & 1u) fail(SPHYNX_ERR_INVALID_ARG, "NaN coordinate");
  if (head[1] & 2u) fail(SPHYNX_ERR_INVALID_ARG, "vertex weight below 1");
  // k * cumW must fit in int64: K <= 2^20 and W < 2^40
  if (wtot >= (1ull << 40)) fail(SPHYNX_ERR_UNSUPPORTED, "total vertex weight >= 2^40");
  int64_t launches = 2;
  if (count == 1) {
    k_mj_level0<<<1, 1, 0, st>>>(tab[0][0], tab[0][1], tab[0][2], n, misc, sec);
    SPX_LAUNCHED();
  } else {
    // first level: graph gi is section gi, vertices [gptr[gi], gptr[gi + 1])
    std::vector<long long> hs(count), he(count), hw(count);
    for (int gi = 0; gi < count; ++gi) {
      hs[gi] = h_gptr[gi];
      he[gi] = h_gptr[gi + 1];
      hw[gi] = h_gptr[gi + 1] - h_gptr[gi];
    }
    SPX_CUDA(cudaMemcpyAsync(tab[0][0], hs.data(), count * 8, cudaMemcpyHostToDevice, st));
    SPX_CUDA(cudaMemcpyAsync(tab[0][1], he.data(), count * 8, cudaMemcpyHostToDevice, st));
    if (vw) {
      k_mj_graph_weights<<<count, 256, 0, st>>>(vw, dgptr, tab[0][2]);
      SPX_LAUNCHED();
      ++launches;
    } else {
      SPX_CUDA(cudaMemcpyAsync(tab[0][2], hw.data(), count * 8, cudaMemcpyHostToDevice, st));
    }
    SPX_CUDA(cudaMemsetAsync(sec, 0, static_cast<size_t>(count) * sizeof(MjSec), st));
    SPX_CUDA(cudaStreamSynchronize(st));   // the host vectors above go out of scope
  }

  int idbits = 1;
  while (idbits < 32 && (1ll << idbits) < n) ++idbits;
  // digits from the top, the key's and then the id's
  std::vector<Digit> digits;
  for (int half = 0; half < 2; ++half) {
    const int total = half ? idbits : (dt == DT::F64 ? 64 : 32);
    for (int top = total; top > 0;) {
      const int w = top < plan.bits ? top : plan.bits;
      top -= w;
      digits.push_back(Digit{half, top, w, digits.empty() ? 1 : 0});
    }
  }
  const unsigned chunks = static_cast<unsigned>((n + kMjChunk - 1) / kMjChunk);
  const size_t hsm = static_cast<size_t>(bins) * (vw ? 12 : 4);
  if (nlev == 1) {   // one part a graph
    const int S = static_cast<int>(levels[0].k.size());
    const int *ks = dtab + off[0];
    k_mj_parts<<<chunks, kMjThreads, 0, st>>>(perm, n, KeySrc{keys, coords, dti, ldc, 0}, tab[0][0], S, ks + S,
                                              ks + 2 * S, sec, ks + 3 * S, part);
    SPX_LAUNCHED();
  }
  int cur = 0;
  for (int l = 0; l + 1 < nlev; ++l) {
    const int S = static_cast<int>(levels[l].k.size());
    const int *ks = dtab + off[l];
    const int *split = ks + S;
    const int *child = ks + 2 * S;
    const int dim = l % dims;
    const KeySrc src{keys, coords, dti, ldc, dim};
    long long *start = tab[cur][0], *end = tab[cur][1], *W = tab[cur][2];
    for (const Digit &d : digits) {
      k_mj_hist<<<chunks, kMjThreads, hsm, st>>>(perm, n, src, vw, start, S, split, sec, d, bins, hist);
      SPX_LAUNCHED();
      k_mj_select<<<S, 256, 0, st>>>(hist, bins, vw ? 0 : 1, split, ks, W, sec, d);
      SPX_LAUNCHED();
    }
    long long *nstart = tab[cur ^ 1][0], *nend = tab[cur ^ 1][1], *nW = tab[cur ^ 1][2];
    k_mj_decide<<<(S + 127) / 128, 128, 0, st>>>(S, split, ks, child, start, end, W, sec, nstart, nend, nW, sec2);
    SPX_LAUNCHED();
    launches += 2 + 2 * static_cast<int64_t>(digits.size());
    if (l + 2 == nlev) {
      const int *lo = dtab + off[nlev - 1] + 3 * levels[nlev - 1].k.size();
      k_mj_parts<<<chunks, kMjThreads, 0, st>>>(perm, n, src, start, S, split, child, sec, lo, part);
      SPX_LAUNCHED();
      break;
    }
    k_mj_scatter<<<chunks, kMjThreads, 0, st>>>(perm, perm2, n, src, keys2, (l + 1) % dims, start, S, split, sec);
    SPX_LAUNCHED();
    std::swap(perm, perm2);
    std::swap(keys, keys2);
    std::swap(sec, sec2);
    cur ^= 1;
  }
  if (ctr) ctr->launches += launches;
}

void run_mj(cudaStream_t st, DT dt, const void *coords, int ldc, int dims, int64_t n, const int64_t *vw, int K,
            int32_t *part, Counters *ctr) {
  size_t bytes = mj_scratch_bytes(n, K, 1, dt);
  std::unique_ptr<Scratch> scratch;
  or_least(bytes, mj_least_bytes(n, K, 1), [&] { scratch.reset(new Scratch(bytes, st)); });
  run_mj_scratch(st, dt, coords, ldc, dims, n, vw, K, part, ctr, scratch->p, bytes, nullptr, 1);
}

}  // namespace sphynx

extern "C" int sphynx_mj(int32_t dtype, const void *coords, int32_t ldc, int32_t dims, int64_t n,
                         const int64_t *vtx_w, int32_t K, int32_t *part_out, void *stream) {
  using namespace sphynx;
  return guarded([&]() -> int {
    if (n > 0 && (!coords || !part_out)) fail(SPHYNX_ERR_INVALID_ARG, "NULL argument");
    if (ldc < dims) fail(SPHYNX_ERR_INVALID_ARG, "ldc < dims");
    if (dtype != SPHYNX_DT_F32 && dtype != SPHYNX_DT_F64) fail(SPHYNX_ERR_INVALID_ARG, "dtype");
    // sizes are checked before the scratch is sized from them
    if (n < 0) fail(SPHYNX_ERR_INVALID_ARG, "n < 0");
    if (K < 1) fail(SPHYNX_ERR_INVALID_ARG, "K must be >= 1");
    if (K > (1 << 20)) fail(SPHYNX_ERR_UNSUPPORTED, "K > 2^20");
    if (n >= (1LL << 31)) fail(SPHYNX_ERR_UNSUPPORTED, "n >= 2^31");
    run_mj(static_cast<cudaStream_t>(stream), static_cast<DT>(dtype), coords, ldc, dims, n, vtx_w, K, part_out,
           nullptr);
    return SPHYNX_OK;
  });
}

// ---- multi-jagged without any device allocation ------------------------------
//
// Some callers cannot let a library call cudaMalloc: a framework whose own
// caching allocator has already reserved the device's memory, or an
// application that budgets all device memory at start-up and allows no
// allocation afterwards.  For them sphynx_mj_noalloc does the same work as
// sphynx_mj with its scratch (permutations, histograms, section tables) in
// this file-scope device array.  Every GPU that loads the library holds the
// array until the process exits.  The call still synchronises its stream
// (run_mj_scratch reads a flag and the total vertex weight back).

constexpr size_t kMjStaticBytes = size_t(16) << 20;   // 16 MiB
static __device__ __align__(256) unsigned char g_mj_static_scratch[kMjStaticBytes];

namespace {

// Device address of the array, per device.  In host code the array's name is
// only a host-side stand-in, so the address comes from cudaGetSymbolAddress,
// called once per device with that device current.
std::mutex g_mj_static_mutex;
void *g_mj_static_ptr[64] = {nullptr};

void *mj_static_scratch() {
  int dev = 0;
  SPX_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) sphynx::fail(SPHYNX_ERR_UNSUPPORTED, "device ordinal %d", dev);
  std::lock_guard<std::mutex> lock(g_mj_static_mutex);
  if (!g_mj_static_ptr[dev]) {
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_mj_static_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      sphynx::fail(SPHYNX_ERR_CUDA, "cudaGetSymbolAddress of the multi-jagged scratch failed: %s", cudaGetErrorString(e));
    }
    g_mj_static_ptr[dev] = p;
  }
  return g_mj_static_ptr[dev];
}

}  // namespace

extern "C" int sphynx_mj_noalloc(int32_t dtype, const void *coords, int32_t ldc, int32_t dims, int64_t n,
                                 const int64_t *vtx_w, int32_t K, int32_t *part_out, void *stream) {
  using namespace sphynx;
  return guarded([&]() -> int {
    if (n > 0 && (!coords || !part_out)) fail(SPHYNX_ERR_INVALID_ARG, "NULL argument");
    if (ldc < dims) fail(SPHYNX_ERR_INVALID_ARG, "ldc < dims");
    if (dtype != SPHYNX_DT_F32 && dtype != SPHYNX_DT_F64) fail(SPHYNX_ERR_INVALID_ARG, "dtype");
    if (n < 0) fail(SPHYNX_ERR_INVALID_ARG, "n < 0");
    if (K < 1) fail(SPHYNX_ERR_INVALID_ARG, "K must be >= 1");
    if (K > (1 << 20)) fail(SPHYNX_ERR_UNSUPPORTED, "K > 2^20");
    const size_t need = mj_least_bytes(n, K, 1);
    if (need > kMjStaticBytes)
      fail(SPHYNX_ERR_UNSUPPORTED,
           "sphynx_mj_noalloc: n = %lld, K = %d need %zu bytes of scratch, more than its fixed %zu "
           "(e.g. n <= 2^20 with K <= 1024 fits); use sphynx_mj",
           static_cast<long long>(n), K, need, kMjStaticBytes);
    void *scratch = mj_static_scratch();
    // run_mj_scratch clears the histograms and counters it relies on and
    // rewrites everything else it reads
    run_mj_scratch(static_cast<cudaStream_t>(stream), static_cast<DT>(dtype), coords, ldc, dims, n, vtx_w, K,
                   part_out, nullptr, scratch, kMjStaticBytes, nullptr, 1);
    return SPHYNX_OK;
  });
}
