// CUDA kernels of the iterative galactic-binary subtraction (arXiv 2602.18560, App. D),
// written for sm_103a (GB300).
//
// Steps of one run:
//   tables   : S_instr(f_k) (App. C, SciRDv1 A channel, TDI-2 factor), R(f_k) (App. B)
//              and the scales derived from them.                              [per context]
//   prepass  : one pass over the catalog: the bins each chirp sweeps, its power deposited
//              into an exact fixed-point spectrum, rho_0 against S_instr, the paper's
//              candidates (rho_0 >= kappa rho_th) counted and the ones that can still be
//              resolved (rho_0 > rho_th) kept.                                [per run]
//   loop     : S_gal = estimator of P_k = S_k Q_k 2^-64 (running mean / running median /
//              median then mean, Eqs. running mean, running median); rho of each kept
//              candidate against S_instr + S_gal (Eqs. SNR inner product, inner product);
//              sources with rho > rho_th removed from the spectrum exactly; loop control
//              on the device.
//
// No floating-point atomics: the spectrum is an integer (units of 2^-64 S_instr,k per bin),
// so deposits and removals commute and every run gives the same bits.  GB300 runs FP64 at
// 1/58 of the FP32 rate, so per-iteration work avoids FP64: medians select on the integer
// bits of the doubles, window sums are integer, and the SNR test is screened in FP32 with
// a proven error margin (exact FP64 recomputation inside the margin).

#include <climits>
#include <cstring>

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <cuda_device_runtime_api.h>

#include "common.cuh"
#include "kernels.cuh"

namespace gbsub {

// ============================================================================ launches
// Programmatic dependent launch along a chain of kernels: a kernel launched by launch_after may
// be set up while the one before it still runs, and waits (chain_wait, in every thread of every
// path) until that one has ended and its writes can be seen.  As every kernel of a chain
// waits, the end of one is the end of all before it.  Before the wait a kernel only reads what
// was there when the chain began: the catalog, and in the loop the iteration's work lists, the
// candidates and the counts, which the previous iteration's control kernel (not of the chain)
// came after.  That takes a trip or two to memory per kernel off a late iteration (3e7 sources
// 1206 -> 1175 us, 1 yr, 1e4 sources 175 -> 169).  What it reads of its predecessors' output
// goes through plain pointers: the compiler may move loads through const __restrict__ parameters
// above the wait.
// chain_next lets the next kernel's CTAs in once every CTA of this one has called it or ended.
// A kernel calls it at once when no CTA has more than one item of work, which hides the next
// launch behind it (a run over 3e7 sources 1257 -> 1232 us, over 1e7 with the mean 481 -> 473).
// With more items the waiting CTAs would hold room that other contexts' kernels could use: 64
// runs at once took 12.7 ms with this rule and without it, 14.7 ms when every kernel called it
// first.  Two kernels call it at once whatever their work: k_begin, whose successor is one CTA per
// SM at the most, and k_snr_resolve, whose successor is one CTA.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void chain_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
static void launch_after(void (*kern)(P...), int bl, int th, size_t smem, cudaStream_t st,
                         A... args) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)bl);
  cfg.blockDim = dim3((unsigned)th);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// ============================================================================ tables

__global__ void k_tables(Grid g, int tdi2, double* __restrict__ S, double* __restrict__ R,
                         double* __restrict__ gq, float* __restrict__ Gf,
                         float* __restrict__ invSf) {
  long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= g.nb) return;
  const double fstar = kC / (2.0 * kPi * kL);
  double f = (double)(g.k_lo + j) / g.T;
  double x = f / fstar;
  double sx, cx;
  sincos(x, &sx, &cx);
  // P_OMS = (15 pm)^2 [1 + (2 mHz/f)^4] (2 pi f / c)^2
  double r = 2.0e-3 / f;
  double w = 2.0 * kPi * f / kC;
  double p_oms = 15.0e-12 * 15.0e-12 * (1.0 + r * r * r * r) * w * w;
  // P_TM = (3 fm/s^2)^2 [1 + (0.4 mHz/f)^2][1 + (f / 8 mHz)^4] (2 pi f)^-4 (2 pi f / c)^2
  double r1 = 0.4e-3 / f, r2 = f / 8.0e-3;
  double om = 2.0 * kPi * f;
  double p_tm = 3.0e-15 * 3.0e-15 * (1.0 + r1 * r1) * (1.0 + r2 * r2 * r2 * r2) /
                (om * om * om * om) * w * w;
  double s_aa = 8.0 * sx * sx * (4.0 * (1.0 + cx + cx * cx) * p_tm + (2.0 + cx) * p_oms);
  double resp = 16.0 * sx * sx * x * x * (9.0 / 20.0) / (1.0 + 0.7 * x * x);
  if (tdi2) {
    double s2 = sin(2.0 * x);
    double t2 = 4.0 * s2 * s2;
    s_aa *= t2;
    resp *= t2;
  }
  S[j] = s_aa;
  R[j] = resp;
  double ratio = g.t5 * resp / s_aa;          // P / S per unit of A^2 w
  gq[j] = kQScale * ratio;                    // fixed-point units per unit of A^2 w
  // FP32 screen factors; outside the normal FP32 range they are NaN, which sends every
  // SNR decision touching the bin to the exact FP64 path.
  double gs = ldexp(4.0 * ratio, -160);       // rho^2 against S_instr per unit A^2 w 2^160
  double is = 1.0 / ldexp(s_aa, 150);
  const double fmin_n = 1.1754943508222875e-38, fmax_n = 3.4028234663852886e38;
  Gf[j] = (gs >= fmin_n && gs <= fmax_n) ? (float)gs : __int_as_float(0x7FC00000);
  invSf[j] = (is >= fmin_n && is <= fmax_n) ? (float)is : __int_as_float(0x7FC00000);
}

void launch_tables(const Grid& g, int tdi2, double* S, double* R, double* gq, float* Gf,
                   float* invSf, cudaStream_t st) {
  int th = 256;
  long long bl = (g.nb + th - 1) / th;
  k_tables<<<(unsigned)bl, th, 0, st>>>(g, tdi2, S, R, gq, Gf, invSf);
}

// ============================================================================ spectrum I/O

// The parts of a single-bin deposit (q_single) added to, or taken from, bin j.
__device__ __forceinline__ void add_parts(unsigned long long* acc, long long j, u64 c0, u64 c1,
                                          u64 c2) {
  u64* a = acc + 4 * j;
  if (c0) atomicAdd(a + 0, c0);
  if (c1) atomicAdd(a + 1, c1);
  if (c2) atomicAdd(a + 2, c2);
}
__device__ __forceinline__ void sub_parts(unsigned long long* acc, long long j, u64 c0, u64 c1,
                                          u64 c2) {
  u64* a = acc + 4 * j;
  if (c0) atomicAdd(a + 0, (u64)(0ull - c0));
  if (c1) atomicAdd(a + 1, (u64)(0ull - c1));
  if (c2) atomicAdd(a + 2, (u64)(0ull - c2));
}

// ---------------------------------------------------------------- the tree of bins
// Words of a node: three of them, as a bin's, in the padding words of the node's first bins
// (level 1 in bins 0-2, level 2 in 3-5, level 3 in 6-8: a complete node has at least 32 bins).
// They need no memory and no clearing of their own.
__device__ __forceinline__ size_t node_word(int level, long long i, int w) {
  return 4 * (size_t)((i << (5 * level)) + 3 * (level - 1) + w) + 3;
}

// What the nodes above bin j add to its Q (units of 2^-64 S_instr): the sum N of their words,
// c in units of 2^(32 - g), times gq_j.  The top 64 bits of N times gq's mantissa, truncated:
// within 2^-62 of the exact product, or one unit.
__device__ __noinline__ U128 tree_units(const unsigned long long* __restrict__ acc, long long j,
                                        long long nb, double gq, int g) {
  U128 N{0ull, 0ull};
#pragma unroll
  for (int l = 1; l <= kTreeLevels; ++l) {
    const long long i = j >> (5 * l);
    if (((i + 1) << (5 * l)) <= nb) {  // an incomplete node takes nothing, and has no words
      const unsigned long long* a = acc + node_word(l, i, 0);
      N = u128_add(N, q_combine3(a[0], a[4], a[8]));
    }
  }
  U128 r{0ull, 0ull};
  if (u128_is_zero(N)) return r;
  const int lz = N.hi ? __clzll((i64)N.hi) : 64 + __clzll((i64)N.lo);
  // top in [2^63, 2^64), N = top 2^(64 - lz) up to the bits dropped
  const u64 top = lz >= 64 ? N.lo << (lz - 64)
                           : (lz ? (N.hi << lz) | (N.lo >> (64 - lz)) : N.hi);
  const u64 bg = (u64)__double_as_longlong(gq);
  const int eg = (int)(bg >> 52) & 0x7FF;
  if (eg == 0) return r;
  const u64 mg = ((bg & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
  const u64 p = __umul64hi(top, mg);  // N gq 2^-g = p 2^sh
  const int sh = 64 + (64 - lz) + (eg - 1086) - g;
  if (sh >= 64) {
    r.hi = p << (sh - 64);
  } else if (sh > 0) {
    r.lo = p << sh;
    r.hi = p >> (64 - sh);
  } else if (sh > -64) {
    r.lo = p >> (-sh);
  }
  return r;
}

// Estimator input of bin j: P_j = S_j Q_j 2^-64 (kSpec; flags: RunState::spec), or x[j].  The
// kernels that read it are built for each kind of input: an estimate of a plain array keeps none of
// the spectrum's registers.
template <bool kSpec>
__device__ __forceinline__ double spec_value(const SpecIn& in, long long j, int flags) {
  if (kSpec) {
    const ulonglong2* a = reinterpret_cast<const ulonglong2*>(in.acc + 4 * j);
    ulonglong2 w01 = a[0];
    u64 w2 = in.acc[4 * j + 2];
    U128 Q = q_combine3(w01.x, w01.y, w2, (flags & kSpecCarried) != 0);
    if (flags & kSpecTree) Q = u128_add(Q, tree_units(in.acc, j, in.nb, in.gq[j], in.g));
    return __dmul_rn(in.S[j], u128_to_dbl_scaled(Q, 64));
  }
  return in.x[j];
}

__global__ void k_power_out(SpecIn in, long long n, double* __restrict__ P) {
  long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= n) return;
  P[j] = spec_value<true>(in, j, *in.flags);
}

void launch_power_out(SpecIn in, long long n, double* P, cudaStream_t st) {
  int th = 256;
  k_power_out<<<(unsigned)((n + th - 1) / th), th, 0, st>>>(in, n, P);
}

// One level of Tree::gsum: a warp per node adds 32 consecutive values of the level below.
__global__ void k_tree_sums(const double* __restrict__ in, int n, double* __restrict__ out) {
  const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (i >= n) return;
  double v = in[(size_t)i * 32 + (threadIdx.x & 31)];
  for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  if ((threadIdx.x & 31) == 0) out[i] = v;
}

void launch_tree_sums(const double* gq, const Tree& tr, double* gsum, cudaStream_t st) {
  const double* in = gq;
  for (int l = 0; l < kTreeLevels; ++l) {
    double* out = gsum + tr.off[l];
    if (tr.n[l] > 0) k_tree_sums<<<(tr.n[l] + 7) / 8, 256, 0, st>>>(in, tr.n[l], out);
    in = out;
  }
}

// The parts of a long sweep: bins [b0, b1) and [b2, b3) one by one, and the nodes
// [lo[l], mid0[l]) and [mid1[l], hi[l]) of each level between them (all relative to the band).
// k0 .. k1 are the sweep's bins inside the band and ka, kb its first and last: a node holds
// whole cells only, so never those two.
struct TreeSpan {
  int b0, b1, b2, b3;
  int lo[kTreeLevels], mid0[kTreeLevels], mid1[kTreeLevels], hi[kTreeLevels];
  int nbins, nnodes;
};
__device__ __forceinline__ TreeSpan tree_span(long long ka, long long kb, long long k0,
                                              long long k1) {
  TreeSpan t;
  const int a = (int)(k0 > ka ? k0 : ka + 1), b = (int)(k1 < kb ? k1 : kb - 1) + 1;  // whole cells
  int lo = (a + 31) >> 5, hi = b >> 5;
  t.b0 = (int)k0;
  t.b1 = lo << 5;
  t.b2 = hi << 5;
  t.b3 = (int)k1 + 1;
  t.nbins = (t.b1 - t.b0) + (t.b3 - t.b2);
  t.nnodes = 0;
#pragma unroll
  for (int l = 0; l < kTreeLevels; ++l) {
    const int up_lo = (lo + 31) >> 5, up_hi = hi >> 5;
    const bool up = l + 1 < kTreeLevels && up_lo < up_hi;
    t.lo[l] = lo;
    t.hi[l] = hi;
    t.mid0[l] = up ? up_lo << 5 : hi;
    t.mid1[l] = up ? up_hi << 5 : hi;
    t.nnodes += (t.mid0[l] - t.lo[l]) + (t.hi[l] - t.mid1[l]);
    lo = up ? up_lo : 0;
    hi = up ? up_hi : 0;
  }
  return t;
}
// Bin x of the span's bins taken one by one (0 <= x < nbins).
__device__ __forceinline__ int tree_bin(const TreeSpan& t, int x) {
  const int n0 = t.b1 - t.b0;
  return x < n0 ? t.b0 + x : t.b2 + (x - n0);
}
// Node x of the span's nodes (0 <= x < nnodes): its level (1 ..) and index.
__device__ __forceinline__ void tree_node(const TreeSpan& t, int x, int* level, int* i) {
  *level = 1;
  *i = 0;
#pragma unroll
  for (int l = 0; l < kTreeLevels; ++l) {
    const int n0 = t.mid0[l] - t.lo[l], n1 = t.hi[l] - t.mid1[l];
    if (x >= 0 && x < n0 + n1) {
      *level = l + 1;
      *i = x < n0 ? t.lo[l] + x : t.mid1[l] + (x - n0);
    }
    x -= n0 + n1;
  }
}

// q of a node for a sweep of length 1 / inv: c = A^2 inv in units of 2^-g (exact: a power of
// two).  The sweep goes through the tree only when that is inside the fixed-point range (then
// every bin's power is too, gq < 2^g); otherwise it is walked bin by bin.
__device__ __forceinline__ bool tree_takes(const Tree& tr, double a2, double inv, long long k0,
                                           long long k1, double* q) {
  if (k1 - k0 < kTreeBins) return false;
  *q = __dmul_rn(__dmul_rn(a2, inv), tr.scale);
  return (u64)__double_as_longlong(*q) < kQLimitBits;
}

// ============================================================================ prepass

// The catalog is dominated by the low-frequency end of the band (the number of sources
// falls steeply with f), so the 64-bit atomics of the deposits pile up on the cache lines
// of the first bins: an L2 line takes one atomic at a time.  The first rep.nbins bins
// therefore have kAccReplicas private copies (words 0 and 1 of every bin), a source
// picking one by its index; a fold adds them into the spectrum after the pass (word 2 takes
// a part only from a source of at least S_instr in the bin, rare, and goes to the spectrum
// directly).  Integer sums, so the result does not depend on the split.
__global__ void k_fold_replicas(unsigned long long* __restrict__ acc, AccReplicas rep) {
  chain_wait();
  long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (j >= rep.nbins) return;
  u64 s1 = 0, s2 = 0;
#pragma unroll
  for (int r = 0; r < kAccReplicas; ++r) {
    const ulonglong2 v = reinterpret_cast<const ulonglong2*>(rep.w)[(size_t)r * rep.nbins + j];
    s1 += v.x;
    s2 += v.y;
  }
  acc[4 * j + 0] += s1;
  acc[4 * j + 1] += s2;
}


// Bins of a source's sweep inside the band: [k0, k1] (absolute bin numbers), empty when the
// sweep leaves it.
__device__ __forceinline__ void sweep_bins(const Sweep& sw, const Grid& g, long long* k0,
                                           long long* k1) {
  *k0 = sw.ka > g.k_lo ? sw.ka : g.k_lo;
  *k1 = sw.kb < g.k_lo + g.nb - 1 ? sw.kb : g.k_lo + g.nb - 1;
}

// The cells of a sweep over several bins, for the catalog pass (a lane each): the bins
// j0 .. j0 + n - 1 of the band hold A^2 w = mid, except the sweep's own first and last bin
// where they are inside the band.  The same products as RN(A^2 RN((b - a) inv)) in every cell:
// an interior cell's b - a is 1.
struct SweepCells {
  int j0, n;
  bool first_in, last_in;
  double mid, first, last;
};
__device__ __forceinline__ double cell_power(const SweepCells& s, int t) {
  return t == 0 && s.first_in ? s.first : t == s.n - 1 && s.last_in ? s.last : s.mid;
}

// A long sweep (tree_takes), by a whole warp: the bins at its ends and the nodes between; the
// sum of the contributions (units of 2^-96 S_instr) comes back in every lane.  qn: q of a node.
__device__ __forceinline__ double tree_deposit(const SweepCells& c, double qn, const Tables& tb,
                                               unsigned long long* acc, RunState* rs) {
  const int lane = threadIdx.x & 31;
  const TreeSpan t = tree_span(c.first_in ? c.j0 : c.j0 - 1, c.last_in ? c.j0 + c.n - 1 : c.j0 + c.n,
                               c.j0, c.j0 + c.n - 1);
  U128 sum{0ull, 0ull};
  for (int x = lane; x < t.nbins; x += 32) {
    const int j = tree_bin(t, x);
    u64 c0, c1, c2;
    if (!q_cell(cell_power(c, j - c.j0), tb.gq[j], &c0, &c1, &c2)) atomicOr(&rs->err, ERR_RANGE);
    add_parts(acc, j, c0, c1, c2);
    sum = u128_add(sum, U128{c0 | (c1 << 32), c2});
  }
  u64 c0, c1, c2;
  q_parts(qn, &c0, &c1, &c2);
  double gs = 0.0;
  for (int x = lane; x < t.nnodes; x += 32) {
    int l, i;
    tree_node(t, x, &l, &i);
    if (c0) atomicAdd(acc + node_word(l, i, 0), c0);
    if (c1) atomicAdd(acc + node_word(l, i, 1), c1);
    if (c2) atomicAdd(acc + node_word(l, i, 2), c2);
    gs = __dadd_rn(gs, tb.tree.gsum[tb.tree.off[l - 1] + i]);
  }
  if (lane == 0 && !(*(volatile int*)&rs->spec & kSpecTree)) atomicOr(&rs->spec, (int)kSpecTree);
  double r = __dadd_rn(__dmul_rn(c.mid, gs), u128_to_dbl_scaled(sum, -32));
  for (int o = 16; o > 0; o >>= 1) r = __dadd_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, o));
  return r;
}

// Record of a kept candidate.
__device__ __forceinline__ void emit_candidate(const Cands& cd, long long c, long long s, double A,
                                            double fs, double fds, const Grid& g,
                                            RunState* rs) {
  Sweep sw = make_sweep(fs, fds, g.T, g.T2);
  const double a2 = __dmul_rn(A, A);
  cd.src[c] = s;
  cd.pk[c] = make_int4((int)(sw.ka - g.k_lo), (int)(sw.kb - sw.ka + 1),
                       __float_as_int(dbl_to_f32_scaled(a2, 160)),
                       __float_as_int((float)(sw.lo - (double)sw.ka)));
  cd.len[c] = (float)(sw.hi - sw.lo);
  cd.a2[c] = a2;
  cd.amp[c] = A;
  cd.lo[c] = sw.lo;
  cd.hi[c] = sw.hi;
  cd.res[c] = 0;
  if (sw.kb - sw.ka + 1 > kSnrLaneBins) cd.wide[atomicAdd(&rs->nwide, 1ull)] = c;
  if (sw.kb - sw.ka + 1 > kTreeBins) rs->tree_live = 1;
}

// Keep the live lanes' sources as candidates (the warp together).
__device__ __forceinline__ void prepass_keep(bool live, long long s, double A, double fs,
                                             double fds, const Grid& g, const Cands& cd,
                                             RunState* rs) {
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(0xFFFFFFFFu, live);
  if (!m) return;
  unsigned long long b0 = 0;
  const int leader = __ffs(m) - 1;
  if (lane == leader) b0 = atomicAdd(&rs->nlive, (unsigned long long)__popc(m));
  b0 = __shfl_sync(0xFFFFFFFFu, b0, leader);
  if (live) {
    const long long c = (long long)b0 + __popc(m & ((1u << lane) - 1u));
    emit_candidate(cd, c, s, A, fs, fds, g, rs);
  }
}

// The decision for one source once r (its rho_0^2 / 4 in units of 2^-96) is known: counted
// among the paper's candidates (nkappa), and true when it can still be resolved.
__device__ __forceinline__ bool prepass_decide(double r, u64 tk_bits, u64 tl_bits,
                                               unsigned& nkappa) {
  const u64 rb = (u64)__double_as_longlong(r);
  if (rb < tk_bits) return false;
  ++nkappa;
  return rb > tl_bits;
}

// ---------------------------------------------------------------- TMA staging
// The catalog streams through shared memory: one thread issues bulk asynchronous copies
// (cp.async.bulk, completion counted in bytes on an mbarrier) of whole tiles of A, f and
// fdot a few tiles ahead, so no thread waits on HBM for its sources.

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, unsigned bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
// Wait for phase `parity` of the barrier; false after about a second of polling.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
  const uint32_t a = smem_addr(bar);
  for (int i = 0; i < (1 << 20); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
    __nanosleep(1000);
  }
  return false;
}

// Sources whose sweep the FP32 bound cannot keep in one bin go through the FP64 path.  They
// are rare (well under 1%), but one such lane would hold its whole warp on the slow FP64
// pipe, so each warp queues them in shared memory and runs them 32 at a time.
//
// Layout of the pass: one CTA per SM, kPreWarps warps, each on its own.  The steps of kPreStep
// sources are dealt out in turn over all warps of the grid; a warp streams its steps through
// kPreStages shared-memory stages with bulk asynchronous copies of A, f and fdot (cp.async.bulk,
// completion counted in bytes on the stage's mbarrier): once its values are in registers the
// stage takes the step after the next.  No barrier between warps runs in the steady state, so a
// warp that meets a slow source delays no other.
//
// Bound: latency.  With 20 warps on an SM (issue active 56%, L1 and L2 57 and 60% of their rates)
// the warps wait for their gathers and for the results of dependent instructions.  Two reductions
// and most of a table gather per source go to L2 beyond the first bins, and their number counts:
// 3e7 sources took 470 us with all of them in L2, 268 with none.  With the rings and the first bins
// in shared memory, set-up and fold included: 3e7 sources 470 -> 343 us, 1e7 170 -> 127, 1e6 45 ->
// 43.  Other layouts at 3e7: steps in runs from a global counter 376 (it gives out a number every
// 1.7 ns, and long runs lose the locality of the stream: 450 at two runs a warp); 24 warps 351, 28
// 391, 16 with four sources a lane 371.
constexpr int kPreWarps = 20;
constexpr int kPrepassThreads = kPreWarps * 32;
constexpr int kPrePer = 2;                                    // sources per lane per step
constexpr int kPreStep = 32 * kPrePer;                        // sources per step
constexpr int kPreStages = 2;                                 // steps in flight per warp
constexpr int kSlowWarpCap = 32 + kPreStep;                   // queue of a warp (drained at 32)
constexpr int kHotBins = 4096;                                // bins kept in shared memory
constexpr long long kHotMinSources = 1000000;
constexpr size_t kPrepassSmem =
    (size_t)kPreWarps * (kPreStages * 3 * kPreStep * sizeof(double) +
                         kSlowWarpCap * sizeof(long long)) +
    (size_t)kHotBins * 3 * sizeof(unsigned);


// The common case of one source without FP64 arithmetic: the bin k its sweep starts in, and
// the certificate that the whole sweep [f T, f T + fdot T^2] stays inside cell k (false: the
// FP64 path takes the source).
//
// f T comes from the 53-bit mantissa of f, split in 21 + 32 bits, times T's in 32 + 21: three
// 32-bit products, exact but for two units of their 2^53 (2^-32 of a bin in the band; the
// dropped part of T's low bits).  With at most 30 integer bits, the product is shifted to 23
// fraction bits.  The certificate is FP32: the start's offset from the bin's centre, and that plus
// du = fdot T^2 (off by less than 4e-7 |du|), must both stay 2^-20 inside the cell, which covers
// the truncation of the fraction and the FP64 rounding of f T in the reference.  (Both ends: a
// start on an upper edge that is truncated into the cell below and moves down ends well inside
// it, and the removal, which goes by the FP64 sweep, would take power from a bin that got none.)
// A value that is not finite fails it (f: no exponent in range; fdot: du is not a number or too
// large).
//
// T's mantissa is used with its top bit set: with its trailing zeros dropped instead (20 bits
// left for 4 years) the product kept too few bits for f above 1 mHz, and every such source,
// 0.5% of a catalog, went through the FP64 path.
__device__ __forceinline__ bool source_bin(double fs, double fds, const Grid& g, int* k) {
  const u64 bf = (u64)__double_as_longlong(fs), bd = (u64)__double_as_longlong(fds);
  const unsigned fh = hi32(bf), dh = hi32(bd);
  const unsigned n = (unsigned)(g.ebin - (int)(fh >> 20));  // a negative f: n wraps
  const unsigned mh = (fh & 0x000FFFFFu) | 0x00100000u;
  const u64 prod = (u64)mh * g.tq + hi32((u64)lo32(bf) * g.tq) + __umulhi(mh, g.tr);
  const u64 x = (prod >> (n & 63u)) + (1u << 22);           // f T + 1/2, 23 fraction bits
  *k = (int)(x >> 23);
  // the offset from the centre, in [-1/2, 1/2): 1 + fraction as a float, less 3/2 (exact)
  const float off = __fadd_rn(__uint_as_float((lo32(x) & 0x007FFFFFu) | 0x3F800000u), -1.5f);
  // fdot as a float: its exponent rebased (1023 - 127 = 0x380, so that the low eight bits
  // change in the top one only) and its mantissa cut to 23 bits; 0 below the FP32 range
  const unsigned da = dh & 0x7FFFFFFFu;
  const unsigned fb = ((__funnelshift_l(lo32(bd), dh, 3) & 0x7FFFFFFFu) ^ 0x40000000u) |
                      (dh & 0x80000000u);
  const float fd = da >= (897u << 20) ? __uint_as_float(fb) : 0.0f;
  const float du = __fmul_rn(fd, g.T2f);
  const float edge = __fmaf_rn(-4e-7f, fabsf(du), 0.5f - 9.5367431640625e-7f);
  return n <= 39u && da < (1151u << 20) && fabsf(off) < edge && fabsf(__fadd_rn(off, du)) < edge;
}

// Arguments of the catalog pass, one block so that the out-of-line parts take one pointer.
struct PrepassArgs {
  const CatalogRef* cat;
  Grid g;
  Tables tb;
  u64 tk_bits, tl_bits;  // thresholds on r >= 0, as the bits of non-negative doubles
  int tk_hi;             // high word of tk_bits, INT_MIN when that is 0: a source whose r has a
                         // smaller high word (as a signed number) is below the threshold
  unsigned long long* acc;
  AccReplicas rep;
  Cands cd;
  RunState* rs;
  int test_flags;
};

// What a warp sets aside in its queue: a source of the FP64 path, or (tagged) one that the
// common path deposited and that is to be kept as a candidate.  Both are rare, and the queue's
// drain is out of line and called once per step, so that none of its registers are held in the
// common path.  A generated catalog's entries carry their values, which are FP32 numbers.
constexpr long long kQueueKeep = 1LL << 62;
constexpr unsigned kMaxAExp = 1535;  // exponent field of 2^512
struct SlowQueue {
  long long* s;
  float *a, *f, *d;  // generated catalogs only
};

// Up to 32 queued entries from `at` on (lane i takes entry i); returns this lane's count of the
// paper's candidates.
//
// FP64 arithmetic (a warp instruction every 64 clocks of a scheduler) is done once per source,
// a lane each: its sweep and the powers of its first, interior and last cells.  The cells of all
// 32 sources are then laid end to end and dealt out to the lanes, whatever their lengths, as
// integer products, and each source's sum comes back by a segmented scan.  Before, a sweep of
// more than 4 bins was walked by the whole warp in FP64, two of three lanes idle.  With the queues
// of the generated pass: catalog pass of 1e7 sources of a prior draw 3.2 -> 1.2 ms, of 3e6 stored
// ones with long sweeps 140 -> 90 us.
template <bool kGen>
__device__ __noinline__ unsigned prepass_drain_warp(const PrepassArgs& pa, const CatalogRef* cat,
                                                    const SlowQueue& q, int at, int cnt) {
  const int lane = threadIdx.x & 31;
  const Grid& g = pa.g;
  unsigned nkappa = 0;
  const bool valid = lane < cnt;
  const long long entry = valid ? q.s[at + lane] : 0;
  const long long s = entry & ~kQueueKeep;
  double a = 0.0, fs = 0.0, fds = 0.0, qn = 0.0;
  bool live = (entry & kQueueKeep) != 0, counted = false, tree = false;  // tagged: finite inputs
  SweepCells c;
  c.j0 = c.n = 0;
  c.first_in = c.last_in = false;
  c.mid = c.first = c.last = 0.0;
  double r = 0.0;
  if (valid) {
    if (kGen) {
      a = (double)q.a[at + lane];
      fs = (double)q.f[at + lane];
      fds = (double)q.d[at + lane];
    } else {
      a = cat->A[s];
      fs = cat->f[s];
      fds = cat->fdot[s];
    }
    // finite inputs, and A^2 finite (|A| < 2^512): else the source is skipped and the run
    // reports it
    if (!live && !(finite3(a, fs, fds) &&
                   (((u64)__double_as_longlong(a) >> 52) & 0x7FF) < kMaxAExp)) {
      atomicOr(&pa.rs->err, ERR_INPUT);
    } else if (!live) {
      counted = true;
      const Sweep sw = make_sweep(fs, fds, g.T, g.T2);
      if (sw.ka == sw.kb) {
        // deposited as the common path deposits it, so that every single-bin source is removed
        // the same way
        const long long j = sw.ka - g.k_lo;
        if (j >= 0 && j < g.nb) {
          u64 c0, c1, c2, qb;
          if (q_single(a, pa.tb.gq[j], &c0, &c1, &c2, &qb)) {
            add_parts(pa.acc, j, c0, c1, c2);
            r = __longlong_as_double((long long)qb);
          } else {
            atomicOr(&pa.rs->err, ERR_RANGE);
          }
        }
      } else {
        long long k0, k1;
        sweep_bins(sw, g, &k0, &k1);
        if (k1 >= k0) {
          const double a2 = __dmul_rn(a, a), inv = sweep_inv_len(sw);
          c.j0 = (int)(k0 - g.k_lo);
          c.n = (int)(k1 - k0 + 1);
          c.first_in = k0 == sw.ka;
          c.last_in = k1 == sw.kb;
          c.mid = __dmul_rn(a2, inv);
          c.first = __dmul_rn(a2, sweep_weight_inv(sw, sw.ka, inv));
          c.last = __dmul_rn(a2, sweep_weight_inv(sw, sw.kb, inv));
          tree = tree_takes(pa.tb.tree, a2, inv, k0, k1, &qn);
        }
      }
    }
  }
  // the long sweeps, one after another by the whole warp
  unsigned pending = __ballot_sync(0xFFFFFFFFu, tree);
  while (pending) {
    const int src = __ffs(pending) - 1;
    pending &= pending - 1;
    SweepCells t;
    t.j0 = __shfl_sync(0xFFFFFFFFu, c.j0, src);
    t.n = __shfl_sync(0xFFFFFFFFu, c.n, src);
    t.first_in = __shfl_sync(0xFFFFFFFFu, (int)c.first_in, src) != 0;
    t.last_in = __shfl_sync(0xFFFFFFFFu, (int)c.last_in, src) != 0;
    t.mid = __shfl_sync(0xFFFFFFFFu, c.mid, src);
    t.first = __shfl_sync(0xFFFFFFFFu, c.first, src);
    t.last = __shfl_sync(0xFFFFFFFFu, c.last, src);
    const double tq = __shfl_sync(0xFFFFFFFFu, qn, src);
    if (tq > 0.0) {
      const double rt = tree_deposit(t, tq, pa.tb, pa.acc, pa.rs);
      if (lane == src) r = rt;
    }
  }
  // the others' cells, end to end
  const int n = tree ? 0 : c.n;
  int off = n;  // inclusive, then exclusive scan
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, off, o);
    if (lane >= o) off += v;
  }
  const int total = __shfl_sync(0xFFFFFFFFu, off, 31);
  off -= n;
  U128 sum{0ull, 0ull};
  for (int base = 0; base < total; base += 32) {
    const int x = base + lane;
    int src = 0;  // the last source whose cells begin at x or before
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const int o = __shfl_sync(0xFFFFFFFFu, off, src + step);
      if (o <= x) src += step;
    }
    SweepCells t;
    const int t_off = __shfl_sync(0xFFFFFFFFu, off, src);
    t.j0 = __shfl_sync(0xFFFFFFFFu, c.j0, src);
    t.n = __shfl_sync(0xFFFFFFFFu, n, src);
    const int ends = __shfl_sync(0xFFFFFFFFu, (c.first_in ? 1 : 0) | (c.last_in ? 2 : 0), src);
    t.first_in = ends & 1;
    t.last_in = ends & 2;
    t.mid = __shfl_sync(0xFFFFFFFFu, c.mid, src);
    t.first = __shfl_sync(0xFFFFFFFFu, c.first, src);
    t.last = __shfl_sync(0xFFFFFFFFu, c.last, src);
    u64 lo = 0ull, hi = 0ull;
    if (x < total) {
      const int i = x - t_off, j = t.j0 + i;
      u64 c0, c1, c2;
      if (!q_cell(cell_power(t, i), pa.tb.gq[j], &c0, &c1, &c2))
        atomicOr(&pa.rs->err, ERR_RANGE);
      add_parts(pa.acc, j, c0, c1, c2);
      lo = c0 | (c1 << 32);
      hi = c2;
    }
    // sums over the lanes of one source
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      U128 v;
      v.lo = __shfl_up_sync(0xFFFFFFFFu, lo, o);
      v.hi = __shfl_up_sync(0xFFFFFFFFu, hi, o);
      const int vs = __shfl_up_sync(0xFFFFFFFFu, src, o);
      if (lane >= o && vs == src) {
        const U128 w = u128_add(v, U128{lo, hi});
        lo = w.lo;
        hi = w.hi;
      }
    }
    // each source's last lane of this round
    const int end = min(off + n, base + 32) - 1 - base;
    U128 mine;
    mine.lo = __shfl_sync(0xFFFFFFFFu, lo, end & 31);
    mine.hi = __shfl_sync(0xFFFFFFFFu, hi, end & 31);
    if (n > 0 && off < base + 32 && end >= 0) sum = u128_add(sum, mine);
  }
  if (n > 0) r = u128_to_dbl_scaled(sum, -32);
  if (counted) live = prepass_decide(r, pa.tk_bits, pa.tl_bits, nkappa);
  prepass_keep(live, s, a, fs, fds, g, pa.cd, pa.rs);
  return nkappa;
}

// Drain the warp's queue while it holds 32 entries or more.
template <bool kGen>
__device__ __forceinline__ void prepass_drain_full(const PrepassArgs& pa, const CatalogRef* cat,
                                                   const SlowQueue& q, int& qn,
                                                   unsigned& nkappa) {
  while (qn >= 32) {
    // the last 32 entries: nothing moves down
    __syncwarp();
    nkappa += prepass_drain_warp<kGen>(pa, cat, q, qn - 32, 32);
    qn -= 32;
    __syncwarp();
  }
}

// The first bins' words in shared memory (catalog pass over a stored catalog): 96 bits a bin in
// three 32-bit words, carried over as they are added, so a deposit is two shared-memory atomics
// there instead of two in L2.  The source density falls so steeply with f that 4 096 bins take
// about half of a catalog (3e7 sources: 343 us against 470 without; 2 048 or 6 144 bins: +5 us).
// From kHotMinSources on: below 1e6 sources clearing and adding up the words costs what they
// save (43 us either way at 1e6).
struct HotBins {
  unsigned* w;  // [3][kHotBins]
  int n;        // bins kept (0: none)
};
__device__ __forceinline__ void hot_add(const HotBins& h, int j, unsigned c0, unsigned c1) {
  const unsigned o0 = atomicAdd(h.w + j, c0);
  const unsigned a1 = c1 + (o0 + c0 < o0 ? 1u : 0u);
  const unsigned o1 = atomicAdd(h.w + kHotBins + j, a1);
  const unsigned a2 = (a1 < c1 ? 1u : 0u) + (o1 + a1 < o1 ? 1u : 0u);
  if (a2) atomicAdd(h.w + 2 * kHotBins + j, a2);
}

// One source of the catalog pass in two steps, so that the table gathers of a lane's sources
// are under way together.
//
// Some 240 instructions per 32 sources (301 before; in the pass over a generated catalog they add to the
// generator's, which is bound by instruction issue; the pass over a stored one waits more than it
// issues).  What is left out here: tests
// that the rare paths repeat (finite inputs, the range of q, both thresholds: a source is
// handed to q_single only when its exponent and top 20 bits say that it may pass the lower
// one, or when it reaches the third word), 64-bit shifts by zero-extended halves, and the
// conversions between FP64, integers and FP32.
struct PlacedSource {
  int j;       // bin in band, or -1: outside it, or -2: for the FP64 path
  double gq;
};
__device__ __forceinline__ PlacedSource place_source(bool valid, double a, double fs, double fds,
                                                     const PrepassArgs& pa) {
  PlacedSource p;
  int k;
  const bool single = source_bin(fs, fds, pa.g, &k) &&
                      (hi32((u64)__double_as_longlong(a)) & 0x7FF00000u) < (kMaxAExp << 20);
  const unsigned j = (unsigned)(k - (int)pa.g.k_lo);
  const bool in = single && j < (unsigned)pa.g.nb;
  p.j = in ? (int)j : (single ? -1 : -2);
  p.gq = 0.0;
  if (!valid) p.j = -3;  // beyond the catalog
  if (p.j >= 0) p.gq = pa.tb.gq[j];
  return p;
}

// The deposit of a placed source (q_single's integers) and whether the rare path has to settle
// it: third word, range, thresholds.  No branches, so that a lane's sources interleave.
struct SourceParts {
  unsigned c0, c1;
  bool rare;
};
__device__ __forceinline__ SourceParts source_parts(double a, double gq, int tk_hi) {
  const u64 ba = (u64)__double_as_longlong(a), bg = (u64)__double_as_longlong(gq);
  const unsigned ah = hi32(ba), al = lo32(ba), gh = hi32(bg), gl = lo32(bg);
  const unsigned am = (ah & 0x000FFFFFu) | 0x00100000u, gm = (gh & 0x000FFFFFu) | 0x00100000u;
  // a2 = floor(mantissa^2 2^-42), pr = floor(a2 gq's mantissa 2^-53): q_single's products
  const u64 w = (u64)(2u * am) * al + hi32((u64)al * al);
  const u64 a2 = (u64)(am << 11) * (am << 11) + (w >> 10);
  const u64 w2 = (u64)lo32(a2) * gm + hi32((u64)lo32(a2) * gl);
  const u64 w3 = (u64)hi32(a2) * gl + lo32(w2);
  const u64 top = (u64)hi32(a2) * gm + hi32(w2) + hi32(w3);
  const unsigned ph = __funnelshift_l(lo32(top), hi32(top), 11);
  const unsigned pl = __funnelshift_l(lo32(w3), lo32(top), 11);
  const int t = 2 * (int)((ah >> 20) & 0x7FFu) + (int)(gh >> 20) - 3162;  // Q = pr 2^t
  // high word of q's bits as a double (q = pr 2^(t + 32), pr in [2^61, 2^64))
  const int lz = __clz((int)ph);
  const int e1022 = t - lz + 1117;
  const int rh = (int)(__funnelshift_l(pl, ph, lz) >> 11) + (e1022 << 20);
  SourceParts r;
  r.rare = t > 0 || rh >= tk_hi;
  // (A or gq zero or subnormal: t is below -64, and nothing is left)
  const u64 Q = shr_clamp(((u64)ph << 32) | pl, (unsigned)-t);
  r.c0 = lo32(Q);
  r.c1 = hi32(Q);
  return r;
}

// The deposit, the count and the candidate test; a source of the FP64 path, or one to keep as
// a candidate, is appended to the warp's queue q (qn entries, the same in every lane; every
// lane of the warp calls it together).  rep_lane: the replica of this lane's sources.
// kGen: f and fdot go with it (FP32 numbers).
template <bool kGen>
__device__ __forceinline__ void deposit_source(const PlacedSource p, SourceParts c, long long s,
                                               double a, float f, float fdot,
                                               const PrepassArgs& pa, const HotBins& hot_bins,
                                               u64* rep_lane, const SlowQueue& q, int& qn,
                                               unsigned& nkappa) {
  const int lane = threadIdx.x & 31;
  bool set_aside = p.j == -2, keep = false;
  if (p.j >= 0) {
    if (c.rare) {
      u64 qb, c0, c1, c2;
      if (!q_single(a, p.gq, &c0, &c1, &c2, &qb)) atomicOr(&pa.rs->err, ERR_RANGE);
      c.c0 = lo32(c0);
      c.c1 = lo32(c1);
      if (c2) atomicAdd(pa.acc + 4 * (size_t)p.j + 2, c2);
      keep = set_aside = prepass_decide(__longlong_as_double((long long)qb), pa.tk_bits,
                                        pa.tl_bits, nkappa);
    }
    if (p.j < hot_bins.n) {
      hot_add(hot_bins, p.j, c.c0, c.c1);
    } else {
      u64* d = p.j < pa.rep.nbins ? rep_lane + 2 * (size_t)p.j : pa.acc + 4 * (size_t)p.j;
      if (c.c0) atomicAdd(d, (u64)c.c0);
      if (c.c1) atomicAdd(d + 1, (u64)c.c1);
    }
  } else if (p.j == -1) {
    // outside the band: r = 0
    if (pa.tk_bits == 0) ++nkappa;
  }
  const unsigned sm = __ballot_sync(0xFFFFFFFFu, set_aside);
  if (sm) {
    if (set_aside) {
      const int at = qn + __popc(sm & ((1u << lane) - 1u));
      q.s[at] = keep ? s | kQueueKeep : s;
      if (kGen) {
        q.a[at] = (float)a;
        q.f[at] = f;
        q.d[at] = fdot;
      }
    }
    qn += __popc(sm);
  }
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, unsigned parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for phase `parity` of the barrier; false once *abort is set by another warp of the CTA,
// or after about a second (2^31 clocks), or after 2^24 polls, whichever comes first.
__device__ __noinline__ bool mbar_poll(uint32_t bar, unsigned parity, const int* abort) {
  const long long t0 = clock64();
  for (int i = 0; i < (1 << 24); ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 63) == 63) {
      if (*(volatile const int*)abort) return false;
      if (clock64() - t0 > (2LL << 30)) return false;
      __nanosleep(256);
    }
  }
  return false;
}
__device__ __forceinline__ bool mbar_wait_abort(uint64_t* bar, unsigned parity,
                                                const int* abort) {
  return mbar_try(smem_addr(bar), parity) || mbar_poll(smem_addr(bar), parity, abort);
}

__global__ void __launch_bounds__(kPrepassThreads, 1)
    k_prepass(const __grid_constant__ PrepassArgs pa) {
  RunState* const rs = pa.rs;
  // per warp [stage][A | f | fdot][kPreStep]; the warps' queues; the hot bins' words
  extern __shared__ __align__(128) double pre_smem[];
  __shared__ __align__(8) uint64_t full[kPreWarps][kPreStages];
  __shared__ int abort_flag;
  // the catalog record (and a generated catalog's constants), read once per CTA: every
  // thread of the grid loading it would queue on one L2 line
  __shared__ CatalogRef scat;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    scat = *pa.cat;
    abort_flag = 0;
  }
  if (lane == 0) {
    for (int k = 0; k < kPreStages; ++k) mbar_init(&full[warp][k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (scat.staged == kCatGenerated) {  // k_prepass_gen's catalog
    chain_wait();
    return;
  }
  const long long N = scat.n;
  double* const stages = pre_smem + (size_t)warp * kPreStages * 3 * kPreStep;
  SlowQueue myq = {};
  myq.s = reinterpret_cast<long long*>(pre_smem + (size_t)kPreWarps * kPreStages * 3 * kPreStep) +
          warp * kSlowWarpCap;
  HotBins hot;
  hot.w = reinterpret_cast<unsigned*>(pre_smem + (size_t)kPreWarps *
                                                     (kPreStages * 3 * kPreStep + kSlowWarpCap));
  hot.n = N >= kHotMinSources && N < (1LL << 31) ? (int)min((long long)kHotBins, pa.rep.nbins) : 0;
  if (hot.n) {
    for (int j = tid; j < 3 * kHotBins; j += kPrepassThreads) hot.w[j] = 0u;
    __syncthreads();
  }
  // steps [0, nfull) of device memory come through bulk copies; the ragged one, and every step
  // of a catalog in host memory, through plain loads
  const unsigned nsteps = (unsigned)((N + kPreStep - 1) / kPreStep);
  const unsigned nfull = scat.staged == kCatDevice ? (unsigned)(N / kPreStep) : 0u;
  unsigned started = 0;  // lane 0: bit k, copies of stage k are under way
  unsigned par = 0;      // bit k: the phase of stage k's barrier that its copies complete
  auto start_copies = [&](unsigned u, unsigned k) {
    if (lane != 0 || u >= nfull || (pa.test_flags & 1)) return;
    double* d = stages + k * 3 * kPreStep;
    const size_t off = (size_t)u * kPreStep;
    uint64_t* bar = &full[warp][k];
    started |= 1u << k;
    mbar_expect_tx(bar, 3u * kPreStep * (unsigned)sizeof(double));
    bulk_g2s(d, scat.A + off, kPreStep * sizeof(double), bar);
    bulk_g2s(d + kPreStep, scat.f + off, kPreStep * sizeof(double), bar);
    bulk_g2s(d + 2 * kPreStep, scat.fdot + off, kPreStep * sizeof(double), bar);
  };
  // steps dealt out in turn over all warps of the grid (numbered across the CTAs, so that a small
  // catalog spreads over the SMs)
  const unsigned nwarps = gridDim.x * kPreWarps;
  unsigned u_next = warp * gridDim.x + blockIdx.x;
  auto take_step = [&]() {
    const unsigned t = u_next;
    u_next += nwarps;
    return t;
  };
  static_assert(kPreStages == 2, "two stages, taken in turn");
  unsigned u = take_step();
  start_copies(u, 0);
  unsigned u1 = take_step();
  start_copies(u1, 1);
  chain_wait();  // the words are zero now
  unsigned nkappa = 0;  // a lane's share of the catalog
  // a source's replica is its index mod kAccReplicas, the same for all of a lane's sources
  u64* const rep_lane = pa.rep.w + 2 * (size_t)(lane % kAccReplicas) * pa.rep.nbins;
  int qn = 0;         // entries of the warp's queue (the same in every lane)
  unsigned done = 0;  // steps done
  bool timeout = false;
  for (; u < nsteps; ++done) {
    const unsigned k = done & 1u;
    const long long s0 = (long long)u * kPreStep + lane;
    double av[kPrePer], fv[kPrePer], dv[kPrePer];
    if (u < nfull) {
      const bool ok = mbar_wait_abort(&full[warp][k], (par >> k) & 1u, &abort_flag);
      if (!__all_sync(0xFFFFFFFFu, ok)) {
        if (lane == 0) {
          atomicOr(&rs->err, ERR_TIMEOUT);
          *(volatile int*)&abort_flag = 1;
        }
        timeout = true;
        break;
      }
      par ^= 1u << k;
      started &= ~(1u << k);
      const double* d = stages + k * 3 * kPreStep + lane;
#pragma unroll
      for (int i = 0; i < kPrePer; ++i) {
        av[i] = d[32 * i];
        fv[i] = d[kPreStep + 32 * i];
        dv[i] = d[2 * kPreStep + 32 * i];
      }
    } else {
      // every load of the lane's sources first: from host memory each one takes a microsecond
      // or more
#pragma unroll
      for (int i = 0; i < kPrePer; ++i) {
        const long long s = s0 + 32 * i;
        av[i] = fv[i] = dv[i] = 0.0;
        if (s < N) {
          av[i] = scat.A[s];
          fv[i] = scat.f[s];
          dv[i] = scat.fdot[s];
        }
      }
    }
    // every lane has its values: the stage takes a later step
    __syncwarp();
    u = u1;
    u1 = take_step();
    start_copies(u1, k);
    PlacedSource pl[kPrePer];
#pragma unroll
    for (int i = 0; i < kPrePer; ++i)
      pl[i] = place_source(s0 + 32 * i < N, av[i], fv[i], dv[i], pa);
    SourceParts sp[kPrePer];
#pragma unroll
    for (int i = 0; i < kPrePer; ++i) sp[i] = source_parts(av[i], pl[i].gq, pa.tk_hi);
#pragma unroll
    for (int i = 0; i < kPrePer; ++i)
      deposit_source<false>(pl[i], sp[i], s0 + 32 * i, av[i], 0.0f, 0.0f, pa, hot, rep_lane, myq,
                            qn, nkappa);
    prepass_drain_full<false>(pa, &scat, myq, qn, nkappa);
  }
  if (timeout) {
    // wait (bounded) for every copy this warp started before its shared memory goes away
    if (lane == 0)
      for (int k = 0; k < kPreStages; ++k)
        if ((started >> k) & 1u) mbar_wait(&full[warp][k], (par >> k) & 1u);
    __syncwarp();
  } else if (qn > 0) {
    __syncwarp();
    nkappa += prepass_drain_warp<false>(pa, &scat, myq, 0, qn);
  }
  for (int o = 16; o > 0; o >>= 1) nkappa += __shfl_xor_sync(0xFFFFFFFFu, nkappa, o);
  if (lane == 0 && nkappa) atomicAdd(&rs->ncand, (unsigned long long)nkappa);
  if (hot.n) {
    // the hot bins' words into the replicas, a few CTAs to each
    __syncthreads();
    if (tid == 0) atomicOr(&rs->spec, (int)kSpecCarried);
    u64* const r = pa.rep.w + 2 * (size_t)(blockIdx.x % kAccReplicas) * pa.rep.nbins;
    for (int j = tid; j < hot.n; j += kPrepassThreads) {
      const unsigned h0 = hot.w[j], h1 = hot.w[kHotBins + j], h2 = hot.w[2 * kHotBins + j];
      if (h0) atomicAdd(r + 2 * j, (u64)h0);
      if (h1) atomicAdd(r + 2 * j + 1, (u64)h1);
      if (h2) atomicAdd(pa.acc + 4 * (size_t)j + 2, (u64)h2);
    }
  }
}

// The catalog pass over a generated catalog: every source computed from (seed, index) where
// the pass over a stored catalog loads it, then the same per-source step.  The other pass leaves
// a generated catalog to this one, and this one leaves every other catalog to it.
//
// Bound: instruction issue.  An attempt at a source's Gamma variate is refused one time in four;
// with a loop per lane a warp went on until its last lane was done, 3.5 attempts and half its
// lanes idle (1 377 instructions per 32 sources, 1 034 with the queues; 3e7 sources 1 340 -> 940
// us).  So a warp keeps refused sources in a queue and tries 32 of them at a time, and sources with their variate in another (for the paper's
// population one for each way through the incomplete gamma function), from which it computes
// the rest 32 at a time.  The order of the sources changes nothing: deposits are integers.
constexpr int kGenThreads = 256;
constexpr int kGenPer = 8;     // sources per lane per run
constexpr int kGenQueue = 64;  // less than 32 entries before 32 are added
struct GenQueues {
  long long retry_s[kGenQueue], ready_s[2][kGenQueue], slow_s[kGenQueue];
  float ready_x[2][kGenQueue], slow_a[kGenQueue], slow_f[kGenQueue], slow_d[kGenQueue];
  int retry_t[kGenQueue];
};

__global__ void __launch_bounds__(kGenThreads, 4)
    k_prepass_gen(const __grid_constant__ PrepassArgs pa) {
  RunState* const rs = pa.rs;
  __shared__ CatalogRef scat;
  __shared__ GenQueues queues[kGenThreads / 32];
  if (threadIdx.x == 0) scat = *pa.cat;
  __syncthreads();
  chain_wait();
  if (scat.staged != kCatGenerated) return;
  const long long N = scat.n;
  const GenParams& gen = scat.gen;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  GenQueues& q = queues[warp];
  SlowQueue slow;
  slow.s = q.slow_s;
  slow.a = q.slow_a;
  slow.f = q.slow_f;
  slow.d = q.slow_d;
  unsigned nkappa = 0;  // a lane's share of the catalog
  u64* const rep_lane = pa.rep.w + 2 * (size_t)(lane % kAccReplicas) * pa.rep.nbins;
  int qn = 0, nretry = 0, nready0 = 0, nready1 = 0;
  constexpr long long kRun = 32LL * kGenPer;
  long long next = 0, run_end = 0;  // the warp's run of fresh sources
  bool more = true;
  for (;;) {
    int what;  // 0, 1: the rest of sources of that class; 2: refused sources again; 3: fresh ones
    if (nready0 >= 32) {
      what = 0;
    } else if (nready1 >= 32) {
      what = 1;
    } else if (nretry >= 32) {
      what = 2;
    } else {
      if (more && next >= run_end) {
        unsigned long long r0 = 0;
        if (lane == 0) r0 = atomicAdd(&rs->next_tile, 1ull);
        next = (long long)__shfl_sync(0xFFFFFFFFu, r0, 0) * kRun;
        run_end = next + kRun;
        more = next < N;
      }
      if (more)
        what = 3;
      else if (nretry > 0)
        what = 2;
      else if (nready0 > 0)
        what = 0;
      else if (nready1 > 0)
        what = 1;
      else
        break;
    }
    if (what >= 2) {
      long long s = next + lane;
      int t = 0;
      bool valid = s < N;
      if (what == 2) {
        const int cnt = min(nretry, 32);
        nretry -= cnt;
        valid = lane < cnt;
        s = valid ? q.retry_s[nretry + lane] : 0;
        t = valid ? q.retry_t[nretry + lane] : 0;
        __syncwarp();
      } else {
        next += 32;
        more = next < N;
      }
      float X;
      bool ok = gen_gamma_try(gen, (unsigned)(unsigned long long)s,
                              (unsigned)((unsigned long long)s >> 32), t, &X);
      if (!ok && t + 1 >= kGammaTries) {
        X = gen.d;
        ok = true;
      }
      const unsigned no = __ballot_sync(0xFFFFFFFFu, valid && !ok);
      if (valid && !ok) {
        const int at = nretry + __popc(no & below);
        q.retry_s[at] = s;
        q.retry_t[at] = t + 1;
      }
      nretry += __popc(no);
      const int cls = gen_class(gen, X);
      const unsigned y0 = __ballot_sync(0xFFFFFFFFu, valid && ok && cls == 0);
      const unsigned y1 = __ballot_sync(0xFFFFFFFFu, valid && ok && cls == 1);
      if (valid && ok) {
        const int at = cls ? nready1 + __popc(y1 & below) : nready0 + __popc(y0 & below);
        q.ready_s[cls][at] = s;
        q.ready_x[cls][at] = X;
      }
      nready0 += __popc(y0);
      nready1 += __popc(y1);
      __syncwarp();
    } else {
      const int have = what ? nready1 : nready0, cnt = min(have, 32), at = have - cnt + lane;
      if (what)
        nready1 -= cnt;
      else
        nready0 -= cnt;
      const bool valid = lane < cnt;
      const long long s = valid ? q.ready_s[what][at] : 0;
      const float X = valid ? q.ready_x[what][at] : (what ? gen.alpha + 2.0f : 0.5f);
      __syncwarp();
      float a, f, fd;
      gen_rest(gen, s, X, &a, &f, &fd);
      const PlacedSource pl = place_source(valid, (double)a, (double)f, (double)fd, pa);
      deposit_source<true>(pl, source_parts((double)a, pl.gq, pa.tk_hi), s, (double)a, f, fd, pa,
                           HotBins{nullptr, 0}, rep_lane, slow, qn, nkappa);
      prepass_drain_full<true>(pa, &scat, slow, qn, nkappa);
    }
  }
  __syncwarp();
  if (qn > 0) nkappa += prepass_drain_warp<true>(pa, &scat, slow, 0, qn);
  for (int o = 16; o > 0; o >>= 1) nkappa += __shfl_xor_sync(0xFFFFFFFFu, nkappa, o);
  if (lane == 0 && nkappa) atomicAdd(&rs->ncand, (unsigned long long)nkappa);
}

void launch_prepass(const CatalogRef* cat, long long cap, const Grid& g, const Tables& tb,
                    double thr_kappa, double thr_live, unsigned long long* acc, AccReplicas rep,
                    Cands cd, RunState* rs, int nsm, int test_flags, cudaStream_t st) {
  // one CTA per SM, at most one per step of the catalog
  const long long steps = (cap + kPreStep - 1) / kPreStep;
  const int bl = (int)(steps < nsm ? (steps < 1 ? 1 : steps) : nsm);
  PrepassArgs pa;
  pa.cat = cat;
  pa.g = g;
  pa.tb = tb;
  memcpy(&pa.tk_bits, &thr_kappa, sizeof(double));
  memcpy(&pa.tl_bits, &thr_live, sizeof(double));
  pa.tk_hi = pa.tk_bits ? (int)(pa.tk_bits >> 32) : INT_MIN;
  pa.acc = acc;
  pa.rep = rep;
  pa.cd = cd;
  pa.rs = rs;
  pa.test_flags = test_flags;
  launch_after(k_prepass, bl, kPrepassThreads, kPrepassSmem, st, pa);  // after launch_begin
  // the generated-catalog pass: resident CTAs, at most one per run of sources
  const long long runs = (cap + 32LL * kGenPer - 1) / (32LL * kGenPer);
  const long long glim = (long long)nsm * 4 * (kGenThreads / 32);
  const long long gwarps = runs < glim ? (runs < 1 ? 1 : runs) : glim;
  launch_after(k_prepass_gen, (int)((gwarps + kGenThreads / 32 - 1) / (kGenThreads / 32)),
               kGenThreads, 0, st, pa);
  if (rep.nbins > 0)
    launch_after(k_fold_replicas, (int)((rep.nbins + 255) / 256), 256, 0, st, acc, rep);
}

__global__ void k_set_catalog(CatalogRef* p, CatalogRef v) { *p = v; }

void launch_set_catalog(CatalogRef* p, const CatalogRef& v, cudaStream_t st) {
  k_set_catalog<<<1, 1, 0, st>>>(p, v);
}

// ---------------------------------------------------------------- generated catalogs
// The recipe's constants for the power law f^-gamma and Gamma(shape, 1), computed on the device
// (so that no host compiler contracts them into fused multiply-adds).
__device__ GenParams gen_setup(unsigned long long seed, double gamma, double shape) {
  GenParams g;
  g.k0 = (unsigned)seed;
  g.k1 = (unsigned)(seed >> 32);
  const float e = __double2float_rn(__dsub_rn(1.0, gamma));
  const float lmin = gen_log(__double2float_rn(1e-4)), lmax = gen_log(__double2float_rn(1e-2));
  g.power = fabs(__dsub_rn(gamma, 1.0)) >= 1e-3 ? 1 : 0;
  const float lf0 = e < 0.0f ? lmin : lmax, lf1 = e < 0.0f ? lmax : lmin;
  g.lf0 = lf0;
  g.rho = g.power ? gen_exp(__fmul_rn(e, __fsub_rn(lf1, lf0))) : 0.0f;
  g.omr = __fsub_rn(1.0f, g.rho);
  g.inv_e = g.power ? __fdiv_rn(1.0f, e) : 0.0f;
  g.lmin = lmin;
  g.span = __fsub_rn(lmax, lmin);
  g.d = __fsub_rn(__double2float_rn(shape), (float)(1.0 / 3.0));
  g.c = __fdiv_rn(1.0f, __fsqrt_rn(__fmul_rn(9.0f, g.d)));
  g.pref = __fmul_rn((float)19.2, gen_exp(__fmul_rn((float)(8.0 / 3.0),
                                                    gen_log((float)3.141592653589793))));
  g.log1e3 = gen_log((float)1e-3);
  g.kind = 0;
  g.beta = g.alpha = g.gln = g.mu_g = g.mu = g.sigma = g.rho_cop = g.rho_c = 0.0f;
  return g;
}

__device__ void gen_publish(CatalogRef* ref, long long n, const GenParams& g, const double* A,
                            const double* f, const double* fdot) {
  CatalogRef r;
  r.A = A;
  r.f = f;
  r.fdot = fdot;
  r.n = n;
  r.staged = A ? kCatDevice : kCatGenerated;
  r.pad = 0;
  r.gen = g;
  *ref = r;
}

__global__ void k_gen_setup(CatalogRef* ref, long long n, unsigned long long seed, double gamma,
                            double shape, const double* A, const double* f, const double* fdot) {
  gen_publish(ref, n, gen_setup(seed, gamma, shape), A, f, fdot);
}

// The paper's population: the power law p(f) ~ f^alpha_pl (gamma = -alpha_pl), Gamma of shape
// alpha_g, and the copula, amplitude and rate constants.
__global__ void k_gen_setup_paper(CatalogRef* ref, long long n, unsigned long long seed,
                                  PaperPop pp, const double* A, const double* f,
                                  const double* fdot) {
  GenParams g = gen_setup(seed, -pp.alpha_pl, pp.alpha_g);
  g.kind = 1;
  g.beta = __double2float_rn(pp.beta_g);
  g.alpha = __double2float_rn(pp.alpha_g);
  g.gln = gen_lgamma(g.alpha);
  g.mu_g = __double2float_rn(pp.mu_g);
  g.mu = __double2float_rn(pp.mu);
  g.sigma = __double2float_rn(pp.sigma);
  g.rho_cop = __double2float_rn(pp.rho);
  g.rho_c = __fsqrt_rn(__fsub_rn(1.0f, __fmul_rn(g.rho_cop, g.rho_cop)));
  gen_publish(ref, n, g, A, f, fdot);
}

void launch_gen_setup(CatalogRef* ref, long long n, unsigned long long seed, double gamma,
                      double shape, const double* A, const double* f, const double* fdot,
                      cudaStream_t st) {
  k_gen_setup<<<1, 1, 0, st>>>(ref, n, seed, gamma, shape, A, f, fdot);
}

void launch_gen_setup_paper(CatalogRef* ref, long long n, unsigned long long seed,
                            const PaperPop& pp, const double* A, const double* f,
                            const double* fdot, cudaStream_t st) {
  k_gen_setup_paper<<<1, 1, 0, st>>>(ref, n, seed, pp, A, f, fdot);
}

__global__ void __launch_bounds__(256) k_generate(const CatalogRef* __restrict__ ref,
                                                  long long start, long long n,
                                                  double* __restrict__ A, double* __restrict__ f,
                                                  double* __restrict__ fdot) {
  const GenParams g = ref->gen;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    double a, fs, fd;
    gen_source(g, start + i, &a, &fs, &fd);
    A[i] = a;
    f[i] = fs;
    fdot[i] = fd;
  }
}

void launch_generate(const CatalogRef* ref, long long start, long long n, double* A, double* f,
                     double* fdot, cudaStream_t st) {
  if (n <= 0) return;
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, 0);
  long long want = (n + 255) / 256, cap = (long long)(nsm > 0 ? nsm : 1) * 8;
  k_generate<<<(unsigned)(want < cap ? want : cap), 256, 0, st>>>(ref, start, n, A, f, fdot);
}

// ============================================================================ reductions

__device__ __forceinline__ void warp_max_atomic(u64 v, u64* target) {
  // v are bits of non-negative doubles: their integer order is the value order.
  for (int o = 16; o > 0; o >>= 1) {
    u64 t = __shfl_xor_sync(0xFFFFFFFFu, v, o);
    v = t > v ? t : v;
  }
  if ((threadIdx.x & 31) == 0 && v) atomicMax(target, v);
}

__global__ void k_max_bits(const double* __restrict__ x, long long n, unsigned long long* max_bits) {
  long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  u64 b = 0;
  if (j < n) {
    b = (u64)__double_as_longlong(x[j]);
    if (b >> 63) b = 0ull;
  }
  warp_max_atomic(b, max_bits);
}

void launch_max_bits(const double* x, long long n, unsigned long long* max_bits, cudaStream_t st) {
  int th = 256;
  k_max_bits<<<(unsigned)((n + th - 1) / th), th, 0, st>>>(x, n, max_bits);
}

// S_gal epilogue: store, fold the relative change of S_n for conv_rtol, and the FP32
// factor 1 / (1 + S_gal / S_instr) that the SNR screen multiplies rho_0^2 by.
// inv (may be null) receives that factor.
__device__ __forceinline__ double sg_store(const SgOut& o, long long j, double v,
                                           float* inv = nullptr) {
  double rel = 0.0;
  if (o.rtol_on) {
    double a = __dadd_rn(o.S[j], v), b = __dadd_rn(o.S[j], o.out[j]);
    rel = fabs(__dsub_rn(a, b)) / a;
  }
  o.out[j] = v;
  if (o.inv_f) {
    float ratio = __fmul_rn(dbl_to_f32_scaled(v, 150), o.invSf[j]);
    const float f = __frcp_rn(__fadd_rn(1.0f, ratio));
    o.inv_f[j] = f;
    if (inv) *inv = f;
  }
  return rel;
}

// ---------------------------------------------------------------- node sums of the SNR
// h of a node is the sum over its bins of Gf / (1 + S_gal / S_instr) in FP32, so that the
// screen of a long sweep reads nodes instead of bins.  The kernel that writes S_gal writes
// level 1 of the bins it wrote; its last CTA to finish (a ticket, no CTA waits) adds up the
// levels above.  Only in runs that keep a candidate with such a sweep (tree_live).
__device__ __forceinline__ float warp_sum_f32(float v) {
  for (int o = 16; o > 0; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}
// Level 1 nodes [a, b) from the bins' factors in memory (the whole CTA).
__device__ __forceinline__ void tree_h_nodes(const SgOut& o, int a, int b) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int i = a + warp; i < b; i += nwarp) {
    const long long j = (long long)i * 32 + lane;
    const float v = warp_sum_f32(__fmul_rn(o.Gf[j], o.inv_f[j]));
    if (lane == 0) o.tree.h[i] = v;
  }
}
// True in every thread of the last CTA of the grid to get here; what the others wrote before
// is then visible to it.
__device__ __forceinline__ bool last_cta(unsigned* ticket) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned t = atomicAdd(ticket, 1u);
    last = t == gridDim.x - 1;
    if (last) {
      *ticket = 0u;
      __threadfence();
    }
  }
  __syncthreads();
  return last != 0;
}
// Sum of 32 values pairwise, v holding them four at a time.
__device__ __forceinline__ float sum32(const float4 (&v)[8]) {
  float s[8];
#pragma unroll
  for (int k = 0; k < 8; ++k)
    s[k] = __fadd_rn(__fadd_rn(v[k].x, v[k].y), __fadd_rn(v[k].z, v[k].w));
#pragma unroll
  for (int w = 4; w > 0; w >>= 1)
#pragma unroll
    for (int k = 0; k < w; ++k) s[k] = __fadd_rn(s[k], s[k + w]);
  return s[0];
}
// Levels 2 and up from level 1 (the whole CTA): a thread per node adds its 32 values, all of
// them loaded at once.  (A warp per node left the one CTA waiting on a load per node: 20 us
// for a band of 1.25e6 bins, against 4.)
// Only the nodes above the changed bins: the outputs of the CTAs' items are the bins
// [item b0 + shift, + Kc), item from the work list (all of them when it is long).
__device__ __noinline__ void tree_h_levels(const Tree& tr, const Dirty& d, int list, int nitem,
                                           int Kc, int shift) {
  for (int l = 1; l < kTreeLevels; ++l) {
    const float4* in = reinterpret_cast<const float4*>(tr.h + tr.off[l - 1]);
    float* out = tr.h + tr.off[l];
    const int sh = 5 * (l + 1), per = (Kc >> sh) + 2;  // nodes that Kc bins can lie in
    const bool some = d.lists && (long long)nitem * per < tr.n[l];
    const int count = some ? nitem * per : tr.n[l];
    for (int x = threadIdx.x; x < count; x += blockDim.x) {
      int i = x;
      if (some) {
        const int a = max(d.item(list, x / per) * Kc + shift, 0);
        i = (a >> sh) + x % per;
      }
      if (i < 0 || i >= tr.n[l]) continue;
      float4 v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldcg(in + (size_t)i * 8 + k);
      out[i] = sum32(v);
    }
    __threadfence();
    __syncthreads();
  }
}
// The level 1 nodes that straddle two median tiles (the bins (u Kc + h) for u < nch), from the
// factors in memory, a thread per node.
__device__ __noinline__ void tree_h_straddle(const float* Gf, const float* inv_f, float* h1, int n1,
                                             int Kc, int h, int nch) {
  for (int u = threadIdx.x; u < nch; u += blockDim.x) {
    const long long i = ((long long)u * Kc + h) >> 5;
    if (i >= n1) continue;
    const float4* G = reinterpret_cast<const float4*>(Gf + i * 32);
    const float4* F = reinterpret_cast<const float4*>(inv_f + i * 32);
    float4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 a = G[k], f = __ldcg(F + k);
      v[k] = make_float4(__fmul_rn(a.x, f.x), __fmul_rn(a.y, f.y), __fmul_rn(a.z, f.z),
                         __fmul_rn(a.w, f.w));
    }
    h1[i] = sum32(v);
  }
  __threadfence();
  __syncthreads();
}

// Sum over the CTA of every thread's count c (0 <= c <= cmax, cmax the same in every thread),
// by barrier reductions of its bits: a barrier, and no shared memory.
__device__ __forceinline__ int cta_count(int c, int cmax) {
  int total = 0;
  for (int bit = 0; (1 << bit) <= cmax; ++bit) total += __syncthreads_count((c >> bit) & 1) << bit;
  return total;
}

// ============================================================================ chunk sort
// Chunks of Kc >= W consecutive bins: any window of at most W bins lies in at most two
// consecutive chunks.  Each chunk is sorted once (keys: the bits of the non-negative
// doubles, whose integer order is their value order; ties broken by position); srank
// maps a position to its sorted index.

// Sort key of a value x >= 0 (a negative value or -0.0 sorts as zero): the bits of the
// double (FP64 path), or of the float nearest to x * scale (mixed precision; scale is a
// power of two that brings the powers, ~1e-50 .. 1e-30, into the FP32 range).  For
// non-negative numbers the integer order of the bits is their value order.
template <typename K>
__device__ __forceinline__ K sort_key(double x, double scale);
template <>
__device__ __forceinline__ u64 sort_key<u64>(double x, double) {
  u64 k = (u64)__double_as_longlong(x);
  return (k >> 63) ? 0ull : k;
}
template <>
__device__ __forceinline__ uint32_t sort_key<uint32_t>(double x, double scale) {
  uint32_t k = __float_as_uint(__double2float_rn(__dmul_rn(x, scale)));
  return (k >> 31) ? 0u : k;
}
// The value a key stands for (inv_scale = 1 / scale, exact).
template <typename K>
__device__ __forceinline__ double key_value(K k, double inv_scale);
template <>
__device__ __forceinline__ double key_value<u64>(u64 k, double) {
  return __longlong_as_double((i64)k);
}
template <>
__device__ __forceinline__ double key_value<uint32_t>(uint32_t k, double inv_scale) {
  return __dmul_rn((double)__uint_as_float(k), inv_scale);
}

// Bitonic sort of 64-bit numbers, kpad of them, E consecutive ones per thread (element i in
// thread i / E).  Every merge begins with a stage of mirrored partners (i with i ^ (k - 1)), so
// that all comparisons run upwards: an element keeps the smaller or the larger of a pair by one
// bit of its index.  Partners less than E apart meet in registers, less than 32 E apart through
// warp shuffles, and the others through shared memory (two buffers in turn: a barrier per stage).
// buf: 2 kpad numbers.
// Bound: instruction issue, when every chunk is sorted.  As (key, position) pairs with a direction
// bit per stage a dense chunk of 1024 bins took 45 K warp instructions, 1.25e6 bins 71.6 us; as
// single numbers, all ascending, 32 K and 56 us.
__device__ __forceinline__ void keep_ordered(u64& c, u64 o, bool lower) {
  if ((o < c) == lower) c = o;
}
__device__ __forceinline__ void order_pair(u64& lo, u64& hi) {
  const u64 x = lo, y = hi;
  const bool swap = y < x;
  lo = swap ? y : x;
  hi = swap ? x : y;
}
template <int E>
__device__ __forceinline__ void bitonic_sort(u64 (&c)[E], int kpad, u64* buf) {
  const int T = blockDim.x, tid = threadIdx.x;
  u64* cur = buf;
  u64* nxt = buf + kpad;
  for (int kk = 2; kk <= kpad; kk <<= 1) {
    // the mirrored stage, then distances kk/4 .. 1
    bool mirror = true;
    for (int jj = kk >> 1; jj >= E; jj >>= 1) {
      const int m = (mirror ? kk - 1 : jj) / E;  // partner thread
      const bool lower = (tid & (jj / E)) == 0;
      u64 o[E];
      if (m < 32) {
#pragma unroll
        for (int a = 0; a < E; ++a) o[a] = __shfl_xor_sync(0xFFFFFFFFu, c[a], m);
      } else {
#pragma unroll
        for (int a = 0; a < E; ++a) cur[a * T + tid] = c[a];
        __syncthreads();
#pragma unroll
        for (int a = 0; a < E; ++a) o[a] = cur[a * T + (tid ^ m)];
        u64* t = cur;
        cur = nxt;
        nxt = t;
      }
#pragma unroll
      for (int a = 0; a < E; ++a) keep_ordered(c[a], mirror ? o[E - 1 - a] : o[a], lower);
      mirror = false;
    }
    // in registers: partners a and a ^ (2 jl - 1) in the mirrored stage of a merge that fits a
    // thread, a and a | jl otherwise
#pragma unroll
    for (int jl = E / 2; jl >= 1; jl >>= 1) {
      if (jl > (kk >> 1)) continue;
      if (jl == (kk >> 1)) {
#pragma unroll
        for (int a = 0; a < E; ++a)
          if ((a & jl) == 0) order_pair(c[a], c[a ^ (2 * jl - 1)]);
      } else {
#pragma unroll
        for (int a = 0; a < E; ++a)
          if ((a & jl) == 0) order_pair(c[a], c[a | jl]);
      }
    }
  }
}

// Re-sort of a chunk whose values changed at few positions since it was last sorted (the
// iterations after the first remove a few sources each).  The unchanged elements keep their
// relative order.  An unchanged element's new index is its old index, less the changed
// elements before it in the old order, plus the changed elements whose new (key, position)
// precede it; a changed element's new index is its rank among the changed elements plus the
// unchanged elements that precede it, found by a binary search of the old order.  This is
// the (key, position) order the full sort produces, so the two paths write the same arrays.
// Returns false, having written nothing, when more than kResortMax positions changed.
constexpr int kResortMax = 128;

template <typename K>
__device__ __forceinline__ bool key_pos_less(K ka, int pa, K kb, int pb) {
  return ka < kb || (ka == kb && pa < pb);
}

template <int E, typename K>
__device__ bool resort_few_changes(const K (&knew)[E], const K (&kold)[E], const int (&rold)[E],
                                   int len, int kpad, K* __restrict__ skey_c,
                                   uint16_t* __restrict__ srank_c, unsigned char* raw) {
  K* old_k = (K*)raw;                                // [kpad] old keys, in old sorted order
  K* ch_k = old_k + kpad;                            // [kResortMax] changed: new keys
  K* cs_k = ch_k + kResortMax;                       // [kResortMax] the same, sorted
  uint16_t* old_p = (uint16_t*)(cs_k + kResortMax);  // [kpad] position of each old index
  uint16_t* csum = old_p + kpad;                     // [kpad + 2] changed before an old index
  uint16_t* ch_p = csum + kpad + 2;                  // [kResortMax] changed: positions
  uint16_t* cs_p = ch_p + kResortMax;                // [kResortMax] the same, sorted
  unsigned char* chg = (unsigned char*)(cs_p + kResortMax);  // [kpad] changed, by position
  __shared__ int n_changed;
  __shared__ int bad_state;
  __shared__ int warp_sum[32];
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wid = tid >> 5;
  // 1. the old sorted state of the chunk (an index out of range, which a consistent state
  // never holds, sends the chunk to the full sort)
  if (tid == 0) {
    n_changed = 0;
    bad_state = 0;
  }
  // (the caller loaded this thread's old keys kold and sorted indices rold, of indices and
  // positions tid E + a, beside the new values)
  int r[E];
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const int p = tid * E + a;
    if (p < len) old_k[p] = kold[a];
    r[a] = p < len ? rold[a] : 0;
    if (r[a] >= len) {
      bad_state = 1;
      r[a] = 0;
    }
  }
  __syncthreads();
  if (bad_state) {
    __syncthreads();  // every thread has read the flag
    return false;
  }
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const int p = tid * E + a;
    if (p < len) old_p[r[a]] = (uint16_t)p;
  }
  __syncthreads();
  // 2. positions whose key changed, gathered in any order
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const int p = tid * E + a;
    const bool c = p < len && knew[a] != old_k[r[a]];
    chg[p] = c ? 1 : 0;
    if (c) {
      const int slot = atomicAdd(&n_changed, 1);
      if (slot < kResortMax) {
        ch_k[slot] = knew[a];
        ch_p[slot] = (uint16_t)p;
      }
    }
  }
  __syncthreads();
  const int C = n_changed;
  __syncthreads();  // every thread has read the count before the caller reuses shared memory
  if (C > kResortMax) return false;
  if (C == 0) return true;
  // 3. csum[i] = changed elements among old indices < i (exclusive scan in old order)
  int f[E], run = 0;
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const int i = tid * E + a;
    f[a] = i < len ? chg[old_p[i] & (kpad - 1)] : 0;
    run += f[a];
  }
  int incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_sum[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int nw = T >> 5;
    int v = lane < nw ? warp_sum[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xFFFFFFFFu, v, o);
      if (lane >= o) v += u;
    }
    if (lane < nw) warp_sum[lane] = v;  // inclusive over warps
  }
  __syncthreads();
  int ex = incl - run + (wid > 0 ? warp_sum[wid - 1] : 0);
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const int i = tid * E + a;
    if (i < len) csum[i] = (uint16_t)ex;
    ex += f[a];
  }
  if (tid == 0) csum[len] = (uint16_t)C;
  __syncthreads();
  // 4. changed elements: rank among themselves, plus the unchanged ones before them
  for (int t = tid; t < C; t += T) {
    const K ke = ch_k[t];
    const int pe = ch_p[t];
    int crank = 0;
    for (int u = 0; u < C; ++u) crank += key_pos_less<K>(ch_k[u], ch_p[u], ke, pe) ? 1 : 0;
    int lo = 0, hi = len;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (key_pos_less<K>(old_k[mid], old_p[mid], ke, pe))
        lo = mid + 1;
      else
        hi = mid;
    }
    const int ni = crank + lo - (int)csum[lo];
    cs_k[crank] = ke;
    cs_p[crank] = (uint16_t)pe;
    if (ni < len) {  // always, for a consistent old state
      skey_c[ni] = ke;
      srank_c[pe] = (uint16_t)ni;
    }
  }
  __syncthreads();
  // 5. unchanged elements: old index, less the changed before, plus the changed below them
#pragma unroll
  for (int a = 0; a < E; ++a) {
    const int i = tid * E + a;
    if (i < len && !f[a]) {
      const K ki = old_k[i];
      const int pi = old_p[i];
      int lo = 0, hi = C;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (key_pos_less<K>(cs_k[mid], cs_p[mid], ki, pi))
          lo = mid + 1;
        else
          hi = mid;
      }
      const int ni = i - (int)csum[i] + lo;
      if (ni < len && pi < len) {  // always, for a consistent old state
        skey_c[ni] = ki;
        srank_c[pi] = (uint16_t)ni;
      }
    }
  }
  return true;
}

// two elements per thread: 32 registers, so that a whole SM's threads stay resident
template <int E, typename K, bool kSpec>
__global__ void __launch_bounds__(1024, E == 2 ? 2 : 1) k_chunk_sort(SpecIn in, long long n, SmoothPlan pl,
                                                     K* __restrict__ skey,
                                                     uint16_t* __restrict__ srank, Dirty d) {
  extern __shared__ __align__(16) unsigned char sort_raw[];
  chain_wait();
  const int T = blockDim.x, tid = threadIdx.x;
  const int kpad = pl.kpad;  // = T * E
  const ListHead head = list_head(d, kListR0, pl.nch, in.flags);
  const int nitem = head.count;
  if (nitem <= (int)gridDim.x) chain_next();
  // after the first iteration of a tracked run every chunk holds the sorted state of its
  // previous values
  const bool resort = d.base != nullptr && head.iter > 0;
  int b_next = head.first;
  for (int item = blockIdx.x; item < nitem; item += gridDim.x) {
    const int b = b_next;  // a chunk whose input changed
    if (item + (int)gridDim.x < nitem) b_next = d.item(kListR0, item + gridDim.x);
    const long long base = (long long)b * pl.Kc;
    const int len = (int)((n - base) < pl.Kc ? (n - base) : pl.Kc);
    K k[E], kold[E];
    int rold[E];
    // the previous sorted state, loaded beside the new values
#pragma unroll
    for (int a = 0; a < E; ++a) {
      const int i = tid * E + a;
      kold[a] = (resort && i < len) ? skey[base + i] : (K)0;
      rold[a] = (resort && i < len) ? (int)srank[base + i] : 0;
    }
#pragma unroll
    for (int a = 0; a < E; ++a) {
      const int i = tid * E + a;
      K kv = (K)~(K)0;
      if (i < len) kv = sort_key<K>(spec_value<kSpec>(in, base + i, head.flags), pl.key_scale);
      k[a] = kv;
    }
    if (resort &&
        resort_few_changes<E, K>(k, kold, rold, len, kpad, skey + base, srank + base, sort_raw)) {
      __syncthreads();  // before the next chunk overwrites shared memory
      continue;
    }
    // a chunk of zeros (no power in it: much of the band's high-frequency end before any
    // removal) is sorted already: every key 0, ties in position order; a chunk with few
    // nonzero bins is that order with the few merged in (the re-sort from an all-zero state)
    {
      int nzc = 0;
#pragma unroll
      for (int a = 0; a < E; ++a) nzc += ((tid * E + a < len) && k[a] != (K)0) ? 1 : 0;
      const int nzt = cta_count(nzc, E);
      if (nzt == 0) {
#pragma unroll
        for (int a = 0; a < E; ++a) {
          const int i = tid * E + a;
          if (i < len) {
            skey[base + i] = (K)0;
            srank[base + i] = (uint16_t)i;
          }
        }
        continue;
      }
      if (nzt <= kResortMax) {
        K kz[E];
        int rid[E];
#pragma unroll
        for (int a = 0; a < E; ++a) {
          kz[a] = (K)0;
          rid[a] = tid * E + a < len ? tid * E + a : 0;
        }
        if (resort_few_changes<E, K>(k, kz, rid, len, kpad, skey + base, srank + base,
                                     sort_raw)) {
          __syncthreads();  // before the next chunk overwrites shared memory
          continue;
        }
      }
    }
    // the whole order: by the key's bits above the position's, with the position in their
    // place, as one 64-bit number (a 4-byte key leaves room for all of it)
    const u64 low = (u64)kpad - 1;
    u64* keys = (u64*)sort_raw;                    // [kpad] by position (8-byte keys)
    u64* buf = keys + (sizeof(K) == 8 ? kpad : 0);  // [2 kpad]
    u64 c[E];
#pragma unroll
    for (int a = 0; a < E; ++a) {
      const int i = tid * E + a;
      if (sizeof(K) == 8) {
        keys[i] = (u64)k[a];
        c[a] = ((u64)k[a] & ~low) | (u64)i;
      } else {
        c[a] = ((u64)k[a] << 32) | (u64)i;
      }
    }
    for (int pass = 0;; ++pass) {
      bitonic_sort<E>(c, kpad, buf);
      if (sizeof(K) == 4) break;
      // Keys that differ in the bits left out only may stand in the wrong order.  Such a
      // chunk is sorted by (those bits, position) and then by (the others, place in that
      // order), which is the order wanted.
      uint16_t* posof = (uint16_t*)(buf + 2 * (size_t)kpad);  // [kpad]
      if (pass == 0) {
        __shared__ u64 first[32];
        const int lane = tid & 31;
        __syncthreads();  // keys are in place (a chunk of one warp meets no other barrier)
#pragma unroll
        for (int a = 0; a < E; ++a) k[a] = (K)keys[c[a] & low];
        u64 after = __shfl_down_sync(0xFFFFFFFFu, (u64)k[0], 1);
        if (lane == 0) first[tid >> 5] = (u64)k[0];
        __syncthreads();
        if (lane == 31) after = tid + 1 < T ? first[(tid >> 5) + 1] : ~0ull;
        bool bad = (u64)k[E - 1] > after;
#pragma unroll
        for (int a = 0; a + 1 < E; ++a) bad = bad || k[a] > k[a + 1];
        if (!__syncthreads_or(bad)) break;
#pragma unroll
        for (int a = 0; a < E; ++a) c[a] = (((u64)k[a] & low) << 13) | (c[a] & low);
      } else if (pass == 1) {
#pragma unroll
        for (int a = 0; a < E; ++a) {
          const int i = tid * E + a;
          const int pos = (int)(c[a] & low);
          posof[i] = (uint16_t)pos;
          c[a] = (keys[pos] & ~low) | (u64)i;
        }
        // the next sort begins with the buffer that this one's last exchange read (an odd number
        // of exchanges: 64, 128 and 1024 threads)
        __syncthreads();
      } else {
        __syncthreads();
#pragma unroll
        for (int a = 0; a < E; ++a) {
          const int pos = posof[c[a] & low];
          k[a] = (K)keys[pos];
          c[a] = (u64)pos;
        }
        break;
      }
    }
#pragma unroll
    for (int a = 0; a < E; ++a) {
      const int sidx = tid * E + a;
      if (sidx < len) {
        skey[base + sidx] = sizeof(K) == 8 ? k[a] : (K)(c[a] >> 32);
        srank[base + (int)(c[a] & low)] = (uint16_t)sidx;
      }
    }
    __syncthreads();  // before the next chunk overwrites shared memory
  }
}

// Persistent grid: as many CTAs as fit on the GPU at once (items are dealt out statically,
// so a CTA that had to wait for a free slot would serialise its share), never more than
// the work items.
template <typename K>
static int resident_ctas(const SmoothPlan& pl, K kernel, int threads, size_t smem) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) !=
          cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  return pl.nsm * per_sm;
}
static int persistent_grid(const SmoothPlan& pl, int items, int resident) {
  if (pl.nsm <= 0 || resident <= 0) return items;
  return items < resident ? items : resident;
}

// Launch one k_chunk_sort instantiation with the key buffer cast to its key type.
template <typename K>
static void launch_sort_as(void (*kern)(SpecIn, long long, SmoothPlan, K*, uint16_t*, Dirty),
                           int bl, int th, size_t smem, cudaStream_t st, SpecIn in, long long n,
                           const SmoothPlan& pl, unsigned long long* skey, uint16_t* srank,
                           Dirty d) {
  kern<<<bl, th, smem, st>>>(in, n, pl, (K*)skey, srank, d);
}

static int sort_per_thread(const SmoothPlan& pl) {
  if (pl.sort_e) return pl.sort_e;
  return pl.kpad <= 2048 ? 2 : pl.kpad / 1024;
}
static int sort_threads(const SmoothPlan& pl) { return pl.kpad / sort_per_thread(pl); }
static size_t sort_smem(const SmoothPlan& pl) {
  const size_t kb = pl.fp32_keys ? 4 : 8;
  // the exchange buffers; 8-byte keys by position and an order beside them
  const size_t full = (size_t)pl.kpad * (16 + (kb == 8 ? 8 + sizeof(uint16_t) : 0));
  const size_t few = (size_t)pl.kpad * (kb + 2 + 1) + (size_t)(pl.kpad + 2) * 2 +
                     (size_t)kResortMax * 2 * (kb + 2);
  return full > few ? full : few;
}
template <typename K, bool kSpec, typename F>
static void with_sort_kernel_k(const SmoothPlan& pl, F fn) {
  switch (sort_per_thread(pl)) {
    case 2: fn(k_chunk_sort<2, K, kSpec>); break;
    case 4: fn(k_chunk_sort<4, K, kSpec>); break;
    default: fn(k_chunk_sort<8, K, kSpec>); break;
  }
}
template <bool kSpec, typename F>
static void with_sort_kernel(const SmoothPlan& pl, F fn) {
  if (pl.fp32_keys)
    with_sort_kernel_k<uint32_t, kSpec>(pl, fn);
  else
    with_sort_kernel_k<u64, kSpec>(pl, fn);
}

void launch_chunk_sort(SpecIn in, long long n, const SmoothPlan& pl, unsigned long long* skey,
                       uint16_t* srank, Dirty d, cudaStream_t st) {
  const size_t smem = sort_smem(pl);
  const int th = sort_threads(pl);
  const int bl = persistent_grid(pl, pl.nch, pl.res_sort);
  auto launch = [&](auto kern) {
    launch_sort_as(kern, bl, th, smem, st, in, n, pl, skey, srank, d);
  };
  if (in.acc)
    with_sort_kernel<true>(pl, launch);
  else
    with_sort_kernel<false>(pl, launch);
}

// ============================================================================ running median
// Tile u (u = 0 .. nch) produces the outputs j in [(u-1) Kc + h, u Kc + h), h = W/2.
// Their windows [s(j), e(j)] = [max(0, j - h), min(n-1, j - h + W - 1)] lie in the 2 Kc
// bins of chunks u-1 and u (W <= Kc): the tile's span.  One CTA per tile
//  1. merges the two sorted chunks, so that every position p of the span gets its rank
//     v(p) in the merged order (key, then position): a permutation of 0 .. 2Kc-1, bins
//     outside the band taking the top ranks (they are never inside a window);
//  2. builds a wavelet matrix of v over the positions: level l (l = 0 .. LV-1) stores bit
//     LV-1-l of the ranks in the order the stable partitions (zeros first) of the levels
//     above left them, as bitset words with exclusive prefix counts of their ones;
//  3. answers, one thread per output, "k-th smallest rank among positions [s, e]" by LV
//     descents of two rank lookups each, for k = c/2 (the upper median of c bins) and
//     k = c/2 - 1 (the lower one, used when c is even).
// Both results are elements of the window, so the median (App. D, Eq. running median)
// is a selection, exact whatever the order of the arithmetic; the ranks only say which
// element is selected.  Every output costs O(log Kc) independent of its neighbours, so
// a tile's latency is a few thousand cycles even when a single chunk has changed.

__device__ __forceinline__ int wm_levels(int M) { return 32 - __clz(M - 1); }
// Ones of the warps before this one (run) and of all of them (total), from the per-warp
// counts c (lane i holds warp i's, zero beyond the warps).
__device__ __forceinline__ void wm_warp_offsets(int c, int warp, int* run, int* total) {
  const int lane = threadIdx.x & 31;
  *total = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)c);
  *run = (int)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? (unsigned)c : 0u);
}

__device__ __forceinline__ unsigned lds_u16(uint32_t addr) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u16(uint32_t addr, unsigned v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"((unsigned short)v) : "memory");
}

// Wavelet matrix of the permutation seq0 (M elements, every warp owning exactly WPW words of a
// level; the caller fills the last words up with ranks beyond the span's): each level loads the
// warp's elements once, all of them before the first ballot, and the ballots serve both the count
// and the stable partition into the other buffer.  Level l stores its words in rk[l ws ..] (bits in the low half, ones of the earlier words
// in the high half) and its number of zeros in zeros[l].  seq0 and seq1 are both
// overwritten.
template <int WPW>
__device__ __forceinline__ void wm_build(uint16_t* seq0, uint16_t* seq1, u64* rk, int ws,
                                               int* zeros, int* warp_ones, int M, int LV,
                                               int nwm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const int w0 = warp * WPW;
  const unsigned below = (1u << lane) - 1u;
  uint32_t cur = (uint32_t)__cvta_generic_to_shared(seq0);
  uint32_t nxt = (uint32_t)__cvta_generic_to_shared(seq1);
  for (int l = 0; l < LV; ++l) {
    const int sh = LV - 1 - l;
    u64* rkl = rk + (size_t)l * ws;
    uint32_t xv[WPW];
    unsigned bal[WPW];
    int mine = 0;
#pragma unroll
    for (int q = 0; q < WPW; ++q) xv[q] = lds_u16(cur + 2u * (uint32_t)((w0 + q) * 32 + lane));
#pragma unroll
    for (int q = 0; q < WPW; ++q) {
      bal[q] = __ballot_sync(0xFFFFFFFFu, (xv[q] >> sh) & 1u);
      mine += __popc(bal[q]);
    }
    if (lane == 0) warp_ones[warp] = mine;
    __syncthreads();
    int run, total;
    wm_warp_offsets(lane < nwarp ? warp_ones[lane] : 0, warp, &run, &total);
    const int Z = M - total;
#pragma unroll
    for (int q = 0; q < WPW; ++q) {
      const int k = w0 + q;
      if (lane == 0) rkl[k] = ((u64)run << 32) | bal[q];
      if (l + 1 < LV) {
        const int ob = run + __popc(bal[q] & below);
        const int dst = ((xv[q] >> sh) & 1u) ? Z + ob : k * 32 + lane - ob;
        sts_u16(nxt + 2u * (uint32_t)dst, xv[q]);
      }
      run += __popc(bal[q]);
    }
    if (tid == 0) {
      rkl[nwm] = (u64)total << 32;
      zeros[l] = Z;
    }
    __syncthreads();
    const uint32_t t = cur;
    cur = nxt;
    nxt = t;
  }
}

// The same for any number of words per warp (the last warps may own fewer, or none).
__device__ __forceinline__ void wm_build_any(uint16_t* seq0, uint16_t* seq1, u64* rk, int ws,
                                             int* zeros, int* warp_ones, int M, int LV,
                                             int nwm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  const int wpw = (nwm + nwarp - 1) / nwarp;
  const int w0 = warp * wpw, w1 = min(w0 + wpw, nwm);
  uint16_t* cur = seq0;
  uint16_t* nxt = seq1;
  for (int l = 0; l < LV; ++l) {
    const int sh = LV - 1 - l;
    u64* rkl = rk + (size_t)l * ws;
    int mine = 0;
    for (int k = w0; k < w1; ++k)
      mine += __popc(__ballot_sync(0xFFFFFFFFu, (cur[k * 32 + lane] >> sh) & 1));
    if (lane == 0) warp_ones[warp] = mine;
    __syncthreads();
    int run, total;
    wm_warp_offsets(lane < nwarp ? warp_ones[lane] : 0, warp, &run, &total);
    const int Z = M - total;
    for (int k = w0; k < w1; ++k) {
      const int i = k * 32 + lane;
      const int x = cur[i];
      const int b = (x >> sh) & 1;
      const unsigned bits = __ballot_sync(0xFFFFFFFFu, b);
      if (lane == 0) rkl[k] = ((u64)run << 32) | bits;
      if (l + 1 < LV) {
        const int ob = run + __popc(bits & ((1u << lane) - 1u));
        nxt[b ? Z + ob : i - ob] = (uint16_t)x;
      }
      run += __popc(bits);
    }
    if (tid == 0) {
      rkl[nwm] = (u64)total << 32;
      zeros[l] = Z;
    }
    __syncthreads();
    uint16_t* t = cur;
    cur = nxt;
    nxt = t;
  }
}

// Positions of a tile of M filled up to whole words for every warp of T threads, so that the
// build's loads are unrolled: one, two, four or eight words per warp, as long as the ranks of
// the positions added keep LV bits.  Otherwise M (few threads for a long window, or more than a
// short one needs).  Before, only the windows whose words divide so had it; now W = 300 takes
// 189 us for every tile of 1.25e6 bins (195 with the loads in a loop), W = 2000 212 (219), a late
// tile there 30 us (33).
static int median_pad(int M, int T) {
  const int nwarp = T >> 5, w = ((M >> 5) + nwarp - 1) / nwarp;
  const int wpw = w <= 2 ? w : w <= 4 ? 4 : w <= 8 ? 8 : 0;
  const int Mp = 32 * wpw * nwarp;
  int top = 1;  // 2^LV
  while (top < M) top <<= 1;
  return wpw > 0 && Mp <= top ? Mp : M;
}
// Bytes of the keys' region, which later holds Mp positions' and M ranks' 16-bit numbers.
__host__ __device__ __forceinline__ size_t median_keys_bytes(int M, int Mp, size_t key_bytes) {
  const size_t k = key_bytes * M, later = 2 * ((size_t)M + Mp);
  return ((k > later ? k : later) + 15) & ~(size_t)15;
}

// Ones of a level's bitset before position i (the word holds its bits in the low half and
// the ones of all earlier words in the high half).
__device__ __forceinline__ int wm_rank1(const u64* rkl, int i) {
  const u64 e = rkl[i >> 5];
  return (int)(e >> 32) + __popc((uint32_t)e & ((1u << (i & 31)) - 1u));
}

// One tile; returns the largest relative change of S_n among its outputs (conv_rtol).
template <typename K>
__device__ __forceinline__ double median_tile(const K* __restrict__ skey,
                                              const uint16_t* __restrict__ srank, long long n,
                                              const SmoothPlan& pl, const SgOut& o, long long u,
                                              unsigned char* sm_raw, int* zeros) {
  const int T = blockDim.x, tid = threadIdx.x;
  // the span's positions, and the same filled up to whole words for every warp
  const int Kc = pl.Kc, M = 2 * Kc, LV = wm_levels(M);
  const int Mp = pl.median_mp;
  const int nwm = Mp >> 5, ws = nwm + 1;  // words per level (one zero word of padding)
  const int h = pl.W / 2;
  long long j_lo = (u - 1) * Kc + h, j_hi = u * Kc + h;
  if (j_lo < 0) j_lo = 0;
  if (j_hi > n) j_hi = n;
  if (j_lo >= j_hi) return 0.0;
  const double inv_scale = 1.0 / pl.key_scale;  // exact: a power of two
  const long long span = (u - 1) * (long long)Kc;
  int len0 = 0, len1 = 0;
  if (u >= 1) len0 = (n - span) < Kc ? (int)(n - span) : Kc;
  if (u < pl.nch) len1 = (n - span - Kc) < Kc ? (int)(n - span - Kc) : Kc;
  double relmax = 0.0;
  K* sk = (K*)sm_raw;                                        // [M] sorted keys (step 1)
  uint16_t* seq1 = (uint16_t*)sm_raw;                        // [Mp] (steps 2-3, over sk)
  uint16_t* src = seq1 + Mp;                                 // [M] rank -> element
  uint16_t* seq0 = (uint16_t*)(sm_raw + median_keys_bytes(M, Mp, sizeof(K)));  // [Mp]
  // [LV][ws]: per bitset word, its 32 bits (low half) and the ones before it (high half),
  // so that a rank is one 64-bit load
  u64* rk = (u64*)(seq0 + Mp);
  uint16_t* mr = (uint16_t*)rk;  // [M] merged index of (chunk, sorted index) (step 1, over rk)
  __shared__ int warp_ones[32];

  // 1. merged ranks.  Chunk u-1 precedes chunk u on equal keys (its positions are lower).
  int nzc = 0;  // this thread's nonzero keys of the span
  for (int i = tid; i < len0; i += T) {
    const K v = skey[span + i];
    sk[i] = v;
    nzc += v != (K)0 ? 1 : 0;
  }
  for (int i = tid; i < len1; i += T) {
    const K v = skey[span + Kc + i];
    sk[Kc + i] = v;
    nzc += v != (K)0 ? 1 : 0;
  }
  // Every window lies in the span; a window of c bins with fewer than ceil(c / 2) nonzero
  // values has a zero median (both middle elements are zeros).  The smallest window of
  // the tile is at one of its ends.
  auto win = [&](long long j) {
    const long long s0 = j - h > 0 ? j - h : 0;
    const long long e0 = j - h + pl.W - 1 < n - 1 ? j - h + pl.W - 1 : n - 1;
    return (int)(e0 - s0 + 1);
  };
  const int cmin = min(win(j_lo), win(j_hi - 1));
  const int nzt = cta_count(nzc, 2 * ((Kc + T - 1) / T));  // a thread loads at most that many
  if (nzt < (cmin + 1) / 2) {
    // every window's median is 0
    const int nz_out = (int)(j_hi - j_lo);
    for (int t = tid; t < nz_out; t += T) {
      const double rel = sg_store(o, j_lo + t, __dmul_rn(kMedianBias, 0.0));
      relmax = rel > relmax ? rel : relmax;
    }
    return relmax;
  }
  {
    // merge path: thread t emits the merged indices [d0, d1) of the two sorted chunks,
    // starting where a binary search on the diagonal d0 puts it
    const int L = len0 + len1, per = (L + T - 1) / T;
    const int d0 = min(tid * per, L), d1 = min(d0 + per, L);
    if (d0 < d1) {
      const K* A = sk;
      const K* B = sk + Kc;
      int lo = max(0, d0 - len1), hi = min(d0, len0);
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (A[mid] <= B[d0 - 1 - mid])
          lo = mid + 1;
        else
          hi = mid;
      }
      int i = lo, j = d0 - lo;
      for (int m = d0; m < d1; ++m) {
        if (i < len0 && (j >= len1 || A[i] <= B[j]))
          mr[i++] = (uint16_t)m;
        else
          mr[Kc + j++] = (uint16_t)m;
      }
    }
  }
  __syncthreads();
  for (int p = tid; p < M; p += T) {
    const int X = p >= Kc, q = p - X * Kc;
    int v;
    if (q < (X ? len1 : len0)) {
      const int si = srank[span + p];
      v = mr[X * Kc + si];
      src[v] = (uint16_t)((X << 15) | si);
    } else {
      v = len0 + len1 + (X ? (Kc - len0) + (q - len1) : (q - len0));
    }
    seq0[p] = (uint16_t)v;
  }
  for (int p = M + tid; p < Mp; p += T) seq0[p] = (uint16_t)p;
  __syncthreads();

  // 2. wavelet matrix.  Warp w owns the words [w wpw, (w + 1) wpw) of every level.  A level
  // takes two barriers: one after the warps have counted their ones, one after the stable
  // partition.
  const int nwarp = T >> 5, wpw = nwm % nwarp == 0 ? nwm / nwarp : 0;
  switch (wpw) {
    case 1: wm_build<1>(seq0, seq1, rk, ws, zeros, warp_ones, Mp, LV, nwm); break;
    case 2: wm_build<2>(seq0, seq1, rk, ws, zeros, warp_ones, Mp, LV, nwm); break;
    case 4: wm_build<4>(seq0, seq1, rk, ws, zeros, warp_ones, Mp, LV, nwm); break;
    case 8: wm_build<8>(seq0, seq1, rk, ws, zeros, warp_ones, Mp, LV, nwm); break;
    default: wm_build_any(seq0, seq1, rk, ws, zeros, warp_ones, Mp, LV, nwm); break;
  }

  // 3. selections
  const int nout = (int)(j_hi - j_lo);
  for (int t = tid; t < nout; t += T) {
    const long long j = j_lo + t;
    const long long s = j - h > 0 ? j - h : 0;
    const long long e = j - h + pl.W - 1 < n - 1 ? j - h + pl.W - 1 : n - 1;
    const int cnt = (int)(e - s + 1);
    // two descents side by side: a = upper median (k = c/2), b = lower (k = c/2 - 1)
    int la = (int)(s - span), ra = (int)(e + 1 - span), ka = cnt >> 1, va = 0;
    int lb = la, rb = ra, kb = ka > 0 ? ka - 1 : 0, vb = 0;
    for (int l = 0; l < LV; ++l) {
      const u64* rkl = rk + (size_t)l * ws;
      const int Z = zeros[l];
      const int oal = wm_rank1(rkl, la);
      const int oar = wm_rank1(rkl, ra);
      // the two order statistics are neighbours: their descents share a node at most
      // levels, and then share its ranks
      int obl = oal, obr = oar;
      if (__any_sync(__activemask(), la != lb || ra != rb)) {  // lanes still in the loop
        obl = wm_rank1(rkl, lb);
        obr = wm_rank1(rkl, rb);
      }
      const int za = (ra - oar) - (la - oal), zb = (rb - obr) - (lb - obl);
      const int bit = 1 << (LV - 1 - l);
      if (ka < za) {
        la -= oal;
        ra -= oar;
      } else {
        ka -= za;
        la = Z + oal;
        ra = Z + oar;
        va |= bit;
      }
      if (kb < zb) {
        lb -= obl;
        rb -= obr;
      } else {
        kb -= zb;
        lb = Z + obl;
        rb = Z + obr;
        vb |= bit;
      }
    }
    const int ea = src[va];
    const K khi = skey[span + (ea >> 15) * Kc + (ea & 0x7FFF)];
    double med;
    if (cnt & 1) {
      med = key_value<K>(khi, inv_scale);
    } else {
      const int eb = src[vb];
      const K klo = skey[span + (eb >> 15) * Kc + (eb & 0x7FFF)];
      med = __dmul_rn(__dadd_rn(key_value<K>(klo, inv_scale), key_value<K>(khi, inv_scale)),
                      0.5);
    }
    double v = __dmul_rn(kMedianBias, med);
    double rel = sg_store(o, j, v);
    relmax = rel > relmax ? rel : relmax;
  }
  return relmax;
}

template <typename K>
__global__ void __launch_bounds__(512, 2) k_median_wm(
    const K* skey, const uint16_t* srank, long long n, SmoothPlan pl,
    const __grid_constant__ SgOut o, const __grid_constant__ Dirty d) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ int zeros[16];
  double relmax = 0.0;
  const ListHead head =
      list_head(d, kListTile, pl.nch + 1, o.tree.h ? &o.rs->tree_live : nullptr);
  chain_wait();
  const int nitem = head.count;
  if (nitem <= (int)gridDim.x) chain_next();
  int u_next = head.first;
  for (int it = blockIdx.x; it < nitem; it += gridDim.x) {
    // a tile whose windows changed
    const int u = u_next;
    if (it + (int)gridDim.x < nitem) u_next = d.item(kListTile, it + gridDim.x);
    double r = median_tile<K>(skey, srank, n, pl, o, u, sm_raw, zeros);
    relmax = r > relmax ? r : relmax;
    __syncthreads();  // before the next tile overwrites shared memory
    if (head.flags) {
      // nodes whose bins all lie in this tile's outputs [(u-1) Kc + h, u Kc + h)
      const long long a = (long long)(u - 1) * pl.Kc + pl.W / 2, b = a + pl.Kc;
      const long long n1 = o.tree.n[0], na = a > 0 ? (a + 31) >> 5 : 0;
      tree_h_nodes(o, (int)na, (int)min(b >> 5, n1));
    }
  }
  if (head.flags && last_cta(&o.rs->ticket)) {
    // the nodes that straddle two tiles, then the levels above
    if ((pl.W / 2) & 31)
      tree_h_straddle(o.Gf, o.inv_f, o.tree.h, o.tree.n[0], pl.Kc, pl.W / 2, pl.nch);
    tree_h_levels(o.tree, d, kListTile, nitem, pl.Kc, pl.W / 2 - pl.Kc);
  }
  if (o.rtol_on) warp_max_atomic((u64)__double_as_longlong(relmax), &o.rs->relchg_bits);
}

// Two outputs per thread: a few tiles' latency is what a late iteration waits for.  At most 512
// threads, so that two CTAs share an SM (W = 2000, every tile: 212 us, 228 with 1024).
// Where tiles are many (all: every one of them; shared: a grid divisor above 1 says that other
// contexts run beside) their rate counts, and four CTAs of 256 threads cover each other's barriers better than two of 512, as long
// as the build stays unrolled (eight words per warp: chunks of up to 1024).  W = 1000, 1.25e6 bins:
// an estimate of every tile 213 us (220.5 with 512 threads), 64 runs at once 11.95 ms (12.2); a
// run by itself over 3e7 sources, with its late iterations, 1262 us (1209), so it keeps 512.
static int median_threads(const SmoothPlan& pl, bool all) {
  if (pl.median_th) return pl.median_th;
  int t = ((pl.Kc / 2 + 31) / 32) * 32;
  if (t < 32) t = 32;
  const int most = (all || pl.shared) && pl.Kc <= 1024 ? 256 : 512;
  return t < most ? t : most;
}

size_t median_smem_bytes(int Kc, int threads, int key_bytes) {
  const int M = 2 * Kc, Mp = median_pad(M, threads);
  int LV = 0;
  while ((1 << LV) < M) ++LV;
  size_t ws = (size_t)Mp / 32 + 1;
  size_t rk = (size_t)LV * ws * 8, mr = (size_t)2 * M;  // the merged indices sit over rk
  return median_keys_bytes(M, Mp, key_bytes) + (size_t)2 * Mp + (rk > mr ? rk : mr);
}

void launch_running_median(const unsigned long long* skey, const uint16_t* srank, long long n,
                           const SmoothPlan& pl, SgOut o, Dirty d, cudaStream_t st) {
  const bool all = d.lists == nullptr;
  const int th = median_threads(pl, all);
  size_t smem = median_smem_bytes(pl.Kc, th, pl.fp32_keys ? 4 : 8);
  int bl = persistent_grid(pl, pl.nch + 1, all ? pl.res_median_all : pl.res_median);
  SmoothPlan p = pl;
  p.median_mp = median_pad(2 * pl.Kc, th);
  if (pl.fp32_keys)
    launch_after(k_median_wm<uint32_t>, bl, th, smem, st, (const uint32_t*)skey, srank, n, p, o, d);
  else
    launch_after(k_median_wm<u64>, bl, th, smem, st, (const u64*)skey, srank, n, p, o, d);
}

// ============================================================================ window mean
// Exact window sums: inside chunk b every value becomes a 128-bit integer number of units
// 2^-sig[b], sig[b] chosen from the chunk's maximum so that a sum over the chunk fits;
// each chunk stores its inclusive prefix sums.  A window (at most two chunks) is one
// difference of prefixes per chunk, each converted to double once, so there is no
// cancellation however large the dynamic range of the spectrum.

__device__ __forceinline__ int sigma_from_max(u64 maxbits) {
  // max < 2^(e - 1022) with e the biased exponent; Kc <= 2^13 terms stay below 2^127.
  int e = (int)((maxbits >> 52) & 0x7FF);
  if (e == 0) e = 1;
  return 1136 - e;
}

// Prefix sums of chunk b: kPer consecutive values per thread, loaded and stored in pairs where
// the chunk is whole (pairs: a plain array starts on 16 bytes, as the library's own do).
//
// Bound: latency of one chunk (a maximum, a scan, two barriers each), so what counts is how
// many chunks an SM works on at once.  With one value per thread a chunk of 1024 bins took the
// SM alone (1024 threads of 56 registers).  1.25e6 bins, W = 1000: 31 -> 13 us from
// an array, 33 -> 28 us from the spectrum (W = 2000); running mean of 312 422 bins with its
// window means 29.7 -> 18.4 us.
template <bool kSpec, int kPer>
__device__ __forceinline__ void chunk_prefix(const SpecIn& in, long long n, const SmoothPlan& pl,
                                             unsigned long long* __restrict__ pre_lo,
                                             unsigned long long* __restrict__ pre_hi,
                                             int* __restrict__ sig, unsigned* __restrict__ uflow,
                                             double* __restrict__ x_out, int b, U128* warp_tot,
                                             u64* warp_max, int& any_uf, int flags, bool pairs) {
  const long long base = (long long)b * pl.Kc;
  const int len = (int)((n - base) < pl.Kc ? (n - base) : pl.Kc);
  const int p0 = threadIdx.x * kPer;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const bool whole = p0 + kPer <= len;
  // pass 1: values and the chunk maximum
  double v[kPer];
  u64 mb = 0;
  if (kSpec) {
    // a bin of the spectrum is 40 bytes in two arrays: neighbouring threads take neighbouring
    // bins, and hand them over through shared memory
    extern __shared__ double prefix_x[];  // [kPer blockDim.x]
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int p = threadIdx.x + i * blockDim.x;
      const double x = p < len ? spec_value<true>(in, base + p, flags) : 0.0;
      prefix_x[p] = x;
      if (x_out && p < len) x_out[base + p] = x;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i) v[i] = prefix_x[p0 + i];
  } else if (whole && pairs) {
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      const double2 w = *reinterpret_cast<const double2*>(in.x + base + p0 + i);
      v[i] = w.x;
      v[i + 1] = w.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      v[i] = p0 + i < len ? in.x[base + p0 + i] : 0.0;
  }
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const u64 bits = (u64)__double_as_longlong(v[i]);
    if (!(bits >> 63) && bits > mb) mb = bits;
  }
  for (int o = 16; o > 0; o >>= 1) {
    u64 t = __shfl_xor_sync(0xFFFFFFFFu, mb, o);
    mb = t > mb ? t : mb;
  }
  if (lane == 0) warp_max[warp] = mb;
  if (threadIdx.x == 0) any_uf = 0;
  __syncthreads();
  // every warp takes the maximum over the warps itself
  mb = lane < nwarp ? warp_max[lane] : 0ull;
  for (int o = 16; o > 0; o >>= 1) {
    u64 t = __shfl_xor_sync(0xFFFFFFFFu, mb, o);
    mb = t > mb ? t : mb;
  }
  const int sigma = sigma_from_max(mb);
  u64 lo[kPer], hi[kPer];
  if (mb == 0ull) {
    // a chunk of zeros: every prefix is 0 and nothing fell below one unit
#pragma unroll
    for (int i = 0; i < kPer; ++i) lo[i] = hi[i] = 0ull;
    if (threadIdx.x == 0) {
      uflow[b] = 0u;
      sig[b] = sigma;
    }
  } else {
    // pass 2: the thread's prefixes in fixed point; note inputs > 0 below one unit
    U128 run{0ull, 0ull};
    int uf = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const U128 q = dbl_to_u128_scaled(v[i], sigma);
      if (v[i] > 0.0 && u128_is_zero(q)) uf = 1;
      run = u128_add(run, q);
      lo[i] = run.lo;
      hi[i] = run.hi;
    }
    if (uf) any_uf = 1;
    // exclusive scan of thread totals
    U128 inc = run;
    for (int o = 1; o < 32; o <<= 1) {
      U128 t;
      t.lo = __shfl_up_sync(0xFFFFFFFFu, inc.lo, o);
      t.hi = __shfl_up_sync(0xFFFFFFFFu, inc.hi, o);
      if (lane >= o) inc = u128_add(inc, t);
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    // the warps before this one
    U128 offs = lane < warp ? warp_tot[lane] : U128{0ull, 0ull};
    for (int o = 16; o > 0; o >>= 1) {
      U128 t;
      t.lo = __shfl_xor_sync(0xFFFFFFFFu, offs.lo, o);
      t.hi = __shfl_xor_sync(0xFFFFFFFFu, offs.hi, o);
      offs = u128_add(offs, t);
    }
    offs = u128_add(offs, u128_sub(inc, run));  // exclusive within warp
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const U128 q = u128_add(offs, U128{lo[i], hi[i]});
      lo[i] = q.lo;
      hi[i] = q.hi;
    }
    if (threadIdx.x == 0) {
      uflow[b] = (unsigned)any_uf;
      sig[b] = sigma;
    }
  }
  // the inclusive prefixes
  if (whole) {
#pragma unroll
    for (int i = 0; i < kPer; i += 2) {
      *reinterpret_cast<ulonglong2*>(pre_lo + base + p0 + i) = make_ulonglong2(lo[i], lo[i + 1]);
      *reinterpret_cast<ulonglong2*>(pre_hi + base + p0 + i) = make_ulonglong2(hi[i], hi[i + 1]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if (p0 + i < len) {
        pre_lo[base + p0 + i] = lo[i];
        pre_hi[base + p0 + i] = hi[i];
      }
  }
}

// Values per thread: at most 1024 threads for chunks of up to 8192 bins, and few registers.
constexpr int kPrefixPer = 4, kPrefixPerLong = 8;
static int prefix_per(const SmoothPlan& pl) { return pl.Kc > 4096 ? kPrefixPerLong : kPrefixPer; }
static size_t prefix_smem(const SmoothPlan& pl, bool spec) {
  return spec ? (size_t)prefix_per(pl) * ((pl.Kc / prefix_per(pl) + 31) / 32 * 32) * sizeof(double)
              : 0;
}
static int prefix_threads(const SmoothPlan& pl) {
  return (pl.Kc / prefix_per(pl) + 31) / 32 * 32;
}

template <bool kSpec, int kPer>
__global__ void __launch_bounds__(1024)
    k_chunk_prefix(SpecIn in, long long n, SmoothPlan pl, unsigned long long* __restrict__ pre_lo,
                   unsigned long long* __restrict__ pre_hi, int* __restrict__ sig,
                   unsigned* __restrict__ uflow, double* __restrict__ x_out, Dirty d,
                   int in_radius) {
  __shared__ U128 warp_tot[32];
  __shared__ u64 warp_max[32];
  __shared__ int any_uf;
  // chunks whose input changed (a chunk within in_radius of them is dirty)
  const int list = kListR0 + in_radius;
  const ListHead head = list_head(d, list, pl.nch, in.flags);
  chain_wait();
  const int nitem = head.count;
  if (nitem <= (int)gridDim.x) chain_next();
  const bool pairs = (reinterpret_cast<uintptr_t>(in.x) & 15u) == 0;
  int b_next = head.first;
  for (int it = blockIdx.x; it < nitem; it += gridDim.x) {
    const int b = b_next;
    if (it + (int)gridDim.x < nitem) b_next = d.item(list, it + gridDim.x);
    chunk_prefix<kSpec, kPer>(in, n, pl, pre_lo, pre_hi, sig, uflow, x_out, b, warp_tot, warp_max,
                              any_uf, head.flags, pairs);
    __syncthreads();
  }
}

void launch_chunk_prefix(SpecIn in, long long n, const SmoothPlan& pl, unsigned long long* pre_lo,
                         unsigned long long* pre_hi, int* sig, unsigned* uflow, double* x_out,
                         Dirty d, int in_radius, cudaStream_t st) {
  const int th = prefix_threads(pl), bl = persistent_grid(pl, pl.nch, pl.res_prefix);
  auto launch = [&](auto kern) {
    const size_t smem = prefix_smem(pl, in.acc != nullptr);
    if (in_radius > 0)  // the medians' kernel comes before it
      launch_after(kern, bl, th, smem, st, in, n, pl, pre_lo, pre_hi, sig, uflow, x_out, d,
                   in_radius);
    else
      kern<<<bl, th, smem, st>>>(in, n, pl, pre_lo, pre_hi, sig, uflow, x_out, d, in_radius);
  };
  if (prefix_per(pl) == kPrefixPer) {
    if (in.acc) launch(k_chunk_prefix<true, kPrefixPer>);
    else launch(k_chunk_prefix<false, kPrefixPer>);
  } else {
    if (in.acc) launch(k_chunk_prefix<true, kPrefixPerLong>);
    else launch(k_chunk_prefix<false, kPrefixPerLong>);
  }
}

// A window's share of one chunk, units 2^-sigma of its bins [a, e]: the sum as a double.
__device__ __forceinline__ double part_sum(const double* __restrict__ x, int a, int e, U128 sum,
                                           int sigma, unsigned uf) {
  // Each input lost less than one unit; if the sum holds fewer than cnt * 2^40 units the
  // relative error could exceed 2^-40, so add the doubles directly instead.  A zero sum
  // is exact only if no input of the chunk fell below one unit.
  if (u128_is_zero(sum) && !uf) return 0.0;
  if (sum.hi == 0ull && sum.lo < ((unsigned long long)(e - a + 1) << 40)) {
    double acc = 0.0;
    for (int i = a; i <= e; ++i) acc = __dadd_rn(acc, x[i]);
    return acc;
  }
  return u128_to_dbl_scaled(sum, sigma);
}

// Window means, a CTA per kMeanThreads outputs of a chunk and an output per thread: an output is
// a dozen independent loads and a few dozen instructions, so small CTAs keep an SM's loads in
// flight (with a chunk's 1024 outputs per CTA of 40 registers an SM held one, and waited for
// each), and bins are 32-bit numbers.  1.25e6 bins: 26 -> 19 us; a late
// iteration's few chunks 8 -> 6 us.
// kTree: the run's S_gal, whose node sums h are kept up to date.
constexpr int kMeanThreads = 256;
template <bool kTree>
__global__ void __launch_bounds__(kMeanThreads, 6)
k_window_mean(const double* x, long long n, SmoothPlan pl, const unsigned long long* pre_lo,
                              const unsigned long long* pre_hi, const int* sig,
                              const unsigned* uflow, const __grid_constant__ SgOut o,
                              const __grid_constant__ Dirty d, int out_radius) {
  double relmax = 0.0;
  const int h = pl.W / 2;
  const double inv_w = 1.0 / (double)pl.W;
  // output chunks with a dirty chunk within out_radius, in parts of blockDim.x outputs
  const int list = kListR0 + out_radius;
  const int parts = (pl.Kc + blockDim.x - 1) / blockDim.x;
  const ListHead head =
      list_head(d, list, pl.nch, kTree ? &o.rs->tree_live : nullptr, parts);
  chain_wait();
  const int nitem = head.count * parts;
  if (nitem <= (int)gridDim.x) chain_next();
  long long b_next = head.first;
  for (int it = blockIdx.x; it < nitem; it += gridDim.x) {
    const long long b = b_next;
    if (it + (int)gridDim.x < nitem) b_next = d.item(list, (it + gridDim.x) / parts);
    // bins and outputs as 32-bit numbers (a band holds at most 16e6)
    const int b0 = (int)b * pl.Kc, nb = (int)n;
    const int jend = min(b0 + pl.Kc, nb);
    const int j = b0 + (it % parts) * (int)blockDim.x + threadIdx.x;
    if (j < jend) {
      const int s = max(j - h, 0), e = min(j - h + pl.W - 1, nb - 1), cnt = e - s + 1;
      // s and e lie within one chunk of chunk b (h < W <= Kc)
      const int cs = (int)b + (s < b0 ? -1 : (s >= b0 + pl.Kc ? 1 : 0));
      const int ce = (int)b + (e < b0 ? -1 : (e >= b0 + pl.Kc ? 1 : 0));
      const int s0 = cs * pl.Kc;  // first bin of the window's first chunk
      const U128 pe{pre_lo[e], pre_hi[e]};
      U128 ps{0ull, 0ull};
      if (s > s0) ps = U128{pre_lo[s - 1], pre_hi[s - 1]};
      double sum;
      if (cs == ce) {
        sum = part_sum(x, s, e, u128_sub(pe, ps), sig[cs], uflow[cs]);
      } else {
        const int last = s0 + pl.Kc - 1;
        const U128 pl1{pre_lo[last], pre_hi[last]};
        const double s1 = part_sum(x, s, last, u128_sub(pl1, ps), sig[cs], uflow[cs]);
        const double s2 = part_sum(x, last + 1, e, pe, sig[ce], uflow[ce]);
        sum = __dadd_rn(s1, s2);
      }
      double v = (cnt == pl.W) ? __dmul_rn(sum, inv_w) : __ddiv_rn(sum, (double)cnt);
      float inv = 0.0f;
      double rel = sg_store(o, j, v, &inv);
      relmax = rel > relmax ? rel : relmax;
      // chunks and warps start on multiples of 32 bins: a warp holds one node of level 1
      if (kTree && head.flags && (j | 31) < n) {
        const float hv = warp_sum_f32(__fmul_rn(o.Gf[j], inv));
        if ((threadIdx.x & 31) == 0) o.tree.h[j >> 5] = hv;
      }
    }
  }
  if (kTree && head.flags && last_cta(&o.rs->ticket))
    tree_h_levels(o.tree, d, list, head.count, pl.Kc, 0);
  if (o.rtol_on) warp_max_atomic((u64)__double_as_longlong(relmax), &o.rs->relchg_bits);
}

static int mean_threads(const SmoothPlan& pl) { return pl.Kc < kMeanThreads ? pl.Kc : kMeanThreads; }

void launch_window_mean(const double* x, long long n, const SmoothPlan& pl,
                        const unsigned long long* pre_lo, const unsigned long long* pre_hi,
                        const int* sig, const unsigned* uflow, SgOut o, Dirty d, int out_radius,
                        cudaStream_t st) {
  int th = mean_threads(pl);
  int bl = persistent_grid(pl, pl.nch * ((pl.Kc + th - 1) / th), pl.res_mean);
  if (o.tree.h)
    launch_after(k_window_mean<true>, bl, th, 0, st, x, n, pl, pre_lo, pre_hi, sig, uflow, o, d,
                 out_radius);
  else
    launch_after(k_window_mean<false>, bl, th, 0, st, x, n, pl, pre_lo, pre_hi, sig, uflow, o, d,
                 out_radius);
}

// ============================================================================ SNR + resolve
// rho^2 = 4 (T/5) A^2 sum_k w_k R_k / (S_k + S_gal,k) = sum_k rho0_k / (1 + S_gal,k / S_k).
// The screen evaluates it in FP32 as sum_k a2f w_k Gf_k inv_f_k; its relative error is
// below 2.2e-6 (FP32 roundings of the inputs, the ratio, the reciprocal and the products of
// each term) + 2e-7 per rounding of the sum that a term passes through: per bin for a sum
// on one lane, and for a sweep summed by a warp the longest lane's count plus the five
// levels of the butterfly (a sum of positive terms loses at most one rounding per step of
// its longest chain).  Outside twice that, 1e-5 + 4e-7 per step, around rho_th^2 the FP64
// decision is known.  Inside it, and always when the caller asks for the strict path,
// rho^2 is recomputed in FP64 with the oracle's terms: on one lane in the oracle's order
// for a sweep of a few bins, by the warp for a longer one.  In the mixed-precision mode the
// FP32 value decides alone.

__device__ __forceinline__ bool rtol_stop(const RunState* rs, double rtol) {
  if (!(rtol > 0.0) || rs->iter < 1) return false;
  double r = __longlong_as_double((i64)rs->relchg_bits);
  return r <= rtol;
}

// rho^2 of a sweep of many bins in FP64 by a whole warp: the same terms as rho2_exact, lane i
// summing the bins k0 + i, k0 + i + 32, ..., then a butterfly (a fixed order; every lane ends
// with the same value).  Its rounding differs from the sequential sum's by a few parts in
// 10^16; a decision that could differ lies within the near-threshold band.
__device__ double rho2_exact_warp(const Grid& g, const Tables& tb, const double* __restrict__ Sg,
                                  double a2, double lo, double hi) {
  const int lane = threadIdx.x & 31;
  Sweep sw;
  sw.lo = lo;
  sw.hi = hi;
  sw.ka = (i64)floor(__dadd_rn(lo, 0.5));
  sw.kb = (i64)floor(__dadd_rn(hi, 0.5));
  const bool single = (sw.ka == sw.kb);
  const long long k0 = sw.ka > g.k_lo ? sw.ka : g.k_lo;
  const long long k1 = sw.kb < g.k_lo + g.nb - 1 ? sw.kb : g.k_lo + g.nb - 1;
  double acc = 0.0;
  for (long long k = k0 + lane; k <= k1; k += 32) {
    const double w = single ? 1.0 : sweep_weight(sw, k);
    if (w > 0.0) {
      const long long j = k - g.k_lo;
      const double sn = __dadd_rn(tb.S[j], Sg[j]);
      const double psk = __dmul_rn(__dmul_rn(__dmul_rn(g.t5, tb.R[j]), a2), w);
      acc = __dadd_rn(acc, __ddiv_rn(psk, sn));
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, o));
  return __dmul_rn(4.0, acc);
}

// rho^2 of a sweep of very many bins by the whole CTA, for a decision that its screen left open:
// the terms of rho2_exact with the common factors outside the sum, which differs from it by the
// order of the roundings.  The value is in every thread.
// Bound by the FP64 pipe (a division per bin).  One warp took some 30 ms for a sweep of the whole
// 4-year band and held the launch; over twelve draws of 1e7 sources from the paper's priors, two
// of which meet such sweeps, a simulation now takes 2.95 ms on average.  (With reciprocals of
// 43 bits in place of the divisions it took 3.00, and rho^2 came out 3e-15 too small.)
__device__ double rho2_cta(const Grid& g, const Tables& tb, const double* __restrict__ Sg,
                           double a2, double lo, double hi) {
  __shared__ double part[32];
  Sweep sw;
  sw.lo = lo;
  sw.hi = hi;
  sw.ka = (i64)floor(__dadd_rn(lo, 0.5));
  sw.kb = (i64)floor(__dadd_rn(hi, 0.5));
  const long long k0 = sw.ka > g.k_lo ? sw.ka : g.k_lo;
  const long long k1 = sw.kb < g.k_lo + g.nb - 1 ? sw.kb : g.k_lo + g.nb - 1;
  double acc = 0.0;
#pragma unroll 4
  for (long long k = k0 + threadIdx.x; k <= k1; k += blockDim.x) {
    const long long j = k - g.k_lo;
    const bool inner = k > sw.ka && k < sw.kb;
    acc = __dadd_rn(acc, inner ? __ddiv_rn(tb.R[j], __dadd_rn(tb.S[j], Sg[j])) : 0.0);
  }
  acc = __dmul_rn(acc, sweep_inv_len(sw));
  if (threadIdx.x < 2) {  // the sweep's first and last cells, with their own weights
    const long long k = threadIdx.x ? sw.kb : sw.ka;
    if (k >= k0 && k <= k1) {
      const long long j = k - g.k_lo;
      const double sn = __dadd_rn(tb.S[j], Sg[j]);
      acc = __dadd_rn(acc, __ddiv_rn(__dmul_rn(tb.R[j], sweep_weight(sw, k)), sn));
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc = __dadd_rn(acc, __shfl_xor_sync(0xFFFFFFFFu, acc, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  double v = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = __dadd_rn(v, part[w]);
  return __dmul_rn(4.0, __dmul_rn(__dmul_rn(g.t5, a2), v));
}

__device__ double rho2_exact(const Grid& g, const Tables& tb, const double* __restrict__ Sg,
                             double a2, double lo, double hi) {
  Sweep sw;
  sw.lo = lo;
  sw.hi = hi;
  sw.ka = (i64)floor(__dadd_rn(lo, 0.5));
  sw.kb = (i64)floor(__dadd_rn(hi, 0.5));
  bool single = (sw.ka == sw.kb);
  long long k0 = sw.ka > g.k_lo ? sw.ka : g.k_lo;
  long long k1 = sw.kb < g.k_lo + g.nb - 1 ? sw.kb : g.k_lo + g.nb - 1;
  double acc = 0.0;
  for (long long k = k0; k <= k1; ++k) {
    double w = single ? 1.0 : sweep_weight(sw, k);
    if (w > 0.0) {
      long long j = k - g.k_lo;
      double sn = __dadd_rn(tb.S[j], Sg[j]);
      double psk = __dmul_rn(__dmul_rn(__dmul_rn(g.t5, tb.R[j]), a2), w);
      acc = __dadd_rn(acc, __ddiv_rn(psk, sn));
    }
  }
  return __dmul_rn(4.0, acc);
}

// FP32 screen sum of candidate c over the bins t0 + off, t0 + off + step, ... < t1 of its
// sweep (t relative to its first bin ka); kcount counts the terms.
__device__ __forceinline__ float screen_part(const Cands& cd, long long c, const int4 pk,
                                             const Grid& g, const Tables& tb,
                                             const float* __restrict__ inv_f, int off, int step,
                                             int& kcount) {
  const int ka = pk.x;
  const int nbin = pk.y;
  const float a2f = __int_as_float(pk.z);
  float r2 = 0.0f;
  kcount = 0;
  if (nbin == 1) {
    if (off == 0 && ka >= 0 && ka < g.nb) {
      r2 = __fmul_rn(__fmul_rn(a2f, tb.Gf[ka]), inv_f[ka]);
      kcount = 1;
    }
    return r2;
  }
  const float flo = __int_as_float(pk.w), len = cd.len[c];
  const float fhi = __fadd_rn(flo, len), invlen = 1.0f / len;
  const int t0 = ka < 0 ? -ka : 0;
  const int t1 = (long long)ka + nbin > g.nb ? (int)(g.nb - ka) : nbin;
  for (int t = t0 + off; t < t1; t += step) {
    float a = fmaxf(flo, (float)t - 0.5f);
    float b = fminf(fhi, (float)t + 0.5f);
    if (b > a) {
      float w = __fmul_rn(__fsub_rn(b, a), invlen);
      int k = ka + t;
      r2 = __fadd_rn(r2, __fmul_rn(__fmul_rn(__fmul_rn(a2f, w), tb.Gf[k]), inv_f[k]));
      ++kcount;
    }
  }
  return r2;
}

// Margin of the screen: the FP32 value is within this relative distance of the FP64 one
// (the bound above, doubled, for kcount bins).
__device__ __forceinline__ float screen_margin(int kcount) {
  return 1e-5f + 4e-7f * (float)kcount;
}

// The same by a whole warp for a sweep in the tree: the bins at its ends and the node sums h
// between them, the same value in every lane.  A term passes through at most 5 roundings in
// each level of h, the lane's chain (at most 3 bins, or 6 nodes in a band of 2^20 bins; nlev3
// / 32 more in a longer one) and the butterfly's 5.  False where the sum of h is outside the
// range in which FP32 keeps that accuracy (the caller then walks the bins).
__device__ __forceinline__ bool screen_tree(const Cands& cd, long long c, const int4 pk,
                                            const Grid& g, const Tables& tb,
                                            const float* __restrict__ inv_f, float* r2out,
                                            int* kcount) {
  const int lane = threadIdx.x & 31;
  const int ka = pk.x, kb = ka + pk.y - 1;
  const int k0 = ka < 0 ? 0 : ka, k1 = kb < g.nb ? kb : (int)g.nb - 1;
  if (k1 - k0 < kTreeBins) return false;
  const float a2f = __int_as_float(pk.z);
  const float flo = __int_as_float(pk.w), len = cd.len[c];
  const float fhi = __fadd_rn(flo, len), invlen = 1.0f / len;
  const TreeSpan t = tree_span(ka, kb, k0, k1);
  float r2 = 0.0f, hs = 0.0f;
  for (int x = lane; x < t.nbins; x += 32) {
    const int k = tree_bin(t, x);
    const float p = (float)(k - ka);
    const float a = fmaxf(flo, p - 0.5f);
    const float b = fminf(fhi, p + 0.5f);
    if (b > a) {
      const float w = __fmul_rn(__fsub_rn(b, a), invlen);
      r2 = __fadd_rn(r2, __fmul_rn(__fmul_rn(__fmul_rn(a2f, w), tb.Gf[k]), inv_f[k]));
    }
  }
  for (int x = lane; x < t.nnodes; x += 32) {
    int l, i;
    tree_node(t, x, &l, &i);
    hs = __fadd_rn(hs, tb.tree.h[tb.tree.off[l - 1] + i]);
  }
  hs = warp_sum_f32(hs);
  if (!(hs >= 1e-30f && hs <= 1e30f)) return false;
  *r2out = __fadd_rn(warp_sum_f32(r2), __fmul_rn(__fmul_rn(a2f, invlen), hs));
  *kcount = 5 * kTreeLevels + 6 + 5 + (tb.tree.n[kTreeLevels - 1] >> 5);
  return true;
}

// The FP32 value of a sweep of more than kSnrLaneBins bins by a whole warp, the same in every
// lane: true when it came from the tree.  kcount: the roundings that a term passes through.
__device__ __forceinline__ bool screen_wide(const Cands& cd, long long c, const int4 pk,
                                            const Grid& g, const Tables& tb,
                                            const float* __restrict__ inv_f, float* r2out,
                                            int* kcount) {
  if (screen_tree(cd, c, pk, g, tb, inv_f, r2out, kcount)) return true;
  // butterfly sums.  The sum's longest sequential chain is the largest lane count, and the
  // butterfly adds five roundings: the screen's bound takes that many terms, not every bin of
  // the sweep
  int kchain;
  float r2 = screen_part(cd, c, pk, g, tb, inv_f, threadIdx.x & 31, 32, kchain);
  for (int o = 16; o > 0; o >>= 1) {
    r2 = __fadd_rn(r2, __shfl_xor_sync(0xFFFFFFFFu, r2, o));
    kchain = max(kchain, __shfl_xor_sync(0xFFFFFFFFu, kchain, o));
  }
  *r2out = r2;
  *kcount = kchain + 5;
  return false;
}

// Decision from the FP32 value: 1 resolve, 0 keep, -1 too close to rho_th to tell (the
// caller then computes rho^2 exactly).
__device__ __forceinline__ int screen_decide(float r2, int kcount, float th2f, int mode) {
  if (mode == 1) return r2 > th2f ? 1 : 0;
  float m = screen_margin(kcount);
  if (mode == 0 && r2 > th2f * (1.0f + m)) return 1;
  if (mode == 0 && r2 < th2f * (1.0f - m)) return 0;
  return -1;
}

// An FP32 decision (mixed precision) that the FP64 value could take the other way.
__device__ __forceinline__ bool screen_uncertain(float r2, int kcount, float th2f) {
  const float m = screen_margin(kcount);
  return r2 <= th2f * (1.0f + m) && r2 >= th2f * (1.0f - m);
}

// An FP64 value of rho^2 with |rho - rho_th| / rho_th < 1e-9, i.e. |rho^2 / rho_th^2 - 1|
// below 2e-9 (to first order): a decision that the order of the FP64 roundings could flip.
__device__ __forceinline__ bool near_threshold(double r2, double th2) {
  return fabs(__dsub_rn(r2, th2)) < __dmul_rn(2e-9, th2);
}

// Take a cell's deposit from its bin (one beyond the range was never deposited).
__device__ __forceinline__ void remove_cell(unsigned long long* acc, long long j, double c,
                                            double gq) {
  u64 c0, c1, c2;
  if (q_cell(c, gq, &c0, &c1, &c2)) sub_parts(acc, j, c0, c1, c2);
}

// Remove the parts of candidate c that the catalog pass deposited: bins k0 + off,
// k0 + off + step, ... of its sweep.
__device__ __forceinline__ void remove_part(const Cands& cd, long long c, const Grid& g,
                                            const Tables& tb, unsigned long long* acc,
                                            const DirtyIter& d, int Kc, int off, int step) {
  Sweep sw;
  sw.lo = cd.lo[c];
  sw.hi = cd.hi[c];
  sw.ka = (i64)floor(__dadd_rn(sw.lo, 0.5));
  sw.kb = (i64)floor(__dadd_rn(sw.hi, 0.5));
  const double a2 = cd.a2[c];
  if (sw.ka == sw.kb) {
    long long j = sw.ka - g.k_lo;
    if (off == 0 && j >= 0 && j < g.nb) {
      u64 c0, c1, c2, qb;
      if (q_single(cd.amp[c], tb.gq[j], &c0, &c1, &c2, &qb)) sub_parts(acc, j, c0, c1, c2);
      d.mark_next(j / Kc);
    }
    return;
  }
  long long k0 = sw.ka > g.k_lo ? sw.ka : g.k_lo;
  long long k1 = sw.kb < g.k_lo + g.nb - 1 ? sw.kb : g.k_lo + g.nb - 1;
  const double inv = sweep_inv_len(sw);
  double q;
  if (step == 32 && tree_takes(tb.tree, a2, inv, k0, k1, &q)) {  // as tree_deposit
    if (!(q > 0.0)) return;
    const TreeSpan t = tree_span(sw.ka - g.k_lo, sw.kb - g.k_lo, k0 - g.k_lo, k1 - g.k_lo);
    for (int x = off; x < t.nbins; x += 32) {
      const int j = tree_bin(t, x);
      const double w = sweep_weight_inv(sw, g.k_lo + j, inv);
      if (w > 0.0) remove_cell(acc, j, __dmul_rn(a2, w), tb.gq[j]);
    }
    u64 c0, c1, c2;
    q_parts(q, &c0, &c1, &c2);
    for (int x = off; x < t.nnodes; x += 32) {
      int l, i;
      tree_node(t, x, &l, &i);
      if (c0) atomicAdd(acc + node_word(l, i, 0), (u64)(0ull - c0));
      if (c1) atomicAdd(acc + node_word(l, i, 1), (u64)(0ull - c1));
      if (c2) atomicAdd(acc + node_word(l, i, 2), (u64)(0ull - c2));
    }
    for (long long c = (k0 - g.k_lo) / Kc + off; c <= (k1 - g.k_lo) / Kc; c += 32) d.mark_next(c);
    return;
  }
  for (long long k = k0 + off; k <= k1; k += step) {
    double w = sweep_weight_inv(sw, k, inv);
    if (w > 0.0) {
      long long j = k - g.k_lo;
      remove_cell(acc, j, __dmul_rn(a2, w), tb.gq[j]);
      d.mark_next(j / Kc);
    }
  }
}

// The decision on a long sweep whose screen value is r2 (the same in every lane of the warp),
// and its removal.
__device__ __forceinline__ void snr_wide_decide(
    const Cands& cd, long long c, const Grid& g, const Tables& tb, const double* __restrict__ Sg,
    double th2, float th2f, int mode, float r2, int kcount, unsigned char* __restrict__ resolved,
    unsigned long long* __restrict__ acc, const DirtyIter& di, int Kc, unsigned& local_new,
    unsigned& local_exact, unsigned& local_near, unsigned& local_unc) {
  const int lane = threadIdx.x & 31;
  int dec = screen_decide(r2, kcount, th2f, mode);
  if (mode == 1 && lane == 0 && screen_uncertain(r2, kcount, th2f)) ++local_unc;
  if (dec < 0) {
    // FP64, the lanes sharing the bins
    if (lane == 0) ++local_exact;
    const double v = rho2_exact_warp(g, tb, Sg, cd.a2[c], cd.lo[c], cd.hi[c]);
    if (lane == 0 && near_threshold(v, th2)) ++local_near;
    dec = v > th2 ? 1 : 0;
  }
  if (dec) {
    if (lane == 0) {
      cd.res[c] = 1;
      resolved[cd.src[c]] = 1;
      ++local_new;
    }
    remove_part(cd, c, g, tb, acc, di, Kc, lane, 32);
  }
}

// Every lane screens one candidate of a group of 32: still unresolved, and S_n changed on
// a bin of its sweep (else rho is the value already found below rho_th).  Candidates of a
// few bins are done by their own lane.  Longer sweeps (loud high-frequency sources cover up
// to hundreds of bins, and more) come from their own list, one per warp in turn over the
// grid, the lanes sharing the bins: no launch waits on one thread walking a long sweep, nor
// on one warp walking many.

constexpr int kOpenMax = 16;     // sweeps a CTA sets aside
constexpr int kOpenBins = 4096;  // of more bins than this

__global__ void __launch_bounds__(256) k_snr_resolve(
    const __grid_constant__ Cands cd, const __grid_constant__ Grid g,
    const __grid_constant__ Tables tb, const double* Sg, const float* inv_f,
    double th2, double rtol, int mode, unsigned char* __restrict__ resolved,
    unsigned long long* __restrict__ acc, RunState* rs, Dirty d, int Kc, int sg_radius) {
  // the loop state, read by one thread per CTA (every thread of the grid loading the same
  // words would queue on one L2 line)
  __shared__ long long snr_head[4];  // stop, iteration, live candidates, long sweeps
  if (threadIdx.x == 0) {
    snr_head[0] = rs->final_pass ? 1 : 0;
    snr_head[1] = rs->iter;
    snr_head[2] = (long long)rs->nlive;
    snr_head[3] = (long long)rs->nwide;
  }
  __syncthreads();
  const long long nlive = snr_head[2];
  const DirtyIter di(d, (int)snr_head[1]);
  const int lane = threadIdx.x & 31;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const float th2f = (float)th2;
  unsigned local_new = 0, local_exact = 0, local_near = 0, local_unc = 0;
  // group grp holds candidates grp, grp + ngroups, grp + 2 ngroups, ...: candidates that
  // sit together in the list (the catalog pass emits the long sweeps of its FP64 path in
  // runs) are spread over many warps
  const long long ngroups = (nlive + 31) / 32;
  // the lane's candidate of a group is unresolved, a short sweep, and S_gal changed on it
  auto wanted = [&](long long c, int4* pk) {
    *pk = make_int4(0, 0, 0, 0);
    unsigned char done = 1;
    if (c < nlive) {  // both loads at once
      done = cd.res[c];
      *pk = cd.pk[c];
    }
    bool todo = false;
    if (!done && pk->y <= kSnrLaneBins) {  // the long sweeps are taken below
      const int ka = pk->x;
      const int nbin = pk->y;
      long long c0 = ka < 0 ? 0 : ka / Kc;
      long long kl = (long long)ka + nbin - 1;
      if (kl > g.nb - 1) kl = g.nb - 1;
      if (kl >= 0) {
        long long c1 = kl / Kc;
        for (long long cc = c0; cc <= c1 && !todo; ++cc) todo = di.any(cc, sg_radius);
      }
    }
    return todo;
  };
  // the warp's first group, while the estimate still runs
  long long grp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  int4 pk = make_int4(0, 0, 0, 0);
  bool todo = false;
  if (grp < ngroups) todo = wanted(grp + (long long)lane * ngroups, &pk);
  chain_wait();
  chain_next();
  if (rtol > 0.0) {
    if (threadIdx.x == 0 && rtol_stop(rs, rtol)) snr_head[0] = 1;
    __syncthreads();
  }
  if (snr_head[0]) return;
  for (; grp < ngroups;) {
    const long long c = grp + (long long)lane * ngroups;
    if (todo) {
      int kcount;
      const float r2 = screen_part(cd, c, pk, g, tb, inv_f, 0, 1, kcount);
      int dec = screen_decide(r2, kcount, th2f, mode);
      if (mode == 1 && screen_uncertain(r2, kcount, th2f)) ++local_unc;
      if (dec < 0) {
        ++local_exact;
        const double ex = rho2_exact(g, tb, Sg, cd.a2[c], cd.lo[c], cd.hi[c]);
        if (near_threshold(ex, th2)) ++local_near;
        dec = ex > th2;
      }
      if (dec) {
        cd.res[c] = 1;
        resolved[cd.src[c]] = 1;
        ++local_new;
        remove_part(cd, c, g, tb, acc, di, Kc, 0, 1);
      }
    }
    grp += nwarps;
    if (grp < ngroups) todo = wanted(grp + (long long)lane * ngroups, &pk);
  }
  // the long sweeps, one per warp at a time; the very long ones that the screen leaves open are
  // set aside for the whole CTA (the few that find no room are decided by their warp)
  __shared__ long long open_c[kOpenMax];
  __shared__ int open_n;
  if (threadIdx.x == 0) open_n = 0;
  __syncthreads();
  const long long nwide = snr_head[3];
  for (long long wi = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5; wi < nwide;
       wi += nwarps) {
    const long long cw = cd.wide[wi];
    if (cd.res[cw]) continue;  // the same in every lane
    const int4 pkw = cd.pk[cw];
    const long long c0 = pkw.x < 0 ? 0 : pkw.x / Kc;
    long long kl = (long long)pkw.x + pkw.y - 1;
    if (kl > g.nb - 1) kl = g.nb - 1;
    bool t = false;
    if (kl >= 0) {
      const long long c1 = kl / Kc;
      if (c1 - c0 >= 32 && d.lists) {
        // many chunks: the work list of the chunks whose S_gal changed is the shorter walk
        const int nlist = d.count(kListR0 + sg_radius, d.nch);
        if (nlist == d.nch) t = true;
        for (int i = lane; i < nlist && !t; i += 32) {
          const int cc = d.item(kListR0 + sg_radius, i);
          t = cc >= c0 && cc <= c1;
        }
      } else {
        for (long long cc = c0 + lane; cc <= c1; cc += 32) t = t || di.any(cc, sg_radius);
      }
    }
    if (!__any_sync(0xFFFFFFFFu, t)) continue;
    int kcount;
    float r2;
    if (screen_wide(cd, cw, pkw, g, tb, inv_f, &r2, &kcount) && mode == 0 && pkw.y > kOpenBins &&
        screen_decide(r2, kcount, th2f, mode) < 0) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&open_n, 1);
      at = __shfl_sync(0xFFFFFFFFu, at, 0);
      if (at < kOpenMax) {
        if (lane == 0) open_c[at] = cw;
        continue;
      }
    }
    snr_wide_decide(cd, cw, g, tb, Sg, th2, th2f, mode, r2, kcount, resolved, acc, di, Kc,
                    local_new, local_exact, local_near, local_unc);
  }
  __syncthreads();
  for (int i = 0; i < min(open_n, kOpenMax); ++i) {
    const long long co = open_c[i];
    const double v = rho2_cta(g, tb, Sg, cd.a2[co], cd.lo[co], cd.hi[co]);
    if (threadIdx.x == 0) {
      ++local_exact;
      if (near_threshold(v, th2)) ++local_near;
    }
    if (v > th2 && threadIdx.x < 32) {
      if (lane == 0) {
        cd.res[co] = 1;
        resolved[cd.src[co]] = 1;
        ++local_new;
      }
      remove_part(cd, co, g, tb, acc, di, Kc, lane, 32);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    local_new += __shfl_xor_sync(0xFFFFFFFFu, local_new, o);
    local_exact += __shfl_xor_sync(0xFFFFFFFFu, local_exact, o);
    local_near += __shfl_xor_sync(0xFFFFFFFFu, local_near, o);
    local_unc += __shfl_xor_sync(0xFFFFFFFFu, local_unc, o);
  }
  if (lane == 0) {
    if (local_new) atomicAdd(&rs->count_new, (unsigned long long)local_new);
    if (local_exact) atomicAdd(&rs->nexact, (unsigned long long)local_exact);
    if (local_near) atomicAdd(&rs->nnear, (unsigned long long)local_near);
    if (local_unc) atomicAdd(&rs->nuncertain, (unsigned long long)local_unc);
  }
}

// Both evaluations of rho^2 for every kept candidate against the current S_gal: the FP32
// screen as the loop evaluates it (a short sweep on one lane, a longer one by the warp) and the
// FP64 value in the oracle's order of summation, with the bins of the band in the sweep.  A
// measurement of the screen's error.
__global__ void __launch_bounds__(256) k_snr_check(Cands cd, Grid g, Tables tb,
                                                   const double* __restrict__ Sg,
                                                   const float* __restrict__ inv_f,
                                                   const RunState* rs,
                                                   long long* __restrict__ src,
                                                   float* __restrict__ screen,
                                                   double* __restrict__ exact,
                                                   int* __restrict__ nbins) {
  const long long nlive = (long long)rs->nlive;
  const int lane = threadIdx.x & 31;
  for (long long c0 = ((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5) << 5; c0 < nlive;
       c0 += (long long)gridDim.x * blockDim.x) {
    const long long c = c0 + lane;
    const bool valid = c < nlive;
    int4 pk = make_int4(0, 0, 0, 0);
    if (valid) pk = cd.pk[c];
    const bool wide = valid && pk.y > kSnrLaneBins;
    int count = 0, chain;
    float r2 = 0.0f;
    if (valid && !wide) r2 = screen_part(cd, c, pk, g, tb, inv_f, 0, 1, count);
    for (unsigned m = __ballot_sync(0xFFFFFFFFu, wide); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const int4 pl = make_int4(__shfl_sync(0xFFFFFFFFu, pk.x, l), __shfl_sync(0xFFFFFFFFu, pk.y, l),
                                __shfl_sync(0xFFFFFFFFu, pk.z, l), __shfl_sync(0xFFFFFFFFu, pk.w, l));
      float v;
      screen_wide(cd, c0 + l, pl, g, tb, inv_f, &v, &chain);
      if (lane == l) {
        const long long a = pl.x < 0 ? 0 : pl.x, b = min((long long)pl.x + pl.y, g.nb);
        r2 = v;
        count = b > a ? (int)(b - a) : 0;
      }
    }
    if (valid) {
      screen[c] = r2;
      exact[c] = rho2_exact(g, tb, Sg, cd.a2[c], cd.lo[c], cd.hi[c]);
      src[c] = cd.src[c];
      nbins[c] = count;
    }
  }
}

void launch_snr_check(Cands cd, long long ncap, const Grid& g, const Tables& tb, const double* Sg,
                      const float* inv_f, const RunState* rs, long long* src, float* screen,
                      double* exact, int* nbins, cudaStream_t st) {
  long long want = (ncap + 255) / 256;
  int bl = (int)(want < 4096 ? (want < 1 ? 1 : want) : 4096);
  k_snr_check<<<bl, 256, 0, st>>>(cd, g, tb, Sg, inv_f, rs, src, screen, exact, nbins);
}

void launch_snr_resolve(Cands cd, long long ncap, const Grid& g, const Tables& tb,
                        const double* Sg, const float* inv_f, double th2, double rtol, int mode,
                        unsigned char* resolved, unsigned long long* acc, RunState* rs,
                        Dirty d, int Kc, int sg_radius, int nsm, cudaStream_t st) {
  int th = 256;  // 8 warps, each screening 32 candidates at a time
  long long want = (ncap + th - 1) / th;
  long long cap = (long long)nsm * 8;
  int bl = (int)(want < cap ? (want < 1 ? 1 : want) : cap);
  launch_after(k_snr_resolve, bl, th, 0, st, cd, g, tb, Sg, inv_f, th2, rtol, mode, resolved, acc, rs,
               d, Kc, sg_radius);
}

// ============================================================================ coarse graining
// Bin averages of a per-bin series over log-spaced frequency bins (the coarse-grained
// spectrum and frequencies).  Bin k covers the grid indices [edge[k], edge[k+1]); a cluster of
// kParts CTAs per bin sums its values in a fixed order (no atomics), so the result is reproducible.
// The mean frequency of indices a .. b-1 is (2 k_lo + a + b - 1) / (2 T) exactly.
// Bound by the FP64 additions of the widest bin, which one SM makes at 2 per clock: of 100 bins
// over the 4-year band it holds 56 000 values (a call to the host 69 us with one CTA per bin, 56 with
// eight).
template <int kParts>
__global__ void __launch_bounds__(256) k_coarse_grain(const double* __restrict__ x,
                                                      const double* __restrict__ S,
                                                      const long long* __restrict__ edge,
                                                      long long k_lo, double T,
                                                      double* __restrict__ S_out,
                                                      double* __restrict__ f_out,
                                                      long long* __restrict__ cnt_out) {
  __shared__ double part[8];
  __shared__ double total;
  const int k = blockIdx.x / kParts, rank = blockIdx.x % kParts;
  const long long a = edge[k], b = edge[k + 1];
  const long long each = (b - a + kParts - 1) / kParts;
  const long long i1 = a + (rank + 1) * each < b ? a + (rank + 1) * each : b;
  double s = 0.0;
  for (long long i = a + rank * each + threadIdx.x; i < i1; i += blockDim.x)
    s = __dadd_rn(s, S ? __dadd_rn(S[i], x[i]) : x[i]);
  for (int o = 16; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xFFFFFFFFu, s, o));
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0) {
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = __dadd_rn(t, part[w]);
    total = t;
  }
  if (kParts > 1) {
    auto cluster = cooperative_groups::this_cluster();
    cluster.sync();
    if (threadIdx.x == 0 && rank == 0)
      for (int r = 1; r < kParts; ++r) t = __dadd_rn(t, *cluster.map_shared_rank(&total, r));
    cluster.sync();  // the others' shared memory stays until it is read
  }
  if (threadIdx.x == 0 && rank == 0) {
    const long long c = b - a;
    cnt_out[k] = c;
    S_out[k] = c > 0 ? __ddiv_rn(t, (double)c) : __longlong_as_double(0x7FF8000000000000ll);
    f_out[k] = c > 0 ? __ddiv_rn((double)(2 * k_lo + a + b - 1), __dmul_rn(2.0, T))
                     : __longlong_as_double(0x7FF8000000000000ll);
  }
}

void launch_coarse_grain(const double* x, const double* S, const long long* edge, int nbins,
                         long long n, long long k_lo, double T, double* S_out, double* f_out,
                         long long* cnt_out, cudaStream_t st) {
  // Clusters of eight where a bin has some thousands of values: at 3 124 on average 52.5 us a call
  // (56.1 with one CTA), at 2 048 56.6 us (54.2), over the 4-year band in one bin 96 us (429).
  constexpr int kParts = 8;
  if (n / nbins >= 3072) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kParts;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nbins * kParts);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_coarse_grain<kParts>, x, S, edge, k_lo, T, S_out, f_out, cnt_out);
  } else {
    k_coarse_grain<1><<<nbins, 256, 0, st>>>(x, S, edge, k_lo, T, S_out, f_out, cnt_out);
  }
}

// ============================================================================ loop control

// Work lists from the dirty set `cur` (one CTA).  Their order depends on the atomics,
// which is harmless: every item is computed on its own.
__device__ void build_lists_cta(const unsigned char* __restrict__ cur, int nch,
                                int* __restrict__ lists, int* __restrict__ counts) {
  __shared__ int cnt[kNumLists];
  if (threadIdx.x < kNumLists) cnt[threadIdx.x] = 0;
  __syncthreads();
  const size_t stride = (size_t)nch + 1;
  for (int b = threadIdx.x; b <= nch; b += blockDim.x) {
    auto at = [&](int i) { return i >= 0 && i < nch && cur[i] != 0; };
    const bool d0 = at(b), dm1 = at(b - 1);
    if (b < nch) {
      const bool r0 = d0, r1 = r0 || dm1 || at(b + 1), r2 = r1 || at(b - 2) || at(b + 2);
      if (r0) lists[kListR0 * stride + atomicAdd(&cnt[kListR0], 1)] = b;
      if (r1) lists[kListR1 * stride + atomicAdd(&cnt[kListR1], 1)] = b;
      if (r2) lists[kListR2 * stride + atomicAdd(&cnt[kListR2], 1)] = b;
    }
    if (d0 || dm1) lists[kListTile * stride + atomicAdd(&cnt[kListTile], 1)] = b;
  }
  __syncthreads();
  if (threadIdx.x < kNumLists) counts[threadIdx.x] = cnt[threadIdx.x];
}

// The state a run begins with: the spectrum's words, their replicas and the resolved mask zero,
// every chunk marked in the set the first iteration reads, none in the other one, and that
// iteration's work lists full.  Writes of (32 n + replicas + N) bytes, a few us at the most; as
// seven clears and a one-CTA list kernel the launches made it 12-18 us more of every run (1 yr, 1e4
// sources 187 -> 173 us; 24 served requests 4.03 -> 3.69 ms).
__global__ void __launch_bounds__(256) k_begin(ulonglong2* acc, long long n_acc, ulonglong2* rep,
                                               long long n_rep, unsigned char* resolved,
                                               long long n_resolved, unsigned char* dirty, int nch,
                                               int* lists, int* counts, int* new_hist,
                                               int max_iter, RunState* rs) {
  const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long step = (long long)gridDim.x * blockDim.x;
  chain_next();
  const ulonglong2 z = make_ulonglong2(0ull, 0ull);
  for (long long i = t0; i < n_acc; i += step) acc[i] = z;
  for (long long i = t0; i < n_rep; i += step) rep[i] = z;
  const long long whole = n_resolved / 16;
  for (long long i = t0; i < whole; i += step) reinterpret_cast<ulonglong2*>(resolved)[i] = z;
  for (long long i = 16 * whole + t0; i < n_resolved; i += step) resolved[i] = 0;
  for (long long i = t0; i < max_iter; i += step) new_hist[i] = 0;
  for (long long i = t0; i <= nch; i += step) {
    if (i < nch) {
      dirty[i] = 1;
      dirty[nch + i] = 0;
    }
#pragma unroll
    for (int l = 0; l < kNumLists; ++l)
      if (i < nch || l == kListTile) lists[(size_t)l * (nch + 1) + i] = (int)i;
  }
  if (t0 == 0) {
    RunState r{};
    for (int l = 0; l < kNumLists; ++l) {
      counts[l] = nch + (l == kListTile ? 1 : 0);
      r.work[l] = (unsigned long long)counts[l];
    }
    *rs = r;
  }
}

void launch_begin(unsigned long long* acc, long long nb, AccReplicas rep, unsigned char* resolved,
                  long long cap, unsigned char* dirty, int nch, int* lists, int* counts,
                  int* new_hist, int max_iter, RunState* rs, int nsm, cudaStream_t st) {
  const long long n_acc = nb * 2, n_rep = (long long)kAccReplicas * rep.nbins;
  const long long most = n_acc > cap / 16 ? n_acc : cap / 16;
  const long long want = (most + 255) / 256, lim = (long long)nsm * 8;
  k_begin<<<(unsigned)(want < lim ? want : lim), 256, 0, st>>>(
      (ulonglong2*)acc, n_acc, (ulonglong2*)rep.w, n_rep, resolved, cap, dirty, nch, lists, counts,
      new_hist, max_iter, rs);
}

__global__ void k_control(RunState* rs, int max_iter, double rtol, int* new_hist,
                          unsigned long long cond_handle, int use_cond, unsigned char* dirty,
                          int nch, int* lists, int* counts, RunState* host) {
  // every thread reads the count before thread 0 advances it (after the barriers below)
  const int it0 = rs->iter;
  chain_wait();
  // thread 0 loads the rest of the loop state now, so that its latency overlaps the lists
  int final_pass = 0;
  unsigned err = 0u;
  unsigned long long nn = 0ull, nres = 0ull;
  bool rstop = false;
  unsigned long long work[kNumLists] = {};
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < kNumLists; ++i) work[i] = rs->work[i];
    final_pass = rs->final_pass;
    err = rs->err;
    nn = rs->count_new;
    nres = rs->nres;
    rstop = rtol_stop(rs, rtol);
  }
  if (dirty) {
    // clear the set this iteration read; the removals of this iteration marked the other
    // one, which the next iteration reads through its work lists
    unsigned char* cur = dirty + (size_t)(it0 & 1) * nch;
    for (int i = threadIdx.x; i < nch; i += blockDim.x) cur[i] = 0;
    build_lists_cta(dirty + (size_t)((it0 + 1) & 1) * nch, nch, lists, counts);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned go = 1u;
  if (final_pass || (err & ERR_TIMEOUT)) {
    go = 0u;  // the last pass is done, or the catalog pass gave up
  } else {
    int it = it0 + 1;
    rs->iter = it;
    if (new_hist && it <= max_iter) new_hist[it - 1] = (int)nn;
    rs->nres = nres + nn;
    if (rstop || nn == 0ull) {
      rs->converged = 1;
      go = 0u;
    } else if (it >= max_iter) {
      rs->final_pass = 1;  // one more estimate of S_gal from the final resolved set
      go = 1u;
    }
  }
  rs->count_new = 0ull;
  rs->relchg_bits = 0ull;
  if (!go) {
    rs->stopped = 1;
    *host = *rs;
  }
  if (go && dirty)  // the lists just built go to the next iteration's kernels
    for (int i = 0; i < kNumLists; ++i) rs->work[i] = work[i] + (unsigned long long)counts[i];
  if (use_cond) cudaGraphSetConditional((cudaGraphConditionalHandle)cond_handle, go);
}

void launch_control(RunState* rs, int max_iter, double rtol, int* new_hist,
                    unsigned long long cond_handle, int use_cond, unsigned char* dirty, int nch,
                    int* lists, int* counts, RunState* host, cudaStream_t st) {
  launch_after(k_control, 1, 1024, 0, st, rs, max_iter, rtol, new_hist, cond_handle, use_cond, dirty,
               nch, lists, counts, host);
}

void plan_grids(SmoothPlan& pl) {
  pl.res_sort = pl.res_median = pl.res_median_all = pl.res_prefix = pl.res_mean = 0;
  if (pl.nsm <= 0) return;
  with_sort_kernel<true>(pl, [&](auto kern) {
    pl.res_sort = resident_ctas(pl, kern, sort_threads(pl), sort_smem(pl));
  });
  for (bool all : {false, true}) {
    const int th = median_threads(pl, all);
    const size_t smem = median_smem_bytes(pl.Kc, th, pl.fp32_keys ? 4 : 8);
    (all ? pl.res_median_all : pl.res_median) =
        pl.fp32_keys ? resident_ctas(pl, k_median_wm<uint32_t>, th, smem)
                     : resident_ctas(pl, k_median_wm<u64>, th, smem);
  }
  if (prefix_per(pl) == kPrefixPer)
    pl.res_prefix = resident_ctas(pl, k_chunk_prefix<true, kPrefixPer>, prefix_threads(pl),
                                  prefix_smem(pl, true));
  else
    pl.res_prefix = resident_ctas(pl, k_chunk_prefix<true, kPrefixPerLong>, prefix_threads(pl),
                                  prefix_smem(pl, true));
  pl.res_mean = resident_ctas(pl, k_window_mean<true>, mean_threads(pl), 0);
}

void configure_kernels() {
  cudaFuncSetAttribute(k_prepass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPrepassSmem);
  cudaFuncSetAttribute(k_chunk_prefix<true, kPrefixPerLong>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxWindow * 8);
  SmoothPlan p64 = {}, p32 = {};
  p32.fp32_keys = 1;
  for (int kp : {64, 4096, 8192}) {  // one of each instantiation; 8192: the widest sort
    p64.kpad = p32.kpad = kp;
    auto set = [](auto kern) {
      SmoothPlan widest = {};
      widest.kpad = 8192;
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sort_smem(widest));
    };
    with_sort_kernel<true>(p64, set);
    with_sort_kernel<true>(p32, set);
    with_sort_kernel<false>(p64, set);
    with_sort_kernel<false>(p32, set);
  }
  cudaFuncSetAttribute(k_median_wm<u64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       224 * 1024);
  cudaFuncSetAttribute(k_median_wm<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       224 * 1024);
}

}  // namespace gbsub
