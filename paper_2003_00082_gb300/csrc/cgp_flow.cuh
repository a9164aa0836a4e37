// The resident solvers' iterations in dataflow form: no grid barrier and no
// memory fence inside the loop.
//
// A block needs two things from the others every iteration: the totals of the
// three dot products, and w = K u of the rows its product reads (its halo).
// They travel in words that show by themselves whether they are the ones waited
// for, so a reader polls exactly the data it will use:
//   - partial sums in tagged 128-bit words (FP64: one per component, {sum,
//     exponent, tag}; FP32: one for all three) on lines that no other block
//     writes;
//   - w of a row that another block reads, with the reduction's number, in one
//     128-bit (FP64) or 64-bit (FP32) word.
// The halo rows' r and s are not published at all: a reader keeps copies of
// them (ghost rows) and applies the owner's own operations to them every
// iteration, so both hold the same bits.
//
// The FP64 sums travel in two parts.  (r,u) and (r,r) are known as soon as r is
// updated, before the product: they go out first (the early words), and their
// exchange, decoding, the stop test and beta cost nothing, because the product
// runs meanwhile on other warps.  Only (w,u) is left after the product (the late
// word): one component to sum, store, poll and convert, and one quotient.
// Meanwhile the warps with rows form p, x and s = w + beta s.
//
// Words of a kind live in two banks by the parity of the reduction.  A block
// stores its early words of k + 1 after it has read every late word of k, and
// its late word of k + 1 after it has read all early and late words of k (the
// stored sums depend on what it read); it overwrites a bank at k + 2 only after
// it has seen every block's words of k + 1, so no word is overwritten before its
// readers have it.
//
// What bounds it: 152 blocks that exchange one flag each way take 8.1k clocks
// an exchange through a release/acquire counter, 5.4k through slots 16 bytes
// apart (the pollers queue on the shared lines), 3.5k through slots on lines
// of their own stored with release, 2.6k stored relaxed; a line read on the
// other die just after it was written costs about 1.7k of that.  Polling loads
// the same network that the words travel on, so a round has one lane a block and
// one load a word.  The rest of an iteration is a chain of short steps (warp
// sums, block sums, totals, scalars), each written for latency here.
#pragma once

#include "cgp_solver.cuh"

namespace cgp {
namespace {

constexpr int kMaxShares = 8;   // groups of blocks whose words are folded by one warp each

// What only the dataflow iterations keep in shared memory beside Shared: it leads
// the dynamic part, so that the other forms' blocks stay as small as they are
// (whole 16-byte units; flow_smem_bytes counts them).
struct Flow64Shared {
  unsigned long long plo[3][kMaxShares];   // the polling warps' shares of the totals
  long long phi[3][kMaxShares];
  int pexp[3][kMaxShares];
  double ea[2], eb[2];            // alpha and beta by iteration parity
  double ev[2][MAX_BLOCK / 2];    // the rows' parts of (r,u) and (r,r)
  unsigned long long sig[2];      // signals: beta ready, (w,u) stored
};
struct Flow32Shared {
  float pf[3][kMaxShares];        // the polling warps' shares of the totals
  float abf[2][2];                // alpha and beta by iteration parity
};
static_assert(sizeof(Flow64Shared) % 16 == 0 && sizeof(Flow32Shared) % 16 == 0, "the vectors that follow are aligned");

// Dynamic shared memory of a dataflow block of `chunk` rows beyond the barrier
// form's: the state above and a byte per row (published or not).
inline size_t flow_smem_bytes(bool mixed, int chunk) {
  return (mixed ? sizeof(Flow32Shared) : sizeof(Flow64Shared)) + ((size_t)chunk + 15) / 16 * 16;
}

// A block's line of bank (red & 1): kind 0 early words, 1 the late word.
__device__ __forceinline__ unsigned char* flow_line(const Desc& d, int kind, int red, int blk) {
  return reinterpret_cast<unsigned char*>(d.tpart) + ((size_t)blk * 4 + 2 * kind + (red & 1)) * kLineBytes;
}

// Limit of a polling loop: d.spin_ns of wall-clock time, or as soon as another
// block has given up.
struct PollLimit {
  int* timeout;
  long long spin_ns;
  unsigned long long t0 = 0;
  unsigned spins = 0;
  __device__ PollLimit(const Desc& d) : timeout(&d.res->timeout), spin_ns(d.spin_ns) {}
  __device__ bool expired() {
    if ((++spins & 63u) != 0) return false;
    if (*(volatile int*)timeout) return true;
    const unsigned long long now = global_ns();
    if (t0 == 0) {
      t0 = now;
    } else if ((long long)(now - t0) > spin_ns) {
      atomicExch(timeout, 1);
      return true;
    }
    return false;
  }
};

// One-shot signals inside a block on shared-memory barriers of one arrival a
// phase: the waiting warps are suspended by the hardware, so they neither take
// issue slots from the warps at work (spinning on a shared word made small
// systems 10 % slower) nor poll the network before there can be anything to
// read.  `phase` is the parity of the signals given before.
__device__ __forceinline__ unsigned shared_address(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void signal_init(unsigned long long* mb) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(shared_address(mb)) : "memory");
}
__device__ __forceinline__ void signal_give(unsigned long long* mb) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(shared_address(mb)) : "memory");
}
__device__ __forceinline__ bool signal_wait(unsigned long long* mb, unsigned phase, const Desc& d) {
  PollLimit lim(d);
  while (true) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(shared_address(mb)), "r"(phase)
        : "memory");
    if (done) return true;
    if (lim.expired()) return false;
  }
}

// Groups the blocks of a solve are polled in (32 blocks a pass each) by at most
// `most` warps.
__device__ __forceinline__ int flow_groups(int nblk, int most) {
  const int g = (nblk + 31) / 32, m = most < kMaxShares ? most : kMaxShares;
  return g < m ? g : m;
}
// Row il's product with columns and values in shared memory (columns renumbered
// into ext), its entries taken eight at a time with their loads issued together
// (a row of a triangular mesh has about seven).
template <typename V>
__device__ __forceinline__ V row_product(const int* __restrict__ col, const V* __restrict__ val, const V* ext, int k0,
                                         int k1) {
  constexpr int B = 8;
  V s = V(0);
  for (int k = k0; k < k1; k += B) {
    int c[B];
    V a[B];
#pragma unroll
    for (int q = 0; q < B; ++q) c[q] = k + q < k1 ? col[k + q] : 0;
#pragma unroll
    for (int q = 0; q < B; ++q) a[q] = k + q < k1 ? val[k + q] : V(0);
#pragma unroll
    for (int q = 0; q < B; ++q) {
      const V u = ext[c[q]];
      if (k + q < k1) s = fma(a[q], u, s);
    }
  }
  return s;
}

// Rows below nloc of the calling thread among nt threads, T lanes per row.
template <int T, typename V, typename Op>
__device__ __forceinline__ void flow_rows(const int* __restrict__ row, const int* __restrict__ col,
                                          const V* __restrict__ val, const V* ext, int nloc, int t, int nt, Op op) {
  if constexpr (T == 1) {
    for (int il = t; il < nloc; il += nt) op(il, row_product(col, val, ext, row[il], row[il + 1]));
  } else {
    const int g = t / T, l = t % T, ng = nt / T;
    for (int base = 0; base < nloc; base += ng) {
      const int il = base + g;
      V s = V(0);
      if (il < nloc) {
        const int k1 = row[il + 1];
        for (int k = row[il] + l; k < k1; k += T) s = fma(val[k], ext[col[k]], s);
      }
#pragma unroll
      for (int o = T / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, T);
      if (il < nloc && l == 0) op(il, s);
    }
  }
}

// ---- FP64 -------------------------------------------------------------------

// The sums are those of put_partials (cgp_fixed.h): 128-bit integers aligned to
// the largest exponent, value X 2^(E - 1129).  A block's sum travels in one word
// (fx::pack_word: 94 bits below its largest term; two words with all of X took
// 3700 clocks more of an iteration on 152 blocks, since polling loads the network), and
// the fold over the blocks is 128 bits wide again.  A warp's sum is five
// redux.sync of 27-bit limbs.  Sums of 57-bit images, truncated 2^-54 below the
// largest term of a warp, block or group, took 7 % less of a solve at 512x256 and
// 321x163 and 12 % less at 64x32; the 128-bit steps written out on 32-bit words
// were no faster than the compiler's.
__device__ __forceinline__ fx::I128 warp_sum_wide(fx::I128 x) {
  unsigned s[fx::kLimbs];
#pragma unroll
  for (int i = 0; i < fx::kLimbs; ++i) s[i] = __reduce_add_sync(0xffffffffu, fx::limb(x, i));
  return fx::limbs_value(s);
}

// Exact warp sum of one value per lane into the block's table.
__device__ __forceinline__ void flow_warp_sum(double v, int c, int slot, Shared& sh) {
  const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)fx::exponent_of(v));
  const fx::I128 X = warp_sum_wide(E < fx::kBadExp ? fx::image(v, E) : (fx::I128)0);
  if ((threadIdx.x & 31) == 0) {
    sh.wlo[c][slot] = (unsigned long long)X;
    sh.whi[c][slot] = (long long)(X >> 64);
    sh.wexp[c][slot] = E;
  }
}
// One warp: the block's sum of component c over `act` warps, stored at p.
__device__ __forceinline__ void flow_block_sum(int c, int act, void* p, int red, Shared& sh) {
  const int lane = threadIdx.x & 31;
  const fx::I128 xw = lane < act ? ((fx::I128)sh.whi[c][lane] << 64) | (fx::I128)sh.wlo[c][lane] : (fx::I128)0;
  const int ew = lane < act ? sh.wexp[c][lane] : 1;
  const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)ew);
  const fx::I128 X = warp_sum_wide(E < fx::kBadExp ? fx::sar(xw, E - ew) : (fx::I128)0);
  uint64_t lo, hi;
  fx::pack_word(X, E, red, lo, hi);
  if (lane == 0) st_relaxed_b128(p, lo, hi);
}

// Polling warp q < G: wait for NC words of kind `kind` of the blocks 32 q + lane
// (+ 32 G ...); the warp's shares of the totals go to fs.plo/phi/pexp[c0 + c][q].
// The warp that has the early words (kind 0) loads its late word at once, into
// `late`, so that the load travels while the early words are decoded; the wait
// for the late words (kind 1) starts from `late`.  False (on every lane) when the
// wait gave up.
template <int NC>
__device__ __forceinline__ bool flow_poll(const Desc& d, int kind, int red, int q, int G, int c0, ulonglong2& late,
                                          Flow64Shared& fs) {
  const int lane = threadIdx.x & 31;
  PollLimit lim(d);
  fx::I128 acc[NC];
  int Ea[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    acc[c] = 0;
    Ea[c] = 1;
  }
  for (int base = 32 * q; base < d.nblk; base += 32 * G) {
    const int j = base + lane;
    const unsigned char* line = flow_line(d, kind, red, j < d.nblk ? j : base);
    ulonglong2 w[NC];
    bool loaded = kind == 1 && base == 32 * q;
    if (loaded) w[0] = late;
    while (true) {
      bool have = true;
      if (!loaded) {
#pragma unroll
        for (int c = 0; c < NC; ++c) w[c] = ld_relaxed_b128(line + 16 * c);
      }
      loaded = false;
#pragma unroll
      for (int c = 0; c < NC; ++c) have = have && fx::word_current(w[c].y, red);
      if (__all_sync(0xffffffffu, have)) break;
      if (__any_sync(0xffffffffu, lim.expired())) return false;
    }
    if (kind == 0 && base + 32 * G >= d.nblk) late = ld_relaxed_b128(flow_line(d, 1, red, min(32 * q + lane, d.nblk - 1)));
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int e = j < d.nblk ? fx::word_exponent(w[c].y) : 1;
      const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
      const fx::I128 S = fx::sar(fx::word_sum(w[c].x, w[c].y), E - e);
      const fx::I128 t = warp_sum_wide(j < d.nblk && E < fx::kBadExp ? S : (fx::I128)0);
      if (base == 32 * q) {
        acc[c] = t;
        Ea[c] = E;
      } else {
        const int F = max(Ea[c], E);
        acc[c] = fx::sar(acc[c], F - Ea[c]) + fx::sar(t, F - E);
        Ea[c] = F;
      }
    }
  }
  if (lane < NC) {
    const fx::I128 a = NC == 2 && lane == 1 ? acc[NC - 1] : acc[0];
    fs.plo[c0 + lane][q] = (unsigned long long)a;
    fs.phi[c0 + lane][q] = (long long)(a >> 64);
    fs.pexp[c0 + lane][q] = NC == 2 && lane == 1 ? Ea[NC - 1] : Ea[0];
  }
  return true;
}

// One warp: the total of component c from its G shares, on every lane.
__device__ __forceinline__ double flow_total(int c, int G, const Flow64Shared& fs) {
  const int lane = threadIdx.x & 31;
  const fx::I128 x = lane < G ? ((fx::I128)fs.phi[c][lane] << 64) | (fx::I128)fs.plo[c][lane] : (fx::I128)0;
  const int e = lane < G ? fs.pexp[c][lane] : 1;
  const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  return fx::to_double_normal(warp_sum_wide(E < fx::kBadExp ? fx::sar(x, E - e) : (fx::I128)0),
                              E < fx::kBadExp ? E + fx::kWordShift : E);
}

// A reciprocal of a normal a to about 22 bits, its exponent set by integer
// operations.
__device__ __forceinline__ double reciprocal_seed(double a) {
  const unsigned long long b = fx::dbits(a);
  const float m = __uint_as_float(0x3F800000u | (unsigned)((b >> 29) & 0x7FFFFFull));   // [1, 2)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));                                 // [0.5, 1]
  const unsigned f = __float_as_uint(r);
  const int e = (int)(f >> 23) - 127 + 2046 - (int)((b >> 52) & 0x7FF);
  return fx::from_bits(((unsigned long long)e << 52) | ((unsigned long long)(f & 0x7FFFFFu) << 29));
}
// Positive and within 2^-500 .. 2^500: the quotient of two such numbers and the
// remainders of flow_late are normal.
__device__ __forceinline__ bool moderate(double a) {
  const int e = __double2hiint(a) >> 20;
  return e > 523 && e < 1523;
}

// The scalars of an iteration, by one warp:
//   beta = gamma / gamma_old, alpha = gamma / (delta - beta gamma / alpha_old).
// An FP64 operation takes 64 clocks from issue to use whatever the number of
// active lanes, and the compiler's division about nine of them in a chain (564
// clocks).  What depends on gamma and (r,r) alone is done while the product runs
// (flow_early), 1 / (gamma alpha) of the iteration before while the early words
// travel; after delta one operation gives the denominator, and the quotient takes
// five more: lane 0 corrects it twice by its remainder (Markstein), first with the
// reciprocal that lane 1 has after one Newton step, then with the one it has after
// two.  After the first correction the quotient is one unit in the last place off
// in 1 of 100,000 cases; the second remainder is then exact and the result the
// correctly rounded quotient, as of a division.
struct EarlyScalars {
  double g, rr, m;         // gamma, (r,r), -gamma^2
  double inv_g, inv_ga;    // 1 / gamma and, of the iteration before, 1 / (gamma alpha)
  int st;                  // stop status so far (-1: go on)
};
// Leaves beta in fs.eb[k & 1] and gives sig[0] once it is there.
__device__ __forceinline__ void flow_early(EarlyScalars& q, int G, int k, bool last, Flow64Shared& fs, Shared& sh) {
  q.g = flow_total(0, G, fs);
  const double beta = k > 0 ? q.g * q.inv_g : 0.0;
  if ((threadIdx.x & 31) == 0) {
    fs.eb[k & 1] = beta;
    signal_give(&fs.sig[0]);
  }
  q.rr = flow_total(1, G, fs);
  q.st = -1;
  if (!finite_bits(q.g) || !finite_bits(q.rr)) q.st = CGP_ERR_NONFINITE;
  else if (nonneg_le(q.rr, sh.sc[4])) q.st = CGP_OK;   // (r,r) and (tol |b|)^2 are >= 0
  else if (last) q.st = CGP_ERR_NOT_CONVERGED;
  q.m = -q.g * q.g;
  q.inv_g = 1.0 / q.g;
  if ((threadIdx.x & 31) == 0) sh.sc[5] = q.rr;
}
// Leaves alpha in fs.ea[k & 1] and the stop status in sh.isc[0].
__device__ __forceinline__ void flow_late(EarlyScalars& q, int G, int k, Flow64Shared& fs, Shared& sh) {
  const int lane = threadIdx.x & 31;
  const double dl = flow_total(2, G, fs);
  const double den = k > 0 ? fma(q.m, q.inv_ga, dl) : dl;
  double alpha;
  int st = q.st;
  if (moderate(den) && moderate(q.g)) {
    const double y0 = reciprocal_seed(den);
    const bool quo = lane == 0;
    const double t1 = fma(quo ? q.g : -den, y0, quo ? 0.0 : 1.0);              // q0; 1 - den y0
    const double t2 = fma(quo ? -den : t1, quo ? t1 : y0, quo ? q.g : y0);     // g - den q0; y1
    const double y1 = __shfl_sync(0xffffffffu, t2, 1);
    const double t3 = fma(quo ? t2 : -den, y1, quo ? t1 : 1.0);                // q1; 1 - den y1
    const double t4 = fma(quo ? -den : t3, quo ? t3 : y1, quo ? q.g : y1);     // g - den q1; y2
    alpha = fma(t4, __shfl_sync(0xffffffffu, t4, 1), t3);                      // lane 0: q1 + rem y2
  } else {
    if (!finite_bits(dl)) st = CGP_ERR_NONFINITE;
    alpha = q.g / den;
  }
  if (lane == 0) {
    if (st < 0 && !(positive_bits(q.g) && positive_bits(alpha) && finite_bits(alpha))) st = CGP_ERR_BREAKDOWN;
    sh.isc[0] = st;
    fs.ea[k & 1] = alpha;
  }
}

// Word of row j's w in the publication of reduction `red`.
__device__ __forceinline__ ulonglong2* flow_w64(const Desc& d, int red, int j) {
  return reinterpret_cast<ulonglong2*>(d.pub64) + (size_t)(red & 1) * d.n + j;
}

// Thread t of nt: w of the rows hid[0 .. nh) in reduction `red`, as their owners
// store them.  False when the wait gave up.
__device__ __forceinline__ bool flow_fetch64(const Desc& d, int red, const int* hid, int nh, double* gw, int t, int nt) {
  const unsigned long long tag = (unsigned long long)red + 1;
  PollLimit lim(d);
  constexpr int B = 4;   // loads of a thread in flight
  bool ok = true;
  for (int h = t; h < nh; h += B * nt) {
    ulonglong2 a[B];
#pragma unroll
    for (int q = 0; q < B; ++q)
      a[q] = h + q * nt < nh ? ld_relaxed_b128(flow_w64(d, red, hid[h + q * nt])) : make_ulonglong2(0ull, tag);
#pragma unroll
    for (int q = 0; q < B; ++q) {
      while (a[q].y != tag && !lim.expired()) a[q] = ld_relaxed_b128(flow_w64(d, red, hid[h + q * nt]));
      ok = ok && a[q].y == tag;
      if (h + q * nt < nh) gw[h + q * nt] = fx::from_bits(a[q].x);
    }
  }
  return ok;
}

// FP64 Jacobi-PCG in the single-reduction form (solve_fp64_sr describes the
// recurrences) with rows resident in shared memory and dataflow iterations.
// The passes around the loop (projections, true residual) use the group
// barrier.
//
// Roles (a block has at least eight warps): the first half (ct threads) holds
// the rows; four warps with an operation always ready fill the FP64 pipe, so
// eight lose nothing in the product.  The other half sums and stores the early
// words, polls, fetches the halo's w, derives the scalars and updates the ghost
// rows, each on warps of its own.  Keeping the rows' r, s, w, u in registers (four rows a thread) was
// slower: 7.4 against 6.3 us an iteration.
//
// Measured at 512x256 on 152 blocks in O-grid tiles: 6.83 us an iteration with
// the counter barrier and slots 16 bytes apart, 6.34 us with all sums after the
// product, 5.59 us in this form with 57-bit images, 5.9 us with 128-bit ones.
constexpr int kFlowMinBlock = 256;
template <int T>
__device__ void solve_fp64_flow(const Desc& d, int lb, Shared& sh) {
  extern __shared__ __align__(16) unsigned char dsm[];
  const int tid = threadIdx.x, bd = blockDim.x, warp = tid >> 5, nw = bd >> 5;
  const int chunk = (d.n + d.nblk - 1) / d.nblk;
  const int r0 = min(d.n, lb * chunk), r1 = min(d.n, r0 + chunk), nloc = r1 - r0;
  const size_t n = d.n;
  Group grp{d.bar, &d.res->timeout, (unsigned)d.nblk, 0u, d.spin_ns};
  int red = 0;
  const int ow = nw / 2, ct = 32 * ow;                  // warps and threads with rows
  const int act = min(ow, (nloc * T + 31) / 32);        // of those, warps that have any
  const int G = flow_groups(d.nblk, nw - ow - 2);       // warps ow .. ow + G - 1 poll, warp ow + G derives the scalars
  // With many rows the product outlasts the early words: the warps that poll for
  // what it gives wait until this block's own part is done.  In the bisection
  // order this pays from about 500 rows a block (a solve with 429 rows: 5.06 ms
  // without, 5.11 with; 529 rows: 6.54 and 6.40; 866 rows: 9.86 and 9.75), on
  // O-grid tiles, whose product is shorter, from about 850 (583 rows: 6.37 and
  // 6.51; 866 rows: 8.85 and 8.75); with few rows the wait costs a round trip.
  const bool patient = chunk >= 512;
  double* const R0 = d.pub64 + 4 * n;                // r of a pass's start, for the ghost rows
  int* const mark = reinterpret_cast<int*>(d.z);     // rows that another block reads

  // shared memory: this form's state, own vectors, the product's input (CSR: own rows and halo;
  // stencil: the padded box), D^-1 and ghost r, s, w of the halo, the system,
  // its indices, and one byte per own row (published or not)
  const bool st = d.stencil;
  Flow64Shared& fs = *reinterpret_cast<Flow64Shared*>(dsm);
  double* base = reinterpret_cast<double*>(dsm + sizeof(Flow64Shared));
  double* x = base;
  double* r = base + chunk;
  double* ua = base + 2 * chunk;     // u_k and u_(k+1) alternate
  double* ub = base + 3 * chunk;
  double* w = base + 4 * chunk;
  double* p = base + 5 * chunk;
  double* s = base + 6 * chunk;
  double* di = base + 7 * chunk;
  double* bp = base + 8 * chunk;
  double* ext = base + 9 * chunk;
  double* dih = ext + (st ? d.box_cap : chunk + d.halo_cap);
  double* val = dih + d.halo_cap;                    // CSR: [nnz_cap]; stencil: [7][chunk] planes
  double* gr = val + (st ? 7 * chunk : d.res_nnz_cap);
  double* gs = gr + d.halo_cap;
  double* gw = gs + d.halo_cap;
  int* row = reinterpret_cast<int*>(gw + d.halo_cap);   // CSR: offsets [chunk + 1]; stencil: box positions [chunk]
  int* col = row + chunk + 1;
  int* hid = st ? row + chunk : col + d.res_nnz_cap;    // global row of each halo entry
  int* hpos = hid + d.halo_cap;                         // stencil: its box position
  unsigned char* pub = reinterpret_cast<unsigned char*>(st ? hpos + d.halo_cap : hid + d.halo_cap);
  const int h0 = d.hptr[lb], nh = d.hptr[lb + 1] - h0;
  int Ba = 0;
  if (st) {
    Ba = d.bdim[lb];
    for (int q = tid; q < d.box_cap; q += bd) ext[q] = 0.0;   // the ring outside the domain stays zero
    for (int k = 0; k < 7; ++k)
      for (int i = tid; i < nloc; i += bd) val[k * chunk + i] = d.planes[(size_t)k * n + r0 + i];
    for (int i = tid; i < nloc; i += bd) row[i] = d.bpos[r0 + i];
    for (int h = tid; h < nh; h += bd) hpos[h] = d.hpos[h0 + h];
  } else {
    const int k0 = nloc > 0 ? d.rowptr[r0] : 0;
    const int nnzl = nloc > 0 ? d.rowptr[r1] - k0 : 0;
    for (int i = tid; i <= nloc; i += bd) row[i] = d.rowptr[r0 + i] - k0;
    for (int k = tid; k < nnzl; k += bd) {
      col[k] = d.lcol[k0 + k];
      val[k] = d.val[k0 + k];
    }
  }
  for (int h = tid; h < nh; h += bd) {
    const int j = d.hidx[h0 + h];
    hid[h] = j;
    dih[h] = d.dinv[j];
  }
  for (int i = tid; i < nloc; i += bd) di[i] = d.dinv[r0 + i];

  auto own_at = [&](int i) { return st ? row[i] : i; };
  auto halo_at = [&](int h) { return st ? hpos[h] : nloc + h; };
  // the product's rows of thread t among nt
  auto rows = [&](int t, int nt, auto op) {
    if (st) spmv_box(row, val, chunk, ext, Ba, nloc, t, nt, op);
    else flow_rows<T>(row, col, val, ext, nloc, t, nt, op);
  };
  // this block's words start empty, its rows unmarked; the barrier of the first
  // reduction orders that before any block polls or marks
  if (tid < 8) st_relaxed_b128(flow_line(d, tid / 4, tid / 2, lb) + 16 * (tid % 2), 0ull, 0ull);   // both kinds and banks
  for (int i = tid; i < nloc; i += bd) {
    *flow_w64(d, 0, r0 + i) = make_ulonglong2(0ull, 0ull);
    *flow_w64(d, 1, r0 + i) = make_ulonglong2(0ull, 0ull);
    mark[r0 + i] = 0;
  }
  // ---- means of b and x0 ----
  {
    double v2[2] = {0.0, 0.0};
    for (int i = tid; i < nloc; i += bd) {
      v2[0] += d.b[r0 + i];
      if (d.use_x0) v2[1] += d.x[r0 + i];
    }
    put_partials<2>(d, lb, red, v2, sh);
    if (!grp.sync(sh)) return;
    get_totals<2>(d, red, sh);
    ++red;
  }
  for (int h = tid; h < nh; h += bd) mark[hid[h]] = 1;
  // ---- projected b and x0; x0 published for the first product ----
  {
    const double mb = d.fixed ? 0.0 : sh.tot[0] / d.n, mx = d.fixed ? 0.0 : sh.tot[1] / d.n;
    double v1[1] = {0.0};
    for (int i = tid; i < nloc; i += bd) {
      const double bi = is_fixed(d, r0 + i) ? 0.0 : d.b[r0 + i] - mb;
      bp[i] = bi;
      v1[0] += bi * bi;
      const double xi = (d.use_x0 && !is_fixed(d, r0 + i)) ? d.x[r0 + i] - mx : 0.0;
      x[i] = xi;
      d.x[r0 + i] = xi;
    }
    put_partials<1>(d, lb, red, v1, sh);
    if (!grp.sync(sh)) return;
    get_totals<1>(d, red, sh);
    ++red;
  }
  for (int i = tid; i < nloc; i += bd) pub[i] = (unsigned char)__ldcg(mark + r0 + i);
  const double bnorm = sqrt(sh.tot[0]);
  if (!isfinite(bnorm)) { finish(d, lb, CGP_ERR_NONFINITE, 0, 0, 0.0, 0.0, bnorm); return; }
  if (bnorm == 0.0) {
    for (int i = tid; i < nloc; i += bd) d.x[r0 + i] = 0.0;
    finish(d, lb, CGP_OK, 0, 0, 0.0, 0.0, 0.0);
    return;
  }
  const double stop = d.tol * bnorm, stop2 = stop * stop;
  if (tid < 2) signal_init(&fs.sig[tid]);   // the barriers of the next passes order that before any use
  if (tid == 0) sh.sc[4] = stop2;   // the test ||r||^2 <= (tol ||b||)^2 needs no square root

  int its = 0, restarts = 0, status = CGP_ERR_NOT_CONVERGED, pending = -1;
  unsigned phase = 0;   // of the block's signals, one of each an iteration
  double rr_rec = 0.0, rr_true = 0.0;
  bool first = true;
  while (true) {
    // ---- true residual of the projected, published x: r = bp - K x, u = D^-1 r; r published ----
    {
      double v1[1] = {0.0};
      for (int i = tid; i < nloc; i += bd) ext[own_at(i)] = x[i];
      for (int h = tid; h < nh; h += bd) ext[halo_at(h)] = __ldcg(d.x + hid[h]);
      __syncthreads();
      rows(tid, bd, [&](int il, double sum) {
        const double t = bp[il] - sum;
        r[il] = t;
        ua[il] = di[il] * t;
        R0[r0 + il] = t;
        v1[0] += t * t;
      });
      put_partials<1>(d, lb, red, v1, sh);
      if (!grp.sync(sh)) return;   // also publishes r for the ghost rows
      get_totals<1>(d, red, sh);
      ++red;
    }
    rr_true = sh.tot[0];
    if (first) rr_rec = rr_true;
    if (!isfinite(rr_true)) { status = CGP_ERR_NONFINITE; break; }
    if (rr_true <= stop2) { status = CGP_OK; break; }
    if (pending >= 0) { status = pending; break; }
    if (its >= d.max_it || restarts >= kMaxRestarts) { status = CGP_ERR_NOT_CONVERGED; break; }
    if (!first) ++restarts;
    first = false;

    // ---- u_0 and the ghost rows; then iterations from the product w_0 = K u_0 ----
    for (int h = tid; h < nh; h += bd) {
      const double rj = __ldcg(R0 + hid[h]);
      gr[h] = rj;
      ext[halo_at(h)] = dih[h] * rj;
    }
    if (tid < ct) {
      double g = 0.0, rr = 0.0;
      for (int i = tid; i < nloc; i += ct) {
        const double ri = r[i], ui = ua[i];
        ext[own_at(i)] = ui;
        g = fma(ri, ui, g);
        rr = fma(ri, ri, rr);
      }
      fs.ev[0][tid] = g;
      fs.ev[1][tid] = rr;
    }
    if (tid == 0) sh.tflag = 1;
    int k = 0;                           // products formed in this pass, less one
    EarlyScalars es;                     // warp ow + G
    es.inv_g = es.inv_ga = 0.0;
    while (true) {
      double* const uc = (k & 1) ? ub : ua;   // u_k
      double* const up = (k & 1) ? ua : ub;   // u_(k-1), then u_(k+1)
      const unsigned long long tag = (unsigned long long)red + 1;
      __syncthreads();
      if (tid < ct) {
        // ---- w_k = K u_k, published where another block reads it; (w,u) ----
        double v = 0.0;
        rows(tid, ct, [&](int il, double sum) {
          const double ui = uc[il];
          const bool out = pub[il];
          w[il] = sum;
          v = fma(sum, ui, v);
          if (out) st_relaxed_b128(flow_w64(d, red, r0 + il), fx::dbits(sum), tag);
        });
        if (warp < act) flow_warp_sum(v, 2, warp, sh);
        named_sync(2, ct);
        if (warp == 0) {
          flow_block_sum(2, act, flow_line(d, 1, red, lb), red, sh);
          if (tid == 0) signal_give(&fs.sig[1]);
        }
        // ---- p_(k-1) = u_(k-1) + beta p_(k-2), x += alpha p_(k-1) while the word travels ----
        if (k > 0) {
          const double alpha = fs.ea[(k - 1) & 1], beta = fs.eb[(k - 1) & 1];
          for (int i = tid; i < nloc; i += ct) {
            const double pi = k == 1 ? up[i] : fma(beta, p[i], up[i]);
            p[i] = pi;
            x[i] = fma(alpha, pi, x[i]);
          }
        }
        // ---- s_k = w_k + beta_k s_(k-1), once beta_k is known ----
        if (!signal_wait(&fs.sig[0], phase, d)) sh.tflag = 0;
        const double beta = fs.eb[k & 1];
        for (int i = tid; i < nloc; i += ct) s[i] = k == 0 ? w[i] : fma(beta, s[i], w[i]);
      } else {
        const int nt = bd - ct, cw = warp - ow;
        // ---- the early words: (r,u) and (r,r) ----
        if (cw < act) {
          flow_warp_sum(fs.ev[0][tid - ct], 0, cw, sh);
          flow_warp_sum(fs.ev[1][tid - ct], 1, cw, sh);
        }
        named_sync(3, nt);
        if (warp >= nw - 2) {   // two warps that do not poll
          const int c = warp - (nw - 2);
          flow_block_sum(c, act, flow_line(d, 0, red, lb) + 16 * c, red, sh);
        }
        if (cw < G) {
          ulonglong2 late = make_ulonglong2(0ull, 0ull);
          if (!flow_poll<2>(d, 0, red, cw, G, 0, late, fs)) sh.tflag = 0;
          named_sync(1, 32 * (G + 1));
          if (patient && !signal_wait(&fs.sig[1], phase, d)) sh.tflag = 0;
          if (!flow_poll<1>(d, 1, red, cw, G, 2, late, fs)) sh.tflag = 0;
          named_sync(1, 32 * (G + 1));
        } else if (cw == G) {
          if (k > 0) es.inv_ga = es.inv_g * (1.0 / fs.ea[(k - 1) & 1]);
          named_sync(1, 32 * (G + 1));
          flow_early(es, G, k, its + k >= d.max_it, fs, sh);
          named_sync(1, 32 * (G + 1));
          flow_late(es, G, k, fs, sh);
        } else {
          // ---- the halo's w: other blocks store theirs about when this one does ----
          if (patient && !signal_wait(&fs.sig[1], phase, d)) sh.tflag = 0;
          if (!flow_fetch64(d, red, hid, nh, gw, bd - 1 - tid, nt - 32 * (G + 1))) sh.tflag = 0;
        }
      }
      __syncthreads();
      if (!sh.tflag) return;
      ++red;
      phase ^= 1u;
      const int stop_st = sh.isc[0];
      if (stop_st >= 0) {
        if (stop_st != CGP_OK) pending = stop_st;
        break;
      }
      const double alpha = fs.ea[k & 1], beta = fs.eb[k & 1];
      if (tid < ct) {
        // ---- own rows: r, u_(k+1) and their dot products ----
        double g = 0.0, rr = 0.0;
        for (int i = tid; i < nloc; i += ct) {
          const double ri = fma(-alpha, s[i], r[i]);
          r[i] = ri;
          const double ui = di[i] * ri;
          up[i] = ui;
          ext[own_at(i)] = ui;
          g = fma(ri, ui, g);
          rr = fma(ri, ri, rr);
        }
        fs.ev[0][tid] = g;
        fs.ev[1][tid] = rr;
      } else {
        // ---- ghost rows: s, r, u_(k+1) ----
        for (int h = bd - 1 - tid; h < nh; h += bd - ct) {
          const double sj = k == 0 ? gw[h] : fma(beta, gs[h], gw[h]);
          gs[h] = sj;
          const double rj = fma(-alpha, sj, gr[h]);
          gr[h] = rj;
          ext[halo_at(h)] = dih[h] * rj;
        }
      }
      ++k;
    }
    its += k;
    rr_rec = sh.sc[5];
    // ---- x -= mean(x), published for the true residual ----
    {
      double v1[1] = {0.0};
      for (int i = tid; i < nloc; i += bd) v1[0] += x[i];
      put_partials<1>(d, lb, red, v1, sh);
      if (!grp.sync(sh)) return;
      get_totals<1>(d, red, sh);
      ++red;
    }
    const double mxf = d.fixed ? 0.0 : sh.tot[0] / d.n;
    for (int i = tid; i < nloc; i += bd) {
      const double xi = x[i] - mxf;
      x[i] = xi;
      d.x[r0 + i] = xi;
    }
    if (!grp.sync(sh)) return;
  }
  finish(d, lb, status, its, restarts, sqrt(rr_rec) / bnorm, sqrt(rr_true) / bnorm, bnorm);
}

// ---- FP32 (the inner iterations of MIXED) -----------------------------------

// The block's partial sums of three per-thread values as its word of reduction
// `red`: {v0, v1, v2, red + 1}.
__device__ __forceinline__ void flow_put_f(const Desc& d, int lb, int red, int act, const float (&v)[3], Shared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < act) {
    float t[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) t[c] = warp_sum(v[c]);
    if (lane < 3) sh.fred[lane][warp] = lane == 0 ? t[0] : (lane == 1 ? t[1] : t[2]);
  }
  if (threadIdx.x == 0) sh.tflag = 1;
  __syncthreads();
  if (warp == 0) {
    float t[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      t[c] = lane < act ? sh.fred[c][lane] : 0.0f;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) t[c] += __shfl_xor_sync(0xffffffffu, t[c], o);   // at most 16 warps
    }
    if (lane == 0)
      st_relaxed_b128(flow_line(d, 0, red, lb),
                      ((unsigned long long)__float_as_uint(t[1]) << 32) | __float_as_uint(t[0]),
                      ((unsigned long long)(unsigned)(red + 1) << 32) | __float_as_uint(t[2]));
  }
}

// Warp q < G: wait for the words of the blocks 32 q + lane (+ 32 G ...); the
// warp's share of the totals goes to fs.pf[c][q] (fixed order: the same bits
// in every block).
__device__ __forceinline__ bool flow_poll_f(const Desc& d, int red, int q, int G, Flow32Shared& fs) {
  const int lane = threadIdx.x & 31;
  PollLimit lim(d);
  const unsigned tag = (unsigned)(red + 1);
  float acc[3] = {0.0f, 0.0f, 0.0f};
  for (int base = 32 * q; base < d.nblk; base += 32 * G) {
    const int j = base + lane;
    const void* line = flow_line(d, 0, red, j < d.nblk ? j : base);
    ulonglong2 a;
    while (true) {
      a = ld_relaxed_b128(line);
      if (__all_sync(0xffffffffu, (unsigned)(a.y >> 32) == tag)) break;
      if (__any_sync(0xffffffffu, lim.expired())) return false;
    }
    if (j < d.nblk) {
      acc[0] += __uint_as_float((unsigned)a.x);
      acc[1] += __uint_as_float((unsigned)(a.x >> 32));
      acc[2] += __uint_as_float((unsigned)a.y);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) acc[c] = warp_sum(acc[c]);
  if (lane < 3) fs.pf[lane][q] = lane == 0 ? acc[0] : (lane == 1 ? acc[1] : acc[2]);
  return true;
}

__device__ __forceinline__ bool finite_bits(float x) { return ((__float_as_uint(x) >> 23) & 0xFFu) != 0xFFu; }

// One warp: the totals and the scalars of the next FP32 update: abf[k & 1]
// alpha and beta, fsc[3] ||r_0||^2 of the sweep, fsc[4] and fsc[5] the stop
// bounds, isc[0] the stop flag (0: stop, 1: non-finite, 2: breakdown); gamma
// and alpha of the last iteration stay with the warp in old[].
__device__ __forceinline__ void flow_scalars_f(int G, int k, bool last, float (&old)[2], Flow32Shared& fs,
                                                Shared& sh) {
  const int lane = threadIdx.x & 31, c = lane >> 3, q = lane & 7;
  float v = c < 3 && q < G ? fs.pf[c][q] : 0.0f;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const float g = __shfl_sync(0xffffffffu, v, 0), dl = __shfl_sync(0xffffffffu, v, 8);
  const float rr = __shfl_sync(0xffffffffu, v, 16);
  float beta = 0.0f, den = dl;
  if (k > 0) {   // two quotients of known terms side by side, then the one that needs the totals' difference
    beta = g / old[0];
    den = dl - beta * (g / old[1]);
  }
  const float alpha = g / den;
  const float rr0 = k == 0 ? rr : sh.fsc[3];
  int st = -1;
  if (!finite_bits(rr) || !finite_bits(g) || !finite_bits(dl)) st = 1;
  else if (rr <= fmaxf(sh.fsc[4] * rr0, sh.fsc[5])) st = 0;   // inner tolerance reached
  else if (last) st = 0;
  if (st < 0 && !(g > 0.0f && alpha > 0.0f && finite_bits(alpha))) st = 2;
  __syncwarp();
  if (lane == 0) {
    if (k == 0) sh.fsc[3] = rr;
    sh.isc[0] = st;
    fs.abf[k & 1][0] = alpha;
    fs.abf[k & 1][1] = beta;
  }
  old[0] = g;
  old[1] = alpha;
}

__device__ __forceinline__ unsigned long long* flow_w32(const Desc& d, int red, int j) {
  return reinterpret_cast<unsigned long long*>(d.f32pub) + (size_t)(red & 1) * d.n + j;
}

// As flow_fetch64.
__device__ __forceinline__ bool flow_fetch32(const Desc& d, int red, const int* hid, int nh, float* gw, int t, int nt) {
  const unsigned tag = (unsigned)(red + 1);
  PollLimit lim(d);
  constexpr int B = 4;   // loads of a thread in flight
  bool ok = true;
  for (int h = t; h < nh; h += B * nt) {
    unsigned long long a[B];
#pragma unroll
    for (int q = 0; q < B; ++q)
      a[q] = h + q * nt < nh ? ld_relaxed_u64(flow_w32(d, red, hid[h + q * nt])) : (unsigned long long)tag << 32;
#pragma unroll
    for (int q = 0; q < B; ++q) {
      while ((unsigned)(a[q] >> 32) != tag && !lim.expired()) a[q] = ld_relaxed_u64(flow_w32(d, red, hid[h + q * nt]));
      ok = ok && (unsigned)(a[q] >> 32) == tag;
      if (h + q * nt < nh) gw[h + q * nt] = __uint_as_float((unsigned)a[q]);
    }
  }
  return ok;
}

// Mixed precision with rows resident: the FP64 refinement and the FP32 inner
// recurrences of solve_mixed, the inner iterations in dataflow form.
//
// An inner iteration's arithmetic is small; what it costs besides the exchange
// is shared-memory instructions.  R > 0 (one lane per row, at most R rows a
// thread) therefore keeps r, s, w, u, D^-1 of a thread's rows and the first
// eight entries of each (values, 16-bit positions in the product's input) in
// registers: a row's product is eight independent gathers, and longer rows go
// on from the shared-memory slice.  R = 0 keeps everything in shared memory.
// At 512x256 on 152 blocks an inner iteration takes 2.55 us (3.69 us with the
// counter barrier), at 64x32 on 9 blocks 2.0 us (4.0 us).
//
// The sums go out together after the product: its 0.8k clocks are too few to
// hide a second exchange (early and late words as in solve_fp64_flow: 2.82 us).
template <int T, int R>
__device__ void solve_mixed_flow(const Desc& d, int lb, Shared& sh) {
  extern __shared__ __align__(16) unsigned char dsm[];
  static_assert(R == 0 || T == 1, "register rows take one lane each");
  constexpr int NR = R > 0 ? R : 1;
  constexpr int NE = 8;                              // entries of a row in registers
  const int tid = threadIdx.x, bd = blockDim.x, warp = tid >> 5, nw = bd >> 5;
  const int chunk = (d.n + d.nblk - 1) / d.nblk;
  const int r0 = min(d.n, lb * chunk), r1 = min(d.n, r0 + chunk), nloc = r1 - r0;
  const size_t n = d.n;
  Group grp{d.bar, &d.res->timeout, (unsigned)d.nblk, 0u, d.spin_ns};
  int red = 0;
  const int act = min(nw, (nloc * T + 31) / 32);     // warps with rows
  const int G = flow_groups(d.nblk, nw);
  const int f0 = G < nw ? 32 * G : 0;                // threads from here on fetch the halo's w
  float* const R0 = d.f32pub + 4 * n;                // r of a sweep's start, for the ghost rows
  int* const mark = reinterpret_cast<int*>(d.z);     // rows that another block reads

  Flow32Shared& fs = *reinterpret_cast<Flow32Shared*>(dsm);
  float* f = reinterpret_cast<float*>(dsm + sizeof(Flow32Shared));
  float* ir = f;
  float* iu = f + chunk;
  float* iw = f + 2 * chunk;
  float* ip = f + 3 * chunk;
  float* is = f + 4 * chunk;
  float* ie = f + 5 * chunk;
  float* di = f + 6 * chunk;
  float* ext = f + 7 * chunk;                   // [chunk + halo_cap]
  float* dih = ext + chunk + d.halo_cap;        // [halo_cap]
  float* val = dih + d.halo_cap;                // [nnz_cap]
  float* gr = val + d.res_nnz_cap;              // [halo_cap] each: ghost r, s and fetched w
  float* gs = gr + d.halo_cap;
  float* gw = gs + d.halo_cap;
  int* row = reinterpret_cast<int*>(gw + d.halo_cap);
  int* col = row + chunk + 1;
  int* hid = col + d.res_nnz_cap;
  unsigned char* pub = reinterpret_cast<unsigned char*>(hid + d.halo_cap);
  const int h0 = d.hptr[lb], nh = d.hptr[lb + 1] - h0;
  {
    const int k0 = nloc > 0 ? d.rowptr[r0] : 0;
    const int nnzl = nloc > 0 ? d.rowptr[r1] - k0 : 0;
    for (int i = tid; i <= nloc; i += bd) row[i] = d.rowptr[r0 + i] - k0;
    for (int k = tid; k < nnzl; k += bd) {
      col[k] = d.lcol[k0 + k];
      val[k] = d.val32[k0 + k];
    }
    for (int h = tid; h < nh; h += bd) {
      const int j = d.hidx[h0 + h];
      hid[h] = j;
      dih[h] = d.dinv32[j];
    }
    for (int i = tid; i < nloc; i += bd) di[i] = d.dinv32[r0 + i];
  }
  // outer FP64 storage (global)
  double* x = d.x + r0;
  double* bp = d.bp + r0;
  double* r64 = d.r + r0;

  // the calling thread's own rows: g(q, i), register slot q
  auto own_rows = [&](auto g) {
    if constexpr (R > 0) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int i = tid + q * bd;
        if (i < nloc) g(q, i);
      }
    } else {
      for (int i = tid; i < nloc; i += bd) g(0, i);
    }
  };

  // this block's words start empty, its rows unmarked; the barrier of the first
  // reduction orders that before any block polls or marks
  if (tid < 2) st_relaxed_b128(flow_line(d, 0, tid, lb), 0ull, 0ull);
  for (int i = tid; i < nloc; i += bd) {
    *flow_w32(d, 0, r0 + i) = 0ull;
    *flow_w32(d, 1, r0 + i) = 0ull;
    mark[r0 + i] = 0;
  }
  // ---- projected b and x0 ----
  {
    double v2[2] = {0.0, 0.0};
    for (int i = tid; i < nloc; i += bd) {
      v2[0] += d.b[r0 + i];
      if (d.use_x0) v2[1] += x[i];
    }
    put_partials<2>(d, lb, red, v2, sh);
    if (!grp.sync(sh)) return;
    get_totals<2>(d, red, sh);
    ++red;
  }
  for (int h = tid; h < nh; h += bd) mark[hid[h]] = 1;
  {
    const double mb = d.fixed ? 0.0 : sh.tot[0] / d.n, mx = d.fixed ? 0.0 : sh.tot[1] / d.n;
    double v1[1] = {0.0};
    for (int i = tid; i < nloc; i += bd) {
      const double bi = is_fixed(d, r0 + i) ? 0.0 : d.b[r0 + i] - mb;
      bp[i] = bi;
      v1[0] += bi * bi;
      x[i] = (d.use_x0 && !is_fixed(d, r0 + i)) ? x[i] - mx : 0.0;
    }
    put_partials<1>(d, lb, red, v1, sh);
    if (!grp.sync(sh)) return;
    get_totals<1>(d, red, sh);
    ++red;
  }
  for (int i = tid; i < nloc; i += bd) pub[i] = (unsigned char)__ldcg(mark + r0 + i);
  const double bnorm = sqrt(sh.tot[0]);
  if (!isfinite(bnorm)) { finish(d, lb, CGP_ERR_NONFINITE, 0, 0, 0.0, 0.0, bnorm); return; }
  if (bnorm == 0.0) {
    for (int i = tid; i < nloc; i += bd) x[i] = 0.0;
    finish(d, lb, CGP_OK, 0, 0, 0.0, 0.0, 0.0);
    return;
  }
  // FP64 view of the local rows for the outer residual (global arrays)
  Local L;
  L.row = d.rowptr + r0;
  L.col = d.col;
  L.val = d.val;

  // register rows: the first NE entries (absent ones: value 0 at the row's own
  // position) and whether a row goes on after them
  float rq[NR], sq[NR], wq[NR], uq[NR], vq[NR], dq[NR], aq[NR][NE];
  unsigned cq[NR][NE / 2];
  unsigned out = 0, more = 0;                        // rows to publish; rows longer than NE
  if constexpr (R > 0) {
    __syncthreads();
#pragma unroll
    for (int q = 0; q < R; ++q) {
      dq[q] = rq[q] = sq[q] = wq[q] = uq[q] = vq[q] = 0.0f;
#pragma unroll
      for (int e = 0; e < NE; ++e) aq[q][e] = 0.0f;
#pragma unroll
      for (int e = 0; e < NE / 2; ++e) cq[q][e] = 0u;
    }
    own_rows([&](int q, int i) {
      const int k0 = row[i], k1 = row[i + 1];
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const bool in = k0 + e < k1;
        aq[q][e] = in ? val[k0 + e] : 0.0f;
        cq[q][e / 2] |= (unsigned)(in ? col[k0 + e] : i) << (16 * (e & 1));
      }
      dq[q] = di[i];
      if (pub[i]) out |= 1u << q;
      if (k1 - k0 > NE) more |= 1u << q;
    });
  }

  int total = 0, sweeps = 0, status = CGP_ERR_NOT_CONVERGED;
  double rel = 0.0;
  while (true) {
    // ---- FP64 residual r = bp - K x, projected; x is complete (barrier above) ----
    {
      double v1[1] = {0.0};
      spmv_local<T, double>(
          L, r0, nloc, [&](int jl) { return x[jl]; }, [&](int j) { return __ldcg(d.x + j); },
          [&](int il, double s) {
            const double ri = bp[il] - s;
            r64[il] = ri;
            v1[0] += ri;
          });
      put_partials<1>(d, lb, red, v1, sh);
      if (!grp.sync(sh)) return;
      get_totals<1>(d, red, sh);
      ++red;
    }
    {
      const double mr = d.fixed ? 0.0 : sh.tot[0] / d.n;
      double v1[1] = {0.0};
      for (int i = tid; i < nloc; i += bd) {
        const double ri = r64[i] - mr;
        v1[0] += ri * ri;
        const float rf = (float)ri;
        ir[i] = rf;
        iu[i] = di[i] * rf;
        ie[i] = 0.0f;
        R0[r0 + i] = rf;
      }
      put_partials<1>(d, lb, red, v1, sh);
      if (!grp.sync(sh)) return;   // also publishes r_0 for the ghost rows
      get_totals<1>(d, red, sh);
      ++red;
    }
    rel = sqrt(sh.tot[0]) / bnorm;
    if (!isfinite(rel)) { status = CGP_ERR_NONFINITE; break; }
    if (rel <= d.tol) { status = CGP_OK; break; }
    if (sweeps >= d.max_sweeps || total >= d.max_it) { status = CGP_ERR_NOT_CONVERGED; break; }

    // ---- FP32 inner solve: u_0 and the ghost rows, then iterations from the product w_0 = A u_0 ----
    for (int i = tid; i < nloc; i += bd) ext[i] = iu[i];
    for (int h = tid; h < nh; h += bd) {
      const float rj = __ldcg(R0 + hid[h]);
      gr[h] = rj;
      ext[nloc + h] = dih[h] * rj;
    }
    if constexpr (R > 0) {
      own_rows([&](int q, int i) {
        rq[q] = ir[i];
        uq[q] = iu[i];
      });
    }
    if (tid == 0) {
      sh.fsc[4] = (float)(d.inner_tol * d.inner_tol);
      // below half the outer target the correction would already pass the outer test
      const double floor = 0.5 * d.tol * bnorm;
      sh.fsc[5] = (float)(floor * floor);
    }
    int k = 0;                           // products formed in this sweep, less one
    float old[2] = {0.0f, 0.0f};         // flow_scalars_f's last gamma and alpha (warp 0)
    bool bad = false;
    while (true) {
      __syncthreads();
      // ---- w_k = A u_k, published where another block reads it; the partial sums ----
      float v3[3] = {0.0f, 0.0f, 0.0f};
      const unsigned tag = (unsigned)(red + 1);
      if constexpr (R > 0) {
        own_rows([&](int q, int i) {
          float g[NE];
#pragma unroll
          for (int e = 0; e < NE; ++e) g[e] = ext[(cq[q][e / 2] >> (16 * (e & 1))) & 0xFFFFu];
          float s = 0.0f;
#pragma unroll
          for (int e = 0; e < NE; ++e) s = fmaf(aq[q][e], g[e], s);
          wq[q] = s;
        });
        if (more) {
          own_rows([&](int q, int i) {
            if (more & (1u << q))
              for (int e = row[i] + NE; e < row[i + 1]; ++e) wq[q] = fmaf(val[e], ext[col[e]], wq[q]);
          });
        }
        own_rows([&](int q, int i) {
          if (out & (1u << q))
            st_relaxed_u64(flow_w32(d, red, r0 + i), ((unsigned long long)tag << 32) | __float_as_uint(wq[q]));
          v3[0] = fmaf(rq[q], uq[q], v3[0]);
          v3[1] = fmaf(wq[q], uq[q], v3[1]);
          v3[2] = fmaf(rq[q], rq[q], v3[2]);
        });
      } else {
        flow_rows<T>(row, col, val, ext, nloc, tid, bd, [&](int il, float s) {
          const float u = ext[il], r = ir[il];
          iw[il] = s;
          if (pub[il]) st_relaxed_u64(flow_w32(d, red, r0 + il), ((unsigned long long)tag << 32) | __float_as_uint(s));
          v3[0] = fmaf(r, u, v3[0]);
          v3[1] = fmaf(s, u, v3[1]);
          v3[2] = fmaf(r, r, v3[2]);
        });
      }
      flow_put_f(d, lb, red, act, v3, sh);
      // ---- p_(k-1) = u_(k-1) + beta p_(k-2), e += alpha p_(k-1), while the words travel ----
      if (k > 0) {
        const float alpha = fs.abf[(k - 1) & 1][0], beta = fs.abf[(k - 1) & 1][1];
        own_rows([&](int q, int i) {
          const float uo = R > 0 ? vq[q] : iu[i];   // u_(k-1)
          const float pi = k == 1 ? uo : fmaf(beta, ip[i], uo);
          ip[i] = pi;
          ie[i] = fmaf(alpha, pi, ie[i]);
          if constexpr (R == 0) iu[i] = ext[i];
        });
      }
      // ---- the halo's w, then the sums ----
      if (tid >= f0) {
        if (!flow_fetch32(d, red, hid, nh, gw, tid - f0, bd - f0)) sh.tflag = 0;
      }
      if (warp < G && !flow_poll_f(d, red, warp, G, fs)) sh.tflag = 0;
      __syncthreads();
      if (warp == 0) flow_scalars_f(G, k, total + k >= d.max_it, old, fs, sh);
      __syncthreads();
      if (!sh.tflag) return;
      ++red;
      const int st = sh.isc[0];
      if (st >= 0) {
        bad = st == 1;
        break;
      }
      const float alpha = fs.abf[k & 1][0], beta = fs.abf[k & 1][1];
      // ---- own rows and ghost rows: s, r, u_(k+1) ----
      own_rows([&](int q, int i) {
        const float wi = R > 0 ? wq[q] : iw[i];
        const float si = k == 0 ? wi : fmaf(beta, R > 0 ? sq[q] : is[i], wi);
        const float ri = fmaf(-alpha, si, R > 0 ? rq[q] : ir[i]);
        const float ui = (R > 0 ? dq[q] : di[i]) * ri;
        if constexpr (R > 0) {
          sq[q] = si;
          rq[q] = ri;
          vq[q] = uq[q];
          uq[q] = ui;
        } else {
          is[i] = si;
          ir[i] = ri;
        }
        ext[i] = ui;
      });
      for (int h = bd - 1 - tid; h < nh; h += bd) {
        const float sj = k == 0 ? gw[h] : fmaf(beta, gs[h], gw[h]);
        gs[h] = sj;
        const float rj = fmaf(-alpha, sj, gr[h]);
        gr[h] = rj;
        ext[nloc + h] = dih[h] * rj;
      }
      ++k;
    }
    total += k;
    if (bad) { status = CGP_ERR_NONFINITE; break; }
    // ---- FP64 correction and projection; x published for the next residual ----
    {
      double v1[1] = {0.0};
      for (int i = tid; i < nloc; i += bd) {
        const double xi = x[i] + (double)ie[i];
        x[i] = xi;
        v1[0] += xi;
      }
      put_partials<1>(d, lb, red, v1, sh);
      if (!grp.sync(sh)) return;
      get_totals<1>(d, red, sh);
      ++red;
      const double mx = d.fixed ? 0.0 : sh.tot[0] / d.n;
      for (int i = tid; i < nloc; i += bd) x[i] -= mx;
      if (!grp.sync(sh)) return;
    }
    ++sweeps;
    if (k == 0 && total < d.max_it) { status = CGP_ERR_BREAKDOWN; break; }  // no inner progress
  }
  finish(d, lb, status, total, sweeps, rel, rel, bnorm);
}

// The solve loop of a system in the general kernels: dataflow iterations where
// the launch asked for them (d.flow: rows resident, reductions tagged, blocks of
// at least kFlowMinBlock threads; cgp_flow.cu has kernels of their own for the
// FP32 register rows), the barrier forms otherwise.
template <int T, bool RES>
__device__ __forceinline__ void solve_any(const Desc& d, int lb, Shared& sh) {
  if (d.mixed) {
    if constexpr (RES) {
      if (d.flow) {
        solve_mixed_flow<T, 0>(d, lb, sh);
        return;
      }
    }
    solve_mixed<T, RES>(d, lb, sh);
  } else if (d.classic) {
    solve_fp64<T, RES>(d, lb, sh);
  } else {
    if constexpr (RES) {
      if (d.flow) {
        solve_fp64_flow<T>(d, lb, sh);
        return;
      }
    }
    solve_fp64_sr<T, RES>(d, lb, sh);
  }
}

}  // namespace
}  // namespace cgp
