// Spectral Score Smoothing: one thread block per head, the whole transform chain on chip.
//
// A real sequence of even length n is packed into a complex one of length N = n/2
// (odd n: length N = n with zero imaginary part). The complex transform is an in-place
// mixed-radix decimation-in-frequency FFT: radices 2 to 19 one butterfly per thread, larger primes
// as a product with the p x p cosine and sine matrices, register-tiled. Its output is left in digit-reversed order
// and addressed through a table, and the inverse is the matching decimation-in-time chain, so no reordering pass
// and no second buffer is needed. Lengths with a large prime factor go through a chirp-z
// (Bluestein) convolution of a length M >= 2N - 1 made of small radices.
// The work buffer lives in shared memory when it fits. A longer one lies in a per-block global scratch (it stays in
// L2): the first pass, and the last of the inverse, run there; after it the transform falls apart into contiguous
// blocks, which are brought into shared memory a chunk at a time for everything in between.
//
// What bounds it: a head is a chain of short phases with a barrier between them, each a few thousand cycles of
// shared-memory traffic and index arithmetic on one SM; HBM sees only the scores coming in and the indices going out.
// So the block reads the scores once into shared memory, 512 threads keep eight or more independent accesses in
// flight each (128 registers), every access to shared memory is a compile-time LDS / STS through a swizzle
// that keeps the power-of-two strides of the passes and the digit-reversed reads of the spectrum off the same banks,
// and twiddles come from a two-level table of roots of unity in shared memory. Heads are taken from a queue, since what a
// head costs shows only in its scores. 112 heads of 8160 tokens, no transform: 27 us; 192 heads of 16352 tokens, two
// transforms each of 16 * 7 * 73 points: 195 us (two turns on 148 SMs).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "select.cuh"

namespace akv {
namespace {

constexpr int kT = kSssThreads;
constexpr int kWarps = kT / 32;

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {  // a * conj(b)
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 mul_i(float2 a) { return make_float2(-a.y, a.x); }    // i * a
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }   // -i * a

// ---- work buffers ------------------------------------------------------------------------
// Shared memory: element e sits at e + e / 16 + e / 256. Sixteen float2 are one turn of the banks: neighbours come out on
// different banks, so do the power-of-two strides of late passes, and the two divisors together keep the strides of the
// digit-reversed reads of the spectrum apart to a few. (An exclusive-or of the low four bits with the next twelve
// has fewer conflicts still, but six operations per access instead of four; a radix-8 pass has sixteen accesses.)
extern __shared__ __align__(16) float2 g_sbuf[];
struct SmemBuf {
  static __device__ __forceinline__ int slot(int e) { return e + (e >> 4) + (e >> 8); }
  __device__ __forceinline__ float2 ld(int e) const { return g_sbuf[slot(e)]; }
  __device__ __forceinline__ void st(int e, float2 v) const { g_sbuf[slot(e)] = v; }
};
struct GlobBuf {
  float2* p;
  __device__ __forceinline__ float2 ld(int e) const { return p[e]; }
  __device__ __forceinline__ void st(int e, float2 v) const { p[e] = v; }
};

// The n scores of a head as transform entries: entry m = tokens 2m and 2m + 1 (packed) or token m and zero.
struct Scores {
  const float* x;
  bool packed, pairs;  // pairs: packed, and the head starts on an 8-byte boundary
  __device__ __forceinline__ float2 pair(int m) const { return *reinterpret_cast<const float2*>(x + 2 * m); }
  __device__ __forceinline__ float2 single(int m) const {
    const int j = packed ? 2 * m : m;
    const float v = x[j], w = x[packed ? j + 1 : j];
    return make_float2(v, packed ? w : 0.f);
  }
  __device__ __forceinline__ float2 entry(int m) const { return pairs ? pair(m) : single(m); }
};

// Loops of the block over [0, n). An access to L2 takes some 700 cycles from here, and with 16 warps on the SM it is
// the number of accesses in flight that decides the time of every phase: get(i) is therefore issued for U elements
// before the first use(i, value), with no branch in between (a branch, even a uniform one, keeps the compiler from
// moving the loads of one element above the use of another: the sweep that reads a head's 32736 scores took 23 k cycles
// that way, 32 round trips one after another).
template <int U, class Get, class Use>
__device__ __forceinline__ void batched(int n, Get get, Use use) {
  batched_loop<kT, U>(n, get, use);
}

// use(m, entry m) for every entry of the head's scores.
template <int U, class Use>
__device__ __forceinline__ void for_entries(const Scores& sc, int n, Use use) {
  if (sc.pairs) batched<U>(n, [&](int m) { return sc.pair(m); }, use);
  else batched<U>(n, [&](int m) { return sc.single(m); }, use);
}

// Roots of unity e^{-2 pi i e / Q} of one order Q, 0 <= e < Q: the product, in double precision, of two table entries in
// shared memory, 256 fine ones and Q / 256 coarse ones, rounded once. Every twiddle, chirp and post-twiddle of a head
// comes from here, and is the correctly rounded value that a table of all Q of them would hold.
// (Tables of whole passes in global memory were tried first: all blocks then read the same lines at the same time, and
// L2 delivered 6 bytes per clock and SM: one sweep over 15840 twiddles took 23 k cycles, more than the
// butterflies it belonged to. A table of all Q in shared memory fits beside the shorter buffers only. Products of
// single-precision entries are twice as fast, but off by an ulp or two, and the selection behind the transform sees
// the last bit: with attention sinks every other rounding of the transform moves a token across the threshold in 5 % of the
// heads at n = 16352.)
__device__ __forceinline__ double2 zmul(double2 a, double2 b) { return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x)); }
__device__ __forceinline__ float2 rounded(double2 a) { return make_float2(static_cast<float>(a.x), static_cast<float>(a.y)); }
struct Roots {
  int at;    // where the fine entries lie in g_sbuf, in float2 (even); the coarse ones follow
  int mult;  // order of the table / order asked for
  __device__ __forceinline__ double2 exact(int e) const {
    const double2* tab = reinterpret_cast<const double2*>(g_sbuf + at);
    e *= mult;
    return zmul(tab[e & 255], tab[256 + (e >> 8)]);
  }
  __device__ __forceinline__ float2 operator()(int e) const { return rounded(exact(e)); }
};

// ---- shared state ------------------------------------------------------------------------
constexpr int kDirectBins = 12;
constexpr int kDirectRows = 128;  // entries per thread the table covers: even n up to 131072, odd n up to 65535

// First bins of the spectrum without a transform (see direct_bins).
struct DirectSmem {
  float2 tab[kDirectRows][kDirectBins];     // tab[i][k] = w_k^{a kT i}
  float2 part[kWarps][kDirectBins];         // per warp: bins 1 .. kDirectBins - 1
  double energy[kDirectBins];               // |F_k|^2 as it counts towards the cumulative energy
  double tot[3];                            // F_0 (= sum x), the energy threshold rho E, the margin of a decision
  float2 bin[kDirectBins];                  // F_k
  int kstar;                                // stage 1: k*, -1: left to the transform, -2: the bins decide
  int k_hi;                                 // last bin to evaluate; after stage 3: k* or -1
};

constexpr int kMaxChunks = 2 * (65536 / 64 + 1);  // energy sums: 32 bins each, from both ends of the spectrum
constexpr int kPreInts = 832;                     // prefix sums of the selection, for a buffer in shared memory

struct SssShared {
  FftPlan pl;
  // the head at hand; kept here and not in registers, which the passes want all to themselves
  const float* x;
  float* y;
  float2* g;
  int32_t *out, *kstar_out;
  int k_keep;
  double sums[3];      // sum x, sum x^2, alternating sum
  int kstar, slot;
  int loaded;          // plan whose roots lie in shared memory
  uint32_t kmin, kmax;
  int pre[kPreInts];
  alignas(16) union {  // never alive at the same time
    DirectSmem ds;
    double energy[kMaxChunks];
    SelectSmem sel;
  };
};
__shared__ __align__(16) SssShared S;

// While a pass runs none of the union is alive: a prime pass stages rows of its matrix there.
constexpr int kPassScratch = sizeof(double) * kMaxChunks / sizeof(float4);
__device__ __forceinline__ float4* pass_scratch() { return reinterpret_cast<float4*>(S.energy); }

// ---- passes ------------------------------------------------------------------------------
// cos / sin of 2 pi t / R, 0 <= t < R, for the odd radices handled in registers (t is a compile-time constant at every use).
template <int R>
__device__ __forceinline__ constexpr float rcos(int t) {
  constexpr float c3[2] = {1.f, -0.5f};
  constexpr float c5[3] = {1.f, 0.30901699437494745f, -0.8090169943749475f};
  constexpr float c7[4] = {1.f, 0.6234898018587336f, -0.2225209339563144f, -0.9009688679024191f};
  constexpr float c11[6] = {1.f, 0.84125353283118121f, 0.41541501300188644f, -0.142314838273285f, -0.65486073394528499f,
                            -0.95949297361449737f};
  constexpr float c13[7] = {1.f, 0.88545602565320991f, 0.56806474673115592f, 0.12053668025532301f,
                            -0.35460488704253545f, -0.74851074817110119f, -0.97094181742605201f};
  constexpr float c17[9] = {1.f, 0.9324722294043558f, 0.73900891722065912f, 0.44573835577653827f, 0.092268359463302f,
                            -0.27366299007208286f, -0.60263463637925639f, -0.85021713572961415f, -0.98297309968390178f};
  constexpr float c19[10] = {1.f, 0.94581724170063468f, 0.7891405093963936f, 0.54694815812242687f, 0.24548548714079915f,
                             -0.08257934547233232f, -0.40169542465296946f, -0.67728157162574107f, -0.87947375120648907f,
                             -0.98636130340272237f};
  const int i = 2 * t > R ? R - t : t;
  return R == 3 ? c3[i < 2 ? i : 0] : R == 5 ? c5[i < 3 ? i : 0] : R == 7 ? c7[i < 4 ? i : 0] : R == 11 ? c11[i < 6 ? i : 0]
         : R == 13 ? c13[i < 7 ? i : 0] : R == 17 ? c17[i < 9 ? i : 0] : c19[i];
}
template <int R>
__device__ __forceinline__ constexpr float rsin(int t) {
  constexpr float s3[2] = {0.f, 0.8660254037844386f};
  constexpr float s5[3] = {0.f, 0.9510565162951535f, 0.5877852522924731f};
  constexpr float s7[4] = {0.f, 0.7818314824680298f, 0.9749279121818236f, 0.4338837391175581f};
  constexpr float s11[6] = {0.f, 0.54064081745559756f, 0.90963199535451833f, 0.9898214418809328f, 0.75574957435425827f,
                            0.28173255684142967f};
  constexpr float s13[7] = {0.f, 0.46472317204376851f, 0.82298386589365635f, 0.99270887409805397f, 0.93501624268541483f,
                            0.66312265824079519f, 0.23931566428755768f};
  constexpr float s17[9] = {0.f, 0.36124166618715295f, 0.67369564364655721f, 0.89516329135506232f, 0.99573417629503452f,
                            0.96182564317281907f, 0.7980172272802395f, 0.5264321628773558f, 0.18374951781657033f};
  constexpr float s19[10] = {0.f, 0.32469946920468349f, 0.61421271268966782f, 0.83716647826252857f, 0.96940026593933042f,
                             0.99658449300666985f, 0.91577332665505744f, 0.73572391067313162f, 0.47594739303707354f,
                             0.16459459028073389f};
  const int i = 2 * t > R ? R - t : t;
  const float v = R == 3 ? s3[i < 2 ? i : 0] : R == 5 ? s5[i < 3 ? i : 0] : R == 7 ? s7[i < 4 ? i : 0]
                : R == 11 ? s11[i < 6 ? i : 0] : R == 13 ? s13[i < 7 ? i : 0] : R == 17 ? s17[i < 9 ? i : 0] : s19[i];
  return 2 * t > R ? -v : v;
}

// In-register DFT of R points: X_c = sum_s v_s exp(-/+ 2 pi i s c / R)  (INV: plus sign).
template <int R, bool INV>
__device__ __forceinline__ void dft_small(float2 (&v)[R]) {
  auto rot = [](float2 a) { return INV ? mul_i(a) : mul_mi(a); };  // times exp(-/+ i pi / 2)
  if constexpr (R == 2) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  } else if constexpr (R == 4) {
    const float2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]), t2 = cadd(v[1], v[3]), t3 = rot(csub(v[1], v[3]));
    v[0] = cadd(t0, t2);
    v[2] = csub(t0, t2);
    v[1] = cadd(t1, t3);
    v[3] = csub(t1, t3);
  } else {
    constexpr int H = (R - 1) / 2;
    float2 p[H + 1], q[H + 1];
#pragma unroll
    for (int s = 1; s <= H; ++s) {
      p[s] = cadd(v[s], v[R - s]);
      q[s] = csub(v[s], v[R - s]);
    }
    const float2 v0 = v[0];
    float2 sum = v0;
#pragma unroll
    for (int s = 1; s <= H; ++s) sum = cadd(sum, p[s]);
    v[0] = sum;
#pragma unroll
    for (int c = 1; c <= H; ++c) {
      float2 A = v0, B = make_float2(0.f, 0.f);
#pragma unroll
      for (int s = 1; s <= H; ++s) {
        const float cc = rcos<R>((s * c) % R), ss = rsin<R>((s * c) % R);
        A.x = fmaf(p[s].x, cc, A.x);
        A.y = fmaf(p[s].y, cc, A.y);
        B.x = fmaf(q[s].x, ss, B.x);
        B.y = fmaf(q[s].y, ss, B.y);
      }
      // forward: X_c = A - i B, X_{R-c} = A + i B; inverse: the other way round
      const float2 iB = mul_i(B);
      v[c] = INV ? cadd(A, iB) : csub(A, iB);
      v[R - c] = INV ? csub(A, iB) : cadd(A, iB);
    }
  }
}

// v[c] times w1^c (INV: times its conjugate), c = 1 .. R - 1; the powers are formed in double precision and rounded each.
template <int R, bool INV>
__device__ __forceinline__ void twiddle(float2 (&v)[R], double2 w1) {
  double2 w = w1;
#pragma unroll
  for (int c = 1; c < R; ++c) {
    const float2 r = rounded(w);
    v[c] = INV ? cmulc(v[c], r) : cmul(v[c], r);
    if (c + 1 < R) w = zmul(w, w1);
  }
}

// t / m for t < 2^32 / m by a multiplication: magic = ceil(2^32 / m). (t m <= (length / R)^2 < 2^32 for every pass.)
struct FastDiv {
  uint32_t m, magic;
  __device__ __forceinline__ explicit FastDiv(int d) : m(d), magic(d > 1 ? 0xffffffffu / static_cast<uint32_t>(d) + 1u : 0u) {}
  __device__ __forceinline__ int div(int t) const { return m > 1 ? static_cast<int>(__umulhi(static_cast<uint32_t>(t), magic)) : t; }
};

// One in-place pass of radix R over `total` elements that fall into sub-transforms of length ns (thread per butterfly).
// Forward (decimation in frequency): DFT_R, then multiply output c by W_ns^{j c}.
// Inverse (decimation in time): multiply input c by W_ns^{-j c}, then inverse DFT_R.
// `in` and `out` are the same buffer, or two views of it (the element is then moved on the way).
template <int R, bool INV, class In, class Out>
__device__ __forceinline__ void pass_small(const In& in, const Out& out, int total, int ns, int N, const Roots& root) {
  const int m = ns / R, nb = total / R, step = N / ns;
  const FastDiv dm(m);
#pragma unroll 1
  for (int t = threadIdx.x; t < nb; t += kT) {
    const int b = dm.div(t), j = t - b * m;
    const int e0 = b * ns + j;
    float2 v[R];
#pragma unroll
    for (int s = 0; s < R; ++s) v[s] = in.ld(e0 + s * m);
    if (INV && m > 1) twiddle<R, true>(v, root.exact(j * step));
    dft_small<R, INV>(v);
    if (!INV && m > 1) twiddle<R, false>(v, root.exact(j * step));
#pragma unroll
    for (int s = 0; s < R; ++s) out.st(e0 + s * m, v[s]);
  }
  __syncthreads();
}

// The same for the two radices that want most of a thread's registers, out of the way of the others.
template <int R, bool INV, class Buf>
__device__ __noinline__ void pass_mid(const Buf buf, int total, int ns, int N, const Roots root) {
  pass_small<R, INV>(buf, buf, total, ns, N, root);
}

// Two passes of small radices in one trip through shared memory: R1 on sub-transforms of length ns, then R2 on the R1 pieces
// of each. A thread holds the R1 x R2 elements that meet; operations and roundings are those of the two passes one after
// the other, so only the number of barriers and of loads and stores changes.
template <int R1, int R2, bool INV>
__device__ __forceinline__ void pass_pair(int total, int ns, int N, const Roots& root) {
  const SmemBuf buf;
  const int m1 = ns / R1, m2 = m1 / R2, step = N / ns;
  const FastDiv dm(m2);
#pragma unroll 1
  for (int t = threadIdx.x; t < total / (R1 * R2); t += kT) {
    const int b = dm.div(t), j = t - b * m2;
    const int e0 = b * ns + j;
    float2 x[R2][R1];
#pragma unroll
    for (int s2 = 0; s2 < R2; ++s2)
#pragma unroll
      for (int s1 = 0; s1 < R1; ++s1) x[s2][s1] = buf.ld(e0 + s1 * m1 + s2 * m2);
    const double2 w2 = root.exact(R1 * j * step);
    auto outer = [&]() {  // the pass of radix R1
#pragma unroll
      for (int s2 = 0; s2 < R2; ++s2) {
        const double2 w1 = root.exact((j + s2 * m2) * step);
        if (INV) twiddle<R1, true>(x[s2], w1);
        dft_small<R1, INV>(x[s2]);
        if (!INV) twiddle<R1, false>(x[s2], w1);
      }
    };
    if (!INV) outer();
#pragma unroll
    for (int c = 0; c < R1; ++c) {
      float2 u[R2];
#pragma unroll
      for (int s2 = 0; s2 < R2; ++s2) u[s2] = x[s2][c];
      if (INV && m2 > 1) twiddle<R2, true>(u, w2);
      dft_small<R2, INV>(u);
      if (!INV && m2 > 1) twiddle<R2, false>(u, w2);
#pragma unroll
      for (int s2 = 0; s2 < R2; ++s2) x[s2][c] = u[s2];
    }
    if (INV) outer();
#pragma unroll
    for (int s2 = 0; s2 < R2; ++s2)
#pragma unroll
      for (int s1 = 0; s1 < R1; ++s1) buf.st(e0 + s1 * m1 + s2 * m2, x[s2][s1]);
  }
  __syncthreads();
}
// Whether two passes of these radices go through pass_pair. Only in a chirp-z, which runs every pass four times: a direct
// transform runs it once a direction, mostly from a cold instruction cache, and the pair's longer code costs what its
// shorter way saves (N = 496: 41 -> 44 us; 11985: 122 -> 127). And only where half the threads get a share. The smoothing kernel
// at n = 12170 (M = 12288): 121 -> 100 us; at 8564: 98 -> 88.
__device__ __forceinline__ bool pairable(int r1, int r2, int total) {
  if (!S.pl.bluestein || total < kT / 2 * r1 * r2) return false;
  return (r1 == 4 && r2 == 4) || (r1 == 4 && r2 == 2) || (r1 == 3 && r2 == 4) || (r1 == 3 && r2 == 3) || (r1 == 5 && r2 == 3);
}
// The pair at pass i (sub-transforms of length ns there).
template <bool INV>
__device__ __forceinline__ void one_pair(int total, int ns, const FftSeq& sq, int i, const Roots& root) {
  const int N = sq.N;
  switch (sq.radix[i] * 8 + sq.radix[i + 1]) {
    case 4 * 8 + 4: pass_pair<4, 4, INV>(total, ns, N, root); break;
    case 4 * 8 + 2: pass_pair<4, 2, INV>(total, ns, N, root); break;
    case 3 * 8 + 4: pass_pair<3, 4, INV>(total, ns, N, root); break;
    case 3 * 8 + 3: pass_pair<3, 3, INV>(total, ns, N, root); break;
    default: pass_pair<5, 3, INV>(total, ns, N, root); break;
  }
}

// The same pass for an odd prime radix p, kMaxSmall < p <= kMaxPrime. With inputs s and p - s folded into P_s = a_s + a_{p-s}
// and Q_s = a_s - a_{p-s}, outputs c and p - c come from the same real-by-complex sums, X_c = A_c -/+ i B_c,
// A_c = a_0 + sum_s P_s cos(2 pi s c / p), B_c = sum_s Q_s sin(2 pi s c / p): a product of a small matrix with as many
// columns as there are butterflies. A thread computes a tile of TO outputs x TC butterflies in registers: per s it reads TC
// values of P and of Q and TO (cos, sin) pairs, the latter the same for most of a warp and staged in shared memory, for 4 TO TC
// FMAs. 8 x 2 or 8 x 1 where that makes tiles for five warps, in one round (4815 = 45 x 107: 71 -> 59 us against three rounds of
// 2 x 1), 2 x 1 for few butterflies (which are latency: a length of 7 x 167 has 44 tiles of 8 x 2, two warps' worth). The folding sweep (inverse) and the write-back (forward) carry the
// pass twiddles. (An earlier version gave a thread 5 outputs of one butterfly and looked the cosines up by (s c mod p): the
// radix-73 pass of N = 8176 took 45-55 k cycles, seven loads and their index arithmetic for every 20 FMAs.)
template <bool INV, class Buf, int TO, int TC>
__device__ __forceinline__ void prime_product(const Buf& buf, int ns, int p, int m, int nb, int step, const Roots& root,
                                              const float2* __restrict__ mat) {
  const int H = (p - 1) / 2, Cp = fft_mat_cols(p);
  const FastDiv dm(m);
  const int n_ct = Cp / TO;                 // tiles of outputs
  const int tiles = (nb + TC - 1) / TC;     // tiles of butterflies
  const int n_round = (tiles * n_ct + kT - 1) / kT;
  const int per_round = min((tiles + n_round - 1) / n_round, kT / n_ct);  // rounds of equal size
  float4* s_mat = pass_scratch();
  const int s_rows = min(H, kPassScratch / (Cp / 2));  // matrix rows staged at a time
  int staged = -1;
  for (int p0 = 0; p0 < tiles; p0 += per_round) {
    const int np = min(per_round, tiles - p0);
    const int ct = static_cast<int>(threadIdx.x) / np;  // neighbouring threads: the same outputs of neighbouring butterflies
    const int jt = p0 + static_cast<int>(threadIdx.x) - ct * np;
    const bool live = ct < n_ct;
    int e[TC], j[TC];
    float2 A[TC][TO], B[TC][TO];
#pragma unroll
    for (int h = 0; h < TC; ++h) {
      const int col = min(TC * jt + h, nb - 1), b = dm.div(col);
      j[h] = col - b * m;
      e[h] = b * ns + j[h];
#pragma unroll
      for (int i = 0; i < TO; ++i) {
        A[h][i] = buf.ld(e[h]);
        B[h][i] = make_float2(0.f, 0.f);
      }
    }
    for (int s0 = 0; s0 < H; s0 += s_rows) {
      const int rows = min(s_rows, H - s0);
      if (staged != s0) {
        __syncthreads();
        const float4* src = reinterpret_cast<const float4*>(mat + s0 * Cp);
        batched<4>(rows * (Cp / 2), [&](int t) { return __ldg(src + t); }, [&](int t, float4 v) { s_mat[t] = v; });
        staged = s0;
        __syncthreads();
      }
      if (live) {
        const float4* w4 = s_mat + ct * (TO / 2);
#pragma unroll 2
        for (int s = s0 + 1; s <= s0 + rows; ++s) {
          float2 P[TC], Q[TC];
#pragma unroll
          for (int h = 0; h < TC; ++h) {
            P[h] = buf.ld(e[h] + s * m);
            Q[h] = buf.ld(e[h] + (p - s) * m);
          }
#pragma unroll
          for (int i = 0; i < TO; i += 2) {
            const float4 w = w4[i >> 1];  // (cos, sin) of outputs i and i + 1
#pragma unroll
            for (int h = 0; h < TC; ++h) {
              A[h][i].x = fmaf(P[h].x, w.x, A[h][i].x);
              A[h][i].y = fmaf(P[h].y, w.x, A[h][i].y);
              B[h][i].x = fmaf(Q[h].x, w.y, B[h][i].x);
              B[h][i].y = fmaf(Q[h].y, w.y, B[h][i].y);
              A[h][i + 1].x = fmaf(P[h].x, w.z, A[h][i + 1].x);
              A[h][i + 1].y = fmaf(P[h].y, w.z, A[h][i + 1].y);
              B[h][i + 1].x = fmaf(Q[h].x, w.w, B[h][i + 1].x);
              B[h][i + 1].y = fmaf(Q[h].y, w.w, B[h][i + 1].y);
            }
          }
          w4 += Cp / 2;
        }
      }
    }
    __syncthreads();  // every thread of the round has read its inputs
    if (live) {
#pragma unroll
      for (int h = 0; h < TC; ++h) {
        if (TC * jt + h >= nb) continue;
#pragma unroll
        for (int i = 0; i < TO; ++i) {
          const int c = ct * TO + i;
          if (c > H) continue;
          if (c == 0) {
            buf.st(e[h], A[h][i]);
            continue;
          }
          const float2 iB = mul_i(B[h][i]);
          float2 xc = INV ? cadd(A[h][i], iB) : csub(A[h][i], iB), xq = INV ? csub(A[h][i], iB) : cadd(A[h][i], iB);
          if (!INV && m > 1) {
            xc = cmul(xc, root(j[h] * c * step));
            xq = cmul(xq, root(j[h] * (p - c) * step));
          }
          buf.st(e[h] + c * m, xc);
          buf.st(e[h] + (p - c) * m, xq);
        }
      }
    }
  }
  __syncthreads();
}
template <bool INV, class Buf>
__device__ __noinline__ void pass_prime(const Buf buf, int total, int ns, int N, int p, const Roots root,
                                        const float2* __restrict__ mat) {
  if (p <= kMaxSmall) {  // asked here and not with the smaller radices, which would make every transform 0.3 to 1 us longer
    if (p == 17) pass_mid<17, INV, Buf>(buf, total, ns, N, root);
    else pass_mid<19, INV, Buf>(buf, total, ns, N, root);
    return;
  }
  const int m = ns / p, nb = total / p, H = (p - 1) / 2, step = N / ns;
  const FastDiv dm(m), dn(nb);
#pragma unroll 2
  for (int t = threadIdx.x; t < nb * H; t += kT) {
    const int s = dn.div(t) + 1, col = t - (s - 1) * nb;
    const int b = dm.div(col), j = col - b * m;
    const int e0 = b * ns + j + s * m, e1 = b * ns + j + (p - s) * m;
    float2 x = buf.ld(e0), y = buf.ld(e1);
    if (INV && m > 1) {
      x = cmulc(x, root(j * s * step));
      y = cmulc(y, root(j * (p - s) * step));
    }
    buf.st(e0, cadd(x, y));
    buf.st(e1, csub(x, y));
  }
  if (nb * fft_mat_cols(p) >= 16 * 160) prime_product<INV, Buf, 8, 2>(buf, ns, p, m, nb, step, root, mat);
  else if (nb * fft_mat_cols(p) >= 8 * 160) prime_product<INV, Buf, 8, 1>(buf, ns, p, m, nb, step, root, mat);
  else prime_product<INV, Buf, 2, 1>(buf, ns, p, m, nb, step, root, mat);
}

// Pass i of a sequence, on `total` elements whose sub-transforms have length ns.
template <bool INV, class Buf>
__device__ __forceinline__ void one_pass(const Buf& buf, int total, int ns, const FftSeq& sq, int i, const Roots& root,
                                         const float2* __restrict__ tables) {
  const int N = sq.N;
  switch (sq.radix[i]) {
    case 4: pass_small<4, INV>(buf, buf, total, ns, N, root); break;
    case 2: pass_small<2, INV>(buf, buf, total, ns, N, root); break;
    case 3: pass_small<3, INV>(buf, buf, total, ns, N, root); break;
    case 5: pass_small<5, INV>(buf, buf, total, ns, N, root); break;
    case 7: pass_small<7, INV>(buf, buf, total, ns, N, root); break;
    case 11: pass_small<11, INV>(buf, buf, total, ns, N, root); break;
    case 13: pass_small<13, INV>(buf, buf, total, ns, N, root); break;
    default: pass_prime<INV, Buf>(buf, total, ns, N, sq.radix[i], root, tables + sq.base + sq.mat[i]); break;
  }
}
// Passes [i0, i1) of a transform, forward in order or inverse in reverse order, on a buffer of `total` elements; ns:
// length of the sub-transforms at pass i0.
template <class Buf>
__device__ __noinline__ void passes_fwd(const Buf buf, int total, int ns, const FftSeq& sq, int i0, int i1, const Roots root,
                                        const float2* __restrict__ tables) {
#pragma unroll 1
  for (int i = i0; i < i1; ++i) {
    if constexpr (std::is_same<Buf, SmemBuf>::value) {
      if (i + 1 < i1 && pairable(sq.radix[i], sq.radix[i + 1], total)) {
        one_pair<false>(total, ns, sq, i, root);
        ns /= sq.radix[i] * sq.radix[i + 1];
        ++i;
        continue;
      }
    }
    one_pass<false>(buf, total, ns, sq, i, root, tables);
    ns /= sq.radix[i];
  }
}
template <class Buf>
__device__ __noinline__ void passes_inv(const Buf buf, int total, int ns, const FftSeq& sq, int i0, int i1, const Roots root,
                                        const float2* __restrict__ tables) {
  for (int i = i0; i < i1; ++i) ns /= sq.radix[i];
#pragma unroll 1
  for (int i = i1 - 1; i >= i0; --i) {
    ns *= sq.radix[i];
    if constexpr (std::is_same<Buf, SmemBuf>::value) {
      if (i > i0 && pairable(sq.radix[i - 1], sq.radix[i], total)) {
        --i;
        ns *= sq.radix[i];
        one_pair<true>(total, ns, sq, i, root);
        continue;
      }
    }
    one_pass<true>(buf, total, ns, sq, i, root, tables);
  }
}

// A direct transform of a buffer in global memory: the first g passes couple elements that lie far apart and run on the
// global buffer; after them the transform falls apart into contiguous blocks of length len, of which `chunk` elements'
// worth at a time go through shared memory for the remaining passes. The inverse runs the steps backwards.
template <bool INV>
__device__ __noinline__ void fft_big(float2* g, const FftPlan& pl, const Roots root, const float2* __restrict__ tables) {
  const FftSeq& sq = pl.seq;
  const GlobBuf gb{g};
  const SmemBuf sb;
  int len = sq.N;
  for (int i = 0; i < pl.g_pass; ++i) len /= sq.radix[i];
  if (!INV) passes_fwd(gb, sq.N, sq.N, sq, 0, pl.g_pass, root, tables);
  for (int c0 = 0; c0 < sq.N; c0 += pl.chunk) {
    const int n = min(pl.chunk, sq.N - c0);
    batched<8>(n, [&](int t) { return g[c0 + t]; }, [&](int t, float2 v) { sb.st(t, v); });
    __syncthreads();
    if (!INV) passes_fwd(sb, n, len, sq, pl.g_pass, sq.n_pass, root, tables);
    else passes_inv(sb, n, len, sq, pl.g_pass, sq.n_pass, root, tables);
    for (int t = threadIdx.x; t < n; t += kT) g[c0 + t] = sb.ld(t);
    __syncthreads();
  }
  if (INV) passes_inv(gb, sq.N, sq.N, sq, 0, pl.g_pass, root, tables);
}

// Where the forward transform leaves bin k.
__device__ __forceinline__ int seq_pos(const FftSeq& sq, int k) {
  int len = sq.N, p = 0;
  for (int i = 0; i < sq.n_pass; ++i) {
    const int r = sq.radix[i];
    len /= r;
    const int q = k / r;
    p += (k - q * r) * len;
    k = q;
  }
  return p;
}

// ---- chirp-z -----------------------------------------------------------------------------
// The last forward pass of a convolution (radix R, no twiddles), the product with the transformed filter and the first
// inverse pass work on the same R neighbours: one sweep in registers does all three.
template <int R>
__device__ __forceinline__ void pass_filter(int total, const float2* __restrict__ filt) {
  const SmemBuf sb;
  struct Piece {
    float4 f[R / 2];
  };
  const float4* f4 = reinterpret_cast<const float4*>(filt);  // filters start on 16-byte boundaries
  batched<4>(total / R,
             [&](int t) {
               Piece p;
#pragma unroll
               for (int s = 0; s < R / 2; ++s) p.f[s] = __ldg(f4 + R / 2 * t + s);
               return p;
             },
             [&](int t, const Piece& p) {
               float2 v[R];
#pragma unroll
               for (int s = 0; s < R; ++s) v[s] = sb.ld(R * t + s);
               dft_small<R, false>(v);
#pragma unroll
               for (int s = 0; s < R / 2; ++s) {
                 v[2 * s] = cmul(v[2 * s], make_float2(p.f[s].x, p.f[s].y));
                 v[2 * s + 1] = cmul(v[2 * s + 1], make_float2(p.f[s].z, p.f[s].w));
               }
               dft_small<R, true>(v);
#pragma unroll
               for (int s = 0; s < R; ++s) sb.st(R * t + s, v[s]);
             });
  __syncthreads();
}
__device__ __forceinline__ void apply_filter(const FftSeq& sq, int total, const float2* __restrict__ filt) {
  if (sq.radix[sq.n_pass - 1] == 4) pass_filter<4>(total, filt);
  else pass_filter<2>(total, filt);  // convolution lengths are multiples of 4
}

// The chirp e^{-i pi j^2 / N} = e^{-2 pi i (j^2 mod 2N) / 2N}, j < N.
struct Chirp {
  Roots root;  // of order 2N
  uint32_t two_n, magic;
  __device__ __forceinline__ Chirp(const Roots& r, int N) : root(r), two_n(2 * N), magic(0xffffffffu / (2u * N)) {}
  __device__ __forceinline__ float2 operator()(int j) const {
    const uint64_t q = static_cast<uint64_t>(j) * static_cast<uint64_t>(j);  // j < 2^17
    // the quotient from the upper bits is short by a little; the remainder is put right
    uint32_t r = static_cast<uint32_t>(q) - __umulhi(static_cast<uint32_t>(q >> 4), magic) * 16u * two_n;
    while (r >= 16u * two_n) r -= 16u * two_n;
    r -= __umulhi(r, magic) * two_n;
    while (r >= two_n) r -= two_n;
    return root(static_cast<int>(r));
  }
};

// Views of the global buffer at the two ends of a long convolution: the chirp goes on with the first pass's reads and off
// with the last pass's writes. conj: conjugate on the way in and out, which turns the forward transform into the
// unnormalised inverse.
struct ChirpIn {
  Scores sc;
  const float2* g;  // null: the head's scores
  Chirp chirp;
  int n_in;
  bool conj;
  __device__ __forceinline__ float2 ld(int e) const {
    if (e >= n_in) return make_float2(0.f, 0.f);
    float2 v = g ? g[e] : sc.entry(e);
    if (conj) v = cconj(v);
    return cmul(v, chirp(e));
  }
};
struct ChirpOut {
  float2* g;
  Chirp chirp;
  int n_out;
  bool conj;
  __device__ __forceinline__ void st(int e, float2 v) const {
    if (e >= n_out) return;
    v = cmul(v, chirp(e));
    g[e] = conj ? cconj(v) : v;
  }
};
template <bool INV, class In, class Out>
__device__ __noinline__ void end_pass(const In in, const Out out, const FftSeq& sq, const Roots root) {
  const int M = sq.N;
  switch (sq.radix[0]) {  // convolution lengths are made of 7, 5, 3 and 2
    case 7: pass_small<7, INV>(in, out, M, M, M, root); break;
    case 5: pass_small<5, INV>(in, out, M, M, M, root); break;
    case 3: pass_small<3, INV>(in, out, M, M, M, root); break;
    default: pass_small<4, INV>(in, out, M, M, M, root); break;
  }
}

// Chirp-z: entries [0, n_in) (natural order; the rest counts as zero) in, bins 0..n_out-1 of DFT_N (natural order) out.
// `filt` is the transformed wrapped chirp that fits this pair of ranges: the plan's filter for n_in = n_out = N, and for
// a half plan the filter (N in, (N+1)/2 out) or filter2 ((N+1)/2 in, N out). Short: the work buffer in shared memory.
// Long: scratch g; from_scores: the input is read from the scores. root: of order M; rootn: of order 2N.
template <bool CONJ>
__device__ __forceinline__ void chirp_z_smem(const FftPlan& pl, const Roots& root, const Roots& rootn,
                                             const float2* __restrict__ tables, int n_in, int n_out,
                                             const float2* __restrict__ filt) {
  const SmemBuf sb;
  const Chirp chirp(rootn, pl.N);
  const int M = pl.M, last = pl.seq.n_pass - 1;
#pragma unroll 2
  for (int j = threadIdx.x; j < n_in; j += kT) {
    const float2 v = sb.ld(j);
    sb.st(j, cmul(CONJ ? cconj(v) : v, chirp(j)));
  }
  for (int j = n_in + threadIdx.x; j < M; j += kT) sb.st(j, make_float2(0.f, 0.f));
  __syncthreads();
  passes_fwd(sb, M, M, pl.seq, 0, last, root, tables);
  apply_filter(pl.seq, M, filt);
  passes_inv(sb, M, M, pl.seq, 0, last, root, tables);
#pragma unroll 2
  for (int j = threadIdx.x; j < n_out; j += kT) {
    const float2 v = cmul(sb.ld(j), chirp(j));
    sb.st(j, CONJ ? cconj(v) : v);
  }
  __syncthreads();
}
__device__ __noinline__ void chirp_z_big(const Scores sc, bool from_scores, bool conj, float2* g, const FftPlan& pl, const Roots root,
                                         const Roots rootn, const float2* __restrict__ tables, int n_in, int n_out,
                                         const float2* __restrict__ filt) {
  const FftSeq& sq = pl.seq;
  const Chirp chirp(rootn, pl.N);
  const int M = pl.M, last = sq.n_pass - 1;
  const SmemBuf sb;
  const GlobBuf gb{g};
  int len = M;
  for (int i = 0; i < pl.g_pass; ++i) len /= sq.radix[i];
  end_pass<false>(ChirpIn{sc, from_scores ? nullptr : g, chirp, n_in, conj}, gb, sq, root);
  passes_fwd(gb, M, M / sq.radix[0], sq, 1, pl.g_pass, root, tables);
  for (int c0 = 0; c0 < M; c0 += pl.chunk) {
    const int n = min(pl.chunk, M - c0);
    batched<8>(n, [&](int t) { return g[c0 + t]; }, [&](int t, float2 v) { sb.st(t, v); });
    __syncthreads();
    passes_fwd(sb, n, len, sq, pl.g_pass, last, root, tables);
    apply_filter(sq, n, filt + c0);
    passes_inv(sb, n, len, sq, pl.g_pass, last, root, tables);
    for (int t = threadIdx.x; t < n; t += kT) g[c0 + t] = sb.ld(t);
    __syncthreads();
  }
  passes_inv(gb, M, M / sq.radix[0], sq, 1, pl.g_pass, root, tables);
  end_pass<true>(gb, ChirpOut{g, chirp, n_out, conj}, sq, root);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Inclusive prefix of v over the warp.
__device__ __forceinline__ double warp_prefix(double v) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) >= o) v += t;
  }
  return v;
}

// ---- low cut-offs without a transform ---------------------------------------------------------------------------
// Attention scores are positive, so where a head attends evenly their mean carries most of the energy and k* is a
// handful of bins. The block then evaluates those bins directly, O(n (k* + T)) operations instead of two transforms of
// n points: the total energy comes from Parseval's identity (sum of squares in fp64), the first kDirectBins bins from
// their definition. The shortcut is taken only when those bins decide k* with a clear margin and k* + T lies inside
// them; otherwise the transform path decides.
// Entry m = t + kT i of thread t holds token m (odd n) or tokens 2m and 2m + 1 (even n): token j = a m + b.
// With w_k = e^{-2 pi i k / n},  w_k^j = w_k^{a t} * w_k^b * w_k^{a kT i}: the first factor is a power of one
// rotation per thread, the second a power of one rotation per head, the third comes from a table of
// rows x kDirectBins entries built once per head. A bin then costs one read of the table and two FMAs per token.
// e^{-2 pi i (j k mod n) / n}: the product is reduced exactly in integers, the angle then lies in [-pi, pi] where the
// fast sine and cosine are good to 5e-7.
__device__ __forceinline__ float2 unit_root(int j, int k, int n, float inv_n, float two_pi_over_n) {
  const int jk = j * k;                                   // j <= 2^17, k < 16
  int m = jk - n * __float2int_rd(static_cast<float>(jk) * inv_n);
  m += m < 0 ? n : 0;
  m -= m >= n ? n : 0;
  m -= 2 * m > n ? n : 0;                                 // (-n/2, n/2]
  float sn, cs;
  __sincosf(static_cast<float>(m) * two_pi_over_n, &sn, &cs);
  return make_float2(cs, -sn);
}

// e^{-2 pi i j / n} for 0 <= j < 2^22, to fp32 rounding
__device__ __forceinline__ float2 unit_root_exact(int j, int n) {
  int m = j % n;
  m -= 2 * m > n ? n : 0;  // (-n/2, n/2]: the quotient below is rounded relative to an angle of at most pi
  float sn, cs;
  sincospif(static_cast<float>(2 * m) / static_cast<float>(n), &sn, &cs);
  return make_float2(cs, -sn);
}

struct DirectGeom {
  int a, M, rows;          // tokens per entry, entries, entries per thread
  float2 wt, v;            // w_1^{a t}, w_1
};

__device__ __forceinline__ DirectGeom direct_geom(int n, bool packed) {
  DirectGeom g;
  g.a = packed ? 2 : 1;
  g.M = n / g.a;
  g.rows = (g.M + kT - 1) / kT;
  // one accurate rotation per thread, w_1^t; w_1 is the ratio of two neighbours' and w_1^{2t} its square
  const float2 w = unit_root_exact(threadIdx.x, n);
  const float2 w_l0 = make_float2(__shfl_sync(0xffffffffu, w.x, 0), __shfl_sync(0xffffffffu, w.y, 0));
  const float2 w_l1 = make_float2(__shfl_sync(0xffffffffu, w.x, 1), __shfl_sync(0xffffffffu, w.y, 1));
  g.v = cmulc(w_l1, w_l0);
  g.wt = packed ? cmul(w, w) : w;
  return g;
}

// Stage 1, from three sums over the block (s[0] = sum x, s[1] = sum x^2, s[2] = alternating sum; one thread): the mean
// bin F_0 and, by Parseval, the total over the bins 0 .. floor(n/2). Often that settles the cut-off at bin 0, and only
// the T bins of the cosine band are needed; it also tells the heads for which the other eleven bins are not worth
// evaluating (a matter of time only: both paths compute the same function): a spectrum without a strong low end
// would have to hold the missing energy there in an eighth of what lies outside the mean.
__device__ __forceinline__ void direct_stage1(const double* s, int n, int smooth_mode, float rho, float kappa, int T, DirectSmem* ds) {
  const int Kb = n / 2;
  const double F0 = s[0], FN = s[2];
  const double total = 0.5 * (static_cast<double>(n) * s[1] + F0 * F0 + ((n & 1) ? 0.0 : FN * FN));
  const bool no_mean = smooth_mode == AUDIOKV_SMOOTH_ENERGY_NO_MEAN;
  const double rest = fmax(total - F0 * F0, 0.0), whole = no_mean ? rest : total;
  const double thr = static_cast<double>(rho) * whole;
  // The rotations are good to about 1e-6, so a bin's energy is off by up to 2e-6 |F_k| F_0: a decision is taken
  // here only when it is clear of the threshold by several times the sum of that over the bins.
  const double margin = 1e-5 * (whole + fabs(F0) * static_cast<double>(sqrtf(static_cast<float>(rest))));
  int ks = -2, k_hi = kDirectBins - 1;  // -2: the bins have to decide
  if (smooth_mode == AUDIOKV_SMOOTH_FIXED_FRACTION) {
    ks = static_cast<int>(floor(static_cast<double>(kappa) * Kb));
  } else if (!(whole > 0.0)) {
    ks = -1;
  } else if (!no_mean && F0 * F0 >= thr + margin) {
    ks = 0;
  } else if ((no_mean ? 0.0 : F0 * F0) + 0.125 * rest < thr) {
    ks = -1;
  }
  if (ks >= 0) {
    k_hi = ks + T;
    if (k_hi >= kDirectBins || k_hi >= Kb) ks = -1;
  }
  ds->tot[0] = F0;
  ds->tot[1] = thr;
  ds->tot[2] = margin;
  ds->bin[0] = make_float2(static_cast<float>(F0), 0.f);
  ds->energy[0] = no_mean ? 0.0 : F0 * F0;
  ds->k_hi = k_hi;
  ds->kstar = ks;
}

// Stages 2 and 3, where stage 1 did not send the head to the transform. entry(m): the head's scores. Returns k* (and
// leaves the bins in ds->bin and the table in ds->tab) or -1 when the transform has to decide.
template <class Entry>
__device__ __forceinline__ int direct_bins(Entry entry, int n, bool packed, const DirectGeom& g, int T, DirectSmem* ds) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    const float inv_n = 1.f / static_cast<float>(n), tpn = 6.283185307179586f * inv_n;
    for (int e = threadIdx.x; e < g.rows * kDirectBins; e += kT) {
      const int i = e / kDirectBins, k = e - i * kDirectBins;
      ds->tab[i][k] = unit_root(g.a * kT * i, k, n, inv_n, tpn);
    }
  }
  __syncthreads();
  const int k_hi = ds->k_hi;
  // bins 1 .. k_hi from their definition, four at a time
  float2 pk = make_float2(1.f, 0.f), vk = pk;
#pragma unroll 1
  for (int k0 = 1; k0 <= k_hi; k0 += 4) {
    float2 A0[4], A1[4];  // at most 128 entries per thread: their sums stay in fp32
#pragma unroll
    for (int q = 0; q < 4; ++q) A0[q] = A1[q] = make_float2(0.f, 0.f);
    batched<4>(g.M, entry, [&](int m, float2 x) {
      const float2* tb = &ds->tab[m / kT][0];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 t = tb[min(k0 + q, kDirectBins - 1)];
        A0[q].x = fmaf(x.x, t.x, A0[q].x);
        A0[q].y = fmaf(x.x, t.y, A0[q].y);
        A1[q].x = fmaf(x.y, t.x, A1[q].x);
        A1[q].y = fmaf(x.y, t.y, A1[q].y);
      }
    });
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      pk = cmul(pk, g.wt);  // w_k^{a t}
      vk = cmul(vk, g.v);   // w_k
      float2 F = A0[q];
      if (packed) F = cadd(F, cmul(A1[q], vk));
      F = cmul(F, pk);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        F.x += __shfl_xor_sync(0xffffffffu, F.x, o);
        F.y += __shfl_xor_sync(0xffffffffu, F.y, o);
      }
      if (lane == 0 && k0 + q <= k_hi) ds->part[warp][k0 + q] = F;
    }
  }
  __syncthreads();
  // warp k adds up bin k over the warps' parts (lane w reads warp w's)
  if (warp >= 1 && warp <= k_hi) {
    float2 t = lane < kWarps ? ds->part[lane][warp] : make_float2(0.f, 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
      t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
    }
    if (lane == 0) {
      ds->energy[warp] = static_cast<double>(t.x) * t.x + static_cast<double>(t.y) * t.y;
      ds->bin[warp] = t;
    }
  }
  __syncthreads();
  if (ds->kstar >= 0) return ds->kstar;  // settled in stage 1
  // Stage 3: the first bin at which the cumulative energy reaches the threshold, if it does so clearly
  if (threadIdx.x == 0) {
    const int Kb = n / 2;
    const double thr = ds->tot[1], margin = ds->tot[2];
    int ks = -1;
    double run = 0.0;
#pragma unroll 1
    for (int k = 0; k < kDirectBins; ++k) {
      const double before = run;
      run += ds->energy[k];
      if (run >= thr) {
        if (run >= thr + margin && (k == 0 || before <= thr - margin)) ks = k;
        break;
      }
    }
    if (ks < 0 || ks + T >= kDirectBins || ks + T >= Kb) ks = -1;
    ds->k_hi = ks;
  }
  __syncthreads();
  return ds->k_hi;
}

// The residual mix of every token from the masked bins c_k = mask_k F_k (1 up to k*, raised cosine over the T bins
// after it): y_j = alpha (1/n) [c_0 + 2 sum_k Re(c_k conj(w_k^j))] + (1 - alpha) x_j. emit(m, x, y) gets the scores and
// the results of entry m.
template <class Entry, class Emit>
__device__ __forceinline__ void direct_apply(Entry entry, Emit emit, int n, bool packed, const DirectGeom& g, int kstar, int T, float al, const DirectSmem* ds) {
  constexpr int kRows = 8;
  const float om = 1.f - al, c0 = ds->bin[0].x, inv_n = 1.f / static_cast<float>(n);
  const float band = 3.14159265358979f / static_cast<float>(T + 1);
#pragma unroll 1
  for (int i0 = 0; i0 < g.rows; i0 += kRows) {
    float acc0[kRows], acc1[kRows];
#pragma unroll
    for (int ii = 0; ii < kRows; ++ii) acc0[ii] = acc1[ii] = 0.f;
    float2 pk = make_float2(1.f, 0.f), vk = pk;
#pragma unroll 1
    for (int k = 1; k <= kstar + T; ++k) {
      pk = cmul(pk, g.wt);
      vk = cmul(vk, g.v);
      const float mask = k <= kstar ? 1.f : 0.5f * (1.f + __cosf(static_cast<float>(k - kstar) * band));
      const float2 g0 = cscale(cmulc(ds->bin[k], pk), mask);  // c_k conj(w_k^{a t})
      const float2 g1 = cmulc(g0, vk);
#pragma unroll
      for (int ii = 0; ii < kRows; ++ii) {
        const float2 tb = ds->tab[min(i0 + ii, kDirectRows - 1)][k];
        acc0[ii] = fmaf(g0.x, tb.x, fmaf(g0.y, tb.y, acc0[ii]));  // Re(g conj(tb))
        acc1[ii] = fmaf(g1.x, tb.x, fmaf(g1.y, tb.y, acc1[ii]));
      }
    }
#pragma unroll
    for (int ii = 0; ii < kRows; ++ii) {
      const int m = threadIdx.x + kT * (i0 + ii);
      if (m < g.M) {
        const float2 x = entry(m);
        emit(m, make_float2(fmaf(al, fmaf(2.f, acc0[ii], c0) * inv_n, om * x.x),
                            fmaf(al, fmaf(2.f, acc1[ii], c0) * inv_n, om * x.y)));
      }
    }
  }
}

// ---- the kernel --------------------------------------------------------------------------
__device__ __forceinline__ Scores scores_of_head() {
  const bool packed = S.pl.packed != 0;
  return Scores{S.x, packed, packed && (reinterpret_cast<uintptr_t>(S.x) & 7) == 0};
}

// The first `count` entries of the plan's tables of roots, into shared memory.
__device__ __forceinline__ void load_roots(const FftPlan& pl, const float2* __restrict__ tables, int count) {
  const float4* src = reinterpret_cast<const float4*>(tables + pl.root_offset);
  float4* dst = reinterpret_cast<float4*>(g_sbuf + pl.root_at);
  batched<2>(count, [&](int t) { return __ldg(src + t); }, [&](int t, float4 v) { dst[t] = v; });
}

// A work buffer of either kind, for the steps around the transforms.
template <bool BIG>
struct Work {
  float2* g;
  __device__ __forceinline__ float2 ld(int e) const {
    if constexpr (BIG) return g[e];
    else return SmemBuf().ld(e);
  }
  __device__ __forceinline__ void st(int e, float2 v) const {
    if constexpr (BIG) g[e] = v;
    else SmemBuf().st(e, v);
  }
};

// Smoothing of one head by transforms: the entries of `sc` (BIG = false: already in the buffer) become the masked
// spectrum's inverse in the buffer, natural order; *inv_scale is what that still has to be multiplied with.
template <bool BIG>
__device__ __noinline__ void transform_head(const Shape& sh, const float2* __restrict__ tables) {
  const FftPlan& pl = S.pl;
  float2* g = S.g;
  const Scores sc = scores_of_head();
  const Work<BIG> buf{g};
  const int n = pl.n, N = pl.N, Kb = n / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool packed = pl.packed != 0, direct = pl.bluestein == 0, half = pl.half != 0;
  // the slots of bins k and N - k after the forward passes: in order for a chirp-z, else from the plan
  const uint32_t* __restrict__ rec = reinterpret_cast<const uint32_t*>(tables + pl.pos_offset);
  auto slots_of = [&](int k) -> uint2 {
    if (!direct) return make_uint2(k, k == 0 ? 0 : N - k);
    if (pl.wide_pos) return make_uint2(__ldg(rec + 2 * k), __ldg(rec + 2 * k + 1));
    const uint32_t r = __ldg(rec + k);
    return make_uint2(r & 0xffffu, r >> 16);
  };
  const Roots root{pl.root_at, pl.root_mult};                              // of the passes
  const Roots rootn{direct ? pl.root_at : pl.root_at + 2 * pl.root_count, 1};  // of order 2N (odd n, direct: not used)
  if (S.loaded != pl.id) {
    load_roots(pl, tables, pl.root_count + pl.root_count2);
    __syncthreads();
    if (threadIdx.x == 0) S.loaded = pl.id;
  }

  // 1. forward complex transform; bin k then sits at pos(k)
  if constexpr (BIG) {
    if (direct) {
      for_entries<8>(sc, N, [&](int m, float2 v) { g[m] = v; });
      __syncthreads();
      fft_big<false>(g, pl, root, tables);
    } else {
      chirp_z_big(sc, true, false, g, pl, root, rootn, tables, N, half ? Kb + 1 : N, tables + pl.filter_offset);
    }
  } else {
    if (direct) passes_fwd(SmemBuf(), N, N, pl.seq, 0, pl.seq.n_pass, root, tables);
    else chirp_z_smem<false>(pl, root, rootn, tables, N, half ? Kb + 1 : N, tables + pl.filter_offset);
  }

  // 2. The spectrum of the real sequence and the cut-off, the smallest k with E(k) = sum_{i<=k} |F_i|^2 >= rho E(Kb) (fp64).
  //    packed: Z is turned into F pairwise in place (the slot of bin 0 holds (F_0, F_N), both real). Energies are summed by
  //    chunks of 32 neighbouring bins (one warp's share): chunk i of the low bins at energy[i], chunk i of their partners
  //    N - k, which count downwards, at energy[2 nc - 1 - i].
  //    The threshold is taken from the sum of all bins. Parseval's identity gives a total before that, but the bins are
  //    fp32 and their own sum is off from it by some 1e-7 of the energy, which near rho = 1 is many bins of a spectrum that falls
  //    off. So it serves only to end the sums early, 2048 low bins at a time, and only for a cut-off that is clear of the
  //    threshold by more than the two totals can differ.
  const bool no_mean = sh.smooth_mode == AUDIOKV_SMOOTH_ENERGY_NO_MEAN;  // variant: bin 0 adds no energy
  const int n_low = packed ? N / 2 + 1 : Kb + 1;
  const int nc = (n_low + 31) / 32, n_chunk = packed ? 2 * nc : nc;
  auto sq_abs = [](float2 f) -> double { return fma(static_cast<double>(f.x), static_cast<double>(f.x), static_cast<double>(f.y) * f.y); };
  // the spectrum's bins k and N - k from the two values of the packed transform. Bin 0 and the middle bin of an even N are
  // their own partners; the formulas give them what they should (bin 0: F_0 and F_N).
  auto split = [&](int k, float2 a, float2 b, float2& fk, float2& fq) {
    const float2 zq = cconj(b);
    const float2 E = cscale(cadd(a, zq), 0.5f), T = cmul(mul_mi(cscale(csub(a, zq), 0.5f)), rootn(k));
    fk = cadd(E, T);
    fq = cconj(csub(E, T));
  };
  const bool fixed = sh.smooth_mode == AUDIOKV_SMOOTH_FIXED_FRACTION;  // variant: no energies needed
  int summed = 0;  // chunks of low bins that have their sums and, packed, have been split with their partners
  if (fixed) {
    if (threadIdx.x == 0) S.kstar = min(static_cast<int>(floor(static_cast<double>(sh.smooth_kappa) * Kb)), Kb);
    __syncthreads();
  } else {
    double whole = 0.0, margin = 0.0, early = INFINITY;
    if (nc > 64 && sh.rho < 1.f) {  // more than one turn of sums
      const double F0 = S.sums[0], FN = S.sums[2];
      const double total = 0.5 * (static_cast<double>(n) * S.sums[1] + F0 * F0 + ((n & 1) ? 0.0 : FN * FN));
      // The transform is off by less than kOff of the spectrum's norm (33 roundings; six were the most seen), the energies by this:
      constexpr double kOff = 2e-6;
      whole = no_mean ? fmax(total - F0 * F0, 0.0) : total;
      margin = 2.0 * kOff * sqrt(whole * total) + kOff * kOff * total;
      early = static_cast<double>(sh.rho) * whole + margin;
    }
    double run = 0.0;
    constexpr int U = 4;
    static_assert(U * kWarps == 64, "two chunks per lane and round");
#pragma unroll 1
    for (bool last = false;; last = true) {
#pragma unroll 1
      while (summed < nc && (last || !(run >= early))) {
        uint2 at[U];
#pragma unroll
        for (int q = 0; q < U; ++q) at[q] = slots_of(min(32 * (summed + q * kWarps + warp) + lane, n_low - 1));
#pragma unroll
        for (int q = 0; q < U; ++q) {
          const int c = summed + q * kWarps + warp, k = 32 * c + lane;
          double el = 0.0, eh = 0.0;
          if (k < n_low) {
            float2 fk = buf.ld(at[q].x);
            if (packed) {
              float2 fq;
              split(k, fk, buf.ld(at[q].y), fk, fq);
              buf.st(at[q].x, k == 0 ? make_float2(fk.x, fq.x) : fk);
              if (k > 0) buf.st(at[q].y, fq);
              eh = 2 * k == N ? 0.0 : sq_abs(fq);
            }
            el = k == 0 && no_mean ? 0.0 : sq_abs(fk);
          }
          // both sums in one tree: the lower half of the warp goes on with the low bins, the upper half with the others
          const double ol = __shfl_xor_sync(0xffffffffu, el, 16), oh = __shfl_xor_sync(0xffffffffu, eh, 16);
          double v = (lane & 16) ? eh + oh : el + ol;
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (c < nc) {
            if (lane == 0) S.energy[c] = v;
            if (lane == 16 && packed) S.energy[2 * nc - 1 - c] = v;
          }
        }
        summed += U * kWarps;
        __syncthreads();
        if (summed < nc && !last) run += warp_sum(S.energy[summed - 64 + lane] + S.energy[summed - 32 + lane]);
      }
      const bool exact = summed >= nc;
      if (warp == 0) {
        // every lane sums a run of chunks; then the lane, the chunk and the bin that reach the threshold
        const int avail = exact ? n_chunk : summed, per = (avail + 31) / 32, c0 = min(avail, lane * per), c1 = min(avail, c0 + per);
        double own = 0.0;
        for (int c = c0; c < c1; ++c) own += S.energy[c];
        const double inc = warp_prefix(own), all = __shfl_sync(0xffffffffu, inc, 31), sum = exact ? all : whole;
        // all of a total above zero is reached at the last bin, whatever the rounding of the sums
        const double thr = sh.rho < 1.f || !(sum > 0.0) ? static_cast<double>(sh.rho) * sum : INFINITY;
        const uint32_t hit = __ballot_sync(0xffffffffu, inc >= thr);
        int ks = exact ? Kb : -1;
        if (hit) {
          double before = inc - own;
          int chunk = c0;
          while (chunk + 1 < c1 && !(before + S.energy[chunk] >= thr)) before += S.energy[chunk++];
          chunk = __shfl_sync(0xffffffffu, chunk, __ffs(hit) - 1);
          before = __shfl_sync(0xffffffffu, before, __ffs(hit) - 1);
          // the chunk's bins in ascending order, one per lane
          const bool upper = packed && chunk >= nc;
          const int k = upper ? N - (32 * (2 * nc - 1 - chunk) + 31 - lane) : 32 * chunk + lane;
          const bool in = upper ? (k >= N - N / 2 && 2 * k != N && k <= N) : k < n_low;
          double e = 0.0;
          if (in) {
            if (packed && (k == N || k == 0)) {
              const float2 f = buf.ld(0);
              e = k == N ? static_cast<double>(f.y) * f.y : no_mean ? 0.0 : static_cast<double>(f.x) * f.x;
            } else if (!(k == 0 && no_mean)) {
              const uint2 at = slots_of(upper ? N - k : k);
              e = sq_abs(buf.ld(upper ? at.y : at.x));
            }
          }
          const double up_to = before + warp_prefix(e);
          const uint32_t reach = __ballot_sync(0xffffffffu, in && up_to >= thr);
          const uint32_t any = __ballot_sync(0xffffffffu, in);
          const int at_lane = reach ? __ffs(reach) - 1 : 31 - __clz(any | 1u);  // rounding of the two sums: the chunk's last bin
          ks = min(max(__shfl_sync(0xffffffffu, k, at_lane), 0), Kb);
          const int clear = up_to >= thr + margin && (ks == 0 || up_to - e <= thr - margin);
          if (!__shfl_sync(0xffffffffu, clear, at_lane) && !exact) ks = -1;
        }
        if (lane == 0) S.kstar = ks;
      }
      __syncthreads();
      if (S.kstar >= 0) break;  // else close: with the sums of all bins
      __syncthreads();
    }
  }
  const int kstar = S.kstar;

  // 3. mask (1 up to k*, raised-cosine tail of T bins, 0 beyond) and back to the packed transform
  const int T = sh.transition_bins, k_hi = kstar + min(T, n);  // last bin that is not masked away
  auto weight = [&](int k) -> float {
    if (k <= kstar) return 1.f;
    if (k <= k_hi) return 0.5f * (1.f + cospif(static_cast<float>(k - kstar) / static_cast<float>(T + 1)));
    return 0.f;
  };
  if (packed) {
    batched<4>(n_low, slots_of, [&](int k, uint2 at) {
      float2 ok = make_float2(0.f, 0.f), oq = ok;
      if (k <= k_hi) {  // else its partner, further up, is masked away as well
        float2 fk = buf.ld(at.x), fq = buf.ld(at.y);
        if (k >= 32 * summed) {
          split(k, fk, fq, fk, fq);
        } else if (k == 0) {
          fq = make_float2(fk.y, 0.f);
          fk.y = 0.f;
        }
        fk = cscale(fk, weight(k));
        fq = cconj(cscale(fq, weight(N - k)));
        const float2 E = cscale(cadd(fk, fq), 0.5f), O = cmulc(cscale(csub(fk, fq), 0.5f), rootn(k));
        ok = cadd(E, mul_i(O));
        oq = cconj(csub(E, mul_i(O)));
      }
      buf.st(at.x, ok);
      if (k > 0) buf.st(at.y, oq);
    });
  } else if (half) {
    // bins 0 .. Kb alone go back: x_j = (2 / N) Re sum_{k <= Kb} h_k e^{+2 pi i j k / N}, h_0 = F_0 / 2, h_k = F_k
    for (int k = threadIdx.x; k <= Kb; k += kT) buf.st(k, cscale(buf.ld(k), k == 0 ? 0.5f * weight(0) : weight(k)));
  } else {
    batched<4>(Kb + 1, slots_of, [&](int k, uint2 at) {
      const float w = weight(k);
      buf.st(at.x, cscale(buf.ld(at.x), w));
      if (k > 0) buf.st(at.y, cscale(buf.ld(at.y), w));
    });
  }
  __syncthreads();

  // 4. inverse complex transform (unnormalised), natural order out
  if constexpr (BIG) {
    if (direct) fft_big<true>(g, pl, root, tables);
    else chirp_z_big(sc, false, true, g, pl, root, rootn, tables, half ? Kb + 1 : N, N, tables + (half ? pl.filter2_offset : pl.filter_offset));
  } else {
    if (direct) passes_inv(SmemBuf(), N, N, pl.seq, 0, pl.seq.n_pass, root, tables);
    else chirp_z_smem<true>(pl, root, rootn, tables, half ? Kb + 1 : N, N, tables + (half ? pl.filter2_offset : pl.filter_offset));
  }
}

// Top-k of the keys in the work buffer. Bit masks and their prefix sums: over the histogram and in S.pre when the buffer
// is on chip, else in the idle dynamic area.
template <bool BIG, bool PAIR>
__device__ __noinline__ void select_head(int window, int* status) {
  const Work<BIG> buf{S.g};
  const int N = S.pl.N;
  uint32_t* words = BIG ? reinterpret_cast<uint32_t*>(g_sbuf) : reinterpret_cast<uint32_t*>(S.sel.hist);
  int* pre = BIG ? reinterpret_cast<int*>(g_sbuf) + select_words(N, PAIR) : S.pre;
  select_entries<kT, PAIR>([&](int m) -> float2 { return buf.ld(m); }, N, S.pl.n, window, S.k_keep, S.kmin, S.kmax, S.out,
                           &S.sel, words, pre, status);
}

// One head from its scores to its smoothed scores and, with `sel`, its kept tokens.
template <bool BIG>
__device__ __noinline__ void smooth_head(const Shape& sh, const float2* __restrict__ tables, bool sel, int* status) {
  const FftPlan& pl = S.pl;
  const Work<BIG> buf{S.g};
  const int n = pl.n, N = pl.N;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool packed = pl.packed != 0;

  // The scores go into the buffer (or stay where they are when it is not on chip); plain, squared and alternating
  // sums are taken on the way, in fp64.
  double sx = 0.0, sxx = 0.0, salt = 0.0;
  {
    const bool even_entry = packed || (threadIdx.x & 1) == 0;  // kT is even: all of a thread's tokens m alike
    const Scores sc = scores_of_head();
    for_entries<8>(sc, N, [&](int m, float2 v) {
      if (!BIG) buf.st(m, v);
      const double d0 = static_cast<double>(v.x), d1 = static_cast<double>(v.y);
      sx += d0 + d1;
      sxx = fma(d0, d0, fma(d1, d1, sxx));
      salt += even_entry ? d0 - d1 : -d0;
    });
  }
  sx = warp_sum(sx);
  sxx = warp_sum(sxx);
  salt = warp_sum(salt);
  if (threadIdx.x == 0) {
    S.kmin = 0xffffffffu;
    S.kmax = 0u;
  }
  double* part = S.energy;  // [3][kWarps]
  if (lane == 0) {
    part[warp] = sx;
    part[kWarps + warp] = sxx;
    part[2 * kWarps + warp] = salt;
  }
  __syncthreads();
  if (warp < 3) {
    const double v = warp_sum(lane < kWarps ? part[warp * kWarps + lane] : 0.0);
    if (lane == 0) S.sums[warp] = v;
  }
  __syncthreads();

  // A low cut-off is settled from the first few bins of the spectrum, without a transform.
  const bool direct_ok = n >= 4 * kDirectBins && N <= kDirectRows * kT;
  int kd = -1;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  auto emit = [&](int m, float2 v) {  // entry m's smoothed scores: to memory, and as keys into the buffer
    const int j = packed ? 2 * m : m;
    if (float* y = S.y) {
      y[j] = v.x;
      if (packed) y[j + 1] = v.y;
    }
    if (sel) {
      const uint32_t a = score_key(v.x), b = packed ? score_key(v.y) : a;
      kmin = min(kmin, min(a, b));
      kmax = max(kmax, max(a, b));
      buf.st(m, make_float2(__uint_as_float(a), __uint_as_float(b)));
    }
  };
  if (direct_ok) {
    if (threadIdx.x == 0) direct_stage1(S.sums, n, sh.smooth_mode, sh.rho, sh.smooth_kappa, sh.transition_bins, &S.ds);
    __syncthreads();
    if (S.ds.kstar != -1) {
      const DirectGeom dg = direct_geom(n, packed);
      auto entry = [&](int m) -> float2 {
        if constexpr (BIG) return scores_of_head().entry(m);
        else return buf.ld(m);
      };
      kd = direct_bins(entry, n, packed, dg, sh.transition_bins, &S.ds);
      if (kd >= 0) direct_apply(entry, emit, n, packed, dg, kd, sh.transition_bins, sh.alpha, &S.ds);
    }
    __syncthreads();  // S.ds makes room for the energies
  }
  if (kd >= 0) {
    if (threadIdx.x == 0 && S.kstar_out) *S.kstar_out = kd;
  } else {
    transform_head<BIG>(sh, tables);
    if (threadIdx.x == 0 && S.kstar_out) *S.kstar_out = S.kstar;
    // residual mix
    const float inv = (pl.half ? 2.f : 1.f) / static_cast<float>(N), al = sh.alpha, om = 1.f - sh.alpha;
    const Scores sc = scores_of_head();
    for_entries<8>(sc, N, [&](int m, float2 v) {
      const float2 z = buf.ld(m);
      emit(m, make_float2(fmaf(al, z.x * inv, om * v.x), fmaf(al, z.y * inv, om * v.y)));
    });
  }
  if (!sel) return;
  // top-k of the smoothed scores, straight from the work buffer
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) {
    atomicMin(&S.kmin, kmin);
    atomicMax(&S.kmax, kmax);
  }
  __syncthreads();
  if (packed) select_head<BIG, true>(sh.window, status);
  else select_head<BIG, false>(sh.window, status);
}

// Variant: local pooling instead of the spectral filter: pooled over |i - j| <= pool_kernel / 2 (average: zero padding counts in
// the divisor; maximum: padding never wins), mixed with alpha and written out; the selection then reads it back. The
// sequence goes through shared memory, in stretches when it is longer; scores and smoothed may be the same array, so what a
// stretch needs from before its start comes from the stretch before.
__device__ __noinline__ void pool_head(const Shape& sh, bool sel, int* status) {
  const int n = S.pl.n;
  const float* x = S.x;
  float* y = S.y;
  float* st = reinterpret_cast<float*>(g_sbuf);  // st[i - base] = x[i]
  if (threadIdx.x == 0) {
    S.kmin = 0xffffffffu;
    S.kmax = 0u;
  }
  const int hw = sh.pool_kernel / 2;  // at most 511
  static_assert(kT > 511, "a thread per value carried over");
  const bool is_max = sh.smooth_mode == AUDIOKV_SMOOTH_MAX_POOL;
  const float inv_pool = 1.f / static_cast<float>(sh.pool_kernel), al = sh.alpha, om = 1.f - sh.alpha;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  const int room = 2 * S.pl.root_at, stretch = n <= room ? n : room - 2 * hw;
  int base = 0;
#pragma unroll 1
  for (int c0 = 0; c0 < n; c0 += stretch) {
    const int c1 = min(n, c0 + stretch), end = min(n, c1 + hw);
    if (c0 > 0) {
      const int t = threadIdx.x;
      const float keep = t < hw ? st[c0 - hw + t - base] : 0.f;
      __syncthreads();
      if (t < hw) st[t] = keep;
      base = c0 - hw;
    }
    batched<8>(end - c0, [&](int t) { return x[c0 + t]; }, [&](int t, float v) { st[c0 + t - base] = v; });
    __syncthreads();
    auto mix = [&](int j, float acc) {
      const float v = fmaf(al, is_max ? acc : acc * inv_pool, om * st[j - base]);
      if (y) y[j] = v;
      kmin = min(kmin, score_key(v));
      kmax = max(kmax, score_key(v));
    };
    // Four tokens of a thread at a time, their reads in flight together, where no window reaches over an end.
    constexpr int Q = 4;
    for (int j0 = c0 + threadIdx.x; j0 < c1; j0 += Q * kT) {
      if (j0 >= hw && j0 + (Q - 1) * kT < c1 && j0 + (Q - 1) * kT + hw < n) {
        const float* p = st + j0 - hw - base;
        float acc[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[q] = is_max ? -INFINITY : 0.f;
        if (is_max) {
#pragma unroll 4
          for (int i = 0; i < sh.pool_kernel; ++i)
#pragma unroll
            for (int q = 0; q < Q; ++q) acc[q] = fmaxf(acc[q], p[i + q * kT]);
        } else {
#pragma unroll 4
          for (int i = 0; i < sh.pool_kernel; ++i)
#pragma unroll
            for (int q = 0; q < Q; ++q) acc[q] += p[i + q * kT];
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) mix(j0 + q * kT, acc[q]);
      } else {
#pragma unroll 1
        for (int j = j0; j < min(c1, j0 + Q * kT); j += kT) {
          const float* p = st - base;
          const int lo = max(0, j - hw), hi = min(n - 1, j + hw);
          float acc = is_max ? -INFINITY : 0.f;
          if (is_max) {
#pragma unroll 8
            for (int i = lo; i <= hi; ++i) acc = fmaxf(acc, p[i]);
          } else {
#pragma unroll 8
            for (int i = lo; i <= hi; ++i) acc += p[i];
          }
          mix(j, acc);
        }
      }
    }
    __syncthreads();  // everybody is done with the stretch
  }
  if (threadIdx.x == 0 && S.kstar_out) *S.kstar_out = 0;
  if (!sel) return;
  if (y == nullptr) {
    if (threadIdx.x == 0) atomicExch(status, AUDIOKV_EDEVICE);
    return;
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&S.kmin, kmin);
    atomicMax(&S.kmax, kmax);
  }
  __syncthreads();  // y is complete; the sequence makes room for the masks
  int* words = reinterpret_cast<int*>(g_sbuf);
  select_entries<kT, false>([&](int j) -> float2 { return make_float2(__uint_as_float(score_key(y[j])), 0.f); }, n, n, sh.window,
                            S.k_keep, S.kmin, S.kmax, S.out, &S.sel, reinterpret_cast<uint32_t*>(words),
                            words + select_words(n, false), status);
}

__global__ void __launch_bounds__(kT, 1)
sss_kernel(Shape sh, const ReqDesc* __restrict__ reqs, const FftPlan* __restrict__ plans,
           const float2* __restrict__ tables, const float* scores, float* smoothed /* may alias scores */,
           int32_t* __restrict__ kstar_out, float2* __restrict__ scratch, int64_t scratch_per_block,
           const int32_t* __restrict__ order, int n_order, int first_head, const int32_t* __restrict__ budgets,
           const int32_t* __restrict__ cu_kept, int32_t* __restrict__ kept_idx, int* __restrict__ status,
           int* __restrict__ queue, HeadQueue hq) {
  // A gather that follows head by head is set up when every block here has started, on the SMs that come free.
  if (hq.done) chain_release();
  // Launched as a programmatic dependent: the block is brought in while the kernel before it drains, reads its plan
  // (written when the plan was made, not by the kernels of the pass), and waits for that kernel only where it first
  // touches the scores.
  bool waited = false;
  if (threadIdx.x == 0) S.loaded = -1;
  const bool sel = budgets != nullptr;

  // A block's first head is its own; after that it takes the next one nobody has. Whether a head needs transforms shows only in
  // its scores, so a deal beforehand leaves some blocks with transforms and others with few bins to evaluate. queue[0] counts the heads taken, queue[1]
  // the blocks that are through; the last of them leaves both at zero for the next launch.
  auto next_slot = [&]() -> int {
    if (n_order <= static_cast<int>(gridDim.x)) return n_order;
    __syncthreads();
    if (threadIdx.x == 0) S.slot = gridDim.x + atomicAdd(queue, 1);
    __syncthreads();
    return S.slot;
  };
  for (int slot = blockIdx.x; slot < n_order; slot = next_slot()) {
    const int u = order ? order[slot] : first_head + slot;  // no list: heads first_head, first_head + 1, ...
    const int r = u / sh.heads_per_req;
    const ReqDesc rq = reqs[r];
    __syncthreads();
    {
      const int* src = reinterpret_cast<const int*>(plans + rq.fft_plan);
      for (int i = threadIdx.x; i < static_cast<int>(sizeof(FftPlan) / 4); i += kT) reinterpret_cast<int*>(&S.pl)[i] = src[i];
    }
    const int64_t base = rq.score_offset + static_cast<int64_t>(u - rq.head_base) * rq.P;
    const int P = rq.P, W = sh.window;
    if (!waited) {
      chain_wait();
      waited = true;
    }
    if (threadIdx.x == 0) {
      if (S.loaded != rq.fft_plan) S.loaded = -1;  // this head's work buffer may run over the roots of the plan before
      S.x = scores + base;
      S.y = smoothed ? smoothed + base : nullptr;
      S.g = scratch + static_cast<int64_t>(blockIdx.x) * scratch_per_block;
      S.kstar_out = kstar_out ? kstar_out + u : nullptr;
      if (sel) {
        int k = budgets[u] - W;
        if (k < 0 || k > P) {
          atomicExch(status, AUDIOKV_EDEVICE);
          k = k < 0 ? 0 : P;
        }
        S.k_keep = k;
        S.out = kept_idx + cu_kept[u];
      }
    }
    __syncthreads();
    if (sh.smooth_mode >= AUDIOKV_SMOOTH_AVG_POOL) pool_head(sh, sel, status);
    else if (S.pl.in_smem) smooth_head<false>(sh, tables, sel, status);
    else smooth_head<true>(sh, tables, sel, status);
    if (hq.done && threadIdx.x == 0) hq.finished(u, S.k_keep + W);  // the selection ends with a barrier
  }
  // Only now: the other gather, whose blocks would sit on the SMs that are through and keep the others' places, is brought in
  // when the last block ends, and its launch is hidden behind that.
  if (!hq.done) chain_release();
  if (n_order > static_cast<int>(gridDim.x) && threadIdx.x == 0) {
    if (atomicAdd(queue + 1, 1) == static_cast<int>(gridDim.x) - 1) {
      atomicExch(queue, 0);
      atomicExch(queue + 1, 0);
    }
  }
}

// ---- tables ---------------------------------------------------------------------------
__device__ __forceinline__ float2 root_of_unity(int64_t num, int den) {  // exp(-2 pi i num / den)
  double s, c;
  sincospi(2.0 * static_cast<double>(num % den) / den, &s, &c);
  return make_float2(static_cast<float>(c), static_cast<float>(-s));
}

// A plan's bytes travel to the device as arguments: of the two table kernels, 4 us for the two together, whatever they hold,
// where a copy out of pinned memory takes 5 us up to 16 KB and 12 above, in front of the table kernel (28 layers of 4 heads
// make 36 KB; reading the pinned memory from the kernel took 40 us). What does not fit these two goes ahead in kernels of
// its own. Each thread reads its own 16 bytes of the argument bank, so the copy is spread over blocks.
struct PlanPart {
  uint4 v[kPlanPartBytes / 16];
};
__device__ __forceinline__ void put_part(const PlanPart& part, uint4* to, int n16, int block, int blocks) {
  for (int i = block * blockDim.x + threadIdx.x; i < n16; i += blocks * blockDim.x) to[i] = part.v[i];
}

__global__ void __launch_bounds__(256) plan_part_kernel(const __grid_constant__ PlanPart part, int n16, uint4* to) {
  put_part(part, to, n16, blockIdx.x, gridDim.x);
}

// Writes the tables of every transform plan, 32 blocks each, and the first n16 x 16 bytes of the workspace from `part`. The
// transform plans, at byte plans_at of the workspace, are read from `part` when they travel in it.
__global__ void __launch_bounds__(256)
fft_table_kernel(const __grid_constant__ PlanPart part, int n16, char* ws, size_t plans_at, float2* __restrict__ tables) {
  chain_wait();  // set up while the pass before drains, which reads what is overwritten here
  chain_release();
  __shared__ FftPlan pl;
  {
    const char* from = (n16 ? reinterpret_cast<const char*>(part.v) : ws) + plans_at + sizeof(FftPlan) * blockIdx.y;
    for (int i = threadIdx.x; i < static_cast<int>(sizeof(FftPlan) / 4); i += blockDim.x)
      reinterpret_cast<int*>(&pl)[i] = reinterpret_cast<const int*>(from)[i];
  }
  put_part(part, reinterpret_cast<uint4*>(ws), n16, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
  __syncthreads();
  const int gid = blockIdx.x * blockDim.x + threadIdx.x, gsz = gridDim.x * blockDim.x;
  // roots: 256 fine entries and the coarse ones, of the order the passes want and, for a chirp-z, of order 2N
  for (int t = gid; t < pl.root_count + pl.root_count2; t += gsz) {
    const bool second = t >= pl.root_count;
    const int i = second ? t - pl.root_count : t, order = second ? 2 * pl.N : pl.seq.N * pl.root_mult;
    double sn, cs;
    sincospi(2.0 * static_cast<double>(i < 256 ? i : (i - 256) * 256) / order, &sn, &cs);
    reinterpret_cast<double2*>(tables + pl.root_offset)[t] = make_double2(cs, -sn);
  }
  for (int i = 0; i < pl.seq.n_pass; ++i) {
    const int R = pl.seq.radix[i];
    if (R > kMaxSmall) {
      const int H = (R - 1) / 2, Cp = fft_mat_cols(R);
      for (int t = gid; t < H * Cp; t += gsz) {
        const int s = t / Cp + 1, c = t - (s - 1) * Cp;
        const float2 w = root_of_unity(static_cast<int64_t>(s) * c, R);
        tables[pl.seq.base + pl.seq.mat[i] + t] = make_float2(w.x, -w.y);  // (cos, sin)
      }
    }
  }
  if (!pl.bluestein) {
    uint32_t* rec = reinterpret_cast<uint32_t*>(tables + pl.pos_offset);
    for (int k = gid; k <= pl.N / 2; k += gsz) {
      const uint32_t a = seq_pos(pl.seq, k), b = seq_pos(pl.seq, k == 0 ? 0 : pl.N - k);
      if (pl.wide_pos) {
        rec[2 * k] = a;
        rec[2 * k + 1] = b;
      } else {
        rec[k] = a | b << 16;
      }
    }
  }
  if (pl.bluestein) {
    const int N = pl.N, M = pl.M;
    // Wrapped conjugate chirp b[d] = exp(+i pi d^2 / N) at position d for index differences d = out - in >= 0 and at
    // M - |d| for d < 0, zero elsewhere. Full plan: |d| < N both ways. Half plan: the forward filter serves d in
    // [-(N-1), Kb] (N inputs, Kb + 1 outputs), the inverse one d in [-Kb, N-1].
    const int Kb = (pl.n - 1) / 2;
    const int pos_f = pl.half ? Kb + 1 : N, neg_f = N;       // forward filter: d in (-neg_f, pos_f)
    const int pos_i = N, neg_i = pl.half ? Kb + 1 : N;       // inverse filter (half plans only)
    auto chirp_at = [&](int d) -> float2 {  // exp(+i pi d^2 / N), the exponent reduced exactly
      const long long q = (static_cast<long long>(d) * d) % (2LL * N);
      double s, c;
      sincospi(static_cast<double>(q) / N, &s, &c);
      return make_float2(static_cast<float>(c), static_cast<float>(s));
    };
    for (int j = gid; j < M; j += gsz) {
      // position j holds difference +j inside the positive support, difference -(M - j) inside the negative one
      // (they never collide: M is at least their total length), zero in between
      const int d = j < N ? j : M - j;
      const float2 b = d < N ? chirp_at(d) : make_float2(0.f, 0.f), zero = make_float2(0.f, 0.f);
      const float2 bn = j < N && M - j < N ? chirp_at(M - j) : b;  // the value on the negative side, should j lie there
      auto wrapped = [&](int pos, int neg) -> float2 { return j < pos ? b : M - j < neg ? bn : zero; };
      tables[pl.filter_offset + j] = wrapped(pos_f, neg_f);
      if (pl.half) tables[pl.filter2_offset + j] = wrapped(pos_i, neg_i);
    }
  }
}

// Transforms each chirp-z filter in place and folds in the 1/M of the inverse: one block per plan and filter. The blocks from
// y = 2 on write the rest of the plan (n16 x 16 bytes) from `part`.
__global__ void __launch_bounds__(kT, 1)
fft_filter_kernel(const __grid_constant__ PlanPart part, int n16, uint4* rest, const FftPlan* __restrict__ plans, float2* __restrict__ tables) {
  const FftPlan& pl = S.pl;
  chain_wait();
  if (blockIdx.y >= 2) {
    put_part(part, rest, n16, (blockIdx.y - 2) * gridDim.x + blockIdx.x, (gridDim.y - 2) * gridDim.x);
    return;
  }
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(FftPlan) / 4); i += kT)
    reinterpret_cast<int*>(&S.pl)[i] = reinterpret_cast<const int*>(plans + blockIdx.x)[i];
  __syncthreads();
  if (!pl.bluestein || (blockIdx.y == 1 && !pl.half)) return;
  const Roots root{pl.root_at, pl.root_mult};
  load_roots(pl, tables, pl.root_count);
  __syncthreads();
  float2* f = tables + (blockIdx.y ? pl.filter2_offset : pl.filter_offset);
  const float inv = 1.f / static_cast<float>(pl.M);
  if (pl.in_smem) {
    const SmemBuf sb;
    batched<8>(pl.M, [&](int j) { return f[j]; }, [&](int j, float2 v) { sb.st(j, v); });
    __syncthreads();
    passes_fwd(sb, pl.M, pl.M, pl.seq, 0, pl.seq.n_pass, root, tables);
#pragma unroll 4
    for (int j = threadIdx.x; j < pl.M; j += kT) f[j] = cscale(sb.ld(j), inv);
  } else {
    fft_big<false>(f, pl, root, tables);
#pragma unroll 4
    for (int j = threadIdx.x; j < pl.M; j += kT) f[j] = cscale(f[j], inv);
  }
}

}  // namespace

int sss_static_smem() { return static_cast<int>(sizeof(SssShared)); }

cudaError_t launch_fft_tables(int n_plans, const char* h_blob, size_t blob_bytes, size_t early_bytes, char* ws, size_t plans_at,
                              float2* d_tables, size_t smem_bytes, Launch ln) {
  cudaError_t e = cudaFuncSetAttribute(fft_filter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
  if (e != cudaSuccess) return e;
  PlanPart part;
  // two parts go with the table kernels, the second with the one that kernels behind may not have waited for
  size_t first = 0, rest = 0;
  if (h_blob && blob_bytes <= 2 * kPlanPartBytes && early_bytes <= kPlanPartBytes) {
    first = std::min(blob_bytes, kPlanPartBytes);
    rest = blob_bytes - first;
  } else if (h_blob) {
    for (size_t at = 0; at < blob_bytes; at += kPlanPartBytes) {  // a transfer: not counted as a launch
      const size_t bytes = std::min(blob_bytes - at, kPlanPartBytes);
      memcpy(part.v, h_blob + at, bytes);
      plan_part_kernel<<<8, 256, 0, ln.stream>>>(part, static_cast<int>(bytes / 16), reinterpret_cast<uint4*>(ws + at));
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  if (first) memcpy(part.v, h_blob, first);
  e = launch_chained(fft_table_kernel, dim3(32, n_plans), dim3(256), 0, ln.stream, part, static_cast<int>(first / 16), ws, plans_at,
                     d_tables);
  ln.done("fft_table");
  if (e != cudaSuccess) return e;
  if (rest) memcpy(part.v, h_blob + first, rest);
  e = launch_chained(fft_filter_kernel, dim3(n_plans, rest ? 2 + (8 + n_plans - 1) / n_plans : 2), dim3(kT), smem_bytes, ln.stream, part,
                     static_cast<int>(rest / 16), reinterpret_cast<uint4*>(ws + first),
                     reinterpret_cast<const FftPlan*>(ws + plans_at), d_tables);
  ln.done("fft_filter");
  return e;
}

cudaError_t launch_sss(const Shape& sh, const ReqDesc* d_reqs, const FftPlan* d_plans, const float2* d_tables,
                       const float* scores, float* smoothed, int32_t* kstar, float2* scratch,
                       int64_t scratch_per_block, int grid, size_t smem_bytes, const int32_t* order, int n_order,
                       int first_head, const int32_t* budgets, const int32_t* cu_kept, int32_t* kept_idx, int* status,
                       int* queue, HeadQueue hq, Launch ln) {
  cudaError_t e = cudaFuncSetAttribute(sss_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
  if (e != cudaSuccess) return e;
  e = launch_chained(sss_kernel, dim3(grid), dim3(kT), smem_bytes, ln.stream, sh, d_reqs, d_plans, d_tables, scores,
                     smoothed, kstar, scratch, scratch_per_block, order, n_order, first_head, budgets, cu_kept, kept_idx,
                     status, queue, hq);
  ln.done(budgets ? "sss_select" : "sss");
  return e;
}

}  // namespace akv
