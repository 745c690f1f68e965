// The Conjugate Gradient of Appendix A with the whole iteration state on the chip.
//
// solver.cu's k_cg streams the state of every node (x, r, p, q: 32 bytes in FP32) through
// HBM or L2 once per iteration and pays a kernel launch, a pipeline ramp and a serial
// finaliser each time.  A GB300 has 152 SMs with 256 KB of registers and 227 KB of shared
// memory each: the state of 2.2 million FP32 nodes (0.7 million in FP64) fits.  Here a
// variant is cut into blocks, one CTA per block, and the CTAs of the variant run its CG
// iterations to the inner stopping test without leaving the kernel:
//   * x, r and p live in shared memory, q in registers (FP64: in shared memory); blocks with
//     displaced cells keep their operator rows' weights there too (FP32), so that an iteration
//     reads nothing but its neighbours' edges from outside;
//   * per iteration the CTAs exchange q at the block edges (each keeps r and p of its halo
//     nodes and advances them itself, bit for bit as their owner does) and partial sums (four
//     dot products and the collapsed body rows).  The variant's first block adds them in a
//     fixed order, forms alpha, beta and the bodies' p, and broadcasts those;
//   * an exchanged value travels in 8-byte words whose upper half is the iteration's
//     number: the reader polls the word itself, with no flag, fence or atomic.  Words are
//     double-buffered by parity: a block writes iteration k+2 only after the broadcast of k+1,
//     which follows every block's sums of k+1, hence its reads of k.
// Batches larger than the chip are queued: CTAs take (variant, block) items from a ticket
// counter, items of a variant next to each other, so at most one variant is partly staffed
// while the others run to their end (the launch is cooperative: all CTAs are resident).
//
// The recurrences, the operator's coefficients and the precision of the dot products are
// k_cg's: FP32 state with two-float dot products, or FP64.  The order of summation differs.
//
// Thread layout: a block is w columns by ns strips of H*ha rows (H = 2 in FP32, 1 in FP64);
// thread t works on column t % w of strip t / w.  In FP32 the two halves of a strip are
// packed: row a of the first half and row a of the second are the two lanes of one 64-bit
// register and of one 8-byte shared-memory element, so the recurrences, the rectangle
// stencil and the dot products run on packed f32x2 instructions with no shuffling of
// lanes.  Rows next to a half's end are kept a second time in the neighbouring half's
// halo slot.
//
// What bounds it (GB300, 2070 MHz): per iteration about 2 us between a CTA's partial sums and
// the next alpha (two hops through L2 of 0.4 us, and the first block's FP64 sums and division
// at 64 cycles a dependent instruction), the rest instruction latency at eight warps per
// scheduler pair.  In the first block four warps sum the dot products and the other four the
// bodies' rows, four bodies at a time with eight lanes each: with all eight warps taking whole sums
// in turn, variants of five and more bodies waited for a second round (five 403x201 channels 8.6
// -> 7.7 us an iteration, one 1024x512 grid in FP64 43 -> 40 us).  Measured, time per CG
// iteration, streaming kernel -> here: five 403x201 channel variants, FP32, 25.5 -> 8.1 us; one
// 128x64 cylinder, FP64, 14.1 (24 with the idle launches of its chunks) -> 8.0 us; 16 solves of
// 256x128, FP32, 18.6 -> 8.9 us; one 1024x512 grid, FP64, 54 -> 40 us (FP64 arithmetic).  256
// variants (62 M nodes): 1.50 -> 1.75 s a solve, hence the limit on the queue.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "batch.h"

namespace pfq4 {

namespace {

constexpr int RNT = 256;                  // threads per CTA
constexpr int RWARPS = RNT / 32;
static_assert(RWARPS > 4, "four warps sum the dot products, the others the bodies");
constexpr int HITER = 3;                  // halo nodes per thread at most
constexpr int HMAX = HITER * RNT;
constexpr int NSMAX = 8;                  // strips per block at most
constexpr int PITCH = RNT + 2 * NSMAX;    // elements of p in one row of all strips, with their side halos

typedef unsigned long long u64;

// ---------------------------------------------------------------- packed arithmetic
__device__ __forceinline__ u64 vfma(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 vadd(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 vsub(u64 a, u64 b) {
  u64 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 vmul(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }

template <typename T> struct VT;
template <> struct VT<float> {
  using V = u64;
  static constexpr int H = 2;
  static constexpr bool REG = true;        // q in registers
  static constexpr int ROWS = 14;          // rows of a half strip at most (shared memory of two CTAs per SM)
  static constexpr int GROWS1 = 6;         // 1 + rows at most where the block's weights lie in shared memory
  static __device__ __forceinline__ V make(const float (&c)[2]) {
    V v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(c[0]), "f"(c[1]));
    return v;
  }
  static __device__ __forceinline__ void split(V v, float (&c)[2]) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c[0]), "=f"(c[1]) : "l"(v));
  }
  static __device__ __forceinline__ V bcast(float x) {
    const float c[2] = {x, x};
    return make(c);
  }
};
template <> struct VT<double> {
  using V = double;
  static constexpr int H = 1;
  static constexpr bool REG = false;       // r and q in shared memory: rolled loops, the FP64 pipe is the bound
  static constexpr int ROWS = 9;           // rows of a strip at most (shared memory of two CTAs per SM)
  static constexpr int GROWS1 = 10;
  static __device__ __forceinline__ V make(const double (&c)[1]) { return c[0]; }
  static __device__ __forceinline__ void split(V v, double (&c)[1]) { c[0] = v; }
  static __device__ __forceinline__ V bcast(double x) { return x; }
};

// ---------------------------------------------------------------- dot products of one iteration
// FP32: the two-float accumulation of k_cg (ff_add_prod), on both halves of a strip at a time.
// Every product is split exactly (TwoProd), added with TwoSum, and the two errors go to the low
// word: ten packed operations per product, about 2^-48 relative error per addition.  (Sums on a
// grid fixed per warp took four, and 0.4 us less an iteration of five 403x201 channels, but kept
// 6e-12 of sum |p q| where magnitudes are spread and lost |r| below 1e-19 a decade earlier.)
template <typename T> struct Dots;
template <> struct Dots<float> {
  u64 s[4], l[4];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = l[k] = 0ull;
  }
  // sum k of (x, y), with ny = -y
  __device__ __forceinline__ void add(int k, u64 x, u64 y, u64 ny) {
    const u64 np = vmul(x, ny);             // -p
    const u64 e = vfma(x, y, np);           // p + e = x y exactly
    const u64 t = vsub(s[k], np);
    const u64 bb = vsub(t, s[k]);
    const u64 err = vsub(vsub(s[k], vsub(t, bb)), vadd(np, bb));
    s[k] = t;
    l[k] = vadd(l[k], vadd(err, e));
  }
  __device__ __forceinline__ void add_row(u64 r, u64 p, u64 q) {
    const u64 nr = vsub(0ull, r), nq = vsub(0ull, q);
    add(0, r, r, nr);
    add(1, p, q, nq);
    add(2, r, q, nq);
    add(3, q, q, nq);
  }
  static __device__ __forceinline__ FF shfl(FF a, int o) {
    return FF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
  }
  static __device__ __forceinline__ double value(FF a) { return (double)a.hi + (double)a.lo; }
  // ff_add of two pairs of sums at once
  struct F2 { u64 hi, lo; };
  static __device__ __forceinline__ F2 plus(F2 a, F2 b) {
    const u64 t = vadd(a.hi, b.hi), bb = vsub(t, a.hi);
    const u64 err = vadd(vadd(vsub(a.hi, vsub(t, bb)), vsub(b.hi, bb)), vadd(a.lo, b.lo));
    const u64 h = vadd(t, err);
    return F2{h, vsub(err, vsub(h, t))};
  }
  // both halves of sums k and k + 1
  __device__ __forceinline__ F2 halves(int k) const {
    float a[2], b[2], c[2], d[2];
    VT<float>::split(s[k], a);
    VT<float>::split(s[k + 1], b);
    VT<float>::split(l[k], c);
    VT<float>::split(l[k + 1], d);
    const float h0[2] = {a[0], b[0]}, h1[2] = {a[1], b[1]}, l0[2] = {c[0], d[0]}, l1[2] = {c[1], d[1]};
    return plus(F2{VT<float>::make(h0), VT<float>::make(l0)}, F2{VT<float>::make(h1), VT<float>::make(l1)});
  }
  // the four sums over the warp: lane k returns sum k (k < 4); each exchange step halves the
  // number of sums a lane carries
  __device__ __forceinline__ double warp_sums(int lane) const {
    const bool up = lane & 16, up8 = lane & 8;
    const F2 a = halves(0), b = halves(2), keep = up ? b : a, give = up ? a : b;
    const F2 f = plus(keep, F2{__shfl_xor_sync(0xffffffffu, give.hi, 16), __shfl_xor_sync(0xffffffffu, give.lo, 16)});
    float h[2], w[2];
    VT<float>::split(f.hi, h);
    VT<float>::split(f.lo, w);
    FF c = ff_add(up8 ? FF{h[1], w[1]} : FF{h[0], w[0]}, shfl(up8 ? FF{h[0], w[0]} : FF{h[1], w[1]}, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) c = ff_add(c, shfl(c, o));
    return __shfl_sync(0xffffffffu, value(c), (lane & 3) * 8);
  }
};
template <> struct Dots<double> {
  double s[4];
  __device__ __forceinline__ void zero() { s[0] = s[1] = s[2] = s[3] = 0.0; }
  __device__ __forceinline__ void add_row(double r, double p, double q) {
    s[0] = fma(r, r, s[0]);
    s[1] = fma(p, q, s[1]);
    s[2] = fma(r, q, s[2]);
    s[3] = fma(q, q, s[3]);
  }
  // each exchange step halves the number of sums a lane carries: 6 additions per lane, not 20
  __device__ __forceinline__ double warp_sums(int lane) const {
    const bool up = lane & 16, up8 = lane & 8;
    const double k0 = up ? s[2] : s[0], k1 = up ? s[3] : s[1], g0 = up ? s[0] : s[2], g1 = up ? s[1] : s[3];
    const double b0 = k0 + __shfl_xor_sync(0xffffffffu, g0, 16), b1 = k1 + __shfl_xor_sync(0xffffffffu, g1, 16);
    double c = (up8 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, up8 ? b0 : b1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    return __shfl_sync(0xffffffffu, c, (lane & 3) * 8);
  }
};

// Sum of single values: two-float in FP32 mode.
template <typename T> struct BodySum;
template <> struct BodySum<float> {
  FF s{0.0f, 0.0f};
  __device__ __forceinline__ void add(float x) { ff_add_value(s, x); }
  __device__ __forceinline__ double warp_sum() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = ff_add(s, Dots<float>::shfl(s, o));
    return Dots<float>::value(s);
  }
};
template <> struct BodySum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ double warp_sum() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
  }
};

// ---------------------------------------------------------------- exchanged words
__device__ __forceinline__ u64 ld_word(const u64* p) {
  u64 w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void ld_word2(const u64* p, u64& a, u64& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_word(u64* p, u64 w) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ void st_word2(u64* p, u64 a, u64 b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void put_double(u64* p, double x, unsigned ep) {
  const u64 b = (u64)__double_as_longlong(x), e = (u64)ep << 32;
  st_word2(p, e | (b & 0xffffffffull), e | (b >> 32));
}
__device__ __forceinline__ double word_double(u64 a, u64 b) {
  return __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
}
__device__ __forceinline__ bool fresh(u64 a, u64 b, unsigned ep) {
  return (unsigned)(a >> 32) == ep && (unsigned)(b >> 32) == ep;
}

// A node's exchanged q: two (FP32) or four (FP64) words in the node's record of the state
// buffer of the other parity, which this kernel does not use for anything else.
template <typename T> struct QWord;
template <> struct QWord<float> {
  u64 w;
  static __device__ __forceinline__ u64* at(u64* words, long long n, unsigned ep) { return words + 2 * n + (ep & 1); }
  __device__ __forceinline__ void load(const u64* p) { w = ld_word(p); }
  __device__ __forceinline__ bool ready(unsigned ep) const { return (unsigned)(w >> 32) == ep; }
  __device__ __forceinline__ float value() const { return __int_as_float((int)(unsigned)w); }
  static __device__ __forceinline__ void put(u64* p, float x, unsigned ep) {
    st_word(p, ((u64)ep << 32) | (unsigned)__float_as_int(x));
  }
};
template <> struct QWord<double> {
  u64 a, b;
  static __device__ __forceinline__ u64* at(u64* words, long long n, unsigned ep) {
    return words + 4 * n + 2 * (ep & 1);
  }
  __device__ __forceinline__ void load(const u64* p) { ld_word2(p, a, b); }
  __device__ __forceinline__ bool ready(unsigned ep) const { return fresh(a, b, ep); }
  __device__ __forceinline__ double value() const { return word_double(a, b); }
  static __device__ __forceinline__ void put(u64* p, double x, unsigned ep) { put_double(p, x, ep); }
};

// ---------------------------------------------------------------- the kernel
template <typename T> __device__ __forceinline__ const T* rect_of(const DevVariant& V);
template <> __device__ __forceinline__ const float* rect_of<float>(const DevVariant& V) { return V.kr32; }
template <> __device__ __forceinline__ const double* rect_of<double>(const DevVariant& V) { return V.kr64; }

struct RItem {               // one block: columns i0 .. i0+w-1, rows j0 .. j0+ns*H*ha-1
  int v, part;               // variant, number of the block in it
  int i0, w, j0;
  int ns, ha;                // strips, rows of a half strip
  int gen;                   // some node's operator row needs stored coefficients
};

struct RVar {                // a variant's blocks
  int part0, parts;          // first partial-sum slot, number of blocks
};

template <typename T>
struct ResArgs {
  MeshDev m;
  VarState* st;
  const SolveParams* prm;
  State4<T>* s[2];           // state records; the other parity's buffer carries the exchanged q
  T* sb;                     // [4][B] body x, r, p, q
  int B;
  const RVar* var;           // [nv]
  const RItem* items;        // a variant's blocks next to each other
  int n_items;
  int* ticket;
  int* join;                 // [nv] blocks of the variant that have started
  u64* pw;                   // [2][4 + nb][blocks][2] partial sums, per variant at 2 qs part0
  long long pw_half;         // words of one parity
  u64* bc;                   // [nv][2][bc_len] what the first block broadcasts: alpha, beta, stop, body p
  u64* pbm;                  // [blocks] bodies with nodes in the block
  int* blist;                // per variant and body: the blocks with its nodes
  int qs;                    // 4 + most bodies of a variant
  unsigned* epoch;           // [nv] number of the variant's last exchange
  int* err;
  int* n_done;
  int poll_limit;
  int test_drop;
  int max_it;
};

constexpr int LISTMAX = 384;             // entries of the first block's lists kept in shared memory
constexpr int JOIN_LIMIT = 1 << 26;       // waits of about a microsecond for a variant's CTAs to start

// Offsets in a block's dynamic shared memory, in bytes (host and device).
template <typename T>
struct Lay {
  using X = VT<T>;
  static constexpr int VB = X::H * (int)sizeof(T);
  int x, r, q, hr, hw, hp, qe, ew, w4, total;
  __host__ __device__ Lay(int ha, int gen) {
    int o = (ha + 2) * PITCH * VB;                           // p with halo
    x = o; o += ha * RNT * VB;
    r = o; o += ha * RNT * VB;
    q = o; if (!X::REG) o += ha * RNT * VB;
    hr = o; o += HMAX * (int)sizeof(T);                      // halo: r,
    hw = o; o += HMAX * 4;                                   //   whose node,
    hp = o; o += HMAX * 4;                                   //   where in p
    qe = o; o += HMAX * (int)sizeof(T);                      // q at the block's edge
    ew = o; o += HMAX * 4;                                   //   and whose node, -1: not published
    w4 = o; if (X::REG && gen) o += 4 * X::GROWS1 * PITCH * VB;   // weights towards E, N, NE and NW neighbours
    total = o;
  }
};

template <typename T>
__global__ void __launch_bounds__(RNT, 2) k_cg_resident(ResArgs<T> g) {
  using X = VT<T>;
  using V = typename X::V;
  constexpr int H = X::H, ROWS = X::ROWS;
  constexpr bool REG = X::REG;
  constexpr int UNR = REG ? ROWS : 1, GUNR = REG ? X::GROWS1 - 1 : 1;
  constexpr int WPV = (int)sizeof(T) / 4;  // words of a broadcast value
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double s_red[RWARPS][4];
  __shared__ double s_yb[RWARPS][MAXB];
  __shared__ double s_tot[4 + MAXB];
  __shared__ T s_b[4][MAXB];               // body x, r, p, q of the current iteration
  __shared__ T s_pb[MAXB];                 // p of each body, as its nodes see it
  __shared__ T s_alpha, s_beta;
  __shared__ unsigned s_bm[2];             // bodies with nodes in this block
  __shared__ struct { double gamma_start, thr, thr_rel, thr_abs2; long long iters, inner, k_max; } s_root;
  __shared__ T s_kr[6];                    // rectangle constants
  __shared__ int s_first[MAXB];            // first block: where a body's list starts in s_list, -1: in global memory
  __shared__ int s_cnt[MAXB];              // first block: blocks with nodes of each body
  __shared__ unsigned short s_list[LISTMAX];   // first block: those blocks, body after body
  __shared__ int s_item, s_stop, s_abort;
  // values of the block that all threads share and that the loops need now and then: kept here
  // rather than in registers, which hold the state (a spill costs far more than these loads)
  __shared__ struct {
    u64 *words, *pw_var, *bc;
    const int* blist;
    VarState* S;
    long long base;
    int P, w, bh, i0, j0, nx, ny, nbu, parts, see;
  } sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // (a wait that gave up in the launch before: its words are not to be continued)
  if (tid == 0) s_abort = *(volatile int*)g.err != 0;
  for (;;) {
    __syncthreads();
    if (s_abort) return;
    if (tid == 0) s_item = atomicAdd(g.ticket, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= g.n_items) return;
    const RItem I = g.items[item];
    const int v = I.v, part = I.part;
    VarState* const S = &g.st[v];
    if (S->phase != PH_CG) continue;       // (a variant cannot finish before this block has joined it)

    // ---- the block
    const RVar R = g.var[v];
    const DevVariant& Vg = g.m.var[v];
    const int nx = Vg.nx, ny = Vg.ny, P = Vg.P, nb = Vg.nb, body0 = Vg.body0;
    const long long base = Vg.base;
    const int w = I.w, ns = I.ns, ha = I.ha, pw = w + 2, bh = ns * H * ha, i0 = I.i0, j0 = I.j0;
    const bool fixed = g.prm->fixed_bodies != 0;
    const int nbu = fixed ? 0 : nb;
    const Lay<T> L(ha, I.gen);
    V* const P2 = reinterpret_cast<V*>(smem);
    T* const Pt = reinterpret_cast<T*>(smem);
    V* const X2 = reinterpret_cast<V*>(smem + L.x);
    T* const Xt = reinterpret_cast<T*>(smem + L.x);
    V* const R2 = reinterpret_cast<V*>(smem + L.r);
    V* const Q2 = reinterpret_cast<V*>(smem + L.q);
    T* const hr = reinterpret_cast<T*>(smem + L.hr);
    int* const hw = reinterpret_cast<int*>(smem + L.hw);     // node offset, -1: none, -2 - k: node of body k
    unsigned* const hp = reinterpret_cast<unsigned*>(smem + L.hp);   // place in Pt | second place << 16
    T* const qe = reinterpret_cast<T*>(smem + L.qe);
    int* const ew = reinterpret_cast<int*>(smem + L.ew);
    V* const W4 = reinterpret_cast<V*>(smem + L.w4);
    constexpr int WPL = X::GROWS1 * PITCH;                   // elements of one weight plane
    const int strip = tid / w, col = tid - strip * w, i = i0 + col;
    const bool on = strip < ns && i <= nx;
    // p of row a, strip s, column c: element (a + 1) PITCH + s (w + 2) + c + 1 (rows a = -1 and
    // ha and columns -1 and w are halo); x: element a RNT + thread.  The strides are constants,
    // so every access of the unrolled loops is a base register and an immediate
    const int p0 = PITCH + strip * pw + col + 1;
    const int plast = p0 + ha * PITCH;                       // the strip's lower halo row
    State4<T>* const rec = g.s[S->buf];
    u64* const words = reinterpret_cast<u64*>(g.s[S->buf ^ 1]);
    auto row_of = [&](int a, int h) { return (strip * H + h) * ha + a; };

    for (int k = tid; k < (ha + 2) * PITCH; k += RNT) P2[k] = V(0);
    for (int k = tid; k < HMAX; k += RNT) qe[k] = T(0);
    if (tid < 2) s_bm[tid] = 0u;
    __syncthreads();

    // ---- kinds of the thread's nodes; do all of them have four undisplaced active cells?
    unsigned freeM = 0, bodyM = 0;
    int kb = -1;                           // the thread's body nodes: none (-1), all of body kb, of several (-2)
    bool gen = false;
    if (on) {
      constexpr uint8_t GEN = sizeof(T) == 4 ? CELL_GEN32 : CELL_GENERAL;
      constexpr uint8_t FL = CELL_ACTIVE | GEN;
      for (int k = 0; k < H * ha; ++k) {
        const int j = j0 + strip * H * ha + k;
        if (j > ny) break;
        const long long n = base + (long long)j * P + i;
        const int kind = g.m.tag[n] & KIND_MASK;
        const unsigned bit = 1u << ((k >= ha ? 16 + k - ha : k));
        if (kind == K_FREE) freeM |= bit;
        else if (kind == K_BODY) bodyM |= bit;
        else continue;
        const bool inner = i > 0 && j > 0 && i < nx && j < ny;
        gen |= !inner || (g.m.tag[n] & FL) != CELL_ACTIVE || (g.m.tag[n - 1] & FL) != CELL_ACTIVE ||
               (g.m.tag[n - P - 1] & FL) != CELL_ACTIVE || (g.m.tag[n - P] & FL) != CELL_ACTIVE;
        if (kind == K_BODY) {
          const int k1 = g.m.bid[n];
          atomicOr(&s_bm[k1 >> 5], 1u << (k1 & 31));
          kb = kb == -1 || kb == k1 ? k1 : -2;
        }
      }
    }
    const bool act = (freeM | bodyM) != 0;
    const unsigned half = 0xffffffffu >> (32 - ha), fullM = H == 2 ? (half | (half << 16)) : half;
    const bool wgen = __any_sync(0xffffffffu, gen);
    const bool wmask = __any_sync(0xffffffffu, act && freeM != fullM);
    auto body_at = [&](int a, int h, int pit) {
      return kb >= 0 ? kb : g.m.bid[base + (long long)(j0 + row_of(a, h)) * pit + i];
    };

    // p at row a, half h of this thread: its element and, next to a half's end, the halo
    // slot of the neighbouring half
    auto put_p = [&](int a, int h, T val) {
      Pt[(p0 + a * PITCH) * H + h] = val;
      if (a == 0) {
        if (h > 0) Pt[plast * H + h - 1] = val;
        else if (strip > 0) Pt[(plast - pw) * H + H - 1] = val;
      }
      if (a == ha - 1) {
        if (h < H - 1) Pt[(p0 - PITCH) * H + h + 1] = val;
        else if (strip < ns - 1) Pt[(p0 - PITCH + pw) * H] = val;
      }
    };

    // ---- state of the own nodes (q passes through x's place on its way to registers)
    V q[REG ? ROWS : 1];
    auto fetch = [&](int field) {
      if (!on) return;
#pragma unroll 1
      for (int k = 0; k < H * ha; ++k) {
        const int h = k >= ha ? 1 : 0, a = k - h * ha;
        T val = T(0);
        if ((freeM >> (16 * h + a)) & 1u)
          val = reinterpret_cast<const T*>(rec + base + (long long)(j0 + row_of(a, h)) * P + i)[field];
        if (field == 2) { if (val != T(0)) put_p(a, h, val); }
        else if (field == 1) reinterpret_cast<T*>(R2)[(a * RNT + tid) * H + h] = val;
        else Xt[(a * RNT + tid) * H + h] = val;
      }
    };
    fetch(3);
#pragma unroll UNR
    for (int a = 0; a < (REG ? ROWS : ha); ++a) {
      V t = V(0);
      if (a < ha && on) t = X2[a * RNT + tid];
      if (REG) q[a] = t;
      else if (on) Q2[a * RNT + tid] = t;
    }
    fetch(0);
    fetch(1);
    fetch(2);

    // ---- weights of the block's operator rows: per pair of neighbouring nodes, the sum of
    // the (one or two) element entries, added in FP64 and rounded once
    if (REG && I.gen) {
      const double* const K = g.m.K64;
      const long long pl = g.m.Vtot;
      const int cols = w + 1, per = cols * (ha + 1);
      for (int e = tid; e < ns * H * per; e += RNT) {
        const int sg = e / per, a = (e - sg * per) / cols - 1, c = e - sg * per - (a + 1) * cols - 1;
        const int ii = i0 + c, jj = j0 + sg * ha + a;
        double wE = 0.0, wN = 0.0, wD = 0.0, wA = 0.0;
        if (ii >= 0 && jj >= 0 && ii <= nx && jj <= ny) {
          const long long n = base + (long long)jj * P + ii;
          if (ii < nx && jj < ny) {
            wE = K[n];
            wN = K[2 * pl + n];
            wD = K[pl + n];
            wA = K[4 * pl + n];
          }
          if (ii < nx && jj > 0) wE += K[5 * pl + n - P];
          if (ii > 0 && jj < ny) wN += K[3 * pl + n - 1];
        }
        T* const W = reinterpret_cast<T*>(W4) + ((a + 1) * PITCH + (sg / H) * pw + c + 1) * H + sg % H;
        W[0] = (T)wE;
        W[WPL * H] = (T)wN;
        W[2 * WPL * H] = (T)wD;
        W[3 * WPL * H] = (T)wA;
      }
    }

    // ---- halo nodes: the ring of the block
    const int n_halo = 2 * pw + 2 * bh;
    bool near = bodyM != 0;                // body nodes here or next to the block
    T qh[HITER];
#pragma unroll
    for (int k = 0; k < HITER; ++k) {
      const int h = tid + k * RNT;
      qh[k] = T(0);
      if (h < n_halo) {
        int row, c;
        if (h < pw) { row = -1; c = h - 1; }
        else if (h < 2 * pw) { row = bh; c = h - pw - 1; }
        else if (h < 2 * pw + bh) { row = h - 2 * pw; c = -1; }
        else { row = h - 2 * pw - bh; c = w; }
        const int hi = i0 + c, hj = j0 + row;
        int code = -1;
        unsigned pl = 0;
        T rh = T(0);
        if (hi >= 0 && hj >= 0 && hi <= nx && hj <= ny) {
          const long long off = (long long)hj * P + hi;
          const int kind = g.m.tag[base + off] & KIND_MASK;
          // half strip and row in it; rows -1 and bh are the outer slots of the first and last one
          int sg = row < 0 ? 0 : row / ha, a = row < 0 ? -1 : row - sg * ha;
          if (row == bh) { sg = ns * H - 1; a = ha; }
          auto place = [&](int s2, int a2) { return (unsigned)(((a2 + 1) * PITCH + (s2 / H) * pw + c + 1) * H + s2 % H); };
          pl = place(sg, a);
          unsigned second = 0xffffu;
          if (row >= 0 && row < bh) {
            if (a == 0 && sg > 0) second = place(sg - 1, ha);
            else if (a == ha - 1 && sg < ns * H - 1) second = place(sg + 1, -1);
          }
          if (kind == K_FREE) {
            const State4<T> o = rec[base + off];
            code = (int)off;
            rh = o.r;
            qh[k] = o.q;
            Pt[pl] = o.p;
          } else if (kind == K_BODY) {
            code = -2 - g.m.bid[base + off];
          }
          pl |= second << 16;
        }
        if (code < -1) near = true;
        hw[h] = code;
        hp[h] = pl;
        hr[h] = rh;
      }
    }

    // ---- nodes at the block's edges that other blocks see
    const bool see_l = i0 > 0, see_r = i0 + w <= nx, see_t = j0 > 0, see_b = j0 + bh <= ny;
    for (int e = tid; e < 2 * w + 2 * bh; e += RNT) {
      int row, c;
      bool see;
      if (e < w) { row = 0; c = e; see = see_t; }
      else if (e < 2 * w) { row = bh - 1; c = e - w; see = see_b; }
      else if (e < 2 * w + bh) { row = e - 2 * w; c = 0; see = see_l; }
      else { row = e - 2 * w - bh; c = w - 1; see = see_r; }
      ew[e] = see && i0 + c <= nx && j0 + row <= ny ? (j0 + row) * P + i0 + c : -1;
    }

    // ---- body values and scalars; the first iteration starts from the state's alpha, beta
    {
      const T al = (T)S->alpha, be = (T)S->beta;
      if (tid < nb) {
        const int gb = body0 + tid;
        const T xb = g.sb[gb], rb = g.sb[g.B + gb], pb = g.sb[2 * g.B + gb], qb = g.sb[3 * g.B + gb];
        const T rn = rb - al * qb;
        const T pn = rn + be * pb;
        s_b[0][tid] = xb + al * pb;
        s_b[1][tid] = rn;
        s_b[2][tid] = pn;
        s_pb[tid] = fixed ? T(0) : pn;
      }
      if (tid < 6) s_kr[tid] = rect_of<T>(Vg)[tid];
      if (tid == 0) {
        s_alpha = al;
        s_beta = be;
        s_stop = 0;
        s_root.gamma_start = S->gamma_start;
        s_root.thr_rel = S->thr_rel;
        s_root.thr_abs2 = S->thr_abs2;
        s_root.thr = fmax(S->thr_rel * S->gamma_start, S->thr_abs2);   // (a first iteration sets it)
        s_root.iters = S->iters;
        s_root.inner = S->inner_iters;
        s_root.k_max = g.prm->k_max;
      }
    }
    unsigned ep = g.epoch[v] + 1;
    // the thread's places in qe
    const bool ecol = act && ((col == 0 && see_l) || (col == w - 1 && see_r));
    const int ecol_at = 2 * w + (col == 0 ? 0 : bh) + strip * H * ha;
    const bool etop = act && strip == 0 && see_t, ebot = act && strip == ns - 1 && see_b;

    // ---- every block of the variant has started and has told which bodies it holds
    const bool near_body = __syncthreads_or(near);
    const u64 bm = (u64)s_bm[0] | ((u64)s_bm[1] << 32);
    if (tid == 0) {
      st_word(&g.pbm[R.part0 + part], bm);
      atom_add_acq_rel_gpu(&g.join[v], 1);
      int tries = 0;
      while (*(volatile int*)&g.join[v] < R.parts) {
        __nanosleep(500);
        if (++tries > JOIN_LIMIT || *(volatile int*)g.err) {
          atomicExch(g.err, 1);
          s_abort = 1;
          break;
        }
      }
      __threadfence();
    }
    __syncthreads();
    if (s_abort) return;
    // the first block sums every block's partial sums; of a body, only those that hold its nodes
    int* const blist = g.blist + (long long)R.part0 * (g.qs - 4);
    if (part == 0) {
      for (int k = warp; k < nbu; k += RWARPS) {
        int n = 0;
        for (int p1 = 0; p1 < R.parts; p1 += 32) {
          const bool has = p1 + lane < R.parts && ((ld_word(&g.pbm[R.part0 + p1 + lane]) >> k) & 1ull);
          const unsigned m = __ballot_sync(0xffffffffu, has);
          if (has) blist[(long long)k * R.parts + n + __popc(m & ((1u << lane) - 1u))] = p1 + lane;
          n += __popc(m);
        }
        if (lane == 0) s_cnt[k] = n;
      }
      __syncthreads();
      if (tid == 0) {
        int at = 0;
        for (int k = 0; k < nbu; ++k) {
          s_first[k] = at + s_cnt[k] <= LISTMAX && R.parts < 65536 ? at : -1;
          at += s_cnt[k];
        }
      }
      __syncthreads();
      for (int k = warp; k < nbu; k += RWARPS)
        if (s_first[k] >= 0)
          for (int e = lane; e < s_cnt[k]; e += 32) s_list[s_first[k] + e] = (unsigned short)blist[(long long)k * R.parts + e];
    }
    if (tid == 0) {
      sh.words = words + base * (2 * WPV);   // (from the variant's first node on)
      sh.pw_var = g.pw + (long long)R.part0 * g.qs * 2;
      sh.bc = g.bc + (long long)v * 2 * (g.qs - 1) * WPV;
      sh.blist = blist;
      sh.S = S;
      sh.base = base;
      sh.P = P;
      sh.w = w;
      sh.bh = bh;
      sh.i0 = i0;
      sh.j0 = j0;
      sh.nx = nx;
      sh.ny = ny;
      sh.nbu = nbu;
      sh.parts = R.parts;
      sh.see = near_body ? 16 : 0;
    }
    // the thread's part of the block in one word
    const int fl = (act ? 1 : 0) | (wgen ? 2 : 0) | (wmask ? 4 : 0) | (ecol ? 8 : 0) | (etop ? 16 : 0) | (ebot ? 32 : 0) |
                   (strip > 0 ? 64 : 0) | (strip < ns - 1 ? 128 : 0) | ((kb + 2) << 8) |
                   (__any_sync(0xffffffffu, kb >= 0) ? 0x10000 : 0);
    __syncthreads();

    for (int it = 0;; ++it, ++ep) {
      const bool act = fl & 1, wgen = fl & 2, etop = fl & 16, ebot = fl & 32, above = fl & 64, below = fl & 128;
      const int kb = ((fl >> 8) & 0xff) - 2;
      // (hidden from the compiler, which would otherwise make two copies of the unrolled loops)
      int mask = fl & 4, ec = fl & 8, bodies = fl & 0x10000;
      asm volatile("" : "+r"(mask), "+r"(ec), "+r"(bodies));
      const int pw = sh.w + 2, n_edge = 2 * sh.w + 2 * sh.bh, n_halo = n_edge + 4;
      u64* const words_v = sh.words;
      auto body_of = [&](int a, int h) {
        return kb >= 0 ? kb : g.m.bid[sh.base + (long long)(sh.j0 + (strip * H + h) * ha + a) * sh.P + i];
      };

      // ---- r -= alpha q, x += alpha p, p = r + beta p, on the block and its halo
      const T al = s_alpha, be = s_beta;
      if (act) {
        const V nal = X::bcast(-al), val = X::bcast(al), vbe = X::bcast(be);
        const T pbody = kb >= 0 ? s_pb[kb] : T(0);
        V pn = V(0);
        T c[H];
#pragma unroll UNR
        for (int a = 0; a < (REG ? ROWS : ha); ++a) {
          if (a < ha) {
            const V po = P2[p0 + a * PITCH];
            const V rn = vfma(nal, REG ? q[REG ? a : 0] : Q2[a * RNT + tid], R2[a * RNT + tid]);
            R2[a * RNT + tid] = rn;
            X2[a * RNT + tid] = vfma(val, po, X2[a * RNT + tid]);
            pn = vfma(vbe, po, rn);
            X::split(pn, c);
            if (bodies) {
#pragma unroll
              for (int h = 0; h < H; ++h)
                if (bodyM & (1u << (16 * h + a))) c[h] = pbody;
              pn = X::make(c);
            }
            P2[p0 + a * PITCH] = pn;
            if (a == 0) {
              if (H == 2) Pt[plast * H] = c[H - 1];
              if (above) Pt[(plast - pw) * H + H - 1] = c[0];
            }
          }
        }
        // the last row of each half
        if (H == 2) Pt[(p0 - PITCH) * H + 1] = c[0];
        if (below) Pt[(p0 - PITCH + pw) * H] = c[H - 1];
        if (kb == -2) {                    // nodes of several bodies
#pragma unroll 1
          for (unsigned b = bodyM; b; b &= b - 1) {
            const int bit = __ffs(b) - 1, h = bit >> 4, a = bit & 15;
            put_p(a, h, s_pb[body_of(a, h)]);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < HITER; ++k) {
        const int h = tid + k * RNT;
        if (h < n_halo) {
          const int code = hw[h];
          if (code != -1) {
            const unsigned pl = hp[h];
            T pn;
            if (code >= 0) {
              const T rn = hr[h] - al * qh[k];
              hr[h] = rn;
              pn = rn + be * Pt[pl & 0xffffu];
            } else {
              pn = s_pb[-2 - code];
            }
            Pt[pl & 0xffffu] = pn;
            if ((pl >> 16) != 0xffffu) Pt[pl >> 16] = pn;
          }
        }
      }
      __syncthreads();

      // ---- q = A p and the dot products
      BodySum<T> yb;                       // the thread's rows of A p at the nodes of body kb
      if (act) {
        V yl = V(0);                       // q of the last row
        // a finished row: mask the rows of other nodes, edges
        auto finish = [&](int a, V y) {
          T c[H];
          X::split(y, c);
          if (mask) {
#pragma unroll
            for (int h = 0; h < H; ++h) {
              const unsigned bit = 1u << (16 * h + a);
              if (bodyM & bit) {
                yb.add(c[h]);
                if (kb == -2) Xt[(a * RNT + tid) * H + h] = c[h];   // (a body node has no x)
              }
              if (!(freeM & bit)) c[h] = T(0);
            }
            y = X::make(c);
          }
          if (REG) q[REG ? a : 0] = y;
          else Q2[a * RNT + tid] = y;
          if (ec) {
#pragma unroll
            for (int h = 0; h < H; ++h) qe[ecol_at + h * ha + a] = c[h];
          }
          if (a == 0 && etop) qe[col] = c[0];
          yl = y;
        };
        if (!wgen) {
          // four undisplaced active cells around every node: with S the second difference
          // along the row and w that along the column,
          //   y = 2 K01 S_j + K02 (S_{j-1} + S_{j+1}) + 2 (K02 + K03) w
          const T* const kr = s_kr;
          const V c1 = X::bcast(T(2) * kr[0]), c2 = X::bcast(T(2) * (kr[1] + kr[2])), c3 = X::bcast(kr[1]);
          auto row = [&](int a, V& C) {
            const V* p = P2 + p0 + a * PITCH;
            C = p[0];
            return vadd(vsub(p[-1], C), vsub(p[1], C));
          };
          V Cm, C0, C1;
          V Sm = row(-1, Cm), S0 = row(0, C0), S1;
          V vm = vsub(C0, Cm);
#pragma unroll UNR
          for (int a = 0; a < (REG ? ROWS : ha); ++a) {
            if (a < ha) {
              S1 = row(a + 1, C1);
              const V vn = vsub(C1, C0);
              finish(a, vfma(c3, vadd(Sm, S1), vfma(c2, vsub(vn, vm), vmul(c1, S0))));
              Sm = S0; S0 = S1; C0 = C1; vm = vn;
            }
          }
        } else if constexpr (REG) {
          // the weights of the block's shared memory
          const V* const W = W4 + p0;      // row a = 0 of the weight planes: the place of p's row 0
          const V* p = P2 + p0;
          V sw = p[-PITCH - 1], so = p[-PITCH], se = p[-PITCH + 1];
          V we = p[-1], ce = p[0], ea = p[1];
          V Nm = W[WPL - PITCH];
#pragma unroll GUNR
          for (int a = 0; a < X::GROWS1 - 1; ++a) {
            if (a < ha) {
              const V nw = p[(a + 1) * PITCH - 1], no = p[(a + 1) * PITCH], ne = p[(a + 1) * PITCH + 1];
              const V N = W[WPL + a * PITCH];
              V y = vmul(W[a * PITCH], vsub(ea, ce));
              y = vfma(W[a * PITCH - 1], vsub(we, ce), y);
              y = vfma(N, vsub(no, ce), y);
              y = vfma(Nm, vsub(so, ce), y);
              y = vfma(W[2 * WPL + a * PITCH], vsub(ne, ce), y);
              y = vfma(W[2 * WPL + (a - 1) * PITCH - 1], vsub(sw, ce), y);
              y = vfma(W[3 * WPL + a * PITCH - 1], vsub(nw, ce), y);
              y = vfma(W[3 * WPL + (a - 1) * PITCH], vsub(se, ce), y);
              finish(a, y);
              Nm = N;
              sw = we; so = ce; se = ea;
              we = nw; ce = no; ea = ne;
            }
          }
        } else {
          // FP64: the element coefficients from global memory (the arithmetic hides the loads)
          const double* const K = g.m.K64;
          const long long pl = g.m.Vtot;
          const bool has_l = i > 0;
          const int jb = sh.j0 + strip * H * ha, ny = sh.ny, pit = sh.P;
          long long n = sh.base + (long long)jb * pit + i;
          // cells below the node: K12 K02 K23 of the left one, K03 K13 K23 of the right one
          T l1 = T(0), l3 = T(0), l5 = T(0), m2 = T(0), m4 = T(0), m5 = T(0);
          if (jb > 0 && jb <= ny) {
            const long long c = n - pit;
            if (has_l) { l1 = K[pl + c - 1]; l3 = K[3 * pl + c - 1]; l5 = K[5 * pl + c - 1]; }
            m2 = K[2 * pl + c]; m4 = K[4 * pl + c]; m5 = K[5 * pl + c];
          }
          const T* pr = Pt + p0;
          T sw = pr[-PITCH - 1], se = pr[-PITCH + 1], we = pr[-1], ce = pr[0], ea = pr[1];
          T dS = pr[-PITCH] - ce;
#pragma unroll 1
          for (int a = 0; a < ha && jb + a <= ny; ++a, n += pit) {
            T b0 = T(0), b1 = T(0), b3 = T(0), b4 = T(0), b5 = T(0);
            if (has_l) {
              b0 = K[n - 1]; b1 = K[pl + n - 1]; b3 = K[3 * pl + n - 1]; b4 = K[4 * pl + n - 1]; b5 = K[5 * pl + n - 1];
            }
            const T a0 = K[n], a1 = K[pl + n], a2 = K[2 * pl + n], a4 = K[4 * pl + n], a5 = K[5 * pl + n];
            pr += PITCH;
            const T nw = pr[-1], no = pr[0], ne = pr[1];
            const T dE = ea - ce, dW = we - ce, dN = no - ce;
            T y = a0 * dE + a1 * (ne - ce) + a2 * dN;
            y += b0 * dW + b3 * dN + b4 * (nw - ce);
            y += l1 * (sw - ce) + l3 * dS + l5 * dW;
            y += m2 * dS + m4 * (se - ce) + m5 * dE;
            finish(a, y);
            l1 = b1; l3 = b3; l5 = b5;
            m2 = a2; m4 = a4; m5 = a5;
            sw = we; se = ea; dS = -dN;
            we = nw; ce = no; ea = ne;
          }
        }
        if (ebot) {
          T c[H];
          X::split(yl, c);
          qe[w + col] = c[H - 1];
        }
      }

      // ---- dot products: threads, warps, then the CTA
      Dots<T> d;
      d.zero();
      if (act) {
#pragma unroll UNR
        for (int a = 0; a < (REG ? ROWS : ha); ++a) {
          if (a < ha) {
            d.add_row(R2[a * RNT + tid], P2[p0 + a * PITCH], REG ? q[REG ? a : 0] : Q2[a * RNT + tid]);
          }
        }
      }
      {
        const double s = d.warp_sums(lane);
        if (lane < 4) s_red[warp][lane] = s;
        if (sh.nbu > 0) {
          for (u64 b = (u64)s_bm[0] | ((u64)s_bm[1] << 32); b; b &= b - 1) {
            const int k = __ffsll((long long)b) - 1;
            double y = 0.0;
            if (__any_sync(0xffffffffu, kb == k || kb == -2)) {
              BodySum<T> b = kb == k ? yb : BodySum<T>();
              if (kb == -2) {
#pragma unroll 1
                for (unsigned c = bodyM; c; c &= c - 1) {
                  const int bit = __ffs(c) - 1, h = bit >> 4, a = bit & 15;
                  if (body_of(a, h) == k) b.add(Xt[(a * RNT + tid) * H + h]);
                }
              }
              y = b.warp_sum();
            }
            if (lane == 0) s_yb[warp][k] = y;
          }
        }
      }
      __syncthreads();

      // ---- publish q at the edges that other blocks see, and the block's sums
      {
        const bool drop = g.test_drop && part == 0 && it == 0;   // test hook: the waits give up
        const int parts = sh.parts;
        u64* const mine = sh.pw_var + (ep & 1) * g.pw_half + (long long)part * 2;
        if (warp == 0) {
          double s = (lane & 7) < RWARPS ? s_red[lane & 7][lane >> 3] : 0.0;
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if ((lane & 7) == 0 && !drop) put_double(mine + (long long)(lane >> 3) * parts * 2, s, ep);
        } else if (tid - 32 < sh.nbu && ((s_bm[(tid - 32) >> 5] >> ((tid - 32) & 31)) & 1u)) {
          const int k = tid - 32;
          double s = 0.0;
          for (int u = 0; u < RWARPS; ++u) s += s_yb[u][k];
          if (!drop) put_double(mine + (long long)(4 + k) * parts * 2, s, ep);
        }
#pragma unroll
        for (int k = 0; k < HITER; ++k) {
          // (from the last warp down: the first one sums)
          const int e = RNT - 1 - tid + k * RNT;
          if (e < n_edge && ew[e] >= 0) QWord<T>::put(QWord<T>::at(words_v, ew[e], ep), qe[e], ep);
        }
      }

      // ---- the neighbours' q: asked for now, looked at when alpha and beta are there
      QWord<T> hq[HITER];
      int hc[HITER];
#pragma unroll
      for (int k = 0; k < HITER; ++k) {
        const int h = tid + k * RNT;
        hc[k] = h < n_halo ? hw[h] : -1;
        if (hc[k] >= 0) hq[k].load(QWord<T>::at(words_v, hc[k], ep));
      }
      bool gave_up = false;
      auto give_up = [&](int& tries) {
        return ++tries > g.poll_limit || ((tries & 255) == 0 && *(volatile int*)g.err);
      };
      u64* const bc = sh.bc + (ep & 1) * (long long)(g.qs - 1) * WPV;
      const int nbu = sh.nbu, parts = sh.parts;
      if (part == 0) {
        // ---- first block: all partial sums, in block order, then the scalars
        // (a dot product per warp; of the bodies, which few blocks hold, four per warp)
        const u64* const now = sh.pw_var + (ep & 1) * g.pw_half;
        auto wait_sum = [&](const u64* at) {
          u64 wa, wb;
          ld_word2(at, wa, wb);
          int tries = 0;
          while (!fresh(wa, wb, ep)) {
            if (give_up(tries)) {
              gave_up = true;
              break;
            }
            ld_word2(at, wa, wb);
          }
          return word_double(wa, wb);
        };
        if (warp < 4) {
          const u64* const all = now + (long long)warp * parts * 2;
          double s = 0.0;
          for (int pp = lane; pp < parts; pp += 128) {
            u64 wa[4], wb[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (pp + 32 * u < parts) ld_word2(all + 2 * (pp + 32 * u), wa[u], wb[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (pp + 32 * u < parts)
                s += fresh(wa[u], wb[u], ep) ? word_double(wa[u], wb[u]) : wait_sum(all + 2 * (pp + 32 * u));
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (lane == 0) s_tot[warp] = s;
        } else {
          for (int k0 = 4 * (warp - 4); k0 < nbu; k0 += 4 * (RWARPS - 4)) {
            const int k = k0 + (lane >> 3), n = k < nbu ? s_cnt[k] : 0, first = k < nbu ? s_first[k] : 0;
            const u64* const all = now + (long long)(4 + k) * parts * 2;
            double s = 0.0;
            for (int e = lane & 7; e < n; e += 8)
              s += wait_sum(all + 2 * (first >= 0 ? s_list[first + e] : sh.blist[(long long)k * parts + e]));
            __syncwarp();
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((lane & 7) == 0 && k < nbu) s_tot[4 + k] = s;
          }
        }
        if (gave_up) {
          atomicExch(g.err, 1);
          s_abort = 1;
        }
        __syncthreads();
        if (warp == 0 && !s_abort) {
          // the bodies' part of the dot products: eight lanes per dot product
          const int dot = lane >> 3;
          double c = 0.0;
          for (int k = lane & 7; k < nbu; k += 8) {
            const T qn = (T)s_tot[4 + k], rn = s_b[1][k], pn = s_b[2][k];
            if (dot == 0) s_b[3][k] = qn;
            c += (double)(dot == 1 ? pn : dot == 3 ? qn : rn) * (double)(dot == 0 ? rn : qn);
          }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1)
            if (nbu > o) c += __shfl_xor_sync(0xffffffffu, c, o);   // (lanes past the bodies hold zeros)
          c = s_tot[dot] + c;
          const double ga = __shfl_sync(0xffffffffu, c, 0), pi = __shfl_sync(0xffffffffu, c, 8),
                       rho = __shfl_sync(0xffffffffu, c, 16), mu = __shfl_sync(0xffffffffu, c, 24);
          __syncwarp();
          double nal = 0.0, nbe = 0.0;
          int stop = 0;                    // 1: residual check, 2: breakdown, 3: pause (the launch's iteration limit)
          if (lane == 0) {
            // (FP64 arithmetic takes 64 cycles an instruction here, so comparisons of doubles of
            // known sign go through their bits)
            const long long gab = __double_as_longlong(ga), pib = __double_as_longlong(pi);
            constexpr long long INF = 0x7ff0000000000000ll;
            bool capped = false;
            const long long iters = s_root.iters + 1, inner = s_root.inner + 1;
            s_root.iters = iters;
            s_root.inner = inner;
            if (inner == 1) {
              s_root.gamma_start = ga;
              s_root.thr = fmax(s_root.thr_rel * ga, s_root.thr_abs2);
            }
            if ((gab & INF) == INF || pib <= 0 || pib >= INF) {      // r.r not finite, or p.Ap not positive and finite
              stop = ga == 0.0 ? 1 : 2;
            } else if (gab <= __double_as_longlong(s_root.thr)) {    // (both are non-negative)
              stop = 1;
            } else if (iters >= s_root.k_max) {
              stop = 1;
              capped = true;
            } else {
              // alpha = r.r / p.q, beta = (r.r - 2 alpha r.q + alpha^2 q.q) / r.r
              const double inv = 1.0 / pi;
              nal = ga * inv;
              const double b = fma(fma(nal, mu, -2.0 * rho), inv, 1.0);
              nbe = __double_as_longlong(b) > 0 ? b : 0.0;
              if (it + 1 >= g.max_it) stop = 3;
            }
            if (stop) {
              VarState* const S = sh.S;
              S->iters = iters;
              S->inner_iters = inner;
              S->gamma_start = s_root.gamma_start;
              S->gamma = ga;
              S->pi = pi;
              S->rho = rho;
              S->mu = mu;
              if (stop == 1) {
                if (capped) S->capped = 1;
                S->phase = PH_RESID;
              } else if (stop == 2) {
                S->status = PF_EBREAKDOWN;
                S->phase = PH_DONE;
                atomicAdd(g.n_done, 1);
              } else {
                S->alpha = nal;
                S->beta = nbe;
              }
              g.epoch[S - g.st] = ep;
            }
          }
          stop = __shfl_sync(0xffffffffu, stop, 0);
          const T alT = (T)__shfl_sync(0xffffffffu, nal, 0), beT = (T)__shfl_sync(0xffffffffu, nbe, 0);
          if (lane == 0) {
            QWord<T>::put(bc, alT, ep);
            QWord<T>::put(bc + WPV, beT, ep);
            QWord<T>::put(bc + 2 * WPV, (T)stop, ep);
            s_alpha = alT;
            s_beta = beT;
            s_stop = stop;
          }
          for (int k = lane; k < nbu; k += 32) {
            const T pb = s_b[2][k];
            const T rn = s_b[1][k] - alT * s_b[3][k];
            const T pn = rn + beT * pb;
            QWord<T>::put(bc + (3 + k) * WPV, pn, ep);
            if (stop == 0) {               // (else the state stays that of this iteration)
              s_b[0][k] = s_b[0][k] + alT * pb;
              s_b[1][k] = rn;
              s_b[2][k] = pn;
              s_pb[k] = pn;
            }
          }
        }
      } else if (warp == 0) {
        // ---- the others take alpha, beta and the body values (bodies only if there are any here)
        const int n = 3 + ((sh.see & 16) ? nbu : 0);
        for (int e = lane; e < n; e += 32) {
          QWord<T> w0;
          int tries = 0;
          w0.load(bc + e * WPV);
          while (!w0.ready(ep)) {
            if (give_up(tries)) {
              gave_up = true;
              break;
            }
            w0.load(bc + e * WPV);
          }
          const T val = w0.value();
          if (e == 0) s_alpha = val;
          else if (e == 1) s_beta = val;
          else if (e == 2) s_stop = (int)val;
          else s_pb[e - 3] = val;
        }
        if (gave_up) {
          atomicExch(g.err, 1);
          s_abort = 1;
        }
      }
      __syncthreads();
      if (s_abort) return;
      if (s_stop) break;
#pragma unroll
      for (int k = 0; k < HITER; ++k) {
        if (hc[k] >= 0) {
          const u64* const at = QWord<T>::at(words_v, hc[k], ep);
          int tries = 0;
          while (!hq[k].ready(ep)) {
            if (give_up(tries)) {
              gave_up = true;
              break;
            }
            hq[k].load(at);
          }
          qh[k] = hq[k].value();
        }
      }
      if (gave_up) {                       // seen by the block at the end of the next iteration's waits
        atomicExch(g.err, 1);
        s_abort = 1;
      }
    }

    // ---- state back to the records (every block has read its halo long before)
    int pit = P;
    asm volatile("" : "+r"(pit));
    auto store = [&](int field) {
#pragma unroll 1
      for (int k = 0; k < H * ha; ++k) {
        const int h = k >= ha ? 1 : 0, a = k - h * ha;
        if ((freeM >> (16 * h + a)) & 1u)
          reinterpret_cast<T*>(rec + base + (long long)(j0 + row_of(a, h)) * pit + i)[field] =
              field == 2 ? Pt[(p0 + a * PITCH) * H + h]
                         : field == 1 ? reinterpret_cast<const T*>(R2)[(a * RNT + tid) * H + h] : Xt[(a * RNT + tid) * H + h];
      }
    };
    store(0);
    store(1);
    store(2);
#pragma unroll UNR
    for (int a = 0; a < (REG ? ROWS : ha); ++a)
      if (a < ha) X2[a * RNT + tid] = REG ? q[REG ? a : 0] : Q2[a * RNT + tid];
    store(3);
    if (part == 0 && tid < nbu) {
      const int gb = body0 + tid;
      g.sb[gb] = s_b[0][tid];
      g.sb[g.B + gb] = s_b[1][tid];
      g.sb[2 * g.B + gb] = s_b[2][tid];
      g.sb[3 * g.B + gb] = s_b[3][tid];
    }
  }
}

// ---------------------------------------------------------------- host side
template <typename T>
const void* kernel() { return (const void*)k_cg_resident<T>; }

// Blocks of one variant.  The columns are cut into nbx equal parts; each column part into
// blocks of ns strips from the top down.  `rows`: rows of a half strip at most in blocks of
// undisplaced cells only, `grows` in the others (stored coefficients: more shared memory in
// FP32, more arithmetic in FP64), so that the blocks of a variant take about the same time.
struct Cutter {
  int W, R, H;                         // nodes per row, rows, halves of a strip
  int tx = 0, ty = 0;                  // 64 x 16 tiles
  std::vector<uint8_t> stored;         // [ty][tx] some operator row needs stored coefficients
  std::vector<std::vector<int>> ends;  // [column parts][part][ty] where plain runs end, made when first asked for

  // rows to which tile rows of the column parts of width w without stored coefficients run on: 0
  // where the tile row has stored ones.  (Kept: every candidate of the search asks for the same.)
  const int* runs(int nbx, int w) {
    if ((int)ends.size() <= nbx) ends.resize(nbx + 1);
    std::vector<int>& e = ends[nbx];
    if (e.empty()) {
      e.assign((size_t)nbx * ty, 0);
      for (int p = 0; p < nbx; ++p) {
        const int c0 = p * w / CTX, c1 = std::min(W - 1, (p + 1) * w - 1) / CTX;
        int* const to = e.data() + (size_t)p * ty;
        for (int t = ty - 1; t >= 0; --t) {
          bool st = false;
          for (int c = c0; c <= c1 && !st; ++c) st = stored[(size_t)t * tx + c] != 0;
          if (!st) to[t] = t + 1 < ty && to[t + 1] ? to[t + 1] : std::min(R, (t + 1) * CTY);
        }
      }
    }
    return e.data();
  }
  // Blocks of `threads` threads with at most that many rows of a half strip: no cut has fewer.  A
  // block without stored rows holds no node of a stored tile.
  double least(int rows, int grows, int threads) const {
    double st = 0.0;
    for (int t = 0; t < ty; ++t)
      for (int c = 0; c < tx; ++c)
        if (stored[(size_t)t * tx + c]) st += (double)std::min(CTX, W - c * CTX) * std::min(CTY, R - t * CTY);
    return (st / std::min(rows, grows) + ((double)W * R - st) / std::max(rows, grows)) / ((double)threads * H);
  }
  struct Part { int i0, w, ns, unit, rows, grows; };

  // Blocks of a column part from row j down, each as high as it may be: their number, and their
  // rows in `slots`.  Where a plain run ends in a low block, that may join the stored block below,
  // and the last block of a stored run may stop with it or run on.  Of these two ways the one
  // with fewer blocks is taken, `forks` times per column part (once: 16 grids of 257x129 nodes
  // with an airfoil each need 256 blocks in place of 320, so that all of them fit the chip; more
  // often costs host time that doubles with every fork and gains under 2 % of the blocks).
  int down(const Part& c, const int* plain_to, int j, int forks, double& slots, std::vector<RItem>* out) const {
    int n = 0;
    while (j < R) {
      const int end = plain_to[j / CTY], left = (R - j + c.unit - 1) / c.unit;
      const int full = std::max(2, std::min(c.grows, left));
      int ha = 0, gen = 1;
      auto fewer = [&](int h1, int h2) {         // blocks below a block of h1 rows against one of h2
        double s = 0.0;
        return down(c, plain_to, j + c.unit * h1, forks, s, nullptr) < down(c, plain_to, j + c.unit * h2, forks, s, nullptr);
      };
      if (end) {
        const int fit = end == R ? left : (end - j) / c.unit;
        ha = std::min(fit, c.rows);
        if (fit > ha && fit - ha < 2 && ha > 3) ha = fit - 2;       // leave no single row
        if (end == R) ha = std::max(ha, 2);
        if (ha >= 2) gen = 0;
        if (!gen && end < R && fit <= c.rows && forks > 0) {
          --forks;
          gen = fewer(full, ha);
        }
      }
      if (gen) {
        ha = full;
        int t = j / CTY;
        while (t < ty && plain_to[t]) ++t;                  // (the plain rest that joined)
        while (t < ty && !plain_to[t]) ++t;
        const int need = std::max(2, (std::min(R, t * CTY) - j + c.unit - 1) / c.unit);
        if (need < full && forks > 0) {
          --forks;
          if (!fewer(full, need)) ha = need;
        }
      }
      if (out) out->push_back(RItem{0, 0, c.i0, c.w, j, c.ns, ha, gen});
      ++n;
      slots += ha;
      j += c.unit * ha;
    }
    return n;
  }

  // column part p: appends (j0, ha, gen); false if the exchange lists would overflow
  bool column(int p, const int* ends_w, int w, int ns, int rows, int grows, std::vector<RItem>* out, int& parts, double& slots) const {
    const int unit = ns * H, fit = (HMAX - 2 * (w + 2)) / (2 * unit);
    if (fit < 2) return false;
    const Part c{p * w, w, ns, unit, std::min(rows, fit), std::min(grows, fit)};
    parts += down(c, ends_w + (size_t)p * ty, 0, 1, slots, out);
    return true;
  }

  // the cut with the fewest blocks (ties: fewer rows in all)
  bool best(int rows, int grows, int threads, std::vector<RItem>& out) {
    double best_cost = 1e300;
    int bn = 0, bw = 0, bns = 0;
    for (int nbx = (W + threads - 1) / threads; nbx <= W; ++nbx) {
      const int w = (W + nbx - 1) / nbx;
      if (w < 32 && nbx > 1) break;
      if ((nbx - 1) * w >= W) continue;                // the last column part would be empty
      const int most = std::min(NSMAX, threads / w);
      const int* const e = runs(nbx, w);
      for (int ns = most; ns >= std::max(1, most - 1); --ns) {
        if (w * ns < threads / 2 && W >= threads) continue;   // half the threads idle
        int parts = 0;
        double slots = 0.0;
        bool ok = true;
        for (int bx = 0; bx < nbx && ok && parts < best_cost; ++bx) ok = column(bx, e, w, ns, rows, grows, nullptr, parts, slots);
        const double cost = parts + 0.01 * slots;
        if (ok && cost < best_cost) {
          best_cost = cost;
          bn = nbx;
          bw = w;
          bns = ns;
        }
      }
    }
    out.clear();
    if (bw == 0) return false;
    int parts = 0;
    double slots = 0.0;
    for (int p = 0; p < bn; ++p) column(p, runs(bn, bw), bw, bns, rows, grows, &out, parts, slots);
    return true;
  }
};

void free_plan(Batch& b, ResPlan& R) {
  for (void* p : {R.d_var, R.d_items, (void*)R.d_ctrl, (void*)R.d_epoch, (void*)R.d_pw, (void*)R.d_bc,
                  (void*)R.d_pbm, (void*)R.d_blist})
    if (p) dev_free(b, p);
  R = ResPlan{};
}

// Exchange numbers start again at 1: no word carries one.  (The q words lie in the state
// records, which every solve clears.)
void clear_exchange(Batch& b, ResPlan& R) {
  PF_CUDA(cudaMemsetAsync(R.d_epoch, 0, b.nv * sizeof(unsigned), b.stream));
  PF_CUDA(cudaMemsetAsync(R.d_pw, 0, 2 * R.pw_half * sizeof(u64), b.stream));
  PF_CUDA(cudaMemsetAsync(R.d_bc, 0, R.bc_words * sizeof(u64), b.stream));
  R.open = false;
}

}  // namespace

// Can this batch's CG run with its state on the chip, and how is it cut?  Made once per
// handle and precision (and again when the coordinates change: the cut follows the cells that
// need stored coefficients).  If every variant fits the chip at once, the blocks are cut for
// the shortest iteration; up to twice that, blocks are as large as a CTA holds and the variants
// queue.  Larger batches, and variants that need more blocks than there are resident CTAs,
// take the streaming kernel of solver.cu: it is then bound by bytes, no longer by latency.
static bool make_plan(Batch& b, int precision);

// ... and does it pay with `chunk` iterations a launch (0: as many as the inner solve takes)?  A
// launch carries the state from and to memory.  Time of the streaming kernel over that of this one,
// FP32, at chunks of 4, 6, 8, 12, 16: one 1900x951 grid 0.91, 1.07, 1.18, 1.36, 1.46; twenty of
// 400x200, which queue, 0.63, 0.76, 0.86, 0.98, 1.07.
bool resident_ready(Batch& b, int precision, int chunk) {
  ResPlan& R = b.res[precision];
  if (!R.made) make_plan(b, precision);
  if (!R.ok || (chunk > 0 && chunk < (R.queued ? 16 : 6))) return false;
  // after a solve that was broken off (a wait that gave up) the last numbers in use are not known
  if (R.open) clear_exchange(b, R);
  return true;
}

static bool make_plan(Batch& b, int precision) {
  ResPlan& R = b.res[precision];
  R.made = true;
  R.ok = false;
  const bool f64 = precision == PF_FP64;
  const int H = f64 ? VT<double>::H : VT<float>::H;
  const int rows = f64 ? VT<double>::ROWS : VT<float>::ROWS;
  const int grows = f64 ? VT<double>::GROWS1 - 1 : VT<float>::GROWS1 - 1;
  const void* f = f64 ? kernel<double>() : kernel<float>();
  long long cells = 0;
  for (auto& h : b.hv) cells = std::max(cells, (long long)(h.g.ny + 1) * b.P);
  if (cells >= (1LL << 31)) return false;
  int coop = 0;
  PF_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, b.device));
  if (!coop) return false;
  // the largest block of each kind decides the shared memory of all CTAs
  R.smem = f64 ? std::max(Lay<double>(rows, 0).total, Lay<double>(grows, 1).total)
               : std::max(Lay<float>(rows, 0).total, Lay<float>(grows, 1).total);
  PF_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R.smem));
  int occ = 0;
  PF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, RNT, R.smem));
  const long long G = (long long)occ * b.nsm;
  if (G < 1) return false;
  double nodes = 0.0;
  for (auto& h : b.hv) nodes += (double)(h.g.nx + 1) * (h.g.ny + 1);
  if (nodes > 2.0 * G * RNT * H * rows) return false;
  // tile flags
  const long long T = b.Tcg;
  std::vector<int2> ij(T);
  std::vector<int> var(T);
  std::vector<uint8_t> fl(T);
  PF_CUDA(cudaMemcpyAsync(ij.data(), b.tile_cg_ij, T * sizeof(int2), cudaMemcpyDeviceToHost, b.stream));
  PF_CUDA(cudaMemcpyAsync(var.data(), b.tile_cg_var, T * sizeof(int), cudaMemcpyDeviceToHost, b.stream));
  PF_CUDA(cudaMemcpyAsync(fl.data(), b.tile_cg_gen, T, cudaMemcpyDeviceToHost, b.stream));
  PF_CUDA(cudaStreamSynchronize(b.stream));
  std::vector<Cutter> cut(b.nv);
  for (int v = 0; v < b.nv; ++v) {
    Cutter& c = cut[v];
    c.W = b.hv[v].g.nx + 1;
    c.R = b.hv[v].g.ny + 1;
    c.H = H;
    c.tx = (c.W + CTX - 1) / CTX;
    c.ty = (c.R + CTY - 1) / CTY;
    c.stored.assign((size_t)c.tx * c.ty, 0);
    if ((double)c.W * c.R > (double)G * RNT * H * rows) return false;
  }
  const uint8_t bit = f64 ? TILE_ROW64 : TILE_ROW32;
  for (long long t = 0; t < T; ++t)
    if (fl[t] & bit) cut[var[t]].stored[(size_t)(ij[t].y / CTY) * cut[var[t]].tx + ij[t].x / CTX] = 1;
  std::vector<std::vector<RItem>> blocks(b.nv);
  long long total = 0;
  auto plan = [&](int cap, int gcap, int threads, long long most) {
    total = 0;
    for (int v = 0; v < b.nv && total <= most; ++v) {
      if (!cut[v].best(cap, std::max(2, std::min(grows, gcap)), threads, blocks[v])) return false;
      total += (long long)blocks[v].size();
    }
    return total <= most;
  };
  auto least = [&](int cap, int gcap, int threads) {
    double n = 0.0;
    for (auto& c : cut) n += std::max(1.0, std::ceil(c.least(cap, std::max(2, std::min(grows, gcap)), threads) * (1.0 - 1e-9)));
    return n;
  };
  // all at once: the cut whose iteration is estimated shortest.  An iteration's fixed part costs
  // about as much as five rows; a row with stored coefficients 1.6 times (FP64: 1.5 times) a row
  // without; two blocks on one SM share it.  From the least estimate up, as far as one can still
  // win, and cut only where the least number of blocks leaves room.  A handle's first solve is
  // longer than its second by 0.95 ms with five 403x201 channels (every candidate in turn: 2.6),
  // 0.85 with one 1024x512 grid in FP64 (4.4), 0.8 on 6000x60 cells (4.6), and 0.75 where two
  // 2048x1024 grids do not fit (2.1)
  struct Candidate { double cost; int threads, cap, gc; };
  std::vector<Candidate> cand;
  for (int threads : {64, 128, RNT})
    for (int cap = 2; cap <= rows; ++cap)
      for (int gc = std::max(2, cap / 2); gc <= std::min(cap, grows); ++gc)
        if (nodes <= (double)G * threads * H * cap)
          cand.push_back({(5.0 + std::max((double)cap, (f64 ? 1.5 : 1.6) * gc)) * threads / RNT, threads, cap, gc});
  std::vector<int> by_cost(cand.size());
  for (size_t k = 0; k < cand.size(); ++k) by_cost[k] = (int)k;
  std::stable_sort(by_cost.begin(), by_cost.end(), [&](int x, int y) { return cand[x].cost < cand[y].cost; });
  double best_cost = 1e300;
  int best = -1, planned = -1;           // (of two with one cost the first in the loops' order)
  for (int k : by_cost) {
    const Candidate& c = cand[k];
    if (c.cost > best_cost) break;
    const double n = least(c.cap, c.gc, c.threads), low = c.cost * std::ceil(n / b.nsm);
    if (n > (double)G || low > best_cost || (low == best_cost && k > best)) continue;
    planned = k;
    if (!plan(c.cap, c.gc, c.threads, G)) continue;
    const double c2 = c.cost * (double)((total + b.nsm - 1) / b.nsm);
    if (c2 < best_cost || (c2 == best_cost && k < best)) {
      best_cost = c2;
      best = k;
    }
  }
  if (best >= 0) {
    if (planned != best) plan(cand[best].cap, cand[best].gc, cand[best].threads, G);
  } else if (least(rows, grows, RNT) > 2.0 * G || !plan(rows, grows, RNT, 2 * G)) {
    return false;                        // else the largest blocks, and the variants queue
  }
  size_t most = 0;
  for (auto& x : blocks) most = std::max(most, x.size());
  if ((long long)most > G || total > (1 << 24)) return false;
  // queued variants start with the longest: iterations grow with the grid's width and height
  std::vector<int> ord(b.nv);
  for (int v = 0; v < b.nv; ++v) ord[v] = v;
  std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) {
    return std::max(b.hv[x].g.nx, b.hv[x].g.ny) > std::max(b.hv[y].g.nx, b.hv[y].g.ny);
  });
  R.queued = best < 0;
  if (R.queued && f64) {
    // In FP64 a full chip gains little over the streaming kernel (both wait for the FP64 pipe), so
    // a queue has to pack well: few large variants leave CTAs without work (two 842x411 grids, one
    // after the other, 90 against 57 us an iteration), many small ones do not (63 of 155x66: 32
    // against 67).  Times of an iteration of the longest variant, fitted to 86 measured batches (5.5
    // and 9 us rms): with the chip filled `span` times over, and for the streaming kernel, whose
    // variants drop out as they finish.  At 0.88 none of them is slower here, two in five gain.
    // (FP32: 69 batches, 0.98 to 2.2 times as fast; no rule.)
    std::vector<double> tiles(b.nv, 0.0), gen(b.nv, 0.0);
    for (long long t = 0; t < T; ++t) {
      tiles[var[t]] += 1.0;
      if (fl[t] & TILE_GEN64) gen[var[t]] += 1.0;
    }
    std::vector<std::pair<double, long long>> run;     // running variants: end, blocks (a heap, earliest first)
    const auto later = [](const std::pair<double, long long>& x, const std::pair<double, long long>& y) { return x.first > y.first; };
    double now = 0.0, span = 0.0, area = 0.0, nt = 0.0, ng = 0.0;
    long long left = G;
    const double longest = std::max(b.hv[ord[0]].g.nx, b.hv[ord[0]].g.ny);
    for (int v : ord) {
      const double w = std::max(b.hv[v].g.nx, b.hv[v].g.ny) / longest;
      const long long n = (long long)blocks[v].size();
      while (left < n) {
        std::pop_heap(run.begin(), run.end(), later);
        now = run.back().first;
        left += run.back().second;
        run.pop_back();
      }
      left -= n;
      run.push_back({now + w, n});
      std::push_heap(run.begin(), run.end(), later);
      span = std::max(span, now + w);
      area += w * (double)n / (double)G;
      nt += w * tiles[v];
      ng += w * gen[v];
    }
    const double here = (31.0 + 6.0 * ng / nt) * span + 7.5 * area;
    const double streamed = 31.0 + 0.0385 * nt + 0.0214 * ng + 0.19 * b.nv;
    if (here > 0.88 * streamed) return false;
  }
  std::vector<RItem> items;
  std::vector<RVar> vars(b.nv);
  items.reserve(total);
  int nbm = 0;
  for (int v : ord) {
    nbm = std::max(nbm, b.hv[v].nb);
    vars[v].part0 = (int)items.size();
    vars[v].parts = (int)blocks[v].size();
    for (size_t k = 0; k < blocks[v].size(); ++k) {
      RItem x = blocks[v][k];
      x.v = v;
      x.part = (int)k;
      items.push_back(x);
    }
  }
  R.grid = (int)std::min<long long>(G, total);
  R.n_items = (int)total;
  R.qs = 4 + nbm;
  R.pw_half = total * R.qs * 2;
  const size_t WPV = f64 ? 2 : 1;
  R.bc_words = (size_t)b.nv * 2 * (R.qs - 1) * WPV;
  try {
    R.d_var = dev_alloc(b, b.nv * sizeof(RVar));
    R.d_items = dev_alloc(b, items.size() * sizeof(RItem));
    R.d_ctrl = (int*)dev_alloc(b, (1 + b.nv) * sizeof(int));
    R.d_epoch = (unsigned*)dev_alloc(b, b.nv * sizeof(unsigned));
    R.d_pw = (unsigned long long*)dev_alloc(b, 2 * R.pw_half * sizeof(u64));
    R.d_bc = (unsigned long long*)dev_alloc(b, R.bc_words * sizeof(u64));
    R.d_pbm = (unsigned long long*)dev_alloc(b, total * sizeof(u64));
    R.d_blist = (int*)dev_alloc(b, std::max<long long>(1, total * nbm) * sizeof(int));
  } catch (const Error& e) {
    if (e.code != PF_ENOMEM) throw;
    free_plan(b, R);                     // no room for the exchange buffers: the streaming kernel solves
    R.made = true;
    return false;
  }
  PF_CUDA(cudaMemcpyAsync(R.d_var, vars.data(), b.nv * sizeof(RVar), cudaMemcpyHostToDevice, b.stream));
  PF_CUDA(cudaMemcpyAsync(R.d_items, items.data(), items.size() * sizeof(RItem), cudaMemcpyHostToDevice, b.stream));
  clear_exchange(b, R);
  PF_CUDA(cudaStreamSynchronize(b.stream));
  R.ok = true;
  return true;
}

// The plan is made again on the next solve (node coordinates were replaced).
void drop_resident(Batch& b) {
  for (ResPlan& R : b.res) free_plan(b, R);
}

template <typename T>
static void launch(Batch& b, ResPlan& R, State4<T>* const st[2], T* sb, int max_it) {
  ResArgs<T> a;
  a.m.var = b.d_var;
  a.m.tag = b.tag;
  a.m.bid = b.bid;
  a.m.body_ptr = b.body_ptr;
  a.m.body_nodes = b.body_nodes;
  a.m.K64 = b.K64;
  a.m.K32 = b.K32;
  a.m.Vtot = b.Vtot;
  a.st = b.state;
  a.prm = b.params;
  a.s[0] = st[0];
  a.s[1] = st[1];
  a.sb = sb;
  a.B = std::max(1, b.B);
  a.var = (const RVar*)R.d_var;
  a.items = (const RItem*)R.d_items;
  a.n_items = R.n_items;
  a.ticket = R.d_ctrl;
  a.join = R.d_ctrl + 1;
  a.pw = R.d_pw;
  a.pw_half = R.pw_half;
  a.bc = R.d_bc;
  a.pbm = R.d_pbm;
  a.blist = R.d_blist;
  a.qs = R.qs;
  a.epoch = R.d_epoch;
  a.err = b.d_err;
  a.n_done = b.n_done;
  a.poll_limit = b.test_drop ? 1024 : MBAR_POLL_LIMIT;
  a.test_drop = b.test_drop;
  a.max_it = max_it;
  R.open = true;
  PF_CUDA(cudaMemsetAsync(R.d_ctrl, 0, (1 + b.nv) * sizeof(int), b.stream));
  PF_CUDA(cudaFuncSetAttribute(kernel<T>(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)R.smem));
  void* args[] = {&a};
  PF_CUDA(cudaLaunchCooperativeKernel(kernel<T>(), dim3(R.grid), dim3(RNT), args, R.smem, b.stream));
}

// Every variant in the CG phase runs its CG to the inner stopping test, or for max_it
// iterations (one launch).  The caller ends the solve with end_resident once every launch
// has come to its end without a wait that gave up.
void launch_resident(Batch& b, int precision, int max_it) {
  ResPlan& R = b.res[precision];
  if (precision == PF_FP64) launch<double>(b, R, b.st64, b.sb64, max_it);
  else launch<float>(b, R, b.st32, b.sb32, max_it);
}

void end_resident(Batch& b, int precision) { b.res[precision].open = false; }

}  // namespace pfq4
