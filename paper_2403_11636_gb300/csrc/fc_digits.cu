// fc_digits.cu -- FP64 products with rows that many nodes share, on the tensor
// cores.
//
// Away from obstacles and walls the operator's stencil and the cached patch
// rows are the same for every fluid node, so the smoother residual y = L x and
// the patch apply y = Inv r are products of one short matrix W (d+1 rows; 27 or
// 59 slots in 2D, 402 for the patch in 3D) with vectors gathered around each
// node.  FP64 is the bound of both on this part (a warp FMA takes 64 clocks of
// an SM partition), so the products are formed from digits whose products and
// sums are exact (the slices of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms
// 59, 2012, on a tile's common exponent):
//
//  - a CTA takes a tile of nodes and its halo, finds the largest exponent E of
//    the values that the tile's products read, and rounds each value to a
//    62-bit fixed-point number v 2^(62-E) in eight signed base-256 digits,
//    held as half-precision integers in [-128, 127];
//  - the rows W have the same form in ten digits with an exponent per row
//    (setup), the velocity and pressure columns first brought to one scale by a
//    power of two (delta), as D L D equilibrates the blocks;
//  - S_d = sum_slots sum_{s+t=d} w_s v_t, d = 0..9, is one matrix product: a
//    node is a row of the left operand (K = slot, digit), a row of W and an
//    antidiagonal d a column of the right one (w_{d-s} at digit s), and
//    y = 2^(Ew+E-12) sum_d S_d 2^(-8d), rounded to double once.  (3D: 40 columns
//    of N = 48; with N = 32 and eight antidiagonals the sums that are left out
//    would be 2^-58 of max|w| max|v|.)
//
// The digits of a component lie 16 bytes a node, nodes in the order of the
// halo tile, so the left operand of a pair of slots is read in place: 128
// consecutive nodes are a tcgen05 tile, a slot is an offset of its descriptor
// (8 x 16-byte core matrices 128 bytes apart; the second slot at the leading
// offset).  Rows of the halo are computed too and dropped.  Accumulators stay
// in tensor memory; a thread then reads all S_d of one node.
//
// Accuracy: products are integers of at most 2^14 and float32 sums of integers
// are exact below 2^24.  digit_rows_kernel adds up the magnitudes of W's
// digits: in 2D no sum can reach 2^24, in 3D none of d <= 5 (or the class is
// not used); those of d >= 6, of weight 2^-48 and less, could in 3D round by a
// unit if nearly all digits were largest and of one sign.  What is lost is the
// rounding of the values, at most 2^(E-63) sum|w| (the antidiagonals that are
// left out and W's own rounding are 2^-66 of 2^(Ew+E) at most).  That is relative
// to the tile's largest value, not to what a node reads, so each node's sum |w||v|
// is formed beside it in float32, and a node where it is below 2^(E-11) sum|w|
// for some row leaves the digits: a result's error is at most about 2^-52
// sum |w||v|, where a chain of FP64 fused multiply-adds can round every partial
// sum by 2^-53 of it (measured: see kFloor).  The nodes that leave, and all of a
// tile that holds an infinity or NaN, whose exponent is extreme, or whose
// products do not come in time, are formed in FP64 by the tile's CTA as the
// general kernels do.
//
// Which nodes: `cls` of the plan.  Fictitious nodes (alpha-scaled rows) read
// values far below their tile's largest in nearly every field (sum |w||v| from
// 2^-9 to 2^-28 of the largest; fluid nodes 2^-2 to 2^-6), so they are left,
// with all other nodes, to the FP64 kernels (plan list).
#include <cuda_fp16.h>
#include <math.h>
#include <stdlib.h>

#include <algorithm>
#include <type_traits>

#include "fc_node.cuh"

namespace fc {

namespace {

// KIND 0: patch apply (velocities of the 5^d box, pressures of the 3^d box),
// KIND 1: operator (all components of the 3^d box; 2D: in 3D the tile's halo
// and the rows of the halo cost more than the 270 FMA of a node).
template <int DIM, int KIND>
struct Dig {
  static constexpr int ND = DIM + 1, R = KIND == 0 ? 2 : 1;
  static constexpr int NSLOT = KIND == 0 ? SlotDims<DIM>::NSLOT : (DIM == 3 ? 27 : 9) * ND;
  static constexpr int STEPS = (NSLOT + 1) / 2;  // K = 16: two slots
  // tile: NBLK blocks of 128 rows cover the tile's nodes in halo order
  static constexpr int TX = DIM == 3 ? 16 : 32, TY = DIM == 3 ? 8 : 14, TZ = DIM == 3 ? 4 : 1;
  static constexpr int HX = TX + 2 * R, HY = TY + 2 * R, HZ = DIM == 3 ? TZ + 2 * R : 1;
  static constexpr int NHALO = HX * HY * HZ;
  static constexpr int LAST = (TX - 1) + HX * ((TY - 1) + HY * (TZ - 1));
  static constexpr int NBLK = LAST / 128 + 1;
  // columns of the right operand: ND rows x NA antidiagonals, filled up to a multiple of 16
  static constexpr int NA = 10, N = (ND * NA + 15) / 16 * 16;
  static constexpr int TMEM = NBLK * N <= 128 ? 128 : NBLK * N <= 256 ? 256 : 512;  // columns
  // largest offset of a slot's node from the corner, and the nodes of a plane
  // that some row of a block can read
  static constexpr int FAR = 2 * R * (1 + HX + (DIM == 3 ? HX * HY : 0));
  static constexpr int PLANE = NBLK * 128 + FAR + 8;
  static constexpr int THREADS = 256, PER_SM = DIM == 3 ? 1 : 3;  // CTAs an SM, by shared memory
  // W is read in pieces of CS steps, NST pieces in flight
  static constexpr int CS = DIM == 3 ? 12 : STEPS, NST = DIM == 3 ? 3 : 1, NCH = (STEPS + CS - 1) / CS;
  static constexpr int STEPB = 2 * N * 16;  // bytes of W a step
  // node rows of a warp, and those that one of the warps 1-7 checks
  static constexpr int NWR = NBLK * 4, NCHK = (NWR + THREADS / 32 - 2) / (THREADS / 32 - 1);
  static constexpr int CHUNK = 8, CHK = (NSLOT + CHUNK - 1) / CHUNK * CHUNK;
  static constexpr size_t O_ROWS = (size_t)PLANE * 16 * ND;
  static constexpr size_t O_WABS = O_ROWS + (size_t)NST * CS * STEPB;     // |w| 2^-Ew, float4 a slot
  static constexpr size_t O_MAG = O_WABS + (size_t)CHK * 16;              // |v| 2^-E, float
  static constexpr size_t O_OFFS = O_MAG + (size_t)PLANE * ND * 4;
  static constexpr size_t O_CHK = O_OFFS + (size_t)STEPS * sizeof(unsigned);  // offsets of O_WABS's slots
  static constexpr size_t O_CLS = O_CHK + (size_t)CHK * 2;
  static constexpr size_t O_LEFT = (O_CLS + NHALO + 1) / 2 * 2;           // nodes that leave the digits
  static constexpr size_t BYTES = (O_LEFT + (size_t)NBLK * 128 * 2 + 15) / 16 * 16;
  static_assert((size_t)NSLOT * 4 <= (size_t)NST * CS * STEPB, "the slot table takes W's place");
};

// Slots in the order of their digits' addresses (component, then node).
// Offset of the slot's node, its component; the slot's index in the cached
// rows (KIND 0) or in (node, component) order (KIND 1)
template <int DIM, int KIND>
__device__ __forceinline__ void slot_of(int j, int* o, int* c, int* src) {
  using P = SlotDims<DIM>;
  constexpr int NV = KIND == 0 ? P::NU : (DIM == 3 ? 27 : 9);
  int t, w, h;
  if (j < NV * DIM) {
    *c = j / NV;
    t = j % NV;
    w = KIND == 0 ? 5 : 3;
  } else {
    *c = DIM;
    t = j - NV * DIM;
    w = 3;
  }
  h = w / 2;
  o[0] = t % w - h;
  o[1] = DIM == 3 ? (t / w) % w - h : t / w - h;
  o[2] = DIM == 3 ? t / (w * w) - h : 0;
  if (KIND == 0) *src = *c < DIM ? t * DIM + *c : P::NU * DIM + t;
  else *src = t * (DIM + 1) + *c;
}

// eight base-256 digits of V + 0x80..80 (most significant first), as halves
__device__ __forceinline__ uint4 digits_of(long long V) {
  const unsigned long long T = (unsigned long long)V + 0x8080808080808080ull;
  const unsigned hi = (unsigned)(T >> 32), lo = (unsigned)T;
  // 0x6400 + u is the half 1024 + u; less 1152 leaves the digit u - 128
  const __half2 m = __half2half2(__ushort_as_half(0x6480));
  unsigned w[4] = {__byte_perm(hi, 0x64646464u, 0x4243), __byte_perm(hi, 0x64646464u, 0x4041),
                   __byte_perm(lo, 0x64646464u, 0x4243), __byte_perm(lo, 0x64646464u, 0x4041)};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    __half2 h = *reinterpret_cast<__half2*>(&w[k]);
    h = __hsub2(h, m);
    w[k] = *reinterpret_cast<unsigned*>(&h);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// v 2^(62 - E) rounded, for |v| < 2^E with E = emax - 1022 and e the biased
// exponent of v (shifted by delta for pressures)
__device__ __forceinline__ long long fixed_point(double v, int emax, int shift) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu);
  if (e == 0) return 0;  // zero or subnormal
  const int sh = emax - (e + shift);
  if (sh > 62) return 0;
  const unsigned long long m = ((((unsigned long long)(hi & 0xfffffu) | 0x100000ull) << 32) | lo) << 9;
  const long long V = (long long)((m + ((1ull << sh) >> 1)) >> sh);
  return (hi >> 31) ? -V : V;
}

// |v| 2^-E as float, truncated; not zero where v is not
__device__ __forceinline__ float magnitude(double v, int emax, int shift) {
  const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu, lo = (unsigned)__double2loint(v);
  const int e = (int)(hi >> 20), f = 126 + (e + shift) - emax;
  if ((hi | lo) == 0u) return 0.0f;
  if (e == 0 || f < 1) return 1.1754943508222875e-38f;
  return __uint_as_float(((unsigned)f << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
}

// The ten digits of w 2^(78 - E), rounded (setup)
__device__ __forceinline__ void row_digits(double v, int emax, int shift, int* d) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int e = (int)((hi >> 20) & 0x7ffu), sh = emax - (e + shift);
  __int128 V = 0;
  if (e != 0 && sh <= 78) {
    const __int128 m = (__int128)((((unsigned long long)(hi & 0xfffffu) | 0x100000ull) << 32) | lo) << 25;
    V = (m + (((__int128)1 << sh) >> 1)) >> sh;
    if (hi >> 31) V = -V;
  }
  for (int k = 9; k > 0; --k) {
    d[k] = (int)((V + 128) & 255) - 128;
    V = (V - d[k]) >> 8;
  }
  d[0] = (int)V;
}

__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// ---- tcgen05, mbarrier and bulk copies
// A wait gives up after a second (the wait for products after the plan's wait_ns)
constexpr unsigned long long kWaitNs = 1000000000ull;

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, unsigned long long limit = kWaitNs) {
  if (limit == 0ull) return false;
  unsigned long long start = 0ull;
  for (;;) {
    unsigned done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    unsigned long long now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (start == 0ull) start = now;
    else if (now - start > limit) return false;
  }
}
// global -> shared copy of `bytes` (a multiple of 16) that completes on bar
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tc_mma(unsigned d, unsigned long long a, unsigned long long b, unsigned idesc,
                                       bool add) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"((unsigned)add)
      : "memory");
}
// one lane of a full warp; a branch on it keeps the descriptors in uniform
// registers (43 clocks from product to product; 84 behind a test of threadIdx)
__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(p));
  return p != 0u;
}
__device__ __forceinline__ void tc_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// N columns of a thread's row: 32, or 40 (one block of instructions, for the
// values are there after the wait only)
template <int N>
__device__ __forceinline__ void tc_load(unsigned addr, unsigned* v) {
  static_assert(N == 32 || N == 40, "columns");
  if constexpr (N == 40)
    asm volatile(
        "{\ntcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%40];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%32,%33,%34,%35,%36,%37,%38,%39}, [%41];\n"
        "tcgen05.wait::ld.sync.aligned;\n}"
        : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7]),
          "=&r"(v[8]), "=&r"(v[9]), "=&r"(v[10]), "=&r"(v[11]), "=&r"(v[12]), "=&r"(v[13]), "=&r"(v[14]), "=&r"(v[15]),
          "=&r"(v[16]), "=&r"(v[17]), "=&r"(v[18]), "=&r"(v[19]), "=&r"(v[20]), "=&r"(v[21]), "=&r"(v[22]), "=&r"(v[23]),
          "=&r"(v[24]), "=&r"(v[25]), "=&r"(v[26]), "=&r"(v[27]), "=&r"(v[28]), "=&r"(v[29]), "=&r"(v[30]), "=&r"(v[31]),
          "=&r"(v[32]), "=&r"(v[33]), "=&r"(v[34]), "=&r"(v[35]), "=&r"(v[36]), "=&r"(v[37]), "=&r"(v[38]), "=&r"(v[39])
        : "r"(addr), "r"(addr + 32)
        : "memory");
  else
    asm volatile(
        "{\ntcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;\n}"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(addr)
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

struct DigArgs {
  const unsigned char* cls;
  const uint4* rows;
  const float4* wabs;
  const unsigned short* chk;
  const DigitScale* sc;
  unsigned* err;
  unsigned long long wait_ns;
  const int* list;
  int nlist, list_blocks;
  // KIND 0: v = padded residual, x updated.  KIND 1: v = x, r and rpad
  // (nullable) receive b - L x (L x when b is null)
  const double* v;
  const double* b;
  double* x;
  double* r;
  double* rpad;
  double omega;
  // the FP64 products of the list and of the nodes that leave the digits
  const double* coef;  // KIND 0 rows, KIND 1 stencil
  const unsigned char* mask;
  const int* prow;
};

// x + omega y (own = x, scale includes omega), or b - y (own = b; y without b)
template <int DIM, int KIND>
__device__ __forceinline__ void store_product(const LevelGeom& g, const DigArgs& a, const int* ia, const double* own,
                                              const double* y, const double* scale) {
  constexpr int ND = DIM + 1;
  const long long n = ia[0] + (long long)g.nn[0] * (ia[1] + (long long)(DIM == 3 ? g.nn[1] : 1) * ia[2]);
  double v[ND];
#pragma unroll
  for (int c = 0; c < ND; ++c) {
    if (KIND == 0) v[c] = own[c] + scale[c] * y[c];
    else v[c] = a.b ? own[c] - scale[c] * y[c] : scale[c] * y[c];
  }
  if (KIND == 0) {
#pragma unroll
    for (int c = 0; c < ND; ++c) a.x[n * ND + c] = v[c];
    return;
  }
  if (a.r) {
#pragma unroll
    for (int c = 0; c < ND; ++c) a.r[n * ND + c] = v[c];
  }
  if (a.rpad) {
    double* p = a.rpad + pad_node(g, ia[0], ia[1], ia[2]) * ND;
#pragma unroll
    for (int c = 0; c < ND; ++c) p[c] = v[c];
  }
}

// A node takes its digits' result where sum |w||v| >= 2^kFloor 2^E sum|w| in every
// row: the values' rounding is then at most 2^-52 sum |w||v|, and at random below
// that of the FP64 sums.  Error in 2^-53 sum |w||v|, root mean square (largest), of
// nodes that read random values 2^-k times those of a few others in the tile,
// all by digits / by the FP64 kernels: patch apply 2D k = 4 0.11 (0.6) / 0.31
// (1.7), k = 10 0.11 (0.6), k = 11 0.57 (2.7), k = 14 3.7; 3D k = 4 0.08 (0.4) /
// 0.38 (2.2), k = 9 0.15, k = 10 0.25 (1.5), k = 11 0.65 (4.1); operator k = 4 0.18
// (0.9) / 0.55 (3.4), k = 9 0.30, k = 10 0.47 (3.2), k = 11 1.2 (9.6).  Random
// values have half their bound in the mean, so -11 is k = 10.
constexpr int kFloor = -11;

// 2D: the first list_blocks CTAs take the nodes of the plan's list in FP64.
// The others take a tile each.  (CTAs that keep W and walk over the tiles, the
// next tile's values loaded during the products, were slower: 196 against 164
// us for the 1537^2 patch apply.)
template <int DIM, int KIND>
__global__ void __launch_bounds__(Dig<DIM, KIND>::THREADS, Dig<DIM, KIND>::PER_SM)
    digit_product_kernel(LevelGeom g, DigArgs a, int tiles_x, int tiles_y) {
  using D = Dig<DIM, KIND>;
  constexpr int ND = D::ND, R = D::R;
  constexpr int TPP = DIM == 3 ? 8 : 4;  // lanes of a node in FP64
  extern __shared__ uint4 dsm[];
  if (DIM == 2 && (int)blockIdx.x < a.list_blocks) {
    const int gi = (int)((blockIdx.x * 256u + threadIdx.x) / TPP);
    const bool valid = gi < a.nlist;
    const int node = a.list[valid ? gi : a.nlist - 1];
    if constexpr (KIND == 0) {
      int* soff = reinterpret_cast<int*>(dsm);
      slot_table<DIM>(g, soff);
      apply_fp64_patch<DIM, TPP>(g, a.coef, a.mask, a.v, a.omega, a.x, a.prow, soff, (unsigned)node, valid);
    } else {
      residual_node<DIM, 0, TPP>(g, a.coef, a.mask, a.v, a.b, a.r, a.rpad, nullptr, node, valid);
    }
    return;
  }
  char* smem = reinterpret_cast<char*>(dsm);
  float* smag = reinterpret_cast<float*>(smem + D::O_MAG);
  float4* swabs = reinterpret_cast<float4*>(smem + D::O_WABS);
  unsigned* soffs = reinterpret_cast<unsigned*>(smem + D::O_OFFS);
  unsigned short* schk = reinterpret_cast<unsigned short*>(smem + D::O_CHK);
  unsigned char* scls = reinterpret_cast<unsigned char*>(smem + D::O_CLS);
  unsigned short* sleft = reinterpret_cast<unsigned short*>(smem + D::O_LEFT);
  constexpr int NH = (D::NHALO + D::THREADS - 1) / D::THREADS;
  // W arrived [NST], W used [NST], products done [per block where W is one
  // piece], drained.  Every arrival is waited for before the CTA ends: a block
  // without class nodes and a place that takes no further piece of W are not
  // committed.
  constexpr int NDONE = D::NCH == 1 ? D::NBLK : 1;
  __shared__ __align__(8) unsigned long long sbar[2 * D::NST + NDONE + 1];
  __shared__ int semax, sbad, sfail, snleft;
  __shared__ unsigned sblk, stmem, spass[D::NWR];
  const int tid = threadIdx.x, lane = tid & 31, wib = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(smem);
  const unsigned bar0 = (unsigned)__cvta_generic_to_shared(sbar);
  const unsigned bar_done = bar0 + 8 * 2 * D::NST, bar_drain = bar_done + 8 * NDONE;
  const unsigned tile = blockIdx.x - (unsigned)a.list_blocks, tq = tile / (unsigned)tiles_x;
  // the first R layers of a grid hold no class node (their boxes leave it): of
  // 2^k + 1 nodes, a multiple of the tile and a remainder are left
  const int bx = (int)(tile - tq * (unsigned)tiles_x) * D::TX + R;
  const int by = (int)(DIM == 3 ? tq % (unsigned)tiles_y : tq) * D::TY + R;
  const int bz = DIM == 3 ? (int)(tq / (unsigned)tiles_y) * D::TZ + R : 0;
  // ---- the tile and its halo: every load is issued before the first is used
  unsigned char hc[NH];
  double hv[NH][ND];
#pragma unroll
  for (int q = 0; q < NH; ++q) {
    const int n = q * D::THREADS + tid;
    const int hx = n % D::HX, hy = (n / D::HX) % D::HY, hz = n / (D::HX * D::HY);
    const int i = bx + hx - R, j = by + hy - R, k = DIM == 3 ? bz + hz - R : 0;
    const bool in =
        n < D::NHALO && i >= 0 && i < g.nn[0] && j >= 0 && j < g.nn[1] && (DIM == 2 || (k >= 0 && k < g.nn[2]));
    const long long at = in ? i + (long long)g.nn[0] * (j + (long long)(DIM == 3 ? g.nn[1] : 1) * k) : 0;
    const double* v = a.v + (KIND == 0 ? (in ? pad_node(g, i, j, k) : 0) : at) * ND;
    hc[q] = in ? a.cls[at] : (unsigned char)0;
    if (KIND == 0 && ND == 4) {  // (own buffer: 16-byte aligned; x is the caller's)
      const double2 v0 = in ? reinterpret_cast<const double2*>(v)[0] : make_double2(0.0, 0.0);
      const double2 v1 = in ? reinterpret_cast<const double2*>(v)[1] : make_double2(0.0, 0.0);
      hv[q][0] = v0.x; hv[q][1] = v0.y; hv[q][2] = v1.x; hv[q][ND - 1] = v1.y;
    } else {
#pragma unroll
      for (int c = 0; c < ND; ++c) hv[q][c] = in ? v[c] : 0.0;
    }
  }
  const int delta = a.sc->delta;
  const bool sc_ok = a.sc->ok != 0;
  if (tid == 0) {
    for (int k = 0; k < 2 * D::NST + NDONE + 1; ++k) mbar_init(bar0 + 8 * k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    semax = -100000;
    sblk = 0u;
    sbad = 0;
    sfail = 0;
    snleft = 0;
  }
  for (int t = tid; t < D::CHK; t += D::THREADS) {
    swabs[t] = a.wabs[t];
    schk[t] = a.chk[t];
  }
  // operand offsets of a step: first slot's digits, and the second's distance
  for (int t = tid; t < D::STEPS; t += D::THREADS) {
    unsigned at[2];
    for (int h = 0; h < 2; ++h) {
      int o[3], c, src;
      const int j = 2 * t + h;
      slot_of<DIM, KIND>(j < D::NSLOT ? j : j - 1, o, &c, &src);
      at[h] = (unsigned)(c * D::PLANE + (o[0] + R) + D::HX * ((o[1] + R) + (DIM == 3 ? D::HY * (o[2] + R) : 0)));
      if (j >= D::NSLOT) at[h] += 1;  // an odd count's last slot: any digits, W's are zero
    }
    soffs[t] = at[0] | ((at[1] - at[0]) << 16);  // in units of 16 bytes
  }
  // past the halo: zeros, read by rows whose results are dropped
  for (int t = tid; t < (D::PLANE - D::NHALO) * ND; t += D::THREADS) {
    const int c = t / (D::PLANE - D::NHALO), n = D::NHALO + t % (D::PLANE - D::NHALO);
    *reinterpret_cast<uint4*>(smem + ((size_t)c * D::PLANE + n) * 16) = make_uint4(0u, 0u, 0u, 0u);
    smag[c * D::PLANE + n] = 0.0f;
  }
  // W in pieces of CS steps through NST places
  auto load_w = [&](int k) {
    const int st = k % D::NST;
    const unsigned steps = (unsigned)min(D::CS, D::STEPS - k * D::CS);
    bulk_load(sbase + (unsigned)D::O_ROWS + st * D::CS * D::STEPB,
              reinterpret_cast<const char*>(a.rows) + (size_t)k * D::CS * D::STEPB, steps * D::STEPB, bar0 + 8 * st);
  };
  // row m of the blocks (node m of the halo order, seen from the tile) is a class node
  auto row_class = [&](int m) {
    const int l0 = m % D::HX, l1 = DIM == 3 ? (m / D::HX) % D::HY : m / D::HX, l2 = DIM == 3 ? m / (D::HX * D::HY) : 0;
    if (l0 >= D::TX || l1 >= D::TY || l2 >= D::TZ) return false;
    return (scls[(l0 + R) + D::HX * ((l1 + R) + (DIM == 3 ? D::HY * (l2 + R) : 0))] & 1) != 0;
  };
#pragma unroll
  for (int q = 0; q < NH; ++q)
    if (q * D::THREADS + tid < D::NHALO) scls[q * D::THREADS + tid] = hc[q];
  __syncthreads();
  // ---- largest exponent of the values
  int emt = -100000;
#pragma unroll
  for (int q = 0; q < NH; ++q) {
    if (!(hc[q] & 2)) continue;
#pragma unroll
    for (int c = 0; c < ND; ++c) {
      const int e = (__double2hiint(hv[q][c]) >> 20) & 0x7ff;
      if (e == 0x7ff) sbad = 1;
      const bool none = ((__double2hiint(hv[q][c]) & 0x7fffffff) | __double2loint(hv[q][c])) == 0;
      emt = max(emt, none ? -100000 : e + (c == DIM ? delta : 0));
    }
  }
  emt = __reduce_max_sync(0xffffffffu, emt);
  if (lane == 0 && emt > -100000) atomicMax(&semax, emt);
  // ---- blocks that hold class nodes; a thread's own nodes: row tid % 128 of
  // every second block
  constexpr int NB = (D::NBLK + 1) / 2;
  bool rc[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int blk = 2 * q + (wib >> 2);
    rc[q] = blk < D::NBLK && row_class(blk * 128 + (wib & 3) * 32 + lane);
    const bool any = __any_sync(0xffffffffu, rc[q]);
    if (lane == 0 && any) atomicOr(&sblk, 1u << blk);
  }
  __syncthreads();
  const unsigned blocks = sblk;
  if (blocks == 0u) return;
  const int em = semax;
  const bool zero = !sbad && em == -100000;  // nothing but zeros: so are the products
  const bool digits = !sbad && sc_ok && em >= 1022 - 500 && em <= 1022 + 500;
  if (digits) {
    // ---- W on its way while the digits are written
    if (tid == 0)
      for (int k = 0; k < D::NST && k < D::NCH; ++k) load_w(k);
    if (wib == 1) {
      const unsigned at = (unsigned)__cvta_generic_to_shared(&stmem);
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(at), "n"(D::TMEM)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // ---- digits; zeros where no product reads a value
#pragma unroll
    for (int q = 0; q < NH; ++q) {
      const int n = q * D::THREADS + tid;
      if (n >= D::NHALO) continue;
#pragma unroll
      for (int c = 0; c < ND; ++c) {
        const bool read = (hc[q] & 2) != 0;
        const int shift = c == DIM ? delta : 0;
        *reinterpret_cast<uint4*>(smem + ((size_t)c * D::PLANE + n) * 16) =
            read ? digits_of(fixed_point(hv[q][c], em, shift)) : make_uint4(0u, 0u, 0u, 0u);
        smag[c * D::PLANE + n] = read ? magnitude(hv[q][c], em, shift) : 0.0f;
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }
  const unsigned tmem = stmem;
  unsigned owed = 0;  // the issuing thread: barriers with a commit, a bit each
  unsigned owed_parity = 0;
  if (digits && wib == 0) {
    if (elect_one()) {
      // ---- one thread: the products of each piece of W for every block.
      // Descriptors: no swizzle, core matrices of 8 rows x 16 bytes; left
      // operand: rows 16 bytes apart, groups of 8 rows 128; right: the
      // halves of K 16 N bytes apart, the columns' groups 128
      const unsigned long long hi = ((unsigned long long)(128 >> 4) << 32) | (1ull << 46);
      const unsigned idesc = (1u << 4) | ((unsigned)(D::N >> 3) << 17) | ((128u >> 4) << 24);
      const unsigned a0 = sbase >> 4;
      auto commit = [&](int b, unsigned parity) {
        tc_commit(bar0 + 8 * b);
        owed |= 1u << b;
        owed_parity = (owed_parity & ~(1u << b)) | (parity << b);
      };
      bool ok = true;
      int loaded = D::NST < D::NCH ? D::NST : D::NCH, waited = 0;
      for (int k = 0; k < D::NCH; ++k) {
        const int st = k % D::NST;
        if (k > 0 && k - 1 + D::NST < D::NCH) {
          // the piece before has been issued; when its products are done its place takes another
          const int u = k - 1;
          ok = ok && mbar_wait(bar0 + 8 * (D::NST + u % D::NST), (unsigned)((u / D::NST) & 1));
          if (ok) load_w(loaded++);
        }
        ok = ok && mbar_wait(bar0 + 8 * st, (unsigned)((k / D::NST) & 1));
        if (!ok) break;
        ++waited;
        tc_fence_after();
        const unsigned b0 =
            ((sbase + (unsigned)D::O_ROWS + st * D::CS * D::STEPB) >> 4) | ((unsigned)D::N << 16);
        const int t0 = k * D::CS, t1 = min(t0 + D::CS, D::STEPS);
        // A product reads 4 KB of digits and 32 N bytes of W at 128 bytes a
        // clock: 40 clocks (3D: 44).  W in one piece: block by block, so that
        // the results of one are taken while the next runs
        if (D::NCH == 1) {
#pragma unroll
          for (int blk = 0; blk < D::NBLK; ++blk) {
            if ((blocks >> blk) & 1u) {
#pragma unroll 6
              for (int t = 0; t < D::STEPS; ++t)
                tc_mma(tmem + blk * D::N, hi | (unsigned long long)(soffs[t] + (a0 + blk * 128)),
                       hi | (unsigned long long)(b0 + (unsigned)t * (D::STEPB / 16)), idesc, t > 0);
              commit(2 * D::NST + blk, 0u);
            }
          }
        } else {
          unsigned so = soffs[t0] + a0;
#pragma unroll 2
          for (int t = t0; t < t1; ++t) {
            const unsigned next = soffs[t + 1 < t1 ? t + 1 : t] + a0;
            const unsigned long long db = hi | (unsigned long long)(b0 + (unsigned)(t - t0) * (D::STEPB / 16));
#pragma unroll
            for (int blk = 0; blk < D::NBLK; ++blk)
              if ((blocks >> blk) & 1u)
                tc_mma(tmem + blk * D::N, hi | (unsigned long long)(so + blk * 128), db, idesc, t > 0);
            so = next;
          }
        }
        if (k + D::NST < D::NCH) commit(D::NST + st, (unsigned)((k / D::NST) & 1));
      }
      if (D::NCH > 1 && ok) commit(2 * D::NST, 0u);
      if (!ok) {
        // give up: once more for the copies on their way; what waits for the
        // products gives up at its own limit, the products on their way are
        // waited for at the end
        sfail = 1;
        for (int k = waited; k < loaded; ++k) mbar_wait(bar0 + 8 * (k % D::NST), (unsigned)((k / D::NST) & 1));
      }
    }
    __syncwarp();
  }
  // ---- what the thread's nodes bring besides the product, loaded meanwhile
  double own[NB][ND];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    if (!rc[q]) continue;
    const int m = (2 * q + (wib >> 2)) * 128 + (wib & 3) * 32 + lane;
    const int i = bx + m % D::HX, j = by + (DIM == 3 ? (m / D::HX) % D::HY : m / D::HX);
    const int k = DIM == 3 ? bz + m / (D::HX * D::HY) : 0;
    const long long n = i + (long long)g.nn[0] * (j + (long long)(DIM == 3 ? g.nn[1] : 1) * k);
    const double* from = KIND == 0 ? a.x : a.b;
#pragma unroll
    for (int c = 0; c < ND; ++c) own[q][c] = from ? from[n * ND + c] : 0.0;
  }
  if (digits) {
    // ---- sum |w||v| of every class node, by warps 1-7 while the products run
    // (warp 0 issues them), a warp's NCHK rows of nodes side by side.  Slots
    // come largest weight first and a part of the sum is enough, so most warps
    // end after CHUNK or two: shared memory is what the products are bound by.
    constexpr int NW = D::THREADS / 32 - 1;
    if (wib > 0) {
      float S[D::NCHK][ND], floor[ND];
      int at[D::NCHK];
      bool pass[D::NCHK];
#pragma unroll
      for (int r = 0; r < ND; ++r) floor[r] = a.sc->floor[r];
#pragma unroll
      for (int q = 0; q < D::NCHK; ++q) {
        const int w = wib - 1 + q * NW, m = w * 32 + lane;
        at[q] = m;
        pass[q] = w >= D::NWR || !((blocks >> (w >> 2)) & 1u) || !row_class(m);
        if (pass[q]) at[q] = 0;
#pragma unroll
        for (int r = 0; r < ND; ++r) S[q][r] = 0.0f;
      }
      for (int t0 = 0; t0 < D::CHK; t0 += D::CHUNK) {
        bool all = true;
#pragma unroll
        for (int q = 0; q < D::NCHK; ++q) all = all && pass[q];
        if (__all_sync(0xffffffffu, all)) break;
#pragma unroll
        for (int t = t0; t < t0 + D::CHUNK; ++t) {
          const float4 w = swabs[t];
          const int o = schk[t];
#pragma unroll
          for (int q = 0; q < D::NCHK; ++q) {
            const float v = smag[o + at[q]];
            S[q][0] = fmaf(w.x, v, S[q][0]);
            S[q][1] = fmaf(w.y, v, S[q][1]);
            S[q][2] = fmaf(w.z, v, S[q][2]);
            if (ND == 4) S[q][ND - 1] = fmaf(w.w, v, S[q][ND - 1]);
          }
        }
#pragma unroll
        for (int q = 0; q < D::NCHK; ++q) {
          bool p = true;
#pragma unroll
          for (int r = 0; r < ND; ++r) p = p && S[q][r] >= floor[r];
          pass[q] = pass[q] || p;
        }
      }
#pragma unroll
      for (int q = 0; q < D::NCHK; ++q) {
        // (a row that reads nothing but zeros is zero)
        bool p = true;
#pragma unroll
        for (int r = 0; r < ND; ++r) p = p && (S[q][r] >= floor[r] || S[q][r] == 0.0f);
        const int w = wib - 1 + q * NW;
        const unsigned b = __ballot_sync(0xffffffffu, pass[q] || p);
        if (w < D::NWR && lane == 0) spass[w] = b;
      }
      __threadfence_block();
      asm volatile("bar.arrive 2, %0;" ::"n"(D::THREADS) : "memory");
      asm volatile("bar.sync 1, %0;" ::"n"(D::THREADS - 32) : "memory");
    } else {
      asm volatile("bar.sync 2, %0;" ::"n"(D::THREADS) : "memory");
    }
  }
  double scale[ND];
#pragma unroll
  for (int n = 0; n < ND; ++n) {
    scale[n] = digits ? pow2(a.sc->rowexp[n] + (em - 1022) - 36) : 0.0;
    if (KIND == 0) scale[n] = a.omega * scale[n];
  }
  bool gave_up = false;
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int blk = 2 * q + (wib >> 2);
    if (blk >= D::NBLK || !((blocks >> blk) & 1u)) continue;
    const int m = blk * 128 + (wib & 3) * 32 + lane;
    double y[ND];
    bool have = zero;
#pragma unroll
    for (int n = 0; n < ND; ++n) y[n] = 0.0;
    if (digits && !gave_up) {
      // (the warp agrees: tcgen05.ld needs all of it)
      if (!__all_sync(0xffffffffu, mbar_wait(bar_done + 8 * (NDONE > 1 ? blk : 0), 0u, a.wait_ns))) {
        gave_up = true;  // no products: say so, and form them in FP64, these and the warp's others
        if (lane == 0) {
          atomicOr(a.err, kErrTimeout);
          sfail = 1;
        }
      } else {
        have = (spass[blk * 4 + (wib & 3)] >> lane) & 1u;
        tc_fence_after();
        constexpr int NCOL = ND * D::NA > 32 ? 40 : 32;
        unsigned v[NCOL];
        tc_load<NCOL>(tmem + ((unsigned)(wib & 3) << 21) + blk * D::N, v);
#pragma unroll
        for (int n = 0; n < ND; ++n) {
          // hi = S_0 2^24 + S_1 2^16 + S_2 2^8 + S_3, lo likewise of S_4..S_7,
          // and of S_8 and S_9 to lo's unit (2^-69 of 2^(Ew+E))
          long long h[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const unsigned* S = v + n * D::NA + k * 4;
            const int s0 = __float2int_rn(__uint_as_float(S[0])), s1 = __float2int_rn(__uint_as_float(S[1]));
            const int s2 = __float2int_rn(__uint_as_float(S[2])), s3 = __float2int_rn(__uint_as_float(S[3]));
            h[k] = (((long long)s0 * 256 + s1) << 16) + ((long long)s2 * 256 + s3);
          }
          const float s8 = __uint_as_float(v[n * D::NA + 8]), s9 = __uint_as_float(v[n * D::NA + 9]);
          h[1] += __float2int_rn(fmaf(s9, 0x1p-16f, s8 * 0x1p-8f));
          // hi + lo 2^-32 without integer conversions (both below 2^51)
          y[n] = (__longlong_as_double(0x4338000000000000ll + h[0]) - (6755399441055744.0 + 1572864.0)) +
                 __longlong_as_double(0x4138000000000000ll + h[1]);
        }
      }
    }
    if (rc[q] && have) {
      const int ia[3] = {bx + m % D::HX, by + (DIM == 3 ? (m / D::HX) % D::HY : m / D::HX),
                         DIM == 3 ? bz + m / (D::HX * D::HY) : 0};
      store_product<DIM, KIND>(g, a, ia, own[q], y, scale);
    }
    const unsigned left = __ballot_sync(0xffffffffu, rc[q] && !have);
    if (left) {
      int at = 0;
      if (lane == 0) at = atomicAdd(&snleft, __popc(left));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (rc[q] && !have) sleft[at + __popc(left & ((1u << lane) - 1u))] = (unsigned short)m;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (sfail) {
    // products may be on their way: the thread that issued them waits for them
    // and for what its commits have not signalled yet, before tensor and shared
    // memory are given back
    if (wib == 0 && elect_one()) {
      tc_commit(bar_drain);
      mbar_wait(bar_drain, 0u);
      for (int b = 0; b < 2 * D::NST + NDONE; ++b)
        if ((owed >> b) & 1u) mbar_wait(bar0 + 8 * b, (owed_parity >> b) & 1u);
    }
    __syncthreads();
  }
  if (digits && wib == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(D::TMEM) : "memory");
  // ---- the nodes that left the digits, in FP64 (the slot table takes W's place)
  const int nleft = snleft;
  if (nleft == 0) return;
  int* soff = reinterpret_cast<int*>(smem + D::O_ROWS);
  if constexpr (KIND == 0) {
    slot_table<DIM>(g, soff);
  } else if (nleft >= D::THREADS / 2) {
    // many: a thread each (1025 x 257 nodes at the solution, 10,000 nodes in few
    // tiles: 43 -> 34 us a launch)
    for (int t = tid; t < nleft; t += D::THREADS) {
      const int m = sleft[t];
      residual_node<DIM, 0, 1>(g, a.coef, a.mask, a.v, a.b, a.r, a.rpad, nullptr,
                               bx + m % D::HX + g.nn[0] * (by + m / D::HX), true);
    }
    return;
  }
  auto by_lanes = [&](auto lanes) {
    constexpr int L = decltype(lanes)::value;
    for (int base = 0; base < nleft; base += D::THREADS / L) {
      const int gi = base + tid / L;
      const bool valid = gi < nleft;
      const int m = sleft[valid ? gi : nleft - 1];
      const int i = bx + m % D::HX, j = by + (DIM == 3 ? (m / D::HX) % D::HY : m / D::HX);
      const int k = DIM == 3 ? bz + m / (D::HX * D::HY) : 0;
      const int node = i + g.nn[0] * (j + (DIM == 3 ? g.nn[1] : 1) * k);
      if constexpr (KIND == 0)
        apply_fp64_patch<DIM, L>(g, a.coef, a.mask, a.v, a.omega, a.x, a.prow, soff, (unsigned)node, valid);
      else
        residual_node<DIM, 0, L>(g, a.coef, a.mask, a.v, a.b, a.r, a.rpad, nullptr, node, valid);
    }
  };
  // (3D: 3.6 us for 8 nodes at a warp each, 13 us for 32 at 8 lanes)
  if (DIM == 3 && nleft <= 24) by_lanes(std::integral_constant<int, 32>());
  else by_lanes(std::integral_constant<int, TPP>());
}

// ---- plan ------------------------------------------------------------------

// class nodes: those whose whole box is in the grid, unconstrained and fluid
// (KIND 0: node classes over the 5^d box; KIND 1: the node's own class, free
// neighbours)
template <int DIM, int KIND>
__global__ void digit_class_kernel(LevelGeom g, const unsigned char* __restrict__ nclass,
                                   const unsigned char* __restrict__ mask, unsigned char* __restrict__ cls,
                                   int* __restrict__ rep) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (unsigned)g.nnodes) return;
  int ia[3];
  decode_node<DIM>(g, i, ia);
  constexpr int R = Dig<DIM, KIND>::R, RZ = DIM == 3 ? R : 0;
  bool c = nclass[i] == 1;
  for (int dz = -RZ; dz <= RZ && c; ++dz)
    for (int dy = -R; dy <= R && c; ++dy)
      for (int dx = -R; dx <= R && c; ++dx) {
        const int b0 = ia[0] + dx, b1 = ia[1] + dy, b2 = ia[2] + dz;
        if (b0 < 0 || b0 > g.n[0] || b1 < 0 || b1 > g.n[1] || (DIM == 3 && (b2 < 0 || b2 > g.n[2]))) { c = false; break; }
        const long long bn = b0 + (long long)g.nn[0] * (b1 + (long long)g.nn[1] * b2);
        if (mask[bn] & 7) c = false;
        if (KIND == 0 && nclass[bn] != 1) c = false;
      }
  cls[i] = c ? 1 : 0;
  if (c) atomicMin(rep, (int)i);
}

// KIND 1: a node whose stencil is not the representative's is no class node
template <int DIM>
__global__ void digit_compare_kernel(LevelGeom g, const double* __restrict__ st, unsigned char* __restrict__ cls,
                                     const int* __restrict__ rep) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (unsigned)g.nnodes) return;
  if (!cls[i]) return;
  const int r = *rep;
  constexpr int N = (DIM == 3 ? 27 : 9) * (2 * DIM + 2);
  bool same = true;
  for (int t = 0; t < N; ++t) same = same && st[(long long)t * g.nnodes + i] == st[(long long)t * g.nnodes + r];
  if (!same) cls[i] = 0;
}

// bit 1: a product reads the node; counts the class nodes
template <int DIM, int KIND>
__global__ void digit_tag_kernel(LevelGeom g, const unsigned char* __restrict__ in, unsigned char* __restrict__ out,
                                 int* __restrict__ count) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = 0;
  if (i < (unsigned)g.nnodes) {
    int ia[3];
    decode_node<DIM>(g, i, ia);
    constexpr int R = Dig<DIM, KIND>::R, RZ = DIM == 3 ? R : 0;
    int tag = 0;
    for (int dz = -RZ; dz <= RZ; ++dz)
      for (int dy = -R; dy <= R; ++dy)
        for (int dx = -R; dx <= R; ++dx) {
          const int b0 = ia[0] + dx, b1 = ia[1] + dy, b2 = ia[2] + dz;
          if (b0 < 0 || b0 > g.n[0] || b1 < 0 || b1 > g.n[1] || (DIM == 3 && (b2 < 0 || b2 > g.n[2]))) continue;
          tag |= in[b0 + (long long)g.nn[0] * (b1 + (long long)g.nn[1] * b2)] & 1;
        }
    c = in[i] & 1;
    out[i] = (unsigned char)(c | (tag << 1));
  }
  const int n = __popc(__ballot_sync(0xffffffffu, c != 0));
  if ((threadIdx.x & 31) == 0 && n) atomicAdd(count, n);
}

// counts the tiles that hold class nodes (a CTA each)
template <int DIM, int KIND>
__global__ void __launch_bounds__(128) digit_tiles_kernel(LevelGeom g, const unsigned char* __restrict__ cls, int tiles_x,
                                                          int tiles_y, int* __restrict__ count) {
  using D = Dig<DIM, KIND>;
  const int tq = blockIdx.x / tiles_x;
  const int b0 = blockIdx.x % tiles_x * D::TX + D::R, b1 = (DIM == 3 ? tq % tiles_y : tq) * D::TY + D::R;
  const int b2 = DIM == 3 ? tq / tiles_y * D::TZ + D::R : 0;
  bool any = false;
  for (int t = threadIdx.x; t < D::TX * D::TY * D::TZ; t += blockDim.x) {
    const int i = b0 + t % D::TX, j = b1 + t / D::TX % D::TY, k = b2 + t / (D::TX * D::TY);
    if (i < g.nn[0] && j < g.nn[1] && (DIM == 2 || k < g.nn[2]))
      any = any || (cls[i + (long long)g.nn[0] * (j + (long long)(DIM == 3 ? g.nn[1] : 1) * k)] & 1);
  }
  if (__syncthreads_or(any) && threadIdx.x == 0) atomicAdd(count, 1);
}

// the nodes without a class, in order
constexpr int kListBlock = 1024;
__global__ void digit_list_count_kernel(int n, const unsigned char* __restrict__ cls, int* __restrict__ counts) {
  __shared__ int sm;
  if (threadIdx.x == 0) sm = 0;
  __syncthreads();
  const int i = blockIdx.x * kListBlock + threadIdx.x;
  const int f = __popc(__ballot_sync(0xffffffffu, i < n && !(cls[i] & 1)));
  if ((threadIdx.x & 31) == 0) atomicAdd(&sm, f);
  __syncthreads();
  if (threadIdx.x == 0) counts[blockIdx.x] = sm;
}
// exclusive scan by one CTA
__global__ void __launch_bounds__(1024) digit_list_scan_kernel(int nb, int* __restrict__ counts) {
  __shared__ int sm[32];
  int run = 0;
  for (int b0 = 0; b0 < nb; b0 += 1024) {
    const int b = b0 + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int c = b < nb ? counts[b] : 0;
    int s = c;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane == 31) sm[w] = s;
    __syncthreads();
    int before = 0, total = 0;
    for (int k = 0; k < 32; ++k) {
      if (k < w) before += sm[k];
      total += sm[k];
    }
    if (b < nb) counts[b] = run + before + s - c;
    run += total;
    __syncthreads();
  }
}
__global__ void digit_list_place_kernel(int n, const unsigned char* __restrict__ cls, const int* __restrict__ offs,
                                        int* __restrict__ list) {
  __shared__ int sm[32];
  const int i = blockIdx.x * kListBlock + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool f = i < n && !(cls[i] & 1);
  const unsigned bal = __ballot_sync(0xffffffffu, f);
  if (lane == 0) sm[w] = __popc(bal);
  __syncthreads();
  int before = offs[blockIdx.x];
  for (int k = 0; k < w; ++k) before += sm[k];
  if (f) list[before + __popc(bal & ((1u << lane) - 1u))] = i;
}

// W in slot order (one CTA): the representative's cached rows or stencil; then
// scales, the right operand and the magnitudes.
template <int DIM, int KIND>
__global__ void __launch_bounds__(256)
    digit_rows_kernel(LevelGeom g, const double* __restrict__ src, const int* __restrict__ prow,
                      const int* __restrict__ rep, double* __restrict__ W, uint4* __restrict__ rows,
                      float4* __restrict__ wabs, unsigned short* __restrict__ chk, DigitScale* __restrict__ sc) {
  using D = Dig<DIM, KIND>;
  constexpr int ND = D::ND, NSLOT = D::NSLOT, NA = D::NA;
  const int tid = threadIdx.x;
  const int i = *rep;
  __shared__ int smax[4 + 2], sok;
  __shared__ int sdig[4][NA];  // sum over the slots of |digit|
  if (tid < 6) smax[tid] = -100000;
  if (tid < 4 * NA) sdig[tid / NA][tid % NA] = 0;
  if (tid == 0) sok = 1;
  __syncthreads();
  if (i == 0x7fffffff) {  // no class node
    if (tid == 0) {
      for (int r = 0; r < 4; ++r) {
        sc->rowexp[r] = 0;
        sc->floor[r] = 0.0f;
      }
      sc->delta = 0;
      sc->ok = 0;
    }
    return;
  }
  for (int t = tid; t < NSLOT * ND; t += blockDim.x) {
    const int j = t / ND, r = t % ND;
    int o[3], k, at;
    slot_of<DIM, KIND>(j, o, &k, &at);
    double v;
    if (KIND == 0) {
      const int pr = prow[i];
      v = src[((size_t)(pr < 0 ? -pr - 1 : pr) * NSLOT + at) * ND + r];
    } else {
      constexpr int SP = 2 * DIM + 2;
      const int nb = at / ND;
      int e = -1;  // velocity components do not couple
      if (r < DIM) e = k == r ? 0 : (k == DIM ? 1 + r : -1);
      else e = k < DIM ? 1 + DIM + k : 1 + 2 * DIM;
      v = e >= 0 ? src[((long long)nb * SP + e) * g.nnodes + i] : 0.0;
    }
    W[t] = v;
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    if (e == 0x7ff) sok = 0;
    if (e != 0 && (r < DIM) == (k < DIM)) atomicMax(&smax[r < DIM ? 4 : 5], e);
  }
  __syncthreads();
  const int eu = smax[4], ep = smax[5];
  const int d2 = eu > -100000 && ep > -100000 ? ep - eu : 0;
  const int delta = (d2 + (d2 < 0 ? -1 : 1)) / 2;
  for (int t = tid; t < NSLOT * ND; t += blockDim.x) {
    int o[3], k, at;
    slot_of<DIM, KIND>(t / ND, o, &k, &at);
    const int e = (__double2hiint(W[t]) >> 20) & 0x7ff;
    if (e != 0) atomicMax(&smax[t % ND], e - (k == DIM ? delta : 0));
  }
  __syncthreads();
  // right operand: per slot the columns r NA + d of eight values s, w_{d-s};
  // stored [step][slot of the pair][column][s]
  for (int t = tid; t < D::STEPS * 2 * D::N; t += blockDim.x) {
    const int slot = t / D::N, r = t % D::N / NA, d = t % D::N % NA;
    unsigned v[4] = {0u, 0u, 0u, 0u};
    if (slot < NSLOT && r < ND) {
      int o[3], k, at, dg[NA];
      slot_of<DIM, KIND>(slot, o, &k, &at);
      row_digits(W[(size_t)slot * ND + r], smax[r], k == DIM ? -delta : 0, dg);
      for (int s = 0; s < 8 && s <= d; ++s)
        v[s / 2] |= (unsigned)__half_as_ushort(__int2half_rn(dg[d - s])) << (16 * (s & 1));
      atomicAdd(&sdig[r][d], abs(dg[d]));
    }
    rows[t] = make_uint4(v[0], v[1], v[2], v[3]);
  }
  // magnitudes relative to the row's 2^Ew, at least 2^-22 where not zero (with
  // the smallest magnitude of a value the product is not zero either), slots by
  // their largest one, with their offset from a node in the tile
  __shared__ float skey[NSLOT];
  auto weight = [&](int j, float* m) {
    int o[3], k, at;
    slot_of<DIM, KIND>(j, o, &k, &at);
    for (int r = 0; r < 4; ++r) {
      const double v = r < ND ? W[(size_t)j * ND + r] : 0.0;
      m[r] = v != 0.0 ? fmaxf(magnitude(v, smax[r < ND ? r : 0], k == DIM ? -delta : 0), 0x1p-22f) : 0.0f;
    }
    return k * D::PLANE + (o[0] + D::R) + D::HX * ((o[1] + D::R) + (DIM == 3 ? D::HY * (o[2] + D::R) : 0));
  };
  for (int j = tid; j < NSLOT; j += blockDim.x) {
    float m[4];
    weight(j, m);
    skey[j] = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
  }
  __syncthreads();
  for (int j = tid; j < D::CHK; j += blockDim.x) {
    float m[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    int at = 0, rank = j;
    if (j < NSLOT) {
      at = weight(j, m);
      rank = 0;
      for (int i = 0; i < NSLOT; ++i) rank += skey[i] > skey[j] || (skey[i] == skey[j] && i < j);
    }
    wabs[rank] = make_float4(m[0], m[1], m[2], m[3]);
    chk[rank] = (unsigned short)at;
  }
  __syncthreads();
  if (tid < 4) {
    float sum = 0.0f;
    for (int t = 0; t < NSLOT; ++t) sum += tid == 0 ? wabs[t].x : tid == 1 ? wabs[t].y : tid == 2 ? wabs[t].z : wabs[t].w;
    sc->floor[tid] = ldexpf(sum, kFloor);
  }
  if (tid == 0) {
    for (int r = 0; r < 4; ++r) {
      const int e = r < ND && smax[r] > -100000 ? smax[r] - 1022 : 0;
      if (e < -400 || e > 400) sok = 0;
      sc->rowexp[r] = e;
      // |S_d| <= sum over s <= d of (sum |w_s|) max |v_{d-s}|; a leading digit is at most 64
      for (int d = 0; d <= (DIM == 3 ? 5 : NA - 1); ++d) {
        long long b = 0;
        for (int s = max(0, d - 7); s <= d; ++s) b += (long long)sdig[r][s] * (s == d ? 64 : 128);
        if (b >= (1 << 24)) sok = 0;
      }
    }
    if (delta < -200 || delta > 200) sok = 0;
    sc->delta = delta;
    sc->ok = sok;
  }
}

template <int DIM, int KIND>
void tiles_of(const LevelGeom& g, int* tx, int* ty, int* tz) {
  using D = Dig<DIM, KIND>;
  *tx = (g.nn[0] - 2 * D::R + D::TX - 1) / D::TX;
  *ty = (g.nn[1] - 2 * D::R + D::TY - 1) / D::TY;
  *tz = DIM == 3 ? (g.nn[2] - 2 * D::R + D::TZ - 1) / D::TZ : 1;
}

// Class nodes that a wave of tiles (one on every place of the GPU) has to take
// off the FP64 kernels to pay for its time.  GB300, measured where both sides
// are equal: 3D apply 16,300 to 18,500 a wave at 49^3, 57^3, 65^3, 73^3 and 81^3
// nodes with 0 to 100 spheres (49^3, 318 us in FP64: 0 spheres, 79,500 class
// nodes, 212; 12, 61,500, 251; 40, 26,000, 346.  65^3, 715 us: 0, 205,000, 364;
// 40, 102,000, 605; 100, 43,000, 753); 2D apply 37,000 and 2D operator 89,000 by
// the times of grids without obstacles (a wave 15 and 10 us).
template <int DIM, int KIND>
constexpr long long kPerWave = DIM == 3 ? 18500 : KIND == 0 ? 40000 : 100000;

// The plan's list in FP64.  A short one is taken by the first CTAs of the same
// launch (a launch less).  A long one has a launch of its own: beside tiles,
// whose shared memory leaves 24 warps an SM, it is bound by latency (326,000
// nodes of 1537^2, residual 205 us in one launch and 164 in two, patch apply
// 395 and 272; 36,000 of 513^2, 31 and 29, 49 and 52).  3D: always (a tile's
// CTA takes an SM's shared memory; run beside one, the FP64 products lost more
// to the smaller L1 than they gained).
constexpr long long kListLaunch = 65536;

template <int DIM>
__global__ void __launch_bounds__(256) residual_list_kernel(LevelGeom g, DigArgs a, int n, const int* __restrict__ list) {
  const int t = (int)(blockIdx.x * 256u + threadIdx.x);
  if (t < n) residual_node<DIM, 0, 1>(g, a.coef, a.mask, a.v, a.b, a.r, a.rpad, nullptr, list[t], true);
}

template <int DIM, int KIND>
cudaError_t run_product(const LevelGeom& g, const DigitPlan& p, DigArgs a, cudaStream_t s) {
  using D = Dig<DIM, KIND>;
  a.cls = p.cls;
  a.rows = p.rows;
  a.wabs = p.wabs;
  a.chk = p.chk;
  a.sc = p.sc;
  a.err = p.err;
  a.wait_ns = p.wait_ns;
  a.list = p.list;
  a.nlist = (int)p.nlist;
  if (DIM == 2 && p.nlist < kListLaunch) {
    a.list_blocks = (int)((p.nlist + 63) / 64);  // 4 lanes a node
  } else if (p.nlist > 0) {
    cudaError_t e;
    if constexpr (KIND == 0) {
      e = launch_patch_apply(g, FC_PREC_FP64, a.coef, a.mask, a.v, nullptr, a.omega, a.x, a.prow, s, p.list, p.nlist);
    } else {
      residual_list_kernel<DIM><<<(unsigned)((p.nlist + 255) / 256), 256, 0, s>>>(g, a, (int)p.nlist, p.list);
      note_launches(1);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
  }
  auto kern = digit_product_kernel<DIM, KIND>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D::BYTES);
  if (e != cudaSuccess) return e;
  int tx, ty, tz;
  tiles_of<DIM, KIND>(g, &tx, &ty, &tz);
  kern<<<(unsigned)a.list_blocks + (unsigned)tx * ty * tz, D::THREADS, D::BYTES, s>>>(g, a, tx, ty);
  note_launches(1);
  return cudaGetLastError();
}

template <int DIM, int KIND>
cudaError_t build_plan(const LevelGeom& g, const double* src, const unsigned char* nclass, const unsigned char* mask,
                       const int* prow, DigitPlan* p, const DigitScratch& t, cudaStream_t s) {
  using D = Dig<DIM, KIND>;
  const char* env = getenv("FC_DIGIT_WAIT_NS");
  p->wait_ns = env ? strtoull(env, nullptr, 10) : kWaitNs;
  const unsigned blocks = (unsigned)((g.nnodes + 255) / 256);
  const int n = (int)g.nnodes, nb = (n + kListBlock - 1) / kListBlock;
  const int init[3] = {0x7fffffff, 0, 0};  // representative, class nodes, tiles with some
  cudaError_t e = cudaMemcpyAsync(t.rep, init, sizeof(init), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  digit_class_kernel<DIM, KIND><<<blocks, 256, 0, s>>>(g, nclass, mask, t.cls, t.rep);
  if (KIND == 1) digit_compare_kernel<DIM><<<blocks, 256, 0, s>>>(g, src, t.cls, t.rep);
  digit_tag_kernel<DIM, KIND><<<blocks, 256, 0, s>>>(g, t.cls, p->cls, t.rep + 1);
  int tx, ty, tz;
  tiles_of<DIM, KIND>(g, &tx, &ty, &tz);
  if (tx > 0 && ty > 0 && tz > 0)
    digit_tiles_kernel<DIM, KIND><<<(unsigned)tx * ty * tz, 128, 0, s>>>(g, p->cls, tx, ty, t.rep + 2);
  digit_list_count_kernel<<<nb, kListBlock, 0, s>>>(n, p->cls, t.counts);
  digit_list_scan_kernel<<<1, 1024, 0, s>>>(nb, t.counts);
  digit_list_place_kernel<<<nb, kListBlock, 0, s>>>(n, p->cls, t.counts, p->list);
  digit_rows_kernel<DIM, KIND><<<1, 256, 0, s>>>(g, src, prow, t.rep, t.w, p->rows, p->wabs, p->chk, p->sc);
  note_launches(7 + KIND);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  int got[2] = {0, 0}, dev = 0, nsm = 0;
  e = cudaMemcpyAsync(got, t.rep + 1, sizeof(got), cudaMemcpyDeviceToHost, s);
  DigitScale sc;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&sc, p->sc, sizeof(sc), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  p->nlist = g.nnodes - got[0];
  const long long places = std::max(1, D::PER_SM * nsm);
  p->on = sc.ok && got[0] > 0 && got[0] >= kPerWave<DIM, KIND> * ((got[1] + places - 1) / places);
  return e;
}

}  // namespace

size_t digit_plan_rows_bytes(int dim, int kind) {
  return dim == 3 ? (size_t)Dig<3, 0>::STEPS * Dig<3, 0>::STEPB
                  : kind == 0 ? (size_t)Dig<2, 0>::STEPS * Dig<2, 0>::STEPB : (size_t)Dig<2, 1>::STEPS * Dig<2, 1>::STEPB;
}
int digit_plan_slots(int dim, int kind) {
  return dim == 3 ? Dig<3, 0>::CHK : kind == 0 ? Dig<2, 0>::CHK : Dig<2, 1>::CHK;
}
int digit_plan_counts(long long nnodes) { return (int)((nnodes + kListBlock - 1) / kListBlock); }

cudaError_t build_digit_plan(const LevelGeom& g, int kind, const double* src, const unsigned char* nclass,
                             const unsigned char* mask, const int* prow, DigitPlan* p, const DigitScratch& t,
                             cudaStream_t s) {
  if (g.dim == 2)
    return kind == 0 ? build_plan<2, 0>(g, src, nclass, mask, prow, p, t, s)
                     : build_plan<2, 1>(g, src, nclass, mask, prow, p, t, s);
  return build_plan<3, 0>(g, src, nclass, mask, prow, p, t, s);
}

cudaError_t launch_digit_apply(const LevelGeom& g, const DigitPlan& p, const double* coef, const unsigned char* mask,
                               const double* rpad, double omega, double* x, const int* prow, cudaStream_t s) {
  DigArgs a{};
  a.v = rpad;
  a.x = x;
  a.omega = omega;
  a.coef = coef;
  a.mask = mask;
  a.prow = prow;
  return g.dim == 2 ? run_product<2, 0>(g, p, a, s) : run_product<3, 0>(g, p, a, s);
}

cudaError_t launch_digit_residual(const LevelGeom& g, const DigitPlan& p, const double* st, const unsigned char* mask,
                                  const double* x, const double* b, double* r, double* rpad, cudaStream_t s) {
  DigArgs a{};
  a.v = x;
  a.b = b;
  a.r = r;
  a.rpad = rpad;
  a.coef = st;
  a.mask = mask;
  return run_product<2, 1>(g, p, a, s);
}

}  // namespace fc
