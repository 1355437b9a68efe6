// FP64 matrix products of the FP64 form on the tensor cores.
//
// GB300 issues about two FP64 multiply-adds per SM and clock (1.2 TFLOP/s for the chip), so a
// contraction of the FP64 form is bound by the FP64 pipe 50 to 100 times above the time its
// bytes take.  Here each real operand is cut into eight signed 8-bit digits, the digit
// products run as BF16 MMAs on tcgen05 and are summed as integers (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 95 (2012)):
//
//   x = 2^(e - 1084) sum_s d_s 256^(7 - s),  |d_s| <= 128, |d_0| <= 64,
//
// with one exponent e per row of A (column of B) and segment of the contraction (at most 256 terms), the one
// of its largest entry there: an entry is held to 2^-62 of 2^e.  Digits are small integers, exact in BF16.  The products
// d_s d'_t of one order o = s + t have one common weight 256^-o and a TMEM accumulator of their own; orders
// 0..7 are formed (36 MMAs per 16-element K step).  The dropped ones weigh at most 2^-57 of 2^e 2^e' per term (typically 2^-60).
// An FP32 accumulator is exact while its sum of integers stays up to 2^24: at most o + 1 products of 2^14 (2^13 with a
// leading digit) over 256 terms, so the orders 0..4 never round, and 5..7 do so only where the digits of nearly every term are
// close to 128 and of one sign, by a few units of 2^-50 2^e 2^e'.  At the end of
// a segment the accumulators go into 64-bit integers (hi: orders 0..3, lo: orders 4..7), whose sum is
// rounded once to FP64; the segments of a long contraction are added in FP64.  (One exponent for a whole row
// of 32768 terms lost a factor ten against FP64 multiply-adds in the gradients of sparse cotangents.)
//
// All this is relative to the largest entries, while FP64 multiply-adds err by parts of sum |a| |b|, which is far
// smaller where entries of very different size meet: far from the diagonal of decaying matrices, beside one huge matrix
// element, in the imaginary parts of nearly real data.  So one more MMA per K step sums the magnitudes, as BF16
// numbers (magnitude()), and an element with 0 < sum |a| |b| < 2^e 2^e' / 16 is taken from FP64 multiply-adds instead
// (plain_elements(), and the reduction of long contractions).  From that line on the digits err by at most n 2^-53 sum |a| |b|
// over the n <= 256 terms of the segment, the a-priori bound of n multiply-adds; at the line typically by 1.5 of 2^-53 sum |a| |b|
// (multiply-adds: 0.3 for terms of mixed sign, 0.4 sqrt(n / 3) for one sign), above it by less in proportion.
// Seeded bases have 1e-6 or fewer such elements, up to one in 200 in the source term at times when n is nearly 1/2 (GW, nb = 64:
// mode products 370 us, 470 on average in such a step).  Sparse or decaying operands have as many as they need: the 4 x 4
// cluster (noise of 1e-17 beside entries of 1) one in ten, for which its gradients take 68 ms instead of 31 with none (160 with
// all products on the CUDA cores).
//
// Against an extended-precision reference the right-hand side of a seeded basis at nb = 24 errs by 2.6e-16 (GW) and 3.8e-16
// (TPP, complex w) in the 2-norm; FP64 multiply-adds by 6.2e-16 and 9.3e-16, plain FP64 torch by 6.0e-16 and 9.0e-16.
//
// The digits are cut on the integer pipe, and the sums converted on both (fixed_to_double_*): FP64 instructions
// alone would cost as much as the MMAs (two per SM and clock).  A row or column that holds an Inf or a NaN has
// no digits; its elements are taken from FP64 multiply-adds too.
#include "g1g2_internal.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <new>
#include <type_traits>

namespace g1g2 {

namespace {

using namespace tc;

constexpr int kDig = 8;                    // digits per real operand
constexpr int kOrd = 8;                    // orders of digit products
// A row's exponent comes with the number of its real terms that are not zero
constexpr int kExpBits = 11, kExpMask = (1 << kExpBits) - 1;
constexpr int kTM = 128;                   // rows of A per tile (TMEM lanes)
constexpr int kTNMax = 128;                // real columns per tile, at most
constexpr int kKB = 16;                    // K elements per block: one MMA step, 32-byte rows
constexpr int kSeg = 16;                   // K blocks of a segment (256 terms)
constexpr uint32_t kADig = kTM * 32;       // one digit plane of an A block: 4 KB
constexpr int kStages = 3;
constexpr int kEpiWarps = 12;              // 128 registers per thread (16 warps: 96, spilled in the epilogue's loop, 412 us
                                           // instead of 346 per mode product at nb = 64; 8 warps: 378 us)
constexpr int kThreads = 64 + 32 * kEpiWarps;   // loader warp, MMA warp, epilogue warps
constexpr int kPerQuarter = kEpiWarps / 4;        // epilogue warps per quarter of the TMEM lanes
constexpr int kMaxGroups = (kTNMax / 8 + kPerQuarter - 1) / kPerQuarter;   // groups of eight columns per epilogue warp
static_assert(kMaxGroups * 4 <= 32, "one lane per column exponent");
constexpr int kStgPitch = 5;               // complex per staged row (4 used)
constexpr uint32_t kStgWarp = 32 * kStgPitch * 16;
// A and B blocks (at most 128 columns) per stage, and the staging tiles
constexpr size_t kSmem = 1024 + kStages * 2 * kDig * kADig + kEpiWarps * kStgWarp + 256;
static_assert(kSmem <= 227 * 1024, "shared memory of a CTA");

constexpr int kNonFinite = 2047;           // row exponent of a row with an Inf or a NaN
constexpr int kZeroRow = 1023;             // of a row of zeros (any other would do: its digits are zero)
constexpr int kSafeLo = 600, kSafeHi = 1450;   // rows and columns in this range have kMinE <= e <= kMaxE (see fixed_to_double_*)

// ---------------------------------------------------------------------------
// Digits
// ---------------------------------------------------------------------------
// One strided complex operand: row r = (b, x) with x < X, element k at p[b sb + x sx + (k / kin) kout + (k % kin) sk].
struct Operand {
  const cplx *p;
  long long sb, sx, sk, kout;
  int X, kin;
  int rows, K;
  int conj;
};
__device__ __forceinline__ long long row_offset(const Operand &o, int r) {
  const int b = r / o.X;
  return (long long)b * o.sb + (long long)(r - b * o.X) * o.sx;
}
__device__ __forceinline__ long long k_offset(const Operand &o, int k) {
  const int b = k / o.kin;
  return (long long)b * o.kout + (long long)(k - b * o.kin) * o.sk;
}

// The digits of x at row exponent emax as one word: d_s + 128 is byte 7 - s (a balanced base-256 expansion is the plain
// one of X + 128 (256^0 + ..)).  X = x 2^(1084 - emax) to nearest, |X| < 2^62, so |d_0| <= 64.
__device__ __forceinline__ unsigned long long digits(double x, int emax) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32) | lo;
  unsigned long long q;                      // floor(2 |X|); shifts of 64 and more give 0
  asm("shr.u64 %0, %1, %2;" : "=l"(q) : "l"(m << 10), "r"(emax - max(e, 1)));
  q = (q + 1) >> 1;
  const long long s = (long long)((int)hi >> 31);
  return (q ^ (unsigned long long)s) + (0x8080808080808080ull - (unsigned long long)s);
}

// |x| 2^(1023 - emax) cut to BF16, at least 2^-60 unless x is zero.  A sum of products of these is a lower bound of
// sum |a| |b| in units of the two rows' exponents (the floor adds less than 2^-50), and zero only if every product is.
__device__ __forceinline__ uint32_t magnitude(double x, int emax) {
  const uint32_t hi = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  const int v = hi >= 0x100000u ? (int)(hi >> 13) - ((emax - 127) << 7) : 0;   // a subnormal x: the floor
  return (hi | (uint32_t)__double2loint(x)) == 0 ? 0u : (uint32_t)max(v, (127 - 60) << 7);
}

// d_s of two neighbouring elements as a BF16 pair.  A byte b = d + 128 below 128 becomes (128 + b) - 256, one from 128 on
// b - 128, where 128 + (b mod 128) is a BF16 number with the seven low bits of b as its mantissa: both differences are exact.
template <int S>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long a, unsigned long long b) {
  constexpr int byte = kDig - 1 - S;
  const uint32_t wa = byte < 4 ? (uint32_t)a : (uint32_t)(a >> 32), wb = byte < 4 ? (uint32_t)b : (uint32_t)(b >> 32);
  const uint32_t w = __byte_perm(wa, wb, (byte & 3) | (4 | (byte & 3)) << 8);
  uint32_t d;
  asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"((w & 0x007f007fu) | 0x43004300u), "r"((w & 0x00800080u) ^ 0x43804380u));
  return d;
}

// Digit planes in global memory, ready for the MMA: block (tile of TR rows, K block) holds kDig planes
// of TR rows x 32 bytes in the 32-byte-swizzled K-major layout, so that the GEMM brings the leading planes
// of a block in with one contiguous bulk copy and no tensor map.  The plane of magnitudes is an array of its own: those
// of eight K blocks come with one copy.
__device__ __forceinline__ void store_digits(uint8_t *out, uint8_t *mag, int TR, int KB, int row, int q,
                                             const unsigned long long (&w)[8], uint32_t flip, const uint4 &m) {
  const int tile = row / TR, rr = row - tile * TR, kb = q >> 1, c2 = q & 1;
  const uint32_t plane = (uint32_t)TR * 32;
  const size_t block = (size_t)tile * KB + kb, at = rr * 32 + ((c2 ^ ((rr >> 2) & 1)) << 4);
  uint8_t *o = out + block * (kDig * plane) + at;
#define G1G2_PUT(S)                                                                              \
  *reinterpret_cast<uint4 *>(o + S * plane) =                                                    \
      make_uint4(digit_pair<S>(w[0], w[1]) ^ flip, digit_pair<S>(w[2], w[3]) ^ flip,             \
                 digit_pair<S>(w[4], w[5]) ^ flip, digit_pair<S>(w[6], w[7]) ^ flip)
  G1G2_PUT(0); G1G2_PUT(1); G1G2_PUT(2); G1G2_PUT(3); G1G2_PUT(4); G1G2_PUT(5); G1G2_PUT(6); G1G2_PUT(7);
#undef G1G2_PUT
  *reinterpret_cast<uint4 *>(mag + block * plane + at) = m;
}

// How a complex operand becomes real rows:
//   kRows    row r: [re | im] along K' (the A side of a complex product)
//   kReal    rows 2 r, 2 r + 1: [re | -im], [im | re] (its B side: columns re, im of the product)
//   kPlanes  rows 2 r, 2 r + 1: re, im over K (both sides of a long contraction; the four
//            real products are combined at the end)
enum Form : int { kRows = 0, kReal = 1, kPlanes = 2 };

constexpr int kCutVals = 4096;   // complex values of an operand per CTA: one segment of kCutVals / K rows
__host__ __device__ constexpr int seg_k(int form) { return form == kPlanes ? 256 : 128; }   // operand K values per segment
__host__ __device__ constexpr int cut_rows(int form) { return kCutVals / seg_k(form); }

// Cuts rows x K of an operand into digits and magnitudes, and finds the exponents and the numbers of nonzero terms.  A CTA
// stages one segment of 32 rows (16 for kPlanes) in shared memory, read along whichever index is contiguous in memory, takes
// the largest exponent of each row there, and every thread then cuts eight consecutive K values of one row at a time into nine
// 16-byte stores; a warp writes 16 rows x 32 bytes, 512 contiguous bytes, per plane.  Bound by its 16
// bytes read and 36 written per complex element (72 for kReal).  The phases of a CTA only overlap with those of others:
// five CTAs per SM.  nb = 64 operand (268 MB read, 604 MB written): 181 us (4.8 TB/s); six CTAs (40 registers) 180,
// but 203 instead of 199 in GW products and 15.6 instead of 15.2 at nb = 27.
struct CutJob {
  Operand o;               // o.rows: rows of the panel
  int r_begin, TR;
  int *rexp;
  uint8_t *out, *mag;
};
template <int FORM>
__device__ __forceinline__ void cut_digits(const CutJob &job, int block, int k_begin, int Klen, int Kp, int KB, int SK) {
  constexpr int SR = cut_rows(FORM);
  extern __shared__ double sh[];
  __shared__ long long roff[SR], koff[seg_k(FORM)];
  __shared__ int emax[SR];
  const Operand &A = job.o;
  const int r_begin = job.r_begin, TR = job.TR;
  int *__restrict__ rexp = job.rexp;
  uint8_t *__restrict__ out = job.out, *__restrict__ mag = job.mag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = block * SR;                              // within the panel
  const int nr = min(SR, A.rows - r0);                    // A.rows: rows of the panel
  const int seg = blockIdx.y, k0 = seg * SK;
  const int kt = min(SK, Kp - k0);                        // padded K values of this segment (multiple of 8)
  const int pitch = kt + 1;
  double *re = sh, *im = sh + SR * pitch;
  if (tid < SR) roff[tid] = row_offset(A, r_begin + r0 + min(tid, nr - 1));
  if (tid < SK) koff[tid] = (k0 + tid < Klen) ? k_offset(A, k_begin + k0 + tid) : -1;
  __syncthreads();
  const int flip_im = A.conj ? (int)0x80000000u : 0;
  // kLoads loads in flight per thread, consecutive lanes along the index that is contiguous in memory
  constexpr int kLoads = 4;
  const int total = SR * kt;
  const unsigned inv = ((1u << 22) + kt - 1) / kt;        // idx / kt = idx inv >> 22 for idx kt < 2^22
  const cplx *p = A.p;
  for (int i0 = tid; i0 < total; i0 += 256 * kLoads) {
    cplx v[kLoads];
    int at[kLoads];
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      const int idx = i0 + 256 * i;
      int r, k;
      if (A.sk == 1) { r = (int)((unsigned)idx * inv >> 22); k = idx - r * kt; }
      else { k = idx / SR; r = idx % SR; }
      at[i] = r * pitch + k;
      v[i] = {0.0, 0.0};
      if (idx < total && koff[k] >= 0) v[i] = p[roff[r] + koff[k]];
    }
#pragma unroll
    for (int i = 0; i < kLoads; ++i) {
      if (i0 + 256 * i < total) {
        re[at[i]] = v[i].x;
        im[at[i]] = __hiloint2double(__double2hiint(v[i].y) ^ flip_im, __double2loint(v[i].y));
      }
    }
  }
  __syncthreads();
  {
    constexpr int T = 256 / SR;                           // threads per row
    const int r = tid / T, j = tid % T;
    int e = 0, terms = 0;
    for (int k = j; k < kt; k += T) {
      const double x = re[r * pitch + k], y = im[r * pitch + k];
      const int hx = __double2hiint(x) & 0x7fffffff, hy = __double2hiint(y) & 0x7fffffff;
      const int nx = (hx | __double2loint(x)) != 0, ny = (hy | __double2loint(y)) != 0;
      e = max(e, max(hx, hy));
      terms += nx + ny;
    }
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) {
      e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
      terms += __shfl_xor_sync(0xffffffffu, terms, o);
    }
    e = terms == 0 ? kZeroRow : max(e >> 20, 1);
    if (j == 0) {
      emax[r] = e;
      if (r < nr) rexp[(size_t)seg * A.rows + r0 + r] = e | terms << kExpBits;
    }
  }
  __syncthreads();
  const int c2 = lane & 1, rs = lane >> 1;
  const int nch = kt >> 3;                                // chunks of 8 per plane; pairs of them over both planes
  for (int g = warp; g < nch * (SR / 16); g += 8) {
    const int r = (g % (SR / 16)) * 16 + rs, qq = (g / (SR / 16)) * 2 + c2;
    const int u = qq >= nch ? 1 : 0, kc = qq - u * nch;
    if (r >= nr) continue;
    const double *src = (u ? im : re) + r * pitch + kc * 8;
    const int e = emax[r];
    unsigned long long w[8];
    uint32_t mg[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double x = e == kNonFinite ? 0.0 : src[i];
      w[i] = digits(x, e);
      mg[i / 2] = i & 1 ? mg[i / 2] | magnitude(x, e) << 16 : magnitude(x, e);
    }
    const uint4 m = make_uint4(mg[0], mg[1], mg[2], mg[3]);
    const int q0 = seg * (SK / (FORM == kPlanes ? 8 : 4)), row = r0 + r;          // 16-byte chunks before this segment
    if (FORM == kRows) {
      store_digits(out, mag, TR, KB, row, q0 + u * nch + kc, w, 0u, m);
    } else if (FORM == kReal) {
      store_digits(out, mag, TR, KB, 2 * row, q0 + u * nch + kc, w, u ? 0x80008000u : 0u, m);
      store_digits(out, mag, TR, KB, 2 * row + 1, q0 + (1 - u) * nch + kc, w, 0u, m);
    } else {
      store_digits(out, mag, TR, KB, 2 * row + u, q0 + kc, w, 0u, m);
    }
  }
}

// Both operands of a product in one launch: blocks below xblocks cut x, the others y.  (The column operand is small: as
// a launch of its own it took 5 us of the 50 us of a mode product at nb = 32.)
template <int FX, int FY>
__global__ void __launch_bounds__(256, 5) cut_digits_kernel(const CutJob x, const CutJob y, int xblocks, int k_begin, int Klen,
                                                         int Kp, int KB, int SK) {
  dependent_begin();
  if ((int)blockIdx.x < xblocks) cut_digits<FX>(x, blockIdx.x, k_begin, Klen, Kp, KB, SK);
  else cut_digits<FY>(y, blockIdx.x - xblocks, k_begin, Klen, Kp, KB, SK);
}

// ---------------------------------------------------------------------------
// GEMM
// ---------------------------------------------------------------------------
struct TcGemm {
  const uint8_t *A, *B;       // digit blocks
  const uint8_t *MA, *MB;     // magnitudes
  int KB, segs, kseg;         // K blocks of a row tile, in segments of kseg
  int nt;                     // real columns per tile (multiple of 16)
  int mtiles, ntiles;         // unit = (split mtiles + m_tile) ntiles + n_tile
  int splits, segs_per_split; // long contractions: segments cut over the units
  int *err;
  long long *sums;            // per CTA: [hi, lo][column][row] of a segment
  double *part;               // FP64 sums over segments [unit (long contractions) or CTA][column][row]
  int accumulate;             // long contractions: part holds earlier panels
  uint32_t *flags, *any;      // long contractions: masks of the elements left to the reduction, [tile][column group][row][segment],
                              // and their union over the segments of a unit, [unit][column group][row]
  int all_segs, seg_begin;    // segments of all panels, the first one of this panel
  Operand X, Y;               // rows r_begin + m of X, columns y_begin + y of Y, K from k_begin
  const int *ex, *ey;         // exponents [segment][row of the panel]
  int exs, eys;               // rows of the panel
  int r_begin, y_begin, k_begin;
  int rows, cols;             // complex rows and columns of this panel
  cplx *C;
  long long scb, scx, scy;
  int unit_alpha;             // alpha = i^unit_alpha
  int beta;                   // 0 or 1
};

// K-major operand tile with 32-byte rows and 32-byte swizzling (8-row atoms of 256 bytes)
__device__ __forceinline__ uint64_t smem_desc_sw32(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);          // start address
  d |= (uint64_t)1 << 16;                            // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(256u >> 4) << 32;                  // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                            // descriptor version
  d |= (uint64_t)6 << 61;                            // 32-byte swizzle
  return d;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
// the loaded registers carry no value before the wait: tie them to a point after it
__device__ __forceinline__ void after_wait(uint32_t (&r)[8]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Whether s = sum |a| |b|, in units of the two rows' exponents, is too small for the digits: below it their error may pass
// n 2^-53 s (see the head of the file)
__device__ __forceinline__ bool too_small(float s) { return s > 0.f && s < 0.0625f; }

// (hi 2^32 + lo) 2^e as FP64, rounded to nearest, without a branch, for |hi| < 2^62, |lo| < 2^62 and kMinE <= e <= kMaxE (no
// subnormal or infinite result then).  Two forms, because either alone is bound by its own pipe:
//   fixed_to_double_add: the upper 52 bits and the lower 44 as mantissas at 1.5 2^96 and 1.5 2^52; two FP64 additions
//       (64 cycles of the FP64 pipe per warp each), the first exact, and ten integer instructions;
//   fixed_to_double_int: the 96-bit magnitude is shifted left to its leading one by whole words and a funnel shift: about
//       forty integer instructions.
// The real parts take the one and the imaginary parts the other; long contractions, which add segments up on the FP64 pipe,
// the second alone.  Mode product at nb = 64 (seven digits), us: additions only 378, integers only 343, both 341.
constexpr int kMinE = -1022, kMaxE = 927;
__device__ __forceinline__ double fixed_to_double_add(long long hi, long long lo, int e) {
  hi += lo >> 32;
  const int es = e << 20;
  const double x0 = __hiloint2double((int)((0x43380000u + (uint32_t)es) | ((uint32_t)hi & 0xfffu)), (int)(uint32_t)lo);
  const long long top = hi >> 12;
  const double x1 = __longlong_as_double(top + ((long long)(0x45F80000 + es) << 32));
  const double c = __hiloint2double(0x45F80000 + es, 0x180);   // 1.5 2^96 + 1.5 2^52
  return __dadd_rn(__dsub_rn(x1, c), x0);
}
__device__ __forceinline__ double fixed_to_double_int(long long hi, long long lo, int e) {
  hi += lo >> 32;
  uint32_t w0 = (uint32_t)lo;
  const uint32_t s = (uint32_t)(int)(hi >> 63);
  w0 = (w0 ^ s) - s;
  hi = (hi ^ (long long)(int)s) + ((s & 1u) & (w0 == 0 ? 1u : 0u));
  uint32_t w2 = (uint32_t)(hi >> 32), w1 = (uint32_t)hi;
  int p = 1022 + 95 + e;                         // biased exponent - 1 of the result, minus the shift
  if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; p -= 32; }
  if (w2 == 0) { w2 = w1; w1 = 0; p -= 32; }
  const int lz = __clz((int)w2);
  const uint32_t t1 = __funnelshift_l(w1, w2, lz), t0 = __funnelshift_l(w0, w1, lz);
  p -= lz;
  uint32_t mhi = t1 >> 11, mlo = __funnelshift_r(t0, t1, 11);
  const uint32_t up = (t0 >> 10) & 1u;
  mlo += up;
  mhi += (mlo < up) ? 1u : 0u;
  const uint32_t out = w2 == 0 ? 0u : ((mhi + ((uint32_t)p << 20)) | (s & 0x80000000u));
  return __hiloint2double((int)out, (int)mlo);
}
// 2^k times a result at the end of that range, for any other e (a subnormal result is rounded a second time)
__device__ __noinline__ double beyond_range(double x, int k) { return ldexp(x, k); }

// alpha z for alpha = i^u: signs by the integer pipe
__device__ __forceinline__ cplx mul_unit(cplx z, int u) {
  const uint32_t sx = (u == 1 || u == 2) ? 0x80000000u : 0u, sy = (u >= 2) ? 0x80000000u : 0u;   // of the results
  const double x = (u & 1) ? z.y : z.x, y = (u & 1) ? z.x : z.y;
  return {__hiloint2double(__double2hiint(x) ^ sx, __double2loint(x)),
          __hiloint2double(__double2hiint(y) ^ sy, __double2loint(y))};
}

__device__ __forceinline__ bool is_zero(const cplx &v) {   // on the integer pipe
  return (((__double2hiint(v.x) | __double2hiint(v.y)) & 0x7fffffff) | __double2loint(v.x) | __double2loint(v.y)) == 0;
}
__device__ __forceinline__ bool is_finite(const cplx &v) {
  return max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff) < 0x7ff00000;
}
__device__ __forceinline__ double flip(double v, int sign) {
  return __hiloint2double(__double2hiint(v) ^ sign, __double2loint(v));
}
// s += u v, conjugated where fu, fv is the sign bit
__device__ __forceinline__ void plain_fma(cplx &s, const cplx &u, const cplx &v, int fu, int fv) {
  const double ui = flip(u.y, fu), vi = flip(v.y, fv);
  s = {fma(u.x, v.x, fma(-ui, vi, s.x)), fma(u.x, vi, fma(ui, v.x, s.y))};
}
// One segment (k0..k1) of the elements that the digits do not give, by FP64 multiply-adds, into the slots of their high
// sums: bit c = 4 i + j of a lane's mask is complex column y0 + 12 i + j of its row, xt the terms of that row that are not
// zero, yt those of column c = lane.  Three ways, by the cycles that they keep the FP64 pipe busy (64 per warp and term, 32 per
// sum over two lanes): a row at a time with the columns over the lanes and a column with the rows over the lanes, which
// leave terms with a zero out (such operands are mostly sparse; not with an Inf or a NaN among them), and a list of
// elements, each over as many lanes as there are for it.  (One element of the list after another, its terms over the whole
// warp, waited for memory: one in 400 elements took a product at nb = 64 from 371 to 920 us, now to 620.  Columns four at a time,
// all their terms looked at, took 137 us per mode product of the 4 x 4 cluster, now 79.)
__device__ __noinline__ void plain_elements(const TcGemm &p, uint32_t mask, bool finite, int xt, int yt, int row0, int y0, int k0,
                                            int k1, uint16_t *list, long long *hi) {
  const int lane = threadIdx.x & 31, K = k1 - k0;
  const Operand &X = p.X, &Y = p.Y;
  const int fx = X.conj ? (int)0x80000000u : 0, fy = Y.conj ? (int)0x80000000u : 0;
  auto row = [&](int m) { return X.p + row_offset(X, p.r_begin + min(m, p.rows - 1)); };   // lanes beyond the panel: its last
  auto put = [&](int y, int r, const cplx &s) {
    __stcg(hi + (size_t)(2 * y) * kTM + r, __double_as_longlong(s.x));
    __stcg(hi + (size_t)(2 * y + 1) * kTM + r, __double_as_longlong(s.y));
  };
  const uint32_t cols = __reduce_or_sync(0xffffffffu, mask);
  const int total = __reduce_add_sync(0xffffffffu, __popc(mask));
  const int by_rows = __reduce_add_sync(0xffffffffu, mask ? min(K, xt) : 0);
  const int by_cols = __reduce_add_sync(0xffffffffu, cols >> lane & 1u ? min(K, yt) : 0);
  int L = 1;                                                       // lanes per element of the list
  while (L < 32 && 2 * L * total <= 32) L *= 2;
  const int listed = (total * L + 31) / 32 * ((K + L - 1) / L + (31 - __clz(L)) / 2);
  __syncwarp();
  if (listed <= min(by_rows, by_cols)) {
    int at = __popc(mask);
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const int v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    at -= __popc(mask);
    for (uint32_t b = mask; b; b &= b - 1) list[at++] = (uint16_t)(lane | (__ffs((int)b) - 1) << 5);
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < total; i += 32 / L) {
      const int e = i + lane / L, c = list[min(e, total - 1)], r = c & 31, y = 4 * kPerQuarter * (c >> 7) + ((c >> 5) & 3);
      const cplx *a = row(row0 + r), *b = Y.p + row_offset(Y, p.y_begin + y0) + y * Y.sx;
      cplx s = {0.0, 0.0};
#pragma unroll 4
      for (int k = k0 + lane % L; k < k1; k += L) plain_fma(s, a[k * X.sk], b[k * Y.sk], fx, fy);
      for (int o = L / 2; o > 0; o /= 2) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
      }
      if (lane % L == 0 && e < total) put(y, r, s);
    }
  } else if (by_rows < by_cols) {
    const int y = 4 * kPerQuarter * (lane >> 2) + (lane & 3);      // this lane's column
    const cplx *b = Y.p + row_offset(Y, p.y_begin + y0) + y * Y.sx;
    uint32_t rows = __ballot_sync(0xffffffffu, mask != 0);
    int r = __ffs((int)rows) - 1, kb = k0;
    auto load = [&]() { return kb + lane < k1 ? row(row0 + r)[(kb + lane) * X.sk] : cplx{0.0, 0.0}; };
    cplx next = load(), s = {0.0, 0.0};
    while (r >= 0) {
      const cplx u = next;
      const int r_now = r, kb_now = kb;
      kb += 32;
      if (kb >= k1) {                                              // the next row's terms are loaded ahead
        kb = k0;
        rows &= rows - 1;
        r = __ffs((int)rows) - 1;
      }
      if (r >= 0) next = load();
      const bool mine = __shfl_sync(0xffffffffu, mask, r_now) >> lane & 1u;
      uint32_t nz = __ballot_sync(0xffffffffu, kb_now + lane < k1 && !(finite && is_zero(u)));
      for (; nz; nz &= nz - 1) {
        const int q = __ffs((int)nz) - 1;
        const cplx uq = {__shfl_sync(0xffffffffu, u.x, q), __shfl_sync(0xffffffffu, u.y, q)};
        if (mine) plain_fma(s, uq, b[(kb_now + q) * Y.sk], fx, fy);
      }
      if (kb == k0) {
        if (mine) put(y, r_now, s);
        s = {0.0, 0.0};
      }
    }
  } else {
    const cplx *a = row(row0 + lane), *b = Y.p + row_offset(Y, p.y_begin + y0);
    uint32_t rest = cols;
    int c = __ffs((int)rest) - 1, kb = k0;
    auto column = [&](int i) { return 4 * kPerQuarter * (i >> 2) + (i & 3); };
    auto load = [&]() { return kb + lane < k1 ? b[column(c) * Y.sx + (kb + lane) * Y.sk] : cplx{0.0, 0.0}; };
    cplx next = load(), s = {0.0, 0.0};
    while (c >= 0) {
      const cplx v = next;
      const int c_now = c, kb_now = kb;
      kb += 32;
      if (kb >= k1) {                                              // the next column's terms are loaded ahead
        kb = k0;
        rest &= rest - 1;
        c = __ffs((int)rest) - 1;
      }
      if (c >= 0) next = load();
      const bool mine = mask >> c_now & 1u;
      uint32_t nz = __ballot_sync(0xffffffffu, kb_now + lane < k1 && !(finite && is_zero(v)));
      while (nz) {
        constexpr int kAhead = 4;                                  // rows' terms on their way
        int q[kAhead];
        cplx u[kAhead];
#pragma unroll
        for (int t = 0; t < kAhead; ++t) {
          q[t] = __ffs((int)nz) - 1;
          nz &= nz - 1;
          u[t] = (mine && q[t] >= 0) ? a[(kb_now + q[t]) * X.sk] : cplx{0.0, 0.0};
        }
#pragma unroll
        for (int t = 0; t < kAhead; ++t) {
          if (q[t] < 0) continue;
          const cplx vq = {__shfl_sync(0xffffffffu, v.x, q[t]), __shfl_sync(0xffffffffu, v.y, q[t])};
          if (mine && !(finite && is_zero(u[t]))) plain_fma(s, u[t], vq, fx, fy);
        }
      }
      if (kb == k0) {
        if (mine) put(column(c_now), lane, s);
        s = {0.0, 0.0};
      }
    }
  }
  __syncwarp();
}

__device__ __forceinline__ float max_abs3(float a, float b, float c) {
  float d;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// 256 (256 (256 q0 + q1) + q2) + q3 of eight columns, q_o the integer values of four FP32 accumulators.  An
// integer up to 2^22 shows in the low bits of its sum with 1.5 2^23; larger ones (sums of digit
// products near their bound) are converted one by one, at a quarter of the rate.
__device__ __forceinline__ void join_orders(const uint32_t (&v)[4][8], long long (&s)[8]) {
  float mx = 0.f;
#pragma unroll
  for (int o = 0; o < 4; ++o)
#pragma unroll
    for (int j = 0; j < 8; j += 2) mx = max_abs3(mx, __uint_as_float(v[o][j]), __uint_as_float(v[o][j + 1]));
  if (__any_sync(0xffffffffu, !(mx <= 4194304.f))) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      s[j] = 0;
#pragma unroll
      for (int o = 0; o < 4; ++o) s[j] = s[j] * 256 + __float2int_rn(__uint_as_float(v[o][j]));
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint32_t q[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) q[o] = __float_as_uint(__uint_as_float(v[o][j]) + 12582912.f);   // 0x4B400000 + q_o
    const int a = (int)((q[0] << 8) + q[1] - 0x8B400000u), b = (int)((q[2] << 8) + q[3] - 0x8B400000u);
    s[j] = (long long)a * 65536ll + b;
  }
}

// Persistent over units of one 128-row tile x nt real columns x a range of segments.  Roles: warp 0 loads
// digit blocks (bulk copies, three stages of one 16-element K step), warp 1 issues the MMAs, warps 2-13 drain
// the accumulators at the end of a segment (a warp reads its lane quarter, every third group of eight columns) into
// integer sums in global memory, which stay in L2, and read them back, convert and store (or add up) while the
// next MMAs run.  (With the sums in registers the loops over columns had to be unrolled into 70 to 140 KB of
// code, and instruction fetches made the epilogue three times the MMA time.)
//
// An MMA costs the larger of its N / 2 cycles and its operands' shared-memory reads, about (4096 + 32 N) / 88
// (70 cycles at N = 64, 93 at 128), so wide tiles halve the cost per column.  TMEM holds 512 columns:
//   G = 8: tiles of up to 64 columns, all eight orders at once (36 MMAs per K step);
//   G = 4: tiles of up to 128 columns in two phases over a segment, orders 4..7 (26 MMAs), which the conversion of
//          the last segment overlaps, then orders 0..3 (ten MMAs, four digit planes loaded);
// a last phase sums the magnitudes (one MMA per K step, eight steps' planes per stage).  It costs the wait for the tile before and
// after: with seven digits and without it a mode product at nb = 64 took 341 us, now 370, the pair product of GW 14.3 ms,
// now 15.0.
// kKind: 0 one segment per unit, 1 several, 2 a long contraction (several, real products of re and im rows).
template <int G, int kKind>
__global__ void __launch_bounds__(kThreads, 1) fp64_tc_gemm_kernel(const __grid_constant__ TcGemm p) {
  constexpr bool kSplit = kKind == 2;
  constexpr int kMain = kOrd / G, kPhases = kMain + 1;   // of the digits, and the magnitudes
  constexpr int kTN = 512 / G;                       // TMEM columns per accumulator
  constexpr uint32_t kABlk = kDig * kADig, kStageBytes = 2 * kABlk;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *stg_all = smem + kStages * kStageBytes;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kSmem - 1024 - 256);
  uint64_t *full = bars, *empty = bars + kStages, *tfull = bars + 2 * kStages, *tempty = tfull + 1, *fin = tempty + 1;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(fin + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bdig = (uint32_t)p.nt * 32, bblk = kDig * bdig;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(tfull, 1);
    mbar_init(tempty, 32 * kEpiWarps);
    mbar_init(fin, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  dependent_begin();
  const int units = p.mtiles * p.ntiles * p.splits;

  if (warp == 0) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int nt = u % p.ntiles, mt = (u / p.ntiles) % p.mtiles, sp = u / (p.ntiles * p.mtiles);
        const int s0 = sp * p.segs_per_split, s1 = min(p.segs, s0 + p.segs_per_split);
        for (int sf = s0 * kPhases; sf < s1 * kPhases && ok; ++sf) {
          const int f = sf % kPhases, kb0 = (sf / kPhases) * p.kseg, kb1 = min(p.KB, kb0 + p.kseg);
          // a stage: the digits of one K block (all, or the four leading ones), or the magnitudes of up to kDig
          const bool mags = f == kMain;
          for (int kb = kb0; kb < kb1; kb += mags ? kDig : 1) {
            if (!mbar_wait(&empty[s], ph ^ 1u, p.err)) { ok = false; break; }
            uint8_t *st = smem + (size_t)s * kStageBytes;
            const size_t ka = (size_t)mt * p.KB + kb, kc = (size_t)nt * p.KB + kb;
            const uint32_t np = mags ? (uint32_t)min(kDig, kb1 - kb) : f == 1 ? 4u : (uint32_t)kDig;   // planes
            mbar_arrive_expect_tx(&full[s], np * (kADig + bdig));
            bulk_load(st, mags ? p.MA + ka * kADig : p.A + ka * kABlk, np * kADig, &full[s]);
            bulk_load(st + kABlk, mags ? p.MB + kc * bdig : p.B + kc * bblk, np * bdig, &full[s]);
            if (++s == kStages) { s = 0; ph ^= 1u; }
          }
        }
      }
      wait_loads(full, kStages, s, ph);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(kTM, p.nt);
      int s = 0;
      uint32_t ph = 0, acc_ph = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
        const int sp = u / (p.ntiles * p.mtiles);
        const int s0 = sp * p.segs_per_split, s1 = min(p.segs, s0 + p.segs_per_split);
        for (int seg = s0; seg < s1 && ok; ++seg) {
          const int kb0 = seg * p.kseg, kb1 = min(p.KB, kb0 + p.kseg);
#pragma unroll
          for (int f = 0; f < kPhases; ++f) {
            if (!ok || !mbar_wait(tempty, acc_ph ^ 1u, p.err)) { ok = false; break; }
            tc_fence_after();
            for (int kb = kb0; kb < kb1; kb += f == kMain ? kDig : 1) {
              if (!mbar_wait(&full[s], ph, p.err)) { ok = false; break; }
              tc_fence_after();
              const uint32_t sa = smem_u32(smem + (size_t)s * kStageBytes), sb = sa + kABlk;
              uint64_t a[kDig], b[kDig];
#pragma unroll
              for (int q = 0; q < kDig; ++q) {
                a[q] = smem_desc_sw32(sa + q * kADig);
                b[q] = smem_desc_sw32(sb + q * bdig);
              }
              if (f == kMain) {
#pragma unroll
                for (int q = 0; q < kDig; ++q)
                  if (kb + q < kb1) mma_bf16(tmem, a[q], b[q], idesc, (kb == kb0 && q == 0) ? 0u : 1u);
              } else {
#pragma unroll
                for (int g = 0; g < G; ++g) {
                  const int o = (kMain - 1 - f) * G + g, q0 = o < kDig ? 0 : o - kDig + 1;
#pragma unroll
                  for (int q = q0; q <= o && q < kDig; ++q)
                    mma_bf16(tmem + (uint32_t)(g * kTN), a[q], b[o - q], idesc, (q == q0 && kb == kb0) ? 0u : 1u);
                }
              }
              mma_commit(&empty[s]);
              if (++s == kStages) { s = 0; ph ^= 1u; }
            }
            if (!ok) break;
            mma_commit(tfull);
            acc_ph ^= 1u;
          }
        }
      }
      mma_commit(fin);
      mbar_wait_own(fin, 0);
    }
  } else {
    const int quarter = warp & 3, cg = (warp - 2) >> 2;
    const int r = 32 * quarter + lane;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const int ngroups = p.nt >> 3;
    cplx *stg = reinterpret_cast<cplx *>(stg_all + (warp - 2) * kStgWarp);
    uint32_t acc_ph = 0;
    bool ok = true;
    long long *sums = p.sums + (size_t)blockIdx.x * 2 * kTNMax * kTM + r;
    for (int u = blockIdx.x; u < units && ok; u += gridDim.x) {
      const int ntile = u % p.ntiles, mt = (u / p.ntiles) % p.mtiles, sp = u / (p.ntiles * p.mtiles);
      const int s0 = sp * p.segs_per_split, s1 = min(p.segs, s0 + p.segs_per_split);
      double *part = p.part + (size_t)(kSplit ? u : blockIdx.x) * kTNMax * kTM + r;
      // this lane's row, its exponents and its place in C (a long contraction has rows 2 i + re / im)
      const int m = mt * kTM + r, mc = kSplit ? m >> 1 : m;
      const bool valid = mc < p.rows;
      const int y_tile = (ntile * p.nt) >> 1;           // first complex column of the tile
      long long off = 0;
      if (!kSplit && valid) {
        const int row = p.r_begin + m, b = row / p.X.X;
        off = (long long)b * p.scb + (long long)(row - b * p.X.X) * p.scx;
      }
      uint32_t any = 0;
      for (int seg = s0; seg < s1 && ok; ++seg) {
        // exponents, loaded before the MMAs are waited for: lane 4 i + j holds that of column j of this warp's
        // i-th group
        const int yl = y_tile + 4 * (cg + kPerQuarter * (lane >> 2)) + (lane & 3);
        const int xr = valid ? p.ex[(size_t)seg * p.exs + mc] : kZeroRow;
        const int yr = (lane < kMaxGroups * 4 && yl < p.cols) ? p.ey[(size_t)seg * p.eys + yl] : kZeroRow;
        const int ea = xr & kExpMask, eyl = yr & kExpMask;
#pragma unroll 1
        for (int f = 0; f < kMain; ++f) {
          if (!__all_sync(0xffffffffu, mbar_wait(tfull, acc_ph, p.err))) { ok = false; break; }
          tc_fence_after();
#pragma unroll 1
          for (int g = cg; g < ngroups; g += kPerQuarter) {
#pragma unroll
            for (int w = 0; w < G / 4; ++w) {
              long long *q = sums + (size_t)(8 * g) * kTM + ((G == 8 ? w : 1 - f) ? kTNMax * kTM : 0);
              long long s[8];
              uint32_t v[4][8];
#pragma unroll
              for (int o = 0; o < 4; ++o)
                tmem_ld8(tmem + lane_base + (uint32_t)((4 * w + o) * kTN + 8 * g), v[o]);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int o = 0; o < 4; ++o) after_wait(v[o]);
              join_orders(v, s);
#pragma unroll
              for (int j = 0; j < 8; ++j) __stcg(q + j * kTM, s[j]);
            }
          }
          tc_fence_before();
          mbar_arrive(tempty);
          acc_ph ^= 1u;
        }
        if (!ok) break;
        // elements whose sum of magnitudes is too small for the digits, or with an Inf or a NaN (bit 4 i + j: column j of
        // this lane's i-th group)
        if (!__all_sync(0xffffffffu, mbar_wait(tfull, acc_ph, p.err))) { ok = false; break; }
        tc_fence_after();
        uint32_t plain = 0;
#pragma unroll 1
        for (int g = cg, gl = 0; g < ngroups; g += kPerQuarter, gl += 4) {
          uint32_t v[8];
          tmem_ld8(tmem + lane_base + (uint32_t)(8 * g), v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          after_wait(v);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int yj = __shfl_sync(0xffffffffu, yr, gl + j);
            const bool low = too_small(__uint_as_float(v[2 * j])) || too_small(__uint_as_float(v[2 * j + 1]));
            if ((low || max(ea, yj & kExpMask) == kNonFinite) && y_tile + 4 * g + j < p.cols) plain |= 1u << (gl + j);
          }
        }
        if (!valid) plain = 0;
        tc_fence_before();
        mbar_arrive(tempty);
        acc_ph ^= 1u;
        const bool some = __any_sync(0xffffffffu, plain != 0);
        if constexpr (kSplit) {                         // fp64_tc_reduce_kernel adds them: here they may fill a few CTAs' segments
          p.flags[((size_t)((mt * p.ntiles + ntile) * kPerQuarter + cg) * kTM + r) * p.all_segs + p.seg_begin + seg] = plain;
          any |= plain;
        } else if (some) {
          const bool finite = !__any_sync(0xffffffffu, max(ea, eyl) == kNonFinite);
          const int k0 = seg * seg_k(kRows);
          plain_elements(p, plain, finite, xr >> kExpBits, yr >> kExpBits, mt * kTM + 32 * quarter, y_tile + 4 * cg, k0,
                         min(p.X.K, k0 + seg_k(kRows)), reinterpret_cast<uint16_t *>(stg),
                         sums - lane + (size_t)(8 * cg) * kTM);
        }
        // those, or results that may leave the range of fixed_to_double_*
        const bool care = some || __any_sync(0xffffffffu, min(ea, eyl) < kSafeLo || max(ea, eyl) > kSafeHi);
        const bool first = seg == s0 && !(kSplit && p.accumulate), last = seg == s1 - 1;
        // two copies: with the calls of the careful one in its loop, the plain one spilled registers
        auto convert = [&](auto careful) {
        constexpr bool kCare = decltype(careful)::value;
#pragma unroll 1
        for (int g = cg, gl = 0; g < ngroups; g += kPerQuarter, gl += 4) {
          const int y0 = y_tile + 4 * g;                 // first complex column of the group
          const int ny = min(4, p.cols - y0);
          if (ny <= 0) break;
          const long long *q = sums + (size_t)(8 * g) * kTM;
          double *pq = part + (size_t)(8 * g) * kTM;
          long long hi[8], lo[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            hi[j] = __ldcg(q + j * kTM);
            lo[j] = __ldcg(q + j * kTM + kTNMax * kTM);
          }
          double v[8];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int e0 = ea + __shfl_sync(0xffffffffu, eyl, gl + j) - 2112;
            const int e = kCare ? min(max(e0, kMinE), kMaxE) : e0;
            v[2 * j] = kSplit ? fixed_to_double_int(hi[2 * j], lo[2 * j], e) : fixed_to_double_add(hi[2 * j], lo[2 * j], e);
            v[2 * j + 1] = fixed_to_double_int(hi[2 * j + 1], lo[2 * j + 1], e);
            if constexpr (kCare) {
              if (e != e0) {
                v[2 * j] = beyond_range(v[2 * j], e0 - e);
                v[2 * j + 1] = beyond_range(v[2 * j + 1], e0 - e);
              }
              if (plain >> (gl + j) & 1u) {
                v[2 * j] = kSplit ? 0.0 : __longlong_as_double(hi[2 * j]);
                v[2 * j + 1] = kSplit ? 0.0 : __longlong_as_double(hi[2 * j + 1]);
              }
            }
          }
          if (kKind != 0 && !first) {   // (in one-segment kernels the compiler would add a zero, on the slow FP64 pipe)
            double o[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) o[j] = __ldcg(pq + j * kTM);
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] += o[j];
          }
          if (kKind != 0 && (kSplit || !last)) {
#pragma unroll
            for (int j = 0; j < 8; ++j) __stcg(pq + j * kTM, v[j]);
          }
          if (kSplit || (kKind != 0 && !last)) continue;
          cplx z[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) z[j] = mul_unit({v[2 * j], v[2 * j + 1]}, p.unit_alpha);
          if (p.scy != 1) {
            // rows contiguous in C (or neither): a lane stores its own row, loads of the old values first
            cplx *c = p.C + off + (long long)(p.y_begin + y0) * p.scy;
            if (p.beta) {
              cplx c0[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) c0[j] = (valid && j < ny) ? c[(long long)j * p.scy] : cplx{0.0, 0.0};
#pragma unroll
              for (int j = 0; j < 4; ++j) z[j] = {z[j].x + c0[j].x, z[j].y + c0[j].y};
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (valid && j < ny) c[(long long)j * p.scy] = z[j];
          } else {
            // columns contiguous in C: through the warp's staging tile, then 64 contiguous bytes of eight
            // rows per store
            const int j = lane & 3;
            cplx *c = p.C + p.y_begin + y0 + j;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) stg[lane * kStgPitch + i] = z[i];
            __syncwarp();
            long long ro[4];
            bool in[4];
            cplx t[4];
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              const int rr = 8 * it + (lane >> 2);
              ro[it] = __shfl_sync(0xffffffffu, off, rr);
              in[it] = mt * kTM + 32 * quarter + rr < p.rows && j < ny;
              t[it] = stg[rr * kStgPitch + j];
            }
            if (p.beta) {
              cplx c0[4];
#pragma unroll
              for (int it = 0; it < 4; ++it) c0[it] = in[it] ? c[ro[it]] : cplx{0.0, 0.0};
#pragma unroll
              for (int it = 0; it < 4; ++it) t[it] = {t[it].x + c0[it].x, t[it].y + c0[it].y};
            }
#pragma unroll
            for (int it = 0; it < 4; ++it)
              if (in[it]) c[ro[it]] = t[it];
          }
        }
        };
        if (care) convert(std::true_type{});
        else convert(std::false_type{});
      }
      if constexpr (kSplit) {
        uint32_t *a = p.any + (size_t)(u * kPerQuarter + cg) * kTM + r;
        *a = p.accumulate ? *a | any : any;
      }
    }
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Sums the units of a long contraction in a fixed order and combines the four real products:
// C[i][j] = alpha ((re re - im im) + i (re im + im re)) + beta C.  One CTA per output element, which also adds the
// segments that the digits do not give, by FP64 multiply-adds (bits of rows 2 i and 2 i + 1 for column j).  Here the whole chip
// shares them: taken in the GEMM they kept one SM busy for 540 us with the sparse cotangents of the 4 x 4 cluster; 202 us here
// with one warp per element, 141 with a CTA, 106 with terms of zeros left out.  The next kernel may start once these are done: its
// CTAs would take the L1 from their loads.
constexpr int kRedThreads = 128;
__global__ void __launch_bounds__(kRedThreads) fp64_tc_reduce_kernel(const TcGemm p) {
  __shared__ double sx[kRedThreads / 32], sy[kRedThreads / 32];
  dependent_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i = blockIdx.x / p.cols, j = blockIdx.x - i * p.cols;
  const int mt = 2 * i / kTM, nt = 2 * j / p.nt, rr = 2 * i - mt * kTM, cc = 2 * j - nt * p.nt;
  const int grp = cc >> 3, cg = grp % kPerQuarter, bit = 4 * (grp / kPerQuarter) + ((cc >> 1) & 3);
  double x = 0.0, y = 0.0;
  uint32_t any = 0;
  for (int sp = tid; sp < p.splits; sp += kRedThreads) {
    const size_t unit = (size_t)(sp * p.mtiles + mt) * p.ntiles + nt;
    const double *q = p.part + unit * kTNMax * kTM + (size_t)cc * kTM + rr;
    x += q[0] - q[kTM + 1];
    y += q[kTM] + q[1];
    const uint32_t *a = p.any + (unit * kPerQuarter + cg) * kTM + rr;
    any |= (a[0] | a[1]) >> bit & 1u;
  }
  if (__syncthreads_or(any)) {
    const uint32_t *fl = p.flags + ((size_t)((mt * p.ntiles + nt) * kPerQuarter + cg) * kTM + rr) * p.all_segs;
    const cplx *a = p.X.p + row_offset(p.X, i), *b = p.Y.p + row_offset(p.Y, j);
    const int fx = p.X.conj ? (int)0x80000000u : 0, fy = p.Y.conj ? (int)0x80000000u : 0, len = p.kseg * kKB;
    for (int s0 = 32 * warp; s0 < p.all_segs; s0 += kRedThreads) {
      const bool in = s0 + lane < p.all_segs;
      const uint32_t re = __ballot_sync(0xffffffffu, in && (fl[s0 + lane] >> bit & 1u));
      const uint32_t im = __ballot_sync(0xffffffffu, in && (fl[p.all_segs + s0 + lane] >> bit & 1u));
      for (uint32_t m = re | im; m; m &= m - 1) {
        const int s = __ffs((int)m) - 1, k1 = min(p.X.K, (s0 + s + 1) * len);
        const bool r = re >> s & 1u, t = im >> s & 1u;
        double xs = 0.0, ys = 0.0;   // by segment: fewer roundings in a row than in one sum over all
#pragma unroll 8
        for (int k = (s0 + s) * len + lane; k < k1; k += 32) {
          const cplx u = a[k_offset(p.X, k)], v = b[k_offset(p.Y, k)];
          if ((is_zero(u) && is_finite(v)) || (is_zero(v) && is_finite(u))) continue;
          const double ui = flip(u.y, fx), vi = flip(v.y, fy);
          if (r) { xs = fma(u.x, v.x, xs); ys = fma(u.x, vi, ys); }
          if (t) { xs = fma(-ui, vi, xs); ys = fma(ui, v.x, ys); }
        }
        x += xs;
        y += ys;
      }
    }
  }
  dependent_launch();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, o);
    y += __shfl_xor_sync(0xffffffffu, y, o);
  }
  if (lane == 0) { sx[warp] = x; sy[warp] = y; }
  __syncthreads();
  if (tid != 0) return;
  for (int w = 1; w < kRedThreads / 32; ++w) { x += sx[w]; y += sy[w]; }
  cplx z = mul_unit({x, y}, p.unit_alpha);
  cplx *c = p.C + (long long)i * p.scx + (long long)j * p.scy;
  if (p.beta) z = {z.x + c->x, z.y + c->y};
  *c = z;
}

int unit_of(cplx a) {
  if (a.x == 1.0 && a.y == 0.0) return 0;
  if (a.x == 0.0 && a.y == 1.0) return 1;
  if (a.x == -1.0 && a.y == 0.0) return 2;
  if (a.x == 0.0 && a.y == -1.0) return 3;
  return -1;
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Real columns per tile: as few tiles of at most 128 as the columns need, evenly filled.  Up to 64 columns
// run with all orders in TMEM at once (G = 8).
int even_tiles(int real_cols, int tiles) { return round_up((real_cols + tiles - 1) / tiles, 16); }
int tile_columns(int real_cols) { return even_tiles(real_cols, (real_cols + kTNMax - 1) / kTNMax); }
// The same for a product of several segments, which lasts as many rounds of MMAs as the busiest CTA has tiles: the width
// with the least rounds times cost of an MMA (see the kernel).  128 columns everywhere left nb = 24 (45 tiles) and nb = 27
// (72) with most SMs idle: 177 and 242 us.
int tile_columns(int real_cols, int mtiles, int sms) {
  int best = 0;
  long long cost = 0;
  for (int w = kTNMax; w >= 16; w -= 16) {
    const int nt = even_tiles(real_cols, (real_cols + w - 1) / w);
    const long long units = (long long)mtiles * ((real_cols + nt - 1) / nt);
    const long long c = (units + sms - 1) / sms * (4096 + 32 * nt);
    if (!best || c < cost) { best = nt; cost = c; }
  }
  return best;
}

template <int kKind>
void launch_gemm(Launcher &L, const TcGemm &t, int ctas, const char *tag) {
  L.before(tag);
  if (t.nt <= 64) launch_dependent(fp64_tc_gemm_kernel<8, kKind>, ctas, kThreads, kSmem, L.stream, t);
  else launch_dependent(fp64_tc_gemm_kernel<4, kKind>, ctas, kThreads, kSmem, L.stream, t);
  L.after_launch();
}

CutJob cut_job(const Operand &o, int r_begin, int rows, int TR, int *rexp, uint8_t *out, uint8_t *mag) {
  CutJob j{o, r_begin, TR, rexp, out, mag};
  j.o.rows = rows;
  return j;
}

// x and y (where they have rows) in segments of SK <= seg_k(FX) values
template <int FX, int FY>
void cut(Launcher &L, const CutJob &x, const CutJob &y, int k_begin, int Klen, int Kp, int KB, int SK) {
  static_assert(seg_k(FX) == seg_k(FY), "one grid of segments");
  constexpr int SR = cut_rows(FX);
  const size_t sh = (size_t)2 * SR * (std::min(SK, Kp) + 1) * sizeof(double);
  const int xb = (x.o.rows + SR - 1) / SR, yb = (y.o.rows + SR - 1) / SR;
  if (xb + yb == 0) return;
  dim3 grid(xb + yb, (Kp + SK - 1) / SK);
  L.before("fp64_tc_digits");
  launch_dependent(cut_digits_kernel<FX, FY>, grid, 256, sh, L.stream, x, y, xb, k_begin, Klen, Kp, KB, SK);
  L.after_launch();
}

}  // namespace

constexpr int kMinK = 8, kMinCols = 8;
// Complex multiply-adds from which a product is faster here than on zgemm_kernel, whose time grows with them while digits,
// product and reduction here cost their launches and one round of MMAs.  Per launch with an event on either side: mode product 13 us
// there at nb = 15 (34 at nb = 20 by its growth), 25 us here at nb = 16 and 30 at nb = 20; long contraction 25 us there
// at nb = 15 (45 at nb = 20), 48 us here at nb = 16 and 43 at nb = 24; nb^2 x nb^2 x nb^2 product 43 and 39 us at nb = 12 (3e6).
constexpr double kMinWork = 2.2e6, kMinWorkLong = 4e6;

// nb^5 products pass kMinWork from nb = 19 on; nb^4 products with the factors of a factorised interaction (nfac <= nb^2) may below
int fp64_tc_min_nb(bool pair_products, bool factorised) { return pair_products ? 12 : factorised ? 17 : 19; }

struct Fp64Tc {
  uint8_t *A = nullptr, *B = nullptr;   // digit blocks of the two operands
  uint8_t *MA = nullptr, *MB = nullptr; // their magnitudes, an eighth of the size
  size_t a_bytes = 0, b_bytes = 0;
  int *ex = nullptr, *ey = nullptr;     // exponents
  long long exps = 0;                   // of each
  long long *sums = nullptr;            // hi and lo sums of a tile per CTA
  double *part = nullptr;               // FP64 sums of a tile per CTA
  uint32_t *flags = nullptr, *any = nullptr;   // elements of long contractions that the digits do not give
  long long flag_words = 0;
  int *err = nullptr;
  int sms = 0;
  size_t a_panel = 0, b_panel = 0;      // what a product uses of A and B (at most a_bytes and b_bytes)
  int yK = 0, ycols = 0, ynt = 0;       // shape of the column operand whose digits B holds whole (0: none), and that operand
  Operand y{};
};

void fp64_tc_destroy(Fp64Tc *f) {
  if (!f) return;
  for (void *p : {(void *)f->A, (void *)f->B, (void *)f->MA, (void *)f->MB, (void *)f->ex, (void *)f->ey, (void *)f->sums, (void *)f->part, (void *)f->flags,
                  (void *)f->any, (void *)f->err})
    if (p) cudaFree(p);
  delete f;
}

Fp64Tc *fp64_tc_create(int nb, bool pair_products) {
  const long long N = nb, N2 = N * N, N3 = N2 * N;
  Fp64Tc *f = new (std::nothrow) Fp64Tc;
  if (!f) return nullptr;
  // digit blocks: all of a big operand up to kPanelBytes, panels of it above
  constexpr size_t kPanelBytes = (size_t)1 << 30;
  auto blocks = [](long long rows, long long Kp) { return (size_t)((rows + 127) / 128 * 128) * (size_t)Kp * 2 * kDig; };
  const size_t big = blocks(N3, 2 * ((N + 7) / 8 * 8)), pair = pair_products ? blocks(2 * N2 + kTNMax, 2 * ((N2 + 7) / 8 * 8)) : 0;
  const size_t lng = blocks(2 * N, (N3 + 255) / 256 * 256);
  f->a_bytes = std::min(kPanelBytes, std::max({big, pair, lng}));
  f->b_bytes = std::min(kPanelBytes, std::max({blocks(2 * N, 2 * ((N + 7) / 8 * 8)), pair, lng}));
  f->a_panel = f->a_bytes;
  f->b_panel = f->b_bytes;
  f->exps = std::max({N3, N2 * ((N2 + 127) / 128), N * ((N3 + 127) / 128)});
  f->flag_words = (N3 + 127) / 128 * ((2 * N + kTM - 1) / kTM) * ((2 * N + kTNMax - 1) / kTNMax) * kPerQuarter * kTM;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&f->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    goto bad;
  if (cudaMalloc(&f->A, f->a_bytes) != cudaSuccess || cudaMalloc(&f->B, f->b_bytes) != cudaSuccess ||
      cudaMalloc(&f->MA, f->a_bytes / kDig) != cudaSuccess || cudaMalloc(&f->MB, f->b_bytes / kDig) != cudaSuccess ||
      cudaMalloc(&f->ex, sizeof(int) * (size_t)f->exps) != cudaSuccess ||
      cudaMalloc(&f->ey, sizeof(int) * (size_t)f->exps) != cudaSuccess ||
      cudaMalloc(&f->sums, (size_t)f->sms * 2 * kTNMax * kTM * sizeof(long long)) != cudaSuccess ||
      cudaMalloc(&f->part, (size_t)f->sms * kTNMax * kTM * sizeof(double)) != cudaSuccess ||
      cudaMalloc(&f->flags, sizeof(uint32_t) * (size_t)f->flag_words) != cudaSuccess ||
      cudaMalloc(&f->any, sizeof(uint32_t) * (size_t)f->sms * kPerQuarter * kTM) != cudaSuccess ||
      cudaMalloc(&f->err, sizeof(int)) != cudaSuccess || cudaMemset(f->err, 0, sizeof(int)) != cudaSuccess)
    goto bad;
  for (const void *k : {(const void *)fp64_tc_gemm_kernel<8, 0>, (const void *)fp64_tc_gemm_kernel<8, 1>,
                        (const void *)fp64_tc_gemm_kernel<8, 2>, (const void *)fp64_tc_gemm_kernel<4, 0>,
                        (const void *)fp64_tc_gemm_kernel<4, 1>, (const void *)fp64_tc_gemm_kernel<4, 2>})
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem) != cudaSuccess) goto bad;
  {
    const int sh = 2 * (kCutVals + 32) * (int)sizeof(double);
    for (const void *k : {(const void *)cut_digits_kernel<kRows, kReal>, (const void *)cut_digits_kernel<kPlanes, kPlanes>})
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, sh) != cudaSuccess) goto bad;
  }
  return f;
bad:
  cudaGetLastError();
  fp64_tc_destroy(f);
  return nullptr;
}

void fp64_tc_set_panel(Fp64Tc *f, size_t bytes) {
  f->a_panel = std::min(f->a_bytes, bytes);
  f->b_panel = std::min(f->b_bytes, bytes);
}

void fp64_tc_inject_error(Fp64Tc *f, cudaStream_t stream) { cudaMemsetAsync(f->err, 1, sizeof(int), stream); }

int fp64_tc_error(Fp64Tc *f, cudaStream_t stream) {
  int e = 0;
  if (cudaMemcpyAsync(&e, f->err, sizeof(int), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess) {
    set_error_detail("reading the FP64 tensor-core error word failed");
    return G1G2_ECUDA;
  }
  if (e == 0) return G1G2_OK;
  cudaMemsetAsync(f->err, 0, sizeof(int), stream);
  set_error_detail("a barrier wait of an FP64 tensor-core kernel gave up");
  return G1G2_ETIMEOUT;
}

// C_b = alpha A_b B_b + beta C_b.  The operand with the batch (or the more rows) gives the tile rows, the other the
// columns.
bool fp64_tc_zgemm(Launcher &L, const ZGemm &g) {
  Fp64Tc *f = L.ftc;
  if (!f) return false;
  // digits of the last product's column operand, when that product ran here and the caller says that it is the same
  const int yK = g.same_small ? f->yK : 0;
  f->yK = 0;
  const int alpha = unit_of(g.alpha);
  if (alpha < 0 || (g.beta != 0.0 && g.beta != 1.0)) return false;
  if (g.batch > 1 && g.sa_b != 0 && g.sb_b != 0) return false;
  const bool a_rows = g.batch > 1 ? g.sa_b != 0 : g.M >= g.N;
  Operand X{}, Y{};
  Operand a{g.A, g.sa_b, g.sa_m, g.sa_k, 0, g.M, g.K, g.M, g.K, g.conjA ? 1 : 0};
  Operand b{g.B, g.sb_b, g.sb_n, g.sb_k, 0, g.N, g.K, g.N, g.K, g.conjB ? 1 : 0};
  X = a_rows ? a : b;
  Y = a_rows ? b : a;
  const long long rows = (long long)X.X * g.batch;
  const int cols = Y.X;
  if (g.K < kMinK || cols < kMinCols || (double)rows * cols * g.K < kMinWork) return false;
  const int Kp = round_up(g.K, 8), KB = 2 * Kp / kKB, segs = (KB + kSeg - 1) / kSeg;
  if (std::max<long long>(rows, cols) * segs > f->exps) return false;
  X.rows = (int)rows;
  const int nt = segs == 1 ? tile_columns(2 * cols) : tile_columns(2 * cols, (int)((rows + kTM - 1) / kTM), f->sms);
  // panels of whole tiles
  const size_t a_tile = (size_t)KB * kDig * kADig, b_tile = (size_t)KB * kDig * nt * 32;
  const int all_m = (int)((rows + kTM - 1) / kTM), all_n = (2 * cols + nt - 1) / nt;
  const int pm = (int)std::min<size_t>(all_m, f->a_panel / a_tile), pn = (int)std::min<size_t>(all_n, f->b_panel / b_tile);
  if (pm < 1 || pn < 1) return false;
  for (int n0 = 0; n0 < all_n; n0 += pn) {
    const int y0 = n0 * nt / 2, ny = std::min(cols - y0, std::min(pn, all_n - n0) * nt / 2);
    // (the caller's word covers the contents; where and how they are read is looked at)
    const bool kept = pn >= all_n && yK == g.K && f->ycols == cols && f->ynt == nt && f->y.p == Y.p && f->y.sx == Y.sx &&
                      f->y.sk == Y.sk && f->y.conj == Y.conj;
    for (int m0 = 0; m0 < all_m; m0 += pm) {
      const int r0 = m0 * kTM, nr = (int)std::min<long long>(rows - r0, (long long)std::min(pm, all_m - m0) * kTM);
      cut<kRows, kReal>(L, cut_job(X, r0, (n0 == 0 || pm < all_m) ? nr : 0, kTM, f->ex, f->A, f->MA),
                        cut_job(Y, y0, (m0 == 0 && !kept) ? ny : 0, nt, f->ey, f->B, f->MB), 0, g.K, Kp, KB, seg_k(kRows));
      TcGemm t{};
      t.A = f->A; t.B = f->B; t.MA = f->MA; t.MB = f->MB; t.KB = KB; t.segs = segs; t.kseg = kSeg; t.nt = nt;
      t.mtiles = (nr + kTM - 1) / kTM; t.ntiles = (2 * ny + nt - 1) / nt;
      t.splits = 1; t.segs_per_split = segs; t.err = f->err; t.sums = f->sums; t.part = f->part;
      t.X = X; t.Y = Y; t.ex = f->ex; t.ey = f->ey; t.exs = nr; t.eys = ny;
      t.r_begin = r0; t.y_begin = y0; t.rows = nr; t.cols = ny;
      t.C = g.C; t.scb = g.sc_b; t.scx = a_rows ? g.sc_m : g.sc_n; t.scy = a_rows ? g.sc_n : g.sc_m;
      t.unit_alpha = alpha; t.beta = g.beta != 0.0;
      const int ctas = std::min(f->sms, t.mtiles * t.ntiles);
      if (segs == 1) launch_gemm<0>(L, t, ctas, "fp64_tc_gemm");
      else launch_gemm<1>(L, t, ctas, "fp64_tc_gemm_pair");
    }
  }
  if (pn >= all_n) {
    f->yK = g.K;
    f->ycols = cols;
    f->ynt = nt;
    f->y = Y;
  }
  return true;
}

// C = alpha sum_b A_b B_b + beta C: one contraction over c = (b, k), both operands as re and im rows.
bool fp64_tc_zgemm_reduce(Launcher &L, const ZGemm &g) {
  Fp64Tc *f = L.ftc;
  if (!f) return false;
  f->yK = 0;
  const int alpha = unit_of(g.alpha);
  if (alpha < 0 || (g.beta != 0.0 && g.beta != 1.0)) return false;
  const long long Kl = (long long)g.K * g.batch;
  if (Kl > (1ll << 30) || std::min(g.M, g.N) < kMinCols || (double)g.M * g.N * Kl < kMinWorkLong) return false;
  const int K = (int)Kl;
  Operand X{g.A, 0, g.sa_m, g.sa_k, g.sa_b, g.M, g.K, g.M, K, g.conjA ? 1 : 0};
  Operand Y{g.B, 0, g.sb_n, g.sb_k, g.sb_b, g.N, g.K, g.N, K, g.conjB ? 1 : 0};
  const int nt = tile_columns(2 * g.N);
  const int mtiles = (2 * g.M + kTM - 1) / kTM, ntiles = (2 * g.N + nt - 1) / nt;
  const int splits_max = f->sms / (mtiles * ntiles);   // one unit per CTA
  if (splits_max < 1) return false;
  // segments of 256 terms, or 128 where those leave half of the SMs idle (nb <= 26: 34 -> 24 us at nb = 24)
  const int kseg = 2 * ((K + kSeg * kKB - 1) / (kSeg * kKB)) * mtiles * ntiles <= f->sms ? kSeg / 2 : kSeg;
  const size_t a_seg = (size_t)mtiles * kseg * kDig * kADig, b_seg = (size_t)ntiles * kseg * kDig * nt * 32;   // bytes per segment
  const int all_segs = (K + kseg * kKB - 1) / (kseg * kKB);
  int ps = (int)std::min<size_t>(all_segs, std::min(f->a_panel / a_seg, f->b_panel / b_seg));
  ps = (int)std::min<long long>(ps, f->exps / std::max(g.M, g.N));
  if (ps < 1 || (long long)all_segs * mtiles * ntiles * kPerQuarter * kTM > f->flag_words) return false;
  TcGemm t{};
  for (int sg0 = 0; sg0 < all_segs; sg0 += ps) {
    const int ns = std::min(ps, all_segs - sg0), k0 = sg0 * kseg * kKB, Klen = std::min(K - k0, ns * kseg * kKB);
    const int Kp = round_up(Klen, kKB), KB = Kp / kKB;
    cut<kPlanes, kPlanes>(L, cut_job(X, 0, g.M, kTM, f->ex, f->A, f->MA), cut_job(Y, 0, g.N, nt, f->ey, f->B, f->MB), k0, Klen, Kp, KB,
                           kseg * kKB);
    t.A = f->A; t.B = f->B; t.MA = f->MA; t.MB = f->MB; t.KB = KB; t.segs = ns; t.kseg = kseg; t.nt = nt; t.mtiles = mtiles; t.ntiles = ntiles;
    // the first panel is the longest: its split count holds for the later ones
    if (sg0 == 0) {
      t.segs_per_split = (ns + splits_max - 1) / splits_max;
      t.splits = (ns + t.segs_per_split - 1) / t.segs_per_split;
    } else {
      t.segs_per_split = (ns + t.splits - 1) / t.splits;
    }
    t.err = f->err; t.X = X; t.Y = Y; t.ex = f->ex; t.ey = f->ey; t.exs = g.M; t.eys = g.N; t.rows = g.M; t.cols = g.N;
    t.k_begin = k0;
    t.C = g.C; t.scx = g.sc_m; t.scy = g.sc_n; t.unit_alpha = alpha; t.beta = g.beta != 0.0;
    t.sums = f->sums; t.part = f->part; t.accumulate = sg0 > 0;
    t.flags = f->flags; t.any = f->any; t.all_segs = all_segs; t.seg_begin = sg0;
    launch_gemm<2>(L, t, t.splits * mtiles * ntiles, "fp64_tc_gemm_long");
  }
  L.before("fp64_tc_reduce");
  launch_dependent(fp64_tc_reduce_kernel, g.M * g.N, kRedThreads, 0, L.stream, t);
  L.after_launch();
  return true;
}

}  // namespace g1g2
