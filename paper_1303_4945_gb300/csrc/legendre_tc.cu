// legendre_tc.cu -- the mixed form's Legendre synthesis (Eq. syn2) with the
// contraction of a_lm against Lambda_lm on the tensor cores (tcgen05).
//
// For one m and the 128 ring pairs of a CTA the synthesis is a product
// F[pair][col] = sum_l Lambda[pair][l] B[l][col] (Sect. 3.2's inner loop over l,
// Fig. 1), with B the a_lm values arranged by column (real and imaginary parts,
// the even/odd-l split of the ring-pair parity, the +s / -s spin combinations).
// Lambda is still generated on the fly by the double-float recursion of Sect. 4.1
// (one thread per ring pair, as in legendre_mixed.cu); the product runs as bf16
// matrix products with FP32 accumulation, made exact by splitting both operands
// into digits on a common grid (an Ozaki-style error-free split):
//
//  * Lambda = L0 + L1 + L2 + r.  The digits Lj are multiples of qj = u 2^(-7-8j)
//    with |Lj| <= 128 qj, where u is a power of two bounding the ring pair's own
//    |Lambda_lm| from its join block to lmax + 1 (its join record: one walk of the
//    recursion at plan creation; not below 2^-16 of the plan-wide bound
//    sqrt((2 lmax + 3)/(4 pi)), |d^l| <= 1); each digit fits a bf16 exactly.  One
//    row of the product is one pair, so rows on different grids never share a sum.
//    The FP32 remainder r (|r| <= q2/2) is contracted on the CUDA cores (one FFMA
//    per output column), so Lambda enters to ~2^-43 u.
//  * B = B0 + ... + B5 with digits on the grid u_c 2^(-7-8j), u_c a power of two
//    bounding column c of B over a window of 256 degrees: a value enters to
//    2^-47 u_c (the last digit's rounding and that of the low word's entry; with
//    five digits the truncation at 2^-40 u_c was the larger error).
//  * The products Li Bj with i + j = k are accumulated in TMEM level k (k <= 5;
//    the dropped products sum to below 2^-47 of the bounds).  Every product is a
//    multiple of the level's quantum and a level's sum over one window stays
//    below 2^24 quanta, so the FP32 accumulation is exact whatever its rounding.
//  * After each window the six levels are read from TMEM and added in
//    double-float, together with the CUDA-core remainder sums.
//
// MMA shape: M = 128 ring pairs (one TMEM lane per pair: thread t reads lane t),
// K = 16 degrees per instruction, N = 2 NCW: one instruction reads two
// consecutive a_lm digit tiles (NCW >= 8 columns each) and so adds L_i B_j and
// L_i B_(j+1) into two consecutive levels of NCW TMEM columns (level k at column
// k NCW), which keeps the narrow shapes' MMAs free of padding columns: 8 MMAs per
// Lambda set and K-step instead of 14.
// A (the Lambda digits) and B (the a_lm digit stack) are K-major in shared memory
// without swizzle, 8x16-byte core matrices 128 bytes apart along K and 256 bytes
// apart along M / N.  One thread issues a K-step's MMAs in program order (the
// first ones of a window overwrite every level read later); the recursion's
// digits of K-step s + 1 are written once the MMAs of s have completed, and B is
// rebuilt then too.
//
// What bounds it (GB300, spin 2, one E/B pair, lmax 4095; lmax 2047 under ncu): the
// FP32 pipe (58% busy) and issue (67%), with the K-step's barrier the largest stall;
// 20 warps per SM.  A step takes about 73 FP32 lane operations (recursions 45, digits
// 20, remainders 8), so at the pipe's measured rate the kernel needs 29 ms.  History:
// 54.3 ms with scalar recursions of three coefficients, 49.6 with the unit-coefficient
// recursion, 39.9 with both recursions packed, on Lambda / u_p and with the signs in
// the recursion, 38.7 with 16-byte digit stores and B built between the halves (8
// spin-0 maps at lmax 2047: 10.2 -> 8.7).  The B build split evenly over the threads
// was slower (40.5 against 39.9), four CTAs per SM with more registers too (42.9).
#include "dual.cuh"
#include "tcgen05.cuh"

namespace sht {
namespace tc {

constexpr int kRows = 128;          // ring pairs per CTA = MMA M = TMEM lanes
constexpr int kK = 16;              // degrees per MMA (bf16 K)
constexpr int kWin = 16;            // K-steps per TMEM window (256 degrees)
constexpr int kLamDigits = 3;       // bf16 digits of Lambda (plus an FP32 remainder)
constexpr int kAlmDigits = 6;       // bf16 digits of the a_lm columns
constexpr int kLevels = 6;          // TMEM levels read: digit products with i + j <= 5
constexpr int kATile = kRows * kK * 2;  // bytes of one 128 x 16 bf16 tile
// the warp issuing the MMAs (an elected lane): the last, whose threads neither load
// the staged rows nor build B (threads 0-63 at one E/B pair), so that the warps
// reach the K-step's barrier together (152.4 -> 151.8 ms per headline pair)
constexpr int kIssuerWarp = 3;
// Shapes: NCOL output columns per pair (spin: N1, S4, N2, S3 as re/im per job;
// spin 0: even-l and odd-l sums as re/im per job), NCW = max(NCOL, 8) TMEM columns
// per level and rows per a_lm digit tile, MMA width N = 2 NCW (two digit tiles, two
// levels), NV a_lm values per degree (spin: P = E + iB and M = E - iB, re and im;
// spin 0: re, im).  A set's digit stack holds the tiles of digits -1 .. 5, that of
// digit -1 zero: Lambda digit i meets the windows of digits
// (j0, j0 + 1) with j0 = -(i mod 2), j0 + 2, ..., which start on even levels i + j0,
// so every MMA writes the 2 NCW columns of a level pair at a multiple of N.
//
// TWO (spin 0, one or two maps): a thread runs two neighbouring pairs as the two lanes
// of Dual, whose digits are two A sets meeting the same B in accumulators of their own.
template <int NJ, bool SPIN, bool TWO>
struct Shape {
  static constexpr bool DUAL = TWO;
  // degrees of digits held in registers before a shared-memory store: eight, but four
  // where the remainder sums of four E/B pairs make the unrolled code of three step
  // forms outgrow the instruction cache (lmax 511 546 us at eight, 387 at four; 1023 2.37, 2.05 ms)
  static constexpr int PACK = SPIN && NJ >= 4 ? 4 : 8;
  static constexpr int NP = DUAL ? 2 : 1;         // ring pairs per thread
  static constexpr int NL = SPIN || DUAL ? 2 : 1; // A sets
  static constexpr int NB = SPIN ? 2 : 1;         // B stacks
  static constexpr int NCOL = SPIN ? 8 * NJ : 4 * NJ;
  static constexpr int NCW = NCOL < 8 ? 8 : NCOL;
  static constexpr int N = 2 * NCW;
  static constexpr int NDT = kAlmDigits + 1;  // digit tiles per Lambda set: -1 .. 5
  static constexpr int COLS1 = kLevels * NCW; // TMEM: levels 0 .. 5
  static constexpr int COLS = NP * COLS1;
  static constexpr int TCOLS = COLS <= 32 ? 32 : (COLS <= 64 ? 64 : (COLS <= 128 ? 128 : 256));
  static constexpr int NV = SPIN ? 4 * NJ : 2 * NJ;
  static constexpr int DTILE = NCW * kK * 2;  // bytes of one a_lm digit tile
  static constexpr int A_BYTES = NL * kLamDigits * kATile;
  static constexpr int B_BYTES = NB * NDT * DTILE;
  // per degree of a K-step, staged in shared memory one K-step ahead: the float4
  // of its recursion coefficients and one float4 per a_lm table row read
  static constexpr int NARR = SPIN ? 2 * NJ : NJ;
  static constexpr int ROW = 1 + NARR;
  static constexpr int STG = kK * ROW;                 // float4 per K-step
  static constexpr int PF = (STG + kRows - 1) / kRows;  // of them per thread
  static constexpr int ST_BYTES = 2 * STG * 16;        // two buffers
  static constexpr int ACC_BYTES = NP * NCOL * kRows * 8;  // the double-float column sums [pair of the thread][col][thread]
  static constexpr int SMEM = A_BYTES + ST_BYTES + B_BYTES + ACC_BYTES + 2 * NV * 4;
  // CTAs per SM the kernel is compiled for, and the dynamic shared memory
  // requested: at least enough that no more than 512 / TCOLS CTAs fit on an SM,
  // so their TMEM allocations never wait for one another
  static constexpr int MINB = TCOLS <= 64 ? 5 : (TCOLS == 128 ? 4 : 2);
  static constexpr int SMEM_FLOOR = (228 * 1024) / (512 / TCOLS + 1) - 1024 + 1;
  static constexpr int SMEM_LAUNCH = SMEM > SMEM_FLOOR ? SMEM : SMEM_FLOOR;
  static_assert(N % 16 == 0 && N <= 256 && NCW % 8 == 0, "MMA width; digit tiles of whole core-matrix rows");
  static_assert(kLevels % 2 == 0 && kLamDigits <= 3, "level pairs");
  static_assert(COLS <= TCOLS && COLS1 % 2 == 0, "TMEM allocation");
  static_assert(!TWO || (!SPIN && NJ <= 2), "two pairs a thread: spin 0, one or two maps");
  static_assert(NCOL <= 32, "tensor-core synthesis: at most 32 output columns");
  static_assert(128 % NV == 0, "a_lm values per degree must divide the CTA");
};



// the double-float a_lm value v (Shape::NV of them per degree) at table index ci
template <int NJ, bool SPIN>
__device__ __forceinline__ f2 alm_value(const MixArgs &a, int64_t ci, int v) {
  if (SPIN) {
    const float4 q = __ldg(a.alm32 + (int64_t)(2 * (v / 4) + ((v & 2) ? 1 : 0)) * a.ncoef + ci);
    return (v & 1) ? f2{q.z, q.w} : f2{q.x, q.y};
  }
  const float4 q = __ldg(a.alm32 + (int64_t)(v / 2) * a.ncoef + ci);
  return (v & 1) ? f2{q.z, q.w} : f2{q.x, q.y};
}

// the double-float a_lm value v from a staged degree row (coefficients, then the tables)
template <int NJ, bool SPIN>
__device__ __forceinline__ f2 staged_value(const float4 *row, int v) {
  const float4 q = SPIN ? row[1 + 2 * (v / 4) + ((v & 2) ? 1 : 0)] : row[1 + v / 2];
  return (v & 1) ? f2{q.z, q.w} : f2{q.x, q.y};
}

// Column bounds of one window (degrees lw0..lw1): umax[v] = max |value v| over
// the window (atomically, as FP32 bit patterns of non-negative numbers).  The
// caller synchronises before the bounds are read.
template <int NJ, bool SPIN>
__device__ __forceinline__ void window_bounds(const MixArgs &a, int64_t co, int lw0, int lw1, float *umax) {
  using S = Shape<NJ, SPIN, false>;
  const int v = threadIdx.x % S::NV;
  float mx = 0.f;
  for (int l = lw0 + (int)threadIdx.x / S::NV; l <= lw1; l += kRows / S::NV)
    mx = fmaxf(mx, fabsf(alm_value<NJ, SPIN>(a, co + l, v).h));
  // lanes holding the same v differ in the bits above log2(NV): reduce over them
#pragma unroll
  for (int o = S::NV; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) < S::NV) atomicMax(reinterpret_cast<int *>(umax) + v, __float_as_int(mx));
}

// The a_lm digit stacks of a K-step from its staged rows (zero past lmax; M times s =
// (-1)^(l - l0)): value v of degree lb + k split into kAlmDigits digits on its window's
// grid and written into the rows of the columns that read it (see the column layout
// in tc_syn_body).  Set t's
// stack holds NDT digit tiles of NCW rows, digit j at rows (j + 1) NCW ..; rows no
// value writes (the other set's columns, padding columns, the tile of digit -1)
// stay zero from the kernel's start.
template <int NJ, bool SPIN>
__device__ __forceinline__ void build_b(const float4 *stg, const float *umax, unsigned char *Bt) {
  using S = Shape<NJ, SPIN, false>;
  // byte offset of (row r of the stack, degree k) in the K-major core-matrix layout
  auto at = [](int r, int k) { return (r / 8) * 256 + (r % 8) * 16 + (k / 8) * 128 + (k % 8) * 2; };
  for (int t = threadIdx.x; t < kK * S::NV; t += kRows) {
    const int k = t % kK, v = t / kK;
    const f2 x = staged_value<NJ, SPIN>(stg + k * S::ROW, v);  // zero past lmax
    const float s0 = pow2_above(umax[v]) * 98304.0f;  // 1.5 * 2^23 * (bound * 2^-7)
    float d[kAlmDigits];
    float r = x.h;
    d[0] = round_to(r, s0);
    r = __fsub_rn(r, d[0]);
    d[1] = round_to(r, s0 * 0x1p-8f);
    r = __fsub_rn(r, d[1]);
    d[2] = round_to(r, s0 * 0x1p-16f);
    r = __fadd_rn(__fsub_rn(r, d[2]), x.l);
    d[3] = round_to(r, s0 * 0x1p-24f);
    r = __fsub_rn(r, d[3]);
    d[4] = round_to(r, s0 * 0x1p-32f);
    r = __fsub_rn(r, d[4]);
    d[5] = round_to(r, s0 * 0x1p-40f);
    // (set, column) pairs of this value; spin: P.re -> (+, 8j) and (-, 8j+6), P.im ->
    // (+, 8j+1) and (-, 8j+7), s M.re -> (+, 8j+2) and (-, 8j+4), s M.im -> (+, 8j+3) and
    // (-, 8j+5); spin 0: the even- or odd-l column of its job
    int col0, col1 = 0, zcol = 0;
    if (SPIN) {
      const int j = v / 4, c = v % 4;
      col0 = 8 * j + c;
      col1 = 8 * j + (c < 2 ? 6 + c : 2 + c);
    } else {
      const bool odd = k & 1;
      const int j = v / 2, c = v % 2;
      col0 = 4 * j + (odd ? 2 : 0) + c;
      zcol = 4 * j + (odd ? 0 : 2) + c;
    }
#pragma unroll
    for (int dj = 0; dj < kAlmDigits; ++dj) {
      const int r = (dj + 1) * S::NCW;
      *reinterpret_cast<uint16_t *>(Bt + at(r + col0, k)) = bf16_of(d[dj]);
      if (SPIN)
        *reinterpret_cast<uint16_t *>(Bt + S::NDT * S::DTILE + at(r + col1, k)) = bf16_of(d[dj]);
      else
        *reinterpret_cast<uint16_t *>(Bt + at(r + zcol, k)) = 0;
    }
  }
}

}  // namespace tc

// ---------------------------------------------------------------------------
// synthesis, spin 0 and spin s
//
// Columns of the product (per job j): spin, 8j + {0,1} N1 = sum P l+, {2,3}
// S4 = sum s M l+, {4,5} N2 = sum M l-, {6,7} S3 = sum s P l- (re, im; s =
// (-1)^(l - l0), P = E + iB, M = E - iB); spin 0, 4j + {0,1} the even-l and
// 4j + {2,3} the odd-l sums of a_lm lambda.  A set 0 holds the digits of l+, set 1
// those of s l-, so both meet B rows holding P and s M.  All sums run on Lambda / u_p
// (u_p the pair's bound) and are multiplied by u_p at the end.
// ---------------------------------------------------------------------------
template <int NJ, bool SPIN, bool TWO>
__device__ __forceinline__ void tc_syn_body(const TcArgs &ta, const int2 item, unsigned char *smem) {
  using S = tc::Shape<NJ, SPIN, TWO>;
  constexpr int NL = S::NL, NCOL = S::NCOL;
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tslot;
  __shared__ volatile int stop;
  const MixArgs &a = ta.m;
  // the warp's number from a shuffle, so that the compiler sees it uniform
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int mi = item.x;
  constexpr int NP = S::NP;
  // the pairs of the item: one tile of kRows, or (DUAL) as many as kSynTwoTiles says
  const int p0 = item.y & ~kSynTwoTiles, np = S::DUAL && (item.y & kSynTwoTiles) ? 2 * tc::kRows : tc::kRows;
  int pr[NP], lj[NP];
  bool valid[NP];
  const float4 *jrec[NP];
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    pr[t] = p0 + NP * tid + t;
    valid[t] = pr[t] < min(a.npairs, p0 + np);
  }
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax;
  const int nks = (lmax - l0 + tc::kK) / tc::kK;
  const int64_t co = a.coef_off[mi] - l0;
  const float4 *__restrict__ cf = a.coef32 + co;
  unsigned char *const Abuf = smem;
  float4 *const stage = reinterpret_cast<float4 *>(smem + S::A_BYTES);
  unsigned char *const Bt = smem + S::A_BYTES + S::ST_BYTES;
  // column c of pair t of this thread at accs[(t NCOL + c) * 128 + tid]
  f2 *const accs = reinterpret_cast<f2 *>(Bt + S::B_BYTES);
  float *const umax = reinterpret_cast<float *>(Bt + S::B_BYTES + S::ACC_BYTES);

  // the staged rows of K-step ks: thread t loads entries t, t + 128, ... (zero past lmax)
  float4 pf[S::PF];
  auto prefetch = [&](int ks) {
    const int lb = l0 + ks * tc::kK;
#pragma unroll
    for (int i = 0; i < S::PF; ++i) {
      const int e = tid + i * tc::kRows;
      pf[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e < S::STG) {
        const int k = e / S::ROW, c = e % S::ROW, l = lb + k;
        if (l <= lmax) pf[i] = c < 1 ? __ldg(cf + l) : __ldg(a.alm32 + (int64_t)(c - 1) * a.ncoef + co + l);
        if (SPIN && c > 0 && !(c & 1) && (k & 1)) pf[i] = make_float4(-pf[i].x, -pf[i].y, -pf[i].z, -pf[i].w);  // s M
      }
    }
  };
  auto stage_store = [&](int ks) {
    float4 *dst = stage + (ks & 1) * S::STG;
#pragma unroll
    for (int i = 0; i < S::PF; ++i) {
      const int e = tid + i * tc::kRows;
      if (e < S::STG) dst[e] = pf[i];
    }
  };
  __shared__ int kstart[tc::kRows / 32];
  // the K-step (block of 16 degrees) at which this pair's terms start (join record);
  // the CTA starts at its pairs' earliest
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    jrec[t] = a.join + ((size_t)mi * a.npairs + (valid[t] ? pr[t] : 0)) * 3;
    lj[t] = valid[t] ? __float_as_int(__ldg(jrec[t] + 2).z) : lmax + 1;
  }
  const int jmin = min(lj[0], lj[NP - 1]);
  {
    const int kj = jmin <= lmax ? (jmin - l0) / tc::kK : nks;
    const int wmin = __reduce_min_sync(0xffffffffu, kj);
    if ((tid & 31) == 0) kstart[warp] = wmin;
  }
  if (warp == 0) tc::tmem_alloc(&tslot, S::TCOLS);
  if (tid == 0) {
    tc::bar_init(&mbar);
    stop = 0;
  }
  for (int i = tid; i < S::B_BYTES / 16; i += tc::kRows) reinterpret_cast<uint4 *>(Bt)[i] = make_uint4(0, 0, 0, 0);
  if (tid < 2 * S::NV) umax[tid] = 0.f;
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = tslot;
  const uint32_t lane = tbase + ((uint32_t)(warp * 32) << 16);
  int ks0 = kstart[0];
#pragma unroll
  for (int w = 1; w < tc::kRows / 32; ++w) ks0 = min(ks0, kstart[w]);
  if (ks0 < nks) {  // its rows; the first K-step's window barrier orders them before any read
    prefetch(ks0);
    stage_store(ks0);
  }
#pragma unroll
  for (int c = 0; c < NP * NCOL; ++c) accs[c * tc::kRows + tid] = f2{0.f, 0.f};

  // the recursions, on Lambda / u_p: zero until the pair joins (no terms, and a
  // recursion of zeros).  Spin 0 without DUAL runs one lane.
  double xd[NP];
  bool near = false;
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    xd[t] = a.pairs[valid[t] ? pr[t] : 0].x;
    near = near || near_pole(xd[t], valid[t]);
  }
  const bool polar = __any_sync(0xffffffffu, near);
  Dual<!S::DUAL, S::DUAL ? kPacked : kCalled> rec;
  rec.p = rec.q = d2{both(0.f), both(0.f)};
#pragma unroll
  for (int t = 0; t < NP; ++t) rec.x[t] = node_of(xd[t], polar);
  int sc0 = 0, sc1 = 0;
  const int lfast = SPIN ? fast_from(as, rec.x[0].h, valid[0], lmax) : 0;
  float racc[NP][NCOL];
#pragma unroll
  for (int t = 0; t < NP; ++t)
#pragma unroll
    for (int c = 0; c < NCOL; ++c) racc[t][c] = 0.f;
  float2 wf = both(1.f);  // weights of the two lanes' values; scales change only at the rescale checks
  bool settled = false;   // every lane of the warp at scale 0 (warp-uniform; scales only rise)

  // one step of the recursions with a row's coefficients
  auto advance = [&](const StepMode mode, const float4 &c) {
    if (SPIN || S::DUAL) {
      rec.step(mode, c);
    } else {
      f2 lc = lane0(rec.p), lp = lane0(rec.q);
      step_s0(Coef32{{c.x, c.y}, {0.f, 0.f}}, rec.x[0], mode == kPolar, lc, lp);
      rec.start(0, lc, lp, 1.f);
    }
  };
  // PACK degrees from rows (lb - l0 even): digits (quanta 2^-7, 2^-15, 2^-23) packed
  // per pair of degrees into pk[set][digit][q / 2], remainders contracted into racc,
  // recursion advanced.  Unless every lane is at scale 0 (kFast; a polar warp tests
  // too) the values take their weights, and every second degree the warp votes: if
  // every lane's values are negligible for the next two steps (as in the double-float
  // kernels) the digits are zero and only the recursion runs.
  auto part = [&](const StepMode mode, const float4 *rows,
                  uint32_t (&pk)[NL][tc::kLamDigits][S::PACK / 2]) __attribute__((always_inline)) {
    constexpr float s0 = 98304.0f, s1 = s0 * 0x1p-8f, s2 = s0 * 0x1p-16f;  // 1.5 * 2^23 * quantum
    float2 dlo[tc::kLamDigits];
    bool dead = false;
#pragma unroll
    for (int q = 0; q < S::PACK; ++q) {
      // past lmax the staged rows are zero: the recursion runs on zero coefficients
      // (values of one degree's size, alternating) and meets zero a_lm, so those degrees
      // add nothing and need no test
      const bool odd = q & 1;
      if (!odd && mode != kFast)
        dead = !settled && __all_sync(0xffffffffu, negligible(lane0(rec.p), sc0) && (NL == 1 || negligible(lane1(rec.p), sc1)));
      const float4 *row = rows + q * S::ROW;  // this degree's staged coefficients and a_lm
      float2 d[tc::kLamDigits] = {both(0.f), both(0.f), both(0.f)};
      if (mode == kFast || !dead) {
        float2 h = rec.p.h, lo = rec.p.l;
        if (mode != kFast) {
          const float2 f = make_float2(wf.x, (SPIN && mode == kPolar && odd) ? -wf.y : wf.y);
          h = mul2(h, f);
          lo = mul2(lo, f);
        }
        float2 rr;
        if (NL == 2) {
          auto round2 = [](float2 r, float c) { return add2(add2(r, both(c)), both(-c)); };
          d[0] = round2(h, s0);
          rr = sub2(h, d[0]);
          d[1] = round2(rr, s1);
          rr = sub2(rr, d[1]);
          d[2] = round2(rr, s2);
          rr = add2(sub2(rr, d[2]), lo);
        } else {
          d[0].x = tc::round_to(h.x, s0);
          float r = __fsub_rn(h.x, d[0].x);
          d[1].x = tc::round_to(r, s1);
          r = __fsub_rn(r, d[1].x);
          d[2].x = tc::round_to(r, s2);
          rr.x = __fadd_rn(__fsub_rn(r, d[2].x), lo.x);
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          if (SPIN) {
            const float4 P = row[1 + 2 * j];
            const float4 M = row[2 + 2 * j];  // s M
            racc[0][8 * j + 0] = __fmaf_rn(rr.x, P.x, racc[0][8 * j + 0]);
            racc[0][8 * j + 1] = __fmaf_rn(rr.x, P.z, racc[0][8 * j + 1]);
            racc[0][8 * j + 2] = __fmaf_rn(rr.x, M.x, racc[0][8 * j + 2]);
            racc[0][8 * j + 3] = __fmaf_rn(rr.x, M.z, racc[0][8 * j + 3]);
            racc[0][8 * j + 4] = __fmaf_rn(rr.y, M.x, racc[0][8 * j + 4]);
            racc[0][8 * j + 5] = __fmaf_rn(rr.y, M.z, racc[0][8 * j + 5]);
            racc[0][8 * j + 6] = __fmaf_rn(rr.y, P.x, racc[0][8 * j + 6]);
            racc[0][8 * j + 7] = __fmaf_rn(rr.y, P.z, racc[0][8 * j + 7]);
          } else {
            const float4 v = row[1 + j];
            const int c = 4 * j + (odd ? 2 : 0);
            racc[0][c] = __fmaf_rn(rr.x, v.x, racc[0][c]);
            racc[0][c + 1] = __fmaf_rn(rr.x, v.z, racc[0][c + 1]);
            if (S::DUAL) {
              racc[NP - 1][c] = __fmaf_rn(rr.y, v.x, racc[NP - 1][c]);
              racc[NP - 1][c + 1] = __fmaf_rn(rr.y, v.z, racc[NP - 1][c + 1]);
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < tc::kLamDigits; ++i) {
        if (!odd) {
          dlo[i] = d[i];
        } else {
          pk[0][i][q / 2] = tc::pack_bf16(dlo[i].x, d[i].x);
          if (NL == 2) pk[NL - 1][i][q / 2] = tc::pack_bf16(dlo[i].y, d[i].y);
        }
      }
      advance(mode, row[0]);
    }
  };
  // enhanced exponent: rescale every eight degrees (see mixed_common.cuh)
  auto rescale = [&]() {
    if (settled) return;
    rec.rescale(sc0, sc1);
    wf = make_float2(scale_weight(sc0), scale_weight(sc1));
    settled = __all_sync(0xffffffffu, sc0 == 0 && sc1 == 0);
  };
  // this thread's digits of degrees q0 .. q0 + PACK - 1 of the K-step into the A tiles
  auto store_a = [&](int q0, const uint32_t (&pk)[NL][tc::kLamDigits][S::PACK / 2]) {
#pragma unroll
    for (int t = 0; t < NL; ++t)
#pragma unroll
      for (int i = 0; i < tc::kLamDigits; ++i) {
        unsigned char *dst = Abuf + (t * tc::kLamDigits + i) * tc::kATile + (tid / 8) * 256 + (q0 / 8) * 128 +
                             (tid % 8) * 16 + (q0 % 8) * 2;
        if constexpr (S::PACK == 8)
          *reinterpret_cast<uint4 *>(dst) = make_uint4(pk[t][i][0], pk[t][i][1], pk[t][i][2], pk[t][i][3]);
        else
          *reinterpret_cast<uint2 *>(dst) = make_uint2(pk[t][i][0], pk[t][i][1]);
      }
  };

  // the MMAs of one K-step, issued in order by one thread: for each Lambda set t and
  // digit i, the a_lm digit windows (j0, j0 + 1), j0 = -(i mod 2), j0 + 2, ... up to
  // the last digit with i + j <= 5, into levels (i + j0, i + j0 + 1); in a window's
  // first K-step the set-0, digit-0 products come first and overwrite levels 0 .. 5
  // (every level written), the rest accumulate.  The zero tile of digit -1 fills
  // the odd windows' first halves; the i = 2 windows end at digit 3.
  const uint64_t adesc0 = tc::mat_desc(tc::smem_u32(Abuf), 128, 256);
  const uint64_t bdesc0 = tc::mat_desc(tc::smem_u32(Bt), 128, 256);
  auto issue = [&](int ks) {
    tc::fence_after();
    constexpr uint32_t idesc = tc::instr_desc(tc::kRows, S::N);
    const bool first = (ks % tc::kWin) == 0 || ks == ks0;
#pragma unroll
    for (int t = 0; t < NL; ++t)
#pragma unroll
      for (int i = 0; i < tc::kLamDigits; ++i)
#pragma unroll
        for (int j0 = -(i & 1); j0 <= tc::kAlmDigits - 1 && i + j0 < tc::kLevels; j0 += 2) {
          const uint64_t ad = adesc0 + (uint64_t)(((t * tc::kLamDigits + i) * tc::kATile) >> 4);
          const int tb = SPIN ? t : 0, td = S::DUAL ? t : 0;  // B stack, accumulators
          const uint64_t bd = bdesc0 + (uint64_t)((tb * S::NDT * S::DTILE + (j0 + 1) * S::DTILE) >> 4);
          tc::mma_bf16(tbase + td * S::COLS1 + (i + j0) * S::NCW, ad, bd, idesc,
                       (first && t == td && i == 0) ? 0u : 1u);
        }
    tc::mma_commit(&mbar);
  };

  // after a window: the six levels of this thread's lane plus the remainder sums,
  // added to the double-float column sums
  auto readout = [&]() {
#pragma unroll
    for (int cc = 0; cc < NP * NCOL; cc += NCOL < 8 ? NCOL : 8) {
      const int pt = cc / NCOL, c0 = cc % NCOL;
      uint32_t dv[tc::kLevels][8];
#pragma unroll
      for (int k = 0; k < tc::kLevels; ++k) tc::tmem_ld8(lane + pt * S::COLS1 + k * S::NCW + c0, dv[k]);
      tc::tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c0 + c >= NCOL) break;
        f2 t = {__uint_as_float(dv[0][c]), 0.f};
#pragma unroll
        for (int k = 1; k < tc::kLevels; ++k) t = f2_add_lazy(t, f2{__uint_as_float(dv[k][c]), 0.f});
        t = f2_add_lazy(t, f2{racc[pt][c0 + c], 0.f});
        racc[pt][c0 + c] = 0.f;
        f2 &acc = accs[(pt * NCOL + c0 + c) * tc::kRows + tid];
        acc = f2_add(acc, t);
      }
    }
  };

  int ncommit = 0, nwaited = 0;
  bool ok = true;
  // waits for the last commit (mostly done: no clock read); a wait that gives up sets
  // `stop`, which ends the later ones at once, and the CTA leaves at its window's end
  auto wait_mma = [&]() -> bool {
    const uint32_t par = (uint32_t)(ncommit - 1) & 1u;
    return tc::bar_try(&mbar, par) || tc::bar_wait_or(&mbar, par, &stop);
  };
  for (int ks = ks0; ks < nks; ++ks) {
    const int lb = l0 + ks * tc::kK;
    if (ks % tc::kWin == 0 || ks == ks0) {  // column bounds of this window's a_lm (from lb on)
      float *um = umax + ((ks / tc::kWin) & 1) * S::NV;
      if (tid < S::NV) umax[(((ks / tc::kWin) & 1) ^ 1) * S::NV + tid] = 0.f;  // the other window's, for later
      const int lw1 = l0 + (ks / tc::kWin + 1) * tc::kWin * tc::kK - 1;
      tc::window_bounds<NJ, SPIN>(a, co, lb, lw1 < lmax ? lw1 : lmax, um);
      __syncthreads();
    }
    // pairs joining here take the recursion state where their terms start, over u_p
    bool joins = false;
#pragma unroll
    for (int t = 0; t < NP; ++t)
      if (lj[t] == lb) {
        const JoinRec r = ld_join(jrec[t], polar);
        const float ulx = __int_as_float((127 - r.lexp) << 23);
        rec.start(t, r.lpc, r.lpp, ulx);
        (t ? sc1 : sc0) = r.scp;
        if (SPIN) {  // lane 1 holds s l- (l- itself in a polar warp): the previous degree's sign is -1
          rec.start(1, r.lmc, polar ? r.lmp : neg(r.lmp), ulx);
          sc1 = r.scm;
        }
        wf = make_float2(scale_weight(sc0), scale_weight(sc1));
        joins = true;
      }
    if (__any_sync(0xffffffffu, joins)) settled = __all_sync(0xffffffffu, sc0 == 0 && sc1 == 0);
    // a warp none of whose lanes has joined holds zeros: it skips the recursion
    const bool wlive = __any_sync(0xffffffffu, jmin <= lb);
    const float4 *rows = stage + (ks & 1) * S::STG;
    if (ks + 1 < nks) prefetch(ks + 1);  // its latency hides behind this K-step's work
    bool fail = false;
#pragma unroll 1
    for (int q0 = 0; q0 < tc::kK; q0 += S::PACK) {
      uint32_t pk[NL][tc::kLamDigits][S::PACK / 2];
      if (wlive) {
        if (polar) part(kPolar, rows + q0 * S::ROW, pk);
        else if (settled && lb >= lfast) part(kFast, rows + q0 * S::ROW, pk);
        else part(kCareful, rows + q0 * S::ROW, pk);
      } else {  // no lane of the warp has joined: zero digits, and nothing to advance
#pragma unroll
        for (int t = 0; t < NL; ++t)
#pragma unroll
          for (int i = 0; i < tc::kLamDigits; ++i)
#pragma unroll
            for (int q = 0; q < S::PACK / 2; ++q) pk[t][i][q] = 0u;
      }
      if ((q0 + S::PACK) % 8 == 0) rescale();  // after every eight degrees
      // the previous K-step's MMAs read the A and B tiles: wait for them before
      // the first write (they have long finished by now)
      if (q0 == 0 && ncommit > nwaited) {
        fail = !wait_mma();
        nwaited = ncommit;
      }
      if (!fail) store_a(q0, pk);
      // (between the halves: the warps that build B reach the barrier later by less)
      if (q0 == 0 && !fail) tc::build_b<NJ, SPIN>(rows, umax + ((ks / tc::kWin) & 1) * S::NV, Bt);
    }
    if (ks + 1 < nks) stage_store(ks + 1);  // its buffer's last readers finished before the previous barrier
    tc::fence_async_smem();
    if (fail) stop = 1;
    __syncthreads();
    if (warp == tc::kIssuerWarp && tc::elect_one()) issue(ks);
    ++ncommit;
    if (ks % tc::kWin == tc::kWin - 1 || ks == nks - 1) {
      fail = !wait_mma();
      nwaited = ncommit;
      if (__syncthreads_or(fail || stop)) {
        ok = false;
        break;
      }
      tc::fence_after();
      readout();
      tc::fence_before();
    }
  }
  if (!ok) {  // a wait gave up: flag it, give the MMAs in flight a bounded wait, release TMEM
    if (tid == 0) atomicOr(ta.err, 1);
    if (ncommit > nwaited) tc::bar_wait(&mbar, (uint32_t)(ncommit - 1) & 1u);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, S::TCOLS);
  if (!ok) return;
#pragma unroll
  for (int t = 0; t < NP; ++t) {
    if (!valid[t]) continue;
    const int p = pr[t], lexp = __float_as_int(__ldg(jrec[t] + 2).w);
    const double u = __hiloint2double((1023 + lexp) << 20, 0);  // u_p
    auto colsum = [&](int c) { return u * f2_val(accs[(t * NCOL + c) * tc::kRows + tid]); };
    if (SPIN) {
      const double sig = (as & 1) ? -1.0 : 1.0;
      const double h0 = ((l0 + m) & 1) ? -0.5 : 0.5;
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const double n1r = colsum(8 * j + 0), n1i = colsum(8 * j + 1);
        const double s4r = colsum(8 * j + 2), s4i = colsum(8 * j + 3);
        const double n2r = colsum(8 * j + 4), n2i = colsum(8 * j + 5);
        const double s3r = colsum(8 * j + 6), s3i = colsum(8 * j + 7);
        const double ar = n1r + sig * n2r, ai = n1i + sig * n2i;
        const double br = sig * n2r - n1r, bi = sig * n2i - n1i;
        const double cr = s3r + sig * s4r, ci = s3i + sig * s4i;
        const double dr = sig * s4r - s3r, di = sig * s4i - s3i;
        double2 qn = make_double2(-0.5 * ar, -0.5 * ai);
        double2 un = make_double2(0.5 * bi, -0.5 * br);
        double2 qs = make_double2(-h0 * cr, -h0 * ci);
        double2 us = make_double2(h0 * di, -h0 * dr);
        if (m == 0) qn.y = qs.y = un.y = us.y = 0.0;
        double2 *oq = a.phase + (((size_t)(2 * j) * a.nm + mi) * a.npairs + p) * 2;
        double2 *ou = a.phase + (((size_t)(2 * j + 1) * a.nm + mi) * a.npairs + p) * 2;
        oq[0] = qn;
        oq[1] = qs;
        ou[0] = un;
        ou[1] = us;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const double e0 = colsum(4 * j + 0), e1 = colsum(4 * j + 1);
        const double o0 = colsum(4 * j + 2), o1 = colsum(4 * j + 3);
        double2 fn = make_double2(e0 + o0, e1 + o1), fs = make_double2(e0 - o0, e1 - o1);
        if (m == 0) fn.y = fs.y = 0.0;
        double2 *o = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
        o[0] = fn;
        o[1] = fs;
      }
    }
  }
}

}  // namespace sht

namespace sht {

template <int NJ, bool SPIN, bool TWO>
__global__ void __launch_bounds__(tc::kRows, tc::Shape<NJ, SPIN, TWO>::MINB) tc_syn(TcArgs ta) {
  extern __shared__ __align__(128) unsigned char tc_smem[];
  tc_syn_body<NJ, SPIN, TWO>(ta, ta.m.syn_items[blockIdx.x], tc_smem);
}

// batches: item (mi, first pair, -, record); the record holds the plan's arguments
template <int NJ, bool SPIN, bool TWO>
__global__ void __launch_bounds__(tc::kRows, tc::Shape<NJ, SPIN, TWO>::MINB)
    tc_syn_batch(const TcArgs *__restrict__ args, const int4 *__restrict__ items) {
  extern __shared__ __align__(128) unsigned char tc_smem[];
  const int4 it = items[blockIdx.x];
  tc_syn_body<NJ, SPIN, TWO>(args[it.w], make_int2(it.x, it.y), tc_smem);
}

template <int NJ, bool SPIN, bool TWO>
static cudaError_t tc_set_smem() {
  // the request, and a shared-memory carveout that lets the compiled number of CTAs fit
  cudaError_t e = cudaFuncSetAttribute(tc_syn_batch<NJ, SPIN, TWO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       tc::Shape<NJ, SPIN, TWO>::SMEM_LAUNCH);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tc_syn<NJ, SPIN, TWO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             tc::Shape<NJ, SPIN, TWO>::SMEM_LAUNCH);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tc_syn_batch<NJ, SPIN, TWO>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(tc_syn<NJ, SPIN, TWO>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  return e;
}

// shared-memory attributes of every instance (once per device, at plan time)
cudaError_t tc_prepare_device() {
  cudaError_t e = tc_set_smem<1, false, false>();
  if (e == cudaSuccess) e = tc_set_smem<1, false, true>();
  if (e == cudaSuccess) e = tc_set_smem<2, false, false>();
  if (e == cudaSuccess) e = tc_set_smem<2, false, true>();
  if (e == cudaSuccess) e = tc_set_smem<4, false, false>();
  if (e == cudaSuccess) e = tc_set_smem<8, false, false>();
  if (e == cudaSuccess) e = tc_set_smem<1, true, false>();
  if (e == cudaSuccess) e = tc_set_smem<2, true, false>();
  if (e == cudaSuccess) e = tc_set_smem<4, true, false>();
  return e;
}

bool tc_supported(int spin, int njobs_pad) {
  return spin == 0 ? njobs_pad <= 8 : njobs_pad <= 4;
}

// One or two spin-0 maps: two pairs a thread where the 128-pair tiles fill the chip at
// least kTwoPerSm times over.  It saves issue slots (the two lanes' recursions and
// digits are packed) but halves the CTAs, whose fixed cost per block of degrees is then
// longer: two maps on Gauss-Legendre rings, one pair a thread against two, lmax 511
// 132 / 156 us, 1023 (27 tiles per SM) 567 / 583, HEALPix 1535 (81) 2128 / 1846, 2047
// (108) 3600 / 3130, 4095 25.6 / 20.9 ms.
bool tc_syn_two_tiles(const sht_plan_s *P, int64_t tiles) {
  constexpr int kTwoPerSm = 40;
  return P->precision == SHT_MIXED && P->spin == 0 && P->njobs_pad <= 2 && tiles >= (int64_t)kTwoPerSm * P->sms;
}

namespace {
// calls f with the shape of a spin class, padded job count and pairs per thread; false: none
template <int NJ, bool SPIN, bool TWO>
struct SynShape {
  static constexpr int nj = NJ;
  static constexpr bool spin = SPIN, two = TWO;
  static constexpr int smem = tc::Shape<NJ, SPIN, TWO>::SMEM_LAUNCH;
};
template <class F>
bool syn_shape(int spin, int nj, bool two, F &&f) {
  if (spin == 0) {
    switch (nj) {
      case 1: two ? f(SynShape<1, false, true>()) : f(SynShape<1, false, false>()); return true;
      case 2: two ? f(SynShape<2, false, true>()) : f(SynShape<2, false, false>()); return true;
      case 4: f(SynShape<4, false, false>()); return true;
      case 8: f(SynShape<8, false, false>()); return true;
    }
  } else {
    switch (nj) {
      case 1: f(SynShape<1, true, false>()); return true;
      case 2: f(SynShape<2, true, false>()); return true;
      case 4: f(SynShape<4, true, false>()); return true;
    }
  }
  return false;
}
}  // namespace

float tc_lambda_bound(int lmax) {
  // |sLambda_lm| <= sqrt((2l + 1) / (4 pi)) (|d^l| <= 1) up to l = lmax + 1 (the
  // kernel computes one value past lmax); the next power of two above it, with
  // room for the recursion's rounding
  const double b = sqrt((2.0 * lmax + 3.0) / (4.0 * M_PI)) * (1.0 + 1e-6);
  return (float)exp2(ceil(log2(b)));
}

size_t tc_args_size() { return sizeof(TcArgs); }

void leg_tc_fill_args(const sht_plan_s *P, int polar, void *out) {
  TcArgs ta;
  leg_mixed_fill_args(P, polar, &ta.m);
  ta.err = P->d_err;
  ta.force = P->quad_off;
  memcpy(out, &ta, sizeof(ta));
}

cudaError_t launch_leg_tc_batch(int spin, int nj, bool two, const void *targs, const int4 *items, int n,
                                cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const TcArgs *a = static_cast<const TcArgs *>(targs);
  const bool ok = syn_shape(spin, nj, two, [&](auto sh) {
    using H = decltype(sh);
    tc_syn_batch<H::nj, H::spin, H::two><<<n, tc::kRows, H::smem, st>>>(a, items);
  });
  return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

cudaError_t launch_leg_tc_syn(const sht_plan_s *P, const void *mixargs, int n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  TcArgs ta;
  memcpy(&ta.m, mixargs, sizeof(MixArgs));
  ta.err = P->d_err;
  ta.force = P->quad_off;
  const bool ok = syn_shape(P->spin, P->njobs_pad, P->syn_two != 0, [&](auto sh) {
    using H = decltype(sh);
    tc_syn<H::nj, H::spin, H::two><<<n, tc::kRows, H::smem, st>>>(ta);
  });
  return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

}  // namespace sht
