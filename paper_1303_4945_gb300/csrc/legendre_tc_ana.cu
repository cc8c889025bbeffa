// legendre_tc_ana.cu -- the mixed form's Legendre analysis (Eq. ana1) with the
// contraction over ring pairs on the tensor cores (tcgen05).
//
// For one m and a tile of 128 ring pairs the analysis adds, for every degree l,
// a[l][c] = sum_p G[c][p] Lambda[p][l]: the columns c are the phase values of the
// ring pairs combined for the parity of l - l0 and the spin (Sect. 3.2's loop over
// rings inside the loop over l, Fig. 2), Lambda comes from the double-float
// recursion of Sect. 4.1, one thread per ring pair walking l.  The contraction
// runs transposed, D[c][l] = sum_p G[c][p] Lambda[p][l]: M = the columns' digit
// rows, K = the ring pairs, N = degrees, so that each thread writes its own pair's
// values along N (the Lambda operand in the MN-major layout) and the G operand is
// built once per tile.  Both operands are split exactly into bf16 digits on common
// grids (an Ozaki-style error-free split):
//
//  * Lambda / u_p = L0 + ... + L5 with quanta q_i = 2^-7, -15, -23, -31, -40, -49, u_p a power of two
//    bounding the pair's true values from its join block on (join record), so
//    |Lambda / u_p| < 1; the pair's factor u_p moves into its G values.
//  * G'[c][p] = G[c][p] u_p = G0 + ... + G5 with quanta v_c q_j, v_c the power of
//    two above column c's largest |G'| over the tile (it enters when the sums are
//    stored, so that the range is FP64's).
//  * Every product Gj Li is a multiple of v_c q_i q_j; a digit is at most 128 of its
//    quanta (192 for digit 3, which takes the low word, 256 for digits 4 and 5, whose
//    quanta are one and two bits finer: at no cost a quarter of the split's error), so
//    a sum over K = 512 entries stays within 512 * 256 * 128 = 2^24 quanta (of
//    512 * 192^2 for the product of two digits 3, level 6, only its rounding below
//    2^-70 could depend on the order) and the FP32 accumulation is exact whatever its
//    order.
//
// One MMA per 16 entries: M = 64 rows (a column's six G digits and two zero rows
// together), N = 48 (the six Lambda digits of 8 degrees), so D holds every digit
// product G_j L_i of a column and degree, each an exact sum; the products with i + j
// <= 2 are added in double-float, those with 3 <= i + j <= 6 in FP32 (below 2^-24 of
// the sum), the rest dropped (below 2^-56).
//
// Each warp owns the K entries of its 32 threads: it writes their Lambda digits and
// issues their MMAs itself, with no CTA barrier per block.  TMEM accumulators of 48
// columns rotate between blocks of 8 degrees; mbarriers order the steps: a warp's own
// commits free its Lambda tiles, every warp's commit (or plain arrival for a warp with
// no joined pair) fills an accumulator, and the warps whose turn it is read its rows,
// zero and release it.  Every wait is bounded; a wait that gives up flags the plan's
// status word and stops the CTA.
//
// What bounds it (GB300, spin 2, lmax 4095): issue slots and dependency latency on the
// CUDA cores (59% issue, FP32 pipe 48%, tensor pipe 25% at 16 warps per SM).  With
// parts left out: recursion and digits 37 ms, MMA issue 3.5, accumulator reads 7.5 (of
// which 6 are warps waiting for one another, 1.2 the TMEM loads), level sums 3.2.
// History: scalar recursions with three coefficients, 128 threads per CTA, every wait
// reading the clock, MMAs issued through a divergent lane 73.9 ms; unit-coefficient
// recursion 65; both recursions as packed lanes 55.7; 256 threads, four accumulators
// read in turn by two groups 57.0; waits that try once before reading the clock and
// MMAs from an elected lane with uniform descriptors 53.5; the block's two halves
// unrolled 51.4.  Coefficients staged in shared memory (56.7 against 55.7) and pairs
// interleaved over the warps (54.4 against 51.4) were slower.
#include <math_constants.h>

#include "dual.cuh"
#include "mix_ana.cuh"
#include "tcgen05.cuh"

namespace sht {
namespace tca {

constexpr int kTile = 128;       // ring pairs per tile of the work lists
constexpr int kBlk = 8;          // degrees per block
constexpr int kDig = 6;          // digits of Lambda / u_p and of G'
constexpr int kN = kDig * kBlk;  // MMA N: every Lambda digit of the block's degrees
constexpr int kColRows = 8;      // A rows per column: its six G digits, two zero rows
constexpr int kDCols = 64;       // TMEM columns per accumulator (kN used)
constexpr int kEStride = kN + 4; // floats per staged D row (rows 16 bytes off the banks of the next)

// Columns per job j: 4j + {0, 1} and 4j + {2, 3} (re, im of the two sums the
// kernel below describes).  A thread runs the two recursions of Dual; its value of
// lane t is K entry t TH + tid.  Column c's six G digit rows and two zero rows make 8
// rows of A and of D.
//
// One job: 256 threads, four accumulators, one column in each TMEM quarter.  Reading
// an accumulator back (waits, loads, zeroing, the sum over the digit products) costs a
// warp about 75 instructions for 8 degrees whatever K is, so twice the pairs per CTA
// halve it, and each group of four warps reads every second block, one column a warp,
// two blocks after its products were issued.  (128 threads, two accumulators, both
// columns of a quarter read by warps 0 and 1, which share their SM quarters with those
// of the other CTAs: 55.7 ms at spin 2, lmax 4095.)  Two jobs take twice the A digits:
// 128 threads, two columns a quarter, every warp reads every block.
//
// Four jobs (spin 0; plans of more run four at a time, QUAD): M = 128, a quarter per job.
// A's six rows per column are packed without the zero rows (an 8-row group's last two
// rows are the next column's first digits, and no one reads their products), so that
// three CTAs fit an SM; the quarter's warp keeps the four degrees of a column's parity
// and sums over its digit rows through a 608-byte buffer, one Lambda digit at a time.
// GB300, lmax 2047, per four maps 5.0 ms (the double-float contraction 10.4; of eight
// maps in one recursion 18.7): 12 warps per SM, as A's digits of 16 columns fill the
// shared memory; eight maps' would leave room for 8 warps.
template <int NJ, bool SPIN>
struct AnaShape {
  static constexpr int TH = NJ == 1 ? 256 : 128;
  static constexpr int WARPS = TH / 32;
  static constexpr int NP = SPIN ? 1 : 2;                // ring pairs per thread
  static constexpr bool QUAD = NJ == 4;
  static constexpr bool GROUPED = QUAD || (SPIN && NJ == 2);  // runs plans of more jobs NJ at a time
  static constexpr int TILE = QUAD ? 2 * kTile : kTile;  // ring pairs per tile of the work list
  static constexpr int TILES = NP * TH / TILE;           // tiles walked at a time
  static constexpr int NACC = NJ == 1 ? 4 : 2;           // accumulators
  static constexpr int GROUPS = WARPS / 4;               // groups of reading warps (block ib: group ib % GROUPS)
  static constexpr int LAG = NJ == 1 ? 2 : 1;            // blocks between issuing and reading (a multiple of GROUPS)
  static constexpr int NSET = 2;
  static constexpr int NC = 4 * NJ;
  static constexpr int CPW = NC / 4;                     // columns per TMEM quarter
  static constexpr int KG = NSET * TH / 8;               // 8-entry K-groups
  // MMA M = 64: D row r lands in TMEM lane 32 (r / 16) + r % 16 (measured): warp w
  // reads quarter w % 4, its columns' rows in lanes 0 .. 8 CPW - 1.  The rows of one
  // K-group are contiguous.  One column a quarter: 8-row groups 64 bytes apart put
  // column c in row group 2c (the odd groups overlap two columns; no one reads them).
  static constexpr int M = QUAD ? 128 : 64;         // MMA M: the columns' digit rows
  static constexpr int A_ROWS = QUAD ? kDig : kColRows;  // rows stored per column
  static constexpr int A_LBO = NC * A_ROWS * 16;    // bytes between K-groups
  static constexpr int A_SBO = QUAD ? A_ROWS * 16 : (CPW == 1 ? 64 : 128);  // bytes between 8-row groups
  static constexpr int A_BYTES = KG * A_LBO;
  // byte offset of (column c, digit row j, K-group h)
  __host__ __device__ static constexpr int a_at(int c, int j, int h) { return h * A_LBO + (A_ROWS * c + j) * 16; }
  static constexpr int KSTRIDE = QUAD ? 128 : 144;  // bytes between 8-pair K-groups of the Lambda tiles
  static constexpr int B_SBO = KG * KSTRIDE;  // bytes between the 8-degree N-groups (one per digit)
  static constexpr int B_BYTES = kDig * B_SBO;
  static constexpr int EROWS = CPW * kColRows;  // staged D rows per warp: lanes 0 .. EROWS - 1
  // staged floats per warp (QUAD: four degrees of eight rows, columns 10 rows apart, off
  // one another's banks)
  static constexpr int E_FLOATS = QUAD ? (3 * 10 + 8) * 4 : EROWS * kEStride;
  static constexpr int E_BYTES = WARPS * E_FLOATS * 4;
  static constexpr int SMEM = A_BYTES + B_BYTES + E_BYTES;
  static constexpr int TCOLS = NACC * kDCols;
  // at most 512 / TCOLS CTAs per SM, so that their TMEM allocations never wait
  static constexpr int SMEM_FLOOR = (228 * 1024) / (512 / TCOLS + 1) - 1024 + 1;
  static constexpr int SMEM_LAUNCH = SMEM > SMEM_FLOOR ? SMEM : SMEM_FLOOR;
  static constexpr int V = (SPIN ? 4 : 2) * NJ;  // partial sums per degree (QUAD: of the CTA's jobs)
  static constexpr int MINB = NJ == 1 ? 2 : 3;
  static_assert(kColRows * NC <= M && (CPW <= 2 || QUAD) && !(QUAD && SPIN), "columns within the MMA's rows");
  static_assert(LAG % GROUPS == 0 && LAG < NACC, "a group reads the blocks it holds the turn of");
  // the MMA reads M / 8 row groups of two K-groups from a K-step's base: from the last
  // one's, inside A and the B tiles that follow it
  static_assert((KG - 1) * A_LBO + (M / 8 - 1) * A_SBO + 128 <= A_BYTES + B_BYTES, "A operand inside shared memory");
  static_assert(A_BYTES % 16 == 0 && B_SBO % 16 == 0, "descriptor alignment");
  static_assert(MINB * (SMEM_LAUNCH + 1024 + 512) <= 228 * 1024, "CTAs per SM");
};

// the exponent of the power of two above a number whose magnitude has the upper word hi
// (kept so that its reciprocal and it are normal numbers)
__device__ __forceinline__ int exp_above(unsigned hi) { return min(max((int)(hi >> 20) - 1022, -1022), 1022); }

// the upper word of a magnitude times 2^e (as a bound: kept within the finite numbers)
__device__ __forceinline__ unsigned add_exp(unsigned hi, int e) { return (unsigned)min(max((int)hi + (e << 20), 0), 0x7fefffff); }
__device__ __forceinline__ bool not_finite(unsigned hi) { return hi >= 0x7ff00000u; }

// six digits of x 2^e, |x 2^e| < 1 (zero unless on), by integer operations: the value in
// quanta of 2^-49, a bias that makes every field below the first one's a digit plus half
// its range, and each field placed under the exponent whose last bit is its quantum.
// (In FP64 the conversions hold the FP64 pipe 80 cycles per value and warp: with them the
// analysis of four maps at lmax 31 took 35.5 us, now 31.8.)
__device__ __forceinline__ void digits6(double x, bool on, int e, float (&d)[kDig]) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int E = (int)((hi >> 20) & 0x7ffu), sh = max(1026 - E - e, 1);
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  uint64_t f = on && E > 0 && sh < 63 ? (m + (1ull << (sh - 1))) >> sh : 0ull;
  if (hi >> 31) f = 0ull - f;
  f += (1ull << 41) + (1ull << 33) + (1ull << 25) + (1ull << 17) + (1ull << 8);
  const uint32_t fh = (uint32_t)(f >> 32), fl = (uint32_t)f;
  // a field of half range h in quanta of 2^-b: 2^(23 - b) + field 2^-b, less 2^(23 - b) + h 2^-b
  auto place = [](uint32_t field, int b, float h) {
    const float base = __uint_as_float((uint32_t)(127 + 23 - b) << 23), q = __uint_as_float((uint32_t)(127 - b) << 23);
    return __fsub_rn(__uint_as_float(__float_as_uint(base) | field), base + h * q);
  };
  d[0] = __fmul_rn(__int2float_rn((int)fh >> 10), 0x1p-7f);
  d[1] = place((fh >> 2) & 255u, 15, 128.f);
  d[2] = place(__funnelshift_r(fl, fh, 26) & 255u, 23, 128.f);
  d[3] = place((fl >> 18) & 255u, 31, 128.f);
  d[4] = place((fl >> 9) & 511u, 40, 256.f);
  d[5] = place(fl & 511u, 49, 256.f);
}

// six digits of two double-float values, |x| < 1: each a multiple of its quantum with at
// most 8 significant bits (at most 128 quanta; 192 for d[3], after the low word enters;
// 256 for d[4] and d[5])
__device__ __forceinline__ void split6(float2 h, float2 l, float2 (&d)[kDig]) {
  constexpr float s0 = 98304.0f;  // 1.5 * 2^23 * 2^-7
  auto round2 = [](float2 r, float s) { return add2(add2(r, both(s)), both(-s)); };
  float2 r = h;
  d[0] = round2(r, s0);
  r = sub2(r, d[0]);
  d[1] = round2(r, s0 * 0x1p-8f);
  r = sub2(r, d[1]);
  d[2] = round2(r, s0 * 0x1p-16f);
  r = add2(sub2(r, d[2]), l);
  d[3] = round2(r, s0 * 0x1p-24f);
  r = sub2(r, d[3]);
  d[4] = round2(r, s0 * 0x1p-33f);
  r = sub2(r, d[4]);
  d[5] = round2(r, s0 * 0x1p-42f);
}

}  // namespace tca

// ---------------------------------------------------------------------------
// Columns' K entries (mixed analysis naming: W+_N, W-_N the north ring's spin
// combinations, W+_S', W-_S' the south ring's times (-1)^(l0 + m)): spin, T1 = sum l+
// W+_N + s l- W+_S' and s T2 = sum l+ W-_S' + s l- W-_N with s = (-1)^(l - l0), so the K
// entries are the +s values and the -s values times s (the two lanes of Dual), and T2
// is s times its row; spin 0, the even-l sum over G_N + G_S and the odd-l sum over
// G_N - G_S, the two lanes two neighbouring pairs.
// ---------------------------------------------------------------------------
template <int NJ, bool SPIN>
__device__ __forceinline__ bool tc_ana_body(const TcArgs &ta, const int4 item_, const int j0, unsigned char *tca_smem) {
  using S = tca::AnaShape<NJ, SPIN>;
  constexpr int NSET = S::NSET, NC = S::NC, kDig = tca::kDig, TH = S::TH, NP = S::NP;
  constexpr int NACC = S::NACC, GROUPS = S::GROUPS, LAG = S::LAG;
  __shared__ __align__(8) uint64_t full[NACC], freeb[NACC], mine[S::WARPS];
  __shared__ uint32_t tslot;
  __shared__ unsigned vmax[NC], eqmax[NC];
  __shared__ int eqok;
  __shared__ int tstart[S::WARPS];
  __shared__ volatile int stop;
  const MixArgs &a = ta.m;
  // the work list's tiles in tiles of this kernel (plans of more than two jobs: 256 pairs)
  const int tmul = S::GROUPED && !S::QUAD && a.nj > NJ ? 2 : 1;
  const int4 item = make_int4(item_.x, item_.y * tmul, ((item_.z >> 8) << 8) | ((item_.z & 255) * tmul), 0);
  const int V = S::GROUPED ? (SPIN ? 4 : 2) * a.nj : S::V;  // the plan's partial sums per degree; the CTA's jobs from j0 on
  // the warp's number from a shuffle: the compiler sees it uniform, and so the MMAs'
  // descriptors, which then live in uniform registers
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int mi = item.x, ng = item.z & 255;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax, nl = lmax - l0 + 1;
  const float4 *__restrict__ cf = a.coef32 + (a.coef_off[mi] - l0);
  double *const outp = a.part + a.part_off[mi] + (int64_t)(item.z >> 8) * nl * V;
  const double sg0 = ((l0 + m) & 1) ? -1.0 : 1.0;
  unsigned char *const Abuf = tca_smem;
  unsigned char *const Bbuf = tca_smem + S::A_BYTES;
  // this warp's staged D rows (kN columns each)
  float *const Ebuf = reinterpret_cast<float *>(tca_smem + S::A_BYTES + S::B_BYTES) + warp * S::E_FLOATS;

  if (warp == 0) tc::tmem_alloc(&tslot, S::TCOLS);
  if (tid == 0) {
#pragma unroll
    for (int x = 0; x < NACC; ++x) {
      tc::bar_init(&full[x], S::WARPS);
      tc::bar_init(&freeb[x], 4);  // the warps of one group read and release it
    }
#pragma unroll
    for (int w = 0; w < S::WARPS; ++w) tc::bar_init(&mine[w], 1);
    stop = 0;
  }
  // A starts at zero: rows 6 and 7 of each column (below its six digits) stay so
  // (QUAD stores no such rows, and every entry of the others is written in each tile)
  if (!S::QUAD) for (int i = tid; i < S::A_BYTES / 16; i += TH) reinterpret_cast<uint4 *>(Abuf)[i] = make_uint4(0, 0, 0, 0);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = tslot;
  const uint32_t tlane = tbase + ((uint32_t)((warp & 3) * 32) << 16);
  // the accumulators start at zero (ordered before any MMA by the tile's barriers)
  if (warp < 4) {
#pragma unroll
    for (int x = 0; x < NACC; ++x)
#pragma unroll
      for (int q = 0; q < tca::kN / 16; ++q) tc::tmem_zero16(tlane + x * tca::kDCols + q * 16);
    tc::tmem_wait_st();
  }
  tc::fence_before();

  const uint64_t adesc0 = tc::mat_desc(tc::smem_u32(Abuf), S::A_LBO, S::A_SBO);
  const uint64_t bdesc0 = tc::mat_desc(tc::smem_u32(Bbuf), S::KSTRIDE, S::B_SBO);
  constexpr uint32_t idesc = tc::instr_desc(S::M, tca::kN, true);

  // the K entries of pair p (spin: both of its lanes; spin 0: lane t) for every column
  auto load_pair = [&](int p, int t, double (&gv)[NSET][NC]) __attribute__((always_inline)) {
    const bool south = a.pairs[p].south;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      if (!SPIN) {
        const double2 *gp = a.phase + (((size_t)(j0 + j) * a.nm + mi) * a.npairs + p) * 2;
        const double2 gn = gp[0], gs = south ? gp[1] : make_double2(0.0, 0.0);
        gv[t][4 * j + 0] = gn.x + gs.x;
        gv[t][4 * j + 1] = gn.y + gs.y;
        gv[t][4 * j + 2] = gn.x - gs.x;
        gv[t][4 * j + 3] = gn.y - gs.y;
      } else {
        const double2 *gq = a.phase + (((size_t)(2 * (j0 + j)) * a.nm + mi) * a.npairs + p) * 2;
        const double2 *gu = a.phase + (((size_t)(2 * (j0 + j) + 1) * a.nm + mi) * a.npairs + p) * 2;
        const double2 qn = gq[0], un = gu[0];
        const double2 qs = south ? gq[1] : make_double2(0.0, 0.0), us = south ? gu[1] : make_double2(0.0, 0.0);
        // W+_N, W-_N, W+_S', W-_S' (re, im)
        const double wpn_r = qn.x - un.y, wpn_i = qn.y + un.x;
        const double wmn_r = qn.x + un.y, wmn_i = qn.y - un.x;
        const double wps_r = sg0 * (qs.x - us.y), wps_i = sg0 * (qs.y + us.x);
        const double wms_r = sg0 * (qs.x + us.y), wms_i = sg0 * (qs.y - us.x);
        gv[0][4 * j + 0] = wpn_r;  // T1: l+ W+_N
        gv[0][4 * j + 1] = wpn_i;
        gv[0][4 * j + 2] = wms_r;  // s T2: l+ W-_S'
        gv[0][4 * j + 3] = wms_i;
        gv[1][4 * j + 0] = wps_r;  // T1: s l- W+_S'
        gv[1][4 * j + 1] = wps_i;
        gv[1][4 * j + 2] = wmn_r;  // s T2: s l- W-_N
        gv[1][4 * j + 3] = wmn_i;
      }
    }
  };
  // Plans that always run this kernel (more than two jobs): whether the item's values range too far for
  // the digits, which lose 2^-50 of a column's largest |G'| where the double-float sums lose
  // 2^-46 of each term; the item is then left to those (false).  At degree l the sum comes
  // from the pairs between some latitude and the equator (l0: next to it), the others' Lambda
  // falls away exponentially, so no |G'| may exceed 2^kWideRange times the largest of the 32
  // pairs next to the equator, and the last of them has to start near its bound at l0.
  // (White maps without ring weights range over u_p, 2^5 at lmax 2047, and their extremes.)
  constexpr int kWideRange = 8;
  bool wide = false;
  const bool guard = S::QUAD || (S::GROUPED && a.nj > NJ);
  if (guard && warp == 0) {
    const int p = a.npairs - 1 - lane;
    unsigned mx[NC];
    {
      double gv[NSET][NC];
#pragma unroll
      for (int t = 0; t < NSET; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) gv[t][c] = 0.0;
      JoinRec r = {};
      if (p >= 0) {
        r = ld_join(a.join + ((size_t)mi * a.npairs + p) * 3);
        load_pair(p, 0, gv);
      }
      if (lane == 0) {
        const float low = SPIN ? fminf(fabsf(r.lpc.h), fabsf(r.lmc.h)) : fabsf(r.lpc.h);
        eqok = !ta.force && r.lj == l0 && r.scp == 0 && (!SPIN || r.scm == 0) && low >= ldexpf(1.f, r.lexp - 6);
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        mx[c] = 0u;
#pragma unroll
        for (int t = 0; t < (SPIN ? 2 : 1); ++t) {
          const unsigned hi = (unsigned)__double2hiint(gv[t][c]) & 0x7fffffffu;
          if (p >= 0 && r.lj <= lmax && hi > 0u) mx[c] = max(mx[c], tca::not_finite(hi) ? 0x7ff00000u : tca::add_exp(hi, r.lexp));
        }
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const unsigned e = __reduce_max_sync(0xffffffffu, mx[c]);
      if (lane == 0) eqmax[c] = e;
    }
  }

  int ib = 0;                    // blocks walked by the CTA over all its tiles: accumulator ib % NACC
  int nmine = 0, nmine_done = 0;  // this warp's commits to mine[warp], and those waited for
  bool ok = true;
  // a bounded wait of the whole warp (false for every lane if any lane gave up)
  auto wait_warp = [&](uint64_t *bar, uint32_t parity) -> bool {
    if (__all_sync(0xffffffffu, tc::bar_try(bar, parity))) return true;  // mostly: no clock read
    const bool r = tc::bar_wait_or(bar, parity, &stop);
    return __all_sync(0xffffffffu, r);
  };
  auto give_up = [&]() {
    if (lane == 0) stop = 1;
    ok = false;
  };

  // a thread's ring pairs: one (spin), or two neighbours (spin 0: they join at about
  // the same degree; pairs TH apart took 28.6 ms at lmax 4095, neighbours 27.2)
#pragma unroll 1
  for (int gi = 0; gi < ng; gi += S::TILES) {
    int pr[NP], lj[NP], lexp[NP];
    bool valid[NP];
    const float4 *jrec[NP];
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      pr[t] = (item.y + gi) * S::TILE + NP * tid + t;
      valid[t] = pr[t] < min(a.npairs, (item.y + ng) * S::TILE);
      jrec[t] = a.join + ((size_t)mi * a.npairs + (valid[t] ? pr[t] : 0)) * 3;
      lj[t] = lmax + 1;
      lexp[t] = 0;
      if (valid[t]) {
        const float4 c = __ldg(jrec[t] + 2);
        lj[t] = __float_as_int(c.z);
        lexp[t] = __float_as_int(c.w);
      }
    }
    const int jmin = min(lj[0], lj[NP - 1]);
    // the K entries of every column; their factors u_p = 2^lexp, the pairs' Lambda bounds
    // (zero for a pair that never joins), enter with the column's scale
    double gv[NSET][NC];
#pragma unroll
    for (int t = 0; t < NSET; ++t)
#pragma unroll
      for (int c = 0; c < NC; ++c) gv[t][c] = 0.0;
#pragma unroll
    for (int t = 0; t < NP; ++t)
      if (valid[t]) load_pair(pr[t], t, gv);
    __syncthreads();  // the previous tile's products are complete (its last accumulator was read)
    if (stop) {       // read after a barrier: the same for every warp
      ok = false;
      break;
    }
    if (tid < NC) vmax[tid] = 0u;
    {
      const int wmin = __reduce_min_sync(0xffffffffu, jmin);
      if (lane == 0) tstart[warp] = wmin;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {  // column bounds over the tile (upper words of |G'|)
      unsigned mx = 0u;
#pragma unroll
      for (int t = 0; t < NSET; ++t) {
        const unsigned hi = (unsigned)__double2hiint(gv[t][c]) & 0x7fffffffu;
        const int q = t < NP ? t : 0;  // an infinity or NaN counts whether or not its pair joins
        mx = max(mx, tca::not_finite(hi) ? 0x7ff00000u : lj[q] <= lmax ? tca::add_exp(hi, lexp[q]) : 0u);
      }
      const unsigned w = __reduce_max_sync(0xffffffffu, mx);
      if (lane == 0) atomicMax(&vmax[c], w);
    }
    __syncthreads();
    if (guard) {
      wide = !eqok;
#pragma unroll
      for (int c = 0; c < NC; ++c)  // (a column that is not finite: below)
        wide = wide || (vmax[c] > 0u && !tca::not_finite(vmax[c]) && !tca::not_finite(eqmax[c]) &&
                        (vmax[c] >> 20) > (eqmax[c] >> 20) + kWideRange);
      if (wide) break;  // the same for every thread; no product is in flight here
    }
    int lstart = tstart[0];
#pragma unroll
    for (int w = 1; w < S::WARPS; ++w) lstart = min(lstart, tstart[w]);
    // the G' digits of this pair into A: column c's digit j at its row j of the
    // pair's K-group, entry tid % 8 (rows 6 and 7 stay zero)
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int e = tca::exp_above(vmax[c]);
#pragma unroll
      for (int t = 0; t < NSET; ++t) {
        float d[kDig];
        tca::digits6(gv[t][c], lj[t < NP ? t : 0] <= lmax, lexp[t < NP ? t : 0] - e, d);
        unsigned char *dst = Abuf + S::a_at(c, 0, t * (TH / 8) + tid / 8) + (tid % 8) * 2;
#pragma unroll
        for (int j = 0; j < kDig; ++j) *reinterpret_cast<uint16_t *>(dst + j * 16) = tc::bf16_of(d[j]);
      }
    }
    // the slot's degrees before the tile's first block are zero (later tiles add to them);
    // a column that holds an infinity or a NaN makes all its degrees NaN
    bool bad = false;
#pragma unroll
    for (int c = 0; c < NC; ++c) bad = bad || tca::not_finite(vmax[c]);
    if (gi == 0 || bad)
      for (int i = tid; i < (min(lstart, lmax + 1) - l0) * S::V; i += TH) {
        const int v = i % S::V;
        const bool nan = bad && tca::not_finite(vmax[SPIN ? v : 4 * (v >> 1) + (v & 1)]);
        if (gi == 0 || nan) outp[(int64_t)(i / S::V) * V + (SPIN ? 4 : 2) * j0 + v] = nan ? CUDART_NAN : 0.0;
      }
    // v_c of the column that this lane sums (epi_sum, epi_quad)
    const int vcol = S::QUAD ? 4 * (warp & 3) + ((lane >> 2) & 3) : (S::CPW == 1 ? (warp & 3) : 2 * (warp & 3) + ((lane >> 3) & 1));
    const double vscale =
        tca::not_finite(vmax[vcol]) ? CUDART_NAN : __hiloint2double((1023 + tca::exp_above(vmax[vcol])) << 20, 0);
    tc::fence_async_smem();
    __syncthreads();
    if (lstart > lmax) continue;

    // the walk over the tile's blocks of 8 degrees (from its pairs' earliest join):
    // the recursions run on Lambda / u_p
    Dual<SPIN, kPacked> rec;
    rec.p = rec.q = d2{both(0.f), both(0.f)};
    int sc0 = 0, sc1 = 0;
    double xd[NP];
    bool near = false;
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      xd[t] = valid[t] ? a.pairs[pr[t]].x : 0.0;
      near = near || near_pole(xd[t], valid[t]);
    }
    const bool polar = __any_sync(0xffffffffu, near);
#pragma unroll
    for (int t = 0; t < NP; ++t) rec.x[t] = node_of(xd[t], polar);
    const int lfast = SPIN ? fast_from(as, rec.x[0].h, valid[0], lmax) : 0;
    float2 wf = both(0.f);  // weights of the two lanes' values (zero until they join)
    bool settled = false;   // every lane of the warp at scale 0 (warp-uniform)

    // 4 degrees from lb4 (lb4 - l0 even): the digits packed per pair of degrees into
    // pk[set][digit][q / 2]; recursion advanced.  (Values of a joined pair are not
    // tested for negligibility: the join record already skips the stretch before its
    // first non-negligible degree pair, and later values below the digits' grid give
    // zero digits.)  kFast: settled, weights 1.
    auto part = [&](const StepMode mode, int lb4, uint32_t (&pk)[NSET][kDig][2]) __attribute__((always_inline)) {
      float2 hold[kDig];
      float4 cv[4];
      // past lmax the entries of the next m (or the table's zero tail) give finite
      // values no output reads
#pragma unroll
      for (int q = 0; q < 4; ++q) cv[q] = __ldg(cf + lb4 + q);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool odd = q & 1;
        float2 d[kDig];
        if (mode == kFast) {
          tca::split6(rec.p.h, rec.p.l, d);
        } else {
          const float2 f = make_float2(wf.x, (SPIN && mode == kPolar && odd) ? -wf.y : wf.y);
          tca::split6(mul2(rec.p.h, f), mul2(rec.p.l, f), d);
        }
#pragma unroll
        for (int i = 0; i < kDig; ++i) {
          if (!odd) {
            hold[i] = d[i];
          } else {
            pk[0][i][q >> 1] = tc::pack_bf16(hold[i].x, d[i].x);
            pk[1][i][q >> 1] = tc::pack_bf16(hold[i].y, d[i].y);
          }
        }
        rec.step(mode, cv[q]);
      }
    };
    // the enhanced exponent's check after every block of 8 degrees (see mixed_common.cuh)
    auto rescale = [&]() {
      if (settled) return;
      rec.rescale(sc0, sc1);
      if (lj[0] <= lmax) wf.x = scale_weight(sc0);
      if (lj[NP - 1] <= lmax) wf.y = scale_weight(sc1);
      settled = __all_sync(0xffffffffu, sc0 == 0 && sc1 == 0);
    };
    // this warp's digits of degrees 4h .. 4h + 3 of the block: entry tid % 8 of K-group
    // (set, tid / 8), N-group = digit, bytes 8h .. 8h + 7 of the 16-byte row
    auto store_b = [&](int h, const uint32_t (&pk)[NSET][kDig][2]) {
#pragma unroll
      for (int t = 0; t < NSET; ++t)
#pragma unroll
        for (int i = 0; i < kDig; ++i) {
          unsigned char *dst = Bbuf + i * S::B_SBO + (t * (TH / 8) + tid / 8) * S::KSTRIDE + (tid % 8) * 16 + h * 8;
          *reinterpret_cast<uint2 *>(dst) = make_uint2(pk[t][i][0], pk[t][i][1]);
        }
    };
    // this warp's MMAs of a block into accumulator xb: one per K-step (16 entries:
    // two K-groups) of each set
    auto issue = [&](int xb) {
      tc::fence_after();
#pragma unroll
      for (int t = 0; t < NSET; ++t)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int kk = t * (TH / 16) + 2 * warp + hh;
          const uint64_t ad = adesc0 + (uint64_t)((2 * kk * S::A_LBO) >> 4);
          const uint64_t bd = bdesc0 + (uint64_t)((2 * kk * S::KSTRIDE) >> 4);
          tc::mma_bf16(tbase + xb * tca::kDCols, ad, bd, idesc, 1u);
        }
      tc::mma_commit(&mine[warp]);
      tc::mma_commit(&full[xb]);
    };
    // block ibp's D rows of this warp's quarter into shared memory; the accumulator
    // zeroed and released
    auto epi_read = [&](int ibp) {
      const int xb = ibp % NACC;
      if (!wait_warp(&full[xb], (uint32_t)(ibp / NACC) & 1u)) {
        give_up();
        return;
      }
      tc::fence_after();
      const uint32_t ta = tlane + xb * tca::kDCols;
      uint32_t v[tca::kN / 16][16];
#pragma unroll
      for (int q = 0; q < tca::kN / 16; ++q) tc::tmem_ld16(ta + q * 16, v[q]);
      tc::tmem_wait_ld();
#pragma unroll
      for (int q = 0; q < tca::kN / 16; ++q) tc::tmem_zero16(ta + q * 16);
      if (lane < S::EROWS) {
        float4 *er = reinterpret_cast<float4 *>(Ebuf + lane * tca::kEStride);
#pragma unroll
        for (int q = 0; q < tca::kN / 16; ++q)
#pragma unroll
          for (int r = 0; r < 4; ++r)
            er[4 * q + r] = make_float4(__uint_as_float(v[q][4 * r]), __uint_as_float(v[q][4 * r + 1]),
                                        __uint_as_float(v[q][4 * r + 2]), __uint_as_float(v[q][4 * r + 3]));
      }
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::bar_arrive(&freeb[xb]);
    };
    // the column and degree a lane sums (one column a quarter: four lanes share a
    // degree, epart 0 .. 3, and lane epart 0 writes it); the slot entry written for
    // block lbp (nullptr: none; neg: add the negation)
    const int odeg = lane & 7, epart = lane >> 3;
    const int ocol = S::CPW == 1 ? (warp & 3) : 2 * (warp & 3) + (epart & 1);
    const bool oact = S::CPW == 1 ? epart == 0 : lane < S::EROWS;
    auto out_at = [&](int lbp, bool &neg) -> double * {
      if (S::QUAD) {  // job = quarter, column = lane / 4, every second degree; the upper lanes sum odd digit rows
        const int c = (lane >> 2) & 3, lq = lbp + 2 * (lane & 3) + (c >> 1);
        neg = false;
        return lane < 16 && lq <= lmax ? outp + (int64_t)(lq - l0) * V + 2 * (j0 + (warp & 3)) + (c & 1) : nullptr;
      }
      const int l = lbp + odeg, j = ocol >> 2, cc = ocol & 3;
      neg = false;
      if (!oact || l > lmax) return nullptr;
      if (SPIN) {
        neg = cc >= 2 && (odeg & 1);  // T2 = s (s T2)
        return outp + (int64_t)(l - l0) * V + 4 * (j0 + j) + cc;
      }
      // spin 0: the even-l columns at even l - l0, the odd ones at odd
      return (cc >> 1) == (odeg & 1) ? outp + (int64_t)(l - l0) * V + 2 * j + (cc & 1) : nullptr;
    };
    // the staged digit products by level: levels 0 to 2 exact in FP32 (at most three
    // sums of 2^22 quanta), added in double-float; levels 3 to 6 in FP32; the slot
    // entry written (prev: its value from the group's earlier tiles).  D(i, j) = sum of
    // G_j L_i.
    auto epi_sum = [&](double *o, bool neg, double prev) {
      float L0, L1, L2, lo = 0.f;
      if (S::CPW == 1) {
        // lane epart q takes row j = q, and of rows 4 and 5 lane 2 + (j - 4) takes one
        const float *e = Ebuf + epart * tca::kEStride + odeg;
        float v[kDig];
#pragma unroll
        for (int i = 0; i < kDig; ++i) v[i] = e[i * 8];
        const float *e2 = e + 2 * tca::kEStride;  // parts 2, 3: rows 4, 5 (others': not used)
        const float w0 = e2[0], w1 = e2[8], w2 = e2[16];
        lo = __fadd_rn(epart < 2 ? v[5] : w1, epart < 3 ? v[4] : 0.f);
        lo = __fadd_rn(lo, epart == 2 ? w2 : 0.f);
        lo = __fadd_rn(lo, v[3]);
        lo = __fadd_rn(lo, epart < 2 ? 0.f : w0);
        lo = __fadd_rn(lo, epart < 1 ? 0.f : v[2]);
        lo = __fadd_rn(lo, epart < 2 ? 0.f : v[1]);
        lo = __fadd_rn(lo, epart < 3 ? 0.f : v[0]);
        lo = __fadd_rn(lo, __shfl_xor_sync(0xffffffffu, lo, 16));
        lo = __fadd_rn(lo, __shfl_xor_sync(0xffffffffu, lo, 8));
        L0 = v[0];
        L1 = __fadd_rn(v[1], __shfl_down_sync(0xffffffffu, v[0], 8));
        L2 = __fadd_rn(__fadd_rn(v[2], __shfl_down_sync(0xffffffffu, v[1], 8)), __shfl_down_sync(0xffffffffu, v[0], 16));
      } else {
        const float *e = Ebuf + (epart & 1) * tca::kColRows * tca::kEStride + odeg;
        auto D = [&](int i, int j) { return e[j * tca::kEStride + i * 8]; };
        L0 = D(0, 0);
        L1 = __fadd_rn(D(1, 0), D(0, 1));
        L2 = __fadd_rn(__fadd_rn(D(2, 0), D(1, 1)), D(0, 2));
#pragma unroll
        for (int k = 6; k >= 3; --k)
#pragma unroll
          for (int i = 0; i < kDig; ++i)
            if (k - i >= 0 && k - i < kDig) lo = __fadd_rn(lo, D(i, k - i));
      }
      if (o) {
        f2 t = two_sum(L0, L1);
        t = f2_add_lazy(t, f2{L2, 0.f});
        t = fast_two_sum(t.h, __fadd_rn(t.l, lo));
        *o = fma(f2_val(t), neg ? -vscale : vscale, prev);
      }
      __syncwarp();
    };

    // four jobs: block ibp's rows of this warp's quarter read, zeroed and released; then,
    // one Lambda digit at a time, the four degrees of each row's parity go through shared
    // memory to lanes of (column, degree), the lower 16 taking the even digit rows j and
    // the upper the odd ones.  S[k] of a lower lane: level k, of an upper one level k + 1.
    auto epi_quad = [&](int ibp, double *o, double prev) {
      const int xb = ibp % NACC;
      if (!wait_warp(&full[xb], (uint32_t)(ibp / NACC) & 1u)) {
        give_up();
        return;
      }
      tc::fence_after();
      const uint32_t ta = tlane + xb * tca::kDCols;
      uint32_t v[tca::kN / 16][16];
#pragma unroll
      for (int q = 0; q < tca::kN / 16; ++q) tc::tmem_ld16(ta + q * 16, v[q]);
      tc::tmem_wait_ld();
#pragma unroll
      for (int q = 0; q < tca::kN / 16; ++q) tc::tmem_zero16(ta + q * 16);
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::bar_arrive(&freeb[xb]);
      float4 *const put = reinterpret_cast<float4 *>(Ebuf) + 10 * (lane >> 3) + (lane & 7);
      const float *const get = Ebuf + (10 * ((lane >> 2) & 3) + (lane >> 4)) * 4 + (lane & 3);
      const bool par = lane >= 16;
      float S5[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < kDig; ++i) {
        auto w = [&](int d) { return __uint_as_float(par ? v[i / 2][8 * (i & 1) + 2 * d + 1] : v[i / 2][8 * (i & 1) + 2 * d]); };
        *put = make_float4(w(0), w(1), w(2), w(3));
        __syncwarp();
#pragma unroll
        for (int jj = 0; jj < 3; ++jj) {
          const int k = i + 2 * jj;
          if (k <= 6) S5[k < 4 ? k : 4] = __fadd_rn(S5[k < 4 ? k : 4], get[8 * jj]);
        }
        __syncwarp();
      }
      const float q0 = __shfl_xor_sync(0xffffffffu, S5[0], 16), q1 = __shfl_xor_sync(0xffffffffu, S5[1], 16);
      const float q2 = __shfl_xor_sync(0xffffffffu, __fadd_rn(__fadd_rn(S5[4], S5[3]), S5[2]), 16);
      if (o) {
        f2 t = two_sum(S5[0], __fadd_rn(S5[1], q0));
        t = f2_add_lazy(t, f2{__fadd_rn(S5[2], q1), 0.f});
        t = fast_two_sum(t.h, __fadd_rn(t.l, __fadd_rn(__fadd_rn(S5[4], q2), S5[3])));
        *o = fma(f2_val(t), vscale, prev);
      }
    };

    int lb = lstart;
    const int ib0 = ib;
#pragma unroll 1
    for (; lb <= lmax; lb += tca::kBlk, ++ib) {
      const int xb = ib % NACC;
      // this warp's turn to read: block ib - LAG.  The slot entry its lanes add that
      // block to is read now, its latency hidden behind this block's recursion.
      const bool turn = ib - LAG >= ib0 && (GROUPS == 1 || (ib & 1) == (warp >> 2));
      bool neg_prev = false;
      double *const o_prev = turn ? out_at(lb - LAG * tca::kBlk, neg_prev) : nullptr;
      double prev = 0.0;
      if (o_prev && gi > 0) asm volatile("ld.global.f64 %0, [%1];" : "=d"(prev) : "l"(o_prev));
      // pairs joining here take the recursion state where their terms start, over u_p
      bool joins = false;
#pragma unroll
      for (int t = 0; t < NP; ++t)
        if (lj[t] == lb) {
          const JoinRec r = ld_join(jrec[t], polar);
          const float ulx = __int_as_float((127 - lexp[t]) << 23);
          if (t == 0) {
            rec.start(0, r.lpc, r.lpp, ulx);
            sc0 = r.scp;
            wf.x = scale_weight(sc0);
          } else {
            rec.start(1, r.lpc, r.lpp, ulx);
            sc1 = r.scp;
            wf.y = scale_weight(sc1);
          }
          if (SPIN) {  // lane 1 holds s l- (l- itself in a polar warp): the previous degree's sign is -1
            rec.start(1, r.lmc, polar ? r.lmp : neg(r.lmp), ulx);
            sc1 = r.scm;
            wf.y = scale_weight(sc1);
          }
          joins = true;
        }
      if (__any_sync(0xffffffffu, joins)) settled = __all_sync(0xffffffffu, sc0 == 0 && sc1 == 0);
      // a warp none of whose pairs has joined adds nothing: no digits, no products,
      // a plain arrival.  Every warp first waits until the reading warps have released
      // the accumulator's previous block, so that no arrival (or commit) of this block
      // can fall into the phase of the block NACC before.
      const bool live = __any_sync(0xffffffffu, jmin <= lb);
      if (live) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t pk[NSET][kDig][2];
          if (polar) part(kPolar, lb + 4 * h, pk);
          else if (settled && lb >= lfast) part(kFast, lb + 4 * h, pk);
          else part(kCareful, lb + 4 * h, pk);
          // this warp's products of its previous block read the tiles: wait for them
          // before the first write (they have long finished by now)
          if (h == 0 && nmine > nmine_done) {
            if (!wait_warp(&mine[warp], (uint32_t)(nmine - 1) & 1u)) break;
            nmine_done = nmine;
          }
          store_b(h, pk);
        }
        if (nmine > nmine_done) {  // the wait above gave up
          give_up();
          break;
        }
        rescale();
        tc::fence_async_smem();
        __syncwarp();
      }
      if (ib >= NACC && !wait_warp(&freeb[xb], (uint32_t)(ib / NACC - 1) & 1u)) {
        give_up();
        break;
      }
      if (live) {
        if (tc::elect_one()) issue(xb);
        __syncwarp();
        ++nmine;
      } else if (lane == 0) {
        tc::bar_arrive(&full[xb]);
      }
      if (turn) {
        if (S::QUAD) {
          epi_quad(ib - LAG, o_prev, prev);
          if (!ok) break;
        } else {
          epi_read(ib - LAG);
          if (!ok) break;
          epi_sum(o_prev, neg_prev, prev);
        }
      }
    }
    if (!ok) continue;  // to the next tile's barrier, where the CTA stops
    // the tile's last blocks
#pragma unroll 1
    for (int k = ib - LAG > ib0 ? ib - LAG : ib0; k < ib; ++k) {
      if (GROUPS > 1 && (k & 1) != (warp >> 2)) continue;
      bool neg;
      double *o = out_at(lb - (ib - k) * tca::kBlk, neg);
      const double prev = (o && gi > 0) ? *o : 0.0;
      if (S::QUAD) {
        epi_quad(k, o, prev);
        if (!ok) break;
        continue;
      }
      epi_read(k);
      if (!ok) break;
      epi_sum(o, neg, prev);
    }
  }

  // leave: flag a wait that gave up (each warp its own: the two groups wait for different
  // accumulators, and after the last tile no barrier tells the others), let this warp's
  // products in flight finish (bounded), release TMEM
  if (!ok && lane == 0) atomicOr(ta.err, 1);
  if (nmine > nmine_done) tc::bar_wait(&mine[warp], (uint32_t)(nmine - 1) & 1u);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, S::TCOLS);
  return !wide;
}

template <int NJ, bool SPIN>
__device__ __forceinline__ void tc_ana_item(const TcArgs &ta, const int4 item, const int j0, unsigned char *smem) {
  using S = tca::AnaShape<NJ, SPIN>;
  if (tc_ana_body<NJ, SPIN>(ta, item, j0, smem)) return;
  if constexpr (S::GROUPED) {  // the item's tiles of 256 pairs in double-float
    static_assert(sizeof(MixAnaShared) <= S::SMEM, "its table in the digits' shared memory");
    __syncthreads();
    mix_ana_body<NJ, 2, SPIN>(ta.m, item, *reinterpret_cast<MixAnaShared *>(smem), j0, (SPIN ? 4 : 2) * ta.m.nj, true);
  }
}

// a plan of more than four jobs: consecutive CTAs take its groups of four
template <int NJ, bool SPIN>
__global__ void __launch_bounds__((tca::AnaShape<NJ, SPIN>::TH), (tca::AnaShape<NJ, SPIN>::MINB))
    tc_ana(TcArgs ta, int groups) {
  extern __shared__ __align__(128) unsigned char tca_smem[];
  constexpr bool G = tca::AnaShape<NJ, SPIN>::GROUPED;
  const int g = G ? blockIdx.x % groups : 0, i = G ? blockIdx.x / groups : blockIdx.x;
  tc_ana_item<NJ, SPIN>(ta, ta.m.ana_items[i], NJ * g, tca_smem);
}

// batches: item (mi, first tile, slot << 8 | tiles, record); the record holds the plan's arguments
template <int NJ, bool SPIN>
__global__ void __launch_bounds__((tca::AnaShape<NJ, SPIN>::TH), (tca::AnaShape<NJ, SPIN>::MINB))
    tc_ana_batch(const TcArgs *__restrict__ args, const int4 *__restrict__ items, int groups) {
  extern __shared__ __align__(128) unsigned char tca_smem[];
  constexpr bool G = tca::AnaShape<NJ, SPIN>::GROUPED;
  const int g = G ? blockIdx.x % groups : 0;
  const int4 it = items[G ? blockIdx.x / groups : blockIdx.x];
  tc_ana_item<NJ, SPIN>(args[it.w], make_int4(it.x, it.y, it.z, 0), NJ * g, tca_smem);
}

template <int NJ, bool SPIN>
static cudaError_t tca_set_smem() {
  cudaError_t e = cudaSuccess;
  for (const void *k : {(const void *)tc_ana<NJ, SPIN>, (const void *)tc_ana_batch<NJ, SPIN>}) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, tca::AnaShape<NJ, SPIN>::SMEM_LAUNCH);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  }
  return e;
}

cudaError_t tc_ana_prepare_device() {
  cudaError_t e = tca_set_smem<1, false>();
  if (e == cudaSuccess) e = tca_set_smem<2, false>();
  if (e == cudaSuccess) e = tca_set_smem<4, false>();
  if (e == cudaSuccess) e = tca_set_smem<1, true>();
  if (e == cudaSuccess) e = tca_set_smem<2, true>();
  return e;
}

bool tc_ana_supported(int spin, int njobs_pad) {
  (void)spin;
  return njobs_pad <= 2;
}

// Spin s, more than two E/B pairs, two at a time: four pairs, lmax 31 20 us against 54 for
// the double-float contraction, 511 0.41 ms against 1.11, 2047 18.6 against 41.6; eight, lmax
// 1023 5.1 against 15.1.
// Spin 0, more than two maps: faster than the double-float contraction at every size
// (four maps, lmax 31: 22.5 us against 24.4; 255: 74 / 112; 2047: 4.99 / 10.35 ms; sixteen
// maps, lmax 31: 22 / 107 us, 2047: 20.2 / 65.7 ms), which has no instance for them.  Error
// against the FP64 form: lmax 31 2.3e-14 to 2.4e-14 (that contraction 2.1e-14 to 2.4e-14),
// 255 8.4e-14 (8.4e-14), 511 1.0e-13 (1.2e-13), 2047 3.7e-13 (3.7e-13).
bool tc_ana_quad(const sht_plan_s *P) { return P->precision == SHT_MIXED && P->njobs_pad >= 4; }

int tc_ana_tiles(int spin, int njobs_pad) {
  if (spin == 0) return njobs_pad == 1 ? tca::AnaShape<1, false>::TILES : tca::AnaShape<2, false>::TILES;
  return njobs_pad == 1 ? tca::AnaShape<1, true>::TILES : tca::AnaShape<2, true>::TILES;
}

namespace {
// calls f with the shape of a spin class and padded job count; false: none
template <int NJ, bool SPIN>
struct AnaLaunch {
  static constexpr int nj = NJ, th = tca::AnaShape<NJ, SPIN>::TH, smem = tca::AnaShape<NJ, SPIN>::SMEM_LAUNCH;
  static constexpr bool spin = SPIN;
};
template <class F>
bool tca_shape(int spin, int nj, F &&f) {
  if (spin == 0) {
    if (nj == 1) f(AnaLaunch<1, false>());
    else if (nj == 2) f(AnaLaunch<2, false>());
    else f(AnaLaunch<4, false>());
    return true;
  }
  if (nj == 1) f(AnaLaunch<1, true>());
  else f(AnaLaunch<2, true>());
  return true;
}
}  // namespace

cudaError_t launch_leg_tc_ana_batch(int spin, int nj, const void *targs, const int4 *items, int n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const TcArgs *a = static_cast<const TcArgs *>(targs);
  const bool ok = tca_shape(spin, nj, [&](auto sh) {
    using H = decltype(sh);
    const int groups = nj / H::nj;
    tc_ana_batch<H::nj, H::spin><<<n * groups, H::th, H::smem, st>>>(a, items, groups);
  });
  return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

cudaError_t launch_leg_tc_ana(const sht_plan_s *P, const void *mixargs, int n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  TcArgs ta;
  memcpy(&ta.m, mixargs, sizeof(MixArgs));
  ta.err = P->d_err;
  ta.force = P->quad_off;
  const bool ok = tca_shape(P->spin, P->njobs_pad, [&](auto sh) {
    using H = decltype(sh);
    const int groups = P->njobs_pad / H::nj;
    tc_ana<H::nj, H::spin><<<n * groups, H::th, H::smem, st>>>(ta, groups);
  });
  return ok ? cudaGetLastError() : cudaErrorInvalidValue;
}

}  // namespace sht
