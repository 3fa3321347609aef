// Fused sweep: enumerate -> evaluate -> filter -> reduce -> emit, nothing materialised,
// one launch and one block per model (top-k: per model and capacity).  A block walks the
// model's factorisations ("units") in segments, and everywhere a lane owns a unit: it
// forms the unit's shard quantities, and what a (Theta, Omega, G) triple's own bytes are held
// against, in registers (the screening: bounds in rounded figures, without a division; top-k's first
// pass, which counts points: a bound per activation variant and digit, LaneUnit; the other passes: the
// least activation bytes, LeastUnit); then the lanes of a warp walk the triples together.  A
// triple's bytes are a sum of three terms, one per state, and what is uniform (modes, allowed
// digits, coefficients) comes from small tables of the block.
//
// Screening.  Every unit: its points are compared with their bounds in rounded figures, two
// to an instruction (the four variants of the offloaded digit have the same bytes: 17
// compares for 20 points), masked by the flags that the placement code and the composition
// allow.  It leaves the list of the units that may have survivors (an eighth of them on the
// stress configuration), which the next two passes walk densely and in whole bytes.  (With
// ps_filter.skip_rejected the list is made from the composition tests alone; top-k without
// required flags lists all units.)
//
// First pass, over the cells of a histogram (an eighth of an octave each).
//   Pareto: the least communication of the candidates whose bytes fall into a cell
//   (atomicMin).  The prefix minimum is a staircase of strictly dominating points.
//   Top-k: the number of survivors whose communication falls into a cell.  The first cell
//   up to which there are k bounds the k-th smallest.
// Second pass: appends to the block's buffer only what the staircase does not beat, or
// what lies within the bounding cell.  A full buffer is cut back (Pareto: to its frontier;
// top-k: to its k smallest, the last of which is then a threshold) and the warps resume
// where they stopped.  Nothing is inserted into a sorted list one by one.  The few that are
// left at the end are resolved to points and indices by a thread each, in code of its own:
// the passes stay small enough for the instruction cache.
// The block then emits the entries, evaluating each again from its index as a self-check.
// A frontier that outgrows the buffer takes a slow exact path.
//
// What bounds it: the issue slots of the screening, and the latency of a block's phases (five
// blocks of four warps share an SM).  4096 models of the stress configuration, 6.96e9 points:
// top-k 1.94 -> 0.57 ms, Pareto 2.37 -> 0.54 ms against a sweep whose warps took a unit each (the
// set-up of a unit paid by a whole warp, candidates inserted one by one into a sorted list per
// warp, the lists merged by a second kernel); 1024 models skipping rejected factorisations 0.41
// -> 0.072 ms.  The screening takes 0.23 and 0.27 ms of the former two.
#include <type_traits>
#include "ps_device.cuh"
#include "ps_internal.h"
#include "ps_lane.cuh"

namespace {

typedef uint16_t u16;

constexpr u64 U64MAX = ~0ull;
constexpr int SEG = 1024;                  // units of a segment
constexpr int CELLS = 512;                 // cells of the histogram
constexpr int CAND_CAP = 512;              // candidates the block's buffer holds
constexpr int KEEP_CAP = PS_FRONTIER_FAST; // Pareto: frontier entries that can be emitted from the buffer
constexpr int MAX_TRIPLES = 125;
constexpr u32 NO_CODE = 0xffffffffu;       // an empty entry
constexpr u32 ALL_STEPS = 0xffffffffu;
constexpr int STEP_CAP = 128;              // entries that a step of the second pass appends at most: four a lane
// (top-k: a cut leaves k candidates and what ties with the last of them in its unit, see cut_candidates;
// a candidate becomes at most ten points)
static_assert(PS_TOPK_MAX <= KEEP_CAP && PS_TOPK_MAX + 2 * MAX_TRIPLES <= CAND_CAP - STEP_CAP &&
                  CAND_CAP - PS_TOPK_MAX >= 320,
              "what a step brings fits an emptied buffer");

struct Key {
  u64 a, b;   // Pareto: (mem, comm); top-k: (comm, mem)
  u32 i;      // index within the model
};
__device__ __forceinline__ bool key_less(const Key& x, const Key& y) {
  if (x.a != y.a) return x.a < y.a;
  if (x.b != y.b) return x.b < y.b;
  return x.i < y.i;
}
__device__ __forceinline__ Key key_shfl_xor(const Key& x, int lanes) {
  Key o;
  o.a = __shfl_xor_sync(0xffffffffu, x.a, lanes);
  o.b = __shfl_xor_sync(0xffffffffu, x.b, lanes);
  o.i = __shfl_xor_sync(0xffffffffu, x.i, lanes);
  return o;
}

// What a (Theta, Omega, G) triple contributes, the same for every unit.  With E = elements
// of a state on one (t, k) position, s = its largest data-axis shard, u = the
// reconstruction unit and x = the ring volume in elements (all four the same for Theta,
// Omega and G), a triple's
//   bytes          = ka * E + kb * s + kc * u     (Theorem 1, widths of Remark 1)
//   communication  = kx * x                       (Theorem 2 [+ unpriced traffic])
//   host bytes     = kh * s                       (mode O)
// with small integer coefficients that depend only on the triple's modes and the model's
// byte widths.
struct __align__(16) Triple {
  double k[3];          // ka, kb, kc
  u64 kh, kx;           // as the sweep's type
  u32 allowed;          // allowed activation digits: bits 0..4, 8..12, 16..20 for the three CLS_* of a unit;
                        // bits 24.. reductions to shards (2 bits) and all-reduces (1 bit) beyond kx * x, where
                        // shards have copies
  u32 pad;
};

// the cell of a whole number below 2^63: exponent and three bits of the fraction of it as a
// double, so that a lower cell means a strictly smaller number (rounding keeps the order);
// 0 has a cell of its own
__device__ __forceinline__ int cell_of(double m) {
  return max((__double2hiint(m) >> 17) - (1023 << 3) + 1, 0);
}
__device__ __forceinline__ int cell_of(u64 m) { return cell_of(as<double>(m)); }

// what decides whether one triple dominates another (see dominated)
struct Rank {
  u32 bytes;            // ka, ka + kb, kc, a byte each
  u32 volume;           // kx, kh
  u32 allowed;          // as in Triple
};

struct BlockShared {
  ModelRec rec;
  Triple tri[MAX_TRIPLES];
  float4 pair[25];                         // Theta and Omega, by NM * (Theta's digit) + Omega's: the coefficients of
                                           // E, s and u, and that of the host bytes
  alignas(8) u32 mask[3][25][10];                     // FIX_TOPS where the flags allow a point, by CLS_*, pair and G's digit: the
                                           // activation digits that keep bytes (ScreenUnit leaves out those that they
                                           // never allow), the offloaded one
  u32 digits;                              // activation digits that the flags allow with any triple, a byte each CLS_*
  alignas(16) u64 cell[CELLS];             // the histogram
  u64 scan[4];                             // of its four quarters
  u64 cand_a[CAND_CAP], cand_b[CAND_CAP];  // the buffer: Pareto (mem, comm), top-k (comm, least mem)
  u32 cand_i[CAND_CAP];
  unsigned char place[CAND_CAP];           // candidates that stay
  int kept;
  u32 flags[SEG / 32];                     // units of the segment with survivors
  alignas(8) u16 heavy[SEG];               // the same as a list
  alignas(8) u32 least_cell[SEG];                     // top-k: the lowest cell that a survivor of a listed unit falls into
                                           // (Pareto: drop_tied's indices)
  unsigned char live[MAX_TRIPLES + 3];     // the triples the passes walk
  Rank rank[MAX_TRIPLES];
  unsigned char alive[MAX_TRIPLES + 3];
  u32 n_live, n_heavy, next1, next2, n_cand, full, limit_cell, survivors;
};

// Three arrays in the place of others that are not read any more when they are written.
struct Scratch {
  u64* a;
  u64* b;
  u32* i;
};
// a ranking's result on its way into the buffer.  Pareto (KEEP_CAP entries): a model's last ranking, behind
// the passes.  Top-k (PAIRWISE entries, in the place of the screening's masks): also behind the passes, since a cut
// inside them sorts in place -- the buffer is full then, and a later segment is screened with the masks.
template <int KIND> __device__ __forceinline__ Scratch ranked_scratch(BlockShared& sh);
// top-k: the candidates that are left, while their points fill the buffer (CAND_CAP entries, behind the passes)
__device__ __forceinline__ Scratch hits(BlockShared& sh);

// the composition bits of a factorisation against the required ones (ps_filter.skip_rejected:
// a factorisation that misses one has no survivor, so it need not be evaluated)
__device__ __forceinline__ bool unit_rejected(const SpaceDev& sp, const ModelRec& rec, const Fact& f, u32 req_cv) {
  const bool t_heads = rec.heads % f.T == 0, k_layers = rec.L % f.K == 0, tp_le = f.T <= sp.tp_max_valid;
  const bool whole = (u64)f.T * f.K * f.D == (u64)f.N;
  u32 cv = (t_heads ? PS_F_T_DIV_HEADS : 0) | (k_layers ? PS_F_K_DIV_LAYERS : 0) | (tp_le ? PS_F_TP_LE_MAX : 0) |
           PS_F_AXIS_FORM;
  if (t_heads && k_layers && tp_le && whole) cv |= PS_F_CV;
  return (cv & req_cv) != req_cv;
}

// ------------------------------------------------------------------ screening
// Bytes as 16-bit figures, two of them in a word: a unit is some fraction of the capacity (or of
// the host budget), everything held is rounded down and everything that bounds it up.  So a point
// that fits fits here too, and one that fits here but not in whole bytes is within a few units of
// the capacity; what the screening lets through is tested in whole bytes by the passes.  A field
// of a bound is 2^15 + the units that are left (-1: it cannot fit), a field held at most 2^15 - 2:
// after one subtraction for both halves their top bits say which of the two points fit, with no
// borrow from one half to the other.  Against a compare of doubles per point (two cycles of the
// fp64 pipe, chained through predicates; as many instructions as points) the screening of 4096
// models of the stress configuration takes 230 us instead of 517 (top-k) and 270 instead of 581
// (Pareto, with a host budget), the sweeps 621 instead of 768 and 656 instead of 824.
constexpr u32 FIX_TERM = 16383;            // a term held, at most: above every bound, and two of them below 2^15
constexpr float FIX_CAP = 16382.0f;        // the capacity in units
constexpr u32 FIX_NEVER = 0x7fff7fffu;     // bounds that nothing is below
constexpr u32 FIX_TOPS = 0x80008000u;

struct Scale {
  float unit;                              // units per byte
  float room;                              // the capacity in units, rounded up, and one
};
__device__ __forceinline__ Scale scale_of(u64 cap) {
  Scale r;
  r.unit = cap <= (u64)FIX_CAP ? 1.0f : __fdiv_rd(FIX_CAP, __ull2float_ru(cap));
  r.room = __fadd_ru(__fmul_ru(__ull2float_ru(cap), r.unit), 1.0f);
  return r;
}
__device__ __forceinline__ u32 both_halves(u32 x) { return x * 0x10001u; }
__device__ __forceinline__ u32 term_of(float x) { return __float2uint_rd(fminf(x, (float)FIX_TERM)); }
// what is left of a capacity beside `held`, as the field of a bound less that of FIX_NEVER
__device__ __forceinline__ u32 room_beside(const Scale& c, float held) {
  return __float2uint_rd(fminf(fmaxf(__fsub_ru(c.room, held), 0.0f), (float)FIX_TERM));
}
// below 1 / x for a whole x below 2^24 (rcp.approx is right to one unit in the last place)
__device__ __forceinline__ float below_reciprocal(u32 x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"((float)x));
  return __fmul_rd(r, 1.0f - 0x1p-22f);
}

// A unit as a lane holds it for the screening, no figure above what LaneUnit has for it.
template <int NM, bool HOST_LIMITED>
struct ScreenUnit {
  float E, s, u, shard;                    // as LaneUnit's, in units
  u32 gr_mem[NM], gr_host;                 // G's terms, in both halves
  u32 bound[NM][2], host_bound[2];         // by activation variant; the halves are the tensor-axis variants
  u32 room, host_room;                     // the capacity and the host budget, in both halves
  u32 cls;

  __device__ __forceinline__ void load(const SpaceDev& sp, const ModelRec& rec, const Fact& f, u32 modemap,
                                       const Scale& cap, const Scale& host, u32 digits_of_any) {
    const u32 G = sp.repl > 1 ? f.D / gcd_u32(sp.repl, f.D) : f.D;
    cls = f.D == 1 ? CLS_ONE_DEVICE : (G == 1 ? CLS_ALL_COPIES : CLS_SHARDED);
    const float over_t = below_reciprocal(f.T), over_tk = below_reciprocal(f.T * f.K), over_g = below_reciprocal(G);
    const float P = __ull2float_rd(rec.P);
    E = __fmul_rd(__fmul_rd(P, cap.unit), over_tk);
    s = G == 1 ? E : __fmul_rd(E, over_g);
    u = __fmul_rd(__fmul_rd(__ull2float_rd(rec.unit), cap.unit), over_t);
    const float ss = (float)sp.sstar_units;
    auto held = [&](u32 mode, float full, float part, float unit) {      // Theorem 1, as mu_elems
      const float p = mode == PS_MODE_R ? full : (in_set(SET_SHARDLIKE, mode) ? part : 0.0f);
      return mode == PS_MODE_SG ? __fmaf_rd(unit, ss, p) : (mode == PS_MODE_M ? unit : p);
    };
#pragma unroll
    for (int d = 0; d < NM; ++d)
      gr_mem[d] = both_halves(term_of(__fmul_rd(held(digit_mode(modemap, d), E, s, u), (float)rec.wG)));
    room = FIX_NEVER + both_halves(room_beside(cap, 0.0f));
    if (HOST_LIMITED) {
      shard = __fmul_rd(__fmul_rd(__fmul_rd(P, host.unit), over_tk), over_g);
      gr_host = both_halves(term_of(__fmul_rd(shard, (float)(2 * rec.wG))));
      host_room = FIX_NEVER + both_halves(room_beside(host, 0.0f));
    }
    const u32 digits = digits_of_any >> (8 * cls);       // that the flags allow in a unit of this class
#pragma unroll
    for (u32 v = 0; v < 2; ++v) {
      u32 left[NM][2], host_left[2] = {0, 0};
#pragma unroll
      for (u32 tau = 0; tau < 2; ++tau) {
        const bool have = v < sp.nv && tau < sp.nt;
        const float A = __ull2float_rd(rec.A[v]), over = tau == 0 ? over_t : 1.0f;
        const float EA = __fmul_rd(__fmul_rd(A, cap.unit), over);
        const float uA = __fmul_rd(__fmul_rd(__ull2float_rd(rec.UA[v]), cap.unit), over);
        const float shA = G == 1 ? EA : __fmul_rd(EA, over_g);
#pragma unroll
        for (int d = 0; d < NM; ++d) {
          const u32 mode = digit_mode(modemap, d);       // (the offloaded digit's points: `room`)
          left[d][tau] = have && mode != PS_MODE_O && ((digits >> d) & 1u) ? room_beside(cap, held(mode, EA, shA, uA)) : 0;
        }
        if (HOST_LIMITED && have)
          host_left[tau] = room_beside(host, __fmul_rd(__fmul_rd(__fmul_rd(A, host.unit), over), (float)(2 * sp.accum)));
      }
#pragma unroll
      for (int d = 0; d < NM; ++d) bound[d][v] = FIX_NEVER + left[d][0] + (left[d][1] << 16);
      if (HOST_LIMITED) host_bound[v] = FIX_NEVER + host_left[0] + (host_left[1] << 16);
    }
  }
};

// May any point of the lane's unit whose (Theta, Omega) pair lies in [p0, p1) survive?
template <int NM, bool HOST_LIMITED>
__device__ __forceinline__ bool screen_pairs(const BlockShared& sh, const ScreenUnit<NM, HOST_LIMITED>& su, u32 modemap,
                                             u32 p0, u32 p1) {
  u32 any = 0;
#pragma unroll 1
  for (u32 p = p0; p < p1; ++p) {
    const float4 k = sh.pair[p];
    const u32 to_mem = both_halves(term_of(__fmaf_rd(su.E, k.x, __fmaf_rd(su.s, k.y, __fmul_rd(su.u, k.z)))));
    u32 fits_host[2] = {FIX_TOPS, FIX_TOPS}, fits_off[2] = {FIX_TOPS, FIX_TOPS};   // (G not offloaded, offloaded)
    if (HOST_LIMITED) {
      // the triple's own host bytes against the budget, and with offloaded activations beside them
      const u32 h = both_halves(term_of(__fmul_rd(su.shard, k.w)));
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const u32 with_g = o ? h + su.gr_host : h;
        fits_host[o] = su.host_room - with_g;
        fits_off[o] = (su.host_bound[0] - with_g) | (su.host_bound[1] - with_g);
      }
    }
    u32 mask[2 * NM];                                    // by G's digit: activation digits that keep bytes, and the offloaded one
    {
      const uint2* row = reinterpret_cast<const uint2*>(sh.mask[su.cls][p]);
#pragma unroll
      for (int gr = 0; gr < NM; ++gr) { const uint2 w = row[gr]; mask[2 * gr] = w.x; mask[2 * gr + 1] = w.y; }
    }
#pragma unroll
    for (int gr = 0; gr < NM; ++gr) {
      const u32 m = to_mem + su.gr_mem[gr];
      u32 fit = 0;
#pragma unroll
      for (int d = 0; d < NM; ++d)
        if (NM < 5 || digit_mode(modemap, d) != PS_MODE_O) fit |= (su.bound[d][0] - m) | (su.bound[d][1] - m);
      // (the variants of the offloaded digit have the same bytes: one compare)
      const u32 off = su.room - m;
      const bool g_off = digit_mode(modemap, gr) == PS_MODE_O;
      any |= (fit & mask[2 * gr] & (g_off ? fits_host[1] : fits_host[0])) |
             (off & mask[2 * gr + 1] & (g_off ? fits_off[1] : fits_off[0]));
    }
  }
  return (any & FIX_TOPS) != 0;
}

// Pareto: the classes of units in which triple t can never add to a frontier because triple
// a has, in every unit, a point with no more bytes, volume and host bytes wherever t has one
// -- and fewer bytes, or a smaller index for the same pair.  (E >= s >= 1: bytes are compared
// as ka (E - s) + (ka + kb) s + kc u.)  Bits 0, 8 and 16 for the three CLS_*.
__device__ __forceinline__ u32 dominated(const Rank& t, const Rank& a, bool a_first) {
  const bool less = (a.bytes & 0xff00u) < (t.bytes & 0xff00u);
  const u32 copies_t = t.allowed >> 24, copies_a = a.allowed >> 24;
  if (__vcmpgtu4(a.bytes, t.bytes) | __vcmpgtu2(a.volume, t.volume)) return 0;
  if (!(less || a_first) || (copies_a & 3u) > (copies_t & 3u) || (copies_a & 4u) > (copies_t & 4u)) return 0;
  const u32 misses = t.allowed & ~a.allowed & 0x1f1f1fu; // digits that t may use and a may not
  return __vcmpeq4(misses, 0u) & 0x010101u;
}

// ------------------------------------------------------------------ the buffer
// The block's n candidates, sorted by key (a bitonic network over shared memory).
__device__ __noinline__ void sort_candidates(BlockShared& sh, int n) {
  const int tid = threadIdx.x, threads = blockDim.x;
  u64* const a = sh.cand_a;
  u64* const b = sh.cand_b;
  u32* const ix = sh.cand_i;
  int size = 32;
  while (size < n) size <<= 1;
  for (int p = n + tid; p < size; p += threads) { a[p] = U64MAX; b[p] = U64MAX; ix[p] = NO_CODE; }
  for (int k = 2; k <= size; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      __syncthreads();
      for (int t = tid; t < size / 2; t += threads) {
        const int lo = 2 * t - (t & (j - 1)), hi = lo + j;       // the pair's places, j apart
        const Key x{a[lo], b[lo], ix[lo]}, y{a[hi], b[hi], ix[hi]};
        if (key_less(y, x) == ((lo & k) == 0)) {
          a[lo] = y.a; b[lo] = y.b; ix[lo] = y.i;
          a[hi] = x.a; b[hi] = x.b; ix[hi] = x.i;
        }
      }
    }
  __syncthreads();
}

// Up to this many candidates every thread tests its own against all others (no barrier in
// the loop); more are sorted, whose work grows more slowly.  With 64 instead of 128 the stress
// configuration takes 586 us for top-k instead of 591, but the frontiers 555 instead of 546 and
// those of 1024 models 86 instead of 83.
constexpr int PAIRWISE = 128;

static_assert(CAND_CAP > PAIRWISE, "a full buffer is sorted in place: a ranking would overwrite the masks of later segments");
static_assert(sizeof(BlockShared::cell) >= CAND_CAP * sizeof(u64) && sizeof(BlockShared::least_cell) >= CAND_CAP * sizeof(u64) &&
                  sizeof(BlockShared::heavy) >= CAND_CAP * sizeof(u32) && CAND_CAP >= KEEP_CAP &&
                  sizeof(BlockShared::mask) >= PAIRWISE * (2 * sizeof(u64) + sizeof(u32)),
              "scratch in the place of others");
__device__ __forceinline__ Scratch hits(BlockShared& sh) {
  return Scratch{sh.cell, reinterpret_cast<u64*>(sh.least_cell), reinterpret_cast<u32*>(sh.heavy)};
}
template <> __device__ __forceinline__ Scratch ranked_scratch<PS_REDUCE_PARETO>(BlockShared& sh) { return hits(sh); }
template <> __device__ __forceinline__ Scratch ranked_scratch<PS_REDUCE_TOPK>(BlockShared& sh) {
  u64* const a = reinterpret_cast<u64*>(sh.mask);
  return Scratch{a, a + PAIRWISE, reinterpret_cast<u32*>(a + 2 * PAIRWISE)};
}

// Closes up the candidates p < n for which `keep(p, its key)` holds, by one warp, 32 at a
// time; returns how many are left.  (`keep` is called by all lanes; a code of NO_CODE and keys
// of U64MAX stand for the places from n on.)
template <typename F>
__device__ __forceinline__ int close_up(BlockShared& sh, int n, F&& keep) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    int left = 0;
    for (int base = 0; base < n; base += 32) {
      const int p = base + lane;
      const Key e = p < n ? Key{sh.cand_a[p], sh.cand_b[p], sh.cand_i[p]} : Key{U64MAX, U64MAX, NO_CODE};
      const bool stays = keep(p, e);
      const u32 votes = __ballot_sync(0xffffffffu, stays);
      if (stays) {
        const int to = left + __popc(votes & ((1u << lane) - 1u));
        sh.cand_a[to] = e.a; sh.cand_b[to] = e.b; sh.cand_i[to] = e.i;
      }
      left += __popc(votes);
      __syncwarp();
    }
    if (lane == 0) sh.kept = left;
  }
  __syncthreads();
  return sh.kept;
}

// Pareto: drops the candidates that another one beats strictly, and (of more than PAIRWISE) of
// those with the same pair all but the smallest unit's, whose points have the smaller indices;
// returns how many are left.  (Points that cost nothing are the same pair in every unit: kept
// side by side, they alone would fill the buffer, 1360 of them in a model of the stress
// configuration.)  Those of one pair in one unit all stay: the indices of their points are not known.
__device__ __noinline__ int drop_dominated(BlockShared& sh, int n) {
  const int tid = threadIdx.x, lane = tid & 31, threads = blockDim.x;
  __syncthreads();
  if (n <= PAIRWISE) {
    for (int p = tid; p < n; p += threads) {
      const u64 a = sh.cand_a[p], b = sh.cand_b[p];
      bool keep = a != U64MAX;
#pragma unroll 4
      for (int q = 0; q < n; ++q) {
        const u64 oa = sh.cand_a[q], ob = sh.cand_b[q];
        if (oa <= a && ob <= b && (oa < a || ob < b)) keep = false;
      }
      sh.place[p] = keep ? 1 : 0;
    }
    __syncthreads();
    return close_up(sh, n, [&](int p, const Key&) { return p < n && sh.place[p] != 0; });
  }
  sort_candidates(sh, n);
  // In the order of (bytes, communication, unit) a candidate stays if nothing before it has as
  // little communication, or only its own pair in its own unit.
  u64 least = U64MAX, least_at = 0;                      // the least communication before these 32, the bytes
  u32 least_unit = 0;                                    // and the unit that it came with first
  return close_up(sh, n, [&](int, const Key& e) {
    u64 m = e.b, at = e.a;
    bool tied = least == e.b && least_at == e.a;         // with the candidate before
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 mu = __shfl_up_sync(0xffffffffu, m, o), au = __shfl_up_sync(0xffffffffu, at, o);
      if (o == 1 && lane > 0) tied = mu == e.b && au == e.a;
      if (lane >= o && mu <= m) { m = mu; at = au; }
    }
    if (least <= m) { m = least; at = least_at; }        // (m: the least up to here, earliest first)
    // the unit of the pair's first candidate
    const u32 firsts = __ballot_sync(0xffffffffu, !tied) & (0xffffffffu >> (31 - lane));
    u32 unit = __shfl_sync(0xffffffffu, e.i >> 8, firsts ? 31 - __clz(firsts) : 0);
    if (firsts == 0) unit = least_unit;
    const bool keep = e.a != U64MAX && m == e.b && at == e.a && unit == e.i >> 8;
    const u32 kept = __ballot_sync(0xffffffffu, keep);
    if (kept) least_unit = __shfl_sync(0xffffffffu, unit, 31 - __clz(kept));
    least = __shfl_sync(0xffffffffu, m, 31);
    least_at = __shfl_sync(0xffffffffu, at, 31);
    return keep;
  });
}

// Pareto: the first `front` of the n candidates are the frontier that a cut left, in ascending
// order of bytes; of the others drops those that one of them beats, or that are its pair in a
// larger unit.  A search per candidate where a cut sorts: where a cell of the histogram holds
// many points (28 ragged shapes, every valid placement of every composition: a quarter of all
// candidates get past the staircase) the sweep takes 0.54 ms instead of 0.78.
__device__ __noinline__ int drop_beaten(BlockShared& sh, int front, int n) {
  __syncthreads();
  for (int p = front + threadIdx.x; p < n; p += blockDim.x) {
    const u64 mem = sh.cand_a[p], comm = sh.cand_b[p];
    int lo = 0, hi = front;                              // lo: the entries with as many bytes at most
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (sh.cand_a[mid] <= mem) lo = mid + 1; else hi = mid;
    }
    bool keep = mem != U64MAX;
    if (lo > 0 && sh.cand_b[lo - 1] <= comm)
      keep = sh.cand_a[lo - 1] == mem && sh.cand_b[lo - 1] == comm && sh.cand_i[lo - 1] >> 8 >= sh.cand_i[p] >> 8;
    sh.place[p] = keep ? 1 : 0;
  }
  __syncthreads();
  return close_up(sh, n, [&](int p, const Key&) { return p < n && (p < front || sh.place[p] != 0); });
}

// The n candidates sorted by key, without those of a pair that a smaller index has (Pareto,
// after drop_dominated and with indices), or the k smallest of them (top-k).  Returns how many
// stay; more than KEEP_CAP are not all written.
template <int KIND>
__device__ __noinline__ int rank_candidates(BlockShared& sh, int n, int k_keep) {
  constexpr bool PARETO = KIND == PS_REDUCE_PARETO;
  const int tid = threadIdx.x, threads = blockDim.x;
  __syncthreads();
  if (!PARETO && n > PAIRWISE) {
    sort_candidates(sh, n);
    return min(n, k_keep);
  }
  const Scratch sorted = ranked_scratch<KIND>(sh);
  if (tid == 0) sh.kept = 0;
  if (PARETO)
    for (int p = tid; p < n; p += threads) {
      const u64 a = sh.cand_a[p];
      const u32 ix = sh.cand_i[p];
      bool keep = true;
      for (int q = 0; q < n; ++q)
        if (sh.cand_a[q] == a && sh.cand_i[q] < ix) keep = false;
      sh.place[p] = keep ? 1 : 0;
    }
  __syncthreads();
  for (int p = tid; p < n; p += threads) {
    const Key e{sh.cand_a[p], sh.cand_b[p], sh.cand_i[p]};
    if (PARETO && sh.place[p] == 0) continue;
    int rank = 0;
#pragma unroll 4
    for (int q = 0; q < n; ++q) {
      if (PARETO) rank += (sh.place[q] != 0 && sh.cand_a[q] < e.a) ? 1 : 0;
      else rank += key_less(Key{sh.cand_a[q], sh.cand_b[q], sh.cand_i[q]}, e) ? 1 : 0;
    }
    if (PARETO) atomicAdd(&sh.kept, 1);
    if (rank < KEEP_CAP) { sorted.a[rank] = e.a; sorted.b[rank] = e.b; sorted.i[rank] = e.i; }
  }
  __syncthreads();
  const int stay = PARETO ? sh.kept : min(n, k_keep);
  for (int p = tid; p < min(stay, KEEP_CAP); p += threads) {
    sh.cand_a[p] = sorted.a[p]; sh.cand_b[p] = sorted.b[p]; sh.cand_i[p] = sorted.i[p];
  }
  __syncthreads();
  return stay;
}

// Top-k: the n candidates sorted by (communication, least bytes, unit), cut to the k smallest and
// those that are the same in all three as the last of these (the order of points inside a unit is
// not known here).  Each of the k stands for a point of its own, the least of its points, and the
// points of a larger unit have larger indices: so what is dropped has none of the k smallest.
// Returns how many stay.
__device__ __noinline__ int cut_candidates(BlockShared& sh, int n, int k) {
  __syncthreads();
  if (n <= k) return n;
  if (n > PAIRWISE) sort_candidates(sh, n);
  else rank_candidates<PS_REDUCE_TOPK>(sh, n, n);
  const u64 a = sh.cand_a[k - 1], b = sh.cand_b[k - 1];
  const u32 unit = sh.cand_i[k - 1] >> 8;
  if (threadIdx.x == 0) sh.kept = k;
  __syncthreads();
  for (int p = k + threadIdx.x; p < n; p += blockDim.x)
    if (sh.cand_a[p] == a && sh.cand_b[p] == b && sh.cand_i[p] >> 8 == unit) atomicAdd(&sh.kept, 1);
  __syncthreads();
  return sh.kept;
}

// ------------------------------------------------------------------ candidates to points
// A (unit, triple, tensor-axis variant) that the second pass let through: its points, in
// index order, by one thread.  `visit(mem, idx)` sees those that the flags, the capacity
// and the host budget allow, until it returns false.
template <int NM, int DEGREES, typename F>
__device__ __forceinline__ void points_of(const SpaceDev& sp, const BlockShared& sh, u32 code, u32 modemap, u64 cap_x,
                                          u64 host_x, F&& visit) {
  constexpr u32 N3 = NM * NM * NM, NC = N3 * NM;
  const ModelRec& rec = sh.rec;
  const u32 unit = code >> 8, t = (code >> 1) & 127u, tau = code & 1u;
  const Fact f = sp.facts[unit];
  const UnitBase ub = unit_of<DEGREES>(sp, rec, f);
  const u32 modes[3] = {digit_mode(modemap, t % NM), digit_mode(modemap, (t / NM) % NM), digit_mode(modemap, t / (NM * NM))};
  const u32 width[3] = {rec.wT, rec.wO, rec.wG};
  u64 mem = 0, host = 0;
#pragma unroll
  for (int st = 0; st < 3; ++st) {
    mem += mad_small(mu_elems(modes[st], ub.E2, ub.sh, ub.u, sp.sstar_units), width[st], 0);
    if (modes[st] == PS_MODE_O) host += mad_small(ub.sh, (st == 0 ? 2 * sp.accum + 1 : 2) * width[st], 0);
  }
  const u32 allowed = sh.tri[t].allowed >> (8 * ub.cls);
#pragma unroll 1
  for (u32 v = 0; v < sp.nv; ++v) {
    const ActBase ab = act_of<DEGREES>(sp, rec, f, ub, v, tau);
    const bool host_fits = host + 2 * ab.EA * sp.accum < host_x;
#pragma unroll 1
    for (u32 d = 0; d < NM; ++d) {
      const u32 mode = digit_mode(modemap, d);
      const u64 m = mem + mu_elems(mode, ab.EA, ab.shA, ab.uA, sp.sstar_units);
      if (((allowed >> d) & 1u) && m < cap_x && (mode != PS_MODE_O || host_fits) &&
          !visit(m, (unit * sp.nvt + v * sp.nt + tau) * NC + t + d * N3))
        return;
    }
  }
}

// Pareto: the index of each candidate's point, the smallest with the candidate's bytes
template <int NM, int DEGREES>
__device__ __noinline__ void resolve_candidates(const SpaceDev& sp, BlockShared& sh, int n, u32 modemap, u64 cap_x,
                                                u64 host_x, u32* index) {
  __syncthreads();
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    const u32 code = sh.cand_i[p];
    const u64 want = sh.cand_a[p];
    points_of<NM, DEGREES>(sp, sh, code, modemap, cap_x, host_x, [&](u64 m, u32 idx) {
      if (m == want) index[p] = idx;
      return m != want;
    });
  }
  __syncthreads();
}

// Pareto, where drop_dominated leaves too many: of the candidates of one pair in one unit only
// the one with the smallest index stays.
template <int NM, int DEGREES>
__device__ __noinline__ int drop_tied(const SpaceDev& sp, BlockShared& sh, int n, u32 modemap, u64 cap_x, u64 host_x) {
  u32* const index = sh.least_cell;                      // (top-k's)
  resolve_candidates<NM, DEGREES>(sp, sh, n, modemap, cap_x, host_x, index);
  for (int p = threadIdx.x; p < n; p += blockDim.x) {
    bool keep = true;
    for (int q = 0; q < n; ++q)
      if (sh.cand_a[q] == sh.cand_a[p] && index[q] < index[p]) keep = false;   // (same bytes: same pair)
    sh.place[p] = keep ? 1 : 0;
  }
  __syncthreads();
  return close_up(sh, n, [&](int p, const Key&) { return p < n && sh.place[p] != 0; });
}

// top-k: the points of the buffer's n candidates take their places, as many candidates at a
// time as surely fit, the smallest first; those at or above the k-th smallest point so far are
// left out.  Returns the number of points.
template <int NM, int DEGREES>
__device__ __noinline__ int resolve_points(const SpaceDev& sp, BlockShared& sh, int n, int k, u32 modemap, u64 cap_x,
                                           u64 host_x) {
  const int tid = threadIdx.x, threads = blockDim.x;
  const u32 per_unit = sp.nvt * NM * NM * NM * NM;
  const Scratch hit = hits(sh);
  __syncthreads();
  for (int p = tid; p < n; p += threads) { hit.a[p] = sh.cand_a[p]; hit.b[p] = sh.cand_b[p]; hit.i[p] = sh.cand_i[p]; }
  if (tid == 0) sh.n_cand = 0;
  __syncthreads();
  Key threshold{U64MAX, U64MAX, NO_CODE};
  for (int base = 0; base < n;) {
    int room = (CAND_CAP - (int)sh.n_cand) / (2 * NM);
    if (room < min(n - base, 32)) {
      const int left = rank_candidates<PS_REDUCE_TOPK>(sh, (int)sh.n_cand, k);
      if (left == k) threshold = Key{sh.cand_a[k - 1], sh.cand_b[k - 1], sh.cand_i[k - 1]};
      __syncthreads();
      if (tid == 0) sh.n_cand = (u32)left;
      room = (CAND_CAP - left) / (2 * NM);
    }
    __syncthreads();
    const int now = min(n - base, room);
    for (int j = base + tid; j < base + now; j += threads) {
      const u64 comm = hit.a[j];
      const u32 code = hit.i[j];
      if (!key_less(Key{comm, hit.b[j], (code >> 8) * per_unit}, threshold)) continue;
      points_of<NM, DEGREES>(sp, sh, code, modemap, cap_x, host_x, [&](u64 m, u32 idx) {
        if (key_less(Key{comm, m, idx}, threshold)) {
          const u32 at = atomicAdd(&sh.n_cand, 1u);
          sh.cand_a[at] = comm; sh.cand_b[at] = m; sh.cand_i[at] = idx;
        }
        return true;
      });
    }
    base += now;
    __syncthreads();
  }
  return (int)sh.n_cand;
}

// ------------------------------------------------------------------ one point, the slow exact path
// one point of a model from its index, as an output entry
template <int DEGREES>
__device__ __forceinline__ PointOut eval_local(const SpaceDev& sp, const ModelRec& rec, u32 lidx) {
  const LocalPoint lp = decode_local(sp, lidx);
  const Fact f = sp.facts[lp.unit];
  const UnitBase ub = unit_of<DEGREES>(sp, rec, f);
  return eval_point_from(rec, f, ub, act_of<DEGREES>(sp, rec, f, ub, lp.v, lp.tau), lp.tau, digit_mode(sp.modemap, lp.dth),
                         digit_mode(sp.modemap, lp.dom), digit_mode(sp.modemap, lp.dgr), digit_mode(sp.modemap, lp.dac),
                         sp.tp_coll, sp.sstar_units, sp.accum);
}

__device__ __forceinline__ void write_entry(ps_front_entry* out, const PointOut& po, u64 comm, u64 idx) {
  ps_front_entry e;
  e.mem = po.mem; e.comm = comm; e.host = po.host; e.idx = idx; e.flags = po.flags | PS_F_FEASIBLE; e.pad = 0;
  *out = e;
}
__device__ __forceinline__ void write_empty(ps_front_entry* out) {
  ps_front_entry e;
  e.mem = 0; e.comm = 0; e.host = 0; e.idx = 0; e.flags = 0; e.pad = 0;
  *out = e;
}

// A frontier with more than KEEP_CAP entries does not fit the block's buffer.  The block
// then computes the model's frontier by the definition, one entry per pass over the
// model's points: the next entry is the survivor with the fewest bytes among those with
// more bytes and less communication than the last entry (fewest communication, then
// smallest index, on ties).  Slow (passes = frontier length), bounded memory, any length.
// Not inlined, so that it does not weigh on the sweep's registers.
template <int DEGREES>
__device__ __noinline__ void frontier_by_definition(const SpaceDev& sp, const SweepArgs& args, const ModelRec& rec,
                                                    u32 model, u64* a, u64* b, u32* ix) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, threads = blockDim.x;
  u32 found[PS_MAX_CAPS];
  for (u32 ci = 0; ci < PS_MAX_CAPS; ++ci) found[ci] = 0;
  u64 last_mem = 0, last_comm = U64MAX;
  bool have_last = false;
  const u32 ppm = (u32)sp.ppm;
  for (u32 pass = 0; pass <= ppm; ++pass) {             // a frontier has at most ppm entries
    Key best{U64MAX, U64MAX, 0xffffffffu};
    for (u64 lidx = tid; lidx < ppm; lidx += threads) {
      const PointOut po = eval_local<DEGREES>(sp, rec, (u32)lidx);
      const u64 comm = args.comm_kind == PS_COMM_PAPER ? po.comm_paper : po.comm_paper + po.comm_ext;
      const bool survivor = po.mem <= args.cap_max && po.host <= args.host_cap &&
                            (po.flags & args.require_flags) == args.require_flags;
      const bool beyond = !have_last || (po.mem > last_mem && comm < last_comm);
      const Key key{po.mem, comm, (u32)lidx};
      if (survivor && beyond && key_less(key, best)) best = key;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const Key other = key_shfl_xor(best, o);
      if (key_less(other, best)) best = other;
    }
    __syncthreads();
    if (lane == 0) { a[warp] = best.a; b[warp] = best.b; ix[warp] = best.i; }      // the warps' best candidates of the pass
    __syncthreads();
    best = Key{a[0], b[0], ix[0]};
    for (int w = 1; w < threads >> 5; ++w) {
      const Key other{a[w], b[w], ix[w]};
      if (key_less(other, best)) best = other;
    }
    if (best.i == 0xffffffffu) break;                   // nothing beyond the last entry: done
    for (u32 ci = 0; ci < args.n_caps; ++ci) {
      if (best.a > args.caps[ci]) continue;
      const u32 slot = found[ci]++;
      if (slot < args.max_entries && tid == 0)
        write_entry(args.out + ((u64)model * args.n_caps + ci) * args.max_entries + slot, eval_local<DEGREES>(sp, rec, best.i),
                    best.b, (u64)model * sp.ppm + best.i);
    }
    last_mem = best.a; last_comm = best.b; have_last = true;
  }
  for (u32 ci = 0; ci < args.n_caps; ++ci) {
    ps_front_entry* out = args.out + ((u64)model * args.n_caps + ci) * args.max_entries;
    for (u64 p = found[ci] + (u64)tid; p < args.max_entries; p += threads) write_empty(out + p);
    if (tid == 0) {
      args.counts[(u64)model * args.n_caps + ci] = found[ci];
      if (found[ci] > args.max_entries) report(args.status, ST_TRUNCATED);
    }
  }
}

// ------------------------------------------------------------------ the sweep
// Registers of a thread.  With powers of two the frontier passes fit 96, and five blocks of four warps
// share an SM instead of four (4096 models of the stress configuration 577 -> 543 us); the divisions of other
// degrees spill then (ragged counts 83 -> 102 us).  The first pass of top-k holds twenty bounds and spills
// at 96, so it is compiled for both, and launch_sweep_d chooses.  At 80 the passes spill in any case.
constexpr int FEW_REGISTERS = 96, ALL_REGISTERS = 128;

// KIND: the reduction; NM: allowed modes; T: the type of byte counts and volumes (see
// LaneUnit); HOST_LIMITED: the filter has a host budget (without one the host bytes are
// never formed).  The number of warps is the launch's (see launch_sweep).
template <int KIND, int NM, typename T, bool HOST_LIMITED, int DEGREES, int REGISTERS>
__global__ void __maxnreg__(REGISTERS) k_sweep(const __grid_constant__ SpaceDev sp, const __grid_constant__ SweepArgs args) {
  constexpr int N2 = NM * NM, N3 = NM * NM * NM;
  constexpr bool PARETO = KIND == PS_REDUCE_PARETO;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BlockShared& sh = *reinterpret_cast<BlockShared*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, threads = blockDim.x, warps = threads >> 5;

  // blocks are handed out in grid order: the models with the most expected work first
  const u32 model = sp.order[blockIdx.x];
  if (tid < (int)(sizeof(ModelRec) / 16))
    reinterpret_cast<uint4*>(&sh.rec)[tid] = reinterpret_cast<const uint4*>(&sp.recs[model])[tid];
  if (tid == 0) { sh.survivors = 0; sh.n_cand = 0; sh.digits = 0; }
  for (int j = tid; j < CELLS; j += threads) sh.cell[j] = PARETO ? U64MAX : 0;
  __syncthreads();
  const ModelRec& rec = sh.rec;

  const u32 req = args.require_flags;
  const bool ext_in_objective = args.comm_kind == PS_COMM_PAPER_PLUS_EXT;
  // capacities as exclusive bounds (memory stays below 2^61)
  const u64 cap_x = min(PARETO ? args.cap_max : args.caps[blockIdx.y], (u64)1 << 62) + 1;
  const u64 host_x = min(args.host_cap, HOST_BYTES_END) + 1;
  const T cap_room = as<T>(cap_x), host_room = as<T>(host_x);
  constexpr u32 CV_BITS = PS_F_CV | PS_F_T_DIV_HEADS | PS_F_K_DIV_LAYERS | PS_F_TP_LE_MAX | PS_F_AXIS_FORM;
  const u32 req_cv = req & CV_BITS;
  // with all five modes allowed digit d is mode d: the compiler then knows every
  // per-digit property below (which digit offloads, which keep a replica's own
  // activations) and drops the tests
  const u32 modemap = (NM == 5) ? 0x43210u : sp.modemap;
  constexpr u32 all = (1u << NM) - 1u;
  u32 is_o = 0;
#pragma unroll
  for (int d = 0; d < NM; ++d)
    if (digit_mode(modemap, d) == PS_MODE_O) is_o |= 1u << d;

  const bool skip = args.skip_rejected && req_cv != 0;
  // Top-k without a required flag: the first pass counts every point itself and nothing is screened
  // for (4096 models of the stress configuration in 2.16 ms instead of 2.30).
  const bool take_all = !PARETO && req == 0, screened = !skip && !take_all;

  // ---- the block's tables of triples and of states
  u32 digits_of_any = 0;
  for (int t = tid; t < N3; t += threads) {
    // activation-digit classes (Theorem 3: a replica needs its own activations)
    u32 own = 0, not_mo = 0;
    for (int d = 0; d < NM; ++d) {
      const u32 ac = digit_mode(modemap, d);
      if (in_set(SET_ACT_OWN, ac)) own |= 1u << d;
      if (!in_set(SET_M_OR_O, ac)) not_mo |= 1u << d;
    }
    const u32 th = digit_mode(modemap, t % NM), om = digit_mode(modemap, (t / NM) % NM), gr = digit_mode(modemap, t / N2);
    const bool on_shard = in_set(SET_UPDATE_ON_SHARD, om);
    const u32 modes[3] = {th, om, gr}, width[3] = {rec.wT, rec.wO, rec.wG};
    u32 a = 0, b = 0, c = 0;
    for (int st = 0; st < 3; ++st) {
      if (modes[st] == PS_MODE_R) a += width[st];
      if (in_set(SET_SHARDLIKE, modes[st])) b += width[st];
      if (modes[st] == PS_MODE_SG) c += width[st] * sp.sstar_units;   // one or two unit buffers
      if (modes[st] == PS_MODE_M) c += width[st];
    }
    const u32 h = (th == PS_MODE_O ? (2 * sp.accum + 1) * rec.wT : 0) + (om == PS_MODE_O ? 2 * rec.wO : 0) +
                  (gr == PS_MODE_O ? 2 * rec.wG : 0);
    // Theorem 2: all-reduce of replicated gradients, reduce-scatter of sharded
    // ones, two all-gathers of gathered parameters for each micro-batch
    u32 ct = (th == PS_MODE_SG) ? 2 * sp.accum : 0, co = 0;
    u32 cg = (gr == PS_MODE_R) ? 2 : (gr == PS_MODE_S ? 1 : 0);
    // With several copies of every shard (k-way replication) the communication is kx * x
    // plus what reducing gradients to shards and all-reducing them cost beyond that: x2
    // per reduction to shards, x3 per all-reduce over all devices
    u32 n2 = gr == PS_MODE_S ? 1u : 0u, n3 = gr == PS_MODE_R ? 1u : 0u;
    if (ext_in_objective) {                  // traffic the theorem does not price
      if (th == PS_MODE_O) ct += 2 * sp.accum;
      if (th == PS_MODE_R && on_shard) ct += 1;
      if (om == PS_MODE_SG) co = 1;
      if (gr == PS_MODE_SG) { cg += 2; n2 += 1; }
      if (gr == PS_MODE_M) { cg += on_shard ? 1 : 2; if (on_shard) n2 += 1; else n3 += 1; }
      if (gr == PS_MODE_O) { cg += 1; n2 += 1; }
    }
    if (sp.repl == 1) n2 = n3 = 0;           // (x2 and x3 are zero)
    const u32 a_many = allowed_act_digits(triple_bits(th, om, gr, CLS_SHARDED), req, all, own, is_o, not_mo);
    const u32 a_one = allowed_act_digits(triple_bits(th, om, gr, CLS_ONE_DEVICE), req, all, all, is_o, not_mo);
    const u32 a_copies = allowed_act_digits(triple_bits(th, om, gr, CLS_ALL_COPIES), req, all, all, is_o, not_mo);
    Triple& tr = sh.tri[t];
    tr.k[0] = a; tr.k[1] = b; tr.k[2] = c;
    tr.kh = bits<T>(as<T>(h));
    tr.kx = bits<T>(as<T>(ct * rec.wT + co * rec.wO + cg * rec.wG));
    tr.allowed = a_many | (a_one << 8) | (a_copies << 16) | (n2 << 24) | (n3 << 26);
    tr.pad = 0;
    sh.rank[t] = Rank{a | ((a + b) << 8) | (c << 16), (ct * rec.wT + co * rec.wO + cg * rec.wG) | (h << 16), tr.allowed};
    if (screened) {
      const u32 pair = (t % NM) * NM + (t / NM) % NM, gr_digit = t / N2;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const u32 digits = (tr.allowed >> (8 * c)) & all;
        *reinterpret_cast<uint2*>(&sh.mask[c][pair][2 * gr_digit]) =
            make_uint2((digits & ~is_o) ? FIX_TOPS : 0, (digits & is_o) ? FIX_TOPS : 0);
      }
    }
    digits_of_any |= tr.allowed;
  }
  digits_of_any = __reduce_or_sync(0xffffffffu, digits_of_any & 0x1f1f1fu);
  if (lane == 0 && digits_of_any) atomicOr(&sh.digits, digits_of_any);
  for (int t = tid; screened && t < N2; t += threads) {
    const u32 modes[2] = {digit_mode(modemap, t / NM), digit_mode(modemap, t % NM)}, width[2] = {rec.wT, rec.wO};
    u32 a = 0, b = 0, c = 0, h = 0;
#pragma unroll
    for (int st = 0; st < 2; ++st) {
      if (modes[st] == PS_MODE_R) a += width[st];
      if (in_set(SET_SHARDLIKE, modes[st])) b += width[st];
      if (modes[st] == PS_MODE_SG) c += width[st] * sp.sstar_units;
      if (modes[st] == PS_MODE_M) c += width[st];
      if (modes[st] == PS_MODE_O) h += (st == 0 ? 2 * sp.accum + 1 : 2) * width[st];
    }
    sh.pair[t] = make_float4((float)a, (float)b, (float)c, (float)h);
  }

  // ---- the triples that the passes walk: those that the flags allow; for Pareto only those
  // that no triple differing in one mode dominates (55 of 95 with valid points required)
  __syncthreads();
  for (int t = tid; t < N3; t += threads) {
    const Rank own = sh.rank[t];
    // (0x01 in the byte of a class with allowed digits)
    u32 used = __vcmpgtu4(own.allowed & 0x1f1f1fu, 0u) & 0x010101u;
    if (PARETO) {
      const int digit[3] = {t % NM, (t / NM) % NM, t / N2}, weight[3] = {1, NM, N2};
#pragma unroll
      for (int st = 0; st < 3; ++st)
#pragma unroll
        for (int k = 1; k < (NM > 1 ? NM : 0); ++k) {
          const int d = digit[st] + k < NM ? digit[st] + k : digit[st] + k - NM;
          used &= ~dominated(own, sh.rank[t + (d - digit[st]) * weight[st]], d < digit[st]);
        }
    }
    sh.alive[t] = used != 0;
  }
  __syncthreads();
  if (warp == 0) {
    u32 n = 0;
    for (int base = 0; base < N3; base += 32) {
      const int t = base + lane;
      const bool live = t < N3 && sh.alive[t] != 0;
      const u32 votes = __ballot_sync(0xffffffffu, live);
      if (live) sh.live[n + __popc(votes & ((1u << lane) - 1u))] = (unsigned char)t;
      n += __popc(votes);
    }
    if (lane == 0) sh.n_live = n;
  }

  int front = 0;                                     // Pareto: the buffer's first entries that are a frontier, in order
  // top-k: no candidate above these (communication, least bytes, unit) is wanted
  T most_comm = T(U64MAX), most_mem = T(U64MAX);
  u32 most_unit = NO_CODE;
  u32 survivors = 0;
  bool overflowed = false;                           // the same for every thread
  const Scale cap_scale = scale_of(cap_x - 1), host_scale = scale_of(host_x - 1);

  for (u32 seg = 0; seg < sp.n_facts; seg += SEG) {
    const u32 seg_n = min((u32)SEG, sp.n_facts - seg), n_batches = (seg_n + 31) / 32;
    __syncthreads();
    for (int j = tid; j < SEG / 32; j += threads) sh.flags[j] = 0;
    if (tid == 0) { sh.next1 = 0; sh.next2 = 0; }
    __syncthreads();
    if (take_all) {
      if (tid < SEG / 32)
        sh.flags[tid] = seg_n >= 32u * tid + 32 ? ~0u : seg_n > 32u * tid ? (1u << (seg_n - 32u * tid)) - 1u : 0u;
    } else if (skip) {
      for (u32 b = warp; b < n_batches; b += warps) {
        const u32 p = b * 32 + lane;
        const u32 votes = __ballot_sync(0xffffffffu, p < seg_n && !unit_rejected(sp, rec, sp.facts[seg + min(p, seg_n - 1)], req_cv));
        if (lane == 0) sh.flags[b] = votes;
      }
    } else {
      // ---- screening.  A batch of 32 units is shared by several warps, a part of the
      // (Theta, Omega) pairs each, where there are more warps than batches.
      const u32 parts = min(max((u32)warps / n_batches, 1u), (u32)N2);
      for (u32 item = warp; item < n_batches * parts; item += warps) {
        const u32 b = item / parts, part = item - b * parts, p = b * 32 + lane;
        const Fact f = sp.facts[seg + min(p, seg_n - 1)];
        ScreenUnit<NM, HOST_LIMITED> su;
        su.load(sp, rec, f, modemap, cap_scale, host_scale, sh.digits);
        const bool any = screen_pairs(sh, su, modemap, part * N2 / parts, (part + 1) * N2 / parts);
        const u32 votes = __ballot_sync(0xffffffffu, any && p < seg_n && !unit_rejected(sp, rec, f, req_cv));
        if (lane == 0 && votes) atomicOr(&sh.flags[b], votes);
      }
    }
    __syncthreads();
    // the flagged units as a list, a warp for each word of flags
    {
      const u32 set_here = __popc(sh.flags[lane]);
      for (u32 w = warp; w < n_batches; w += warps) {
        const u32 word = sh.flags[w];
        u32 at = __reduce_add_sync(0xffffffffu, (u32)lane < w ? set_here : 0u);
        if ((word >> lane) & 1u) {
          at += __popc(word & ((1u << lane) - 1u));
          if (!PARETO) sh.least_cell[at] = CELLS;        // (before the barrier: the first pass lowers it from any warp)
          sh.heavy[at] = (u16)(32 * w + lane);
        }
      }
      const u32 total = __reduce_add_sync(0xffffffffu, set_here);
      if (tid == 0) sh.n_heavy = total;
    }
    __syncthreads();
    const u32 n_live = sh.n_live;
    u32 n_heavy = sh.n_heavy;
    if (n_heavy == 0 || n_live == 0) continue;

    // ---- the two passes.  An item is a batch of 32 listed units and a part of the triples.
    u32 parts, n_items;
    auto deal = [&]() {
      const u32 batches = (n_heavy + 31) / 32;
      parts = min(max((u32)warps / batches, 1u), (n_live + 1) / 2);
      n_items = batches * parts;
    };
    deal();
    // walks an item's triples from place `from` of the list on; returns the place at which the
    // buffer was full, or none
    auto walk = [&](auto second, u32 item, u32 from) -> u32 {
      constexpr bool SECOND = decltype(second)::value;
      const u32 b = item / parts, part = item - b * parts, k = b * 32 + lane;
      const u32 unit = seg + sh.heavy[min(k, n_heavy - 1)];
      const Fact f = sp.facts[unit];
      const UnitBase ub = unit_of<DEGREES>(sp, rec, f);
      constexpr bool COUNTS = !PARETO && !SECOND;    // top-k's first pass counts points, the others want the least bytes
      typename std::conditional<COUNTS, LaneUnit<NM, T, HOST_LIMITED, DEGREES>, LeastUnit<NM, T, HOST_LIMITED, DEGREES>>::type lu;
      const bool live = k < n_heavy && (ub.cv & req_cv) == req_cv;
      if constexpr (COUNTS) lu.load(sp, rec, f, ub, modemap, cap_x, host_x, live);
      else lu.load(sp, rec, f, ub, modemap, cap_x, host_x, (sh.digits >> (8 * ub.cls)) & all & ~is_o, live);
      const T x = as<T>(ub.x);
      const T gx2 = as<T>((u64)rec.wG * ub.x2), gx3 = as<T>((u64)rec.wG * ub.x3);
      T axis[2];
#pragma unroll
      for (u32 tau = 0; tau < 2; ++tau)
        axis[tau] = as<T>(ext_in_objective ? model_axis_traffic(rec, f, ub, tau, sp.tp_coll, sp.accum) : 0);
      const u32 t_end = (part + 1) * n_live / parts;
      u32 lowest = CELLS;                            // top-k, first pass: the lowest cell of a survivor
      // Two triples at a time, all four candidates side by side and one vote for them: what
      // a step waits for (table loads, dependent fp64 operations, votes) is waited for once.
#pragma unroll 1
      for (u32 t0 = max(part * n_live / parts, from); t0 < t_end; t0 += 2) {
        double m[2];
        T c[2], h[2];
        u32 allowed[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const Triple& tr = sh.tri[sh.live[min(t0 + j, t_end - 1)]];
          allowed[j] = t0 + j < t_end ? (tr.allowed >> lu.shift) & lu.allowed : 0u;
          m[j] = fma(lu.E, tr.k[0], fma(lu.s, tr.k[1], lu.u * tr.k[2]));
          h[j] = T(0);
          if (HOST_LIMITED) {
            h[j] = mul_add(lu.shard, from_bits<T>(tr.kh), T(0));
            if (!(h[j] < host_room)) allowed[j] = 0;     // the triple's own host bytes against the budget
          }
          c[j] = mul_add(x, from_bits<T>(tr.kx), T(0));
          if (sp.repl > 1) c[j] += (T)((tr.allowed >> 24) & 3u) * gx2 + (T)((tr.allowed >> 26) & 1u) * gx3;
        }
        if (!__any_sync(0xffffffffu, allowed[0] | allowed[1])) continue;
        if constexpr (COUNTS) {
          // the survivors of the triples, by tensor-axis variant
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            float n[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int d = 0; d < NM; ++d) {
              if (HOST_LIMITED && digit_mode(modemap, d) == PS_MODE_O) {
                count_offloaded(n, m[j], lu.bounds(d), h[j], lu.host_bound, allowed[j] & (1u << d));
              } else {
                count_variants(n, m[j], lu.bounds(d), allowed[j] & (1u << d));
              }
            }
            const float n0 = n[0] + n[2], n1 = n[1] + n[3];
            survivors += (u32)(n0 + n1);
            const int cell0 = cell_of(c[j] + axis[0]), cell1 = cell_of(c[j] + axis[1]);
            if (n0 != 0.0f) { atomicAdd(reinterpret_cast<u32*>(&sh.cell[cell0]), (u32)n0); lowest = min(lowest, (u32)cell0); }
            if (n1 != 0.0f) { atomicAdd(reinterpret_cast<u32*>(&sh.cell[cell1]), (u32)n1); lowest = min(lowest, (u32)cell1); }
          }
        } else {
          // For a triple and a tensor-axis variant the communication does not depend on the
          // activation variant and digit, so of those that are allowed only the one with the
          // least bytes can be on a frontier -- and if it does not fit, none does.  The offloaded
          // digit keeps none.  (Where it is the only one allowed and the host budget keeps it out, the
          // capacity stands for the activations' bytes: with a test of its own for that in `cand` the
          // passes lose 5 to 12 %, 1024 models skipping rejected factorisations 83 us instead of 74.)
          bool cand[4];
          T mem[4], comm[4];
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            const int j = w >> 1, tau = w & 1;
            comm[w] = c[j] + axis[tau];
            const bool off = (allowed[j] & is_o) != 0 && (!HOST_LIMITED || h[j] < lu.host_most[tau]);
            const bool keeps = !HOST_LIMITED || (allowed[j] & ~is_o) != 0;
            mem[w] = whole<T>(m[j]) + (off ? T(0) : keeps ? lu.act[tau] : cap_room);
            cand[w] = allowed[j] != 0 && mem[w] < cap_room && (u32)tau < sp.nt;
            const int cell = cell_of(PARETO ? mem[w] : comm[w]);
            if (!SECOND) {
              if (cand[w] && bits<T>(comm[w]) < sh.cell[cell])
                atomicMin(reinterpret_cast<unsigned long long*>(&sh.cell[cell]), (unsigned long long)bits<T>(comm[w]));
            } else if (PARETO) {
              // (the first cell holds one number, zero: its own least is a bound as well)
              const u64 least = sh.cell[max(cell, 1) - 1];
              cand[w] = cand[w] && (cell == 0 ? bits<T>(comm[w]) <= least : bits<T>(comm[w]) < least);
            } else {
              cand[w] = cand[w] && cell <= (int)sh.limit_cell &&
                        (comm[w] < most_comm || (comm[w] == most_comm &&
                                                 (mem[w] < most_mem || (mem[w] == most_mem && unit <= most_unit))));
            }
          }
          if (SECOND && __any_sync(0xffffffffu, cand[0] | cand[1] | cand[2] | cand[3])) {
            u32 mine = 0;
#pragma unroll
            for (int w = 0; w < 4; ++w) mine += cand[w] ? 1u : 0u;
            u32 incl = mine;                           // inclusive prefix sum over the lanes
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const u32 up = __shfl_up_sync(0xffffffffu, incl, o);
              if (lane >= o) incl += up;
            }
            const u32 total = __shfl_sync(0xffffffffu, incl, 31);
            u32 at = 0;
            if (lane == 0) at = atomicAdd(&sh.n_cand, total);
            at = __shfl_sync(0xffffffffu, at, 0);
            // (a group that does not fit leaves empty entries where there were places)
            const bool room = at + total <= CAND_CAP;
            at += incl - mine;
#pragma unroll
            for (int w = 0; w < 4; ++w)
              if (cand[w]) {
                if (at < CAND_CAP) {
                  sh.cand_a[at] = room ? (u64)(PARETO ? mem[w] : comm[w]) : U64MAX;
                  sh.cand_b[at] = room ? (u64)(PARETO ? comm[w] : mem[w]) : U64MAX;
                  sh.cand_i[at] = room ? (unit << 8) | ((u32)sh.live[min(t0 + (w >> 1), t_end - 1)] << 1) | (w & 1) : NO_CODE;
                }
                ++at;
              }
            if (!room) return t0;
          }
        }
      }
      if (!PARETO && !SECOND && lowest < CELLS) atomicMin(&sh.least_cell[k], lowest);
      return ALL_STEPS;
    };

    for (;;) {
      u32 item = 0;
      if (lane == 0) item = atomicAdd(&sh.next1, 1u);
      item = __shfl_sync(0xffffffffu, item, 0);
      if (item >= n_items) break;
      walk(std::false_type{}, item, 0);
    }
    __syncthreads();
    // Four warps, four cells a thread.
    constexpr int SCAN_WARPS = 4, PER = CELLS / (SCAN_WARPS * 32);
    static_assert(PER == 4, "cells of a thread: two 16-byte accesses");
    if (PARETO) {
      // cell j then holds the least communication of any survivor so far in cells 0..j
      u64 c[PER], incl = U64MAX;
      if (warp < SCAN_WARPS) {
        const ulonglong2* const from = reinterpret_cast<const ulonglong2*>(sh.cell + tid * PER);
        const ulonglong2 lo = from[0], hi = from[1];
        c[0] = lo.x; c[1] = min(c[0], (u64)lo.y); c[2] = min(c[1], (u64)hi.x); c[3] = min(c[2], (u64)hi.y);
        incl = c[3];
        for (int o = 1; o < 32; o <<= 1) {
          const u64 up = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl = min(incl, up);
        }
        if (lane == 31) sh.scan[warp] = incl;
      }
      __syncthreads();
      if (warp < SCAN_WARPS) {
        u64 before = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) before = U64MAX;
        for (int w = 0; w < warp; ++w) before = min(before, sh.scan[w]);
        ulonglong2* const to = reinterpret_cast<ulonglong2*>(sh.cell + tid * PER);
        to[0] = make_ulonglong2(min(c[0], before), min(c[1], before));
        to[1] = make_ulonglong2(min(c[2], before), min(c[3], before));
      }
    } else {
      // the first cell up to which there are k survivors (the last one if there are fewer)
      u32 c[PER], incl = 0;
      if (warp < SCAN_WARPS) {
        const ulonglong2* const from = reinterpret_cast<const ulonglong2*>(sh.cell + tid * PER);
        const ulonglong2 lo = from[0], hi = from[1];
        c[0] = (u32)lo.x; c[1] = c[0] + (u32)lo.y; c[2] = c[1] + (u32)hi.x; c[3] = c[2] + (u32)hi.y;
        incl = c[3];
        for (int o = 1; o < 32; o <<= 1) {
          const u32 up = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += up;
        }
        if (lane == 31) sh.scan[warp] = incl;
      }
      if (tid == 0) sh.limit_cell = CELLS - 1;
      __syncthreads();
      if (warp < SCAN_WARPS) {
        u32 before = incl - c[PER - 1];
        for (int w = 0; w < warp; ++w) before += (u32)sh.scan[w];
        if (before < args.max_entries && before + c[PER - 1] >= args.max_entries) {
          int q = 0;
          while (before + c[q] < args.max_entries) ++q;
          sh.limit_cell = tid * PER + q;
        }
      }
      __syncthreads();
      if (warp == 0) {
        // and only the units with a survivor that low are walked again
        const u32 limit = sh.limit_cell;
        u32 n = 0;
        for (u32 base = 0; base < n_heavy; base += 32) {
          const bool again = base + lane < n_heavy && sh.least_cell[base + lane] <= limit;
          const u16 p = sh.heavy[min(base + lane, n_heavy - 1)];
          const u32 votes = __ballot_sync(0xffffffffu, again);
          if (again) sh.heavy[n + __popc(votes & ((1u << lane) - 1u))] = p;
          n += __popc(votes);
          __syncwarp();
        }
        if (lane == 0) sh.n_heavy = n;
      }
    }
    __syncthreads();
    if (!PARETO) {
      n_heavy = sh.n_heavy;
      if (n_heavy == 0) continue;
      deal();
    }
    u32 item = ALL_STEPS, from = 0;                  // the warp's item in hand and the triple to resume at
    for (;;) {
      if (tid == 0) sh.full = 0;
      __syncthreads();
      for (;;) {
        if (item == ALL_STEPS) {
          u32 k = 0;
          if (lane == 0) k = atomicAdd(&sh.next2, 1u);
          item = __shfl_sync(0xffffffffu, k, 0);
          from = 0;
        }
        if (item >= n_items) break;
        from = walk(std::true_type{}, item, from);
        if (from != ALL_STEPS) {
          if (lane == 0) sh.full = 1;
          break;
        }
        item = ALL_STEPS;
      }
      __syncthreads();
      if (!sh.full) break;
      int n = min((int)sh.n_cand, CAND_CAP);
      if (PARETO) {
        if (front != 0) n = drop_beaten(sh, front, n);
        if (front == 0 || n > CAND_CAP / 2) {
          n = drop_dominated(sh, n);                 // (sorts: more than PAIRWISE)
          if (n > CAND_CAP - STEP_CAP) n = drop_tied<NM, DEGREES>(sp, sh, n, modemap, cap_x, host_x);
          if (n > CAND_CAP - STEP_CAP) { overflowed = true; break; }
          front = n;
        }
      } else {
        const int k = (int)args.max_entries;
        n = cut_candidates(sh, n, k);
        most_comm = as<T>(sh.cand_a[k - 1]); most_mem = as<T>(sh.cand_b[k - 1]); most_unit = sh.cand_i[k - 1] >> 8;
      }
      __syncthreads();
      if (tid == 0) sh.n_cand = (u32)n;
    }
    if (overflowed) break;
  }

  // ---- the model's result, sorted, in the buffer
  __syncthreads();
  int n_list = 0;
  if (!overflowed) {
    if (PARETO) {
      n_list = drop_dominated(sh, (int)sh.n_cand);
      resolve_candidates<NM, DEGREES>(sp, sh, n_list, modemap, cap_x, host_x, sh.cand_i);
      n_list = rank_candidates<KIND>(sh, n_list, 0);
    } else {
      for (int o = 16; o > 0; o >>= 1) survivors += __shfl_xor_sync(0xffffffffu, survivors, o);
      if (lane == 0 && survivors) atomicAdd(&sh.survivors, survivors);
      n_list = cut_candidates(sh, (int)sh.n_cand, (int)args.max_entries);
      n_list = resolve_points<NM, DEGREES>(sp, sh, n_list, (int)args.max_entries, modemap, cap_x, host_x);
      n_list = rank_candidates<KIND>(sh, n_list, (int)args.max_entries);
    }
    overflowed = PARETO && n_list > KEEP_CAP;
    __syncthreads();
  }
  if (overflowed) {
    frontier_by_definition<DEGREES>(sp, args, rec, model, sh.cand_a, sh.cand_b, sh.cand_i);
    return;
  }

  // ---- emit.  Each entry is evaluated again from its index (host bytes and flags come
  // from there; mem and comm must agree).  Pareto: a tighter capacity keeps the head of the
  // staircase (dominance only ever looks at entries with smaller-or-equal memory).  Top-k:
  // a block per capacity, so everything in the list already fits.
  const u32 c_begin = PARETO ? 0 : blockIdx.y, c_end = PARETO ? args.n_caps : blockIdx.y + 1;
  ps_front_entry* const rows = args.out + (u64)model * args.n_caps * args.max_entries;
  for (u32 ci = c_begin; ci < c_end; ++ci) {
    int n_cap = n_list;
    if (PARETO) {
      int lo = 0, hi = n_list;
      while (lo < hi) { const int mid = (lo + hi) >> 1; if (sh.cand_a[mid] <= args.caps[ci]) lo = mid + 1; else hi = mid; }
      n_cap = lo;
    }
    if (tid == 0) {
      args.counts[(u64)model * args.n_caps + ci] = PARETO ? (u32)n_cap : sh.survivors;
      // a frontier that does not fit the caller's rows: its head is written, the count is the true one
      if (PARETO && (u32)n_cap > args.max_entries) report(args.status, ST_TRUNCATED);
    }
    for (u64 p = (u64)n_cap + tid; p < args.max_entries; p += threads) write_empty(rows + (u64)ci * args.max_entries + p);
  }
  for (int p = tid; p < n_list && (u32)p < args.max_entries; p += threads) {
    const u32 lidx = sh.cand_i[p];
    const PointOut po = eval_local<DEGREES>(sp, rec, lidx);
    const u64 comm = args.comm_kind == PS_COMM_PAPER ? po.comm_paper : po.comm_paper + po.comm_ext;
    const u64 list_mem = PARETO ? sh.cand_a[p] : sh.cand_b[p];
    const u64 list_comm = PARETO ? sh.cand_b[p] : sh.cand_a[p];
    if (po.mem != list_mem || comm != list_comm) report(args.status, ST_SELF_CHECK);
    for (u32 ci = c_begin; ci < c_end; ++ci)
      if (!PARETO || po.mem <= args.caps[ci])
        write_entry(rows + (u64)ci * args.max_entries + p, po, comm, (u64)model * sp.ppm + lidx);
  }
}

}  // namespace

// ------------------------------------------------------------------ launchers
template <int KIND, int NM, typename T, bool HOST_LIMITED, int DEGREES, int REGISTERS = ALL_REGISTERS>
static cudaError_t launch_sweep_p(const SpaceDev& sp, const SweepArgs& a, int warps, cudaStream_t stream) {
  const dim3 grid(sp.n_models, KIND == PS_REDUCE_PARETO ? 1 : a.n_caps);
  const size_t smem = sizeof(BlockShared);
  const auto kernel = k_sweep<KIND, NM, T, HOST_LIMITED, DEGREES, REGISTERS>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<grid, warps * 32, smem, stream>>>(sp, a);
  return cudaGetLastError();
}

// Top-k with powers of two: 96 registers where five blocks an SM instead of four outweigh the spills.  A table
// of one round of blocks never gains (300 models of the stress configuration 138 -> 144 us, with a host budget 139 -> 156).
// Beyond it, with 128 -> 96 registers:
//   up to 32 factorisations, blocks that last alike: 700 models of a data axis 78 -> 64 us, skipping rejected
//     factorisations 73 -> 61, 1100 105 -> 92 (900 76.5 -> 78.6, the worst);
//   four modes, 8 bytes of spills: up to five blocks an SM 128 is better (700 models of a grid 87 -> 97), beyond
//     96 (900: 111 -> 98, with a host budget 119 -> 113; 1180 skipping 107 -> 95);
//   five modes, 48 bytes of spills, 104 with a host budget: up to eight blocks an SM 128 is better (700 models of the
//     stress configuration 148 -> 163, 1000 skipping 115 -> 121, with a host budget as well 116 -> 133), beyond 96
//     (1350: 232 -> 220, 2400: 375 -> 356, skipping 206 -> 192);
//   without required flags the blocks last alike and long: where 96 make it a single round, 700 models 448 -> 374.
static bool few_registers(const SpaceDev& sp, const SweepArgs& a, int sm_count) {
  const u64 blocks = (u64)sp.n_models * a.n_caps, sms = (u64)sm_count;
  const u64 most = sp.n_facts <= 32 ? 4 : sp.nm <= 4 ? 5 : 8;
  return blocks > most * sms || (a.require_flags == 0 && blocks > 4 * sms && blocks <= 5 * sms);
}

template <int KIND, int NM, bool HOST_LIMITED>
static cudaError_t launch_sweep_d(const SpaceDev& sp, const SweepArgs& a, int sm_count, int warps, cudaStream_t stream) {
  if (!sp.all_pow2) return launch_sweep_p<KIND, NM, double, HOST_LIMITED, DEGREES_ANY>(sp, a, warps, stream);
  constexpr int MANY = KIND == PS_REDUCE_PARETO ? FEW_REGISTERS : ALL_REGISTERS;
  return few_registers(sp, a, sm_count)
             ? launch_sweep_p<KIND, NM, double, HOST_LIMITED, DEGREES_POW2, FEW_REGISTERS>(sp, a, warps, stream)
             : launch_sweep_p<KIND, NM, double, HOST_LIMITED, DEGREES_POW2, MANY>(sp, a, warps, stream);
}

template <int KIND, int NM>
static cudaError_t launch_sweep_t(const SpaceDev& sp, const SweepArgs& a, int sm_count, int warps, cudaStream_t stream) {
  // every byte count exact in a double
  if (sp.all_small && a.cap_max < ((u64)1 << 53) - 1)
    return NM < 4 || a.host_cap < HOST_BYTES_END ? launch_sweep_d<KIND, NM, true>(sp, a, sm_count, warps, stream)
                                                 : launch_sweep_d<KIND, NM, NM < 4>(sp, a, sm_count, warps, stream);
  return launch_sweep_p<KIND, NM, u64, true, DEGREES_EITHER>(sp, a, warps, stream);
}

template <int KIND>
static cudaError_t launch_sweep_k(const SpaceDev& sp, const SweepArgs& a, int sm_count, int warps, cudaStream_t stream) {
  switch (sp.nm) {
    case 1: return launch_sweep_t<KIND, 1>(sp, a, sm_count, warps, stream);
    case 2: return launch_sweep_t<KIND, 2>(sp, a, sm_count, warps, stream);
    case 3: return launch_sweep_t<KIND, 3>(sp, a, sm_count, warps, stream);
    case 4: return launch_sweep_t<KIND, 4>(sp, a, sm_count, warps, stream);
    default: return launch_sweep_t<KIND, 5>(sp, a, sm_count, warps, stream);
  }
}

cudaError_t launch_sweep(int kind, const SpaceDev& sp, const SweepArgs& a, int sm_count, cudaStream_t stream) {
  // Warps of a block: as many as give every SM about sixteen, four at least (a table of
  // many models) and sixteen at most (a few models, where one block's latency is the call's).
  const u64 blocks = (u64)sp.n_models * (kind == PS_REDUCE_PARETO ? 1 : a.n_caps);
  int warps = 4;
  while (warps < SWEEP_MAX_WARPS && blocks * warps * 2 <= (u64)sm_count * 16) warps *= 2;
  return kind == PS_REDUCE_PARETO ? launch_sweep_k<PS_REDUCE_PARETO>(sp, a, sm_count, warps, stream)
                                  : launch_sweep_k<PS_REDUCE_TOPK>(sp, a, sm_count, warps, stream);
}
