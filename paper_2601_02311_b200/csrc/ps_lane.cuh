// A factorisation ("unit") of a model as one lane holds it, for the kernels in which the
// lanes of a warp own units and walk the (Theta, Omega, G) triples together.
#pragma once
#include <type_traits>
#include "ps_device.cuh"

// ------------------------------------------------------------------ small arithmetic
// a * k + acc for a 64-bit a and a small 32-bit k: two multiply-adds
__device__ __forceinline__ u64 mad_small(u64 a, u32 k, u64 acc) {
  u64 r = (u64)(u32)a * (u64)k + acc;
  r += (u64)((u32)(a >> 32) * k) << 32;
  return r;
}
__device__ __forceinline__ u64 mul_add(u64 a, u64 k, u64 acc) { return mad_small(a, (u32)k, acc); }
__device__ __forceinline__ double mul_add(double a, double k, double acc) { return fma(a, k, acc); }

// ------------------------------------------------------------------ a lane's unit
template <typename T> __device__ __forceinline__ T as(u64 x);
template <> __device__ __forceinline__ u64 as<u64>(u64 x) { return x; }
template <> __device__ __forceinline__ double as<double>(u64 x) { return (double)(long long)x; }
template <typename T> __device__ __forceinline__ T whole(double x);      // a whole number
template <> __device__ __forceinline__ u64 whole<u64>(double x) { return (u64)(long long)x; }
template <> __device__ __forceinline__ double whole<double>(double x) { return x; }
template <typename T> __device__ __forceinline__ u64 bits(T x);
template <> __device__ __forceinline__ u64 bits<u64>(u64 x) { return x; }
template <> __device__ __forceinline__ u64 bits<double>(double x) { return (u64)__double_as_longlong(x); }
template <typename T> __device__ __forceinline__ T from_bits(u64 x);
template <> __device__ __forceinline__ u64 from_bits<u64>(u64 x) { return x; }
template <> __device__ __forceinline__ double from_bits<double>(u64 x) { return __longlong_as_double((long long)x); }

// Which degrees a kernel is compiled for: powers of two (every division a shift), any (the
// divisions), or both with a uniform branch.  The code for the other kind is not just jumped over,
// it takes the place of code that runs in the instruction cache.
enum { DEGREES_ANY = 0, DEGREES_POW2 = 1, DEGREES_EITHER = 2 };
template <int DEGREES = DEGREES_EITHER>
__device__ __forceinline__ UnitBase unit_of(const SpaceDev& sp, const ModelRec& rec, const Fact& f) {
  if (DEGREES == DEGREES_POW2 || (DEGREES == DEGREES_EITHER && sp.all_pow2)) return unit_base_pow2(rec, f, pow2_of(f, sp.repl), sp.tp_max_valid, true);
  return unit_base(rec, f, sp.tp_max_valid, true, sp.repl);
}
template <int DEGREES = DEGREES_EITHER>
__device__ __forceinline__ ActBase act_of(const SpaceDev& sp, const ModelRec& rec, const Fact& f, const UnitBase& ub,
                                          u32 v, u32 tau) {
  if (DEGREES == DEGREES_POW2 || (DEGREES == DEGREES_EITHER && sp.all_pow2)) return act_base_pow2(rec, pow2_of(f, sp.repl), v, tau);
  return act_base(rec, f, v, tau, ub.G);
}

// A unit as a lane holds it.  A triple's own device bytes are doubles: they stay below 2^52 (48
// bytes of each of 2^46 elements and of two units of 2^36), where doubles are exact, and a bound
// on them that is rounded, above 2^53, lies above them all the same.  T is the type of volumes,
// host bytes and whole points' bytes: double where all of a space are below 2^53, else u64.  (With
// the triple's bytes in 64-bit integers there too, top-k of 2048 shapes of the stress
// configuration with 64 micro-batches a step took 2.40 ms without required flags instead of
// 1.27.)  Variants are slots q = 2 v + tau; a slot that the space does not have bounds
// everything out.
template <int NM, typename T, bool HOST_LIMITED, int DEGREES = DEGREES_EITHER>
struct LaneUnit {
  double E, s, u;            // elements of a state, of its largest shard, of a reconstruction unit
  double gr_mem[NM];         // G's terms
  T shard, gr_host;          // for host bytes; only mode O has any
  // a triple whose own bytes are below bound[d][q] fits the capacity with activation digit
  // d under variant q.  The offloaded digit keeps no activation bytes: its bound is the
  // capacity for every variant the space has, and its host bytes have to fit too.
  T bound[NM][4], host_bound[4];
  double rounded[std::is_same<T, double>::value ? 1 : NM][4];              // bound as doubles, where T is not
  u32 allowed, shift;        // digits of a triple that count for this unit: (bits >> shift) & allowed

  __device__ __forceinline__ void load(const SpaceDev& sp, const ModelRec& rec, const Fact& f, const UnitBase& ub,
                                       u32 modemap, u64 cap_x, u64 host_x, bool live) {
    E = as<double>(ub.E2); s = as<double>(ub.sh); u = as<double>(ub.u);
    shard = as<T>(ub.sh);
    gr_host = as<T>(mad_small(ub.sh, 2 * rec.wG, 0));
#pragma unroll
    for (int d = 0; d < NM; ++d)
      gr_mem[d] = as<double>(mad_small(mu_elems(digit_mode(modemap, d), ub.E2, ub.sh, ub.u, sp.sstar_units), rec.wG, 0));
#pragma unroll
    for (u32 q = 0; q < 4; ++q) {
      const u32 v = q >> 1, tau = q & 1;
      const bool have = v < sp.nv && tau < sp.nt;
      const ActBase ab = act_of<DEGREES>(sp, rec, f, ub, v, tau);
#pragma unroll
      for (int d = 0; d < NM; ++d) {
        const u64 am = mu_elems(digit_mode(modemap, d), ab.EA, ab.shA, ab.uA, sp.sstar_units);
        bound[d][q] = as<T>(have && am < cap_x ? cap_x - am : 0);
        if constexpr (!std::is_same<T, double>::value) rounded[d][q] = as<double>(bound[d][q]);
      }
      if (HOST_LIMITED) {
        const u64 ah = 2 * ab.EA * sp.accum;             // offload after fwd, reload for bwd, per micro-batch
        // (rounded only above 2^53, where no host figure of the double case reaches)
        host_bound[q] = as<T>(have && ah < host_x ? host_x - ah : 0);
      }
    }
    shift = 8 * ub.cls;
    allowed = live ? (1u << NM) - 1u : 0u;
  }
  __device__ __forceinline__ const double* bounds(int d) const {
    if constexpr (std::is_same<T, double>::value) return bound[d];
    else return rounded[d];
  }
};

// A unit as a lane holds it where only the least bytes of a (triple, tensor-axis variant) count.  The flags
// allow the digits that keep activation bytes all together or not at all: whether one of them may stand
// beside a triple depends on the triple only for the offloaded digit (allowed_act_digits).  So their least
// bytes are a figure of the unit, and no bound per digit and variant is held (40 registers in doubles).
template <int NM, typename T, bool HOST_LIMITED, int DEGREES>
struct LeastUnit {
  double E, s, u;
  T shard;
  T act[2], host_most[2];    // by tensor-axis variant: least activation bytes of `digits`, at most the capacity, and the
                             // most that a triple's host bytes may be below, with offloaded activations beside them
  u32 allowed, shift;

  // digits: those that keep bytes and are allowed in a unit of this class
  __device__ __forceinline__ void load(const SpaceDev& sp, const ModelRec& rec, const Fact& f, const UnitBase& ub,
                                       u32 modemap, u64 cap_x, u64 host_x, u32 digits, bool live) {
    E = as<double>(ub.E2); s = as<double>(ub.sh); u = as<double>(ub.u);
    shard = as<T>(ub.sh);
#pragma unroll
    for (u32 tau = 0; tau < 2; ++tau) {
      u64 least = cap_x, most = 0;
#pragma unroll
      for (u32 v = 0; v < 2; ++v) {
        const bool have = v < sp.nv && tau < sp.nt;
        const ActBase ab = act_of<DEGREES>(sp, rec, f, ub, v, tau);
#pragma unroll
        for (int d = 0; d < NM; ++d)
          if (have && ((digits >> d) & 1u))
            least = min(least, mu_elems(digit_mode(modemap, d), ab.EA, ab.shA, ab.uA, sp.sstar_units));
        const u64 ah = 2 * ab.EA * sp.accum;
        if (HOST_LIMITED && have && ah < host_x) most = max(most, host_x - ah);
      }
      act[tau] = as<T>(least);
      host_most[tau] = as<T>(most);
    }
    shift = 8 * ub.cls;
    allowed = live ? (1u << NM) - 1u : 0u;
  }
};

// Survivors of the lane's unit among the four variants of one activation digit: a compare
// per point on the fp64 pipe, masked by its input predicate, counted with predicated fp32
// adds (small integers are exact).
__device__ __forceinline__ void count_variants(float* n, double m, const double* b, u32 on) {
  asm("{\n\t"
      ".reg .pred q, p0, p1, p2, p3;\n\t"
      "setp.ne.u32 q, %9, 0;\n\t"
      "setp.lt.and.f64 p0, %4, %5, q;\n\t"
      "setp.lt.and.f64 p1, %4, %6, q;\n\t"
      "setp.lt.and.f64 p2, %4, %7, q;\n\t"
      "setp.lt.and.f64 p3, %4, %8, q;\n\t"
      "@p0 add.f32 %0, %0, 0f3F800000;\n\t"
      "@p1 add.f32 %1, %1, 0f3F800000;\n\t"
      "@p2 add.f32 %2, %2, 0f3F800000;\n\t"
      "@p3 add.f32 %3, %3, 0f3F800000;\n\t"
      "}"
      : "+f"(n[0]), "+f"(n[1]), "+f"(n[2]), "+f"(n[3])
      : "d"(m), "d"(b[0]), "d"(b[1]), "d"(b[2]), "d"(b[3]), "r"(on));
}
// The same for the offloaded digit under a host budget: a bound for the triple's host bytes each as well.  Left
// to the compiler as conditions, a top-k sweep with a host budget waited for the additions one after the other:
// 300 models of the stress configuration without required flags 323 -> 282 us, 500 skipping 115 -> 99.
__device__ __forceinline__ void count_offloaded(float* n, double m, const double* b, double h, const double* hb, u32 on) {
  asm("{\n\t"
      ".reg .pred q, p0, p1, p2, p3;\n\t"
      "setp.ne.u32 q, %9, 0;\n\t"
      "setp.lt.and.f64 p0, %10, %11, q;\n\t"
      "setp.lt.and.f64 p1, %10, %12, q;\n\t"
      "setp.lt.and.f64 p2, %10, %13, q;\n\t"
      "setp.lt.and.f64 p3, %10, %14, q;\n\t"
      "setp.lt.and.f64 p0, %4, %5, p0;\n\t"
      "setp.lt.and.f64 p1, %4, %6, p1;\n\t"
      "setp.lt.and.f64 p2, %4, %7, p2;\n\t"
      "setp.lt.and.f64 p3, %4, %8, p3;\n\t"
      "@p0 add.f32 %0, %0, 0f3F800000;\n\t"
      "@p1 add.f32 %1, %1, 0f3F800000;\n\t"
      "@p2 add.f32 %2, %2, 0f3F800000;\n\t"
      "@p3 add.f32 %3, %3, 0f3F800000;\n\t"
      "}"
      : "+f"(n[0]), "+f"(n[1]), "+f"(n[2]), "+f"(n[3])
      : "d"(m), "d"(b[0]), "d"(b[1]), "d"(b[2]), "d"(b[3]), "r"(on), "d"(h), "d"(hb[0]), "d"(hb[1]), "d"(hb[2]), "d"(hb[3]));
}
__device__ __forceinline__ void count_offloaded(float* n, double m, const double* b, u64 h, const u64* hb, u32 on) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if ((on != 0) & (m < b[q]) & (h < hb[q])) n[q] += 1.0f;
}
