// ig_meet.cuh -- what the CTAs of a resident solve exchange through L2: posted values.
#pragma once

#include "ig_device.cuh"

namespace ig {
namespace {

// One posted value: the number of the meeting beside it, written and read as one 16-byte word, so
// that a reader that sees the number has the value. Slots alternate between two buffers: a CTA
// posts for meeting i + 2 only after meeting i + 1, for which every CTA had read the slots of i.
struct __align__(16) Slot {
  double value;
  unsigned long long number;
};

// Ahead of a mesh's slots. word: the one-launch solves of the mesh so far (times 2^16) plus the CTAs of the
// current one that have begun. The last of them moves it on to the next solve: by then every CTA has its
// number, whenever it began. team: the solve (its number + 1, times 2^16) that was settled last and how many
// CTAs share it.
struct __align__(16) MeetHead {
  unsigned long long word, team;
};
static_assert(sizeof(MeetHead) == sizeof(Slot), "one slot");

// The CTAs of a solve wait for one another, so those that share it must all run at once, and nothing makes
// sure that a grid starts as a whole when other work holds some of the SMs. So they settle who takes part:
// the last of them to begin settles on all; one that has waited long enough (enough(polls)) settles on
// those that have begun by then (they run and will see it), and a CTA that begins after that leaves at
// once. One word decides (compare-and-swap), so all read the same. ALL: all or none.
struct Team {
  unsigned long long solve;  // number of the solve
  int rank;                  // in the order of beginning; takes part if below size
  int size;                  // CTAs that share the solve (-1: not settled within the limits)
};
__device__ __forceinline__ unsigned long long load_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
struct Arrival {  // the words as a CTA that begins finds them
  unsigned long long word, team;
};
__device__ __forceinline__ Arrival arrive(MeetHead* h, int count) {
  if (count == 1) return {atomicAdd(&h->word, 1ull << 16), 0ull};
  const unsigned long long s = load_relaxed(&h->team);
  return {atomicAdd(&h->word, 1ull), s};
}
template <bool ALL = false, typename Enough>
__device__ __forceinline__ Team join_team(MeetHead* h, int count, const Arrival& a, long long limit,
                                          const Enough& enough) {
  if (count == 1) return Team{a.word >> 16, 0, 1};
  unsigned long long s = a.team;
  Team t{a.word >> 16, (int)(a.word & 0xffffu), -1};
  const unsigned long long mark = t.solve + 1ull;
  auto settle = [&](unsigned long long size) {  // a failed swap found this solve settled already
    const unsigned long long was = atomicCAS(&h->team, s, mark << 16 | size);
    s = was == s ? (mark << 16 | size) : was;
  };
  if (t.rank == count - 1) {
    if (s >> 16 != mark) settle((unsigned long long)count);
    atomicExch(&h->word, mark << 16);  // (one that sees this first looks at team again)
  } else {
    for (long long spins = 0; s >> 16 != mark && spins < limit; ++spins) {
      const bool now = enough(spins);
      const unsigned long long begun = now ? load_relaxed(&h->word) : 0ull;
      if (now && begun >> 16 == t.solve) settle(ALL ? 0ull : begun & 0xffffu);
      else s = load_relaxed(&h->team);
    }
  }
  if (s >> 16 == mark) t.size = (int)(s & 0xffffu);
  return t;
}

__device__ __forceinline__ double not_a_number() { return __longlong_as_double(0x7ff8000000000000ll); }

__device__ __forceinline__ void post(Slot* s, double value, unsigned long long number) {
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(s),
               "l"(__double_as_longlong(value)), "l"(number)
               : "memory");
}
// ACQUIRE: with the value comes what its CTA released (an acquire load per slot: a fence after
// relaxed loads took the geodesic case from 8.3 to 9.6 us an iteration).
template <bool ACQUIRE>
__device__ __forceinline__ bool peek(const Slot* s, unsigned long long number, double& value) {
  unsigned long long a, b;
  if constexpr (ACQUIRE)
    asm volatile("{\n\t.reg .b128 t;\n\tld.acquire.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(a), "=l"(b)
                 : "l"(s)
                 : "memory");
  else
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(a), "=l"(b)
                 : "l"(s)
                 : "memory");
  value = __longlong_as_double((long long)a);
  return b == number;
}
// `count` posted partials buf[8 * i + value], on the kWarps warps of a CTA (PartialMap: a lane takes a few
// tiles of one value, all polled together, 0 past the last). late is set when a wait ran out.
template <int NV>
constexpr int kLaneTiles = (kResMaxCtas + PartialMap<NV>::kStride - 1) / PartialMap<NV>::kStride;
template <int NV, bool ACQUIRE>
__device__ __forceinline__ void collect(const Slot* buf, int count, unsigned long long number, int patience,
                                        double (&b)[kLaneTiles<NV>], bool& late) {
  using Map = PartialMap<NV>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, val = Map::value(lane);
  const int first = Map::first(warp, lane);
  constexpr int J = kLaneTiles<NV>;
  unsigned want = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    b[j] = 0.0;
    if (val < NV && first + j * Map::kStride < count) want |= 1u << j;
  }
  // all the missing slots of a round are loaded before any is looked at
  for (int spins = 0; want != 0 && !late; late = ++spins > patience) {
    double x[J];
    bool there[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const bool ask = (want >> j & 1u) != 0;
      there[j] = peek<ACQUIRE>(buf + (ask ? 8 * (size_t)(first + j * Map::kStride) + val : 0), number, x[j]) && ask;
    }
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (there[j]) {
        b[j] = x[j];
        want &= ~(1u << j);
      }
  }
}
// The lane's sum of them.
template <int NV, bool ACQUIRE>
__device__ __forceinline__ double collect_sum(const Slot* buf, int count, unsigned long long number, int patience,
                                              bool& late) {
  constexpr int J = kLaneTiles<NV>;
  double b[J];
  collect<NV, ACQUIRE>(buf, count, number, patience, b, late);
  const int steps = (count + PartialMap<NV>::kStride - 1) / PartialMap<NV>::kStride;
  double a = 0.0;
#pragma unroll
  for (int j = 0; j < J; ++j)
    if (j < steps) a += b[j];
  return a;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

}  // namespace
}  // namespace ig
