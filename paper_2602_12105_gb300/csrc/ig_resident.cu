// ig_resident.cu -- the FP64 conjugate-gradient solve of a single mesh in one launch, with the mesh's
// rows held in shared memory (the solve of ig_pcg.cu: the same row arithmetic, tiles and order of the
// sums, so the same bits).
//
// A mesh of at most kResMaxRows rows per SM gets one tile per CTA and at most one CTA per SM
// (the tile rule in ig_api.cu). Its CTAs keep their rows' operator, direction, residual and solution
// on chip through the whole solve; only z = D^-1 r, which the neighbours' rows gather, goes through
// global memory (L2). Per iteration the CTAs meet twice, to add p.q and then r.z and r.r; every CTA adds
// all the tiles' partials and runs the finish step on its own copy of the solve state,
// so no step waits for one last CTA, and no kernel boundary or graph node lies in the loop.
//
// A CTA of a large mesh takes all of an SM's shared memory, so other kernels on the GPU (another stream's)
// can keep some of the CTAs from starting. The solve waits some 0.2 ms for them and then goes on with those
// that have begun (join_team, solve_shared), from global memory. 184,470 rows, k = 4, while another kernel
// holds SMs for 10 ms: 1.8 ms with none held, 2.8 with one held and 3.1 with 30 (the two-kernel graph loop
// 2.6 in all of these; a cooperative launch, which starts only as a whole, 11.4).
//
// Measured, per iteration (the two-kernel graph loop before, and this): 163,842 rows k = 3 41 -> 25 us
// and k = 4 47 -> 31 us, 66,049 rows k = 1 23 -> 7.4 us, 5,917 rows k = 1 20.6 -> 6.3 us, 642 rows k = 3
// (a cluster of 6 CTAs; three CTAs of 256 rows before) 10 -> 6 us.
//
// What bounds it: on large meshes FP64 instructions (of 26 us, 163,842 rows, k = 3: 3 go without the
// gathers, 11 without the SpMV's multiplications, 5.5 without the update; 7.7 are the two meetings). A warp's FP64
// instruction occupies its SM sub-partition for 64 cycles (16 per SM), so the 45 per row and iteration
// (three columns) take 11.7 us on 163,842 rows; eight row warps are enough to issue them, and fewer
// threads leave fewer sums to add (the sums of 32 warps would take 2.2 us of FP64 issue in the
// update alone, those of 8 a quarter). On small meshes the chain of an iteration: two gathers, two
// meetings of about 1 us (a store to L2, then a load that sees it), and sums (in fixed point where that is
// shorter) and divisions whose every FP64 step costs 64 cycles.
#include "ig_meet.cuh"
#include "ig_tiles64.cuh"

namespace ig {

namespace {

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double peer_load(const double* p, int rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

// What the host lays out in dynamic shared memory: rows of rp entries; aw slots of the operator (a
// wider slice's further slots are read from global memory), and the solution when it fits.
struct ResLayout {
  int rp;      // rows per CTA
  int aw;      // operator slots per row on chip
  int x_on;    // the solution is on chip
  int bytes;
};

struct ResShared {
  MeshDev md;
  SolveScal st;
  double red[8 * kWarps];
  double tot[8];
  double box[2][8];          // cluster: this CTA's posted sums, by parity of the meeting
  Team team;                 // the CTAs that share the solve
  int width[kResMaxRows / 32];
};

constexpr int kResThreads = kBlock + 32;  // eight warps take the rows; the ninth finishes a meeting

// Where the CTAs meet. CLUSTER: all of them form one thread-block cluster (at most 16 CTAs).
//
// A meeting adds per-thread sums over all tiles, a warp to a value, in fixed point: the row warps
// leave their totals in red; after a barrier the tile's sums are added and posted; the row warps collect every
// tile's; after another barrier warp v adds those of value v into tot[v].
template <bool CLUSTER>
struct Meeting {
  Slot* slots;
  double* gathered;  // [value][tile]
  int nct;
  int patience;  // polls of a wait before the solve is given up
  unsigned long long number;

  // One meeting up to the barrier after which tot is complete; true when a wait ran out. RELEASE: what a
  // CTA wrote to global memory before is visible to all CTAs after it. (The product's meeting needs no order
  // beyond its data: its sums depend on every z the CTA gathered, and the z written next depends on
  // the sums.)
  template <int NV, bool RELEASE>
  __device__ __forceinline__ bool meet(ResShared& sh, double (&v)[NV], bool row_warp) {
    ++number;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (row_warp) warp_totals_fixed<NV>(v, sh.red);
    __syncthreads();
    bool late = false;
    const int parity = (int)(number & 1);
    Slot* const box = slots + (size_t)parity * 8 * (size_t)nct;
    double a = 0.0;
    int value = NV;  // the lane's value to post
    if constexpr (kFixedWarps<NV>) {
      if (warp < NV) {
        a = add_warps_fixed(sh.red, warp);
        if (lane == 0) value = warp;
      }
    } else if (!row_warp) {
      a = add_warps<NV>(sh.red);
      if ((lane & 3) == 0) value = lane >> 2;
    }
    if constexpr (CLUSTER) {
      if (value < NV) sh.box[parity][value] = a;
    } else {
      if (RELEASE && (kFixedWarps<NV> ? warp < NV : !row_warp)) fence_gpu();
      if (value < NV) post(box + 8 * (size_t)blockIdx.x + value, a, number);
    }
    constexpr int S = kFixedTiles;
    if constexpr (CLUSTER) {
      cluster_sync_all();
    } else {
      // eight lanes take a tile's values, which share a 128-byte line: a warp to a value would ask for
      // 32 lines with each load (26 -> 28 us an iteration on 163,842 rows)
      if (row_warp) {
        using Map = PartialMap<NV>;
        double b[kLaneTiles<NV>];
        collect<NV, RELEASE>(box, nct, number, patience, b, late);
        const int val = Map::value(lane), first = Map::first(warp, lane);
        if (val < NV) {
#pragma unroll
          for (int j = 0; j < kLaneTiles<NV>; ++j)
            if (first + j * Map::kStride < S) gathered[val * S + first + j * Map::kStride] = b[j];
        }
      }
      __syncthreads();
    }
    if (warp < NV) {
      constexpr int J = CLUSTER ? 1 : S / 32;
      double x[J];
#pragma unroll
      for (int j = 0; j < J; ++j) x[j] = 0.0;
      if constexpr (CLUSTER) {
        if (lane < nct) x[0] = peer_load(&sh.box[parity][warp], lane);
      } else {
#pragma unroll
        for (int j = 0; j < J; ++j) x[j] = gathered[warp * S + 32 * j + lane];
      }
      const double b = warp_sum_fixed<J>(x);
      if (lane == 0) sh.tot[warp] = b;
    }
    return __syncthreads_or(late) != 0;
  }
};

// Four operator slots of one row: values and the gathered rows of z.
template <int K>
struct Slots4 {
  double a[4], v[4][K];
  __device__ __forceinline__ void load(const MeshDev& md, const double* sa, const int* sc, int rp, int i, int j0,
                                       int on) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < on) {
        a[u] = sa[(j0 + u) * rp + i];
        const int col = sc[(j0 + u) * rp + i];
        load_row<K>(md.z, IG_IN_RANGE(col, md.n, md.err) ? col : 0, v[u]);
      }
  }
  __device__ __forceinline__ void add_to(double (&w)[K], int j0, int on) const {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < on) {
#pragma unroll
        for (int c = 0; c < K; ++c) w[c] = fma(a[u], v[u][c], w[c]);
      }
  }
};

// The slots from the ninth on of a wide row: on chip up to `on`, the rest from global memory.
template <int K>
__device__ __forceinline__ void wide_slots(const MeshDev& md, const double* sa, const int* sc, int rp, int i, int on,
                                           int width, long row, double (&w)[K]) {
  for (int j = 8; j < on; ++j) {
    const int col = sc[j * rp + i];
    double v[K];
    load_row<K>(md.z, IG_IN_RANGE(col, md.n, md.err) ? col : 0, v);
#pragma unroll
    for (int c = 0; c < K; ++c) w[c] = fma(sa[j * rp + i], v[c], w[c]);
  }
  const long e = __ldg(md.sell_ptr + (row >> 5)) + (row & 31);
  for (int j = on; j < width; ++j) {
    const double a = __ldg(md.A + e + 32 * j);
    const int col = __ldg(md.sell_col + e + 32 * j);
    double v[K];
    load_row<K>(md.z, IG_IN_RANGE(col, md.n, md.err) ? col : 0, v);
#pragma unroll
    for (int c = 0; c < K; ++c) w[c] = fma(a, v[c], w[c]);
  }
}

// The solve by fewer CTAs than the mesh has tiles (the others had not begun in time: join_team): a CTA takes
// the tiles rank, rank + size, ... with the rows in global memory, through the tile bodies of the loop
// kernels, and adds all the tiles' sums itself. The same arithmetic and order, the same bits. Only the
// eight row warps come here. Two meetings per iteration, each after a half of the partial sums is
// complete: a half is written again only after the meeting of the other.
struct SharedScratch {  // at the start of the dynamic shared memory
  ScalSnap sn;
  double red[2][8 * kWarps];
  double tot[8];
};
static_assert(sizeof(SharedScratch) <= 128 * 4 * 8, "fits where the smallest tile's rows would be");
template <int K>
__device__ __noinline__ void solve_shared(ResShared& sh, SharedScratch& w, Slot* slots, const double* in, double* out,
                                          int rhs_mass, double tol, int max_iter, int cap, int patience) {
  const MeshDev& md = sh.md;
  const int tid = threadIdx.x, nt = md.ntiles, size = sh.team.size, rank = sh.team.rank;
  const long nn = md.n;
  double* const part_spmv = md.part;
  double* const part_update = md.part + (long)nt * kPartStride;
  unsigned long long number = sh.team.solve << 32;
  bool late = false;
  auto meet = [&]() {  // what any of the CTAs wrote before is visible to all of them after
    ++number;
    Slot* const box = slots + (size_t)(number & 1) * 8 * (size_t)nt;
    __syncthreads();
    if (tid == 0) {
      fence_gpu();
      post(box + 8 * (size_t)rank, 0.0, number);
    }
    bool mine = false;
    if (tid < size) {
      double x;
      for (int spins = 0; !peek<true>(box + 8 * (size_t)tid, number, x) && !mine; mine = ++spins > patience) {
      }
    }
    late = __syncthreads_or(mine) != 0;
    return !late;
  };
  int b = 0;
  for (int tile = rank; tile < nt; tile += size, b ^= 1) {
    const long t0 = (long)tile * md.tile_rows, t1 = t0 + md.tile_rows < nn ? t0 + md.tile_rows : nn;
    double acc[2 * K];
#pragma unroll
    for (int i = 0; i < 2 * K; ++i) acc[i] = 0.0;
    for (long row = t0 + tid; row < t1; row += kBlock) {
      const double dinv = md.Dinv[row], mass = rhs_mass ? md.M[row] : 1.0;
      double zo[K], zero[K];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        const double v = rhs_mass ? mass * in[row * K + c] : in[row * K + c];
        zo[c] = dinv * v;
        zero[c] = 0.0;
        md.x[c * nn + row] = 0.0;
        md.r[c * nn + row] = v;
        md.q[c * nn + row] = 0.0;
        acc[c] = fma(v, zo[c], acc[c]);
        acc[K + c] = fma(v, v, acc[K + c]);
      }
      store_row<K>(md.z, row, zo);
      store_row<K>(md.p, row, zero);
    }
    tile_reduce<2 * K, kFixed>(acc, w.red[b], part_update + (long)tile * kPartStride);
  }
  if (meet()) {
    combine_tiles<2 * K, kFixed>(part_update, nt, w.red[0], w.tot);
    if (tid == 0) finish_init(&sh.st, K, w.tot, tol, max_iter);
    __syncthreads();
  }
  for (int it = 0; it < cap && !late && !sh.st.done; ++it) {
    if (tid < kMaxK) w.sn.beta[tid] = sh.st.beta[tid];
    __syncthreads();
    for (int tile = rank; tile < nt; tile += size, b ^= 1)
      spmv_tile<K>(md, tile, w.sn, w.red[b], part_spmv + (long)tile * kPartStride);
    if (!meet()) break;
    combine_tiles<K, kFixed>(part_spmv, nt, w.red[0], w.tot);
    if (tid < 32) finish_spmv_step(&sh.st, sh.st, K, w.tot);
    __syncthreads();
    if (sh.st.done) break;
    if (tid < kMaxK) w.sn.alpha[tid] = sh.st.alpha[tid];
    __syncthreads();
    for (int tile = rank; tile < nt; tile += size, b ^= 1)
      update_tile<K>(md, tile, w.sn, w.red[b], part_update + (long)tile * kPartStride);
    if (!meet()) break;
    combine_tiles<2 * K, kFixed>(part_update, nt, w.red[0], w.tot);
    if (tid < 32) finish_update_step(&sh.st, sh.st, K, w.tot);
    __syncthreads();
  }
  for (int tile = rank; tile < nt; tile += size) {
    const long t0 = (long)tile * md.tile_rows, t1 = t0 + md.tile_rows < nn ? t0 + md.tile_rows : nn;
    for (long row = t0 + tid; row < t1; row += kBlock) {
#pragma unroll
      for (int c = 0; c < K; ++c) out[row * K + c] = late ? not_a_number() : md.x[c * nn + row];
    }
  }
  if (tid == 0) {
    if (late) {
      atomicOr(md.err, kErrStopped);
      sh.st.status = IG_ERR_CUDA;
      sh.st.done = 1;
    }
    sh.st.members = size;
    sh.st.off_chip = 1;
  }
  __syncthreads();
  if (rank == 0) {
    for (int j = tid; j < (int)(sizeof(SolveScal) / 4); j += kBlock)
      reinterpret_cast<unsigned*>(md.s)[j] = reinterpret_cast<const unsigned*>(&sh.st)[j];
  }
}

// The calling thread settles who takes part (in line: out of line 163,842 rows, k = 3, take 25.65 us an
// iteration instead of 24.98).
__device__ __forceinline__ void resident_join(ResShared& sh, int begin, int patience) {
  MeetHead* h = reinterpret_cast<MeetHead*>(sh.md.meet);
  sh.team = join_team(h, (int)gridDim.x, arrive(h, (int)gridDim.x), (long long)begin + patience,
                      [=](long long polls) { return polls >= begin; });
}

template <int K, bool CLUSTER>
__global__ void __launch_bounds__(kResThreads, 1) solve_resident_kernel(const MeshDev* __restrict__ mds,
                                                                        const double* __restrict__ in,
                                                                        double* __restrict__ out, int rhs_mass,
                                                                        double tol, int max_iter, int cap,
                                                                        int begin_patience, int patience,
                                                                        ResLayout lay) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ ResShared sh;
  {
    static_assert(sizeof(MeshDev) % 4 == 0 && sizeof(SolveScal) % 4 == 0, "copied as 4-byte words");
    const unsigned* src = reinterpret_cast<const unsigned*>(mds);
    for (int j = threadIdx.x; j < (int)(sizeof(MeshDev) / 4); j += kResThreads)
      reinterpret_cast<unsigned*>(&sh.md)[j] = __ldg(src + j);
    __syncthreads();
    for (int j = threadIdx.x; j < (int)(sizeof(SolveScal) / 4); j += kResThreads)
      reinterpret_cast<unsigned*>(&sh.st)[j] = __ldcg(reinterpret_cast<const unsigned*>(sh.md.s) + j);
  }
  const MeshDev& md = sh.md;
  const int tid = threadIdx.x;
  const bool row_warp = tid < kBlock;
  const long nn = md.n;
  const long t0 = (long)blockIdx.x * md.tile_rows;
  // the ninth warp has no rows
  const int rows = !row_warp ? 0 : (int)(nn - t0 < md.tile_rows ? nn - t0 : md.tile_rows);
  const int rp = lay.rp, aw = lay.aw;
  double* q = reinterpret_cast<double*>(dyn);
  double* p = q + K * rp;
  double* r = p + K * rp;
  double* dinv = r + K * rp;
  double* sa = dinv + rp;
  double* xs = sa + (size_t)aw * rp;
  double* sums = xs + (lay.x_on ? K * rp : 0);
  int* sc = reinterpret_cast<int*>(sums + 2 * K * kFixedTiles);
  double* x = lay.x_on ? xs : md.x + t0;   // component c of row i at x[c * xn + i]
  const long xn = lay.x_on ? rp : nn;
  double* z = md.z;

  // (the ninth warp, while the others load)
  if (!CLUSTER && tid == kBlock)
    resident_join(sh, begin_patience, patience);

  // the rows' operator on chip; slices of 32 rows, one per warp and step
  for (int i = tid; i < rows; i += kBlock) {
    const long row = t0 + i;
    const int sl = (int)(row >> 5);
    const int b0 = __ldg(md.sell_ptr + sl), w = (__ldg(md.sell_ptr + sl + 1) - b0) >> 5;
    if ((i & 31) == 0) sh.width[i >> 5] = w;
    const long e = b0 + (row & 31);
    for (int j = 0; j < (w < aw ? w : aw); ++j) {
      sa[j * rp + i] = __ldg(md.A + e + 32 * j);
      sc[j * rp + i] = __ldg(md.sell_col + e + 32 * j);
    }
    dinv[i] = md.Dinv[row];
  }

  Meeting<CLUSTER> mt;
  mt.slots = reinterpret_cast<Slot*>(md.meet) + 1;
  mt.gathered = sums;
  mt.nct = gridDim.x;
  mt.patience = patience;
  mt.number = 0;

  if constexpr (!CLUSTER) {
    __syncthreads();  // nothing is written to global memory before it is settled who takes part
    if (__builtin_expect(sh.team.size != (int)gridDim.x, 0)) {
      if (!row_warp || sh.team.rank >= sh.team.size) {
        if (sh.team.size < 0) {  // not settled: a failed solve
          for (int i = tid; i < rows; i += kBlock)
#pragma unroll
            for (int c = 0; c < K; ++c) out[(t0 + i) * K + c] = not_a_number();
          if (tid == 0) atomicOr(md.err, kErrStopped);
        }
        return;
      }
      solve_shared<K>(sh, *reinterpret_cast<SharedScratch*>(dyn), mt.slots, in, out, rhs_mass, tol, max_iter, cap,
                      patience);
      return;
    }
    mt.number = sh.team.solve << 32;  // above those of every solve of the mesh before
  }

  // start: rhs = M * in or in; r = rhs, z = D^-1 r, p = q = x = 0; r.z and |rhs|^2
  bool late;
  {
    double acc[2 * K];
#pragma unroll
    for (int c = 0; c < 2 * K; ++c) acc[c] = 0.0;
    for (int i = tid; i < rows; i += kBlock) {
      const long row = t0 + i;
      const double d = dinv[i];
      const double mass = rhs_mass ? md.M[row] : 1.0;
      double zo[K];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        const double b = rhs_mass ? mass * in[row * K + c] : in[row * K + c];
        zo[c] = d * b;
        x[c * xn + i] = 0.0;
        p[c * rp + i] = 0.0;
        q[c * rp + i] = 0.0;
        r[c * rp + i] = b;
        acc[c] = fma(b, zo[c], acc[c]);
        acc[K + c] = fma(b, b, acc[K + c]);
      }
      store_row<K>(z, row, zo);
    }
    late = mt.template meet<2 * K, true>(sh, acc, row_warp);
    if (tid == kBlock) finish_init(&sh.st, K, sh.tot, tol, max_iter);
  }

  for (int it = 0; it < cap && !late; ++it) {
    // p = z + beta p, q = A z + beta q, p.q. A row's product needs only z, which is there: the row
    // warps start on their first row's while the ninth warp finishes the meeting before (beta, done).
    {
      double beta[K], pq[K];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        beta[c] = 0.0;
        pq[c] = 0.0;
      }
      // The slots are taken four at a time, and the loads run ahead of the arithmetic: the second
      // four are under way while the first are added, the next row's first four while the rest of
      // this row is. Two warps share a sub-partition's FP64 unit and would otherwise wait for their
      // loads together.
      bool waiting = true;
      Slots4<K> s0, s1;
      int width = 0, on = 0;
      if ((tid & ~31) < rows) {
        width = sh.width[tid >> 5];
        on = width < aw ? width : aw;
        s0.load(md, sa, sc, rp, tid < rows ? tid : rows - 1, 0, on);
      }
      for (int i = tid; (i & ~31) < rows; i += kBlock) {  // whole warps: a barrier is inside
        const int ii = i < rows ? i : rows - 1;
        double w[K];
#pragma unroll
        for (int c = 0; c < K; ++c) w[c] = 0.0;
        double zi[K];
        s1.load(md, sa, sc, rp, ii, 4, on);
        load_row<K>(z, t0 + ii, zi);
        s0.add_to(w, 0, on);
        const int on_i = on, width_i = width, next = i + kBlock;
        if ((next & ~31) < rows) {
          width = sh.width[next >> 5];
          on = width < aw ? width : aw;
          s0.load(md, sa, sc, rp, next < rows ? next : rows - 1, 0, on);
        }
        s1.add_to(w, 4, on_i);
        if (width_i > 8 || on_i < width_i) wide_slots<K>(md, sa, sc, rp, ii, on_i, width_i, t0 + i, w);
        if (waiting) {
          waiting = false;
          __syncthreads();
          if (sh.st.done) break;
#pragma unroll
          for (int c = 0; c < K; ++c) beta[c] = sh.st.beta[c];
        }
        if (i < rows) {
#pragma unroll
          for (int c = 0; c < K; ++c) {
            const double pn = fma(beta[c], p[c * rp + i], zi[c]);
            const double qn = fma(beta[c], q[c * rp + i], w[c]);
            p[c * rp + i] = pn;
            q[c * rp + i] = qn;
            pq[c] = fma(pn, qn, pq[c]);
          }
        }
      }
      if (waiting) __syncthreads();
      if (sh.st.done) break;
      late = mt.template meet<K, false>(sh, pq, row_warp);
      if (late) break;
      if (!row_warp) finish_spmv_step(&sh.st, sh.st, K, sh.tot);
      __syncthreads();
      if (sh.st.done) break;  // a breakdown: no update, as in the multi-CTA loop
    }
    // x += alpha p, r -= alpha q, z = D^-1 r, r.z and r.r
    {
      double alpha[K], acc[2 * K];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        alpha[c] = sh.st.alpha[c];
        acc[c] = 0.0;
        acc[K + c] = 0.0;
      }
      for (int i = tid; i < rows; i += kBlock) {
        const double d = dinv[i];
        double rn[K], zo[K];
#pragma unroll
        for (int c = 0; c < K; ++c) {
          rn[c] = fma(-alpha[c], q[c * rp + i], r[c * rp + i]);
          zo[c] = d * rn[c];
          r[c * rp + i] = rn[c];
        }
        store_row<K>(z, t0 + i, zo);
#pragma unroll
        for (int c = 0; c < K; ++c) {
          x[c * xn + i] = fma(alpha[c], p[c * rp + i], x[c * xn + i]);
          acc[c] = fma(rn[c], zo[c], acc[c]);
          acc[K + c] = fma(rn[c], rn[c], acc[K + c]);
        }
      }
      late = mt.template meet<2 * K, true>(sh, acc, row_warp);
      if (late) break;
      if (!row_warp) finish_update_step(&sh.st, sh.st, K, sh.tot);
    }
  }
  for (int i = tid; i < rows; i += kBlock) {
#pragma unroll
    for (int c = 0; c < K; ++c) out[(t0 + i) * K + c] = late ? not_a_number() : x[c * xn + i];
  }
  if (late && tid == kBlock) {  // a CTA stayed away past the limit: a failed solve, for every caller to see
    atomicOr(md.err, kErrStopped);
    sh.st.status = IG_ERR_CUDA;
    sh.st.done = 1;
  }
  if (tid == 0) sh.st.members = (int)gridDim.x;
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int j = tid; j < (int)(sizeof(SolveScal) / 4); j += kResThreads)
      reinterpret_cast<unsigned*>(md.s)[j] = reinterpret_cast<const unsigned*>(&sh.st)[j];
  }
  if constexpr (CLUSTER) cluster_sync_all();  // no CTA leaves while another reads its sums
}

constexpr int kResBytes = 227 * 1024 - (int)sizeof(ResShared) - 256;  // most dynamic shared memory of a CTA

// Shared memory of a CTA of rp rows: everything, less the solution, then less operator slots, as far
// as the SM's 227 KB demand.
template <int K>
ResLayout layout(int rp, int wmax) {
  const int room = kResBytes;
  const int fixed = rp * 8 * (3 * K + 1) + 2 * K * kFixedTiles * 8;
  ResLayout l{};
  l.rp = rp;
  l.x_on = fixed + rp * 8 * K + 12 * rp * wmax <= room;
  const int left = room - fixed - (l.x_on ? rp * 8 * K : 0);
  l.aw = left / (12 * rp) < wmax ? left / (12 * rp) : wmax;
  l.bytes = fixed + (l.x_on ? rp * 8 * K : 0) + 12 * rp * l.aw;
  return l;
}

template <int K, bool CLUSTER>
bool launch_k(Group& g, const double* in, double* out, int rhs_mass, const ig_solve_opts& o, cudaStream_t st) {
  const MeshDev& md = g.host_mds[0];
  auto kern = solve_resident_kernel<K, CLUSTER>;
  const ResLayout lay = layout<K>(md.tile_rows, md.sell_wmax);
  // (the same limit whatever the mesh: it is the kernel's, and a thread with a smaller mesh could lower it
  // between another's call here and its launch)
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kResBytes) != cudaSuccess ||
      (CLUSTER && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(md.ntiles, 1, 1);
  cfg.blockDim = dim3(kResThreads, 1, 1);
  cfg.dynamicSmemBytes = lay.bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  if (CLUSTER) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = md.ntiles;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  }
  // (Not a cooperative launch: that starts as a whole, once no other work holds any SM it needs. See join_team.)
  cfg.attrs = attr;
  cfg.numAttrs = CLUSTER ? 1 : 0;
  if (CLUSTER) {
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg) != cudaSuccess || clusters < 1) {
      cudaGetLastError();
      return false;
    }
  }
  if (cudaLaunchKernelEx(&cfg, kern, (const MeshDev*)g.mds, in, out, rhs_mass, o.rel_tol, o.max_iter, o.max_iter + 2,
                         g.waits->begin, g.waits->meet, lay) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

template <int K>
bool launch(Group& g, const double* in, double* out, int rhs_mass, const ig_solve_opts& o, cudaStream_t st) {
  if (g.host_mds[0].ntiles <= kClusterTiles && launch_k<K, true>(g, in, out, rhs_mass, o, st)) return true;
  if (capturing(st)) return false;
  return launch_k<K, false>(g, in, out, rhs_mass, o, st);
}

}  // namespace

size_t meet_bytes(int parts) { return sizeof(Slot) * (1 + 2 * 8 * (size_t)parts); }

bool launch_resident(Group& g, int k, const double* in, double* out, int rhs_mass, const ig_solve_opts& o,
                     cudaStream_t st) {
  if (g.nmesh != 1 || !g.host_mds[0].resident) return false;
  switch (k) {
    case 1: return launch<1>(g, in, out, rhs_mass, o, st);
    case 2: return launch<2>(g, in, out, rhs_mass, o, st);
    case 3: return launch<3>(g, in, out, rhs_mass, o, st);
    case 4: return launch<4>(g, in, out, rhs_mass, o, st);
    default: return false;
  }
}

}  // namespace ig
