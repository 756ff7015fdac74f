// ig_resident32.cu -- the mixed-precision solve (ig_pcg_mixed.cu) of the meshes of a group in one launch,
// each mesh by a gang of CTAs that hold its rows on chip: the FP32 operator, residual, product and
// solution of a CTA's tiles stay in shared memory through the whole solve, and only p, which the
// neighbours' rows gather, and the FP64 vectors of the refinement go through global memory. The row
// arithmetic, the tiles and the order of the sums are those of the multi-CTA kernels: the same bits,
// alone and in any batch.
//
// The CTAs draw tickets; the tickets of a mesh are consecutive, the longest solves
// first, so that a CTA that is done with a mesh goes on to the next one without waiting for the rest
// of the group: a batch takes no launch, and no idle CTA, per iteration, where the multi-CTA loop took
// four launches per iteration of its slowest mesh. A CTA that draws a ticket waits for the rest of its
// gang: those CTAs are at work on meshes drawn before, and the lowest gang that is not complete always
// gets the next tickets, so every wait ends. Where CTAs have not been able to start (other kernels hold
// their SMs), a gang that is not whole in some 0.2 ms leaves its mesh to the kernel that writes the results
// (finish_gang_kernel), whose CTAs fit beside other work.
//
// A CTA holds a group of four tiles and posts their sums together. Per iteration a gang meets three
// times: for p.q, for r.z and r.r, and after p is written (see ig_meet.cuh); each meeting takes about
// 1.2 us for the exchange alone. A single mesh takes CTAs of four workers of kBlock threads, one per
// SM; a batch of small tiles takes CTAs of two workers, two per SM, so that one computes while the other
// meets.
//
// Measured: 256 icospheres of 162 to 40,962 vertices (a forward and an adjoint solve of the batch), 21
// and 23 ms in the multi-CTA loop, 11.1 and 11.4 ms here (13.3 and 13.5 with one CTA per SM and the
// meshes in order of size); a grid of 251,819 vertices 45 -> 17 us an iteration. What bounds it: the
// chain of an iteration (three meetings, their FP64 sums and divisions), then the latency of the
// gathers; the L1 data path is busy 36% of the time, DRAM not at all.
#include <algorithm>
#include <cmath>

#include "ig_meet.cuh"
#include "ig_mixed.cuh"

namespace ig {

namespace {


// Dynamic shared memory of a CTA of W workers: what GangShared leaves of an SM's 227 KB, or of half of
// them.
template <int W>
constexpr int kGangBytes = W == 4 ? 222 * 1024 : 108 * 1024;

// Operator slots per row that fit on chip beside three K-vectors and the preconditioner.
__host__ __device__ inline int gang_slots(int bytes, int rows, int k, int wmax) {
  const int fit = (bytes / rows - 4 * (3 * k + 1)) / 8;
  return fit < wmax ? fit : wmax;
}

struct GangShared {
  MeshDev md;
  SolveScal st;
  double red[4][8 * kWarps];               // warp totals of the four tiles
  double red2[8 * kWarps];
  double tot[8];
  float alpha[kMaxK], beta[kMaxK];         // as floats (a conversion in every warp costs FP64 issue)
  int ticket;
  Team team;                               // whether the mesh's gang is whole
  int groups, member;                      // the mesh's groups of four tiles, and this CTA's
  int width[kGangMaxRows / 32];
};

struct GangRows {  // what a CTA holds of its mesh, in dynamic shared memory
  int rp;          // rows held (a multiple of 32)
  int aw;          // operator slots per row on chip; a wider slice's further slots are read from global memory
  float *a, *r, *x, *q, *d;
  int* c;
};

struct Gang {
  Slot* slots;
  int member, nct;     // this CTA and the CTAs of the whole gang: as many as the mesh has groups of four tiles
  unsigned long long number;
  int patience;        // polls before a wait is given up

  __device__ __forceinline__ Slot* buffer() const { return slots + (number & 1) * (8 * (size_t)nct); }

  // A meeting for sums. First those of this CTA's four tiles (warp totals in sh.red) are posted ...
  template <int NV>
  __device__ __forceinline__ void post_sums(GangShared& sh) {
    ++number;
    post_group<NV>(sh, member);
  }
  template <int NV>
  __device__ __forceinline__ void post_group(GangShared& sh, int group) const {
    const int lane = threadIdx.x & 31;
    __syncthreads();
    if (threadIdx.x < 32) {  // lane = value * 4 + tile, then over the four tiles
      const int v = lane >> 2, t = lane & 3;
      double s = v < NV ? add_warps_of<kGroups>(&sh.red[t][v * kWarps]) : 0.0;
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (t == 0 && v < NV) post(buffer() + 8 * (size_t)group + v, s, number);
    }
  }
  // ... then all groups' are collected: the mesh's totals are in sh.tot on warp 0. False in every
  // thread when a wait ran out.
  template <int NV>
  __device__ __forceinline__ bool collect_sums(GangShared& sh) {
    const int warp = threadIdx.x >> 5;
    bool late = false;
    if (warp < kWarps)
      PartialMap<NV>::to_warp_total(collect_sum<NV, false>(buffer(), nct, number, patience, late), sh.red2);
    if (__syncthreads_or(late)) return false;
    if (warp == 0) {
      add_warps_to<NV>(sh.red2, sh.tot);
      __syncwarp();
    }
    return true;
  }

  // A meeting without values: what any CTA of the gang wrote to global memory before is visible to
  // all of them after. False in every thread when a wait ran out.
  __device__ __forceinline__ bool meet_writes() { return meet_writes(member, nct); }
  __device__ __forceinline__ bool meet_writes(int rank, int size) {
    ++number;
    __syncthreads();
    if (threadIdx.x == 0) {
      fence_gpu();
      post(buffer() + 8 * (size_t)rank, 0.0, number);
    }
    bool late = false;
    if ((int)threadIdx.x < size) {
      const Slot* theirs = buffer() + 8 * (size_t)threadIdx.x;
      double x;
      for (int spins = 0; !peek<true>(theirs, number, x) && !late; late = ++spins > patience) {
      }
    }
    return __syncthreads_or(late) == 0;
  }
};

// Tile i of a CTA's four, and its rows.
struct GangTile {
  int tile, t0, rows, local;  // rows t0 .. t0 + rows of the mesh, local .. of the CTA
};
__device__ __forceinline__ GangTile gang_tile(const MeshDev& md, int member, int i) {
  GangTile g;
  g.tile = 4 * member + i;
  g.local = i * md.tile_rows32;
  g.t0 = g.tile * md.tile_rows32;
  g.rows = g.tile < md.ntiles32 ? min(md.tile_rows32, md.n - g.t0) : 0;
  return g;
}

// One slot's loop of a mesh's solve by its gang: see ig_pcg_mixed.cu for the phases.
template <int K, int W>
__device__ __forceinline__ bool gang_solve(GangShared& sh, const GangRows& gr, Gang& gang, int cap) {
  const MeshDev& md = sh.md;
  const int worker = threadIdx.x / kBlock, tid = threadIdx.x % kBlock, warp = tid >> 5, lane = tid & 31;
  const int n = md.n, rp = gr.rp;
  const long nn = n;
  float* p = as_global(md.p32);
  double* x64 = as_global(md.x);
  double* r64 = as_global(md.r);

  for (int it = 0; it < cap && !sh.st.done; ++it) {
    if (sh.st.phase == kPhaseApply) {
      // r64 = rhs - A x64 and its norms, once every CTA's x64 is there; the sums in tile order
      if (!gang.meet_writes()) return false;
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        double acc[K];
#pragma unroll
        for (int c = 0; c < K; ++c) acc[c] = 0.0;
        for (int o = tid; o < t.rows; o += kBlock) {
          const long row = t.t0 + o;
          double ax[K];
          if (md.geom32) row_product<K>(md, md.A32, row, GatherSoA64<K>{md.x, nn}, ax);
          else row_product<K>(md, md.A, row, GatherSoA64<K>{md.x, nn}, ax);
#pragma unroll
          for (int c = 0; c < K; ++c) {
            const double res = md.rhs[c * nn + row] - ax[c];
            r64[c * nn + row] = res;
            acc[c] = fma(res, res, acc[c]);
          }
        }
        const double w = warp_sum_transposed<K>(acc, lane);
        const int idx = warp_sum_index<K>(lane);
        if (warp_sum_writer<K>(lane) && idx < K) sh.red[i4][idx * kWarps + warp] = w;
      }
      __syncthreads();
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        if (tid < K && t.rows > 0)
          __stcg(md.part + (long)t.tile * kPartStride + tid, add_warps_of<kInOrder>(&sh.red[i4][tid * kWarps]));
      }
      if (!gang.meet_writes()) return false;
      double v[K];
      if (worker == 0) {
        gather_in_order<K>(md.part, md.ntiles32, v);
        warp_totals<K>(v, sh.red2);
      }
      __syncthreads();
      if (threadIdx.x < 32) {
        if (threadIdx.x < K) sh.tot[threadIdx.x] = add_warps_of<kInOrder>(sh.red2 + threadIdx.x * kWarps);
        __syncwarp();
        finish_residual(&sh.st, sh.st, K, sh.tot);
      }
      __syncthreads();
      if (sh.st.done) break;
    }
    if (sh.st.phase == kPhaseInner) {
      // q = A p and p.q
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        float pq[K];
#pragma unroll
        for (int c = 0; c < K; ++c) pq[c] = 0.f;
        for (int o = tid; o < t.rows; o += kBlock) {
          const int i = t.local + o, row = t.t0 + o;
          const int width = sh.width[i >> 5], on = width < gr.aw ? width : gr.aw;
          float q[K];
#pragma unroll
          for (int c = 0; c < K; ++c) q[c] = 0.f;
          for (int j0 = 0; j0 < on; j0 += 4) {
            float v[4][K];
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (j0 + u < on) {
                const int col = gr.c[(j0 + u) * rp + i];
                load_row32<K>(p, IG_IN_RANGE(col, n, md.err) ? col : 0, v[u]);
              }
#pragma unroll
            for (int u = 0; u < 4; ++u)
              if (j0 + u < on) {
                const float a = gr.a[(j0 + u) * rp + i];
#pragma unroll
                for (int c = 0; c < K; ++c) q[c] = fmaf(a, v[u][c], q[c]);
              }
          }
          if (on < width) {  // slots that did not fit on chip
            const long e = __ldg(md.sell_ptr + (row >> 5)) + (row & 31);
            for (int j = on; j < width; ++j) {
              const float a = __ldg(md.A32 + e + 32 * j);
              const int col = __ldg(md.sell_col + e + 32 * j);
              float v[K];
              load_row32<K>(p, IG_IN_RANGE(col, n, md.err) ? col : 0, v);
#pragma unroll
              for (int c = 0; c < K; ++c) q[c] = fmaf(a, v[c], q[c]);
            }
          }
          float pi[K];
          load_row32<K>(p, row, pi);
#pragma unroll
          for (int c = 0; c < K; ++c) {
            gr.q[c * rp + i] = q[c];
            pq[c] = fmaf(pi[c], q[c], pq[c]);
          }
        }
        const float w = warp_sum_transposed<K>(pq, lane);
        const int idx = warp_sum_index<K>(lane);
        if (warp_sum_writer<K>(lane) && idx < K) sh.red[i4][idx * kWarps + warp] = to_double(w);
      }
      gang.post_sums<K>(sh);
      if (!gang.collect_sums<K>(sh)) return false;
      if (threadIdx.x < 32) {
        finish_spmv_step(&sh.st, sh.st, K, sh.tot);
        if (threadIdx.x < K) sh.alpha[threadIdx.x] = f64_to_f32_rn(sh.st.alpha[threadIdx.x]);
      }
      __syncthreads();
      if (sh.st.done) break;
    }
    // Inner: r -= alpha q; Restart: r = r64 / ||r64||, x = 0; r.z and r.r
    const bool inner = sh.st.phase == kPhaseInner;
    {
      float alpha[K];
      double inv[K];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        alpha[c] = sh.alpha[c];
        inv[c] = inner ? 0.0 : 1.0 / sh.st.scale[c];
      }
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        float acc[2 * K];
#pragma unroll
        for (int i = 0; i < 2 * K; ++i) acc[i] = 0.f;
        for (int o = tid; o < t.rows; o += kBlock) {
          const int i = t.local + o;
          const float d = gr.d[i];
#pragma unroll
          for (int c = 0; c < K; ++c) {
            float rv;
            if (inner) {
              rv = fmaf(-alpha[c], gr.q[c * rp + i], gr.r[c * rp + i]);
            } else {
              rv = sh.st.active64[c] ? (float)(r64[c * nn + t.t0 + o] * inv[c]) : 0.f;
              gr.x[c * rp + i] = 0.f;
            }
            gr.r[c * rp + i] = rv;
            acc[c] = fmaf(rv, d * rv, acc[c]);
            acc[K + c] = fmaf(rv, rv, acc[K + c]);
          }
        }
        const float w = warp_sum_transposed<2 * K>(acc, lane);
        const int idx = warp_sum_index<2 * K>(lane);
        if (warp_sum_writer<2 * K>(lane) && idx < 2 * K) sh.red[i4][idx * kWarps + warp] = to_double(w);
      }
    }
    gang.post_sums<2 * K>(sh);
    if (inner) {
      // x += alpha p while the sums are on their way
      float alpha[K];
#pragma unroll
      for (int c = 0; c < K; ++c) alpha[c] = sh.alpha[c];
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        for (int o = tid; o < t.rows; o += kBlock) {
          float pi[K];
          load_row32<K>(p, t.t0 + o, pi);
#pragma unroll
          for (int c = 0; c < K; ++c) {
            float* x = gr.x + c * rp + t.local + o;
            *x = fmaf(alpha[c], pi[c], *x);
          }
        }
      }
    }
    if (!gang.collect_sums<2 * K>(sh)) return false;
    if (threadIdx.x < 32) {
      if (inner) finish_update_mixed_step(&sh.st, sh.st, K, sh.tot);
      else finish_restart_step(&sh.st, sh.st, K, sh.tot);
      if (threadIdx.x < K) sh.beta[threadIdx.x] = f64_to_f32_rn(sh.st.beta[threadIdx.x]);
    }
    __syncthreads();
    if (sh.st.done) break;
    if (sh.st.phase == kPhaseInner) {
      // p = D^-1 r + beta p
      float beta[K];
#pragma unroll
      for (int c = 0; c < K; ++c) beta[c] = sh.beta[c];
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        for (int o = tid; o < t.rows; o += kBlock) {
          const int i = t.local + o;
          float pi[K];
          load_row32<K>(p, t.t0 + o, pi);
          const float d = gr.d[i];
#pragma unroll
          for (int c = 0; c < K; ++c) pi[c] = fmaf(beta[c], pi[c], d * gr.r[c * rp + i]);
          store_row32<K>(p, t.t0 + o, pi);
        }
      }
      if (!gang.meet_writes()) return false;
    } else {
      // x64 += ||r64|| x
      double sc[K];
#pragma unroll
      for (int c = 0; c < K; ++c) sc[c] = sh.st.scale[c];
      for (int i4 = worker; i4 < 4; i4 += W) {
        const GangTile t = gang_tile(md, gang.member, i4);
        for (int o = tid; o < t.rows; o += kBlock) {
          const long row = t.t0 + o;
#pragma unroll
          for (int c = 0; c < K; ++c)
            x64[c * nn + row] = fma(sc[c], (double)gr.x[c * rp + t.local + o], x64[c * nn + row]);
        }
      }
    }
  }
  return true;
}

// The calling thread waits for the rest of the gang of the CTA's mesh: CTAs at work on meshes drawn before for
// as long as such a solve takes, but not those that have not been able to start. (Out of line, like
// gang_failed: the loop has all the registers.)
__device__ __noinline__ void gang_join(GangShared& sh, Arrival a, const unsigned* started, unsigned ctas, int begin,
                                       int patience, long long longest) {
  sh.team = join_team<true>(reinterpret_cast<MeetHead*>(sh.md.meet), sh.groups, a, longest + patience,
                            [=](long long polls) {
                              return polls >= longest || (polls >= begin && __ldcg(started) < ctas);
                            });
}
// A wait ran out: a failed solve, for every caller to see.
template <int K>
__device__ __noinline__ void gang_failed(GangShared& sh) {
  const MeshDev& md = sh.md;
  const int first = 4 * sh.member * md.tile_rows32;
  for (int i = first + threadIdx.x; i < md.n && i < first + 4 * md.tile_rows32; i += blockDim.x)
#pragma unroll
    for (int c = 0; c < K; ++c) md.x[(long)c * md.n + i] = not_a_number();
  if (threadIdx.x == 0) {
    atomicOr(md.err, kErrStopped);
    sh.st.status = IG_ERR_CUDA;
    sh.st.done = 1;
  }
}

template <int K, int W>
__global__ void __launch_bounds__(W * kBlock, W == 4 ? 1 : 2) solve_gang_kernel(const MeshDev* __restrict__ mds,
                                                                                const int4* __restrict__ plan, int nplan,
                                                                                int tickets, unsigned* ticket, int cap,
                                                                                int begin, int patience,
                                                                                long long longest) {
  constexpr int kGangThreads = W * kBlock;
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ GangShared sh;
  // ticket[0]: the next ticket, [1]: CTAs of the launch that have started, [2]: a mesh is left to finish_gang_kernel
  if (threadIdx.x == 0) atomicAdd(ticket + 1, 1u);
  for (;;) {
    __syncthreads();  // every thread is done with the mesh before
    if (threadIdx.x == 0) sh.ticket = (int)atomicAdd(ticket, 1u);
    __syncthreads();
    if (sh.ticket >= tickets) return;
    int lo = 0, hi = nplan - 1;  // the last entry whose first ticket is not above this one
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(&plan[mid].y) <= sh.ticket) lo = mid;
      else hi = mid - 1;
    }
    const int4 e = __ldg(plan + lo);  // mesh, first ticket, CTAs
    if (threadIdx.x == 0) {
      sh.groups = e.z;
      sh.member = sh.ticket - e.y;
    }
    for (int j = threadIdx.x; j < (int)(sizeof(MeshDev) / 4); j += kGangThreads)
      reinterpret_cast<unsigned*>(&sh.md)[j] = __ldg(reinterpret_cast<const unsigned*>(mds + e.x) + j);
    __syncthreads();
    const MeshDev& md = sh.md;
    for (int j = threadIdx.x; j < (int)(sizeof(SolveScal) / 4); j += kGangThreads)
      reinterpret_cast<unsigned*>(&sh.st)[j] = __ldcg(reinterpret_cast<const unsigned*>(md.s) + j);
    Gang gang;
    gang.member = sh.ticket - e.y;
    gang.nct = e.z;
    gang.slots = reinterpret_cast<Slot*>(md.meet) + 1;
    gang.patience = patience;
    Arrival arrival{};
    if (threadIdx.x == kGangThreads - 32) arrival = arrive(reinterpret_cast<MeetHead*>(md.meet), gang.nct);

    // the rows on chip
    GangRows gr;
    const int first_row = 4 * gang.member * md.tile_rows32;
    gr.rp = 4 * md.tile_rows32;
    const int held = min(gr.rp, md.n - first_row);
    gr.aw = gang_slots(kGangBytes<W>, gr.rp, K, md.sell_wmax);
    gr.r = reinterpret_cast<float*>(dyn);
    gr.x = gr.r + K * gr.rp;
    gr.q = gr.x + K * gr.rp;
    gr.d = gr.q + K * gr.rp;
    gr.a = gr.d + gr.rp;
    gr.c = reinterpret_cast<int*>(gr.a + gr.aw * gr.rp);
    for (int i = threadIdx.x; i < held; i += kGangThreads) {
      const int row = first_row + i, sl = row >> 5;
      const int b0 = __ldg(md.sell_ptr + sl), w = (__ldg(md.sell_ptr + sl + 1) - b0) >> 5;
      if ((i & 31) == 0) sh.width[i >> 5] = w;
      const int at = b0 + (row & 31);
      for (int j = 0; j < (w < gr.aw ? w : gr.aw); ++j) {
        gr.a[j * gr.rp + i] = __ldg(md.A32 + at + 32 * j);
        gr.c[j * gr.rp + i] = __ldg(md.sell_col + at + 32 * j);
      }
      gr.d[i] = __ldg(md.Dinv32 + row);
    }
    if (threadIdx.x == kGangThreads - 32) gang_join(sh, arrival, ticket + 1, gridDim.x, begin, patience, longest);
    __syncthreads();
    if (sh.team.size == 0) {  // left to finish_gang_kernel
      if (threadIdx.x == 0) {
        md.s->off_chip = 1;
        ticket[2] = 1u;
      }
      continue;
    }
    gang.number = sh.team.solve << 32;  // above those of every solve of the mesh before

    const bool met = sh.team.size > 0 && gang_solve<K, W>(sh, gr, gang, cap);
    __syncthreads();
    if (!met) gang_failed<K>(sh);
    if (gang.member == 0) {
      if (threadIdx.x == 0) sh.st.members = gang.nct;
      __syncthreads();
      for (int j = threadIdx.x; j < (int)(sizeof(SolveScal) / 4); j += kGangThreads)
        reinterpret_cast<unsigned*>(md.s)[j] = reinterpret_cast<const unsigned*>(&sh.st)[j];
    }
  }
}

// After the gangs: the solutions written to io.out, and the meshes whose gang was not whole in time solved (CTAs
// could not start: other work held their SMs; some 0.2 ms are waited for that). The CTAs of such a mesh's
// tiles need little of an SM; those that have begun share the solve, group by group of four tiles (rank,
// rank + size, ...) with the rows in global memory, in the arithmetic and order of gang_solve: the same bits.
template <int K>
__device__ __noinline__ bool gang_solve_shared(GangShared& sh, int cap, int patience) {
  const MeshDev& md = sh.md;
  const int rank = sh.team.rank, size = sh.team.size, groups = sh.groups;
  Gang gang{reinterpret_cast<Slot*>(md.meet) + 1, rank, groups, sh.team.solve << 32, patience};
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = md.n;
  const long nn = n;
  float *r32 = as_global(md.r32), *x32 = as_global(md.x32), *q32 = as_global(md.q32);
  const float* d32 = as_global(md.Dinv32);
  float* p = as_global(md.p32);
  double* x64 = as_global(md.x);
  double* r64 = as_global(md.r);

  for (int it = 0; it < cap && !sh.st.done; ++it) {
    if (sh.st.phase == kPhaseApply) {
      // r64 = rhs - A x64 and its norms, once every CTA's x64 is there; the sums in tile order
      if (!gang.meet_writes(rank, size)) return false;
      for (int g = rank; g < groups; g += size) {
        __syncthreads();  // the group before has been added
        for (int i4 = 0; i4 < 4; ++i4) {
          const GangTile t = gang_tile(md, g, i4);
          double acc[K];
#pragma unroll
          for (int c = 0; c < K; ++c) acc[c] = 0.0;
          for (int o = tid; o < t.rows; o += kBlock) {
            const long row = t.t0 + o;
            double ax[K];
            if (md.geom32) row_product<K>(md, md.A32, row, GatherSoA64<K>{md.x, nn}, ax);
            else row_product<K>(md, md.A, row, GatherSoA64<K>{md.x, nn}, ax);
#pragma unroll
            for (int c = 0; c < K; ++c) {
              const double res = md.rhs[c * nn + row] - ax[c];
              r64[c * nn + row] = res;
              acc[c] = fma(res, res, acc[c]);
            }
          }
          const double w = warp_sum_transposed<K>(acc, lane);
          const int idx = warp_sum_index<K>(lane);
          if (warp_sum_writer<K>(lane) && idx < K) sh.red[i4][idx * kWarps + warp] = w;
        }
        __syncthreads();
        for (int i4 = 0; i4 < 4; ++i4) {
          const GangTile t = gang_tile(md, g, i4);
          if (tid < K && t.rows > 0)
            __stcg(md.part + (long)t.tile * kPartStride + tid, add_warps_of<kInOrder>(&sh.red[i4][tid * kWarps]));
        }
      }
      if (!gang.meet_writes(rank, size)) return false;
      double v[K];
      gather_in_order<K>(md.part, md.ntiles32, v);
      warp_totals<K>(v, sh.red2);
      __syncthreads();
      if (threadIdx.x < 32) {
        if (threadIdx.x < K) sh.tot[threadIdx.x] = add_warps_of<kInOrder>(sh.red2 + threadIdx.x * kWarps);
        __syncwarp();
        finish_residual(&sh.st, sh.st, K, sh.tot);
      }
      __syncthreads();
      if (sh.st.done) break;
    }
    if (sh.st.phase == kPhaseInner) {
      // q = A p and p.q
      ++gang.number;
      for (int g = rank; g < groups; g += size) {
        __syncthreads();  // the group before has been added
        for (int i4 = 0; i4 < 4; ++i4) {
          const GangTile t = gang_tile(md, g, i4);
          float pq[K];
#pragma unroll
          for (int c = 0; c < K; ++c) pq[c] = 0.f;
          for (int o = tid; o < t.rows; o += kBlock) {
            const int row = t.t0 + o, b0 = __ldg(md.sell_ptr + (row >> 5));
            const int width = (__ldg(md.sell_ptr + (row >> 5) + 1) - b0) >> 5;
            const long e = b0 + (row & 31);
            float q[K];
#pragma unroll
            for (int c = 0; c < K; ++c) q[c] = 0.f;
            for (int j = 0; j < width; ++j) {
              const float a = __ldg(md.A32 + e + 32 * j);
              const int col = __ldg(md.sell_col + e + 32 * j);
              float v[K];
              load_row32<K>(p, IG_IN_RANGE(col, n, md.err) ? col : 0, v);
#pragma unroll
              for (int c = 0; c < K; ++c) q[c] = fmaf(a, v[c], q[c]);
            }
            float pi[K];
            load_row32<K>(p, row, pi);
#pragma unroll
            for (int c = 0; c < K; ++c) {
              q32[c * nn + row] = q[c];
              pq[c] = fmaf(pi[c], q[c], pq[c]);
            }
          }
          const float w = warp_sum_transposed<K>(pq, lane);
          const int idx = warp_sum_index<K>(lane);
          if (warp_sum_writer<K>(lane) && idx < K) sh.red[i4][idx * kWarps + warp] = to_double(w);
        }
        gang.template post_group<K>(sh, g);
      }
      if (!gang.template collect_sums<K>(sh)) return false;
      if (threadIdx.x < 32) {
        finish_spmv_step(&sh.st, sh.st, K, sh.tot);
        if (threadIdx.x < K) sh.alpha[threadIdx.x] = f64_to_f32_rn(sh.st.alpha[threadIdx.x]);
      }
      __syncthreads();
      if (sh.st.done) break;
    }
    // Inner: r -= alpha q; Restart: r = r64 / ||r64||, x = 0; r.z and r.r
    const bool inner = sh.st.phase == kPhaseInner;
    ++gang.number;
    for (int g = rank; g < groups; g += size) {
      __syncthreads();  // the group before has been added
      float alpha[K];
      double inv[K];
#pragma unroll
      for (int c = 0; c < K; ++c) {
        alpha[c] = sh.alpha[c];
        inv[c] = inner ? 0.0 : 1.0 / sh.st.scale[c];
      }
      for (int i4 = 0; i4 < 4; ++i4) {
        const GangTile t = gang_tile(md, g, i4);
        float acc[2 * K];
#pragma unroll
        for (int i = 0; i < 2 * K; ++i) acc[i] = 0.f;
        for (int o = tid; o < t.rows; o += kBlock) {
          const int i = t.t0 + o;
          const float d = d32[i];
#pragma unroll
          for (int c = 0; c < K; ++c) {
            float rv;
            if (inner) {
              rv = fmaf(-alpha[c], q32[c * nn + i], r32[c * nn + i]);
            } else {
              rv = sh.st.active64[c] ? (float)(r64[c * nn + i] * inv[c]) : 0.f;
              x32[c * nn + i] = 0.f;
            }
            r32[c * nn + i] = rv;
            acc[c] = fmaf(rv, d * rv, acc[c]);
            acc[K + c] = fmaf(rv, rv, acc[K + c]);
          }
        }
        const float w = warp_sum_transposed<2 * K>(acc, lane);
        const int idx = warp_sum_index<2 * K>(lane);
        if (warp_sum_writer<2 * K>(lane) && idx < 2 * K) sh.red[i4][idx * kWarps + warp] = to_double(w);
      }
      gang.template post_group<2 * K>(sh, g);
    }
    if (inner) {
      // x += alpha p while the sums are on their way
      float alpha[K];
#pragma unroll
      for (int c = 0; c < K; ++c) alpha[c] = sh.alpha[c];
      for (int g = rank; g < groups; g += size) {
        for (int i4 = 0; i4 < 4; ++i4) {
          const GangTile t = gang_tile(md, g, i4);
          for (int o = tid; o < t.rows; o += kBlock) {
            float pi[K];
            load_row32<K>(p, t.t0 + o, pi);
#pragma unroll
            for (int c = 0; c < K; ++c) {
              float* x = x32 + c * nn + t.t0 + o;
              *x = fmaf(alpha[c], pi[c], *x);
            }
          }
        }
      }
    }
    if (!gang.template collect_sums<2 * K>(sh)) return false;
    if (threadIdx.x < 32) {
      if (inner) finish_update_mixed_step(&sh.st, sh.st, K, sh.tot);
      else finish_restart_step(&sh.st, sh.st, K, sh.tot);
      if (threadIdx.x < K) sh.beta[threadIdx.x] = f64_to_f32_rn(sh.st.beta[threadIdx.x]);
    }
    __syncthreads();
    if (sh.st.done) break;
    if (sh.st.phase == kPhaseInner) {
      // p = D^-1 r + beta p
      float beta[K];
#pragma unroll
      for (int c = 0; c < K; ++c) beta[c] = sh.beta[c];
      for (int g = rank; g < groups; g += size) {
        for (int i4 = 0; i4 < 4; ++i4) {
          const GangTile t = gang_tile(md, g, i4);
          for (int o = tid; o < t.rows; o += kBlock) {
            const int i = t.t0 + o;
            float pi[K];
            load_row32<K>(p, i, pi);
            const float d = d32[i];
#pragma unroll
            for (int c = 0; c < K; ++c) pi[c] = fmaf(beta[c], pi[c], d * r32[c * nn + i]);
            store_row32<K>(p, i, pi);
          }
        }
      }
      if (!gang.meet_writes(rank, size)) return false;
    } else {
      // x64 += ||r64|| x
      double sc[K];
#pragma unroll
      for (int c = 0; c < K; ++c) sc[c] = sh.st.scale[c];
      for (int g = rank; g < groups; g += size) {
        for (int i4 = 0; i4 < 4; ++i4) {
          const GangTile t = gang_tile(md, g, i4);
          for (int o = tid; o < t.rows; o += kBlock) {
            const long row = t.t0 + o;
#pragma unroll
            for (int c = 0; c < K; ++c)
              x64[c * nn + row] = fma(sc[c], (double)x32[c * nn + row], x64[c * nn + row]);
          }
        }
      }
    }
  }
  return true;
}

template <int K>
__global__ void __launch_bounds__(kBlock) finish_gang_kernel(const MeshDev* __restrict__ mds,
                                                             const int2* __restrict__ tiles, IoTable io, int cap,
                                                             int begin, int patience,
                                                             const unsigned* __restrict__ left) {
  const unsigned any = __ldcg(left);  // whether some mesh is left (beside the loads that follow)
  const int2 tl = tiles[blockIdx.x];
  const MeshDev& gmd = mds[tl.x];
  const long nn = gmd.n;
  double* __restrict__ out = io.out[tl.x];
  if (any == 0u || !gmd.s->off_chip) {
    const long t0 = (long)tl.y * gmd.tile_rows, t1 = t0 + gmd.tile_rows < nn ? t0 + gmd.tile_rows : nn;
    for (long row = t0 + threadIdx.x; row < t1; row += kBlock) {
#pragma unroll
      for (int c = 0; c < K; ++c) out[row * K + c] = gmd.x[c * nn + row];
    }
    return;
  }
  __shared__ GangShared sh;
  const int groups = (gmd.ntiles32 + 3) / 4, count = gmd.ntiles < groups ? gmd.ntiles : groups;
  if (tl.y >= count) return;
  for (int j = threadIdx.x; j < (int)(sizeof(MeshDev) / 4); j += kBlock)
    reinterpret_cast<unsigned*>(&sh.md)[j] = __ldg(reinterpret_cast<const unsigned*>(mds + tl.x) + j);
  for (int j = threadIdx.x; j < (int)(sizeof(SolveScal) / 4); j += kBlock)
    reinterpret_cast<unsigned*>(&sh.st)[j] = __ldcg(reinterpret_cast<const unsigned*>(gmd.s) + j);
  if (threadIdx.x == 0) {
    sh.groups = groups;
    MeetHead* h = reinterpret_cast<MeetHead*>(gmd.meet);
    sh.team = join_team(h, count, arrive(h, count), (long long)begin + patience,
                        [&](long long polls) { return polls >= begin; });
  }
  __syncthreads();
  const int rank = sh.team.rank, size = sh.team.size;
  if (size >= 0 && rank >= size) return;  // settled without this CTA
  const bool met = size > 0 && gang_solve_shared<K>(sh, cap, patience);
  __syncthreads();
  const int rows = 4 * gmd.tile_rows32;
  for (int g = size > 0 ? rank : tl.y; g < groups; g += size > 0 ? size : count)
    for (long i = (long)g * rows + threadIdx.x; i < nn && i < (long)(g + 1) * rows; i += kBlock) {
#pragma unroll
      for (int c = 0; c < K; ++c) out[i * K + c] = met ? gmd.x[c * nn + i] : not_a_number();
    }
  if (threadIdx.x == 0) {
    sh.st.members = size;
    if (!met) {
      atomicOr(gmd.err, kErrStopped);
      sh.st.status = IG_ERR_CUDA;
      sh.st.done = 1;
    }
  }
  __syncthreads();
  if (rank == 0)
    for (int j = threadIdx.x; j < (int)(sizeof(SolveScal) / 4); j += kBlock)
      reinterpret_cast<unsigned*>(gmd.s)[j] = reinterpret_cast<const unsigned*>(&sh.st)[j];
}

// (1 KB of an SM's shared memory is the system's for each CTA)
static_assert(sizeof(GangShared) <= 4 * 1024, "shared memory of a gang CTA");

template <int K, int W>
bool launch_w(Group& g, int cap, cudaStream_t st) {
  auto kern = solve_gang_kernel<K, W>;
  const int ctas = g.num_sms * (W == 4 ? 1 : 2);
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGangBytes<W>) != cudaSuccess ||
      cudaMemsetAsync(g.gang_ticket, 0, 3 * sizeof(unsigned), st) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g.gang_tickets < ctas ? g.gang_tickets : ctas, 1, 1);
  cfg.blockDim = dim3(W * kBlock, 1, 1);
  cfg.dynamicSmemBytes = kGangBytes<W>;
  cfg.stream = st;
  // a wait for the rest of a gang lasts as long as the solve of a mesh drawn before
  const long long longest = g.waits->meet + (g.waits->meet == WaitLimits{}.meet ? 256ll * cap : 0ll);
  if (cudaLaunchKernelEx(&cfg, kern, (const MeshDev*)g.mds, (const int4*)g.gang_plan, g.nmesh, g.gang_tickets,
                         g.gang_ticket, cap, g.waits->begin, g.waits->meet, longest) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

template <int K>
bool launch(Group& g, int cap, const IoTable& io, cudaStream_t st, cudaError_t& e) {
  if (!(g.gang_workers == 2 ? launch_w<K, 2>(g, cap, st) : launch_w<K, 4>(g, cap, st))) return false;
  finish_gang_kernel<K><<<g.ntiles, kBlock, 0, st>>>(g.mds, g.tiles, io, cap, g.waits->begin, g.waits->meet,
                                                   g.gang_ticket + 2);
  e = cudaGetLastError();
  return true;
}

}  // namespace

// The gangs of a group: mesh, first ticket, CTAs; empty when some mesh is too large. The meshes with the
// longest solves come first, so that none of them is still running when the rest is done: iterations
// grow with the square root of the time step over the squared edge length, that is of t n on meshes of
// one size (t null: equal steps). CTAs of two workers (two per SM) when there are more of them than
// SMs and their tiles are small enough.
//
// Empty too for batches that the multi-CTA loop solves sooner. A CTA of four workers has an SM to itself, and
// gangs of more than half the SMs run one after another, so the chain of an iteration (some 12.5 us in any
// gang) is not hidden: n gangs at a time take 12.5 / n us an iteration and mesh, the loop 40 us an
// iteration and 40 us per million rows (fitted to 102 batches, leaning to the gangs; weights: iterations as
// the square root of the rows). 163,842 rows each, k = 3: 4 meshes 5.6 ms in gangs and 6.4 in the loop, 8
// 11.2 and 10.7, 16 22.2 and 19.6; one of these and 40 of 40,962 rows 10.9 and 9.5; of 250,000 rows each, 8
// 7.0 and 7.9, 32 27.7 and 25.7. In CTAs of two workers no batch was slower than in the loop by more than 2%.
std::vector<int4> gang_plan(const MeshDev* mds, const double* t, int nmesh, int num_sms, int* tickets, int* workers) {
  std::vector<int4> plan;
  std::vector<double> work((size_t)nmesh);
  int rows = 0;
  for (int i = 0; i < nmesh; ++i) {
    const int g = (mds[i].ntiles32 + 3) / 4;
    if (!mds[i].meet || g > num_sms || g > kResMaxCtas || 4 * mds[i].tile_rows32 > kGangMaxRows) return {};
    rows = std::max(rows, 4 * mds[i].tile_rows32);
    work[(size_t)i] = (t ? t[i] : 1.0) * mds[i].n;
    plan.push_back(make_int4(i, 0, g, 0));
  }
  std::stable_sort(plan.begin(), plan.end(),
                   [&work](const int4& a, const int4& b) { return work[(size_t)a.x] > work[(size_t)b.x]; });
  int first = 0;
  for (int4& e : plan) {
    e.y = first;
    first += e.z;
  }
  *tickets = first;
  *workers = first > num_sms && rows <= kGangMaxRows / 2 - 32 ? 2 : 4;
  if (first > num_sms && *workers == 4) {
    int most = 1;
    for (int i = 0; i < nmesh; ++i) most = std::max(most, mds[i].n);
    double gangs = 0.0, loop = 40.0;  // us per iteration of the largest mesh
    for (const int4& e : plan) {
      const double n = mds[e.x].n, w = std::sqrt(n / most);
      gangs += w * 12.5 / (num_sms / e.z);
      loop += w * 40.0 * 1e-6 * n;
    }
    if (gangs > loop) return {};
  }
  return plan;
}

bool launch_gang(Group& g, int k, int cap, const IoTable& io, cudaStream_t st, cudaError_t& e) {
  if (!g.gang_plan || capturing(st)) return false;
  switch (k) {
    case 1: return launch<1>(g, cap, io, st, e);
    case 2: return launch<2>(g, cap, io, st, e);
    case 3: return launch<3>(g, cap, io, st, e);
    case 4: return launch<4>(g, cap, io, st, e);
    default: return false;
  }
}

}  // namespace ig
