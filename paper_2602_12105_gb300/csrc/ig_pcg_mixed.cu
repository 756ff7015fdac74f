// ig_pcg_mixed.cu -- mixed-precision solve of A X = RHS (forward and adjoint systems of §7.1 /
// §5.2) to an FP64 relative residual: FP32 Jacobi-PCG on the FP32 copy of A inside an FP64
// iterative refinement whose residuals use the FP64 operator.
//
//   x64 = 0, r64 = rhs
//   repeat:  r32 = r64 / ||r64||            (per column; unit-norm inner right-hand side)
//            solve A32 d = r32 by FP32 Jacobi-PCG to inner_tol (dot products summed in FP64)
//            x64 += ||r64|| d
//            r64 = rhs - A64 x64 in FP64; stop when ||r64|| / ||rhs|| <= rel_tol
//
// It runs inside the same three-kernel iteration as the FP64 solver, with a per-mesh phase:
//   Inner   : spmv q32 = A32 p32 | update r32, (r.z, r.r) | pupdate x32, p32
//   Apply   : set by update when the inner solve converged; pupdate adds ||r64|| d into x64
//   (next)  : spmv computes r64 = rhs - A64 x64 and its norms (the refinement residual)
//   Restart : update forms r32 = r64 / ||r64||, d = 0; pupdate sets p32 = z32
// so a refinement costs one iteration slot whose SpMV runs in FP64, and no extra launches.
// FP64 arithmetic is used only for the residual SpMV, the x64 update and the reductions.
#include "ig_mixed.cuh"

namespace ig {

namespace {

// The mixed-precision kernels take a tile in passes of kTileRows rows (kRowsPerThread per thread);
// a thread adds its rows' FP32 products across the passes of a tile (at most 64 passes, 256
// terms), the warps add their lanes in FP32 and the tile's warps and tiles are added in FP64.
template <int NV>
struct PassSum {
  float s[NV];
  __device__ __forceinline__ PassSum() {
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] = 0.f;
  }
  __device__ __forceinline__ void add(const float (&x)[NV]) {
#pragma unroll
    for (int i = 0; i < NV; ++i) s[i] += x[i];
  }
};

// ------------------------------------------------------------------------------- kernels
template <int K>
__global__ void __launch_bounds__(kBlock) init_mixed_kernel(const MeshDev* __restrict__ mds,
                                                            const int2* __restrict__ tiles, IoTable io, int rhs_mass,
                                                            LoopCtl* ctl, double tol, double inner_tol, int max_iter,
                                                            int max_refine, int cap) {
  const int2 tl = tiles[blockIdx.x];
  const MeshDev& md = mds[tl.x];
  const long nn = md.n;
  const long t0 = (long)tl.y * md.tile_rows32;
  const long t1 = t0 + md.tile_rows32 < nn ? t0 + md.tile_rows32 : nn;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->cnt = 0u;
    ctl->iter = 0;
    ctl->all_done = 0;
    ctl->any_apply = 0;
    ctl->ndone_start = 1 << 30;  // a whole solve stops only when every mesh is done
    ctl->cap = cap;
  }
  const double* __restrict__ src = io.in[tl.x];
  double acc[K];
#pragma unroll
  for (int c = 0; c < K; ++c) acc[c] = 0.0;
  for (long base = t0; base < t1; base += kTileRows) {
#pragma unroll
    for (int rr = 0; rr < kRowsPerThread; ++rr) {
      const long row = base + rr * kBlock + threadIdx.x;
      if (row < t1) {
        const double mass = rhs_mass ? md.M[row] : 1.0;
#pragma unroll
        for (int c = 0; c < K; ++c) {
          const double b = rhs_mass ? mass * src[row * K + c] : src[row * K + c];
          md.rhs[c * nn + row] = b;
          md.r[c * nn + row] = b;
          md.x[c * nn + row] = 0.0;
          acc[c] = fma(b, b, acc[c]);
        }
      }
    }
  }
  if (reduce_tiles<K, kInOrder>(acc, md.part, tl.y, md.ntiles32, &md.s->cnt[2]) && threadIdx.x == 0)
    finish_init_mixed(md.s, K, acc, tol, inner_tol, max_iter, max_refine);
}

template <int K>
__global__ void __launch_bounds__(kBlock, 4) spmv_mixed_kernel(const MeshDev* __restrict__ mds, LoopCtl* ctl, ListRef L) {
  __shared__ TileCtx tc;
  tile_loop<K, kGroups>(
      mds, L, 3, 0, tc, [](const ScalSnap& x) { return !x.done && x.phase == kPhaseInner; },
      [&](const MeshDev& md, int tile, double* red, double* out) {
        const int n = md.n, nsl = (n + 31) >> 5, lane = threadIdx.x & 31;
        const int rb = tile / md.s32_ncb, cb = tile - rb * md.s32_ncb;
        const float* __restrict__ A = as_global(md.A32);
        const float* __restrict__ p = as_global(md.p32);
        float* __restrict__ q32 = as_global(md.q32);
        // This warp's slices of the block, line by line. A line's products are added in FP32 over the
        // warp, the lines in FP64.
        const int warp = threadIdx.x >> 5, w = md.tile_rows32 >> 5;
        double sum = 0.0;
        for (int l = rb * md.s32_h; l < (rb + 1) * md.s32_h; ++l) {
          const int s0 = (l * md.s32_ncb + cb) * w;
          if (s0 >= nsl) break;
          const unsigned bits = pattern_bits(md, s0, nsl);
          float pq[K];
#pragma unroll
          for (int k = 0; k < K; ++k) pq[k] = 0.f;
          for (int c = warp; c < w; c += kWarps) {
            const int sl = s0 + c, row = sl * 32 + lane;
            if (row < n) {
              float q[K];
              row_product32<K>(md, A, p, sl, row, (bits >> c & 1u) != 0, q);
              float pi[K];
              load_row32<K>(p, row, pi);
#pragma unroll
              for (int k = 0; k < K; ++k) {
                q32[(long)k * n + row] = q[k];
                pq[k] = fmaf(pi[k], q[k], pq[k]);
              }
            }
          }
          const double line = to_double(warp_sum_transposed<K>(pq, lane));
          sum = l == rb * md.s32_h ? line : sum + line;
        }
        if (warp_sum_writer<K>(lane) && warp_sum_index<K>(lane) < K) red[warp_sum_index<K>(lane) * kWarps + warp] = sum;
        __syncthreads();
        if (threadIdx.x < K) out[threadIdx.x] = add_warps_of<kGroups>(red + threadIdx.x * kWarps);
      },
      [](const MeshDev& md, const SolveScal& cur, const double* v) { finish_spmv(md.s, cur, K, v); });
}

// Apply phase: r64 = rhs - A64 x64 in FP64 and its squared norms (the refinement residual).
// Kept out of the FP32 SpMV kernel so that the hot FP32 kernel stays small; it walks the Apply
// list (the meshes in that phase), which the previous update launch built.
template <int K>
__global__ void __launch_bounds__(kBlock, 4) resid_mixed_kernel(const MeshDev* __restrict__ mds, LoopCtl* ctl, ListRef L) {
  __shared__ TileCtx tc;
  if (!ctl->any_apply) return;  // no mesh of the group is in the Apply phase
  tile_loop<K, kInOrder>(
      mds, L, 1, 0, tc, [](const ScalSnap& x) { return !x.done && x.phase == kPhaseApply; },
      [&](const MeshDev& md, int tile, double* red, double* out) {
        const long nn = md.n;
        const long t0 = (long)tile * md.tile_rows32;
        const long t1 = t0 + md.tile_rows32 < nn ? t0 + md.tile_rows32 : nn;
        const double* __restrict__ x = as_global(md.x);
        const bool geom32 = md.geom32 != 0;  // the operator is the FP32 one: its values, exactly
        double acc[K];
#pragma unroll
        for (int c = 0; c < K; ++c) acc[c] = 0.0;
        // tiles of at most kTileRows rows: one pass
#pragma unroll
        for (int rr = 0; rr < kRowsPerThread; ++rr) {
          const long row = t0 + rr * kBlock + threadIdx.x;
          if (row < t1) {
            double ax[K];
            if (geom32) row_product<K>(md, md.A32, row, GatherSoA64<K>{x, nn}, ax);
            else row_product<K>(md, md.A, row, GatherSoA64<K>{x, nn}, ax);
#pragma unroll
            for (int c = 0; c < K; ++c) {
              const double res = md.rhs[c * nn + row] - ax[c];
              md.r[c * nn + row] = res;
              acc[c] = fma(res, res, acc[c]);
            }
          }
        }
        tile_reduce<K, kInOrder>(acc, red, out);
      },
      [](const MeshDev& md, const SolveScal& cur, const double* v) { finish_residual(md.s, cur, K, v); });
}

// Inner phase: r32 -= alpha q32 and the tile's sums r.z, r.r (x32 += alpha p32 waits for the p-update,
// which reads p32 anyway: 16 bytes a row less per iteration); all loads of a thread's rows are issued
// before its stores. Restart phase: r32 = r64 / ||r64||, x32 = 0.
template <int K>
__global__ void __launch_bounds__(kBlock, 4) update_mixed_kernel(const MeshDev* __restrict__ mds, LoopCtl* ctl, ListRef L,
    cudaGraphConditionalHandle handle, int use_graph) {
  __shared__ TileCtx tc;
  __shared__ int s_single, s_iter, s_cap, s_phase;
  if (threadIdx.x == 0) {
    s_single = (__ldcg(&ctl->nmesh) == 1);
    s_iter = __ldcg(&ctl->iter);
    s_cap = __ldcg(&ctl->cap);
    s_phase = kPhaseInner;
    tc.last = 0;
    // a group of one mesh that takes no part in this launch (done: its residual met the tolerance
    // in this iteration, or the loop stopped): no CTA completes it, so the loop is stopped here
    if (s_single && blockIdx.x == 0 && (__ldcg(&ctl->all_done) || __ldcg(&mds[0].s->done))) {
      ctl->all_done = 1;
      if (use_graph) cudaGraphSetConditional(handle, 0u);
    }
  }
  __syncthreads();
  tile_loop<2 * K, kGroups>(
      mds, L, 2, 1, tc,
      [](const ScalSnap& x) { return !x.done && x.phase != kPhaseApply; },
      [&](const MeshDev& md, int tile, double* red, double* out) {
        const long nn = md.n;
        const long t0 = (long)tile * md.tile_rows32u;
        const long t1 = t0 + md.tile_rows32u < nn ? t0 + md.tile_rows32u : nn;
        PassSum<2 * K> sum;
        const float* __restrict__ D32 = as_global(md.Dinv32);
        float* __restrict__ x32 = as_global(md.x32);
        float* __restrict__ r32 = as_global(md.r32);
        if (tc.sn.phase == kPhaseInner) {
          const float* __restrict__ q32 = as_global(md.q32);
          const int n32 = md.n;
          float alpha[K];
#pragma unroll
          for (int c = 0; c < K; ++c) alpha[c] = tc.sn.alpha32[c];
          for (long base = t0; base < t1; base += kTileRows) {
            float acc[2 * K];
#pragma unroll
            for (int i = 0; i < 2 * K; ++i) acc[i] = 0.f;
            constexpr int RB = kRowsPerThread;
            float d[RB], qs[RB][K], rs[RB][K];
#pragma unroll
            for (int u = 0; u < RB; ++u) {
              const int row = (int)base + u * kBlock + threadIdx.x;
              if (row < (int)t1) {
                d[u] = D32[row];
#pragma unroll
                for (int c = 0; c < K; ++c) {
                  qs[u][c] = q32[(long)c * n32 + row];
                  rs[u][c] = r32[(long)c * n32 + row];
                }
              }
            }
#pragma unroll
            for (int u = 0; u < RB; ++u) {
              const int row = (int)base + u * kBlock + threadIdx.x;
              if (row < (int)t1) {
#pragma unroll
                for (int c = 0; c < K; ++c) {
                  const float rv = fmaf(-alpha[c], qs[u][c], rs[u][c]);
                  r32[(long)c * n32 + row] = rv;
                  acc[c] = fmaf(rv, d[u] * rv, acc[c]);
                  acc[K + c] = fmaf(rv, rv, acc[K + c]);
                }
              }
            }
            sum.add(acc);
          }
        } else {
          // Restart: r32 = r64 / ||r64|| for columns still above tol, d = 0
          double inv[K];
          int act[K];
#pragma unroll
          for (int c = 0; c < K; ++c) {
            act[c] = tc.sn.act64[c];
            inv[c] = 1.0 / tc.sn.scale[c];
          }
          const double* __restrict__ r64 = as_global(md.r);
          for (long base = t0; base < t1; base += kTileRows) {
            float acc[2 * K];
#pragma unroll
            for (int i = 0; i < 2 * K; ++i) acc[i] = 0.f;
#pragma unroll
            for (int rr = 0; rr < kRowsPerThread; ++rr) {
              const long row = base + rr * kBlock + threadIdx.x;
              if (row < t1) {
                const float dinv = D32[row];
#pragma unroll
                for (int c = 0; c < K; ++c) {
                  const float rv = act[c] ? (float)(r64[c * nn + row] * inv[c]) : 0.f;
                  r32[c * nn + row] = rv;
                  x32[c * nn + row] = 0.f;
                  acc[c] = fmaf(rv, dinv * rv, acc[c]);
                  acc[K + c] = fmaf(rv, rv, acc[K + c]);
                }
              }
            }
            sum.add(acc);
          }
        }
        tile_reduce<2 * K, kGroups>(sum.s, red, out);
      },
      [&](const MeshDev& md, const SolveScal& cur, const double* v) {
        const int phase = cur.phase == kPhaseInner ? finish_update_mixed(md.s, cur, K, v)
                                                   : finish_restart(md.s, cur, K, v);
        if (threadIdx.x == 0) s_phase = phase;
      });
  if (!s_single) {
    loop_control(mds, ctl, handle, use_graph);
  } else if (tc.last) {
    // the CTA that completed the mesh (flush_tiles ended in a barrier, so s_phase is visible): the
    // next iteration recomputes the FP64 residual when the inner solve just ended; the Apply list
    // is rebuilt by the whole CTA
    const int apply = s_phase == kPhaseApply;
    if (apply && ctl->app_mesh) rebuild_apply(mds, ctl);
    if (threadIdx.x == 0) {
      ctl->any_apply = apply;
      single_loop_control(s_phase < 0, s_iter, s_cap, ctl, handle, use_graph);
    }
  }
}

// x32 += alpha p32, then in the Inner phase p32 = D^-1 r32 + beta p32 (loads of a thread's rows before
// its stores), in the Apply phase x64 += ||r64|| x32.
template <int K>
// In the graph loop of a single mesh (use_graph), CTA 0 also sets the condition of the IF node that
// holds the next iteration's residual kernel: whether the mesh recomputes its FP64 residual then
// (any_apply, as the update launch before this one left it). Iterations without a refinement so
// skip that launch.
__global__ void __launch_bounds__(kBlock, 4) pupdate_mixed_kernel(const MeshDev* __restrict__ mds, LoopCtl* ctl, ListRef L,
                                                                  cudaGraphConditionalHandle apply_handle,
                                                                  int use_graph) {
  __shared__ TileCtx tc;
  if (use_graph && blockIdx.x == 0 && threadIdx.x == 0)
    cudaGraphSetConditional(apply_handle, __ldcg(&ctl->any_apply) ? 1u : 0u);
  tile_loop_plain(mds, L, 1, tc,
                  [](const ScalSnap& x) { return !x.done && (x.phase == kPhaseInner || x.phase == kPhaseApply); },
                  [&](const MeshDev& md, int tile) {
                    const long nn = md.n;
                    const long t0 = (long)tile * md.tile_rows32;
                    const long t1 = t0 + md.tile_rows32 < nn ? t0 + md.tile_rows32 : nn;
                    // x32 += alpha p32 of this slot's iteration (none when it restarted)
                    const bool step = tc.sn.inner_iter > 0;
                    float alpha[K];
#pragma unroll
                    for (int c = 0; c < K; ++c) alpha[c] = tc.sn.alpha32[c];
                    float* __restrict__ x32 = as_global(md.x32);
                    float* __restrict__ p32 = as_global(md.p32);
                    if (tc.sn.phase == kPhaseInner) {
                      float beta[K];
#pragma unroll
                      for (int c = 0; c < K; ++c) beta[c] = tc.sn.beta32[c];
                      const float* __restrict__ D32 = as_global(md.Dinv32);
                      const float* __restrict__ r32 = as_global(md.r32);
                      constexpr int R = 2;  // rows in flight
#pragma unroll
                      for (int r0 = 0; r0 < kRowsPerThread; r0 += R) {
                        float d[R], pi[R][K], rs[R][K], xs[R][K];
#pragma unroll
                        for (int u = 0; u < R; ++u) {
                          const long row = t0 + (r0 + u) * kBlock + threadIdx.x;
                          if (row < t1) {
                            d[u] = D32[row];
                            load_row32<K>(p32, row, pi[u]);
#pragma unroll
                            for (int c = 0; c < K; ++c) {
                              rs[u][c] = r32[c * nn + row];
                              if (step) xs[u][c] = x32[c * nn + row];
                            }
                          }
                        }
#pragma unroll
                        for (int u = 0; u < R; ++u) {
                          const long row = t0 + (r0 + u) * kBlock + threadIdx.x;
                          if (row < t1) {
                            float pn[K];
#pragma unroll
                            for (int c = 0; c < K; ++c) {
                              if (step) x32[c * nn + row] = fmaf(alpha[c], pi[u][c], xs[u][c]);
                              pn[c] = fmaf(beta[c], pi[u][c], d[u] * rs[u][c]);
                            }
                            store_row32<K>(p32, row, pn);
                          }
                        }
                      }
                    } else {
                      double sc[K];
#pragma unroll
                      for (int c = 0; c < K; ++c) sc[c] = tc.sn.scale[c];
                      double* __restrict__ x = as_global(md.x);
#pragma unroll
                      for (int rr = 0; rr < kRowsPerThread; ++rr) {
                        const long row = t0 + rr * kBlock + threadIdx.x;
                        if (row < t1) {
                          float pi[K];
                          if (step) load_row32<K>(p32, row, pi);
#pragma unroll
                          for (int c = 0; c < K; ++c) {
                            float xv = x32[c * nn + row];
                            if (step) xv = fmaf(alpha[c], pi[c], xv);
                            x[c * nn + row] = fma(sc[c], (double)xv, x[c * nn + row]);
                          }
                        }
                      }
                    }
                  });
}

template <int K>
cudaError_t build_plan_mixed(Group& g, SolvePlan& pl) {
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaGraphCreate(&graph, 0);
  if (e != cudaSuccess) return e;
  cudaGraphConditionalHandle handle;
  e = cudaGraphConditionalHandleCreate(&handle, graph, 1u, cudaGraphCondAssignDefault);
  if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = handle;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  e = cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &cp);
  if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  cudaStream_t cs = g.capture_stream;
  // A group of one mesh: the body is an IF node holding the residual kernel (its condition set by
  // the p-update of the iteration before; the value it starts a solve with is irrelevant, since no
  // mesh recomputes its residual in a solve's first iteration and the kernel itself returns when
  // none does), then the SpMV, the update and the p-update. A group of many meshes has some mesh
  // refining in most iterations, where the IF node costs more than it saves: its body launches the
  // residual kernel every iteration.
  const bool use_if = g.nmesh == 1;
  cudaGraphConditionalHandle apply_handle{};
  cudaGraphNode_t if_node = nullptr;
  cudaGraph_t captured = nullptr;
  cudaError_t le = cudaSuccess;
  if (use_if) {
    e = cudaGraphConditionalHandleCreate(&apply_handle, body, 1u, 0u);
    if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
    cudaGraphNodeParams ip = {};
    ip.type = cudaGraphNodeTypeConditional;
    ip.conditional.handle = apply_handle;
    ip.conditional.type = cudaGraphCondTypeIf;
    ip.conditional.size = 1;
    e = cudaGraphAddNode(&if_node, body, nullptr, nullptr, 0, &ip);
    if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
    cudaGraph_t resid_body = ip.conditional.phGraph_out[0];
    e = cudaStreamBeginCaptureToGraph(cs, resid_body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
    resid_mixed_kernel<K><<<g.grid32, kBlock, 0, cs>>>(g.mds, g.ctl, g.listapp);
    le = cudaGetLastError();
    e = cudaStreamEndCapture(cs, &captured);
    if (le != cudaSuccess) e = le;
    if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
    e = cudaStreamBeginCaptureToGraph(cs, body, &if_node, nullptr, 1, cudaStreamCaptureModeThreadLocal);
  } else {
    e = cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
  }
  if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
  if (!use_if) resid_mixed_kernel<K><<<g.grid32, kBlock, 0, cs>>>(g.mds, g.ctl, g.listapp);
  spmv_mixed_kernel<K><<<g.grid32, kBlock, 0, cs>>>(g.mds, g.ctl, g.list32);
  update_mixed_kernel<K><<<g.grid32, kBlock, 0, cs>>>(g.mds, g.ctl, g.list32, handle, 1);
  pupdate_mixed_kernel<K><<<g.grid32, kBlock, 0, cs>>>(g.mds, g.ctl, g.list32, apply_handle, use_if ? 1 : 0);
  le = cudaGetLastError();
  e = cudaStreamEndCapture(cs, &captured);
  if (le != cudaSuccess) e = le;
  if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
  cudaGraphExec_t exec = nullptr;
  e = cudaGraphInstantiate(&exec, graph, 0);
  if (e != cudaSuccess) { cudaGraphDestroy(graph); return e; }
  pl.k = K;
  pl.mixed = 1;
  pl.graph = graph;
  pl.exec = exec;
  return cudaSuccess;
}

int slot_cap(const ig_solve_opts& o) { return o.max_iter + 3 * o.max_refine + 4; }

template <int K>
cudaError_t init_mixed_k(Group& g, const IoTable& io, int rhs_mass, const ig_solve_opts& o, cudaStream_t st) {
  init_mixed_kernel<K><<<g.ntiles32, kBlock, 0, st>>>(g.mds, g.tiles32, io, rhs_mass, g.ctl, o.rel_tol, o.inner_tol,
                                                      o.max_iter, o.max_refine, slot_cap(o));
  return cudaGetLastError();
}

template <int K>
cudaError_t begin_mixed_k(Group& g, const IoTable& io, int rhs_mass, const ig_solve_opts& o, cudaStream_t st) {
  IG_PROF("pcg_init", st);
  cudaError_t e = init_mixed_k<K>(g, io, rhs_mass, o, st);
  if (e != cudaSuccess) return e;
  list_kernel<<<1, kBlock, 0, st>>>(g.mds, g.ctl);
  return cudaGetLastError();
}

template <int K>
cudaError_t host_loop_mixed_k(Group& g, int max_it, int poll, cudaStream_t st) {
  cudaError_t e = group_done_word(g);
  if (e != cudaSuccess) return e;
  for (int it = 0; it < max_it; ++it) {
    {
      IG_PROF("pcg32_resid64", st);
      resid_mixed_kernel<K><<<g.grid32, kBlock, 0, st>>>(g.mds, g.ctl, g.listapp);
    }
    {
      IG_PROF("pcg32_spmv", st);
      spmv_mixed_kernel<K><<<g.grid32, kBlock, 0, st>>>(g.mds, g.ctl, g.list32);
    }
    {
      IG_PROF("pcg32_update", st);
      update_mixed_kernel<K><<<g.grid32, kBlock, 0, st>>>(g.mds, g.ctl, g.list32, cudaGraphConditionalHandle{}, 0);
    }
    {
      IG_PROF("pcg32_pupdate", st);
      pupdate_mixed_kernel<K><<<g.grid32, kBlock, 0, st>>>(g.mds, g.ctl, g.list32, cudaGraphConditionalHandle{}, 0);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (prof_on() || (it % poll) == poll - 1 || it == max_it - 1) {
      e = cudaMemcpyAsync(g.done_host, &g.ctl->all_done, sizeof(int), cudaMemcpyDeviceToHost, st);
      if (e != cudaSuccess) return e;
      e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) return e;
      if (*g.done_host) break;
    }
  }
  return cudaSuccess;
}

template <int K>
cudaError_t solve_mixed_k(Group& g, const IoTable& io, int rhs_mass, const ig_solve_opts& o, cudaStream_t st) {
  const bool graph = o.launch == IG_LAUNCH_GRAPH && !prof_on();
  cudaError_t e;
  if (graph && g.gang_plan) {
    if ((e = init_mixed_k<K>(g, io, rhs_mass, o, st)) != cudaSuccess) return e;
    if (launch_gang(g, K, slot_cap(o), io, st, e)) {
      g.route = IG_ROUTE_ONE_LAUNCH;
      return e;
    }
  }
  e = begin_mixed_k<K>(g, io, rhs_mass, o, st);
  if (e != cudaSuccess) return e;
  if (graph) {
    SolvePlan& pl = g.plans[1][K];
    if (!pl.exec) {
      e = build_plan_mixed<K>(g, pl);
      if (e != cudaSuccess) return e;
    }
    g.route = IG_ROUTE_GRAPH;
    e = cudaGraphLaunch(pl.exec, st);
  } else {
    g.route = IG_ROUTE_HOST;
    e = host_loop_mixed_k<K>(g, slot_cap(o), 16, st);
  }
  if (e != cudaSuccess) return e;
  IG_PROF("pcg_finalize", st);
  finalize_kernel<K><<<g.ntiles, kBlock, 0, st>>>(g.mds, g.tiles, io);
  return cudaGetLastError();
}

}  // namespace

int solver_blocks_per_sm_mixed() {
  int a = 0, b = 0, c = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, spmv_mixed_kernel<3>, kBlock, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, update_mixed_kernel<3>, kBlock, 0);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, pupdate_mixed_kernel<3>, kBlock, 0);
  int m = a < b ? a : b;
  m = m < c ? m : c;
  return m > 0 ? m : 1;
}

cudaError_t group_begin_mixed(Group& g, int k, const IoTable& io, int rhs_mass, const ig_solve_opts& o,
                              cudaStream_t st) {
  switch (k) {
    case 1: return begin_mixed_k<1>(g, io, rhs_mass, o, st);
    case 2: return begin_mixed_k<2>(g, io, rhs_mass, o, st);
    case 3: return begin_mixed_k<3>(g, io, rhs_mass, o, st);
    case 4: return begin_mixed_k<4>(g, io, rhs_mass, o, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t group_host_loop_mixed(Group& g, int k, int budget, cudaStream_t st) {
  switch (k) {
    case 1: return host_loop_mixed_k<1>(g, budget, 8, st);
    case 2: return host_loop_mixed_k<2>(g, budget, 8, st);
    case 3: return host_loop_mixed_k<3>(g, budget, 8, st);
    case 4: return host_loop_mixed_k<4>(g, budget, 8, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t group_solve_mixed(Group& g, int k, const IoTable& io, int rhs_mass, const ig_solve_opts& o,
                              cudaStream_t st) {
  switch (k) {
    case 1: return solve_mixed_k<1>(g, io, rhs_mass, o, st);
    case 2: return solve_mixed_k<2>(g, io, rhs_mass, o, st);
    case 3: return solve_mixed_k<3>(g, io, rhs_mass, o, st);
    case 4: return solve_mixed_k<4>(g, io, rhs_mass, o, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ig
