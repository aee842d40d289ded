// Launch code of the matrix-free operator (Section 2, Eq. fe-problem; BR2 of
// Section 4.4): the kernels around the tile work of apply_kernel.cuh,
// apply2_kernel.cuh, apply3_kernel.cuh and apply_map_kernel.cuh, their
// shared-memory sizing and grids.
#include "apply_map_kernel.cuh"
#include "apply2_kernel.cuh"
#include "kernels.cuh"

namespace dg {

// ============================================================== operator
__global__ void __launch_bounds__(kThreads) trace_kernel(const ApplyArgs A) {
  pdl_entry();
  const ApplyTile T = A.tiles[blockIdx.x];
  switch (T.p) {
    case 1: trace_tile<1>(A, T); break;
    case 2: trace_tile<2>(A, T); break;
    case 3: trace_tile<3>(A, T); break;
    case 4: trace_tile<4>(A, T); break;
    case 5: trace_tile<5>(A, T); break;
    case 6: trace_tile<6>(A, T); break;
    case 7: trace_tile<7>(A, T); break;
    case 8: trace_tile<8>(A, T); break;
    default: break;
  }
}

// Inside PCG, after the solve has stopped: no operator, and alpha = 0, so that
// the updates riding on the preconditioner change nothing.
__device__ __forceinline__ bool pcg_stopped(const ApplyArgs& A) {
  if (!A.pcg_sc || A.pcg_sc[SC_STATUS] == 0.0) return false;
  if (blockIdx.x == 0 && threadIdx.x == 0) A.pcg_sc[SC_ALPHA] = 0.0;
  return true;
}

// End of a persistent operator launch: the last CTA to leave resets the tile
// counter and sums the tile partials of x . y in tile order.  Inside PCG
// (pcg_sc set, x = p, y = q) it also forms the step alpha = (r.z) / (p.q) once
// for the kernels that apply the update r -= alpha q, x += alpha p.
template <int NT>
__device__ __forceinline__ void apply_exit(const ApplyArgs& A, double* red) {
  __shared__ unsigned s_last;
  pdl_trigger();   // this CTA's tiles are done: the next kernel may start launching
  // the scalars alpha needs, loaded before the ticket so that their latency
  // overlaps it (no kernel writes them while the operator runs)
  double rz = 0.0;
  if (threadIdx.x == 0) {
    if (A.pcg_sc) rz = A.pcg_sc[SC_RZ];
    __threadfence();
    s_last = (atomicAdd(A.sched + 1, 1u) == gridDim.x - 1) ? 1u : 0u;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    if (A.dot_partial) {
      double v = 0.0;
      for (int i = threadIdx.x; i < A.n_tiles; i += NT) v += __ldcg(A.dot_partial + i);
      v = block_sum<NT>(v, red);
      if (threadIdx.x == 0) {
        *A.dot_out = v;
        if (A.pcg_sc) A.pcg_sc[SC_ALPHA] = rz / v;
      }
    }
    if (threadIdx.x == 0) {
      A.sched[0] = 0u;
      A.sched[1] = 0u;
    }
  }
}

// Persistent operator kernel: a grid sized to the resident capacity, CTA b
// starting on tile b (consecutive CTAs land on different SMs) and then taking
// tiles from an atomic counter, heaviest first (tiles are degree-sorted), so
// the uneven tiles balance across SMs.  The next tile's number is fetched
// while a tile runs (two slots, so that a fast warp's fetch cannot overwrite
// the number a slow one has yet to read).  The last CTA to leave resets the
// counter and, when a dot product is requested, sums the tile partials in
// tile order (deterministic whichever CTA ran which tile).
template <bool BR2>
__global__ void __launch_bounds__(kThreads) apply_kernel(const ApplyArgs A) {
  pdl_entry();
  extern __shared__ __align__(16) double smem[];
  __shared__ double red[kThreads];
  if (pcg_stopped(A)) return;
  __shared__ int s_next[2];
  for (int t = blockIdx.x, par = 0; t < A.n_tiles; par ^= 1) {
    if (threadIdx.x == 0) s_next[par] = (int)(gridDim.x + atomicAdd(A.sched, 1u));
    const ApplyTile T = A.tiles[t];
    switch (T.p) {
      case 1: apply_tile<1, BR2>(A, T, t, smem, red); break;
      case 2: apply_tile<2, BR2>(A, T, t, smem, red); break;
      case 3: apply_tile<3, BR2>(A, T, t, smem, red); break;
      case 4: apply_tile<4, BR2>(A, T, t, smem, red); break;
      case 5: apply_tile<5, BR2>(A, T, t, smem, red); break;
      case 6: apply_tile<6, BR2>(A, T, t, smem, red); break;
      case 7: apply_tile<7, BR2>(A, T, t, smem, red); break;
      case 8: apply_tile<8, BR2>(A, T, t, smem, red); break;
      default: break;
    }
    __syncthreads();
    t = s_next[par];
  }
  apply_exit<kThreads>(A, red);
}

#define DG_CASES_2 \
    DG_CASE_2(1) DG_CASE_2(2) DG_CASE_2(3) DG_CASE_2(4) DG_CASE_2(5) DG_CASE_2(6) DG_CASE_2(7) DG_CASE_2(8)

// Modes and traces of x on large square meshes.  UPDATE (inside PCG): p = z + beta p
// (first: p = z, and the initial scalars and loop condition) takes the place of
// x.
template <bool UPDATE>
__global__ void __launch_bounds__(kThreads3)
modal2_kernel(const ApplyArgs A, double* p, const double* z, double* sc, cudaGraphConditionalHandle h,
              int use_cond, int first) {
  __shared__ __align__(16) double smem[modal2_doubles()];
  const ApplyTile T = A.tiles[blockIdx.x];
  const int4 hang = __ldg(A.hang2_tile + blockIdx.x);
  switch (T.p) {   // the tables: written by no kernel, fetched before the wait
#define DG_CASE_2(PP) \
    case PP: modal2_tables<PP>(A, smem); break;
    DG_CASES_2
#undef DG_CASE_2
    default: break;
  }
  pdl_entry();
  double beta = 0.0;
  if (UPDATE) {
    if (!first && sc[SC_STATUS] != 0.0) return;   // stopped: the loop condition is already clear
    if (!first) beta = sc[SC_BETA];
  }
  if (A.skip && A.skip[(int64_t)T.inst * A.skip_stride] != 0.0) return;
  switch (T.p) {
#define DG_CASE_2(PP) \
    case PP: modal2_tile<PP, UPDATE>(A, T, hang, smem, p, z, beta, first != 0); break;
    DG_CASES_2
#undef DG_CASE_2
    default: break;
  }
  if (UPDATE && first) pcg_first_scalars(sc, h, use_cond);
}

// The operator of large square meshes, a tile per CTA; the last CTA to leave sums the
// tile partials of x . y in tile order.
template <bool BR2>
__global__ void __launch_bounds__(kThreads3) apply2_kernel(const ApplyArgs A) {
  __shared__ __align__(16) double smem[apply2_doubles()];
  const ApplyTile T = A.tiles[blockIdx.x];
  const int4 hang = __ldg(A.hang2_tile + blockIdx.x);
  Side2 first;
  const int n = modal_table_doubles(T.p);
  for (int i = threadIdx.x; i < n; i += kThreads3) smem[i] = __ldg(A.tab + A.moff3[T.p] + i);
  switch (T.p) {
#define DG_CASE_2(PP) \
    case PP: side2_fetch<PP, BR2>(A, T, hang, first); break;
    DG_CASES_2
#undef DG_CASE_2
    default: break;
  }
  pdl_entry();
  if (pcg_stopped(A)) return;
  if (A.skip && A.skip[(int64_t)T.inst * A.skip_stride] != 0.0) {
    if (A.dot_partial && threadIdx.x == 0) A.dot_partial[blockIdx.x] = 0.0;
  } else {
    double part = 0.0;
    switch (T.p) {
#define DG_CASE_2(PP) \
      case PP: part = apply2_tile<PP, BR2>(A, T, hang, smem, first); break;
      DG_CASES_2
#undef DG_CASE_2
      default: break;
    }
    if (A.dot_partial && threadIdx.x < 32) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
      if (threadIdx.x == 0) A.dot_partial[blockIdx.x] = part;
    }
  }
  if (!A.dot_partial) return;
  __syncthreads();   // the tile's partial before the CTA's ticket
  apply_exit<kThreads3>(A, smem);
}

// Weights of every sub-face of a mapped mesh.
template <bool BR2>
__global__ void __launch_bounds__(kThreads3) map_face_kernel(const ApplyArgs A) {
  pdl_entry();
  extern __shared__ __align__(16) double smem[];
  map_face_tile<BR2>(A, A.mface_tiles[blockIdx.x], smem);
}

// Persistent operator kernel of mapped squares (same scheduling as on boxes).  Its
// shared memory leaves room for three or four CTAs per SM; left to itself the
// compiler takes 48 registers and spills 28 bytes for more (98k unknowns, whole
// apply 43.8 -> 42.6 us).
__global__ void __launch_bounds__(kThreads, 4) apply_map_kernel(const ApplyArgs A) {
  pdl_entry();
  extern __shared__ __align__(16) double smem[];
  __shared__ double red[kThreads];
  if (pcg_stopped(A)) return;
  __shared__ int s_next[2];
  for (int t = blockIdx.x, par = 0; t < A.n_tiles; par ^= 1) {
    if (threadIdx.x == 0) s_next[par] = (int)(gridDim.x + atomicAdd(A.sched, 1u));
    const ApplyTile T = A.tiles[t];
    switch (T.p) {
      case 1: apply_map_tile<1>(A, T, t, smem, red); break;
      case 2: apply_map_tile<2>(A, T, t, smem, red); break;
      case 3: apply_map_tile<3>(A, T, t, smem, red); break;
      case 4: apply_map_tile<4>(A, T, t, smem, red); break;
      case 5: apply_map_tile<5>(A, T, t, smem, red); break;
      case 6: apply_map_tile<6>(A, T, t, smem, red); break;
      case 7: apply_map_tile<7>(A, T, t, smem, red); break;
      case 8: apply_map_tile<8>(A, T, t, smem, red); break;
      default: break;
    }
    __syncthreads();
    t = s_next[par];
  }
  apply_exit<kThreads>(A, red);
}

// Modes and side traces of x on cube meshes.  UPDATE (inside PCG): p = z +
// beta p (first: p = z, and the initial scalars and loop condition) takes the
// place of x.
template <bool UPDATE>
__global__ void __launch_bounds__(kThreads3)
modal3_kernel(const ApplyArgs A, double* p, const double* z, double* sc, cudaGraphConditionalHandle h,
              int use_cond, int first) {
  pdl_entry();
  extern __shared__ __align__(16) double smem[];
  double beta = 0.0;
  if (UPDATE) {
    if (!first && sc[SC_STATUS] != 0.0) return;   // stopped: the loop condition is already clear
    if (!first) beta = sc[SC_BETA];
  }
  const ApplyTile T = A.tiles[blockIdx.x];
  switch (T.p) {
#define DG_MODAL_CASE(PP) \
    case PP: modal3_tile<PP, UPDATE>(A, T, smem, p, z, beta, first != 0); break;
    DG_MODAL_CASE(1) DG_MODAL_CASE(2) DG_MODAL_CASE(3) DG_MODAL_CASE(4)
    DG_MODAL_CASE(5) DG_MODAL_CASE(6) DG_MODAL_CASE(7) DG_MODAL_CASE(8)
#undef DG_MODAL_CASE
    default: break;
  }
  if (UPDATE && first) pcg_first_scalars(sc, h, use_cond);
}

// Residuals of both sides of every hanging sub-face of a cube mesh.
template <bool BR2>
__global__ void __launch_bounds__(kThreads3) hang3_kernel(const ApplyArgs A) {
  pdl_entry();
  extern __shared__ __align__(16) double smem[];
  const HangTile T = A.hang_tiles[blockIdx.x];
  switch (T.p) {
#define DG_HANG_CASE(PP) \
    case PP: hang3_tile<PP, BR2>(A, T, smem); break;
    DG_HANG_CASE(1) DG_HANG_CASE(2) DG_HANG_CASE(3) DG_HANG_CASE(4)
    DG_HANG_CASE(5) DG_HANG_CASE(6) DG_HANG_CASE(7) DG_HANG_CASE(8)
#undef DG_HANG_CASE
    default: break;
  }
}

// Persistent operator kernel of cube meshes (same scheduling as on squares).
template <bool BR2>
__global__ void __launch_bounds__(kThreads3) apply3_kernel(const ApplyArgs A) {
  pdl_entry();
  extern __shared__ __align__(16) double smem[];
  __shared__ double red[kThreads3];
  if (pcg_stopped(A)) return;
  __shared__ int s_next[2];
  for (int t = blockIdx.x, par = 0; t < A.n_tiles; par ^= 1) {
    if (threadIdx.x == 0) s_next[par] = (int)(gridDim.x + atomicAdd(A.sched, 1u));
    const ApplyTile T = A.tiles[t];
    switch (T.p) {
      case 1: apply3_tile<1, BR2>(A, T, t, smem, red); break;
      case 2: apply3_tile<2, BR2>(A, T, t, smem, red); break;
      case 3: apply3_tile<3, BR2>(A, T, t, smem, red); break;
      case 4: apply3_tile<4, BR2>(A, T, t, smem, red); break;
      case 5: apply3_tile<5, BR2>(A, T, t, smem, red); break;
      case 6: apply3_tile<6, BR2>(A, T, t, smem, red); break;
      case 7: apply3_tile<7, BR2>(A, T, t, smem, red); break;
      case 8: apply3_tile<8, BR2>(A, T, t, smem, red); break;
      default: break;
    }
    __syncthreads();
    t = s_next[par];
  }
  apply_exit<kThreads3>(A, red);
}

// static shared-memory layout of a degree-p tile up to the item partials (doubles)
static int apply_shape_smem(int p) {
  switch (p) {
    case 1: return ApplyShape<1>::PART;
    case 2: return ApplyShape<2>::PART;
    case 3: return ApplyShape<3>::PART;
    case 4: return ApplyShape<4>::PART;
    case 5: return ApplyShape<5>::PART;
    case 6: return ApplyShape<6>::PART;
    case 7: return ApplyShape<7>::PART;
    default: return ApplyShape<8>::PART;
  }
}

static int map_shape_smem(int p) {
  switch (p) {
    case 1: return MapShape<1>::SMEM;
    case 2: return MapShape<2>::SMEM;
    case 3: return MapShape<3>::SMEM;
    case 4: return MapShape<4>::SMEM;
    case 5: return MapShape<5>::SMEM;
    case 6: return MapShape<6>::SMEM;
    case 7: return MapShape<7>::SMEM;
    default: return MapShape<8>::SMEM;
  }
}

int64_t apply_smem_for(const dg_mesh& M) {
  if (M.host.dim == 3) return M.apply3_smem;
  if (M.host.mapped) {
    int64_t mx = 0;
    for (int t = 0; t < M.n_tiles; ++t) mx = std::max<int64_t>(mx, map_shape_smem(M.h_tiles[t].p));
    return 8 * mx;
  }
  if (M.modal2) return 0;   // static
  // the layout of the tile's degree plus its sub-face item partials
  int64_t mx = 0;
  for (int t = 0; t < M.n_tiles; ++t) {
    const ApplyTile& T = M.h_tiles[t];
    const int64_t nit = M.h_item_ptr.empty() ? 0 : M.h_item_ptr[t + 1] - M.h_item_ptr[t];
    mx = std::max<int64_t>(mx, apply_shape_smem(T.p) + 2 * nit * (T.p + 1));
  }
  return 8 * mx;
}

ApplyArgs make_apply_args(const dg_mesh& M, const double* x, double* y, Reduce red) {
  ApplyArgs A;
  A.x = x;
  A.y = y;
  A.off = M.d_off;
  A.aih = M.d_aih;
  A.tr = M.d_tr;
  A.sf_ptr = M.d_sf_ptr;
  A.face_items = M.d_face_items;
  A.face_br2 = M.d_face_br2;
  A.sfm2 = M.d_sfm2;
  A.side2 = reinterpret_cast<const int2*>(M.d_side2);
  A.hang2 = reinterpret_cast<const int2*>(M.d_hang2);
  A.hang2_tile = reinterpret_cast<const int4*>(M.d_hang2_tile);
  A.sfm3 = M.d_sfm3;
  A.erec3 = M.d_erec3;
  A.hang3 = M.d_hang3;
  A.hang_tiles = M.d_hang_tiles;
  A.xm = M.d_xm;
  for (int p = 0; p <= kMaxP; ++p) A.moff3[p] = M.moff3[p];
  A.tab = M.d_tables;
  A.order = M.d_order;
  A.tiles = M.d_tiles;
  A.item_ptr = M.d_item_ptr;
  A.side_items = reinterpret_cast<const int2*>(M.d_side_items);
  A.dot_partial = red.partial;
  A.dot_out = red.out;
  A.pcg_sc = nullptr;
  A.skip = M.skip_status;
  A.skip_stride = M.skip_stride;
  A.n_tiles = M.n_tiles;
  A.sched = M.d_sched;
  for (int p = 0; p <= kMaxP; ++p) A.boff[p] = M.boff[p];
  A.mface = M.d_mface;
  A.mface_tiles = M.d_mface_tiles;
  A.mside = M.d_mside;
  A.mw = M.d_mw;
  A.gvol = M.d_gvol;
  A.goff = M.d_goff;
  A.gface = M.d_gface;
  A.gbr2 = M.d_gbr2;
  A.g2off = M.d_g2off;
  for (int p = 0; p <= kMaxP; ++p) A.moff[p] = M.moff[p];
  return A;
}

int apply_kernel_setup(const dg_mesh& M) {
  // The shared-memory opt-in is an attribute of the kernel function on the
  // current device, shared by every mesh: raise it to the device limit (a
  // mesh's own size could lower it under an earlier mesh's needs), and size the
  // resident grid of this mesh's persistent launch from its own tile layout.
  int dev = 0, sms = 0, per = 0, optin = 0;
  DG_CUDA(cudaGetDevice(&dev));
  DG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  optin -= 4 * 1024;   // room for the kernels' static shared memory
  const bool br2 = M.opts.form == DG_FORM_BR2;
  if (M.host.dim == 3) {
    const int smem = (int)M.apply3_smem;
    DG_REQUIRE(smem <= optin && M.modal3_smem <= optin, "operator tile needs too much shared memory");
    DG_CUDA(cudaFuncSetAttribute(modal3_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    DG_CUDA(cudaFuncSetAttribute(modal3_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    DG_CUDA(cudaFuncSetAttribute(apply3_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    DG_CUDA(cudaFuncSetAttribute(apply3_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    if (br2) DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, apply3_kernel<true>, kThreads3, smem));
    else DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, apply3_kernel<false>, kThreads3, smem));
    return sms * (per > 0 ? per : 1);
  }
  if (M.modal2) return M.n_tiles;   // a CTA per tile
  const int smem = (int)M.apply_smem;
  DG_REQUIRE(smem <= optin, "operator tile needs too much shared memory");
  if (M.host.mapped) {
    DG_CUDA(cudaFuncSetAttribute(apply_map_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
    DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, apply_map_kernel, kThreads, smem));
    return sms * (per > 0 ? per : 1);
  }
  DG_CUDA(cudaFuncSetAttribute(apply_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
  DG_CUDA(cudaFuncSetAttribute(apply_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, optin));
  if (br2)
    DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, apply_kernel<true>, kThreads, smem));
  else
    DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, apply_kernel<false>, kThreads, smem));
  return sms * (per > 0 ? per : 1);
}

static void launch_hang3(const dg_mesh& M, const ApplyArgs& A, cudaStream_t s) {
  const int g = (int)M.h_hang_tiles.size();
  if (g == 0) return;
  const size_t smem = (size_t)M.hang3_smem;
  if (M.opts.form == DG_FORM_BR2) launch_k(hang3_kernel<true>, g, kThreads3, smem, s, A);
  else launch_k(hang3_kernel<false>, g, kThreads3, smem, s, A);
}

static void launch_modal3(const dg_mesh& M, const ApplyArgs& A, cudaStream_t s) {
  launch_k(modal3_kernel<false>, M.n_tiles, kThreads3, (size_t)M.modal3_smem, s, A, (double*)nullptr,
           (const double*)nullptr, (double*)nullptr, (cudaGraphConditionalHandle)0, 0, 0);
  launch_hang3(M, A, s);
}

static void launch_map_faces(const dg_mesh& M, const ApplyArgs& A, cudaStream_t s) {
  const int g = (int)M.h_mface_tiles.size();
  const size_t smem = (size_t)M.mface_smem;
  if (M.opts.form == DG_FORM_BR2) launch_k(map_face_kernel<true>, g, kThreads3, smem, s, A);
  else launch_k(map_face_kernel<false>, g, kThreads3, smem, s, A);
}

// what an apply needs of x beside x itself: the side traces (modes, weights)
static void launch_sides(const dg_mesh& M, const ApplyArgs& A, cudaStream_t s) {
  if (M.host.dim == 3) {
    launch_modal3(M, A, s);
  } else if (M.modal2) {
    launch_k(modal2_kernel<false>, M.n_tiles, kThreads3, 0, s, A, (double*)nullptr, (const double*)nullptr,
             (double*)nullptr, (cudaGraphConditionalHandle)0, 0, 0);
  } else {
    launch_k(trace_kernel, M.n_tiles, kThreads, 0, s, A);
    if (M.host.mapped) launch_map_faces(M, A, s);
  }
}

void launch_trace(const dg_mesh& M, const double* x, cudaStream_t s) {
  if (M.n_tiles == 0) return;
  const ApplyArgs A = make_apply_args(M, x, nullptr, Reduce{});
  launch_sides(M, A, s);
  DG_CUDA(cudaGetLastError());
}

void launch_apply(const dg_mesh& M, const double* x, double* y, Reduce red, cudaStream_t s,
                  bool with_trace, double* pcg_sc) {
  if (M.n_tiles == 0) return;
  DG_REQUIRE(!pcg_sc || red.partial, "the PCG step needs the p . q reduction");
  ApplyArgs A = make_apply_args(M, x, y, red);
  A.pcg_sc = pcg_sc;
  if (with_trace) launch_sides(M, A, s);
  const int grid = M.n_tiles < M.apply_grid ? M.n_tiles : M.apply_grid;
  const bool br2 = M.opts.form == DG_FORM_BR2;
  const size_t smem = (size_t)(M.host.dim == 3 ? M.apply3_smem : M.apply_smem);
  if (M.host.dim == 3) {
    if (br2) launch_k(apply3_kernel<true>, grid, kThreads3, smem, s, A);
    else launch_k(apply3_kernel<false>, grid, kThreads3, smem, s, A);
  } else if (M.host.mapped) {
    launch_k(apply_map_kernel, grid, kThreads, smem, s, A);
  } else if (M.modal2) {
    if (br2) launch_k(apply2_kernel<true>, M.n_tiles, kThreads3, 0, s, A);
    else launch_k(apply2_kernel<false>, M.n_tiles, kThreads3, 0, s, A);
  } else if (br2) {
    launch_k(apply_kernel<true>, grid, kThreads, smem, s, A);
  } else {
    launch_k(apply_kernel<false>, grid, kThreads, smem, s, A);
  }
  DG_CUDA(cudaGetLastError());
}

void launch_faces_of_traces(const dg_mesh& M, const double* x, cudaStream_t s) {
  launch_map_faces(M, make_apply_args(M, x, nullptr, Reduce{}), s);
  DG_CUDA(cudaGetLastError());
}

void launch_modal_update(const dg_mesh& M, double* p, const double* z, double* sc,
                          unsigned long long cond_handle, int use_cond, int first, cudaStream_t s) {
  const ApplyArgs A = make_apply_args(M, p, nullptr, Reduce{});
  if (M.host.dim == 2) {
    launch_k(modal2_kernel<true>, M.n_tiles, kThreads3, 0, s, A, p, z, sc, (cudaGraphConditionalHandle)cond_handle,
             use_cond, first);
    DG_CUDA(cudaGetLastError());
    return;
  }
  launch_k(modal3_kernel<true>, M.n_tiles, kThreads3, (size_t)M.modal3_smem, s, A, p, z, sc,
           (cudaGraphConditionalHandle)cond_handle, use_cond, first);
  launch_hang3(M, A, s);
  DG_CUDA(cudaGetLastError());
}

// ============================================================== tile tuner
// Time of one operator kernel (side traces in place) as a solve runs it:
// kReps launches captured into a CUDA graph (programmatic edges between them, as
// in the PCG graph), the graph launched once to warm up and then timed with CUDA
// events, best of kRuns, on a private stream ordered after the work already
// queued on s.
static double time_apply_ms(const dg_mesh& M, const double* x, double* y, cudaStream_t s) {
  constexpr int kReps = 20, kRuns = 3;
  cudaStream_t ts = nullptr;
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ge = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  auto release = [&]() {
    if (ts) {
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      if (cudaStreamIsCapturing(ts, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) {
        cudaGraph_t part = nullptr;
        cudaStreamEndCapture(ts, &part);
        if (part) cudaGraphDestroy(part);
      }
      cudaStreamSynchronize(ts);
    }
    if (ge) cudaGraphExecDestroy(ge);
    if (g) cudaGraphDestroy(g);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (ts) cudaStreamDestroy(ts);
  };
  float best = 0.0f;
  try {
    DG_CUDA(cudaStreamCreateWithFlags(&ts, cudaStreamNonBlocking));
    DG_CUDA(cudaEventCreate(&e0));
    DG_CUDA(cudaEventCreate(&e1));
    DG_CUDA(cudaEventRecord(e0, s));
    DG_CUDA(cudaStreamWaitEvent(ts, e0, 0));
    DG_CUDA(cudaStreamBeginCapture(ts, cudaStreamCaptureModeThreadLocal));
    for (int i = 0; i < kReps; ++i) launch_apply(M, x, y, Reduce{}, ts, false);
    DG_CUDA(cudaStreamEndCapture(ts, &g));
    DG_CUDA(cudaGraphInstantiate(&ge, g, 0));
    DG_CUDA(cudaGraphLaunch(ge, ts));
    for (int r = 0; r < kRuns; ++r) {
      DG_CUDA(cudaEventRecord(e0, ts));
      DG_CUDA(cudaGraphLaunch(ge, ts));
      DG_CUDA(cudaEventRecord(e1, ts));
      DG_CUDA(cudaEventSynchronize(e1));
      float t = 0.0f;
      DG_CUDA(cudaEventElapsedTime(&t, e0, e1));
      if (r == 0 || t < best) best = t;
    }
  } catch (...) {
    release();
    throw;
  }
  release();
  return best / kReps;
}

void tune_tiles(dg_mesh* M, cudaStream_t s, void (*retile)(dg_mesh*, void*), void* ctx) {
  if (M->n_tiles == 0) return;
  DevArena scratch;
  try {
    const int64_t n = M->n_dofs;
    double* x = scratch.alloc<double>(n);
    double* y = scratch.alloc<double>(n);
    // x = 1 everywhere: the kernel's work and timing do not depend on the values
    std::vector<double> ones(n, 1.0);
    DG_CUDA(cudaMemcpyAsync(x, ones.data(), n * sizeof(double), cudaMemcpyHostToDevice, s));
    auto measure = [&]() {
      retile(M, ctx);
      upload_tiles(M, s);
      launch_trace(*M, x, s);
      return time_apply_ms(*M, x, y, s);
    };
    const double fixed_ms = measure();
    double best_ms = fixed_ms;
    if (M->host.dim == 3) {
      // shared-memory budget of a tile: 4, 3 (the fixed rule) or 2 tiles per SM
      const int64_t fixed_budget = M->apply3_budget, budgets[3] = {6656, 9216, 13312};
      int64_t best = fixed_budget;
      for (int64_t b : budgets) {
        if (b == fixed_budget) continue;
        M->apply3_budget = b;
        const double t = measure();
        if (t < 0.99 * best_ms) {
          best_ms = t;
          best = b;
        }
      }
      M->apply3_budget = best;
    } else {
      bool present[kMaxP + 1] = {false};
      for (const ApplyTile& T : M->h_tiles) present[T.p] = true;
      // highest degrees first: their tiles set the length of the launch
      for (int P = kMaxP; P >= 1; --P) {
        if (!present[P]) continue;
        const int cap = M->modal2 ? apply2_epb(P) : apply_epb(P), start = M->tile_epb[P];
        const int cand[3] = {cap, std::max(1, (3 * cap + 3) / 4), std::max(1, cap / 2)};
        int best = start;
        for (int c : cand) {
          if (c == start) continue;
          M->tile_epb[P] = c;
          const double t = measure();
          if (t < 0.99 * best_ms) {
            best_ms = t;
            best = c;
          }
        }
        M->tile_epb[P] = best;
      }
    }
    retile(M, ctx);
    upload_tiles(M, s);
    M->stats.tiles_tuned = 1;
    M->stats.apply_ms_fixed = fixed_ms;
    M->stats.apply_ms_tuned = best_ms;
  } catch (...) {
    scratch.release();
    throw;
  }
  scratch.release();
  for (int p = 0; p <= kMaxP; ++p) M->stats.tile_elems[p] = M->host.dim == 2 ? M->tile_epb[p] : 0;
  M->stats.tile_smem_budget = M->host.dim == 3 ? 8 * M->apply3_budget : 0;
}

}  // namespace dg
