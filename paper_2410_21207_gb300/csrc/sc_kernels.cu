// Whole-image kernels of libsc_gb300: packing, transposition, the e1 energy, and the per-seam
// local energy refresh and row compaction (arXiv 2410.21207, sections "Energy Mapping" and
// "Removal of Seams"; horizontal seams by transposition, section "Design Techniques").
#include "sc_internal.cuh"
#include "sc_ptx.cuh"
#include "sc_rowops.cuh"

namespace sc {

// ---- pack: HWC uint8 (C in {1,3,4}) -> one uint32 word per pixel, channel c in byte c ----
__global__ void k_pack(const uint8_t *__restrict__ src, int H, int W, int C, uint32_t *__restrict__ img,
                       int pitch) {
  const int64_t n = (int64_t)H * W;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(p / W), j = (int)(p % W);
    img[(int64_t)i * pitch + j] = pack_pixel(src + p * C, C);
  }
}

// ---- unpack: words -> HWC uint8 ----
__global__ void k_unpack(const uint32_t *__restrict__ img, int pitch, int H, int W, int C, uint8_t *__restrict__ dst) {
  const int64_t n = (int64_t)H * W;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(p / W), j = (int)(p % W);
    unpack_pixel(img[(int64_t)i * pitch + j], dst + p * C, C);
  }
}

// ---- transpose of a word image through 32x32 shared-memory tiles (coalesced both ways) ----
__global__ void k_transpose(const uint32_t *__restrict__ src, int ps, int H, int W, uint32_t *__restrict__ dst,
                            int pd) {
  __shared__ uint32_t tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int i = by + r, j = bx + threadIdx.x;
    if (i < H && j < W) tile[r][threadIdx.x] = src[(int64_t)i * ps + j];
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += 8) {
    const int j = bx + r, i = by + threadIdx.x;   // dst row j, column i
    if (i < H && j < W) dst[(int64_t)j * pd + i] = tile[threadIdx.x][r];
  }
}

// ---- e1 energy: sum over the packed channels of |right - left| + |down - up|, clamped ----
__global__ void k_energy(const uint32_t *__restrict__ img, int pitch, int H, int W, uint16_t *__restrict__ E,
                         int pe) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (j >= W || i >= H) return;
  E[(int64_t)i * pe + j] = (uint16_t)energy_at(img, pitch, H, W, i, j);
}

// ---- e1 energy straight from HWC bytes (sc_energy: no word image is kept) ----
// Bound by memory: C + 2 bytes a pixel. One pass instead of a packing pass and a pass over its words
// (4 bytes a pixel written and read again). A thread takes 4 columns of ENERGY_ROWS rows: per row it
// loads the aligned words that hold its 6 pixels (columns j0 - 1 .. j0 + 4), all rows' loads in flight at
// once, and every row serves as its own centre and as its neighbours' upper and lower row. On the device:
// 1920x1080x3 20.1 -> 5.1 us, 3840x2160x3 58.5 -> 14.6 us (2.8 TB/s), 64x48 3.0 -> 1.8 us.
constexpr int ENERGY_ROWS = 4;

template <int C>
__global__ void __launch_bounds__(128) k_energy_bytes(const uint8_t *__restrict__ src, int H, int W,
                                                      uint16_t *__restrict__ E) {
  constexpr int NWD = (6 * C + 3 + 3) / 4;   // words that hold 6 pixels from any byte offset
  const int j0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int i0 = blockIdx.y * ENERGY_ROWS;
  if (j0 >= W) return;
  // words counted from the aligned word holding the image's first byte to the one holding its last
  const uint32_t mis = (uint32_t)((uintptr_t)src & 3u);
  const uint32_t *base = reinterpret_cast<const uint32_t *>(src - mis);
  const int64_t last = ((int64_t)H * W * C - 1 + mis) >> 2;
  uint32_t w[ENERGY_ROWS + 2][NWD];
  uint32_t sh[ENERGY_ROWS + 2];
  const int jf = j0 > 0 ? j0 - 1 : 0;   // first column loaded
#pragma unroll
  for (int r = 0; r < ENERGY_ROWS + 2; ++r) {
    const int i = min(max(i0 + r - 1, 0), H - 1);   // edge rows replicated
    const int64_t b = ((int64_t)i * W + jf) * C + mis;
    sh[r] = (uint32_t)(b & 3) * 8;
#pragma unroll
    for (int n = 0; n < NWD; ++n) {
      const int64_t q = (b >> 2) + n;
      w[r][n] = __ldg(base + (q < last ? q : last));
    }
  }
  // pixels of columns j0 - 1 .. j0 + 4 of a loaded row, channel c in byte c
  auto pixels = [&](int r, uint32_t (&p)[6]) {
    uint32_t v[NWD];
#pragma unroll
    for (int n = 0; n < NWD; ++n) v[n] = __funnelshift_r(w[r][n], n + 1 < NWD ? w[r][n + 1 < NWD ? n + 1 : n] : 0u, sh[r]);
    uint32_t x[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int bit = k * C * 8, n = bit >> 5;
      const uint32_t hi = n + 1 < NWD ? v[n + 1 < NWD ? n + 1 : n] : 0u;
      x[k] = __funnelshift_r(v[n], hi, bit & 31) & (C == 4 ? 0xFFFFFFFFu : (1u << (C * 8)) - 1u);
    }
    // column 0 has no left neighbour: it stands in for it
    p[0] = x[0];
#pragma unroll
    for (int k = 1; k < 6; ++k) p[k] = j0 > 0 ? x[k] : x[k - 1];
  };
  uint32_t up[6], mid[6], dn[6];
  pixels(0, up);
  pixels(1, mid);
#pragma unroll
  for (int r = 0; r < ENERGY_ROWS; ++r) {
    pixels(r + 2, dn);
    const int i = i0 + r;
    uint32_t e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t right = j0 + k + 1 < W ? mid[k + 2] : mid[k + 1];
      e[k] = sad4(right, mid[k]) + sad4(dn[k + 1], up[k + 1]);
    }
    if (i < H) {
      uint16_t *o = E + (int64_t)i * W + j0;
      if ((W & 3) == 0 && ((uintptr_t)E & 7u) == 0) {
        *reinterpret_cast<uint2 *>(o) = make_uint2(e[0] | (e[1] << 16), e[2] | (e[3] << 16));
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (j0 + k < W) o[k] = (uint16_t)e[k];
      }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      up[k] = mid[k];
      mid[k] = dn[k];
    }
  }
}

// ---- forward energy: the CU, DL, DR planes (plane p at E + p * pstride) ----
__global__ void k_forward(const uint32_t *__restrict__ img, int pitch, int H, int W, uint16_t *__restrict__ E, int pe,
                          int64_t pstride) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (j >= W || i >= H) return;
  uint32_t cu, dl, dr;
  forward_at([&](int r, int c) { return img[(int64_t)r * pitch + c]; }, W, i, j, cu, dl, dr);
  E[(int64_t)i * pe + j] = (uint16_t)cu;
  E[pstride + (int64_t)i * pe + j] = (uint16_t)dl;
  E[2 * pstride + (int64_t)i * pe + j] = (uint16_t)dr;
  // the search from the bottom steps out of the row below the last one, which has no costs (where the planes
  // have no such row, the next plane's row 0 holds zeros, or a tensor copy reads them)
  if (i == H - 1 && (int64_t)H * pe < pstride) E[pstride + (int64_t)H * pe + j] = 0;
}

// ---- caller forward planes -> padded layout. DL in row 0 and column 0 and DR in row 0 and the
// last column are never used (no such predecessor) and are stored as 0. A cell whose
// CU + max(DL, DR) exceeds `limit` sets the map's gate: its seam sums may not fit the 24-bit cost
// field, and the wide-cost search takes the map (one atomic per warp). ----
__global__ void k_copy_planes(const uint16_t *__restrict__ cu, const uint16_t *__restrict__ dl,
                              const uint16_t *__restrict__ dr, int H, int W, uint16_t *__restrict__ E, int pe,
                              int64_t pstride, uint32_t limit, int *gate) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  bool over = false;
  if (j < W && i < H) {
    const int64_t q = (int64_t)i * W + j;
    const uint32_t u = cu[q];
    const uint32_t l = (i >= 1 && j >= 1) ? dl[q] : 0u;
    const uint32_t r = (i >= 1 && j + 1 < W) ? dr[q] : 0u;
    E[(int64_t)i * pe + j] = (uint16_t)u;
    E[pstride + (int64_t)i * pe + j] = (uint16_t)l;
    E[2 * pstride + (int64_t)i * pe + j] = (uint16_t)r;
    over = u + (l > r ? l : r) > limit;
  }
  if (__any_sync(0xffffffffu, over) && (threadIdx.x & 31) == 0) atomicOr(gate, ERR_ENERGY_RANGE);
}

// ---- caller energy -> padded layout; an energy above `limit` sets the map's gate (its seam sums
// may not fit the 24-bit cost field: the wide-cost search takes the map; one atomic per warp) ----
__global__ void k_copy_energy(const uint16_t *__restrict__ src, int H, int W, uint16_t *__restrict__ E, int pe,
                              uint32_t limit, int *gate) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  bool over = false;
  if (j < W && i < H) {
    const uint16_t v = src[(int64_t)i * W + j];
    E[(int64_t)i * pe + j] = v;
    over = v > limit;
  }
  if (__any_sync(0xffffffffu, over) && (threadIdx.x & 31) == 0) atomicOr(gate, ERR_ENERGY_RANGE);
}

__global__ void k_unpad_energy(const uint16_t *__restrict__ E, int pe, int H, int W, uint16_t *__restrict__ dst) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (j >= W || i >= H) return;
  dst[(int64_t)i * W + j] = E[(int64_t)i * pe + j];
}

// ---- the per-seam refresh, one warp per row: the refreshed energy pair through the pending-removal
// lists, the removal added to the row's list, the energy row's tail shifted left past the seam ----
// It sits between one seam's search and the next, so what counts is its chain of memory round trips
// after the seam is known. Launched as a programmatic dependent it is resident while the search runs,
// and the search starts its dependents only after it has itself waited for the kernel before it: the
// energies, lists and image words are then in their final state (nothing writes them until this kernel
// does), complete in L2, where the search's wait left them; only this kernel's own wait would say
// anything of an SM's L1, so these loads go past it. So everything that does not need the seam is loaded
// before the wait: the whole energy row into registers (R chunks of 8 elements per lane) and the three
// rows' lists. After the wait: the
// seam columns, one round trip; the tail goes out of the registers while eight lanes fetch the eight
// pixels of the refreshed pair, a second one. From the end of the search to the end of the refresh:
// 1920x1080 5.5 -> 3.2 us (carve 14.6 -> 12.6 ms), 1279x853 4.9 -> 3.1 us (carve 11.6 -> 9.7 ms).
template <int R>
__global__ void __launch_bounds__(256) k_refresh(const uint32_t *__restrict__ img, int pitch, uint16_t *E, int pe, int H,
                                                 int W, const int32_t *__restrict__ seam,
                                                 const int16_t *__restrict__ lists_in, int16_t *__restrict__ lists_out,
                                                 int m, int *err) {
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  pdl_launch_dependents();
  if (i >= H) return;
  uint16_t *const er = E + (int64_t)i * pe;
  const int c_hi = (W - 2) >> 3;   // the chunk holding the new last column
  uint4 x[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int c = lane + 32 * r;
    x[r] = make_uint4(0u, 0u, 0u, 0u);
    if (c <= c_hi + 1) x[r] = __ldcg(reinterpret_cast<const uint4 *>(er + 8 * c));
  }
  const RefreshLane f = refresh_lane(lists_in, m, H, i, lane);
  pdl_wait_prerequisites();   // the seam of the search that precedes this launch
  const int s = __ldcg(seam + i);
  const int sr = __ldcg(seam + f.row);
  if (s < 0 || s >= W) {
    if (lane == 0) atomicOr(err, ERR_BAD_SEAM);
    return;
  }
  const uint32_t px = refresh_pixel(f, img, pitch, W, s, sr, lane);
  if (lane == 0) list_insert(f.list, lists_out + (int64_t)i * RPEND, s);
  if (s < W - 1) {
    const int c_lo = s >> 3;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      // the first element of the next chunk: lane + 1's, or the first lane's next one
      const uint32_t first = (lane == 0 && r + 1 < R) ? x[r + 1 < R ? r + 1 : r].x : x[r].x;
      const uint32_t nx = __shfl_sync(0xffffffffu, first, (lane + 1) & 31);
      const int c = lane + 32 * r;
      if (c >= c_lo && c <= c_hi) *reinterpret_cast<uint4 *>(er + 8 * c) = shift_chunk(x[r], nx, s - 8 * c);
    }
  }
  __syncwarp();   // the pair goes over the chunk holding s
  const uint32_t e = refresh_energy(px);
  if (lane == 0 && s >= 1) er[s - 1] = (uint16_t)e;
  if (lane == 4 && s <= W - 2) er[s] = (uint16_t)e;
}

// rows wider than the registers hold: chunk by chunk, everything after the wait
__global__ void k_refresh_wide(const uint32_t *__restrict__ img, int pitch, uint16_t *__restrict__ E, int pe, int H, int W,
                               const int32_t *__restrict__ seam, const int16_t *__restrict__ lists_in,
                               int16_t *__restrict__ lists_out, int m, int *err) {
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  pdl_launch_dependents();
  if (i >= H) return;
  const RefreshLane f = refresh_lane(lists_in, m, H, i, lane);
  pdl_wait_prerequisites();
  const int s = seam[i], sr = seam[f.row];
  if (s < 0 || s >= W) {
    if (lane == 0) atomicOr(err, ERR_BAD_SEAM);
    return;
  }
  uint16_t *const er = E + (int64_t)i * pe;
  const uint32_t px = refresh_pixel(f, img, pitch, W, s, sr, lane);
  if (lane == 0) list_insert(f.list, lists_out + (int64_t)i * RPEND, s);
  shift_row_u16(er, s, W, lane);
  const uint32_t e = refresh_energy(px);
  if (lane == 0 && s >= 1) er[s - 1] = (uint16_t)e;
  if (lane == 4 && s <= W - 2) er[s] = (uint16_t)e;
}

// The same for the three forward-energy planes (plane p at E + p * pstride; R chunks per lane and plane): lanes
// 0..2 fetch the pixels left and right of and above the new column s-1, lanes 4..6 those of column s.
template <int R>
__global__ void __launch_bounds__(128) k_refresh_fwd(const uint32_t *__restrict__ img, int pitch, uint16_t *E, int pe,
                                                     int64_t pstride, int H, int W, const int32_t *__restrict__ seam,
                                                     const int16_t *__restrict__ lists_in,
                                                     int16_t *__restrict__ lists_out, int m, int *err) {
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  pdl_launch_dependents();
  if (i >= H) return;
  uint16_t *const er = E + (int64_t)i * pe;
  const int c_hi = (W - 2) >> 3;   // the chunk holding the new last column
  uint4 x[3][R];
#pragma unroll
  for (int pl = 0; pl < 3; ++pl)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int c = lane + 32 * r;
      x[pl][r] = make_uint4(0u, 0u, 0u, 0u);
      if (c <= c_hi + 1) x[pl][r] = __ldcg(reinterpret_cast<const uint4 *>(er + pl * pstride + 8 * c));
    }
  const int row = (lane & 2) ? max(i - 1, 0) : i;
  const LazyRow list = lazy_row_l2(lists_in + (int64_t)row * RPEND, m);
  pdl_wait_prerequisites();   // the seam of the search that precedes this launch
  const int s = __ldcg(seam + i);
  const int sr = __ldcg(seam + row);
  if (s < 0 || s >= W) {
    if (lane == 0) atomicOr(err, ERR_BAD_SEAM);
    return;
  }
  const int col = (lane & 4) ? s : s - 1;   // the new column this lane works for
  const int j = clampi((lane & 2) ? col : ((lane & 1) ? col + 1 : col - 1), 0, W - 2);
  const int xs = j + (j >= sr ? 1 : 0);     // column in the width-W image
  const uint32_t px = img[(int64_t)row * pitch + xs + lazy_count(list, xs)];
  if (lane == 0) list_insert(list, lists_out + (int64_t)i * RPEND, s);
  if (s < W - 1) {
    const int c_lo = s >> 3;
#pragma unroll
    for (int pl = 0; pl < 3; ++pl)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const uint32_t first = (lane == 0 && r + 1 < R) ? x[pl][r + 1 < R ? r + 1 : r].x : x[pl][r].x;
        const uint32_t nx = __shfl_sync(0xffffffffu, first, (lane + 1) & 31);
        const int c = lane + 32 * r;
        if (c >= c_lo && c <= c_hi)
          *reinterpret_cast<uint4 *>(er + pl * pstride + 8 * c) = shift_chunk(x[pl][r], nx, s - 8 * c);
      }
  }
  __syncwarp();   // the refreshed values go over the chunk holding s
  const uint32_t pl = __shfl_sync(0xffffffffu, px, lane & 4), pr = __shfl_sync(0xffffffffu, px, (lane & 4) | 1),
                 up = __shfl_sync(0xffffffffu, px, (lane & 4) | 2);
  const bool left = col >= 1, right = col + 1 < W - 1;
  const uint32_t cu = left && right ? sad4(pr, pl) : 0u, dl = i >= 1 && left ? sad4(up, pl) : 0u,
                 dr = i >= 1 && right ? sad4(up, pr) : 0u;
  const int plane = lane & 3;
  if (lane < 8 && plane < 3 && col >= 0 && col <= W - 2)
    er[plane * pstride + col] = (uint16_t)(plane == 0 ? cu : (plane == 1 ? dl : dr));
}

__global__ void k_refresh_fwd_wide(const uint32_t *__restrict__ img, int pitch, uint16_t *__restrict__ E, int pe,
                              int64_t pstride, int H, int W, const int32_t *__restrict__ seam,
                              const int16_t *__restrict__ lists_in, int16_t *__restrict__ lists_out, int m, int *err) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  pdl_launch_dependents();
  pdl_wait_prerequisites();
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < H; i += warps)
    if (!refresh_row_fwd(img, pitch, E, pe, pstride, H, W, seam, lists_in, lists_out, m, i, lane) && lane == 0)
      atomicOr(err, ERR_BAD_SEAM);
}

__global__ void k_compact_lazy(uint32_t *__restrict__ img, int pitch, int H, int w, const int16_t *__restrict__ lists,
                               int m) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  pdl_launch_dependents();
  pdl_wait_prerequisites();
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < H; i += warps)
    compact_row_lazy(img + (int64_t)i * pitch, lists + (int64_t)i * RPEND, m, w, lane);
}

// ---- launchers ----
// launch as a programmatic dependent of the previous kernel on the stream (the kernels of the seam
// loop wait for their predecessor with griddepcontrol.wait before touching its results)
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), int blocks, int threads, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

static int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > 152 * 64) b = 152 * 64;
  return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_pack(const uint8_t *src, int H, int W, int C, uint32_t *img, int pitch, cudaStream_t st) {
  k_pack<<<grid_for((int64_t)H * W, 256), 256, 0, st>>>(src, H, W, C, img, pitch);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const uint32_t *img, int pitch, int H, int W, int C, bool transposed, uint8_t *dst,
                          cudaStream_t st) {
  (void)transposed;  // the caller transposes first when needed
  k_unpack<<<grid_for((int64_t)H * W, 256), 256, 0, st>>>(img, pitch, H, W, C, dst);
  return cudaGetLastError();
}

cudaError_t launch_transpose(const uint32_t *src, int ps, int H, int W, uint32_t *dst, int pd, cudaStream_t st) {
  dim3 grid((W + 31) / 32, (H + 31) / 32), block(32, 8);
  k_transpose<<<grid, block, 0, st>>>(src, ps, H, W, dst, pd);
  return cudaGetLastError();
}

cudaError_t launch_energy(const uint32_t *img, int pitch, int H, int W, uint16_t *E, int pe, cudaStream_t st) {
  dim3 grid((W + 127) / 128, H);
  k_energy<<<grid, 128, 0, st>>>(img, pitch, H, W, E, pe);
  return cudaGetLastError();
}

cudaError_t launch_energy_bytes(const uint8_t *src, int H, int W, int C, uint16_t *E, cudaStream_t st) {
  if (H > 65535) return cudaErrorInvalidConfiguration;   // rows are a grid dimension
  const int threads = W > 256 ? 128 : 32;
  const dim3 grid(((W + 3) / 4 + threads - 1) / threads, (H + ENERGY_ROWS - 1) / ENERGY_ROWS);
  if (C == 1) k_energy_bytes<1><<<grid, threads, 0, st>>>(src, H, W, E);
  else if (C == 3) k_energy_bytes<3><<<grid, threads, 0, st>>>(src, H, W, E);
  else k_energy_bytes<4><<<grid, threads, 0, st>>>(src, H, W, E);
  return cudaGetLastError();
}

cudaError_t launch_copy_energy(const uint16_t *src, int H, int W, uint16_t *E, int pe, int *gate, cudaStream_t st) {
  // the 24-bit search keeps costs below 2^24: every seam sum must fit
  const uint32_t limit = (uint32_t)((((uint64_t)1 << 24) - 1) / (uint64_t)H);
  dim3 grid((W + 127) / 128, H);
  k_copy_energy<<<grid, 128, 0, st>>>(src, H, W, E, pe, limit, gate);
  return cudaGetLastError();
}

cudaError_t launch_forward(const uint32_t *img, int pitch, int H, int W, uint16_t *E, int pe, int64_t pstride,
                           cudaStream_t st) {
  dim3 grid((W + 127) / 128, H);
  k_forward<<<grid, 128, 0, st>>>(img, pitch, H, W, E, pe, pstride);
  return cudaGetLastError();
}

cudaError_t launch_copy_planes(const uint16_t *cu, const uint16_t *dl, const uint16_t *dr, int H, int W, uint16_t *E,
                               int pe, int64_t pstride, int *gate, cudaStream_t st) {
  const uint32_t limit = (uint32_t)((((uint64_t)1 << 24) - 1) / (uint64_t)H);
  dim3 grid((W + 127) / 128, H);
  k_copy_planes<<<grid, 128, 0, st>>>(cu, dl, dr, H, W, E, pe, pstride, limit, gate);
  return cudaGetLastError();
}

cudaError_t launch_unpad_energy(const uint16_t *E, int pe, int H, int W, uint16_t *dst, cudaStream_t st) {
  dim3 grid((W + 127) / 128, H);
  k_unpad_energy<<<grid, 128, 0, st>>>(E, pe, H, W, dst);
  return cudaGetLastError();
}

}  // namespace sc

namespace sc {

cudaError_t launch_refresh(const uint32_t *img, int pitch, uint16_t *E, int pe, int H, int W, const int32_t *seam,
                           const int16_t *lists_in, int16_t *lists_out, int m, int *err, cudaStream_t st) {
  // registers for rows up to 1024, 2048 or 4096 elements
  auto *const k = W <= 1024 ? k_refresh<4> : (W <= 2048 ? k_refresh<8> : (W <= 4096 ? k_refresh<16> : k_refresh_wide));
  // rows per block: small blocks start and end sooner (per seam, blocks of 8 / 4 / 2 / 1 rows: 1920x1080 24.25 /
  // 23.9 / 24.1 / 24.1 us, 700x500 15.1 / 14.6 / 14.6 / 14.7; 3840x2160 makes no difference)
  const int rows = W <= 2048 ? 4 : 8;
  return launch_pdl(k, (H + rows - 1) / rows, 32 * rows, st, img, pitch, E, pe, H, W, seam, lists_in, lists_out, m, err);
}

cudaError_t launch_refresh_fwd(const uint32_t *img, int pitch, uint16_t *E, int pe, int64_t pstride, int H, int W,
                               const int32_t *seam, const int16_t *lists_in, int16_t *lists_out, int m, int *err,
                               cudaStream_t st) {
  if (W <= 1024)
    return launch_pdl(k_refresh_fwd<4>, (H + 3) / 4, 128, st, img, pitch, E, pe, pstride, H, W, seam, lists_in, lists_out,
                      m, err);
  if (W <= 2048)
    return launch_pdl(k_refresh_fwd<8>, (H + 3) / 4, 128, st, img, pitch, E, pe, pstride, H, W, seam, lists_in, lists_out,
                      m, err);
  // three planes of wider rows do not fit the registers: everything after the wait
  const int warps_per_block = 8;
  int blocks = (H + warps_per_block - 1) / warps_per_block;
  if (blocks > 152 * 8) blocks = 152 * 8;
  return launch_pdl(k_refresh_fwd_wide, blocks, warps_per_block * 32, st, img, pitch, E, pe, pstride, H, W, seam, lists_in,
                    lists_out, m, err);
}

cudaError_t launch_compact_lazy(uint32_t *img, int pitch, int H, int w, const int16_t *lists, int m, cudaStream_t st) {
  const int warps_per_block = 8;
  int blocks = (H + warps_per_block - 1) / warps_per_block;
  if (blocks > 152 * 8) blocks = 152 * 8;
  return launch_pdl(k_compact_lazy, blocks, warps_per_block * 32, st, img, pitch, H, w, lists, m);
}

}  // namespace sc

namespace sc {

// ---- Algorithm 2 (greedy): start at the leftmost minimum of the bottom row, climb by the
// leftmost minimum of the (in-range) upper neighbours. One warp per map: the bottom-row argmin is a
// warp reduction; the climb is serial, so the warp stages the 65-column window it can reach in
// the next 32 rows into shared memory and lane 0 walks it. ----
constexpr int GREEDY_ROWS = 32;
constexpr int GREEDY_COLS = 2 * GREEDY_ROWS + 1;

__global__ void __launch_bounds__(32) k_greedy(const uint16_t *__restrict__ e, int H, int W,
                                               int32_t *__restrict__ seam, int64_t *__restrict__ cost) {
  __shared__ uint32_t win[GREEDY_ROWS][GREEDY_COLS + 1];
  const int lane = threadIdx.x;
  unsigned long long best = ~0ull;   // (energy << 32) | column, leftmost minimum
  const uint16_t *last = e + (int64_t)(H - 1) * W;
  for (int j = lane; j < W; j += 32) {
    const unsigned long long k = ((unsigned long long)last[j] << 32) | (unsigned)j;
    best = k < best ? k : best;
  }
  for (int off = 16; off > 0; off >>= 1) {
    const unsigned long long o = __shfl_xor_sync(0xffffffffu, best, off);
    best = o < best ? o : best;
  }
  int j = (int)(best & 0xFFFFFFFFu);
  int64_t total = (int64_t)(best >> 32);
  if (lane == 0) seam[H - 1] = j;
  for (int top = H - 1; top > 0; top -= GREEDY_ROWS) {
    const int rows = top < GREEDY_ROWS ? top : GREEDY_ROWS;   // rows top-1 .. top-rows
    const int c0 = j - GREEDY_ROWS;
    // stage 8 rows at a time with all their loads in flight (3 columns per lane per row)
    for (int rb = 0; rb < rows; rb += 8) {
      uint32_t v[8][3];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int r = rb + q;
        const uint16_t *row = e + (int64_t)(top - 1 - (r < rows ? r : 0)) * W;
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int c = lane + 32 * u, col = c0 + c;
          v[q][u] = (r < rows && c < GREEDY_COLS && col >= 0 && col < W) ? (uint32_t)row[col] : 0x10000u;
        }
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int c = lane + 32 * u;
          if (rb + q < rows && c < GREEDY_COLS) win[rb + q][c] = v[q][u];   // 0x10000: above any energy
        }
      }
    }
    __syncwarp();
    if (lane == 0) {
      int x = j - c0;
      for (int r = 0; r < rows; ++r) {
        int b = x - 1;
        if (win[r][x] < win[r][b]) b = x;
        if (win[r][x + 1] < win[r][b]) b = x + 1;
        x = b;
        total += win[r][x];
        seam[top - 1 - r] = c0 + x;
      }
      j = c0 + x;
    }
    j = __shfl_sync(0xffffffffu, j, 0);
    __syncwarp();
  }
  if (lane == 0 && cost) *cost = total;
}

cudaError_t launch_greedy(const uint16_t *e, int H, int W, int32_t *seam, int64_t *cost, cudaStream_t st) {
  k_greedy<<<1, 32, 0, st>>>(e, H, W, seam, cost);
  return cudaGetLastError();
}

}  // namespace sc

namespace sc {

// ---- self-test of the bounded waits: one thread waits on an mbarrier that nothing completes,
// with a limit of limit_ns, exactly as the search's waits do; when the limit runs out it records
// ERR_TIMEOUT and returns (no trap, no fault), so the host sees SC_ETIMEOUT and the context stays
// usable. ----
__global__ void k_wait_selftest(uint64_t limit_ns, int *err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);   // one arrival expected; none comes
  fence_mbar_init();
  if (!mbar_wait_bounded(&bar, 0u, limit_ns)) atomicOr(err, ERR_TIMEOUT);
}

cudaError_t launch_wait_selftest(uint64_t limit_ns, int *err, cudaStream_t st) {
  k_wait_selftest<<<1, 32, 0, st>>>(limit_ns, err);
  return cudaGetLastError();
}

}  // namespace sc
