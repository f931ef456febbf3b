// Per-pixel and per-row operations shared by the whole-image kernels (sc_kernels.cu) and the
// batched persistent kernel (sc_batch.cuh): the e1 energy of a pixel ("Energy Mapping", item e1),
// the two refreshed energies of a row after a removal, and the row compactions ("Removal of
// Seams"). Pixels are uint32 words, channel c in byte c (unused bytes 0).
#pragma once
#include <cstdint>

#include "sc_ptx.cuh"

namespace sc {

// sum over the four bytes of |a_b - b_b|
__device__ __forceinline__ uint32_t sad4(uint32_t a, uint32_t b) { return __vsadu4(a, b); }

__device__ __forceinline__ int clampi(int x, int lo, int hi) { return x < lo ? lo : (x > hi ? hi : x); }

// e1 energy of pixel (i, j) of a rows x cols word image with edge replication
__device__ __forceinline__ uint32_t energy_at(const uint32_t *img, int pitch, int rows, int cols, int i, int j) {
  const uint32_t *row = img + (int64_t)i * pitch;
  const int jl = j > 0 ? j - 1 : 0, jr = j + 1 < cols ? j + 1 : cols - 1;
  const int iu = i > 0 ? i - 1 : 0, id = i + 1 < rows ? i + 1 : rows - 1;
  return sad4(row[jr], row[jl]) + sad4(img[(int64_t)id * pitch + j], img[(int64_t)iu * pitch + j]);
}

// Eight uint16 elements x moved down one, the first of the next eight (nx, low half) shifted in; the
// leading `keep` elements (none when keep <= 0) stay where they are.
__device__ __forceinline__ uint4 shift_chunk(const uint4 &x, uint32_t nx, int keep) {
  uint4 o;
  o.x = __funnelshift_r(x.x, x.y, 16);
  o.y = __funnelshift_r(x.y, x.z, 16);
  o.z = __funnelshift_r(x.z, x.w, 16);
  o.w = __funnelshift_r(x.w, nx, 16);
  // (branch-free: a warp whose lane 0 took a branch here would wait for it on every row)
  auto merge = [keep](uint32_t in, uint32_t sh, int q) {
    const uint32_t m = keep > 2 * q + 1 ? 0xFFFFFFFFu : (keep > 2 * q ? 0x0000FFFFu : 0u);
    return (in & m) | (sh & ~m);
  };
  o.x = merge(x.x, o.x, 0);
  o.y = merge(x.y, o.y, 1);
  o.z = merge(x.z, o.z, 2);
  o.w = merge(x.w, o.w, 3);
  return o;
}

// In-place left shift by one of a 16-byte-aligned uint16 row, row[s+1 .. W-1] -> row[s .. W-2],
// by one warp, 8 elements (one 16-byte load and store) at a time: chunk c of the result is chunk c of the input moved down one element, with the first
// element of chunk c+1 shifted in; every lane reads its chunks and the element after each chunk
// before any lane of the warp writes. The first chunk keeps its elements left of s. Elements from
// W-1 to the end of the last chunk are left undefined (they lie in the row's padding or in the
// column that the shift drops).
__device__ __forceinline__ void shift_row_u16(uint16_t *row, int s, int W, int lane) {
  constexpr int R = 4;
  if (s >= W - 1) return;
  const int c_lo = s >> 3, c_hi = (W - 2) >> 3;
  for (int cb = c_lo; cb <= c_hi; cb += 32 * R) {
    uint4 x[R];
    uint32_t nx[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int c = cb + r * 32 + lane;
      if (c <= c_hi) {
        x[r] = *reinterpret_cast<const uint4 *>(row + 8 * c);
        nx[r] = row[8 * c + 8];
      }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int c = cb + r * 32 + lane;
      if (c <= c_hi) {
        *reinterpret_cast<uint4 *>(row + 8 * c) = shift_chunk(x[r], nx[r], s - 8 * c);
      }
    }
    __syncwarp();
  }
}

__device__ __forceinline__ uint32_t pack_pixel(const uint8_t *s, int C) {
  uint32_t w = s[0];
  if (C >= 3) w |= ((uint32_t)s[1] << 8) | ((uint32_t)s[2] << 16);
  if (C == 4) w |= (uint32_t)s[3] << 24;
  return w;
}

__device__ __forceinline__ void unpack_pixel(uint32_t w, uint8_t *d, int C) {
  d[0] = (uint8_t)w;
  if (C >= 3) {
    d[1] = (uint8_t)(w >> 8);
    d[2] = (uint8_t)(w >> 16);
  }
  if (C == 4) d[3] = (uint8_t)(w >> 24);
}

}  // namespace sc

namespace sc {

// ---- lazy compaction of the image words ----
// The stored words of a row are compacted only every RPEND seams. Between compactions each row
// keeps the sorted stored columns o_0 < o_1 < ... < o_(m-1) of its m removed pixels. Current column
// j (after the m removals) is stored column j + #{q : o_q - q <= j}: o_q - q is the number of kept
// pixels left of o_q, so the q-th removal is passed exactly when j reaches it.
constexpr int RPEND = 16;

// A row's pending removals in registers: the thresholds t_q = o_q - q, two 16-bit values per word,
// from two 16-byte loads (the lists are 32-byte rows); entries q >= m get t_q = 0x7FFF, above every
// column (columns stay below 2^15). Current column j is stored column j + #{q : t_q <= j}. A count
// is four instructions per word: for 16-bit halves a = 0x8000 + j and b = t_q <= 0x7FFF, a - b
// stays in [1, 0xFFFF] (no borrow between halves) and has bit 15 set exactly when t_q <= j.
// No load per entry on the way to a pixel.
struct LazyRow {
  uint32_t t[RPEND / 2];
};

__device__ __forceinline__ LazyRow lazy_row_of(const uint4 a, const uint4 b, int m) {
  const uint32_t w[RPEND / 2] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  LazyRow r;
#pragma unroll
  for (int k = 0; k < RPEND / 2; ++k) {
    // entries past m become 0x7FFF + q before the subtraction (o_q >= q for the others: no borrow)
    const uint32_t lo = (2 * k < m) ? (w[k] & 0xFFFFu) : 0x7FFFu + 2 * k;
    const uint32_t hi = (2 * k + 1 < m) ? (w[k] >> 16) : 0x7FFFu + 2 * k + 1;
    r.t[k] = (lo | (hi << 16)) - ((uint32_t)(2 * k) | ((uint32_t)(2 * k + 1) << 16));
  }
  return r;
}

__device__ __forceinline__ LazyRow lazy_row(const int16_t *list, int m) {
  const uint4 *const p = reinterpret_cast<const uint4 *>(list);
  return lazy_row_of(p[0], p[1], m);
}
// past L1: for the loads a kernel makes ahead of its griddepcontrol.wait
__device__ __forceinline__ LazyRow lazy_row_l2(const int16_t *list, int m) {
  const uint4 *const p = reinterpret_cast<const uint4 *>(list);
  return lazy_row_of(__ldcg(p), __ldcg(p + 1), m);
}

// removals passed by current column j (0 <= j < 2^15)
__device__ __forceinline__ int lazy_count(const LazyRow &r, int j) {
  const uint32_t jj = ((uint32_t)j * 0x10001u) | 0x80008000u;
  int c = 0;
#pragma unroll
  for (int k = 0; k < RPEND / 2; ++k) c += __popc((jj - r.t[k]) & 0x80008000u);
  return c;
}

// The two energies of row i that the removal of `seam` changes. After deleting seam s from a
// W-wide image, the energy of the (W-1)-wide image equals the old energy shifted left past s_i,
// except at the new columns s_i - 1 and s_i (their left/right neighbour changed, and, since
// |s_i - s_(i+-1)| <= 1, they are the only pixels whose upper/lower neighbour can change). They
// are computed from the old image seen through the removal: new pixel (r, j) = old (r, j + [j >= s_r]).
// Returns (e(s-1) | e(s) << 16); a value is 0 when its column does not exist. The image is read
// through the pending-removal lists of the width-W image the seam was found in: lc is row i's (seam
// column s), lu and ld those of the rows above and below, iu and id (edge rows replicated), whose
// seam columns are su and sd.
__device__ __forceinline__ uint32_t patch_pair(const uint32_t *img, int pitch, int W, int i, int s, int iu, int su,
                                               const LazyRow &lu, const LazyRow &lc, int id, int sd,
                                               const LazyRow &ld) {
  const int Wn = W - 1;
  // new pixel (r, j), j clamped to the new width, of a row r whose seam column is sr and list L
  auto pix = [&](int r, const LazyRow &L, int sr, int j) -> uint32_t {
    j = clampi(j, 0, Wn - 1);
    const int x = j + (j >= sr ? 1 : 0);                    // column in the width-W image
    return img[(int64_t)r * pitch + x + lazy_count(L, x)];
  };
  // columns s-1 and s of the rows above and below (edge rows replicated)
  const uint32_t up0 = pix(iu, lu, su, s - 1), up1 = pix(iu, lu, su, s);
  const uint32_t dn0 = pix(id, ld, sd, s - 1), dn1 = pix(id, ld, sd, s);
  const uint32_t p0 = (s >= 1) ? sad4(pix(i, lc, s, s), pix(i, lc, s, s - 2)) + sad4(dn0, up0) : 0u;
  const uint32_t p1 = (s <= Wn - 1) ? sad4(pix(i, lc, s, s + 1), pix(i, lc, s, s - 1)) + sad4(dn1, up1) : 0u;
  return p0 | (p1 << 16);
}

// patch_pair of row i, its seam columns and lists read here (lists: row r at lists + r*RPEND, m
// entries each); row i's list comes back in *li for the insertion that follows, and *bad is set
// when the seam column is out of range.
__device__ __forceinline__ uint32_t patch_row_lazy(const uint32_t *img, int pitch, int H, int W, const int32_t *seam,
                                                   const int16_t *lists, int m, int i, bool *bad, LazyRow *li) {
  const int s = seam[i];
  *li = lazy_row(lists + (int64_t)i * RPEND, m);
  if (s < 0 || s >= W) {
    *bad = true;
    return 0u;
  }
  const int iu = i > 0 ? i - 1 : 0, id = i + 1 < H ? i + 1 : H - 1;
  const LazyRow lu = lazy_row(lists + (int64_t)iu * RPEND, m);
  const LazyRow ld = lazy_row(lists + (int64_t)id * RPEND, m);
  return patch_pair(img, pitch, W, i, s, iu, seam[iu], lu, *li, id, seam[id], ld);
}

// Add a row's removal at current column s to its sorted list (L: the row's m entries): the removals
// it passes are exactly the first c = lazy_count(s) (t_q never decreases with q), so the stored
// column o = s + c goes in at position c. out gets m + 1 entries (two 16-byte stores).
__device__ __forceinline__ void list_insert(const LazyRow &L, int16_t *out, int s) {
  const int c = lazy_count(L, s);
  const uint32_t o = (uint32_t)(s + c);
  uint32_t raw[RPEND / 2], v[RPEND / 2];
#pragma unroll
  for (int k = 0; k < RPEND / 2; ++k) raw[k] = L.t[k] + ((uint32_t)(2 * k) | ((uint32_t)(2 * k + 1) << 16));   // o_q
#pragma unroll
  for (int k = 0; k < RPEND / 2; ++k) {
    const uint32_t up = k > 0 ? __funnelshift_l(raw[k - 1], raw[k], 16) : (raw[0] << 16);   // entries moved up one
    uint32_t x = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = 2 * k + h;
      const uint32_t keep = (raw[k] >> (16 * h)) & 0xFFFFu, moved = (up >> (16 * h)) & 0xFFFFu;
      x |= (q < c ? keep : (q == c ? o : moved)) << (16 * h);
    }
    v[k] = x;
  }
  *reinterpret_cast<uint4 *>(out) = make_uint4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<uint4 *>(out + 8) = make_uint4(v[4], v[5], v[6], v[7]);
}

// The refreshed pairs and pending-removal list updates of the rows one thread handles (local rows
// q = t0, t0 + tstride, ... of nq; image row row0 + q * rstride): pairs[q] gets row q's pair (as
// patch_row_lazy) and lists_out its list with this seam's removal added. Returns true when a seam
// column was out of range (the rows after it are left alone).
__device__ __forceinline__ bool refresh_pairs(const uint32_t *img, int pitch, int H, int W, const int32_t *seam,
                                           const int16_t *lists_in, int16_t *lists_out, int m, int nq, int row0,
                                           int rstride, uint32_t *pairs, int t0, int tstride) {
  bool bad = false;
#pragma unroll 1
  for (int q = t0; q < nq; q += tstride) {
    const int i = row0 + q * rstride;
    LazyRow li;
    pairs[q] = patch_row_lazy(img, pitch, H, W, seam, lists_in, m, i, &bad, &li);
    if (!bad) list_insert(li, lists_out + (size_t)i * RPEND, seam[i]);
  }
  return bad;
}

// Compact one row of stored words in place by one warp: current column j <- its stored column, for
// j < w. Sources never lie left of their destination and the row is processed left to right in
// chunks read completely before they are written, so nothing is overwritten before it is read.
__device__ __forceinline__ void compact_row_lazy(uint32_t *row, const int16_t *list, int m, int w, int lane) {
  constexpr int R = 4;
  int l[RPEND];   // o_q - q (the output column where the q-th removal is passed), padded high
#pragma unroll
  for (int q = 0; q < RPEND; ++q) l[q] = q < m ? (int)list[q] - q : 0x7FFFFFFF;
  int first = w;   // columns left of the first removal keep their place
  if (m > 0) first = l[0];
  for (int base = first; base < w; base += 32 * R) {
    uint32_t x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int j = base + r * 32 + lane;
      if (j < w) {
        int c = 0;
#pragma unroll
        for (int q = 0; q < RPEND; ++q) c += (l[q] <= j) ? 1 : 0;
        x[r] = row[j + c];
      }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int j = base + r * 32 + lane;
      if (j < w) row[j] = x[r];
    }
    __syncwarp();
  }
}

}  // namespace sc

namespace sc {

// The refreshed pair of row i by one warp, eight lanes fetching one pixel each (see patch_pair for what
// changes): lanes 0, 1 the new columns s and s-2 of the row itself and lanes 2, 3 column s-1 below and
// above, which make e(s-1); lanes 4, 5 columns s+1 and s-1 and lanes 6, 7 column s below and above,
// which make e(s). The other lanes repeat lanes 0..7.
struct RefreshLane {
  LazyRow list;   // pending removals of the lane's row
  int row;        // the row its pixel lies in (i, or a neighbour; edge rows replicated)
};
__device__ __forceinline__ RefreshLane refresh_lane(const int16_t *lists, int m, int H, int i, int lane) {
  RefreshLane f;
  const int q = lane & 7;
  f.row = (q & 2) == 0 ? i : ((q & 1) ? max(i - 1, 0) : min(i + 1, H - 1));
  f.list = lazy_row_l2(lists + (int64_t)f.row * RPEND, m);
  return f;
}
// the lane's pixel; s: row i's seam column, sr: that of the lane's row
__device__ __forceinline__ uint32_t refresh_pixel(const RefreshLane &f, const uint32_t *img, int pitch, int W, int s,
                                                  int sr, int lane) {
  const int q = lane & 7;
  // new column: s, s-2, s-1, s-1 | s+1, s-1, s, s
  const int j = clampi(s + ((q & 2) ? ((q & 4) ? 0 : -1) : ((q & 4) ? 1 : 0) - ((q & 1) ? 2 : 0)), 0, W - 2);
  const int x = j + (j >= sr ? 1 : 0);   // column in the width-W image
  return img[(int64_t)f.row * pitch + x + lazy_count(f.list, x)];
}
// from every lane's pixel: e(s-1) in lanes 0..3, e(s) in lanes 4..7
__device__ __forceinline__ uint32_t refresh_energy(uint32_t px) {
  const uint32_t d = sad4(px, __shfl_xor_sync(0xffffffffu, px, 1));
  return d + __shfl_xor_sync(0xffffffffu, d, 2);
}

// The energy shift of every row this warp owns (local rows q = warp, warp + nwarps, ... of nq; image
// row row0 + q * rstride), each followed by its refreshed pair (pairs[q]: e(s-1) | e(s) << 16), NR rows
// at a time through registers: a lane holds chunks cb + lane and cb + 32 + lane (8 elements each, cb first
// the chunk holding s) of each row, takes the element after each chunk from the next lane, and writes the
// chunk one element to the left; longer tails go on block by block from the left, each read before it
// is written. Rows whose seam is out of range are skipped (the caller records the error).
// Bound by the latency of its instruction stream: no branch depends on a row's tail length (a branch and
// its reconvergence per load and store cost as much as the loads: 1254x944 173.2 -> 170.9 us a seam,
// 2500x1332 98.2 -> 94.5 on its cluster), and nothing goes through shared memory. Against tails staged there
// by bulk copies and written back chunk by chunk, per seam of one image: 400x900 96.2 -> 90.8 us, 1254x944
// 176.1 -> 170.9 us, 2500x1332 on a cluster of 8-row tiles 223.6 -> 207.9. Slower: two rows of 6 chunks per
// lane, eight rows of one, four of four.
// Not inlined (nor is compact_rows_staged): a separate function gets its own register allocation, and inlined
// the two phases cost the one-CTA batched kernel ~160 bytes of spills.
static __device__ __noinline__ void shift_rows(uint16_t *E, int pe, int nq, int row0, int rstride, int w,
                                               const int32_t *seam, const uint32_t *pairs, int warp, int nwarps,
                                               int lane) {
  constexpr int R = 2, NR = 4;
  const int c_last = (w - 2) >> 3;   // the chunk holding the new last column
  const int nk = warp < nq ? (nq - warp + nwarps - 1) / nwarps : 0;
  const int64_t rowstep = (int64_t)nwarps * rstride * pe;
  uint16_t *e0 = E + (int64_t)(row0 + warp * rstride) * pe;   // the group's first row
#pragma unroll 1
  for (int k0 = 0; k0 < nk; k0 += 32) {
    const int kl = k0 + lane;
    const int sl = kl < nk ? seam[row0 + (warp + kl * nwarps) * rstride] : -1;
    const uint32_t pl = kl < nk ? pairs[warp + kl * nwarps] : 0u;
    const int n = min(32, nk - k0);
#pragma unroll 1
    for (int t = 0; t < n; t += NR, e0 += NR * rowstep) {
      int s[NR], cb[NR];
      uint16_t *er[NR];
      bool any = false;
#pragma unroll
      for (int v = 0; v < NR; ++v) {
        s[v] = __shfl_sync(0xffffffffu, sl, t + v);   // (t + v <= 31: t is a multiple of NR)
        er[v] = e0 + (t + v < n ? v : 0) * rowstep;
        // past the last row, a seam out of range, or one in the last column: nothing to shift
        cb[v] = (t + v >= n || s[v] < 0 || s[v] >= w - 1) ? c_last + 1 : s[v] >> 3;
        any |= cb[v] <= c_last;
      }
      while (any) {
        // no branches: lanes past the tail load its last chunk again, and only the stores are predicated
        uint4 x[NR][R];
        uint32_t after[NR];
#pragma unroll
        for (int v = 0; v < NR; ++v) {
#pragma unroll
          for (int r = 0; r < R; ++r)
            x[v][r] = __ldcg(reinterpret_cast<const uint4 *>(er[v] + 8 * min(cb[v] + 32 * r + lane, c_last + 1)));
          // the element after the block's last chunk
          after[v] = __ldcg(er[v] + 8 * min(cb[v] + 32 * R, c_last + 1));
        }
        any = false;
#pragma unroll
        for (int v = 0; v < NR; ++v) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const uint32_t first = lane > 0 ? x[v][r].x : (r + 1 < R ? x[v][r + 1 < R ? r + 1 : r].x : after[v]);
            const uint32_t nx = __shfl_sync(0xffffffffu, first, (lane + 1) & 31);
            const int c = cb[v] + 32 * r + lane;
            const uint4 o = shift_chunk(x[v][r], nx, r == 0 ? s[v] - 8 * c : 0);
            if (c <= c_last) *reinterpret_cast<uint4 *>(er[v] + 8 * c) = o;
          }
          cb[v] += 32 * R;
          any |= cb[v] <= c_last;
        }
      }
      __syncwarp();
      // the pairs, one lane per row
      const uint32_t pr = __shfl_sync(0xffffffffu, pl, (t + (lane & (NR - 1))) & 31);
      const int sr = __shfl_sync(0xffffffffu, sl, (t + (lane & (NR - 1))) & 31);
      if (lane < NR && t + lane < n && sr >= 0 && sr < w) {
        uint16_t *er = e0 + lane * rowstep;
        if (sr >= 1) er[sr - 1] = (uint16_t)(pr & 0xFFFFu);
        if (sr <= w - 2) er[sr] = (uint16_t)(pr >> 16);
      }
    }
  }
}

// compact_row_lazy for every row this warp owns (local rows q = warp, warp + nwarps, ... of nq;
// image row row0 + q * rstride), staged through a shared-memory buffer of buf_words words
// (16-byte aligned): the stored tail of a row is copied in with cp.async in pieces, then every
// output word is gathered from the buffer. The removals are held one per lane (o_q - q in lane q);
// for 32 consecutive outputs one ballot counts those left of the first and a second finds the few
// that fall inside, instead of comparing every output with every removal.
static __device__ __noinline__ void compact_rows_staged(uint32_t *img, int pitch, int nq, int row0, int rstride,
                                           const int16_t *lists, int m, int w, int warp, int nwarps, int lane,
                                           uint32_t *buf, int buf_words) {
  const int piece = ((buf_words - 24) / 32) * 32;   // outputs per staged piece
  for (int q = warp; q < nq; q += nwarps) {
    const int r = row0 + q * rstride;
    uint32_t *row = img + (int64_t)r * pitch;
    const int16_t *list = lists + (int64_t)r * RPEND;
    if (piece < 32) {   // no room to stage: the direct form
      compact_row_lazy(row, list, m, w, lane);
      continue;
    }
    const int lq = lane < m ? (int)list[lane] - lane : 0x7FFFFFFF;
    const int first = m > 0 ? __shfl_sync(0xffffffffu, lq, 0) : w;   // the list is sorted
    for (int j0 = first; j0 < w; j0 += piece) {
      const int j1 = min(w, j0 + piece);
      const int a = j0 & ~3, b = (j1 + m + 3) & ~3;   // stored words j0 .. j1 + m - 1, 16-byte aligned
      for (int x = a + 4 * lane; x < b; x += 128) cp_async16(buf + (x - a), row + x);
      cp_async_wait_all();
      __syncwarp();
      // 4 x 32 outputs at a time, their gathers in flight together
#pragma unroll 1
      for (int jb = j0; jb < j1; jb += 128) {
        uint32_t v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int b0 = jb + 32 * u, j = b0 + lane;
          int c = __popc(__ballot_sync(0xffffffffu, lq <= b0));
          unsigned in = __ballot_sync(0xffffffffu, lq > b0 && lq < b0 + 32);
          while (in) {
            const int bq = __ffs(in) - 1;
            in &= in - 1;
            const int lv = __shfl_sync(0xffffffffu, lq, bq);
            c += (j >= lv) ? 1 : 0;
          }
          v[u] = (j < j1) ? buf[j + c - a] : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (jb + 32 * u + lane < j1) row[jb + 32 * u + lane] = v[u];
      }
      __syncwarp();   // the buffer is reused by the next piece
    }
  }
}

// ---- forward energy ----
// The three cost planes of pixel (i, j) of a rows x cols word image: CU = |P(i,j+1) - P(i,j-1)|
// (0 at the first and last column), DL = |P(i-1,j) - P(i,j-1)| (0 in row 0 and column 0),
// DR = |P(i-1,j) - P(i,j+1)| (0 in row 0 and the last column), each summed over the channels.
// pix(r, c) returns the word of pixel (r, c) (r, c inside the image).
template <typename Pix>
__device__ __forceinline__ void forward_at(Pix pix, int cols, int i, int j, uint32_t &cu, uint32_t &dl, uint32_t &dr) {
  const bool left = j >= 1, right = j + 1 < cols;
  const uint32_t pl = left ? pix(i, j - 1) : 0u, pr = right ? pix(i, j + 1) : 0u;
  cu = (left && right) ? sad4(pr, pl) : 0u;
  dl = dr = 0u;
  if (i >= 1) {
    const uint32_t up = pix(i - 1, j);
    if (left) dl = sad4(up, pl);
    if (right) dr = sad4(up, pr);
  }
}

// The forward-energy planes at the new columns s-1 and s of row i after removing `seam` (the
// other columns are shifted copies: the dirty set of the e1 refresh holds for all three planes),
// the image read through the pending-removal lists. out[plane] = value(s-1) | value(s) << 16.
__device__ __forceinline__ void patch_row_lazy_fwd(const uint32_t *img, int pitch, int H, int W, const int32_t *seam,
                                                   const int16_t *lists, int m, int i, uint32_t (&out)[3], bool *bad,
                                                   LazyRow *li) {
  const int Wn = W - 1;
  const int iu = i > 0 ? i - 1 : 0;
  const int s = seam[i], su = seam[iu];
  const LazyRow lc = lazy_row(lists + (int64_t)i * RPEND, m);
  const LazyRow lu = lazy_row(lists + (int64_t)iu * RPEND, m);
  *li = lc;
  out[0] = out[1] = out[2] = 0u;
  if (s < 0 || s >= W) {
    *bad = true;
    return;
  }
  // rows i (forward_at's row) and i - 1 (read only when i >= 1)
  auto pix = [&](int r, int j) -> uint32_t {
    const LazyRow &L = r == i ? lc : lu;
    const int x = j + (j >= (r == i ? s : su) ? 1 : 0);      // column in the width-W image
    return img[(int64_t)r * pitch + x + lazy_count(L, x)];
  };
  uint32_t cu, dl, dr;
  if (s >= 1) {
    forward_at(pix, Wn, i, s - 1, cu, dl, dr);
    out[0] = cu; out[1] = dl; out[2] = dr;
  }
  if (s <= Wn - 1) {
    forward_at(pix, Wn, i, s, cu, dl, dr);
    out[0] |= cu << 16; out[1] |= dl << 16; out[2] |= dr << 16;
  }
}

// refresh_row for the three forward-energy planes (plane p at E + p * pstride)
__device__ __forceinline__ bool refresh_row_fwd(const uint32_t *img, int pitch, uint16_t *E, int pe, int64_t pstride,
                                                int H, int W, const int32_t *seam, const int16_t *lists_in,
                                                int16_t *lists_out, int m, int i, int lane) {
  const int s = seam[i];
  if (s < 0 || s >= W) return false;
  uint32_t pr[3] = {0u, 0u, 0u};
  if (lane == 0) {
    bool bad = false;
    LazyRow li;
    patch_row_lazy_fwd(img, pitch, H, W, seam, lists_in, m, i, pr, &bad, &li);
    list_insert(li, lists_out + (int64_t)i * RPEND, s);
  }
#pragma unroll
  for (int pl = 0; pl < 3; ++pl) {
    const uint32_t v = __shfl_sync(0xffffffffu, pr[pl], 0);
    uint16_t *er = E + pl * pstride + (int64_t)i * pe;
    shift_row_u16(er, s, W, lane);
    if (lane == 0) {
      if (s >= 1) er[s - 1] = (uint16_t)(v & 0xFFFFu);
      if (s <= W - 2) er[s] = (uint16_t)(v >> 16);
    }
  }
  return true;
}

}  // namespace sc
