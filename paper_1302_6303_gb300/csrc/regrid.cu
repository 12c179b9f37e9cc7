// Dynamic regridding (Sec. 5).
//
// nrd_regrid_boxes: Berger-Rigoutsos clustering of tagged cells into the
// boxes of a new hierarchy (host C++, off the stepping path).  Level by level
// from the coarsest: the cells of the new level l that carry a selected tag
// (a cell that does not exist on level l of the current hierarchy inherits
// the tag of the finest current cell that contains it) are dilated by
// `buffer` cells and kept only where a finer level can be properly nested
// (every level-l neighbour of the cell, inside the domain, belongs to the new
// level l).  The tagged set is clustered recursively:
//   shrink the box to the bounding box of its tags (drop it if none);
//   accept it when tags/volume >= efficiency, every cell may hold the finer
//   level, and no side exceeds max_side/2 cells;
//   otherwise cut it, trying in turn
//     (1) a zero of a tag signature (the count of tags per plane), axes taken
//         longest first, the zero nearest the middle (lower one on a tie);
//         the empty plane itself is dropped,
//     (2) the strongest sign change of the signature's second difference,
//         over all axes with at least 4 planes (first one on a tie),
//     (3) the middle of the longest side,
//   where a cut must leave both parts at least min_side/2 planes wide unless
//   the box holds cells that cannot take the finer level (then any cut is
//   allowed); a box that cannot be cut is accepted as it is.
// Accepted boxes, refined by 2, are the boxes of level l+1, in the order the
// recursion accepts them (lower part first).
//
// The tagged and nestable fields of a level and their summed-area tables are
// formed on the device (scatter, box filters, scans), for small levels on the
// host; the recursion reads the tables on the host, 8 entries per count.
//
// nrd_transfer: conservative limited-linear transfer of state vectors from an
// old to a new hierarchy, one device kernel that looks every new cell's source
// up in the old hierarchy's maps.  The
// old vectors are first made composite (covered cells := mean of their
// children).  A new cell that exists on the same level of the old hierarchy
// copies it; any other new cell evaluates, at its centre, the limited linear
// reconstruction of the old cell that contains it on the finest old level
// present there:
//   u = u_c + sum_d s_d (x_d - x_{c,d}) / h_{c,d},
//   s_d = minmod(u_c - u_{c-e_d}, u_{c+e_d} - u_c)  (0 if a neighbour is missing),
// whose mean over the children of the coarse cell is u_c (conservative) and
// which takes no value outside the neighbouring old values (no new extrema,
// so positivity is kept).
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <optional>
#include <string>
#include <vector>

#include "nrd_internal.h"

namespace {

struct IBox {
  int lo[3], hi[3];
  long vol() const {
    return (long)(hi[0] - lo[0] + 1) * (hi[1] - lo[1] + 1) * (hi[2] - lo[2] + 1);
  }
  int side(int d) const { return hi[d] - lo[d] + 1; }
};

// One axis of a box filter of a dense 0/1 field of n[0] x n[1] x n[2] cells:
// v[c] := AND (MIN) or OR (!MIN) of v over the cells within r of c along
// axis d that lie inside the field.  v is viewed as [outer][n[d]][inner],
// and each output row along the contiguous inner index combines 2r + 1
// input rows.
template <bool MIN>
void box_filter_t(std::vector<uint8_t>& v, const int n[3], int d, int r) {
  const long inner = d == 0 ? 1 : (d == 1 ? (long)n[0] : (long)n[0] * n[1]);
  const long outer = (long)v.size() / (inner * n[d]);
  const int m = n[d];
  std::vector<uint8_t> w(v.size());
  auto op = [](uint8_t a, uint8_t b) -> uint8_t { return MIN ? (a & b) : (a | b); };
  for (long o = 0; o < outer; o++) {
    const uint8_t* vo = &v[o * m * inner];
    uint8_t* wo = &w[o * m * inner];
    if (inner == 1) {  // along the row: combine the row with its shifts
      std::memcpy(wo, vo, m);
      for (int s = 1; s <= r && s < m; s++) {
        for (int x = 0; x + s < m; x++) wo[x] = op(wo[x], vo[x + s]);
        for (int x = s; x < m; x++) wo[x] = op(wo[x], vo[x - s]);
      }
      continue;
    }
    for (int x = 0; x < m; x++) {
      const int y0 = std::max(0, x - r), y1 = std::min(m - 1, x + r);
      uint8_t* dst = wo + x * inner;
      std::memcpy(dst, vo + y0 * inner, inner);
      for (int y = y0 + 1; y <= y1; y++) {
        const uint8_t* src = vo + y * inner;
        for (long t = 0; t < inner; t++) dst[t] = op(dst[t], src[t]);
      }
    }
  }
  v.swap(w);
}

void box_filter(std::vector<uint8_t>& v, const int n[3], int d, int r, bool take_min) {
  if (take_min)
    box_filter_t<true>(v, n, d, r);
  else
    box_filter_t<false>(v, n, d, r);
}

// Counts over boxes in O(1): a summed-area table of a dense 0/1 field,
// S(i, j, k) = number of set cells in [0, i) x [0, j) x [0, k); without a table
// every cell is set.
struct BoxSum {
  int n[3];
  const int* S;
  BoxSum(const int* table, const int nn[3]) : S(table) {
    for (int d = 0; d < 3; d++) n[d] = nn[d];
  }
  // the table of a host field
  static std::vector<int> table(const std::vector<uint8_t>& v, const int n[3]) {
    const long sx = n[0] + 1, sxy = sx * (n[1] + 1);
    std::vector<int> S(sxy * (n[2] + 1), 0);
    for (int k = 0; k < n[2]; k++)
      for (int j = 0; j < n[1]; j++) {
        const uint8_t* row = &v[(long)n[0] * (j + (long)n[1] * k)];
        int* o = &S[(k + 1) * sxy + (j + 1) * sx];
        const int* dn = o - sx;        // (j, k + 1)
        const int* bk = o - sxy;       // (j + 1, k)
        const int* db = o - sx - sxy;  // (j, k)
        int line = 0;                  // running sum along the row
        for (int i = 0; i < n[0]; i++) {
          line += row[i] ? 1 : 0;
          o[i + 1] = line + dn[i + 1] + bk[i + 1] - db[i + 1];
        }
      }
    return S;
  }
  long count(const int lo[3], const int hi[3]) const {
    if (!S) return (long)(hi[0] - lo[0] + 1) * (hi[1] - lo[1] + 1) * (hi[2] - lo[2] + 1);
    const long sx = n[0] + 1, sxy = sx * (n[1] + 1);
    auto at = [&](int i, int j, int k) { return (long)S[k * sxy + j * sx + i]; };
    const int a0 = lo[0], a1 = lo[1], a2 = lo[2], b0 = hi[0] + 1, b1 = hi[1] + 1, b2 = hi[2] + 1;
    return at(b0, b1, b2) - at(a0, b1, b2) - at(b0, a1, b2) - at(b0, b1, a2) + at(a0, a1, b2) +
           at(a0, b1, a2) + at(b0, a1, a2) - at(a0, a1, a2);
  }
};

struct Clusterer {
  const BoxSum& tag;   // level-l tags
  const BoxSum& ok;    // level-l cells that may hold the finer level
  int n[3];
  double eff;
  int max_side, min_side;            // in level-l cells
  std::vector<IBox>& out;

  // sig[x] = tags in the plane lo[d] + x of the box, along axis d
  void signature(const IBox& b, int d, std::vector<long>& sig) const {
    sig.assign(b.side(d), 0);
    int lo[3] = {b.lo[0], b.lo[1], b.lo[2]}, hi[3] = {b.hi[0], b.hi[1], b.hi[2]};
    for (int x = 0; x < b.side(d); x++) {
      lo[d] = hi[d] = b.lo[d] + x;
      sig[x] = tag.count(lo, hi);
    }
  }

  // the box cut down to the bounding box of its tags; false if it has none
  bool shrink(IBox& b, long& cnt) const {
    cnt = tag.count(b.lo, b.hi);
    if (!cnt) return false;
    std::vector<long> sig;
    for (int d = 0; d < 3; d++) {
      signature(b, d, sig);
      int f = 0, l = b.side(d) - 1;
      while (!sig[f]) f++;
      while (!sig[l]) l--;
      const int lo = b.lo[d];
      b.lo[d] = lo + f;
      b.hi[d] = lo + l;
    }
    return true;
  }

  bool all_ok(const IBox& b) const { return ok.count(b.lo, b.hi) == b.vol(); }

  void run(IBox b) {
    long cnt;
    if (!shrink(b, cnt)) return;
    int longest = 0;
    for (int d = 1; d < 3; d++)
      if (b.side(d) > b.side(longest)) longest = d;
    const bool nested = all_ok(b);
    if (nested && b.side(longest) <= max_side && (double)cnt >= eff * (double)b.vol()) {
      out.push_back(b);
      return;
    }
    const int mn = nested ? std::max(1, min_side) : 1;
    const int order[3] = {longest, (longest + 1) % 3, (longest + 2) % 3};
    std::vector<long> sig;
    // (1) a hole of a signature: parts [lo, lo+i-1] and [lo+i+1, hi]
    for (int q = 0; q < 3; q++) {
      const int d = order[q], s = b.side(d), mid = s / 2;
      if (s < 3) continue;
      signature(b, d, sig);
      int best = -1, bestdist = 1 << 30;
      for (int i = 1; i + 1 < s; i++)
        if (sig[i] == 0 && i >= mn && s - 1 - i >= mn && std::abs(i - mid) < bestdist) {
          best = i;
          bestdist = std::abs(i - mid);
        }
      if (best >= 0) {
        IBox a = b, c = b;
        a.hi[d] = b.lo[d] + best - 1;
        c.lo[d] = b.lo[d] + best + 1;
        run(a);
        run(c);
        return;
      }
    }
    // (2) an inflection: parts [lo, lo+i] and [lo+i+1, hi]
    int sd = -1, cut = -1;
    long bestv = 0;
    for (int q = 0; q < 3; q++) {
      const int d = order[q], s = b.side(d);
      if (s < 4) continue;
      signature(b, d, sig);
      for (int i = 1; i + 2 < s; i++) {
        const long l1 = sig[i + 1] - 2 * sig[i] + sig[i - 1];
        const long l2 = sig[i + 2] - 2 * sig[i + 1] + sig[i];
        if ((l1 < 0) == (l2 < 0)) continue;
        if (i + 1 < mn || s - 1 - i < mn) continue;
        const long v = std::labs(l2 - l1);
        if (v > bestv) {
          bestv = v;
          sd = d;
          cut = i;
        }
      }
    }
    if (sd >= 0) {
      IBox a = b, c = b;
      a.hi[sd] = b.lo[sd] + cut;
      c.lo[sd] = b.lo[sd] + cut + 1;
      run(a);
      run(c);
      return;
    }
    // (3) bisection of the longest side: [lo, lo+s/2-1] and [lo+s/2, hi]
    const int s = b.side(longest);
    if (s >= 2 && s / 2 >= mn && s - s / 2 >= mn) {
      IBox a = b, c = b;
      a.hi[longest] = b.lo[longest] + s / 2 - 1;
      c.lo[longest] = b.lo[longest] + s / 2;
      run(a);
      run(c);
      return;
    }
    out.push_back(b);
  }
};

// Small levels form their fields on the host: a copy of the tags and byte loops
// (about 0.85 ns per cell and window cell) take less there than ten launches, the
// tables' copy back (40 us) and 0.26 us per plane of running sums.  Whole calls for
// 2 levels, host against device form (us): 4^3 23 against 57, 16^3 47 against 68
// (buffer 8: 65 against 66), 18^3 59 against 70 (buffer 4: 74 against 69), 20^3 98
// against 99, 24^3 101 against 82, 4x4x512 144 against 214.
bool host_fields(const int n[3], int up, int buffer) {   // n of a level, `up` levels finer
  const long cells = ((long)n[0] * n[1] * n[2]) << (3 * up), planes = ((long)n[1] + n[2]) << up;
  return cells * (std::min(buffer, 8192) + 6L) <= 44000 + 300 * planes;
}

// ---- device side of the clustering: dense fields of one level
struct Dims {
  int n0, n1, n2;
  __device__ long at(int i, int j, int k) const { return i + (long)n0 * (j + (long)n1 * k); }
};

// raw[q] := tag of the level-lc cell holding q, for every level-lc cell of the
// current hierarchy; called from the coarsest level to min(l, finest), so that
// the finest cell's tag stays.  Grid (patches, blocks per patch).
__global__ void k_rg_scatter(const PatchDev* __restrict__ patches, const uint8_t* __restrict__ tags,
                             int bits, int shift, Dims D, uint8_t* __restrict__ raw) {
  const PatchDev P = patches[blockIdx.x];
  const int nc = P.n[0] * P.n[1] * P.n[2], r = 1 << shift;
  for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < nc; c += gridDim.y * blockDim.x) {
    const int q = c / P.n[0], i = P.lo[0] + c - q * P.n[0];
    const int k = q / P.n[1], j = P.lo[1] + q - k * P.n[1], kk = P.lo[2] + k;
    const uint8_t t = (tags[P.off + c] & bits) ? 1 : 0;
    for (int z = 0; z < r; z++)
      for (int y = 0; y < r; y++)
        for (int x = 0; x < r; x++) raw[D.at(i * r + x, j * r + y, kk * r + z)] = t;
  }
}

// in[q] := 1 on the boxes of the new level.  Grid (boxes, blocks per box).
__global__ void k_rg_boxes(const int* __restrict__ boxes, Dims D, uint8_t* __restrict__ in) {
  const int* b = boxes + 6 * blockIdx.x;
  const int s0 = b[3] - b[0] + 1, s1 = b[4] - b[1] + 1, nc = s0 * s1 * (b[5] - b[2] + 1);
  for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < nc; c += gridDim.y * blockDim.x) {
    const int q = c / s0, k = q / s1;
    in[D.at(b[0] + c - q * s0, b[1] + q - k * s1, b[2] + k)] = 1;
  }
}

// one axis of the box filters: hit := OR of raw within r cells (of cells that
// are in the level, where in is given), ok := AND of in within 1 cell, both
// inside the domain.  first: the x axis, where raw counts on the level only.
__global__ void k_rg_filter(Dims D, int axis, int r, bool first, const uint8_t* __restrict__ raw,
                            const uint8_t* __restrict__ in0, const uint8_t* __restrict__ in,
                            uint8_t* __restrict__ hit, uint8_t* __restrict__ ok) {
  const long nn = (long)D.n0 * D.n1 * D.n2;
  const long st = axis == 0 ? 1 : (axis == 1 ? (long)D.n0 : (long)D.n0 * D.n1);
  const int m = axis == 0 ? D.n0 : (axis == 1 ? D.n1 : D.n2);
  for (long q = blockIdx.x * (long)blockDim.x + threadIdx.x; q < nn;
       q += (long)gridDim.x * blockDim.x) {
    const int x = (int)((q / st) % m);
    uint8_t h = 0;
    for (int d = -min(r, x); d <= min(r, m - 1 - x); d++) {
      const uint8_t v = raw[q + d * st];
      h |= (first && in0) ? (v & in0[q + d * st]) : v;
    }
    hit[q] = h;
    if (in) {
      uint8_t o = in[q];
      if (x > 0) o &= in[q - st];
      if (x < m - 1) o &= in[q + st];
      ok[q] = o;
    }
  }
}

// Summed-area tables of the tagged field (tag on nestable cells) and, where
// there is one, the nestable field (blockIdx.y = 1): first the rows (one warp
// each, a scan per 32 cells), then running sums along y and z.  S: tables of
// (n0 + 1)(n1 + 1)(n2 + 1) entries, one after the other, zeroed.
__global__ void k_rg_rows(Dims D, const uint8_t* __restrict__ hit, const uint8_t* __restrict__ ok,
                          int* __restrict__ S) {
  const long sx = D.n0 + 1, sxy = sx * (D.n1 + 1), tab = sxy * (D.n2 + 1);
  const int f = blockIdx.y, lane = threadIdx.x & 31;
  const long rows = (long)D.n1 * D.n2;
  for (long w = (blockIdx.x * (long)blockDim.x + threadIdx.x) >> 5; w < rows;
       w += ((long)gridDim.x * blockDim.x) >> 5) {
    const int j = (int)(w % D.n1), k = (int)(w / D.n1);
    int* o = S + f * tab + (k + 1) * sxy + (j + 1) * sx + 1;
    int base = 0;
    for (int i0 = 0; i0 < D.n0; i0 += 32) {
      const int i = i0 + lane;
      int v = 0;
      if (i < D.n0) {
        const long q = D.at(i, j, k);
        const uint8_t a = ok ? ok[q] : 1;
        v = f ? a : (a & hit[q]);
      }
      for (int s = 1; s < 32; s <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, s);
        if (lane >= s) v += u;
      }
      if (i < D.n0) o[i] = base + v;
      base += __shfl_sync(0xffffffffu, v, 31);
    }
  }
}
// axis 1: along y for every (i, k); axis 2: along z for every (i, j)
__global__ void k_rg_sums(Dims D, int axis, int* __restrict__ S) {
  const long sx = D.n0 + 1, sxy = sx * (D.n1 + 1), tab = sxy * (D.n2 + 1);
  const int other = axis == 1 ? D.n2 : D.n1, m = axis == 1 ? D.n1 : D.n2;
  const long so = axis == 1 ? sxy : sx, st = axis == 1 ? sx : sxy;
  const long lines = (long)D.n0 * other;
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < lines;
       t += (long)gridDim.x * blockDim.x) {
    int* p = S + blockIdx.y * tab + (t % D.n0) + 1 + (t / D.n0 + 1) * so + st;
    int acc = 0;
#pragma unroll 8
    for (int x = 0; x < m; x++, p += st) {
      acc += *p;
      *p = acc;
    }
  }
}

int rg_blocks(long n) { return (int)std::max(1L, std::min(152L * 8, (n + 255) / 256)); }

// Device scratch of a context for the two calls here, both of which synchronise
// before they return: kept up to kKeep bytes (an allocation and its release
// cost more than the kernels of a 64^3 level: 170 of 400 us), else given back by
// xfer_done.  null when the allocation fails.
constexpr size_t kKeep = 256u << 20;
void* xfer_reserve(nrd_ctx* c, size_t bytes) {
  if (bytes > c->xfer_bytes) {
    if (c->d_xfer) cudaFree(c->d_xfer);
    c->d_xfer = nullptr;
    c->xfer_bytes = 0;
    if (cudaMalloc(&c->d_xfer, bytes) != cudaSuccess) {
      cudaGetLastError();
      c->d_xfer = nullptr;
      return nullptr;
    }
    c->xfer_bytes = bytes;
  }
  return c->d_xfer;
}
void xfer_done(nrd_ctx* c) {
  if (c->xfer_bytes <= kKeep) return;
  cudaFree(c->d_xfer);
  c->d_xfer = nullptr;
  c->xfer_bytes = 0;
}

// One call's hold on that scratch; while another thread's call has it (several
// may transfer from one context), an allocation of the call's own in its stream's
// order, so that neither call waits for the other's work.
struct Scratch {
  nrd_ctx* c;
  cudaStream_t s;
  std::unique_lock<std::mutex> lock;
  void* own = nullptr;
  Scratch(nrd_ctx* ctx, cudaStream_t st) : c(ctx), s(st), lock(ctx->xfer_mu, std::try_to_lock) {}
  Scratch(const Scratch&) = delete;
  void* get(size_t bytes) {
    if (lock.owns_lock()) return xfer_reserve(c, bytes);
    if (cudaMallocAsync(&own, bytes, s) != cudaSuccess) {
      cudaGetLastError();
      own = nullptr;
    }
    return own;
  }
  ~Scratch() {
    if (own) {
      cudaFreeAsync(own, s);
      cudaStreamSynchronize(s);   // the pool gives it back here
    } else if (lock.owns_lock()) {
      xfer_done(c);   // before the lock is released
    }
  }
};

// the device fields and tables of one level
struct RgDevice {
  Scratch scratch;
  explicit RgDevice(nrd_ctx* ctx) : scratch(ctx, nullptr) {}
  // tables of the tagged cells and (unless the level covers the domain) of the
  // nestable cells, on the host; false when the device had no memory for it
  bool tables(const Hier& H, const uint8_t* tags, int bits, int buffer, int l, const int n[3],
              const std::vector<IBox>& boxes, std::vector<int>& S, cudaError_t& e) {
    const long nn = (long)n[0] * n[1] * n[2];
    const long tab = (long)(n[0] + 1) * (n[1] + 1) * (n[2] + 1);
    const bool full = l == 0;                      // one box: the whole domain
    const int nt = full ? 1 : 2;
    const size_t pad = (nn + 255) / 256 * 256;
    const size_t bytes = 6 * pad + nt * tab * sizeof(int) + 6 * boxes.size() * sizeof(int);
    uint8_t* buf = (uint8_t*)scratch.get(bytes);
    if (!buf) return false;
    uint8_t *raw = buf, *in = raw + pad, *h1 = in + pad, *o1 = h1 + pad, *h2 = o1 + pad,
            *o2 = h2 + pad;
    int* dS = (int*)(buf + 6 * pad);
    int* dB = dS + nt * tab;
    const Dims D{n[0], n[1], n[2]};
    for (int lc = 0; lc <= std::min(l, H.L - 1); lc++) {
      const LevelInfo& Lv = H.lev[lc];
      const int per = (int)std::max(1L, std::min(152L * 8L / Lv.np + 1, (Lv.ncell / Lv.np + 255L) / 256));
      k_rg_scatter<<<dim3(Lv.np, per), 256>>>(H.d_patches + Lv.p0, tags, bits, l - lc, D, raw);
    }
    if (!full) {
      std::vector<int> hb;
      for (const IBox& b : boxes) {
        hb.insert(hb.end(), b.lo, b.lo + 3);
        hb.insert(hb.end(), b.hi, b.hi + 3);
      }
      cudaMemcpy(dB, hb.data(), hb.size() * sizeof(int), cudaMemcpyHostToDevice);
      cudaMemsetAsync(in, 0, nn);
      k_rg_boxes<<<dim3((unsigned)boxes.size(), 8), 256>>>(dB, D, in);
    }
    cudaMemsetAsync(dS, 0, nt * tab * sizeof(int));
    const int g = rg_blocks(nn);
    const uint8_t* i0 = full ? nullptr : in;
    k_rg_filter<<<g, 256>>>(D, 0, buffer, true, raw, i0, i0, h1, o1);
    k_rg_filter<<<g, 256>>>(D, 1, buffer, false, h1, nullptr, full ? nullptr : o1, h2, o2);
    k_rg_filter<<<g, 256>>>(D, 2, buffer, false, h2, nullptr, full ? nullptr : o2, h1, o1);
    k_rg_rows<<<dim3(rg_blocks((long)n[1] * n[2] * 32), nt), 256>>>(D, h1, full ? nullptr : o1, dS);
    k_rg_sums<<<dim3(rg_blocks((long)n[0] * n[2]), nt), 256>>>(D, 1, dS);
    k_rg_sums<<<dim3(rg_blocks((long)n[0] * n[1]), nt), 256>>>(D, 2, dS);
    S.resize(nt * tab);
    e = cudaMemcpy(S.data(), dS, nt * tab * sizeof(int), cudaMemcpyDeviceToHost);
    return true;
  }
};

// ---- transfer
__device__ __forceinline__ double minmod(double a, double b) {
  if (a * b <= 0.0) return 0.0;
  return (fabs(a) < fabs(b)) ? a : b;
}

// The old hierarchy's cell look-up: dense maps up to the level below the
// finest; a finest cell is the child of a covered cell there (slot: index of
// a level L - 2 cell in the covered list, or -1).  One level: the box itself.
struct OldCells {
  int L;
  int n[NRD_MAX_LEVELS][3];
  const int* lmap[NRD_MAX_LEVELS];
  const int4* cov;
  const int* slot;
  int off;                       // first cell of level L - 2
  __device__ int find(int l, int x, int y, int z) const {
    if (l >= L || x < 0 || y < 0 || z < 0 || x >= n[l][0] || y >= n[l][1] || z >= n[l][2])
      return -1;
    if (l == 0 && L == 1) return x + n[0][0] * (y + n[0][1] * z);
    if (l < L - 1) return lmap[l][x + (long)n[l][0] * (y + (long)n[l][1] * z)];
    const int p = lmap[l - 1][(x >> 1) + (long)n[l - 1][0] * ((y >> 1) + (long)n[l - 1][1] * (z >> 1))];
    if (p < 0) return -1;
    const int e = slot[p - off];
    if (e < 0) return -1;
    const int4 c = cov[e];
    return c.y + (x & 1) + (y & 1) * c.z + (z & 1) * c.w;
  }
};

__global__ void k_cov_slots(const int4* __restrict__ cov, int n, int off, int* __restrict__ slot) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x)
    slot[cov[q].x - off] = q;
}

// One new cell per thread over the new hierarchy's tiles: a cell that exists on
// its level of the old hierarchy is copied, any other takes the limited linear
// reconstruction of the finest old cell holding it.
__global__ void k_transfer(const TileDev* __restrict__ tiles, const PatchDev* __restrict__ patches,
                           int tx, int ty, OldCells O, int N, int Nold, int nvec,
                           const double* __restrict__ uo, double* __restrict__ un) {
  const TileDev tile = tiles[blockIdx.x];
  const PatchDev P = patches[tile.patch];
  const int ex = min(tx, P.n[0] - tile.i0), ey = min(ty, P.n[1] - tile.j0);
  const int nc = ex * ey * (tile.k1 - tile.k0), l = P.level;
  for (int t = threadIdx.x; t < nc; t += blockDim.x) {
    const int r0 = t / ex, i = tile.i0 + t - r0 * ex;
    const int rk = r0 / ey, j = tile.j0 + r0 - rk * ey, k = tile.k0 + rk;
    const int c = P.off + i + P.n[0] * (j + P.n[1] * k);
    const int q[3] = {P.lo[0] + i, P.lo[1] + j, P.lo[2] + k};
    int lc = min(l, O.L - 1), src = -1, cq[3] = {0, 0, 0};
    for (; lc >= 0; lc--) {
      for (int d = 0; d < 3; d++) cq[d] = q[d] >> (l - lc);
      src = O.find(lc, cq[0], cq[1], cq[2]);
      if (src >= 0) break;
    }
    if (lc == l) {
      for (int f = 0; f < 2 * nvec; f++) un[(long)f * N + c] = uo[(long)f * Nold + src];
      continue;
    }
    // (the base level covers the domain, so src >= 0)
    const int r = 1 << (l - lc);
    int nb[6];
    double off[3];
    for (int d = 0; d < 3; d++) {
      // centre of the new cell relative to the old one, in old cells (a
      // multiple of 1/2^(l - lc + 1), exact)
      off[d] = (2.0 * (q[d] - cq[d] * r) + 1.0 - r) / (2.0 * r);
      for (int sd = 0; sd < 2; sd++) {
        int nq[3] = {cq[0], cq[1], cq[2]};
        nq[d] += sd ? 1 : -1;
        nb[2 * d + sd] = O.find(lc, nq[0], nq[1], nq[2]);
      }
    }
    for (int f = 0; f < 2 * nvec; f++) {
      const double* u = uo + (long)f * Nold;
      const double uc = u[src];
      double v = uc;
      for (int a = 0; a < 3; a++) {
        const int im = nb[2 * a], ip = nb[2 * a + 1];
        if (im >= 0 && ip >= 0) v += minmod(uc - u[im], u[ip] - uc) * off[a];
      }
      un[(long)f * N + c] = v;
    }
  }
}

}  // namespace

extern "C" {

int nrd_regrid_boxes(nrd_ctx* c, const uint8_t* tags, int tag_bits, int buffer,
                     double efficiency, int min_side, int max_side, int max_levels,
                     int max_boxes, int* nlevels_out, int* nboxes_out, int* boxes_out,
                     int* total_out) {
  if (!c) return NRD_EINVAL;
  if (!c->have_hier) {
    c->err = "no hierarchy";
    return NRD_ESTATE;
  }
  if (step_pending_check(c, false, nullptr)) return NRD_ESTATE;
  if (!tags || !nlevels_out || !nboxes_out || !boxes_out || !total_out || buffer < 0 ||
      !(efficiency > 0.0 && efficiency <= 1.0) || min_side < 2 || max_side < min_side ||
      (min_side % 2) || (max_side % 2) || max_levels < 1 || max_levels > NRD_MAX_LEVELS ||
      max_boxes < 1 || (tag_bits & 0xff) == 0) {
    c->err = "bad argument to nrd_regrid_boxes";
    return NRD_EINVAL;
  }
  // the work below goes to the legacy default stream, after the tags
  if (c->tag_ev && cudaStreamWaitEvent(nullptr, c->tag_ev, 0) != cudaSuccess) {
    c->err = "wait for the tags failed";
    return NRD_ECUDA;
  }
  const Hier& H = c->H;
  std::vector<uint8_t> htags;   // of the levels up to one done on the host
  const int n0[3] = {H.lev[0].n[0], H.lev[0].n[1], H.lev[0].n[2]};
  // tag of the current cell (l, q), or -1 if the current hierarchy has none
  auto cur_tag = [&](int l, const int q[3]) -> int {
    if (l >= H.L) return -1;
    const LevelInfo& Lv = H.lev[l];
    const int ci = H.lmap[l][q[0] + (long)Lv.n[0] * (q[1] + (long)Lv.n[1] * q[2])];
    return ci < 0 ? -1 : ((htags[ci] & tag_bits) ? 1 : 0);
  };
  std::vector<std::vector<IBox>> levels(1);
  levels[0].push_back(IBox{{0, 0, 0}, {n0[0] - 1, n0[1] - 1, n0[2] - 1}});
  for (int l = 0; l + 1 < max_levels; l++) {
    const int n[3] = {n0[0] << l, n0[1] << l, n0[2] << l};
    const long lsize = (long)n[0] * n[1] * n[2];
    if ((long)(n[0] + 1) * (n[1] + 1) * (n[2] + 1) > (long)INT32_MAX) {
      c->err = "nrd_regrid_boxes: a level is too large for int32 box counts";
      return NRD_EINVAL;
    }
    // on the host where that is faster (host_fields) or the device's memory does
    // not allow the fields
    std::vector<int> tables, osum_h;
    RgDevice dev{c};
    cudaError_t e = cudaSuccess;
    const bool on_device =
        !host_fields(n, 0, buffer) && dev.tables(H, tags, tag_bits, buffer, l, n, levels[l], tables, e);
    if (on_device && (e != cudaSuccess || cudaGetLastError() != cudaSuccess)) {
      c->err = "clustering kernels failed";
      return NRD_ECUDA;
    }
    const int* ttab = tables.data();
    const int* otab = nullptr;   // null: every cell is nestable
    if (on_device && l > 0) otab = tables.data() + (long)(n[0] + 1) * (n[1] + 1) * (n[2] + 1);
    if (!on_device) {
      // the tags of the levels up to this one, at once for all that will be done
      // here (cells ascend by level)
      int lt = std::min(l, H.L - 1);
      while (lt + 1 < std::min(H.L, max_levels - 1) && host_fields(n, lt + 1 - l, buffer)) lt++;
      const size_t need = (size_t)H.lev[lt].off + H.lev[lt].ncell;
      if (htags.size() < need) {
        htags.resize(need);
        if (cudaMemcpy(htags.data(), tags, need, cudaMemcpyDeviceToHost) != cudaSuccess) {
          c->err = "copy of the tags failed";
          return NRD_ECUDA;
        }
      }
      auto li = [&](int i, int j, int k) { return i + (long)n[0] * (j + (long)n[1] * k); };
      std::vector<uint8_t> in(lsize, 0), raw(lsize, 0), tg(lsize, 0), ok(lsize, 0);
      for (const IBox& b : levels[l])
        for (int k = b.lo[2]; k <= b.hi[2]; k++)
          for (int j = b.lo[1]; j <= b.hi[1]; j++)
            for (int i = b.lo[0]; i <= b.hi[0]; i++) {
              in[li(i, j, k)] = 1;
              int t = -1;
              for (int lc = std::min(l, H.L - 1); lc >= 0 && t < 0; lc--) {
                const int q[3] = {i >> (l - lc), j >> (l - lc), k >> (l - lc)};
                t = cur_tag(lc, q);
              }
              raw[li(i, j, k)] = t > 0 ? 1 : 0;
            }
      // ok: every neighbour of the 3x3x3 block inside the domain is in the new
      // level (proper nesting); tg: a raw tag within `buffer` cells (inside the
      // domain), on ok cells.  Both are box filters, done one axis at a time:
      // the minimum of `in` over windows of 3 (outside the domain counts as
      // in), the maximum of `raw` over windows of 2 buffer + 1 (outside counts
      // as untagged).
      ok = in;
      for (int d = 0; d < 3; d++) box_filter(ok, n, d, 1, true);
      std::vector<uint8_t> hit = raw;
      for (int d = 0; d < 3; d++) box_filter(hit, n, d, buffer, false);
      for (long q = 0; q < lsize; q++) tg[q] = (ok[q] && hit[q]) ? 1 : 0;
      tables = BoxSum::table(tg, n);
      osum_h = BoxSum::table(ok, n);
      ttab = tables.data();
      otab = osum_h.data();
    }
    std::vector<IBox> coarse;
    const BoxSum tsum(ttab, n), osum(otab, n);
    Clusterer C{tsum, osum, {n[0], n[1], n[2]}, efficiency, max_side / 2, min_side / 2, coarse};
    C.run(IBox{{0, 0, 0}, {n[0] - 1, n[1] - 1, n[2] - 1}});
    if (coarse.empty()) break;
    levels.emplace_back();
    for (const IBox& b : coarse) {
      IBox f;
      for (int d = 0; d < 3; d++) {
        f.lo[d] = 2 * b.lo[d];
        f.hi[d] = 2 * b.hi[d] + 1;
      }
      levels[l + 1].push_back(f);
    }
  }
  int total = 0;
  for (const auto& lv : levels) total += (int)lv.size();
  *total_out = total;
  *nlevels_out = (int)levels.size();
  if (total > max_boxes) {
    c->err = "the new hierarchy has more than max_boxes boxes";
    return NRD_EINVAL;
  }
  int q = 0;
  for (int l = 0; l < max_levels; l++) {
    nboxes_out[l] = l < (int)levels.size() ? (int)levels[l].size() : 0;
    if (l >= (int)levels.size()) continue;
    for (const IBox& b : levels[l]) {
      for (int d = 0; d < 3; d++) boxes_out[6 * q + d] = b.lo[d];
      for (int d = 0; d < 3; d++) boxes_out[6 * q + 3 + d] = b.hi[d];
      q++;
    }
  }
  return NRD_OK;
}

int nrd_transfer(nrd_ctx* src, nrd_ctx* dst, const double* u_src, double* u_dst, int nvec,
                 cudaStream_t s) {
  if (!src || !dst) return NRD_EINVAL;
  if (!src->have_hier || !dst->have_hier) {
    dst->err = "both contexts need a hierarchy";
    return NRD_ESTATE;
  }
  if (step_pending_check(src, false, nullptr) || step_pending_check(dst, false, nullptr))
    return NRD_ESTATE;
  if (!u_src || !u_dst || nvec < 1) {
    dst->err = "bad argument to nrd_transfer";
    return NRD_EINVAL;
  }
  const Hier& A = src->H;
  const Hier& B = dst->H;
  for (int d = 0; d < 3; d++)
    if (A.lev[0].n[d] != B.lev[0].n[d]) {
      dst->err = "the hierarchies have different base grids";
      return NRD_EINVAL;
    }
  const size_t No = (size_t)A.N;
  // composite copies of the old vectors (with finer levels) and the covered
  // slots of the level below the finest, in a buffer the old context keeps
  const bool comp = A.L > 1;
  const size_t comp_bytes = comp ? 2 * No * nvec * sizeof(double) : 0;
  const size_t slot_bytes = comp ? (size_t)A.lev[A.L - 2].ncell * sizeof(int) : 0;
  std::optional<Scratch> scratch;   // until the call returns: its kernels have ended then
  char* buf = nullptr;
  if (comp) {
    scratch.emplace(src, s);
    buf = (char*)scratch->get(comp_bytes + slot_bytes);
    if (!buf) {
      dst->err = "allocation failed";
      return NRD_ENOMEM;
    }
  }
  OldCells O{};
  O.L = A.L;
  for (int l = 0; l < A.L; l++) {
    for (int d = 0; d < 3; d++) O.n[l][d] = A.lev[l].n[d];
    O.lmap[l] = A.d_lmap[l];
  }
  const double* old = u_src;
  dst->timer.begin(NRD_TK_TRANSFER, s);
  if (comp) {
    const int lp = A.L - 2;
    double* d_comp = (double*)buf;
    int* slot = (int*)(buf + comp_bytes);
    cudaMemcpyAsync(d_comp, u_src, comp_bytes, cudaMemcpyDeviceToDevice, s);
    launch_average_down(A, d_comp, 2 * nvec, (int)No, s);
    cudaMemsetAsync(slot, 0xff, slot_bytes, s);
    if (A.ncov[lp])
      k_cov_slots<<<rg_blocks(A.ncov[lp]), 256, 0, s>>>(A.d_cov[lp], A.ncov[lp], A.lev[lp].off,
                                                        slot);
    O.cov = A.d_cov[lp];
    O.slot = slot;
    O.off = A.lev[lp].off;
    old = d_comp;
  }
  k_transfer<<<(int)B.tiles.size(), 256, 0, s>>>(B.d_tiles, B.d_patches, B.tile_x, B.tile_y, O,
                                                 B.N, (int)No, nvec, old, u_dst);
  dst->timer.end(NRD_TK_TRANSFER, s);
  const cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) {
    dst->err = "transfer kernel failed";
    return NRD_ECUDA;
  }
  return NRD_OK;
}

}  // extern "C"
