// The renderer of Section 6: level-of-detail node selection and pixel-sized
// splats that keep the closest sample per pixel with a 64-bit atomicMin on
// (float bits of depth << 32 | rgba), drawn straight from the octree's chunk
// lists. It reads the octree as the update left it (stream order) and
// changes nothing in it.
//
// Selection, per node in parallel: a node is drawn when it is in the view
// frustum, it is a leaf or not larger than 2^G pixels on screen (the voxel
// resolution of an inner node), and its parent is larger than 2^G pixels (or
// it is the root). Because a child's projected box lies inside its parent's,
// this selects exactly the nodes of the paper's top-down rule (an inner node
// larger than 2^G pixels is hidden and its children are drawn instead).
//
// Projection: clip = M (x, y, z, 1) with M row-major; depth = clip w; a
// sample at screen s = (clip.xy / w * 0.5 + 0.5) * (width, height) with w > 0
// and s inside the screen lands in pixel floor(s). A cube is culled when all
// 8 corners are outside one plane of x < -w, x > w, y < -w, y > w, w <= 0;
// its size on screen is the larger side of its corners' screen box
// (infinite when a corner has w <= 0). Every float operation is one IEEE
// single-precision operation in the written order (no contraction), so the
// result is reproducible bit for bit.
#pragma once

#include "device.cuh"

namespace SL_NS {

struct View {
  float m[16];
  float W, H, lod;
  uint32_t width, height;
};

__device__ __forceinline__ float dot4(float a, float x, float b, float y, float c, float z, float d) {
  return __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(a, x), __fmul_rn(b, y)), __fmul_rn(c, z)), d);
}

__device__ __forceinline__ float screen_coord(float c, float w, float extent) {
  return __fmul_rn(__fadd_rn(__fmul_rn(__fdiv_rn(c, w), 0.5f), 0.5f), extent);
}

// Frustum test and size on screen of the cube [mn, mn + 2^L).
__device__ __forceinline__ void cube_view(const View& v, const long long (&mn)[3], uint32_t L,
                                          bool& culled, float& size) {
  int out0 = 0, out1 = 0, out2 = 0, out3 = 0, out4 = 0;
  bool behind = false;
  float x0 = __int_as_float(0x7f800000), x1 = -x0, y0 = x0, y1 = -x0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float x = __ll2float_rn(mn[0] + ((long long)(k & 1) << L));
    const float y = __ll2float_rn(mn[1] + ((long long)((k >> 1) & 1) << L));
    const float z = __ll2float_rn(mn[2] + ((long long)((k >> 2) & 1) << L));
    const float cx = dot4(v.m[0], x, v.m[1], y, v.m[2], z, v.m[3]);
    const float cy = dot4(v.m[4], x, v.m[5], y, v.m[6], z, v.m[7]);
    const float cw = dot4(v.m[12], x, v.m[13], y, v.m[14], z, v.m[15]);
    out0 += cx < -cw;
    out1 += cx > cw;
    out2 += cy < -cw;
    out3 += cy > cw;
    out4 += !(cw > 0.0f);
    if (!(cw > 0.0f)) {
      behind = true;
      continue;
    }
    const float sx = screen_coord(cx, cw, v.W), sy = screen_coord(cy, cw, v.H);
    if (sx < x0) x0 = sx;
    if (sx > x1) x1 = sx;
    if (sy < y0) y0 = sy;
    if (sy > y1) y1 = sy;
  }
  culled = out0 == 8 || out1 == 8 || out2 == 8 || out3 == 8 || out4 == 8;
  if (behind) {
    size = __int_as_float(0x7f800000);
  } else {
    const float w = __fsub_rn(x1, x0), h = __fsub_rn(y1, y0);
    size = w > h ? w : h;
  }
}

__device__ __forceinline__ bool node_drawn(const Ctx& c, const View& v, uint32_t id) {
  const NodeMeta& m = c.meta[id];
  const uint32_t level = m.level;
  const uint32_t L = c.rlog2 - level;
  const long long mn[3] = {m.min[0], m.min[1], m.min[2]};
  bool culled;
  float size;
  cube_view(v, mn, L, culled, size);
  if (culled) return false;
  if (c.child[id] != NONE && size > v.lod) return false;  // hidden: its children are drawn
  if (level == 0) return true;
  long long pmn[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    pmn[a] = c.rmin[a] + (((mn[a] - c.rmin[a]) >> (L + 1)) << (L + 1));
  float psize;
  cube_view(v, pmn, L + 1, culled, psize);
  return psize > v.lod;
}

// Clear the frame (clear != 0: n_px words of all ones) and list the drawn
// nodes, one thread per node (warp-aggregated appends). The clear streams
// 8 bytes per pixel and would be a launch of its own; here its stores drain
// while the node tests wait for the node table.
__global__ void k_render_select(Ctx c, View v, uint32_t* vis, unsigned long long* fb,
                                uint64_t n_px, int clear) {
  after_previous();
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  // (nothing writes these during the frame: plain loads, most of them from L1)
  const uint32_t err = c.ctl->error, n_nodes = c.ctl->n_nodes;
  if (clear) {
    // the frame is 8-byte aligned; 16-byte stores from its first 16-byte boundary
    const uint64_t head = (reinterpret_cast<uintptr_t>(fb) & 15u) ? 1u : 0u;
    ulonglong2* fb2 = reinterpret_cast<ulonglong2*>(fb + head);
    const uint64_t pairs = (n_px - head) / 2;
    for (uint64_t i = t; i < pairs; i += stride) fb2[i] = make_ulonglong2(~0ull, ~0ull);
    if (t == 0) {
      if (head) fb[0] = ~0ull;
      if ((n_px - head) & 1u) fb[n_px - 1u] = ~0ull;
    }
  }
  // an octree whose last update failed is not drawn: ids that a failing build
  // reserved have no metadata (the host learns of the error at its next look)
  const uint32_t n = __any_sync(FULL_MASK, err != 0u) ? 0u : n_nodes;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b < n; b += stride) {
    const uint64_t id = b + lane;
    const bool d = id < n && id < c.max_nodes && node_drawn(c, v, (uint32_t)id);
    const unsigned mm = __ballot_sync(FULL_MASK, d);
    if (mm == 0u) continue;
    uint32_t o = 0;
    if (lane == 0) o = atomicAdd(&c.ctl->vis_count, (uint32_t)__popc(mm));
    o = __shfl_sync(FULL_MASK, o, 0);
    if (d) vis[o + __popc(mm & ((1u << lane) - 1u))] = (uint32_t)id;
  }
}

__device__ __forceinline__ void splat(const View& v, int4 r, unsigned long long* fb) {
  const float x = (float)r.x, y = (float)r.y, z = (float)r.z;
  const float cw = dot4(v.m[12], x, v.m[13], y, v.m[14], z, v.m[15]);
  if (!(cw > 0.0f)) return;
  const float cx = dot4(v.m[0], x, v.m[1], y, v.m[2], z, v.m[3]);
  const float cy = dot4(v.m[4], x, v.m[5], y, v.m[6], z, v.m[7]);
  const float sx = screen_coord(cx, cw, v.W), sy = screen_coord(cy, cw, v.H);
  if (!(sx >= 0.0f && sx < v.W && sy >= 0.0f && sy < v.H)) return;
  const uint32_t px = __float2uint_rz(sx), py = __float2uint_rz(sy);
  const unsigned long long key =
      ((unsigned long long)__float_as_uint(cw) << 32) | (uint32_t)r.w;
  atomicMin(fb + (uint64_t)py * v.width + px, key);
}

// A piece of a drawn node: records [first, first + n) of the chunk or array
// at ref, a chunk's or about as many, so that a node's records spread over many
// warps.
// (Compaction: n records of the chunk at ref that go to records first, ... of
// the array at arr.)
struct DrawUnit {
  uint32_t ref, first, n, arr;
};
static_assert(sizeof(DrawUnit) == sizeof(SpillTask), "draw units use the spill-task region");

__device__ __forceinline__ void draw_records(const Ctx& c, const View& v, const DrawUnit& u,
                                             uint32_t lo, uint32_t hi, unsigned long long* fb) {
  const int4* recs = chunk_recs(c, u.ref) + u.first;
  constexpr uint32_t U = 4;  // records per lane in flight
  for (uint32_t q = lo + lane_id(); q < hi; q += 32u * U) {
    int4 r[U];
#pragma unroll
    for (uint32_t k = 0; k < U; ++k) {
      if (q + 32u * k < hi) r[k] = __ldcg(recs + q + 32u * k);
    }
#pragma unroll
    for (uint32_t k = 0; k < U; ++k) {
      if (q + 32u * k < hi) splat(v, r[k], fb);
    }
  }
}

// All 32 lanes call: lane i hands out its unit u (when on) at index at.
// Units that do not fit the region (arrays cut into more pieces than the
// data region has chunks) are drawn here.
__device__ __forceinline__ void put_unit(const Ctx& c, const View& v, DrawUnit* units, bool on,
                                         uint64_t at, const DrawUnit& u, unsigned long long* fb) {
  const bool fits = at < c.max_chunks;
  if (on && fits) units[at] = u;
  unsigned over = __ballot_sync(FULL_MASK, on && !fits);
  while (over) {
    const int l = __ffs(over) - 1;
    over &= over - 1u;
    DrawUnit w;
    w.ref = __shfl_sync(FULL_MASK, u.ref, l);
    w.first = __shfl_sync(FULL_MASK, u.first, l);
    w.n = __shfl_sync(FULL_MASK, u.n, l);
    w.arr = 0;
    draw_records(c, v, w, 0, w.n, fb);
  }
}

// The chunks of one node, in list order: all 32 lanes call, and so does f(on, j,
// ref) for 32 chunks at a time (lane with `on`: chunk j is at ref). A leaf's
// chunks are in its directory (dir != nullptr). An inner node's chunk list has
// to be walked, one memory round trip per link; the chunks of one allocation
// lie one after another in the data region, so the warp reads the next links
// of 32 such successors at once and keeps as many as the list confirms (a link
// that points elsewhere ends the run: the walk goes on from there). Returns how
// many chunks it found; fewer than nch when the list is broken (an error).
template <typename F>
__device__ __forceinline__ uint32_t walk_chunks(const Ctx& c, uint32_t head, uint32_t nch,
                                                const uint32_t* dir, F&& f) {
  const uint32_t lane = lane_id();
  if (dir) {
    for (uint32_t j0 = 0; j0 < nch; j0 += 32u) {
      const bool in = j0 + lane < nch;
      const uint32_t ref = in ? dir[j0 + lane] : NONE;
      const bool ok = in && ref_ok(c, ref, c.chunk_bytes);
      if (in && !ok) set_error(c, E_INTERNAL);
      f(ok, j0 + lane, ref);
      const unsigned bad = __ballot_sync(FULL_MASK, in && !ok);
      if (bad) return j0 + (uint32_t)__ffs(bad) - 1u;
    }
    return nch;
  }
  uint32_t ref = head, j0 = 0;
  while (j0 < nch) {
    const uint32_t mine = ref + lane * c.chunk_units;
    const bool in = j0 + lane < nch && ref != NONE && ref_ok(c, mine, c.chunk_bytes);
    const uint32_t nxt = in ? *chunk_next(c, mine) : NONE;
    // the run: lanes whose predecessors' links all lead to the next lane
    const unsigned brk = __ballot_sync(FULL_MASK, !in || nxt != mine + c.chunk_units);
    const uint32_t run = brk ? (uint32_t)__ffs(brk) : 32u;  // lanes before run are in the list
    const bool ok = __shfl_sync(FULL_MASK, in ? 1 : 0, (int)run - 1) != 0;
    f(lane < run && in, j0 + lane, mine);
    if (lane < run && j0 + lane < nch && !in) set_error(c, E_INTERNAL);
    if (!ok) return min(j0 + run - 1u, nch);
    j0 += run;
    ref = __shfl_sync(FULL_MASK, nxt, (int)run - 1);
  }
  return nch;
}

// Directory of a leaf whose chunks are all in it, else nullptr.
__device__ __forceinline__ const uint32_t* leaf_dir(const Ctx& c, uint32_t id, const NodeMeta& m) {
  return c.child[id] == NONE && m.n_chunks <= c.dir_cap && ref_ok(c, m.dir, c.dir_bytes)
             ? dir_entries(c, m.dir)
             : nullptr;
}

// Records of chunk j of a node with n records.
__device__ __forceinline__ uint32_t chunk_fill(const Ctx& c, uint32_t j, uint32_t n) {
  const unsigned long long at = (unsigned long long)j * c.C;
  return at < n ? (uint32_t)min((unsigned long long)c.C, n - at) : 0u;
}

// All 32 lanes call: draw the n records of up to 32 chunks at once, C of them in
// each but the last; lane j holds the reference of chunk j (of those in `have`).
__device__ __forceinline__ void draw_chunks(const Ctx& c, const View& v, uint32_t ref,
                                            unsigned have, uint32_t n, unsigned long long* fb) {
#pragma unroll 2
  for (uint32_t q0 = 0; q0 < n; q0 += 32u) {
    const uint32_t q = q0 + lane_id(), j = div_by(q, c.C, c.C_mul, c.C_shift);
    const uint32_t from = __shfl_sync(FULL_MASK, ref, (int)(j & 31u));
    if (q < n && ((have >> (j & 31u)) & 1u)) splat(v, __ldcg(chunk_recs(c, from) + (q - j * c.C)), fb);
  }
}

// Cut the drawn nodes' records into draw units of one chunk, or `piece` records of
// a compacted node's array. A warp looks at up to 32 nodes at once, one per lane
// (fewer nodes than warps: one node a warp); the block takes their unit numbers
// with one atomic, and each lane hands out the chunks of its own node when it need
// not follow a list of them. The other nodes are walked one after another by all
// lanes; chunks of less than a warp's records are drawn on the way. (A warp and an
// atomic per node, and a unit for every chunk: a frame of 17,764 nodes of 60 points
// 61 us, of 282k nodes of 4 points 296, where one warp had drawn each in 45 and 252.)
constexpr uint32_t LANE_CHUNKS = 4;
__global__ void k_render_units(Ctx c, View v, const uint32_t* vis, DrawUnit* units, uint32_t piece,
                               unsigned long long* fb) {
  __shared__ uint32_t s_first[32], s_u0;
  after_previous();
  const uint32_t nv = min(vload(&c.ctl->vis_count), c.max_nodes);
  const uint32_t lane = threadIdx.x & 31u, wi = threadIdx.x / 32u, wpb = blockDim.x / 32u;
  const uint64_t nwarps = (uint64_t)gridDim.x * wpb;
  unsigned long long samples = 0;
  for (uint64_t b = (uint64_t)blockIdx.x * wpb; b < nv; b += 32u * nwarps) {
    const uint64_t k = b + wi + lane * nwarps;
    uint32_t n = 0, nch = 0, head = NONE;
    bool compact = false;
    const uint32_t* dir = nullptr;
    if (k < nv) {
      const uint32_t id = vis[k];
      const NodeMeta& m = c.meta[id];
      n = c.num[id];
      head = m.head;
      compact = m.compact != 0u;
      nch = compact ? (uint32_t)(((unsigned long long)n + piece - 1) / piece) : m.n_chunks;
      if (n == 0) nch = 0;
      if (!compact) dir = leaf_dir(c, id, m);
      samples += n;
    }
    const bool own = nch == 1u ? !compact : dir && nch <= LANE_CHUNKS;
    const uint32_t take = own || compact || c.C >= 32u ? nch : 0u;  // units
    uint32_t upto = take;  // of the lanes up to this one
    for (uint32_t d = 1; d < 32u; d <<= 1) {
      const uint32_t o = __shfl_up_sync(FULL_MASK, upto, d);
      if (lane >= d) upto += o;
    }
    if (lane == 31u) s_first[wi] = upto;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t all = 0;
      for (uint32_t w = 0; w < wpb; ++w) {
        const uint32_t t = s_first[w];
        s_first[w] = all;
        all += t;
      }
      s_u0 = all ? atomicAdd(&c.ctl->draw_units, all) : 0u;
    }
    __syncthreads();
    const uint32_t u0 = s_u0 + s_first[wi] + upto - take;  // the first of this lane's node
    __syncthreads();
    for (uint32_t j = 0; __any_sync(FULL_MASK, own && j < nch); ++j) {
      const bool on = own && j < nch;
      const uint32_t ref = !on ? NONE : nch == 1u ? head : dir[j];
      const bool ok = on && ref_ok(c, ref, c.chunk_bytes);
      if (on && !ok) set_error(c, E_INTERNAL);
      put_unit(c, v, units, on, (uint64_t)u0 + j,
               ok ? DrawUnit{ref, 0, chunk_fill(c, j, n), 0} : DrawUnit{0, 0, 0, 0}, fb);
    }
    for (unsigned rest = __ballot_sync(FULL_MASK, nch != 0u && !own); rest; rest &= rest - 1u) {
      const int l = __ffs(rest) - 1;
      const uint32_t ln = __shfl_sync(FULL_MASK, n, l), lnch = __shfl_sync(FULL_MASK, nch, l);
      const uint32_t lhead = __shfl_sync(FULL_MASK, head, l);
      const uint32_t ltake = __shfl_sync(FULL_MASK, take, l);
      const uint64_t lu = __shfl_sync(FULL_MASK, u0, l);
      const uint32_t* ldir = reinterpret_cast<const uint32_t*>(
          __shfl_sync(FULL_MASK, reinterpret_cast<unsigned long long>(dir), l));
      uint32_t got = 0;
      if (!__shfl_sync(FULL_MASK, (int)compact, l)) {
        got = walk_chunks(c, lhead, lnch, ldir, [&](bool on, uint32_t j, uint32_t ref) {
          if (ltake) {
            put_unit(c, v, units, on, lu + j, DrawUnit{ref, 0, chunk_fill(c, j, ln), 0}, fb);
          } else {
            const unsigned have = __ballot_sync(FULL_MASK, on);
            const unsigned long long first = (unsigned long long)(j - lane) * c.C;
            if (first < ln)
              draw_chunks(c, v, ref, have,
                          min(ln - (uint32_t)first, (32u - (uint32_t)__clz(have)) * c.C), fb);
          }
        });
      } else if (array_ok(c, lhead, ln)) {
        for (; got < lnch; got += 32u) {
          const uint32_t j = got + lane;
          const unsigned long long at = (unsigned long long)j * piece;
          put_unit(c, v, units, j < lnch, lu + j,
                   DrawUnit{lhead, (uint32_t)at, at < ln ? min(piece, ln - (uint32_t)at) : 0u, 0},
                   fb);
        }
      } else if (lane == 0) {
        set_error(c, E_INTERNAL);
      }
      // a broken list: the rest of the reserved units draw nothing
      for (uint32_t j = got + lane; j < ltake; j += 32u)
        if (lu + j < c.max_chunks) units[lu + j] = DrawUnit{0, 0, 0, 0};
    }
  }
  for (uint32_t d = 16; d; d >>= 1) samples += __shfl_down_sync(FULL_MASK, samples, d);
  if (lane == 0 && samples) atomicAdd(&c.ctl->render_samples, samples);
}

// Splat the units, `parts` warps per unit (parts * part >= C and the pieces): about 256
// records a warp, so that a frame of a few nodes with tens of thousands of
// records each fills the GPU. One warp per node (the first form) left the
// longest node's chain of loads in charge: 0.43 ms for 3 nodes of 65k points
// in all, 0.87-0.97 ms for frames of 1M to 13M samples alike. Two 1080p frames
// of a 12M-point terrain (2.5M samples in the overview) went from 1.93 to
// 0.11 ms. What is left is the three launches and, for frames of tens of
// millions of samples, the 64-bit minimums on the frame in L2.
__global__ void k_render_draw(Ctx c, View v, const DrawUnit* units, uint32_t parts, uint32_t part,
                              unsigned long long* fb) {
  after_previous();
  const uint64_t nu = min((uint64_t)vload(&c.ctl->draw_units), (uint64_t)c.max_chunks);
  const uint64_t warp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  const uint64_t nwarps = (uint64_t)gridDim.x * blockDim.x / 32;
  for (uint64_t w = warp; w < nu * parts; w += nwarps) {
    const DrawUnit u = units[w / parts];
    const uint32_t lo = (uint32_t)(w % parts) * part, hi = min(lo + part, u.n);
    if (lo < hi) draw_records(c, v, u, lo, hi, fb);
  }
}

}  // namespace SL_NS
