// Corner turn (Sec. 2.1, "Transpose": [input, frequency] -> [frequency,
// input]) and FP64 normalisation of the integrated visibilities.
#include <algorithm>

#include "xe_device.cuh"

namespace xe {
namespace {

// ---------------------------------------------------------------- corner turn
// in[t][g][k] -> out[k][g][t] for byte samples, through a 256 (t) x 128 (k)
// shared-memory tile of 32-bit words.  Word w of tile row r is stored at
// r * 32 + (w ^ 4 * (r >> 5)): the 16-byte chunk index is XOR-ed with the
// row's 32-row band, which makes both the row-wise stores and the
// column-wise loads below free of bank conflicts without padding.
constexpr int kTT = 256, kTK = 128;

__device__ __forceinline__ void transpose4x4(uint32_t& a0, uint32_t& a1, uint32_t& a2,
                                             uint32_t& a3) {
  const uint32_t t0 = __byte_perm(a0, a1, 0x5140), t1 = __byte_perm(a0, a1, 0x7362);
  const uint32_t t2 = __byte_perm(a2, a3, 0x5140), t3 = __byte_perm(a2, a3, 0x7362);
  a0 = __byte_perm(t0, t2, 0x5410);
  a1 = __byte_perm(t0, t2, 0x7632);
  a2 = __byte_perm(t1, t3, 0x5410);
  a3 = __byte_perm(t1, t3, 0x7632);
}

__device__ __forceinline__ void ld32B(const uint8_t* p, uint32_t (&r)[8]) {
  asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}
__device__ __forceinline__ void st32B(uint8_t* p, const uint32_t (&r)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// 16 bytes from any address: the two aligned 16-byte words around it (one if
// it is aligned) and a byte shift.  A word that reaches outside [begin, end)
// is not read: its bytes come one by one, and those outside are zero.
__device__ __forceinline__ void ld16_any(const uint8_t* p, const uint8_t* begin, const uint8_t* end,
                                         uint32_t (&r)[4]) {
  const uint32_t a = (uint32_t)(reinterpret_cast<uintptr_t>(p) & 15);
  const uint8_t* q = p - a;
  if (q >= begin && q + (a ? 32 : 16) <= end) {
    const uint4 lo = __ldg(reinterpret_cast<const uint4*>(q));
    uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, 0u, 0u, 0u, 0u};
    if (a) {
      const uint4 hi = __ldg(reinterpret_cast<const uint4*>(q + 16));
      w[4] = hi.x, w[5] = hi.y, w[6] = hi.z, w[7] = hi.w;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = (a & 8) ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = (a & 4) ? w[i + 1] : w[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) r[i] = __funnelshift_r(w[i], w[i + 1], 8 * (a & 3));
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      r[i] = 0;
      for (int b = 0; b < 4; ++b)
        if (p + 4 * i + b >= begin && p + 4 * i + b < end) r[i] |= (uint32_t)p[4 * i + b] << (8 * b);
    }
  }
}

__device__ __forceinline__ int tile_word(int row, int w) { return row * 32 + (w ^ ((row >> 5) << 2)); }

// barrier of one 256-thread group (id 0 is the whole CTA of a 256-thread launch)
__device__ __forceinline__ void group_bar(int id) {
  asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory");
}

// Store phase of a tile held in `tile`: each thread transposes 4 x 32 bytes
// in registers and writes 32-byte pieces of [k][g][t] rows (vec: the rows are
// aligned to and padded to 32 bytes), or single bytes.
__device__ __forceinline__ void turn_tile_store(uint8_t* __restrict__ out, int T, int K, int G,
                                                long long os, int pair_rows, int t0, int k0,
                                                int g, const uint32_t* tile, int tid, bool full, bool vec) {
  const int warp = tid >> 5, lane = tid & 31;
  // store: thread = 4 consecutive k (word kq) x 32 consecutive t (segment ts);
  // the eight lanes of a k-quad cover one 256-byte stretch of each output row
  const int kq = 4 * warp + (lane >> 3), ts = lane & 7;
  uint32_t a[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) a[j] = tile[tile_word(ts * 32 + j, kq)];
#pragma unroll
  for (int j = 0; j < 32; j += 4) transpose4x4(a[j], a[j + 1], a[j + 2], a[j + 3]);
  // a[4w + c] now holds t = ts*32 + 4w .. +3 of k = 4 kq + c
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int k = k0 + 4 * kq + c;
    const int tb = t0 + ts * 32;
    const long long row =
        pair_rows ? ((long long)(k >> 1) * G + g) * 2 + (k & 1) : (long long)k * G + g;
    uint8_t* o = out + row * os + tb;
    if (full || (vec && k < K && tb < T)) {  // the last piece of a row runs into its padding (zeros)
      const uint32_t r[8] = {a[c], a[4 + c], a[8 + c], a[12 + c],
                             a[16 + c], a[20 + c], a[24 + c], a[28 + c]};
      st32B(o, r);
    } else if (!vec && k < K) {
      for (int b = 0; b < 32; ++b)
        if (tb + b < T) o[b] = (uint8_t)(a[4 * (b >> 2) + c] >> ((b & 3) * 8));
    }
  }
}


// Which accesses of a turn may be 32 bytes wide.
enum : int { kTurnIn = 1, kTurnOut = 2 };

// Load of a tile at an edge, or of unaligned rows: 16-byte pieces from any
// address, zeros past K and T.  Not inlined: its registers stay out of the
// kernels' main path.
__device__ __noinline__ void turn_tile_edge_load(const uint8_t* __restrict__ in, int T, int G, int K,
                                                 long long ks, int t0, int k0, int g, uint32_t* tile,
                                                 int tid) {
  const uint8_t* const end = in + ((long long)T * G - 1) * ks + K;
#pragma unroll 4
  for (int it = 0; it < 8; ++it) {
    const int e = it * 256 + tid, r = e >> 3, c = e & 7;
    uint32_t x[4] = {0u, 0u, 0u, 0u};
    if (t0 + r < T && k0 + 16 * c < K)
      ld16_any(in + ((long long)(t0 + r) * G + g) * ks + k0 + 16 * c, in, end, x);
    *reinterpret_cast<uint4*>(&tile[tile_word(r, 4 * c)]) = make_uint4(x[0], x[1], x[2], x[3]);
  }
}

// One tile: 256 threads (tid 0..255) move spectra t0 .. t0+255 of byte rows
// k0 .. k0+127 of group g through `tile`, meeting at barrier `bar`.  Input
// row (t, g) starts at in + (t G + g) ks: ks = K, or more for a range of
// rows cut from a wider block.  Tiles at the edges, and every tile of a block
// whose rows are not 32-byte aligned, load through ld16_any (HBM-bound as
// the aligned ones: a 100-input, 333-channel, 3001-spectra block, pushed and
// dumped, takes 0.132 ms, against 0.630 ms with byte loads and stores).
__device__ __forceinline__ void turn_tile(const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                          int T, int G, int K, long long ks, long long os, int vec,
                                          int pair_rows, int t0, int k0, int g, uint32_t* tile,
                                          int tid, int bar) {
  // load: 256 rows x 128 bytes as 32-byte pieces, four per thread, all
  // issued before any of them is stored
  const bool full = vec == (kTurnIn | kTurnOut) && t0 + kTT <= T && k0 + kTK <= K;
  if (full) {
    uint32_t v[4][8];
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int e = it * 256 + tid, r = e >> 2, p = e & 3;
      ld32B(in + ((long long)(t0 + r) * G + g) * ks + k0 + 32 * p, v[it]);
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int e = it * 256 + tid, r = e >> 2, p = e & 3;
      // odd rows store their second 16-byte half first: the two rows of a
      // quarter-warp then hit disjoint banks
      const bool odd = r & 1;
      const uint4 lo = make_uint4(v[it][0], v[it][1], v[it][2], v[it][3]);
      const uint4 hi = make_uint4(v[it][4], v[it][5], v[it][6], v[it][7]);
      *reinterpret_cast<uint4*>(&tile[tile_word(r, 8 * p + (odd ? 4 : 0))]) = odd ? hi : lo;
      *reinterpret_cast<uint4*>(&tile[tile_word(r, 8 * p + (odd ? 0 : 4))]) = odd ? lo : hi;
    }
  } else {
    turn_tile_edge_load(in, T, G, K, ks, t0, k0, g, tile, tid);
  }
  group_bar(bar);
  turn_tile_store(out, T, K, G, os, pair_rows, t0, k0, g, tile, tid, full, (vec & kTurnOut) != 0);
}

__global__ void __launch_bounds__(256, 4) turn_kernel(const uint8_t* __restrict__ in,
                                                      uint8_t* __restrict__ out, int T, int G,
                                                      int K, long long ks, long long os,
                                                      int vec, int pair_rows) {
  __shared__ __align__(16) uint32_t tile[kTT * 32];
  turn_tile(in, out, T, G, K, ks, os, vec, pair_rows, blockIdx.x * kTT, blockIdx.y * kTK,
            blockIdx.z, tile, threadIdx.x, 0);
}

// The same tiles from a fixed number of CTAs, one per SM, for a corner turn
// confined to a few SMs while the cross-multiply of the previous block holds
// the others.  Confined to a few SMs, the turn is bound by the bytes each SM
// keeps in flight, not by HBM: each of the kTurnGroups 256-thread groups of a
// CTA walks its own tiles through kTurnBufs 32 KB buffers, with the 16-byte
// cp.async copies of the next kTurnBufs - 1 tiles in flight while one tile is
// transposed and stored.  Edge tiles load synchronously.
#ifndef XE_TURN_GROUPS
#define XE_TURN_GROUPS 3
#endif
#ifndef XE_TURN_BUFS
#define XE_TURN_BUFS 2
#endif
constexpr int kTurnGroups = XE_TURN_GROUPS;
constexpr int kTurnBufs = XE_TURN_BUFS;
constexpr int kTurnAhead = kTurnBufs - 1;  // tiles in flight per group
constexpr int kTileWords = kTT * 32;
static_assert(kTurnBufs >= 2 && kTurnAhead <= 7, "cp.async.wait_group takes 0..7 here");
static_assert(kTurnGroups * kTurnBufs * kTileWords * 4 <= 227 * 1024,
              "the buffers must fit in one CTA's shared memory");

template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void cp_async16(uint32_t* dst, const uint8_t* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// Issue the copies of a full tile into `tile`, the same word placement as
// the register path of turn_tile: bytes 16c .. 16c+15 of a row go to words
// 4c .. 4c+3.  Consecutive threads take consecutive 16-byte chunks, so each
// warp instruction covers four whole 128-byte rows (every sector requested
// once, not half of it by each of two instructions).
__device__ __forceinline__ void tile_prefetch(const uint8_t* __restrict__ in, int G, long long ks, int t0,
                                              int k0, int g, uint32_t* tile, int tid) {
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int e = it * 256 + tid, r = e >> 3, c = e & 7;
    cp_async16(&tile[tile_word(r, 4 * c)], in + ((long long)(t0 + r) * G + g) * ks + k0 + 16 * c);
  }
}

__global__ void __launch_bounds__(256 * kTurnGroups, 1)
    turn_persist_kernel(const uint8_t* __restrict__ in, uint8_t* __restrict__ out, int T, int G,
                        int K, long long ks, long long os, int vec, int pair_rows) {
  extern __shared__ __align__(16) uint32_t tiles[];
  const int grp = threadIdx.x >> 8, tid = threadIdx.x & 255, bar = 1 + grp;
  uint32_t* const mine = tiles + kTurnBufs * grp * kTileWords;  // this group's buffers
  // tile indices in 32 bits (the host keeps their count below 2^31): the
  // per-tile index arithmetic is a visible share of this kernel's issue slots
  const unsigned gx = (unsigned)(T + kTT - 1) / kTT, gy = (unsigned)(K + kTK - 1) / kTK;
  const unsigned n = gx * gy * (unsigned)G;
  const unsigned stride = gridDim.x * kTurnGroups;
  auto coords = [&](unsigned w, int& t0, int& k0, int& g) {
    const unsigned r = w / gx, q = r / gy;
    t0 = (int)(w - r * gx) * kTT;
    k0 = (int)(r - q * gy) * kTK;
    g = (int)q;
  };
  auto is_full = [&](int t0, int k0) { return vec == (kTurnIn | kTurnOut) && t0 + kTT <= T && k0 + kTK <= K; };
  // copies of full tile w into buffer b; one commit group per tile, empty
  // for edge tiles and past the end, so that group i is always tile i
  auto prefetch = [&](unsigned w, int b) {
    if (w < n) {
      int t0, k0, g;
      coords(w, t0, k0, g);
      if (is_full(t0, k0)) tile_prefetch(in, G, ks, t0, k0, g, mine + b * kTileWords, tid);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  unsigned w = blockIdx.x * kTurnGroups + grp;
#pragma unroll
  for (int d = 0; d < kTurnAhead; ++d) prefetch(w + d * stride, d);
  // tile i sits in buffer i mod kTurnBufs; tile i + kTurnAhead goes into the
  // buffer of tile i - 1, released by the barrier that ended its iteration
  for (int b = 0; w < n; w += stride) {
    const int bn = b == 0 ? kTurnBufs - 1 : b - 1;
    prefetch(w + kTurnAhead * stride, bn);
    cp_async_wait<kTurnAhead>();  // the copies of this tile are in
    int t0, k0, g;
    coords(w, t0, k0, g);
    uint32_t* tile = mine + b * kTileWords;
    if (is_full(t0, k0)) {
      group_bar(bar);
      turn_tile_store(out, T, K, G, os, pair_rows, t0, k0, g, tile, tid, true, true);
    } else {
      turn_tile(in, out, T, G, K, ks, os, vec, pair_rows, t0, k0, g, tile, tid, bar);
    }
    group_bar(bar);
    if (++b == kTurnBufs) b = 0;
  }
  cp_async_wait<0>();
}

// ---------------------------------------------------------------- packet turn
// A block assembled in packet order -- [slot][fid][xid][8 spectra][chans_pkt
// x inputs_pkt bytes] -- becomes the X-engine's [c][i][t] rows.  For one
// (fid, xid) and 128 consecutive bytes k of a packet row, the spectra
// t = 8 slot + tt form a 256 x 128 tile like the corner turn's, except that
// a tile row's address steps by the packet stream stride every 8 spectra and
// each byte k names its own output row: channel xid chans_pkt + k / inputs_pkt,
// input fid inputs_pkt + k mod inputs_pkt.
struct PktGeom {
  int n_fids, inputs_pkt, n_xids, chans_pkt, T;
  long long os;
  int vec_in;   // 32-byte aligned packet rows
  int width;    // widest store every output row's 32-byte pieces allow: 32, 16, 8 or 1 byte(s)
};

__device__ __noinline__ void pkt_tile_edge_load(const uint8_t* __restrict__ in,
                                                const uint8_t* __restrict__ base, int T, int rowb,
                                                long long slot_stride, int t0, int k0, uint32_t* tile,
                                                int tid) {
  const uint8_t* const end = in + (long long)(T >> 3) * slot_stride;
#pragma unroll 4
  for (int it = 0; it < 8; ++it) {
    const int e = it * 256 + tid, r = e >> 3, c = e & 7, t = t0 + r;
    uint32_t x[4] = {0u, 0u, 0u, 0u};
    if (t < T && k0 + 16 * c < rowb)
      ld16_any(base + (long long)(t >> 3) * slot_stride + (long long)(t & 7) * rowb + k0 + 16 * c, in, end, x);
    *reinterpret_cast<uint4*>(&tile[tile_word(r, 4 * c)]) = make_uint4(x[0], x[1], x[2], x[3]);
  }
}

__global__ void __launch_bounds__(256, 4) pkt_turn_kernel(const uint8_t* __restrict__ in,
                                                          uint8_t* __restrict__ out, PktGeom q) {
  __shared__ __align__(16) uint32_t tile[kTT * 32];
  const int rowb = q.chans_pkt * q.inputs_pkt;           // bytes of one spectrum of a packet
  const long long P = 8LL * rowb;                        // payload bytes
  const long long slot_stride = (long long)q.n_fids * q.n_xids * P;
  const int t0 = blockIdx.x * kTT, k0 = blockIdx.y * kTK;
  const int stream = blockIdx.z, fid = stream / q.n_xids, xid = stream % q.n_xids;
  const int N = q.n_fids * q.inputs_pkt;
  const uint8_t* base = in + ((long long)fid * q.n_xids + xid) * P;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool full = q.vec_in && t0 + kTT <= q.T && k0 + kTK <= rowb;
  if (full) {
    uint32_t v[4][8];
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int e = it * 256 + tid, r = e >> 2, p = e & 3, t = t0 + r;
      ld32B(base + (long long)(t >> 3) * slot_stride + (long long)(t & 7) * rowb + k0 + 32 * p, v[it]);
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int e = it * 256 + tid, r = e >> 2, p = e & 3;
      const bool odd = r & 1;
      const uint4 lo = make_uint4(v[it][0], v[it][1], v[it][2], v[it][3]);
      const uint4 hi = make_uint4(v[it][4], v[it][5], v[it][6], v[it][7]);
      *reinterpret_cast<uint4*>(&tile[tile_word(r, 8 * p + (odd ? 4 : 0))]) = odd ? hi : lo;
      *reinterpret_cast<uint4*>(&tile[tile_word(r, 8 * p + (odd ? 0 : 4))]) = odd ? lo : hi;
    }
  } else {
    pkt_tile_edge_load(in, base, q.T, rowb, slot_stride, t0, k0, tile, tid);
  }
  __syncthreads();
  const int kq = 4 * warp + (lane >> 3), ts = lane & 7;
  uint32_t a[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) a[j] = tile[tile_word(ts * 32 + j, kq)];
#pragma unroll
  for (int j = 0; j < 32; j += 4) transpose4x4(a[j], a[j + 1], a[j + 2], a[j + 3]);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int k = k0 + 4 * kq + c;
    if (k >= rowb) continue;
    const int ch = xid * q.chans_pkt + k / q.inputs_pkt, inp = fid * q.inputs_pkt + k % q.inputs_pkt;
    const int tb = t0 + ts * 32;
    uint8_t* o = out + ((long long)ch * N + inp) * q.os + tb;
    const uint32_t r[8] = {a[c], a[4 + c], a[8 + c], a[12 + c],
                           a[16 + c], a[20 + c], a[24 + c], a[28 + c]};
    if (full && q.width == 32) {
      st32B(o, r);
      continue;
    }
    const int n = q.T - tb;  // spectra left of the row: a multiple of 8
    if (n <= 0) continue;
    if (q.width == 32 && n >= 32) {
      st32B(o, r);
    } else if (q.width >= 16 && n >= 32) {
      *reinterpret_cast<uint4*>(o) = make_uint4(r[0], r[1], r[2], r[3]);
      *reinterpret_cast<uint4*>(o + 16) = make_uint4(r[4], r[5], r[6], r[7]);
    } else if (q.width >= 8) {
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (8 * b < n) *reinterpret_cast<uint2*>(o + 8 * b) = make_uint2(r[2 * b], r[2 * b + 1]);
    } else {
#pragma unroll
      for (int b = 0; b < 32; ++b)
        if (b < n) o[b] = (uint8_t)(r[b >> 2] >> ((b & 3) * 8));
    }
  }
}

// ---------------------------------------------------------------- plane split
// out[r][p][t] = in[r][t][p] for 8-bit complex samples: 16 samples (32 bytes,
// any alignment) per thread become 16 real and 16 imaginary bytes.  The last
// 16 of a row run into its padding (vec: rows aligned to and padded to 16).
__global__ void split_planes_kernel(const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                    long long rows, int T, long long os, int vec) {
  const int per_row = (T + 15) / 16;
  const long long total = rows * per_row;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / per_row;
    const int t = (int)(e - r * per_row) * 16;
    const uint8_t* src = in + (r * T + t) * 2;
    uint8_t* dre = out + (2 * r) * os + t;
    uint8_t* dim = dre + os;
    if (vec) {
      uint32_t a[4], b[4];
      ld16_any(src, in, in + rows * T * 2, a);
      ld16_any(src + 16, in, in + rows * T * 2, b);
      // even bytes are real parts, odd bytes imaginary parts
      *reinterpret_cast<uint4*>(dre) =
          make_uint4(__byte_perm(a[0], a[1], 0x6420), __byte_perm(a[2], a[3], 0x6420),
                     __byte_perm(b[0], b[1], 0x6420), __byte_perm(b[2], b[3], 0x6420));
      *reinterpret_cast<uint4*>(dim) =
          make_uint4(__byte_perm(a[0], a[1], 0x7531), __byte_perm(a[2], a[3], 0x7531),
                     __byte_perm(b[0], b[1], 0x7531), __byte_perm(b[2], b[3], 0x7531));
    } else {
      for (int k = 0; k < 16 && t + k < T; ++k) {
        dre[k] = src[2 * k];
        dim[k] = src[2 * k + 1];
      }
    }
  }
}

// ---------------------------------------------------------------- row padding
// 4-bit [c][i][t] rows of T bytes (any alignment) copied to rows os bytes
// apart (aligned to and padded to 32 bytes), one 32-byte piece a thread.
__global__ void pad_rows_kernel(const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                long long rows, int T, long long os) {
  const int per_row = (T + 31) / 32;
  const long long total = rows * per_row;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long r = e / per_row;
    const int t = (int)(e - r * per_row) * 32;
    const uint8_t* src = in + r * T + t;
    uint32_t a[4], b[4];
    ld16_any(src, in, in + rows * T, a);
    ld16_any(src + 16, in, in + rows * T, b);
    const uint32_t w[8] = {a[0], a[1], a[2], a[3], b[0], b[1], b[2], b[3]};
    st32B(out + r * os + t, w);
  }
}

// ---------------------------------------------------------------- normalise
// rho = V / sqrt(V_ii V_jj) for a range of one channel's baselines.
//
// The FP64 pipe is 80 times narrower on this chip than FP32 (1.59 FMAs a cycle
// per SM, measured), and a square root and two divisions on it cost a baseline
// far more than its 32 bytes.  So both are made from float pairs and integers.
// A block keeps 1 / sqrt(V_ii) and sqrt(V_ii) of its channel's inputs in shared
// memory (one root per input, not per baseline) as float pairs.  Their
// products, and those with V's parts, give the 53-bit significands of the
// denominator and of the quotients to about 2^-45.  The remainders
// D - s^2 and a - q s are then below 2^63 and exact in the low 64 bits of
// integer products; they give the correction to within half a unit and a
// little, and the new remainder's sign against half a unit the last step.  So
// the results are those of sqrt and /.  One FP64 product a baseline is left,
// the denominator's square.  What bounds it now is the issue of some 230
// instructions a baseline (74% of the slots), then the 32 bytes (0.09 ms).
// The call (192 inputs x 1024 channels): 163 us; 345 with the roundings by
// FP64 residuals (7 operations of that pipe), 471 with the estimates in FP64
// too (11), 1700 with sqrt and two divisions.  64 x 512: 25 us.
constexpr int kNormThreads = 256;

// A correctly rounded square root: m 2^(e - 52), m in [2^52, 2^53), and
// 2^e over it as a float pair, good to 2^-45.
struct NormRoot {
  uint64_t m;
  int e;
  float yh, yl;
};

// The significand h + l, a float pair in units of its last bit over 2^28, as an integer.
__device__ __forceinline__ uint64_t sig_of(float h, float l) {
  return (uint64_t)(uint32_t)__float2int_rn(h) * (1u << 28) + (uint64_t)(2ll * __float2int_rn(l * 134217728.0f));
}
// Bits 32 .. 63 of p q.
__device__ __forceinline__ uint32_t product_word1(uint64_t p, uint64_t q) {
  const uint32_t pl = (uint32_t)p, ph = (uint32_t)(p >> 32), ql = (uint32_t)q, qh = (uint32_t)(q >> 32);
  return __umulhi(pl, ql) + pl * qh + ph * ql;
}
// A correction of c units, |c| < 2^10 and good to 2^-13, as an integer k; near
// says that c is too close to half a unit for its nearest integer to be sure.
__device__ __forceinline__ int nearest(float c, bool& near) {
  const float t = c + 12582912.0f;  // 1.5 2^23
  near = fabsf(c - (t - 12582912.0f)) > 0.499f;
  return (int)(__float_as_uint(t) - 0x4B400000u);
}

// sqrt(den2), den2 >= 1, from the pairs of 1 / sqrt(den2) and sqrt(den2).
__device__ __forceinline__ NormRoot norm_root(double den2, float yh, float yl, float sh, float sl) {
  const uint32_t hi = (uint32_t)__double2hiint(den2), lo = (uint32_t)__double2loint(den2);
  const int x = (int)(hi >> 20) - 1023;
  NormRoot r;
  r.e = x >> 1;
  const float up = __uint_as_float((uint32_t)(127 + r.e) << 23);
  const float dn = __uint_as_float((uint32_t)(151 - r.e) << 23);  // 2^24 over it
  r.yh = yh * up;
  r.yl = yl * up;
  const uint64_t m = sig_of(sh * dn, sl * dn);
  // den2 is n 2^(2 e - 104), n an integer of up to 106 bits: its low 64 are the
  // last 12 of den2's significand (doubled for odd exponents)
  const uint32_t n1 = lo << (20 + (x & 1));
  bool near;
  const int k = nearest((float)(int)(n1 - product_word1(m, m)) * (r.yh * 0x1p-21f), near);
  r.m = m + (uint64_t)(long long)k;
  if (near) {  // (m +- 1/2)^2 = m^2 +- m + 1/4
    const long long rem = (long long)(((uint64_t)n1 << 32) - r.m * r.m), mk = (long long)r.m;
    r.m += rem > mk ? 1 : rem <= -mk ? -1 : 0;
  }
  return r;
}

// a over the root's significand, a = |w| 2^(53 - bits) in [2^52, 2^53) and ah +
// al its leading bits as a float pair in [1, 2): the quotient, correctly
// rounded, with w's sign.
__device__ __forceinline__ double norm_quotient(uint64_t a, float ah, float al, int bits, uint32_t sign,
                                                const NormRoot& r) {
  const bool big = a >= r.m;  // the quotient of the significands is at least 1
  const float scale = big ? 0x1p24f : 0x1p25f;
  const float qh = ah * r.yh, ql = fmaf(al, r.yh, fmaf(ah, r.yl, fmaf(ah, r.yh, -qh)));
  uint64_t q = sig_of(qh * scale, ql * scale);
  const uint32_t a1 = (uint32_t)a << (big ? 20 : 21);  // bits 32 .. 63 of a 2^52, a 2^53
  bool near;
  const int k = nearest((float)(int)(a1 - product_word1(q, r.m)) * (r.yh * 0x1p-20f), near);
  q += (uint64_t)(long long)k;
  if (near) {
    const long long rem = (long long)(((uint64_t)a1 << 32) - q * r.m);
    q += 2 * rem > (long long)r.m ? 1 : 2 * rem < -(long long)r.m ? -1 : 0;
  }
  const uint32_t x = (uint32_t)(bits - 1 - r.e - (big ? 0 : 1) + 1022);
  return __hiloint2double((int)((x << 20) + (uint32_t)(q >> 32) + (sign & 0x80000000u)), (int)(uint32_t)q);
}

__device__ __noinline__ double norm_divide_wide(long long w, const NormRoot r) {
  const uint64_t u = (uint64_t)llabs(w);
  if (u >> 53)  // rounded to a double first
    return (double)w / __longlong_as_double((long long)(((uint64_t)(r.e + 1022) << 52) + r.m));
  const int z = __clzll((long long)u);
  const uint64_t a = u << z >> 11;
  const float ah = __uint_as_float((uint32_t)(a >> 29) + 0x3F000000u);
  const float al = (__uint_as_float(((uint32_t)a << 3 >> 9) | 0x3F800000u) - 1.0f) * 0x1p-23f;
  return norm_quotient(a, ah, al, 64 - z, (uint32_t)(w >> 32), r);
}
// w over the root, correctly rounded.
__device__ __forceinline__ double norm_divide(long long w, const NormRoot& r) {
  const int x = (int)w;
  if (w != (long long)x || x == (int)0x80000000) return norm_divide_wide(w, r);
  const uint32_t u = (uint32_t)abs(x);
  if (u == 0) return 0.0;
  const int z = __clz((int)u);
  const uint32_t t = u << z;
  const float ah = __uint_as_float((t >> 8) + 0x3F000000u);
  const float al = (__uint_as_float((t & 0xFFu) | 0x3F800000u) - 1.0f) * 0x1p-8f;
  return norm_quotient((uint64_t)t * (1u << 21), ah, al, 32 - z, (uint32_t)x, r);
}

// An input's factors: the power V_ii, and 1 / sqrt(V_ii) and sqrt(V_ii) as
// float pairs.
struct NormInput {
  double p;
  float yh, yl, rh, rl;
};

__global__ void __launch_bounds__(kNormThreads, 6)
    normalise_kernel(const int64_t* __restrict__ acc, double* __restrict__ rho,
                     uint8_t* __restrict__ zero_flag, int nbl, int per_block, int vec_ok) {
  extern __shared__ __align__(16) NormInput norm_sm[];
  const long long c = blockIdx.y;
  const int b0 = blockIdx.x * per_block, b1 = min(nbl, b0 + per_block);
  const int64_t* v = acc + c * nbl * 2;
  auto input_of = [](int b) {  // i with i (i + 1) / 2 <= b < (i + 1) (i + 2) / 2; 8 b + 1 < 2^24
    const float x = (float)(8 * b + 1);
    int i = (int)((x * rsqrtf(x) - 1.0f) * 0.5f);  // within one
    if (i * (i + 1) / 2 > b) --i;
    if ((i + 1) * (i + 2) / 2 <= b) ++i;
    return i;
  };
  const int last = input_of(b1 - 1);  // no baseline of the range has a larger input
  for (int i = threadIdx.x; i <= last; i += kNormThreads) {
    NormInput n;
    const long long p = v[i * (i + 3)];
    n.p = (double)p;
    // |p| as a float pair; a Newton step from the FP32 estimate, in pairs:
    // y + y e / 2 + 3 y e^2 / 8 with e = 1 - p y^2
    const float ph = (float)p, pl = (float)(p - (long long)ph), y = rsqrtf(fabsf(ph));
    const float ah = fabsf(ph), al = ph < 0.f ? -pl : pl, t = y * y;
    const float e = fmaf(-al, t, fmaf(-ah, fmaf(y, y, -t), fmaf(-ah, t, 1.0f)));
    n.yh = y;
    n.yl = y * fmaf(0.375f * e, e, 0.5f * e);
    n.rh = ah * y;
    n.rl = fmaf(al, y, fmaf(ah, n.yl, fmaf(ah, y, -n.rh)));
    norm_sm[i] = n;
  }
  __syncthreads();
  int i = input_of(b0 + (int)threadIdx.x), j = b0 + (int)threadIdx.x - i * (i + 1) / 2;
  for (int b = b0 + (int)threadIdx.x; b < b1; b += kNormThreads, j += kNormThreads) {
    for (; j > i; j -= ++i) {
    }
    const long long e = c * nbl + b;
    long long vr, vi;
    if (vec_ok) {
      ld_s64x2(v + 2 * b, vr, vi);
    } else {
      vr = v[2 * b];
      vi = v[2 * b + 1];
    }
    const NormInput ni = norm_sm[i], nj = norm_sm[j];
    const double den2 = ni.p * nj.p;
    double re = 0.0, im = 0.0;
    const int top = __double2hiint(den2);  // |den2| is 0 or at least 1: its sign and zero from the high word
    if (top > 0) {
      // 1 / sqrt(den2) and sqrt(den2) as float pairs
      const float yh = ni.yh * nj.yh;
      const float yl = fmaf(ni.yl, nj.yh, fmaf(ni.yh, nj.yl, fmaf(ni.yh, nj.yh, -yh)));
      const float sh = ni.rh * nj.rh;
      const float sl = fmaf(ni.rl, nj.rh, fmaf(ni.rh, nj.rl, fmaf(ni.rh, nj.rh, -sh)));
      const NormRoot root = norm_root(den2, yh, yl, sh, sl);
      re = norm_divide(vr, root);
      im = norm_divide(vi, root);
    } else if ((top << 1) != 0) {
      re = im = sqrt(den2);  // not a power: NaN
    }
    if (vec_ok) {
      *reinterpret_cast<double2*>(rho + 2 * e) = make_double2(re, im);
    } else {
      rho[2 * e] = re;
      rho[2 * e + 1] = im;
    }
    if (zero_flag) zero_flag[e] = (top << 1) == 0 ? 1 : 0;
  }
}

}  // namespace

cudaError_t turn_launch(const uint8_t* in, uint8_t* out, int T, int G, int K, long long out_stride,
                        cudaStream_t s, bool pair_rows, int persist_ctas) {
  return turn_launch_strided(in, out, T, G, K, K, out_stride, s, pair_rows, persist_ctas);
}

cudaError_t turn_launch_strided(const uint8_t* in, uint8_t* out, int T, int G, int K,
                                long long in_stride, long long out_stride, cudaStream_t s,
                                bool pair_rows, int persist_ctas) {
  if (in_stride < K) return cudaErrorInvalidValue;
  const int vec =
      (in_stride % 32 == 0 && reinterpret_cast<uintptr_t>(in) % 32 == 0 ? kTurnIn : 0) |
      (out_stride % 32 == 0 && reinterpret_cast<uintptr_t>(out) % 32 == 0 ? kTurnOut : 0);
  const long long n_tiles = (long long)((T + kTT - 1) / kTT) * ((K + kTK - 1) / kTK) * G;
  if (persist_ctas > 0 && n_tiles + (long long)persist_ctas * kTurnGroups * kTurnBufs < (1LL << 31)) {
    constexpr int smem = kTurnGroups * kTurnBufs * kTileWords * (int)sizeof(uint32_t);
    static bool attr = false;
    if (!attr) {
      cudaError_t e = cudaFuncSetAttribute(turn_persist_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
      if (e != cudaSuccess) return e;
      attr = true;
    }
    turn_persist_kernel<<<persist_ctas, 256 * kTurnGroups, smem, s>>>(
        in, out, T, G, K, in_stride, out_stride, vec, pair_rows ? 1 : 0);
    return cudaGetLastError();
  }
  dim3 grid((T + kTT - 1) / kTT, (K + kTK - 1) / kTK, G);
  turn_kernel<<<grid, 256, 0, s>>>(in, out, T, G, K, in_stride, out_stride, vec, pair_rows ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t split_planes_launch(const uint8_t* in, uint8_t* out, long long rows, int T,
                                long long out_stride, cudaStream_t s) {
  const int vec = out_stride % 16 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0;
  const long long total = rows * ((T + 15) / 16);
  long long blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  if (blocks < 1) blocks = 1;
  split_planes_kernel<<<(unsigned)blocks, 256, 0, s>>>(in, out, rows, T, out_stride, vec);
  return cudaGetLastError();
}

cudaError_t pad_rows_launch(const uint8_t* in, uint8_t* out, long long rows, int T,
                            long long out_stride, cudaStream_t s) {
  if (out_stride % 32 != 0 || out_stride < T || reinterpret_cast<uintptr_t>(out) % 32 != 0)
    return cudaErrorInvalidValue;
  const long long blocks = (rows * ((T + 31) / 32) + 255) / 256;
  pad_rows_kernel<<<(unsigned)std::min<long long>(blocks, device_sm_count() * 64), 256, 0, s>>>(
      in, out, rows, T, out_stride);
  return cudaGetLastError();
}

cudaError_t pkt_turn_launch(const uint8_t* in, uint8_t* out, int n_fids, int inputs_pkt, int n_xids,
                            int chans_pkt, int T, long long out_stride, cudaStream_t s) {
  PktGeom q{n_fids, inputs_pkt, n_xids, chans_pkt, T, out_stride, 0, 1};
  const int rowb = chans_pkt * inputs_pkt;
  q.vec_in = rowb % 32 == 0 && reinterpret_cast<uintptr_t>(in) % 32 == 0;
  for (int w : {8, 16, 32})
    if (out_stride % w == 0 && reinterpret_cast<uintptr_t>(out) % w == 0) q.width = w;
  dim3 grid((T + kTT - 1) / kTT, (rowb + kTK - 1) / kTK, n_fids * n_xids);
  pkt_turn_kernel<<<grid, 256, 0, s>>>(in, out, q);
  return cudaGetLastError();
}

bool needs_turn(int layout, int bits) { return layout != 2 || bits == 8; }

bool turn_can_persist(int layout, int bits) { return needs_turn(layout, bits) && layout != 2; }

cudaError_t turn_rows(const uint8_t* in, uint8_t* out, int layout, int bits, int n_inputs,
                      int n_chans, int n_time, long long out_stride, cudaStream_t s,
                      int persist_ctas) {
  const int N = n_inputs, C = n_chans, T = n_time;
  const bool eight = bits == 8;
  const int R = eight ? 2 * N : N;
  // [t][c][i] is one transpose of a T x (C N) byte matrix, [t][i][c] is N
  // transposes of T x C.  8-bit samples are byte pairs: [t][c][i][p] turns as
  // T x (C 2N); [t][i][c][p] as N transposes of T x 2C with each (c, p) row
  // sent to row (c, i, p); [c][i][t][p] only splits the planes.
  if (layout == 0) return turn_launch(in, out, T, 1, C * R, out_stride, s, false, persist_ctas);
  if (layout == 1)
    return eight ? turn_launch(in, out, T, N, 2 * C, out_stride, s, true, persist_ctas)
                 : turn_launch(in, out, T, N, C, out_stride, s, false, persist_ctas);
  if (eight) return split_planes_launch(in, out, (long long)C * N, T, out_stride, s);
  return cudaSuccess;
}

cudaError_t turn_rows_chans(const uint8_t* in, uint8_t* out, int layout, int bits, int n_inputs,
                            int n_chans, int n_time, int c0, int c1, long long out_stride,
                            cudaStream_t s, int persist_ctas) {
  const int N = n_inputs, C = n_chans, T = n_time;
  if (bits != 4 || c0 < 0 || c1 > C || c0 >= c1) return cudaErrorInvalidValue;
  // channels c0 .. c1-1 are output rows c N + i for c0 <= c < c1
  uint8_t* o = out + (long long)c0 * N * out_stride;
  if (layout == 0)  // [t][c][i]: bytes c0 N .. c1 N of each spectrum
    return turn_launch_strided(in + (long long)c0 * N, o, T, 1, (c1 - c0) * N, (long long)C * N,
                               out_stride, s, false, persist_ctas);
  if (layout == 1)  // [t][i][c]: bytes c0 .. c1 of each (spectrum, input) row
    return turn_launch_strided(in + c0, o, T, N, c1 - c0, C, out_stride, s, false, persist_ctas);
  return cudaErrorInvalidValue;
}

// One thread: copy the status word into a slot of pinned host memory
// (written through its device mapping) and clear it, in stream order.
__global__ void take_status_kernel(int* status, int* host_slot) {
  *host_slot = *status;
  *status = 0;
}

cudaError_t take_status_launch(int* status, int* host_slot, cudaStream_t s) {
  take_status_kernel<<<1, 1, 0, s>>>(status, host_slot);
  return cudaGetLastError();
}

cudaError_t normalise_launch(const int64_t* acc, double* rho, uint8_t* zero_flag, int n_inputs,
                             int n_chans, cudaStream_t s) {
  const int nbl = n_inputs * (n_inputs + 1) / 2;  // at most 524800 (1024 inputs)
  // Blocks of a few thousand baselines: enough of them to fill the SMs several
  // times over, large enough that the inputs' rsqrt stay a small share.
  const int want = std::max(1, device_sm_count() * 32 / n_chans);
  const int per = std::max(kNormThreads, (nbl + want - 1) / want);
  const int vec_ok = reinterpret_cast<uintptr_t>(acc) % 16 == 0 && reinterpret_cast<uintptr_t>(rho) % 16 == 0;
  const size_t smem = (size_t)n_inputs * sizeof(NormInput);
  for (int c0 = 0; c0 < n_chans; c0 += 65535) {  // grid.y
    const int nc = std::min(65535, n_chans - c0);
    const long long e0 = (long long)c0 * nbl;
    normalise_kernel<<<dim3((nbl + per - 1) / per, nc), kNormThreads, smem, s>>>(
        acc + 2 * e0, rho + 2 * e0, zero_flag ? zero_flag + e0 : nullptr, nbl, per, vec_ok);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace xe
