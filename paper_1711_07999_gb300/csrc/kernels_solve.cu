// kernels_solve.cu -- point-to-plane residuals and the pose Jacobian (Eq. residual, Sec. 4.2), the
// reduction [J r]^T [J r] (Eqs. JTJ, JTr), the damped least-squares step with the pose prior and its
// energy test (Sec. 4.2), and the per-vertex shape step (Eq. r_warp, Sec. 4.3).
//
// Reductions are deterministic: per-block partial sums over fixed vertex ranges, then a second pass
// that adds the partials in a fixed order (error-free FP32 within a warp, FP64 across warps).  The LM
// retries of one iteration (damping lambda, 10 lambda, ..., 10^5 lambda) are solved side by side, one CTA
// each, and their energies evaluated over the vertices; the first candidate that does not raise the
// energy is taken on the device, which gives the same result as trying them one after the other without
// any host round trip.
#include <mutex>

#include "tcgen05.cuh"
#include "trk_internal.cuh"

namespace trk {

constexpr int kBlock = 256;

__device__ __forceinline__ float3 f3(float4 a) { return make_float3(a.x, a.y, a.z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// L(c, h) = -c_w h_vec + h_w c_vec + h_vec x c_vec: for a pure quaternion (0, xi),
// <c, (0, xi) h> = xi . L(c, h).
__device__ __forceinline__ float3 Lfun(float4 c, float4 h) {
  return make_float3(-c.x * h.y + h.x * c.y + (h.z * c.w - h.w * c.z),
                     -c.x * h.z + h.x * c.z + (h.w * c.y - h.y * c.w),
                     -c.x * h.w + h.x * c.w + (h.y * c.z - h.z * c.y));
}

// ---------------------------------------------------------------------------------------------
// Residual r_i = n_i . (p~_i - v_i) and Jacobian row dr_i/dTheta for every vertex of A, followed by
// the block's partial [J r]^T [J r].
//
// Jacobian: with c = n^T dT/dH (an 8-vector: the normal pulled back through the homogeneous point map
// at H_iSigma) and dH_iSigma/dtheta_k = sum_b w_b s_b Xi_k H_{b,Delta} over the bones b below k,
//   J_ik = -sum_b w_b s_b <c, Xi_k H_{b,Delta}> = -sum_b Xi_k . e_b,
//   e_b = w_b s_b (L(c_r, h_r) + L(c_d, h_d), L(c_d, h_r)),
// so each bone costs one 6-vector and each ancestor link one 6-term dot product.
//   c_r = (-2 N a X - 2 N b - 2 (n.v) a) / |a|^2,  c_d = 2 N a / |a|^2,  N = (0, n), X = (0, x).
// The block's rows (compacted to A) are staged in shared memory; 16 x 16 threads each own a TxT tile
// of the (16T) x (16T) product and sweep the rows.
// ---------------------------------------------------------------------------------------------
// Copies the link tables this block needs to shared memory: H_Delta, and per link eight floats (the twist
// Xi, the parent's index as bits, unused), read as two 16-byte pieces in the Jacobian's walk.
__device__ __forceinline__ void load_link_tables(const Dev& d, DQ* sHd, float* sXi) {
  for (int t = threadIdx.x; t < 2 * d.L; t += kBlock) {
    reinterpret_cast<float4*>(sHd)[t] = reinterpret_cast<const float4*>(d.Hd)[t];
    float4 x = reinterpret_cast<const float4*>(d.xi)[t];
    if (t & 1) x.z = __int_as_float(d.links->parent[t >> 1]);
    reinterpret_cast<float4*>(sXi)[t] = x;
  }
}

// This block's vertices in A (c_i >= 1 and a valid normal) and each one's row slot, compacted in vertex
// order, with every input of the vertex's row (all loaded at once: one round trip, the point data of
// vertices outside A read and dropped).  Contains a __syncthreads; returns the number of rows (the same
// in every thread).
struct RowSlot {
  int i, slot, base;  // vertex, its row among the vertex block's rows, the record index of row 0
  bool inA;
  Acc4 a4;
  float4 nn, v, x0, ph, bw;
  uchar4 bi;
};
__device__ __forceinline__ int block_rows(const Dev& d, int blk, int row_base, int phi_buf, int* s_warp,
                                         RowSlot& rs) {
  const int tid = threadIdx.x;
  rs.i = blk * kBlock + tid;
  rs.base = row_base;
  rs.inA = false;
  rs.a4 = Acc4{0, 0, 0, 0};
  rs.nn = make_float4(0.f, 0.f, 0.f, 0.f);
  rs.v = rs.x0 = rs.ph = rs.bw = rs.nn;
  rs.bi = make_uchar4(0, 0, 0, 0);
  if (rs.i < d.V) {
    rs.a4 = d.acc[rs.i];
    rs.nn = d.n[rs.i];
    rs.v = d.v[rs.i];
    rs.x0 = d.v0[rs.i];
    rs.ph = d.phi[phi_buf][rs.i];
    rs.bi = d.bidx[rs.i];
    rs.bw = d.bw[rs.i];
    rs.inA = rs.a4.w >= 1 && rs.nn.w > 0.f;
  }
  const unsigned m = __ballot_sync(0xffffffffu, rs.inA);
  const int lane = tid & 31, w = tid >> 5;
  if (lane == 0) s_warp[w] = __popc(m);
  __syncthreads();
  int off = 0, total = 0;
  for (int k = 0; k < kBlock / 32; ++k) {
    off += k < w ? s_warp[k] : 0;
    total += s_warp[k];
  }
  rs.slot = off + __popc(m & ((1u << lane) - 1u));
  return total;
}

// Writes this thread's [J r] row (if its vertex is in A) to Js row rs.slot (stride ROW, columns
// [0, width) with width >= NP, zero beyond NP) and sets r2 = r_i^2 (0 outside A).  The link tables must
// be in shared memory; the caller synchronises before reading Js.
__device__ __forceinline__ void jacobian_row(const Dev& d, const RowSlot& rs, int phi_buf, float* Js, int ROW,
                                             int width, const DQ* sHd, const float* sXi, float& r2) {
  r2 = 0.f;
  if (!rs.inA) return;
  const Acc4 a4 = rs.a4;
  float* row = Js + rs.slot * ROW;
  if ((ROW & 3) == 0 && (width & 3) == 0) {  // 16-byte rows: 128-bit stores
    for (int k = 0; k < width; k += 4) *reinterpret_cast<float4*>(row + k) = make_float4(0.f, 0.f, 0.f, 0.f);
  } else {
    for (int k = 0; k < width; ++k) row[k] = 0.f;
  }
  const float inv = 1.f / ((float)a4.w * kFix);
  const float3 pm = make_float3((float)a4.x * inv, (float)a4.y * inv, (float)a4.z * inv);
  const float3 n = f3(rs.nn);
  const float r = dot3(n, pm);
  row[d.L] = r;
  r2 = r * r;
  float sg[4];
  const uchar4 bi = rs.bi;
  const float4 bw = rs.bw;
  const DQ H = blend_bones(sHd, bi, bw, sg);
  const float4 x0 = rs.x0, ph = rs.ph, v = rs.v;
  const float4 X = make_float4(0.f, x0.x + ph.x, x0.y + ph.y, x0.z + ph.z);
  {  // the row's record for the candidate energies: p~ = v + pm, n, x = x0 + phi, bones and weights
    float4* rec = d.arec + (size_t)(rs.base + rs.slot) * 4;
    unsigned bits;
    memcpy(&bits, &bi, 4);
    rec[0] = make_float4(v.x + pm.x, v.y + pm.y, v.z + pm.z, n.x);
    rec[1] = make_float4(n.y, n.z, X.y, X.z);
    rec[2] = make_float4(X.w, bw.x, bw.y, bw.z);
    rec[3] = make_float4(bw.w, __uint_as_float(bits), 0.f, 0.f);
  }
  const float4 Np = make_float4(0.f, n.x, n.y, n.z);
  const float invN = 1.f / qdot(H.r, H.r);
  const float4 Na = qmul(Np, H.r);
  const float4 cr = qscale(qadd(qadd(qmul(Na, X), qmul(Np, H.d)), qscale(H.r, dot3(n, f3(v)))), -2.f * invN);
  const float4 cd = qscale(Na, 2.f * invN);
  const int idx[4] = {bi.x, bi.y, bi.z, bi.w};
  const float ws[4] = {bw.x, bw.y, bw.z, bw.w};
  // e_b of every weighted bone, keyed by its link (-1: no weight)
  int key[4];
  float es[4][6];
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    key[s] = -1;
#pragma unroll
    for (int c = 0; c < 6; ++c) es[s][c] = 0.f;
    if (!(ws[s] > 0.f)) continue;
    key[s] = idx[s];
    const DQ h = sHd[idx[s]];
    const float sc = ws[s] * sg[s];
    const float3 e1 = Lfun(cr, h.r), e2 = Lfun(cd, h.d), e3 = Lfun(cd, h.r);
    es[s][0] = sc * (e1.x + e2.x);
    es[s][1] = sc * (e1.y + e2.y);
    es[s][2] = sc * (e1.z + e2.z);
    es[s][3] = sc * e3.x;
    es[s][4] = sc * e3.y;
    es[s][5] = sc * e3.z;
  }
  // J_ik = -Xi_k . (sum of e_b over the bones b at or below k).  The bones, sorted by link (parents
  // precede their children), are walked to the root from the deepest one; a bone met on the way joins
  // the running sum, so a link shared by several bones' chains is visited once.  A bone on another
  // branch is not met and starts its own walk afterwards (sums are linear, so every bone still reaches
  // each of its ancestors exactly once).
  auto cswap = [&](int a, int b) {
    if (key[a] < key[b]) {
      const int t = key[a];
      key[a] = key[b];
      key[b] = t;
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const float u = es[a][c];
        es[a][c] = es[b][c];
        es[b][c] = u;
      }
    }
  };
  cswap(0, 1);
  cswap(2, 3);
  cswap(0, 2);
  cswap(1, 3);
  cswap(1, 2);
  auto pop = [&]() {  // drops the head of the sorted queue
    key[0] = key[1];
    key[1] = key[2];
    key[2] = key[3];
    key[3] = -1;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      es[0][c] = es[1][c];
      es[1][c] = es[2][c];
      es[2][c] = es[3][c];
    }
  };
  while (key[0] >= 0) {
    int k = key[0];
    float E[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) E[c] = es[0][c];
    pop();
    while (k >= 0) {
      const float4 xa = *reinterpret_cast<const float4*>(sXi + 8 * k), xb = *reinterpret_cast<const float4*>(sXi + 8 * k + 4);
      const float old = row[k];
      while (key[0] == k) {
#pragma unroll
        for (int c = 0; c < 6; ++c) E[c] += es[0][c];
        pop();
      }
      row[k] = old - (xa.x * E[0] + xa.y * E[1] + xa.z * E[2] + xa.w * E[3] + xb.x * E[4] + xb.y * E[5]);
      k = __float_as_int(xb.z);
    }
  }
}

// Row stride of the staged rows: 16T columns, padded so that rows of even T start on 16 bytes (vector loads
// of a tile's T entries) and rows of odd T fall on distinct banks.
__host__ __device__ constexpr int jtj_row_stride(int T) { return 16 * T + (T % 2 == 0 ? 4 : 1); }
constexpr int kMaxRowGroups = 4;

// Packed FP32 pairs: fma.rn.f32x2 rounds each lane as fmaf does, so a tile updated pairwise holds the same
// bits as one updated entry by entry.
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(unsigned long long v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void f2_fma(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// One thread's T x T tile of the product: acc[a][b] += ra[a] rb[b] over the rows it sweeps.
template <int T>
struct TileAcc {
  static constexpr bool kPaired = T % 2 == 0;
  unsigned long long p[kPaired ? T : 1][kPaired ? T / 2 : 1];
  float f[kPaired ? 1 : T][kPaired ? 1 : T];
  __device__ __forceinline__ void zero() {
    if constexpr (kPaired) {
#pragma unroll
      for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T / 2; ++b) p[a][b] = 0ull;
    } else {
#pragma unroll
      for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) f[a][b] = 0.f;
    }
  }
  // adds one staged row: entries [ty T, ty T + T) and [tx T, tx T + T)
  __device__ __forceinline__ void add_row(const float* row, int ty, int tx) {
    float ra[T], rb[T];
    if constexpr (T == 4) {
      const float4 A = *reinterpret_cast<const float4*>(row + ty * 4);
      const float4 B = *reinterpret_cast<const float4*>(row + tx * 4);
      ra[0] = A.x, ra[1] = A.y, ra[2] = A.z, ra[3] = A.w;
      rb[0] = B.x, rb[1] = B.y, rb[2] = B.z, rb[3] = B.w;
    } else {
#pragma unroll
      for (int a = 0; a < T; ++a) {
        ra[a] = row[ty * T + a];
        rb[a] = row[tx * T + a];
      }
    }
    if constexpr (kPaired) {
      unsigned long long B2[T / 2];
#pragma unroll
      for (int b = 0; b < T / 2; ++b) B2[b] = f2_pack(rb[2 * b], rb[2 * b + 1]);
#pragma unroll
      for (int a = 0; a < T; ++a) {
        const unsigned long long A2 = f2_pack(ra[a], ra[a]);
#pragma unroll
        for (int b = 0; b < T / 2; ++b) f2_fma(p[a][b], A2, B2[b]);
      }
    } else {
#pragma unroll
      for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) f[a][b] = fmaf(ra[a], rb[b], f[a][b]);
    }
  }
  __device__ __forceinline__ float get(int a, int b) const {
    if constexpr (kPaired) {
      float lo, hi;
      f2_unpack(p[a][b / 2], lo, hi);
      return (b & 1) ? hi : lo;
    } else {
      return f[a][b];
    }
  }
  __device__ __forceinline__ void add(int a, int b, float x) {
    if constexpr (kPaired) {
      float lo, hi;
      f2_unpack(p[a][b / 2], lo, hi);
      if (b & 1) hi += x; else lo += x;
      p[a][b / 2] = f2_pack(lo, hi);
    } else {
      f[a][b] += x;
    }
  }
};

// Every input of vertex i's row (RowSlot of a vertex known to be in A; slot and base set by the caller).
__device__ __forceinline__ void row_inputs(const Dev& d, int i, int phi_buf, RowSlot& rs) {
  rs.i = i;
  rs.inA = true;
  rs.a4 = d.acc[i];
  rs.nn = d.n[i];
  rs.v = d.v[i];
  rs.x0 = d.v0[i];
  rs.ph = d.phi[phi_buf][i];
  rs.bi = d.bidx[i];
  rs.bw = d.bw[i];
}

// A [J r] block covers jtj_group consecutive blocks of 256 vertices.  Its vertices in A are listed first,
// in vertex order (a vertex's thread tests c_i >= 1 and a valid normal: two small loads), and their rows
// are then formed 256 at a time by consecutive threads -- every thread of a chunk holds a row, instead of
// the third of a vertex block's threads whose vertices are in A -- staged, and added to the same tiles,
// so the block writes one partial for up to 256 G rows.
// The symmetric product needs only the tiles (ty, tx) with ty <= tx among the nt x nt tiles that hold
// columns < NP; S groups of nt (nt + 1) / 2 threads (S = 2 for NP <= 60 at T = 4) each sweep every S-th
// staged row, and the first group adds the other groups' tiles, in group order, before the block writes
// its partial: a fixed order, so the partial is the same in any launch.
template <int T>
__device__ __forceinline__ void resid_jtj_impl(const Dev& d, BlockPos bp, int phi_buf) {
  constexpr int ROW = jtj_row_stride(T);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* Js = reinterpret_cast<float*>(smem_raw);
  DQ* sHd = reinterpret_cast<DQ*>(Js + kBlock * ROW);
  float* sXi = reinterpret_cast<float*>(sHd + d.L);
  __shared__ int s_cnt[kMaxJtjGroup * (kBlock / 32)];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, G = d.jtj_group;
  const int NP = d.NP;
  const int nt = (NP + T - 1) / T;
  const int ntiles = nt * (nt + 1) / 2;
  const int S = min(kMaxRowGroups, kBlock / ntiles);
  const int h = tid / ntiles;  // this thread's row group (h >= S: idle in the product)
  int ty = 0, k = tid - h * ntiles;
  while (ty < nt && k >= nt - ty) {  // the k-th tile of the upper triangle, row-major
    k -= nt - ty;
    ++ty;
  }
  const int tx = ty + k;
  // the block's rows: membership of A of vertex tid of each vertex block, counted per (block, warp)
  unsigned m[kMaxJtjGroup];
#pragma unroll
  for (int sub = 0; sub < kMaxJtjGroup; ++sub) {
    const int i = (bp.x * G + sub) * kBlock + tid;
    bool inA = false;
    if (sub < G && i < d.V) inA = d.acc[i].w >= 1 && d.n[i].w > 0.f;
    m[sub] = __ballot_sync(0xffffffffu, inA);
    if (lane == 0) s_cnt[sub * (kBlock / 32) + w] = __popc(m[sub]);
  }
  load_link_tables(d, sHd, sXi);
  __syncthreads();
  int total = 0;
  for (int q = 0; q < G * (kBlock / 32); ++q) total += s_cnt[q];
  if (total == 0) {  // nothing to add: the reduction skips this block's (unwritten) partial
    if (tid == 0) d.jtj_rows[bp.x] = 0;
    return;
  }
  {  // the list, in vertex order, staged where the rows go (each thread takes its entries before any row)
    int* s_idx = reinterpret_cast<int*>(Js);
    int off = 0;
#pragma unroll
    for (int sub = 0; sub < kMaxJtjGroup; ++sub) {
      if (sub >= G) break;
      int before = off;
      for (int q = sub * (kBlock / 32); q < sub * (kBlock / 32) + w; ++q) before += s_cnt[q];
      if ((m[sub] >> lane) & 1u) s_idx[before + __popc(m[sub] & ((1u << lane) - 1u))] = (bp.x * G + sub) * kBlock + tid;
      for (int q = 0; q < kBlock / 32; ++q) off += s_cnt[sub * (kBlock / 32) + q];
    }
  }
  __syncthreads();
  int mine[kMaxJtjGroup];
#pragma unroll
  for (int c = 0; c < kMaxJtjGroup; ++c) mine[c] = c * kBlock + tid < total ? reinterpret_cast<const int*>(Js)[c * kBlock + tid] : -1;
  __syncthreads();
  TileAcc<T> acc;
  acc.zero();
#pragma unroll
  for (int c = 0; c < kMaxJtjGroup; ++c) {
    const int c0 = c * kBlock;
    if (c0 >= total) break;
    const int rows = min(kBlock, total - c0);
    if (c > 0) __syncthreads();  // the previous chunk's rows have been added
    if (mine[c] >= 0) {
      RowSlot rs;
      row_inputs(d, mine[c], phi_buf, rs);
      rs.slot = tid;
      rs.base = bp.x * kBlock * G + c0;
      float r2;
      jacobian_row(d, rs, phi_buf, Js, ROW, 16 * T, sHd, sXi, r2);
    }
    __syncthreads();
    if (h < S) {
      // eight rows' loads ahead of their products (a row at a time waits for its loads: 62 cycles a row, not 25)
      int s = h;
#pragma unroll 1
      for (; s + 7 * S < rows; s += 8 * S) {
#pragma unroll
        for (int u = 0; u < 8; ++u) acc.add_row(Js + (s + u * S) * ROW, ty, tx);
      }
#pragma unroll 1
      for (; s < rows; s += S) acc.add_row(Js + s * ROW, ty, tx);
    }
  }
  const int done = total;
  if (S > 1) {  // the groups' tiles, added into group 0's in group order
    __syncthreads();  // every group's sweep is done: the staged rows are free
    float* red = Js;
    if (h >= 1 && h < S)
#pragma unroll
      for (int a = 0; a < T; ++a)
#pragma unroll
        for (int b = 0; b < T; ++b) red[((h - 1) * T * T + a * T + b) * ntiles + (tid - h * ntiles)] = acc.get(a, b);
    __syncthreads();
    if (h == 0)
      for (int g2 = 1; g2 < S; ++g2)
#pragma unroll
        for (int a = 0; a < T; ++a)
#pragma unroll
          for (int b = 0; b < T; ++b) acc.add(a, b, red[((g2 - 1) * T * T + a * T + b) * ntiles + tid]);
  }
  if (h == 0) {
    float* out = d.partial + (size_t)bp.x * NP * NP;
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
      for (int b = 0; b < T; ++b) {
        const int r = ty * T + a, c = tx * T + b;
        if (r < NP && c < NP && r <= c) out[r * NP + c] = acc.get(a, b);  // the upper triangle (the reduction mirrors)
      }
  }
  if (tid == 0) {
    d.jtj_rows[bp.x] = done;
    atomicAdd(&d.stats[1], done);
  }
}

template <int T>
__global__ void __launch_bounds__(kBlock, 3) k_resid_jtj(BatchGrid g, Dev d0, int phi_buf) {
  if (g.map == nullptr) {
    resid_jtj_impl<T>(d0, grid_pos(), phi_buf);
    return;
  }
  __shared__ Dev sd;
  resid_jtj_impl<T>(sd, batch_block(g, sd), phi_buf);
}

// ---------------------------------------------------------------------------------------------
// The same rows contracted on the tensor cores (split-BF16x3 or 3xTF32, PREC 1 / 2): the block's rows
// are taken in chunks of TL::K (64 BF16 / 32 TF32 rows), split into hi + lo K-major tiles and multiplied
// by one issuing thread into an FP32 accumulator in tensor memory (128 lanes x N columns; lane = parameter
// a, column = parameter b).  The energy entry [r]^T [r] is summed on the FP32 cores instead, so that the
// LM acceptance test compares energies formed the same way in every precision mode.  One stage of tiles
// (the next chunk waits for the previous chunk's MMAs) keeps the block at ~105 KB of shared memory, two
// blocks per SM; their 2 x 128 TMEM columns fit the 512 of an SM, so tcgen05.alloc never waits.
// ---------------------------------------------------------------------------------------------
template <int PREC, int NB>
__device__ __forceinline__ void resid_jtj_tc_impl(const Dev& d, BlockPos bp, int phi_buf) {
  using TL = tc::Tile<PREC, 8>;
  constexpr int N = 16 * NB, ROW = N + 1, T = TL::T;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* tiles = smem_raw;  // hi tile, lo tile
  float* Js = reinterpret_cast<float*>(smem_raw + TL::STAGE);
  DQ* sHd = reinterpret_cast<DQ*>(Js + kBlock * ROW);
  float* sXi = reinterpret_cast<float*>(sHd + d.L);
  __shared__ int s_warp[kBlock / 32];
  __shared__ float s_e[kBlock / 32];
  __shared__ uint64_t bar;
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int NP = d.NP, G = d.jtj_group;
  // The rows of the block's G vertex blocks go into the same TMEM accumulator, chunk after chunk; the
  // tensor memory is taken when the first rows appear (a block without rows takes none).
  int done = 0, gq = 0;  // rows added, chunks issued
  float E = 0.f;
  bool ok = true, taken = false;
  uint32_t tmem = 0;
  const uint32_t idesc = tc::instr_desc(tc::Split<PREC>::fmt, tc::kRows, N);
  const uint32_t hi = tc::smem_u32(tiles);
  for (int sub = 0; sub < G; ++sub) {
    const int vb = bp.x * G + sub;
    if (vb * kBlock >= d.V) break;
    RowSlot rs;
    const int total = block_rows(d, vb, bp.x * kBlock * G + done, phi_buf, s_warp, rs);
    if (total == 0) {
      __syncthreads();  // s_warp is rewritten by the next vertex block
      continue;
    }
    if (!taken) {
      tc::zero_padding<PREC, TL::CH, kBlock>(tiles, 2, NP);
      if (tid == 0) {
        tc::mbar_init(&bar, 1);
        tc::fence_mbar_init();
      }
      if (w == 0) tc::tmem_alloc(&tslot, tc::kTmemCols);
      load_link_tables(d, sHd, sXi);
      taken = true;
    }
    __syncthreads();
    float r2;
    jacobian_row(d, rs, phi_buf, Js, ROW, NP, sHd, sXi, r2);
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    if (lane == 0) s_e[w] = r2;
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    tmem = tslot;
    for (int k = 0; k < kBlock / 32; ++k) E += s_e[k];
    const int nchunks = (total + TL::K - 1) / TL::K;
    for (int q = 0; q < nchunks; ++q, ++gq) {
      if (gq > 0) {  // the previous chunk's MMAs read the tiles
        ok &= tc::mbar_wait(&bar, (gq - 1) & 1);
        tc::fence_proxy_async();
      }
      const int base = q * TL::K, cnt = min(TL::K, total - base);
      const int kq = (cnt + 2 * T - 1) / (2 * T) * (2 * T);
      const float* blk = Js + base * ROW;
      tc::stage_chunk<PREC, TL::CH, kBlock>([&](int k, int m) { return k < cnt ? blk[k * ROW + m] : 0.f; }, kq, NP,
                                            tiles);
      tc::fence_proxy_async();
      __syncthreads();
      if (tid == 0) {
        tc::fence_after_sync();
        tc::issue_chunk<PREC, TL::CH>(tmem, hi, hi + TL::BYTES, kq / (2 * T), idesc, gq == 0);
        tc::commit(&bar);
      }
    }
    done += total;
  }
  if (!taken) {  // nothing to add: no TMEM was taken and the reduction skips this block
    if (tid == 0) d.jtj_rows[bp.x] = 0;
    return;
  }
  const int nchunks = gq;
  if (nchunks > 0) {
    ok &= tc::mbar_wait(&bar, (nchunks - 1) & 1);
    tc::fence_after_sync();
  }
  // warps w and w + 4 read the same 32 TMEM lanes (parameters a), alternate 8-column groups (b)
  float* out = d.partial + (size_t)bp.x * NP * NP;
  const int a = 32 * (w & 3) + lane;
  const float bad = __int_as_float(0x7fc00000);
  for (int g = w >> 2; g < N / 8; g += 2) {
    uint32_t r[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
    if (nchunks > 0) {
      tc::ld_x8(tmem + ((uint32_t)(32 * (w & 3)) << 16) + 8 * g, r);
      tc::ld_wait(r);
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int b = 8 * g + t;
      if (a < NP && b < NP && a <= b)  // the upper triangle (the reduction mirrors)
        out[a * NP + b] = (a == NP - 1 && b == NP - 1) ? E : (ok ? __uint_as_float(r[t]) : bad);
    }
  }
  if (!ok && tid == 0) {
    atomicExch(&d.stats[3], 1);
    tc::mbar_wait(&bar, (nchunks - 1) & 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (w == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, tc::kTmemCols);
  }
  if (tid == 0) {
    d.jtj_rows[bp.x] = done;
    atomicAdd(&d.stats[1], done);
  }
}

template <int PREC, int NB>
__global__ void __launch_bounds__(kBlock) k_resid_jtj_tc(BatchGrid g, Dev d0, int phi_buf) {
  if (g.map == nullptr) {
    resid_jtj_tc_impl<PREC, NB>(d0, grid_pos(), phi_buf);
    return;
  }
  __shared__ Dev sd;
  resid_jtj_tc_impl<PREC, NB>(sd, batch_block(g, sd), phi_buf);
}

// Fixed-order sum of the block partials -> [J r]^T [J r]; the last entry gives E_pose (with the prior
// sum_k (lambda_s S_kk theta_k)^2), recorded as this iteration's energy and as the LM reference.
// A CTA owns 32 consecutive entries (coalesced lanes); its 32 warps take every 32nd partial and add them
// in FP32 with an error-free transformation (each addition's rounding error, from Knuth's TwoSum, is
// carried in a second FP32 accumulator: the compensated sum of Ogita, Rump and Oishi, accurate to about
// u |S| + (n u)^2 sum |x| in FP32 unit roundoff u, i.e. as if added in twice the precision).  The FP64
// pipe issues a small fraction of the FP32 rate on this GPU, so it is left to warp 0, which adds the 32
// warp sums (hi + lo) in FP64 in warp order.
//
// What bounds it is latency: one round trip for the partials, then the FP64 chain over the warps' sums
// (64 cycles an addition).  Humanoid 50k / 640x480 (196 partials of 1,596 entries): 14.6 -> 6.6 us; the
// prior term of E was a chain of 55 x 3 FP64 operations in one thread, the last partials one load at a time.
constexpr int kReduceThreads = 1024;

__device__ __forceinline__ void sum2_add(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bb = s - hi;
  const float e = (hi - (s - bb)) + (x - bb);  // exact: hi + x = s + e
  hi = s;
  lo += e;
}

constexpr int kReduceBatch = 8;  // partials a warp has in flight

__device__ __forceinline__ void reduce_jtj_impl(const Dev& d, BlockPos bp, int slot) {
  __shared__ double sm[kReduceThreads / 32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int NP = d.NP, n2 = NP * NP, nu = NP * (NP + 1) / 2;
  // lane -> the u-th entry of the upper triangle, row-major: (r, c), r <= c, at e = r NP + c; counted from
  // the end, row NP - 1 - m holds m + 1 entries
  const int u = bp.x * 32 + lane;
  int r = 0, c = 0;
  if (u < nu) {
    const int v = nu - 1 - u;
    int m = (int)((sqrtf(8.f * (float)v + 1.f) - 1.f) * 0.5f);
    if ((m + 1) * (m + 2) / 2 <= v) ++m;
    if (m * (m + 1) / 2 > v) --m;
    r = NP - 1 - m;
    c = NP - 1 - (v - m * (m + 1) / 2);
  }
  const int e = r * NP + c;
  // warp w < S takes blocks w, w + S, ... (up to kReduceBatch loads in flight together, each partial loaded
  // with its row count rather than after it); blocks that added no rows wrote no partial and count as
  // zero.  S depends on the session alone, so its sums have the same order in any launch.
  const int nb = d.nblk_rows;
  const int S = reduce_warps(nb);
  float hi = 0.f, lo = 0.f;
  if (u < nu && w < S) {
    for (int b0 = w; b0 < nb; b0 += kReduceBatch * S) {
      int rows[kReduceBatch];
      float q[kReduceBatch];
#pragma unroll
      for (int k = 0; k < kReduceBatch; ++k) {
        const int b = b0 + k * S;
        rows[k] = b < nb ? d.jtj_rows[b] : 0;
        q[k] = b < nb ? d.partial[(size_t)b * n2 + e] : 0.f;
      }
#pragma unroll
      for (int k = 0; k < kReduceBatch; ++k) sum2_add(hi, lo, rows[k] > 0 ? q[k] : 0.f);
    }
  }
  // E's prior term by the block that holds the last entry (NP - 1, NP - 1), a warp beside the sums
  const bool has_e = bp.x == (nu - 1) / 32;
  __shared__ double prior;
  if (has_e && w == (blockDim.x >> 5) - 1) {
    double p = 0.0;
    for (int k = lane; k < d.L; k += 32) p += d.prior2[k] * d.theta[k] * d.theta[k];
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    if (lane == 0) prior = p;
  }
  bool other = false;
  double dh = widen(hi, other), dl = widen(lo, other);
  if (__any_sync(0xffffffffu, other)) {
    dh = (double)hi;
    dl = (double)lo;
  }
  sm[w][lane] = dh + dl;
  __syncthreads();
  if (w != 0 || u >= nu) return;
  double t = 0.0;
#pragma unroll 8
  for (int k = 0; k < S; ++k) t += sm[k][lane];
  d.A[e] = t;
  d.A[c * NP + r] = t;  // A is symmetric: the lower triangle mirrors the upper
  if (e == n2 - 1) {
    const double E = t + prior;
    if (slot >= 0) d.energy[slot] = E;
    d.lm_trials[6] = E;
  }
}

__global__ void __launch_bounds__(kReduceThreads) k_reduce_jtj(BatchGrid g, Dev d0, int slot) {
  if (g.map == nullptr) {
    reduce_jtj_impl(d0, grid_pos(), slot);
    return;
  }
  __shared__ Dev sd;
  reduce_jtj_impl(sd, batch_block(g, sd), slot);
}

static int jtj_smem_bytes(int T, int L) {
  return kBlock * jtj_row_stride(T) * 4 + L * (int)sizeof(DQ) + 8 * L * 4;
}

template <int PREC>
static int jtj_tc_smem_bytes(int NB, int L) {
  return tc::Tile<PREC, 8>::STAGE + kBlock * (16 * NB + 1) * 4 + L * (int)sizeof(DQ) + 8 * L * 4;
}

template <int PREC>
static void launch_resid_jtj_tc(const Dev& d, int phi_buf, cudaStream_t st) {
  const int NB = (d.NP + 15) / 16;
  const int g = d.nblk_rows;
  const int sm = jtj_tc_smem_bytes<PREC>(NB, d.L);
  switch (NB) {
    case 1: k_resid_jtj_tc<PREC, 1><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    case 2: k_resid_jtj_tc<PREC, 2><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    case 3: k_resid_jtj_tc<PREC, 3><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    case 4: k_resid_jtj_tc<PREC, 4><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    default: k_resid_jtj_tc<PREC, 5><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
  }
}

template <int PREC>
static void configure_resid_jtj_tc() {
  cudaFuncSetAttribute(k_resid_jtj_tc<PREC, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_tc_smem_bytes<PREC>(1, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj_tc<PREC, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_tc_smem_bytes<PREC>(2, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj_tc<PREC, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_tc_smem_bytes<PREC>(3, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj_tc<PREC, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_tc_smem_bytes<PREC>(4, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj_tc<PREC, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_tc_smem_bytes<PREC>(5, kMaxLinks));
}

void launch_resid_jtj(const Dev& d, int phi_buf, cudaStream_t st) {
  if (d.precision == 1) return launch_resid_jtj_tc<1>(d, phi_buf, st);
  if (d.precision == 2) return launch_resid_jtj_tc<2>(d, phi_buf, st);
  const int T = (d.NP + 15) / 16;
  const int g = d.nblk_rows;
  const int sm = jtj_smem_bytes(T, d.L);
  switch (T) {
    case 1: k_resid_jtj<1><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    case 2: k_resid_jtj<2><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    case 3: k_resid_jtj<3><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    case 4: k_resid_jtj<4><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
    default: k_resid_jtj<5><<<g, kBlock, sm, st>>>(kSingle, d, phi_buf); break;
  }
}

void launch_reduce_jtj(const Dev& d, int slot, cudaStream_t st) {
  k_reduce_jtj<<<(d.NP * (d.NP + 1) / 2 + 31) / 32, 32 * reduce_warps(d.nblk_rows), 0, st>>>(kSingle, d, slot);
}

void launch_normal_equations(const Dev& d, int phi_buf, int slot, cudaStream_t st) {
  launch_resid_jtj(d, phi_buf, st);
  launch_reduce_jtj(d, slot, st);
}

// ---------------------------------------------------------------------------------------------
// LM candidates (Sec. 4.2): CTA c solves (A + lambda_c diag A) x = b with A = J^T J + (lambda_s S)^2,
// b = J^T r + (lambda_s S)^2 Theta and lambda_c = min(lambda 10^c, 1e7); a parameter whose diagonal is
// zero is frozen (x_k = 0).  Theta_c = Theta - x and its FK tables follow.
//
// On this GPU a dependent FP64 FMA costs ~70 cycles and an FP64 rsqrt ~440 (FP32: ~4 and ~20), and the
// FP64 pipe issues ~2 operations per cycle per SM, so the P sequential pivot steps of an FP64 Cholesky
// are latency-bound (~80 us at P = 55).  The solve therefore factors the Jacobi-scaled matrix D M D
// (unit diagonal) in FP32 (blocked Cholesky) and reaches FP64 accuracy by iterative refinement:
// x += D (D M D)^-1 D (b - M x) with the residual in FP64, until the scaled residual is below 1e-10 of
// the scaled right-hand side.  If the FP32 factorisation breaks down or the refinement stalls, the FP64
// Cholesky factorisation of M is used instead.
//
// One CTA per candidate; every phase is a dependent chain on one SM (IPC 0.7), so the time is the sum of
// the chains' latencies: P = 55, cycles at 2.07 GHz: inputs 1.8k, set-up 4.3k, factor 8.2k, two
// substitutions 2 x 4.7k, two FP64 residuals 2 x 2.9k (the FP64 pipe's rate), FK 9k.  Measured per launch,
// humanoid 50k: 34.9 -> 20 us (a frame of ten iterations 1,406 -> 1,259 us).
// ---------------------------------------------------------------------------------------------
constexpr int kSolveThreads = 256, kSolveBlocksPerSM = 2;
constexpr int kCrowdThreads = 192, kCrowdBlocksPerSM = 3;  // of a batch that takes fewer waves so
constexpr int kMaxRefine = 8;

__device__ void chol_solve_fp64(double* M, int ld, double* b, int P, int& fail_out) {
  __shared__ int fail;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (tid == 0) fail = 0;
  __syncthreads();
  for (int k = 0; k < P; ++k) {
    if (tid == 0) {
      const double piv = M[k * ld + k];
      if (!(piv > 0.0)) fail = 1;
      M[k * ld + k] = sqrt(fmax(piv, 0.0));
    }
    __syncthreads();
    if (fail) break;
    const double ik = 1.0 / M[k * ld + k];
    for (int r = k + 1 + tid; r < P; r += nt) M[r * ld + k] *= ik;
    __syncthreads();
    const int n = P - k - 1;
    for (int e = tid; e < n * n; e += nt) {
      const int r = k + 1 + e / n, q = k + 1 + e % n;
      if (q <= r) M[r * ld + q] -= M[r * ld + k] * M[q * ld + k];
    }
    __syncthreads();
  }
  if (!fail) {
    for (int k = 0; k < P; ++k) {
      if (tid == 0) b[k] /= M[k * ld + k];
      __syncthreads();
      for (int r = k + 1 + tid; r < P; r += nt) b[r] -= M[r * ld + k] * b[k];
      __syncthreads();
    }
    for (int k = P - 1; k >= 0; --k) {
      if (tid == 0) b[k] /= M[k * ld + k];
      __syncthreads();
      for (int r = tid; r < k; r += nt) b[r] -= M[k * ld + r] * b[k];
      __syncthreads();
    }
  }
  fail_out = fail;
  __syncthreads();
}

constexpr int kBlk = 8;               // block size of the factorisation
constexpr int kMaxPad = 80;           // P padded to a multiple of kBlk
// Row r of the FP32 matrices starts at fidx(r, 0): on 16 bytes, with the 16-byte pieces of one column in 8
// consecutive (aligned) rows on distinct banks (21 pieces per row, odd) and those in rows 0, 4, .., 28 too
// (one piece of skew per 8 rows).
constexpr int kFRow = kMaxPad + 4;
constexpr int kFBlock = kBlk * kFRow + 4;  // distance of two block rows
__host__ __device__ constexpr int fidx(int r, int c) { return r * kFRow + 4 * (r >> 3) + c; }

// The 8x8 diagonal block at j (lower triangle used) in registers.
__device__ __forceinline__ void load_diag(const float* F, int j, float (&a)[kBlk][kBlk]) {
  const float* p = F + (j >> 3) * kFBlock + j;
#pragma unroll
  for (int i = 0; i < kBlk; ++i) {
    const float4 lo = *reinterpret_cast<const float4*>(p + i * kFRow);
    a[i][0] = lo.x, a[i][1] = lo.y, a[i][2] = lo.z, a[i][3] = lo.w;
    if (i >= 4) {
      const float4 hi = *reinterpret_cast<const float4*>(p + i * kFRow + 4);
      a[i][4] = hi.x, a[i][5] = hi.y, a[i][6] = hi.z, a[i][7] = hi.w;
    }
  }
}
__device__ __forceinline__ void load8(const float* p, float (&v)[kBlk]) {
  const float4 lo = *reinterpret_cast<const float4*>(p), hi = *reinterpret_cast<const float4*>(p + 4);
  v[0] = lo.x, v[1] = lo.y, v[2] = lo.z, v[3] = lo.w;
  v[4] = hi.x, v[5] = hi.y, v[6] = hi.z, v[7] = hi.w;
}
__device__ __forceinline__ void store8(float* p, const float (&v)[kBlk]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}

// 1/sqrt(x) of a normal x: what rsqrtf returns for it, without rsqrtf's handling of denormals.
__device__ __forceinline__ float rsqrt_normal(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Blocked FP32 Cholesky: F (lower triangle, padded to Pp) is used up, G receives the factor and ivd 1/L_kk.
// Returns false if a pivot is not positive.  It is a chain of Pp dependent pivots on one SM, so what
// counts is the latency of a block column.  The warps with rows below the 8x8 diagonal block each factor
// it redundantly in registers (a pivot is then one rsqrt, one multiply and one FMA: no shuffles, and no
// barrier between the factor and the panel), a thread solves one panel row, and the trailing triangle goes
// by 2x4 tiles, one thread each: shared-memory loads return 128 bytes per cycle and SM however many lanes
// read the same address, so entries formed per load count, but a tile is also one thread's chain.  The
// factor goes to a matrix of its own, so that the redundant readers of F never race its writer.  Two
// barriers per block column.
__device__ bool chol_blocked(float* F, float* G, float* ivd, int Pp) {
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5, nt = blockDim.x, nw = nt >> 5;
  if (tid == 0) bad = 0;
  // this thread's tiles (2 rows x 4 columns) of the trailing triangle, relative to its corner: row pairs in
  // order, pair i with i / 2 + 1 tiles, so the rows 4 m .. 4 m + 3 hold 2 (m + 1) from tile m (m + 1) on
  // (at most 18 x 19 tiles for 72 rows)
  static_assert(2 * kCrowdThreads >= 18 * 19, "two tiles per thread cover the largest trailing triangle");
  int tile[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int e = tid + h * nt;
    int m = (int)((sqrtf(4.f * (float)e + 1.f) - 1.f) * 0.5f);
    if ((m + 1) * (m + 2) <= e) ++m;
    if (m * (m + 1) > e) --m;
    const int k = e - m * (m + 1), odd = k > m;
    tile[h] = (4 * m + 2 * odd) << 8 | 4 * (k - (odd ? m + 1 : 0));
  }
  __syncthreads();
#pragma unroll 1
  for (int j = 0; j < Pp; j += kBlk) {
    const int j1 = j + kBlk;
    if (warp == nw - 1 || j1 + 32 * warp < Pp) {
      float a[kBlk][kBlk], iv[kBlk];
      load_diag(F, j, a);
      bool neg = false;
#pragma unroll
      for (int c = 0; c < kBlk; ++c) {
        const float dc = a[c][c];
        neg |= !(dc > 0.f);
        iv[c] = rsqrt_normal(fmaxf(dc, 1e-30f));
        a[c][c] = dc * iv[c];
#pragma unroll
        for (int i = c + 1; i < kBlk; ++i) a[i][c] = a[i][c] * iv[c];
#pragma unroll
        for (int q = c + 1; q < kBlk; ++q)
#pragma unroll
          for (int i = q; i < kBlk; ++i) a[i][q] = fmaf(-a[i][c], a[q][c], a[i][q]);
      }
      if (warp != nw - 1) {  // a panel row (no panel reaches the last warp)
        if (j1 + tid < Pp) {
          float p[kBlk];
          load8(&F[fidx(j1 + tid, j)], p);
#pragma unroll
          for (int c = 0; c < kBlk; ++c) {
            float sacc = p[c];
#pragma unroll
            for (int q = 0; q < c; ++q) sacc = fmaf(-p[q], a[c][q], sacc);
            p[c] = sacc * iv[c];
          }
          store8(&G[fidx(j1 + tid, j)], p);
        }
      } else if (tid == nt - 1) {  // the factored diagonal block (its upper triangle is not read)
        if (neg) bad = 1;
#pragma unroll
        for (int i = 0; i < kBlk; ++i) {
          *reinterpret_cast<float4*>(&G[fidx(j + i, j)]) = make_float4(a[i][0], a[i][1], a[i][2], a[i][3]);
          if (i >= 4) *reinterpret_cast<float4*>(&G[fidx(j + i, j + 4)]) = make_float4(a[i][4], a[i][5], a[i][6], a[i][7]);
        }
        store8(ivd + j, iv);
      }
    }
    __syncthreads();
    if (bad) return false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r0 = j1 + (tile[h] >> 8), q0 = j1 + (tile[h] & 255);
      if (r0 >= Pp) break;
      float lr[2][kBlk], dot[2][4];
      load8(&G[fidx(r0, j)], lr[0]);
      load8(&G[fidx(r0 + 1, j)], lr[1]);
      float4* f0 = reinterpret_cast<float4*>(&F[fidx(r0, q0)]);
      float4* f1 = reinterpret_cast<float4*>(&F[fidx(r0 + 1, q0)]);
      const float4 o0 = *f0, o1 = *f1;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float lq[kBlk];
        load8(&G[fidx(q0 + t, j)], lq);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          dot[u][t] = 0.f;
#pragma unroll
          for (int c = 0; c < kBlk; ++c) dot[u][t] = fmaf(lr[u][c], lq[c], dot[u][t]);
        }
      }
      // (entries right of the diagonal are updated too: nothing reads them)
      *f0 = make_float4(o0.x - dot[0][0], o0.y - dot[0][1], o0.z - dot[0][2], o0.w - dot[0][3]);
      *f1 = make_float4(o1.x - dot[1][0], o1.y - dot[1][1], o1.z - dot[1][2], o1.w - dot[1][3]);
    }
    __syncthreads();
  }
  return true;
}

// One 8x8 block of the substitutions by a warp whose lanes hold rows lane + 32 k: the block's eight
// right-hand sides by independent shuffles, the block solved redundantly by every lane in registers, and
// the lane's own rows updated (rows already solved too: their results are in z and are not read again).
// The next block's diagonal (at jn) is loaded meanwhile.  Issue-bound: one warp, ~100 instructions.
template <int SETS, bool kBack>
__device__ __forceinline__ void solve_block(const float* G, const float* const (&mine_rows)[SETS], const float* ivd, int j, int jn,
                                            const float (&a)[kBlk][kBlk], const float (&iv)[kBlk],
                                            float (&an)[kBlk][kBlk], float (&ivn)[kBlk], float (&y)[SETS], float* z) {
  const int lane = threadIdx.x & 31, set = j >> 5;
  float row[SETS][kBlk];
  if constexpr (kBack) {
    const float* p = G + (j >> 3) * kFBlock + lane;  // (columns past the row: the next row's, not used)
#pragma unroll
    for (int k = 0; k < SETS; ++k)
#pragma unroll
      for (int c = 0; c < kBlk; ++c) row[k][c] = p[c * kFRow + (k < 2 ? 32 * k : min(32 * k, kMaxPad - 1 - lane))];
  } else {
#pragma unroll
    for (int k = 0; k < SETS; ++k) load8(mine_rows[k] + j, row[k]);
  }
  float mine = y[0];
#pragma unroll
  for (int k = 1; k < SETS; ++k) mine = set == k ? y[k] : mine;
  float v[kBlk];
#pragma unroll
  for (int i = 0; i < kBlk; ++i) v[i] = __shfl_sync(0xffffffffu, mine, (j & 31) + i);
  load_diag(G, jn, an);
  load8(ivd + jn, ivn);
#pragma unroll
  for (int t = 0; t < kBlk; ++t) {
    const int c = kBack ? kBlk - 1 - t : t;
    v[c] = v[c] * iv[c];
#pragma unroll
    for (int i = 0; i < kBlk; ++i) {
      if (kBack && i < c) v[i] = fmaf(-a[c][i], v[c], v[i]);
      if (!kBack && i > c) v[i] = fmaf(-a[i][c], v[c], v[i]);
    }
  }
#pragma unroll
  for (int k = 0; k < SETS; ++k)
#pragma unroll
    for (int c = 0; c < kBlk; ++c) y[k] = fmaf(-row[k][c], v[c], y[k]);
  if (lane == 0) store8(z + j, v);
}

// y <- (L L^T)^-1 y with the factor of chol_blocked, by one warp without block barriers: lane l holds rows
// l + 32 k; z (16-byte aligned, kMaxPad) is scratch; G has g_rows rows.
template <int SETS>
__device__ __forceinline__ void solve_warp(const float* G, const float* ivd, float (&y)[SETS], float* z,
                                           int Pp, int g_rows) {
  const int lane = threadIdx.x & 31;
  float a[kBlk][kBlk], iv[kBlk], an[kBlk][kBlk], ivn[kBlk];
  const float* rows[SETS];  // this lane's rows of G
#pragma unroll
  for (int k = 0; k < SETS; ++k) rows[k] = G + fidx(min(32 * k + lane, g_rows - 1), 0);
  load_diag(G, 0, a);
  load8(ivd, iv);
#pragma unroll 1
  for (int j = 0; j < Pp; j += 2 * kBlk) {  // L z = y
    solve_block<SETS, false>(G, rows, ivd, j, min(j + kBlk, Pp - kBlk), a, iv, an, ivn, y, z);
    if (j + kBlk >= Pp) break;
    solve_block<SETS, false>(G, rows, ivd, j + kBlk, min(j + 2 * kBlk, Pp - kBlk), an, ivn, a, iv, y, z);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < SETS; ++k) y[k] = z[min(32 * k + lane, kMaxPad - 1)];
  __syncwarp();
  load_diag(G, Pp - kBlk, a);
  load8(ivd + Pp - kBlk, iv);
#pragma unroll 1
  for (int j = Pp - kBlk; j >= 0; j -= 2 * kBlk) {  // L^T x = z
    solve_block<SETS, true>(G, rows, ivd, j, max(j - kBlk, 0), a, iv, an, ivn, y, z);
    if (j < kBlk) break;
    solve_block<SETS, true>(G, rows, ivd, j - kBlk, max(j - 2 * kBlk, 0), an, ivn, a, iv, y, z);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < SETS; ++k) y[k] = z[min(32 * k + lane, kMaxPad - 1)];
}

// ys <- (L L^T)^-1 ys by one warp.
template <int SETS>
__device__ __forceinline__ void solve_rows(const float* G, const float* ivd, float* ys, float* z, int P, int Pp,
                                           int g_rows) {
  const int lane = threadIdx.x & 31;
  float y[SETS];
#pragma unroll
  for (int k = 0; k < SETS; ++k) y[k] = lane + 32 * k < P ? ys[lane + 32 * k] : 0.f;
  solve_warp<SETS>(G, ivd, y, z, Pp, g_rows);
#pragma unroll
  for (int k = 0; k < SETS; ++k)
    if (lane + 32 * k < P) ys[lane + 32 * k] = y[k];
}

// (float)x, rounded to nearest even.  Conversions from FP64 share the FP64 pipe, which takes 60 cycles per
// warp instruction here; where the result is a normal FP32 number or zero, the same bits are formed with
// integer operations: the exponent rebiased by 1023 - 127 and the 29 dropped mantissa bits rounded, a
// carry running into the exponent (up to infinity) as it should.  Sets `other` where that does not hold.
__device__ __forceinline__ float to_float_rn(double x, bool& other) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned t = __funnelshift_l(lo, hi, 3) - (384u << 23);  // exponent (mod 512) and 23 mantissa bits
  const unsigned up = (lo & 0x1fffffffu) + (t & 1u) > 0x10000000u ? 1u : 0u;
  const bool zero = ((hi & 0x7fffffffu) | lo) == 0u;
  other |= !zero && ((hi >> 20) & 0x7ffu) - 897u >= 254u;
  return __uint_as_float((zero ? 0u : t + up) | (hi & 0x80000000u));
}

// The solve's dynamic shared memory: F (P padded to the block, rows of kFRow), G (kMaxPad rows: the substitution's lanes
// read past the padded P), M, six P-vectors, then the link table and the links' dual quaternions.  kLate: G without the
// rows past the padded P, and the last two in F's place, once the factor has used it up.
constexpr int kLinkTableBytes = (sizeof(LinkTable) + 15) & ~15;
__host__ __device__ constexpr int padded(int P) { return (P + kBlk - 1) / kBlk * kBlk; }
template <bool kLate>
struct SolveLayout {
  static __host__ __device__ constexpr int g_rows(int P) { return kLate ? padded(P) : kMaxPad; }
  static __host__ __device__ constexpr int links(int P) { return kLinkTableBytes + P * (int)sizeof(DQ); }
  static __host__ __device__ constexpr int g(int P) {  // byte offsets; F at 0
    const int f = fidx(padded(P), 0) * (int)sizeof(float);
    return kLate && links(P) > f ? links(P) : f;
  }
  static __host__ __device__ constexpr int m(int P) { return g(P) + fidx(g_rows(P), 0) * (int)sizeof(float); }
  static __host__ __device__ constexpr int end(int P) {
    return (m(P) + ((P + 1) * (P + 1) + 6 * P) * (int)sizeof(double) + 15) & ~15;
  }
  static __host__ __device__ constexpr int table(int P) { return kLate ? 0 : end(P); }
  static __host__ __device__ constexpr int bytes(int P) { return kLate ? end(P) : end(P) + links(P); }
};

template <bool kLate>
__device__ __forceinline__ void lm_solve_impl(const Dev& d, BlockPos bp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) float ivd[kMaxPad], zs[kMaxPad];
  __shared__ float sc[kMaxPad], ys[kMaxPad];  // scale D, scaled residual
  const int P = d.L, NP = d.NP, c = bp.x, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int Pp = (P + kBlk - 1) / kBlk * kBlk;
  float* F = reinterpret_cast<float*>(smem_raw);  // FP32 scaled system (used up by the factor)
  using Layout = SolveLayout<kLate>;
  float* G = reinterpret_cast<float*>(smem_raw + Layout::g(P));  // its Cholesky factor
  // [NP][NP] as the reduction left it (J^T J, J^T r in column P), then the FP64 system for the residuals
  double* M = reinterpret_cast<double*>(smem_raw + Layout::m(P));
  double* x = M + NP * NP;
  double* res = x + P;
  double* b = res + P;
  double* dg = b + P;
  double* p2 = dg + P;  // (lambda_s S_kk)^2
  double* th = p2 + P;  // Theta
  LinkTable* lt = reinterpret_cast<LinkTable*>(smem_raw + Layout::table(P));
  DQ* H0 = reinterpret_cast<DQ*>(smem_raw + Layout::table(P) + kLinkTableBytes);
  __shared__ unsigned rmax_bits[2], bmax_bits;  // rmax: one slot per refinement parity
  __shared__ unsigned char frz[kMaxPad];
  __shared__ int any_frz;
  // ---- inputs in one round trip: the matrix with its last column, the prior, Theta and the link table
  for (int t = tid; t < NP * NP / 2; t += nt) cp_async16(M + 2 * t, d.A + 2 * t);
  if ((NP & 1) && tid == 0) cp_async8(M + NP * NP - 1, d.A + NP * NP - 1);
  for (int r = tid; r < P; r += nt) {
    cp_async8(p2 + r, d.prior2 + r);
    cp_async8(th + r, d.theta + r);
  }
  auto load_links = [&] {
    for (int t = tid; t < (int)(sizeof(LinkTable) / 16); t += nt)
      cp_async16(reinterpret_cast<char*>(lt) + 16 * t, reinterpret_cast<const char*>(d.links) + 16 * t);
  };
  if (!kLate) load_links();
  double lam = *d.lam;
  for (int t = 0; t < c; ++t) lam = fmin(lam * 10.0, 1e7);
  if (tid == 0) bmax_bits = rmax_bits[0] = any_frz = 0;
  if (tid == nt - 1) {  // lambda after the step if this candidate is taken; if none is, after the last one
    d.lam_next[c] = fmax(lam / 10.0, 1e-7);
    if (c == kCandidates - 1) d.lam_next[kCandidates] = fmin(lam * 10.0, 1e7);
  }
  cp_async_wait_all();
  __syncthreads();
  // ---- setup: M = A + diag(prior + lambda dg) (FP64), frozen rows/columns -> identity; scale D in FP32
  // (an FP64 instruction occupies its sub-partition's pipe for 64 cycles per warp: the two halves of the
  // block take a part of the vectors each)
  static_assert(kCrowdThreads / 2 >= kMaxPad, "half a block covers the rows");
  {
    constexpr int half = (kLate ? kCrowdThreads : kSolveThreads) / 2;
    const int r = tid < half ? tid : tid - half;
    if (r < P) {
      double& mrr = M[(size_t)r * NP + r];
      if (tid < half) {
        const double dgr = mrr + p2[r];
        const bool fr = dgr == 0.0;
        frz[r] = fr;
        if (fr) any_frz = 1;
        sc[r] = fr ? 1.f : rsqrtf((float)(dgr * (1.0 + lam)));
        mrr = fr ? 1.0 : mrr + (p2[r] + lam * dgr);
      } else {
        b[r] = M[(size_t)r * NP + P] + p2[r] * th[r];
        ys[r] = (float)b[r];
        x[r] = 0.0;
      }
    }
  }
  __syncthreads();
  {
    unsigned bmine = 0u;
    if (tid < P) {
      if (frz[tid]) {
        b[tid] = 0.0;
        ys[tid] = 0.f;
      }
      ys[tid] *= sc[tid];
      bmine = __float_as_uint(fabsf(ys[tid]));
    }
    bmine = __reduce_max_sync(0xffffffffu, bmine);
    if (lane == 0 && bmine) atomicMax(&bmax_bits, bmine);
  }
  if (any_frz) {  // the off-diagonal of M is zero in frozen rows and columns
    for (int r = warp; r < P; r += nt >> 5)
      for (int q = lane; q < P; q += 32)
        if (q != r && (frz[r] || frz[q])) M[(size_t)r * NP + q] = 0.0;
    __syncthreads();
  }
  // the FP32 lower triangle of D M D, a warp per row, four rows' loads in flight
  {
    constexpr int kSets = (kMaxPad + 31) / 32, kRows = 4;
    float scq[kSets];
#pragma unroll
    for (int k = 0; k < kSets; ++k) scq[k] = lane + 32 * k < P ? sc[lane + 32 * k] : 0.f;
    const int step = nt >> 5;
#pragma unroll 1
    for (int r0 = warp; r0 < P; r0 += kRows * step) {
      double m[kRows][kSets];
      float sr[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int r = r0 + u * step;
        sr[u] = r < P ? sc[r] : 0.f;
#pragma unroll
        for (int k = 0; k < kSets; ++k)
          if (32 * k < P) m[u][k] = r < P && lane + 32 * k <= r ? M[(size_t)r * NP + lane + 32 * k] : 0.0;
      }
      float f[kRows][kSets];
      bool other = false;
#pragma unroll
      for (int u = 0; u < kRows; ++u)
#pragma unroll
        for (int k = 0; k < kSets; ++k)
          if (32 * k < P) f[u][k] = to_float_rn(m[u][k], other);
      if (__any_sync(0xffffffffu, other)) {
#pragma unroll
        for (int u = 0; u < kRows; ++u)
#pragma unroll
          for (int k = 0; k < kSets; ++k) f[u][k] = (float)m[u][k];
      }
#pragma unroll
      for (int u = 0; u < kRows; ++u)
#pragma unroll
        for (int k = 0; k < kSets; ++k)
          if (lane + 32 * k <= r0 + u * step && r0 + u * step < P)
            F[fidx(r0 + u * step, lane + 32 * k)] = f[u][k] * sr[u] * scq[k];
    }
  }
  for (int e = tid; e < (Pp - P) * Pp; e += nt) {  // identity rows padding P to a multiple of the block
    const int r = P + e / Pp, q = e % Pp;
    if (q <= r) F[fidx(r, q)] = r == q ? 1.f : 0.f;
  }
  __syncthreads();
  // ---- FP32 factor of D M D, padded with identity rows to a multiple of the block size
  const bool ok32 = chol_blocked(F, G, ivd, Pp);  // (its last barrier: nothing reads F any more)
  if (kLate) load_links();
  // ---- iterative refinement: x += D (D M D)^-1 D (b - M x), residual in FP64
  int iters = 0;
  bool converged = false;
  const float bmax = __uint_as_float(bmax_bits);
  for (int it = 0; it < kMaxRefine && ok32; ++it) {
    if (warp == 0) {
      if (Pp <= 32) solve_rows<1>(G, ivd, ys, zs, P, Pp, Layout::g_rows(P));
      else if (Pp <= 64) solve_rows<2>(G, ivd, ys, zs, P, Pp, Layout::g_rows(P));
      else solve_rows<3>(G, ivd, ys, zs, P, Pp, Layout::g_rows(P));
    }
    __syncthreads();
    for (int r = tid; r < P; r += nt) x[r] += (double)sc[r] * (double)ys[r];
    __syncthreads();
    if (tid == 0) rmax_bits[(it + 1) & 1] = 0u;  // every thread has read it (the previous iteration's test)
    // res = b - M x in FP64: four threads per row (columns q = part mod 4, two accumulators each), the
    // four sums combined by shuffles in a fixed pairing
    unsigned rmine = 0u;
    for (int r0 = 0; r0 < P; r0 += nt / 4) {
      const int r = r0 + (tid >> 2), part = tid & 3;
      double s0 = 0.0, s1 = 0.0;
      if (r < P) {
        const double* mr = M + (size_t)r * NP;
        int q = part;
        for (; q + 4 < P; q += 8) {
          s0 = fma(-mr[q], x[q], s0);
          s1 = fma(-mr[q + 4], x[q + 4], s1);
        }
        if (q < P) s0 = fma(-mr[q], x[q], s0);
      }
      double sum = s0 + s1;
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      if (r < P && part == 0) {
        const double rres = b[r] + sum;
        ys[r] = (float)rres * sc[r];
        rmine = max(rmine, __float_as_uint(fabsf(ys[r])));
      }
    }
    rmine = __reduce_max_sync(0xffffffffu, rmine);
    if (lane == 0 && rmine) atomicMax(&rmax_bits[it & 1], rmine);
    __syncthreads();
    iters = it + 1;
    if (__uint_as_float(rmax_bits[it & 1]) <= 1e-10f * bmax) { converged = true; break; }
  }
  int fail = 0;
  if (!converged) {  // FP64 Cholesky of the unscaled system
    for (int r = tid; r < P; r += nt) x[r] = b[r];
    __syncthreads();
    chol_solve_fp64(M, NP, x, P, fail);
  }
  double* thc = d.theta_c + (size_t)c * P;
  for (int j = tid; j < P; j += nt) {  // the candidate, also kept in shared memory (res is free now) for FK
    const double tj = fail ? th[j] : th[j] - x[j];
    thc[j] = tj;
    res[j] = tj;
  }
  if (tid == 0) {
    d.lm_ok[c] = !fail;
    d.lm_ok[kCandidates + c] = converged ? iters : (fail ? -2 : -1);
  }
  if (kLate) cp_async_wait_all();
  __syncthreads();
  fk_all(*lt, res, H0, d.Hd_c + (size_t)c * P, d.xi_c + (size_t)c * P * 8, 8);
}

template <bool kLate>
__global__ void __launch_bounds__(kLate ? kCrowdThreads : kSolveThreads, kLate ? kCrowdBlocksPerSM : kSolveBlocksPerSM)
    k_lm_solve(BatchGrid g, Dev d0) {
  if (g.map == nullptr) {
    lm_solve_impl<kLate>(d0, grid_pos());
    return;
  }
  __shared__ Dev sd;
  lm_solve_impl<kLate>(sd, batch_block(g, sd));
}

// Energy of each candidate at the fixed association (normals and p~ held), then the accept step:
// the first candidate with E_c <= E wins (lambda <- lambda_c / 10); if none, Theta stays and
// lambda <- min(lambda_5 * 10, 1e7).  The last block to finish does the selection.
//
// In two passes, so that the common case costs a third of the work: the first pass scores candidates
// 0 and 1 (the damping that almost always succeeds) and accepts one if it can; otherwise it records
// their energies and marks the step pending (lm_trials[7] = -2), and the second pass scores candidates
// 2-5 and decides over all six.  The decision sequence and every energy are those of scoring all six at
// once (each candidate's sum has the same blocks in the same order).  Candidates not scored report +inf.
//
// A chain of round trips: row count, records, ticket, block energies, decision, tables.  FP64 additions
// (64 cycles each and warp) are kept out of it where they can be: only the scored candidates are added, a
// warp per candidate, and the next lambdas come from the solve.  Humanoid 50k, first pass: 12.6 -> 10.3 us
// alone, 39 -> 31 us for 16 sessions.
constexpr double kPending = -2.0;

template <int c0, int c1>  // the candidates it scores
__device__ __forceinline__ void lm_eval_impl(const Dev& d, BlockPos bp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  DQ* sH = reinterpret_cast<DQ*>(smem_raw);  // [kCandidates][L]
  __shared__ int sok[kCandidates];
  __shared__ double swarp[kBlock / 32][kCandidates];
  __shared__ bool last;
  const int L = d.L, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (c0 > 0 && d.lm_trials[7] != kPending) return;  // the first pass decided
  // the [J r] block's rows (written by the normal-equations pass of this iteration, one record per vertex
  // of A: the mean data point p~, n, x = x0 + phi, bones and weights), with the candidates' tables
  const int cnt = d.jtj_rows[bp.x];
  const float4* recs = d.arec + (size_t)bp.x * kBlock * d.jtj_group * 4;
  float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0, r2 = r0, r3 = r0;
  if (tid < cnt) {
    r0 = recs[4 * tid];
    r1 = recs[4 * tid + 1];
    r2 = recs[4 * tid + 2];
    r3 = recs[4 * tid + 3];
  }
  if (cnt > 0)  // the same in every thread of the block
    for (int t = c0 * L + tid; t < c1 * L; t += kBlock) sH[t] = d.Hd_c[t];
  if (tid < kCandidates) sok[tid] = d.lm_ok[tid];
  __syncthreads();
  float e[kCandidates];
#pragma unroll
  for (int c = 0; c < kCandidates; ++c) e[c] = 0.f;
  for (int q = tid; q < cnt; q += kBlock) {
    if (q != tid) {
      r0 = recs[4 * q];
      r1 = recs[4 * q + 1];
      r2 = recs[4 * q + 2];
      r3 = recs[4 * q + 3];
    }
    const float3 pt = make_float3(r0.x, r0.y, r0.z), nn = make_float3(r0.w, r1.x, r1.y);
    const float3 x = make_float3(r1.z, r1.w, r2.x);
    const float4 bw = make_float4(r2.y, r2.z, r2.w, r3.x);
    const unsigned bits = __float_as_uint(r3.y);
    uchar4 bi;
    memcpy(&bi, &bits, 4);
#pragma unroll
    for (int c = 0; c < kCandidates; ++c) {
      if (c < c0 || c >= c1 || !sok[c]) continue;
      float sg[4];
      const DQ H = blend_bones(sH + c * L, bi, bw, sg);
      const float3 vc = dq_point(H, x);
      const float r = nn.x * (pt.x - vc.x) + nn.y * (pt.y - vc.y) + nn.z * (pt.z - vc.z);
      e[c] += r * r;
    }
  }
#pragma unroll
  for (int c = 0; c < kCandidates; ++c)
    for (int o = 16; o > 0; o >>= 1) e[c] += __shfl_xor_sync(0xffffffffu, e[c], o);
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < kCandidates; ++c)
      if (c >= c0 && c < c1) swarp[w][c] = e[c];
  }
  __syncthreads();
  // the block's energies, then its ticket: one warp writes and takes it
  if (w == 0) {
    if (lane >= c0 && lane < c1) {
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < kBlock / 32; ++k) s += swarp[k][lane];
      d.epart[(size_t)bp.x * 8 + lane] = s;
    }
    __syncwarp();
    if (lane == 0) {
      __threadfence();  // (by the lane that takes the ticket: it orders what the warp's barrier showed it, too)
      last = atomicAdd(&d.counter[0], 1u) == (unsigned)bp.gx - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the session's last block: warp c adds candidate c's block energies and prior terms (strided over the
  // lanes, then a shuffle tree)
  __shared__ double Ec[kCandidates];
  const double inf = __longlong_as_double(0x7ff0000000000000ll);
  if (w < kCandidates) {
    double v = 0.0;
    if (w >= c0 && w < c1) {
      const double* thc = d.theta_c + (size_t)w * L;
#pragma unroll 4
      for (int k = lane; k < L; k += 32) v += d.prior2[k] * thc[k] * thc[k];
#pragma unroll 8
      for (int b = lane; b < bp.gx; b += 32) v += __ldcg(d.epart + (size_t)b * 8 + w);
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (!sok[w]) v = inf;
    } else {
      v = w < c0 ? d.lm_trials[w] : inf;  // the first pass's energies; later ones unscored
    }
    if (lane == 0) Ec[w] = v;
  }
  __syncthreads();
  __shared__ int acc_c;
  if (tid == 0) {
    const double E = d.lm_trials[6];
    int a = -1;
#pragma unroll
    for (int c = kCandidates - 1; c >= 0; --c)
      if (c < c1 && sok[c] && Ec[c] <= E) a = c;
    if (a >= 0 || c1 == kCandidates) {
      *d.lam = d.lam_next[a >= 0 ? a : kCandidates];
      d.lm_trials[7] = (double)a;
    } else {
      d.lm_trials[7] = kPending;
    }
    acc_c = a;
    d.counter[0] = 0;
  }
  if (tid < kCandidates) d.lm_trials[tid] = tid < c1 ? Ec[tid] : inf;
  __syncthreads();
  const int a = acc_c;
  if (a >= 0) {  // the accepted candidate's Theta and tables, in 16-byte pieces (a piece per thread)
    const float4* H = reinterpret_cast<const float4*>(d.Hd_c + (size_t)a * L);
    const float4* X = reinterpret_cast<const float4*>(d.xi_c + (size_t)a * L * 8);
    for (int t = tid; t < 4 * L; t += kBlock) {
      if (t < 2 * L) reinterpret_cast<float4*>(d.Hd)[t] = H[t];
      else reinterpret_cast<float4*>(d.xi)[t - 2 * L] = X[t - 2 * L];
    }
    for (int j = tid; j < L; j += kBlock) d.theta[j] = d.theta_c[(size_t)a * L + j];
  }
}

constexpr int kFirstPass = 2;  // candidates scored by the first pass

template <int c0, int c1>
__global__ void __launch_bounds__(kBlock) k_lm_eval(BatchGrid g, Dev d0) {
  if (g.map == nullptr) {
    lm_eval_impl<c0, c1>(d0, grid_pos());
    return;
  }
  // the second pass mostly has nothing to do: looked up before the descriptor is staged
  if (c0 > 0 && g.devs[g.map[blockIdx.x].x].lm_trials[7] != kPending) return;
  __shared__ Dev sd;
  lm_eval_impl<c0, c1>(sd, batch_block(g, sd));
}

void launch_lm_solve(const Dev& d, cudaStream_t st) {
  k_lm_solve<false><<<kCandidates, kSolveThreads, SolveLayout<false>::bytes(d.L), st>>>(kSingle, d);
}

void launch_lm_eval(const Dev& d, int /*phi_buf: the rows' records already hold x0 + phi*/, cudaStream_t st) {
  const size_t sm = kCandidates * d.L * sizeof(DQ);
  k_lm_eval<0, kFirstPass><<<d.nblk_rows, kBlock, sm, st>>>(kSingle, d);
  k_lm_eval<kFirstPass, kCandidates><<<d.nblk_rows, kBlock, sm, st>>>(kSingle, d);
}

void launch_lm(const Dev& d, int phi_buf, cudaStream_t st) {
  launch_lm_solve(d, st);
  launch_lm_eval(d, phi_buf, st);
}

// ---------------------------------------------------------------------------------------------
// Sec. 4.3 shape step (per vertex, neighbours frozen): e_i = [i in A] r_i^2 + lambda_phi |phi_i|^2 +
// lambda_N sum_n |phi_i - phi_n|^2 with g_i = dr_i/dphi_i = -R(a^_i)^T n_i; one damped 3x3 Gauss-Newton
// solve (M + lambda_w diag M) delta = -(g r + lambda_phi phi_i + lambda_N sum_n (phi_i - phi_n)),
// M = g g^T + (lambda_phi + lambda_N |N(i)|) I, written to the other Jacobi buffer.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ float3 solve3_damped(float3 g, float cdiag, float lw, float3 rhs) {
  // M + lw diag(M), M = g g^T + cdiag I  (Cramer's rule)
  float m00 = g.x * g.x + cdiag, m11 = g.y * g.y + cdiag, m22 = g.z * g.z + cdiag;
  const float m01 = g.x * g.y, m02 = g.x * g.z, m12 = g.y * g.z;
  m00 += lw * m00; m11 += lw * m11; m22 += lw * m22;
  const float c00 = m11 * m22 - m12 * m12, c01 = m02 * m12 - m01 * m22, c02 = m01 * m12 - m02 * m11;
  const float det = m00 * c00 + m01 * c01 + m02 * c02;
  if (det == 0.f) return make_float3(0.f, 0.f, 0.f);
  const float c11 = m00 * m22 - m02 * m02, c12 = m01 * m02 - m00 * m12, c22 = m00 * m11 - m01 * m01;
  const float id = 1.f / det;
  return make_float3((c00 * rhs.x + c01 * rhs.y + c02 * rhs.z) * id, (c01 * rhs.x + c11 * rhs.y + c12 * rhs.z) * id,
                     (c02 * rhs.x + c12 * rhs.y + c22 * rhs.z) * id);
}

// Sum of v[0 .. kBlock) as a binary tree over the threads (v[t] += v[t + h], h = 128, .., 1), in thread 0; the
// last five levels by shuffles.  The caller has synchronised after writing v.
__device__ __forceinline__ double block_tree(double* v) {
  for (int h = kBlock / 2; h >= 32; h >>= 1) {
    if (threadIdx.x < h) v[threadIdx.x] += v[threadIdx.x + h];
    __syncthreads();
  }
  double x = threadIdx.x < 32 ? v[threadIdx.x] : 0.0;
  if (threadIdx.x < 32)
    for (int h = 16; h > 0; h >>= 1) x += __shfl_down_sync(0xffffffffu, x, h);
  return x;
}

__device__ __forceinline__ void block_energy_to_slot(const Dev& d, BlockPos bp, float e, int slot, int ticket) {
  __shared__ double sw[kBlock];
  __shared__ bool last;
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) s += sw[w];
    d.epart[(size_t)bp.x * 8] = s;
    __threadfence();
    last = atomicAdd(&d.counter[ticket], 1u) == (unsigned)bp.gx - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double s = 0.0;  // fixed order: strided per thread, then a tree over the threads
  for (int b = threadIdx.x; b < bp.gx; b += kBlock) s += __ldcg(d.epart + (size_t)b * 8);
  sw[threadIdx.x] = s;
  __syncthreads();
  const double total = block_tree(sw);
  if (threadIdx.x == 0) {
    if (slot >= 0) d.energy[slot] = total;
    d.counter[ticket] = 0;
  }
}

// r_i (the mean offset of the associated pixels along n_i) and g_i = dr_i/dphi_i = -R(a^_i)^T n_i.
__device__ __forceinline__ void vertex_r_g(const DQ* sHd, uchar4 bi, float4 bw, const Acc4& a4, const float4& nn,
                                           float& r, float3& g) {
  const float inv = 1.f / ((float)a4.w * kFix);
  r = nn.x * (float)a4.x * inv + nn.y * (float)a4.y * inv + nn.z * (float)a4.z * inv;
  float sg[4];
  const DQ H = blend_bones(sHd, bi, bw, sg);
  const float4 ah = qscale(H.r, rsqrtf(qdot(H.r, H.r)));
  const float4 q = qmul(qmul(qconj(ah), make_float4(0.f, nn.x, nn.y, nn.z)), ah);  // R^T n
  g = make_float3(-q.y, -q.z, -q.w);
}

__device__ __forceinline__ void shape_impl(const Dev& d, BlockPos bp, int src, int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  DQ* sHd = reinterpret_cast<DQ*>(smem_raw);
  const int i = bp.x * kBlock + threadIdx.x;
  bool anyA = false;
  if (i < d.V) anyA = d.acc[i].w >= 1 && d.n[i].w > 0.f;
  if (__syncthreads_or(anyA)) {  // the pose tables are needed only where a vertex of A is
    for (int j = threadIdx.x; j < d.L; j += kBlock) sHd[j] = d.Hd[j];
    __syncthreads();
  }
  float e = 0.f;
  int inA_count = 0;
  if (i < d.V) {
    const float4* phi = d.phi[src];
    const float4 p4 = phi[i];
    const float3 pi = f3(p4);
    const Acc4 a4 = d.acc[i];
    const float4 nn = d.n[i];
    const bool inA = a4.w >= 1 && nn.w > 0.f;
    float r = 0.f;
    float3 g = make_float3(0.f, 0.f, 0.f);
    if (inA) {
      inA_count = 1;
      vertex_r_g(sHd, d.bidx[i], d.bw[i], a4, nn, r, g);
    }
    e = r * r + d.lambda_phi * dot3(pi, pi);
    float3 sd = make_float3(0.f, 0.f, 0.f);
    int nn_count = 0;
    const int4 nb = d.nbr[i];
    const int nbs[4] = {nb.x, nb.y, nb.z, nb.w};
    float4 qn[4];  // the neighbours' offsets, all in flight before they are used
#pragma unroll
    for (int t = 0; t < 4; ++t) qn[t] = t < d.knn && nbs[t] >= 0 ? phi[nbs[t]] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (t >= d.knn || nbs[t] < 0) continue;
      const float3 q = f3(qn[t]);
      const float3 df = make_float3(pi.x - q.x, pi.y - q.y, pi.z - q.z);
      e += d.lambda_N * dot3(df, df);
      sd.x += df.x; sd.y += df.y; sd.z += df.z;
      ++nn_count;
    }
    const float3 grad = make_float3(g.x * r + d.lambda_phi * pi.x + d.lambda_N * sd.x,
                                    g.y * r + d.lambda_phi * pi.y + d.lambda_N * sd.y,
                                    g.z * r + d.lambda_phi * pi.z + d.lambda_N * sd.z);
    const float3 dl = solve3_damped(g, d.lambda_phi + d.lambda_N * nn_count, d.lambda_w,
                                    make_float3(-grad.x, -grad.y, -grad.z));
    d.phi[1 - src][i] = make_float4(pi.x + dl.x, pi.y + dl.y, pi.z + dl.z, 0.f);
    d.rg[i] = make_float4(g.x, g.y, g.z, r);
    d.phi0[i] = p4;
  }
  const unsigned m = __ballot_sync(0xffffffffu, inA_count != 0);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(&d.stats[1], __popc(m));
  block_energy_to_slot(d, bp, e, slot, 1);
}

__global__ void __launch_bounds__(kBlock) k_shape(BatchGrid g, Dev d0, int src, int slot) {
  if (g.map == nullptr) {
    shape_impl(d0, grid_pos(), src, slot);
    return;
  }
  __shared__ Dev sd;
  shape_impl(sd, batch_block(g, sd), src, slot);
}

// A batch's launch: registers sized for kBatchMinBlocks resident blocks (a few spills for occupancy).
__global__ void __launch_bounds__(kBlock, kBatchMinBlocks) k_shape_b(BatchGrid g, int src, int slot) {
  __shared__ Dev sd;
  shape_impl(sd, batch_block(g, sd), src, slot);
}

// Further Jacobi sweeps: r_i is updated linearly, r_i = r0_i + g_i . (phi_i - phi0_i).
__device__ __forceinline__ void shape_sweep_impl(const Dev& d, BlockPos bp, int src) {
  const int i = bp.x * kBlock + threadIdx.x;
  if (i >= d.V) return;
  const float4* phi = d.phi[src];
  const float3 pi = f3(phi[i]);
  const float4 rg = d.rg[i];
  const float3 g = f3(rg), p0 = f3(d.phi0[i]);
  const float r = rg.w + g.x * (pi.x - p0.x) + g.y * (pi.y - p0.y) + g.z * (pi.z - p0.z);
  float3 sd = make_float3(0.f, 0.f, 0.f);
  int nn_count = 0;
  const int4 nb = d.nbr[i];
  const int nbs[4] = {nb.x, nb.y, nb.z, nb.w};
  float4 qn[4];
#pragma unroll
  for (int t = 0; t < 4; ++t) qn[t] = t < d.knn && nbs[t] >= 0 ? phi[nbs[t]] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (t >= d.knn || nbs[t] < 0) continue;
    const float3 q = f3(qn[t]);
    sd.x += pi.x - q.x; sd.y += pi.y - q.y; sd.z += pi.z - q.z;
    ++nn_count;
  }
  const float3 grad = make_float3(g.x * r + d.lambda_phi * pi.x + d.lambda_N * sd.x,
                                  g.y * r + d.lambda_phi * pi.y + d.lambda_N * sd.y,
                                  g.z * r + d.lambda_phi * pi.z + d.lambda_N * sd.z);
  const float3 dl = solve3_damped(g, d.lambda_phi + d.lambda_N * nn_count, d.lambda_w,
                                  make_float3(-grad.x, -grad.y, -grad.z));
  d.phi[1 - src][i] = make_float4(pi.x + dl.x, pi.y + dl.y, pi.z + dl.z, 0.f);
}

__global__ void __launch_bounds__(kBlock) k_shape_sweep(BatchGrid g, Dev d0, int src) {
  if (g.map == nullptr) {
    shape_sweep_impl(d0, grid_pos(), src);
    return;
  }
  __shared__ Dev sd;
  shape_sweep_impl(sd, batch_block(g, sd), src);
}

// ---------------------------------------------------------------------------------------------
// Coupled shape step (the whole shape energy of Sec. 4.3, linearised in r): (H + lambda_w diag H) delta
// = -b with H_ii = [A] g g^T + (lambda_phi + lambda_N deg_i) I and H_ij = -lambda_N I per neighbourhood
// edge (either direction), by conjugate gradients preconditioned with the 3x3 diagonal blocks.  Vectors
// in FP32, dot products in FP64 with fixed-order block sums (deterministic); a breakdown (r.z = 0 or
// p.Ap <= 0) stops the iteration as in exact arithmetic.  One kernel per CG phase.
// ---------------------------------------------------------------------------------------------
// Block sum of v (FP64) into epart[bp.x * 8 + slot]; returns true in every thread of the session's last
// block, with the fixed-order total of all its blocks in thread 0's `total`.
__device__ __forceinline__ bool block_total(const Dev& d, BlockPos bp, double v, int slot, int ticket, double& total) {
  __shared__ double sw[kBlock / 32];
  __shared__ double red[kBlock];
  __shared__ bool last;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kBlock / 32; ++w) s += sw[w];
    d.epart[(size_t)bp.x * 8 + slot] = s;
    __threadfence();
    last = atomicAdd(&d.counter[ticket], 1u) == (unsigned)bp.gx - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double s = 0.0;
  for (int b = threadIdx.x; b < bp.gx; b += kBlock) s += __ldcg(d.epart + (size_t)b * 8 + slot);
  red[threadIdx.x] = s;
  __syncthreads();
  total = block_tree(red);
  if (threadIdx.x == 0) d.counter[ticket] = 0;
  return true;
}

// a.b in FP64 (products of FP32 numbers are exact there), whole warps; the conversions without the FP64 pipe.
__device__ __forceinline__ double dot3_fp64(float3 a, float3 b) {
  bool other = false;
  double ax = widen(a.x, other), ay = widen(a.y, other), az = widen(a.z, other);
  double bx = widen(b.x, other), by = widen(b.y, other), bz = widen(b.z, other);
  if (__any_sync(0xffffffffu, other)) {
    ax = (double)a.x, ay = (double)a.y, az = (double)a.z;
    bx = (double)b.x, by = (double)b.y, bz = (double)b.z;
  }
  return ax * bx + ay * by + az * bz;
}

// B_i = M_i + lambda_w diag(M_i), M_i = g g^T + c I (g = 0 outside A): B_i p and B_i^-1 p.
__device__ __forceinline__ float3 block_apply(float3 g, float c, float lw, float3 p) {
  const float gp = g.x * p.x + g.y * p.y + g.z * p.z;
  return make_float3(g.x * gp + c * p.x + lw * (g.x * g.x + c) * p.x, g.y * gp + c * p.y + lw * (g.y * g.y + c) * p.y,
                     g.z * gp + c * p.z + lw * (g.z * g.z + c) * p.z);
}

// r_i, g_i, E_shape (energy[slot]) as the Jacobi step; b; x = 0, r = -b, z = B^-1 r, p = z, rz = r.z.
__device__ __forceinline__ void cg_init_impl(const Dev& d, BlockPos bp, int src, int slot) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  DQ* sHd = reinterpret_cast<DQ*>(smem_raw);
  const int i = bp.x * kBlock + threadIdx.x;
  bool anyA = false;
  if (i < d.V) anyA = d.acc[i].w >= 1 && d.n[i].w > 0.f;
  if (__syncthreads_or(anyA)) {
    for (int j = threadIdx.x; j < d.L; j += kBlock) sHd[j] = d.Hd[j];
    __syncthreads();
  }
  float e = 0.f;
  float3 rr = make_float3(0.f, 0.f, 0.f), z = rr;
  int inA_count = 0;
  if (i < d.V) {
    const float4* phi = d.phi[src];
    const float4 p4 = phi[i];
    const float3 pi = f3(p4);
    const Acc4 a4 = d.acc[i];
    const float4 nn = d.n[i];
    float r = 0.f;
    float3 g = make_float3(0.f, 0.f, 0.f);
    if (a4.w >= 1 && nn.w > 0.f) {
      inA_count = 1;
      vertex_r_g(sHd, d.bidx[i], d.bw[i], a4, nn, r, g);
    }
    e = r * r + d.lambda_phi * dot3(pi, pi);
    const int4 nb = d.nbr[i];
    const int nbs[4] = {nb.x, nb.y, nb.z, nb.w};
    for (int t = 0; t < d.knn; ++t) {
      if (nbs[t] < 0) continue;
      const float3 q = f3(phi[nbs[t]]);
      const float3 df = make_float3(pi.x - q.x, pi.y - q.y, pi.z - q.z);
      e += d.lambda_N * dot3(df, df);
    }
    float3 sd = make_float3(0.f, 0.f, 0.f);
    const int a0 = d.adj_off[i], a1 = d.adj_off[i + 1];
    for (int t = a0; t < a1; ++t) {
      const float3 q = f3(phi[d.adj[t]]);
      sd.x += pi.x - q.x; sd.y += pi.y - q.y; sd.z += pi.z - q.z;
    }
    rr = make_float3(-(g.x * r + d.lambda_phi * pi.x + d.lambda_N * sd.x),
                     -(g.y * r + d.lambda_phi * pi.y + d.lambda_N * sd.y),
                     -(g.z * r + d.lambda_phi * pi.z + d.lambda_N * sd.z));
    z = solve3_damped(g, d.lambda_phi + d.lambda_N * (float)(a1 - a0), d.lambda_w, rr);
    d.rg[i] = make_float4(g.x, g.y, g.z, r);
    d.phi0[i] = p4;
    d.cg_x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    d.cg_r[i] = make_float4(rr.x, rr.y, rr.z, 0.f);
    d.cg_z[i] = make_float4(z.x, z.y, z.z, 0.f);
    d.cg_p[i] = make_float4(z.x, z.y, z.z, 0.f);
  }
  const double rz = dot3_fp64(rr, z);
  const unsigned m = __ballot_sync(0xffffffffu, inA_count != 0);
  if ((threadIdx.x & 31) == 0 && m) atomicAdd(&d.stats[1], __popc(m));
  double tot;
  if (block_total(d, bp, rz, 1, 2, tot) && threadIdx.x == 0) {
    d.cg[0] = tot;
    d.cg[3] = tot > 0.0 ? 0.0 : 1.0;  // stopped if the preconditioned residual is already zero
  }
  block_energy_to_slot(d, bp, e, slot, 1);
}

// The direction of iteration k: of odd ones in the Phi buffer that receives the result (nothing reads that before the
// last iteration, and there each thread only its own entry, before it writes the result over it).
__device__ __forceinline__ float4* cg_direction(const Dev& d, int src, int k) { return k & 1 ? d.phi[1 - src] : d.cg_p; }

// Iteration k > 0: p = z + beta p first (the neighbours' too, each formed from its z and old p, so that the
// direction needs no pass of its own; p is written to the other buffer).  Ap = (B - lambda_N Adj) p;
// alpha = r.z / p.Ap (0 and stop on a breakdown).  Bound by the latency of its gathers, which warps hide
// better than loads ahead do: one neighbour at a time in 32 registers, eight blocks per SM (a coupled step of
// eight iterations at 55k and 200k vertices and of sixteen sessions of 50k: 180, 307 and 769 us; eight
// neighbours ahead in 80 registers: 188, 322 and 904; a pass of its own for p, in 40: 213, 330 and 796).
__device__ __forceinline__ void cg_apply_impl(const Dev& d, BlockPos bp, int src, int k) {
  const int i = bp.x * kBlock + threadIdx.x;
  float3 p = make_float3(0.f, 0.f, 0.f), ap = p;
  if (i < d.V) {
    const float beta = (float)d.cg[2];
    const float4* old = cg_direction(d, src, k - 1);
    auto direction = [&](int j) {
      if (k == 0) return f3(d.cg_p[j]);
      const float3 z = f3(d.cg_z[j]), q = f3(old[j]);
      return make_float3(z.x + beta * q.x, z.y + beta * q.y, z.z + beta * q.z);
    };
    const float4 rg = d.rg[i];
    p = direction(i);
    if (k > 0) cg_direction(d, src, k)[i] = make_float4(p.x, p.y, p.z, 0.f);
    const int a0 = d.adj_off[i], a1 = d.adj_off[i + 1];
    ap = block_apply(f3(rg), d.lambda_phi + d.lambda_N * (float)(a1 - a0), d.lambda_w, p);
#pragma unroll 1
    for (int t = a0; t < a1; ++t) {
      const float3 q = direction(d.adj[t]);
      ap.x -= d.lambda_N * q.x; ap.y -= d.lambda_N * q.y; ap.z -= d.lambda_N * q.z;
    }
    d.cg_ap[i] = make_float4(ap.x, ap.y, ap.z, 0.f);
  }
  const double pap = dot3_fp64(p, ap);
  double tot;
  if (block_total(d, bp, pap, 2, 3, tot) && threadIdx.x == 0) {
    const bool go = d.cg[3] == 0.0 && tot > 0.0;
    d.cg[1] = go ? d.cg[0] / tot : 0.0;
    if (!go) d.cg[3] = 1.0;
  }
}

// x += alpha p, r -= alpha Ap, z = B^-1 r; beta = r.z_new / r.z.  The last iteration: phi[1 - src] =
// phi[src] + x.
__device__ __forceinline__ void cg_update_impl(const Dev& d, BlockPos bp, int src, int k, bool last) {
  const int i = bp.x * kBlock + threadIdx.x;
  float3 r = make_float3(0.f, 0.f, 0.f), z = r;
  if (i < d.V) {
    const float alpha = (float)d.cg[1];
    const float4 rg = d.rg[i];
    const float3 p = f3(cg_direction(d, src, k)[i]), ap = f3(d.cg_ap[i]);
    float3 x = f3(d.cg_x[i]);
    r = f3(d.cg_r[i]);
    x.x += alpha * p.x; x.y += alpha * p.y; x.z += alpha * p.z;
    r.x -= alpha * ap.x; r.y -= alpha * ap.y; r.z -= alpha * ap.z;
    const int deg = d.adj_off[i + 1] - d.adj_off[i];
    z = solve3_damped(f3(rg), d.lambda_phi + d.lambda_N * (float)deg, d.lambda_w, r);
    d.cg_x[i] = make_float4(x.x, x.y, x.z, 0.f);
    d.cg_r[i] = make_float4(r.x, r.y, r.z, 0.f);
    d.cg_z[i] = make_float4(z.x, z.y, z.z, 0.f);
    if (last) {
      const float4 f = d.phi[src][i];
      d.phi[1 - src][i] = make_float4(f.x + x.x, f.y + x.y, f.z + x.z, 0.f);
    }
  }
  const double rz = dot3_fp64(r, z);
  double tot;
  if (block_total(d, bp, rz, 1, 2, tot) && threadIdx.x == 0) {
    const bool go = d.cg[3] == 0.0 && d.cg[0] > 0.0;
    d.cg[2] = go ? tot / d.cg[0] : 0.0;
    d.cg[0] = tot;
    if (!(tot > 0.0)) d.cg[3] = 1.0;
  }
}

#define TRK_CG_KERNEL(name, impl, blocks_per_sm)                                           \
  __global__ void __launch_bounds__(kBlock, blocks_per_sm) name(BatchGrid g, Dev d0 ARGS_##name) {         \
    if (g.map == nullptr) {                                                                  \
      impl(d0, grid_pos() CALL_##name);                                                      \
      return;                                                                                \
    }                                                                                        \
    __shared__ Dev sd;                                                                       \
    impl(sd, batch_block(g, sd) CALL_##name);                                                \
  }
#define ARGS_k_cg_init , int src, int slot
#define CALL_k_cg_init , src, slot
#define ARGS_k_cg_apply , int src, int k
#define CALL_k_cg_apply , src, k
#define ARGS_k_cg_update , int src, int k, bool last
#define CALL_k_cg_update , src, k, last
TRK_CG_KERNEL(k_cg_init, cg_init_impl, 5)
TRK_CG_KERNEL(k_cg_apply, cg_apply_impl, 8)
TRK_CG_KERNEL(k_cg_update, cg_update_impl, 8)

// The whole coupled step (g, n: the block table and its size for a batch; kSingle and nblk_v alone).
static void launch_shape_pcg(const BatchGrid& g, int n, const Dev& d0, int max_links, int iters, int src, int slot,
                             cudaStream_t st) {
  if (n <= 0) return;
  k_cg_init<<<n, kBlock, max_links * sizeof(DQ), st>>>(g, d0, src, slot);
  for (int k = 0; k < iters; ++k) {
    k_cg_apply<<<n, kBlock, 0, st>>>(g, d0, src, k);
    k_cg_update<<<n, kBlock, 0, st>>>(g, d0, src, k, k + 1 == iters);
  }
}

// Returns the buffer that holds Phi after the step.
int launch_shape(const Dev& d, int phi_src, int slot, cudaStream_t st) {
  if (d.shape_solver == 1) {
    launch_shape_pcg(kSingle, d.nblk_v, d, d.L, d.shape_sweeps, phi_src, slot, st);
    return 1 - phi_src;
  }
  k_shape<<<d.nblk_v, kBlock, d.L * sizeof(DQ), st>>>(kSingle, d, phi_src, slot);
  int cur = 1 - phi_src;
  for (int s = 1; s < d.shape_sweeps; ++s) {
    k_shape_sweep<<<d.nblk_v, kBlock, 0, st>>>(kSingle, d, cur);
    cur = 1 - cur;
  }
  return cur;
}

// ---- batched launches ------------------------------------------------------------------------
template <int PREC>
static void launch_resid_jtj_tc_b(const BatchGrid& g, int nblk, int max_np, int max_links, int phi_buf,
                                  cudaStream_t st) {
  const int NB = (max_np + 15) / 16;
  const int sm = jtj_tc_smem_bytes<PREC>(NB, max_links);
  switch (NB) {
    case 1: k_resid_jtj_tc<PREC, 1><<<nblk, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
    case 2: k_resid_jtj_tc<PREC, 2><<<nblk, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
    case 3: k_resid_jtj_tc<PREC, 3><<<nblk, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
    case 4: k_resid_jtj_tc<PREC, 4><<<nblk, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
    default: k_resid_jtj_tc<PREC, 5><<<nblk, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
  }
}

// gj[t - 1], nj[t - 1]: the blocks of the sessions whose [J r] tile width class is t = ceil(NP / 16)
// (one launch per class, so a small skeleton does not pay for the largest one's tiles).  A class of a few
// sessions does not fill the chip, so the classes run beside each other where the caller has the streams for it
// (eight uneven sessions, four classes of 86 to 492 blocks: one after the other they took 108 us).
void launch_normal_equations_b(const BatchGrid* gj, const int* nj, const BatchGrid& gr, int nr, int max_links,
                               int precision, int phi_buf, int slot, cudaStream_t main, int reduce_threads,
                               const ForkStreams* fork) {
  int last = 0;
  for (int T = 1; T <= 5; ++T)
    if (nj[T - 1] > 0) last = T;
  int sides = 0;
  for (int T = 1; T <= 5; ++T) {
    const BatchGrid& g = gj[T - 1];
    const int n = nj[T - 1];
    if (n == 0) continue;
    cudaStream_t st = main;
    if (fork && T != last) {
      if (sides == 0) cudaEventRecord(fork->fork, main);
      st = fork->side[sides];
      cudaStreamWaitEvent(st, fork->fork, 0);
    }
    if (precision == 1) {
      launch_resid_jtj_tc_b<1>(g, n, 16 * T, max_links, phi_buf, st);
    } else if (precision == 2) {
      launch_resid_jtj_tc_b<2>(g, n, 16 * T, max_links, phi_buf, st);
    } else {
      const int sm = jtj_smem_bytes(T, max_links);
      switch (T) {
        case 1: k_resid_jtj<1><<<n, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
        case 2: k_resid_jtj<2><<<n, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
        case 3: k_resid_jtj<3><<<n, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
        case 4: k_resid_jtj<4><<<n, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
        default: k_resid_jtj<5><<<n, kBlock, sm, st>>>(g, Dev{}, phi_buf); break;
      }
    }
    if (st != main) cudaEventRecord(fork->join[sides++], st);
  }
  for (int k = 0; k < sides; ++k) cudaStreamWaitEvent(main, fork->join[k], 0);
  if (nr > 0) k_reduce_jtj<<<nr, reduce_threads, 0, main>>>(gr, Dev{}, slot);
}

void launch_lm_b(const BatchGrid& glm, int nlm, const BatchGrid& gv, int nv, int max_links, int phi_buf,
                 cudaStream_t st) {
  // 3 x 192 threads per SM where that takes fewer waves than 2 x 256: 64 sessions of 55 links 50 us against 70, 52
  // sessions 48 against 66, 100 sessions (two waves either way) 80 against 72
  auto waves = [nlm](int blocks_per_sm) { return (nlm + 152 * blocks_per_sm - 1) / (152 * blocks_per_sm); };
  if (waves(kCrowdBlocksPerSM) < waves(kSolveBlocksPerSM)) {
    k_lm_solve<true><<<nlm, kCrowdThreads, SolveLayout<true>::bytes(max_links), st>>>(glm, Dev{});
  } else if (nlm > 0) {
    k_lm_solve<false><<<nlm, kSolveThreads, SolveLayout<false>::bytes(max_links), st>>>(glm, Dev{});
  }
  if (nv > 0) {
    const size_t sm = kCandidates * max_links * sizeof(DQ);
    k_lm_eval<0, kFirstPass><<<nv, kBlock, sm, st>>>(gv, Dev{});
    k_lm_eval<kFirstPass, kCandidates><<<nv, kBlock, sm, st>>>(gv, Dev{});
  }
}

int launch_shape_b(const BatchGrid& gv, int nv, int max_links, int sweeps, int solver, int phi_src, int slot,
                   cudaStream_t st) {
  if (solver == 1) {
    launch_shape_pcg(gv, nv, Dev{}, max_links, sweeps, phi_src, slot, st);
    return 1 - phi_src;
  }
  if (nv > 0) k_shape_b<<<nv, kBlock, max_links * sizeof(DQ), st>>>(gv, phi_src, slot);
  int cur = 1 - phi_src;
  for (int s = 1; s < sweeps; ++s) {
    if (nv > 0) k_shape_sweep<<<nv, kBlock, 0, st>>>(gv, Dev{}, cur);
    cur = 1 - cur;
  }
  return cur;
}

static void configure_batched() {
  cudaFuncSetAttribute(k_lm_solve<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       SolveLayout<true>::bytes(kMaxLinks));
}

void configure_tc_kernels();

void configure_kernels() {
  configure_tc_kernels();
  configure_batched();
  configure_resid_jtj_tc<1>();
  configure_resid_jtj_tc<2>();
  cudaFuncSetAttribute(k_resid_jtj<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_smem_bytes(1, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_smem_bytes(2, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_smem_bytes(3, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_smem_bytes(4, kMaxLinks));
  cudaFuncSetAttribute(k_resid_jtj<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, jtj_smem_bytes(5, kMaxLinks));
  cudaFuncSetAttribute(k_lm_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       SolveLayout<false>::bytes(kMaxLinks));
}

// Sets the kernels' shared-memory limits once per device (the attributes are per device).
void ensure_configured() {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev]) {
    configure_kernels();
    done[dev] = true;
  }
}

}  // namespace trk
