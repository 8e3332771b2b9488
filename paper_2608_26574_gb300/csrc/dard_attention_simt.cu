// dard_attention_simt.cu - the fp32 attention kernel on CUDA cores (dtype F32): the
// validation path and the kernel of fp32 workloads. Same mask as the tensor-core kernels
// (Sec. 3.1 Eq. 2; Sec. 3.2 query blocks 1-6, Eq. 3), through key_visible(), and the same
// RoPE positions (dard_rope.cuh).
#include "dard_attn_common.cuh"

namespace dard {
namespace {

// ---------------------------------------------------------------- fp32 CUDA-core path
// A CTA holds 32 query rows of one head (a quarter of a 128-row query tile), four threads per
// row in each of four key groups, 512 threads: thread `part` of a row owns the four-element
// vectors 16 v + 4 part .. 16 v + 4 part + 3 (v = 0 .. D/16 - 1) of q and of its O
// accumulator, so that the row's four threads read 64 contiguous bytes of a shared-memory
// key row per vector (one 16-byte load each, no bank conflict). The sequence's keys pass
// through shared memory 32 rows at a time (K and V, read as broadcasts; four tiles in
// flight by cp.async, the first four issued before the block's metadata is read, so that a
// short sequence waits for memory once); key group `grp` takes
// keys 8 grp .. 8 grp + 7 of every tile, four at a time: four independent partial dot
// products, which the row's four threads add up with two shuffles each, then one online
// softmax step over the four. At the end the four groups' (maximum, sum, accumulator) of a
// row are merged through shared memory. Masking as on the tensor-core path, by
// key_visible().
constexpr int kSimtParts = 4;     // threads per query row and key group
constexpr int kSimtGroups = 4;    // key groups
constexpr int kSimtGroupThreads = kSimtRows * kSimtParts;
constexpr int kSimtThreads = kSimtGroupThreads * kSimtGroups;
constexpr int kSimtStages = 4;    // K/V tiles in shared memory
constexpr int kSimtKeys = 32;     // keys per tile
constexpr int kSimtSplit = kSimtCtasPerTile;  // CTAs per 128-row query tile
static_assert(kSimtSplit * kSimtRows == kBM, "the CTAs cover a 128-row query tile");

template <int D>
__global__ void __launch_bounds__(kSimtThreads) attn_simt(const __grid_constant__ AttnParams p) {
  constexpr int kV = D / 16;                   // float4 vectors per thread
  constexpr int kKT = kSimtKeys;               // keys per shared-memory tile
  constexpr int kKG = kKT / kSimtGroups;       // keys of a tile per key group
  static_assert(kKG % 4 == 0, "four keys per step");
  static_assert(kKT >= kSimtRows, "the merge reuses the K and V tile buffers, one row block each");
  __shared__ BlockInfo bi;
  extern __shared__ __align__(16) float smem[];  // kSimtStages tiles of K, then of V
  using Tile = float[kKT][D];
  Tile* const sKs = reinterpret_cast<Tile*>(smem);
  Tile* const sVs = sKs + kSimtStages;
  __shared__ float s_m[kSimtGroups][kSimtRows], s_l[kSimtGroups][kSimtRows];
  int seq, qt, h;
  decode_work(p, blockIdx.x / kSimtSplit, seq, qt, h);
  const int sub = blockIdx.x % kSimtSplit;
  const SeqDesc sd = p.seq[seq];
  const int rows_seq = sd.n_orig + sd.slen;
  const int r0 = sd.q_start + qt * kBM + sub * kSimtRows;  // first (sequence-relative) query row
  if (r0 >= rows_seq) return;
  const int g = h / (p.hq / p.hkv);
  const float* K = static_cast<const float*>(p.k);
  const float* V = static_cast<const float*>(p.v);
  // the rows of keys kt0 .. kt0 + 31 into a stage (rows past the sequence as zeros)
  auto copy_rows = [&](Tile& dst, const float* src, int kt0) {
#pragma unroll
    for (int u = 0; u < kKT * D / 4 / kSimtThreads; ++u) {
      const int idx = static_cast<int>(threadIdx.x) + u * kSimtThreads;
      const int kr = kt0 + idx / (D / 4), c4 = idx % (D / 4);
      if (kt0 >= rows_seq) break;
      const bool in = kr < rows_seq;
      const size_t off =
          (static_cast<size_t>(sd.row_base + (in ? kr : 0)) * p.hkv + g) * D + 4 * c4;
      cp_async16(&dst[0][0] + 4 * idx, src + off, in ? 16 : 0);
    }
  };
  // K and V of a tile into stage st; every thread commits one group per tile, copies or none
  auto copy_tile = [&](int kt0, int st) {
    copy_rows(sKs[st], K, kt0);
    copy_rows(sVs[st], V, kt0);
    cp_async_commit();
  };
  static_assert(kKT * D / 4 % kSimtThreads == 0, "a tile splits evenly over the threads");
  // The first tiles before anything else: they land while the block is read. With RoPE the keys
  // come from the pass launched before this kernel, which is waited for only once the block has
  // been read and the query row rotated (one call of 96 rows and four heads with head_dim 64, us:
  // waited for first 20.8, so 18.4); V does not depend on it.
#pragma unroll
  for (int st = 0; st < kSimtStages; ++st) {
    if (p.rope) copy_rows(sVs[st], V, st * kKT);
    else copy_tile(st * kKT, st);
  }
  if (threadIdx.x < 128)  // warps 0-3
    load_block_info(p, sd, bi, qt == 0 && h == 0 && sub == 0);
  __syncthreads();
  const int grp = threadIdx.x / kSimtGroupThreads, local = threadIdx.x % kSimtGroupThreads;
  const int t = local / kSimtParts, part = local % kSimtParts;
  const unsigned quad = 0xfu << ((threadIdx.x & 31) & ~3);  // the row's four threads
  const int r = r0 + t;  // sequence-relative query row
  const bool active = r < rows_seq;
  RowInfo q{0, kStateU, 0.f, -1, 0};
  if (active) q = row_info(sd, bi, r);
  const bool live = active && q.store;
  const float* Q = static_cast<const float*>(p.q);
  float* O = static_cast<float*>(p.o);
  // vector v of this thread: float4 index 4 v + part of the row
  const size_t qoff4 = (static_cast<size_t>(sd.row_base + r) * p.hq + h) * (D / 4) + part;
  float4 qv[kV], acc[kV];
#pragma unroll
  for (int v = 0; v < kV; ++v) {
    qv[v] = live ? reinterpret_cast<const float4*>(Q)[qoff4 + 4 * v] : make_float4(0.f, 0.f, 0.f, 0.f);
    acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (p.rope && live) {  // RoPE of this row; its pairs lie within one thread
    const int pos = rope_position(p, sd, r);
    auto rot = [](float& a, float& b, float c, float s) {
      const float x = a, y = b;
      a = fmaf(x, c, -y * s);
      b = fmaf(x, s, y * c);
    };
    if (p.rope_style == DARD_ROPE_INTERLEAVED) {
      // elements (d, d + 1) of a vector, d = 16 v + 4 part + {0, 2}: frequency d / 2
#pragma unroll
      for (int v = 0; v < kV; ++v) {
        const int i = 8 * v + 2 * part;
        float c0, s0, c1, s1;
        rope_cos_sin(pos, p.rope_f[2 * i], p.rope_f[2 * i + 1], c0, s0);
        rope_cos_sin(pos, p.rope_f[2 * i + 2], p.rope_f[2 * i + 3], c1, s1);
        rot(qv[v].x, qv[v].y, c0, s0);
        rot(qv[v].z, qv[v].w, c1, s1);
      }
    } else {
      // element d = 16 v + 4 part + k < D/2 pairs with d + D/2 (vector v + kV/2): frequency d
#pragma unroll
      for (int v = 0; v < kV / 2; ++v) {
        const int i = 16 * v + 4 * part;
        float c[4], s[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) rope_cos_sin(pos, p.rope_f[2 * (i + k)], p.rope_f[2 * (i + k) + 1], c[k], s[k]);
        float4& a = qv[v];
        float4& b = qv[v + kV / 2];
        rot(a.x, b.x, c[0], s[0]);
        rot(a.y, b.y, c[1], s[1]);
        rot(a.z, b.z, c[2], s[2]);
        rot(a.w, b.w, c[3], s[3]);
      }
    }
  }
  if (p.rope) {
    grid_dep_wait();  // the key pass is complete
#pragma unroll
    for (int st = 0; st < kSimtStages; ++st) {
      copy_rows(sKs[st], K, st * kKT);
      cp_async_commit();  // the first group: every V tile so far, and K(0)
    }
  }
  float m = -INFINITY, l = 0.f;
  for (int kt0 = 0, t0 = 0; kt0 < rows_seq; kt0 += kKT, ++t0) {
    if (t0 > 0 && kt0 + (kSimtStages - 1) * kKT < rows_seq) {
      __syncthreads();  // the tile before has been read: its stage takes the tile kSimtStages on
      copy_tile(kt0 + (kSimtStages - 1) * kKT, (t0 - 1) % kSimtStages);
    } else if (t0 > 0) {
      cp_async_commit();
    }
    cp_async_wait<kSimtStages - 1>();
    __syncthreads();  // this tile has landed
    const auto& sK = sKs[t0 % kSimtStages];
    const auto& sV = sVs[t0 % kSimtStages];
    if (!live) continue;
    const int k_end = min(kKT, rows_seq - kt0);
    // four keys per step: four independent dot-product chains, one maximum and at most one
    // rescale per step (keys past the sequence or hidden by the mask weigh 0)
    for (int kk = grp * kKG; kk < grp * kKG + kKG && kk < k_end; kk += 4) {
      // Four keys before the shadow rows and outside the block are seen by every row, and nothing is
      // looked up (the same branch for a whole warp): that pays for leaving hidden keys out below
      // (564 rows, four heads, us: head_dim 64 67.6 without either, 66.6 and 61.4 with the second and
      // with both; head_dim 128 98.4, 100.3, 94.3).
      const int k0 = kt0 + kk;
      const bool open = k0 + 4 <= sd.n_orig && (k0 + 4 <= sd.b0 || k0 >= sd.b0 + sd.blen);
      bool vis[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        vis[u] = open || (kk + u < k_end && key_visible(q, bi, sd, k0 + u));  // the same for the row
      if (!(vis[0] || vis[1] || vis[2] || vis[3])) continue;
      float dot[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int v = 0; v < kV; ++v) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 kx = reinterpret_cast<const float4*>(sK[kk + u])[4 * v + part];
          dot[u] = fmaf(qv[v].x, kx.x, dot[u]);
          dot[u] = fmaf(qv[v].y, kx.y, dot[u]);
          dot[u] = fmaf(qv[v].z, kx.z, dot[u]);
          dot[u] = fmaf(qv[v].w, kx.w, dot[u]);
        }
      }
      float z[4];
      float zmax = -INFINITY;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        dot[u] += __shfl_xor_sync(quad, dot[u], 1);
        dot[u] += __shfl_xor_sync(quad, dot[u], 2);
        z[u] = vis[u] ? dot[u] * p.scale : -INFINITY;
        zmax = fmaxf(zmax, z[u]);
      }
      if (zmax > m) {
        const float alpha = (m == -INFINITY) ? 0.f : expf(m - zmax);
        l *= alpha;
#pragma unroll
        for (int v = 0; v < kV; ++v) {
          acc[v].x *= alpha;
          acc[v].y *= alpha;
          acc[v].z *= alpha;
          acc[v].w *= alpha;
        }
        m = zmax;
      }
      float pz[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        pz[u] = vis[u] ? expf(z[u] - m) : 0.f;
      }
      l += (pz[0] + pz[1]) + (pz[2] + pz[3]);
      // V of a key that the row does not see may hold anything, a NaN too: it is left out, not
      // multiplied by 0. The four products are summed apart, then added to the
      // accumulator: the error against 64 bits falls from 2.2e-7 to 1.4e-7 (8 heads of 64, 564 rows), the
      // same as attn_f32's, at 0 to 1 % of the time.
#pragma unroll
      for (int v = 0; v < kV; ++v) {
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 vx = reinterpret_cast<const float4*>(sV[kk + u])[4 * v + part];
          sum.x = vis[u] ? fmaf(pz[u], vx.x, sum.x) : sum.x;
          sum.y = vis[u] ? fmaf(pz[u], vx.y, sum.y) : sum.y;
          sum.z = vis[u] ? fmaf(pz[u], vx.z, sum.z) : sum.z;
          sum.w = vis[u] ? fmaf(pz[u], vx.w, sum.w) : sum.w;
        }
        acc[v].x += sum.x;
        acc[v].y += sum.y;
        acc[v].z += sum.z;
        acc[v].w += sum.w;
      }
    }
  }
  // Merge the key groups: groups 2 and 3 hand their state to groups 0 and 1, then group 1
  // to group 0, through the K and V tile buffers (free once every group is past its last
  // tile): group half + k writes into buffer k (sK for k = 0, sV for k = 1).
  Tile& sK = sKs[0];
  Tile& sV = sVs[0];
  if (part == 0) {
    s_m[grp][t] = m;
    s_l[grp][t] = l;
  }
  __syncthreads();
#pragma unroll
  for (int half = 2; half >= 1; half >>= 1) {
    if (grp >= half && grp < 2 * half) {
      float4* slot = reinterpret_cast<float4*>(grp == half ? &sK[0][0] : &sV[0][0]);
#pragma unroll
      for (int v = 0; v < kV; ++v) slot[t * (D / 4) + 4 * v + part] = acc[v];
    }
    __syncthreads();
    if (grp < half) {
      const float4* slot = reinterpret_cast<const float4*>(grp == 0 ? &sK[0][0] : &sV[0][0]);
      const float mo = s_m[grp + half][t], lo = s_l[grp + half][t];
      const float mn = fmaxf(m, mo);
      const float a = (m == -INFINITY) ? 0.f : expf(m - mn);
      const float b = (mo == -INFINITY) ? 0.f : expf(mo - mn);
      l = l * a + lo * b;
#pragma unroll
      for (int v = 0; v < kV; ++v) {
        const float4 o = slot[t * (D / 4) + 4 * v + part];
        acc[v].x = acc[v].x * a + o.x * b;
        acc[v].y = acc[v].y * a + o.y * b;
        acc[v].z = acc[v].z * a + o.z * b;
        acc[v].w = acc[v].w * a + o.w * b;
      }
      m = mn;
    }
    __syncthreads();
    if (grp < half && part == 0) {
      s_m[grp][t] = m;
      s_l[grp][t] = l;
    }
    __syncthreads();
  }
  if (live && grp == 0) {
    const float inv_l = 1.0f / l;
#pragma unroll
    for (int v = 0; v < kV; ++v)
      reinterpret_cast<float4*>(O)[qoff4 + 4 * v] =
          make_float4(acc[v].x * inv_l, acc[v].y * inv_l, acc[v].z * inv_l, acc[v].w * inv_l);
  }
}

template <int D>
cudaError_t launch_simt(const AttnParams& p, cudaStream_t stream) {
  static std::atomic<uint64_t> attr_done{0};
  const size_t smem = 2 * kSimtStages * kSimtKeys * D * sizeof(float);
  const cudaError_t e = ensure_smem_attr(attn_simt<D>, smem, attr_done);
  if (e != cudaSuccess) return e;
  const AttnLaunch L(p.total_work * kSimtSplit, kSimtThreads, smem, stream, 1, p.rope != 0);
  return cudaLaunchKernelEx(&L.cfg, attn_simt<D>, p);
}

}  // namespace

cudaError_t launch_simt_attention(const AttnParams& p, cudaStream_t stream) {
  return p.head_dim == 64 ? launch_simt<64>(p, stream) : launch_simt<128>(p, stream);
}

}  // namespace dard
