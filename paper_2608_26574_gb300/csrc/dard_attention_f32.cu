// dard_attention_f32.cu - the fp32 attention kernel for more than a few query tiles (dtype
// F32; attn_simt takes the small calls). Same mask as the tensor-core kernels (Sec. 3.1 Eq. 2;
// Sec. 3.2 query blocks 1-6, Eq. 3) and the same RoPE positions (dard_rope.cuh); fp32 FMAs
// throughout.
#include <type_traits>

#include "dard_attn_common.cuh"

namespace dard {
namespace {

// A CTA holds 64 query rows of one head, 128 threads: thread (ty, tx) = (tid / 16, tid % 16)
// owns rows 8 i + ty (i < 8). The keys pass through shared memory 32 rows at a time
// (two CTAs fit on an SM):
//   S = Q K^T: the thread's 8 x 2 scores (keys tx + 16 c), summed over pairs of d as packed
//     FMAs: 10 16-byte shared loads per 64 multiply-adds;
//   softmax: row maxima over the 16 threads of a row by shuffles, the weights P (fp32) to
//     shared memory, row sums kept per thread until the end;
//   O += P V: the thread's 8 rows x D / 16 columns (columns 4 tx + 64 c ..), packed FMAs over
//     pairs of columns.
// K(j + 1) is copied (cp.async) while the softmax and P V of tile j run, V(j) while S(j) runs.
// Bound: the FMA pipe (two products of 64 x 32 x D per tile), next the shared-memory loads;
// rows are padded so that the 16-byte loads of a warp hit each bank at most twice.
constexpr int kFRows = 64;   // query rows per CTA
constexpr int kFKeys = 32;   // keys per tile
constexpr int kNC = kFKeys / 16;  // keys per thread
constexpr int kFThreads = 128;
static_assert(kF32CtasPerTile * kFRows == kBM, "the CTAs cover a 128-row query tile");

template <int D>
struct __align__(16) F32Smem {
  float q[kFRows][D + 4];
  float k[kFKeys][D + 4];
  float v[kFKeys][D];
  float p[kFRows][kFKeys + 4];
  BlockInfo bi;
  RowMasks rm[kFRows];
  int32_t store[kFRows];
};

template <int D>
__global__ void __launch_bounds__(kFThreads) attn_f32(const __grid_constant__ AttnParams p) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  F32Smem<D>& sm = *reinterpret_cast<F32Smem<D>*>(smem_raw);
  int seq, qt, h;
  decode_work(p, blockIdx.x / kF32CtasPerTile, seq, qt, h);
  const int sub = blockIdx.x % kF32CtasPerTile;
  const SeqDesc sd = p.seq[seq];
  const int rows_seq = sd.n_orig + sd.slen;
  const int r0 = sd.q_start + qt * kBM + sub * kFRows;  // first (sequence-relative) query row
  if (r0 >= rows_seq) return;
  const int g = h / (p.hq / p.hkv);
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  const float* Q = static_cast<const float*>(p.q);
  const float* K = static_cast<const float*>(p.k);
  const float* V = static_cast<const float*>(p.v);

  // n rows of D floats, rows past the sequence as zeros
  auto copy_rows = [&](float* dst, int dst_pitch, const float* src, int heads, int head, int row, int n) {
#pragma unroll 4
    for (int i = tid; i < n * D / 4; i += kFThreads) {
      const int r = i / (D / 4), c = i % (D / 4);
      const bool in = row + r < rows_seq;
      const size_t off =
          (static_cast<size_t>(sd.row_base + (in ? row + r : 0)) * heads + head) * D + 4 * c;
      cp_async16(dst + r * dst_pitch + 4 * c, src + off, in ? 16 : 0);
    }
    cp_async_commit();
  };
  copy_rows(&sm.q[0][0], D + 4, Q, p.hq, h, r0, kFRows);
  load_block_info(p, sd, sm.bi, qt == 0 && h == 0 && sub == 0);
  grid_dep_wait();  // the RoPE key pass launched before this kernel (if any) is complete
  copy_rows(&sm.k[0][0], D + 4, K, p.hkv, g, 0, kFKeys);
  __syncthreads();
  if (tid < kFRows) {
    const RowInfo ri = row_info(sd, sm.bi, r0 + tid);
    sm.rm[tid] = row_masks(ri, sm.bi, sd);
    sm.store[tid] = ri.store;
  }
  if (p.rope) {  // RoPE of the query rows in shared memory, two threads per row
    cp_async_wait_all();
    __syncthreads();
    const int r = tid / 2;
    if (r0 + r < rows_seq) {
      const int pos = rope_position(p, sd, r0 + r);
      const bool half = p.rope_style == DARD_ROPE_HALF;
#pragma unroll 4
      for (int i = tid % 2; i < D / 2; i += 2) {
        float c, s;
        rope_cos_sin(pos, p.rope_f[2 * i], p.rope_f[2 * i + 1], c, s);
        float& a = sm.q[r][half ? i : 2 * i];
        float& b = sm.q[r][half ? i + D / 2 : 2 * i + 1];
        const float x = a, y = b;
        a = fmaf(x, c, -y * s);
        b = fmaf(x, s, y * c);
      }
    }
  }

  constexpr int kC = D / 64;  // 4-column groups of O per thread
  uint64_t acc[8][2 * kC];    // O as column pairs
  float m[8], l[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 2 * kC; ++c) acc[i][c] = 0;
  }
  const int n_kt = (rows_seq + kFKeys - 1) / kFKeys;
  for (int j = 0; j < n_kt; ++j) {
    const int kt0 = j * kFKeys;
    cp_async_wait_all();
    __syncthreads();  // K(j) (and Q) landed; P V of the tile before has read V and P
    copy_rows(&sm.v[0][0], D, V, p.hkv, g, kt0, kFKeys);
    // S: 32 values of d at a time, sums over even and odd d apart, then added up (short
    // chains: the rounding errors stay as small as with a sum split over several threads)
    float z[8][kNC];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < kNC; ++c) z[i][c] = 0.f;
#pragma unroll 1
    for (int d0 = 0; d0 < D; d0 += 32) {
      uint64_t s2[8][kNC];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < kNC; ++c) s2[i][c] = 0;
#pragma unroll 4
      for (int d = d0; d < d0 + 32; d += 4) {
        ulonglong2 kv[kNC];
#pragma unroll
        for (int c = 0; c < kNC; ++c)
          kv[c] = *reinterpret_cast<const ulonglong2*>(&sm.k[tx + 16 * c][d]);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const ulonglong2 qv = *reinterpret_cast<const ulonglong2*>(&sm.q[8 * i + ty][d]);
#pragma unroll
          for (int c = 0; c < kNC; ++c) {
            s2[i][c] = f2_fma(qv.x, kv[c].x, s2[i][c]);
            s2[i][c] = f2_fma(qv.y, kv[c].y, s2[i][c]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < kNC; ++c) {
          float a, b;
          f2_unpack(s2[i][c], a, b);
          z[i][c] += a + b;
        }
    }
    const bool masked = kt0 + kFKeys > sd.n_orig ||
                        (sd.blen > 0 && kt0 < sd.b0 + sd.blen && kt0 + kFKeys > sd.b0);
    float al[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
      for (int c = 0; c < kNC; ++c) z[i][c] *= p.scale;
      uint64_t vis = ~0ull;
      if (masked) {
        vis = vis64(sd, kt0, sm.rm[8 * i + ty]) >> tx;
#pragma unroll
        for (int c = 0; c < kNC; ++c) z[i][c] = ((vis >> (16 * c)) & 1ull) ? z[i][c] : -INFINITY;
      }
      float mt = z[i][0];
#pragma unroll
      for (int c = 1; c < kNC; ++c) mt = fmaxf(mt, z[i][c]);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, o));
      const float mn = fmaxf(m[i], mt);
      al[i] = m[i] == -INFINITY ? 0.f : (mn == m[i] ? 1.f : expf(m[i] - mn));
      m[i] = mn;
      const float ref = mn == -INFINITY ? 0.f : mn;
      float sum = 0.f;
#pragma unroll
      for (int c = 0; c < kNC; ++c) {
        // a key that the row does not see weighs -0, by which PV leaves it out
        const float w = !((vis >> (16 * c)) & 1ull) ? -0.f
                        : z[i][c] == -INFINITY      ? 0.f
                                                    : expf(z[i][c] - ref);
        sum += w;
        sm.p[8 * i + ty][tx + 16 * c] = w;
      }
      l[i] = l[i] * al[i] + sum;
    }
    cp_async_wait_all();
    __syncthreads();  // V(j) landed, P is stored, K(j) has been read
    if (j + 1 < n_kt) copy_rows(&sm.k[0][0], D + 4, K, p.hkv, g, kt0 + kFKeys, kFKeys);
    // the tile's P V apart, then added to O (short chains again)
    uint64_t part[8][2 * kC];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 2 * kC; ++c) part[i][c] = 0;
    const auto add_pv = [&](auto tile_masked) {
      constexpr bool kMasked = decltype(tile_masked)::value;
#pragma unroll 2
      for (int kk = 0; kk < kFKeys; kk += 4) {
        float4 pv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) pv[i] = *reinterpret_cast<const float4*>(&sm.p[8 * i + ty][kk]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          ulonglong2 vv[kC];
#pragma unroll
          for (int c = 0; c < kC; ++c)
            vv[c] = *reinterpret_cast<const ulonglong2*>(&sm.v[kk + u][4 * tx + 64 * c]);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float w = u == 0 ? pv[i].x : u == 1 ? pv[i].y : u == 2 ? pv[i].z : pv[i].w;
            // V of a key that the row does not see may hold anything, a NaN too
            if (kMasked && __float_as_int(w) == INT_MIN) continue;
            const uint64_t w2 = f2_pack(w, w);
#pragma unroll
            for (int c = 0; c < kC; ++c) {
              part[i][2 * c] = f2_fma(w2, vv[c].x, part[i][2 * c]);
              part[i][2 * c + 1] = f2_fma(w2, vv[c].y, part[i][2 * c + 1]);
            }
          }
        }
      }
    };
    if (masked) add_pv(std::true_type{});
    else add_pv(std::false_type{});
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 2 * kC; ++c)
        acc[i][c] = f2_fma(acc[i][c], f2_pack(al[i], al[i]), part[i][c]);
  }
  float* O = static_cast<float*>(p.o);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float sum = l[i];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const int row = 8 * i + ty;
    if (r0 + row >= rows_seq || !sm.store[row]) continue;
    const float inv = 1.0f / sum;
    float* out = O + (static_cast<size_t>(sd.row_base + r0 + row) * p.hq + h) * D + 4 * tx;
#pragma unroll
    for (int c = 0; c < kC; ++c) {
      float4 v;
      f2_unpack(acc[i][2 * c], v.x, v.y);
      f2_unpack(acc[i][2 * c + 1], v.z, v.w);
      v.x *= inv;
      v.y *= inv;
      v.z *= inv;
      v.w *= inv;
      *reinterpret_cast<float4*>(out + 64 * c) = v;
    }
  }
}

template <int D>
cudaError_t launch(const AttnParams& p, cudaStream_t stream) {
  static std::atomic<uint64_t> attr_done{0};
  const cudaError_t e = ensure_smem_attr(attn_f32<D>, sizeof(F32Smem<D>), attr_done);
  if (e != cudaSuccess) return e;
  const AttnLaunch L(p.total_work * kF32CtasPerTile, kFThreads, sizeof(F32Smem<D>), stream, 1, p.rope != 0);
  return cudaLaunchKernelEx(&L.cfg, attn_f32<D>, p);
}

}  // namespace

cudaError_t launch_f32_attention(const AttnParams& p, cudaStream_t stream) {
  return p.head_dim == 64 ? launch<64>(p, stream) : launch<128>(p, stream);
}

}  // namespace dard
