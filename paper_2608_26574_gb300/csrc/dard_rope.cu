// dard_rope.cu - the RoPE pass over the key rows of an attention call (rope_theta > 0).
//
// Every key row is read by every query tile of its sequence and every query head of its
// group, so the keys are rotated once here, into k_rope, rather than in each CTA that loads
// them; the attention kernel launched next on the stream waits for this grid
// (griddepcontrol) before its first key load, and rotates its own query tiles as it loads
// them. Positions and arithmetic: dard_rope.cuh.
//
// One thread per (row, group of eight frequencies, four heads): the eight cos/sin pairs are
// formed once, while the thread's loads are in flight, and applied to its elements of each of
// its heads. Interleaved pairing: a group is 16 consecutive elements; half pairing: eight
// elements of the first half and the eight D/2 later. All loads and stores are 16 bytes.
// Bound: memory (each key row read and written once).
#include <cuda_bf16.h>

#include "dard_ptx.cuh"
#include "dard_rope.cuh"

namespace dard {
namespace {

constexpr int kRopeThreads = 256;
constexpr int kRopeHeads = 4;  // heads per thread

// Sequence of global row `row` (rows are stored sequence after sequence).
__device__ __forceinline__ int seq_of_row(const AttnParams& p, int row) {
  int lo = 0, hi = p.num_seqs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.seq[mid].row_base <= row) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void rot(float& a, float& b, float c, float s) {
  const float x = a, y = b;
  a = fmaf(x, c, -y * s);
  b = fmaf(x, s, y * c);
}

// Eight values of T as 16-byte vectors, to and from floats.
template <typename T>
struct Eight {
  static constexpr int kVecs = 8 * sizeof(T) / 16;
  uint4 u[kVecs];
  __device__ void load(const T* p) {
#pragma unroll
    for (int k = 0; k < kVecs; ++k) u[k] = reinterpret_cast<const uint4*>(p)[k];
  }
  __device__ void store(T* p) const {
#pragma unroll
    for (int k = 0; k < kVecs; ++k) reinterpret_cast<uint4*>(p)[k] = u[k];
  }
  __device__ void get(float (&x)[8]) const {
    const uint32_t* w = &u[0].x;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if constexpr (sizeof(T) == 2) x[e] = (e & 1) ? bf_hi(w[e / 2]) : bf_lo(w[e / 2]);
      else x[e] = __uint_as_float(w[e]);
    }
  }
  __device__ void set(const float (&x)[8]) {
    uint32_t* w = &u[0].x;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if constexpr (sizeof(T) == 2) {
        if (e & 1) w[e / 2] = bf_pack(x[e - 1], x[e]);
      } else {
        w[e] = __float_as_uint(x[e]);
      }
    }
  }
};

template <typename T, int D>
__global__ void __launch_bounds__(kRopeThreads) rope_keys(const __grid_constant__ AttnParams p) {
  grid_dep_launch();  // the attention kernel may be scheduled; it waits for this grid's end
  constexpr int kGroups = D / 16;  // groups of eight frequencies per row
  const int hblocks = (p.hkv + kRopeHeads - 1) / kRopeHeads;
  const long long idx = static_cast<long long>(blockIdx.x) * kRopeThreads + threadIdx.x;
  const long long total = static_cast<long long>(p.total_rows) * hblocks * kGroups;
  if (idx >= total) return;
  const int grp = static_cast<int>(idx % kGroups);
  const long long rest = idx / kGroups;
  const int hb = static_cast<int>(rest % hblocks);
  const int row = static_cast<int>(rest / hblocks);
  const bool half = p.rope_style == DARD_ROPE_HALF;
  // element offsets of the group within a head: [e0, e0 + 8) and [e1, e1 + 8)
  const int e0 = half ? 8 * grp : 16 * grp;
  const int e1 = half ? D / 2 + 8 * grp : 16 * grp + 8;
  const T* src = static_cast<const T*>(p.k_src);
  T* dst = static_cast<T*>(const_cast<void*>(p.k));
  const int h0 = hb * kRopeHeads;
  // every head's loads first (they are independent), then the rotations and the stores
  Eight<T> u0[kRopeHeads], u1[kRopeHeads];
#pragma unroll
  for (int hh = 0; hh < kRopeHeads; ++hh) {
    if (h0 + hh >= p.hkv) break;
    const size_t base = (static_cast<size_t>(row) * p.hkv + h0 + hh) * D;
    u0[hh].load(src + base + e0);
    u1[hh].load(src + base + e1);
  }
  // the angles while the loads are in flight
  const SeqDesc& sd = p.seq[seq_of_row(p, row)];
  const int pos = rope_position(p, sd, row - sd.row_base);
  float c[8], s[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int i = 8 * grp + e;  // frequency index
    rope_cos_sin(pos, p.rope_f[2 * i], p.rope_f[2 * i + 1], c[e], s[e]);
  }
#pragma unroll
  for (int hh = 0; hh < kRopeHeads; ++hh) {
    if (h0 + hh >= p.hkv) break;
    float x[8], y[8];
    u0[hh].get(x);
    u1[hh].get(y);
    if (half) {
#pragma unroll
      for (int e = 0; e < 8; ++e) rot(x[e], y[e], c[e], s[e]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        rot(x[2 * e], x[2 * e + 1], c[e], s[e]);
        rot(y[2 * e], y[2 * e + 1], c[4 + e], s[4 + e]);
      }
    }
    u0[hh].set(x);
    u1[hh].set(y);
    const size_t base = (static_cast<size_t>(row) * p.hkv + h0 + hh) * D;
    u0[hh].store(dst + base + e0);
    u1[hh].store(dst + base + e1);
  }
}

template <typename T>
cudaError_t launch_typed(const AttnParams& p, cudaStream_t stream) {
  const long long hblocks = (p.hkv + kRopeHeads - 1) / kRopeHeads;
  const long long threads = static_cast<long long>(p.total_rows) * hblocks * (p.head_dim / 16);
  const long long blocks = (threads + kRopeThreads - 1) / kRopeThreads;
  if (blocks < 1) return cudaSuccess;
  if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
  if (p.head_dim == 64)
    rope_keys<T, 64><<<static_cast<unsigned>(blocks), kRopeThreads, 0, stream>>>(p);
  else
    rope_keys<T, 128><<<static_cast<unsigned>(blocks), kRopeThreads, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rope_keys(const AttnParams& p, int dtype, cudaStream_t stream) {
  return dtype == DARD_BF16 ? launch_typed<__nv_bfloat16>(p, stream)
                            : launch_typed<float>(p, stream);
}

}  // namespace dard
