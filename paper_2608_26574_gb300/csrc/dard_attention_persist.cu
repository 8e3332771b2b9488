// dard_attention_persist.cu - state-masked attention of more than one wave of work items
// (bf16, tcgen05): the arithmetic and products of attn_tc2 (dard_attention.cu: the order of S
// and PV in the tensor pipe, P's own TMEM columns, the elected issue, the reference maximum),
// in persistent CTAs.
//
// attn_persist: one CTA per SM. A work item is one or two query tiles of 128 rows that share a
// sequence and a key/value head, so that every K/V tile serves up to 256 rows; how tiles make
// items is the launcher's choice (plan_items). 12 warps:
//   warps 4q .. 4q + 3  softmax and epilogue of the item's tile q, one thread per query row;
//   warp 8              TMA producer: the Q tiles, then K and V through 2 stages each;
//   warp 9              TMEM allocator and S issuer;
//   warp 10             PV issuer;
//   warp 11             decodes the CTA's items and gathers their block information into
//                       shared memory ahead of their users.
//   TMEM: the S buffer [0, 128), P_0, P_1 [128, 256), O_0, O_1 [256, 256 + 2D); at D = 64 a
//   second S buffer [384, 512), so that each tile has its own.
// Every role walks the CTA's items by itself: the producer and the S issuer run ahead into
// the next item while the softmax still finishes this one, so that an item's loads, its first
// products and the CTA's set-up hide behind the item before.
//
// Bound: the tensor pipe (2064 cycles of products per key tile and pair of tiles, about 2300 in
// the steady state); between items the softmax warps wait for the last PV (750 cycles) and
// store O (the stores of all SMs together run at L2's write rate). Against one CTA per item
// (attn_tc2, forced, the same build otherwise): 32 sequences of 500 to 2300 rows 811 -> 759 us,
// 8 of 1248 rows 173 -> 165 us, a GQA sequence of 5184 rows 217 -> 221 us; a launch of at most
// one item per SM has nothing to hide and its start is later (8B layer 15.4 -> 17.7 us): those
// stay with attn_tc1 and attn_tc2. (Single launches; back to back for seconds the board is at its
// power limit, and the first and the last take 845 and 243 us.)
//
// Tried and slower: the rows of a last V tile that belong to the next sequence cleared, so that a
// NaN there stays out (24 sequences of 264 rows 91.0 us, by the PV issuer 94.5, by warp 11 100.4);
// both tile slots on a lone query tile, every other key tile each, merged at the end (the loop's code got worse: GQA 221 -> 240 us, a lone-tile launch 14.7 -> 16.4 us);
// P stored and handed over in two halves (226 us); the exponentials in explicit batches of 16
// (239 us with the split above, as without batches); O stored by each row's own thread with
// 32-byte stores (ragged batch 790 -> 822 us).
#include <algorithm>

#include "dard_attn_common.cuh"

namespace dard {
namespace {

constexpr int kPersThreads = 384;  // 2 x 4 softmax warps, TMA producer, S and PV issuers, item decoder
constexpr int kQT = 2;    // query tiles per work item at most (one sequence and K/V head)
constexpr int kNK = 2;    // TMA stages for K
constexpr int kNV = 2;    // TMA stages for V
constexpr int kPvGo = 4;  // slots of the S-before-PV hand-off
constexpr int kItems = 3;  // decoded work items ahead
constexpr int kItemUsers = 4 * kQT + 3;  // softmax warps, producer, issuers
constexpr int kWProd = 4 * kQT;    // warp 8: TMA producer
constexpr int kWMma = kWProd + 1;  // warp 9: TMEM allocator and S issuer
constexpr int kWPv = kWProd + 2;   // warp 10: PV issuer
constexpr int kWItem = kWProd + 3;  // warp 11: item decoder
// Register split (setmaxnreg): the launch gives 384 threads 168 registers each; the
// warpgroup of warps 8-11 (producer, issuers, decoder) drops to 40 and the two softmax
// warpgroups rise to 232, so that a thread holds its row's 128 scores and 64 words of
// weights at once: 128 x 40 + 256 x 232 = 384 x 168.
constexpr uint32_t kPersLaunchRegs = 168, kPersSideRegs = 40, kPersSoftmaxRegs = 232;
static_assert(128 * kPersSideRegs + 256 * kPersSoftmaxRegs == kPersThreads * kPersLaunchRegs,
              "the register shares must add up to the launch's registers");
static_assert(kPersThreads * kPersLaunchRegs <= 65536, "one CTA per SM");

// P = 2^(s * sl - mL) of keys 64 hh .. 64 hh + 63 of the row's scores as bf16 pairs, and their
// sum: of the rounded values, so that the output is a convex combination of V rows with exactly
// the weights the PV product uses.
template <int hh>
__device__ __forceinline__ void tile_row_exp(const uint32_t (&sv)[128], uint64_t sl2,
                                             uint64_t nmL2, uint64_t (&acc)[4],
                                             uint32_t (&pk)[32]) {
#pragma unroll
  for (int e = 0; e < 32; ++e) {
    float x0, x1;
    f2_unpack(f2_fma(f2_pack(__uint_as_float(sv[64 * hh + 2 * e]),
                             __uint_as_float(sv[64 * hh + 2 * e + 1])), sl2, nmL2), x0, x1);
    pk[e] = pack_bf16x2(ex2_approx(x0), ex2_approx(x1));
    acc[e & 3] = f2_add(acc[e & 3], f2_pack(__uint_as_float(pk[e] << 16),
                                            __uint_as_float(pk[e] & 0xffff0000u)));
  }
}

// One work item: nq query tiles, tile q being rows [r[q], r[q] + 128) of head h[q] against key
// tiles [0, nk[q]), and its sequence's layout. nq = 0 ends the CTA's items.
struct __align__(16) TcItem {
  SeqDesc sd;
  int32_t g, nq, first;  // first: the sequence's first item (reports bad states once)
  int32_t r[kQT], h[kQT], nk[kQT], n_kt;  // n_kt: the larger of nk
};

// Barrier protocol. Every barrier completes one phase per use, counted over the CTA's items;
// use u of a ring of r waits for parity (u / r) & 1, and no waiter is ever two phases behind
// (the parity would alias): each wait for use u is preceded, in the same thread or through a
// chain of waits, by the completion of use u - r. Below, n counts a tile slot's key tiles
// over the items.
struct __align__(16) PersistCtl {
  uint64_t item_full[kItems], item_empty[kItems];
  uint64_t bi_full[kItems];  // the item's block information is there
  uint64_t q_full[kQT];   // the item's query tile q landed
  uint64_t q_rot[kQT];    // RoPE: the softmax warps of tile q rotated it in shared memory
  uint64_t q_empty[kQT];  // the item's last S_q completed: the next Q tile may land
  uint64_t k_full[kNK], k_empty[kNK], v_full[kNV], v_empty[kNV];
  uint64_t s_full[kQT];   // S_q(n) landed in TMEM
  uint64_t s_free[kQT];   // per S buffer: the softmax read the scores into registers
  uint64_t p_full[kQT];   // the softmax of tile q stored P_q(n) (and, on an item's first key
                          // tile, has read the item before out of O_q)
  // S_q(n + 1) has been issued: PV_q(n) may follow it into the pipe. A ring, since S runs
  // ahead: S_q(n + 4) is only issued once the softmax has read S_q(n + 2) (its buffer, or one
  // before it in turn), so has stored P_q(n + 1), which waits for PV_q(n): the issuer of PV
  // has taken its slot before the slot's next use.
  uint64_t pv_go[kQT][kPvGo];
  uint64_t pv_done[kQT];  // PV_q(n) completed: P_q(n + 1) may replace P_q(n), and after an item's
                          // last key tile O_q is final
  uint64_t drained;       // every product both issuers launched has completed (two commits)
  uint32_t tmem_base;
  TcItem item[kItems];
  BlockInfo bi[kItems];   // the block of each item's sequence
  RowMasks rm[kQT][kBM];  // each row's masks, read on the tiles that need them
  uint4 stage[4 * kQT][128];  // epilogue: 32 rows x 32 columns of each softmax warp
};

template <int D>
constexpr size_t persist_smem_bytes() {
  // alignment slack + kQT query tiles + kNK K stages + kNV V stages (128 rows each) + control
  return 1024 + (kQT + kNK + kNV) * static_cast<size_t>(kTN) * D * 2 + sizeof(PersistCtl);
}

__device__ __forceinline__ void flag_timeout(const AttnParams& p) {
  if (p.status) atomicOr(p.status, DARD_STATUS_TIMEOUT);
}

// n / d for 0 <= n < 2^31 by the host's ceil(2^64 / d) (0 for d = 1).
__device__ __forceinline__ int div_by(int n, uint64_t magic) {
  return magic == 0 ? n : static_cast<int>(__umul64hi(static_cast<uint64_t>(n), magic));
}

// The CTA's k-th item (rows of the grid in alternating direction: sequences are ordered
// longest first, so that the CTAs' shares come out even); nq = 0 after the last.
__device__ __forceinline__ TcItem tc_item(const AttnParams& p, int k) {
  TcItem it{};
  const int grid = static_cast<int>(gridDim.x), b = static_cast<int>(blockIdx.x);
  const long long w64 = static_cast<long long>(k) * grid + ((k & 1) ? grid - 1 - b : b);
  if (w64 >= p.total_items) return it;
  const int w = static_cast<int>(w64);
  int lo = 0, hi = p.num_seqs;  // item_prefix[lo] <= w < item_prefix[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (p.item_prefix[mid] <= w) lo = mid; else hi = mid;
  }
  const int seq = p.num_seqs == 1 ? 0 : p.order[lo];  // (spares a cold parameter read)
  const SeqDesc sd = p.seq[seq];
  const int rows = sd.n_orig + sd.slen;
  const int local = lo == 0 ? w : w - p.item_prefix[lo];
  it.sd = sd;
  it.first = local == 0;
  int nq, r0, r1, nk0, nk1;
  if (p.by_group) {
    // units (query tile, head of the group), head minor; an item takes two of them
    const int group = p.group;
    const int i = div_by(local, p.div_hkv), g = local - i * p.hkv, u = i * kQT;
    const int t0 = div_by(u, p.div_group), t1 = div_by(u + 1, p.div_group);
    nq = min(kQT, sd.n_qtiles * group - u);
    r0 = sd.q_start + t0 * kBM;
    r1 = sd.q_start + t1 * kBM;
    it.g = g;
    it.h[0] = g * group + u - t0 * group;
    it.h[1] = g * group + u + 1 - t1 * group;
    nk0 = key_tiles(sd, r0, min(r0 + kBM, rows));  // tiles of shadow keys only are skipped
    nk1 = nq > 1 ? key_tiles(sd, r1, min(r1 + kBM, rows)) : 0;
  } else {
    // two consecutive query tiles of one head, both against the key tiles of their rows
    const int i = div_by(local, p.div_hq), h = local - i * p.hq;
    nq = min(kQT, sd.n_qtiles - i * kQT);
    r0 = sd.q_start + i * (kQT * kBM);
    r1 = r0 + kBM;
    it.g = div_by(h, p.div_group);
    it.h[0] = it.h[1] = h;
    nk0 = key_tiles(sd, r0, min(r0 + nq * kBM, rows));
    nk1 = nq > 1 ? nk0 : 0;
  }
  it.nq = nq;
  it.r[0] = r0;
  it.r[1] = r1;
  it.nk[0] = nk0;
  it.nk[1] = nk1;
  it.n_kt = max(nk0, nk1);
  return it;
}

// kRope: the launch applies RoPE to the query tiles (a separate instantiation, so that the
// kernel without RoPE keeps its register allocation).
template <int D, bool kRope>
__global__ void __launch_bounds__(kPersThreads, 1)
    attn_persist(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tmq,
            const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv) {
  constexpr int kSub = D / 64;                   // 128-byte (64 x bf16) column blocks
  constexpr uint32_t kKSub = kTN * 128;          // one 128-row x 128-byte swizzled block
  constexpr uint32_t kTileBytes = kSub * kKSub;  // one 128-row tile of Q, K or V
  constexpr bool kOneX = D == 128;               // one S buffer in TMEM for both tiles
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sQ = base;                     // kQT query tiles
  uint8_t* sK = sQ + kQT * kTileBytes;    // kNK stages
  uint8_t* sV = sK + kNK * kTileBytes;    // kNV stages
  PersistCtl& ctl = *reinterpret_cast<PersistCtl*>(sV + kNV * kTileBytes);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const long long wlim = p.wait_cycles > 0 ? p.wait_cycles : kWaitCycles;

  // K or V tile j of an item into its stage (use: counted over the items)
  auto load_kv = [&](const TcItem& t, int j, int use, bool k_or_v) {
    const int b = use % (k_or_v ? kNK : kNV);
    uint64_t* bar = k_or_v ? &ctl.k_full[b] : &ctl.v_full[b];
    uint8_t* dst = (k_or_v ? sK : sV) + b * kTileBytes;
    const void* map = k_or_v ? static_cast<const void*>(&tmk) : static_cast<const void*>(&tmv);
    mbar_arrive_expect_tx(bar, kTileBytes);
    if (k_or_v && j == p.test_drop_kv) return;  // test hook: this K copy is never issued
    const int row0 = t.sd.row_base;
#pragma unroll
    for (int s = 0; s < kSub; ++s)
      tma_load_2d(dst + s * kKSub, map, bar, t.g * D + s * 64, row0 + j * kTN);
  };
  auto load_q = [&](const TcItem& t, int q) {
    mbar_arrive_expect_tx(&ctl.q_full[q], kTileBytes);
    const int row = t.sd.row_base + t.r[q], col = t.h[q] * D;
#pragma unroll
    for (int s = 0; s < kSub; ++s)
      tma_load_2d(sQ + q * kTileBytes + s * kKSub, &tmq, &ctl.q_full[q], col + s * 64, row);
  };
  // The producer lane initialises the barriers and issues Q0 and K0; the other threads touch
  // the barriers only after the block sync.
  TcItem first;
  if (warp == kWProd || warp == kWItem) first = tc_item(p, 0);
  if (warp == kWProd && lane == 0) {
    // Q0 and K0 only, and before the other barriers: the first S product needs nothing else,
    // and with every CTA of the launch starting at once they land sooner alone (the rest
    // follows in the producer)
    mbar_init(&ctl.q_full[0], 1);
    mbar_init(&ctl.k_full[0], 1);
    fence_barrier_init();
    load_q(first, 0);
    grid_dep_wait();  // the RoPE key pass launched before this kernel (if any) is complete
    load_kv(first, 0, 0, true);
    for (int i = 0; i < kItems; ++i) {
      mbar_init(&ctl.item_full[i], 1);
      mbar_init(&ctl.item_empty[i], kItemUsers);
      mbar_init(&ctl.bi_full[i], 1);
    }
    for (int q = 0; q < kQT; ++q) {
      if (q > 0) mbar_init(&ctl.q_full[q], 1);
      mbar_init(&ctl.q_rot[q], 4);  // the tile's softmax warps
      mbar_init(&ctl.q_empty[q], 1);
      mbar_init(&ctl.s_full[q], 1);
      mbar_init(&ctl.s_free[q], 4);
      mbar_init(&ctl.p_full[q], 4);
      for (int b = 0; b < kPvGo; ++b) mbar_init(&ctl.pv_go[q][b], 1);
      mbar_init(&ctl.pv_done[q], 1);
    }
    for (int b = 0; b < kNK; ++b) {
      if (b > 0) mbar_init(&ctl.k_full[b], 1);
      mbar_init(&ctl.k_empty[b], 1);
    }
    for (int b = 0; b < kNV; ++b) {
      mbar_init(&ctl.v_full[b], 1);
      mbar_init(&ctl.v_empty[b], 1);
    }
    mbar_init(&ctl.drained, 2);
    fence_barrier_init();
    tma_prefetch_desc(&tmv);
  }
  if (warp == kWMma) {
    tmem_alloc<kTmemCols>(&ctl.tmem_base);
    tmem_relinquish();
  }
  if (warp == kWItem && lane == 0) ctl.item[0] = first;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tX0 = ctl.tmem_base;
  const uint32_t tP0 = ctl.tmem_base + kTN;
  const uint32_t tO0 = ctl.tmem_base + 2 * kTN;
  auto s_buf = [&](int q) { return tX0 + (!kOneX && q != 0 ? 3 * kTN : 0); };

  // The CTA's k-th item for one of its users; `done_with` returns the slot.
  auto item_at = [&](int k, bool& ok) -> const TcItem& {
    // (the first item has been there since the block sync)
    ok = k == 0 || mbar_wait(&ctl.item_full[k % kItems], (k / kItems) & 1, wlim);
    return ctl.item[k % kItems];
  };
  auto done_with = [&](int k) { mbar_arrive(&ctl.item_empty[k % kItems]); };

  // The register split: each branch below starts with its warpgroup's setmaxnreg (warps 8-11
  // give registers up, the softmax warps 0-7 take them), so that it covers the branch's code.
  if (warp == kWProd) {
    // ------------------------------------------------------------ TMA producer
    reg_dealloc<kPersSideRegs>();
    if (lane == 0) {
      int uk = 1, uv = 0, dropped = -1;  // K and V uses issued; the last use the test hook dropped
      int iq0 = 1, iq1 = 0;              // Q tiles issued per slot
      if (p.test_drop_kv == 0) dropped = 0;
      // the other first loads once Q0 and K0 have landed
      bool ok = mbar_wait(&ctl.q_full[0], 0, wlim) && mbar_wait(&ctl.k_full[0], 0, wlim);
      for (int k = 0; ok; ++k) {
        const TcItem& it = item_at(k, ok);
        if (!ok || it.nq == 0) break;
        const int n_kt = it.n_kt;
        for (int j = 0; j < n_kt && ok; ++j) {
          if (k > 0 || j > 0) {
            ok = uk < kNK || mbar_wait(&ctl.k_empty[uk % kNK], (uk / kNK - 1) & 1, wlim);
            if (!ok) break;
            if (j == p.test_drop_kv) dropped = uk;
            load_kv(it, j, uk++, true);
          }
          if (j == 0) {
            if (k > 0) {
              ok = mbar_wait(&ctl.q_empty[0], (iq0 - 1) & 1, wlim);
              if (!ok) break;
              load_q(it, 0);
              ++iq0;
            }
            if (it.nq > 1) {
              ok = iq1 == 0 || mbar_wait(&ctl.q_empty[1], (iq1 - 1) & 1, wlim);
              if (!ok) break;
              load_q(it, 1);
              ++iq1;
            }
          }
          ok = uv < kNV || mbar_wait(&ctl.v_empty[uv % kNV], (uv / kNV - 1) & 1, wlim);
          if (!ok) break;
          load_kv(it, j, uv++, false);
        }
        done_with(k);
      }
      if (!ok) flag_timeout(p);
      // Every copy issued lands before shared memory is released (after a normal run they all
      // have: the waits return at once): the latest use of each stage (earlier uses landed
      // before their stage was reused). A copy the test hook dropped was never issued.
      for (int u = max(0, uk - kNK); u < uk; ++u)
        if (u != dropped) mbar_wait(&ctl.k_full[u % kNK], (u / kNK) & 1, wlim);
      for (int u = max(0, uv - kNV); u < uv; ++u)
        mbar_wait(&ctl.v_full[u % kNV], (u / kNV) & 1, wlim);
      mbar_wait(&ctl.q_full[0], (iq0 - 1) & 1, wlim);
      if (iq1 > 0) mbar_wait(&ctl.q_full[1], (iq1 - 1) & 1, wlim);
    }
  } else if (warp == kWMma) {
    // ------------------------------------------------------------ S issuer
    reg_dealloc<kPersSideRegs>();
    // S_q(j) = Q_q K(j)^T once K(j) has landed and the softmax has read the scores that the
    // buffer held out of it. The whole warp runs the loop and an elected lane issues:
    // descriptors and addresses then stay in uniform registers, where the instruction wants
    // them (in a one-lane branch each MMA took about 100 cycles to issue, more than the 64
    // that it runs). The PV products come from a second warp, whose waits between products
    // then hide behind this one's products and the other way round.
    constexpr uint32_t kIdS = idesc_bf16_f32(kBM, kTN, 0, 0);
    const uint64_t dq = smem_desc_sw128(smem_u32(sQ), 16, 1024);
    const uint64_t dk = smem_desc_sw128(smem_u32(sK), 16, 1024);
    bool ok = true;
    int uk = 0;               // K uses
    int us0 = 0, us1 = 0;     // S products per buffer (one buffer: all in us0)
    int go0 = 0, go1 = 0;     // hand-offs to the PV issuer per slot
    int iq0 = 0, iq1 = 0;     // items per slot
    auto issue = [&](int q, int j, int nk, int& us, int& go, int& iq, uint64_t db) {
      if (j == 0) {
        if (!warp_wait(kRope ? &ctl.q_rot[q] : &ctl.q_full[q], iq & 1, wlim)) return false;
        ++iq;
      }
      if (us > 0 && !warp_wait(&ctl.s_free[kOneX ? 0 : q], (us - 1) & 1, wlim)) return false;
      ++us;
      tc_fence_after();
      const uint64_t da = dq + q * (kTileBytes >> 4);
      const uint32_t td = s_buf(q);
      if (elect_one()) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t off = ((ks >> 2) * kKSub + (ks & 3) * 32) >> 4;
          mma_ss(td, da + off, db + off, kIdS, ks > 0);
        }
        mma_commit(&ctl.s_full[q]);
        if (j > 0) mbar_arrive(&ctl.pv_go[q][go % kPvGo]);  // PV_q(j - 1) may follow
        if (j == nk - 1) mma_commit(&ctl.q_empty[q]);
      }
      __syncwarp();
      go += j > 0 ? 1 : 0;
      return true;
    };
#pragma unroll 1
    for (int k = 0; ok; ++k) {
      const TcItem& it = item_at(k, ok);
      ok = __all_sync(0xffffffffu, ok);
      const int nk0 = __shfl_sync(0xffffffffu, it.nk[0], 0), nk1 = __shfl_sync(0xffffffffu, it.nk[1], 0), n_kt = max(nk0, nk1), nq = __shfl_sync(0xffffffffu, it.nq, 0);
      __syncwarp();
      if (ok && lane == 0) done_with(k);
      if (!ok || nq == 0) break;
#pragma unroll 1
      for (int j = 0; j < n_kt && ok; ++j, ++uk) {
        ok = warp_wait(&ctl.k_full[uk % kNK], (uk / kNK) & 1, wlim);
        const uint64_t db = dk + (uk % kNK) * (kTileBytes >> 4);
        if (ok && j < nk0) ok = issue(0, j, nk0, us0, go0, iq0, db);
        if (ok && j < nk1) ok = issue(1, j, nk1, kOneX ? us0 : us1, go1, iq1, db);
        if (ok && elect_one()) mma_commit(&ctl.k_empty[uk % kNK]);
        __syncwarp();
      }
    }
    if (!ok && lane == 0) flag_timeout(p);
    if (elect_one()) mma_commit(&ctl.drained);  // completes once every S product issued has
    __syncwarp();
  } else if (warp == kWPv) {
    // ------------------------------------------------------------ PV issuer
    reg_dealloc<kPersSideRegs>();
    // O_q += P_q(j) V(j) once V(j) has landed, the softmax of tile q has stored P_q(j) and
    // S_q(j + 1) is in the pipe.
    constexpr uint32_t kIdO = idesc_bf16_f32(kBM, D, 0, 1);
    const uint64_t dv = smem_desc_sw128(smem_u32(sV), kKSub, 1024);
    bool ok = true;
    int uv = 0;            // V uses
    int n0 = 0, n1 = 0;    // PV products per slot
    int go0 = 0, go1 = 0;  // hand-offs taken per slot
    auto issue = [&](int q, int j, int nk, int& n, int& go, uint64_t db) {
      if (!warp_wait(&ctl.p_full[q], n & 1, wlim)) return false;
      ++n;
      if (j < nk - 1) {
        if (!warp_wait(&ctl.pv_go[q][go % kPvGo], (go / kPvGo) & 1, wlim)) return false;
        ++go;
      }
      tc_fence_after();
      const uint32_t td = tO0 + q * D, ta = tP0 + q * 64;
      if (elect_one()) {
#pragma unroll
        for (int ks = 0; ks < kTN / 16; ++ks)
          mma_ts(td, ta + ks * 8, db + ks * (2048 >> 4), kIdO, (j > 0 || ks > 0) ? 1u : 0u);
        mma_commit(&ctl.pv_done[q]);
      }
      __syncwarp();
      return true;
    };
#pragma unroll 1
    for (int k = 0; ok; ++k) {
      const TcItem& it = item_at(k, ok);
      ok = __all_sync(0xffffffffu, ok);
      const int nk0 = __shfl_sync(0xffffffffu, it.nk[0], 0), nk1 = __shfl_sync(0xffffffffu, it.nk[1], 0), n_kt = max(nk0, nk1), nq = __shfl_sync(0xffffffffu, it.nq, 0);
      __syncwarp();
      if (ok && lane == 0) done_with(k);
      if (!ok || nq == 0) break;
#pragma unroll 1
      for (int j = 0; j < n_kt && ok; ++j, ++uv) {
        ok = warp_wait(&ctl.v_full[uv % kNV], (uv / kNV) & 1, wlim);
        const uint64_t db = dv + (uv % kNV) * (kTileBytes >> 4);
        if (ok && j < nk0) ok = issue(0, j, nk0, n0, go0, db);
        if (ok && j < nk1) ok = issue(1, j, nk1, n1, go1, db);
        if (ok && elect_one()) mma_commit(&ctl.v_empty[uv % kNV]);
        __syncwarp();
      }
    }
    if (!ok && lane == 0) flag_timeout(p);
    if (elect_one()) mma_commit(&ctl.drained);  // completes once every PV product issued has
    __syncwarp();
  } else if (warp < kWProd) {
    // ------------------------------------------------------------ softmax + epilogue
    // Warps 4q .. 4q + 3 own tile slot q; thread t = query row t of the tile (TMEM lane t).
    reg_alloc<kPersSoftmaxRegs>();
    const int q = warp >> 2, quarter = warp & 3;
    const int t = quarter * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t tX = s_buf(q) + lane_off, tP = tP0 + q * 64 + lane_off, tO = tO0 + q * D + lane_off;
    const float sl = p.scale_log2;
    const uint64_t sl2 = f2_pack(sl, sl);
    int n = 0;        // key tiles of this slot
    int iq = 0;       // items of this slot
    bool ok = true;
#pragma unroll 1
    for (int k = 0; ok; ++k) {
      const TcItem& it = item_at(k, ok);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok || it.nq == 0) break;
      if (q >= it.nq) {
        __syncwarp();
        if (lane == 0) done_with(k);
        continue;
      }
      const SeqDesc& sd = it.sd;
      const BlockInfo& bi = ctl.bi[k % kItems];
      const int n_kt = __shfl_sync(0xffffffffu, it.nk[q], 0);
      if (kRope) {
        // RoPE of this thread's query row in shared memory, before the first S product reads it
        ok = mbar_wait(&ctl.q_full[q], iq & 1, wlim);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        const int r = it.r[q] + t;
        if (r < sd.n_orig + sd.slen) rope_tile_row<D>(p, sQ + q * kTileBytes, t, rope_position(p, sd, r));
        fence_proxy_async_smem();  // the generic-proxy writes, before the MMAs read the tile
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl.q_rot[q]);
      }
      bool have_rm = false;  // ctl.rm[q][t] holds this row's masks
      float ref = -INFINITY, l_run = 0.f;  // the row's reference in powers of two, its sum
      // the key tiles that need the mask (tile_needs_mask): those of the block, [jb0, jb1), and
      // those from jm on
      const int jb0 = sd.b0 / kTN, jb1 = sd.blen > 0 ? (sd.b0 + sd.blen + kTN - 1) / kTN : 0;
      const int jm = sd.n_orig / kTN;
      bool fresh = true;  // some row of the warp has seen no finite score
#pragma unroll 1
      for (int j = 0; j < n_kt; ++j) {
        ok = mbar_wait(&ctl.s_full[q], n & 1, wlim);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        tc_fence_after();
        // the tile's 128 scores of this row in registers
        uint32_t sv[128];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          tmem_ld32(tX + 32 * c, *reinterpret_cast<uint32_t(*)[32]>(sv + 32 * c));
        tmem_wait_ld();
        // the buffer may take the next S product
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl.s_free[kOneX ? 0 : q]);
        if (j >= jm || (j >= jb0 && j < jb1)) {
          if (!have_rm) {
            ok = mbar_wait(&ctl.bi_full[k % kItems], (k / kItems) & 1, wlim);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            ctl.rm[q][t] = row_masks(row_info(sd, bi, it.r[q] + t), bi, sd);
            have_rm = true;
          }
          mask_row(vis64(sd, j * kTN, ctl.rm[q][t]), vis64(sd, j * kTN + 64, ctl.rm[q][t]), sv);
        }
        // The tile's weights against the reference so far, the maximum of the row's first tile
        // with a finite score. Only where their sum comes out at kRescaleMax or more, and before
        // the first finite score, is the maximum formed and the reference raised beyond it, the
        // weights are computed (again) and O is rescaled.
        float ls = 0.f, alpha = 1.f;
        uint32_t pk[32], pk1[32];
        bool rescale = false;
        bool raise = fresh, over = false;  // over: the second pass, for rows whose sum was
#pragma unroll 1
        while (true) {
          if (raise) {
            const float top = tile_row_max(sv) * sl;
            fresh = __any_sync(0xffffffffu, ref == -INFINITY && top == -INFINITY);
            if (ref == -INFINITY) {
              ref = top;
            } else if (!(ls < kRescaleMax) && top > ref) {  // (no other row matters)
              rescale = true;
              alpha = ex2_approx(ref - (top + kRaiseRoom));
              ref = top + kRaiseRoom;
            }
          }
          const float mL = ref == -INFINITY ? 0.f : ref;
          const uint64_t nmL2 = f2_pack(-mL, -mL);
          uint64_t acc[4] = {0, 0, 0, 0};  // bit pattern 0 = +0.0f
          tile_row_exp<0>(sv, sl2, nmL2, acc, pk);
          tile_row_exp<1>(sv, sl2, nmL2, acc, pk1);
          float a0, a1, b0, b1;
          f2_unpack(f2_add(acc[0], acc[1]), a0, a1);
          f2_unpack(f2_add(acc[2], acc[3]), b0, b1);
          ls = (a0 + a1) + (b0 + b1);
          if (over || !__any_sync(0xffffffffu, !(ls < kRescaleMax))) break;
          raise = over = true;
        }
        // P_q(n) replaces P_q(n - 1), and O_q may be rescaled, once PV_q(n - 1) has completed
        // (an item's first tile: waited for at the end of the item before)
        if (j > 0) ok = mbar_wait(&ctl.pv_done[q], (n - 1) & 1, wlim);
        ++n;
        tc_fence_after();
        if (__any_sync(0xffffffffu, !ok || rescale)) {
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
#pragma unroll 1
          for (int c = 0; c < D / 32 && j > 0; ++c) {
            uint32_t o[32];
            tmem_ld32(tO + 32 * c, o);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st32(tO + 32 * c, o);
          }
        }
        tmem_st32(tP, pk);
        tmem_st32(tP + 32, pk1);
        l_run = fmaf(l_run, alpha, ls);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&ctl.p_full[q]);
      }
      if (ok) ok = mbar_wait(&ctl.pv_done[q], (n - 1) & 1, wlim) &&
                   mbar_wait(&ctl.bi_full[k % kItems], (k / kItems) & 1, wlim);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      ++iq;
      tc_fence_after();
      // O row / row sum -> bf16, 32 columns at a time through the warp's own 2 KB of shared
      // memory (16-byte chunks XOR-swizzled), so that a store instruction writes 64
      // contiguous bytes of eight rows; no other warp is waited for.
      const float inv_l = 1.0f / l_run;
      // rows of the call's output (not past the sequence's end, no invalid shadow row)
      const uint32_t rows_out =
          __ballot_sync(0xffffffffu, row_info(sd, bi, it.r[q] + t).store != 0);
      uint4* stage = ctl.stage[warp];
      __nv_bfloat16* out = static_cast<__nv_bfloat16*>(p.o) +
                           (static_cast<size_t>(sd.row_base + it.r[q] + quarter * 32) * p.hq +
                            it.h[q]) * D;
      const size_t pitch = static_cast<size_t>(p.hq) * D;
      // before the stores, which an arrival would wait for
      __syncwarp();
      if (lane == 0) done_with(k);
      uint32_t rr[D];
#pragma unroll
      for (int c = 0; c < D / 32; ++c)
        tmem_ld32(tO + 32 * c, *reinterpret_cast<uint32_t(*)[32]>(rr + 32 * c));
      tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            w[e] = pack_bf16x2(__uint_as_float(rr[32 * c + 8 * v + 2 * e]) * inv_l,
                               __uint_as_float(rr[32 * c + 8 * v + 2 * e + 1]) * inv_l);
          stage[4 * lane + (v ^ ((lane >> 1) & 3))] = make_uint4(w[0], w[1], w[2], w[3]);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = 8 * i + (lane >> 2), v = lane & 3;
          const uint4 u = stage[4 * row + (v ^ ((row >> 1) & 3))];
          if ((rows_out >> row) & 1u)
            *reinterpret_cast<uint4*>(out + row * pitch + 32 * c + 8 * v) = u;
        }
        __syncwarp();
      }
      // the reads of O come before the first P_q of the next item, which lets PV_q write O
      tc_fence_before();
    }
    if (!ok && lane == 0) flag_timeout(p);
  } else {
    // ------------------------------------------------------------ item decoder
    // One warp decodes the items (searches and cold parameter reads, about 1000 cycles) and
    // gathers their block information (about 1500) ahead of the others.
    reg_dealloc<kPersSideRegs>();
    bool ok = true;
#pragma unroll 1
    for (int k = 0; ok; ++k) {
      const int b = k % kItems;
      ok = k < kItems || warp_wait(&ctl.item_empty[b], (k / kItems - 1) & 1, wlim);
      if (!ok) break;
      TcItem it = first;
      if (k > 0) {
        it = tc_item(p, k);
        if (lane == 0) ctl.item[b] = it;  // (the first is there: its users do not wait)
      }
      if (lane == 0) mbar_arrive(&ctl.item_full[b]);
      if (it.nq == 0) break;
      publish_block_info_warp(p, it.sd, ctl.bi[b], it.first);
      if (lane == 0) mbar_arrive(&ctl.bi_full[b]);
      __syncwarp();
    }
    if (!ok && lane == 0) flag_timeout(p);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWMma) {
    // no product is still writing TMEM (both issuers committed `drained` last)
    if (lane == 0 && !mbar_wait(&ctl.drained, 0, wlim)) flag_timeout(p);
    __syncwarp();
    tc_fence_after();
    tmem_dealloc<kTmemCols>(ctl.tmem_base);
  }
}

// ---------------------------------------------------------------- host side

template <int D, bool kRope>
cudaError_t launch(const AttnParams& p, cudaStream_t stream) {
  static std::atomic<uint64_t> attr_done{0};
  static std::atomic<int> regs{0};
  CUtensorMap mq, mk, mv;
  if (!make_map(&mq, p.q, p.hq, D, p.total_rows, kBM) ||
      !make_map(&mk, p.k, p.hkv, D, p.total_rows, kTN) ||
      !make_map(&mv, p.v, p.hkv, D, p.total_rows, kTN))
    return cudaErrorInvalidValue;
  const size_t smem = persist_smem_bytes<D>();
  cudaError_t e = check_launch_regs(attn_persist<D, kRope>, kPersLaunchRegs, regs);
  if (e == cudaSuccess) e = ensure_smem_attr(attn_persist<D, kRope>, smem, attr_done);
  if (e != cudaSuccess) return e;
  const AttnLaunch L(persist_ctas(p), kPersThreads, smem, stream, 1, kRope);
  return cudaLaunchKernelEx(&L.cfg, attn_persist<D, kRope>, p, mq, mk, mv);
}

}  // namespace

void plan_items(AttnParams& p, bool by_group) {
  const auto magic = [](int d) { return d == 1 ? 0ull : ~0ull / static_cast<uint64_t>(d) + 1; };
  p.group = p.hq / p.hkv;
  p.div_hq = magic(p.hq);
  p.div_hkv = magic(p.hkv);
  p.div_group = magic(p.group);
  p.by_group = by_group;
  long long items = 0;
  for (int r = 0; r < p.num_seqs; ++r) {
    p.item_prefix[r] = static_cast<int32_t>(items);
    const long long tiles = p.seq[p.order[r]].n_qtiles;
    items += by_group ? (tiles * p.group + kQT - 1) / kQT * p.hkv : (tiles + kQT - 1) / kQT * p.hq;
  }
  p.item_prefix[p.num_seqs] = static_cast<int32_t>(items);
  p.total_items = static_cast<int32_t>(items);
}

int persist_ctas(const AttnParams& p) { return std::min(p.total_items, sm_count()); }

cudaError_t launch_persist_attention(const AttnParams& p, cudaStream_t stream) {
  if (p.head_dim == 64) return p.rope ? launch<64, true>(p, stream) : launch<64, false>(p, stream);
  return p.rope ? launch<128, true>(p, stream) : launch<128, false>(p, stream);
}

}  // namespace dard
