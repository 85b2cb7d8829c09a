// Fused runs by direct addressing (Sec. II.D.2: the branches that agree on
// every bit a run does not write form a coherent group, and the run acts on
// each group by itself).
//
// When few key bits vary over a state, a branch's group and its place in the
// group can be addressed instead of sorted for: the varying bits, packed with
// the run's targets lowest, number a slot, the group a range of 2^k slots.
//   k_slot_scatter  applies the queued operations and stores every branch's
//                   amplitude at its slot, with a presence byte: no sort, no
//                   counters, no atomics.
//   k_slot_run      takes areas of whole groups (up to 2^12 slots) into shared
//                   memory and applies the run's items one after another:
//                   interference steps and phases.  Per step the pairs with a
//                   member present and the controls met are listed first (one
//                   ballot per 32 pairs of presence bits), pairs of two members
//                   apart from single ones, so that every lane of the FP64
//                   sequence holds a pair that acts; survivors are appended to
//                   the dense output.
// Each step evaluates children() with the presence flags of its pair and
// prunes with keep_amp(), so the result is that of the steps one by one, bit
// for bit.  Because a pair's full key is known from its slot, a step may read
// (controls, angle register, table address) the targets of other steps of the
// run and a target may come again, which the sorted form (sqs_group.cu) does
// not allow.
//
// What bounds it: FP64 issue of the rotations (12 FP64 instructions a pair and
// register-valued step) while the areas hold branches, latency of a step's two
// barriers while they do not; DRAM is idle.  Measured, rotations with their
// loads and unloads as one step included: an N = 1024 walk step (0.9 M branches
// on average, 98 steps) 8.4 -> 1.7 ms, three steps of an N = 128 walk in
// non-Hermitian form 10.4 -> 1.6 ms, two of 64 systems batched 13.5 -> 2.0 ms,
// readout included, where partition and pair took 73 us a step at 10^6 branches
// and 15 us at the smallest.
#include <cuda_runtime.h>
#include <stdint.h>

#include "sqs_device.cuh"
#include "sqs_internal.h"

namespace sqs {
namespace {

constexpr int kRunThreads = 512;
constexpr uint32_t kAreaLog2Max = 12;
static_assert(kMaxRun <= (int)kAreaLog2Max, "a group fits the area");

// The slot of key k (bits moved run by run), and the key of a slot.
template <class K>
__device__ __forceinline__ uint32_t slot_of(const SlotMap& m, K k) {
  const uint64_t w0 = lo64(k), w1 = hi64(k);
  uint32_t s = 0;
#pragma unroll 1
  for (uint32_t i = 0; i < m.n; ++i) {
    const BitMove v = m.mv[i];
    const uint64_t w = v.src < 64 ? w0 : w1;
    s |= ((uint32_t)(w >> (v.src & 63u)) & ((1u << v.len) - 1u)) << v.dst;
  }
  return s;
}
template <int KW>
__device__ __forceinline__ typename KT<KW>::T key_of(const SlotMap& m, uint32_t s) {
  uint64_t w0 = m.base[0], w1 = m.base[1];
#pragma unroll 1
  for (uint32_t i = 0; i < m.n; ++i) {
    const BitMove v = m.mv[i];
    const uint64_t f = (uint64_t)((s >> v.dst) & ((1u << v.len) - 1u)) << (v.src & 63u);
    if (KW == 1 || v.src < 64)
      w0 |= f;
    else
      w1 |= f;
  }
  return mk<KW>(w0, w1);
}

constexpr int kScatterILP = 4;

template <int KW, class AT, class LT>
__global__ void __launch_bounds__(kStreamThreads)
    k_slot_scatter(Ctl* ctl, Arr in, int in_slot, const __grid_constant__ LT ops,
                   const __grid_constant__ SlotMap map, AT* amp, uint8_t* pres) {
  typedef typename KT<KW>::T K;
  __shared__ AT tab[LT::kTab];
  __shared__ DevOp sops[LT::kOps];
  __shared__ uint16_t ulist[kStreamThreads];
  __shared__ unsigned int n_ulist;
  pdl_next();
  load_ops(ops, sops, tab);
  pdl_wait();
  if (ctl->err) return;
  const uint64_t n_dense = ctl->cnt[in_slot];
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(&ctl->peak, n_dense);
  for_units(in, n_dense, kScatterILP * blockDim.x, ulist, &n_ulist,
            [&](uint64_t base, uint32_t lim) {
    K k[kScatterILP];
    AT v[kScatterILP];
    bool live[kScatterILP];
#pragma unroll
    for (int q = 0; q < kScatterILP; ++q) {
      const uint32_t j = q * blockDim.x + threadIdx.x;
      live[q] = j < lim;
      k[q] = 0;
      v[q].x = v[q].y = 0;
      if (live[q]) {
        k[q] = ld_key<KW>(in, base + j);
        v[q] = ((const AT*)in.amp)[base + j];
      }
    }
    if (ops.n) apply_ops_n<KW, AT, kScatterILP>(ops.n, sops, tab, k, v, live);
#pragma unroll
    for (int q = 0; q < kScatterILP; ++q) {
      if (live[q]) {
        const uint32_t s = slot_of(map, k[q]);
        amp[s] = v[q];
        pres[s] = 1;
      }
    }
  });
}

// Shared state of a CTA that runs items over an area of slots.  Dynamic: the
// area's amplitudes, then
//   pres   presence bits, 32 slots a word
//   wbase  survivors before each presence word (emission)
//   list   u16 per pair: pairs of two members from the front, single ones
//          from the back
template <class AT>
__host__ __device__ constexpr size_t run_smem_bytes(uint32_t area_log2) {
  return ((size_t)sizeof(AT) << area_log2) + ((size_t)8 << (area_log2 - 5)) +
         ((size_t)2 << (area_log2 - 1));
}
template <class AT>
struct Area {
  uint32_t log2;
  AT* amp;
  uint32_t *pres, *wbase;
  uint16_t* list;
  __device__ Area(unsigned char* smem, uint32_t area_log2) : log2(area_log2) {
    amp = (AT*)smem;
    pres = (uint32_t*)(smem + ((size_t)sizeof(AT) << area_log2));
    wbase = pres + (1u << (area_log2 - 5));
    list = (uint16_t*)(wbase + (1u << (area_log2 - 5)));
  }
};
struct RunShared {
  unsigned int lc[2][2];  // list counters: [parity][two members, single]
  unsigned int stage[kMaxItems];
  unsigned int wsum[4];
  unsigned long long base_out;
  unsigned int last, next, dead;
};

// Applies the run's items to the area, one after another.  keys.ok(it, s)
// tells whether item it acts on slot s, a present one or the other of its pair
// (its predicate; the same for both), keys.key(s) the key of slot s.  Called by the whole CTA with the
// area's amplitudes and presence bits written and a barrier passed; returns
// past a barrier.
template <int KW, class AT, class Keys>
__device__ __forceinline__ void run_items(const RunProg& prog, const Area<AT>& A, RunShared& sh,
                                          uint32_t& par, const Keys& keys) {
  const uint32_t area = 1u << A.log2, npairs = area >> 1, nwords = area >> 5;
  AT* const amp = A.amp;
  uint32_t* const pres = A.pres;
  uint16_t* const list = A.list;
  const uint32_t lane = threadIdx.x & 31u;
  const unsigned int lt = (1u << lane) - 1u;
  for (uint32_t i = 0; i < prog.n; ++i) {
    const RunItem& it = prog.it[i];
    if (it.phase) {
      AT f;
      to_amp(f, make_double2(it.g.u[0], it.g.u[1]));
      for (uint32_t s = threadIdx.x; s < area; s += blockDim.x)
        if (((pres[s >> 5] >> (s & 31u)) & 1u) && keys.ok(it, s)) amp[s] = cmul(amp[s], f);
      __syncthreads();
      continue;
    }
    const Gate1& g = it.g;
    const uint32_t low = (1u << it.j) - 1u;
    // The pairs that act.  (npairs is a multiple of 32: whole warps.)
    for (uint32_t p = threadIdx.x; p < npairs; p += blockDim.x) {
      const uint32_t s0 = ((p & ~low) << 1) | (p & low), s1 = s0 | (1u << it.j);
      const unsigned int h0 = (pres[s0 >> 5] >> (s0 & 31u)) & 1u;
      const unsigned int h1 = (pres[s1 >> 5] >> (s1 & 31u)) & 1u;
      const bool act = (h0 | h1) && keys.ok(it, s0);
      const unsigned int b2 = __ballot_sync(0xffffffffu, act && (h0 & h1));
      const unsigned int b1 = __ballot_sync(0xffffffffu, act && !(h0 & h1));
      if (b1 | b2) {
        unsigned int at2 = 0, at1 = 0;
        if (lane == 0) {
          if (b2) at2 = atomicAdd(&sh.lc[par][0], (unsigned int)__popc(b2));
          if (b1) at1 = atomicAdd(&sh.lc[par][1], (unsigned int)__popc(b1));
        }
        at2 = __shfl_sync(0xffffffffu, at2, 0);
        at1 = __shfl_sync(0xffffffffu, at1, 0);
        if ((b2 >> lane) & 1u) list[at2 + __popc(b2 & lt)] = (uint16_t)p;
        if ((b1 >> lane) & 1u) list[npairs - 1u - (at1 + __popc(b1 & lt))] = (uint16_t)p;
      }
    }
    __syncthreads();
    const uint32_t n2 = sh.lc[par][0], n1 = sh.lc[par][1];
    par ^= 1u;
    if (threadIdx.x < 2) sh.lc[par][threadIdx.x] = 0u;  // the next step's
    const uint32_t n2w = (n2 + 31u) & ~31u;
    for (uint32_t q = threadIdx.x; q < n2w + n1; q += blockDim.x) {
      const bool two = q < n2;
      if (!two && q < n2w) continue;
      const uint32_t p = two ? list[q] : list[npairs - 1u - (q - n2w)];
      const uint32_t s0 = ((p & ~low) << 1) | (p & low), s1 = s0 | (1u << it.j);
      const uint32_t m0 = 1u << (s0 & 31u), m1 = 1u << (s1 & 31u);
      const uint64_t av = g.mode == 1 ? angle_value(g, keys.key(s0)) : 0ull;
      bool h0 = true, h1 = true;
      AT o0, o1;
      if (two) {
        children<AT>(g, av, true, amp[s0], true, amp[s1], o0, o1);
      } else {
        h0 = (pres[s0 >> 5] & m0) != 0u;
        h1 = !h0;
        const AT a = amp[h0 ? s0 : s1];
        if (h0)
          children<AT>(g, av, true, a, false, a, o0, o1);
        else
          children<AT>(g, av, false, a, true, a, o0, o1);
      }
      const bool k0 = keep_amp(o0, g.eps, g.epsf, g.eps2);
      const bool k1 = keep_amp(o1, g.eps, g.epsf, g.eps2);
      amp[s0] = o0;
      amp[s1] = o1;
      if (k0 != h0) atomicXor(&pres[s0 >> 5], m0);
      if (k1 != h1) atomicXor(&pres[s1 >> 5], m1);
    }
    __syncthreads();
    // Branches after the step (the words change again only after the next
    // step's list barrier).
    if (threadIdx.x < nwords) {
      unsigned int c = __popc(pres[threadIdx.x]);
      for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      if (lane == 0 && c) atomicAdd(&sh.stage[i], c);
    }
  }
}

// Appends the area's survivors to the dense output; ends with a barrier.
template <int KW, class AT, class Keys>
__device__ __forceinline__ void emit_area(Ctl* ctl, const Area<AT>& A, RunShared& sh,
                                          const Keys& keys, const Arr& out, int out_slot,
                                          uint32_t seq) {
  const uint32_t area = 1u << A.log2, nwords = area >> 5;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  unsigned int c = 0, incl = 0;
  if (threadIdx.x < nwords) {
    c = incl = __popc(A.pres[threadIdx.x]);
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    if (lane == 31) sh.wsum[warp] = incl;
  }
  __syncthreads();
  if (threadIdx.x < nwords) {
    unsigned int before = incl - c;
    for (uint32_t w = 0; w < warp; ++w) before += sh.wsum[w];
    A.wbase[threadIdx.x] = before;
    if (threadIdx.x == nwords - 1u) {
      const unsigned int sum = before + c;
      sh.base_out = sum ? atomicAdd(&ctl->cnt[out_slot], (unsigned long long)sum) : 0ull;
      if (sum && sh.base_out + sum > out.cap)
        raise_err(ctl, kErrCapacity, seq, sh.base_out + sum);
    }
  }
  __syncthreads();
  const unsigned long long ob = sh.base_out;
#pragma unroll 2
  for (uint32_t s = threadIdx.x; s < area; s += blockDim.x) {
    const uint32_t w = A.pres[s >> 5];
    if ((w >> lane) & 1u) {  // s & 31 == lane
      const uint64_t pos = ob + A.wbase[s >> 5] + __popc(w & lt);
      if (pos < out.cap) {
        st_key<KW>(out, pos, keys.key(s));
        ((AT*)out.amp)[pos] = A.amp[s];
      }
    }
  }
  __syncthreads();  // the area is reused
}

// The counts after each step; the last CTA raises the peak and clears them
// (and the work counter) for the next run.
__device__ __forceinline__ void finish_run(Ctl* ctl, const RunProg& prog, RunShared& sh) {
  for (uint32_t i = threadIdx.x; i < prog.n; i += blockDim.x)
    if (sh.stage[i]) atomicAdd(&ctl->stage[i], (unsigned long long)sh.stage[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) sh.last = atomicAdd(&ctl->run_done, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (sh.last) {
    __threadfence();
    for (uint32_t i = threadIdx.x; i < prog.n; i += blockDim.x) {
      const unsigned long long v = atomicExch(&ctl->stage[i], 0ull);
      if (v) atomicMax(&ctl->peak, v);
    }
    if (threadIdx.x == 0) ctl->run_done = ctl->run_next = 0u;
  }
}

__device__ __forceinline__ void begin_run(Ctl* ctl, RunShared& sh, int out_slot) {
  pdl_next();
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->cnt[(out_slot + 1) & 3] = 0;
  for (uint32_t i = threadIdx.x; i < kMaxItems; i += blockDim.x) sh.stage[i] = 0u;
  if (threadIdx.x < 4) sh.lc[threadIdx.x >> 1][threadIdx.x & 1u] = 0u;
  // Work is drawn one piece at a time (the next index while the current piece
  // is processed): branches cluster in some areas, and with a fixed share per
  // CTA half the SMs idled (a 64-system walk batch: 580 us a run).
  if (threadIdx.x == 0) {
    sh.next = atomicAdd(&ctl->run_next, 1u);
    sh.dead = ctl->err;  // one answer for the CTA: another may raise an error any time
  }
  __syncthreads();
}

// Slots of an addressed run: predicates are masks of the slot number.
template <int KW>
struct SlotKeys {
  const SlotMap& map;
  uint32_t first;  // slot of the area's slot 0
  __device__ __forceinline__ bool ok(const RunItem& it, uint32_t s) const {
    return ((first + s) & it.smask) == it.sval;
  }
  __device__ __forceinline__ typename KT<KW>::T key(uint32_t s) const {
    return key_of<KW>(map, first + s);
  }
};

template <int KW, class AT>
__global__ void __launch_bounds__(kRunThreads, 2)
    k_slot_run(Ctl* ctl, AT* gamp, uint8_t* gpres, const __grid_constant__ SlotMap map,
               const __grid_constant__ RunProg prog, Arr out, int out_slot, uint32_t seq) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RunShared sh;
  const Area<AT> A(smem, prog.area_log2);
  const uint32_t area = 1u << prog.area_log2;
  uint32_t par = 0;
  begin_run(ctl, sh, out_slot);
  // After an error the presence bytes are still cleared: they are zero between
  // runs.
  const bool dead = sh.dead != 0u;
  for (uint32_t b = sh.next; b < prog.n_areas; b = sh.next) {
    uint32_t drawn = 0u;
    if (threadIdx.x == 0) drawn = atomicAdd(&ctl->run_next, 1u);
    const uint32_t s0g = b << prog.area_log2;  // first slot of the area
    // Presence bytes to bits (16 slots a thread), cleared behind.
    bool some = false;
    if (threadIdx.x < area / 16u) {
      uint4* const src = (uint4*)(gpres + s0g) + threadIdx.x;
      const uint4 v = *src;
      unsigned int m = 0u;
      if (v.x | v.y | v.z | v.w) {
        // Bytes are 0 or 1: the multiply gathers a word's four into its top nibble.
        m = ((v.x * 0x10204080u) >> 28) | (((v.y * 0x10204080u) >> 28) << 4) |
            (((v.z * 0x10204080u) >> 28) << 8) | (((v.w * 0x10204080u) >> 28) << 12);
        *src = make_uint4(0u, 0u, 0u, 0u);
        some = true;
      }
      ((uint16_t*)A.pres)[threadIdx.x] = (uint16_t)m;
    }
    const bool empty = !__syncthreads_or(some);  // every thread has read `next`
    if (threadIdx.x == 0) sh.next = drawn;
    __syncthreads();
    if (empty || dead) continue;
#pragma unroll 4
    for (uint32_t s = threadIdx.x; s < area; s += blockDim.x)
      if ((A.pres[s >> 5] >> (s & 31u)) & 1u) A.amp[s] = gamp[s0g + s];
    __syncthreads();
    const SlotKeys<KW> keys{map, s0g};
    run_items<KW, AT>(prog, A, sh, par, keys);
    emit_area<KW, AT>(ctl, A, sh, keys, out, out_slot, seq);
  }
  finish_run(ctl, prog, sh);
}

// ---------------------------------------------------------------------------
// Bucketed runs: where too many key bits vary to address slots, k_partition
// scatters the branches by a hash of the key with the run's few targets
// cleared, so that every group (at most 2^kMaxHashRun branches) lies in one
// bucket.  k_bucket_run numbers a bucket's groups through an open-addressing
// table in shared memory (over the amplitude area, which is free then), lays
// batches of them out as 2^k slots each and runs the items as above.  A round
// of the QRAM workload (4 rotations and their inverses on 2^20 two-word
// branches, 2^24 in between) took 8 partitions and 8 pair launches, 3.6 ms;
// the state in between now never leaves shared memory.
constexpr uint32_t kBucketCap = 2048;
constexpr uint32_t kBucketTable = 2 * kBucketCap;
constexpr uint32_t kBucketAreaLog2 = 12;

template <int KW, class AT>
struct BucketSmem {
  typedef typename KT<KW>::T K;
  static constexpr size_t key_off = run_smem_bytes<AT>(kBucketAreaLog2);
  static constexpr size_t gid_off = key_off + kBucketCap * sizeof(K);
  static constexpr size_t rep_off = gid_off + kBucketCap * 2;
  static constexpr size_t bytes = rep_off + kBucketCap * 2;
  static_assert(kBucketTable * 4 <= (sizeof(AT) << kBucketAreaLog2), "the table fits the area");
  static_assert(bytes <= 112u * 1024u, "two CTAs per SM");
};

// Slots of a batch of groups: slot (group, index) with the group's first
// branch as its representative.
template <int KW>
struct GroupKeys {
  typedef typename KT<KW>::T K;
  const SlotMap& map;  // moves between the k index bits and the key
  const K* skey;
  const uint16_t* rep;  // of the batch's groups
  uint32_t k;
  K tmask;
  __device__ __forceinline__ K rest(uint32_t s) const { return skey[rep[s >> k]] & ~tmask; }
  __device__ __forceinline__ bool ok(const RunItem& it, uint32_t s) const {
    if ((s & it.smask) != it.sval) return false;
    if ((it.rmask[0] | it.rmask[1]) == 0ull) return true;
    return (rest(s) & mk<KW>(it.rmask[0], it.rmask[1])) == mk<KW>(it.rval[0], it.rval[1]);
  }
  __device__ __forceinline__ K key(uint32_t s) const {
    return rest(s) | key_of<KW>(map, s & ((1u << k) - 1u));
  }
};

template <int KW, class AT>
__global__ void __launch_bounds__(kRunThreads, 2)
    k_bucket_run(Ctl* ctl, Arr bk, const __grid_constant__ SlotMap map,
                 const __grid_constant__ RunProg prog, uint32_t k, uint64_t tm0, uint64_t tm1,
                 Arr out, int out_slot, uint32_t seq) {
  typedef typename KT<KW>::T K;
  typedef BucketSmem<KW, AT> L;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ RunShared sh;
  __shared__ unsigned int n_groups;
  const Area<AT> A(smem, kBucketAreaLog2);
  K* const skey = (K*)(smem + L::key_off);
  uint16_t* const gid = (uint16_t*)(smem + L::gid_off);
  uint16_t* const rep = (uint16_t*)(smem + L::rep_off);
  unsigned int* const slot = (unsigned int*)smem;  // over the area
  const K tmask = mk<KW>(tm0, tm1);
  const uint32_t per_batch = 1u << (kBucketAreaLog2 - k);
  uint32_t par = 0;
  begin_run(ctl, sh, out_slot);
  const uint32_t nb = sh.dead ? 0u : ctl->buckets;
  for (uint32_t b = sh.next; b < nb; b = sh.next) {
    uint32_t drawn = 0u;
    if (threadIdx.x == 0) {
      drawn = atomicAdd(&ctl->run_next, 1u);
      n_groups = 0u;
    }
    unsigned int* const bcnt = &bk.seg_cnt[(uint64_t)b << kBucketCntLog2];
    const uint32_t cnt = *bcnt;
    const uint32_t n = cnt > kBucketCap ? 0u : cnt;  // overflow: flagged by the partition
    const uint64_t base = (uint64_t)b << bk.seg_log2;
    // 1. Keys, and the group of every branch: first its representative (the
    //    branch that claimed the group's table slot), then the group's number.
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) skey[i] = ld_key<KW>(bk, base + i);
    for (uint32_t i = threadIdx.x; i < kBucketTable; i += blockDim.x) slot[i] = 0u;
    __syncthreads();
    if (threadIdx.x == 0) {
      sh.next = drawn;
      *bcnt = 0u;  // the bucket is clean for the next use
    }
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
      const K p = skey[i] & ~tmask;
      uint32_t h = (uint32_t)khash(p) & (kBucketTable - 1u);
      // n <= half the table: a free slot or the group is found within it.
      for (uint32_t probe = 0; probe < kBucketTable; ++probe) {
        const unsigned int old = atomicCAS(&slot[h], 0u, i + 1u);
        if (old == 0u) {
          const unsigned int id = atomicAdd(&n_groups, 1u);
          rep[id] = (uint16_t)i;
          break;
        }
        if ((skey[old - 1u] & ~tmask) == p) break;
        h = (h + 1u) & (kBucketTable - 1u);
      }
      gid[i] = (uint16_t)h;  // the group's table slot
    }
    __syncthreads();
    const uint32_t G = n_groups;
    // Table slot -> group number (a slot holds its representative).
    for (uint32_t q = threadIdx.x; q < G; q += blockDim.x) {
      const K p = skey[rep[q]] & ~tmask;
      uint32_t h = (uint32_t)khash(p) & (kBucketTable - 1u);
      while (slot[h] != (unsigned int)rep[q] + 1u) h = (h + 1u) & (kBucketTable - 1u);
      slot[h] = (q << 16) | 0x8000u;  // no branch index: read as a number below
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) gid[i] = (uint16_t)(slot[gid[i]] >> 16);
    __syncthreads();
    // 2. Batches of whole groups.
    for (uint32_t g0 = 0; g0 < G; g0 += per_batch) {
      const uint32_t gn = G - g0 < per_batch ? G - g0 : per_batch;
      for (uint32_t w = threadIdx.x; w < (1u << (kBucketAreaLog2 - 5)); w += blockDim.x)
        A.pres[w] = 0u;
      __syncthreads();
      for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        const uint32_t q = (uint32_t)gid[i] - g0;  // wraps below the batch
        if (q < gn) {
          const uint32_t s = (q << k) | slot_of(map, skey[i]);
          A.amp[s] = ((const AT*)bk.amp)[base + i];
          atomicOr(&A.pres[s >> 5], 1u << (s & 31u));
        }
      }
      __syncthreads();
      const GroupKeys<KW> keys{map, skey, rep + g0, k, tmask};
      run_items<KW, AT>(prog, A, sh, par, keys);
      emit_area<KW, AT>(ctl, A, sh, keys, out, out_slot, seq);
    }
    if (G == 0) __syncthreads();  // every thread has left the shared state
  }
  finish_run(ctl, prog, sh);
}

template <int KW, class AT>
cudaError_t scatter_t(const Launch& L, Ctl* ctl, Arr in, int in_slot, const OpList& ops,
                      const SlotMap& map, void* amp, uint8_t* pres) {
  const uint64_t per = (uint64_t)kScatterILP * kStreamThreads;
  uint64_t grid = (L.n_hint + per - 1) / per;
  const uint64_t cap = (uint64_t)L.sm_count * 8;
  grid = grid < 1 ? 1 : (grid > cap ? cap : grid);
  if (!fits_small(ops))
    return launch_next(k_slot_scatter<KW, AT, OpList>, grid, kStreamThreads, 0, L.stream, ctl, in,
                       in_slot, ops, map, (AT*)amp, pres);
  OpListSmall s;
  copy_small(ops, s);
  return launch_next(k_slot_scatter<KW, AT, OpListSmall>, grid, kStreamThreads, 0, L.stream, ctl,
                     in, in_slot, s, map, (AT*)amp, pres);
}

template <int KW, class AT>
cudaError_t run_t(const Launch& L, Ctl* ctl, void* amp, uint8_t* pres, const SlotMap& map,
                  const RunProg& prog, Arr out, int out_slot) {
  static std::atomic<unsigned long long> configured{0};  // opt-in above 48 KB, per device
  cudaError_t e = ensure_smem_optin((const void*)k_slot_run<KW, AT>,
                                    run_smem_bytes<AT>(kAreaLog2Max), configured);
  if (e != cudaSuccess) return e;
  const uint32_t wave = (uint32_t)L.sm_count * 2u;
  const uint32_t grid = prog.n_areas < wave ? prog.n_areas : wave;
  return launch_next(k_slot_run<KW, AT>, grid, kRunThreads, run_smem_bytes<AT>(prog.area_log2),
                     L.stream, ctl, (AT*)amp, pres, map, prog, out, out_slot, L.seq);
}

template <int KW, class AT>
cudaError_t bucket_t(const Launch& L, Ctl* ctl, Arr bk, const SlotMap& map, const RunProg& prog,
                     uint32_t k, const uint64_t tmask[2], Arr out, int out_slot) {
  static std::atomic<unsigned long long> configured{0};  // opt-in above 48 KB, per device
  const size_t smem = BucketSmem<KW, AT>::bytes;
  cudaError_t e = ensure_smem_optin((const void*)k_bucket_run<KW, AT>, smem, configured);
  if (e != cudaSuccess) return e;
  const uint32_t wave = (uint32_t)L.sm_count * 2u;
  const uint32_t grid = bk.n_seg < wave ? bk.n_seg : wave;
  return launch_next(k_bucket_run<KW, AT>, grid ? grid : 1u, kRunThreads, smem, L.stream, ctl, bk,
                     map, prog, k, tmask[0], tmask[1], out, out_slot, L.seq);
}

}  // namespace

cudaError_t launch_bucket_run(const Launch& L, int kw, bool amp32, Ctl* ctl, Arr bk,
                              const SlotMap& map, const RunProg& prog, uint32_t k,
                              const uint64_t tmask[2], Arr out, int out_slot) {
  if (prog.n > (uint32_t)kMaxItems || k > (uint32_t)kMaxHashRun ||
      (1u << bk.seg_log2) != kBucketCap)
    return cudaErrorInvalidValue;
  if (kw == 2)
    return amp32 ? bucket_t<2, float2>(L, ctl, bk, map, prog, k, tmask, out, out_slot)
                 : bucket_t<2, double2>(L, ctl, bk, map, prog, k, tmask, out, out_slot);
  return amp32 ? bucket_t<1, float2>(L, ctl, bk, map, prog, k, tmask, out, out_slot)
               : bucket_t<1, double2>(L, ctl, bk, map, prog, k, tmask, out, out_slot);
}

cudaError_t launch_slot_scatter(const Launch& L, int kw, bool amp32, Ctl* ctl, Arr in, int in_slot,
                                const OpList& ops, const SlotMap& map, void* amp, uint8_t* pres) {
  if (kw == 2)
    return amp32 ? scatter_t<2, float2>(L, ctl, in, in_slot, ops, map, amp, pres)
                 : scatter_t<2, double2>(L, ctl, in, in_slot, ops, map, amp, pres);
  return amp32 ? scatter_t<1, float2>(L, ctl, in, in_slot, ops, map, amp, pres)
               : scatter_t<1, double2>(L, ctl, in, in_slot, ops, map, amp, pres);
}

// Slots per shared-memory area: one group, at least 2^10 slots (a full block's
// work per step).  More groups to an area mean fewer barriers, but also fewer
// areas to balance over the SMs: a 64-system walk batch spends 191 us a run
// with 2^12 slots, 149 us with the smallest areas, the N = 1024 walk the same.
uint32_t run_area_log2(uint32_t k) { return k > 10u ? k : 10u; }

cudaError_t launch_slot_run(const Launch& L, int kw, bool amp32, Ctl* ctl, void* amp,
                            uint8_t* pres, const SlotMap& map, const RunProg& prog, Arr out,
                            int out_slot) {
  if (prog.n > (uint32_t)kMaxItems || prog.area_log2 > kAreaLog2Max || prog.area_log2 < 10u)
    return cudaErrorInvalidValue;
  if (kw == 2)
    return amp32 ? run_t<2, float2>(L, ctl, amp, pres, map, prog, out, out_slot)
                 : run_t<2, double2>(L, ctl, amp, pres, map, prog, out, out_slot);
  return amp32 ? run_t<1, float2>(L, ctl, amp, pres, map, prog, out, out_slot)
               : run_t<1, double2>(L, ctl, amp, pres, map, prog, out, out_slot);
}

}  // namespace sqs
