// Long runs of queued operations in place, on bit planes (Sec. II.D.1).
//
// Branch by branch a run is bound by integer issue: a controlled X is about
// eight instructions a branch, an addition fourteen, and over few branches each
// operation is 0.2 us of latency.  Here a thread takes 32 branches and turns
// their keys into planes -- bit i of plane b is bit b of branch i -- in its own
// column of shared memory, where an operation treats all 32 at once: a Toffoli
// is three loads, one logic instruction and one store, an addition a ripple over
// the field's planes, a phase one plane of each factor index.  No thread touches
// another's column, so there is no barrier inside a run.  The 32x32 bit
// transposition is done in registers (256 instructions a key word and way, 8 a
// branch); the branches of a thread lie a block apart, so that every load and
// store of keys and amplitudes is coalesced.  Bit for bit the results of
// apply_ops: the same table entry multiplies each amplitude.
//
// What bounds it now is FP64 issue of the factors (four instructions a branch and
// table) where a list has them, the way into planes and back where it has not.
// Measured, 2^24 branches of one 32-bit key, branch by branch against planes: 90
// X, CNOT and Toffoli 630 -> 163 us, 90 additions and swaps 1669 -> 283, 90 mixed
// with phases (three lists) 1390 -> 873; sizes and lists for which it is taken:
// planes_pay in sqs_api.cu.
//
// (Planes spread over the lanes of a warp were slower than branch by branch: an
// AND over the lanes costs two issue slots of the SM's one reduction unit.)
#include <cuda_runtime.h>
#include <stdint.h>

#include "sqs_device.cuh"
#include "sqs_internal.h"

namespace sqs {
namespace {

constexpr int kPlaneThreads = 128;
constexpr uint32_t kPlaneTile = 32u * kPlaneThreads;  // branches per CTA and round

// Bits d of the two indices exchanged, d = 4, 2, 1.
template <int D>
__device__ __forceinline__ void transpose_bits(uint32_t (&a)[32]) {
  constexpr uint32_t m = D == 4 ? 0x0f0f0f0fu : D == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    if (k & D) continue;
    const uint32_t x = a[k], y = a[k + D];
    a[k] = (x & m) | ((y << D) & ~m);
    a[k + D] = ((x >> D) & m) | (y & ~m);
  }
}

// a[i] bit p <-> a[p] bit i.
__device__ __forceinline__ void transpose32(uint32_t (&a)[32]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint32_t x = a[k], y = a[k + 16];
    a[k] = __byte_perm(x, y, 0x5410u);
    a[k + 16] = __byte_perm(x, y, 0x7632u);
  }
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    if (k & 8) continue;
    const uint32_t x = a[k], y = a[k + 8];
    a[k] = __byte_perm(x, y, 0x6240u);
    a[k + 8] = __byte_perm(x, y, 0x7351u);
  }
  transpose_bits<4>(a);
  transpose_bits<2>(a);
  transpose_bits<1>(a);
}

// 32-bit word v of the keys.
template <int KW>
__device__ __forceinline__ uint32_t* key_words(const Arr& a, int v) {
  return (uint32_t*)(v < 2 ? a.k0 : a.k1) + (v & 1);
}

template <int KW, class AT, class PL>
__global__ void __launch_bounds__(kPlaneThreads)
    k_apply_planes(Ctl* ctl, Arr a, int slot, const __grid_constant__ PL ops) {
  extern __shared__ uint32_t planes[];  // [ops.bits + kPlaneIdx][kPlaneThreads]
  __shared__ AT tab[PL::kTab];
  __shared__ PlaneOp sops[kMaxOps];
  __shared__ uint8_t sctrl[kPlaneCtrl];
  __shared__ uint16_t ulist[kPlaneThreads];
  __shared__ unsigned int n_ulist;
  pdl_next();
  const uint32_t* const pop = param_ptr((const uint32_t*)ops.op);
  const uint8_t* const pctrl = param_ptr(ops.ctrl);
  const double2* const ptab = param_ptr(ops.tab);
  for (uint32_t i = threadIdx.x; i < ops.n * (uint32_t)(sizeof(PlaneOp) / 4); i += blockDim.x)
    ((uint32_t*)sops)[i] = pop[i];
  for (uint32_t i = threadIdx.x; i < ops.n_ctrl; i += blockDim.x) sctrl[i] = pctrl[i];
  for (uint32_t i = threadIdx.x; i < ops.n_tab; i += blockDim.x) to_amp(tab[i], ptab[i]);
  __syncthreads();
  pdl_wait();
  if (ctl->err) return;
  const uint64_t n_dense = ctl->cnt[slot];
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(&ctl->peak, n_dense);
  uint32_t* const P = planes + threadIdx.x;
  uint32_t* const I = P + ops.bits * kPlaneThreads;  // planes of the factor index
  auto at = [](uint32_t b) { return b * (uint32_t)kPlaneThreads; };
  for_units(a, n_dense, kPlaneTile, ulist, &n_ulist, [&](uint64_t base, uint32_t lim) {
#pragma unroll 1
    for (int v = 0; v < 2 * KW && 32u * v < ops.bits; ++v) {
      uint32_t r[32];
      const uint32_t* const src = key_words<KW>(a, v) + 2 * base;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const uint32_t j = (uint32_t)i * kPlaneThreads + threadIdx.x;
        r[i] = j < lim ? src[2 * j] : 0u;
      }
      transpose32(r);
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (32u * v + i < ops.bits) P[at(32u * v + i)] = r[i];
    }
#pragma unroll 1
    for (uint32_t o = 0; o < ops.n; ++o) {
      const PlaneOp op = sops[o];
      uint32_t on = 0xffffffffu;  // branches the predicate holds on
      for (uint32_t c = 0; c < op.n_ctrl; ++c) {
        const uint32_t q = sctrl[op.ctrl + c];
        const uint32_t x = P[at(q & 127u)];
        on &= q & 128u ? ~x : x;
      }
      if (op.kind == OP_XOR) {
        for (uint32_t c = 0; c < op.w; ++c) P[at(sctrl[op.dst + c])] ^= on;
      } else if (op.kind == OP_MUL || op.kind == OP_MUL_XOR) {
        if (op.sel < 128) {
          const uint32_t one = P[at(op.sel)];
          I[at(op.shift)] = on & ~one;
          I[at(op.shift + 1u)] = on & one;
        } else {
          I[at(op.shift)] = on;
        }
        if (op.kind == OP_MUL_XOR) P[at(op.dst)] ^= on;
      } else if (op.kind == OP_TABLE) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = i < kPlaneIdx && (uint32_t)i < op.w ? I[at(i)] : 0u;
        transpose32(r);
        AT* const amp = (AT*)a.amp + base;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const uint32_t j = (uint32_t)i * kPlaneThreads + threadIdx.x;
          if (r[i] && j < lim) amp[j] = cmul(amp[j], tab[op.dst + r[i]]);
        }
      } else if (op.kind == OP_SWAP) {
        for (uint32_t i = 0; i < op.w; ++i) {
          const uint32_t x = P[at(op.dst + i)], y = P[at(op.src + i)], t = (x ^ y) & on;
          P[at(op.dst + i)] = x ^ t;
          P[at(op.src + i)] = y ^ t;
        }
      } else {  // additions: carry or borrow from plane to plane
        const bool sub = op.kind == OP_SUB_REG, reg = op.kind != OP_ADD_CONST;
        uint32_t carry = 0u;
        for (uint32_t i = 0; i < op.w; ++i) {
          const uint32_t x = P[at(op.dst + i)];
          const uint32_t b = reg ? (i < op.src_w ? P[at(op.src + i)] : 0u)
                                 : 0u - (uint32_t)((op.constant >> i) & 1ull);
          P[at(op.dst + i)] = x ^ ((b ^ carry) & on);
          const uint32_t y = sub ? ~x : x;
          carry = (y & b) | (y & carry) | (b & carry);
        }
      }
    }
    if (ops.touches_keys)
#pragma unroll 1
      for (int v = 0; v < 2 * KW && 32u * v < ops.bits; ++v) {
        uint32_t r[32];
        uint32_t* const dst = key_words<KW>(a, v) + 2 * base;
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = 32u * v + i < ops.bits ? P[at(32u * v + i)] : 0u;
        transpose32(r);
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const uint32_t j = (uint32_t)i * kPlaneThreads + threadIdx.x;
          if (j < lim) dst[2 * j] = r[i];
        }
      }
  });
}

template <int KW, class AT, class PL>
cudaError_t planes_t(const Launch& L, Ctl* ctl, Arr a, int slot, const PL& ops) {
  const auto kern = k_apply_planes<KW, AT, PL>;
  constexpr size_t most = (size_t)(64 * KW + kPlaneIdx) * kPlaneThreads * 4;
  static std::atomic<unsigned long long> configured{0};  // opt-in above 48 KB, per device
  cudaError_t e = ensure_smem_optin((const void*)kern, most, configured);
  if (e != cudaSuccess) return e;
  uint64_t grid = (L.n_hint + kPlaneTile - 1) / kPlaneTile;
  const uint64_t cap = (uint64_t)L.sm_count * 8;
  grid = grid < 1 ? 1 : (grid > cap ? cap : grid);
  return launch_next(kern, grid, kPlaneThreads, (size_t)(ops.bits + kPlaneIdx) * kPlaneThreads * 4,
                     L.stream, ctl, a, slot, ops);
}

template <class PL>
cudaError_t planes_of(const Launch& L, int kw, bool amp32, Ctl* ctl, Arr a, int slot,
                      const PL& ops) {
  if (kw == 2)
    return amp32 ? planes_t<2, float2>(L, ctl, a, slot, ops)
                 : planes_t<2, double2>(L, ctl, a, slot, ops);
  return amp32 ? planes_t<1, float2>(L, ctl, a, slot, ops)
               : planes_t<1, double2>(L, ctl, a, slot, ops);
}

}  // namespace

cudaError_t launch_apply_planes(const Launch& L, int kw, bool amp32, Ctl* ctl, Arr a, int slot,
                                const PlaneList& ops) {
  if (ops.n_tab > (uint32_t)PlaneListSmall::kTab)
    return planes_of(L, kw, amp32, ctl, a, slot, ops);
  PlaneListSmall s;
  s.n = ops.n;
  s.n_ctrl = ops.n_ctrl;
  s.n_tab = ops.n_tab;
  s.bits = ops.bits;
  s.touches_keys = ops.touches_keys;
  for (uint32_t i = 0; i < ops.n; ++i) s.op[i] = ops.op[i];
  for (uint32_t i = 0; i < ops.n_ctrl; ++i) s.ctrl[i] = ops.ctrl[i];
  for (uint32_t i = 0; i < ops.n_tab; ++i) s.tab[i] = ops.tab[i];
  return planes_of(L, kw, amp32, ctl, a, slot, s);
}

// The list on planes; false when it holds operations on values, prunes, or
// more predicate bits than a list takes.
bool plane_list(const OpList& L, uint32_t total_bits, PlaneList& p) {
  p.n = L.n;
  p.n_ctrl = 0;
  p.n_tab = L.n_tab;
  p.bits = total_bits;
  p.touches_keys = L.touches_keys;
  if (L.drops) return false;
  for (uint32_t i = 0; i < L.n_tab; ++i) p.tab[i] = L.tab[i];
  uint32_t idx_bits = 0;  // of the factor index since the last table
  for (uint32_t i = 0; i < L.n; ++i) {
    const DevOp& d = L.op[i];
    PlaneOp& o = p.op[i];
    o = PlaneOp{};
    o.kind = (uint8_t)d.kind;
    o.ctrl = (uint16_t)p.n_ctrl;
    for (uint32_t q = 0; q < total_bits; ++q)
      if ((d.pmask[q >> 6] >> (q & 63)) & 1ull) {
        if (p.n_ctrl >= (uint32_t)kPlaneCtrl || o.n_ctrl == 255) return false;
        p.ctrl[p.n_ctrl++] = (uint8_t)(q | (((d.pval[q >> 6] >> (q & 63)) & 1ull) ? 0u : 128u));
        o.n_ctrl++;
      }
    switch (d.kind) {
      case OP_XOR:  // the planes to flip, listed after the predicate
        o.dst = (uint16_t)p.n_ctrl;
        for (uint32_t q = 0; q < total_bits; ++q)
          if ((d.xmask[q >> 6] >> (q & 63)) & 1ull) {
            if (p.n_ctrl >= (uint32_t)kPlaneCtrl) return false;
            p.ctrl[p.n_ctrl++] = (uint8_t)q;
            o.w++;
          }
        break;
      case OP_MUL_XOR:
        if (__builtin_popcountll(d.xmask[0]) + __builtin_popcountll(d.xmask[1]) != 1) return false;
        o.dst = (uint16_t)(d.xmask[0] ? __builtin_ctzll(d.xmask[0])
                                      : 64 + __builtin_ctzll(d.xmask[1]));
        break;
      case OP_MUL:
      case OP_TABLE:
      case OP_ADD_REG:
      case OP_SUB_REG:
      case OP_ADD_CONST:
      case OP_SWAP:
        break;
      default:
        return false;
    }
    if (d.kind == OP_MUL || d.kind == OP_MUL_XOR) {
      o.sel = (uint8_t)(d.sel_bit < 128 ? d.sel_bit : 128);
      o.shift = (uint8_t)d.shift;
      idx_bits = d.shift + (d.sel_bit < 128 ? 2u : 1u);
      if (idx_bits > (uint32_t)kPlaneIdx) return false;
    } else if (d.kind == OP_TABLE) {
      o.dst = (uint16_t)d.tab_off;
      o.w = (uint8_t)idx_bits;
      idx_bits = 0;
    } else if (d.kind != OP_XOR) {
      o.dst = (uint16_t)d.dst_off;
      o.w = (uint8_t)d.dst_w;
      o.src = (uint16_t)d.src_off;
      o.src_w = (uint8_t)d.src_w;
      o.constant = d.constant;
    }
  }
  return true;
}

}  // namespace sqs
