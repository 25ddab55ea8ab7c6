// rtlfs_device.h -- device helpers shared by the faulty-machine kernels: op evaluation, the
// fault function, and the search for the next cycle in which a fault acts by itself.
#pragma once
#include "rtlfs_internal.h"

namespace rtlfs {

__device__ __forceinline__ uint64_t wmask(uint32_t w) {
    return w >= 64 ? ~0ull : ((1ull << w) - 1ull);
}

__device__ __forceinline__ int n_operands(uint32_t op) {
    return op == OP_CONST ? 0
         : (op == OP_NOT || op == OP_SHL || op == OP_SHR || op == OP_SLICE) ? 1
         : op == OP_MUX2 ? 3 : 2;
}

// One word-level op on zero-extended operands, masked to the node width.
__device__ __forceinline__ uint64_t eval_op(uint4 d, uint64_t a, uint64_t b, uint64_t c) {
    const uint32_t m = d.w, k = meta_k(m);
    uint64_t r;
    switch (meta_op(m)) {
    case OP_AND:    r = a & b; break;
    case OP_OR:     r = a | b; break;
    case OP_XOR:    r = a ^ b; break;
    case OP_NOT:    r = ~a; break;
    case OP_ADD:    r = a + b; break;
    case OP_SUB:    r = a - b; break;
    case OP_MUX2:   r = a ? b : c; break;
    case OP_EQ:     r = (a == b) ? 1ull : 0ull; break;
    case OP_LT:     r = (a < b) ? 1ull : 0ull; break;
    case OP_SHL:    r = k >= 64 ? 0ull : (a << k); break;
    case OP_SHR:
    case OP_SLICE:  r = k >= 64 ? 0ull : (a >> k); break;
    case OP_CONCAT: r = (k >= 64 ? 0ull : (a << k)) | b; break;
    default:        r = ((uint64_t)d.y << 32) | d.x; break;   // CONST
    }
    return r & wmask(meta_w(m));
}

// eval_op with the operands in their value slots (x, y; s: the MUX2 select), without branches:
// the lanes of a warp hold nodes of any op. x is shifted first (by 0 for most ops); the logic
// ops, the shifts, CONCAT and MUX2 are then (x & y & A) ^ (x & B) ^ (y & C) ^ D with masks the
// record names (PM_*), a MUX2's B and C chosen by s.
__device__ __forceinline__ uint64_t pack_eval(uint4 d, uint64_t x, uint64_t y, uint64_t s) {
    uint32_t w = d.w;
    if (s) w ^= PM_B | PM_C;
    const uint32_t k = meta_k(w), op = meta_op(w);
    uint64_t xl, xr;   // shl/shr by more than 63 give 0
    asm("shl.b64 %0, %1, %2;" : "=l"(xl) : "l"(x), "r"(k));
    asm("shr.u64 %0, %1, %2;" : "=l"(xr) : "l"(x), "r"(k));
    const uint64_t xs = w & PM_LEFT ? xl : xr;
    auto mask = [&](uint32_t bit) -> uint64_t {
        const uint32_t m = w & bit ? ~0u : 0u;
        return (uint64_t)m << 32 | m;
    };
    uint64_t r = (xs & y & mask(PM_A)) ^ (xs & mask(PM_B)) ^ (y & mask(PM_C)) ^ mask(PM_D);
    const uint64_t neg = op == OP_SUB ? ~0ull : 0ull;
    r = w & PM_SUM ? x + (y ^ neg) - neg : r;
    const bool cmp = op == OP_EQ ? x == y : x < y;
    r = w & PM_CMP ? (cmp ? 1ull : 0ull) : r;
    r = op == OP_CONST ? (uint64_t)d.y << 32 | d.x : r;
    return r & (~0ull >> (64u - meta_w(w)));
}

// The fault function at a fault's site (Sec. IV-A: applied wherever the site's value is
// produced; a virtual function in the paper, a switch on the kind here): stuck-at 0 or 1
// forces the bit in every cycle; a transient flip (an SEU on a register, an SET on an
// input or node net) inverts it during cycle t0 only. A port fault (port != NO_PORT) acts
// on what one output port observes of the site net and on nothing else.
struct FaultSite {
    uint32_t site, port, kind, t0;
    uint64_t bm;   // one-hot mask of the faulted bit
    __device__ __forceinline__ uint64_t apply(uint64_t v, uint32_t t) const {
        return kind == FK_SA0 ? (v & ~bm) : kind == FK_SA1 ? (v | bm) : (t == t0 ? v ^ bm : v);
    }
    // whether the fault function changes anything in cycle t (a stuck-at fault: always)
    __device__ __forceinline__ bool acts(uint32_t t) const { return kind != FK_FLIP || t == t0; }
};

__device__ __forceinline__ FaultSite load_fault(const DevFaults &f, uint32_t fid) {
    FaultSite s;
    s.site = f.site[fid];
    s.kind = f.val[fid];
    s.bm = 1ull << f.bit[fid];
    s.port = f.port ? f.port[fid] : NO_PORT;
    s.t0 = f.t0 ? f.t0[fid] : 0u;
    return s;
}

// Loads issued where they stand: volatile, so the compiler does not sink them into the
// branch that consumes them and they travel together with the operand loads.
__device__ __forceinline__ uint32_t ld_early_u32(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t ld_early_u16(const uint16_t *p) {
    unsigned short v;
    asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// First cycle in [t, tend) where the fault is active by itself, or tend.
__device__ __forceinline__ uint32_t next_active(const uint64_t *__restrict__ fact, uint32_t t, uint32_t tend) {
    while (t < tend) {
        const uint64_t w = __ldg(fact + (t >> 6)) >> (t & 63u);
        if (w) {
            const uint32_t a = t + (uint32_t)(__ffsll((long long)w) - 1);
            return a < tend ? a : tend;
        }
        t = (t | 63u) + 1;
    }
    return tend;
}

}  // namespace rtlfs
