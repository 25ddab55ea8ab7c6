// rtlfs_pack.cu -- the packed faulty-machine kernel: a warp simulates 32 / LPS faults, each in
// the hands of LPS lanes, and takes a step of every fault per round.
//
// The rounds are asynchronous across faults: every fault is at a cycle and a topological
// level of its own. In a round each lane takes one item of its fault: a dirty node (some
// operand differs) of the fault's lowest level that has any, or, when the fault has no dirty
// node left -- its cycle is complete, it latches and moves to its next cycle, or is replaced
// from the queue -- a seed of the new cycle (a latched register diff or the faulted site).
// Both kinds then share one piece of code: compare with the good value, and hand the value to
// the consumers. So the lanes of a warp stay together on the nodes of many faults, instead of
// walking one fault's levels with two busy lanes, or diverging over 32 private loops.
//
// A fault owns a hash table of TPL x LPS entries in shared memory, one per dirty node of the
// cycle, keyed by net. The net that differs stores its value into the operand slot of each
// consumer's entry (an edge of the op graph knows which operands it feeds: two value slots
// and, for a MUX2 select, one bit), so evaluating a node needs no search: an operand that was
// delivered is in the entry, any other is the good value. Insertion (compare-and-swap) makes
// each dirty node an item once. A 16-bit tag per entry holds a pending item's level above the
// entry's place among the TPL its lane owns, so the minimum over a lane's tags (two per
// instruction) is both the fault's next level and an item of it, without any list. Register diffs
// go to a private double buffer.
//
// Tiers: one lane per fault for the many faults with a handful of dirty nodes, then 8, a warp,
// and a CTA of 256. A fault that outgrows its table or buffer is handed to the next tier
// with its start-of-cycle register diffs; behind the last is the heavy kernel, with its
// state in global memory, which also takes the last tier's faults where they are too many for it
// (plan_pack). Which faults count as light or heavy (evaluation counters, promotions) does not
// depend on the tier or on the kernel: a fault is heavy from the first cycle with more
// evaluations or register diffs than light_cap names. (The light kernel promotes by what is pending or
// differs at once instead, so the two forms' counts differ; their sums do not.)
//
// What bounds it: a warp instruction takes 7 to 8 cycles (2.2 of fixed latency, 1.2-1.9 of global
// loads, 1.1 of branches), and a warp's tables take 9 to 15 KB of shared memory, so 3 to 7 warps a
// tier are resident on an SM. With many faults (20k nodes, 100k faults, a window of 64 cycles) the
// tiers issue in 12 to 22% of the slots, 16% for the busiest; with few (5,003 faults) a tier lasts as
// long as its slowest fault's chain of rounds, about a microsecond per level. Neither memory nor
// issue is near a limit. Light and heavy kernels -> packed (whole calls, with the good trace's own
// gains): tiny list 6.8 -> 2.4 ms, 2.8k nodes 61 -> 15 ms, 20k nodes with 5k faults 286 -> 82 ms, with
// 100k faults over 10k cycles 1125 -> 850 ms, transient list 270 -> 152 ms, no-drop 131 -> 72 to 80 ms, twelve
// designs 193 -> 88 ms, 200k nodes 169 -> 62 to 65 ms.
// With few faults the last tier sets the pace, and its level the barriers and instructions of its
// rounds. Slower there (before its reductions took one barrier): items listed and dealt to the lanes
// evenly (recorded loads 103 against 83 ms: few rounds have two items on a lane), consumers' records
// prefetched into L1 when they are marked (88), 128 or 64 lanes (no-drop with another fault list 247,
// 258 against 115: tables overflow).
#include "rtlfs_device.h"
#include "rtlfs_internal.h"

namespace rtlfs {

constexpr uint32_t FULL = 0xFFFFFFFFu;
constexpr uint32_t PK_EMPTY = 0xFFFFFFFFu;     // no key
constexpr uint32_t PK_IDLE = 0xFFFFu;          // tag of an entry with nothing pending
constexpr uint32_t PK_NET = 0x07FFFFFFu;       // key: net, and what was delivered:
constexpr uint32_t PK_F0 = 1u << 27, PK_F1 = 1u << 28;   // value slots 0 and 1
constexpr uint32_t PK_FV = 1u << 30;   // and that the MUX2 select (bit 29) is not 0
constexpr uint32_t PK_RING = 16;               // long fan-out ranges marked together

// The shared memory of one unit: a warp, or the CTA when it works on one fault (N lanes;
// pack_unit_bytes sizes the same layout).
struct PackSmem {
    uint64_t *val;           // [2][N TPL] delivered operand values
    uint64_t *regv;          // [2][N RPL] register diffs: value
    uint32_t *key;           // [N TPL] net | PK_F*
    uint32_t *regr;          // [2][N RPL] and register
    uint16_t *tag;           // [N TPL] level << 4 | place, or PK_IDLE
    uint32_t *nnew;          // [32] register diffs latched by a fault this cycle
    uint32_t *fail;          // [32] the fault outgrew its table or buffer
    uint32_t *n_ring;
    uint32_t *ring;          // [PK_RING][5] {slot, first, end, value} of fan-out entries
};

__host__ __device__ constexpr size_t pack_unit_bytes(int n, int tpl, int rpl) {
    return (size_t)n * tpl * 22 + (size_t)2 * n * rpl * 12 + (64 + 8 + 5 * PK_RING) * 4;
}

template <int N, int TPL, int RPL>
__device__ __forceinline__ PackSmem pack_layout(unsigned char *sm) {
    PackSmem m;
    m.val = reinterpret_cast<uint64_t *>(sm);
    m.regv = m.val + 2 * N * TPL;
    m.key = reinterpret_cast<uint32_t *>(m.regv + 2 * N * RPL);
    m.regr = m.key + N * TPL;
    m.tag = reinterpret_cast<uint16_t *>(m.regr + 2 * N * RPL);
    m.nnew = reinterpret_cast<uint32_t *>(m.tag + N * TPL);
    m.fail = m.nnew + 32;
    m.n_ring = m.fail + 32;
    m.ring = m.n_ring + 8;
    return m;
}

// Compare-and-swap of an empty key where `on`; PK_EMPTY when it was empty or not on. Without
// a branch around it.
__device__ __forceinline__ uint32_t cas_if(bool on, uint32_t *key, uint32_t w) {
    uint32_t old;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.u32 p, %3, 0;\n\t"
                 "mov.u32 %0, 0xffffffff;\n\t"
                 "@p atom.shared.cas.b32 %0, [%1], 0xffffffff, %2;\n\t}"
                 : "=&r"(old) : "r"((uint32_t)__cvta_generic_to_shared(key)), "r"(w), "r"((uint32_t)on) : "memory");
    return old;
}

template <int LPS, int TPL, int RPL, bool MULTI>
__global__ void __launch_bounds__(LPS > 32 ? LPS : PACK_MAX_WARPS * 32, 1)
pack_kernel(const DevDesign *__restrict__ designs, const __grid_constant__ DevDesign D0, DevFaults f, const __grid_constant__ PackArgs q) {
    constexpr uint32_t E = TPL * LPS;   // table entries of a fault (a power of two)
    constexpr uint32_t R = RPL * LPS;   // register diffs of a fault
    constexpr uint32_t PROBES = E < 32 ? E : 32;
    constexpr int EBITS = E == 8 ? 3 : E == 16 ? 4 : E == 32 ? 5 : E == 64 ? 6 : E == 128 ? 7 : E == 256 ? 8 : E == 512 ? 9 : E == 1024 ? 10 : E == 2048 ? 11 : E == 4096 ? 12 : 13;
    static_assert(E == 1u << EBITS, "table size");
    static_assert(TPL == 8 || TPL == 16, "tags are scanned 8 at a time and hold 4 bits of place");
    extern __shared__ __align__(16) unsigned char psm[];
    constexpr bool BLOCK = LPS > 32;           // the whole CTA works on one fault
    constexpr uint32_t N = BLOCK ? LPS : 32;   // lanes that share tables
    constexpr uint32_t G = N / LPS;            // faults (slots) among them
    const uint32_t lane = BLOCK ? threadIdx.x : threadIdx.x & 31u, slot = lane / LPS, sub = lane % LPS;
    const uint32_t gmask = LPS >= 32 ? FULL : ((1u << (LPS & 31)) - 1u) << (slot * LPS);
    const PackSmem sm = pack_layout<N, TPL, RPL>(psm + (BLOCK ? 0 : (threadIdx.x >> 5) * pack_unit_bytes(N, TPL, RPL)));
    const bool nodrop = f.mism != nullptr;
    const uint32_t n_carry = q.n_carry_in ? *q.n_carry_in : 0u;
    const uint32_t item0 = q.item_begin ? *q.item_begin : 0u;
    const uint32_t n_list = q.live_in ? (q.n_live_in ? *q.n_live_in : q.n_live) : *q.item_end - item0;
    const uint32_t n_items = n_carry + n_list;
    const bool crowded = LPS > 1 && n_items > q.tier_limit;
    if (BLOCK && crowded) return;   // the heavy kernel takes them
    // few faults: spread them over all units
    const uint32_t n_units = BLOCK ? gridDim.x : gridDim.x * (blockDim.x >> 5);
    const bool use_slot = slot < (n_items + n_units - 1) / n_units;
    const DevDesign *const only = &D0;

    auto usync = [&]() { if (BLOCK) __syncthreads(); else __syncwarp(); };   // all lanes of the unit
    auto uany = [&](bool x) { return BLOCK ? x : __any_sync(FULL, x) != 0; };   // (BLOCK: the same in every lane)
    auto gshfl = [&](auto v) {   // the owner's value
        if constexpr (BLOCK) {
            __shared__ unsigned long long b;
            if (sub == 0) b = (unsigned long long)v;
            __syncthreads();
            v = (decltype(v))b;
            __syncthreads();
            return v;
        } else {
            return LPS == 1 ? v : __shfl_sync(gmask, v, slot * LPS);
        }
    };
    auto gsum = [&](uint32_t v) {
        if constexpr (BLOCK) {
            __shared__ uint32_t w[N / 32];
            v = __reduce_add_sync(FULL, v);
            if ((lane & 31u) == 0) w[lane >> 5] = v;
            __syncthreads();
            v = 0u;
#pragma unroll
            for (uint32_t k = 0; k < N / 32; ++k) v += w[k];
        } else {
#pragma unroll
            for (int o = 1; o < LPS; o <<= 1) v += __shfl_xor_sync(gmask, v, o);
        }
        return v;
    };
    auto gmin = [&](uint32_t v) {
        // A CTA's lanes meet once per reduction (its warps' results side by side; calls lie another
        // barrier apart): with an atomic per warp and a second barrier a level of its one fault took
        // an eighth longer (recorded loads 83 -> 75 ms, transient list 157 -> 138).
        if constexpr (BLOCK) {
            __shared__ uint32_t w[N / 32];
            v = __reduce_min_sync(FULL, v);
            if ((lane & 31u) == 0) w[lane >> 5] = v;
            __syncthreads();
            v = FULL;
#pragma unroll
            for (uint32_t k = 0; k < N / 32; ++k) v = min(v, w[k]);
        } else if constexpr (LPS == 32) {
            v = __reduce_min_sync(FULL, v);
        } else {
#pragma unroll
            for (int o = 1; o < LPS; o <<= 1) v = min(v, __shfl_xor_sync(gmask, v, o));
        }
        return v;
    };

    // ---- this group's fault (the same in its LPS lanes) ---------------------------------
    FaultSite fs{};
    const DevDesign *D = only;   // MULTI: its design
    auto DD = [&]() -> const DevDesign & { return *(MULTI ? D : only); };
    const uint64_t *dg = D0.gcol;
    const uint4 *dr = D0.rec;
    uint32_t dT = D0.T, dI = D0.I, dIR = D0.I + D0.R;
    auto gcol = [&]() -> const uint64_t * { return MULTI ? dg : D0.gcol; };
    auto recs = [&]() -> const uint4 * { return MULTI ? dr : D0.rec; };
    auto cycles = [&]() -> uint32_t { return MULTI ? dT : D0.T; };
    unsigned long long before = 0;                   // evaluations before this run (budget checks)
    unsigned long long ev_light = 0, ev_heavy = 0;   // evaluations of this run
    unsigned long long acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;   // evaluations, fault-cycles: light, heavy
    uint32_t fid = 0, tend = 0, t = 0, t_begin = 0;
    uint32_t nreg = 0, cur = 0;                // register diffs entering cycle t, and their buffer
    uint32_t seeded = 0;                       // seeds of the cycle taken so far
    bool seeding = false, has_site = false;    // has_site: this lane met the faulted register's diff
    uint32_t t_heavy = 0, mism = 0;            // first cycle counted as heavy
    bool active = false, heavy = false, seen = false;
    bool more = use_slot;                      // the queue may hold further items
    // of the running cycle, per lane: evaluations and lowest differing port
    uint32_t my_ev = 0, my_port = NI_NO_PORT;
    uint32_t fr_begin = 0;                     // first unexpanded ring entry

    // ---- table ------------------------------------------------------------------------
    auto home = [&](uint32_t e) -> uint32_t { return ((e & PK_NET) * 0x9E3779B1u) >> (32 - EBITS); };
    // what edge e (consumer net | operands it feeds, as in the key) delivers of value v
    auto want = [&](uint32_t e, uint64_t v) -> uint32_t { return e | (v ? (e << 1) & PK_FV : 0u); };
    // Consumer w (as want() gives it) of slot sl becomes dirty; its home i was not free: it was
    // there, or another net is.
    auto settle = [&](uint32_t sl, uint32_t w, uint32_t i, uint32_t old) -> uint32_t {
        uint32_t h = i - sl * E;
#pragma unroll 1
        for (uint32_t p = 0; old != PK_EMPTY && ((old ^ w) & PK_NET); ++p) {
            if (p == PROBES) { sm.fail[sl] = 1u; return PK_EMPTY; }
            h = (h + 1) & (E - 1);
            old = atomicCAS(&sm.key[sl * E + h], PK_EMPTY, w);
        }
        i = sl * E + h;
        if (old != PK_EMPTY) atomicOr(&sm.key[i], w);
        return i;
    };
    // its value and tag (lv: its level << 4)
    auto deliver = [&](uint32_t sl, uint32_t w, uint32_t lv, uint64_t v, uint32_t i, uint32_t old) {
        if (old != PK_EMPTY) {
            i = settle(sl, w, i, old);
            if (i == PK_EMPTY) return;
        }
        if (w & PK_F0) sm.val[i] = v;
        if (w & PK_F1) sm.val[N * TPL + i] = v;
        sm.tag[i] = (uint16_t)(lv | (i & (TPL - 1)));
    };
    auto mark = [&](uint32_t sl, uint32_t e, uint32_t lv, uint64_t v) {
        const uint32_t w = want(e, v), i = sl * E + home(w);
        deliver(sl, w, lv, v, i, atomicCAS(&sm.key[i], PK_EMPTY, w));
    };

    // ---- a fault's comings and goings -----------------------------------------------------
    // its counts so far go to the campaign's; `end` = first cycle not simulated here
    auto flush = [&](uint32_t end) {
        if (sub) return;
        f.load[fid] = before + ev_light + ev_heavy;
        if (nodrop && mism) f.mism[fid] += mism;
        acc0 += ev_light;
        acc2 += ev_heavy;
        const uint32_t th = heavy ? t_heavy : end;
        if (th > t_begin) acc1 += th - t_begin;
        if (heavy && end > th) acc3 += end - th;
    };
    // the fault's final result: undetected, detected at t on `port`, or over the budget
    auto finish = [&](bool detected, bool budget, uint32_t port) {
        if (sub || (!detected && !budget && nodrop)) return;
        f.res_det[fid] = detected ? 1 : budget ? 255 : 0;
        f.res_cycle[fid] = detected ? (int32_t)t : -1;
        f.res_port[fid] = detected ? (int32_t)port : -1;
        if (budget) atomicAdd(q.budget_hit, 1ull);
    };
    auto append_one = [&](uint32_t *count) -> uint32_t {   // one position per calling lane
        const unsigned m = __activemask();
        const int leader = __ffs(m) - 1;
        uint32_t base = 0;
        if ((int)lane == leader) base = atomicAdd(count, (uint32_t)__popc(m));
        base = __shfl_sync(m, base, leader);
        return base + __popc(m & ((1u << lane) - 1u));
    };
    auto reg_at = [&](uint32_t half, uint32_t k) -> uint32_t { return (half * G + slot) * R + k; };
    // alive at the end of the window: onto the survivors' list with its register diffs
    auto survive = [&]() {
        if (sub == 0) q.cls[fid] = heavy;
        if (LPS == 1) {
            q.st_nreg[fid] = (uint8_t)nreg;
#pragma unroll 1
            for (uint32_t k = 0; k < nreg; ++k) {
                q.st_r[(size_t)k * f.F + fid] = sm.regr[reg_at(cur, k)];
                q.st_v[(size_t)k * f.F + fid] = sm.regv[reg_at(cur, k)];
            }
            q.live_out[append_one(q.n_live_out)] = fid;
            return;
        }
        unsigned long long off = 0;
        if (sub == 0) off = atomicAdd(q.pool_top, (unsigned long long)nreg);
        off = gshfl(off);
        if (off + nreg > q.pool_cap) {
            if (sub == 0) atomicOr(q.err, 2u);
            return;
        }
#pragma unroll 1
        for (uint32_t k = sub; k < nreg; k += LPS) {
            q.pool_r[off + k] = sm.regr[reg_at(cur, k)];
            q.pool_v[off + k] = sm.regv[reg_at(cur, k)];
        }
        if (sub == 0) q.carry_out[atomicAdd(q.n_carry_out, 1u)] = HeavyCarry{fid, nreg, off};
    };
    // To the next tier from the start of cycle t; the register diffs come from this warp's
    // buffer or, when they never fitted it, from where they were to be loaded.
    auto promote = [&](const uint32_t *src_r, const uint64_t *src_v, size_t stride) {
        unsigned long long off = 0;
        if (sub == 0) {
            q.cls[fid] = heavy;
            off = atomicAdd(q.prom_top, (unsigned long long)nreg);
        }
        off = gshfl(off);
        if (off + nreg > q.prom_cap) {
            if (sub == 0) atomicOr(q.err, 2u);
            return;
        }
#pragma unroll 1
        for (uint32_t k = sub; k < nreg; k += LPS) {
            q.prom_r[off + k] = src_r ? src_r[k * stride] : sm.regr[reg_at(cur, k)];
            q.prom_v[off + k] = src_r ? src_v[k * stride] : sm.regv[reg_at(cur, k)];
        }
        if (sub == 0) q.items_out[atomicAdd(q.n_items_out, 1u)] = PackItem{fid, t, nreg, (uint32_t)off};
    };
    // A detection at cycle t on `port`: true when the fault is dropped.
    auto detect = [&](uint32_t port) -> bool {
        if (!nodrop) return true;
        if (!seen && sub == 0) {
            f.res_det[fid] = 1;
            f.res_cycle[fid] = (int32_t)t;
            f.res_port[fid] = (int32_t)port;
        }
        seen = true;
        ++mism;
        return false;
    };
    // after a completed cycle, before cycle t; not at the end of one of the caller's windows
    auto over_budget = [&]() -> bool {
        return q.fault_budget && before + ev_light + ev_heavy > q.fault_budget && (t < tend || (q.budget_at_end && t < cycles()));
    };
    // What becomes of the fault at cycle t.
    enum { RUN, DETECTED, BUDGET, END, PROMOTE };
    uint32_t port = NI_NO_PORT;   // the detecting port
    // With nothing latched, move on to the next cycle in which the fault acts by itself.
    auto advance = [&]() -> int {
#pragma unroll 1
        for (;;) {
            if (t >= tend) return END;
            if (nreg) return RUN;
            if (fs.kind == FK_FLIP) {
                t = t <= fs.t0 ? min(fs.t0, tend) : tend;
            } else if (f.act) {
                t = next_active(f.act + (size_t)fid * f.act_stride, t, tend);
            } else {
                const uint64_t *scol = gcol() + (size_t)fs.site * cycles();
                const uint64_t want = fs.kind == FK_SA1 ? fs.bm : 0ull;
#pragma unroll 1
                while (t < tend && (__ldg(scol + t) & fs.bm) == want) ++t;
            }
            if (t >= tend) continue;
            if (fs.port == NO_PORT) return RUN;
            // a port fault changes only what its port observes of the site net
            (heavy ? ev_heavy : ev_light) += 1;
            port = fs.port;
            if (detect(port)) return DETECTED;
            ++t;
            if (over_budget()) return BUDGET;
        }
    };

    // ---- scan: the group's lowest pending level, and this lane's first item of it ------------
    constexpr uint32_t NONE = PK_IDLE >> 4;   // no level
    uint32_t level = NONE, item = PK_EMPTY;
    auto scan = [&]() {
        uint32_t m = FULL;
#pragma unroll
        for (int k = 0; k < TPL / 8; ++k) {
            const uint4 x = reinterpret_cast<const uint4 *>(sm.tag)[lane * (TPL / 8) + k];
            m = __vminu2(m, __vminu2(__vminu2(x.x, x.y), __vminu2(x.z, x.w)));
        }
        m = min(m & 0xFFFFu, m >> 16);
        const uint32_t mine = m >> 4;
        level = gmin(mine);
        item = mine == level && m != PK_IDLE ? lane * TPL + (m & 15u) : PK_EMPTY;
    };

#pragma unroll
    for (int k = 0; k < TPL / 8; ++k) reinterpret_cast<uint4 *>(sm.tag)[lane * (TPL / 8) + k] = make_uint4(~0u, ~0u, ~0u, ~0u);
    if (lane == 0) *sm.n_ring = 0u;
    usync();
    if (!uany(more)) return;

    for (;;) {
        scan();
        const bool turn = level == NONE && !seeding && (active || more);
        if (uany(turn)) {
            if (turn) {
                int next = RUN;
                const uint32_t *src_r = nullptr;   // register diffs that were never loaded
                const uint64_t *src_v = nullptr;
                size_t stride = 1;
                // (1) the completed cycle
                if (active) {
                    const uint32_t ev = gsum(my_ev), nr = sm.nnew[slot];
                    port = gmin(my_port);
                    // the capacity rule: more register diffs or evaluations in a cycle than a light
                    // fault may have make the fault heavy, that cycle included; so does a cycle
                    // that not even the last tier holds (its table and buffer are far beyond the
                    // rule), which the heavy kernel simulates without looking at the class
                    const bool full = sm.fail[slot] != 0u;
                    if (!heavy && (full ? BLOCK : nr > q.cap_regs || ev > q.cap_evals)) {
                        heavy = true;
                        t_heavy = t;
                        if (sub == 0) atomicAdd(q.prom_total, 1u);
                    }
                    if (full) {
                        next = PROMOTE;
                    } else {
                        (heavy ? ev_heavy : ev_light) += ev;
                        if (port != NI_NO_PORT && detect(port)) {
                            next = DETECTED;
                        } else {
                            cur ^= 1u;
                            nreg = nr;
                            ++t;
                            if (over_budget()) next = BUDGET;
                            else if (t < tend && ev > q.tier_evals) next = PROMOTE;   // slow here
                        }
                    }
                }
                // (2) its next cycle, or the next fault
#pragma unroll 1
                for (;;) {
                    if (active && next == RUN) next = advance();
                    if (next != RUN) {
                        flush(next == DETECTED ? t + 1 : t);
                        if (next == PROMOTE) promote(src_r, src_v, stride);
                        else if (next == END && tend < cycles()) survive();
                        else finish(next == DETECTED, next == BUDGET, port);
                        active = false;
                        next = RUN;
                    }
                    if (active || !more) break;
                    unsigned long long base = 0;
                    if (LPS == 1) {
                        const unsigned m = __activemask();
                        const int leader = __ffs(m) - 1;
                        if ((int)lane == leader) base = atomicAdd(q.head, (unsigned long long)__popc(m));
                        base = __shfl_sync(m, base, leader) + __popc(m & ((1u << lane) - 1u));
                    } else {
                        if (sub == 0) base = atomicAdd(q.head, 1ull);
                        base = gshfl(base);
                    }
                    if (base >= n_items) { more = false; break; }
                    const uint32_t qi = (uint32_t)base;
                    src_r = nullptr;
                    stride = 1;
                    nreg = 0;
                    t = q.t0;
                    if (qi < n_carry) {   // back to front: the slowest of the last window first
                        const HeavyCarry c = q.carry_in[n_carry - 1 - qi];
                        fid = c.fault;
                        nreg = c.nreg;
                        src_r = q.pool_r_in + c.off;
                        src_v = q.pool_v_in + c.off;
                        heavy = q.cls[fid];
                    } else if (LPS == 1) {
                        const uint32_t li = qi - n_carry;
                        fid = q.live_in[q.reverse ? n_list - 1 - li : li];
                        heavy = q.fresh ? li < q.n_heavy : q.cls[fid];
                        if (!q.fresh) nreg = q.st_nreg[fid];
                        src_r = q.st_r + fid;
                        src_v = q.st_v + fid;
                        stride = f.F;
                    } else {
                        const PackItem it = q.items[item0 + qi - n_carry];
                        fid = it.fault;
                        t = it.t;
                        nreg = it.nreg;
                        src_r = q.prom_r_in + it.off;
                        src_v = q.prom_v_in + it.off;
                        heavy = q.cls[fid];
                    }
                    active = true;
                    cur = 0;
                    fs = load_fault(f, fid);
                    if (MULTI) {
                        D = designs + f.design[fid];
                        dg = D->gcol; dr = D->rec; dT = D->T; dI = D->I; dIR = D->I + D->R;
                    }
                    tend = min(q.t1, cycles());
                    t_begin = t_heavy = t;
                    before = f.load[fid];
                    ev_light = ev_heavy = 0;
                    mism = 0;
                    seen = nodrop && f.res_det[fid] == 1;
                    if (nreg > R || (LPS > 1 && crowded)) {   // never fits this tier, or too many do
                        next = PROMOTE;
                        continue;
                    }
#pragma unroll 1
                    for (uint32_t k = sub; k < nreg; k += LPS) {
                        sm.regr[reg_at(0, k)] = src_r[k * stride];
                        sm.regv[reg_at(0, k)] = src_v[k * stride];
                    }
                    src_r = nullptr;
                }
                // (3) a new cycle
                if (active) {
                    my_ev = 0;
                    my_port = NI_NO_PORT;
                    seeding = true;
                    has_site = false;
                    seeded = 0;
                    const uint4 ones = make_uint4(~0u, ~0u, ~0u, ~0u);
                    uint4 *kp = reinterpret_cast<uint4 *>(sm.key) + slot * (E / 4);
#pragma unroll
                    for (uint32_t k = 0; k < TPL / 4; ++k) kp[k * LPS + sub] = ones;   // the slot's keys
                    if (sub == 0) { sm.nnew[slot] = 0u; sm.fail[slot] = 0u; }
                }
            }
            if (!uany(active)) break;
            usync();
        }
        // (4) this lane's item: a seed or a dirty node
        const uint32_t I = MULTI ? dI : D0.I, IR = MULTI ? dIR : D0.I + D0.R, T = cycles();
        uint32_t net = 0, key = 0;
        uint64_t v = 0;
        bool have = false, site_now = false;
        if (seeding) {
            item = PK_EMPTY;
            if (seeded < nreg) {
                const uint32_t k = seeded + sub;
                if (k < nreg) {
                    net = I + sm.regr[reg_at(cur, k)];
                    v = sm.regv[reg_at(cur, k)];
                    have = true;
                    if (net == fs.site) { v = fs.apply(v, t); has_site = true; }
                }
                seeded += LPS;
            } else {
                // an input or register without a latched diff, or a node while no other net
                // differs (its operands are good): the faulty value follows from the good one
                const bool met = LPS == 1 ? has_site : gsum(has_site) != 0u;
                seeding = false;
                if (sub == 0) {
                    net = fs.site;
                    site_now = net < IR ? !met : fs.acts(t) && nreg == 0;
                    have = site_now;
                    if (site_now && net >= IR) my_ev = 1;
                    if (!site_now && net >= IR && fs.acts(t))
                        mark(slot, net, (uint32_t)__ldg(DD().node_level + net - IR) << 4, 0ull);
                }
            }
        } else if (item != PK_EMPTY) {
            key = sm.key[item];
            net = key & PK_NET;
            sm.tag[item] = (uint16_t)PK_IDLE;
            have = true;
        }
        if (have) {
            const uint64_t *__restrict__ gt = gcol() + t;
            const uint4 *rec = recs() + (size_t)net * 8;
            const uint4 d = __ldg(rec), ni = __ldg(rec + 1), ea = __ldg(rec + 2), eb = __ldg(rec + 3), lv = __ldg(rec + 4);
            const uint64_t g = __ldg(gt + (size_t)net * T);
            if (item != PK_EMPTY) {
                // operands: delivered, or good
                uint64_t x0 = 0, x1 = 0, xs = key & PK_FV ? 1ull : 0ull;
                const uint32_t need = d.w & ~(key >> 23);   // PACK_NEED bits without what was delivered
                if (need & 0x10u) x0 = __ldg(gt + (size_t)d.x * T);
                if (need & 0x20u) x1 = __ldg(gt + (size_t)d.y * T);
                if (need & 0x40u) xs = __ldg(gt + (size_t)d.z * T);
                if (key & PK_F0) x0 = sm.val[item];
                if (key & PK_F1) x1 = sm.val[N * TPL + item];
                v = pack_eval(d, x0, x1, xs);
                if (net == fs.site) v = fs.apply(v, t);
                ++my_ev;
            } else if (site_now) {
                v = fs.apply(g, t);
            }
            // (5) what a net that differs leads to: its port, the registers it drives, its consumers
            if (v != g) {
                my_port = min(my_port, ni_port(ni.w));
                uint32_t nr = ni_nreg(ni.w);
                auto latch = [&](uint32_t rr) {   // register | width << 25
                    const uint64_t wm = wmask(rr >> 25), qv = v & wm;
                    if (qv == (g & wm)) return;
                    const uint32_t k = LPS == 1 ? sm.nnew[slot]++ : atomicAdd(&sm.nnew[slot], 1u);
                    if (k >= R) { sm.fail[slot] = 1u; return; }
                    sm.regr[reg_at(cur ^ 1u, k)] = rr & 0x1FFFFFFu;
                    sm.regv[reg_at(cur ^ 1u, k)] = qv;
                };
                if (nr) {   // the first register is in the record
                    if (nr == 255u) nr = __ldg(DD().dreg_off + net + 1) - ni.z;
#pragma unroll 1
                    for (uint32_t e = 0; e < nr; ++e)   // a single one is in the record
                        latch(nr == 1 ? ni.z : __ldg(DD().dreg_rec + ni.z + e));
                }
                const uint32_t nf = ni.y - ni.x;
                uint32_t here = nf;   // consumers marked by this lane
                if (nf > 8) {
                    if (nf > E) {
                        sm.fail[slot] = 1u;
                        here = 0;
                    } else if (LPS > 1) {   // a long list: by all lanes, unless the ring is full
                        const uint32_t k = atomicAdd(sm.n_ring, 1u);
                        if (k - fr_begin < PK_RING) {
                            uint32_t *r = sm.ring + 5 * (k % PK_RING);
                            r[0] = slot; r[1] = ni.x; r[2] = ni.y; r[3] = (uint32_t)v; r[4] = (uint32_t)(v >> 32);
                            here = 0;
                        }
                    }
                }
                // the first eight are in the record: the first probes of four go out together
                auto four = [&](uint32_t k0, uint4 e, uint32_t la, uint32_t lb) {
                    const uint32_t w[4] = {want(e.x, v), want(e.y, v), want(e.z, v), want(e.w, v)};
                    const uint32_t l4[4] = {la & 0xFFFFu, la >> 16, lb & 0xFFFFu, lb >> 16};
                    uint32_t at[4], old[4];
#pragma unroll
                    for (uint32_t k = 0; k < 4; ++k) {
                        at[k] = slot * E + home(w[k]);
                        old[k] = cas_if(k0 + k < here, &sm.key[at[k]], w[k]);
                    }
                    if ((old[0] & old[1] & old[2] & old[3]) != PK_EMPTY) {   // some home was not free
#pragma unroll
                        for (uint32_t k = 0; k < 4; ++k)
                            if (old[k] != PK_EMPTY) at[k] = settle(slot, w[k], at[k], old[k]);
                    }
#pragma unroll
                    for (uint32_t k = 0; k < 4; ++k) {
                        const bool on = k0 + k < here && at[k] != PK_EMPTY;
                        if (on && (w[k] & PK_F0)) sm.val[at[k]] = v;
                        if (on && (w[k] & PK_F1)) sm.val[N * TPL + at[k]] = v;
                        if (on) sm.tag[at[k]] = (uint16_t)(l4[k] | (at[k] & (TPL - 1)));
                    }
                };
                four(0, ea, lv.x, lv.y);
                if (here > 4) {
                    four(4, eb, lv.z, lv.w);
#pragma unroll 1
                    for (uint32_t k = 8; k < here; ++k)
                        mark(slot, __ldg(DD().fo_edge + ni.x + k), (uint32_t)__ldg(DD().fo_lvl + ni.x + k) << 4, v);
                }
            }
        }
        usync();
        if (LPS > 1) {
            const uint32_t rend = *sm.n_ring;
            if (rend != fr_begin) {   // long fan-out lists, marked by all lanes
                const uint32_t n = min(rend - fr_begin, PK_RING);
#pragma unroll 1
                for (uint32_t k = 0; k < n; ++k) {
                    const uint32_t *r = sm.ring + 5 * ((fr_begin + k) % PK_RING);
                    const uint32_t sl = r[0], e1 = r[2];
                    const uint64_t rv = (uint64_t)r[4] << 32 | r[3];
                    const DevDesign *Ds = !MULTI ? only : BLOCK ? D : reinterpret_cast<const DevDesign *>(__shfl_sync(FULL, reinterpret_cast<unsigned long long>(D), sl * LPS & 31));
                    const DevDesign &DR = *(MULTI ? Ds : only);
#pragma unroll 1
                    for (uint32_t x = r[1] + lane; x < e1 && !sm.fail[sl]; x += N)
                        mark(sl, __ldg(DR.fo_edge + x), (uint32_t)__ldg(DR.fo_lvl + x) << 4, rv);
                    usync();
                }
                fr_begin = rend;
            }
        }
    }
    if (acc0) atomicAdd(q.counters_light + 0, acc0);
    if (acc1) atomicAdd(q.counters_light + 1, acc1);
    if (acc2) atomicAdd(q.counters_heavy + 0, acc2);
    if (acc3) atomicAdd(q.counters_heavy + 1, acc3);
}

// Everything the packed kernel reads of a net in one 128-byte record, a thread per net. On the host
// the records of 22k nets took 0.56 ms of 3.6 for loading the design, and their copy 0.1.
__global__ void __launch_bounds__(128)
records_kernel(const __grid_constant__ DevDesign D, uint4 *__restrict__ out) {
    const uint32_t e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= D.n_net) return;
    const uint32_t IR = D.I + D.R;
    uint4 d = make_uint4(0, 0, 0, 0), ni = D.netinfo[e];
    uint32_t c[8], l[8], end = 0;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
        const bool on = k < ni.y - ni.x;
        c[k] = on ? D.fo_edge[ni.x + k] : 0u;
        l[k] = on ? (uint32_t)(uint16_t)(D.fo_lvl[ni.x + k] << 4) : 0u;
    }
    if (e >= IR) {
        d = D.desc[e - IR];
        const uint32_t op = meta_op(d.w);
        if (op == OP_MUX2) d = make_uint4(d.y, d.z, d.x, d.w);
        const int no = n_operands(op);
        d.w |= (no >= 3 ? 7u : no == 2 ? 3u : no == 1 ? 1u : 0u) << 4;
        switch (op) {
        case OP_AND: d.w |= PM_A; break;
        case OP_OR: d.w |= PM_A | PM_B | PM_C; break;
        case OP_XOR: d.w |= PM_B | PM_C; break;
        case OP_NOT: d.w |= PM_B | PM_D; break;
        case OP_ADD: case OP_SUB: d.w |= PM_SUM; break;
        case OP_EQ: case OP_LT: d.w |= PM_CMP; break;
        case OP_MUX2: d.w |= PM_C; break;
        case OP_SHL: d.w |= PM_B | PM_LEFT; break;
        case OP_CONCAT: d.w |= PM_B | PM_C | PM_LEFT; break;
        case OP_SHR: case OP_SLICE: d.w |= PM_B; break;
        default: break;
        }
        end = D.lvl_start[D.node_level[e - IR] + 1];
    }
    if (ni_nreg(ni.w) == 1) ni.z = D.dreg_rec[ni.z];
    uint4 *const r = out + (size_t)e * 8;
    r[0] = d;
    r[1] = ni;
    r[2] = make_uint4(c[0], c[1], c[2], c[3]);
    r[3] = make_uint4(c[4], c[5], c[6], c[7]);
    r[4] = make_uint4(l[0] | l[1] << 16, l[2] | l[3] << 16, l[4] | l[5] << 16, l[6] | l[7] << 16);
    r[5] = make_uint4(end, 0, 0, 0);
    r[6] = r[7] = make_uint4(0, 0, 0, 0);
}

cudaError_t launch_records(const DevDesign &d, uint4 *rec, cudaStream_t stream) {
    if (!d.n_net) return cudaSuccess;
    records_kernel<<<(d.n_net + 127) / 128, 128, 0, stream>>>(d, rec);
    return cudaGetLastError();
}

// The tiers: lanes per fault, table entries per lane.
constexpr int TIER_LPS[PACK_TIERS] = {1, 8, 32, 256}, TIER_TPL[PACK_TIERS] = {8, 16, 16, 16};

template <bool MULTI>
static const void *pack_fn(int tier) {
    return tier == 0 ? (const void *)pack_kernel<TIER_LPS[0], TIER_TPL[0], PACK_RPL, MULTI>
         : tier == 1 ? (const void *)pack_kernel<TIER_LPS[1], TIER_TPL[1], PACK_RPL, MULTI>
         : tier == 2 ? (const void *)pack_kernel<TIER_LPS[2], TIER_TPL[2], PACK_RPL, MULTI>
                     : (const void *)pack_kernel<TIER_LPS[3], TIER_TPL[3], PACK_RPL, MULTI>;
}

size_t pack_smem_bytes(int tier, int warps) {
    return TIER_LPS[tier] > 32 ? pack_unit_bytes(TIER_LPS[tier], TIER_TPL[tier], PACK_RPL)
                               : warps * pack_unit_bytes(32, TIER_TPL[tier], PACK_RPL);
}

cudaError_t launch_pack(int tier, bool multi, const DevDesign *d_designs, const DevDesign &d0, DevFaults f,
                        const PackArgs &q, int warps, int grid, cudaStream_t stream) {
    const void *fn = multi ? pack_fn<true>(tier) : pack_fn<false>(tier);
    const size_t smem = pack_smem_bytes(tier, warps);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[] = {(void *)&d_designs, (void *)&d0, (void *)&f, (void *)&q};
    return cudaLaunchKernel(fn, dim3(grid), dim3(TIER_LPS[tier] > 32 ? TIER_LPS[tier] : warps * 32), args, smem, stream);
}

}  // namespace rtlfs
