// rtlfs_static.cu -- allocation-free fault simulation: kernels with a warp, or for very large
// designs a thread, per fault, whose scratch lives in one file-scope device array instead of
// memory obtained from cudaMalloc.
//
// Who needs it: callers that cannot obtain device memory from cudaMalloc where they run --
// a process whose device memory is owned by another allocator (a framework's caching pool
// that has reserved the GPU, which this library cannot call into), and latency-critical
// paths that cannot afford an allocation or the device-wide synchronisation cudaMalloc
// and cudaFree can imply. Such a caller passes its own device buffers for the faults and
// the results; the design and its good trace come from a context that was set up earlier.
//
// The array below is part of the library image: every GPU that loads the library keeps
// its 64 MiB until the process exits. Every call shares it, it keeps the contents the last
// call left, and two calls whose work overlaps on the GPU race on it.
#include "rtlfs_device.h"
#include "rtlfs_static.h"

#include <algorithm>
#include <mutex>

namespace rtlfs {

static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

// Host side: the device address of g_static_scratch, looked up once per device. In host
// code the name g_static_scratch is only a host-side stand-in, not a device address.
cudaError_t static_scratch_address(int device, void **out) {
    static std::mutex mu;
    static void *addr[STATIC_MAX_DEVICES] = {};
    if (device < 0 || device >= STATIC_MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[device]) {
        int prev = 0;
        cudaError_t e = cudaGetDevice(&prev);
        if (e != cudaSuccess) return e;
        e = cudaSetDevice(device);
        if (e != cudaSuccess) return e;
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        cudaSetDevice(prev);
        if (e != cudaSuccess) return e;
        addr[device] = p;
    }
    *out = addr[device];
    return cudaSuccess;
}

// A fault that no context ever checked: false, with the result that says so, if it is out of range.
__device__ __forceinline__ bool static_site(const DevDesign &D, const uint32_t *ext2int, const StaticFault &fx, uint32_t *err,
                                            StaticResult *out, uint32_t *site) {
    out->cycle = -1;
    out->port = -1;
    out->detected = 0;
    out->reserved[0] = out->reserved[1] = out->reserved[2] = 0;
    if (fx.net < D.n_net && fx.stuck <= 1) {
        *site = ext2int[fx.net];
        if (fx.bit < D.net_w[*site]) return true;
    }
    atomicOr(err, 1u);
    out->detected = 254;
    return false;
}

// Shared memory of one warp of static_kernel.
struct StaticWarp {
    uint32_t *bm, *top;      // dirty nodes, and the words of bm that hold one
    uint32_t *df, *dtop;     // nets that differ this cycle, and the words of df that hold one
    uint32_t *n_new;         // registers latched with a difference
    uint16_t *list;          // [1024] a level's dirty nodes in 32 words of bm
};

__host__ __device__ inline uint32_t static_words(uint32_t n) { return (n + 31) / 32; }
__host__ __device__ inline size_t static_warp_bytes(uint32_t n_node, uint32_t n_net) {
    const uint32_t a = static_words(n_node), b = static_words(n_net);
    return 4 * ((size_t)a + static_words(a) + b + static_words(b) + 4) + 2048;
}

// One warp per fault; a warp takes the next fault when it is done with one. A cycle in which the
// machine has no register difference and the site's good bit is the stuck value is skipped
// (32 cycles a look); in the others the warp takes the lowest level that has dirty nodes, its
// lanes a node each, until none is left. Which nets differ is a bitmap in shared memory, so an
// operand is one load, of the faulty value (in the slot's part of the scratch array) or of the
// good one. What bounds it is the chain of a level, some 1000 cycles: the search for its nodes,
// their 128-byte records, their operands. 1500 faults of 1200 nodes over 300 cycles: 11.6 ms with a
// thread per fault and its heap of dirty nodes in the scratch array, 3.4 so. (One to four faults: 0.2 to
// 1.6 times a thread's time; an idle fault's cycles are skipped, a busy one's level costs more.)
// THIN: for designs with a few nodes per level, where a level's search is most of its cost. 20 and
// 2000 faults of a 1000-level chain over 50 cycles took 56 and 64 ms without the walk (a thread per
// fault: 44 and 49), 18 and 22 with it. Elsewhere it costs 3% (1200 nodes), so it is left out there.
template <bool THIN>
__global__ void __launch_bounds__(128)
static_kernel(const DevDesign *__restrict__ designs, uint32_t design, const StaticFault *__restrict__ faults,
              StaticResult *results, uint32_t n_faults, unsigned char *arena, StaticLayout L) {
    extern __shared__ __align__(16) unsigned char ssm[];
    constexpr uint32_t FULL = 0xFFFFFFFFu;
    const DevDesign &D = designs[design];
    const uint32_t I = D.I, IR = D.I + D.R, T = D.T, n_net = D.n_net, lane = threadIdx.x & 31u;
    const uint32_t nw = static_words(D.N), nt = static_words(nw), dw = static_words(n_net), dt = static_words(dw);
    const uint32_t slot = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    StaticWarp m;
    m.bm = reinterpret_cast<uint32_t *>(ssm + (threadIdx.x >> 5) * static_warp_bytes(D.N, n_net));
    m.top = m.bm + nw;
    m.df = m.top + nt;
    m.dtop = m.df + dw;
    m.n_new = m.dtop + dt;
    m.list = reinterpret_cast<uint16_t *>(m.n_new + 4);
    for (uint32_t i = lane; i < nw + nt + dw + dt + 1; i += 32) m.bm[i] = 0u;
    __syncwarp();
    const uint64_t *__restrict__ const gcol = D.gcol;
    const uint4 *__restrict__ const rec = D.rec;
    const uint32_t *ext2int = reinterpret_cast<const uint32_t *>(arena + L.ext2int_off);
    uint32_t *const err = reinterpret_cast<uint32_t *>(arena + L.err_off), *const head = err + 1;
    unsigned char *const base = arena + L.thread_off + (size_t)slot * L.per_thread;
    uint64_t *const val = reinterpret_cast<uint64_t *>(base), *const regv = val + n_net;
    uint32_t *const regr = reinterpret_cast<uint32_t *>(regv + 2 * (size_t)L.sreg);

    for (;;) {
        uint32_t fi = 0;
        if (lane == 0) fi = atomicAdd(head, 1u);
        fi = __shfl_sync(FULL, fi, 0);
        if (fi >= n_faults) return;
        const StaticFault fx = faults[fi];
        StaticResult out;
        uint32_t site = 0;
        if (!static_site(D, ext2int, fx, err, &out, &site)) {
            if (lane == 0) results[fi] = out;
            continue;
        }
        const uint64_t bm1 = 1ull << fx.bit;
        const bool sv = fx.stuck != 0;
        auto force = [&](uint64_t x) { return sv ? (x | bm1) : (x & ~bm1); };
        const uint64_t *const scol = gcol + (size_t)site * T;
        uint32_t nreg = 0, cur = 0, t = 0;
        while (t < T) {
            if (nreg == 0) {   // the next cycle in which the fault acts
                uint32_t hit = 0;
                for (; t < T; t += 32) {
                    const bool on = t + lane < T && force(__ldg(scol + min(t + lane, T - 1))) != __ldg(scol + min(t + lane, T - 1));
                    hit = __ballot_sync(FULL, on);
                    if (hit) break;
                }
                if (!hit) break;
                t += __ffs((int)hit) - 1;
            }
            const uint32_t nb = cur ^ 1u;
            uint32_t port = NI_NO_PORT;
            auto mark = [&](uint32_t n) {
                const uint32_t w = n >> 5;
                atomicOr(m.bm + w, 1u << (n & 31u));
                atomicOr(m.top + (w >> 5), 1u << (w & 31u));
            };
            // where a net that differs is seen: its port and latches (ni: its netinfo)
            auto observe = [&](uint32_t net, uint64_t v, uint64_t g, uint4 ni) {
                port = min(port, ni_port(ni.w));
                uint32_t nl = ni_nreg(ni.w);
                if (nl == 255u) nl = D.dreg_off[net + 1] - ni.z;
                for (uint32_t e = 0; e < nl; ++e) {   // a single one is in the record
                    const uint32_t rr = nl == 1 ? ni.z : __ldg(D.dreg_rec + ni.z + e);
                    const uint64_t wm = wmask(rr >> 25);
                    if ((v & wm) == (g & wm)) continue;
                    const uint32_t k = atomicAdd(m.n_new, 1u);
                    regr[nb * L.sreg + k] = rr & 0x1FFFFFFu;
                    regv[nb * L.sreg + k] = v & wm;
                }
            };
            // and its value and consumers
            auto keep = [&](uint32_t net, uint64_t v, uint64_t g, uint4 ni, const uint4 *r) {
                observe(net, v, g, ni);
                val[net] = v;
                const uint32_t w = net >> 5;
                atomicOr(m.df + w, 1u << (net & 31u));
                atomicOr(m.dtop + (w >> 5), 1u << (w & 31u));
                const uint32_t nf = ni.y - ni.x;
                if (nf <= 8) {
                    const uint4 e0 = r[2], e1 = r[3];
                    const uint32_t e[8] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
#pragma unroll
                    for (uint32_t k = 0; k < 8; ++k)
                        if (k < nf) mark((e[k] & (PACK_NETS - 1)) - IR);
                } else {
                    for (uint32_t e = ni.x; e < ni.y; ++e) mark(__ldg(D.fo_idx + e));
                }
            };
            bool seeded = false;
            for (uint32_t k = lane; k < nreg; k += 32) {
                const uint32_t net = I + regr[cur * L.sreg + k];
                uint64_t qv = regv[cur * L.sreg + k];
                if (net == site) { qv = force(qv); seeded = true; }
                const uint64_t g = __ldg(gcol + (size_t)net * T + t);
                if (qv != g) keep(net, qv, g, __ldg(rec + 8 * (size_t)net + 1), rec + 8 * (size_t)net);
            }
            seeded = __any_sync(FULL, seeded);
            if (lane == 0) {
                const uint64_t g = __ldg(scol + t);
                if (force(g) != g) {   // else the site's own evaluation or register decides
                    if (site >= IR) mark(site - IR);
                    else if (!seeded) keep(site, force(g), g, __ldg(rec + 8 * (size_t)site + 1), rec + 8 * (size_t)site);
                }
            }
            __syncwarp();
            uint32_t tp = 0;   // no word of top before it is set
            for (;;) {
                uint32_t word = FULL;   // the first word with a dirty node
                for (; tp < nt; tp += 32) {
                    const uint32_t x = tp + lane < nt ? m.top[tp + lane] : 0u;
                    const uint32_t any = __ballot_sync(FULL, x != 0u);
                    if (!any) continue;
                    const int src = __ffs((int)any) - 1;
                    word = (tp + src) * 32 + __ffs((int)__shfl_sync(FULL, x, src)) - 1;
                    break;
                }
                if (word == FULL) break;
                // Each lane reads and clears a word of its own of the 32 looked at; the first one's
                // lowest node n0 names the level.
                const uint32_t wi = word + lane;
                const uint32_t all = wi < nw ? m.bm[wi] : 0u;
                const uint32_t w0 = __shfl_sync(FULL, all, 0), n0 = word * 32 + __ffs((int)w0) - 1;
                const uint4 *const r0 = rec + 8 * (size_t)(IR + n0);
                const uint32_t end = __ldg(&r0[5].x);
                auto operand = [&](uint4 d, uint32_t x, uint32_t bit) -> uint64_t {
                    if (!(d.w & bit)) return 0ull;
                    return m.df[x >> 5] >> (x & 31u) & 1u ? val[x] : __ldg(gcol + (size_t)x * T + t);
                };
                if constexpr (THIN) {
                    // Alone in its level: the next dirty node n1 is one of a later level, or none of these
                    // words. One lane walks on while what differs has a single consumer before n1: its value
                    // stays in a register, and the consumer's record is on its way while the node's
                    // operands are.
                    const uint32_t rest = lane == 0 ? all & (all - 1) : all, more = __ballot_sync(FULL, rest != 0u);
                    const uint32_t src = more ? __ffs((int)more) - 1 : 0u;
                    const uint32_t wr = __shfl_sync(FULL, rest, src);
                    const uint32_t n1 = more ? (word + src) * 32 + __ffs((int)wr) - 1 : (word + 32) * 32;
                    if (n1 >= end) {
                        if (lane == 0) {
                            m.bm[word] = w0 & (w0 - 1);
                            if (m.bm[word] == 0u) atomicAnd(m.top + (word >> 5), ~(1u << (word & 31u)));
                            uint4 d = __ldg(r0), ni = __ldg(r0 + 1), e = __ldg(r0 + 2);
                            uint64_t g = __ldg(gcol + (size_t)(IR + n0) * T + t);
                            uint32_t net = IR + n0, fed = 0;   // fed: the slots that `fv` feeds, from bit 27
                            uint64_t fv = 0;
                            for (;;) {
                                const uint32_t nx = e.x & (PACK_NETS - 1);
                                const bool on = ni.y - ni.x == 1 && nx < IR + n1;
                                const size_t to = on ? nx : net;   // no condition on the loads: their values are not merged
                                const uint4 d2 = __ldg(rec + 8 * to), ni2 = __ldg(rec + 8 * to + 1), e2 = __ldg(rec + 8 * to + 2);
                                const uint64_t g2 = __ldg(gcol + to * T + t);
                                const uint64_t x = fed >> 27 & 1u ? fv : operand(d, d.x, 1u << 4), y = fed >> 28 & 1u ? fv : operand(d, d.y, 1u << 5);
                                const uint64_t s = fed >> 29 & 1u ? fv : operand(d, d.z, 1u << 6);
                                uint64_t v = pack_eval(d, x, y, s);
                                if (net == site) v = force(v);
                                if (v == g) break;
                                if (!on) { keep(net, v, g, ni, rec + 8 * (size_t)net); break; }
                                observe(net, v, g, ni);
                                fed = e.x;
                                fv = v;
                                net = nx;
                                d = d2; ni = ni2; e = e2; g = g2;
                            }
                        }
                        __syncwarp();
                        continue;
                    }
                }
                // its dirty nodes into the list
                uint32_t bits = 0, at = 0;
                if (wi < nw && wi * 32 < end) {
                    bits = end - wi * 32 >= 32 ? all : all & ((1u << (end - wi * 32)) - 1u);
                    if (bits) {
                        m.bm[wi] = all ^ bits;
                        if (all == bits) atomicAnd(m.top + (wi >> 5), ~(1u << (wi & 31u)));
                    }
                }
                const uint32_t mine = __popc(bits);
                uint32_t sum = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(FULL, sum, o);
                    if (lane >= (uint32_t)o) sum += x;
                }
                at = sum - mine;
                const uint32_t total = __shfl_sync(FULL, sum, 31);
                for (; bits; bits &= bits - 1) m.list[at++] = (uint16_t)(lane * 32 + __ffs((int)bits) - 1);
                __syncwarp();
                for (uint32_t k = lane; k < total; k += 32) {
                    const uint32_t net = IR + word * 32 + m.list[k];
                    const uint4 *const r = rec + 8 * (size_t)net;
                    const uint4 d = __ldg(r), ni = __ldg(r + 1);
                    const uint64_t g = __ldg(gcol + (size_t)net * T + t);
                    const uint64_t x = operand(d, d.x, 1u << 4), y = operand(d, d.y, 1u << 5), s = operand(d, d.z, 1u << 6);
                    uint64_t v = pack_eval(d, x, y, s);
                    if (net == site) v = force(v);
                    if (v != g) keep(net, v, g, ni, r);
                }
                __syncwarp();
            }
            for (uint32_t i = 0; i < dt; i += 32) {   // clear df: all lanes share a word of dtop
                const uint32_t x = i + lane < dt ? m.dtop[i + lane] : 0u;
                for (uint32_t any = __ballot_sync(FULL, x != 0u); any; any &= any - 1) {
                    const int src = __ffs((int)any) - 1;
                    if (__shfl_sync(FULL, x, src) >> lane & 1u) m.df[(i + src) * 32 + lane] = 0u;
                }
                if (x) m.dtop[i + lane] = 0u;
            }
            port = __reduce_min_sync(FULL, port);
            nreg = *(volatile uint32_t *)m.n_new;
            __syncwarp();
            if (lane == 0) *m.n_new = 0u;
            __syncwarp();
            if (port != NI_NO_PORT) {
                out.detected = 1;
                out.cycle = (int32_t)t;
                out.port = (int32_t)port;
                break;
            }
            cur = nb;
            ++t;
        }
        if (lane == 0) results[fi] = out;
    }
}

int static_warps(uint32_t n_node, uint32_t n_net) {
    const size_t one = static_warp_bytes(n_node, n_net);
    return (int)std::min<size_t>(4, STATIC_SMEM / one);
}

cudaError_t launch_static(const DevDesign *d_designs, uint32_t design, uint32_t n_node, uint32_t n_levels, uint32_t n_net, const void *faults,
                          void *results, uint32_t n_faults, uint32_t blocks, uint32_t warps, void *arena, StaticLayout L, cudaStream_t stream) {
    const size_t smem = warps * static_warp_bytes(n_node, n_net);
    // chains: where levels have a few nodes, one lane walks along them
    const auto fn = n_node <= 8ull * n_levels ? static_kernel<true> : static_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    fn<<<blocks, warps * 32, smem, stream>>>(d_designs, design, (const StaticFault *)faults, (StaticResult *)results,
                                                        n_faults, (unsigned char *)arena, L);
    return cudaGetLastError();
}

// The form for designs whose bitmaps do not fit in a warp's shared memory (static_warps is 0).
// One thread per fault of this wave; the wave's scratch is carved from the static array:
// [ext2int: n_net u32][error word][per thread: values u64, stamps u32, queued u32, heap u32,
// register diffs 2 x (u32 reg, u64 value)]. Stamps must be zero before the wave.
__global__ void __launch_bounds__(128)
plain_static_kernel(const DevDesign *__restrict__ designs, uint32_t design,
                    const StaticFault *__restrict__ faults, StaticResult *results,
                    uint32_t first, uint32_t count, unsigned char *arena, StaticLayout L) {
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid >= count) return;
    const uint32_t fi = first + tid;
    const DevDesign &D = designs[design];
    const uint32_t I = D.I, IR = D.I + D.R, T = D.T;
    const uint64_t *gcol = D.gcol;
    const uint32_t *ext2int = reinterpret_cast<const uint32_t *>(arena + L.ext2int_off);
    uint32_t *err = reinterpret_cast<uint32_t *>(arena + L.err_off);
    unsigned char *base = arena + L.thread_off + (size_t)tid * L.per_thread;
    uint64_t *fval = reinterpret_cast<uint64_t *>(base);
    uint64_t *regv = fval + L.sn;
    uint32_t *stamp = reinterpret_cast<uint32_t *>(regv + 2 * (size_t)L.sreg);
    uint32_t *qst = stamp + L.sn;
    uint32_t *hp = qst + L.snode;
    uint32_t *regr = hp + L.snode;

    const StaticFault fx = faults[fi];
    StaticResult out;
    uint32_t site = 0;
    if (!static_site(D, ext2int, fx, err, &out, &site)) {
        results[fi] = out;
        return;
    }
    const uint64_t bm = 1ull << fx.bit;
    const bool sv = fx.stuck != 0;
    auto force = [&](uint64_t x) { return sv ? (x | bm) : (x & ~bm); };
    uint32_t nreg = 0, cur = 0, epoch = 0;
    for (uint32_t t = 0; t < T; ++t) {
        ++epoch;
        const uint32_t nb = cur ^ 1u;
        uint32_t nh = 0, nreg_new = 0, minport = NO_PORT;
        auto push = [&](uint32_t x) {
            if (qst[x] == epoch) return;
            qst[x] = epoch;
            uint32_t i = nh++;
            while (i > 0) {
                const uint32_t p = (i - 1) >> 1;
                if (hp[p] <= x) break;
                hp[i] = hp[p];
                i = p;
            }
            hp[i] = x;
        };
        auto pop = [&]() -> uint32_t {
            const uint32_t top = hp[0];
            const uint32_t x = hp[--nh];
            uint32_t i = 0;
            for (;;) {
                uint32_t c = 2 * i + 1;
                if (c >= nh) break;
                if (c + 1 < nh && hp[c + 1] < hp[c]) ++c;
                if (x <= hp[c]) break;
                hp[i] = hp[c];
                i = c;
            }
            if (nh > 0) hp[i] = x;
            return top;
        };
        auto keep = [&](uint32_t net, uint64_t v, uint64_t g) {
            stamp[net] = epoch;
            fval[net] = v;
            const uint32_t p = D.outport[net];
            minport = p < minport ? p : minport;
            for (uint32_t e = D.fo_off[net]; e < D.fo_off[net + 1]; ++e) push(D.fo_idx[e]);
            for (uint32_t e = D.dreg_off[net]; e < D.dreg_off[net + 1]; ++e) {
                const uint32_t r = D.dreg_idx[e];
                const uint64_t wm = wmask(D.net_w[I + r]);
                if ((v & wm) != (g & wm)) {
                    regr[nb * L.sreg + nreg_new] = r;
                    regv[nb * L.sreg + nreg_new] = v & wm;
                    ++nreg_new;
                }
            }
        };
        auto lookup = [&](uint32_t x) -> uint64_t {
            return stamp[x] == epoch ? fval[x] : gcol[(size_t)x * T + t];
        };
        bool site_seeded = false;
        for (uint32_t k = 0; k < nreg; ++k) {
            const uint32_t net = I + regr[cur * L.sreg + k];
            uint64_t qv = regv[cur * L.sreg + k];
            if (net == site) { qv = force(qv); site_seeded = true; }
            const uint64_t g = gcol[(size_t)net * T + t];
            if (qv != g) keep(net, qv, g);
        }
        if (site < IR && !site_seeded) {
            const uint64_t g = gcol[(size_t)site * T + t];
            const uint64_t fv = force(g);
            if (fv != g) keep(site, fv, g);
        }
        if (site >= IR) push(site - IR);
        while (nh > 0) {
            const uint32_t n = pop();
            const uint4 d = D.desc[n];
            const int no = n_operands(meta_op(d.w));
            uint64_t a = 0, b = 0, c = 0;
            if (no >= 1) a = lookup(d.x);
            if (no >= 2) b = lookup(d.y);
            if (no >= 3) c = lookup(d.z);
            const uint32_t net = IR + n;
            uint64_t v = eval_op(d, a, b, c);
            if (net == site) v = force(v);
            const uint64_t g = gcol[(size_t)net * T + t];
            if (v != g) keep(net, v, g);
        }
        if (minport != NO_PORT) {
            out.detected = 1;
            out.cycle = (int32_t)t;
            out.port = (int32_t)minport;
            break;
        }
        nreg = nreg_new;
        cur = nb;
    }
    results[fi] = out;
}

cudaError_t launch_plain_static(const DevDesign *d_designs, uint32_t design, const void *faults,
                                void *results, uint32_t first, uint32_t count, void *arena,
                                StaticLayout L, cudaStream_t stream) {
    if (!count) return cudaSuccess;
    plain_static_kernel<<<(count + 127) / 128, 128, 0, stream>>>(
        d_designs, design, (const StaticFault *)faults, (StaticResult *)results, first, count,
        (unsigned char *)arena, L);
    return cudaGetLastError();
}

}  // namespace rtlfs
