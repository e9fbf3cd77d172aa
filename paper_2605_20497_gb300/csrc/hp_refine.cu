// hp_refine.cu -- one level of refinement (Sec. VI): Theta repetitions of
//   pins(p,e) lists  -> move proposal by gain (Eq. 13, Sec. VI-B)
//   -> sort (p_s asc, gain desc, node asc) -> chaining (Sec. VI-C)
//   -> chain order -> in-sequence gains (Eq. 14-15, exact change of
//   connectivity) -> event-based validity of every prefix (Sec. VI-D)
//   -> apply the best valid prefix.
// pins(p,e) is kept as a short list per hyperedge, sorted by partition id, at
// the hyperedge's own pin segment: (p, pins(p,e), pins_in(p,e)).
#include <cuda_runtime.h>

#include <cstring>

#include <algorithm>
#include <climits>
#include <initializer_list>

#include "hp_cluster.cuh"
#include "hp_internal.cuh"

namespace hp {

static int grid_of(int64_t n, int block) {
    int64_t g = cdiv(n, block);
    int64_t cap = (int64_t)num_sms() * 32;
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}
#define GRID_STRIDE(i, n) \
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

struct Plist {
    int32_t *p = nullptr, *cnt = nullptr, *cin = nullptr;  // [np]
    int32_t *lam = nullptr;                                // [e] entries per hyperedge
};

// slot of key x in a table of mask + 1 (a power of two, >= 2) slots: the top
// bits of a Fibonacci product, so that keys with equal low bits spread out
__device__ __forceinline__ uint32_t hslot(int32_t x, uint32_t mask) {
    return mask ? ((uint32_t)x * 0x9E3779B1u) >> __clz(mask) : 0u;
}

template <int G> __device__ __forceinline__ void gsync() {
    if (G == 32) __syncwarp();
    else __syncthreads();
}

// ---------------------------------------------------------------- pins(p,e)
// One group of G threads builds the sorted list of hyperedge e.  Its table
// of `cap` slots (keys/cnt/cin) is clean (keys -1, counters 0) on entry and
// is left clean; the entry buffers hold >= |e| slots.  Both live in shared
// or global memory private to the group.  Optionally adds D(p) (distinct
// inbound hyperedges per part) and saving(v) for the hyperedge's pins (v
// alone in its part, |e| >= 2).
template <int G>
__device__ void plist_edge(int32_t e, int gt, const int32_t *off, const int32_t *pin, const int32_t *nsrc,
                           const int32_t *w, const int32_t *rho, int32_t *keys, int32_t *tc, int32_t *tci, uint32_t cap,
                           int32_t *ent_s, int32_t *ent_p, int32_t *ent_c, int32_t *ent_ci, int32_t *g_cnt, Plist PL,
                           int32_t *D, long long *saving) {
    const uint32_t mask = cap - 1;
    const int32_t a = off[e], b = off[e + 1], dst0 = a + nsrc[e];
    if (gt == 0) *g_cnt = 0;
    gsync<G>();
    for (int64_t j = (int64_t)a + gt; j < b; j += G) {
        int32_t p = rho[pin[j]];
        uint32_t h = hslot(p, mask);
        for (uint32_t probe = 0; probe < cap; probe++) {
            int32_t k = ((volatile int32_t *)keys)[h];
            if (k == -1) {
                int32_t old = atomicCAS(&keys[h], -1, p);
                if (old == -1) {
                    ent_s[atomicAdd(g_cnt, 1)] = (int32_t)h;
                    k = p;
                } else {
                    k = old;
                }
            }
            if (k == p) {
                atomicAdd(&tc[h], 1);
                if (j >= dst0) atomicAdd(&tci[h], 1);
                break;
            }
            h = (h + 1) & mask;
        }
    }
    gsync<G>();
    const int32_t lam = *(volatile int32_t *)g_cnt;
    if (saving && b - a >= 2) {
        const long long we = w[e];
        for (int64_t j = (int64_t)a + gt; j < b; j += G) {
            int32_t v = pin[j], p = rho[v];
            uint32_t h = hslot(p, mask);
            for (uint32_t probe = 0; probe < cap && keys[h] != p; probe++) h = (h + 1) & mask;
            if (keys[h] == p && tc[h] == 1) atomicAdd((unsigned long long *)&saving[v], (unsigned long long)we);
        }
    }
    for (int32_t i = gt; i < lam; i += G) {
        int32_t h = ent_s[i];
        ent_p[i] = keys[h];
        ent_c[i] = tc[h];
        ent_ci[i] = tci[h];
    }
    gsync<G>();
    for (int32_t i = gt; i < lam; i += G) {
        int32_t p = ent_p[i], r = 0;
        for (int32_t k = 0; k < lam; k++) r += ent_p[k] < p;
        PL.p[a + r] = p;
        PL.cnt[a + r] = ent_c[i];
        PL.cin[a + r] = ent_ci[i];
        if (D && ent_ci[i] > 0) atomicAdd(&D[p], 1);
        int32_t h = ent_s[i];
        keys[h] = -1;
        tc[h] = 0;
        tci[h] = 0;
    }
    if (gt == 0) PL.lam[e] = lam;
    gsync<G>();
}

constexpr int PLW_T = 128;  // warp-per-edge kernel: 4 warps
constexpr int32_t MID_SPLIT = 128;   // warp-tier hyperedges up to this size get small tables

// edges with |e| <= small_max, one warp each, tables in shared memory
__global__ void __launch_bounds__(PLW_T) k_plist_small(const int32_t *off, const int32_t *pin, const int32_t *nsrc,
                                                       const int32_t *w, const int32_t *rho, int32_t e,
                                                       const int32_t *list, int32_t small_max, uint32_t cap, Plist PL,
                                                       int32_t *D, long long *saving, int32_t skip_below,
                                                       int32_t skip_above) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) int32_t sm[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // table of cap slots; entry buffers of cap / 2 >= lambda(e) entries
    const int per = 5 * (int)cap + 1, ent = (int)cap / 2;
    int32_t *base = sm + wid * per;
    int32_t *keys = base, *tc = base + cap, *tci = base + 2 * cap;
    int32_t *es = base + 3 * cap, *ep = es + ent, *ec = ep + ent, *eci = ec + ent, *gcnt = eci + ent;
    for (uint32_t i = lane; i < cap; i += 32) {
        keys[i] = -1;
        tc[i] = 0;
        tci[i] = 0;
    }
    __syncwarp();
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    // all hyperedges up to small_max pins, or the given list (count e) skipping
    // the ones of at most skip_below or more than skip_above pins
    for (int64_t i = warp; i < e; i += nw) {
        const int32_t ed = list ? list[i] : (int32_t)i;
        const int32_t sz = off[ed + 1] - off[ed];
        if ((!list && sz > small_max) || sz <= skip_below || sz > skip_above) continue;
        plist_edge<32>(ed, lane, off, pin, nsrc, w, rho, keys, tc, tci, cap, es, ep, ec, eci, gcnt, PL, D, saving);
    }
}

// The same for up to PB_PARTS parts, a warp per hyperedge of the list, of at
// most 512 pins: counters indexed by part (pins in the low half word, inbound
// pins in the high one) and a bit per part in use, both in shared memory.  The
// bits give the entries in ascending part order, so nothing is probed, ranked
// or sorted: a lane owns 32 parts, and a warp prefix sum over the lanes' bit
// counts places its entries.  D(p) is summed per CTA.  Bound by the gather of
// rho behind the pins.  Against the hashed form above: 1M Gaussian net 1.01 ->
// 0.89 s a call, 16,384-node random net 151 -> 140 ms, 20k irregular net 68.0
// -> 64.7 ms.
constexpr int PP_T = 256;
constexpr int32_t PB_PARTS = 1024;   // most parts with a bit row (here, and of the gains from part bits)
__host__ __device__ inline size_t plist_parts_smem(int32_t nparts) {
    const size_t words = (size_t)(nparts + 31) / 32;
    return 4 * ((PP_T / 32) * (words * 32 + 32) + words * 32);
}
// The applied moves of the repetition before: node v moved when its sequence
// position lies below *applied, from the part of its move.
struct Applied {
    const int32_t *mvpos, *seqmove, *src, *applied;
    __device__ __forceinline__ int32_t old_part(int32_t v, int32_t now, int32_t len) const {
        const int32_t k = mvpos[v];
        return k >= 0 && k < len ? src[seqmove[k]] : now;
    }
};
// UPDATE: the list holds the hyperedges that may have a pin among the applied
// moves (*count_p of them); the ones that do take their old contributions to
// D(p) and saving(v) back, read off their old pins list, before they are
// rebuilt; their pins and new list entries are counted into acc[0] and acc[1].
template <bool UPDATE>
__global__ void __launch_bounds__(PP_T) k_plist_parts(const int32_t *off, const int32_t *pin, const int32_t *nsrc,
                                                      const int32_t *w, const int32_t *rho, const int32_t *list,
                                                      int32_t count, const int32_t *count_p, Applied M, int32_t nparts,
                                                      Plist PL, int32_t *D, long long *saving,
                                                      unsigned long long *acc) {
    HP_KERNEL_ENTER();
    int32_t len = 0;
    unsigned long long n_pins = 0, n_ent = 0;
    if (UPDATE) {
        count = *count_p;
        len = *M.applied;
        if ((int64_t)blockIdx.x * (PP_T / 32) >= count) return;
    }
    extern __shared__ __align__(16) uint32_t smw[];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwb = PP_T / 32;
    const int words = (nparts + 31) / 32;
    uint32_t *cnt = smw + wid * (words * 32 + 32), *used = cnt + words * 32;
    uint32_t *s_d = smw + nwb * (words * 32 + 32);
    for (int i = threadIdx.x; i < nwb * (words * 32 + 32) + words * 32; i += PP_T) smw[i] = 0;
    __syncthreads();
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    constexpr int R = 4;   // pins a lane holds at a time
    for (int64_t x = w0; x < count; x += nw) {
        const int32_t e = list[x];
        // (positions within the hyperedge: the level's last pin may be number 2^31 - 2)
        const int32_t a = off[e], sz = off[e + 1] - a, dst0 = nsrc[e];
        const unsigned long long we = (unsigned long long)w[e];
        int32_t vv[R], pp[R];
        auto load = [&](int32_t j0) {
#pragma unroll
            for (int k = 0; k < R; k++) {
                const int32_t j = j0 + 32 * k + lane;
                vv[k] = j < sz ? pin[a + j] : -1;
            }
#pragma unroll
            for (int k = 0; k < R; k++) pp[k] = vv[k] >= 0 ? rho[vv[k]] : 0;
        };
        if (UPDATE) {
            bool moved = false;
            for (int32_t j0 = 0; j0 < sz; j0 += 32 * R) {
                load(j0);
#pragma unroll
                for (int k = 0; k < R; k++) moved |= vv[k] >= 0 && M.old_part(vv[k], pp[k], len) != pp[k];
            }
            if (!__any_sync(FULL, moved)) continue;
            const int32_t lam = PL.lam[e];
            for (int32_t x2 = lane; x2 < lam; x2 += 32) {
                const int32_t p = PL.p[a + x2], ci = PL.cin[a + x2];
                cnt[p] = (uint32_t)PL.cnt[a + x2];
                if (ci > 0) atomicAdd(&s_d[p], 0xffffffffu);
            }
            __syncwarp();
            for (int32_t j0 = 0; j0 < sz; j0 += 32 * R) {
                if (sz > 32 * R) load(j0);
#pragma unroll
                for (int k = 0; k < R; k++)
                    if (vv[k] >= 0 && cnt[M.old_part(vv[k], pp[k], len)] == 1u)
                        atomicAdd((unsigned long long *)&saving[vv[k]], 0ull - we);
            }
            __syncwarp();
            for (int32_t x2 = lane; x2 < lam; x2 += 32) cnt[PL.p[a + x2]] = 0;
            __syncwarp();
        }
        for (int32_t j0 = 0; j0 < sz; j0 += 32 * R) {
            load(j0);
#pragma unroll
            for (int k = 0; k < R; k++)
                if (vv[k] >= 0) {
                    atomicAdd(&cnt[pp[k]], j0 + 32 * k + lane >= dst0 ? 0x10001u : 1u);
                    atomicOr(&used[pp[k] >> 5], 1u << (pp[k] & 31));
                }
        }
        __syncwarp();
        uint32_t mine = used[lane];   // 32 words, those past the parts stay 0
        int32_t at = __popc(mine), inc = at;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(FULL, inc, o);
            if (lane >= o) inc += u;
        }
        at = a + inc - at;
        // a pin alone in its part can be spared a cut
        for (int32_t j0 = 0; j0 < sz; j0 += 32 * R) {
            if (sz > 32 * R) load(j0);
#pragma unroll
            for (int k = 0; k < R; k++)
                if (vv[k] >= 0 && (cnt[pp[k]] & 0xffffu) == 1u) atomicAdd((unsigned long long *)&saving[vv[k]], we);
        }
        __syncwarp();
        for (; mine; mine &= mine - 1, at++) {
            const int32_t p = 32 * lane + __ffs(mine) - 1;
            const uint32_t c = cnt[p];
            cnt[p] = 0;
            PL.p[at] = p;
            PL.cnt[at] = (int32_t)(c & 0xffffu);
            PL.cin[at] = (int32_t)(c >> 16);
            if (c >> 16) atomicAdd(&s_d[p], 1u);
        }
        used[lane] = 0;
        if (lane == 31) {
            PL.lam[e] = inc;
            n_pins += (unsigned long long)sz;
            n_ent += (unsigned long long)inc;
        }
        __syncwarp();
    }
    __shared__ unsigned long long s_acc[2];
    if (UPDATE && threadIdx.x < 2) s_acc[threadIdx.x] = 0;
    __syncthreads();
    for (int32_t p = threadIdx.x; p < nparts; p += PP_T)
        if (s_d[p]) atomicAdd(&D[p], (int32_t)s_d[p]);
    if (UPDATE) {
        if (lane == 31 && n_pins) {
            atomicAdd(&s_acc[0], n_pins);
            atomicAdd(&s_acc[1], n_ent);
        }
        __syncthreads();
        if (threadIdx.x < 2 && s_acc[threadIdx.x]) atomicAdd(&acc[threadIdx.x], s_acc[threadIdx.x]);
    }
}

// edges with |e| > small_max, one CTA each, tables in global memory
__global__ void __launch_bounds__(256) k_plist_big(const int32_t *off, const int32_t *pin, const int32_t *nsrc,
                                                   const int32_t *w, const int32_t *rho, const int32_t *list,
                                                   int32_t count, uint32_t cap, int32_t *gtab, int32_t max_e, Plist PL,
                                                   int32_t *D, long long *saving) {
    HP_KERNEL_ENTER();
    __shared__ int32_t gcnt;
    int32_t *mine = gtab + (int64_t)blockIdx.x * (3 * (int64_t)cap + 4 * (int64_t)max_e);
    int32_t *keys = mine, *tc = mine + cap, *tci = mine + 2 * cap;
    int32_t *es = mine + 3 * cap, *ep = es + max_e, *ec = ep + max_e, *eci = ec + max_e;
    for (uint32_t i = threadIdx.x; i < cap; i += 256) {
        keys[i] = -1;
        tc[i] = 0;
        tci[i] = 0;
    }
    __syncthreads();
    for (int32_t k = blockIdx.x; k < count; k += gridDim.x)
        plist_edge<256>(list[k], threadIdx.x, off, pin, nsrc, w, rho, keys, tc, tci, cap, es, ep, ec, eci, &gcnt, PL,
                        D, saving);
}

__global__ void k_big_edges(const int32_t *off, int32_t e, int32_t small_max, int32_t *list, int32_t *cnt,
                            int32_t *maxe) {
    HP_KERNEL_ENTER();
    GRID_STRIDE(i, (int64_t)e) {
        int32_t sz = off[i + 1] - off[i];
        if (sz > small_max) {
            list[atomicAdd(cnt, 1)] = (int32_t)i;
            atomicMax(maxe, sz);
        }
    }
}

__global__ void k_max_edge(const int32_t *off, int32_t e, int32_t *maxe) {
    HP_KERNEL_ENTER();
    int32_t m = 0;
    GRID_STRIDE(i, (int64_t)e) m = max(m, off[i + 1] - off[i]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(maxe, m);
}

static uint32_t pow2_at_least(int64_t x) {
    uint32_t c = 1;
    while ((int64_t)c < x) c <<= 1;
    return c;
}

static void build_plist(const Level &L, const int32_t *w, const int32_t *rho, int32_t max_e, Plist &PL, int32_t *D,
                        long long *saving, Arena &A) {
    cudaStream_t s = A.stream();
    if (L.e == 0) return;
    const int32_t small_max = std::min<int32_t>(std::max<int32_t>(max_e, 1), 512);
    const uint32_t cap = pow2_at_least(2 * (int64_t)small_max);
    const int per = 5 * (int)cap + 1;
    size_t sm = (size_t)per * 4 * (PLW_T / 32);
    int occ = prepare_kernel((const void *)k_plist_small, PLW_T, sm);
    int grid = (int)std::min<int64_t>(cdiv(L.e, PLW_T / 32), (int64_t)num_sms() * std::max(occ, 1));
    launch_k(k_plist_small, std::max(grid, 1), PLW_T, sm, s, L.off, L.pin, L.nsrc, w, rho, L.e, nullptr, small_max, cap,
             PL, D, saving, 0, INT32_MAX);
    HP_LAUNCH_CHECK();
    if (max_e > small_max) {
        int32_t *list = A.get<int32_t>(L.e);
        int32_t *cnt = A.get<int32_t>(2);
        HPC(cudaMemsetAsync(cnt, 0, 2 * sizeof(int32_t), s));
        launch_k(k_big_edges, grid_of(L.e, 256), 256, 0, s, L.off, L.e, small_max, list, cnt, cnt + 1);
        HP_LAUNCH_CHECK();
        int32_t hc[2];
        fetch_bytes(hc, cnt, sizeof hc, s);
        if (hc[0] > 0) {
            uint32_t bcap = pow2_at_least(2 * (int64_t)hc[1]);
            int nb = std::min<int>(hc[0], num_sms() * 2);
            int32_t *gtab = A.get<int32_t>((int64_t)nb * (3 * (int64_t)bcap + 4 * (int64_t)hc[1]));
            launch_k(k_plist_big, nb, 256, 0, s, L.off, L.pin, L.nsrc, w, rho, list, hc[0], bcap, gtab, hc[1], PL, D,
                     saving);
            HP_LAUNCH_CHECK();
            A.release(gtab);
        }
        A.release(list);
        A.release(cnt);
    }
}

// ---------------------------------------------------------------- objective
__global__ void k_objective(const int32_t *lam, const int32_t *w, int32_t e, unsigned long long *conn,
                            unsigned long long *cutnet) {
    HP_KERNEL_ENTER();
    unsigned long long c = 0, cn = 0;
    GRID_STRIDE(i, (int64_t)e) {
        int32_t l = lam[i];
        c += (unsigned long long)w[i] * (unsigned long long)(l - 1);
        if (l > 1) cn += (unsigned long long)w[i];
    }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_down_sync(0xffffffffu, c, o);
        cn += __shfl_down_sync(0xffffffffu, cn, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(conn, c);
        atomicAdd(cutnet, cn);
    }
}

// ---------------------------------------------------------------- objective in one pass
// Eq. 1 and Eq. 16 of a part vector without pins lists: a warp per hyperedge
// sets a bit per part it meets (shared memory; a lane owns every 32nd word)
// and counts the bits; the next hyperedge's pins are loaded while the
// current one's parts are gathered.  D (optional, up to PB_PARTS parts): adds
// the hyperedge to the distinct inbound count of the parts that hold a
// destination pin.
// CHECK: pins and parts come straight from a caller: a pin outside [0, n) or
// equal to its hyperedge's source raises E_DUP / E_PIN, destinations that do
// not ascend raise PS_UNSORTED (duplicates among them are then to be looked
// for elsewhere), parts outside [0, nparts) are skipped (the caller's check
// reports them), and nothing is read when *pre, left by an earlier kernel, has
// a bit of `stop`.  Bound by the chain pin -> part -> shared memory of each hyperedge.
// Sorting the incidence to find duplicates and building pins lists to count
// their entries took 6.5 ms on the 80 M pins of the 1M Gaussian net; this 0.43.
// BIG: hyperedges of more than PS_BIG pins are left to k_part_scan_big below (a
// warp takes 2.4 us for 128 pins).  A form of its own, which the host takes where
// there are such hyperedges: the test alone made 0.44 ms of the calls above 0.47.
constexpr int PS_T = 256;
constexpr int32_t PS_PARTS = 32768;   // bit rows of up to 4 KB a warp
constexpr uint32_t PS_UNSORTED = 1u << 31, PS_HAS_BIG = 1u << 30;
constexpr int PSB_T = 1024;
// (from 2,048 pins on, 20,000 hyperedges of 3,000 pins take 0.28 ms instead of
// 0.18; from 32,768 on, one of 20,000 takes 0.24 instead of 0.07)
constexpr int32_t PS_BIG = 8192;
inline size_t part_scan_smem(int32_t nparts, bool d) {
    const size_t words = (size_t)cdiv(std::max(nparts, 1), 1024) * 32;
    return 4 * ((PS_T / 32) * words * (d ? 2 : 1) + (d ? words * 32 : 0));
}
template <bool CHECK, bool BIG>
__global__ void __launch_bounds__(PS_T) k_part_scan(const int32_t *off, const int32_t *pin, const int32_t *nsrc,
                                                    const int32_t *w, int32_t e, const int32_t *part, int32_t n,
                                                    int32_t nparts, int32_t *D, unsigned long long *conn,
                                                    unsigned long long *cutnet, const uint32_t *pre, uint32_t stop,
                                                    uint32_t *err) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) uint32_t smw[];
    __shared__ unsigned long long s_sum[2];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int words = (nparts + 1023) / 1024 * 32;   // a multiple of 32
    const int rows = (PS_T / 32) * words * (D ? 2 : 1);
    uint32_t *bm = smw + (size_t)wid * words * (D ? 2 : 1), *bd = bm + words, *s_d = smw + rows;
    if (CHECK && (*pre & stop)) return;
    for (int i = threadIdx.x; i < rows + (D ? words * 32 : 0); i += PS_T) smw[i] = 0;
    if (threadIdx.x < 2) s_sum[threadIdx.x] = 0;
    __syncthreads();
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    constexpr int R = 4;   // pins a lane holds at a time
    uint32_t na = 0, nb = 0;
    int32_t nv[R];
    // (unsigned positions: they may pass 2^31 behind the last pin)
    auto pins_of = [&](uint32_t j0, uint32_t b, int32_t (&v)[R]) {
#pragma unroll
        for (int k = 0; k < R; k++) v[k] = j0 + 32 * k + lane < b ? pin[j0 + 32 * k + lane] : -1;
    };
    if (w0 < e) {
        na = off[w0];
        nb = off[w0 + 1];
        pins_of(na, nb, nv);
    }
    unsigned long long c = 0, cn = 0;
    uint32_t bad = 0;
    for (int64_t i = w0; i < e; i += nw) {
        const uint32_t a = na, b = nb;
        int32_t vv[R];
#pragma unroll
        for (int k = 0; k < R; k++) vv[k] = nv[k];
        if (i + nw < e) {
            na = off[i + nw];
            nb = off[i + nw + 1];
            pins_of(na, nb, nv);
        }
        if (BIG && b - a > PS_BIG) continue;
        const uint32_t dst0 = D ? a + nsrc[i] : a + 1;
        int32_t src = 0, last = INT32_MIN;   // CHECK: the source; the last pin of the chunk before
        if (CHECK) src = __shfl_sync(FULL, vv[0], 0);
        for (uint32_t j0 = a; j0 < b; j0 += 32 * R) {
            if (j0 != a) pins_of(j0, b, vv);
#pragma unroll
            for (int k = 0; k < R; k++) {
                const uint32_t j = j0 + 32 * k + lane;
                const bool in = j < b;
                bool ok = in;
                if (CHECK) {
                    int32_t pv = __shfl_up_sync(FULL, vv[k], 1);
                    if (lane == 0) pv = last;
                    last = __shfl_sync(FULL, vv[k], 31);
                    if (in && (vv[k] < 0 || vv[k] >= n)) {
                        bad |= E_PIN;
                        ok = false;
                    }
                    if (in && j > a && vv[k] == src) bad |= E_DUP;
                    if (in && j > a + 1 && vv[k] <= pv) bad |= PS_UNSORTED;
                }
                if (ok) {
                    const uint32_t p = (uint32_t)part[vv[k]];
                    if (!CHECK || p < (uint32_t)nparts) {
                        const uint32_t bit = 1u << (p & 31);
                        if (!(*(volatile uint32_t *)&bm[p >> 5] & bit)) atomicOr(&bm[p >> 5], bit);
                        if (D && j >= dst0 && !(*(volatile uint32_t *)&bd[p >> 5] & bit)) atomicOr(&bd[p >> 5], bit);
                    }
                }
            }
        }
        __syncwarp();
        uint32_t lam = 0;
        for (int x = lane; x < words; x += 32) {
            lam += __popc(bm[x]);
            bm[x] = 0;
            if (D) {
                for (uint32_t y = bd[x]; y; y &= y - 1) atomicAdd(&s_d[32 * x + __ffs(y) - 1], 1u);
                bd[x] = 0;
            }
        }
        lam = __reduce_add_sync(FULL, lam);
        if (lane == 0 && lam > 1) {
            const unsigned long long we = w ? (unsigned long long)w[i] : 1ull;
            c += we * (lam - 1);
            cn += we;
        }
    }
    if (CHECK && bad) atomicOr(err, bad);
    if (lane == 0 && cn) {
        atomicAdd(&s_sum[0], c);
        atomicAdd(&s_sum[1], cn);
    }
    __syncthreads();
    if (threadIdx.x == 0 && s_sum[1]) {
        atomicAdd(conn, s_sum[0]);
        atomicAdd(cutnet, s_sum[1]);
    }
    if (D)
        for (int32_t p = threadIdx.x; p < nparts; p += PS_T)
            if (s_d[p]) atomicAdd(&D[p], (int32_t)s_d[p]);
}
// The same for the listed hyperedges of more than PS_BIG pins, a CTA each
// (the row of bits, its checks and its counts are k_part_scan's).  One
// hyperedge of 30 M pins: 575 ms by a warp, 180 by the pins lists before.
template <bool CHECK>
__global__ void __launch_bounds__(PSB_T) k_part_scan_big(const int32_t *off, const int32_t *pin, const int32_t *nsrc,
                                                         const int32_t *w, const int32_t *list,
                                                         const int32_t *count_p, const int32_t *part, int32_t n, int32_t nparts, int32_t *D, unsigned long long *conn,
                                                         unsigned long long *cutnet, uint32_t *err) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) uint32_t smw[];
    __shared__ int32_t s_lam;
    const int words = (nparts + 1023) / 1024 * 32;
    uint32_t *bm = smw, *bd = smw + words, *s_d = bd + words;
    const int32_t count = *count_p;
    if ((int32_t)blockIdx.x >= count) return;
    for (int i = threadIdx.x; i < words * (D ? 34 : 1); i += PSB_T) smw[i] = 0;
    if (threadIdx.x == 0) s_lam = 0;
    __syncthreads();
    uint32_t bad = 0;
    for (int32_t x = blockIdx.x; x < count; x += gridDim.x) {
        const int32_t i = list[x], a = off[i], len = off[i + 1] - a;
        const int32_t *pe = pin + a;
        const int32_t dst0 = D ? nsrc[i] : 1, src = CHECK ? pe[0] : 0;
        constexpr int R = 4;
        for (int64_t j0 = threadIdx.x; j0 < len; j0 += R * PSB_T) {
            int32_t v[R], pv[R];
#pragma unroll
            for (int k = 0; k < R; k++) {
                const int64_t j = j0 + k * PSB_T;
                v[k] = j < len ? pe[j] : -1;
                pv[k] = CHECK && j > 1 && j < len ? pe[j - 1] : INT32_MIN;
            }
#pragma unroll
            for (int k = 0; k < R; k++) {
                const int64_t j = j0 + k * PSB_T;
                if (j >= len) break;
                if (CHECK) {
                    if (j > 0 && v[k] == src) bad |= E_DUP;
                    if (v[k] <= pv[k] && j > 1) bad |= PS_UNSORTED;
                    if (v[k] < 0 || v[k] >= n) {
                        bad |= E_PIN;
                        continue;
                    }
                }
                const uint32_t p = (uint32_t)part[v[k]];
                if (CHECK && p >= (uint32_t)nparts) continue;
                const uint32_t bit = 1u << (p & 31);
                if (!(*(volatile uint32_t *)&bm[p >> 5] & bit)) atomicOr(&bm[p >> 5], bit);
                if (D && j >= dst0 && !(*(volatile uint32_t *)&bd[p >> 5] & bit)) atomicOr(&bd[p >> 5], bit);
            }
        }
        __syncthreads();
        int32_t lam = 0;
        for (int y = threadIdx.x; y < words; y += PSB_T) {
            lam += __popc(bm[y]);
            bm[y] = 0;
            if (D) {
                for (uint32_t z = bd[y]; z; z &= z - 1) atomicAdd(&s_d[32 * y + __ffs(z) - 1], 1u);
                bd[y] = 0;
            }
        }
        if (lam) atomicAdd(&s_lam, lam);
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned long long we = w ? (unsigned long long)w[i] : 1ull;
            if (s_lam > 1) {
                atomicAdd(conn, we * (unsigned long long)(s_lam - 1));
                atomicAdd(cutnet, we);
            }
            s_lam = 0;
        }
        __syncthreads();
    }
    if (CHECK && bad) atomicOr(err, bad);
    if (D)
        for (int32_t p = threadIdx.x; p < nparts; p += PSB_T)
            if (s_d[p]) atomicAdd(&D[p], (int32_t)s_d[p]);
}
// part_scan: k_part_scan alone; with `big`, without the hyperedges of more than
// PS_BIG pins, and k_part_scan_big for these
template <bool CHECK>
static void part_scan(const int32_t *off, const int32_t *pin, const int32_t *nsrc, const int32_t *w, int32_t e,
                      const int32_t *part, int32_t n, int32_t nparts, int32_t *D, int64_t *conn, int64_t *cutnet,
                      const uint32_t *pre, uint32_t stop, uint32_t *err, bool big, Arena &A) {
    cudaStream_t s = A.stream();
    unsigned long long *c = (unsigned long long *)conn, *cn = (unsigned long long *)cutnet;
    size_t sm = part_scan_smem(nparts, D != nullptr);
    auto scan = [&](auto kern) {
        const int occ = prepare_kernel((const void *)kern, PS_T, sm);
        launch_k(kern, (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(e, PS_T / 32), (int64_t)num_sms() * occ)), PS_T,
                 sm, s, off, pin, nsrc, w, e, part, n, nparts, D, c, cn, pre, stop, err);
        HP_LAUNCH_CHECK();
    };
    if (!big) return scan(k_part_scan<CHECK, false>);
    scan(k_part_scan<CHECK, true>);
    int32_t *list = A.get<int32_t>(2 + (size_t)std::min<int64_t>(e, (int64_t(1) << 31) / PS_BIG)), *cnt = list, *maxe = list + 1;
    HPC(cudaMemsetAsync(cnt, 0, 2 * sizeof(int32_t), s));
    launch_k(k_big_edges, grid_of(e, 256), 256, 0, s, off, e, PS_BIG, list + 2, cnt, maxe);
    HP_LAUNCH_CHECK();
    sm = 4 * (size_t)cdiv(std::max(nparts, 1), 1024) * 32 * (D ? 34 : 1);
    const int occ = prepare_kernel((const void *)k_part_scan_big<CHECK>, PSB_T, sm);
    launch_k(k_part_scan_big<CHECK>, num_sms() * occ, PSB_T, sm, s, off, pin, nsrc, w, list + 2, cnt, part, n, nparts,
             D, c, cn, err);
    HP_LAUNCH_CHECK();
    A.release(list);
}

// A caller's offsets, weights and parts, before any pin is read.
__global__ void k_conn_check(const int32_t *off, int32_t e, const int32_t *weights, const int32_t *part, int32_t n,
                             int32_t nparts, uint32_t *err, unsigned long long *wsum, uint32_t *bad_part) {
    HP_KERNEL_ENTER();
    uint32_t bad = 0;
    unsigned long long ws = 0;
    GRID_STRIDE(i, (int64_t)e) {
        if (off[i + 1] <= off[i]) bad |= E_OFFSETS;
        else if ((int64_t)off[i + 1] - off[i] > PS_BIG) bad |= PS_HAS_BIG;
        if (weights) {
            const int32_t x = weights[i];
            if (x < 1 || x > 65536) bad |= E_WEIGHT;
            ws += (unsigned long long)max(x, 0);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && off[0] != 0) bad |= E_OFFSETS;
    bool pbad = false;
    GRID_STRIDE(v, (int64_t)n) pbad |= part[v] < 0 || part[v] >= nparts;
    for (int o = 16; o > 0; o >>= 1) ws += __shfl_down_sync(0xffffffffu, ws, o);
    bad = __reduce_or_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) {
        if (bad & (E_OFFSETS | PS_HAS_BIG)) atomicOr(err, bad & (E_OFFSETS | PS_HAS_BIG));
        if (bad & E_WEIGHT) atomicOr(err + 1, E_WEIGHT);   // (the pins are still to be checked)
        if (ws) atomicAdd(wsum, ws);
    }
    if (pbad) atomicOr(bad_part, 1u);
}
// Connectivity and cut-net of a caller's hypergraph (one source each) and
// part vector: offsets, weights and parts are checked, then one pass over the
// pins checks and counts.  Returns the error bits; PS_UNSORTED among them:
// nothing is known of duplicate pins.  *bad_part: some part id is out of range.
uint32_t connectivity_scan(const int32_t *pins, const int32_t *offsets, int32_t e, int32_t n, const int32_t *weights,
                           const int32_t *part, int32_t nparts, int64_t *conn, int64_t *cutnet, uint32_t *bad_part,
                           Arena &A) {
    cudaStream_t s = A.stream();
    struct Box {
        uint32_t err, werr, bad_part, scan_err;
        unsigned long long wsum;
        int64_t conn, cutnet;
    };
    Box *box = A.get<Box>(1), hb;
    HPC(cudaMemsetAsync(box, 0, sizeof(Box), s));
    launch_k(k_conn_check, grid_of(std::max(e, n), 256), 256, 0, s, offsets, e, weights, part, n, nparts, &box->err,
             &box->wsum, &box->bad_part);
    HP_LAUNCH_CHECK();
    auto scan = [&](uint32_t stop, bool big) {
        part_scan<true>(offsets, pins, nullptr, weights, e, part, n, nparts, nullptr, &box->conn, &box->cutnet, &box->err,
                        stop, &box->scan_err, big, A);
    };
    if (e > 0) scan(E_OFFSETS | PS_HAS_BIG, false);
    fetch_bytes(&hb, box, sizeof hb, s);
    if (hb.err == PS_HAS_BIG) {   // nothing scanned yet
        scan(E_OFFSETS, true);
        fetch_bytes(&hb, box, sizeof hb, s);
    }
    hb.err &= ~PS_HAS_BIG;
    A.release(box);
    *conn = hb.conn;
    *cutnet = hb.cutnet;
    *bad_part = hb.bad_part;
    return hb.err | hb.werr | hb.scan_err | (hb.wsum > (1ull << 37) ? E_WSUM : 0u);
}
bool connectivity_scan_takes(int32_t nparts) { return nparts <= PS_PARTS; }

void objective(const Level &L, const int32_t *w, const int32_t *rho, int32_t nparts, int32_t max_e, int64_t *conn_dev,
               int64_t *cutnet_dev, Arena &A) {
    cudaStream_t s = A.stream();
    HPC(cudaMemsetAsync(conn_dev, 0, sizeof(int64_t), s));
    HPC(cudaMemsetAsync(cutnet_dev, 0, sizeof(int64_t), s));
    if (L.e == 0) return;
    if (nparts <= PS_PARTS) {
        part_scan<false>(L.off, L.pin, L.nsrc, w, L.e, rho, L.n, nparts, nullptr, conn_dev, cutnet_dev, nullptr, 0,
                         nullptr, max_e > PS_BIG, A);
        return;
    }
    int32_t *maxe = A.get<int32_t>(1);
    HPC(cudaMemsetAsync(maxe, 0, sizeof(int32_t), s));
    launch_k(k_max_edge, grid_of(L.e, 256), 256, 0, s, L.off, L.e, maxe);
    HP_LAUNCH_CHECK();
    int32_t me = fetch<int32_t>(maxe, s);
    Plist PL;
    PL.p = A.get<int32_t>(L.np);
    PL.cnt = A.get<int32_t>(L.np);
    PL.cin = A.get<int32_t>(L.np);
    PL.lam = A.get<int32_t>(L.e);
    build_plist(L, w, rho, me, PL, nullptr, nullptr, A);
    launch_k(k_objective, grid_of(L.e, 256), 256, 0, s, PL.lam, w, L.e, (unsigned long long *)conn_dev,
             (unsigned long long *)cutnet_dev);
    HP_LAUNCH_CHECK();
    A.release(PL.p);
    A.release(PL.cnt);
    A.release(PL.cin);
    A.release(PL.lam);
    A.release(maxe);
}

// ---------------------------------------------------------------- Eq. 13 gains
struct Moves {
    int32_t *node, *src, *dst;
    long long *gain;
    int32_t *count;
};

constexpr int GN_T = 128;

// gain(v,p) = saving(v) - loss(v,p) with loss = W(v) - conn(v,p), conn(v,p) =
// sum of w(e) over e in I(v) with pins(p,e) > 0 (singleton hyperedges cancel).
__device__ void gains_node(int32_t v, const int32_t *off, const int32_t *ioff, const int32_t *cutn, const int32_t *inc,
                           const int32_t *w,
                           const int32_t *rho, const int32_t *size, const long long *psize, const long long *saving,
                           const long long *wns, Plist PL, int32_t omega, int second_half, int32_t *keys,
                           long long *conn, int32_t *slots, uint32_t cap, uint32_t limit, int32_t *s_cnt, int *s_flag,
                           Moves M,
                           int32_t *ovf, int32_t *ovf_n, long long *s_rg, int32_t *s_rp) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t mask = cap - 1;
    const int32_t s = rho[v];
    auto add = [&](int32_t p, long long we) {
        uint32_t h = hslot(p, mask);
        for (uint32_t probe = 0; probe < cap; probe++) {
            int32_t kk = ((volatile int32_t *)keys)[h];
            if (kk == -1) {
                int32_t old = atomicCAS(&keys[h], -1, p);
                if (old == -1) {
                    const uint32_t slot = (uint32_t)atomicAdd(s_cnt, 1);
                    if (slot < limit) slots[slot] = (int32_t)h;
                    else *(volatile int *)s_flag = 1;
                    kk = p;
                } else {
                    kk = old;
                }
            }
            if (kk == p) {
                atomicAdd((unsigned long long *)&conn[h], (unsigned long long)we);
                return;
            }
            h = (h + 1) & mask;
        }
    };
    // one cut hyperedge per thread.  The k-th entries of the pins lists of a
    // warp's 32 hyperedges are combined by part across the warp (match_any)
    // before one table update per distinct part, so that the few parts a
    // node touches are not hammered by every lane.
    {
        // (unsigned positions, here and in the other gain kernels: they may pass 2^31
        // behind the last incidence entry)
        const uint32_t c0 = ioff[v], c1 = c0 + cutn[v];
        for (uint32_t base = c0; base < c1; base += blockDim.x) {
            if (__any_sync(0xffffffffu, *(volatile int *)s_flag)) break;
            const uint32_t t = base + threadIdx.x;
            int32_t a = 0, lam = 0;
            uint32_t we = 0;
            if (t < c1) {
                const int32_t e = inc[t];
                lam = PL.lam[e];
                a = off[e];
                we = (uint32_t)w[e];
            }
            const int kmax = __reduce_max_sync(0xffffffffu, (unsigned)lam);
            for (int k = 0; k < kmax; k++) {
                int32_t p = k < lam ? PL.p[a + k] : -1;
                if (p == s) p = -1;
                const unsigned m = __match_any_sync(0xffffffffu, p);
                uint32_t sw[1] = {we};
                group_sum(m, p >= 0, sw);
                if (p >= 0 && lane == __ffs(m) - 1) add(p, (long long)sw[0]);
            }
        }
    }
    __syncthreads();
    const int overflow = *s_flag;
    long long bg = 0;
    int32_t bp = -1;
    const long long base = saving[v] - wns[v];
    if (overflow) {
        // the slot list is incomplete: clear the whole table, redo the node in a larger one
        for (uint32_t h = threadIdx.x; h < cap; h += blockDim.x) {
            keys[h] = -1;
            conn[h] = 0;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            ovf[atomicAdd(ovf_n, 1)] = v;
            *s_flag = 0;
            *s_cnt = 0;
        }
        __syncthreads();
        return;
    }
    const int32_t used = *(volatile int32_t *)s_cnt;
    for (int32_t i = threadIdx.x; i < used; i += blockDim.x) {
        const int32_t h = slots[i];
        const int32_t p = keys[h];
        if (!second_half || (long long)size[v] + psize[p] <= omega) {
            long long g = base + conn[h];
            if (bp < 0 || g > bg || (g == bg && p > bp)) {
                bg = g;
                bp = p;
            }
        }
        keys[h] = -1;
        conn[h] = 0;
    }
    for (int o = 16; o > 0; o >>= 1) {
        long long og = __shfl_down_sync(0xffffffffu, bg, o);
        int32_t op = __shfl_down_sync(0xffffffffu, bp, o);
        if (op >= 0 && (bp < 0 || og > bg || (og == bg && op > bp))) {
            bg = og;
            bp = op;
        }
    }
    if (lane == 0) {
        s_rg[wid] = bg;
        s_rp[wid] = bp;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < nw; k++) {
            if (s_rp[k] >= 0 && (bp < 0 || s_rg[k] > bg || (s_rg[k] == bg && s_rp[k] > bp))) {
                bg = s_rg[k];
                bp = s_rp[k];
            }
        }
        if (bp >= 0 && bg > 0) {
            int32_t i = atomicAdd(M.count, 1);
            M.node[i] = v;
            M.src[i] = s;
            M.dst[i] = bp;
            M.gain[i] = bg;
        }
        *s_cnt = 0;
    }
    __syncthreads();
}

struct GainArgs {
    const int32_t *off, *ioff, *cutn, *inc, *w, *rho, *size;   // cut hyperedges of v: inc[ioff[v] .. ioff[v] + cutn[v])
    const long long *psize, *saving, *wns;
    Plist PL;
    int32_t omega;
    int second_half;
    Moves M;
};

template <int BT>
__global__ void __launch_bounds__(BT) k_gains_smem(GainArgs G, const int32_t *list, const int32_t *count_p,
                                                     uint32_t cap, int32_t *ovf, int32_t *ovf_n) {
    HP_KERNEL_ENTER();
    const int32_t count = *count_p;
    extern __shared__ __align__(16) unsigned char smem[];
    long long *conn = reinterpret_cast<long long *>(smem);
    int32_t *keys = reinterpret_cast<int32_t *>(conn + cap);
    int32_t *slots = keys + cap;
    __shared__ int32_t s_cnt;
    __shared__ int s_flag;
    __shared__ long long s_rg[32];
    __shared__ int32_t s_rp[32];
    for (uint32_t i = threadIdx.x; i < cap; i += BT) {
        keys[i] = -1;
        conn[i] = 0;
    }
    if (threadIdx.x == 0) {
        s_cnt = 0;
        s_flag = 0;
    }
    __syncthreads();
    for (int32_t k = blockIdx.x; k < count; k += gridDim.x)
        gains_node(list[k], G.off, G.ioff, G.cutn, G.inc, G.w, G.rho, G.size, G.psize, G.saving, G.wns, G.PL, G.omega,
                   G.second_half, keys, conn, slots, cap, cap * 3 / 4, &s_cnt, &s_flag, G.M, ovf, ovf_n, s_rg, s_rp);
}

__global__ void __launch_bounds__(GN_T) k_gains_global(GainArgs G, const int32_t *list, const int32_t *count_p,
                                                       uint32_t cap, int32_t *gkeys, long long *gconn, int32_t *bad,
                                                       int32_t *bad_n) {
    HP_KERNEL_ENTER();
    const int32_t count = *count_p;
    if (count == 0) return;
    __shared__ int32_t s_cnt;
    __shared__ int s_flag;
    __shared__ long long s_rg[8];
    __shared__ int32_t s_rp[8];
    int32_t *keys = gkeys + (int64_t)blockIdx.x * 2 * cap;
    int32_t *slots = keys + cap;
    long long *conn = gconn + (int64_t)blockIdx.x * cap;
    for (uint32_t i = threadIdx.x; i < cap; i += GN_T) {
        keys[i] = -1;
        conn[i] = 0;
    }
    if (threadIdx.x == 0) {
        s_cnt = 0;
        s_flag = 0;
    }
    __syncthreads();
    for (int32_t k = blockIdx.x; k < count; k += gridDim.x)
        gains_node(list[k], G.off, G.ioff, G.cutn, G.inc, G.w, G.rho, G.size, G.psize, G.saving, G.wns, G.PL, G.omega,
                   G.second_half, keys, conn, slots, cap, cap - 1, &s_cnt, &s_flag, G.M, bad, bad_n, s_rg, s_rp);
}

// Nodes with at most GW_DEG cut hyperedges: one warp each, with a warp-private
// table of GW_SLOTS parts in shared memory.  Entries of the lanes' hyperedges
// are combined by part across the warp before each table update.  A node
// whose neighbouring parts outgrow `limit` is handed to the CTA kernel's list.
constexpr int GW_T = 256, GW_SLOTS = 256;
__global__ void __launch_bounds__(GW_T) k_gains_warp(GainArgs G, const int32_t *list, const int32_t *count_p,
                                                     uint32_t limit, int32_t *spill, int32_t *spill_n) {
    HP_KERNEL_ENTER();
    __shared__ int32_t s_keys[GW_T / 32][GW_SLOTS];
    __shared__ long long s_conn[GW_T / 32][GW_SLOTS];
    __shared__ int32_t s_used[GW_T / 32];
    const unsigned FULL = 0xffffffffu;
    const int32_t count = *count_p;
    if (count == 0) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *keys = s_keys[wid];
    long long *conn = s_conn[wid];
    for (int h = lane; h < GW_SLOTS; h += 32) {
        keys[h] = -1;
        conn[h] = 0;
    }
    if (lane == 0) s_used[wid] = 0;
    __syncwarp();
    const int64_t gw = (int64_t)blockIdx.x * (GW_T / 32) + wid, nw = (int64_t)gridDim.x * (GW_T / 32);
    for (int64_t k = gw; k < count; k += nw) {
        const int32_t v = list[k];
        const int32_t s = G.rho[v];
        const uint32_t c0 = G.ioff[v], c1 = c0 + G.cutn[v];
        for (uint32_t base = c0; base < c1; base += 32) {
            if (*(volatile int32_t *)&s_used[wid] > (int32_t)limit) break;   // same value for the whole warp
            const uint32_t t = base + lane;
            int32_t a = 0, lam = 0;
            uint32_t we = 0;
            if (t < c1) {
                const int32_t e = G.inc[t];
                lam = G.PL.lam[e];
                a = G.off[e];
                we = (uint32_t)G.w[e];
            }
            const int kmax = (int)__reduce_max_sync(FULL, (unsigned)lam);
            for (int k2 = 0; k2 < kmax; k2++) {
                int32_t p = k2 < lam ? G.PL.p[a + k2] : -1;
                if (p == s) p = -1;
                const unsigned m = __match_any_sync(FULL, p);
                uint32_t sw[1] = {we};
                group_sum(m, p >= 0, sw);
                if (p >= 0 && lane == __ffs(m) - 1) {
                    uint32_t h = hslot(p, GW_SLOTS - 1);
                    for (int probe = 0; probe < GW_SLOTS; probe++) {
                        int32_t kk = ((volatile int32_t *)keys)[h];
                        if (kk == -1) {
                            const int32_t old = atomicCAS(&keys[h], -1, p);
                            if (old == -1) {
                                atomicAdd(&s_used[wid], 1);
                                kk = p;
                            } else {
                                kk = old;
                            }
                        }
                        if (kk == p) {
                            atomicAdd((unsigned long long *)&conn[h], (unsigned long long)sw[0]);
                            break;
                        }
                        h = (h + 1) & (GW_SLOTS - 1);
                    }
                }
            }
            __syncwarp();
        }
        __syncwarp();
        const bool spilled = *(volatile int32_t *)&s_used[wid] > (int32_t)limit;
        const long long basev = G.saving[v] - G.wns[v];
        long long bg = 0;
        int32_t bp = -1;
        for (int h = lane; h < GW_SLOTS; h += 32) {
            const int32_t p = keys[h];
            if (p >= 0 && !spilled && (!G.second_half || (long long)G.size[v] + G.psize[p] <= G.omega)) {
                const long long g = basev + conn[h];
                if (bp < 0 || g > bg || (g == bg && p > bp)) {
                    bg = g;
                    bp = p;
                }
            }
            keys[h] = -1;
            conn[h] = 0;
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long og = __shfl_down_sync(FULL, bg, o);
            const int32_t op = __shfl_down_sync(FULL, bp, o);
            if (op >= 0 && (bp < 0 || og > bg || (og == bg && op > bp))) {
                bg = og;
                bp = op;
            }
        }
        if (lane == 0) {
            if (spilled) {
                spill[atomicAdd(spill_n, 1)] = v;
            } else if (bp >= 0 && bg > 0) {
                const int32_t i = atomicAdd(G.M.count, 1);
                G.M.node[i] = v;
                G.M.src[i] = s;
                G.M.dst[i] = bp;
                G.M.gain[i] = bg;
            }
            s_used[wid] = 0;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------- gains from part bits
// Levels whose cut hyperedges span many parts (random nets: lambda(e) near
// |e|).  k_part_bits writes, for every cut hyperedge, one row of 4 * WQ words
// with bit p set when e touches part p; k_gains_bits then reads a node's rows
// instead of its pins lists.  A lane owns the parts p = 32 k + lane: the row's
// words arrive by a warp-uniform 16-byte load and every lane adds w(e) to the
// counters of its set bits, so a row costs two instructions per 32 parts and
// neither a hash probe nor an atomic.  The list form needs a match, a warp
// reduction and a shared-memory update per list entry.  Bound by the L1 return
// of the uniform loads (a row's bytes to 32 lanes).  Measured per repetition,
// summed over the node lists: 16,384-node random net, 413 parts, lambda about
// 100: 7.4 ms of list kernels, 0.33 ms of bit kernels, 30 us for the rows;
// 20,011-node irregular net, 206 parts, lambda about 26: 1.93 and 0.13 ms.
constexpr int PB_T = 256, PB_MAXQ = 8;
static_assert(PB_PARTS == PB_MAXQ * 128, "a bit per part");
constexpr int64_t PB_BYTES = int64_t(1) << 30;
__global__ void __launch_bounds__(PB_T) k_part_bits(const int32_t *off, Plist PL, int32_t e, int wq, uint4 *bits) {
    HP_KERNEL_ENTER();
    __shared__ __align__(16) uint32_t s_row[PB_T / 32][PB_MAXQ * 4];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t *row = s_row[wid];
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = w0; i < e; i += nw) {
        const int32_t a = off[i];
        if (off[i + 1] - a < 2) continue;   // single-pin hyperedges have no pins list
        const int32_t lam = PL.lam[i];
        if (lam < 2) continue;              // not cut: no node lists it
        if (lane < 4 * wq) row[lane] = 0;
        __syncwarp();
        for (int32_t k = lane; k < lam; k += 32) {
            const int32_t p = PL.p[a + k];
            atomicOr(&row[p >> 5], 1u << (p & 31));
        }
        __syncwarp();
        if (lane < wq) bits[i * wq + lane] = reinterpret_cast<const uint4 *>(row)[lane];
        __syncwarp();
    }
}

// One node per CTA of NW warps (from list and then list2, which may be none),
// the warps taking its cut hyperedges in chunks of 32.  The counters are 32 bits wide: the host takes this path only when
// the sum of all weights is below 2^32.
template <int WQ, int NW>
__global__ void __launch_bounds__(NW * 32) k_gains_bits(GainArgs G, const uint4 *bits, int32_t nparts,
                                                        const int32_t *list, const int32_t *count_p,
                                                        const int32_t *list2, const int32_t *count2_p) {
    HP_KERNEL_ENTER();
    __shared__ uint32_t s_conn[WQ * 128];
    __shared__ long long s_rg[NW];
    __shared__ int32_t s_rp[NW];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t my = 1u << lane;
    const int32_t n1 = *count_p, count = n1 + (list2 ? *count2_p : 0);
    for (int i = threadIdx.x; i < WQ * 128; i += NW * 32) s_conn[i] = 0;
    __syncthreads();
    for (int32_t k = blockIdx.x; k < count; k += gridDim.x) {
        const int32_t v = k < n1 ? list[k] : list2[k - n1], s = G.rho[v];
        const uint32_t c0 = G.ioff[v], c1 = c0 + G.cutn[v];
        uint32_t acc[WQ * 4];
#pragma unroll
        for (int q = 0; q < WQ * 4; q++) acc[q] = 0;
        for (uint32_t base = c0 + wid * 32; base < c1; base += NW * 32) {
            const uint32_t t = base + lane;
            int32_t e = 0;
            uint32_t we = 0;
            if (t < c1) {
                e = G.inc[t];
                we = (uint32_t)G.w[e];
            }
            const int cnt = (int)min(32u, c1 - base);
#pragma unroll 4
            for (int u = 0; u < cnt; u++) {
                const uint4 *r = bits + (int64_t)__shfl_sync(FULL, e, u) * WQ;
                const uint32_t wu = __shfl_sync(FULL, we, u);
#pragma unroll
                for (int q = 0; q < WQ; q++) {
                    const uint4 x = __ldg(r + q);
                    if (x.x & my) acc[4 * q] += wu;
                    if (x.y & my) acc[4 * q + 1] += wu;
                    if (x.z & my) acc[4 * q + 2] += wu;
                    if (x.w & my) acc[4 * q + 3] += wu;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < WQ * 4; q++)
            if (acc[q]) atomicAdd(&s_conn[32 * q + lane], acc[q]);
        __syncthreads();
        // the best part (gain, then the larger id) of the ones v touches
        long long bg = 0;
        int32_t bp = -1;
        const long long basev = G.saving[v] - G.wns[v];
        const long long room = (long long)G.omega - G.size[v];
        for (int32_t p = threadIdx.x; p < nparts; p += NW * 32) {
            const uint32_t c = s_conn[p];
            s_conn[p] = 0;
            if (c == 0 || p == s || (G.second_half && G.psize[p] > room)) continue;
            const long long g = basev + (long long)c;
            if (bp < 0 || g >= bg) {   // p ascends
                bg = g;
                bp = p;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long og = __shfl_down_sync(FULL, bg, o);
            const int32_t op = __shfl_down_sync(FULL, bp, o);
            if (op >= 0 && (bp < 0 || og > bg || (og == bg && op > bp))) {
                bg = og;
                bp = op;
            }
        }
        if (lane == 0) {
            s_rg[wid] = bg;
            s_rp[wid] = bp;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int x = 1; x < NW; x++)
                if (s_rp[x] >= 0 && (bp < 0 || s_rg[x] > bg || (s_rg[x] == bg && s_rp[x] > bp))) {
                    bg = s_rg[x];
                    bp = s_rp[x];
                }
            if (bp >= 0 && bg > 0) {
                const int32_t i = atomicAdd(G.M.count, 1);
                G.M.node[i] = v;
                G.M.src[i] = s;
                G.M.dst[i] = bp;
                G.M.gain[i] = bg;
            }
        }
    }
}

// ---------------------------------------------------------------- per level constants
// The level's classes and constants, in one pass over its nodes, hyperedges
// and incidence (all independent of one another):
// - parts holding at least one node (lambda(e) never exceeds their number
//   within a level: moves only go to parts that exist);
// - hyperedges of 2..TINY_E pins (one thread each), up to SMALL_EDGE (a warp
//   each) and larger ones (a CTA each), and the largest;
// - per node, Wns(v) = sum of w(e) over incident hyperedges with |e| >= 2, and
//   the number of singleton hyperedges {v} that hold v as a destination.
//   Singleton hyperedges cancel in every gain (they are spared and re-created
//   by any move) and change only the distinct-inbound count, by one per
//   singleton at p_s (-) and at p_d (+): they are handled per node.
// Appends take one atomic per CTA and list: 229,376 hyperedges a warp at a
// time queued 7,000 atomics on one word, most of the 12 us that took.
constexpr int TINY_E = 8;
constexpr int32_t SMALL_EDGE = 512;
// largest hyperedge handled a warp each: the level's largest, at least 2, at most SMALL_EDGE
inline int32_t level_small_max(int32_t max_e) { return max_e < 2 ? 2 : (max_e > SMALL_EDGE ? SMALL_EDGE : max_e); }
// counters of a level: larger hyperedges, the largest, tiny ones, middle ones, parts in use
enum { V_BIG, V_MAX, V_TINY, V_MID, V_PARTS, V_N };
constexpr int LP_T = 256;
__global__ void __launch_bounds__(LP_T) k_level_prep(Level L, const int32_t *w, const int32_t *rho, int32_t *pmark,
                                                     int32_t *big, int32_t *tiny, int32_t *mid, int32_t *cnt,
                                                     long long *wns, int32_t *singin) {
    HP_KERNEL_ENTER();
    __shared__ int32_t s_n[3][LP_T / 32], s_max, s_used;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    if (threadIdx.x == 0) s_max = s_used = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * LP_T;
    int32_t used = 0, mx = 0;
    GRID_STRIDE(v, (int64_t)L.n) {
        if (pmark[rho[v]] == 0 && atomicExch(&pmark[rho[v]], 1) == 0) used++;
    }
    for (int64_t base = (int64_t)blockIdx.x * LP_T; base < L.e; base += step) {
        const int64_t i = base + threadIdx.x;
        const int32_t sz = i < L.e ? L.off[i + 1] - L.off[i] : 0;
        mx = max(mx, sz);
        const int cls = sz < 2 ? -1 : sz <= TINY_E ? 0 : sz <= SMALL_EDGE ? 1 : 2;
        unsigned m[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            m[c] = __ballot_sync(FULL, cls == c);
            if (lane == 0) s_n[c][wid] = __popc(m[c]);
        }
        __syncthreads();
        if (threadIdx.x < 3) {   // the warps' places in their lists
            int32_t tot = 0;
            for (int x = 0; x < LP_T / 32; x++) tot += s_n[threadIdx.x][x];
            int32_t at = tot ? atomicAdd(&cnt[threadIdx.x == 0 ? V_TINY : threadIdx.x == 1 ? V_MID : V_BIG], tot) : 0;
            for (int x = 0; x < LP_T / 32; x++) {
                const int32_t k = s_n[threadIdx.x][x];
                s_n[threadIdx.x][x] = at;
                at += k;
            }
        }
        __syncthreads();
        if (cls == 0) tiny[s_n[0][wid] + __popc(m[0] & lt)] = (int32_t)i;
        if (cls == 1) mid[s_n[1][wid] + __popc(m[1] & lt)] = (int32_t)i;
        if (cls == 2) big[s_n[2][wid] + __popc(m[2] & lt)] = (int32_t)i;
        __syncthreads();
    }
    mx = __reduce_max_sync(FULL, mx);
    used = __reduce_add_sync(FULL, used);
    if (lane == 0) {
        atomicMax(&s_max, mx);
        if (used) atomicAdd(&s_used, used);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (s_max) atomicMax(&cnt[V_MAX], s_max);
        if (s_used) atomicAdd(&cnt[V_PARTS], s_used);
    }
    for (int64_t base = (int64_t)blockIdx.x * LP_T + (threadIdx.x & ~31u); base < L.np; base += step) {
        const int64_t t = base + lane;
        const bool valid = t < L.np;
        const int32_t v = valid ? L.inode[t] : -1 - lane;
        long long a = 0;
        int32_t c = 0;
        if (valid) {
            const int32_t e = L.inc[t];
            const int32_t sz = L.off[e + 1] - L.off[e];
            if (sz >= 2) a = w[e];
            else if (t < L.ioff[v] + L.nin[v]) c = 1;
        }
        bool tail = warp_run_sum(v, a);
        warp_run_sum(v, c);
        if (valid && tail) {
            if (a) atomicAdd((unsigned long long *)&wns[v], (unsigned long long)a);
            if (c) atomicAdd(&singin[v], c);
        }
    }
}

// pins(p, e) list of a hyperedge of 2..TINY_E pins by one thread.  D(p) and
// saving(v) updates are combined across the warp by key (match_any) first:
// a coarse node or a part shared by many neighbouring hyperedges would
// otherwise take one global atomic per hyperedge.
__global__ void k_plist_tiny(const int32_t *off, const int32_t *pin, const int32_t *nsrc, const int32_t *w,
                             const int32_t *rho, const int32_t *list, int32_t count, Plist PL, int32_t *D,
                             long long *saving) {
    HP_KERNEL_ENTER();
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < count; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = base + threadIdx.x;
        const bool live = k < count;
        int32_t a = 0, sz = 0, dst0 = 0;
        uint32_t we = 0;
        if (live) {
            const int32_t e = list[k];
            a = off[e];
            sz = off[e + 1] - a;
            dst0 = nsrc[e];
            we = (uint32_t)w[e];
        }
        int32_t vv[TINY_E], pp[TINY_E], up[TINY_E], uc[TINY_E], uci[TINY_E];
        int32_t nu = 0;
#pragma unroll
        for (int j = 0; j < TINY_E; j++) {
            vv[j] = -1;
            pp[j] = -1;
            up[j] = 0x7fffffff;
            uc[j] = 0;
            uci[j] = 0;
        }
#pragma unroll
        for (int j = 0; j < TINY_E; j++) {
            if (j < sz) {
                vv[j] = pin[a + j];
                pp[j] = rho[vv[j]];
            }
        }
#pragma unroll
        for (int j = 0; j < TINY_E; j++) {
            if (j >= sz) break;
            const int32_t p = pp[j];
            int32_t f = -1;
#pragma unroll
            for (int u = 0; u < TINY_E; u++)
                if (u < nu && up[u] == p) f = u;
            if (f < 0) f = nu++;
#pragma unroll
            for (int u = 0; u < TINY_E; u++)
                if (u == f) {
                    up[u] = p;
                    uc[u]++;
                    uci[u] += j >= dst0;
                }
        }
        // sorted by part id: rank of each distinct entry
#pragma unroll
        for (int u = 0; u < TINY_E; u++) {
            if (u < nu) {
                int32_t r = 0;
#pragma unroll
                for (int x = 0; x < TINY_E; x++)
                    if (x < nu && up[x] < up[u]) r++;
                PL.p[a + r] = up[u];
                PL.cnt[a + r] = uc[u];
                PL.cin[a + r] = uci[u];
            }
        }
        if (live) PL.lam[list[k]] = nu;
        if (D) {
#pragma unroll
            for (int u = 0; u < TINY_E; u++) {
                const int32_t key = (u < nu && uci[u] > 0) ? up[u] : -1;
                const unsigned m = __match_any_sync(FULL, key);
                if (key >= 0 && lane == __ffs(m) - 1) atomicAdd(&D[key], __popc(m));
            }
        }
        if (saving) {
#pragma unroll
            for (int j = 0; j < TINY_E; j++) {
                int32_t c = 0;
#pragma unroll
                for (int u = 0; u < TINY_E; u++)
                    if (u < nu && up[u] == pp[j]) c = uc[u];
                const int32_t key = (j < sz && c == 1) ? vv[j] : -1;
                const unsigned m = __match_any_sync(FULL, key);
                uint32_t sw[1] = {we};
                group_sum(m, key >= 0, sw);
                if (key >= 0 && lane == __ffs(m) - 1)
                    atomicAdd((unsigned long long *)&saving[key], (unsigned long long)sw[0]);
            }
        }
    }
}

// words of `upd`: hyperedges of 2..TINY_E pins and larger ones among the moved
// nodes', and two 64-bit sums over them, pins and new list entries
enum { U_TINY, U_MID, U_ACC, U_N = U_ACC + 4 };
// After a repetition that applied few moves, the next one updates the
// partition-dependent state where they changed it instead of rebuilding it:
// |p| and the single-pin hyperedges' share of D(p) per move, and the pins
// list, D(p) and saving(v) of the hyperedges with a moved pin.  All are sums
// of integers, so the result is the rebuilt one.  406 rebuilds on the 1M
// Gaussian net (88 moves applied in each on average) took 63 and 36 ms in the
// pins-list kernels; 69 rebuilds and 337 updates take 4 + 10 and 6 + 3 ms, and
// 6 to list the hyperedges: 719 -> 640 ms a call.
__global__ void k_move_nodes(Applied M, const int32_t *node, const int32_t *dst, const int32_t *size,
                             const int32_t *singin, long long *psize, int32_t *D0, int32_t *upd) {
    HP_KERNEL_ENTER();
    const int32_t len = *M.applied;
    if (blockIdx.x == 0 && threadIdx.x < U_N) upd[threadIdx.x] = 0;
    GRID_STRIDE(k, (int64_t)len) {
        const int32_t i = M.seqmove[k], v = node[i], ps = M.src[i], pd = dst[i];
        const unsigned long long sz = (unsigned long long)size[v];
        atomicAdd((unsigned long long *)&psize[ps], 0ull - sz);
        atomicAdd((unsigned long long *)&psize[pd], sz);
        if (singin[v]) {
            atomicAdd(&D0[ps], -singin[v]);
            atomicAdd(&D0[pd], singin[v]);
        }
    }
}
// the hyperedges of the moved nodes (a CTA per node: hubs have ten thousand),
// each once: `mark` holds the number of the last update that listed a hyperedge
__global__ void __launch_bounds__(256) k_moved_edges(Applied M, const int32_t *node, const int32_t *off, const int32_t *ioff, const int32_t *inc,
                              int32_t epoch, int32_t *mark, int32_t *tiny, int32_t *mid, int32_t *upd) {
    HP_KERNEL_ENTER();
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    const int32_t len = *M.applied;
    for (int32_t k = blockIdx.x; k < len; k += gridDim.x) {
        const int32_t v = node[M.seqmove[k]];
        const uint32_t i1 = ioff[v + 1];
        for (uint32_t t0 = ioff[v] + (threadIdx.x & ~31u); t0 < i1; t0 += 256) {
            int cls = -1;
            int32_t e = 0;
            if (t0 + lane < i1) {
                e = inc[t0 + lane];
                const int32_t sz = off[e + 1] - off[e];
                if (sz >= 2 && atomicExch(&mark[e], epoch) != epoch) cls = sz <= TINY_E ? 0 : 1;
            }
#pragma unroll
            for (int c = 0; c < 2; c++) {
                const unsigned m = __ballot_sync(FULL, cls == c);
                if (!m) continue;
                int32_t at = 0;
                if (lane == 0) at = atomicAdd(&upd[c], __popc(m));
                at = __shfl_sync(FULL, at, 0);
                if (cls == c) (c ? mid : tiny)[at + __popc(m & lt)] = e;
            }
        }
    }
}
// hyperedges of 2..TINY_E pins from the list, one thread each
__global__ void k_plist_tiny_update(const int32_t *off, const int32_t *pin, const int32_t *nsrc, const int32_t *w,
                                    const int32_t *rho, const int32_t *list, const int32_t *count_p, Applied M, Plist PL,
                                    int32_t *D, long long *saving, unsigned long long *acc) {
    HP_KERNEL_ENTER();
    const int32_t count = *count_p, len = *M.applied;
    if ((int64_t)blockIdx.x * blockDim.x >= count) return;
    __shared__ unsigned long long s_acc[2];
    if (threadIdx.x < 2) s_acc[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long n_pins = 0, n_ent = 0;
    GRID_STRIDE(x, (int64_t)count) {
        const int32_t e = list[x], a = off[e], sz = off[e + 1] - a;
        int32_t vv[TINY_E], np[TINY_E], op[TINY_E];
        bool moved = false;
#pragma unroll
        for (int j = 0; j < TINY_E; j++) {
            vv[j] = np[j] = op[j] = -1;
            if (j < sz) {
                vv[j] = pin[a + j];
                np[j] = rho[vv[j]];
                op[j] = M.old_part(vv[j], np[j], len);
                moved |= op[j] != np[j];
            }
        }
        if (!moved) continue;
        const int32_t dst0 = nsrc[e];
        const long long we = w[e];
        int32_t lam = 0;
#pragma unroll
        for (int j = 0; j < TINY_E; j++) {
            if (j >= sz) break;
            int32_t co = 0, cn = 0, ci = 0, rank = 0;   // pins of j's old and new part; inbound ones; smaller new parts
            bool nfirst = true, odst = j >= dst0, ndst = j >= dst0;   // first pin of its new part; first destination of its parts
#pragma unroll
            for (int k = 0; k < TINY_E; k++) {
                if (k >= sz) break;
                co += op[k] == op[j];
                if (np[k] == np[j]) {
                    cn++;
                    ci += k >= dst0;
                    if (k < j) nfirst = false;
                    if (k < j && k >= dst0) ndst = false;
                }
                if (op[k] == op[j] && k < j && k >= dst0) odst = false;
                if (np[k] < np[j]) {
                    bool first = true;
#pragma unroll
                    for (int q = 0; q < TINY_E; q++)
                        if (q < k && np[q] == np[k]) first = false;
                    rank += first;
                }
            }
            const long long ds = (cn == 1 ? we : 0) - (co == 1 ? we : 0);
            if (ds) atomicAdd((unsigned long long *)&saving[vv[j]], (unsigned long long)ds);
            if (odst != ndst || op[j] != np[j]) {
                if (odst) atomicAdd(&D[op[j]], -1);
                if (ndst) atomicAdd(&D[np[j]], 1);
            }
            if (nfirst) {
                PL.p[a + rank] = np[j];
                PL.cnt[a + rank] = cn;
                PL.cin[a + rank] = ci;
                lam++;
            }
        }
        PL.lam[e] = lam;
        n_pins += (unsigned long long)sz;
        n_ent += (unsigned long long)lam;
    }
    for (int o = 16; o > 0; o >>= 1) {
        n_pins += __shfl_down_sync(0xffffffffu, n_pins, o);
        n_ent += __shfl_down_sync(0xffffffffu, n_ent, o);
    }
    if ((threadIdx.x & 31) == 0 && n_pins) {
        atomicAdd(&s_acc[0], n_pins);
        atomicAdd(&s_acc[1], n_ent);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_acc[threadIdx.x]) atomicAdd(&acc[threadIdx.x], s_acc[threadIdx.x]);
}

// counters of one repetition (device)
enum { C_CAND, C_MOVES, C_OVF, C_BAD, C_NH, C_BAD0, C_APPLIED, C_NV, C_HUB, C_CW, C_TOUCH, C_PAD,
       C_ACC,          // three 64-bit byte counters (even index: 8-byte aligned), see k_cut_bits
       C_UPD = C_ACC + 6,   // the two 64-bit sums of an update (upd[U_ACC])
       C_N = C_UPD + 4 };

// moves of at most SMALLM are validated by one CTA (k_val_small) with the
// sorts in shared memory; moves of at most sq_max<uint64_t>() are sequenced by one
// thread-block cluster (k_seq_cluster); more take the multi-kernel path
constexpr int SMALLM = 6144, SEQ_T = 1024;
// refinement levels of at most this many nodes run their repetitions on the
// cluster kernels with one read-back each (every move count fits them)
constexpr int32_t SMALL_LEVEL = 32768;
// pins of a level from which on few moves update its state: from 2^16 on a
// 16,384-node Gaussian net takes 42.3 ms instead of 42.0, from 2^22 on a 262k one
// 218.5 instead of 213.5 and the 262k layered net 186.9 instead of 185.6
constexpr int64_t UPDATE_NP = int64_t(1) << 19;

#define STRIDE(i, n, t0, nt) for (int64_t i = (t0); i < (int64_t)(n); i += (nt))
#define G_T0 (blockIdx.x * (int64_t)blockDim.x + threadIdx.x)
#define G_NT ((int64_t)gridDim.x * blockDim.x)

struct RepArrays {
    int32_t n, e, nparts, rounds;
    int32_t *cnt, *linked;
    int32_t *D0;
    long long *psize, *saving;
    int32_t *cutn;   // cut hyperedges of every candidate node
    int32_t *pc;
    int32_t *pred, *succ, *chain, *mvpos;
    long long *cgain;
    unsigned long long *gseq, *acc0;
    int32_t *dDs, *dDd, *viol;
};

__device__ __forceinline__ int64_t rep_zero_span(const RepArrays &R) {
    return max(max((int64_t)R.n, (int64_t)R.nparts + 1), max((int64_t)C_N, (int64_t)R.rounds + 1));
}
// keep 1: the partition is the one of the previous repetition (it applied
// nothing), so D(p), |p|, saving(v) and the cut lists are still valid; keep 2:
// the first three have been updated, and `upd` says what that took
__global__ void k_rep_zero(RepArrays R, int keep, const int32_t *upd) {
    HP_KERNEL_ENTER();
    GRID_STRIDE(i, rep_zero_span(R)) {
        if (i < R.nparts && !keep) {
            R.D0[i] = 0;
            R.psize[i] = 0;
        }
        if (i <= R.nparts) R.pc[i] = 0;
        if (i < R.n) {
            if (!keep) R.saving[i] = 0;
            if (keep != 1) R.cutn[i] = 0;
            R.pred[i] = -1;
            R.succ[i] = -1;
            R.chain[i] = -1;
            R.mvpos[i] = -1;
            R.cgain[i] = 0;
            R.gseq[i] = 0;
            R.acc0[i] = 0;
            R.dDs[i] = 0;
            R.dDd[i] = 0;
            R.viol[i] = 0;
        }
        if (i < C_N) R.cnt[i] = keep == 2 && i >= C_UPD ? upd[U_ACC + i - C_UPD] : 0;
        if (i <= R.rounds) R.linked[i] = 0;
    }
}

// |p| and the single-pin hyperedges' share of D(p).  Up to RN_PARTS parts are
// summed per CTA first: a million nodes over a few hundred parts otherwise
// queue on as many addresses.
constexpr int32_t RN_PARTS = 2048;
__global__ void __launch_bounds__(256) k_rep_nodes(const int32_t *rho, const int32_t *size, const int32_t *singin,
                                                   int32_t n, int32_t nparts, long long *psize, int32_t *D0) {
    HP_KERNEL_ENTER();
    __shared__ uint32_t s_size[RN_PARTS], s_d[RN_PARTS];   // sizes sum to the level-0 node count: 32 bits
    if (nparts > RN_PARTS) {
        GRID_STRIDE(v, (int64_t)n) {
            const int32_t p = rho[v];
            atomicAdd((unsigned long long *)&psize[p], (unsigned long long)size[v]);
            if (singin[v]) atomicAdd(&D0[p], singin[v]);
        }
        return;
    }
    for (int32_t p = threadIdx.x; p < nparts; p += blockDim.x) s_size[p] = s_d[p] = 0;
    __syncthreads();
    GRID_STRIDE(v, (int64_t)n) {
        const int32_t p = rho[v];
        atomicAdd(&s_size[p], (uint32_t)size[v]);
        if (singin[v]) atomicAdd(&s_d[p], (uint32_t)singin[v]);
    }
    __syncthreads();
    for (int32_t p = threadIdx.x; p < nparts; p += blockDim.x) {
        if (s_size[p]) atomicAdd((unsigned long long *)&psize[p], (unsigned long long)s_size[p]);
        if (s_d[p]) atomicAdd(&D0[p], (int32_t)s_d[p]);
    }
}

// Cut hyperedges (|e| >= 2 and more than one part), one bit each: the only
// ones that add to conn(v, p) for p != rho(v).  Also counts, for the step's
// algorithmic bytes, the pins-list entries of the level (sum of lambda(e)),
// the cut incidence entries (sum of |e| over cut hyperedges) and the list
// entries the gain kernels walk for them (sum of |e| lambda(e)), into acc[0..2].
__global__ void k_cut_bits(const int32_t *off, const int32_t *lam, int32_t e, uint32_t *bits, unsigned long long *acc) {
    HP_KERNEL_ENTER();
    const int lane = threadIdx.x & 31;
    unsigned long long lsum = 0, cuts = 0, clam = 0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31u); base < e; base += step) {
        const int64_t i = base + lane;
        bool cut = false;
        if (i < e) {
            const int32_t sz = off[i + 1] - off[i];
            if (sz >= 2) {   // single-pin hyperedges have no pins list
                const int32_t l = lam[i];
                cut = l >= 2;
                lsum += (unsigned long long)l;
                if (cut) {
                    cuts += (unsigned long long)sz;
                    clam += (unsigned long long)sz * (unsigned long long)l;
                }
            }
        }
        const uint32_t word = __ballot_sync(0xffffffffu, cut);
        if (lane == 0) bits[base >> 5] = word;
    }
    // one update of each counter per CTA (all CTAs hit the same three words)
    __shared__ unsigned long long s_acc[3];
    if (threadIdx.x < 3) s_acc[threadIdx.x] = 0;
    __syncthreads();
    for (int o = 16; o > 0; o >>= 1) {
        lsum += __shfl_down_sync(0xffffffffu, lsum, o);
        cuts += __shfl_down_sync(0xffffffffu, cuts, o);
        clam += __shfl_down_sync(0xffffffffu, clam, o);
    }
    if (lane == 0 && (lsum | cuts | clam)) {
        atomicAdd(&s_acc[0], lsum);
        atomicAdd(&s_acc[1], cuts);
        atomicAdd(&s_acc[2], clam);
    }
    __syncthreads();
    if (threadIdx.x < 3 && s_acc[threadIdx.x]) atomicAdd(&acc[threadIdx.x], s_acc[threadIdx.x]);
}
// The cut hyperedges of every candidate (saving(v) > 0), gathered at the front
// of v's own incidence segment (in no particular order: the gains are sums):
// one pass over the incidence, a warp's entries of one node taking their
// places by one atomic.  Bound by the reads of the incidence (8 B an entry, 4
// where no node of a warp is a candidate).  Flagging, scanning and filling
// lists of all nodes took 166 + 45 + 62 us a repetition on the 1M Gaussian net.
__global__ void k_cut_lists(const int32_t *ioff, const int32_t *inc, const int32_t *inode, int64_t np,
                            const long long *saving, const uint32_t *bits, int32_t *cut, int32_t *cutn) {
    HP_KERNEL_ENTER();
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31u); base < np; base += step) {
        const int64_t t = base + lane;
        const int32_t v = t < np ? inode[t] : -1;
        const bool cand = v >= 0 && saving[v] > 0;
        if (!__any_sync(FULL, cand)) continue;
        int32_t e = 0;
        bool f = false;
        if (cand) {
            e = inc[t];
            f = (bits[e >> 5] >> (e & 31)) & 1u;
        }
        // the lanes of v: from the last head up to this lane to the one before the next head
        const int32_t pv = __shfl_up_sync(FULL, v, 1);
        const unsigned heads = __ballot_sync(FULL, lane == 0 || pv != v), fm = __ballot_sync(FULL, f);
        const unsigned upto = (2u << lane) - 1u;
        const int first = 31 - __clz((int)(heads & upto));
        const unsigned later = heads & ~upto;
        const unsigned run = fm & ~((1u << first) - 1u) & (later ? (later & (0u - later)) - 1u : FULL);
        int32_t at = 0;
        if (lane == first && run) at = atomicAdd(&cutn[v], __popc(run));
        at = __shfl_sync(FULL, at, first);
        if (f) cut[ioff[v] + at + __popc(run & ((1u << lane) - 1u))] = e;
    }
}

// candidates: nodes that can spare a cut, by number of cut hyperedges:
// up to GW_DEG a warp each, up to HUB_DEG a CTA each, more a large CTA each
constexpr int32_t HUB_DEG = 1024, GW_DEG = 256;
__global__ void k_candidates(const long long *saving, const int32_t *cutn, int32_t n, int32_t *list, int32_t *cnt,
                             int32_t *hubs, int32_t *hcnt, int32_t *wlist, int32_t *wcnt) {
    HP_KERNEL_ENTER();
    GRID_STRIDE(v, (int64_t)n) {
        if (saving[v] > 0) {
            const int32_t d = cutn[v];
            if (d > HUB_DEG) hubs[atomicAdd(hcnt, 1)] = (int32_t)v;
            else if (d <= GW_DEG) wlist[atomicAdd(wcnt, 1)] = (int32_t)v;
            else list[atomicAdd(cnt, 1)] = (int32_t)v;
        }
    }
}

// ---------------------------------------------------------------- phases
// Each phase is a strided loop (t0, nt): a kernel runs it over its grid, the
// single-CTA sequence kernels over their block, with a barrier in between.

// sort keys (p_s, gbound - gain, node): ascending = (p_s asc, gain desc, node asc)
__device__ void ph_move_keys(const Moves &M, int32_t m, long long gbound, int gb, int nb, int field, uint64_t *keys,
                             uint32_t *idx, int init_idx, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        if (init_idx) idx[i] = (uint32_t)i;
        uint32_t k = idx[i];
        uint64_t g = (uint64_t)(gbound - M.gain[k]);
        if (field < 0) keys[i] = ((uint64_t)M.src[k] << (gb + nb)) | (g << nb) | (uint64_t)M.node[k];
        else keys[i] = field == 0 ? (uint64_t)M.node[k] : field == 1 ? g : (uint64_t)M.src[k];
    }
}
// the moves in sorted order, with the size and |in| of each moved node
__device__ void ph_gather(const Moves &M, const uint32_t *idx, int32_t m, const Moves &S, int32_t *pc,
                          const int32_t *size, const int32_t *nin, int32_t *msz, int32_t *mni, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        uint32_t k = idx[i];
        const int32_t v = M.node[k];
        S.node[i] = v;
        S.src[i] = M.src[k];
        S.dst[i] = M.dst[k];
        S.gain[i] = M.gain[k];
        msz[i] = size[v];
        mni[i] = nin[v];
        atomicAdd(&pc[M.src[k]], 1);
    }
}

struct ChainCtx {
    int32_t window;
    const int32_t *node, *src, *dst, *size, *nin;
    const int32_t *msz, *mni;   // size and |in| of the node of each sorted move
    const long long *gain;
    const int32_t *first;   // [nparts+1]: moves leaving p are [first[p], first[p+1])
    int32_t *pred, *succ, *choice;
    unsigned long long *pen, *minpen;     // general acceptance
    int32_t *accnode;
    unsigned long long *acc[3];           // packed acceptance (penalty < 2^32)
    int32_t *linked;                      // linked[r]: round r linked something
};

// The pick of one free chain end i by its warp (packed acceptance, 64-bit
// grades: |G| < 2^62 when the weights sum to at most 2^38): among the first
// `window` moves of [j0, jend) not taken and not i, the one of maximum grade
// G = gain * 10^7 - penalty, earliest on ties; lanes over moves.  The moves
// leaving a part are sorted by gain, and no penalty is negative, so the scan
// ends at the first move whose gain * 10^7 does not exceed the best grade
// found: usually after the moves that tie with the best gain.  Bound by the
// latency of the scan's steps.  A thread per free end, four moves at a time
// from L2 and to the window's end, took 372 us a call of k_seq_cluster on the
// 262k layered net (1,831 moves, 13 rounds on average), 556 us on the 20k
// irregular net (1,543 moves, 6.5 rounds) and 45 us a round of the device-wide
// form on the 1M Gaussian net; a warp per free end, from shared memory in the
// cluster kernel: 116, 119 and 12.6 us.
template <class Taken, class Gain, class Sn>
__device__ __forceinline__ int32_t warp_pick(int32_t i, int32_t jbeg, int32_t jend, int32_t window, int32_t szi,
                                             int32_t nii, Taken taken, Gain gain, Sn sn, uint32_t &pen_out) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    long long bG = LLONG_MIN;
    int32_t best = -1, seen = 0;
    uint32_t bpen = 0;
    for (int32_t j0 = jbeg; j0 < jend && seen < window; j0 += 32) {
        const int32_t j = j0 + lane;
        const bool in = j < jend;
        const long long top = in ? gain(j) * 10000000ll : 0;
        if (__any_sync(FULL, bG >= __shfl_sync(FULL, top, 0))) break;
        bool ok = in && j != i && !taken(j);
        const unsigned bal = __ballot_sync(FULL, ok);
        ok = ok && seen + __popc(bal & lt) < window;
        if (ok) {
            const int2 x = sn(j);
            const long long ds = (long long)szi - x.x, di = (long long)nii - x.y;
            const long long pen = 10 * (ds < 0 ? -ds : ds) + (di < 0 ? -di : di);
            if (top - pen > bG) {
                bG = top - pen;
                best = j;
                bpen = (uint32_t)pen;
            }
        }
        seen += __popc(bal);
    }
    // maximum grade over the lanes (high word, then low word), then the earliest move
    const int32_t hi = (int32_t)(bG >> 32);
    const int32_t mhi = __reduce_max_sync(FULL, hi);
    const uint32_t mlo = __reduce_max_sync(FULL, hi == mhi ? (uint32_t)bG : 0u);
    const bool top_lane = best >= 0 && hi == mhi && (uint32_t)bG == mlo;
    const uint32_t bj = __reduce_min_sync(FULL, top_lane ? (uint32_t)best : 0xffffffffu);
    if (bj == 0xffffffffu) return -1;
    pen_out = __shfl_sync(FULL, bpen, (int)(bj - (uint32_t)jbeg) & 31);
    return (int32_t)bj;
}

// Sec. VI-C: every free chain end picks, among the first `window` moves
// leaving its destination that have no predecessor, the one of maximum
// grade G = gain(m)*10^7 - 10|size(n)-size(m)| - |nin(n)-nin(m)|, earliest on
// ties.  For a chosen move all choosers share gain(m), so the acceptor of
// maximum (G, node id) is the chooser of minimum penalty, then maximum id.
__device__ void ph_choose(const ChainCtx &C, int32_t m, int64_t t0, int64_t nt) {
    constexpr int B = 4;   // candidates loaded together, ahead of their evaluation
    STRIDE(i0, m, t0, nt) {
        int32_t i = (int32_t)i0;
        C.choice[i] = -1;
        C.minpen[i] = ~0ull;
        C.accnode[i] = -1;
        if (C.succ[i] >= 0) continue;
        const int32_t d = C.dst[i];
        int32_t seen = 0, best = -1;
        __int128 bG = 0;
        unsigned long long bpen = 0;
        const int32_t szi = C.msz[i], nii = C.mni[i];
        const int32_t jend = C.first[d + 1];
        for (int32_t j0 = C.first[d]; j0 < jend && seen < C.window; j0 += B) {
            int32_t pr[B], sz[B], ni[B];
            long long gn[B];
#pragma unroll
            for (int u = 0; u < B; u++) {
                const int32_t j = j0 + u;
                const bool ok = j < jend;
                pr[u] = ok ? C.pred[j] : 0;
                sz[u] = ok ? C.msz[j] : 0;
                ni[u] = ok ? C.mni[j] : 0;
                gn[u] = ok ? C.gain[j] : 0;
            }
#pragma unroll
            for (int u = 0; u < B; u++) {
                const int32_t j = j0 + u;
                if (j >= jend || seen >= C.window) break;
                if (best >= 0 && (__int128)gn[u] * 10000000 <= bG) {   // none from here on has a higher grade
                    seen = C.window;
                    break;
                }
                if (pr[u] >= 0 || j == i) continue;
                seen++;
                const long long ds = (long long)szi - sz[u], di = (long long)nii - ni[u];
                const unsigned long long pen =
                    10ull * (unsigned long long)(ds < 0 ? -ds : ds) + (unsigned long long)(di < 0 ? -di : di);
                const __int128 G = (__int128)gn[u] * 10000000 - (__int128)pen;
                if (best < 0 || G > bG) {
                    best = j;
                    bG = G;
                    bpen = pen;
                }
            }
        }
        C.choice[i] = best;
        C.pen[i] = bpen;
    }
}
__device__ void ph_accept_min(const ChainCtx &C, int32_t m, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        int32_t j = C.choice[i];
        if (j >= 0) atomicMin(&C.minpen[j], C.pen[i]);
    }
}
__device__ void ph_accept_id(const ChainCtx &C, int32_t m, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        int32_t j = C.choice[i];
        if (j >= 0 && C.pen[i] == C.minpen[j]) atomicMax(&C.accnode[j], C.node[i]);
    }
}
// link the winners; clear the packed slots of the next round
__device__ void ph_link(const ChainCtx &C, int r, int packed, int32_t m, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        int32_t j = C.choice[i];
        bool won = false;
        if (j >= 0) {
            if (packed)
                won = ((r & 1) ? C.acc[1] : C.acc[0])[j] ==
                      (((0xffffffffull - C.pen[i]) << 32) | (unsigned long long)(uint32_t)C.node[i]);
            else
                won = C.pen[i] == C.minpen[j] && C.accnode[j] == C.node[i];
        }
        if (won) {
            C.pred[j] = (int32_t)i;
            C.succ[i] = j;
            C.linked[r] = 1;
        }
        if (packed) ((r & 1) ? C.acc[0] : C.acc[1])[i] = 0;
    }
}

// One chaining round with one barrier (packed acceptance only).  Round r's
// winners are linked in round r + 1's pass instead of a pass of their own:
// the chooser of a move j won it in round r iff acc_r[j] holds its key, and a
// move j already has a predecessor in round r + 1 iff pred[j] >= 0 (rounds
// before r) or acc_r[j] != 0 (round r: every chosen move gets exactly one
// winner).  The slots rotate over three arrays, round r in acc[r % 3]; the
// pass of round r clears acc[(r + 1) % 3], which the pass of round r - 1 read
// and the pass of round r + 1 fills.  The links of the last round are made by
// ph_link_last.  The result equals the two-pass round above.
__device__ __forceinline__ unsigned long long chain_key(unsigned long long pen, int32_t node) {
    return ((0xffffffffull - pen) << 32) | (unsigned long long)(uint32_t)node;
}
// The free ends are dealt to the warps a lane at a time (a warp of few moves
// otherwise scans for 32 of them one after another).
template <class Taken, class Gain, class Sn>
__device__ void ph_round(const ChainCtx &C, int r, int32_t m, int gw, int nw, Taken taken, Gain gain, Sn sn) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned long long *accr = C.acc[r % 3], *accp = C.acc[(r + 2) % 3], *accn = C.acc[(r + 1) % 3];
    for (int32_t base = 0; base < m; base += 32 * nw) {
        const int32_t i = base + lane * nw + gw;
        bool free_end = false;
        int32_t j0 = 0, jend = 0, szi = 0, nii = 0, vi = 0;
        if (i < m) {
            free_end = C.succ[i] < 0;
            vi = C.node[i];
            if (r > 0) {
                const int32_t j = C.choice[i];
                if (j >= 0 && accp[j] == chain_key(C.pen[i], vi)) {
                    C.pred[j] = i;
                    C.succ[i] = j;
                    free_end = false;
                }
            }
            accn[i] = 0;
            if (free_end) {
                const int32_t d = C.dst[i];
                j0 = C.first[d];
                jend = C.first[d + 1];
                szi = C.msz[i];
                nii = C.mni[i];
            }
        }
        int32_t best = -1;
        uint32_t pen = 0;
        unsigned todo = __ballot_sync(FULL, free_end && j0 < jend);
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            uint32_t p = 0;
            const int32_t x = warp_pick(__shfl_sync(FULL, i, l), __shfl_sync(FULL, j0, l), __shfl_sync(FULL, jend, l),
                                        C.window, __shfl_sync(FULL, szi, l), __shfl_sync(FULL, nii, l), taken, gain,
                                        sn, p);
            if (lane == l) {
                best = x;
                pen = p;
            }
        }
        if (i < m) {
            C.choice[i] = best;
            C.pen[i] = pen;
            if (best >= 0) {
                atomicMax(&accr[best], chain_key(pen, vi));
                C.linked[r] = 1;
            }
        }
    }
}
// the links of round r, the last round run (nothing when it chose nothing)
__device__ void ph_link_last(const ChainCtx &C, int r, int32_t m, int64_t t0, int64_t nt) {
    const unsigned long long *accr = C.acc[r % 3];
    STRIDE(i0, m, t0, nt) {
        const int32_t i = (int32_t)i0, j = C.choice[i];
        if (j >= 0 && accr[j] == chain_key(C.pen[i], C.node[i])) {
            C.pred[j] = i;
            C.succ[i] = j;
        }
    }
}

struct SeqCtx {
    const int32_t *node, *pred, *succ;
    const long long *gain;
    int32_t *chain, *pos, *clen;
    long long *cgain;
    uint32_t *err;
};
__device__ void ph_path_heads(const SeqCtx &S, int32_t m, int64_t t0, int64_t nt) {
    STRIDE(i0, m, t0, nt) {
        int32_t i = (int32_t)i0;
        if (S.pred[i] >= 0) continue;
        long long g = 0;
        int32_t k = 0;
        for (int32_t j = i; j >= 0; j = S.succ[j]) {
            if (k > m) {
                atomicOr(S.err, E_TIMEOUT);
                break;
            }
            S.chain[j] = i;
            S.pos[j] = k++;
            g += S.gain[j];
        }
        S.clen[i] = k;
        S.cgain[i] = g;
    }
}
// moves left unassigned lie on cycles; the member of smallest node id heads it
__device__ void ph_cycle_heads(const SeqCtx &S, int32_t m, int64_t t0, int64_t nt) {
    STRIDE(i0, m, t0, nt) {
        int32_t i = (int32_t)i0;
        if (S.chain[i] >= 0) continue;
        int32_t mn = S.node[i], k = 0;
        for (int32_t j = S.succ[i]; j != i; j = S.succ[j]) {
            if (j < 0 || ++k > m) {
                atomicOr(S.err, E_INTERNAL);
                mn = -1;
                break;
            }
            mn = min(mn, S.node[j]);
        }
        if (mn != S.node[i]) continue;
        long long g = 0;
        int32_t c = 0, j = i;
        do {
            S.chain[j] = i;
            S.pos[j] = c++;
            g += S.gain[j];
            j = S.succ[j];
        } while (j != i && c <= m);
        S.clen[i] = c;
        S.cgain[i] = g;
    }
}
__device__ void ph_head_collect(const SeqCtx &S, int32_t m, uint32_t *heads, int32_t *nh, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        if (S.chain[i] == (int32_t)i) heads[atomicAdd(nh, 1)] = (uint32_t)i;
    }
}
// key (cgbound - chain gain, head node): ascending = (total gain desc, head node asc)
__device__ void ph_head_keys(const uint32_t *heads, int32_t nh, const long long *cgain, const int32_t *node,
                             long long cgbound, int nb, int field, uint64_t *keys, int64_t t0, int64_t nt) {
    STRIDE(k, nh, t0, nt) {
        uint32_t h = heads[k];
        uint64_t gk = (uint64_t)(cgbound - cgain[h]);
        if (field < 0) keys[k] = (gk << nb) | (uint64_t)node[h];
        else keys[k] = field == 0 ? (uint64_t)node[h] : gk;
    }
}
__device__ void ph_chain_lens(const uint32_t *heads, int32_t nh, const int32_t *clen, int64_t cap, int32_t *lens,
                              int64_t t0, int64_t nt) {
    STRIDE(k, cap, t0, nt) lens[k] = k < nh ? clen[heads[k]] : 0;
}
__device__ void ph_chain_start(const uint32_t *heads, int32_t nh, const int32_t *starts, int32_t *cstart, int64_t t0,
                               int64_t nt) {
    STRIDE(k, nh, t0, nt) cstart[heads[k]] = starts[k];
}
__device__ void ph_seq_pos(const int32_t *chain, const int32_t *pos, const int32_t *cstart, int32_t m,
                           const int32_t *node, int32_t *seqmove, int32_t *mvpos, int64_t t0, int64_t nt) {
    STRIDE(i, m, t0, nt) {
        int32_t k = cstart[chain[i]] + pos[i];
        seqmove[k] = (int32_t)i;
        mvpos[node[i]] = k;
    }
}

// Sec. VI-D: two capacity entries per move k, in sequence order: at p_s
// (-size, dD_s) and at p_d (+size, dD_d); sorted stably by part, each part's
// entries are walked in sequence order and each change of its validity is
// recorded at the move that caused it.
struct ValCtx {
    const int32_t *seqmove, *size, *singin, *dDs, *dDd, *D0;
    const unsigned long long *gseq;
    Moves S;
    const long long *psize;
    uint32_t *vkey, *vidx;
    long long *vsz;
    int32_t *vdd, *viol;
    int32_t omega, delta;
    long long *gsz, *gdd, *esz, *edd;  // [2m] events in part order; their exclusive prefix sums
    int32_t *vhead;                    // [nparts] first event of each part
};
__device__ void ph_val_entries(const ValCtx &V, int32_t m, int64_t t0, int64_t nt) {
    STRIDE(k, m, t0, nt) {
        int32_t i = V.seqmove[k];
        int32_t v = V.S.node[i];
        long long sz = V.size[v];
        V.vkey[2 * k] = (uint32_t)V.S.src[i];
        V.vidx[2 * k] = (uint32_t)(2 * k);
        V.vsz[2 * k] = -sz;
        V.vdd[2 * k] = V.dDs[k] - V.singin[v];
        V.vkey[2 * k + 1] = (uint32_t)V.S.dst[i];
        V.vidx[2 * k + 1] = (uint32_t)(2 * k + 1);
        V.vsz[2 * k + 1] = sz;
        V.vdd[2 * k + 1] = V.dDd[k] + V.singin[v];
    }
}
// Validity of every prefix (Sec. VI-D) from the c = 2m capacity events
// sorted by part (stably, so in sequence order within a part).  A part's
// running size and distinct-inbound count after each of its events are
// global prefix sums minus the prefix at the part's first event; every event
// at which the part turns valid or invalid adds -1 / +1 to the violation
// count of its move.
__device__ void ph_val_gather(const ValCtx &V, int32_t c, int64_t t0, int64_t nt) {
    STRIDE(j, c, t0, nt) {
        const uint32_t x = V.vidx[j];
        V.gsz[j] = V.vsz[x];
        V.gdd[j] = V.vdd[x];
        const uint32_t p = V.vkey[j];
        if (j == 0 || V.vkey[j - 1] != p) V.vhead[p] = (int32_t)j;
    }
}
__device__ void ph_val_trans(const ValCtx &V, int32_t c, int64_t t0, int64_t nt) {
    STRIDE(j, c, t0, nt) {
        const uint32_t p = V.vkey[j];
        const int32_t h = V.vhead[p];
        const long long bs = V.psize[p] + (V.esz[j] - V.esz[h]), bd = (long long)V.D0[p] + (V.edd[j] - V.edd[h]);
        const long long as = bs + V.gsz[j], ad = bd + V.gdd[j];
        const bool vb = bs <= V.omega && bd <= V.delta, va = as <= V.omega && ad <= V.delta;
        if (vb != va) atomicAdd(&V.viol[V.vidx[j] >> 1], va ? -1 : 1);
    }
}
__device__ int32_t ph_initial_bad(const long long *psize, const int32_t *D0, int32_t nparts, int32_t omega,
                                  int32_t delta, int64_t t0, int64_t nt) {
    int32_t c = 0;
    STRIDE(p, nparts, t0, nt) c += (psize[p] > omega || D0[p] > delta) ? 1 : 0;
    return c;
}
__device__ void ph_apply(const int32_t *seqmove, const int32_t *node, const int32_t *dst, int32_t L, int32_t *rho,
                         int64_t t0, int64_t nt) {
    STRIDE(k, L, t0, nt) {
        int32_t i = seqmove[k];
        rho[node[i]] = dst[i];
    }
}

// ---- block-level helpers of the single-CTA kernels (blockDim = SEQ_T)
// the same for int64 values, in place allowed (in == out)
__device__ void block_scan_excl_ll(const long long *in, long long *out, int64_t n, long long *s_tmp) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    long long carry = 0;
    for (int64_t base = 0; base < n; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        long long x = i < n ? in[i] : 0, inc = x;
        for (int o = 1; o < 32; o <<= 1) {
            long long u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) s_tmp[wid] = inc;
        __syncthreads();
        if (wid == 0) {
            long long y = lane < nw ? s_tmp[lane] : 0, yi = y;
            for (int o = 1; o < 32; o <<= 1) {
                long long u = __shfl_up_sync(0xffffffffu, yi, o);
                if (lane >= o) yi += u;
            }
            if (lane < nw) s_tmp[lane] = yi - y;
            if (lane == nw - 1) s_tmp[32] = yi;
        }
        __syncthreads();
        if (i < n) out[i] = carry + s_tmp[wid] + inc - x;
        carry += s_tmp[32];
        __syncthreads();
    }
}

// best prefix (Sec. VI-D): max cumulative gain over prefixes with zero
// invalid parts, longest on ties; one CTA of 1024 threads
__device__ void best_prefix_block(const unsigned long long *gseq, const int32_t *violc, int32_t m, int32_t bad0,
                                  int32_t *best_len, long long *best_gain) {
    __shared__ long long s_g[32];
    __shared__ int32_t s_k[32];
    __shared__ long long s_carry_g;
    __shared__ int32_t s_carry_v;
    if (threadIdx.x == 0) {
        s_carry_g = 0;
        s_carry_v = bad0;
    }
    __syncthreads();
    long long bestg = 0;
    int32_t bestk = 0;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int32_t base = 0; base < m; base += 1024) {
        int32_t k = base + threadIdx.x;
        long long g = k < m ? (long long)gseq[k] : 0;
        int32_t dv = k < m ? violc[k] : 0;
        long long gi = g;
        int32_t vi = dv;
        for (int o = 1; o < 32; o <<= 1) {
            long long ug = __shfl_up_sync(0xffffffffu, gi, o);
            int32_t uv = __shfl_up_sync(0xffffffffu, vi, o);
            if (lane >= o) {
                gi += ug;
                vi += uv;
            }
        }
        if (lane == 31) {
            s_g[wid] = gi;
            s_k[wid] = vi;
        }
        __syncthreads();
        if (wid == 0) {
            long long x = s_g[lane];
            int32_t y = s_k[lane];
            long long xi = x;
            int32_t yi = y;
            for (int o = 1; o < 32; o <<= 1) {
                long long ux = __shfl_up_sync(0xffffffffu, xi, o);
                int32_t uy = __shfl_up_sync(0xffffffffu, yi, o);
                if (lane >= o) {
                    xi += ux;
                    yi += uy;
                }
            }
            s_g[lane] = xi - x;
            s_k[lane] = yi - y;
        }
        __syncthreads();
        long long cum = s_carry_g + s_g[wid] + gi;
        int32_t vio = s_carry_v + s_k[wid] + vi;
        if (k < m && vio == 0 && cum >= bestg) {
            bestg = cum;
            bestk = k + 1;
        }
        __syncthreads();
        if (threadIdx.x == 1023) {
            s_carry_g = cum;
            s_carry_v = vio;
        }
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) {
        long long og = __shfl_down_sync(0xffffffffu, bestg, o);
        int32_t ok = __shfl_down_sync(0xffffffffu, bestk, o);
        if (og > bestg || (og == bestg && ok > bestk)) {
            bestg = og;
            bestk = ok;
        }
    }
    if (lane == 0) {
        s_g[wid] = bestg;
        s_k[wid] = bestk;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 32; k++)
            if (s_g[k] > bestg || (s_g[k] == bestg && s_k[k] > bestk)) {
                bestg = s_g[k];
                bestk = s_k[k];
            }
        *best_gain = bestg;
        *best_len = bestg > 0 ? bestk : 0;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- multi-kernel path
__global__ void k_move_keys(const Moves M, const int32_t *cntp, long long gbound, int gb, int nb, int field,
                            uint64_t *keys, uint32_t *idx, int init_idx) {
    HP_KERNEL_ENTER();
    ph_move_keys(M, *cntp, gbound, gb, nb, field, keys, idx, init_idx, G_T0, G_NT);
}
__global__ void k_gather_moves(const Moves M, const uint32_t *idx, const int32_t *cntp, Moves S, int32_t *pc,
                               const int32_t *size, const int32_t *nin, int32_t *msz, int32_t *mni) {
    HP_KERNEL_ENTER();
    ph_gather(M, idx, *cntp, S, pc, size, nin, msz, mni, G_T0, G_NT);
}
__global__ void k_choose(ChainCtx C, const int32_t *mcount, int r) {
    HP_KERNEL_ENTER();
    if (r > 0 && !C.linked[r - 1]) return;
    ph_choose(C, *mcount, G_T0, G_NT);
}
// packed acceptance: a warp per free end
__global__ void __launch_bounds__(128) k_choose_warp(ChainCtx C, const int32_t *mcount, int r) {
    HP_KERNEL_ENTER();
    if (r > 0 && !C.linked[r - 1]) return;
    const int32_t m = *mcount;
    const int lane = threadIdx.x & 31;
    unsigned long long *acc = (r & 1) ? C.acc[1] : C.acc[0];
    for (int64_t x = G_T0 >> 5; x < m; x += G_NT >> 5) {
        const int32_t i = (int32_t)x;
        int32_t best = -1;
        uint32_t pen = 0;
        if (C.succ[i] < 0) {
            const int32_t d = C.dst[i];
            best = warp_pick(i, C.first[d], C.first[d + 1], C.window, C.msz[i], C.mni[i],
                             [&](int32_t j) { return C.pred[j] >= 0; }, [&](int32_t j) { return C.gain[j]; },
                             [&](int32_t j) { return make_int2(C.msz[j], C.mni[j]); }, pen);
        }
        if (lane == 0) {
            C.choice[i] = best;
            C.pen[i] = pen;
            if (best >= 0) atomicMax(&acc[best], chain_key(pen, C.node[i]));
        }
    }
}
__global__ void k_accept_min(ChainCtx C, const int32_t *mcount, int r) {
    HP_KERNEL_ENTER();
    if (r > 0 && !C.linked[r - 1]) return;
    ph_accept_min(C, *mcount, G_T0, G_NT);
}
__global__ void k_accept_id(ChainCtx C, const int32_t *mcount, int r) {
    HP_KERNEL_ENTER();
    if (r > 0 && !C.linked[r - 1]) return;
    ph_accept_id(C, *mcount, G_T0, G_NT);
}
__global__ void k_link(ChainCtx C, const int32_t *mcount, int r, int packed) {
    HP_KERNEL_ENTER();
    if (r > 0 && !C.linked[r - 1]) return;
    ph_link(C, r, packed, *mcount, G_T0, G_NT);
}

__global__ void k_path_heads(SeqCtx S, const int32_t *mcount) { HP_KERNEL_ENTER(); ph_path_heads(S, *mcount, G_T0, G_NT); }
__global__ void k_cycle_heads(SeqCtx S, const int32_t *mcount) { HP_KERNEL_ENTER(); ph_cycle_heads(S, *mcount, G_T0, G_NT); }
__global__ void k_head_collect(SeqCtx S, const int32_t *mcount, uint32_t *heads, int32_t *nh) {
    HP_KERNEL_ENTER();
    ph_head_collect(S, *mcount, heads, nh, G_T0, G_NT);
}
__global__ void k_head_keys(const uint32_t *heads, const int32_t *nh, const long long *cgain, const int32_t *node,
                            long long cgbound, int nb, int field, uint64_t *keys) {
    HP_KERNEL_ENTER();
    ph_head_keys(heads, *nh, cgain, node, cgbound, nb, field, keys, G_T0, G_NT);
}
__global__ void k_chain_lens(const uint32_t *heads, const int32_t *nh, const int32_t *clen, int32_t cap,
                             int32_t *lens) {
    HP_KERNEL_ENTER();
    ph_chain_lens(heads, *nh, clen, cap, lens, G_T0, G_NT);
}
__global__ void k_chain_start(const uint32_t *heads, const int32_t *nh, const int32_t *starts, int32_t *cstart) {
    HP_KERNEL_ENTER();
    ph_chain_start(heads, *nh, starts, cstart, G_T0, G_NT);
}
__global__ void k_seq_pos(const int32_t *chain, const int32_t *pos, const int32_t *cstart, const int32_t *mcount,
                          const int32_t *node, int32_t *seqmove, int32_t *mvpos) {
    HP_KERNEL_ENTER();
    ph_seq_pos(chain, pos, cstart, *mcount, node, seqmove, mvpos, G_T0, G_NT);
}
__global__ void k_val_entries(ValCtx V, const int32_t *mcount, int32_t *nv) {
    HP_KERNEL_ENTER();
    const int32_t m = *mcount;
    if (blockIdx.x == 0 && threadIdx.x == 0) *nv = 2 * m;
    ph_val_entries(V, m, G_T0, G_NT);
}
__global__ void k_val_gather(ValCtx V, const int32_t *nv) { HP_KERNEL_ENTER(); ph_val_gather(V, *nv, G_T0, G_NT); }
__global__ void k_val_trans(ValCtx V, const int32_t *nv) { HP_KERNEL_ENTER(); ph_val_trans(V, *nv, G_T0, G_NT); }
__global__ void k_initial_bad(const long long *psize, const int32_t *D0, int32_t nparts, int32_t omega, int32_t delta,
                              int32_t *bad) {
    HP_KERNEL_ENTER();
    int32_t c = ph_initial_bad(psize, D0, nparts, omega, delta, G_T0, G_NT);
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(bad, c);
}
__global__ void __launch_bounds__(1024) k_best_prefix(const unsigned long long *gseq, const int32_t *violc,
                                                      const int32_t *mcount, const int32_t *bad0, int32_t *best_len,
                                                      long long *best_gain) {
    HP_KERNEL_ENTER();
    best_prefix_block(gseq, violc, *mcount, *bad0, best_len, best_gain);
}
__global__ void k_apply(const int32_t *seqmove, const int32_t *node, const int32_t *dst, const int32_t *lenp,
                        int32_t *rho) {
    HP_KERNEL_ENTER();
    ph_apply(seqmove, node, dst, *lenp, rho, G_T0, G_NT);
}

// ---------------------------------------------------------------- cluster path (M <= sq_max<uint64_t>())
// Sort of the moves, chaining rounds, chain order and sequence positions of
// one repetition by one thread-block cluster (hp_cluster.cuh): every phase is
// a strided loop over the cluster's threads on the global arrays (L2
// resident at these sizes), separated by cluster barriers; the two sorts are
// cluster radix sorts.  Eight times the threads of one CTA, so the latency of
// each phase's global loads is spread over 8 SMs.
static_assert(SQ_T == SEQ_T, "cluster CTA size");
constexpr int32_t SEQ_CLUSTER_M = 4096;   // moves of a larger level sequenced by one cluster
// moves whose gain, size and |in| (16 bytes each) fit the sort buffers of one CTA
constexpr int32_t CHAIN_SMEM_M = (int32_t)(SQ_SMEM / 16);
static_assert(CHAIN_SMEM_M / 32 <= 32 * 256, "their taken bits fit the digit counters");
static_assert(SMALL_LEVEL <= sq_max<uint64_t>() && 2 * SMALL_LEVEL <= sq_max<uint32_t>(),
              "a small level's moves fit the cluster sorts");

struct ClusterSeqArgs {
    Moves M, S;
    uint64_t *keys, *hkeys;
    uint32_t *idx, *heads;
    int32_t *first, *lens, *starts, *cstart, *seqmove, *mvpos, *cnt;
    ChainCtx C;
    SeqCtx Q;
    int32_t nparts, rounds, packed, gb, nb, sb, cgb;
    long long gbound, cgbound;
};

// first[p] = number of sorted moves leaving a part below p, for p in [0, nparts]
__device__ void ph_first_of(const int32_t *src, int32_t m, int32_t nparts, int32_t *first, int64_t t0, int64_t nt) {
    STRIDE(p, (int64_t)nparts + 1, t0, nt) {
        int32_t a = 0, b = m;
        while (a < b) {
            const int32_t mid = (a + b) >> 1;
            if (src[mid] < (int32_t)p) a = mid + 1;
            else b = mid;
        }
        first[p] = a;
    }
}

// The chaining rounds of at most CHAIN_SMEM_M moves by one cluster (packed
// acceptance).  Every CTA keeps a copy of what the window scans read: gain,
// size and |in| of each move, and a bit per move with a predecessor, to which
// each round adds the moves chosen in the one before; a thread keeps its own
// moves' state in registers, so a round reads nothing but the previous
// round's slots: one trip to L2, the scans, one cluster barrier.  Keeping that
// state in global memory cost four dependent trips a round (8.6 us a round of
// 1,800 moves on the 262k layered net; 6.2 this way).
__device__ __forceinline__ void chain_rounds_smem(const ChainCtx &C, const Moves &S, int rounds, int32_t m,
                                                  cg::cluster_group &cl, unsigned char *smem, uint32_t *s_taken) {
    constexpr int NS = (CHAIN_SMEM_M + SQ_CS * SQ_T - 1) / (SQ_CS * SQ_T);   // moves a thread owns
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int gw = (int)cl.block_rank() * (SQ_T / 32) + wid, nw = SQ_CS * (SQ_T / 32);
    long long *c_gain = reinterpret_cast<long long *>(smem);
    int2 *c_sn = reinterpret_cast<int2 *>(c_gain + CHAIN_SMEM_M);
    for (int32_t j = threadIdx.x; j < m; j += SQ_T) {
        c_gain[j] = S.gain[j];
        c_sn[j] = make_int2(C.msz[j], C.mni[j]);
    }
    for (int32_t x = threadIdx.x; x < (m + 31) / 32; x += SQ_T) s_taken[x] = 0;
    // the free ends are dealt to the warps a lane at a time (a warp of few
    // moves otherwise scans for 32 of them one after another)
    int32_t j0[NS], jend[NS], vi[NS], choice[NS];
    uint32_t pen[NS];
    bool free_end[NS];
#pragma unroll
    for (int q = 0; q < NS; q++) {
        const int32_t i = q * (32 * nw) + lane * nw + gw;
        j0[q] = jend[q] = vi[q] = 0;
        choice[q] = -1;
        pen[q] = 0;
        free_end[q] = i < m;
        if (i < m) {
            const int32_t d = S.dst[i];
            j0[q] = C.first[d];
            jend[q] = C.first[d + 1];
            vi[q] = S.node[i];
        }
    }
    __syncthreads();
    // links the winners of the round whose slots are acc
    auto link = [&](const unsigned long long *acc) {
#pragma unroll
        for (int q = 0; q < NS; q++) {
            const int32_t i = q * (32 * nw) + lane * nw + gw, j = choice[q];
            if (j >= 0 && acc[j] == chain_key(pen[q], vi[q])) {
                C.pred[j] = i;
                C.succ[i] = j;
                free_end[q] = false;
            }
        }
    };
    int rr = 0;
    for (; rr < rounds; rr++) {
        unsigned long long *accr = C.acc[rr % 3], *accp = C.acc[(rr + 2) % 3], *accn = C.acc[(rr + 1) % 3];
        if (rr > 0) {
            const int32_t go = *(volatile int32_t *)&C.linked[rr - 1];
            for (int32_t x = wid; x < (m + 31) / 32; x += SQ_T / 32) {
                const int32_t j = 32 * x + lane;
                const unsigned b = __ballot_sync(FULL, j < m && accp[j] != 0ull);
                if (lane == 0) s_taken[x] |= b;
            }
            if (!go) break;   // the same for the whole cluster
            link(accp);
            __syncthreads();
        }
        bool any = false;
#pragma unroll
        for (int q = 0; q < NS; q++) {
            const int32_t i = q * (32 * nw) + lane * nw + gw;
            if (i < m) accn[i] = 0;
            choice[q] = -1;
            int2 sn = make_int2(0, 0);
            if (i < m) sn = c_sn[i];
            unsigned todo = __ballot_sync(FULL, free_end[q] && j0[q] < jend[q]);
            while (todo) {
                const int l = __ffs(todo) - 1;
                todo &= todo - 1;
                uint32_t p = 0;
                const int32_t x = warp_pick(__shfl_sync(FULL, i, l), __shfl_sync(FULL, j0[q], l),
                                            __shfl_sync(FULL, jend[q], l), C.window, __shfl_sync(FULL, sn.x, l),
                                            __shfl_sync(FULL, sn.y, l),
                                            [&](int32_t j) { return (s_taken[j >> 5] >> (j & 31)) & 1u; },
                                            [&](int32_t j) { return c_gain[j]; }, [&](int32_t j) { return c_sn[j]; }, p);
                if (lane == l) {
                    choice[q] = x;
                    pen[q] = p;
                }
            }
            if (choice[q] >= 0) {
                atomicMax(&accr[choice[q]], chain_key(pen[q], vi[q]));
                any = true;
            }
        }
        if (__any_sync(FULL, any) && lane == 0) C.linked[rr] = 1;
        cl.sync();
    }
    // the links of the last round run (rounds cut off by the limit)
    if (rr == rounds && rounds > 0) link(C.acc[(rounds - 1) % 3]);
    cl.sync();
}

__global__ void __cluster_dims__(SQ_CS, 1, 1) __launch_bounds__(SEQ_T) k_seq_cluster(ClusterSeqArgs A) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wc[32 * 256];
    __shared__ uint32_t s_tot[256];
    __shared__ uint32_t s_base[512];
    __shared__ int32_t s_tmp[40];
    __shared__ int32_t s_part;
    __shared__ long long s_ll[40];
    cg::cluster_group cl = cg::this_cluster();
    const int32_t m = A.cnt[C_MOVES];
    if (m == 0 || m > sq_max<uint64_t>()) return;   // uniform: no CTA of the cluster runs on
    const int64_t t0 = (int64_t)cl.block_rank() * blockDim.x + threadIdx.x, nt = (int64_t)SQ_CS * blockDim.x;
    const SqBuf<uint64_t> B(smem);
    // key widths from this repetition's moves
    long long gmx = 0, smx = 0, nmx = 0;
    STRIDE(i, m, t0, nt) {
        gmx = max(gmx, A.M.gain[i]);
        smx = max(smx, (long long)A.M.src[i]);
        nmx = max(nmx, (long long)A.M.node[i]);
    }
    cluster_max3_ll(cl, gmx, smx, nmx, s_ll);
    const int gb = dev_bits((unsigned long long)gmx), nb = dev_bits((unsigned long long)nmx),
              sb = dev_bits((unsigned long long)smx);
    // sort (p_s asc, gain desc, node asc)
    if (sb + gb + nb <= 64) {
        ph_move_keys(A.M, m, gmx, gb, nb, -1, A.keys, A.idx, 1, t0, nt);
        cl.sync();
        cluster_radix_sort<uint64_t>(cl, A.keys, A.idx, m, (sb + gb + nb + 7) / 8, B, s_wc, s_tot, s_base);
    } else {
        const int fb[3] = {A.nb, A.gb, A.sb};
        for (int f = 0; f < 3; f++) {
            ph_move_keys(A.M, m, A.gbound, A.gb, A.nb, f, A.keys, A.idx, f == 0, t0, nt);
            cl.sync();
            cluster_radix_sort<uint64_t>(cl, A.keys, A.idx, m, (fb[f] + 7) / 8, B, s_wc, s_tot, s_base);
        }
    }
    // the moves in sorted order, with the size and |in| of each moved node
    STRIDE(i, m, t0, nt) {
        const uint32_t k = A.idx[i];
        const int32_t v = A.M.node[k];
        A.S.node[i] = v;
        A.S.src[i] = A.M.src[k];
        A.S.dst[i] = A.M.dst[k];
        A.S.gain[i] = A.M.gain[k];
        const_cast<int32_t *>(A.C.msz)[i] = A.C.size[v];
        const_cast<int32_t *>(A.C.mni)[i] = A.C.nin[v];
    }
    cl.sync();
    ph_first_of(A.S.src, m, A.nparts, A.first, t0, nt);
    cl.sync();
    // chaining rounds (Sec. VI-C)
    const int gw = (int)(t0 >> 5), nwarps = (int)(nt >> 5);
    if (A.packed && m <= CHAIN_SMEM_M) {
        chain_rounds_smem(A.C, A.S, A.rounds, m, cl, smem, s_wc);
    } else if (A.packed) {
        for (int rr = 0; rr < A.rounds; rr++) {
            if (rr > 0 && !*(volatile int32_t *)&A.C.linked[rr - 1]) break;
            const unsigned long long *accp = A.C.acc[(rr + 2) % 3];
            ph_round(A.C, rr, m, gw, nwarps,
                     [&](int32_t j) { return A.C.pred[j] >= 0 || (rr > 0 && accp[j] != 0ull); },
                     [&](int32_t j) { return A.S.gain[j]; },
                     [&](int32_t j) { return make_int2(A.C.msz[j], A.C.mni[j]); });
            cl.sync();
        }
        if (A.rounds > 0 && *(volatile int32_t *)&A.C.linked[A.rounds - 1]) {
            ph_link_last(A.C, A.rounds - 1, m, t0, nt);
            cl.sync();
        }
    } else {
        for (int rr = 0; rr < A.rounds; rr++) {
            if (rr > 0 && !*(volatile int32_t *)&A.C.linked[rr - 1]) break;
            ph_choose(A.C, m, t0, nt);
            cl.sync();
            ph_accept_min(A.C, m, t0, nt);
            cl.sync();
            ph_accept_id(A.C, m, t0, nt);
            cl.sync();
            ph_link(A.C, rr, 0, m, t0, nt);
            cl.sync();
        }
    }
    // chains, ordered by (total gain desc, head node asc)
    ph_path_heads(A.Q, m, t0, nt);
    cl.sync();
    ph_cycle_heads(A.Q, m, t0, nt);
    cl.sync();
    ph_head_collect(A.Q, m, A.heads, &A.cnt[C_NH], t0, nt);
    cl.sync();
    const int32_t nh = *(volatile int32_t *)&A.cnt[C_NH];
    long long cmx = 0;
    STRIDE(k, nh, t0, nt) cmx = max(cmx, A.Q.cgain[A.heads[k]]);
    cmx = cluster_max_ll(cl, cmx, s_ll);
    const int cgb = dev_bits((unsigned long long)cmx);
    if (cgb + nb <= 64) {
        ph_head_keys(A.heads, nh, A.Q.cgain, A.S.node, cmx, nb, -1, A.hkeys, t0, nt);
        cl.sync();
        cluster_radix_sort<uint64_t>(cl, A.hkeys, A.heads, nh, (cgb + nb + 7) / 8, B, s_wc, s_tot, s_base);
    } else {
        for (int f = 0; f < 2; f++) {
            ph_head_keys(A.heads, nh, A.Q.cgain, A.S.node, A.cgbound, A.nb, f, A.hkeys, t0, nt);
            cl.sync();
            cluster_radix_sort<uint64_t>(cl, A.hkeys, A.heads, nh, ((f == 0 ? A.nb : A.cgb) + 7) / 8, B, s_wc,
                                         s_tot, s_base);
        }
    }
    ph_chain_lens(A.heads, nh, A.Q.clen, nh, A.lens, t0, nt);
    cl.sync();
    cluster_scan_excl<int32_t>(cl, A.lens, A.starts, nh, s_tmp, &s_part);
    ph_chain_start(A.heads, nh, A.starts, A.cstart, t0, nt);
    cl.sync();
    ph_seq_pos(A.Q.chain, A.Q.pos, A.cstart, m, A.S.node, A.seqmove, A.mvpos, t0, nt);
    cl.sync();   // no CTA leaves while another may still read its shared memory
}

// validity of every prefix, best prefix, apply
__global__ void __launch_bounds__(SEQ_T) k_val_small(ValCtx V, int32_t *cnt, int32_t nparts, int sb, long long *bgain,
                                                     int32_t *rho) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wc[32 * 256];
    __shared__ uint32_t s_hist[256 + 33];
    __shared__ int32_t s_tmp[40];
    __shared__ long long s_ll[40];
    const int32_t m = cnt[C_MOVES];
    if (m == 0 || m > SMALLM) return;
    const int64_t t0 = threadIdx.x, nt = blockDim.x;
    ph_val_entries(V, m, t0, nt);
    block_radix_sort<uint32_t>(V.vkey, V.vidx, 2 * m, (sb + 7) / 8, 2 * SMALLM, smem, s_wc, s_hist);
    __syncthreads();
    ph_val_gather(V, 2 * m, t0, nt);
    __syncthreads();
    block_scan_excl_ll(V.gsz, V.esz, 2 * m, s_ll);
    block_scan_excl_ll(V.gdd, V.edd, 2 * m, s_ll);
    ph_val_trans(V, 2 * m, t0, nt);
    int32_t bad = block_sum(ph_initial_bad(V.psize, V.D0, nparts, V.omega, V.delta, t0, nt), s_tmp);
    __syncthreads();
    best_prefix_block(V.gseq, V.viol, m, bad, &cnt[C_APPLIED], bgain);
    const int32_t L = *(volatile int32_t *)&cnt[C_APPLIED];
    ph_apply(V.seqmove, V.S.node, V.S.dst, L, rho, t0, nt);
}

// The same on one thread-block cluster, for up to sq_max<uint32_t>() / 2
// moves: events, cluster radix sort by part, the two prefix sums, the
// validity transitions, the count of invalid parts, the best prefix and the
// apply, separated by cluster barriers.
__global__ void __cluster_dims__(SQ_CS, 1, 1) __launch_bounds__(SQ_T)
    k_val_cluster(ValCtx V, int32_t *cnt, int32_t nparts, int sb, long long *bgain, int32_t *rho) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wc[32 * 256];
    __shared__ uint32_t s_tot[256];
    __shared__ uint32_t s_base[512];
    __shared__ long long s_ll[40];
    __shared__ int32_t s_tmp[40];
    __shared__ long long s_part;
    __shared__ int32_t s_ipart;
    __shared__ long long s_bg[32];
    __shared__ int32_t s_bk[32];
    cg::cluster_group cl = cg::this_cluster();
    const int32_t m = cnt[C_MOVES];
    if (m == 0 || 2 * (int64_t)m > sq_max<uint32_t>()) return;   // uniform over the cluster
    const int r = (int)cl.block_rank(), t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = blockDim.x >> 5;
    const int64_t t0 = (int64_t)r * blockDim.x + t, nt = (int64_t)SQ_CS * blockDim.x;
    const int32_t c = 2 * m;
    ph_val_entries(V, m, t0, nt);
    cl.sync();
    cluster_radix_sort<uint32_t>(cl, V.vkey, V.vidx, c, (sb + 7) / 8, SqBuf<uint32_t>(smem), s_wc, s_tot, s_base);
    ph_val_gather(V, c, t0, nt);
    cl.sync();
    cluster_scan_excl<long long>(cl, V.gsz, V.esz, c, s_ll, &s_part);
    cluster_scan_excl<long long>(cl, V.gdd, V.edd, c, s_ll, &s_part);
    ph_val_trans(V, c, t0, nt);
    const int32_t bad0 = cluster_sum_i32(cl, ph_initial_bad(V.psize, V.D0, nparts, V.omega, V.delta, t0, nt), s_tmp,
                                         &s_ipart);
    // best prefix (Sec. VI-D): the largest cumulative gain over prefixes with
    // no invalid part, the longest on ties; this CTA takes moves [lo, hi)
    const int32_t chunk = (m + SQ_CS - 1) / SQ_CS, lo = min(m, r * chunk), hi = min(m, lo + chunk);
    long long gl = 0;
    int32_t vl = 0;
    for (int32_t k = lo + t; k < hi; k += blockDim.x) {
        gl += (long long)V.gseq[k];
        vl += V.viol[k];
    }
    gl = block_sum_ll(gl, s_ll);
    vl = block_sum(vl, s_tmp);
    if (t == 0) {
        s_ll[36] = gl;
        s_ll[37] = vl;
    }
    cl.sync();
    long long gc = 0, vc = bad0;   // sums over the moves before lo
    for (int q = 0; q < r; q++) {
        const long long *o = cl.map_shared_rank(s_ll, q);
        gc += o[36];
        vc += o[37];
    }
    long long bestg = 0;
    int32_t bestk = 0;
    for (int32_t base = lo; base < hi; base += blockDim.x) {
        const int32_t k = base + t;
        const long long g = k < hi ? (long long)V.gseq[k] : 0;
        const long long dv = k < hi ? V.viol[k] : 0;
        long long gi = g, vi = dv;
        for (int o = 1; o < 32; o <<= 1) {
            const long long ug = __shfl_up_sync(0xffffffffu, gi, o), uv = __shfl_up_sync(0xffffffffu, vi, o);
            if (lane >= o) {
                gi += ug;
                vi += uv;
            }
        }
        if (lane == 31) {
            s_ll[wid] = gi;
            s_bg[wid] = vi;
        }
        __syncthreads();
        if (wid == 0) {
            const long long x = lane < nw ? s_ll[lane] : 0, y = lane < nw ? s_bg[lane] : 0;
            long long xi = x, yi = y;
            for (int o = 1; o < 32; o <<= 1) {
                const long long ux = __shfl_up_sync(0xffffffffu, xi, o), uy = __shfl_up_sync(0xffffffffu, yi, o);
                if (lane >= o) {
                    xi += ux;
                    yi += uy;
                }
            }
            if (lane < nw) {
                s_ll[lane] = xi - x;
                s_bg[lane] = yi - y;
            }
            if (lane == nw - 1) {
                s_ll[32] = xi;
                s_ll[33] = yi;
            }
        }
        __syncthreads();
        const long long cum = gc + s_ll[wid] + gi, vio = vc + s_bg[wid] + vi;
        if (k < hi && vio == 0 && cum >= bestg) {
            bestg = cum;
            bestk = k + 1;
        }
        gc += s_ll[32];
        vc += s_ll[33];
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) {
        const long long og = __shfl_down_sync(0xffffffffu, bestg, o);
        const int32_t ok = __shfl_down_sync(0xffffffffu, bestk, o);
        if (og > bestg || (og == bestg && ok > bestk)) {
            bestg = og;
            bestk = ok;
        }
    }
    if (lane == 0) {
        s_bg[wid] = bestg;
        s_bk[wid] = bestk;
    }
    __syncthreads();
    if (t == 0) {
        for (int k = 1; k < nw; k++)
            if (s_bg[k] > bestg || (s_bg[k] == bestg && s_bk[k] > bestk)) {
                bestg = s_bg[k];
                bestk = s_bk[k];
            }
        s_ll[38] = bestg;
        s_ll[39] = bestk;
    }
    cl.sync();
    if (r == 0 && t == 0) {
        for (int q = 1; q < SQ_CS; q++) {
            const long long *o = cl.map_shared_rank(s_ll, q);
            if (o[38] > bestg || (o[38] == bestg && o[39] > bestk)) {
                bestg = o[38];
                bestk = (int32_t)o[39];
            }
        }
        *bgain = bestg;
        cnt[C_APPLIED] = bestg > 0 ? bestk : 0;
    }
    cl.sync();
    const int32_t L = *(volatile int32_t *)&cnt[C_APPLIED];
    ph_apply(V.seqmove, V.S.node, V.S.dst, L, rho, t0, nt);
    cl.sync();   // no CTA leaves while another may still read its shared memory
}

// ---------------------------------------------------------------- in-sequence gains
// Per hyperedge e with moved pins: its moved pins in sequence order; the
// running pins(p,e) / pins_in(p,e) of the parts they touch start from the
// pins list.  A move that empties e in p_s spares w(e), one that enters an
// empty p_d costs w(e) (Eq. 14-15 read as the exact change of connectivity);
// an inbound count crossing 1 -> 0 at p_s or 0 -> 1 at p_d changes the
// distinct-inbound count of that part at that move (Sec. VI-D).
struct SeqSim {
    const int32_t *off, *pin, *nsrc, *w, *mvpos, *seqmove, *src, *dst;
    Plist PL;
    unsigned long long *gseq;
    int32_t *dDs, *dDd;
};

__device__ __forceinline__ int32_t plist_find(const Plist &PL, int32_t a, int32_t lam, int32_t p) {
    int32_t lo = 0, hi = lam;
    while (lo < hi) {
        int32_t mid = (lo + hi) >> 1;
        if (PL.p[a + mid] < p) lo = mid + 1;
        else hi = mid;
    }
    return (lo < lam && PL.p[a + lo] == p) ? a + lo : -1;
}

// group of G threads; buffers: bk/bd/ord >= |e|, tp/tc/tci >= 2|e|.
// The running counts are not simulated move by move: the move at sequence
// rank r sees pins(p,e) = the pins list's count + (moves of ranks < r into p)
// - (moves of ranks < r out of p), and pins_in(p,e) the same over the moves
// of destination pins, so every rank is evaluated at once (threads over
// ranks, each counting over the ranks before it in shared memory).
template <int G>
__device__ void inseq_edge(const SeqSim &Q, int32_t e, int gt, int32_t *bk, int32_t *bd, int32_t *ord, int32_t *tp,
                           int32_t *tc, int32_t *tci, int32_t *g_cnt) {
    const int32_t a = Q.off[e], b = Q.off[e + 1], dst0 = a + Q.nsrc[e];
    if (gt == 0) *g_cnt = 0;
    gsync<G>();
    for (int64_t j = (int64_t)a + gt; j < b; j += G) {
        int32_t k = Q.mvpos[Q.pin[j]];
        if (k >= 0) {
            int32_t s = atomicAdd(g_cnt, 1);
            bk[s] = k;
            bd[s] = j >= dst0;
        }
    }
    gsync<G>();
    const int32_t c = *(volatile int32_t *)g_cnt;
    if (c == 0) {
        gsync<G>();
        return;
    }
    for (int32_t i = gt; i < c; i += G) {
        int32_t k = bk[i], r = 0;
        for (int32_t t = 0; t < c; t++) r += bk[t] < k;
        ord[r] = i;
    }
    gsync<G>();
    // by rank: source part, destination part, destination-pin flag
    int32_t *rs = tp, *rd = tp + c, *rf = tc;
    for (int32_t r = gt; r < c; r += G) {
        const int32_t i = ord[r], mi = Q.seqmove[bk[i]];
        rs[r] = Q.src[mi];
        rd[r] = Q.dst[mi];
        rf[r] = bd[i];
    }
    gsync<G>();
    const long long we = Q.w[e];
    const int32_t lam = Q.PL.lam[e];
    for (int32_t r = gt; r < c; r += G) {
        const int32_t ps = rs[r], pd = rd[r];
        const int32_t fs = plist_find(Q.PL, a, lam, ps), fd = plist_find(Q.PL, a, lam, pd);
        int32_t cs = fs >= 0 ? Q.PL.cnt[fs] : 0, cd = fd >= 0 ? Q.PL.cnt[fd] : 0;
        int32_t is = fs >= 0 ? Q.PL.cin[fs] : 0, id = fd >= 0 ? Q.PL.cin[fd] : 0;
        for (int32_t t = 0; t < r; t++) {
            const int32_t xs = rs[t], xd = rd[t];
            const int32_t ds = (xd == ps) - (xs == ps), dd = (xd == pd) - (xs == pd);
            cs += ds;
            cd += dd;
            if (rf[t]) {
                is += ds;
                id += dd;
            }
        }
        const int32_t k = bk[ord[r]];
        long long g = 0;
        if (cs == 1) g += we;
        if (cd == 0) g -= we;
        if (g) atomicAdd(&Q.gseq[k], (unsigned long long)g);
        if (rf[r]) {
            if (is == 1) atomicAdd(&Q.dDs[k], -1);
            if (id == 0) atomicAdd(&Q.dDd[k], 1);
        }
    }
    gsync<G>();
}

// The hyperedges of `list` that hold a moved pin (lanes take one hyperedge
// each; those of more than 32 pins are scanned by the whole warp).
__global__ void k_touched(const int32_t *off, const int32_t *pin, const int32_t *mvpos, const int32_t *list,
                          int32_t count, int32_t *out, int32_t *out_n, const int32_t *mcount) {
    HP_KERNEL_ENTER();
    if (*mcount == 0) return;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < count; base += step) {
        const int64_t i = base + lane;
        int32_t e = -1, a = 0, b = 0;
        if (i < count) {
            e = list[i];
            a = off[e];
            b = off[e + 1];
        }
        bool hit = false;
        if (e >= 0 && b - a <= 32)
            for (int32_t j = a; j < b && !hit; j++) hit = mvpos[pin[j]] >= 0;
        unsigned big = __ballot_sync(FULL, e >= 0 && b - a > 32);
        while (big) {
            const int l = __ffs(big) - 1;
            big &= big - 1;
            const int32_t ea = __shfl_sync(FULL, a, l), eb = __shfl_sync(FULL, b, l);
            bool found = false;
            for (int64_t j0 = ea; j0 < eb; j0 += 32) {
                const bool h = j0 + lane < eb && mvpos[pin[j0 + lane]] >= 0;
                if (__any_sync(FULL, h)) {
                    found = true;
                    break;
                }
            }
            if (lane == l) hit = found;
        }
        if (hit) out[atomicAdd(out_n, 1)] = e;
    }
}

constexpr int IS_T = 128;
// hyperedges of lo < |e| <= emax pins from the list, a warp each
__global__ void __launch_bounds__(IS_T) k_inseq_small(SeqSim Q, const int32_t *list, const int32_t *count_p,
                                                      int32_t emax, const int32_t *mcount, int32_t lo) {
    HP_KERNEL_ENTER();
    if (*mcount == 0) return;
    const int32_t count = *count_p;
    extern __shared__ __align__(16) int32_t sm[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int32_t *base = sm + wid * (9 * emax + 1);
    int32_t *bk = base, *bd = bk + emax, *ord = bd + emax, *tp = ord + emax, *tc = tp + 2 * emax,
            *tci = tc + 2 * emax, *gc = tci + 2 * emax;
    int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = warp; i < count; i += nw) {
        const int32_t e = list[i], sz = Q.off[e + 1] - Q.off[e];
        if (sz > lo && sz <= emax) inseq_edge<32>(Q, e, lane, bk, bd, ord, tp, tc, tci, gc);
    }
}
// The same for up to PB_PARTS parts: the running counts of every part sit in
// a table indexed by part (pins in the low half word, inbound pins in the high
// one), loaded from the pins list.  The moves are taken 32 sequence ranks at a
// time, a lane each: a lane's counts are the table's plus what the chunk's
// earlier lanes change at its two parts (32 broadcasts); the table then takes
// the chunk's changes.  Against counting over all earlier ranks from the list:
// work c instead of c^2 / 2 a hyperedge with c moved pins, and no binary
// searches.  A warp per hyperedge of lo < |e| <= emax <= 512 pins.
__host__ __device__ inline size_t inseq_parts_smem(int32_t nparts, int32_t emax) {
    return 4 * (size_t)(IS_T / 32) * (nparts + 2 * (size_t)emax + 1);
}
__global__ void __launch_bounds__(IS_T) k_inseq_parts(SeqSim Q, const int32_t *list, const int32_t *count_p,
                                                      int32_t emax, int32_t nparts, const int32_t *mcount, int32_t lo) {
    HP_KERNEL_ENTER();
    if (*mcount == 0) return;
    const int32_t count = *count_p;
    extern __shared__ __align__(16) uint32_t smw[];
    const unsigned FULL = 0xffffffffu;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    // running counts; moved pins (sequence position << 1 | destination pin) as found, then by rank
    uint32_t *tab = smw + (size_t)wid * (nparts + 2 * emax + 1), *mv = tab + nparts, *srt = mv + emax;
    for (int32_t p = lane; p < nparts; p += 32) tab[p] = 0;
    __syncwarp();
    const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t x = w0; x < count; x += nw) {
        const int32_t e = list[x];
        const int32_t a = Q.off[e], sz = Q.off[e + 1] - a;
        if (sz <= lo || sz > emax) continue;
        const int32_t dst0 = Q.nsrc[e], lam = Q.PL.lam[e];
        const long long we = Q.w[e];
        int32_t c = 0;
        for (int32_t j0 = 0; j0 < sz; j0 += 32) {
            const int32_t j = j0 + lane;
            const int32_t k = j < sz ? Q.mvpos[Q.pin[a + j]] : -1;
            const unsigned m = __ballot_sync(FULL, k >= 0);
            if (k >= 0) mv[c + __popc(m & lt)] = ((uint32_t)k << 1) | (j >= dst0 ? 1u : 0u);
            c += __popc(m);
        }
        if (c == 0) continue;
        for (int32_t k = lane; k < lam; k += 32)
            tab[Q.PL.p[a + k]] = (uint32_t)Q.PL.cnt[a + k] | ((uint32_t)Q.PL.cin[a + k] << 16);
        __syncwarp();
        for (int32_t i = lane; i < c; i += 32) {   // positions are distinct
            const uint32_t k = mv[i];
            int32_t r = 0;
            for (int32_t t = 0; t < c; t++) r += mv[t] < k;
            srt[r] = k;
        }
        __syncwarp();
        for (int32_t r0 = 0; r0 < c; r0 += 32) {
            const bool on = r0 + lane < c;
            const int n = min(32, c - r0);
            int32_t k = 0, ps = -1, pd = -1;
            uint32_t dv = 0, cs = 0, cd = 0;
            if (on) {
                const uint32_t y = srt[r0 + lane];
                k = (int32_t)(y >> 1);
                dv = (y & 1u) ? 0x10001u : 1u;
                const int32_t mi = Q.seqmove[k];
                ps = Q.src[mi];
                pd = Q.dst[mi];
                cs = tab[ps];
                cd = tab[pd];
            }
            __syncwarp();
            for (int t = 0; t + 1 < n; t++) {
                const int32_t xs = __shfl_sync(FULL, ps, t), xd = __shfl_sync(FULL, pd, t);
                const uint32_t xv = __shfl_sync(FULL, dv, t);
                if (lane > t) {
                    if (xd == ps) cs += xv;
                    if (xs == ps) cs -= xv;
                    if (xd == pd) cd += xv;
                    if (xs == pd) cd -= xv;
                }
            }
            if (on) {
                long long g = 0;
                if ((cs & 0xffffu) == 1u) g += we;
                if ((cd & 0xffffu) == 0u) g -= we;
                if (g) atomicAdd(&Q.gseq[k], (unsigned long long)g);
                if (dv >> 16) {
                    if ((cs >> 16) == 1u) atomicAdd(&Q.dDs[k], -1);
                    if ((cd >> 16) == 0u) atomicAdd(&Q.dDd[k], 1);
                }
                atomicAdd(&tab[ps], 0u - dv);
                atomicAdd(&tab[pd], dv);
            }
            __syncwarp();
        }
        // clean the table: the list's parts and the parts moved to
        for (int32_t k = lane; k < lam; k += 32) tab[Q.PL.p[a + k]] = 0;
        for (int32_t i = lane; i < c; i += 32) tab[Q.dst[Q.seqmove[srt[i] >> 1]]] = 0;
        __syncwarp();
    }
}
__global__ void __launch_bounds__(256) k_inseq_big(SeqSim Q, const int32_t *list, int32_t count, int32_t emax,
                                                   int32_t *gbuf, const int32_t *mcount) {
    HP_KERNEL_ENTER();
    if (*mcount == 0) return;
    __shared__ int32_t gc;
    int32_t *base = gbuf + (int64_t)blockIdx.x * 9 * (int64_t)emax;
    int32_t *bk = base, *bd = bk + emax, *ord = bd + emax, *tp = ord + emax, *tc = tp + 2 * emax,
            *tci = tc + 2 * emax;
    for (int32_t k = blockIdx.x; k < count; k += gridDim.x)
        inseq_edge<256>(Q, list[k], threadIdx.x, bk, bd, ord, tp, tc, tci, &gc);
}


// In-sequence gains of hyperedges of at most TINY_E pins (all of the level's:
// listing the ones with a moved pin first reads what this reads), one thread each:
// the moved pins are taken in sequence order (ranks among at most TINY_E
// distinct positions) and the parts they leave or enter are tracked in a
// per-thread table of 2 TINY_E entries in shared memory.  The r-th moves of
// a warp's hyperedges are combined by sequence position (match_any) before
// their atomics: a moved node with many hyperedges is one position.
constexpr int IST_T = 128;
__global__ void __launch_bounds__(IST_T) k_inseq_tiny(SeqSim Q, const int32_t *list, int32_t count,
                                                       const int32_t *mcount) {
    HP_KERNEL_ENTER();
    __shared__ int32_t s_tab[IST_T * 6 * TINY_E];
    if (*mcount == 0) return;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t lt = (1u << lane) - 1u;
    int32_t *tp = s_tab + threadIdx.x * 6 * TINY_E, *tc = tp + 2 * TINY_E, *tci = tc + 2 * TINY_E;
    const int64_t step = (int64_t)gridDim.x * IST_T;
    for (int64_t base = blockIdx.x * (int64_t)IST_T + (threadIdx.x & ~31u); base < count; base += step) {
        const int64_t i = base + lane;
        int32_t e = 0, a = 0, sz = 0, d0 = 0, lam = 0;
        long long we = 0;
        if (i < count) {
            e = list[i];
            a = Q.off[e];
            sz = Q.off[e + 1] - a;
        }
        int32_t kk[TINY_E];
        int nm = 0;
#pragma unroll
        for (int j = 0; j < TINY_E; j++) {
            kk[j] = 0x7fffffff;
            if (j < sz) {
                const int32_t k = Q.mvpos[Q.pin[a + j]];
                if (k >= 0) {
                    kk[j] = k;
                    nm++;
                }
            }
        }
        const int rmax = (int)__reduce_max_sync(FULL, (unsigned)nm);
        if (nm > 0) {
            d0 = Q.nsrc[e];
            we = Q.w[e];
            lam = Q.PL.lam[e];
        }
        int nt = 0;
        for (int r = 0; r < rmax; r++) {
            int32_t k = -1;
            int g = 0, ds = 0, dd = 0;
            if (r < nm) {
                // the moved pin of rank r (positions are distinct)
                bool isdst = false;
#pragma unroll
                for (int j = 0; j < TINY_E; j++) {
                    int32_t rk = 0;
#pragma unroll
                    for (int x = 0; x < TINY_E; x++) rk += kk[x] < kk[j];
                    if (kk[j] != 0x7fffffff && rk == r) {
                        k = kk[j];
                        isdst = j >= d0;
                    }
                }
                const int32_t mi = Q.seqmove[k];
                const int32_t ps[2] = {Q.src[mi], Q.dst[mi]};
                int32_t sl[2];
                for (int h = 0; h < 2; h++) {
                    int32_t x = 0;
                    while (x < nt && tp[x] != ps[h]) x++;
                    if (x == nt) {
                        const int32_t f = plist_find(Q.PL, a, lam, ps[h]);
                        tp[x] = ps[h];
                        tc[x] = f >= 0 ? Q.PL.cnt[f] : 0;
                        tci[x] = f >= 0 ? Q.PL.cin[f] : 0;
                        nt++;
                    }
                    sl[h] = x;
                }
                if (tc[sl[0]] == 1) g += (int)we;
                if (tc[sl[1]] == 0) g -= (int)we;
                tc[sl[0]]--;
                tc[sl[1]]++;
                if (isdst) {
                    if (--tci[sl[0]] == 0) ds = -1;
                    if (++tci[sl[1]] == 1) dd = 1;
                }
            }
            // |g| <= 65536 per lane, so the warp sums fit 32 bits
            const unsigned grp = __match_any_sync(FULL, k);
            uint32_t sum[3] = {(uint32_t)g, (uint32_t)ds, (uint32_t)dd};
            group_sum(grp, k >= 0, sum);
            const int gs = (int)sum[0], dss = (int)sum[1], dds = (int)sum[2];
            if (k >= 0 && (grp & lt) == 0u) {
                if (gs) atomicAdd(&Q.gseq[k], (unsigned long long)(long long)gs);
                if (dss) atomicAdd(&Q.dDs[k], dss);
                if (dds) atomicAdd(&Q.dDd[k], dds);
            }
        }
    }
}

// ---------------------------------------------------------------- workspace
// Allocated once per call for the largest level and reused by every level
// and repetition.
struct LevelWs {
    // capacities
    int32_t cn, ce, nparts, cmax_e;
    int64_t cnp;
    // per level
    int32_t n, max_e, small_max, n_big;
    uint32_t pcap;
    int32_t *big;
    long long *wns;
    int32_t *singin;
    Plist PL;
    RepArrays R;
    int32_t *cl, *hubs, *cw;
    uint32_t *cutbits;                       // a bit per cut hyperedge
    int32_t *cut;                            // cut hyperedges of the candidates (k_cut_lists)
    int32_t *tiny, n_tiny;                   // hyperedges of 2..8 pins
    int32_t *mid, n_mid;                     // hyperedges of 9..small_max pins
    int32_t parts_used;                      // parts holding a node at the level's start
    cudaStream_t side = nullptr, side2 = nullptr;   // side streams of the gain kernels
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    // algorithmic bytes of the repetitions (host): running total, and the cut
    // entries and their list entries of the last rebuilt repetition
    int64_t alg_bytes = 0, cuts = 0, cut_lam = 0;
    bool bits_valid = false;
    uint4 *bits = nullptr;   // [ce][wq] parts of every cut hyperedge (k_part_bits), or none
    int wq = 0;
    int32_t *touched, *ttouched;             // hyperedges of mid (of tiny) with a moved pin
    int32_t *emark, *upd;                    // [ce] last update that listed a hyperedge; its counts (U_N words)
    int32_t epoch = 0;
    Moves M, S;
    uint64_t *keys;
    uint32_t *idx;
    int32_t *msz, *mni;
    int32_t *first, *choice, *accnode, *pos, *clen, *lens, *starts, *cstart, *seqmove;
    unsigned long long *pen, *minpen, *acc1, *acc2;
    uint32_t *heads;
    uint64_t *hkeys;
    uint32_t *vkey, *vidx;
    long long *vsz;
    int32_t *vdd;
    long long *gsz, *gdd, *esz, *edd;
    int32_t *vhead;
    int32_t *ovf, *gk;
    long long *gc;
    uint32_t gcap;
    int gnb;
    int32_t *ptab, *ibuf;
    uint32_t bcap;
    int pnb;
    long long *bgain;
    int32_t *lvl;   // per-level counters
    int32_t *pmark; // [nparts] parts in use
    int32_t *pnew;  // [nparts] their ranks
};

// rows of part bits (16 * wq bytes per hyperedge) for the current number of
// parts, where every sum of weights fits their 32-bit counters and they take
// at most PB_BYTES, and no more than 8 bytes a pin (beyond a megabyte): rows
// longer than their hyperedges' lists do not pay
static void part_bits_rows(LevelWs &W, const Params &P, Arena &A) {
    if (W.nparts > PB_PARTS || P.wsum >= (1ll << 32) || P.o.debug_table_cap != 0) return;
    W.wq = (int)pow2_at_least(std::max<int64_t>(cdiv(W.nparts, 128), 1));
    if (!W.bits && (int64_t)W.ce * W.wq * 16 <= std::min(PB_BYTES, 8 * W.cnp + (int64_t(1) << 20))) W.bits = A.get<uint4>((int64_t)W.ce * W.wq);
}

static LevelWs *refine_workspace_body(LevelWs *W, int32_t n, int64_t np, int32_t e, int32_t nparts, int32_t max_e,
                                      const Params &P, Arena &A);

// on a failure half-way, the stream and events made so far are destroyed
// (the arena frees the device memory taken so far)
LevelWs *refine_workspace(int32_t n, int64_t np, int32_t e, int32_t nparts, int32_t max_e, const Params &P,
                          Arena &A) {
    LevelWs *W = new LevelWs();
    try {
        return refine_workspace_body(W, n, np, e, nparts, max_e, P, A);
    } catch (...) {
        for (cudaStream_t x : {W->side, W->side2})
            if (x) cudaStreamDestroy(x);
        for (cudaEvent_t x : W->ev)
            if (x) cudaEventDestroy(x);
        delete W;
        throw;
    }
}

static LevelWs *refine_workspace_body(LevelWs *W, int32_t n, int64_t np, int32_t e, int32_t nparts, int32_t max_e,
                                      const Params &P, Arena &A) {
    cudaStream_t s = A.stream();
    if (!t_one_stream) {
        for (cudaStream_t *x : {&W->side, &W->side2}) HPC(cudaStreamCreateWithFlags(x, cudaStreamNonBlocking));
        for (cudaEvent_t &x : W->ev) HPC(cudaEventCreateWithFlags(&x, cudaEventDisableTiming));
    }
    W->cn = n;
    W->cnp = np;
    W->ce = e;
    W->nparts = nparts;
    W->cmax_e = max_e;
    W->big = A.get<int32_t>(e);
    W->wns = A.get<long long>(n);
    W->singin = A.get<int32_t>(n);
    W->PL.p = A.get<int32_t>(np);
    W->PL.cnt = A.get<int32_t>(np);
    W->PL.cin = A.get<int32_t>(np);
    W->PL.lam = A.get<int32_t>(e);
    RepArrays &R = W->R;
    R.nparts = nparts;
    R.rounds = P.o.chain_rounds;
    R.cnt = A.get<int32_t>(C_N);
    R.linked = A.get<int32_t>(P.o.chain_rounds + 1);
    R.D0 = A.get<int32_t>(nparts);
    R.psize = A.get<long long>(nparts);
    R.saving = A.get<long long>(n);
    R.pc = A.get<int32_t>(nparts + 1);
    R.pred = A.get<int32_t>(n);
    R.succ = A.get<int32_t>(n);
    R.chain = A.get<int32_t>(n);
    R.mvpos = A.get<int32_t>(n);
    R.cgain = A.get<long long>(n);
    R.gseq = A.get<unsigned long long>(n);
    R.acc0 = A.get<unsigned long long>(n);
    R.dDs = A.get<int32_t>(n);
    R.dDd = A.get<int32_t>(n);
    R.viol = A.get<int32_t>(n);
    W->cl = A.get<int32_t>(n);
    W->hubs = A.get<int32_t>(n);
    W->cw = A.get<int32_t>(n);
    W->cutbits = A.get<uint32_t>(e / 32 + 1);
    W->cut = A.get<int32_t>(np);
    R.cutn = A.get<int32_t>(n);
    W->tiny = A.get<int32_t>(e);
    W->mid = A.get<int32_t>(e);
    W->touched = A.get<int32_t>(e);
    W->ttouched = A.get<int32_t>(e);
    W->emark = A.get<int32_t>(std::max(e, 1));
    W->upd = A.get<int32_t>(U_N);
    HPC(cudaMemsetAsync(W->emark, 0, sizeof(int32_t) * std::max(e, 1), s));
    for (Moves *m : {&W->M, &W->S}) {
        m->node = A.get<int32_t>(n);
        m->src = A.get<int32_t>(n);
        m->dst = A.get<int32_t>(n);
        m->gain = A.get<long long>(n);
        m->count = R.cnt + C_MOVES;
    }
    W->keys = A.get<uint64_t>(n);
    W->idx = A.get<uint32_t>(n);
    W->msz = A.get<int32_t>(n);
    W->mni = A.get<int32_t>(n);
    W->first = A.get<int32_t>(nparts + 1);
    W->choice = A.get<int32_t>(n);
    W->accnode = A.get<int32_t>(n);
    W->pen = A.get<unsigned long long>(n);
    W->minpen = A.get<unsigned long long>(n);
    W->acc1 = A.get<unsigned long long>(n);
    W->acc2 = A.get<unsigned long long>(n);
    W->pos = A.get<int32_t>(n);
    W->clen = A.get<int32_t>(n);
    W->lens = A.get<int32_t>(n);
    W->starts = A.get<int32_t>(n);
    W->cstart = A.get<int32_t>(n);
    W->seqmove = A.get<int32_t>(n);
    W->heads = A.get<uint32_t>(n);
    W->hkeys = A.get<uint64_t>(n);
    W->vkey = A.get<uint32_t>(2 * (int64_t)n);
    W->vidx = A.get<uint32_t>(2 * (int64_t)n);
    W->vsz = A.get<long long>(2 * (int64_t)n);
    W->vdd = A.get<int32_t>(2 * (int64_t)n);
    W->gsz = A.get<long long>(2 * (int64_t)n);
    W->gdd = A.get<long long>(2 * (int64_t)n);
    W->esz = A.get<long long>(2 * (int64_t)n);
    W->edd = A.get<long long>(2 * (int64_t)n);
    W->vhead = A.get<int32_t>(std::max<int64_t>(nparts, 1));
    W->bgain = A.get<long long>(1);
    W->lvl = A.get<int32_t>(V_N);
    W->pmark = A.get<int32_t>(std::max(nparts, 1));
    W->pnew = A.get<int32_t>(std::max(nparts, 1));
    // overflow tables of the gain kernel, one per CTA of its fallback grid
    W->gcap = pow2_at_least(2 * (int64_t)nparts + 2);
    W->gnb = (int)std::min<int64_t>(num_sms(), std::max<int64_t>(1, ((int64_t)1 << 27) / ((int64_t)W->gcap * 12)));
    W->ovf = A.get<int32_t>(n);
    W->gk = A.get<int32_t>((int64_t)W->gnb * 2 * W->gcap);
    W->gc = A.get<long long>((int64_t)W->gnb * W->gcap);
    fill_i32(W->gk, (int64_t)W->gnb * 2 * W->gcap, -1, s);
    HPC(cudaMemsetAsync(W->gc, 0, sizeof(long long) * W->gnb * W->gcap, s));
    part_bits_rows(*W, P, A);
    // hyperedges above 512 pins: tables and buffers in global memory
    W->ptab = W->ibuf = nullptr;
    W->pnb = 0;
    if (max_e > SMALL_EDGE) {
        W->bcap = pow2_at_least(2 * (int64_t)max_e);
        W->pnb = num_sms() * 2;
        W->ptab = A.get<int32_t>((int64_t)W->pnb * (3 * (int64_t)W->bcap + 4 * (int64_t)max_e));
        W->ibuf = A.get<int32_t>((int64_t)W->pnb * 9 * (int64_t)max_e);
    }
    return W;
}

void refine_workspace_free(LevelWs *W, Arena &A) {
    if (!W) return;
    // side-stream work must be done before the arena hands its memory back
    // (it is, unless the call is ending early on an error)
    for (cudaStream_t x : {W->side, W->side2})
        if (x) {
            (void)cudaStreamSynchronize(x);
            cudaStreamDestroy(x);
        }
    for (cudaEvent_t x : W->ev)
        if (x) cudaEventDestroy(x);
    for (void *p : std::initializer_list<void *>{
             W->big, W->wns, W->singin, W->PL.p, W->PL.cnt, W->PL.cin, W->PL.lam, W->R.cnt, W->R.linked,
             W->R.D0, W->R.psize, W->R.saving, W->R.pc, W->R.pred, W->R.succ, W->R.chain, W->R.mvpos, W->R.cgain,
             W->R.gseq, W->R.acc0, W->R.dDs, W->R.dDd, W->R.viol, W->cl, W->hubs, W->cw, W->cutbits, W->cut, W->R.cutn, W->tiny, W->mid, W->touched, W->ttouched, W->emark, W->upd, W->M.node, W->M.src, W->M.dst, W->M.gain,
             W->S.node, W->S.src, W->S.dst, W->S.gain, W->keys, W->idx, W->msz, W->mni, W->first, W->choice, W->accnode, W->pen,
             W->minpen, W->acc1, W->acc2, W->pos, W->clen, W->lens, W->starts, W->cstart, W->seqmove, W->heads, W->hkeys,
             W->vkey, W->vidx, W->vsz, W->vdd, W->gsz, W->gdd, W->esz, W->edd, W->vhead, W->bgain, W->lvl, W->pmark, W->pnew, W->ovf, W->gk, W->gc, W->ptab, W->ibuf, W->bits})
        A.release(p);
    delete W;
}

// the level's counters and per-part / per-node sums start at zero (one
// launch instead of four memsets, which would each end the overlap of a
// launch with its predecessor)
__global__ void k_prep_zero(int32_t *lvl, int32_t *pmark, int32_t nparts, long long *wns, int32_t *singin, int32_t n) {
    HP_KERNEL_ENTER();
    GRID_STRIDE(i, (int64_t)max(max(n, nparts), (int32_t)V_N)) {
        if (i < V_N) lvl[i] = 0;
        if (i < nparts) pmark[i] = 0;
        if (i < n) {
            wns[i] = 0;
            singin[i] = 0;
        }
    }
}

static void level_prepare(const Level &L, const int32_t *w, const int32_t *rho, LevelWs &W, Arena &A) {
    cudaStream_t s = A.stream();
    const int32_t n = L.n, e = L.e;
    W.n = n;
    W.R.n = n;
    W.R.e = e;
    launch_k(k_prep_zero, grid_of(std::max(std::max(n, W.nparts), (int32_t)V_N), 256), 256, 0, s, W.lvl, W.pmark, W.nparts,
             W.wns, W.singin, n);
    HP_LAUNCH_CHECK();
    launch_k(k_level_prep, grid_of(std::max<int64_t>(std::max(n, e), L.np), LP_T), LP_T, 0, s, L, w, rho, W.pmark, W.big,
             W.tiny, W.mid, W.lvl, W.wns, W.singin);
    HP_LAUNCH_CHECK();
    int32_t hc[V_N];
    fetch_bytes(hc, W.lvl, sizeof hc, s);
    W.max_e = hc[V_MAX];
    W.small_max = level_small_max(W.max_e);
    W.n_big = hc[V_BIG];
    W.n_tiny = hc[V_TINY];
    W.n_mid = hc[V_MID];
    W.parts_used = hc[V_PARTS];
    // pins lists of the level hold at most min(small_max, parts in use) entries
    W.pcap = pow2_at_least(2 * (int64_t)std::max<int32_t>(2, std::min<int32_t>(W.small_max, W.parts_used)));
    if (W.n_big > 0 && !W.ptab) throw Error(HP_ERR_INTERNAL, "large hyperedge buffers missing");
}

// Whether the gains of the next repetition are computed from part bits: the
// average number of list entries behind a cut incidence entry, as counted by
// the last repetition that rebuilt the lists (of this level, or of the coarser
// one, whose lambda(e) the projection keeps), against the row's words.  At
// one entry per word the bits win (262k-node Gaussian net with the learned
// first level, lambda about 3 and 8 to 16 words: 462.8 ms by this rule, 483.1
// with bits from a quarter of an entry per word on; 4,096-node random net,
// 25 entries to 4 words: 27.0 ms against 46.1 without bits).
static bool bits_pay(const Level &L, const LevelWs &W) {
    if (!W.bits) return false;
    if (W.cuts == 0) return L.np >= 16 * (int64_t)L.e;
    return W.cut_lam >= W.cuts * 4 * W.wq;
}

// Side streams of the gain kernels: fork_side lets one start after the work
// queued on s, end_side marks the end of its work, join_side lets s wait for
// that (all on s itself where the thread keeps to one stream).
static cudaStream_t fork_side(const LevelWs &W, cudaStream_t s, cudaStream_t side) {
    if (t_one_stream) return s;
    HPC(cudaEventRecord(W.ev[0], s));
    HPC(cudaStreamWaitEvent(side, W.ev[0], 0));
    return side;
}
static void end_side(const LevelWs &W, cudaStream_t side, int k) {
    if (!t_one_stream) HPC(cudaEventRecord(W.ev[k], side));
}
static void join_side(const LevelWs &W, cudaStream_t s, int k) {
    if (!t_one_stream) HPC(cudaStreamWaitEvent(s, W.ev[k], 0));
}

// ---------------------------------------------------------------- gains by part
// The list form for up to PB_PARTS parts and weight sums below 2^32: the
// node's conn(v, p) in 32-bit counters indexed by part, so no table can
// overflow and the node classes need not wait for one another.  NW warps per
// node (one: several nodes a CTA); the k-th list entries of a warp's 32
// hyperedges are combined by part before one update per distinct part, the
// next entries and the next hyperedges loaded ahead.  Bound by the latency of
// those loads.  Hashed tables with a spill from class to class took 100, 83
// and 53 ms of kernel time (the last two one after the other) in the 466
// repetitions of the 1M Gaussian net; these 48, 38 and 54, side by side.
template <int NW>
__global__ void __launch_bounds__(NW == 1 ? 256 : NW * 32)
    k_gains_parts(GainArgs G, int32_t nparts, const int32_t *list, const int32_t *count_p) {
    HP_KERNEL_ENTER();
    extern __shared__ __align__(16) uint32_t smw[];
    __shared__ long long s_rg[32];
    __shared__ int32_t s_rp[32];
    constexpr int GROUPS = NW == 1 ? 8 : 1;   // nodes a CTA has in hand
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int grp = NW == 1 ? wid : 0, gt = NW == 1 ? lane : (int)threadIdx.x;
    const int words = (nparts + 31) / 32;
    uint32_t *conn = smw + (size_t)grp * (words * 32 + 32), *used = conn + words * 32;
    const int32_t count = *count_p;
    if ((int64_t)blockIdx.x * GROUPS >= count) return;
    for (int i = gt; i < words * 32 + 32; i += NW * 32) conn[i] = 0;
    gsync<NW * 32>();
    for (int64_t x = (int64_t)blockIdx.x * GROUPS + grp; x < count; x += (int64_t)gridDim.x * GROUPS) {
        const int32_t v = list[x], s = G.rho[v];
        const uint32_t c0 = G.ioff[v], c1 = c0 + G.cutn[v];
        auto hedge = [&](uint32_t t, int32_t &a, int32_t &lam, uint32_t &we) {
            a = lam = 0;
            we = 0;
            if (t < c1) {
                const int32_t e = G.inc[t];
                lam = G.PL.lam[e];
                a = G.off[e];
                we = (uint32_t)G.w[e];
            }
        };
        int32_t na, nlam;
        uint32_t nwe;
        hedge(c0 + gt, na, nlam, nwe);
        const int w32 = NW == 1 ? 0 : wid * 32;
        for (uint32_t base = c0 + w32; base < c1; base += NW * 32) {
            const int32_t a = na, lam = nlam;
            const uint32_t we = nwe;
            if (base + NW * 32 < c1) hedge(base + NW * 32 + lane, na, nlam, nwe);
            const int kmax = (int)__reduce_max_sync(FULL, (unsigned)lam);
            int32_t pn = lam > 0 ? G.PL.p[a] : -1;
            for (int k = 0; k < kmax; k++) {
                int32_t p = pn;
                pn = k + 1 < lam ? G.PL.p[a + k + 1] : -1;
                if (p == s) p = -1;
                const unsigned m = __match_any_sync(FULL, p);
                uint32_t sw[1] = {we};
                group_sum(m, p >= 0, sw);
                if (p >= 0 && lane == __ffs(m) - 1) {
                    atomicAdd(&conn[p], sw[0]);
                    atomicOr(&used[p >> 5], 1u << (p & 31));
                }
            }
        }
        gsync<NW * 32>();
        // the best part: the largest gain, the larger id on ties
        long long bg = 0;
        int32_t bp = -1;
        const long long basev = G.saving[v] - G.wns[v];
        const long long room = (long long)G.omega - G.size[v];
        auto look = [&](int32_t p) {
            const uint32_t c = conn[p];
            conn[p] = 0;
            if (G.second_half && G.psize[p] > room) return;
            const long long g = basev + (long long)c;
            if (bp < 0 || g > bg || (g == bg && p > bp)) {
                bg = g;
                bp = p;
            }
        };
        if (NW == 1) {
            for (uint32_t b = used[lane]; b; b &= b - 1) look(32 * lane + __ffs(b) - 1);
            used[lane] = 0;
        } else {
            for (int32_t p = threadIdx.x; p < nparts; p += NW * 32)
                if ((used[p >> 5] >> (p & 31)) & 1u) look(p);
        }
        for (int o = 16; o > 0; o >>= 1) {
            const long long og = __shfl_down_sync(FULL, bg, o);
            const int32_t op = __shfl_down_sync(FULL, bp, o);
            if (op >= 0 && (bp < 0 || og > bg || (og == bg && op > bp))) {
                bg = og;
                bp = op;
            }
        }
        if (NW > 1) {
            if (lane == 0) {
                s_rg[wid] = bg;
                s_rp[wid] = bp;
            }
            __syncthreads();
            if (threadIdx.x < 32) used[threadIdx.x] = 0;
            if (threadIdx.x == 0)
                for (int q = 1; q < NW; q++)
                    if (s_rp[q] >= 0 && (bp < 0 || s_rg[q] > bg || (s_rg[q] == bg && s_rp[q] > bp))) {
                        bg = s_rg[q];
                        bp = s_rp[q];
                    }
        }
        if (gt == 0 && bp >= 0 && bg > 0) {
            const int32_t i = atomicAdd(G.M.count, 1);
            G.M.node[i] = v;
            G.M.src[i] = s;
            G.M.dst[i] = bp;
            G.M.gain[i] = bg;
        }
        gsync<NW * 32>();
    }
}
// the three node classes side by side
static void gains_parts(const GainArgs &G, const LevelWs &W, const int32_t *cnt, int32_t n, cudaStream_t s) {
    const size_t sm = 4 * (size_t)(cdiv(W.nparts, 32) * 32 + 32);
    const cudaStream_t sh = fork_side(W, s, W.side), sm2 = fork_side(W, s, W.side2);
    const int occ_h = prepare_kernel((const void *)k_gains_parts<32>, 1024, sm);
    launch_k(k_gains_parts<32>, std::max(1, std::min<int>(n, num_sms() * occ_h)), 1024, sm, sh, G, W.nparts, W.hubs,
             cnt + C_HUB);
    HP_LAUNCH_CHECK();
    end_side(W, sh, 1);
    const int occ_m = prepare_kernel((const void *)k_gains_parts<8>, 256, sm);
    launch_k(k_gains_parts<8>, std::max(1, std::min<int>(n, num_sms() * occ_m)), 256, sm, sm2, G, W.nparts, W.cl,
             cnt + C_CAND);
    HP_LAUNCH_CHECK();
    end_side(W, sm2, 2);
    const int occ = prepare_kernel((const void *)k_gains_parts<1>, 256, 8 * sm);
    launch_k(k_gains_parts<1>, std::max(1, std::min<int>((int)cdiv(n, 8), num_sms() * occ)), 256, 8 * sm, s, G, W.nparts,
             W.cw, cnt + C_CW);
    HP_LAUNCH_CHECK();
    join_side(W, s, 1);
    join_side(W, s, 2);
}

template <int WQ>
static void gains_bits(const GainArgs &G, const LevelWs &W, const int32_t *cnt, int32_t n, cudaStream_t s) {
    // hub nodes on the side stream, beside the two lists of smaller ones
    const cudaStream_t sh = fork_side(W, s, W.side);
    // (16 warps a hub while the registers let two CTAs of them on an SM: wider
    // rows hold 74 a thread, and one such CTA an SM took 130.7 instead of 126.4
    // ms on the 16,384-node random net)
    constexpr int HW = WQ <= 2 ? 16 : 8;
    const int occ_h = prepare_kernel((const void *)k_gains_bits<WQ, HW>, HW * 32, 0);
    launch_k(k_gains_bits<WQ, HW>, std::max(1, std::min<int>(n, num_sms() * occ_h)), HW * 32, 0, sh, G, W.bits, W.nparts,
             W.hubs, cnt + C_HUB, nullptr, nullptr);
    HP_LAUNCH_CHECK();
    end_side(W, sh, 1);
    const int occ = prepare_kernel((const void *)k_gains_bits<WQ, 4>, 128, 0);
    const int grid = std::max(1, std::min<int>(n, num_sms() * occ));
    launch_k(k_gains_bits<WQ, 4>, grid, 128, 0, s, G, W.bits, W.nparts, W.cl, cnt + C_CAND, W.cw, cnt + C_CW);
    HP_LAUNCH_CHECK();
    join_side(W, s, 1);
}

// One repetition; returns the number of moves applied.
// reuse: rho is unchanged since the previous repetition of this level (which
// applied nothing), so its pins lists, D(p), |p|, saving(v) and cut lists,
// all functions of rho, are reused instead of rebuilt
// update: the previous repetition of this level applied that many moves, and
// the first four of these are updated for them instead of rebuilt
static int32_t rep_run(const Level &L, const int32_t *w, const Params &P, int32_t *rho, int second_half, LevelWs &W,
                       Arena &A, uint32_t *err_dev, const RepDebug *dbg, bool reuse = false, int32_t update = 0) {
    cudaStream_t s = A.stream();
    const int32_t n = L.n, nparts = W.nparts;
    RepArrays &R = W.R;
    int32_t *cnt = R.cnt;
    const int64_t zspan = std::max<int64_t>(std::max<int64_t>(n, (int64_t)nparts + 1),
                                            std::max<int64_t>((int64_t)C_N, (int64_t)P.o.chain_rounds + 1));
    const Applied moved{R.mvpos, W.seqmove, W.S.src, cnt + C_APPLIED};
    unsigned long long *uacc = reinterpret_cast<unsigned long long *>(W.upd + U_ACC);
    if (update > 0) {
        // the previous repetition applied `update` moves
        launch_k(k_move_nodes, grid_of(update, 256), 256, 0, s, moved, W.S.node, W.S.dst, L.size, W.singin, R.psize, R.D0,
                 W.upd);
        HP_LAUNCH_CHECK();
        launch_k(k_moved_edges, std::min(update, 16 * num_sms()), 256, 0, s, moved, W.S.node, L.off, L.ioff, L.inc,
                 ++W.epoch, W.emark, W.ttouched, W.touched, W.upd);
        HP_LAUNCH_CHECK();
        if (W.n_mid > 0) {
            const size_t sm = plist_parts_smem(nparts);
            const int occ = prepare_kernel((const void *)k_plist_parts<true>, PP_T, sm);
            const int grid = (int)std::min<int64_t>(cdiv(W.n_mid, PP_T / 32), (int64_t)num_sms() * occ);
            launch_k(k_plist_parts<true>, grid, PP_T, sm, s, L.off, L.pin, L.nsrc, w, rho, W.touched, 0, W.upd + U_MID, moved,
                     nparts, W.PL, R.D0, R.saving, uacc);
            HP_LAUNCH_CHECK();
        }
        if (W.n_tiny > 0) {
            launch_k(k_plist_tiny_update, std::min(grid_of(W.n_tiny, 128), 8 * num_sms()), 128, 0, s, L.off, L.pin, L.nsrc,
                     w, rho, W.ttouched, W.upd + U_TINY, moved, W.PL, R.D0, R.saving, uacc);
            HP_LAUNCH_CHECK();
        }
    }
    launch_k(k_rep_zero, grid_of(zspan, 256), 256, 0, s, R, reuse ? 1 : update ? 2 : 0, W.upd);
    HP_LAUNCH_CHECK();
    if (!reuse && update == 0) {
        // (a few CTAs an SM: each ends with a pass over the parts; the step call takes any sizes)
        launch_k(k_rep_nodes, std::min(grid_of(n, 256), 4 * num_sms()), 256, 0, s, rho, L.size, W.singin, n, dbg ? RN_PARTS + 1 : nparts,
                 R.psize, R.D0);
        HP_LAUNCH_CHECK();
        // pins(p,e), pins_in(p,e), D(p), saving(v)
        if (W.n_mid > 0 && nparts <= PB_PARTS) {
            const size_t sm = plist_parts_smem(nparts);
            const int occ = prepare_kernel((const void *)k_plist_parts<false>, PP_T, sm);
            const int grid = (int)std::min<int64_t>(cdiv(W.n_mid, PP_T / 32), (int64_t)num_sms() * occ);
            launch_k(k_plist_parts<false>, grid, PP_T, sm, s, L.off, L.pin, L.nsrc, w, rho, W.mid, W.n_mid, nullptr, moved,
                     nparts, W.PL, R.D0, R.saving, nullptr);
            HP_LAUNCH_CHECK();
        } else if (W.n_mid > 0) {
            // hyperedges of up to MID_SPLIT pins in small tables (many warps
            // per SM), the rest of the warp tier in tables for small_max pins
            auto plist_mid = [&](uint32_t cap, int32_t lo, int32_t hi) {
                const int per = 5 * (int)cap + 1;
                size_t sm = (size_t)per * 4 * (PLW_T / 32);
                int occ = prepare_kernel((const void *)k_plist_small, PLW_T, sm);
                int grid = (int)std::min<int64_t>(cdiv(W.n_mid, PLW_T / 32), (int64_t)num_sms() * occ);
                launch_k(k_plist_small, std::max(grid, 1), PLW_T, sm, s, L.off, L.pin, L.nsrc, w, rho, W.n_mid, W.mid,
                         W.small_max, cap, W.PL, R.D0, R.saving, lo, hi);
                HP_LAUNCH_CHECK();
            };
            if (W.pcap > pow2_at_least(2 * MID_SPLIT)) {
                plist_mid(pow2_at_least(2 * MID_SPLIT), 0, MID_SPLIT);
                plist_mid(W.pcap, MID_SPLIT, INT32_MAX);
            } else {
                plist_mid(W.pcap, 0, INT32_MAX);
            }
        }
        if (W.n_tiny > 0) {
            launch_k(k_plist_tiny, grid_of(W.n_tiny, 128), 128, 0, s, L.off, L.pin, L.nsrc, w, rho, W.tiny, W.n_tiny, W.PL, R.D0,
                     R.saving);
            HP_LAUNCH_CHECK();
        }
        if (W.n_big > 0) {
            launch_k(k_plist_big, W.pnb, 256, 0, s, L.off, L.pin, L.nsrc, w, rho, W.big, W.n_big, W.bcap, W.ptab, W.cmax_e,
                     W.PL, R.D0, R.saving);
            HP_LAUNCH_CHECK();
        }
    }
    if (!reuse) {
        W.bits_valid = false;
        // moves in isolation (Eq. 13)
        if (L.np > 0) {
            launch_k(k_cut_bits, grid_of(L.e, 256), 256, 0, s, L.off, W.PL.lam, L.e, W.cutbits,
                     reinterpret_cast<unsigned long long *>(cnt + C_ACC));
            HP_LAUNCH_CHECK();
            launch_k(k_cut_lists, grid_of(L.np, 256), 256, 0, s, L.ioff, L.inc, L.inode, L.np, R.saving, W.cutbits, W.cut,
                     R.cutn);
            HP_LAUNCH_CHECK();
        }
    }
    launch_k(k_candidates, grid_of(n, 256), 256, 0, s, R.saving, R.cutn, n, W.cl, cnt + C_CAND, W.hubs, cnt + C_HUB,
             W.cw, cnt + C_CW);
    HP_LAUNCH_CHECK();
    GainArgs G{L.off, L.ioff, R.cutn, W.cut, w, rho, L.size, R.psize, R.saving, W.wns, W.PL, P.omega, second_half, W.M};
    if (bits_pay(L, W)) {
        if (!reuse || !W.bits_valid) {
            launch_k(k_part_bits, grid_of((int64_t)L.e * 32, PB_T), PB_T, 0, s, L.off, W.PL, L.e, W.wq, W.bits);
            HP_LAUNCH_CHECK();
            W.bits_valid = true;
        }
        if (W.wq == 1) gains_bits<1>(G, W, cnt, n, s);
        else if (W.wq == 2) gains_bits<2>(G, W, cnt, n, s);
        else if (W.wq == 4) gains_bits<4>(G, W, cnt, n, s);
        else gains_bits<8>(G, W, cnt, n, s);
    } else if (nparts <= PB_PARTS && P.wsum < (1ll << 32) && P.o.debug_table_cap == 0) {
        gains_parts(G, W, cnt, n, s);
    } else {
        uint32_t gcap_smem = 2048;
        if (P.o.debug_table_cap > 0) gcap_smem = (uint32_t)P.o.debug_table_cap;
        const size_t gsm = (size_t)gcap_smem * 12 + (size_t)(gcap_smem * 3 / 4) * 4;
        {
            // hub nodes on the side stream, beside the warp and CTA tiers (disjoint
            // node lists; all append to the same move and overflow lists by atomics)
            const cudaStream_t sh = fork_side(W, s, W.side);
            const int occ_h = prepare_kernel((const void *)k_gains_smem<1024>, 1024, gsm);
            launch_k(k_gains_smem<1024>, num_sms() * std::max(occ_h, 1), 1024, gsm, sh, G, W.hubs, cnt + C_HUB, gcap_smem,
                     W.ovf, cnt + C_OVF);
            HP_LAUNCH_CHECK();
            end_side(W, sh, 1);
        }
        {
            const uint32_t wlimit = P.o.debug_table_cap > 0 ? std::min<uint32_t>(GW_SLOTS * 3 / 4, P.o.debug_table_cap / 2)
                                                            : GW_SLOTS * 3 / 4;
            int occ = prepare_kernel((const void *)k_gains_warp, GW_T, 0);
            int grid = (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(n, GW_T / 32), (int64_t)num_sms() * occ));
            launch_k(k_gains_warp, grid, GW_T, 0, s, G, W.cw, cnt + C_CW, wlimit, W.cl, cnt + C_CAND);
            HP_LAUNCH_CHECK();
        }
        {
            int occ = prepare_kernel((const void *)k_gains_smem<GN_T>, GN_T, gsm);
            int grid = std::max(1, std::min<int>(n, num_sms() * occ));
            launch_k(k_gains_smem<GN_T>, grid, GN_T, gsm, s, G, W.cl, cnt + C_CAND, gcap_smem, W.ovf, cnt + C_OVF);
            HP_LAUNCH_CHECK();
            join_side(W, s, 1);
            launch_k(k_gains_global, W.gnb, GN_T, 0, s, G, W.ovf, cnt + C_OVF, W.gcap, W.gk, W.gc, W.cl, cnt + C_BAD);
            HP_LAUNCH_CHECK();
        }
    }
    // The rest of the repetition; `end` reads its counters back (the one
    // host read of a repetition on a small level) and returns the moves applied.
    auto end = [&]() -> int32_t {
        int32_t hc[C_N];
        fetch_bytes(hc, cnt, sizeof hc, s);
        if (hc[C_BAD]) throw Error(HP_ERR_INTERNAL, "gain table overflow");
        // algorithmic bytes (scope of Sec. VI-B..VI-D): a rebuilt repetition
        // reads each pin and its part (8 B) and writes the pins-list entries
        // (12 B each), an updated one those of the hyperedges with a moved pin;
        // both scan the incidence for cut hyperedges (4 B per entry); every
        // repetition reads the cut entries (4 B) and the list entries behind
        // them (12 B), and moves 48 B per proposed move (sort read and write,
        // sequence, in-sequence gain, two capacity events, apply)
        unsigned long long acc[5];   // C_ACC, C_UPD
        std::memcpy(acc, hc + C_ACC, sizeof acc);
        if (!reuse) {
            W.alg_bytes += 4 * L.np + (update > 0 ? 8 * (int64_t)acc[3] + 12 * (int64_t)acc[4]
                                                  : 8 * L.np + 12 * (int64_t)acc[0]);
            W.cuts = (int64_t)acc[1];
            W.cut_lam = (int64_t)acc[2];
        }
        W.alg_bytes += 4 * W.cuts + 12 * W.cut_lam + 48 * (int64_t)hc[C_MOVES];
        return hc[C_APPLIED];
    };
    // Levels of at most SMALL_LEVEL nodes have at most that many moves, which
    // the cluster kernels sequence and validate whatever their number (none
    // included): no read-back is needed before the end of the repetition.
    const bool small_level = n <= SMALL_LEVEL && !dbg;
    int32_t m = n;   // an upper bound of the moves on small levels
    if (!small_level) {
        int32_t hc[C_N];
        fetch_bytes(hc, cnt, sizeof hc, s);
        if (hc[C_BAD]) throw Error(HP_ERR_INTERNAL, "gain table overflow");
        m = hc[C_MOVES];
        if (dbg) *dbg->m = m;
        if (m == 0) return end();
    }

    const long long gbound = std::max<long long>(P.wsum, 1);
    const int nb = bits_for((uint64_t)std::max(n - 1, 1)), gb = bits_for((uint64_t)gbound),
              sb = bits_for((uint64_t)std::max(nparts - 1, 1));
    const long long cgbound = (long long)std::min<double>((double)gbound * (double)std::max(n, 1), 9.0e18);
    const int cgb = bits_for((uint64_t)cgbound);
    // packed acceptance and 64-bit grades: penalties below 2^32, gains of at most 2^38
    const int packed = (10ll * P.omega + (long long)P.delta) < 0xffffffffll && P.wsum <= (1ll << 38);
    ChainCtx C;
    C.window = P.o.chain_window;
    C.node = W.S.node;
    C.src = W.S.src;
    C.dst = W.S.dst;
    C.size = L.size;
    C.nin = L.nin;
    C.msz = W.msz;
    C.mni = W.mni;
    C.gain = W.S.gain;
    C.first = W.first;
    C.pred = R.pred;
    C.succ = R.succ;
    C.choice = W.choice;
    C.pen = W.pen;
    C.minpen = W.minpen;
    C.accnode = W.accnode;
    C.acc[0] = R.acc0;
    C.acc[1] = W.acc1;
    C.acc[2] = W.acc2;
    C.linked = R.linked;
    SeqCtx Q{W.S.node, R.pred, R.succ, W.S.gain, R.chain, W.pos, W.clen, R.cgain, err_dev};
    ValCtx V{W.seqmove, L.size, W.singin, R.dDs, R.dDd, R.D0, R.gseq, W.S, R.psize, W.vkey, W.vidx, W.vsz, W.vdd,
             R.viol, P.omega, P.delta, W.gsz, W.gdd, W.esz, W.edd, W.vhead};
    // one CTA sequences the moves unless the chaining window scans would be
    // long: every free end scans up to min(window, moves per part) moves of
    // its destination, each round (few parts in use make that quadratic)
    const int64_t per_part = cdiv(m, std::max<int32_t>(W.parts_used, 1));
    const int64_t scan_work = (int64_t)m * std::min<int64_t>(P.o.chain_window, per_part);
    // (on a larger level the device-wide path takes over above a few thousand
    // moves: the cluster's eight SMs then lose to the whole GPU's phases)
    const bool small = m <= SMALLM,
               one_cluster = small_level || (m <= SEQ_CLUSTER_M && scan_work <= (int64_t(1) << 21));
    if (one_cluster) {
        ClusterSeqArgs SA{W.M, W.S, W.keys, W.hkeys, W.idx, W.heads, W.first, W.lens, W.starts, W.cstart,
                          W.seqmove, R.mvpos, cnt, C, Q, nparts, P.o.chain_rounds, packed, gb, nb, sb, cgb, gbound,
                          cgbound};
        const size_t sm = SQ_SMEM;
        prepare_kernel((const void *)k_seq_cluster, SEQ_T, sm);
        launch_k(k_seq_cluster, SQ_CS, SEQ_T, sm, s, SA);
        HP_LAUNCH_CHECK();
    } else {
        // sort (p_s asc, gain desc, node asc)
        if (sb + gb + nb <= 64) {
            launch_k(k_move_keys, grid_of(m, 256), 256, 0, s, W.M, cnt + C_MOVES, gbound, gb, nb, -1, W.keys, W.idx, 1);
            HP_LAUNCH_CHECK();
            radix_sort_dev(W.keys, W.idx, cnt + C_MOVES, m, sb + gb + nb, A);
        } else {
            const int fb[3] = {nb, gb, sb};
            for (int f = 0; f < 3; f++) {
                launch_k(k_move_keys, grid_of(m, 256), 256, 0, s, W.M, cnt + C_MOVES, gbound, gb, nb, f, W.keys, W.idx,
                         f == 0);
                HP_LAUNCH_CHECK();
                radix_sort_dev(W.keys, W.idx, cnt + C_MOVES, m, fb[f], A);
            }
        }
        launch_k(k_gather_moves, grid_of(m, 256), 256, 0, s, W.M, W.idx, cnt + C_MOVES, W.S, R.pc, L.size, L.nin, W.msz,
                 W.mni);
        HP_LAUNCH_CHECK();
        scan_excl(R.pc, W.first, nparts + 1, nullptr, A);
        // chaining (Sec. VI-C)
        // (two passes per round here: on these levels the window scans are
        // long, and the one-pass round's extra slot read per scanned move
        // costs more than the barrier it saves)
        for (int32_t r = 0; r < P.o.chain_rounds; r++) {
            if (packed) {
                launch_k(k_choose_warp, grid_of((int64_t)m * 32, 128), 128, 0, s, C, cnt + C_MOVES, r);
                HP_LAUNCH_CHECK();
            } else {
                launch_k(k_choose, grid_of(m, 128), 128, 0, s, C, cnt + C_MOVES, r);
                HP_LAUNCH_CHECK();
                launch_k(k_accept_min, grid_of(m, 256), 256, 0, s, C, cnt + C_MOVES, r);
                HP_LAUNCH_CHECK();
                launch_k(k_accept_id, grid_of(m, 256), 256, 0, s, C, cnt + C_MOVES, r);
                HP_LAUNCH_CHECK();
            }
            launch_k(k_link, grid_of(m, 256), 256, 0, s, C, cnt + C_MOVES, r, packed);
            HP_LAUNCH_CHECK();
        }
        // chains in order of (total gain desc, head node asc)
        launch_k(k_path_heads, grid_of(m, 256), 256, 0, s, Q, cnt + C_MOVES);
        HP_LAUNCH_CHECK();
        launch_k(k_cycle_heads, grid_of(m, 256), 256, 0, s, Q, cnt + C_MOVES);
        HP_LAUNCH_CHECK();
        launch_k(k_head_collect, grid_of(m, 256), 256, 0, s, Q, cnt + C_MOVES, W.heads, cnt + C_NH);
        HP_LAUNCH_CHECK();
        if (cgb + nb <= 64) {
            launch_k(k_head_keys, grid_of(m, 256), 256, 0, s, W.heads, cnt + C_NH, R.cgain, W.S.node, cgbound, nb, -1,
                     W.hkeys);
            HP_LAUNCH_CHECK();
            radix_sort_dev(W.hkeys, W.heads, cnt + C_NH, m, cgb + nb, A);
        } else {
            for (int f = 0; f < 2; f++) {
                launch_k(k_head_keys, grid_of(m, 256), 256, 0, s, W.heads, cnt + C_NH, R.cgain, W.S.node, cgbound, nb, f,
                         W.hkeys);
                HP_LAUNCH_CHECK();
                radix_sort_dev(W.hkeys, W.heads, cnt + C_NH, m, f == 0 ? nb : cgb, A);
            }
        }
        launch_k(k_chain_lens, grid_of(m, 256), 256, 0, s, W.heads, cnt + C_NH, W.clen, m, W.lens);
        HP_LAUNCH_CHECK();
        scan_excl(W.lens, W.starts, m, nullptr, A);
        launch_k(k_chain_start, grid_of(m, 256), 256, 0, s, W.heads, cnt + C_NH, W.starts, W.cstart);
        HP_LAUNCH_CHECK();
        launch_k(k_seq_pos, grid_of(m, 256), 256, 0, s, R.chain, W.pos, W.cstart, cnt + C_MOVES, W.S.node, W.seqmove,
                 R.mvpos);
        HP_LAUNCH_CHECK();
    }
    if (dbg) {
        HPC(cudaMemcpyAsync(dbg->node, W.S.node, sizeof(int32_t) * m, cudaMemcpyDeviceToDevice, s));
        HPC(cudaMemcpyAsync(dbg->src, W.S.src, sizeof(int32_t) * m, cudaMemcpyDeviceToDevice, s));
        HPC(cudaMemcpyAsync(dbg->dst, W.S.dst, sizeof(int32_t) * m, cudaMemcpyDeviceToDevice, s));
        HPC(cudaMemcpyAsync(dbg->gain, W.S.gain, sizeof(long long) * m, cudaMemcpyDeviceToDevice, s));
        HPC(cudaMemcpyAsync(dbg->seq, W.seqmove, sizeof(int32_t) * m, cudaMemcpyDeviceToDevice, s));
    }

    // in-sequence gains and distinct-inbound changes per move
    SeqSim Z{L.off, L.pin, L.nsrc, w, R.mvpos, W.seqmove, W.S.src, W.S.dst, W.PL, R.gseq, R.dDs, R.dDd};
    if (W.n_tiny > 0) {
        launch_k(k_inseq_tiny, grid_of(W.n_tiny, IST_T), IST_T, 0, s, Z, W.tiny, W.n_tiny, cnt + C_MOVES);
        HP_LAUNCH_CHECK();
    }
    if (W.n_mid > 0) {
        launch_k(k_touched, grid_of(W.n_mid, 256), 256, 0, s, L.off, L.pin, R.mvpos, W.mid, W.n_mid, W.touched, cnt + C_TOUCH,
                 cnt + C_MOVES);
        HP_LAUNCH_CHECK();
        auto inseq_mid = [&](int32_t lo, int32_t emax) {
            if (nparts <= PB_PARTS) {
                const size_t sm = inseq_parts_smem(nparts, emax);
                const int occ = prepare_kernel((const void *)k_inseq_parts, IS_T, sm);
                const int grid = (int)std::min<int64_t>(cdiv(W.n_mid, IS_T / 32), (int64_t)num_sms() * occ);
                launch_k(k_inseq_parts, std::max(grid, 1), IS_T, sm, s, Z, W.touched, cnt + C_TOUCH, emax, nparts,
                         cnt + C_MOVES, lo);
                HP_LAUNCH_CHECK();
                return;
            }
            size_t sm = (size_t)(9 * emax + 1) * 4 * (IS_T / 32);
            int occ = prepare_kernel((const void *)k_inseq_small, IS_T, sm);
            int grid = (int)std::min<int64_t>(cdiv(W.n_mid, IS_T / 32), (int64_t)num_sms() * occ);
            launch_k(k_inseq_small, std::max(grid, 1), IS_T, sm, s, Z, W.touched, cnt + C_TOUCH, emax, cnt + C_MOVES, lo);
            HP_LAUNCH_CHECK();
        };
        // (two launches on larger levels: the smaller buffers let more warps in)
        if (W.small_max > MID_SPLIT && !(small_level && nparts <= PB_PARTS)) {
            inseq_mid(0, MID_SPLIT);
            inseq_mid(MID_SPLIT, W.small_max);
        } else {
            inseq_mid(0, W.small_max);
        }
    }
    if (W.n_big > 0) {
        launch_k(k_inseq_big, W.pnb, 256, 0, s, Z, W.big, W.n_big, W.cmax_e, W.ibuf, cnt + C_MOVES);
        HP_LAUNCH_CHECK();
    }

    // validity of every prefix (Sec. VI-D), best valid prefix, apply
    if (small_level) {
        prepare_kernel((const void *)k_val_cluster, SQ_T, SQ_SMEM);
        launch_k(k_val_cluster, SQ_CS, SQ_T, SQ_SMEM, s, V, cnt, nparts, sb, W.bgain, rho);
        HP_LAUNCH_CHECK();
    } else if (small) {
        size_t sm = (size_t)2 * SMALLM * 2 * (4 + 4);
        prepare_kernel((const void *)k_val_small, SEQ_T, sm);
        launch_k(k_val_small, 1, SEQ_T, sm, s, V, cnt, nparts, sb, W.bgain, rho);
        HP_LAUNCH_CHECK();
    } else {
        launch_k(k_val_entries, grid_of(m, 256), 256, 0, s, V, cnt + C_MOVES, cnt + C_NV);
        HP_LAUNCH_CHECK();
        radix_sort_dev(W.vkey, W.vidx, cnt + C_NV, 2 * (int64_t)m, sb, A);
        launch_k(k_val_gather, grid_of(2 * (int64_t)m, 256), 256, 0, s, V, cnt + C_NV);
        HP_LAUNCH_CHECK();
        scan_excl((const int64_t *)W.gsz, (int64_t *)W.esz, 2 * (int64_t)m, nullptr, A);
        scan_excl((const int64_t *)W.gdd, (int64_t *)W.edd, 2 * (int64_t)m, nullptr, A);
        launch_k(k_val_trans, grid_of(2 * (int64_t)m, 256), 256, 0, s, V, cnt + C_NV);
        HP_LAUNCH_CHECK();
        launch_k(k_initial_bad, grid_of(nparts, 256), 256, 0, s, R.psize, R.D0, nparts, P.omega, P.delta, cnt + C_BAD0);
        HP_LAUNCH_CHECK();
        launch_k(k_best_prefix, 1, 1024, 0, s, R.gseq, R.viol, cnt + C_MOVES, cnt + C_BAD0, cnt + C_APPLIED, W.bgain);
        HP_LAUNCH_CHECK();
        launch_k(k_apply, grid_of(m, 256), 256, 0, s, W.seqmove, W.S.node, W.S.dst, cnt + C_APPLIED, rho);
        HP_LAUNCH_CHECK();
    }
    if (dbg) {
        HPC(cudaMemcpyAsync(dbg->gseq, R.gseq, sizeof(long long) * m, cudaMemcpyDeviceToDevice, s));
        HPC(cudaMemcpyAsync(dbg->best_gain, W.bgain, sizeof(long long), cudaMemcpyDeviceToDevice, s));
    }
    return end();
}

__global__ void k_max_edge_i(const int32_t *off, int32_t e, int32_t *maxe) {
    HP_KERNEL_ENTER();
    int32_t m = 0;
    GRID_STRIDE(i, (int64_t)e) m = max(m, off[i + 1] - off[i]);
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(maxe, m);
}

int32_t max_edge_size(const Level &L, Arena &A) {
    cudaStream_t s = A.stream();
    int32_t *mx = A.get<int32_t>(1);
    HPC(cudaMemsetAsync(mx, 0, sizeof(int32_t), s));
    if (L.e > 0) {
        launch_k(k_max_edge_i, grid_of(L.e, 256), 256, 0, s, L.off, L.e, mx);
        HP_LAUNCH_CHECK();
    }
    const int32_t r = fetch<int32_t>(mx, s);
    A.release(mx);
    return r;
}

int32_t refine_rep_debug(const Level &L, const int32_t *w, int32_t nparts, const Params &P, int32_t *rho,
                         int second_half, Arena &A, uint32_t *err_dev, const RepDebug &dbg) {
    *dbg.m = 0;
    if (L.n == 0) return 0;
    const int32_t max_e = max_edge_size(L, A);
    LevelWs *W = refine_workspace(L.n, L.np, L.e, nparts, max_e, P, A);
    level_prepare(L, w, rho, *W, A);
    int32_t k = rep_run(L, w, P, rho, second_half, *W, A, err_dev, &dbg);
    refine_workspace_free(W, A);
    return k;
}

__global__ void k_relabel(const int32_t *newid, int32_t n, int32_t *rho) {
    HP_KERNEL_ENTER();
    GRID_STRIDE(v, (int64_t)n) rho[v] = newid[rho[v]];
}
// Parts that have emptied never hold a node again, so once half of the ids
// are out of use the parts in use are renumbered in ascending order, which no
// decision can tell from the old ids (ties go by their order).  A net that
// stops coarsening at ten thousand nodes and ends in a hundred parts then has
// the tables, keys and part-indexed kernels of a hundred parts.
static void renumber_parts(const Level &L, const Params &P, int32_t *rho, LevelWs &W, Arena &A) {
    if (2 * (int64_t)W.parts_used > W.nparts) return;
    scan_excl(W.pmark, W.pnew, W.nparts, nullptr, A);
    launch_k(k_relabel, grid_of(L.n, 256), 256, 0, A.stream(), W.pnew, L.n, rho);
    HP_LAUNCH_CHECK();
    W.nparts = W.R.nparts = W.parts_used;
    part_bits_rows(W, P, A);
}

RefineOut refine_level(const Level &L, const int32_t *w, const Params &P, int32_t *rho, LevelWs *W, Arena &A,
                       uint32_t *err_dev) {
    RefineOut out;
    if (L.n == 0 || P.o.theta == 0) return out;
    level_prepare(L, w, rho, *W, A);
    renumber_parts(L, P, rho, *W, A);
    const int64_t bytes0 = W->alg_bytes;
    const int32_t half = P.o.theta / 2;
    bool same_rho = false;   // the previous repetition applied nothing
    int32_t applied = 0;     // moves the previous one applied
    for (int32_t rep = 0; rep < P.o.theta; rep++) {
        // an update touches the moved nodes' hyperedges only; on small levels a
        // rebuild is as short as the update's four launches (UPDATE_NP), and with
        // many moves most hyperedges have one (1M Gaussian net: up to an eighth
        // of the nodes 620.4 ms, a half 621.0, a 128th 623.0)
        const int32_t update = L.np >= UPDATE_NP && W->n_big == 0 && W->nparts <= PB_PARTS && 8 * (int64_t)applied <= L.n
                                   ? applied : 0;
        const int32_t k = rep_run(L, w, P, rho, rep >= half, *W, A, err_dev, nullptr, same_rho, update);
        applied = k;
        same_rho = k == 0;
        out.reps++;
        out.moves += k;
        if (k == 0) {
            if (rep < half) rep = half - 1;
            else break;
        }
    }
    out.alg_bytes = W->alg_bytes - bytes0;
    return out;
}

// ---------------------------------------------------------------- final statistics
__global__ void k_part_sizes(const int32_t *part, int32_t n, long long *psize) {
    HP_KERNEL_ENTER();
    GRID_STRIDE(v, (int64_t)n) atomicAdd((unsigned long long *)&psize[part[v]], 1ull);
}
__global__ void k_part_max(const long long *psize, const int32_t *D, int32_t nparts, int32_t omega, int32_t delta,
                           long long *out) {
    HP_KERNEL_ENTER();
    long long ms = 0, md = 0, bad = 0;
    GRID_STRIDE(p, (int64_t)nparts) {
        ms = max(ms, psize[p]);
        md = max(md, (long long)D[p]);
        bad += (psize[p] > omega || D[p] > delta) ? 1 : 0;
    }
    for (int o = 16; o > 0; o >>= 1) {
        ms = max(ms, __shfl_down_sync(0xffffffffu, ms, o));
        md = max(md, __shfl_down_sync(0xffffffffu, md, o));
        bad += __shfl_down_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax((unsigned long long *)&out[2], (unsigned long long)ms);
        atomicMax((unsigned long long *)&out[3], (unsigned long long)md);
        atomicAdd((unsigned long long *)&out[4], (unsigned long long)bad);
    }
}

// out (device int64[5]): connectivity, cut-net, max part size, max distinct
// inbound hyperedges of a part, parts violating Omega or Delta; max_e: the largest hyperedge
void part_stats(const Level &L, const int32_t *w, const int32_t *part, int32_t nparts, int32_t max_e, int32_t omega,
                int32_t delta, int64_t *out, Arena &A) {
    cudaStream_t s = A.stream();
    HPC(cudaMemsetAsync(out, 0, 5 * sizeof(int64_t), s));
    if (nparts <= 0) return;
    int32_t *D = A.get<int32_t>(nparts);
    long long *psize = A.get<long long>(nparts);
    HPC(cudaMemsetAsync(D, 0, sizeof(int32_t) * nparts, s));
    HPC(cudaMemsetAsync(psize, 0, sizeof(long long) * nparts, s));
    if (L.e > 0 && nparts <= PB_PARTS) {
        part_scan<false>(L.off, L.pin, L.nsrc, w, L.e, part, L.n, nparts, D, out, out + 1, nullptr, 0, nullptr,
                         max_e > PS_BIG, A);
    } else if (L.e > 0) {
        int32_t *maxe = A.get<int32_t>(1);
        HPC(cudaMemsetAsync(maxe, 0, sizeof(int32_t), s));
        launch_k(k_max_edge, grid_of(L.e, 256), 256, 0, s, L.off, L.e, maxe);
        HP_LAUNCH_CHECK();
        int32_t me = fetch<int32_t>(maxe, s);
        Plist PL;
        PL.p = A.get<int32_t>(L.np);
        PL.cnt = A.get<int32_t>(L.np);
        PL.cin = A.get<int32_t>(L.np);
        PL.lam = A.get<int32_t>(L.e);
        build_plist(L, w, part, me, PL, D, nullptr, A);
        launch_k(k_objective, grid_of(L.e, 256), 256, 0, s, PL.lam, w, L.e, (unsigned long long *)out,
                 (unsigned long long *)(out + 1));
        HP_LAUNCH_CHECK();
        A.release(PL.p);
        A.release(PL.cnt);
        A.release(PL.cin);
        A.release(PL.lam);
        A.release(maxe);
    }
    launch_k(k_part_sizes, grid_of(L.n, 256), 256, 0, s, part, L.n, psize);
    HP_LAUNCH_CHECK();
    launch_k(k_part_max, grid_of(nparts, 256), 256, 0, s, psize, D, nparts, omega, delta, (long long *)out);
    HP_LAUNCH_CHECK();
    A.release(D);
    A.release(psize);
}

}  // namespace hp
