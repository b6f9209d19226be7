// Force pass by contact items: FP64 mode (walk and lists) and the FP32 walk of few particles.
//
//   k_items  steps 5-8 and 1 (walk: also the new cell key of step 2) for a block of
//            ITEM_THREADS threads on `tile` consecutive stored particles (16 to 128).
//            1. all threads search: the particles' list entries, or the 27 cells as 9 rows of
//               three x-adjacent cells, against the FP32 prefilter;
//            2. what passes becomes one item per pair, in shared memory: a pair of two
//               particles of the block is one item (its evaluations from the two sides are
//               exact negatives of each other), a pair across blocks one per block;
//            3. every thread evaluates items (contact decision, spring, law) and leaves force,
//               torque arm and spring in shared memory;
//            4. one thread per particle adds its contacts up in list (walk: stored) order,
//               then walls, gravity, update, as in k_list and k_force.
//
// Why: GB300's FP64 pipe does 0.58 T fused operations per second for the whole chip, so what
// an FP64 pass costs is the number of warp instructions it sends there. A thread per particle
// evaluated every pair twice, with the lanes of a warp holding 0 to 12 contacts each. Items
// evaluate 0.7 of the contacts (two thirds of a 128-particle tile's pairs are inside it) with
// all lanes busy. And a small scene leaves most of the chip idle with a thread per particle;
// here a particle's contacts run side by side on the threads of its block.
// If the items of a block do not fit (ITEM_MAX), it takes its particles in several rounds and
// evaluates every pair from both sides. The sums do not depend on any of this.
// Measured (GB300, dense boxes, per step, thread per particle -> items): 2,048 spheres walking
// 230 -> 50 us, 262,144 with lists 1,026 -> 539 us, one force evaluation of 65,537 (with load and
// sort) 564 -> 301 us. Tiles of 64 particles take 713 us with lists (fewer pairs inside; 256 would
// be more than ITEM_MAX items), 85 registers and three blocks per SM 563 us and 10% more on 2,048.
#include <algorithm>

#include <cuda_runtime.h>

#include "dem_domain.h"
#include "dem_policy.cuh"

namespace demgb {

constexpr uint32_t ITEM_THREADS = 256;
constexpr uint32_t ITEM_MAX = 768;      // items of a round (a particle has at most 64 + a few)
constexpr uint32_t ENTRY_MAX = 1280;    // near candidates of a round
constexpr uint16_t NO_ITEM = 0xFFFFu;

template <class PR>
struct ItemArgs {
    using T = typename PR::T;
    const SceneDev* scenes;
    int nscenes;
    uint32_t n, cap, tile, hcap;
    int maxc, stiffness;
    typename PR::State S0, S1;
    CtrlDev* ctrl;
    // lists
    const uint32_t* ncnt;
    const uint32_t* nl;
    const uint2* nl4;
    const uint32_t* halo;
    const uint32_t* nhalo;
    const float4* ref;           // lists: positions at the last sort; walk: FP32 (x, y, z, r) of the sorted particles
    int interval;
    const uint32_t* wmask;
    uint64_t* hmask[2];
    int loop;
    // walk
    const uint32_t* skey;
    const uint32_t* cs;
    uint32_t* key;
    uint32_t* rank;
    uint32_t* cnt;
    // both
    const uint32_t* perm;
    uint32_t* hcnt[2];
    Spring<T>* hs[2];
    int hin;                     // walk: history buffer read (lists: ctrl->hcur)
    StatusDev* st;
    double* dbgF;
    double* dbgT;
    int halt;
    int once;                    // both particles of a pair hold its spring
};

// Values an item leaves per contact: force, torque arm n x F_t, spring, and with the optional
// terms the rolling moment; the simple law has its force alone.
template <int MODEL>
struct ItemRes {
    static constexpr uint32_t N = MODEL == 1 ? 3u : (MODEL == 2 ? 12u : 9u);
};

// Bytes of shared memory, and where each array starts (the kernel and its launcher).
template <class PR, bool LIST, int MODEL>
struct ItemMem {
    uint32_t res, delta, pre, gid, nb, near, src, cold, om, sc, pid, ent, itm, own, slot, item, total;
    __host__ __device__ ItemMem(uint32_t P, uint32_t hcap, uint32_t maxc) {
        uint32_t o = 0;
        auto put = [&](uint32_t& at, uint32_t bytes) {
            at = o;
            o += (bytes + 15u) & ~15u;
        };
        const uint32_t E = P + hcap;
        put(res, ItemRes<MODEL>::N * ITEM_MAX * (uint32_t)sizeof(typename PR::T));
        put(delta, ITEM_MAX * 4);
        put(pre, LIST ? E * 16 : 0);
        put(gid, LIST ? E * 4 : 0);
        put(nb, (P + 1) * 4);
        put(near, LIST ? P * 8 : P * 18);       // lists: mask of the entries; walk: counts of 9 rows
        put(src, P * 4);
        put(cold, P * 4);
        put(om, LIST ? P * 8 : 0);
        put(sc, P * 4);
        put(pid, LIST || MODEL == 1 ? 0 : P * maxc * 4);
        put(ent, ENTRY_MAX * 4);
        put(itm, ENTRY_MAX * 2);
        put(own, ENTRY_MAX);
        put(slot, LIST ? ENTRY_MAX : 0);
        put(item, ITEM_MAX * 2);
        total = o;
    }
};

// Whether two stored particles touch, as PF64::exact_j decides it (out of line: few blocks ask).
__device__ __noinline__ bool touch(const double* x, const double* y, const double* z, const float* r, uint32_t i,
                                   uint32_t j) {
    const double dx = __dsub_rn(x[j], x[i]), dy = __dsub_rn(y[j], y[i]), dz = __dsub_rn(z[j], z[i]);
    const double R = __dadd_rn((double)r[i], (double)r[j]);
    return __fma_rn(dz, dz, __fma_rn(dy, dy, __dmul_rn(dx, dx))) < __dmul_rn(R, R);
}

template <class PR, bool LIST, int MODEL, bool EVAL>
__global__ void __launch_bounds__(ITEM_THREADS, 2) k_items(ItemArgs<PR> a) {
    using T = typename PR::T;
    constexpr bool PRACT = MODEL != 1;
    constexpr bool TERMS = MODEL == 2;
    constexpr int STIFF = MODEL == 2 ? 2 : (MODEL == 3 ? 1 : 0);
    const unsigned full = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char mem[];
    __shared__ uint32_t s_sum[3], s_max[3], s_flag, s_items, s_warp[ITEM_THREADS / 32];
    __shared__ int s_void;
    if (!EVAL && LIST && a.loop && a.ctrl->stop != LOOP_GO) return;   // (written between passes only)
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5;
    if (tid == 0) s_void = a.ctrl->rebuild & DEM_HALT;
    if (tid < 3) s_sum[tid] = s_max[tid] = 0u;
    if (tid == 3) s_flag = 0u;
    __syncthreads();
    if (!EVAL && s_void) return;   // a void step
    const int cur = a.ctrl->cur;
    const typename PR::State A = cur ? a.S1 : a.S0;
    const typename PR::State B = cur ? a.S0 : a.S1;
    const bool pv = a.ctrl->perm_valid != 0;
    const int hi = LIST ? a.ctrl->hcur : a.hin, ho = 1 - hi;
    if (!EVAL && LIST && blockIdx.x == 0 && tid == 0) {
        a.ctrl->hlast = ho;
        if (a.interval > 0 && a.ctrl->since + 1 >= a.interval) atomicOr(&a.ctrl->rebuild, 1);
    }
    const Spring<T>* __restrict__ hin = hi ? a.hs[1] : a.hs[0];
    const uint32_t* __restrict__ hin_cnt = hi ? a.hcnt[1] : a.hcnt[0];
    uint32_t* __restrict__ hout_cnt = ho ? a.hcnt[1] : a.hcnt[0];
    Spring<T>* __restrict__ hout = ho ? a.hs[1] : a.hs[0];
    const uint32_t maxc = (uint32_t)a.maxc, P = a.tile, G = ITEM_THREADS / P;
    const size_t cap = a.cap;
    const ItemMem<PR, LIST, MODEL> M(P, a.hcap, maxc);
    T* res = (T*)(mem + M.res);
    float* delta_of = (float*)(mem + M.delta);   // overlap of an item; -1: no contact
    float4* t_pre = (float4*)(mem + M.pre);
    uint32_t* t_gid = (uint32_t*)(mem + M.gid);
    uint32_t* nb = (uint32_t*)(mem + M.nb);      // first near candidate of each particle
    uint32_t* near = (uint32_t*)(mem + M.near);
    uint16_t* rows = (uint16_t*)(mem + M.near);
    uint32_t* s_src = (uint32_t*)(mem + M.src);
    uint32_t* s_cold = (uint32_t*)(mem + M.cold);
    uint32_t* s_om = (uint32_t*)(mem + M.om);
    uint32_t* s_sc = (uint32_t*)(mem + M.sc);    // scene, or ~0: no particle (or a frozen one)
    uint32_t* s_pid = (uint32_t*)(mem + M.pid);
    uint32_t* ent = (uint32_t*)(mem + M.ent);    // near candidates: tile entry (direct tiles, walk: stored index)
    uint16_t* itm = (uint16_t*)(mem + M.itm);    // their items
    uint8_t* own = (uint8_t*)(mem + M.own);      // whose they are
    uint8_t* slot = (uint8_t*)(mem + M.slot);    // lists: which list entry
    uint16_t* item = (uint16_t*)(mem + M.item);  // near candidate of each item

    // ---- the particles of the block
    uint32_t q0, np, tile_scene = 0;
    if (LIST) {
        tile_scene = (uint32_t)scene_of_tile(a.scenes, a.nscenes, blockIdx.x);
        const SceneDev& S = a.scenes[tile_scene];
        const uint32_t off = (blockIdx.x - S.t0) * P;
        q0 = S.p0 + off;
        np = min(P, S.np - off);
    } else {
        q0 = blockIdx.x * P;
        np = min(P, a.n - q0);
    }
    const bool mine = tid < np;     // this thread's own particle, from the search to the update
    const uint32_t q = q0 + tid;
    bool live = false;
    if (tid < P) {
        uint32_t src = 0, cold = 0, sc = 0xFFFFFFFFu;
        uint2 om = make_uint2(0u, 0u);
        if (mine) {
            const uint32_t s = LIST ? tile_scene : (uint32_t)scene_of(a.scenes, a.nscenes, q);
            const SceneDev& S = a.scenes[s];
            live = S.active != 0;
            src = pv ? __ldg(&a.perm[q]) : q;
            if (PRACT || !live) {
                cold = min(__ldg(&hin_cnt[src]), maxc);
                if (LIST) om = __ldg((const uint2*)&(hi ? a.hmask[1] : a.hmask[0])[q]);
            }
            if (live) sc = s;
            else if (!EVAL) {
                // frozen scene: carry state and springs unchanged
                PR::store(B, q, PR::load(A, q));
                for (uint32_t k = 0; k < cold; ++k) hout[k * cap + q] = hin[k * cap + src];
                hout_cnt[q] = cold;
                if (LIST) {
                    *(uint2*)&(ho ? a.hmask[1] : a.hmask[0])[q] = om;
                } else {
                    const uint32_t kk = a.skey[q];
                    a.key[q] = kk;
                    a.rank[q] = atomicAdd(&a.cnt[kk], 1u);
                }
            } else {
                hout_cnt[q] = 0;
            }
        }
        s_src[tid] = src;
        s_cold[tid] = live ? cold : 0u;
        s_sc[tid] = sc;
        if (LIST) {
            s_om[2 * tid] = om.x;
            s_om[2 * tid + 1] = om.y;
            near[2 * tid] = near[2 * tid + 1] = 0u;
        }
    }
    const uint32_t nh = LIST ? __ldg(&a.nhalo[blockIdx.x]) : HALO_NONE;
    const bool direct = nh == HALO_NONE;   // (lists: the halo does not fit)
    if (LIST && !direct) {
        if (mine) {
            t_pre[tid] = PR::pre(A, q);
            t_gid[tid] = q;
        }
        const uint32_t* __restrict__ halo = a.halo + (size_t)blockIdx.x * a.hcap;
        for (uint32_t k = tid; k < nh; k += ITEM_THREADS) {
            const uint32_t j = __ldg(&halo[k]);
            t_pre[P + k] = PR::pre(A, j);
            t_gid[P + k] = j;
        }
    }
    __syncthreads();

    // ---- search: thread (p, sub) takes every G-th piece of particle p's candidates
    const uint32_t p = tid & (P - 1u), sub = tid / P;   // (P a power of two)
    const uint32_t psc = s_sc[p];
    const bool plive = psc != 0xFFFFFFFFu;
    const SceneDev& PS = a.scenes[plive ? psc : 0u];
    float4 pp = make_float4(0.f, 0.f, 0.f, 0.f);
    float peps = 0.f;
    uint32_t pm = 0;
    int pix = 0, piy = 0, piz = 0;
    if (plive) {
        pp = LIST ? (direct ? PR::pre(A, q0 + p) : t_pre[p]) : PR::pre(A, q0 + p);
        peps = PR::pre_eps(PS, pp);
        if (LIST) {
            pm = min(__ldg(&a.ncnt[q0 + p]), (uint32_t)DEM_LIST_CAP);
        } else {
            const uint32_t local = a.skey[q0 + p] - PS.c0;
            const uint32_t t1 = local / (uint32_t)PS.dims[0];
            pix = (int)(local % (uint32_t)PS.dims[0]);
            piy = (int)(t1 % (uint32_t)PS.dims[1]);
            piz = (int)(t1 / (uint32_t)PS.dims[1]);
        }
    }
    // candidates of row r of particle p's 27 cells (walk)
    auto row = [&](uint32_t r, uint32_t& j0, uint32_t& j1) {
        const int z = piz + (int)(r / 3u) - 1, y = piy + (int)(r % 3u) - 1;
        j0 = j1 = 0;
        if (z < 0 || z >= PS.dims[2] || y < 0 || y >= PS.dims[1]) return;
        const uint32_t base = PS.c0 + (uint32_t)((z * PS.dims[1] + y) * PS.dims[0]);
        j0 = __ldg(&a.cs[base + (uint32_t)max(pix - 1, 0)]);
        j1 = __ldg(&a.cs[base + (uint32_t)min(pix + 1, PS.dims[0] - 1) + 1u]);
    };
    auto walk_near = [&](uint32_t j) {
        if (sizeof(T) == 4) return j != q0 + p && near_f(pp, PR::pre(A, j), peps);   // (as k_force)
        return j != q0 + p && !far_f(pp, __ldg(&a.ref[j]), peps);
    };
    bool exact = false;   // FP64: candidates are contacts (below)
    auto touches = [&](uint32_t j) {
        if constexpr (sizeof(T) == 8) return touch(A.x, A.y, A.z, A.r, q0 + p, j);
        else return true;
    };
    auto count_rows = [&](auto passes) {
        for (uint32_t r = sub; r < 9u; r += G) {
            uint32_t c = 0;
            if (plive) {
                uint32_t j0, j1;
                row(r, j0, j1);
                for (uint32_t j = j0; j < j1; ++j) c += passes(j) ? 1u : 0u;
            }
            rows[p * 9u + r] = (uint16_t)min(c, 0xFFFFu);
        }
    };
    if (LIST) {
        if (!direct) {
            for (uint32_t k = 4u * sub; k < pm; k += 4u * G) {
                const uint2 u = __ldg(&a.nl4[(size_t)(k >> 2) * cap + q0 + p]);
                uint32_t b = near_f(pp, t_pre[u.x & 0xffffu], peps) ? 1u : 0u;
                b |= near_f(pp, t_pre[u.x >> 16], peps) ? 2u : 0u;
                b |= near_f(pp, t_pre[u.y & 0xffffu], peps) ? 4u : 0u;
                b |= near_f(pp, t_pre[u.y >> 16], peps) ? 8u : 0u;
                if (k + 4u > pm) b &= (1u << (pm - k)) - 1u;   // (the last element is padded)
                if (b) atomicOr(&near[2 * p + (k >> 5)], b << (k & 31u));
            }
        } else {
            for (uint32_t k = sub; k < pm; k += G)
                if (near_f(pp, PR::pre(A, __ldg(&a.nl[k * cap + q0 + p])), peps))
                    atomicOr(&near[2 * p + (k >> 5)], 1u << (k & 31u));
        }
    } else {
        count_rows(walk_near);
        if (PRACT) {
            const uint32_t c = s_cold[p], src = s_src[p];
            for (uint32_t k = sub; k < c; k += G) s_pid[k * P + p] = __ldg(&hin[k * cap + src].pid);
        }
    }
    __syncthreads();
    // ---- how many each particle has, and where they start
    uint32_t mycnt = 0;
    if (mine && live) {
        if (LIST) {
            mycnt = (uint32_t)(__popc(near[2 * tid]) + __popc(near[2 * tid + 1]));
        } else {
            for (uint32_t r = 0; r < 9u; ++r) mycnt += rows[tid * 9u + r];
        }
    }
    if (!LIST) {
        // FP64: the prefilter's margin grows with the coordinates, and far from the origin it
        // passes spheres that are nowhere near: a block with a particle that has more of them
        // than a round holds counts contacts instead
        if (sizeof(T) == 8 && __syncthreads_or(mycnt > ITEM_MAX ? 1 : 0)) {
            exact = true;
            count_rows([&](uint32_t j) { return walk_near(j) && touches(j); });
            __syncthreads();
            mycnt = 0;
            if (mine && live)
                for (uint32_t r = 0; r < 9u; ++r) mycnt += rows[tid * 9u + r];
        }
        // more candidates than slots: FP32 counts what passes the prefilter, FP64 contacts
        // (below); no particle has more than a round holds
        const uint32_t most = sizeof(T) == 8 ? ITEM_MAX : maxc;
        if (mycnt > most) {
            raise_status(a.st, ST_CAPACITY, (int32_t)q);
            if (!EVAL && a.halt) atomicOr(&s_flag, DEM_HALT);
            mycnt = most;
        }
    }
    {
        uint32_t inc = mycnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(full, inc, o);
            if (lane >= (uint32_t)o) inc += t;
        }
        if (lane == 31u) s_warp[wid] = inc;
        __syncthreads();
        uint32_t before = 0;
        for (uint32_t w = 0; w < wid; ++w) before += s_warp[w];
        if (tid < P) nb[tid + 1u] = before + inc;
        if (tid == 0) nb[0] = 0u;
    }
    __syncthreads();

    // ---- rounds: normally one, with every pair inside the block evaluated once
    V3<T> F = mk(T(0), T(0), T(0)), Tq = mk(T(0), T(0), T(0));
    uint32_t nnew = 0, nm0 = 0, nm1 = 0;
    float c_maxov = 0.f;
    bool once = a.once && nb[P] <= ENTRY_MAX;
    for (uint32_t g0 = 0; g0 < P;) {
        uint32_t g1 = P;
        if (!once) {
            g1 = g0 + 1u;
            while (g1 < P && nb[g1 + 1u] - nb[g0] <= ITEM_MAX) ++g1;
        }
        const uint32_t base = nb[g0];
        if (tid == 0) s_items = 0u;
        __syncthreads();
        // near candidates and items of particles [g0, g1)
        auto add = [&](uint32_t k, uint32_t what, uint32_t local, uint32_t e) {
            ent[k] = what;
            own[k] = (uint8_t)p;
            if (LIST) slot[k] = (uint8_t)e;
            uint16_t it = NO_ITEM;
            if (!(once && local < p)) {
                const uint32_t i = atomicAdd(&s_items, 1u);
                if (i < ITEM_MAX) {
                    item[i] = (uint16_t)k;
                    it = (uint16_t)i;
                }
            }
            itm[k] = it;
        };
        if (plive && p >= g0 && p < g1) {
            const uint32_t first = nb[p] - base, limit = nb[p + 1u] - base;
            if (LIST) {
                for (uint32_t w = sub; w < 2u; w += G) {
                    uint32_t k = first + (w ? (uint32_t)__popc(near[2 * p]) : 0u);
                    for (uint32_t m = near[2 * p + w]; m; m &= m - 1u, ++k) {
                        const uint32_t e = 32u * w + (uint32_t)__ffs((int)m) - 1u;
                        const uint32_t j = direct ? __ldg(&a.nl[(size_t)e * cap + q0 + p])
                                                  : __ldg((const uint16_t*)(a.nl4 + (size_t)(e >> 2) * cap + q0 + p) +
                                                          (e & 3u));
                        const uint32_t local = direct ? j - q0 : j;
                        add(k, j, local < P ? local : P, e);
                    }
                }
            } else {
                for (uint32_t r = sub; r < 9u; r += G) {
                    uint32_t k = first, j0, j1;
                    for (uint32_t t = 0; t < r; ++t) k += rows[p * 9u + t];
                    if (rows[p * 9u + r] == 0) continue;
                    row(r, j0, j1);
                    for (uint32_t j = j0; j < j1 && k < limit; ++j)
                        if (walk_near(j) && (!exact || touches(j))) {
                            const uint32_t local = j - q0;
                            add(k++, j, local < P ? local : P, 0u);
                        }
                }
            }
        }
        __syncthreads();
        const uint32_t items = s_items;
        if (items > ITEM_MAX) {   // (only with pairs taken once: a round of the other kind fits)
            once = false;
            __syncthreads();
            continue;
        }
        // the items
        for (uint32_t i = tid; i < items; i += ITEM_THREADS) {
            const uint32_t k = item[i], o = own[k];
            const SceneDev& S = a.scenes[LIST ? tile_scene : s_sc[o]];
            const typename PR::Self me = PR::load(A, q0 + o);
            const typename PR::Partner pj = PR::load_partner(A, LIST && !direct ? t_gid[ent[k]] : ent[k]);
            V3<T> n;
            T delta;
            float rj;
            if (!PR::exact_p(A, pj, me, n, delta, rj)) {
                delta_of[i] = -1.f;
                continue;
            }
            delta_of[i] = (float)delta;
            const Law<T> L = law_of(S, a.stiffness, T());
            V3<T> vj, wj;
            PR::partner_vw(pj, vj, wj);
            const V3<T> v = me.v - vj;
            T* r = res + i;
            if (PRACT) {
                // the owner's spring
                V3<T> dold = mk(T(0), T(0), T(0));
                const uint32_t src = s_src[o];
                if (LIST) {
                    const uint32_t e = slot[k], lo = s_om[2 * o], up = s_om[2 * o + 1];
                    const uint32_t word = e < 32u ? lo : up, bit = 1u << (e & 31u);
                    if (word & bit) {
                        const uint32_t h = (uint32_t)__popc(word & (bit - 1u)) + (e < 32u ? 0u : (uint32_t)__popc(lo));
                        const Spring<T> s = load_spring(&hin[h * cap + src]);
                        dold = mk(s.x, s.y, s.z);
                    }
                } else {
                    dold = find_spring(s_pid, P, o, s_cold[o], pj.id, hin, cap, src);
                }
                const T ri = (T)me.r, rjT = (T)rj;
                const V3<T> rw = mk(sym_madd(ri, me.w.x, rjT, wj.x), sym_madd(ri, me.w.y, rjT, wj.y),
                                    sym_madd(ri, me.w.z, rjT, wj.z));
                const T mi = PR::mass(S, me.r), mj = PR::mass(S, rj);
                const T meff = law_div(mi * mj, mi + mj);
                const T Reff = STIFF == 0 ? T(0) : law_div(ri * rjT, ri + rjT);
                V3<T> Fc, Ftc, dnew, Mr;
                law_practical<TERMS, STIFF>(L, n, delta, v, rw, Reff, meff, dold, Fc, Ftc, dnew, me.w - wj, Mr);
                const V3<T> c = cross(n, Ftc);
                r[0] = Fc.x; r[ITEM_MAX] = Fc.y; r[2 * ITEM_MAX] = Fc.z;
                r[3 * ITEM_MAX] = c.x; r[4 * ITEM_MAX] = c.y; r[5 * ITEM_MAX] = c.z;
                r[6 * ITEM_MAX] = dnew.x; r[7 * ITEM_MAX] = dnew.y; r[8 * ITEM_MAX] = dnew.z;
                if (TERMS) { r[9 * ITEM_MAX] = Mr.x; r[10 * ITEM_MAX] = Mr.y; r[11 * ITEM_MAX] = Mr.z; }
            } else {
                const V3<T> Fc = law_simple(L, n, delta, v);
                r[0] = Fc.x; r[ITEM_MAX] = Fc.y; r[2 * ITEM_MAX] = Fc.z;
            }
        }
        __syncthreads();
        // the sums of particles [g0, g1), in the order of their candidates
        if (mine && live && tid >= g0 && tid < g1) {
            const T ri = (T)PR::radius(A, q);
            for (uint32_t k = nb[tid] - base; k < nb[tid + 1u] - base; ++k) {
                const uint32_t what = ent[k];
                uint32_t it = itm[k], pid_at = what;
                T sg = T(1);
                if (it == NO_ITEM) {
                    // evaluated by the partner, in this block: its candidate that is this particle
                    const uint32_t t = LIST && !direct ? what : what - q0;
                    const uint32_t self = LIST && !direct ? tid : q;
                    // (not among them: one of the two prefilters, each of which passes every
                    // contact, says that they do not touch)
                    uint32_t f = nb[t] - base;
                    const uint32_t f1 = nb[t + 1u] - base;
                    while (f < f1 && ent[f] != self) ++f;
                    if (f == f1 || itm[f] == NO_ITEM) continue;
                    it = itm[f];
                    sg = T(-1);
                }
                const float dl = delta_of[it];
                if (!(dl >= 0.f)) continue;
                const T* r = res + it;
                F = axpy(mk(r[0], r[ITEM_MAX], r[2 * ITEM_MAX]), sg, F);
                if (PRACT) {
                    Tq = axpy(mk(r[3 * ITEM_MAX], r[4 * ITEM_MAX], r[5 * ITEM_MAX]), ri, Tq);
                    if (TERMS) Tq = axpy(mk(r[9 * ITEM_MAX], r[10 * ITEM_MAX], r[11 * ITEM_MAX]), sg, Tq);
                }
                if ((PRACT || EVAL) && nnew < maxc) {
                    const uint32_t j = LIST && !direct ? t_gid[pid_at] : pid_at;
                    const V3<T> d = PRACT ? scale(mk(r[6 * ITEM_MAX], r[7 * ITEM_MAX], r[8 * ITEM_MAX]), sg)
                                          : mk(T(0), T(0), T(0));
                    store_spring(&hout[nnew * cap + q], d, __ldg(&A.id[j]));
                    if (LIST) {
                        const uint32_t e = slot[k];
                        if (e < 32u) nm0 |= 1u << e;
                        else nm1 |= 1u << (e - 32u);
                    }
                }
                ++nnew;
                c_maxov = fmaxf(c_maxov, dl);
            }
        }
        __syncthreads();
        g0 = g1;
    }

    // ---- walls (step 8), gravity, update
    uint32_t c_pp = 0, c_wc = 0, c_clamp = 0, c_nnew = 0;
    float c_disp2 = 0.f;
    if (mine && live) {
        const SceneDev& S = a.scenes[s_sc[tid]];
        const typename PR::Self me = PR::load(A, q);
        const Law<T> L = law_of(S, a.stiffness, T());
        const T ri = (T)me.r, mi = PR::mass(S, me.r);
        const uint32_t src = s_src[tid], cold = s_cold[tid];
        c_pp = nnew;
        for (uint32_t wm = LIST ? __ldg(&a.wmask[q]) : (1u << S.nwalls) - 1u; wm; wm &= wm - 1u) {
            const int w = __ffs((int)wm) - 1;
            const WallDev& W = S.walls[w];
            V3<T> n, cp;
            T delta;
            if (!PR::wall(W, me, S, n, delta, cp)) continue;
            const V3<T> v = me.v - PR::wall_vel(W, cp);
            const uint32_t gid = DEM_WALL_BASE + (uint32_t)w;
            if (PRACT) {
                const V3<T> rw = scale(me.w, ri);
                V3<T> dold = mk(T(0), T(0), T(0));
                // (lists: wall springs follow the particles' ones)
                for (uint32_t k = LIST ? (uint32_t)(__popc(s_om[2 * tid]) + __popc(s_om[2 * tid + 1])) : 0u; k < cold; ++k) {
                    const Spring<T> r = load_spring(&hin[k * cap + src]);
                    if (r.pid == gid) dold = mk(r.x, r.y, r.z);
                }
                V3<T> Fc, Ftc, dnew, Mr;
                law_practical<TERMS, STIFF>(L, n, delta, v, rw, ri, mi, dold, Fc, Ftc, dnew, me.w - PR::wall_omega(W), Mr);
                F = add(F, Fc);
                Tq = axpy(cross(n, Ftc), ri, Tq);
                if (TERMS) Tq = add(Tq, Mr);
                if (nnew < maxc) store_spring(&hout[nnew * cap + q], dnew, gid);
            } else {
                F = add(F, law_simple(L, n, delta, v));
                if (EVAL && nnew < maxc) store_spring(&hout[nnew * cap + q], mk(T(0), T(0), T(0)), gid);
            }
            ++nnew;
            ++c_wc;
            c_maxov = fmaxf(c_maxov, (float)delta);
        }
        if (nnew > maxc) {
            raise_status(a.st, ST_CAPACITY, (int32_t)q);
            if (!EVAL && a.halt) atomicOr(&s_flag, DEM_HALT);
        }
        c_nnew = nnew;
        if (PRACT || EVAL) hout_cnt[q] = min(nnew, maxc);
        if (LIST && PRACT && !EVAL) *(uint2*)&(ho ? a.hmask[1] : a.hmask[0])[q] = make_uint2(nm0, nm1);
        {
            const T gx = sizeof(T) == 8 ? (T)S.g[0] : (T)S.g_f[0];
            const T gy = sizeof(T) == 8 ? (T)S.g[1] : (T)S.g_f[1];
            const T gz = sizeof(T) == 8 ? (T)S.g[2] : (T)S.g_f[2];
            F = axpy(mk(gx, gy, gz), mi, F);
        }
        if (EVAL) {
            const size_t o = 3 * (size_t)me.id;
            if (a.dbgF) { a.dbgF[o] = F.x; a.dbgF[o + 1] = F.y; a.dbgF[o + 2] = F.z; }
            if (a.dbgT) { a.dbgT[o] = Tq.x; a.dbgT[o + 1] = Tq.y; a.dbgT[o + 2] = Tq.z; }
        } else {
            bool clamped = false, finite = true;
            float4 pnew;
            const uint32_t kk = PR::template integrate<!LIST>(B, q, me, F, Tq, S, mi, clamped, finite, pnew);
            if (!finite) raise_status(a.st, ST_NONFINITE, (int32_t)q);
            c_clamp = clamped ? 1u : 0u;
            c_disp2 = pnew.w;
            if (LIST) {
                const float4 r0 = __ldg(&a.ref[q]);
                const float ex = pnew.x - r0.x, ey = pnew.y - r0.y, ez = pnew.z - r0.z;
                if (ex * ex + ey * ey + ez * ez > S.thresh2_f || !finite) atomicOr(&s_flag, 1u);
            } else {
                a.key[q] = kk;
                a.rank[q] = atomicAdd(&a.cnt[kk], 1u);
            }
        }
    }
    const uint32_t w_pp = __reduce_add_sync(full, c_pp);
    const uint32_t w_wc = __reduce_add_sync(full, c_wc);
    const uint32_t w_cl = __reduce_add_sync(full, c_clamp);
    const uint32_t w_mx = __reduce_max_sync(full, c_nnew);
    const uint32_t w_ov = __reduce_max_sync(full, __float_as_uint(c_maxov));
    const uint32_t w_dp = __reduce_max_sync(full, __float_as_uint(c_disp2));
    if (lane == 0) {
        if (w_pp) atomicAdd(&s_sum[0], w_pp);
        if (w_wc) atomicAdd(&s_sum[1], w_wc);
        if (w_cl) atomicAdd(&s_sum[2], w_cl);
        if (w_mx) atomicMax(&s_max[0], w_mx);
        if (w_ov) atomicMax(&s_max[1], w_ov);
        if (w_dp) atomicMax(&s_max[2], w_dp);
    }
    __syncthreads();
    if (tid == 0) {
        if (s_sum[0]) atomicAdd(&a.st->live.ncontacts, s_sum[0]);
        if (s_sum[1]) atomicAdd(&a.st->live.nwallc, s_sum[1]);
        if (s_sum[2]) atomicAdd(&a.st->live.clamped, s_sum[2]);
        if (s_max[0]) atomicMax(&a.st->live.max_nnew, s_max[0]);
        if (s_max[1]) atomicMax(&a.st->live.max_overlap_bits, s_max[1]);
        if (s_max[2]) atomicMax(&a.st->live.max_disp2_bits, s_max[2]);
        if (s_flag) atomicOr(&a.ctrl->rebuild, (int)s_flag);
    }
}

// ======================================================================= launchers
template <class PR, bool LIST>
static cudaError_t items_impl(Domain& d, const typename PR::State& S0, const typename PR::State& S1, uint32_t P, bool eval,
                              double* dbgF, double* dbgT) {
    using T = typename PR::T;
    ItemArgs<PR> a{};
    a.scenes = d.d_scenes;
    a.nscenes = d.nscenes;
    a.n = d.n;
    a.cap = d.cap;
    a.tile = P;
    a.hcap = LIST ? halo_cap(P) : 0u;
    a.maxc = d.maxc;
    a.stiffness = d.stiffness;
    a.S0 = S0;
    a.S1 = S1;
    a.ctrl = d.ctrl;
    a.ncnt = d.ncnt;
    a.nl = d.nl;
    a.nl4 = d.nl4;
    a.halo = d.halo;
    a.nhalo = d.nhalo;
    a.ref = d.ref;
    a.interval = d.interval;
    a.wmask = d.wmask;
    a.loop = d.in_loop;
    a.skey = d.skey;
    a.cs = d.cs;
    a.key = d.key;
    a.rank = d.rank;
    a.cnt = d.cnt;
    a.perm = d.perm;
    for (int k = 0; k < 2; ++k) {
        a.hcnt[k] = d.hcnt[k];
        a.hs[k] = (Spring<T>*)d.hs[k];
        a.hmask[k] = d.hmask[k];
    }
    a.hin = d.h_cur;
    a.st = d.st;
    a.dbgF = dbgF;
    a.dbgT = dbgT;
    a.halt = d.regrow;
    a.once = d.both_springs;
    const uint32_t grid = LIST ? d.ntiles : (d.n + P - 1) / P;
    auto launch = [&](auto kern, uint32_t smem) -> cudaError_t {
        if (smem > 32 * 1024) {   // (with the static shared memory above the default limit)
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        kern<<<grid, ITEM_THREADS, smem, d.stream>>>(a);
        return cudaSuccess;
    };
    const uint32_t mc = (uint32_t)d.maxc;
    const int model = d.model != 0 ? 1 : (d.terms != 0 ? 2 : (d.stiffness != 0 ? 3 : 0));
    cudaError_t e;
#define DEM_ITEMS(MODEL)                                                                              \
    (eval ? launch(k_items<PR, LIST, MODEL, true>, ItemMem<PR, LIST, MODEL>(P, a.hcap, mc).total)     \
          : launch(k_items<PR, LIST, MODEL, false>, ItemMem<PR, LIST, MODEL>(P, a.hcap, mc).total))
    if (model == 0) e = DEM_ITEMS(0);
    else if (model == 1) e = DEM_ITEMS(1);
    else if (model == 2) e = DEM_ITEMS(2);
    else e = DEM_ITEMS(3);
#undef DEM_ITEMS
    if (e != cudaSuccess) return e;
    ++d.launches;
    return cudaGetLastError();
}

// Particles per block of the walk by items: 128, and less for few particles, so that the
// blocks reach every SM.
static uint32_t walk_tile(const Domain& d) {
    uint32_t P = 128;
    while (P > 16 && d.n / P < (uint32_t)(d.sort_blocks / 8)) P /= 2;
    return P;
}

cudaError_t run_force_items(Domain& d, bool eval, double* dbgF, double* dbgT) {
    if (d.n == 0) return cudaSuccess;
    if (d.list_mode) return items_impl<PF64, true>(d, d.S64[0], d.S64[1], d.tile, eval, dbgF, dbgT);
    return d.precision == 0 ? items_impl<PF64, false>(d, d.S64[0], d.S64[1], walk_tile(d), eval, dbgF, dbgT)
                            : items_impl<PF32, false>(d, d.S32[0], d.S32[1], walk_tile(d), eval, dbgF, dbgT);
}

}  // namespace demgb
