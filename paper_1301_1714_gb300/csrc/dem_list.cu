// List mode (re-sort only after some particle moved skin/2): the force pass over the
// neighbour lists built at each sort (the lists and tiles themselves: dem_nlist.cu), FP32
// mode (FP64: dem_items.cu).
//
//   k_list   steps 5-8 and 1 for one thread block per tile of consecutive stored particles,
//            one thread per particle. The tile's particles and its halo (the particles
//            outside it that are on some list of the tile, found at the sort) are copied
//            to shared memory; phase 1 keeps the list entries that pass the contact
//            prefilter as a 64-bit mask; phase 2 takes them one after another (contact
//            decision, Eq. 1 or Eqs. 2-10, the spring); then the walls the last sort found
//            within reach (step 8), gravity, the update (step 1) and the displacement test
//            that decides whether this step ends with a sort.
//
// Every particle evaluates all of its contacts (each pair twice, once from each side, with
// arithmetic that makes the two results exact negatives), so a step is one pass with no
// exchange between particles; springs are stored per particle in list order, and a 64-bit
// mask per particle says which list entries have one, so that a contact finds its spring by
// counting bits. No floating-point atomics: a particle's sums run in list order (ascending
// partner id), so results depend neither on the tile size nor on when the sorts happened.
#include <algorithm>

#include <cuda_runtime.h>

#include "dem_domain.h"
#include "dem_policy.cuh"

namespace demgb {

using PR = PF32;
using T = float;

struct ListArgs {
    const SceneDev* scenes;
    int nscenes;
    uint32_t cap, tile, hcap;
    int maxc, stiffness;
    StateF32 S0, S1;             // the two state sets; ctrl->cur names the current one
    CtrlDev* ctrl;
    const uint32_t* ncnt;        // list lengths
    const uint32_t* nl;          // list entries (stored index), slot-major
    const uint2* nl4;            // the same as tile entries, four 16-bit indices per element
    const uint32_t* halo;        // hcap stored indices per tile
    const uint32_t* nhalo;       // how many of them; HALO_NONE: the tile has no entry indices
    const float4* ref;           // positions at the last sort
    int interval;                // sort at least every `interval` steps (0: never forced)
    const uint32_t* perm;
    const uint32_t* wmask;       // walls each particle can reach until the next sort
    uint32_t* hcnt[2];           // springs: ctrl->hcur names the buffer read, the other is written
    Spring<T>* hs[2];
    uint64_t* hmask[2];          // list entries that have a spring
    StatusDev* st;
    double* dbgF;
    double* dbgT;
    int halt;                    // 1: a capacity overflow makes the step void (DEM_HALT)
    int loop;                    // 1: a pass of the step loop, idle unless ctrl->stop says go
};

// ------------------------------------------------------------------- force pass

// MODEL: 0 the practical law with linear stiffness, 1 the simple law (Eq. 1), 2 the practical
// law with the scene's optional terms, 3 the practical law with Hertz stiffness (the paper's
// two stiffnesses have a variant each: the other's constants would take registers).
// EVAL: forces and torques by id instead of the update.
template <int MODEL, bool EVAL>
__global__ void __launch_bounds__(PR::LIST_THREADS, PR::LIST_BLOCKS) k_list(ListArgs a) {
    constexpr bool PRACT = MODEL != 1;
    constexpr bool TERMS = MODEL == 2;
    constexpr int STIFF = MODEL == 2 ? 2 : (MODEL == 3 ? 1 : 0);
    const unsigned full = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char t_mem[];
    __shared__ uint32_t s_sum[3], s_max[3], s_flag;   // counters of the block; bits for ctrl->rebuild
    __shared__ int s_void;
    __shared__ __align__(16) unsigned char s_law[64];
    if (!EVAL && a.loop && a.ctrl->stop != LOOP_GO) return;   // (written between passes only)
    const uint32_t tid = threadIdx.x, lane = tid & 31u;
    if (tid == 0) s_void = a.ctrl->rebuild & DEM_HALT;
    if (tid < 3) s_sum[tid] = s_max[tid] = 0u;
    if (tid == 3) s_flag = 0u;
    __syncthreads();
    if (!EVAL && s_void) return;   // an earlier launch (or another block) overflowed: a void step
    const int cur = a.ctrl->cur;
    const StateF32 A = cur ? a.S1 : a.S0;
    const StateF32 B = cur ? a.S0 : a.S1;
    const bool pv = a.ctrl->perm_valid != 0;
    const int hi = a.ctrl->hcur, ho = 1 - hi;
    if (!EVAL && blockIdx.x == 0 && tid == 0) {
        a.ctrl->hlast = ho;
        if (a.interval > 0 && a.ctrl->since + 1 >= a.interval) atomicOr(&a.ctrl->rebuild, 1);
    }
    const Spring<T>* __restrict__ hin = hi ? a.hs[1] : a.hs[0];
    uint32_t* __restrict__ hout_cnt = ho ? a.hcnt[1] : a.hcnt[0];
    Spring<T>* __restrict__ hout = ho ? a.hs[1] : a.hs[0];
    uint64_t* __restrict__ mout = ho ? a.hmask[1] : a.hmask[0];
    const uint32_t maxc = (uint32_t)a.maxc, E = a.tile + a.hcap;
    const size_t cap = a.cap;
    const SceneDev& S = a.scenes[scene_of_tile(a.scenes, a.nscenes, blockIdx.x)];
    const uint32_t off = (blockIdx.x - S.t0) * a.tile;
    const uint32_t q = S.p0 + off + tid;
    const bool valid = off + tid < S.np;
    uint32_t src = 0, cnt_old = 0, m = 0;
    uint32_t om_lo = 0, om_hi = 0;   // list entries that have a stored spring
    if (valid) {
        src = pv ? __ldg(&a.perm[q]) : q;
        if (PRACT || !S.active) {
            cnt_old = min(__ldg(&(hi ? a.hcnt[1] : a.hcnt[0])[src]), maxc);
            const uint2 u = __ldg((const uint2*)&(hi ? a.hmask[1] : a.hmask[0])[q]);
            om_lo = u.x;
            om_hi = u.y;
        }
    }
    if (!S.active) {
        // frozen scene: carry state and springs unchanged
        if (!valid) return;
        if (!EVAL) {
            PR::store(B, q, PR::load(A, q));
            for (uint32_t k = 0; k < cnt_old; ++k) hout[k * cap + q] = hin[k * cap + src];
            hout_cnt[q] = cnt_old;
            *(uint2*)&mout[q] = make_uint2(om_lo, om_hi);
        } else {
            hout_cnt[q] = 0;
        }
        return;
    }
    // ---- the tile and its halo into shared memory
    const uint32_t nh = __ldg(&a.nhalo[blockIdx.x]);
    const bool direct = nh == HALO_NONE;   // (more halo than fits: partners are read from global memory)
    if (valid) {
        m = min(__ldg(&a.ncnt[q]), (uint32_t)DEM_LIST_CAP);
        PR::tile_fetch(A, q, t_mem, E, tid);
        if (!direct) {
            // the list and the stored springs stream from DRAM: start their line fills now
            for (uint32_t k = 0; k < m; k += 4) prefetch_l1(&a.nl4[(size_t)(k >> 2) * cap + q]);
        }
        for (uint32_t k = 0; k < cnt_old; ++k) prefetch_l1(&hin[k * cap + src]);
    }
    if (!direct) {
        const uint32_t* __restrict__ halo = a.halo + (size_t)blockIdx.x * a.hcap;
        for (uint32_t k = tid; k < nh; k += blockDim.x) PR::tile_fetch(A, __ldg(&halo[k]), t_mem, E, a.tile + k);
    }
    if (tid == 0) PR::put_law(law_of(S, a.stiffness, T()), s_law);
    copies_done();
    __syncthreads();
    uint32_t c_pp = 0, c_wc = 0, c_clamp = 0, c_nnew = 0;
    float c_maxov = 0.f, c_disp2 = 0.f;
    if (valid) {
        const PR::Self me = PR::tile_self(A, q, t_mem, E, tid);
        // ---- phase 1: list entries that pass the prefilter (near[0]: entries 0-31, near[1]: 32-63)
        uint32_t near0 = 0, near1 = 0;
        {
            const float4 p = PR::pre(me);
            const float eps = PR::pre_eps(S, p);
            if (!direct) {
                const uint2* lp = a.nl4 + q;
                const float4* t4 = (const float4*)t_mem;
                for (uint32_t k = 0; k < m; k += 4, lp += cap) {
                    const uint2 u = __ldg(lp);
                    uint32_t b = near_f(p, t4[u.x & 0xffffu], eps) ? 1u : 0u;
                    b |= near_f(p, t4[u.x >> 16], eps) ? 2u : 0u;
                    b |= near_f(p, t4[u.y & 0xffffu], eps) ? 4u : 0u;
                    b |= near_f(p, t4[u.y >> 16], eps) ? 8u : 0u;
                    if (k < 32) near0 |= b << k;
                    else near1 |= b << (k - 32);
                }
                // (the last element is padded)
                if (m < 32) near0 &= (1u << m) - 1u;
                else if (m < 64) near1 &= (1u << (m - 32)) - 1u;
            } else {
                for (uint32_t k = 0; k < m; ++k)
                    if (near_f(p, PR::pre(A, __ldg(&a.nl[k * cap + q])), eps)) {
                        if (k < 32) near0 |= 1u << k;
                        else near1 |= 1u << (k - 32);
                    }
            }
        }
        // ---- phase 2: the near candidates, in list order
        const Law<T> L = law_of(S, a.stiffness, T());
        const T mi = PR::mass(S, me.r);
        const T ri = (T)me.r;
        V3<T> F = mk(T(0), T(0), T(0)), Tq = mk(T(0), T(0), T(0));
        uint32_t nnew = 0;
        uint32_t om = om_lo, nm = 0, nm_lo = 0;
        const Spring<T>* hp = hin + src;   // slots of the mask word's springs start here
        Spring<T>* op = hout + q;
        uint32_t e0 = 0;
        for (;;) {
            if (near0 == 0) {
                // the upper mask word (a list of more than 32 entries)
                if (e0 != 0 || near1 == 0) break;
                e0 = 32;
                near0 = near1;
                hp += (size_t)__popc(om_lo) * cap;
                om = om_hi;
                nm_lo = nm;
                nm = 0;
            }
            const uint32_t e = (uint32_t)__ffs((int)near0) - 1u;
            const uint32_t bit = 1u << e;
            near0 &= near0 - 1u;
            PR::Partner pj;
            if (!direct)
                pj = PR::tile_partner(
                    A, t_mem, E, __ldg((const uint16_t*)(a.nl4 + (size_t)((e0 + e) >> 2) * cap + q) + (e & 3u)));
            else
                pj = PR::load_partner(A, __ldg(&a.nl[(size_t)(e0 + e) * cap + q]));
            V3<T> n;
            T delta;
            float rj;
            if (!PR::exact_p(A, pj, me, n, delta, rj)) continue;
            V3<T> vj, wj;
            PR::partner_vw(pj, vj, wj);
            const V3<T> v = PR::self_v(me, t_mem, E, tid) - vj;
            const Law<T> Lc = PR::law(L, s_law);
            if (PRACT) {
                const V3<T> wi = PR::self_w(me, t_mem, E, tid);
                V3<T> dold = mk(T(0), T(0), T(0));
                if (om & bit) {
                    const Spring<T> r = load_spring(hp + (size_t)__popc(om & (bit - 1u)) * cap);
                    dold = mk(r.x, r.y, r.z);
                }
                const T rjT = (T)rj;
                const V3<T> rw = mk(sym_madd(ri, wi.x, rjT, wj.x), sym_madd(ri, wi.y, rjT, wj.y),
                                    sym_madd(ri, wi.z, rjT, wj.z));
                const T mj = PR::mass(S, rj);
                const T meff = law_div(mi * mj, mi + mj);
                const T Reff = (STIFF == 0) ? T(0) : law_div(ri * rjT, ri + rjT);
                V3<T> Fc, Ftc, dnew, Mr;
                law_practical<TERMS, STIFF>(Lc, n, delta, v, rw, Reff, meff, dold, Fc, Ftc, dnew, wi - wj, Mr);
                F = add(F, Fc);
                Tq = axpy(cross(n, Ftc), ri, Tq);
                if (TERMS) Tq = add(Tq, Mr);
                if (nnew < maxc) {
                    store_spring(op, dnew, pj.id);
                    op += cap;
                    nm |= bit;
                }
            } else {
                F = add(F, law_simple(Lc, n, delta, v));
                if (EVAL && nnew < maxc) {
                    store_spring(op, mk(T(0), T(0), T(0)), pj.id);
                    op += cap;
                }
            }
            ++nnew;
            c_maxov = fmaxf(c_maxov, (float)delta);
        }
        c_pp = nnew;
        const PR::Self me2 = PR::tile_again(me, t_mem, E, tid);
        // ---- walls (step 8), those the last sort found within reach; their springs follow
        // the particles' ones
        const uint32_t w_first = (uint32_t)(__popc(om_lo) + __popc(om_hi));
        for (uint32_t wm = __ldg(&a.wmask[q]); wm; wm &= wm - 1) {
            const int w = __ffs(wm) - 1;
            const WallDev& W = S.walls[w];
            V3<T> n, cp;
            T delta;
            if (!PR::wall(W, me2, S, n, delta, cp)) continue;
            const V3<T> v = me2.v - PR::wall_vel(W, cp);
            const uint32_t gid = DEM_WALL_BASE + (uint32_t)w;
            if (PRACT) {
                const V3<T> rw = scale(me2.w, ri);
                V3<T> dold = mk(T(0), T(0), T(0));
                for (uint32_t k = w_first; k < cnt_old; ++k) {
                    const Spring<T> r = load_spring(&hin[k * cap + src]);
                    if (r.pid == gid) dold = mk(r.x, r.y, r.z);
                }
                V3<T> Fc, Ftc, dnew, Mr;
                law_practical<TERMS, STIFF>(L, n, delta, v, rw, ri, mi, dold, Fc, Ftc, dnew, me2.w - PR::wall_omega(W), Mr);
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
        if (PRACT && !EVAL) *(uint2*)&mout[q] = e0 ? make_uint2(nm_lo, nm) : make_uint2(nm, 0u);
        // gravity, once per particle
        {
            F = axpy(mk(S.g_f[0], S.g_f[1], S.g_f[2]), mi, F);
        }
        if (EVAL) {
            const size_t o = 3 * (size_t)me2.id;
            if (a.dbgF) { a.dbgF[o] = F.x; a.dbgF[o + 1] = F.y; a.dbgF[o + 2] = F.z; }
            if (a.dbgT) { a.dbgT[o] = Tq.x; a.dbgT[o + 1] = Tq.y; a.dbgT[o + 2] = Tq.z; }
        } else {
            bool clamped = false, finite = true;
            float4 pnew;
            PR::integrate<false>(B, q, me2, F, Tq, S, mi, clamped, finite, pnew);
            if (!finite) raise_status(a.st, ST_NONFINITE, (int32_t)q);
            c_clamp = clamped ? 1u : 0u;
            c_disp2 = pnew.w;
            // a particle that moved skin/2 (less the FP32 margin) since the last sort makes
            // this step end with a sort and new lists
            const float4 r0 = __ldg(&a.ref[q]);
            const float ex = pnew.x - r0.x, ey = pnew.y - r0.y, ez = pnew.z - r0.z;
            if (ex * ex + ey * ey + ez * ez > S.thresh2_f || !finite) atomicOr(&s_flag, 1u);
        }
    }
    // counters of the block (every thread reaches this point): one global atomic per counter
    // and block; one per warp meant 131,072 x 5 atomics on one 32-byte sector for the drum
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
#define DEM_LAUNCH_CHECK()                          \
    do {                                            \
        ++d.launches;                               \
        cudaError_t e_ = cudaGetLastError();        \
        if (e_ != cudaSuccess) return e_;           \
    } while (0)

cudaError_t run_force_list(Domain& d, bool eval, double* dbgF, double* dbgT) {
    if (d.n == 0) return cudaSuccess;
    ListArgs a;
    a.scenes = d.d_scenes;
    a.nscenes = d.nscenes;
    a.cap = d.cap;
    a.tile = d.tile;
    a.hcap = halo_cap(d.tile);
    a.maxc = d.maxc;
    a.stiffness = d.stiffness;
    a.S0 = d.S32[0];
    a.S1 = d.S32[1];
    a.ctrl = d.ctrl;
    a.ncnt = d.ncnt;
    a.nl = d.nl;
    a.nl4 = d.nl4;
    a.halo = d.halo;
    a.nhalo = d.nhalo;
    a.ref = d.ref;
    a.interval = d.interval;
    a.perm = d.perm;
    a.wmask = d.wmask;
    for (int k = 0; k < 2; ++k) {
        a.hcnt[k] = d.hcnt[k];
        a.hs[k] = (Spring<T>*)d.hs[k];
        a.hmask[k] = d.hmask[k];
    }
    a.st = d.st;
    a.dbgF = dbgF;
    a.dbgT = dbgT;
    a.halt = d.regrow;
    a.loop = d.in_loop;
    const size_t smem = (size_t)(a.tile + a.hcap) * PR::TILE_BYTES;
    const int model = d.model != 0 ? 1 : (d.terms != 0 ? 2 : (d.stiffness != 0 ? 3 : 0));
    auto launch = [&](auto kern) -> cudaError_t {
        if (smem > 32 * 1024) {   // (with the static shared memory above the default limit)
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        kern<<<d.ntiles, d.tile, smem, d.stream>>>(a);
        return cudaSuccess;
    };
    cudaError_t e;
    if (model == 0) e = eval ? launch(k_list<0, true>) : launch(k_list<0, false>);
    else if (model == 2) e = eval ? launch(k_list<2, true>) : launch(k_list<2, false>);
    else if (model == 3) e = eval ? launch(k_list<3, true>) : launch(k_list<3, false>);
    else e = eval ? launch(k_list<1, true>) : launch(k_list<1, false>);
    if (e != cudaSuccess) return e;
    DEM_LAUNCH_CHECK();
    return cudaSuccess;
}

}  // namespace demgb
