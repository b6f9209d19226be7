// List mode: the neighbour lists of a sort (Eq. 12's 27 cells, candidates within
// r_i + r_j + skin, in ascending partner id) and the walls each particle can reach before
// the next sort, and the tiles. The force passes that read them: dem_list.cu (FP32),
// dem_items.cu (FP64).
#include <algorithm>

#include <cuda_runtime.h>

#include "dem_domain.h"
#include "dem_policy.cuh"

namespace demgb {

// ------------------------------------------------------------------ list build
// Walls the particle can touch before the next sort: walls do not move (their velocity
// only enters the contact law), and a particle moves less than skin/2 between sorts, so
// every wall within r + skin/2 (+ the FP32 margin) of it now; bit w marks wall w.
// The test is a conservative FP32 distance (to a plane, from a cylinder's axis, from a
// half-plate's plane) with four times the FP32 position margin.
template <class PR>
__device__ __forceinline__ uint32_t reachable_walls(const typename PR::Self& me, const SceneDev& S) {
    const float4 x = PR::pos_f(me);
    const float eps = 4.f * S.eps_f;
    const float reach = me.r + 0.5f * S.skin_f + eps;
    uint32_t m = 0;
    for (int w = 0; w < S.nwalls; ++w) {
        const WallDev& W = S.walls[w];
        const float qx = x.x - W.pf[0], qy = x.y - W.pf[1], qz = x.z - W.pf[2];
        const float h = W.nf[0] * qx + W.nf[1] * qy + W.nf[2] * qz;
        bool near;
        if (W.kind == 1) {
            // distance from the axis (through p along n) against the radius
            const float rho2 = fmaxf(qx * qx + qy * qy + qz * qz - h * h, 0.f);
            const float lim = W.rad_hi - reach - eps;
            near = !(lim > 0.f && rho2 <= lim * lim);
        } else if (W.kind == 0) {
            near = h < reach;                 // signed distance into the domain
        } else {
            near = fabsf(h) < reach;          // either face of a half-plate, wherever its edge is
        }
        if (near) m |= 1u << w;
    }
    return m;
}

template <class PR>
__global__ void __launch_bounds__(256) k_wall_masks(uint32_t n, const SceneDev* scenes, int nscenes,
                                                    typename PR::State S0, typename PR::State S1, const CtrlDev* ctrl,
                                                    uint32_t* __restrict__ wmask) {
    const typename PR::State A = ctrl->cur ? S1 : S0;
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x)
        wmask[q] = reachable_walls<PR>(PR::load(A, q), scenes[scene_of(scenes, nscenes, q)]);
}

// Candidates of particle q at a sort: every particle of the 27 cells around q's cell
// (Eq. 12; list mode numbers the cells brick by brick, so each cell is looked up on its
// own) within r_i + r_j + skin (+ the FP32 margin), the skin of q's scene. With cells of
// edge >= 2 r_max + skin no pair that comes into contact before some particle has moved
// skin/2 is missed. A list is kept in ascending partner id, so the force pass sums a
// particle's contacts in that order whenever the list was built: results do not depend on
// when sorts happen (a batch sorts all its scenes together, and each scene still gets the
// bits of its own run). A list longer than DEM_LIST_CAP is reported (the step returns
// DEM_ERR_CAPACITY).
//
// One warp per cell: the particles of a cell have the same 27 cells around them, so the
// lanes look the cells up together (one each), number the candidates through by a scan of
// the counts, read up to NLIST_REGS x 32 of them into registers once, and test all 32 lanes'
// candidates against one particle of the cell at a time; the accepted ones are ranked by id
// in shared memory. (One thread per particle walked 27 x 0-5 candidates with its neighbours
// in the warp on other cells, and sorted its list by insertion in local memory: 2.9 ms per
// sort of the 4,194,304-sphere bed at 59 candidates and 10 list entries per particle, 1.6 now.)
// A warp takes `per` consecutive positions: 32, and less for few particles, whose warps would
// otherwise walk their 10 to 16 cells one after another with most of the chip idle (9,217
// spheres: 49.8 us with 32, 15.0 with 4; 500: 43.2 and 13.3).
constexpr int NLIST_REGS = 3;

template <class PR>
__global__ void __launch_bounds__(256) k_nlist(uint32_t n, uint32_t per, const SceneDev* __restrict__ scenes, int nscenes, typename PR::State S0,
                                               typename PR::State S1, const CtrlDev* ctrl,
                                               const uint32_t* __restrict__ key, const uint32_t* __restrict__ canon,
                                               const uint32_t* __restrict__ cs, const uint32_t* __restrict__ fin,
                                               uint32_t* __restrict__ ncnt, uint32_t* __restrict__ nl, size_t cap,
                                               uint32_t* __restrict__ wmask, StatusDev* st) {
    if (ctrl->rebuild != 1) return;   // no sort this step (or a void step)
    const unsigned full = 0xffffffffu;
    __shared__ uint32_t s_idx[8][DEM_LIST_CAP], s_id[8][DEM_LIST_CAP];
    const typename PR::State A = ctrl->cur ? S1 : S0;
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t* acc = s_idx[wid];
    uint32_t* aid = s_id[wid];
    // the lane's cell of the 27 (lanes 27-31: none)
    const int dx = (int)(lane % 3u) - 1, dy = (int)((lane / 3u) % 3u) - 1, dz = (int)(lane / 9u) - 1;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    for (uint32_t base = (blockIdx.x * (blockDim.x >> 5) + wid) * per; base < n; base += warps * per) {
        // `per` (cell, id) positions: stored position, cell and FP32 position of each
        const uint32_t s = base + lane;
        const bool valid = lane < per && s < n;
        uint32_t q = 0, kk = 0xFFFFFFFFu;
        int sidx = 0, ix = 0, iy = 0, iz = 0;
        float4 p = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
            q = fin[s];
            kk = key[canon[s]];
            sidx = scene_of(scenes, nscenes, s);
            const SceneDev& S = scenes[sidx];
            cell_coords(S, kk - S.c0, ix, iy, iz);
            const typename PR::Self me = PR::load(A, q);
            p = PR::pre(me);
            wmask[q] = reachable_walls<PR>(me, S);
        }
        const uint32_t before = __shfl_up_sync(full, kk, 1);
        uint32_t runs = __ballot_sync(full, valid && (lane == 0 || before != kk));   // first of each cell
        const uint32_t nvalid = (uint32_t)__popc(__ballot_sync(full, valid));
        while (runs) {
            const int a = __ffs((int)runs) - 1;
            runs &= runs - 1u;
            const int b = runs ? __ffs((int)runs) - 1 : (int)nvalid;
            const SceneDev& S = scenes[__shfl_sync(full, sidx, a)];
            const int cx = __shfl_sync(full, ix, a) + dx, cy = __shfl_sync(full, iy, a) + dy,
                      cz = __shfl_sync(full, iz, a) + dz;
            uint32_t first = 0, cnt = 0;
            if (lane < 27u && cx >= 0 && cy >= 0 && cz >= 0 && cx < S.dims[0] && cy < S.dims[1] && cz < S.dims[2]) {
                const uint32_t c = S.c0 + cell_index(S, (uint32_t)cx, (uint32_t)cy, (uint32_t)cz);
                first = __ldg(&cs[c]);
                cnt = __ldg(&cs[c + 1]) - first;
            }
            uint32_t upto = cnt;   // candidates of this lane's cell and the ones before it
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(full, upto, o);
                if (lane >= (uint32_t)o) upto += t;
            }
            const uint32_t total = __shfl_sync(full, upto, 31);
            const float extra = S.skin_f + S.eps_f;
            // candidate k of the 27 cells: its stored index (or none)
            auto candidate = [&](uint32_t k) -> uint32_t {
                uint32_t c = 0;
#pragma unroll
                for (uint32_t o = 16; o; o >>= 1) {
                    const uint32_t t = __shfl_sync(full, upto, c + o - 1u);
                    if (t <= k) c += o;
                }
                c = min(c, 31u);
                const uint32_t f = __shfl_sync(full, first, c), u = __shfl_sync(full, upto - cnt, c);
                return k < total ? fin[f + (k - u)] : 0xFFFFFFFFu;
            };
            uint32_t jr[NLIST_REGS];
            float4 pr[NLIST_REGS];
#pragma unroll
            for (int r = 0; r < NLIST_REGS; ++r) {
                jr[r] = 0xFFFFFFFFu;
                pr[r] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (r * 32u < total) {
                    jr[r] = candidate(r * 32u + lane);
                    if (jr[r] != 0xFFFFFFFFu) pr[r] = PR::pre(A, jr[r]);
                }
            }
            for (int i = a; i < b; ++i) {
                const uint32_t qi = __shfl_sync(full, q, i);
                const float4 pi = make_float4(__shfl_sync(full, p.x, i), __shfl_sync(full, p.y, i),
                                              __shfl_sync(full, p.z, i), __shfl_sync(full, p.w, i));
                uint32_t m = 0;
                auto take = [&](uint32_t j, float4 pj) {
                    const bool in = j != 0xFFFFFFFFu && j != qi && near_f(pi, pj, extra);
                    const uint32_t bl = __ballot_sync(full, in);
                    const uint32_t at = m + (uint32_t)__popc(bl & lt);
                    if (in && at < DEM_LIST_CAP) acc[at] = j;
                    m += (uint32_t)__popc(bl);
                };
#pragma unroll
                for (int r = 0; r < NLIST_REGS; ++r)
                    if (r * 32u < total) take(jr[r], pr[r]);
                for (uint32_t k0 = NLIST_REGS * 32u; k0 < total; k0 += 32u) {
                    const uint32_t j = candidate(k0 + lane);
                    take(j, j != 0xFFFFFFFFu ? PR::pre(A, j) : make_float4(0.f, 0.f, 0.f, 0.f));
                }
                __syncwarp();
                const uint32_t mm = min(m, (uint32_t)DEM_LIST_CAP);
                for (uint32_t k = lane; k < mm; k += 32u) aid[k] = __ldg(&A.id[acc[k]]);
                __syncwarp();
                for (uint32_t k = lane; k < mm; k += 32u) {
                    const uint32_t id = aid[k];
                    uint32_t r = 0;
                    for (uint32_t t = 0; t < mm; ++t) r += aid[t] < id ? 1u : 0u;
                    nl[(size_t)r * cap + qi] = acc[k];
                }
                if (lane == 0) {
                    ncnt[qi] = mm;
                    if (m > DEM_LIST_CAP) raise_status(st, ST_LIST, (int32_t)qi);
                }
                __syncwarp();   // (the buffers are filled again by the next particle)
            }
        }
    }
}

// ------------------------------------------------------------------ tiles
// A tile is `tile` consecutive stored particles of one scene (the last of a scene may hold
// fewer): the work of one block of the force pass, which keeps the tile and its halo in
// shared memory. One block here per tile: the stored indices outside the tile that occur on
// its lists are collected in a hash table in shared memory, sorted (the force pass then
// copies them in nearly coalesced runs), and every list entry is rewritten as a 16-bit index
// into (tile, halo). A tile whose halo does not fit is marked HALO_NONE. The same pass marks
// the list entries that have a stored spring: a particle's springs and its list are both in
// ascending partner id, so it is a merge. A spring whose partner is not on the new list (the pair
// has moved apart by more than the skin, or the springs were set from outside) moves behind the
// wall springs: no contact reads it there, and it is still part of the history.
constexpr uint32_t TILE_HASH = 2048;   // entries: a tile inserts at most halo_cap + 512 before it stops
constexpr uint32_t TILE_SORT = 1024;   // >= halo_cap, power of two

template <class T>
__device__ __forceinline__ void swap_springs(Spring<T>* h, size_t a, size_t b) {
    const Spring<T> t = h[a];
    h[a] = h[b];
    h[b] = t;
}

template <class PR>
__global__ void __launch_bounds__(512) k_tile(const SceneDev* scenes, int nscenes, uint32_t tile, uint32_t ntiles,
                                              uint32_t hcap, typename PR::State S0, typename PR::State S1,
                                              const CtrlDev* ctrl, int always, const uint32_t* __restrict__ ncnt,
                                              const uint32_t* __restrict__ nl, uint2* __restrict__ nl4,
                                              uint32_t* __restrict__ halo, uint32_t* __restrict__ nhalo, size_t cap,
                                              const uint32_t* __restrict__ perm, const uint32_t* hcnt0, const uint32_t* hcnt1,
                                              Spring<typename PR::T>* hs0, Spring<typename PR::T>* hs1, uint64_t* hm0,
                                              uint64_t* hm1, uint32_t maxc) {
    if (!always && ctrl->rebuild != 1) return;   // no sort this step (or a void step)
    __shared__ uint32_t s_key[TILE_HASH], s_list[TILE_SORT];
    __shared__ uint16_t s_val[TILE_HASH];
    __shared__ uint32_t s_n;
    const typename PR::State A = ctrl->cur ? S1 : S0;
    const int hl = ctrl->hlast;
    const uint32_t* hcnt = hl ? hcnt1 : hcnt0;
    Spring<typename PR::T>* hs = hl ? hs1 : hs0;
    uint64_t* hm = hl ? hm1 : hm0;
    const uint32_t tid = threadIdx.x, bd = blockDim.x;
    for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const SceneDev& S = scenes[scene_of_tile(scenes, nscenes, t)];
        const uint32_t off = (t - S.t0) * tile;
        const uint32_t q0 = S.p0 + off, n = min(tile, S.np - off);
        const uint32_t q = q0 + tid;
        const bool valid = tid < n;
        const uint32_t m = valid ? ncnt[q] : 0u;
        for (uint32_t k = tid; k < TILE_HASH; k += bd) s_key[k] = 0xFFFFFFFFu;
        for (uint32_t k = tid; k < TILE_SORT; k += bd) s_list[k] = 0xFFFFFFFFu;
        if (tid == 0) s_n = 0u;
        __syncthreads();
        // ---- the halo; and the spring mask by a merge of the list with the stored springs
        uint64_t mask = 0;
        {
            const uint32_t src = valid ? perm[q] : 0u;
            const uint32_t c = valid ? min(hcnt[src], maxc) : 0u;
            uint32_t o = 0, kept = 0, pid = c ? hs[src].pid : DEM_WALL_BASE;
            for (uint32_t k0 = 0; k0 < m; k0 += 4) {
                // four entries and their ids in flight together
                uint32_t jj[4], id[4];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) jj[u] = k0 + u < m ? nl[(size_t)(k0 + u) * cap + q] : q0;
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) id[u] = o < c ? __ldg(&A.id[jj[u]]) : 0u;
                auto pick = [](const uint32_t (&a)[4], uint32_t u) {
                    return u == 0 ? a[0] : (u == 1 ? a[1] : (u == 2 ? a[2] : a[3]));
                };
#pragma unroll 1   // (unrolled: 94 -> 99 us at 500,009 spheres, 31.6 -> 34.8 at 9,217)
                for (uint32_t u = 0; u < 4; ++u) {
                    const uint32_t k = k0 + u, j = pick(jj, u), idj = pick(id, u);
                    if (k >= m) break;
                    if (o < c && pid < DEM_WALL_BASE) {
                        while (o < c && pid < idj) {   // a partner that left the list
                            ++o;
                            pid = o < c ? hs[(size_t)o * cap + src].pid : DEM_WALL_BASE;
                        }
                        if (o < c && pid == idj) {
                            if (kept != o) swap_springs(hs, (size_t)kept * cap + src, (size_t)o * cap + src);
                            ++kept;
                            mask |= 1ull << k;
                            ++o;
                            pid = o < c ? hs[(size_t)o * cap + src].pid : DEM_WALL_BASE;
                        }
                    }
                    if (j - q0 >= n && *(volatile uint32_t*)&s_n <= hcap) {
                        uint32_t h = (j * 2654435761u) >> 21;   // 11 bits
                        for (;;) {
                            const uint32_t old = atomicCAS(&s_key[h], 0xFFFFFFFFu, j);
                            if (old == 0xFFFFFFFFu) {
                                const uint32_t at = atomicAdd(&s_n, 1u);
                                if (at < hcap) s_list[at] = j;
                                break;
                            }
                            if (old == j) break;
                            h = (h + 1) & (TILE_HASH - 1);
                        }
                    }
                }
            }
            while (o < c && pid < DEM_WALL_BASE) {   // partners beyond the list's last
                ++o;
                pid = o < c ? hs[(size_t)o * cap + src].pid : DEM_WALL_BASE;
            }
            if (kept != o)   // the wall springs move up
                for (; o < c; ++o, ++kept) swap_springs(hs, (size_t)kept * cap + src, (size_t)o * cap + src);
            if (valid) hm[q] = mask;
        }
        __syncthreads();
        const uint32_t nh = s_n;
        if (nh > hcap) {
            if (tid == 0) nhalo[t] = HALO_NONE;
            __syncthreads();
            continue;
        }
        uint32_t w = 32;
        while (w < nh) w <<= 1;
        for (uint32_t k = 2; k <= w; k <<= 1)
            for (uint32_t j = k >> 1; j > 0; j >>= 1) {
                for (uint32_t i = tid; i < w; i += bd) {
                    const uint32_t o = i ^ j;
                    if (o > i) {
                        const uint32_t a = s_list[i], b = s_list[o];
                        if ((a > b) == ((i & k) == 0)) {
                            s_list[i] = b;
                            s_list[o] = a;
                        }
                    }
                }
                __syncthreads();
            }
        for (uint32_t i = tid; i < nh; i += bd) {
            const uint32_t j = s_list[i];
            halo[(size_t)t * hcap + i] = j;
            uint32_t h = (j * 2654435761u) >> 21;
            while (s_key[h] != j) h = (h + 1) & (TILE_HASH - 1);
            s_val[h] = (uint16_t)(tile + i);
        }
        if (tid == 0) nhalo[t] = nh;
        __syncthreads();
        for (uint32_t k = 0; k < m; k += 4) {
            uint32_t e[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                e[u] = tid;   // pad: the particle itself (the force pass masks it out)
                if (k + u < m) {
                    const uint32_t j = nl[(size_t)(k + u) * cap + q];
                    if (j - q0 < n) e[u] = j - q0;
                    else {
                        uint32_t h = (j * 2654435761u) >> 21;
                        while (s_key[h] != j) h = (h + 1) & (TILE_HASH - 1);
                        e[u] = s_val[h];
                    }
                }
            }
            nl4[(size_t)(k >> 2) * cap + q] = make_uint2(e[0] | (e[1] << 16), e[2] | (e[3] << 16));
        }
        __syncthreads();   // the table is cleared by the next tile
    }
}

// ======================================================================= launchers
static inline uint32_t nblk(uint32_t n, uint32_t b) { return (n + b - 1) / b; }
static inline uint32_t sgrid(const Domain& d, uint32_t n) {
    return std::max(1u, std::min(nblk(n, 256), (uint32_t)std::max(d.sort_blocks, 1)));
}

#define DEM_LAUNCH_CHECK()                          \
    do {                                            \
        ++d.launches;                               \
        cudaError_t e_ = cudaGetLastError();        \
        if (e_ != cudaSuccess) return e_;           \
    } while (0)

cudaError_t run_lists(Domain& d) {
    if (d.n == 0) return cudaSuccess;
    // 16 warps per SM, as far as warps of at least four positions reach
    uint32_t per = 32;
    while (per > 4 && d.n / per < 2u * (uint32_t)d.sort_blocks) per /= 2;
    const uint32_t grid = std::max(1u, std::min(nblk(d.n, 8 * per), (uint32_t)std::max(d.sort_blocks, 1)));
    if (d.precision == 0)
        k_nlist<PF64><<<grid, 256, 0, d.stream>>>(d.n, per, d.d_scenes, d.nscenes, d.S64[0], d.S64[1], d.ctrl, d.key,
                                                  d.canon, d.cs, d.fin, d.ncnt, d.nl, d.cap, d.wmask, d.st);
    else
        k_nlist<PF32><<<grid, 256, 0, d.stream>>>(d.n, per, d.d_scenes, d.nscenes, d.S32[0], d.S32[1], d.ctrl, d.key,
                                                  d.canon, d.cs, d.fin, d.ncnt, d.nl, d.cap, d.wmask, d.st);
    DEM_LAUNCH_CHECK();
    return run_tiles(d, false);
}

template <class PR>
static void launch_tiles(Domain& d, const typename PR::State& S0, const typename PR::State& S1, bool always) {
    using Sp = Spring<typename PR::T>;
    const uint32_t g = std::max(1u, std::min(d.ntiles, (uint32_t)std::max(d.sort_blocks, 1)));
    k_tile<PR><<<g, d.tile, 0, d.stream>>>(d.d_scenes, d.nscenes, d.tile, d.ntiles, halo_cap(d.tile), S0, S1, d.ctrl,
                                           always ? 1 : 0, d.ncnt, d.nl, d.nl4, d.halo, d.nhalo, d.cap, d.perm,
                                           d.hcnt[0], d.hcnt[1], (Sp*)d.hs[0], (Sp*)d.hs[1], d.hmask[0], d.hmask[1],
                                           (uint32_t)d.maxc);
}

// The tiles of the lists just built (always: also when no sort is due, for springs that
// were set after it).
cudaError_t run_tiles(Domain& d, bool always) {
    if (d.n == 0) return cudaSuccess;
    if (d.precision == 0) launch_tiles<PF64>(d, d.S64[0], d.S64[1], always);
    else launch_tiles<PF32>(d, d.S32[0], d.S32[1], always);
    DEM_LAUNCH_CHECK();
    return cudaSuccess;
}

cudaError_t run_wall_masks(Domain& d) {
    if (d.n == 0) return cudaSuccess;
    if (d.precision == 0)
        k_wall_masks<PF64><<<sgrid(d, d.n), 256, 0, d.stream>>>(d.n, d.d_scenes, d.nscenes, d.S64[0], d.S64[1], d.ctrl,
                                                               d.wmask);
    else
        k_wall_masks<PF32><<<sgrid(d, d.n), 256, 0, d.stream>>>(d.n, d.d_scenes, d.nscenes, d.S32[0], d.S32[1], d.ctrl,
                                                               d.wmask);
    DEM_LAUNCH_CHECK();
    return cudaSuccess;
}

}  // namespace demgb
