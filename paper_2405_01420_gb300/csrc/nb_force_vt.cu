// Force kernel over gathered tiles (the pruned list in its packed form).
//
// After a prune, each half i-cluster (rows 0-3 or 4-7 of an 8-atom cluster)
// has a list of 4 x 8 tiles whose 8 j atoms are gathered from all its
// cluster pairs: only j atoms within r_inner of at least one of the 4 rows
// appear, each with its own periodic shift (nb_prune.cu writes them). The
// arithmetic per pair is that of the cluster-pair kernel (nb_pair with
// d = (y_a - y_b) + S), so both kernels make the same in-range decisions.
//
// Layout (j-stationary): a warp takes one half at a time and reads its
// tiles in groups of 4, i.e. 32 j atoms, one per lane; each lane computes
// its j atom against the half's 4 i rows. On water at rc 1.0 / r_inner
// 1.04 nm about 60% of these pair slots are in range, against 40% for 8 x 8
// cluster tiles with empty half-tiles skipped.
//
//  - The pair arithmetic runs on the packed two-wide FP32 instructions:
//    rows (0, 1) and (2, 3) of the half are two row pairs, each evaluated
//    against the lane's j atom by nb_pair_x2 (one packed operation for two
//    pairs, same rounding per pair as nb_pair). The kernel is bound by
//    instruction issue, and packing halves the issue slots of the FP32 work.
//  - j data (coordinates and charge, type, mask word) of group g + 1 are
//    loaded into registers while group g is computed, their slot words one
//    group earlier still. (Staged through shared memory with cp.async, the
//    gathers cost 7.5 shared-memory wavefronts per copy and the data path of
//    L1 was 67% busy; with plain loads it is 37%: 898 -> 851 us per force
//    call at 1,000,002 atoms, 24.4 -> 23.5 at 11,997.)
//  - Groups whose j atoms all sit at the center image skip the addition of
//    S = 0 and its shared loads (851 -> 821 us at 1,000,002 atoms).
//  - The row pairs' positions and charges and their LJ coefficients by j
//    type sit in per-warp shared tables, already in packed order.
//  - j forces stay in registers over the 4 rows and go out with one
//    16-byte vector atomic per lane (fsort is float4 per slot).
//  - i forces stay in registers over the whole half and are reduced across
//    the warp at its end, one vector atomic per row.
//  - Energies: FP32 over a half (per lane, then across the warp), FP64
//    across halves in a per-warp shared pair (no registers held across
//    halves), FP64 atomics per system when the warp moves to another
//    system or finishes. The pair forces are the same bits with and without
//    energies (nb_pair_x2).
//  - Halves are handed out in cluster order. Half lists make the first
//    clusters' lists the longest and the last ones' the shortest, so the
//    launch ends with short items as it would in sorted order, and neither
//    an order array nor the sorting before it is needed (sorted: 1 us
//    slower per call at 96,000 atoms, 4 us at 1,000,002).
//  - First items (FIRST_BY_INDEX): from the work counter, or from the warp's index in
//    the grid. The counter serves one warp per 1.3 ns, so 3,040 warps start
//    over 4 us: a loss when each takes only a few halves (12,000 atoms: 23.3
//    us per call from the counter, 18.6 from the index), a gain of up to 6%
//    when it takes many (the warps' phases are spread from the start).
#include "nb_pair_x2.cuh"
#include "nb_warp.cuh"

namespace {

constexpr unsigned kStreams = 16u;   // places of a batch that are worked on at a time, with energies
constexpr unsigned kMaxPieces = 4u;  // pieces of a half's list in a small system

struct VtParams {
    const float4 *xq;
    const int *tsort;
    float *fsort;             // float4 per slot, viewed as floats
    const int *vt_slot;       // 8 per tile: slot | shift << 27
    const unsigned *vt_mask;  // 4 x 8 bits per tile
    const int *half_start;
    const int *half_len;
    const float *ljparams;
    nb_dev_state *st;
    double *energies;         // [2 nsys]
    const float4 *sys_shift;  // [27 nsys]
    const int *clus_sys;
    int ntype;
    float rc6inv, rc12inv;
    nb_coul cc;
    nb_coul2 cc2;             // the same constants in packed form
    float stale_prune2;
    int pad_slot;             // never holds an atom: far away, q = 0, type 0
    int reg0, nreg;           // regions of gathered tiles to compute (0 local or all, 1 non-local)
    int reg_stride;           // 2 nc_max: halves per region in half_start / half_len
    const int *nl_list;       // with a halo: the halves with non-local tiles (the prune's list), else NULL
    int finalize;             // move the displacement maxima of this evaluation to last_*
};

// Adds a warp's energies of one system (Coulomb in e[0], LJ in e[1]) to
// that system's pair (E_LJ, E_C) and clears them; lane 0 only.
__device__ __forceinline__ void flush_energies_vt(double *e, double *out) {
    atomicAdd(&out[0], e[1]);
    atomicAdd(&out[1], e[0]);
    e[0] = 0.0;
    e[1] = 0.0;
}

// The lane's slot word of group g of the half with tiles [t0, t1): its j
// atom's slot and shift, or the pad slot past the end (the load then reads
// tile t0, so that no lane branches).
__device__ __forceinline__ int slot_word(const VtParams &p, int t0, int t1, int g, int lane) {
    const int tile = t0 + 4 * g + (lane >> 3);
    const bool live = tile < t1;
    const int tc = live ? tile : t0;
    const int w = p.vt_slot[8 * (size_t)tc + (lane & 7)];
    return live ? w : (int)((unsigned)p.pad_slot | ((unsigned)NB_SHIFT_CENTER << 27));
}

// The lane's j atom of one group: coordinates and charge, type, mask word of
// its tile (0 past the end).
struct VtJ {
    float4 x;
    int t;
    unsigned m;
};

__device__ __forceinline__ VtJ load_j(const VtParams &p, int v, int t0, int t1, int g, int lane) {
    const int tile = t0 + 4 * g + (lane >> 3);
    const int slot = v & 0x07ffffff;
    VtJ j;
    j.m = 0u;
    if (tile < t1) j.m = p.vt_mask[tile];
    j.x = p.xq[slot];
    j.t = p.tsort[slot];
    return j;
}

// Pieces of each half's groups, one work item each (a small system without
// energies, whose sums would depend on the split). Whole halves against up to
// 4 pieces, force call: 1,536 atoms 13.8 -> 10.4 us, 4,500 16.2 -> 12.8; up
// to 8 pieces the same.
template <bool SPLIT>
__device__ __forceinline__ unsigned vt_pieces(unsigned grid_warps, unsigned halves) {
    return SPLIT ? min(nb_work_split(grid_warps, halves), kMaxPieces) : 1u;
}

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// The next work item: from the counter, past the items handed out by index.
__device__ __forceinline__ unsigned take_item(const VtParams &p, unsigned by_index, int lane) {
    unsigned w = 0;
    if (lane == 0) w = atomicAdd(&p.st->work, 1u);
    return __shfl_sync(0xffffffffu, w, 0) + by_index;
}

// j-stationary kernel over gathered tiles. A warp takes one half i-cluster
// (4 i rows) at a time; its tiles are read in groups of 4 (32 j atoms, one
// per lane), and each lane computes its j atom against the 4 rows, two row
// pairs of packed arithmetic. j forces stay in registers for the 4 pairs
// and go out with one 16-byte vector atomic per lane (fsort is float4 per
// slot); i forces stay in registers for the whole half and are reduced
// across the warp at its end. Group g + 1's j atoms load while group g is
// computed, and group g + 2's slot words meanwhile.
// Dynamic shared memory: the ntype x ntype LJ table, then per warp 3 float4
// per j type (see s_lj2).
// Bound by the FMA pipe and instruction issue together, 64 and 61% busy at
// 96,000 atoms without energies, 63 and 62% with them
// (a packed instruction holds the pipe for 2 cycles), with 5 warps per
// scheduler to cover a half's chain of dependent loads. RES x THREADS
// resident threads per SM set the register cap; pick_shape says which is
// taken when.
template <bool ENERGY, bool COUNT, int THREADS, int RES, bool FIRST_BY_INDEX, int COUL, bool BATCH>
__global__ void __launch_bounds__(THREADS, RES) k_force_vt(VtParams p) {
    constexpr int kWarps = THREADS / 32;
    extern __shared__ float4 s_lj[];
    __shared__ float4 s_shift[kWarps][27];  // the warp's copy of its system's shift vectors
    int shift_sys = -1;
    __shared__ float4 s_xi[kWarps][4];
    __shared__ int s_tr[kWarps][4];
    __shared__ float4 s_xp[kWarps][2][2];  // row pair k: (x_a, x_b, y_a, y_b), (z_a, z_b, fq_a, fq_b)
    __shared__ double s_e[kWarps][2];      // the warp's energies of its current system: Coulomb, LJ
    if (FIRST_BY_INDEX && !BATCH && p.nreg == 1 && p.reg0 == 0) {
        // the warp's first tiles, which the prune wrote, on their way while the gather runs
        const unsigned nh = 2u * (unsigned)p.st->nc, k = blockIdx.x * kWarps + (threadIdx.x >> 5);
        const unsigned pieces = vt_pieces<FIRST_BY_INDEX && !ENERGY>(gridDim.x * kWarps, nh), u = k / pieces;
        if (u < nh) {
            int g0, g1;
            const int len = p.half_len[u], lane = threadIdx.x & 31;
            nb_piece((len + 3) >> 2, k - u * pieces, pieces, g0, g1);
            const int tile = 4 * g0 + (lane >> 3);
            if (tile < len) {
                const size_t t = (size_t)p.half_start[u] + tile;
                prefetch_l1(p.vt_slot + 8 * t + (lane & 7));
                prefetch_l1(p.vt_mask + t);
            }
            prefetch_l1(p.clus_sys + (u >> 1));
        }
    }
    nb_pdl_wait();  // launched with nb_launch_pdl: the gather has completed from here on
    nb_pdl_release();
    const int nt2 = p.ntype * p.ntype;
    for (int k = threadIdx.x; k < nt2; k += blockDim.x) {
        const float c6 = p.ljparams[2 * k], c12 = p.ljparams[2 * k + 1];
        s_lj[k] = make_float4(c6, c12, c12 * p.rc12inv - c6 * p.rc6inv, 0.0f);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const unsigned ds = p.st->cur_d2_search, dp = p.st->cur_d2_prune;
        if (p.finalize) {
            p.st->last_d2_search = ds;
            p.st->last_d2_prune = dp;
            p.st->cur_d2_search = 0u;
            p.st->cur_d2_prune = 0u;
        }
        if (__uint_as_float(dp) > p.stale_prune2) atomicOr(&p.st->err, NB_DEV_STALE_PRUNE);
    }
    __syncthreads();

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // per warp, for the current half, by j type t: (C6, C6, C12, C12) of
    // row pairs (0, 1) and (2, 3) at [3t], [3t + 1], minus the 4 rows' LJ
    // shifts at [3t + 2]
    float4 *s_lj2 = s_lj + nt2 + 3 * p.ntype * warp;
    // Work items: region 0 (every pair without a halo, the local pairs with one) is every half, in
    // the list order; region 1 (non-local) is the prune's list of the halves that have such tiles
    const unsigned nhalf = 2u * (unsigned)p.st->nc;  // halves per region
    const unsigned n0 = p.reg0 == 0 ? nhalf : 0u;
    const unsigned n1 = p.reg0 + p.nreg == 2 ? (p.nl_list ? p.st->nl_count : nhalf) : 0u;
    const unsigned nseg = vt_pieces<FIRST_BY_INDEX && !ENERGY>(gridDim.x * kWarps, n0 + n1);
    // BATCH (with energies): the halves of kStreams places of the batch in turn, 8 neighbours at a
    // time. In plain order all warps work in one system or two at any time, and every half's energies
    // queue on the same addresses: 190 boxes at rc 0.7 2,913 -> 2,520 us, 60 small ones 630 -> 546
    const unsigned chunk = BATCH ? 8u * ((n0 + 8u * kStreams - 1u) / (8u * kStreams)) : 0u;
    const unsigned nwork = BATCH ? kStreams * chunk : (n0 + n1) * nseg;
    if (ENERGY && lane == 0) s_e[warp][0] = s_e[warp][1] = 0.0;
    int cur_sys = -1;
    unsigned cnt = 0;

    const unsigned by_index = FIRST_BY_INDEX ? gridDim.x * kWarps : 0u;
    unsigned w = FIRST_BY_INDEX ? blockIdx.x * kWarps + warp : 0u;
    if (!FIRST_BY_INDEX) w = take_item(p, 0u, lane);
    for (;;) {
        unsigned reg = 0u, hw = 0u;
        const unsigned u = nseg == 1u ? w : w / nseg, seg = w - u * nseg;
        int ci = 0;
        if (BATCH) {
            const unsigned a = w >> 3;
            hw = (a % kStreams) * chunk + 8u * (a / kStreams) + (w & 7u);
            if (w < nwork && hw >= n0) {  // past the last half of the batch
                w = take_item(p, by_index, lane);
                continue;
            }
            ci = (int)(hw >> 1);
        } else if (u < n0) {
            hw = u;
            ci = (int)(hw >> 1);
        } else if (w < nwork) {
            reg = 1u;
            hw = p.nl_list ? (unsigned)p.nl_list[u - n0] : u - n0;
            ci = (int)(hw >> 1);
        }
        const int h = (int)(hw & 1u);
        const int csys = (w < nwork) ? p.clus_sys[ci] : -1;
        if (ENERGY && csys != cur_sys) {
            if (cur_sys >= 0 && lane == 0) flush_energies_vt(s_e[warp], p.energies + 2 * cur_sys);
            cur_sys = csys;
        }
        if (w >= nwork) break;
        const size_t hidx = (size_t)reg * p.reg_stride + 2 * ci + h;
        int t0 = p.half_start[hidx], t1 = t0 + p.half_len[hidx];
        if (nseg > 1u) {
            int g0, g1;
            nb_piece((t1 - t0 + 3) >> 2, seg, nseg, g0, g1);
            t1 = min(t1, t0 + 4 * g1);
            t0 += 4 * g0;
        }
        if (t1 <= t0) {
            w = take_item(p, by_index, lane);
            continue;
        }
        if (csys != shift_sys) {
            if (lane < 27) s_shift[warp][lane] = p.sys_shift[27 * csys + lane];
            shift_sys = csys;
        }
        const int ibase = ci * NB_CLUSTER + 4 * h;
        int v = slot_word(p, t0, t1, 0, lane);
        VtJ j = load_j(p, v, t0, t1, 0, lane);
        int vnext = slot_word(p, t0, t1, 1, lane);
        if (lane < 4) {
            const float4 x = p.xq[ibase + lane];
            s_xi[warp][lane] = make_float4(x.x, x.y, x.z, x.w * NB_COULOMB_F);
            s_tr[warp][lane] = p.tsort[ibase + lane] * p.ntype;
        }
        float2 fix[2], fiy[2], fiz[2];  // row pair k: rows 2k (.x) and 2k + 1 (.y)
#pragma unroll
        for (int k = 0; k < 2; ++k) fix[k] = fiy[k] = fiz[k] = make_float2(0.f, 0.f);
        float2 ec2 = make_float2(0.f, 0.f), elj2 = make_float2(0.f, 0.f);
        const int ngroups = (t1 - t0 + 3) >> 2;
        __syncwarp();
        if (lane < 2) {
            const float4 a = s_xi[warp][2 * lane], b = s_xi[warp][2 * lane + 1];
            s_xp[warp][lane][0] = make_float4(a.x, b.x, a.y, b.y);
            s_xp[warp][lane][1] = make_float4(a.z, b.z, a.w, b.w);
        }
        for (int t = lane; t < p.ntype; t += 32) {
            const float4 c0 = s_lj[s_tr[warp][0] + t], c1 = s_lj[s_tr[warp][1] + t];
            const float4 c2 = s_lj[s_tr[warp][2] + t], c3 = s_lj[s_tr[warp][3] + t];
            s_lj2[3 * t + 0] = make_float4(c0.x, c1.x, c0.y, c1.y);
            s_lj2[3 * t + 1] = make_float4(c2.x, c3.x, c2.y, c3.y);
            if (ENERGY) s_lj2[3 * t + 2] = make_float4(-c0.z, -c1.z, -c2.z, -c3.z);
        }
        __syncwarp();
        for (int g = 0; g < ngroups; ++g) {
            const float4 xj = j.x;
            const int tj = j.t;
            const unsigned mrow = j.m >> (lane & 7);  // bit 8a: row a
            const int slot = v & 0x07ffffff;
            const float2 nxjx = nb_f2(-xj.x), nxjy = nb_f2(-xj.y), nxjz = nb_f2(-xj.z), qj = nb_f2(xj.w);
            // d = (y_a - y_b) + S; a group whose atoms all sit at the center image skips S = 0
            float2 dx[2], dy[2], dz[2], qi[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float4 xa = s_xp[warp][k][0], xb = s_xp[warp][k][1];
                dx[k] = __fadd2_rn(make_float2(xa.x, xa.y), nxjx);
                dy[k] = __fadd2_rn(make_float2(xa.z, xa.w), nxjy);
                dz[k] = __fadd2_rn(make_float2(xb.x, xb.y), nxjz);
                qi[k] = make_float2(xb.z, xb.w);
            }
            if (__any_sync(0xffffffffu, ((unsigned)v >> 27) != NB_SHIFT_CENTER)) {
                const float4 S = s_shift[warp][(unsigned)v >> 27];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    dx[k] = __fadd2_rn(dx[k], nb_f2(S.x));
                    dy[k] = __fadd2_rn(dy[k], nb_f2(S.y));
                    dz[k] = __fadd2_rn(dz[k], nb_f2(S.z));
                }
            }
            float4 nsh = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ENERGY) nsh = s_lj2[3 * tj + 2];
            float2 gjx = make_float2(0.f, 0.f), gjy = gjx, gjz = gjx;
            // the next group's j atoms load during this whole group, and the slot words after it
            // a group ahead (past the last group: the pad slot)
            j = load_j(p, vnext, t0, t1, g + 1, lane);
            const int vafter = slot_word(p, t0, t1, g + 2, lane);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int c2 = nb_pair_x2<ENERGY, COUL>(
                    dx[k], dy[k], dz[k], qi[k], qj, s_lj2[3 * tj + k],
                    k == 0 ? make_float2(nsh.x, nsh.y) : make_float2(nsh.z, nsh.w), ((mrow >> (16 * k)) & 1u) != 0u,
                    ((mrow >> (16 * k + 8)) & 1u) != 0u, p.cc.rc2, p.cc2, fix[k], fiy[k], fiz[k], gjx, gjy, gjz, ec2,
                    elj2);
                if (COUNT) cnt += c2;
            }
            if (slot != p.pad_slot)  // all padding lanes share one slot: no atomics there
                atomicAdd(reinterpret_cast<float4 *>(p.fsort) + slot,
                          make_float4(-(gjx.x + gjx.y), -(gjy.x + gjy.y), -(gjz.x + gjz.y), 0.0f));
            v = vnext;
            vnext = vafter;
        }
        // i forces: row a component c is value 4a + c; lanes 2k hold value k
        float r[16];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            r[8 * k + 0] = fix[k].x;
            r[8 * k + 1] = fiy[k].x;
            r[8 * k + 2] = fiz[k].x;
            r[8 * k + 3] = 0.0f;
            r[8 * k + 4] = fix[k].y;
            r[8 * k + 5] = fiy[k].y;
            r[8 * k + 6] = fiz[k].y;
            r[8 * k + 7] = 0.0f;
        }
        reduce_scatter<16>(r, lane);
        // lane 8a holds row a's x; its y and z sit 2 and 4 lanes up
        const float ry = __shfl_down_sync(0xffffffffu, r[0], 2);
        const float rz = __shfl_down_sync(0xffffffffu, r[0], 4);
        if ((lane & 7) == 0)
            atomicAdd(reinterpret_cast<float4 *>(p.fsort) + ibase + (lane >> 3), make_float4(r[0], ry, rz, 0.0f));
        if (ENERGY) {
            float ec = ec2.x + ec2.y, el = elj2.x + elj2.y;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                ec += __shfl_xor_sync(0xffffffffu, ec, o);
                el += __shfl_xor_sync(0xffffffffu, el, o);
            }
            if (lane == 0) {
                s_e[warp][0] += (double)ec;
                s_e[warp][1] += (double)el;
            }
        }
        __syncwarp();
        w = take_item(p, by_index, lane);
    }
    if (COUNT) {
        unsigned long long c64 = cnt;
        for (int o = 16; o > 0; o >>= 1) c64 += __shfl_xor_sync(0xffffffffu, c64, o);
        if (lane == 0) atomicAdd(&p.st->npairs, c64);
    }
}

using VtFn = void (*)(VtParams);

// Launch shapes (threads, resident CTAs per SM, first items by index). The
// default of 128 threads picks by the halves there are per warp of the grid;
// microseconds per force call at 5 CTAs from the counter, then the shape
// taken (rc 1.0, water; replays of 20 or more calls without energies):
//   without energies, up to 3.5 halves per warp: 5 CTAs by index
//     (6,000 atoms 21.9 -> 15.7, 24,000 28.6 -> 27.6, 36,000 37.5 -> 37.5;
//     96,000 84.4 -> 84.7, 1,000,002 825 -> 880; RF 12,000 17.4 -> 15.4)
//   reaction field without energies, from 10 halves per warp: 6 CTAs (80
//     registers; 96,000 59.9 -> 59.8, 192,000 128 -> 122). Ewald gains
//     nothing by it (192,000 164 -> 166, 1,000,002 825 -> 827)
//   with energies, up to 6 halves per warp of 4 CTAs: 4 CTAs by index
//     (6,000 25.4 -> 17.2, 24,000 36.1 -> 34.2, 48,000 57.4 -> 55.5;
//     96,000 102.3 -> 106.8)
// Counting kernels and 256 threads have one shape.
enum { kShape256, kShapeCounter, kShapeIndex, kShapeMany, kShapes };

int pick_shape(bool energy, bool count, int threads, int coul, long long halves, int num_sms) {
    if (threads == 256) return kShape256;
    if (count) return kShapeCounter;
    const long long per_cta = 4LL * num_sms;  // warps of the grid per resident CTA
    if (energy) return halves <= 6 * 4 * per_cta ? kShapeIndex : kShapeCounter;
    if (2 * halves <= 7 * 5 * per_cta) return kShapeIndex;
    return coul == NB_COULK_RF && halves >= 10 * 5 * per_cta ? kShapeMany : kShapeCounter;
}

template <bool E, bool C, int K, bool B>
VtFn pick_vt_shape(int shape) {
    if (shape == kShape256) return k_force_vt<E, C, 256, 2, false, K, B>;
    if constexpr (!C) {
        if (shape == kShapeIndex) return k_force_vt<E, C, 128, E ? 4 : 5, true, K, B>;
        if constexpr (!E && K == NB_COULK_RF)
            if (shape == kShapeMany) return k_force_vt<E, C, 128, 6, false, K, B>;
    }
    return k_force_vt<E, C, 128, 5, false, K, B>;
}

template <bool E, bool C, int K>
VtFn pick_vt_coul(int shape, bool batch) {
    if constexpr (E)
        if (batch) return pick_vt_shape<E, C, K, true>(shape);
    return pick_vt_shape<E, C, K, false>(shape);
}

template <bool E, bool C>
VtFn pick_vt(int shape, int coul, bool batch) {
    if (coul == NB_COULK_RF) return pick_vt_coul<E, C, NB_COULK_RF>(shape, batch);
    if constexpr (E)
        if (coul == NB_COULK_EWALD_SHIFT) return pick_vt_coul<E, C, NB_COULK_EWALD_SHIFT>(shape, batch);
    return pick_vt_coul<E, C, NB_COULK_EWALD>(shape, batch);  // the shift does not change forces
}

struct Occ {
    size_t smem;
    int per_sm;
};
Occ g_vt_occ[3][2][2][2][kShapes] = {};

}  // namespace

cudaError_t nb_launch_force_vt(nb_pairlist *pl, int ntype, const float *ljparams, float rc, float beta,
                               double *energies, float stale_prune2, int part, cudaStream_t s) {
    VtParams p;
    // regions: without a halo one (every pair); with one, 0 = local, 1 = non-local
    p.reg0 = part == NB_PART_NONLOCAL ? 1 : 0;
    p.nreg = (part == NB_PART_ALL && pl->vt_parts == 2) ? 2 : 1;
    p.reg_stride = 2 * pl->nc_max;
    p.nl_list = pl->vt_parts == 2 ? pl->nl_list : nullptr;
    p.finalize = part != NB_PART_LOCAL;
    p.xq = pl->xq;
    p.tsort = pl->tsort;
    p.fsort = reinterpret_cast<float *>(pl->fsort);
    p.vt_slot = pl->vt_slot;
    p.vt_mask = pl->vt_mask;
    p.half_start = pl->half_start;
    p.half_len = pl->half_len;
    p.ljparams = ljparams;
    p.st = pl->st;
    p.energies = energies;
    p.sys_shift = pl->sys_shift;
    p.clus_sys = pl->clus_sys;
    p.ntype = ntype;
    const double rc6 = 1.0 / ((double)rc * rc * rc * rc * rc * rc);
    p.rc6inv = (float)rc6;
    p.rc12inv = (float)(rc6 * rc6);
    const int coul = nb_fill_coul(p.cc, rc, beta, pl->coul_kind, pl->eps_rf, pl->coul_flags);
    p.cc2 = nb_pack_coul(p.cc);
    p.stale_prune2 = stale_prune2;
    p.pad_slot = pl->nc_max * NB_CLUSTER;
    const int e = energies ? 1 : 0;
    const int c = (pl->flags & NB_FLAG_COUNT_PAIRS) ? 1 : 0;
    const int threads = pl->force_threads == 256 ? 256 : 128;
    // halves of all systems: one cluster per 8 atoms and at most one more per column
    const long long halves = 2LL * (pl->n_atoms / NB_CLUSTER + pl->ncol);
    const int shape = pick_shape(e, c, threads, coul, halves, pl->num_sms);
    const bool batch = e && pl->nsys > 1;
    VtFn fn = e ? (c ? pick_vt<true, true>(shape, coul, batch) : pick_vt<true, false>(shape, coul, batch))
                : (c ? pick_vt<false, true>(shape, coul, batch) : pick_vt<false, false>(shape, coul, batch));
    const size_t smem = sizeof(float4) * ((size_t)ntype * ntype + 3 * (size_t)ntype * (threads / 32));
    Occ &occ = g_vt_occ[coul][e][c][batch][shape];
    if (occ.per_sm == 0 || occ.smem != smem) {  // resident CTAs for this LJ table size
        int n = 0;
        cudaError_t err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, (const void *)fn, threads, smem);
        if (err != cudaSuccess) return err;
        occ.smem = smem;
        occ.per_sm = n < 1 ? 1 : n;
    }
    const int per_sm = occ.per_sm;
    const int use = pl->force_blocks_per_sm > 0 ? min(pl->force_blocks_per_sm, per_sm) : per_sm;
    int blocks = pl->num_sms * use;
    const long long items = 2LL * p.nreg * pl->nc_max * (shape == kShapeIndex && !e ? kMaxPieces : 1u);
    blocks = (int)min((long long)blocks, (items + threads / 32 - 1) / (threads / 32));
    return nb_launch_pdl(fn, max(blocks, 1), threads, smem, s, p);
}
