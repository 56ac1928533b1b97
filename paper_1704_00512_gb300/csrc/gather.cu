// Gather plan of the column-order kernel built on the device (Eq. 3 restricted
// to the pattern; column independence, Sec. "Expansion in Chebyshev
// polynomials"): from the device block-CSR patterns of P_out and of the
// operator, with the same panels, groups, warp streams and entry words as the
// host builder in colstep.cu (bit for bit).
//
//   k_gp_spans   a warp per block column: where a panel that starts there ends (P
//                columns, or the next column's new rows would overflow the union
//                capacity);
//   k_gp_panels  one thread follows the starts, its block writes the panels;
//   k_gp_rows    one thread block per panel: the union of the panel's
//                columns' rows as a bitmap with ranks (slot = rank) and per union
//                row a bitmap of its operator slots; one warp groups the rows by
//                fours; per group its merged slots and their count, and -- in the
//                fill pass -- the groups dealt to the NW warps
//                by decreasing quad count (each to the warp with the least work so
//                far, ties to the lowest warp), the group words, the entry streams
//                padded with zero-block entries, and the union slot of every P_out
//                block of the panel;
//   k_gp_scan    offsets of the panels' quads and groups.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "kernels.cuh"
#include "plan.cuh"

namespace cheb {

constexpr int GP_NT = 512;
constexpr int GP_NWARP = GP_NT / 32;
constexpr int GP_MAXU = 1 << COL_SLOT_BITS;  // union slots
constexpr int GP_MAXG = GP_MAXU / 4;         // groups, and quads of a group
constexpr int GP_STATIC = 12 * 1024;         // static shared memory of k_gp_rows at most
static_assert(GP_NWARP == COL_NW, "one warp of the builder per warp stream of the step kernel");

// Block-wide integer sum, returned to every thread.
__device__ __forceinline__ int64_t gp_block_sum(int64_t v, int64_t *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    int64_t r = 0;
#pragma unroll
    for (int i = 0; i < GP_NWARP; ++i) r += sh[i];
    __syncthreads();
    return r;
}
__device__ __forceinline__ int gp_block_max(int v, int *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    int r = 0;
#pragma unroll
    for (int i = 0; i < GP_NWARP; ++i) r = max(r, sh[i]);
    __syncthreads();
    return r;
}

// The panel walk shared by every panel set: within each system [sys_col[s],
// sys_col[s+1]) the block columns are taken in order, and a panel is closed when P
// columns are in it or the next column would take its union of rows above ucap or its
// blocks above bcap.  Where a panel that starts at column j ends depends on j alone, so
// a warp per column finds that for every column (span[j]: columns, union rows, blocks,
// system), and one thread follows the starts.  (One thread block that walked the
// columns one after the other took 2.2 ms a panel set at 1,500 columns; now 0.07.)
__global__ void __launch_bounds__(256) k_gp_spans(const int64_t *rp, const int32_t *ci, int64_t nbr, int P, int64_t ucap,
                                                  int64_t bcap, const int64_t *sys_col, int nsys, int4 *span) {
    const int64_t j = (blockIdx.x * (int64_t)256 + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= nbr) return;
    int lo = 0, hi = nsys - 1;  // the last system that starts at or before j
    while (lo < hi) {
        const int m = (lo + hi + 1) >> 1;
        if (sys_col[m] <= j) lo = m; else hi = m - 1;
    }
    const int64_t end = sys_col[lo + 1];
    int64_t cnt = 0, nblk = 0;
    int q = 0;
    for (; q < P && j + q < end; ++q) {
        const int64_t r0 = rp[j + q], r1 = rp[j + q + 1];
        int add = 0;  // rows of this column in none before it
        for (int64_t e = r0 + lane; e < r1; e += 32) {
            const int x = ci[e];
            bool fresh = true;
            for (int k = 0; k < q && fresh; ++k) {
                int64_t a = rp[j + k], b = rp[j + k + 1];
                const int64_t stop = b;
                while (a < b) {
                    const int64_t m = (a + b) >> 1;
                    if (ci[m] < x) a = m + 1; else b = m;
                }
                fresh = !(a < stop && ci[a] == x);
            }
            add += fresh;
        }
        add = __reduce_add_sync(0xffffffffu, add);
        if (cnt + add > ucap || nblk + (r1 - r0) > bcap) break;
        cnt += add;
        nblk += r1 - r0;
    }
    if (lane == 0) span[j] = make_int4(q, (int)cnt, (int)nblk, lo);
}
// panels: (first column, columns, union rows, system) per panel; aux (or NULL):
// (blocks, system) per panel.  out[0] = panels, out[1] = largest union, out[2]
// = 1 if a single column does not fit, out[3] = most blocks of a panel.
constexpr int GP_WIN = 32768;
__global__ void __launch_bounds__(GP_NT) k_gp_panels(const int4 *span, int64_t nbr, int32_t *panels, int32_t *aux,
                                                     int64_t *out) {
    __shared__ unsigned char w[GP_WIN];
    __shared__ int64_t s_np;
    __shared__ int s_max[2];
    const int tid = threadIdx.x;
    int64_t j = 0, np = 0;  // (thread 0's)
    if (tid < 2) s_max[tid] = 0;
    for (int64_t base = 0; base < nbr; base += GP_WIN) {
        const int n = (int)min((int64_t)GP_WIN, nbr - base);
        __syncthreads();
        for (int i = tid; i < n; i += GP_NT) w[i] = (unsigned char)span[base + i].x;
        __syncthreads();
        if (tid == 0) {
            while (np >= 0 && j < base + n) {
                const int c = w[j - base];
                if (c == 0) {
                    np = -1;  // a single column does not fit
                } else {
                    panels[4 * np++] = (int32_t)j;
                    j += c;
                }
            }
        }
    }
    if (tid == 0) s_np = np;
    __syncthreads();
    if (s_np < 0) {
        if (tid == 0) out[2] = 1;
        return;
    }
    for (int64_t p = tid; p < s_np; p += GP_NT) {
        const int4 v = span[panels[4 * p]];
        panels[4 * p + 1] = v.x;
        panels[4 * p + 2] = v.y;
        panels[4 * p + 3] = v.w;
        if (aux) {
            aux[2 * p] = v.z;
            aux[2 * p + 1] = v.w;
        }
        atomicMax(&s_max[0], v.y);
        atomicMax(&s_max[1], v.z);
    }
    __syncthreads();
    if (tid == 0) {
        out[0] = s_np;
        out[1] = s_max[0];
        out[2] = 0;
        out[3] = s_max[1];
    }
}

struct GpArgs {
    const int64_t *rp;
    const int32_t *ci;
    int64_t nbr;
    const int64_t *lrp;
    const int32_t *lci;
    int64_t nnzL;
    const int32_t *panels;
    // count pass
    int64_t *cnt_chunks, *cnt_rows;
    int32_t *cnt_maxrow;
    // fill pass
    const int64_t *chunk_off, *row_off;
    int32_t *wchunk, *wrow;
    uint32_t *rows, *ent;
    uint16_t *slot;
    int32_t *err;
    // dynamic shared memory: the union as a bitmap, the prefix count of each of its words,
    // the operator slots of the union rows, and for each of the fill warps its group's
    // merged slots and their places (ucap each)
    int off_pre, off_ub, off_list, ucap, fill_warps;
};

template <bool FILL>
__global__ void __launch_bounds__(GP_NT) k_gp_rows(const GpArgs a) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ int ulist[GP_MAXU];
    __shared__ int work[GP_MAXG], gch[GP_MAXG], gro[GP_MAXG];
    __shared__ int16_t order[GP_MAXG];
    __shared__ uint8_t wsel[GP_MAXG];
    __shared__ int hist[GP_MAXG + 1];
    __shared__ int16_t group[GP_MAXG][4];
    __shared__ int wsum[32];
    __shared__ int64_t sh[GP_NWARP];
    __shared__ int shi[GP_NWARP];
    __shared__ int bin_ch[COL_NW + 1], bin_ro[COL_NW + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t p = blockIdx.x;
    const int j0 = a.panels[4 * p], nc = a.panels[4 * p + 1], nu_plan = a.panels[4 * p + 2];
    const int64_t nw = (a.nbr + 31) / 32;
    uint32_t *bits = reinterpret_cast<uint32_t *>(dsm);
    uint16_t *pre = reinterpret_cast<uint16_t *>(dsm + a.off_pre);
    auto rank = [&](int K) {  // union slot of block row K, or -1
        const uint32_t w = bits[K >> 5], b = 1u << (K & 31);
        return w & b ? (int)pre[K >> 5] + __popc(w & (b - 1u)) : -1;
    };

    // 1. union bitmap of the panel's columns' rows, ranks, sorted union list
    for (int64_t w = tid; w < nw; w += GP_NT) bits[w] = 0u;
    __syncthreads();
    for (int q = 0; q < nc; ++q)
        for (int64_t e = a.rp[j0 + q] + tid; e < a.rp[j0 + q + 1]; e += GP_NT) {
            const int K = a.ci[e];
            atomicOr(&bits[K >> 5], 1u << (K & 31));
        }
    __syncthreads();
    const int64_t chunk = (nw + GP_NT - 1) / GP_NT;
    const int64_t wb = min(nw, (int64_t)tid * chunk), we = min(nw, wb + chunk);
    int cnt = 0;
    for (int64_t w = wb; w < we; ++w) cnt += __popc(bits[w]);
    int total;
    int run = block_excl_scan<GP_NWARP>(cnt, wsum, &total);
    const int nu = total, ng = (nu + 3) / 4;
    if (nu != nu_plan || nu >= GP_MAXU) {  // uniform
        if (tid == 0) atomicExch(a.err, 1);
        return;
    }
    for (int64_t w = wb; w < we; ++w) {
        unsigned m = bits[w];
        pre[w] = (uint16_t)run;
        while (m) {
            const int b = __ffs(m) - 1;
            ulist[run++] = (int)(w * 32 + b);
            m &= m - 1u;
        }
    }
    __syncthreads();
    if (FILL)
        for (int q = 0; q < nc; ++q)
            for (int64_t e = a.rp[j0 + q] + tid; e < a.rp[j0 + q + 1]; e += GP_NT)
                a.slot[e] = (uint16_t)rank(a.ci[e]);

    // 2. operator slots of every union row
    const int uw = (nu + 31) / 32;
    uint32_t *ub = reinterpret_cast<uint32_t *>(dsm + a.off_ub);
    for (int i = tid; i < nu * uw; i += GP_NT) ub[i] = 0u;
    __syncthreads();
    for (int u = warp; u < nu; u += GP_NWARP) {
        const int I = ulist[u];
        for (int64_t e = a.lrp[I] + lane; e < a.lrp[I + 1]; e += 32) {
            const int sl = rank(a.lci[e]);
            if (sl >= 0) atomicOr(&ub[u * uw + (sl >> 5)], 1u << (sl & 31));
        }
    }
    __syncthreads();
    // groups: the first row left, then three times, among the COL_WINDOW rows left
    // after it, the one with the smallest 2 (new slots) - (slots), the first of
    // those.  Lane l holds the candidates l and l + 32 in order (-1: none).
    if (warp == 0) {
        int c0 = lane < nu ? lane : -1, c1 = 32 + lane < nu ? 32 + lane : -1, next = 64;
        auto drop = [&](int k) {  // remove candidate k, fill up from the rows behind
            const int up0 = __shfl_down_sync(0xffffffffu, c0, 1), first1 = __shfl_sync(0xffffffffu, c1, 0);
            const int up1 = __shfl_down_sync(0xffffffffu, c1, 1);
            if (lane >= k) c0 = lane < 31 ? up0 : first1;
            if (lane + 32 >= k) c1 = lane < 31 ? up1 : (next < nu ? next : -1);
            ++next;
        };
        for (int i = 0; i < ng; ++i) {
            uint32_t cur = 0u;  // the group's slots, a word per lane
            for (int r = 0; r < 4; ++r) {
                int best = 0;
                if (r > 0) {
                    int k0 = 0, k1 = 0;
                    for (int w = 0; w < uw; ++w) {
                        const uint32_t m = __shfl_sync(0xffffffffu, cur, w);
                        const uint32_t x = c0 >= 0 ? ub[c0 * uw + w] : 0u, y = c1 >= 0 ? ub[c1 * uw + w] : 0u;
                        k0 += 2 * __popc(x & ~m) - __popc(x);
                        k1 += 2 * __popc(y & ~m) - __popc(y);
                    }
                    // (cost, place) as one key; no candidate: the largest
                    const unsigned q0 = c0 >= 0 ? ((unsigned)(k0 + 2048) << 6) | (unsigned)lane : 0xffffffffu;
                    const unsigned q1 = c1 >= 0 ? ((unsigned)(k1 + 2048) << 6) | (unsigned)(lane + 32) : 0xffffffffu;
                    best = (int)(__reduce_min_sync(0xffffffffu, min(q0, q1)) & 63u);
                }
                const int u0 = __shfl_sync(0xffffffffu, c0, best & 31), u1 = __shfl_sync(0xffffffffu, c1, best & 31);
                const int u = __shfl_sync(0xffffffffu, c0, 0) < 0 ? -1 : best < 32 ? u0 : u1;  // -1: no row left
                if (lane == 0) group[i][r] = (int16_t)u;
                if (u < 0) continue;
                if (lane < uw) cur |= ub[u * uw + lane];
                drop(best);
            }
        }
    }
    __syncthreads();
    // per group: the merged slots (one word of the bitmap per lane), quads (even)
    auto merge = [&](int i) {
        uint32_t m = 0u;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int u = group[i][r];
            if (u >= 0 && lane < uw) m |= ub[u * uw + lane];
        }
        return m;
    };
    int mymax = 0;
    int64_t mych = 0;
    for (int i = warp; i < ng; i += GP_NWARP) {
        const int k = __reduce_add_sync(0xffffffffu, __popc(merge(i)));
        const int wk = max(2, (k + 7) / 8 * 2);
        if (lane == 0) {
            work[i] = wk;
            mymax = max(mymax, wk);
            mych += wk;
        }
    }
    const int64_t chunks = gp_block_sum(mych, sh);  // (barrier: work[] complete)
    const int maxrow = gp_block_max(mymax, shi);
    if (!FILL) {
        if (tid == 0) {
            a.cnt_chunks[p] = chunks;
            a.cnt_rows[p] = ng;
            a.cnt_maxrow[p] = maxrow;
        }
        return;
    }

    // 3. groups to warps: decreasing quad count (stable), each to the warp with
    // the fewest quads so far (the lowest such warp)
    if (warp == 0) {
        for (int v = lane; v <= maxrow; v += 32) hist[v] = 0;
        __syncwarp();
        if (lane == 0) {
            for (int i = 0; i < ng; ++i) ++hist[work[i]];
            int at = 0;
            for (int v = maxrow; v >= 0; --v) {
                const int t = hist[v];
                hist[v] = at;
                at += t;
            }
            for (int i = 0; i < ng; ++i) order[hist[work[i]]++] = (int16_t)i;
        }
        __syncwarp();
        // lane w keeps the load of stream w; the lane with the smallest (load, w) takes the group
        int load = 0, rows = 0;
        for (int i = 0; i < ng; ++i) {
            const int gi = order[i];
            const unsigned key = lane < COL_NW ? ((unsigned)load << 5) | (unsigned)lane : 0xffffffffu;
            const int best = (int)(__reduce_min_sync(0xffffffffu, key) & 31u);
            if (lane == best) {
                load += work[gi];
                ++rows;
                wsel[gi] = (uint8_t)lane;
            }
        }
        int ch = load, ro = rows;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, ch, o), y = __shfl_up_sync(0xffffffffu, ro, o);
            if (lane >= o) {
                ch += x;
                ro += y;
            }
        }
        if (lane < COL_NW) {
            bin_ch[lane] = ch - load;
            bin_ro[lane] = ro - rows;
            a.wchunk[p * (COL_NW + 1) + lane] = (int32_t)(a.chunk_off[p] + ch - load);
            a.wrow[p * (COL_NW + 1) + lane] = (int32_t)(a.row_off[p] + ro - rows);
            if (lane == COL_NW - 1) {
                a.wchunk[p * (COL_NW + 1) + COL_NW] = (int32_t)(a.chunk_off[p] + ch);
                a.wrow[p * (COL_NW + 1) + COL_NW] = (int32_t)(a.row_off[p] + ro);
            }
        }
    }
    __syncthreads();

    // 4. warp w lays out the groups of stream w in increasing order
    {
        const unsigned lt = (1u << lane) - 1u;
        int ro = bin_ro[warp], ch = bin_ch[warp];
        for (int base = 0; base < ng; base += 32) {
            const int i = base + lane;
            const bool sel = i < ng && wsel[i] == warp;
            const unsigned m = __ballot_sync(0xffffffffu, sel);
            const int wk = sel ? work[i] : 0;
            int incl = wk;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            if (sel) {
                gro[i] = ro + __popc(m & lt);
                gch[i] = ch + incl - wk;
            }
            ro += __popc(m);
            ch += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    __syncthreads();

    // 5. group words and entry streams
    const uint32_t zero_blk = (uint32_t)a.nnzL;
    if (warp >= a.fill_warps) return;
    uint16_t *list = reinterpret_cast<uint16_t *>(dsm + a.off_list) + 2 * warp * a.ucap, *place = list + a.ucap;
    for (int i = warp; i < ng; i += a.fill_warps) {
        const uint32_t mine = merge(i);
        const int quads = work[i];
        if (lane == 0) {
            uint32_t sl[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) sl[r] = group[i][r] >= 0 ? (uint32_t)group[i][r] : (1u << COL_SLOT_BITS) - 1u;
            uint32_t *out = a.rows + 2 * (a.row_off[p] + gro[i]);
            out[0] = sl[0] | (sl[1] << COL_SLOT_BITS) | (sl[2] << (2 * COL_SLOT_BITS));
            out[1] = sl[3] | ((uint32_t)quads << COL_SLOT_BITS);
        }
        uint32_t *ent = a.ent + (a.chunk_off[p] + gch[i]) * COL_CW;
        auto word = [&](int pl, int r) -> uint32_t & {
            return ent[(pl >> 2) * COL_CW + ((r & 1) * 4 + (pl & 3)) * 2 + (r >> 1)];
        };
        // the merged slots ascending, then eight at a time to their places; the
        // empty places name zero blocks
        const int c = __popc(mine);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += x;
        }
        const int all = __shfl_sync(0xffffffffu, incl, 31);
        int pl = incl - c;
        for (uint32_t m = mine; m; m &= m - 1u, ++pl) list[pl] = (uint16_t)(lane * 32 + __ffs(m) - 1);
        __syncwarp();
        for (int ch = lane; ch < quads / 2; ch += 32) {
            uint8_t at[8];
            unsigned taken = 0u;
            const int n = max(0, min(8, all - 8 * ch));
            col_places(list + 8 * ch, n, at);
            for (int k = 0; k < n; ++k) {
                const int s = list[8 * ch + k];
                place[s] = (uint16_t)(8 * ch + at[k]);
                taken |= 1u << at[k];
#pragma unroll
                for (int x = 0; x < 4; ++x) word(8 * ch + at[k], x) = (zero_blk << COL_SLOT_BITS) | (uint32_t)s;
            }
            for (int k = 0; k < 8; ++k)
                if (!((taken >> k) & 1u))
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        word(8 * ch + k, x) = (zero_blk << COL_SLOT_BITS) | (uint32_t)((k & 3) < nu ? k & 3 : 0);
        }
        __syncwarp();
        for (int x = 0; x < 4 && group[i][x] >= 0; ++x) {
            const int I = ulist[group[i][x]];
            for (int64_t e = a.lrp[I] + lane; e < a.lrp[I + 1]; e += 32) {
                const int sl = rank(a.lci[e]);
                if (sl >= 0) word(place[sl], x) = ((uint32_t)e << COL_SLOT_BITS) | (uint32_t)sl;
            }
        }
        __syncwarp();
    }
}

// off[i] = sum of v[0..i), off[n] = total (one thread block of 1024)
__global__ void __launch_bounds__(1024) k_gp_scan(const int64_t *v, int64_t n, int64_t *off) {
    __shared__ int64_t part[1024];
    const int tid = threadIdx.x;
    const int64_t per = (n + 1023) / 1024, b = min(n, (int64_t)tid * per), e = min(n, b + per);
    int64_t s = 0;
    for (int64_t i = b; i < e; ++i) s += v[i];
    part[tid] = s;
    __syncthreads();
    if (tid == 0) {
        int64_t run = 0;
        for (int i = 0; i < 1024; ++i) {
            const int64_t t = part[i];
            part[i] = run;
            run += t;
        }
        off[n] = run;
    }
    __syncthreads();
    int64_t run = part[tid];
    for (int64_t i = b; i < e; ++i) {
        off[i] = run;
        run += v[i];
    }
}

// ---------------------------------------------------------------------------
// The plan of P_out itself, on the device: checks, transposition map, the
// longest block row.

// first[0]: first row whose row_ptr range is decreasing or leaves [0, nnzb];
// first[1]: first row with a column out of range; first[2]: first row whose
// columns do not strictly ascend; first[3]: first row without its diagonal
// block (nbr where none).  *maxlen: the longest row.
__global__ void k_pc_check(const int64_t *rp, const int32_t *ci, int64_t nbr, int64_t nnzb, int64_t *first,
                           int32_t *maxlen) {
    const int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (I >= nbr) return;
    const int64_t a = rp[I], b = rp[I + 1];
    if (a < 0 || b > nnzb || b < a) {
        atomicMin(reinterpret_cast<long long *>(first), (long long)I);
        return;
    }
    atomicMax(maxlen, (int32_t)(b - a < (int64_t)INT32_MAX ? b - a : (int64_t)INT32_MAX));
    bool diag = false;
    for (int64_t p = a; p < b; ++p) {
        const int32_t c = ci[p];
        if (c < 0 || c >= nbr) {
            atomicMin(reinterpret_cast<long long *>(first + 1), (long long)I);
            return;
        }
        if (p > a && c <= ci[p - 1]) {
            atomicMin(reinterpret_cast<long long *>(first + 2), (long long)I);
            return;
        }
        diag |= c == I;
    }
    if (!diag) atomicMin(reinterpret_cast<long long *>(first + 3), (long long)I);
}

// tperm[p] = position of block (J, I) for block p = (I, J); *bad = the first
// block without a transpose (nnzb where none).  Runs on a checked pattern.
__global__ void k_pc_tperm(const int64_t *rp, const int32_t *ci, int64_t nbr, int64_t nnzb, int32_t *tperm,
                           int64_t *bad) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (p >= nnzb) return;
    const int64_t I = row_of(rp, nbr, p);
    const int64_t q = find_in_row(rp, ci, ci[p], (int32_t)I);
    if (q < 0)
        atomicMin(reinterpret_cast<long long *>(bad), (long long)p);
    else
        tperm[p] = (int32_t)q;
}

// Checks of an operator pattern (n blocks): first[0] rows decreasing or out of
// [0, n] or longer than 65536 blocks; first[1] a column out of range; first[2] columns
// that do not strictly ascend.
__global__ void k_op_check(const int64_t *rp, const int32_t *ci, int64_t nbr, int64_t n, int64_t *first) {
    const int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (I >= nbr) return;
    const int64_t a = rp[I], b = rp[I + 1];
    if (a < 0 || b > n || b < a || b - a > 65536) {
        atomicMin(reinterpret_cast<long long *>(first), (long long)I);
        return;
    }
    for (int64_t p = a; p < b; ++p) {
        if (ci[p] < 0 || ci[p] >= nbr) {
            atomicMin(reinterpret_cast<long long *>(first + 1), (long long)I);
            return;
        }
        if (p > a && ci[p] <= ci[p - 1]) atomicMin(reinterpret_cast<long long *>(first + 2), (long long)I);
    }
}

// Row lists of one panel set (the FP64 step kernel's and the resident
// kernel's): per panel (pairs[2p], pairs[2p+1] = first column, columns), per
// union row in increasing order, the operator row's blocks whose column is in
// the union as (offset in the operator row << 16 | union slot).  Count pass:
// cnt[p] entries, nrow[p] = union rows + 1.  Fill pass: row pointers from
// row_base[p] (global entry offsets from ent_off[p]) and the entries.
template <bool FILL>
__global__ void __launch_bounds__(GP_NT) k_rl_rows(const int64_t *rp, const int32_t *ci, int64_t nbr,
                                                   const int64_t *lrp, const int32_t *lci, const int32_t *pairs,
                                                   int maxu, int64_t *cnt, int64_t *nrow, const int64_t *ent_off,
                                                   const int64_t *row_base, int32_t *lrow_ptr, uint32_t *lent,
                                                   int32_t *err) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ int wsum[32];
    const int tid = threadIdx.x;
    const int64_t p = blockIdx.x;
    const int j0 = pairs[2 * p], nc = pairs[2 * p + 1];
    const int64_t nw = (nbr + 31) / 32;
    uint2 *bits = reinterpret_cast<uint2 *>(dsm);
    int *ulist = reinterpret_cast<int *>(dsm + (((size_t)nw * sizeof(uint2) + 15) & ~(size_t)15));
    for (int64_t w = tid; w < nw; w += GP_NT) bits[w] = make_uint2(0u, 0u);
    __syncthreads();
    for (int q = 0; q < nc; ++q)
        for (int64_t e = rp[j0 + q] + tid; e < rp[j0 + q + 1]; e += GP_NT) {
            const int K = ci[e];
            atomicOr(&bits[K >> 5].x, 1u << (K & 31));
        }
    __syncthreads();
    const int64_t chunk = (nw + GP_NT - 1) / GP_NT;
    const int64_t wb = min(nw, (int64_t)tid * chunk), we = min(nw, wb + chunk);
    int c = 0;
    for (int64_t w = wb; w < we; ++w) c += __popc(bits[w].x);
    int nu;
    int run = block_excl_scan<GP_NWARP>(c, wsum, &nu);
    if (nu > maxu) {  // uniform
        if (tid == 0) atomicExch(err, 1);
        return;
    }
    for (int64_t w = wb; w < we; ++w) {
        unsigned m = bits[w].x;
        bits[w].y = (unsigned)run;
        while (m) {
            const int b = __ffs(m) - 1;
            ulist[run++] = (int)(w * 32 + b);
            m &= m - 1u;
        }
    }
    __syncthreads();
    // thread t takes union rows [u0, u1) in order; a block scan gives offsets
    const int rch = (nu + GP_NT - 1) / GP_NT, u0 = min(nu, tid * rch), u1 = min(nu, u0 + rch);
    int mine = 0;
    for (int u = u0; u < u1; ++u) {
        const int I = ulist[u];
        for (int64_t a = lrp[I]; a < lrp[I + 1]; ++a) mine += rank_of(bits, lci[a]) >= 0;
    }
    int total;
    int off = block_excl_scan<GP_NWARP>(mine, wsum, &total);
    if (!FILL) {
        if (tid == 0) {
            cnt[p] = total;
            nrow[p] = nu + 1;
        }
        return;
    }
    const int64_t e0 = ent_off[p], r0 = row_base[p];
    for (int u = u0; u < u1; ++u) {
        const int I = ulist[u];
        lrow_ptr[r0 + u] = (int32_t)(e0 + off);
        for (int64_t a = lrp[I]; a < lrp[I + 1]; ++a) {
            const int sl = rank_of(bits, lci[a]);
            if (sl >= 0) lent[e0 + off++] = ((uint32_t)(a - lrp[I]) << 16) | (uint32_t)sl;
        }
    }
    if (tid == 0) lrow_ptr[r0 + nu] = (int32_t)(e0 + total);
}

int col_build_device(cheb_plan *plan, const cheb_bsr *L, cudaStream_t s) {
    ColLists c;
    const bool wide = wide_elements(plan->precision);
    c.P = col_width(plan->precision);
    c.NW = COL_NW;
    c.nnzL = L->nnzb;
    c.ucap = col_ucap(c.P);
    const int64_t nbr = plan->nbr, nnzL = L->nnzb;
    if (!col_wanted(plan, nnzL)) return CHEB_ERR_NOSPACE;
    // dynamic shared memory of k_gp_rows; where it is short, fewer warps fill the lists
    // (FP32: all 16 up to about 640,000 block rows, one at 860,000)
    GpArgs a{};
    const size_t nw = (size_t)((nbr + 31) / 32), o_pre = align_up(nw * 4, 16), o_ub = align_up(o_pre + nw * 2, 16),
                 o_list = o_ub + align_up((size_t)c.ucap * ((c.ucap + 31) / 32) * 4, 16);
    size_t dyn = 0;
    for (a.fill_warps = GP_NWARP; a.fill_warps > 0; a.fill_warps /= 2) {
        dyn = o_list + (size_t)a.fill_warps * c.ucap * 4;
        if (dyn + GP_STATIC <= (size_t)CHEB_MAX_DYN_SMEM) break;
    }
    if (a.fill_warps == 0) return CHEB_ERR_NOSPACE;
    a.off_pre = (int)o_pre;
    a.off_ub = (int)o_ub;
    a.off_list = (int)o_list;
    a.ucap = c.ucap;
    // scratch: spans, panels (at most one per column), counts and offsets
    const size_t n1 = (size_t)nbr + 1;
    size_t off = 0;
    auto at = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes);
        return o;
    };
    const size_t o_span = at(nbr * 16), o_pan = at(4 * nbr * 4), o_out = at(8 * 8), o_chunks = at(nbr * 8),
                 o_rows = at(nbr * 8), o_max = at(nbr * 4), o_choff = at(n1 * 8), o_rooff = at(n1 * 8),
                 o_sys = at(plan->h_sys_col.size() * 8);
    char *scr = nullptr;
    CHEB_CUDA(cudaMalloc(&scr, off));
    struct Free {
        char *p;
        ~Free() { cudaFree(p); }
    } free_scr{scr};
    int4 *span = reinterpret_cast<int4 *>(scr + o_span);
    int32_t *pan = reinterpret_cast<int32_t *>(scr + o_pan);
    int64_t *out = reinterpret_cast<int64_t *>(scr + o_out);
    int64_t *cnt_chunks = reinterpret_cast<int64_t *>(scr + o_chunks), *cnt_rows = reinterpret_cast<int64_t *>(scr + o_rows);
    int32_t *cnt_max = reinterpret_cast<int32_t *>(scr + o_max);
    int64_t *choff = reinterpret_cast<int64_t *>(scr + o_choff), *rooff = reinterpret_cast<int64_t *>(scr + o_rooff);
    int64_t *dsys = reinterpret_cast<int64_t *>(scr + o_sys);
    int32_t *err = reinterpret_cast<int32_t *>(out + 4);
    CHEB_CUDA(cudaMemsetAsync(out, 0, 8 * 8, s));
    CHEB_CUDA(cudaMemcpyAsync(dsys, plan->h_sys_col.data(), plan->h_sys_col.size() * 8, cudaMemcpyHostToDevice, s));
    k_gp_spans<<<(unsigned)((nbr + 7) / 8), 256, 0, s>>>(plan->rp, plan->ci, nbr, c.P, c.ucap, INT64_MAX, dsys, plan->nsys, span);
    k_gp_panels<<<1, GP_NT, 0, s>>>(span, nbr, pan, nullptr, out);
    CHEB_TRY(check_launch("k_gp_panels", 2));
    int64_t h_out[3];
    CHEB_CUDA(cudaMemcpyAsync(h_out, out, sizeof(h_out), cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    if (h_out[2]) return CHEB_ERR_NOSPACE;  // a single column does not fit: no column kernel
    const int64_t np = h_out[0];
    c.n_panels = np;
    c.max_union = (int32_t)h_out[1];
    a.rp = plan->rp;
    a.ci = plan->ci;
    a.nbr = nbr;
    a.lrp = L->row_ptr;
    a.lci = L->col_idx;
    a.nnzL = nnzL;
    a.panels = pan;
    a.cnt_chunks = cnt_chunks;
    a.cnt_rows = cnt_rows;
    a.cnt_maxrow = cnt_max;
    a.err = err;
    CHEB_TRY(allow_shared(k_gp_rows<false>));
    CHEB_TRY(allow_shared(k_gp_rows<true>));
    k_gp_rows<false><<<(unsigned)np, GP_NT, dyn, s>>>(a);
    CHEB_TRY(check_launch("k_gp_rows count"));
    k_gp_scan<<<1, 1024, 0, s>>>(cnt_chunks, np, choff);
    k_gp_scan<<<1, 1024, 0, s>>>(cnt_rows, np, rooff);
    CHEB_TRY(check_launch("k_gp_scan", 2));
    std::vector<int32_t> h_max(np);
    std::vector<int32_t> h_pan(4 * np);
    std::vector<int64_t> h_quads(np);
    int64_t tot[2];
    int32_t h_err = 0;
    CHEB_CUDA(cudaMemcpyAsync(h_max.data(), cnt_max, np * 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(h_quads.data(), cnt_chunks, np * 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(h_pan.data(), pan, 4 * np * 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(&tot[0], choff + np, 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(&tot[1], rooff + np, 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    if (h_err) return fail(CHEB_ERR_INVALID, "gather plan: inconsistent panel union (code %d)", h_err);
    for (const int32_t m : h_max) c.max_row = std::max(c.max_row, m);
    if ((tot[0] + COL_TAIL) * COL_CW >= (int64_t)INT32_MAX || (wide && c.max_row > COL_MAX_QUADS64)) return CHEB_ERR_NOSPACE;
    c.n_entries = (tot[0] + COL_TAIL) * COL_CW;
    c.n_rows = 2 * tot[1];
    c.n_slot = plan->nnzb;
    c.h_sys_panel.assign(plan->nsys + 1, (int32_t)np);
    for (int64_t p = np - 1; p >= 0; --p) c.h_sys_panel[h_pan[4 * p + 3]] = (int32_t)p;
    c.n_sys = (int64_t)c.h_sys_panel.size();
    c.h_order = col_order(h_quads);
    // the lists, in device memory of their own until cheb_plan_bind_operator
    // copies them into the operator workspace
    c.built = true;  // (sizes complete: bytes() counts them from here on)
    const size_t nbytes = c.bytes();
    CHEB_CUDA(cudaMalloc(&c.tmp, nbytes));
    struct FreeOnError {
        ColLists &c;
        bool armed = true;
        ~FreeOnError() {
            if (armed) col_free(c);
        }
    } guard{c};
    Carve cv(c.tmp, nbytes);
    c.d_panels = cv.take<int32_t>(4 * np);
    c.d_wchunk = cv.take<int32_t>(np * (COL_NW + 1));
    c.d_wrow = cv.take<int32_t>(np * (COL_NW + 1));
    c.d_rows = cv.take<uint32_t>(std::max<int64_t>(c.n_rows, 1));
    c.d_ent = cv.take<uint32_t>(std::max<int64_t>(c.n_entries, 1));
    c.d_slot = cv.take<uint16_t>(c.n_slot);
    c.d_sys_panel = cv.take<int32_t>(c.n_sys);
    c.d_order = cv.take<int32_t>(np);
    CHEB_CUDA(cudaMemcpyAsync(c.d_sys_panel, c.h_sys_panel.data(), c.n_sys * 4, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_order, c.h_order.data(), np * 4, cudaMemcpyHostToDevice, s));
    CHEB_CUDA(cudaMemcpyAsync(c.d_panels, pan, 4 * np * 4, cudaMemcpyDeviceToDevice, s));
    CHEB_CUDA(cudaMemsetAsync(c.d_ent + tot[0] * COL_CW, 0, COL_TAIL * COL_CW * 4, s));
    a.chunk_off = choff;
    a.row_off = rooff;
    a.wchunk = c.d_wchunk;
    a.wrow = c.d_wrow;
    a.rows = c.d_rows;
    a.ent = c.d_ent;
    a.slot = c.d_slot;
    k_gp_rows<true><<<(unsigned)np, GP_NT, dyn, s>>>(a);
    CHEB_TRY(check_launch("k_gp_rows fill"));
    CHEB_CUDA(cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    if (h_err) return fail(CHEB_ERR_INVALID, "gather plan: inconsistent row lists (code %d)", h_err);
    c.device = true;
    guard.armed = false;
    plan->col = std::move(c);
    return CHEB_OK;
}

}  // namespace cheb

namespace cheb {

// ---------------------------------------------------------------------------
// Host-side launchers of the plan kernels (plan.cu drives them).

int gp_check_pattern(const int64_t *rp, const int32_t *ci, int64_t nbr, int64_t nnzb, int64_t first[4],
                     int32_t *maxlen, cudaStream_t s) {
    int64_t *d = nullptr;
    CHEB_CUDA(cudaMallocAsync(&d, 5 * 8, s));
    const int64_t init[5] = {nbr, nbr, nbr, nbr, 0};
    CHEB_CUDA(cudaMemcpyAsync(d, init, sizeof(init), cudaMemcpyHostToDevice, s));
    k_pc_check<<<(unsigned)((nbr + 255) / 256), 256, 0, s>>>(rp, ci, nbr, nnzb, d,
                                                           reinterpret_cast<int32_t *>(d + 4));
    const int rc = check_launch("k_pc_check");
    int64_t h[5] = {0, 0, 0, 0, 0};
    if (rc == CHEB_OK) CHEB_CUDA(cudaMemcpyAsync(h, d, sizeof(h), cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaFreeAsync(d, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    CHEB_TRY(rc);
    for (int i = 0; i < 4; ++i) first[i] = h[i];
    int32_t ml;
    std::memcpy(&ml, &h[4], 4);
    *maxlen = ml;
    return CHEB_OK;
}

int gp_tperm(const int64_t *rp, const int32_t *ci, int64_t nbr, int64_t nnzb, int32_t *tperm, int64_t *bad,
             cudaStream_t s) {
    int64_t *d = nullptr;
    CHEB_CUDA(cudaMallocAsync(&d, 8, s));
    CHEB_CUDA(cudaMemcpyAsync(d, &nnzb, 8, cudaMemcpyHostToDevice, s));
    k_pc_tperm<<<(unsigned)((nnzb + 255) / 256), 256, 0, s>>>(rp, ci, nbr, nnzb, tperm, d);
    const int rc = check_launch("k_pc_tperm");
    if (rc == CHEB_OK) CHEB_CUDA(cudaMemcpyAsync(bad, d, 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaFreeAsync(d, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    return rc;
}

int gp_walk(const int64_t *rp, const int32_t *ci, int64_t nbr, int P, int64_t ucap, int64_t bcap,
            const std::vector<int64_t> &sys_col, std::vector<int32_t> &panels4, std::vector<int32_t> &aux,
            int64_t out[4], cudaStream_t s) {
    const int nsys = (int)sys_col.size() - 1;
    size_t off = 0;
    auto at = [&](size_t bytes) {
        const size_t o = off;
        off = align_up(off + bytes);
        return o;
    };
    const size_t o_span = at(nbr * 16), o_pan = at(4 * nbr * 4), o_aux = at(2 * nbr * 4), o_out = at(4 * 8),
                 o_sys = at(sys_col.size() * 8);
    char *scr = nullptr;
    CHEB_CUDA(cudaMalloc(&scr, off));
    struct Free {
        char *p;
        ~Free() { cudaFree(p); }
    } free_scr{scr};
    int4 *span = reinterpret_cast<int4 *>(scr + o_span);
    int32_t *pan = reinterpret_cast<int32_t *>(scr + o_pan), *ax = reinterpret_cast<int32_t *>(scr + o_aux);
    int64_t *dout = reinterpret_cast<int64_t *>(scr + o_out), *dsys = reinterpret_cast<int64_t *>(scr + o_sys);
    CHEB_CUDA(cudaMemsetAsync(dout, 0, 4 * 8, s));
    CHEB_CUDA(cudaMemcpyAsync(dsys, sys_col.data(), sys_col.size() * 8, cudaMemcpyHostToDevice, s));
    k_gp_spans<<<(unsigned)((nbr + 7) / 8), 256, 0, s>>>(rp, ci, nbr, P, ucap, bcap, dsys, nsys, span);
    k_gp_panels<<<1, GP_NT, 0, s>>>(span, nbr, pan, ax, dout);
    CHEB_TRY(check_launch("k_gp_panels", 2));
    CHEB_CUDA(cudaMemcpyAsync(out, dout, 4 * 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    if (out[2]) return CHEB_OK;  // the caller reports the column that does not fit
    panels4.resize(4 * out[0]);
    aux.resize(2 * out[0]);
    CHEB_CUDA(cudaMemcpyAsync(panels4.data(), pan, panels4.size() * 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(aux.data(), ax, aux.size() * 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    return CHEB_OK;
}

int gp_check_operator(const cheb_bsr *L, int64_t nbr, int64_t first[3], cudaStream_t s) {
    int64_t *d = nullptr;
    CHEB_CUDA(cudaMallocAsync(&d, 3 * 8, s));
    const int64_t init[3] = {nbr, nbr, nbr};
    CHEB_CUDA(cudaMemcpyAsync(d, init, sizeof(init), cudaMemcpyHostToDevice, s));
    k_op_check<<<(unsigned)((nbr + 255) / 256), 256, 0, s>>>(L->row_ptr, L->col_idx, nbr, L->nnzb, d);
    const int rc = check_launch("k_op_check");
    if (rc == CHEB_OK) CHEB_CUDA(cudaMemcpyAsync(first, d, 3 * 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaFreeAsync(d, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    return rc;
}

int row_lists_device(const int64_t *rp, const int32_t *ci, int64_t nbr, const cheb_bsr *L, const int32_t *pairs,
                     int64_t np, int maxu, RowLists &out, cudaStream_t s) {
    if (np == 0) return CHEB_OK;
    const size_t dyn = (((size_t)((nbr + 31) / 32) * sizeof(uint2) + 15) & ~(size_t)15) + (size_t)maxu * 4;
    if (dyn > (size_t)CHEB_MAX_DYN_SMEM - 2048)
        return fail(CHEB_ERR_NOSPACE, "cheb_plan_attach_operator: %zu bytes of panel bitmap and union", dyn);
    CHEB_TRY(allow_shared(k_rl_rows<false>));
    CHEB_TRY(allow_shared(k_rl_rows<true>));
    int64_t *scr = nullptr;  // cnt, nrow [np]; ent_off, row_base [np + 1]; error flag
    CHEB_CUDA(cudaMalloc(&scr, (4 * np + 3) * 8));
    struct Free {
        int64_t *p;
        ~Free() { cudaFree(p); }
    } free_scr{scr};
    int64_t *cnt = scr, *nrow = scr + np, *ent_off = scr + 2 * np, *row_base = scr + 3 * np + 1;
    int32_t *err = reinterpret_cast<int32_t *>(scr + 4 * np + 2);
    CHEB_CUDA(cudaMemsetAsync(err, 0, 4, s));
    k_rl_rows<false><<<(unsigned)np, GP_NT, dyn, s>>>(rp, ci, nbr, L->row_ptr, L->col_idx, pairs, maxu, cnt, nrow,
                                                      nullptr, nullptr, nullptr, nullptr, err);
    k_gp_scan<<<1, 1024, 0, s>>>(cnt, np, ent_off);
    k_gp_scan<<<1, 1024, 0, s>>>(nrow, np, row_base);
    CHEB_TRY(check_launch("row lists count", 3));
    int64_t tot[2];
    int32_t h_err = 0;
    CHEB_CUDA(cudaMemcpyAsync(&tot[0], ent_off + np, 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(&tot[1], row_base + np, 8, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaMemcpyAsync(&h_err, err, 4, cudaMemcpyDeviceToHost, s));
    CHEB_CUDA(cudaStreamSynchronize(s));
    if (h_err) return fail(CHEB_ERR_INVALID, "cheb_plan_attach_operator: panel union above the plan's maximum");
    if (tot[0] >= (int64_t)INT32_MAX)
        return fail(CHEB_ERR_NOSPACE, "cheb_plan_attach_operator: %lld list entries exceed the int32 offsets",
                    (long long)tot[0]);
    out.device = true;
    out.n_base = np;
    out.n_ptr = tot[1];
    out.n_ent = tot[0];
    CHEB_CUDA(cudaMalloc(&out.tmp, out.bytes()));
    Carve cv(out.tmp, out.bytes());
    out.d_base = cv.take<int64_t>(np);
    out.d_ptr = cv.take<int32_t>(std::max<int64_t>(out.n_ptr, 1));
    out.d_ent = cv.take<uint32_t>(std::max<int64_t>(out.n_ent, 1));
    CHEB_CUDA(cudaMemcpyAsync(out.d_base, row_base, np * 8, cudaMemcpyDeviceToDevice, s));
    k_rl_rows<true><<<(unsigned)np, GP_NT, dyn, s>>>(rp, ci, nbr, L->row_ptr, L->col_idx, pairs, maxu, nullptr,
                                                     nullptr, ent_off, row_base, out.d_ptr, out.d_ent, err);
    CHEB_TRY(check_launch("row lists fill"));
    CHEB_CUDA(cudaStreamSynchronize(s));
    return CHEB_OK;
}

}  // namespace cheb
