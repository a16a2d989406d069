// gather_plan.cu -- the lists of the gather assembly (gather.cuh), one block per
// patch.  A block stages its owned rows' columns in shared memory, finds every
// closure pair's entry there, counts the contributions of each entry, lists them,
// and sorts each entry's short list, so that the lists do not depend on the order in
// which the atomics were served.  The closure's element order is the colour order of
// the scatter kernels, so an entry is the same sum, bit for bit, on either path.
#include <algorithm>
#include <type_traits>

#include "block_prims.cuh"
#include "elem_ops.cuh"
#include "gather.cuh"
#include "mesh.cuh"
#include "phases.cuh"

namespace fem {

struct GatherPlanSmem {
    size_t col, gid, own, roff, rows, cnt, start, lst, cw, ln, rp, pe, total;
};

static size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }

static GatherPlanSmem gather_plan_smem(const Plan &P, const Closure &cl, int npe) {
    GatherPlanSmem L{};
    const size_t n = (size_t)std::max(P.max_acc, P.max_own) + 16;
    size_t o = 0;
    L.col = o;
    o = up16(o + n * 4);
    L.gid = o;
    o = up16(o + (size_t)cl.max_cnodes * 4);
    L.own = o;
    o = up16(o + (size_t)cl.max_cnodes * 2);
    L.roff = o;
    o = up16(o + (size_t)(P.max_own + 1) * 4);
    L.rows = o;
    o = up16(o + (size_t)(P.max_own + 1) * 4);
    L.cnt = o;
    o = up16(o + n * 4);
    L.start = o;
    o = up16(o + n * 4);
    L.lst = o;
    o = up16(o + (size_t)cl.max_celems * (npe * (npe - 1) / 2 > npe ? npe * (npe - 1) / 2 : npe) * 2);
    L.cw = o;
    o = up16(o + (n / 32 + 2) * 4);
    L.ln = o;
    o = up16(o + (size_t)cl.max_celems * npe * 2);
    L.rp = o;
    o = up16(o + (size_t)P.max_own * 8);
    L.pe = o;
    o = up16(o + (size_t)cl.max_celems * (npe * (npe - 1) / 2) * 2);
    L.total = o;
    return L;
}

// Sorts the lists of n entries (list k: lst[start[k] .. start[k] + cnt[k])) and sets
// cw[chunk] to the words a lane of the chunk needs (half the longest list of its 32
// entries, rounded up).
__device__ static void sort_lists(uint16_t *lst, const int *start, const int *cnt, int n, int *cw) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int c = warp; 32 * c < n; c += nw) {
        const int k = 32 * c + lane;
        int m = 0;
        if (k < n) {
            m = cnt[k];
            uint16_t *l = lst + start[k];
            for (int i = 1; i < m; ++i) {
                const uint16_t v = l[i];
                int j = i - 1;
                for (; j >= 0 && l[j] > v; --j) l[j + 1] = l[j];
                l[j + 1] = v;
            }
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) cw[c] = (m + 1) / 2;
    }
}

// The chunk words of n entries from word offset `at` of the block on.
__device__ static void write_words(uint32_t *out, const int *off, const int *cw, const uint16_t *lst, const int *start,
                                   const int *cnt, int n, uint32_t zero) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int c = warp; 32 * c < n; c += nw) {
        const int k = 32 * c + lane, m = k < n ? cnt[k] : 0, b = k < n ? start[k] : 0;
        for (int w = 0; w < cw[c]; ++w) {
            const uint32_t lo = 2 * w < m ? lst[b + 2 * w] : zero, hi = 2 * w + 1 < m ? lst[b + 2 * w + 1] : zero;
            out[off[c] + 32 * w + lane] = lo | (hi << 16);
        }
    }
}

template <int NPE>
__device__ __forceinline__ void load_lnodes_smem(const uint16_t *s, int i, uint16_t (&ln)[NPE]) {
    if constexpr (NPE == 8) {
        const uint4 v = reinterpret_cast<const uint4 *>(s)[i];
        ln[0] = v.x & 0xffff; ln[1] = v.x >> 16; ln[2] = v.y & 0xffff; ln[3] = v.y >> 16;
        ln[4] = v.z & 0xffff; ln[5] = v.z >> 16; ln[6] = v.w & 0xffff; ln[7] = v.w >> 16;
    } else {
        const uint2 v = reinterpret_cast<const uint2 *>(s)[i];
        ln[0] = v.x & 0xffff; ln[1] = v.x >> 16; ln[2] = v.y & 0xffff; ln[3] = v.y >> 16;
    }
}

template <int NPE>
__global__ void __launch_bounds__(512) k_gather_lists(PlanView pv, const int32_t *__restrict__ col, GatherPlanSmem L,
                                                      int top_step,
                                                      uint32_t zero, GatherPatch *__restrict__ patch,
                                                      uint32_t *__restrict__ words, unsigned long long *cursor,
                                                      unsigned long long cap, unsigned long long *empty_row) {
    constexpr int NP = ElemTraits<NPE>::NP;
    extern __shared__ __align__(16) unsigned char gp_smem[];
    int32_t *s_col = reinterpret_cast<int32_t *>(gp_smem + L.col);
    int32_t *s_gid = reinterpret_cast<int32_t *>(gp_smem + L.gid);
    int16_t *s_own = reinterpret_cast<int16_t *>(gp_smem + L.own);
    int *s_roff = reinterpret_cast<int *>(gp_smem + L.roff);
    int *s_rows = reinterpret_cast<int *>(gp_smem + L.rows);
    int *cnt = reinterpret_cast<int *>(gp_smem + L.cnt);
    int *start = reinterpret_cast<int *>(gp_smem + L.start);
    uint16_t *lst = reinterpret_cast<uint16_t *>(gp_smem + L.lst);
    int *cw = reinterpret_cast<int *>(gp_smem + L.cw);
    uint16_t *s_ln = reinterpret_cast<uint16_t *>(gp_smem + L.ln);
    int64_t *s_rp = reinterpret_cast<int64_t *>(gp_smem + L.rp);
    uint16_t *s_pe = reinterpret_cast<uint16_t *>(gp_smem + L.pe);  // each off-diagonal pair's entry (0xffff: not owned)
    __shared__ int ws[32];
    __shared__ int64_t s_base;
    const int tid = threadIdx.x, nthr = blockDim.x;
    for (int64_t p = blockIdx.x; p < pv.n_patches; p += gridDim.x) {
        GatherPatch d{};
        d.nb = pv.patch_node_ptr[p], d.n_own = (int)(pv.patch_node_ptr[p + 1] - d.nb);
        d.cb = pv.patch_cnode_ptr[p], d.n_cnodes = (int)(pv.patch_cnode_ptr[p + 1] - d.cb);
        d.eb = pv.patch_elem_ptr[p], d.n_elems = (int)(pv.patch_elem_ptr[p + 1] - d.eb);
        const int nacc = pv.patch_acc[p];
        d.n_off = nacc - d.n_own;  // every row ends with its diagonal
        const int nch = d.n_chunks();
        for (int j = tid; j < d.n_cnodes; j += nthr) {
            s_gid[j] = pv.cnode_gid[d.cb + j];
            s_own[j] = (int16_t)pv.cnode_own[d.cb + j];
        }
        for (int k = tid; k < d.n_own; k += nthr) {
            s_roff[k] = pv.own_acc[d.nb + k];
            s_rp[k] = pv.own_rowptr[d.nb + k];
        }
        using Row = typename std::conditional<NPE == 8, uint4, uint2>::type;  // an element's local nodes
        for (int i = tid; i < d.n_elems; i += nthr)
            reinterpret_cast<Row *>(s_ln)[i] = __ldg(reinterpret_cast<const Row *>(pv.celem_lnode) + d.eb + i);
        if (tid == 0) s_roff[d.n_own] = nacc;
        for (int i = tid; i < d.n_off; i += nthr) cnt[i] = 0;
        __syncthreads();
        // columns of the owned rows, and which rows have off-diagonals
        bool empty = false;  // a node of no element: a row without its diagonal
#pragma unroll 4
        for (int k = tid / 8; k < d.n_own; k += nthr / 8) {
            const int o = s_roff[k], len = s_roff[k + 1] - o, j = tid & 7;
            const int32_t *src = col + s_rp[k];
            if (j < len) s_col[o + j] = __ldg(src + j);
            if (j + 8 < len) s_col[o + j + 8] = __ldg(src + j + 8);
            for (int l = j + 16; l < len; l += 8) s_col[o + l] = __ldg(src + l);
            if (j == 0) s_rows[k] = len > 1;
            empty = empty || len < 1;
        }
        if (__syncthreads_or(empty)) {
            if (tid == 0) *empty_row = 1;  // the caller drops the lists
            return;
        }
        d.n_rows = block_scan(s_rows, d.n_own, ws);
        // every off-diagonal pair's entry among the owned off-diagonals, counted and kept
        constexpr int PAIRS = NPE * (NPE - 1) / 2;
        {
            for (int i = tid; i < d.n_elems; i += nthr) {
                uint16_t ln[NPE];
                load_lnodes_smem<NPE>(s_ln, i, ln);
                int g[NPE], own[NPE];
#pragma unroll
                for (int a = 0; a < NPE; ++a) g[a] = s_gid[ln[a]], own[a] = s_own[ln[a]];
                // binary searches of a fixed number of steps, a few pairs side by side
                // (one pair at a time, each step waits for the one before)
                constexpr int B = NPE == 8 ? 7 : 6;
                int a0 = 1, b0 = 0;
#pragma unroll
                for (int g0 = 0; g0 < PAIRS; g0 += B) {
                    int k[B], gc[B], at[B], end[B];
#pragma unroll
                    for (int j = 0; j < B; ++j) {
                        const bool up = g[a0] > g[b0];
                        k[j] = up ? own[a0] : own[b0];
                        gc[j] = up ? g[b0] : g[a0];
                        at[j] = k[j] >= 0 ? s_roff[k[j]] : 0;
                        end[j] = k[j] >= 0 ? s_roff[k[j] + 1] : 1;
                        if (++b0 == a0) ++a0, b0 = 0;
                    }
                    for (int step = top_step; step > 0; step >>= 1)
#pragma unroll
                        for (int j = 0; j < B; ++j) {
                            const int mid = at[j] + step;
                            if (mid < end[j] && s_col[mid] <= gc[j]) at[j] = mid;
                        }
#pragma unroll
                    for (int j = 0; j < B; ++j)
                    {
                        const int e = k[j] >= 0 ? at[j] - k[j] : 0xffff;
                        s_pe[i * PAIRS + g0 + j] = (uint16_t)e;
                        if (k[j] >= 0) atomicAdd(&cnt[e], 1);
                    }
                }
            }
        }
        __syncthreads();
        for (int i = tid; i < d.n_off; i += nthr) start[i] = cnt[i];
        __syncthreads();
        block_scan(start, d.n_off, ws);
        for (int i = tid; i < d.n_off; i += nthr) cnt[i] = 0;
        __syncthreads();
        for (int i = tid; i < d.n_elems; i += nthr) {
            const uint16_t *pe = s_pe + i * PAIRS;
#pragma unroll
            for (int a = 1; a < NPE; ++a)
#pragma unroll
                for (int b = 0; b < a; ++b) {
                    const int e = pe[a * (a - 1) / 2 + b];
                    if (e != 0xffff) lst[start[e] + atomicAdd(&cnt[e], 1)] = (uint16_t)(i * NP + a * (a + 1) / 2 + b);
                }
        }
        __syncthreads();
        sort_lists(lst, start, cnt, d.n_off, cw);
        __syncthreads();
        // the block's size: tables, then the words of the off-diagonals and the diagonals
        int *off = s_col;  // the columns are done with: chunk offsets
        for (int c = tid; c < nch; c += nthr) off[c] = 32 * cw[c];
        __syncthreads();
        const int wtot = block_scan(off, nch, ws);
        const int ndc = d.n_diag();
        const int row_at = 4 * (nch + ndc), dst_at = row_at + 2 * d.n_rows, idx_at = dst_at + 2 * d.n_own;
        int *doff = off + nch + 1, *dcw = doff + ndc + 1;
        int *inc = s_gid;  // the closure ids are done with (every owned node is a closure node)
        for (int k = tid; k < d.n_own; k += nthr) inc[k] = 0;
        __syncthreads();
        auto each_node = [&](auto &&f) {
            for (int i = tid; i < d.n_elems; i += nthr) {
                uint16_t ln[NPE];
                load_lnodes_smem<NPE>(s_ln, i, ln);
#pragma unroll
                for (int a = 0; a < NPE; ++a) {
                    const int k = s_own[ln[a]];
                    if (k >= 0) f(k, i * NP + a * (a + 3) / 2);
                }
            }
        };
        each_node([&](int k, int) { atomicAdd(&inc[k], 1); });
        __syncthreads();
        for (int c = tid >> 5; c < ndc; c += nthr >> 5) {
            const int k = 32 * c + (tid & 31);
            const int m = __reduce_max_sync(0xffffffffu, k < d.n_own ? inc[k] : 0);
            if ((tid & 31) == 0) dcw[c] = (m + 1) / 2, doff[c] = 32 * ((m + 1) / 2);
        }
        __syncthreads();
        const int dtot = block_scan(doff, ndc, ws);
        const int total = (idx_at + wtot + dtot + 3) & ~3;
        d.n_words = total;
        if (tid == 0) s_base = (int64_t)atomicAdd(cursor, (unsigned long long)total);
        __syncthreads();
        d.list = s_base;
        if (tid == 0) patch[p] = d;
        if ((unsigned long long)(s_base + total) <= cap) {  // else the caller sees the cursor and calls again
            uint32_t *B = words + s_base;
            int64_t *rowd = reinterpret_cast<int64_t *>(B + row_at), *diag = reinterpret_cast<int64_t *>(B + dst_at);
            // (s_rows[k]: the rows with off-diagonals before row k)
            for (int k = tid; k < d.n_own; k += nthr) {
                const int64_t rp = s_rp[k];
                const int len = s_roff[k + 1] - s_roff[k];
                diag[k] = rp + len - 1;
                if (len > 1) rowd[s_rows[k]] = rp - (s_roff[k] - k);
            }
            uint4 *tab = reinterpret_cast<uint4 *>(B);
            for (int c = tid; c < nch; c += nthr) {
                // the row holding entry 32 c: the last one that starts at or before it
                int lo = 0, hi = d.n_own - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_roff[mid] - mid <= 32 * c) lo = mid; else hi = mid - 1;
                }
                uint32_t marks = 1;
                for (int k = lo + 1; k < d.n_own && s_roff[k] - k < 32 * c + 32; ++k)
                    if (s_roff[k + 1] - s_roff[k] > 1) marks |= 1u << (s_roff[k] - k - 32 * c);
                tab[c] = make_uint4((uint32_t)(idx_at + off[c]), (uint32_t)cw[c], (uint32_t)s_rows[lo], marks);
            }
            for (int c = tid >> 5; c < ndc; c += nthr >> 5) {
                const int k = 32 * c + (tid & 31);
                const uint32_t hv = __ballot_sync(0xffffffffu, k < d.n_own && pv.own_hv[d.nb + k] != 0);
                if ((tid & 31) == 0)
                    tab[nch + c] = make_uint4((uint32_t)(idx_at + wtot + doff[c]), (uint32_t)dcw[c], 0u, hv);
            }
            write_words(B + idx_at, off, cw, lst, start, cnt, d.n_off, zero);
            __syncthreads();
            // diagonals: the same over the owned nodes
            for (int k = tid; k < d.n_own; k += nthr) start[k] = inc[k];
            __syncthreads();
            block_scan(start, d.n_own, ws);
            for (int k = tid; k < d.n_own; k += nthr) cnt[k] = 0;
            __syncthreads();
            each_node([&](int k, int q) { lst[start[k] + atomicAdd(&cnt[k], 1)] = (uint16_t)q; });
            __syncthreads();
            sort_lists(lst, start, cnt, d.n_own, cw);
            __syncthreads();
            write_words(B + idx_at + wtot, doff, cw, lst, start, cnt, d.n_own, zero);
        }
        __syncthreads();
    }
}

// The largest layout is the fused FP64 one (the batched FP64 builds), and positions are
// 16-bit.  A closure holds at least the nodes its patch owns.
bool lists_fit(fem_mesh m, const Closure &cl) {
    const Plan &P = m->plan;
    int dev = 0, limit = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    GatherMax gm;
    gm.max_acc = P.max_acc, gm.max_own = P.max_own;
    gm.max_cnodes = std::max(cl.max_cnodes, P.max_own), gm.max_celems = cl.max_celems;
    return cl.max_celems * m->np < 65536 && P.max_own < 32767 &&
           gather_smem_layout(gm, m->npe, true, 8, 8, 8).total + 1024 <= (size_t)limit &&
           gather_plan_smem(P, cl, m->npe).total + 1024 <= (size_t)limit;
}

// Builds the lists of the full closure (all patches); leaves lists.ready false when
// the patches are out of the gather kernels' range.  FEM_ERR_BUDGET if the budget
// cannot hold them.
fem_status build_gather_lists(fem_mesh m, Closure &cl, cudaStream_t s) {
    Plan &P = m->plan;
    GatherLists &G = cl.lists;
    G.free();
    const GatherPlanSmem L = gather_plan_smem(P, cl, m->npe);
    P.max_cnodes = cl.max_cnodes, P.max_celems = cl.max_celems;
    if (cl.total_celems == 0 || !lists_fit(m, cl)) return FEM_OK;
    const int64_t np_ = cl.p1 - cl.p0;
    const int np = m->npe * (m->npe + 1) / 2;
    G.zero = (int)(cl.max_celems * np);
    FEM_TRY(G.patch.alloc(m->arena, np_, "gather patches"));
    DevBuf<unsigned long long> cursor;
    FEM_TRY(cursor.alloc(m->arena, 2, "gather list cursor"));
    // About: an off-diagonal entry of a brick mesh takes two words (an edge of four
    // bricks), of a tetrahedral mesh three to four, a diagonal half the incidence.
    const size_t off = (size_t)(m->nnz - m->n_nodes), N = (size_t)m->n_nodes;
    size_t cap = off * (m->npe == 8 ? 2 : 4) + N * (m->npe == 8 ? 4 : 16) + off / 8 + 6 * N + 512 * (size_t)np_;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(np_, (int64_t)num_sms() * 4));
    int top_step = 1;  // the largest power of two below the longest row's length
    while (2 * top_step < m->max_row_len) top_step *= 2;
    auto f = m->npe == 8 ? k_gather_lists<8> : k_gather_lists<4>;
    FEM_CUDA(allow_smem(f, L.total));
    for (int pass = 0; pass < 2; ++pass) {
        FEM_TRY(G.words.alloc(m->arena, cap, "gather lists"));
        FEM_CUDA(cudaMemsetAsync(cursor.ptr, 0, 2 * sizeof(unsigned long long), s));
        f<<<grid, 512, L.total, s>>>(P.view(cl), m->col.ptr, L, top_step, (uint32_t)G.zero, G.patch.ptr, G.words.ptr, cursor.ptr,
                                     cap, cursor.ptr + 1);
        FEM_LAUNCHED("k_gather_lists");
        unsigned long long h[2] = {0, 0};
        FEM_CUDA(cudaMemcpyAsync(h, cursor.ptr, sizeof(h), cudaMemcpyDeviceToHost, s));
        FEM_CUDA(cudaStreamSynchronize(s));
        const unsigned long long used = h[0];
        if (h[1]) {
            G.free();
            return FEM_OK;
        }
        if (used <= cap) {
            G.ready = true;
            return FEM_OK;
        }
        G.words.free();
        cap = used;  // the first pass wrote what fitted and counted the rest
    }
    set_error("gather lists outgrew their second allocation");
    return FEM_ERR_CUDA;
}

}  // namespace fem
