// gather.cu -- the gather assembly: builds of K without accumulators or colours.
//
// A block integrates every element of its patch's closure into shared memory (or
// copies the staged element matrices there), and after one barrier each owned CSR
// entry is summed by one thread from the patch's lists (gather.cuh) and stored
// straight to its place: consecutive lanes hold consecutive entries of the rows.
//
// What bounds it, and why this form.  The scatter it replaces (numeric.cu's k_patch)
// spent, of 226 us on 1M bricks, 34 us ordering its colour phases, 30 us in
// read-modify-write adds with random bank conflicts (17 M shared-memory wavefronts,
// 54 us of that pipe), 27 us waiting for the adds' targets and 38 us writing rows
// four lanes at a time (8 cache lines a store instruction).  Here an element matrix
// leaves a thread in nine conflict-free 16-byte stores, an entry is read 2.5 times
// on average and never written back, a store instruction covers about four lines,
// and a block passes two barriers a patch.  While the entries of one patch are
// summed, cp.async brings the next patch's coordinates and coefficients.  Patches are
// smaller than the scatter's (the matrices of 500 bricks fill half an SM's shared
// memory), so more border elements are integrated twice; on balance 1M bricks went
// from 228 to 167 us, 27M from 4.87 to 3.75 ms, 512 meshes in one launch from 3.17 to
// 2.66 ms, 3.07M tetrahedra from 160 to 146 us, and the assembly of 1M bricks' FP64
// matrices from 0.36 to 0.28 ms.  What bounds it now: latency at 16 warps an SM (113
// registers; 20 or 24 warps at 96 or 80 registers measured slower), about two thirds
// of it in the integration.
#include "elem_ops.cuh"
#include "gather.cuh"
#include "mesh.cuh"
#include "numeric.cuh"
#include "phases.cuh"

namespace fem {

__device__ __forceinline__ void g_cp4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void g_cp8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void g_cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void g_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Asks L2 for [p, p + bytes) (rounded inwards to 16-byte units).
__device__ __forceinline__ void g_prefetch(const void *p, size_t bytes) {
    const uint64_t a = (reinterpret_cast<uint64_t>(p) + 15) & ~15ull, e = (reinterpret_cast<uint64_t>(p) + bytes) & ~15ull;
    if (e > a)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(e - a)) : "memory");
}
template <typename T>
__device__ __forceinline__ void g_cp(T *dst, const T *src) {
    if constexpr (sizeof(T) == 4) g_cp4(dst, src);
    else g_cp8(dst, src);
}

// One element matrix to its row of shared memory, in the widest stores its stride
// allows (36 floats or doubles and 10 doubles: 16 bytes; 10 floats: 8 bytes).  The
// strides of 36 and 10 words put the lanes of a store's phase on distinct banks.
template <int NP>
__device__ __forceinline__ void put_matrix(float *dst, const float (&k)[NP]) {
    if constexpr (NP % 4 == 0) {
#pragma unroll
        for (int w = 0; w < NP / 4; ++w)
            reinterpret_cast<float4 *>(dst)[w] = make_float4(k[4 * w], k[4 * w + 1], k[4 * w + 2], k[4 * w + 3]);
    } else {
#pragma unroll
        for (int w = 0; w < NP / 2; ++w) reinterpret_cast<float2 *>(dst)[w] = make_float2(k[2 * w], k[2 * w + 1]);
    }
}
template <int NP>
__device__ __forceinline__ void put_matrix(double *dst, const double (&k)[NP]) {
#pragma unroll
    for (int w = 0; w < NP / 2; ++w) reinterpret_cast<double2 *>(dst)[w] = make_double2(k[2 * w], k[2 * w + 1]);
}

// What a patch needs of its mesh's plan, read once a patch (from a batch's table the
// fields would be loaded again after every store).
struct PatchPlan {
    const uint16_t *lnode;  // the patch's first element's local nodes
    const uint32_t *lists;  // its list block
    int64_t val_off, nnz, n_nodes, n_elems;
    int zero;
    __device__ __forceinline__ PatchPlan(const PlanView &v, const GatherPatch &d, int npe)
        : lnode(v.celem_lnode + d.eb * npe), lists(v.gwords + d.list), val_off(v.val_off), nnz(v.nnz),
          n_nodes(v.n_nodes), n_elems(v.n_elems), zero(v.gzero) {}
};

// The summation of a patch's owned entries.  A warp takes every (warps of the
// block)-th chunk, U at a time, side by side and without branches between them: a
// block has only two warps a scheduler in this phase, so the loads and additions of
// one chunk alone wait out their latencies (1M bricks, 3,584 entries a patch: 220 us
// chunk by chunk, of which removing every load and store of the phase took 15).  The
// words of a batch are loaded together, the first batch and the diagonals before the
// barrier that completes the element matrices.
template <int NPE, typename AccT, bool MIXED>
struct GatherRows {
    static constexpr int U = 4, PRE = NPE == 8 ? 2 : 3;  // chunks of a batch, words of each loaded ahead
    static constexpr int DPRE = NPE == 8 ? 4 : 12;       // the same of a chunk of diagonals
    const PatchPlan &pv;
    const GatherPatch &d;
    const uint4 *tab;      // shared: chunk table
    const int64_t *rowd;   // shared: row starts
    const uint32_t *L;     // global: the list block
    int lane, warp, nw, n_chunks;
    uint32_t none;         // a word of two zeros' positions
    uint32_t w[U][PRE], dw[DPRE];
    int64_t dat;           // CSR position of the lane's diagonal

    __device__ __forceinline__ GatherRows(const PatchPlan &v, const GatherPatch &p, const uint4 *t, const int64_t *r)
        : pv(v), d(p), tab(t), rowd(r), L(v.lists), lane(threadIdx.x & 31), warp(threadIdx.x >> 5),
          nw(blockDim.x >> 5), n_chunks(p.n_chunks()), none((uint32_t)v.zero * 0x10001u) {}

    __device__ __forceinline__ void load(int c0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + u * nw;
            const uint2 t = c < n_chunks ? *reinterpret_cast<const uint2 *>(tab + c) : make_uint2(0u, 0u);
#pragma unroll
            for (int j = 0; j < PRE; ++j) w[u][j] = j < (int)t.y ? __ldg(L + t.x + 32 * j + lane) : none;
        }
    }
    // chunks of diagonals go to the warps from the last on
    __device__ __forceinline__ int first_diag() const { return nw - 1 - warp; }
    __device__ __forceinline__ void load_diag(int c) {
        const bool here = 32 * c < d.n_own;
        const uint2 t = here ? *reinterpret_cast<const uint2 *>(tab + n_chunks + c) : make_uint2(0u, 0u);
#pragma unroll
        for (int j = 0; j < DPRE; ++j) dw[j] = j < (int)t.y ? __ldg(L + t.x + 32 * j + lane) : none;
        const int64_t *ddst = reinterpret_cast<const int64_t *>(L + 4 * (n_chunks + d.n_diag())) + d.n_rows;
        dat = 32 * c + lane < d.n_own ? __ldg(ddst + 32 * c + lane) : 0;
    }

    __device__ __forceinline__ AccT term(const AccT *ke, uint32_t i, int *status) const {
        (void)status;
        if (!FEM_IN_BOUNDS((int)i <= pv.zero, status)) return AccT(0);
        return ke[i];
    }

    __device__ __forceinline__ void run(const AccT *ke, AccT *__restrict__ vals, int *status) {
        const int64_t val_off = pv.val_off;
        for (int c0 = warp; c0 < n_chunks; c0 += U * nw) {
            uint32_t v[U][PRE];
            uint4 t[U];
            AccT s[U];
            int deep = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
#pragma unroll
                for (int j = 0; j < PRE; ++j) v[u][j] = w[u][j];
                t[u] = tab[min(c0 + u * nw, n_chunks - 1)];
                s[u] = AccT(0);
                deep = max(deep, (int)t[u].y);
            }
            if (c0 + U * nw < n_chunks) load(c0 + U * nw);
#pragma unroll
            for (int j = 0; j < PRE; ++j) {
                AccT x[U][2];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    x[u][0] = term(ke, v[u][j] & 0xffffu, status);
                    x[u][1] = term(ke, v[u][j] >> 16, status);
                }
#pragma unroll
                for (int u = 0; u < U; ++u) s[u] = (s[u] + x[u][0]) + x[u][1];
            }
            for (int j = PRE; j < deep; ++j)
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (j < (int)t[u].y) {
                        const uint32_t q = __ldg(L + t[u].x + 32 * j + lane);
                        s[u] = (s[u] + term(ke, q & 0xffffu, status)) + term(ke, q >> 16, status);
                    }
            int64_t at[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int r = (int)t[u].z + __popc(t[u].w & (0xffffffffu >> (31 - lane))) - 1;
                at[u] = rowd[r] + (32 * (c0 + u * nw) + lane) - val_off;
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (32 * (c0 + u * nw) + lane < d.n_off && FEM_IN_BOUNDS(at[u] >= 0 && at[u] < pv.nnz, status))
                    vals[at[u]] = s[u];
        }
    }

    // Diagonals, one owned row a lane; in mixed precision those of high-valence rows
    // (marked in the table) are summed FP64-accurately, as by k_patch.
    __device__ __forceinline__ void run_diag(const AccT *ke, AccT *__restrict__ vals, unsigned mode, int *status) {
        for (int c = first_diag(); 32 * c < d.n_own; c += nw) {
            const uint4 t = tab[n_chunks + c];
            const int c2 = (int)t.y;
            const int64_t at = dat - pv.val_off;
            AccT x[DPRE][2];
#pragma unroll
            for (int j = 0; j < DPRE; ++j)
                x[j][0] = term(ke, dw[j] & 0xffffu, status), x[j][1] = term(ke, dw[j] >> 16, status);
            AccT s = AccT(0);
            if (MIXED && t.w != 0) {
                const bool hv = (t.w >> lane & 1u) != 0;
                if (mode & FP64_SUMS) {
                    double ds = 0.0;
                    auto add = [&](AccT v) { s += v, ds += (double)v; };
#pragma unroll
                    for (int j = 0; j < DPRE; ++j) add(x[j][0]), add(x[j][1]);
                    for (int j = DPRE; j < c2; ++j) {
                        const uint32_t q = __ldg(L + t.x + 32 * j + lane);
                        add(term(ke, q & 0xffffu, status)), add(term(ke, q >> 16, status));
                    }
                    if (hv) s = (AccT)ds;
                } else {
                    // a plain sum is the high part of the TwoSum pair
                    float2 pr = make_float2(0.f, 0.f);
#pragma unroll
                    for (int j = 0; j < DPRE; ++j) two_sum_acc(pr, (float)x[j][0]), two_sum_acc(pr, (float)x[j][1]);
#pragma unroll 4
                    for (int j = DPRE; j < c2; ++j) {
                        const uint32_t q = __ldg(L + t.x + 32 * j + lane);
                        two_sum_acc(pr, (float)term(ke, q & 0xffffu, status));
                        two_sum_acc(pr, (float)term(ke, q >> 16, status));
                    }
                    s = hv ? (AccT)(pr.x + pr.y) : (AccT)pr.x;
                }
            } else {
#pragma unroll
                for (int j = 0; j < DPRE; ++j) s = (s + x[j][0]) + x[j][1];
#pragma unroll 4
                for (int j = DPRE; j < c2; ++j) {
                    const uint32_t q = __ldg(L + t.x + 32 * j + lane);
                    s = (s + term(ke, q & 0xffffu, status)) + term(ke, q >> 16, status);
                }
            }
            if (32 * c + lane < d.n_own && FEM_IN_BOUNDS(at >= 0 && at < pv.nnz, status)) vals[at] = s;
            if (32 * (c + nw) < d.n_own) load_diag(c + nw);
        }
    }
};

// The patches desc[w0 + blockIdx.x], + gridDim.x, ... below w1.  BATCH: desc holds the
// patches of many meshes, items[pad] their plan, inputs and outputs.
template <int NPE, typename AccT, typename S, typename CT, bool FUSED, bool MIXED, bool BATCH>
__device__ __forceinline__ void gather_patches(const PlanView &pv0, const S *__restrict__ X0,
                                               const CT *__restrict__ c0, const AccT *__restrict__ ke0,
                                               AccT *__restrict__ vals0, const float *xrank0, float thr0,
                                               const BatchItem *__restrict__ items,
                                               const GatherPatch *__restrict__ desc, int64_t w0, int64_t w1,
                                               const GatherSmem &L, unsigned mode, int *status) {
    constexpr int NP = ElemTraits<NPE>::NP;
    constexpr bool X4 = sizeof(S) == 4;       // FP32 coordinates: one 16-byte row a node
    constexpr int XW = X4 ? 4 : 3;
    extern __shared__ __align__(16) unsigned char g_smem[];
    __shared__ GatherPatch sd[3];  // this, the next and the next but one patch
    AccT *ke = reinterpret_cast<AccT *>(g_smem + L.ke);
    S(*xs)[XW] = reinterpret_cast<S(*)[XW]>(g_smem + L.xs);
    CT *cs = reinterpret_cast<CT *>(g_smem + L.cs);
    int32_t *gid = reinterpret_cast<int32_t *>(g_smem + L.gid);
    int32_t *eid = reinterpret_cast<int32_t *>(g_smem + L.eid);
    uint4 *tab = reinterpret_cast<uint4 *>(g_smem + L.tab);
    int64_t *rowd = reinterpret_cast<int64_t *>(g_smem + L.rowd);
    uint32_t *bad = reinterpret_cast<uint32_t *>(g_smem + L.bad);  // distorted elements, a bit each
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int64_t step = gridDim.x;
    auto view = [&](const GatherPatch &d) -> const PlanView & {
        if constexpr (BATCH) return items[d.pad].pv;
        else return pv0;
    };
    const float4 *Xr = X4 && !BATCH ? reinterpret_cast<const float4 *>(xrank0) : nullptr;
    // first copies of a patch: its closure's node ids (ranks, where the coordinates
    // come in locality order) and element ids
    auto copy_ids = [&](const GatherPatch &d) {
        const PlanView &pv = view(d);
        if constexpr (FUSED) {
            const int32_t *src = Xr ? pv.cnode_rank : pv.cnode_gid;
            for (int j = tid; j < d.n_cnodes; j += nthr) g_cp4(gid + j, src + d.cb + j);
        }
        for (int j = tid; j < d.n_elems; j += nthr) g_cp4(eid + j, pv.celem_id + d.eb + j);
    };
    // second copies: coordinates and coefficients of the ids this thread copied
    auto copy_inputs = [&](const GatherPatch &d) {
        const PlanView &pv = view(d);
        const S *X = BATCH ? static_cast<const S *>(items[d.pad].X) : X0;
        const CT *cf = BATCH ? static_cast<const CT *>(items[d.pad].c) : c0;
        g_wait();
        for (int j = tid; j < d.n_cnodes; j += nthr) {
            int64_t g = gid[j];
#ifdef FEM_DEBUG_BOUNDS
            // testing the checks: one planted out-of-range node id per patch
            if ((mode & PLANT_ID) && j == 0) g = pv.n_nodes;
#endif
            if (!FEM_IN_BOUNDS(g >= 0 && g < pv.n_nodes, status)) g = 0;
            if (Xr) {
                g_cp16(&xs[j][0], Xr + g);
            } else {
#pragma unroll
                for (int k = 0; k < 3; ++k) g_cp(&xs[j][k], X + 3 * g + k);
            }
        }
        for (int j = tid; j < d.n_elems; j += nthr) {
            int64_t e = eid[j];
            if (!FEM_IN_BOUNDS(e >= 0 && e < pv.n_elems, status)) e = 0;
            g_cp(cs + j, cf + e);
        }
    };
    // chunk table and row starts of the patch's lists; a warp copies the table entries
    // of its own chunks
    auto copy_tables = [&](const GatherPatch &d) {
        const uint32_t *B = view(d).gwords + d.list;
        const int total = d.n_chunks() + d.n_diag(), nw = nthr >> 5;
        const int nch = d.n_chunks(), warp = tid >> 5;
        for (int c = warp + (tid & 31) * nw; c < nch; c += nthr) g_cp16(tab + c, reinterpret_cast<const uint4 *>(B) + c);
        for (int c = nch + nw - 1 - warp + (tid & 31) * nw; c < total; c += nthr)
            g_cp16(tab + c, reinterpret_cast<const uint4 *>(B) + c);
        for (int r = tid; r < d.n_rows; r += nthr) g_cp8(rowd + r, reinterpret_cast<const int64_t *>(B + 4 * total) + r);
    };
    // matrices of the patch's distorted elements
    auto fix_distorted = [&](const GatherPatch &d) {
        if constexpr (FUSED && MIXED && NPE == 8) {
            const PlanView &pv = view(d);
            const int lane = tid & 31, nw = nthr >> 5;
            for (int j = tid >> 5; j < (d.n_elems + 31) / 32; j += nw) {
                for (uint32_t b = bad[j]; b;) {
                    // the word's next four elements, one for each eight lanes (the last
                    // again where there are fewer)
                    int i = 32 * j;
                    for (int k = 0; k < 4; ++k) {
                        if (b) {
                            const int e = 32 * j + __ffs(b) - 1;
                            b &= b - 1;
                            if (k <= lane >> 3) i = e;
                        }
                    }
                    uint16_t ln[NPE];
                    load_lnodes<NPE>(pv.celem_lnode, d.eb + i, ln);
                    S x[NPE][3];
#pragma unroll
                    for (int a = 0; a < NPE; ++a) {
                        if (!FEM_IN_BOUNDS(ln[a] < d.n_cnodes, status)) ln[a] = 0;
#pragma unroll
                        for (int k = 0; k < 3; ++k) x[a][k] = xs[ln[a]][k];
                    }
                    AccT kv[NP];
                    brick_distorted_shared<S>(x, (float)cs[i], (mode & OP_MASS) != 0, kv);
                    if (!isfinite(kv[0])) atomicOr(status, STATUS_NONFINITE);
                    if ((lane & 7) == 0) put_matrix<NP>(ke + i * NP, kv);
                }
                __syncwarp();
                if (lane == 0) bad[j] = 0;
            }
        }
    };
    // the lists and local node indices of a patch to come, into L2
    auto ahead = [&](const GatherPatch &d) {
        const PlanView &pv = view(d);
        g_prefetch(pv.gwords + d.list, (size_t)d.n_words * 4);
        if constexpr (FUSED) g_prefetch(pv.celem_lnode + d.eb * NPE, (size_t)d.n_elems * NPE * 2);
    };
    int64_t w = w0 + blockIdx.x;
    if (w >= w1) return;
    if constexpr (FUSED && MIXED && NPE == 8)
        for (int j = tid; j < L.n_bad; j += nthr) bad[j] = 0;
    if (tid < 8 && w + (tid >> 2) * step < w1)
        reinterpret_cast<uint4 *>(&sd[tid >> 2])[tid & 3] =
            __ldg(reinterpret_cast<const uint4 *>(desc + w + (tid >> 2) * step) + (tid & 3));
    __syncthreads();
    if (tid == 0) ahead(sd[0]);
    copy_ids(sd[0]);
    if constexpr (FUSED) copy_inputs(sd[0]);
    for (int it = 0;; it = it == 2 ? 0 : it + 1, w += step) {
        const GatherPatch &d = sd[it], &dn = sd[it == 2 ? 0 : it + 1];
        const PatchPlan pv(view(d), d, NPE);
        g_wait();
        __syncthreads();  // the patch's inputs are visible; the previous patch's matrices have been read
        const bool more = w + step < w1;
        bool distorted = false;
        (void)distorted;
        if (more && tid == 0) ahead(dn);
        if (w + 2 * step < w1 && tid < 4)
            g_cp16(reinterpret_cast<uint4 *>(&sd[it == 0 ? 2 : it - 1]) + tid,
                   reinterpret_cast<const uint4 *>(desc + w + 2 * step) + tid);
        copy_tables(d);
        if constexpr (FUSED) {
            if (more) copy_ids(dn);
            const float thr = BATCH ? items[d.pad].thr : thr0;
            for (int i = tid; i < d.n_elems; i += nthr) {
                uint16_t ln[NPE];
                load_lnodes<NPE>(pv.lnode, i, ln);
                S xc[NPE][3];
#pragma unroll
                for (int a = 0; a < NPE; ++a) {
                    if (!FEM_IN_BOUNDS(ln[a] < d.n_cnodes, status)) ln[a] = 0;
                    if constexpr (X4) {
                        const float4 v = *reinterpret_cast<const float4 *>(xs[ln[a]]);
                        xc[a][0] = v.x, xc[a][1] = v.y, xc[a][2] = v.z;
                    } else {
                        xc[a][0] = xs[ln[a]][0];
                        xc[a][1] = xs[ln[a]][1];
                        xc[a][2] = xs[ln[a]][2];
                    }
                }
                AccT kv[NP];
                if (element_matrix_fast<NPE, AccT, S, MIXED>(xc, cs[i], thr, mode, kv)) {
                    atomicOr(&bad[i >> 5], 1u << (i & 31));
                    distorted = true;
                }
                // k_00 (m_00) is positive and finite for any element of nonzero volume
                // (a distorted brick's FP32 value may not be; its own is tested below)
                else if (!isfinite(kv[0])) atomicOr(status, STATUS_NONFINITE);
                put_matrix<NP>(ke + i * NP, kv);
            }
        } else {
            constexpr int UNIT = NP * sizeof(AccT) % 16 == 0 ? 16 : 8, Q = NP * sizeof(AccT) / UNIT;
            const int n = d.n_elems * Q;
            for (int t = tid; t < n; t += nthr) {
                int64_t e = eid[t / Q];
                if (!FEM_IN_BOUNDS(e >= 0 && e < pv.n_elems, status)) e = 0;
                unsigned char *dst = reinterpret_cast<unsigned char *>(ke) + t * UNIT;
                const unsigned char *src = reinterpret_cast<const unsigned char *>(ke0) + (e * Q + t % Q) * UNIT;
                if constexpr (UNIT == 16) g_cp16(dst, src);
                else g_cp8(dst, src);
            }
        }
        g_wait();
        __syncwarp();
        GatherRows<NPE, AccT, MIXED> rows(pv, d, tab, rowd);
        rows.load(rows.warp);
        rows.load_diag(rows.first_diag());
        if (tid == 0) ke[pv.zero] = AccT(0);
        // the closure's element matrices are complete ...
        if constexpr (FUSED && MIXED && NPE == 8) {
            // ... but for the distorted elements': four at a time by each warp
            if (__syncthreads_or(distorted)) {
                fix_distorted(d);
                __syncthreads();
            }
        } else {
            __syncthreads();
        }
        if (more) {
            if constexpr (FUSED) copy_inputs(dn);
            else copy_ids(dn);
        }
        AccT *vals = BATCH ? static_cast<AccT *>(items[d.pad].vals) : vals0;
        rows.run_diag(ke, vals, mode, status);
        rows.run(ke, vals, status);
        if (!more) break;
    }
}

// Registers: 128 a thread lets two 256-thread blocks of bricks share an SM;
// tetrahedra need fewer (three blocks).
template <int NPE, bool FUSED, bool MIXED>
__host__ __device__ constexpr int gather_max_threads() { return NPE == 4 && FUSED && MIXED ? 256 : 512; }
template <int NPE, bool FUSED, bool MIXED>
__host__ __device__ constexpr int gather_min_blocks() { return NPE == 4 && FUSED && MIXED ? 3 : 1; }

template <int NPE, typename AccT, typename S, typename CT, bool FUSED, bool MIXED>
__global__ void __launch_bounds__((gather_max_threads<NPE, FUSED, MIXED>()), (gather_min_blocks<NPE, FUSED, MIXED>()))
    k_gather(PlanView pv, const S *__restrict__ X, const CT *__restrict__ c, const AccT *__restrict__ ke,
             AccT *__restrict__ vals, const float *__restrict__ xrank, float thr, int64_t w0, int64_t w1, GatherSmem L, unsigned mode, int *status) {
    gather_patches<NPE, AccT, S, CT, FUSED, MIXED, false>(pv, X, c, ke, vals, xrank, thr, nullptr, pv.gpatch, w0, w1, L, mode, status);
}

template <int NPE, typename AccT, bool MIXED>
__global__ void __launch_bounds__((gather_max_threads<NPE, true, MIXED>()), (gather_min_blocks<NPE, true, MIXED>()))
    k_gather_batched(const BatchItem *__restrict__ items, const GatherPatch *__restrict__ desc, int64_t n,
                     GatherSmem L, unsigned mode, int *status) {
    PlanView none{};
    gather_patches<NPE, AccT, AccT, AccT, true, MIXED, true>(none, nullptr, nullptr, nullptr, nullptr, nullptr, 0.f, items,
                                                             desc, 0, n, L, mode, status);
}

// X of the nodes in locality order, one 16-byte row each (see gather_patches).
__global__ void __launch_bounds__(256) k_order_x(const int32_t *__restrict__ order, const float *__restrict__ X,
                                                 int64_t n, float4 *__restrict__ out) {
    const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (r >= n) return;
    const int64_t g = __ldg(order + r);
    out[r] = make_float4(__ldg(X + 3 * g), __ldg(X + 3 * g + 1), __ldg(X + 3 * g + 2), 0.f);
}

fem_status launch_order_x(const Plan &P, const float *X, float *xrank, cudaStream_t s) {
    k_order_x<<<(unsigned)cdiv(P.n_nodes, 256), 256, 0, s>>>(P.own_row.ptr, X, P.n_nodes,
                                                             reinterpret_cast<float4 *>(xrank));
    FEM_LAUNCHED("k_order_x");
    return FEM_OK;
}

XrankUse::XrankUse(fem_mesh m, bool mixed, fem_dtype xd, cudaStream_t s) : m_(m), s_(s) {
    if (!mixed || xd != FEM_F32 || !m->plan.full.lists.ready || m->xrank.n < 4 * (size_t)m->n_nodes) return;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return;
    }
    lock_ = std::unique_lock<std::mutex>(m->xrank_mu);
    if ((m->xrank_read || cudaEventCreateWithFlags(&m->xrank_read, cudaEventDisableTiming) == cudaSuccess) &&
        cudaStreamWaitEvent(s, m->xrank_read, 0) == cudaSuccess) {
        ptr_ = m->xrank.ptr;
    } else {
        cudaGetLastError();
        lock_.unlock();
    }
}

XrankUse::~XrankUse() {
    if (ptr_ && cudaEventRecord(m_->xrank_read, s_) != cudaSuccess) cudaStreamSynchronize(s_);
}

GatherSmem gather_smem_layout(const GatherMax &g, int npe, bool fused, size_t accsize, size_t xsize, size_t csize) {
    GatherSmem L{};
    auto up = [](size_t v) { return (v + 15) & ~(size_t)15; };
    size_t o = 0;
    L.tab = o;
    o = up(o + (size_t)(g.max_acc / 32 + g.max_own / 32 + 2) * 16);
    L.rowd = o;
    o = up(o + (size_t)g.max_own * 8);
    L.bad = o;
    L.n_bad = (int)((g.max_celems + 31) / 32);
    if (fused && npe == 8) o = up(o + (size_t)L.n_bad * 4);
    L.ke = o;
    o = up(o + ((size_t)g.max_celems * (npe * (npe + 1) / 2) + 1) * accsize);
    L.xs = o;
    if (fused) o = up(o + (size_t)g.max_cnodes * (xsize == 4 ? 4 : 3) * xsize);
    L.cs = o;
    if (fused) o = up(o + (size_t)g.max_celems * csize);
    L.gid = o;
    if (fused) o = up(o + (size_t)g.max_cnodes * sizeof(int32_t));
    L.eid = o;
    o = up(o + (size_t)g.max_celems * sizeof(int32_t));
    L.total = o;
    return L;
}

// Resident blocks of f at `threads` threads and L bytes, opted in; 0 if none fits.
template <typename F>
static fem_status resident(F *f, int threads, size_t bytes, int *per_sm) {
    FEM_CUDA(allow_smem(f, bytes));
    FEM_CUDA(resident_blocks(per_sm, f, threads, bytes));
    if (*per_sm < 1) {
        set_error("the gather kernel cannot be resident with %d threads and %zu bytes of shared memory", threads, bytes);
        return FEM_ERR_UNSUPPORTED;
    }
    return FEM_OK;
}

template <int NPE, typename AccT, typename S, typename CT, bool FUSED, bool MIXED>
static fem_status launch_gather_t(const PatchArgs &a, cudaStream_t s) {
    const Plan &P = *a.plan;
    const Closure &cl = a.closure ? *a.closure : P.full;
    const int64_t q0 = std::max(a.p0, cl.p0) - cl.p0, q1 = std::min(a.p1, cl.p1) - cl.p0;
    if (q1 <= q0) return FEM_OK;
    GatherMax gm;
    gm.add(P);
    const GatherSmem L = gather_smem_layout(gm, NPE, FUSED, sizeof(AccT), sizeof(S), sizeof(CT));
    auto f = k_gather<NPE, AccT, S, CT, FUSED, MIXED>;
    const int threads = std::min(a.threads, gather_max_threads<NPE, FUSED, MIXED>());
    int per_sm = 0;
    FEM_TRY(resident(f, threads, L.total, &per_sm));
    if (a.blocks_per_sm > 0 && a.blocks_per_sm < per_sm) per_sm = a.blocks_per_sm;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(q1 - q0, (int64_t)num_sms() * per_sm));
    PlanView pv = P.view(cl);
    pv.val_off = a.val_off;
    const float *xr = nullptr;
    if constexpr (FUSED && sizeof(S) == 4) {
        if (a.xrank) {
            xr = a.xrank;
            if (!a.x_ordered) FEM_TRY(launch_order_x(P, (const float *)a.X, a.xrank, s));
        }
    }
    f<<<grid, threads, L.total, s>>>(pv, (const S *)a.X, (const CT *)a.c, (const AccT *)a.ke, (AccT *)a.vals, xr, a.thr,
                                     q0, q1, L, a.mode, a.wait.status);
    FEM_LAUNCHED("k_gather");
    return FEM_OK;
}

int gather_blocks_per_sm(int npe, int threads) {
    int n = 0;
    const cudaError_t e =
        npe == 8 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gather<8, float, float, float, true, true>, threads, 0)
                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_gather<4, float, float, float, true, true>, threads, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 2;
    }
    return std::max(1, n);
}

fem_status launch_gather(const PatchArgs &a, cudaStream_t s) {
#define FEM_G(NPE, ACC, S, CT, FU, MX) return launch_gather_t<NPE, ACC, S, CT, FU, MX>(a, s)
    if (!a.mixed) {
        if (a.fused) {
            if (a.npe == 8) FEM_G(8, double, double, double, true, false);
            FEM_G(4, double, double, double, true, false);
        }
        if (a.npe == 8) FEM_G(8, double, double, double, false, false);
        FEM_G(4, double, double, double, false, false);
    }
    if (!a.fused) {
        if (a.npe == 8) FEM_G(8, float, float, float, false, true);
        FEM_G(4, float, float, float, false, true);
    }
    if (a.npe == 8) {
        if (a.xd == FEM_F32 && a.cd == FEM_F32) FEM_G(8, float, float, float, true, true);
        if (a.xd == FEM_F32 && a.cd == FEM_F64) FEM_G(8, float, float, double, true, true);
        if (a.xd == FEM_F64 && a.cd == FEM_F32) FEM_G(8, float, double, float, true, true);
        FEM_G(8, float, double, double, true, true);
    }
    if (a.xd == FEM_F32 && a.cd == FEM_F32) FEM_G(4, float, float, float, true, true);
    if (a.xd == FEM_F32 && a.cd == FEM_F64) FEM_G(4, float, float, double, true, true);
    if (a.xd == FEM_F64 && a.cd == FEM_F32) FEM_G(4, float, double, float, true, true);
    FEM_G(4, float, double, double, true, true);
#undef FEM_G
}

template <int NPE, typename T, bool MIXED>
static fem_status gather_batched_config_t(const GatherMax &gm, int threads, int blocks_per_sm, BatchLaunch *out) {
    out->gl = gather_smem_layout(gm, NPE, true, sizeof(T), sizeof(T), sizeof(T));
    out->threads = std::min(threads, gather_max_threads<NPE, true, MIXED>());
    int per_sm = 0;
    FEM_TRY(resident(k_gather_batched<NPE, T, MIXED>, out->threads, out->gl.total, &per_sm));
    if (blocks_per_sm > 0 && blocks_per_sm < per_sm) per_sm = blocks_per_sm;
    out->grid = num_sms() * per_sm;
    return FEM_OK;
}

bool gather_batch_fits(int npe, bool mixed, const GatherMax &gm) {
    int dev = 0, limit = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return false;
    const size_t w = mixed ? 4 : 8;
    return gather_smem_layout(gm, npe, true, w, w, w).total + 1024 <= (size_t)limit;  // (and the static part)
}

fem_status gather_batched_config(int npe, bool mixed, const GatherMax &gm, int threads, int blocks_per_sm,
                                 BatchLaunch *out) {
    out->npe = npe;
    out->mixed = mixed;
    out->gather = true;
    if (mixed) return npe == 8 ? gather_batched_config_t<8, float, true>(gm, threads, blocks_per_sm, out)
                               : gather_batched_config_t<4, float, true>(gm, threads, blocks_per_sm, out);
    return npe == 8 ? gather_batched_config_t<8, double, false>(gm, threads, blocks_per_sm, out)
                    : gather_batched_config_t<4, double, false>(gm, threads, blocks_per_sm, out);
}

fem_status launch_gather_batched_kernel(const BatchLaunch &bl, cudaStream_t s) {
#define FEM_B(NPE, T, MX)                                                                                       \
    k_gather_batched<NPE, T, MX><<<bl.grid, bl.threads, bl.gl.total, s>>>(bl.items, bl.gpatch, bl.n_work, bl.gl, \
                                                                          bl.mode, bl.wait.status)
    if (bl.mixed) {
        if (bl.npe == 8) FEM_B(8, float, true); else FEM_B(4, float, true);
    } else {
        if (bl.npe == 8) FEM_B(8, double, false); else FEM_B(4, double, false);
    }
#undef FEM_B
    FEM_LAUNCHED("k_gather_batched");
    return FEM_OK;
}

__global__ void k_gather_table(const GatherPatch *src, int64_t n, int mesh, GatherPatch *out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        GatherPatch d = src[i];
        d.pad = mesh;
        out[i] = d;
    }
}

fem_status launch_gather_table(const GatherPatch *src, int64_t n, int mesh, GatherPatch *out, cudaStream_t s) {
    if (n <= 0) return FEM_OK;
    k_gather_table<<<(unsigned)cdiv(n, 256), 256, 0, s>>>(src, n, mesh, out);
    FEM_LAUNCHED("k_gather_table");
    return FEM_OK;
}

}  // namespace fem
