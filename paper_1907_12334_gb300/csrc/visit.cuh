// visit.cuh -- one visit half of Algorithm 1 on one grid above the on-chip diagonals.
//
// k_visit runs a visit half (PRE: nu1 sweeps, residual, restriction; POST:
// prolongation, nu2 sweeps) of one (item, grid) with a cluster of C CTAs (C = 1:
// a single one), each on a slab of ny / C rows.  What bounds a visit is DRAM on
// the large grids and, on the small ones, the chain first touch - half sweeps -
// barriers; so every input is read once, all of a thread's loads are in flight
// together, and between the load and the store nothing leaves the SM:
//  - a thread owns pairs (2m, 2m + 1) of neighbouring nodes of a row, one red and
//    one black, with their coefficients and b, scaled by the diagonal, in
//    registers (the Pair of mid.cuh);
//  - u sits in shared memory, one row of nx words per grid row, column 0 the west
//    boundary and the east boundary of the row before it, with a halo row on each side;
//  - a CTA writes the nodes of its first and last row also into its neighbours'
//    halo rows (distributed shared memory) before the cluster barrier that ends
//    a half sweep, so every read is local.
// The largest grid a cluster of 16 holds has 2^16 cells in FP32 and 2^15 in FP64
// (visit_takes); larger ones, and thin ones with too few rows for their cluster, are left
// to the one-CTA kernels in global memory.
// The slabs and the number of pairs per thread regroup independent per-node
// updates: they do not change a bit of the result.
#pragma once

namespace msg {

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// store v at the address that `a` (this CTA's shared memory) has in CTA `rank` of the cluster
template <class T>
__device__ __forceinline__ void store_peer(uint32_t a, int rank, T v)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    if constexpr (sizeof(T) == 4) asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(r), "f"(v) : "memory");
    else asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(r), "d"(v) : "memory");
}

constexpr int kVisitClusterMax = 16;
// pairs per thread: two keep the registers of a float thread under 64, so a CTA can have
// 1024 of them and a grid of 4096 cells needs no cluster (four: 108 registers and 1.3 times
// the time on diagonals 8 and 9; one, with twice the threads: 1.1 to 1.9 times)
template <class T> constexpr int visit_threads_max() { return sizeof(T) == 4 ? 1024 : 512; }
constexpr int kVisitPairs = 2;

// words of a slab of a grid 2^p x 2^q in a cluster of C: u with its halo rows, r with its lower halo
__host__ __device__ __forceinline__ int visit_words(int p, int q, int C)
{
    const int nx = 1 << p, R = (1 << q) / C;
    return (R + 2) * nx + 4 + (R + 1) * (nx >> 1);
}

template <class T, int NP, bool CL>
__global__ void __launch_bounds__(visit_threads_max<T>())
    k_visit(DevCtx cx, T* su, T* sbx, T* sby, const T* ax, const T* ay, int pre, int zero, int nu, T omega, int C)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Segment* sg = &cx.segs[blockIdx.y];
    const int at = CL ? blockIdx.x / C : blockIdx.x, rank = CL ? blockIdx.x - at * C : 0;
    launch_next();
    // The whole cluster.  A CTA that leaves here has not waited for the kernel before this one, so
    // the chain holds only while some CTA of every launch goes on: the host makes no segment
    // without samples.
    if ((int64_t)at >= sg->count) return;
    if (CL) cluster_arrive();              // a peer's shared memory is written once all have started
    const int smp = cx.slist[sg->list_off + at];
    const int64_t scr = sg->scr0 + (int64_t)cx.gpos[smp] * sg->scr_per, node = cx.samples[smp].node_off + sg->co;
    const int p = sg->p, q = sg->q, nx = 1 << p, ny = 1 << q, W = nx + 1, hx2 = nx >> 1, R = ny / C, j0 = rank * R;
    const bool hx = p < sg->pi, hy = q < sg->qi;  // parents that have restricted into b
    const T* fx = ax + node + j0 * W;  // the slab's first row of each array
    const T* fy = ay + node + j0 * W;
    const T* bx = sbx + scr + sg->so + j0 * W;
    const T* by = sby + scr + sg->so + j0 * W;
    T* gu = su + scr + sg->so + j0 * W;
    const Sm<T> U = Sm<T>{(uint32_t)__cvta_generic_to_shared(smem_raw)}.at(nx);  // row lj at lj nx, halo rows lj = -1 and R
    const Sm<T> Rr = U.at((R + 1) * nx + 4 + hx2);  // red residual of each pair, lower halo row lj = -1
    const int nt = blockDim.x;  // NP nt = R nx / 2 pairs
    const bool below = CL && rank > 0, above = CL && rank < C - 1;
    Pair<T> P[NP];
    T aw[NP], am[NP], ae[NP], sA[NP], sB[NP], nA[NP], nB[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int cA = 2 * (threadIdx.x + k * nt), i = cA & (nx - 1), lj = cA >> p;
        const bool ok = j0 + lj > 0;
        const int o = lj * W + i, w = ok && i > 0 ? o - 1 : o, s = ok ? o - W : o;
        aw[k] = fx[w]; am[k] = fx[o]; ae[k] = fx[o + 1];
        nA[k] = fy[o]; nB[k] = fy[o + 1]; sA[k] = fy[s]; sB[k] = fy[s + 1];
    }
    wait_previous();
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int cA = 2 * (threadIdx.x + k * nt), i = cA & (nx - 1), lj = cA >> p, j = j0 + lj;
        const bool ok = j > 0, hasA = ok && i > 0, redB = j & 1;
        const int o = lj * W + i;
        T bA, bB, uA = T(0), uB = T(0);
        if (hx && hy) {
            bA = T(0.5) * bx[o] + T(0.5) * by[o];
            bB = T(0.5) * bx[o + 1] + T(0.5) * by[o + 1];
        } else {
            const T* b = hy ? by : bx;  // (no parent: the item's own residual, in bx)
            bA = b[o];
            bB = b[o + 1];
        }
        if (!zero) {
            uA = gu[o];
            uB = gu[o + 1];
        }
        // b and u at boundary nodes are whatever the scratch held: not used
        T iR, iK;
        pair_set(P[k], U.at(cA).a, nx, ok, hasA, redB, aw[k], am[k], ae[k], sA[k], sB[k], nA[k], nB[k], hasA ? bA : T(0),
                 ok ? bB : T(0), hasA ? uA : T(0), ok ? uB : T(0), iR, iK);
    }
    if (!pre) {  // Eq. (2.4) at the black nodes (the first red half sweep overwrites the red ones)
        const T* ucx = su + scr + sg->cxo + j0 * (hx2 + 1);
        const T* ucy = su + scr + sg->cyo + (j0 >> 1) * W;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            Pair<T>& a = P[k];
            const int cA = 2 * (threadIdx.x + k * nt), i = cA & (nx - 1), lj = cA >> p;
            const bool redB = (j0 + lj) & 1;
            if (a.w == 0 || (redB && i == 0)) continue;
            T vx = T(0), vy = T(0);
            if (p > 1) {  // child (p-1, q): black is column i (even) of an odd row, i + 1 of an even one
                const T* c = ucx + lj * (hx2 + 1) + (i >> 1);
                vx = redB ? c[0] : T(0.5) * (c[0] + c[1]);
            }
            if (q > 1) {  // child (p, q-1)
                const T* c = ucy + (lj >> 1) * W + (redB ? i : i + 1);
                vy = redB ? T(0.5) * (c[0] + c[W]) : c[0];
            }
            T e = p > 1 ? vx : vy;
            if (p > 1 && q > 1) {
                const T c1 = a.pK + a.oK, c2 = a.sK + a.nK, x2 = c1 * c1, y2 = c2 * c2, w = rcp_of(x2 + y2);
                e = (x2 * w) * vx + (y2 * w) * vy;
            }
            a.uK += omega * e;
        }
    }
    // both nodes of a pair (a pair of row 0 and column 0 of every row: zeros)
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int cA = 2 * (threadIdx.x + k * nt);
        const bool redB = (j0 + (cA >> p)) & 1;
        U.at(cA).st2(redB ? P[k].uK : P[k].uR, redB ? P[k].uR : P[k].uK);
    }
    // halo rows: zeros at the grid's boundary and in column 0; with neighbours, PRE from a
    // nonzero u takes their black nodes from memory (the only ones read before the
    // neighbour has written its red ones).  The red node in the last column of row -1 lies
    // before column 0 of row 0, which reads it with weight zero: it must be a number.
    for (int i = threadIdx.x; i < nx; i += nt) {
        if (!below || i == 0 || i == nx - 1) U.at(i - nx).st(T(0));
        else if (pre && !zero && ((i + j0 - 1) & 1)) U.at(i - nx).st(gu[i - W]);
        if (!above || i == 0) U.at(R * nx + i).st(T(0));
        else if (pre && !zero && ((i + j0 + R) & 1)) U.at(R * nx + i).st(gu[R * W + i]);
    }
    if (CL) cluster_wait();
    // write a node's value (u at address a): here, and in the halo of a neighbouring slab
    const uint32_t first = U.at(nx).a, last = U.at((R - 1) * nx).a, slab = (uint32_t)(R * nx * sizeof(T));
    auto put = [&](uint32_t a, T v) {
        Sm<T>{a}.st(v);
        if (CL) {
            if (below && a < first) store_peer(a + slab, rank - 1, v);
            if (above && a >= last) store_peer(a - slab, rank + 1, v);
        }
    };
    auto sync = [&] {
        if (CL) {
            cluster_arrive();
            cluster_wait();
        } else {
            __syncthreads();
        }
    };
    if (CL && !pre) {
#pragma unroll
        for (int k = 0; k < NP; ++k) put(P[k].aR - P[k].e, P[k].uK);
    }
    sync();
    for (int s = 0; s < nu; ++s) {
        // a half sweep reads nodes of the other colour only: all its loads come before its stores
        if (s == 0 && zero) {
#pragma unroll
            for (int k = 0; k < NP; ++k) P[k].uR = P[k].bR;
        } else {
#pragma unroll
            for (int k = 0; k < NP; ++k) P[k].uR = pair_red(P[k]);
        }
#pragma unroll
        for (int k = 0; k < NP; ++k) put(P[k].aR, P[k].uR);
        sync();
#pragma unroll
        for (int k = 0; k < NP; ++k) P[k].uK = pair_black(P[k]);
        if (pre || s + 1 < nu) {
#pragma unroll
            for (int k = 0; k < NP; ++k) put(P[k].aR - P[k].e, P[k].uK);
            sync();
        }
    }
    if (pre) {  // the residual of a black node is zero up to rounding after a black half sweep
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const Pair<T>& a = P[k];
            const int m = threadIdx.x + k * nt;
            const T r = a.dR * (pair_red(a) - a.uR);
            Rr.at(m).st(r);
            if (above && m >= (R - 1) * hx2) store_peer(Rr.at(m - R * hx2).a, rank + 1, r);
        }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {  // boundary nodes of column 0 and row 0 as zeros
        const int cA = 2 * (threadIdx.x + k * nt), i = cA & (nx - 1), lj = cA >> p;
        const bool redB = (j0 + lj) & 1;
        gu[lj * W + i] = redB ? P[k].uK : P[k].uR;
        gu[lj * W + i + 1] = redB ? P[k].uR : P[k].uK;
    }
    if (!pre) return;
    if (zero) {  // the other boundary nodes: scratch may hold an earlier stage's hierarchy
        for (int l = threadIdx.x; l < R; l += nt) gu[l * W + nx] = T(0);
        if (rank == C - 1)
            for (int i = threadIdx.x; i <= nx; i += nt) gu[R * W + i] = T(0);
    }
    sync();
    // Eq. (2.3) of the red residual; half of the weights meet black nodes
    if (p > 1) {  // child (p-1, q), node (ic, j) around column 2 ic
        T* cb = sbx + scr + sg->cxo + j0 * (hx2 + 1);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int m = threadIdx.x + k * nt, ic = m & (hx2 - 1), lj = m >> (p - 1), j = j0 + lj;
            const Sm<T> r = Rr.at(m);
            const T r0 = r.ld(), v = (j & 1) ? T(0.25) * (r.at(-1).ld() + r0) : T(0.5) * r0;
            if (ic > 0 && j > 0) cb[lj * (hx2 + 1) + ic] = v;
        }
    }
    if (q > 1) {  // child (p, q-1), node (i, jc) around row 2 jc
        T* cb = sby + scr + sg->cyo + (j0 >> 1) * W;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int m = threadIdx.x + k * nt, i = m & (nx - 1), l = m >> p;
            const Sm<T> r = Rr.at(l * nx + (i >> 1));
            const T v = (i & 1) ? T(0.25) * (r.at(-hx2).ld() + r.at(hx2).ld()) : T(0.5) * r.ld();
            if (i > 0 && j0 + l > 0) cb[l * W + i] = v;
        }
    }
}

}  // namespace msg
