// mid.cuh -- mu-cycles of Algorithm 1 with a whole item hierarchy on chip.
//
// Two kernels run the recursion for one item per CTA, every grid they touch in
// shared memory:
//   k_item  an item of a low stage from its interpolated initial guess to
//           convergence (FP64 residual, stopping decision, cycle, FP64 update,
//           repeated inside the kernel);
//   k_mid   the mu calls on the diagonals at and below kMidD inside the W-cycle
//           of a larger item.
//
// Why.  A W-cycle visits diagonal d 2^(L-d) times, so its cost is a chain of
// small dependent phases, two thirds of them on diagonals <= 3 (at most 102
// unknowns).  What bounds it is the latency of that chain, not bytes or flops:
// run as phases, the two calls at diagonal 4 took 65 us with the GPU otherwise
// idle, and 132 us at 192 samples of 256 x 256.  Two things shorten it:
//
//  - The mu calls on diagonal 3 start from u = 0 and are linear in their
//    right-hand side, so per sample and clipped triangle they are one matrix
//    M (at most 72 x 72).  k_lowop builds its columns by running the calls on
//    unit vectors, once per solve, in the arithmetic of the cycles; a
//    call is then one matrix-vector product instead of about 170 phases.
//  - Launch boundaries between visits become CTA barriers, and a visit keeps
//    each thread's coefficients and right-hand side in registers.
//
// Layout.  Grid (p,q) is stored as its 2^(p+q) cells, cell (i,j) at j 2^p + i,
// i < nx, j < ny.  Column 0 and row 0 are boundary nodes; the east
// boundary of a row is the next row's column 0, and the north boundary is row 0
// of the next grid (grids of a diagonal are ordered by p, so the next row 0 is
// at least as long) or the pad behind the diagonal.  All boundary values of u
// are therefore zeros at c +- 1 and c +- nx, every grid of diagonal d takes
// exactly 2^(d+2) words, and the east and north faces of a node sit at the
// node's own index.
//
// Work split.  A thread owns pairs of neighbouring cells (2m, 2m+1) of a
// diagonal, all its grids in one index range; a pair holds one red and one
// black node, so every half sweep uses every thread, and the face between the
// two and the partner's value never leave the registers.
#pragma once

namespace msg {

constexpr int kOpD = 3;      // the diagonal replaced by its matrix
constexpr int kOpN = 72;     // unknowns of the full diagonal kOpD
constexpr int kMidD = 6;     // highest diagonal of k_mid: 72 KB an item in FP32, 104 KB with records (kept.cuh; two an SM)
constexpr int kMidMax = 9;   // highest diagonal of any hierarchy held on chip
constexpr int kItemL32 = 9;  // stages solved whole by k_item (FP32 cycles): (5,6) takes 149 KB, with records 206 KB
constexpr int kItemL64 = 8;  // the same in FP64: (5,5) takes 209 KB
constexpr int kMidThreads = 256;

// ---------------------------------------------------------------- matrices --

// Clipped triangles below diagonal kOpD that items of stage > kOpD have:
// (pic, qic) = (min(p, 4), min(q, 4)), p + q >= kOpD + 3.
constexpr int kOpClasses = 8;
__host__ __device__ constexpr int op_pic(int c) { return c == 0 ? 1 : c == 1 ? 4 : c == 2 ? 2 : c == 3 ? 4 : c == 4 ? 3 : c == 5 ? 3 : 4; }
__host__ __device__ constexpr int op_qic(int c) { return c == 0 ? 4 : c == 1 ? 1 : c == 2 ? 4 : c == 3 ? 2 : c == 4 ? 3 : c == 5 ? 4 : c == 6 ? 3 : 4; }
// unknowns of the class on diagonal kOpD, and the row stride of its matrix:
// two threads share a row, and half a row, four times an odd number of words, keeps their
// 16-byte loads on disjoint banks (kept_matrix: eight threads, an odd number of words each)
__host__ __device__ constexpr int op_n(int pic, int qic)
{
    int n = 0;
    for (int p = 1; p <= 4; ++p) {
        const int q = kOpD + 2 - p;
        if (p <= pic && q <= qic) n += ((1 << p) - 1) * ((1 << q) - 1);
    }
    return n;
}
__host__ __device__ constexpr int op_ld(int n) { return n <= 24 ? 24 : n <= 40 ? 40 : n <= 56 ? 56 : 72; }
// does a sample with finest grid (P, Q) have items of the class?
__host__ __device__ constexpr bool op_has(int pic, int qic, int P, int Q)
{
    return pic <= P && qic <= Q && (pic < 4 ? pic : P) + (qic < 4 ? qic : Q) >= kOpD + 3;
}
// offset of the class's matrix in the sample's block; (0, 0): size of the block
__host__ __device__ inline int op_offset(int pic, int qic, int P, int Q)
{
    int o = 0;
    for (int c = 0; c < kOpClasses; ++c) {
        if (op_pic(c) == pic && op_qic(c) == qic) return o;
        const int n = op_n(op_pic(c), op_qic(c));
        if (op_has(op_pic(c), op_qic(c), P, Q)) o += n * op_ld(n);
    }
    return o;
}
// row / column of interior node (i, j) of grid (p, kOpD + 2 - p) in a class's matrix
__host__ __device__ inline int op_index(int p, int i, int j, int qic)
{
    int o = 0;
    for (int pp = 1; pp < p; ++pp)
        if (kOpD + 2 - pp <= qic) o += ((1 << pp) - 1) * ((1 << (kOpD + 2 - pp)) - 1);
    return o + (j - 1) * ((1 << p) - 1) + (i - 1);
}

// One matrix per CTA: sample blockIdx.x, class kOpClasses - 1 - blockIdx.y (the largest
// first).  A lane runs the mu calls on the unit vector of its column through the phase
// program of the low-diagonal tables (below), whose entries are uniform over the lanes;
// the rows of the block share the entries of a phase.  Bound by the latency of about 170
// short phases in FP32 and by the FP64 pipe in FP64, so what does not depend on the
// column (faces, the reciprocal of the diagonal, the kappa weights) is made once per node
// of the triangle, and all classes run side by side.  Measured, against one launch per
// class with the reciprocals in every lane: FP64, 64 samples 2.85 -> 0.8 ms; FP32, 6 samples
// 0.48 -> 0.12 ms.
constexpr int kOpThreads = 768;
template <class T>
struct __align__(16) OpNode {
    T aw, ae, as, an;
    T d, rd;   // diagonal and its reciprocal
    T kx, ky;  // kappa weights of the two children
};
template <class T>
__host__ __device__ __forceinline__ size_t op_smem(int nent, int nops, const LowPlanes& lp, int n)
{
    return sizeof(uint4) * nent + sizeof(uint2) * ((nops + 1) & ~1) + sizeof(OpNode<T>) * lp.nu + sizeof(T) * (size_t)(2 * lp.nu + lp.nr) * n;
}
template <class T>
__global__ void __launch_bounds__(kOpThreads) k_lowop(const SampleInfo* samples, const T* img, int64_t istride, int ify,
                                                     const LowDesc* desc, const uint4* ent, const uint2* rprog, LowPlanes lp,
                                                     int mu, T omega, T* op)
{
    const SampleInfo S = samples[blockIdx.x];
    const int cls = kOpClasses - 1 - blockIdx.y, pic = op_pic(cls), qic = op_qic(cls);
    if (!op_has(pic, qic, S.P, S.Q)) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const LowDesc& D = desc[cls];
    const int n = op_n(pic, qic), ld = op_ld(n), nc = n, nent = D.e1 - D.e0, nops = D.nops;
    uint4* sent = (uint4*)smem_raw;
    uint2* sprog = (uint2*)(sent + nent);
    OpNode<T>* node = (OpNode<T>*)(sprog + ((nops + 1) & ~1));  // [slot]
    T* u = (T*)(node + lp.nu);                                 // [slot][column]
    T* b = u + lp.nu * nc;
    T* r = b + lp.nu * nc;
    const int tid = threadIdx.x;
    constexpr int nt = kOpThreads;
    for (int k = tid; k < nent; k += nt) sent[k] = ent[D.e0 + k];
    for (int k = tid; k < nops; k += nt) sprog[k] = rprog[D.prog + k];
    for (int k = tid; k < 2 * lp.nu * nc; k += nt) u[k] = T(0);
    __syncthreads();
    const T *fx = img + (int64_t)blockIdx.x * istride, *fy = fx + ify;
    for (int d = 0; d <= kOpD; ++d) {
        for (int e = tid; e < D.cnt[d][LK_RESID]; e += nt) {  // every node of the diagonal
            const uint4 v = sent[D.off[d][LK_RESID] - D.e0 + e];
            const int xw = v.z >> 16, ys = v.w & 0xFFFF;
            OpNode<T>& N = node[v.x & 0xFFFF];
            N.aw = fx[xw]; N.ae = fx[xw + 1]; N.as = fy[ys]; N.an = fy[ys + 1];
            N.d = N.aw + N.ae + N.as + N.an;
            N.rd = rcp_of(N.d);
            const T cx = N.aw + N.ae, cy = N.as + N.an, x2 = cx * cx, y2 = cy * cy, s = rcp_of(x2 + y2);
            N.kx = x2 * s;
            N.ky = y2 * s;
        }
    }
    const int bx = (n + 31) & ~31, g = tid / bx, col = tid - g * bx, ng = nt / bx;
    const bool on = col < nc && g < ng;
    // slot of unknown t in the u and b planes
    auto slot_of = [&](int t) {
        for (int k = 0; k < lp.ngrid; ++k) {
            const LowGrid G = lp.g[k];
            if (G.p + G.q - 2 != kOpD || G.p > pic || G.q > qic) continue;
            const int nx1 = (1 << G.p) - 1, ny1 = (1 << G.q) - 1;
            if (t < nx1 * ny1) return G.gu + low_rb(nx1, ny1, 1 + t % nx1, 1 + t / nx1);
            t -= nx1 * ny1;
        }
        return 0;
    };
    if (g == 0 && on) b[slot_of(col) * nc + col] = T(1);
    __syncthreads();
    for (int call = 0; call < mu; ++call)
        for (int o = 0; o < nops; ++o) {
            const uint2 w = sprog[o];
            const int kind = w.x & 7, cnt = (int)(w.x >> 3), off = (int)w.y;
            if (on)
                for (int e = g; e < cnt; e += ng) {
                    const uint4 v = sent[off + e];
                    auto U = [&](uint32_t s) { return u[s * nc + col]; };
                    const uint32_t c = v.x & 0xFFFF;
                    const OpNode<T>& N = node[c];
                    if (kind <= LK_RESID) {
                        const T x = N.aw * U(v.x >> 16) + N.ae * U(v.y & 0xFFFF), y = N.as * U(v.y >> 16) + N.an * U(v.z & 0xFFFF);
                        if (kind == LK_RESID) r[(v.w >> 16) * nc + col] = b[c * nc + col] - (N.d * U(c) - x - y);
                        else u[c * nc + col] = (b[c * nc + col] + (x + y)) * N.rd;
                    } else if (kind == LK_RESTRICT) {
                        const int rx = v.x >> 16, ry = v.y & 0xFFFF, wy = v.y >> 16;
                        const bool hx = v.z & 1, hy = v.z & 2;
                        T vx = T(0), vy = T(0);
                        if (hx) vx = T(0.25) * (r[(rx - 1) * nc + col] + T(2) * r[rx * nc + col] + r[(rx + 1) * nc + col]);
                        if (hy) vy = T(0.25) * (r[(ry - wy) * nc + col] + T(2) * r[ry * nc + col] + r[(ry + wy) * nc + col]);
                        b[c * nc + col] = (hx && hy) ? T(0.5) * vx + T(0.5) * vy : (hx ? vx : vy);
                        u[c * nc + col] = T(0);
                    } else {
                        const bool hx = (v.w >> 16) & 1, hy = (v.w >> 17) & 1;
                        T vx = T(0), vy = T(0);
                        if (hx) vx = T(0.5) * (U(v.y >> 16) + U(v.z & 0xFFFF));
                        if (hy) vy = T(0.5) * (U(v.z >> 16) + U(v.w & 0xFFFF));
                        const T corr = (hx && hy) ? N.kx * vx + N.ky * vy : (hx ? vx : vy);
                        u[c * nc + col] += omega * corr;
                    }
                }
            __syncthreads();
        }
    T* M = op + S.op_off + op_offset(pic, qic, S.P, S.Q);
    for (int k = tid; k < n * ld; k += nt) {
        const int t = k / ld, s = k - t * ld;
        M[k] = s < n ? u[slot_of(t) * nc + s] : T(0);
    }
}

// ------------------------------------------------------------------ visits --

// An array of T in shared memory by its 32-bit address: element addresses are one
// integer add, and an access is one instruction with an immediate offset.  (Through
// C++ pointers the visits spent 90 % of their instructions on 64-bit address
// arithmetic and control.)
template <class T> struct Vec2;
template <> struct Vec2<float> { typedef float2 V; };
template <> struct Vec2<double> { typedef double2 V; };
template <class T>
struct Sm {
    uint32_t a;
    typedef typename Vec2<T>::V V;
    __device__ __forceinline__ Sm at(int i) const { return Sm{a + (uint32_t)i * (uint32_t)sizeof(T)}; }
    __device__ __forceinline__ T ld() const
    {
        T v;
        if constexpr (sizeof(T) == 4) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
        else asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
        return v;
    }
    __device__ __forceinline__ V ld2() const  // two elements, 2 sizeof(T) aligned
    {
        V v;
        if constexpr (sizeof(T) == 4) asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
        else asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
        return v;
    }
    __device__ __forceinline__ void st(T v) const
    {
        if constexpr (sizeof(T) == 4) asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
        else asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
    }
    __device__ __forceinline__ void st2(T x, T y) const
    {
        if constexpr (sizeof(T) == 4) asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
        else asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(x), "d"(y) : "memory");
    }
};

// The launches of a cycle are a chain of short dependent kernels.  Each lets the next one
// start at once and waits for the one before it only when it has read what does not
// change during a solve (lists, coefficients, matrices): what follows launch_next in a
// kernel up to wait_previous runs under its predecessor.  A kernel that waits waits for the
// end of the whole previous kernel, hence of all before it.  Measured with FP32 cycles:
// 180 samples of 4 to 128 cells a side 32.0 -> 26.4 ms, 192 of 256 x 256 327 -> 308 ms.
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One item's hierarchy (pic, qic: its top grid clipped to the diagonals held)
// on chip: diagonals lo..hi; below lo (when lo = kOpD + 1) the matrix.
template <class T>
struct MidItem {
    Sm<T> u;   // per diagonal: cells of its grids, then a pad of zeros (the last grid's north boundary)
    Sm<T> b;   // cells
    Sm<T> ax;  // cells
    Sm<T> ay;
    Sm<T> r;   // residual of the diagonal being restricted: the red node of each pair (every cell when nu1 = 0)
    Sm<T> di;  // FP64: 1 / diagonal of each cell, 0 at a boundary cell
    Sm<T> kp;  // FP64: kappa weight of the x-child at the black node of each pair
    Sm<T> M;   // the matrix (lo = kOpD + 1)
    Sm<T> b3;  // its right-hand side, compact
    Sm<T> u3;  // its result: the cells of diagonal kOpD
    const int2* at;  // first word of each diagonal in b, ax, ay (x) and in u (y)
    int pic, qic, lo, klo, hi;
    int n3, ld3;
};

__host__ __device__ __forceinline__ int mid_plo(int d, int qic) { return d + 2 - qic > 1 ? d + 2 - qic : 1; }
__host__ __device__ __forceinline__ int mid_phi(int d, int pic) { return d + 1 < pic ? d + 1 : pic; }
__host__ __device__ __forceinline__ int mid_cells(int d, int pic, int qic)
{
    const int ng = mid_phi(d, pic) - mid_plo(d, qic) + 1;
    return ng > 0 ? ng << (d + 2) : 0;
}
__host__ __device__ __forceinline__ int mid_pad(int d, int pic) { return 4 + (1 << mid_phi(d, pic)); }

// words of the arrays of an item: cells of the diagonals whose coefficients and b are
// stored (klo..hi; the ones below are kept in registers), cells of all, their pads, the residual
struct MidWords { int cells, ucells, pads, r; };
__host__ __device__ __forceinline__ MidWords mid_words(int pic, int qic, int lo, int klo, int hi, int nu1)
{
    MidWords w{0, 0, 0, 0};
    for (int d = lo; d <= hi; ++d) {
        const int c = mid_cells(d, pic, qic), r = nu1 == 0 ? c : c >> 1;
        w.cells += d >= klo ? c : 0;
        w.ucells += c;
        w.pads += mid_pad(d, pic);
        w.r = r > w.r ? r : w.r;
    }
    return w;
}
// In FP64 a reciprocal is a dozen operations of the pipe that bounds the cycles, so the
// diagonals' and the kappa weights are made once per launch: words per pair of cells.  (FP32
// has the MUFU pipe for them, and kept.cuh.)  With the sums of pair_red as chains: FP64 solve
// of 64 samples of 32 x 32 8.53 -> 6.61 ms, convergence study on 64 x 64 24.8 -> 20.5 ms.
template <class T> constexpr int mid_aux() { return sizeof(T) == 8 ? 3 : 0; }
constexpr int kU3 = 4 * 32 + 20;  // cells of diagonal kOpD and their pad
template <class T>
__host__ __device__ __forceinline__ int mid_total(int pic, int qic, int lo, int klo, int hi, int nu1)
{
    const MidWords w = mid_words(pic, qic, lo, klo, hi, nu1);
    int t = 3 * w.cells + w.ucells + w.pads + w.r + mid_aux<T>() * (w.cells >> 1);
    if (lo > 0) {
        const int n = op_n(pic < 4 ? pic : 4, qic < 4 ? qic : 4);
        t += n * op_ld(n) + kOpN + kU3;
    }
    return t;
}

// The pointers of an item whose words start at sm (16-byte aligned), and the table
// of its diagonals (written by thread 0; a CTA barrier comes before its first use).
template <class T>
__device__ __forceinline__ MidItem<T> mid_item(T* sm, int2* at, int pic, int qic, int lo, int klo, int hi, int nu1)
{
    MidItem<T> m;
    const MidWords w = mid_words(pic, qic, lo, klo, hi, nu1);
    m.pic = pic; m.qic = qic; m.lo = lo; m.klo = klo; m.hi = hi;
    m.n3 = op_n(pic < 4 ? pic : 4, qic < 4 ? qic : 4);
    m.ld3 = op_ld(m.n3);
    m.M = Sm<T>{(uint32_t)__cvta_generic_to_shared(sm)};
    m.b3 = m.M.at(lo > 0 ? m.n3 * m.ld3 : 0);
    m.u3 = m.b3.at(lo > 0 ? kOpN : 0);
    m.ax = m.u3.at(lo > 0 ? kU3 : 0);
    m.ay = m.ax.at(w.cells);
    m.b = m.ay.at(w.cells);
    m.r = m.b.at(w.cells);
    m.u = m.r.at(w.r);
    m.di = m.u.at(w.ucells + w.pads);
    m.kp = m.di.at(w.cells);
    m.at = at;
    if (threadIdx.x == 0) {
        int c = 0, u = 0;
        for (int d = lo; d <= hi; ++d) {
            at[d] = make_int2(c, u);
            const int n = mid_cells(d, pic, qic);
            c += d >= klo ? n : 0;
            u += n + mid_pad(d, pic);
        }
    }
    return m;
}

// arrays of one diagonal
template <class T>
struct MidDiag {
    Sm<T> u, b, ax, ay, di, kp;
    int plo, ng;
};
template <class T>
__device__ __forceinline__ MidDiag<T> mid_diag(const MidItem<T>& m, int d)
{
    MidDiag<T> v;
    const int2 o = m.at[d];
    v.u = m.u.at(o.y);
    v.b = m.b.at(o.x);
    v.ax = m.ax.at(o.x);
    v.ay = m.ay.at(o.x);
    if constexpr (mid_aux<T>() > 0) {
        v.di = m.di.at(o.x);
        v.kp = m.kp.at(o.x >> 1);
    }
    v.plo = mid_plo(d, m.qic);
    v.ng = mid_phi(d, m.pic) - v.plo + 1;
    return v;
}

// A thread's pair of nodes during a visit: the red and the black one.  The
// coefficients and b are divided by the node's diagonal, so that an update is
// u = b + sum a u and the residual is diagonal * (b + sum a u - u); the kappa
// weights, ratios of squared coefficients of one node, do not see the division.
// A boundary node takes part with zero coefficients and stays zero, so the half
// sweeps have no branches; a pair of row 0 or past the end keeps both
// nodes on one zero word (eR = nx = 0).
template <class T>
struct Pair {
    T pR, oR, sR, nR, bR, uR;  // red: face to the partner, outer horizontal, south and north face
    T pK, oK, sK, nK, bK, uK;  // black
    T dR;                      // diagonal of the red node
    uint32_t aR;               // address of u at the red node; the black one's: aR - e
    uint32_t e;                // bytes to the red node's outer horizontal neighbour (the black one's: -e)
    uint32_t w;                // bytes of a row
};

// The pair from its faces and values (below) and the reciprocals iA, iB of the diagonals.
template <class T>
__device__ __forceinline__ void pair_scale(Pair<T>& P, uint32_t aA, int nx, bool ok, bool redB, T aw, T am, T ae, T sA, T sB,
                                           T nA, T nB, T bA, T bB, T uA, T uB, T iA, T iB, T& iR, T& iK)
{
    constexpr uint32_t es = sizeof(T);
    const T oR = redB ? ae : aw, sR = redB ? sB : sA, nR = redB ? nB : nA;
    iR = redB ? iB : iA;
    iK = redB ? iA : iB;
    P.w = ok ? nx * es : 0u;
    P.aR = aA + (ok && redB ? es : 0u);
    P.e = ok ? (redB ? es : 0u - es) : 0u;
    P.dR = oR + am + sR + nR;
    P.pR = iR * am; P.pK = iK * am;
    P.oR = iR * oR; P.oK = iK * (redB ? aw : ae);
    P.sR = iR * sR; P.sK = iK * (redB ? sA : sB);
    P.nR = iR * nR; P.nK = iK * (redB ? nA : nB);
    P.bR = iR * (redB ? bB : bA); P.bK = iK * (redB ? bA : bB);
    P.uR = redB ? uB : uA; P.uK = redB ? uA : uB;
}

// From the faces and values of nodes A (even column, u at address aA) and B: aw, am,
// ae the faces west of A, between, east of B; s, n the south and north ones.  ok: a row
// of nodes; hasA: A is not the west boundary; redB: B is the red node.  iR, iK: what the
// nodes' values were scaled with.
template <class T>
__device__ __forceinline__ void pair_set(Pair<T>& P, uint32_t aA, int nx, bool ok, bool hasA, bool redB, T aw, T am, T ae,
                                         T sA, T sB, T nA, T nB, T bA, T bB, T uA, T uB, T& iR, T& iK)
{
    const T dA = aw + am + sA + nA, dB = am + ae + sB + nB;
    const T iA = hasA ? rcp_of(dA) : T(0), iB = ok ? rcp_of(dB) : T(0);
    pair_scale(P, aA, nx, ok, redB, aw, am, ae, sA, sB, nA, nB, bA, bB, uA, uB, iA, iB, iR, iK);
    P.dR = redB ? dB : dA;
}

// Pair m of diagonal d; dump: the zero word for pairs past the end.
template <class T>
__device__ __forceinline__ void pair_load(Pair<T>& P, const MidDiag<T>& g, int d, int m, int np, int dump)
{
    const bool in = m < np;
    const int cA = in ? 2 * m : dump, p = g.plo + (in ? m >> (d + 1) : 0), cell = cA & ((4 << d) - 1);
    const int nx = 1 << p, i = cell & (nx - 1), j = cell >> p;
    const bool ok = in && j > 0, hasA = ok && i > 0, redB = j & 1;  // (i, j), i even, is red when j is even
    const int c = ok ? cA : 1 << g.plo;  // any node's cell where there is none
    const Sm<T> x = g.ax.at(c), y = g.ay.at(c);
    const T aw = x.at(-1).ld();
    const auto ae = x.ld2(), an = y.ld2(), as = y.at(ok ? -nx : 0).ld2(), bb = g.b.at(c).ld2(), uu = g.u.at(c).ld2();
    T iR, iK;
    if constexpr (mid_aux<T>() > 0) {
        const auto ii = g.di.at(c).ld2();
        pair_scale(P, g.u.at(cA).a, nx, ok, redB, aw, ae.x, ae.y, as.x, as.y, an.x, an.y, bb.x, bb.y, ok ? uu.x : T(0),
                   ok ? uu.y : T(0), ok ? ii.x : T(0), ok ? ii.y : T(0), iR, iK);
    } else {
        pair_set(P, g.u.at(cA).a, nx, ok, hasA, redB, aw, ae.x, ae.y, as.x, as.y, an.x, an.y, bb.x, bb.y, ok ? uu.x : T(0),
                 ok ? uu.y : T(0), iR, iK);
    }
}

// b + sum a u of the red / black node.  FP64: as four operations of its pipe instead of six
// (in FP32 the sum of two pairs and the chain take the same time: 256 x 256 0.5 % apart).
template <class T>
__device__ __forceinline__ T pair_red(const Pair<T>& a)
{
    const T o = Sm<T>{a.aR + a.e}.ld(), s = Sm<T>{a.aR - a.w}.ld(), n = Sm<T>{a.aR + a.w}.ld();
    if constexpr (sizeof(T) == 8) return fma(a.pR, a.uK, fma(a.oR, o, fma(a.sR, s, fma(a.nR, n, a.bR))));
    return a.bR + ((a.pR * a.uK + a.oR * o) + (a.sR * s + a.nR * n));
}
template <class T>
__device__ __forceinline__ T pair_black(const Pair<T>& a)
{
    const uint32_t k = a.aR - a.e;
    const T o = Sm<T>{k - a.e}.ld(), s = Sm<T>{k - a.w}.ld(), n = Sm<T>{k + a.w}.ld();
    if constexpr (sizeof(T) == 8) return fma(a.pK, a.uR, fma(a.oK, o, fma(a.sK, s, fma(a.nK, n, a.bK))));
    return a.bK + ((a.pK * a.uR + a.oK * o) + (a.sK * s + a.nK * n));
}

// nu red-black Gauss-Seidel sweeps over the thread's pairs; zero: u is zero on
// entry, so the first red half sweep has no neighbours to read.  A half sweep reads
// nodes of the other colour only: all its loads come before its stores.
// on: bit k, this warp has pairs in round k (the same for its lanes).
template <class T, int NP>
__device__ __forceinline__ void mid_sweeps(Pair<T> (&P)[NP], uint32_t on, int nu, bool zero)
{
    for (int s = 0; s < nu; ++s) {
#pragma unroll
        for (int k = 0; k < NP; ++k)
            if (on >> k & 1) P[k].uR = zero ? P[k].bR : pair_red(P[k]);
#pragma unroll
        for (int k = 0; k < NP; ++k)
            if (on >> k & 1) Sm<T>{P[k].aR}.st(P[k].uR);
        zero = false;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < NP; ++k)
            if (on >> k & 1) P[k].uK = pair_black(P[k]);
#pragma unroll
        for (int k = 0; k < NP; ++k)
            if (on >> k & 1) Sm<T>{P[k].aR - P[k].e}.st(P[k].uK);
        __syncthreads();
    }
}

template <int NP>
__device__ __forceinline__ uint32_t pairs_of_warp(int np)
{
    uint32_t on = 0;
#pragma unroll
    for (int k = 0; k < NP; ++k) on |= (uint32_t)((threadIdx.x & ~31) + k * blockDim.x < np) << k;
    return on;
}

// Eq. (2.3) into the children of diagonal d from m.r.  RED: m.r holds the red
// node of each pair (pair k of a row: column 2k of an even row, 2k + 1 of an odd
// one) and the black nodes are zero, so half of the weights drop out.
template <class T, bool RED>
__device__ __forceinline__ void mid_restrict(const MidItem<T>& m, int d)
{
    const int pplo = mid_plo(d, m.qic), plo = mid_plo(d - 1, m.qic), ngc = mid_phi(d - 1, m.pic) - plo + 1;
    const bool op = d == m.lo && m.lo > 0;
    const int2 o = m.at[op ? d : d - 1];
    const Sm<T> cb = m.b.at(o.x), cu = m.u.at(o.y);  // not used when op
    for (int k = threadIdx.x; k < (ngc << d); k += blockDim.x) {
        // cells A = (i, j), i even, and B = (i + 1, j) of child (p, q)
        const int cA = 2 * k, p = plo + (k >> d), q = d + 1 - p, cell = cA & ((2 << d) - 1);
        const int nx = 1 << p, i = cell & (nx - 1), j = cell >> p;
        if (j == 0) continue;
        const bool hx = p < m.pic, hy = q < m.qic;
        T xA = T(0), xB = T(0), yA = T(0), yB = T(0);
        if constexpr (RED) {
            if (hx) {  // grid (p+1, q): row j has nx pairs, around columns 2i and 2i + 2
                const Sm<T> r = m.r.at(((p + 1 - pplo) << (d + 1)) + (j << p) + i);
                const T rm = r.at(-1).ld(), r0 = r.ld(), r1 = r.at(1).ld();
                xA = (j & 1) ? T(0.25) * (rm + r0) : T(0.5) * r0;
                xB = (j & 1) ? T(0.25) * (r0 + r1) : T(0.5) * r1;
            }
            if (hy) {  // grid (p, q+1): rows 2j - 1 .. 2j + 1 of nx / 2 pairs
                const int h = nx >> 1;
                const Sm<T> r = m.r.at(((p - pplo) << (d + 1)) + j * nx + (i >> 1));
                yA = T(0.5) * r.ld();
                yB = T(0.25) * (r.at(-h).ld() + r.at(h).ld());
            }
        } else {
            if (hx) {
                const Sm<T> r = m.r.at(((p + 1 - pplo) << (d + 2)) + (j << (p + 1)) + 2 * i);
                const T rm = r.at(-1).ld();
                const auto r0 = r.ld2(), r2 = r.at(2).ld2();
                xA = T(0.25) * (rm + T(2) * r0.x + r0.y);
                xB = T(0.25) * (r0.y + T(2) * r2.x + r2.y);
            }
            if (hy) {
                const Sm<T> r = m.r.at(((p - pplo) << (d + 2)) + (j << (p + 1)) + i);
                const auto r0 = r.at(-nx).ld2(), r1 = r.ld2(), r2 = r.at(nx).ld2();
                yA = T(0.25) * (r0.x + T(2) * r1.x + r2.x);
                yB = T(0.25) * (r0.y + T(2) * r1.y + r2.y);
            }
        }
        T vA = (hx && hy) ? T(0.5) * xA + T(0.5) * yA : (hx ? xA : yA);
        const T vB = (hx && hy) ? T(0.5) * xB + T(0.5) * yB : (hx ? xB : yB);
        if (op) {
            const Sm<T> t = m.b3.at(op_index(p, i, j, m.qic));  // unknown of cell A; B is the next one
            if (i > 0) t.st(vA);
            t.at(1).st(vB);
        } else {
            if (i == 0) vA = T(0);  // the boundary stays zero
            cb.at(cA).st2(vA, vB);
            cu.at(cA).st2(T(0), T(0));
        }
    }
}

// First half of a visit of diagonal d: nu1 sweeps, the residual, Eq. (2.3) into
// diagonal d-1 (whose correction restarts from zero).  After a black half sweep
// the residual of a black node is zero up to the rounding of its own update, so
// only the red nodes' is formed.
template <class T, int NP, bool RESTRICT = true>
__device__ __forceinline__ void mid_pre(const MidItem<T>& m, int d, int nu1, bool zero)
{
    const MidDiag<T> g = mid_diag(m, d);
    const int np = g.ng << (d + 1), tid = threadIdx.x, nt = blockDim.x, dump = 2 * np + (1 << (g.plo + g.ng - 1));
    const uint32_t on = pairs_of_warp<NP>(np);
    Pair<T> P[NP] = {};
#pragma unroll
    for (int k = 0; k < NP; ++k)
        if (on >> k & 1) pair_load(P[k], g, d, tid + k * nt, np, dump);
    if (d == 0) {  // one unknown: solved exactly
        if (on & 1) Sm<T>{P[0].aR}.st(P[0].bR);
        __syncthreads();
        return;
    }
    mid_sweeps<T, NP>(P, on, nu1, zero);
    if (nu1 > 0) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            if (!(on >> k & 1)) continue;
            const T r = P[k].dR * (pair_red(P[k]) - P[k].uR);
            if (tid + k * nt < np) m.r.at(tid + k * nt).st(r);
        }
        __syncthreads();
        if (!RESTRICT) return;
        mid_restrict<T, true>(m, d);
    } else {
        for (int k = tid; k < (g.ng << (d + 2)); k += nt) {
            const int p = g.plo + (k >> (d + 2)), cell = k & ((4 << d) - 1), nx = 1 << p;
            if ((cell & (nx - 1)) == 0 || cell < nx) continue;
            const Sm<T> x = g.ax.at(k), y = g.ay.at(k), u = g.u.at(k);
            const T aw = x.at(-1).ld(), ae = x.ld(), as = y.at(-nx).ld(), an = y.ld();
            m.r.at(k).st(g.b.at(k).ld() - ((aw + ae + as + an) * u.ld() - (aw * u.at(-1).ld() + ae * u.at(1).ld()) -
                                           (as * u.at(-nx).ld() + an * u.at(nx).ld())));
        }
        __syncthreads();
        mid_restrict<T, false>(m, d);
    }
    __syncthreads();
}

// Second half: Eq. (2.4) with the kappa weights of Eq. (2.5), then nu2 sweeps.
// The first red half sweep reads black nodes only and overwrites the red ones, so
// the correction is formed at the black nodes (at both when nu2 = 0).
template <class T, int NP>
__device__ __forceinline__ void mid_post(const MidItem<T>& m, int d, int nu2, T omega)
{
    const MidDiag<T> g = mid_diag(m, d);
    const int np = g.ng << (d + 1), tid = threadIdx.x, nt = blockDim.x, dump = 2 * np + (1 << (g.plo + g.ng - 1));
    const uint32_t on = pairs_of_warp<NP>(np);
    const int plo = mid_plo(d - 1, m.qic);
    const bool op = d == m.lo && m.lo > 0;
    const Sm<T> cu{op ? m.u3.a : m.u.at(m.at[op ? d : d - 1].y).a};
    Pair<T> P[NP] = {};
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int mm = tid + k * nt;
        Pair<T>& a = P[k];
        if (!(on >> k & 1)) continue;
        pair_load(a, g, d, mm, np, dump);
        if (a.w == 0) continue;
        const int p = g.plo + (mm >> (d + 1)), q = d + 2 - p, cell = (2 * mm) & ((4 << d) - 1);
        const int nx = 1 << p, i = cell & (nx - 1), j = cell >> p;
        const bool hx = p > 1, hy = q > 1, redB = j & 1;
        const Sm<T> cx = cu.at(((p - 1 - plo) << (d + 1)) + (j << (p - 1)) + (i >> 1));  // grid (p-1, q): row j, from column i/2
        const Sm<T> cy = cu.at(((p - plo) << (d + 1)) + ((j >> 1) << p) + i);            // grid (p, q-1): from row j/2
        // correction at node A (B = 0) or B (B = 1) from the scaled coefficients
        auto corr = [&](int B, T h0, T h1, T v0, T v1, bool black) {
            T x = T(0), y = T(0);
            if (hx) {
                x = cx.ld();
                if (B) x = T(0.5) * (x + cx.at(1).ld());
            }
            if (hy) {
                y = cy.at(B).ld();
                if (redB) y = T(0.5) * (y + cy.at(nx + B).ld());
            }
            if (!(hx && hy)) return hx ? x : y;
            if constexpr (mid_aux<T>() > 0)
                if (black) return y + g.kp.at(mm).ld() * (x - y);
            const T c1 = h0 + h1, c2 = v0 + v1, x2 = c1 * c1, y2 = c2 * c2, w = rcp_of(x2 + y2);
            return (x2 * w) * x + (y2 * w) * y;
        };
        if (!redB || i > 0) {
            a.uK += omega * corr(redB ? 0 : 1, a.pK, a.oK, a.sK, a.nK, true);
            Sm<T>{a.aR - a.e}.st(a.uK);
        }
        if (nu2 == 0 && (redB || i > 0)) {
            a.uR += omega * corr(redB ? 1 : 0, a.pR, a.oR, a.sR, a.nR, false);
            Sm<T>{a.aR}.st(a.uR);
        }
    }
    __syncthreads();
    mid_sweeps<T, NP>(P, on, nu2, false);
}

// u3 = M b3: two threads a row.
template <class T>
__device__ __forceinline__ void mid_matrix(const MidItem<T>& m)
{
    const int half = m.ld3 >> 1;
    for (int t2 = threadIdx.x; t2 < ((2 * m.n3 + 31) & ~31); t2 += blockDim.x) {
        const int t = t2 >> 1, h = t2 & 1;
        T s0 = T(0), s1 = T(0), s2 = T(0), s3 = T(0);
        if (t < m.n3) {
            const Sm<T> row = m.M.at(t * m.ld3 + h * half), v = m.b3.at(h * half);
            for (int k = 0; k < half; k += 4) {
                const auto a = row.at(k).ld2(), b = row.at(k + 2).ld2(), x = v.at(k).ld2(), y = v.at(k + 2).ld2();
                s0 += a.x * x.x;
                s1 += a.y * x.y;
                s2 += b.x * y.x;
                s3 += b.y * y.y;
            }
        }
        T s = (s0 + s1) + (s2 + s3);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        if (h == 0 && t < m.n3) {
            // cell of unknown t
            const int plo = mid_plo(kOpD, m.qic);
            int p = plo, o = t;
            for (;; ++p) {
                const int nn = ((1 << p) - 1) * ((1 << (kOpD + 2 - p)) - 1);
                if (o < nn) break;
                o -= nn;
            }
            const int nx1 = (1 << p) - 1, j = 1 + o / nx1, i = 1 + o - (j - 1) * nx1;
            m.u3.at(((p - plo) << (kOpD + 2)) + (j << p) + i).st(s);
        }
    }
    __syncthreads();
}

template <class T>
__device__ __forceinline__ void mid_pre_any(const MidItem<T>& m, int d, int nu1, bool zero)
{
    const int np = mid_cells(d, m.pic, m.qic) >> 1;
    if (np <= blockDim.x) mid_pre<T, 1>(m, d, nu1, zero);
    else if (np <= 2 * blockDim.x) mid_pre<T, 2>(m, d, nu1, zero);
    else mid_pre<T, 4>(m, d, nu1, zero);
}
template <class T>
__device__ __forceinline__ void mid_post_any(const MidItem<T>& m, int d, int nu2, T omega)
{
    const int np = mid_cells(d, m.pic, m.qic) >> 1;
    if (np <= blockDim.x) mid_post<T, 1>(m, d, nu2, omega);
    else if (np <= 2 * blockDim.x) mid_post<T, 2>(m, d, nu2, omega);
    else mid_post<T, 4>(m, d, nu2, omega);
}

// One mu-cycle of Algorithm 1 on diagonal m.hi, the recursion as a loop:
// `made` counts the calls already made below each diagonal, four bits each.
// Diagonal 0 does not change between the mu calls of one visit (one unknown,
// solved exactly), so it is called once.
template <class T>
__device__ __forceinline__ void mid_cycle(const MidItem<T>& m, int mu, int nu1, int nu2, T omega, bool zero)
{
    int d = m.hi;
    uint64_t made = 0;
    for (;;) {
        mid_pre_any(m, d, nu1, zero);
        if (d > m.lo) {
            made &= ~(15ull << (4 * d));
            zero = true;
            --d;
            continue;
        }
        if (m.lo > 0) {
            mid_matrix(m);
            mid_post_any(m, d, nu2, omega);
        }
        for (;;) {
            if (d == m.hi) return;
            ++d;
            made += 1ull << (4 * d);
            const int k = (int)(made >> (4 * d)) & 15;
            if (k < (d == 1 ? 1 : mu)) {
                zero = false;
                --d;
                break;
            }
            mid_post_any(m, d, nu2, omega);
        }
    }
}

// Coefficients, zeros and the matrix of an item into shared memory.
template <class T>
__device__ __forceinline__ void mid_fill(const MidItem<T>& m, const SampleInfo& S, const T* ax, const T* ay, const T* op)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    const MidWords w = mid_words(m.pic, m.qic, m.lo, m.klo, m.hi, 1);
    const T *gx = ax + S.node_off, *gy = ay + S.node_off;
    int c0 = 0;
    for (int d = m.klo; d <= m.hi; ++d) {
        const int nc = mid_cells(d, m.pic, m.qic), plo = mid_plo(d, m.qic);
#pragma unroll 2
        for (int k = tid; k < nc; k += nt) {  // cell (i, j) is node (i, j) of rows of 2^p + 1
            const int p = plo + (k >> (d + 2)), cell = k & ((4 << d) - 1);
            const int o = grid_offset32(p, d + 2 - p, S.Q) + cell + (cell >> p);
            const T x = gx[o], y = gy[o];
            m.ax.at(c0 + k).st(x);
            m.ay.at(c0 + k).st(y);
            if constexpr (mid_aux<T>() > 0) {
                const int i = cell & ((1 << p) - 1), j = cell >> p;
                T inv = T(0), kx = T(0);
                if (i > 0 && j > 0) {
                    const T aw = gx[o - 1], as = gy[o - (1 << p) - 1], cx = aw + x, cy = as + y, x2 = cx * cx, y2 = cy * cy;
                    inv = rcp_of(cx + cy);
                    kx = x2 * rcp_of(x2 + y2);
                }
                m.di.at(c0 + k).st(inv);
                if ((i + j) & 1) m.kp.at((c0 + k) >> 1).st(kx);
            }
        }
        c0 += nc;
    }
    for (int k = tid; k < w.cells; k += nt) m.b.at(k).st(T(0));  // boundary nodes read it (with zero coefficients)
    for (int k = tid; k < w.ucells + w.pads; k += nt) m.u.at(k).st(T(0));
    if (m.lo > 0) {
        const T* M = op + S.op_off + op_offset(m.pic < 4 ? m.pic : 4, m.qic < 4 ? m.qic : 4, S.P, S.Q);
        for (int k = 2 * tid; k < m.n3 * m.ld3; k += 2 * nt) {
            const auto v = *reinterpret_cast<const typename Vec2<T>::V*>(M + k);
            m.M.at(k).st2(v.x, v.y);
        }
        for (int k = tid; k < kOpN; k += nt) m.b3.at(k).st(T(0));
        for (int k = tid; k < kU3; k += nt) m.u3.at(k).st(T(0));
    }
}

// b of diagonal kMidD from the restrictions its parents left in the item's scratch, and u
// back to it.
template <class T>
__device__ __forceinline__ void mid_take(const MidItem<T>& m, int64_t scr, int pi, int qi, const T* sbx, const T* sby)
{
    const MidDiag<T> g = mid_diag(m, kMidD);
    const T *bx = sbx + scr, *by = sby + scr;
#pragma unroll 2
    for (int k = threadIdx.x; k < g.ng << (kMidD + 2); k += blockDim.x) {
        const int p = g.plo + (k >> (kMidD + 2)), q = kMidD + 2 - p, cell = k & ((4 << kMidD) - 1);
        const int o = grid_offset32(p, q, qi) + cell + (cell >> p);
        const bool hx = p < pi, hy = q < qi;
        const T v = (hx && hy) ? T(0.5) * bx[o] + T(0.5) * by[o] : (hx ? bx[o] : by[o]);
        if (cell >> p && cell & ((1 << p) - 1)) g.b.at(k).st(v);
    }
}
template <class T>
__device__ __forceinline__ void mid_give(const MidItem<T>& m, int64_t scr, int qi, T* su)
{
    const MidDiag<T> g = mid_diag(m, kMidD);
    T* dst = su + scr;
    for (int k = threadIdx.x; k < g.ng << (kMidD + 2); k += blockDim.x) {  // column 0 and row 0 are zeros of the layout
        const int p = g.plo + (k >> (kMidD + 2)), q = kMidD + 2 - p, cell = k & ((4 << kMidD) - 1);
        const int o = grid_offset32(p, q, qi) + cell + (cell >> p);
        dst[o] = g.u.at(k).ld();
        if ((cell & ((1 << p) - 1)) == (1 << p) - 1) dst[o + 1] = T(0);  // the other two sides
        if (cell >> p == (1 << q) - 1) {
            dst[o + (1 << p) + 1] = T(0);
            if ((cell & ((1 << p) - 1)) == (1 << p) - 1) dst[o + (1 << p) + 2] = T(0);
        }
    }
}

// The mu calls at diagonal kMidD inside a visit of diagonal kMidD + 1 of a larger item.
template <class T>
__global__ void __launch_bounds__(kMidThreads, sizeof(T) == 4 ? 3 : 1)
    k_mid(DevCtx cx, T* su, const T* sbx, const T* sby, const T* ax, const T* ay, const T* op, CycleParams cp)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const TaskRef t = resolve(cx);
    const SampleInfo& S = cx.samples[t.s];
    const int pi = t.seg->pi, qi = t.seg->qi;
    __shared__ int2 at[kMidMax + 1];
    const MidItem<T> m = mid_item<T>((T*)smem_raw, at, min(pi, kMidD + 1), min(qi, kMidD + 1), kOpD + 1, kOpD + 1, kMidD, cp.nu1);
    mid_fill(m, S, ax, ay, op);
    __syncthreads();
    mid_take(m, t.scr, pi, qi, sbx, sby);
    __syncthreads();
    for (int call = 0; call < cp.mu; ++call) mid_cycle(m, cp.mu, cp.nu1, cp.nu2, (T)cp.omega, call == 0);
    mid_give(m, t.scr, qi, su);
}

// The decision of k_residual: does the item take another cycle?  first: its relative
// residual before the first one (set at step 0).
__device__ __forceinline__ int item_goes_on(int step, double rr, double& first, int max_cycles, double eps, int* status)
{
    if (step == 0) {
        first = rr;
        return 1;
    }
    if (!(rr == rr) || isinf(rr)) {
        atomicOr(status, MSG_SAMPLE_NONFINITE);
        return 0;
    }
    if (rr <= eps) return 0;
    if (step >= max_cycles || (rr > 1.0 && rr > first)) {
        atomicOr(status, MSG_SAMPLE_NOT_CONVERGED);
        return 0;
    }
    return 1;
}

// An item of a low stage, solved whole: Algorithm 2's initial guess, then
// defect-correction cycles until the residual meets eps (or the item stops), the
// decision of k_residual.
template <class T>
__global__ void __launch_bounds__(sizeof(T) == 4 ? 512 : 256) k_item(DevCtx cx, int L, double* u64, const double* ax64, const double* ay64,
                                                          const T* ax, const T* ay, const T* op, CycleParams cp, int max_cycles,
                                                          double eps, int* cycles, double* relres, int* status)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_act;
    const TaskRef t = resolve(cx);
    const SampleInfo& S = cx.samples[t.s];
    const int p = t.seg->pi, q = t.seg->qi, nx = 1 << p, ny = 1 << q, W = nx + 1;
    const int64_t off = S.node_off + grid_offset(p, q, S.Q);
    double* u = u64 + off;
    const double* fx = ax64 + off;
    const double* fy = ay64 + off;
    __shared__ int2 at[kMidMax + 1];
    const int lo = L > kOpD ? kOpD + 1 : 0;
    const MidItem<T> m = mid_item<T>((T*)smem_raw, at, p, q, lo, lo, L, cp.nu1);
    mid_fill(m, S, ax, ay, op);
    item_guess(S, p, q, u64, ax64, ay64);
    __syncthreads();
    const MidDiag<T> g = mid_diag(m, L);
    const int n = (nx - 1) * (ny - 1);
    double first = 0.0;
    for (int step = 0;; ++step) {
        __syncthreads();
        double acc = 0.0;
        for (int k = nx + threadIdx.x; k < nx * ny; k += blockDim.x) {
            const int i = k & (nx - 1), j = k >> p, c = j * W + i;
            if (i == 0) continue;
            const double aw = fx[c - 1], ae = fx[c], as = fy[c - W], an = fy[c];
            const double Au = (aw + ae + as + an) * u[c] - (aw * u[c - 1] + ae * u[c + 1]) - (as * u[c - W] + an * u[c + W]);
            const double r = 1.0 - Au;
            acc += r * r;
            g.b.at(k).st((T)r);
            g.u.at(k).st(T(0));
        }
        const double ss = block_sum(acc);
        if (threadIdx.x == 0) {
            const double rr = sqrt(ss / (double)n);
            const int act = item_goes_on(step, rr, first, max_cycles, eps, &status[t.s]);
            s_act = act;
            if (!act) {
                cycles[t.item] = step;
                relres[t.item] = rr;
            }
        }
        __syncthreads();
        if (!s_act) return;
        mid_cycle(m, cp.mu, cp.nu1, cp.nu2, (T)cp.omega, true);
        for (int k = nx + threadIdx.x; k < nx * ny; k += blockDim.x) {
            const int i = k & (nx - 1), j = k >> p;
            if (i > 0) u[j * W + i] += (double)g.u.at(k).ld();
        }
    }
}

// Convergence study on hierarchies that fit one CTA: residual history of MSG cycles
// on (u, b = 1) from u = 0, FP64, one CTA per sample.
__global__ void __launch_bounds__(256) k_history_chip(DevCtx cx, int L, const double* ax, const double* ay, const double* op,
                                                      CycleParams cp, int ncycles, double* hist)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int2 at[kMidMax + 1];
    const TaskRef t = resolve(cx);
    const SampleInfo& S = cx.samples[t.s];
    const int p = t.seg->pi, q = t.seg->qi, nx = 1 << p, ny = 1 << q;
    const int lo = L > kOpD ? kOpD + 1 : 0;
    const MidItem<double> m = mid_item<double>((double*)smem_raw, at, p, q, lo, lo, L, cp.nu1);
    mid_fill(m, S, ax, ay, op);
    __syncthreads();
    const MidDiag<double> g = mid_diag(m, L);
    for (int k = nx + threadIdx.x; k < nx * ny; k += blockDim.x)
        if (k & (nx - 1)) g.b.at(k).st(1.0);
    const double nb = sqrt((double)(nx - 1) * (ny - 1));
    for (int cyc = 0; cyc <= ncycles; ++cyc) {
        __syncthreads();
        if (cyc > 0) mid_cycle(m, cp.mu, cp.nu1, cp.nu2, cp.omega, cyc == 1);
        double acc = 0.0;
        for (int k = nx + threadIdx.x; k < nx * ny; k += blockDim.x) {
            if ((k & (nx - 1)) == 0) continue;
            const Sm<double> x = g.ax.at(k), y = g.ay.at(k), u = g.u.at(k);
            const double aw = x.at(-1).ld(), ae = x.ld(), as = y.at(-nx).ld(), an = y.ld();
            const double r = 1.0 - ((aw + ae + as + an) * u.ld() - (aw * u.at(-1).ld() + ae * u.at(1).ld()) -
                                    (as * u.at(-nx).ld() + an * u.at(nx).ld()));
            acc += r * r;
        }
        const double ss = block_sum(acc);
        if (threadIdx.x == 0) hist[(int64_t)t.s * (ncycles + 1) + cyc] = sqrt(ss) / nb;
    }
}

// The same on larger hierarchies, between the launches of the cycles (b in sbx, u in su
// of each sample's scratch): start values of the top grid of sample blockIdx.x (blockIdx.y: a
// slice of it; the other way round a study had at most 65535 samples), and one entry of the
// history.
__global__ void k_history_start(int P, int Q, int64_t R, double* su, double* sbx)
{
    const int W = (1 << P) + 1, n = W * ((1 << Q) + 1);
    const int64_t o = (int64_t)blockIdx.x * R + grid_offset(P, Q, Q);
    for (int k = blockIdx.y * blockDim.x + threadIdx.x; k < n; k += gridDim.y * blockDim.x) {
        su[o + k] = 0.0;
        sbx[o + k] = 1.0;  // (the boundary's is not read)
    }
}

__global__ void __launch_bounds__(1024) k_history_norm(int P, int Q, int64_t R, const double* su, const double* ax,
                                                       const double* ay, double* hist, int stride)
{
    const int nx = 1 << P, ny = 1 << Q, W = nx + 1;
    const int64_t o = (int64_t)blockIdx.x * R + grid_offset(P, Q, Q);
    const double *u = su + o, *x = ax + o, *y = ay + o;
    double acc = 0.0;
    for (int k = nx + threadIdx.x; k < nx * ny; k += blockDim.x) {
        const int i = k & (nx - 1), c = k + (k >> P);
        if (i == 0) continue;
        const double aw = x[c - 1], ae = x[c], as = y[c - W], an = y[c];
        const double r = 1.0 - ((aw + ae + as + an) * u[c] - (aw * u[c - 1] + ae * u[c + 1]) - (as * u[c - W] + an * u[c + W]));
        acc += r * r;
    }
    const double ss = block_sum(acc);
    if (threadIdx.x == 0) hist[(int64_t)blockIdx.x * stride] = sqrt(ss) / sqrt((double)(nx - 1) * (ny - 1));
}

}  // namespace msg
