// kept.cuh -- the on-chip cycles with the lowest diagonals' pairs prepared once per launch (FP32).
//
// k_mid and k_item (mid.cuh) make a diagonal's pairs from its coefficients for every visit
// half: index arithmetic, nine loads, two reciprocals and the scaling, about half of its
// instructions, and all of it in front of the visit's first half sweep.  The lowest diagonals
// are visited most (diagonal 4 eight times as often as diagonal 7) and have the fewest pairs,
// so here their pairs are made once: a record of five 16-byte words in shared memory
// (scaled coefficients, scale factors and b, addresses, transfer addresses), read by the
// thread that owns the pair (one a thread and diagonal).  The restriction into such a diagonal
// is computed by the owner of the pair, straight into its b, which also saves the
// barrier behind it.  One piece of code serves all these diagonals: a visit is a chain of a
// few hundred instructions on few warps, and what bounds it is their latency and their
// fetching (with the pairs of three diagonals in registers the code was three times as long
// and a visit half of diagonal 4 took 1400 to 1900 cycles).  Measured, a call of diagonals 3 to
// 6 at nu = (2, 2): 83 us in k_mid, 63.6 us here for the 2688 items of 192 samples (58 and
// 43.7 us for one wave of CTAs).  Tried: records of three diagonals with 896 threads 94 us,
// pairs of three diagonals in registers with 896 threads 94 us.
#pragma once

namespace msg {

constexpr int kKeepMid = 2;        // diagonals 4, 5 of k_mid_kept
constexpr int kKeepItem = 3;       // diagonals 4, 5, 6 of items of stage > 3
constexpr int kKeepLow = 4;        // diagonals 0..3 of items of stage <= 3
constexpr int kKeptThreads = 448;  // of k_mid_kept: a pair of diagonal 5 each, two of diagonal 6
enum { KF_X = 1, KF_Y = 2, KF_REDB = 4, KF_PX = 8, KF_PY = 16, KF_A = 32, KF_OK = 64 };

// Records behind the arrays of an item: per kept diagonal a row for each of its pairs (whole
// warps); field f of row k at (f rows + k) 16 bytes:
//   0  pR oR sR nR      1  pK oK sK nK      2  iR iK bR bK      3  aR e w dR
//   4  {black node's child column | flags << 24, its child row, the pair's residuals in its
//      x-parent, in its y-parent} as addresses
// then, for the children of diagonal lo = kOpD + 1, a row per pair of them, and the cells of
// the matrix's unknowns.
constexpr int kFields = 5;
__host__ __device__ __forceinline__ int kept_rows(int d, int pic, int qic) { return ((mid_cells(d, pic, qic) >> 1) + 31) & ~31; }
__host__ __device__ __forceinline__ int kept_total(int pic, int qic, int lo, int keep, int hi, int nu1)
{
    int t = (mid_total<float>(pic, qic, lo, lo + keep, hi, nu1) + 3) & ~3;
    for (int d = lo; d < lo + keep && d <= hi; ++d) t += 4 * kFields * kept_rows(d, pic, qic);
    return t + (lo > 0 ? 4 * 64 + kOpN : 0);
}

__device__ __forceinline__ uint4 lds4(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts4(uint32_t a, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

struct KeptTables {
    uint32_t rec;     // this thread's row of diagonal lo, field 0
    uint32_t field;   // bytes from one field to the next
    uint32_t opc;     // rows of the children of diagonal lo
    uint32_t rows;    // u3 address of each unknown of the matrix
    uint32_t on;      // bit x: this warp has pairs of diagonal lo + x
    uint32_t last;    // bit x: this thread has one
    int row[4];       // rows before diagonal lo + x
};
template <class T>
__device__ __forceinline__ KeptTables kept_tables(const MidItem<T>& m, int keep, int nu1)
{
    KeptTables t;
    const uint32_t base = m.M.a + (uint32_t)sizeof(T) * ((mid_total<T>(m.pic, m.qic, m.lo, m.klo, m.hi, nu1) + 3) & ~3);
    int n = 0;
    t.on = t.last = 0;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        t.row[x] = n;
        if (x >= keep || m.lo + x > m.hi) continue;
        const int np = mid_cells(m.lo + x, m.pic, m.qic) >> 1;
        n += kept_rows(m.lo + x, m.pic, m.qic);
        t.on |= (uint32_t)((int)(threadIdx.x & ~31) < np) << x;
        t.last |= (uint32_t)((int)threadIdx.x < np) << x;
    }
    t.rec = base + 16 * threadIdx.x;
    t.field = 16 * n;
    t.opc = base + kFields * t.field;
    t.rows = t.opc + 16 * 64;
    return t;
}
// this thread's row of diagonal lo + x
__device__ __forceinline__ uint32_t kept_row(const KeptTables& t, int x)
{
    return t.rec + 16 * (x == 0 ? 0 : x == 1 ? t.row[1] : x == 2 ? t.row[2] : t.row[3]);
}
__device__ __forceinline__ float4 lds4f(uint32_t a)
{
    const uint4 v = lds4(a);
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}
__device__ __forceinline__ uint4 bits4(float x, float y, float z, float w)
{
    return make_uint4(__float_as_uint(x), __float_as_uint(y), __float_as_uint(z), __float_as_uint(w));
}

// The record of this thread's pair of diagonal d.
template <class T>
__device__ __forceinline__ void kept_load(const MidItem<T>& m, const KeptTables& t, int d, const SampleInfo& S, const T* ax,
                                          const T* ay)
{
    if (!(t.on >> (d - m.lo) & 1)) return;
    const int np = mid_cells(d, m.pic, m.qic) >> 1, plo = mid_plo(d, m.qic), tid = threadIdx.x;
    const bool in = tid < np;
    const int p = plo + (in ? tid >> (d + 1) : 0), q = d + 2 - p, nx = 1 << p, W = nx + 1;
    const int cA = in ? 2 * tid : 2 * np + (1 << mid_phi(d, m.pic)), cell = in ? cA & ((4 << d) - 1) : 0;
    const int i = cell & (nx - 1), j = cell >> p;
    const bool ok = in && j > 0, hasA = ok && i > 0, redB = j & 1;
    const int o = grid_offset32(p, q, S.Q) + (ok ? j * W + i : W);
    ax += S.node_off;
    ay += S.node_off;
    const T aw = ax[o - 1], am = ax[o], ae = ax[o + 1], nA = ay[o], nB = ay[o + 1], sA = ay[o - W], sB = ay[o + 1 - W];
    Pair<T> P;
    T iR, iK;
    pair_set(P, m.u.at(m.at[d].y + cA).a, nx, ok, hasA, redB, aw, am, ae, sA, sB, nA, nB, T(0), T(0), T(0), T(0), iR, iK);
    const bool op = d == m.lo && m.lo > 0, hx = ok && p > 1, hy = ok && q > 1;
    const bool px = ok && d < m.hi && p < m.pic, py = ok && d < m.hi && q < m.qic;
    uint4 g = make_uint4(0, 0, 0, 0);
    if (d > 0) {
        const Sm<T> cu{op ? m.u3.a : m.u.at(m.at[op ? d : d - 1].y).a};
        const int cplo = mid_plo(d - 1, m.qic);
        if (hx) g.x = cu.at(((p - 1 - cplo) << (d + 1)) + (j << (p - 1)) + (i >> 1)).a;
        if (hy) g.y = cu.at(((p - cplo) << (d + 1)) + ((j >> 1) << p) + (redB ? i : i + 1)).a;
    }
    const int pplo = mid_plo(d + 1, m.qic);
    if (px) g.z = m.r.at(((p + 1 - pplo) << (d + 2)) + (j << p) + i).a;
    if (py) g.w = m.r.at(((p - pplo) << (d + 2)) + j * nx + (i >> 1)).a;
    g.x |= (uint32_t)((hx ? KF_X : 0) | (hy ? KF_Y : 0) | (redB ? KF_REDB : 0) | (px ? KF_PX : 0) | (py ? KF_PY : 0) |
                      (hasA ? KF_A : 0) | (ok ? KF_OK : 0)) << 24;
    const uint32_t a = kept_row(t, d - m.lo);
    sts4(a, bits4(P.pR, P.oR, P.sR, P.nR));
    sts4(a + t.field, bits4(P.pK, P.oK, P.sK, P.nK));
    sts4(a + 2 * t.field, bits4(iR, iK, 0.f, 0.f));
    sts4(a + 3 * t.field, make_uint4(P.aR, P.e, P.w, __float_as_uint(P.dR)));
    sts4(a + 4 * t.field, g);
}

// Tables of the matrix: the unknowns' cells, and per pair of children of diagonal lo
// {residuals in the x-parent, in the y-parent, its unknowns in b3, row bytes | flags << 24}.
template <class T>
__device__ __forceinline__ void kept_op(const MidItem<T>& m, const KeptTables& t)
{
    const int d = m.lo, plo = mid_plo(d - 1, m.qic), n = (mid_phi(d - 1, m.pic) - plo + 1) << d, pplo = mid_plo(d, m.qic);
    for (int k = threadIdx.x; k < 64; k += blockDim.x) {
        uint4 g = make_uint4(0, 0, 0, 0);
        if (k < n) {
            const int p = plo + (k >> d), q = d + 1 - p, cell = (2 * k) & ((2 << d) - 1), nx = 1 << p, i = cell & (nx - 1), j = cell >> p;
            if (j > 0) {
                const bool px = p < m.pic, py = q < m.qic;
                if (px) g.x = m.r.at(((p + 1 - pplo) << (d + 1)) + (j << p) + i).a;
                if (py) g.y = m.r.at(((p - pplo) << (d + 1)) + j * nx + (i >> 1)).a;
                g.z = m.b3.at(op_index(p, i, j, m.qic)).a;
                g.w = nx * (uint32_t)sizeof(T) | (uint32_t)((px ? KF_PX : 0) | (py ? KF_PY : 0) | (i > 0 ? KF_A : 0) | KF_OK | ((j & 1) ? KF_REDB : 0)) << 24;
            }
        }
        sts4(t.opc + 16 * k, g);
    }
    for (int k = threadIdx.x; k < m.n3; k += blockDim.x) {
        int p = mid_plo(kOpD, m.qic), o = k;
        const int p0 = p;
        for (;; ++p) {
            const int nn = ((1 << p) - 1) * ((1 << (kOpD + 2 - p)) - 1);
            if (o < nn) break;
            o -= nn;
        }
        const int nx1 = (1 << p) - 1, j = 1 + o / nx1, i = 1 + o - (j - 1) * nx1;
        const uint32_t a = m.u3.at(((p - p0) << (kOpD + 2)) + (j << p) + i).a;
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(t.rows + 4 * k), "r"(a) : "memory");
    }
}

// Eq. (2.3) at a pair of child nodes A, B from the red residuals (see mid_restrict).
template <class T>
__device__ __forceinline__ void kept_weights(uint32_t rx, uint32_t ry, uint32_t w, uint32_t fl, T& vA, T& vB)
{
    constexpr uint32_t es = sizeof(T);
    T xA = T(0), xB = T(0), yA = T(0), yB = T(0);
    if (fl & KF_PX) {
        const T rm = Sm<T>{rx - es}.ld(), r0 = Sm<T>{rx}.ld(), r1 = Sm<T>{rx + es}.ld();
        xA = (fl & KF_REDB) ? T(0.25) * (rm + r0) : T(0.5) * r0;
        xB = (fl & KF_REDB) ? T(0.25) * (r0 + r1) : T(0.5) * r1;
    }
    if (fl & KF_PY) {
        yA = T(0.5) * Sm<T>{ry}.ld();
        yB = T(0.25) * (Sm<T>{ry - (w >> 1)}.ld() + Sm<T>{ry + (w >> 1)}.ld());
    }
    const bool both = (fl & KF_PX) && (fl & KF_PY);
    vA = both ? T(0.5) * xA + T(0.5) * yA : ((fl & KF_PX) ? xA : yA);
    vB = both ? T(0.5) * xB + T(0.5) * yB : ((fl & KF_PX) ? xB : yB);
    if (!(fl & KF_A)) vA = T(0);
}

// the record's pair, without u
__device__ __forceinline__ void kept_pair(Pair<float>& P, const KeptTables& t, uint32_t a)
{
    const float4 r = lds4f(a), k = lds4f(a + t.field), b = lds4f(a + 2 * t.field);
    const uint4 g = lds4(a + 3 * t.field);
    P.pR = r.x; P.oR = r.y; P.sR = r.z; P.nR = r.w;
    P.pK = k.x; P.oK = k.y; P.sK = k.z; P.nK = k.w;
    P.bR = b.z; P.bK = b.w;
    P.aR = g.x; P.e = g.y; P.w = g.z;
    P.dR = __uint_as_float(g.w);  // (the sum of the faces: the reciprocal of iR is up to three ulp off)
}

// b of the record's pair from nodes' values A and B
__device__ __forceinline__ void kept_b(const KeptTables& t, uint32_t a, bool redB, float vA, float vB)
{
    const Sm<float> f{a + 2 * t.field};
    const float2 i = f.ld2();
    f.at(2).st2(i.x * (redB ? vB : vA), i.y * (redB ? vA : vB));
}

// PRE of a kept diagonal up to the residual
__device__ __forceinline__ void kept_pre(const MidItem<float>& m, const KeptTables& t, int x, int nu1, bool zero)
{
    const uint32_t on = t.on >> x & 1;
    Pair<float> P[1] = {};
    if (on) {
        kept_pair(P[0], t, kept_row(t, x));
        if (!zero) P[0].uK = Sm<float>{P[0].aR - P[0].e}.ld();  // the first red half sweep overwrites the red node
    }
    if (m.lo + x == 0) {  // one unknown: solved exactly
        if (on) Sm<float>{P[0].aR}.st(P[0].bR);
    } else {
        mid_sweeps<float, 1>(P, on, nu1, zero);
        if (on) {
            const float r = P[0].dR * (pair_red(P[0]) - P[0].uR);
            if (t.last >> x & 1) m.r.at(threadIdx.x).st(r);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void kept_post(const KeptTables& t, int x, int nu2, float omega)
{
    const uint32_t on = t.on >> x & 1;
    Pair<float> P[1] = {};
    if (on) {
        Pair<float>& a = P[0];
        const uint32_t row = kept_row(t, x);
        const uint4 g = lds4(row + 4 * t.field);
        kept_pair(a, t, row);
        const uint32_t fl = g.x >> 24;
        a.uK = Sm<float>{a.aR - a.e}.ld();
        if ((fl & KF_OK) && ((fl & KF_A) || !(fl & KF_REDB))) {  // the black node exists
            float cx = 0.f, cy = 0.f;
            if (fl & KF_X) {
                const Sm<float> c{g.x & 0xffffffu};
                cx = c.ld();
                if (!(fl & KF_REDB)) cx = 0.5f * (cx + c.at(1).ld());
            }
            if (fl & KF_Y) {
                cy = Sm<float>{g.y}.ld();
                if (fl & KF_REDB) cy = 0.5f * (cy + Sm<float>{g.y + a.w}.ld());
            }
            float e = (fl & KF_X) ? cx : cy;
            if ((fl & KF_X) && (fl & KF_Y)) {
                const float c1 = a.pK + a.oK, c2 = a.sK + a.nK, x2 = c1 * c1, y2 = c2 * c2, w = rcp_of(x2 + y2);
                e = (x2 * w) * cx + (y2 * w) * cy;
            }
            a.uK += omega * e;
            Sm<float>{a.aR - a.e}.st(a.uK);
        }
    }
    __syncthreads();
    mid_sweeps<float, 1>(P, on, nu2, false);
}

// u3 = M b3, eight threads a row.
template <class T>
__device__ __forceinline__ void kept_matrix(const MidItem<T>& m, const KeptTables& t)
{
    const int part = m.ld3 >> 3, h = threadIdx.x & 7;
    for (int e = threadIdx.x; e < ((8 * m.n3 + 31) & ~31); e += blockDim.x) {
        const int r = e >> 3;
        T s0 = T(0), s1 = T(0);
        if (r < m.n3) {
            const Sm<T> a = m.M.at(r * m.ld3 + h * part), v = m.b3.at(h * part);
            s0 = a.ld() * v.ld();
            for (int k = 1; k < part; k += 2) {  // part is odd
                s0 += a.at(k).ld() * v.at(k).ld();
                s1 += a.at(k + 1).ld() * v.at(k + 1).ld();
            }
        }
        T s = s0 + s1;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        if (h == 0 && r < m.n3) {
            uint32_t a;
            asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a) : "r"(t.rows + 4 * r) : "memory");
            Sm<T>{a}.st(s);
        }
    }
    __syncthreads();
}

// mid_cycle with diagonals lo .. lo + keep - 1 kept (nu1, nu2 > 0); ALL: there is none above.
template <class T, bool ALL>
__device__ __forceinline__ void kept_cycle(const MidItem<T>& m, const KeptTables& t, int keep, int mu, int nu1, int nu2, T omega,
                                           bool zero)
{
    int d = m.hi;
    uint64_t made = 0;
    const int nt = blockDim.x;
    bool up = false;  // POST of d is next, else PRE
    for (;;) {
        const int x = d - m.lo;
        if (up) {
            if (ALL || x < keep) kept_post(t, x, nu2, omega);
            else if (mid_cells(d, m.pic, m.qic) <= 2 * nt) mid_post<T, 1>(m, d, nu2, omega);
            else mid_post<T, 2>(m, d, nu2, omega);
        } else {
            if (ALL || x < keep) kept_pre(m, t, x, nu1, zero);
            else if (mid_cells(d, m.pic, m.qic) <= 2 * nt) mid_pre<T, 1, false>(m, d, nu1, zero);
            else mid_pre<T, 2, false>(m, d, nu1, zero);
            if (d > m.lo) {
                if (ALL || x - 1 < keep) {
                    if (t.on >> (x - 1) & 1) {
                        const uint32_t a = kept_row(t, x - 1);
                        const uint4 g = lds4(a + 4 * t.field);
                        const uint32_t w = lds4(a + 3 * t.field).z;
                        T vA, vB;
                        kept_weights<T>(g.z, g.w, w, g.x >> 24, vA, vB);
                        kept_b(t, a, (g.x >> 24) & KF_REDB, vA, vB);
                    }
                } else {
                    mid_restrict<T, true>(m, d);
                    __syncthreads();
                }
                made &= ~(15ull << (4 * d));
                zero = true;
                --d;
                continue;
            }
            if (m.lo > 0) {
                for (int k = threadIdx.x; k < 64; k += nt) {
                    const uint4 g = lds4(t.opc + 16 * k);
                    const uint32_t fl = g.w >> 24;
                    if (fl & KF_OK) {
                        T vA, vB;
                        kept_weights<T>(g.x, g.y, g.w & 0xffffffu, fl, vA, vB);
                        if (fl & KF_A) Sm<T>{g.z}.st(vA);
                        Sm<T>{g.z}.at(1).st(vB);
                    }
                }
                __syncthreads();
                kept_matrix(m, t);
                up = true;
                continue;
            }
        }
        // the visit of d is done: another call on it, or the parent's second half
        if (d == m.hi) return;
        ++d;
        made += 1ull << (4 * d);
        up = ((int)(made >> (4 * d)) & 15) >= (d == 1 ? 1 : mu);
        if (!up) {
            zero = false;
            --d;
        }
    }
}

// k_mid with diagonals 4 and 5 kept.  Diagonal 6 has most of the pairs and the fewest
// visits: its coefficients stay as they are, so that two items fit one SM.
template <class T>
__global__ void __launch_bounds__(kKeptThreads, 2)
    k_mid_kept(DevCtx cx, T* su, const T* sbx, const T* sby, const T* ax, const T* ay, const T* op, CycleParams cp)
{
    launch_next();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int2 at[kMidMax + 1];
    const TaskRef t = resolve(cx);
    const SampleInfo& S = cx.samples[t.s];
    const int pi = t.seg->pi, qi = t.seg->qi;
    const MidItem<T> m = mid_item<T>((T*)smem_raw, at, min(pi, kMidD + 1), min(qi, kMidD + 1), kOpD + 1, kOpD + 1 + kKeepMid, kMidD, cp.nu1);
    const KeptTables tb = kept_tables(m, kKeepMid, cp.nu1);
    __syncthreads();  // the table of diagonals
    mid_fill(m, S, ax, ay, op);
    for (int x = 0; x < kKeepMid; ++x) kept_load(m, tb, kOpD + 1 + x, S, ax, ay);
    kept_op(m, tb);
    wait_previous();
    __syncthreads();
    mid_take(m, t.scr, pi, qi, sbx, sby);
    __syncthreads();
    for (int call = 0; call < cp.mu; ++call)
        kept_cycle<T, false>(m, tb, kKeepMid, cp.mu, cp.nu1, cp.nu2, (T)cp.omega, call == 0);
    mid_give(m, t.scr, qi, su);
}

// k_item with the diagonals lo .. lo + keep - 1 kept (stages <= 3: all of them).
template <class T, bool ALL>
__global__ void __launch_bounds__(512, 1)
    k_item_kept(DevCtx cx, int L, double* u64, const double* ax64, const double* ay64, const T* ax, const T* ay, const T* op,
                CycleParams cp, int max_cycles, double eps, int* cycles, double* relres, int* status)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int2 at[kMidMax + 1];
    __shared__ int s_act;
    launch_next();
    const TaskRef t = resolve(cx);
    const SampleInfo& S = cx.samples[t.s];
    const int p = t.seg->pi, q = t.seg->qi, nx = 1 << p, ny = 1 << q, W = nx + 1, tid = threadIdx.x;
    const int64_t off = S.node_off + grid_offset(p, q, S.Q);
    double* u = u64 + off;
    const double* fx = ax64 + off;
    const double* fy = ay64 + off;
    const int lo = L > kOpD ? kOpD + 1 : 0, keep = L > kOpD ? kKeepItem : kKeepLow;
    const MidItem<T> m = mid_item<T>((T*)smem_raw, at, p, q, lo, lo + keep, L, cp.nu1);
    const KeptTables tb = kept_tables(m, keep, cp.nu1);
    __syncthreads();
    mid_fill(m, S, ax, ay, op);
    for (int d = lo; d < lo + keep && d <= L; ++d) kept_load(m, tb, d, S, ax, ay);
    if (lo > 0) kept_op(m, tb);
    wait_previous();
    item_guess(S, p, q, u64, ax64, ay64);
    __syncthreads();
    const MidDiag<T> g = mid_diag(m, L);
    const bool ktop = L < lo + keep;
    const int n = (nx - 1) * (ny - 1);
    auto residual = [&](int c) {
        const double aw = fx[c - 1], ae = fx[c], as = fy[c - W], an = fy[c];
        return 1.0 - ((aw + ae + as + an) * u[c] - (aw * u[c - 1] + ae * u[c + 1]) - (as * u[c - W] + an * u[c + W]));
    };
    const int cell = 2 * tid, ci = cell & (nx - 1), cj = cell >> p;  // the pair of a kept top diagonal
    double first = 0.0;
    for (int step = 0;; ++step) {
        __syncthreads();
        double acc = 0.0;
        if (ktop) {
            if (cell < nx * ny && cj > 0) {
                const double rA = ci > 0 ? residual(cj * W + ci) : 0.0, rB = residual(cj * W + ci + 1);
                acc = rA * rA + rB * rB;
                kept_b(tb, kept_row(tb, L - lo), cj & 1, (T)rA, (T)rB);
            }
        } else {
            for (int k = nx + tid; k < nx * ny; k += blockDim.x) {
                if ((k & (nx - 1)) == 0) continue;
                const double r = residual(k + (k >> p));
                acc += r * r;
                g.b.at(k).st((T)r);
                g.u.at(k).st(T(0));
            }
        }
        const double ss = block_sum(acc);
        if (tid == 0) {
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
        kept_cycle<T, ALL>(m, tb, keep, cp.mu, cp.nu1, cp.nu2, (T)cp.omega, true);
        for (int k = nx + tid; k < nx * ny; k += blockDim.x)
            if (k & (nx - 1)) u[k + (k >> p)] += (double)g.u.at(k).ld();
    }
}

}  // namespace msg
