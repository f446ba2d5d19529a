// Fused all-principal-minors (Schur-complement tree with pivot correction) and
// CDet connected-sum recursion, FP64, one CTA per matrix, persistent over the
// batch.
//
// Paper: Section II (Eq. dets_schur, lemma1, lemma2, Eq. minor, Alg. 1, the
// pivot-correction paragraph and the depth-first remark), Section V.A
// (a[S] = det M_up[S] det M_dn[S], Eq. recursion).
//
// Layout on chip (doubles, for n <= 12 in shared memory, else in per-CTA global
// scratch):  MA[2^n]  minors, then a[]      MC[max(2^n,16)]  tree scratch, then c[]
//            MU[2^n]  (only with a separate A_dn) minors of A_dn
//
// Minors (per matrix):
//   The tree node of mask m over the elements < l holds the Schur complement of
//   A with respect to A[m], restricted to the elements l..n-1 (size (n-l)^2).
//   Its (1,1) entry p gives det A[m | {l}] = det A[m] * p (Eq. minor). The left
//   child (element l excluded) is the same matrix without its first row and
//   column; the right child (l included) is its Schur complement with respect
//   to p. Levels 0..L-1 (L = n-4) are expanded breadth first across the CTA
//   (per level: one thread per node for its minor and pivot reciprocal, then
//   the pivot rows scaled and the child entries formed, one entry per thread
//   step); the 2^L nodes of level L (4x4 each) are finished by one thread each:
//   one more Schur step on the node's first element (a pivot like the others,
//   corrected when tiny) and the 8 minors of each 3x3 child in closed form (56
//   FP64 operations per node against 73 for a 4x4 closed form). Level buffers
//   alternate between MC and the not yet written upper part of MA, so the tree
//   needs no memory beyond MA and MC.
//   Pivot correction: a pivot with |p| <= thr is shifted by C; the node's minor
//   is stored with p + C and the right subtree is built from the shifted
//   matrix. The shift equals adding C to A_ll for every mask of that subtree, so
//   by linearity in row l the exact minors follow from
//       det[m] = det~[m] - C det[m \ {l}]
//   for every mask of its right subtree below the node, applied deepest level
//   first (a shallower correction must see deeper ones already removed). The
//   node's own minor is written as det[m \ {l}] p with the logged unshifted
//   pivot: the subtraction would leave it with an error of eps C |det[m \ {l}]|,
//   large next to the minor itself when p is tiny.
//
// Connected sums: popcount layers k = 2..n in order (every proper subset of a
// k-set lies in an earlier layer). For S with lowest element j and
// S' = S \ {j}, c[S] = a[S] - sum_{U proper subset of S'} c[{j} u U] a[S' \ U].
// A group of g lanes (g = 2^r chosen per layer by a cost model) shares one S:
// lane t fixes the lowest r elements of S' to the bits of t and walks the
// submasks of the rest; the group sum is reduced with warp shuffles.
#include <cuda_runtime.h>
#include <stdint.h>

#include "apm_internal.cuh"

namespace apm {

constexpr int kBlkB = 10;  // low elements per block of the blocked recursion (orders above 12)

__device__ uint16_t g_popmasks[1 << 16];  // masks < 2^16 ordered by (popcount, value)
__device__ int g_popoff[18];              // first index of each popcount class
__constant__ int c_binom[17][17];

struct __align__(16) CdetSmemHdr {
    double log_p[kCorrCap];  // the unshifted pivot (C = sign(p) shift)
    int log_x[kCorrCap];
    int log_l[kCorrCap];
    double red[kCdetThreads / 32];
    unsigned long long red_u[kCdetThreads / 32];
    int ncorr;
    int flags;
    double anorm;
};

// doubles of global scratch per CTA slot: MA, MC, MU
__host__ __device__ inline size_t slot_doubles(int n) {
    const size_t N = size_t(1) << n;
    return 2 * N + (N > 16 ? N : 16);
}

struct CdetKernelParams {
    CdetArgs a;
    unsigned long long gsel;    // 3 bits per popcount layer k: log2 of the lane-group size
    unsigned long long gsel_b;  // the same for blocks of kBlkB elements (orders above 12)
};

struct VarlenParams {
    CdetArgs a;                    // batch, mode, flags, base pointers, gscratch
    const int64_t *a_off;          // element offset of each input matrix
    const int *n_arr;              // order of each matrix
    const int64_t *c_off;          // element offset of each output row (2^n entries)
    const int *order;              // processing order (longest first)
    unsigned *ctr;                 // work counter, zeroed by varlen_order_kernel
    int smem_max_n;
    int n_max;
    int split_to;                  // items of orders smem_max_n + 1 .. split_to with flag 0 are done elsewhere
    const unsigned *width;         // the threads of the CTAs that run, where both widths are launched
    unsigned long long gsel[17];   // lane-group table per order
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Bulk (TMA engine) copy of `bytes` from shared to global memory; issued by one
// thread after a CTA barrier that ordered the shared-memory writes.
__device__ __forceinline__ void bulk_store(double *gdst, const double *ssrc, uint32_t bytes) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst),
                 "r"(smem_u32(ssrc)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------

// max |A_ij| and finiteness of one n x n matrix, on integer bit patterns (the
// magnitude order of finite doubles is the order of their bits without sign).
// over (if not NULL): the scale to use instead of the matrix's own max (a leaf
// of a larger matrix takes that matrix's ||A||max).
__device__ __forceinline__ void matrix_norm(const double *__restrict__ Ag, int n, CdetSmemHdr &h,
                                            const double *over) {
    const int tid = threadIdx.x;
    unsigned long long mx = 0ull;
    int bad = 0;
    for (int i = tid; i < n * n; i += blockDim.x) {
        unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(__ldg(Ag + i)));
        u &= 0x7fffffffffffffffull;
        if (u >= 0x7ff0000000000000ull) bad = 1;
        else if (u > mx) mx = u;
    }
    for (int o = 16; o > 0; o >>= 1) {
        unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = v > mx ? v : mx;
    }
    bad = __any_sync(0xffffffffu, bad);
    if ((tid & 31) == 0) {
        h.red_u[tid >> 5] = mx;
        if (bad) atomicOr(&h.flags, APM_ST_NONFINITE_INPUT);
    }
    __syncthreads();
    if (tid == 0) {
        unsigned long long m = 0ull;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = h.red_u[w] > m ? h.red_u[w] : m;
        double an = over ? *over : __longlong_as_double(static_cast<long long>(m));
        h.anorm = an > 0.0 ? an : 1.0;
    }
    __syncthreads();
}

// Node bookkeeping when a BFS-level matrix's (1,1) entry v is final: store the
// node's minor det[x | {lev}] = det[x] * p (Eq. minor), correct p if it is
// tiny, and replace v by 1/p for the Schur step of the next level.
__device__ __forceinline__ void node_pivot(int x, int lev, double &v, double *MA, double thr,
                                           double shift, CdetSmemHdr &h) {
    double piv = v;
    if (fabs(piv) <= thr) {
        const int slot = atomicAdd(&h.ncorr, 1);
        if (slot < kCorrCap) {
            h.log_x[slot] = x;
            h.log_l[slot] = lev;
            h.log_p[slot] = piv;
        }
        piv += piv >= 0.0 ? shift : -shift;
    }
    MA[x | (1 << lev)] = MA[x] * piv;
    v = 1.0 / piv;
}

// All 15 principal minors of a 4x4 matrix w (row-major) times `pre`, written to
// MA[m | X << L] for X = 1 .. 2^s - 1 (s = min(n,4)); closed-form cofactor and
// Laplace expansions, no division.
__device__ __forceinline__ void bottom4(const double *__restrict__ w, double pre, double *MA, int m,
                                        int L, int s) {
    const double a = w[0], b = w[1], c = w[2], d = w[3];
    const double e = w[4], f = w[5], g = w[6], hh = w[7];
    const double i = w[8], j = w[9], k = w[10], l = w[11];
    const double mm = w[12], nn = w[13], o = w[14], p = w[15];
    // 2x2 principal
    const double d01 = fma(a, f, -b * e);
    const double d02 = fma(a, k, -c * i);
    const double d03 = fma(a, p, -d * mm);
    const double d12 = fma(f, k, -g * j);
    const double d13 = fma(f, p, -hh * nn);
    const double d23 = fma(k, p, -l * o);
    // off-principal 2x2 minors used by the 3x3 and 4x4 expansions
    const double ek_gi = fma(e, k, -g * i);
    const double ej_fi = fma(e, j, -f * i);
    const double ep_hm = fma(e, p, -hh * mm);
    const double en_fm = fma(e, nn, -f * mm);
    const double ip_lm = fma(i, p, -l * mm);
    const double io_km = fma(i, o, -k * mm);
    const double jp_ln = fma(j, p, -l * nn);
    const double jo_kn = fma(j, o, -k * nn);
    // 3x3 principal (cofactor expansion along the first row of each subset)
    const double d012 = fma(a, d12, fma(-b, ek_gi, c * ej_fi));
    const double d013 = fma(a, d13, fma(-b, ep_hm, d * en_fm));
    const double d023 = fma(a, d23, fma(-c, ip_lm, d * io_km));
    const double d123 = fma(f, d23, fma(-g, jp_ln, hh * jo_kn));
    // 4x4 by Laplace expansion along rows 0,1
    const double s02 = fma(a, g, -c * e);
    const double s03 = fma(a, hh, -d * e);
    const double s12 = fma(b, g, -c * f);
    const double s13 = fma(b, hh, -d * f);
    const double s23 = fma(c, hh, -d * g);
    const double c01 = fma(i, nn, -j * mm);
    double d0123 = d01 * d23;
    d0123 = fma(-s02, jp_ln, d0123);
    d0123 = fma(s03, jo_kn, d0123);
    d0123 = fma(s12, ip_lm, d0123);
    d0123 = fma(-s13, io_km, d0123);
    d0123 = fma(s23, c01, d0123);
    MA[m | (1 << L)] = pre * a;
    if (s < 2) return;
    MA[m | (2 << L)] = pre * f;
    MA[m | (3 << L)] = pre * d01;
    if (s < 3) return;
    MA[m | (4 << L)] = pre * k;
    MA[m | (5 << L)] = pre * d02;
    MA[m | (6 << L)] = pre * d12;
    MA[m | (7 << L)] = pre * d012;
    if (s < 4) return;
    MA[m | (8 << L)] = pre * p;
    MA[m | (9 << L)] = pre * d03;
    MA[m | (10 << L)] = pre * d13;
    MA[m | (11 << L)] = pre * d013;
    MA[m | (12 << L)] = pre * d23;
    MA[m | (13 << L)] = pre * d023;
    MA[m | (14 << L)] = pre * d123;
    MA[m | (15 << L)] = pre * d0123;
}

// The 7 principal minors other than the empty one of a 3 x 3 node C (row-major
// stride 4 from c) with node minor d, written to MA[base | X << sh] for
// X = 1..7: row 0 scaled by d first, the 2 x 2 minors directly, the whole by
// expansion along row 0 (no division).
__device__ __forceinline__ void cf3_store(const double *c, int st, double d, double *MA, int base, int sh) {
    const double c00 = c[0], c01 = c[1], c02 = c[2];
    const double c10 = c[st], c11 = c[st + 1], c12 = c[st + 2];
    const double c20 = c[2 * st], c21 = c[2 * st + 1], c22 = c[2 * st + 2];
    const double a0 = d * c00, a1 = d * c01, a2 = d * c02;
    const double m12 = fma(c11, c22, -c12 * c21);
    const double m02 = fma(c10, c22, -c12 * c20);
    const double m01 = fma(c10, c21, -c11 * c20);
    MA[base | (1 << sh)] = a0;
    MA[base | (2 << sh)] = d * c11;
    MA[base | (3 << sh)] = fma(a0, c11, -a1 * c10);
    MA[base | (4 << sh)] = d * c22;
    MA[base | (5 << sh)] = fma(a0, c22, -a2 * c20);
    MA[base | (6 << sh)] = d * m12;
    MA[base | (7 << sh)] = fma(a0, m12, fma(-a1, m02, a2 * m01));
}

// The 15 principal minors of a 4x4 node w (elements L..L+3, node minor MA[m])
// by one Schur step on its first element, a pivot of the tree, and the closed
// forms of the two 3x3 children. A tiny pivot p is shifted by C as on the
// other levels, but its correction is finished here: the node's right subtree
// is the 7 minors of its kept child, all in this thread, and this is the
// deepest level with pivots, so det[m] = det~[m] - C det[m without element L]
// is applied at once (before the logged corrections of the shallower levels),
// and the node's own minor is written with the unshifted pivot. No log entry.
__device__ __forceinline__ void bottom43(const double *__restrict__ w, double *MA, int m, int L, double thr,
                                         double shift, CdetSmemHdr &h) {
    const double p = w[0], d = MA[m];
    const bool corr = fabs(p) <= thr;
    const double C = corr ? (p >= 0.0 ? shift : -shift) : 0.0;
    const double piv = p + C;
    const double v = 1.0 / piv;
    const int mk = m | (1 << L);
    MA[mk] = d * p;
    const double g1 = w[4] * v, g2 = w[8] * v, g3 = w[12] * v;
    double S[9];
    S[0] = fma(-g1, w[1], w[5]);
    S[1] = fma(-g1, w[2], w[6]);
    S[2] = fma(-g1, w[3], w[7]);
    S[3] = fma(-g2, w[1], w[9]);
    S[4] = fma(-g2, w[2], w[10]);
    S[5] = fma(-g2, w[3], w[11]);
    S[6] = fma(-g3, w[1], w[13]);
    S[7] = fma(-g3, w[2], w[14]);
    S[8] = fma(-g3, w[3], w[15]);
    cf3_store(w + 5, 4, d, MA, m, L + 1);      // element L dropped
    cf3_store(S, 3, d * piv, MA, mk, L + 1);   // element L kept (shifted minor when corrected)
    if (corr) {
#pragma unroll
        for (int X = 1; X < 8; ++X) MA[mk | (X << (L + 1))] = fma(-C, MA[m | (X << (L + 1))], MA[mk | (X << (L + 1))]);
        atomicOr(&h.flags, APM_ST_PIVOT_CORRECTED);
    }
}

// All principal minors of the n x n matrix Ag, times root (the minor of the
// empty set), into MA[0 .. 2^n), MC as scratch.
__device__ __forceinline__ void fpm_tree(const double *__restrict__ Ag, int n, double *MA, double *MC, double thr,
                         double shift, CdetSmemHdr &h, double root = 1.0) {
    const int tid = threadIdx.x, T = blockDim.x;
    const int L = n > 4 ? n - 4 : 0;
    double *const bufA = MA + (1 << L);
    // level-l buffer: MC when L-l is even, else the upper part of MA
#define APM_BUF(lv) ((((L) - (lv)) & 1) ? bufA : MC)
    double *W0 = APM_BUF(0);
    if (n >= 4) {
        for (int t = tid; t < n * n; t += T) W0[t] = __ldg(Ag + t);
    } else {
        for (int t = tid; t < 16; t += T) {
            const int r = t >> 2, q = t & 3;
            W0[t] = (r < n && q < n) ? __ldg(Ag + r * n + q) : (r == q ? 1.0 : 0.0);
        }
    }
    if (tid == 0) MA[0] = root;
    __syncthreads();
    for (int l = 0; l < L; ++l) {
        const int s = n - l, s1 = s - 1, ss = s * s, ss1 = s1 * s1, P = 1 << l;
        double *Wl = APM_BUF(l);
        double *Wn = APM_BUF(l + 1);
        // one thread per node: the node's minor and pivot (the division runs
        // with a lane per node, not one lane of a warp busy with Schur entries),
        // then its pivot row scaled by 1/p; row 0 is not part of the left child,
        // so it can be scaled in place (Wl[0] keeps 1/p)
        for (int m = tid; m < P; m += T) {
            double *Wm = Wl + m * ss;
            double v = Wm[0];
            node_pivot(m, l, v, MA, thr, shift, h);
            Wm[0] = v;
        }
        __syncthreads();
        // the pivot rows scaled by 1/p, one entry per thread step
        for (int e = tid; e < P * s1; e += T) {
            const int m = e / s1, q = e - m * s1 + 1;
            Wl[m * ss + q] *= Wl[m * ss];
        }
        __syncthreads();
        const int E = 2 * P * ss1;
        for (int e = tid; e < E; e += T) {
            const int x = e / ss1;
            const int rem = e - x * ss1;
            const int p = rem / s1;
            const int q = rem - p * s1;
            const double *Wp = Wl + (x & (P - 1)) * ss;
            double v = Wp[(p + 1) * s + q + 1];
            if (x >> l)  // right child: Schur complement w.r.t. the pivot
                v = fma(-Wp[(p + 1) * s], Wp[q + 1], v);
            Wn[x * ss1 + rem] = v;
        }
        __syncthreads();
    }
    const double *WL = APM_BUF(L);
#undef APM_BUF
    if (n >= 4) {
        for (int m = tid; m < (1 << L); m += T) bottom43(WL + m * 16, MA, m, L, thr, shift, h);
    } else {
        const int s = n;
        for (int m = tid; m < (1 << L); m += T) bottom4(WL + m * 16, MA[m], MA, m, L, s);
    }
    __syncthreads();
    // back-propagation of pivot corrections, deepest level first (the log is in
    // non-decreasing level order: each level's pivots are logged in its own
    // pivot phase, after a barrier that ends the previous level)
    const int nc = h.ncorr;
    if (nc > kCorrCap) {
        for (int t = tid; t < (1 << n); t += T) MA[t] = __longlong_as_double(0x7ff8000000000000ll);
        if (tid == 0) h.flags |= APM_ST_CORRECTION_OVERFLOW;
        __syncthreads();
        return;
    }
    for (int ci = nc - 1; ci >= 0; --ci) {
        const int x = h.log_x[ci], lv = h.log_l[ci];
        const double pv = h.log_p[ci];
        const double cs = pv >= 0.0 ? shift : -shift;
        const int cnt = 1 << (n - lv - 1);
        for (int t = tid; t < cnt; t += T) {
            const int src = x | (t << (lv + 1));
            const int tgt = src | (1 << lv);
            MA[tgt] = t == 0 ? MA[src] * pv : fma(-cs, MA[src], MA[tgt]);
        }
        __syncthreads();
    }
    if (nc > 0 && tid == 0) h.flags |= APM_ST_PIVOT_CORRECTED;
}

// sum over UH within H, in descending order, of c[j u UL u UH] a[S' less UL and
// UH], four terms a step, their operands loaded a step ahead: with few warps on
// an SM the chain of FMAs is what a set costs, not the loads before each (65536
// rows of order 12 32.6 -> 30.0 ms, one of order 10 22.8 -> 18.7 us, against a
// loop of one term). first (uniform over the warp): the first term is U = S', whose c[S] is still
// zero, and is left out.
__device__ __forceinline__ double cdet_walk(const double *c, const double *a, int j, int Sp, int UL, int H,
                                            bool first = false) {
    const int e0 = H & (-H), H1 = H ^ e0, e1 = H1 & (-H1), H2 = H1 ^ e1;
    double acc = 0.0;
    if (H1 == 0) {  // one or two terms
        if (H && !first) acc = fma(c[j | UL | H], a[Sp ^ (UL | H)], acc);
        return fma(c[j | UL], a[Sp ^ UL], acc);
    }
    int X = H2, cu = j | UL | H2, au = Sp ^ (UL | H2);
    double c3 = c[cu | e1 | e0], a3 = a[au ^ (e1 | e0)], c2 = c[cu | e1], a2 = a[au ^ e1];
    double c1 = c[cu | e0], a1 = a[au ^ e0], c0 = c[cu], a0 = a[au];
    if (first) {
        acc = fma(c0, a0, fma(c1, a1, fma(c2, a2, acc)));
        if (X == 0) return acc;
        X = (X - 1) & H2;
        cu = j | UL | X;
        au = Sp ^ (UL | X);
        c3 = c[cu | e1 | e0], a3 = a[au ^ (e1 | e0)], c2 = c[cu | e1], a2 = a[au ^ e1];
        c1 = c[cu | e0], a1 = a[au ^ e0], c0 = c[cu], a0 = a[au];
    }
    while (X) {
        X = (X - 1) & H2;
        cu = j | UL | X;
        au = Sp ^ (UL | X);
        const double d3 = c[cu | e1 | e0], b3 = a[au ^ (e1 | e0)], d2 = c[cu | e1], b2 = a[au ^ e1];
        const double d1 = c[cu | e0], b1 = a[au ^ e0], d0 = c[cu], b0 = a[au];
        acc = fma(c0, a0, fma(c1, a1, fma(c2, a2, fma(c3, a3, acc))));
        c3 = d3, a3 = b3, c2 = d2, a2 = b2, c1 = d1, a1 = b1, c0 = d0, a0 = b0;
    }
    return fma(c0, a0, fma(c1, a1, fma(c2, a2, fma(c3, a3, acc))));
}

// one group step of a layer: lane's set S, its lanes' shares UL, the rest H
struct CdetSet {
    int S, j, Sp, UL, H, gl;
};
__device__ __forceinline__ CdetSet cdet_set(int S, int r, int lane) {
    CdetSet q;
    q.S = S;
    q.j = S & (-S);
    q.Sp = S ^ q.j;
    q.gl = lane & ((1 << r) - 1);
    q.UL = 0;
    q.H = q.Sp;
    for (int i = 0; i < r; ++i) {
        const int bt = q.H & (-q.H);
        q.H ^= bt;
        if ((q.gl >> i) & 1) q.UL |= bt;
    }
    return q;
}

// Connected sums c[S] = init[S] - sum_{U proper subset of S'} c[{j} u U] a[S' \ U]
// (init = a for the plain recursion) for all masks of n elements.
__device__ __forceinline__ void cdet_layers(const double *init, const double *a, double *c, int n,
                                            unsigned long long gsel) {
    const int tid = threadIdx.x, T = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    for (int t = tid; t < (1 << n); t += T) c[t] = 0.0;
    __syncthreads();
    for (int x = tid; x < n; x += T) c[1 << x] = init[1 << x];
    __syncthreads();
    for (int k = 2; k <= n; ++k) {
        const int cnt = c_binom[n][k];
        const uint16_t *masks = g_popmasks + g_popoff[k];
        const int r = static_cast<int>((gsel >> (3 * k)) & 7ull);
        const int spw = 32 >> r;  // sets per warp step
        for (int base = warp * spw; base < cnt; base += nw * spw) {
            const int G = base + (lane >> r);
            const bool act = G < cnt;
            const CdetSet q = cdet_set(masks[act ? G : cnt - 1], r, lane);
            // c[S] itself (U = S') is still 0 here (c[] of this layer is zeroed
            // before the layer): the term adds exactly 0. Where a lane has the
            // whole set it is left out, else it needs no test
            double acc = cdet_walk(c, a, q.j, q.Sp, q.UL, q.H, r == 0);
            for (int o = (1 << r) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (act && q.gl == 0) c[q.S] = init[q.S] - acc;
        }
        __syncthreads();
    }
}

// acc[S] += sum over all U subset of S' of cb[{j} u U] ab[S' \ U] for every
// nonempty mask S of b elements (j = lowest element of S, S' = S \ {j}): the
// contribution of one off-diagonal block pair of the blocked recursion. All
// masks are independent; lane groups as in cdet_layers.
__device__ __forceinline__ void block_conv(const double *cb, const double *ab, double *acc, int b,
                                           unsigned long long gsel) {
    const int tid = threadIdx.x, T = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    for (int k = 1; k <= b; ++k) {
        const int cnt = c_binom[b][k];
        const uint16_t *masks = g_popmasks + g_popoff[k];
        const int r = static_cast<int>((gsel >> (3 * k)) & 7ull);
        const int spw = 32 >> r;
        for (int base = warp * spw; base < cnt; base += nw * spw) {
            const int G = base + (lane >> r);
            const bool act = G < cnt;
            const CdetSet q = cdet_set(masks[act ? G : cnt - 1], r, lane);
            double sum = cdet_walk(cb, ab, q.j, q.Sp, q.UL, q.H);
            for (int o = (1 << r) >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (act && q.gl == 0) acc[q.S] += sum;
        }
    }
}

// Connected sums for n > kBlkB, blocked over the lowest kBlkB elements:
// S = S_H u S_L. For each S_H (increasing), every proper T_H of S_H contributes
// the block convolution of c[T_H u .] with a[(S_H \ T_H) u .] (with j in the
// low part, T_L = S_L allowed), the S_L = {} entry only when the lowest element
// of S_H lies in T_H; then the diagonal block solves its own recursion with
// init a[S_H u S_L] - acc[S_L] and the pure-low block a[0 u .]. a (global) and
// c (global output row) are read block-wise into shared memory (blk: 6 x 2^kBlkB)
// by asynchronous 16-byte copies (both rows and every block are 16-byte aligned).
__device__ void cdet_blocked(const double *a, double *c, int n, double *blk, unsigned long long gsel_b) {
    const int tid = threadIdx.x, T = blockDim.x;
    const int b = kBlkB, NB = 1 << kBlkB, h = n - b;
    double *cb = blk, *ab = blk + NB, *acc = blk + 2 * NB, *cs = blk + 3 * NB, *as = blk + 4 * NB,
           *a0 = blk + 5 * NB;
    for (int t = tid; t < NB / 2; t += T) cp_async16(a0 + 2 * t, a + 2 * t);
    for (int SH = 0; SH < (1 << h); ++SH) {
        const double *aS = a + (static_cast<size_t>(SH) << b);
        for (int t = tid; t < NB / 2; t += T) cp_async16(as + 2 * t, aS + 2 * t);
        for (int t = tid; t < NB; t += T) acc[t] = 0.0;
        const int jH = SH & (-SH);
        cp_async_wait_all();
        __syncthreads();
        if (SH) {
            for (int TH = (SH - 1) & SH;; TH = (TH - 1) & SH) {
                const double *cT = c + (static_cast<size_t>(TH) << b), *aR = a + (static_cast<size_t>(SH ^ TH) << b);
                for (int t = tid; t < NB / 2; t += T) {
                    cp_async16(cb + 2 * t, cT + 2 * t);
                    cp_async16(ab + 2 * t, aR + 2 * t);
                }
                cp_async_wait_all();
                __syncthreads();
                block_conv(cb, ab, acc, b, gsel_b);
                if (tid == 0 && (TH & jH)) acc[0] = fma(cb[0], ab[0], acc[0]);
                __syncthreads();
                if (TH == 0) break;
            }
        }
        for (int t = tid; t < NB; t += T) as[t] -= acc[t];
        __syncthreads();
        cdet_layers(as, a0, cs, b, gsel_b);
        for (int t = tid; t < NB; t += T)
            c[(static_cast<size_t>(SH) << b) + t] = (t == 0) ? (SH ? as[0] : 0.0) : cs[t];
        __syncthreads();
    }
}

// One matrix: minors (and optionally the connected sums) into the output rows.
// MA/MC/MU are on chip (in_smem) or in the CTA's global scratch slot. given:
// the warp-per-matrix minors kernel has already left this matrix's minors in
// mo (in co when mo is NULL) and its status; only the weights and the
// connected sums remain.
__device__ __forceinline__ void cdet_item(const CdetArgs &p, int n, const double *Au, const double *Ad,
                                          const double *ain, double *mo, double *co, uint32_t *st,
                                          double *MA, double *MC, double *MU, bool in_smem,
                                          unsigned long long gsel, unsigned long long gsel_b, double *blk,
                                          CdetSmemHdr &h, const double *anorm_over, double root,
                                          bool given = false) {
    const int tid = threadIdx.x;
    const int N = 1 << n;
    if (tid == 0) bulk_wait_read();  // the previous item's bulk stores have read their source
    if (tid == 0) {
        h.ncorr = 0;
        h.flags = 0;
    }
    __syncthreads();
    if (p.mode == kModeWeights) {
        for (int t = tid; t < N; t += blockDim.x) MA[t] = t ? __ldg(ain + t) : 1.0;  // a[0] is not read
        __syncthreads();
    } else if (given) {
        // the weights from the given minors (one matrix: det^2, or det)
        const double *src = mo ? mo : co;
        for (int t = tid; t < N; t += blockDim.x) {
            const double m = src[t];
            MA[t] = p.single_det ? m : m * m;
        }
        __syncthreads();
    } else {
        if (p.two_mats) {
            matrix_norm(Ad, n, h, anorm_over);
            fpm_tree(Ad, n, MA, MC, p.piv_thr * h.anorm, p.piv_shift * h.anorm, h);
            for (int t = tid; t < N; t += blockDim.x) MU[t] = MA[t];
            if (tid == 0) h.ncorr = 0;
            __syncthreads();
        }
        matrix_norm(Au, n, h, anorm_over);
        fpm_tree(Au, n, MA, MC, p.piv_thr * h.anorm, p.piv_shift * h.anorm, h, root);
        if (mo) {
            if (in_smem) {
                if (tid == 0) {
                    bulk_store(mo, MA, N * 8u);
                    if (p.two_mats) bulk_store(mo + N, MU, N * 8u);
                    bulk_wait_read();
                }
            } else {
                for (int t = tid; t < N; t += blockDim.x) {
                    mo[t] = MA[t];
                    if (p.two_mats) mo[N + t] = MU[t];
                }
            }
        }
        if (tid == 0 && st) *st = static_cast<uint32_t>(h.flags);
        __syncthreads();
        if (p.mode == kModeMinors) return;
        if (!p.single_det) {
            if (p.two_mats)
                for (int t = tid; t < N; t += blockDim.x) MA[t] *= MU[t];
            else
                for (int t = tid; t < N; t += blockDim.x) MA[t] *= MA[t];
        }
        __syncthreads();
    }
    if (p.weights_only) return;
    if (in_smem) {
        cdet_layers(MA, MA, MC, n, gsel);
        if (tid == 0) bulk_store(co, MC, N * 8u);
    } else if (p.fsc_from_n && n >= p.fsc_from_n) {
        // the weights go to the output row; the fast subset convolution that
        // follows in its own launch turns them into the connected sums in place
        for (int t = tid; t < N; t += blockDim.x) co[t] = MA[t];
    } else {
        cdet_blocked(MA, co, n, blk, gsel_b);
    }
    // the next item's first barrier orders these reads before any overwrite
}

template <bool kSmemArrays>
__global__ void __launch_bounds__(kCdetThreads, 3) fpm_cdet_kernel(const CdetKernelParams P) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    CdetSmemHdr &h = *reinterpret_cast<CdetSmemHdr *>(smem_raw);
    const CdetArgs &p = P.a;
    const int n = p.n;
    const int N = 1 << n;
    const int NC = N > 16 ? N : 16;
    double *const sbase = reinterpret_cast<double *>(smem_raw + ((sizeof(CdetSmemHdr) + 127) & ~size_t(127)));
    double *base;
    if (kSmemArrays)
        base = sbase;
    else
        base = p.gscratch + static_cast<size_t>(blockIdx.x) * slot_doubles(n);
    double *MA = base;
    double *MC = base + N;
    double *MU = MC + NC;
    const int64_t mat = static_cast<int64_t>(n) * n;
    auto item = [&](int64_t b) {
        if (p.weights_only && p.wflag && !p.wflag[b]) return;
        cdet_item(p, n, p.A_up ? p.A_up + b * mat : nullptr, p.A_dn ? p.A_dn + b * mat : nullptr,
                  p.a_in ? p.a_in + b * N : nullptr,
                  p.minors_out ? p.minors_out + b * (p.two_mats ? 2 * N : N) : nullptr,
                  p.c_out ? p.c_out + b * N : nullptr, p.status ? p.status + b : nullptr, MA, MC, MU,
                  kSmemArrays, P.gsel, P.gsel_b, sbase, h, p.anorm_in ? p.anorm_in + (b >> p.anorm_shift) : nullptr,
                  p.pre ? p.pre[b] : 1.0, p.wflag && n >= p.warp_from_n && !p.wflag[b]);
    };
    if (p.redo_list) {
        // only the matrices the warp-per-matrix minors kernel flagged (usually none)
        const int64_t cnt = *p.redo_count < p.batch ? static_cast<int64_t>(*p.redo_count) : p.batch;
        for (int64_t i = blockIdx.x; i < cnt; i += gridDim.x) item(p.redo_list[i]);
    } else {
        for (int64_t b = blockIdx.x; b < p.batch; b += gridDim.x) item(b);
    }
    if (threadIdx.x == 0) bulk_wait_all();
}

// ---------------------------------------------------------------------------
// Orders 11 and 12, few matrices: a cluster of CTAs per matrix
// ---------------------------------------------------------------------------
// One matrix of order 12 is 9400 FP64 warp instructions on one SM, 109 us, with
// the other SMs idle. Here 2^lc CTAs hold a copy of a[] and c[] each. The tree's
// first lc levels are expanded by all of them, below those a CTA has the nodes
// whose masks end in its rank; their minors go to the other CTAs' shared memory.
// A layer's set groups are dealt out to the warps of all CTAs, each finished c[S]
// goes to every copy, and a cluster barrier ends the layer. Every value is formed
// by the operations of fpm_cdet_kernel, in their order: the same bits.
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// all threads of the cluster; orders their shared memory accesses, remote ones too
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_put(double *local, uint32_t rank, double v) {
    uint32_t addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_u32(local)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_or(int *local, uint32_t rank, int v) {
    uint32_t addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_u32(local)), "r"(rank));
    asm volatile("red.shared::cluster.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// the corrections logged at levels lo .. hi - 1, deepest first (as in fpm_tree)
__device__ __forceinline__ void cluster_backprop(double *MA, int n, double shift, const CdetSmemHdr &h, int lo, int hi) {
    for (int ci = h.ncorr - 1; ci >= 0; --ci) {
        const int x = h.log_x[ci], lv = h.log_l[ci];
        if (lv < lo || lv >= hi) continue;
        const double pv = h.log_p[ci], cs = pv >= 0.0 ? shift : -shift;
        for (int t = threadIdx.x; t < (1 << (n - lv - 1)); t += blockDim.x) {
            const int src = x | (t << (lv + 1)), tgt = src | (1 << lv);
            MA[tgt] = t == 0 ? MA[src] * pv : fma(-cs, MA[src], MA[tgt]);
        }
        __syncthreads();
    }
}

// fpm_tree over the cluster (n - 4 > lc, and fewer nodes above the 4 x 4 ones
// than the log holds): every CTA's MA complete and corrected on return.
__device__ __forceinline__ void cluster_tree(const double *__restrict__ Ag, int n, double *MA, double *MC, double thr,
                                             double shift, CdetSmemHdr &h, int rank, int lc) {
    const int tid = threadIdx.x, T = blockDim.x, L = n - 4;
    double *const bufA = MA + (1 << L);
    auto buf = [&](int lv) { return ((L - lv) & 1) ? bufA : MC; };
    double *W0 = buf(0);
    for (int t = tid; t < n * n; t += T) W0[t] = __ldg(Ag + t);
    if (tid == 0) MA[0] = 1.0;
    __syncthreads();
    for (int l = 0; l < L; ++l) {
        const int s = n - l, s1 = s - 1, ss = s * s, ss1 = s1 * s1;
        const bool own = l >= lc;                       // node i is mask (i << lc) | rank, else mask i
        const int P = own ? 1 << (l - lc) : 1 << l;
        double *Wl = buf(l), *Wn = buf(l + 1);
        for (int i = tid; i < P; i += T) {
            double v = Wl[i * ss];
            node_pivot(own ? (i << lc) | rank : i, l, v, MA, thr, shift, h);
            Wl[i * ss] = v;
        }
        __syncthreads();
        for (int e = tid; e < P * s1; e += T) {
            const int m = e / s1, q = e - m * s1 + 1;
            Wl[m * ss + q] *= Wl[m * ss];
        }
        __syncthreads();
        // the children: all of them, or at the last shared level only this CTA's
        const bool one = l + 1 == lc;
        const int E = (one ? 1 : 2 * P) * ss1;
        for (int e = tid; e < E; e += T) {
            const int x = e / ss1, rem = e - x * ss1, p = rem / s1, q = rem - p * s1;
            const int xi = one ? rank : x;
            const double *Wp = Wl + (xi & (P - 1)) * ss;
            double v = Wp[(p + 1) * s + q + 1];
            if (xi >= P) v = fma(-Wp[(p + 1) * s], Wp[q + 1], v);
            Wn[x * ss1 + rem] = v;
        }
        __syncthreads();
    }
    for (int i = tid; i < (1 << (L - lc)); i += T) bottom43(MC + i * 16, MA, (i << lc) | rank, L, thr, shift, h);
    __syncthreads();
    cluster_backprop(MA, n, shift, h, lc, L);
    // this CTA's status bits are complete before the barrier: after it the other
    // CTAs' bits arrive in the first one's word
    if (tid == 0 && h.ncorr > 0) h.flags |= APM_ST_PIVOT_CORRECTED;
    cluster_barrier();  // nobody's MA or MC holds tree nodes any more
    for (int i = tid; i < (1 << (n - lc)); i += T) {
        const int m = (i << lc) | rank;
        const double v = MA[m];
        for (int q = 1; q < (1 << lc); ++q) cluster_put(MA + m, rank ^ q, v);
    }
    if (tid == 0 && rank && h.flags) cluster_or(&h.flags, 0, h.flags);
    cluster_barrier();
    cluster_backprop(MA, n, shift, h, 0, lc);
}

__global__ void __launch_bounds__(kCdetThreads, 2) fpm_cdet_cluster_kernel(const CdetKernelParams P, int lc) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    CdetSmemHdr &h = *reinterpret_cast<CdetSmemHdr *>(smem_raw);
    const CdetArgs &p = P.a;
    const int n = p.n, N = 1 << n, tid = threadIdx.x, T = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    const int rank = static_cast<int>(cluster_rank()), size = 1 << lc;
    const int64_t b = blockIdx.x >> lc;
    double *MA = reinterpret_cast<double *>(smem_raw + ((sizeof(CdetSmemHdr) + 127) & ~size_t(127)));
    double *MC = MA + N, *MU = MC + N;
    const int s0 = rank << (n - lc), s1 = (rank + 1) << (n - lc);  // this CTA's slice of the output rows
    if (tid == 0) {
        h.ncorr = 0;
        h.flags = 0;
    }
    __syncthreads();
    if (p.mode == kModeWeights) {
        for (int t = tid; t < N; t += T) MA[t] = t ? __ldg(p.a_in + b * N + t) : 1.0;  // a[0] is not read
        __syncthreads();
    } else {
        const int64_t mat = static_cast<int64_t>(n) * n;
        if (p.two_mats) {
            matrix_norm(p.A_dn + b * mat, n, h, nullptr);
            cluster_tree(p.A_dn + b * mat, n, MA, MC, p.piv_thr * h.anorm, p.piv_shift * h.anorm, h, rank, lc);
            for (int t = tid; t < N; t += T) MU[t] = MA[t];
            if (tid == 0) h.ncorr = 0;
            __syncthreads();
        }
        matrix_norm(p.A_up + b * mat, n, h, nullptr);
        cluster_tree(p.A_up + b * mat, n, MA, MC, p.piv_thr * h.anorm, p.piv_shift * h.anorm, h, rank, lc);
        if (p.minors_out) {
            double *mo = p.minors_out + b * (p.two_mats ? 2 * N : N);
            for (int t = s0 + tid; t < s1; t += T) {
                mo[t] = MA[t];
                if (p.two_mats) mo[N + t] = MU[t];
            }
        }
        if (tid == 0 && rank == 0 && p.status) p.status[b] = static_cast<uint32_t>(h.flags);
        __syncthreads();
        if (!p.single_det)
            for (int t = tid; t < N; t += T) MA[t] *= p.two_mats ? MU[t] : MA[t];
        __syncthreads();
    }
    for (int t = tid; t < N; t += T) MC[t] = t & (t - 1) ? 0.0 : (t ? MA[t] : 0.0);
    cluster_barrier();  // every copy of c[] is ready for the others' sums
    for (int k = 2; k <= n; ++k) {
        const int cnt = c_binom[n][k];
        const uint16_t *masks = g_popmasks + g_popoff[k];
        const int r = static_cast<int>((P.gsel >> (3 * k)) & 7ull), spw = 32 >> r;
        for (int base = (warp * size + rank) * spw; base < cnt; base += nw * size * spw) {
            const int G = base + (lane >> r);
            const CdetSet q = cdet_set(masks[G < cnt ? G : cnt - 1], r, lane);
            double acc = cdet_walk(MC, MA, q.j, q.Sp, q.UL, q.H, r == 0);
            for (int o = (1 << r) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (G < cnt) {  // all lanes of the group hold the sum
                const double v = MA[q.S] - acc;
                for (int to = q.gl; to < size; to += 1 << r) cluster_put(MC + q.S, to, v);
            }
        }
        cluster_barrier();
    }
    for (int t = s0 + tid; t < s1; t += T) p.c_out[b * N + t] = MC[t];
}

// ---------------------------------------------------------------------------
// Orders 13..15, few matrices: the blocked recursion of cdet_blocked with a
// matrix's blocks on many CTAs
// ---------------------------------------------------------------------------
// One CTA per matrix leaves 24 matrices on 24 of 152 SMs, 1.5 ms each at order
// 14. The blocks S_H of one popcount depend only on those of smaller popcounts,
// so the recursion runs level by level over the whole batch, two launches per
// level: the off-diagonal contributions of every block (its masks S_L dealt out
// to `parts` CTAs, each walking all T_H), left in the block's own place in the
// output row, then the diagonal recursion of every block. Each mask's terms are
// added in the order of cdet_blocked: the results are the same bits.

// The matrices of such a launch: `batch` fixed-order ones (weights a + i astride,
// sums c + (i << n)), or the items order[*first + i], i < *count, of one order of
// an uneven batch (sums c + c_off[item]) less the flagged ones, which its
// persistent kernel takes.
struct SplitArgs {
    const double *a;
    size_t astride;
    double *c;
    const int *order;
    const int64_t *c_off;
    const unsigned *first, *count;
    const unsigned *on;  // 0: the persistent kernel takes all of them (varlen_split_pays)
    const uint8_t *flag;
    double *rows;  // scratch rows of 2^kBlkB doubles, `cap` of them
    int64_t cap, batch;
    int n;
    unsigned long long gsel;
    __device__ __forceinline__ int64_t items() const { return order ? (*on ? static_cast<int64_t>(*count) : 0) : batch; }
    __device__ __forceinline__ int64_t item(int64_t i) const { return order ? order[static_cast<int64_t>(*first) + i] : i; }
    __device__ __forceinline__ bool skip(int64_t i) const { return order && flag[item(i)]; }
    __device__ __forceinline__ double *out(int64_t i) const { return order ? c + c_off[item(i)] : c + (i << n); }
    // whether the terms of level k get a row per T_H
    __device__ __forceinline__ bool in_rows(int64_t blocks, int k) const {
        return rows && blocks * ((1 << k) - 1) <= cap;
    }
};

// Weights of the matrices the warp-per-matrix kernel has not flagged, from
// their minors (rows laid out as the sums) into the rows of P.a, passed as `to`. Where
// an uneven batch's items do not go by blocks (P.on), their flags get bit 1 instead:
// the persistent kernel leaves out those with flag 0.
__global__ void __launch_bounds__(256) cdet_square_kernel(const SplitArgs P, double *to,
                                                          const double *__restrict__ minors, uint8_t *flag,
                                                          int single) {
    if (P.order && !*P.on) {
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < static_cast<int>(*P.count); i += gridDim.x * blockDim.x)
            flag[P.item(i)] |= 2;
        return;
    }
    const int64_t pairs = int64_t(1) << (P.n - 1), all = P.items() << (P.n - 1);
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < all;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t b = i >> (P.n - 1), t = 2 * (i & (pairs - 1));
        if (flag[P.item(b)]) continue;
        double2 m = *reinterpret_cast<const double2 *>(minors + (P.out(b) - P.c) + t);
        if (!single) m = make_double2(m.x * m.x, m.y * m.y);
        *reinterpret_cast<double2 *>(to + b * P.astride + t) = m;
    }
}

// first index of popcount class k in g_popmasks, from the constant bank
__device__ __forceinline__ int cdet_popoff(int k) {
    int o = 0;
    for (int i = 0; i < k; ++i) o += c_binom[16][i];
    return o;
}
// the masks of kBlkB elements by (popcount, value) into pop, one independent
// load per mask
__device__ __forceinline__ void cdet_block_masks(uint16_t *pop) {
    for (int t = threadIdx.x; t < (1 << kBlkB); t += blockDim.x) {
        int rest = t, src = t, k = 0;
        for (; k < kBlkB && rest >= c_binom[kBlkB][k]; ++k) {
            rest -= c_binom[kBlkB][k];
            src += c_binom[16][k] - c_binom[kBlkB][k];
        }
        pop[t] = g_popmasks[src];
    }
}

// Off-diagonal contributions of the blocks with |S_H| = k. Task = (matrix,
// block, part); the warps of a block's parts take the set groups of all layers
// in turn, and the next T_H's operand blocks arrive while the current ones are
// used; the sums go to the block's place in the rows of c. Of few matrices
// (in_rows) a task is one T_H alone instead, (matrix, block, T_H, part), and its
// terms go to a row of their own, which the diagonal launch adds in T_H's order.
// As many parts as give every resident CTA a task.
__global__ void __launch_bounds__(kCdetThreads, 3) cdet_split_conv_kernel(const SplitArgs P, int k) {
    constexpr int b = kBlkB, NB = 1 << kBlkB;
    __shared__ __align__(16) double cb[2][NB], ab[2][NB], acc[NB];
    __shared__ uint16_t pop[NB];
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31;
    const int n = P.n, h = n - b, nblk = c_binom[h][k], pk = cdet_popoff(k);
    const int64_t blocks = P.items() * nblk;
    const bool in_rows = P.in_rows(blocks, k);
    const int nth = in_rows ? (1 << k) - 1 : 1;
    int lparts = 0;
    while (lparts < (in_rows ? 2 : 3) && (blocks * nth << lparts) < (in_rows ? 152 : 6 * 152)) ++lparts;
    const int parts = 1 << lparts, W = (T >> 5) << lparts;
    double *const rows = in_rows ? P.rows : nullptr;
    const unsigned long long gsel = P.gsel;
    if (blockIdx.x >= (blocks * nth) << lparts) return;
    cdet_block_masks(pop);
    for (int64_t task = blockIdx.x; task < (blocks * nth) << lparts; task += gridDim.x) {
        const int part = static_cast<int>(task & (parts - 1));
        const int64_t row = task >> lparts, mb = row / nth, mat = mb / nblk;
        if (P.skip(mat)) continue;
        const int SH = g_popmasks[pk + static_cast<int>(mb - mat * nblk)], jH = SH & (-SH);
        const double *am = P.a + mat * P.astride;
        double *cm = P.out(mat);
        const int wg = part * (T >> 5) + (tid >> 5);
        // f(first lane's set) for the sets of this warp, in every layer
        auto sets = [&](auto &&f) {
            int done = 0, off = 1;
            for (int kk = 1; kk <= b; ++kk) {
                const int cnt = c_binom[b][kk];
                const int r = static_cast<int>((gsel >> (3 * kk)) & 7ull), spw = 32 >> r;
                const int steps = (cnt + spw - 1) >> (5 - r);
                int s0 = wg - done % W;
                if (s0 < 0) s0 += W;
                for (int s = s0; s < steps; s += W) {
                    const int G = s * spw + (lane >> r);
                    f(pop[off + (G < cnt ? G : cnt - 1)], r, G < cnt);
                }
                done += steps;
                off += cnt;
            }
        };
        auto fetch = [&](int TH, int q) {
            const double *cT = cm + (static_cast<size_t>(TH) << b), *aR = am + (static_cast<size_t>(SH ^ TH) << b);
            for (int t = tid; t < NB / 2; t += T) {
                cp_async16(cb[q] + 2 * t, cT + 2 * t);
                cp_async16(ab[q] + 2 * t, aR + 2 * t);
            }
        };
        int T0 = (SH - 1) & SH;
        if (rows)
            for (int i = static_cast<int>(row - mb * nth); i > 0; --i) T0 = (T0 - 1) & SH;
        fetch(T0, 0);
        for (int t = tid; t < NB; t += T) acc[t] = 0.0;
        int q = 0;
        for (int TH = T0;; TH = (TH - 1) & SH, q ^= 1) {
            cp_async_wait_all();
            __syncthreads();
            if (TH && !rows) fetch((TH - 1) & SH, q ^ 1);
            sets([&](int S, int r, bool act) {
                const CdetSet g = cdet_set(S, r, lane);
                double sum = cdet_walk(cb[q], ab[q], g.j, g.Sp, g.UL, g.H);
                for (int o = (1 << r) >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (act && g.gl == 0) acc[S] += sum;
            });
            if (rows) break;
            if (tid == 0 && part == 0 && (TH & jH)) acc[0] = fma(cb[q][0], ab[q][0], acc[0]);
            if (TH == 0) break;
        }
        __syncthreads();
        double *out = rows ? rows + (row << b) : cm + (static_cast<size_t>(SH) << b);
        sets([&](int S, int r, bool act) {
            if (act && (lane & ((1 << r) - 1)) == 0) out[S] = acc[S];
        });
        if (tid == 0 && part == 0) out[0] = acc[0];
        __syncthreads();
    }
}

// The diagonal recursion of the blocks with |S_H| = k, one CTA each.
__global__ void __launch_bounds__(kCdetThreads, 3) cdet_split_diag_kernel(const SplitArgs P, int k) {
    constexpr int b = kBlkB, NB = 1 << kBlkB;
    __shared__ __align__(16) double cs[NB], as[NB], a0[NB];
    __shared__ uint16_t pop[NB];
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = T >> 5;
    const int nblk = c_binom[P.n - b][k], pk = cdet_popoff(k);
    const int64_t blocks = P.items() * nblk;
    const double *const rows = P.in_rows(blocks, k) ? P.rows : nullptr;
    const unsigned long long gsel = P.gsel;
    if (blockIdx.x >= blocks) return;
    cdet_block_masks(pop);
    for (int64_t task = blockIdx.x; task < blocks; task += gridDim.x) {
        const int64_t mat = task / nblk;
        if (P.skip(mat)) continue;
        const int SH = g_popmasks[pk + static_cast<int>(task - mat * nblk)];
        const double *am = P.a + mat * P.astride;
        double *cm = P.out(mat), *out = cm + (static_cast<size_t>(SH) << b);
        for (int t = tid; t < NB; t += T) {
            a0[t] = t ? am[t] : 1.0;
            double sum = 0.0;
            if (SH && !rows) {
                sum = out[t];
            } else if (SH && t) {
                const double *pr = rows + ((task * ((1 << k) - 1)) << b) + t;
                for (int i = 0; i < (1 << k) - 1; i += 8) {  // the loads of eight rows in flight
                    double v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (i + e < (1 << k) - 1) v[e] = pr[static_cast<size_t>(i + e) << b];
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (i + e < (1 << k) - 1) sum += v[e];
                }
            } else if (SH) {
                for (int TH = (SH - 1) & SH; TH; TH = (TH - 1) & SH)
                    if (TH & SH & -SH)
                        sum = fma(cm[static_cast<size_t>(TH) << b], am[static_cast<size_t>(SH ^ TH) << b], sum);
            }
            const double v = am[(static_cast<size_t>(SH) << b) + t] - sum;
            as[t] = v;
            cs[t] = (t & (t - 1)) ? 0.0 : v;  // sets of one element are their own sums
        }
        __syncthreads();
        for (int kk = 2, off = 1 + b; kk <= b; off += c_binom[b][kk], ++kk) {
            const int cnt = c_binom[b][kk];
            const int r = static_cast<int>((gsel >> (3 * kk)) & 7ull), spw = 32 >> r;
            for (int base = warp * spw; base < cnt; base += nw * spw) {
                const int G = base + (lane >> r);
                const CdetSet g = cdet_set(pop[off + (G < cnt ? G : cnt - 1)], r, lane);
                double acc = cdet_walk(cs, a0, g.j, g.Sp, g.UL, g.H, r == 0);
                for (int o = (1 << r) >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (G < cnt && g.gl == 0) cs[g.S] = as[g.S] - acc;
            }
            __syncthreads();
        }
        for (int t = tid; t < NB; t += T) out[t] = (t == 0) ? (SH ? as[0] : 0.0) : cs[t];
        __syncthreads();
    }
}

// Uneven batch: items taken longest-first from `order` through a global
// counter; arrays on chip for n <= smem_max_n, else in the CTA's scratch slot.
// kWidths: launched with both widths of CTAs, of which V.width names the one that
// runs (an instantiation of its own: the test alone, before the first items are
// taken, let them gather on fewer SMs, 1700 of orders 4..9 51 -> 61 us).
template <bool kWidths>
__global__ void __launch_bounds__(kCdetThreads, 3) fpm_cdet_varlen_kernel(const VarlenParams V) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    CdetSmemHdr &h = *reinterpret_cast<CdetSmemHdr *>(smem_raw);
    __shared__ unsigned long long gsel_s[17];
    __shared__ int item_s;
    const CdetArgs &p = V.a;
    if (kWidths && *V.width != blockDim.x) return;
    if (threadIdx.x < 17) gsel_s[threadIdx.x] = V.gsel[threadIdx.x];
    double *const sbase = reinterpret_cast<double *>(smem_raw + ((sizeof(CdetSmemHdr) + 127) & ~size_t(127)));
    double *const gbase = p.gscratch ? p.gscratch + static_cast<size_t>(blockIdx.x) * slot_doubles(V.n_max) : nullptr;
    while (true) {
        __syncthreads();  // gsel_s ready; item_s free for reuse
        if (threadIdx.x == 0) item_s = static_cast<int>(atomicAdd(V.ctr, 1u));
        __syncthreads();
        const int item = item_s;
        if (item >= p.batch) break;
        const int b = V.order[item];
        const int n = V.n_arr[b];
        if (n < 1 || n > V.n_max) {
            if (threadIdx.x == 0 && p.status) p.status[b] = APM_ST_BAD_ORDER;
            continue;
        }
        if (n > V.smem_max_n && n <= V.split_to && !p.wflag[b]) continue;
        const int N = 1 << n;
        const int NC = N > 16 ? N : 16;
        const bool in_smem = n <= V.smem_max_n;
        double *MA = in_smem ? sbase : gbase;
        double *MC = MA + N;
        double *MU = MC + NC;
        const int64_t ao = V.a_off[b], co = V.c_off[b];
        cdet_item(p, n, p.A_up ? p.A_up + ao : nullptr, p.A_dn ? p.A_dn + ao : nullptr,
                  p.a_in ? p.a_in + co : nullptr,
                  p.minors_out ? p.minors_out + (p.two_mats ? 2 * co : co) : nullptr,
                  p.c_out ? p.c_out + co : nullptr, p.status ? p.status + b : nullptr, MA, MC, MU, in_smem,
                  gsel_s[n], gsel_s[kBlkB], sbase, h, nullptr, 1.0,
                  p.wflag && p.warp_from_n && n >= p.warp_from_n && !(p.wflag[b] & 1));
    }
    if (threadIdx.x == 0) bulk_wait_all();
}

// Whether the items of orders 13..to of an uneven batch go by blocks on many CTAs,
// order after order, or all orders together with one CTA per matrix. Each side's
// time from hist, the items per order: of the first a launch's fixed part and a part
// per item; of the second what its work takes on 3 CTAs per SM, but not less than
// the rounds of any one order, whose last takes less with fewer CTAs on an SM (after
// a full one few items do not spread over all SMs).
// 4 % in favour of the second. Measured, us per call (blocks | one CTA per matrix):
//   orders 13, 14: 100 items 656 | 1125, 456 1885 | 2256, 912 3483 | 3064
//   order 13: 100 308 | 404, 300 651 | 559, 500 1038 | 1288, 912 1761 | 1571
//   orders 13..15: 456 3993 | 6584, 1024 7924 | 7162;  4..14: 1024 1181 | 2230
__device__ __noinline__ int varlen_split_pays(const int *hist, int64_t batch, int to) {
    constexpr int kCtas = 456;  // 3 per SM
    // orders 13..16 (16 only where the recursion takes it): us at 1, 2, 3 per SM; us, 10 ns
    constexpr int kWhole[4][3] = {{404, 557, 797}, {1093, 1571, 2288}, {3137, 4585, 6650}, {12450, 14840, 19650}};
    constexpr int kFixed[4] = {150, 250, 400, 300}, kItem[4] = {175, 485, 1430, 4250};
    const int low = (256 * hist[12] + 99 * hist[11] + 43 * hist[10] + 25 * hist[9]) / kCtas;
    const int depth = batch <= 152 ? 0 : batch <= 304 ? 1 : 2;
    int blocks = low, work = 0, least = 0;
    for (int m = 13; m <= to; ++m) {
        const int c = hist[m], i = m - 13;
        if (c == 0) continue;
        blocks += kFixed[i] + kItem[i] * c / 100;
        work += kWhole[i][2] * c;
        const int full = c / kCtas, rest = c - full * kCtas;
        const int last = rest == 0 ? 0 : full && rest <= 152 ? (kWhole[i][0] + kWhole[i][1]) / 2 : kWhole[i][(rest - 1) / 152];
        const int rounds = full * kWhole[i][2] + last;
        least = max(least, max(rounds, kWhole[i][depth]));
    }
    return 104 * blocks <= 100 * max(work / kCtas + low, least);
}

// Threads of the CTAs of an uneven batch of orders up to n_max = 9, 10 or 11, of a
// size where it depends on hist, the items per order: wide (256) while one round of
// wide CTAs holds the items of the largest order (at order 9, narrow CTAs of 64
// threads, those of order 8 count by half), else narrow; wide again for two to three
// rounds of order 11 alone, which narrow CTAs (912 at a time) take in two of their
// own. us per call, narrow | wide:
//   orders 4..9: 600 items 36 | 28, 1024 41 | 37;  8, 9: 700 38 | 45;   order 9: 600 37 | 50, 1200 50 | 73
//   orders 4..10: 912 76 | 48, 1700 79 | 70;       9, 10: 1024 78 | 90; order 10: 600 58 | 88, 1200 126 | 130
//   orders 4..11: 912 175 | 103, 3200 191 | 187;   10, 11: 1200 191 | 200, 2000 299 | 317
//   order 11: 600 133 | 171, 1200 302 | 266, 2300 486 | 519
__device__ unsigned varlen_width(const int *hist, int64_t batch, int n_max) {
    const int c = hist[n_max];
    if (n_max == 9) return c + hist[8] / 2 <= 360 ? kCdetThreads : 64u;
    const bool wide = c <= 456 || (n_max == 11 && c > 912 && c <= 1368 && 10 * c > 9 * batch);
    return wide ? kCdetThreads : 128u;
}

// Longest-first order of an uneven batch: counting sort by decreasing order n
// (one CTA), and reset of the work counter of the consumer kernel; per order m
// the first index and the count of its items (ctr[2 + 2m], ctr[3 + 2m]), and the
// choices of varlen_split_pays for orders 13..split_to (ctr[kCtrSplit]) and, with
// by_width, of varlen_width (ctr[kCtrWidth]).
constexpr int kCtrSplit = 36, kCtrWidth = 37;
template <bool kChoose>
__global__ void __launch_bounds__(1024) varlen_order_kernel(const int *__restrict__ n_arr, int64_t batch,
                                                            int n_max, int *order, unsigned *ctr, int fsc_from_n,
                                                            int split_to, int by_width) {
    __shared__ int hist[18];
    __shared__ int start[18];
    if (threadIdx.x < 18) hist[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t b = threadIdx.x; b < batch; b += blockDim.x) {
        int n = n_arr[b];
        n = (n < 1 || n > n_max) ? 0 : n;  // invalid orders go last (bucket 0)
        atomicAdd(&hist[n], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int pos = 0;
        for (int n = 17; n >= 0; --n) {
            start[n] = pos;
            pos += hist[n];
        }
        ctr[0] = 0u;
        // items of the orders that take the fast subset convolution: the first
        // ones of the longest-first order
        int nf = 0;
        for (int n = fsc_from_n; n <= 16; ++n) nf += hist[n];
        ctr[1] = static_cast<unsigned>(nf);
        if constexpr (kChoose) {
            if (by_width) ctr[kCtrWidth] = varlen_width(hist, batch, n_max);
            if (split_to) ctr[kCtrSplit] = static_cast<unsigned>(varlen_split_pays(hist, batch, split_to));
        }
        for (int n = 0; n <= 16; ++n) {
            ctr[2 + 2 * n] = static_cast<unsigned>(start[n]);
            ctr[3 + 2 * n] = static_cast<unsigned>(hist[n]);
        }
    }
    __syncthreads();
    for (int64_t b = threadIdx.x; b < batch; b += blockDim.x) {
        int n = n_arr[b];
        n = (n < 1 || n > n_max) ? 0 : n;
        const int slot = atomicAdd(&start[n], 1);
        order[slot] = static_cast<int>(b);
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

static inline size_t hdr_bytes() { return (sizeof(CdetSmemHdr) + 127) & ~size_t(127); }

size_t cdet_slot_doubles(int n) { return slot_doubles(n); }

size_t cdet_smem_bytes(int n, bool two_mats, bool smem_arrays) {
    if (!smem_arrays) return hdr_bytes() + 6 * sizeof(double) * (size_t(1) << kBlkB);
    const size_t N = size_t(1) << n;
    return hdr_bytes() + 8 * ((two_mats ? 2 : 1) * N + (N > 16 ? N : 16));
}

int cdet_smem_max_n(bool two_mats) {
    (void)two_mats;
    return 12;  // above: a[] and c[] in global memory, recursion blocked through shared memory
}

void cdet_group_table(int n, int threads, uint8_t *gsel) {
    // Per popcount layer k: choose the group size g = 2^r lanes per set that
    // minimises the FP64 warp-instructions of the layer,
    //   ceil(C(n,k) g / 32) * (2^{k-1-r} + r + 1),
    // breaking near-ties (within 3%) toward larger groups, whose lanes read
    // neighbouring subsets (fewer shared-memory bank conflicts).
    (void)threads;
    for (int k = 0; k <= 16; ++k) gsel[k] = 0;
    double binom[17][17] = {};
    for (int a = 0; a <= 16; ++a) {
        binom[a][0] = 1;
        for (int b = 1; b <= a; ++b) binom[a][b] = binom[a - 1][b - 1] + (b <= a - 1 ? binom[a - 1][b] : 0);
    }
    for (int k = 2; k <= n; ++k) {
        const double cnt = binom[n][k];
        double best = 1e300;
        int rb = 0;
        double cost[6];
        const int rmax = (k - 1) < 5 ? (k - 1) : 5;
        for (int r = 0; r <= rmax; ++r) {
            const double tasks = ceil(cnt * double(1 << r) / 32.0);
            cost[r] = tasks * (double(1 << (k - 1 - r)) + r + 1);
            if (cost[r] < best) { best = cost[r]; rb = r; }
        }
        for (int r = rmax; r > rb; --r)
            if (cost[r] <= best * 1.03) { rb = r; break; }
        gsel[k] = static_cast<uint8_t>(rb);
    }
}

// Lane-group tables installed by apm_cdet_tune_set (0 = use the cost model).
static unsigned long long g_tuned[17] = {};
// Knobs installed by apm_tune_options_set: the order from which the connected
// sums take the fast subset convolution, and the persistent CTAs per SM of the
// uneven batch (0: as many as fit).
static int g_fsc_from_n = kFscFromN;
static int g_varlen_ctas = 0;

int cdet_fsc_from_n() { return g_fsc_from_n; }
int cdet_varlen_ctas_per_sm() { return g_varlen_ctas; }
void cdet_tune_options_set(int fsc_from_n, int cdet_ctas_per_sm) {
    g_fsc_from_n = fsc_from_n;
    g_varlen_ctas = cdet_ctas_per_sm;
}

unsigned long long cdet_gsel_packed(int n) {
    if (n >= 0 && n <= 16 && g_tuned[n]) return g_tuned[n];
    uint8_t gsel[17];
    cdet_group_table(n, kCdetThreads, gsel);
    unsigned long long packed = 0ull;
    for (int k = 0; k <= 16; ++k) packed |= static_cast<unsigned long long>(gsel[k] & 7) << (3 * k);
    return packed;
}

void cdet_tune_set(const unsigned long long *table) {
    for (int n = 0; n <= 16; ++n) g_tuned[n] = table ? table[n] : 0ull;
}

// Threads of a CTA at order n <= 12. A small order's phases have
// too little to do for 256 threads, and every barrier of its tree and its layers
// stops the whole CTA: more, smaller CTAs on an SM (its registers hold 768
// threads of this kernel in any case) fill each other's waits. Wide CTAs are the
// faster only while one round of them holds the batch, or where it fills their last
// round and not the narrow ones'. Measured, us per call (256 | 128 | 64 threads;
// device time):
//   n = 8:  304 matrices 17 | 17 | 18, 1216 46 | 35 | 24, 16384 511 | 284 | 256
//   n = 9:  304 22 | 22 | 28, 777 46 | 35 | 38, 1216 67 | 57 | 44, 16384 740 | 539 | 526
//   n = 10: 456 43 | 46 | 52, 777 82 | 74 | 76, 1216 121 | 111 | 94, 1500 152 | 129 | 115,
//           1672 160 | 140 | 158, 2000 191 | 165 | 170, 16384 1413 | 1240 | 1223
//   n = 11: 456 99 | 104 | 122, 912 194 | 185 | 191, 1368 286 | 301 | 331, 2000 441 | 424 | 477,
//           16384 3315 | 3233 | 3299
//   n = 12: 456 252 | 259 | 290, 16384 8643 | 8808 | 9680
// With a second matrix the arrays of a narrow CTA leave room for 7 (n = 10, 64
// threads) or 4 on an SM (n = 11, 128 threads) instead of 10 and 6:
//   n = 10: 1216 158 | 142 | 164, 1672 209 | 176 | 188, 16384 1849 | 1542 | 1593
//   n = 11: 608 200 | 151 | 176, 912 232 | 271 | 321, 1216 343 | 298 | 337, 1368 344 | 391 | 466,
//           2736 678 | 710 | 802, 3648 899 | 886 | 984
static int cdet_threads(int n, int64_t batch, bool two_mats) {
    if (n > 11) return kCdetThreads;
    const int64_t round = 3 * 152;  // resident CTAs of 256 threads
    if (n <= 8) return batch <= 2 * round ? 128 : 64;
    if (batch <= round) return kCdetThreads;
    if (n == 9) return batch <= 2 * round ? 128 : 64;
    if (n == 10) return !two_mats && batch > 2 * round && batch <= 10 * 152 ? 64 : 128;
    if (two_mats) {  // a round of 4 x 152 narrow CTAs takes 5 / 4 of one of wide ones
        const int64_t wide = (batch + round - 1) / round, narrow = (batch + 4 * 152 - 1) / (4 * 152);
        return 4 * wide <= 5 * narrow ? kCdetThreads : 128;
    }
    return batch > 8 * 152 && batch <= 9 * 152 ? kCdetThreads : 128;
}

int cdet_grid(int n, int64_t batch, bool two_mats, bool smem_arrays, int *err, int threads) {
    const size_t smem = cdet_smem_bytes(n, two_mats, smem_arrays);
    if (threads == 0) threads = cdet_threads(n, batch, two_mats);
    int64_t g = smem_arrays ? resident_ctas(fpm_cdet_kernel<true>, threads, smem,
                                            cdet_smem_bytes(cdet_smem_max_n(true), true, true), err)
                            : resident_ctas(fpm_cdet_kernel<false>, kCdetThreads, smem, smem, err);
    if (*err) return 0;
    if (batch < g) g = batch;
    return static_cast<int>(g < 1 ? 1 : g);
}

// Rows (of 2^kBlkB doubles) that the levels' terms may take, at most 64 MB; does
// not shrink as the batch grows.
constexpr int64_t kSplitMaxRows = 8192;
static int64_t cdet_split_rows(int n, int64_t batch) {
    const int h = n - kBlkB;
    if (h < 3 || h > 6) return 0;
    const int most = h == 3 ? 9 : h == 4 ? 28 : h == 5 ? 75 : 225;  // max over k of C(h, k) (2^k - 1)
    return batch < kSplitMaxRows / most ? batch * most : kSplitMaxRows;
}

size_t cdet_scratch_bytes(int n, int64_t batch, bool two_mats, int *err) {
    const int grid = cdet_grid(n, batch, two_mats, false, err);
    if (*err) return 0;
    return (static_cast<size_t>(grid) * slot_doubles(n) +
            (static_cast<size_t>(cdet_split_rows(n, batch)) << kBlkB)) * sizeof(double);
}

int ensure_tables() {
    static int done_mask = 0;  // bit per device id < 32
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 32 && (done_mask >> dev) & 1) return 0;
    static uint16_t masks[1 << 16];
    int off[18];
    int pos = 0;
    for (int k = 0; k <= 16; ++k) {
        off[k] = pos;
        for (int S = 0; S < (1 << 16); ++S)
            if (__builtin_popcount(static_cast<unsigned>(S)) == k) masks[pos++] = static_cast<uint16_t>(S);
    }
    off[17] = pos;
    int binom[17][17] = {};
    for (int a = 0; a <= 16; ++a) {
        binom[a][0] = 1;
        for (int b = 1; b <= a; ++b) binom[a][b] = binom[a - 1][b - 1] + (b <= a - 1 ? binom[a - 1][b] : 0);
    }
    e = cudaMemcpyToSymbol(g_popmasks, masks, sizeof(masks));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_popoff, off, sizeof(off));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_binom, binom, sizeof(binom));
    if (e != cudaSuccess) return e;
    if (dev < 32) done_mask |= 1 << dev;
    return 0;
}

// The recursion above order 12 with every matrix's blocks on many CTAs, for at
// most `most` matrices.
static int launch_cdet_split(const SplitArgs &P, int64_t most, cudaStream_t s) {
    const int h = P.n - kBlkB;
    const int64_t ctas = 8 * 3 * 152;
    for (int k = 0, nblk = 1; k <= h; nblk = nblk * (h - k) / (k + 1), ++k) {
        const int64_t blocks = most * nblk, tasks = blocks * 8 * (k < 4 ? 1 << k : 16);  // at least as many as there are
        if (k)
            cdet_split_conv_kernel<<<static_cast<int>(tasks < ctas ? tasks : ctas), kCdetThreads, 0, s>>>(P, k);
        cdet_split_diag_kernel<<<static_cast<int>(blocks < ctas ? blocks : ctas), kCdetThreads, 0, s>>>(P, k);
    }
    return static_cast<int>(cudaGetLastError());
}

// Whether a launch (or the last, partial round of one) of this many matrices
// above order 12 goes level by level over many CTAs rather than with one CTA
// per matrix, whose time depends on the most of them that share an SM only: level
// by level up to most of two on every SM, and again up to most of three. After full
// rounds the last one's matrices go to the CTAs that finish first, more of them on
// an SM: level by level up to most of three.
// Measured, us per call (one CTA per matrix | level by level):
//   n = 13: 1 matrix 377 | 130, 24 375 | 168, 152 386 | 360, 230 552 | 541, 260 553 | 582, 304 555 | 651,
//           305 776 | 688, 360 790 | 786, 370 791 | 796, 400 790 | 823
//   n = 14: 1 1069 | 167, 24 1074 | 270, 152 1096 | 915, 270 1577 | 1563, 290 1578 | 1632, 305 2239 | 1788,
//           405 2259 | 2205, 420 2279 | 2385
//   n = 15: 1 3129 | 231, 24 3145 | 554, 152 3199 | 2613, 280 4649 | 4564, 304 4651 | 4818, 305 6578 | 4957,
//           400 6642 | 6279, 430 6649 | 6740
//   n = 16 (from weights): 1 12451 | 299, 300 14857 | 13042, 455 19657 | 19456
//   456 more: n = 13: 152 1285 | 1126, 235 1316 | 1333, 270 1538 | 1386, 340 1539 | 1497, 400 1563 | 1610
//     n = 14: 152 3746 | 3164, 296 4480 | 3900, 400 4489 | 4447, 430 4493 | 4635;  n = 15: 400 13249 | 12926, 430 13273 | 13398
static bool cdet_split_pays(int n, int64_t batch, bool after_rounds) {
    if (n >= 16) return true;
    if (batch <= 2 * 152 && !after_rounds) return batch <= (n == 13 ? 235 : n == 14 ? 275 : 287);
    return batch <= (n == 13 ? 360 : n == 14 ? 405 : 422);
}

// CTAs per matrix (log2) of a launch of so many matrices, 0 for one: at most a CTA
// per SM (two on an SM share its FP64 pipe). us per call, 1, 2, 4 and 8 CTAs:
//   n = 12: 1 matrix 109, 76, 58, 55; 38 109, 76, 76, 117; 100 109, 109
//   n = 11: 1 51, 45, 39, 39; 38 51, 45, 45, 77
//   n = 10: 1 29, 33, 31, 31: a layer's barrier costs what its other lanes save
static int cdet_cluster_log2(int n, int64_t batch) {
    if (n < 11 || n > 12 || batch > 76) return 0;
    return batch > 32 ? 1 : n == 12 && batch <= 10 ? 3 : 2;
}

static int launch_cdet_cluster(const CdetKernelParams &P, int lc, cudaStream_t s) {
    const bool two = P.a.two_mats != 0;
    const size_t smem = cdet_smem_bytes(P.a.n, two, true);
    int err = 0;
    resident_ctas(fpm_cdet_cluster_kernel, kCdetThreads, smem, cdet_smem_bytes(cdet_smem_max_n(true), true, true), &err);
    if (err) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(P.a.batch << lc));
    cfg.blockDim = dim3(kCdetThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1u << lc;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return static_cast<int>(cudaLaunchKernelEx(&cfg, fpm_cdet_cluster_kernel, P, lc));
}

int launch_fpm_cdet(const CdetArgs &a, cudaStream_t s) {
    // before any route, the lane groups' too, which read none of the tables: a
    // later call on this device may be one under capture, where they cannot be
    // uploaded
    int err = ensure_tables();
    if (err) return err;
    if (!a.redo_list && !a.pre && !a.anorm_in) {
        const int lg = cdet_lanes_log2(a.n, a.batch, a.mode);
        if (lg >= 0) return launch_cdet_lanes(a, lg, s);
    }
    CdetKernelParams P;
    P.a = a;
    P.gsel = cdet_gsel_packed(a.n);
    P.gsel_b = cdet_gsel_packed(kBlkB);
    const bool smem_arrays = a.n <= cdet_smem_max_n(a.two_mats != 0);
    // (a redo launch, which usually finds nothing to do, in the fewest CTAs: the
    // 12 per SM of 64 threads cost minors of 4096 matrices of order 9 1.4 of 43 us)
    const int threads = a.redo_list ? kCdetThreads : cdet_threads(a.n, a.batch, a.two_mats != 0);
    const int grid = cdet_grid(a.n, a.batch, a.two_mats != 0, smem_arrays, &err, threads);
    if (err) return err;
    const size_t smem = cdet_smem_bytes(a.n, a.two_mats != 0, smem_arrays);
    const bool fsc = a.mode == kModeCdet && a.n >= g_fsc_from_n;
    P.a.fsc_from_n = fsc ? g_fsc_from_n : 0;
    if (a.wflag && a.warp_from_n && a.n >= a.warp_from_n) {
        // the minors first, one warp per matrix (its stack in the slots' region,
        // which the fused kernel takes over after it)
        err = launch_fpm_warp_route(a.A_up, a.n, a.batch, a.minors_out ? a.minors_out : a.c_out, a.piv_thr,
                                    a.wflag, a.status, a.gscratch, nullptr, nullptr, nullptr, nullptr, nullptr, s);
        if (err) return err;
    }
    // (weights that the sums overwrite in place have to be copied to the slots)
    const bool in_place = a.mode == kModeWeights && a.a_in < a.c_out + (a.batch << a.n) &&
                          a.c_out < a.a_in + (a.batch << a.n);
    if (!smem_arrays && !fsc && a.mode != kModeMinors && !in_place) {
        // full rounds of one CTA per matrix, then the rest
        const int full = cdet_grid(a.n, INT64_MAX, a.two_mats != 0, false, &err);
        if (err) return err;
        const int64_t part = a.batch % full, rest = cdet_split_pays(a.n, part, a.batch > part) ? part : 0, b0 = a.batch - rest;
        if (b0) {
            P.a.batch = b0;
            fpm_cdet_kernel<false><<<grid, kCdetThreads, smem, s>>>(P);
            err = static_cast<int>(cudaGetLastError());
        }
        if (err || !rest) return err;
        const size_t slot = slot_doubles(a.n), row = size_t(1) << a.n, mats = a.two_mats ? 2 : 1;
        SplitArgs Q = {};
        Q.c = a.c_out + b0 * row;
        Q.rows = a.gscratch + grid * slot;
        Q.cap = cdet_split_rows(a.n, rest);
        Q.batch = rest;
        Q.n = a.n;
        Q.gsel = P.gsel_b;
        Q.a = a.mode == kModeWeights ? a.a_in + b0 * row : a.gscratch;
        Q.astride = a.mode == kModeWeights ? row : slot;
        if (a.mode == kModeWeights) return launch_cdet_split(Q, rest, s);
        P.a.batch = rest;
        P.a.weights_only = 1;
        P.a.A_up += b0 * a.n * a.n;
        if (a.A_dn) P.a.A_dn += b0 * a.n * a.n;
        P.a.c_out = Q.c;
        if (a.minors_out) P.a.minors_out += b0 * row * mats;
        if (a.status) P.a.status += b0;
        if (a.wflag) {
            P.a.wflag += b0;
            cdet_square_kernel<<<static_cast<int>(((rest << (a.n - 1)) + 255) / 256), 256, 0, s>>>(
                Q, a.gscratch, a.minors_out ? P.a.minors_out : Q.c, P.a.wflag, a.single_det);
        }
        fpm_cdet_kernel<false><<<static_cast<int>(rest), kCdetThreads, smem, s>>>(P);
        err = static_cast<int>(cudaGetLastError());
        if (err) return err;
        return launch_cdet_split(Q, rest, s);
    }
    if (smem_arrays && a.mode != kModeMinors && !a.redo_list) {
        const int lc = cdet_cluster_log2(a.n, a.batch);
        if (lc) return launch_cdet_cluster(P, lc, s);
    }
    if (smem_arrays)
        fpm_cdet_kernel<true><<<grid, threads, smem, s>>>(P);
    else
        fpm_cdet_kernel<false><<<grid, kCdetThreads, smem, s>>>(P);
    err = static_cast<int>(cudaGetLastError());
    if (err || !fsc) return err;
    // the workspace holds the fused kernel's slots, then the ranked arrays
    return launch_fsc(a.c_out, a.n, a.batch, a.c_out, a.gscratch, s);
}

// ---------------------------------------------------------------------------
// uneven batches
// ---------------------------------------------------------------------------

constexpr int kVarlenSmemMaxN = 12;
// Threads of a CTA, from the largest order present and the batch. Narrow CTAs
// (four or two times as many on an SM) pay once the batch is several rounds of wide
// ones: below that the call waits for the items of the largest order, which a wide
// CTA finishes soonest. Where that depends on how many there are of it (0), both are
// launched and the kernel that sorts the items chooses (varlen_width; the other's
// CTAs return at once). us per call, 64 | 128 | 256 threads (device time):
//   orders 4..8:  304 items 21 | 20 | 20, 600 22 | 22 | 23, 1500 27 | 27 | 44, 16384 159 | 207 | 361
//   orders 4..9:  64 31 | 24 | 23, 456 33 | 29 | 28, 1200 42 | 40 | 41, 16384 218 | 268 | 430
//   orders 4..10: 456 56 | 49 | 46, 2100 82 | 79 | 83, 4096 119 | 110 | 151
//   orders 4..11: 456 129 | 108 | 103, 3648 197 | 191 | 214;  order 11: 4096 935 | 839 | 856
static int varlen_narrow(int n_max) { return n_max <= 9 ? 64 : 128; }
static int varlen_threads(int n_max, int64_t batch) {
    if (n_max > 11) return kCdetThreads;
    if (n_max <= 6) return 64;  // the same at any size below a round, the fastest above
    if (batch <= 456) return kCdetThreads;
    if (n_max <= 8) return 64;
    return batch <= (n_max == 9 ? 1100 : n_max == 10 ? 2000 : 3100) ? 0 : varlen_narrow(n_max);
}
// Largest uneven batch whose items of orders 13..15 may go by blocks on many CTAs: a
// CTA takes 3 to 4 ms for one of order 15 by itself, which is the whole call then
// (300 walkers of orders 4..14 1672 -> 818 us, 100 of 10..16 3872 -> 1764, 1000 of
// 4..16 9174 -> 5078). Whether they do: varlen_split_pays, on the device, where the
// orders are. Their weights, 2^15 doubles each at most, fit the region of the slots
// (456 x 3 times the largest order's).
constexpr int64_t kVarlenSplitMax = 1024;
// The order a CTA's shared arrays hold: the largest present rather than 12 leaves
// room for the narrow CTAs.
static int varlen_smem_n(int n_max) { return n_max < kVarlenSmemMaxN ? n_max : kVarlenSmemMaxN; }

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

static int cdet_varlen_grid(int n_max, int threads, bool two_mats, bool widths, int *err) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        *err = static_cast<int>(e);
        return 0;
    }
    const size_t smem = cdet_smem_bytes(varlen_smem_n(n_max), two_mats, true);
    const size_t allow = cdet_smem_bytes(kVarlenSmemMaxN, true, true);
    int per_sm = (widths ? resident_ctas(fpm_cdet_varlen_kernel<true>, threads, smem, allow, err)
                         : resident_ctas(fpm_cdet_varlen_kernel<false>, threads, smem, allow, err)) / sms;
    if (*err) return 0;
    // the tuned limit counts CTAs of kCdetThreads threads
    const int most = g_varlen_ctas * (kCdetThreads / threads);
    if (most > 0 && most < per_sm) per_sm = most;
    return sms * per_sm;
}

// Orders from which the connected-sum paths of one matrix per item take their
// minors from the warp-per-matrix kernel (0: never).
static int warp_route_from(int n_max, bool two_mats) {
    return !two_mats && n_max >= kWarpRouteFromN ? kWarpRouteFromN : 0;
}

// Workspace of an uneven batch: [counter 256 B][order: batch int32]
// [flags of the warp-kernel minors: batch bytes, with orders >= 13 of one
// matrix per item][varlen_region][rows of terms of the items done by blocks]
// Doubles of the region that holds the CTAs' slots, and before and after them the
// warp kernel's stacks, the weights of the items done by blocks and the ranked arrays.
static int varlen_region(int n_max, int64_t batch, bool two_mats, int grid, size_t *doubles) {
    int err = 0;
    size_t bytes = static_cast<size_t>(grid) * slot_doubles(n_max) * sizeof(double);
    if (n_max >= g_fsc_from_n) {
        const size_t f = fsc_workspace_bytes(n_max, batch, &err);
        if (err) return err;
        if (f > bytes) bytes = f;
    }
    if (warp_route_from(n_max, two_mats)) {
        const size_t st = fpm_warp_route_stack_bytes(n_max, batch, &err);
        if (err) return err;
        if (st > bytes) bytes = st;
    }
    *doubles = align256(bytes) / sizeof(double);
    return 0;
}

// Rows of terms of the items done by blocks: as many as all items would take, were
// they of the largest such order (a batch too large for blocks: the most a smaller
// one takes).
static int64_t varlen_split_rows(int n_max, int64_t batch) {
    const int to = n_max < g_fsc_from_n ? n_max : g_fsc_from_n - 1;
    return batch <= kVarlenSplitMax ? cdet_split_rows(to, batch) : kSplitMaxRows;
}

size_t cdet_varlen_workspace(int n_max, int64_t batch, bool two_mats, int *err) {
    *err = 0;
    size_t bytes = 256 + align256(static_cast<size_t>(batch) * sizeof(int));
    if (n_max <= kVarlenSmemMaxN) return bytes;
    const int grid = cdet_varlen_grid(n_max, kCdetThreads, two_mats, false, err);  // of orders above 12
    if (*err) return 0;
    size_t region = 0;
    *err = varlen_region(n_max, batch, two_mats, grid, &region);
    if (*err) return 0;
    bytes += region * sizeof(double);
    if (warp_route_from(n_max, two_mats))
        bytes += align256(static_cast<size_t>(batch)) +
                 static_cast<size_t>(varlen_split_rows(n_max, batch) << kBlkB) * sizeof(double);
    return bytes;
}

int launch_order(const int *n_arr, int64_t batch, int n_max, int *order, unsigned *ctr, cudaStream_t s,
                 int fsc_from_n, int split_to, int by_width) {
    const auto kern = split_to || by_width ? varlen_order_kernel<true> : varlen_order_kernel<false>;
    kern<<<1, 1024, 0, s>>>(n_arr, batch, n_max, order, ctr, fsc_from_n, split_to, by_width);
    return static_cast<int>(cudaGetLastError());
}

int launch_cdet_varlen(const CdetArgs &a, const int64_t *a_off, const int *n_arr, const int64_t *c_off,
                       int n_max, void *workspace, cudaStream_t s) {
    int err = ensure_tables();
    if (err) return err;
    const bool two = a.two_mats != 0;
    const int threads = varlen_threads(n_max, a.batch);  // 0: both widths, varlen_width chooses
    const int grid = cdet_varlen_grid(n_max, threads ? threads : kCdetThreads, two, threads == 0, &err);
    if (err) return err;
    const int narrow = threads ? 0 : cdet_varlen_grid(n_max, varlen_narrow(n_max), two, true, &err);
    if (err) return err;
    unsigned char *ws = static_cast<unsigned char *>(workspace);
    unsigned *ctr = reinterpret_cast<unsigned *>(ws);
    int *order = reinterpret_cast<int *>(ws + 256);
    size_t off = 256 + align256(static_cast<size_t>(a.batch) * sizeof(int));
    const int wfrom = n_max > kVarlenSmemMaxN && a.mode == kModeCdet ? warp_route_from(n_max, two) : 0;
    uint8_t *wflag = wfrom ? ws + off : nullptr;
    if (wfrom) off += align256(static_cast<size_t>(a.batch));
    double *slots = reinterpret_cast<double *>(ws + off);
    const int fsc_from = g_fsc_from_n;
    // few items: those of orders 13..15 by blocks on many CTAs, if that pays
    int split_to = 0;
    size_t region = 0;  // of the slots, in doubles; the rows of terms come after it
    if (wfrom) {
        err = varlen_region(n_max, a.batch, two, grid, &region);
        if (err) return err;
        const int to = n_max < fsc_from ? n_max : fsc_from - 1;
        if (a.batch <= kVarlenSplitMax && static_cast<size_t>(a.batch) << to <= region) split_to = to;
    }
    err = launch_order(n_arr, a.batch, n_max, order, ctr, s, fsc_from, split_to, narrow > 0);
    if (err) return err;
    // the minors of the items of orders >= wfrom, one launch per order from its
    // first index and count in the sorted list, the flags zeroed before them
    // (a small batch's matrices are several warps each, which only set them)
    if (wfrom) {
        err = static_cast<int>(cudaMemsetAsync(wflag, 0, static_cast<size_t>(a.batch), s));
        if (err) return err;
    }
    for (int m = n_max; wfrom && m >= wfrom && !err; --m)
        err = launch_fpm_warp_route(a.A_up, m, a.batch, a.minors_out ? a.minors_out : a.c_out, a.piv_thr, wflag,
                                    a.status, slots, order, a_off, c_off, ctr + 2 + 2 * m, ctr + 3 + 2 * m, s);
    if (err) return err;
    // the split orders one after the other, their weights in the slots' region (the
    // persistent kernel, which takes it over after them, finds only the flagged ones
    // of these orders)
    if (split_to) {
        SplitArgs Q = {};
        Q.a = slots;
        Q.c = a.c_out;
        Q.order = order;
        Q.c_off = c_off;
        Q.on = ctr + kCtrSplit;
        Q.flag = wflag;
        Q.rows = slots + region;
        Q.cap = varlen_split_rows(n_max, a.batch);
        Q.batch = a.batch;
        Q.gsel = cdet_gsel_packed(kBlkB);
        for (int m = split_to; m > kVarlenSmemMaxN; --m) {
            Q.n = m;
            Q.astride = size_t(1) << m;
            Q.first = ctr + 2 + 2 * m;
            Q.count = ctr + 3 + 2 * m;
            cdet_square_kernel<<<8 * 152, 256, 0, s>>>(Q, slots, a.minors_out ? a.minors_out : a.c_out, wflag,
                                                       a.single_det);
            err = launch_cdet_split(Q, a.batch, s);
            if (err) return err;
        }
    }
    VarlenParams V;
    V.a = a;
    V.split_to = split_to;
    V.width = narrow ? ctr + kCtrWidth : nullptr;
    V.a.wflag = wflag;
    V.a.warp_from_n = wfrom;
    V.a.gscratch = n_max > kVarlenSmemMaxN ? slots : nullptr;
    V.a_off = a_off;
    V.n_arr = n_arr;
    V.c_off = c_off;
    V.order = order;
    V.ctr = ctr;
    V.smem_max_n = kVarlenSmemMaxN;
    V.n_max = n_max;
    for (int n = 0; n <= 16; ++n) V.gsel[n] = cdet_gsel_packed(n);
    const bool fsc = a.mode == kModeCdet && n_max >= fsc_from;
    V.a.fsc_from_n = fsc ? fsc_from : 0;
    const size_t smem = cdet_smem_bytes(varlen_smem_n(n_max), two, true);
    const auto ctas = [&](int most) { return static_cast<int>(a.batch < most ? a.batch : most); };
    if (narrow) {
        fpm_cdet_varlen_kernel<true><<<ctas(grid), kCdetThreads, smem, s>>>(V);
        fpm_cdet_varlen_kernel<true><<<ctas(narrow), varlen_narrow(n_max), smem, s>>>(V);
    } else {
        fpm_cdet_varlen_kernel<false><<<ctas(grid), threads, smem, s>>>(V);
    }
    err = static_cast<int>(cudaGetLastError());
    if (err || !fsc) return err;
    // the items of the orders >= fsc_from (the longest-first prefix), one launch
    // per order from its first index and count as the order kernel left them,
    // in place on their output rows
    for (int m = n_max; m >= fsc_from && !err; --m)
        err = launch_fsc_items(a.c_out, c_off, order, ctr + 2 + 2 * m, ctr + 3 + 2 * m, a.batch, m, slots, s);
    return err;
}

}  // namespace apm
