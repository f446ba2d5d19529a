// Minors and connected sums of small orders (n <= 8), a few lanes per matrix.
//
// Paper: Section II (Eq. minor, Alg. 1) and Section V.A (Eq. recursion), as in
// the one-CTA-per-matrix kernel; the same operations on the same operands in
// the same order, so every output is bit-identical to that kernel's, whatever
// the batch size decides.
//
// What bounds it: the FP64 pipe, which is charged a whole warp instruction (16
// SM cycles) whatever the number of active lanes. At these orders a CTA of 256
// threads on one matrix leaves most lanes idle and waits at a barrier per tree
// level and per popcount layer. Here a warp holds 32 / LPM matrices, LPM lanes
// each, and nothing wider than a warp is ever synchronised:
//   * tree: a lane carries its node's Schur complement in registers. The first
//     log2(LPM) levels are one path per lane (bit l of the lane's index within
//     the matrix keeps or drops element l), the subtree below it is the lane's
//     own, unrolled, down to the 4 x 4 closed step;
//   * recursion: a lane takes whole sets S and walks all their submask groups
//     itself; only where a layer has fewer sets than the matrix has lanes do
//     lanes share a set (their partial sums meet by shuffles).
// a[] and c[] are in shared memory, entry (mask, matrix) at mask * STR +
// matrix, STR odd, so that both the lanes' accesses (matrices side by side) and
// the transposed reads that write the rows out are free of bank conflicts.
#include <cuda_runtime.h>
#include <stdint.h>

#include "apm_internal.cuh"

namespace apm {

constexpr int kLanesMaxN = 8;

__host__ __device__ constexpr int cl_binom(int n, int k) {
    int r = 1;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return r;
}

struct LanesParams {
    CdetArgs a;
    unsigned long long gsel;  // 3 bits per popcount layer k: log2 of the partial sums a set is split into
};

template <int N, int LG>
struct Lanes {
    static constexpr int LPM = 1 << LG, MPW = 32 >> LG, STR = MPW > 1 ? MPW + 1 : 1;
    static constexpr int L = N > 4 ? N - 4 : 0;  // tree levels above the 4 x 4 nodes
    static constexpr int TOP = LG < L ? LG : L;  // levels walked as one path per lane
    static constexpr int NODES = (1 << L) - 1;   // their nodes, each with a pivot that may be corrected
    static constexpr int SLOTS = NODES > 0 ? NODES : 1;

    struct Smem {
        double log_p[SLOTS][MPW];  // the unshifted pivot of node (level, x) at slot 2^level - 1 + x
        unsigned corr[MPW];        // the corrected nodes of each matrix
        uint8_t pop[1 << N];       // masks by (popcount, value)
    };

    // lane's state while its matrix's tree is walked
    struct Ctx {
        Smem &s;
        double *D;  // minors, entry (mask, m) at mask * STR + m
        int m, q;
        double thr, shift;
        unsigned fl;
        __device__ __forceinline__ void put(int mask, double v, bool mine) {
            if (mine) D[mask * STR + m] = v;
        }
    };

    // the 7 principal minors other than the empty one of the 3 x 3 block of M
    // at (o, o), node minor d: row 0 scaled by d, the whole by expansion along row 0
    template <int K>
    static __device__ __forceinline__ void cf3(const double (&M)[K][K], int o, double d, double (&v)[8]) {
        const double c00 = M[o][o], c01 = M[o][o + 1], c02 = M[o][o + 2];
        const double c10 = M[o + 1][o], c11 = M[o + 1][o + 1], c12 = M[o + 1][o + 2];
        const double c20 = M[o + 2][o], c21 = M[o + 2][o + 1], c22 = M[o + 2][o + 2];
        const double a0 = d * c00, a1 = d * c01, a2 = d * c02;
        const double m12 = fma(c11, c22, -c12 * c21);
        const double m02 = fma(c10, c22, -c12 * c20);
        const double m01 = fma(c10, c21, -c11 * c20);
        v[1] = a0;
        v[2] = d * c11;
        v[3] = fma(a0, c11, -a1 * c10);
        v[4] = d * c22;
        v[5] = fma(a0, c22, -a2 * c20);
        v[6] = d * m12;
        v[7] = fma(a0, m12, fma(-a1, m02, a2 * m01));
    }

    // a 4 x 4 node of mask x over elements L..L+3 with minor d: one Schur step
    // on its first element (its own correction finished at once) and the
    // closed forms of the two 3 x 3 children
    static __device__ __forceinline__ void node4(const double (&w)[4][4], double d, int x, Ctx &t, bool mine) {
        const double p = w[0][0];
        const bool corr = fabs(p) <= t.thr;
        const double C = corr ? (p >= 0.0 ? t.shift : -t.shift) : 0.0;
        const double piv = p + C;
        const double v = 1.0 / piv;
        const int xk = x | (1 << L);
        t.put(xk, d * p, mine);
        const double g1 = w[1][0] * v, g2 = w[2][0] * v, g3 = w[3][0] * v;
        double S[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            S[0][c] = fma(-g1, w[0][c + 1], w[1][c + 1]);
            S[1][c] = fma(-g2, w[0][c + 1], w[2][c + 1]);
            S[2][c] = fma(-g3, w[0][c + 1], w[3][c + 1]);
        }
        double lo[8], hi[8];
        cf3(w, 1, d, lo);
        cf3(S, 0, d * piv, hi);
        if (corr) {
#pragma unroll
            for (int X = 1; X < 8; ++X) hi[X] = fma(-C, lo[X], hi[X]);
            t.fl |= APM_ST_PIVOT_CORRECTED;
        }
#pragma unroll
        for (int X = 1; X < 8; ++X) {
            t.put(x | (X << (L + 1)), lo[X], mine);
            t.put(xk | (X << (L + 1)), hi[X], mine);
        }
    }

    // node of size K at level N - K with mask x and minor d
    template <int K>
    static __device__ __forceinline__ void node(const double (&M)[K][K], double d, int x, Ctx &t, bool mine) {
        if constexpr (K == 4) {
            node4(M, d, x, t, mine);
        } else {
            constexpr int lev = N - K;
            double piv = M[0][0];
            // a node of the lanes' paths is shared: the first of its lanes writes
            const bool w = mine && (lev >= TOP || (t.q >> lev) == 0);
            if (fabs(piv) <= t.thr) {
                if (w) {
                    const int slot = (1 << lev) - 1 + x;
                    t.s.log_p[slot][t.m] = piv;
                    atomicOr(&t.s.corr[t.m], 1u << slot);
                }
                piv += piv >= 0.0 ? t.shift : -t.shift;
            }
            const double dk = d * piv;
            t.put(x | (1 << lev), dk, w);
            const double iv = 1.0 / piv;
            double S[K - 1][K - 1];
            if constexpr (lev < TOP) {
                const bool keep = (t.q >> lev) & 1;
#pragma unroll
                for (int c = 0; c < K - 1; ++c) {
                    const double f = M[0][c + 1] * iv;
#pragma unroll
                    for (int r = 0; r < K - 1; ++r)
                        S[r][c] = keep ? fma(-M[r + 1][0], f, M[r + 1][c + 1]) : M[r + 1][c + 1];
                }
                node<K - 1>(S, keep ? dk : d, keep ? x | (1 << lev) : x, t, mine);
            } else {
#pragma unroll
                for (int c = 0; c < K - 1; ++c) {
                    const double f = M[0][c + 1] * iv;
#pragma unroll
                    for (int r = 0; r < K - 1; ++r) S[r][c] = fma(-M[r + 1][0], f, M[r + 1][c + 1]);
                }
                node<K - 1>(S, dk, x | (1 << lev), t, mine);
#pragma unroll
                for (int r = 0; r < K - 1; ++r)
#pragma unroll
                    for (int c = 0; c < K - 1; ++c) S[r][c] = M[r + 1][c + 1];
                node<K - 1>(S, d, x, t, mine);
            }
        }
    }

    // orders 1..3: the closed forms of the matrix bordered by a unit block
    static __device__ __forceinline__ void small(const double (&w)[4][4], Ctx &t, bool mine) {
        const double a = w[0][0], b = w[0][1], c = w[0][2], e = w[1][0], f = w[1][1], g = w[1][2];
        const double i = w[2][0], j = w[2][1], k = w[2][2];
        t.put(1, a, mine);
        if constexpr (N >= 2) {
            t.put(2, f, mine);
            t.put(3, fma(a, f, -b * e), mine);
        }
        if constexpr (N >= 3) {
            const double d12 = fma(f, k, -g * j), ek_gi = fma(e, k, -g * i), ej_fi = fma(e, j, -f * i);
            t.put(4, k, mine);
            t.put(5, fma(a, k, -c * i), mine);
            t.put(6, d12, mine);
            t.put(7, fma(a, d12, fma(-b, ek_gi, c * ej_fi)), mine);
        }
    }

    // all minors of matrix A (this lane's share) into D
    static __device__ __forceinline__ void tree(const double *__restrict__ A, double *D, const CdetArgs &p, Smem &s,
                                                int m, int q, unsigned &fl) {
        constexpr int K = N < 4 ? 4 : N;
        double M[K][K];
        unsigned long long mx = 0ull;
        if (q == 0) s.corr[m] = 0u;
#pragma unroll
        for (int r = 0; r < K; ++r)
#pragma unroll
            for (int c = 0; c < K; ++c) {
                if (r < N && c < N) {
                    const double x = __ldg(A + r * N + c);
                    M[r][c] = x;
                    const unsigned long long u =
                        static_cast<unsigned long long>(__double_as_longlong(x)) & 0x7fffffffffffffffull;
                    if (u >= 0x7ff0000000000000ull) fl |= APM_ST_NONFINITE_INPUT;
                    else if (u > mx) mx = u;
                } else {
                    M[r][c] = r == c ? 1.0 : 0.0;
                }
            }
        __syncwarp();
        double an = __longlong_as_double(static_cast<long long>(mx));
        an = an > 0.0 ? an : 1.0;
        Ctx t = {s, D, m, q, p.piv_thr * an, p.piv_shift * an, 0u};
        t.put(0, 1.0, q == 0);
        if constexpr (N < 4) small(M, t, q == 0);
        else node<K>(M, 1.0, 0, t, (q >> TOP) == 0);
        fl |= t.fl;
        __syncwarp();
        if constexpr (NODES > 0) {
            // back-propagation, deepest level first; nodes of one level touch disjoint masks
            const unsigned corr = s.corr[m];
            if (__any_sync(0xffffffffu, corr != 0u)) {
                for (int slot = NODES - 1; slot >= 0; --slot) {
                    if ((corr >> slot) & 1u) {
                        const int lv = 31 - __clz(slot + 1), x = slot + 1 - (1 << lv);
                        const double pv = s.log_p[slot][m], cs = pv >= 0.0 ? t.shift : -t.shift;
                        for (int e = q; e < (1 << (N - lv - 1)); e += LPM) {
                            const int src = x | (e << (lv + 1)), tgt = src | (1 << lv);
                            const double vs = D[src * STR + m];
                            D[tgt * STR + m] = e == 0 ? vs * pv : fma(-cs, vs, D[tgt * STR + m]);
                        }
                    }
                    __syncwarp();
                }
                if (corr) fl |= APM_ST_PIVOT_CORRECTED;
            }
        }
    }

    // sum over the submasks UH of H, in descending order, of c[j u UL u UH]
    // a[S' less them]; the term that is the whole of S' (c[S] itself) is left out
    static __device__ __forceinline__ double leaf(const double *c, const double *a, int j, int Sp, int UL, int H) {
        double acc = 0.0;
        int UH = H;
        if ((UL | H) == Sp) {
            if (H == 0) return 0.0;
            UH = (H - 1) & H;
        }
        while (true) {
            const int U = UL | UH;
            acc = fma(c[(j | U) * STR], a[(Sp ^ U) * STR], acc);
            if (UH == 0) break;
            UH = (UH - 1) & H;
        }
        return acc;
    }

    // Eq. recursion. A set's sum is split into 2^r partial sums by its r lowest
    // elements of S' (r per layer, gsel) which are added pairwise, the highest
    // of the r first: 2^sh of them on lanes of their own, the rest in the lane.
    static __device__ __forceinline__ void layers(const double *a, double *c, unsigned long long gsel, const Smem &s,
                                                  int m, int q) {
        const double *am = a + m;
        double *cm = c + m;
        if (q == 0) {
            cm[0] = 0.0;
#pragma unroll
            for (int x = 0; x < N; ++x) cm[(1 << x) * STR] = am[(1 << x) * STR];
        }
        __syncwarp();
        int off = 1 + N;
        for (int k = 2, cnt = N * (N - 1) / 2; k <= N; off += cnt, cnt = cnt * (N - k) / (k + 1), ++k) {
            const int r = static_cast<int>((gsel >> (3 * k)) & 7ull);
            int sh = 0;
            while (sh < LG && sh < r && (cnt << (sh + 1)) <= LPM) ++sh;
            const int R = r - sh, spw = LPM >> sh, gl = q & ((1 << sh) - 1);
            for (int g0 = 0; g0 < cnt; g0 += spw) {
                const int G = g0 + (q >> sh);
                const bool act = G < cnt;
                const int S = s.pop[off + (act ? G : cnt - 1)];
                const int j = S & -S, Sp = S ^ j;
                int UL = 0, rest = Sp, eb[5];
                for (int i = 0; i < sh; ++i) {
                    const int bt = rest & -rest;
                    rest ^= bt;
                    if ((gl >> i) & 1) UL |= bt;
                }
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    eb[i] = 0;
                    if (i < R) {
                        eb[i] = rest & -rest;
                        rest ^= eb[i];
                    }
                }
                double v = 0.0, st0 = 0.0, st1 = 0.0, st2 = 0.0, st3 = 0.0, st4 = 0.0;
                for (int t = 0; t < (1 << R); ++t) {
                    int U = UL;
#pragma unroll
                    for (int i = 0; i < 5; ++i)
                        if (i < R && ((t >> (R - 1 - i)) & 1)) U |= eb[i];
                    v = leaf(cm, am, j, Sp, U, rest);
                    // add equal-sized runs pairwise (a binary counter of runs)
                    if (!(t & 1)) { st0 = v; continue; }
                    v = st0 + v;
                    if (!(t & 2)) { st1 = v; continue; }
                    v = st1 + v;
                    if (!(t & 4)) { st2 = v; continue; }
                    v = st2 + v;
                    if (!(t & 8)) { st3 = v; continue; }
                    v = st3 + v;
                    if (!(t & 16)) { st4 = v; continue; }
                    v = st4 + v;
                }
                for (int o = (1 << sh) >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o * MPW);
                if (act && gl == 0) cm[S * STR] = am[S * STR] - v;
            }
            __syncwarp();
        }
    }

    // rows base .. base+rows-1 (2^N doubles each, row stride rs) from D
    static __device__ __forceinline__ void store(double *out, int64_t base, int rows, int64_t rs, const double *D,
                                                 int lane) {
        for (int i = lane; i < (rows << (N - 1)); i += 32) {
            const int mm = i >> (N - 1), t = 2 * (i & ((1 << (N - 1)) - 1));
            *reinterpret_cast<double2 *>(out + (base + mm) * rs + t) =
                make_double2(D[t * STR + mm], D[(t + 1) * STR + mm]);
        }
    }
};

template <int N, int LG>
__global__ void __launch_bounds__(32) cdet_lanes_kernel(const LanesParams P) {
    using T = Lanes<N, LG>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename T::Smem &s = *reinterpret_cast<typename T::Smem *>(smem_raw);
    double *const MA = reinterpret_cast<double *>(smem_raw + ((sizeof(typename T::Smem) + 15) & ~size_t(15)));
    double *const MC = MA + (T::STR << N);
    double *const MU = MC + (T::STR << N);  // with a second matrix only
    const CdetArgs &p = P.a;
    const int lane = threadIdx.x, m = lane & (T::MPW - 1), q = lane / T::MPW;
    for (int t = lane; t < (1 << N); t += 32) {
        // position of t: the smaller classes, then its rank within its own
        int pos = 0, i = 0;
        const int pc = __popc(t);
        for (int k = 0; k < pc; ++k) pos += cl_binom(N, k);
        for (int r = t; r; r &= r - 1) {
            ++i;
            const int e = __ffs(r) - 1;
            if (i <= e) pos += cl_binom(e, i);
        }
        s.pop[pos] = static_cast<uint8_t>(t);
    }
    __syncwarp();
    const int64_t NN = int64_t(1) << N;
    for (int64_t base = static_cast<int64_t>(blockIdx.x) * T::MPW; base < p.batch;
         base += static_cast<int64_t>(gridDim.x) * T::MPW) {
        const int rows = p.batch - base < T::MPW ? static_cast<int>(p.batch - base) : T::MPW;
        const int64_t b = base + (m < rows ? m : rows - 1);
        if (p.mode == kModeWeights) {
            for (int i = lane; i < (T::MPW << N); i += 32) {
                const int mm = i >> N, t = i & ((1 << N) - 1);
                MA[t * T::STR + mm] = mm < rows ? __ldg(p.a_in + (base + mm) * NN + t) : 0.0;
            }
        } else {
            unsigned fl = 0u;
            if (p.two_mats) T::tree(p.A_dn + b * N * N, MU, p, s, m, q, fl);
            T::tree(p.A_up + b * N * N, MA, p, s, m, q, fl);
#pragma unroll
            for (int o = T::MPW; o < 32; o <<= 1) fl |= __shfl_xor_sync(0xffffffffu, fl, o);
            if (p.status && q == 0 && m < rows) p.status[b] = fl;
            if (p.minors_out) {
                T::store(p.minors_out, base, rows, p.two_mats ? 2 * NN : NN, MA, lane);
                if (p.two_mats) T::store(p.minors_out + NN, base, rows, 2 * NN, MU, lane);
            }
            __syncwarp();
            if (p.mode == kModeMinors) continue;
            if (!p.single_det) {
                for (int i = lane; i < (T::STR << N); i += 32) MA[i] *= p.two_mats ? MU[i] : MA[i];
            }
        }
        __syncwarp();
        T::layers(MA, MC, P.gsel, s, m, q);
        T::store(p.c_out, base, rows, NN, MC, lane);
        __syncwarp();
    }
}

template <int N, int LG>
static int lanes_launch(const LanesParams &P, cudaStream_t s) {
    using T = Lanes<N, LG>;
    const size_t arrays = P.a.two_mats ? 3 : 2;
    const size_t smem = ((sizeof(typename T::Smem) + 15) & ~size_t(15)) + arrays * (T::STR << N) * sizeof(double);
    const size_t allow = ((sizeof(typename T::Smem) + 15) & ~size_t(15)) + 3 * (T::STR << N) * sizeof(double);
    int err = 0;
    const int64_t most = resident_ctas(cdet_lanes_kernel<N, LG>, 32, smem, allow, &err);
    if (err) return err;
    const int64_t need = (P.a.batch + T::MPW - 1) / T::MPW;
    cdet_lanes_kernel<N, LG><<<static_cast<int>(need < most ? need : most), 32, smem, s>>>(P);
    return static_cast<int>(cudaGetLastError());
}

// Fewest and most lanes per matrix (log2) that cdet_lanes_log2 gives out; nothing
// beyond them is compiled.
__host__ __device__ constexpr int lanes_least(int n) { return n > 6 ? n - 6 : 0; }
__host__ __device__ constexpr int lanes_most(int n) { return n < 4 ? 2 : n == 5 ? 4 : n == 7 ? 2 : 3; }

// Lanes per matrix (log2) at order n and this batch, or -1 for the
// one-CTA-per-matrix kernel (of 64 or 128 threads here). Both sides measured on
// a GB300, device us per call (CTA | this):
//   minors and sums: n = 4: 457 matrices 8.7 | 8.8;  n = 5: 1500 14.4 | 15.3, 2000 18 | 16, 16384 105 | 24
//     n = 6: 2000 20.7 | 21.6, 2300 25.6 | 21.8, 16384 126 | 48
//     n = 7: 4096 49 | 60, 5500 64 | 65, 6000 71 | 65, 16384 175 | 128
//     n = 8: 16384 255 | 276, 20000 312 | 341, 24000 374 | 359, 65536 1018 | 921
//   minors: n = 5: 1824 12 | 12, 2300 15 | 11;  n = 6: 2000 15 | 14, 8000 50 | 17;  n = 7: 3648 28 | 27,
//     4096 30 | 32, 6000 44 | 36;  n = 8: 9000 72 | 81, 11000 88 | 86, 16384 129 | 113
//   sums from weights: n = 4: 1500 5.6 | 5.9, 2300 8.3 | 6.0;  n = 5: 2100 7.0 | 8.9, 2200 10.0 | 8.9, 3200 10.3 | 9.6
//     n = 6: 8000 23 | 28, 11000 29 | 31, 13000 34 | 31, 16384 41 | 31
//     n = 7: 12000 52 | 51, 14000 60 | 77, 18000 75 | 80, 24000 97 | 87, 65536 266 | 205;  n = 8: 65536 489 | 596
// (256-thread CTAs took 1220, 1581 and 2210 us on 65536 of order 6, 7 and 8.)
// As few lanes per matrix as fill the chip (6 warps per SM) waste the fewest;
// below `least` lanes a warp's arrays leave too few warps per SM (n = 8, 65536:
// 918 us with 8 lanes, 1046 with 4, 1442 with 2).
int cdet_lanes_log2(int n, int64_t batch, int mode) {
    if (n > kLanesMaxN) return -1;
    static const int from[3][kLanesMaxN + 1] = {
        {0, 0, 0, 0, 457, 2000, 2000, 5000, 10500},        // minors
        {0, 0, 0, 0, 457, 1800, 2200, 5600, 22000},        // minors and sums
        {0, 0, 0, 0, 1900, 2200, 11500, 20000, 1 << 30}};  // sums from weights
    if (batch < from[mode][n]) return -1;
    const int least = mode == kModeMinors ? lanes_least(n) : (n > 5 ? n - 5 : n == 5 ? 1 : 0);
    int lg = least;
    while (lg < lanes_most(n) && (batch << (lg + 1)) <= int64_t(32) * 6 * 152) ++lg;
    return lg;
}

template <int N, int LG = lanes_least(N)>
static int lanes_for(const LanesParams &P, int lg, cudaStream_t s) {
    if constexpr (LG <= lanes_most(N)) return lg == LG ? lanes_launch<N, LG>(P, s) : lanes_for<N, LG + 1>(P, lg, s);
    return static_cast<int>(cudaErrorInvalidValue);
}

int launch_cdet_lanes(const CdetArgs &a, int lg, cudaStream_t s) {
    LanesParams P;
    P.a = a;
    P.gsel = cdet_gsel_packed(a.n);
    switch (a.n) {
        case 1: return lanes_for<1>(P, lg, s);
        case 2: return lanes_for<2>(P, lg, s);
        case 3: return lanes_for<3>(P, lg, s);
        case 4: return lanes_for<4>(P, lg, s);
        case 5: return lanes_for<5>(P, lg, s);
        case 6: return lanes_for<6>(P, lg, s);
        case 7: return lanes_for<7>(P, lg, s);
        default: return lanes_for<8>(P, lg, s);
    }
}

}  // namespace apm
