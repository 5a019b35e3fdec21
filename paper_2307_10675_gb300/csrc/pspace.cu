// Start vectors of the batched Davidson from a small exact eigenproblem (a
// "P-space" guess), and single Hamiltonian matrix elements.
//
// The lowest singlet of a body set can be a charge-transfer state whose
// leading determinant is not the one of lowest diagonal energy; started from
// that determinant plus a small random part, the Davidson iteration can meet
// its residual tolerance on an excited state before the ground-state component
// has grown.  The guess here diagonalises H exactly in the span of the
// spin-flip-symmetric pair functions u_K of the kPsp lowest-diagonal
// determinants K = (I_a, I_b), I_a <= I_b,
//   u_K = (|I_a I_b> + |I_b I_a>) / sqrt 2   (I_a != I_b),   u_K = |I_a I_a>,
// and starts from its lowest eigenvector.
//
// Matrix elements <I|H|J> of H = sum_pq h_pq E_pq + 1/2 sum_pqrs (pq|rs)
// (E_pq E_rs - delta_qr E_ps) between determinants (alpha string, beta string)
// follow the Slater–Condon rules on the bit masks: zero beyond double
// excitations; for a single excitation j -> a (spin s) the sign is the parity
// of the orbitals occupied strictly between a and j; a same-spin double is two
// such excitations applied in turn; an opposite-spin double is the product of
// the two single signs.
#include "dav_driver.cuh"
#include "hamiltonian.cuh"
#include "slater.cuh"

namespace ifci {

namespace {

constexpr int kPsp = kPspMax;   // pair functions in the guess space
constexpr int kSelThreads = 256;
constexpr int kSelPer = 4;      // candidates kept per thread during selection
constexpr int kSelCand = kSelThreads * kSelPer;

// Per problem: the kPsp lowest-diagonal canonical determinants (I_a <= I_b).
// Each thread keeps its kSelPer lowest over a strided scan, then the block
// sorts the candidates (bitonic, by value then index).
__device__ __forceinline__ void psp_select_kernel_body(const DavProb *__restrict__ probs, long long *__restrict__ pidx, int *__restrict__ pcount, int w_) {
    const DavProb p = probs[w_];
    __shared__ double sv[kSelCand];
    __shared__ long long si[kSelCand];
    double bv[kSelPer];
    long long bi[kSelPer];
#pragma unroll
    for (int u = 0; u < kSelPer; u++) {
        bv[u] = 1e300;
        bi[u] = 0x7fffffffffffffffll;
    }
    const int n = p.nb;
    for (long long I = threadIdx.x; I < p.ndet; I += kSelThreads) {
        const int a = (int)(I / n), b = (int)(I % n);
        if (p.sym && a > b) continue;
        double v = p.hd[I];
        long long i = I;
        if (v < bv[kSelPer - 1] || (v == bv[kSelPer - 1] && i < bi[kSelPer - 1])) {
#pragma unroll
            for (int u = 0; u < kSelPer; u++) {   // insertion into the sorted list
                if (v < bv[u] || (v == bv[u] && i < bi[u])) {
                    const double tv = bv[u];
                    const long long ti = bi[u];
                    bv[u] = v;
                    bi[u] = i;
                    v = tv;
                    i = ti;
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < kSelPer; u++) {
        sv[threadIdx.x * kSelPer + u] = bv[u];
        si[threadIdx.x * kSelPer + u] = bi[u];
    }
    __syncthreads();
    for (int size = 2; size <= kSelCand; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < kSelCand; t += kSelThreads) {
                const int partner = t ^ stride;
                if (partner > t) {
                    const bool up = (t & size) == 0;
                    const bool gt = sv[t] > sv[partner] || (sv[t] == sv[partner] && si[t] > si[partner]);
                    if (gt == up) {
                        const double tv = sv[t];
                        const long long ti = si[t];
                        sv[t] = sv[partner];
                        si[t] = si[partner];
                        sv[partner] = tv;
                        si[partner] = ti;
                    }
                }
            }
            __syncthreads();
        }
    }
    const long long nsym = p.ndim;
    const int pmax = p.gc ? kPspBlock : kPsp;
    const int P = nsym < pmax ? (int)nsym : pmax;
    if (threadIdx.x < kPsp) pidx[w_ * kPsp + threadIdx.x] = threadIdx.x < P ? si[threadIdx.x] : -1;
    if (threadIdx.x == 0) pcount[w_] = P;
}

__global__ void __launch_bounds__(kSelThreads) psp_select_kernel(const DavProb *__restrict__ probs, long long *__restrict__ pidx, int *__restrict__ pcount, int nprob_) {
    for (int w = blockIdx.x; w < nprob_; w += gridDim.x) {
        if (probs[w].seed) continue;   // started from its own vector: no P-space
        psp_select_kernel_body(probs, pidx, pcount, w);
        __syncthreads();   // shared memory is reused by the next body
    }
}

// Row-cyclic Jacobi on the symmetric P x P matrix A (shared memory, row
// stride LD), in two forms.  Sweeps end once the off-diagonal part is below
// 1e-26 of |A|_F^2 (a start guess needs no more); a rotation whose A_pq is
// below 1e-18 (|A_pp| + |A_qq|) only sets A_pq = A_qp = 0.  Zero couplings
// (other sectors, pair functions beyond a double excitation apart) are skipped.
// The order of rotations and every rounding are those of one rotation at a
// time: columns p, q <- fma(c, a_p, -(s a_q)), fma(s, a_p, c a_q), then rows,
// then V, whoever computes them.
//
// One warp: every lane derives the same rotation from the settled entries, then
// rotates the columns of its rows, and after a warp barrier its columns' rows
// and V.  The chain of dependent FP64 operations of one rotation bounds it.
// Serves the small blocks of sectored spaces, sixteen to an SM.
template <int MAXP>
__device__ __forceinline__ void psp_jacobi_cyclic(double *A, double *V, int P, double *red, double *red2) {
    constexpr int LD = MAXP + 1, R = (MAXP + 31) / 32;
    const int lane = threadIdx.x;
    for (int sweep = 0; sweep < 40; sweep++) {
#pragma unroll
        for (int u = 0; u < R; u++) {
            const int t = lane + 32 * u;
            if (t >= P) continue;
            double off = 0.0, all = 0.0;
            for (int c = 0; c < P; c++) {
                const double a2 = A[t * LD + c] * A[t * LD + c];
                all += a2;
                if (c != t) off += a2;
            }
            red[t] = off;
            red2[t] = all;
        }
        __syncwarp();
        double tot = 0.0, fro = 0.0;
        for (int i = 0; i < P; i++) {
            tot += red[i];
            fro += red2[i];
        }
        __syncwarp();
        if (tot <= 1e-26 * fro || tot == 0.0) break;
        for (int pp = 0; pp < P - 1; pp++)
            for (int q = pp + 1; q < P; q++) {
                const double apq = A[pp * LD + q];
                if (dmag(apq) < dbits(1e-300)) continue;
                const double app = A[pp * LD + pp], aqq = A[q * LD + q];
                __syncwarp();   // every lane has read the rotation's entries
                if (jacobi_negligible(app, aqq, apq)) {
                    if (lane == 0) A[pp * LD + q] = A[q * LD + pp] = 0.0;
                    __syncwarp();
                    continue;
                }
                double c, sn;
                jacobi_rotation(app, aqq, apq, c, sn);
#pragma unroll
                for (int u = 0; u < R; u++) {
                    const int t = lane + 32 * u;
                    if (t >= P) continue;
                    const double arp = A[t * LD + pp], arq = A[t * LD + q];
                    A[t * LD + pp] = c * arp - sn * arq;
                    A[t * LD + q] = sn * arp + c * arq;
                }
                __syncwarp();
#pragma unroll
                for (int u = 0; u < R; u++) {
                    const int t = lane + 32 * u;
                    if (t >= P) continue;
                    const double apr = A[pp * LD + t], aqr = A[q * LD + t];
                    A[pp * LD + t] = c * apr - sn * aqr;
                    A[q * LD + t] = sn * apr + c * aqr;
                    const double vrp = V[t * LD + pp], vrq = V[t * LD + q];
                    V[t * LD + pp] = c * vrp - sn * vrq;
                    V[t * LD + q] = sn * vrp + c * vrq;
                }
                __syncwarp();
            }
    }
}

// bar.sync and bar.arrive on a numbered barrier of all kPairThreads threads
constexpr int kPairThreads = 160;
__device__ __forceinline__ void pair_sync(int id) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kPairThreads) : "memory");
}
__device__ __forceinline__ void pair_arrive(int id) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kPairThreads) : "memory");
}

// Five warps: one derives the rotations, four apply them.  An SM sub-partition's
// FP64 pipe takes 64 clk for a warp instruction however few lanes are in it, so
// what bounds a rotation is the chain from its 2 x 2 block to the next one.
// The deriving warp therefore runs ahead: from the rows p and q as they stand
// before rotation (p, q) it computes row p and A_pp after it, which with the
// untouched diagonal is all that (p, q + 1) needs, while the four warps rotate
// A and V.  Where that does not find the next rotation (the end of a row, or an
// entry to be set to zero) it scans A.
// The others: lane l the p and lane l + 16 the q element of one row, then of
// one column, then of one row of V, a multiply and an FMA each.  Only the 2 x 2
// block needs both mixes of A; its rows and columns belong to one warp, so no
// barrier is needed between.
// Barrier 1: a rotation is applied to A (the four arrive, the deriving warp
// waits); barrier 2: the next one is in shared memory (it arrives, they wait).
template <int MAXP>
__device__ __forceinline__ void psp_jacobi_ahead(double *A, double *V, int P, double *red, double *red2) {
    static_assert(MAXP == 64, "sixteen rows to each of four warps");
    constexpr int LD = MAXP + 1;
    __shared__ double rot_c, rot_s;
    __shared__ int rot_p, rot_q;                   // rot_q < 0: the sweep is over
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, half = lane >> 4;
    for (int sweep = 0; sweep < 40; sweep++) {
        if (t < P) {
            double off = 0.0, all = 0.0;
            for (int c = 0; c < P; c++) {
                const double a2 = A[t * LD + c] * A[t * LD + c];
                all += a2;
                if (c != t) off += a2;
            }
            red[t] = off;
            red2[t] = all;
        }
        __syncthreads();
        const double *part = lane & 1 ? red2 : red;   // even lanes add up the off-diagonal part, odd lanes all
        double sum = 0.0;
        for (int i = 0; i < P; i++) sum += part[i];
        const double tot = __shfl_sync(0xffffffffu, sum, 0), fro = __shfl_sync(0xffffffffu, sum, 1);
        __syncthreads();
        if (tot <= 1e-26 * fro || tot == 0.0) break;
        if (warp == 4) {
            int p = 0, q = 0, nq = -1;             // the last rotation; nq >= 0: the next one is (p, nq)
            bool applied = true;                   // A has had the last one
            double app = 0.0, aqq = 0.0, apq = 0.0;
            while (true) {
                if (nq < 0) {
                    if (!applied) pair_sync(1);
                    applied = true;
                    int sp = p, sq = q + 1;
                    while (sp < P - 1) {
                        // first coupling of row sp from column sq on that is not zero
                        int f = P;
                        for (int c0 = sq; c0 < P; c0 += 32) {
                            const bool nz = c0 + lane < P && dmag(A[sp * LD + c0 + lane]) >= dbits(1e-300);
                            const unsigned m = __ballot_sync(0xffffffffu, nz);
                            if (m) {
                                f = c0 + __ffs(m) - 1;
                                break;
                            }
                        }
                        if (f >= P) {
                            sp++;
                            sq = sp + 1;
                            continue;
                        }
                        apq = A[sp * LD + f];
                        app = A[sp * LD + sp];
                        aqq = A[f * LD + f];
                        if (!jacobi_negligible(app, aqq, apq)) {
                            p = sp;
                            nq = f;
                            break;
                        }
                        __syncwarp();
                        if (lane == 0) A[sp * LD + f] = A[f * LD + sp] = 0.0;
                        __syncwarp();
                        sq = f + 1;
                    }
                    if (nq < 0) {
                        if (lane == 0) rot_q = -1;
                        __syncwarp();
                        pair_arrive(2);
                        break;
                    }
                }
                double c, s;
                jacobi_rotation(app, aqq, apq, c, s);
                if (jacobi_negligible(app, aqq, apq)) {   // found ahead, but to be set to zero
                    nq = -1;
                    continue;
                }
                q = nq;
                if (!applied) pair_sync(1);
                if (lane == 0) {
                    rot_p = p;
                    rot_q = q;
                    rot_c = c;
                    rot_s = s;
                }
                const int col = q + 1 + lane;
                const bool in = col < P;
                const double rp = in ? A[p * LD + col] : 0.0, rq = in ? A[q * LD + col] : 0.0;
                const double dg = in ? A[col * LD + col] : 0.0, aqp = A[q * LD + p];
                const double ms = dflip(s, 0x80000000u);
                // columns p of rows p and q, then row p; row p at the columns ahead
                const double xp = __fma_rn(c, app, __dmul_rn(ms, apq)), yp = __fma_rn(c, aqp, __dmul_rn(ms, aqq));
                const double row = __fma_rn(c, rp, __dmul_rn(ms, rq));
                app = __fma_rn(c, xp, __dmul_rn(ms, yp));
                const unsigned m = __ballot_sync(0xffffffffu, in && dmag(row) >= dbits(1e-300));
                nq = m ? q + __ffs(m) : -1;
                apq = __shfl_sync(0xffffffffu, row, __ffs(m) - 1);
                aqq = __shfl_sync(0xffffffffu, dg, __ffs(m) - 1);
                pair_arrive(2);
                applied = false;
            }
        } else {
            while (true) {
                pair_sync(2);
                const int q = rot_q, p = rot_p;
                if (q < 0) break;
                const double c = rot_c, s = rot_s;
                const double x = half ? s : c, y = half ? c : dflip(s, 0x80000000u);
                // slots 0 and 1 hold rows (columns) p and q, whose own slots get 0 and 1
                const int slot = 16 * warp + (lane & 15);
                int r = slot == 1 ? q : slot == q ? 1 : slot;
                r = r == 0 ? p : r == p ? 0 : r;
                const bool on = r < P;
                double ap = 0.0, aq = 0.0;
                if (on) {
                    ap = A[r * LD + p];
                    aq = A[r * LD + q];
                }
                __syncwarp();
                if (on) A[r * LD + (half ? q : p)] = __fma_rn(x, ap, __dmul_rn(y, aq));
                __syncwarp();
                if (on) {
                    ap = A[p * LD + r];
                    aq = A[q * LD + r];
                }
                __syncwarp();
                if (on) A[(half ? q : p) * LD + r] = __fma_rn(x, ap, __dmul_rn(y, aq));
                __syncwarp();
                pair_arrive(1);
                if (slot < P) {
                    ap = V[slot * LD + p];
                    aq = V[slot * LD + q];
                }
                __syncwarp();
                if (slot < P) V[slot * LD + (half ? q : p)] = __fma_rn(x, ap, __dmul_rn(y, aq));
                __syncwarp();
            }
        }
        __syncthreads();
    }
}

// The same by NT threads in round-robin order: a step rotates n / 2 disjoint
// index pairs at once, so every 2 x 2 block (pair i, pair j) of A changes on
// its own, A' = R_i^T A_ij R_j, and a sweep is n - 1 steps of two barriers
// instead of n (n - 1) / 2 dependent rotations.  The FP64 pipe (~1.8 FMA per
// clock and SM on this part) bounds it: per step 16 operations per block above
// the diagonal (the other half is its mirror image) and 4 per element pair of
// V.  n4 = P rounded up to a multiple of 4; the padding rows are zero and never
// rotate.
// T = float: a first pass that leaves few FP64 sweeps to do (psp_jacobi_refined);
// it stops at 1e-11 of |A|_F^2, near FP32's own rounding.
__device__ __forceinline__ bool pair_rotation(double app, double aqq, double apq, double &c, double &s, bool &zero) {
    if (dmag(apq) < dbits(1e-300)) return false;
    zero = jacobi_negligible(app, aqq, apq);
    if (!zero) jacobi_rotation(app, aqq, apq, c, s);
    return !zero;
}
__device__ __forceinline__ bool pair_rotation(float app, float aqq, float apq, float &c, float &s, bool &) {
    if (!(fabsf(apq) > 1e-9f * (fabsf(app) + fabsf(aqq)))) return false;
    const float tau = (aqq - app) / (2.0f * apq);
    const float t = (tau >= 0.0f ? 1.0f : -1.0f) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
    c = rsqrtf(1.0f + t * t);
    s = t * c;
    return true;
}

template <int MAXP, int NT, typename T>
__device__ __forceinline__ void psp_jacobi_pairs(T *A, T *V, int P, int sweeps, T small, T *red, T *red2) {
    static_assert(MAXP % 4 == 0 && NT >= MAXP && NT / 32 <= MAXP, "P-space sizes");
    constexpr int LD = MAXP + 1;
    __shared__ T rc[MAXP / 2], rsn[MAXP / 2];
    __shared__ int rp[MAXP / 2], rq[MAXP / 2];       // the step's index pairs; rq < 0: no rotation
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n4 = (P + 3) & ~3, npr = n4 / 2;
    for (int e = t; e < n4 * n4; e += NT) {
        const int r = e / n4, c = e % n4;
        if (r >= P || c >= P) A[r * LD + c] = T(0);
    }
    __syncthreads();
    for (int sweep = 0; sweep < sweeps; sweep++) {
        T off = T(0), all = T(0);
        for (int e = t; e < P * P; e += NT) {
            const int r = e / P, c = e % P;
            const T a = A[r * LD + c];
            all += a * a;
            if (c != r) off += a * a;
        }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        __syncthreads();   // red is free again
        if (lane == 0) {
            red[warp] = off;
            red2[warp] = all;
        }
        __syncthreads();
        off = all = T(0);
        for (int w = 0; w < NT / 32; w++) {
            off += red[w];
            all += red2[w];
        }
        if (off <= small * all || off == T(0)) break;
        for (int step = 0; step < n4 - 1; step++) {
            if (t < npr) {
                // index n4 - 1 stays, the others turn
                const int a = t == 0 ? n4 - 1 : (step + t) % (n4 - 1), b = t == 0 ? step : (step + n4 - 1 - t) % (n4 - 1);
                const int pp = min(a, b), q = max(a, b);
                const T app = A[pp * LD + pp], aqq = A[q * LD + q], apq = A[pp * LD + q];
                T c = T(1), sn = T(0);
                bool zero = false;
                const bool rot = pair_rotation(app, aqq, apq, c, sn, zero);
                if (zero) A[pp * LD + q] = A[q * LD + pp] = T(0);
                if (rot) {
                    const T xp = c * app - sn * apq, xq = sn * app + c * apq;   // columns of row p
                    const T yp = c * apq - sn * aqq, yq = sn * apq + c * aqq;   // columns of row q
                    A[pp * LD + pp] = c * xp - sn * yp;
                    A[q * LD + q] = sn * xq + c * yq;
                    A[pp * LD + q] = A[q * LD + pp] = c * xq - sn * yq;
                    rc[t] = c;
                    rsn[t] = sn;
                }
                rp[t] = pp;
                rq[t] = rot ? q : -1 - q;
            }
            __syncthreads();
            // blocks (i, j), i < j, of the npr pairs (npr is even): row r of the
            // folded triangle holds pair row r and pair row npr - 1 - r
            for (int e = t; e < npr / 2 * (npr - 1); e += NT) {
                const int r = e / (npr - 1), c = e % (npr - 1);
                const int i = c >= r ? r : npr - 1 - r, j = c >= r ? c + 1 : npr - 1 - c;
                int qi = rq[i], qj = rq[j];
                if (qi < 0 && qj < 0) continue;
                const T ci = qi >= 0 ? rc[i] : T(1), si = qi >= 0 ? rsn[i] : T(0);
                const T cj = qj >= 0 ? rc[j] : T(1), sj = qj >= 0 ? rsn[j] : T(0);
                const int pi = rp[i], pj = rp[j];
                if (qi < 0) qi = -1 - qi;
                if (qj < 0) qj = -1 - qj;
                const T a00 = A[pi * LD + pj], a01 = A[pi * LD + qj], a10 = A[qi * LD + pj], a11 = A[qi * LD + qj];
                const T x00 = cj * a00 - sj * a01, x01 = sj * a00 + cj * a01;
                const T x10 = cj * a10 - sj * a11, x11 = sj * a10 + cj * a11;
                const T b00 = ci * x00 - si * x10, b10 = si * x00 + ci * x10;
                const T b01 = ci * x01 - si * x11, b11 = si * x01 + ci * x11;
                A[pi * LD + pj] = A[pj * LD + pi] = b00;
                A[pi * LD + qj] = A[qj * LD + pi] = b01;
                A[qi * LD + pj] = A[pj * LD + qi] = b10;
                A[qi * LD + qj] = A[qj * LD + qi] = b11;
            }
            for (int e = t; e < npr * P; e += NT) {
                const int i = e / P, r = e % P, q = rq[i];
                if (q < 0) continue;
                const T c = rc[i], sn = rsn[i], vp = V[r * LD + rp[i]], vq = V[r * LD + q];
                V[r * LD + rp[i]] = c * vp - sn * vq;
                V[r * LD + q] = sn * vp + c * vq;
            }
            __syncthreads();
        }
    }
}

// P x P product X^T Y (or X Y with TX = false), every thread its elements into
// registers: element e = t + NT i of the result is (e / P, e % P).
template <int MAXP, int NT, bool TX>
__device__ __forceinline__ void psp_product(const double *X, const double *Y, int P, double (&out)[MAXP * MAXP / NT]) {
    constexpr int LD = MAXP + 1;
#pragma unroll
    for (int i = 0; i < MAXP * MAXP / NT; i++) {
        const int e = threadIdx.x + NT * i, r = e / P, c = e % P;
        out[i] = 0.0;
        if (e < P * P)
            for (int k = 0; k < P; k++) out[i] = fma(X[TX ? k * LD + r : r * LD + k], Y[k * LD + c], out[i]);
    }
}
template <int MAXP, int NT>
__device__ __forceinline__ void psp_store(double *X, int P, const double (&v)[MAXP * MAXP / NT]) {
    __syncthreads();   // every thread has read the operands
#pragma unroll
    for (int i = 0; i < MAXP * MAXP / NT; i++) {
        const int e = threadIdx.x + NT * i;
        if (e < P * P) X[e / P * (MAXP + 1) + e % P] = v[i];
    }
    __syncthreads();
}

// The FP64 sweeps from the eigenvectors of an FP32 solve: those, made orthogonal
// in FP64 by two Newton-Schulz steps X <- X + X (1 - X^T X) / 2 (1e-6 -> 1e-12
// -> rounding; E32 holds 1 - X^T X, whose own rounding the second step sees),
// turn A into X^T A X with off-diagonal elements ~1e-6 of the others, and about
// two FP64 sweeps are left of seven.  32 problems of 64 functions: 2.4 ms, 3.5 ms
// in FP64 throughout.  Blocks of A stay blocks (zeros stay zero in every step).  An
// FP32 solve that went wrong (numbers beyond its range) is dropped.
template <int MAXP, int NT>
__device__ __forceinline__ void psp_jacobi_refined(double *A, double *V, float *E32, int P, double *red, double *red2) {
    constexpr int LD = MAXP + 1, R = MAXP * MAXP / NT;
    const int t = threadIdx.x;
    if (P >= 8) {
        float *A32 = reinterpret_cast<float *>(V), *V32 = A32 + MAXP * LD;   // V is not needed yet
        for (int e = t; e < P * P; e += NT) {
            const int r = e / P, c = e % P;
            A32[r * LD + c] = d2f(A[r * LD + c]);
            V32[r * LD + c] = r == c ? 1.0f : 0.0f;
        }
        __syncthreads();
        psp_jacobi_pairs<MAXP, NT, float>(A32, V32, P, 12, 1e-11f, reinterpret_cast<float *>(red), reinterpret_cast<float *>(red2));
        __syncthreads();
        double v[R];
#pragma unroll
        for (int i = 0; i < R; i++) {
            const int e = t + NT * i;
            v[i] = e < P * P ? f2d(V32[e / P * LD + e % P]) : 0.0;
        }
        psp_store<MAXP, NT>(V, P, v);
        bool bad = false;
        for (int step = 0; step < 2 && !bad; step++) {
            psp_product<MAXP, NT, true>(V, V, P, v);
#pragma unroll
            for (int i = 0; i < R; i++) {
                const int e = t + NT * i;
                if (e >= P * P) continue;
                const float d = d2f((e / P == e % P ? 1.0 : 0.0) - v[i]);
                E32[e / P * LD + e % P] = d;
                if (!(fabsf(d) < 1e-3f)) bad = true;
            }
            bad = __syncthreads_or(bad);
            // X + X E / 2
#pragma unroll
            for (int i = 0; i < R; i++) {
                const int e = t + NT * i, r = e / P, c = e % P;
                v[i] = 0.0;
                if (e >= P * P) continue;
                float x = 0.0f;   // X E is at most 1e-3: FP32 keeps the first step's result to 1e-9, the second's to 1e-16
                for (int k = 0; k < P; k++) x = fmaf(d2f(V[r * LD + k]), E32[k * LD + c], x);
                v[i] = V[r * LD + c] + 0.5 * f2d(x);
            }
            psp_store<MAXP, NT>(V, P, v);
        }
        if (!bad) {
            psp_product<MAXP, NT, false>(A, V, P, v);
            psp_store<MAXP, NT>(A, P, v);
            psp_product<MAXP, NT, true>(V, A, P, v);
            psp_store<MAXP, NT>(A, P, v);
        } else {
            for (int e = t; e < P * P; e += NT) V[e / P * LD + e % P] = e / P == e % P ? 1.0 : 0.0;
            __syncthreads();
        }
    }
    psp_jacobi_pairs<MAXP, NT, double>(A, V, P, 40, 1e-26, red, red2);
}

// Per problem (one block of NT threads): H in the pair functions, its lowest
// eigenvectors, written to the start slots 0..nv-1; the random start vector is
// cleared on the P-space determinants.
//
// NT = 256 runs the round-robin sweeps, the others the cyclic ones.  The
// round-robin order is the faster one for a 64-function problem (2.2 ms, against
// 20.1 ms with one rotation at a time; less after an FP32 solve) and serves the
// whole spaces of FP64 solves, where a last-bit change of the start vector stays
// one, and of direct batches in every precision, whose energies it moves by
// 1e-13 (FP64E) to 3e-11 (mixed) of themselves (32 spaces CAS(4e,10o) in FP64E:
// 27.5 ms, 8.1 ms with the Rayleigh-Ritz problems in that order too).  In an
// expansion with a quantised contraction (FP64E and the mixed modes that end on
// it) such a change turns up at the contraction's own level, ~5e-11 Eh, in
// increments that are differences of energies; it moves them without taking them
// farther from FP64 (davidson.cu, jacobi_pairs).  Those and HBCI keep the order of
// rotations, and with it every bit of their start vectors, on five warps a
// problem: 64 functions 20.1 ms on one warp, 13.8 ms; 298 such problems at once
// 21.9 ms, 15.7 ms; the P-space solves of an expansion of 298 sets 58.9 ms,
// 42.9 ms.  So do the blocks of sectored spaces (MAXP = 24), which come by the
// hundred thousand and share an SM sixteen at a time, a warp each.
template <int MAXP, int NT>
__device__ __forceinline__ void psp_solve_kernel_body(const DavProb *__restrict__ probs, const HdiagDesc *__restrict__ hdd, const long long *__restrict__ pidx,
                 const int *__restrict__ pcount, int max_space, double *__restrict__ blk_energy, int w_) {
    constexpr int LD = MAXP + 1;
    extern __shared__ double psm[];
    double *A = psm;                       // [MAXP][LD]
    double *V = psm + MAXP * LD;           // [MAXP][LD]
    __shared__ double red[MAXP], red2[MAXP];
    __shared__ unsigned long long adj[MAXP];
    __shared__ int comp[MAXP], order[MAXP], blk[MAXP], cols[kStartP];
    const DavProb p = probs[w_];
    const HdiagDesc d = hdd[w_];
    const int P = pcount[w_];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n = p.nb;
    const double rs2 = 0.7071067811865476;
    // <u_r|H|u_c>, every term of the pair functions written out (in an
    // off-diagonal block, whose spin-flip image is not iterated, u_K = |K>)
    for (int e = t; e < P * P; e += NT) {
        const int r = e / P, c = e % P;
        const long long K = pidx[w_ * kPsp + r], L = pidx[w_ * kPsp + c];
        const int ka = (int)(K / n), kb = (int)(K % n), la = (int)(L / n), lb = (int)(L % n);
        const int nbra = (ka == kb || !p.sym) ? 1 : 2, nket = (la == lb || !p.sym) ? 1 : 2;
        const double f = (nbra == 2 ? rs2 : 1.0) * (nket == 2 ? rs2 : 1.0);
        double v = 0.0;
        for (int x = 0; x < nbra; x++)
            for (int y = 0; y < nket; y++) {
                // (row, column) local indices of the bra and ket determinants
                const int ba = x ? kb : ka, bb = x ? ka : kb, ca = y ? lb : la, cb = y ? la : lb;
                v += h_element(d.n, d.h1, d.eri, (uint32_t)d.strings[blk_row(p, ba)],
                               (uint32_t)d.strings[blk_col(p, bb)], (uint32_t)d.strings[blk_row(p, ca)],
                               (uint32_t)d.strings[blk_col(p, cb)]);
            }
        A[r * LD + c] = f * v;
        V[r * LD + c] = r == c ? 1.0 : 0.0;
    }
    __syncthreads();
    // blocks of the P-space: connected components of the coupling graph
    // (|A_ij| above 1e-12 of the largest element); distant bodies make H split
    // into (nearly) decoupled sectors, and the start block takes the lowest
    // eigenvector of each of the lowest blocks first
    {
        double amax = 0.0;
        for (int e = t; e < P * P; e += NT) amax = fmax(amax, fabs(A[(e / P) * LD + e % P]));
        for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        if (lane == 0) red[warp] = amax;   // NT / 32 <= MAXP
        __syncthreads();
        for (int w = 0; w < NT / 32; w++) amax = fmax(amax, red[w]);
        for (int r = t; r < P; r += NT) {
            unsigned long long m = 0ull;
            for (int c = 0; c < P; c++)
                if (fabs(A[r * LD + c]) > 1e-12 * amax) m |= 1ull << c;
            adj[r] = m;
        }
        __syncthreads();
        if (t == 0) {
            unsigned long long left = P == 64 ? ~0ull : (1ull << P) - 1ull;
            for (int ncomp = 0; left; ncomp++) {
                unsigned long long front = left & (~left + 1ull), members = 0ull;
                while (front) {
                    const int u = __ffsll((long long)front) - 1;
                    members |= 1ull << u;
                    comp[u] = ncomp;
                    front = (front | (adj[u] & left)) & ~members;
                }
                left &= ~members;
            }
        }
    }
    __syncthreads();
    if constexpr (NT == 32) psp_jacobi_cyclic<MAXP>(A, V, P, red, red2);
    else if constexpr (NT == kPairThreads) psp_jacobi_ahead<MAXP>(A, V, P, red, red2);
    else psp_jacobi_refined<MAXP, NT>(A, V, reinterpret_cast<float *>(psm + 2 * MAXP * LD), P, red, red2);
    __syncthreads();
    int nv, ns;
    start_block(p.ndim, max_space, false, &nv, &ns);
    // eigenvalues in ascending order; each eigenvector's block is the block of
    // its largest component (entries that are not numbers keep their own place)
    for (int r = t; r < P; r += NT) {
        order[r] = r;
        blk[r] = comp[r];
    }
    __syncthreads();
    for (int r = t; r < P; r += NT) {
        const double ev = A[r * LD + r];
        int rank = 0, g = 0;
        for (int i = 0; i < P; i++) {
            const double o = A[i * LD + i];
            if (o < ev || (o == ev && i < r)) rank++;
            if (fabs(V[i * LD + r]) > fabs(V[g * LD + r])) g = i;
        }
        order[rank] = r;
        blk[rank] = comp[g];
    }
    __syncthreads();
    if (t == 0) {
        // rank of each block by its lowest eigenvalue: first[] = the eigenpair
        // index (in ascending order) that opens block rank 0, 1, ...
        int first[MAXP], nb = 0;
        unsigned long long seen = 0ull, taken = 0ull;
        for (int r = 0; r < P; r++)
            if (!(seen >> blk[r] & 1ull)) {
                seen |= 1ull << blk[r];
                first[nb++] = r;
            }
        if (blk_energy) {
            blk_energy[2 * w_] = A[order[first[0]] * LD + order[first[0]]];
            blk_energy[2 * w_ + 1] = nb > 1 ? A[order[first[1]] * LD + order[first[1]]] : 1e300;
        }
        int nc = 0;
        const int seed = p.seed_block;
        if (seed > 0 && seed < nb) {
            // second pass: that block's lowest vector first, then the lowest
            // eigenvectors outside the blocks ranked below it
            cols[nc++] = order[first[seed]];
            taken |= 1ull << first[seed];
            for (int r = 0; r < P && nc < nv; r++) {
                bool lower = false;
                for (int q = 0; q < seed; q++)
                    if (blk[r] == blk[first[q]]) lower = true;
                if (!(taken >> r & 1ull) && !lower) {
                    cols[nc++] = order[r];
                    taken |= 1ull << r;
                }
            }
        } else {
            // first the lowest eigenvector of each block (in order of those
            // eigenvalues), then the next lowest eigenvectors
            for (int k = 0; k < nb && nc < nv; k++) {
                cols[nc++] = order[first[k]];
                taken |= 1ull << first[k];
            }
        }
        for (int r = 0; r < P && nc < nv; r++)
            if (!(taken >> r & 1ull)) {
                cols[nc++] = order[r];
                taken |= 1ull << r;
            }
    }
    __syncthreads();
    // the nv chosen columns, each sign fixed by its largest component
    for (int u = t; u < P; u += NT) {
        const long long K = pidx[w_ * kPsp + u];
        const int ka = (int)(K / n), kb = (int)(K % n);
        const long long KT = (long long)kb * n + ka;
        for (int r = 0; r < nv; r++) {
            const int col = cols[r];
            int g = 0;
            for (int i = 1; i < P; i++)
                if (fabs(V[i * LD + col]) > fabs(V[g * LD + col])) g = i;
            const double y = (V[g * LD + col] < 0 ? -1.0 : 1.0) * V[u * LD + col];
            double *Br = p.B + (long long)r * p.ndet;
            if (ka == kb || !p.sym) {
                Br[K] = y;
            } else {
                Br[K] = y * rs2;
                Br[KT] = y * rs2;
            }
        }
        if (ns >= 0) {   // the random vector becomes exactly orthogonal to the block
            double *Bn = p.B + (long long)ns * p.ndet;
            Bn[K] = 0.0;
            if (p.sym) Bn[KT] = 0.0;
        }
    }
}

// Whole spaces (MAXP = 64) or blocks of sectored spaces (MAXP = 24); a problem
// started from its own vector needs no P-space guess.
template <int MAXP, int NT>
__global__ void __launch_bounds__(NT) psp_solve_kernel(const DavProb *__restrict__ probs, const HdiagDesc *__restrict__ hdd, const long long *__restrict__ pidx,
                 const int *__restrict__ pcount, int max_space, double *__restrict__ blk_energy, int nprob_) {
    for (int w = blockIdx.x; w < nprob_; w += gridDim.x) {
        if (probs[w].seed || (probs[w].gc != nullptr) != (MAXP < kPsp)) continue;
        psp_solve_kernel_body<MAXP, NT>(probs, hdd, pidx, pcount, max_space, blk_energy, w);
        __syncthreads();   // shared memory is reused by the next body
    }
}

// partial |.|^2 of the random start vector per vector work item
__device__ __forceinline__ void norm_part_kernel_body(const DavProb *__restrict__ probs,
                                                        const DavState *__restrict__ st,
                                                        const WorkItem *__restrict__ items, double *__restrict__ part, int w_) {
    const WorkItem it = items[w_];
    const DavProb &p = probs[it.prob];
    const int ns = st[it.prob].noise_slot;
    double acc = 0.0;
    const long long end = min(it.start + (long long)kVecChunk, p.ndet);
    if (ns >= 0) {
        const double *v = p.B + (long long)ns * p.ndet;
        for (long long I = it.start + threadIdx.x; I < end; I += blockDim.x) acc += v[I] * v[I];
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ double red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < 8; i++) s += red[i];
        part[(long long)w_ * kNP] = s;
    }
}

__global__ void __launch_bounds__(256) norm_part_kernel(const DavProb *__restrict__ probs,
                                                        const DavState *__restrict__ st,
                                                        const WorkItem *__restrict__ items, double *__restrict__ part, int nitem_) {
    for (int w = blockIdx.x; w < nitem_; w += gridDim.x) {
        norm_part_kernel_body(probs, st, items, part, w);
        __syncthreads();   // shared memory is reused by the next body
    }
}

// <bra_k|H|ket_k> for determinant index pairs (C entry point below)
__global__ void h_elements_kernel(int n, int nstr, const uint64_t *__restrict__ strings,
                                  const double *__restrict__ h1, const double *__restrict__ eri, long long count,
                                  const long long *__restrict__ bra, const long long *__restrict__ ket,
                                  double *__restrict__ out) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const long long I = bra[i], J = ket[i];
    out[i] = h_element(n, h1, eri, (uint32_t)strings[I / nstr], (uint32_t)strings[I % nstr],
                       (uint32_t)strings[J / nstr], (uint32_t)strings[J % nstr]);
}

}  // namespace

size_t psp_workspace_bytes(int nprob) {
    return ws_round((size_t)nprob * kPsp * sizeof(long long)) + ws_round((size_t)nprob * sizeof(int));
}

// Fills the P-space slots of every problem's start block, clears the random
// start vector on the P-space determinants and stores its |.|^2 per item in
// part (the caller normalises it).
int launch_pspace_start(ifci_handle_t h, const DavBatch &b, const HdiagDesc *d_hd, cudaStream_t s) {
    long long *pidx = b.d_pidx;
    int *pcount = b.d_pcount;
    if (!pidx || !pcount) return set_error(h, IFCI_ERR_OOM, "davidson: workspace (P-space)");
    {
        ProfScope ps(h, s, PK_SETUP);
        psp_select_kernel<<<stride_grid(h->device, b.nprob, 8), kSelThreads, 0, s>>>(b.d_probs, pidx, pcount, b.nprob);
        IFCI_LAUNCH_CHECK(h);
    }
    bool whole = false, sector = false;
    for (const DavProb &p : b.probs) {
        whole = whole || (!p.gc && !p.seed);
        sector = sector || (p.gc && !p.seed);
    }
    constexpr int smem = 2 * kPsp * (kPsp + 1) * (int)sizeof(double);   // 65 KB
    if (whole && b.any_order) {
        static SmemOptIn opt;
        constexpr int smem_refined = smem + kPsp * (kPsp + 1) * (int)sizeof(float);   // 82 KB
        IFCI_CUDA_TRY(h, ensure_smem(opt, h->device, psp_solve_kernel<kPsp, 256>, smem_refined));
        ProfScope ps(h, s, PK_PSPACE);
        psp_solve_kernel<kPsp, 256><<<stride_grid(h->device, b.nprob, 2), 256, smem_refined, s>>>(
            b.d_probs, d_hd, pidx, pcount, b.max_space, b.d_blk_energy, b.nprob);
        IFCI_LAUNCH_CHECK(h);
    } else if (whole) {
        static SmemOptIn opt;
        IFCI_CUDA_TRY(h, ensure_smem(opt, h->device, psp_solve_kernel<kPsp, kPairThreads>, smem));
        ProfScope ps(h, s, PK_PSPACE);
        psp_solve_kernel<kPsp, kPairThreads><<<stride_grid(h->device, b.nprob, 3), kPairThreads, smem, s>>>(
            b.d_probs, d_hd, pidx, pcount, b.max_space, b.d_blk_energy, b.nprob);
        IFCI_LAUNCH_CHECK(h);
    }
    if (sector) {
        constexpr int smem24 = 2 * kPspBlock * (kPspBlock + 1) * (int)sizeof(double);   // 9.6 KB
        ProfScope ps(h, s, PK_PSPACE);
        psp_solve_kernel<kPspBlock, 32><<<stride_grid(h->device, b.nprob, 16), 32, smem24, s>>>(
            b.d_probs, d_hd, pidx, pcount, b.max_space, b.d_blk_energy, b.nprob);
        IFCI_LAUNCH_CHECK(h);
    }
    ProfScope ps(h, s, PK_SETUP);
    norm_part_kernel<<<stride_grid(h->device, (long long)b.vitems.size(), 8), 256, 0, s>>>(b.d_probs, b.d_state, b.d_vitems, b.d_part, (int)b.vitems.size());
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

}  // namespace ifci

extern "C" int ifci_h_elements(ifci_handle_t h, const ifci_strings_t *str, const double *h1, const double *eri,
                               long long count, const long long *bra, const long long *ket, double *out,
                               ifci_stream_t stream) {
    using namespace ifci;
    if (!h) return IFCI_ERR_INVALID_ARG;
    if (!str || !str->strings || !h1 || !eri || count < 0 || (count > 0 && (!bra || !ket || !out)))
        return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_h_elements: bad arguments");
    int nstr = 0, nexc = 0;
    if (ifci_string_counts(str->norb, str->nelec_spin, &nstr, &nexc) != IFCI_OK || nstr != str->nstr)
        return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_h_elements: inconsistent string table");
    if (count == 0) return IFCI_OK;
    IFCI_CUDA_TRY(h, cudaSetDevice(h->device));
    const int threads = 128;
    const long long blocks = (count + threads - 1) / threads;
    h_elements_kernel<<<(unsigned)blocks, threads, 0, as_cuda(stream)>>>(str->norb, nstr, str->strings, h1, eri,
                                                                          count, bra, ket, out);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}
