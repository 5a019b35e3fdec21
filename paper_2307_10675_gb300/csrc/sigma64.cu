// Plain FP64 sigma build, every nonzero element of H once.
//
//   sigma[Ia][Ib] = sum_J  h[Ia][J] c[J][Ib]                       (alpha alpha)
//                 + sum_J  h[Ib][J] c[Ia][J]                       (beta beta)
//                 + sum_{A in exc(Ib)} sum_{B in exc(Ia)} s_A s_B (A|B) c[J_B][J_A]
//
// h is the Hamiltonian of one spin's strings (one-electron part and same-spin
// repulsion, Slater-Condon): 1 + m (n-m) + C(m,2) C(n-m,2) elements per string,
// the same columns for every problem of a (norb, nelec_spin) class.  exc(I) are
// the nexc = m (n - m + 1) single excitations of a string (diagonal ones
// included), (A|B) the packed two-electron integrals.
//
// GB300 issues ~1.8 FP64 FMAs per clock and SM, so the count of FMAs decides:
// nexc^2 + 2 nnz per determinant (33^2 + 2 x 166 for CAS(6e,13o)) against the
// npair^2 (91^2) of a dense contraction over all orbital pairs, whose
// intermediates also went through HBM.  Next to one FMA (18 clocks per warp)
// the two shared-memory reads that feed it (one row element of c, one integral,
// both at lane-dependent addresses) hide.
//
// One block per alpha string Ia.  The rows c[J_B] and the integral columns of
// kb excitations B at a time sit in shared memory (the sign s_B is taken into
// the rows), each thread owns determinants Ib = t, t + blockDim, ...; s_A flips
// the accumulator's sign bit instead of costing a multiplication.  58.9 KB per
// block (54 KB of rows, 2.5 KB of lists, 1 KB of the system's) leave three blocks
// on an SM, whose loads overlap another's FMAs.  Rows cut to 53.5 KB let a fourth
// in: CAS(12e,12o) 4.49 ms, 3.86 ms; 64 problems of CAS(4e,12o) 4 % faster; but
// eight of CAS(6e,12o) 22.6 ms, 22.9 ms, and CAS(6e,13o) 285 us, 289 us.
//
// Measured: CAS(6e,13o) 240 us and 9 us for the lists (dense contraction 1634 us,
// gather and scatter 103 us before), 1.16e8 FMAs at 0.88 of a DGEMM's rate.
#include <algorithm>

#include "sigma.cuh"
#include "slater.cuh"

namespace ifci {

namespace {

constexpr int kMaxThreads64 = 512;
constexpr int kList = 128;              // alpha-alpha elements staged at a time
constexpr int kMaxExc = (kMaxNorb + 1) * (kMaxNorb + 1) / 4;   // most excitations m (n - m + 1) of a string
constexpr int kCapSmall = 6912, kCapMid = 13824, kCapLarge = 28160;   // doubles: 3, 2 or 1 blocks per SM

// the input row and the sums are kept in shared memory too, unless the strings
// are too many for that
__host__ __device__ inline int rows64(int nstr, int np) { return 3ll * nstr + np <= kCapLarge ? 2 : 0; }
// doubles a problem takes with kb excitations per pass
__host__ __device__ inline long long need64(int nstr, int np, int kb) {
    return (long long)nstr * (kb + rows64(nstr, np)) + (long long)np * (kb | 1);
}
// most excitations per pass that fit into cap doubles
__host__ __device__ inline int fit64(int nstr, int np, int nexc, long long cap) {
    long long kb = (cap - (long long)rows64(nstr, np) * nstr) / (nstr + np);
    if (kb > nexc) kb = nexc;
    while (kb > 0 && need64(nstr, np, (int)kb) > cap) kb--;
    return (int)kb;
}

__device__ __forceinline__ void sigma64_body(const SigmaProb &p, int ka, int cap) {
    extern __shared__ double sm[];
    __shared__ double lv[kList];
    __shared__ int lj[kList], lx[kMaxExc];
    if (p.active && !*p.active) return;
    const int nstr = p.nstr, nexc = p.nexc, np = p.np, nnz = p.nnz, t = threadIdx.x, nt = blockDim.x;
    const double *__restrict__ c = p.cbase + (p.cslot ? (long long)*p.cslot : 0ll) * p.stride;
    double *__restrict__ out = p.sbase + (p.sslot ? (long long)*p.sslot : 0ll) * p.stride + (long long)ka * nstr;
    const int32_t *__restrict__ exc = p.exc;
    const double *__restrict__ hval = p.hval;
    const int *__restrict__ hidx = p.hidx;
    const int rows = rows64(nstr, np);
    const double *row = rows ? sm : c + (long long)ka * nstr;
    double *acc = rows ? sm + nstr : out, *Cs = sm + rows * nstr;
    const int kb = fit64(nstr, np, nexc, cap), ldv = kb | 1;
    double *Vs = Cs + (size_t)kb * nstr;
    if (rows)
        for (int i = t; i < nstr; i += nt) sm[i] = c[(long long)ka * nstr + i];
    for (int i = t; i < nexc; i += nt) lx[i] = exc[(size_t)ka * nexc + i];
    __syncthreads();
    // beta beta: the string's own elements, the row from shared memory
    for (int ib = t; ib < nstr; ib += nt) {
        double a0 = 0.0, a1 = 0.0;
        int e = 0;
#pragma unroll 4
        for (; e + 1 < nnz; e += 2) {
            a0 = fma(hval[(size_t)e * nstr + ib], row[hidx[(size_t)e * nstr + ib]], a0);
            a1 = fma(hval[(size_t)(e + 1) * nstr + ib], row[hidx[(size_t)(e + 1) * nstr + ib]], a1);
        }
        if (e < nnz) a0 = fma(hval[(size_t)e * nstr + ib], row[hidx[(size_t)e * nstr + ib]], a0);
        acc[ib] = a0 + a1;
    }
    // alpha alpha: whole rows of c, the same for every Ib
    for (int e0 = 0; e0 < nnz; e0 += kList) {
        const int ne = min(kList, nnz - e0);
        __syncthreads();
        for (int i = t; i < ne; i += nt) {
            lv[i] = hval[(size_t)(e0 + i) * nstr + ka];
            lj[i] = hidx[(size_t)(e0 + i) * nstr + ka];
        }
        __syncthreads();
        for (int ib = t; ib < nstr; ib += nt) {
            double a0 = 0.0, a1 = 0.0;
            int e = 0;
#pragma unroll 2
            for (; e + 1 < ne; e += 2) {
                a0 = fma(lv[e], c[(long long)lj[e] * nstr + ib], a0);
                a1 = fma(lv[e + 1], c[(long long)lj[e + 1] * nstr + ib], a1);
            }
            if (e < ne) a0 = fma(lv[e], c[(long long)lj[e] * nstr + ib], a0);
            acc[ib] += a0 + a1;
        }
    }
    // alpha beta, kb alpha excitations at a time
    for (int k0 = 0; k0 < nexc; k0 += kb) {
        const int kn = min(kb, nexc - k0);
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < kn; k++) {   // loads of several excitations in flight
            const int32_t x = lx[k0 + k];
            const uint32_t neg = (uint32_t)(x & 1) << 31;
            const double *src = c + (long long)exc_J(x) * nstr, *v = p.eri + (long long)exc_pair(x) * np;
            for (int i = t; i < nstr; i += nt) Cs[(size_t)k * nstr + i] = dflip(src[i], neg);
            for (int A = t; A < np; A += nt) Vs[A * ldv + k] = v[A];
        }
        __syncthreads();
        for (int ib = t; ib < nstr; ib += nt) {
            const int32_t *eb = exc + (size_t)ib * nexc;
            double a0 = 0.0, a1 = 0.0;
            uint32_t cur = 0;   // sign the accumulators carry
            for (int e = 0; e < nexc; e++) {
                const int32_t x = eb[e];
                const uint32_t neg = (uint32_t)(x & 1) << 31;
                a0 = dflip(a0, cur ^ neg);
                a1 = dflip(a1, cur ^ neg);
                cur = neg;
                const double *v = Vs + exc_pair(x) * ldv, *cs = Cs + exc_J(x);
                int k = 0;
#pragma unroll 2
                for (; k + 1 < kn; k += 2) {
                    a0 = fma(v[k], cs[(size_t)k * nstr], a0);
                    a1 = fma(v[k + 1], cs[(size_t)(k + 1) * nstr], a1);
                }
                if (k < kn) a0 = fma(v[k], cs[(size_t)k * nstr], a0);
            }
            acc[ib] += dflip(a0, cur) + dflip(a1, cur);
        }
    }
    if (rows)
        for (int ib = t; ib < nstr; ib += nt) out[ib] = acc[ib];   // own elements
}

// one problem by value, or a plan's items
__global__ void __launch_bounds__(kMaxThreads64) sigma64_one_kernel(const SigmaProb p, int cap) {
    sigma64_body(p, blockIdx.x, cap);
}
__global__ void __launch_bounds__(kMaxThreads64)
sigma64_kernel(const SigmaProb *__restrict__ probs, const WorkItem *__restrict__ items, int cap) {
    const WorkItem it = items[blockIdx.x];
    sigma64_body(probs[it.prob], (int)it.start, cap);
}

// Element list of the string Hamiltonian: entry 0 the diagonal, then the
// single, then the double excitations (occupied major), at [entry][string].
// val and idx may each be nullptr.  A lane owns one of kStringHChunk strings,
// a warp one entry at a time (the same kind of element in all lanes); the
// gridDim.y parts of a problem share its entries.  The binomials that rank and
// unrank strings sit in shared memory: lanes read them at addresses of their
// own, which a kernel parameter serves one after the other.
// CAS(6e,13o), 166 entries of 286 strings: 9.4 us; 9 blocks, a string unranked for
// each element from the parameter, took 56 us.
__device__ __forceinline__ void string_h_body(const StringHDesc &d, int I0, const StringBinom &B) {
    const int n = d.n, m = d.m, nv = n - m, ns = m * nv, nvp = nv * (nv - 1) / 2, lane = threadIdx.x % kStringHChunk;
    __shared__ int bin[32][33];
    for (int t = threadIdx.x; t < n * (m + 1); t += 256) bin[t / (m + 1)][t % (m + 1)] = B.c[t / (m + 1)][t % (m + 1)];
    __syncthreads();
    const int I = I0 + lane;
    if (I >= d.nstr) return;
    const uint32_t bra = string_of_rank(I, n, m, bin), vir = ~bra & (n == 32 ? ~0u : (1u << n) - 1u);
    auto nth = [](uint32_t x, int k) {
        for (; k > 0; k--) x &= x - 1;
        return x & (~x + 1u);
    };
    for (int e = blockIdx.y * (256 / kStringHChunk) + threadIdx.x / kStringHChunk; e < d.nnz; e += gridDim.y * (256 / kStringHChunk)) {
        uint32_t ket = bra;
        if (e > ns) {
            int o = (e - 1 - ns) / nvp, v = (e - 1 - ns) % nvp, i = 0, a = 0;
            while (o >= m - 1 - i) o -= m - 1 - i++;       // pair (i, i + 1 + o) of the occupied
            while (v >= nv - 1 - a) v -= nv - 1 - a++;     // and of the empty orbitals
            ket ^= nth(bra, i) | nth(bra, i + 1 + o) | nth(vir, a) | nth(vir, a + 1 + v);
        } else if (e > 0) {
            ket ^= nth(bra, (e - 1) / nv) | nth(vir, (e - 1) % nv);
        }
        if (d.idx) d.idx[(size_t)e * d.nstr + I] = string_rank_of(ket, bin);
        if (d.val) d.val[(size_t)e * d.nstr + I] = h_element(n, d.h1, d.eri, bra, 0u, ket, 0u);
    }
}

__global__ void __launch_bounds__(256) string_h_one_kernel(const StringHDesc d, const StringBinom B) {
    string_h_body(d, blockIdx.x * kStringHChunk, B);
}
__global__ void __launch_bounds__(256) string_h_kernel(const StringHDesc *__restrict__ desc, const WorkItem *__restrict__ items,
                                                       const StringBinom B) {
    const WorkItem it = items[blockIdx.x];
    string_h_body(desc[it.prob], (int)it.start, B);
}

// parts of a problem's entries: about two blocks per SM, eight entries to a part
static int string_h_parts(ifci_handle_t h, int nblk, int nnz) {
    return std::max(1, std::min((nnz + 7) / 8, 2 * device_sm_count(h->device) / nblk));
}

int cap64(const SigmaProb *probs, int nprob) {
    for (int cap : {kCapSmall, kCapMid}) {
        bool ok = true;
        for (int i = 0; i < nprob && ok; i++) {
            const SigmaProb &p = probs[i];
            ok = fit64(p.nstr, p.np, p.nexc, cap) >= std::min(p.nexc, 4);
        }
        if (ok) return cap;
    }
    return kCapLarge;
}

}  // namespace

StringBinom string_binom() {
    StringBinom B;
    for (int i = 0; i < 32; i++)
        for (int j = 0; j < 32; j++) B.c[i][j] = (int)std::min<long long>(binom(i, j), 0x7fffffff);
    return B;
}

bool sigma64_supported(int np, int nstr, int nexc) { return fit64(nstr, np, nexc, kCapLarge) >= 1; }

int string_h_nnz(int n, int m) { return 1 + m * (n - m) + m * (m - 1) / 2 * ((n - m) * (n - m - 1) / 2); }

int launch_string_h(ifci_handle_t h, const StringHDesc &one, cudaStream_t s) {
    const int nblk = (one.nstr + kStringHChunk - 1) / kStringHChunk;
    string_h_one_kernel<<<dim3(nblk, string_h_parts(h, nblk, one.nnz)), 256, 0, s>>>(one, string_binom());
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

int launch_string_h_batch(ifci_handle_t h, const StringHDesc *d_desc, const WorkItem *d_items, int nitem, cudaStream_t s) {
    if (nitem <= 0) return IFCI_OK;
    string_h_kernel<<<dim3(nitem, string_h_parts(h, nitem, 64)), 256, 0, s>>>(d_desc, d_items, string_binom());
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

// Threads of a block: one per determinant of a row, while that is at most 512
// (few blocks in all) or 256.  With 128 threads a CAS(6e,13o) row of 286 takes
// its first warp three times round, the chain of dependent FMAs three times as
// long: 455 us against 253 us for the sigma of its 286 blocks.
static int threads64(ifci_handle_t h, int nstr, int nitem) {
    const int most = nitem < 4 * device_sm_count(h->device) ? kMaxThreads64 : 256;
    return std::min(most, (nstr + 31) / 32 * 32);
}

// One problem, its descriptor passed by value (no copies to the device).
int run_sigma64_one(ifci_handle_t h, const SigmaProb &p, cudaStream_t s) {
    const int cap = cap64(&p, 1);
    static SmemOptIn opt;
    IFCI_CUDA_TRY(h, ensure_smem(opt, h->device, sigma64_one_kernel, cap * (int)sizeof(double)));
    ProfScope ps(h, s, PK_CONTRACT);
    sigma64_one_kernel<<<p.nstr, threads64(h, p.nstr, p.nstr), cap * sizeof(double), s>>>(p, cap);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

int run_sigma64(ifci_handle_t h, const SigmaPlan &plan, const SigmaWave &w, cudaStream_t s) {
    const int cap = cap64(plan.probs.data() + w.prob0, w.nprob);
    static SmemOptIn opt;
    IFCI_CUDA_TRY(h, ensure_smem(opt, h->device, sigma64_kernel, cap * (int)sizeof(double)));
    ProfScope ps(h, s, PK_CONTRACT);
    int nstr = 0;
    for (int i = w.prob0; i < w.prob0 + w.nprob; i++) nstr = std::max(nstr, plan.probs[i].nstr);
    sigma64_kernel<<<w.nitem, threads64(h, nstr, w.nitem), cap * sizeof(double), s>>>(plan.d_probs, plan.d_items + w.item0, cap);
    IFCI_LAUNCH_CHECK(h);
    return IFCI_OK;
}

}  // namespace ifci
