// Gradient of the iFCI energy with respect to the integrals (reverse mode of
// Eqs. 1-5): Hellmann–Feynman on every E_Y, summed with the expansion weights
//   E_iFCI = E_0 + sum_{|X|<=n} eps_X = (1 - sum_Y w_Y) E_0 + sum_Y w_Y E_Y,
//   w_Y = (-1)^(n-|Y|) C(N-|Y|-1, n-|Y|).
//
// Per body set Y with converged vector c (spin-flip-even, normalised):
//   D+[A][K] = <K|E+_A|c>                     (the gather of the sigma build)
//   M[A][B]  = sum_K D+[A][K] D+[B][K] = <c|E+_A E+_B|c>    (SYRK, split over K)
//   gamma+_A = sum_K c_K D+[A][K]             (an extra row of D+ holding c)
// so the packed active 2-RDM is Gamma+_AB = M[A][B] - sum_{pq in A, rs in B}
// delta_qr gamma_ps.  The frozen core enters through the chain rule of
// E_core and h1 (Coulomb and exchange with the core orbitals).  Contributions
// of all body sets are summed with FP64 atomics into dh and dV; dV is
// symmetrised at the end (the packed entries V[A][B] and V[B][A] are one
// parameter of the symmetric H).
#include <algorithm>
#include <cmath>
#include <map>

#include "dav_driver.cuh"
#include "hamiltonian.cuh"
#include "system.cuh"

namespace ifci {

namespace {

constexpr int kSyrkT = 16;          // SYRK output tile
constexpr int kSyrkChunk = 512;     // fewest determinants of a split-K chunk
constexpr int kSyrkJobsPerSm = 64;  // jobs a wave is cut into, about, if it has more determinants than that
constexpr int kSyrkWarps = 4, kSyrkPer = 4;             // warps of a block, tiles each keeps in registers
constexpr int kSyrkGroup = kSyrkWarps * kSyrkPer;       // tiles of one job
constexpr int kSyrkK = 16;          // determinants staged at a time
__host__ __device__ inline int syrk_side(int np) { return (np + 1 + kSyrkT - 1) / kSyrkT; }
__host__ __device__ inline int syrk_tiles(int np) { return syrk_side(np) * (syrk_side(np) + 1) / 2; }   // ta <= tb
__host__ __device__ inline int syrk_groups(int np) { return (syrk_tiles(np) + kSyrkGroup - 1) / kSyrkGroup; }

struct RdmProb {
    int n, np, nstr, nexc, nA, nC;
    long long ndet;
    const int32_t *exc;
    const double *c;        // converged vector
    const int *orbs;        // [active nA ..., core nC ...] global orbital indices
    double w;               // expansion weight x grad_out
    long long doff;         // element offset of this problem's (np+1) x ndet block of D+
    int chunk0, nchunk;     // split-K chunks of this problem in the partial buffer
    double *M;              // (np+1)^2 reduced moments
};

struct SyrkJob {
    int prob, chunk, group;
};

// D+[A][K] for A < np (merge of the sorted alpha/beta lists) and D+[np][K] = c_K
__global__ void __launch_bounds__(256) rdm_gather_kernel(const RdmProb *__restrict__ probs,
                                                         const WorkItem *__restrict__ items, double *__restrict__ D) {
    const WorkItem it = items[blockIdx.x];
    const RdmProb &p = probs[it.prob];
    const long long K = it.start + threadIdx.x;
    if (K >= p.ndet) return;
    const int nstr = p.nstr, nexc = p.nexc, np = p.np;
    const long long ndet = p.ndet;
    const int ka = (int)(K / nstr), kb = (int)(K % nstr);
    const double *c = p.c;
    const int32_t *ea = p.exc + (size_t)ka * nexc, *eb = p.exc + (size_t)kb * nexc;
    int ia = 0, ib = 0;
    int32_t xa = ea[0], xb = eb[0];
    int pa = exc_pair(xa), pb = exc_pair(xb);
    double *out = D + p.doff + K;
    for (int A = 0; A < np; A++) {
        double v = 0.0;
        if (pa == A) {
            v += exc_sign(xa) * c[(long long)exc_J(xa) * nstr + kb];
            if (++ia < nexc) { xa = ea[ia]; pa = exc_pair(xa); } else pa = -1;
        }
        if (pb == A) {
            v += exc_sign(xb) * c[(long long)ka * nstr + exc_J(xb)];
            if (++ib < nexc) { xb = eb[ib]; pb = exc_pair(xb); } else pb = -1;
        }
        out[(long long)A * ndet] = v;
    }
    out[(long long)np * ndet] = c[K];
}

// partial[job][tile][i][j] = sum_{K in chunk} D+[16 ta + i][K] D+[16 tb + j][K]
// for the 16 tiles (ta <= tb) of the job's group.  An SM sub-partition takes 64
// clocks per FP64 warp instruction, so the sum is bound by the FMAs issued, and
// by their even spread over the chip: 16 x 16 tiles compute 3,840 products per
// determinant for 79 rows (12,288 with 64 x 64 tiles, 3,160 needed), and chunks
// of 512 determinants make a job of half a millisecond at most (16 ms with
// 16,384, of which a gradient over 63 sets had fewer than two per SM).  The
// gradient of 63 sets up to CAS(6e,12o): 18.2 ms before, 1.6 ms.
__global__ void __launch_bounds__(32 * kSyrkWarps) rdm_syrk_kernel(const RdmProb *__restrict__ probs,
                                                                   const SyrkJob *__restrict__ jobs, int chunk,
                                                                   const double *__restrict__ D, double *__restrict__ part) {
    const SyrkJob jb = jobs[blockIdx.x];
    const RdmProb &p = probs[jb.prob];
    const int rows = p.np + 1, T = syrk_side(p.np), nt = syrk_tiles(p.np), ld = T * kSyrkT + 2;
    const long long ndet = p.ndet;
    const long long k0 = (long long)(jb.chunk - p.chunk0) * chunk, k1 = min(ndet, k0 + chunk);
    const double *Dp = D + p.doff;
    extern __shared__ double Ds[];   // [kSyrkK][ld]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // lane: 4 rows x 2 columns of each of its warp's tiles
    const int r0 = (lane >> 3) * 4, c0 = (lane & 7) * 2;
    int oa[kSyrkPer], ob[kSyrkPer];
    bool on[kSyrkPer];
#pragma unroll
    for (int u = 0; u < kSyrkPer; u++) {
        // neighbouring tiles go to different warps: a short group still uses all
        int t = jb.group * kSyrkGroup + u * kSyrkWarps + warp, ta = 0;
        on[u] = t < nt;
        if (!on[u]) t = 0;
        while (t >= T - ta) t -= T - ta++;
        oa[u] = ta * kSyrkT + r0;
        ob[u] = (ta + t) * kSyrkT + c0;
    }
    double acc[kSyrkPer][4][2];
#pragma unroll
    for (int u = 0; u < kSyrkPer; u++)
#pragma unroll
        for (int i = 0; i < 4; i++) acc[u][i][0] = acc[u][i][1] = 0.0;
    for (long long kk = k0; kk < k1; kk += kSyrkK) {
        __syncthreads();
        for (int e = threadIdx.x; e < T * kSyrkT * kSyrkK; e += 32 * kSyrkWarps) {
            const int k = e % kSyrkK, A = e / kSyrkK;
            Ds[k * ld + A] = A < rows && kk + k < k1 ? Dp[(long long)A * ndet + kk + k] : 0.0;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < kSyrkK; k++) {
            const double *d = Ds + k * ld;
#pragma unroll
            for (int u = 0; u < kSyrkPer; u++) {
                if (!on[u]) continue;
                const double b0 = d[ob[u]], b1 = d[ob[u] + 1];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const double a = d[oa[u] + i];
                    acc[u][i][0] = fma(a, b0, acc[u][i][0]);
                    acc[u][i][1] = fma(a, b1, acc[u][i][1]);
                }
            }
        }
    }
    double *out = part + (size_t)blockIdx.x * kSyrkGroup * kSyrkT * kSyrkT;
#pragma unroll
    for (int u = 0; u < kSyrkPer; u++)
        if (on[u])
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 2; j++)
                    out[(u * kSyrkWarps + warp) * kSyrkT * kSyrkT + (r0 + i) * kSyrkT + c0 + j] = acc[u][i][j];
}

// M = sum over the problem's chunks of the partial tiles (fixed order), symmetric
// fill; blocks (problem, part)
__global__ void rdm_reduce_kernel(const RdmProb *__restrict__ probs, const int *__restrict__ job0,
                                  const double *__restrict__ part) {
    const int pi = blockIdx.x;
    const RdmProb &p = probs[pi];
    const int rows = p.np + 1, T = syrk_side(p.np), ng = syrk_groups(p.np);
    for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < rows * rows; e += gridDim.y * blockDim.x) {
        const int A = e / rows, B = e % rows;
        const int a = min(A, B), b = max(A, B);
        const int ta = a / kSyrkT, tb = b / kSyrkT;
        const int t = ta * T - ta * (ta - 1) / 2 + (tb - ta);   // index of (ta, tb) among ta <= tb
        const double *src = part + ((size_t)job0[pi] + t / kSyrkGroup) * kSyrkGroup * kSyrkT * kSyrkT +
                            (size_t)(t % kSyrkGroup) * kSyrkT * kSyrkT + (a - ta * kSyrkT) * kSyrkT + (b - tb * kSyrkT);
        double s = 0.0;
        for (int ch = 0; ch < p.nchunk; ch++) s += src[(size_t)ch * ng * kSyrkGroup * kSyrkT * kSyrkT];
        p.M[e] = s;
    }
}

__device__ __forceinline__ int pair_local(int P, int Q) { return P >= Q ? P * (P + 1) / 2 + Q : Q * (Q + 1) / 2 + P; }

// Weighted contributions of one body set to dh (norb^2) and dV (npair_g^2).
__global__ void rdm_accum_kernel(const RdmProb *__restrict__ probs, int norb, double *__restrict__ dh,
                                 double *__restrict__ dV) {
    const RdmProb &p = probs[blockIdx.x];
    const int n = p.nA, nC = p.nC, np = p.np, rows = np + 1;
    const double w = p.w;
    if (w == 0.0) return;
    const long long npg = (long long)norb * (norb + 1) / 2;
    const int *act = p.orbs, *core = p.orbs + n;
    const double *M = p.M;
    auto gam = [&](int a, int b) -> double {   // active 1-RDM gamma_ab
        const double g = M[(long long)pair_local(a, b) * rows + np];
        return a == b ? g : 0.5 * g;
    };
    auto Vg = [&](int P, int Q, int R, int S) -> double * {
        return dV + (long long)pair_of(P, Q) * npg + pair_of(R, S);
    };
    // (i) one-electron: dh = gamma (active), 2 (core)
    for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
        const int a = t / n, b = t % n;
        atomicAdd(dh + (long long)act[a] * norb + act[b], w * gam(a, b));
    }
    for (int k = threadIdx.x; k < nC; k += blockDim.x) atomicAdd(dh + (long long)core[k] * norb + core[k], 2.0 * w);
    // (ii) active 2-RDM, packed: 1/2 (M[A][B] - sum_{pq in A, rs in B} d_qr gamma_ps)
    for (int t = threadIdx.x; t < np * np; t += blockDim.x) {
        const int A = t / np, B = t % np;
        int P = 0;
        while ((P + 1) * (P + 2) / 2 <= A) P++;
        const int Q = A - P * (P + 1) / 2;
        int R = 0;
        while ((R + 1) * (R + 2) / 2 <= B) R++;
        const int S = B - R * (R + 1) / 2;
        double corr = 0.0;
        const int pq[2][2] = {{P, Q}, {Q, P}}, rs[2][2] = {{R, S}, {S, R}};
        const int na = P == Q ? 1 : 2, nb = R == S ? 1 : 2;
        for (int u = 0; u < na; u++)
            for (int v = 0; v < nb; v++)
                if (pq[u][1] == rs[v][0]) corr += gam(pq[u][0], rs[v][1]);
        const double g2 = M[(long long)A * rows + B] - corr;
        atomicAdd(Vg(act[P], act[Q], act[R], act[S]), 0.5 * w * g2);
    }
    // (iii) h1 = h + sum_c [2 (pq|cc) - (pc|cq)]: Coulomb and exchange with the core
    for (int t = threadIdx.x; t < np * nC; t += blockDim.x) {
        const int A = t / nC, k = t % nC;
        int P = 0;
        while ((P + 1) * (P + 2) / 2 <= A) P++;
        const int Q = A - P * (P + 1) / 2;
        const double gplus = M[(long long)A * rows + np];
        atomicAdd(Vg(act[P], act[Q], core[k], core[k]), 2.0 * w * gplus);
    }
    for (int t = threadIdx.x; t < n * n * nC; t += blockDim.x) {
        const int a = t / (n * nC), b = (t / nC) % n, k = t % nC;
        atomicAdd(Vg(act[a], core[k], core[k], act[b]), -w * gam(a, b));
    }
    // (iv) E_core = sum_c 2 h_cc + sum_{c,d} [2 (cc|dd) - (cd|dc)]
    for (int t = threadIdx.x; t < nC * nC; t += blockDim.x) {
        const int k = t / nC, l = t % nC;
        atomicAdd(Vg(core[k], core[k], core[l], core[l]), 2.0 * w);
        atomicAdd(Vg(core[k], core[l], core[l], core[k]), -w);
    }
}

// E_0 terms with weight w0 over the bonding orbitals.
__global__ void rdm_reference_kernel(const int *__restrict__ bond, int nb, double w0, int norb, double *__restrict__ dh,
                                     double *__restrict__ dV) {
    const long long npg = (long long)norb * (norb + 1) / 2;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nb * nb; t += gridDim.x * blockDim.x) {
        const int k = t / nb, l = t % nb;
        const int c = bond[k], d = bond[l];
        if (k == l) atomicAdd(dh + (long long)c * norb + c, 2.0 * w0);
        atomicAdd(dV + (long long)pair_of(c, c) * npg + pair_of(d, d), 2.0 * w0);
        atomicAdd(dV + (long long)pair_of(c, d) * npg + pair_of(d, c), -w0);
    }
}

// dV <- (dV + dV^T) / 2
__global__ void rdm_symmetrise_kernel(long long npg, double *__restrict__ dV) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < npg * npg;
         t += (long long)gridDim.x * blockDim.x) {
        const long long A = t / npg, B = t % npg;
        if (A < B) {
            const double s = 0.5 * (dV[A * npg + B] + dV[B * npg + A]);
            dV[A * npg + B] = s;
            dV[B * npg + A] = s;
        }
    }
}

long long expansion_weight(int nbody, int k, int max_order) {
    // (-1)^(n-|Y|) C(N-|Y|-1, n-|Y|); a set of all N bodies has weight 1
    if (k == nbody) return 1;
    long long c = binom(nbody - k - 1, max_order - k);
    return ((max_order - k) & 1) ? -c : c;
}

// Determinants of a split-K chunk for problems [first, last): 512, which spreads
// small sets over the chip, while that makes at most 64 jobs per SM; then the
// least multiple of it that does.  A job leaves 32 KB of partial sums, which the
// reduction adds up one chunk after the other: with 512 throughout, CAS(8e,20o)
// held 10.5 GB of them next to 39.6 GB of rows and took 1,191 ms (1,067 ms so,
// 0.3 GB), CAS(8e,16o) 0.64 GB and 74.9 ms (0.32 GB, 70.7 ms).  A wave of up to
// 64 jobs per SM, such as 63 sets up to CAS(6e,12o), keeps 512.
int syrk_chunk(const std::vector<RdmProb> &probs, int first, int last, int sms) {
    long long jobs = 0;
    for (int x = first; x < last; x++) jobs += (probs[x].ndet + kSyrkChunk - 1) / kSyrkChunk * syrk_groups(probs[x].np);
    const long long most = (long long)kSyrkJobsPerSm * sms;
    return (int)(kSyrkChunk * std::max(1ll, (jobs + most - 1) / most));
}

}  // namespace

}  // namespace ifci

extern "C" int ifci_rdm_backward(ifci_handle_t h, const ifci_system_t *sys, int max_order,
                                 const ifci_davidson_opts_t *opts, double grad_out, double *dh, double *deri,
                                 int recompute_vectors, ifci_stream_t stream) {
    using namespace ifci;
    if (!h) return IFCI_ERR_INVALID_ARG;
    IFCI_TRY(validate_system(h, sys, max_order));
    if (!dh || !deri) return set_error(h, IFCI_ERR_INVALID_ARG, "rdm_backward: null output");
    if (opts && opts->hbci_max_rounds > 0)
        return set_error(h, IFCI_ERR_UNSUPPORTED, "rdm_backward: no gradient of the HBCI energy (its PT2 part)");
    IFCI_CUDA_TRY(h, cudaSetDevice(h->device));
    cudaStream_t s = as_cuda(stream);
    const int norb = sys->norb;
    const long long npg = (long long)norb * (norb + 1) / 2;
    bool have = h->kept.valid && h->kept.nbody == sys->nbody && h->kept.max_order == max_order &&
                h->kept.norb == norb &&
                std::equal(h->kept.body_offset.begin(), h->kept.body_offset.end(), sys->body_offset);
    if (!recompute_vectors && !have)
        return set_error(h, IFCI_ERR_INVALID_ARG, "rdm_backward: no kept vectors for this system (run "
                                                   "ifci_increments first or ask for recomputation)");
    if (recompute_vectors || !have) {
        long long ns = 0;
        ifci_num_subsets(sys->nbody, max_order, &ns);
        std::vector<double> eps(ns);
        double e0 = 0, et = 0;
        ifci_davidson_opts_t o;
        ifci_davidson_default_opts(&o);
        if (opts) o = *opts;
        if (o.refine < 0) o.refine = 1;   // the vectors must be kept
        IFCI_TRY(ifci_increments(h, sys, max_order, &o, &e0, nullptr, eps.data(), &et, nullptr, nullptr, stream));
    }
    SubsetPlan P;
    plan_subsets(sys, max_order, P);
    // expansion weights: closed form, or (screened expansion) the derivative of
    // the recursion of Eqs. 2-5 at the forward call's inclusion pattern; the
    // screened sets (no vector, weight 0) leave the plan
    std::vector<double> wts(P.subsets.size());
    std::vector<long long> kvec_off;
    {
        const bool scr = h->kept.screened && h->kept.included.size() == P.subsets.size();
        if (scr) wts = screened_weights(P, h->kept.included);
        else
            for (size_t x = 0; x < P.subsets.size(); x++)
                wts[x] = (double)expansion_weight(sys->nbody, (int)P.subsets[x].size(), max_order);
        SubsetPlan Q;
        Q.orbs = P.orbs;
        std::vector<double> w2;
        for (size_t x = 0; x < P.subsets.size(); x++) {
            if (scr && !h->kept.included[x]) continue;
            Q.subsets.push_back(P.subsets[x]);
            Q.nA.push_back(P.nA[x]);
            Q.nC.push_back(P.nC[x]);
            Q.orb_off.push_back(P.orb_off[x]);
            kvec_off.push_back(h->kept.vec_off[x]);
            w2.push_back(wts[x]);
        }
        P = std::move(Q);
        wts = std::move(w2);
    }
    const int ns = (int)P.subsets.size();

    // problems, D+ waves and split-K jobs
    std::vector<RdmProb> probs(ns);
    double wsum = 0.0;
    long long dtotal = 0, maxd = 0;
    for (int x = 0; x < ns; x++) {
        RdmProb &r = probs[x];
        r.n = P.nA[x];
        r.nC = P.nC[x];
        r.nA = r.n;
        r.np = r.n * (r.n + 1) / 2;
        const int m = (int)P.subsets[x].size();
        r.nstr = (int)binom(r.n, m);
        r.nexc = m * (r.n - m + 1);
        r.ndet = (long long)r.nstr * r.nstr;
        r.c = h->kept.vec + kvec_off[x];
        const double wy = wts[x];
        r.w = wy * grad_out;
        wsum += wy;
        const long long need = (long long)(r.np + 1) * r.ndet;
        maxd = std::max(maxd, need);
        dtotal += need;
    }
    const long long budget = std::max(maxd, std::min(dtotal, 1ll << 28));
    // string tables per class
    size_t need = ws_round(ns * sizeof(RdmProb)) + ws_round(P.orbs.size() * 4) + ws_round(sys->nbody * 4) +
                  ws_round((size_t)budget * 8);
    std::map<std::pair<int, int>, int> cls;
    size_t tab_bytes = 0;
    long long mtot = 0;
    for (int x = 0; x < ns; x++) {
        auto key = std::make_pair(probs[x].n, (int)P.subsets[x].size());
        if (!cls.count(key)) {
            cls[key] = 1;
            tab_bytes += ws_round((size_t)probs[x].nstr * 8) + ws_round((size_t)probs[x].nstr * probs[x].nexc * 4);
        }
        mtot += (long long)(probs[x].np + 1) * (probs[x].np + 1);
    }
    need += tab_bytes + ws_round((size_t)mtot * 8);
    // per-wave work lists and partials are sized for the largest wave below
    std::vector<std::pair<int, int>> waves;
    {
        int first = 0;
        long long acc = 0;
        for (int x = 0; x < ns; x++) {
            const long long d = (long long)(probs[x].np + 1) * probs[x].ndet;
            if (acc + d > budget && x > first) {
                waves.push_back({first, x});
                first = x;
                acc = 0;
            }
            acc += d;
        }
        waves.push_back({first, ns});
    }
    size_t wave_max = 0;
    for (auto &wv : waves) {
        long long items = 0, jobs = 0;
        const int chunk = syrk_chunk(probs, wv.first, wv.second, device_sm_count(h->device));
        for (int x = wv.first; x < wv.second; x++) {
            const long long nch = (probs[x].ndet + chunk - 1) / chunk;
            items += (probs[x].ndet + 255) / 256;
            jobs += nch * syrk_groups(probs[x].np);
        }
        wave_max = std::max(wave_max, ws_round(items * sizeof(WorkItem)) + ws_round(jobs * sizeof(SyrkJob)) +
                                          ws_round(jobs * kSyrkGroup * kSyrkT * kSyrkT * 8) + ws_round((wv.second - wv.first) * 4));
    }
    need += wave_max + 4096;
    IFCI_TRY(ws_reserve(h, need));
    auto *d_probs = ws_take<RdmProb>(h, ns);
    int *d_orbs = ws_take<int>(h, P.orbs.size());
    int *d_bond = ws_take<int>(h, sys->nbody);
    double *D = ws_take<double>(h, budget);
    double *Mall = ws_take<double>(h, mtot);
    if (!d_probs || !d_orbs || !d_bond || !D || !Mall) return set_error(h, IFCI_ERR_OOM, "rdm_backward: workspace");
    std::map<std::pair<int, int>, int32_t *> tables;
    for (int x = 0; x < ns; x++) {
        auto key = std::make_pair(probs[x].n, (int)P.subsets[x].size());
        if (!tables.count(key)) {
            uint64_t *st = ws_take<uint64_t>(h, probs[x].nstr);
            int32_t *ex = ws_take<int32_t>(h, (size_t)probs[x].nstr * probs[x].nexc);
            if (!st || !ex) return set_error(h, IFCI_ERR_OOM, "rdm_backward: workspace (strings)");
            IFCI_TRY(ifci_build_strings(h, key.first, key.second, st, ex, stream));
            tables[key] = ex;
        }
    }
    {
        long long moff = 0;
        for (int x = 0; x < ns; x++) {
            probs[x].exc = tables[{probs[x].n, (int)P.subsets[x].size()}];
            probs[x].orbs = d_orbs + P.orb_off[x];
            probs[x].M = Mall + moff;
            moff += (long long)(probs[x].np + 1) * (probs[x].np + 1);
        }
    }
    std::vector<int> bond(sys->nbody);
    for (int b = 0; b < sys->nbody; b++) bond[b] = sys->body_offset[b];
    IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_orbs, P.orbs.data(), P.orbs.size() * 4, cudaMemcpyHostToDevice, s));
    IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_bond, bond.data(), sys->nbody * 4, cudaMemcpyHostToDevice, s));
    IFCI_CUDA_TRY(h, cudaMemsetAsync(dh, 0, (size_t)norb * norb * 8, s));
    IFCI_CUDA_TRY(h, cudaMemsetAsync(deri, 0, (size_t)npg * npg * 8, s));
    const size_t mark = h->ws_top;
    for (auto &wv : waves) {
        h->ws_top = mark;
        std::vector<WorkItem> items;
        std::vector<SyrkJob> jobs;
        std::vector<int> job0;
        long long doff = 0;
        const int len = syrk_chunk(probs, wv.first, wv.second, device_sm_count(h->device));
        int chunk = 0, max_np = 0;
        for (int x = wv.first; x < wv.second; x++) {
            RdmProb &r = probs[x];
            r.doff = doff;
            doff += (long long)(r.np + 1) * r.ndet;
            for (long long s0 = 0; s0 < r.ndet; s0 += 256) items.push_back(WorkItem{x - wv.first, 0, s0});
            const int ng = syrk_groups(r.np);
            max_np = std::max(max_np, r.np);
            r.nchunk = (int)((r.ndet + len - 1) / len);
            r.chunk0 = chunk;
            job0.push_back((int)jobs.size());
            for (int ch = 0; ch < r.nchunk; ch++)
                for (int g = 0; g < ng; g++) jobs.push_back(SyrkJob{x - wv.first, chunk + ch, g});
            chunk += r.nchunk;
        }
        const int nw = wv.second - wv.first;
        auto *d_items = ws_take<WorkItem>(h, items.size());
        auto *d_jobs = ws_take<SyrkJob>(h, jobs.size());
        double *part = ws_take<double>(h, jobs.size() * kSyrkGroup * kSyrkT * kSyrkT);
        int *d_job0 = ws_take<int>(h, nw);
        if (!d_items || !d_jobs || !part || !d_job0) return set_error(h, IFCI_ERR_OOM, "rdm_backward: workspace (wave)");
        RdmProb *d_wp = d_probs + wv.first;
        IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_wp, probs.data() + wv.first, nw * sizeof(RdmProb), cudaMemcpyHostToDevice, s));
        IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_items, items.data(), items.size() * sizeof(WorkItem), cudaMemcpyHostToDevice, s));
        IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_jobs, jobs.data(), jobs.size() * sizeof(SyrkJob), cudaMemcpyHostToDevice, s));
        IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_job0, job0.data(), nw * 4, cudaMemcpyHostToDevice, s));
        rdm_gather_kernel<<<(int)items.size(), 256, 0, s>>>(d_wp, d_items, D);
        IFCI_LAUNCH_CHECK(h);
        const int smem = kSyrkK * (syrk_side(max_np) * kSyrkT + 2) * (int)sizeof(double);   // 64 KB at 496 pairs
        static SmemOptIn opt;
        IFCI_CUDA_TRY(h, ensure_smem(opt, h->device, rdm_syrk_kernel, smem));
        rdm_syrk_kernel<<<(int)jobs.size(), 32 * kSyrkWarps, smem, s>>>(d_wp, d_jobs, len, D, part);
        IFCI_LAUNCH_CHECK(h);
        rdm_reduce_kernel<<<dim3(nw, std::max(1, std::min(32, (max_np + 1) * (max_np + 1) / 256))), 256, 0, s>>>(d_wp, d_job0, part);
        IFCI_LAUNCH_CHECK(h);
        rdm_accum_kernel<<<nw, 256, 0, s>>>(d_wp, norb, dh, deri);
        IFCI_LAUNCH_CHECK(h);
        // the host vectors above are staged by cudaMemcpyAsync before it returns;
        // synchronise before the next wave reuses the workspace
        IFCI_CUDA_TRY(h, cudaStreamSynchronize(s));
    }
    const double w0 = (1.0 - wsum) * grad_out;
    rdm_reference_kernel<<<4, 256, 0, s>>>(d_bond, sys->nbody, w0, norb, dh, deri);
    IFCI_LAUNCH_CHECK(h);
    rdm_symmetrise_kernel<<<1024, 256, 0, s>>>(npg, deri);
    IFCI_LAUNCH_CHECK(h);
    IFCI_CUDA_TRY(h, cudaStreamSynchronize(s));
    return IFCI_OK;
}
