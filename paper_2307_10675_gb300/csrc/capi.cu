// C entry points for single CI spaces: ifci_sigma and ifci_frozen_core.
#include <algorithm>

#include "hamiltonian.cuh"
#include "sigma.cuh"

namespace ifci {
int launch_convert_w(ifci_handle_t h, int nprob, const SigmaProb *d_probs, cudaStream_t s);
}

extern "C" {

int ifci_sigma(ifci_handle_t h, const ifci_strings_t *str, const double *h1, const double *eri, const double *c,
               double *sigma, int precision, ifci_stream_t stream) {
    using namespace ifci;
    if (!h) return IFCI_ERR_INVALID_ARG;
    if (!str || !h1 || !eri || !c || !sigma || !str->exc)
        return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_sigma: null argument");
    int nstr = 0, nexc = 0;
    if (ifci_string_counts(str->norb, str->nelec_spin, &nstr, &nexc) != IFCI_OK || nstr != str->nstr ||
        nexc != str->nexc || str->nelec_spin < 1)
        return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_sigma: inconsistent string table (norb=%d nelec=%d)",
                         str->norb, str->nelec_spin);
    if (c == sigma) return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_sigma: sigma aliases c");
    const bool sym_req = (precision & IFCI_SIGMA_SPIN_SYMMETRIC) != 0;
    precision &= ~IFCI_SIGMA_SPIN_SYMMETRIC;
    if (precision < IFCI_FP64 || precision > IFCI_FP64E)
        return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_sigma: precision %d", precision);
    const bool tc = precision == IFCI_BF16 || precision == IFCI_TF32;
    const bool oz = precision == IFCI_FP64E;
    if (tc && !tc_supported(precision))
        return set_error(h, IFCI_ERR_UNSUPPORTED, "ifci_sigma: precision %d not built", precision);
    IFCI_CUDA_TRY(h, cudaSetDevice(h->device));
    cudaStream_t s = as_cuda(stream);
    const int n = str->norb, np = n * (n + 1) / 2, ld = np;
    const long long ndet = (long long)nstr * nstr;

    if (precision == IFCI_FP64) {
        // string Hamiltonian, then one fused kernel; descriptors by value
        if (!sigma64_supported(np, nstr, nexc))
            return set_error(h, IFCI_ERR_OOM, "ifci_sigma: %d strings are beyond the shared memory of an SM", nstr);
        const int nnz = string_h_nnz(n, str->nelec_spin);
        IFCI_TRY(ws_reserve(h, ws_round((size_t)nnz * nstr * 8) + ws_round((size_t)nnz * nstr * 4)));
        double *hval = ws_take<double>(h, (size_t)nnz * nstr);
        int *hidx = ws_take<int>(h, (size_t)nnz * nstr);
        SigmaProb q{};
        q.n = n; q.nstr = nstr; q.nexc = nexc; q.np = np;
        q.ndet = ndet; q.stride = ndet; q.exc = str->exc; q.eri = eri;
        q.hval = hval; q.hidx = hidx; q.nnz = nnz;
        q.cbase = c; q.sbase = sigma;
        IFCI_TRY(launch_string_h(h, StringHDesc{n, str->nelec_spin, nstr, nnz, h1, eri, hval, hidx}, s));
        return run_sigma64_one(h, q, s);
    }
    SigmaPlan plan;
    SigmaProb p{};
    p.n = n; p.nstr = nstr; p.nexc = nexc; p.np = np; p.ld = ld;
    p.ndet = ndet; p.stride = ndet; p.exc = str->exc;
    p.cbase = c; p.sbase = sigma;
    const bool sym = sym_req && (tc || oz) && 2 * ndet < (1ll << 31);
    p.sym = sym ? 1 : 0;   // the pair map is placed below, before the plan is uploaded
    plan.probs.push_back(p);
    IFCI_TRY(plan_sigma(h, plan, sigma_elems(np, ndet), precision));   // one wave
    const size_t eb = sigma_elem_bytes(precision);
    const long long delems_D = oz ? plan.max_qelems : std::max(plan.max_delems, plan.max_qelems);
    const int ldj = oz ? oz_map_ld(nstr) : 0;
    size_t need = ws_round(sizeof(FoldDesc)) + ws_round((size_t)ld * ld * 8) + ws_round((size_t)ld * ld * 4) +
                  (tc ? ws_round((size_t)tc_operand_bytes(np, precision)) : 0) +
                  (oz ? ws_round((size_t)oz_operand_bytes(np)) + ws_round(8) : 0) +
                  (oz ? ws_round(oz_map_elems(np, nstr) * 2) : 0) + (tc ? ws_round((size_t)nstr * kBlk16Stride) : 0) +
                  (sym && tc ? ws_round((size_t)nstr * pmap_ld(np) * 4) : 0) + plan_device_bytes(plan) +
                  ws_round((size_t)delems_D * eb) + ws_round((size_t)plan.max_delems * eb);
    IFCI_TRY(ws_reserve(h, need));
    auto *fd = ws_take<FoldDesc>(h, 1);
    double *W = ws_take<double>(h, (size_t)ld * ld);
    float *Wf = ws_take<float>(h, (size_t)ld * ld);
    void *Wtc = tc ? (void *)ws_take<char>(h, tc_operand_bytes(np, precision)) : nullptr;
    char *Woz = oz ? ws_take<char>(h, oz_operand_bytes(np)) : nullptr;
    plan.probs[0].W = W;
    plan.probs[0].Wf = Wf;
    plan.probs[0].Wtc = Wtc;
    plan.probs[0].Woz = Woz;
    plan.probs[0].Wexp = oz ? (double *)(Woz + (oz_operand_bytes(np) - 256)) : nullptr;
    plan.probs[0].dscale = 2.0;
    uint16_t *jmap = oz ? ws_take<uint16_t>(h, oz_map_elems(np, nstr)) : nullptr;
    plan.probs[0].jmap = jmap;
    plan.probs[0].ldj = ldj;
    uint8_t *blk = tc ? ws_take<uint8_t>(h, (size_t)nstr * kBlk16Stride) : nullptr;
    plan.probs[0].blk = blk;
    int32_t *pmap = sym && tc ? ws_take<int32_t>(h, (size_t)nstr * pmap_ld(np)) : nullptr;
    plan.probs[0].pmap = pmap;
    FoldDesc f{n, 2 * str->nelec_spin, ld, h1, eri, W};
    void *D, *G;
    if (oz) {
        unsigned long long *mx = ws_take<unsigned long long>(h, 2);
        IFCI_TRY(upload_plan(h, plan, s));
        D = ws_take<char>(h, (size_t)delems_D * eb);
        G = ws_take<char>(h, (size_t)plan.max_delems * eb);
        if (!D || !G || !mx) return set_error(h, IFCI_ERR_OOM, "ifci_sigma: workspace");
        return run_sigma_oz_one(h, plan, f, c, jmap, mx, D, G, s);
    }
    IFCI_CUDA_TRY(h, cudaMemcpyAsync(fd, &f, sizeof(f), cudaMemcpyHostToDevice, s));
    IFCI_TRY(launch_fold(h, 1, fd, np, s));
    if (blk && !pmap) IFCI_TRY(launch_exc_blocks(h, nstr, nexc, str->exc, blk, s));
    if (pmap) IFCI_TRY(launch_pair_map(h, nstr, nexc, np, str->exc, pmap, s));
    IFCI_TRY(upload_plan(h, plan, s));
    if (precision == IFCI_FP32) IFCI_TRY(launch_convert_w(h, 1, plan.d_probs, s));
    if (tc) IFCI_TRY(launch_tc_pack_w(h, 1, plan.d_probs, precision, np, s));
    D = ws_take<char>(h, (size_t)delems_D * eb);
    G = ws_take<char>(h, (size_t)plan.max_delems * eb);
    if (!D || !G) return set_error(h, IFCI_ERR_OOM, "ifci_sigma: workspace");
    return run_sigma(h, plan, precision, D, G, s);
}

int ifci_frozen_core(ifci_handle_t h, const ifci_system_t *sys, int nx, const int *bodies, double *h1,
                     double *eri_x, double *e_core, ifci_stream_t stream) {
    using namespace ifci;
    if (!h) return IFCI_ERR_INVALID_ARG;
    if (!sys || !bodies || !h1 || !eri_x || !e_core || nx < 1 || nx > sys->nbody)
        return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_frozen_core: bad arguments");
    for (int i = 0; i < nx; i++)
        if (bodies[i] < 0 || bodies[i] >= sys->nbody || (i && bodies[i] <= bodies[i - 1]))
            return set_error(h, IFCI_ERR_INVALID_ARG, "ifci_frozen_core: bodies must be ascending and in range");
    IFCI_CUDA_TRY(h, cudaSetDevice(h->device));
    cudaStream_t s = as_cuda(stream);
    const int norb = sys->norb;
    const long long npg = (long long)norb * (norb + 1) / 2;
    std::vector<int> orbs;
    std::vector<char> inx(sys->nbody, 0);
    for (int i = 0; i < nx; i++) inx[bodies[i]] = 1;
    for (int b = 0; b < sys->nbody; b++)
        if (inx[b])
            for (int p = sys->body_offset[b]; p < sys->body_offset[b + 1]; p++) orbs.push_back(p);
    const int nA = (int)orbs.size();
    for (int b = 0; b < sys->nbody; b++)
        if (!inx[b]) orbs.push_back(sys->body_offset[b]);
    const int nC = (int)orbs.size() - nA;
    size_t need = ws_round(sizeof(FrozenDesc)) + ws_round(orbs.size() * sizeof(int)) + ws_round(8) +
                  (sys->on_host ? ws_round((size_t)norb * norb * 8) + ws_round((size_t)npg * npg * 8) : 0);
    IFCI_TRY(ws_reserve(h, need));
    auto *fd = ws_take<FrozenDesc>(h, 1);
    int *d_orbs = ws_take<int>(h, orbs.size());
    double *d_ec = ws_take<double>(h, 1);
    const double *dh = sys->h, *dV = sys->eri;
    if (sys->on_host) {
        double *th = ws_take<double>(h, (size_t)norb * norb);
        double *tV = ws_take<double>(h, (size_t)npg * npg);
        IFCI_CUDA_TRY(h, cudaMemcpyAsync(th, sys->h, (size_t)norb * norb * 8, cudaMemcpyHostToDevice, s));
        IFCI_CUDA_TRY(h, cudaMemcpyAsync(tV, sys->eri, (size_t)npg * npg * 8, cudaMemcpyHostToDevice, s));
        dh = th;
        dV = tV;
    }
    FrozenDesc f{nA, nC, 0, h1, eri_x, d_ec};
    IFCI_CUDA_TRY(h, cudaMemcpyAsync(fd, &f, sizeof(f), cudaMemcpyHostToDevice, s));
    IFCI_CUDA_TRY(h, cudaMemcpyAsync(d_orbs, orbs.data(), orbs.size() * sizeof(int), cudaMemcpyHostToDevice, s));
    IFCI_TRY(launch_frozen_core(h, 1, fd, d_orbs, dh, dV, norb, s));
    IFCI_CUDA_TRY(h, cudaMemcpyAsync(e_core, d_ec, 8, cudaMemcpyDeviceToHost, s));
    IFCI_CUDA_TRY(h, cudaStreamSynchronize(s));
    return IFCI_OK;
}

}  // extern "C"
