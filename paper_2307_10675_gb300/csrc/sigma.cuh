// Batched sigma build: gather D = E+ c, contraction G = W D, scatter sigma = E+ G.
#pragma once
#include "common.cuh"

namespace ifci {

// One CI problem as seen by the sigma kernels.  The input vector is
// cbase + (*cslot) * stride and the output sbase + (*sslot) * stride, so a
// Davidson iteration can move its slots on the device.
struct SigmaProb {
    int n, nstr, nexc, np;   // active orbitals, strings, excitations per string, pairs
    int ld;                  // row stride of W (>= np)
    int sym;                 // 1: the vector is spin-flip symmetric (C = C^T); the tensor-core paths gather
                             // alpha excitations only and return S + S^T (set by plan_sigma; BF16 and TF32
                             // need pmap, FP64E jmap)
    long long ndet;
    long long stride;
    const int32_t *exc;      // [nstr * nexc] excitation table of (n, nelec_spin)
    const uint8_t *blk;      // [nstr * kBlk16Stride] entry offsets per 16-pair block (tensor-core paths)
    const int32_t *pmap;     // [nstr * pmap_ld(np)] dense pair map (spin-flip-symmetric gathers) or nullptr
    const double *W;         // [ld * ld] folded contraction matrix, FP64
    const float *Wf;         // [ld * ld] FP32 copy (FP32 path) or nullptr
    const void *Wtc;         // tensor-core operand image (BF16 path) or nullptr
    const void *Woz;         // sliced operand image of the FP64-emulating path or nullptr
    double *Wexp;            // its power-of-two scale
    double dscale;           // scale of the digits of c, a power of two above max |c| (twice that where sym; FP64E)
    const uint16_t *jmap;    // excitation map over the contracted pairs (FP64-emulating path) or nullptr
    int ldj;
    long long qoff;          // element offset of the quantised copies of c in their wave buffer
    // plain FP64 path: the integrals, and the string Hamiltonian (nnz elements per string)
    const double *eri;
    const double *hval;      // [nnz][nstr]
    const int *hidx;         // [nnz][nstr]
    int nnz;
    const double *cbase;
    double *sbase;
    const int *cslot;        // device slot index or nullptr (= 0)
    const int *sslot;        // device slot index or nullptr (= 0)
    const int *active;       // device flag or nullptr (= active)
    long long doff;          // element offset of this problem's D and G blocks in a wave
    // FP64-emulating sigma over a subset of the pairs (a sectored space, whose
    // H' has no integral joining two groups): the npc pairs act[0..npc) in
    // ascending order, and pinv[pair] = their index or -1.  act = nullptr:
    // every pair (npc = np).
    int npc;
    const int32_t *act;
    const int16_t *pinv;
    const uint8_t *kcnt;     // [nstr] active pairs each string has an excitation on (nullptr: nexc)
};

// D/G elements one problem takes in a wave (the quantised +-c copies of the
// symmetric tensor-core gathers share the D buffer and need 2 ndet)
inline long long sigma_elems(int np, long long ndet) { return (long long)(np < 2 ? 2 : np) * ndet; }

struct WorkItem {
    int prob;
    int sub;                 // GEMM: first output pair row of the tile; FP64E: pass, or column tile of the finish
    long long start;         // first determinant; FP64E: alpha string, or row tile of the finish
};

constexpr int kGatherChunk = 256;   // determinants per gather/scatter block
constexpr int kGemmTM = 64, kGemmTN = 64, kGemmTK = 16;

struct SigmaWave {
    int prob0, nprob;        // problems of the wave (consecutive in the plan)
    int item0, nitem;        // gather/scatter items
    int tile0, ntile;        // contraction tiles
    int tc0, ntc;            // tensor-core tiles (BF16/TF32) or FP64E items
    int nwide;               // FP64E items of problems with long excitation lists (after the ntc others)
    int nfin;                // FP64E: finish tiles, from tile0
    long long delems;        // D (and G) elements of the wave; FP64E: elements of S
    long long qelems;        // 8-byte elements of the quantised copies of c
};

// Host-side plan over a fixed problem set; device arrays live in caller memory.
struct SigmaPlan {
    std::vector<SigmaProb> probs;
    std::vector<SigmaWave> waves;
    std::vector<WorkItem> items, tiles, tctiles;
    long long max_delems = 0;
    long long max_qelems = 0;   // largest set of quantised copies of a wave (the D buffer of the tensor-core paths)
    bool any_sym = false;    // some problem uses the spin-flip-symmetric gathers
    SigmaProb *d_probs = nullptr;
    WorkItem *d_items = nullptr, *d_tiles = nullptr, *d_tctiles = nullptr;
};

// Splits probs into waves of at most `budget` D elements (FP64E: 8-byte
// elements of digit planes and S), each problem whole; one problem above the
// budget fails with IFCI_ERR_OOM (FP64E: takes a wave of its own).
int plan_sigma(ifci_handle_t h, SigmaPlan &plan, long long budget, int precision);
size_t plan_device_bytes(const SigmaPlan &plan);
// Copies the plan's descriptor arrays to device memory taken from the workspace.
int upload_plan(ifci_handle_t h, SigmaPlan &plan, cudaStream_t s);
// The same into device arrays the caller has already set in the plan.
int upload_plan_to(ifci_handle_t h, SigmaPlan &plan, cudaStream_t s);
// Launches every wave: D, G are device buffers of at least max_delems
// elements of the precision's storage type (8 B for FP64, 4 B otherwise);
// FP64E: max_qelems and max_delems elements of 8 B.
int run_sigma(ifci_handle_t h, const SigmaPlan &plan, int precision, void *D, void *G, cudaStream_t s);
size_t sigma_elem_bytes(int precision);

// plain FP64 sigma (sigma64.cu)
constexpr int kStringHChunk = 32;              // strings per block of the list build
struct StringHDesc {
    int n, m, nstr, nnz;
    const double *h1, *eri;
    double *val;             // [nnz][nstr] or nullptr
    int *idx;                // [nnz][nstr] or nullptr
};
int string_h_nnz(int n, int m);
bool sigma64_supported(int np, int nstr, int nexc);   // one excitation of every string fits an SM's shared memory
int launch_string_h(ifci_handle_t h, const StringHDesc &one, cudaStream_t s);
int launch_string_h_batch(ifci_handle_t h, const StringHDesc *d_desc, const WorkItem *d_items, int nitem, cudaStream_t s);
int run_sigma64_one(ifci_handle_t h, const SigmaProb &p, cudaStream_t s);
int run_sigma64(ifci_handle_t h, const SigmaPlan &plan, const SigmaWave &w, cudaStream_t s);

// FP64-accurate sigma on FP16 tensor cores (sigma_oz.cu)
int oz_operand_bytes(int np);                  // bytes of one problem's sliced W image (+ scale)
int oz_map_ld(int nstr);                       // strings a row of the excitation map holds
size_t oz_map_elems(int np, int nstr);         // 16-bit elements of an excitation map
// a sectored unit's map: its class's restricted to npc active pairs
struct OzMapDesc {
    int npc, ldj, nstr;
    const int32_t *act;
    const uint16_t *map;
    uint16_t *out;
    uint8_t *kcnt;           // [nstr] active pairs each string has an excitation on
};
int launch_oz_compact_maps(ifci_handle_t h, int n, const OzMapDesc *d_desc, cudaStream_t s);
long long oz_plane_elems(int nstr, bool sym);  // FP16 elements of the digit planes of one problem
bool oz_supported(int np, int nstr, int nexc);
bool oz_wide(int nexc);
int launch_oz_map(ifci_handle_t h, int nstr, int nexc, int np, const int32_t *exc, uint16_t *jmap, cudaStream_t s);
int launch_oz_pack_w(ifci_handle_t h, int nprob, const SigmaProb *d_probs, int max_np, cudaStream_t s);
int run_sigma_oz(ifci_handle_t h, const SigmaPlan &plan, const SigmaWave &w, void *D, void *G, cudaStream_t s);
// The one problem of a plan, from its integrals and the caller's vector: builds
// W, its image, the excitation map and the scales (mx: two words of scratch) too.
struct FoldDesc;
int run_sigma_oz_one(ifci_handle_t h, const SigmaPlan &plan, const FoldDesc &f, const double *c, uint16_t *jmap,
                     unsigned long long *mx, void *D, void *G, cudaStream_t s);

// tensor-core contraction (sigma_tc.cu)
int tc_supported(int precision);
int tc_operand_bytes(int np, int precision);   // bytes of one problem's W image
int launch_tc_pack_w(ifci_handle_t h, int nprob, const SigmaProb *d_probs, int precision, int max_np, cudaStream_t s);
int launch_tc_contract(ifci_handle_t h, const SigmaPlan &plan, const SigmaWave &w, int precision,
                       const void *D, void *G, cudaStream_t s);

}  // namespace ifci
