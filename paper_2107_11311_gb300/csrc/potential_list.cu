// Evaluation over neighbour lists: launch of the list build and of the
// list-driven potential (kernels in list_kernels.cuh).
#include <algorithm>

#include "list_kernels.cuh"

namespace aenet {
namespace {

using namespace detail;

// Direct rows of one slice of atoms are limited to this many bytes; more atoms are
// evaluated in slices (water: 441,000 atoms a slice; a slice's last atoms leave a
// few warps busy for about 10 us of its 1.5 ms).
constexpr size_t kMaxRowBytes = size_t(1) << 30;

// Staged image-atoms of a build CTA: 1.25 x the mean neighbourhood of a cell
// before the reach filter, which removes about a quarter of it in large boxes.
int build_tile(const Context &c, const Grid &g, int n) {
    const double want = 1.25 * n / std::max(1, g.ncell) * g.n_off + 64.0;
    return want > 2048.0 ? 2048 : std::max(128, ((int)want + 31) / 32 * 32);
}

cudaError_t launch_build(Context &c, const Grid &g, int n, int a_lo, int a_hi, bool codes, bool clear) {
    const int tile = c.batch_sinfo ? c.caps.tile : build_tile(c, g, n);  // (batches: the tuned tile)
    const size_t smem = make_build_layout(g.n_off, tile).total;
    // with few cells each is divided, so that the build does not leave most SMs
    // idle (a part restages the neighbourhood); a part has at least 4 atoms
    const double per_cell = (double)n / std::max(1, g.ncell);
    const int parts =
        std::max(1, std::min((4 * std::max(1, c.n_sm) + g.ncell - 1) / std::max(1, g.ncell), (int)(per_cell / 4.0)));
    const int ctas = c.batch_sinfo ? c.batch_items : g.ncell * parts;  // (a batch: parts of each structure's own)
    auto kern = c.batch_sinfo ? k_list_build<true, false> : codes ? k_list_build<false, true> : k_list_build<false, false>;
    cudaError_t e = allow_max_smem(kern);
    if (e != cudaSuccess) return e;
    return launch_after(
        c.pdl, kern, ctas, kBuildThreads, smem, c.stream, g, c.batch_sinfo, c.batch_n,
        codes ? c.caps.rc_list : c.basis.rc_max, tile, parts, a_lo, a_hi, c.d_pos4,
        c.d_cell_start, c.d_rows, c.d_vl, codes ? c.caps.vl_cap : row_cap(c.caps), c.caps.vl_jbits,
        codes ? c.d_vl_count : c.d_list_count, clear ? c.d_F4 : nullptr, clear ? c.d_stats : nullptr, c.d_err);
}

// Warps of a list CTA (one CTA per SM): as many as the atoms of an SM need, at
// least 8 (the parameters are staged by all of them), at most `most` and what
// shared memory holds; 0 if not even one fits. (MD of 1,536 atoms: 11 warps 48 us
// a step, 20 warps 58; of 12,288 atoms, 81 an SM: 20 warps 100 us, 17, which
// divide the atoms more evenly, 102.)
int list_warps(const Context &c, size_t fixed, size_t per_warp, int n, int most) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    const size_t room = optin > 4096 ? (size_t)optin - 4096 : 0;  // (less the kernel's static shared memory)
    if (room < fixed + per_warp) return 0;
    const int fit = (int)std::min<size_t>((room - fixed) / per_warp, (size_t)most);
    const int sm = std::max(1, c.n_sm);
    return std::max(1, std::min(fit, std::max(8, (n + sm - 1) / sm)));
}

template <int KRT, int KAT, bool EXACT>
FusedNet list_net(const Context &c) {
    return make_list_net<KRT, KAT>(c.net);
}

// What a launch of the list kernel computes, and over which rows.
struct ListLaunch {
    int mode = kFused;
    bool codes = false;
    int a_lo = 0, a_hi = 0;
    int part0 = 0;  // first partial row
};

template <int KRT, int KAT, bool EXACT>
cudaError_t launch_list(Context &c, const Grid &g, const ListLaunch &q, int *parts) {
    const bool fused = q.mode == kFused;
    const FusedNet net = fused ? list_net<KRT, KAT, EXACT>(c) : FusedNet{};
    constexpr int most = list_max_warps<KRT, KAT, EXACT>();
    constexpr bool sh = sh_angular<KRT, KAT, EXACT>();
    Caps caps = c.caps;
    if (!q.codes) caps.vl_cap = row_cap(caps);
    const ListLayout L = make_list_layout(q.codes ? g.n_off : 0, caps.nb, caps.ang, fused ? c.basis.n_species : 0,
                                          net.stride, sh, 1);
    const int n = q.a_hi - q.a_lo;
    const int nw = list_warps(c, L.warp_base, L.warp_bytes, n, most);
    if (nw <= 0) return cudaErrorInvalidConfiguration;
    const bool batch = c.batch_sinfo != nullptr;
    auto kern = k_potential_list<KRT, KAT, EXACT, kFused, 32, false, false>;
    if (q.mode == kDescriptor)
        kern = k_potential_list<KRT, KAT, EXACT, kDescriptor, 32, false, false>;
    else if (q.mode == kForces)
        kern = batch ? k_potential_list<KRT, KAT, EXACT, kForces, 32, false, true>
                     : k_potential_list<KRT, KAT, EXACT, kForces, 32, false, false>;
    else if (batch)
        kern = net.hb == 32 ? k_potential_list<KRT, KAT, EXACT, kFused, 32, false, true>
                            : k_potential_list<KRT, KAT, EXACT, kFused, 16, false, true>;
    else if (q.codes)
        kern = net.hb == 32 ? k_potential_list<KRT, KAT, EXACT, kFused, 32, true, false>
                            : k_potential_list<KRT, KAT, EXACT, kFused, 16, true, false>;
    else if (net.hb == 16)
        kern = k_potential_list<KRT, KAT, EXACT, kFused, 16, false, false>;
    cudaError_t e = allow_max_smem(kern);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min(c.n_sm, n));
    float *out = fused ? (c.keep_act ? c.d_act : nullptr) : c.d_G;  // activation records or G rows
    *parts = grid;
    return launch_after(
        c.pdl, kern, grid, nw * 32, L.warp_base + L.warp_bytes * nw, c.stream, c.basis, net, g, caps, q.a_lo, q.a_hi,
        c.d_pos4, c.d_rows, c.d_vl, q.codes ? c.d_vl_count : c.d_list_count, c.d_pnet, c.d_F4, c.d_eatom, out,
        c.d_dEdG, c.d_vl_epart + q.part0, c.d_vl_vpart + 9 * (size_t)q.part0, c.d_vir_atom, c.d_stats, c.d_err,
        c.d_work);
}

template <int KRT, int KAT, bool EXACT>
cudaError_t pack_net(Context &c) {
    const FusedNet net = list_net<KRT, KAT, EXACT>(c);
    const int total = c.basis.n_species * net.stride;
    if (!c.d_pnet) {
        const cudaError_t e = cudaMalloc(&c.d_pnet, sizeof(float) * (size_t)total);
        if (e != cudaSuccess) return e;
    }
    k_pack_list_net<KRT, KAT, EXACT><<<(total + 255) / 256, 256, 0, c.stream>>>(c.basis, net, c.d_params, c.d_shift,
                                                                               c.d_scale, c.d_pnet);
    return cudaGetLastError();
}

template <int KRT, int KAT, bool EXACT>
size_t list_smem(const Context &c) {
    return make_list_layout(0, c.caps.nb, c.caps.ang, c.basis.n_species, list_net<KRT, KAT, EXACT>(c).stride,
                            sh_angular<KRT, KAT, EXACT>(), 1)
        .total;
}

// The kernel form of a basis: the two exact forms, or the smallest bound.
#define AENET_BY_BASIS(c, FN, ...)                                                                   \
    ((c).basis.Kr == 17 && (c).basis.Ka == 9   ? FN<17, 9, true>(__VA_ARGS__)                        \
     : (c).basis.Kr == 21 && (c).basis.Ka == 7 ? FN<21, 7, true>(__VA_ARGS__)                        \
     : (c).basis.Kr <= 8 && (c).basis.Ka <= 6  ? FN<8, 6, false>(__VA_ARGS__)                        \
     : (c).basis.Kr <= 20 && (c).basis.Ka <= 12 ? FN<20, 12, false>(__VA_ARGS__)                     \
                                               : FN<24, 8, false>(__VA_ARGS__))

cudaError_t clear_sums(Context &c, int n) {
    cudaError_t e = cudaMemsetAsync(c.d_stats, 0, sizeof(unsigned long long) * 4, c.stream);
    if (e != cudaSuccess) return e;
    return cudaMemsetAsync(c.d_F4, 0, sizeof(float4) * (size_t)(n > 0 ? n : 1), c.stream);
}

}  // namespace

size_t list_smem_bytes(const Context &c) { return AENET_BY_BASIS(c, list_smem, c); }

// Atoms of one slice of direct rows.
int list_slice(const Context &c, int n) {
    const size_t most = std::max<size_t>(1, kMaxRowBytes / (sizeof(float4) * (size_t)std::max(1, row_cap(c.caps))));
    return (int)std::min<size_t>((size_t)std::max(1, n), most);
}

int potential_list_max_ctas(const Context &c) { return std::max(1, c.n_sm); }

cudaError_t pack_list_net(Context &c) { return AENET_BY_BASIS(c, pack_net, c); }

cudaError_t launch_rows_build(Context &c, const Grid &g, int n, int a_lo, int a_hi, bool clear) {
    // with one slice the build clears what the list kernel accumulates into; with
    // more, an earlier slice's forces already lie on a later slice's atoms
    const bool one = a_lo == 0 && a_hi >= n;
    cudaError_t e;
    if (clear && !one && a_lo == 0 && (e = clear_sums(c, n)) != cudaSuccess) return e;
    return launch_build(c, g, n, a_lo, a_hi, false, clear && one);
}

cudaError_t launch_rows_potential(Context &c, const Grid &g, RowsMode mode, int a_lo, int a_hi, int *parts) {
    ListLaunch q;
    q.mode = mode == RowsMode::descriptor ? kDescriptor : mode == RowsMode::forces ? kForces : kFused;
    q.a_lo = a_lo;
    q.a_hi = a_hi;
    q.part0 = *parts;
    int got = 0;
    const cudaError_t e = AENET_BY_BASIS(c, launch_list, c, g, q, &got);
    *parts += got;
    c.last.epart = c.d_vl_epart;
    c.last.vpart = c.d_vl_vpart;
    c.last.eparts = c.last.vparts = c.pot_parts = *parts;
    c.last_grid = got;
    return e;
}

cudaError_t launch_vl_build(Context &c, const Grid &g, int n) { return launch_build(c, g, n, 0, n, true, false); }

cudaError_t launch_potential_list(Context &c, const Grid &g, int n) {
    cudaError_t e;
    if (!c.md_prezeroed && (e = clear_sums(c, n)) != cudaSuccess) return e;
    ListLaunch q;
    q.codes = true;
    q.a_hi = n;
    int parts = 0;
    if ((e = AENET_BY_BASIS(c, launch_list, c, g, q, &parts)) != cudaSuccess) return e;
    c.last.epart = c.d_vl_epart;
    c.last.vpart = c.d_vl_vpart;
    c.last.eparts = c.last.vparts = parts;
    return cudaSuccess;
}

}  // namespace aenet
