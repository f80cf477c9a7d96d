// Internal declarations of the GB300 ANN-potential library: device model
// constants, the cell grid, the context, and the launch wrappers of every
// kernel. Only the .cu files of this library include it.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>
#include <vector_types.h>

#include "aenet_gpu.h"
#include "cell_grid.cuh"

namespace aenet {

constexpr int kMaxSpecies = 8;
constexpr int kMaxD = 64;       // descriptor length handled by the 64-slot warp reduction
constexpr int kMaxWidth = 64;   // hidden-layer width limit
constexpr int kMaxLayers = 5;   // weight layers
constexpr int kMaxOrder = 31;

// Device error word bits (set by kernels, read by the host after a sync).
constexpr unsigned kErrNbCap = 1u;      // neighbour list overflow
constexpr unsigned kErrAngCap = 2u;     // angular list overflow
constexpr unsigned kErrOverlap = 4u;    // |d| < 1e-6 A
constexpr unsigned kErrNonfinite = 8u;  // non-finite coordinate
constexpr unsigned kErrType = 16u;      // species index out of range
constexpr unsigned kErrTimeout = 32u;   // a bounded in-kernel wait ran out

// Descriptor basis and species constants, passed by value to the kernels.
struct Basis {
    int n_species;
    int Kr, Ka, D;          // Kr = order_rad + 1, Ka = order_ang + 1, D = 2 (Kr + Ka)
    float rc_rad, rc_ang, rc_max;
    float type_weight[kMaxSpecies];
    float sh_b[7][7];       // Legendre coefficients of T_a (a, l <= 6): the angular form through spherical harmonics
};

// Network shape (per species identical), passed by value.
struct Net {
    int n_species;
    int n_layers;                  // weight layers
    int widths[kMaxLayers + 1];
    int n_params;                  // floats per species: W^1 b^1 W^2 b^2 ...
    int act_len;                   // sum of widths (activation storage per atom)
};

// One structure of a batch: its own cell grid inside a global cell index space
// (cells cell0 .. cell0 + ncell - 1) and its atoms (atom0 .. atom0 + natoms - 1
// in input order).
struct StructInfo {
    Grid g;
    int cell0, ncell, atom0, natoms;
    // the list build's CTAs of the structure are item0 .. item0 + ncell parts - 1: a cell
    // is divided into parts of about 24 atoms, since a small box is one cell of up to some
    // hundred atoms that see thousands of image-atoms (a solid of 250 atoms: 6,750)
    int item0, parts;
};

// Energy and virial partial rows of one evaluation (read by the MD reductions).
struct Partials {
    const double *epart = nullptr, *vpart = nullptr;
    int eparts = 0, vparts = 0;
};

// Capacities of the per-warp neighbour lists of the potential kernel, and the
// shape of the Verlet list (MD with a skin).
struct Caps {
    int nb;     // entries with r <= rc_max
    int ang;    // entries with r <= rc_ang
    int tile;   // staged neighbour-cell atoms per chunk (fused kernel)
    int vl_cap = 0;        // Verlet-list entries per atom (r <= rc_max + skin at the build, and kRowSlack)
    int vl_jbits = 0;      // bits of the sorted atom index in an entry; the rest: image-offset code
    float rc_list = 0.f;   // rc_max + skin
};

// Entries of a list row beyond those an atom may have: the list build keeps the atom
// itself and, by its rounding margin, now and then a pair just outside the cutoff. The
// kernel that reads the row drops both, so an atom with exactly caps.nb neighbours fits.
constexpr int kRowSlack = 8;
inline int row_cap(const Caps &k) { return k.nb + kRowSlack; }

struct Context {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int precision = AENET_FP32;
    bool fuse_network = true;      // BF16 forms: tensor-core network inside the fused kernel
    bool pdl = false;              // set while a chain of kernels without event records is enqueued (pdl.cuh)
    int eval_n = 0;                // atoms of the evaluation being set up (tc_fused_supported)
    bool batch_call = false;       // set during the batch entry points
    bool cell_search = false;      // set while an MD step with AENET_MD_LIST_OFF is enqueued
    bool pipeline = false;         // FP32 fused form: the pipelined kernel (one CTA of 16 warps per SM)
    Basis basis{};
    Net net{};
    std::vector<double> mass;      // [n_species], empty if none
    std::string err;

    // model on the device
    float *d_params = nullptr;     // [n_species * n_params] FP32
    float *d_shift = nullptr;      // [n_species * D]
    float *d_scale = nullptr;      // [n_species * D]
    uint16_t *d_wbf = nullptr;     // BF16 warp-MMA operand fragments (hi, lo) and biases, see ann_bf16.cu
    unsigned char *d_wtc = nullptr;  // tcgen05 B operands and biases per species, see ann_tcgen05.cu
    size_t wbf_elems = 0;
    double *d_mass = nullptr;      // [n_species]

    // work buffers (grown on demand)
    int cap_atoms = 0;
    int cap_cells = 0;
    int cap_blocks = 0;
    float4 *d_pos4 = nullptr;      // sorted cell-local coordinates, .w = species (int bits)
    float4 *d_tmp4 = nullptr;      // same, input order
    int *d_perm = nullptr;         // sorted slot -> input index
    int *d_cell_of = nullptr;      // input index -> cell
    int *d_slot = nullptr;         // input index -> rank inside its cell
    int *d_cell_count = nullptr;   // [ncell]
    int *d_cell_start = nullptr;   // [ncell + 1]
    float *d_G = nullptr;          // [n * D] sorted order (descriptor calls and the split path)
    size_t cap_G = 0;
    float *d_dEdG = nullptr;       // [n * D] sorted order (split path)
    size_t cap_dEdG = 0;
    float *d_eatom = nullptr;      // [n] sorted order
    float4 *d_F4 = nullptr;        // [n] force accumulators, sorted order
    double *d_vir_part = nullptr;  // [cells * 9]
    double *d_e_part = nullptr;    // [blocks]
    double *d_ke_part = nullptr;   // [MD CTAs * 11] per-CTA energy, virial and kinetic-energy sums
    double *d_result = nullptr;    // [10]: energy, virial[9]
    double *h_res = nullptr;       // mapped host memory [12]: energy, virial[9], -, error word
    // mapped host memory for the arrays of small calls made with host pointers: the
    // kernels read positions and species from it and write forces and E_i to it
    unsigned char *h_stage = nullptr;
    size_t cap_hstage = 0;
    bool err_stale = false;        // the error word may hold an asynchronous call's error
    unsigned *d_err = nullptr;     // device error word
    unsigned long long *d_stats = nullptr;  // [4] radial entries, angular entries, angular pairs
    int *d_step = nullptr;         // MD record counter
    unsigned *d_done = nullptr;    // last-CTA counter of the MD reduction (left at 0)

    // per-atom activation records for dE/dW (optional)
    bool keep_act = false;
    bool act_valid = false;        // records of the last evaluation are in d_act
    int act_atoms = 0;             // atoms of that evaluation
    int cap_act = 0;
    float *d_act = nullptr;        // [n * rec_len] sorted order
    float *d_wpart = nullptr;      // dE/dW partial sums per (species, chunk)
    size_t cap_wpart = 0;
    int2 *d_wpairs = nullptr;      // [n_params] record indices of each weight's factors
    double *d_dEdW = nullptr;      // [n_species * n_params]

    // species grouping of the BF16 network kernel
    int *d_sp_cnt = nullptr;       // [kMaxSpecies], kept at 0 between evaluations
    int *d_sp_off = nullptr;       // [kMaxSpecies]
    int *d_sp_rank = nullptr;      // [n]
    int *d_sp_list = nullptr;      // [n] sorted indices grouped by species
    int cap_sp = 0;

    // staging of host arrays
    int cap_stage = 0;
    double *d_pos = nullptr, *d_vel = nullptr, *d_forces = nullptr, *d_eatom_out = nullptr;
    int32_t *d_types = nullptr;
    int cap_rec = 0;
    double *d_rec = nullptr;       // [2 * cap_rec] e_pot, e_kin records

    Caps caps{};

    // batched evaluation: per-structure grids (device), valid during a batch call
    int cap_struct = 0;
    StructInfo *d_sinfo = nullptr;     // [n_struct]
    double *d_bres = nullptr;          // [n_struct * 10]: energy, virial[9]
    const StructInfo *batch_sinfo = nullptr;  // non-NULL while a batch is enqueued
    int batch_n = 0;
    int batch_items = 0;               // CTAs of its list build

    // Verlet neighbour list with a skin (MD steps of the fused FP32 form; skin 0 =
    // the cell list every step). Entries: sorted index | image-offset code << jbits,
    // built by k_list_build (code rows), rebuilt inside the captured step (a graph
    // conditional node) whenever an atom moved more than skin/2 since the build.
    double skin = 0.0;
    // MD steps without a skin: AENET_MD_LIST_AUTO (0), _OFF (1: the fused kernel searches the cells
    // itself) or _ON (2: the exact list is built in every step and the list kernel evaluates it)
    int md_list = 0;
    int md_path = 0;                   // AENET_PATH_* flags of the captured MD step
    // tilt factors xy, xz, yz of the restricted triclinic cell of single-structure
    // calls (zero: orthorhombic)
    double tilt[3] = {0.0, 0.0, 0.0};
    int cap_vl_atoms = 0;
    long long cap_vl_entries = 0;
    int *d_vl = nullptr;               // [atoms * vl_cap] sorted order
    int *d_vl_count = nullptr;         // [atoms]
    double *d_vl_origin = nullptr;     // [atoms * 3] origin of atom i's FP32 coordinates (input order)
    double *d_vl_ref = nullptr;        // [atoms * 3] positions at the last build (input order)
    unsigned *d_vl_flag = nullptr;     // [2]: rebuild flag, last-CTA counter
    unsigned long long *d_vl_builds = nullptr;  // list builds so far
    // neighbour lists built for every evaluation (direct rows: displacement, index and species)
    float4 *d_rows = nullptr;          // [atoms of a slice * row_cap(caps)]
    size_t cap_rows = 0;
    int *d_list_count = nullptr;       // [atoms]
    int cap_list = 0;
    float *d_pnet = nullptr;           // network parameters packed in the list kernel's layout
    float *d_vir_atom = nullptr;       // [atoms * 6] virial of every atom (batches)
    int cap_vir_atom = 0;
    int cap_parts = 0;
    double *d_vl_epart = nullptr;      // [SMs * slices] energy partials of the list kernel
    double *d_vl_vpart = nullptr;      // [SMs * slices * 9] virial partials
    bool vl_valid = false;             // list, origins and cell maps describe the MD state
    cudaStream_t aux_stream = nullptr; // captures the body of the rebuild conditional
    int maps_n = -1;                   // atoms of the evaluation that last wrote the cell maps
    // partials of the last potential evaluation, and those that the captured MD step writes: a
    // replay makes them the last again (frame 0 of its call may have taken another form)
    Partials last, md_last;

    // Berendsen thermostat of the MD path (tau <= 0: NVE). d_lambda holds the
    // velocity scale of the next step, written by the closing kick.
    double thermo_T0 = 0.0, thermo_tau = 0.0, thermo_dt = 0.0;
    double *d_lambda = nullptr;
    bool lambda_valid = false;         // d_lambda was computed with the current settings

    // Berendsen barostat of the MD path (baro_every 0: off): after every
    // baro_every-th step of a call, positions and cell scaled by
    // mu = (1 - (baro_every dt / baro_tau) (baro_P0 - P) / baro_modulus)^(1/3).
    double baro_P0 = 0.0, baro_tau = 0.0, baro_modulus = 0.0;  // bar, ps, bar
    int baro_every = 0;
    double md_box[3] = {0.0, 0.0, 0.0};  // edges of the cell after the last MD call
    bool md_box_valid = false;

    // Generation of the work buffers: bumped whenever one is reallocated, so a
    // captured graph (which holds their addresses) knows it must be re-captured.
    unsigned buf_gen = 0;

    // persistent form of the potential kernel (used by the batched evaluation)
    int n_sm = 0;                      // SMs of the device
    bool persist = false;              // CTAs take cells from a global counter (batches only)
    int persist_ctas = 0;              // CTAs of the persistent launch (0 = all resident)
    unsigned *d_work = nullptr;        // [2] item counter, exit counter (each launch leaves both 0)
    const int *batch_order = nullptr;  // cell order of the batch being enqueued, heaviest first
    int *d_order = nullptr;            // [cap_order] that order for aenet_compute_batch
    int cap_order = 0;
    int last_grid = 0;                 // CTAs of the last potential launch
    bool last_pipe = false;            // the last fused FP32 launch was the pipelined form
    // set while an MD step is enqueued: its kick + drift kernel has already cleared the force
    // accumulators and the neighbour statistics, so the potential launch needs no memset
    bool md_prezeroed = false;
    int pot_parts = 0;                 // energy / virial partial rows of the last potential launch

    // prepared batch (aenet_batch_prepare): its own layout buffers, the tuned
    // launch and the captured evaluation
    cudaGraphExec_t batch_exec = nullptr;
    StructInfo *d_psinfo = nullptr;    // [n_struct]
    int *d_porder = nullptr;           // [total_cells]
    struct {
        bool valid = false;
        int n_struct = 0, n_atoms = 0, total_cells = 0;
        Grid gall{};
        const double *pos = nullptr;
        const int32_t *types = nullptr;
        double *energies = nullptr, *forces = nullptr, *virials = nullptr;
        bool persist = false;
        int tile = 0, ctas = 0, kernels = 0;
        float ms = 0.f;
        Caps caps{};
        unsigned gen = 0;
        cudaStream_t stream = nullptr;
    } plan;
    std::vector<StructInfo> plan_layout;  // host copy of the prepared layout
    std::vector<int> plan_order;

    // captured MD step (kick + drift + binning ... closing kick), and the part of a
    // call between two drifts (sort, potential, k_md_turn), each with what it was
    // captured for
    struct MdKey {
        int n = -1;
        double *pos = nullptr, *vel = nullptr;
        const int32_t *types = nullptr;
        double box[3] = {0, 0, 0};
        double dt = 0;
        double *rec = nullptr;
        cudaStream_t stream = nullptr;
        int nb = 0, ang = 0, tile = 0, vl_cap = 0;
        unsigned gen = 0;
        double skin = 0.0;
        unsigned ev_mask = 0;
        double thermo_T0 = 0.0, thermo_tau = 0.0;
        bool operator==(const MdKey &o) const {
            return n == o.n && pos == o.pos && vel == o.vel && types == o.types && box[0] == o.box[0] &&
                   box[1] == o.box[1] && box[2] == o.box[2] && dt == o.dt && rec == o.rec && stream == o.stream &&
                   nb == o.nb && ang == o.ang && tile == o.tile && vl_cap == o.vl_cap && gen == o.gen &&
                   skin == o.skin && ev_mask == o.ev_mask && thermo_T0 == o.thermo_T0 &&
                   thermo_tau == o.thermo_tau;
        }
    };
    cudaGraphExec_t md_exec = nullptr, turn_exec = nullptr;
    MdKey md_key, turn_key;
    unsigned ev_mask = 0;              // stage events recorded while an MD step is captured

    // stage timing of the captured MD step (events recorded inside the graph)
    static constexpr int kStages = 6;  // kick+drift+bin, sort, descriptor, network, forces, kick+reductions
    cudaEvent_t ev[kStages + 1] = {};
    int md_kernels = 0;                // kernel nodes in the captured step
};

// Allow a kernel the device's largest dynamic shared memory. Launches of one
// kernel with different sizes (captured graphs among them) then never depend on
// which size was set last; each launcher still checks its own size.
template <class K>
inline cudaError_t allow_max_smem(K kern) {
    int dev = 0, optin = 0;
    cudaFuncAttributes fa{};
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);  // static shared memory counts against the limit
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 optin - (int)fa.sharedSizeBytes);
    return e;
}

// ---------------------------------------------------------------- launchers
// All launchers enqueue on ctx.stream and return the launch status.

// Wrap, bin and sort atoms by cell (the periodic cell list).
cudaError_t launch_cells(Context &c, const Grid &g, int n, const double *pos, const int32_t *types);
// The scan + scatter half of launch_cells (after the counts are in place).
cudaError_t launch_scan(Context &c, const Grid &g);  // cell counts -> cell starts (k_scan_cells)
cudaError_t launch_scatter(Context &c, int n);  // the sort after a binning kernel that also scanned
cudaError_t launch_sort(Context &c, const Grid &g, int n);
// Binning of a batch: every atom into the cell grid of its structure.
cudaError_t launch_cells_batch(Context &c, int n, int total_cells, const double *pos, const int32_t *types);
// Per-structure energy (FP64 sum of E_i) and virial (FP64 sum of cell partials)
// into c.d_bres rows, or (when given) straight into energies[S], virials[S*9].
// The virials come from the cells' partial rows, or with atoms from every atom's
// (c.d_vir_atom, the list kernel).
cudaError_t launch_batch_reduce(Context &c, bool atoms, double *energies = nullptr, double *virials = nullptr);

// Per-species networks: E_i and dE/dG_i (Sec. II.A, Eq. ANN-layer), energy block partials.
cudaError_t launch_ann(Context &c, int n);

// Energy and virial reductions (E = sum_i E_i, Sec. II.A) over n_eparts energy partials and the
// virial partials of the last evaluation, and outputs in input order (each or NULL); to_host:
// energy, virial and the error word also to c.h_res.
cudaError_t launch_finalize(Context &c, int n, int n_eparts, double *forces, double *e_atom, double *energy,
                            double *virial, bool to_host);

// BF16 tensor-core networks (precision forms; two hidden layers <= 32).
bool bf16_supported(const Net &net);
// The three-kernel path's network kernel: tcgen05 (TMEM accumulators) over
// 128-atom species tiles. Energy partials: one per CTA.
int tcgen05_tiles(const Context &c, int n);
int tcgen05_eparts(const Context &c, int n);
cudaError_t launch_ann_tcgen05(Context &c, int n);
// Its weights, packed into the B-operand layout (c.d_wtc) from c.d_params.
cudaError_t pack_tcgen05_weights(Context &c);

// Length of the per-atom activation record (g, then x_l and delta_l per hidden layer).
int activation_record_len(const Net &net);
// Group the sorted atoms by species (d_sp_list, d_sp_off).
cudaError_t launch_species_group(Context &c, int n);
// dE/dW and dE/db of every species from the activation records (FP64 result in d_dEdW).
cudaError_t launch_grad_weights(Context &c, int n);
std::vector<int2> grad_pairs(const Net &net);
int grad_max_params();

// Work items per cell of a single-structure potential launch (persistent CTAs
// take cell parts from a counter); partial buffers hold kMaxSplit rows per cell.
constexpr int kMaxSplit = 4;
int potential_split(const Context &c, const Grid &g, int *split_from, int wave = 0);
bool pipe_supported(const Context &c, const Grid &g);

// Fused descriptor + network + forces kernel (FP32 form, hidden widths <= 32).
bool fused_supported(const Context &c);
cudaError_t launch_fused_potential(Context &c, const Grid &g, int n);
// Fused kernel with the networks on the tensor cores (BF16 forms; two hidden
// layers <= 32 wide; the water (16, 8) and solid (20, 6) bases), unless the context
// asked for the three-kernel path (AENET_OPT_FUSED_NETWORK 0): the form, and
// whether the evaluation of c.eval_n atoms takes it (at most kTcFusedAtoms or
// kTcFusedAtomsSolid; more take the three kernels).
bool tc_fused_form(const Context &c);
bool tc_fused_supported(const Context &c);
cudaError_t launch_fused_tc(Context &c, const Grid &g, int n);
// Either fused form: descriptor, networks and forces in one kernel.
inline bool fused_path(const Context &c) { return fused_supported(c) || tc_fused_supported(c); }
// Atoms up to which the BF16 forms run the networks inside the potential kernel:
// its one launch wins where launches count, the three kernels over neighbour lists
// where the chip is full. Split BF16, one evaluation, fused against three kernels
// (us): water 1,536 77 / 103, 3,072 121 / 124, 6,144 142 / 133, 12,288 188 / 160,
// 98,304 920 / 627, 331,776 2955 / 1929; device calls in a row, water 192 42 / 66,
// 384 82 / 75, 768 76 / 77, 1,536 55 / 75, 3,072 89 / 91, 4,095 105 / 102.
// The solid's cells hold more work per atom, and its fused time goes by how the
// cells fill the chip: 32 82 / 93, 64 97 / 85, 128 186 / 94, 256 481 / 116, 512 123 /
// 91, 700 162 / 99, 1,024 80 / 95, 2,000 189 / 135, 27,000 668 / 367. So its line is
// the largest size at which the fused form is known to win, not a crossover: between
// 64 and 1,000 atoms the three kernels (AENET_OPT_FUSED_NETWORK 0) are the faster.
constexpr int kTcFusedAtoms = 4096, kTcFusedAtomsSolid = 1024;
// Whether evaluations go over neighbour rows: the FP32 fused form, except (for one
// structure) the pipelined kernel and MD steps asked to search the cells in the
// fused kernel.
inline bool rows_form(const Context &c) {
    return fused_supported(c) && (c.batch_call || (!c.pipeline && !c.cell_search));
}
int ann_blocks(int n);

// Forces to input order (FP64) only.
cudaError_t launch_finalize_forces(Context &c, int n, double *forces);

// Descriptor rows to input order (float), and the error word to c.h_res[11].
cudaError_t launch_unsort_G(Context &c, int n, float *G);

// Velocity Verlet (the propagation step of the MD cycle, Fig. 1).
// One MD half: kick (v += dt/2 F/m c) + drift (x += dt v) fused with the binning
// of the new positions (integration and cell list); the scan and scatter follow.
cudaError_t launch_md_kick_drift_bin(Context &c, const Grid &g, int n, double dt, double *pos, double *vel,
                                     const int32_t *types);
// The closing kick (v += dt/2 F/m c) with the kinetic energy, fused with the
// FP64 reduction of energy, virial and kinetic energy (last-CTA pattern) into
// c.d_result and, when rec_pot != NULL, the record of step *c.d_step. The
// partials are those of the last potential evaluation (c.last_*). With
// clear_vl, the last CTA also counts a list build and clears the rebuild flag.
cudaError_t launch_md_kick_finish(Context &c, int n, double dt, double *vel, const int32_t *types,
                                  double *rec_pot, double *rec_kin, bool clear_vl = false);
// The closing kick and reduction of one step and the opening kick, drift and
// binning (with the scan) of the next in one kernel (NVE).
cudaError_t launch_md_turn(Context &c, const Grid &g, int n, double dt, double *pos, double *vel,
                           const int32_t *types, double *rec_pot, double *rec_kin);
// x *= mu for count doubles (the barostat's isotropic scaling of positions).
cudaError_t launch_scale(Context &c, double *x, long long count, double mu);

// Verlet form of the opening half-kick and drift (no binning): refresh the FP32
// coordinates relative to the origins of the last list build, raise the rebuild
// flag if an atom moved more than skin/2, and set the graph conditional.
cudaError_t launch_md_vl_kick_drift(Context &c, int n, double dt, double *pos, double *vel, const int32_t *types,
                                    cudaGraphConditionalHandle cond);
// Rebuild, part 1: bin the current positions, record each atom's origin and
// reference position (then launch_sort and launch_vl_build).
cudaError_t launch_md_vl_bin(Context &c, const Grid &g, int n, const double *pos, const int32_t *types);
// Rebuild, part 2: the Verlet list of every atom (k_list_build, code rows).
cudaError_t launch_vl_build(Context &c, const Grid &g, int n);
// The fused potential over the Verlet list (persistent CTAs, atoms from a
// counter); sets c.last_* to its partials.
cudaError_t launch_potential_list(Context &c, const Grid &g, int n);
// Largest CTA count of a list-kernel launch (sizes its partial buffers).
int potential_list_max_ctas(const Context &c);
// Evaluation over lists built for it, for the sorted atoms [a_lo, a_hi) (slices
// of list_slice(c, n) atoms): the list build (direct rows) and the list kernel.
// The first build also clears the forces and statistics when clear;
// the kernel appends its partial rows after *parts and sets c.last_*.
int list_slice(const Context &c, int n);
cudaError_t launch_rows_build(Context &c, const Grid &g, int n, int a_lo, int a_hi, bool clear);
// What the list kernel evaluates: everything, the G rows (c.d_G) only, or forces
// and virial from given dE/dG rows (c.d_dEdG).
enum class RowsMode { fused, descriptor, forces };
cudaError_t launch_rows_potential(Context &c, const Grid &g, RowsMode mode, int a_lo, int a_hi, int *parts);
// Network parameters into the list kernel's layout (c.d_pnet), on c.stream.
cudaError_t pack_list_net(Context &c);
// Dynamic shared memory of one list CTA of a single warp (what must fit).
size_t list_smem_bytes(const Context &c);

// Message reported by aenet_last_error(NULL) for calls made without a context.
void set_context_free_error(const char *msg);

// Dynamic shared memory bytes of the potential kernel in the context's mode.
size_t potential_smem_bytes(const Context &c, const Grid &g);
size_t ann_smem_bytes(const Context &c);

}  // namespace aenet
