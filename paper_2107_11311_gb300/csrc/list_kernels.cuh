// Neighbour lists in global memory and the potential evaluated over them.
//
// k_list_build (one CTA per cell or cell part) finds every image-atom within
// the cutoff of each atom from the sorted cells and writes one list row per
// atom; k_potential_list (persistent CTAs, one warp per atom) reads the rows
// and runs descriptor (Sec. II.B), network (Sec. II.A) and chain rule. Between
// the two there is nothing to wait for inside a CTA: no staging tile, no block
// barrier, so the potential kernel holds only per-warp state.
//
// Two row formats. A direct row holds the displacement of every entry and its
// sorted index and species, float4 (dx, dy, dz, j | species << 28): it is used
// where the list is rebuilt for every evaluation, and needs no gather, no image
// table and no cell grid in the potential kernel (16 B per entry, streamed once
// out and once in). A code row holds 4-byte entries (j | image-offset code <<
// jbits) and serves the Verlet list with a skin, whose displacements change
// from step to step.
#pragma once

#include <type_traits>

#include "pdl.cuh"
#include "potential_kernels.cuh"

namespace aenet {

namespace {

using namespace detail;

constexpr int kEntryIndex = 0x0fffffff;  // sorted index of a list entry; the bits above: species

// ------------------------------------------------------------------ the build

constexpr int kBuildThreads = 128;
constexpr int kBuildAtoms = 3;  // atoms a warp tests every staged image-atom against

struct BuildLayout {
    size_t off_start, off_prefix, off_shift, s_pos, total;
};

__host__ __device__ inline BuildLayout make_build_layout(int n_off, int tile) {
    BuildLayout L{};
    size_t p = 0;
    L.off_start = p;
    p = align16(p + sizeof(int) * n_off);
    L.off_prefix = p;
    p = align16(p + sizeof(int) * (n_off + 1));
    L.off_shift = p;
    p = align16(p + sizeof(float4) * n_off);
    L.s_pos = p;
    p = align16(p + sizeof(float4) * tile);
    L.total = p;
    return L;
}

// One CTA: the list rows of the atoms of one cell (or of one of its `parts`
// consecutive ranges) that lie in the sorted range [a_lo, a_hi).
//  1. The neighbour cells' atoms, shifted into the cell's frame, go to shared
//     memory; in an orthorhombic box only those within the cutoff of the cell
//     itself (about 72% of a 27-cell neighbourhood). More than `tile` of them
//     are taken in chunks.
//  2. Each warp tests the staged atoms against three atoms at a time (whole
//     evaluation: water 12,288 atoms, two at 12 CTAs per SM 94 us, three at 10
//     91 us; water 98,304, four at 8 515 us, two at 12 507 us). With
//     t = |p|^2 - 2 p.u the test is t <= rc^2 - |u|^2, three FMAs per pair; its
//     rounding is covered by a margin (the potential kernel applies the exact
//     cutoff to the displacement). The atom itself passes the test and is
//     dropped there too (kRowSlack).
// It also clears the atoms' force accumulators and the neighbour statistics (F4
// and stats, when given).
template <bool BATCH, bool CODES>
__global__ void __launch_bounds__(kBuildThreads, 10)
    k_list_build(Grid g_one, const StructInfo *__restrict__ sinfo, int n_struct, float rc, int tile, int parts,
                 int a_lo, int a_hi, const float4 *pos4, const int *cell_start, float4 *__restrict__ rows,
                 int *__restrict__ codes, int cap, int jbits, int *__restrict__ count, float4 *__restrict__ F4,
                 unsigned long long *__restrict__ stats, unsigned *__restrict__ err) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_kept, s_next;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    pdl_wait();
    if (stats && blockIdx.x == 0 && tid < 4) stats[tid] = 0ull;
    int cell, part, sidx = 0;
    if constexpr (BATCH) {  // the structure whose CTAs (cells x parts) this is one of
        int lo = 0, hi = n_struct - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (sinfo[mid].item0 <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        sidx = lo;
        parts = sinfo[sidx].parts;
        const int k = (int)blockIdx.x - sinfo[sidx].item0;
        cell = k / parts;
        part = k - cell * parts;
        cell += sinfo[sidx].cell0;
    } else {
        cell = blockIdx.x / parts;
        part = blockIdx.x - cell * parts;
    }
    int first = cell_start[cell], n = cell_start[cell + 1] - first;
    {
        const int lo = part * n / parts, hi = (part + 1) * n / parts;
        const int f0 = max(first + lo, a_lo), f1 = min(first + hi, a_hi);
        first = f0;
        n = f1 - f0;
    }
    if (n <= 0) return;

    const BuildLayout L = make_build_layout(g_one.n_off, tile);
    int *off_start = reinterpret_cast<int *>(smem + L.off_start);
    int *off_prefix = reinterpret_cast<int *>(smem + L.off_prefix);
    float4 *off_shift = reinterpret_cast<float4 *>(smem + L.off_shift);
    float4 *s_pos = reinterpret_cast<float4 *>(smem + L.s_pos);
    const Grid &g = BATCH ? sinfo[sidx].g : g_one;
    const int cell0 = BATCH ? sinfo[sidx].cell0 : 0;
    const int n_off = g.n_off;
    const int lcell = cell - cell0;
    const int cx = lcell % g.nc[0], cy = (lcell / g.nc[0]) % g.nc[1], cz = lcell / (g.nc[0] * g.nc[1]);
    const int wx = 2 * g.m[0] + 1, wy = 2 * g.m[1] + 1;
    for (int o = tid; o < n_off; o += kBuildThreads) {
        const int ox = o % wx - g.m[0], oy = (o / wx) % wy - g.m[1], oz = o / (wx * wy) - g.m[2];
        const int ux = cx + ox, uy = cy + oy, uz = cz + oz;
        const int vx = ux - floor_div(ux, g.nc[0]) * g.nc[0];
        const int vy = uy - floor_div(uy, g.nc[1]) * g.nc[1];
        const int vz = uz - floor_div(uz, g.nc[2]) * g.nc[2];
        const int nc = cell0 + (vz * g.nc[1] + vy) * g.nc[0] + vx;
        const int s0 = cell_start[nc];
        off_start[o] = s0;
        off_prefix[o] = cell_start[nc + 1] - s0;  // counts, scanned below
        off_shift[o] = make_float4(ox * g.hf[0] + oy * g.htf[0] + oz * g.htf[1], oy * g.hf[1] + oz * g.htf[2],
                                   oz * g.hf[2], 0.f);
    }
    __syncthreads();
    if (warp == 0) {
        int carry = 0;
        for (int base = 0; base < n_off; base += 32) {
            const int o = base + lane;
            const int v = o < n_off ? off_prefix[o] : 0;
            int x = v;
#pragma unroll
            for (int s = 1; s < 32; s <<= 1) {
                const int y = __shfl_up_sync(kFull, x, s);
                if (lane >= s) x += y;
            }
            if (o < n_off) off_prefix[o] = carry + x - v;
            carry += __shfl_sync(kFull, x, 31);
        }
        if (lane == 0) off_prefix[n_off] = carry;
    }
    if (tid == 0) s_kept = 0;
    __syncthreads();
    const int total = off_prefix[n_off];
    const float rc2 = rc * rc;
    const float rc2stage = rc2 * 1.00001f;  // pairs at the cutoff to the last ulp
    const bool filter = !g.tri;
    const int n_chunks = (total + tile - 1) / tile;
    for (int chunk = 0; chunk < n_chunks; ++chunk) {
        const int q1 = min(total, (chunk + 1) * tile);
        for (int q0 = chunk * tile; q0 < q1; q0 += kBuildThreads) {
            const int q = q0 + tid;
            bool keep = false;
            float4 sp = make_float4(0.f, 0.f, 0.f, 0.f);
            if (q < q1) {
                int lo = 0, hi = n_off - 1;  // largest o with off_prefix[o] <= q
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (off_prefix[mid] <= q) lo = mid; else hi = mid - 1;
                }
                const int j = off_start[lo] + (q - off_prefix[lo]);
                const float4 p = pos4[j], sh = off_shift[lo];
                const int bits = CODES ? (j | (lo << jbits)) : (j | (__float_as_int(p.w) << 28));
                sp = make_float4(p.x + sh.x, p.y + sh.y, p.z + sh.z, __int_as_float(bits));
                keep = true;
                if (filter) {
                    const float dx = fmaxf(fmaxf(-sp.x, sp.x - g.hf[0]), 0.f);
                    const float dy = fmaxf(fmaxf(-sp.y, sp.y - g.hf[1]), 0.f);
                    const float dz = fmaxf(fmaxf(-sp.z, sp.z - g.hf[2]), 0.f);
                    keep = dx * dx + dy * dy + dz * dz <= rc2stage;
                }
            }
            const unsigned mk = __ballot_sync(kFull, keep);
            int at = 0;
            if (lane == 0) at = atomicAdd(&s_kept, __popc(mk));
            at = __shfl_sync(kFull, at, 0) + __popc(mk & lt_mask);
            if (keep) s_pos[at] = sp;
        }
        if (tid == 0) s_next = 0;
        __syncthreads();
        const int len = s_kept;
        if (warp == 0 && (len & 31) && lane >= (len & 31)) s_pos[(len & ~31) + lane] = make_float4(1e15f, 0.f, 0.f, 0.f);
        __syncthreads();
        for (;;) {
            int a = 0;
            if (lane == 0) a = atomicAdd(&s_next, kBuildAtoms);
            a = __shfl_sync(kFull, a, 0);
            if (a >= n) break;
            float mx[kBuildAtoms], my[kBuildAtoms], mz[kBuildAtoms], lim[kBuildAtoms];  // -2u; rc^2 - |u|^2
            int cnt[kBuildAtoms];
            typename std::conditional<CODES, size_t, unsigned>::type row[kBuildAtoms];  // (a slice: < 2^26 entries)
#pragma unroll
            for (int b = 0; b < kBuildAtoms; ++b) {
                const int i = first + min(a + b, n - 1);
                row[b] = (decltype(row[b] + 0))(i - (CODES ? 0 : a_lo)) * cap;
                const float4 u = pos4[i];
                const float u2 = u.x * u.x + u.y * u.y + u.z * u.z, ur = sqrtf(u2) + rc;
                mx[b] = -2.f * u.x;
                my[b] = -2.f * u.y;
                mz[b] = -2.f * u.z;
                // |p| <= |u| + rc for an entry, so the sum's terms are at most 3 (|u| + rc)^2
                // and its rounding error is below 1e-6 of (|u| + rc)^2
                lim[b] = a + b < n ? rc2stage - u2 + 1e-6f * ur * ur : -3e38f;
                cnt[b] = chunk ? count[i] : 0;
            }
            __syncwarp();
            for (int base = 0; base < len; base += 32) {
                const int k = base + lane;
                const float4 p = s_pos[k];  // (the tile is padded to whole rounds with atoms out of reach)
                const float pp = p.x * p.x + p.y * p.y + p.z * p.z;
#pragma unroll
                for (int b = 0; b < kBuildAtoms; ++b) {
                    const float t = fmaf(p.x, mx[b], fmaf(p.y, my[b], fmaf(p.z, mz[b], pp)));
                    const bool in = t <= lim[b];
                    const unsigned m = __ballot_sync(kFull, in);
                    const int slot = cnt[b] + __popc(m & lt_mask);
                    if (in && slot < cap) {
                        if constexpr (CODES)
                            codes[row[b] + slot] = __float_as_int(p.w);
                        else
                            rows[row[b] + slot] = make_float4(fmaf(0.5f, mx[b], p.x), fmaf(0.5f, my[b], p.y),
                                                   fmaf(0.5f, mz[b], p.z), p.w);
                    }
                    cnt[b] += __popc(m);
                }
            }
#pragma unroll
            for (int b = 0; b < kBuildAtoms; ++b)
                if (a + b < n && lane == b) {
                    count[first + a + b] = min(cnt[b], cap);
                    if (cnt[b] > cap) atomicOr(err, kErrNbCap);
                    if (F4 && chunk == 0) F4[first + a + b] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
        }
        __syncthreads();  // the tile, s_kept and the counts are used again
        if (tid == 0) s_kept = 0;
        __syncthreads();
    }
}

// -------------------------------------------------------------- the potential

// Warps of a CTA (one CTA per SM): 20 at 96 registers for the pair form (water
// 98,304 atoms, whole evaluation: 521 us; 24 warps at 80 registers spill, 534 us;
// 16 at 128, 552 us), 16 at 128 for the spherical-harmonic form, whose
// accumulators need them (solid 27,000: 273 us; 12 warps, 287 us).
template <int KRT, int KAT, bool EXACT>
__host__ __device__ constexpr int list_max_warps() {
    return sh_angular<KRT, KAT, EXACT>() ? 16 : 20;
}

// Descriptor slots in the list kernel: [radial | angular | radial_w | angular_w]
// of widths KRT, KAT as in potential_kernels.cuh; a lane s < P = KRT + KAT holds
// slot s and its species-weighted copy s + P. NS = slots the layer-1 sums run
// over; the row stride of W1 is NS or NS + 4 floats, an odd multiple of 16 B, so
// that the 128-bit loads of eight lanes reading eight rows are free of bank
// conflicts.
template <int KRT, int KAT>
__host__ __device__ constexpr int list_inputs(int hb) {
    return hb == 16 ? (2 * (KRT + KAT) + 7) / 8 * 8 : (2 * (KRT + KAT) + 3) / 4 * 4;
}
template <int KRT, int KAT>
__host__ __device__ constexpr int list_w1_stride(int hb) {
    return (list_inputs<KRT, KAT>(hb) / 4) % 2 ? list_inputs<KRT, KAT>(hb) : list_inputs<KRT, KAT>(hb) + 4;
}

// G column of a lane's slot and of its weighted copy (-1 if unused).
template <int KRT, int KAT>
__device__ __forceinline__ int lane_col(int lane, int copy, int Kr, int Ka) {
    return lane < KRT + KAT ? slot_col<KRT, KAT>(lane + copy * (KRT + KAT), Kr, Ka) : -1;
}

// The FusedNet block of one species with the list kernel's W1 row stride.
template <int KRT, int KAT>
inline FusedNet make_list_net(const Net &net) {
    FusedNet f = make_fused_net(net);
    const int hb = f.hb, w1 = hb * list_w1_stride<KRT, KAT>(hb);
    const int d = w1 - hb * kW1Stride;  // only the first block's length differs
    for (int l = 1; l <= f.L; ++l) {
        if (l > 1) f.offW[l] += d;
        f.offB[l] += d;
    }
    f.offWL += d;
    f.offBL += d;
    f.offShift = (f.offShift + d + 3) & ~3;
    f.offScale = f.offShift + kSlots;
    f.stride = f.offScale + kSlots;
    return f;
}

// Every species' block packed in global memory (once per parameter set), so
// that a CTA copies it with 128-bit loads.
template <int KRT, int KAT, bool EXACT>
__global__ void k_pack_list_net(Basis B, FusedNet net, const float *__restrict__ params,
                                const float *__restrict__ shift, const float *__restrict__ scale,
                                float *__restrict__ out) {
    const int Kr = EXACT ? KRT : B.Kr, Ka = EXACT ? KAT : B.Ka, D = 2 * (Kr + Ka);
    const int hb = net.hb, w1s = list_w1_stride<KRT, KAT>(hb);
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < B.n_species * net.stride;
         idx += gridDim.x * blockDim.x) {
        const int t = idx / net.stride, p = idx - t * net.stride;
        const float *src = params + (size_t)t * net.n_params;
        float v = 0.f;
        if (p < net.offB[1]) {
            const int o = p / w1s, col = slot_col<KRT, KAT>(p - o * w1s, Kr, Ka);
            if (o < net.H[1] && col >= 0) v = src[net.srcOff[1] + o * D + col];
        } else if (p < net.offB[1] + hb) {
            const int o = p - net.offB[1];
            if (o < net.H[1]) v = src[net.srcOff[1] + net.H[1] * D + o];
        } else if (p >= net.offShift) {
            const bool sc = p >= net.offScale;
            const int col = slot_col<KRT, KAT>(p - (sc ? net.offScale : net.offShift), Kr, Ka);
            if (col >= 0) v = sc ? scale[t * D + col] : shift[t * D + col];
        } else if (p >= net.offBL) {
            if (p == net.offBL) v = src[net.srcOffL + net.Hlast];
        } else if (p >= net.offWL) {
            if (p - net.offWL < net.Hlast) v = src[net.srcOffL + p - net.offWL];
        } else {
#pragma unroll
            for (int l = 2; l < kMaxLayers; ++l) {
                if (l >= net.L || p < net.offW[l] || p >= net.offB[l] + hb) continue;
                const int Hi = net.H[l - 1], Ho = net.H[l];
                if (p < net.offB[l]) {
                    const int q = p - net.offW[l], o = q / (hb + 4), k = q - o * (hb + 4);
                    if (o < Ho && k < Hi) v = src[net.srcOff[l] + o * Hi + k];
                } else if (p - net.offB[l] < Ho) {
                    v = src[net.srcOff[l] + Ho * Hi + p - net.offB[l]];
                }
            }
        }
        out[idx] = v;
    }
}

constexpr int kRedStride = 20;  // floats per lane of the reduction buffer (5 x 16 B: conflict-free)

struct ListLayout {
    size_t params, off_shift, warp_base, warp_bytes, total;
    size_t e_d, e_j, a_u, a_s, red, coef, sh;  // inside a warp region
};

__host__ __device__ inline ListLayout make_list_layout(int n_off, int nb, int ang, int n_species, int stride, bool sh,
                                                       int nw) {
    ListLayout L{};
    size_t p = 0;
    L.off_shift = p;  // code rows only
    p = align16(p + sizeof(float4) * n_off);
    L.params = p;
    p = align16(p + sizeof(float) * (size_t)n_species * stride);
    L.warp_base = p;
    size_t q = 0;
    L.e_d = q;  // (dx, dy, dz, r): angular entries from the front, the others from the back
    q = align16(q + sizeof(float4) * nb);
    L.e_j = q;
    q = align16(q + sizeof(int) * nb);
    L.a_u = q;  // angular entries: (u, f_c); the pair form repeats the first ones after the last
    q = align16(q + sizeof(float4) * (ang + (sh ? 0 : 20)));
    L.a_s = q;  // their species weights
    q = align16(q + sizeof(float) * (ang + (sh ? 0 : 20)));
    L.red = q;  // reduction buffer; later dE/du sums of the angular entries (float4 each)
    const size_t red = sizeof(float) * 32 * kRedStride, grad = sizeof(float4) * ang;
    q = align16(q + (red > grad ? red : grad));
    L.coef = q;  // network inputs, then the coefficient pairs (a, a_w) of every order (64 floats)
    q = align16(q + sizeof(float2) * 32);
    L.sh = q;  // component sums and coefficients of the spherical-harmonic form
    if (sh) q = align16(q + sizeof(float) * kShScratch);
    L.warp_bytes = q;
    L.total = p + q * nw;
    return L;
}

// |d|^2 (one rounding order wherever r and 1/r are derived from it)
__device__ __forceinline__ float length2(float x, float y, float z) { return fmaf(z, z, fmaf(x, x, y * y)); }

struct ListWarp {
    float4 *e_d, *a_u, *a_g;
    float *a_s, *red, *coef, *sh;
    int *e_j;
};

// Entry k of round r of the main list: rounds 0 .. nra-1 hold the angular
// entries (front), the later ones the others (back of the buffer, descending).
struct Rounds {
    int nra, nang, front, back, low;  // back - 32 r: index in a later round; low: the last of them
    __device__ __forceinline__ Rounds(int nang_, int nrest, int nb, int lane)
        : nra((nang_ + 31) >> 5), nang(nang_), front(lane), back(nb - 1 - lane + 32 * ((nang_ + 31) >> 5)),
          low(nb - nrest) {}
    __device__ __forceinline__ bool at(int r, int &k) const {
        const bool ang = r < nra;  // (uniform)
        k = ang ? front + 32 * r : back - 32 * r;
        return ang ? k < nang : k >= low;
    }
};

// Warp totals of 8 pairs of partial sums (one pair per lane and order): lane l
// returns the pair of order 2 (l & 3) + (l >> 4). Each lane leaves its 16 values
// in its row of the buffer, lane (c, g) = (l & 3, l >> 2) adds column quad c of
// rows 4g .. 4g + 3, and the eight g are joined by shuffles that halve the quad
// first: 27 instructions where a shuffle-only transposed reduction takes 78.
__device__ __forceinline__ float2 reduce8(const float2 (&v)[8], float *red, int lane) {
    float4 *row = reinterpret_cast<float4 *>(red + lane * kRedStride);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) row[q] = make_float4(v[2 * q].x, v[2 * q].y, v[2 * q + 1].x, v[2 * q + 1].y);
    __syncwarp();
    const float4 *col = reinterpret_cast<const float4 *>(red + (lane & ~3) * kRedStride) + (lane & 3);
    float2 lo = dup2(0.f), hi = lo;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 x = col[i * (kRedStride / 4)];
        if (i == 0) {
            lo = make_float2(x.x, x.y);
            hi = make_float2(x.z, x.w);
        } else {
            lo = __fadd2_rn(lo, make_float2(x.x, x.y));
            hi = __fadd2_rn(hi, make_float2(x.z, x.w));
        }
    }
    const bool up = lane & 16;
    float2 send = up ? lo : hi, t = up ? hi : lo;
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) {
        const float2 in = make_float2(__shfl_xor_sync(kFull, send.x, o), __shfl_xor_sync(kFull, send.y, o));
        t = __fadd2_rn(t, in);
        send = t;
    }
    return t;
}
__device__ __forceinline__ int reduce8_order(int lane) { return 2 * (lane & 3) + (lane >> 4); }

// Two pairs (10 shuffles; the buffer would move 16): lane l returns the pair l >> 4.
__device__ __forceinline__ float2 reduce2(float2 v0, float2 v1, int lane) {
    const bool up = lane & 16;
    float2 send = up ? v0 : v1, t = up ? v1 : v0;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        t = __fadd2_rn(t, make_float2(__shfl_xor_sync(kFull, send.x, o), __shfl_xor_sync(kFull, send.y, o)));
        send = t;
    }
    return t;
}

// The totals of orders [0, N) of v (a compile-time count), times scale, to
// dst[2 (at + order)] and [.. + 1].
template <int N>
__device__ __forceinline__ void reduce_orders(const float2 *v, float *red, float *dst, int at, int lane) {
#pragma unroll
    for (int b = 0; b < N; b += 8) {
        if (N - b <= 2) {
            const float2 t = reduce2(v[b], N - b == 2 ? v[b + 1 < N ? b + 1 : b] : dup2(0.f), lane);
            const int o = b + (lane >> 4);
            if ((lane & 15) == 0 && o < N) *reinterpret_cast<float2 *>(dst + 2 * (at + o)) = t;
            continue;
        }
        float2 w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = b + q < N ? v[b + q] : dup2(0.f);
        const float2 t = reduce8(w, red, lane);
        const int o = b + reduce8_order(lane);
        if ((lane & 12) == 0 && o < N) *reinterpret_cast<float2 *>(dst + 2 * (at + o)) = t;
    }
}

// Angular pairs in one block of at most 32 entries: lane l owns entry l, and at
// shift t it meets entry (l + t) mod n, t = 1 .. n/2, so that every unordered
// pair occurs once (at t = n/2 with n even twice, once from each side). The
// first n/2 + 1 entries are repeated after the last, so the partner's address
// needs no wrap. Two shifts per iteration, their Chebyshev recurrences packed.
//
// Forward: S_q = sum_pairs w T_q(cos), plain and species-weighted.
template <int KAT, bool EXACT>
__device__ __forceinline__ void ring_forward(int n, int Ka, const ListWarp &W, int lane, float2 (&pp)[KAT],
                                             float2 (&pw)[KAT]) {
    const int self = lane < n ? lane : 0;
    float4 uj = W.a_u[self];
    const float sj = W.a_s[self];
    if (lane >= n) uj.w = 0.f;
    const float4 *pu = W.a_u + self + 1;
    const float *ps = W.a_s + self + 1;
    const float2 fj = dup2(uj.w);
    auto two = [&](float2 f) {  // two shifts; f: uj.w times the weight of each
        const float4 ua = pu[0], ub = pu[1];
        const float2 c = make_float2(uj.x * ua.x + uj.y * ua.y + uj.z * ua.z,
                                     uj.x * ub.x + uj.y * ub.y + uj.z * ub.z);
        const float2 w = make_float2(f.x * ua.w, f.y * ub.w);
        const float2 ww = make_float2(w.x * (sj * ps[0]), w.y * (sj * ps[1]));
        const float2 x2 = __fadd2_rn(c, c);
        float2 tm = dup2(1.0f), tc = c;
        pp[0] = __fadd2_rn(pp[0], w);
        pw[0] = __fadd2_rn(pw[0], ww);
#pragma unroll
        for (int q = 1; q < KAT; ++q) {
            if (EXACT || q < Ka) {
                pp[q] = ffma2(tc, w, pp[q]);
                pw[q] = ffma2(tc, ww, pw[q]);
                const float2 tn = ffma2(x2, tc, make_float2(-tm.x, -tm.y));
                tm = tc;
                tc = tn;
            }
        }
        pu += 2;
        ps += 2;
    };
    if (n < 2) return;
    const int full = (n - 1) >> 1;  // shifts that meet every pair once
    for (int i = full >> 1; i > 0; --i) two(fj);
    // what is left: a full shift (odd `full`), then the half-weighted one (even n)
    if ((full & 1) || !(n & 1))
        two((full & 1) ? make_float2(uj.w, (n & 1) ? 0.f : 0.5f * uj.w) : make_float2(0.5f * uj.w, 0.f));
}

// One step of Clenshaw's recurrence for two arguments (clenshaw_d2): the
// coefficient a0 + w a1 of each, then b and the halved derivative chain D. The
// coefficients are scalars: two scalar FMAs take as long as one packed one, and
// need no duplicated operand in registers or shared memory.
struct Clenshaw2 {
    float2 x2, b1, b2, D1, D2;
    __device__ __forceinline__ explicit Clenshaw2(float2 x) : x2(__fadd2_rn(x, x)), b1(dup2(0.f)) { b2 = D1 = D2 = b1; }
    __device__ __forceinline__ void step(float a0, float a1, float2 w) {
        const float2 m1 = dup2(-1.0f), a = make_float2(fmaf(w.x, a1, a0), fmaf(w.y, a1, a0));
        const float2 b = ffma2(x2, b1, ffma2(m1, b2, a));
        const float2 D = ffma2(x2, D1, ffma2(m1, D2, b1));
        b2 = b1;
        b1 = b;
        D2 = D1;
        D1 = D;
    }
    __device__ __forceinline__ void finish(float a0, float a1, float2 w, float2 x, float2 &S, float2 &dS) {
        const float2 a = make_float2(fmaf(w.x, a1, a0), fmaf(w.y, a1, a0));
        S = ffma2(x, b1, ffma2(dup2(-1.0f), b2, a));
        dS = ffma2(x2, D1, ffma2(dup2(-2.0f), D2, b1));
    }
};

// S = sum_q a_q T_q(x) and dS = sum_q a_q T_q'(x) of two arguments, a_q = a0_q +
// w a1_q, the coefficient pairs (a0, a1) of orders 0 .. KT - 1 read from shared
// memory, two orders per 128-bit load (KT registers each would not fit).
template <int KT, bool EXACT>
__device__ __forceinline__ void clenshaw_shared(float2 x, float2 w, const float2 *coef, int K, float2 &S, float2 &dS) {
    // (a compiler barrier: the loads stay inside the caller's loop)
    asm volatile("" ::: "memory");
    Clenshaw2 c(x);
    const float4 *two = reinterpret_cast<const float4 *>(coef);
#pragma unroll
    for (int h = (KT - 1) / 2; h >= 1; --h) {
        const float4 k = two[h];
        if (2 * h + 1 < KT && (EXACT || 2 * h + 1 < K)) c.step(k.z, k.w, w);
        if (EXACT || 2 * h < K) c.step(k.x, k.y, w);
    }
    const float4 k = two[0];
    if (KT > 1 && (EXACT || K > 1)) c.step(k.z, k.w, w);
    c.finish(k.x, k.y, w, x, S, dS);
}

// The same with the coefficients in registers.
template <int KT, bool EXACT>
__device__ __forceinline__ void clenshaw_regs(float2 x, float2 w, const float (&a0)[KT], const float (&a1)[KT], int K,
                                              float2 &S, float2 &dS) {
    Clenshaw2 c(x);
#pragma unroll
    for (int q = KT - 1; q >= 1; --q)
        if (EXACT || q < K) c.step(a0[q], a1[q], w);
    c.finish(a0[0], a1[0], w, x, S, dS);
}

// Coefficient pairs of the KAT angular orders into registers.
template <int KAT>
__device__ __forceinline__ void load_coef(const float2 *coef, float (&a0)[KAT], float (&a1)[KAT]) {
#pragma unroll
    for (int q = 0; q < KAT; ++q) {
        const float2 k = coef[q];
        a0[q] = k.x;
        a1[q] = k.y;
    }
}

// Backward: with S_jk = sum_q a_q T_q(c), S'_jk its derivative and f the cutoff
// values, the gradient with respect to d_j is
//   dE/dd_j = f_j' B_j u_j + (f_j / r_j) (V_j - (V_j . u_j) u_j),
//   B_j = sum_k S_jk f_k,  V_j = sum_k S'_jk f_k u_k
// (sum_k S'_jk f_k cos_jk = V_j . u_j), so a pair adds four products per side;
// the rest is done once per entry. Each lane adds its own side and takes S and
// S' of the pair it is the partner of by two shuffles.
template <int KAT, bool EXACT>
__device__ __forceinline__ float4 ring_backward(int n, int Ka, const ListWarp &W, const float2 *coef, int lane) {
    float a0[KAT], a1[KAT];
    load_coef(coef, a0, a1);
    const int self = lane < n ? lane : 0;
    const float4 uj = W.a_u[self];
    const float sj = W.a_s[self];
    const float4 *pu = W.a_u + self + 1;
    const float *ps = W.a_s + self + 1;
    float4 V = make_float4(0.f, 0.f, 0.f, 0.f);  // V_j, B_j
    int sa = lane == 0 ? n - 1 : lane - 1;       // lane (l - t) mod n
    // two shifts: j: the second one is inside the range; ka, kb: their pairs are met
    // once, so that the other side has to be added too
    auto two = [&](bool j, bool ka, bool kb) {
        const float4 ua = pu[0], ub = pu[1];
        const float2 w = make_float2(sj * ps[0], sj * ps[1]);
        const float2 c = make_float2(uj.x * ua.x + uj.y * ua.y + uj.z * ua.z,
                                     uj.x * ub.x + uj.y * ub.y + uj.z * ub.z);
        float2 S, dS;
        clenshaw_regs<KAT, EXACT>(c, w, a0, a1, Ka, S, dS);
        const float fa = ua.w, fb = j ? ub.w : 0.f;
        const float ga = dS.x * fa, gb = dS.y * fb;
        V.x = fmaf(ga, ua.x, fmaf(gb, ub.x, V.x));
        V.y = fmaf(ga, ua.y, fmaf(gb, ub.y, V.y));
        V.z = fmaf(ga, ua.z, fmaf(gb, ub.z, V.z));
        V.w = fmaf(S.x, fa, fmaf(S.y, fb, V.w));
        // the other side: this lane is the partner of lane (l - t) mod n
        const int sb = sa == 0 ? n - 1 : sa - 1;
        const float dSa = __shfl_sync(kFull, dS.x, sa), Sa = __shfl_sync(kFull, S.x, sa);
        const float dSb = __shfl_sync(kFull, dS.y, sb), Sb = __shfl_sync(kFull, S.y, sb);
        const float4 va = W.a_u[sa], vb = W.a_u[sb];
        const float ha = ka ? va.w : 0.f, hb = kb ? vb.w : 0.f;
        const float ma = dSa * ha, mb = dSb * hb;
        V.x = fmaf(ma, va.x, fmaf(mb, vb.x, V.x));
        V.y = fmaf(ma, va.y, fmaf(mb, vb.y, V.y));
        V.z = fmaf(ma, va.z, fmaf(mb, vb.z, V.z));
        V.w = fmaf(Sa, ha, fmaf(Sb, hb, V.w));
        sa = sb == 0 ? n - 1 : sb - 1;
        pu += 2;
        ps += 2;
    };
    if (n < 2) return V;
    const int full = (n - 1) >> 1;
    for (int i = full >> 1; i > 0; --i) two(true, true, true);
    if ((full & 1) || !(n & 1)) two((full & 1) && !(n & 1), full & 1, false);
    return V;
}

// More than 32 angular entries: nblk blocks of bs (at most 32) entries, every
// pair of blocks (A <= Bk). Inside a block the ring of its entries; between two
// blocks lane l of A meets column (l + t) mod bs of Bk, t = 0 .. bs - 1.
struct BlockStep {
    int k;      // partner entry (a valid one where v is false)
    float v;    // 1, 1/2 (a pair met from both sides) or 0
};
__device__ __forceinline__ BlockStep block_step(bool diag, int t, int nA, int nB, int bs, int baseB, int lane,
                                                bool vj) {
    BlockStep s;
    const int ring = diag ? nA : bs;
    int cc = lane + t;
    if (cc >= ring) cc -= ring;
    const bool v = vj && cc < nB && (!diag || 2 * t <= nA) && t < ring;
    s.k = v ? baseB + cc : baseB;
    s.v = v ? (diag && 2 * t == nA ? 0.5f : 1.0f) : 0.f;
    return s;
}

template <int KAT, bool EXACT>
__device__ __forceinline__ void blocks_forward(int n, int Ka, const ListWarp &W, int lane, float2 (&pp)[KAT],
                                               float2 (&pw)[KAT]) {
    const int nblk = (n + 31) >> 5, bs = (n + nblk - 1) / nblk;
    for (int A = 0; A * bs < n; ++A) {
        const int nA = min(bs, n - A * bs);
        const bool vj = lane < nA;
        const int self = A * bs + (vj ? lane : 0);
        const float4 uj = W.a_u[self];
        const float sj = W.a_s[self];
        for (int Bk = A; Bk * bs < n; ++Bk) {
            const int nB = min(bs, n - Bk * bs);
            const bool diag = Bk == A;
            const int t0 = diag ? 1 : 0, t1 = diag ? nA / 2 : bs - 1;
            for (int t = t0; t <= t1; t += 2) {
                const BlockStep a = block_step(diag, t, nA, nB, bs, Bk * bs, lane, vj);
                const BlockStep b = block_step(diag, t + 1, nA, nB, bs, Bk * bs, lane, vj && t < t1);
                const float4 ua = W.a_u[a.k], ub = W.a_u[b.k];
                const float2 c = make_float2(uj.x * ua.x + uj.y * ua.y + uj.z * ua.z,
                                             uj.x * ub.x + uj.y * ub.y + uj.z * ub.z);
                const float2 w = make_float2(uj.w * ua.w * a.v, uj.w * ub.w * b.v);
                const float2 ww = make_float2(w.x * (sj * W.a_s[a.k]), w.y * (sj * W.a_s[b.k]));
                const float2 x2 = __fadd2_rn(c, c);
                float2 tm = dup2(1.0f), tc = c;
                pp[0] = __fadd2_rn(pp[0], w);
                pw[0] = __fadd2_rn(pw[0], ww);
#pragma unroll
                for (int q = 1; q < KAT; ++q) {
                    if (EXACT || q < Ka) {
                        pp[q] = ffma2(tc, w, pp[q]);
                        pw[q] = ffma2(tc, ww, pw[q]);
                        const float2 tn = ffma2(x2, tc, make_float2(-tm.x, -tm.y));
                        tm = tc;
                        tc = tn;
                    }
                }
            }
        }
    }
}

// (a_g: the sums (V, B) of every entry, zeroed and filled here)
template <int KAT, bool EXACT>
__device__ __forceinline__ void blocks_backward(int n, int Ka, const ListWarp &W, const float2 *coef, int lane) {
    float a0[KAT], a1[KAT];
    load_coef(coef, a0, a1);
    const int nblk = (n + 31) >> 5, bs = (n + nblk - 1) / nblk;
    for (int k = lane; k < n; k += 32) W.a_g[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();
    for (int A = 0; A * bs < n; ++A) {
        const int nA = min(bs, n - A * bs);
        const bool vj = lane < nA;
        const int self = A * bs + (vj ? lane : 0);
        const float4 uj = W.a_u[self];
        const float sj = W.a_s[self];
        float4 V = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int Bk = A; Bk * bs < n; ++Bk) {
            const int nB = min(bs, n - Bk * bs);
            const bool diag = Bk == A;
            const int ring = diag ? nA : bs;
            const int t0 = diag ? 1 : 0, t1 = diag ? nA / 2 : bs - 1;
            float4 U = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int t = t0; t <= t1; t += 2) {
                const BlockStep a = block_step(diag, t, nA, nB, bs, Bk * bs, lane, vj);
                const BlockStep b = block_step(diag, t + 1, nA, nB, bs, Bk * bs, lane, vj && t < t1);
                const float4 ua = W.a_u[a.k], ub = W.a_u[b.k];
                const float2 c = make_float2(uj.x * ua.x + uj.y * ua.y + uj.z * ua.z,
                                             uj.x * ub.x + uj.y * ub.y + uj.z * ub.z);
                float2 S, dS;
                clenshaw_regs<KAT, EXACT>(c, make_float2(sj * W.a_s[a.k], sj * W.a_s[b.k]), a0, a1, Ka, S, dS);
                const float fa = a.v != 0.f ? ua.w : 0.f, fb = b.v != 0.f ? ub.w : 0.f;
                const float ga = dS.x * fa, gb = dS.y * fb;
                V.x = fmaf(ga, ua.x, fmaf(gb, ub.x, V.x));
                V.y = fmaf(ga, ua.y, fmaf(gb, ub.y, V.y));
                V.z = fmaf(ga, ua.z, fmaf(gb, ub.z, V.z));
                V.w = fmaf(S.x, fa, fmaf(S.y, fb, V.w));
                int sa = lane - t, sb = sa - 1;
                if (sa < 0) sa += ring;
                if (sb < 0) sb += ring;
                sa &= 31;  // (lanes past the ring: any lane, masked below)
                sb &= 31;
                const float dSa = __shfl_sync(kFull, dS.x, sa), Sa = __shfl_sync(kFull, S.x, sa);
                const float dSb = __shfl_sync(kFull, dS.y, sb), Sb = __shfl_sync(kFull, S.y, sb);
                const bool ra = lane < nB && sa < nA && !(diag && 2 * t == nA);
                const bool rb = lane < nB && sb < nA && t < t1 && !(diag && 2 * (t + 1) == nA);
                const float4 va = W.a_u[A * bs + (ra ? sa : 0)], vb = W.a_u[A * bs + (rb ? sb : 0)];
                const float ha = ra ? va.w : 0.f, hb = rb ? vb.w : 0.f;
                const float ka = dSa * ha, kb = dSb * hb;
                U.x = fmaf(ka, va.x, fmaf(kb, vb.x, U.x));
                U.y = fmaf(ka, va.y, fmaf(kb, vb.y, U.y));
                U.z = fmaf(ka, va.z, fmaf(kb, vb.z, U.z));
                U.w = fmaf(Sa, ha, fmaf(Sb, hb, U.w));
            }
            if (lane < nB) {  // each entry is written by its owner lane only
                float4 o = W.a_g[Bk * bs + lane];
                W.a_g[Bk * bs + lane] = make_float4(o.x + U.x, o.y + U.y, o.z + U.z, o.w + U.w);
            }
        }
        if (vj) {
            float4 o = W.a_g[self];
            W.a_g[self] = make_float4(o.x + V.x, o.y + V.y, o.z + V.z, o.w + V.w);
        }
    }
}

// Spherical-harmonic form (sh_angular.cuh): the component sums of the atom's
// angular entries, interleaved (plain, weighted) at sh[2c], sh[2c + 1] for the 49
// components c, and sum w_j^2, sum (s_j w_j)^2 at c = 49. Two column groups; an
// entry's components are computed once and enter both copies by one packed FMA.
template <int M0, int M1, bool W2>
__device__ __forceinline__ void sh_sum_group(int nang, const ListWarp &W, int lane) {
    constexpr int c0 = sh_comp(M0, M0, 0), N = (W2 ? kShComps + 1 : sh_comp(M1 + 1, M1 + 1, 0)) - c0;
    float2 acc[N];
#pragma unroll
    for (int k = 0; k < N; ++k) acc[k] = dup2(0.f);
    for (int k = lane; k < nang; k += 32) {
        const float4 u = W.a_u[k];
        const float2 w = make_float2(u.w, u.w * W.a_s[k]);
        float cm = 1.f, sm = 0.f, pmm = 1.f;  // C_m, S_m, (2m - 1)!!
#pragma unroll
        for (int m = 0; m <= M1; ++m) {
            if (m > 0) {
                const float c1 = u.x * cm - u.y * sm, s1 = fmaf(u.x, sm, u.y * cm);
                cm = c1;
                sm = s1;
                pmm *= (float)(2 * m - 1);
            }
            if (m < M0) continue;
            const float2 wc = __fmul2_rn(w, dup2(cm)), ws = __fmul2_rn(w, dup2(sm));
            float p2 = 0.f, p1 = pmm;
#pragma unroll
            for (int l = m; l <= kShL; ++l) {
                float p;
                if (l == m) {
                    p = p1;
                } else if (l == m + 1) {
                    p = (float)(2 * m + 1) * u.z * p1;
                } else {
                    const float fa = (float)(2 * l - 1) / (float)(l - m), fb = (float)(l + m - 1) / (float)(l - m);
                    p = fmaf(fa * u.z, p1, -fb * p2);
                }
                if (l > m) {
                    p2 = p1;
                    p1 = p;
                }
                acc[sh_comp(l, m, 0) - c0] = ffma2(dup2(p), wc, acc[sh_comp(l, m, 0) - c0]);
                if (m > 0) acc[sh_comp(l, m, 1) - c0] = ffma2(dup2(p), ws, acc[sh_comp(l, m, 1) - c0]);
            }
        }
        if constexpr (W2) acc[kShComps - c0] = ffma2(w, w, acc[kShComps - c0]);
    }
    reduce_orders<N>(acc, W.red, W.sh, c0, lane);
}

__device__ __forceinline__ void sh_sums(int nang, const ListWarp &W, int lane) {
    sh_sum_group<0, 2, false>(nang, W, lane);
    sh_sum_group<3, kShL, true>(nang, W, lane);
    __syncwarp();
}

// S_a = sum_c b_{a l(c)} N_c^2 A_c^2 - sum w^2 of both copies into the rows of orders
// KRT .. KRT + KAT - 1 of dst (without the last term): each lane takes its two
// components for every order, with the coefficients b N^2 of the table (rounded
// once, as sh_fingerprint does), and the pairs are reduced across the warp.
constexpr int kShTabList = kShTab + 7 * kShComps;  // the table with b_{a l(c)} N_c^2 at kShTab + 49 a + c
template <int KRT, int KAT>
__device__ __forceinline__ void sh_fingerprints(const ListWarp &W, const float *tab, float *dst, int lane) {
    float2 acc[KAT];
#pragma unroll
    for (int a = 0; a < KAT; ++a) acc[a] = dup2(0.f);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        if (c < kShComps) {
            const float2 A = *reinterpret_cast<const float2 *>(W.sh + 2 * c);
#pragma unroll
            for (int a = 0; a < KAT; ++a)
                acc[a] = ffma2(__fmul2_rn(dup2(tab[kShTab + kShComps * a + c]), A), A, acc[a]);
        }
    }
    reduce_orders<KAT>(acc, W.red, dst, KRT, lane);
}

// Where the contraction's coefficients of component c lie in the warp's scratch:
// m = 0: the pairs (D, D') of l = 0 .. 6 at [2l]; m > 0: the quad (D_cos, D_sin,
// D'_cos, D'_sin) of (l, m) at [16 + 4 q], q counting the (l, m) column by column.
constexpr int kShQuads = 16;

// E = sum_c k_c v_c(u) and F = sum_c k_c grad_u v_c(u) of one entry, k_c = D_c + s
// D'_c (sh_contract with cosine and sine parts packed: one 128-bit load and three
// packed FMAs per (l, m)). Called by all 32 lanes together.
__device__ __forceinline__ void sh_contract2(float x, float y, float z, float s, const float *D, float &E, float &Fx,
                                             float &Fy, float &Fz) {
    __syncwarp();  // (keeps the loads of one column from moving above the one before)
    const float2 s2 = dup2(s), z2 = dup2(z);
    float h0 = 0.f, d0 = 0.f;
    {
        float p2 = 0.f, p1 = 1.f, q2 = 0.f, q1 = 0.f;  // P_l and P_l'
#pragma unroll
        for (int l = 0; l <= kShL; ++l) {
            float p = p1, d = 0.f;
            if (l == 1) {
                p = z;
                d = 1.f;
            } else if (l > 1) {
                const float fa = (float)(2 * l - 1) / (float)l, fb = (float)(l - 1) / (float)l;
                p = fmaf(fa * z, p1, -fb * p2);
                d = fmaf(fa, fmaf(z, q1, p1), -fb * q2);
            }
            if (l > 0) {
                p2 = p1;
                p1 = p;
                q2 = q1;
                q1 = d;
            }
            const float2 kc = *reinterpret_cast<const float2 *>(D + 2 * l);
            const float k = fmaf(s, kc.y, kc.x);
            h0 = fmaf(k, p, h0);
            d0 = fmaf(k, d, d0);
        }
    }
    E = h0;
    Fz = d0;
    Fx = Fy = 0.f;
    float cm = 1.f, sm = 0.f, pmm = 1.f;
    int q = 0;
#pragma unroll
    for (int m = 1; m <= kShL; ++m) {
        const float cp = cm, sp = sm;  // C_{m-1}, S_{m-1}
        cm = x * cp - y * sp;
        sm = fmaf(x, sp, y * cp);
        pmm *= (float)(2 * m - 1);
        __syncwarp();
        float2 h = dup2(0.f), dh = h;              // cosine and sine sums of k Pbar and k Pbar'
        float2 p2 = h, p1 = dup2(pmm), q2 = h, q1 = h;
#pragma unroll
        for (int l = m; l <= kShL; ++l, ++q) {
            float2 p = p1, d = dup2(0.f);
            if (l == m + 1) {
                d = dup2((float)(2 * m + 1) * pmm);
                p = __fmul2_rn(d, z2);
            } else if (l > m + 1) {
                const float fa = (float)(2 * l - 1) / (float)(l - m), fb = (float)(l + m - 1) / (float)(l - m);
                const float2 nb = dup2(-fb);
                p = ffma2(__fmul2_rn(dup2(fa), z2), p1, __fmul2_rn(nb, p2));
                d = ffma2(dup2(fa), ffma2(z2, q1, p1), __fmul2_rn(nb, q2));
            }
            if (l > m) {
                p2 = p1;
                p1 = p;
                q2 = q1;
                q1 = d;
            }
            const float4 kq = *reinterpret_cast<const float4 *>(D + kShQuads + 4 * q);
            const float2 k = ffma2(s2, make_float2(kq.z, kq.w), make_float2(kq.x, kq.y));
            h = ffma2(k, p, h);
            if (l > m) dh = ffma2(k, d, dh);
        }
        E = fmaf(h.x, cm, fmaf(h.y, sm, E));
        Fz = fmaf(dh.x, cm, fmaf(dh.y, sm, Fz));
        Fx = fmaf((float)m, fmaf(h.x, cp, h.y * sp), Fx);
        Fy = fmaf((float)m, fmaf(h.y, cp, -h.x * sp), Fy);
    }
}

// (V, B) of every angular entry: with the coefficients (D_c, D'_c) = 2 N_c^2 (A_c
// k_l, A'_c k'_l), k_l = sum_a g_a b_al, written over the component sums, V is the
// contraction's gradient F and B = E - 2 w (sum_a g_a + s^2 sum_a g'_a).
template <int KRT, int KAT>
__device__ __forceinline__ void sh_gradients(int nang, const ListWarp &W, const float2 *coef, const float *tab,
                                             int lane) {
    float gsum = 0.f, gwsum = 0.f;
    float dv[2], dwv[2];
#pragma unroll
    for (int a = 0; a < KAT; ++a) {
        gsum += coef[KRT + a].x;
        gwsum += coef[KRT + a].y;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        dv[h] = dwv[h] = 0.f;
        if (c < kShComps) {
            const int l = (int)tab[kShTabL + c];
            float kl = 0.f, klw = 0.f;
#pragma unroll
            for (int a = 0; a < KAT; ++a) {
                const float b = tab[kShTabB + a * (kShL + 1) + l];
                kl = fmaf(coef[KRT + a].x, b, kl);
                klw = fmaf(coef[KRT + a].y, b, klw);
            }
            const float n2 = 2.0f * tab[kShTabN + c];
            dv[h] = n2 * W.sh[2 * c] * kl;
            dwv[h] = n2 * W.sh[2 * c + 1] * klw;
        }
    }
    __syncwarp();  // every lane has read its sums
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        // components 7, 8, 9, ...: cosine and sine of the (l, m) in turn (sh_comp)
        const int at = c <= kShL ? 2 * c : kShQuads + 4 * ((c - kShL - 1) >> 1) + ((c - kShL - 1) & 1);
        if (c < kShComps) {
            W.sh[at] = dv[h];
            W.sh[at + (c <= kShL ? 1 : 2)] = dwv[h];
        }
    }
    __syncwarp();
    for (int base = 0; base < nang; base += 32) {  // (sh_contract2 synchronises the warp)
        const int k = base + lane < nang ? base + lane : 0;
        const float4 u = W.a_u[k];
        const float s = W.a_s[k];
        float E, Fx, Fy, Fz;
        sh_contract2(u.x, u.y, u.z, s, W.sh, E, Fx, Fy, Fz);
        if (base + lane < nang) W.a_g[k] = make_float4(Fx, Fy, Fz, E - 2.0f * u.w * fmaf(s * s, gwsum, gsum));
    }
}

// The atom's network (Sec. II.A, Eq. ANN-layer; FP32) from the descriptor pair
// (G0, G1) of this lane's order, and back-propagation to dE/dG: E is returned
// in every lane, the lane's two coefficients in (c0, c1). Lanes own neurons; see
// process_atom in potential_kernels.cuh for the half-warp split of HB = 16.
template <int KRT, int KAT, int HB>
__device__ __forceinline__ float list_network(const FusedNet &net, const float *Pt, float *xs, int lane, float G0,
                                              float G1, float *rec, int Kr, int Ka, float &c0, float &c1) {
    constexpr int NS = list_inputs<KRT, KAT>(HB), WS = list_w1_stride<KRT, KAT>(HB);
    constexpr int HS = HB + 4, NK1 = HB == 16 ? NS / 2 : NS, NKH = HB == 16 ? 8 : 32;
    constexpr int P = KRT + KAT;
    const int s0 = lane < P ? lane : 0;  // (lanes past the last slot: slot 0's parameters, results unused)
    const float *shift = Pt + net.offShift + s0, *scale = Pt + net.offScale + s0;
    const float sc0 = scale[0], sc1 = scale[P];
    const float x0 = (G0 - shift[0]) * sc0, x1 = (G1 - shift[P]) * sc1;
    if (rec) {
        const int k0 = lane_col<KRT, KAT>(lane, 0, Kr, Ka), k1 = lane_col<KRT, KAT>(lane, 1, Kr, Ka);
        if (k0 >= 0) rec[k0] = x0;
        if (k1 >= 0) rec[k1] = x1;
    }
    const int o = lane & (HB - 1), h = HB == 16 ? lane >> 4 : 0;
    if (lane < P) {
        xs[lane] = x0;
        xs[lane + P] = x1;
    }
    if (2 * P + lane < NS) xs[2 * P + lane] = 0.f;
    __syncwarp();
    const float *W1 = Pt;  // (offW[1] == 0)
    float z;
    {
        const float *wr = W1 + o * WS + h * NK1, *gx = xs + h * NK1;
        float2 za = dup2(0.f);
#pragma unroll 4
        for (int k = 0; k < NK1; k += 4) {
            const float4 gv = *reinterpret_cast<const float4 *>(gx + k);
            const float4 wv = *reinterpret_cast<const float4 *>(wr + k);
            za = ffma2(make_float2(wv.x, wv.y), make_float2(gv.x, gv.y), za);
            za = ffma2(make_float2(wv.z, wv.w), make_float2(gv.z, gv.w), za);
        }
        z = za.x + za.y;
        if constexpr (HB == 16) z += __shfl_xor_sync(kFull, z, 16);
    }
    float xl[kMaxLayers];
    xl[1] = tanh_exp(z + Pt[net.offB[1] + o]);
    if (rec && lane < net.H[1]) rec[net.rec_x[1] + lane] = xl[1];
#pragma unroll
    for (int l = 2; l < kMaxLayers; ++l) {
        if (l < net.L) {
            __syncwarp();
            if (lane < HB) xs[lane] = xl[l - 1];
            __syncwarp();
            const float *wr = Pt + net.offW[l] + o * HS + h * NKH, *xv = xs + h * NKH;
            float2 za = dup2(0.f);
#pragma unroll 4
            for (int k = 0; k < NKH; k += 4) {
                const float4 gv = *reinterpret_cast<const float4 *>(xv + k);
                const float4 wv = *reinterpret_cast<const float4 *>(wr + k);
                za = ffma2(make_float2(wv.x, wv.y), make_float2(gv.x, gv.y), za);
                za = ffma2(make_float2(wv.z, wv.w), make_float2(gv.z, gv.w), za);
            }
            float zz = za.x + za.y;
            if constexpr (HB == 16) zz += __shfl_xor_sync(kFull, zz, 16);
            xl[l] = tanh_exp(zz + Pt[net.offB[l] + o]);
            if (rec && lane < net.H[l]) rec[net.rec_x[l] + lane] = xl[l];
        }
    }
    float xlast = 0.f;
#pragma unroll
    for (int l = 1; l < kMaxLayers; ++l)
        if (l == net.L - 1) xlast = xl[l];
    const float wL = Pt[net.offWL + o];
    float E = wL * xlast;
#pragma unroll
    for (int m = HB / 2; m >= 1; m >>= 1) E += __shfl_xor_sync(kFull, E, m);
    E += Pt[net.offBL];
    float delta = (1.0f - xlast * xlast) * wL;
    if (rec && lane < net.Hlast) rec[net.rec_dlast + lane] = delta;
#pragma unroll
    for (int l = kMaxLayers - 1; l >= 2; --l) {
        if (l < net.L) {
            __syncwarp();
            if (lane < HB) xs[lane] = delta;
            __syncwarp();
            const float *wc = Pt + net.offW[l] + h * NKH * HS + o, *dv = xs + h * NKH;
            float2 da = dup2(0.f);
#pragma unroll 2
            for (int q = 0; q < NKH; q += 4) {
                const float4 d4 = *reinterpret_cast<const float4 *>(dv + q);
                da = ffma2(make_float2(wc[(q + 0) * HS], wc[(q + 1) * HS]), make_float2(d4.x, d4.y), da);
                da = ffma2(make_float2(wc[(q + 2) * HS], wc[(q + 3) * HS]), make_float2(d4.z, d4.w), da);
            }
            float dx = da.x + da.y;
            if constexpr (HB == 16) dx += __shfl_xor_sync(kFull, dx, 16);
            delta = (1.0f - xl[l - 1] * xl[l - 1]) * dx;
            if (rec && lane < net.H[l - 1]) rec[net.rec_d[l - 1] + lane] = delta;
        }
    }
    // dE/dg of the lane's slot and its weighted copy: sums over even and odd neurons
    // in the two halves of a packed accumulator
    __syncwarp();
    if (lane < HB) xs[lane] = delta;
    __syncwarp();
    float2 d0 = dup2(0.f), d1 = d0;
    const float *wq = W1 + s0;
#pragma unroll 2
    for (int q = 0; q < HB; q += 4) {
        const float4 d = *reinterpret_cast<const float4 *>(xs + q);
        const float *w = wq + q * WS;
        d0 = ffma2(make_float2(w[0], w[WS]), make_float2(d.x, d.y), d0);
        d1 = ffma2(make_float2(w[P], w[WS + P]), make_float2(d.x, d.y), d1);
        d0 = ffma2(make_float2(w[2 * WS], w[3 * WS]), make_float2(d.z, d.w), d0);
        d1 = ffma2(make_float2(w[2 * WS + P], w[3 * WS + P]), make_float2(d.z, d.w), d1);
    }
    c0 = (d0.x + d0.y) * sc0;
    c1 = (d1.x + d1.y) * sc1;
    __syncwarp();  // every lane has read the deltas
    return E;
}

// Per-CTA scalars kept in shared memory, so that they hold no registers
// through the atom loop.
template <int NW>
struct ListSums {
    double e[NW];
    double vir[NW][6];
    unsigned long long st[NW][4];
};

// One warp per atom, atoms from a counter. For its atom the warp
//   1. reads the list row, applies the exact cutoff, and compacts the entries
//      into shared memory, the angular ones at the front;
//   2. evaluates the descriptor, reduced across the warp;
//   3. runs the network and back-propagates to dE/dG;
//   4. applies the chain rule: the angular sums of every entry, then one pass
//      over the entries that adds the radial part, the force atomics and the
//      virial.
// MODE: kFused, or kDescriptor (G rows to G_out) or kForces (dE/dG rows from
// dEdG_in). BATCH: the virial of every atom goes to vir_atom (summed per
// structure afterwards) instead of the CTA's partial row.
template <int KRT, int KAT, bool EXACT, int MODE, int HB, bool CODES, bool BATCH>
__global__ void __launch_bounds__(32 * list_max_warps<KRT, KAT, EXACT>(), 1)
    k_potential_list(Basis B, FusedNet net, Grid g, Caps caps, int a_lo, int a_hi, const float4 *pos4,
                     const float4 *rows, const int *codes, const int *count, const float *__restrict__ pnet,
                     float4 *__restrict__ F4, float *__restrict__ eatom, float *__restrict__ G_out,
                     const float *dEdG_in, double *__restrict__ e_part, double *__restrict__ vir_part,
                     float *__restrict__ vir_atom, unsigned long long *__restrict__ stats,
                     unsigned *__restrict__ err, unsigned *__restrict__ work) {
    constexpr bool kSh = sh_angular<KRT, KAT, EXACT>();
    constexpr int NW = list_max_warps<KRT, KAT, EXACT>();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ float s_tw[kMaxSpecies];
    __shared__ float s_sh[kSh ? kShTabList : 1];
    __shared__ ListSums<NW> s_sum;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int Kr = EXACT ? KRT : B.Kr, Ka = EXACT ? KAT : B.Ka;
    const ListLayout L = make_list_layout(CODES ? g.n_off : 0, caps.nb, caps.ang, MODE == kFused ? B.n_species : 0,
                                          net.stride, kSh, 1);
    float4 *off_shift = reinterpret_cast<float4 *>(smem + L.off_shift);
    float *s_par = reinterpret_cast<float *>(smem + L.params);
    unsigned char *wb = smem + L.warp_base + L.warp_bytes * warp;
    ListWarp W;
    W.e_d = reinterpret_cast<float4 *>(wb + L.e_d);
    W.e_j = reinterpret_cast<int *>(wb + L.e_j);
    W.a_u = reinterpret_cast<float4 *>(wb + L.a_u);
    W.a_s = reinterpret_cast<float *>(wb + L.a_s);
    W.red = reinterpret_cast<float *>(wb + L.red);
    W.a_g = reinterpret_cast<float4 *>(wb + L.red);
    W.coef = reinterpret_cast<float *>(wb + L.coef);
    W.sh = reinterpret_cast<float *>(wb + L.sh);
    const float2 *coef = reinterpret_cast<const float2 *>(W.coef);  // (a, a_w) of every order
#pragma unroll
    for (int t = 0; t < kMaxSpecies; ++t)
        if (tid == t) s_tw[t] = B.type_weight[t];
    if constexpr (kSh) {  // (the table's loader takes thread indices up to 64, a CTA may be one or two warps)
        for (int t = tid; t <= 64; t += blockDim.x) load_sh_table(B.sh_b, s_sh, t);
    }
    // the parameters arrive while the first atoms' descriptors are computed
    if constexpr (MODE == kFused) {
        const unsigned dst = (unsigned)__cvta_generic_to_shared(s_par);
        for (int k = tid; k < B.n_species * net.stride / 4; k += blockDim.x)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * k), "l"(pnet + 4 * k) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    bool staged = MODE != kFused;
    auto wait_params = [&]() {  // once per warp (a CTA barrier): every thread's copies are complete
        if (staged) return;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        staged = true;
    };
    if constexpr (CODES) {
        const int wx = 2 * g.m[0] + 1, wy = 2 * g.m[1] + 1;
        for (int o = tid; o < g.n_off; o += blockDim.x) {  // image shift of every list code
            const int ox = o % wx - g.m[0], oy = (o / wx) % wy - g.m[1], oz = o / (wx * wy) - g.m[2];
            off_shift[o] = make_float4(ox * g.hf[0] + oy * g.htf[0] + oz * g.htf[1], oy * g.hf[1] + oz * g.htf[2],
                                       oz * g.hf[2], 0.f);
        }
    }
    if (lane < 4) s_sum.st[warp][lane] = 0ull;
    if (lane == 0) s_sum.e[warp] = 0.0;
    if (lane < 6) s_sum.vir[warp][lane] = 0.0;
    __syncthreads();
    if constexpr (kSh) {
        for (int k = tid; k < 7 * kShComps; k += blockDim.x) {
            const int al = k / kShComps, c = k - al * kShComps;
            s_sh[kShTab + k] = s_sh[kShTabB + al * (kShL + 1) + (int)s_sh[kShTabL + c]] * s_sh[kShTabN + c];
        }
        __syncthreads();
    }
    // (what is above reads only what the kernels of the evaluation leave alone)
    pdl_wait();

    const float inv_rcr = 1.0f / B.rc_rad, inv_rca = 1.0f / B.rc_ang, rc2max = B.rc_max * B.rc_max;
    const int nb = caps.nb;
    // The first two rounds of an atom's row, its length and its species are loaded
    // while the atom before is in its last phase.
    struct Ahead {
        float4 e0, e1;
        int c0, c1;  // code rows
        int cnt, type;
    } nx;
    auto fetch = [&](int i) {
        if (i >= a_hi) return;
        nx.cnt = count[i];
        nx.type = __float_as_int(pos4[i].w);
        if constexpr (CODES) {
            const int *row = codes + (size_t)i * caps.vl_cap;
            nx.c0 = __ldcg(row + lane);  // (rows hold at least 64 entries; those past the count are not used)
            nx.c1 = __ldcg(row + 32 + lane);
        } else {
            const float4 *row = rows + (size_t)(i - a_lo) * caps.vl_cap;
            nx.e0 = __ldcs(row + lane);
            nx.e1 = __ldcs(row + 32 + lane);
        }
    };
    const int n_static = nw * (int)gridDim.x;
    int a = a_lo + warp * (int)gridDim.x + (int)blockIdx.x;
    fetch(a);
    while (a < a_hi) {
        int next = 0;  // the counter's reply is needed only at the end of the atom
        if (lane == 0) next = a_lo + n_static + (int)atomicAdd(work, 1u);

        // ---- 1. the list, and the radial sums of the descriptor as it is read (in
        // row order: sorted by distance the FP32 sums would be biased)
        const int cnt = nx.cnt, type = nx.type;
        float c0, c1;  // dE/dG of this lane's order and its weighted copy
        if constexpr (MODE == kForces) {
            const int D = 2 * (Kr + Ka);
            const int k0 = lane_col<KRT, KAT>(lane, 0, Kr, Ka), k1 = lane_col<KRT, KAT>(lane, 1, Kr, Ka);
            c0 = k0 >= 0 ? dEdG_in[(size_t)a * D + k0] : 0.f;
            c1 = k1 >= 0 ? dEdG_in[(size_t)a * D + k1] : 0.f;
        }
        int nang = 0, nrest = 0;
        bool over = false;
        constexpr bool kDesc = MODE != kForces;
        constexpr int LR = kSh ? 0 : KRT % 8, RB = KRT - LR;  // radial orders reduced on their own
        float2 acc[kDesc ? KRT : 1];
        if constexpr (kDesc) {
#pragma unroll
            for (int q = 0; q < KRT; ++q) acc[q] = dup2(0.f);
        }
        auto append = [&](bool in, float dx, float dy, float dz, int bits) {
            const float r2 = length2(dx, dy, dz);
            in = in && r2 <= rc2max && !(r2 == 0.f && (bits & kEntryIndex) == a);  // not the atom itself
            float inv = rsqrtf(r2), r = r2 * inv;
            if (in && r2 < 1e-12f) {  // r < 1e-6 A
                atomicOr(err, kErrOverlap);
                r = 1e-6f;
                inv = 1e6f;
            }
            if (!in) r = B.rc_rad;
            const float s = s_tw[in ? bits >> 28 : 0];
            const bool ina = in && r <= B.rc_ang;
            const unsigned m = __ballot_sync(kFull, in), ma = __ballot_sync(kFull, ina);
            const int na = __popc(ma), nr = __popc(m) - na;
            if (nang + nrest + na + nr > nb) {  // (uniform) no room: reported, results invalid
                over = true;
                return;
            }
            if (in) {
                const int slot = ina ? nang + __popc(ma & lt_mask) : nb - 1 - nrest - __popc(m & ~ma & lt_mask);
                W.e_d[slot] = make_float4(dx, dy, dz, r);
                W.e_j[slot] = bits;
                if (ina && slot < caps.ang) {
                    float sn, cs;
                    __sincosf(3.14159265358979f * (r * inv_rca), &sn, &cs);  // argument in [0, pi]
                    W.a_u[slot] = make_float4(dx * inv, dy * inv, dz * inv, 0.5f * (cs + 1.0f));
                    W.a_s[slot] = s;
                }
            }
            nang += na;
            nrest += nr;
            if constexpr (kDesc) {
                float fc, dfc;
                radial_cutoff(r, inv_rcr, fc, dfc);
                fc = in && r <= B.rc_rad ? fc : 0.f;
                const float x = 2.0f * r * inv_rcr - 1.0f;
                const float2 f = make_float2(fc, s * fc), x2 = dup2(2.0f * x);
                float2 tm = dup2(1.0f), t = dup2(x);
                acc[0] = __fadd2_rn(acc[0], f);
#pragma unroll
                for (int q = 1; q < KRT; ++q) {
                    if (EXACT || q < Kr) {
                        acc[q] = ffma2(t, f, acc[q]);
                        const float2 tn = ffma2(x2, t, make_float2(-tm.x, -tm.y));
                        tm = t;
                        t = tn;
                    }
                }
            }
        };
        // (the loads of the next round are in flight while a round is worked on)
        if constexpr (CODES) {
            const int jmask = (1 << caps.vl_jbits) - 1;
            const float4 ui = pos4[a];
            const int *row = codes + (size_t)a * caps.vl_cap;
            auto code = [&](int base) { return base + lane < cnt ? __ldcg(row + base + lane) : -1; };  // (entries >= 0)
            auto gather = [&](int e) { return e >= 0 ? pos4[e & jmask] : make_float4(0.f, 0.f, 0.f, 0.f); };
            int e0 = lane < cnt ? nx.c0 : -1, e1 = 32 + lane < cnt ? nx.c1 : -1;
            float4 p0 = gather(e0);
            for (int base = 0; base < cnt; base += 32) {
                const float4 p1 = gather(e1);
                const int e2 = code(base + 64);
                const float4 sh = off_shift[e0 >= 0 ? e0 >> caps.vl_jbits : 0];
                append(e0 >= 0, (p0.x + sh.x) - ui.x, (p0.y + sh.y) - ui.y, (p0.z + sh.z) - ui.z,
                       (e0 & jmask) | (__float_as_int(p0.w) << 28));
                e0 = e1;
                e1 = e2;
                p0 = p1;
            }
        } else {
            const float4 *row = rows + (size_t)(a - a_lo) * caps.vl_cap;
            auto load = [&](int base) {
                return base + lane < cnt ? __ldcs(row + base + lane) : make_float4(0.f, 0.f, 0.f, 0.f);
            };
            float4 e0 = nx.e0, e1 = nx.e1;
            for (int base = 0; base < cnt; base += 32) {
                const float4 e2 = load(base + 64);
                append(base + lane < cnt, e0.x, e0.y, e0.z, __float_as_int(e0.w));
                e0 = e1;
                e1 = e2;
            }
        }
        if (lane == 0 && over) atomicOr(err, kErrNbCap);
        if (lane < 3)
            s_sum.st[warp][lane] += lane == 0 ? (unsigned long long)(nang + nrest)
                                   : lane == 1 ? (unsigned long long)nang
                                               : (unsigned long long)((unsigned)nang * (unsigned)(nang - 1) / 2);
        if (nang > caps.ang) {
            if (lane == 0) atomicOr(err, kErrAngCap);
            nang = caps.ang;
        }
        __syncwarp();
        if constexpr (!kSh) {
            if (nang <= 32) {  // the ring's repeated entries
                if (lane <= (nang >> 1) && lane < nang) {
                    W.a_u[nang + lane] = W.a_u[lane];
                    W.a_s[nang + lane] = W.a_s[lane];
                }
                __syncwarp();
            }
        }
        const Rounds rounds(nang, nrest, nb, lane);
        const int nra = rounds.nra, nrounds = nra + ((nrest + 31) >> 5);

        // ---- 2. the descriptor
        float G0 = 0.f, G1 = 0.f;  // coefficient `lane` of [radial | angular], plain and weighted
        if constexpr (MODE != kForces) {
            float2 tail[kSh ? 1 : LR + KAT];  // left-over radial orders, then the angular ones
            reduce_orders<RB>(acc, W.red, W.coef, 0, lane);
            if constexpr (!kSh) {
#pragma unroll
                for (int q = 0; q < LR; ++q) tail[q] = acc[RB + q];
            }
            if constexpr (!kSh) {
                float2 pp[KAT], pw[KAT];
#pragma unroll
                for (int q = 0; q < KAT; ++q) pp[q] = pw[q] = dup2(0.f);
                if (nang <= 32)
                    ring_forward<KAT, EXACT>(nang, Ka, W, lane, pp, pw);
                else
                    blocks_forward<KAT, EXACT>(nang, Ka, W, lane, pp, pw);
#pragma unroll
                for (int q = 0; q < KAT; ++q) tail[LR + q] = make_float2(pp[q].x + pp[q].y, pw[q].x + pw[q].y);
                reduce_orders<LR + KAT>(tail, W.red, W.coef, RB, lane);
                __syncwarp();
                const float2 G = *reinterpret_cast<const float2 *>(W.coef + 2 * lane);
                const float two = lane >= KRT ? 2.0f : 1.0f;  // the ordered-pair sum
                G0 = lane < KRT + KAT ? two * G.x : 0.f;
                G1 = lane < KRT + KAT ? two * G.y : 0.f;
            } else {
                sh_sums(nang, W, lane);
                sh_fingerprints<KRT, KAT>(W, s_sh, W.coef, lane);
                __syncwarp();
                const float2 G = *reinterpret_cast<const float2 *>(W.coef + 2 * lane);
                const float2 w2 = *reinterpret_cast<const float2 *>(W.sh + 2 * kShComps);  // the j = k terms
                G0 = lane < KRT ? G.x : lane < KRT + KAT ? G.x - w2.x : 0.f;
                G1 = lane < KRT ? G.y : lane < KRT + KAT ? G.y - w2.y : 0.f;
            }
            __syncwarp();  // the row is written again
        }
        if constexpr (MODE == kDescriptor) {
            const int D = 2 * (Kr + Ka);
            const int k0 = lane_col<KRT, KAT>(lane, 0, Kr, Ka), k1 = lane_col<KRT, KAT>(lane, 1, Kr, Ka);
            if (k0 >= 0) G_out[(size_t)a * D + k0] = G0;
            if (k1 >= 0) G_out[(size_t)a * D + k1] = G1;
            next = __shfl_sync(kFull, next, 0);
            fetch(next);
        } else {
            // ---- 3. the network
            if constexpr (MODE == kFused) {
                wait_params();
                const float E = list_network<KRT, KAT, HB>(net, s_par + type * net.stride, W.coef, lane, G0, G1,
                                                           G_out ? G_out + (size_t)a * net.rec_len : nullptr, Kr, Ka,
                                                           c0, c1);
                if (lane == 0) {
                    s_sum.e[warp] += (double)E;
                    eatom[a] = E;
                }
            } else {  // dE/dG given
                if constexpr (kSh) sh_sums(nang, W, lane);
            }
            if (!kSh && lane >= KRT) {  // the ordered-pair sum's factor
                c0 *= 2.0f;
                c1 *= 2.0f;
            }
            if (lane < KRT + KAT) reinterpret_cast<float2 *>(W.coef)[lane] = make_float2(c0, c1);
            __syncwarp();

            // ---- 4. the chain rule: (V, B) of every angular entry
            if constexpr (kSh) {
                sh_gradients<KRT, KAT>(nang, W, coef, s_sh, lane);
            } else if (nang <= 32) {
                const float4 V = ring_backward<KAT, EXACT>(nang, Ka, W, coef + KRT, lane);
                __syncwarp();
                if (lane < nang) W.a_g[lane] = V;
            } else {
                blocks_backward<KAT, EXACT>(nang, Ka, W, coef + KRT, lane);
            }
            __syncwarp();
            next = __shfl_sync(kFull, next, 0);
            fetch(next);
            // every entry: two rounds at a time, their Clenshaw sums packed
            float fix = 0.f, fiy = 0.f, fiz = 0.f;
            const float k2 = 2.0f * inv_rcr;
            float vir[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) vir[k] = 0.f;
            for (int r = 0; r < nrounds; r += 2) {
                int ka, kb;
                const bool va = rounds.at(r, ka), vb = rounds.at(r + 1, kb);  // (none past the last round)
                float4 ea = make_float4(1.f, 0.f, 0.f, 1.f), eb = ea;
                int ja = 0, jb = 0;
                if (va) {
                    ea = W.e_d[ka];
                    ja = W.e_j[ka];
                }
                if (vb) {
                    eb = W.e_d[kb];
                    jb = W.e_j[kb];
                }
                const float2 x = make_float2(2.0f * ea.w * inv_rcr - 1.0f, 2.0f * eb.w * inv_rcr - 1.0f);
                float2 S, dS;
                clenshaw_shared<KRT, EXACT>(x, make_float2(s_tw[ja >> 28], s_tw[jb >> 28]), coef, Kr, S, dS);
                auto entry = [&](bool v, const float4 &e, int j, float S1, float dS1, int round, int k) {
                    float fc, dfc;
                    radial_cutoff(e.w, inv_rcr, fc, dfc);
                    // d/dr [T(x) f_c(r)] = T'(x) (2/R_c) f_c + T f_c'
                    float al = e.w <= B.rc_rad ? __fdividef(fmaf(dS1, k2 * fc, S1 * dfc), e.w) : 0.f;
                    float gx = 0.f, gy = 0.f, gz = 0.f;
                    if (round < nra) {  // (uniform) angular entries
                        const float4 Vg = W.a_g[v ? k : 0];
                        const float inv = rsqrtf(length2(e.x, e.y, e.z));  // as the unit vectors' 1/r
                        float sn, cs;
                        __sincosf(3.14159265358979f * (e.w * inv_rca), &sn, &cs);
                        const float be = 0.5f * (cs + 1.0f) * inv, df = -0.5f * 3.14159265358979f * inv_rca * sn;
                        const float vu = (Vg.x * e.x + Vg.y * e.y + Vg.z * e.z) * inv;
                        al = fmaf(fmaf(df, Vg.w, -be * vu), inv, al);
                        gx = be * Vg.x;
                        gy = be * Vg.y;
                        gz = be * Vg.z;
                    }
                    if (v) {  // force on the neighbour: -dE_i/dd
                        gx = fmaf(-al, e.x, -gx);
                        gy = fmaf(-al, e.y, -gy);
                        gz = fmaf(-al, e.z, -gz);
                        atomicAdd(&F4[j & kEntryIndex], make_float4(gx, gy, gz, 0.f));
                        fix -= gx;
                        fiy -= gy;
                        fiz -= gz;
                        vir[0] = fmaf(e.x, gx, vir[0]);
                        vir[1] = fmaf(e.x, gy, vir[1]);
                        vir[2] = fmaf(e.x, gz, vir[2]);
                        vir[3] = fmaf(e.y, gy, vir[3]);
                        vir[4] = fmaf(e.y, gz, vir[4]);
                        vir[5] = fmaf(e.z, gz, vir[5]);
                    }
                };
                entry(va, ea, ja, S.x, dS.x, r, ka);
                entry(vb, eb, jb, S.y, dS.y, r + 1, kb);
            }
            // the atom's own force and its virial. FP32 sums end with the atom: its virial is
            // added up in FP64, per warp or (a batch) per structure, so that the rounding
            // of the total does not grow with the atoms a warp takes.
            __syncwarp();
            const float2 sums[8] = {make_float2(fix, fiy), make_float2(fiz, 0.f), make_float2(vir[0], vir[1]),
                                    make_float2(vir[2], vir[3]), make_float2(vir[4], vir[5]),
                                    dup2(0.f), dup2(0.f), dup2(0.f)};
            const float2 t = reduce8(sums, W.red, lane);
            const int o = reduce8_order(lane);
            // (one vector atomic; three scalar ones: water 331,776 1% slower)
            const float tz = __shfl_sync(kFull, t.x, 16);  // order 1
            if (lane == 0) atomicAdd(&F4[a], make_float4(t.x, t.y, tz, 0.f));
            if ((lane & 12) == 0 && o > 1 && o < 5) {
                if constexpr (BATCH) {
                    *reinterpret_cast<float2 *>(vir_atom + (size_t)a * 6 + 2 * (o - 2)) = t;
                } else {
                    double *v = s_sum.vir[warp] + 2 * (o - 2);
                    v[0] += (double)t.x;
                    v[1] += (double)t.y;
                }
            }
        }
        __syncwarp();
        a = next;
    }

    wait_params();  // (a warp without atoms)
    // ---- the CTA's partial sums
    __syncthreads();  // every warp has left the loop
    if (tid == 0) release_work_counter(work);
    if (MODE != kForces && tid < 3) {
        unsigned long long t = 0;
        for (int w = 0; w < nw; ++w) t += s_sum.st[w][tid];
        if (t) atomicAdd(&stats[tid], t);
    }
    if constexpr (MODE != kDescriptor && !BATCH) {
        if (tid < 9) {  // the virial of an atom is symmetric: six sums
            const int ra = tid / 3, rb = tid - 3 * ra, lo = min(ra, rb), hi = max(ra, rb);
            const int k = lo == 0 ? hi : lo == 1 ? 2 + hi : 5;
            double t = 0.0;
            for (int w = 0; w < nw; ++w) t += s_sum.vir[w][k];
            vir_part[(size_t)blockIdx.x * 9 + tid] = t;
        }
    }
    if constexpr (MODE == kFused) {
        if (tid == 32 || (nw == 1 && tid == 0)) {
            double t = 0.0;
            for (int w = 0; w < nw; ++w) t += s_sum.e[w];
            e_part[blockIdx.x] = t;
        }
    }
}

}  // namespace
}  // namespace aenet
