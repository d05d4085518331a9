// hd_kernels.cu -- per-phase kernels of libhdslide (sm_103a).
//
// One step of the batched path, per replica (Kim & Falk, Sec. 2.2-2.3):
//   [k_bin, k_cellsort, k_nlist]    Verlet list rebuild, only for replicas
//                                   whose rebuild flag is set
//   k_pair{64,32}                   LJ force + energy (Eq. 9) and H.(r - r_O)
//                                   in one sweep of the list; per-tile sums
//   k_scalar                        per replica: d (Eq. 7), sigma (Eq. 5),
//                                   DeltaV_1 (Eq. 14), rigid-body force, clocks
//   k_update{64,32}                 bias force + BAOAB kicks/drifts/noise
// The quench (steepest descent / FIRE) reuses the list and pair kernels on a
// copy of the positions (k_pair<true>, k_qscalar, k_qupdate).
//
// Tiles: a CTA handles one tile = up to blockDim atoms of ONE replica, so any
// per-replica quantity is a fixed-order sum of per-tile sums (deterministic).
#include <map>
#include <mutex>
#include <utility>

#include "hd_internal.cuh"
#include "hd_launch.h"

namespace hd {

// ---------------------------------------------------------------- packed FP32x2
__device__ __forceinline__ float2 f2c(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2i(int a, int b) { return make_float2((float)a, (float)b); }
__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __fadd2_rn(a, f2neg(b)); }
__device__ __forceinline__ float2 f2fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// ---------------------------------------------------------------- reductions
// Sums NV per-thread values over the CTA in a fixed order and writes them to
// out[0..NV).  Slot `maxslot` (if >= 0) is reduced with max instead of +.
template <int NV>
__device__ __forceinline__ void cta_reduce(double (&v)[NV], double *out, int maxslot) {
    __shared__ double sm[32][NV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = (q == maxslot) ? warp_max(v[q]) : warp_sum(v[q]);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sm[w][q] = v[q];
    __syncthreads();
    if (threadIdx.x < NV) {
        const int q = threadIdx.x;
        double a = sm[0][q];
        for (int k = 1; k < nw; ++k) a = (q == maxslot) ? fmax(a, sm[k][q]) : a + sm[k][q];
        out[q] = a;
    }
    __syncthreads();
}

// Warp sums of up to four doubles in 6 additions (one each: 20): the lanes
// split between the values as they halve, so after two exchanges each holds
// a partial sum of one value.  The sum of v[q] ends in lane 8 q.  The FP64
// pipe takes a warp instruction every 16 cycles an SM, so these sums, not
// their latency, were a quarter of the pair sweep's time.
__device__ __forceinline__ double warp_sum4(double v0, double v1, double v2, double v3) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16, up2 = lane & 8;
    // lanes 0-15 keep (v0, v1), lanes 16-31 keep (v2, v3)
    const double s0 = up ? v0 : v2, s1 = up ? v1 : v3;
    const double k0 = (up ? v2 : v0) + __shfl_xor_sync(full, s0, 16), k1 = (up ? v3 : v1) + __shfl_xor_sync(full, s1, 16);
    double k = (up2 ? k1 : k0) + __shfl_xor_sync(full, up2 ? k0 : k1, 8);
    k += __shfl_xor_sync(full, k, 4);
    k += __shfl_xor_sync(full, k, 2);
    k += __shfl_xor_sync(full, k, 1);
    return k;
}

// Tile sums of the split form.  Per-atom values are FP64 (products of FP32
// factors, exact in FP64) where sigma = G / d (Eq. 5) or the sign of FIRE's
// power depends on them: sum[0..3], summed in FP64.  sf[0..nf) are FP32
// per-atom values (rigid atoms) summed in FP32 within a warp, xr the rigid
// positions, both only where some lane holds a rigid atom (few warps do).
// fm: largest of an FP32 value, or negative for none.  Warp results are
// combined in FP64 in warp order.  out: slots in the order of `slot`.
struct TileSlots {
    int sum[4], f0, x0, max;      // out index of the sums (-1: unused), first FP32 sum, first position, the maximum
};
template <int NF>
__device__ __forceinline__ void tile_reduce(double v0, double v1, double v2, double v3, const float (&sf)[NF],
                                            const double (&xr)[3], bool anyrig, float fm, TileSlots L, double *out) {
    __shared__ double sm[8][NPART];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if (lane < NPART) sm[w][lane] = 0.0;
    __syncwarp();
    const double s = warp_sum4(v0, v1, v2, v3);
    const int q = L.sum[lane >> 3];
    if ((lane & 7) == 0 && q >= 0) sm[w][q] = s;
    if (L.max >= 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fm = fmaxf(fm, __shfl_xor_sync(0xffffffffu, fm, o));
        if (lane == 0) sm[w][L.max] = (double)fm;
    }
    if (anyrig) {
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            const float a = warp_sum(sf[k]);
            if (lane == 0) sm[w][L.f0 + k] = (double)a;
        }
        const double x = warp_sum4(xr[0], xr[1], xr[2], 0.0);
        if ((lane & 7) == 0 && lane < 24) sm[w][L.x0 + (lane >> 3)] = x;
    }
    __syncthreads();
    if (threadIdx.x < NPART) {
        const int k = threadIdx.x;
        double a = sm[0][k];
        for (int m = 1; m < nw; ++m) a = k == L.max ? fmax(a, sm[m][k]) : a + sm[m][k];
        out[k] = a;
    }
    __syncthreads();
}

// ---------------------------------------------------------------- init
// Fixed-point image, r - r_O, and (where asked) Maxwell-Boltzmann velocities
// from Philox calls 2 and 3 at the current step.
__global__ void k_init(Dev D, const int *draw_vel) {
    const int t = blockIdx.x, r = D.tile_rep[t];
    if (threadIdx.x >= D.tile_n[t]) return;
    const int i = D.tile_start[t] + threadIdx.x;
    const RepDev &R = D.rep[r];
    dbl4 x = D.x[i], xo = D.xo[i];
    int4 p = D.p[i];  // w (type | role << 8) preset by the host
    p = fix_pos(R, x, p.w);
    D.p[i] = p;
    D.pfixb[i] = p;
    const int role = (p.w >> 8) & 0xff;
    if (D.prec == HD_FP64) {
        D.dr64[i] = make_dbl4(x.x - xo.x, x.y - xo.y, x.z - xo.z, 0.0);
    } else {
        D.po[i] = fix_pos(R, xo, 0);
    }
    if (draw_vel[r]) {
        double v0 = 0, v1 = 0, v2 = 0;
        if (role == ROLE_MOBILE) {
            const double sd = sqrt(R.kT);
            double z0, z1, z2, z3;
            normals64(philox_draw(D, D.st[r].step, D.orig[i], R.rep_id, 2), z0, z1);
            v0 = sd * z0;
            v1 = sd * z1;
            if (R.dim == 3) {
                normals64(philox_draw(D, D.st[r].step, D.orig[i], R.rep_id, 3), z2, z3);
                v2 = sd * z2;
            }
        }
        D.v64[i] = make_dbl4(v0, v1, v2, 0.0);
    }
}

// ---------------------------------------------------------------- neighbour list
// A list rebuild touches only the replicas whose flag is set.  rb_list[k] is
// the k-th such replica in ascending order, rb_off[k] / rb_aoff[k] its first
// cell / atom in the compacted range, rb_meta = {count, cells, atoms}.  The
// rebuild kernels run fixed grids that stride over that compacted range.  Most
// steps rebuild few replicas or none, so their launches are what a rebuild
// pass costs: every CTA of k_bin makes the plan for itself (a warp's ballots
// over the flags) instead of waiting for a launch that makes it, and the cell
// counts are cleared by the scalar kernel that retires the flag, so that they
// are zero whenever a binning starts.  With the plan and the clearing as
// launches of their own the preparation took 19.8 us of a step of 64 x 14,272
// atoms (16.8 now) and 64 quench iterations of 16 x 421 atoms 2.05 ms (1.83).
struct Plan {
    int n, cells, atoms;
};
__device__ __forceinline__ Plan rebuild_plan(const Dev &D, int *list, int *off, int *aoff) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int nrb = 0, coff = 0, ao = 0;
    for (int base = 0; base < D.nrep; base += 32) {
        const int r = base + lane;
        const bool f = r < D.nrep && D.rebuild[r] != 0;
        const unsigned m = __ballot_sync(full, f);
        if (m == 0) continue;
        const int nc = f ? D.rep[r].ncell : 0, na = f ? D.rep[r].n : 0;
        int c = nc, a = na;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int tc = __shfl_up_sync(full, c, o), ta = __shfl_up_sync(full, a, o);
            if (lane >= o) {
                c += tc;
                a += ta;
            }
        }
        if (f) {
            const int k = nrb + __popc(m & ((1u << lane) - 1u));
            list[k] = r;
            off[k] = coff + c - nc;
            aoff[k] = ao + a - na;
        }
        nrb += __popc(m);
        coff += __shfl_sync(full, c, 31);
        ao += __shfl_sync(full, a, 31);
    }
    return {nrb, coff, ao};
}

// Entry k of the compacted replicas that holds compacted index idx.
__device__ __forceinline__ int rb_find(const int *off, int n, int idx) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= idx) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void dev_bin_atom(const Dev &D, int r, int i) {
    const RepDev &R = D.rep[r];
    const int4 p = D.p[i];
    const dbl4 x = D.x[i];
    const int cx = cell_of(R, 0, x.x), cy = cell_of(R, 1, x.y), cz = cell_of(R, 2, x.z);
    D.cellid[i] = cx | (cy << 10) | (cz << 20);
    const int c = R.cell0 + (cz * R.nc[1] + cy) * R.nc[0] + cx;
    const int slot = atomicAdd(&D.cell_cnt[c], 1);
    if (slot < D.cell_cap) D.cell_atoms[(size_t)c * D.cell_cap + slot] = i;
    else set_err(D, HD_ERR_OVERFLOW, i, r);
    D.pfixb[i] = p;
}
// planned: the plan is in global memory already (k_rebuild_plan, for batches
// whose plan does not fit a CTA's shared memory).
__global__ void __launch_bounds__(256) k_bin(Dev D, bool planned) {
    extern __shared__ int pl[];
    int *list = planned ? D.rb_list : pl, *aoff = planned ? D.rb_aoff : pl + D.nrep, *off = pl + 2 * D.nrep;
    __shared__ Plan P;
    if (planned) {
        if (threadIdx.x == 0) P = {D.rb_meta[0], D.rb_meta[1], D.rb_meta[2]};
    } else if (threadIdx.x < 32) {
        const Plan p = rebuild_plan(D, list, off, aoff);
        if (threadIdx.x == 0) {
            P = p;
            if (blockIdx.x == 0) {
                D.rb_off[p.n] = p.cells;
                D.rb_aoff[p.n] = p.atoms;
                D.rb_meta[0] = p.n;
                D.rb_meta[1] = p.cells;
                D.rb_meta[2] = p.atoms;
            }
        }
    }
    __syncthreads();
    const int n = P.n, total = P.atoms;
    if (blockIdx.x == 0 && !planned)
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            D.rb_list[k] = list[k];
            D.rb_off[k] = off[k];
            D.rb_aoff[k] = aoff[k];
        }
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
        const int k = rb_find(aoff, n, idx);
        const int r = list[k];
        dev_bin_atom(D, r, D.rep[r].atom0 + idx - aoff[k]);
    }
}
__global__ void k_rebuild_plan(Dev D) {
    const Plan p = rebuild_plan(D, D.rb_list, D.rb_off, D.rb_aoff);
    if (threadIdx.x == 0) {
        D.rb_off[p.n] = p.cells;
        D.rb_aoff[p.n] = p.atoms;
        D.rb_meta[0] = p.n;
        D.rb_meta[1] = p.cells;
        D.rb_meta[2] = p.atoms;
    }
}

// The list of a replica has been used: its cells' counts go back to zero.
__device__ __forceinline__ void clear_cells(const Dev &D, const RepDev &R) {
    for (int c = threadIdx.x; c < R.ncell; c += blockDim.x) D.cell_cnt[R.cell0 + c] = 0;
}

// Each cell's atom list in ascending slot order: one warp per cell copies the
// list to shared memory and writes every entry at its rank (slot indices are
// distinct).  With atoms stored cell-major, walking the neighbour cells in
// ascending cell order then yields candidates in (almost) ascending j.
__device__ __forceinline__ void dev_cellsort_warp(const Dev &D, const RepDev &R, int c, int *buf) {
    const int lane = threadIdx.x & 31;
    int *a = D.cell_atoms + (size_t)(R.cell0 + c) * D.cell_cap;
    const int m = min(D.cell_cnt[R.cell0 + c], D.cell_cap);
    for (int k = lane; k < m; k += 32) buf[k] = a[k];
    __syncwarp();
    for (int k = lane; k < m; k += 32) {
        const int v = buf[k];
        int rank = 0;
        for (int q = 0; q < m; ++q) rank += buf[q] < v;
        a[rank] = v;
    }
    __syncwarp();
}
__global__ void __launch_bounds__(128) k_cellsort(Dev D) {
    extern __shared__ int cs_buf[];
    const int w = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    const int n = D.rb_meta[0], total = D.rb_meta[1];
    for (int idx = blockIdx.x * nwb + w; idx < total; idx += gridDim.x * nwb) {
        const int k = rb_find(D.rb_off, n, idx);
        dev_cellsort_warp(D, D.rep[D.rb_list[k]], idx - D.rb_off[k], cs_buf + w * D.cell_cap);
    }
}

// Row i = every j != i whose FP64 minimum-image squared distance is below
// (rc + skin)^2.  One CTA builds the rows of one cell's atoms.  It first
// stages the candidates of the cell's stencil (the 27, or 9 in 2-D,
// surrounding cells in ascending cell order, each cell's atoms ascending) in
// shared memory.  Then one warp per atom of the cell takes two passes.
//
// 1. All candidates (~675 in a dense 3-D crystal, of which ~76 are neighbours),
//    64 at a time: the FP32 distance, one compare, and the place of each
//    accepted candidate goes to the warp's buffer, packed by ballot.  This is
//    where the instructions are, so positions are staged as FP32 offsets from
//    the cell's centre (three packed subtractions and three packed products
//    per 64) and nothing else is decided here.  An offset is the exact integer
//    difference of the images, rounded: r^2 is good to ~1e-6, far inside the
//    2^-12 wide band that pass 2 decides exactly.  A periodic axis of three
//    cells or one has no such offsets (a neighbour may be nearer around the
//    box); a replica with one stages the images and subtracts those.
// 2. The accepted ones: the atom itself leaves, the thin band around the
//    radius takes the oracle's FP64 test operation for operation, and each j
//    gets a class: A (first shell) FP32 r^2 < rA^2, the pairs that can come
//    within the range where the pair sweep takes the exact r^2; B the rest of
//    the pairs within rc at build time; C (skin shell) the rest of the row.
//    The class decides the place in the row, and with it the order in which
//    the sweep adds up forces, so next to its two bounds it is taken from the
//    images themselves: it must not depend on which cell's centre was near.
//
// The row is then written as A | B | C, each block in candidate order, so the
// lanes of the pair sweep leave the first shell, and later the cutoff, at
// nearly the same k; a lane writes a group of four.  The row order is a
// deterministic function of the cell lists (sorted by k_cellsort); reads
// return each row ascending in j.
//
// Bound by instruction issue and the latency of the staging.
// Row-build CTA: 8 warps share one staged stencil (the cell's atoms split among them).
constexpr int NL_THREADS = 256;
// Accepted candidates a warp holds between the passes: the longest row and
// room for the atom itself and the band's candidates that pass 2 takes out.
constexpr int NL_BUF = 256;

struct NlSmem {
    int nst, tot, kc;
    int cell[27], off[28], centre[3];
};

// Shared memory of a row-build CTA: the staged candidates (x, y, z as FP32
// offsets or images; slot, top bit its type), then per warp the accepted
// candidates and the row.
__host__ __device__ inline int nl_cand(const Dev &D) { return (27 * D.cell_cap + 63) / 64 * 64; }
__host__ __device__ inline size_t nl_warp_bytes(const Dev &D) { return NL_BUF * 2 + (size_t)D.ngrp * sizeof(int4); }
struct NlStage {
    float *x, *y, *z;
    int *j;
    char *warp;
};

// FP32 r^2 of two images, from their exact integer differences
__device__ __forceinline__ float img_r2(const RepDev &R, int4 a, int4 b) {
    const int4 d = img_diff(a, b);
    const float dx = (float)d.x * R.fx_lsb[0], dy = (float)d.y * R.fx_lsb[1], dz = (float)d.z * R.fx_lsb[2];
    return dx * dx + dy * dy + dz * dz;
}

template <bool LOCAL>
__device__ __forceinline__ void dev_nlist_rows(const Dev &D, const RepDev &R, int r, int m, const NlSmem &M, const NlStage &T) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int tot = M.tot, cap = D.maxnb;
    const float lx = R.fx_lsb[0], ly = R.fx_lsb[1], lz = R.fx_lsb[2], rA2 = R.rA2f;
    const float lo = D.rl2_lo_f, hi = D.rl2_hi_f, rc2 = D.rc2_lo_f;
    unsigned short *buf = reinterpret_cast<unsigned short *>(T.warp + w * nl_warp_bytes(D));
    int *row = reinterpret_cast<int *>(buf + NL_BUF);
    // difference of two staged coordinates
    auto diff = [](float a, float b, float l) {
        return LOCAL ? a - b : (float)(int)(__float_as_uint(a) - __float_as_uint(b)) * l;
    };
    for (int a = w; a < m; a += nw) {
        const int slot = M.off[M.kc] + a;
        const float xi = T.x[slot], yi = T.y[slot], zi = T.z[slot];
        const int i = T.j[slot] & 0x7fffffff;
        int cnt = 0;
        for (int base = 0; base < tot; base += 64) {
            const int q = base + 2 * lane;
            const float2 xj = *reinterpret_cast<const float2 *>(T.x + q), yj = *reinterpret_cast<const float2 *>(T.y + q),
                         zj = *reinterpret_cast<const float2 *>(T.z + q);
            float2 dx, dy, dz;
            if (LOCAL) {
                dx = f2sub(f2c(xi), xj);
                dy = f2sub(f2c(yi), yj);
                dz = f2sub(f2c(zi), zj);
            } else {
                dx = make_float2(diff(xi, xj.x, lx), diff(xi, xj.y, lx));
                dy = make_float2(diff(yi, yj.x, ly), diff(yi, yj.y, ly));
                dz = make_float2(diff(zi, zj.x, lz), diff(zi, zj.y, lz));
            }
            const float2 r2 = f2fma(dx, dx, f2fma(dy, dy, f2mul(dz, dz)));
            // offsets past the last candidate are far away; images are not
            const bool ina = r2.x < hi && (LOCAL || q < tot), inb = r2.y < hi && (LOCAL || q + 1 < tot);
            const unsigned ma = __ballot_sync(full, ina), mb = __ballot_sync(full, inb);
            int at = cnt + __popc(ma & below) + __popc(mb & below);
            if (ina && at < NL_BUF) buf[at] = (unsigned short)q;
            at += ina;
            if (inb && at < NL_BUF) buf[at] = (unsigned short)(q + 1);
            cnt += __popc(ma) + __popc(mb);
        }
        const int have = min(cnt, NL_BUF);
        __syncwarp();
        int nA = 0, nB = 0, nC = 0;
        unsigned mixed = (unsigned)T.j[slot] >> 31;
        for (int base = 0; base < have; base += 32) {
            int cl = 3;
            const int e = base + lane;
            const int q = e < have ? buf[e] : slot;
            if (q != slot) {
                const int jt = T.j[q], j = jt & 0x7fffffff;
                const float dx = diff(xi, T.x[q], lx), dy = diff(yi, T.y[q], ly), dz = diff(zi, T.z[q], lz);
                float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (r2 < lo || exact_r2(R, D.x[i], D.x[j]) < D.rl2) {
                    if (fabsf(r2 - rA2) < rA2 * 0x1p-16f || fabsf(r2 - rc2) < rc2 * 0x1p-16f) r2 = img_r2(R, D.p[i], D.p[j]);
                    cl = r2 < rA2 ? 0 : (r2 < rc2 ? 1 : 2);
                    mixed |= (unsigned)jt >> 31;
                }
            }
            if (e < have) buf[e] = (unsigned short)(q | (cl << 14));
            nA += __popc(__ballot_sync(full, cl == 0));
            nB += __popc(__ballot_sync(full, cl == 1));
            nC += __popc(__ballot_sync(full, cl == 2));
        }
        __syncwarp();
        const int n = nA + nB + nC, kept = min(n, cap);
        int bA = 0, bB = nA, bC = nA + nB;
        for (int base = 0; base < have; base += 32) {
            const int e = base + lane;
            const int v = e < have ? buf[e] : 3 << 14, cl = v >> 14;
            const unsigned mA = __ballot_sync(full, cl == 0), mB = __ballot_sync(full, cl == 1),
                           mC = __ballot_sync(full, cl == 2);
            const int pos = cl == 0 ? bA + __popc(mA & below) : (cl == 1 ? bB + __popc(mB & below) : bC + __popc(mC & below));
            if (cl < 3 && pos < cap) row[pos] = T.j[v & 0x3fff] & 0x7fffffff;
            bA += __popc(mA);
            bB += __popc(mB);
            bC += __popc(mC);
        }
        if (kept + lane < ((kept + 3) & ~3)) row[kept + lane] = i;     // fill up the last group
        __syncwarp();
        const size_t row4 = nbr_row4(D, R, i);
        for (int g = lane; g < (kept + 3) >> 2; g += 32)
            reinterpret_cast<int4 *>(D.nbr)[row4 + 32 * (size_t)g] = reinterpret_cast<const int4 *>(row)[g];
        const bool mx = __any_sync(full, mixed != 0);
        if (lane == 0) {
            D.nnb[i] = kept | (mx ? NB_MIXED : 0);
            if (n > cap || cnt > NL_BUF) set_err(D, HD_ERR_OVERFLOW, i, r);
        }
        __syncwarp();
    }
}

__device__ __forceinline__ void dev_nlist_cell(const Dev &D, int r, int c, NlSmem &M, const NlStage &T) {
    const RepDev &R = D.rep[r];
    const int cell0 = R.cell0 + c;
    const int m = min(D.cell_cnt[cell0], D.cell_cap);
    if (m == 0) return;  // uniform: every thread reads the same count
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w == 0) {
        // lane k < 27: stencil cell (k % 3, k / 3 % 3, k / 9) of the per-axis
        // lists, each list ascending (a periodic wrap puts nc-1 after 0 and 1)
        const int ci[3] = {c % R.nc[0], (c / R.nc[0]) % R.nc[1], c / (R.nc[0] * R.nc[1])};
        int cs[3], ncs[3];
        const int pick[3] = {lane % 3, (lane / 3) % 3, lane / 9};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int nc = R.nc[a], q = pick[a];
            int list[3] = {0, 0, 0}, n = 0;
            if (nc == 1) {
                list[n++] = 0;
            } else {
                const int c0 = ci[a] - 1, c2 = ci[a] + 1;
                if (R.periodic[a]) {
                    if (c0 < 0) { list[0] = 0; list[1] = 1; list[2] = nc - 1; }
                    else if (c2 >= nc) { list[0] = 0; list[1] = nc - 2; list[2] = nc - 1; }
                    else { list[0] = c0; list[1] = ci[a]; list[2] = c2; }
                    n = 3;
                } else {
                    if (c0 >= 0) list[n++] = c0;
                    list[n++] = ci[a];
                    if (c2 < nc) list[n++] = c2;
                }
            }
            ncs[a] = n;
            cs[a] = q < n ? list[q] : 0;
        }
        const bool valid = lane < 27 && pick[0] < ncs[0] && pick[1] < ncs[1] && pick[2] < ncs[2];
        const int nst = ncs[0] * ncs[1] * ncs[2];
        const int k = valid ? (pick[2] * ncs[1] + pick[1]) * ncs[0] + pick[0] : 0;
        const int cc = R.cell0 + (cs[2] * R.nc[1] + cs[1]) * R.nc[0] + cs[0];
        if (valid) {
            M.cell[k] = cc;
            M.off[k] = min(D.cell_cnt[cc], D.cell_cap);   // the count, until the scan below
            if (cc == cell0) M.kc = k;
        }
        __syncwarp();
        // exclusive scan of the counts in stencil order
        const int cnt = lane < nst ? M.off[lane] : 0;
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        __syncwarp();
        if (lane < nst) M.off[lane] = incl - cnt;
        if (lane == nst - 1) {
            M.off[nst] = incl;
            M.tot = incl;
            M.nst = nst;
        }
        // the cell's centre in the fixed-point image
        if (lane < 3) {
            const int ca = lane == 0 ? ci[0] : (lane == 1 ? ci[1] : ci[2]);
            const double x = R.periodic[lane] ? (ca + 0.5) * (R.L[lane] / R.nc[lane]) : R.cell_lo + (ca + 0.5) / R.cell_inv_w;
            M.centre[lane] = R.periodic[lane] || lane == R.vert ? fix_coord(R, lane, x) : 0;
        }
    }
    __syncthreads();
    // stage the stencil: every thread takes candidates idx, idx + blockDim, ...,
    // four at a time so that their loads are in flight together
    {
        const int tot = M.tot, nst = M.nst;
        const bool local = R.nl_local != 0;
        const float lx = R.fx_lsb[0], ly = R.fx_lsb[1], lz = R.fx_lsb[2];
        const int cx = M.centre[0], cy = M.centre[1], cz = M.centre[2];
        for (int base = threadIdx.x; base < tot; base += 4 * blockDim.x) {
            int jj[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = base + u * blockDim.x;
                jj[u] = -1;
                if (idx < tot) {
                    int lo = 0, hi = nst - 1;          // last stencil cell with off <= idx
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (M.off[mid] <= idx) lo = mid;
                        else hi = mid - 1;
                    }
                    jj[u] = D.cell_atoms[(size_t)M.cell[lo] * D.cell_cap + (idx - M.off[lo])];
                }
            }
            int4 pp[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) pp[u] = jj[u] >= 0 ? D.p[jj[u]] : make_int4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = base + u * blockDim.x;
                if (idx < tot) {
                    const int4 p = pp[u];
                    const int ox = (int)((unsigned)p.x - (unsigned)cx), oy = (int)((unsigned)p.y - (unsigned)cy),
                              oz = (int)((unsigned)p.z - (unsigned)cz);
                    T.x[idx] = local ? (float)ox * lx : __int_as_float(p.x);
                    T.y[idx] = local ? (float)oy * ly : __int_as_float(p.y);
                    T.z[idx] = local ? (float)oz * lz : __int_as_float(p.z);
                    T.j[idx] = jj[u] | (p.w << 31);      // top bit: the type
                }
            }
        }
        // the last 64 are read whole
        for (int idx = tot + threadIdx.x; idx < (tot + 63) / 64 * 64; idx += blockDim.x) T.x[idx] = T.y[idx] = T.z[idx] = 1e18f;
    }
    __syncthreads();
    if (R.nl_local) dev_nlist_rows<true>(D, R, r, m, M, T);
    else dev_nlist_rows<false>(D, R, r, m, M, T);
    __syncthreads();  // the staging buffers are reused by the next cell
}

__device__ __forceinline__ NlStage nl_smem_carve(const Dev &D, char *base) {
    const int n = nl_cand(D);
    NlStage T;
    T.x = reinterpret_cast<float *>(base);
    T.y = T.x + n;
    T.z = T.y + n;
    T.j = reinterpret_cast<int *>(T.z + n);
    T.warp = reinterpret_cast<char *>(T.j + n);
    return T;
}

__global__ void __launch_bounds__(NL_THREADS) k_nlist(Dev D) {
    extern __shared__ __align__(16) char nl_smem[];
    __shared__ NlSmem M;
    const NlStage T = nl_smem_carve(D, nl_smem);
    const int n = D.rb_meta[0], total = D.rb_meta[1];
    for (int idx = blockIdx.x; idx < total; idx += gridDim.x) {
        const int k = rb_find(D.rb_off, n, idx);
        dev_nlist_cell(D, D.rb_list[k], idx - D.rb_off[k], M, T);
    }
}

// ---------------------------------------------------------------- pair sweep
// F_i = sum_j -phi'(r)/r r_ij; e_i = sum_j phi(r)/2;
// (H dr)_i = sum_j [A (dr_i - dr_j) + B ((dr_i - dr_j) . r_ij) r_ij],
// A = phi'/r, B = (phi'' - phi'/r)/r^2, with s = sigma_ab/r:
//   -A = 24 eps s^6 (2 s^6 - 1)/r^2,   B = 96 eps s^6 (7 s^6 - 2)/r^4.
// Q (quench): positions of the quench copy, quench partial sums.  E: per-atom
// energies.  H: the Hessian term.
// S: lanes of a warp that share one row (lane s takes groups s, s + S, ... of
// four entries, the sums meet in a shuffle tree).  A tile is cut into D.split
// units of block / split atoms, one CTA each, of S threads an atom.
template <bool Q, bool E, bool H, int S>
__device__ __forceinline__ void dev_pair64(const Dev &D, int unit) {
    const int t = unit / D.split;
    const int r = D.tile_rep[t];
    if (Q && D.st[r].q_done) return;
    const RepDev &R = D.rep[r];
    const int sub = S > 1 ? (int)(threadIdx.x % S) : 0;
    const int at = (unit % D.split) * (D.block / D.split) + (int)threadIdx.x / S;     // atom of the tile
    const bool has = at < D.tile_n[t], act = has && sub == 0;
    const int i = D.tile_start[t] + (has ? at : 0);
    const dbl4 xi = D.x[i];
    const int ti = (int)xi.w;
    const dbl4 dri = Q ? make_dbl4(0, 0, 0, 0) : D.dr64[i];
    double fx = 0, fy = 0, fz = 0, e = 0, hx = 0, hy = 0, hz = 0;
    const int nn = has ? NB_LEN(D.nnb[i]) : 0;
    const size_t row4 = nbr_row4(D, R, i);
    const double rc2 = D.rc2;
    for (int k = 4 * sub; k < nn; k += (k & 3) == 3 ? 4 * S - 3 : 1) {
        const int j = D.nbr[nbr_at(row4, k)];
        const dbl4 xj = D.x[j];
        const double dx = mi64(R, 0, xi.x - xj.x), dy = mi64(R, 1, xi.y - xj.y), dz = mi64(R, 2, xi.z - xj.z);
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (r2 < rc2) {
            const int tj = (int)xj.w;
            const double eps = R.eps[ti][tj];
            const double ir2 = 1.0 / r2;
            const double s2 = R.sig2[ti][tj] * ir2;
            const double s6 = s2 * s2 * s2;
            const double fr = 24.0 * eps * ir2 * s6 * (2.0 * s6 - 1.0);
            fx += fr * dx;
            fy += fr * dy;
            fz += fr * dz;
            if (E) e += 0.5 * (4.0 * eps * s6 * (s6 - 1.0) - R.shift[ti][tj]);
            if (H) {
                const dbl4 drj = D.dr64[j];
                const double ux = dri.x - drj.x, uy = dri.y - drj.y, uz = dri.z - drj.z;
                const double rdu = dx * ux + dy * uy + dz * uz;
                const double B = 96.0 * eps * ir2 * ir2 * s6 * (7.0 * s6 - 2.0);
                hx += -fr * ux + B * rdu * dx;
                hy += -fr * uy + B * rdu * dy;
                hz += -fr * uz + B * rdu * dz;
            }
        }
    }
    // harmonic bonds of Eq. 12, phi = k (r - r_b)^2 / 2 at any distance:
    // A = phi'/r = k (r - r_b)/r, B = (phi'' - A)/r^2 = k r_b / r^3
    if (R.nbond > 0 && act) {
        for (int b = D.bond_off[i]; b < D.bond_off[i + 1]; ++b) {
            const int j = D.bond_j[b];
            const dbl4 xj = D.x[j];
            const double dx = mi64(R, 0, xi.x - xj.x), dy = mi64(R, 1, xi.y - xj.y), dz = mi64(R, 2, xi.z - xj.z);
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double rr = sqrt(r2), db = rr - R.rbond;
            const double A = R.kbond * db / rr;
            fx -= A * dx;
            fy -= A * dy;
            fz -= A * dz;
            if (E) e += 0.5 * (0.5 * R.kbond * db * db);
            if (H) {
                const dbl4 drj = D.dr64[j];
                const double ux = dri.x - drj.x, uy = dri.y - drj.y, uz = dri.z - drj.z;
                const double rdu = dx * ux + dy * uy + dz * uz;
                const double B = (R.kbond - A) / r2;
                hx += A * ux + B * rdu * dx;
                hy += A * uy + B * rdu * dy;
                hz += A * uz + B * rdu * dz;
            }
        }
    }
    if (S > 1) {
#pragma unroll
        for (int o = 1; o < S; o <<= 1) {
            fx += __shfl_xor_sync(0xffffffffu, fx, o);
            fy += __shfl_xor_sync(0xffffffffu, fy, o);
            fz += __shfl_xor_sync(0xffffffffu, fz, o);
            if (E) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (H) {
                hx += __shfl_xor_sync(0xffffffffu, hx, o);
                hy += __shfl_xor_sync(0xffffffffu, hy, o);
                hz += __shfl_xor_sync(0xffffffffu, hz, o);
            }
        }
    }
    const int role = act ? ((D.p[i].w >> 8) & 0xff) : -1;
    if (H && role == ROLE_RIGID) {
        hx += R.kr_n * dri.x;
        if (R.dim == 3) hy += R.kr_n * dri.y;
    }
    if (act) {
        D.f64[i] = make_dbl4(fx, fy, fz, e);
        if (H) D.h64[i] = make_dbl4(hx, hy, hz, 0.0);
    }
    const bool rig = role == ROLE_RIGID;
    if (!Q) {
        double v[NPART] = {};
        if (act) {
            v[PART_D2] = dri.x * dri.x + dri.y * dri.y + dri.z * dri.z;
            v[PART_G] = -(fx * dri.x + fy * dri.y + fz * dri.z);
            v[PART_V] = e;
        }
        if (rig) {
            v[PART_FRIG] = fx; v[PART_FRIG + 1] = fy; v[PART_FRIG + 2] = fz;
            v[PART_HRIG] = hx; v[PART_HRIG + 1] = hy; v[PART_HRIG + 2] = hz;
            v[PART_DRRIG] = dri.x; v[PART_DRRIG + 1] = dri.y; v[PART_DRRIG + 2] = dri.z;
            v[PART_XRIG] = xi.x; v[PART_XRIG + 1] = xi.y; v[PART_XRIG + 2] = xi.z;
        }
        cta_reduce<NPART>(v, D.part + (size_t)unit * NPART, -1);
    } else {
        double v[QPART] = {};
        if (role == ROLE_MOBILE) {
            const dbl4 vv = D.v64[i];
            v[QP_FMAX2] = fx * fx + fy * fy + fz * fz;
            v[QP_P] = fx * vv.x + fy * vv.y + fz * vv.z;
            v[QP_VV] = vv.x * vv.x + vv.y * vv.y + vv.z * vv.z;
            v[QP_FF] = v[QP_FMAX2];
        }
        if (rig) {
            v[QP_FRIG] = fx; v[QP_FRIG + 1] = fy; v[QP_FRIG + 2] = fz;
            v[QP_XRIG] = xi.x; v[QP_XRIG + 1] = xi.y; v[QP_XRIG + 2] = xi.z;
        }
        cta_reduce<QPART>(v, D.part + (size_t)unit * NPART, QP_FMAX2);
    }
}

// ---- split form
// Positions are differenced exactly in 32-bit fixed point, the pair
// arithmetic is FP32, per-tile sums are carried in FP64.
//
// Near the LJ minimum the force holds the cancelling factor w = 2 s^6 - 1; it
// is evaluated as t (3 + 3 t + t^2) with t = (r_0^2 - r^2) / r^2.  Where
// |t| < 1/4, and the FP32 r^2 would cost w its relative accuracy, r^2 is taken
// exactly, as hi + lo, from the integer separations; elsewhere the FP32 r^2
// gives w to a few ulps.  The row builder puts the pairs that can need the
// exact r^2 at the head of each row, so a warp leaves that form after its
// first groups of four.  With c = 2 s^6 = (1 + t)^3 the force is 12 eps c w /
// r^2 r_ij and the Hessian term -f u + 12 eps c (14 c - 8) (r.u) / r^4 r_ij.
//
// With a lane to a row, what its entries give is added up one after another,
// in the row's order, whichever entries share a packed instruction: a force is
// then a function of the row alone, to the last bit.  It matters because the
// LJ force jumps by 0.04 where it is cut at rc: where two trajectories part by
// rounding (~1e-8 in positions), a pair that close to rc is cut a step sooner
// in one of them and positions part by 1e-6 a step (a replica of 14,272 atoms
// meets such a pair in one of ten runs of 40 steps).  Packed sums and lengths
// in units of the fixed point, which round otherwise, did that: a step of 64 x
// 14,272 atoms took 307 us with them and takes 315.  Four lanes to a row (small
// batches) add up their own entries and meet in a tree; keeping the order there
// too, through shared memory, made a step of 8 x 1,983 atoms 57.5 us for 53.8.
//
// The sweep is bound by instruction issue (and next by the L1 wavefronts of
// its gathers), so it is laid out to spend few instructions per list entry:
// four list entries are one 16-byte load, the row's position in the list is an
// immediate offset, the neighbour's record is 16 bytes, two entries at a time
// go through packed FP32x2 arithmetic (the same roundings as one by one); and
// r - r_O of a pair is its separation minus that of the two r_O's images, so
// only the Hessian term reads a second record.
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// 1/x to FP32 rounding: the hardware approximation refined by one Newton
// step, y + y (1 - x y), so that its error carries no bias into the forces
// (an unrefined approximation shifts every pair force the same way, and the
// slope sigma of Eq. 5 sums them over the whole replica).
__device__ __forceinline__ float2 rcp_refined(float2 x) {
    const float2 y = make_float2(rcp_approx(x.x), rcp_approx(x.y));
    return f2fma(y, f2fma(f2neg(x), y, f2c(1.f)), y);
}

// What two entries of a row give: force factor, Hessian factor and r - r_O of
// the pair, energy.
struct PairTerms {
    float2 fr, B, ux, uy, uz, ee;
};

// S, unit: as in dev_pair64.
template <bool Q, bool E, bool H, int S>
__device__ __forceinline__ void dev_pair32(const Dev &D, int unit) {
    const int t = unit / D.split;
    const int r = D.tile_rep[t];
    if (Q && D.st[r].q_done) return;
    const RepDev &R = D.rep[r];
    const int sub = S > 1 ? (int)(threadIdx.x % S) : 0;
    const int at = (unit % D.split) * (D.block / D.split) + (int)threadIdx.x / S;     // atom of the tile
    const bool act = at < D.tile_n[t];
    const int i = D.tile_start[t] + (act ? at : 0);
    const int4 pi = D.p[i];
    const int4 poi = H ? D.po[i] : make_int4(0, 0, 0, 0);
    const int ti = pi.w & 1;
    const float lx = R.fx_lsb[0], ly = R.fx_lsb[1], lz = R.fx_lsb[2];
    // 12 eps as FP32 hi + lo: an eps such as 0.2 is not an FP32 number, and
    // its rounding would scale every such pair force alike
    const float a0 = R.eps12f[ti][0], a1 = R.eps12f[ti][1], al0 = R.eps12l[ti][0], al1 = R.eps12l[ti][1];
    const float q0h = R.r0sq_hi[ti][0], q1h = R.r0sq_hi[ti][1], q0l = R.r0sq_lo[ti][0], q1l = R.r0sq_lo[ti][1];
    const float rc_lo = D.rc2_lo_f, rc_hi = D.rc2_hi_f;
    const bool exact = R.exact_r2 != 0;
    // the rounding of the fixed-point unit, undone in r^2 (all axes share it
    // when they share the unit)
    const float corr = exact ? 2.f * R.lsb_rel[0] : 0.f;
    const int len = act ? D.nnb[i] : 0, nn = NB_LEN(len);
    const bool mix = __any_sync(0xffffffffu, (len & NB_MIXED) != 0);
    // In stages without branches.  An entry outside the cutoff (or past the
    // row's end) takes part at r^2 = 3e38, where every product below is zero.
    // MIX: some lane's row or atom is of the tip; without one the parameters
    // are the substrate's and nothing is selected.  vote: the whole warp is
    // here, and takes the exact r^2 if one of its lanes needs it.
    constexpr float FAR = 3.0e38f;
    auto two = [&](bool vote, bool mix, int4 pa, int4 pb, int4 poa, int4 pob, int ixa, int ixb, int iya, int iyb, int iza,
                   int izb, float2 dx, float2 dy, float2 dz, float2 r2, PairTerms &o) {
        const bool ta = mix && (pa.w & 1), tb = mix && (pb.w & 1);
        const float2 r0h = make_float2(ta ? q1h : q0h, tb ? q1h : q0h), r0l = make_float2(ta ? q1l : q0l, tb ? q1l : q0l);
        const float2 r2c = f2fma(r2, f2c(corr), r2);
        float2 ir2 = rcp_refined(r2c);
        float2 tt = f2mul(f2add(f2sub(r0h, r2c), r0l), ir2);
        const bool na = exact && r2.x < FAR && fabsf(tt.x) < 0.25f, nb = exact && r2.y < FAR && fabsf(tt.y) < 0.25f;
        if (vote ? __any_sync(0xffffffffu, na || nb) : (na || nb)) {
            float ha, la, hb, lb;
            r2_split(R, ixa, iya, iza, ha, la);
            r2_split(R, ixb, iyb, izb, hb, lb);
            const float2 h = make_float2(ha, hb), ih = rcp_refined(h);
            const float2 th = f2mul(f2add(f2sub(r0h, h), f2sub(r0l, make_float2(la, lb))), ih);
            ir2 = make_float2(na ? ih.x : ir2.x, nb ? ih.y : ir2.y);
            tt = make_float2(na ? th.x : tt.x, nb ? th.y : tt.y);
        }
        const float2 c1 = f2add(tt, f2c(1.f));
        const float2 c = f2mul(f2mul(c1, c1), c1);                               // 2 s^6
        const float2 w = f2mul(tt, f2fma(tt, f2add(tt, f2c(3.f)), f2c(3.f)));    // 2 s^6 - 1
        const float2 eh = make_float2(ta ? a1 : a0, tb ? a1 : a0), el = make_float2(ta ? al1 : al0, tb ? al1 : al0);
        const float2 pf = f2mul(f2mul(ir2, c), w);
        o.fr = f2fma(pf, el, f2mul(pf, eh));
        if (E) {
            const float sa = 0.5f * c.x, sb = 0.5f * c.y;
            const float ea = fmaf(4.f * R.epsf[ti][ta] * sa, sa - 1.f, -R.shiftf[ti][ta]);
            const float eb = fmaf(4.f * R.epsf[ti][tb] * sb, sb - 1.f, -R.shiftf[ti][tb]);
            o.ee = make_float2(r2.x < FAR ? ea : 0.f, r2.y < FAR ? eb : 0.f);
        }
        if (H) {
            o.ux = f2mul(f2i(ixa - (int)((unsigned)poi.x - (unsigned)poa.x), ixb - (int)((unsigned)poi.x - (unsigned)pob.x)), f2c(lx));
            o.uy = f2mul(f2i(iya - (int)((unsigned)poi.y - (unsigned)poa.y), iyb - (int)((unsigned)poi.y - (unsigned)pob.y)), f2c(ly));
            o.uz = f2mul(f2i(iza - (int)((unsigned)poi.z - (unsigned)poa.z), izb - (int)((unsigned)poi.z - (unsigned)pob.z)), f2c(lz));
            const float2 rdu = f2fma(dx, o.ux, f2fma(dy, o.uy, f2mul(dz, o.uz)));
            const float2 pb2 = f2mul(f2mul(f2mul(f2mul(ir2, ir2), c), f2fma(c, f2c(14.f), f2c(-8.f))), rdu);
            o.B = f2fma(pb2, el, f2mul(pb2, eh));
        }
    };
    auto sep = [](int a, int b) { return (int)((unsigned)a - (unsigned)b); };
    float fx = 0.f, fy = 0.f, fz = 0.f, e = 0.f, hx = 0.f, hy = 0.f, hz = 0.f;
    float2 Fx = make_float2(0.f, 0.f), Fy = Fx, Fz = Fx, Hx = Fx, Hy = Fx, Hz = Fx;     // four lanes: packed sums
    auto add = [&](float fr, float B, float ux, float uy, float uz, float ee, float dx, float dy, float dz) {
        fx = fmaf(fr, dx, fx);
        fy = fmaf(fr, dy, fy);
        fz = fmaf(fr, dz, fz);
        if (E) e = fmaf(0.5f, ee, e);
        if (H) {
            hx = fmaf(-fr, ux, fmaf(B, dx, hx));
            hy = fmaf(-fr, uy, fmaf(B, dy, hy));
            hz = fmaf(-fr, uz, fmaf(B, dz, hz));
        }
    };
    bool band = false;
    const int ngroup = (nn + 3) >> 2;
    int itmax = (ngroup - sub + S - 1) / S;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) itmax = max(itmax, __shfl_xor_sync(0xffffffffu, itmax, o));
    const int4 *row = reinterpret_cast<const int4 *>(D.nbr) + nbr_row4(D, R, i) + 32 * sub;
    int4 J = make_int4(i, i, i, i);
    if (sub < ngroup) J = row[0];
    for (int it = 0; it < itmax; ++it) {
        const int left = nn - 4 * (sub + S * it);         // entries of this lane from here on
        const int j4[4] = {J.x, J.y, J.z, J.w};
        int4 p4[4], po4[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) p4[u] = D.p[j4[u]];   // the builder fills a row's last group up with i
#pragma unroll
        for (int u = 0; u < 4; ++u) po4[u] = H ? D.po[j4[u]] : make_int4(0, 0, 0, 0);
        row += 32 * S;
        if (left > 4 * S) J = *row;
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
            const int ixa = sep(pi.x, p4[u].x), iya = sep(pi.y, p4[u].y), iza = sep(pi.z, p4[u].z);
            const int ixb = sep(pi.x, p4[u + 1].x), iyb = sep(pi.y, p4[u + 1].y), izb = sep(pi.z, p4[u + 1].z);
            const float2 dx = f2mul(f2i(ixa, ixb), f2c(lx)), dy = f2mul(f2i(iya, iyb), f2c(ly)),
                         dz = f2mul(f2i(iza, izb), f2c(lz));
            float2 r2 = f2fma(dx, dx, f2fma(dy, dy, f2mul(dz, dz)));
            const bool ina = u < left && r2.x < rc_lo, inb = u + 1 < left && r2.y < rc_lo;
            band |= (u < left && r2.x < rc_hi && !ina) || (u + 1 < left && r2.y < rc_hi && !inb);
            r2.x = ina ? r2.x : FAR;
            r2.y = inb ? r2.y : FAR;
            if (!__any_sync(0xffffffffu, ina || inb)) continue;      // the skin shell
            PairTerms o;
            if (mix) two(true, true, p4[u], p4[u + 1], po4[u], po4[u + 1], ixa, ixb, iya, iyb, iza, izb, dx, dy, dz, r2, o);
            else two(true, false, p4[u], p4[u + 1], po4[u], po4[u + 1], ixa, ixb, iya, iyb, iza, izb, dx, dy, dz, r2, o);
            if (S == 1) {
                add(o.fr.x, o.B.x, o.ux.x, o.uy.x, o.uz.x, o.ee.x, dx.x, dy.x, dz.x);
                add(o.fr.y, o.B.y, o.ux.y, o.uy.y, o.uz.y, o.ee.y, dx.y, dy.y, dz.y);
            } else {
                Fx = f2fma(o.fr, dx, Fx);
                Fy = f2fma(o.fr, dy, Fy);
                Fz = f2fma(o.fr, dz, Fz);
                if (E) e = fmaf(0.5f, o.ee.y, fmaf(0.5f, o.ee.x, e));
                if (H) {
                    const float2 nfr = f2neg(o.fr);
                    Hx = f2fma(nfr, o.ux, f2fma(o.B, dx, Hx));
                    Hy = f2fma(nfr, o.uy, f2fma(o.B, dy, Hy));
                    Hz = f2fma(nfr, o.uz, f2fma(o.B, dz, Hz));
                }
            }
        }
    }
    if (S > 1) {
        fx = Fx.x + Fx.y; fy = Fy.x + Fy.y; fz = Fz.x + Fz.y;
        hx = Hx.x + Hx.y; hy = Hy.x + Hy.y; hz = Hz.x + Hz.y;
    }
    // Rare: pairs in a thin band around rc are cut by the oracle's FP64 test
    // (same operations), so no pair is cut at a different step than in FP64.
    if (band) {
        const dbl4 xi64 = D.x[i];
        const size_t row4 = nbr_row4(D, R, i);
        const int4 zero = make_int4(0, 0, 0, 0);
        for (int k = 4 * sub; k < nn; k += (k & 3) == 3 ? 4 * S - 3 : 1) {
            const int j = D.nbr[nbr_at(row4, k)];
            const int4 pj = D.p[j];
            const int ix = sep(pi.x, pj.x), iy = sep(pi.y, pj.y), iz = sep(pi.z, pj.z);
            const float dx = (float)ix * lx, dy = (float)iy * ly, dz = (float)iz * lz;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            if (r2 >= rc_lo && r2 < rc_hi && exact_r2(R, xi64, D.x[j]) < D.rc2) {
                PairTerms o;
                two(false, true, pj, zero, H ? D.po[j] : zero, zero, ix, 0, iy, 0, iz, 0, make_float2(dx, 0.f),
                    make_float2(dy, 0.f), make_float2(dz, 0.f), make_float2(r2, FAR), o);
                add(o.fr.x, o.B.x, o.ux.x, o.uy.x, o.uz.x, o.ee.x, dx, dy, dz);
            }
        }
    }
    if (S > 1) {
#pragma unroll
        for (int o = 1; o < S; o <<= 1) {
            fx += __shfl_xor_sync(0xffffffffu, fx, o);
            fy += __shfl_xor_sync(0xffffffffu, fy, o);
            fz += __shfl_xor_sync(0xffffffffu, fz, o);
            if (E) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (H) {
                hx += __shfl_xor_sync(0xffffffffu, hx, o);
                hy += __shfl_xor_sync(0xffffffffu, hy, o);
                hz += __shfl_xor_sync(0xffffffffu, hz, o);
            }
        }
    }
    const bool own = act && sub == 0;
    const int4 dfi = Q ? make_int4(0, 0, 0, 0) : img_diff(pi, H ? poi : D.po[i]);
    const float4 dri = make_float4((float)dfi.x * lx, (float)dfi.y * ly, (float)dfi.z * lz, 0.f);
    // harmonic bonds of Eq. 12 at any distance, from the exact r^2 where the
    // axes share one unit (r - r_b is a small difference of two numbers near
    // r_b); A = k (r - r_b)/r, B = k r_b / r^3
    if (R.nbond > 0 && own) {
        for (int b = D.bond_off[i]; b < D.bond_off[i + 1]; ++b) {
            const int j = D.bond_j[b];
            const int4 pj = D.p[j];
            const int ix = (int)((unsigned)pi.x - (unsigned)pj.x);
            const int iy = (int)((unsigned)pi.y - (unsigned)pj.y);
            const int iz = (int)((unsigned)pi.z - (unsigned)pj.z);
            const float dx = (float)ix * lx, dy = (float)iy * ly, dz = (float)iz * lz;
            float r2h = fmaf(dx, dx, fmaf(dy, dy, dz * dz)), r2l = 0.f;
            if (exact) r2_split(R, ix, iy, iz, r2h, r2l);
            const float rh = sqrtf(r2h);
            const float rr = rh + (fmaf(-rh, rh, r2h) + r2l) * (0.5f / rh);
            const float db = (rr - R.rbond_hi) - R.rbond_lo;
            const float ir = 1.f / rr;
            const float A = R.kbondf * db * ir;
            fx = fmaf(-A, dx, fx);
            fy = fmaf(-A, dy, fy);
            fz = fmaf(-A, dz, fz);
            if (E) e = fmaf(0.25f * R.kbondf * db, db, e);
            if (H) {
                const int4 poj = D.po[j];
                const float ux = (float)(int)((unsigned)ix - ((unsigned)poi.x - (unsigned)poj.x)) * lx;
                const float uy = (float)(int)((unsigned)iy - ((unsigned)poi.y - (unsigned)poj.y)) * ly;
                const float uz = (float)(int)((unsigned)iz - ((unsigned)poi.z - (unsigned)poj.z)) * lz;
                const float rdu = fmaf(dx, ux, fmaf(dy, uy, dz * uz));
                const float B = (R.kbondf - A) * ir * ir * rdu;
                hx = fmaf(A, ux, fmaf(B, dx, hx));
                hy = fmaf(A, uy, fmaf(B, dy, hy));
                hz = fmaf(A, uz, fmaf(B, dz, hz));
            }
        }
    }
    // undo the FP32 rounding of the per-axis fixed-point unit (uniform per axis)
    fx = fmaf(fx, R.lsb_rel[0], fx);
    fy = fmaf(fy, R.lsb_rel[1], fy);
    fz = fmaf(fz, R.lsb_rel[2], fz);
    const int role = own ? ((pi.w >> 8) & 0xff) : -1;
    if (H && role == ROLE_RIGID) {
        hx += R.kr_nf * dri.x;
        if (R.dim == 3) hy += R.kr_nf * dri.y;
    }
    if (own) {
        D.f32[i] = make_float4(fx, fy, fz, e);
        if (H) D.h32[i] = make_float4(hx, hy, hz, 0.f);
    }
    const bool rig = role == ROLE_RIGID;
    const bool anyrig = __any_sync(0xffffffffu, rig);
    double xr[3] = {0.0, 0.0, 0.0};
    if (rig) {
        const dbl4 xi = D.x[i];
        xr[0] = xi.x; xr[1] = xi.y; xr[2] = xi.z;
    }
    double *out = D.part + (size_t)unit * NPART;
    if (!Q) {
        float v[9] = {};
        double d2 = 0.0, g = 0.0;
        if (own) {
            const double rx = dri.x, ry = dri.y, rz = dri.z;
            d2 = rx * rx + ry * ry + rz * rz;
            g = -((double)fx * rx + (double)fy * ry + (double)fz * rz);
        }
        if (rig) {
            v[0] = fx; v[1] = fy; v[2] = fz;
            v[3] = hx; v[4] = hy; v[5] = hz;
            v[6] = dri.x; v[7] = dri.y; v[8] = dri.z;
        }
        const TileSlots L = {{PART_D2, PART_G, PART_V, -1}, PART_FRIG, PART_XRIG, -1};
        tile_reduce<9>(d2, g, E && own ? (double)e : 0.0, 0.0, v, xr, anyrig, -1.f, L, out);
    } else {
        float v[3] = {}, fm = 0.f;
        double pw = 0.0, vv2 = 0.0, ff = 0.0;
        if (role == ROLE_MOBILE) {
            const float4 vv = D.v32[i];
            fm = fx * fx + fy * fy + fz * fz;
            const double gx = fx, gy = fy, gz = fz, ux = vv.x, uy = vv.y, uz = vv.z;
            pw = gx * ux + gy * uy + gz * uz;
            vv2 = ux * ux + uy * uy + uz * uz;
            ff = gx * gx + gy * gy + gz * gz;
        }
        if (rig) {
            v[0] = fx; v[1] = fy; v[2] = fz;
        }
        const TileSlots L = {{QP_P, QP_VV, QP_FF, -1}, QP_FRIG, QP_XRIG, QP_FMAX2};
        tile_reduce<3>(pw, vv2, ff, 0.0, v, xr, anyrig, fm, L, out);
    }
}

template <bool Q, bool E, bool H, int S>
__global__ void __launch_bounds__(256) k_pair64(Dev D) { dev_pair64<Q, E, H, S>(D, blockIdx.x); }
// The Hessian term only for the replicas expected to need it (see
// expect_slope).  Both kinds share the launch: an FP64 sweep is as long as one
// row takes until the batch fills the chip twice, so two sweeps one after the
// other took twice that (100 x 113 atoms, some in their band: 105 us a step, 74
// now; all in their band 79 and 73; 4 x 14,272 atoms, one in its band: 9.5 and
// 8.3 ms for 20 steps).
template <int S>
__global__ void __launch_bounds__(256) k_pair64_lazy(Dev D) {
    if (D.sc[D.tile_rep[blockIdx.x / D.split]].need_h) dev_pair64<false, false, true, S>(D, blockIdx.x);
    else dev_pair64<false, false, false, S>(D, blockIdx.x);
}

// Which replicas a split-form MD sweep covers: all of them; those that go
// without the Hessian term (k_pair_hot sweeps the others: the sweep without it
// runs in 64 registers, with it in 80).
enum { SWEEP_ALL = 0, SWEEP_PLAIN = 1 };
template <bool Q, bool E, bool H, int S>
__global__ void __launch_bounds__(256, H ? 3 : 4) k_pair32(Dev D, int sweep) {
    if (sweep == SWEEP_PLAIN && D.sc[D.tile_rep[blockIdx.x / D.split]].need_h) return;
    dev_pair32<Q, E, H, S>(D, blockIdx.x);
}

// Sweeps with the Hessian term over the listed replicas only; true in the
// last CTA to finish (all others' results visible to it).  The list is empty
// in most steps, so the grid is a fixed few CTAs an SM that stride over the
// listed tiles.  (In the split form only batches of one lane a row get here.)
// A CTA looks for its tiles 32 replicas at a time, every warp alike: with one
// replica after another, a step of 3,900 x 113 atoms that were all listed took
// 1,347 us.
template <int PREC, int S>
__device__ __forceinline__ bool sweep_listed(const Dev &D, const int *list, int n, unsigned *ticket) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    int pos = blockIdx.x, base = 0;       // place in the listed replicas' tiles, one after another
    for (int q0 = 0; q0 < n; q0 += 32) {
        int mine = 0, t0 = 0;
        if (q0 + lane < n) {
            const RepDev &R = D.rep[list[q0 + lane]];
            mine = R.ntile * D.split;
            t0 = R.tile0 * D.split;
        }
        int upto = mine;                  // tiles of the replicas up to this lane's
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(full, upto, o);
            if (lane >= o) upto += u;
        }
        const int all = __shfl_sync(full, upto, 31);
        t0 -= upto - mine;
        for (; pos < base + all; pos += gridDim.x) {
            const int k = __ffs(__ballot_sync(full, upto > pos - base)) - 1;
            const int unit = __shfl_sync(full, t0, k) + pos - base;
            if (PREC == HD_FP64) dev_pair64<false, false, true, S>(D, unit);
            else dev_pair32<false, false, true, S>(D, unit);
        }
        base += all;
    }
    __shared__ unsigned s_tick;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_tick = atomicAdd(ticket, 1u);
    }
    __syncthreads();
    if (s_tick != gridDim.x - 1) return false;
    __threadfence();
    return true;
}

// The replicas of the split form predicted to need the Hessian term (h_meta[0] of them).
__global__ void __launch_bounds__(256, 3) k_pair_hot(Dev D) {
    const int n = D.h_meta[0];
    if (n == 0) return;
    if (sweep_listed<HD_FP32_SPLIT, 1>(D, D.h_list, n, (unsigned *)D.h_meta + 2) && threadIdx.x == 0) {
        D.h_meta[0] = 0;
        D.h_meta[2] = 0;
    }
}

// ---------------------------------------------------------------- per-replica scalars
// Gathers the replica's tile sums (warp q sums slot q over the tiles in a
// fixed order) and evaluates, in FP64:
//   x_T = centre of the rigid layer, spring/load gradient gs;
//   G = grad V . dr (LJ part + gs . sum_rigid dr / n_rig);
//   d = sqrt(sum dr^2) (Eq. 7), sigma = G / d (Eq. 5), DeltaV_1 (Eq. 14);
//   bias coefficients: F_tot = F + ca (H dr - F) + cb dr, ca = -DeltaV'/d,
//   cb = DeltaV' sigma / d^2 (from grad sigma = (H dr + g)/d - sigma dr/d^2);
//   rigid-body force = sum_rigid F - gs - DeltaV' sum_rigid grad sigma;
//   body kicks and the clocks: t_h += dt exp(DeltaV / kT) (Eq. 3).
// need_hess: the caller has no H.dr of this configuration; with DeltaV' != 0
// nothing is changed then and the result is false.  ksum: the mobile atoms'
// kinetic energy, or null to leave S.K as it is.
//
// One warp evaluates it (every lane calls; S and C may be in shared or global
// memory): lane a < 3 holds axis a.  The chain of FP64 operations is all of
// its time, so it is kept short: one square root and one division (1/d), the
// other quotients by reciprocals that the host set, the exponential only
// inside the band (its value at DeltaV_max is the host's, at 0 it is 1).  With
// one thread for all of it, 22 divisions one after another, a step of 16 x 421
// atoms in one launch took 30.8 us; with the warp it took 19.3, and the kernel of
// 8 x 1,983 atoms 13 us where it took 21.
__device__ bool scalar_eval(const Dev &D, int r, int mode, const double *acc, const double *ksum, RepState &S, Scal &C,
                            bool need_hess = false) {
    const unsigned full = 0xffffffffu;
    const RepDev &R = D.rep[r];
    const int lane = threadIdx.x & 31, a = lane < 3 ? lane : 2;
    const int dim = R.dim, vert = R.vert;
    const bool rig = R.nrig > 0, mine = lane < 3;
    const double inr = R.inv_nrig, h = D.dt, k = R.kspring, fn = R.fnormal;
    const long long step = S.step;
    const double vb0 = S.vbody[a], xs = slider_x(R, step, h);
    const bool spring = a == 0 || (a == 1 && dim == 3);           // else the load, on the vertical axis
    const double xT = rig ? acc[PART_XRIG + a] * inr : 0.0;
    const double off = xT - (a == 0 ? xs : R.slider[1]);
    const double gs = !rig ? 0.0 : (a == vert ? fn : (spring ? k * off : 0.0));
    auto sum3 = [&](double v) { return (__shfl_sync(full, v, 0) + __shfl_sync(full, v, 1)) + __shfl_sync(full, v, 2); };
    const double gd = sum3(gs * acc[PART_DRRIG + a]);
    const double ext = sum3(!rig ? 0.0 : (a == vert ? fn * xT : (spring ? 0.5 * k * off * off : 0.0)));
    const double G = acc[PART_G] + (rig ? gd * inr : 0.0);
    const double d = sqrt(acc[PART_D2]), id = d > 0.0 ? 1.0 / d : 0.0;
    const double sig = G * id;
    double dV = 0.0, dVp = 0.0, dVe = 0.0, d1 = 0.0, d2 = 0.0;
    if (D.bias_on) dv1(R, sig, dV, dVp);
    d1 = dV;
    if (D.bias_on && R.eig_on) {
        // Eq. 13: DeltaV = DeltaV_1 + DeltaV_2 - DeltaV_1 DeltaV_2 / DeltaV_max
        double dvp1 = dVp, dvp2 = 0.0;
        dv2(R, S.eig, d2, dvp2);
        if (R.dvmax > 0.0) {
            dV = d1 + d2 - d1 * d2 / R.dvmax;
            dVp = (1.0 - d2 / R.dvmax) * dvp1;
            dVe = (1.0 - d1 / R.dvmax) * dvp2;
        } else {
            dV = dVp = dVe = 0.0;
        }
    }
    if (need_hess && dVp != 0.0) return false;
    const double ca = -dVp * id, cb = dVp * sig * (id * id);
    double fb = 0.0;
    if (rig) {
        const double F = acc[PART_FRIG + a];
        const double srig = (acc[PART_HRIG + a] + (gs - F)) * id - sig * acc[PART_DRRIG + a] * (id * id);
        fb = F - gs - (dVp != 0.0 ? dVp * srig : 0.0);
    }
    if (dVe != 0.0 && rig) {
        // the rigid layer's share of -dDeltaV/depsilon grad epsilon, summed per tile
        double e = 0.0;
        for (int t = R.tile0; t < R.tile0 + R.ntile; ++t) e += D.epart[(size_t)t * 4 + a];
        fb -= dVe * e;
    }
    // the rigid body
    const double kick = rig && a < dim ? 0.5 * h * fb * inr : 0.0;
    double vb = vb0, vfull = S.vbody_full[a];
    if (mode & MODE_CLOSE) {
        vb += kick;
        vfull = vb;
    }
    const double vmid = vb;
    if (mode & MODE_OPEN) vb += kick;
    const double v2 = sum3(vfull * vfull);
    double boost = 1.0;
    if (mode & MODE_OPEN) boost = dV == 0.0 ? 1.0 : (dV == R.dvmax ? R.boost_max : exp(dV * R.beta));
    __syncwarp();                       // every lane has read S
    if (mine) {
        C.xT[a] = xT;
        C.fbody[a] = fb;
        C.vb_mid[a] = vmid;
        C.vb_new[a] = vb;
        S.vbody[a] = vb;
        S.vbody_full[a] = vfull;
    }
    if (lane == 0) {
        C.ce = -dVe;
        C.dV1 = d1;
        C.dV2 = d2;
        C.d = d; C.sigma = sig; C.dV = dV; C.dVp = dVp; C.G = G;
        C.Vlj = acc[PART_V];
        C.V = acc[PART_V] + ext;
        C.FR = k * (xs - xT);
        C.xS = xs;
        C.ca = ca; C.cb = cb;
        C.step_cur = step;
        if (mode & MODE_OPEN) {
            // Eq. 3
            S.t_h += h * boost;
            S.t_md += h;
            S.step = step + 1;
            S.n_dv[dV <= 0.0 ? 0 : (dV >= R.dvmax ? 2 : 1)] += 1;
        }
        if (ksum) S.K = *ksum + 0.5 * (double)R.nrig * v2;
    }
    __syncwarp();
    return true;
}

// Sums of one replica's tile parts into acc[0..NPART) and of its kinetic parts
// into acc[NPART].  A warp reads two parts (256 bytes) at a time, lane l slot
// l % 16, and every warp takes every nw-th pair, so the loads are coalesced and
// each lane adds its own slot; the warps' sums meet in shared memory in warp
// order.  The order is a function of the block size alone.  MAXSLOT is reduced
// with max (-1: none).  K: the kinetic parts are wanted.
template <int MAXSLOT, bool K = true>
__device__ __forceinline__ void dev_scalar_acc(const Dev &D, int r, double *acc) {
    __shared__ double sm[17][NPART + 1];
    const RepDev &R = D.rep[r];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5, slot = lane & 15;
    const int p0 = R.tile0 * D.split, np = R.ntile * D.split;
    const bool mx = slot == MAXSLOT;
    double v = 0.0, k = 0.0;
    const double *p = D.part + (size_t)p0 * NPART;
    // eight loads in flight: a warp alone (the smallest units) would wait for each
    for (int t = 2 * w + (lane >> 4); t < np; t += 16 * nw) {
        double x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = t + 2 * nw * u < np ? p[(size_t)(t + 2 * nw * u) * NPART + slot] : 0.0;
#pragma unroll
        for (int h = 4; h > 0; h >>= 1)
#pragma unroll
            for (int u = 0; u < h; ++u) x[u] = mx ? fmax(x[u], x[u + h]) : x[u] + x[u + h];
        v = mx ? fmax(v, x[0]) : v + x[0];
    }
    const double o = __shfl_down_sync(0xffffffffu, v, 16);
    v = mx ? fmax(v, o) : v + o;
    if (K && MAXSLOT < 0) {
        for (int t = (int)threadIdx.x; t < R.ntile * D.ksplit; t += blockDim.x) k += D.kpart[R.tile0 * D.ksplit + t];
        k = warp_sum(k);
    }
    if (lane < NPART) sm[w][lane] = v;
    if (lane == 0) sm[w][NPART] = k;
    __syncthreads();
    if (threadIdx.x <= NPART) {
        const int q = threadIdx.x;
        double s = sm[0][q];
        for (int m = 1; m < nw; ++m) s = q == MAXSLOT ? fmax(s, sm[m][q]) : s + sm[m][q];
        acc[q] = s;
    }
    __syncthreads();
}

// H.(r - r_O) enters the dynamics only through DeltaV', which is zero outside
// the band of Eq. 14; sigma itself needs the forces alone.  So the sweeps of
// a large batch leave the Hessian term out for the replicas that are not
// expected in their band (lazy = 1): it costs the sweep a second gather and
// nearly doubles its time (322 and 172 us at 913,408 atoms).  After each
// evaluation the next slope is expected within two of the largest recent changes of the slope; a replica
// whose band reaches there is swept with H (split form: by k_pair_hot, from a
// list).  If another one lands in its band all the same, its evaluation is put off
// (h_meta[1], k_scalar_late) until k_scalar_late has swept it with H, so the
// result never depends on the guess.  list = 0: the next sweep takes H for
// everyone (the last step of a call, whose H can be read), or the form is FP64.
__device__ void expect_slope(const Dev &D, int r, RepState &S, Scal &C, int list) {
    const RepDev &R = D.rep[r];
    const double step = fabs(C.sigma - S.h_sig);
    S.h_step = fmax(step, 0.9 * S.h_step);
    S.h_sig = C.sigma;
    const double m = 2.0 * S.h_step;
    C.need_h = D.bias_on && R.dvmax != 0.0 && C.sigma > R.sig_lo - m && C.sigma < R.sig_hi + m;
    if (list && C.need_h) D.h_list[atomicAdd(D.h_meta, 1)] = r;
}

// threads of a scalar kernel's CTA: what its replica's tile sums can use
static inline int sc_threads(const Dev &D) { return D.max_parts > 256 ? 512 : 256; }
constexpr int SC_MAX = 512;

__global__ void __launch_bounds__(SC_MAX) k_scalar(Dev D, int mode, int lazy, int list) {
    const int r = blockIdx.x;
    __shared__ double acc[NPART + 1];
    const int f = D.rebuild[r];
    if (f) clear_cells(D, D.rep[r]);
    dev_scalar_acc<-1>(D, r, acc);
    if (threadIdx.x < 32) {
        Scal &C = D.sc[r];
        const bool done = scalar_eval(D, r, mode, acc, acc + NPART, D.st[r], C, lazy && !C.need_h);
        if (threadIdx.x == 0) {
            if (!done) D.h_late[atomicAdd(D.h_meta + 1, 1)] = r;
            else if (D.lazy_h) expect_slope(D, r, D.st[r], C, list);
            // the list (if rebuilt this step) has been used; count displacement-triggered builds
            if (f) {
                if (f == 1) D.st[r].n_rebuild += 1;
                D.rebuild[r] = 0;
            }
        }
    }
}

// The replicas whose evaluation k_scalar put off: their sweep with H, then,
// in the last CTA to finish, their scalars.
template <int PREC, int S>
__global__ void __launch_bounds__(256, PREC == HD_FP64 ? 1 : 3) k_scalar_late(Dev D, int mode, int list) {
    const int n = D.h_meta[1];
    if (n == 0) return;
    if (!sweep_listed<PREC, S>(D, D.h_late, n, (unsigned *)D.h_meta + 3)) return;
    __shared__ double acc[NPART + 1];
    for (int q = 0; q < n; ++q) {
        const int r = D.h_late[q];
        dev_scalar_acc<-1>(D, r, acc);
        if (threadIdx.x < 32) {
            scalar_eval(D, r, mode, acc, acc + NPART, D.st[r], D.sc[r]);
            if (threadIdx.x == 0) expect_slope(D, r, D.st[r], D.sc[r], list);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        D.h_meta[1] = 0;
        D.h_meta[3] = 0;
    }
}

// Kinetic energy of the last full step (observables only).
__global__ void k_obs(Dev D) {
    const int r = blockIdx.x;
    const RepDev &R = D.rep[r];
    RepState &S = D.st[r];
    double a = 0.0;
    for (int t = (int)threadIdx.x; t < R.ntile * D.ksplit; t += 32) a += D.kpart[R.tile0 * D.ksplit + t];
    a = warp_sum(a);
    if (threadIdx.x == 0)
        S.K = a + 0.5 * (double)R.nrig * (S.vbody_full[0] * S.vbody_full[0] + S.vbody_full[1] * S.vbody_full[1] +
                                          S.vbody_full[2] * S.vbody_full[2]);
}

// ---------------------------------------------------------------- Nose-Hoover chain
// One half step of the chain (Sec. 3.1.1; the reversible Trotter splitting of
// Martyna, Tuckerman, Tobias and Klein, 1996, one stage): quarter kicks of
// the chain velocities from the top down with exp(-v_{j+1} h/8) damping on
// both sides, the particle scale s = exp(-v_1 h/2), the chain positions by
// h/2, then the kicks from the bottom up.  k2 = sum m v^2 of the mobile atoms
// is updated to its scaled value; returns s.
__device__ double nhc_half(const RepDev &R, RepState &S, double &k2, double h) {
    const int M = R.nhc_len;
    const double kT = R.kT;
    double *v = S.nhc_v;
    auto force = [&](int j) {
        return j == 0 ? (k2 - R.nhc_nf * kT) / R.nhc_Q[0] : (R.nhc_Q[j - 1] * v[j - 1] * v[j - 1] - kT) / R.nhc_Q[j];
    };
    v[M - 1] += 0.25 * h * force(M - 1);
    for (int j = M - 2; j >= 0; --j) {
        const double damp = exp(-0.125 * h * v[j + 1]);
        v[j] *= damp;
        v[j] += 0.25 * h * force(j);
        v[j] *= damp;
    }
    const double sc = exp(-0.5 * h * v[0]);
    k2 *= sc * sc;
    for (int j = 0; j < M; ++j) S.nhc_xi[j] += 0.5 * h * v[j];
    for (int j = 0; j < M - 1; ++j) {
        const double damp = exp(-0.125 * h * v[j + 1]);
        v[j] *= damp;
        v[j] += 0.25 * h * force(j);
        v[j] *= damp;
    }
    v[M - 1] += 0.25 * h * force(M - 1);
    return sc;
}

// The chain between two kicks.  mode KIN: remember k2 of the current
// velocities.  CLOSE: the closing half step of the step that ends (k2 from
// the kinetic sums of the closing kick just made); OPEN: the opening half
// step of the next one (k2 carried over).  C.nhc_scale is the product of the
// particle scales, applied by the next update pass.
__device__ void nhc_eval(const Dev &D, int r, int mode, double ksum, RepState &S, Scal &C) {
    const RepDev &R = D.rep[r];
    C.nhc_scale = 1.0;
    if (R.nhc_len <= 0) return;
    if (mode & MODE_KIN) {
        S.nhc_k2 = 2.0 * ksum;
        return;
    }
    double k2 = (mode & MODE_CLOSE) ? 2.0 * ksum : S.nhc_k2, sc = 1.0;
    if (mode & MODE_CLOSE) sc *= nhc_half(R, S, k2, D.dt);
    if (mode & MODE_OPEN) sc *= nhc_half(R, S, k2, D.dt);
    S.nhc_k2 = k2;
    C.nhc_scale = sc;
}

__global__ void k_nhc(Dev D, int mode) {
    const int r = blockIdx.x;
    const RepDev &R = D.rep[r];
    double a = 0.0;
    for (int t = (int)threadIdx.x; t < R.ntile * D.ksplit; t += 32) a += D.kpart[R.tile0 * D.ksplit + t];
    a = warp_sum(a);
    if (threadIdx.x == 0) nhc_eval(D, r, mode, a, D.st[r], D.sc[r]);
}

// ---------------------------------------------------------------- integrator
// BAOAB (reading: Langevin in place of the paper's Nose-Hoover chain):
//   CLOSE: v += dt/2 F_tot                      (end of the previous step)
//   OPEN:  v += dt/2 F_tot; x += dt/2 v; v = c v + s xi; x += dt/2 v
// Mobile atoms only; rigid atoms follow the body velocity; fixed atoms stay.
__device__ __forceinline__ int4 post_move(const Dev &D, const RepDev &R, int r, int i, dbl4 x, int4 p, int *moved) {
    const int4 q = fix_pos(R, x, p.w);
    D.p[i] = q;
    const int4 b = D.pfixb[i];
    const float ex = (float)(int)((unsigned)q.x - (unsigned)b.x) * R.fx_lsb[0];
    const float ey = (float)(int)((unsigned)q.y - (unsigned)b.y) * R.fx_lsb[1];
    const float ez = (float)(int)((unsigned)q.z - (unsigned)b.z) * R.fx_lsb[2];
    if (ex * ex + ey * ey + ez * ez > D.half_skin2_f) *moved = 1;
    const double zv = R.vert == 2 ? x.z : x.y;
    if (!(fabs(zv - R.fx_origin[R.vert]) < R.open_lim) || !isfinite(x.x) || !isfinite(x.y) || !isfinite(x.z))
        set_err(D, HD_ERR_NUMERIC, i, r);
    return q;
}

// Split form: the new fixed-point image, the checks of post_move, and that
// r - r_O (the difference of the images of r and r_O) has not wrapped.  It
// wraps at L / 2^(k+1) >= 4 (rc + skin); an atom is reported (HD_ERR_NUMERIC)
// when it has moved 3/4 of that from its r_O.
__device__ __forceinline__ void post_move32(const Dev &D, const RepDev &R, int r, int i, dbl4 x, int4 p, int *moved) {
    const int4 q = fix_pos(R, x, p.w);
    const int4 d = img_diff(q, D.po[i]);
    D.p[i] = q;
    const int4 b = D.pfixb[i];
    const float ex = (float)(int)((unsigned)q.x - (unsigned)b.x) * R.fx_lsb[0];
    const float ey = (float)(int)((unsigned)q.y - (unsigned)b.y) * R.fx_lsb[1];
    const float ez = (float)(int)((unsigned)q.z - (unsigned)b.z) * R.fx_lsb[2];
    if (ex * ex + ey * ey + ez * ez > D.half_skin2_f) *moved = 1;
    const double zv = R.vert == 2 ? x.z : x.y;
    const int lim = 3 << 29;
    if (!(fabs(zv - R.fx_origin[R.vert]) < R.open_lim) || !isfinite(x.x) || !isfinite(x.y) || !isfinite(x.z) ||
        abs(d.x) > lim || abs(d.y) > lim || abs(d.z) > lim)
        set_err(D, HD_ERR_NUMERIC, i, r);
}

// The atoms a CTA updates: a tile of the per-phase kernels; a unit of the
// persistent launch (block / split atoms, with more threads than that), whose
// kinetic sum has its own slot.  *moved is set where an atom has moved half the
// skin since the last list build: the replica's flag, or the CTA's own.
struct UpdateSpan {
    int t, first, n, slot, r;
    int *moved;
};
__device__ __forceinline__ UpdateSpan update_tile(const Dev &D, int t) {
    const int r = D.tile_rep[t];
    return {t, D.tile_start[t], D.tile_n[t], t * D.ksplit, r, D.rebuild + r};
}
__device__ __forceinline__ UpdateSpan update_unit(const Dev &D, int unit, int *moved) {
    const int t = unit / D.split;
    const UnitSpan a = unit_span(D.tile_start[t], D.tile_n[t], D.block / D.split, unit % D.split);
    return {t, a.first, a.n, unit, D.tile_rep[t], moved};
}

__device__ __forceinline__ void dev_update64(const Dev &D, const UpdateSpan &U, int mode, const Scal &C) {
    const int r = U.r;
    const RepDev &R = D.rep[r];
    const bool act = (int)threadIdx.x < U.n;
    const int i = U.first + (act ? threadIdx.x : 0);
    const int4 p = D.p[i];
    const int role = act ? ((p.w >> 8) & 0xff) : ROLE_FIXED;
    double kin = 0.0;
    if (role != ROLE_FIXED) {
        const double h = D.dt;
        dbl4 x = D.x[i], v = D.v64[i];
        if (role == ROLE_MOBILE) {
            const dbl4 F = D.f64[i], H = D.h64[i], dr = D.dr64[i];
            const double ca = C.ca, cb = C.cb;
            double Fx = F.x + ca * (H.x - F.x) + cb * dr.x;
            double Fy = F.y + ca * (H.y - F.y) + cb * dr.y;
            double Fz = F.z + ca * (H.z - F.z) + cb * dr.z;
            if (C.ce != 0.0) {               // eigenvalue bias (Eq. 13, Eq. 15)
                const dbl4 g = D.eg[i];
                Fx += C.ce * g.x;
                Fy += C.ce * g.y;
                Fz += C.ce * g.z;
            }
            const bool three = R.dim == 3;
            const bool chain = R.nhc_len > 0;
            if (mode & MODE_KIN) kin = 0.5 * (v.x * v.x + v.y * v.y + v.z * v.z);
            if (mode & MODE_SCALE) {
                if (chain) {
                    v.x *= C.nhc_scale;
                    v.y *= C.nhc_scale;
                    v.z *= C.nhc_scale;
                }
                kin = 0.5 * (v.x * v.x + v.y * v.y + v.z * v.z);
            }
            if (mode & MODE_CLOSE) {
                v.x += 0.5 * h * Fx;
                v.y += 0.5 * h * Fy;
                if (three) v.z += 0.5 * h * Fz;
                kin = 0.5 * (v.x * v.x + v.y * v.y + v.z * v.z);
            }
            if (mode & MODE_OPEN) {
                if (chain && (mode & MODE_NHC)) {
                    v.x *= C.nhc_scale;
                    v.y *= C.nhc_scale;
                    v.z *= C.nhc_scale;
                }
                v.x += 0.5 * h * Fx;
                v.y += 0.5 * h * Fy;
                if (three) v.z += 0.5 * h * Fz;
                x.x += 0.5 * h * v.x;
                x.y += 0.5 * h * v.y;
                if (three) x.z += 0.5 * h * v.z;
                if (!chain) {
                    double n0, n1, n2, n3;
                    normals64(philox_draw(D, C.step_cur, D.orig[i], R.rep_id, 0), n0, n1);
                    v.x = R.c_ou * v.x + R.s_ou * n0;
                    v.y = R.c_ou * v.y + R.s_ou * n1;
                    if (three) {
                        normals64(philox_draw(D, C.step_cur, D.orig[i], R.rep_id, 1), n2, n3);
                        v.z = R.c_ou * v.z + R.s_ou * n2;
                    }
                }
                x.x += 0.5 * h * v.x;
                x.y += 0.5 * h * v.y;
                if (three) x.z += 0.5 * h * v.z;
            }
        } else {
            if (mode & MODE_CLOSE) v = make_dbl4(C.vb_mid[0], C.vb_mid[1], C.vb_mid[2], 0.0);
            if (mode & MODE_OPEN) {
                x.x += 0.5 * h * C.vb_new[0];
                x.y += 0.5 * h * C.vb_new[1];
                x.z += 0.5 * h * C.vb_new[2];
                x.x += 0.5 * h * C.vb_new[0];
                x.y += 0.5 * h * C.vb_new[1];
                x.z += 0.5 * h * C.vb_new[2];
                v = make_dbl4(C.vb_new[0], C.vb_new[1], C.vb_new[2], 0.0);
            }
        }
        D.v64[i] = v;
        if (mode & MODE_OPEN) {
            D.x[i] = x;
            const dbl4 xo = D.xo[i];
            D.dr64[i] = make_dbl4(x.x - xo.x, x.y - xo.y, x.z - xo.z, 0.0);
            post_move(D, R, r, i, x, p, U.moved);
        }
    }
    if (mode & (MODE_CLOSE | MODE_KIN | MODE_SCALE)) {
        double v1[1] = {kin};
        cta_reduce<1>(v1, D.kpart + U.slot, -1);
    }
}

__device__ __forceinline__ void dev_update32(const Dev &D, const UpdateSpan &U, int mode, const Scal &C) {
    // split form: FP32 forces, FP64 velocities and positions (FP32 velocities
    // would round every kick and thermostat step at 2^-24 of |v|, which after
    // 100 steps puts sigma and the boosted clock beyond 1e-6 of FP64); r - r_O
    // from the fixed-point images of r and r_O
    const int r = U.r;
    const RepDev &R = D.rep[r];
    const bool act = (int)threadIdx.x < U.n;
    const int i = U.first + (act ? threadIdx.x : 0);
    const int4 p = D.p[i];
    const int role = act ? ((p.w >> 8) & 0xff) : ROLE_FIXED;
    // the closing half kick of one step and the opening one of the next see
    // the same force: between steps of one call a Langevin replica takes one
    // full kick in FP64 (this GPU's FP64 rate is a small fraction of its FP32
    // rate).  The kinetic energy at the half step is an observable there, not
    // an input, and is summed only on the closing half of a call's last step.
    const bool fused = R.nhc_len == 0 && (mode & MODE_CLOSE) && (mode & MODE_OPEN);
    float kin = 0.f;
    if (role != ROLE_FIXED) {
        const double hh = 0.5 * D.dt;
        dbl4 v = D.v64[i];
        dbl4 x = D.x[i];
        if (role == ROLE_MOBILE) {
            const float4 F = D.f32[i], H = D.h32[i];
            const int4 di = img_diff(p, D.po[i]);
            const float4 dr = make_float4((float)di.x * R.fx_lsb[0], (float)di.y * R.fx_lsb[1],
                                          (float)di.z * R.fx_lsb[2], 0.f);
            const float ca = (float)C.ca, cb = (float)C.cb;
            double Fx = (double)fmaf(ca, H.x - F.x, fmaf(cb, dr.x, F.x));
            double Fy = (double)fmaf(ca, H.y - F.y, fmaf(cb, dr.y, F.y));
            double Fz = (double)fmaf(ca, H.z - F.z, fmaf(cb, dr.z, F.z));
            if (C.ce != 0.0) {               // eigenvalue bias (Eq. 13, Eq. 15), FP64
                const dbl4 g = D.eg[i];
                Fx += C.ce * g.x;
                Fy += C.ce * g.y;
                Fz += C.ce * g.z;
            }
            const bool three = R.dim == 3;
            const bool chain = R.nhc_len > 0;
            if (fused) {
                v.x = fma(D.dt, Fx, v.x);
                v.y = fma(D.dt, Fy, v.y);
                if (three) v.z = fma(D.dt, Fz, v.z);
            } else {
                if (mode & MODE_KIN) kin = (float)(0.5 * (v.x * v.x + v.y * v.y + v.z * v.z));
                if (mode & MODE_SCALE) {
                    if (chain) {
                        v.x *= C.nhc_scale;
                        v.y *= C.nhc_scale;
                        v.z *= C.nhc_scale;
                    }
                    kin = (float)(0.5 * (v.x * v.x + v.y * v.y + v.z * v.z));
                }
                if (mode & MODE_CLOSE) {
                    v.x += hh * Fx;
                    v.y += hh * Fy;
                    if (three) v.z += hh * Fz;
                    kin = (float)(0.5 * (v.x * v.x + v.y * v.y + v.z * v.z));
                }
                if (mode & MODE_OPEN) {
                    if (chain && (mode & MODE_NHC)) {
                        v.x *= C.nhc_scale;
                        v.y *= C.nhc_scale;
                        v.z *= C.nhc_scale;
                    }
                    v.x += hh * Fx;
                    v.y += hh * Fy;
                    if (three) v.z += hh * Fz;
                }
            }
            if (mode & MODE_OPEN) {
                const double ax = v.x, ay = v.y, az = v.z;
                if (!chain) {
                    float n0, n1, n2, n3;
                    normals32(philox_draw(D, C.step_cur, D.orig[i], R.rep_id, 0), n0, n1);
                    v.x = R.c_ou * v.x + R.s_ou * (double)n0;
                    v.y = R.c_ou * v.y + R.s_ou * (double)n1;
                    if (three) {
                        normals32(philox_draw(D, C.step_cur, D.orig[i], R.rep_id, 1), n2, n3);
                        v.z = R.c_ou * v.z + R.s_ou * (double)n2;
                    }
                }
                x.x += hh * (ax + v.x);
                x.y += hh * (ay + v.y);
                if (three) x.z += hh * (az + v.z);
            }
        } else {
            if (mode & MODE_CLOSE) v = make_dbl4(C.vb_mid[0], C.vb_mid[1], C.vb_mid[2], 0.0);
            if (mode & MODE_OPEN) {
                x.x += hh * C.vb_new[0];
                x.y += hh * C.vb_new[1];
                x.z += hh * C.vb_new[2];
                x.x += hh * C.vb_new[0];
                x.y += hh * C.vb_new[1];
                x.z += hh * C.vb_new[2];
                v = make_dbl4(C.vb_new[0], C.vb_new[1], C.vb_new[2], 0.0);
            }
        }
        D.v64[i] = v;
        if (mode & MODE_OPEN) {
            D.x[i] = x;
            post_move32(D, R, r, i, x, p, U.moved);
        }
    }
    if ((mode & (MODE_CLOSE | MODE_KIN | MODE_SCALE)) && !fused) {
        double v1[1] = {(double)kin};    // FP64 sums: how atoms share warps must not show in K
        cta_reduce<1>(v1, D.kpart + U.slot, -1);
    }
}

__global__ void __launch_bounds__(256) k_update64(Dev D, int mode) {
    dev_update64(D, update_tile(D, blockIdx.x), mode, D.sc[D.tile_rep[blockIdx.x]]);
}
__global__ void __launch_bounds__(256) k_update32(Dev D, int mode) {
    dev_update32(D, update_tile(D, blockIdx.x), mode, D.sc[D.tile_rep[blockIdx.x]]);
}

// ---------------------------------------------------------------- quench
// |x - r_O|^2 in FP64, in the transition test's operation order.  Positions
// and r_O are never wrapped, so below L/2 per axis this is the minimum-image
// value bit for bit; beyond it it is larger, which only delays an early stop.
__device__ __forceinline__ double disp2(dbl4 a, dbl4 b) {
    const double d0 = __dsub_rn(a.x, b.x), d1 = __dsub_rn(a.y, b.y), d2 = __dsub_rn(a.z, b.z);
    return __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
}

// Split form: |x - r_O|^2 in FP32 from the difference of the fixed-point
// images of x and r_O (exact integers; no FP64 instruction).  A difference
// beyond 3/4 of the image range reads as far.  The early stop compares it
// with (theta/2)^2, where FP32 rounding can only matter within ~1e-7 of it.
__device__ __forceinline__ float disp2_img(const RepDev &R, int4 q, int4 po) {
    const int4 d = img_diff(q, po);
    const int lim = 3 << 29;
    if (abs(d.x) > lim || abs(d.y) > lim || abs(d.z) > lim) return 3.0e38f;
    const float dx = (float)d.x * R.fx_lsb[0], dy = (float)d.y * R.fx_lsb[1], dz = (float)d.z * R.fx_lsb[2];
    return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Largest m over the CTA into qgate[r] (non-negative doubles order as their
// bit patterns).  Every thread of the CTA calls it.
__device__ __forceinline__ void gate_max(const Dev &D, int r, double m) {
    __shared__ double sm[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    m = warp_max(m);
    if (lane == 0) sm[w] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = sm[0];
        for (int k = 1; k < nw; ++k) a = fmax(a, sm[k]);
        atomicMax(D.qgate + r, (unsigned long long)__double_as_longlong(a));
    }
}
// The same over FP32 values, converted once per CTA.
__device__ __forceinline__ void gate_max_f(const Dev &D, int r, float m) {
    __shared__ float smf[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
    if (lane == 0) smf[w] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        float a = smf[0];
        for (int k = 1; k < nw; ++k) a = fmaxf(a, smf[k]);
        atomicMax(D.qgate + r, (unsigned long long)__double_as_longlong((double)a));
    }
}

__global__ void k_qinit(Dev Q, Dev M) {
    // Q: quench view (x = copy), M: MD view
    const int t = blockIdx.x, r = Q.tile_rep[t];
    if (threadIdx.x == 0 && t == Q.rep[r].tile0) {
        RepState &S = Q.st[r];
        S.q_dt = Q.q_step;
        S.q_alpha = 0.1;
        S.q_npos = 0;
        S.q_iter = 0;
        S.q_done = 0;
        S.q_flag = 0;
        S.q_stay = 0;
        S.q_fmax = 0.0;
        S.q_vb[0] = S.q_vb[1] = S.q_vb[2] = 0.0;
        Q.qdisp[r] = 0ull;
        Q.rebuild[r] = 2;
    }
    double m = 0.0;
    float mf = 0.f;
    if (threadIdx.x < Q.tile_n[t]) {
        const int i = Q.tile_start[t] + threadIdx.x;
        const dbl4 x = M.x[i];
        const int4 p = M.p[i];
        Q.x[i] = x;
        Q.p[i] = p;
        if (Q.prec == HD_FP64) Q.v64[i] = make_dbl4(0, 0, 0, 0);
        else Q.v32[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (Q.q_ftol_stay > 0.0) {
            if (Q.prec == HD_FP64) m = disp2(x, Q.xo[i]);
            else mf = disp2_img(Q.rep[r], p, Q.po[i]);
        }
    }
    if (Q.q_ftol_stay > 0.0) {
        if (Q.prec == HD_FP64) gate_max(Q, r, m);
        else gate_max_f(Q, r, mf);
    }
}

// Convergence test and FIRE bookkeeping (reading of Bitzek et al. 2006: mix
// with the alpha of this step, then grow/shrink dt and alpha).
__global__ void __launch_bounds__(SC_MAX) k_qscalar(Dev D, int max_iter) {
    const int r = blockIdx.x;
    const RepDev &R = D.rep[r];
    RepState &S = D.st[r];
    Scal &C = D.sc[r];
    // this iteration's list rebuild (if any) has been used by the pair pass
    if (D.rebuild[r]) clear_cells(D, R);
    const bool done = S.q_done != 0;
    __syncthreads();
    if (threadIdx.x == 0) D.rebuild[r] = 0;
    if (done) return;
    __shared__ double acc[NPART + 1];
    dev_scalar_acc<QP_FMAX2>(D, r, acc);
    if (threadIdx.x != 0) return;
    const double inr = R.inv_nrig;
    const int nr = R.nrig, dim = R.dim;
    double fb[3] = {0, 0, 0};
    double fm2 = acc[QP_FMAX2];
    if (nr > 0) {
        double xT[3], gs[3] = {0, 0, 0};
        for (int a = 0; a < 3; ++a) xT[a] = acc[QP_XRIG + a] * inr;
        gs[0] = R.kspring * (xT[0] - slider_x(R, S.step, D.dt));   // the slider stands still during a quench
        if (dim == 3) gs[1] = R.kspring * (xT[1] - R.slider[1]);
        gs[R.vert] = R.fnormal;
        for (int a = 0; a < 3; ++a) fb[a] = acc[QP_FRIG + a] - gs[a];
        fm2 = fmax(fm2, fb[0] * fb[0] + fb[1] * fb[1] + fb[2] * fb[2]);
    }
    const double fmax_ = sqrt(fm2);
    S.q_fmax = fmax_;
    // early stop inside the basin: every atom within theta/2 of r_O and the
    // force below ftol_stay rule a transition out (Sec. 2.3 transition test)
    bool stay = false;
    if (D.q_ftol_stay > 0.0) {
        const double g2 = __longlong_as_double((long long)D.qgate[r]);
        D.qgate[r] = 0ull;
        stay = fmax_ < D.q_ftol_stay && g2 < D.q_keep2;
    }
    if (fmax_ < D.q_ftol || stay || S.q_iter >= max_iter) {
        S.q_done = 1;
        S.q_stay = stay && !(fmax_ < D.q_ftol);
        C.q_active = 0;
        return;
    }
    C.q_active = 1;
    for (int a = 0; a < 3; ++a) C.q_fbody[a] = fb[a];
    if (D.q_method == 1) {
        double pw = acc[QP_P], vv = acc[QP_VV], ff = acc[QP_FF];
        if (nr > 0)
            for (int a = 0; a < dim; ++a) {
                pw += fb[a] * S.q_vb[a];
                vv += (double)nr * S.q_vb[a] * S.q_vb[a];
                ff += fb[a] * fb[a] * inr;
            }
        double alpha = S.q_alpha, dt = S.q_dt;
        double vb[3] = {S.q_vb[0], S.q_vb[1], S.q_vb[2]};
        if (pw > 0.0) {
            const double mix = ff > 0.0 ? alpha * sqrt(vv / ff) : 0.0;
            C.q_mix = mix;
            C.q_zero = 0;
            if (nr > 0)
                for (int a = 0; a < dim; ++a) vb[a] = (1.0 - alpha) * vb[a] + mix * fb[a] * inr;
            S.q_npos += 1;
            if (S.q_npos > 5) {
                dt = dt * 1.1 < 10.0 * D.q_step ? dt * 1.1 : 10.0 * D.q_step;
                alpha *= 0.99;
            }
        } else {
            C.q_mix = 0.0;
            C.q_zero = 1;
            vb[0] = vb[1] = vb[2] = 0.0;
            dt *= 0.5;
            alpha = 0.1;
            S.q_npos = 0;
        }
        C.q_alpha = S.q_alpha;   // the alpha this step mixes with
        C.q_dt = dt;             // the dt this step moves with
        S.q_alpha = alpha;
        S.q_dt = dt;
        if (nr > 0)
            for (int a = 0; a < dim; ++a) vb[a] += dt * fb[a] * inr;
        for (int a = 0; a < 3; ++a) { S.q_vb[a] = vb[a]; C.q_vb[a] = vb[a]; }
    }
    S.q_iter += 1;
}

// Per-atom quench move.  SD: x += a F (body: a F_body / n_rig).  FIRE: mix,
// or zero, the velocity, then a semi-implicit Euler step.
template <typename V4>
__device__ __forceinline__ dbl4 qmove(const Dev &D, const RepDev &R, const Scal &C, int r, int i, int4 p, int role,
                                      double fx, double fy, double fz, V4 *vq, int4 *img) {
    dbl4 x = D.x[i];
    const int dim = R.dim;
    if (D.q_method == 0) {
        const double a = D.q_step;
        if (role == ROLE_MOBILE) {
            x.x += a * fx;
            x.y += a * fy;
            if (dim == 3) x.z += a * fz;
        } else {
            const double inr = 1.0 / (double)R.nrig;
            x.x += a * C.q_fbody[0] * inr;
            x.y += a * C.q_fbody[1] * inr;
            if (dim == 3) x.z += a * C.q_fbody[2] * inr;
        }
    } else {
        const double dt = C.q_dt;
        if (role == ROLE_MOBILE) {
            V4 v = vq[i];
            double vx = v.x, vy = v.y, vz = v.z;
            if (C.q_zero) {
                vx = vy = vz = 0.0;
            } else {
                vx = (1.0 - C.q_alpha) * vx + C.q_mix * fx;
                vy = (1.0 - C.q_alpha) * vy + C.q_mix * fy;
                vz = (1.0 - C.q_alpha) * vz + C.q_mix * fz;
            }
            vx += dt * fx;
            vy += dt * fy;
            if (dim == 3) vz += dt * fz;
            else vz = 0.0;
            x.x += dt * vx;
            x.y += dt * vy;
            if (dim == 3) x.z += dt * vz;
            v.x = vx; v.y = vy; v.z = vz;
            vq[i] = v;
        } else {
            x.x += dt * C.q_vb[0];
            x.y += dt * C.q_vb[1];
            if (dim == 3) x.z += dt * C.q_vb[2];
        }
    }
    D.x[i] = x;
    *img = post_move(D, R, r, i, x, p, D.rebuild + r);
    return x;
}

// The split form's FIRE move in FP32 (its velocities are FP32 and its forces
// FP32 already): only the position, kept in FP64, takes FP64 adds.
__device__ __forceinline__ int4 qmove32(const Dev &D, const RepDev &R, const Scal &C, int r, int i, int4 p, int role,
                                        float fx, float fy, float fz) {
    if (D.q_method == 0) {
        int4 q;
        qmove(D, R, C, r, i, p, role, (double)fx, (double)fy, (double)fz, D.v32, &q);
        return q;
    }
    dbl4 x = D.x[i];
    const bool three = R.dim == 3;
    const float dt = (float)C.q_dt;
    if (role == ROLE_MOBILE) {
        float4 v = D.v32[i];
        if (C.q_zero) {
            v.x = v.y = v.z = 0.f;
        } else {
            const float keep = (float)(1.0 - C.q_alpha), mix = (float)C.q_mix;
            v.x = fmaf(keep, v.x, mix * fx);
            v.y = fmaf(keep, v.y, mix * fy);
            v.z = fmaf(keep, v.z, mix * fz);
        }
        v.x = fmaf(dt, fx, v.x);
        v.y = fmaf(dt, fy, v.y);
        v.z = three ? fmaf(dt, fz, v.z) : 0.f;
        x.x += (double)(dt * v.x);
        x.y += (double)(dt * v.y);
        if (three) x.z += (double)(dt * v.z);
        D.v32[i] = v;
    } else {
        x.x += C.q_dt * C.q_vb[0];
        x.y += C.q_dt * C.q_vb[1];
        if (three) x.z += C.q_dt * C.q_vb[2];
    }
    D.x[i] = x;
    return post_move(D, R, r, i, x, p, D.rebuild + r);
}

__global__ void __launch_bounds__(256) k_qupdate(Dev D) {
    const int t = blockIdx.x, r = D.tile_rep[t];
    const Scal &C = D.sc[r];
    if (!C.q_active || D.st[r].q_done) return;        // the same for the whole CTA
    // displacement from r_O of the new iterate (every atom, as in the
    // transition test), for the next convergence test
    const bool gate = D.q_ftol_stay > 0.0;
    double m = 0.0;
    float mf = 0.f;
    if (threadIdx.x < D.tile_n[t]) {
        const int i = D.tile_start[t] + threadIdx.x;
        const RepDev &R = D.rep[r];
        const int4 p = D.p[i];
        const int role = (p.w >> 8) & 0xff;
        if (D.prec == HD_FP64) {
            dbl4 x;
            int4 q;
            if (role == ROLE_FIXED) {
                if (gate) x = D.x[i];
            } else {
                const dbl4 f = D.f64[i];
                x = qmove(D, R, C, r, i, p, role, f.x, f.y, f.z, D.v64, &q);
            }
            if (gate) m = disp2(x, D.xo[i]);
        } else {
            int4 q = p;
            if (role != ROLE_FIXED) {
                const float4 f = D.f32[i];
                q = qmove32(D, R, C, r, i, p, role, f.x, f.y, f.z);
            }
            if (gate) mf = disp2_img(R, q, D.po[i]);
        }
    }
    if (gate) {
        if (D.prec == HD_FP64) gate_max(D, r, m);
        else gate_max_f(D, r, mf);
    }
}

// Largest displacement of the quenched copy from r_O per replica (minimum
// image, FP64, the oracle's operation order); stored as the bits of the
// non-negative double so that an integer max is the FP64 max.
// One atomic per CTA: with one per atom the 14,272 of a replica ran one after
// another (508 us for 64 of them; 26 now).  Below half a box the nearest integer to
// d / L is 0 and the division, which the FP64 pipe takes ten instructions for,
// is left out.
__global__ void __launch_bounds__(256) k_qdisp(Dev Q) {
    __shared__ unsigned long long most;
    const int t = blockIdx.x, r = Q.tile_rep[t];
    if (threadIdx.x == 0) most = 0ull;
    __syncthreads();
    unsigned long long bits = 0ull;
    if (threadIdx.x < Q.tile_n[t]) {
        const int i = Q.tile_start[t] + threadIdx.x;
        const RepDev &R = Q.rep[r];
        const dbl4 a = Q.x[i], b = Q.xo[i];
        auto image = [&](int ax, double d) {
            if (!R.periodic[ax] || fabs(d) < 0.499 * R.L[ax]) return d;
            return __dsub_rn(d, __dmul_rn(R.L[ax], rint(__ddiv_rn(d, R.L[ax]))));
        };
        const double d0 = image(0, a.x - b.x), d1 = image(1, a.y - b.y), d2 = image(2, a.z - b.z);
        const double m = __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
        bits = (unsigned long long)__double_as_longlong(m);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, bits, o);
        bits = u > bits ? u : bits;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(&most, bits);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(Q.qdisp + r, most);
}

// r_O <- quenched copy for replicas with adopt[r] != 0; refresh r - r_O.
__global__ void k_adopt(Dev Q, Dev M, const int *adopt) {
    const int t = blockIdx.x, r = M.tile_rep[t];
    if (!adopt[r] || threadIdx.x >= M.tile_n[t]) return;
    const int i = M.tile_start[t] + threadIdx.x;
    const dbl4 q = Q.x[i];
    M.xo[i] = make_dbl4(q.x, q.y, q.z, 0.0);
    const dbl4 x = M.x[i];
    if (M.prec == HD_FP64) M.dr64[i] = make_dbl4(x.x - q.x, x.y - q.y, x.z - q.z, 0.0);
    else M.po[i] = fix_pos(M.rep[r], make_dbl4(q.x, q.y, q.z, 0.0), 0);
}

// ---------------------------------------------------------------- persistent driver
// One launch steps every replica n times.  Replica r owns CTAs
// [pg_first[r], pg_first[r] + pg_count[r]); each takes the replica's units
// (see dev_pair64) round robin and runs the same phases as the per-phase
// kernels; the compiler may contract multiply-adds differently where a phase
// is inlined here, so the two drivers agree to rounding.
//
// Small replicas are what this driver is for, and a step of theirs is latency:
// two barriers, the sweep of a row, the scalars and the update.  So a unit is
// small (8 atoms where the batch leaves SMs idle: an FP64 sweep is bound by
// the FP64 pipe of the SMs it is on), a CTA updates the atoms it sweeps, states
// go to global memory at the end of the call only, and a barrier carries the
// flag that a list is due.  Against a tile's threads, separate flags and
// fences a step of 16 x 421 atoms takes 16.2 us in place of 18.7, of 8 x 113 in
// the FP64 form 33.2 in place of 36.5.
//
// Phases of one replica are separated by that replica's own barrier: a 64-bit
// counter in global memory (reset before each launch) whose low half counts
// arrivals and whose high half counts CTAs that saw an atom move half the skin
// in the update before (a call of very many steps is cut into launches, so the
// low half never carries: persist_steps_max).  An arrival releases the CTA's writes, the poll
// acquires the others'.  Polling is bounded: after ~2^24 polls the CTA records
// HD_ERR_TIMEOUT, raises the abort word err[3], and every CTA leaves at its
// next barrier.  The launch is cooperative, so all CTAs are resident.  A
// one-CTA replica uses only __syncthreads().
struct GrpBar {
    unsigned epoch, moved;       // barriers passed; high half of the counter at the last one
    bool due;                    // a CTA arrived with `moved` since then
};
__device__ __forceinline__ bool grp_barrier(const Dev &D, int r, int nc, GrpBar &B, int *s_moved) {
    __shared__ int s_ok;
    __shared__ unsigned s_hi;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned mine = s_moved && *s_moved ? 1u : 0u;
        unsigned hi = B.moved + mine;
        if (s_moved) *s_moved = 0;
        if (nc > 1) {
            unsigned long long *ctr = reinterpret_cast<unsigned long long *>(D.bar) + r;
            const unsigned target = (B.epoch + 1u) * (unsigned)nc;
            // test hook: one CTA of replica fault_rep skips its first arrival
            const bool skip = D.fault_rep == r && B.epoch == 0 && blockIdx.x == (unsigned)D.pg_first[r];
            const unsigned long long add = ((unsigned long long)mine << 32) | 1ull;
            if (!skip) asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(ctr), "l"(add) : "memory");
            unsigned polls = 0;
            unsigned long long v;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ctr) : "memory");
                if ((unsigned)v >= target) break;
                if ((++polls & 63u) == 0) {
                    if (*((volatile int *)(D.err + 3)) != 0) { ok = 0; break; }
                    if (polls > (1u << 24)) {
                        set_err(D, HD_ERR_TIMEOUT, -1, r);
                        atomicExch(D.err + 3, 1);
                        ok = 0;
                        break;
                    }
                    __nanosleep(64);
                }
            }
            hi = (unsigned)(v >> 32);
        }
        s_hi = hi;
        s_ok = ok;
    }
    __syncthreads();
    ++B.epoch;
    // at the other barriers the high half may already hold the next update's
    if (s_moved) {
        B.due = s_hi != B.moved;
        B.moved = s_hi;
    }
    return s_ok != 0;
}

template <int PREC, int S>
__global__ void __launch_bounds__(128, 4) k_persist(Dev D, int nsteps) {
    const int r = D.cta_rep[blockIdx.x];
    if (r < 0) return;
    const RepDev &R = D.rep[r];
    const int nc = D.pg_count[r], me = blockIdx.x - D.pg_first[r];
    const int u0 = R.tile0 * D.split + me, u1 = (R.tile0 + R.ntile) * D.split;
    const bool leader = me == 0;
    __shared__ RepState St;
    __shared__ Scal C;
    __shared__ double acc[NPART + 1];
    __shared__ int s_moved;
    __shared__ NlSmem M;
    extern __shared__ __align__(16) char nl_smem[];
    const NlStage T = nl_smem_carve(D, nl_smem);
    if (threadIdx.x == 0) {
        St = D.st[r];
        C = D.sc[r];
        s_moved = D.rebuild[r] != 0;
    }
    __syncthreads();
    GrpBar B = {0u, 0u, false};
    // The kinetic parts are left alone here: a CTA that is through goes on to
    // update() and writes its own while another may still be in here.  K is
    // formed when it is read (k_obs).
    auto scalars = [&](int mode) {
        dev_scalar_acc<-1, false>(D, r, acc);
        if (threadIdx.x < 32) scalar_eval(D, r, mode, acc, nullptr, St, C);
        __syncthreads();
    };
    auto update = [&](int mode) {
        for (int u = u0; u < u1; u += nc) {
            if (PREC == HD_FP64) dev_update64(D, update_unit(D, u, &s_moved), mode, C);
            else dev_update32(D, update_unit(D, u, &s_moved), mode, C);
        }
    };
    // the chain between the kicks (every CTA evaluates it alike from the
    // replica's kinetic sums)
    auto chain = [&](int mode) {
        dev_scalar_acc<-1>(D, r, acc);
        if (threadIdx.x == 0) nhc_eval(D, r, mode, acc[NPART], St, C);
        __syncthreads();
    };
    const bool nhc = D.any_nhc != 0;
    // opening half of the first step, from the forces of the last call
    scalars(MODE_OPEN);
    if (nhc) chain(MODE_OPEN);
    update(nhc ? (MODE_OPEN | MODE_NHC) : MODE_OPEN);
    if (!grp_barrier(D, r, nc, B, &s_moved)) return;
    for (int k = 1; k <= nsteps; ++k) {
        if (B.due) {
            for (int i = R.atom0 + me * blockDim.x + threadIdx.x; i < R.atom0 + R.n; i += nc * blockDim.x) dev_bin_atom(D, r, i);
            if (!grp_barrier(D, r, nc, B, nullptr)) return;
            {
                const int wib = threadIdx.x >> 5, nwb = blockDim.x >> 5;
                int *buf = reinterpret_cast<int *>(nl_smem) + wib * D.cell_cap;
                for (int c = me * nwb + wib; c < R.ncell; c += nc * nwb) dev_cellsort_warp(D, R, c, buf);
                __syncthreads();
            }
            if (!grp_barrier(D, r, nc, B, nullptr)) return;
            if (threadIdx.x == 0) St.n_rebuild += 1;
            // rows are built cell by cell, so a CTA's units take rows other CTAs wrote
            for (int c = me; c < R.ncell; c += nc) dev_nlist_cell(D, r, c, M, T);
            if (!grp_barrier(D, r, nc, B, nullptr)) return;
            // the counts go back to zero for the next binning, whoever does it
            for (int c = me * blockDim.x + threadIdx.x; c < R.ncell; c += nc * blockDim.x) D.cell_cnt[R.cell0 + c] = 0;
        }
        for (int u = u0; u < u1; u += nc) {
            // per-atom energies (observables only) on the last step of the call
            // and H.(r - r_O) there and wherever a bias may use it
            if (PREC == HD_FP64) {
                if (k == nsteps) dev_pair64<false, true, true, S>(D, u);
                else if (D.bias_on) dev_pair64<false, false, true, S>(D, u);
                else dev_pair64<false, false, false, S>(D, u);
            } else {
                if (k == nsteps) dev_pair32<false, true, true, S>(D, u);
                else if (D.bias_on) dev_pair32<false, false, true, S>(D, u);
                else dev_pair32<false, false, false, S>(D, u);
            }
        }
        if (!grp_barrier(D, r, nc, B, nullptr)) return;
        const int mode = k < nsteps ? (MODE_CLOSE | MODE_OPEN) : MODE_CLOSE;
        scalars(mode);
        if (!nhc) {
            update(mode);
        } else {
            update(MODE_CLOSE);
            if (!grp_barrier(D, r, nc, B, nullptr)) return;
            chain(mode);
            // MODE_SCALE writes the kinetic sums that chain() has read
            if (!(mode & MODE_OPEN) && !grp_barrier(D, r, nc, B, nullptr)) return;
            update((mode & MODE_OPEN) ? (MODE_OPEN | MODE_NHC) : MODE_SCALE);
        }
        if (!grp_barrier(D, r, nc, B, &s_moved)) return;
    }
    if (leader && threadIdx.x == 0) {
        D.st[r] = St;
        D.sc[r] = C;
        D.rebuild[r] = 0;
    }
}

// ---------------------------------------------------------------- launchers
static inline int nthr(const Dev &D) { return D.block; }

// Dynamic shared memory of the list build.
size_t nl_smem_bytes(const Dev &D, int nwarps) {
    return (size_t)nl_cand(D) * 16 + nwarps * nl_warp_bytes(D);
}
// threads of a CTA of the pair sweep and of the persistent launch: its unit's atoms times the lanes of a row
static int unit_threads(const Dev &D) { return D.block / D.split * D.lanes; }
static size_t persist_smem_bytes(const Dev &D) { return nl_smem_bytes(D, (unit_threads(D) + 31) / 32); }
typedef void (*persist_fn)(Dev, int);
static persist_fn persist_kernel(const Dev &D) {
    if (D.prec == HD_FP64) return D.lanes == 4 ? k_persist<HD_FP64, 4> : k_persist<HD_FP64, 1>;
    return D.lanes == 4 ? k_persist<HD_FP32_SPLIT, 4> : k_persist<HD_FP32_SPLIT, 1>;
}
// Lets kernel f use `bytes` of dynamic shared memory.  The limit belongs to the
// kernel on a device, not to a context, and contexts of different size live
// side by side, so it is never lowered.
static cudaError_t allow_smem(const void *f, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, int> most;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    int &m = most[std::make_pair(dev, f)];
    const int want = bytes > m ? bytes : m;
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, want);
    if (e == cudaSuccess) m = want;
    return e;
}
cudaError_t nl_configure(const Dev &D, int *nl_blocks_per_sm) {
    const int bytes = (int)nl_smem_bytes(D, NL_THREADS / 32), pbytes = (int)persist_smem_bytes(D);
    cudaError_t e = allow_smem((const void *)k_nlist, bytes);
    if (e != cudaSuccess) return e;
    // the row builder is latency-bound: launch as many CTAs as fit
    *nl_blocks_per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(nl_blocks_per_sm, k_nlist, NL_THREADS, bytes);
    if (e != cudaSuccess) return e;
    return allow_smem((const void *)persist_kernel(D), pbytes);
}

void launch_init(const Dev &D, const int *draw_vel, cudaStream_t s) {
    k_init<<<D.ntile, nthr(D), 0, s>>>(D, draw_vel);
}
void launch_rebuild_prep(const Dev &D, cudaStream_t s) {
    const bool big = D.nrep > PLAN_MAX;
    if (big) k_rebuild_plan<<<1, 32, 0, s>>>(D);
    k_bin<<<D.nl_grid, 256, big ? 0 : 3 * D.nrep * sizeof(int), s>>>(D, big);
    k_cellsort<<<D.nl_grid, 128, 4 * D.cell_cap * sizeof(int), s>>>(D);
}
void launch_nlist(const Dev &D, cudaStream_t s) {
    k_nlist<<<D.nl_grid, NL_THREADS, nl_smem_bytes(D, NL_THREADS / 32), s>>>(D);
}
void launch_rebuild(const Dev &D, cudaStream_t s) {
    launch_rebuild_prep(D, s);
    launch_nlist(D, s);
}
template <int S>
static void pair_of(const Dev &D, int kind, cudaStream_t s) {
    const int grid = D.ntile * D.split, n = unit_threads(D);
    if (D.prec == HD_FP64) {
        if (kind == PAIR_QUENCH) k_pair64<true, false, false, S><<<grid, n, 0, s>>>(D);
        else if (kind == PAIR_ENERGY) k_pair64<false, true, true, S><<<grid, n, 0, s>>>(D);
        else if (kind == PAIR_FULL) k_pair64<false, false, true, S><<<grid, n, 0, s>>>(D);
        else if (D.bias_on) k_pair64_lazy<S><<<grid, n, 0, s>>>(D);
        else k_pair64<false, false, false, S><<<grid, n, 0, s>>>(D);
    } else {
        if (kind == PAIR_QUENCH) k_pair32<true, false, false, S><<<grid, n, 0, s>>>(D, SWEEP_ALL);
        else if (kind == PAIR_ENERGY) k_pair32<false, true, true, S><<<grid, n, 0, s>>>(D, SWEEP_ALL);
        else if (kind == PAIR_FULL) k_pair32<false, false, true, S><<<grid, n, 0, s>>>(D, SWEEP_ALL);
        else k_pair32<false, false, false, S><<<grid, n, 0, s>>>(D, SWEEP_PLAIN);
        if (kind == PAIR_LAZY && D.bias_on) k_pair_hot<<<D.hot_grid, n, 0, s>>>(D);
    }
}
void launch_pair(const Dev &D, int kind, cudaStream_t s) {
    if (D.lanes == 4) pair_of<4>(D, kind, s);
    else pair_of<1>(D, kind, s);
}
void launch_scalar(const Dev &D, int mode, bool lazy, bool list, cudaStream_t s) {
    const bool more = D.lazy_h && D.bias_on;
    const int n = unit_threads(D), g = D.hot_grid, li = list && more && D.prec != HD_FP64;
    k_scalar<<<D.nrep, sc_threads(D), 0, s>>>(D, mode, lazy && more, li);
    if (!lazy || !more) return;
    if (D.prec != HD_FP64) k_scalar_late<HD_FP32_SPLIT, 1><<<g, n, 0, s>>>(D, mode, li);
    else if (D.lanes == 4) k_scalar_late<HD_FP64, 4><<<g, n, 0, s>>>(D, mode, li);
    else k_scalar_late<HD_FP64, 1><<<g, n, 0, s>>>(D, mode, li);
}
void launch_update(const Dev &D, int mode, cudaStream_t s) {
    if (D.prec == HD_FP64) k_update64<<<D.ntile, nthr(D), 0, s>>>(D, mode);
    else k_update32<<<D.ntile, nthr(D), 0, s>>>(D, mode);
}
void launch_obs(const Dev &D, cudaStream_t s) { k_obs<<<D.nrep, 32, 0, s>>>(D); }
void launch_nhc(const Dev &D, int mode, cudaStream_t s) { k_nhc<<<D.nrep, 32, 0, s>>>(D, mode); }
void launch_qinit(const Dev &Q, const Dev &M, cudaStream_t s) { k_qinit<<<Q.ntile, nthr(Q), 0, s>>>(Q, M); }
void launch_qiter(const Dev &Q, int max_iter, cudaStream_t s) {
    launch_rebuild(Q, s);
    launch_pair(Q, PAIR_QUENCH, s);
    k_qscalar<<<Q.nrep, sc_threads(Q), 0, s>>>(Q, max_iter);
    k_qupdate<<<Q.ntile, nthr(Q), 0, s>>>(Q);
}
void launch_qdisp(const Dev &Q, cudaStream_t s) { k_qdisp<<<Q.ntile, nthr(Q), 0, s>>>(Q); }
int persist_blocks_per_sm(const Dev &D) {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, persist_kernel(D), unit_threads(D), persist_smem_bytes(D));
    return nb;
}
cudaError_t launch_persist(const Dev &D, int grid, int nsteps, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(D.bar, 0, sizeof(unsigned long long) * D.nrep, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(D.err + 3, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(unit_threads(D));
    cfg.dynamicSmemBytes = persist_smem_bytes(D);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, persist_kernel(D), D, nsteps);
}
void launch_adopt(const Dev &Q, const Dev &M, const int *adopt, cudaStream_t s) {
    k_adopt<<<M.ntile, nthr(M), 0, s>>>(Q, M, adopt);
}

}  // namespace hd
