// hd_static.cu -- hd_nlist_static: the neighbour-list build of one replica
// with no device allocation at all.
//
// Some callers cannot let a library allocate device memory: a host program
// that budgets every byte of the GPU itself, or a loop that cannot afford
// the latency or the failure of an allocation.  This entry point takes only
// the caller's input and output buffers and keeps its scratch (fixed-point
// positions, cell ids, cell counts and cell lists, an error word) in one
// file-scope device array of fixed size, which every GPU that loads the
// library holds until the process exits.
//
// The first call on a device looks up that array's device address
// (cudaGetSymbolAddress, with that device current) and keeps it.  Under
// CUDA's lazy module loading that first call is also when the module, and
// with it the array, is committed on the device, so it can itself fail for
// want of memory: make it at start-up, before the program reserves the rest
// of the GPU's memory (or run with CUDA_MODULE_LOADING=EAGER).  Every call
// synchronises its stream (it reads back the error word), so no call may be
// made while that stream is being captured into a graph.  Every call shares the array and
// it keeps the last call's contents: the counts, the extent and the error
// word are cleared at the start of each call.  Calls on one device therefore
// take turns: each holds that device's lock from its first launch until its
// stream is synchronised.  (The row build takes the grid and the atoms from the
// array, so a call that overlapped another would write rows of its atoms.)
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <mutex>

#include "hd_internal.cuh"

namespace {

constexpr int S_MAX_ATOMS = 65536;
constexpr int S_MAX_CELLS = 16384;
constexpr int S_CELL_CAP = 64;
constexpr int S_MAX_NB = 160;
constexpr int S_SPARSE = 6;      // mean atoms a cell below which the row build takes a warp a row
constexpr int S_THREADS = 256;   // row build: 8 warps share one cell's staged stencil

struct Grid {
    int nc[3], periodic[3], ncell;
    double L[3], invL[3], scale[3], origin[3], lo[3], inv_w[3];
    float lsb[3];
    double rl, rl2;
    float rl2_lo, rl2_hi;
};

// What a call clears comes first, so that one memset clears it: cell counts,
// the positions' extent and the error word.
struct StaticScratch {
    int cell_cnt[S_MAX_CELLS];
    unsigned long long ext[6];   // per axis: max of the complement (the minimum), then max, of the ordered bits
    int err[4];
    Grid grid;
    int4 pfix[S_MAX_ATOMS];
    int cell_atoms[S_MAX_CELLS * S_CELL_CAP];
};

static __device__ __align__(256) StaticScratch g_static_scratch;

// Cell along one axis: exact integer map of the fixed-point image on a
// periodic axis; FP64 quotient on an open axis (an FP32 quotient would round
// by more than the cells' 1e-4 width margin near 1000 cells).
__device__ __forceinline__ int s_cell(const Grid &G, int a, int q, double x) {
    if (G.nc[a] <= 1) return 0;
    if (G.periodic[a]) return (int)(((unsigned long long)(unsigned int)q * (unsigned long long)G.nc[a]) >> 32);
    const int c = (int)floor((x - G.lo[a]) * G.inv_w[a]);
    return c < 0 ? 0 : (c >= G.nc[a] ? G.nc[a] - 1 : c);
}

// Order-preserving map of a double onto unsigned 64-bit integers, so that
// integer atomicMin/atomicMax give the FP64 minimum and maximum.
__device__ __forceinline__ unsigned long long ord_bits(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__host__ __device__ inline double ord_value(unsigned long long u) {
    const unsigned long long b = (u >> 63) ? (u & 0x7FFFFFFFFFFFFFFFull) : ~u;
    double x;
    memcpy(&x, &b, 8);
    return x;
}

// Extent of the positions along every axis.  The minimum is kept as the
// maximum of the complemented bits, so that zero is the start of both.  One
// atomic per axis end and CTA: with one per atom the 14,272 additions to each
// of the six words ran one after another.
__global__ void k_s_extent(StaticScratch *S, const double *pos, int n) {
    __shared__ unsigned long long sm[6];
    if (threadIdx.x < 6) sm[threadIdx.x] = 0ull;
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    for (int a = 0; a < 3; ++a) {
        unsigned long long hi = i < n ? ord_bits(pos[3 * i + a]) : 0ull, lo = i < n ? ~hi : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long th = __shfl_down_sync(0xffffffffu, hi, o), tl = __shfl_down_sync(0xffffffffu, lo, o);
            hi = th > hi ? th : hi;
            lo = tl > lo ? tl : lo;
        }
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&sm[2 * a], lo);
            atomicMax(&sm[2 * a + 1], hi);
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) atomicMax(&S->ext[threadIdx.x], sm[threadIdx.x]);
}

// The cell grid: cells at least rl wide (periodic axes tile the box exactly;
// an open axis spans the positions of this call).  It is made on the device,
// from the extent that k_s_extent left there, so that a call waits for the
// GPU once and not twice.  Returns 0 or the error the call ends with.
__device__ int s_grid(const StaticScratch *S, Grid &G, const double *box, bool need_ext) {
    double mn[3] = {0, 0, 0}, mx[3] = {0, 0, 0};
    if (need_ext)
        for (int a = 0; a < 3; ++a) {
            mn[a] = ord_value(~S->ext[2 * a]);
            mx[a] = ord_value(S->ext[2 * a + 1]);
            if (!isfinite(mn[a]) || !isfinite(mx[a])) return HD_ERR_NUMERIC;
        }
    long long ncell = 1;
    for (int a = 0; a < 3; ++a) {
        if (G.periodic[a]) {
            if (!(box[a] > 0.0)) return HD_ERR_ARG;
            G.L[a] = box[a];
            G.invL[a] = 1.0 / box[a];
            G.scale[a] = 4294967296.0 / box[a];
            G.lsb[a] = (float)(box[a] / 4294967296.0);
            const double nc = floor(box[a] / (G.rl * (1.0 + 1e-6)));
            G.nc[a] = nc >= 3.0 ? (nc < 1024.0 ? (int)nc : 1024) : 1;
        } else if (mx[a] > mn[a]) {
            double span = 64.0;
            while (span < 4.0 * (mx[a] - mn[a]) + 64.0) span *= 2.0;
            G.origin[a] = 0.5 * (mn[a] + mx[a]);
            G.scale[a] = 4294967296.0 / span;
            G.lsb[a] = (float)(span / 4294967296.0);
            const double w = G.rl * (1.0 + 1e-4);
            G.inv_w[a] = 1.0 / w;
            G.lo[a] = mn[a] - 1.0;
            const double nc = ceil((mx[a] + 1.0 - G.lo[a]) / w);
            G.nc[a] = nc >= 1.0 ? (nc < 1024.0 ? (int)nc : 1024) : 1;
        }
        if (G.nc[a] >= 1024) return HD_ERR_ARG;
        ncell *= G.nc[a];
    }
    if (ncell > S_MAX_CELLS) return HD_ERR_ARG;
    G.ncell = (int)ncell;
    return 0;
}

__device__ __forceinline__ double s_r2(const Grid &G, const double *a, const double *b) {
    double d[3];
    for (int k = 0; k < 3; ++k) {
        d[k] = __dsub_rn(a[k], b[k]);
        if (G.periodic[k]) d[k] = __dsub_rn(d[k], __dmul_rn(G.L[k], rint(d[k] * G.invL[k])));
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
}

// Every CTA makes the grid for itself (a few divisions); the first one also
// leaves it for the row build, or the error that ends the call there.
__global__ void k_s_bin(StaticScratch *S, Grid G0, double bx, double by, double bz, bool need_ext, const double *pos,
                        int n) {
    __shared__ Grid G;
    __shared__ int bad;
    if (threadIdx.x == 0) {
        const double box[3] = {bx, by, bz};
        Grid g = G0;
        bad = s_grid(S, g, box, need_ext);
        G = g;
        if (blockIdx.x == 0) {
            if (bad) {
                g.ncell = 0;
                atomicCAS(&S->err[0], 0, bad);
            }
            S->grid = g;
        }
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (bad || i >= n) return;
    int q[3];
    for (int a = 0; a < 3; ++a) {
        if (G.scale[a] == 0.0) { q[a] = 0; continue; }
        const long long v = __double2ll_rn((pos[3 * i + a] - G.origin[a]) * G.scale[a]);
        q[a] = (int)(unsigned int)(unsigned long long)v;
    }
    const int cx = s_cell(G, 0, q[0], pos[3 * i]), cy = s_cell(G, 1, q[1], pos[3 * i + 1]),
              cz = s_cell(G, 2, q[2], pos[3 * i + 2]);
    const int c = (cz * G.nc[1] + cy) * G.nc[0] + cx;
    S->pfix[i] = make_int4(q[0], q[1], q[2], c);
    const int slot = atomicAdd(&S->cell_cnt[c], 1);
    if (slot < S_CELL_CAP) S->cell_atoms[c * S_CELL_CAP + slot] = i;
    else atomicCAS(&S->err[0], 0, HD_ERR_OVERFLOW);
}

// Stencil cell of `lane` around cell c: (lane % 3, lane / 3 % 3, lane / 9) of
// -1, 0, 1 along each axis, as far as it exists; its atoms (0 where there is none).
__device__ __forceinline__ int s_stencil(const StaticScratch *S, const Grid &G, int c, int lane, int &cell) {
    const int ci[3] = {c % G.nc[0], (c / G.nc[0]) % G.nc[1], c / (G.nc[0] * G.nc[1])};
    const int d[3] = {lane % 3 - 1, (lane / 3) % 3 - 1, lane / 9 - 1};
    bool ok = lane < 27;
    int q[3];
    for (int a = 0; a < 3; ++a) {
        q[a] = ci[a] + d[a];
        if (G.nc[a] == 1) {
            ok = ok && d[a] == 0;
            q[a] = 0;
        } else if (G.periodic[a]) {
            q[a] = (q[a] + G.nc[a]) % G.nc[a];
        } else {
            ok = ok && q[a] >= 0 && q[a] < G.nc[a];
        }
    }
    cell = ok ? (q[2] * G.nc[1] + q[1]) * G.nc[0] + q[0] : 0;
    return ok ? min(S->cell_cnt[cell], S_CELL_CAP) : 0;
}

// Sum over the lanes up to this one.
__device__ __forceinline__ int s_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Is j (image pj) in row i: the FP32 test on exact fixed-point differences
// decides outside a thin band.
__device__ __forceinline__ bool s_in(const Grid &G, const double *pos, int i, int4 pi, int j, int4 pj) {
    if (j == i) return false;
    const float dx = (float)(int)((unsigned)pi.x - (unsigned)pj.x) * G.lsb[0];
    const float dy = (float)(int)((unsigned)pi.y - (unsigned)pj.y) * G.lsb[1];
    const float dz = (float)(int)((unsigned)pi.z - (unsigned)pj.z) * G.lsb[2];
    const float r2 = dx * dx + dy * dy + dz * dz;
    if (r2 < G.rl2_lo) return true;
    if (r2 >= G.rl2_hi) return false;
    return s_r2(G, pos + 3 * (size_t)i, pos + 3 * (size_t)j) < G.rl2;
}

// A warp adds its accepted candidates to the row in buf (cnt so far).
__device__ __forceinline__ int s_add(bool in, int j, int lane, int maxnb, int cnt, int *buf) {
    const unsigned hit = __ballot_sync(0xffffffffu, in);
    const int at = cnt + __popc(hit & ((1u << lane) - 1u));
    if (in && at < maxnb) buf[at] = j;
    return cnt + __popc(hit);
}

// The warp sorts the cnt entries in buf by rank (the count of smaller ones)
// and writes row i.
__device__ __forceinline__ void s_write_row(StaticScratch *S, int i, int cnt, int maxnb, int lane, int *buf, int *srt,
                                            int *nbr, int *nnb) {
    if (cnt > maxnb) {
        if (lane == 0) atomicCAS(&S->err[0], 0, HD_ERR_OVERFLOW);
        cnt = maxnb;
    }
    // fill the last group of four so that it ranks after every entry
    if (lane < 4 && (cnt & ~3) + lane >= cnt && (cnt & ~3) + lane < S_MAX_NB) buf[(cnt & ~3) + lane] = 0x7fffffff;
    __syncwarp();
    const int4 *b4 = reinterpret_cast<const int4 *>(buf);
    for (int k = lane; k < cnt; k += 32) {
        const int v = buf[k];
        int rank = 0;
        for (int q = 0; q < (cnt + 3) >> 2; ++q) {
            const int4 u = b4[q];
            rank += (u.x < v) + (u.y < v) + (u.z < v) + (u.w < v);
        }
        srt[rank] = v;
    }
    __syncwarp();
    int *row = nbr + (size_t)i * maxnb;
    for (int k = lane; k < maxnb; k += 32) row[k] = k < cnt ? srt[k] : -1;
    if (lane == 0) nnb[i] = cnt;
    __syncwarp();
}

// Row i: every j != i with FP64 minimum-image r^2 < rl^2, ascending j.
//
// One CTA builds the rows of one cell's atoms: it stages the cell's stencil
// (27 cells, ~675 candidates in a dense crystal) in shared memory once, then
// a warp per atom tests 32 candidates at a time, packs the accepted ones by
// ballot and sorts them by rank (read four at a time from shared memory).
// Both loops are issue-bound: ~21 x 20 + 480
// instructions an atom.  A thread per atom that kept its row sorted in global
// memory by insertion made a call at 14,272 atoms (rows of 76) take 978 us;
// with this build, and one wait for the GPU instead of two, it takes 92 us.
//
// Where cells hold few atoms (below S_SPARSE on the average: a gas, a thin
// film under much vacuum) a CTA a cell leaves most warps without a row and
// waits at the staging barriers instead.  There a warp takes a row by itself
// and reads the candidates where they lie: 20,000 atoms in 15,625 cells 59 us
// a call, with a CTA a cell 143, with a thread an atom 120.  1,728 cells of 6
// atoms on the average 50 us and 58, of 8 atoms 69 and 62, of 12 94 and 82.
__global__ void __launch_bounds__(S_THREADS) k_s_list(StaticScratch *S, const double *pos, int n, int maxnb, int *nbr,
                                                     int *nnb) {
    __shared__ Grid G;
    __shared__ int s_off[28], s_cell_id[27], s_nst;
    __shared__ int4 sp[27 * S_CELL_CAP];
    __shared__ __align__(16) int buf[S_THREADS / 32][S_MAX_NB];
    __shared__ int srt[S_THREADS / 32][S_MAX_NB];
    if (threadIdx.x == 0) G = S->grid;
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    if (n < S_SPARSE * G.ncell) {
        for (int i = blockIdx.x * (S_THREADS / 32) + w; i < n; i += gridDim.x * (S_THREADS / 32)) {
            const int4 pi = S->pfix[i];
            int cell;
            const int mine = s_stencil(S, G, pi.w, lane, cell), incl = s_scan(mine, lane);
            const int tot = __shfl_sync(full, incl, 31), first = cell * S_CELL_CAP - (incl - mine);
            int cnt = 0;
            for (int base = 0; base < tot; base += 32) {
                const int t = base + lane;
                int k = 0;        // stencil cell of candidate t: the first one whose sum is above t
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
                    if (__shfl_sync(full, incl, k + o - 1) <= t) k += o;
                const int at = __shfl_sync(full, first, k) + t;
                const int j = t < tot ? S->cell_atoms[at] : i;
                cnt = s_add(s_in(G, pos, i, pi, j, S->pfix[j]), j, lane, maxnb, cnt, buf[w]);
            }
            s_write_row(S, i, cnt, maxnb, lane, buf[w], srt[w], nbr, nnb);
        }
        return;
    }
    for (int c = blockIdx.x; c < G.ncell; c += gridDim.x) {
        const int m = min(S->cell_cnt[c], S_CELL_CAP);
        if (m == 0) continue;   // the same for every thread
        if (w == 0) {
            int cell;
            const int cnt = s_stencil(S, G, c, lane, cell), incl = s_scan(cnt, lane);
            const unsigned has = __ballot_sync(full, cnt > 0);
            if (cnt > 0) {
                const int k = __popc(has & ((1u << lane) - 1u));
                s_cell_id[k] = cell;
                s_off[k] = incl - cnt;
            }
            if (lane == 31) {
                s_nst = __popc(has);
                s_off[__popc(has)] = incl;
            }
        }
        __syncthreads();
        const int nst = s_nst, tot = s_off[nst];
        // stage: a warp per stencil cell
        for (int k = w; k < nst; k += S_THREADS / 32) {
            const int o = s_off[k], mk = s_off[k + 1] - o, base = s_cell_id[k] * S_CELL_CAP;
            for (int q = lane; q < mk; q += 32) {
                const int j = S->cell_atoms[base + q];
                int4 p = S->pfix[j];
                p.w = j;
                sp[o + q] = p;
            }
        }
        __syncthreads();
        for (int a = w; a < m; a += S_THREADS / 32) {
            const int i = S->cell_atoms[c * S_CELL_CAP + a];
            const int4 pi = S->pfix[i];
            int cnt = 0;
            for (int base = 0; base < tot; base += 32) {
                const int4 pj = base + lane < tot ? sp[base + lane] : make_int4(0, 0, 0, i);
                cnt = s_add(s_in(G, pos, i, pi, pj.w, pj), pj.w, lane, maxnb, cnt, buf[w]);
            }
            s_write_row(S, i, cnt, maxnb, lane, buf[w], srt[w], nbr, nnb);
        }
        __syncthreads();   // the staging buffer is reused by the next cell
    }
}

std::mutex g_mu[64];
StaticScratch *g_addr[64] = {};

}  // namespace

extern "C" hd_status hd_nlist_static(const double *d_pos, int n_atoms, const double box[3],
                                     const uint8_t periodic[3], double rl, int maxnb, int32_t *d_nbr,
                                     int32_t *d_nnb, void *cuda_stream) {
    if (!d_pos || !d_nbr || !d_nnb || !box || !periodic) return HD_ERR_ARG;
    if (n_atoms <= 0 || n_atoms > S_MAX_ATOMS) return HD_ERR_ARG;
    if (maxnb <= 0 || maxnb > S_MAX_NB || !(rl > 0.0)) return HD_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return HD_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_mu[dev]);
    if (!g_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) return HD_ERR_CUDA;
        g_addr[dev] = static_cast<StaticScratch *>(p);
    }
    StaticScratch *S = g_addr[dev];
    cudaStream_t s = (cudaStream_t)cuda_stream;
    Grid G;
    memset(&G, 0, sizeof G);
    G.rl = rl;
    G.rl2 = rl * rl;
    G.rl2_lo = (float)(G.rl2 * (1.0 - 1.0 / 4096.0));
    G.rl2_hi = (float)(G.rl2 * (1.0 + 1.0 / 4096.0));
    bool need_ext = false;
    for (int a = 0; a < 3; ++a) {
        G.periodic[a] = periodic[a] ? 1 : 0;
        G.nc[a] = 1;
        need_ext |= !periodic[a];
    }
    if (cudaMemsetAsync(S, 0, offsetof(StaticScratch, grid), s) != cudaSuccess) return HD_ERR_CUDA;
    const int nb = (n_atoms + 127) / 128;
    if (need_ext) k_s_extent<<<nb, 128, 0, s>>>(S, d_pos, n_atoms);
    k_s_bin<<<nb, 128, 0, s>>>(S, G, box[0], box[1], box[2], need_ext, d_pos, n_atoms);
    // the number of cells stays on the device: a fixed grid (five CTAs an SM
    // fit beside their shared memory) strides over them
    k_s_list<<<std::min(760, n_atoms), S_THREADS, 0, s>>>(S, d_pos, n_atoms, maxnb, d_nbr, d_nnb);
    if (cudaGetLastError() != cudaSuccess) return HD_ERR_CUDA;
    int err[4];
    if (cudaMemcpyAsync(err, S->err, sizeof err, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return HD_ERR_CUDA;
    return err[0] ? (hd_status)err[0] : HD_OK;
}
