// noalloc.cu -- md_forces_static: pair forces for a small system without any device allocation.
//
// Some callers cannot allocate device memory at the point where they need forces: host code
// inside another runtime or framework that hands out only pre-planned buffers and owns the
// device allocator, plug-ins that run between someone else's kernels where a cudaMalloc/cudaFree
// would take the device-wide synchronisation these calls can imply, or code that has no
// workspace to hand.  For them this entry point keeps its cell-list scratch (occupancy counts,
// prefix sums, cell order, cell-local positions) in one file-scope __device__ array of fixed
// size, instead of a caller-provided workspace.  The computation is the force pass of
// md_compute_forces on a plain cell list of side >= r_c (no neighbour matrix): FP32 pair
// arithmetic on cell-local coordinates, per-atom sums in a fixed order (the nine rows of cells
// around an atom one lane each, their atoms in cell order and ascending within a cell, then the
// nine sums in a fixed tree), so repeated calls on the same input give the same bits.
//
// A call of a few thousand atoms is bound by its launches, so up to NA_CLUSTER_ATOMS the cell list
// is made by one kernel, a cluster of 8 CTAs that meet between its phases.
//
// Limits and sharing:
//   * at most NA_MAX_ATOMS atoms and NA_MAX_CELLS cells (both 65536); larger requests fail with
//     MD_ERR_INVALID_ARG before any work is queued;
//   * every GPU that loads the library keeps the NA_BYTES array until the process exits;
//   * all calls share the array and it keeps the last call's contents: each call clears the
//     occupancy counters itself, and calls whose work overlaps on the GPU (different streams
//     without ordering between them) race on the array and must not be issued;
//   * the host needs the array's device address: the first call on each device looks it up
//     (cudaGetSymbolAddress) with that device current, so that first call should come before any
//     stream capture; the address is kept for the life of the process, so the entry point must
//     not be used after cudaDeviceReset on that device.
#include <mutex>
#include <string>

#include "gbmd_internal.cuh"

namespace {

constexpr int NA_MAX_ATOMS = 1 << 16;
constexpr int NA_MAX_CELLS = 1 << 16;
constexpr int NA_THREADS = 128;
constexpr size_t NA_COUNT_OFF = 0;                                              // int32[cells]
constexpr size_t NA_START_OFF = NA_COUNT_OFF + sizeof(int32_t) * NA_MAX_CELLS;  // int32[cells+1]
constexpr size_t NA_PERM_OFF = NA_START_OFF + sizeof(int32_t) * (NA_MAX_CELLS + 64);
constexpr size_t NA_CELL_OFF = NA_PERM_OFF + sizeof(int32_t) * NA_MAX_ATOMS;
constexpr size_t NA_LAYER_OFF = NA_CELL_OFF + sizeof(int32_t) * NA_MAX_ATOMS;
constexpr size_t NA_POS_OFF = NA_LAYER_OFF + sizeof(int32_t) * NA_MAX_ATOMS;     // float4[atoms]
constexpr size_t NA_SPOS_OFF = NA_POS_OFF + sizeof(float4) * NA_MAX_ATOMS;       // float4[atoms], cell order
constexpr size_t NA_TOTAL_OFF = NA_SPOS_OFF + sizeof(float4) * NA_MAX_ATOMS;     // int32[64]
constexpr size_t NA_BYTES = NA_TOTAL_OFF + sizeof(int32_t) * 64;                 // 3.25 MiB

// The cluster works on 8 SMs, whose FP64 pipes the binning fills.  Whole calls, cluster / separate
// kernels (/ before either, with a thread per atom in the forces): 5003 WCA atoms 34 / 43 (60) us, LJ
// 56 / 61 (180) us, 12000 LJ atoms 69 / 65 (225) us; the line is where each thread has one atom.
constexpr int NA_CLUSTER = 8;
constexpr int NA_CLUSTER_THREADS = 1024;
constexpr int NA_CLUSTER_ATOMS = NA_CLUSTER * NA_CLUSTER_THREADS;

static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

struct NaView {
    int32_t* count;
    int32_t* start;
    int32_t* perm;
    int32_t* cell;
    int32_t* layer;           // layer slot in the cell; after the ordering the packed cell, in cell order
    float4* pos;
    float4* spos;             // cell-local positions in cell order, the atom's index in .w
    int32_t* total;           // atoms in the cells of each CTA of the cluster
};

struct NaGeom {
    double L[3], w[3], s[3];
    float wf[3];
    float wlo[3];          // (float) (w - wf), added after o wf to keep the distances unbiased
    int nc[3];
    int ncells;
    int n;
    float rc2f, sig2f, eps4f, eps48f, ucf;
};

NaView view_of(void* base)
{
    unsigned char* b = static_cast<unsigned char*>(base);
    return NaView{reinterpret_cast<int32_t*>(b + NA_COUNT_OFF), reinterpret_cast<int32_t*>(b + NA_START_OFF),
                  reinterpret_cast<int32_t*>(b + NA_PERM_OFF), reinterpret_cast<int32_t*>(b + NA_CELL_OFF),
                  reinterpret_cast<int32_t*>(b + NA_LAYER_OFF), reinterpret_cast<float4*>(b + NA_POS_OFF),
                  reinterpret_cast<float4*>(b + NA_SPOS_OFF), reinterpret_cast<int32_t*>(b + NA_TOTAL_OFF)};
}

// cell of atom i and its cell-local FP32 position, which go to V.cell and V.pos; returns the cell
__device__ __forceinline__ int na_place(const NaView& V, const NaGeom& G, const double* __restrict__ x, int i)
{
    int c[3];
    float l[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double xa = x[3 * i + a];
        // inside [0, L) on the bit patterns (for x >= 0 they order as the values do), which keeps the
        // comparisons off the FP64 pipe
        if (static_cast<unsigned long long>(__double_as_longlong(xa)) >=
            static_cast<unsigned long long>(__double_as_longlong(G.L[a]))) {
            if (xa < 0.0) xa += G.L[a];
            if (xa >= G.L[a]) xa -= G.L[a];
            if (!(xa >= 0.0 && xa < G.L[a])) {       // more than one period away: whole periods
                xa -= G.L[a] * floor(xa / G.L[a]);
                if (xa < 0.0) xa += G.L[a];
                if (xa >= G.L[a]) xa -= G.L[a];
            }
        }
        int ca = int(floor(xa * G.s[a]));
        ca = min(max(ca, 0), G.nc[a] - 1);
        c[a] = ca;
        l[a] = __double2float_rn(xa - double(ca) * G.w[a]);
    }
    const int cell = (c[2] * G.nc[1] + c[1]) * G.nc[0] + c[0];
    V.pos[i] = make_float4(l[0], l[1], l[2], __uint_as_float(gbmd::pack_cell(c[0], c[1], c[2])));
    V.cell[i] = cell;
    return cell;
}

// place of atom i in the cell order: its rank among its cell's atoms (listed in perm in the order of
// the atomic layer slots)
__device__ __forceinline__ void na_order(const NaView& V, int i, int cell, int b, int e)
{
    int rank = 0;
    for (int k = b; k < e; ++k) rank += (__ldcg(V.perm + k) < i) ? 1 : 0;
    const float4 p = __ldcg(V.pos + i);
    V.spos[b + rank] = make_float4(p.x, p.y, p.z, __int_as_float(i));
    V.layer[b + rank] = int(__float_as_uint(p.w));   // the layer slots have been read
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The whole cell list of a small system: counters cleared, atoms binned, prefix sum, atoms listed by
// cell, ordered within cells.  The CTAs of the cluster meet after each phase; what they read of each
// other's goes through L2.
__global__ void __cluster_dims__(NA_CLUSTER, 1, 1) __launch_bounds__(NA_CLUSTER_THREADS)
    k_na_cells(NaView V, NaGeom G, const double* __restrict__ x)
{
    __shared__ int sh[33];
    const int cta = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int tid = cta * NA_CLUSTER_THREADS + threadIdx.x;
    constexpr int STRIDE = NA_CLUSTER * NA_CLUSTER_THREADS;
    constexpr int MINE = (NA_CLUSTER_ATOMS + STRIDE - 1) / STRIDE;        // atoms per thread
    for (int c = tid; c < G.ncells; c += STRIDE) V.count[c] = 0;
    cluster_sync();
    int cell[MINE], layer[MINE];
#pragma unroll
    for (int q = 0; q < MINE; ++q) {
        const int i = tid + q * STRIDE;
        if (i < G.n) {
            cell[q] = na_place(V, G, x, i);
            layer[q] = atomicAdd(&V.count[cell[q]], 1);
        }
    }
    cluster_sync();
    // prefix sum: this CTA's contiguous share of the cells, `per` consecutive ones per thread
    const int share = (G.ncells + NA_CLUSTER - 1) / NA_CLUSTER, per = (share + NA_CLUSTER_THREADS - 1) / NA_CLUSTER_THREADS;
    const int c0 = cta * share + threadIdx.x * per;
    const int c1 = min(min(c0 + per, (cta + 1) * share), G.ncells);
    int mine = 0;
    for (int c = c0; c < c1; ++c) mine += __ldcg(V.count + c);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int wv = sh[lane];
        int wi = wv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        sh[lane] = wi - wv;
        if (lane == 31) V.total[cta] = wi;
    }
    __syncthreads();
    cluster_sync();
    int run = sh[wid] + incl - mine;
    for (int q = 0; q < cta; ++q) run += __ldcg(V.total + q);
    for (int c = c0; c < c1; ++c) {
        V.start[c] = run;
        run += __ldcg(V.count + c);
    }
    if (tid == 0) V.start[G.ncells] = G.n;
    cluster_sync();
    int b[MINE];
#pragma unroll
    for (int q = 0; q < MINE; ++q) {
        const int i = tid + q * STRIDE;
        if (i < G.n) {
            b[q] = __ldcg(V.start + cell[q]);
            V.perm[b[q] + layer[q]] = i;
        }
    }
    cluster_sync();
#pragma unroll
    for (int q = 0; q < MINE; ++q) {
        const int i = tid + q * STRIDE;
        if (i < G.n) na_order(V, i, cell[q], b[q], __ldcg(V.start + cell[q] + 1));
    }
}

// the same in separate kernels: cell of each atom, cell-local FP32 position, layer slot in its cell
__global__ void __launch_bounds__(NA_THREADS) k_na_bin(NaView V, NaGeom G, const double* __restrict__ x)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.n) return;
    V.layer[i] = atomicAdd(&V.count[na_place(V, G, x, i)], 1);
}

// exclusive prefix sum of the occupancies, one block
__global__ void __launch_bounds__(1024) k_na_scan(NaView V, NaGeom G)
{
    __shared__ int sh[33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int carry = 0;
    for (int c0 = 0; c0 < G.ncells; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const int v = (c < G.ncells) ? V.count[c] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) sh[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            const int wv = sh[lane];
            int wi = wv;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            sh[lane] = wi - wv;
            if (lane == 31) sh[32] = wi;
        }
        __syncthreads();
        if (c < G.ncells) V.start[c] = carry + sh[wid] + incl - v;
        carry += sh[32];
        __syncthreads();
    }
    if (threadIdx.x == 0) V.start[G.ncells] = carry;
}

__global__ void __launch_bounds__(NA_THREADS) k_na_scatter(NaView V, NaGeom G)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < G.n) V.perm[V.start[V.cell[i]] + V.layer[i]] = i;
}

// the atomic layer slots leave the order inside a cell to chance; ranking each cell's atoms by
// index fixes the summation order of every force, so repeated calls give identical bits
__global__ void __launch_bounds__(NA_THREADS) k_na_order(NaView V, NaGeom G)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.n) return;
    const int c = V.cell[i];
    na_order(V, i, c, V.start[c], V.start[c + 1]);
}

// F1 over the 27 cells around each atom; force on i is g (x_i - x_j).  Nine lanes per atom, one per
// row of cells, whose three cells are one run of the cell order (or three, where the row wraps): a
// thread per atom walked its 27 cells one dependent load after the other.  Lane r's sums are added
// as ((r, r+3, r+6), then r = 0, 1, 2).
constexpr int NA_GROUP = 3;                                  // atoms per warp
__global__ void __launch_bounds__(NA_THREADS) k_na_forces(NaView V, NaGeom G, double* __restrict__ f,
                                                          double* __restrict__ u)
{
    const int lane = threadIdx.x & 31, a = lane / 9, r = lane - 9 * a;
    const int k = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * NA_GROUP + a;
    const bool act = a < NA_GROUP && k < G.n;
    float fx = 0.f, fy = 0.f, fz = 0.f, ui = 0.f;
    int i = 0;
    if (act) {
        const float4 pi = __ldg(V.spos + k);
        i = __float_as_int(pi.w);
        int cx, cy, cz;
        gbmd::unpack_cell(uint32_t(__ldg(V.layer + k)), cx, cy, cz);
        const int oy = r % 3 - 1, oz = r / 3 - 1;
        int ny = cy + oy; ny += (ny < 0) ? G.nc[1] : 0; ny -= (ny >= G.nc[1]) ? G.nc[1] : 0;
        int nz = cz + oz; nz += (nz < 0) ? G.nc[2] : 0; nz -= (nz >= G.nc[2]) ? G.nc[2] : 0;
        const int32_t* __restrict__ row = V.start + (nz * G.nc[1] + ny) * G.nc[0];
        auto run = [&](int kb, int ke, int k1, int k2) {     // o_x + 1 = (q >= k1) + (q >= k2)
            for (int q = kb; q < ke; ++q) {
                const float4 pj = __ldg(V.spos + q);
                const float ox = float(int(q >= k1) + int(q >= k2) - 1);
                const float dx = fmaf(ox, G.wlo[0], fmaf(ox, G.wf[0], pj.x - pi.x));
                const float dy = fmaf(float(oy), G.wlo[1], fmaf(float(oy), G.wf[1], pj.y - pi.y));
                const float dz = fmaf(float(oz), G.wlo[2], fmaf(float(oz), G.wf[2], pj.z - pi.z));
                const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
                if (r2 < G.rc2f && q != k) {
                    const float ri2 = __frcp_rn(r2);
                    const float sr2 = G.sig2f * ri2;
                    const float sr6 = sr2 * sr2 * sr2;
                    const float fs = G.eps48f * sr6 * (sr6 - 0.5f) * ri2;
                    fx = fmaf(-fs, dx, fx);
                    fy = fmaf(-fs, dy, fy);
                    fz = fmaf(-fs, dz, fz);
                    ui += fmaf(G.eps4f * sr6, sr6 - 1.0f, -G.ucf);
                }
            }
        };
        constexpr int FAR = 0x7fffffff;
        if (cx > 0 && cx < G.nc[0] - 1) {
            run(row[cx - 1], row[cx + 2], row[cx], row[cx + 1]);
        } else {
            const int xm = (cx == 0) ? G.nc[0] - 1 : cx - 1, xp = (cx == G.nc[0] - 1) ? 0 : cx + 1;
            run(row[xm], row[xm + 1], FAR, FAR);
            run(row[cx], row[cx + 1], 0, FAR);
            run(row[xp], row[xp + 1], 0, 0);
        }
    }
    float v[4] = {fx, fy, fz, ui};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float p = __shfl_down_sync(0xffffffffu, v[q], 3), t = __shfl_down_sync(0xffffffffu, v[q], 6);
        v[q] = (v[q] + p) + t;
        const float p1 = __shfl_down_sync(0xffffffffu, v[q], 1), t1 = __shfl_down_sync(0xffffffffu, v[q], 2);
        v[q] = (v[q] + p1) + t1;
    }
    if (act && r == 0) {
        f[3 * i + 0] = v[0];
        f[3 * i + 1] = v[1];
        f[3 * i + 2] = v[2];
        if (u) u[i] = v[3];
    }
}

std::mutex g_na_mutex;
void* g_na_addr[256] = {nullptr};

int na_fail(int code, const std::string& msg) { return gbmd::set_last_error(code, msg.c_str()); }

}  // namespace

extern "C" {

int md_forces_static(const md_params* p, int64_t n, const double* x, double* f, double* u, void* stream)
{
    if (!p || !x || !f) return na_fail(MD_ERR_INVALID_ARG, "params, x and f are required");
    if (n <= 0 || n > NA_MAX_ATOMS)
        return na_fail(MD_ERR_INVALID_ARG, "md_forces_static handles 1.." + std::to_string(NA_MAX_ATOMS) + " atoms, got " +
                                               std::to_string(n));
    if (!(p->rc > 0.0) || !(p->eps > 0.0) || !(p->sigma > 0.0)) return na_fail(MD_ERR_INVALID_ARG, "bad potential");
    NaGeom G;
    G.ncells = 1;
    for (int a = 0; a < 3; ++a) {
        const double L = p->box[a];
        if (!(L > 0.0)) return na_fail(MD_ERR_INVALID_ARG, "box sides must be > 0");
        const double q = std::floor(L / p->rc);
        if (q < 3.0) return na_fail(MD_ERR_BOX_TOO_SMALL, "fewer than 3 cells of side >= rc");
        if (q > gbmd::MAX_NC) return na_fail(MD_ERR_INVALID_ARG, "more than 1023 cells along an axis");
        G.nc[a] = int(q);
        G.L[a] = L;
        G.w[a] = L / q;
        G.s[a] = q / L;
        G.wf[a] = float(G.w[a]);
        G.wlo[a] = float(G.w[a] - double(G.wf[a]));
        if (int64_t(G.ncells) * G.nc[a] > NA_MAX_CELLS)
            return na_fail(MD_ERR_INVALID_ARG, "md_forces_static handles at most " + std::to_string(NA_MAX_CELLS) +
                                                   " cells of side >= rc");
        G.ncells *= G.nc[a];
    }
    G.n = int(n);
    const double rc2 = p->rc * p->rc, sig2 = p->sigma * p->sigma;
    double uc = 0.0;
    if (p->shift_energy) {
        const double q2 = sig2 / rc2, q6 = q2 * q2 * q2;
        uc = 4.0 * p->eps * (q6 * q6 - q6);
    }
    G.rc2f = float(rc2);
    G.sig2f = float(sig2);
    G.eps4f = float(4.0 * p->eps);
    G.eps48f = float(48.0 * p->eps);
    G.ucf = float(uc);

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_fail(MD_ERR_CUDA, cudaGetErrorString(e));
    if (dev < 0 || dev >= 256) return na_fail(MD_ERR_CUDA, "device ordinal out of range");
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_na_mutex);
        if (!g_na_addr[dev]) {
            void* ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
            if (e != cudaSuccess || !ptr)
                return na_fail(MD_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
            g_na_addr[dev] = ptr;
        }
        base = g_na_addr[dev];
    }
    const NaView V = view_of(base);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    (void)cudaGetLastError();        // an earlier, unrelated launch error is not this call's failure
    const int blocks = int((n + NA_THREADS - 1) / NA_THREADS);
    if (n <= NA_CLUSTER_ATOMS) {
        k_na_cells<<<NA_CLUSTER, NA_CLUSTER_THREADS, 0, st>>>(V, G, x);
    } else {
        e = cudaMemsetAsync(V.count, 0, sizeof(int32_t) * size_t(G.ncells), st);
        if (e != cudaSuccess) return na_fail(MD_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
        k_na_bin<<<blocks, NA_THREADS, 0, st>>>(V, G, x);
        k_na_scan<<<1, 1024, 0, st>>>(V, G);
        k_na_scatter<<<blocks, NA_THREADS, 0, st>>>(V, G);
        k_na_order<<<blocks, NA_THREADS, 0, st>>>(V, G);
    }
    const int per_cta = NA_GROUP * (NA_THREADS / 32);
    k_na_forces<<<int((n + per_cta - 1) / per_cta), NA_THREADS, 0, st>>>(V, G, f, u);
    e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(MD_ERR_CUDA, cudaGetErrorString(e));
    return MD_OK;
}

}  // extern "C"
