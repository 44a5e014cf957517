// kernels_rebuild.cu -- cell binning, cell ordering, reordering and neighbour-matrix build.
//
// Sec. 2.3 of the paper lists the steps N1-N5; Sec. 2.4 item 4 the reorder vector s obtained
// there by a serial host pass over H and, as the GPU alternative it names, by a prefix sum of
// the cell occupancies k_c.  Here everything runs on the GPU:
//   k_bin          N1 + N2: cell of every atom from its FP64 position, layer l_i = atomic slot
//                  in the cell (the occupancy counter k_c); max k_c (N3) per replica.
//   k_scan_*       prefix sum of k_c -> cstart (the row offsets of H, Sec. 2.4 item 4).
//   k_scatter      N4: H flattened, in layer order.
//   k_order        the atomic layer order is indeterminate (Sec. 2.3 notes the resulting
//                  irreproducibility); ranking each atom among its cell's slots makes the order,
//                  and every result after it, deterministic.  It also writes the candidate array
//                  psort that the build reads.
//   k_reorder_copy Sec. 4.1 item 1: the atoms into cell order, from the scratch that k_order filled.
//   k_build_group  N5: W from the 27 neighbouring cells, units of 10 atoms per warp and a lane per
//                  atom and z plane; W stored row-major for coalescing (Sec. 4.1 item 6).
//   k_tile_windows the slot window of each tile's W entries per row of neighbour cells, read by
//                  the step kernel that stages neighbour positions (step kernel 3 only).
// Only replicas whose rebuild flag is set do work; kernels return at once when none is set, so
// the whole sequence can sit in every step of md_integrate.
#include <algorithm>

#include "gbmd_internal.cuh"

namespace gbmd {

// ------------------------------------------------------------------------------------------
// The largest occupancy (N3) is kept per thread over a CTA's contiguous run of tiles and folded in once
// per replica: one block reduction and one atomic, instead of an atomic per warp on the same address.
// All threads of the CTA call this.
// ------------------------------------------------------------------------------------------
__device__ void flush_max(int* dst, int mx)
{
    __shared__ int sh_max[TILE / 32];
    mx = warp_max_i(mx);
    if ((threadIdx.x & 31) == 0) sh_max[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        int m = 0;
        for (int w = 0; w < TILE / 32; ++w) m = max(m, sh_max[w]);
        if (m > 0) atomicMax(dst, m);
    }
    __syncthreads();
}

// ------------------------------------------------------------------------------------------
// The tiles of the replicas that rebuild in this step, listed contiguously so that the rebuild
// kernels share them evenly among their CTAs (in a batch only some replicas rebuild per step).
// Every CTA computes the replicas' positions in the list and fills those of its share of them, a
// warp per replica: one CTA filling all of them in turn took 44 us of a step of 512 replicas.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_rebuild_list(Arrays A, Scal S)
{
    if (!A.g->any_rebuild) return;
    __shared__ int sh[33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int carry = 0;
    for (int r0 = 0; r0 < S.nrep; r0 += blockDim.x) {
        const int r = r0 + threadIdx.x;
        const int v = (r < S.nrep && A.rs[r].rebuild) ? A.rep[r].ntiles : 0;
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
        const int base = carry + sh[wid] + incl - v;
        carry += sh[32];
        // this CTA's warps of replicas
        const int w0 = (r0 >> 5) + wid;               // the replicas 32 w0 .. 32 w0 + 31
        if (w0 % int(gridDim.x) == int(blockIdx.x)) {
            for (unsigned todo = __ballot_sync(0xffffffffu, v > 0); todo; todo &= todo - 1) {
                const int l = __ffs(todo) - 1;
                const int nt = __shfl_sync(0xffffffffu, v, l), b = __shfl_sync(0xffffffffu, base, l);
                const int t0 = A.rep[32 * w0 + l].tile0;
                for (int k = lane; k < nt; k += 32) A.rb_tiles[b + k] = t0 + k;
            }
        }
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) A.g->n_rb_tiles = carry;
}

// The it-th tile of the rebuild and its replica.  A single system's list is all its tiles: no need to
// wait for two loads, one after the other, before the replica's geometry.
__device__ __forceinline__ int rebuild_tile(const Arrays& A, const Scal& S, int it) { return S.nrep == 1 ? it : A.rb_tiles[it]; }
__device__ __forceinline__ int tile_replica(const Arrays& A, const Scal& S, int t) { return S.nrep == 1 ? 0 : A.tile_rep[t]; }

// ------------------------------------------------------------------------------------------
// N1 + N2
// ------------------------------------------------------------------------------------------
template <int MODE>
__global__ void __launch_bounds__(TILE) k_bin(Arrays A, Scal S, int cur, int from_set)
{
    if (!A.g->any_rebuild) return;
    const int nrb = A.g->n_rb_tiles;                  // tiles of the rebuilding replicas
    const int per = (nrb + gridDim.x - 1) / gridDim.x;
    const int t_begin = blockIdx.x * per, t_end = min(nrb, t_begin + per);
    int run_r = -1, run_occ = 0;
    for (int it = t_begin; it < t_end; ++it) {
        const int t = rebuild_tile(A, S, it);
        const int r = tile_replica(A, S, t);
        if (r != run_r) {
            if (run_r >= 0) flush_max(&A.rs[run_r].max_occ, run_occ);
            run_r = r;
            run_occ = 0;
        }
        const Rep& R = A.rep[r];
        if (t == R.tile0 && threadIdx.x == 0) {
            A.rs[r].sum_nbrs = 0;
            A.rs[r].max_nbrs = 0;
        }
        const int64_t slot = int64_t(t) * TILE + threadIdx.x;
        const int64_t j = slot - R.slot0;
        int occ = 0;
        int cell_bin = -1;            // this lane's cell, -1 for padding slots
        if (j < R.n && from_set) {
            // exact binning of a global position (the definition the oracle follows):
            // wrap into [0, L), c = floor(x n_c / L) clamped, local = x - c w, all in FP64
            double x[3] = {A.xl[0][slot], A.xl[1][slot], A.xl[2][slot]};
            int c[3];
            double loc[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                double xa = x[a];
                // inside [0, L) on the bit patterns (for x >= 0 they order as the values do): the FP64
                // pipe, which bounds this pass, is left the arithmetic
                if (static_cast<unsigned long long>(__double_as_longlong(xa)) >=
                    static_cast<unsigned long long>(__double_as_longlong(R.L[a]))) {
                    if (!isfinite(xa)) {              // reported; the atom goes to cell 0
                        atomicOr(&A.g->err, ERR_NONFINITE);
                        xa = 0.0;
                    }
                    if (xa < 0.0) xa = __dadd_rn(xa, R.L[a]);
                    if (xa >= R.L[a]) xa = __dsub_rn(xa, R.L[a]);
                    if (!(xa >= 0.0 && xa < R.L[a])) {    // more than one period away: whole periods
                        xa = __dsub_rn(xa, __dmul_rn(R.L[a], floor(xa / R.L[a])));
                        if (xa < 0.0) xa = __dadd_rn(xa, R.L[a]);
                        if (xa >= R.L[a]) xa = __dsub_rn(xa, R.L[a]);
                    }
                }
                // xa >= 0, so rounding towards zero is the floor (xa in a hair's breadth of 0 or L after
                // the wraps is clamped)
                int ca = __double2int_rz(__dmul_rn(xa, R.s[a]));
                ca = min(max(ca, 0), R.nc[a] - 1);
                c[a] = ca;
                loc[a] = __dsub_rn(xa, __dmul_rn(double(ca), R.w[a]));
            }
            const uint32_t packed = pack_cell(c[0], c[1], c[2]);
            if (MODE == MD_FP64) {
                A.pos64[cur][slot] = make_double4_32a(loc[0], loc[1], loc[2], cell_word_d(packed));
            } else {
                A.pos32[cur][slot] = make_float4(__double2float_rn(loc[0]), __double2float_rn(loc[1]),
                                                 __double2float_rn(loc[2]), cell_word_f(packed));
            }
            if (MODE != MD_FP32) {
                A.xl[0][slot] = loc[0]; A.xl[1][slot] = loc[1]; A.xl[2][slot] = loc[2];
            }
            const int cell = cell_index(R, c[0], c[1], c[2]);
            A.cell[slot] = cell;
            cell_bin = cell;
        } else if (j < R.n) {
            // during a run every atom is within skin/2 < w of its cell: it stays or moves to the
            // adjacent cell along each axis; its local coordinate shifts by -s w (s in -1, 0, 1)
            int c[3], sh[3];
            bool moved = false;
            if (MODE == MD_FP64) {
                const double4_32a p = A.pos64[cur][slot];
                unpack_cell(cell_bits(p.w), c[0], c[1], c[2]);
                const double l[3] = {p.x, p.y, p.z};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    sh[a] = (l[a] < 0.0) ? -1 : ((l[a] >= R.w[a]) ? 1 : 0);
                    moved |= sh[a] != 0;
                    if (!(l[a] >= -R.w[a] && l[a] < 2.0 * R.w[a])) atomicOr(&A.g->err, ERR_NONFINITE);
                }
                if (moved) {
                    double nl[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        nl[a] = sh[a] ? __dsub_rn(l[a], double(sh[a]) * R.w[a]) : l[a];
                        int ca = c[a] + sh[a];
                        ca += (ca < 0) ? R.nc[a] : 0;
                        ca -= (ca >= R.nc[a]) ? R.nc[a] : 0;
                        c[a] = ca;
                        A.xl[a][slot] = nl[a];
                    }
                    A.pos64[cur][slot] = make_double4_32a(nl[0], nl[1], nl[2], cell_word_d(pack_cell(c[0], c[1], c[2])));
                }
            } else {
                const float4 p = A.pos32[cur][slot];
                unpack_cell(__float_as_uint(p.w), c[0], c[1], c[2]);
                const float l[3] = {p.x, p.y, p.z};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    sh[a] = (l[a] < 0.0f) ? -1 : ((l[a] >= R.wf[a]) ? 1 : 0);
                    moved |= sh[a] != 0;
                    if (!(l[a] >= -R.wf[a] && l[a] < 2.0f * R.wf[a])) atomicOr(&A.g->err, ERR_NONFINITE);
                }
                if (moved) {
                    float nl[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        if (MODE == MD_MIXED) {
                            const double x = sh[a] ? __dsub_rn(A.xl[a][slot], double(sh[a]) * R.w[a]) : A.xl[a][slot];
                            if (sh[a]) A.xl[a][slot] = x;
                            nl[a] = __double2float_rn(x);
                        } else {
                            nl[a] = sh[a] ? __fsub_rn(l[a], float(sh[a]) * R.wf[a]) : l[a];
                        }
                        int ca = c[a] + sh[a];
                        ca += (ca < 0) ? R.nc[a] : 0;
                        ca -= (ca >= R.nc[a]) ? R.nc[a] : 0;
                        c[a] = ca;
                    }
                    A.pos32[cur][slot] = make_float4(nl[0], nl[1], nl[2], cell_word_f(pack_cell(c[0], c[1], c[2])));
                }
            }
            const int cell = cell_index(R, c[0], c[1], c[2]);
            if (moved) A.cell[slot] = cell;
            cell_bin = cell;
        }
        // N2 layer slots: lanes of a warp that share a cell (common, the atoms are cell-sorted)
        // take consecutive layers from one atomic on the cell's counter
        {
            const unsigned peers = __match_any_sync(0xffffffffu, cell_bin);
            const int lane = threadIdx.x & 31;
            const int leader = __ffs(peers) - 1;
            const int rank = __popc(peers & ((1u << lane) - 1u));
            int base = 0;
            if (cell_bin >= 0 && lane == leader) base = atomicAdd(&A.ccount[cell_bin], __popc(peers));
            base = __shfl_sync(0xffffffffu, base, leader);
            if (cell_bin >= 0) {
                A.layer[slot] = base + rank;
                occ = base + rank + 1;
            }
        }
        run_occ = max(run_occ, occ);
    }
    if (run_r >= 0) flush_max(&A.rs[run_r].max_occ, run_occ);
}

// ------------------------------------------------------------------------------------------
// prefix sum of the cell occupancies (three passes, no inter-block waiting)
// ------------------------------------------------------------------------------------------
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_PER_THREAD = SCAN_CHUNK / SCAN_THREADS;

__device__ __forceinline__ int block_exclusive_scan(int v, int* sh_warp, int& total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh_warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        int w = (lane < (blockDim.x >> 5)) ? sh_warp[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < (blockDim.x >> 5)) sh_warp[lane] = wi - w;
        if (lane == (blockDim.x >> 5) - 1) sh_warp[32] = wi;
    }
    __syncthreads();
    total = sh_warp[32];
    const int r = sh_warp[wid] + incl - v;
    __syncthreads();
    return r;
}

// The scan of the cells' occupancies into cstart (ncells + 1 entries), through per-chunk totals; up
// to SCAN_SOLO chunks in one launch whose CTAs each add up the counts before theirs (three launches
// of a few us otherwise).  The scatter clears the counters for the next binning.  Only the cells of rebuilding replicas have
// atoms counted, and only their starts are read: a chunk of cells without any is passed over (in a
// batch about a tenth of the replicas rebuilds in a step).
__device__ __forceinline__ bool chunk_live(const Arrays& A, const Scal& S, int64_t c0)
{
    if (S.nrep == 1) return true;
    const int r0 = A.cell_rep[c0], r1 = A.cell_rep[min(c0 + SCAN_CHUNK, int64_t(S.ncells)) - 1];
    bool live = false;
    for (int r = r0 + int(threadIdx.x); r <= r1; r += blockDim.x) live |= A.rs[r].rebuild != 0;
    return __syncthreads_or(live) != 0;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_chunks(Arrays A, Scal S)
{
    if (!A.g->any_rebuild) return;
    __shared__ int sh[33];
    const int64_t c0 = int64_t(blockIdx.x) * SCAN_CHUNK;
    int total = 0;
    if (chunk_live(A, S, c0)) {
        const int64_t base = c0 + threadIdx.x * SCAN_PER_THREAD;
        int s = 0;
#pragma unroll
        for (int k = 0; k < SCAN_PER_THREAD; ++k) {
            const int64_t c = base + k;
            if (c < S.ncells) s += A.ccount[c];
        }
        block_exclusive_scan(s, sh, total);
    }
    if (threadIdx.x == 0) A.chunk[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_scan_top(Arrays A, Scal S)
{
    if (!A.g->any_rebuild) return;
    __shared__ int sh[33];
    int carry = 0;
    for (int b0 = 0; b0 < S.nchunks; b0 += blockDim.x) {
        const int b = b0 + threadIdx.x;
        const int v = (b < S.nchunks) ? A.chunk[b] : 0;
        int total;
        const int ex = block_exclusive_scan(v, sh, total);
        if (b < S.nchunks) A.chunk[b] = carry + ex;
        carry += total;
    }
}

template <bool SOLO>
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_apply(Arrays A, Scal S)
{
    if (!A.g->any_rebuild) return;
    __shared__ int sh[33];
    const int64_t c0 = int64_t(blockIdx.x) * SCAN_CHUNK;
    if (!chunk_live(A, S, c0)) return;
    int before = 0;
    if (SOLO) {
        // cells of replicas that do not rebuild count zero; c0 is a multiple of 4
        const int4* __restrict__ cnt = reinterpret_cast<const int4*>(A.ccount);
        int s = 0;
        for (int q = threadIdx.x; q < int(c0 >> 2); q += SCAN_THREADS) {
            const int4 v = __ldg(cnt + q);
            s += (v.x + v.y) + (v.z + v.w);
        }
        block_exclusive_scan(s, sh, before);
    } else {
        before = A.chunk[blockIdx.x];
    }
    const int64_t base = c0 + threadIdx.x * SCAN_PER_THREAD;
    int v[SCAN_PER_THREAD];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        const int64_t c = base + k;
        v[k] = (c < S.ncells) ? A.ccount[c] : 0;
        s += v[k];
    }
    int total;
    int run = before + block_exclusive_scan(s, sh, total);
    const int64_t end = min(c0 + SCAN_CHUNK, int64_t(S.ncells));
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        const int64_t c = base + k;
        if (c < end) {
            A.cstart[c] = run;
            run += v[k];
            if (c == end - 1) A.cstart[end] = run;      // also the start of the next chunk, if that is passed over
        }
    }
}

constexpr int SCAN_SOLO = 32;
static bool solo_scan(const Scal& S) { return S.nchunks <= SCAN_SOLO; }

static void launch_scan(const Arrays& A, const Scal& S, cudaStream_t st)
{
    if (solo_scan(S)) {
        k_scan_apply<true><<<S.nchunks, SCAN_THREADS, 0, st>>>(A, S);
        return;
    }
    k_scan_chunks<<<S.nchunks, SCAN_THREADS, 0, st>>>(A, S);
    k_scan_top<<<1, 1024, 0, st>>>(A, S);
    k_scan_apply<false><<<S.nchunks, SCAN_THREADS, 0, st>>>(A, S);
}

// ------------------------------------------------------------------------------------------
// N4 and the deterministic order within cells
// ------------------------------------------------------------------------------------------
// What a rebuild keeps of cell c of a replica: its run of candidates, its counter cleared for the next
// binning, and (keep) its slot range for the list-free step kernel.
__device__ __forceinline__ void cell_done(const Arrays& A, const Rep& R, const int32_t* __restrict__ cs, int c, int k0, int P0,
                                          int keep)
{
    const int ncx = R.nc[0], prow = c / ncx, cx = c - prow * ncx;
    const int32_t* row = cs + R.cell0 + prow * ncx;
    const int rs = row[0];
    const int base = cand_place(R, prow, rs) - P0;
    A.crun[R.cell0 + c] = make_int2((base + ((row[max(cx - 1, 0)] - rs) & ~3)) >> 2,
                                    (base + ((row[min(cx + 1, ncx - 1) + 1] - rs + 3) & ~3)) >> 2);
    A.ccount[R.cell0 + c] = 0;
    if (keep) A.ckeep[R.cell0 + c] = make_int2(row[cx] - k0, row[cx + 1] - k0);
}

// A tile does its share of its replica's cells.  In a dilute gas that is far more cells than slots
// (one tile of 128 atoms in 10^6 cells: 2.63 ms a binning and build); replicas beyond CELLS_PER_TILE have theirs
// done in chunks by all CTAs instead (S.dilute; 61 us, 20000 atoms in 8 10^6 cells 281 -> 137).
constexpr int CELLS_PER_TILE = 256, CELL_CHUNK = 4 * TILE;

__host__ __device__ __forceinline__ bool dilute_rep(const Rep& R) { return R.ncells > int64_t(CELLS_PER_TILE) * R.ntiles; }

bool dilute_cells(const std::vector<Rep>& reps)
{
    for (const Rep& R : reps)
        if (dilute_rep(R)) return true;
    return false;
}

__global__ void __launch_bounds__(TILE) k_scatter(Arrays A, Scal S, int keep)
{
    if (!A.g->any_rebuild) return;
    const int nrb = A.g->n_rb_tiles;
    const int32_t* __restrict__ cs = A.cstart;
    for (int it = blockIdx.x; it < nrb; it += gridDim.x) {
        const int t = rebuild_tile(A, S, it);
        const int r = tile_replica(A, S, t);
        const Rep& R = A.rep[r];
        const int64_t slot = int64_t(t) * TILE + threadIdx.x;
        if (slot - R.slot0 < R.n) A.tmp_i[0][cs[A.cell[slot]] + A.layer[slot]] = int32_t(slot);
        if (S.dilute && dilute_rep(R)) continue;
        const int tt = t - R.tile0;
        const int c_end = int(int64_t(R.ncells) * (tt + 1) / R.ntiles);
        const int k0 = cs[R.cell0], P0 = cand_place(R, 0, k0);
        for (int c = int(int64_t(R.ncells) * tt / R.ntiles) + int(threadIdx.x); c < c_end; c += TILE)
            cell_done(A, R, cs, c, k0, P0, keep);
    }
    if (!S.dilute) return;
    for (int64_t c0 = int64_t(blockIdx.x) * CELL_CHUNK; c0 < S.ncells; c0 += int64_t(gridDim.x) * CELL_CHUNK) {
        const int64_t c1 = min(c0 + CELL_CHUNK, int64_t(S.ncells));
        const int r1 = (S.nrep == 1) ? 0 : A.cell_rep[c1 - 1];
        for (int r = (S.nrep == 1) ? 0 : A.cell_rep[c0]; r <= r1; ++r) {
            const Rep& R = A.rep[r];
            if (!A.rs[r].rebuild || !dilute_rep(R)) continue;
            const int k0 = cs[R.cell0], P0 = cand_place(R, 0, k0);
            const int end = int(min(c1 - R.cell0, int64_t(R.ncells)));
            for (int c = int(max(c0 - R.cell0, int64_t(0))) + int(threadIdx.x); c < end; c += TILE)
                cell_done(A, R, cs, c, k0, P0, keep);
        }
    }
}

// One thread per atom: its rank among the slots of its cell (the scatter left them in atomic
// order) is its place in the cell order, perm.  The thread also writes the atom's entry of the
// build's candidate array at that place: position in the replica's frame, the slot it will have
// after a reorder that is due, and the packed cell.  A thread per cell sorting its slots in
// place was a serial chain of dependent loads (cells of 18 atoms: 428 us for 16.4M atoms, 22 us
// for 4000); the rank takes one pass over the cell's slots, which the lanes of a cell share.
template <int MODE>
__global__ void __launch_bounds__(TILE) k_order(Arrays A, Scal S, int cur, int move)
{
    if (!A.g->any_rebuild) return;
    const int nrb = A.g->n_rb_tiles;
    const int32_t* __restrict__ unsorted = A.tmp_i[0];
    const int32_t* __restrict__ cs = A.cstart;
    for (int it = blockIdx.x; it < nrb; it += gridDim.x) {
        const int t = rebuild_tile(A, S, it);
        const int r = tile_replica(A, S, t);
        const Rep& R = A.rep[r];
        const int64_t slot = int64_t(t) * TILE + threadIdx.x;
        if (slot - R.slot0 >= R.n) continue;
        const int c = A.cell[slot];
        const int b = cs[c], e = cs[c + 1];
        int rank = 0;
        for (int k = b; k < e; ++k) rank += (unsorted[k] < int(slot)) ? 1 : 0;
        const int k = b + rank;
        A.perm[k] = int32_t(slot);
        float G[3];
        uint32_t pc;
        int cc[3];
        if constexpr (MODE == MD_FP64) {
            const double4_32a p = A.pos64[cur][slot];
            pc = cell_bits(p.w);
            unpack_cell(pc, cc[0], cc[1], cc[2]);
            G[0] = __double2float_rn(fma(double(cc[0]), R.w[0], p.x));
            G[1] = __double2float_rn(fma(double(cc[1]), R.w[1], p.y));
            G[2] = __double2float_rn(fma(double(cc[2]), R.w[2], p.z));
        } else {
            const float4 p = A.pos32[cur][slot];
            pc = __float_as_uint(p.w);
            unpack_cell(pc, cc[0], cc[1], cc[2]);
            G[0] = fmaf(float(cc[0]), R.wf[0], p.x);
            G[1] = fmaf(float(cc[1]), R.wf[1], p.y);
            G[2] = fmaf(float(cc[2]), R.wf[2], p.z);
        }
        const int prow = row_pos(R, cc[1], cc[2]);
        const int rs = cs[R.cell0 + prow * R.nc[0]], re = cs[R.cell0 + (prow + 1) * R.nc[0]];
        const int P = cand_place(R, prow, rs) + (k - rs);
        const bool reorder = A.rs[r].reorder != 0;
        const int64_t out_slot = reorder ? R.slot0 + (k - cs[R.cell0]) : slot;
        if (move && reorder) {                        // the atom's state to its new place in the scratch
            if (MODE == MD_FP64) A.tmp_p64[out_slot] = A.pos64[cur][slot];
            else A.tmp_p32[out_slot] = A.pos32[cur][slot];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (MODE == MD_FP32) {
                    A.tmp_v[a][out_slot] = double(A.v32[a][slot]);
                } else {
                    A.tmp_d[a][out_slot] = A.xl[a][slot];
                    A.tmp_v[a][out_slot] = A.v[a][slot];
                }
            }
            A.tmp_i[1][out_slot] = c;
            A.tmp_id[out_slot] = A.id[slot];
        }
        cand_store(A.psort, A.pent, P, G[0], G[1], G[2], (uint32_t(out_slot) << IDX_SHIFT) | uint32_t(cc[0] & 3));
        A.pcell[k] = pc;
        if (k == re - 1)                              // far-away entries up to the group of 4
            for (int q = P + 1; q & 3; ++q) cand_store(A.psort, A.pent, q, CAND_FAR, CAND_FAR, CAND_FAR, 0u);
    }
}

// ------------------------------------------------------------------------------------------
// reorder (Sec. 4.1 item 1): new slot slot0 + j takes the j-th atom in cell order, from the scratch
// that k_order or k_reorder_gather has filled
// ------------------------------------------------------------------------------------------
// Larger systems gather the scratch in a launch of its own: k_order's scattered writes take longer there
// (4M atoms: 253 us against 52 + 110), and the launch they save is nothing.  New positions to W built,
// WCA, written by k_order / gathered: 2048 atoms 77 / 83 us, 108k 109 / 110, 256k 151 / 158, 500k 237 /
// 237, 1M 416 / 397, 4M 1471 / 1344 (LJ 256k 285 / 285, 1M 888 / 866); moves_in_order draws the line at
// 2048 tiles (262k atoms), within the sizes where the two are level.
template <int MODE>
__global__ void __launch_bounds__(TILE) k_reorder_gather(Arrays A, Scal S, int cur)
{
    if (!A.g->any_reorder) return;
    const int nrb = A.g->n_rb_tiles;
    for (int it = blockIdx.x; it < nrb; it += gridDim.x) {
        const int t = rebuild_tile(A, S, it);
        const int r = tile_replica(A, S, t);
        if (!A.rs[r].reorder) continue;
        const Rep& R = A.rep[r];
        const int64_t slot = int64_t(t) * TILE + threadIdx.x;
        const int64_t j = slot - R.slot0;
        if (j >= R.n) continue;
        const int32_t src = A.perm[A.cstart[R.cell0] + j];
        if (MODE == MD_FP64) A.tmp_p64[slot] = A.pos64[cur][src];
        else A.tmp_p32[slot] = A.pos32[cur][src];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if (MODE == MD_FP32) {
                A.tmp_v[a][slot] = double(A.v32[a][src]);
            } else {
                A.tmp_d[a][slot] = A.xl[a][src];
                A.tmp_v[a][slot] = A.v[a][src];
            }
        }
        A.tmp_i[1][slot] = A.cell[src];
        A.tmp_id[slot] = A.id[src];
    }
}

template <int MODE>
__global__ void __launch_bounds__(TILE) k_reorder_copy(Arrays A, Scal S, int cur)
{
    if (!A.g->any_reorder) return;
    const int nrb = A.g->n_rb_tiles;
    for (int it = blockIdx.x; it < nrb; it += gridDim.x) {
        const int t = rebuild_tile(A, S, it);
        const int r = tile_replica(A, S, t);
        if (!A.rs[r].reorder) continue;
        const Rep& R = A.rep[r];
        const int64_t slot = int64_t(t) * TILE + threadIdx.x;
        const int64_t j = slot - R.slot0;
        if (j >= R.n) continue;
        if (MODE == MD_FP32) {
            A.pos32[cur][slot] = A.tmp_p32[slot];
            for (int a = 0; a < 3; ++a) A.v32[a][slot] = float(A.tmp_v[a][slot]);
        } else {
            if (MODE == MD_FP64) A.pos64[cur][slot] = A.tmp_p64[slot];
            else A.pos32[cur][slot] = A.tmp_p32[slot];
            for (int a = 0; a < 3; ++a) {
                A.xl[a][slot] = A.tmp_d[a][slot];
                A.v[a][slot] = A.tmp_v[a][slot];
            }
        }
        const int32_t id = A.tmp_id[slot];
        A.id[slot] = id;
        A.slot_of_id[id] = int32_t(slot);
        A.cell[slot] = A.tmp_i[1][slot];
        A.perm[A.cstart[R.cell0] + int(j)] = int32_t(slot);
    }
}

// ------------------------------------------------------------------------------------------
// N5: neighbour matrix.  Criterion (exact, shared with nothing): with lf the cell-local
// coordinates and o the periodic cell offset, d = (lf_j - lf_i) + o * wf (two roundings),
// r2 = fma(d_z, d_z, fma(d_y, d_y, d_x * d_x)), neighbour iff r2 < (r_c + skin)^2.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// The criterion itself, for the atoms of slots me and j whose cells lie o apart: negative when j
// is a neighbour.  ox is the unwrapped difference of the cells along x (sx the periodic shift of
// j's run of cells); cells more than one apart hold no neighbours.
template <int MODE>
__device__ __noinline__ float criterion(const void* pos, const Rep* Rp, double rl2d, float rl2f, int me, int j, int sx,
                                        int oy, int oz)
{
    const Rep& R = *Rp;
    int ci[3], cj[3];
    if constexpr (MODE == MD_FP64) {
        const double4_32a pi = static_cast<const double4_32a*>(pos)[me], pj = static_cast<const double4_32a*>(pos)[j];
        unpack_cell(cell_bits(pi.w), ci[0], ci[1], ci[2]);
        unpack_cell(cell_bits(pj.w), cj[0], cj[1], cj[2]);
        const int ox = cj[0] + sx - ci[0];
        if (ox < -1 || ox > 1) return 1.0f;
        const double dx = add_rn(sub_rn(pj.x, pi.x), double(ox) * R.w[0]);
        const double dy = add_rn(sub_rn(pj.y, pi.y), double(oy) * R.w[1]);
        const double dz = add_rn(sub_rn(pj.z, pi.z), double(oz) * R.w[2]);
        return fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx))) < rl2d ? -1.0f : 1.0f;
    } else {
        const float4 pi = static_cast<const float4*>(pos)[me], pj = static_cast<const float4*>(pos)[j];
        unpack_cell(__float_as_uint(pi.w), ci[0], ci[1], ci[2]);
        unpack_cell(__float_as_uint(pj.w), cj[0], cj[1], cj[2]);
        const int ox = cj[0] + sx - ci[0];
        if (ox < -1 || ox > 1) return 1.0f;
        const float dx = add_rn(sub_rn(pj.x, pi.x), float(ox) * R.wf[0]);
        const float dy = add_rn(sub_rn(pj.y, pi.y), float(oy) * R.wf[1]);
        const float dz = add_rn(sub_rn(pj.z, pi.z), float(oz) * R.wf[2]);
        return fma_rn(dz, dz, fma_rn(dy, dy, mul_rn(dx, dx))) < rl2f ? -1.0f : 1.0f;
    }
}

// ------------------------------------------------------------------------------------------
// N5, the build of W.  A warp takes a unit of BG_ATOMS atoms consecutive in cell order; lane
// (a, plane) scans, for atom a, the three rows of cells of one z plane of the 27 around it, so the
// three planes of an atom are scanned at the same time.
//
// A candidate is tested on its position in the replica's frame (cand_store), two per packed
// FP32x2 operation: d = |r|^2 - (r_c + skin)^2.  That differs from the criterion's expression by at
// most R.band; where |d| is below the band (a few pairs in 10^4) the criterion itself decides, so
// the sets are the criterion's exactly.  A run of candidates starts and ends at a multiple of 4:
// an atom of a cell more than one away is farther than r_c + skin, so it needs no bounds, and rows
// of cells end in far-away entries.  An accepted candidate is appended to the lane's own list in
// shared memory by predicated instructions, without a branch.  After the three rows the warp joins
// each atom's three lists (planes in order, so the entries of a column come in the order rows,
// cells, slots) and writes W row by row: consecutive lanes write consecutive slots.
//
// Bounds: the loads of candidates (12 bytes to each of 32 lanes, SM load pipe 63-72 % busy) and
// issue (44-60 %); what waits is their latency, so as many warps as fit matter: with 16-bit list
// entries 31 of them at the LJ cutoff (0.67 ms per binning and build of 864k atoms; 20 with 32-bit
// ones 0.77, 16 0.90), 32 at WCA.  Measured against one thread per atom walking its nine rows and
// branching at every append (per rebuild): LJ r_c + skin = 2.8: 16.4M atoms 27.7 -> 11.5 ms, 256k
// atoms 513 -> 200 us, 4000 atoms 388 -> 31 us; WCA: 100k atoms 110 -> 30 us, 4M atoms 0.76 ->
// 0.75 ms; FP64, 2048 atoms 71 -> 9 us (positions tested in FP32, the criterion in FP64).  One run
// shared by a unit's atoms of a row (fewer distinct addresses per load, more candidates) lost:
// 0.69 against 0.59 ms at 2M WCA atoms; so did loads one pass ahead (registers) and passes of 8.
// ------------------------------------------------------------------------------------------
constexpr int BG_ATOMS = 10;
constexpr int BG_UNITS = (TILE + BG_ATOMS - 1) / BG_ATOMS;       // units per rebuild tile
constexpr int BG_STEP = 4;                                       // candidates per pass of the scan
constexpr int BG_TABLE = 12 * 32 * 4;                            // bytes of a warp's table of run starts
constexpr uint32_t BG_ROW = 32 * 2;                              // bytes of one row of the lists

// append v to the list at shared address w where d < 0.  The appends tell the compiler of no memory, so
// that loads of candidates can pass them; the lists are read through a pointer it takes to be
// unrelated, behind lists_fence() (volatile, as the appends are, and so in order with them), and a
// second one lies between those reads and the next unit's appends.
__device__ __forceinline__ void list_append(uint32_t& w, float d, uint32_t v)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.f32 p, %1, 0f00000000;\n\t@p st.shared.u16 [%0], %2;\n\t"
                 "@p add.u32 %0, %0, 64;\n\t}"
                 : "+r"(w) : "f"(d), "h"(uint16_t(v)));
}
__device__ __forceinline__ void lists_fence()
{
    __syncwarp();
    asm volatile("" ::: "memory");
}
// the same where also e != self (NE) or e > self (unsigned)
template <bool GT>
__device__ __forceinline__ void list_append_if(uint32_t& w, float d, uint32_t v, uint32_t e, uint32_t self)
{
    if constexpr (GT)
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.gt.u32 q, %3, %4;\n\tsetp.lt.and.f32 p, %1, 0f00000000, q;\n\t"
                     "@p st.shared.u16 [%0], %2;\n\t@p add.u32 %0, %0, 64;\n\t}"
                     : "+r"(w) : "f"(d), "h"(uint16_t(v)), "r"(e), "r"(self));
    else
        asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %3, %4;\n\tsetp.lt.and.f32 p, %1, 0f00000000, q;\n\t"
                     "@p st.shared.u16 [%0], %2;\n\t@p add.u32 %0, %0, 64;\n\t}"
                     : "+r"(w) : "f"(d), "h"(uint16_t(v)), "r"(e), "r"(self));
}

// List entries, 16 bits: the candidate's number within its run, the row's o_y + 1 and the periodic
// shift of the run in x (1: from the left image, 2: from the right one).  The start of each run is
// kept in a table per lane, so that the place, the slot and the code of W follow when the lists are
// joined.  A unit with a run of more than BG_RUN candidates goes through build_column.
constexpr int BG_RUN = 4096, BG_OY = 12, BG_IMG = 14;

struct ScanLane {               // what a lane keeps while it scans
    float2 nx, ny, nz;          // minus the atom's coordinates, as seen from the row's cells
    float band;
    uint32_t self;              // its own W word (slot << IDX_SHIFT | c_x mod 4)
    uint32_t w, wlim, lost;     // list position and its limit; bytes of entries beyond it
    bool far;                   // a run was too long for the entries
};

// Candidate groups [g0, g1) of one run.  SELF: the run may hold the atom itself, whose list entry
// would be `mine`.
template <int MODE, bool HALF, bool SELF>
__device__ __forceinline__ void scan_run(const float4* __restrict__ ps, const uint32_t* __restrict__ pent, int g0, int g1,
                                         ScanLane& L, int* runs, float rl2f, double rl2d, uint32_t tag, uint32_t mine,
                                         const void* pos, const Rep* Rp, int sx, int oy, int oz)
{
    const float2 nrl2 = make_float2(-rl2f, -rl2f);
    runs[32 * (tag >> BG_OY)] = BG_STEP * g0;
    L.far |= g1 - g0 > BG_RUN / BG_STEP;
    for (int g = g0; g < g1; ++g) {
        const float4 x = __ldg(ps + 3 * g), y = __ldg(ps + 3 * g + 1), z = __ldg(ps + 3 * g + 2);
        const float2 dx0 = __fadd2_rn(make_float2(x.x, x.y), L.nx), dx1 = __fadd2_rn(make_float2(x.z, x.w), L.nx);
        const float2 dy0 = __fadd2_rn(make_float2(y.x, y.y), L.ny), dy1 = __fadd2_rn(make_float2(y.z, y.w), L.ny);
        const float2 dz0 = __fadd2_rn(make_float2(z.x, z.y), L.nz), dz1 = __fadd2_rn(make_float2(z.z, z.w), L.nz);
        const float2 q0 = __ffma2_rn(dz0, dz0, __ffma2_rn(dy0, dy0, __ffma2_rn(dx0, dx0, nrl2)));
        const float2 q1 = __ffma2_rn(dz1, dz1, __ffma2_rn(dy1, dy1, __ffma2_rn(dx1, dx1, nrl2)));
        float d[BG_STEP] = {q0.x, q0.y, q1.x, q1.y};
        if (fminf(fminf(fabsf(d[0]), fabsf(d[1])), fminf(fabsf(d[2]), fabsf(d[3]))) < L.band) {
#pragma unroll
            for (int u = 0; u < BG_STEP; ++u)
                if (fabsf(d[u]) < L.band)
                    d[u] = criterion<MODE>(pos, Rp, rl2d, rl2f, int(L.self >> IDX_SHIFT),
                                           int(pent[BG_STEP * g + u] >> IDX_SHIFT), sx, oy, oz);
        }
        const uint32_t v = uint32_t(BG_STEP * (g - g0)) | tag;
#pragma unroll
        for (int u = 0; u < BG_STEP; ++u) {
            if (HALF) list_append_if<true>(L.w, d[u], v | uint32_t(u), pent[BG_STEP * g + u], L.self | 63u);
            else if (SELF) list_append_if<false>(L.w, d[u], v | uint32_t(u), uint32_t(BG_STEP * g + u), mine);
            else list_append(L.w, d[u], v | uint32_t(u));
        }
        if (L.w > L.wlim) {                           // a full list counts on, writing past its end
            L.lost += L.w - L.wlim;
            L.w = L.wlim;
        }
    }
}

// The column of one atom entry by entry, for a unit in which a list overflowed: the criterion on
// every atom of the 27 cells, in the same order.
template <int MODE>
__device__ __noinline__ int build_column(const void* pos, const Rep* Rp, const int32_t* cs, const int32_t* perm,
                                         uint32_t* W, int64_t nslots, int cap, double rl2d, float rl2f, int half, int me,
                                         uint32_t pc)
{
    const Rep& R = *Rp;
    int c[3];
    unpack_cell(pc, c[0], c[1], c[2]);
    int m = 0;
    for (int oz = -1; oz <= 1; ++oz)
        for (int oy = -1; oy <= 1; ++oy)
            for (int ox = -1; ox <= 1; ++ox) {
                int n[3] = {c[0] + ox, c[1] + oy, c[2] + oz};
                const int sx = (n[0] < 0) ? -R.nc[0] : ((n[0] >= R.nc[0]) ? R.nc[0] : 0);
                for (int q = 0; q < 3; ++q) { n[q] += (n[q] < 0) ? R.nc[q] : 0; n[q] -= (n[q] >= R.nc[q]) ? R.nc[q] : 0; }
                const int g = cell_index(R, n[0], n[1], n[2]);
                for (int k = cs[g]; k < cs[g + 1]; ++k) {
                    const int j = perm[k];
                    if (half ? j <= me : j == me) continue;
                    if (criterion<MODE>(pos, Rp, rl2d, rl2f, me, j, sx, oy, oz) >= 0.0f) continue;
                    if (m < cap)
                        W[int64_t(m) * nslots + me] =
                            (uint32_t(j) << IDX_SHIFT) | uint32_t(ox + 1) | (uint32_t(oy + 1) << 2) | (uint32_t(oz + 1) << 4);
                    ++m;
                }
            }
    return m;
}

// Bookkeeping after a rebuild, by one CTA.
__device__ void rebuild_finish(const Arrays& A, const Scal& S, int in_graph)
{
    for (int r = threadIdx.x; r < S.nrep; r += blockDim.x) {
        RepState& st = A.rs[r];
        if (!st.rebuild) continue;
        if (st.reorder) {
            st.last_reorder = st.step;
            st.reorders += 1;
        }
        st.reorder = 0;
        st.rebuild = 0;
        st.D = 0.0;
        st.rebuilds += 1;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        A.g->any_rebuild = 0;
        A.g->any_reorder = 0;
        if (in_graph) A.g->graph_rebuilds += 1;
    }
}

// finish: 1 when no kernel of the rebuild follows, so that the last CTA closes it (in_graph as
// for k_rebuild_finish)
template <int MODE, bool HALF, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 1) k_build_group(Arrays A, Scal S, int cur, int rows, int finish, int in_graph)
{
    extern __shared__ uint32_t s_list[];              // [warps][rows + BG_STEP][32]
    if (!A.g->any_rebuild) return;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    // per warp: the table of run starts [12][32], then the lists [rows + BG_STEP][32]
    unsigned char* const mem = reinterpret_cast<unsigned char*>(s_list) + wl * (BG_TABLE + (rows + BG_STEP) * int(BG_ROW));
    int* const my_runs = reinterpret_cast<int*>(mem);
    const uint16_t* const my_lists = reinterpret_cast<const uint16_t*>(mem + BG_TABLE);
    const int a = lane % BG_ATOMS, pl = lane / BG_ATOMS;          // atom of the unit, z plane (3: idle lane)
    const int32_t* __restrict__ cs = A.cstart;
    const void* const pos = (MODE == MD_FP64) ? static_cast<const void*>(A.pos64[cur]) : static_cast<const void*>(A.pos32[cur]);
    const int nunits = A.g->n_rb_tiles * BG_UNITS;
    // every CTA takes a contiguous run of units, its warps side by side: neighbouring units read the
    // same rows of candidates
    const int wpc = blockDim.x >> 5;
    const int per = (nunits + int(gridDim.x) - 1) / int(gridDim.x), u_begin = int(blockIdx.x) * per;
    const int u_end = min(nunits, u_begin + per);
    ScanLane L;
    L.wlim = smem_u32(my_lists) + 2 * lane + uint32_t(rows) * BG_ROW;
    int run_r = -1, run_max = 0;
    long long run_sum = 0;
    auto flush_warp = [&]() {
        const long long ws = warp_sum_ll(run_sum);
        const int wm = warp_max_i(run_max);
        if (lane == 0) {
            if (ws) atomicAdd(reinterpret_cast<unsigned long long*>(&A.rs[run_r].sum_nbrs), static_cast<unsigned long long>(ws));
            if (wm > 0) atomicMax(&A.rs[run_r].max_nbrs, wm);
        }
    };
    for (int uid = u_begin + wl; uid < u_end; uid += wpc) {
        const int it = uid / BG_UNITS, u = uid - it * BG_UNITS;
        const int t = rebuild_tile(A, S, it);
        const int r = tile_replica(A, S, t);
        const Rep& R = A.rep[r];
        const int j0 = (t - R.tile0) * TILE + u * BG_ATOMS;
        const int na = min(min(BG_ATOMS, TILE - u * BG_ATOMS), R.n - j0);
        if (na <= 0) continue;
        if (r != run_r) {
            if (run_r >= 0) flush_warp();
            run_r = r;
            run_sum = 0;
            run_max = 0;
        }
        const bool act = pl < 3 && a < na;
        const int k0 = cs[R.cell0];
        const int k = k0 + j0 + min(a, na - 1);
        const uint32_t pc = A.pcell[k];
        int cx, cy, cz;
        unpack_cell(pc, cx, cy, cz);
        const int ncx = R.nc[0], ncy = R.nc[1], ncz = R.nc[2];
        const int P0 = cand_place(R, 0, k0);          // the replica's part of the candidate array
        const float4* __restrict__ ps = A.psort + int64_t(3) * (P0 >> 2);
        const uint32_t* __restrict__ pent = A.pent + P0;
        float X, Y, Z;
        uint32_t mine;                                // the atom's own place
        {
            const int prow = row_pos(R, cy, cz);
            const int rs = cs[R.cell0 + prow * ncx];
            mine = uint32_t(cand_place(R, prow, rs) - P0 + (k - rs));
            const float* f = reinterpret_cast<const float*>(ps) + 12 * (mine >> 2) + (mine & 3u);
            X = f[0];
            Y = f[4];
            Z = f[8];
            L.self = pent[mine];
        }
        const int oz = pl - 1;
        int nz = cz + oz;
        float wz = 0.0f;                              // shift of the atom into the frame of wrapped cells
        if (nz < 0) { nz += ncz; wz = float(ncz) * R.wf[2]; }
        else if (nz >= ncz) { nz -= ncz; wz = -float(ncz) * R.wf[2]; }
        L.nz = make_float2(-(Z + wz), -(Z + wz));
        L.w = L.wlim - uint32_t(rows) * BG_ROW;
        L.lost = 0;
        L.far = false;
        const bool lo = act && cx == 0, hi = act && cx == ncx - 1;
        const bool any_lo = __any_sync(0xffffffffu, lo), any_hi = __any_sync(0xffffffffu, hi);
        const float band = R.band;
#pragma unroll 1
        for (int oy = -1; oy <= 1; ++oy) {
            int ny = cy + oy;
            float wy = 0.0f;
            if (ny < 0) { ny += ncy; wy = float(ncy) * R.wf[1]; }
            else if (ny >= ncy) { ny -= ncy; wy = -float(ncy) * R.wf[1]; }
            L.ny = make_float2(-(Y + wy), -(Y + wy));
            const uint32_t tag = uint32_t(oy + 1) << BG_OY;
            const int prow = row_pos(R, ny, nz < ncz ? nz : 0);
            const int row = R.cell0 + prow * ncx;
            if (any_lo) {                             // the row's last cell, seen across the boundary
                const float xs = X + float(ncx) * R.wf[0];
                L.nx = make_float2(-xs, -xs);
                L.band = 4.0f * band;
                const int rs = cs[row], base = cand_place(R, prow, rs) - P0;
                const int g0 = (base + ((cs[row + ncx - 1] - rs) & ~3)) >> 2;
                const int g1 = lo ? (base + ((cs[row + ncx] - rs + 3) & ~3)) >> 2 : g0;
                scan_run<MODE, HALF, false>(ps, pent, g0, g1, L, my_runs + lane, S.rl2f, S.rl2d, tag | (1u << BG_IMG), 0u, pos, &R, -ncx, oy, oz);
            }
            {
                L.nx = make_float2(-X, -X);
                L.band = (wy != 0.0f || wz != 0.0f) ? 4.0f * band : band;
                const int2 run = A.crun[row + cx];
                const int g1 = act ? run.y : run.x;
                if (oy == 0)
                    scan_run<MODE, HALF, true>(ps, pent, run.x, g1, L, my_runs + lane, S.rl2f, S.rl2d, tag, mine, pos, &R, 0, oy, oz);
                else
                    scan_run<MODE, HALF, false>(ps, pent, run.x, g1, L, my_runs + lane, S.rl2f, S.rl2d, tag, 0u, pos, &R, 0, oy, oz);
            }
            if (any_hi) {                             // the row's first cell, seen across the boundary
                const float xs = X - float(ncx) * R.wf[0];
                L.nx = make_float2(-xs, -xs);
                L.band = 4.0f * band;
                const int rs = cs[row], g0 = (cand_place(R, prow, rs) - P0) >> 2;
                const int g1 = hi ? g0 + ((cs[row + 1] - rs + 3) >> 2) : g0;
                scan_run<MODE, HALF, false>(ps, pent, g0, g1, L, my_runs + lane, S.rl2f, S.rl2d, tag | (2u << BG_IMG), 0u, pos, &R, ncx, oy, oz);
            }
        }
        // join the planes: entry m of atom a comes from plane 0, 1 or 2
        const int cnt = int((L.w - (L.wlim - uint32_t(rows) * BG_ROW) + L.lost) / BG_ROW);
        lists_fence();
        const int c0 = __shfl_sync(0xffffffffu, cnt, a), c1 = __shfl_sync(0xffffffffu, cnt, a + BG_ATOMS);
        const int c2 = __shfl_sync(0xffffffffu, cnt, a + 2 * BG_ATOMS);
        int m = c0 + c1 + c2;
        const int slot = int(L.self >> IDX_SHIFT);
        // o_x + 1 = cell of j, shifted by its run's image, - cell of i + 1 (mod 4)
        const uint32_t cadd = uint32_t(1 - cx);
        if (__any_sync(0xffffffffu, act && (L.far || (rows < S.cap && L.lost != 0)))) {
            if (act && pl == 0)
                m = build_column<MODE>(pos, &R, cs, A.perm, A.W, S.nslots, S.cap, S.rl2d, S.rl2f, HALF ? 1 : 0, slot, pc);
        } else if (act) {
            const int mc = min(m, S.cap);
            uint32_t* wp = A.W + int64_t(pl) * S.nslots + slot;
            for (int q0 = pl; q0 < mc; q0 += 12, wp += 12 * S.nslots) {
                uint32_t e[4], img[4], code[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int q = q0 + 3 * u;
                    const int oz1 = (q < c0) ? 0 : ((q < c0 + c1) ? 1 : 2), from = a + BG_ATOMS * oz1;
                    const int m0 = (oz1 == 0) ? 0 : ((oz1 == 1) ? c0 : c0 + c1);
                    const uint32_t v = q < mc ? my_lists[(q - m0) * 32 + from] : 0u;
                    e[u] = __ldg(pent + (q < mc ? my_runs[32 * (v >> BG_OY) + from] + int(v & (BG_RUN - 1)) : 0));
                    img[u] = v >> BG_IMG;
                    code[u] = (((v >> BG_OY) & 3u) << 2) | (uint32_t(oz1) << 4);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const uint32_t ox = (e[u] + cadd + (img[u] == 2u ? uint32_t(ncx) : 0u) - (img[u] == 1u ? uint32_t(ncx) : 0u)) & 3u;
                    if (q0 + 3 * u < mc) wp[int64_t(3 * u) * S.nslots] = (e[u] & ~63u) | ox | code[u];
                }
            }
        }
        lists_fence();
        if (act && pl == 0) {
            A.nbr_count[slot] = m;
            if (S.rule == MD_REBUILD_DISP) {
                if constexpr (MODE == MD_FP64) {
                    const double4_32a p = A.pos64[cur][slot];
                    A.xref[slot] = make_float4(float(p.x), float(p.y), float(p.z), 0.0f);
                } else {
                    const float4 p = A.pos32[cur][slot];
                    A.xref[slot] = make_float4(p.x, p.y, p.z, 0.0f);
                }
            }
            if (m > S.cap) {
                atomicOr(&A.g->err, ERR_NBR_OVERFLOW);
                atomicMax(&A.g->max_nbr_seen, m);
            }
            run_sum += m;
            run_max = max(run_max, m);
        }
    }
    if (run_r >= 0) flush_warp();
    if (finish) {
        // every CTA has read the rebuild flags by the time it counts itself in
        __shared__ int last;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(&A.g->build_done, 1) == int(gridDim.x) - 1;
        }
        __syncthreads();
        if (!last) return;
        if (threadIdx.x == 0) A.g->build_done = 0;
        __threadfence();
        rebuild_finish(A, S, in_graph);
    }
}

// ------------------------------------------------------------------------------------------
// Slot windows of each rebuilt tile's neighbours, for the step kernel that stages neighbour
// positions in shared memory: for every (o_y, o_z) row code, the smallest and largest slot among
// the tile's W entries of that code whose neighbour cell is reached without a periodic wrap
// (wrapped entries are gathered from global memory).  With atoms in cell order (reorder at every
// rebuild) each window spans the tile's cells plus one halo cell at either end, in one row of
// cells; otherwise windows can be wide, and the step kernel then stages what fits its budget.
// One CTA per tile; empty rows get lo > hi.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(TILE) k_tile_windows(Arrays A, Scal S, int cur, int enabled)
{
    __shared__ int sh_lo[9], sh_hi[9];
    if (!enabled || !A.g->any_rebuild || !A.tile_win) return;
    const int nrb = A.g->n_rb_tiles;
    for (int it = blockIdx.x; it < nrb; it += gridDim.x) {
        const int t = rebuild_tile(A, S, it);
        const Rep& R = A.rep[tile_replica(A, S, t)];
        if (threadIdx.x < 9) {
            sh_lo[threadIdx.x] = INT32_MAX;
            sh_hi[threadIdx.x] = -1;
        }
        __syncthreads();
        const int64_t slot = int64_t(t) * TILE + threadIdx.x;
        if (slot - R.slot0 < R.n) {
            int cx, cy, cz;
            unpack_cell(__float_as_uint(A.pos32[cur][slot].w), cx, cy, cz);
            // codes whose neighbour cell lies across the periodic boundary for this atom
            const bool wxl = cx == 0, wxh = cx == R.nc[0] - 1, wyl = cy == 0, wyh = cy == R.nc[1] - 1;
            const bool wzl = cz == 0, wzh = cz == R.nc[2] - 1;
            int lo[9], hi[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                lo[q] = INT32_MAX;
                hi[q] = -1;
            }
            const int mm = min(A.nbr_count[slot], S.cap);
            constexpr int B = 4;                 // rows of W loaded together
            for (int m0 = 0; m0 < mm; m0 += B) {
              uint32_t eb[B];
#pragma unroll
              for (int u = 0; u < B; ++u) eb[u] = (m0 + u < mm) ? __ldcs(A.W + int64_t(m0 + u) * S.nslots + slot) : 0u;
#pragma unroll
              for (int u = 0; u < B; ++u) {
                if (m0 + u >= mm) break;
                const uint32_t e = eb[u];
                const uint32_t ox = e & 3u, oy = (e >> 2) & 3u, oz = (e >> 4) & 3u;
                const bool wrap = (ox == 0 && wxl) || (ox == 2 && wxh) || (oy == 0 && wyl) || (oy == 2 && wyh) ||
                                  (oz == 0 && wzl) || (oz == 2 && wzh);
                if (wrap) continue;
                const int j = int(e >> IDX_SHIFT);
                const int q = int(oy + 3 * oz);
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    if (k == q) {
                        lo[k] = min(lo[k], j);
                        hi[k] = max(hi[k], j);
                    }
                }
              }
            }
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                if (hi[k] >= 0) {
                    atomicMin(&sh_lo[k], lo[k]);
                    atomicMax(&sh_hi[k], hi[k]);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x < 9) A.tile_win[int64_t(t) * 9 + threadIdx.x] = make_int2(sh_lo[threadIdx.x], sh_hi[threadIdx.x]);
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------------------
// bookkeeping after a rebuild
// ------------------------------------------------------------------------------------------
// (k_build_group's last CTA; a launch of its own when there is no build)
__global__ void k_rebuild_finish(Arrays A, Scal S, int in_graph)
{
    if (!A.g->any_rebuild) return;
    rebuild_finish(A, S, in_graph);
}

// Mark every replica for a rebuild (creation, md_set_state, md_bin_cells).
__global__ void k_force_rebuild(Arrays A, Scal S, int reorder)
{
    for (int r = threadIdx.x; r < S.nrep; r += blockDim.x) {
        A.rs[r].rebuild = 1;
        A.rs[r].reorder = reorder;
        A.rs[r].max_occ = 0;
    }
    if (threadIdx.x == 0) {
        A.g->any_rebuild = 1;
        A.g->any_reorder = reorder;
    }
}

// ------------------------------------------------------------------------------------------
// launch wrappers
// ------------------------------------------------------------------------------------------
static int tile_grid(const Scal& S, const Launch& L)
{
    return std::max(1, std::min(L.grid, S.ntiles));
}

// Grid of a rebuild kernel over tiles or other items that holds nothing across them (binning,
// scatter, order, reorder): every CTA the device can keep resident.  They wait on memory and
// atomics, so each resident warp adds requests in flight.  The occupancy of each kernel is looked
// up once.
template <auto Kernel>
static int resident_grid(const Scal& S, const Launch& L, int items = 0)
{
    static const int per_sm = [] {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, Kernel, TILE, 0) != cudaSuccess) b = 0;
        return b;
    }();
    const int g = (per_sm > 0) ? L.nsm * per_sm : L.grid;
    return std::max(1, std::min(g, items > 0 ? items : S.ntiles));
}

// looks the occupancies up outside any stream capture
void prime_rebuild_grids(const Scal& S, const Launch& L)
{
    (void)resident_grid<k_bin<MD_FP64>>(S, L);
    (void)resident_grid<k_bin<MD_MIXED>>(S, L);
    (void)resident_grid<k_bin<MD_FP32>>(S, L);
    (void)resident_grid<k_scatter>(S, L);
    (void)resident_grid<k_order<MD_FP64>>(S, L);
    (void)resident_grid<k_order<MD_MIXED>>(S, L);
    (void)resident_grid<k_order<MD_FP32>>(S, L);
    (void)resident_grid<k_reorder_copy<MD_FP64>>(S, L);
    (void)resident_grid<k_reorder_gather<MD_FP64>>(S, L);
    (void)resident_grid<k_reorder_copy<MD_MIXED>>(S, L);
    (void)resident_grid<k_reorder_gather<MD_MIXED>>(S, L);
    (void)resident_grid<k_reorder_copy<MD_FP32>>(S, L);
    (void)resident_grid<k_reorder_gather<MD_FP32>>(S, L);
}

cudaError_t launch_force_rebuild(const Arrays& A, const Scal& S, const Launch& L, int reorder)
{
    k_force_rebuild<<<1, 256, 0, L.stream>>>(A, S, reorder);
    return cudaGetLastError();
}

static bool moves_in_order(const Scal& S) { return S.ntiles <= 2048; }

cudaError_t launch_bin_order(const Arrays& A, const Scal& S, const Launch& L, int cur, bool from_set)
{
    // a single system rebuilds all its tiles, always (rebuild_tile; n_rb_tiles is set at creation)
    if (S.nrep > 1) k_rebuild_list<<<std::min((S.nrep + 31) / 32, L.nsm), 1024, 0, L.stream>>>(A, S);
    const int fs = from_set ? 1 : 0, move = moves_in_order(S) ? 1 : 0;
    if (S.mode == MD_FP64) k_bin<MD_FP64><<<resident_grid<k_bin<MD_FP64>>(S, L), TILE, 0, L.stream>>>(A, S, cur, fs);
    else if (S.mode == MD_MIXED) k_bin<MD_MIXED><<<resident_grid<k_bin<MD_MIXED>>(S, L), TILE, 0, L.stream>>>(A, S, cur, fs);
    else k_bin<MD_FP32><<<resident_grid<k_bin<MD_FP32>>(S, L), TILE, 0, L.stream>>>(A, S, cur, fs);
    launch_scan(A, S, L.stream);
    const int items = S.dilute ? std::max(S.ntiles, int((int64_t(S.ncells) + CELL_CHUNK - 1) / CELL_CHUNK)) : S.ntiles;
    k_scatter<<<resident_grid<k_scatter>(S, L, items), TILE, 0, L.stream>>>(A, S, L.step_kernel == 4 ? 1 : 0);
    if (S.mode == MD_FP64) k_order<MD_FP64><<<resident_grid<k_order<MD_FP64>>(S, L), TILE, 0, L.stream>>>(A, S, cur, move);
    else if (S.mode == MD_MIXED) k_order<MD_MIXED><<<resident_grid<k_order<MD_MIXED>>(S, L), TILE, 0, L.stream>>>(A, S, cur, move);
    else k_order<MD_FP32><<<resident_grid<k_order<MD_FP32>>(S, L), TILE, 0, L.stream>>>(A, S, cur, move);
    return cudaGetLastError();
}

cudaError_t launch_reorder(const Arrays& A, const Scal& S, const Launch& L, int cur)
{
#define GBMD_GATHER(M) k_reorder_gather<M><<<resident_grid<k_reorder_gather<M>>(S, L), TILE, 0, L.stream>>>(A, S, cur)
    if (moves_in_order(S)) {
    } else if (S.mode == MD_FP64) GBMD_GATHER(MD_FP64);
    else if (S.mode == MD_MIXED) GBMD_GATHER(MD_MIXED);
    else GBMD_GATHER(MD_FP32);
#undef GBMD_GATHER
#define GBMD_REORDER(M) k_reorder_copy<M><<<resident_grid<k_reorder_copy<M>>(S, L), TILE, 0, L.stream>>>(A, S, cur)
    if (S.mode == MD_FP64) GBMD_REORDER(MD_FP64);
    else if (S.mode == MD_MIXED) GBMD_REORDER(MD_MIXED);
    else GBMD_REORDER(MD_FP32);
#undef GBMD_REORDER
    return cudaGetLastError();
}

cudaError_t launch_bin_only(const Arrays& A, const Scal& S, const Launch& L, int cur, bool from_set)
{
    cudaError_t e = launch_bin_order(A, S, L, cur, from_set);
    if (e != cudaSuccess) return e;
    return launch_reorder(A, S, L, cur);
}

// the list-free step kernel reads no neighbour matrix; it is built only where the exact
// displacement rule needs the positions at the rebuild (written by the build)
static bool skip_w(const Scal& S, const Launch& L) { return L.step_kernel == 4 && S.rule != MD_REBUILD_DISP; }

int reorder_kernels(const Scal& S) { return moves_in_order(S) ? 1 : 2; }

int bin_kernels(const Scal& S, const Launch&) { return (S.nrep > 1 ? 1 : 0) + (solo_scan(S) ? 4 : 6); }

int build_kernels(const Scal& S, const Launch& L)
{
    return skip_w(S, L) ? (L.step_kernel == 3 ? 2 : 1) : (L.step_kernel == 3 ? 3 : 1);
}

// The lists of k_build_group hold one z plane's neighbours of an atom.  A slab of thickness w >= r_l
// around it holds up to 69 % of them; a third as many again and 12 leave room for fluctuations, at
// the largest mean density or, as far as 60 % of the capacity allows, in the densest liquid
// (mean_nbrs, dense_nbrs), so that a droplet's lists fit.  A capacity beyond that must not cost warps:
// 256k WCA atoms with room for 1000 neighbours each had 601 rows and 5 warps per SM, 260 us a binning
// and build against 106 with 29.  A longer list sends its unit through build_column.  One CTA per SM
// with as many warps as their lists allow, up to 32; with room for fewer than 24 the kernel compiled
// for 20, which has more registers.
// The opt-in limit is raised at each call: it belongs to the kernel in the context that is current, so
// one raised for a system on another device says nothing about this one.
template <int MODE, bool HALF, int WARPS>
static cudaError_t group_limit(int smem_per_cta)
{
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, k_build_group<MODE, HALF, WARPS>);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_build_group<MODE, HALF, WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                smem_per_cta - int(fa.sharedSizeBytes));
}

// F(MODE, HALF, WARPS) for the system's precision, list and list length
#define GBMD_BUILD_WARPS(M, H, F) { if (L.bg_warps == 32) F(M, H, 32); else F(M, H, 20); }
#define GBMD_BUILD_DISPATCH(F)                                                                          \
    if (S.mode == MD_FP64) GBMD_BUILD_WARPS(MD_FP64, false, F)                                           \
    else if (S.mode == MD_MIXED) { if (S.half_list) GBMD_BUILD_WARPS(MD_MIXED, true, F) else GBMD_BUILD_WARPS(MD_MIXED, false, F) } \
    else { if (S.half_list) GBMD_BUILD_WARPS(MD_FP32, true, F) else GBMD_BUILD_WARPS(MD_FP32, false, F) }

cudaError_t build_group_shape(const Scal& S, Launch& L, double mean_nbrs, double dense_nbrs, int smem_per_cta)
{
    const int room = smem_per_cta - 2048;
    auto for_mean = [](double nbrs) { return 0.69 * 1.35 * nbrs + 12.0; };
    const double want = std::max(for_mean(mean_nbrs), std::min(0.6 * S.cap, for_mean(dense_nbrs)));
    int rows = std::min(S.cap, int(std::min(want, 1.0e6)) + 1);
    rows = std::min(rows, (room - BG_TABLE) / int(BG_ROW) - BG_STEP);
    const int fit = room / (BG_TABLE + (rows + BG_STEP) * int(BG_ROW));
    L.bg_warps = fit >= 24 ? 32 : 20;
    L.bg_block = 32 * std::min(L.bg_warps, fit);
    L.bg_rows = rows;
    L.bg_smem = (BG_TABLE + (rows + BG_STEP) * int(BG_ROW)) * (L.bg_block / 32);
    cudaError_t e = cudaSuccess;
#define GBMD_LIMIT(M, H, B) e = group_limit<M, H, B>(smem_per_cta)
    GBMD_BUILD_DISPATCH(GBMD_LIMIT)
#undef GBMD_LIMIT
    return e;
}

cudaError_t launch_build_only(const Arrays& A, const Scal& S, const Launch& L, int cur)
{
    const int finish = (!skip_w(S, L) && L.step_kernel != 3) ? 1 : 0;
    if (!skip_w(S, L)) {
        // no more warps per CTA than units per SM (a CTA of 32 warps and 200 KB starts later)
        const int64_t units = int64_t(S.ntiles) * BG_UNITS;
        const int g = int(std::max<int64_t>(1, std::min<int64_t>(L.nsm, units)));
        const int warps = int(std::min<int64_t>(L.bg_block / 32, (units + g - 1) / g));
        const int block = 32 * warps, smem = L.bg_smem / (L.bg_block / 32) * warps;
#define GBMD_BUILD(M, H, B) k_build_group<M, H, B><<<g, block, smem, L.stream>>>(A, S, cur, L.bg_rows, finish, L.in_graph)
        GBMD_BUILD_DISPATCH(GBMD_BUILD)
#undef GBMD_BUILD
    }
    if (L.step_kernel == 3) k_tile_windows<<<tile_grid(S, L), TILE, 0, L.stream>>>(A, S, cur, 1);
    if (!finish) k_rebuild_finish<<<1, 256, 0, L.stream>>>(A, S, L.in_graph);
    return cudaGetLastError();
}

cudaError_t launch_rebuild(const Arrays& A, const Scal& S, const Launch& L, int cur, bool from_set)
{
    cudaError_t e = launch_bin_only(A, S, L, cur, from_set);
    if (e != cudaSuccess) return e;
    return launch_build_only(A, S, L, cur);
}

}  // namespace gbmd
