// Periodic counting sort of one species (histogram, exclusive scan, scatter),
// dropping dead slots.  The FP64 path sorts by linear cell index; the mixed
// path by tile (blocks of tile[0] x tile[1] x tile[2] cells, tile-major, the
// cells of a tile row-major inside it), so that each tile's particles occupy
// one contiguous slot range, which the push hands to one thread block; where that
// pays the electrons' order by cell is made in two passes (two_passes_pay).  The
// order of particles inside a cell is not fixed (atomic scatter); nothing in a
// step depends on it: the deposit is an exact integer sum and the random
// numbers are keyed on particle ids.
#include <algorithm>

#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 4;
constexpr int kScanBlock = kScanThreads * kScanPer;

// sort key geometry: tiles of tx x ty x tz cells, ntx x nty tiles per plane;
// order: 0 one key per cell, 1 one key per tile (no order inside it), 2 one key
// per block of 2 x 2 x 2 cells inside the tile, kByTile the tile index itself
constexpr int kByTile = 3;
struct KeyGeo {
    int tx, ty, tz, ntx, nty, order;
};

// mixed: tile index * (cells per tile) + the cell's row-major index inside its
// tile (or of its block of 2 x 2 x 2 cells, or only the tile's first key: the
// sort order), or -1 for a dead slot
__device__ __forceinline__ int key_of(const float4& p, const KeyGeo& g)
{
    const int c = __float_as_int(p.w);   // packed i | j << 10 | k << 20
    if (c < 0) return -1;
    const int i = c & 1023, j = (c >> 10) & 1023, k = c >> 20;
    const int ti = i / g.tx, tj = j / g.ty, tk = k / g.tz;
    const int tile = (tk * g.nty + tj) * g.ntx + ti;
    if (g.order == kByTile) return tile;
    if (g.order == 1) return tile * (g.tx * g.ty * g.tz);
    if (g.order == 2) {
        const int bx = (g.tx + 1) >> 1, by = (g.ty + 1) >> 1;
        return tile * (g.tx * g.ty * g.tz) + (((k - tk * g.tz) >> 1) * by + ((j - tj * g.ty) >> 1)) * bx +
               ((i - ti * g.tx) >> 1);
    }
    return tile * (g.tx * g.ty * g.tz) + ((k - tk * g.tz) * g.ty + (j - tj * g.ty)) * g.tx + (i - ti * g.tx);
}
// FP64: the linear cell index (k*ny + j)*nx + i held in w
__device__ __forceinline__ int key_of(const double4& p, const KeyGeo&) { return p.w < 0.0 ? -1 : (int)p.w; }

// particles per thread and round of the histogram and scatter loops: their
// loads are all issued before the first key's atomic, so one round costs one
// memory latency instead of one per particle
constexpr int kSortUnroll = 4;

template <typename T4>
__global__ void k_hist(const T4* __restrict__ pos, const unsigned long long* nslot, int sp, unsigned int* hist,
                       KeyGeo kg)
{
    const unsigned long long n = nslot[sp];
    const int lane = threadIdx.x & 31;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    // the loop runs on the warp's first index, so every lane of a warp takes the
    // same rounds (the warp-wide match and shuffle below need all 32)
    for (unsigned long long w0 = blockIdx.x * (unsigned long long)blockDim.x + (threadIdx.x & ~31u); w0 < n;
         w0 += kSortUnroll * stride) {
        const unsigned long long q0 = w0 + (unsigned long long)lane;
        int key[kSortUnroll];
#pragma unroll
        for (int u = 0; u < kSortUnroll; ++u) {
            const unsigned long long q = q0 + u * stride;
            key[u] = q < n ? key_of(pos[q], kg) : -1;
        }
#pragma unroll
        for (int u = 0; u < kSortUnroll; ++u) {
            // lanes with the same key (common in nearly sorted input) add once
            const unsigned m = __match_any_sync(0xffffffffu, key[u]);
            if (key[u] >= 0 && lane == __ffs(m) - 1) atomicAdd(hist + key[u], (unsigned int)__popc(m));
        }
    }
}

// exclusive scan of one block of 1024 values; the block total goes to sums[blockIdx]
__global__ void k_scan_block(const unsigned int* in, unsigned int* out, unsigned int* sums, size_t n)
{
    __shared__ unsigned int warp_tot[kScanThreads / 32];
    const size_t base = (size_t)blockIdx.x * kScanBlock + (size_t)threadIdx.x * kScanPer;
    unsigned int v[kScanPer];
    unsigned int s = 0;
#pragma unroll
    for (int t = 0; t < kScanPer; ++t) {
        v[t] = (base + t < n) ? in[base + t] : 0u;
        s += v[t];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int incl = s;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        unsigned int w = lane < kScanThreads / 32 ? warp_tot[lane] : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned int y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        if (lane < kScanThreads / 32) warp_tot[lane] = w;
    }
    __syncthreads();
    unsigned int run = (incl - s) + (warp > 0 ? warp_tot[warp - 1] : 0u);
#pragma unroll
    for (int t = 0; t < kScanPer; ++t) {
        if (base + t < n) out[base + t] = run;
        run += v[t];
    }
    if (threadIdx.x == kScanThreads - 1) sums[blockIdx.x] = run;
}

__global__ void k_scan_add(unsigned int* out, const unsigned int* offs, size_t n)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x)
        out[q] += offs[q / kScanBlock];
}

// (mixed precision also lists the new slots of particles in MD cells for the
// next step: md_next / next_n, null for FP64)
template <typename T4>
__global__ void k_scatter(const T4* __restrict__ pos, const T4* __restrict__ vel, const unsigned long long* nslot,
                          int sp, unsigned int* cursor, T4* __restrict__ pos_out, T4* __restrict__ vel_out, KeyGeo kg,
                          int nx, int ny, const int* cell_ng, unsigned int* md_next, unsigned int* next_n)
{
    const unsigned long long n = nslot[sp];
    const int lane = threadIdx.x & 31;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    // the loop runs on the warp's first index, so every lane of a warp takes the
    // same rounds (the warp-wide match and shuffle below need all 32)
    for (unsigned long long w0 = blockIdx.x * (unsigned long long)blockDim.x + (threadIdx.x & ~31u); w0 < n;
         w0 += kSortUnroll * stride) {
        const unsigned long long q0 = w0 + (unsigned long long)lane;
        T4 p[kSortUnroll], v[kSortUnroll];
        int key[kSortUnroll];
        unsigned int dst[kSortUnroll];
#pragma unroll
        for (int u = 0; u < kSortUnroll; ++u) {
            const unsigned long long q = q0 + u * stride;
            if (q < n) {
                p[u] = pos[q];
                v[u] = vel[q];
            }
            key[u] = q < n ? key_of(p[u], kg) : -1;
        }
#pragma unroll
        for (int u = 0; u < kSortUnroll; ++u) {
            // one cursor atomic per group of lanes with the same key; the
            // group's lanes take consecutive slots in lane order
            const unsigned m = __match_any_sync(0xffffffffu, key[u]);
            const int leader = __ffs(m) - 1;
            unsigned int base = 0;
            if (key[u] >= 0 && lane == leader) base = atomicAdd(cursor + key[u], (unsigned int)__popc(m));
            dst[u] = base;
            dst[u] = __shfl_sync(0xffffffffu, dst[u], leader) + (unsigned int)__popc(m & ((1u << lane) - 1u));
        }
#pragma unroll
        for (int u = 0; u < kSortUnroll; ++u) {
            if (key[u] < 0) continue;
            const unsigned int d = dst[u];
            pos_out[d] = p[u];
            vel_out[d] = v[u];
            if (md_next) {
                const int pc = __float_as_int(p[u].w);   // mixed: packed cell
                if (cell_ng[((pc >> 20) * ny + ((pc >> 10) & 1023)) * nx + (pc & 1023)] != 0)
                    md_next[atomicAdd(next_n, 1u)] = d;
            }
        }
    }
}

// live records (key >= 0) among the slots in use, one add per warp
template <typename T4>
__global__ void k_count_live(const T4* __restrict__ pos, const unsigned long long* nslot, int sp,
                             unsigned long long* live)
{
    const unsigned long long n = nslot[sp];
    const KeyGeo kg{1, 1, 1, 1, 1, 1};
    unsigned int mine = 0;
    for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < n;
         q += (unsigned long long)gridDim.x * blockDim.x)
        mine += key_of(pos[q], kg) >= 0 ? 1u : 0u;
    const unsigned int w = __reduce_add_sync(0xffffffffu, mine);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(live + sp, (unsigned long long)w);
}

__global__ void k_set_nslot(unsigned long long* nslot, int sp, const unsigned int* total)
{
    nslot[sp] = *total;
}

// first slot of every tile after a scatter, which leaves cursor[key] at the end
// of the key's range: tile t starts where key t * per_tile - 1 ends
__global__ void k_tile_ranges(const unsigned int* cursor, unsigned int* tstart, long long ntiles, int per_tile)
{
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t <= ntiles;
         t += (long long)gridDim.x * blockDim.x)
        tstart[t] = t == 0 ? 0u : cursor[t * per_tile - 1];
}

// The second pass of the electrons' sort: one block per tile puts the tile's
// particles in cell order, from the buffers that the first pass sorted by tile
// into the others, slot range for slot range.  Counts per cell in shared memory,
// their exclusive scan, then each particle's place; up to kPermMax particles as
// a permutation (reads scattered inside the tile's few ten KB, writes in whole
// lines), more of them written to their places directly.
constexpr int kOrderThreads = 256;
constexpr int kOrderCells = 1024;   // largest tile, in cells
constexpr int kPermMax = 8192;

__global__ void __launch_bounds__(kOrderThreads) k_order_cells(const float4* __restrict__ pos, const float4* __restrict__ vel,
                                                               const unsigned int* __restrict__ tstart,
                                                               float4* __restrict__ pos_out, float4* __restrict__ vel_out,
                                                               KeyGeo kg, int nx, int ny, const unsigned char* tile_md,
                                                               const int* cell_ng, unsigned int* md_next, unsigned int* next_n)
{
    extern __shared__ unsigned int s_cell[];          // per cell: count, then next place
    __shared__ unsigned int warp_tot[kOrderThreads / 32];
    __shared__ unsigned short perm[kPermMax];
    const unsigned int first = tstart[blockIdx.x], n = tstart[blockIdx.x + 1] - first;
    if (n == 0u) return;
    const int per = kg.tx * kg.ty * kg.tz, t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int k_first = (int)blockIdx.x * per;        // key of the tile's first cell
    for (int q = t; q < per; q += kOrderThreads) s_cell[q] = 0u;
    __syncthreads();
    for (unsigned int q = t; q < n; q += kOrderThreads) atomicAdd(&s_cell[key_of(pos[first + q], kg) - k_first], 1u);
    __syncthreads();
    // exclusive scan: a run of cells per thread
    const int each = (per + kOrderThreads - 1) / kOrderThreads, c0 = min(t * each, per), c1 = min(c0 + each, per);
    unsigned int sum = 0u;
    for (int q = c0; q < c1; ++q) sum += s_cell[q];
    unsigned int incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned int y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    unsigned int run = incl - sum;
    for (int q = 0; q < w; ++q) run += warp_tot[q];
    for (int q = c0; q < c1; ++q) {
        const unsigned int here = s_cell[q];
        s_cell[q] = run;
        run += here;
    }
    __syncthreads();
    const bool md = md_next && tile_md[blockIdx.x];   // (the tile's own cells lie in its window)
    auto list_md = [&](const float4& p, unsigned int slot) {
        const int pc = __float_as_int(p.w);
        if (cell_ng[((pc >> 20) * ny + ((pc >> 10) & 1023)) * nx + (pc & 1023)] != 0) md_next[atomicAdd(next_n, 1u)] = slot;
    };
    if (n <= kPermMax) {
        for (unsigned int q = t; q < n; q += kOrderThreads)
            perm[atomicAdd(&s_cell[key_of(pos[first + q], kg) - k_first], 1u)] = (unsigned short)q;
        __syncthreads();
#pragma unroll 4
        for (unsigned int q = t; q < n; q += kOrderThreads) {
            const unsigned int from = first + perm[q];
            const float4 p = pos[from], v = vel[from];
            pos_out[first + q] = p;
            vel_out[first + q] = v;
            if (md) list_md(p, first + q);
        }
    } else {
        for (unsigned int q = t; q < n; q += kOrderThreads) {
            const float4 p = pos[first + q], v = vel[first + q];
            const unsigned int to = first + atomicAdd(&s_cell[key_of(p, kg) - k_first], 1u);
            pos_out[to] = p;
            vel_out[to] = v;
            if (md) list_md(p, to);
        }
    }
}

// exclusive scan of n values in place through the per-level scratch buffers;
// returns where the device finds their sum
unsigned int* scan(pic_ctx* c, unsigned int* data, size_t n, int level)
{
    const size_t nb = (n + kScanBlock - 1) / kScanBlock;
    unsigned int* sums = c->scan_tmp[level];
    k_scan_block<<<(unsigned)nb, kScanThreads, 0, c->stream>>>(data, data, sums, n);
    c->launches += 1;
    if (nb == 1) return sums;
    unsigned int* total = scan(c, sums, nb, level + 1);
    k_scan_add<<<grid_for((int64_t)n, 256, 152 * 8), 256, 0, c->stream>>>(data, sums, n);
    c->launches += 1;
    return total;
}

}  // namespace

void scan_cells(pic_ctx* c, unsigned int* data) { scan(c, data, c->cells, 0); }

// scratch: one block-sum buffer per scan level, for a key range of nkeys and for the
// cells (of the Coulomb pass).  Shorter ranges use the same buffers, so a caller
// asks anew only for a range longer than all before it; the old ones stay where the
// new cannot be had.
bool sort_scratch_setup(pic_ctx* c, size_t nkeys)
{
    std::vector<unsigned int*> tmp;
    for (size_t n = std::max(nkeys, c->cells);;) {
        n = (n + kScanBlock - 1) / kScanBlock;
        unsigned int* p = (unsigned int*)dev_alloc(c, sizeof(unsigned int) * n);
        if (!p) return false;
        tmp.push_back(p);
        if (n <= 1) break;
    }
    c->scan_tmp = tmp;
    return true;
}

void count_live(pic_ctx* c)
{
    cudaMemsetAsync(c->d_live, 0, 2 * sizeof(unsigned long long), c->stream);
    for (int sp = 0; sp < 2; ++sp) {
        const int grid = grid_for(c->cap[sp], 256, 152 * 8);
        if (c->prec == PIC_MIXED)
            k_count_live<float4><<<grid, 256, 0, c->stream>>>((const float4*)c->pos[sp], c->d_nslot, sp, c->d_live);
        else
            k_count_live<double4><<<grid, 256, 0, c->stream>>>((const double4*)c->pos[sp], c->d_nslot, sp, c->d_live);
    }
    c->launches += 2;
}

// Electrons in cell order can take two passes: by tile, then by cell inside each
// tile.  They cross about a third of a cell per step and axis, so a few steps after
// a sort a tile's electrons are spread over three times its cells: a scatter
// straight to cells is 32 separate 16-byte writes per warp and nearly one
// returning atomic per particle.  Most of a warp goes to one or a few tiles,
// though, and inside a tile the rest is local.  2.5e8 electrons on 256 x 256 x
// 1024 cells, sorted every 5 steps: histogram 1.6 and scatter 14.8 ms in one
// pass; 1.1, 3.0 and 3.7 ms in two (16 GB each of records read and written:
// 2.6 ms is the memory's).  Ions hardly move between sorts: their one pass writes
// whole lines already (3.4 ms).
//
// The second pass gives a tile to one block, whatever it holds, so it pays only
// where many tiles hold a fair number of particles each, and where the electrons
// have moved.  Particle half of a step with 1 to 2.4e8 electrons, sorted every
// 5 steps (others in brackets), two passes against one:
//   tiles (8 x 8 x 8)        131072 0.85  65536 0.88-0.98  16384 0.90-0.99  8192 0.95-0.99
//                            4096 0.96-1.01 [1.23]  2048 0.98-1.24 [1.66]  16 1.18 [1.89]
//   4096 tiles, per tile     977: 0.98  2441: 0.96-0.99  4882: 1.00-1.01 [1.07]
//   16384 tiles, per tile    488: 0.95  6104: 0.90  7019: 0.93  9155 (beyond kPermMax in part): 1.03 [1.41]
//   cells per tile           64: 1.00 at 122 to 305 a tile, 0.89 at 457 to 763  256: 0.85-0.96
//                            1024: 0.90-0.98 (8192 tiles or more)  2048: 1.03-1.16 [1.33]  4096: 1.06-1.19 [1.39]
//   cells crossed per sort   16384 tiles 0.04: 1.13-1.22  0.36: 1.00-1.14  0.54: 0.98-1.01  0.73: 0.95-1.00
//                            1.8: 0.90-0.99  3.6: 0.95-1.00  7.3: 0.98-1.01; 131072 tiles 0.36: 0.96
//                            8192 tiles 3.6: 0.96-1.00  7.3: 1.00-1.03
// `cells crossed` takes electrons of 3 eV, the workloads' temperature; the particle
// count is the run's first.
bool two_passes_pay(const pic_ctx* c)
{
    if (c->prec != PIC_MIXED || c->sort_order != 0) return false;
    const double cells = (double)c->tile[0] * c->tile[1] * c->tile[2];
    const double tiles = (double)c->ntiles, each = (double)c->n_first[0] / tiles;
    const double crossed = c->sort_every * c->dt * 7.3e5 / c->dx;
    return cells >= 64 && cells <= kOrderCells && each <= kPermMax * 7 / 8 && each + cells >= 500 &&
           (tiles >= 8192 || (tiles >= 4096 && each <= 2500)) && crossed >= (tiles >= 65536 ? 0.3 : 0.6) &&
           crossed <= tiles / 2048;
}

bool sort_swaps(const pic_ctx* c, int sp) { return !(sp == 0 && c->two_pass); }

void sort_particles(pic_ctx* c, int sp)
{
    const bool mixed = c->prec == PIC_MIXED, two = !sort_swaps(c, sp);
    const int per = c->tile[0] * c->tile[1] * c->tile[2];
    const size_t nk = two ? (size_t)c->ntiles : c->nkeys;
    KeyGeo kg{c->tile[0], c->tile[1], c->tile[2], c->ntile[0], c->ntile[1], two ? kByTile : c->sort_order};
    cudaMemsetAsync(c->cursor, 0, sizeof(unsigned int) * nk, c->stream);
    const int grid = grid_for(c->cap[sp], 256, 152 * 8);
    if (mixed)
        k_hist<float4><<<grid, 256, 0, c->stream>>>((const float4*)c->pos[sp], c->d_nslot, sp, c->cursor, kg);
    else
        k_hist<double4><<<grid, 256, 0, c->stream>>>((const double4*)c->pos[sp], c->d_nslot, sp, c->cursor, kg);
    const unsigned int* total = scan(c, c->cursor, nk, 0);
    if (mixed) cudaMemsetAsync(c->d_lists + 4 + sp, 0, sizeof(unsigned int), c->stream);
    if (mixed)
        k_scatter<float4><<<grid, 256, 0, c->stream>>>((const float4*)c->pos[sp], (const float4*)c->vel[sp],
                                                       c->d_nslot, sp, c->cursor, (float4*)c->pos_alt[sp],
                                                       (float4*)c->vel_alt[sp], kg, c->nx, c->ny, c->cell_ng,
                                                       two ? nullptr : c->md_next[sp], c->d_lists + 4 + sp);
    else
        k_scatter<double4><<<grid, 256, 0, c->stream>>>((const double4*)c->pos[sp], (const double4*)c->vel[sp],
                                                        c->d_nslot, sp, c->cursor, (double4*)c->pos_alt[sp],
                                                        (double4*)c->vel_alt[sp], kg, c->nx, c->ny, c->cell_ng,
                                                        (unsigned int*)nullptr, (unsigned int*)nullptr);
    // the last scan level's single block sum is the number of live particles
    k_set_nslot<<<1, 1, 0, c->stream>>>(c->d_nslot, sp, total);
    c->launches += 3;
    if (mixed) {
        k_tile_ranges<<<grid_for(c->ntiles + 1, 256, 152 * 4), 256, 0, c->stream>>>(
            c->cursor, c->tstart[sp], (long long)c->ntiles, two ? 1 : per);
        c->launches += 1;
    }
    if (two) {
        kg.order = 0;
        k_order_cells<<<(unsigned)c->ntiles, kOrderThreads, sizeof(unsigned int) * (size_t)per, c->stream>>>(
            (const float4*)c->pos_alt[sp], (const float4*)c->vel_alt[sp], c->tstart[sp], (float4*)c->pos[sp],
            (float4*)c->vel[sp], kg, c->nx, c->ny, c->tile_md, c->cell_ng, c->md_next[sp], c->d_lists + 4 + sp);
        c->launches += 1;
        return;
    }
    std::swap(c->pos[sp], c->pos_alt[sp]);
    std::swap(c->vel[sp], c->vel_alt[sp]);
}

}  // namespace pic
