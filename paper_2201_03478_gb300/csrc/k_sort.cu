// k_sort.cu -- binning of the pointings before interpolation (the cube is read
// through p x p stencils, Sect. 2.1 interpolation step): a counting sort of
// the samples by grid cell, plus a per-sample stencil record.
//
// A sample's cell is (base row i, base column j) of its stencil.  Cells are
// grouped into tiles of kTileRows x tile_cols; the sort key is either the tile
// (coarse) or the cell in tile-major order (fine), so that both orders list
// each tile's samples contiguously.  With fine keys the samples of one cell
// are adjacent and neighbouring threads read the same cube nodes.
//
//   k_bin:        pointing -> (i, j) in double; key; record {theta - theta(i-1),
//                 phi fraction, [reduced psi], cell}; key histogram
//   k_scan_local / (k_scan_blocks) / k_scan_add:  exclusive prefix sum of the histogram
//                 -> first position of every key (and a cursor copy)
//   k_scatter_agg: perm[cursor[key]++] = s, the cursor atomics aggregated per
//                 chunk of samples in shared memory (order within a key unspecified)
//   k_tile_chunks: work items of at most kChunk samples per tile (adjoint)
#include "sl_internal.cuh"

namespace sl {

constexpr int kChunk = kWorkChunk;
constexpr int kScanBlock = 4096;    // keys per CTA of k_scan_local (1024 threads x 4)

// Runs of equal keys among the warp's lanes (the active lanes are a prefix of
// the warp: lanes 0 .. nact - 1): the run of this lane starts at lane *head and
// holds *cnt lanes.  One atomic per run replaces one per lane; lanes of a scan
// that share a cell are almost always adjacent, and a key that recurs after
// another key just starts another run.  (Grouping all equal keys with
// __match_any_sync costs a multi-pass instruction per lane group, which bound
// the binning and the scatter.)
__device__ __forceinline__ void key_run(unsigned key, bool ok, unsigned lane, int *head, unsigned *cnt) {
    const unsigned prev = __shfl_up_sync(0xffffffffu, key, 1);
    const unsigned act = __ballot_sync(0xffffffffu, ok);
    const unsigned heads = __ballot_sync(0xffffffffu, ok && (lane == 0 || key != prev));
    const unsigned upto = (lane == 31) ? 0xffffffffu : ((2u << lane) - 1u);   // lanes 0 .. lane
    *head = 31 - __clz(heads & upto);
    const unsigned after = heads & ~upto;
    const int next = after ? __ffs(after) - 1 : 32;
    const int nact = __popc(act);
    *cnt = (unsigned)(min(next, nact) - *head);
}

// Samples [*beg, *end) of this CTA in k_bin: one contiguous slice
// of the TOD per CTA (a multiple of blockDim.x long), walked blockDim.x at a
// time.  A scan repeats the same circle on the sky every few thousand samples,
// so a grid-stride walk -- every resident CTA on one contiguous stretch of the
// TOD -- sends hundreds of warps to the same cells' counters at once, and
// their atomics serialise; slices put the CTAs on different stretches.
__device__ __forceinline__ void cta_slice(int64_t n, int64_t *beg, int64_t *end) {
    const int64_t per = ((n + gridDim.x - 1) / gridDim.x + blockDim.x - 1) / blockDim.x * blockDim.x;
    *beg = min(n, (int64_t)blockIdx.x * per);
    *end = min(n, *beg + per);
}

template <bool REC64>
__global__ void __launch_bounds__(256) k_bin(const InterpGeom g, int fine, const double *__restrict__ theta,
                                             const double *__restrict__ phi, const double *__restrict__ psi,
                                             int64_t n, unsigned *__restrict__ keys, void *__restrict__ rec,
                                             unsigned *__restrict__ hist) {
    const unsigned lane = threadIdx.x & 31;
    int64_t sbeg, send;
    cta_slice(n, &sbeg, &send);
    for (int64_t s0 = sbeg; s0 < send; s0 += blockDim.x) {
        const int64_t s = s0 + threadIdx.x;
        const bool ok = s < send;
        unsigned key = 0xffffffffu;
        if (ok) {
            const double th = theta[s];
            const int i = locate_row(g, th);
            unsigned long long fr;
            int sh;
            const int j = locate_col_fix(g, phi[s], fr, sh);
            // tile_cols is 8, 16 or 32 and i + 1 >= 0: shifts and masks instead of divisions
            const int tlg = __ffs(g.tile_cols) - 1;
            const int tr = (int)((unsigned)(i + 1) / kTileRows), li = (i + 1) - tr * kTileRows;
            const int tc = j >> tlg, lj = j & (g.tile_cols - 1);
            const unsigned tile = (unsigned)tr * (unsigned)g.ntc + (unsigned)tc;
            key = fine ? tile * (unsigned)(kTileRows * g.tile_cols) + (unsigned)(li * g.tile_cols + lj) : tile;
            [[maybe_unused]] const unsigned nkeys = (unsigned)(g.ntr * g.ntc) * (fine ? (unsigned)(kTileRows * g.tile_cols) : 1u);
            if (!SL_GUARD(i >= -1 && i < g.R && j >= 0 && j < g.nphi && key < nkeys, 0x101u)) key = 0;
            keys[s] = key;
            // theta - theta(i0), i0 = i - p/2 + 1 the first stencil row (index i0 + half = i + 1),
            // in 2^-60 fixed point (exact for theta >= 2^-8)
            long long tf = 0;
            const bool tfix = to_fix<60>(th, tf);
            const long long dfix = tf - __ldg(g.ring_fix + i + 1);
            const unsigned cell = ((unsigned)(i + 1) << 16) | (unsigned)j;
            if (REC64) {
                const double dth = tfix ? fix_to_d<60>(dfix) : th - __ldg(g.ring_ext + i + 1);
                reinterpret_cast<StencilRec64 *>(rec)[s] = StencilRec64{dth, frac_bits_d(fr, sh), cell, 0u};
            } else {
                const float dth = tfix ? fix_to_f<60>(dfix) : d2f_bits(th - __ldg(g.ring_ext + i + 1));
                // psi reduced to [-pi, pi] in 2^-59 fixed point; |psi| >= 8 (and NaN) in FP64
                const double ps = psi[s];
                long long pf;
                float psr;
                if (to_fix<59>(ps, pf)) {
                    constexpr long long kPi59 = 1811004864519280711ll, k2Pi59 = 3622009729038561421ll;
                    if (pf > kPi59) pf -= k2Pi59;
                    else if (pf < -kPi59) pf += k2Pi59;
                    psr = fix_to_f<59>(pf);
                } else {
                    psr = d2f_bits(ps - 6.283185307179586 * rint(ps * 0.15915494309189535));
                }
                reinterpret_cast<StencilRec32 *>(rec)[s] = StencilRec32{dth, frac_bits_f(fr, sh), psr, cell};
            }
        }
        int head;
        unsigned cnt;
        key_run(key, ok, lane, &head, &cnt);
        if (ok && (int)lane == head) atomicAdd(hist + key, cnt);
    }
}

// Block-wide exclusive scan of 1024 values (one per thread); returns the total.
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned &excl) {
    __shared__ unsigned s_w[32];
    __shared__ unsigned s_tot;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned a = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, a, o);
        if ((int)lane >= o) a += y;
    }
    if (lane == 31) s_w[warp] = a;
    __syncthreads();
    if (warp == 0) {
        unsigned w = s_w[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
            if ((int)lane >= o) w += y;
        }
        s_w[lane] = w;
        if (lane == 31) s_tot = w;
    }
    __syncthreads();
    excl = (warp ? s_w[warp - 1] : 0u) + a - v;
    const unsigned tot = s_tot;
    __syncthreads();
    return tot;
}

// Sum of x over the CTA (1024 threads), in every thread.
__device__ __forceinline__ unsigned block_sum(unsigned x) {
    __shared__ unsigned s_part[32];
    x = __reduce_add_sync(0xffffffffu, x);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = x;
    __syncthreads();
    x = __reduce_add_sync(0xffffffffu, s_part[threadIdx.x & 31]);
    __syncthreads();
    return x;
}

// Four words from data + base on (zero from n on), one 16-byte access where data is aligned.
__device__ __forceinline__ uint4 load4(const unsigned *data, int64_t base, int64_t n) {
    if (base + 3 < n && ((uintptr_t)data & 15) == 0) return *reinterpret_cast<const uint4 *>(data + base);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (base < n) v.x = data[base];
    if (base + 1 < n) v.y = data[base + 1];
    if (base + 2 < n) v.z = data[base + 2];
    if (base + 3 < n) v.w = data[base + 3];
    return v;
}
__device__ __forceinline__ void store4(unsigned *data, int64_t base, int64_t n, uint4 v) {
    if (base + 3 < n && ((uintptr_t)data & 15) == 0) {
        *reinterpret_cast<uint4 *>(data + base) = v;
        return;
    }
    if (base < n) data[base] = v.x;
    if (base + 1 < n) data[base + 1] = v.y;
    if (base + 2 < n) data[base + 2] = v.z;
    if (base + 3 < n) data[base + 3] = v.w;
}

// Per CTA: exclusive scan of data[b*4096 .. +4096) in place, block total to bsum[b] and, with nz,
// the number of nonzero entries to nz[b].
__global__ void __launch_bounds__(1024) k_scan_local(int64_t n, unsigned *__restrict__ data,
                                                      unsigned *__restrict__ bsum, unsigned *__restrict__ nz) {
    const int64_t base = (int64_t)blockIdx.x * kScanBlock + 4 * threadIdx.x;
    const uint4 v = load4(data, base, n);
    unsigned ex;
    const unsigned tot = block_exclusive_scan(v.x + v.y + v.z + v.w, ex);
    store4(data, base, n, make_uint4(ex, ex + v.x, ex + v.x + v.y, ex + v.x + v.y + v.z));
    const unsigned nonzero = nz ? block_sum((v.x != 0u) + (v.y != 0u) + (v.z != 0u) + (v.w != 0u)) : 0u;
    if (threadIdx.x == 0) {
        bsum[blockIdx.x] = tot;
        if (nz) nz[blockIdx.x] = nonzero;
    }
}

// Exclusive scan of bsum[0 .. nb) in place, bsum[nb] = total, by one CTA.
__global__ void __launch_bounds__(1024) k_scan_blocks(int nb, unsigned *__restrict__ bsum) {
    unsigned carry = 0;
    for (int base = 0; base < nb; base += kScanBlock) {
        const int i = base + 4 * threadIdx.x;
        const uint4 v = load4(bsum, i, nb);
        unsigned ex;
        const unsigned tot = block_exclusive_scan(v.x + v.y + v.z + v.w, ex);
        ex += carry;
        store4(bsum, i, nb, make_uint4(ex, ex + v.x, ex + v.x + v.y, ex + v.x + v.y + v.z));
        carry += tot;
    }
    if (threadIdx.x == 0) bsum[nb] = carry;
}

// Adds the totals of the CTAs before to k_scan_local's sums and copies them to cursor; the
// last CTA also writes data[n] = total and, with occ, *occ = the sum of nz.  Up to kScanQuadratic
// CTAs every one sums the earlier totals itself (nb^2 / 2 words from L2, 0.5 MB at 1024 x 2048
// cells): a scan of them by one CTA in between, and of the tiles' chunks by another, cost the small
// and sparse sorts two launches, and with the tiles' strided words more than the rest of the scan
// (1500 x 3000 cells: 17 + 5 + 12 + 4 + 66 us, now 10 + 11 + 37).  The work grows with the square of
// the cells, so beyond (SCANNED) k_scan_blocks runs in between: 16384^2 cells 1.23 -> 0.95 ms,
// 32768 x 16384 3.71 -> 1.88.
constexpr int64_t kScanQuadratic = 65536;

template <bool SCANNED>
__global__ void __launch_bounds__(1024) k_scan_add(int64_t n, unsigned *__restrict__ data, const unsigned *__restrict__ bsum,
                                                    const unsigned *__restrict__ nz, unsigned *__restrict__ cursor,
                                                    unsigned *__restrict__ occ) {
    const int64_t base = (int64_t)blockIdx.x * kScanBlock + 4 * threadIdx.x;
    uint4 v = load4(data, base, n);
    unsigned before = 0;
    if (SCANNED) {
        before = bsum[blockIdx.x];
    } else {
        for (unsigned i = threadIdx.x; i < blockIdx.x; i += 1024) before += bsum[i];
        before = block_sum(before);
    }
    v = make_uint4(before + v.x, before + v.y, before + v.z, before + v.w);
    store4(data, base, n, v);
    store4(cursor, base, n, v);
    if (blockIdx.x != gridDim.x - 1) return;
    if (occ) {
        unsigned o = 0;
        for (unsigned i = threadIdx.x; i < gridDim.x; i += 1024) o += nz[i];
        o = block_sum(o);
        if (threadIdx.x == 0) *occ = o;
    }
    if (threadIdx.x == 0) data[n] = SCANNED ? bsum[gridDim.x] : before + bsum[blockIdx.x];
}

// The scatter with its atomics aggregated per chunk of kAggChunk samples: a
// shared-memory hash table gives every sample of the chunk its rank among the
// chunk's samples of the same key (a shared atomic); then one global atomic per
// distinct key reserves the key's range, these atomics issued eight at a time
// and independent of each other, so their round trips overlap; last, each
// sample goes to its range start plus its rank.  Along a scan a 4096-sample
// chunk holds about two visits of every cell of a circle; a per-lane scatter
// (one returning atomic per run of equal keys in a warp) waited for one
// round trip per warp and 32 samples.
// PER samples a thread: 16 where that fills the chip; 2 below, so that a short TOD spreads over
// more CTAs and each clears and walks an eighth of the table (1e5 uniform samples 22 -> 8 us, 1e6 29
// -> 20; from 1.2e6 on the larger chunk's fewer global atomics are as good: 3e6 65 us).
constexpr int kAggThreads = 256;
constexpr int agg_chunk(int per) { return kAggThreads * per; }
constexpr int agg_log(int per) { return per == 16 ? 13 : 10; }   // slots: 2 x the chunk's samples
static_assert((1 << agg_log(16)) == 2 * agg_chunk(16) && (1 << agg_log(2)) == 2 * agg_chunk(2),
              "the hash table must hold every distinct key of a chunk");
constexpr unsigned kNoKey = 0xffffffffu;

template <int PER>
__global__ void __launch_bounds__(kAggThreads) k_scatter_agg(int64_t n, int64_t nkeys, const unsigned *__restrict__ keys,
                                                             unsigned *__restrict__ cursor,
                                                             unsigned *__restrict__ perm) {
    constexpr int CHUNK = agg_chunk(PER), LOG = agg_log(PER), SLOTS = 1 << LOG;
    constexpr int NQ = SLOTS / kAggThreads < 8 ? SLOTS / kAggThreads : 8;   // atomics in flight a thread
    extern __shared__ __align__(16) unsigned agg_smem[];
    unsigned *hkey = agg_smem, *hval = agg_smem + SLOTS;   // key per slot; count, then range start
    const int64_t per = (n + (int64_t)gridDim.x * CHUNK - 1) / ((int64_t)gridDim.x * CHUNK) * CHUNK;
    const int64_t sbeg = min(n, (int64_t)blockIdx.x * per), send = min(n, sbeg + per);
    for (int64_t c0 = sbeg; c0 < send; c0 += CHUNK) {
        for (int i = threadIdx.x; i < SLOTS / 4; i += kAggThreads) {
            reinterpret_cast<uint4 *>(hkey)[i] = make_uint4(kNoKey, kNoKey, kNoKey, kNoKey);
            reinterpret_cast<uint4 *>(hval)[i] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
        unsigned slot[PER], rank[PER];
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int64_t s = c0 + (int64_t)j * kAggThreads + threadIdx.x;
            slot[j] = SLOTS;
            rank[j] = 0u;
            if (s < send) {
                unsigned key = keys[s];
                if (!SL_GUARD(key < nkeys, 0x102u)) key = 0;
                unsigned h = (key * 2654435761u) >> (32 - LOG);
                // linear probing; the table holds more slots than the chunk has samples,
                // so a free or matching slot is always found within SLOTS probes
                for (int probe = 0; probe < SLOTS; ++probe) {
                    const unsigned prev = atomicCAS(&hkey[h], kNoKey, key);
                    if (prev == kNoKey || prev == key) break;
                    h = (h + 1u) & (SLOTS - 1);
                }
                slot[j] = h;
                rank[j] = atomicAdd(&hval[h], 1u);
            }
        }
        __syncthreads();
        for (int i0 = threadIdx.x; i0 < SLOTS; i0 += NQ * kAggThreads) {
            unsigned got[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int i = i0 + q * kAggThreads;
                const unsigned k = hkey[i];
                got[q] = (k != kNoKey) ? atomicAdd(cursor + k, hval[i]) : 0u;
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int i = i0 + q * kAggThreads;
                if (hkey[i] != kNoKey) hval[i] = got[q];
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (slot[j] >= SLOTS) continue;
            const int64_t s = c0 + (int64_t)j * kAggThreads + threadIdx.x;
            const unsigned pos = hval[slot[j]] + rank[j];
            if (SL_GUARD(pos < n, 0x103u)) perm[pos] = (unsigned)s;
        }
        __syncthreads();   // the table is cleared for the next chunk
    }
}

// chunk_off[t] = sum over the tiles before t of ceil(#samples / kChunk), chunk_off[ntiles] = total.
// One CTA per 1024 tiles, which up to kTilesQuadratic tiles also sums the chunks of the tiles before its
// own (37 us at 1500 x 3000 cells, bound by its strided reads; the counts and a single CTA's scan
// took 4 + 66).  That is the square of the tiles (3000 x 6000 cells still as fast, 4096 x 8192 0.06 ms
// slower, 32768 x 16384 63 ms of a call of 73), so beyond (tot given) the CTAs scan their own tiles and
// leave their totals, and k_chunk_add adds those before (calls of 1e5 FP32 samples: 4096 x 8192 cells
// 1.63 -> 1.24 ms, 8192 x 16384 5.9 -> 2.0, 32768 x 16384 73 -> 4.0).
constexpr int kTilesQuadratic = 160000;

__global__ void __launch_bounds__(1024) k_tile_chunks(int ntiles, int ncell, const unsigned *__restrict__ start,
                                                       unsigned *__restrict__ chunk_off, unsigned *__restrict__ tot) {
    auto chunks = [&](int t) {
        return (start[(int64_t)(t + 1) * ncell] - start[(int64_t)t * ncell] + kChunk - 1) / kChunk;
    };
    const int t0 = blockIdx.x * 1024, t = t0 + threadIdx.x;
    unsigned before = 0;
    if (!tot) {
#pragma unroll 4
        for (int i = threadIdx.x; i < t0; i += 1024) before += chunks(i);
        before = block_sum(before);
    }
    unsigned ex;
    const unsigned own = block_exclusive_scan(t < ntiles ? chunks(t) : 0u, ex);
    if (t < ntiles) chunk_off[t] = before + ex;
    if (threadIdx.x != 0) return;
    if (tot) tot[blockIdx.x] = own;
    else if (t0 + 1024 >= ntiles) chunk_off[ntiles] = before + own;
}

__global__ void __launch_bounds__(1024) k_chunk_add(int ntiles, const unsigned *__restrict__ tot, unsigned *__restrict__ chunk_off) {
    unsigned before = 0;
    for (unsigned i = threadIdx.x; i < blockIdx.x; i += 1024) before += tot[i];
    before = block_sum(before);
    const int t = blockIdx.x * 1024 + threadIdx.x;
    if (t < ntiles) chunk_off[t] += before;
    if (threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) chunk_off[ntiles] = before + tot[blockIdx.x];
}

SL_CHECK_READER(chk_sort)

constexpr int kAggFull = 304;   // chunks of 4096 samples that fill the chip (two CTAs an SM)

static unsigned grid_for(int64_t n, int bs) {
    int64_t b = (n + bs - 1) / bs;
    const int64_t cap = 152 * 16;
    return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

int64_t sort_nkeys(const sl_plan *p, int fine) {
    return fine ? (int64_t)p->ntiles * kTileRows * p->geom.tile_cols : (int64_t)p->ntiles;
}

int64_t sort_nbsum(int64_t nkeys) { return (nkeys + kScanBlock - 1) / kScanBlock; }

sl_status launch_sort_into(sl_plan *p, const SortBufs &b, const double *theta, const double *phi,
                           const double *psi, int64_t n, int fine, int rec64, int with_chunks) {
    const int64_t nkeys = sort_nkeys(p, fine), nb = sort_nbsum(nkeys);
    const int ncell = fine ? kTileRows * p->geom.tile_cols : 1;
    sl_status st = cuda_check(cudaMemsetAsync(b.hist, 0, (nkeys + 1) * sizeof(unsigned), p->stream), "memset hist");
    if (st != SL_OK) return st;
    int slot = timing_begin(p, "bin");
    if (rec64)
        k_bin<true><<<grid_for(n, 256), 256, 0, p->stream>>>(p->geom, fine, theta, phi, psi, n, b.keys, b.rec, b.hist);
    else
        k_bin<false><<<grid_for(n, 256), 256, 0, p->stream>>>(p->geom, fine, theta, phi, psi, n, b.keys, b.rec, b.hist);
    timing_end(p, slot);
    if ((st = cuda_check(cudaGetLastError(), "k_bin launch")) != SL_OK) return st;
    slot = timing_begin(p, "scan");
    unsigned *nz = b.occ ? b.occ + 1 : nullptr;
    k_scan_local<<<(unsigned)nb, 1024, 0, p->stream>>>(nkeys, b.hist, b.bsum, nz);
    if (nb > kScanQuadratic) {
        k_scan_blocks<<<1, 1024, 0, p->stream>>>((int)nb, b.bsum);
        k_scan_add<true><<<(unsigned)nb, 1024, 0, p->stream>>>(nkeys, b.hist, b.bsum, nz, b.cursor, b.occ);
    } else {
        k_scan_add<false><<<(unsigned)nb, 1024, 0, p->stream>>>(nkeys, b.hist, b.bsum, nz, b.cursor, b.occ);
    }
    timing_end(p, slot);
    if ((st = cuda_check(cudaGetLastError(), "k_scan launch")) != SL_OK) return st;
    slot = timing_begin(p, "scatter");
    {
        const bool big = n >= (int64_t)kAggFull * agg_chunk(16);
        auto kern = big ? k_scatter_agg<16> : k_scatter_agg<2>;
        const int chunk = agg_chunk(big ? 16 : 2);
        const size_t sm = 4 * (size_t)chunk * sizeof(unsigned);
        if ((st = cuda_check(allow_dyn_smem(kern, sm), "k_scatter_agg smem attribute")) != SL_OK) return st;
        const int64_t nchunk = (n + chunk - 1) / chunk;
        const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nchunk, 152 * 3 * 4));
        kern<<<grid, kAggThreads, sm, p->stream>>>(n, nkeys, b.keys, b.cursor, b.perm);
    }
    timing_end(p, slot);
    if ((st = cuda_check(cudaGetLastError(), "k_scatter_agg launch")) != SL_OK) return st;
    if (with_chunks) {
        // the totals go over the block sums, which are done with: 1024 tiles take more than 4096 keys
        const unsigned nc = (unsigned)((p->ntiles + 1023) / 1024);
        const bool apart = fine && p->ntiles > kTilesQuadratic;
        k_tile_chunks<<<nc, 1024, 0, p->stream>>>(p->ntiles, ncell, b.hist, b.chunk_off, apart ? b.bsum : nullptr);
        if (apart) k_chunk_add<<<nc, 1024, 0, p->stream>>>(p->ntiles, b.bsum, b.chunk_off);
        st = cuda_check(cudaGetLastError(), "k_tile_chunks launch");
    }
    return st;
}

}  // namespace sl
