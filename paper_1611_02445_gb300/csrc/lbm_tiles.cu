// lbm_tiles.cu -- tile-map builder (Algorithm 1 on the GPU), per-tile metadata,
// equilibrium initialisation, FP64 invariant reduction, macroscopic export and the
// dense <-> tile-major conversions of liblbm_gb300.
#include <algorithm>

#include "lbm_internal.cuh"
#include "lbm_df.cuh"
#include "lbm_store.cuh"

namespace lbm {

// ----------------------------------------------------------------------------------
// Algorithm 1 (Sec. 3.1) as flag -> exclusive scan -> scatter. The scan runs over the
// linear tile index t = tx + Tx (ty + Ty tz), which is the loop order of Algorithm 1,
// so ranks equal the paper's discovery order.

// flag[t] = 1 when some node of tile t is not solid; padding nodes count as solid.
__global__ void k_tile_flags(const uint8_t* __restrict__ nt, int nx, int ny, int nz, int Tx, int Ty,
                             int Tz, uint8_t* __restrict__ flag, int* __restrict__ bad) {
    const int64_t nT = (int64_t)Tx * Ty * Tz;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nT;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int tx = (int)(t % Tx);
        const int64_t r = t / Tx;
        const int ty = (int)(r % Ty);
        const int tz = (int)(r / Ty);
        int any = 0, badv = 0;
        for (int dz = 0; dz < TILE; dz++) {
            const int z = TILE * tz + dz;
            if (z >= nz) break;
            for (int dy = 0; dy < TILE; dy++) {
                const int y = TILE * ty + dy;
                if (y >= ny) break;
                const uint8_t* row = nt + ((int64_t)z * ny + y) * nx;
                for (int dx = 0; dx < TILE; dx++) {
                    const int x = TILE * tx + dx;
                    if (x >= nx) break;
                    const uint8_t v = row[x];
                    any |= (v != LBM_SOLID);
                    badv |= (v > LBM_OUTLET);
                }
            }
        }
        flag[t] = (uint8_t)any;
        if (badv) atomicOr(bad, 1);
    }
}

constexpr int SCAN_BLOCK = 1024;

// Exclusive prefix sum of v over the 1024 threads of a block; *total gets the sum.
__device__ int64_t block_exclusive_scan(int64_t v, int64_t* total) {
    __shared__ int64_t warp_sums[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int64_t s = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        warp_sums[lane] = s;   // inclusive over warps
    }
    __syncthreads();
    const int64_t before = (warp > 0 ? warp_sums[warp - 1] : 0) + x - v;
    *total = warp_sums[31];
    __syncthreads();
    return before;
}

__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_sums(const uint8_t* __restrict__ flag, int64_t n,
                                                          int64_t* __restrict__ block_sums) {
    const int64_t t = blockIdx.x * (int64_t)SCAN_BLOCK + threadIdx.x;
    const int64_t v = t < n ? flag[t] : 0;
    int64_t total;
    block_exclusive_scan(v, &total);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

// One block: exclusive scan of the block sums in chunks of 1024 with a running carry.
__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_top(int64_t* __restrict__ block_sums, int64_t nb,
                                                         int64_t* __restrict__ d_count) {
    int64_t carry = 0;
    for (int64_t base = 0; base < nb; base += SCAN_BLOCK) {
        const int64_t i = base + threadIdx.x;
        const int64_t v = i < nb ? block_sums[i] : 0;
        int64_t total;
        const int64_t ex = block_exclusive_scan(v, &total);
        if (i < nb) block_sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) *d_count = carry;
}

__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_scatter(const uint8_t* __restrict__ flag, int64_t n,
                                                             const int64_t* __restrict__ block_off,
                                                             int32_t* __restrict__ tile_map,
                                                             uint32_t* __restrict__ non_empty) {
    const int64_t t = blockIdx.x * (int64_t)SCAN_BLOCK + threadIdx.x;
    const int64_t v = t < n ? flag[t] : 0;
    int64_t total;
    const int64_t rank = block_off[blockIdx.x] + block_exclusive_scan(v, &total);
    if (t < n) {
        tile_map[t] = v ? (int32_t)rank : -1;
        if (v) non_empty[rank] = (uint32_t)t;
    }
}

int64_t scan_block_count(int64_t n) { return (n + SCAN_BLOCK - 1) / SCAN_BLOCK; }

cudaError_t launch_tile_flags(const uint8_t* nt, int nx, int ny, int nz, int Tx, int Ty, int Tz,
                              uint8_t* flag, int* bad, cudaStream_t st) {
    const int64_t nT = (int64_t)Tx * Ty * Tz;
    const int64_t blocks = std::min<int64_t>((nT + 255) / 256, 152 * 64);
    k_tile_flags<<<(unsigned)std::max<int64_t>(blocks, 1), 256, 0, st>>>(nt, nx, ny, nz, Tx, Ty, Tz, flag, bad);
    return cudaGetLastError();
}

cudaError_t launch_scan_flags(const uint8_t* flag, int64_t n, int32_t* tile_map, uint32_t* non_empty,
                              int64_t* d_count, int64_t* block_sums, int64_t nblocks, cudaStream_t st) {
    k_scan_sums<<<(unsigned)nblocks, SCAN_BLOCK, 0, st>>>(flag, n, block_sums);
    k_scan_top<<<1, SCAN_BLOCK, 0, st>>>(block_sums, nblocks, d_count);
    k_scan_scatter<<<(unsigned)nblocks, SCAN_BLOCK, 0, st>>>(flag, n, block_sums, tile_map, non_empty);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Per-tile metadata: node types in slot order, the solid mask, the boundary flag and
// the 3x3x3 neighbourhood of tile ranks (the local tileMap copy of Sec. 3.4), wrapped on
// periodic axes. One 64-thread block per kept tile, thread s = slot s.
__global__ void __launch_bounds__(64) k_tile_meta(const uint8_t* __restrict__ nt, int nx, int ny, int nz,
                                                  int Tx, int Ty, int Tz, unsigned periodic,
                                                  const int32_t* __restrict__ tile_map,
                                                  const uint32_t* __restrict__ non_empty, int64_t n_tiles,
                                                  int32_t* __restrict__ nbr, uint64_t* __restrict__ smask,
                                                  uint32_t* __restrict__ tflags, uint8_t* __restrict__ ntype,
                                                  unsigned long long* __restrict__ n_nonsolid) {
    __shared__ uint32_t s_solid[2], s_bc[2];
    const int s = threadIdx.x, lane = s & 31, warp = s >> 5;
    for (int64_t k = blockIdx.x; k < n_tiles; k += gridDim.x) {
        const uint32_t t = non_empty[k];
        const int tx = (int)(t % (uint32_t)Tx);
        const int ty = (int)((t / (uint32_t)Tx) % (uint32_t)Ty);
        const int tz = (int)(t / ((uint32_t)Tx * (uint32_t)Ty));
        const int x = TILE * tx + (s & 3), y = TILE * ty + ((s >> 2) & 3), z = TILE * tz + (s >> 4);
        uint8_t v = LBM_SOLID;
        if (x < nx && y < ny && z < nz) v = nt[x + (int64_t)nx * (y + (int64_t)ny * z)];
        ntype[k * SLOTS + s] = v;
        const uint32_t solid_bits = __ballot_sync(0xffffffffu, v == LBM_SOLID);
        const uint32_t bc_bits = __ballot_sync(0xffffffffu, v == LBM_INLET || v == LBM_OUTLET);
        if (lane == 0) {
            s_solid[warp] = solid_bits;
            s_bc[warp] = bc_bits;
            atomicAdd(n_nonsolid, (unsigned long long)(32 - __popc(solid_bits)));
        }
        if (s < NBR) {
            const int d[3] = {s % 3 - 1, (s / 3) % 3 - 1, s / 9 - 1};
            int c[3] = {tx + d[0], ty + d[1], tz + d[2]};
            const int T[3] = {Tx, Ty, Tz};
            bool inside = true;
            for (int a = 0; a < 3; a++) {
                if (c[a] < 0 || c[a] >= T[a]) {
                    if (periodic & (1u << a)) c[a] = (c[a] + T[a]) % T[a];
                    else inside = false;
                }
            }
            nbr[k * NBR_STRIDE + s] = inside ? tile_map[c[0] + (int64_t)Tx * (c[1] + (int64_t)Ty * c[2])] : -1;
        } else if (s == NBR) {
            nbr[k * NBR_STRIDE + s] = -1;
        }
        __syncthreads();
        if (s == 0) {
            smask[k] = (uint64_t)s_solid[0] | ((uint64_t)s_solid[1] << 32);
            tflags[k] = (s_bc[0] | s_bc[1]) ? FLAG_HAS_BC : 0;
        }
        __syncthreads();
    }
}

cudaError_t launch_tile_meta(lbm_ctx* c, const uint8_t* nt) {
    unsigned long long* d_cnt = reinterpret_cast<unsigned long long*>(c->d_out);
    cudaError_t e = cudaMemsetAsync(d_cnt, 0, sizeof(unsigned long long), c->stream);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::min<int64_t>(c->n_tiles, 1 << 20);
    if (blocks > 0)
        k_tile_meta<<<(unsigned)blocks, 64, 0, c->stream>>>(nt, c->nx, c->ny, c->nz, c->Tx, c->Ty, c->Tz,
                                                            c->periodic, c->tile_map, c->non_empty,
                                                            c->n_tiles, c->nbr, c->smask, c->tflags,
                                                            c->ntype, d_cnt);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Per-node gather words: for every non-solid node, which of the 18 moving directions
// bounce back (their source x - c_i is solid, in a dropped tile or outside a
// non-periodic box), plus the node type. Built once; the step kernel then needs no
// neighbour masks.
__global__ void __launch_bounds__(64) k_node_words(const int32_t* __restrict__ nbr, const uint64_t* __restrict__ smask,
                                                   const uint8_t* __restrict__ ntype, int64_t n_tiles,
                                                   uint32_t* __restrict__ nword) {
    const int s = threadIdx.x;
    const int x = s & 3, y = (s >> 2) & 3, z = s >> 4;
    for (int64_t k = blockIdx.x; k < n_tiles; k += gridDim.x) {
        const uint32_t type = ntype[k * SLOTS + s];
        uint32_t w = 0;
        if (type != LBM_SOLID) {
            w = type << WORD_TYPE_SHIFT;
#pragma unroll
            for (int i = 1; i < Q; i++) {
                const int sx = x - cx(i), sy = y - cy(i), sz = z - cz(i);
                const int nb = 13 + (sx >> 2) + 3 * (sy >> 2) + 9 * (sz >> 2);
                const int ss = (sx & 3) | ((sy & 3) << 2) | ((sz & 3) << 4);
                const int32_t nk = nbr[k * NBR_STRIDE + nb];
                const bool bounce = nk < 0 || ((smask[nk] >> ss) & 1);
                if (bounce) w |= 1u << i;
            }
        }
        nword[k * SLOTS + s] = w;
    }
}

cudaError_t launch_node_words(lbm_ctx* c) {
    const int64_t blocks = std::min<int64_t>(c->n_tiles, 1 << 20);
    if (blocks > 0) k_node_words<<<(unsigned)blocks, 64, 0, c->stream>>>(c->nbr, c->smask, c->ntype, c->n_tiles, c->nword);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Equilibrium initial state f = f^eq(rho0, u0) (Eq. 3) of every non-solid node, in both
// copies. The 19 values are the same everywhere: a CTA forms them once in FP64 and keeps them
// stored in shared memory. (Formed per node they were all FP64-pipe time: 364 us on a 128^3
// pack in FP32.)
template <int DT>
__global__ void k_init(typename Store<DT>::T* __restrict__ f0, typename Store<DT>::T* __restrict__ f1,
                       const uint64_t* __restrict__ smask, const int32_t* __restrict__ tlane, int64_t n_tiles,
                       double rho0, double ux, double uy, double uz, int eq) {
    using T = typename Store<DT>::T;
    __shared__ T value[Q];
    if (threadIdx.x == 0) {
        const double uu = ux * ux + uy * uy + uz * uz;
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const double cu = cx(i) * ux + cy(i) * uy + cz(i) * uz;
            // Eq. 3, or Eq. 4 for the incompressible model
            const double fe = eq == LBM_EQ_INCOMPR ? wgt(i) * (rho0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
                                                   : wgt(i) * rho0 * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu);
            value[i] = from_f64<DT>(fe, i);
        }
    }
    __syncthreads();
    const int64_t n = n_tiles * SLOTS;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx >> 6;
        const int s = (int)(idx & 63);
        const uint64_t sm = smask[k];
        if ((sm >> s) & 1) continue;   // solid slots have no storage
        const uint32_t P = node_lane((uint32_t)tlane[k], sm, s);
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const T v = value[i];
            f0[data_index(P, i)] = v;
            f1[data_index(P, i)] = v;
        }
    }
}

// The per-lane lists of the step's work groups (fword, fidx), from what the host decided
// per tile while forming the groups: the non-solid nodes of tile k take lanes lane0[k],
// lane0[k] + 1, ... in slot order, and lt[k] is the tile's index within its group. One CTA
// of 64 threads per tile, one thread per slot; a slot's rank is the popcount of the
// tile's non-solid mask below it.
__global__ void k_lane_lists(const uint32_t* __restrict__ nword, const uint64_t* __restrict__ smask,
                             const int32_t* __restrict__ nbr, const int64_t* __restrict__ lane0,
                             const uint8_t* __restrict__ lt, int64_t k0, int64_t k1, uint32_t* __restrict__ fword,
                             uint32_t* __restrict__ fidx, uint4* __restrict__ frank) {
    const int s = threadIdx.x;
    const int x = s & 3, y = (s >> 2) & 3, z = s >> 4;
    const uint64_t below = (1ull << s) - 1ull;   // s < 64
    for (int64_t k = k0 + blockIdx.x; k < k1; k += gridDim.x) {
        const uint64_t sm = smask[k];
        const uint32_t l = lt[k - k0];
        if (!((sm >> s) & 1ull)) {
            const int64_t idx = lane0[k - k0] + __popcll(~sm & below);
            const uint32_t w = nword[k * SLOTS + s];
            fword[idx] = w | (l << WORD_LT_SHIFT) | ((uint32_t)s << WORD_SLOT_SHIFT);
            fidx[idx] = (uint32_t)(k * SLOTS + s);
            uint32_t r[4] = {0u, 0u, 0u, 0u};
            for (int i = 1; i < Q; i++) {
                if ((w >> i) & 1u) continue;   // bounced: no source in another slot
                const int sx = x - cx(i), sy = y - cy(i), sz = z - cz(i);
                const int nb = 13 + (sx >> 2) + 3 * (sy >> 2) + 9 * (sz >> 2);
                const int ss = (sx & 3) | ((sy & 3) << 2) | ((sz & 3) << 4);
                const int32_t nk = nbr[k * NBR_STRIDE + nb];   // >= 0: the link does not bounce
                const uint32_t rank = (uint32_t)__popcll(~smask[nk] & ((1ull << ss) - 1ull));
                r[(i - 1) / 5] |= rank << (6 * ((i - 1) % 5));
            }
            frank[idx] = make_uint4(r[0], r[1], r[2], r[3]);
        }
    }
}

cudaError_t launch_lane_lists(lbm_ctx* c, const int64_t* lane0, const uint8_t* lt) {
    const int64_t n = c->own_k1 - c->own_k0;
    if (n <= 0) return cudaSuccess;
    k_lane_lists<<<(unsigned)std::min<int64_t>(n, 1 << 20), SLOTS, 0, c->stream>>>(
        c->nword, c->smask, c->nbr, lane0, lt, c->own_k0, c->own_k1, c->fword, c->fidx, c->frank);
    return cudaGetLastError();
}

// The step's neighbour records: for each kept tile and each of its 27 neighbourhood
// entries, the index of the neighbour's first non-solid node in data block 0 of a copy
// (zero for a dropped or out-of-box neighbour, and in the padding entry). One thread per
// record.
__global__ void k_node_records(const int32_t* __restrict__ nbr, const int32_t* __restrict__ tlane, int64_t n_tiles,
                               int64_t* __restrict__ nrec) {
    const int64_t n = n_tiles * NBR_STRIDE;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)(idx % NBR_STRIDE);
        const int32_t r = e < NBR ? nbr[idx] : -1;
        nrec[idx] = r >= 0 && r < n_tiles ? data_index((uint32_t)tlane[r], 0) : 0;
    }
}

static unsigned grid_for(int64_t n, int threads) {
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + threads - 1) / threads, 152 * 32));
}

cudaError_t launch_node_records(lbm_ctx* c) {
    if (c->n_tiles <= 0) return cudaSuccess;
    k_node_records<<<grid_for(c->n_tiles * NBR_STRIDE, 256), 256, 0, c->stream>>>(c->nbr, c->tlane, c->n_tiles,
                                                                                 c->nrec);
    return cudaGetLastError();
}

// Import lists and staged offsets of FP16 storage, one CTA per work group, one thread per node.
// A group's imports (pulls whose source lies in another storage group) are numbered direction by
// direction and lane by lane, so that a direction's imports read runs of other groups' blocks; a
// group with more than fit its list sets *too_many.
__global__ void __launch_bounds__(GROUP_LANES) k_imports(const int4* __restrict__ groups, const uint32_t* __restrict__ fword,
                                                         const uint32_t* __restrict__ fidx, const int32_t* __restrict__ nbr,
                                                         const uint64_t* __restrict__ smask,
                                                         const int32_t* __restrict__ tlane, int64_t sg0,
                                                         int* __restrict__ too_many, int2* __restrict__ imports, uint32_t* __restrict__ entries,
                                                         uint32_t* __restrict__ fsrc, uint32_t* __restrict__ fsrc8) {
    __shared__ int warp_n[GROUP_LANES / 32];
    const int64_t g = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int4 h = groups[g];
    const bool on = t < h.w;
    const int64_t n = (int64_t)h.z + t;
    uint32_t w = 0, gi = 0;
    if (on) {
        w = fword[n];
        gi = fidx[n];
    }
    const int64_t k = gi >> 6;
    const int s = (int)(gi & 63u), x = s & 3, y = (s >> 2) & 3, z = s >> 4;
    const uint32_t base = (uint32_t)(sg0 + g);
    uint32_t* list = entries + g * GROUP_MAX_IMPORTS;
    int count = 0;   // imports of the directions so far
    uint32_t off[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int i = 1; i < Q; i++) {
        uint32_t o = (uint32_t)(inv(i) * GROUP_LANES + t) * 2u, P = 0;
        bool import = false;
        if (on && !((w >> i) & 1u)) {
            const int sx = x - cx(i), sy = y - cy(i), sz = z - cz(i);
            const int nb = 13 + (sx >> 2) + 3 * (sy >> 2) + 9 * (sz >> 2);
            const int ss = (sx & 3) | ((sy & 3) << 2) | ((sz & 3) << 4);
            const int32_t r = nbr[k * NBR_STRIDE + nb];   // >= 0: the link does not bounce
            P = node_lane((uint32_t)tlane[r], smask[r], ss);
            import = P / GROUP_LANES != base;
            o = (uint32_t)(i * GROUP_LANES + (P % GROUP_LANES)) * 2u;
        }
        const uint32_t b = __ballot_sync(0xffffffffu, import);
        if (lane == 0) warp_n[warp] = __popc(b);
        __syncthreads();
        int before = count;
        for (int v = 0; v < GROUP_LANES / 32; v++) {
            if (v < warp) before += warp_n[v];
            count += warp_n[v];
        }
        __syncthreads();
        if (import) {
            const int slot = before + __popc(b & ((1u << lane) - 1u));
            const int64_t e = data_index(P, i);
            if (slot < GROUP_MAX_IMPORTS) list[slot] = (uint32_t)(e >> 1);
            o = (uint32_t)(Q * GROUP_LANES * 2 + 4 * slot) + 2u * (uint32_t)(e & 1);
        }
        off[(i - 1) >> 1] |= (i & 1) ? o : o << 16;
    }
    if (count > GROUP_MAX_IMPORTS) {
        if (t == 0) *too_many = 1;
        return;
    }
    if (t == 0) imports[g] = make_int2((int)(g * GROUP_MAX_IMPORTS), count);
    if (t < (4 - (count & 3)) % 4) list[count + t] = 0;   // padding: word 0 of the copy
    if (on) {
#pragma unroll
        for (int j = 0; j < 8; j++) fsrc[n * 8 + j] = off[j];
        fsrc8[n] = off[8];
    }
}

cudaError_t launch_imports(lbm_ctx* c, int* too_many) {
    k_imports<<<(unsigned)c->n_groups, GROUP_LANES, 0, c->stream>>>(c->groups, c->fword, c->fidx, c->nbr, c->smask, c->tlane,
                                                                   c->p.sg0, too_many, c->imports, c->entries,
                                                                   reinterpret_cast<uint32_t*>(c->fsrc), c->fsrc8);
    return cudaGetLastError();
}

cudaError_t launch_init(lbm_ctx* c, double rho0, const double u0[3]) {
    const unsigned g = std::min(grid_for(c->n_tiles * SLOTS, 256), 152u * 8u);
    switch (c->dtype) {
        case LBM_F64:
            k_init<LBM_F64><<<g, 256, 0, c->stream>>>((double*)c->f[0], (double*)c->f[1], c->smask, c->tlane,
                                                      c->n_tiles, rho0, u0[0], u0[1], u0[2], c->p.eq);
            break;
        case LBM_F32:
            k_init<LBM_F32><<<g, 256, 0, c->stream>>>((float*)c->f[0], (float*)c->f[1], c->smask, c->tlane,
                                                      c->n_tiles, rho0, u0[0], u0[1], u0[2], c->p.eq);
            break;
        default:
            k_init<LBM_F16S><<<g, 256, 0, c->stream>>>((__half*)c->f[0], (__half*)c->f[1], c->smask, c->tlane,
                                                       c->n_tiles, rho0, u0[0], u0[1], u0[2], c->p.eq);
    }
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Moments of the stored populations: the FP64 invariants (k_reduce) and the macroscopic
// export (k_macro). Both walk the work groups, one thread per non-solid node: the loads of
// a direction are one contiguous run of a data block and no lane idles on a solid slot.
// GB300 runs FP64, and every conversion from or to it, on 2 lanes per SM, so the moments are
// formed with integer (FP64 storage) or FP32 (the other formats) instructions, and FP64 is
// left for what needs it. Measured against one thread per tile slot with FP64 moments and
// divisions: k_reduce<F64> 103 -> 45 us on a 160^3 pack (1.4 M nodes, 219 MB: 4.9 TB/s);
// reduction and FP64 fields together 322 -> 159 us there; the FP32 fields of a 256^3 pack
// (5.9 M nodes) 640 us less. k_macro<F32, float> issues 65 % of cycles (the TwoSums).
constexpr int MOM_THREADS = GROUP_LANES;   // one thread per lane of a work group
static_assert(GROUP_MAX_NODES == MOM_THREADS && GROUP_MAX_NODES_F64 == MOM_THREADS, "one thread per lane");

// FP64 storage: exact moments in 64-bit fixed point (2^-58). The integer conversion of a
// population in [2^-6, 16) is exact; a node with any other value converts all 19 again with
// the general routine (round to nearest), reading them once more in a rolled loop, so that
// this rare path holds no registers of the common one. That routine maps NaN and Inf to
// finite integers, so a non-finite population is found on its exponent bits and makes every
// moment of the node NaN (what the mass watchdog of lbm_reduce looks for).
struct FixMoments {
    int64_t r, j[3];
    bool nonfinite;
};
__device__ __forceinline__ FixMoments fix_node_moments(const double* __restrict__ f) {
    FixMoments m;
    m.nonfinite = false;
    bool bad = false;
    int64_t q[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) q[i] = fix_from_double_fast(f[i * GROUP_LANES], bad);
    fix_moments(q, m.r, m.j[0], m.j[1], m.j[2]);
    if (bad) {
        uint64_t r = 0, j[3] = {0, 0, 0};   // unsigned: values of 16 and more may wrap
#pragma unroll 1
        for (int i = 0; i < Q; i++) {
            const double v = f[i * GROUP_LANES];
            m.nonfinite |= (~bits_of(v) & 0x7ff0000000000000ull) == 0;
            const uint64_t w = (uint64_t)fix_from_double(v);
            r += w;
            j[0] += (uint64_t)(int64_t)cx(i) * w;
            j[1] += (uint64_t)(int64_t)cy(i) * w;
            j[2] += (uint64_t)(int64_t)cz(i) * w;
        }
        m.r = (int64_t)r;
        for (int a = 0; a < 3; a++) m.j[a] = (int64_t)j[a];
    }
    return m;
}
// FP32 and FP16 storage: the h values are FP32 numbers; each moment (rho - 1, j) is summed
// with Knuth's TwoSum into a running sum and the sum of its rounding errors, so a moment is
// the pair s + e (relative error about 2^-48).
struct PairMoments {
    float s[4], e[4];
    __device__ __forceinline__ void add(int c, float v) {
        const dfl t = two_sum(s[c], v);
        s[c] = t.h;
        e[c] = __fadd_rn(e[c], t.l);
    }
};
template <int DT>
__device__ __forceinline__ void add_node_moments(const typename Store<DT>::T* __restrict__ f, PairMoments& m) {
    float h[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) h[i] = to_arith<DT>(f[i * GROUP_LANES], i);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        m.add(0, h[i]);
        if (cx(i)) m.add(1, cx(i) > 0 ? h[i] : -h[i]);
        if (cy(i)) m.add(2, cy(i) > 0 ? h[i] : -h[i]);
        if (cz(i)) m.add(3, cz(i) > 0 ? h[i] : -h[i]);
    }
}

// FP64 mass and momentum. FP64 storage adds the nodes' fixed-point moments in 128-bit integers,
// exactly, over a warp. The other formats add each node's pair to a triple of FP32 numbers, which
// keeps the rounding errors of both parts, and that to FP64 sums every RED_FLUSH nodes. (A pair
// carried over four nodes lost the last bits of small populations beside large ones: the
// momentum of FP32 populations from 1e-9 to 5e-3 was 30 times further off. Pairs added in FP64
// node by node: 254 us a call on the 256^3 pack in FP32; 152 us so, as with the carried pair.) Then
// a warp shuffle tree, one partial per block and a fixed-order single-block pass. No atomics, so
// the result depends only on the launch shape, which is fixed per context. What is the same at
// every node (half a uniform force, and the 1 of rho = 1 + sum h) enters the final sum once:
// subtracted per node or thread its rounding is the same everywhere and adds up. The half force
// of a field is summed per warp.
constexpr int RED_THREADS = MOM_THREADS;
constexpr int RED_FLUSH = 16;
struct TripleMoments {
    float s[4], e[4], ee[4];
    __device__ __forceinline__ void add(const PairMoments& m) {
        for (int c = 0; c < 4; c++) {
            const dfl t = two_sum(s[c], m.s[c]), u = two_sum(e[c], t.l), v = two_sum(u.h, m.e[c]);
            s[c] = t.h;
            e[c] = v.h;
            ee[c] = __fadd_rn(ee[c], __fadd_rn(u.l, v.l));
        }
    }
    // far from the largest FP32 number, which a sum of RED_FLUSH moments then cannot reach
    __device__ __forceinline__ bool moderate() const {
        return fmaxf(fmaxf(fabsf(s[0]), fabsf(s[1])), fmaxf(fabsf(s[2]), fabsf(s[3]))) < 0x1p100f;
    }
};

// resident CTAs per SM, and the grid: the 128-bit sums of FP64 storage need the registers
template <int DT> constexpr int red_ctas() { return DT == LBM_F64 ? 3 : 4; }

template <int DT>
__global__ void __launch_bounds__(RED_THREADS, red_ctas<DT>()) k_reduce(const typename Store<DT>::T* __restrict__ f,
                                                        const int4* __restrict__ groups,
                                                        const typename Store<DT>::R* __restrict__ gfield_c,
                                                        int64_t n_groups, StepParams p,
                                                        double* __restrict__ partials) {
    __shared__ double sh[RED_THREADS / 32][4], sh_fx[RED_THREADS / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    double fx = 0.0;
    if constexpr (DT == LBM_F64) {
        __int128 sum[4] = {0, 0, 0, 0};
        bool nonfinite = false;
        for (int64_t g = blockIdx.x; g < n_groups; g += gridDim.x) {
            const int4 h = groups[g];
            if (t >= h.w) continue;
            const FixMoments m = fix_node_moments(f + (p.sg0 + g) * (Q * GROUP_LANES) + t);
            sum[0] += m.r;
            for (int a = 0; a < 3; a++) sum[1 + a] += m.j[a];
            nonfinite |= m.nonfinite;
            if (gfield_c) fx += gfield_c[h.z + t];
        }
        nonfinite = __any_sync(0xffffffffu, nonfinite);
#pragma unroll
        for (int c = 0; c < 4; c++)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const uint64_t lo = __shfl_down_sync(0xffffffffu, (uint64_t)sum[c], o);
                const uint64_t hi = __shfl_down_sync(0xffffffffu, (uint64_t)(sum[c] >> 64), o);
                sum[c] += (__int128)(((unsigned __int128)hi << 64) | lo);
            }
        for (int c = 0; c < 4 && lane == 0; c++) {
            // of the magnitude, so that a small negative sum has no large low word
            const bool neg = sum[c] < 0;
            const unsigned __int128 a = neg ? -(unsigned __int128)sum[c] : (unsigned __int128)sum[c];
            const double hi = __ull2double_rn((uint64_t)(a >> 64)), lo = __ull2double_rn((uint64_t)a);
            const double v = __fma_rn(hi, 18446744073709551616.0, lo) * (1.0 / (double)(1ull << FIX_SHIFT));
            sh[warp][c] = nonfinite ? __longlong_as_double(0x7ff8000000000000ll) : neg ? -v : v;
        }
    } else {
        TripleMoments m = {};
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        int held = 0;
        auto flush = [&]() {
            for (int c = 0; c < 4; c++) {
                double e = (double)m.e[c];
                if (m.ee[c] != 0.f) e += (double)m.ee[c];   // 0 for a single node: 8 FP64 operations less
                acc[c] += (double)m.s[c] + e;
            }
            m = {};
            held = 0;
        };
        for (int64_t g = blockIdx.x; g < n_groups; g += gridDim.x) {
            const int4 h = groups[g];
            if (t >= h.w) continue;
            PairMoments node = {};
            add_node_moments<DT>(f + (p.sg0 + g) * (Q * GROUP_LANES) + t, node);
            m.add(node);
            if (++held == RED_FLUSH || !m.moderate()) flush();
            if (gfield_c) fx += (double)gfield_c[h.z + t];
        }
        if (held) flush();
#pragma unroll
        for (int c = 0; c < 4; c++) {
            double v = acc[c];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) sh[warp][c] = v;
        }
    }
    if (gfield_c) {
        for (int o = 16; o > 0; o >>= 1) fx += __shfl_down_sync(0xffffffffu, fx, o);
        if (lane == 0) sh_fx[warp] = fx;
    }
    __syncthreads();
    if (t < 4) {
        double v = 0.0;
        for (int w = 0; w < RED_THREADS / 32; w++) v += gfield_c && t == 1 ? sh[w][t] - 0.5 * sh_fx[w] : sh[w][t];
        partials[blockIdx.x * 4 + t] = v;
    }
}

// a + b - fl(a + b), exactly (two_sum in FP64)
__device__ __forceinline__ double sum_error(double a, double b) {
    const double s = __dadd_rn(a, b), bb = __dadd_rn(s, -a);
    return __dadd_rn(__dadd_rn(a, __dadd_rn(bb, -s)), __dadd_rn(b, -bb));
}

// Fixed-order sum of the blocks' partials: 64 threads per component add every 64th partial, then
// a shuffle tree over the eight of a warp and one over the warps, which keeps the rounding errors,
// as does the addition of n_nodes times `each`, the part that every node has alike. (With plain
// additions, eight in a row at the end, the mass was off by 1.0 half units in the last place, rms.)
struct NodeConst {
    double each[4];
};
__global__ void __launch_bounds__(RED_THREADS) k_reduce_final(const double* __restrict__ partials, int nb, double n_nodes,
                                                              NodeConst k, double* __restrict__ out) {
    __shared__ double sh[RED_THREADS / 32][4];
    const int c = threadIdx.x & 3;
    double v = 0.0;
    for (int b = threadIdx.x >> 2; b < nb; b += RED_THREADS / 4) v += partials[b * 4 + c];
#pragma unroll
    for (int o = 16; o >= 4; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) < 4) sh[threadIdx.x >> 5][c] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        // the sums first, then their errors, which depend on the sums alone
        double s = sh[threadIdx.x >> 2][c], a[3], b[3];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            a[k] = s;
            b[k] = __shfl_down_sync(0xffffffffu, s, 16 >> k);
            s = __dadd_rn(a[k], b[k]);
        }
        double e = sum_error(a[0], b[0]);
        e += __shfl_down_sync(0xffffffffu, e, 8);
        e += sum_error(a[1], b[1]);
        e += __shfl_down_sync(0xffffffffu, e, 4);
        e += sum_error(a[2], b[2]);
        if (threadIdx.x < 4) {
            const double each = c == 0 ? k.each[0] : c == 1 ? k.each[1] : c == 2 ? k.each[2] : k.each[3];
            const double all = __dmul_rn(n_nodes, each);
            e += __fma_rn(n_nodes, each, -all);
            out[c] = __dadd_rn(s, all) + (e + sum_error(s, all));
        }
    }
}
static_assert(RED_THREADS / 32 == 8, "the last tree is over eight warps");

int reduce_blocks(int64_t n_tiles) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((n_tiles * SLOTS + RED_THREADS - 1) / RED_THREADS, 152 * 4));
}

// The per-node force in group order, if one is set.
template <int DT> static const typename Store<DT>::R* force_c(const lbm_ctx* c) {
    return c->gfield ? static_cast<const typename Store<DT>::R*>(c->gfield_c) : nullptr;
}

template <int DT> static int reduce_dt(lbm_ctx* c) {
    const int64_t fits = std::min<int64_t>(c->n_partials, 152 * red_ctas<DT>());
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(fits, c->n_groups));
    k_reduce<DT><<<nb, RED_THREADS, 0, c->stream>>>(static_cast<const typename Store<DT>::T*>(c->f[c->cur]), c->groups,
                                                    force_c<DT>(c), c->n_groups, c->p, c->partials);
    return nb;
}

cudaError_t launch_reduce(lbm_ctx* c, double* d_out) {
    const int nb = c->dtype == LBM_F64 ? reduce_dt<LBM_F64>(c) : c->dtype == LBM_F32 ? reduce_dt<LBM_F32>(c)
                                                                                     : reduce_dt<LBM_F16S>(c);
    const NodeConst k = {{c->dtype == LBM_F64 ? 0.0 : 1.0, c->gfield ? 0.0 : -0.5 * c->p.g[0], -0.5 * c->p.g[1],
                          -0.5 * c->p.g[2]}};
    k_reduce_final<<<1, RED_THREADS, 0, c->stream>>>(c->partials, nb, (double)c->n_own_nonsolid, k, d_out);
    return cudaGetLastError();
}

// Macroscopic export from the stored post-collision populations: rho = sum f*,
// u = (sum c f* - F/2)/rho (Eq. 5; Eq. 6 without the division for the incompressible
// model), into dense arrays (already zeroed by the caller).
//
// x / r from ir, 1/r to 2^-46 or better: one Newton correction of x ir, which rounds like
// the division (to half an ulp and a little) in three FP64 operations, where a division takes
// about ten and a reciprocal as many.
__device__ __forceinline__ double div_by(double x, double r, double ir) {
    const double q = __dmul_rn(x, ir);
    return __fma_rn(__fma_rn(-q, r, x), ir, q);
}
// The same in pairs for an FP32 result.
__device__ __forceinline__ float pair_value(dfl x) { return __fadd_rn(x.h, x.l); }

// What one node exports, from its exact moments (double) or from pairs (float).
template <typename O> struct NodeFields {
    O rho, u[3];
};
__device__ __forceinline__ NodeFields<double> fields_of(const double m[4], const double half[3], bool inc) {
    NodeFields<double> o;
    o.rho = m[0];
    for (int a = 0; a < 3; a++) o.u[a] = inc ? m[1 + a] - half[a] : (m[1 + a] - half[a]) / m[0];
    return o;
}
// FP64 results of FP64 storage for a density in [5/8, 7/4): 1/rho in pairs, widened with integer
// instructions, so that FP64 is left with the force and three operations per component.
__device__ __forceinline__ NodeFields<double> fields_of(const FixMoments& m, const double half[3], bool inc, bool& ok) {
    NodeFields<double> o;
    ok = !m.nonfinite && m.r >= (5ll << (FIX_SHIFT - 3)) && m.r < (7ll << (FIX_SHIFT - 2));
    o.rho = fix_to_double(m.r);
    const double ir = df_to_double_pos(df_recip(df_from_fix(m.r)));
    for (int a = 0; a < 3; a++) {
        double x = fix_to_double(m.j[a]);
        if (half[a] != 0.0) x -= half[a];
        o.u[a] = inc ? x : div_by(x, o.rho, ir);
    }
    return o;
}
// Valid for a density in [2^-20, 2^20]; `ok` says whether the result can be used.
__device__ __forceinline__ NodeFields<float> fields_of(const dfl r, const dfl j[3], const dfl half[3], bool inc, bool& ok) {
    NodeFields<float> o;
    o.rho = pair_value(r);
    ok = o.rho >= 0x1p-20f && o.rho <= 0x1p20f;
    const dfl ir = df_recip(r);
    for (int a = 0; a < 3; a++) {
        const dfl x = df_sub(j[a], half[a]);
        o.u[a] = pair_value(inc ? x : df_mul(x, ir));
        ok = ok && fabsf(o.u[a]) <= 0x1p20f;   // false for NaN
    }
    return o;
}

template <int DT, typename O>
__global__ void __launch_bounds__(MOM_THREADS, 4) k_macro(const typename Store<DT>::T* __restrict__ f,
                                                       const int4* __restrict__ groups,
                                                       const uint32_t* __restrict__ fidx,
                                                       const uint32_t* __restrict__ non_empty,
                                                       const typename Store<DT>::R* __restrict__ gfield_c,
                                                       int64_t n_groups, int nx, int ny, int nz, int Tx, int Ty,
                                                       StepParams p, O* __restrict__ rho, O* __restrict__ u) {
    const int64_t N = (int64_t)nx * ny * nz;
    const int t = threadIdx.x;
    const bool inc = p.eq == LBM_EQ_INCOMPR;
    const double hg[3] = {0.5 * p.g[0], 0.5 * p.g[1], 0.5 * p.g[2]};
    for (int64_t g = blockIdx.x; g < n_groups; g += gridDim.x) {
        const int4 hd = groups[g];
        if (t >= hd.w) continue;
        const typename Store<DT>::T* src = f + (p.sg0 + g) * (Q * GROUP_LANES) + t;
        const uint32_t gi = fidx[hd.z + t];
        NodeFields<O> o;
        FixMoments fm;
        PairMoments pm = {};
        if constexpr (DT == LBM_F64) fm = fix_node_moments(src);
        else add_node_moments<DT>(src, pm);
        // the plain FP64 form: FP64 results of the other formats, and nodes whose density lies
        // outside the ranges of the forms below
        auto wide = [&]() {
            double m[4];
            if constexpr (DT == LBM_F64) {
                const double nan = __longlong_as_double(0x7ff8000000000000ll);
                m[0] = fm.nonfinite ? nan : fix_to_double(fm.r);
                for (int a = 0; a < 3; a++) m[1 + a] = fm.nonfinite ? nan : fix_to_double(fm.j[a]);
            } else {
                for (int c = 0; c < 4; c++) m[c] = (double)pm.s[c] + (double)pm.e[c];
                m[0] += 1.0;
            }
            const double half[3] = {0.5 * (gfield_c ? (double)gfield_c[hd.z + t] : p.g[0]), 0.5 * p.g[1], 0.5 * p.g[2]};
            const NodeFields<double> w = fields_of(m, half, inc);
            o.rho = (O)w.rho;
            for (int a = 0; a < 3; a++) o.u[a] = (O)w.u[a];
        };
        if constexpr (sizeof(O) == 8) {
            if constexpr (DT == LBM_F64) {
                bool ok;
                const double half[3] = {gfield_c ? 0.5 * gfield_c[hd.z + t] : hg[0], hg[1], hg[2]};
                o = fields_of(fm, half, inc, ok);
                if (!ok) wide();
            } else {
                wide();
            }
        } else {
            dfl r, j[3], half[3] = {p.dfc.Fx, {}, {}};
            bool pair_force = true;
            if constexpr (DT == LBM_F64) {
                if (gfield_c) {
                    const double Fx = gfield_c[hd.z + t];
                    half[0] = df_from_double(Fx);
                    // the range of that conversion: [2^-60, 2), or 0
                    const uint64_t e = bits_of(Fx) << 1;
                    pair_force = e == 0 || (uint32_t)(e >> 53) - 963u <= 60u;
                }
            } else if (gfield_c) {
                half[0] = df_make(gfield_c[hd.z + t], 0.f);
            }
            half[0] = df_scale2(half[0], 0.5f);
            half[1] = df_scale2(p.dfc.Fy, 0.5f);
            half[2] = df_scale2(p.dfc.Fz, 0.5f);
            bool ok;
            if constexpr (DT == LBM_F64) {
                r = df_from_fix(fm.r);
                for (int a = 0; a < 3; a++) j[a] = df_from_fix(fm.j[a]);
                o = fields_of(r, j, half, inc, ok);
                ok = ok && !fm.nonfinite && pair_force;
            } else {
                r = df_add_dom(df_make(1.0f, 0.0f), df_make(pm.s[0], pm.e[0]));
                for (int a = 0; a < 3; a++) j[a] = df_make(pm.s[1 + a], pm.e[1 + a]);
                o = fields_of(r, j, half, inc, ok);
                ok = ok && fabsf(pm.s[0]) <= 1.0f;   // 1 dominates
            }
            if (!ok) wide();
        }
        const uint32_t tile = non_empty[gi >> 6];
        const int s = (int)(gi & 63u);
        const uint32_t row = tile / (uint32_t)Tx;
        const int x = TILE * (int)(tile - row * (uint32_t)Tx) + (s & 3);
        const int y = TILE * (int)(row % (uint32_t)Ty) + ((s >> 2) & 3);
        const int z = TILE * (int)(row / (uint32_t)Ty) + (s >> 4);
        const int64_t node = x + (int64_t)nx * (y + (int64_t)ny * z);
        rho[node] = o.rho;
        for (int a = 0; a < 3; a++) u[a * N + node] = o.u[a];
    }
}

template <int DT, typename O> static void macro_dt(lbm_ctx* c, void* rho, void* u) {
    const unsigned g = (unsigned)std::min<int64_t>(c->n_groups, 152 * 32);
    k_macro<DT, O><<<g, MOM_THREADS, 0, c->stream>>>(static_cast<const typename Store<DT>::T*>(c->f[c->cur]), c->groups,
                                                     c->fidx, c->non_empty, force_c<DT>(c), c->n_groups, c->nx, c->ny,
                                                     c->nz, c->Tx, c->Ty, c->p, static_cast<O*>(rho),
                                                     static_cast<O*>(u));
}

template <int DT> static void macro_out(lbm_ctx* c, void* rho, void* u, int out_f64) {
    if (out_f64) macro_dt<DT, double>(c, rho, u);
    else macro_dt<DT, float>(c, rho, u);
}

cudaError_t launch_macroscopic(lbm_ctx* c, void* rho, void* u, int out_f64) {
    if (c->n_groups == 0) return cudaSuccess;
    if (c->dtype == LBM_F64) macro_out<LBM_F64>(c, rho, u, out_f64);
    else if (c->dtype == LBM_F32) macro_out<LBM_F32>(c, rho, u, out_f64);
    else macro_out<LBM_F16S>(c, rho, u, out_f64);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Box export: out[i][bz][by][bx] in FP64; NaN for solid, dropped or outside nodes.
template <int DT>
__global__ void k_get_box(const typename Store<DT>::T* __restrict__ f, const int32_t* __restrict__ tile_map,
                          const uint64_t* __restrict__ smask, const int32_t* __restrict__ tlane, int nx, int ny, int nz, int Tx, int Ty,
                          unsigned periodic, int x0, int y0, int z0, int bx, int by, int bz,
                          double* __restrict__ out) {
    const int64_t B = (int64_t)bx * by * bz;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < B;
         b += (int64_t)gridDim.x * blockDim.x) {
        int p[3] = {x0 + (int)(b % bx), y0 + (int)((b / bx) % by), z0 + (int)(b / ((int64_t)bx * by))};
        const int n[3] = {nx, ny, nz};
        bool inside = true;
        for (int a = 0; a < 3; a++) {
            if (p[a] < 0 || p[a] >= n[a]) {
                if (periodic & (1u << a)) p[a] = ((p[a] % n[a]) + n[a]) % n[a];
                else inside = false;
            }
        }
        int64_t k = -1;
        uint32_t P = 0;
        if (inside) {
            k = tile_map[p[0] / TILE + (int64_t)Tx * (p[1] / TILE + (int64_t)Ty * (p[2] / TILE))];
            const int s = (p[0] & 3) + 4 * (p[1] & 3) + 16 * (p[2] & 3);
            if (k >= 0 && ((smask[k] >> s) & 1)) k = -1;
            if (k >= 0) P = node_lane((uint32_t)tlane[k], smask[k], s);
        }
#pragma unroll
        for (int i = 0; i < Q; i++)
            out[i * B + b] = k >= 0 ? to_f64<DT>(f[data_index(P, i)], i) : __longlong_as_double(0x7ff8000000000000ll);
    }
}

cudaError_t launch_get_box(lbm_ctx* c, int x0, int y0, int z0, int bx, int by, int bz, double* d_out) {
    const unsigned g = grid_for((int64_t)bx * by * bz, 256);
    const void* A = c->f[c->cur];
#define LBM_BOX(DT, TT)                                                                                   \
    k_get_box<DT><<<g, 256, 0, c->stream>>>((const TT*)A, c->tile_map, c->smask, c->tlane, c->nx, c->ny, c->nz, c->Tx, \
                                            c->Ty, c->periodic, x0, y0, z0, bx, by, bz, d_out)
    if (c->dtype == LBM_F64) LBM_BOX(LBM_F64, double);
    else if (c->dtype == LBM_F32) LBM_BOX(LBM_F32, float);
    else LBM_BOX(LBM_F16S, __half);
#undef LBM_BOX
    return cudaGetLastError();
}

// Dense FP64 import of the non-solid nodes into both copies.
template <int DT>
__global__ void k_set_dense(typename Store<DT>::T* __restrict__ f0, typename Store<DT>::T* __restrict__ f1,
                            const double* __restrict__ dense, const uint64_t* __restrict__ smask,
                            const int32_t* __restrict__ tlane, const uint32_t* __restrict__ non_empty,
                            int64_t n_tiles, int nx, int ny, int nz, int Tx, int Ty) {
    using T = typename Store<DT>::T;
    const int64_t n = n_tiles * SLOTS;
    const int64_t N = (int64_t)nx * ny * nz;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx >> 6;
        const int s = (int)(idx & 63);
        const uint64_t sm = smask[k];
        if ((sm >> s) & 1) continue;   // solid slots have no storage
        const uint32_t P = node_lane((uint32_t)tlane[k], sm, s);
        const uint32_t t = non_empty[k];
        const int x = TILE * (int)(t % (uint32_t)Tx) + (s & 3);
        const int y = TILE * (int)((t / (uint32_t)Tx) % (uint32_t)Ty) + ((s >> 2) & 3);
        const int z = TILE * (int)(t / ((uint32_t)Tx * (uint32_t)Ty)) + (s >> 4);
        const int64_t node = x + (int64_t)nx * (y + (int64_t)ny * z);
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const T v = from_f64<DT>(dense[i * N + node], i);
            f0[data_index(P, i)] = v;
            f1[data_index(P, i)] = v;
        }
    }
}

cudaError_t launch_set_dense(lbm_ctx* c, const double* d_dense) {
    const unsigned g = grid_for(c->n_tiles * SLOTS, 256);
#define LBM_SET(DT, TT)                                                                                   \
    k_set_dense<DT><<<g, 256, 0, c->stream>>>((TT*)c->f[c->cur], (TT*)c->f[1 - c->cur], d_dense, c->smask, \
                                              c->tlane, c->non_empty, c->n_tiles, c->nx, c->ny, c->nz, c->Tx, c->Ty)
    if (c->dtype == LBM_F64) LBM_SET(LBM_F64, double);
    else if (c->dtype == LBM_F32) LBM_SET(LBM_F32, float);
    else LBM_SET(LBM_F16S, __half);
#undef LBM_SET
    return cudaGetLastError();
}

// Dense per-node x force -> tile-major copy in the arithmetic precision.
template <typename G>
__global__ void k_gfield(G* __restrict__ gt, const double* __restrict__ dense, const uint32_t* __restrict__ non_empty,
                         int64_t n_tiles, int nx, int ny, int nz, int Tx, int Ty) {
    const int64_t n = n_tiles * SLOTS;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx >> 6;
        const int s = (int)(idx & 63);
        const uint32_t t = non_empty[k];
        const int x = TILE * (int)(t % (uint32_t)Tx) + (s & 3);
        const int y = TILE * (int)((t / (uint32_t)Tx) % (uint32_t)Ty) + ((s >> 2) & 3);
        const int z = TILE * (int)(t / ((uint32_t)Tx * (uint32_t)Ty)) + (s >> 4);
        const bool in = x < nx && y < ny && z < nz;
        gt[idx] = in ? (G)dense[x + (int64_t)nx * (y + (int64_t)ny * z)] : (G)0;
    }
}

// Tile-major force -> the compact per-fluid-node copy read by the step kernel.
template <typename G>
__global__ void k_gfield_compact(G* __restrict__ gc, const G* __restrict__ gt, const uint32_t* __restrict__ fidx,
                                 int64_t n_fluid) {
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < n_fluid; n += (int64_t)gridDim.x * blockDim.x)
        gc[n] = gt[fidx[n]];
}

cudaError_t launch_gfield_compact(lbm_ctx* c) {
    const unsigned g = grid_for(c->n_own_nonsolid, 256);
    if (c->dtype == LBM_F64)
        k_gfield_compact<double><<<g, 256, 0, c->stream>>>((double*)c->gfield_c, (const double*)c->gfield, c->fidx,
                                                           c->n_own_nonsolid);
    else
        k_gfield_compact<float><<<g, 256, 0, c->stream>>>((float*)c->gfield_c, (const float*)c->gfield, c->fidx,
                                                          c->n_own_nonsolid);
    return cudaGetLastError();
}

// Mark (or clear, face < 0) the compact words of the nodes on a box face: x = 0 (face 0),
// x = nx - 1 (1), y = 0 (2), y = ny - 1 (3), z = 0 (4), z = nz - 1 (5).
__global__ void k_mark_lid(uint32_t* __restrict__ fword, const uint32_t* __restrict__ fidx,
                           const uint32_t* __restrict__ non_empty, int64_t n_nodes, int Tx, int Ty, int nx, int ny,
                           int nz, int face) {
    for (int64_t n = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; n < n_nodes;
         n += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t gi = fidx[n];
        const uint32_t t = non_empty[gi >> 6];
        const int s = (int)(gi & 63u);
        const int p[3] = {TILE * (int)(t % (uint32_t)Tx) + (s & 3),
                          TILE * (int)((t / (uint32_t)Tx) % (uint32_t)Ty) + ((s >> 2) & 3),
                          TILE * (int)(t / ((uint32_t)Tx * (uint32_t)Ty)) + (s >> 4)};
        const int dims[3] = {nx, ny, nz};
        bool on = false;
        if (face >= 0) {
            const int a = face >> 1;
            on = (face & 1) ? p[a] == dims[a] - 1 : p[a] == 0;
        }
        const uint32_t w = fword[n] & ~(1u << WORD_LID_BIT);
        fword[n] = on ? (w | (1u << WORD_LID_BIT)) : w;
    }
}

cudaError_t launch_mark_lid(lbm_ctx* c, int face) {
    if (c->n_own_nonsolid == 0) return cudaSuccess;
    k_mark_lid<<<grid_for(c->n_own_nonsolid, 256), 256, 0, c->stream>>>(c->fword, c->fidx, c->non_empty,
                                                                       c->n_own_nonsolid,
                                                                   c->Tx, c->Ty, c->nx, c->ny, c->nz, face);
    return cudaGetLastError();
}

cudaError_t launch_gfield(lbm_ctx* c, const double* d_dense) {
    const unsigned g = grid_for(c->n_tiles * SLOTS, 256);
    if (c->dtype == LBM_F64)
        k_gfield<double><<<g, 256, 0, c->stream>>>((double*)c->gfield, d_dense, c->non_empty, c->n_tiles, c->nx,
                                                   c->ny, c->nz, c->Tx, c->Ty);
    else
        k_gfield<float><<<g, 256, 0, c->stream>>>((float*)c->gfield, d_dense, c->non_empty, c->n_tiles, c->nx,
                                                  c->ny, c->nz, c->Tx, c->Ty);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Halo of a slab context (lbm_create_slab): the populations that cross the cut between
// two slabs. A node of the lowest own plane pulls from the plane below through the five
// directions with c_z = +1, one of the highest own plane from the plane above through
// the five with c_z = -1. Pack copies the own boundary plane's values of the directions
// its neighbour reads (side 0: the lowest plane, for the slab below, c_z = -1; side 1:
// the highest, for the slab above, c_z = +1) from the current copy into buf, laid out
// [direction][tile][64] with NaN in the solid slots; unpack copies the non-solid slots of
// buf into the ghost plane on that side (side 0: c_z = +1, side 1: c_z = -1). Both slabs
// hold the plane's tiles in the same order with the same masks, so the layout agrees.
struct HaloDirs {
    int d[5];
};

template <int DT>
__global__ void k_halo(typename Store<DT>::T* __restrict__ f, const uint64_t* __restrict__ smask,
                       const int32_t* __restrict__ tlane, int64_t n_tiles, HaloDirs dirs, int pack,
                       typename Store<DT>::T* __restrict__ buf) {
    const int64_t n = n_tiles * SLOTS;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx >> 6;
        const int s = (int)(idx & 63);
        const uint64_t sm = smask[k];
        const bool solid = (sm >> s) & 1;
        const uint32_t P = solid ? 0u : node_lane((uint32_t)tlane[k], sm, s);
#pragma unroll
        for (int d = 0; d < 5; d++) {
            if (pack) buf[d * n + idx] = solid ? nan_value<DT>() : f[data_index(P, dirs.d[d])];
            else if (!solid) f[data_index(P, dirs.d[d])] = buf[d * n + idx];
        }
    }
}

cudaError_t launch_halo(lbm_ctx* c, int side, int pack, void* buf) {
    HaloDirs down = {{6, 12, 14, 16, 18}};   // c_z = -1
    HaloDirs up = {{5, 11, 13, 15, 17}};     // c_z = +1
    int64_t k0, n;
    HaloDirs dirs;
    if (pack) {
        k0 = side == 0 ? c->own_k0 : c->own_k1 - c->bnd_hi;
        n = side == 0 ? c->bnd_lo : c->bnd_hi;
        dirs = side == 0 ? down : up;
    } else {
        k0 = side == 0 ? 0 : c->own_k1;
        n = side == 0 ? c->own_k0 : c->n_tiles - c->own_k1;
        dirs = side == 0 ? up : down;
    }
    if (n == 0) return cudaSuccess;
    const unsigned g = grid_for(n * SLOTS, 256);
#define LBM_HALO(DT, TT)                                                                                     \
    k_halo<DT><<<g, 256, 0, c->stream>>>((TT*)c->f[c->cur], c->smask + k0, c->tlane + k0, n, dirs, pack, (TT*)buf)
    if (c->dtype == LBM_F64) LBM_HALO(LBM_F64, double);
    else if (c->dtype == LBM_F32) LBM_HALO(LBM_F32, float);
    else LBM_HALO(LBM_F16S, __half);
#undef LBM_HALO
    return cudaGetLastError();
}

}  // namespace lbm
