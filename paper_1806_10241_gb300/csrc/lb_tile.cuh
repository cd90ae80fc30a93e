// Several time steps per launch on tiles held in shared memory (included by
// lb_kernels.cu inside its anonymous namespace; FP32 arithmetic, FP32 / FP16 /
// BF16 storage).
//
// A block owns a tile of the lattice: `rows` rows of 64 columns, all 19
// planes, fetched once by TMA, and with them the macroscopic fields of the
// stored state (u_x, u_y, u_theta, T) in FP32.  It takes T time steps on the
// tile without leaving the SM; each step is valid one row and one column less
// on every open side of the tile, so the last one is valid on the tile less a
// margin of T, which the block writes to the destination buffer.  Neighbouring
// tiles overlap by their margins and recompute them: no block waits for
// another one.
//
// Why tiles: one launch boundary, one fetch and one pass over memory serve T
// steps, and a row update needs less: the fields of the stored state are
// written by the warp that has the new values in registers, and the radial
// neighbours' fields are plain shared-memory reads instead of shuffles and
// recomputed halo columns (640 warp instructions per 64 columns of result in
// FP32, recomputed margins included, against 809 of the marching step).
// Measured per step (one step per launch before, tiles now): 100 x 100 FP32 7.1
// -> 2.4 us, 40 x 400 FP32 7.4 -> 2.8 us, 256 x 512 FP32 11.6 -> 5.0 us, 301 x
// 257 BF16 12.8 -> 4.7 us.  What bounds a small tile now is the latency of a
// row update, about 1.3 us, and 2.5 us per launch.

template <typename S> struct TileGeom {
    static constexpr int cols = 64;
    static constexpr int row_bytes = NQ * cols * (int)sizeof(S);   // all planes of one row
    static constexpr int field_bytes = 4 * cols * (int)sizeof(float);
    static constexpr int slot_bytes = row_bytes + field_bytes;
    static_assert(row_bytes % 128 == 0, "TMA destinations stay 128-byte aligned");
};

// The tiles of a lattice.  Tile j of window w holds the columns [w * cs, w * cs
// + 64) and, on a lattice with end walls, the rows [j * rs, j * rs + rows); on a
// periodic one the rows [j * rs - rm, (j + 1) * rs + rm), modulo nz.  Made for
// passes of rm steps, they serve shorter ones as well.
struct TileShape {
    int rows;       // rows loaded by a full tile
    int rm, cm;     // margins in rows and columns
    int rs, cs;     // distance of consecutive tiles: rows - 2 rm, 64 - 2 cm
    int nw;         // windows across
};

// Rows of a tile as they lie in shared memory.  The state after step t of
// local row r sits in slot r + T - 1 - t: a step moves every row down by one
// slot, so a group of rows can be written while the next group still reads
// its unmodified lower neighbour.
template <typename S>
__device__ __forceinline__ F2 unpack_stored(uint32_t d, float is)
{
    return LoadScaled<S>::pair(reinterpret_cast<const S *>(&d), is);
}

// Store of one plane of a pair into the tile; v becomes the value a reader of
// the tile gets.
template <typename S>
__device__ __forceinline__ void tile_put(S *p, F2 &v, uint32_t w, float is)
{
    if constexpr (sizeof(S) == 4) {
        *reinterpret_cast<float2 *>(p) = v.v;
    } else {
        const uint32_t d = PairIO<S>::round(v, w);
        *reinterpret_cast<uint32_t *>(p) = d;
        v = unpack_stored<S>(d, is);
    }
}

template <typename S>
__device__ __forceinline__ float *fields_of(S *slot)
{
    return reinterpret_cast<float *>(slot + NQ * TileGeom<S>::cols);
}
template <typename S>
__device__ __forceinline__ const float *fields_of(const S *slot)
{
    return reinterpret_cast<const float *>(slot + NQ * TileGeom<S>::cols);
}

template <typename S>
__device__ __forceinline__ void put_fields(S *slot, int cA, const PM2 &m)
{
    float *f = fields_of(slot);
    *reinterpret_cast<float2 *>(f + cA) = m.ux.v;
    *reinterpret_cast<float2 *>(f + 64 + cA) = m.uy.v;
    *reinterpret_cast<float2 *>(f + 128 + cA) = m.ut.v;
    *reinterpret_cast<float2 *>(f + 192 + cA) = m.T.v;
}

__device__ __forceinline__ F2 fpair(const float *f, int cA)
{
    F2 r;
    r.v = *reinterpret_cast<const float2 *>(f + cA);
    return r;
}

// One node pair of one row from the slots b_m, b_0, b_p of rows i - 1, i, i + 1.
template <typename S>
__device__ __forceinline__ void tile_row(const KP<float> &k, const Lane2 &L, const S *b_m, const S *b_0, const S *b_p,
                                         bool has_m, bool has_p, NodeOut2 &o)
{
    // without a neighbour row the wall rules replace what it would have given:
    // the row itself is read in its place, and no load is conditional (1024 x
    // 2048 FP16: 46.2 -> 44.6 us per step)
    b_m = has_m ? b_m : b_0;
    b_p = has_p ? b_p : b_0;
    const float *f_m = fields_of(b_m), *f_0 = fields_of(b_0), *f_p = fields_of(b_p);
    constexpr int C = TileGeom<S>::cols;
    const int cA = 2 * L.lane;
    const float is = k.inv_scale;
    F2 fv[9], gv[5], hv5[5];
    OwnStage<S, C> own{b_0, cA, is, 0.0f, 0.0f};
    StageRd<S, C> rd{b_m, cA, is};
    fv[1] = rd.pair(1);
    fv[5] = rd.left(5);
    fv[8] = rd.right(8);
    gv[1] = rd.pair(G0 + 1);
    hv5[1] = rd.pair(H0 + 1);
    rd.b = b_0;
    fv[0] = rd.pair(0);
    fv[2] = rd.left(2);
    fv[4] = rd.right(4);
    gv[0] = rd.pair(G0 + 0);
    gv[2] = rd.left(G0 + 2);
    gv[4] = rd.right(G0 + 4);
    hv5[0] = rd.pair(H0 + 0);
    hv5[2] = rd.left(H0 + 2);
    hv5[4] = rd.right(H0 + 4);
    rd.b = b_p;
    fv[3] = rd.pair(3);
    fv[6] = rd.left(6);
    fv[7] = rd.right(7);
    gv[3] = rd.pair(G0 + 3);
    hv5[3] = rd.pair(H0 + 3);
    if (L.edge_warp) {
        own.m8v = StageRd<S, C>{b_m, cA, is}.pair(8).v.x;
        own.p7v = rd.pair(7).v.x;
    }
    wall_rules(k, own, L, L.edge_warp, has_m, has_p, fv, gv, hv5);
    // central differences of the stored-state fields
    const Sides2 c{fpair(f_0, cA), fpair(f_0 + 64, cA), fpair(f_0 + 128, cA), fpair(f_0 + 192, cA)};
    F2 uy_xm = fpair(f_m + 64, cA), uy_xp = fpair(f_p + 64, cA);
    if (!has_m) uy_xm = end_ghost_uy(k, L, 0, c.uy);
    if (!has_p) uy_xp = end_ghost_uy(k, L, 1, c.uy);
    Sides2 l{mk2(f_0[cA - 1], c.ux.v.x), mk2(f_0[63 + cA], c.uy.v.x), mk2(f_0[127 + cA], c.ut.v.x),
             mk2(f_0[191 + cA], c.T.v.x)};
    Sides2 r{mk2(c.ux.v.y, f_0[cA + 2]), mk2(c.uy.v.y, f_0[66 + cA]), mk2(c.ut.v.y, f_0[130 + cA]),
             mk2(c.T.v.y, f_0[194 + cA])};
    if (L.edge_warp) lateral_ghosts(k, L, c, l, r);
    auto across = [](F2 right, F2 left) { return mk2(right.v.x - left.v.x, right.v.y - left.v.y); };
    update_node2<Scaled<S>::value>(k.pc, k.explicit_src, geo_of(k.pc, L.iy), fv, gv, hv5, uy_xp - uy_xm, across(r.ux, l.ux), across(r.uy, l.uy),
                                   across(r.ut, l.ut), across(r.T, l.T), o);
}

// Registers per thread: FP32 tiles run 12 warps on an SM (shared memory), 168
// registers each; 16-bit ones 16 warps of 128 (FP32 at 128: 4-5 % slower;
// 16-bit at 168: 12 warps, 14-18 % slower on the 1024 x 2048 lattice).
template <typename S> constexpr int kTileRegs = sizeof(S) == 4 ? 168 : 128;

template <typename S>
__host__ __device__ size_t tile_smem_bytes(int slots)
{
    return (size_t)slots * TileGeom<S>::slot_bytes + 128;
}

// fields of the stored state of a row just fetched
template <typename S>
__device__ __forceinline__ void tile_fields(const KP<float> &k, S *slot, int cA)
{
    const StageRd<S, TileGeom<S>::cols> rd{slot, cA, k.inv_scale};
    F2 v[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] = rd.pair(q);
    put_fields<S>(slot, cA, moments2(v, k));
}

// the new state of a row into a slot, with its fields
template <typename S>
__device__ __forceinline__ void tile_store(const KP<float> &k, S *slot, int cA, int row, int A, uint32_t salt,
                                           const NodeOut2 &o)
{
    RoundWords w((uint32_t)row * (uint32_t)k.pitch + (uint32_t)A, salt);
    F2 v[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        v[q] = o.v[q];
        tile_put<S>(slot + q * TileGeom<S>::cols + cA, v[q], PairIO<S>::rounds ? w.next() : 0u, k.inv_scale);
    }
    put_fields<S>(slot, cA, moments2(v, k));
}

// one row of all planes by TMA into a slot
template <typename S>
__device__ __forceinline__ void tile_fetch(const CUtensorMap *map, uint32_t slot, int c0, int row, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(slot),
        "l"((unsigned long long)map), "r"(c0), "r"(row), "r"(0), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tile_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ int wrap_row(int row, int nz)
{
    row %= nz;
    return row < 0 ? row + nz : row;
}

// The rounding salts of the steps of a pass, behind the barriers (visible after
// the next barrier of the block).
template <typename S>
__device__ __forceinline__ uint32_t *tile_salts(unsigned char *smem, int slots, int T, unsigned long long step)
{
    uint32_t *salts = reinterpret_cast<uint32_t *>(smem + (size_t)slots * TileGeom<S>::slot_bytes + 64);
    if (PairIO<S>::rounds && (int)threadIdx.x < T) salts[threadIdx.x] = salt_of(step + threadIdx.x);
    return salts;
}

// T steps on one tile by a block.  smem: (sh.rows + T - 1) slots and 128 bytes.
template <typename S>
__device__ __forceinline__ void tile_steps(const KP<float> &k, const CUtensorMap *map, S *__restrict__ dst,
                                           const TileShape &sh, int T, int win, int tile, unsigned long long step,
                                           int *status, unsigned char *smem)
{
    constexpr int SB = TileGeom<S>::slot_bytes / (int)sizeof(S);
    const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int nz = k.nz, c0 = win * sh.cs;
    // rows of this tile: local row 0 is lattice row r0
    const int r0 = k.xper ? tile * sh.rs - sh.rm : tile * sh.rs;
    const int n = k.xper ? min(sh.rs, nz - tile * sh.rs) + 2 * sh.rm : min(sh.rows, nz - r0);
    const bool bottom = !k.xper && r0 == 0, top = !k.xper && r0 + n == nz;

    S *slots = reinterpret_cast<S *>(smem);
    const uint32_t bar = smem_u32(smem + (size_t)(sh.rows + T - 1) * TileGeom<S>::slot_bytes);
    const int groups = (n + W - 1) / W;
    uint32_t *salts = tile_salts<S>(smem, sh.rows + T - 1, T, step);
    if (threadIdx.x == 0) {
        for (int g = 0; g < groups && g < 8; ++g)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8u * g) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const Lane2 L = lane2(k, c0);
    __syncthreads();
    grid_dependency_wait();
    if (warp == 0) {
        if (lane < 8) {
            // group g of W rows (the last barrier takes all the rows from its group on)
            const int first = lane * W, last = lane == 7 ? n : min(n, first + W);
            if (first < n) tile_expect(bar + 8u * lane, (uint32_t)(TileGeom<S>::row_bytes * (last - first)));
        }
        __syncwarp();
        const uint32_t base = smem_u32(smem) + (uint32_t)(T - 1) * TileGeom<S>::slot_bytes;
        for (int r = lane; r < n; r += 32)
            tile_fetch<S>(map, base + (uint32_t)r * TileGeom<S>::slot_bytes, c0, k.xper ? wrap_row(r0 + r, nz) : r0 + r,
                          bar + 8u * min(r / W, 7));
    }

    bool ok = true;
    const int cA = 2 * lane;
    for (int g = 0; g < groups; ++g) {
        if (g < 8) ok &= mbar_wait_bounded(bar + 8u * g, 0u, kTmaWaitLimit);
        const int r = g * W + warp;
        if (r < n) tile_fields<S>(k, slots + (r + T - 1) * SB, cA);
    }
    if (__syncthreads_or(!ok)) {
        if (threadIdx.x == 0) atomicExch(status, (int)LB_ERR_TIMEOUT);
        return;
    }

    const int vlo = win == 0 ? 0 : c0 + sh.cm, vhi = win == sh.nw - 1 ? k.nr : c0 + TileGeom<S>::cols - sh.cm;
    const bool out_cols = L.A >= vlo && L.A < vhi;
    const int out_lo = bottom ? 0 : sh.rm, out_hi = top ? n : n - sh.rm;  // T < rm: rows of the margin are not stored
    for (int t = 0; t < T; ++t) {
        const bool last = t == T - 1;
        const int lo = bottom ? 0 : t + 1, hi = top ? n : n - (t + 1);
        const uint32_t salt = PairIO<S>::rounds ? salts[t] : 0u;
        for (int g = lo; g < hi; g += W) {
            const int r = g + warp;
            const bool active = r < hi;
            NodeOut2 o;
            const int row = k.xper ? wrap_row(r0 + r, nz) : r0 + r;
            S *b_0 = slots + (r + T - 1 - t) * SB;
            if (active) tile_row<S>(k, L, b_0 - SB, b_0, b_0 + SB, !bottom || r > 0, !top || r < n - 1, o);
            if (last) {
                if (active && out_cols && r >= out_lo && r < out_hi) store_row<S>(k, dst, row, L.A, salt, o);
                continue;
            }
            __syncthreads();  // the group's reads are done: its slots may be written
            if (active) tile_store<S>(k, b_0 - SB, cA, row, L.A, salt, o);
        }
        if (!last) __syncthreads();
    }
}

// The same on a long strip of rows, for lattices that do not fit on the device
// as resident tiles: no rows are recomputed between the groups of a strip, and
// the rows of the next group are on their way while this one is worked on.
// The strip is marched through a ring of 2 W + 2 T slots: in tick m the warps
// take the fields of rows m W .. m W + W - 1 and then step t on the rows
// m W - 1 - t .., one row per warp.  State t of row r sits in slot (r - t) mod
// the ring.  A slot is refilled one tick after its last read (2 W + 2 T slots
// are exactly what is live: W rows on their way, W of this tick, and 2 T of
// the lower neighbours' states).  1024 x 2048: FP32 52.0 us per step with one
// step per launch, 40.6 us with strips of two steps; what bounds it is the
// latency of dependent instructions at 12 warps per SM (47 % issue), not
// memory.  FP16 49.1 -> 44.6 us at that size.
// kRunning: the position in the ring, the lattice row and the limits of the
// active rows run along with t instead of being formed from it (10 % fewer
// instructions in 16-bit storage, 2 % in FP32: 41.3 -> 39.8 us).  FP32 batches,
// whose parameters are in shared memory, have no registers left for that (40
// lattices of 64 to 128 columns: 18.7 us formed, 19.9 running).
template <typename S, bool kRunning>
__device__ __forceinline__ void strip_steps(const KP<float> &k, const CUtensorMap *map, S *__restrict__ dst,
                                            const TileShape &sh, int T, int win, int tile, unsigned long long step,
                                            int *status, unsigned char *smem, int part = 0, unsigned *begun = nullptr,
                                            unsigned pass = 0)
{
    constexpr int SB = TileGeom<S>::slot_bytes / (int)sizeof(S);
    const int warp = __shfl_sync(FULL, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31, W = blockDim.x >> 5;
    const int nz = k.nz, R = 2 * W + 2 * T, c0 = win * sh.cs;
    const int r0 = k.xper ? tile * sh.rs - sh.rm : tile * sh.rs;
    const int n = k.xper ? min(sh.rs, nz - tile * sh.rs) + 2 * sh.rm : min(sh.rows, nz - r0);
    const bool bottom = !k.xper && r0 == 0, top = !k.xper && r0 + n == nz;

    S *slots = reinterpret_cast<S *>(smem);
    const uint32_t ring = smem_u32(smem), bar = ring + (uint32_t)(R * TileGeom<S>::slot_bytes);
    uint32_t *salts = tile_salts<S>(smem, R, T, step);
    if (threadIdx.x == 0) {
        for (int g = 0; g < 2; ++g)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar + 8u * g) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const Lane2 L = lane2(k, c0);
    __syncthreads();
    if (part != 2) grid_dependency_wait();
    if (part == 1) {  // the pass before is complete: say so to part 2 (k_tiles)
        if (blockIdx.x == 0) {
            if (threadIdx.x == 0) st_release_gpu(begun, pass);
            __syncthreads();
        }
        grid_dependency_trigger();
    }
    bool told = true;
    if (part == 2 && warp == 0) {  // which issues the fetches, the first access to the lattice
        int polls = 0;
        while (ld_acquire_gpu(begun) != pass && (told = ++polls <= kFlagWaitLimit)) __nanosleep(100);
        asm volatile("fence.proxy.async.global;" ::: "memory");
    }
    auto fetch = [&](int m, int slot0) {  // the rows of tick m (warp 0)
        const int first = m * W, cnt = min(W, n - first);
        if (cnt <= 0) return;
        if (lane == 0) tile_expect(bar + 8u * (m & 1), (uint32_t)(TileGeom<S>::row_bytes * cnt));
        __syncwarp();
        if (lane < cnt) {
            int slot = slot0 + lane;
            slot -= slot >= R ? R : 0;
            tile_fetch<S>(map, ring + (uint32_t)(slot * TileGeom<S>::slot_bytes), c0,
                          k.xper ? wrap_row(r0 + first + lane, nz) : r0 + first + lane, bar + 8u * (m & 1));
        }
    };
    if (warp == 0 && __all_sync(FULL, told)) {  // (else the wait for the first rows runs out)
        fetch(0, 0);
        fetch(1, W);
    }

    const int vlo = win == 0 ? 0 : c0 + sh.cm, vhi = win == sh.nw - 1 ? k.nr : c0 + TileGeom<S>::cols - sh.cm;
    const bool out_cols = L.A >= vlo && L.A < vhi;
    const int out_lo = bottom ? 0 : sh.rm, out_hi = top ? n : n - sh.rm;  // T < rm: rows of the margin are not stored
    const int cA = 2 * lane;
    const int ticks = ((top ? n + T : n) + W - 1) / W;
    // rows r of step t that the strip advances: from lo + t dlo on, below hi + t dhi, with r + t for r
    const int lo = bottom ? 0 : 1, dlo = bottom ? 1 : 2, hi = top ? n : n - 1, dhi = top ? 1 : 0;
    int s0 = 0;  // slot of row m W, state 0
    int row0 = wrap_row(r0 - 1 + warp, nz);  // lattice row of step 0 in this tick
    for (int m = 0; m < ticks; ++m) {
        bool ok = true;
        const int rf = m * W + warp;
        if (m * W < n) ok = mbar_wait_bounded(bar + 8u * (m & 1), (uint32_t)((m >> 1) & 1), kTmaWaitLimit);
        int sf = s0 + warp;
        sf -= sf >= R ? R : 0;
        if (rf < n) tile_fields<S>(k, slots + sf * SB, cA);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) atomicExch(status, (int)LB_ERR_TIMEOUT);
            if (m == 0 && W < n) (void)mbar_wait_bounded(bar + 8u, 0u, kTmaWaitLimit);  // tick 1 is in flight
            return;
        }
        // every warp is done with tick m - 1: its slots take the rows of tick m + 1
        if (m > 0 && warp == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            int s1 = s0 + W;
            s1 -= s1 >= R ? R : 0;
            fetch(m + 1, s1);
        }
        int sl = sf == 0 ? R - 1 : sf - 1;  // slot of the warp's row in step t, state t
        int row = row0;
        for (int t = 0, lo_t = lo, hi_t = hi; t < T; ++t, lo_t += dlo, hi_t += dhi) {
            const int r = rf - 1 - t;
            if constexpr (!kRunning) {
                lo_t = t + (bottom ? 0 : t + 1);
                hi_t = t + (top ? n : n - (t + 1));
                row = k.xper ? wrap_row(r0 + r, nz) : r0 + r;
                sl = s0 + warp - 1 - 2 * t;
                sl += sl < 0 ? R : 0;
                sl -= sl >= R ? R : 0;
            }
            const bool last = t == T - 1, active = rf - 1 >= lo_t && rf - 1 < hi_t;
            S *b_0 = slots + sl * SB, *b_m = sl == 0 ? slots + (R - 1) * SB : b_0 - SB,
              *b_p = sl == R - 1 ? slots : b_0 + SB;
            const uint32_t salt = PairIO<S>::rounds ? salts[t] : 0u;
            NodeOut2 o;
            if (active) tile_row<S>(k, L, b_m, b_0, b_p, !bottom || r > 0, !top || r < n - 1, o);
            if (last) {
                if (active && out_cols && r >= out_lo && r < out_hi) store_row<S>(k, dst, row, L.A, salt, o);
            } else {
                __syncthreads();  // the reads of step t are done: its slots may be written
                if (active) tile_store<S>(k, b_m, cA, row, L.A, salt, o);
                __syncthreads();
            }
            row = row == 0 ? nz - 1 : row - 1;
            sl -= 2;
            sl += sl < 0 ? R : 0;
        }
        s0 += W;
        s0 -= s0 >= R ? R : 0;
        row0 += W;
        if (row0 >= nz) row0 = wrap_row(row0, nz);
    }
}

// One lattice: block b of the launch takes tile `first + b` (rev: from the last
// one back), windows running fastest.
// A pass cut into two launches (part 1 and 2; 0: the only one) runs them side
// by side, the second filling the SMs as the blocks of the first finish: it
// reads the state of the pass before and writes other rows, so it does not
// wait for the first at its start.  What it needs is that the pass before is
// complete and its writes are visible.  Part 1 waits for that pass, then writes
// the number of its own pass to *begun with release semantics and only then
// allows the dependent launch; a block of part 2 reads *begun with acquire
// semantics before its first access to the lattice (it holds that number by
// then; the wait is bounded all the same).  Pass numbers are those of the
// lattice's life, and a call that can be replayed from a graph has an even
// number of such passes, so that the pass before always has another number.
// A block of part 2 waits for part 1 before it ends: a launch that waits for
// part 2 then finds both complete.  (1024 x 2048 FP32: 43.3 us per step with
// part 2 waiting for part 1 at its start, 41.2 as one launch of two waves, 40.6
// so; 2048 x 2048: 79.1, 77.6, 76.1.)
template <typename S, bool kStrip>
__global__ void __maxnreg__(kTileRegs<S>)
    k_tiles(const __grid_constant__ KP<float> k, const __grid_constant__ CUtensorMap map, S *__restrict__ dst,
            const TileShape sh, int T, int first, unsigned long long step, int *status, int rev, int part,
            unsigned *begun, unsigned pass)
{
    extern __shared__ __align__(128) unsigned char smem[];
    if (sizeof(S) != 4 || part != 1) grid_dependency_trigger();
    const int b = first + (rev ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x);
    if constexpr (kStrip)
        strip_steps<S, true>(k, &map, dst, sh, T, b % sh.nw, b / sh.nw, step, status, smem, sizeof(S) == 4 ? part : 0,
                             begun, pass);
    else tile_steps<S>(k, &map, dst, sh, T, b % sh.nw, b / sh.nw, step, status, smem);
    if (sizeof(S) == 4 && part == 2) grid_dependency_wait();
}
