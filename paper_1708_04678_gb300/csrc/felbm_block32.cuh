// Blocked FP32 solve: several Richardson steps of a node block per launch.
// Included by felbm.cu after the DevMesh/Bufs definitions and the
// programmatic-launch helpers.
//
// The steps are those of k_sweep32,
//     x_{k+1,i} = x_{k,i} + tau_k m_i^{-1} (b_i - sum_j M_ij x_{k,j}),
// with the same arithmetic per row in the same order, so both give the same
// bits.  A step at a time is bound by moving the vectors: every step reads
// x_k and b, gathers seven neighbours of every node from L1/L2 and writes
// x_{k+1}.  Here a thread block owns a contiguous run of at most kBlockCore
// nodes; for one plane of right-hand sides after another it loads x_k on the
// run and the K layers of nodes around it into shared memory once, advances K
// steps, each on one layer less, and writes x_{k+K} of the run.  The rows of
// the matrix and 1/m of a thread's nodes stay in registers for the whole
// block, b and the node's own x for the K steps of a plane; x ping-pongs
// between two shared arrays, while cp.async brings the next plane's x and b
// into a third.  The nodes of the layers are computed by every block that
// needs them.
//
// What bounds it: shared-memory wavefronts (LSU data pipe 70 % busy with three
// steps a launch on 520,704 nodes), six 16-byte gathers a node and plane per
// step and about 1.4 times the conflict-free count; DRAM is 20 % busy.  Solve
// phase of the time step, field update included (GB300):
//                                    step at a time   blocked
//   2,082,816 nodes, FP32, 10 steps      1,098 us      758 us
//     131,072 nodes, FP32, 10 steps        109 us       82 us (rows of 9)
//     520,704 nodes, FP64, 3 x 14        2,019 us    1,280 us (FP64 refinement included)
//       2,112 nodes, FP64, 3 x 14          164 us       43 us
// Blocks of 512 nodes at 64 registers put two thread blocks on a
// multiprocessor, one computing while the other loads.  With blocks of 1,024
// nodes, 128 registers and one thread block the 2.08M-node phase took 1,157 us,
// without the cp.async prefetch 942 us, with two steps a launch 889 us (blocked
// phase then 792 us).
constexpr int kHaloMax = 504;          // largest first layer of a tile (felbm_sweep_tiled's limit)
constexpr int kBlockThreads = 512;
constexpr int kBlockNpt = kBlockNodes / kBlockThreads;      // nodes per thread
// Fewer blocks than this per multiprocessor run one plane per thread block (all
// planes in one leave the chip idle); from one block per multiprocessor on, five
// planes on the same rows are the faster form: 84 us against 88 us for the solve
// on 131,072 nodes (256 blocks), 1,618 against 1,771 us on 520,704 (FP64).
// Where even nine thread blocks per block fit the chip one to a multiprocessor,
// one pair of right-hand sides each: 72 us a step against 78 on 2,112 nodes (8
// blocks, FP64); on 18,432 nodes (64 blocks) 160 against 148.
constexpr int kSplitPlanesBelow = 1;
static bool split_pairs(int n_blocks, int n_sm) { return 9 * n_blocks <= n_sm; }

struct BlockTau {
    float tau[kBlockSteps];
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// A piece of the FP32 vectors: NV consecutive values of node i at x + off +
// kStride i -- a plane of vec_at (NV 4, stride 4; rest plane NV 2, stride 2) or
// half of a float4 plane (NV 2, stride 4).
__device__ __forceinline__ uint32_t plane_off(int Np, int p) { return (p < 4 ? 4u * p : 16u) * (uint32_t)Np; }
template <int NV, int kStride>
__device__ __forceinline__ void cp_async_piece(float* dst, const float* x, uint32_t off, int i) {
    const float* src = x + off + (size_t)kStride * i;
    if constexpr (NV == 4)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// Shared memory of a block: three copies of x (two for the steps, one that
// receives the next plane's) and the next plane's b.
struct BlockSmem {
    float x[3][kBlockNodes * 4];
    float b[kBlockNodes * 4];
    int cnt[kBlockSteps + 1];          // nodes up to each layer
};
// With the field update in the last launch: the increments of the block's own
// nodes, piece by piece ([18][kBlockCore] floats).
struct BlockUpdateSmem : BlockSmem {
    alignas(16) float d[18 * kBlockCore];
};

// Queue the copies of the piece at off: x_k on the region into x[buf], b on the nodes
// that are stepped (kFromRhs: b on the whole region and no x).
template <int NV, int kStride, bool kFromRhs>
__device__ __forceinline__ void block_fetch(BlockSmem& sm, const DevMesh& m, const Bufs& b, const float* cur, int K, uint32_t off,
                                            int buf, const int (&node)[kBlockNpt]) {
#pragma unroll
    for (int n = 0; n < kBlockNpt; ++n) {
        const int r = (int)threadIdx.x + n * kBlockThreads;
        if (r < sm.cnt[kFromRhs ? K : K - 1]) cp_async_piece<NV, kStride>(sm.b + r * NV, b.r32, off, node[n]);
        if (!kFromRhs && r < sm.cnt[K]) cp_async_piece<NV, kStride>(sm.x[buf] + r * NV, cur, off, node[n]);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The K steps of the piece at off, whose copies into x[buf] and b were queued by this
// thread; queues those of plane `next` (kPlanes: none) into the third buffer,
// which it returns.
template <int NV, int kStride, int kW, bool kFromRhs, bool kUpdate>
__device__ __forceinline__ int block_plane(BlockSmem& sm, const DevMesh& m, const Bufs& b, const float* cur,
                                           float* nxt, const BlockTau& bt, int K, float tau0, uint32_t off, int next, int buf, const int (&node)[kBlockNpt],
                                           const float (&val)[kBlockNpt][kW], const uint32_t (&col)[kBlockNpt][kW / 2],
                                           const float (&im)[kBlockNpt]) {
    const int tid = (int)threadIdx.x;
    float x[kBlockNpt][NV], rr[kBlockNpt][NV];
    int ia = buf, ib = buf == 2 ? 0 : buf + 1;
    const int free = ib == 2 ? 0 : ib + 1;
    asm volatile("cp.async.wait_all;" ::: "memory");
    // a thread reads only its own copies here; after the barrier all of x[buf]
    // is there, and the free buffer's last readers (the previous plane) are done
#pragma unroll
    for (int n = 0; n < kBlockNpt; ++n) {
        const int r = tid + n * kBlockThreads;
        if (r < sm.cnt[kFromRhs ? K : K - 1]) {
            load_shared(rr[n], sm.b + r * NV);
            if constexpr (kFromRhs) {
                const float s = im[n] * tau0;
#pragma unroll
                for (int c = 0; c < NV; ++c) x[n][c] = rr[n][c] * s;
                store_shared(sm.x[buf] + r * NV, x[n]);
            } else {
                load_shared(x[n], sm.x[buf] + r * NV);
            }
        }
    }
    __syncthreads();
    if (next < 4)
        block_fetch<4, 4, kFromRhs>(sm, m, b, cur, K, plane_off(m.Np, next), free, node);
    else if (next == 4)
        block_fetch<2, 2, kFromRhs>(sm, m, b, cur, K, plane_off(m.Np, 4), free, node);
    for (int step = 1; step <= K; ++step) {
        const int nc = sm.cnt[K - step];
        const float tau = bt.tau[step - 1];
        const float* xa = sm.x[ia];
        float* xb = sm.x[ib];
#pragma unroll
        for (int n = 0; n < kBlockNpt; ++n) {
            const int r = tid + n * kBlockThreads;
            if (r < nc) {
                float acc[NV];
#pragma unroll
                for (int c = 0; c < NV; ++c) acc[c] = fmaf(val[n][0], x[n][c], 0.0f);
#pragma unroll
                for (int k = 1; k < kW; ++k) {
                    const uint32_t at = (k & 1) ? col[n][k / 2] & 0xffffu : col[n][k / 2 - 1] >> 16;
                    float g[NV];
                    load_shared(g, xa + at * NV);
#pragma unroll
                    for (int c = 0; c < NV; ++c) acc[c] = fmaf(val[n][k], g[c], acc[c]);
                }
                const float s = tau * im[n];
#pragma unroll
                for (int c = 0; c < NV; ++c) x[n][c] = fmaf(s, rr[n][c] - acc[c], x[n][c]);
                if (step < K)
                    store_shared(xb + r * NV, x[n]);
                else
                    store_shared(kUpdate ? nxt + (size_t)(off / (uint32_t)m.Np) * kBlockCore + kStride * r
                                         : nxt + off + (size_t)kStride * node[n],
                                 x[n]);
            }
        }
        if (step < K) __syncthreads();
        const int t = ia;
        ia = ib;
        ib = t;
    }
    return free;
}

// kW: ELL width; kFromRhs: x_0 = tau_0 b / m formed here.  n4: float4 planes in
// use (the first n4 of them, and always the rest plane).  Grid: blocks x 1 (all
// planes in use of a block in turn), blocks x (n4 + 1) (a plane each) or, kPair,
// blocks x (2 n4 + 1) (a pair of right-hand sides each).  kUpdate (first form,
// all planes): the last iterate is the increment of the time step; it stays in
// shared memory and the fields and deviations are updated here, which saves
// writing and reading it: solve phase 788 -> 758 us on 2,082,816 nodes.
template <int kW, bool kFromRhs, bool kPair, bool kUpdate = false>
__global__ void __launch_bounds__(kBlockThreads, kW <= 9 ? 2 : 1)
    k_block32(DevMesh m, Phys c, Bufs b, const float* cur, float* nxt, const __grid_constant__ BlockTau bt, int K,
              float tau0, int n4) {
    static_assert(!(kPair && kUpdate), "the update needs all planes");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    BlockSmem& sm = *reinterpret_cast<BlockSmem*>(smem_raw);
    pdl_release();
    const int blk = (int)blockIdx.x, tid = (int)threadIdx.x;
    if (tid <= kBlockSteps) sm.cnt[tid] = m.blk_cnt[blk * (kBlockSteps + 1) + tid];
    const int s0 = m.blk_ptr[blk], ni = m.blk_ptr[blk + 1] - s0;
    const int32_t* halo = m.blk_halo + m.blk_halo_ptr[blk] - ni;
    const int r0 = m.blk_row[blk], rstride = m.blk_row[blk + 1] - r0;
    const float* bval = m.blk_val + (size_t)kW * r0;
    const uint32_t* bcol = m.blk_col + (size_t)(kW / 2) * r0;
    __syncthreads();
    const int nreg = sm.cnt[K], nrow = sm.cnt[K - 1];
    int node[kBlockNpt];
    float val[kBlockNpt][kW], im[kBlockNpt];
    uint32_t col[kBlockNpt][kW / 2];
#pragma unroll
    for (int n = 0; n < kBlockNpt; ++n) {
        const int r = tid + n * kBlockThreads;
        node[n] = r < ni ? s0 + r : (r < nreg ? halo[r] : s0);
        im[n] = m.inv_lumped32[node[n]];
    }
    const int y = (int)blockIdx.y;
    const bool one = gridDim.y > 1;
    const int p0 = one ? y : 0, p1 = one ? min(y + 1, n4) : n4;      // float4 planes [p0, p1)
    const bool rest = kPair ? y == 2 * n4 : (!one || y == n4);
    const uint32_t half = plane_off(m.Np, y >> 1) + 2 * (y & 1);
    pdl_wait();
    if (kPair && !rest)
        block_fetch<2, 4, kFromRhs>(sm, m, b, cur, K, half, 0, node);
    else if (!kPair && p0 < p1)
        block_fetch<4, 4, kFromRhs>(sm, m, b, cur, K, plane_off(m.Np, p0), 0, node);
    else
        block_fetch<2, 2, kFromRhs>(sm, m, b, cur, K, plane_off(m.Np, 4), 0, node);
#pragma unroll
    for (int n = 0; n < kBlockNpt; ++n) {
        const int r = tid + n * kBlockThreads;
        if (r < nrow) {
#pragma unroll
            for (int k = 0; k < kW; ++k) val[n][k] = bval[k * rstride + r];
#pragma unroll
            for (int k = 0; k < kW / 2; ++k) col[n][k] = bcol[k * rstride + r];
        }
    }
    int buf = 0;
    if constexpr (kUpdate) nxt = static_cast<BlockUpdateSmem&>(sm).d;
    if constexpr (kPair) {
        if (!rest)
            block_plane<2, 4, kW, kFromRhs, false>(sm, m, b, cur, nxt, bt, K, tau0, half, kPlanes, 0, node, val, col, im);
    } else {
        for (int p = p0; p < p1; ++p)
            buf = block_plane<4, 4, kW, kFromRhs, kUpdate>(sm, m, b, cur, nxt, bt, K, tau0, plane_off(m.Np, p),
                                                  p + 1 < p1 ? p + 1 : (rest ? 4 : kPlanes), buf, node, val, col, im);
    }
    if (rest)
        block_plane<2, 2, kW, kFromRhs, kUpdate>(sm, m, b, cur, nxt, bt, K, tau0, plane_off(m.Np, 4), kPlanes, buf, node, val, col,
                                        im);
    if constexpr (kUpdate) {
        __syncthreads();
        if (tid < ni) {
            float d[18];
#pragma unroll
            for (int p = 0; p < kPlanes; ++p)
#pragma unroll
                for (int v = 0; v < (p < 4 ? 4 : 2); ++v)
                    d[vec_row(p, v)] = nxt[(4 * p) * kBlockCore + (p < 4 ? 4 : 2) * tid + v];
            dev32_update(m, c, b, s0 + tid, d);
        }
    }
}

// The field and deviation update from the solve's last iterate (FP32-deviation
// states): psi^{n+1} = psi_hat + d.
__global__ void __launch_bounds__(128) k_update32(DevMesh m, Phys c, Bufs b, const float* x) {
    pdl_release();
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.N) return;
    float d[18];
    load_all(d, x, m.Np, i);
    dev32_update(m, c, b, i, d);
}
