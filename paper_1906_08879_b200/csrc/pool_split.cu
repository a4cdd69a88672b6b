// Step 3 of the policy (Sec. 2.2 step 3 of the Placeto paper) for d = 32 with single-layer ReLU l_i
// on the tensor cores: the per-set sums
//   sum_{u in S_i(c)} l_i(e_u),   e_u = [h_down_u || h_up_u || x_u],
// over a chunk of nodes of a state, written as the partial sums that the head kernel adds up.
//
// Rows (node, state) depend on nothing, so this is a throughput problem: 32 (64 + F) multiply-adds a
// row. On the FP32 units (policy_d32.cu) that is what bounds it: 219 us for 992 nodes in 992 states,
// F = 12 (106 here; 1080 nodes x 256 states, F = 8: 63 and 37). Here sixteen rows of a (state, set) are the 16 rows of mma.sync.m16n8k16, on exact pieces of
// three bfloat16 numbers (Bf16x3, six products), which the pipe takes in a quarter of the time.
//   - A warp owns items (state, chunk of nodes) and walks the three sets one by one; it compacts the
//     relation row of the state into the set's node list and takes the list sixteen at a time.
//   - The rows go from memory straight into A fragments: the inner index is permuted so that the four
//     numbers a lane needs of a 16-wide step are adjacent (one 128-bit load, 64 contiguous bytes of a row per step).
//   - The weights' pieces lie in shared memory as B fragments, split once per block; reading them costs
//     half of what the instructions they feed take.
// Warps never wait for one another; sixteen of them per SM cover the loads (the tensor pipe is busy 58 % of the time. Reading a
// tile's rows during the tile before, at twelve or sixteen warps, takes registers from the chains: 108 and 114 us). Products of the leading pieces
// are kept in two chains and the small ones in a third, since the tensor core's accumulation truncates.
// Summation order is fixed, so results are reproducible bit for bit.
#include <algorithm>

#include "kernels.cuh"
#include "split_mma.cuh"

namespace placeto {

namespace {

using split::Bf16x3;

constexpr int kD = 32, kNT = kD / 8, kKS = 2 * kD / 16 + 1;     // output tiles, 16-wide steps (the last: raw features)
constexpr int kWarps = 16, kThreads = kWarps * 32, kTile = 16;
constexpr int kMaxChunk = 1024;
constexpr int kPieces = Bf16x3::kPieces;
constexpr int kFragments = 3 * kKS * kPieces * 2 * 32;          // uint4 of weight fragments

struct PoolSplitPlan {
    int chunk_nodes, chunks, items;
};

size_t smem_bytes(int chunk_nodes) {
    return (size_t)kFragments * sizeof(uint4) + 3 * kD * sizeof(float) + (size_t)kWarps * ((chunk_nodes + 7) & ~7) * sizeof(uint16_t);
}

template <bool kCompact, bool kVec>      // raw features from compact states; in rows of whole 16-byte pieces
__global__ void __launch_bounds__(kThreads, 1)
pool_split_kernel(const PoolArgs a, const PoolSplitPlan p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dependents_may_start();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int n = a.n, B = a.B, F = a.F;
    uint4 *frag = reinterpret_cast<uint4 *>(smem_raw);                  // [set][step][piece][half of the tiles][lane]
    float *bias_s = reinterpret_cast<float *>(frag + kFragments);       // [3][32]
    uint16_t *list = reinterpret_cast<uint16_t *>(bias_s + 3 * kD) + (size_t)warp * ((p.chunk_nodes + 7) & ~7);

    // ---- weights as fragments: lane (g, t) of tile nt holds rows 16 ks + 4 t .. + 3 of column 8 nt + g
    for (int i = threadIdx.x; i < 3 * kKS * kNT * 32; i += kThreads) {
        const int l = i & 31, nt = (i >> 5) % kNT, ks = (i >> 5) / kNT % kKS, set = (i >> 5) / (kNT * kKS);
        const float *W = a.l[set].W1;
        const int k0 = 16 * ks + 4 * (l & 3), col = 8 * nt + (l >> 2);
        float w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = k0 + j < 2 * kD + F ? W[(k0 + j) * kD + col] : 0.f;
        unsigned lo[kPieces], hi[kPieces];
        Bf16x3::pieces(w[0], w[1], lo);
        Bf16x3::pieces(w[2], w[3], hi);
#pragma unroll
        for (int q = 0; q < kPieces; ++q)
            reinterpret_cast<uint2 *>(frag + (((set * kKS + ks) * kPieces + q) * 2 + nt / 2) * 32 + l)[nt & 1] = make_uint2(lo[q], hi[q]);
    }
    if (threadIdx.x < 3 * kD) bias_s[threadIdx.x] = a.l[threadIdx.x / kD].b1[threadIdx.x % kD];
    __syncthreads();
    dependency_wait();          // the embeddings may come from a kernel that is still running

    for (int item = blockIdx.x + gridDim.x * warp; item < p.items; item += gridDim.x * kWarps) {
        const int chunk = item / B, b = item - chunk * B;
        const int u0 = chunk * p.chunk_nodes, nu = min(n - u0, p.chunk_nodes);
        const int c = a.cur[b];
        const bool valid = c >= 0 && c < n;
        PLACETO_DEBUG_CHECK(a.status, valid);
        const uint8_t *rel = a.relation + (size_t)(valid ? c : 0) * n + u0;
        float *out = a.partial + ((size_t)chunk * B + b) * 3 * kD;
#pragma unroll 1
        for (int set = 0; set < 3; ++set) {
            int count = 0;
            for (int base = 0; base < nu; base += 32) {
                const bool in = base + lane < nu && valid && rel[base + lane] == set;
                const unsigned mask = __ballot_sync(0xffffffffu, in);
                if (in) list[count + __popc(mask & ((1u << lane) - 1))] = (uint16_t)(base + lane);
                count += __popc(mask);
            }
            __syncwarp();
            float total[kNT][2];
#pragma unroll
            for (int nt = 0; nt < kNT; ++nt) total[nt][0] = total[nt][1] = 0.f;
            const uint4 *fr = frag + (size_t)set * kKS * kPieces * 2 * 32 + lane;
#pragma unroll 1
            for (int first = 0; first < count; first += kTile) {
                // rows past the end repeat the last one
                const int u[2] = {u0 + list[min(first + g, count - 1)], u0 + list[min(first + 8 + g, count - 1)]};
                float4 x[kKS][2];
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const size_t row = (size_t)u[r] * B + b;
#pragma unroll
                    for (int ks = 0; ks < kKS - 1; ++ks)
                        x[ks][r] = *reinterpret_cast<const float4 *>(a.H[ks >= 2] + row * kD + 16 * (ks & 1) + 4 * t);
                    float4 &f = x[kKS - 1][r];
                    f = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (kCompact) {
                        // [cost, bytes, one-hot_m(device), u == current, visited], this lane's four
                        const unsigned state = a.compact.state[row];
                        const int dev = (int)(state & 63u) + 2, m = a.compact.m;
                        float v[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int k = 4 * t + j;
                            v[j] = k == m + 2 ? (u[r] == c ? 1.f : 0.f) : k == m + 3 ? (float)(state >> 7) : k == dev && k < m + 2 ? 1.f : 0.f;
                        }
                        if (t == 0) { v[0] = a.compact.cost[u[r]]; v[1] = a.compact.bytes[u[r]]; }
                        f = make_float4(v[0], v[1], v[2], v[3]);
                    } else if (kVec) {
                        if (4 * t < F) f = *reinterpret_cast<const float4 *>(a.X + row * F + 4 * t);
                    } else {
                        float *v = &f.x;
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (4 * t + j < F) v[j] = a.X[row * F + 4 * t + j];
                    }
                }
                // chains: leading products of the first steps, of the others, and all small ones
                float acc[3][kNT][4];
#pragma unroll
                for (int ks = 0; ks < kKS; ++ks) {
                    unsigned A[kPieces][4];
                    {
                        unsigned q[4][kPieces];
                        Bf16x3::pieces(x[ks][0].x, x[ks][0].y, q[0]);
                        Bf16x3::pieces(x[ks][1].x, x[ks][1].y, q[1]);
                        Bf16x3::pieces(x[ks][0].z, x[ks][0].w, q[2]);
                        Bf16x3::pieces(x[ks][1].z, x[ks][1].w, q[3]);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int k = 0; k < kPieces; ++k) A[k][i] = q[i][k];
                    }
                    // products (piece of the rows, piece of the weights) in the order in which the weights' pieces are read
                    auto product = [&](auto chain, auto fresh, const unsigned (&rows)[4], const uint4 (&w)[2]) {
                        constexpr int ch = decltype(chain)::value;
#pragma unroll
                        for (int nt = 0; nt < kNT; ++nt) {
                            const unsigned b0 = (nt & 1) ? w[nt / 2].z : w[nt / 2].x, b1 = (nt & 1) ? w[nt / 2].w : w[nt / 2].y;
                            if (decltype(fresh)::value) Bf16x3::mma_zero(acc[ch][nt], rows, b0, b1);
                            else Bf16x3::mma(acc[ch][nt], rows, b0, b1);
                        }
                    };
                    typedef std::integral_constant<int, 0> lead0;
                    typedef std::integral_constant<int, 1> lead1;
                    typedef std::integral_constant<int, 2> small;
                    const uint4 *w_at = fr + ks * kPieces * 2 * 32;
                    uint4 w[2] = {w_at[128], w_at[160]};                             // third piece
                    if (ks == 0) product(small(), std::true_type(), A[0], w);
                    else product(small(), std::false_type(), A[0], w);
                    w[0] = w_at[64]; w[1] = w_at[96];                                // second
                    product(small(), std::false_type(), A[0], w);
                    product(small(), std::false_type(), A[1], w);
                    w[0] = w_at[0]; w[1] = w_at[32];
                    product(small(), std::false_type(), A[2], w);
                    product(small(), std::false_type(), A[1], w);
                    if (ks == 0) product(lead0(), std::true_type(), A[0], w);
                    else if (ks == 1) product(lead0(), std::false_type(), A[0], w);
                    else if (ks == 2) product(lead1(), std::true_type(), A[0], w);
                    else product(lead1(), std::false_type(), A[0], w);
                }
                const bool live[2] = {first + g < count, first + 8 + g < count};
#pragma unroll
                for (int nt = 0; nt < kNT; ++nt) {
                    const float2 bias = *reinterpret_cast<const float2 *>(bias_s + set * kD + 8 * nt + 2 * t);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float v = ((acc[0][nt][i] + acc[1][nt][i]) + acc[2][nt][i]) + ((i & 1) ? bias.y : bias.x);
                        total[nt][i & 1] += live[i >> 1] ? fmaxf(v, 0.f) : 0.f;
                    }
                }
            }
            __syncwarp();       // the list is read
#pragma unroll
            for (int nt = 0; nt < kNT; ++nt) {
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    total[nt][0] += __shfl_xor_sync(0xffffffffu, total[nt][0], o);
                    total[nt][1] += __shfl_xor_sync(0xffffffffu, total[nt][1], o);
                }
                if (g == nt) *reinterpret_cast<float2 *>(out + set * kD + 8 * nt + 2 * t) = make_float2(total[nt][0], total[nt][1]);
            }
        }
    }
}

bool relu1(const DevMlp &m, int in) {
    return m.n_layers == 1 && m.in_dim == in && m.out_dim == kD && m.act == 0 && m.final_act == 1;
}

}  // namespace

bool pool_split_applicable(const PoolArgs &a) {
    if (a.d != kD || a.F < 1 || a.F > 16) return false;
    for (int i = 0; i < 3; ++i)
        if (!relu1(a.l[i], 2 * kD + a.F)) return false;
    return true;
}

// Below 4096 rows the FMA kernel, whose weights need no splitting, is faster (pooling and head together: 279 nodes x 1
// state 14.1 us there, 14.7 here; 300 x 16: 16.4 and 14.5; 300 x 64: 17.3 and 16.5; 279 x 256: 23.7 and 21.3).
// A warp takes whole items, so the batch costs (items per warp, rounded up) x (tiles per item); a set's last tile is
// half empty on average.
void pool_split_chunks(int n, int B, const DeviceInfo &di, int *chunk_nodes, int *chunks) {
    const long warps = (long)di.sm_count * kWarps;
    double best = 0;
    *chunks = 0;
    if ((long)n * B < 4096) return;
    for (int c = (n + kMaxChunk - 1) / kMaxChunk; c <= std::max(1, n / 16); ++c) {
        const int nodes = (n + c - 1) / c;
        if ((n + nodes - 1) / nodes != c) continue;
        const double cost = (double)(((long)B * c + warps - 1) / warps) * (nodes / (double)kTile + 1.5 + 0.5);
        if (*chunks == 0 || cost < best) { best = cost; *chunks = c; *chunk_nodes = nodes; }
    }
    if (*chunks == 0) { *chunk_nodes = std::min(n, kMaxChunk); *chunks = (n + *chunk_nodes - 1) / *chunk_nodes; }
}

cudaError_t launch_pool_split(const PoolArgs &a, const DeviceInfo &di, cudaStream_t stream, bool overlap) {
    PoolSplitPlan p;
    p.chunk_nodes = a.chunk_nodes;
    p.chunks = a.chunks;
    p.items = a.B * a.chunks;
    const size_t bytes = smem_bytes(p.chunk_nodes);
    if (bytes > (size_t)di.max_smem_optin || p.chunk_nodes > kMaxChunk) return cudaErrorNotSupported;
    auto kern = a.compact.state ? pool_split_kernel<true, true> : (a.F & 3) == 0 ? pool_split_kernel<false, true> : pool_split_kernel<false, false>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (err != cudaSuccess) return err;
    const int grid = std::min(di.sm_count, p.items);
    err = launch_overlapped(overlap, kern, dim3(grid), dim3(kThreads), bytes, stream, a, p);
    count_launch();
    return err;
}

}  // namespace placeto
