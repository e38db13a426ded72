// Soft backward of a LUT layer with its input gradient, on packed fp32 pairs
// (packed.cuh), for fan-in 3 to 6 and any batch size and alignment.
//
// dtheta_a = t_a (1 - t_a) sum_s g_s w_a(x_s) and, per edge (j, i), the term
// g_s dy_j/dx_i(s), from the node's k input rows and its output gradient.  A
// lane owns whole samples: it holds the node's 2^k table values (as packed
// Moebius quads) and 2^k accumulators in registers, element h of every pair
// being the half of the table under top input h, so one packed instruction
// does both halves.
//
// What bounds it: register operand reads of the tree (lut_codes.cu) and, for
// wide layers, the term rows that it writes.  16000 nodes of fan-in 6, forward
// and backward with the input gradient: 1000 samples 329 -> 324 us (315 with
// the packed forward) against a kernel with a sample split over two lanes and
// 12 warps per SM (the tree alone is 13% shorter here, with 8 warps to hide the
// copies behind); batches
// that are no multiple of four, which had a scalar kernel, 907 samples 600 ->
// 325 us, 64000 nodes x 2047 samples 6.01 -> 2.83 ms; fan-in 4 244 -> 167 us,
// fan-in 5 (8000 nodes x 1001) 198 -> 133 us.  One or two samples per loop
// body, 3 or 6 stages: 335-340 us at the first size.
#include "lut_packed.cuh"
#include "packed.cuh"

namespace bitlogic {
namespace {

#ifndef BITLOGIC_PACKED_BLOCKS
#define BITLOGIC_PACKED_BLOCKS 8
#endif
#ifndef BITLOGIC_PACKED_BLOCKS5
#define BITLOGIC_PACKED_BLOCKS5 12
#endif
#ifndef BITLOGIC_PACKED_BLOCKS4
#define BITLOGIC_PACKED_BLOCKS4 16
#endif
#ifndef BITLOGIC_PACKED_STAGES
#define BITLOGIC_PACKED_STAGES 4
#endif
#ifndef BITLOGIC_PACKED_UNROLL
#define BITLOGIC_PACKED_UNROLL 4
#endif
constexpr int kPackedStages = BITLOGIC_PACKED_STAGES;
constexpr int kPackedUnroll = BITLOGIC_PACKED_UNROLL;   // samples of a lane in one loop body
constexpr int kStageSamples = 128;

template <int k>
__host__ __device__ constexpr int packed_blocks() {
    return k >= 6 ? BITLOGIC_PACKED_BLOCKS : k == 5 ? BITLOGIC_PACKED_BLOCKS5 : BITLOGIC_PACKED_BLOCKS4;
}

template <int k>
constexpr int packed_smem() {
    return (kPackedStages * (k + 1) * kStageSamples + (1 << k)) * (int)sizeof(float);
}

// Persistent one-warp blocks: block b takes nodes b, b + G, ... (G blocks, one
// wave) over the whole batch.  The node's input rows and gradient row stream
// through a cp.async ring of 128-sample stages that runs across node
// boundaries; the logits and term positions of the next node are loaded one
// node ahead.  Lane l evaluates samples l, l + 32, l + 64 and l + 96 of a
// stage.  VEC (B % 4 == 0, 16-byte aligned rows): 16-byte copies, which other
// lanes read; otherwise each lane copies its own samples, 4 bytes each.
// TERMS: the gradient is summed from the upstream term rows instead (in
// increasing position, as csr_reduce does), NB rows in flight and the next
// stage's prefetched to L2: with one row at a time the chain of loads bounded
// the kernel (step of 8000 x 8000 nodes, 1024 samples, with layer 1's input
// gradient and fused terms: fan-in 3 204 -> 136 us, 4 254 -> 178, 6 543 -> 372;
// 64000 x 64000 at fan-in 6 3.77 -> 2.61 ms; in a kernel with a sample split
// over two lanes and more warps 140, 178, 372 us and 2.59 ms).  dtheta is
// reduced by a fixed butterfly inside the warp.
template <int k, bool VEC, bool TERMS>
__global__ void __launch_bounds__(32, packed_blocks<k>())
lut_backward_packed_kernel(const float* __restrict__ X, int w_in, long long B, const int* __restrict__ conn,
                           const float* __restrict__ theta, int w, int node, GradSource gs,
                           float* __restrict__ dtheta, float* __restrict__ P, const int* __restrict__ epos,
                           float* __restrict__ dY_out) {
    constexpr int K = 1 << k, H = K / 2, R = TERMS ? k : k + 1, CH = kStageSamples, NS = kPackedStages;
    constexpr int NF = K >= 32 ? K / 32 : 1;   // table entries per lane
    constexpr int SH = K >= 32 ? 0 : 5 - k;    // lanes sharing an entry (K < 32)
    constexpr int NB = k == 4 || k == 5 ? 4 : 8;   // term rows in flight (eight spill registers at fan-in 4 and 5)
    extern __shared__ __align__(16) float smem[];
    const int lane = threadIdx.x;
    float* ring = smem;
    float* sT = smem + NS * R * CH;
    const int G = gridDim.x;
    const int nst = (int)((B + CH - 1) / CH);
    const int e0 = K >= 32 ? lane * NF : lane >> SH;   // this lane's first entry

    // issue stream: stage si of node ji, NS - 1 stages ahead of the compute
    // stream; the rows of the node after ji are loaded ahead
    int ji = blockIdx.x, si = 0, ib = 0;
    int ri[k], rn[k];
    auto rows_of = [&](int j, int (&r)[k]) {
#pragma unroll
        for (int i = 0; i < k; ++i) r[i] = j < w ? __ldg(conn + (long long)j * k + i) : 0;
    };
    auto check = [&](int (&r)[k]) {   // when the node is reached: checking at the load would wait for it
        bool bad = false;
#pragma unroll
        for (int i = 0; i < k; ++i)
            if ((unsigned)r[i] >= (unsigned)w_in) { bad = true; r[i] = 0; }
        if (bad && lane == 0) flag_index_error();
    };
    rows_of(ji, ri);
    check(ri);
    rows_of(ji + G, rn);
    const float* gi = TERMS ? nullptr : gs.dY + (long long)(ji / gs.group) * B;
    auto issue = [&]() {
        if (ji < w) {
            const long long s0 = (long long)si * CH;
            if constexpr (VEC) {
                const long long s4 = s0 + 4 * lane;
                if (s4 < B) {
                    float* buf = ring + ib * (R * CH) + 4 * lane;
#pragma unroll
                    for (int r = 0; r < k; ++r) cp_async16(buf + r * CH, X + (long long)ri[r] * B + s4);
                    if constexpr (!TERMS) cp_async16(buf + k * CH, gi + s4);
                }
            } else {
                float* buf = ring + ib * (R * CH) + lane;
                const int left = (int)min((long long)CH, B - s0) - lane;   // this lane's samples: left > 32 c
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float* row = (r < k ? X + (long long)ri[r < k ? r : 0] * B : gi) + s0 + lane;
#pragma unroll
                    for (int c = 0; c < CH / 32; ++c)
                        if (left > 32 * c) cp_async4(buf + r * CH + 32 * c, row + 32 * c);
                }
            }
            if (++si == nst) {
                si = 0;
                ji += G;
                if constexpr (!TERMS)
                    if (ji < w) gi = gs.dY + (long long)(ji / gs.group) * B;
#pragma unroll
                for (int i = 0; i < k; ++i) ri[i] = rn[i];
                check(ri);
                rows_of(ji + G, rn);
            }
        }
        cp_async_commit();
        ib = (ib + 1 == NS) ? 0 : ib + 1;
    };
    // logits and term rows of the warp's next node
    float thn[NF];
    int posn = 0, t0n = 0, t1n = 0;
    auto term_id = [&](int e, int end) {
        int id = -1;
        if (e < end) {
            id = gs.edge ? __ldg(gs.edge + e) : e;
            if ((unsigned)id >= (unsigned)gs.n_edges) {
                flag_index_error();
                id = -1;
            }
        }
        return id;
    };
    auto ahead = [&](int j) {
        if (j < w) {
            if constexpr (TERMS) {
                t0n = __ldg(gs.off + j);
                t1n = __ldg(gs.off + j + 1);
            }
#pragma unroll
            for (int i = 0; i < NF; ++i) thn[i] = __ldg(theta + (long long)j * K + e0 + i);
            if (epos && lane < k) posn = __ldg(epos + (long long)j * k + lane);
        }
    };
#pragma unroll
    for (int i = 0; i < NF; ++i) thn[i] = 0.f;
    ahead(blockIdx.x);
#pragma unroll 1
    for (int i = 0; i < NS - 1; ++i) issue();

    int rb = 0;
#pragma unroll 1
    for (int j = blockIdx.x; j < w; j += G) {
        float sg[NF];   // sigmoids of this lane's entries, for the epilogue
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            sg[i] = sigmoidf(thn[i]);
            const int a = e0 + i;   // the table's halves interleaved, as packed_quads reads them
            if ((lane & ((1 << SH) - 1)) == 0)
                sT[2 * (a & (H - 1)) + (a >> (k - 1))] = table_value(thn[i], sg[i], node);
        }
        float* pst[k];
#pragma unroll
        for (int i = 0; i < k; ++i) {
            long long row = (long long)j * k + i;
            if (epos) {
                const int r = __shfl_sync(0xffffffffu, posn, i);
                if (r >= 0 && (long long)r < (long long)w * k) row = r;
                else if (lane == 0) flag_index_error();   // stored at its own row, inside the buffer
            }
            pst[i] = P + row * B + lane;
        }
        // the node's term positions, and row ids: lane u that of position t0 + u
        // (-1 past the end or out of range)
        int t0 = 0, t1 = 0, ids = -1;
        if constexpr (TERMS) {
            t0 = t0n;
            t1 = t1n;
            if (t0 < 0 || t1 < t0 || t1 > gs.n_edges) {
                if (lane == 0) flag_index_error();
                t0 = t1 = 0;
            }
            ids = term_id(t0 + lane, t1);
        }
        __syncwarp();
        f32x2 cq[H], acc[H];
        packed_quads<k>(sT, cq);
#pragma unroll
        for (int a = 0; a < H; ++a) acc[a] = 0ull;
        ahead(j + G);
#pragma unroll 1
        for (int sc = 0; sc < nst; ++sc) {
            issue();
            cp_async_wait<NS - 1>();
            if constexpr (VEC) __syncwarp();   // the lanes' copies are visible to each other
            const float* buf = ring + rb * (R * CH) + lane;
            const long long s0 = (long long)sc * CH;
            float gt[TERMS ? CH / 32 : 1];
            if constexpr (TERMS) {
#pragma unroll
                for (int c = 0; c < CH / 32; ++c) gt[c] = 0.f;
                // loads of NB rows are issued before the first add (samples past
                // the batch read its first ones, unused; past the end row 0)
                long long at[CH / 32];
#pragma unroll
                for (int c = 0; c < CH / 32; ++c) at[c] = s0 + 32 * c + lane < B ? s0 + 32 * c + lane : 0;
#pragma unroll 1
                for (int q = 0; q < t1 - t0; q += NB) {
                    if (q > 0 && q % 32 == 0) ids = term_id(t0 + q + lane, t1);
                    float v[NB][CH / 32];
                    bool add[NB];
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        const int id = __shfl_sync(0xffffffffu, ids, (q + u) & 31);
                        add[u] = id >= 0;
                        const float* row = gs.terms + (long long)max(id, 0) * B;
#pragma unroll
                        for (int c = 0; c < CH / 32; ++c) v[u][c] = __ldg(row + at[c]);
                    }
#pragma unroll
                    for (int u = 0; u < NB; ++u)
#pragma unroll
                        for (int c = 0; c < CH / 32; ++c)
                            if (add[u]) gt[c] += v[u][c];
                }
                if (t1 - t0 > 32) ids = term_id(t0 + lane, t1);   // the first ones again, for the next stage
                if (ids >= 0) {   // the next stage's rows on their way to L2, a row per lane
#pragma unroll
                    for (int c = 0; c < CH / 32; ++c)
                        if (s0 + CH + 32 * c < B) prefetch_l2(gs.terms + (long long)ids * B + s0 + CH + 32 * c);
                }
            }
            auto sample = [&](int c, bool in) {
                float x[k], dx[k];
#pragma unroll
                for (int i = 0; i < k; ++i) x[i] = in ? buf[i * CH + 32 * c] : 0.f;
                float g;
                if constexpr (TERMS) g = in ? gt[c] : 0.f;
                else g = in ? buf[k * CH + 32 * c] : 0.f;
                node_sample2<k>(cq, x, g, dx, acc);
                if (in) {
#pragma unroll
                    for (int i = 0; i < k; ++i) pst[i][s0 + 32 * c] = dx[i];
                    if (dY_out) dY_out[(long long)j * B + s0 + 32 * c + lane] = g;
                }
            };
            constexpr int kUnroll = TERMS ? CH / 32 : kPackedUnroll, kRagged = TERMS ? CH / 32 : 1;
            if (s0 + CH <= B) {
#pragma unroll kUnroll
                for (int c = 0; c < CH / 32; ++c) sample(c, true);
            } else {
#pragma unroll kRagged
                for (int c = 0; c < CH / 32; ++c) {
                    if (!TERMS && s0 + 32 * c >= B) break;   // warp-uniform
                    sample(c, s0 + 32 * c + lane < B);
                }
            }
            if constexpr (VEC) __syncwarp();   // every lane has read the slot that the next issue refills
            rb = (rb + 1 == NS) ? 0 : rb + 1;
        }
        __syncwarp();   // the table is read before the next node rewrites it
        float sum[K];
#pragma unroll
        for (int a = 0; a < H; ++a) unpack2(acc[a], sum[a], sum[a + H]);
        warp_reduce_scatter<K, 16>(sum, lane);
        if ((lane & ((1 << SH) - 1)) == 0) {
#pragma unroll
            for (int i = 0; i < NF; ++i) dtheta[(long long)j * K + e0 + i] = sg[i] * (1.0f - sg[i]) * sum[i];
        }
    }
    cp_async_wait<0>();
}

template <int k>
int launch_packed(const float* X, int w_in, long long B, const int* conn, const float* theta, int w, int node,
                  const GradSource& gs, float* dtheta, float* P, const int* epos, float* dY_out, cudaStream_t st) {
    constexpr int smem = packed_smem<k>();
    const bool vec = B % 4 == 0 && aligned16(X) && (gs.terms || aligned16(gs.dY));
    auto kern = gs.terms ? (vec ? lut_backward_packed_kernel<k, true, true> : lut_backward_packed_kernel<k, false, true>)
                         : (vec ? lut_backward_packed_kernel<k, true, false>
                                : lut_backward_packed_kernel<k, false, false>);
    static_assert(smem <= 40 * 1024, "fits the default limit");
    const long long resident = (long long)sm_count() * packed_blocks<k>();
    kern<<<(unsigned)(w < resident ? w : resident), 32, smem, st>>>(X, w_in, B, conn, theta, w, node, gs, dtheta, P,
                                                                   epos, dY_out);
    return launch_status();
}

}  // namespace

int launch_backward_packed(int k, const float* X, int w_in, long long B, const int* conn, const float* theta, int w,
                           int node, const GradSource& gs, float* dtheta, float* P, const int* epos, float* dY_out,
                           cudaStream_t st) {
    switch (k) {
        case 3: return launch_packed<3>(X, w_in, B, conn, theta, w, node, gs, dtheta, P, epos, dY_out, st);
        case 4: return launch_packed<4>(X, w_in, B, conn, theta, w, node, gs, dtheta, P, epos, dY_out, st);
        case 5: return launch_packed<5>(X, w_in, B, conn, theta, w, node, gs, dtheta, P, epos, dY_out, st);
        case 6: return launch_packed<6>(X, w_in, B, conn, theta, w, node, gs, dtheta, P, epos, dY_out, st);
        default: return BITLOGIC_ERR_FANIN;
    }
}

}  // namespace bitlogic

BITLOGIC_ERROR_READER(lut_packed)
