// Layer 2 of the training step on corner codes of layer 1.
//
// Layer 1 reads binary wires, so its output is the table entry that the
// wires select (§2: a soft node on binary inputs returns its table entry):
// y1[i][s] = t_i[a_i(s)], a_i(s) < 2^k1.  These kernels keep the index a_i(s),
// one byte per node and sample, and the table t_i instead of the fp32 rows:
//
//  * codes_forward_kernel (layer 1): the codes and the tables;
//  * coded_forward_kernel (layer 2): gathers its k code rows, a quarter of
//    the bytes of fp32 rows, and reads each input from the k tables in shared
//    memory: the same fp32 values bit for bit;
//  * coded_backward_kernel (layer 2): dtheta as in the fp32 kernels, and the
//    input gradient as layer 1 needs it.  Layer 1's table gradient is
//      dtheta1_i[a] = t'_i[a] sum over s with a_i(s) = a of dL/dy1_i[s],
//    and dL/dy1_i is the sum of its consumer edges' terms, so each edge is
//    reduced here to its 2^k1 corner sums H_e[a] = sum over s with a_i(s) = a
//    of term_e[s]: 2^k1 values per edge leave the chip instead of B;
//  * corner_reduce_kernel (layer 1): adds the corner sums of a node's
//    consumer edges and applies the slope of the sigmoid.
//
// Codes are stored as 4 a (the byte offset into an fp32 table), rows padded
// with zeros to whole 128-sample blocks.  Readers mask them to the offsets of
// a table of 2^k1 entries, so no byte value leads outside it.
#include <type_traits>

#include "common.cuh"
#include "packed.cuh"

namespace bitlogic {
namespace {

#ifndef BITLOGIC_CODED_FWD_BLOCKS
#define BITLOGIC_CODED_FWD_BLOCKS 16
#endif
#ifndef BITLOGIC_CODED_BWD_BLOCKS
#define BITLOGIC_CODED_BWD_BLOCKS 8
#endif
#ifndef BITLOGIC_CODED_BWD_BLOCKS_SMALL
#define BITLOGIC_CODED_BWD_BLOCKS_SMALL 12
#endif
constexpr int kCodesWarps = 8;

// ------------------------------------------------- layer 1: codes, tables --

// A warp per node and range of 1024-sample blocks; lanes and wire words as in
// lut_forward_bits_kernel.
template <int k>
__global__ void __launch_bounds__(kCodesWarps * 32)
codes_forward_kernel(const uint32_t* __restrict__ X, int w_in, long long words, const int* __restrict__ conn,
                     const float* __restrict__ theta, int w, int node, uint8_t* __restrict__ codes, long long stride,
                     float* __restrict__ table, long long chunk_blocks) {
    constexpr int K = 1 << k;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = blockIdx.x * kCodesWarps + warp;
    if (j >= w) return;   // warp-uniform
    const uint32_t* xr[k];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < k; ++i) {
        int c = __ldg(conn + (long long)j * k + i);
        if ((unsigned)c >= (unsigned)w_in) {
            bad = true;
            c = 0;
        }
        xr[i] = X + (long long)c * words + lane;
    }
    if (bad && lane == 0) flag_index_error();
    if (blockIdx.y == 0) {
#pragma unroll
        for (int a = 0; a < K; a += 32) {
            if (a + lane < K) {
                const float th = __ldg(theta + (long long)j * K + a + lane);
                table[(long long)j * K + a + lane] = table_value(th, sigmoidf(th), node);
            }
        }
    }
    const long long nblk = words / 32;
    const long long b0 = (long long)blockIdx.y * chunk_blocks;
    const long long b1 = min(nblk, b0 + chunk_blocks);
    uint8_t* out = codes + (long long)j * stride;
    for (long long blk = b0; blk < b1; ++blk) {
        uint32_t wv[k];
#pragma unroll
        for (int i = 0; i < k; ++i) wv[i] = __ldg(xr[i] + blk * 32);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const long long s4 = blk * kBitBlock + 128 * r + 4 * lane;
            uint32_t v = (wv[k - 1] >> r) & 0x01010101u;
#pragma unroll
            for (int i = k - 2; i >= 0; --i) v = (v << 1) | ((wv[i] >> r) & 0x01010101u);
            if (s4 < stride) *reinterpret_cast<uint32_t*>(out + s4) = v << 2;
        }
    }
}

// fp32 rows from codes and tables (for callers that want the activations).
__global__ void __launch_bounds__(256)
codes_decode_kernel(const uint8_t* __restrict__ codes, long long stride, const float* __restrict__ table, int K, int w,
                    long long B, float* __restrict__ Y) {
    const int j = blockIdx.x;
    for (long long s = threadIdx.x; s < B; s += 256) {
        const int a = (__ldg(codes + (long long)j * stride + s) >> 2) & (K - 1);
        Y[(long long)j * B + s] = __ldg(table + (long long)j * K + a);
    }
}

// ------------------------------------------------------ shared node pieces --

// Copies the k input nodes' tables (2^k1 floats each; cin: lane i < k holds
// input i) to shared memory, 64 floats apart, asynchronously: 16-byte pieces,
// or one 8-byte piece per table when k1 == 1.
template <int k>
__device__ __forceinline__ void copy_tables(float* sTab, const float* __restrict__ table1, int k1, int cin, int lane) {
    const int lg = k1 >= 2 ? k1 - 2 : 0;   // log2 of the pieces per table
    const int n = k << lg;
    for (int q0 = 0; q0 < n; q0 += 32) {
        const int q = q0 + lane;
        const int i = q >> lg;
        const int c = __shfl_sync(0xffffffffu, cin, i < k ? i : 0);
        if (q < n) {
            const int piece = q & ((1 << lg) - 1);
            if (k1 >= 2) {
                cp_async16(sTab + 64 * i + 4 * piece, table1 + ((long long)c << k1) + 4 * piece);
            } else {
                const unsigned s = (unsigned)__cvta_generic_to_shared(sTab + 64 * i);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(table1 + 2ll * c) : "memory");
            }
        }
    }
    cp_async_commit();
}

// Connectivity of node j, slot i on lane i.  The value is loaded a node ahead
// and checked when it is used (checking it here would wait for the load).
template <int k>
__device__ __forceinline__ int load_inputs(const int* __restrict__ conn, int j, int w, int lane) {
    return j < w && lane < k ? __ldg(conn + (long long)j * k + lane) : 0;
}
__device__ __forceinline__ int checked_input(int c, int w_in) {
    if ((unsigned)c < (unsigned)w_in) return c;
    flag_index_error();
    return 0;
}

// Shared-memory accesses by 32-bit address.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float lds(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];\n" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(a), "f"(v) : "memory");
}

// Address of the entry that code c of the four in v selects, in a table at the
// 256-byte aligned address base: the code is the address's low byte, so one
// byte permute builds the address.
__device__ __forceinline__ uint32_t entry_addr(uint32_t v, int c, uint32_t base) {
    return __byte_perm(v, base, 0x7650u + (unsigned)c);
}

// Bits of four codes that lie inside a table of 2^k1 entries.
__device__ __forceinline__ uint32_t code_mask(int k1) { return (((1u << k1) - 1u) << 2) * 0x01010101u; }

// A lane's samples in a 128-sample stage: nc consecutive ones from sample `at`
// of the stage, the bytes of code word `word` from bit `shift` on.  A full
// stage has one word and four samples per lane.  In the TAIL form of the
// layer-2 kernels a last stage with at most 64 (32) samples left puts two
// (four) lanes on a word, so that a half (a quarter) of the steps do for it.
// The form is taken for small batches (short_tail): its second sample loop
// costs the compiler's schedule of the first one more (4.05 -> 4.60 ms for the
// step at 128000 nodes x 2048 samples, which has no tail) than it saves when
// there are several full stages.  30000 x 30000 nodes, fan-in 6, per step:
// 32 samples 187 (per-edge terms) -> 165 us, 64 samples 188 -> 172 us; without
// it 64 samples took about as long as 128 (190 us).
struct LaneSamples {
    int word, shift, at, nc;
};
__device__ __forceinline__ LaneSamples lane_samples(long long left, int lane) {
    const int lg = left > 64 ? 0 : left > 32 ? 1 : 2;   // lanes per word, as a power of two
    const int word = lane & ((32 >> lg) - 1), part = lane >> (5 - lg), nc = 4 >> lg;
    return {word, 8 * nc * part, 4 * word + nc * part, nc};
}

inline bool short_tail(long long B) { return B <= 192 && B % 128 != 0 && B % 128 <= 64; }

// ------------------------------------------------------------ layer 2 value --

// Persistent one-warp blocks, a node over the whole batch; lane = 4
// consecutive samples of a 128-sample stage, the code words of the next stage
// (or node) and the next node's tables in flight.  The table's two halves
// under the top input are evaluated together on packed pairs, with the
// expressions of the fp32 forward (8-entry Moebius subtables under lerps), so
// the results equal it bit for bit.  At 128000 nodes of fan-in 6 and 2048
// samples 0.90 ms against 0.985 ms on fp32 rows, which waits for DRAM (6.9 GB
// at 7 TB/s); here 2.5 GB move, and neither the FP32 pipe (56% active) nor
// issue (51%) is full: the tree's register operand reads and the chain from
// code word to table entry are what is left.  12 or 20 blocks per SM: 1 and 9%
// slower steps.
template <int k, bool TAIL>
__global__ void __launch_bounds__(32, BITLOGIC_CODED_FWD_BLOCKS)
coded_forward_kernel(const uint8_t* __restrict__ codes, long long stride, const float* __restrict__ table1, int w_in,
                     int k1, long long B, const int* __restrict__ conn, const float* __restrict__ theta, int w,
                     int node, float* __restrict__ Y, bool vec) {
    constexpr int K = 1 << k, H = K / 2, NF = K >= 32 ? K / 32 : 1;
    extern __shared__ __align__(256) float smem[];
    const int lane = threadIdx.x;
    float* tab = smem;                 // [2][k][64]: this node's input tables and the next node's
    float* sT = smem + 2 * k * 64;     // [K]
    const int G = gridDim.x, nst = (int)((B + 127) / 128);
    const int e0 = NF * lane;
    const uint32_t cmask = code_mask(k1);

    const uint32_t* src[k];
    uint32_t cw[k];
    float th[NF];
    int cin = checked_input(load_inputs<k>(conn, blockIdx.x, w, lane), w_in), buf = 0;
    auto ahead = [&](int j) {
#pragma unroll
        for (int i = 0; i < NF; ++i) th[i] = (j < w && e0 + i < K) ? __ldg(theta + (long long)j * K + e0 + i) : 0.f;
    };
    const LaneSamples tail = lane_samples(B - 128ll * (nst - 1), lane);   // of the last stage
    // code words of stage st of the current row pointers
    auto words = [&](uint32_t (&c)[k], int st) {
        const int at = 32 * st + (!TAIL ? 0 : st + 1 == nst ? tail.word : lane);
#pragma unroll
        for (int i = 0; i < k; ++i) c[i] = __ldg(src[i] + at);
    };
    // the same of the first stage of the node whose inputs are in cin; then
    // cin moves on to node j
    auto first_words = [&](uint32_t (&c)[k], int j) {
#pragma unroll
        for (int i = 0; i < k; ++i)
            src[i] = reinterpret_cast<const uint32_t*>(codes + (long long)__shfl_sync(0xffffffffu, cin, i) * stride) +
                     (TAIL ? 0 : lane);
        words(c, 0);
        cin = load_inputs<k>(conn, j, w, lane);
    };
    ahead(blockIdx.x);
    copy_tables<k>(tab, table1, k1, cin, lane);
    first_words(cw, blockIdx.x + G);
#pragma unroll
    for (int i = 0; i < k; ++i) cw[i] &= cmask;
#pragma unroll 1
    for (int j = blockIdx.x; j < w; j += G) {
#pragma unroll
        for (int i = 0; i < NF; ++i)
            if (e0 + i < K) sT[e0 + i] = table_value(th[i], sigmoidf(th[i]), node);
        __syncwarp();
        // lane m: subtable m into its subset differences, stored with the
        // table's halves interleaved
        float cs[8];
        if (lane < K / 8) {
#pragma unroll
            for (int a = 0; a < 8; ++a) cs[a] = sT[8 * lane + a];
#pragma unroll
            for (int b = 1; b < 8; b <<= 1)
#pragma unroll
                for (int a = 0; a < 8; ++a)
                    if (a & b) cs[a] -= cs[a ^ b];
        }
        __syncwarp();
        if (lane < K / 8) {
#pragma unroll
            for (int a = 0; a < 8; ++a) sT[2 * ((8 * lane + a) & (H - 1)) + lane / (H / 8)] = cs[a];
        }
        __syncwarp();
        f32x2 cf[H];
#pragma unroll
        for (int a = 0; a < H; a += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(sT + 2 * a);
            cf[a] = v.x;
            cf[a + 1] = v.y;
        }
        ahead(j + G);
        cp_async_wait<0>();
        __syncwarp();   // the node's tables are in place; the other buffer's readers are done
        const uint32_t sTab = smem_addr(tab + buf * (k * 64));
        buf ^= 1;
        if (j + G < w) {
            cin = checked_input(cin, w_in);
            copy_tables<k>(tab + buf * (k * 64), table1, k1, cin, lane);
        }
        float* yr = Y + (long long)j * B;
#pragma unroll 1
        for (int st = 0; st < nst; ++st) {
            uint32_t cn[k];   // the next stage's words, or the next node's first
            if (st + 1 < nst) {
#pragma unroll
                for (int i = 0; i < k; ++i) cn[i] = 0u;
                words(cn, st + 1);
            } else {
                first_words(cn, j + 2 * G);   // past the last node: row 0, unused
            }
            auto value = [&](int c) {   // the node's value at sample c of the lane's words
                f32x2 x[k - 1];
#pragma unroll
                for (int i = 0; i < k - 1; ++i) {
                    const float v = lds(entry_addr(cw[i], c, sTab) + i * 256u);
                    x[i] = pack2(v, v);
                }
                const float xt = lds(entry_addr(cw[k - 1], c, sTab) + (k - 1) * 256u);
                float lo, hi;
                unpack2(fwd_tree2<k - 2, 0>(cf, x), lo, hi);
                return fmaf(xt, hi - lo, lo);
            };
            if (!TAIL || st + 1 < nst) {
                float o[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) o[c] = value(c);
                const long long s4 = 128ll * st + 4 * lane;
                if (vec) {
                    if (s4 < B) *reinterpret_cast<float4*>(yr + s4) = make_float4(o[0], o[1], o[2], o[3]);
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (s4 + c < B) yr[s4 + c] = o[c];
                }
            } else {
#pragma unroll
                for (int i = 0; i < k; ++i) cw[i] >>= tail.shift;
                const long long s = 128ll * st + tail.at;
#pragma unroll 1
                for (int c = 0; c < tail.nc; ++c) {
                    const float v = value(c);
                    if (s + c < B) yr[s + c] = v;
                }
            }
#pragma unroll
            for (int i = 0; i < k; ++i) cw[i] = cn[i] & cmask;   // masked only now: nothing waits for the loads before
        }
    }
    cp_async_wait<0>();
}

// ------------------------------------------------------- layer 2 backward --
//
// One warp per node (persistent one-warp blocks); a lane owns whole samples, 4
// consecutive ones of each 128-sample stage, with the node's table (packed
// Moebius quads) and its 2^k accumulators in registers.
//
// Corner sums live in shared memory as columns: 16 per slot, column p shared
// by the lanes p and p + 16 (h = lane >> 4).  Those two take the slots in
// different orders, lane h starting k/2 slots later (slot_of), and a sample
// adds its terms in steps of k/2 slots: in one step the two lanes are at
// different slots, so no two lanes of an instruction touch one word, and a
// warp barrier separates the steps.  Slot s < 2 (k/2) is half s / (k/2) of
// the rows of array s % (k/2), [64][2][16] words, so the 32 lanes fall into
// the 32 banks whatever their corners (for odd k the last slot has an array
// of its own and meets a 2-way conflict).  For k = 6 that is 24 KB per warp
// and 8 warps per SM, which is also what the registers allow.
//
// The order is the lane's alone: its table is permuted when it is loaded and
// its dtheta permuted back when it is reduced.
//
// What bounds it: register operand reads of the tree's multiply-adds (an
// accumulation with three distinct operands takes 2.45 cycles packed and 1.3
// to 1.6 scalar on an SM quarter, whatever the number of warps).  The tree
// alone takes 2.3 ms at 128000 nodes x 2048 samples in this form, 2.6-2.7 ms
// with a sample split over two lanes (scalar or packed), which repeats the
// per-sample work; the pipe is 58% and issue 46% active (8000 nodes x 1024).
// Measured there: 2.78 ms against 2.76 ms for the fp32-row backward, which in
// addition writes 6.3 GB of per-edge terms that the layer-1 backward reads back
// (1.07 ms; the corner reduction takes 0.05 ms).  Step, with the forward on
// codes: 5.20 -> 3.99 ms; 64000 nodes x 1024 1.363 -> 1.143 ms; 8000 x 1024
// 0.197 -> 0.166 ms.  Forms with a sample split over lanes, 8 warps with own
// columns (two samples in flight) and 12 warps with shared columns: steps of
// 4.69 and 5.16 ms at the first size.

template <int k>
struct Order {
    static constexpr int C = k / 2, K = 1 << k, H = K / 2;
    static constexpr int kArrays = (k + 1) / 2;
    static constexpr int kCopy = K + 4;   // floats of one table copy (padded against bank conflicts)
    // slot of tree input m for lanes of half h
    static __device__ __forceinline__ int slot_of(int h, int m) {
        const int s = m + (h ? C : 0);
        return s >= k ? s - k : s;
    }
    // byte offset of slot s's columns inside a row of array 0
    static __device__ __forceinline__ int column_of(int s) {
        return s < 2 * C ? (s % C) * (64 * 128) + (s / C) * 64 : C * (64 * 128);
    }
    // table index in slot order of index v in the tree order of half h
    static __device__ __forceinline__ int to_slots(int h, int v) {
        return h ? ((v << C) | (v >> (k - C))) & (K - 1) : v;   // tree input m is slot m + C modulo k
    }
    static __device__ __forceinline__ int to_tree(int h, int a) {
        return h ? ((a >> C) | (a << (k - C))) & (K - 1) : a;
    }
};

// Sum over the 16 lanes of a half-warp of N >= 16 values per lane; lane p of
// the half keeps those of index p N / 16 + i.
template <int N, int O, int M>
__device__ __forceinline__ void half_reduce(float (&v)[M], int lane) {
    if constexpr (O > 0) {
        const bool up = (lane & O) != 0;
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const float send = up ? v[i] : v[i + N / 2];
            const float keep = up ? v[i + N / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        }
        half_reduce<N / 2, O / 2>(v, lane);
    }
}

__device__ __forceinline__ float sum4(const float4& v) { return (v.x + v.y) + (v.z + v.w); }

// Column sums of row `code` of an array [64][2][16]; clears the row.
// Lane-rotated 16-byte accesses: any eight consecutive lanes touch all 32
// banks.  Every sum has one order whatever the lane's rotation.
__device__ __forceinline__ void take_row(float* arr, int code, int lane, float (&s)[2]) {
    float4* row = reinterpret_cast<float4*>(arr + 32 * code);
    const int t = (lane >> 2) & 1;
    float r[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int f = 4 * ((i + t) & 1);
        float4 v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            v[e] = row[f + ((lane + e) & 3)];
            row[f + ((lane + e) & 3)] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        r[i] = (sum4(v[0]) + sum4(v[2])) + (sum4(v[1]) + sum4(v[3]));
    }
    s[0] = t ? r[1] : r[0];
    s[1] = t ? r[0] : r[1];
}

template <int k>
__host__ __device__ constexpr int coded_bwd_blocks() {
    return k >= 5 ? BITLOGIC_CODED_BWD_BLOCKS : BITLOGIC_CODED_BWD_BLOCKS_SMALL;
}

// Shared memory: the corner arrays (also scratch for the table copies and the
// dtheta exchange, between nodes), then the input tables, 64 floats each.
template <int k>
constexpr int coded_bwd_smem() {
    return (Order<k>::kArrays * 64 * 32 + k * 64) * (int)sizeof(float);
}

// Samples past the batch in the last stage have a zero output gradient and
// code 0 (the rows' padding), so their terms are zeros, unless the node's
// table or entry 0 of an input table is NaN (a NaN logit): for such a node
// they take the codes of the batch's last sample instead, whose own terms are
// NaN wherever theirs are, so that a NaN reaches only the sums of samples that
// meet it.  FORM: whole stages (no such samples), the last stage partly
// filled, or short_tail.
enum { kWhole, kRagged, kShort };

template <int k, int FORM>
__global__ void __launch_bounds__(32, coded_bwd_blocks<k>())
coded_backward_kernel(const uint8_t* __restrict__ codes, long long stride, const float* __restrict__ table1, int w_in,
                      int k1, long long B, const int* __restrict__ conn, const float* __restrict__ theta, int w,
                      int node, const float* __restrict__ dY, int group, bool vec, float* __restrict__ dtheta,
                      float* __restrict__ corner, const int* __restrict__ epos, float* __restrict__ theta_read) {
    using O = Order<k>;
    constexpr bool TAIL = FORM == kShort;
    constexpr int C = O::C, K = O::K, H = O::H;
    constexpr int NF = K >= 32 ? K / 32 : 1;
    extern __shared__ __align__(256) float smem[];
    const int lane = threadIdx.x, h = lane >> 4, p = lane & 15;
    const int K1 = 1 << k1;
    float* sTab = smem + O::kArrays * 64 * 32;
    const int G = gridDim.x, nst = (int)((B + 127) / 128);
    const int e0 = NF * lane;
    const uint32_t cmask = code_mask(k1);

    // tree input m: address of its table (tb + td), and of its column in row 0
    // less 32 times that address: the column's word of the corner at table
    // address e (corner a: e = table + 4 a, row of 128 bytes) is then 32 e + cb.
    // For even k these are one register per step plus compile-time offsets.
    constexpr int NB = k % 2 == 0 ? 2 : k;   // bases kept
    uint32_t tb[NB], cb[NB];
#pragma unroll
    for (int m = 0; m < NB; ++m) {
        const int s = O::slot_of(h, k % 2 == 0 ? m * C : m);
        tb[m] = smem_addr(sTab + 64 * s);
        cb[m] = smem_addr(smem + p) + (uint32_t)O::column_of(s) - 32u * tb[m];
    }
    auto base = [](int m) { return k % 2 == 0 ? m / C : m; };
    auto table_off = [](int m) { return k % 2 == 0 ? (uint32_t)(m % C) * 256u : 0u; };
    auto column_off = [](int m) { return k % 2 == 0 ? (uint32_t)(m % C) * (64u * 128u) : 0u; };

    const uint32_t* src[k];
    const float* gsrc = nullptr;
    uint32_t cw[k];
    float4 g4;
    float th[NF];
    int cin = load_inputs<k>(conn, blockIdx.x, w, lane), posn = 0;
    auto ahead = [&](int j) {
#pragma unroll
        for (int i = 0; i < NF; ++i) th[i] = (j < w && e0 + i < K) ? __ldg(theta + (long long)j * K + e0 + i) : 0.f;
    };
    const LaneSamples tail = lane_samples(B - 128ll * (nst - 1), lane);   // of the last stage
    // output gradient of the lane's samples of stage st (with TAIL those past
    // nc are not evaluated), and with TAIL their code words
    auto load_g = [&](int st) {
        const bool last = TAIL && st + 1 == nst;
        const long long s = 128ll * st + (last ? tail.at : 4 * lane);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec && !last) {
            if (s < B) v = __ldg(reinterpret_cast<const float4*>(gsrc + s));
        } else {
            if (s < B) v.x = __ldg(gsrc + s);
            if (s + 1 < B) v.y = __ldg(gsrc + s + 1);
            if (s + 2 < B) v.z = __ldg(gsrc + s + 2);
            if (s + 3 < B) v.w = __ldg(gsrc + s + 3);
        }
        return v;
    };
    auto word_of = [&](int st) { return st + 1 == nst ? tail.word : lane; };   // TAIL
    auto start = [&](int j) {   // tables, row pointers and first loads of node j
        cin = checked_input(cin, w_in);
        copy_tables<k>(sTab, table1, k1, cin, lane);
        gsrc = dY + (long long)(j / group) * B;
#pragma unroll
        for (int m = 0; m < k; ++m) {
            const int c = __shfl_sync(0xffffffffu, cin, O::slot_of(h, m));
            src[m] = reinterpret_cast<const uint32_t*>(codes + (long long)c * stride) + (TAIL ? 0 : lane);
            cw[m] = __ldg(src[m] + (TAIL ? word_of(0) : 0));
        }
        g4 = load_g(0);
        cin = load_inputs<k>(conn, j + G, w, lane);
    };
    // inputs of sample i of the code words in cw, in tree order, and the table
    // addresses that they came from
    float x[k];
    uint32_t ea[k];
    auto look = [&](int i) {
#pragma unroll
        for (int m = 0; m < k; ++m) {
            ea[m] = entry_addr(cw[m], i, tb[base(m)]);
            x[m] = lds(ea[m] + table_off(m));
        }
    };
    // the codes of the last sample for those past the batch, once cw holds the
    // last stage's, and their first lookup again
    auto fill = [&] {
        const int last = (int)(B - 1 - 128ll * (nst - 1)), nc = TAIL ? tail.nc : 4;
        const int part = (last & 3) >> (TAIL ? nc - 1 : 2);   // nc 1 or 2 with TAIL
        const int owner = (last >> 2) + part * (8 * nc), r = last & (nc - 1);   // its lane and byte there
        const bool past = (TAIL ? tail.at : 4 * lane) + nc > last;
        const int from = past ? owner : lane;
        const uint32_t bytes = !past || r == 3 ? 0x3210u : r == 2 ? 0x2210u : r == 1 ? 0x1110u : 0u;
        uint32_t v[k];   // by slot: the two lane halves hold the slots in different orders
#pragma unroll
        for (int i = 0; i < k; ++i) {
            v[i] = __shfl_sync(0xffffffffu, h ? cw[(i + k - C) % k] : cw[i], from);
            v[i] = __byte_perm(v[i], 0u, bytes);
        }
#pragma unroll
        for (int m = 0; m < k; ++m) cw[m] = h ? v[(m + C) % k] : v[m];
        look(0);
    };
    ahead(blockIdx.x);
    start(blockIdx.x);
    for (int q = lane; q < O::kArrays * 64 * 32; q += 32) smem[q] = 0.f;
#pragma unroll 1
    for (int j = blockIdx.x; j < w; j += G) {
        if (epos && lane < k) posn = __ldg(epos + (long long)j * k + lane);
        // table copies of the two lane halves, in their orders
        float sg[NF];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            sg[i] = sigmoidf(th[i]);
            const int a = e0 + i;
            if (a < K) {   // the table's halves interleaved, as packed_quads reads them
#pragma unroll
                for (int ah = 0; ah < 2; ++ah) {
                    const int v = O::to_tree(ah, a);
                    smem[ah * O::kCopy + 2 * (v & (H - 1)) + (v >> (k - 1))] = table_value(th[i], sg[i], node);
                }
            }
        }
        __syncwarp();
        f32x2 cp[H], acc[H];
        packed_quads<k>(smem + h * O::kCopy, cp);
#pragma unroll
        for (int a = 0; a < H; ++a) acc[a] = 0ull;
        __syncwarp();
        for (int q = lane; q < 2 * O::kCopy; q += 32) smem[q] = 0.f;
        if (FORM != kWhole && theta_read) {
#pragma unroll
            for (int i = 0; i < NF; ++i)
                if (e0 + i < K) theta_read[(long long)j * K + e0 + i] = th[i];
        }
        ahead(j + G);
        cp_async_wait<0>();
        __syncwarp();
        bool nan = false;   // among the values that samples past the batch would meet
        if constexpr (FORM != kWhole) {
            const float first = sTab[64 * (lane < k ? lane : 0)];
            nan = first != first;
#pragma unroll
            for (int i = 0; i < NF; ++i) nan |= sg[i] != sg[i];
            nan = __any_sync(0xffffffffu, nan);
        }
#pragma unroll
        for (int m = 0; m < k; ++m) cw[m] = (cw[m] & cmask) >> (TAIL && nst == 1 ? tail.shift : 0);
        look(0);
        auto stages = [&](auto nan_met) {
#pragma unroll 1
            for (int st = 0; st < nst; ++st) {
                if (decltype(nan_met)::value && nan && st + 1 == nst) fill();
                uint32_t cn[k];
                float4 gn;
#pragma unroll
                for (int m = 0; m < k; ++m) cn[m] = 0u;
                gn = make_float4(0.f, 0.f, 0.f, 0.f);
                if (st + 1 < nst) {
#pragma unroll
                    for (int m = 0; m < k; ++m) cn[m] = __ldg(src[m] + 32 * (st + 1) + (TAIL ? word_of(st + 1) : 0));
                    gn = load_g(st + 1);
                }
                // one sample: its tree, the inputs of sample `next` of the words in cw
                // (after moving on to the next stage's words when `step`), its terms
                // into the columns
                auto sample = [&](float g, bool step, int next) {
                    float dx[k];
                    node_sample2<k>(cp, x, g, dx, acc);
                    uint32_t at[k];   // this sample's columns
#pragma unroll
                    for (int m = 0; m < k; ++m) at[m] = 32u * ea[m] + cb[base(m)];
                    if (step) {   // on to the next stage
#pragma unroll
                        for (int m = 0; m < k; ++m) cw[m] = (cn[m] & cmask) >> (TAIL && st + 2 == nst ? tail.shift : 0);
                    }
                    look(next);
#pragma unroll
                    for (int m0 = 0; m0 < k; m0 += C) {   // a step: slots m0 .. m0 + C - 1 of this lane's order
                        float old[C];
#pragma unroll
                        for (int i = 0; i < C; ++i)
                            if (m0 + i < k) old[i] = lds(at[m0 + i] + column_off(m0 + i));
#pragma unroll
                        for (int i = 0; i < C; ++i)
                            if (m0 + i < k) sts(at[m0 + i] + column_off(m0 + i), old[i] + dx[m0 + i]);
                        __syncwarp();   // the other lane of these columns comes to them in another step
                    }
                };
                if (!TAIL || st + 1 < nst) {
                    sample(g4.x, false, 1);
                    sample(g4.y, false, 2);
                    sample(g4.z, false, 3);
                    sample(g4.w, true, 0);
                } else {
#pragma unroll 1
                    for (int c = 0; c < tail.nc; ++c) sample(c ? g4.y : g4.x, false, c + 1);   // nc <= 2
                }
                g4 = gn;
            }
        };
        // the check in the loop, or a loop of its own for such nodes: 8000 nodes
        // x 907 samples, step 169.7 us at fan-in 6 without it, 171.9 and 173.7;
        // 82.2 at fan-in 4, 82.3 and 82.1; 88340 nodes of fan-in 4 x 44 samples
        // 187.9, 194.7 and 197.9
        if constexpr (k >= 6 || TAIL) stages(std::integral_constant<bool, FORM != kWhole>{});
        else if (FORM != kWhole && nan) stages(std::true_type{});
        else stages(std::false_type{});
        __syncwarp();
        if (j + G < w) start(j + G);   // the next node's loads fly during the epilogue

        // corner sums out (and columns cleared): lane = corner
        float* rowp[k];
#pragma unroll
        for (int i = 0; i < k; ++i) {
            long long row = (long long)j * k + i;
            if (epos) {
                const int r = __shfl_sync(0xffffffffu, posn, i);
                if (r >= 0 && (long long)r < (long long)w * k) row = r;
                else if (lane == 0) flag_index_error();   // stored at its own row, inside the buffer
            }
            rowp[i] = corner + (row << k1);
        }
        for (int a0 = 0; a0 < K1; a0 += 32) {
            const int a = a0 + lane;
            if (a < K1) {
                float s[2];
#pragma unroll
                for (int m = 0; m < C; ++m) {
                    take_row(smem + m * (64 * 32), a, lane, s);
                    rowp[m][a] = s[0];
                    rowp[m + C][a] = s[1];
                }
                if constexpr (k % 2 != 0) {
                    take_row(smem + C * (64 * 32), a, lane, s);
                    rowp[k - 1][a] = s[0];
                }
            }
        }
        __syncwarp();
        // dtheta: over the lanes of a half, then the two halves
        float sum[K];
#pragma unroll
        for (int a = 0; a < H; ++a) unpack2(acc[a], sum[a], sum[a + H]);
        half_reduce<K, 8>(sum, lane);
        constexpr int NV = K / 16;
        if (h == 0) {
#pragma unroll
            for (int i = 0; i < NV; ++i) smem[p * NV + i] = sum[i];
        }
        __syncwarp();
        if (h == 1) {
#pragma unroll
            for (int i = 0; i < NV; ++i) smem[O::to_slots(1, p * NV + i)] += sum[i];
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NF; ++i)
            if (e0 + i < K) dtheta[(long long)j * K + e0 + i] = sg[i] * (1.0f - sg[i]) * smem[e0 + i];
    }
    cp_async_wait<0>();
}

// --------------------------------------------------- layer 1 table gradient --

// dtheta[j][a] = slope(theta_j[a]) * sum of the corner sums H[edge[p]][a] over
// the CSR positions p of node j (an order of its own when parts > 1: no other
// call forms this sum).  `parts` warps of a block per node, each over
// a run of its positions in increasing p, then the runs in order; lane = table
// entry (two neighbours per lane for 64 entries).  The rows of up to eight
// positions and the logits are in flight together: the kernel reads each byte
// once and is bound by the latency of its two dependent loads at small widths,
// by DRAM at large ones.
template <bool WIDE, bool SPLIT>   // 64 entries; several parts per node
__global__ void __launch_bounds__(256)
corner_reduce_kernel(const float* __restrict__ corner, const int* __restrict__ off, const int* __restrict__ edge,
                     int n_edges, const float* __restrict__ theta, int w, int k, int parts,
                     float* __restrict__ dtheta) {
    constexpr int kRows = 8;
    __shared__ float2 run[SPLIT ? 8 : 1][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, K = 1 << k;
    const int at = SPLIT ? blockIdx.x * (8 / parts) + warp / parts : blockIdx.x * 8 + warp;
    if (!SPLIT && at >= w) return;   // warp-uniform
    const int j = SPLIT ? min(at, w - 1) : at;   // past the end: the last node once more, not written
    int e0 = __ldg(off + j), e1 = __ldg(off + j + 1);
    const long long o = (long long)j * K + (WIDE ? 2 * lane : lane);
    const bool in = WIDE || lane < K;
    float2 th = make_float2(0.f, 0.f);
    // logits and gradient by single values: a caller's parameter may start at
    // any float
    if (in) th.x = __ldg(theta + o);
    if constexpr (WIDE) th.y = __ldg(theta + o + 1);
    if (e0 < 0 || e1 < e0 || e1 > n_edges) {
        if (lane == 0) flag_index_error();
        e0 = e1 = 0;
    }
    if constexpr (SPLIT) {
        const int len = (e1 - e0 + parts - 1) / parts;
        e0 = min(e0 + warp % parts * len, e1);
        e1 = min(e0 + len, e1);
    }
    float2 s = make_float2(0.f, 0.f);
    bool bad = false;
    for (int q = e0; q < e1; q += kRows) {
        // no branch before a load, which keeps the loads of a batch together
        // (64000 x 64000 nodes, 1024 samples, step 1153 -> 1143 us): past the
        // end the last position once more, for a position out of range row 0,
        // neither added
        float2 v[kRows];
        bool add[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const int at_q = min(q + r, e1 - 1), id = edge ? __ldg(edge + at_q) : at_q;
            const bool ok = (unsigned)id < (unsigned)n_edges;
            add[r] = ok && q + r < e1;
            bad |= !ok;
            const float* row = corner + ((long long)(ok ? id : 0) << k);
            if constexpr (WIDE) v[r] = __ldcs(reinterpret_cast<const float2*>(row) + lane);
            else v[r] = make_float2(__ldcs(row + (lane & (K - 1))), 0.f);
        }
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            s.x += add[r] ? v[r].x : 0.f;
            if constexpr (WIDE) s.y += add[r] ? v[r].y : 0.f;
        }
    }
    if (bad && lane == 0) flag_index_error();
    if constexpr (SPLIT) {
        run[warp][lane] = s;
        __syncthreads();
        if (warp % parts != 0 || at >= w) return;
        for (int r = 1; r < parts; ++r) {
            s.x += run[warp + r][lane].x;
            s.y += run[warp + r][lane].y;
        }
    }
    const float t0 = sigmoidf(th.x), t1 = sigmoidf(th.y);
    if (in) dtheta[o] = t0 * (1.0f - t0) * s.x;
    if constexpr (WIDE) dtheta[o + 1] = t1 * (1.0f - t1) * s.y;
}

// ------------------------------------------------------------- launchers --

template <int k>
int launch_codes(const uint32_t* X, int w_in, long long B, const int* conn, const float* theta, int w, int node,
                 uint8_t* codes, long long stride, float* table, cudaStream_t st) {
    const long long nblk = (B + kBitBlock - 1) / kBitBlock;
    // the whole batch per warp unless that leaves fewer than two waves
    const long long warps = 2ll * sm_count() * 64;
    long long chunk = ((long long)w * nblk + warps - 1) / warps;
    if (chunk < 1) chunk = 1;
    const long long ny = (nblk + chunk - 1) / chunk;
    if (ny > 65535) return BITLOGIC_ERR_SHAPE;
    dim3 grid((unsigned)((w + kCodesWarps - 1) / kCodesWarps), (unsigned)ny);
    codes_forward_kernel<k><<<grid, kCodesWarps * 32, 0, st>>>(X, w_in, nblk * 32, conn, theta, w, node, codes, stride,
                                                               table, chunk);
    return launch_status();
}

template <int k>
int launch_coded_forward(const uint8_t* codes, long long stride, const float* table, int w_in, int k1, long long B,
                         const int* conn, const float* theta, int w, int node, float* Y, cudaStream_t st) {
    const size_t smem = ((1 << k) + 2 * k * 64) * sizeof(float);
    const long long resident = (long long)sm_count() * BITLOGIC_CODED_FWD_BLOCKS;
    auto kern = short_tail(B) ? coded_forward_kernel<k, true> : coded_forward_kernel<k, false>;
    kern<<<(unsigned)(w < resident ? w : resident), 32, smem, st>>>(
        codes, stride, table, w_in, k1, B, conn, theta, w, node, Y, B % 4 == 0 && aligned16(Y));
    return launch_status();
}

template <int k>
int launch_coded_backward(const uint8_t* codes, long long stride, const float* table, int w_in, int k1, long long B,
                          const int* conn, const float* theta, int w, int node, const float* dY, int group,
                          float* dtheta, float* corner, const int* epos, float* theta_read, cudaStream_t st) {
    constexpr int smem = coded_bwd_smem<k>();
    // one wave: as many blocks per SM as registers and shared memory (228 KB,
    // 1 KB of it per block) hold
    constexpr int fit = (228 * 1024) / (smem + 1024);
    const long long resident = (long long)sm_count() * (fit < coded_bwd_blocks<k>() ? fit : coded_bwd_blocks<k>());
    auto kern = B % 128 == 0    ? coded_backward_kernel<k, kWhole>
                : short_tail(B) ? coded_backward_kernel<k, kShort>
                                : coded_backward_kernel<k, kRagged>;
    kern<<<(unsigned)(w < resident ? w : resident), 32, smem, st>>>(
        codes, stride, table, w_in, k1, B, conn, theta, w, node, dY, group, B % 4 == 0 && aligned16(dY), dtheta, corner,
        epos, theta_read);
    return launch_status();
}

// Host checks of the layer-2 calls.
int check_coded(const void* codes, const void* table, int32_t w_in, int32_t k_in, int64_t B, const void* conn,
                const void* theta, int32_t w, int32_t k, int32_t node) {
    if (!conn || !theta) return BITLOGIC_ERR_NULL;
    if (B > 0 && (!codes || !table)) return BITLOGIC_ERR_NULL;
    if (w_in <= 0 || w <= 0 || B < 0) return BITLOGIC_ERR_SHAPE;
    if (k < 4 || k > 6 || k > w_in || k_in < 1 || k_in > 6) return BITLOGIC_ERR_FANIN;
    if ((int64_t)w * k > 0x7fffffffLL) return BITLOGIC_ERR_SHAPE;
    if (node != BITLOGIC_NODE_SOFT && node != BITLOGIC_NODE_ST) return BITLOGIC_ERR_NODE;
    if ((reinterpret_cast<uintptr_t>(codes) & 3u) != 0 || !aligned16(table)) return BITLOGIC_ERR_ALIGN;
    return BITLOGIC_OK;
}

long long code_stride(int64_t B) { return (B + 127) / 128 * 128; }

}  // namespace
}  // namespace bitlogic

using namespace bitlogic;

BITLOGIC_ERROR_READER(lut_codes)

extern "C" int bitlogic_lut_forward_codes(const uint32_t* X, int32_t w_in, int64_t B, const int32_t* conn,
                                          const float* theta, int32_t w, int32_t k, int32_t node, uint8_t* codes,
                                          float* table, cudaStream_t stream) {
    if (!conn || !theta) return BITLOGIC_ERR_NULL;
    if (B > 0 && (!X || !codes || !table)) return BITLOGIC_ERR_NULL;
    if (w_in <= 0 || w <= 0 || B < 0) return BITLOGIC_ERR_SHAPE;
    if (k < 1 || k > 6 || k > w_in) return BITLOGIC_ERR_FANIN;
    if ((int64_t)w * k > 0x7fffffffLL) return BITLOGIC_ERR_SHAPE;
    if (node != BITLOGIC_NODE_SOFT && node != BITLOGIC_NODE_ST) return BITLOGIC_ERR_NODE;
    if (B == 0) return BITLOGIC_OK;
    if (((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(codes)) & 3u) != 0) return BITLOGIC_ERR_ALIGN;
    const long long sd = code_stride(B);
    switch (k) {
        case 1: return launch_codes<1>(X, w_in, B, conn, theta, w, node, codes, sd, table, stream);
        case 2: return launch_codes<2>(X, w_in, B, conn, theta, w, node, codes, sd, table, stream);
        case 3: return launch_codes<3>(X, w_in, B, conn, theta, w, node, codes, sd, table, stream);
        case 4: return launch_codes<4>(X, w_in, B, conn, theta, w, node, codes, sd, table, stream);
        case 5: return launch_codes<5>(X, w_in, B, conn, theta, w, node, codes, sd, table, stream);
        default: return launch_codes<6>(X, w_in, B, conn, theta, w, node, codes, sd, table, stream);
    }
}

extern "C" int bitlogic_codes_decode(const uint8_t* codes, const float* table, int32_t w, int32_t k, int64_t B,
                                     float* Y, cudaStream_t stream) {
    if (w <= 0 || B < 0) return BITLOGIC_ERR_SHAPE;
    if (k < 1 || k > 6) return BITLOGIC_ERR_FANIN;
    if (B == 0) return BITLOGIC_OK;
    if (!codes || !table || !Y) return BITLOGIC_ERR_NULL;
    codes_decode_kernel<<<(unsigned)w, 256, 0, stream>>>(codes, code_stride(B), table, 1 << k, w, B, Y);
    return launch_status();
}

extern "C" int bitlogic_lut_forward_coded(const uint8_t* codes, const float* table, int32_t w_in, int32_t k_in,
                                          int64_t B, const int32_t* conn, const float* theta, int32_t w, int32_t k,
                                          int32_t node, float* Y, cudaStream_t stream) {
    int st = check_coded(codes, table, w_in, k_in, B, conn, theta, w, k, node);
    if (st) return st;
    if (B == 0) return BITLOGIC_OK;
    if (!Y) return BITLOGIC_ERR_NULL;
    const long long sd = code_stride(B);
    switch (k) {
        case 4: return launch_coded_forward<4>(codes, sd, table, w_in, k_in, B, conn, theta, w, node, Y, stream);
        case 5: return launch_coded_forward<5>(codes, sd, table, w_in, k_in, B, conn, theta, w, node, Y, stream);
        default: return launch_coded_forward<6>(codes, sd, table, w_in, k_in, B, conn, theta, w, node, Y, stream);
    }
}

// bitlogic_lut_backward_coded; theta_read (or NULL) receives the logits that
// the call read, for a caller that forms more of this backward once theta has
// moved on.  The kernels of partly filled stages store them as they go.
extern "C" int bitlogic_internal_lut_backward_coded(const uint8_t* codes, const float* table, int32_t w_in,
                                                    int32_t k_in, int64_t B, const int32_t* conn, const float* theta,
                                                    int32_t w, int32_t k, int32_t node, const float* dY,
                                                    int32_t dy_group, float* dtheta, float* corner_sums,
                                                    const int32_t* edge_pos, float* theta_read, cudaStream_t stream) {
    int st = check_coded(codes, table, w_in, k_in, B, conn, theta, w, k, node);
    if (st) return st;
    if (!dtheta || !corner_sums || (B > 0 && !dY)) return BITLOGIC_ERR_NULL;
    if (dy_group < 1 || dy_group > w) return BITLOGIC_ERR_SHAPE;
    if (theta_read && B % 128 == 0 &&
        cudaMemcpyAsync(theta_read, theta, sizeof(float) * (size_t)w << k, cudaMemcpyDeviceToDevice, stream) !=
            cudaSuccess)
        return BITLOGIC_ERR_CUDA;
    if (B == 0) {   // empty batch: the batch sums are zero
        if (cudaMemsetAsync(dtheta, 0, sizeof(float) * (size_t)w << k, stream) != cudaSuccess ||
            cudaMemsetAsync(corner_sums, 0, sizeof(float) * (size_t)w * k << k_in, stream) != cudaSuccess)
            return BITLOGIC_ERR_CUDA;
        return BITLOGIC_OK;
    }
    const long long sd = code_stride(B);
#define BITLOGIC_CODED_K(K)                                                                                       \
    return launch_coded_backward<K>(codes, sd, table, w_in, k_in, B, conn, theta, w, node, dY, dy_group, dtheta, \
                                    corner_sums, edge_pos, theta_read, stream)
    switch (k) {
        case 4: BITLOGIC_CODED_K(4);
        case 5: BITLOGIC_CODED_K(5);
        default: BITLOGIC_CODED_K(6);
    }
#undef BITLOGIC_CODED_K
}

extern "C" int bitlogic_lut_backward_coded(const uint8_t* codes, const float* table, int32_t w_in, int32_t k_in,
                                           int64_t B, const int32_t* conn, const float* theta, int32_t w, int32_t k,
                                           int32_t node, const float* dY, int32_t dy_group, float* dtheta,
                                           float* corner_sums, const int32_t* edge_pos, cudaStream_t stream) {
    return bitlogic_internal_lut_backward_coded(codes, table, w_in, k_in, B, conn, theta, w, k, node, dY, dy_group,
                                                dtheta, corner_sums, edge_pos, nullptr, stream);
}

extern "C" int bitlogic_corner_reduce(const float* corner_sums, const int32_t* csr_off, const int32_t* csr_edge,
                                      int32_t n_edges, const float* theta, int32_t w, int32_t k, float* dtheta,
                                      cudaStream_t stream) {
    if (!csr_off || !theta || !dtheta || (n_edges > 0 && !corner_sums)) return BITLOGIC_ERR_NULL;
    if (w <= 0 || n_edges < 0) return BITLOGIC_ERR_SHAPE;
    if (k < 1 || k > 6) return BITLOGIC_ERR_FANIN;
    const bool wide = k == 6;
    if (wide && (reinterpret_cast<uintptr_t>(corner_sums) & 7u) != 0) return BITLOGIC_ERR_ALIGN;
    // more warps per node while they all fit one wave and keep four positions
    // each on average: few nodes with many readers are bound by the chain of
    // their rows (training steps of fan-in 6: 1015 and 9110 nodes at 68 samples
    // 81 -> 69 us; 1015 and 20000 at 1024 samples 386 -> 362 us; fan-in 5, 500
    // and 50000 at 200 samples 349 -> 233 us)
    int parts = 1;
    while (parts < 8 && 2ll * parts * w <= 64ll * sm_count() && n_edges / (2ll * parts * w) >= 4) parts *= 2;
    auto kern = parts > 1 ? (wide ? corner_reduce_kernel<true, true> : corner_reduce_kernel<false, true>)
                          : (wide ? corner_reduce_kernel<true, false> : corner_reduce_kernel<false, false>);
    kern<<<(unsigned)((w * (long long)parts + 7) / 8), 256, 0, stream>>>(corner_sums, csr_off, csr_edge, n_edges, theta,
                                                                       w, k, parts, dtheta);
    return launch_status();
}
