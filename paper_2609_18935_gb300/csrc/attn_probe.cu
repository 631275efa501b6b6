// Attention-probe diagnostics (§5.3; Appendix C): the attention distribution
// of a character's last n_q query tokens over its live KV, reconstructed with
// a float32 reference softmax and averaged over those queries and every query
// head of one attention layer.  Removed records left holes in position space
// only: the compacted cache holds live entries alone, so the softmax
// denominator runs over live tokens (holes excluded) by construction.
//
// Query i of the probe (0 <= i < n_q) is the live entry L - n_q + i; it sees
// live entries 0 .. L - n_q + i (causal in processing order), with scores
// q_i . k_j / sqrt(D) in fp32, q_i rotated at that entry's position.
//
//  probe_rotate : rotate the caller's probe queries (fp64 angle reduced mod
//                 2 pi, fp32 rotation) into an fp32 workspace;
//  probe_scores : S = Q K^T of 64 rows (query, head of the group) of one KV
//                 head and 64 keys a block, in fp32 on the CUDA cores;
//  probe_rows   : per row, the softmax max and one over the denominator;
//  probe_probs  : p = exp(s - max) / sum summed over the rows: the averaged
//                 distribution of each key, and its group's mass (atomic adds)
//                 when groups are given.
//
// The scores are formed once and pass through memory (the attention's partials
// workspace; row blocks that do not fit together are done in turn).  8192 keys,
// 8 queries of 16 heads of 256 (0.54 GFLOP): rotate 4, scores 18,
// rows 5, probs 5 us alone, 48 together, against 210 with the scores formed
// twice by 128 threads a tile and one thread a row merging the tiles.
// Fp32 products throughout: on the tensor cores the queries would have to be
// split, and this is the reference that other paths are judged by.
#include <algorithm>

#include "kvm_internal.cuh"
#include "packed_f32.cuh"

namespace kvm {
namespace {

constexpr double kTwoPiP = 6.283185307179586476925286766559;
constexpr int kScoreThreads = 128;
constexpr int kDims = 32;                      // dims staged per step
constexpr int kPitch = 64 + 4;                 // row pitch of the staged [dim][64] tiles
constexpr int kProbThreads = 256;              // probe_probs: 32 keys, eight threads each

// One block per (query, head).
__global__ void __launch_bounds__(128) probe_rotate_kernel(const __grid_constant__ ProbeParams p) {
    grid_dependency_wait();
    grid_dependents_launch();
    const int i = blockIdx.x / p.Hq, half = p.R / 2;
    const int64_t pos = p.pos[p.slot0 + p.L - p.n_q + i];
    const __nv_bfloat16* q = p.q + (int64_t)blockIdx.x * p.D;
    float* o = p.q_rot + (int64_t)blockIdx.x * p.D;
    for (int d = threadIdx.x; d < half; d += blockDim.x) {
        const double ang = (double)pos * p.inv_freq[d];
        const double r = fma(-rint(ang * (1.0 / kTwoPiP)), kTwoPiP, ang);
        float sn, cs;
        sincosf((float)r, &sn, &cs);
        const float x = __bfloat162float(q[d]), y = __bfloat162float(q[d + half]);
        o[d] = x * cs - y * sn;
        o[d + half] = y * cs + x * sn;
    }
    for (int d = p.R + threadIdx.x; d < p.D; d += blockDim.x) o[d] = __bfloat162float(q[d]);
}

// grid (key tiles, row blocks).  Thread (ty, tx) forms rows 8 ty .. + 7 (in
// packed pairs) and keys 4 tx .. + 3 of the 64 x 64 tile; q and k are staged
// 32 dims at a time as [dim][64].  Row rg of KV head kv is query rg / g, head
// kv g + rg mod g.
__global__ void __launch_bounds__(kScoreThreads) probe_scores_kernel(const __grid_constant__ ProbeParams p) {
    __shared__ __align__(16) float Qs[kDims][kPitch], Ks[kDims][kPitch];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int rows_kv = p.n_q * p.g, blocks_kv = (rows_kv + kProbeRows - 1) / kProbeRows;
    const int rb = p.row_block0 + blockIdx.y;
    const int kv = rb / blocks_kv, r0 = (rb % blocks_kv) * kProbeRows;
    const int D = p.D, j0 = blockIdx.x * kProbeKeys;
    grid_dependency_wait();
    grid_dependents_launch();
    const __nv_bfloat16* kb = p.K + ((int64_t)kv * p.slab_rows + p.slot0 + j0) * D;
    // staging: thread t moves dims 8 (t mod 4) .. + 7 of tile rows t / 4, t / 4 + 32,
    // turned by 8 (t mod 4) columns so that the four pieces of a row meet
    // different banks
    const int c = (tid & 3) * 8, sr = tid >> 2;
    const float* qr[2];
    bool q_in[2], k_in[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int rg = r0 + sr + 32 * i;
        q_in[i] = rg < rows_kv;
        qr[i] = p.q_rot + (q_in[i] ? ((int64_t)(rg / p.g) * p.Hq + kv * p.g + rg % p.g) * D : 0);
        k_in[i] = j0 + sr + 32 * i < p.L;
    }
    uint4 kx[2];
    float4 qx[2][2];
    auto load = [&](int d) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            kx[i] = k_in[i] ? *reinterpret_cast<const uint4*>(kb + (int64_t)(sr + 32 * i) * D + d + c) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int e = 0; e < 2; ++e)
                qx[i][e] = q_in[i] ? *reinterpret_cast<const float4*>(qr[i] + d + c + 4 * e) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    f2 acc[4][4];                                             // [row pair][key]
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0;
    load(0);
    for (int d0 = 0; d0 < D; d0 += kDims) {
        __syncthreads();                                      // the previous step is consumed
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t* w = reinterpret_cast<const uint32_t*>(&kx[i]);
            const float* f = reinterpret_cast<const float*>(&qx[i][0]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                Ks[c + 2 * e][(sr + 32 * i + c) & 63] = __uint_as_float(w[e] << 16);
                Ks[c + 2 * e + 1][(sr + 32 * i + c) & 63] = __uint_as_float(w[e] & 0xffff0000u);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) Qs[c + e][(sr + 32 * i + c) & 63] = f[e];
        }
        __syncthreads();
        if (d0 + kDims < D) load(d0 + kDims);                 // in flight during the products
#pragma unroll 8
        for (int d = 0; d < kDims; ++d) {
            const int turn = d & ~7;                          // dims 8 k .. 8 k + 7 are stored turned by 8 k columns
            const float4 k4 = *reinterpret_cast<const float4*>(&Ks[d][(4 * tx + turn) & 63]);
            const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(&Qs[d][(8 * ty + turn) & 63]);
            const ulonglong2 qb = *reinterpret_cast<const ulonglong2*>(&Qs[d][(8 * ty + 4 + turn) & 63]);
            const f2 kk[4] = {pack2(k4.x, k4.x), pack2(k4.y, k4.y), pack2(k4.z, k4.z), pack2(k4.w, k4.w)};
            const f2 qq[4] = {qa.x, qa.y, qb.x, qb.y};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fma2(qq[a], kk[b], acc[a][b]);
        }
    }
    // rows past the end, keys past the row's causal limit: -inf
    const int j = j0 + 4 * tx, first_q = p.L - p.n_q;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        const int r = 8 * ty + a, rg = r0 + r, lim = rg < rows_kv ? first_q + rg / p.g : -1;
        float s[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float2 x = unpack2(acc[a >> 1][b]);
            s[b] = j + b <= lim ? (a & 1 ? x.y : x.x) * p.scale : -INFINITY;
        }
        if (j < p.pitch)
            *reinterpret_cast<float4*>(p.scores + ((int64_t)blockIdx.y * kProbeRows + r) * p.pitch + j) =
                make_float4(s[0], s[1], s[2], s[3]);
    }
}

// One block per row of the staged row blocks (rows past a head's end have no
// key: max -inf, factor 0).
__global__ void __launch_bounds__(256) probe_rows_kernel(const __grid_constant__ ProbeParams p) {
    grid_dependency_wait();
    grid_dependents_launch();
    __shared__ float red[8];
    const float4* s = reinterpret_cast<const float4*>(p.scores + (int64_t)blockIdx.x * p.pitch);
    const int n4 = p.pitch / 4, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float m = -INFINITY;
#pragma unroll 4
    for (int k = threadIdx.x; k < n4; k += 256) {
        const float4 x = s[k];
        m = fmaxf(m, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red[warp] = m;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) m = fmaxf(m, red[k]);
    __syncthreads();
    float e = 0.f;
    if (m != -INFINITY) {
#pragma unroll 4
        for (int k = threadIdx.x; k < n4; k += 256) {
            const float4 x = s[k];
            e += (expf(x.x - m) + expf(x.y - m)) + (expf(x.z - m) + expf(x.w - m));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) red[warp] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        e = 0.f;
        for (int k = 0; k < 8; ++k) e += red[k];
        p.row_ms[2 * blockIdx.x] = m;
        p.row_ms[2 * blockIdx.x + 1] = m == -INFINITY ? 0.f : 1.f / e;
    }
}

// 32 keys a block, warp w taking every eighth row.  Row blocks done in turn
// add up in probs_out; the last one scales and adds the group masses.
__global__ void __launch_bounds__(kProbThreads) probe_probs_kernel(const __grid_constant__ ProbeParams p) {
    grid_dependency_wait();
    grid_dependents_launch();
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + lane, n = p.n_row_blocks * kProbeRows;
    float acc = 0.f;
    if (j < p.L) {
#pragma unroll 8
        for (int r = w; r < n; r += 8) {
            const float2 ms = *reinterpret_cast<const float2*>(p.row_ms + 2 * r);
            const float s = p.scores[(int64_t)r * p.pitch + j];
            acc += s == -INFINITY ? 0.f : expf(s - ms.x) * ms.y;
        }
    }
    part[w][lane] = acc;
    __syncthreads();
    if (w > 0) return;
    float tot = 0.f;
    if (j < p.L) {
#pragma unroll
        for (int k = 0; k < 8; ++k) tot += part[k][lane];
        if (p.row_block0 > 0) tot += p.probs[j];
        if (p.last) tot /= (float)(p.n_q * p.Hq);
        p.probs[j] = tot;
    }
    if (p.last && p.group_of) {
        const int gid = j < p.L ? p.group_of[j] : -1;
        if (gid >= p.n_groups) atomicOr(p.err, kErrBounds);
        const bool in = gid >= 0 && gid < p.n_groups;
        // a record's entries are neighbours: one addition a group and warp
        uint32_t left = __ballot_sync(0xffffffffu, in);
        while (left) {
            const int lead = __shfl_sync(0xffffffffu, gid, __ffs(left) - 1);
            const bool mine = in && gid == lead;
            float sum = mine ? tot : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == __ffs(left) - 1) atomicAdd(p.group_mass + lead, sum);
            left &= ~__ballot_sync(0xffffffffu, mine);
        }
    }
}

}  // namespace

int probe_row_blocks(int n_q, int Hkv, int g) { return Hkv * ((n_q * g + kProbeRows - 1) / kProbeRows); }

int launch_attn_probe(ProbeParams p, cudaStream_t s) {
    if (p.L <= 0 || p.n_q <= 0) return 0;
    const int tiles = (p.L + kProbeKeys - 1) / kProbeKeys, total = probe_row_blocks(p.n_q, p.Hkv, p.g);
    p.pitch = (p.L + 3) / 4 * 4;
    const int fit = (int)std::min<int64_t>(total, p.scores_cap / ((int64_t)kProbeRows * p.pitch));
    launch_pdl(probe_rotate_kernel, dim3(p.n_q * p.Hq), dim3(128), 0, s, p);
    int launches = 1;
    for (p.row_block0 = 0; p.row_block0 < total; p.row_block0 += p.n_row_blocks, launches += 3) {
        p.n_row_blocks = std::min(fit, total - p.row_block0);
        p.last = p.row_block0 + p.n_row_blocks == total;
        launch_pdl(probe_scores_kernel, dim3(tiles, p.n_row_blocks), dim3(kScoreThreads), 0, s, p);
        launch_pdl(probe_rows_kernel, dim3(p.n_row_blocks * kProbeRows), dim3(256), 0, s, p);
        launch_pdl(probe_probs_kernel, dim3((p.L + 31) / 32), dim3(kProbThreads), 0, s, p);
    }
    return launches;
}

}  // namespace kvm
