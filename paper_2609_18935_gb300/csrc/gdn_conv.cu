// Short convolution of a gated-delta-rule layer with its carried state (the
// convolution part of R_t, §4.1: it continues across rounds without rollback,
// like S).  Each channel c of the layer's q, k and v projections (channels
// ordered q [H][d_k], k [H][d_k], v [H][d_v]) is filtered by a causal
// depthwise convolution of width 4 and passed through SiLU:
//     y_t[c] = silu(sum_{i=0..3} w[c][i] x_{t-3+i}[c]),
// where x_{-3..-1} are the last three inputs of earlier rounds (the conv
// state; zero for a fresh context).  Each head's k is then scaled to unit L2
// norm (the delta rule's keys); q and v are not.  The outputs are rounded to
// bf16, the delta rule's operand type.
//
// Bound by memory: every input is read and every output written once.  A
// thread owns eight channels (16 bytes of a token's row) and walks a strip of
// consecutive packed tokens with the taps and the last three inputs in
// registers, four rows in flight; a head's d_k / 8 neighbouring lanes share
// the norm of k.  Strips are as long as the grid allows: a strip's first
// three rows are read again.  8674 tokens of 6144 channels (213 MB): 60 us, 3.6
// TB/s, against 417 with a block a token and head; the exact SiLU is 7 of it.
//
// blockIdx.y < n_strips: outputs of a strip; beyond: one row of blocks per
// character writes the character's new state (the last three inputs of
// [state; tail]) into the other of two state buffers, so that no block reads
// a state row that another block of the same launch writes.
#include "kvm_internal.cuh"
#include "packed_f32.cuh"

namespace kvm {
namespace {

constexpr int kThreads = 128;
constexpr int kAhead = 4;                    // rows loaded ahead of their use

// Eight bf16 channels as four pairs of floats.
__device__ __forceinline__ void unpack8(const uint4& v, f2* x) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&v);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
        x[e] = pack2(f.x, f.y);
    }
}

// ALIGNED: the inputs lie on the 16-byte grid; otherwise their channels are read
// one by one.
template <bool ALIGNED>
__global__ void __launch_bounds__(kThreads, 4) gdn_conv_kernel(const __grid_constant__ ConvParams p) {
    const int g = blockIdx.x * kThreads + threadIdx.x;       // channels 8 g .. 8 g + 7
    const bool act = 8 * g < p.channels;
    const int hk = p.H * p.dk, c = act ? 8 * g : 0;
    const bool is_k = act && c >= hk && c < 2 * hk;
    // the part's rows are contiguous: [tok][H d_k] or [tok][H d_v]
    const int first = c < hk ? 0 : c < 2 * hk ? hk : 2 * hk;
    const int64_t stride = c < 2 * hk ? hk : p.H * p.dv;
    const __nv_bfloat16* in = (c < hk ? p.xq : c < 2 * hk ? p.xk : p.xv) + (c - first);
    __nv_bfloat16* out = (c < hk ? p.yq : c < 2 * hk ? p.yk : p.yv) + (c - first);
    auto row = [&](int64_t tok) {
        const __nv_bfloat16* x = in + tok * stride;
        if constexpr (ALIGNED) return *reinterpret_cast<const uint4*>(x);
        uint4 v;
        __nv_bfloat16* e = reinterpret_cast<__nv_bfloat16*>(&v);
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = x[i];
        return v;
    };
    auto old_row = [&](int b, int r) {
        return *reinterpret_cast<const uint4*>(p.state_in + ((int64_t)b * 3 + r) * p.channels + c);
    };
    grid_dependency_wait();
    grid_dependents_launch();
    if ((int)blockIdx.y >= p.n_strips) {
        const int b = blockIdx.y - p.n_strips;
        if (b >= p.n_chars) { if (threadIdx.x == 0) atomicOr(p.err, kErrBounds); return; }
        if (!act) return;
        const int M = p.tail_cu[b + 1] - p.tail_cu[b];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int t = M - 3 + r;                         // position in the tail (negative: old state row t + 3)
            *reinterpret_cast<uint4*>(p.state_out + ((int64_t)b * 3 + r) * p.channels + c) =
                t >= 0 ? row(p.tail_cu[b] + t) : old_row(b, t + 3);
        }
        return;
    }
    const int n0 = blockIdx.y * p.strip, n1 = min(p.total, n0 + p.strip);
    int lo = 0, hi = p.n_chars - 1;                          // last b with tail_cu[b] <= n0
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.tail_cu[mid] <= n0) lo = mid; else hi = mid - 1;
    }
    int b = lo, end = p.tail_cu[b + 1];
    f2 w[4][4];                                              // [tap][channel pair]
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float4 f = *(reinterpret_cast<const float4*>(p.w) + c + 2 * e);
        const float4 g = *(reinterpret_cast<const float4*>(p.w) + c + 2 * e + 1);
        w[0][e] = pack2(f.x, g.x); w[1][e] = pack2(f.y, g.y); w[2][e] = pack2(f.z, g.z); w[3][e] = pack2(f.w, g.w);
    }
    f2 x[4][4];                                              // the inputs of taps 0 .. 3
    // the three inputs before token n of character b
    auto history = [&](int n) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const int t = n - p.tail_cu[b] - 3 + i;
            unpack8(t >= 0 ? row(n - 3 + i) : old_row(b, t + 3), x[i]);
        }
    };
    const bool any_k = __any_sync(0xffffffffu, is_k);
    uint4 next[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) next[u] = n0 + u < n1 ? row(n0 + u) : make_uint4(0, 0, 0, 0);
    history(n0);
    for (int n = n0; n < n1; n += kAhead) {
        uint4 now[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            now[u] = next[u];
            if (n + kAhead + u < n1) next[u] = row(n + kAhead + u);
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            if (n + u >= n1) break;                          // uniform per block
            if (n + u == end) {                              // the next character with a tail
                do ++b; while (p.tail_cu[b + 1] == p.tail_cu[b]);
                end = p.tail_cu[b + 1];
                history(n + u);
            }
            unpack8(now[u], x[3]);
            float y[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                f2 acc = 0;                                  // two zeros
#pragma unroll
                for (int i = 0; i < 4; ++i) acc = fma2(w[i][e], x[i][e], acc);
                const float2 a = silu2(acc);
                y[2 * e] = a.x;
                y[2 * e + 1] = a.y;
            }
            if (any_k) {                                     // uniform per warp
                float tot = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) tot = fmaf(y[e], y[e], tot);
                for (int o = p.dk / 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
                if (is_k) {
                    const float inv = tot > 0.f ? rsqrtf(tot) : 0.f;
#pragma unroll
                    for (int e = 0; e < 8; ++e) y[e] *= inv;
                }
            }
            uint4 o4;
            __nv_bfloat162* o2 = reinterpret_cast<__nv_bfloat162*>(&o4);
#pragma unroll
            for (int e = 0; e < 4; ++e) o2[e] = __floats2bfloat162_rn(y[2 * e], y[2 * e + 1]);
            if (act) *reinterpret_cast<uint4*>(out + (int64_t)(n + u) * stride) = o4;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) x[i][e] = x[i + 1][e];
        }
    }
}

}  // namespace

void launch_gdn_conv(const ConvParams& p, cudaStream_t s) {
    if (p.total <= 0) return;
    launch_pdl(p.aligned ? gdn_conv_kernel<true> : gdn_conv_kernel<false>,
               dim3((p.channels / 8 + kThreads - 1) / kThreads, p.n_strips + p.n_chars), dim3(kThreads), 0, s, p);
}

}  // namespace kvm
