// Gated delta rule, token by token, for short tails (Eq. 3 for a recurrent
// layer, §4.1; the recurrence of gdn_scan_tc.cu evaluated as it is written):
//     a = (alpha S) k,  u = beta (v - a),  S <- alpha S + u k^T,
//     o = S q = (alpha S) q + u (k . q).
// Decode steps and short replacements are bound by reading and writing S once
// (64 KB a head at d_k = d_v = 128); the chunked form spends a whole 64-token
// chunk's products, a record in memory and two launches on them.
//
// Without the convolution out may be v itself: a block stores only rows whose v
// it has staged, and no other block reads those.  It may not otherwise overlie the
// inputs (all blocks of a head stage its q, k and gates, in no order; a convolved
// step reads inputs once more after its outputs, to carry them): the caller
// convolves in a launch of its own or takes the chunked form for that.  Carrying v
// ahead of the outputs instead, in registers or stored at once, made a convolved
// step of 8 characters slower (2 tokens 4.8 -> 5.9, 4 tokens 6.7 -> 8.5 us).
//
// One block of four warps per (character, head, 16 NR rows of S).  Eight lanes
// share a row: lane j holds the float4 groups j, j + 8, ... of NR rows in
// registers from the first token to the last, so that S moves once, and a
// row's two dot products take three shuffles.  Tokens are staged in fp32 in
// shared memory, `tile` at a time, by the block itself; with a short
// convolution (see gdn_conv.cu) the staging convolves, so a layer is one
// launch either way.  All arithmetic is fp32 (packed pairs); against 64 bits
// the state is ~1e-7 off, the chunked form's split operands ~2.5e-6.
//
// Measured (16 heads, d_k = d_v = 128, back-to-back layers): a decode step of
// one character 2.3 us against 13.9 for the chunked form, of 32 characters 8.8
// against 88 (67 MB of state, 7.6 TB/s: the state sits in L2).  Longer tails
// are bound by the per-token chain (~0.24 us a token for one character) and the
// fp32 pipe (4 multiply-adds per element of S and token).  Fetching the next
// token's k and q ahead, two accumulators per dot product, and carrying S / prod
// alpha instead of decaying S were each slower (more registers, fewer blocks).
#include "kvm_internal.cuh"
#include "packed_f32.cuh"

namespace kvm {
namespace {

constexpr int kThreads = 128;

__device__ __forceinline__ float sum2(f2 v) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return lo + hi;
}
__device__ __forceinline__ void unpack8(const uint4& v, float* x) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(&v);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
        x[2 * e] = f.x;
        x[2 * e + 1] = f.y;
    }
}
__device__ __forceinline__ void store8(float* dst, const float* x) {
    *reinterpret_cast<float4*>(dst) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4*>(dst + 4) = make_float4(x[4], x[5], x[6], x[7]);
}

// One part (q, k or v) of a head's inputs: row t of the tail starts at
// in + t * stride, the carried conv state's row i (t = i - 3) at state + i *
// state_stride, and the taps of its first channel at w.
struct Part {
    const __nv_bfloat16* in;
    int64_t stride;
    const __nv_bfloat16* state;
    int64_t state_stride;
    const float* w;
    __device__ __forceinline__ uint4 row(int t, int c) const {
        return *reinterpret_cast<const uint4*>(t >= 0 ? in + (int64_t)t * stride + c
                                                      : state + (int64_t)(t + 3) * state_stride + c);
    }
    // convolution and SiLU of channels c .. c + 7 at token t, the taps in gdn_conv_kernel's
    // order (a key's norm is summed in another)
    __device__ __forceinline__ void conv8(int t, int c, float* y) const {
        uint4 r[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) r[i] = row(t - 3 + i, c);
        float x[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i) unpack8(r[i], x[i]);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float4 tap = *(reinterpret_cast<const float4*>(w) + c + e);
            float acc = fmaf(tap.x, x[0][e], 0.f);
            acc = fmaf(tap.y, x[1][e], acc);
            acc = fmaf(tap.z, x[2][e], acc);
            acc = fmaf(tap.w, x[3][e], acc);
            y[e] = acc;
        }
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
            const float2 v = silu2(pack2(y[e], y[e + 1]));
            y[e] = v.x;
            y[e + 1] = v.y;
        }
    }
};

template <int DK, int NR, bool CONV>
__global__ void __launch_bounds__(kThreads) gdn_recur_kernel(const __grid_constant__ RecurParams p) {
    constexpr int ROWS = 16 * NR;                    // rows of S a block
    constexpr int NP = DK / 32;                      // float4 groups of a row a lane
    constexpr int GK = DK / 8;                       // 8-channel pieces of a q or k row
    extern __shared__ __align__(16) float sm[];
    const int T = p.tile;
    float* ks = sm;                                  // [T][DK]
    float* qs = ks + T * DK;                         // [T][DK]
    float* vs = qs + T * DK;                         // [T][ROWS]
    float* ga = vs + T * ROWS;                       // alpha, beta, k . q: [T] each
    float* gb = ga + T;
    float* gkq = gb + T;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int j = lane & 7;
    const int r0 = blockIdx.x * ROWS, h = blockIdx.y, b = blockIdx.z;
    const int row0 = r0 + (warp * 4 + (lane >> 3)) * NR;       // this lane's first row
    const int H = p.H, dv = p.dv;
    const int tok0 = p.tail_cu[b], M = p.tail_cu[b + 1] - tok0;
    const int64_t cs = p.channels;
    const int hk = H * DK;                           // channels of all heads' q (and of k)
    const __nv_bfloat16* st = CONV ? p.state_in + (int64_t)b * 3 * cs : nullptr;
    const Part pq{p.q + ((int64_t)tok0 * H + h) * DK, hk, CONV ? st + h * DK : nullptr, cs, CONV ? p.w + (int64_t)(h * DK) * 4 : nullptr};
    const Part pk{p.k + ((int64_t)tok0 * H + h) * DK, hk, CONV ? st + hk + h * DK : nullptr, cs,
                  CONV ? p.w + (int64_t)(hk + h * DK) * 4 : nullptr};
    const Part pv{p.v + ((int64_t)tok0 * H + h) * dv + r0, (int64_t)H * dv, CONV ? st + 2 * hk + h * dv + r0 : nullptr, cs,
                  CONV ? p.w + (int64_t)(2 * hk + h * dv + r0) * 4 : nullptr};

    grid_dependency_wait();
    grid_dependents_launch();

    // the carried inputs after the tail, into the other state buffer (the
    // blocks of slice 0 also carry the head's q and k channels)
    auto carry = [&]() {
        __nv_bfloat16* nst = p.state_out + (int64_t)b * 3 * cs;
        const int per_row = ROWS / 8 + (blockIdx.x == 0 ? 2 * GK : 0);
        for (int e = tid; e < 3 * per_row; e += kThreads) {
            const int r = e / per_row, g = e % per_row, t = M - 3 + r;
            if (g < ROWS / 8) {
                *reinterpret_cast<uint4*>(nst + r * cs + 2 * hk + h * dv + r0 + 8 * g) = pv.row(t, 8 * g);
            } else if (g < ROWS / 8 + GK) {
                const int c = 8 * (g - ROWS / 8);
                *reinterpret_cast<uint4*>(nst + r * cs + h * DK + c) = pq.row(t, c);
            } else {
                const int c = 8 * (g - ROWS / 8 - GK);
                *reinterpret_cast<uint4*>(nst + r * cs + hk + h * DK + c) = pk.row(t, c);
            }
        }
    };
    if (M <= 0) {                                    // uniform per block
        if constexpr (CONV) carry();
        return;
    }

    float* Sg = p.S + (((int64_t)b * H + h) * dv + row0) * DK + 4 * j;
    f2 s[NR][2 * NP];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Sg + (int64_t)r * DK + 32 * i);
            s[r][2 * i] = x.x;
            s[r][2 * i + 1] = x.y;
        }

    for (int t0 = 0; t0 < M; t0 += T) {
        const int nt = min(T, M - t0);
        if (t0 > 0) __syncthreads();                 // the previous tile is consumed
        // ---- stage the tile
        for (int t = tid; t < nt; t += kThreads) {
            const int64_t at = (int64_t)(tok0 + t0 + t) * H + h;
            ga[t] = p.alpha[at];
            gb[t] = p.beta[at];
        }
        if constexpr (CONV) {
            // pieces of eight channels: every token's k, then q, then v, so
            // that a short tile is one round of loads; whole warps run the
            // loop (a k row's norm is taken over its GK lanes)
            const int nk = nt * GK, all = 2 * nk + nt * (ROWS / 8);
            for (int e0 = 0; e0 < all; e0 += kThreads) {
                const int e = e0 + tid;
                const bool is_k = e < nk, is_v = e >= 2 * nk;
                const int x = is_k ? e : is_v ? e - 2 * nk : e - nk;
                const int t = is_v ? x / (ROWS / 8) : x / GK, c = 8 * (is_v ? x % (ROWS / 8) : x % GK);
                float y[8] = {};
                float sq = 0.f;
                if (e < all) {
                    const Part part = is_k ? pk : is_v ? pv : pq;
                    part.conv8(t0 + t, c, y);
#pragma unroll
                    for (int i = 0; i < 8; ++i) sq = fmaf(y[i], y[i], sq);
                }
                if (e0 < nk) {                       // uniform per block
#pragma unroll
                    for (int o = GK / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
                }
                if (e < all) {
                    const float inv = !is_k ? 1.f : sq > 0.f ? rsqrtf(sq) : 0.f;
#pragma unroll
                    for (int i = 0; i < 8; ++i) y[i] = __bfloat162float(__float2bfloat16_rn(y[i] * inv));
                    store8(is_v ? vs + t * ROWS + c : (is_k ? ks : qs) + t * DK + c, y);
                }
            }
        } else {
#pragma unroll 2
            for (int e = tid; e < nt * GK; e += kThreads) {
                const int t = e / GK, c = 8 * (e % GK);
                const uint4 a = pk.row(t0 + t, c), d = pq.row(t0 + t, c);
                float y[8];
                unpack8(a, y);
                store8(ks + t * DK + c, y);
                unpack8(d, y);
                store8(qs + t * DK + c, y);
            }
            for (int e = tid; e < nt * (ROWS / 8); e += kThreads) {
                const int t = e / (ROWS / 8), c = 8 * (e % (ROWS / 8));
                float y[8];
                unpack8(pv.row(t0 + t, c), y);
                store8(vs + t * ROWS + c, y);
            }
        }
        __syncthreads();
        for (int t = warp; t < nt; t += kThreads / 32) {
            float d = 0.f;
#pragma unroll
            for (int i = 0; i < DK / 32; ++i) d = fmaf(ks[t * DK + lane + 32 * i], qs[t * DK + lane + 32 * i], d);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (lane == 0) gkq[t] = d;
        }
        __syncthreads();
        // ---- the recurrence
        __nv_bfloat16* out = p.out + ((int64_t)(tok0 + t0) * H + h) * dv + row0;
        for (int t = 0; t < nt; ++t) {
            f2 k2[2 * NP], q2[2 * NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(ks + t * DK + 4 * j + 32 * i);
                const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(qs + t * DK + 4 * j + 32 * i);
                k2[2 * i] = x.x; k2[2 * i + 1] = x.y;
                q2[2 * i] = y.x; q2[2 * i + 1] = y.y;
            }
            const float al = ga[t], be = gb[t], kq = gkq[t];
            const f2 al2 = pack2(al, al);
            float a[NR], d[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                f2 sk = 0, sq = 0;                   // two zeros each
#pragma unroll
                for (int i = 0; i < 2 * NP; ++i) {
                    s[r][i] = mul2(al2, s[r][i]);
                    sk = fma2(s[r][i], k2[i], sk);
                    sq = fma2(s[r][i], q2[i], sq);
                }
                a[r] = sum2(sk);
                d[r] = sum2(sq);
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1)
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    a[r] += __shfl_xor_sync(0xffffffffu, a[r], o);
                    d[r] += __shfl_xor_sync(0xffffffffu, d[r], o);
                }
            __nv_bfloat16 o16[NR];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const float u = be * (vs[t * ROWS + row0 - r0 + r] - a[r]);
                const f2 u2 = pack2(u, u);
#pragma unroll
                for (int i = 0; i < 2 * NP; ++i) s[r][i] = fma2(u2, k2[i], s[r][i]);
                o16[r] = __float2bfloat16_rn(fmaf(u, kq, d[r]));
            }
            if (j == 0) {                            // NR neighbouring rows, 2 NR bytes
                __nv_bfloat16* o = out + (int64_t)t * H * dv;
                if constexpr (NR == 4) *reinterpret_cast<uint2*>(o) = *reinterpret_cast<uint2*>(o16);
                else if constexpr (NR == 2) *reinterpret_cast<uint32_t*>(o) = *reinterpret_cast<uint32_t*>(o16);
                else *o = o16[0];
            }
        }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int i = 0; i < NP; ++i)
            *reinterpret_cast<ulonglong2*>(Sg + (int64_t)r * DK + 32 * i) = make_ulonglong2(s[r][2 * i], s[r][2 * i + 1]);
    if constexpr (CONV) carry();
}

template <int DK, int NR, bool CONV>
void launch_nr(const RecurParams& p, cudaStream_t s) {
    const size_t smem = sizeof(float) * (size_t)p.tile * (2 * DK + 16 * NR + 3);
    static unsigned long long configured = 0;   // one bit per device
    int dev = 0;
    cudaGetDevice(&dev);
    if (!(configured >> (dev & 63) & 1ull)) {
        cudaFuncSetAttribute(gdn_recur_kernel<DK, NR, CONV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(float) * kRecurMaxTail * (2 * DK + 16 * NR + 3)));
        configured |= 1ull << (dev & 63);
    }
    launch_pdl(gdn_recur_kernel<DK, NR, CONV>, dim3(p.dv / (16 * NR), p.H, p.n_chars), dim3(kThreads), smem, s, p);
}

template <int DK, bool CONV>
void launch_dk(const RecurParams& p, int nr, cudaStream_t s) {
    if (nr == 4) launch_nr<DK, 4, CONV>(p, s);
    else if (nr == 2) launch_nr<DK, 2, CONV>(p, s);
    else launch_nr<DK, 1, CONV>(p, s);
}

}  // namespace

void launch_gdn_recur(const RecurParams& p, int nr, cudaStream_t s) {
    if (p.dk == 64) p.w ? launch_dk<64, true>(p, nr, s) : launch_dk<64, false>(p, nr, s);
    else if (p.dk == 128) p.w ? launch_dk<128, true>(p, nr, s) : launch_dk<128, false>(p, nr, s);
}

}  // namespace kvm
