// K4, fused form, one token row and K <= 1536 (k4f_decode_fused.cuh has the others and the measurements).
//
// M = 1: a token row is little enough for every warp to quantize all of it for itself, in registers -- no barrier, no exchange
// and no shared memory between X and the products.  Lane l holds the codes of the 8-channel groups l, l + 32, ... and
// multiplies them with the same bytes of the rows of W_q that are its warp's.
#include "k4f_common.cuh"

namespace muxq {
namespace decode {

namespace {

template <int kC>
__global__ void __launch_bounds__(kRowT, 2) k_decode_row(const DecodeFusedArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];  // this CTA's rows of W_q
    __shared__ uint64_t bar_full;
    __shared__ uint32_t s_abort;
    const int t = threadIdx.x, lane = t & 31, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
    const int K = a.K, G = K >> 3;
    const int workers = (int)gridDim.x - 1;
    const bool side = (int)blockIdx.x == workers;
    const int n_begin = side ? 0 : (int)((long long)a.N * blockIdx.x / workers);
    const int rows = side ? 0 : (int)((long long)a.N * (blockIdx.x + 1) / workers) - n_begin;
    if (warp == 0) {
        if (lane == 0) {
            mbar_init(&bar_full, 1);
            s_abort = 0u;
            fence_barrier_init();
            mbar_expect_tx(&bar_full, (uint32_t)(rows * K));
        }
        __syncwarp();
        const int8_t *src = a.w_q + (size_t)n_begin * a.ldw;
        if (a.ldw == K) {
            if (lane == 0 && rows) bulk_load(smem, src, (uint32_t)(rows * K), &bar_full);
        } else {
            for (int r = lane; r < rows; r += 32) bulk_load(smem + (size_t)r * K, src + (size_t)r * a.ldw, (uint32_t)K, &bar_full);
        }
    }
    // this warp's rows, a lane each for scale, bias and result.  The bias is no constant of the layer (it may be what the launch
    // before this one stores, a residual): asked into L2 here, read behind the wait.
    const int per = (rows + kRowWarps - 1) / kRowWarps, r0 = warp * per, mine = max(min(per, rows - r0), 0);
    const int n_mine = n_begin + r0 + lane;
    const float sw = __ldg(a.s_w + (a.per_vec && lane < mine ? n_mine : 0));
    if (a.bias && lane < mine) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.bias + n_mine));
    for (int i = t * (int)gridDim.x + (int)blockIdx.x; i < (K + 63) >> 6; i += kRowT * (int)gridDim.x)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.X + i * 64));  // (see k_decode_fused)
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const float down = __int_as_float((127 - a.exp_factor) << 23);  // 2^-e
    const float qf = (float)a.qmax;
    uint4 v[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (lane + 32 * i < G) v[i] = ld_v4(reinterpret_cast<const uint4 *>(a.X) + lane + 32 * i);
    }
    const float bv = a.bias && lane < mine ? __ldcg(a.bias + n_mine) : 0.0f;
    // |x| > threshold for fp16 x: against the largest fp16 not above the threshold (strict, Section III-C)
    const __half2 tau2 = __half2half2(__float2half_rd(a.tau));
    uint32_t flagged = 0;  // bit i: chunk i of some lane of the warp holds an outlier channel
    float bmax = 0.0f;
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        const __half2 *h = reinterpret_cast<const __half2 *>(&v[i]);
        __half2 m = __hmax2(__hmax2(__habs2(h[0]), __habs2(h[1])), __hmax2(__habs2(h[2]), __habs2(h[3])));
        if (__any_sync(0xffffffffu, __hgt2_mask(m, tau2) != 0u)) {
            flagged |= 1u << i;
            float f[8];
            unpack8(v[i], f);
#pragma unroll
            for (int j = 0; j < 8; ++j) bmax = fmaxf(bmax, fabsf(f[j]) > a.tau ? fabsf(f[j]) * down : fabsf(f[j]));  // Eq. 4: exact
        } else {
            bmax = fmaxf(bmax, fmaxf(__low2float(m), __high2float(m)));
        }
    }
    const uint32_t mx = __reduce_max_sync(0xffffffffu, __float_as_uint(bmax));
    const float s = mx ? __fdiv_rn(__uint_as_float(mx), qf) : 1.0f;  // Eq. 1
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (see k_decode_fused)
    auto mask_of = [&](const uint4 &x) {
        float f[8];
        unpack8(x, f);
        uint32_t mask = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) mask |= (fabsf(f[j]) > a.tau ? 1u : 0u) << j;
        return mask;
    };
    if (side) {
        // ------------------------------------------------------------ reports (k_decode_fused)
        if (warp == 0) {
            int carry = 0;
#pragma unroll
            for (int i = 0; i < kC; ++i) {
                const int g = lane + 32 * i;
                if (g < G) {
                    float f[8];
                    unpack8(v[i], f);
                    reinterpret_cast<float4 *>(a.colmax)[2 * g] = make_float4(fabsf(f[0]), fabsf(f[1]), fabsf(f[2]), fabsf(f[3]));
                    reinterpret_cast<float4 *>(a.colmax)[2 * g + 1] = make_float4(fabsf(f[4]), fabsf(f[5]), fabsf(f[6]), fabsf(f[7]));
                }
                if (!((flagged >> i) & 1u)) continue;
                uint32_t m = mask_of(v[i]);
                const int cnt = __popc(m);
                int incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += n;
                }
                int pos = carry + incl - cnt;
                for (; m; m &= m - 1, ++pos)
                    if (pos < a.cap) a.outlier_idx[pos] = 8 * g + __ffs(m) - 1;
                carry += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) {
                a.ctrl->n_outliers = carry;
                if (a.per_vec) a.s_x_rows[0] = s;
                else {
                    a.ctrl->s_x = s;
                    a.ctrl->inv_s_x = __frcp_rn(s);
                }
                if (carry > a.cap && a.dev_status) atomicMax(a.dev_status, kStatusCapacity);
            }
        }
        return;
    }
    // codes; in flagged chunks also the masks of the outlier channels' bytes
    const float inv = __frcp_rn(s);
    float lo, hi;
    recip_bracket(inv, lo, hi);
    uint2 code[kC];
#pragma unroll
    for (int i = 0; i < kC; ++i) {
        float f[8];
        unpack8(v[i], f);
        uint32_t mask = 0;
        if ((flagged >> i) & 1u) {
            mask = mask_of(v[i]);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if ((mask >> j) & 1u) f[j] *= down;  // exact
        }
        if (bracket8(f, lo, hi, code[i])) code[i] = quotient8(f, inv, s);
        if ((flagged >> i) & 1u) {  // (the values are not needed any more: their place keeps the masks)
            v[i].x = ((mask & 15u) * 0x00204081u & 0x01010101u) * 0xFFu;
            v[i].y = ((mask >> 4) * 0x00204081u & 0x01010101u) * 0xFFu;
        }
    }
    const bool ok = mbar_wait_warp(&bar_full, 0u, &s_abort, a.spin);
    if (!ok) {  // (as in k_decode_fused)
        if (warp == 0)
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        if (lane == 0 && a.dev_status) atomicMax(a.dev_status, kStatusTimeout);
        return;
    }
    int acc = 0;  // lane j: output channel r0 + j
#pragma unroll 1
    for (int j = 0; j < mine; ++j) {
        const uint2 *w = reinterpret_cast<const uint2 *>(smem + (size_t)(r0 + j) * K) + lane;
        int body = 0, aux = 0;
#pragma unroll
        for (int i = 0; i < kC; ++i) {
            if (lane + 32 * i < G) {
                const uint2 x = w[32 * i];
                body = __dp4a((int)x.x, (int)code[i].x, body);
                body = __dp4a((int)x.y, (int)code[i].y, body);
                if ((flagged >> i) & 1u) {  // Aux_q == Body_q[:, O] (Eq. 5, shared scale)
                    aux = __dp4a((int)x.x, (int)(code[i].x & v[i].x), aux);
                    aux = __dp4a((int)x.y, (int)(code[i].y & v[i].y), aux);
                }
            }
        }
        const int sum = __reduce_add_sync(0xffffffffu, body + a.c * aux);  // Eq. 7
        if (lane == j) acc = sum;
    }
    if (lane < mine) {
        if (a.out_kind == 2) {
            reinterpret_cast<int32_t *>(a.Y)[n_mine] = acc;
        } else {
            float y = __fmul_rn(__fmul_rn(s, sw), __int2float_rn(acc));  // Eq. 3
            if (a.bias) y = __fadd_rn(y, bv);
            if (a.out_kind == 1) reinterpret_cast<float *>(a.Y)[n_mine] = y;
            else reinterpret_cast<__half *>(a.Y)[n_mine] = __float2half_rn(y);
        }
    }
}

}  // namespace

cudaError_t launch_row(const DecodeFusedArgs &a, const cudaLaunchConfig_t &cfg, int dev) {
    using Fn = void (*)(DecodeFusedArgs);
    static const Fn fns[5] = {k_decode_row<2>, k_decode_row<3>, k_decode_row<4>, k_decode_row<5>, k_decode_row<kRowMaxChunks>};
    static PerDevice<int> done[5];
    const int chunks = (a.K + 255) / 256, i = chunks <= 2 ? 0 : chunks - 2;
    const cudaError_t e = set_up(reinterpret_cast<const void *>(fns[i]), done[i], dev);
    return e != cudaSuccess ? e : cudaLaunchKernelEx(&cfg, fns[i], a);
}

}  // namespace decode
}  // namespace muxq
