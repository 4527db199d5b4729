// Logits x_i . z_t of a few token rows per warp against CC pivots, by warp-level products; shared by the kernel that
// builds the Gibbs kernel (lot_build.cu) and by the sweep kernel, which rebuilds it when the potentials have moved far.
// Accumulator layout: lane (g = lane / 4, q = lane % 4) holds rows g + 8 h (h < ROWS / 8), columns 8 j + 2 q + e.
#pragma once

#include "lot_common.cuh"

namespace lot {
namespace logits {

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f64(double &c0, double &c1, double a, double b)
{
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                 : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// two floats as N packed bf16 pairs
template <int N> __device__ __forceinline__ void split(float x, float y, uint32_t (&o)[N])
{
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
        o[i] = *reinterpret_cast<const uint32_t *>(&h);
        x -= __low2float(h);
        y -= __high2float(h);
    }
}

// Shared memory of one staged step of pivots.
template <typename T> __host__ __device__ constexpr size_t stage_bytes(int cc) { return sizeof(T) == 2 ? (size_t)cc * 80 * 3 : (size_t)cc * 18 * 8; }

// TERMS: bf16 terms a float32 pivot is taken as (bf16 tokens): 3 is exact, 2 is the precision of the tensor-core paths.
template <typename T, int CC, int ROWS, int THREADS, int TERMS = 3> struct Logits;

// bf16 tokens are exact operands; a float32 pivot is the exact sum of three bf16 terms, so the products are those of
// the float32 evaluation, summed in float32.  The next step's operands are in flight while the current one multiplies.
template <int CC, int THREADS, int TERMS> struct Logits<__nv_bfloat16, CC, 16, THREADS, TERMS> {
    typedef float LT;
    static constexpr int KC = 32, PITCH = 80, PLANE = CC * PITCH;     // 80-byte rows: conflict-free ldmatrix
    static constexpr int NZ = (CC * KC / 2 + THREADS - 1) / THREADS;  // pivot pairs a thread stages per step
    float acc[CC / 8][4];
    __device__ __forceinline__ void run(const __nv_bfloat16 *x, int rows, int d, const float *z, int zrows, uint8_t *stage, int lane)
    {
#pragma unroll
        for (int j = 0; j < CC / 8; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[j][e] = 0.f;
        const int g = lane >> 2, q = lane & 3;
        const uint32_t sb = (uint32_t)__cvta_generic_to_shared(stage);
        uint32_t a[2][4];
        float2 zz[NZ];
        auto fetch = [&](int k0) {
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int row = g + (e & 1) * 8, k = k0 + ks * 16 + (e >> 1) * 8 + 2 * q;
                    a[ks][e] = (row < rows && k < d) ? __ldg(reinterpret_cast<const unsigned *>(x + (size_t)row * d + k)) : 0u;
                }
#pragma unroll
            for (int u = 0; u < NZ; ++u) {
                const int idx = threadIdx.x + u * THREADS, t = idx / (KC / 2), k = k0 + (idx % (KC / 2)) * 2;
                zz[u] = (t < zrows && k < d) ? *reinterpret_cast<const float2 *>(z + (size_t)t * d + k) : make_float2(0.f, 0.f);
            }
        };
        fetch(0);
        for (int k0 = 0; k0 < d; k0 += KC) {
            __syncthreads();                                          // the previous step has been read
#pragma unroll
            for (int u = 0; u < NZ; ++u) {
                const int idx = threadIdx.x + u * THREADS, t = idx / (KC / 2), k = (idx % (KC / 2)) * 2;
                if (CC * KC / 2 % THREADS != 0 && t >= CC) break;
                uint8_t *p = stage + t * PITCH + k * 2;
                float2 v = zz[u];
#pragma unroll
                for (int term = 0; term < TERMS; ++term) {
                    const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
                    *reinterpret_cast<__nv_bfloat162 *>(p + term * PLANE) = h;
                    v.x -= __low2float(h);
                    v.y -= __high2float(h);
                }
            }
            uint32_t ac[2][4];
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                for (int e = 0; e < 4; ++e) ac[ks][e] = a[ks][e];
            __syncthreads();
            if (k0 + KC < d) fetch(k0 + KC);
            if (rows > 0) {
#pragma unroll
                for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                    for (int jp = 0; jp < CC / 16; ++jp) {
                        const uint32_t off = sb + (jp * 16 + (lane & 7) + (lane >> 4) * 8) * PITCH + (ks * 16 + ((lane >> 3) & 1) * 8) * 2;
#pragma unroll
                        for (int term = TERMS - 1; term >= 0; --term) {       // small terms first
                            uint32_t b[4];
                            ldsm4(b, off + term * PLANE);
                            mma_bf16(acc[2 * jp], ac[ks], b[0], b[1]);
                            mma_bf16(acc[2 * jp + 1], ac[ks], b[2], b[3]);
                        }
                    }
            }
        }
    }
    __device__ __forceinline__ LT &at(int j, int h, int e) { return acc[j][2 * h + e]; }
};

// float32 tokens: products and sums in float64 (logits C/eps of magnitude 1e3 need an absolute accuracy far below
// 1e-4).  Lane q of a quad reads four consecutive k of its row at once; product step s uses element s on both sides.
template <int CC, int ROWS, int THREADS, int TERMS> struct Logits<float, CC, ROWS, THREADS, TERMS> {
    typedef double LT;
    static constexpr int MT = ROWS / 8, KC = 16, PITCH = 18;          // pitch of 18 doubles: conflict-free 16-byte reads
    static constexpr int NZ = (CC * KC / 4 + THREADS - 1) / THREADS;
    double acc[MT][CC / 8][2];
    __device__ __forceinline__ void run(const float *x, int rows, int d, const float *z, int zrows, uint8_t *stage, int lane)
    {
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < CC / 8; ++j) { acc[m][j][0] = 0.0; acc[m][j][1] = 0.0; }
        const int g = lane >> 2, q = lane & 3;
        double *sz = reinterpret_cast<double *>(stage);
        float4 xa[MT], zz[NZ];
        auto fetch = [&](int k0) {
#pragma unroll
            for (int m = 0; m < MT; ++m)
                xa[m] = (g + 8 * m < rows && k0 + 4 * q < d) ? __ldg(reinterpret_cast<const float4 *>(x + (size_t)(g + 8 * m) * d + k0 + 4 * q))
                                                             : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < NZ; ++u) {
                const int idx = threadIdx.x + u * THREADS, t = idx / (KC / 4), k = k0 + (idx % (KC / 4)) * 4;
                zz[u] = (t < zrows && k < d) ? __ldg(reinterpret_cast<const float4 *>(z + (size_t)t * d + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        };
        fetch(0);
        for (int k0 = 0; k0 < d; k0 += KC) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < NZ; ++u) {
                const int idx = threadIdx.x + u * THREADS, t = idx / (KC / 4), k = (idx % (KC / 4)) * 4;
                if (CC * KC / 4 % THREADS != 0 && t >= CC) break;
                double *p = sz + t * PITCH + k;
                *reinterpret_cast<double2 *>(p) = make_double2((double)zz[u].x, (double)zz[u].y);
                *reinterpret_cast<double2 *>(p + 2) = make_double2((double)zz[u].z, (double)zz[u].w);
            }
            double xd[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m) { xd[m][0] = xa[m].x; xd[m][1] = xa[m].y; xd[m][2] = xa[m].z; xd[m][3] = xa[m].w; }
            __syncthreads();
            if (k0 + KC < d) fetch(k0 + KC);
            if (rows > 0) {
#pragma unroll
                for (int j = 0; j < CC / 8; ++j) {
                    const double *p = sz + (8 * j + g) * PITCH + 4 * q;
                    const double2 b0 = *reinterpret_cast<const double2 *>(p), b1 = *reinterpret_cast<const double2 *>(p + 2);
                    const double b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
                    for (int s = 0; s < 4; ++s)
#pragma unroll
                        for (int m = 0; m < MT; ++m) mma_f64(acc[m][j][0], acc[m][j][1], xd[m][s], b[s]);
                }
            }
        }
    }
    __device__ __forceinline__ LT &at(int j, int h, int e) { return acc[h][j][e]; }
};

} // namespace logits
} // namespace lot
