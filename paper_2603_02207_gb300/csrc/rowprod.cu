// Row products of CholeskyQR2 on double-float blocks: X R^-1 for an upper triangular R^-1, and the trace
// block [Q | G'] = [Q1 R2^-1 | G - Q1 C'] of Algorithm 3 steps 4 and 6 in one pass over Q1 and G
// (C' = R2^-1 R2^-T Q1^T G, so that Q1 C' = Q Q^T G).
//
// Bound by the double-float multiply-adds (12 f32x2 instructions for two of them) once the staging is
// out of the way: a tile's rows are one contiguous piece of the block, copied as it lies (no index
// arithmetic, no conversion pass), each lane reads its row in 16-byte pairs (two elements' leading and
// trailing parts), and whole pairs are written. One barrier a tile; several CTAs share an SM, so one
// computes while another waits, and every warp takes a short and a long column group.
// CholeskyQR2 and the deflation, against a kernel with a split pass and separate products with Q and G: 128^3,
// k = 33, DF64 6.8 -> 6.1 ms; n = 10^7, k = 10 6.8 -> 4.9 ms; five sketches of n = 2.25 million, k = 10
// 8.4 -> 6.2 ms. (Two CTAs of 18 warps an SM at 56 registers: 60 percent of the FMA pipe either way.)
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace ll {

namespace {

constexpr int RP_MAX_WARPS = 18;

template <int CP>
__device__ __forceinline__ void rp_copy(void* dst, const void* src) {
    if constexpr (CP == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// columns p .. p + cnt - 1 (cnt <= 4) of a row of column pairs: 16 bytes where both columns of a pair are
// the lane's, else the column's two floats
__device__ __forceinline__ void put_columns(float* row, int p, int cnt, const float (&h)[4], const float (&l)[4]) {
    float4* u = reinterpret_cast<float4*>(row + (p >> 1) * 4);
    float* f = reinterpret_cast<float*>(u);
    if (p & 1) {
        f[1] = h[0];
        f[3] = l[0];
        if (cnt > 2) {
            u[1] = make_float4(h[1], h[2], l[1], l[2]);
        } else if (cnt > 1) {
            f[4] = h[1];
            f[6] = l[1];
        }
        if (cnt > 3) {
            f[8] = h[3];
            f[10] = l[3];
        }
    } else {
        if (cnt > 1) {
            u[0] = make_float4(h[0], h[1], l[0], l[1]);
        } else {
            f[0] = h[0];
            f[2] = l[0];
        }
        if (cnt > 3) {
            u[1] = make_float4(h[2], h[3], l[2], l[3]);
        } else if (cnt > 2) {
            f[4] = h[2];
            f[6] = l[2];
        }
    }
}

struct RowProdParams {
    const float* X;        // n x kx double-float pairs, ldx columns (even)
    const double* M1;      // kx x kx upper triangular
    const double* M2;      // kx x kg (with G)
    const double* G;       // n x kg, or null
    float* out;            // double-float pairs, ldo columns
    long long ldx, ldo;
    int n, kx, kg, pad;    // pad: columns after the last set to zero
    int TR, CG1, CG2;      // rows per tile; groups of four columns of both parts
    int bufs;              // tiles in shared memory: 2, or 1 for the widest blocks
};

__global__ void __launch_bounds__(RP_MAX_WARPS * 32, 2) k_rows_df(const RowProdParams q) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int kx = q.kx, kxe = (kx + 1) & ~1;
    const int kc1 = 4 * q.CG1, kc2 = 4 * q.CG2;
    float* const m1h = reinterpret_cast<float*>(smem);
    float* const m1l = m1h + kxe * kc1;
    float* const m2h = m1l + kxe * kc1;
    float* const m2l = m2h + kxe * kc2;
    unsigned char* const stg = reinterpret_cast<unsigned char*>(m2l + kxe * kc2);
    const int xrow = (int)q.ldx * 8, grow = q.G ? q.kg * 8 : 0;
    const int xbytes = q.TR * xrow, gbytes = (q.TR * grow + 15) & ~15;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int ntiles = (int)(((long long)q.n + q.TR - 1) / q.TR);

    auto stage = [&](int tile, int buf) {
        if (tile < ntiles) {
            const int rows = min(q.TR, q.n - tile * q.TR);
            unsigned char* d = stg + (size_t)buf * (xbytes + gbytes);
            const unsigned char* s = reinterpret_cast<const unsigned char*>(q.X) + (size_t)tile * xbytes;
            for (int u = tid * 16; u < rows * xrow; u += nt * 16) rp_copy<16>(d + u, s + u);
            if (q.G) {
                d += xbytes;
                s = reinterpret_cast<const unsigned char*>(q.G) + (size_t)tile * q.TR * grow;
                const int full = rows * grow & ~15;
                for (int u = tid * 16; u < full; u += nt * 16) rp_copy<16>(d + u, s + u);
                if (tid == 0 && full < rows * grow) rp_copy<8>(d + full, s + full);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    stage(blockIdx.x, 0);
    for (int i = tid; i < kxe * kc1; i += nt) {
        const int a = i / kc1, c = i - a * kc1;
        float h = 0.f, l = 0.f;
        if (a < kx && c < kx) split_bits(q.M1[a * kx + c], h, l);
        m1h[i] = h;
        m1l[i] = l;
    }
    for (int i = tid; i < kxe * kc2; i += nt) {
        const int a = i / kc2, c = i - a * kc2;
        float h = 0.f, l = 0.f;
        if (a < kx && c < q.kg) split_bits(q.M2[a * q.kg + c], h, l);
        m2h[i] = h;
        m2l[i] = l;
    }
    const int CGT = q.CG1 + q.CG2, items = CGT * (q.TR / 32), nw = nt >> 5;
    int buf = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();   // the tile is there, and every thread is done with the other buffer
        if (q.bufs == 2) stage(tile + gridDim.x, buf ^ 1);
        const unsigned char* xb = stg + (size_t)buf * (xbytes + gbytes);
        for (int it = tid >> 5; it < items; it += nw) {
            // every other block of rows takes the column groups from the last: a warp's two items are a short
            // and a long one
            const int rb = it / CGT, rr = rb * 32 + lane;
            const int cg = rb & 1 ? CGT - 1 - (it - rb * CGT) : it - rb * CGT;
            const long long row = (long long)tile * q.TR + rr;
            if (row >= q.n) continue;
            const bool first = cg < q.CG1;
            const int g = first ? cg : cg - q.CG1, kc = first ? kc1 : kc2;
            const float* mh = (first ? m1h : m2h) + 4 * g;
            const float* ml = (first ? m1l : m2l) + 4 * g;
            const int amax = first ? min(kx, 4 * g + 4) : kx;
            const float4* x = reinterpret_cast<const float4*>(xb + (size_t)rr * xrow);
            f2x h01 = 0ull, l01 = 0ull, h23 = 0ull, l23 = 0ull;
            auto mac = [&](float xh, float xl, int a) {
                const f2x ah2 = f2_pack(xh, xh), al2 = f2_pack(xl, xl), nah2 = f2_pack(-xh, -xh);
                const ulonglong2 m4h = *reinterpret_cast<const ulonglong2*>(mh + a * kc);
                const ulonglong2 m4l = *reinterpret_cast<const ulonglong2*>(ml + a * kc);
                df2_mac(h01, l01, ah2, al2, nah2, m4h.x, m4l.x);
                df2_mac(h23, l23, ah2, al2, nah2, m4h.y, m4l.y);
            };
            int a = 0;
#pragma unroll 2
            for (; a + 2 <= amax; a += 2) {
                const float4 u = x[a >> 1];
                mac(u.x, u.z, a);
                mac(u.y, u.w, a + 1);
            }
            if (a < amax) {   // (the other half of the pair is a pad column: it may hold anything)
                const float4 u = x[a >> 1];
                mac(u.x, u.z, a);
            }
            float h[4], l[4];
            f2_unpack(h01, h[0], h[1]);
            f2_unpack(h23, h[2], h[3]);
            f2_unpack(l01, l[0], l[1]);
            f2_unpack(l23, l[2], l[3]);
            const int cols = min(4, (first ? kx : q.kg) - 4 * g);
            if (first) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 v = df_norm(h[j], l[j]);
                    h[j] = v.x;
                    l[j] = v.y;
                }
            } else {
                const double* gr = reinterpret_cast<const double*>(xb + xbytes + (size_t)rr * grow) + 4 * g;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j < cols) {
                        // G - (h + l): G split from its bits, TwoSum of the leading parts, renormalised
                        float gh, gl;
                        split_bits(gr[j], gh, gl);
                        const float sd = __fsub_rn(gh, h[j]);
                        const float bb = __fsub_rn(sd, gh);
                        float e = __fadd_rn(__fsub_rn(gh, __fsub_rn(sd, bb)), __fsub_rn(-h[j], bb));
                        e = __fadd_rn(e, __fsub_rn(gl, l[j]));
                        const float2 v = df_norm(sd, e);
                        h[j] = v.x;
                        l[j] = v.y;
                    }
                }
            }
            float* orow = q.out + (size_t)row * q.ldo * 2;
            put_columns(orow, (first ? 0 : kx) + 4 * g, cols, h, l);
            if (cg == CGT - 1)
                for (int z = 0; z < q.pad; ++z) {
                    const int c = kx + q.kg + z;
                    orow[(c >> 1) * 4 + (c & 1)] = 0.f;
                    orow[(c >> 1) * 4 + (c & 1) + 2] = 0.f;
                }
        }
        if (q.bufs == 2) {
            buf ^= 1;
        } else {
            __syncthreads();
            stage(tile + gridDim.x, 0);
        }
    }
}

// Cp = Rinv Rinv^T C (k x k upper triangular Rinv, C k x kc row-major): a warp per column
__global__ void __launch_bounds__(128) k_small_project(const double* Rinv, int k, const double* C, int kc, double* Cp) {
    extern __shared__ __align__(16) double sp[];
    double* R = sp;                                        // k x (k + 1)
    double* v = sp + k * (k + 1) + (threadIdx.x >> 5) * 2 * k;   // the warp's column, then R^-T of it
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < k * k; i += blockDim.x) R[(i / k) * (k + 1) + i % k] = Rinv[i];
    const int c = blockIdx.x * 4 + (threadIdx.x >> 5);
    if (c < kc)
        for (int i = lane; i < k; i += 32) v[i] = C[i * kc + c];
    __syncthreads();
    if (c >= kc) return;
    for (int i = lane; i < k; i += 32) {
        double s = 0.0;
        for (int l = 0; l <= i; ++l) s = fma(R[l * (k + 1) + i], v[l], s);
        v[k + i] = s;
    }
    __syncwarp();
    for (int i = lane; i < k; i += 32) {
        double s = 0.0;
        for (int l = i; l < k; ++l) s = fma(R[i * (k + 1) + l], v[k + l], s);
        Cp[i * kc + c] = s;
    }
}

cudaError_t rows_df_launch(RowProdParams q, cudaStream_t s) {
    if (q.n <= 0 || q.kx < 1) return cudaSuccess;
    if (q.ldx % 2 != 0 || q.kx > 96 || q.kg > 96) return cudaErrorInvalidValue;
    q.CG1 = (q.kx + 3) / 4;
    q.CG2 = q.G ? (q.kg + 3) / 4 : 0;
    const int CGT = q.CG1 + q.CG2;
    const int kxe = (q.kx + 1) & ~1;
    const size_t mats = (size_t)2 * kxe * 4 * CGT * sizeof(float);
    auto stage = [&](int RB) { return (size_t)RB * 32 * q.ldx * 8 + (q.G ? ((size_t)RB * 32 * q.kg * 8 + 15 & ~(size_t)15) : 0); };
    // about a dozen warps to a tile, each with two items of 32 rows x 4 columns; two tiles in shared memory, or
    // one of 32 rows for the widest blocks (k = 96: 147 KB of matrices, 49 KB a tile)
    int RB = 2 * std::max(1, std::min(4, 12 / CGT));
    while (RB > 1 && mats + 2 * stage(RB) > 227 * 1024) RB /= 2;
    q.bufs = mats + 2 * stage(RB) <= 227 * 1024 ? 2 : 1;
    q.TR = 32 * RB;
    const int warps = std::min(std::max(CGT * RB / 2, 1), RP_MAX_WARPS);
    const size_t smem = mats + q.bufs * stage(RB);
    cudaError_t e = allow_smem(k_rows_df);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rows_df, warps * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidValue;
    const int ntiles = (int)(((long long)q.n + q.TR - 1) / q.TR);
    k_rows_df<<<std::min(ntiles, per_sm * 152), warps * 32, smem, s>>>(q);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rows_rinv(const void* X, long long ldx, int n, int k, const double* Rinv, void* out, long long ldo, cudaStream_t s) {
    RowProdParams q{};
    q.X = static_cast<const float*>(X);
    q.M1 = Rinv;
    q.out = static_cast<float*>(out);
    q.ldx = ldx;
    q.ldo = ldo;
    q.n = n;
    q.kx = k;
    return rows_df_launch(q, s);
}

cudaError_t launch_rows_basis(const void* Q1, long long ldx, int n, int k, const double* Rinv, const double* Cp, const double* G, int kg,
                              void* out, long long ldo, int pad, cudaStream_t s) {
    RowProdParams q{};
    q.X = static_cast<const float*>(Q1);
    q.M1 = Rinv;
    q.M2 = Cp;
    q.G = G;
    q.out = static_cast<float*>(out);
    q.ldx = ldx;
    q.ldo = ldo;
    q.n = n;
    q.kx = k;
    q.kg = kg;
    q.pad = pad;
    return rows_df_launch(q, s);
}

cudaError_t launch_small_project(const double* Rinv, int k, const double* C, int kc, double* Cp, cudaStream_t s) {
    const size_t smem = ((size_t)k * (k + 1) + 8 * k) * sizeof(double);
    cudaError_t e = allow_smem(k_small_project);
    if (e != cudaSuccess) return e;
    k_small_project<<<(kc + 3) / 4, 128, smem, s>>>(Rinv, k, C, kc, Cp);
    return cudaGetLastError();
}

}  // namespace ll
