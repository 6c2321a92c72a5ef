// kd_mlp.cu -- the surrogate network: a fully connected MLP with exact-erf GELU hidden
// layers, trained on the batched solver's outputs (seeded parameter draws -> diffraction
// and spin-flip populations).  Hand-written kernels: tiled products with fused gather, bias,
// GELU, GELU derivative and loss epilogues (FP32 on the CUDA cores, or BF16 operands on the
// tcgen05 tensor cores with FP32 accumulation in tensor memory), fixed-order column sums, the
// loss sum and Adam.  Every reduction runs in a fixed order, so training is bitwise
// reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <math.h>

#include <vector>

#include "../../include/kd.h"

namespace kd {
int set_error(int code, const char* msg);  // kd_api.cu
}

struct kd_mlp {
    int device = 0;
    int L = 0;                       // number of layers (weight matrices)
    std::vector<int> w;              // widths, L + 1 entries
    std::vector<size_t> woff, boff;  // parameter offsets of W_l [w[l+1]][w[l]] and b_l
    size_t nparam = 0;
    float* param = nullptr;          // all W and b
    float* grad = nullptr;
    float* m1 = nullptr;             // Adam moments
    float* m2 = nullptr;
    long long adam_t = 0;
    int cap = 0;                     // batch capacity of the activation buffers
    std::vector<float*> z;           // pre-activations per layer [cap][w[l+1]]
    std::vector<float*> a;           // activations per layer output [cap][w[l+1]] (a[0] = input)
    float* dbuf0 = nullptr;          // gradient ping-pong buffers [cap][max width]
    float* dbuf1 = nullptr;
    float* lossbuf = nullptr;        // the loss, then [cap * w[L]] squared errors
    float* part = nullptr;           // partial gradients of layers whose batch is split
    size_t part_cap = 0;             // its floats
    int prec = 0;                    // KD_MLP_FP32 or KD_MLP_BF16 (tensor-core GEMMs)
    int* status = nullptr;           // set when a tensor-core GEMM's bounded wait gave up
};

namespace {

int err(int code, const char* msg) { return kd::set_error(code, msg); }

#define MLP_CUDA(call)                                                                   \
    do {                                                                                 \
        cudaError_t e_ = (call);                                                         \
        if (e_ != cudaSuccess) return err(e_ == cudaErrorMemoryAllocation ? KD_ERR_NOMEM : KD_ERR_CUDA, #call); \
    } while (0)

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// ------------------------------------------------------------ grouped products ----
// Every layer's products of one pass run in ONE launch: forward, one product; backward, the
// gradient for the layer below, the weight gradient and the bias gradient (column sums) side
// by side, since they only share their input dZ.  The network is small (a 256 x 256 x 256
// product is 0.9 us of the FP32 pipe), so a step is bound by the number of launches in its
// chain and by the load latency inside each one, not by arithmetic or memory: everything
// pointwise (gather, bias, GELU and its derivative, the loss' gradient) sits in an epilogue
// or a loader, and a launch starts under its predecessor's tail (programmatic dependent
// launch).  Such a launch may start before its predecessor's stores, so nothing here is read
// through the non-coherent path.  Chain of a training step: L forward launches, L backward
// launches, Adam.
//
// A step at batch 256 / FP32 went from 22 launches and 396 us to 9 launches and 43 us, at batch
// 1024 / BF16 from 401 to 73 us (GB300, the 5-256-256-256-4 network).  What bounds it now is
// the chain: nine dependent launches of 4-8 us, most of it launch and load latency.

// One operand P(row, k) of a product C[m][n] = sum_k A(m, k) B(n, k): element p[row ld + k]
// (kc) or p[k ld + row].  idx (may be null) selects the source row of the dimension that is
// not contiguous (row for kc, else k); an index outside [0, nidx) reads zeros.  vec: 16-byte
// loads along the contiguous dimension are aligned.
struct Operand {
    const float* p;
    long ld;
    const int32_t* idx;
    long nidx;
    int kc, vec;
};
enum Epi { EPI_STORE, EPI_BIAS, EPI_BIAS_GELU, EPI_BIAS_MSE, EPI_GELU_BACK };
// A product with its epilogue: STORE C = v; BIAS C = v + b; BIAS_GELU Z = v + b, C = GELU(Z);
// BIAS_MSE C = v + b, dY = scale (C - T), sq = (C - T)^2; GELU_BACK C = v GELU'(Z).  The k
// range runs in `splits` parts of kper, part s stored at C + s cstride.
struct Product {
    Operand A, B;
    float* C;
    long cstride;
    const float* bias;
    float* Z;
    const float* T;          // targets [nt][N], rows tidx[m] when tidx is set
    const int32_t* tidx;
    long nt;
    float* dY;
    float* sq;
    float scale;
    int M, N, K, epi;
    int bm, mt, nt_tiles, splits, kper;
};
// Column sums out[s][n] = sum over part s of the rows of X [M][N] (32 columns per CTA)
struct ColSum {
    const float* X;
    float* out;
    long ostride;
    int M, N, tiles, splits, mper;
};
// The mean of n squared errors into out[0] (and out2[0] when set), one CTA
struct LossSum {
    const float* sq;
    long n;
    float scale;
    float* out;
    float* out2;
};
struct Group {
    Product prod[2];
    ColSum col;
    LossSum loss;
    int first[5];            // first block of product 0, product 1, column sums, loss; total
    int* status;
};

// The epilogue of NE elements (m + i mstep, n + i nstep) of a tile, values v(i).  One loop
// per kind: a kernel of this size runs its code once, from a cold instruction cache, so the
// kind is decided outside the loop and the loop stays short (unrolled over every kind the
// BF16 epilogue took 14,000 cycles a tile).
template <int NE> __device__ __forceinline__ void epi_prefetch(const Product& q, int m, int mstep, int n, int nstep, float (&z)[NE]) {
    if (q.epi != EPI_GELU_BACK) return;
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        const int mi = m + i * mstep, ni = n + i * nstep;
        z[i] = mi < q.M && ni < q.N ? *(q.Z + (long)mi * q.N + ni) : 0.0f;
    }
}
template <int NE, int UNROLL, typename F>
__device__ __forceinline__ void epilogue(const Product& q, int m, int mstep, int n, int nstep, int split, const float (&z)[NE], F v) {
    auto each = [&](auto f) {
#pragma unroll UNROLL
        for (int i = 0; i < NE; ++i) {
            const int mi = m + i * mstep, ni = n + i * nstep;
            if (mi < q.M && ni < q.N) f(mi, ni, (long)mi * q.N + ni, v(i));
        }
    };
    if (q.epi == EPI_STORE) {
        float* C = q.C + (long)split * q.cstride;
        each([&](int, int, long o, float x) { C[o] = x; });
    } else if (q.epi == EPI_BIAS_GELU) {
        each([&](int, int ni, long o, float x) {
            x += *(q.bias + ni);
            q.Z[o] = x;
            q.C[o] = gelu(x);
        });
    } else if (q.epi == EPI_GELU_BACK) {
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const int mi = m + i * mstep, ni = n + i * nstep;
            if (mi < q.M && ni < q.N) q.C[(long)mi * q.N + ni] = v(i) * gelu_grad(z[i]);
        }
    } else if (q.epi == EPI_BIAS) {
        each([&](int, int ni, long o, float x) { q.C[o] = x + *(q.bias + ni); });
    } else {
        each([&](int mi, int ni, long o, float x) {
            const long r = q.tidx ? q.tidx[mi] : mi;
            const float t = !q.tidx || (r >= 0 && r < q.nt) ? *(q.T + r * q.N + ni) : 0.0f;
            x += *(q.bias + ni);
            q.C[o] = x;
            const float d = x - t;
            q.dY[o] = q.scale * d;
            q.sq[o] = d * d;
        });
    }
}

// fixed-order sum of the squared errors (256 threads)
__device__ void loss_block(const LossSum& l) {
    __shared__ double red[256];
    double s = 0.0;
    for (long i = threadIdx.x; i < l.n; i += 256) s += (double)l.sq[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const float v = (float)(red[0] * l.scale);
        l.out[0] = v;
        if (l.out2) l.out2[0] = v;
    }
}

// 32 columns of one part of the rows: eight row groups, each in order, then their sums in
// order (256 threads; one thread per column took 60 us for 256 rows, this disappears beside
// the products of its launch)
__device__ void colsum_block(const ColSum& c, int blk) {
    __shared__ float red[8][33];
    const int n = (blk % c.tiles) * 32 + (threadIdx.x & 31), split = blk / c.tiles, g = threadIdx.x >> 5;
    const int m1 = min(c.M, (split + 1) * c.mper);
    float s = 0.0f;
    if (n < c.N)
        for (int m = split * c.mper + g; m < m1; m += 8) s += *(c.X + (long)m * c.N + n);
    red[g][threadIdx.x & 31] = s;
    __syncthreads();
    if (g == 0 && n < c.N) {
        for (int i = 1; i < 8; ++i) s += red[i][threadIdx.x];
        c.out[(long)split * c.ostride + n] = s;
    }
}

// FP32 products on the CUDA cores: tiles of 32 columns and 16 or 32 rows (128 or 64 CTAs for a
// 256 x 256 output, where 64 x 64 tiles gave 16), 64-deep k slabs in a ring of four
// shared-memory stages filled by cp.async (zero-filled outside the operand), so that a K = 256
// product waits for the load latency once.  A slab's k range is shared by the eight warps,
// each with the whole tile (4 or 8 x 4 outputs a thread, 16-byte shared loads, two or one and
// a half per 16 FMAs), whose partial sums are added in a fixed order at the end.  A slab
// keeps its operand's own contiguous dimension: [rows][64 k] with 68 floats a row, a thread
// taking every 4th (columns: 8th) row (conflict-free 16-byte reads along k), or [64 k][rows]
// with four floats of padding, a thread taking consecutive rows.  64 x 64 tiles with one k
// group and 16-deep slabs of scalar loads took 44 us for 256^3 under ncu; this takes 5.
namespace fp32 {
constexpr int STAGES = 4, KS = 64, KP = KS + 4;
constexpr int BN = 32, PB = BN + 4, OPB = KS * PB;  // floats of an operand's slab of 32 rows
constexpr int SMEM = STAGES * 2 * OPB * 4;
static_assert(OPB >= BN * KP && STAGES * 2 * OPB >= 8 * 32 * PB, "slabs and reduction fit");

__device__ __forceinline__ void copy16(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy4(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}
// ROWS rows x 64 k of an operand into a slab, zeros outside its R rows and [.., kend): groups
// of four contiguous elements, ROWS / 16 per thread
template <int ROWS, bool KC> __device__ __forceinline__ void slab_load(float* sm, const Operand& o, int r0, int R, int k0, int kend) {
#pragma unroll
    for (int i = 0; i < ROWS / 16; ++i) {
        const int c = threadIdx.x + 256 * i;
        const int row = KC ? c >> 4 : 4 * (c % (ROWS / 4)), k = KC ? 4 * (c & 15) : c / (ROWS / 4);
        float* dst = sm + (KC ? row * KP + k : k * (ROWS + 4) + row);
        const int gr = r0 + row, gk = k0 + k, at = KC ? gk : gr;
        long line = KC ? gr : gk;
        int n = 4;   // elements inside
        if (gr >= R || gk >= kend) n = 0;
        else n = min(4, (KC ? kend : R) - at);
        if (o.idx && n > 0) {
            line = o.idx[line];
            if (line < 0 || line >= o.nidx) n = 0;
        }
        const float* src = n > 0 ? o.p + line * o.ld + at : o.p;
        if (o.vec) {
            copy16(dst, src, 4 * n);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) copy4(dst + e, e < n ? src + e : o.p, e < n ? 4 : 0);
        }
    }
}
// a thread's NT of a slab's LN NT rows at k .. k + 3, element [i][kk]: rows u + LN i of a slab
// contiguous in k, else rows NT u + i
template <int LN, int NT, bool KC> __device__ __forceinline__ void slab_read(const float* sm, int u, int k, float (&v)[NT][4]) {
    if constexpr (KC) {
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            const float4 q = *reinterpret_cast<const float4*>(sm + (u + LN * i) * KP + k);
            v[i][0] = q.x; v[i][1] = q.y; v[i][2] = q.z; v[i][3] = q.w;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < NT; i += 4) {
                const float4 q = *reinterpret_cast<const float4*>(sm + (k + e) * (LN * NT + 4) + NT * u + i);
                v[i][e] = q.x; v[i + 1][e] = q.y; v[i + 2][e] = q.z; v[i + 3][e] = q.w;
            }
    }
}

template <int BM, bool AKC, bool BKC> __device__ __forceinline__ void product(const Product& q, int blk, float* sm) {
    constexpr int TM = BM / 4, OPA = KS * (BM + 4), NE = BM / 8;   // rows a thread, A slab, outputs a thread
    static_assert(OPA >= BM * KP && OPA <= OPB, "A slab");
    const int t = threadIdx.x;
    const int n0 = (blk % q.nt_tiles) * BN, m0 = blk / q.nt_tiles % q.mt * BM, split = blk / (q.nt_tiles * q.mt);
    const int kbeg = split * q.kper, kend = min(q.K, kbeg + q.kper);
    const int nslab = (kend - kbeg + KS - 1) / KS;
    const int g = t >> 5, ty = (t & 31) >> 3, tx = t & 7;
    auto fill = [&](int j) {
        if (j < nslab) {
            float* st = sm + (j % STAGES) * (OPA + OPB);
            slab_load<BM, AKC>(st, q.A, m0, q.M, kbeg + KS * j, kend);
            slab_load<BN, BKC>(st + OPA, q.B, n0, q.N, kbeg + KS * j, kend);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int j = 0; j < STAGES - 1; ++j) fill(j);
    const int re = t / (BN / NE), ce = NE * (t % (BN / NE));   // this thread's outputs: NE of a row
    float z[NE];
    epi_prefetch<NE>(q, m0 + re, 0, n0 + ce, 1, z);
    float acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h) acc[i][h] = 0.0f;
    for (int j = 0; j < nslab; ++j) {
        asm volatile("cp.async.wait_group %0;" :: "n"(STAGES - 2) : "memory");
        __syncthreads();            // slab j has landed, slab j - 1's stage is free
        fill(j + STAGES - 1);
        const float* as = sm + (j % STAGES) * (OPA + OPB);
        const float* bs = as + OPA;
#pragma unroll
        for (int kk = 0; kk < 8; kk += 4) {
            float av[TM][4], bv[4][4];
            slab_read<4, TM, AKC>(as, ty, 8 * g + kk, av);
            slab_read<8, 4, BKC>(bs, tx, 8 * g + kk, bv);
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int i = 0; i < TM; ++i)
#pragma unroll
                    for (int h = 0; h < 4; ++h) acc[i][h] = fmaf(av[i][e], bv[h][e], acc[i][h]);
        }
    }
    // the eight groups' partial sums, through shared memory, added in order
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int h = 0; h < 4; ++h)
            sm[(g * BM + (AKC ? ty + 4 * i : TM * ty + i)) * PB + (BKC ? tx + 8 * h : 4 * tx + h)] = acc[i][h];
    __syncthreads();
    const float* r = sm + re * PB + ce;
    constexpr int G = BM * PB;
    epilogue<NE, NE>(q, m0 + re, 0, n0 + ce, 1, split, z, [&](int j) {
        return ((r[j] + r[G + j]) + (r[2 * G + j] + r[3 * G + j])) + ((r[4 * G + j] + r[5 * G + j]) + (r[6 * G + j] + r[7 * G + j]));
    });
}
}  // namespace fp32

// BF16 products on the 5th-generation tensor cores: the operands are rounded to BF16 (to
// nearest, from FP32) while staging, FP32 accumulation in tensor memory.  A CTA of 256
// threads computes a 128 x 16 tile of C (narrow tiles: the network's products are small, so
// more CTAs share them and each has half the epilogue of a 32-wide one).  The k range runs
// in 128-deep slabs through two shared-memory stages in the no-swizzle K-major canonical
// layout (8-row x 16-byte core matrices) with padded strides (LBO 144 bytes between core
// matrices along k, SBO 2320 between 8-row groups), so that neither load pattern's stores
// serialise on the banks.  While thread 0's tcgen05.mma.kind::f16 (M 128, N 16, K 16; A and
// B both BF16) of slab j run, committed to the stage's mbarrier, the threads load slab
// j + 1, wait for slab j - 1's products (bounded) and store into the stage those freed.
// Four warps read the accumulator rows back (warp w owns TMEM lanes 32 w ...) and hand them
// to all eight through shared memory for the epilogue.  A wait that runs out sets *status,
// the CTA issues no further products, waits (bounded) for those in flight and skips the
// epilogue; the host reports KD_ERR_TIMEOUT.  What bounds it is the latency of the slabs'
// loads (about 2,300 cycles each) and a cold instruction cache, not the matrix units (550
// cycles of waiting per tile), hence the short code paths.  Under ncu 1024 x 256 x 256 takes
// 8.8 us where 64-deep slabs loaded row by row by 128 threads took 15, and the weight
// gradient at batch 1024, split over eight parts of the batch, 11.4 us together with the
// gradient below, where 16 CTAs of 16 serial slabs took 43.
namespace tcg {
constexpr int BN = 16, KS = 128;                         // columns of C per CTA, slab depth
constexpr uint32_t LBO = 144, SBO = (KS / 8) * LBO + 16;
constexpr uint32_t A_BYTES = 16 * SBO, B_BYTES = (BN / 8) * SBO, STAGE = A_BYTES + B_BYTES;
constexpr uint32_t OFF_BAR = 2 * STAGE, OFF_SLOT = OFF_BAR + 16;
constexpr uint32_t SMEM = OFF_SLOT + 16;
constexpr uint32_t TMEM_COLS = 32;
// instruction descriptor (kind::f16): D FP32 (bits 4-5 = 1), A BF16 (bits 7-9 = 1), B BF16
// (bits 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(128 >> 4) << 24);
constexpr long long WAIT_LIMIT = 1ll << 20;
static_assert(STAGE % 16 == 0 && SBO % 16 == 0 && LBO % 16 == 0, "descriptor granularity");

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)((LBO >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((SBO >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const uint32_t a = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo));
    const uint32_t b = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi));
    return a | (b << 16);
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (long long it = 0; it < WAIT_LIMIT; ++it) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}
// ROWS rows x KS k of an operand, ROWS / 8 16-byte loads per thread (256 threads).  kc: a warp
// takes whole rows (512 contiguous bytes); !kc: a thread takes blocks of 4 rows x KB k (a warp
// 512 bytes of a k line, or 64 for 16 rows) and transposes them in registers.
__device__ __forceinline__ unsigned char* cell(unsigned char* dst, int row, int k) {
    return dst + (uint32_t)(row >> 3) * SBO + (uint32_t)(k >> 3) * LBO + (uint32_t)(row & 7) * 16 + (uint32_t)(k & 7) * 2;
}
// 16-deep products of the slab at k0
__device__ __forceinline__ int steps_of(int k0, int kend) { return min(KS, kend - k0 + 15) / 16; }
// A tile is whole (every line and k inside, 16-byte loads), or so small that there is little to
// wait for (few rows, or a single 16-deep step: read element by element at the store), or
// neither: edges, gathered rows, odd strides.  The last kind exists in the CHECKED kernel only,
// which the host picks where such a tile can occur (needs_checks): there too all of a thread's
// loads of the slab are in flight together, with every bound checked, 16-byte ones where the
// lines allow it, else scalar ones side by side across the warp.  (In one kernel with the whole
// tiles' short path the checks cost the 256-wide network's steps 3-4 %.)  With these tiles read
// element by element as well, a load latency per eight, a training step took, us: widths 1024,
// 2048, 2048, 64 on 1024 gathered rows 1361 (now 891), on 32 plain ones 399 (254); widths 511,
// 1023, 1023, 7 at batch 1024 620 (367); widths 5, 256, 256, 256, 4 at batch 200 116 (84).
template <int ROWS> struct Tile {
    float4 v[ROWS / 8];
    bool held;       // v holds the tile; else it is read element by element at the store
};
__host__ __device__ constexpr bool small_tile(int rows, int k) { return rows < 16 || k <= 16; }
template <int ROWS, bool KC, bool CHECKED>
__device__ __forceinline__ void tile_load(const Operand& o, int r0, int R, int k0, int kend, Tile<ROWS>& s) {
    const int t = threadIdx.x;
    constexpr int KB = ROWS == 128 ? 8 : 2;
    // this thread's first line (row, or k if !KC) and its place along the lines: four elements
    // there, side by side or (scalar loads) a quarter of the tile apart
    constexpr int Q = KC ? KS / 4 : ROWS / 4;
    const int line0 = KC ? r0 + (t >> 5) : k0 + KB * (t / Q), at = (KC ? k0 : r0) + (!CHECKED || o.vec ? 4 : 1) * (t % Q);
    const bool whole = o.vec && !o.idx && r0 + ROWS <= R && k0 + KS <= kend;
    s.held = CHECKED ? whole || !small_tile(R - r0, kend - k0) : whole;
    if (!s.held) return;
    if (!CHECKED || whole) {
        const float* p = o.p + (long)line0 * o.ld + at;
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i) {
            const long line = KC ? 8 * i : 64 * (i / KB) + i % KB;
            s.v[i] = *reinterpret_cast<const float4*>(p + line * o.ld);
        }
    } else {
        const int lines = KC ? R : kend, left = (KC ? kend : R) - at;   // elements along the lines
#pragma unroll
        for (int i = 0; i < ROWS / 8; ++i) {
            long line = line0 + (KC ? 8 * i : 64 * (i / KB) + i % KB);
            bool in = line < lines && left > 0;
            if (in && o.idx) {
                line = o.idx[line];
                in = line >= 0 && line < o.nidx;
            }
            float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (in) {
                const float* p = o.p + line * o.ld + at;
                if (o.vec) {   // the extent is a multiple of four, as the stride is
                    x = *reinterpret_cast<const float4*>(p);
                } else {
                    x.x = p[0];
                    if (left > Q) x.y = p[Q];
                    if (left > 2 * Q) x.z = p[2 * Q];
                    if (left > 3 * Q) x.w = p[3 * Q];
                }
            }
            s.v[i] = x;
        }
    }
}
__device__ __forceinline__ float elem(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }
template <int ROWS, bool KC, bool CHECKED>
__device__ __forceinline__ void tile_store(unsigned char* dst, const Operand& o, int r0, int R, int k0, int kend, const Tile<ROWS>& s) {
    const int t = threadIdx.x;
    const bool side = !CHECKED || o.vec;   // a thread's four elements of a line lie side by side
    if (!s.held) {
        // element by element, zeros outside, up to the last 16-deep step that holds any k
#pragma unroll 1
        for (int c = t; c < ROWS * 2 * steps_of(k0, kend); c += 256) {
            const int row = r0 + c % ROWS, k = k0 + 8 * (c / ROWS);
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                bool in = row < R && k + e < kend;
                long line = KC ? row : k + e;
                if (in && o.idx) {
                    line = o.idx[line];
                    in = line >= 0 && line < o.nidx;
                }
                v[e] = in ? *(o.p + line * o.ld + (KC ? k + e : row)) : 0.0f;
            }
            *reinterpret_cast<uint4*>(cell(dst, row - r0, k - k0)) =
                make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
        }
    } else if constexpr (KC) {
        if (side) {
#pragma unroll
            for (int i = 0; i < ROWS / 8; ++i)
                *reinterpret_cast<uint2*>(cell(dst, (t >> 5) + 8 * i, 4 * (t & 31))) =
                    make_uint2(pack_bf16(s.v[i].x, s.v[i].y), pack_bf16(s.v[i].z, s.v[i].w));
        } else {
#pragma unroll
            for (int i = 0; i < ROWS / 8; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    *reinterpret_cast<__nv_bfloat16*>(cell(dst, (t >> 5) + 8 * i, (t & 31) + 32 * e)) = __float2bfloat16_rn(elem(s.v[i], e));
        }
    } else if constexpr (ROWS == 128) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                *reinterpret_cast<uint4*>(cell(dst, side ? 4 * (t & 31) + e : (t & 31) + 32 * e, 8 * (t >> 5) + 64 * i)) =
                    make_uint4(pack_bf16(elem(s.v[8 * i + 0], e), elem(s.v[8 * i + 1], e)),
                               pack_bf16(elem(s.v[8 * i + 2], e), elem(s.v[8 * i + 3], e)),
                               pack_bf16(elem(s.v[8 * i + 4], e), elem(s.v[8 * i + 5], e)),
                               pack_bf16(elem(s.v[8 * i + 6], e), elem(s.v[8 * i + 7], e)));
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
            *reinterpret_cast<uint32_t*>(cell(dst, side ? 4 * (t & 3) + e : (t & 3) + 4 * e, 2 * (t >> 2))) = pack_bf16(elem(s.v[0], e), elem(s.v[1], e));
    }
}
}  // namespace tcg

template <bool AKC, bool BKC, bool CHECKED>
__device__ __forceinline__ void product_bf16(const Product& q, int blk, int* status, unsigned char* sm) {
    const int t = threadIdx.x, w = t >> 5;
    const int n0 = (blk % q.nt_tiles) * tcg::BN, m0 = blk / q.nt_tiles % q.mt * 128, split = blk / (q.nt_tiles * q.mt);
    const int kbeg = split * q.kper, kend = min(q.K, kbeg + q.kper);
    const uint32_t s0 = tcg::su32(sm);
    const uint32_t bar[2] = {s0 + tcg::OFF_BAR, s0 + tcg::OFF_BAR + 8};
    if (w == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(s0 + tcg::OFF_SLOT), "r"(tcg::TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (t == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar[0]));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(bar[1]));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int nslab = (kend - kbeg + tcg::KS - 1) / tcg::KS;
    uint32_t phase[2] = {0u, 0u};
    bool ok = true;
    int issued = 0;          // slabs whose products were issued (and committed)
    int waited = 0;          // slabs whose products were waited for
    tcg::Tile<128> ta;
    tcg::Tile<tcg::BN> tb;
    if (nslab > 0) {
        tcg::tile_load<128, AKC, CHECKED>(q.A, m0, q.M, kbeg, kend, ta);
        tcg::tile_load<tcg::BN, BKC, CHECKED>(q.B, n0, q.N, kbeg, kend, tb);
        tcg::tile_store<128, AKC, CHECKED>(sm, q.A, m0, q.M, kbeg, kend, ta);
        tcg::tile_store<tcg::BN, BKC, CHECKED>(sm + tcg::A_BYTES, q.B, n0, q.N, kbeg, kend, tb);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<const uint32_t*>(sm + tcg::OFF_SLOT);
    for (int j = 0; j < nslab && ok; ++j) {
        const int b = j & 1;
        if (t == 0) {
            const uint32_t sa = s0 + (uint32_t)b * tcg::STAGE;
#pragma unroll
            for (int ks = 0; ks < tcg::KS / 16; ++ks) {
                if (ks >= tcg::steps_of(kbeg + tcg::KS * j, kend)) break;
                const uint64_t da = tcg::sdesc(sa + (uint32_t)ks * 2 * tcg::LBO);
                const uint64_t db = tcg::sdesc(sa + tcg::A_BYTES + (uint32_t)ks * 2 * tcg::LBO);
                const uint32_t acc = (j > 0 || ks > 0) ? 1u : 0u;
                asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                             "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                             :: "r"(tmem), "l"(da), "l"(db), "r"(tcg::IDESC), "r"(acc));
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                         :: "r"(bar[b]) : "memory");
        }
        issued = j + 1;
        // the next slab's global loads run while these products do
        if (j + 1 < nslab) {
            tcg::tile_load<128, AKC, CHECKED>(q.A, m0, q.M, kbeg + tcg::KS * (j + 1), kend, ta);
            tcg::tile_load<tcg::BN, BKC, CHECKED>(q.B, n0, q.N, kbeg + tcg::KS * (j + 1), kend, tb);
        }
        bool got = true;
        if (j >= 1) {   // slab j - 1's products read the stage slab j + 1 goes to
            got = tcg::mbar_wait(bar[b ^ 1], phase[b ^ 1]);
            if (got) {
                phase[b ^ 1] ^= 1u;
                waited = j;
            }
        }
        if (got && j + 1 < nslab) {
            unsigned char* st = sm + (uint32_t)(b ^ 1) * tcg::STAGE;
            tcg::tile_store<128, AKC, CHECKED>(st, q.A, m0, q.M, kbeg + tcg::KS * (j + 1), kend, ta);
            tcg::tile_store<tcg::BN, BKC, CHECKED>(st + tcg::A_BYTES, q.B, n0, q.N, kbeg + tcg::KS * (j + 1), kend, tb);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        ok = __syncthreads_and(got) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    // the last issued slab's products (and, after a failed wait, those still in flight:
    // each wait bounded, the first that runs out ends them)
    while (waited < issued) {
        const int b = waited & 1;
        if (!tcg::mbar_wait(bar[b], phase[b])) {
            ok = false;
            break;
        }
        phase[b] ^= 1u;
        ++waited;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    ok = __syncthreads_and(ok) != 0;
    if (ok && nslab > 0 && w < 4) {
        // row m0 + t's 16 columns from TMEM lane t
        const uint32_t trow = tmem + ((uint32_t)(w * 32) << 16);
        uint32_t r[16];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                     "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                       "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                       "=r"(r[14]), "=r"(r[15])
                     : "r"(trow));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        // transposed through shared memory (the stages' products are done), so that the
        // epilogue's global accesses run along the rows
        float* tr = reinterpret_cast<float*>(sm);
#pragma unroll
        for (int j = 0; j < tcg::BN; ++j) tr[t * 17 + j] = __uint_as_float(r[j]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok && nslab > 0) {
        const float* tr = reinterpret_cast<const float*>(sm) + (t >> 4) * 17 + (t & 15);
        float z[8];
        epi_prefetch<8>(q, m0 + (t >> 4), 16, n0 + (t & 15), 0, z);
        epilogue<8, 2>(q, m0 + (t >> 4), 16, n0 + (t & 15), 0, split, z, [&](int i) { return tr[16 * i * 17]; });
    }
    if (!ok && t == 0) atomicOr(status, 1);
    if (w == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(tcg::TMEM_COLS));
}

// One launch of a pass: the block index selects the product (and its tile and part), the
// column sums or the loss.  KIND 0: FP32; 1: BF16, whole or small tiles; 2: BF16, checked tiles.
template <int KIND> __global__ void __launch_bounds__(256, 2) k_group(const __grid_constant__ Group g) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    const int blk = blockIdx.x;
    if (blk >= g.first[3]) {
        loss_block(g.loss);
    } else if (blk >= g.first[2]) {
        colsum_block(g.col, blk - g.first[2]);
    } else {
        // the orientations that occur: forward (rows x rows), the gradient below (rows x
        // columns), the weight gradient (columns x columns)
        // by value: read once into registers (a reference into the parameter block is read
        // again after every store, 7 us per tile)
        Product q = g.prod[0];
        int b = blk;
        if (blk >= g.first[1]) {
            q = g.prod[1];
            b -= g.first[1];
        }
        extern __shared__ __align__(1024) unsigned char sm[];
        if constexpr (KIND != 0) {
            if (!q.A.kc) product_bf16<false, false, KIND == 2>(q, b, g.status, sm);
            else if (q.B.kc) product_bf16<true, true, KIND == 2>(q, b, g.status, sm);
            else product_bf16<true, false, KIND == 2>(q, b, g.status, sm);
        } else {
            float* f = reinterpret_cast<float*>(sm);
            if (q.bm == 16) {
                if (!q.A.kc) fp32::product<16, false, false>(q, b, f);
                else if (q.B.kc) fp32::product<16, true, true>(q, b, f);
                else fp32::product<16, true, false>(q, b, f);
            } else {
                if (!q.A.kc) fp32::product<32, false, false>(q, b, f);
                else if (q.B.kc) fp32::product<32, true, true>(q, b, f);
                else fp32::product<32, true, false>(q, b, f);
            }
        }
    }
}

// Where the gradient of each layer lies: `parts` partial sums (over parts of the batch) at
// src + s stride, each [W_l | b_l]; off[l] is the layer's first parameter, off[L] the count.
struct GradParts {
    int L;
    long off[17];
    const float* src[16];
    long stride[16];
    int parts[16];
};
__device__ __forceinline__ float grad_of(const GradParts& q, long i) {
    int l = 0;
    while (l + 1 < q.L && i >= q.off[l + 1]) ++l;
    const float* p = q.src[l] + (i - q.off[l]);
    float g = p[0];
    for (int s = 1; s < q.parts[l]; ++s) g += p[s * q.stride[l]];
    return g;
}
__global__ void k_sum_parts(const __grid_constant__ GradParts q, float* out) {
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < q.off[q.L]; i += (long)gridDim.x * blockDim.x)
        out[i] = grad_of(q, i);
}

__global__ void k_adam(float* p, const __grid_constant__ GradParts q, float* m1, float* m2, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;");
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < q.off[q.L]; i += (long)gridDim.x * blockDim.x) {
        const float gi = grad_of(q, i);
        const float a = b1 * m1[i] + (1.0f - b1) * gi;
        const float b = b2 * m2[i] + (1.0f - b2) * gi * gi;
        m1[i] = a;
        m2[i] = b;
        p[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
    }
}

// ---------------------------------------------------------------- host side -------
Operand operand(const float* p, long ld, bool kc, const int32_t* idx = nullptr, long nidx = 0) {
    const bool vec = ld % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0;
    return Operand{p, ld, idx, nidx, kc ? 1 : 0, vec ? 1 : 0};
}

// Tiles of the product at the network's precision, its k range in `splits` parts.  FP32: 16-row
// tiles while 32-row ones would leave SMs without one (256 x 256 outputs: 64 tiles), since what
// counts there is one tile's latency; else 32 rows, which read half as much per output (a step
// at batch 256 42.9 us against 51.2 with 32 rows only; at batch 1024 78.8 with 16 rows only
// against 74.6).  The tiles are drawn for the 256-wide network.  Wider ones read an operand more
// often than 64 x 64 (FP32) and 128 x 32 (BF16) tiles did, and are still faster (widths 1024,
// 2048, 2048, 64 at batch 4096: FP32 10.1 -> 4.8 ms, BF16 3.7 -> 2.7), but for BF16 with rows
// of odd length from 2049 on at batch 1024 and more (1.29 -> 1.50 ms).
void tile(const kd_mlp* n, Product* q, int splits) {
    const bool bf = n->prec == KD_MLP_BF16;
    const int bn = bf ? tcg::BN : fp32::BN;
    q->nt_tiles = (q->N + bn - 1) / bn;
    q->bm = bf ? 128 : ((q->M + 31) / 32 * q->nt_tiles * splits < 152 ? 16 : 32);
    q->mt = (q->M + q->bm - 1) / q->bm;
    q->splits = splits;
    q->kper = (q->K + splits - 1) / splits;
}
long blocks(const Product& q) { return (long)q.mt * q.nt_tiles * q.splits; }

template <typename... KP, typename... KA>
cudaError_t launch_pdl(void (*k)(KP...), long grid, int threads, int smem, cudaStream_t s, KA... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

// Lets the products' kernel of a precision take its dynamic shared memory on the current
// device.  The limit belongs to one device's copy of the kernel, so every network sets it for
// its own device (kd_mlp_create, kd_mlp_set_precision) and nothing remembers it.
cudaError_t allow_smem(int precision) {
    constexpr cudaFuncAttribute attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    if (precision != KD_MLP_BF16) return cudaFuncSetAttribute(k_group<0>, attr, fp32::SMEM);
    const cudaError_t e = cudaFuncSetAttribute(k_group<1>, attr, (int)tcg::SMEM);
    return e == cudaSuccess ? cudaFuncSetAttribute(k_group<2>, attr, (int)tcg::SMEM) : e;
}

// Whether a tile of a BF16 product can be neither whole nor small (tcg::Tile): its operand has
// rows x k elements, k in parts of kper.
bool needs_checks(const Operand& o, int tile_rows, int rows, int k, int kper) {
    if (tcg::small_tile(rows, kper)) return false;
    return !o.vec || o.idx || rows % tile_rows != 0 || k % tcg::KS != 0 || kper % tcg::KS != 0;
}
bool needs_checks(const Group& g, int nprod) {
    for (int i = 0; i < nprod; ++i) {
        const Product& q = g.prod[i];
        if (needs_checks(q.A, 128, q.M, q.K, q.kper) || needs_checks(q.B, tcg::BN, q.N, q.K, q.kper)) return true;
    }
    return false;
}

// A pass's launches in order, all by one kernel: the BF16 kernel with checks for every launch
// if any needs it (alternating between the two, each with a cold instruction cache, a forward
// pass of the 256-wide network at batch 32 took 47 us; 35 with one).
struct Pass {
    Group g[16];
    int nprod[16];
    int n = 0;
};
cudaError_t launch_group(const kd_mlp* n, Group& g, int nprod, bool checks, cudaStream_t s) {
    long b = 0;
    for (int i = 0; i < 2; ++i) {
        g.first[i] = (int)b;
        if (i < nprod) b += blocks(g.prod[i]);
    }
    g.first[2] = (int)b;
    b += (long)g.col.tiles * g.col.splits;
    g.first[3] = (int)b;
    b += g.loss.n > 0 ? 1 : 0;
    g.first[4] = (int)b;
    if (b > 0x7fffffffL) return cudaErrorInvalidValue;
    g.status = n->status;
    const bool bf = n->prec == KD_MLP_BF16;
    // BF16: two 41 KB stages and 32 columns of tensor memory per CTA: two CTAs per SM, whose
    // columns fit the SM's 512, so no allocation waits
    const int smem = bf ? (int)tcg::SMEM : fp32::SMEM;
    if (!bf) return launch_pdl(k_group<0>, b, 256, smem, s, g);
    return checks ? launch_pdl(k_group<2>, b, 256, smem, s, g) : launch_pdl(k_group<1>, b, 256, smem, s, g);
}

cudaError_t launch_pass(const kd_mlp* n, Pass& p, cudaStream_t s) {
    bool checks = false;
    for (int i = 0; i < p.n && n->prec == KD_MLP_BF16; ++i) checks = checks || needs_checks(p.g[i], p.nprod[i]);
    for (int i = 0; i < p.n; ++i) {
        const cudaError_t e = launch_group(n, p.g[i], p.nprod[i], checks, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// KD_ERR_TIMEOUT (and the flag cleared) when a tensor-core GEMM's bounded wait gave up
// since the last check; synchronises the device
int check_status(kd_mlp* n) {
    int st = 0;
    MLP_CUDA(cudaMemcpy(&st, n->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (!st) return KD_OK;
    MLP_CUDA(cudaMemset(n->status, 0, sizeof(int)));
    return err(KD_ERR_TIMEOUT, "kd_mlp: a tensor-core GEMM's wait for its products gave up");
}

int maxw(const kd_mlp* n) {
    int m = 0;
    for (int v : n->w) m = v > m ? v : m;
    return m;
}

// Parts of the batch the weight gradient of an fo x fi layer is summed in: enough for about
// two CTAs on every SM when its tiles alone leave most of them idle, at least 128 (BF16: one
// slab) or 256 rows each, at most eight.
int grad_parts(int precision, int fo, int fi, int rows) {
    const bool bf = precision == KD_MLP_BF16;
    const int bm = bf ? 128 : 32, least = bf ? 128 : 256;
    const int bn = bf ? tcg::BN : 32;
    const long tiles = (long)((fo + bm - 1) / bm) * ((fi + bn - 1) / bn);
    const long fill = (304 + tiles - 1) / tiles, depth = rows / least;
    const long p = fill < depth ? fill : depth;
    return (int)(p < 1 ? 1 : p > 8 ? 8 : p);
}

// Room for the partial gradients of any batch up to `rows` (more rows never take fewer parts) at
// a precision.  Made with the batch buffers and at a change of precision, so that a step at a
// batch size already seen allocates nothing (it may be inside a stream capture).
int ensure_part(kd_mlp* n, int precision, int rows) {
    size_t need = 0;
    for (int l = 0; l < n->L; ++l) {
        const int parts = grad_parts(precision, n->w[l + 1], n->w[l], rows);
        if (parts > 1) need += ((size_t)n->w[l + 1] * n->w[l] + n->w[l + 1]) * parts;
    }
    if (need <= n->part_cap) return KD_OK;
    cudaFree(n->part);
    n->part = nullptr;
    n->part_cap = 0;
    MLP_CUDA(cudaMalloc(&n->part, need * sizeof(float)));
    n->part_cap = need;
    return KD_OK;
}

int ensure_cap(kd_mlp* n, int batch) {
    if (batch <= n->cap) return KD_OK;
    for (float* p : n->z) cudaFree(p);
    for (size_t l = 1; l < n->a.size(); ++l) cudaFree(n->a[l]);
    cudaFree(n->dbuf0);
    cudaFree(n->dbuf1);
    cudaFree(n->lossbuf);
    // nothing is left to use or free again if one of the allocations below fails
    n->cap = 0;
    n->dbuf0 = n->dbuf1 = n->lossbuf = nullptr;
    n->z.assign(n->L, nullptr);
    n->a.assign(n->L + 1, nullptr);
    for (int l = 0; l < n->L; ++l) {
        MLP_CUDA(cudaMalloc(&n->z[l], sizeof(float) * (size_t)batch * n->w[l + 1]));
        MLP_CUDA(cudaMalloc(&n->a[l + 1], sizeof(float) * (size_t)batch * n->w[l + 1]));
    }
    MLP_CUDA(cudaMalloc(&n->dbuf0, sizeof(float) * (size_t)batch * maxw(n)));
    MLP_CUDA(cudaMalloc(&n->dbuf1, sizeof(float) * (size_t)batch * maxw(n)));
    MLP_CUDA(cudaMalloc(&n->lossbuf, sizeof(float) * ((size_t)batch * n->w[n->L] + 1)));
    const int rc = ensure_part(n, n->prec, batch);
    if (rc) return rc;
    n->cap = batch;
    return KD_OK;
}

// A minibatch on the device: rows of x and t (targets, may be null), or rows idx[.] of nsrc
struct Batch {
    const float* x;
    const float* t;
    const int32_t* idx;
    long nsrc;
    int rows;
};

// forward pass: a[l+1] = act(a[l] W_l^T + b_l); the last layer is linear (its output is
// a[L]) and, with targets, also writes the loss' gradient to dbuf0 and the squared errors
int forward(kd_mlp* n, const Batch& in, cudaStream_t s) {
    const long nout = (long)in.rows * n->w[n->L];
    Pass pass{};
    for (int l = 0; l < n->L; ++l) {
        const int fi = n->w[l], fo = n->w[l + 1];
        const bool last = l == n->L - 1;
        pass.nprod[pass.n] = 1;
        Group& g = pass.g[pass.n++];
        Product& q = g.prod[0];
        q.A = l == 0 ? operand(in.x, fi, true, in.idx, in.nsrc) : operand(n->a[l], fi, true);
        q.B = operand(n->param + n->woff[l], fi, true);
        q.C = n->a[l + 1];
        q.bias = n->param + n->boff[l];
        q.Z = last ? nullptr : n->z[l];
        q.M = in.rows;
        q.N = fo;
        q.K = fi;
        q.epi = !last ? EPI_BIAS_GELU : in.t ? EPI_BIAS_MSE : EPI_BIAS;
        if (last && in.t) {
            q.T = in.t;
            q.tidx = in.idx;
            q.nt = in.nsrc;
            q.dY = n->dbuf0;
            q.sq = n->lossbuf + 1;
            q.scale = 2.0f / (float)nout;
        }
        tile(n, &q, 1);
    }
    MLP_CUDA(launch_pass(n, pass, s));
    return KD_OK;
}

// Gradients after forward() with targets: layer l's partial sums where `gp` says, the mean
// squared error in lossbuf[0] (and *loss2).
int backward(kd_mlp* n, const Batch& in, GradParts* gp, float* loss2, cudaStream_t s) {
    const int L = n->L;
    gp->L = L;
    for (int l = 0; l < L; ++l) {
        const size_t cnt = (size_t)n->w[l + 1] * n->w[l] + n->w[l + 1];
        gp->off[l] = (long)n->woff[l];
        gp->parts[l] = grad_parts(n->prec, n->w[l + 1], n->w[l], in.rows);
        gp->stride[l] = (long)cnt;
    }
    gp->off[L] = (long)n->nparam;
    float* at = n->part;
    float* dcur = n->dbuf0;   // dZ_l
    float* dnext = n->dbuf1;
    Pass pass{};
    for (int l = L - 1; l >= 0; --l) {
        const int fi = n->w[l], fo = n->w[l + 1], parts = gp->parts[l];
        float* dst = n->grad + n->woff[l];
        if (parts > 1) {
            dst = at;
            at += gp->stride[l] * parts;
        }
        gp->src[l] = dst;
        Group& g = pass.g[pass.n];
        int np = 0;
        if (l > 0) {  // dZ_{l-1}[b][i] = (sum_o dZ[b][o] W_l[o][i]) GELU'(Z_{l-1}[b][i])
            Product& q = g.prod[np++];
            q.A = operand(dcur, fo, true);
            q.B = operand(n->param + n->woff[l], fi, false);
            q.C = dnext;
            q.Z = n->z[l - 1];
            q.M = in.rows;
            q.N = fi;
            q.K = fo;
            q.epi = EPI_GELU_BACK;
            tile(n, &q, 1);
        }
        // dW_l[o][i] = sum_b dZ[b][o] a_l[b][i];  db_l[o] = sum_b dZ[b][o]
        Product& q = g.prod[np++];
        q.A = operand(dcur, fo, false);
        q.B = l == 0 ? operand(in.x, fi, false, in.idx, in.nsrc) : operand(n->a[l], fi, false);
        q.C = dst;
        q.cstride = gp->stride[l];
        q.M = fo;
        q.N = fi;
        q.K = in.rows;
        q.epi = EPI_STORE;
        tile(n, &q, parts);
        g.col = ColSum{dcur, dst + (size_t)fo * fi, gp->stride[l], in.rows, fo, (fo + 31) / 32, parts, q.kper};
        if (l == L - 1) {
            const long nout = (long)in.rows * fo;
            g.loss = LossSum{n->lossbuf + 1, nout, 1.0f / (float)nout, n->lossbuf, loss2};
        }
        pass.nprod[pass.n++] = np;
        float* tmp = dcur;
        dcur = dnext;
        dnext = tmp;
    }
    MLP_CUDA(launch_pass(n, pass, s));
    return KD_OK;
}

int copy_io(void* dst, const void* src, size_t bytes, int32_t where_dst, int32_t where_src, cudaStream_t s) {
    cudaMemcpyKind k = where_src == KD_HOST ? (where_dst == KD_HOST ? cudaMemcpyHostToHost : cudaMemcpyHostToDevice)
                                            : (where_dst == KD_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice);
    MLP_CUDA(cudaMemcpyAsync(dst, src, bytes, k, s));
    return KD_OK;
}

// the gradients in one buffer (grad): layers summed in parts are added up into it
int gather_grads(kd_mlp* n, GradParts& gp, cudaStream_t s) {
    bool split = false;
    for (int l = 0; l < gp.L; ++l) split = split || gp.parts[l] > 1;
    if (!split) return KD_OK;
    k_sum_parts<<<(int)((n->nparam + 255) / 256), 256, 0, s>>>(gp, n->grad);
    MLP_CUDA(cudaGetLastError());
    return KD_OK;
}

int train_step(kd_mlp* n, const Batch& in, float lr, float* loss_dev, cudaStream_t s) {
    MLP_CUDA(cudaSetDevice(n->device));
    int rc = ensure_cap(n, in.rows);
    if (rc) return rc;
    GradParts gp;
    rc = forward(n, in, s);
    if (!rc) rc = backward(n, in, &gp, loss_dev, s);
    if (rc) return rc;
    ++n->adam_t;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - powf(b1, (float)n->adam_t), c2 = 1.0f - powf(b2, (float)n->adam_t);
    MLP_CUDA(launch_pdl(k_adam, (long)((n->nparam + 255) / 256), 256, 0, s, n->param, gp, n->m1, n->m2, lr, b1, b2,
                        1e-8f, c1, c2));
    return KD_OK;
}

}  // namespace

extern "C" {

int kd_mlp_create(const int32_t* widths, int32_t nlayers, kd_mlp** out) {
    if (!widths || !out || nlayers < 1 || nlayers > 16) return err(KD_ERR_ARG, "kd_mlp_create: need 1..16 layers");
    for (int i = 0; i <= nlayers; ++i)
        if (widths[i] < 1 || widths[i] > 4096) return err(KD_ERR_ARG, "kd_mlp_create: widths must be in [1, 4096]");
    *out = nullptr;
    kd_mlp* n = new kd_mlp();
    if (cudaGetDevice(&n->device) != cudaSuccess) { delete n; return err(KD_ERR_CUDA, "kd_mlp_create: no CUDA device"); }
    n->L = nlayers;
    n->w.assign(widths, widths + nlayers + 1);
    size_t off = 0;
    for (int l = 0; l < nlayers; ++l) {
        n->woff.push_back(off);
        off += (size_t)n->w[l + 1] * n->w[l];
        n->boff.push_back(off);
        off += n->w[l + 1];
    }
    n->nparam = off;
    auto bail = [&](int rc) { kd_mlp_destroy(n); return rc; };
    if (allow_smem(KD_MLP_FP32) != cudaSuccess) return bail(err(KD_ERR_CUDA, "kd_mlp_create: shared-memory limit refused"));
    if (cudaMalloc(&n->param, off * sizeof(float)) != cudaSuccess || cudaMalloc(&n->grad, off * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&n->m1, off * sizeof(float)) != cudaSuccess || cudaMalloc(&n->m2, off * sizeof(float)) != cudaSuccess)
        return bail(err(KD_ERR_NOMEM, "kd_mlp_create: allocation failed"));
    if (cudaMalloc(&n->status, sizeof(int)) != cudaSuccess || cudaMemset(n->status, 0, sizeof(int)) != cudaSuccess)
        return bail(err(KD_ERR_NOMEM, "kd_mlp_create: allocation failed"));
    if (cudaMemset(n->param, 0, off * sizeof(float)) != cudaSuccess || cudaMemset(n->m1, 0, off * sizeof(float)) != cudaSuccess ||
        cudaMemset(n->m2, 0, off * sizeof(float)) != cudaSuccess || cudaMemset(n->grad, 0, off * sizeof(float)) != cudaSuccess)
        return bail(err(KD_ERR_CUDA, "kd_mlp_create: memset failed"));
    n->a.assign(nlayers + 1, nullptr);
    n->z.assign(nlayers, nullptr);
    *out = n;
    return KD_OK;
}

void kd_mlp_destroy(kd_mlp* n) {
    if (!n) return;
    cudaSetDevice(n->device);
    cudaDeviceSynchronize();
    for (float* p : n->z) cudaFree(p);
    for (size_t l = 1; l < n->a.size(); ++l) cudaFree(n->a[l]);
    cudaFree(n->dbuf0);
    cudaFree(n->dbuf1);
    cudaFree(n->lossbuf);
    cudaFree(n->part);
    cudaFree(n->status);
    cudaFree(n->param);
    cudaFree(n->grad);
    cudaFree(n->m1);
    cudaFree(n->m2);
    delete n;
}

int kd_mlp_num_params(kd_mlp* n, int64_t* count) {
    if (!n || !count) return err(KD_ERR_ARG, "kd_mlp_num_params: null argument");
    *count = (int64_t)n->nparam;
    return KD_OK;
}

int kd_mlp_set_params(kd_mlp* n, const float* p, int32_t where) {
    if (!n || !p) return err(KD_ERR_ARG, "kd_mlp_set_params: null argument");
    MLP_CUDA(cudaSetDevice(n->device));
    int rc = copy_io(n->param, p, n->nparam * sizeof(float), KD_DEVICE, where, 0);
    if (rc) return rc;
    MLP_CUDA(cudaMemset(n->m1, 0, n->nparam * sizeof(float)));
    MLP_CUDA(cudaMemset(n->m2, 0, n->nparam * sizeof(float)));
    n->adam_t = 0;
    MLP_CUDA(cudaDeviceSynchronize());
    return KD_OK;
}

int kd_mlp_get_params(kd_mlp* n, float* p, int32_t where) {
    if (!n || !p) return err(KD_ERR_ARG, "kd_mlp_get_params: null argument");
    MLP_CUDA(cudaSetDevice(n->device));
    int rc = copy_io(p, n->param, n->nparam * sizeof(float), where, KD_DEVICE, 0);
    if (rc) return rc;
    MLP_CUDA(cudaDeviceSynchronize());
    return check_status(n);
}

int kd_mlp_set_precision(kd_mlp* n, int32_t precision) {
    if (!n || (precision != KD_MLP_FP32 && precision != KD_MLP_BF16))
        return err(KD_ERR_ARG, "kd_mlp_set_precision: KD_MLP_FP32 or KD_MLP_BF16");
    if (precision != n->prec) {
        MLP_CUDA(cudaSetDevice(n->device));
        MLP_CUDA(allow_smem(precision));
        const int rc = n->cap > 0 ? ensure_part(n, precision, n->cap) : KD_OK;
        if (rc) {   // the buffer for the present precision may be gone: made again with the others
            n->cap = 0;
            return rc;
        }
    }
    n->prec = precision;
    return KD_OK;
}

int kd_mlp_forward(kd_mlp* n, const float* x, int32_t batch, float* y, int32_t where, void* cuda_stream) {
    if (!n || !x || !y || batch <= 0) return err(KD_ERR_ARG, "kd_mlp_forward: bad argument");
    MLP_CUDA(cudaSetDevice(n->device));
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int rc = ensure_cap(n, batch);
    if (rc) return rc;
    const float* xd = x;
    if (where == KD_HOST) {
        rc = copy_io(n->dbuf1, x, sizeof(float) * (size_t)batch * n->w[0], KD_DEVICE, KD_HOST, s);
        if (rc) return rc;
        xd = n->dbuf1;
    }
    rc = forward(n, Batch{xd, nullptr, nullptr, 0, batch}, s);
    if (rc) return rc;
    rc = copy_io(y, n->a[n->L], sizeof(float) * (size_t)batch * n->w[n->L], where, KD_DEVICE, s);
    if (rc) return rc;
    if (where == KD_HOST) {
        MLP_CUDA(cudaStreamSynchronize(s));
        return check_status(n);
    }
    return KD_OK;
}

int kd_mlp_gradients(kd_mlp* n, const float* x, const float* t, int32_t batch, float* loss,
                     float* grads, int32_t where, void* cuda_stream) {
    if (!n || !x || !t || batch <= 0) return err(KD_ERR_ARG, "kd_mlp_gradients: bad argument");
    MLP_CUDA(cudaSetDevice(n->device));
    cudaStream_t s = (cudaStream_t)cuda_stream;
    int rc = ensure_cap(n, batch);
    if (rc) return rc;
    const float* xd = x;
    const float* td = t;
    float* tmp_x = nullptr;
    float* tmp_t = nullptr;
    if (where == KD_HOST) {  // staged through the gradient buffers' tail: copy to device scratch
        MLP_CUDA(cudaMalloc(&tmp_x, sizeof(float) * (size_t)batch * n->w[0]));
        MLP_CUDA(cudaMalloc(&tmp_t, sizeof(float) * (size_t)batch * n->w[n->L]));
        rc = copy_io(tmp_x, x, sizeof(float) * (size_t)batch * n->w[0], KD_DEVICE, KD_HOST, s);
        if (!rc) rc = copy_io(tmp_t, t, sizeof(float) * (size_t)batch * n->w[n->L], KD_DEVICE, KD_HOST, s);
        if (rc) { cudaFree(tmp_x); cudaFree(tmp_t); return rc; }
        xd = tmp_x;
        td = tmp_t;
    }
    const Batch in{xd, td, nullptr, 0, batch};
    GradParts gp;
    rc = forward(n, in, s);
    if (!rc) rc = backward(n, in, &gp, nullptr, s);
    if (!rc && grads) rc = gather_grads(n, gp, s);
    if (!rc && loss) rc = copy_io(loss, n->lossbuf, sizeof(float), where, KD_DEVICE, s);
    if (!rc && grads) rc = copy_io(grads, n->grad, n->nparam * sizeof(float), where, KD_DEVICE, s);
    if (where == KD_HOST) {
        cudaStreamSynchronize(s);
        if (!rc) rc = check_status(n);
    }
    cudaFree(tmp_x);
    cudaFree(tmp_t);
    return rc;
}

int kd_mlp_train_step_gather(kd_mlp* n, const float* x_all, const float* t_all, int64_t n_all,
                             const int32_t* idx, int32_t batch, float lr, float* loss_dev, void* cuda_stream) {
    if (!n || !x_all || !t_all || !idx || n_all <= 0 || batch <= 0 || !(lr > 0))
        return err(KD_ERR_ARG, "kd_mlp_train_step_gather: bad argument");
    return train_step(n, Batch{x_all, t_all, idx, (long)n_all, batch}, lr, loss_dev, (cudaStream_t)cuda_stream);
}

int kd_mlp_train_step(kd_mlp* n, const float* x, const float* t, int32_t batch, float lr,
                      float* loss_dev, void* cuda_stream) {
    if (!n || !x || !t || batch <= 0 || !(lr > 0)) return err(KD_ERR_ARG, "kd_mlp_train_step: bad argument");
    return train_step(n, Batch{x, t, nullptr, 0, batch}, lr, loss_dev, (cudaStream_t)cuda_stream);
}

}  // extern "C"
