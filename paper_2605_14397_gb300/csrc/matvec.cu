// H-matrix product y = E x on the device (the product of Sec. 3.1 on the stored
// H-matrix).
//
//   gather   xc = x[perm]                          cluster order, RHS interleaved
//   phase 1  P = V_t^T xc_t                        every V column (one per rank per leaf)
//   reduce   tb_b = sum of the partials of block b over the leaves of its column cluster
//   phase 2  y_s = [D_s | U_s] z_s, z = xc (near columns) or tb (U columns), written to
//            y[perm] (the solvers keep cluster order)
//
// Phases 1 and 2 are persistent kernels, one CTA per SM.  Their coefficient streams are
// cut into chunks of whole columns of one tile or factor slice (at most 32 KB and 128
// columns) and the chunk list is split into equal byte ranges, one per CTA ("stream-K"):
// every SM streams the same number of bytes.  One producer thread moves each chunk --
// its coefficients and, in phase 2, the contiguous range of operands it multiplies --
// with two cp.async.bulk (TMA) copies into a shared-memory ring of four stages (six in
// k_phase1_mr and some tile shapes) guarded by mbarriers; 8 to 16 consumer warps each take
// columns of the chunk, lanes over rows, and touch no global memory except at leaf
// boundaries.  A row leaf whose columns fall into several CTAs is finished by the last of
// them (atomic arrival count, partials summed in CTA order), so the result is deterministic.
//
// Arithmetic modes over the same FP32/BF16 coefficient streams:
//   F32: float vectors, FP32 accumulation;
//   F64: double vectors; each coefficient a multiplies z = zh + zl (zh = fl32(z),
//        zl = fl32(z - zh)) in the compensated dot product of Ogita, Rump and Oishi
//        (2005): TwoProduct via fmaf, TwoSum of the running sum, rounding errors summed
//        apart, the two parts combined in FP64 -- the stored operator applied to FP64
//        vectors to about 1e-13 relative while the coefficients stream at 4 (or 2) bytes.
#include <algorithm>
#include <type_traits>

#include "hmat_impl.h"
#include "pipeline.cuh"

namespace hm {

namespace {

constexpr int STAGES = 4;
constexpr int STAGE_BYTES = 32768;   // coefficients of one chunk
constexpr int MAX_CHUNK_COLS = 128;
constexpr int BAR_BYTES = 128;
// zeroed bytes after phase 1's ring: a single-RHS column read of up to 32 * 12 rows of
// 4 bytes that starts in the last stage ends inside them
constexpr int P1_TAIL = 2048;
constexpr int MAX_RPL = 12;          // 32-row blocks of the largest leaves (384 rows)
constexpr int VEC_SLACK = 32;        // elements after xc / tb so rounded-up copies stay inside

struct FF {
    float hi, lo;
};
// two FF accumulators side by side, for the packed FP32 instructions
struct FF2 {
    float2 hi, lo;
};
// Right-hand sides of one F64 pass.  A coefficient costs 11 FP32 operations per F64
// right-hand side, so from four on the pass is bound by the FP32 pipe and streaming the
// coefficients again for the next four costs less than the registers of a wider pass:
// six RHS of a 12,892-element fault (615 MB of coefficients) took 2.82 ms in one pass of a
// 16-wide kernel that spilled, 0.55 ms in two passes of three (f64_passes).
constexpr int F64_PASS = 4;

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

template <int MODE>
struct AccT;
// type: accumulator; vec: output vectors (y, partials); zin: the x / t operands as the
// kernels read them -- in F64 mode each double is stored pre-split into (hi, lo) floats
// by the gather and the reduction, so the streaming kernels do no FP64 arithmetic
template <>
struct AccT<0> {
    using type = float;
    using vec = float;
    using zin = float;
};
template <>
struct AccT<1> {
    using type = FF;
    using vec = double;
    using zin = float2;
};

// z operand of the F32 mode
struct Z32 {
    float h;
};

__device__ __forceinline__ Z32 make_z(float v) { return Z32{v}; }
__device__ __forceinline__ float2 split_d(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}

__device__ __forceinline__ void acc_zero(float& a) { a = 0.f; }
__device__ __forceinline__ void acc_zero(FF& a) { a.hi = a.lo = 0.f; }
__device__ __forceinline__ void acc_zero(FF2& a) { a.hi = a.lo = make_float2(0.f, 0.f); }

__device__ __forceinline__ void acc_fma(float& acc, float a, Z32 z) { acc = fmaf(a, z.h, acc); }
// two FP32 accumulators against one coefficient: one packed FMA (sm_100-class FFMA2,
// each half rounded like fmaf), half the instructions of the multi-RHS loops
__device__ __forceinline__ void acc_fma2(float& a0, float& a1, float v, Z32 z0, Z32 z1) {
    const float2 r = __ffma2_rn(make_float2(v, v), make_float2(z0.h, z1.h), make_float2(a0, a1));
    a0 = r.x;
    a1 = r.y;
}
// the operands of one column for NR right-hand sides (a multiple of 4) as pairs (p: the
// column's interleaved values in shared memory, 16-byte aligned)
template <int NR>
__device__ __forceinline__ void load_z2(float2 (&z)[NR / 2], const float* p) {
#pragma unroll
    for (int q = 0; q < NR / 4; ++q) {
        const float4 f = reinterpret_cast<const float4*>(p)[q];
        z[2 * q] = make_float2(f.x, f.y);
        z[2 * q + 1] = make_float2(f.z, f.w);
    }
}
// one step of the compensated dot product: acc += a (zh + zl)
__device__ __forceinline__ void ff_fma(float& hi, float& lo, float a, float zh, float zl) {
    const float p = a * zh;
    const float pe = fmaf(a, zh, -p);
    float s, e;
    two_sum(hi, p, s, e);
    hi = s;
    lo += fmaf(a, zl, e + pe);
}
// Two such steps with the packed FP32 instructions of sm_100 (every half rounded like the
// scalar operation), half the instructions to issue.
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ void ff_fma2(FF2& acc, float2 a, float2 zh, float2 zl) {
    const float2 p = __fmul2_rn(a, zh);
    const float2 pe = __ffma2_rn(a, zh, neg2(p));
    const float2 s = __fadd2_rn(acc.hi, p);
    const float2 bb = sub2(s, acc.hi);
    const float2 e = __fadd2_rn(sub2(acc.hi, sub2(s, bb)), sub2(p, bb));
    acc.hi = s;
    acc.lo = __fadd2_rn(acc.lo, __ffma2_rn(a, zl, __fadd2_rn(e, pe)));
}

__device__ __forceinline__ void acc_add(float& a, float b) { a += b; }
__device__ __forceinline__ void acc_add(FF& a, const FF& b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    a.hi = s;
    a.lo += e + b.lo;
}

__device__ __forceinline__ float acc_shfl(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ FF acc_shfl(const FF& v, int o) {
    return FF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// Sum each of the NR accumulators over the warp, spread over the lanes: halving
// exchanges (each lane sends the half of its values it does not keep, NR - 1 shuffles in
// all) and then plain butterflies over the remaining lane bits.  Afterwards acc[0] of lane
// l holds the warp sum of right-hand side k(l) (returned); lanes with the low log2(32/NR)
// bits clear are the first holder of each k.
template <int NR, class Acc>
__device__ __forceinline__ int warp_reduce_scatter(Acc (&acc)[NR], int lane) {
    int k = 0;
#pragma unroll
    for (int h = NR / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const Acc lo = acc[j], hi = acc[j + h];
            Acc mine = up ? hi : lo;
            acc_add(mine, acc_shfl(up ? lo : hi, o));
            acc[j] = mine;
        }
        if (up) k += h;
    }
#pragma unroll
    for (int o = 16 / NR; o > 0; o >>= 1) acc_add(acc[0], acc_shfl(acc[0], o));
    return k;
}

__device__ __forceinline__ float acc_value(float a) { return a; }
__device__ __forceinline__ double acc_value(const FF& a) { return (double)a.hi + (double)a.lo; }

// the (hi, lo) operands of one column for NR right-hand sides in F64 mode (16-byte aligned
// for an even NR)
template <int NR>
__device__ __forceinline__ void load_z(float2 (&z)[NR], const float2* p) {
    if constexpr (NR % 2 == 0) {
#pragma unroll
        for (int q = 0; q < NR / 2; ++q) {
            const float4 f = reinterpret_cast<const float4*>(p)[q];
            z[2 * q] = make_float2(f.x, f.y);
            z[2 * q + 1] = make_float2(f.z, f.w);
        }
    } else {
#pragma unroll
        for (int k = 0; k < NR; ++k) z[k] = p[k];
    }
}

__device__ __forceinline__ float coef(const float* p, int i) { return p[i]; }
__device__ __forceinline__ float coef(const uint16_t* p, int i) { return __uint_as_float(((uint32_t)p[i]) << 16); }

// ---- tensor-core helpers (mma.sync m16n8k16 BF16 x BF16 -> FP32, ldmatrix fragments)
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// round to nearest even BF16 bits
__device__ __forceinline__ uint32_t bf16_bits(float v) {
    const uint32_t u = __float_as_uint(v);
    return (u + 0x7fffu + ((u >> 16) & 1u)) >> 16;
}
__device__ __forceinline__ float bf16_value(uint32_t b) { return __uint_as_float(b << 16); }

// Programmatic dependent launch: the kernels of a product after the gather are launched
// so that they may start while their predecessor drains; each waits for it (and its
// memory) with griddepcontrol.wait before touching what it produced, and lets its own
// successor launch early with griddepcontrol.launch_dependents.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// xc[dof * np + k] = x[k * ndof + user dof], zero for k >= nrhs (np: the padded count)
__global__ void k_gather(const float* __restrict__ x, float* __restrict__ xc, const int32_t* __restrict__ perm,
                         int64_t N, int nrhs, int np) {
    pdl_trigger();
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t ndof = 3 * N;
    if (q >= ndof * np) return;
    const int64_t r = q / np, k = q % np;
    const int64_t p = r / 3, m = r % 3;
    xc[q] = k < nrhs ? x[k * ndof + 3 * (int64_t)perm[p] + m] : 0.f;
}

// The same padding for operands already in cluster order, interleaved by nr.  (The solver's
// kernels before a product let nothing start early: a phase that finds every right-hand side
// converged returns without waiting for them, and what follows is ordered after the phases
// only.  A wait on that path cost the single-RHS F64 phases 1.5 %.)
__global__ void k_pad(const float* __restrict__ xc, float* __restrict__ xp, int64_t ndof, int nr, int np) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= ndof * np) return;
    const int64_t r = q / np, k = q % np;
    xp[q] = k < nr ? xc[r * nr + k] : 0.f;
}

// F64 gather: xc[pass * xc_pass + dof * width + k] = (hi, lo) split of x[(pass * width + k) * ndof +
// user dof], zero beyond nrhs; perm NULL: x is in cluster order already (a solver's: as k_pad)
__global__ void k_gather_split(const double* __restrict__ x, float2* __restrict__ xc,
                               const int32_t* __restrict__ perm, int64_t N, int nrhs, int width, int64_t xc_pass) {
    if (perm) pdl_trigger();
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t ndof = 3 * N;
    if (q >= ndof * width) return;
    const int64_t r = q / width, k = blockIdx.y * (int64_t)width + q % width;
    const int64_t p = r / 3, m = r % 3;
    xc[blockIdx.y * xc_pass + q] =
        k < nrhs ? split_d(x[k * ndof + 3 * (perm ? (int64_t)perm[p] : p) + m]) : make_float2(0.f, 0.f);
}

__device__ __forceinline__ float to_zin(float v, float*) { return v; }
__device__ __forceinline__ float2 to_zin(double v, float2*) { return split_d(v); }
// BF16 high part in the low 16 bits, BF16 of the remainder in the high 16 bits: the B
// operand of the single-RHS tensor-core phase 2
__device__ __forceinline__ uint32_t to_zin(float v, uint32_t*) {
    const uint32_t hb = bf16_bits(v);
    return hb | (bf16_bits(v - bf16_value(hb)) << 16);
}

// tb[(tb_off + l) nr + k] = sum_q P[(poff[pbase + q] + l) nr + k], one CTA (128 threads)
// (VEC4: FP32 with nr a multiple of 4, each slice read as float4)
// per block (and F64 pass): the n = r nr entries times G = 128 / n interleaved groups of leaf partials,
// four independent loads in flight per thread, groups combined in a fixed order.  In F64
// mode the sums are stored as (hi, lo) float pairs, the form phase 2 reads.
template <class V, class Zt, bool VEC4>
__global__ void __launch_bounds__(128) k_reduce_tb(const FarDesc* __restrict__ far, const int32_t* __restrict__ poff,
                                                   const int32_t* __restrict__ uoff, const V* __restrict__ P,
                                                   Zt* __restrict__ tb, int nrhs, int64_t p_pass, int64_t tb_pass,
                                                   const int* __restrict__ skip) {
    __shared__ V sp[128];
    const int64_t p0 = VEC4 ? 0 : blockIdx.y * p_pass, t0 = VEC4 ? 0 : blockIdx.y * tb_pass;
    pdl_wait();
    pdl_trigger();
    if (skip && *(volatile const int*)skip) return;
    const FarDesc F = far[blockIdx.x];
    const int n = F.rank * nrhs;
    if (n == 0) return;
    // first partial of the block in each leaf of T, staged in shared memory when it fits so
    // that the partial loads do not wait on their index loads
    constexpr int SPO = 2048;
    __shared__ int32_t spo[SPO];
    const int32_t* po = poff + F.pbase;
    if (F.n_tleaves <= SPO) {
        for (int q = threadIdx.x; q < F.n_tleaves; q += 128) spo[q] = po[q];
        __syncthreads();
        po = spo;
    }
    auto at = [&](int q) -> int64_t { return p0 + (int64_t)po[q] * nrhs; };
    if constexpr (VEC4) {
        {
            // several RHS: each slice is rank * nrhs contiguous floats, read as float4
            const int n4 = n >> 2;
            const float4* P4 = reinterpret_cast<const float4*>(P);
            for (int e = threadIdx.x; e < n4; e += 128) {
                float4 s0 = make_float4(0.f, 0.f, 0.f, 0.f), s1 = s0, s2 = s0, s3 = s0;
                int q = 0;
                for (; q + 3 < F.n_tleaves; q += 4) {
                    const float4 v0 = P4[(at(q) >> 2) + e], v1 = P4[(at(q + 1) >> 2) + e];
                    const float4 v2 = P4[(at(q + 2) >> 2) + e], v3 = P4[(at(q + 3) >> 2) + e];
                    s0.x += v0.x; s0.y += v0.y; s0.z += v0.z; s0.w += v0.w;
                    s1.x += v1.x; s1.y += v1.y; s1.z += v1.z; s1.w += v1.w;
                    s2.x += v2.x; s2.y += v2.y; s2.z += v2.z; s2.w += v2.w;
                    s3.x += v3.x; s3.y += v3.y; s3.z += v3.z; s3.w += v3.w;
                }
                for (; q < F.n_tleaves; ++q) {
                    const float4 v0 = P4[(at(q) >> 2) + e];
                    s0.x += v0.x; s0.y += v0.y; s0.z += v0.z; s0.w += v0.w;
                }
                const float4 t = make_float4((s0.x + s1.x) + (s2.x + s3.x), (s0.y + s1.y) + (s2.y + s3.y),
                                             (s0.z + s1.z) + (s2.z + s3.z), (s0.w + s1.w) + (s2.w + s3.w));
                for (int c = 0; c < F.n_sleaves; ++c) {  // one copy per leaf of S
                    float* o = reinterpret_cast<float*>(tb) + (int64_t)uoff[F.ubase + c] * nrhs + 4 * e;
                    o[0] = t.x;
                    o[1] = t.y;
                    o[2] = t.z;
                    o[3] = t.w;
                }
            }
            return;
        }
    }
    if (n >= 128) {
        for (int e = threadIdx.x; e < n; e += 128) {
            V s0 = 0, s1 = 0, s2 = 0, s3 = 0;
            int q = 0;
            for (; q + 3 < F.n_tleaves; q += 4) {
                s0 += P[at(q) + e];
                s1 += P[at(q + 1) + e];
                s2 += P[at(q + 2) + e];
                s3 += P[at(q + 3) + e];
            }
            for (; q < F.n_tleaves; ++q) s0 += P[at(q) + e];
            const Zt t = to_zin((s0 + s1) + (s2 + s3), tb);
            for (int c = 0; c < F.n_sleaves; ++c) tb[t0 + (int64_t)uoff[F.ubase + c] * nrhs + e] = t;
        }
        return;
    }
    const int G = 128 / n;
    const int e = threadIdx.x % n, g = threadIdx.x / n;
    V s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    if (g < G) {
        int q = g;
        for (; q + 3 * G < F.n_tleaves; q += 4 * G) {
            s0 += P[at(q) + e];
            s1 += P[at(q + G) + e];
            s2 += P[at(q + 2 * G) + e];
            s3 += P[at(q + 3 * G) + e];
        }
        for (; q < F.n_tleaves; q += G) s0 += P[at(q) + e];
    }
    sp[threadIdx.x] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (threadIdx.x < n) {
        V s = 0;
        for (int q = 0; q < G; ++q) s += sp[q * n + threadIdx.x];
        const Zt t = to_zin(s, tb);
        for (int c = 0; c < F.n_sleaves; ++c) tb[t0 + (int64_t)uoff[F.ubase + c] * nrhs + threadIdx.x] = t;
    }
}

// 16 right-hand sides with BF16 U slices on tensor cores: the sums of t (float4 slices,
// k_reduce_pack16_mix below), each value split into BF16
// hi + lo (hi = bf16(t), lo = bf16(t - hi)) and stored as the B operand of phase 2:
// 64 bytes per rank entry l, four 16-byte pieces (RHS 0-7 hi, RHS 0-7 lo, RHS 8-15 hi,
// RHS 8-15 lo), piece q stored at position q ^ ((l >> 1) & 3), so that the eight
// consecutive entries one ldmatrix row group reads fall into eight different bank groups.
__device__ __forceinline__ int tb16_piece_pos(int64_t l, int q) { return q ^ (int)((l >> 1) & 3); }

// The same reduction for one RHS in one launch of 256-thread CTAs over a block order
// (red_order) that lists the blocks with more than RED_WARP_LEAVES leaves of T first.
// Each of those gets a CTA: its offset table staged in shared memory, 256 / r groups of
// threads over the leaves, four partials per thread in flight.  The many small blocks get
// a warp each, eight per CTA -- four times the blocks in flight of a CTA per block, whose
// launch was bound by the latency of short load chains rather than by bytes: lanes take
// the rank entries, one load fetches 32 offset-table entries which shuffles broadcast.
// Every block sums its partials in a fixed order.
constexpr int RED_WARP_LEAVES = 32;
template <class V, class Zt>
__global__ void __launch_bounds__(256) k_reduce_mix(const FarDesc* __restrict__ far,
                                                    const int32_t* __restrict__ poff,
                                                    const int32_t* __restrict__ uoff,
                                                    const int32_t* __restrict__ order, int64_t n_big, int64_t n_all,
                                                    const V* __restrict__ P, Zt* __restrict__ tb,
                                                    const int* __restrict__ skip) {
    __shared__ V sp[256];
    constexpr int SPO = 2048;
    __shared__ int32_t spo[SPO];
    pdl_wait();
    pdl_trigger();
    if (skip && *(volatile const int*)skip) return;
    if ((int64_t)blockIdx.x < n_big) {
        const FarDesc F = far[order[blockIdx.x]];
        const int r = F.rank, nt = F.n_tleaves;  // r <= 256 (rank cap)
        const int32_t* po = poff + F.pbase;
        if (nt <= SPO) {
            for (int q = threadIdx.x; q < nt; q += 256) spo[q] = po[q];
            __syncthreads();
            po = spo;
        }
        const int G = 256 / r;
        const int e = threadIdx.x % r, g = threadIdx.x / r;
        V s0 = 0, s1 = 0, s2 = 0, s3 = 0;
        if (g < G) {
            int q = g;
            for (; q + 3 * G < nt; q += 4 * G) {
                s0 += P[(int64_t)po[q] + e];
                s1 += P[(int64_t)po[q + G] + e];
                s2 += P[(int64_t)po[q + 2 * G] + e];
                s3 += P[(int64_t)po[q + 3 * G] + e];
            }
            for (; q < nt; q += G) s0 += P[(int64_t)po[q] + e];
        }
        sp[threadIdx.x] = (s0 + s1) + (s2 + s3);
        __syncthreads();
        if (threadIdx.x < r) {
            V s = 0;
            for (int q = 0; q < G; ++q) s += sp[q * r + threadIdx.x];
            const Zt t = to_zin(s, tb);
            for (int c = 0; c < F.n_sleaves; ++c) tb[uoff[F.ubase + c] + threadIdx.x] = t;
        }
        return;
    }
    const int64_t k = n_big + ((int64_t)blockIdx.x - n_big) * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= n_all) return;
    const int64_t b = order[k];
    const int r = far[b].rank, nt = far[b].n_tleaves;
    const int32_t* po = poff + far[b].pbase;
    const int ns = far[b].n_sleaves;
    const int32_t* uo = uoff + far[b].ubase;
    for (int e0 = 0; e0 < r; e0 += 32) {
        const int e = e0 + lane;
        const bool on = e < r;
        V s0 = 0, s1 = 0, s2 = 0, s3 = 0;
        for (int q0 = 0; q0 < nt; q0 += 32) {
            const int m = min(32, nt - q0);
            const int32_t mine = lane < m ? po[q0 + lane] : 0;
            int q = 0;
            for (; q + 3 < m; q += 4) {
                const int32_t o0 = __shfl_sync(0xffffffffu, mine, q), o1 = __shfl_sync(0xffffffffu, mine, q + 1);
                const int32_t o2 = __shfl_sync(0xffffffffu, mine, q + 2), o3 = __shfl_sync(0xffffffffu, mine, q + 3);
                if (on) {
                    s0 += P[(int64_t)o0 + e];
                    s1 += P[(int64_t)o1 + e];
                    s2 += P[(int64_t)o2 + e];
                    s3 += P[(int64_t)o3 + e];
                }
            }
            for (; q < m; ++q) {
                const int32_t o0 = __shfl_sync(0xffffffffu, mine, q);
                if (on) s0 += P[(int64_t)o0 + e];
            }
        }
        if (on) {
            const Zt t = to_zin((s0 + s1) + (s2 + s3), tb);
            for (int c = 0; c < ns; ++c) tb[uo[c] + e] = t;  // one copy per leaf of S
        }
    }
}

// 16 RHS packed for TC16 over the same block order as k_reduce_mix: blocks with more
// than RED_WARP_LEAVES leaves of T a 256-thread CTA each (float4 groups x subsets of the
// leaves, partials meeting in shared memory in subset order), the others a warp each,
// eight per CTA (lanes over the float4 groups, 32 offsets per load broadcast by
// shuffles, four partials in flight).  Every block sums in a fixed order.
__device__ __forceinline__ void store_pack16(uint16_t* __restrict__ tb, const int32_t* __restrict__ uo, int ns,
                                             int e, float4 a) {
    const float t[4] = {a.x, a.y, a.z, a.w};
    uint32_t hb[4], lb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        hb[i] = bf16_bits(t[i]);
        lb[i] = bf16_bits(t[i] - bf16_value(hb[i]));
    }
    const int k0 = (e & 3) * 4;                  // first of the four RHS
    const int qh = 2 * (k0 >> 3), off = k0 & 7;  // hi piece of these RHS, offset inside it
    for (int c = 0; c < ns; ++c) {               // one copy per leaf of S
        const int64_t l = (int64_t)uo[c] + e / 4;
        uint16_t* row = tb + 32 * l;             // 64 bytes
        *reinterpret_cast<uint2*>(row + 8 * tb16_piece_pos(l, qh) + off) =
            make_uint2(hb[0] | (hb[1] << 16), hb[2] | (hb[3] << 16));
        *reinterpret_cast<uint2*>(row + 8 * tb16_piece_pos(l, qh + 1) + off) =
            make_uint2(lb[0] | (lb[1] << 16), lb[2] | (lb[3] << 16));
    }
}

__device__ __forceinline__ void add4(float4& s, const float4 v) {
    s.x += v.x;
    s.y += v.y;
    s.z += v.z;
    s.w += v.w;
}

__global__ void __launch_bounds__(256) k_reduce_pack16_mix(const FarDesc* __restrict__ far,
                                                           const int32_t* __restrict__ poff,
                                                           const int32_t* __restrict__ uoff,
                                                           const int32_t* __restrict__ order, int64_t n_big,
                                                           int64_t n_all, const float* __restrict__ P,
                                                           uint16_t* __restrict__ tb, const int* __restrict__ skip) {
    __shared__ float4 sp[256];
    constexpr int SPO = 2048;
    __shared__ int32_t spo[SPO];
    pdl_wait();
    pdl_trigger();
    if (skip && *(volatile const int*)skip) return;
    const float4* P4 = reinterpret_cast<const float4*>(P);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if ((int64_t)blockIdx.x < n_big) {
        const FarDesc F = far[order[blockIdx.x]];
        const int n4 = 4 * F.rank, nt = F.n_tleaves;
        const int32_t* po = poff + F.pbase;
        if (nt <= SPO) {
            for (int q = threadIdx.x; q < nt; q += 256) spo[q] = po[q];
            __syncthreads();
            po = spo;
        }
        for (int e0 = 0; e0 < n4; e0 += 256) {
            const int r = min(256, n4 - e0);
            const int G = 256 / r;
            const int e = e0 + threadIdx.x % r, g = threadIdx.x / r;
            float4 s0 = z4, s1 = z4, s2 = z4, s3 = z4;
            if (g < G) {
                int q = g;
                for (; q + 3 * G < nt; q += 4 * G) {
                    add4(s0, P4[(int64_t)po[q] * 4 + e]);
                    add4(s1, P4[(int64_t)po[q + G] * 4 + e]);
                    add4(s2, P4[(int64_t)po[q + 2 * G] * 4 + e]);
                    add4(s3, P4[(int64_t)po[q + 3 * G] * 4 + e]);
                }
                for (; q < nt; q += G) add4(s0, P4[(int64_t)po[q] * 4 + e]);
            }
            add4(s0, s1);
            add4(s2, s3);
            add4(s0, s2);
            sp[threadIdx.x] = s0;
            __syncthreads();
            if (threadIdx.x < r) {
                float4 a = sp[threadIdx.x];
                for (int q = 1; q < G; ++q) add4(a, sp[q * r + threadIdx.x]);
                store_pack16(tb, uoff + F.ubase, F.n_sleaves, e0 + threadIdx.x, a);
            }
            __syncthreads();
        }
        return;
    }
    const int64_t k = n_big + ((int64_t)blockIdx.x - n_big) * 8 + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (k >= n_all) return;
    const int64_t b = order[k];
    const int n4 = 4 * far[b].rank, nt = far[b].n_tleaves;
    const int32_t* po = poff + far[b].pbase;
    // up to RP passes of 32 groups at once: their loads for one leaf are independent
    constexpr int RP = 4;
    for (int e0 = 0; e0 < n4; e0 += 32 * RP) {
        float4 acc[2][RP];  // even and odd leaves: two more loads in flight
#pragma unroll
        for (int p = 0; p < RP; ++p) acc[0][p] = acc[1][p] = z4;
        for (int q0 = 0; q0 < nt; q0 += 32) {
            const int m = min(32, nt - q0);
            const int32_t mine = lane < m ? po[q0 + lane] : 0;
            int q = 0;
            for (; q + 1 < m; q += 2) {
                const int64_t o0 = (int64_t)__shfl_sync(0xffffffffu, mine, q) * 4;
                const int64_t o1 = (int64_t)__shfl_sync(0xffffffffu, mine, q + 1) * 4;
#pragma unroll
                for (int p = 0; p < RP; ++p) {
                    const int e = e0 + 32 * p + lane;
                    if (e < n4) {
                        add4(acc[0][p], P4[o0 + e]);
                        add4(acc[1][p], P4[o1 + e]);
                    }
                }
            }
            if (q < m) {
                const int64_t o0 = (int64_t)__shfl_sync(0xffffffffu, mine, q) * 4;
#pragma unroll
                for (int p = 0; p < RP; ++p) {
                    const int e = e0 + 32 * p + lane;
                    if (e < n4) add4(acc[0][p], P4[o0 + e]);
                }
            }
        }
#pragma unroll
        for (int p = 0; p < RP; ++p) {
            const int e = e0 + 32 * p + lane;
            add4(acc[0][p], acc[1][p]);
            if (e < n4) store_pack16(tb, uoff + far[b].ubase, far[b].n_sleaves, e, acc[0][p]);
        }
    }
}

struct StreamArgs {
    const Chunk* chunks;
    const int32_t* cta_begin;
    const LeafDesc* leaves;
    const LeafSplit* split;
    const float* near;
    const void* ucoef;
    const void* vcoef;
    const void* xc;
    const void* tb;
    void* out;    // yc (phase 2) or P (phase 1)
    void* slots;  // phase-2 partials of split leaves
    int32_t* counters;
    int* err;
    const int32_t* perm;  // phase 2: rows of out in user order (cluster position -> element); NULL: cluster order
    int64_t ndof;
    int nout;     // right-hand sides the caller asked for (the vectors of out); the rest pad the kernel's count
    int ld_max;
    // F64: more right-hand sides than one pass holds run as passes of NR in the same launches
    // (blockIdx.y).  Elements from one pass's xc, P and tb to the next's, and its slots and counters
    int64_t xc_pass, p_pass, tb_pass;
    int slots_pass, counters_pass;
    int wait_x;   // phase 2: xc comes from the kernel just before (no far field, so no kernel in between)
    const int* skip;  // optional device flag: when set, the kernels return at once
    uint64_t wait_ns; // limit of every bounded wait of the copy ring
    // test switch (hm_hmat_set_wait): the producer of phase 2 stops before this chunk of
    // the plan (its copy and every later one of the CTA are never issued), so that the
    // consumers' waits run out; -1: off
    int64_t withhold;
};

template <class V, int NR>
struct ZRange {
    static constexpr int ALIGN = 16 / (int)sizeof(V);  // elements per 16 bytes
    static constexpr int BYTES = ((MAX_CHUNK_COLS * NR + 2 * ALIGN) * (int)sizeof(V) + 127) / 128 * 128;
};

// Columns (or column groups) are dealt to the warps round robin through the chunks of a
// CTA: slot g starts chunk i at column (g - rot) mod G, rot the columns dealt so far.  With
// every chunk dealt from warp 0 the first warps always got the odd columns -- 53 columns
// over 16 warps is 4 for five of them and 3 for the rest, so a fifth of the issue slots of
// the compute-bound variants waited (warps run ahead by the depth of the ring, so the
// chunks need not balance one by one).
template <int G>
__device__ __forceinline__ int deal_start(int g, int rot) {
    return g >= rot ? g - rot : g - rot + G;
}
template <int G>
__device__ __forceinline__ int deal_next(int rot, int n) {
    return (rot + n) % G;
}

// ---- producer: one thread streams this CTA's chunks (and their operands) through the ring
// (WAIT_T: wait for the preceding kernel -- the reduction producing t -- only before the
// first chunk whose operand is t; near tiles read x, complete before that kernel began)
template <class C, class V, int NR, bool WITH_Z, bool WAIT_T = false, int ST = STAGES>
__device__ __forceinline__ void produce(const StreamArgs& a, unsigned char* smem_stage, int stage_stride,
                                        uint64_t* full, uint64_t* empty, int c0, int c1) {
    using ZR = ZRange<V, NR>;
    bool waited = false;
    int issued = c1 - c0;  // copies issued (all of them unless the test switch stops early)
    Chunk nxt = c0 < c1 ? a.chunks[c0] : Chunk{};
    for (int i = c0; i < c1; ++i) {
        if (WITH_Z && i == a.withhold) {
            issued = i - c0;
            break;
        }
        const Chunk ch = nxt;
        if (i + 1 < c1) nxt = a.chunks[i + 1];
        if constexpr (WAIT_T) {
            if (!waited && ch.kind != 0) {
                pdl_wait();
                waited = true;
            }
        }
        const int q = i - c0, s = q % ST;
        const uint32_t ph = (uint32_t)(q / ST) & 1u;
        if (q >= ST) mbar_wait(empty + s, ph ^ 1u, a.err, 4, a.wait_ns);
        unsigned char* stg = smem_stage + (size_t)s * stage_stride;
        const void* src;
        uint32_t bytes;
        if (ch.kind == 0) {
            src = a.near + ch.src;
            bytes = (uint32_t)ch.ncols * ch.ld * 4u;
        } else {
            const C* base = (const C*)(ch.kind == 1 ? a.ucoef : a.vcoef);
            src = base + ch.src;
            bytes = (uint32_t)ch.ncols * ch.ld * (uint32_t)sizeof(C);
        }
        if constexpr (WITH_Z) {
            const V* zsrc = (const V*)(ch.kind == 0 ? a.xc : a.tb);
            const int64_t z0 = ch.zoff * NR;
            const int64_t a0 = z0 & ~(int64_t)(ZR::ALIGN - 1);
            const int64_t a1 = (z0 + (int64_t)ch.ncols * NR + ZR::ALIGN - 1) & ~(int64_t)(ZR::ALIGN - 1);
            const uint32_t zbytes = (uint32_t)((a1 - a0) * (int64_t)sizeof(V));
            mbar_arrive_expect_tx(full + s, bytes + zbytes);
            bulk_g2s(stg, zsrc + a0, zbytes, full + s);
            bulk_g2s(stg + ZR::BYTES, src, bytes, full + s);
        } else {
            mbar_arrive_expect_tx(full + s, bytes);
            bulk_g2s(stg, src, bytes, full + s);
        }
    }
    if constexpr (WAIT_T) {
        if (!waited) pdl_wait();
    }
    // no copy may still be in flight when the CTA exits
    const int n = issued;
    for (int q = std::max(0, n - ST); q < n; ++q)
        mbar_wait(full + (q % ST), (uint32_t)(q / ST) & 1u, a.err, 8, a.wait_ns);
}

template <int ST = STAGES>
__device__ __forceinline__ void init_ring(uint64_t* full, uint64_t* empty, int ncw) {
    if (threadIdx.x == 0) {
        for (int s = 0; s < ST; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, ncw);
        }
        mbar_fence_init();
    }
    __syncthreads();
}

// The F64 mode's columns of phase 2: c0, c0 + step, ... of a chunk against the NA row
// blocks of 32 rows this warp holds (col0: the warp's first row of column 0).  NA is a
// template argument so that the row blocks past a short leaf cost nothing (151-row leaves
// of a 25,700-triangle mesh: 5 blocks instead of 6).  Scalar operations: packing row
// blocks in pairs needs a register move for most operands, and took 208 us on those
// triangles (1.12 GB, 166 us at the copy bandwidth) where this loop takes 197 us and the
// former one, with address arithmetic per column and 192 rows, 225 us.
template <int NA, int NR, int RPW, class E>
__device__ __forceinline__ void ff_columns(FF (&t)[NR][RPW], const E* col0, int ld, const float2* zb, int c0,
                                           int ncols, int step) {
    const E* col = col0 + (size_t)c0 * ld;
    const float2* zc = zb + (size_t)c0 * NR;
    const int cs = step * ld, zs = step * NR;
#pragma unroll 2
    for (int c = c0; c < ncols; c += step, col += cs, zc += zs) {
        float v[NA];
#pragma unroll
        for (int i = 0; i < NA; ++i) v[i] = coef(col, 32 * i);
        float2 z[NR];
        load_z<NR>(z, zc);
#pragma unroll
        for (int k = 0; k < NR; ++k)
#pragma unroll
            for (int i = 0; i < NA; ++i) ff_fma(t[k][i].hi, t[k][i].lo, v[i], z[k].x, z[k].y);
    }
}
// the same for a run-time number of row blocks (1 .. 6)
template <int NR, int RPW, class E>
__device__ __forceinline__ void ff_columns_n(FF (&t)[NR][RPW], int nact, const E* col0, int ld, const float2* zb,
                                             int c0, int ncols, int step) {
    static_assert(RPW == 6, "one variant per row block count");
    if (nact == 6)
        ff_columns<6>(t, col0, ld, zb, c0, ncols, step);
    else if (nact == 5)
        ff_columns<5>(t, col0, ld, zb, c0, ncols, step);
    else if (nact >= 3)
        ff_columns<4>(t, col0, ld, zb, c0, ncols, step);
    else if (nact >= 1)
        ff_columns<2>(t, col0, ld, zb, c0, ncols, step);
}

// Several right-hand sides in F32 mode: columns c0, c0 + step, ... of a chunk against the NA
// row blocks of 32 rows this warp holds, accumulators in RHS pairs for the packed FMA.  The
// row block count is a template argument and the right-hand sides are NR exactly (the host
// pads their number), so a column is its loads and FMAs only (with both tested in the loop a
// column of three blocks and 16 RHS took 62 instructions, 24 of them FMAs).  16 RHS on three
// 100 x 100 planes (1.92 GB, 282 us at the copy bandwidth): 540 us before, 395 now.
template <int NA, int NR, int RPW, class E>
__device__ __forceinline__ void mr_columns(float2 (&t)[RPW][NR / 2], const E* col0, int ld, const float* zb, int c0,
                                           int ncols, int step) {
    const E* col = col0 + (size_t)c0 * ld;
    const float* zc = zb + (size_t)c0 * NR;
    const int cs = step * ld, zs = step * NR;
    for (int c = c0; c < ncols; c += step, col += cs, zc += zs) {
        float v[NA];
#pragma unroll
        for (int i = 0; i < NA; ++i) v[i] = coef(col, 32 * i);
        float2 z[NR / 2];
        load_z2<NR>(z, zc);
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const float2 vv = make_float2(v[i], v[i]);
#pragma unroll
            for (int k = 0; k < NR / 2; ++k) t[i][k] = __ffma2_rn(vv, z[k], t[i][k]);
        }
    }
}
// the same for a run-time row block count (0 .. RPW)
template <int NR, int RPW, class E>
__device__ __forceinline__ void mr_columns_n(float2 (&t)[RPW][NR / 2], int nact, const E* col0, int ld,
                                             const float* zb, int c0, int ncols, int step) {
    static_assert(RPW == 2 || RPW == 3 || RPW == 6, "one variant per row block count");
    if constexpr (RPW <= 3) {
        if (RPW == 3 && nact == 3)
            mr_columns<RPW, NR>(t, col0, ld, zb, c0, ncols, step);
        else if (nact == 2)
            mr_columns<2, NR>(t, col0, ld, zb, c0, ncols, step);
        else if (nact == 1)
            mr_columns<1, NR>(t, col0, ld, zb, c0, ncols, step);
    } else {
        if (nact == 6)
            mr_columns<6, NR>(t, col0, ld, zb, c0, ncols, step);
        else if (nact == 5)
            mr_columns<5, NR>(t, col0, ld, zb, c0, ncols, step);
        else if (nact >= 3)
            mr_columns<4, NR>(t, col0, ld, zb, c0, ncols, step);
        else if (nact >= 1)
            mr_columns<2, NR>(t, col0, ld, zb, c0, ncols, step);
    }
}

// ---- phase 2: y = [D | U] z per row leaf
// RS > 1 splits each column's rows over RS warps (RPL / RS rows per lane each), so that
// many right-hand sides fit in registers with more warps in flight.
//
// BF16 U slices with one RHS (TC2) run on tensor cores: A = the slice (rows x columns,
// column-major in shared memory, so ldmatrix.trans gives the row-major fragments), B
// column 0 = the BF16 high part of t, column 1 the low part (the reduction stores t in
// that packed form), so d(col 0) + d(col 1) = U t for 16 rows.  Warp w = (kg, mg) takes
// the k-tiles kg, kg + 4 of each slice and keeps m-tiles mg, mg + 4, mg + 8 of the leaf
// in registers; at the flush each warp adds them to its own row of the reduction buffer.
template <int MODE, class C, int NR, int RPL, int NCW, int RS, int ST = STAGES, bool TC = true, bool PASSES = false>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) k_phase2(StreamArgs a) {
    static_assert(!PASSES || MODE == 1, "F64 passes");
    constexpr bool TC2 = MODE == 0 && NR == 1 && RS == 1 && NCW == 16 && RPL == 6 &&
                         std::is_same<C, uint16_t>::value;
    // BF16 U slices with 16 RHS (TC16): warp w owns the m-tiles w / 2 and w / 2 + 8 (16 rows
    // of the leaf each) of the n-tile w % 2 (8 RHS); A as
    // in TC2, B = t in the packed BF16 (hi, lo) form of k_reduce_pack16_mix read with
    // ldmatrix.trans, two mma per k-tile in two chains.  The CUDA-core accumulators keep the
    // near tiles; the tensor-core results join them at the flush through ty.
    constexpr bool TC16 = TC && MODE == 0 && NR == 16 && RS == 2 && NCW == 16 && RPL <= 6 &&
                          std::is_same<C, uint16_t>::value;
    constexpr int TC16_MT = 2 * RPL, TY_LD = 196;  // m-tiles of 16 rows; ty row stride (bank spread)
    constexpr int TKG = 4, TMG = 4, TMT = 3;  // k-groups x m-groups = NCW; m-tiles per warp
    static_assert(!TC2 || (TKG * TMG == NCW && TMG * TMT * 16 >= 32 * RPL && TKG * 2 * 16 >= MAX_CHUNK_COLS),
                  "tensor-core phase 2 covers every row and column");
    using Acc = typename AccT<MODE>::type;
    using Vv = typename AccT<MODE>::vec;
    using ZR = ZRange<Vv, NR>;
    constexpr int STRIDE = ZR::BYTES + STAGE_BYTES;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = (uint64_t*)smem;
    uint64_t* empty = full + ST;
    int* s_flag = (int*)(empty + ST);
    uint16_t* zline = (uint16_t*)(smem + 112);  // a zeroed 16-byte line (ldmatrix rows outside a slice)
    static_assert(2 * ST * 8 + 4 <= 112 && 112 + 16 <= BAR_BYTES, "barrier area layout");
    unsigned char* stage = smem + BAR_BYTES;
    constexpr int RPW = RPL / RS;  // rows per lane of one warp
    constexpr int NG = NCW / RS;   // column groups
    static_assert(RPL % RS == 0 && NCW % RS == 0, "row split must divide rows and warps");
    // FP32 vectors with 16 RHS on leaves of up to 64 elements reduce 8 RHS per pass of the
    // flush (4 barriers per leaf instead of 32); the other variants one RHS per pass (their
    // reduction buffer would not fit beside the ring)
    constexpr int KP = (MODE == 0 && NR == 16 && RPL <= 6) ? 8 : 1;
    Acc* red = (Acc*)(stage + (size_t)ST * STRIDE);  // [KP][NG][32 RPL]
    float* ty = (float*)(red + (size_t)KP * NG * 32 * RPL);  // TC16: the leaf's tensor-core sums [16 RHS][TY_LD]

    if (a.skip && *(volatile const int*)a.skip) return;  // every right-hand side already converged
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < 8) zline[threadIdx.x] = 0;
    init_ring<ST>(full, empty, NCW);
    const int c0 = a.cta_begin[blockIdx.x], c1 = a.cta_begin[blockIdx.x + 1];
    pdl_trigger();
    if (w == NCW) {
        // the t operand ranges come from the reduction: the producer waits for it before the
        // first U chunk, so the near tiles ahead of it stream while the reduction runs
        if constexpr (PASSES) {
            a.xc = (const Vv*)a.xc + blockIdx.y * a.xc_pass;
            a.tb = (const Vv*)a.tb + blockIdx.y * a.tb_pass;
        }
        if (lane == 0) {
            if (a.wait_x) pdl_wait();  // (before produce: in its loop the test cost the F64 kernels 0.7 %)
            produce<C, Vv, NR, true, true, ST>(a, stage, STRIDE, full, empty, c0, c1);
        }
        return;
    }
    Vv* yc = (Vv*)a.out;
    Vv* slots = (Vv*)a.slots;
    int nout = a.nout;
    int32_t* counters = a.counters;
    if constexpr (PASSES) {
        nout = min(NR, a.nout - (int)blockIdx.y * NR);
        yc += (int64_t)blockIdx.y * NR * a.ndof;
        slots += (int64_t)blockIdx.y * a.slots_pass * NR * a.ld_max;
        counters += blockIdx.y * a.counters_pass;
    }
    const int g = w / RS, rbase = (w % RS) * 32 * RPW;
    constexpr bool MR = MODE == 0 && NR > 1;  // accumulators in RHS pairs
    Acc acc[MR ? 1 : NR][RPW];
    float2 acc2[MR ? RPW : 1][MR ? NR / 2 : 1];
    float dt[TMT][4];  // TC2: this warp's m-tiles of the leaf (tensor-core part)
    int cur = -1, rot = 0;
    LeafDesc L{};

    // entry r of the leaf in an output vector (matvec's y in user order: the permutation costs
    // the flush a cached load, a kernel of its own over y cost 3 to 6 us a product)
    auto out_at = [&](int k, int r) {
        const int p = L.begin + r / 3;
        return (int64_t)k * a.ndof + 3 * (int64_t)(a.perm ? __ldg(a.perm + p) : p) + r % 3;
    };
    auto flush = [&]() {
        const LeafSplit sp = a.split[cur];
        const int rows = 3 * L.n;
        const bool whole = sp.nparts == 1;
        const int64_t slot = whole ? 0 : (int64_t)(sp.slot_base + (int)blockIdx.x - sp.w_first);
        // KP right-hand sides per reduction pass through red (k unrolled at compile time: a
        // runtime index into acc would move it to local memory)
#pragma unroll
        for (int k0 = 0; k0 < NR; k0 += KP) {
            if (k0 >= nout) break;
#pragma unroll
            for (int kk = 0; kk < KP; ++kk)
#pragma unroll
                for (int i = 0; i < RPW; ++i) {
                    Acc& o = red[((size_t)kk * NG + g) * (32 * RPL) + rbase + lane + 32 * i];
                    if constexpr (MR)
                        o = ((k0 + kk) & 1) ? acc2[i][(k0 + kk) / 2].y : acc2[i][(k0 + kk) / 2].x;
                    else
                        o = acc[k0 + kk][i];
                }
            if constexpr (TC2) {
                // lanes 4 c hold rows 16 mt + c (d0 + d1) and 16 mt + c + 8 (d2 + d3)
                __syncwarp();
                if ((lane & 3) == 0) {
#pragma unroll
                    for (int j = 0; j < TMT; ++j) {
                        Acc* rw = red + (size_t)g * (32 * RPL) + (w % TMG + TMG * j) * 16 + (lane >> 2);
                        rw[0] += dt[j][0] + dt[j][1];
                        rw[8] += dt[j][2] + dt[j][3];
                    }
                }
            }
            consumer_sync(NCW * 32);
            for (int e = threadIdx.x; e < KP * rows; e += NCW * 32) {
                const int kk = e / rows, r = e - kk * rows, k = k0 + kk;
                if (k >= nout) continue;
                const int64_t dst = whole ? out_at(k, r) : (slot * NR + k) * a.ld_max + r;  // (loads before the sum)
                const Acc* rk = red + (size_t)kk * NG * (32 * RPL);
                Acc s = rk[r];
                for (int q = 1; q < NG; ++q) acc_add(s, rk[(size_t)q * (32 * RPL) + r]);
                if constexpr (TC16) acc_add(s, ty[(size_t)k * TY_LD + r]);
                (whole ? yc : slots)[dst] = (Vv)acc_value(s);
            }
            consumer_sync(NCW * 32);
        }
        if (!whole) {
            __threadfence();
            consumer_sync(NCW * 32);
            if (threadIdx.x == 0) {
                const int old = atomicAdd(counters + cur, 1);
                *s_flag = (old == sp.nparts - 1);
            }
            consumer_sync(NCW * 32);
            if (*s_flag) {
                __threadfence();
                // (over all right-hand sides at once: one after the other, 16 of an 84-row leaf
                // were 16 rounds of load latencies for a sixth of the threads)
                for (int e = threadIdx.x; e < nout * rows; e += NCW * 32) {
                    const int k = NR == 1 ? 0 : e / rows, r = e - k * rows;
                    Vv s = 0;
                    for (int p = 0; p < sp.nparts; ++p)
                        s += __ldcg(slots + ((int64_t)(sp.slot_base + p) * NR + k) * a.ld_max + r);
                    yc[out_at(k, r)] = s;
                }
                if (threadIdx.x == 0) counters[cur] = 0;
            }
            consumer_sync(NCW * 32);
        }
    };

    Chunk nxt = c0 < c1 ? a.chunks[c0] : Chunk{};
    for (int i = c0; i < c1; ++i) {
        const Chunk ch = nxt;
        if (i + 1 < c1) nxt = a.chunks[i + 1];
        const int q = i - c0, s = q % ST;
        if (ch.leaf != cur) {
            if (cur >= 0) flush();
            cur = ch.leaf;
            L = a.leaves[cur];
            if constexpr (MR) {
#pragma unroll
                for (int j = 0; j < RPW; ++j)
#pragma unroll
                    for (int k = 0; k < NR / 2; ++k) acc2[j][k] = make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int k = 0; k < NR; ++k)
#pragma unroll
                    for (int j = 0; j < RPW; ++j) acc_zero(acc[k][j]);
            }
#pragma unroll
            for (int j = 0; j < TMT; ++j) dt[j][0] = dt[j][1] = dt[j][2] = dt[j][3] = 0.f;
            if constexpr (TC16) {
                // the entries of ty this lane accumulates (its m-tiles, see below) start at 0
                for (int mt = w >> 1; mt < TC16_MT; mt += 8) {
                    const int r0 = 16 * mt + (lane >> 2);
                    float* col = ty + (size_t)(8 * (w & 1) + 2 * (lane & 3)) * TY_LD;
                    col[r0] = col[TY_LD + r0] = col[r0 + 8] = col[TY_LD + r0 + 8] = 0.f;
                }
            }
        }
        mbar_wait(full + s, (uint32_t)(q / ST) & 1u, a.err, 1, a.wait_ns);
        const unsigned char* stg = stage + (size_t)s * STRIDE;
        const int64_t z0 = ch.zoff * NR;
        using Zin = typename AccT<MODE>::zin;  // same size as Vv
        const Zin* zb = (const Zin*)stg + (z0 - (z0 & ~(int64_t)(ZR::ALIGN - 1)));
        const unsigned char* buf = stg + ZR::BYTES;
        const int rows = 3 * L.n;
        const int cg = deal_start<NG>(g, rot);  // this warp's first column on the CUDA cores
        if constexpr (TC16) {
            if (ch.kind != 0) {
                const uint16_t* ub = (const uint16_t*)buf;
                const int ld = ch.ld, ncols = ch.ncols;
                const int j8 = lane >> 3, i8 = lane & 7, nt = w & 1;
                const uint32_t zaddr = smem_u32(zline);
                // B: matrix j8 = (k half j8 % 2, BF16 high or low part j8 / 2), row i8 = column
                // kb of t in the packed form (64 bytes a column)
                const uint32_t tbase = smem_u32(stg) + 64u * (uint32_t)((j8 & 1) * 8 + i8);
                const int lg0 = (int)(ch.zoff & 7) + (j8 & 1) * 8 + i8, piece = 2 * nt + (j8 >> 1);
                for (int mt = w >> 1; 16 * mt < rows; mt += 8) {
                    const int m0 = 16 * mt + (j8 & 1) * 8;
                    const uint32_t abase = smem_u32(ub + m0);
                    float dh[4] = {0.f, 0.f, 0.f, 0.f}, dl[4] = {0.f, 0.f, 0.f, 0.f};
                    for (int k0 = 0; k0 < ncols; k0 += 16) {
                        // A: this lane addresses slice column k0 + (j8 / 2) 8 + i8, rows m0 ..
                        const int kc = k0 + (j8 >> 1) * 8 + i8, kb = k0 + (j8 & 1) * 8 + i8;
                        const uint32_t aaddr = kc < ncols && m0 < ld ? abase + 2u * (uint32_t)(kc * ld) : zaddr;
                        const uint32_t badd =
                            kb < ncols ? tbase + 64u * (uint32_t)k0 + 16u * (uint32_t)tb16_piece_pos(lg0 + k0, piece)
                                       : zaddr;
                        uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
                        ldsm_x4_t(aaddr, a0, a1, a2, a3);
                        ldsm_x4_t(badd, b0, b1, b2, b3);
                        mma_bf16(dh, a0, a1, a2, a3, b0, b1);  // BF16 high parts of t
                        mma_bf16(dl, a0, a1, a2, a3, b2, b3);  // the low parts
                    }
                    // rows 16 mt + lane / 4 (c0, c1) and + 8 (c2, c3), RHS 8 nt + 2 (lane % 4) +
                    // {0, 1}; summed over the leaf's chunks in ty, read by the flush
                    const int r0 = 16 * mt + (lane >> 2);
                    float* col = ty + (size_t)(8 * nt + 2 * (lane & 3)) * TY_LD;
                    col[r0] += dh[0] + dl[0];
                    col[TY_LD + r0] += dh[1] + dl[1];
                    col[r0 + 8] += dh[2] + dl[2];
                    col[TY_LD + r0 + 8] += dh[3] + dl[3];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty + s);
                continue;
            }
        }
        if constexpr (TC2) {
            if (ch.kind != 0) {
                const uint32_t* zw = (const uint32_t*)zb;  // packed (hi, lo) of t per column
                const uint16_t* ub = (const uint16_t*)buf;
                const int ld = ch.ld, ncols = ch.ncols;
                const int kg = w / TMG, mg = w % TMG, n = lane >> 2;
                const int j8 = lane >> 3, i8 = lane & 7;
                const uint32_t sel = n == 0 ? 0x5410u : 0x7632u;
                const uint32_t zaddr = smem_u32(zline);
#pragma unroll
                for (int tk = 0; tk < 2; ++tk) {
                    const int kt = kg + TKG * tk;
                    if (kt * 16 >= ncols) break;
                    // B: rows k0 + 2 (lane % 4) + {0, 1} and the same + 8; column n
                    uint32_t b[2];
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh) {
                        const int k0 = kt * 16 + hh * 8 + 2 * (lane & 3);
                        const uint32_t w0 = k0 < ncols ? zw[k0] : 0u;
                        const uint32_t w1 = k0 + 1 < ncols ? zw[k0 + 1] : 0u;
                        b[hh] = n < 2 ? __byte_perm(w0, w1, sel) : 0u;
                    }
                    // A: this lane supplies the address of slice column kt*16 + (j8/2)*8 + i8
                    const int kc = kt * 16 + (j8 >> 1) * 8 + i8;
#pragma unroll
                    for (int j = 0; j < TMT; ++j) {
                        const int m0 = (mg + TMG * j) * 16 + (j8 & 1) * 8;
                        const uint32_t addr = (kc < ncols && m0 < ld) ? smem_u32(ub + (size_t)kc * ld + m0) : zaddr;
                        uint32_t a0, a1, a2, a3;
                        ldsm_x4_t(addr, a0, a1, a2, a3);
                        mma_bf16(dt[j], a0, a1, a2, a3, b[0], b[1]);
                    }
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty + s);
                continue;
            }
        }
        // Rows at or beyond `rows` read whatever follows the column in shared memory (the
        // next column, stage or the reduction buffer: always inside the allocation); their
        // accumulators are never flushed, so no bound check is needed per coefficient.
        // Except in the HBM-bound single-RHS F32 loop a warp skips the row blocks past the
        // leaf.
        rot = deal_next<NG>(rot, ch.ncols);
        const int nact = max(0, min(RPW, (rows - rbase + 31) >> 5));
        const float* near_col = (const float*)buf + rbase + lane;
        const C* u_col = (const C*)buf + rbase + lane;
        if constexpr (MODE == 1) {
            if (ch.kind == 0)
                ff_columns_n(acc, nact, near_col, ch.ld, zb, cg, ch.ncols, NG);
            else
                ff_columns_n(acc, nact, u_col, ch.ld, zb, cg, ch.ncols, NG);
        } else if constexpr (MR) {
            if (ch.kind == 0)
                mr_columns_n<NR>(acc2, nact, near_col, ch.ld, zb, cg, ch.ncols, NG);
            else
                mr_columns_n<NR>(acc2, nact, u_col, ch.ld, zb, cg, ch.ncols, NG);
        } else {
            for (int c = cg; c < ch.ncols; c += NG) {
                const Z32 zv = make_z(zb[c]);
                if (ch.kind == 0) {
                    const float* col = near_col + (size_t)c * ch.ld;
#pragma unroll
                    for (int ii = 0; ii < RPW; ++ii) acc_fma(acc[0][ii], col[32 * ii], zv);
                } else {
                    const C* col = u_col + (size_t)c * ch.ld;
#pragma unroll
                    for (int ii = 0; ii < RPW; ++ii) acc_fma(acc[0][ii], coef(col, 32 * ii), zv);
                }
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
    }
    if (cur >= 0) flush();
}

// ---- phase 1: P = V_t^T xc_t, one partial per V column (F32 mode, 1 or 4 right-hand sides)
template <class C, int NR, int RPL, int NCW, int ST = STAGES>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) k_phase1(StreamArgs a) {
    static_assert(NR == 1 || NR == 4, "one right-hand side, or four in pairs");
    using Acc = float;
    using Vv = float;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = (uint64_t*)smem;
    uint64_t* empty = full + ST;
    unsigned char* stage = smem + BAR_BYTES;

    if (a.skip && *(volatile const int*)a.skip) return;  // every right-hand side already converged
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if constexpr (NR == 1) {
        // The single-RHS loop reads whole 32 RPL-row columns without bound checks: rows past
        // a leaf meet x = 0, columns past a chunk are clamped to its last one.  Every byte
        // such a read can reach (the ring and the tail after it) must then be finite, so the
        // ring is zeroed once before the first copy lands in it.
        uint4* z = reinterpret_cast<uint4*>(stage);
        for (int i = threadIdx.x; i < (ST * STAGE_BYTES + P1_TAIL) / 16; i += blockDim.x)
            z[i] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the copies write it
    }
    init_ring<ST>(full, empty, NCW);
    const int c0 = a.cta_begin[blockIdx.x], c1 = a.cta_begin[blockIdx.x + 1];
    pdl_trigger();
    if (w == NCW) {
        // the V coefficients are constant: the copies start while the gather drains
        if (lane == 0) produce<C, Vv, NR, false, false, ST>(a, stage, STAGE_BYTES, full, empty, c0, c1);
        return;
    }
    pdl_wait();  // x in cluster order comes from the preceding kernel
    Vv* P = (Vv*)a.out;
    int cur = -1, rot = 0;
    int rows = 0;
    const float* xs = (const float*)a.xc;
    constexpr bool PAIR = std::is_same<C, uint16_t>::value && NR == 1 && RPL == 6;
    Z32 xr[NR][RPL];
    Chunk nxt = c0 < c1 ? a.chunks[c0] : Chunk{};
    for (int i = c0; i < c1; ++i) {
        const Chunk ch = nxt;
        if (i + 1 < c1) nxt = a.chunks[i + 1];
        const int q = i - c0, s = q % ST;
        if (ch.leaf != cur) {
            cur = ch.leaf;
            const LeafDesc L = a.leaves[cur];
            rows = 3 * L.n;
#pragma unroll
            for (int ii = 0; ii < RPL; ++ii) {
                // BF16 single-RHS columns are read two rows per 32-bit word: lane holds rows
                // 2 lane + 64 (ii / 2) + ii % 2; otherwise rows lane + 32 ii
                const int r = PAIR ? 2 * lane + 64 * (ii >> 1) + (ii & 1) : lane + 32 * ii;
#pragma unroll
                for (int k = 0; k < NR; ++k)
                    xr[k][ii] = make_z(r < rows ? xs[(3 * (int64_t)L.begin + r) * NR + k] : 0.f);
            }
        }
        mbar_wait(full + s, (uint32_t)(q / ST) & 1u, a.err, 1, a.wait_ns);
        const C* buf = (const C*)(stage + (size_t)s * STAGE_BYTES);
        if constexpr (NR == 1) {
            // Four neighbouring columns per pass: their four warp sums share one
            // reduce-scatter (6 shuffles instead of 20) and the loads of four columns are in
            // flight together.
            // (no per-coefficient bound checks: see the ring zeroing at the kernel start)
            constexpr int CG = 4;
            const int units = (ch.ncols + CG - 1) / CG;
            for (int u = deal_start<NCW>(w, rot); u < units; u += NCW) {
                const int c = CG * u;
                Acc acc[CG];
                const C* colp[CG];
#pragma unroll
                for (int j = 0; j < CG; ++j) {
                    acc_zero(acc[j]);
                    colp[j] = buf + (size_t)min(c + j, ch.ncols - 1) * ch.ld;
                }
                if constexpr (PAIR) {
#pragma unroll
                    for (int jj = 0; jj < RPL / 2; ++jj) {
#pragma unroll
                        for (int j = 0; j < CG; ++j) {
                            const uint32_t wv = reinterpret_cast<const uint32_t*>(colp[j])[lane + 32 * jj];
                            acc_fma(acc[j], __uint_as_float(wv << 16), xr[0][2 * jj]);
                            acc_fma(acc[j], __uint_as_float(wv & 0xffff0000u), xr[0][2 * jj + 1]);
                        }
                    }
                } else {
#pragma unroll
                    for (int ii = 0; ii < RPL; ++ii) {
#pragma unroll
                        for (int j = 0; j < CG; ++j) acc_fma(acc[j], coef(colp[j], lane + 32 * ii), xr[0][ii]);
                    }
                }
                const int j = warp_reduce_scatter<CG>(acc, lane);
                const int cj = c + j;
                if ((lane & (32 / CG - 1)) == 0 && cj < ch.ncols) P[ch.zoff + cj] = (Vv)acc_value(acc[0]);
            }
            rot = deal_next<NCW>(rot, units);
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + s);
            continue;
        }
        const int cw = deal_start<NCW>(w, rot);
        rot = deal_next<NCW>(rot, ch.ncols);
        for (int c = cw; c < ch.ncols; c += NCW) {
            const C* col = buf + (size_t)c * ch.ld;
            Acc acc[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) acc_zero(acc[k]);
#pragma unroll
            for (int ii = 0; ii < RPL; ++ii) {
                const int r = lane + 32 * ii;
                const float v = r < rows ? coef(col, r) : 0.f;
#pragma unroll
                for (int k = 0; k < NR; k += 2) acc_fma2(acc[k], acc[k + 1], v, xr[k][ii], xr[k + 1][ii]);
            }
            const int k = warp_reduce_scatter<NR>(acc, lane);
            if ((lane & (32 / NR - 1)) == 0) P[(ch.zoff + c) * NR + k] = (Vv)acc_value(acc[0]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
    }
}

// ---- phase 1 with 5 to 16 right-hand sides (F32 mode)
//
// A warp takes 4 CL neighbouring columns: lane (cg, rl) = (lane / 8, lane % 8) columns
// cg + 4 j (j < CL) and the four rows 4 rl .. 4 rl + 3 of every 32, so that the sums over
// rows meet over 8 lanes only -- 28 shuffles for 8 columns of 16 RHS, where lanes over the
// rows of one column at a time took 16 a column and as many instructions to reduce as to
// multiply (155 a column in all; now about 85).  Coefficients come as 16-byte reads of a
// column (eight lanes read 128 bytes in a row), the leaf's operands from shared memory,
// where they lie so that the eight lanes' 16-byte reads of one row and four RHS are
// contiguous and the four column groups share them; every operand read serves CL columns.
// x past the leaf's rows is zero, and everything an unchecked read can reach is
// finite (the ring is zeroed first), so nothing is bound-checked.  Columns are dealt in units
// of 4 CL across chunks; the ring is six deep because the warps work on about three chunks
// at a time.  16 RHS take eight warps: 64 accumulators and their operands a lane.  Bound by
// the FP32 pipe and shared-memory reads: 16 RHS on three 100 x 100 planes (0.82 GB of V, 0.12 ms at the copy bandwidth): 0.38 ms a column at a time, 0.21 ms now.
template <class C>
__device__ __forceinline__ float4 coef4(const C* p);
template <>
__device__ __forceinline__ float4 coef4<float>(const float* p) {
    return *reinterpret_cast<const float4*>(p);
}
template <>
__device__ __forceinline__ float4 coef4<uint16_t>(const uint16_t* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}

constexpr int MR_STAGES = 6;
// shared-memory float4 index of rows r (of 32 t + 4 rl + i), RHS 4 kq .. 4 kq + 3
template <int NR>
__device__ __forceinline__ int mr_x_index(int t, int i, int kq, int rl) {
    return ((t * 4 + i) * (NR / 4) + kq) * 8 + rl;
}

template <class C, int NR, int NCW>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) k_phase1_mr(StreamArgs a) {
    constexpr int CL = 4, UNIT = 4 * CL;  // columns of a lane, of a warp
    constexpr int NV = CL * NR;           // accumulators of a lane
    static_assert(NR == 8 || NR == 16, "after three halvings a lane holds NV / 8 sums of one column");
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = (uint64_t*)smem;
    uint64_t* empty = full + MR_STAGES;
    unsigned char* stage = smem + BAR_BYTES;
    float4* xs = (float4*)(stage + MR_STAGES * STAGE_BYTES + P1_TAIL);  // the leaf's operands (mr_x_index)
    if (a.skip && *(volatile const int*)a.skip) return;  // every right-hand side already converged
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, cg = lane >> 3, rl = lane & 7;
    {
        uint4* z = reinterpret_cast<uint4*>(stage);
        for (int i = threadIdx.x; i < (MR_STAGES * STAGE_BYTES + P1_TAIL) / 16; i += blockDim.x)
            z[i] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the copies write it
    }
    init_ring<MR_STAGES>(full, empty, NCW);
    const int c0 = a.cta_begin[blockIdx.x], c1 = a.cta_begin[blockIdx.x + 1];
    pdl_trigger();
    if (w == NCW) {
        // the V coefficients are constant: the copies start while the gather drains
        if (lane == 0) produce<C, float, NR, false, false, MR_STAGES>(a, stage, STAGE_BYTES, full, empty, c0, c1);
        return;
    }
    pdl_wait();  // x in cluster order comes from the preceding kernel
    float* P = (float*)a.out;
    const float* xg = (const float*)a.xc;
    int cur = -1, nt = 0, rot = 0;
    Chunk nxt = c0 < c1 ? a.chunks[c0] : Chunk{};
    for (int i = c0; i < c1; ++i) {
        const Chunk ch = nxt;
        if (i + 1 < c1) nxt = a.chunks[i + 1];
        const int q = i - c0, s = q % MR_STAGES;
        if (ch.leaf != cur) {
            consumer_sync(NCW * 32);  // every warp is past the leaf before
            cur = ch.leaf;
            const LeafDesc L = a.leaves[cur];
            const int rows = 3 * L.n;
            nt = (rows + 31) >> 5;
            const float* xl = xg + 3 * (int64_t)L.begin * NR;
            float* xf = reinterpret_cast<float*>(xs);
            for (int e = threadIdx.x; e < nt * 32 * NR; e += NCW * 32) {
                const int r = e / NR, k = e % NR;
                const int at = mr_x_index<NR>(r >> 5, r & 3, k >> 2, (r & 31) >> 2);
                xf[4 * at + (k & 3)] = r < rows ? xl[e] : 0.f;
            }
            consumer_sync(NCW * 32);
        }
        mbar_wait(full + s, (uint32_t)(q / MR_STAGES) & 1u, a.err, 1, a.wait_ns);
        const C* buf = (const C*)(stage + (size_t)s * STAGE_BYTES);
        const int units = (ch.ncols + UNIT - 1) / UNIT;
        for (int u = deal_start<NCW>(w, rot); u < units; u += NCW) {
            const C* colp[CL];
#pragma unroll
            for (int j = 0; j < CL; ++j)
                colp[j] = buf + (size_t)min(u * UNIT + cg + 4 * j, ch.ncols - 1) * ch.ld + 4 * rl;
            float2 acc[CL][NR / 2];
#pragma unroll
            for (int j = 0; j < CL; ++j)
#pragma unroll
                for (int k = 0; k < NR / 2; ++k) acc[j][k] = make_float2(0.f, 0.f);
            for (int t = 0; t < nt; ++t) {
                float v[CL][4];
#pragma unroll
                for (int j = 0; j < CL; ++j) {
                    const float4 f = coef4<C>(colp[j] + 32 * t);
                    v[j][0] = f.x, v[j][1] = f.y, v[j][2] = f.z, v[j][3] = f.w;
                }
#pragma unroll
                for (int i4 = 0; i4 < 4; ++i4) {
#pragma unroll
                    for (int kq = 0; kq < NR / 4; ++kq) {
                        const float4 x = xs[mr_x_index<NR>(t, i4, kq, rl)];
#pragma unroll
                        for (int j = 0; j < CL; ++j) {
                            const float2 vv = make_float2(v[j][i4], v[j][i4]);
                            acc[j][2 * kq] = __ffma2_rn(vv, make_float2(x.x, x.y), acc[j][2 * kq]);
                            acc[j][2 * kq + 1] = __ffma2_rn(vv, make_float2(x.z, x.w), acc[j][2 * kq + 1]);
                        }
                    }
                }
            }
            // NV sums over the 8 row lanes: halving exchanges leave each lane NV / 8 RHS of a column
            float f[NV];
#pragma unroll
            for (int j = 0; j < CL; ++j)
#pragma unroll
                for (int k = 0; k < NR / 2; ++k) {
                    f[j * NR + 2 * k] = acc[j][k].x;
                    f[j * NR + 2 * k + 1] = acc[j][k].y;
                }
            int e = 0;
#pragma unroll
            for (int h = NV / 2, o = 4; o >= 1; h >>= 1, o >>= 1) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int j = 0; j < h; ++j) {
                    const float mine = up ? f[j + h] : f[j], other = up ? f[j] : f[j + h];
                    f[j] = mine + __shfl_xor_sync(0xffffffffu, other, o);
                }
                if (up) e += h;
            }
            const int c = u * UNIT + cg + 4 * (e / NR), k = e % NR;  // this lane: column c, RHS k ...
            if (c < ch.ncols) {
#pragma unroll
                for (int j = 0; j < NV / 8; j += 4)
                    *reinterpret_cast<float4*>(P + (ch.zoff + c) * NR + k + j) =
                        make_float4(f[j], f[j + 1], f[j + 2], f[j + 3]);
            }
        }
        rot = deal_next<NCW>(rot, units);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
    }
}

// ---- phase 1 in F64 mode (1 to 4 right-hand sides)
//
// A warp takes a column at a time, lanes over rows, with four dot products in flight --
// four columns for one RHS, two for two, one for three or four -- packed in pairs (over
// the columns for one RHS, over the RHS otherwise) for the packed FP32 instructions; the
// four sums over the warp share one reduce-scatter.  The leaf's operands stay in registers
// already split.  A partial leaves as a double, hi + lo added in FP64; eight passes wait for
// that (HeldParts), a lane of every eight holding each, so that the addition fills its warp:
// one pass at a time it had kept the FP64 pipe a third busy.  Rows past a leaf meet x = 0,
// and NA, the row blocks of 32 the leaf really has, is a template argument of the column
// loop.
// Bound by the FP32 pipe and its issue (a packed instruction takes the pipe two cycles, so
// packing saves issue slots, not pipe time).  One RHS, 25,700 triangles (444 MB of V,
// 65 us at the copy bandwidth): 116 us with scalar operations over 192 rows, 104 us packed
// over the leaf's row blocks, 92 us with the columns dealt across chunks (deal_start); the
// whole product 358 us before, 309 now.
// The sums of up to eight passes, a lane of every eight holding each.
struct HeldParts {
    FF v;
    int64_t at;  // entry of P; -1: none
    int n;       // passes held
    __device__ __forceinline__ void store(double* P) {
        if (at >= 0) P[at] = acc_value(v);
        at = -1;
        n = 0;
    }
};

constexpr int ff_phase1_group(int NR) { return NR == 1 ? 4 : (NR == 2 ? 2 : 1); }  // columns per pass
template <int NA, int NR, int RPL, class C, class Ld>
__device__ __forceinline__ void ff_phase1_columns(const float2 (&x)[NR][RPL], const C* buf, int ld, int u0, int ncw,
                                                  int ncols, int lane, int64_t zoff, double* P, HeldParts& held,
                                                  Ld load) {
    constexpr int CG = ff_phase1_group(NR);
    for (int c = CG * u0; c < ncols; c += CG * ncw) {
        FF2 acc[2];
        acc_zero(acc[0]);
        acc_zero(acc[1]);
        const C* colp[CG];
#pragma unroll
        for (int j = 0; j < CG; ++j) colp[j] = buf + (size_t)min(c + j, ncols - 1) * ld;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            float v[CG];
#pragma unroll
            for (int j = 0; j < CG; ++j) v[j] = load(colp[j], i);
            if constexpr (NR == 1) {
                const float2 xh = make_float2(x[0][i].x, x[0][i].x), xl = make_float2(x[0][i].y, x[0][i].y);
                ff_fma2(acc[0], make_float2(v[0], v[1]), xh, xl);
                ff_fma2(acc[1], make_float2(v[2], v[3]), xh, xl);
            } else if constexpr (NR == 2) {
                const float2 xh = make_float2(x[0][i].x, x[1][i].x), xl = make_float2(x[0][i].y, x[1][i].y);
                ff_fma2(acc[0], make_float2(v[0], v[0]), xh, xl);
                ff_fma2(acc[1], make_float2(v[1], v[1]), xh, xl);
            } else {
                const float2 vv = make_float2(v[0], v[0]);
                ff_fma2(acc[0], vv, make_float2(x[0][i].x, x[1][i].x), make_float2(x[0][i].y, x[1][i].y));
                if constexpr (NR == 4)
                    ff_fma2(acc[1], vv, make_float2(x[2][i].x, x[3][i].x), make_float2(x[2][i].y, x[3][i].y));
                else
                    ff_fma(acc[1].hi.x, acc[1].lo.x, v[0], x[2][i].x, x[2][i].y);
            }
        }
        FF q[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            q[2 * h] = FF{acc[h].hi.x, acc[h].lo.x};
            q[2 * h + 1] = FF{acc[h].hi.y, acc[h].lo.y};
        }
        const int m = warp_reduce_scatter<4>(q, lane);  // value m: column m (one RHS), m / NR (two), RHS m (more)
        const int cj = c + (NR == 1 ? m : (NR == 2 ? m >> 1 : 0)), k = NR == 1 ? 0 : (NR == 2 ? m & 1 : m);
        if ((lane & 7) == held.n) {  // all eight lanes of a group have the sum
            held.v = q[0];
            held.at = cj < ncols && k < NR ? (zoff + cj) * NR + k : -1;
        }
        if (++held.n == 8) held.store(P);
    }
}

template <class C, int NR, int RPL, int NCW, bool PASSES>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) k_phase1_f64(StreamArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = (uint64_t*)smem;
    uint64_t* empty = full + STAGES;
    unsigned char* stage = smem + BAR_BYTES;
    if (a.skip && *(volatile const int*)a.skip) return;  // every right-hand side already converged
    if constexpr (PASSES) {  // fewer chunks than CTAs: the next pass's CTA takes the SM
        if (a.cta_begin[blockIdx.x] == a.cta_begin[blockIdx.x + 1]) return;
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {  // finite data behind every unchecked column read, as in k_phase1
        uint4* z = reinterpret_cast<uint4*>(stage);
        for (int i = threadIdx.x; i < (STAGES * STAGE_BYTES + P1_TAIL) / 16; i += blockDim.x)
            z[i] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the copies write it
    }
    init_ring(full, empty, NCW);
    const int c0 = a.cta_begin[blockIdx.x], c1 = a.cta_begin[blockIdx.x + 1];
    pdl_trigger();
    if (w == NCW) {
        // the V coefficients are constant: the copies start while the gather drains
        if (lane == 0) produce<C, float2, NR, false>(a, stage, STAGE_BYTES, full, empty, c0, c1);
        return;
    }
    pdl_wait();  // x in cluster order comes from the preceding kernel
    double* P = (double*)a.out;
    const float2* xs = (const float2*)a.xc;
    if constexpr (PASSES) {
        P += blockIdx.y * a.p_pass;
        xs += blockIdx.y * a.xc_pass;
    }
    HeldParts held{FF{0.f, 0.f}, -1, 0};
    int cur = -1, rows = 0, rot = 0;
    float2 x[NR][RPL];
    auto load = [lane](const C* col, int i) { return coef(col, lane + 32 * i); };
    Chunk nxt = c0 < c1 ? a.chunks[c0] : Chunk{};
    for (int i = c0; i < c1; ++i) {
        const Chunk ch = nxt;
        if (i + 1 < c1) nxt = a.chunks[i + 1];
        const int q = i - c0, s = q % STAGES;
        if (ch.leaf != cur) {
            cur = ch.leaf;
            const LeafDesc L = a.leaves[cur];
            rows = 3 * L.n;
#pragma unroll
            for (int ii = 0; ii < RPL; ++ii) {
                const int r = lane + 32 * ii;
#pragma unroll
                for (int k = 0; k < NR; ++k)
                    x[k][ii] = r < rows ? xs[(3 * (int64_t)L.begin + r) * NR + k] : make_float2(0.f, 0.f);
            }
        }
        mbar_wait(full + s, (uint32_t)(q / STAGES) & 1u, a.err, 1, a.wait_ns);
        const C* buf = (const C*)(stage + (size_t)s * STAGE_BYTES);
        const int u0 = deal_start<NCW>(w, rot);
        rot = deal_next<NCW>(rot, (ch.ncols + ff_phase1_group(NR) - 1) / ff_phase1_group(NR));
        if constexpr (RPL == 6) {
            if (rows <= 128)
                ff_phase1_columns<4, NR, RPL>(x, buf, ch.ld, u0, NCW, ch.ncols, lane, ch.zoff, P, held, load);
            else if (rows <= 160)
                ff_phase1_columns<5, NR, RPL>(x, buf, ch.ld, u0, NCW, ch.ncols, lane, ch.zoff, P, held, load);
            else
                ff_phase1_columns<6, NR, RPL>(x, buf, ch.ld, u0, NCW, ch.ncols, lane, ch.zoff, P, held, load);
        } else {
            ff_phase1_columns<RPL, NR, RPL>(x, buf, ch.ld, u0, NCW, ch.ncols, lane, ch.zoff, P, held, load);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
    }
    held.store(P);
}

// ---- phase 1 on tensor cores: BF16 V factors, 16 right-hand sides
//
// P (columns x 16) = V_chunk^T X_leaf as mma.sync m16n8k16 BF16 x BF16 -> FP32: the A
// operand is V^T (row m = V column, k = leaf row; a column of the stream is contiguous in
// shared memory, so ldmatrix reads A fragments directly), the B operand the leaf's rows
// of x, each value split into BF16 hi + lo (two products, x kept to ~16 bits), kept in
// registers for the whole leaf.  Warp w takes n-tile w % 2 (8 RHS) and m-tiles
// w / 2, w / 2 + NCW / 2, ..., dealt across chunks; nothing is bound-checked: rows past the
// leaf meet x = 0 and every byte a read can reach is finite (the ring is zeroed first).
constexpr int TC_KT = 12;  // k-tiles of 16 rows: leaves of up to 192 rows

template <int NCW>
__global__ void __launch_bounds__((NCW + 1) * 32, 1) k_phase1_tc(StreamArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t* full = (uint64_t*)smem;
    uint64_t* empty = full + STAGES;
    unsigned char* stage = smem + BAR_BYTES;

    if (a.skip && *(volatile const int*)a.skip) return;  // every right-hand side already converged
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {  // finite data behind every unchecked read, as in k_phase1
        uint4* z = reinterpret_cast<uint4*>(stage);
        for (int i = threadIdx.x; i < (STAGES * STAGE_BYTES + P1_TAIL) / 16; i += blockDim.x)
            z[i] = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the copies write it
    }
    init_ring(full, empty, NCW);
    const int c0 = a.cta_begin[blockIdx.x], c1 = a.cta_begin[blockIdx.x + 1];
    pdl_trigger();
    if (w == NCW) {
        if (lane == 0) produce<uint16_t, float, 16, false>(a, stage, STAGE_BYTES, full, empty, c0, c1);
        return;
    }
    pdl_wait();
    const float* xc = (const float*)a.xc;
    float* P = (float*)a.out;
    const int nt = w & 1;
    int cur = -1, rows = 0, rot = 0;
    uint32_t bh[TC_KT][2], bl[TC_KT][2];
    Chunk nxt = c0 < c1 ? a.chunks[c0] : Chunk{};
    for (int i = c0; i < c1; ++i) {
        const Chunk ch = nxt;
        if (i + 1 < c1) nxt = a.chunks[i + 1];
        const int q = i - c0, s = q % STAGES;
        if (ch.leaf != cur) {
            cur = ch.leaf;
            const LeafDesc L = a.leaves[cur];
            rows = 3 * L.n;
            // B fragments: b0b1 = X[k0 + 2 (lane % 4) + {0, 1}][n], b2b3 = the same 8 rows on
            // (n = nt * 8 + lane / 4), low half the smaller k
            const int n = nt * 8 + (lane >> 2);
#pragma unroll
            for (int kt = 0; kt < TC_KT; ++kt)
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    uint32_t hi2 = 0, lo2 = 0;
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int k = kt * 16 + hh * 8 + 2 * (lane & 3) + e;
                        const float x = k < rows ? xc[(3 * (int64_t)L.begin + k) * 16 + n] : 0.f;
                        const uint32_t hb = bf16_bits(x);
                        const uint32_t lb = bf16_bits(x - bf16_value(hb));
                        hi2 |= hb << (16 * e);
                        lo2 |= lb << (16 * e);
                    }
                    bh[kt][hh] = hi2;
                    bl[kt][hh] = lo2;
                }
        }
        mbar_wait(full + s, (uint32_t)(q / STAGES) & 1u, a.err, 1, a.wait_ns);
        const uint16_t* buf = (const uint16_t*)(stage + (size_t)s * STAGE_BYTES);
        const int ld = ch.ld, ncols = ch.ncols;
        const int mtiles = (ncols + 15) >> 4;
        const int j8 = lane >> 3, i8 = lane & 7;
        for (int mt = deal_start<NCW / 2>(w >> 1, rot); mt < mtiles; mt += NCW / 2) {
            // this lane's ldmatrix row: a V column; columns past the chunk repeat its last one
            // and are not stored
            const int m = min(mt * 16 + (j8 & 1) * 8 + i8, ncols - 1);
            const uint32_t row = smem_u32(buf + (size_t)m * ld + (j8 >> 1) * 8);
            float d[4] = {0.f, 0.f, 0.f, 0.f}, dl[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kt = 0; kt < TC_KT; ++kt) {
                if (kt * 16 >= rows) break;
                uint32_t a0, a1, a2, a3;
                ldsm_x4(row + 32u * kt, a0, a1, a2, a3);
                mma_bf16(d, a0, a1, a2, a3, bh[kt][0], bh[kt][1]);
                mma_bf16(dl, a0, a1, a2, a3, bl[kt][0], bl[kt][1]);
            }
            // d0, d1: column mt*16 + lane/4, RHS nt*8 + 2 (lane % 4) + {0, 1}; d2, d3: column + 8
            const int col = mt * 16 + (lane >> 2), rhs = nt * 8 + 2 * (lane & 3);
            if (col < ncols)
                *reinterpret_cast<float2*>(P + (ch.zoff + col) * 16 + rhs) = make_float2(d[0] + dl[0], d[1] + dl[1]);
            if (col + 8 < ncols)
                *reinterpret_cast<float2*>(P + (ch.zoff + col + 8) * 16 + rhs) =
                    make_float2(d[2] + dl[2], d[3] + dl[3]);
        }
        rot = deal_next<NCW / 2>(rot, mtiles);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
    }
}

// launch with programmatic stream serialisation (the kernel may start before its
// predecessor on the stream completes; it synchronises through griddepcontrol.wait)
template <class... P, class... A>
void launch_pdl(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    HM_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

constexpr int EV_PER_PRODUCT = 6;
constexpr int EV_POOL = EV_PER_PRODUCT * 1024;

void timing_accumulate(HMat& H) {
    if (H.ev_used == 0) return;
    HM_CUDA(cudaEventSynchronize(H.ev[H.ev_used - 1]));
    for (int s = 0; s < H.ev_used; s += EV_PER_PRODUCT) {
        for (int i = 0; i < 5; ++i) {
            float ms = 0.f;
            HM_CUDA(cudaEventElapsedTime(&ms, H.ev[s + i], H.ev[s + i + 1]));
            H.t_acc[i] += ms;
        }
    }
    H.ev_used = 0;
}

// phase boundary idx (0 before the gather, 4 and 5 after phase 2) of one product
void mark(HMat& H, int idx, cudaStream_t st) {
    if (!H.timing) return;
    if (idx == 0 && H.ev_used + EV_PER_PRODUCT > (int)H.ev.size()) timing_accumulate(H);
    HM_CUDA(cudaEventRecord(H.ev[H.ev_used + idx], st));
    if (idx == EV_PER_PRODUCT - 1) H.ev_used += EV_PER_PRODUCT;
}

// consumer warps of phase 1 and phase 2, and phase 2's row split, per right-hand-side
// count: as many warps as the per-thread registers (accumulators and operands) allow.
// (Left spilling: k_phase1_f64 with three or four right-hand sides on leaves above 64 elements,
// 140 to 292 bytes of its operands, and the BF16 16-RHS phase 2 on 192-row leaves, 56 bytes.)
// Phase 2's row split: two or three row blocks per warp with 16 RHS, else (one F32 RHS apart)
// six
template <int MODE>
constexpr int rs_for(int NR, int RPL) {
    return MODE == 0 && NR == 1 ? 1 : (NR == 16 ? (RPL == 4 ? 2 : RPL / 3) : RPL / 6);
}

// ST: ring depth; NCW1V / NCW2V: consumer warps of phase 1 / phase 2 (0: the default for
// the right-hand-side count).  The tile-shape variants the autotuner chooses from use
// other values for the single-RHS FP32-vector product.
// With the producer warp, 16 consumer warps put five warps on one quarter of the SM and
// leave 96 registers a thread; 15 (14 for an even row split) leave 128, which the 48
// accumulators and split operands of three or four F64 right-hand sides need.
template <int MODE>
constexpr int ncw2_for(int NR, int RS) {
    return MODE == 1 && NR > 2 ? 16 - RS : 16;
}

template <int MODE, class C, int NR, int RPL, int ST = STAGES, int NCW1V = 0, int NCW2V = 0, bool TC = true,
          bool PASSES = false>
void launch_phases(HMat& H, const HMat::Plan& PL, const StreamArgs& base, bool timed, cudaStream_t st) {
    constexpr int NCW = NCW1V ? NCW1V : (MODE == 0 && NR == 16 ? 8 : 16), RS = rs_for<MODE>(NR, RPL),
                  NCW2 = NCW2V ? NCW2V : ncw2_for<MODE>(NR, RS);
    static_assert(MODE == 0 || (NR <= F64_PASS && ST == STAGES), "F64 passes");
    using Acc = typename AccT<MODE>::type;
    using V = typename AccT<MODE>::vec;
    // BF16 factors with 16 RHS on leaves of up to 192 rows: phase 1 on tensor cores
    constexpr bool kTensorPhase1 = TC && MODE == 0 && NR == 16 && std::is_same<C, uint16_t>::value && RPL <= 6;
    constexpr bool MR1 = MODE == 0 && NR > 4 && !kTensorPhase1;  // phase 1 over column groups
    auto* const phase1 = [] {
        if constexpr (kTensorPhase1)
            return k_phase1_tc<NCW>;
        else if constexpr (MR1)
            return k_phase1_mr<C, NR, NCW>;
        else if constexpr (MODE == 0)
            return k_phase1<C, NR, RPL, NCW, ST>;
        else
            return k_phase1_f64<C, NR, RPL, NCW, PASSES>;
    }();
    constexpr size_t smem1_ring = BAR_BYTES + (size_t)(MR1 ? MR_STAGES : ST) * STAGE_BYTES + P1_TAIL;
    constexpr size_t smem1 = smem1_ring + (MR1 ? (size_t)32 * RPL * NR * sizeof(float) : 0);
    // k_phase1_mr is one function for every RPL: its opt-in is that of the largest leaves,
    // whichever instantiation of this one sets it (a smaller one set later would refuse them)
    constexpr size_t smem1_max = smem1_ring + (MR1 ? (size_t)32 * MAX_RPL * NR * sizeof(float) : 0);
    static_assert(RPL <= MAX_RPL, "the opt-in covers every leaf size");
    // BF16 factors with one RHS: the U slices of phase 2 on tensor cores, which read t in
    // packed BF16 (hi, lo) form (phase 1 stays on the CUDA cores: one mma.sync per 16 x 16
    // tile did not keep up with the stream there)
    constexpr bool kTensorPhase2x1 = MODE == 0 && NR == 1 && std::is_same<C, uint16_t>::value && RPL == 6;
    static_assert(!kTensorPhase2x1 || (NCW2 == 16 && RS == 1),
                  "the single-RHS tensor-core phase 2 assumes 16 consumer warps without row split");
    // BF16 factors with 16 RHS: the U slices of phase 2 on tensor cores as well, reading t
    // in the packed BF16 form of k_reduce_pack16_mix
    constexpr bool kTensorPhase2x16 = kTensorPhase1;
    constexpr int KP = (MODE == 0 && NR == 16 && RPL <= 6) ? 8 : 1;  // RHS per flush pass of k_phase2
    const size_t smem2 = BAR_BYTES + (size_t)ST * (ZRange<V, NR>::BYTES + STAGE_BYTES) +
                         (size_t)KP * (NCW2 / RS) * 32 * RPL * sizeof(Acc) + (kTensorPhase2x16 ? 16 * 196 * 4 : 0);
    // shared-memory opt-in, once per device for each instantiation
    static bool attr_done[64] = {};
    int dev = 0;
    HM_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        HM_CUDA(cudaFuncSetAttribute(phase1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1_max));
        HM_CUDA(cudaFuncSetAttribute(k_phase2<MODE, C, NR, RPL, NCW2, RS, ST, TC, PASSES>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2));
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    const unsigned passes = PASSES ? (unsigned)ceil_div(base.nout, NR) : 1u;
    if (H.n_far > 0 && H.p_len > 0) {
        StreamArgs a = base;
        a.chunks = PL.ch1.p;
        a.cta_begin = PL.cta1.p;
        a.out = MODE == 0 ? (void*)H.Pf.p : (void*)H.P.p;
        launch_pdl(phase1, dim3(H.grid, passes), dim3((NCW + 1) * 32), smem1, st, a);
        HM_LAUNCH_CHECK();
        if (timed) mark(H, 2, st);
        using Zt = typename AccT<MODE>::zin;
        // several FP32 RHS in multiples of 4: the float4 variant (nrhs 1 keeps the scalar one);
        // BF16 factors with one RHS: t packed as BF16 (hi, lo) for the tensor-core phase 2
        // one RHS: big blocks a CTA each, the others a warp each (red_order)
        const unsigned gm = (unsigned)std::max<int64_t>(1, H.n_red_big + (H.n_red - H.n_red_big + 7) / 8);
        if constexpr (kTensorPhase2x1)
            launch_pdl(k_reduce_mix<V, uint32_t>, dim3(gm), dim3(256), 0, st, (const FarDesc*)H.far.p,
                       (const int32_t*)H.poff.p, (const int32_t*)H.uoff.p, (const int32_t*)H.red_order.p,
                       H.n_red_big, H.n_red,
                       (const V*)a.out, (uint32_t*)base.tb, base.skip);
        else if constexpr (kTensorPhase2x16)
            launch_pdl(k_reduce_pack16_mix, dim3(gm), dim3(256), 0, st, (const FarDesc*)H.far.p,
                       (const int32_t*)H.poff.p, (const int32_t*)H.uoff.p, (const int32_t*)H.red_order.p,
                       H.n_red_big, H.n_red, (const float*)a.out, (uint16_t*)base.tb, base.skip);
        else if constexpr (NR == 1)
            launch_pdl(k_reduce_mix<V, Zt>, dim3(gm), dim3(256), 0, st, (const FarDesc*)H.far.p,
                       (const int32_t*)H.poff.p, (const int32_t*)H.uoff.p, (const int32_t*)H.red_order.p,
                       H.n_red_big, H.n_red,
                       (const V*)a.out, (Zt*)base.tb, base.skip);
        else
            launch_pdl(k_reduce_tb<V, Zt, MODE == 0>, dim3((unsigned)H.n_far, passes), dim3(128), 0, st,
                       (const FarDesc*)H.far.p, (const int32_t*)H.poff.p, (const int32_t*)H.uoff.p,
                       (const V*)a.out, (Zt*)base.tb, NR, base.p_pass, base.tb_pass, base.skip);
        HM_LAUNCH_CHECK();
        if (timed) mark(H, 3, st);
    } else if (timed) {
        mark(H, 2, st);
        mark(H, 3, st);
    }
    StreamArgs a = base;
    a.chunks = PL.ch2.p;
    a.cta_begin = PL.cta2.p;
    a.split = PL.split.p;
    a.wait_x = !(H.n_far > 0 && H.p_len > 0);
    launch_pdl(k_phase2<MODE, C, NR, RPL, NCW2, RS, ST, TC, PASSES>, dim3(H.grid, passes), dim3((NCW2 + 1) * 32), smem2,
               st, a);
    HM_LAUNCH_CHECK();
    if (timed) mark(H, 4, st);
}

template <int MODE, class C, int NR, bool TC = true, bool PASSES = false>
void launch_rpl(HMat& H, const HMat::Plan& PL, const StreamArgs& a, bool timed, cudaStream_t st) {
    // 16 RHS split a column's rows over two warps, so leaves of at most 128 rows have a
    // variant of their own: with three row blocks a warp, one of 99 rows left the second warp
    // one block (three 150 x 150 planes, BF16: phase 2 1,175 us, 905 with exact counts, 692 with
    // two blocks and two and the finer tensor-core mapping; a split computed from each leaf's
    // rows cost the 176-row leaves of three 100 x 100 planes 10 %)
    if (NR == 16 && H.ld_max <= 128) {
        if constexpr (NR == 16) launch_phases<MODE, C, NR, 4, STAGES, 0, 0, TC, PASSES>(H, PL, a, timed, st);
    } else if (H.ld_max <= 192)
        launch_phases<MODE, C, NR, 6, STAGES, 0, 0, TC, PASSES>(H, PL, a, timed, st);
    else
        launch_phases<MODE, C, NR, MAX_RPL, STAGES, 0, 0, true, PASSES>(H, PL, a, timed, st);
}

// The single-RHS FP32-vector product with the ring depth and consumer-warp count of the
// H-matrix's tile shape (leaves of up to 64 elements); false if the shape is the default.
// BF16 factors keep 16 warps in phase 2 (its tensor-core U slices assume them).
template <class C>
bool launch_shape_variant(HMat& H, const HMat::Plan& PL, const StreamArgs& a, bool timed, cudaStream_t st) {
    const int ring = H.shape.ring, warps = H.shape.warps;
    if (H.ld_max > 192 || (ring == STAGES && warps == 16)) return false;
    constexpr bool b16 = std::is_same<C, uint16_t>::value;
    if (ring == 6 && warps == 16)
        launch_phases<0, C, 1, 6, 6>(H, PL, a, timed, st);
    else if (ring == STAGES && warps == 8)
        launch_phases<0, C, 1, 6, STAGES, 8, b16 ? 16 : 8>(H, PL, a, timed, st);
    else if (ring == 6 && warps == 8)
        launch_phases<0, C, 1, 6, 6, 8, b16 ? 16 : 8>(H, PL, a, timed, st);
    else
        fail(HM_EINVAL, "product: unsupported tile shape");
    return true;
}

template <int MODE, class C>
void launch_nr(HMat& H, const HMat::Plan& PL, const StreamArgs& a, int nrhs, bool timed, cudaStream_t st) {
    if constexpr (MODE == 1) {
        if (a.nout > nrhs) {  // several passes: of three or four
            return nrhs == 3 ? launch_rpl<MODE, C, 3, true, true>(H, PL, a, timed, st)
                             : launch_rpl<MODE, C, 4, true, true>(H, PL, a, timed, st);
        }
        switch (nrhs) {
            case 1: return launch_rpl<MODE, C, 1>(H, PL, a, timed, st);
            case 2: return launch_rpl<MODE, C, 2>(H, PL, a, timed, st);
            case 3: return launch_rpl<MODE, C, 3>(H, PL, a, timed, st);
            case 4: return launch_rpl<MODE, C, 4>(H, PL, a, timed, st);
            default: fail(HM_EINVAL, "product: F64 passes of 1 to 4 right-hand sides");
        }
    } else {
        switch (nrhs) {
            case 1: return launch_rpl<MODE, C, 1>(H, PL, a, timed, st);
            case 4: return launch_rpl<MODE, C, 4>(H, PL, a, timed, st);
            case 8: return launch_rpl<MODE, C, 8>(H, PL, a, timed, st);
            case 16:
                if constexpr (std::is_same<C, uint16_t>::value) {
                    // The tensor-core phases keep about 16 bits of the vectors, which the
                    // interface states for full passes only: 9 to 15 keep FP32 vectors
                    // (12 on three 150 x 150 planes: 1.94 ms; 16 on tensor cores: 1.21).
                    if (a.nout < 16) return launch_rpl<MODE, C, 16, false>(H, PL, a, timed, st);
                }
                return launch_rpl<MODE, C, 16>(H, PL, a, timed, st);
            default: fail(HM_EINVAL, "product: 1, 4, 8 or 16 right-hand sides per F32 pass");
        }
    }
}

// The F32 kernels take 1, 4, 8 or 16 right-hand sides: other counts are padded with zero
// vectors, whose products are not written.  (12 right-hand sides, BF16 factors, three 150 x
// 150 planes: 4.03 ms with kernels that tested the count in their loops, 1.94 padded.)
int padded_rhs(int nr) { return nr == 1 ? 1 : (nr <= 4 ? 4 : (nr <= 8 ? 8 : 16)); }

// The F64 passes that share one set of launches for the first right-hand sides of nr: count of
// them, width of each, right-hand sides covered.  A set of launches costs 12 to 15 us where the
// operator is small: 16 right-hand sides of 256 elements took 90 us in four sets, 58 us in the
// single wide pass those had replaced, and take 31 us as four passes of one set; 12,892
// elements: 1,457 us in four sets, 1,401 us in one.  Where nr does not divide, equal passes are
// padded with zero vectors as long as the work of those (F64_PAD_COEFS stored coefficients,
// about 5 us) is below a set of launches; beyond, the passes of four go first and the rest is a
// set of its own.
struct F64Passes {
    int count, width, nrhs;
};
constexpr int64_t F64_PAD_COEFS = 16 << 20;
F64Passes f64_passes(const HMat& H, int nr) {
    nr = std::min(nr, 16);
    const int count = (int)ceil_div(nr, F64_PASS), width = (int)ceil_div(nr, count);
    if ((count * width - nr) * (H.near_entries + H.far_entries) <= F64_PAD_COEFS) return F64Passes{count, width, nr};
    return F64Passes{nr / F64_PASS, F64_PASS, nr / F64_PASS * F64_PASS};
}
// elements of one pass's interleaved vectors of len entries: the next pass starts 16-byte aligned
int64_t f64_pass_stride(int64_t len, int width) { return (len * width + 1) & ~(int64_t)1; }

// phase 1, reduction and phase 2 on cluster-ordered operands (see hmat_impl.h); F32: xc
// interleaved by padded_rhs(nr); F64: as k_gather_split lays it out for f64_passes(nr).  perm: yc in user order.
void run_core(HMat& H, const void* xc, void* yc, int nr, int dtype, int fac, bool timed, cudaStream_t st,
              const int* skip = nullptr, const int32_t* perm = nullptr) {
    if (!has_factors(H, fac)) fail(HM_EINVAL, "product: the requested factor precision is not stored");
    const HMat::Plan& PL = H.plan[fac];
    StreamArgs a{};
    a.leaves = H.leaves.p;
    a.near = H.near.p;
    a.ucoef = fac == 1 ? (const void*)H.u16.p : (const void*)H.u32.p;
    a.vcoef = fac == 1 ? (const void*)H.v16.p : (const void*)H.v32.p;
    a.counters = H.counters.p;
    a.err = H.err.p;
    a.ndof = H.ndof;
    a.nout = nr;
    a.perm = perm;
    a.ld_max = H.ld_max;
    a.skip = skip;
    a.wait_ns = H.wait_ns;
    a.withhold = H.withhold_chunk;
    a.xc = xc;
    a.out = yc;
    if (dtype == HM_F32) {
        a.tb = H.tbf.p;
        a.slots = H.slotsf.p;
        if (nr == 1 && (fac == 1 ? launch_shape_variant<uint16_t>(H, PL, a, timed, st)
                                 : launch_shape_variant<float>(H, PL, a, timed, st)))
            return;
        if (fac == 1)
            launch_nr<0, uint16_t>(H, PL, a, padded_rhs(nr), timed, st);
        else
            launch_nr<0, float>(H, PL, a, padded_rhs(nr), timed, st);
    } else {
        a.tb = H.tb.p;
        a.slots = H.slotsd.p;
        const F64Passes ps = f64_passes(H, nr);
        if (ps.nrhs != nr) fail(HM_EINVAL, "product: right-hand sides of more than one set of F64 passes");
        a.xc_pass = f64_pass_stride(H.ndof, ps.width);
        a.p_pass = f64_pass_stride(H.p_len, ps.width);
        a.tb_pass = f64_pass_stride(H.tb_len, ps.width);
        a.slots_pass = PL.n_slots;
        a.counters_pass = H.n_leaves;
        if (fac == 1)
            launch_nr<1, uint16_t>(H, PL, a, ps.width, timed, st);
        else
            launch_nr<1, float>(H, PL, a, ps.width, timed, st);
    }
}

}  // namespace

void build_plan_for(HMat& H, HMat::Plan& PLAN, int esz, int G, cudaStream_t st);

void build_product_plan(HMat& H, cudaStream_t st) {
    int dev = 0, nsm = 0;
    HM_CUDA(cudaGetDevice(&dev));
    HM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    H.grid = std::max(1, nsm);
    const int G = H.grid;
    H.ld_max = 0;
    for (const LeafDesc& L : H.h_leaves) H.ld_max = std::max(H.ld_max, L.ld);
    for (int fac = 0; fac < 2; ++fac)
        if (has_factors(H, fac)) build_plan_for(H, H.plan[fac], fac == 1 ? 2 : 4, G, st);
    H.counters.alloc((size_t)H.n_leaves * (16 / F64_PASS));  // per pass of a product
    HM_CUDA(cudaMemsetAsync(H.counters.p, 0, H.counters.bytes(), st));
    // single-RHS reduction order: blocks with many leaves of T first, factorless ones out
    std::vector<int32_t> big, small;
    for (int64_t b = 0; b < H.n_far; ++b) {
        const FarDesc& F = H.h_far[b];
        if (F.rank <= 0) continue;
        if (F.rank > 256) fail(HM_EINVAL, "product plan: rank above 256");
        (F.n_tleaves > RED_WARP_LEAVES ? big : small).push_back((int32_t)b);
    }
    H.n_red_big = (int64_t)big.size();
    H.n_red = H.n_red_big + (int64_t)small.size();
    big.insert(big.end(), small.begin(), small.end());
    if (big.empty()) big.push_back(0);
    H.red_order.upload(big, st);
    H.err.alloc(1);
    HM_CUDA(cudaMemsetAsync(H.err.p, 0, sizeof(int), st));
}

void build_plan_for(HMat& H, HMat::Plan& PLAN, int esz, int G, cudaStream_t st) {

    // cut a segment into chunks: runs of consecutive operand indices, bounded in size
    auto cut = [&](std::vector<Chunk>& out, std::vector<int64_t>& bytes, int leaf, int kind, int64_t src,
                   const std::vector<int32_t>& idx, int cbase, int ncols, int ld, int elem) {
        const int per = std::max(1, std::min(H.shape.chunk_cols, H.shape.chunk_bytes / (ld * elem)));
        int c = 0;
        while (c < ncols) {
            int n = 1;
            while (c + n < ncols && n < per && idx[cbase + c + n] == idx[cbase + c] + n) ++n;
            Chunk ch;
            ch.src = src + (int64_t)c * ld;
            ch.zoff = idx[cbase + c];
            ch.leaf = leaf;
            ch.ncols = n;
            ch.kind = kind;
            ch.ld = ld;
            out.push_back(ch);
            bytes.push_back((int64_t)n * ld * elem);
            c += n;
        }
    };
    auto split_ranges = [&](const std::vector<int64_t>& bytes, std::vector<int32_t>& cta) {
        int64_t tot = 0;
        for (int64_t b : bytes) tot += b;
        cta.assign(G + 1, (int32_t)bytes.size());
        int64_t acc = 0;
        int w = 0;
        cta[0] = 0;
        for (size_t i = 0; i < bytes.size(); ++i) {
            // chunk i goes to the CTA whose share contains its first byte
            while (w + 1 <= G && acc >= (tot * (int64_t)(w + 1)) / G) {
                ++w;
                cta[w] = (int32_t)i;
            }
            acc += bytes[i];
        }
        for (int q = w + 1; q <= G; ++q) cta[q] = (int32_t)bytes.size();
        // A chunk larger than a share would leave the CTAs whose shares it covers without
        // a chunk; such an empty CTA inside a row leaf split over several CTAs would be
        // counted as a part of it and never arrive.  So every CTA gets at least one chunk
        // (with fewer chunks than CTAs, one each and the empty CTAs last).
        const int32_t n = (int32_t)bytes.size();
        if (n < G) {
            for (int q = 0; q <= G; ++q) cta[q] = std::min(q, n);
        } else {
            for (int q = 1; q < G; ++q) cta[q] = std::max(cta[q], cta[q - 1] + 1);
            for (int q = G - 1; q >= 1; --q) cta[q] = std::min(cta[q], cta[q + 1] - 1);
        }
    };

    std::vector<Chunk> c1, c2;
    std::vector<int64_t> b1, b2;
    const int nl = H.n_leaves;
    for (int l = 0; l < nl; ++l) {
        const LeafDesc& L = H.h_leaves[l];
        cut(c2, b2, l, 0, L.near_off, H.h_near_zidx, L.near_cbase, L.near_cols, L.ld, 4);
        // the BF16 streams have their own offsets and padding (bf16_ld)
        const bool b16 = esz == 2;
        cut(c2, b2, l, 1, b16 ? L.u_off16 : L.u_off, H.h_u_zidx, L.u_cbase, L.u_cols, b16 ? L.ld16 : L.ld, esz);
        cut(c1, b1, l, 2, b16 ? L.v_off16 : L.v_off, H.h_v_pidx, L.v_cbase, L.v_cols, b16 ? L.ld16 : L.ld, esz);
    }
    std::vector<int32_t> cta1, cta2;
    split_ranges(b1, cta1);
    split_ranges(b2, cta2);
    // split row leaves
    std::vector<LeafSplit> sp(nl, LeafSplit{0, 0, 0, 0});
    std::vector<int> first(nl, -1), last(nl, -1);
    for (int w = 0; w < G; ++w)
        for (int i = cta2[w]; i < cta2[w + 1]; ++i) {
            const int l = c2[i].leaf;
            if (first[l] < 0) first[l] = w;
            last[l] = w;
        }
    int slots = 0;
    for (int l = 0; l < nl; ++l) {
        if (first[l] < 0) fail(HM_EINVAL, "product plan: a leaf has no columns");
        sp[l].w_first = first[l];
        sp[l].nparts = last[l] - first[l] + 1;
        sp[l].slot_base = sp[l].nparts > 1 ? slots : 0;
        if (sp[l].nparts > 1) slots += sp[l].nparts;
    }
    PLAN.n_slots = slots;
    PLAN.ch1.upload(c1, st);
    PLAN.ch2.upload(c2, st);
    PLAN.cta1.upload(cta1, st);
    PLAN.cta2.upload(cta2, st);
    PLAN.split.upload(sp, st);
    PLAN.ready = true;
}

void ensure_product_scratch(HMat& H, int nrhs, cudaStream_t st) {
    if (nrhs <= H.nrhs_cap) return;
    graphs_clear(H);  // captured products refer to the scratch being replaced
    const int cap = nrhs <= 1 ? 1 : (nrhs <= 4 ? 4 : 16);
    const size_t nv = (size_t)H.ndof * cap + VEC_SLACK;
    const size_t np = (size_t)std::max<int64_t>(H.p_len, 1) * cap + VEC_SLACK;
    const size_t nt = (size_t)std::max<int64_t>(H.tb_len, 1) * cap + VEC_SLACK;
    H.xc.alloc(nv);
    H.xcf.alloc(nv);
    H.P.alloc(np);
    H.tb.alloc(nt);
    H.Pf.alloc(np);
    H.tbf.alloc(nt);
    // the slack read by rounded-up operand copies is never used, but keep it defined
    HM_CUDA(cudaMemsetAsync(H.xc.p, 0, H.xc.bytes(), st));
    HM_CUDA(cudaMemsetAsync(H.xcf.p, 0, H.xcf.bytes(), st));
    HM_CUDA(cudaMemsetAsync(H.tb.p, 0, H.tb.bytes(), st));
    HM_CUDA(cudaMemsetAsync(H.tbf.p, 0, H.tbf.bytes(), st));
    int slots = 1;
    for (const HMat::Plan& p : H.plan) slots = std::max(slots, p.n_slots);
    const size_t sl = (size_t)slots * 16 * std::max(H.ld_max, 1);
    H.slotsf.alloc(sl);
    H.slotsd.alloc(sl);
    H.nrhs_cap = cap;
}

int product_group(const HMat& H, int nr, int dtype) {
    return dtype == HM_F64 ? f64_passes(H, nr).nrhs : std::min(nr, 16);
}

void product_split(HMat& H, const double* z, double* zs, int nr, cudaStream_t st) {
    const F64Passes ps = f64_passes(H, nr);
    k_gather_split<<<dim3((unsigned)ceil_div(H.ndof * ps.width, 256), ps.count), 256, 0, st>>>(
        z, (float2*)zs, nullptr, H.N, nr, ps.width, f64_pass_stride(H.ndof, ps.width));
    HM_LAUNCH_CHECK();
}

void product_core(HMat& H, const void* xc, void* yc, int nr, int dtype, int fac, cudaStream_t st, const int* skip) {
    if (nr < 1 || nr > product_group(H, nr, dtype)) fail(HM_EINVAL, "product: too many right-hand sides at once");
    ensure_product_scratch(H, nr, st);
    if (dtype == HM_F32 && padded_rhs(nr) != nr) {
        const int np = padded_rhs(nr);
        k_pad<<<(unsigned)ceil_div(H.ndof * np, 256), 256, 0, st>>>((const float*)xc, H.xcf.p, H.ndof, nr, np);
        HM_LAUNCH_CHECK();
        xc = H.xcf.p;
    }
    run_core(H, xc, yc, nr, dtype, fac, false, st, skip);
}

void matvec(HMat& H, const void* x, void* y, int nrhs, int dtype, cudaStream_t st, int factors) {
    if (nrhs < 1) fail(HM_EINVAL, "matvec: nrhs must be >= 1");
    if (!x || !y) fail(HM_EINVAL, "matvec: NULL vector");
    if (dtype != HM_F32 && dtype != HM_F64) fail(HM_EINVAL, "matvec: dtype must be HM_F32 or HM_F64");
    if (factors != 0 && factors != HM_F32 && factors != HM_BF16)
        fail(HM_EINVAL, "matvec: factors must be 0, HM_F32 or HM_BF16");
    // FP32 factors when stored, unless the caller asks for a stored precision
    const int fac = factors == HM_BF16 ? 1 : (factors == HM_F32 ? 0 : (has_factors(H, 0) ? 0 : 1));
    if (!has_factors(H, fac)) fail(HM_EINVAL, "matvec: the requested factor precision is not stored");
    ensure_product_scratch(H, std::min(nrhs, 16), st);
    for (int k0 = 0, nr = 0; k0 < nrhs; k0 += nr) {
        // (16 right-hand sides are one group, so the next sixteen start a new one)
        nr = product_group(H, std::min(nrhs - k0, 16 - k0 % 16), dtype);
        if (H.timing && k0 % 16 == 0) ++H.t_count;  // products of up to 16 right-hand sides
        mark(H, 0, st);
        if (dtype == HM_F32) {
            const float* xf = (const float*)x + (int64_t)k0 * H.ndof;
            float* yf = (float*)y + (int64_t)k0 * H.ndof;
            const int np = padded_rhs(nr);
            k_gather<<<(unsigned)ceil_div(H.ndof * np, 256), 256, 0, st>>>(xf, H.xcf.p, H.perm.p, H.N, nr, np);
            mark(H, 1, st);
            run_core(H, H.xcf.p, yf, nr, dtype, fac, true, st, nullptr, H.perm.p);
        } else {
            const double* xd = (const double*)x + (int64_t)k0 * H.ndof;
            double* yd = (double*)y + (int64_t)k0 * H.ndof;
            const F64Passes ps = f64_passes(H, nr);
            k_gather_split<<<dim3((unsigned)ceil_div(H.ndof * ps.width, 256), ps.count), 256, 0, st>>>(
                xd, (float2*)H.xc.p, H.perm.p, H.N, nr, ps.width, f64_pass_stride(H.ndof, ps.width));
            mark(H, 1, st);
            run_core(H, H.xc.p, yd, nr, dtype, fac, true, st, nullptr, H.perm.p);
        }
        HM_LAUNCH_CHECK();
        mark(H, 5, st);
    }
}

void matvec_host(HMat& H, const void* x, void* y, int nrhs, int dtype, cudaStream_t st) {
    if (nrhs < 1) fail(HM_EINVAL, "matvec_host: nrhs must be >= 1");
    if (!x || !y) fail(HM_EINVAL, "matvec_host: NULL vector");
    if (dtype != HM_F32 && dtype != HM_F64) fail(HM_EINVAL, "matvec_host: dtype must be HM_F32 or HM_F64");
    const size_t bytes = (size_t)H.ndof * nrhs * (dtype == HM_F32 ? 4 : 8);
    if (H.xs.n < bytes) {
        H.xs.alloc(bytes);
        H.ys.alloc(bytes);
    }
    HM_CUDA(cudaMemcpyAsync(H.xs.p, x, bytes, cudaMemcpyHostToDevice, st));
    matvec(H, H.xs.p, H.ys.p, nrhs, dtype, st);
    HM_CUDA(cudaMemcpyAsync(y, H.ys.p, bytes, cudaMemcpyDeviceToHost, st));
    HM_CUDA(cudaStreamSynchronize(st));
}

void timing_enable(HMat& H, bool on) {
    if (on) {
        if (H.ev.empty()) {
            H.ev.resize(EV_POOL);
            for (auto& e : H.ev) HM_CUDA(cudaEventCreate(&e));
        }
        for (double& t : H.t_acc) t = 0.0;
        H.t_count = 0;
        H.ev_used = 0;
    } else {
        timing_accumulate(H);
    }
    H.timing = on;
}

void timing_read(HMat& H, double out[6]) {
    timing_accumulate(H);
    for (int i = 0; i < 5; ++i) out[i] = H.t_acc[i];
    out[5] = (double)H.t_count;
}

// Error flags raised by the product kernels since the last check (0 if none); clears them.
int product_error_flags(HMat& H, cudaStream_t st) {
    int e = 0;
    HM_CUDA(cudaMemcpyAsync(&e, H.err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    HM_CUDA(cudaStreamSynchronize(st));
    if (e) {
        HM_CUDA(cudaMemsetAsync(H.err.p, 0, sizeof(int), st));
        // a product that gave up waiting may leave split-leaf arrival counts behind
        HM_CUDA(cudaMemsetAsync(H.counters.p, 0, H.counters.bytes(), st));
        HM_CUDA(cudaStreamSynchronize(st));
    }
    return e;
}

}  // namespace hm
