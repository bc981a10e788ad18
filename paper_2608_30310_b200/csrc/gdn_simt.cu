// fp32 path of the GDN forward: Eq. 1 in blocks of eight tokens with plain FFMA.
//
// Per block with start state S (dv x dk), G_t = product of alpha over the block up to token t, R(t, i) = G_t / G_i (formed as the
// product of the alphas between, so that alpha = 0 is exact):
//     r_t = S k_t,  p_t = S q_t                                                       (state-dependent dot products)
//     y_t = beta_t (v_t - G_t r_t),  M[t][i] = beta_t R(t,i) (k_i . k_t) for i < t,  N[t][i] = R(t,i) (k_i . q_t) for i <= t
//     delta = (I + M)^-1 y,  o_t = G_t p_t + (N (I + M)^-1 y)_t                        (8 x 8 matrices, formed ahead)
//     S = G_8 S + sum_i R(8,i) delta_i k_i^T
// which is 3 dk dv FMAs per token and head; the rows of S are independent of each other.
//
// A CTA owns a slice of 2 RPT NW rows of one chain (request, v-head): NW warps of 2 RPT rows each.  Sixteen lanes share RPT
// rows, DK / 16 columns per lane, all in registers.  The dot products of a token are reduced over the sixteen lanes by a
// reduce-scatter that leaves each lane one of the 2 RPT values (a row's r or p) for all eight tokens, so that the 8 x 8 products run
// inside a lane; eight tokens share the latency (one token at a time, each waited for a shuffle reduction: 400 ns a token).
// Calls with few rows have RPT = 1: eight lanes each have all of a row's r, the other eight its p (see compute_few).  NH helper
// warps run ahead by a stage of 8 NH tokens: they load k, q, g and beta, apply the input stage if asked, and form the 8 x 8
// coefficients.
//
// What bounds it: with RPT = 8 the FMA pipe (240 of its cycles per token and 16 rows, 192 of them the 3 dk dv) and, nearly as
// much, the shared-memory loads: a 16-byte load occupies the SM's load path for four cycles whatever it broadcasts, so a loaded
// k or q value has to serve many rows (8 lanes to 4 rows: 340 cycles a token, bound by the loads; to one row: four times as many).
// Where warps are few, the chain of dependent instructions of a block.
//
// This path serves fp32 io (tolerance 1e-4 rules out tf32/bf16 tensor cores) and every shape the tensor-core path does not cover.
#include "common.cuh"
#include "ptx.cuh"

namespace gdn {
namespace {

using ptx::mul_f32x2;

template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

constexpr int kBlk = 8;            // tokens per block
constexpr int kBufs = 3;           // stages in flight

// coefficients of one block (see the head of the file)
struct __align__(16) Coef {
    float A[2][kBlk][kBlk];               // [0][i][t]  (I + M)^-1 - I;  [1][i][t]  N (I + M)^-1  (zero for i > t)
    float c1[2][kBlk], c2[2][kBlk];       // [0] delta's lanes: beta, -beta G;  [1] the outputs' lanes: 0, G
    float rest[kBlk];                     // R(8, i)
    float gend; float pad[3];             // G_8
};

// what each compute warp keeps of the block: R(8, i) delta_i and v, [token][row];  RPT = 1: v, [row][token]
template <int RPT, int NW> struct __align__(16) Scratch { float dr[NW][kBlk][2 * RPT], v[NW][kBlk][2 * RPT]; };
template <int NW> struct __align__(16) Scratch<1, NW> { float v[NW][2][kBlk]; };

template <int DK, int RPT, int NW, int NH>
struct Smem {
    static constexpr int LD = DK + 4;     // row stride: 16-byte aligned, and eight rows at one column fall into different banks
    float k[kBufs][NH * kBlk][LD], q[kBufs][NH * kBlk][LD];
    Coef coef[kBufs][NH];
    __align__(16) double al[NH][kBlk];                   // helpers: alpha and beta of the block at hand
    float be[NH][kBlk];
    __align__(16) float mn[NH][2][kBlk][kBlk];           // helpers: [0][i][t] -M, [1][i][t] N
    Scratch<RPT, NW> own;
    int4 requests[kSelfSort];                            // the requests, longest first (see sort_requests)
};

// N consecutive values of v as fp32, in one load that stays where it is written (the compiler would sink a prefetch to its first
// use, a block later); zeros where !ok
template <int N> __device__ __forceinline__ void load_early(float (&x)[N], const float* p, bool ok)
{
    uint32_t u[4] = {0u, 0u, 0u, 0u};
    if constexpr (N == 4)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}" : "+r"(u[0]), "+r"(u[1]), "+r"(u[2]), "+r"(u[3]) : "l"(p), "r"((uint32_t)ok));
    else if constexpr (N == 2)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.global.nc.v2.b32 {%0, %1}, [%2];\n\t}" : "+r"(u[0]), "+r"(u[1]) : "l"(p), "r"((uint32_t)ok));
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.global.nc.b32 %0, [%1];\n\t}" : "+r"(u[0]) : "l"(p), "r"((uint32_t)ok));
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = __uint_as_float(u[i]);
}
template <int N> __device__ __forceinline__ void load_early(uint32_t (&u)[(N + 1) / 2], const __nv_bfloat16* p, bool ok)
{
#pragma unroll
    for (int i = 0; i < (N + 1) / 2; ++i) u[i] = 0u;
    if constexpr (N == 4)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p ld.global.nc.v2.b32 {%0, %1}, [%2];\n\t}" : "+r"(u[0]), "+r"(u[1]) : "l"(p), "r"((uint32_t)ok));
    else if constexpr (N == 2)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.global.nc.b32 %0, [%1];\n\t}" : "+r"(u[0]) : "l"(p), "r"((uint32_t)ok));
    else
        asm volatile("{\n\t.reg .pred p;\n\t.reg .b16 h;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.b16 h, 0;\n\t@p ld.global.nc.b16 h, [%1];\n\tmov.b32 %0, {h, 0};\n\t}" : "=r"(u[0]) : "l"(p), "r"((uint32_t)ok));
}
// v of the next block in registers: N values per lane of one token
template <typename T, int N> struct VNext;
template <int N> struct VNext<float, N> {
    float x[N];
    __device__ __forceinline__ void load(const float* p, bool ok) { load_early<N>(x, p, ok); }
    __device__ __forceinline__ float get(int i) const { return x[i]; }
};
template <int N> struct VNext<__nv_bfloat16, N> {
    uint32_t u[(N + 1) / 2];
    __device__ __forceinline__ void load(const __nv_bfloat16* p, bool ok) { load_early<N>(u, p, ok); }
    __device__ __forceinline__ float get(int i) const { return __uint_as_float((i & 1) ? (u[i / 2] & 0xffff0000u) : (u[i / 2] << 16)); }
};

// x += a * (b0, b1), kept in the order written
__device__ __forceinline__ void fma_f32x2_here(float2& x, float2 a, float b0, float b1)
{
    asm volatile("{\n\t.reg .b64 p, q, r;\n\tmov.b64 p, {%0, %1};\n\tmov.b64 q, {%2, %3};\n\tmov.b64 r, {%4, %5};\n\t"
        "fma.rn.f32x2 p, q, r, p;\n\tmov.b64 {%0, %1}, p;\n\t}"
        : "+f"(x.x), "+f"(x.y) : "f"(a.x), "f"(a.y), "f"(b0), "f"(b1));
}

template <int ID> __device__ __forceinline__ void bar_sync(int buf, int n) { asm volatile("bar.sync %0, %1;" ::"r"(ID + buf), "r"(n) : "memory"); }
template <int ID> __device__ __forceinline__ void bar_arrive(int buf, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(ID + buf), "r"(n) : "memory"); }
constexpr int BAR_FULL = 1, BAR_EMPTY = 1 + kBufs;

// n / d and n % d for any n, with m = 0xffffffff / d: the product is at most one short.  (A division takes some 40 instructions, and
// finding an item took ten of them.)
struct Divisor {
    uint32_t d, m;
    __device__ explicit Divisor(uint32_t x) : d(x), m(0xffffffffu / x) {}
    __device__ __forceinline__ uint32_t operator()(uint32_t n, uint32_t& rem) const
    {
        uint32_t q = __umulhi(n, m);
        rem = n - q * d;
        if (rem >= d) { ++q; rem -= d; }
        return q;
    }
};

// Item -> (request, v-head, row slice), longest requests first.  The items are dealt to the SMs in snake order (block b runs on
// SM b modulo their number as long as the GPU is empty): the longest share their SM with the shortest.
struct Item { int n, h, hq, slice, row_begin, row_end; };
template <int SLICES> struct Walk {
    uint32_t sms, pos, r, per, items;                     // SMs and place on them; next row of the deal, rows from item to item of the block
    Divisor heads, group;
    __device__ Walk(const Problem& p, uint32_t n)
        : sms(n), pos(blockIdx.x % n), r(blockIdx.x / n), per((gridDim.x + n - 1) / n), items((uint32_t)p.num_seqs * p.Hv * SLICES),
          heads((uint32_t)p.Hv), group((uint32_t)(p.Hv / p.Hq)) {}
    // the block's next item; false when there is none
    __device__ __forceinline__ bool next(const Problem& p, const Sched& s, const int4* requests, Item& it)
    {
        uint32_t item;
        do {
            if (r * sms >= items) return false;
            item = r * sms + ((r & 1u) ? sms - 1 - pos : pos);
            r += per;
        } while (item >= items);
        it.slice = (int)(item % SLICES);
        uint32_t h, rem;
        const int4 rq = request_at(p, s, requests, heads(item / SLICES, h));
        it.h = (int)h;
        it.hq = (int)group(h, rem);
        it.row_begin = rq.x; it.row_end = rq.y; it.n = rq.z;
        return true;
    }
};

// four values of a 16-byte piece (fp32) or eight (bf16), as fp32
template <typename T> struct Piece { static constexpr int N = 16 / sizeof(T); uint4 u; };
__device__ __forceinline__ void widen(const Piece<float>& x, float (&f)[4])
{
    f[0] = __uint_as_float(x.u.x); f[1] = __uint_as_float(x.u.y); f[2] = __uint_as_float(x.u.z); f[3] = __uint_as_float(x.u.w);
}
__device__ __forceinline__ void widen(const Piece<__nv_bfloat16>& x, float (&f)[8])
{
    const uint32_t w[4] = {x.u.x, x.u.y, x.u.z, x.u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w[i] << 16); f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}

// ---- helper warp: block `hw` of every stage ---------------------------------------------------------------
template <int DK, int SLICES, typename T, int RPT, int NW, int NH>
__device__ void helper(const Problem& p, const Sched& s, Smem<DK, RPT, NW, NH>& sm, Walk<SLICES> walk, int hw, int lane)
{
    constexpr int NTHR = (NW + NH) * 32;
    constexpr int PV = Piece<T>::N, PPR = DK / PV;        // values per 16-byte piece, pieces (lanes) per row
    constexpr int RPL = 32 / PPR, NL = kBlk / RPL;        // rows per warp-wide load, loads per block
    const int prow = lane / PPR, pcol = (lane % PPR) * PV;
    const T* __restrict__ kg = (const T*)p.k;
    const T* __restrict__ qg = (const T*)p.q;
    Piece<T> rk[NL], rq[NL];
    float gb = 0.f;                                       // lanes 0-7: g, lanes 8-15: beta
    auto load = [&](const Item& it, int row0) {
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            const int row = row0 + i * RPL + prow;
            rk[i].u = make_uint4(0u, 0u, 0u, 0u); rq[i].u = make_uint4(0u, 0u, 0u, 0u);
            if (row < it.row_end) {
                const size_t off = ((size_t)row * p.Hq + it.hq) * DK + pcol;
                rk[i].u = *reinterpret_cast<const uint4*>(kg + off);
                rq[i].u = *reinterpret_cast<const uint4*>(qg + off);
            }
        }
        const int row = row0 + (lane & 7);
        gb = 0.f;
        if (lane < 16 && row < it.row_end) gb = (lane < 8 ? p.g : p.beta)[(size_t)row * p.Hv + it.h];
    };

    uint32_t stage = 0;
    Item it;
    while (walk.next(p, s, sm.requests, it)) {
        int row0 = it.row_begin + hw * kBlk;
        if (it.row_begin < it.row_end) load(it, row0);
#pragma unroll 1
        for (int base = it.row_begin; base < it.row_end; base += NH * kBlk, row0 += NH * kBlk, ++stage) {
            const int buf = (int)(stage % kBufs);
            if (stage >= kBufs) bar_sync<BAR_EMPTY>(buf, NTHR);
            if (row0 >= it.row_end) { bar_arrive<BAR_FULL>(buf, NTHR); continue; }     // (nobody reads a block past the end)
            float (*ks)[Smem<DK, RPT, NW, NH>::LD] = &sm.k[buf][hw * kBlk];
            float (*qs)[Smem<DK, RPT, NW, NH>::LD] = &sm.q[buf][hw * kBlk];
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                float fk[PV], fq[PV];
                widen(rk[i], fk); widen(rq[i], fq);
                if (p.input_raw) {
                    // fused input stage: rows L2-normalised, x / sqrt(sum x^2 + eps)
                    float sk = 0.f, sq = 0.f;
#pragma unroll
                    for (int e = 0; e < PV; ++e) { sk = fmaf(fk[e], fk[e], sk); sq = fmaf(fq[e], fq[e], sq); }
#pragma unroll
                    for (int o = PPR / 2; o > 0; o >>= 1) { sk += __shfl_xor_sync(0xffffffffu, sk, o); sq += __shfl_xor_sync(0xffffffffu, sq, o); }
                    const float nk = rsqrtf(sk + kNormEps), nq = rsqrtf(sq + kNormEps);
#pragma unroll
                    for (int e = 0; e < PV; ++e) { fk[e] *= nk; fq[e] *= nq; }
                }
#pragma unroll
                for (int e = 0; e < PV; e += 4) {
                    *reinterpret_cast<float4*>(&ks[i * RPL + prow][pcol + e]) = make_float4(fk[e], fk[e + 1], fk[e + 2], fk[e + 3]);
                    *reinterpret_cast<float4*>(&qs[i * RPL + prow][pcol + e]) = make_float4(fq[e], fq[e + 1], fq[e + 2], fq[e + 3]);
                }
            }
            {
                // Rows past the end: alpha = 1, beta = 0 (k, q are zero).  alpha and its products are formed in fp64 and rounded once
                // where they are used: eight factors rounded to fp32, and their products again, would weigh on the state more than
                // a token-by-token evaluation does, and for equal decays with the same sign in every block (relative error of
                // the state, 256 tokens of g = -0.01: 2.7e-7 token by token, 8.8e-7 with fp32 products, 2.0e-7 so).
                const bool ok = row0 + (lane & 7) < it.row_end;
                const double y = p.input_raw ? 1.0 / (1.0 + exp(-(double)gb)) : exp((double)gb);      // sigmoid of both pre-activations
                if (lane < 8) sm.al[hw][lane] = ok ? y : 1.0;
                else if (lane < 16) sm.be[hw][lane & 7] = p.input_raw ? (ok ? (float)y : 0.f) : gb;
            }
            __syncwarp();
            if (base + NH * kBlk < it.row_end) load(it, row0 + NH * kBlk);
            // Lanes 8 m .. 8 m + 7: the products of k_t and q_t, t = 2 m and 2 m + 1, with all eight k_i, an eighth of the columns
            // per lane; a reduce-scatter leaves each lane four of them: kind (k or q), t, i = 4 b0 .. + 3.
            const int sl = lane & 7, m = lane >> 3;
            float acc[2][2][kBlk];
#pragma unroll
            for (int x = 0; x < 4 * kBlk; ++x) (&acc[0][0][0])[x] = 0.f;
#pragma unroll 1
            for (int c = 4 * sl; c < DK; c += 32) {
                float4 y[2][2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    y[0][b] = *reinterpret_cast<const float4*>(&ks[2 * m + b][c]);
                    y[1][b] = *reinterpret_cast<const float4*>(&qs[2 * m + b][c]);
                }
#pragma unroll
                for (int i = 0; i < kBlk; ++i) {
                    const float4 x = *reinterpret_cast<const float4*>(&ks[i][c]);
#pragma unroll
                    for (int kind = 0; kind < 2; ++kind)
#pragma unroll
                        for (int b = 0; b < 2; ++b) {
                            float& z = acc[kind][b][i];
                            z = fmaf(x.x, y[kind][b].x, z); z = fmaf(x.y, y[kind][b].y, z);
                            z = fmaf(x.z, y[kind][b].z, z); z = fmaf(x.w, y[kind][b].w, z);
                        }
                }
            }
            const bool b2 = (sl & 4) != 0, b1 = (sl & 2) != 0, b0 = (sl & 1) != 0;
            float s2[2][kBlk], s1[kBlk], dot[4];
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int i = 0; i < kBlk; ++i)
                    s2[b][i] = (b2 ? acc[1][b][i] : acc[0][b][i]) + __shfl_xor_sync(0xffffffffu, b2 ? acc[0][b][i] : acc[1][b][i], 4);
#pragma unroll
            for (int i = 0; i < kBlk; ++i) s1[i] = (b1 ? s2[1][i] : s2[0][i]) + __shfl_xor_sync(0xffffffffu, b1 ? s2[0][i] : s2[1][i], 2);
#pragma unroll
            for (int i = 0; i < 4; ++i) dot[i] = (b0 ? s1[4 + i] : s1[i]) + __shfl_xor_sync(0xffffffffu, b0 ? s1[i] : s1[4 + i], 1);
            const int kind = sl >> 2, t = 2 * m + ((sl >> 1) & 1), i0 = 4 * (sl & 1);
            double suf[kBlk];                             // R(t, i): the alphas of the tokens i + 1 .. t (of the last t: to the block's end)
            suf[kBlk - 1] = 1.;
#pragma unroll
            for (int x = kBlk - 1; x > 0; --x) suf[x - 1] = suf[x] * (x <= t ? sm.al[hw][x] : 1.);
            const float bt = sm.be[hw][t], gt = (float)(suf[0] * sm.al[hw][0]);
            Coef& cf = sm.coef[buf][hw];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int ii = i0 + i;
                const float r = (float)(i0 ? suf[4 + i] : suf[i]), rd = r * dot[i];
                sm.mn[hw][kind][ii][t] = kind ? (ii <= t ? rd : 0.f) : (ii < t ? -bt * rd : 0.f);
                if (kind == 0 && t == kBlk - 1) cf.rest[ii] = r;
            }
            if (i0 == 0) { cf.c1[kind][t] = kind ? 0.f : bt; cf.c2[kind][t] = kind ? gt : -bt * gt; }
            if (kind == 0 && i0 == 0 && t == kBlk - 1) cf.gend = gt;
            __syncwarp();
            {
                // lanes j, j + 8, ..: column j of the inverse, by forward substitution, and two rows of N times it
                const int j = lane & 7, t0 = lane >> 3;
                float x[kBlk];
#pragma unroll
                for (int t2 = 0; t2 < kBlk; ++t2) x[t2] = t2 == j ? 1.f : 0.f;
#pragma unroll
                for (int i = 0; i < kBlk; ++i)
#pragma unroll
                    for (int t2 = i + 1; t2 < kBlk; ++t2) x[t2] = fmaf(sm.mn[hw][0][i][t2], x[i], x[t2]);
                float o0 = 0.f, o1 = 0.f;
#pragma unroll
                for (int i = 0; i < kBlk; ++i) {
                    // (up to the token itself: zeros times later tokens' entries would be NaN where those are not finite)
                    if (i < 4 && i <= t0) o0 = fmaf(sm.mn[hw][1][i][t0], x[i], o0);
                    if (i <= t0 + 4) o1 = fmaf(sm.mn[hw][1][i][t0 + 4], x[i], o1);
                }
                cf.A[1][j][t0] = o0; cf.A[1][j][t0 + 4] = o1;
                if (t0 == 0) {
#pragma unroll
                    for (int t2 = 0; t2 < kBlk; ++t2) cf.A[0][j][t2] = t2 == j ? 0.f : x[t2];
                }
            }
            bar_arrive<BAR_FULL>(buf, NTHR);
        }
    }
    for (uint32_t n = stage < kBufs ? 0u : stage - kBufs; n < stage; ++n) bar_sync<BAR_EMPTY>((int)(n % kBufs), NTHR);      // (leave no barrier half arrived)
}

// RPT consecutive state values in global memory (16-byte aligned for RPT >= 4, else 8) <-> x[r] = value row ^ r, in 16-byte pieces,
// or whole 32-byte sectors where the address allows.  Calls of many short requests are bound by the L1 cache, and this is a good
// part of it: one value at a time, a warp's store touched 16 lines for 128 bytes (32,000 chains of 1-8 tokens, d = 64: 593 us that
// way; 465 us in 16-byte pieces; with the divisions and empty blocks out of the way 443 us, and 400 -> 364 us in whole sectors).
template <int RPT, bool STORE>
__device__ __forceinline__ void state_rows(float* g, float (&x)[RPT], int row)
{
    constexpr int W = RPT < 4 ? RPT : 4;
    auto permute = [&]() {
#pragma unroll
        for (int b = 1; b < RPT; b <<= 1) {
            const bool swap = (row & b) != 0;
#pragma unroll
            for (int r = 0; r < RPT; ++r)
                if (!(r & b)) { const float lo = x[r], hi = x[r | b]; x[r] = swap ? hi : lo; x[r | b] = swap ? lo : hi; }
        }
    };
    if (STORE) permute();
    if constexpr (STORE && RPT == 8) {
        if ((reinterpret_cast<uintptr_t>(g) & 31u) == 0) {
            asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(g), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7]) : "memory");
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < RPT; i += W) {
        if constexpr (W == 4) {
            float4* p = reinterpret_cast<float4*>(g + i);
            if (STORE) *p = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
            else { const float4 v = *p; x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w; }
        } else {
            float2* p = reinterpret_cast<float2*>(g + i);
            if (STORE) *p = make_float2(x[i], x[i + 1]);
            else { const float2 v = *p; x[i] = v.x; x[i + 1] = v.y; }
        }
    }
    if (!STORE) permute();
}

// ---- compute warp ---------------------------------------------------------------------------------------------
template <int DK, int DV, typename T, int RPT, int NW, int NH, bool SHORT>
__device__ void compute(const Problem& p, const Sched& s, Smem<DK, RPT, NW, NH>& sm, Walk<DV / (2 * RPT * NW)> walk, int warp, int lane)
{
    constexpr int NTHR = (NW + NH) * 32, R = 2 * RPT * NW, NC = DK / 64;      // NC: 16-byte pieces per lane and row
    constexpr int TB = 16 / RPT;                          // tokens whose dot products are formed together
    const int l = lane & 15, rg = lane >> 4;
    // What the reduce-scatter leaves in this lane: outputs' p (1) or delta's r (0), and which of the RPT rows.  The lane keeps its
    // rows in the order row, row ^ 1, .. and its dot products in the order own type, other type, so that every step of the
    // reduction sends and keeps fixed registers (no selects).
    const int type = l >> 3, row = (l & 7) / (8 / RPT);
    const bool store_o = type == 1 && (l & (8 / RPT - 1)) == 0;
    const int wrow = rg * RPT + row;                      // row within the warp
    const T* __restrict__ vg = (const T*)p.v;
    T* __restrict__ og = (T*)p.out_o;

    uint32_t stage = 0;
    Item it;
    while (walk.next(p, s, sm.requests, it)) {
        const int j0 = it.slice * R + warp * 2 * RPT;     // first row (value index) of the warp
        const size_t st_off = ((size_t)it.n * p.Hv + it.h) * DK * DV + j0 + rg * RPT;
        float2 S[RPT][2 * NC];                            // [row ^ r], piece c: columns 64 c + 4 l .. + 3
        if (p.init_state) {
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float x[RPT];
                    state_rows<RPT, false>(const_cast<float*>(p.init_state) + st_off + (size_t)(64 * c + 4 * l + e) * DV, x, row);
#pragma unroll
                    for (int r = 0; r < RPT; ++r) { if (e & 1) S[r][2 * c + (e >> 1)].y = x[r]; else S[r][2 * c + (e >> 1)].x = x[r]; }
                }
        } else {
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int c = 0; c < 2 * NC; ++c) S[r][c] = make_float2(0.f, 0.f);
        }
        const size_t vstride = (size_t)p.Hv * DV;
        const size_t vo = ((size_t)it.row_begin * p.Hv + it.h) * DV + j0 + wrow;
        T* op = og ? og + vo : nullptr;
        // this lane's part of the next block's v: VPL rows of token lane / 4
        constexpr int VPL = RPT / 2;
        const int vtok = lane >> 2, vrow = VPL * (lane & 3);
        const T* vp = vg + ((size_t)(it.row_begin + vtok) * p.Hv + it.h) * DV + j0 + vrow;
        VNext<T, VPL> vn;
        int left = it.row_end - it.row_begin;             // tokens from the current block on
        vn.load(vp, vtok < left);
#pragma unroll 1
        for (; left > 0; ++stage) {
            const int buf = (int)(stage % kBufs);
            bar_sync<BAR_FULL>(buf, NTHR);
#pragma unroll 1
            for (int sb = 0; sb < NH && left > 0; ++sb, left -= kBlk) {
                const float (*ks)[Smem<DK, RPT, NW, NH>::LD] = &sm.k[buf][sb * kBlk];
                const float (*qs)[Smem<DK, RPT, NW, NH>::LD] = &sm.q[buf][sb * kBlk];
                const Coef& cf = sm.coef[buf][sb];
#pragma unroll
                for (int i = 0; i < VPL; ++i) sm.own.v[warp][vtok][vrow + i] = vn.get(i);
                vp += kBlk * vstride;
                vn.load(vp, vtok < left - kBlk);
                __syncwarp();
                float y[kBlk];
                float Areg[RPT == 2 ? kBlk * kBlk : 1], rreg[RPT == 2 ? kBlk : 1];
                if constexpr (RPT == 2) {
                    // few warps: the coefficients are fetched ahead, so that their latency passes under the dot products
#pragma unroll
                    for (int i = 0; i < kBlk; ++i) {
#pragma unroll
                        for (int t = i; t < kBlk; ++t) Areg[i * kBlk + t] = cf.A[type][i][t];
                        rreg[i] = cf.rest[i];
                    }
#pragma unroll
                    for (int i = 0; i < kBlk; ++i) asm volatile("" ::"f"(Areg[i * kBlk + i]), "f"(Areg[i * kBlk + kBlk - 1]), "f"(rreg[i]));
                }
                const float* const A = RPT == 2 ? Areg : &cf.A[type][0][0];
                const float* const rest = RPT == 2 ? rreg : cf.rest;
                // r_t, p_t of TB tokens at a time: products of all, then the reductions side by side
                const float (*own)[Smem<DK, RPT, NW, NH>::LD] = type ? qs : ks, (*oth)[Smem<DK, RPT, NW, NH>::LD] = type ? ks : qs;
#pragma unroll
                for (int t0 = 0; t0 < kBlk; t0 += TB) {
                    if (SHORT && t0 > 0 && t0 >= left) {               // past the end of the request
#pragma unroll
                        for (int x = 0; x < TB; ++x) y[t0 + x] = 0.f;
                        continue;
                    }
                    float2 a[TB][2][RPT];                 // [token][own type, other type][row]
#pragma unroll
                    for (int x = 0; x < TB; ++x)
#pragma unroll
                        for (int r = 0; r < RPT; ++r) { a[x][0][r] = make_float2(0.f, 0.f); a[x][1][r] = make_float2(0.f, 0.f); }
#pragma unroll
                    for (int c = 0; c < NC; ++c)
#pragma unroll
                        for (int x = 0; x < TB; ++x) {
                            const float4 u = *reinterpret_cast<const float4*>(&own[t0 + x][64 * c + 4 * l]);
                            const float4 w = *reinterpret_cast<const float4*>(&oth[t0 + x][64 * c + 4 * l]);
                            // (one multiplicand stays the same from instruction to instruction: with three new 64-bit operands each, the
                            // register file would feed the pipe every third cycle only)
#pragma unroll
                            for (int r = 0; r < RPT; ++r) fma_f32x2_here(a[x][0][r], S[r][2 * c], u.x, u.y);
#pragma unroll
                            for (int r = 0; r < RPT; ++r) fma_f32x2_here(a[x][1][r], S[r][2 * c], w.x, w.y);
#pragma unroll
                            for (int r = 0; r < RPT; ++r) fma_f32x2_here(a[x][0][r], S[r][2 * c + 1], u.z, u.w);
#pragma unroll
                            for (int r = 0; r < RPT; ++r) fma_f32x2_here(a[x][1][r], S[r][2 * c + 1], w.z, w.w);
                        }
                    float z[TB][RPT];
#pragma unroll
                    for (int r = 0; r < RPT; ++r)
#pragma unroll
                        for (int x = 0; x < TB; ++x)
                            z[x][r] = (a[x][0][r].x + a[x][0][r].y) + __shfl_xor_sync(0xffffffffu, a[x][1][r].x + a[x][1][r].y, 8);
#pragma unroll
                    for (int h = RPT / 2; h > 0; h >>= 1)
#pragma unroll
                        for (int r = 0; r < h; ++r)
#pragma unroll
                            for (int x = 0; x < TB; ++x) z[x][r] += __shfl_xor_sync(0xffffffffu, z[x][r + h], h * (8 / RPT));
#pragma unroll
                    for (int o = 4 / RPT; o > 0; o >>= 1)
#pragma unroll
                        for (int x = 0; x < TB; ++x) z[x][0] += __shfl_xor_sync(0xffffffffu, z[x][0], o);
#pragma unroll
                    for (int x = 0; x < TB; ++x)
                        y[t0 + x] = fmaf(cf.c2[type][t0 + x], z[x][0], cf.c1[type][t0 + x] * sm.own.v[warp][t0 + x][wrow]);
                }
                // delta in the lanes of type 0, the outputs in those of type 1: both from the eight y of the row
                float e[kBlk];
#pragma unroll
                for (int i = 0; i < kBlk; ++i) e[i] = __shfl_sync(0xffffffffu, y[i], lane & ~8);
#pragma unroll
                for (int i = 0; i < kBlk; ++i) {
                    if (SHORT && i >= left) break;
#pragma unroll
                    for (int t = i; t < kBlk; ++t) y[t] = fmaf(A[i * kBlk + t], e[i], y[t]);
                }
                if (l % (8 / RPT) == 0 && type == 0) {
#pragma unroll
                    for (int i = 0; i < kBlk; ++i) sm.own.dr[warp][i][wrow] = y[i] * rest[i];
                }
                __syncwarp();
                if (og) {
                    if (store_o) {
#pragma unroll
                        for (int t = 0; t < kBlk; ++t)
                            if (t < left) op[t * vstride] = from_f32<T>(y[t]);
                    }
                    op += kBlk * vstride;
                }
                // S = G_8 S + sum_i R(8, i) delta_i k_i^T
                const float ge = cf.gend;
#pragma unroll
                for (int r = 0; r < RPT; ++r)
#pragma unroll
                    for (int c = 0; c < 2 * NC; ++c) mul_f32x2(S[r][c].x, S[r][c].y, ge, ge);
#pragma unroll (SHORT ? 2 : 4)
                for (int i = 0; i < (SHORT ? min(left, kBlk) : kBlk); ++i) {
                    float dv[RPT];
#pragma unroll
                    for (int r = 0; r < RPT; ++r) dv[r] = sm.own.dr[warp][i][rg * RPT + (row ^ r)];
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const float4 k4 = *reinterpret_cast<const float4*>(&ks[i][64 * c + 4 * l]);
#pragma unroll
                        for (int r = 0; r < RPT; ++r) fma_f32x2_here(S[r][2 * c], make_float2(dv[r], dv[r]), k4.x, k4.y);
#pragma unroll
                        for (int r = 0; r < RPT; ++r) fma_f32x2_here(S[r][2 * c + 1], make_float2(dv[r], dv[r]), k4.z, k4.w);
                    }
                }
                __syncwarp();                             // the scratch may be overwritten
            }
            bar_arrive<BAR_EMPTY>(buf, NTHR);
        }
        if (p.out_state) {
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    float x[RPT];
#pragma unroll
                    for (int r = 0; r < RPT; ++r) x[r] = (e & 1) ? S[r][2 * c + (e >> 1)].y : S[r][2 * c + (e >> 1)].x;
                    state_rows<RPT, true>(p.out_state + st_off + (size_t)(64 * c + 4 * l + e) * DV, x, row);
                }
        }
    }
}

// ---- compute warp of calls with few rows: one row per sixteen lanes (RPT = 1) -------------------------------------------------
// With a warp to a scheduler nothing but the chain of dependent instructions of a block counts: every lane has all eight r or p of its
// row, delta goes from lane to lane by shuffles, and k serves the products and the update from registers.  us for one request of 512
// tokens and four heads, the mean of five calls that start on an idle GPU: d = 64 50.8 with two rows per sixteen lanes, 34.4 so, 37.3
// with the sums scattered until a lane has one token (half the instructions, but one behind the other), 38.5 so and with k and q
// loaded a block ahead; d = 128: 67.2, 46.3, 47.5, 47.9.  In a long row of calls d = 64 takes 49.8, 33.1, 36.0, 37.5.
template <int DK, int DV, typename T, int NW, int NH>
__device__ void compute_few(const Problem& p, const Sched& s, Smem<DK, 1, NW, NH>& sm, Walk<DV / (2 * NW)> walk, int warp, int lane)
{
    constexpr int NTHR = (NW + NH) * 32, R = 2 * NW, NC = DK / 64;
    const int l = lane & 15, rg = lane >> 4, type = l >> 3;                // type 1: the outputs' lanes, 0: delta's
    const T* __restrict__ vg = (const T*)p.v;
    T* __restrict__ og = (T*)p.out_o;
    float* const vs = &sm.own.v[warp][0][0];              // [row][token]
    uint32_t stage = 0;
    Item it;
    while (walk.next(p, s, sm.requests, it)) {
        const int j0 = it.slice * R + warp * 2;           // first row (value index) of the warp
        const size_t st_off = ((size_t)it.n * p.Hv + it.h) * DK * DV + j0 + rg;
        float2 S[2 * NC];                                 // piece c: columns 64 c + 4 l .. + 3
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float x = p.init_state ? p.init_state[st_off + (size_t)(64 * c + 4 * l + e) * DV] : 0.f;
                if (e & 1) S[2 * c + (e >> 1)].y = x; else S[2 * c + (e >> 1)].x = x;
            }
        const size_t vstride = (size_t)p.Hv * DV;
        // lanes 0-15: v of the next block, token lane / 2, row lane % 2;  lanes 8-15 of either half: a token's output each
        const T* vp = vg + ((size_t)(it.row_begin + (l >> 1)) * p.Hv + it.h) * DV + j0 + (l & 1);
        T* op = og ? og + ((size_t)(it.row_begin + (l & 7)) * p.Hv + it.h) * DV + j0 + rg : nullptr;
        VNext<T, 1> vn;
        int left = it.row_end - it.row_begin;             // tokens from the current block on
        vn.load(vp, rg == 0 && (l >> 1) < left);
#pragma unroll 1
        for (; left > 0; ++stage) {
            const int buf = (int)(stage % kBufs);
            bar_sync<BAR_FULL>(buf, NTHR);
#pragma unroll 1
            for (int sb = 0; sb < NH && left > 0; ++sb, left -= kBlk) {
                const float (*ks)[Smem<DK, 1, NW, NH>::LD] = &sm.k[buf][sb * kBlk];
                const float (*qs)[Smem<DK, 1, NW, NH>::LD] = &sm.q[buf][sb * kBlk];
                const Coef& cf = sm.coef[buf][sb];
                if (rg == 0) vs[(l & 1) * kBlk + (l >> 1)] = vn.get(0);
                vp += kBlk * vstride;
                vn.load(vp, rg == 0 && (l >> 1) < left - kBlk);
                float4 k4[kBlk][NC];
                float ak[kBlk], aq[kBlk];
#pragma unroll
                for (int t = 0; t < kBlk; ++t) {
                    float2 x = make_float2(0.f, 0.f), y = make_float2(0.f, 0.f);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        k4[t][c] = *reinterpret_cast<const float4*>(&ks[t][64 * c + 4 * l]);
                        const float4 q4 = *reinterpret_cast<const float4*>(&qs[t][64 * c + 4 * l]);
                        ptx::fma_f32x2(x.x, x.y, S[2 * c].x, S[2 * c].y, k4[t][c].x, k4[t][c].y);
                        ptx::fma_f32x2(y.x, y.y, S[2 * c].x, S[2 * c].y, q4.x, q4.y);
                        ptx::fma_f32x2(x.x, x.y, S[2 * c + 1].x, S[2 * c + 1].y, k4[t][c].z, k4[t][c].w);
                        ptx::fma_f32x2(y.x, y.y, S[2 * c + 1].x, S[2 * c + 1].y, q4.z, q4.w);
                    }
                    ak[t] = x.x + x.y; aq[t] = y.x + y.y;
                }
                __syncwarp();                             // (v is there)
                float A[kBlk][kBlk], y[kBlk], e[kBlk];
#pragma unroll
                for (int i = 0; i < kBlk; ++i)
#pragma unroll
                    for (int t4 = i & ~3; t4 < kBlk; t4 += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(&cf.A[type][i][t4]);
                        A[i][t4] = x.x; A[i][t4 + 1] = x.y; A[i][t4 + 2] = x.z; A[i][t4 + 3] = x.w;
                    }
#pragma unroll
                for (int t4 = 0; t4 < kBlk; t4 += 4) {
                    const float4 v4 = *reinterpret_cast<const float4*>(&vs[rg * kBlk + t4]), c1 = *reinterpret_cast<const float4*>(&cf.c1[type][t4]);
                    y[t4] = c1.x * v4.x; y[t4 + 1] = c1.y * v4.y; y[t4 + 2] = c1.z * v4.z; y[t4 + 3] = c1.w * v4.w;
                }
                // r in the lanes of type 0, p in those of type 1
                float z[kBlk];
#pragma unroll
                for (int t = 0; t < kBlk; ++t) z[t] = (type ? aq[t] : ak[t]) + __shfl_xor_sync(0xffffffffu, type ? ak[t] : aq[t], 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                    for (int t = 0; t < kBlk; ++t) z[t] += __shfl_xor_sync(0xffffffffu, z[t], o);
#pragma unroll
                for (int t4 = 0; t4 < kBlk; t4 += 4) {
                    const float4 c2 = *reinterpret_cast<const float4*>(&cf.c2[type][t4]);
                    y[t4] = fmaf(c2.x, z[t4], y[t4]); y[t4 + 1] = fmaf(c2.y, z[t4 + 1], y[t4 + 1]);
                    y[t4 + 2] = fmaf(c2.z, z[t4 + 2], y[t4 + 2]); y[t4 + 3] = fmaf(c2.w, z[t4 + 3], y[t4 + 3]);
                }
                // delta in the lanes of type 0, the outputs in those of type 1: both from the eight y of the row
#pragma unroll
                for (int i = 0; i < kBlk; ++i) e[i] = __shfl_sync(0xffffffffu, y[i], lane & ~8);
#pragma unroll
                for (int i = 0; i < kBlk; ++i)
#pragma unroll
                    for (int t = i; t < kBlk; ++t) y[t] = fmaf(A[i][t], e[i], y[t]);
                // S = G_8 S + sum_i R(8, i) delta_i k_i^T
                const float ge = cf.gend;
#pragma unroll
                for (int c = 0; c < 2 * NC; ++c) mul_f32x2(S[c].x, S[c].y, ge, ge);
#pragma unroll
                for (int i = 0; i < kBlk; ++i) {
                    const float d = __shfl_sync(0xffffffffu, y[i] * cf.rest[i], lane & ~8);
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        ptx::fma_f32x2(S[2 * c].x, S[2 * c].y, d, d, k4[i][c].x, k4[i][c].y);
                        ptx::fma_f32x2(S[2 * c + 1].x, S[2 * c + 1].y, d, d, k4[i][c].z, k4[i][c].w);
                    }
                }
                if (og) {
                    // a token's output to each lane of type 1 (all eight have all of them)
                    float x4[4], x2[2];
#pragma unroll
                    for (int i = 0; i < 4; ++i) x4[i] = (l & 4) ? y[i + 4] : y[i];
                    x2[0] = (l & 2) ? x4[2] : x4[0]; x2[1] = (l & 2) ? x4[3] : x4[1];
                    if (type && (l & 7) < left) *op = from_f32<T>((l & 1) ? x2[1] : x2[0]);
                    op += kBlk * vstride;
                }
                __syncwarp();                             // the scratch may be overwritten
            }
            bar_arrive<BAR_EMPTY>(buf, NTHR);
        }
        if (p.out_state) {
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    p.out_state[st_off + (size_t)(64 * c + 4 * l + e) * DV] = (e & 1) ? S[2 * c + (e >> 1)].y : S[2 * c + (e >> 1)].x;
        }
    }
}

template <int DK, int DV, typename T, int RPT, int NW, int NH, bool SHORT>
__global__ void __launch_bounds__((NW + NH) * 32, RPT == 1 ? 1 : 2)
gdn_simt_kernel(const Problem p, const Sched s, const int sms)
{
    extern __shared__ __align__(16) uint8_t raw[];
    Smem<DK, RPT, NW, NH>& sm = *reinterpret_cast<Smem<DK, RPT, NW, NH>*>(raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Walk<DV / (2 * RPT * NW)> walk(p, (uint32_t)sms);       // (divisions: before the wait)
    wait_for_predecessor();
    if (self_sorted(p, s)) {
        sort_requests(p.cu, p.num_seqs, sm.requests, warp, NW + NH, lane);
        __syncthreads();
    }
    if (warp < NW) {
        if constexpr (RPT == 1) compute_few<DK, DV, T, NW, NH>(p, s, sm, walk, warp, lane);
        else compute<DK, DV, T, RPT, NW, NH, SHORT>(p, s, sm, walk, warp, lane);
    } else helper<DK, DV / (2 * RPT * NW), T, RPT, NW, NH>(p, s, sm, walk, warp - NW, lane);
    allow_successor();       // at the end: a successor's blocks placed among this kernel's would land on the SMs in another order
}

template <int DK, int DV, typename T, int RPT, int NW, int NH, bool SHORT = false>
cudaError_t launch_one(const Problem& p, const Sched& s, int dev, int sms, cudaStream_t stream)
{
    constexpr int NTHR = (NW + NH) * 32, SMEM = (int)sizeof(Smem<DK, RPT, NW, NH>);
    static int per_sm[64] = {};                          // resident CTAs per SM; found on the first call per device
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (per_sm[dev] == 0) {
        cudaError_t e = cudaFuncSetAttribute(gdn_simt_kernel<DK, DV, T, RPT, NW, NH, SHORT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
        int n = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, gdn_simt_kernel<DK, DV, T, RPT, NW, NH, SHORT>, NTHR, SMEM);
        if (e != cudaSuccess) return e;
        per_sm[dev] = n > 0 ? n : 1;
    }
    const long long items = (long long)p.num_seqs * p.Hv * (DV / (2 * RPT * NW));
    long long per = (items + sms - 1) / sms;
    if (per > per_sm[dev]) per = per_sm[dev];
    const long long grid = items < sms ? (items > 0 ? items : 1) : per * sms;
    return launch_kernel(gdn_simt_kernel<DK, DV, T, RPT, NW, NH, SHORT>, (unsigned)grid, NTHR, SMEM, stream, 1, p, s, sms);
}

template <int DK, int DV, typename T>
cudaError_t launch_shape(const Problem& p, const Sched& s, cudaStream_t stream)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // Rows per warp: 16 have the lowest cost per row, 8, 4 and 2 the lowest time per token.  The finer splits pay while they find idle
    // SMs (us a call; tests/gpu_utils.py has the same lines).
    // 2 rows a warp up to one CTA per SM, CTAs of 4 rows and then of 8.  512 tokens, 512 / 592 < rows <= 1,184, d = 64: CTAs of 4 rows
    //   34.9 / 65.5-66.3, of 8 rows 43.4 / 43.8-44.2, 4 rows a warp 50.9 / 51.2-51.6; d = 128: 46.7 / 88.6-89.2, 58.3 / 58.7-59.4,
    //   67.6 / 67.7-68.1.  Short calls gain less and lose nothing, 4 rows a warp -> now, 512 and 1,152 rows: one token 3.3 -> 3.1 and
    //   3.4 -> 3.3 at d = 64, 4.5 -> 4.0 and 4.8 -> 4.2 at d = 128; 64 tokens 8.4 -> 6.5, 8.5 -> 7.4, 11.2 -> 8.4, 11.5 -> 9.7.
    // 4 rows (8 per CTA) up to two CTAs per SM, 8 (32 per CTA) up to one and a half.  One request of 1,000 tokens at d = 128 with
    //   4 / 8 / 16 rows a warp: 1,024 rows 128 / 193 / 275, 2,304 rows 175 / 194 / 276, 2,432 rows 300 / 194 / 276, 4,096 rows
    //   347 / 195 / 276, 5,120 to 7,040 rows 474-527 / 310 / 277, 8,192 rows 700 / 310 / 278.  So requests of one length would have
    //   the second line at one CTA per SM, 4,736 rows; it lies higher for ragged ones.  4,737 to 7,104 rows, 8 against 16 rows a
    //   warp: lengths equal or a single request 10-14 % longer; three requests of 60-500 or 250-500 tokens 16 % shorter to 9 %
    //   longer, five to 25 requests 16 % shorter to 2 % longer (d = 128: 113-129 against 135, 25 requests 119 / 135).
    // All this is for a call that has the GPU to itself.  A finer split costs more issue slots per row (every slice has its own
    // helpers), and a CTA with 2 rows a warp fills an SM, so calls on other streams wait once the CTAs outnumber the SMs.  A call of 4
    // heads on each of 2 / 4 / 8 streams, 4 rows a warp -> now: 196 / 201 / 264 -> 129 / 222 / 460 (2,048 tokens, d = 64), 134 / 183 /
    // 313 -> 154 / 302 / 610 (1,024 tokens, d = 128).  With room for two CTAs an SM (four helpers) 133 / 195 / 332 and 149 / 253 / 501,
    // but single calls 2.6 and 12 % longer.  The same requests in one call: 126 / 160 / 254 and 112 / 177 / 198.
    const long long rows = (long long)p.num_seqs * p.Hv * DV;
    // Requests that do not fill a block on average: the instance that leaves out tokens past the end (1,000 requests of 1-8 tokens,
    // 32 heads: 443 -> 365 us at d = 64, 1,565 -> 1,232 us at d = 128; where blocks are full its branches cost 2 %).
    if (rows > 48ll * sms && p.total_tokens <= (int64_t)kBlk * p.num_seqs) return launch_one<DK, DV, T, 8, 4, 2, true>(p, s, dev, sms, stream);
    if (rows > 48ll * sms) return launch_one<DK, DV, T, 8, 4, 2>(p, s, dev, sms, stream);
    if (rows > 16ll * sms) return launch_one<DK, DV, T, 4, 4, 2>(p, s, dev, sms, stream);
    if (rows > 8ll * sms) return launch_one<DK, DV, T, 2, 2, 4>(p, s, dev, sms, stream);
    if (rows > 4ll * sms) return launch_one<DK, DV, T, 1, 4, 4>(p, s, dev, sms, stream);
    return launch_one<DK, DV, T, 1, 2, 6>(p, s, dev, sms, stream);
}

}  // namespace

cudaError_t launch_simt(const Problem& p, const Sched& s, int io_dtype, cudaStream_t stream, int* launches)
{
    cudaError_t e = cudaErrorNotSupported;
#define GDN_SIMT_CASE(DKV, DVV)                                                           \
    if (p.dk == DKV && p.dv == DVV)                                                       \
        e = (io_dtype == GDN_BF16) ? launch_shape<DKV, DVV, __nv_bfloat16>(p, s, stream)  \
                                   : launch_shape<DKV, DVV, float>(p, s, stream);
    GDN_SIMT_CASE(64, 64)
    GDN_SIMT_CASE(64, 128)
    GDN_SIMT_CASE(128, 64)
    GDN_SIMT_CASE(128, 128)
#undef GDN_SIMT_CASE
    if (e == cudaSuccess && launches) *launches += 1;
    return e;
}

}  // namespace gdn
