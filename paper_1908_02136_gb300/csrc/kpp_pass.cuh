// kpp_pass.cuh -- the per-point work of one seeding pass, shared by the
// streamed and persistent forms (Algorithm 2: the per-point loop run in
// parallel over contiguous partitions of the points):
//   - distance of every point of the CTA's row range to the newest centre,
//     d_{m,l} = d(H_m, n_l), in the difference form with FP32 FMAs;
//   - the min-update of the nearest squared distance d_sn (D^2);
//   - the D^2 sum of each warp's contiguous segment of rows, accumulated per
//     lane as FP32 two-sum pairs and reduced across the warp once per pass,
//     and the CTA's sum of its segments.
#pragma once

#include "kpp_device.cuh"

namespace kpp {

// Geometry of one (dtype, d, lanes-per-row) specialisation.
//   WIDE rows (>= 16 bytes): L lanes share a row, each lane reading VPL
//     16-byte vectors of it; a warp covers 32 rows per super-iteration and
//     lane (g, l) ends up owning row base + l * (32 / L) + g.
//   Narrow rows (< 16 bytes): one 16-byte vector holds RPV whole rows; a
//     lane owns RPV consecutive rows and a warp covers 32 * RPV rows.
// Each warp walks a contiguous run of super-iterations (its segment).
template <int DT, int D, int L_>
struct Geom {
    static constexpr int EB = Fmt<DT>::bytes;
    static constexpr int EPV = Fmt<DT>::per16;
    static constexpr int RB = D * EB;
    static constexpr bool WIDE = RB >= 16;
    static constexpr int VPR = WIDE ? RB / 16 : 1;
    static constexpr int L = WIDE ? L_ : 1;
    static constexpr int VPL = WIDE ? VPR / L : 1;
    static constexpr int RPV = WIDE ? 1 : 16 / RB;
    static constexpr int SW = WIDE ? 32 : 32 * RPV; // rows per warp super-iteration
    static constexpr int CREG = WIDE ? VPL * EPV : EPV;
    // slots per batch: 8 vectors per lane per batch (4 for FP8, whose decoded
    // vectors are 4x wider); two batches are in flight with the pipelining
    static constexpr int VB = (DT == KPP_FP8_E4M3) ? 4 : 8;
    static constexpr int JB = WIDE ? ((VB / VPL) < 1 ? 1 : ((VB / VPL) > L ? L : (VB / VPL))) : 1;
    static_assert(!WIDE || (RB % 16 == 0), "wide rows are whole vectors");
    static_assert(!WIDE || (VPR % L == 0 && L >= 1 && L <= 32 && (L & (L - 1)) == 0),
                  "lanes per row must divide the row's vectors");
    static_assert(WIDE || (16 % RB == 0), "narrow rows tile a vector");
    static_assert(!WIDE || (L % JB == 0), "slot batches tile the slots");
    // batches kept in flight by the software pipeline: about 16 vectors per
    // lane whatever the row size (FP8: 8); narrow rows, which also carry
    // RPV prefetched D^2 values per batch, 8 batches at most
    static constexpr int VPB = WIDE ? JB * VPL : 1; // vectors per batch
    static constexpr int PD0 = (2 * VB) / VPB;
    static constexpr int PDW = PD0 < 2 ? 2 : (PD0 > 16 ? 16 : PD0);
    static constexpr int PD = WIDE ? PDW : (RPV <= 2 ? 8 : (RPV == 4 ? 4 : 2));
};

// Any d (D = 0): a lane per row, 32-row groups (GenericPipe below).
template <int DT> struct Geom<DT, 0, 0> {
    static constexpr int EB = Fmt<DT>::bytes;
    static constexpr int EPV = Fmt<DT>::per16;
    static constexpr int RB = 0;
    static constexpr bool WIDE = true;
    static constexpr int L = 0;
    static constexpr int SW = 32;
};

// Packed FP32 pairs for the Blackwell FP32x2 instructions.
using F2 = unsigned long long;

__device__ __forceinline__ F2 f2(float lo, float hi)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void f2_split(F2 v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ F2 f2_sub(F2 a, F2 b)
{
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Per-lane slice of the newest centre, decoded to FP32 once per pass.  For
// FP8 each coordinate is the pair (c_hi, c_lo) of split_fp8_centre.
template <int DT, int D, int L_>
struct CentreRegs {
    using G = Geom<DT, D, L_>;
    static constexpr int NLO = (DT == KPP_FP8_E4M3) ? G::CREG : 1;
    float c[G::CREG];
    float clo[NLO];

    __device__ __forceinline__ void set(int k, float s, float raw)
    {
        if constexpr (DT == KPP_FP8_E4M3)
            split_fp8_centre(s, raw, c[k], clo[k]);
        else
            c[k] = raw;
    }

    __device__ __forceinline__ void load(const void *points, const float *scales, int64_t ci)
    {
        const int lane = threadIdx.x & 31;
        const float sc = (DT == KPP_FP8_E4M3) ? __ldg(scales + ci) : 1.0f;
        const char *row = reinterpret_cast<const char *>(points) + ci * (int64_t)G::RB;
        if constexpr (G::WIDE) {
            const int l = lane % G::L;
#pragma unroll
            for (int v = 0; v < G::VPL; ++v) {
                uint4 x = *reinterpret_cast<const uint4 *>(row + (v * G::L + l) * 16);
                float f[G::EPV];
                decode16<DT>(x, f);
#pragma unroll
                for (int e = 0; e < G::EPV; ++e)
                    set(v * G::EPV + e, sc, f[e]);
            }
        } else {
            float tmp[D];
#pragma unroll
            for (int k = 0; k < D; ++k)
                tmp[k] = decode1<DT>(points, ci * D + k);
#pragma unroll
            for (int e = 0; e < G::EPV; ++e)
                set(e, sc, tmp[e % D]);
        }
    }

    // Adds sum_e (x_e - c_{k0+e})^2 of one decoded vector into (a0, a1):
    // even elements into a0, odd into a1, with packed FP32x2 instructions
    // (each lane of a packed op rounds exactly like the scalar op).
    // `s` is the row scale (FP8 only).
    template <int N>
    __device__ __forceinline__ void accum(const float *f, int k0, float s, float &a0,
                                          float &a1) const
    {
        F2 acc = f2(a0, a1);
#pragma unroll
        for (int e = 0; e < N; e += 2) {
            F2 t;
            if constexpr (DT == KPP_FP8_E4M3) {
                const F2 x = f2_fma(f2(s, s), f2(f[e], f[e + 1]),
                                    f2(-c[k0 + e], -c[k0 + e + 1]));
                t = f2_sub(x, f2(clo[k0 + e], clo[k0 + e + 1]));
            } else {
                t = f2_sub(f2(f[e], f[e + 1]), f2(c[k0 + e], c[k0 + e + 1]));
            }
            acc = f2_fma(t, t, acc);
        }
        f2_split(acc, a0, a1);
    }
};

// Where D^2 lives during a pass.
enum D2Mode {
    D2_INPLACE = 0, // the global D^2 array, read and written in place
    D2_SMEM = 1     // shared memory (copied out to the global array when asked)
};

struct PassIO {
    int64_t r0, r1;        // this CTA's rows
    bool first;            // pass 0: D^2 starts at +infinity
    bool reverse;          // walk each segment last super-iteration first
    const char *gpts;      // points in global memory
    const float *scales;   // FP8 row scales
    char *cache;           // shared-memory copy of the first `cache_supers`
    int64_t cache_supers;  //   super-iterations of every warp's segment, or null
    bool fill_cache;       // this pass loads the cached rows and stores them
    float *d2;             // D2_INPLACE: the global D^2 array
    float *d2_out;         // D2_SMEM: also store this pass's D^2 here, or null
    float *d2s;            // D2_SMEM: shared memory, indexed by row - r0
    float2 *segs;          // segment sums of this CTA, one per warp (global or smem)
    uint64_t policy;       // L2 cache policy of global point loads (0: none)
    Control *ctl;          // status block (debug build: index checks report here)
    uint16_t *lab;         // nearest centre of every row, indexed by row - r0 (shared
                           //   memory for D2_SMEM, else global), or null
    uint16_t lab_new;      // the label of this pass's centre
    int d;                 // any-d passes: features, and the bytes of all points
    int64_t bytes;
};

__device__ __forceinline__ uint4 ld_global_hint(const void *ptr, uint64_t policy)
{
    uint4 v;
    asm volatile(
        "ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
        : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
        : "l"(ptr), "l"(policy));
    return v;
}

__device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// 16-byte shared-memory accesses by explicit shared-window address (the
// cache pointer is chosen at run time between shared and global memory, so
// the compiler could not prove the address space by itself).
__device__ __forceinline__ uint4 lds16(const void *p)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a));
    return v;
}

__device__ __forceinline__ void sts16(void *p, uint4 v)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y),
                 "r"(v.z), "r"(v.w)
                 : "memory");
}

// One 16-byte vector of row data: from the shared-memory cache slot of the
// super-iteration (if cached and not being filled), else from global memory.
__device__ __forceinline__ uint4 load_vec(const PassIO &io, const char *cslot, int64_t rb,
                                          int64_t row, int byte_in_row, int RB)
{
    // the 16 bytes read lie within this CTA's rows (a narrow-row vector
    // covers several whole rows)
    if (!kpp_check(io.ctl,
                   row * RB + byte_in_row >= io.r0 * RB &&
                       row * RB + byte_in_row + 16 <= io.r1 * RB,
                   101))
        return make_uint4(0, 0, 0, 0);
    if (cslot)
        return lds16(cslot + (row - rb) * RB + byte_in_row);
    const char *g = io.gpts + row * RB + byte_in_row;
    return io.policy ? ld_global_hint(g, io.policy) : ld_stream16(g);
}

// The previous D^2 of an owned row, for D2_INPLACE prefetched together with
// the row's points (an L2 round trip that would otherwise stall the warp once
// per super-iteration); unused in pass 0 and for D2_SMEM.
template <int MODE>
__device__ __forceinline__ float prefetch_d2(const PassIO &io, int64_t row, bool in_range)
{
    if (MODE != D2_INPLACE || io.first || !in_range)
        return 0.f;
    if (!kpp_check(io.ctl, row >= io.r0 && row < io.r1, 102))
        return 0.f;
    return __ldcg(io.d2 + row);
}

// min-update of one owned row; returns the row's new D^2.  `pre` is the
// prefetched previous D^2 (D2_INPLACE).
template <int MODE>
__device__ __forceinline__ float update_d2(const PassIO &io, int64_t row, float v, float pre)
{
    if (!kpp_check(io.ctl, row >= io.r0 && row < io.r1, 103))
        return 0.f;
    float *slot = (MODE == D2_INPLACE) ? io.d2 + row : io.d2s + (row - io.r0);
    if (io.first) {
        *slot = v;
    } else {
        const float old = (MODE == D2_INPLACE) ? pre : *slot;
        if (v < old)
            *slot = v;
        else
            v = old;
    }
    if (MODE == D2_SMEM && io.d2_out)
        io.d2_out[row] = v;
    return v;
}

// Squared distances of the rows of one batch (slots [jb, jb + JB) of a
// 32-row group): each lane sums its slice of the rows, then the L lanes
// sharing a row add up.  Lane l of a row group ends with slot l's sum in
// `mine` once the batch holding that slot has been through.
template <int DT, int D, int L_>
__device__ __forceinline__ void batch_d2(const uint4 (&x)[Geom<DT, D, L_>::JB][Geom<DT, D, L_>::VPL],
                                         const float (&sc)[Geom<DT, D, L_>::JB],
                                         const CentreRegs<DT, D, L_> &cr, int jb, float &mine)
{
    using G = Geom<DT, D, L_>;
    const int l = (threadIdx.x & 31) % G::L;
    float part[G::JB];
#pragma unroll
    for (int q = 0; q < G::JB; ++q) {
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int v = 0; v < G::VPL; ++v) {
            float f[G::EPV];
            decode16<DT>(x[q][v], f);
            cr.template accum<G::EPV>(f, v * G::EPV, sc[q], a0, a1);
        }
        part[q] = a0 + a1;
    }
    if constexpr (G::JB == G::L) {
        // every slot of the row group is in this batch: reduce-scatter
        // over the L lanes sharing the rows -- halving the live slots
        // at each step, each lane keeping the half its bit selects --
        // leaves slot l's sum on lane l.  Each lane adds the same
        // partials in the same pairs as the butterfly below, so the
        // sums are bit-identical to it, with log2(L) shuffle rounds
        // for all L rows instead of log2(L) per row.
#pragma unroll
        for (int o = G::L / 2, n = G::JB; o > 0; o >>= 1, n >>= 1) {
            const bool up = (l & o) != 0;
#pragma unroll
            for (int i = 0; i < n / 2; ++i) {
                const float send = up ? part[i] : part[i + n / 2];
                const float keep = up ? part[i + n / 2] : part[i];
                part[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        mine = part[0];
    } else {
#pragma unroll
        for (int q = 0; q < G::JB; ++q) {
            float sum = part[q];
#pragma unroll
            for (int o = G::L / 2; o > 0; o >>= 1)
                sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (l == jb + q)
                mine = sum;
        }
    }
}

// One pass over rows [r0, r1) by all warps of the CTA, each over its own
// segment.  Loads are software-pipelined: the vectors of the next batch of
// rows are requested before the current batch is computed, so every warp
// keeps memory requests in flight continuously.  Writes the warp's segment
// sum and returns it (identical on all lanes of the warp).
template <int DT, int D, int L_, int MODE>
__device__ __forceinline__ Pair pass_rows(const PassIO &io, const CentreRegs<DT, D, L_> &cr)
{
    using G = Geom<DT, D, L_>;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    int64_t seg_first, seg_last;
    segment_rows(io.r0, io.r1 - io.r0, G::SW, nwarps, warp, &seg_first, &seg_last);
    const int64_t nsup = (seg_last - seg_first + G::SW - 1) / G::SW;
    Pair lacc{};

    // super-iteration j of this warp: first row and shared-memory cache slot
    auto super_at = [&](int64_t j, int64_t &rb, char *&slot) {
        const int64_t jj = io.reverse ? (nsup - 1 - j) : j;
        rb = seg_first + jj * G::SW;
        slot = (io.cache != nullptr && jj < io.cache_supers)
                   ? io.cache + ((int64_t)warp * io.cache_supers + jj) * G::SW * G::RB
                   : nullptr;
    };

    if constexpr (G::WIDE) {
        // batch bi = slots [jb, jb + JB) of super-iteration bi / NB
        constexpr int NB = G::L / G::JB;
        const int g = lane / G::L, l = lane % G::L;
        const int64_t nbatch = nsup * NB;
        using Vecs = uint4[G::JB][G::VPL];
        using Scales = float[G::JB];
        auto issue = [&](int64_t bi, Vecs &x, Scales &sc, float &pre) {
            int64_t rb;
            char *slot;
            super_at(bi / NB, rb, slot);
            const int jb = (int)(bi % NB) * G::JB;
            const char *from = io.fill_cache ? nullptr : slot;
            const int64_t row0 = rb + (int64_t)jb * (32 / G::L) + g; // row of slot jb
            constexpr int QB = (32 / G::L) * G::RB;                   // bytes between slots
            pre = 0.f;
            if (jb + G::JB == G::L) { // last batch: the own row's previous D^2
                const int64_t own_row = rb + (int64_t)l * (32 / G::L) + g;
                pre = prefetch_d2<MODE>(io, own_row, own_row < seg_last);
            }
            if (rb + G::SW <= seg_last &&
                kpp_check(io.ctl,
                          row0 >= io.r0 && row0 + (int64_t)(G::JB - 1) * (32 / G::L) < io.r1, 104)) {
                // whole super-iteration in range: no bounds checks, one base
                // address and immediate offsets
                if (from) {
                    const char *p0 = from + (row0 - rb) * G::RB + l * 16;
#pragma unroll
                    for (int q = 0; q < G::JB; ++q)
#pragma unroll
                        for (int v = 0; v < G::VPL; ++v)
                            x[q][v] = lds16(p0 + q * QB + v * G::L * 16);
                } else {
                    const char *p0 = io.gpts + row0 * G::RB + l * 16;
#pragma unroll
                    for (int q = 0; q < G::JB; ++q)
#pragma unroll
                        for (int v = 0; v < G::VPL; ++v)
                            x[q][v] = io.policy ? ld_global_hint(p0 + q * QB + v * G::L * 16, io.policy)
                                                : ld_stream16(p0 + q * QB + v * G::L * 16);
                }
#pragma unroll
                for (int q = 0; q < G::JB; ++q)
                    sc[q] = (DT == KPP_FP8_E4M3) ? __ldg(io.scales + row0 + q * (32 / G::L)) : 1.0f;
                return;
            }
            if (rb + G::SW <= seg_last) { // only after a failed debug check
#pragma unroll
                for (int q = 0; q < G::JB; ++q) {
                    sc[q] = 1.0f;
#pragma unroll
                    for (int v = 0; v < G::VPL; ++v)
                        x[q][v] = make_uint4(0, 0, 0, 0);
                }
                return;
            }
#pragma unroll
            for (int q = 0; q < G::JB; ++q) {
                const int64_t row = row0 + (int64_t)q * (32 / G::L);
                const bool ok = row < seg_last;
                sc[q] = (DT == KPP_FP8_E4M3 && ok) ? __ldg(io.scales + row) : 1.0f;
#pragma unroll
                for (int v = 0; v < G::VPL; ++v)
                    x[q][v] = ok ? load_vec(io, from, rb, row, (v * G::L + l) * 16, G::RB)
                                 : make_uint4(0, 0, 0, 0);
            }
        };
        float mine = 0.f;
        auto consume = [&](int64_t bi, const Vecs &x, const Scales &sc, float pre) {
            int64_t rb;
            char *slot;
            super_at(bi / NB, rb, slot);
            const int jb = (int)(bi % NB) * G::JB;
            if (io.fill_cache && slot) {
#pragma unroll
                for (int q = 0; q < G::JB; ++q) {
                    const int64_t row = rb + (int64_t)(jb + q) * (32 / G::L) + g;
                    if (row < seg_last) {
#pragma unroll
                        for (int v = 0; v < G::VPL; ++v)
                            sts16(slot + (row - rb) * G::RB + (v * G::L + l) * 16, x[q][v]);
                    }
                }
            }
            batch_d2<DT, D, L_>(x, sc, cr, jb, mine);
            if (jb + G::JB == G::L) { // last batch of the super-iteration
                const int64_t own_row = rb + (int64_t)l * (32 / G::L) + g;
                if (own_row < seg_last)
                    lacc.add(update_d2<MODE>(io, own_row, mine, pre));
            }
        };
        // ring of PD batches: batch bi + PD - 1 is requested before batch bi
        // is computed
        constexpr int P = G::PD;
        Vecs x[P];
        Scales sc[P];
        float pre[P];
#pragma unroll
        for (int q = 0; q < P - 1; ++q)
            if (q < nbatch)
                issue(q, x[q], sc[q], pre[q]);
        for (int64_t bi = 0; bi < nbatch; bi += P) {
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int qn = (q + P - 1) % P;
                if (bi + q + P - 1 < nbatch)
                    issue(bi + q + P - 1, x[qn], sc[qn], pre[qn]);
                if (bi + q < nbatch)
                    consume(bi + q, x[q], sc[q], pre[q]);
            }
        }
    } else {
        // narrow rows: one 16-byte vector (RPV rows) per lane and super-iteration
        using Pre = float[G::RPV];
        auto issue = [&](int64_t j, uint4 &x, Pre &pre) {
            int64_t rb;
            char *slot;
            super_at(j, rb, slot);
            const int64_t own = rb + (int64_t)lane * G::RPV;
            x = (own + G::RPV <= seg_last)
                    ? load_vec(io, io.fill_cache ? nullptr : slot, rb, own, 0, G::RB)
                    : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int r = 0; r < G::RPV; ++r)
                pre[r] = prefetch_d2<MODE>(io, own + r, own + r < seg_last);
        };
        auto consume = [&](int64_t j, const uint4 &x, const Pre &pre) {
            int64_t rb;
            char *slot;
            super_at(j, rb, slot);
            const int64_t own_row = rb + (int64_t)lane * G::RPV;
            float f[G::EPV];
            float sc[G::RPV];
            if (own_row + G::RPV <= seg_last) {
                if (io.fill_cache && slot)
                    sts16(slot + (own_row - rb) * G::RB, x);
                decode16<DT>(x, f);
#pragma unroll
                for (int r = 0; r < G::RPV; ++r)
                    sc[r] = (DT == KPP_FP8_E4M3) ? __ldg(io.scales + own_row + r) : 1.0f;
            } else {
                // ragged tail of the segment: element loads from global memory,
                // never past its end (these rows are never cached)
#pragma unroll
                for (int r = 0; r < G::RPV; ++r) {
                    const int64_t row = own_row + r;
                    const bool ok = row < seg_last && kpp_check(io.ctl, row >= io.r0 && row < io.r1, 105);
                    sc[r] = (DT == KPP_FP8_E4M3 && ok) ? __ldg(io.scales + row) : 1.0f;
#pragma unroll
                    for (int k = 0; k < D; ++k)
                        f[r * D + k] = ok ? decode1<DT>(io.gpts, row * D + k) : 0.f;
                }
            }
#pragma unroll
            for (int r = 0; r < G::RPV; ++r) {
                float a0 = 0.f, a1 = 0.f;
                cr.template accum<D>(f + r * D, r * D, sc[r], a0, a1);
                const int64_t row = own_row + r;
                if (row < seg_last)
                    lacc.add(update_d2<MODE>(io, row, a0 + a1, pre[r]));
            }
        };
        constexpr int P = G::PD;
        uint4 x[P];
        Pre pre[P];
#pragma unroll
        for (int q = 0; q < P - 1; ++q)
            if (q < nsup)
                issue(q, x[q], pre[q]);
        for (int64_t j = 0; j < nsup; j += P) {
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int qn = (q + P - 1) % P;
                if (j + q + P - 1 < nsup)
                    issue(j + q + P - 1, x[qn], pre[qn]);
                if (j + q < nsup)
                    consume(j + q, x[q], pre[q]);
            }
        }
    }
    const Pair seg = warp_pair_sum(lacc);
    if (lane == 0)
        io.segs[warp] = make_float2(seg.hi, seg.lo);
    return seg;
}

// ---------------------------------------------------------------------------
// Passes that read only the rows whose D^2 can still fall.
//
// Every row carries the label of its nearest chosen centre a.  For the new
// centre c the triangle inequality gives |x - c| >= |c - a| - |x - a|, so a
// row with 4 D^2 <= |c - a|^2 cannot come nearer (Elkan, "Using the triangle
// inequality to accelerate k-means", ICML 2003; for the seeding, Raff, "Exact
// acceleration of k-means++ and k-means||", IJCAI 2021).  The minimum keeps
// its old value there, so leaving the row unread changes no bit of D^2.  The
// computed squares carry a relative rounding of at most (d + 1) 2^-24 each
// (d <= 4096: 2.5e-4); the test keeps a margin of 2^-8, several times their
// sum.  Squares near the ends of the FP32 range (and NaN) skip nothing, or
// only rows at D^2 = 0.
//
// The plain pass over a large set is bound by HBM, so the rows left out are
// time saved: on mixtures with as many components as seeds a pass has to
// read 34 % of the rows on average (99 % at the first seeds, under 1 % at the
// last).  Whole seedings before and after: 10^7 x 64, K = 1024 FP32 381 -> 152
// ms, BF16 225 -> 92 ms; 2 10^7 x 128, K = 2048 FP8 1337 -> 506 ms; 10^6 x 32,
// K = 256 (in L2) 3.90 -> 3.00 ms; the 512-problem batch 40.6 -> 22.7 ms.
// What data without clusters pays, where no row is ever skipped (normal
// coordinates, ms with every row read / so): far beyond L2 nothing (10^7 x 64,
// K = 64 24.6 / 24.5), narrow and FP8 rows gain from the row pipe (10^7 x 16 8.8 / 6.9,
// 10^6 x 128 FP8, K = 100 3.39 / 3.06), sets in L2 gain a little (10^6 x 32, K = 256
// 3.91 / 3.78; 2 10^5 x 32 1.84 / 1.85).  Where the lists push D^2 out of shared
// memory (1.6 to 8 10^6 points) rows of 128 bytes and more lose 1 to 4 % from 20 GB
// of rows in all passes on, where the plain kernel stands by (kpp_persistent.cuh;
// 2 10^6 x 64, K = 128 9.17 / 9.32, 4 10^6 x 32, K = 64 4.69 / 4.87), and up to 10 % in
// shorter seedings, which in clusters gain as much.
// ---------------------------------------------------------------------------
constexpr int kPruneCentres = 2048; // centres with a bound; rows of later ones are always read
constexpr uint16_t kNoLabel = 0xffff;
constexpr int kPruneProbe = 8; // every so many passes look again for rows to skip
constexpr int kHandRowBytes = 128; // rows from which passes that skip none hand over

// Largest D^2 of a row of centre a that centre c at squared distance s2 from
// a cannot lower (negative: none).
__device__ __forceinline__ float prune_bound(float s2)
{
    if (!(s2 < 1e37f))
        return -1.f;
    return s2 < 1e-30f ? 0.f : s2 * (0.25f * (1.f - 0x1.0p-8f));
}

// Largest number of rows read ahead of their arithmetic by a warp, and the
// list of a warp's rows to read: those, one group short of complete and one
// block of tested rows.
constexpr int kPruneBlock = 8; // 32-row groups tested together
constexpr int kPruneAhead = 128;
constexpr int kPruneList = 512;
static_assert(kPruneList >= kPruneAhead + 32 + 32 + 32 * kPruneBlock, "the list holds them");
constexpr int kPruneRing = 8192; // bytes a warp reads ahead

// 16- and 4-byte asynchronous copies from global to shared memory.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int N> __device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The squared distances of a list of rows to the centre, by one warp, with
// the row groups and the arithmetic of pass_rows (bit-identical results).
// The rows in flight sit in a ring in shared memory instead of registers:
// 8 KB a warp, 128 KB an SM, which is what the plain pass keeps in flight (a
// register ring beside the list's state spills).  Every lane copies, waits
// for and reads its own 16-byte vectors, so the ring needs no barrier.  The
// list grows by whole groups of 32 items; n says how many items count, and the
// last group is read with TAIL, which leaves the items past n out (reading some
// row in their place put every CTA's padding on the same sectors of L2).
//   row_at(i, k)     offset in rows from `base` of item i + k (i a multiple of
//                    32 plus the lane's row group, k a constant below 32)
//   ahead(own)       called when the group of the lane's own item is issued
//                    (copies it makes are waited for with the group)
//   pre(own)         what sink wants of the lane's own item, loaded early
//   sink(own, v, p)  called on the lane that owns the item
template <int DT, int D, int L_, class RowAt, class Ahead, class Pre, class Sink> struct RowPipe {
    using G = Geom<DT, D, L_>;
    static_assert(G::WIDE, "rows of at least 16 bytes");
    static constexpr int JB0 = G::VPL >= 4 ? 1 : 4 / G::VPL;
    static constexpr int JB = JB0 < G::L ? JB0 : G::L; // slots per batch
    static constexpr int NB = G::L / JB;               // batches per group
    static constexpr int BR = JB * (32 / G::L);        // rows per batch
    static constexpr int BB = JB * G::VPL * 512;       // bytes per batch
    static constexpr int R0 = kPruneRing / BB < kPruneAhead / BR ? kPruneRing / BB : kPruneAhead / BR;
    static constexpr int R = R0 < 2 ? 2 : R0; // batches in flight
    static_assert(R * BB <= kPruneRing && (R & (R - 1)) == 0, "the ring holds them");

    const CentreRegs<DT, D, L_> &cr;
    Control *ctl;         // debug build: index checks
    int64_t base, nrows;  //   rows base + row_at() below nrows
    const char *src0;     // this lane's first vector of row 0 of the list's base
    const float *scales0; // its FP8 scale
    uint32_t ring, sring; // this lane's first vector; the FP8 scales of the rows in flight
    RowAt row_at;
    Ahead ahead;
    Pre pre;
    Sink sink;
    int n = 0;        // items of the list so far
    int groups = 0;   // issued
    uint32_t it = 0;  // batches issued
    int done = 0;     // groups consumed
    float part[G::L]; // this lane's share of each slot's row

    __device__ __forceinline__ RowPipe(const PassIO &io, int64_t base_,
                                       const CentreRegs<DT, D, L_> &cr_, char *ring_, RowAt r,
                                       Ahead a, Pre p, Sink s)
        : cr(cr_), ctl(io.ctl), base(base_), nrows(io.bytes / G::RB), row_at(r), ahead(a), pre(p),
          sink(s)
    {
        const int lane = threadIdx.x & 31;
        src0 = io.gpts + base * G::RB + (lane % G::L) * 16;
        scales0 = DT == KPP_FP8_E4M3 ? io.scales + base : nullptr;
        const uint32_t r0 = (uint32_t)__cvta_generic_to_shared(ring_);
        ring = r0 + lane * 16;
        sring = r0 + kPruneRing;
    }

    // offsets of the rows of batch jb of the next group
    __device__ __forceinline__ void rows_of(int jb, uint32_t (&row)[JB]) const
    {
        const int g = (threadIdx.x & 31) / G::L;
#pragma unroll
        for (int q = 0; q < JB; ++q)
            row[q] = row_at(groups * 32 + g, (jb * JB + q) * (32 / G::L));
    }

    template <bool TAIL>
    __device__ __forceinline__ void issue(int jb, const uint32_t (&row)[JB])
    {
        const uint32_t slot = it & (R - 1);
        const uint32_t dst = ring + slot * BB;
#pragma unroll
        for (int q = 0; q < JB; ++q) {
            const char *src = src0 + (uint64_t)row[q] * G::RB;
            const int i = groups * 32 + (jb * JB + q) * (32 / G::L) + (int)(threadIdx.x & 31) / G::L;
            if ((!TAIL || i < n) && kpp_check(ctl, base + row[q] < nrows, 112))
#pragma unroll
                for (int v = 0; v < G::VPL; ++v)
                    cp_async16(dst + (q * G::VPL + v) * 512, src + v * G::L * 16);
        }
        if constexpr (DT == KPP_FP8_E4M3) {
            const int lane = threadIdx.x & 31;
            if ((BR == 32 || lane < BR) && (!TAIL || groups * 32 + jb * BR + lane < n) &&
                kpp_check(ctl, base + row_at(groups * 32 + lane, jb * BR) < nrows, 113))
                cp_async4(sring + (slot * BR + lane) * 4,
                          scales0 + row_at(groups * 32 + lane, jb * BR));
        }
        cp_async_commit();
        ++it;
    }

    // the batch issued `back` batches ago
    __device__ __forceinline__ void consume(int jb, uint32_t back)
    {
        const int lane = threadIdx.x & 31, g = lane / G::L, l = lane % G::L;
        if (DT == KPP_FP8_E4M3)
            __syncwarp(); // the scales were copied by other lanes
        const uint32_t slot = (it - back) & (R - 1);
        const uint32_t src = ring + slot * BB;
        const int own = done * 32 + l * (32 / G::L) + g;
        decltype(pre(0)) mine{};
        if (jb == NB - 1)
            mine = pre(own);
        float sum[JB];
#pragma unroll
        for (int q = 0; q < JB; ++q) {
            float s = 1.0f;
            if constexpr (DT == KPP_FP8_E4M3)
                asm volatile("ld.shared.f32 %0, [%1];"
                             : "=f"(s)
                             : "r"(sring + (slot * BR + q * (32 / G::L) + g) * 4));
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int v = 0; v < G::VPL; ++v) {
                uint4 x;
                asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
                             : "r"(src + (q * G::VPL + v) * 512));
                float f[G::EPV];
                decode16<DT>(x, f);
                cr.template accum<G::EPV>(f, v * G::EPV, s, a0, a1);
            }
            sum[q] = a0 + a1;
        }
#pragma unroll
        for (int q = 0; q < JB; ++q)
            part[jb * JB + q] = sum[q];
        if (DT == KPP_FP8_E4M3)
            __syncwarp(); // the scales are read before their slot is filled again
        if (jb == NB - 1) {
            // reduce-scatter as in pass_rows: the same pairs, slot l's sum on lane l
#pragma unroll
            for (int o = G::L / 2, w = G::L; o > 0; o >>= 1, w >>= 1) {
                const bool up = (l & o) != 0;
#pragma unroll
                for (int i = 0; i < w / 2; ++i) {
                    const float send = up ? part[i] : part[i + w / 2];
                    const float keep = up ? part[i + w / 2] : part[i];
                    part[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            }
            if (own < n)
                sink(own, part[0], mine);
            ++done;
        }
    }

    // reads the next group of 32 items (TAIL: those below n); the oldest
    // batches in flight make room
    template <bool TAIL> __device__ __forceinline__ void group()
    {
#pragma unroll
        for (int jb = 0; jb < NB; ++jb) {
            uint32_t row[JB];
            rows_of(jb, row); // before the wait: off the batch's critical path
            if (it >= (uint32_t)R) {
                cp_async_wait<R - 1>();
                consume((jb + NB * R - R) % NB, R);
            }
            if (jb == 0) {
                const int lane = threadIdx.x & 31;
                const int own = groups * 32 + lane % G::L * (32 / G::L) + lane / G::L;
                if (!TAIL || own < n)
                    ahead(own);
            }
            issue<TAIL>(jb, row);
        }
        ++groups;
    }

    // the batches still in flight
    __device__ __forceinline__ void drain()
    {
        cp_async_wait<0>();
        int left = it < (uint32_t)R ? (int)it : R; // the oldest is batch (it - left) % NB of its group
        while (left > 0) {
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (left > 0 && (it - left) % NB == (uint32_t)b) {
                    consume(b, left);
                    --left;
                }
        }
    }

    __device__ __forceinline__ bool full() const { return n - groups * 32 >= 32; }
    __device__ __forceinline__ bool rest() const { return n > groups * 32; }
};

// The row pipe for any d and any row alignment.  A lane owns a row of the
// 32-row group and adds its features in order -- even ones into one sum, odd
// ones into the other, as the streamed any-d pass does, bit for bit.  A row's
// 16-byte chunks (from the 32-byte boundary at or below its first byte) arrive
// four at a time for all 32 rows: a batch is 2 KB, copied as 64-byte pieces of
// eight rows per instruction and read back one chunk of one row per lane.  The
// two halves of a 32-byte sector stay together in shared memory (apart, each
// is a request of its own to L2); pieces are swizzled by row as far as that
// allows.  The streamed pass
// reads single elements a row apart per lane instead: 300 007 x 50, K = 100 32
// us a pass there, 16 here (bound by shared memory: a batch's chunks are written
// and read there, and its centre features once per chunk).
template <int DT, class RowAt, class Ahead, class Pre, class Sink> struct GenericPipe {
    static constexpr int EB = Fmt<DT>::bytes, EPV = Fmt<DT>::per16;
    static constexpr int CH = 4;       // chunks per batch
    static constexpr int BB = 32 * CH * 16;
    static constexpr int R = kPruneRing / BB; // batches in flight
    static_assert(R == 4, "four scale slots follow the ring");

    Control *ctl; // debug build: index checks
    const char *pts;
    const float *scales;
    int64_t base;  // first row of the list's base
    int64_t bytes; // of all points
    const float *cen; // the centre (FP8: high parts, low parts cen_lo floats on), kCentrePad floats of room before and after
    int cen_lo;
    int d, rb, nc, nb; // row bytes; most chunks of a row; batches per group
    int c_in;          // chunks from here on hold no earlier row's elements
    uint32_t ring, sring;
    RowAt row_at;
    Ahead ahead;
    Pre pre;
    Sink sink;
    int n = 0, groups = 0, done = 0; // items, groups issued and consumed
    int ib = 0, cb = 0;              // batches of the current group issued and consumed
    uint32_t it = 0;
    const char *from[4]; // the rows this lane copies: its chunk of the group's first batch,
    int left[4], cut[4]; //   chunks from there on, bytes from there to the points' end
    float a0 = 0.f, a1 = 0.f; // the row being consumed
    int off = 0;              // elements before its first one in its first chunk

    __device__ __forceinline__ GenericPipe(const PassIO &io, int64_t base_, const float *cen_,
                                           int cen_lo_, char *ring_, RowAt r, Ahead a, Pre p,
                                           Sink s)
        : ctl(io.ctl), pts(io.gpts), scales(io.scales), base(base_), bytes(io.bytes), cen(cen_),
          cen_lo(cen_lo_),
          d(io.d), rb(io.d * EB), row_at(r), ahead(a), pre(p), sink(s)
    {
        // a row starts at a multiple of gcd(rb, 16) past a 32-byte boundary
        const int g = (rb & -rb) < 16 ? (rb & -rb) : 16;
        nc = (32 - g + rb + 15) / 16;
        c_in = g == 16 ? 1 : 2;
        nb = (nc + CH - 1) / CH;
        ring = (uint32_t)__cvta_generic_to_shared(ring_);
        sring = ring + kPruneRing;
    }

    // bytes between the 32-byte boundary at or below a row's first byte and it
    __device__ __forceinline__ int lead(int64_t start) const
    {
        return (int)((reinterpret_cast<uintptr_t>(pts) + start) & 31);
    }

    // (a lane's row of the copies and its own row have (lane >> 2) and lane in
    // place of the swizzle's row; both name the same row's bit)
    __device__ __forceinline__ static int swizzle(int j, int row) { return j ^ ((row & 2) ? 2 : 0); }

    template <bool TAIL> __device__ __forceinline__ void issue()
    {
        const int lane = threadIdx.x & 31, j = lane & 3;
        const uint32_t dst = ring + (it & (R - 1)) * BB + (lane >> 2) * (CH * 16) +
                             swizzle(j, lane >> 2) * 16;
        if (ib == 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { // the group's rows this lane copies chunks of
                const int64_t start = (base + row_at(groups * 32 + (lane >> 2), i * 8)) * rb;
                const int ld = lead(start);
                const int64_t at = start - ld + 16 * j;
                from[i] = pts + at;
                // chunks from this one to the row's last (none past n); the
                // last one of all points may be cut short
                left[i] = TAIL && groups * 32 + (lane >> 2) + i * 8 >= n ? 0 : (ld + rb + 15) / 16 - j;
                if (left[i] && !kpp_check(ctl, start >= 0 && start + rb <= bytes, 115))
                    left[i] = 0;
                const int64_t rem = bytes - at;
                cut[i] = (int)(rem < (1 << 20) ? rem : (1 << 20));
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            // (a chunk before the first point: its array need not begin on a
            // 32-byte boundary)
            if (left[i] > ib * CH && from[i] + ib * (16 * CH) >= pts) {
                const int len = cut[i] - ib * (16 * CH);
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                                 dst + i * 8 * (CH * 16)),
                             "l"(from[i] + ib * (16 * CH)), "r"(len < 16 ? len : 16)
                             : "memory");
            }
        if (ib == 0 && (!TAIL || groups * 32 + lane < n))
            ahead(groups * 32 + lane);
        if (DT == KPP_FP8_E4M3 && ib == 0 && (!TAIL || groups * 32 + lane < n) &&
            kpp_check(ctl, (base + row_at(groups * 32 + lane, 0) + 1) * rb <= bytes, 116))
            cp_async4(sring + ((groups & 3) * 32 + lane) * 4,
                      scales + base + row_at(groups * 32 + lane, 0));
        cp_async_commit();
        ++it;
        if (++ib == nb) {
            ib = 0;
            ++groups;
        }
    }

    // one chunk's elements against the centre's ce[0 ..]; EDGE: only those of
    // features [0, d) count, e0 being the first element's; PAIR: ce is 8-byte
    // aligned (d is even)
    template <bool EDGE, bool PAIR>
    __device__ __forceinline__ void chunk(const uint4 &x, const float *ce, int e0, float s, F2 &acc) const
    {
        float f[EPV];
        decode16<DT>(x, f);
#pragma unroll
        for (int w = 0; w < EPV; w += 2) {
            float2 h, l;
            if (PAIR) {
                h = *reinterpret_cast<const float2 *>(ce + w);
                if (DT == KPP_FP8_E4M3)
                    l = *reinterpret_cast<const float2 *>(ce + cen_lo + w);
            } else {
                h = make_float2(ce[w], ce[w + 1]);
                if (DT == KPP_FP8_E4M3)
                    l = make_float2(ce[cen_lo + w], ce[cen_lo + w + 1]);
            }
            F2 t;
            if constexpr (DT == KPP_FP8_E4M3)
                t = f2_sub(f2_fma(f2(s, s), f2(f[w], f[w + 1]), f2(-h.x, -h.y)), f2(l.x, l.y));
            else
                t = f2_sub(f2(f[w], f[w + 1]), f2(h.x, h.y));
            if (EDGE) {
                float t0, t1;
                f2_split(t, t0, t1);
                t = f2((unsigned)(e0 + w) < (unsigned)d ? t0 : 0.f,
                       (unsigned)(e0 + w + 1) < (unsigned)d ? t1 : 0.f);
            }
            acc = f2_fma(t, t, acc);
        }
    }

    // the first `cnt` of the CH chunks of this lane's row at `src`
    template <bool EDGE, bool PAIR>
    __device__ __forceinline__ void chunks(uint32_t src, const float *ceb, int eb, float s, int cnt,
                                           F2 &acc) const
    {
        uint4 x[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j)
            asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(x[j].x), "=r"(x[j].y), "=r"(x[j].z), "=r"(x[j].w)
                         : "r"(src + swizzle(j, threadIdx.x & 31) * 16));
#pragma unroll
        for (int j = 0; j < CH; ++j)
            if (!EDGE || j < cnt)
                chunk<EDGE, PAIR>(x[j], ceb + j * EPV, eb + j * EPV, s, acc);
    }

    // the batch issued `back` batches ago
    __device__ __forceinline__ void consume(uint32_t back)
    {
        const int lane = threadIdx.x & 31;
        __syncwarp(); // other lanes' copies have landed
        const uint32_t src = ring + ((it - back) & (R - 1)) * BB + lane * (CH * 16);
        const int own = done * 32 + lane;
        if (cb == 0) {
            a0 = a1 = 0.f;
            off = lead((base + row_at(own, 0)) * rb) / EB;
        }
        float s = 1.0f;
        if constexpr (DT == KPP_FP8_E4M3)
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(s) : "r"(sring + ((done & 3) * 32 + lane) * 4));
        F2 acc = f2(a0, a1);
        const int eb = cb * CH * EPV - off; // feature of the batch's first element
        const float *ceb = cen + eb;
        // one straight run over the batch's chunks either way, so that their
        // loads overlap
        const int cnt = nc - cb * CH;
        if (cb * CH >= c_in && (cb + 1) * CH * 16 <= rb) {
            if (d & 1)
                chunks<false, false>(src, ceb, eb, s, cnt, acc);
            else
                chunks<false, true>(src, ceb, eb, s, cnt, acc);
        } else {
            if (d & 1)
                chunks<true, false>(src, ceb, eb, s, cnt, acc);
            else
                chunks<true, true>(src, ceb, eb, s, cnt, acc);
        }
        f2_split(acc, a0, a1);
        if (++cb == nb) {
            cb = 0;
            if (own < n)
                sink(own, a0 + a1, pre(own));
            ++done;
        }
        __syncwarp(); // read before the slot is filled again
    }

    template <bool TAIL> __device__ __forceinline__ void group()
    {
        for (int b = 0; b < nb; ++b) {
            if (it >= (uint32_t)R) {
                cp_async_wait<R - 1>();
                consume(R);
            }
            issue<TAIL>();
        }
    }

    __device__ __forceinline__ void drain()
    {
        cp_async_wait<0>();
        for (uint32_t left = it < (uint32_t)R ? it : R; left > 0; --left)
            consume(left);
    }

    __device__ __forceinline__ bool full() const { return n - groups * 32 >= 32; }
    __device__ __forceinline__ bool rest() const { return n > groups * 32; }
};

// The centre of a pass: registers, or shared memory for any d.
struct GenericCentre {
    const float *c; // features from index 0, with kCentrePad floats of room before and after
    int lo;         // FP8: the low parts start here
};

template <int DT, int D, int L_, class Centre, class RowAt, class Ahead, class Pre, class Sink>
__device__ __forceinline__ auto make_row_pipe(const PassIO &io, int64_t base, const Centre &c,
                                              char *ring, RowAt r, Ahead a, Pre p, Sink s)
{
    if constexpr (D == 0)
        return GenericPipe<DT, RowAt, Ahead, Pre, Sink>(io, base, c.c, c.lo, ring, r, a, p, s);
    else
        return RowPipe<DT, D, L_, RowAt, Ahead, Pre, Sink>(io, base, c, ring, r, a, p, s);
}

// floats before and after a centre in shared memory: a chunk of a row's first
// or last bytes may reach 31 features before it, one past its last 94 after it
// (they count nothing)
constexpr int kCentrePad = 96;

// Shared-memory floats of an any-d centre.
__host__ __device__ __forceinline__ int64_t generic_centre_floats(int dt, int d)
{
    const int64_t one = (d + 2 * kCentrePad + 3) / 4 * 4;
    return dt == KPP_FP8_E4M3 ? 2 * one : one;
}

// A row's new D^2 with its previous one given; stores what changed.
template <int MODE>
__device__ __forceinline__ float keep_nearest(const PassIO &io, int64_t row, float v, float old)
{
    if (!io.first && !(v < old))
        return old;
    if (MODE == D2_INPLACE)
        io.d2[row] = v;
    else
        io.d2s[row - io.r0] = v;
    if (io.lab)
        io.lab[row - io.r0] = io.lab_new;
    return v;
}

// Shared memory of the passes that skip rows, beside the block's D^2 and
// chunk sums (byte offsets from `base`): labels (D^2 in shared memory only),
// the bounds and rows of the chosen centres, the pass's centre (any d), every
// warp's ring (with room for FP8 scales) and list of rows to read, and (D^2 in the output array only)
// the D^2 of those rows.
struct PruneLayout {
    int64_t lab, thr, cidx, cen, ring, list, list_d2, bytes;
};
// (a ring starts on a 128-byte boundary: at 16 bytes past one every 32-byte
// sector lands in two of shared memory and is requested from L2 twice --
// 20.7 GB crossed to the SMs for 10.2 GB of points)
constexpr int kPruneRingBytes = kPruneRing + 4 * kPruneAhead;
static_assert(kPruneRingBytes % 128 == 0, "rings are 128-byte aligned");

template <int MODE> struct ListRow {
    using type = uint32_t;
};
template <> struct ListRow<D2_SMEM> {
    using type = uint16_t; // offsets in a block that fits shared memory
};

__host__ __device__ __forceinline__ PruneLayout prune_layout(int64_t base, int64_t chunk, int K,
                                                             bool d2_in_smem, int nwarps,
                                                             int64_t centre_floats = 0)
{
    PruneLayout p;
    const int64_t kp = K < kPruneCentres ? K : kPruneCentres;
    p.lab = (base + 15) & ~15ll;
    p.thr = p.lab + (d2_in_smem ? ((2 * chunk + 15) & ~15ll) : 0);
    p.cidx = p.thr + 4 * kp;
    p.cen = (p.cidx + 4 * kp + 15) & ~15ll;
    p.ring = (p.cen + 4 * centre_floats + 127) & ~127ll;
    p.list = p.ring + (int64_t)kPruneRingBytes * nwarps;
    p.list_d2 = p.list + (d2_in_smem ? 2ll : 4ll) * kPruneList * nwarps;
    p.bytes = p.list_d2 + (d2_in_smem ? 0 : 4ll * kPruneList * nwarps);
    return p;
}

// The end of a pass over a segment: D^2 to the output array where the pass
// asks for it, the segment's sum.
template <int MODE>
__device__ __forceinline__ void pass_end(const PassIO &io, int64_t seg_first, int rows,
                                         const Pair &lacc)
{
    const int lane = threadIdx.x & 31;
    if (MODE == D2_SMEM && io.d2_out) {
        __syncwarp(); // the rows' last stores came from other lanes
        for (int o = lane; o < rows; o += 32)
            io.d2_out[seg_first + o] = io.d2s[seg_first - io.r0 + o];
    }
    const Pair seg = warp_pair_sum(lacc);
    if (lane == 0)
        io.segs[threadIdx.x >> 5] = make_float2(seg.hi, seg.lo);
}

struct PruneIO {
    int64_t ci;          // the new centre's row
    float *thr;          // room for the bounds of the chosen centres (shared memory)
    const int32_t *cidx; // their rows (shared memory)
    int nc;              // chosen centres to take a bound for (0: read every row)
    float *cen;          // room for the pass's centre (any d; shared)
    char *ring;          // this warp's ring (shared)
    void *list;          // this warp's list of rows to read (shared)
    float *list_d2;      // their D^2, or that of the rows in flight (D2_INPLACE; shared)
    int *active;         // out: rows each warp read (shared)
};

// The pass over this warp's segment that reads only the rows whose D^2 can
// fall, or (pr.nc == 0) all of them.  A block of 32-row groups at a time:
// their D^2 and labels (the next block's loads are in flight meanwhile) are
// tested one row per lane, and the rows left go to the warp's list, which
// feeds the row pipe a full group at a time, so the reads of one block's rows
// are in flight while the next are tested.  A skipped row costs 6 bytes, most
// of them from L2, in place of its own.
template <int DT, int D, int L_, int MODE>
__device__ __forceinline__ void pass_rows_pruned(const PassIO &io, const PruneIO &pr)
{
    using G = Geom<DT, D, L_>;
    using Row = typename ListRow<MODE>::type;
    constexpr int U = kPruneBlock;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    int64_t seg_first, seg_last;
    segment_rows(io.r0, io.r1 - io.r0, G::SW, nwarps, warp, &seg_first, &seg_last);
    const int rows = (int)(seg_last - seg_first); // offsets in the segment are ints
    const int64_t rel = seg_first - io.r0;
    auto centre = [&] {
        if constexpr (D == 0) {
            GenericCentre gc;
            gc.c = pr.cen + kCentrePad;
            gc.lo = (int)generic_centre_floats(KPP_F32, io.d);
            const float s = DT == KPP_FP8_E4M3 ? __ldg(io.scales + pr.ci) : 1.0f;
            for (int k = threadIdx.x; k < io.d; k += blockDim.x) {
                const float v = decode1<DT>(io.gpts, pr.ci * io.d + k);
                if constexpr (DT == KPP_FP8_E4M3)
                    split_fp8_centre(s, v, pr.cen[kCentrePad + k], pr.cen[kCentrePad + gc.lo + k]);
                else
                    pr.cen[kCentrePad + k] = v;
            }
            __syncthreads();
            return gc;
        } else {
            CentreRegs<DT, D, L_> cr;
            cr.load(io.gpts, io.scales, pr.ci);
            return cr;
        }
    };
    const auto cr = centre();
    if (pr.nc > 0) {
        // the distance of the new centre to every chosen one, each warp a
        // share of them
        const int per = (pr.nc + nwarps - 1) / nwarps;
        const int f = warp * per;
        const int n = pr.nc - f < per ? pr.nc - f : per;
        if (n > 0) {
            auto pipe = make_row_pipe<DT, D, L_>(
                io, 0, cr, pr.ring,
                [&](int i, int k) { return (uint32_t)pr.cidx[f + (i + k < n ? i + k : n - 1)]; },
                [](int) {}, [](int) { return 0; },
                [&](int i, float v, int) { pr.thr[f + i] = prune_bound(v); });
            pipe.n = n;
            while (pipe.rest())
                pipe.template group<true>();
            pipe.drain();
        }
        __syncthreads();
    }
    Pair lacc{};
    if (pr.nc == 0) {
        // every row, in order (backwards on reverse passes): no tests, no list;
        // the previous D^2 comes with the group's rows
        float *old = pr.list_d2;
        auto at = [&](int i) { return io.reverse ? rows - 1 - i : i; };
        auto pipe = make_row_pipe<DT, D, L_>(
            io, seg_first, cr, pr.ring, [&](int i, int k) { return (uint32_t)at(i + k); },
            [&](int i) {
                if (MODE == D2_INPLACE && !io.first &&
                    kpp_check(io.ctl, at(i) >= 0 && at(i) < rows, 117))
                    cp_async4((uint32_t)__cvta_generic_to_shared(old + i % kPruneList),
                              io.d2 + seg_first + at(i));
            },
            [&](int i) {
                return MODE == D2_INPLACE ? old[i % kPruneList]
                                          : io.d2s[rel + (i < rows ? at(i) : 0)];
            },
            [&](int i, float v, float o) {
                if (kpp_check(io.ctl, seg_first + at(i) < seg_last, 114))
                    lacc.add(keep_nearest<MODE>(io, seg_first + at(i), v, o));
            });
        pipe.n = rows;
        while (pipe.full())
            pipe.template group<false>();
        if (pipe.rest())
            pipe.template group<true>();
        pipe.drain();
        pass_end<MODE>(io, seg_first, rows, lacc);
        if (lane == 0)
            pr.active[warp] = rows;
        return;
    }
    Row *list = reinterpret_cast<Row *>(pr.list);
    float *list_d2 = pr.list_d2;
    struct Own {
        int row;
        float d2;
    };
    auto pipe = make_row_pipe<DT, D, L_>(
        io, seg_first, cr, pr.ring,
        [&](int i, int k) { return (uint32_t)list[i % kPruneList + k]; }, [](int) {},
        [&](int i) {
            Own o;
            o.row = (int)list[i % kPruneList];
            o.d2 = MODE == D2_INPLACE ? list_d2[i % kPruneList] : io.d2s[rel + o.row];
            return o;
        },
        [&](int, float v, const Own &o) {
            if (kpp_check(io.ctl, seg_first + o.row < seg_last, 111))
                lacc.add(keep_nearest<MODE>(io, seg_first + o.row, v, o.d2));
        });
    const int nblock = (rows + 32 * U - 1) / (32 * U);
    float d2[U];
    uint16_t lb[U];
    auto load = [&](int j) {
        const int b = (io.reverse ? nblock - 1 - j : j) * 32 * U;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int o = b + 32 * u + lane;
            const bool in = o < rows && kpp_check(io.ctl, seg_first + o < io.r1, 110);
            if (MODE == D2_SMEM) {
                d2[u] = in ? io.d2s[rel + o] : 0.f;
                lb[u] = in ? io.lab[rel + o] : 0;
            } else {
                d2[u] = in ? __ldcg(io.d2 + seg_first + o) : 0.f;
                lb[u] = in ? __ldcg(io.lab + rel + o) : 0;
            }
        }
    };
    if (nblock > 0)
        load(0);
    for (int j = 0; j < nblock; ++j) {
        const int b = (io.reverse ? nblock - 1 - j : j) * 32 * U;
        int n = pipe.n;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int o = b + 32 * u + lane;
            const float t = lb[u] < pr.nc ? pr.thr[lb[u]] : -1.f;
            const bool must = o < rows && !(d2[u] <= t);
            const unsigned m = __ballot_sync(0xffffffffu, must);
            if (must) {
                const int at = (n + __popc(m & ((1u << lane) - 1u))) % kPruneList;
                list[at] = (Row)o;
                if (MODE == D2_INPLACE)
                    list_d2[at] = d2[u];
            }
            n += __popc(m);
            lacc.add(must ? 0.f : d2[u]);
        }
        pipe.n = n;
        if (j + 1 < nblock) {
            load(j + 1);
        } else { // the last group's other items are looked at, not read
            list[(n + lane) % kPruneList] = 0;
            if (MODE == D2_INPLACE)
                list_d2[(n + lane) % kPruneList] = 0.f;
        }
        __syncwarp(); // the list is read by other lanes
        while (pipe.full())
            pipe.template group<false>();
    }
    if (pipe.rest())
        pipe.template group<true>();
    pipe.drain();
    pass_end<MODE>(io, seg_first, rows, lacc);
    if (lane == 0)
        pr.active[warp] = pipe.n;
}

// The CTA's D^2 sum: warp pairs added in warp order, rounded once to FP64.
// All threads return it.  `sh` holds 2 floats per warp.
__device__ __forceinline__ double cta_sum(const Pair &wacc, float *sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) {
        sh[2 * warp] = wacc.hi;
        sh[2 * warp + 1] = wacc.lo;
    }
    __syncthreads();
    Pair t{};
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        Pair q;
        q.hi = sh[2 * w];
        q.lo = sh[2 * w + 1];
        t.add(q);
    }
    return t.value();
}

// Generic pass for any d and any row alignment: one thread per row, element
// loads, centre in shared memory (c_sh[0..d) = c_hi, c_sh[d..2d) = c_lo for
// FP8).  Segments as in pass_rows with 32-row super-iterations.
template <int DT>
__device__ __forceinline__ Pair pass_rows_generic(const PassIO &io, int d, const float *c_sh)
{
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    int64_t seg_first, seg_last;
    segment_rows(io.r0, io.r1 - io.r0, 32, nwarps, warp, &seg_first, &seg_last);
    Pair lacc{};
    for (int64_t row = seg_first + lane; row < seg_last; row += 32) {
        const float sc = (DT == KPP_FP8_E4M3) ? __ldg(io.scales + row) : 1.0f;
        float a0 = 0.f, a1 = 0.f;
        int k = 0;
        for (; k + 1 < d; k += 2) {
            float q0 = decode1<DT>(io.gpts, row * d + k);
            float q1 = decode1<DT>(io.gpts, row * d + k + 1);
            float t0, t1;
            if constexpr (DT == KPP_FP8_E4M3) {
                t0 = diff_fp8(sc, q0, c_sh[k], c_sh[d + k]);
                t1 = diff_fp8(sc, q1, c_sh[k + 1], c_sh[d + k + 1]);
            } else {
                t0 = q0 - c_sh[k];
                t1 = q1 - c_sh[k + 1];
            }
            a0 = fmaf(t0, t0, a0);
            a1 = fmaf(t1, t1, a1);
        }
        if (k < d) {
            float q0 = decode1<DT>(io.gpts, row * d + k);
            float t0 = (DT == KPP_FP8_E4M3) ? diff_fp8(sc, q0, c_sh[k], c_sh[d + k])
                                            : q0 - c_sh[k];
            a0 = fmaf(t0, t0, a0);
        }
        lacc.add(update_d2<D2_INPLACE>(io, row, a0 + a1, prefetch_d2<D2_INPLACE>(io, row, true)));
    }
    const Pair seg = warp_pair_sum(lacc);
    if (lane == 0)
        io.segs[warp] = make_float2(seg.hi, seg.lo);
    return seg;
}

template <int DT>
__device__ __forceinline__ void load_centre_smem(const void *points, const float *scales,
                                                 int64_t ci, int d, float *c_sh)
{
    const float s = (DT == KPP_FP8_E4M3) ? __ldg(scales + ci) : 1.0f;
    for (int k = threadIdx.x; k < d; k += blockDim.x) {
        const float q = decode1<DT>(points, ci * d + k);
        if constexpr (DT == KPP_FP8_E4M3)
            split_fp8_centre(s, q, c_sh[k], c_sh[d + k]);
        else
            c_sh[k] = q;
    }
}

} // namespace kpp
