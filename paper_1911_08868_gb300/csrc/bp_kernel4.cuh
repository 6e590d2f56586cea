// Register-resident PP-BP decoder kernel (sm_103a), the bp_decode path (Algorithm 1 of
// arXiv 1911.08868).
//
// What bounds it: instruction issue, and behind it the instruction cache.  The shared-memory and
// tensor-memory kernels spend 60% of their instructions on moving messages (N = 1024: 3.65 k warp
// instructions per frame-iteration, 1.45 k of them PE arithmetic); here it is 1.98 k without an event
// and about 2.6 k under one.  The loops every frame runs have to stay within 10 to 15 KB each: with
// 16 positions a thread, or with the switch below unrolled over its slots, warps waited for
// instructions (2 to 5 stall cycles per issue) and the same instruction counts ran slower than the
// kernels they were to replace.
//
// Layouts.  A frame belongs to one warp up to N = 256 and to N / 256 warps above.  A thread holds
// E = 2^KB positions of a node level (8 from N = 256 on, 4 at N = 128, 2 below): KB position bits are
// register bits, the others thread bits.  A group of up to KB consecutive stages whose bits are
// register bits runs without any exchange; between two groups the level passes once through a
// scratch plane in shared memory, written in one layout and read in the next.  From the second
// group on every layout gives the warps the same position bits, so only the exchange between the
// first two groups needs a barrier of the frame's warps, the others a warp sync.
//
// One slot per level.  Level l (2..n) needs R(l) until stage l-2 of the L sweep has used it, and
// L(l), which that stage produces, until the R sweep has used it to make the new R(l): the two are
// never alive at the same time, so one slot of E registers holds both in turn, and a frame's whole
// state is n-1 such slots and the channel LLRs (N = 1024: 80 of the 128 registers).
//
// Permutation events.  In the event's subgraph (the positions whose low n-m bits equal the block,
// m = hi+1) the stages lo..hi use permuted bits.  The levels up to hi+1 are kept under permuted
// position labels, under which every stage up to hi uses its natural bit (the stages before lo use
// bits that the permutation leaves alone), so the sweeps' code does not change: a sweep relabels
// once, at the boundary hi+1, by an exchange through a second plane at per-thread addresses (the
// event's map in the layout of stage hi).  A switch zeroes the interior levels of the subgraphs it
// leaves and enters (Sec. III) and moves the other levels up to hi+2 and the channel LLRs from the
// old labels to the new; it puts the slots in tensor memory, whose columns a loop can index, and
// takes them back.  A frame's first switch draws its first 32 events, one a lane.
//
// Two copies of the iteration, one for the original graph without any test for events.  The stop
// test comes after the R sweep's last group, which hides the reduction and the warps' skew (N = 1024
// at 3 dB 10.0 -> 9.7 ms on 262,144 frames, N = 2048 at 2 dB 8.2 -> 7.7 ms on 16,384).
//
// Time per frame-iteration against the tensor-memory kernel (14,592 frames of scaled min-sum without
// a stop test, 100 iterations more against 100 fewer; events of 4 stages), in ns, at N = 128, 256, 512,
// 1024 and 2048: without an event 0.27 / 0.51, 0.39 / 0.95, 0.88 / 1.39, 2.22 / 3.59 and 5.20 / 7.62;
// under an event 0.36 / 0.55, 0.55 / 1.24, 1.23 / 1.62, 3.20 / 3.85 and 7.47 / 8.87; a switch 0.86 / 1.69,
// 1.27 / 2.97, 2.89 / 4.63, 6.83 / 7.59 and 16.2 / 16.5.  N = 64 against the shared-memory kernel: 0.13 /
// 0.89, 0.24 / 1.14 and 0.80 / 3.04.
//
// Arithmetic: every floating-point operation and its operand order are those of the other decoder
// kernels (l_layer, r_layer), so the outputs are bit-identical.
#pragma once

#include "bp_kernel3.cuh"

namespace pcbp {

template <int LOGN>
struct G4 {
    static constexpr int n = LOGN;
    static constexpr int N = 1 << LOGN;
    static constexpr int KB = n <= 6 ? 1 : (n == 7 ? 2 : 3);
    static constexpr int E = 1 << KB;
    static constexpr int T = N / E;                          // threads that own positions
    static constexpr int WPF = T > 32 ? T / 32 : 1;          // warps per frame
    static constexpr int LW = n - KB > 5 ? n - KB - 5 : 0;   // log2 WPF
    static constexpr int G = (n + KB - 1) / KB;              // groups of KB stages, the last ones shorter
    static constexpr int NW = N >= 32 ? N / 32 : 1;
    // one CTA per SM: with 128 registers a thread 16 warps, with 80 24
    static constexpr int WARPS = n >= 8 ? 16 : 24;
    // Scratch plane: position j at word (j / 32) P + j % 32.  With P = 36 every access from N = 256
    // on is free of bank conflicts, the last group's in vectors of consecutive registers.
    static constexpr int P = 36;
    static constexpr int PLANE = N >= 32 ? (N / 32) * P : N;

    // First stage of group g: groups of KB stages.  N = 1024 has 3, 3, 2, 2: with 3, 3, 3, 1 the third
    // group's register bits would be position bits 1..3, and a warp's accesses in that layout would
    // meet in pairs on the banks (position bits 0, 4, 5, .. from the lanes); from run_low = 2 on they
    // do not.  Without an event 2.22 against 2.35 ns per frame-iteration, 262,144 PP-BP frames at 3 dB
    // 8.97 against 9.35 ms, 65,536 at 2 dB 14.1 against 14.7.  No other length leaves one stage but
    // N = 128, whose groups are of 2.
    __host__ __device__ static constexpr int first(int g) { return g >= G ? n : (n == 10 && g == 3 ? 8 : g * KB); }
    __host__ __device__ static constexpr int len(int g) { return first(g + 1) - first(g); }
    __host__ __device__ static constexpr int grp(int s) { return n == 10 && s == 8 ? 3 : s / KB; }
    // group g's register bits are position bits run_low .. run_low + KB - 1
    __host__ __device__ static constexpr int run_low(int g)
    {
        return g == G - 1 ? 0 : (n == 10 && g == 2 ? 2 : n - first(g) - KB);
    }
    // position bit of register bit i of group g: in the last group bit i; in the others a bit of the
    // run that no stage of the group uses first, then the stages' bits in stage order
    __host__ __device__ static constexpr int reg_pos(int g, int i)
    {
        if (g == G - 1) return i;
        const int f = KB - len(g);
        return i >= f ? n - 1 - first(g) - (i - f) : n - first(g) + i;
    }
    __host__ __device__ static constexpr int stage_reg(int s)
    {
        return grp(s) == G - 1 ? n - 1 - s : KB - len(grp(s)) + s - first(grp(s));
    }
    __host__ __device__ static constexpr int word_of(int pos) { return (pos >> 5) * P + (pos & 31); }
    __host__ __device__ static constexpr int epos(int g, int e)
    {
        int p = 0;
        for (int i = 0; i < KB; ++i)
            if ((e >> i) & 1) p |= 1 << reg_pos(g, i);
        return p;
    }
    // register bit of position bit b in group g, -1 where it is a thread bit
    __host__ __device__ static constexpr int bit_reg(int g, int b)
    {
        for (int i = 0; i < KB; ++i)
            if (reg_pos(g, i) == b) return i;
        return -1;
    }
    // the same tables for a run-time group, 4 bits an entry
    __host__ __device__ static constexpr uint64_t packed_first()
    {
        uint64_t v = 0;
        for (int g = 0; g <= G; ++g) v |= uint64_t(first(g)) << (4 * g);
        return v;
    }
    __host__ __device__ static constexpr uint64_t packed_run_low()
    {
        uint64_t v = 0;
        for (int g = 0; g < G; ++g) v |= uint64_t(run_low(g)) << (4 * g);
        return v;
    }
    __host__ __device__ static constexpr uint64_t packed_reg_pos(int i)
    {
        uint64_t v = 0;
        for (int g = 0; g < G; ++g) v |= uint64_t(reg_pos(g, i)) << (4 * g);
        return v;
    }
    // whether the iteration under an event has a copy of each group's stages with the tests for a
    // relabelling inside the group, entered where it relabels there: fewer instructions (a test
    // makes the values of both paths meet in the same registers, with moves), more code.  Pays at
    // N = 1024 alone.  PP-BP frames, with the copies against without: N = 1024 8.97 / 9.50 ms (262,144 at
    // 3 dB) and 3.48 / 3.72 (65,536, CRC and G-matrix stop); N = 128 0.87 / 0.85 (100,003); N = 256
    // 0.73 / 0.71 and 1.08 / 1.02, N = 512 1.64 / 1.51 and 2.31 / 2.15 (65,536, CRC stop and both);
    // N = 2048 7.62 / 7.50 (16,384 at 2 dB) and 2.81 / 2.83 (32,768 at 3 dB).  Below N = 128 every group
    // is one stage, and there is nothing to copy.
    static constexpr bool COPY = n == 10;
    // tensor memory: n-1 slots of E columns per warp, WARPS / 4 warps to a lane quarter
    static constexpr int SLOT_COLS = (n - 1) * E;
    __host__ __device__ static constexpr int tm_cols()
    {
        int c = 32;
        while (c < (WARPS / 4) * SLOT_COLS) c *= 2;
        return c;
    }
    // whether the warp bits of the thread index are the top position bits in group g
    __host__ __device__ static constexpr bool top_warps(int g) { return run_low(g) + KB <= n - LW; }
    // CTA shape
    static constexpr int SLOTS = WARPS / WPF;
    static constexpr int VT = E >= 4 ? 4 : 2;                // values per lane-private vector
    // shared memory: CTA tables (priors, CRC table, information positions), then the frames
    static constexpr int CB = E >= 4 && n < 11 ? 4 : 2;      // decisions per entry of the CRC table
    static constexpr int CRC_WORDS = ((E / CB) << CB) * T;
    static constexpr int NWA = (NW + 3) & ~3;
    static constexpr int EVENTS = 32;                        // events drawn at once
    static constexpr int FRAME_WORDS = 2 * PLANE + G * N + 4 * EVENTS + 2 * NWA + 12;
    __host__ __device__ static constexpr size_t table_words(int K)
    {
        return size_t(PLANE) + CRC_WORDS + ((size_t(K) + 7) & ~size_t(7)) / 2;
    }
    __host__ __device__ static constexpr size_t smem_bytes(int K, int slots)
    {
        return 4 * (table_words(K) + size_t(slots) * FRAME_WORDS);
    }
};

template <int A, int B, class F>
__device__ __forceinline__ void sfor(F&& f)
{
    if constexpr (A < B) {
        f(std::integral_constant<int, A>{});
        sfor<A + 1, B>(f);
    }
}

// Index i of `step` consecutive entries, a multiple of step, in a buffer of `limit`.  A build with
// PCBP_CHECKED checks it: out of range, bit `cls` of the status word (when there is one) is set and
// the access redirected to entry 0, so nothing faults.
template <int step = 1>
__device__ __forceinline__ int in_range(unsigned* status, unsigned cls, int i, int limit)
{
#ifdef PCBP_CHECKED
    if (i < 0 || i > limit - step || i % step != 0) {
        chk_fail(status, cls);
        return 0;
    }
#endif
    return i;
}

// A level between a thread's registers and a plane, in the layout of group g: tb is the word of
// the thread's base position, the registers are at compile-time distances from it.
template <int LOGN, int g>
__device__ __forceinline__ void plane_st(float* plane, int tb, const float* v, unsigned* check)
{
    using Geo = G4<LOGN>;
    constexpr int E = Geo::E;
    if constexpr (g == Geo::G - 1) {
#pragma unroll
        for (int e = 0; e < E; e += Geo::VT) {
            float* const d = plane + in_range<Geo::VT>(check, 0, tb + e, Geo::PLANE);
            if constexpr (E >= 4) *reinterpret_cast<float4*>(d) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
            else *reinterpret_cast<float2*>(d) = make_float2(v[e], v[e + 1]);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) plane[in_range(check, 0, tb + Geo::word_of(Geo::epos(g, e)), Geo::PLANE)] = v[e];
    }
}

template <int LOGN, int g>
__device__ __forceinline__ void plane_ld(const float* plane, int tb, float* v, unsigned* check)
{
    using Geo = G4<LOGN>;
    constexpr int E = Geo::E;
    if constexpr (g == Geo::G - 1) {
#pragma unroll
        for (int e = 0; e < E; e += Geo::VT) {
            const float* const s = plane + in_range<Geo::VT>(check, 0, tb + e, Geo::PLANE);
            if constexpr (E >= 4) {
                const float4 w = *reinterpret_cast<const float4*>(s);
                v[e] = w.x; v[e + 1] = w.y; v[e + 2] = w.z; v[e + 3] = w.w;
            } else {
                const float2 w = *reinterpret_cast<const float2*>(s);
                v[e] = w.x; v[e + 1] = w.y;
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = plane[in_range(check, 0, tb + Geo::word_of(Geo::epos(g, e)), Geo::PLANE)];
    }
}

// A slot between a thread's registers and its lane of tensor memory, E columns (valid after
// tm_wait_st() / tm_wait_ld() and tm_fence()).
template <int E>
__device__ __forceinline__ void slot_st(uint32_t a, const float* v)
{
    if constexpr (E == 2)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(a), "f"(v[0]), "f"(v[1]) : "memory");
    else
        tm_st<E>(a, v);
}

template <int E>
__device__ __forceinline__ void slot_ld(uint32_t a, float* v)
{
    if constexpr (E == 2)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(a) : "memory");
    else
        tm_ld<E>(a, v);
}

// Events k0 + lane of a frame (draw_event of bp_kernel.cuh: the same draws, remainders and choices),
// one a lane: x = first permuted stage | last << 8 | block << 16, z | w << 32 the packed order.
static __device__ __noinline__ void draw_events(const DevSched& S, int n, uint64_t frame, int k0, int4* out, int lane)
{
    const uint64_t hk = splitmix_out(splitmix_out(splitmix_out(S.seed) ^ frame) ^ uint64_t(k0 + lane));
    auto draw = [&](int d, uint32_t m) { return int(mod_small(splitmix_out(hk ^ uint64_t(d)), m)); };
    int range = n, level = 1, block = 0;
    if (S.mode != 2) {
        range = S.rho_fixed > 0 ? S.rho_fixed : 2 + draw(0, uint32_t(S.P_range - 1));
        level = min(1 + draw(1, uint32_t(S.P_level)), n - range + 1);
        block = int(splitmix_out(hk ^ 2ull) & ((1ull << (n - level - range + 1)) - 1ull));
    }
    uint64_t ident = 0;
#pragma unroll 1
    for (int i = range - 1; i >= 0; --i) ident = (ident << 4) | uint64_t(i);
    uint64_t ord = ident;
#pragma unroll 1
    for (int attempt = 0; attempt < 8 && ord == ident; ++attempt) {
#pragma unroll 1
        for (int i = range - 1; i >= 1; --i) {
            const int j = draw(3 + 16 * attempt + (range - 1 - i), uint32_t(i + 1));
            const uint64_t x = ((ord >> (4 * i)) ^ (ord >> (4 * j))) & 15u;
            ord ^= (x << (4 * i)) | (x << (4 * j));
        }
    }
    if (ord == ident) ord = (ident >> 4);          // rotation: order[i] = (i + 1) mod range
    out[lane] = make_int4((level - 1) | ((level + range - 2) << 8) | (block << 16), 0, int(uint32_t(ord)),
                          int(uint32_t(ord >> 32)));
}

// PO = 1 (the messages output of bp_decode_posterior, for verification): a frame's last iteration
// completes its R sweep and writes L at node level n+1 and R at node level 1 to J.post.
template <int LOGN, int FK, int WG, int PO>
__device__ __forceinline__ void warp_frames(const WarpParams& P, float* smem, uint32_t tm_base)
{
    using Geo = G4<LOGN>;
    constexpr int n = LOGN, N = Geo::N, E = Geo::E, KB = Geo::KB, T = Geo::T, WPF = Geo::WPF, G = Geo::G;
    constexpr int NWA = Geo::NWA, VT = Geo::VT;

    const FrameJob& J = P.job;
    const DevSched& S = J.S;
    const int K = J.K;
    const int KW = (K + 31) / 32;
    const float alpha = S.alpha, nz = J.neg_zero;
    const int max_iters = J.max_iters;
    constexpr bool want_g = WG != 0;
    static_assert(!(PO && (WG || LOGN < 7)), "the messages output is built for the CRC stop, from N = 128 on");
    const bool want_crc = (S.stop_kind & 1) != 0;

    const float* s_pri = smem;                                             // priors, a plane
    const uint32_t* s_crc = reinterpret_cast<const uint32_t*>(smem + Geo::PLANE);
    const int16_t* s_info = reinterpret_cast<const int16_t*>(smem + Geo::PLANE + Geo::CRC_WORDS);

    const int lane = int(threadIdx.x & 31);
    const int slot = int(threadIdx.x) / (32 * WPF);
    const int tid = WPF > 1 ? int(threadIdx.x) - slot * 32 * WPF : lane & (T - 1);   // T < 32: lanes repeat
    const int warp = WPF > 1 ? tid >> 5 : 0;
    float* const scratch = smem + Geo::table_words(K) + slot * Geo::FRAME_WORDS;
    float* const ev_plane = scratch + Geo::PLANE;                          // the event exchanges' plane
    int* const maps = reinterpret_cast<int*>(scratch + 2 * Geo::PLANE);    // the event's map in each layout
    int4* const events = reinterpret_cast<int4*>(maps + G * N);
    uint32_t* const dec = reinterpret_cast<uint32_t*>(events + Geo::EVENTS);
    uint32_t* const xh = dec + NWA;
    uint32_t* const red = xh + NWA;

    const uint32_t tm = tm_base + (uint32_t(32 * ((threadIdx.x >> 5) & 3)) << 16) + uint32_t((threadIdx.x >> 7) * Geo::SLOT_COLS);

    auto fsync = [&]() {
        if constexpr (WPF == 1) __syncwarp();
        else slot_sync(1u + unsigned(slot), 32 * WPF);
    };

    // the thread's base position in the layout of group g
    auto base_pos = [&](int g) {
        const int rl = Geo::run_low(g);
        return (tid & ((1 << rl) - 1)) | ((tid >> rl) << (rl + KB));
    };
    int tb[G];
#pragma unroll
    for (int g = 0; g < G; ++g) tb[g] = Geo::word_of(base_pos(g));
    // information positions of the thread's run in the last group
    unsigned infow;
    {
        const int p0 = tid << KB;
        infow = ~(P.frozen[p0 >> 5] >> (p0 & 31)) & ((1u << E) - 1u);
    }

    // the event's last stage (-1: no event) and its map in that stage's layout
    int ev_hi = -1, ev_x = 0;
    const int* map_hi = maps;
    float Lc[E];                                   // channel LLRs, layout and labels of stage 0
    float slots[n - 1][E];                         // slot k: level k+2, layout and labels of stage k (R) or k+1 (L)

    // --- exchanges through the scratch plane
    // natural labels, layout a -> layout b: a warp writes the positions that it read last, so no
    // barrier is needed before
    auto exch = [&](auto evc, auto ga, auto gb, float* v) {
        constexpr int a = decltype(ga)::value, b = decltype(gb)::value;
        if constexpr (KB == 1 && n >= 5 && !decltype(evc)::value) {
            // neighbouring layouts swap the register bit with one lane bit: a shuffle (60,000 frames of
            // N = 64 for 100 iterations 1,295 -> 814 us, N = 32 716 -> 680; no gain at N = 8 and 16, and
            // none under an event, where the boundary also has the other exchange)
            constexpr int bit = 1 << (n - 2 - (a < b ? a : b));
            const bool up = (lane & bit) != 0;
            const float y = __shfl_xor_sync(0xffffffffu, up ? v[0] : v[1], bit);
            v[0] = up ? y : v[0];
            v[1] = up ? v[1] : y;
        } else {
            __syncwarp();
            plane_st<LOGN, a>(scratch, tb[a], v, J.check);
            if constexpr (Geo::top_warps(a) && Geo::top_warps(b)) __syncwarp();
            else fsync();
            plane_ld<LOGN, b>(scratch, tb[b], v, J.check);
        }
    };
    // a level at the places of a map (byte distances from the start of a plane)
    auto map_at = [&](const int* map, int i) {
        const int from = int(map - maps);
        return map + (in_range<VT>(J.check, 3, from + i, G * N) - from);
    };
    auto place = [&](int d) { return in_range<4>(J.check, 3, d, 4 * Geo::PLANE); };
    auto map_ld = [&](const float* plane, const int* map, float* v) {
        const char* p = reinterpret_cast<const char*>(plane);
#pragma unroll
        for (int q = 0; q < E / VT; ++q) {
            if constexpr (VT == 4) {
                const int4 w = *reinterpret_cast<const int4*>(map_at(map, (q * T + tid) * 4));
                v[4 * q] = *reinterpret_cast<const float*>(p + place(w.x));
                v[4 * q + 1] = *reinterpret_cast<const float*>(p + place(w.y));
                v[4 * q + 2] = *reinterpret_cast<const float*>(p + place(w.z));
                v[4 * q + 3] = *reinterpret_cast<const float*>(p + place(w.w));
            } else {
                const int2 w = *reinterpret_cast<const int2*>(map_at(map, (q * T + tid) * 2));
                v[2 * q] = *reinterpret_cast<const float*>(p + place(w.x));
                v[2 * q + 1] = *reinterpret_cast<const float*>(p + place(w.y));
            }
        }
    };
    auto map_st = [&](const int* map, const float* v) {
        char* p = reinterpret_cast<char*>(ev_plane);
#pragma unroll
        for (int q = 0; q < E / VT; ++q) {
            if constexpr (VT == 4) {
                const int4 w = *reinterpret_cast<const int4*>(map_at(map, (q * T + tid) * 4));
                *reinterpret_cast<float*>(p + place(w.x)) = v[4 * q];
                *reinterpret_cast<float*>(p + place(w.y)) = v[4 * q + 1];
                *reinterpret_cast<float*>(p + place(w.z)) = v[4 * q + 2];
                *reinterpret_cast<float*>(p + place(w.w)) = v[4 * q + 3];
            } else {
                const int2 w = *reinterpret_cast<const int2*>(map_at(map, (q * T + tid) * 2));
                *reinterpret_cast<float*>(p + place(w.x)) = v[2 * q];
                *reinterpret_cast<float*>(p + place(w.y)) = v[2 * q + 1];
            }
        }
    };
    // event labels (map) -> natural labels in layout b, and back, through the event plane.  lead: a
    // barrier before, where none of the frame's lies between the last reads of the plane and here.
    auto exch_out = [&](auto lead, const int* map, auto gb, float* v) {
        constexpr int b = decltype(gb)::value;
        if constexpr (decltype(lead)::value) fsync();
        else __syncwarp();
        map_st(map, v);
        fsync();
        plane_ld<LOGN, b>(ev_plane, tb[b], v, J.check);
    };
    auto exch_in = [&](auto ga, const int* map, float* v) {
        constexpr int a = decltype(ga)::value;
        __syncwarp();
        plane_st<LOGN, a>(ev_plane, tb[a], v, J.check);
        fsync();
        map_ld(ev_plane, map, v);
    };
    // whether the last reads of the event plane before the L sweep's exchange at boundary b, the R
    // sweep's at b, need a barrier: past the first group the barriers of the exchanges between the
    // first two groups lie in between
    auto lead = [](auto bc) { return std::integral_constant<bool, (decltype(bc)::value <= KB)>{}; };
    // group boundary of the L sweep, from group g to g + 1; EV: under an event
    auto l_boundary = [&](auto evc, auto gc, float* v) {
        constexpr int g = decltype(gc)::value, b = Geo::first(g + 1);
        std::integral_constant<int, g + 1> gn;
        if (decltype(evc)::value && ev_hi == b - 1) exch_out(lead(std::integral_constant<int, b>{}), map_hi, gn, v);
        else exch(evc, gc, gn, v);
    };
    // and of the R sweep, from group g to g - 1
    auto r_boundary = [&](auto evc, auto gc, float* v) {
        constexpr int g = decltype(gc)::value, b = Geo::first(g);
        if (decltype(evc)::value && ev_hi == b - 1) exch_in(gc, map_hi, v);
        else exch(evc, gc, std::integral_constant<int, g - 1>{}, v);
    };
    // R(n+1) in the layout and labels of stage n-1
    auto priors = [&](auto evc, float* v) {
        if (decltype(evc)::value && ev_hi == n - 1) map_ld(s_pri, map_hi, v);
        else plane_ld<LOGN, G - 1>(s_pri, tb[G - 1], v, J.check);
    };
    // --- frame queue: the first frames spread over the SMs, the others from the counter
    // (a batch of 2^31 frames of N >= 512 would hold over 4 TB of LLRs)
    using Index = std::conditional_t<(n >= 9), int, long long>;
    const Index frames = Index(J.B);
    const Index total = Index(gridDim.x) * P.slots;
    Index f = Index(slot) * Index(gridDim.x) + Index(blockIdx.x);
    auto load_llr = [&](Index fi) {
#ifdef PCBP_CHECKED
        if (fi < 0 || fi >= frames) {
            chk_fail(J.check, 5);
            fi = 0;
        }
#endif
        const float* src = J.llr + size_t(fi) * N + tid;     // the first group's thread bits are the low bits
#pragma unroll
        for (int e = 0; e < E; ++e) Lc[e] = __ldg(src + (in_range(J.check, 5, tid + Geo::epos(0, e), N) - tid));
    };
    if (f < frames) load_llr(f);

    while (f < frames) {
        // a2: R = 0
#pragma unroll
        for (int k = 0; k < n - 1; ++k)
#pragma unroll
            for (int e = 0; e < E; ++e) slots[k][e] = 0.f;
        ev_hi = -1;
        int next_reset = S.mode == 1 ? S.T0 : (S.mode == 2 ? S.it_reset_full : 0);
        int kev = 0;
        unsigned um = 0, res = 0;
        int it = 0;

        // one iteration; true when it is the frame's last
        auto iterate = [&](auto evc) -> bool {
            constexpr bool EV = decltype(evc)::value;
            float x[E], pr[E];
            float lu[PO ? E : 1];                  // PO: L(n+1), natural labels
            // ---------------- L sweep
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = Lc[e];
            sfor<0, G>([&](auto gc) {
                constexpr int g = decltype(gc)::value, s0 = Geo::first(g), s1 = Geo::first(g + 1);
                // the group's stages; in: an event may relabel at a boundary inside the group
                auto stages = [&](auto in) {
                    sfor<s0, s1>([&](auto sc) {
                        constexpr int s = decltype(sc)::value;
                        if constexpr (s == n - 1) {
                            priors(evc, pr);
                            l_layer<E, FK>(x, pr, Geo::stage_reg(s), alpha, nz);
                        } else {
                            l_layer<E, FK>(x, slots[s], Geo::stage_reg(s), alpha, nz);
                            if constexpr (s + 1 < s1) {
                                if (decltype(in)::value && s > 0 && ev_hi == s) exch_out(lead(std::integral_constant<int, s + 1>{}), map_hi, gc, x);
#pragma unroll
                                for (int e = 0; e < E; ++e) slots[s][e] = x[e];
                            }
                        }
                    });
                };
                if constexpr (!Geo::COPY || !EV || s1 - s0 == 1) stages(evc);
                else if (ev_hi >= s0 && ev_hi < s1 - 1) stages(std::true_type{});
                else stages(std::false_type{});
                if constexpr (g < G - 1) {
                    l_boundary(evc, gc, x);
#pragma unroll
                    for (int e = 0; e < E; ++e) slots[s1 - 1][e] = x[e];
                }
            });
            // ---------------- a5: decisions u_j = [L(n+1) + R(n+1) < 0] (frozen positions: 0)
            const bool check = S.stop_kind != 0 && it >= S.stop_from;
            bool gtest = false;
            if (check || it == max_iters) {
                if (EV && ev_hi == n - 1) exch_out(std::false_type{}, map_hi, std::integral_constant<int, G - 1>{}, x);
                if constexpr (PO != 0) {
#pragma unroll
                    for (int e = 0; e < E; ++e) lu[e] = x[e];
                }
                // the sign of x + 0 is set exactly where x < 0 (-0 becomes +0)
                um = 0;
#pragma unroll
                for (int e = 0; e < E; e += 2) {
                    const float2 z = __fadd2_rn(make_float2(x[e], x[e + 1]), make_float2(0.f, 0.f));
                    x[e] = z.x;
                    x[e + 1] = z.y;
                }
#pragma unroll
                for (int o = E - 1; o >= 0; --o) um = __funnelshift_l(__float_as_uint(x[o]), um, 1);
                um &= infow;
                // CRC residue: CB decisions a table entry
                res = 0;
                constexpr int CB = Geo::CB;
#pragma unroll
                for (int k = 0; k < E / CB; ++k)
                    res ^= s_crc[in_range(J.check, 2, ((k << CB) + int((um >> (CB * k)) & ((1u << CB) - 1u))) * T + tid, Geo::CRC_WORDS)];
                if (T < 32 && lane >= T) res = 0;
                res = __reduce_xor_sync(0xffffffffu, res);
                if constexpr (WPF > 1) {
                    // (written again only after the barriers of the exchanges in between)
                    if (lane == 0) red[warp] = res;
                }
            }
            // the stop test, after the R sweep's last group (wasted in a frame's last iteration), so that
            // the reduction's latency and the warps' skew pass meanwhile
            auto last_iteration = [&]() -> bool {
                if (!check && it != max_iters) return false;
                if constexpr (WPF > 1) {
                    fsync();
                    res = red[0];
#pragma unroll
                    for (int w = 1; w < WPF; ++w) res ^= red[w];
                }
                gtest = want_g && check && (!want_crc || res == 0u);
                return want_g ? (it == max_iters && !gtest) : ((check && res == 0u) || it == max_iters);
            };
            // ---------------- R sweep
            priors(evc, x);
            auto r_group = [&](auto jc) {
                constexpr int g = G - 1 - decltype(jc)::value, s0 = Geo::first(g), s1 = Geo::first(g + 1);
                std::integral_constant<int, g> gc;
                auto stages = [&](auto in) {
                    sfor<0, s1 - s0>([&](auto kc) {
                        constexpr int s = s1 - 1 - decltype(kc)::value;
                        if constexpr (s > 0) {
                            r_layer<E, FK>(x, slots[s - 1], Geo::stage_reg(s), alpha, nz);
                            if constexpr (s > s0) {
                                if (decltype(in)::value && s > 1 && ev_hi == s - 1) exch_in(gc, map_hi, x);
#pragma unroll
                                for (int e = 0; e < E; ++e) slots[s - 1][e] = x[e];
                            }
                        }
                    });
                };
                if constexpr (!Geo::COPY || !EV || s1 - s0 == 1) stages(evc);
                else if (ev_hi >= s0 && ev_hi < s1 - 1) stages(std::true_type{});
                else stages(std::false_type{});
                if constexpr (g > 0) {
                    r_boundary(evc, gc, x);
#pragma unroll
                    for (int e = 0; e < E; ++e) slots[s0 - 1][e] = x[e];
                }
            };
            r_group(std::integral_constant<int, 0>{});
            const bool last = last_iteration();
            if (!PO && last) return true;
            sfor<1, G>(r_group);
            if constexpr (PO != 0) {
                if (last) {
                    r_layer<E, FK>(x, Lc, Geo::stage_reg(0), alpha, nz);
                    if constexpr (EV) exch_out(std::true_type{}, maps, std::integral_constant<int, 0>{}, x);
                    float* const post = J.post + size_t(f) * 2 * N;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        post[(tid << KB) + e] = lu[e];
                        post[N + tid + Geo::epos(0, e)] = x[e];
                    }
                    return true;
                }
            }
            // ---------------- G-matrix test: u G_N against the hard decisions of L1 + R1
            if (want_g && gtest) {
                r_layer<E, FK>(x, Lc, Geo::stage_reg(0), alpha, nz);
#pragma unroll
                for (int e = 0; e < E; ++e) x[e] = __fadd_rn(Lc[e], x[e]);
                if constexpr (EV) exch_out(std::true_type{}, maps, std::integral_constant<int, 0>{}, x);
                unsigned w0 = 0;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const unsigned b = __ballot_sync(0xffffffffu, x[e] < 0.f);
                    if constexpr (n >= 6) {
                        if (lane == 0) xh[in_range(J.check, 2, (Geo::epos(0, e) >> 5) | warp, Geo::NW)] = b;
                    } else {
                        w0 |= (b & ((1u << (T & 31)) - 1u)) << Geo::epos(0, e);
                    }
                }
                if (n < 6 && lane == 0) xh[0] = w0;
                unsigned v = um << ((tid << KB) & 31);
#pragma unroll
                for (int o = 1; o < 32 / E && o < T; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
                dec[in_range(J.check, 2, (tid << KB) >> 5, Geo::NW)] = v;
                fsync();
                const bool gok = g_check<LOGN>(dec, xh, lane);
                fsync();
                if (gok || it == max_iters) return true;
            }
            return false;
        };

        bool done = max_iters == 0;
        while (!done) {
            // the frame's iterations up to the next switch, on the original graph or under an event
            if (ev_hi < 0) {
                do {
                    ++it;
                    done = iterate(std::false_type{});
                } while (!done && it != next_reset);
            } else {
                do {
                    ++it;
                    done = iterate(std::true_type{});
                } while (!done && it != next_reset);
            }
            if (done) break;
            // ---------------- a6: switch at iter == N_it,reset
            if (S.mode == 2 && S.q_max > 0 && kev >= S.q_max - 1) {
                next_reset = 0;                    // no further switch
                continue;
            }
            if ((kev & (Geo::EVENTS - 1)) == 0) {
                if (warp == 0) draw_events(S, n, S.frame_base + uint64_t(f), kev, events, lane);
            }
            fsync();
            // stages lo..hi of the subgraph of the positions whose low bits (under the mask low) equal
            // beta, and the same of the event being left
            const int4 e4 = events[kev & (Geo::EVENTS - 1)];
            const int ev_lo = ev_x & 0xff, ev_low = (1 << (n - 1 - ev_hi)) - 1, ev_beta = ev_x >> 16;
            const uint64_t ord = (uint64_t(uint32_t(e4.w)) << 32) | uint32_t(e4.z);
            const int lo = e4.x & 0xff, hi = (e4.x >> 8) & 0xff, m = hi + 1;
            const int low = (1 << (n - m)) - 1, beta = e4.x >> 16;
            // R from the old labels to the new, slot by slot out of tensor memory, in a loop over groups
            // and slots (the iterations' code has to stay in the instruction cache: unrolled, this
            // code was larger than both iterations together)
            sfor<0, n - 1>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                slot_st<E>(tm + k * E, slots[k]);
            });
            tm_wait_st();
            // byte weight of position bit b's image under the event's labels, in lane b
            int img = 0;
            {
                const int s = n - 1 - lane;
                const int pb = s >= lo && s <= hi ? n - 1 - lo - order_at(ord, s - lo) : lane;
                img = pb < 5 ? 4 << pb : (4 * Geo::P) << (pb - 5);
            }
            auto image = [&](int b) { return __shfl_sync(0xffffffffu, img, b); };
            auto field = [](uint64_t table, int g) { return int((table >> (4 * g)) & 15u); };
            const int last = max(hi, ev_hi);
#pragma unroll 1
            for (int g = 0; g < G && field(Geo::packed_first(), g) <= last; ++g) {
                const int rl = field(Geo::packed_run_low(), g);
                const int p = (tid & ((1 << rl) - 1)) | ((tid >> rl) << (rl + KB));
                int* const mp = maps + g * N;
                // byte distances of the thread's places: natural (an), old labels (ao), new (aw)
                int an[E], ao[E], aw[E], pe[E];
                an[0] = 4 * (p + (Geo::P - 32) * (p >> 5));
                aw[0] = 0;
                pe[0] = p;
#pragma unroll
                for (int b = 0; b < n; ++b) aw[0] += ((p >> b) & 1) * image(b);
#pragma unroll
                for (int i = 0; i < KB; ++i) {
                    const int b = field(Geo::packed_reg_pos(i), g);
                    const int wn = b < 5 ? 4 << b : (4 * Geo::P) << (b - 5), wi = image(b);
#pragma unroll
                    for (int e = 0; e < (1 << i); ++e) {
                        an[e | (1 << i)] = an[e] + wn;
                        aw[e | (1 << i)] = aw[e] + wi;
                        pe[e | (1 << i)] = pe[e] | (1 << b);
                    }
                }
                unsigned in_old = 0, in_new = 0;           // registers inside the two subgraphs
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    in_old |= (pe[e] & ev_low) == ev_beta ? 1u << e : 0u;
                    const bool in = (pe[e] & low) == beta;
                    in_new |= in ? 1u << e : 0u;
                    if (!in) aw[e] = an[e];
                }
#pragma unroll
                for (int q = 0; q < E / VT; ++q) {
                    int* d = mp + (in_range<VT>(J.check, 3, g * N + (q * T + tid) * VT, G * N) - g * N);
                    if constexpr (VT == 4) {
                        const int4 w = *reinterpret_cast<const int4*>(d);
                        ao[4 * q] = w.x; ao[4 * q + 1] = w.y; ao[4 * q + 2] = w.z; ao[4 * q + 3] = w.w;
                        *reinterpret_cast<int4*>(d) = make_int4(aw[4 * q], aw[4 * q + 1], aw[4 * q + 2], aw[4 * q + 3]);
                    } else {
                        const int2 w = *reinterpret_cast<const int2*>(d);
                        ao[2 * q] = w.x; ao[2 * q + 1] = w.y;
                        // below N = 64 two or more lanes stand for one thread: all of them read the old map
                        // before one writes the new
                        if constexpr (T < 32) __syncwarp();
                        *reinterpret_cast<int2*>(d) = make_int2(aw[2 * q], aw[2 * q + 1]);
                    }
                }
                const int k1 = min(min(field(Geo::packed_first(), g + 1), n - 1), last + 1);
#pragma unroll 1
                for (int k = field(Geo::packed_first(), g); k < k1; ++k) {
                    // slots up to hi have labels; the interior slots lo..hi-1 are zeroed inside the
                    // subgraph, and no label changes outside it
                    const bool zero_old = k >= ev_lo && k < ev_hi, zero_new = k >= lo && k < hi;
                    const bool move_old = k <= ev_hi && !zero_old, move_new = k <= hi && !zero_new;
                    const unsigned z_old = zero_old ? in_old : 0u, z_new = zero_new ? in_new : 0u;
                    float v[E];
                    const uint32_t col = tm + uint32_t(in_range<E>(J.check, 1, k * E, Geo::SLOT_COLS));
                    slot_ld<E>(col, v);
                    tm_wait_ld();
                    tm_fence<E>(v);
                    char* const pl = reinterpret_cast<char*>(ev_plane);
#pragma unroll
                    for (int e = 0; e < E; ++e) v[e] = (z_old >> e) & 1u ? 0.f : v[e];
                    if (move_old || move_new) {
                        fsync();
                        if (move_old) {
#pragma unroll
                            for (int e = 0; e < E; ++e) *reinterpret_cast<float*>(pl + place(ao[e])) = v[e];
                        } else {
#pragma unroll
                            for (int e = 0; e < E; ++e) *reinterpret_cast<float*>(pl + place(an[e])) = v[e];
                        }
                        fsync();
#pragma unroll
                        for (int e = 0; e < E; ++e) v[e] = *reinterpret_cast<const float*>(pl + place(move_new ? aw[e] : an[e]));
                    }
#pragma unroll
                    for (int e = 0; e < E; ++e) v[e] = (z_new >> e) & 1u ? 0.f : v[e];
                    slot_st<E>(col, v);
                }
            }
            tm_wait_st();
            sfor<0, n - 1>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                slot_ld<E>(tm + k * E, slots[k]);
            });
            tm_wait_ld();
            sfor<0, n - 1>([&](auto kc) { tm_fence<E>(slots[decltype(kc)::value]); });
            // the channel LLRs under the new labels
            load_llr(f);
            fsync();
            plane_st<LOGN, 0>(ev_plane, tb[0], Lc, J.check);
            fsync();
            map_ld(ev_plane, maps, Lc);
            fsync();
            ev_hi = hi;
            ev_x = e4.x;
            map_hi = maps + Geo::grp(hi) * N;
            const long long nzc = (1ll << m) * (long long)(hi - lo);
            long long inc;
            if (S.mode == 2) {
                inc = S.it_reset_full;
            } else {
                const long long qz = S.D > 0 ? nzc / S.D : 0;
                inc = qz > S.N_min ? qz : S.N_min;
            }
            next_reset = it + int(inc);
            ++kev;
        }

        // ---------------- a7: outputs; the next frame's LLRs are on their way meanwhile
        // The index is drawn only now: drawn a frame ahead, a frame waits for the long one (up to
        // max_iters) that its warp is at.  N = 256 2.5 dB, 12,800 frames 775 -> 535 us; 50,021 frames at
        // 3 dB 576 -> 472 us; N = 1024 9.18 -> 8.99 ms on 262,144, N = 2048 7.72 -> 7.34 ms on 16,384.
        // Without a counter every frame has its own slot, and total is past the last.
        Index nf = 0;
        if (P.counter && lane == 0 && warp == 0) nf = Index(atomicAdd(P.counter, 1ull));
        __syncwarp();
        if constexpr (WPF > 1) {
            if (tid == 0) *reinterpret_cast<Index*>(red + 8) = nf;
        }
        {
            unsigned v = um << ((tid << KB) & 31);
#pragma unroll
            for (int o = 1; o < 32 / E && o < T; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
            dec[in_range(J.check, 2, (tid << KB) >> 5, Geo::NW)] = v;
        }
        fsync();
        if constexpr (WPF > 1) nf = *reinterpret_cast<const Index*>(red + 8);
        else nf = __shfl_sync(0xffffffffu, nf, 0);
        const Index fo = f;
        f = total + nf;
        if (f < frames) load_llr(f);
        uint32_t w = 0;
        for (int o = warp; o < KW; o += WPF) {
            const int kk = o * 32 + lane;
            uint32_t bit = 0;
            if (kk < K) {
                const int pos = in_range(J.check, 2, s_info[kk], N);
                bit = (dec[pos >> 5] >> (pos & 31)) & 1u;
            }
            const uint32_t word = __ballot_sync(0xffffffffu, bit);
            if (lane == ((o / WPF) & 31)) w = word;
            if (((o / WPF) & 31) == 31 || o + WPF >= KW) {
                const int oo = o - ((o / WPF) & 31) * WPF + lane * WPF;
                if (oo <= o) J.bits[size_t(fo) * KW + in_range(J.check, 4, oo, KW)] = w;
            }
        }
        if (lane == 0 && warp == 0) {
            J.crc_ok[fo] = res == 0u ? 1 : 0;
            J.iters[fo] = it;          // the iteration that stopped, else max_iters
        }
        fsync();
    }
}

template <int LOGN, int FK, int WG, int PO = 0>
__global__ void __launch_bounds__(32 * G4<LOGN>::WARPS, 1)
    bp_decode_warp_kernel(const __grid_constant__ WarpParams P)
{
    // a kernel launched after this one may start as soon as SMs free up
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    using Geo = G4<LOGN>;
    constexpr int N = Geo::N, E = Geo::E, T = Geo::T;
    extern __shared__ __align__(16) float smem4[];
    const int K = P.job.K;
    uint32_t* s_crc = reinterpret_cast<uint32_t*>(smem4 + Geo::PLANE);
    int16_t* s_info = reinterpret_cast<int16_t*>(smem4 + Geo::PLANE + Geo::CRC_WORDS);
    // c_j of every position, in the first frame's area (N words) while the table is made
    uint32_t* cj = reinterpret_cast<uint32_t*>(smem4 + Geo::table_words(K));
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        smem4[Geo::word_of(j)] = prior_of(P.frozen, j);
        cj[j] = 0u;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const int p = P.info_idx[k];
        s_info[k] = int16_t(p);
        cj[p] = P.crc[k];
    }
    // tensor memory for the switches
    __shared__ uint32_t s_tm;
    if (threadIdx.x < 32) {
        const uint32_t dst = uint32_t(__cvta_generic_to_shared(&s_tm));
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "n"(Geo::tm_cols())
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm_base = s_tm;
    constexpr int CB = Geo::CB;
    for (int i = threadIdx.x; i < Geo::CRC_WORDS; i += blockDim.x) {
        const int t = i % T, v = (i / T) % (1 << CB), k = i / (T << CB);
        uint32_t c = 0;
#pragma unroll
        for (int b = 0; b < CB; ++b)
            if ((v >> b) & 1) c ^= cj[t * E + CB * k + b];
        s_crc[i] = c;
    }
    __syncthreads();
    if (int(threadIdx.x) < P.slots * 32 * Geo::WPF) warp_frames<LOGN, FK, WG, PO>(P, smem4, tm_base);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm_base), "n"(Geo::tm_cols()) : "memory");
}

}  // namespace pcbp
