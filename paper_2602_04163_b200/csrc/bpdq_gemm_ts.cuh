// Included by bpdq_gemm.cu (inside its unnamed namespace, after the PTX wrappers): the kernel for up to 128 tokens.
//
// gemm_ts_kernel: decoded weights go from the decode threads' registers straight into TMEM and are the MMA's A operand
// there.  With A in shared memory a 128 x N x 16 MMA takes 39 to 48 clocks for N <= 64 (its 4 KB of A), and writing A costs
// the same shared-memory bandwidth again plus swizzled addresses and a proxy fence; from TMEM it takes N / 2 clocks, and a
// thread stores its row's 64 columns with one tcgen05.st of 32 registers.
//
// Work split: a launch covers one or several linears, one CTA per SM.  With T row tiles of equal length for G CTAs every CTA
// takes floor(T / G) whole tiles; the blocks of the remaining tiles are cut into G equal contiguous shares, which go first.
// A whole tile is written to y directly; the parts of a shared tile are added in the handle's binary32 workspace (under the
// whole tiles' work) and the CTA that delivers the last block rounds them.  Rows of fewer than sixteen blocks are not cut
// (the adds' order would be free for little gain).  A (gate, up) pair goes through the workspace throughout; the CTA that
// delivers the last block of the two tiles applies the gated unit.
//
// Roles (768 threads): warp 0 packed blocks (TMA), warp 3 x tiles (TMA), warps 1 and 2 MMA issuers, four groups of four
// decode warps (thread = row, groups take every fourth block), four epilogue warps, which
// the decode warps join for a CTA's last piece (nothing else is left to do then; with 100 tokens four warps took 12 us).  One issuer needs about 500 clocks per
// block beside the decode warps that share its scheduler (two waits, eight instructions with their operands, a commit), so
// blocks alternate between two, each with an accumulator of its own; up to 64 tokens there are two such pairs, and one is
// drained while the other is being filled.  Rings, each with full / empty barriers: packed blocks, x tiles (one block: two
// 64-column tiles of N rows), A slots (one block: 64 TMEM columns).  A wait by parity has to follow its barrier phase by
// phase: A slots belong to one decode group and one issuer, x slots to one issuer; a packed slot is waited on by different
// groups in turn, but its length is even, so that its blocks share an issuer (the argument is at ts_rings, bpdq_rings.h).
// Bound: the pipe that executes byte-permutes, masks and
// shifts (half rate): 220 to 300 of its instructions per lane and block.
using bpdq::kTsGroups;
using bpdq::kTsSmem;
constexpr int kTsDecodeWarps = 4 * kTsGroups, kTsFirstDecode = 4, kTsFirstEpi = kTsFirstDecode + kTsDecodeWarps;
constexpr int kTsThreads = 32 * (kTsFirstEpi + 4);
constexpr int kTsACols = 64 * kTsGroups;              // A slots: one per decode group
constexpr int kTsJoint = 32 * (kTsDecodeWarps + 4);    // threads that drain a CTA's last piece
constexpr int kTsMaxM = 128;

struct TsLinear {
    CUtensorMap x_map;         // [M][in], boxes of N rows x 64 columns
    const CUtensorMap* maps;   // planes and coefficients of one 128-row x 128-column block
    __half* y;                 // [M][out]
    float* ws;                 // [M][out] binary32, zero between calls
    unsigned* counters;        // blocks delivered per 128-row tile, zero between calls (a pair: the gate's)
    const float* conv_a;       // a pair: the gate's and the up projection's sums
    float* conv_b;             // null unless paired
    const __half* bias_a;      // binary16 [out] added before the rounding, or null
    const __half* bias_b;
    int out, nblocks, gsh;     // rows, 128-column blocks per row, log2(group / 64)
    int u_begin;               // first unit: (row tile, block) pairs of all linears, tile by tile
};
struct TsParams {
    TsLinear lin[BPDQ_BATCH_MAX];
    int n, M, cols;            // linears; tokens; token columns of the operand (M rounded up to 16)
    int* status;
    int whole, nb0;            // whole tiles per CTA and their length; units before the shared ones: whole * CTAs * nb0
    int cut_begin, cut_units;  // the units that are cut into equal shares ...
    int cut_step;              // ... of whole multiples of this many (a row's blocks when rows are not cut)
    int sp, sx;                // slots of the packed and of the x ring
    int nbuf, dcols;           // accumulator pairs; TMEM columns of one accumulator
};
// A CTA's work as pieces of row tiles: its share of the cut units, then its whole tiles.
struct TsPieces {
    int u, end, f;
};
struct TsPiece {
    int li, tile, b0, n;
};
__device__ __forceinline__ int ts_share(const TsParams& p, int s) {
    return p.cut_begin + (int)((long long)(p.cut_units / p.cut_step) * s / gridDim.x) * p.cut_step;
}
__device__ __forceinline__ TsPieces ts_pieces(const TsParams& p) { return {ts_share(p, blockIdx.x), ts_share(p, blockIdx.x + 1), 0}; }
__device__ __forceinline__ bool ts_next(const TsParams& p, TsPieces& w, TsPiece& c) {
    if (w.u >= w.end) {
        if (w.f >= p.whole) return false;
        w.u = ((int)blockIdx.x + (int)gridDim.x * w.f) * p.nb0;
        w.end = w.u + p.nb0;
        ++w.f;
    }
    c.li = 0;
    while (c.li + 1 < p.n && w.u >= p.lin[c.li + 1].u_begin) ++c.li;
    const int nblocks = p.lin[c.li].nblocks, rel = w.u - p.lin[c.li].u_begin;
    c.tile = rel / nblocks;
    c.b0 = rel - c.tile * nblocks;
    c.n = min(nblocks - c.b0, w.end - w.u);
    w.u += c.n;
    return true;
}

template <int K> struct TsCfg {
    static constexpr int kPlaneBytes = bpdq::ts_plane_bytes(K), kCoefBytes = bpdq::ts_coef_bytes(K);
    static constexpr int kSlotBytes = bpdq::ts_slot_bytes(K);
};

__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void umma_f16_ts(unsigned d, unsigned a, uint64_t bdesc, unsigned idesc, unsigned accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d), "r"(a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st32(unsigned t, const unsigned (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(t), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]),
          "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]),
          "r"(v[30]), "r"(v[31]) : "memory");
}

// NG: coefficient groups per block, 1 or 2 (as a parameter of the launch, beside a packed slot that was advanced step by step, it cost 2 to 4 %: 18944 x 3584 at K = 2
// with 24 tokens 13.8 us and 13.3, K = 3 15.1 and 14.7, K = 4, g = 64 25.2 and 24.2)
template <int K, int NG>
__global__ void __launch_bounds__(kTsThreads, 1) gemm_ts_kernel(const __grid_constant__ TsParams p) {
    using C = TsCfg<K>;
    constexpr int NA = kTsGroups;
    extern __shared__ unsigned char smem_raw[];
    const unsigned base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
    const int SP = p.sp, SX = p.sx, N = p.cols;
    const unsigned xbytes = (unsigned)N * 256u;                    // one block of x: two tiles of N rows x 128 bytes
    const unsigned x_base = base, p_base = base + (unsigned)SX * xbytes;
    const unsigned bar_off = (unsigned)SX * xbytes + (unsigned)SP * C::kSlotBytes;
    const unsigned bar_base = base + bar_off;
    auto full_a = [&](int s) { return bar_base + 8u * s; };
    auto empty_a = [&](int s) { return bar_base + 8u * (NA + s); };
    const unsigned acc_full = bar_base + 16u * NA, acc_empty = acc_full + 16u;      // two each
    const unsigned full_x0 = acc_empty + 16u, empty_x0 = full_x0 + 8u * SX, full_p0 = empty_x0 + 8u * SX, empty_p0 = full_p0 + 8u * SP;
    const int nbars = 2 * NA + 4 + 2 * SX + 2 * SP;
    unsigned* tmem_slot = reinterpret_cast<unsigned*>(smem + bar_off + 8 * nbars);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* finish = reinterpret_cast<volatile int*>(tmem_slot + 2);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    TsPieces work = ts_pieces(p);
    TsPiece pc;

    if (tid == 0) {
        for (int s = 0; s < NA; ++s) { mbar_init(full_a(s), 4); mbar_init(empty_a(s), 1); }
        for (int s = 0; s < 2; ++s) { mbar_init(acc_full + 8u * s, 2); mbar_init(acc_empty + 8u * s, 4); }
        for (int s = 0; s < SX; ++s) { mbar_init(full_x0 + 8u * s, 1); mbar_init(empty_x0 + 8u * s, 1); }
        for (int s = 0; s < SP; ++s) { mbar_init(full_p0 + 8u * s, 1); mbar_init(empty_p0 + 8u * s, 4); }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // only now: a CTA of the next kernel that took this SM's TMEM first and then waited for this kernel would keep it
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned tmem = *tmem_slot, tmem_d = tmem + kTsACols;
    const unsigned quad_lanes = (unsigned)((warp & 3) * 32) << 16;     // TMEM lane quadrant this warp may access

    // ---- a finished piece: thread = row.  A whole tile goes to y, a part of one (or of a pair) into the workspace.  `parts`
    // sets of four warps share the token columns; this thread belongs to set `part` and is number et of all ----
    auto drain = [&](const TsPiece& c, const int seq, const int buf, const bool ok, const int part, const int parts, const int et) {
        // (local copies: the compiler would load launch parameters again behind every store)
        const TsLinear& L = p.lin[c.li];
        const int rl = (warp & 3) * 32 + lane, M = p.M, out = L.out, nblocks = L.nblocks;
        float* const ws = L.ws;
        float* const conv_b = L.conv_b;
        __half* const y = L.y;
        unsigned* const counter = L.counters + c.tile;
        const bool whole = c.n == nblocks, pair = conv_b != nullptr;
        const int row0 = c.tile * 128, r = row0 + rl;
        const bool row_ok = r < out;
        const float br = (whole && !pair && row_ok && L.bias_a) ? __half2float(L.bias_a[r]) : 0.f;
        // a part of one block has one issuer's sum only: it is taken for both and halved (exactly)
        const float half = c.n > 1 ? 1.f : 0.5f;
        const unsigned d = tmem_d + quad_lanes + (unsigned)(2 * buf * p.dcols);
        const unsigned d_first = c.n > 1 ? d : d + (unsigned)((seq & 1) * p.dcols), d_second = c.n > 1 ? d + (unsigned)p.dcols : d_first;
        size_t at = (size_t)r + (size_t)(16 * part) * out;
#pragma unroll 1
        for (int c0 = 16 * part; c0 < N && ok; c0 += 16 * parts, at += (size_t)(16 * parts) * out) {
            unsigned v[16], v2[16];
            tmem_ld16(d_first + (unsigned)c0, v);
            tmem_ld16(d_second + (unsigned)c0, v2);
            tmem_ld_wait();
            if (row_ok) {
                const int nt = M - c0;                   // tokens left
                float* wp = ws + at;
                if (!whole) {
#pragma unroll
                    for (int j = 0; j < 16; ++j, wp += out)
                        if (j < nt) asm volatile("red.global.add.f32 [%0], %1;" ::"l"(wp), "f"((__uint_as_float(v[j]) + __uint_as_float(v2[j])) * half));
                } else if (pair) {
#pragma unroll
                    for (int j = 0; j < 16; ++j, wp += out)
                        if (j < nt) __stcg(wp, (__uint_as_float(v[j]) + __uint_as_float(v2[j])) * half);
                } else {
                    __half* yp = y + at;
#pragma unroll
                    for (int j = 0; j < 16; ++j, yp += out)
                        if (j < nt) *yp = __float2half_rn((__uint_as_float(v[j]) + __uint_as_float(v2[j])) * half + br);
                }
            }
        }
        tc_fence_before();
        __syncwarp();
        if (parts == 1 && lane == 0) mbar_arrive(acc_empty + 8u * buf);   // (nothing follows the last piece)
        if (!whole || pair) {
            __threadfence();                             // this thread's parts are out before the tile's counter moves
            bar_sync(1, 128 * parts);
            if (et == 0) {
                const unsigned before = atomicAdd(counter, (unsigned)c.n);
                *finish = before + (unsigned)c.n == (unsigned)(pair ? 2 * nblocks : nblocks);
                if (*finish) *counter = 0u;
            }
            bar_sync(1, 128 * parts);
            if (*finish) {                               // the last part of the tile: finish it, write y, zero the workspace
                __threadfence();
                // a thread keeps its four rows and walks over the tokens
                const int q = row0 + (et & 31) * 4;
                float* const conv_a = const_cast<float*>(L.conv_a);
                const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                float4 ba = zero, bb = zero;
                if (q < out && L.bias_a) ba = bpdq::bias_quad(L.bias_a, q);
                if (q < out && L.bias_b) bb = bpdq::bias_quad(L.bias_b, q);
                constexpr int kAhead = 4;
                const int step = 4 * parts;
                for (int t0 = et >> 5; q < out && t0 < M; t0 += step * kAhead) {
                    float4 v[kAhead], vb[kAhead];
#pragma unroll
                    for (int e = 0; e < kAhead; ++e)
                        if (t0 + step * e < M) {
                            v[e] = __ldcg(reinterpret_cast<const float4*>(conv_a + (size_t)(t0 + step * e) * out + q));
                            if (pair) vb[e] = __ldcg(reinterpret_cast<const float4*>(conv_b + (size_t)(t0 + step * e) * out + q));
                        }
#pragma unroll
                    for (int e = 0; e < kAhead; ++e)
                        if (t0 + step * e < M) {
                            const size_t to = (size_t)(t0 + step * e) * out + q;
                            float4 a = make_float4(v[e].x + ba.x, v[e].y + ba.y, v[e].z + ba.z, v[e].w + ba.w);
                            if (pair) {
                                a.x = bpdq::silu_f32(a.x) * (vb[e].x + bb.x); a.y = bpdq::silu_f32(a.y) * (vb[e].y + bb.y);
                                a.z = bpdq::silu_f32(a.z) * (vb[e].z + bb.z); a.w = bpdq::silu_f32(a.w) * (vb[e].w + bb.w);
                                __stcg(reinterpret_cast<float4*>(conv_b + to), zero);
                            }
                            const __half2 h01 = __floats2half2_rn(a.x, a.y), h23 = __floats2half2_rn(a.z, a.w);
                            uint2 o;
                            o.x = *reinterpret_cast<const unsigned*>(&h01);
                            o.y = *reinterpret_cast<const unsigned*>(&h23);
                            *reinterpret_cast<uint2*>(y + to) = o;
                            __stcg(reinterpret_cast<float4*>(conv_a + to), zero);
                        }
                }
            }
            bar_sync(1, 128 * parts);                    // *finish has been read by all
        }
    };
    if (warp == 0) {
        // ---------------- packed blocks ----------------
        if (elect_one()) {
            int sl = 0;
            unsigned ph = 1u;
            bool ok = true;
            while (ok && ts_next(p, work, pc)) {
                const CUtensorMap* maps = p.lin[pc.li].maps;
                const int gsh = p.lin[pc.li].gsh;
                for (int b = pc.b0; b < pc.b0 + pc.n; ++b) {
                    if (!mbar_wait(empty_p0 + 8u * sl, ph, abort_flag, p.status)) { ok = false; break; }
                    const unsigned dst = p_base + (unsigned)sl * C::kSlotBytes, bar = full_p0 + 8u * sl;
                    mbar_expect_tx(bar, (unsigned)(C::kPlaneBytes + NG * C::kCoefBytes));
                    tma_load_2d(dst, &maps[0], pc.tile * 256, b * K, bar);                    // 8-byte elements: two per row
                    tma_load_2d(dst + C::kPlaneBytes, &maps[1], pc.tile * 32, ((2 * b) >> gsh) * (K + 1), bar);
                    if (++sl == SP) { sl = 0; ph ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp == 3) {
        // ---------------- x tiles ----------------
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (elect_one()) {
            int sl = 0;
            unsigned ph = 1u;
            bool ok = true;
            while (ok && ts_next(p, work, pc)) {
                const CUtensorMap* map = &p.lin[pc.li].x_map;
                for (int b = pc.b0; b < pc.b0 + pc.n; ++b) {
                    if (!mbar_wait(empty_x0 + 8u * sl, ph, abort_flag, p.status)) { ok = false; break; }
                    const unsigned dst = x_base + (unsigned)sl * xbytes, bar = full_x0 + 8u * sl;
                    mbar_expect_tx(bar, xbytes);
                    tma_load_2d(dst, map, b * 128, 0, bar);
                    tma_load_2d(dst + xbytes / 2, map, b * 128 + 64, 0, bar);
                    if (++sl == SX) { sl = 0; ph ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp <= 2) {
        // ---------------- MMA issuers: blocks alternate between the two, each adds into an accumulator of its own ----------------
        const int me = warp - 1;
        const unsigned idesc = instr_desc_f16(BM, N);
        int sx = 0, sa = 0, buf = 0;
        unsigned px = 0u, pa = 0u, pacc = 1u;
        bool ok = true;
        while (ok && ts_next(p, work, pc)) {
            const unsigned d = tmem_d + (unsigned)((2 * buf + me) * p.dcols);
            ok = mbar_wait_warp(acc_empty + 8u * buf, pacc, abort_flag, p.status);
            unsigned more = 0u;                          // this issuer has begun its sum
            for (int k = 0; k < pc.n && ok; ++k) {
                if ((sa & 1) == me) {
                    ok = mbar_wait_warp(full_x0 + 8u * sx, px, abort_flag, p.status) && mbar_wait_warp(full_a(sa), pa, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t d0 = smem_desc_sw128(x_base + (unsigned)sx * xbytes), d1 = d0 + (xbytes >> 5);
                    const unsigned a = tmem + (unsigned)(sa * 64);
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < 8; ++kk)
                            umma_f16_ts(d, a + kk * 8, (kk < 4 ? d0 : d1) + 2u * (kk & 3), idesc, kk == 0 ? more : 1u);
                        umma_commit(empty_a(sa));
                        umma_commit(empty_x0 + 8u * sx);
                    }
                    __syncwarp();
                    more = 1u;
                }
                if (++sx == SX) { sx = 0; px ^= 1u; }
                if (++sa == NA) { sa = 0; pa ^= 1u; }
            }
            if (ok && elect_one()) umma_commit(acc_full + 8u * buf);
            __syncwarp();
            if (++buf == p.nbuf) { buf = 0; pacc ^= 1u; }
        }
    } else if (warp >= kTsFirstDecode && warp < kTsFirstEpi) {
        // ---------------- decode warps: thread = row of the tile ----------------
        const int wg = (warp - kTsFirstDecode) >> 2, rl = (warp & 3) * 32 + lane;
        const unsigned wrot = (unsigned)(rl >> 2) & 3u, sh = (unsigned)(rl & 3) * 8u;
        unsigned off[4];                                 // logical word k takes the bytes of physical words k - wrot and k - wrot - 1
#pragma unroll
        for (unsigned k = 0; k < 4; ++k) off[k] = p_base + (unsigned)rl * 16u + (((k - wrot) & 3u) << 2);
        const unsigned slot = tmem + quad_lanes + (unsigned)(wg * 64);
        int sl = wg % SP;
        unsigned ph = (unsigned)(wg / SP) & 1u, pa = 1u;
        const int nblk = work.end - work.u + p.whole * p.nb0;
        for (int q = wg; q < nblk; q += kTsGroups) {
            if (!mbar_wait_warp(full_p0 + 8u * sl, ph, abort_flag, p.status)) break;
            const unsigned so = (unsigned)sl * C::kSlotBytes;
            unsigned a[K][4];
#pragma unroll
            for (int i = 0; i < K; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a[i][j]) : "r"(so + i * 2048 + off[j]));
            bpdq::ByteTables<K> tab;
            bool ok = true;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (half == 0 || NG == 2) {              // candidate tables of the coefficient group that starts here
                    float c[K + 1];
#pragma unroll
                    for (int i = 0; i <= K; ++i) {
                        unsigned short hb;
                        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(hb) : "r"(p_base + so + C::kPlaneBytes + (half * (K + 1) + i) * 256 + rl * 2));
                        c[i] = __half2float(__ushort_as_half(hb));
                    }
                    bpdq::candidate_byte_tables<K>(c, tab);
                }
                unsigned v[32];
#pragma unroll
                for (int wd = 0; wd < 2; ++wd) {
                    const int k = 2 * half + wd;
                    unsigned w[K], sel[4];
#pragma unroll
                    for (int i = 0; i < K; ++i) w[i] = __funnelshift_l(a[i][(k + 3) & 3], a[i][k], sh);
                    bpdq::code_nibbles_word<K>(w, sel);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint4 d = bpdq::decode8<K>(sel[e], tab);
                        v[16 * wd + 4 * e] = d.x; v[16 * wd + 4 * e + 1] = d.y; v[16 * wd + 4 * e + 2] = d.z; v[16 * wd + 4 * e + 3] = d.w;
                    }
                }
                if (half == 0) {
                    ok = mbar_wait_warp(empty_a(wg), pa, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                }
                tmem_st32(slot + (unsigned)(half * 32), v);
            }
            if (!ok) break;
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(full_a(wg));
                mbar_arrive(empty_p0 + 8u * sl);         // everything read from the slot has been stored as an operand
            }
            pa ^= 1u;
            sl += kTsGroups;                             // (the ring is longer)
            if (sl >= SP) { sl -= SP; ph ^= 1u; }
        }
    } else if (warp >= kTsFirstEpi) {
        // ---------------- epilogue warps: every piece, the last one together with the decode warps ----------------
        asm volatile("griddepcontrol.wait;" ::: "memory");
        int buf = 0, seq = 0;                            // seq: blocks before this piece
        unsigned pacc = 0u;
        bool more = ts_next(p, work, pc);
        while (more) {
            const bool ok = mbar_wait_warp(acc_full + 8u * buf, pacc, abort_flag, p.status);
            tc_fence_after();
            const TsPiece now = pc;
            more = ts_next(p, work, pc);
            if (!more) {
                if (tid == 32 * kTsFirstEpi) *finish = ok;
                tc_fence_before();
                bar_sync(2, kTsJoint);
                tc_fence_after();
            }
            drain(now, seq, buf, ok, more ? 0 : kTsGroups, more ? 1 : kTsGroups + 1, tid - 32 * (more ? kTsFirstEpi : kTsFirstDecode));
            if (++buf == p.nbuf) { buf = 0; pacc ^= 1u; }
            seq += now.n;
        }
    }
    if (warp >= kTsFirstDecode && warp < kTsFirstEpi) {
        // the last piece: the epilogue warps have waited for its sums (barrier 2), twenty warps read them
        asm volatile("griddepcontrol.wait;" ::: "memory");
        int buf = -1, seq = 0, n = 0;
        TsPiece last = {0, 0, 0, 0};
        while (ts_next(p, work, pc)) {
            seq += n;
            last = pc;
            n = pc.n;
            buf = buf + 1 == p.nbuf ? 0 : buf + 1;
        }
        if (n > 0) {
            bar_sync(2, kTsJoint);
            const bool ok = *finish != 0;
            tc_fence_after();
            drain(last, seq, buf, ok, (warp - kTsFirstDecode) >> 2, kTsGroups + 1, tid - 32 * kTsFirstDecode);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    if (*abort_flag) linger();
}
