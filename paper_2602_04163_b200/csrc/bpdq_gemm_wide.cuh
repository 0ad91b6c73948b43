// Included by bpdq_gemm.cu (inside its unnamed namespace, after the PTX wrappers): the prefill kernel for many tokens.
//
// gemm_wide_kernel: one decoded weight stage feeds a token tile of two halves (of up to 256 tokens each), so a weight is decoded once per tile:
// the decode's energy is what the 1 kW cap charges (every further plane costs 8-20 %).  The two halves of TMEM's 512 columns are accumulators.
// Halves above 128 tokens: two warps issue, each multiplies every stage with its own half of x into an accumulator of its own.  Up to
// 128: one issuer multiplies with the whole tile, and tiles alternate between the accumulators, so that one is drained while the other
// fills.  (An MMA reads 4 KB of A from shared memory: two of 80 tokens take 2 x 52 clocks of the pipe where one of 160 takes 80.  The pipe is not what
// bounds that tile: 3584 x 18944 with 777 tokens, K = 2, went from 94.6 to 92.2 us, and a block still takes 980 clocks for 640 of MMAs, the rest
// being the two decode groups' chain and hand-over.  Where drains overlap it gives more: K = 2, halves of 128, 8192 x 8192 with 4096 tokens 3 %,
// 20480 x 1024 with 512 tokens 9 %.)  Above, TMEM is full with
// one tile, so the epilogue does not overlap the next tile's MMAs (about 3 % of a 72B-shaped tile's time); producer and decode warps run
// ahead into the next tile's stages meanwhile.
//
// Stages are 64 columns (128-byte swizzle rows) while four of them fit, i.e. for halves of up to 128 tokens, else 32 columns
// (64-byte rows: five stages of the widest tile): a stage costs its issuers about 330 clocks beside the decode warps that
// share their schedulers, a block of four 32-column ones 1320, which is more than the MMAs of halves below 160 tokens take.
// Packed 128-column blocks (two tensor-map boxes each) come in a ring of two to eight.  Roles (640 threads, 896 with four decode
// groups): warps 0 and 3 producers (x, packed), warps 1-2 MMA issuers, two or four decode groups of four warps (thread =
// output row, taking 128-column blocks of the stage sequence in turn, which continues across tiles), eight epilogue warps (four
// per half).  Barriers per stage: full (both x halves' bytes and one arrival per warp of the owning decode group), one or
// two that release it in turn (one tcgen05.commit per issuer); per packed slot: full_p, empty_p; acc_full (one commit per issuer), acc_empty (one arrival per
// epilogue warp).  All waits are bounded.
using bpdq::kWideMaxHalf;
using bpdq::kWideLongHalf;
using bpdq::kWideSmem;
constexpr int kWideEpiWarps = 8;
constexpr int kWideFirstDecode = 4;

struct WideParams {
    GemmParams g;
    int half;                  // tokens of a half tile, a multiple of 16
    int stages, sp;            // slots of the stage ring and of the packed ring
};

// BKW: columns per stage, 32 (64-byte swizzle rows) or 64 (128-byte ones).  NG: decode groups (wide_groups, bpdq_rings.h).
template <int K, int BKW, int NG> struct WideCfg {
    static constexpr int kATile = BM * BKW * 2;                // 8 or 16 KB
    static constexpr int kPerBlock = 128 / BKW;                // stages per packed block
    static constexpr int kGroups = NG;                         // decode groups; they take blocks in turn
    static constexpr int kFirstEpi = kWideFirstDecode + 4 * kGroups, kThreads = 32 * (kFirstEpi + kWideEpiWarps);
    static constexpr bool kWhole = BKW == 64;                  // a MMA takes the whole token tile (two halves of up to 128)
    static constexpr int kIssuers = kWhole ? 1 : 2;
    static constexpr int kReleases = bpdq::wide_releases(NG);  // release barriers of a stage slot
    static constexpr int kAccs = kWhole ? 2 : 1;               // accumulator barrier sets, which tiles take in turn
    static constexpr int kPlaneBytes = bpdq::wide_plane_bytes(K), kCoefBytes = bpdq::wide_coef_bytes(K);
    static constexpr int kBlockBytes = bpdq::wide_block_bytes(K);
    static_assert(kATile == bpdq::wide_a_bytes(BKW), "bytes of a stage's weights");
};

// Shared-memory matrix descriptor of a K-major tile with 64-byte swizzle whose rows are 64 bytes apart: start address
// / 16, leading byte offset (unused by swizzled K-major layouts) 1, stride byte offset 512 / 16 (distance between
// 8-row groups), descriptor version 1, layout type 4 (64-byte swizzle) in bits 61..63.
__device__ __forceinline__ uint64_t smem_desc_sw64(unsigned addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

template <int K, int BKW, int NG>
__global__ void __launch_bounds__(WideCfg<K, BKW, NG>::kThreads, 1)
gemm_wide_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap planes_map,
                 const __grid_constant__ CUtensorMap coefs_map, const WideParams wp) {
    const GemmParams& p = wp.g;
    using C = WideCfg<K, BKW, NG>;
    constexpr int kPerBlock = C::kPerBlock;
    constexpr bool kWhole = C::kWhole;
    const int S = wp.stages, SP = wp.sp, half = wp.half;
    const unsigned bhalf = (unsigned)half * (BKW * 2), stage = C::kATile + 2u * bhalf;
    extern __shared__ unsigned char smem_raw[];
    const unsigned base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
    const unsigned st_base = base;                                 // S x (A tile, x half 0, x half 1)
    const unsigned p_base = st_base + (unsigned)S * stage;              // SP x packed block
    const unsigned bar_base = p_base + SP * C::kBlockBytes;
    auto full = [&](int s) { return bar_base + 8u * s; };
    // a stage slot's release: uses n = 0, 1, ... of a slot take its R barriers in turn (wide_releases, bpdq_rings.h)
    constexpr int R = C::kReleases;
    auto empty = [&](int s, int n) { return bar_base + 8u * (S + R * s + (n & (R - 1))); };
    auto released = [&](int s, int n) { return empty(s, n - 1); };           // what use n waits for
    auto released_parity = [&](int n) { return (unsigned)((n - 1) >> (R - 1)) & 1u; };
    auto full_p = [&](int s) { return bar_base + 8u * ((1 + R) * S + s); };
    auto empty_p = [&](int s) { return bar_base + 8u * ((1 + R) * S + SP + s); };
    // an accumulator's barriers: one set of both halves' (kIssuers commits), or two that tiles j = 0, 1, ... take in turn
    auto acc_full = [&](int j) { return bar_base + 8u * ((1 + R) * S + 2 * SP + j % C::kAccs); };
    auto acc_empty = [&](int j) { return acc_full(j) + 16u; };
    auto acc_parity = [&](int j) { return (unsigned)(j / C::kAccs) & 1u; };
    unsigned* tmem_slot = reinterpret_cast<unsigned*>(smem + (bar_base - base) + 8 * ((1 + R) * S + 2 * SP + 4));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int nkb = p.in / BKW;                  // stages per tile
    const int nblk = p.in / 128;                     // packed blocks per tile (two or four stages each)
    const int nrt = (p.out + BM - 1) / BM;
    const int ntt = (p.M + 2 * half - 1) / (2 * half);
    const int ntiles = nrt * ntt;
    const int ng = p.group == 64 ? 2 : 1;

    if (tid == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full(s), 1 + 4);                   // the producer (with both x halves' bytes) and four decode warps
            for (int n = 0; n < R; ++n) mbar_init(empty(s, n), C::kIssuers);
        }
        for (int s = 0; s < SP; ++s) { mbar_init(full_p(s), 1); mbar_init(empty_p(s), 4); }
        for (int j = 0; j < C::kAccs; ++j) { mbar_init(acc_full(j), C::kIssuers); mbar_init(acc_empty(j), kWideEpiWarps); }   // a live barrier must not be initialised again
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
    const unsigned tmem_d = *tmem_slot;

    if (warp == 0) {
        // ---------------- x tiles of every stage ----------------
        // A thread needs 100 clocks or more per copy, so packed blocks have a producer of their own, and two halves of up to
        // 128 tokens come as one box.
        asm volatile("griddepcontrol.wait;" ::: "memory");   // the kernel before this one may have written x
        if (elect_one()) {
            const int boxes = 2 * half <= 256 ? 1 : 2;
            int s = 0, n = 0;                            // stage slot and its use, continuing across tiles
            bool ok = true;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int tok0 = (tile / nrt) * (2 * half);
                for (int kb = 0; kb < nkb; ++kb) {
                    if (!mbar_wait(released(s, n), released_parity(n), abort_flag, p.status)) { ok = false; break; }
                    mbar_expect_tx(full(s), 2u * bhalf);
                    const unsigned bdst = st_base + (unsigned)s * stage + C::kATile;
                    tma_load_2d(bdst, &x_map, kb * BKW, tok0, full(s));
                    if (boxes == 2) tma_load_2d(bdst + bhalf, &x_map, kb * BKW, tok0 + half, full(s));
                    if (++s == S) { s = 0; ++n; }
                }
            }
        }
        __syncwarp();
    } else if (warp == 3) {
        // ---------------- packed blocks ----------------
        if (elect_one()) {
            int sp = 0;
            unsigned pp = 1u;
            bool ok = true;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
                const int row0 = (tile % nrt) * BM;
                for (int b = 0; b < nblk; ++b) {
                    if (!mbar_wait(empty_p(sp), pp, abort_flag, p.status)) { ok = false; break; }
                    mbar_expect_tx(full_p(sp), (unsigned)(C::kPlaneBytes + ng * C::kCoefBytes));
                    const unsigned pdst = p_base + sp * C::kBlockBytes;
                    tma_load_2d(pdst, &planes_map, row0 * 2, b * K, full_p(sp));
                    tma_load_2d(pdst + C::kPlaneBytes, &coefs_map, row0 / 4, ((b * 128) / p.group) * (K + 1), full_p(sp));
                    if (++sp == SP) { sp = 0; pp ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp <= 2) {
        // ---------------- MMA issuers: warp 1 + h multiplies every stage with x half h into accumulator h; or warp 1 with all of x ----------------
        // One thread throughout: it has 256 clocks per stage beside the decode warps that share its scheduler, so a stage has
        // one barrier for weights and activations together and nothing in the loop involves the rest of the warp.
        if (warp <= C::kIssuers && elect_one()) {
            const unsigned idesc = instr_desc_f16(BM, kWhole ? 2 * half : half);
            const int h = warp - 1;
            int s = 0, n = 0, j = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++j) {
                // the epilogue must have drained the accumulators of the tile before
                if (!mbar_wait(acc_empty(j), acc_parity(j) ^ 1u, abort_flag, p.status)) break;
                const unsigned d = tmem_d + (unsigned)((kWhole ? j & 1 : h) * 256);
                unsigned more = 0u;
                for (int kb = 0; kb < nkb; ++kb) {
                    ok = mbar_wait(full(s), (unsigned)n & 1u, abort_flag, p.status);
                    if (!ok) break;
                    tc_fence_after();
                    const unsigned a_addr = st_base + (unsigned)s * stage;
                    const unsigned b_addr = a_addr + C::kATile + (kWhole ? 0u : (unsigned)h * bhalf);
                    const uint64_t adesc = BKW == 32 ? smem_desc_sw64(a_addr) : smem_desc_sw128(a_addr);
                    const uint64_t bdesc = BKW == 32 ? smem_desc_sw64(b_addr) : smem_desc_sw128(b_addr);
#pragma unroll
                    for (int k = 0; k < BKW / 16; ++k)                // 16 columns = 32 bytes further along the swizzled row
                        umma_f16(d, adesc + 2u * k, bdesc + 2u * k, idesc, k == 0 ? more : 1u);
                    umma_commit(empty(s, n));
                    more = 1u;
                    if (++s == S) { s = 0; ++n; }
                }
                if (ok) umma_commit(acc_full(j));
            }
        }
        __syncwarp();
    } else if (warp < C::kFirstEpi) {
        // ---------------- decode warps: thread = output row; groups take blocks in turn ----------------
        const int grp = (warp - kWideFirstDecode) >> 2;
        const int rl = ((warp - kWideFirstDecode) & 3) * 32 + lane;     // row inside the tile; row tiles start at multiples of 128
        unsigned a_off[BKW / 8];                         // swizzled byte offset of each 16-byte chunk of this thread's 64- or 128-byte row
#pragma unroll
        for (int ch = 0; ch < BKW / 8; ++ch)
            a_off[ch] = (unsigned)rl * (BKW * 2u) + (((unsigned)ch ^ (unsigned)(BKW == 32 ? (rl >> 1) & 3 : rl & 7)) << 4);
        const unsigned wrot = (unsigned)(rl >> 2) & 3u, sh = (unsigned)(rl & 3) * 8u;
        unsigned off[4];                                 // logical word k takes the bytes of physical words k - wrot and k - wrot - 1
#pragma unroll
        for (unsigned k = 0; k < 4; ++k) off[k] = p_base + (unsigned)rl * 16u + (((k - wrot) & 3u) << 2);
        // Stage slots are shared by the groups; why their waits by parity are safe stands at wide_rings (bpdq_rings.h).
        const int my_tiles = blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
        int s = 0, sp = grp;
        int n = 0;
        unsigned pp = 0u;
        auto advance = [&](int by) { s += by; while (s >= S) { s -= S; ++n; } };
        advance(kPerBlock * grp);
        bool ok = true;
        const long long nbseq = (long long)my_tiles * nblk;
        for (long long bseq = grp; bseq < nbseq && ok; bseq += C::kGroups) {
            if (!mbar_wait_warp(full_p(sp), pp, abort_flag, p.status)) break;
            const unsigned so = (unsigned)(sp * C::kBlockBytes);
            unsigned a[K][4];
#pragma unroll
            for (int i = 0; i < K; ++i)
#pragma unroll
                for (int k = 0; k < 4; ++k) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a[i][k]) : "r"(so + i * (BM * 16) + off[k]));
            bpdq::ByteTables<K> tab;
#pragma unroll
            for (int st = 0; st < kPerBlock; ++st) {     // the block's stages
                constexpr int kWords = BKW / 32;         // 32-column words per stage
                if (st == 0 || (ng == 2 && st * kWords == 2)) {   // candidate tables of the coefficient group that starts here
                    float c[K + 1];
#pragma unroll
                    for (int i = 0; i <= K; ++i) {
                        unsigned short hb;
                        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(hb) : "r"(p_base + so + C::kPlaneBytes + (st * kWords / 2) * C::kCoefBytes + i * (BM * 2) + rl * 2));
                        c[i] = __half2float(__ushort_as_half(hb));
                    }
                    bpdq::candidate_byte_tables<K>(c, tab);
                }
                uint4 v8[BKW / 8];                       // decode first (nothing of it waits for the slot), then wait and store
#pragma unroll
                for (int e = 0; e < kWords; ++e) {
                    const int q = st * kWords + e;
                    unsigned w[K], sel[4];
#pragma unroll
                    for (int i = 0; i < K; ++i) w[i] = __funnelshift_l(a[i][(q + 3) & 3], a[i][q], sh);
                    bpdq::code_nibbles_word<K>(w, sel);
#pragma unroll
                    for (int u = 0; u < 4; ++u) v8[4 * e + u] = bpdq::decode8<K>(sel[u], tab);
                }
                if (!mbar_wait_warp(released(s, n), released_parity(n), abort_flag, p.status)) { ok = false; break; }
                const unsigned dst = st_base + (unsigned)s * stage;
#pragma unroll
                for (int ch = 0; ch < BKW / 8; ++ch)
                    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst + a_off[ch]),
                                 "r"(v8[ch].x), "r"(v8[ch].y), "r"(v8[ch].z), "r"(v8[ch].w) : "memory");
                fence_proxy_async();                     // make the generic-proxy stores visible to the MMA's reads
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(full(s));                // one arrival per warp, after all its lanes' stores and fences
                    if (st == bpdq::wide_release_stage(kPerBlock)) mbar_arrive(empty_p(sp));   // stored stages have used everything loaded from the packed slot
                }
                advance(1);
            }
            advance(kPerBlock * (C::kGroups - 1));              // the other groups' blocks
            sp += C::kGroups;
            if (sp >= SP) { sp -= SP; pp ^= 1u; }
        }
    } else {
        // ---------------- epilogue warps: four per accumulator ----------------
        const int quad = warp & 3, h = (warp - C::kFirstEpi) >> 2;   // TMEM lane quadrant this warp may access; half
        const int rl = quad * 32 + lane;
        const size_t out = (size_t)p.out;
        asm volatile("griddepcontrol.wait;" ::: "memory");   // ... or may still be reading what y overwrites
        int j = 0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++j) {
            if (!mbar_wait_warp(acc_full(j), acc_parity(j), abort_flag, p.status)) break;
            tc_fence_after();
            const unsigned taddr = tmem_d + ((unsigned)(quad * 32) << 16) + (unsigned)(kWhole ? (j & 1) * 256 + h * half : h * 256);
            const int row0 = (tile % nrt) * BM, tok0 = (tile / nrt) * (2 * half) + h * half;
            const int r = row0 + rl;
            const bool row_ok = r < p.out;
            const float br = (p.bias && row_ok) ? __half2float(p.bias[r]) : 0.f;
            __half* yp = p.y + (size_t)tok0 * out + r;
            const int nt = min(half, p.M - tok0);        // tokens of this half
#pragma unroll 1
            for (int c0 = 0; c0 < nt; c0 += 16) {        // warp-uniform
                unsigned v[16];
                tmem_ld16(taddr + (unsigned)c0, v);
                tmem_ld_wait();
                if (row_ok) {
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj, yp += out)
                        if (c0 + jj < nt) *yp = __float2half_rn(__uint_as_float(v[jj]) + br);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty(j));       // one arrival per epilogue warp: the accumulators may be overwritten
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_d, 512);
    }
    if (*abort_flag) linger();
}
