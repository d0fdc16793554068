// Partitioned attention (Eq. 1), two-CTA form with 64 query rows per CTA, for launches that leave SM pairs idle as units of 256 rows.
//
// A pair of CTAs (cta_group::2) with M = 128 works at the full tensor rate (32 cycles for a 128 x 128 x 16 MMA, half of what M = 256 takes), where
// one CTA with M = 64 works at half of it. Units of 128 rows therefore put twice the SMs to work on the same launch, and a stream's last unit wastes
// at most 127 rows instead of 255. What bounds a tile of 128 keys is its softmax chain, 2070 cycles against 1024 of MMAs and some 1500 of
// shared memory (64 KB of Q and K and 48 KB of P and V that the MMAs read, 64 KB that come in, 16 KB of P). Two groups of softmax warps on alternating
// tiles with an accumulator each brought a tile to 1570 cycles and the fixed part up by 1 to 2 k: no faster at any number of tiles that a launch has here.
//
// Such an accumulator fills all lanes of either CTA: lanes 0-63 hold the CTA's 64 rows for the first half of the columns, lanes 64-127 for the second.
// For S the halves are the two 64-key halves of a tile, for O the two halves of the head dimension. A row has four softmax threads, 32 keys and a quarter of
// O's columns each. P goes through shared memory (as an operand in tensor memory it would have to lie in both lane halves).
//
// Every cluster has one unit. With nsplit > 1 the keys are cut into slices: the pairs of a cluster hold the slices of one unit and merge them
// through distributed shared memory (cluster_merge: 2 or 4 slices; pair q finishes a share of the columns), or the pairs leave fp32 partials for
// the merge kernel. Times and the choice between the forms: pair_choose_splits.
// Included by attn_tc.cu (shares its tile geometry and tensor maps).
#pragma once

namespace reflex {

constexpr int kApRows = 64;
constexpr int kApThreads = 64 + 256;      // producer warp, MMA warp, eight softmax warps

template <int HD> struct ApSmem {
    static constexpr int CH = HD / 64, VCH = CH / 2;
    static constexpr int NKS = HD == 256 ? 2 : 4, NVS = NKS;
    static constexpr uint32_t Q_BYTES = CH * kApRows * 128;           // later the output tile on its way out
    static constexpr uint32_t K_STAGE = CH * 64 * 128;                // 64 keys x head_dim
    static constexpr uint32_t V_STAGE = VCH * 128 * 128;              // 128 keys x head_dim / 2
    static constexpr uint32_t V_HALF = VCH * 64 * 128;
    static constexpr uint32_t P_BUF = 2 * kApRows * 128;              // [key half][64 rows][64 keys]
    static constexpr uint32_t OFF_Q = 0;
    static constexpr uint32_t OFF_K = OFF_Q + Q_BYTES;                // later the inbox of a merge, or the partial tile on its way out
    static constexpr uint32_t OFF_V = OFF_K + NKS * K_STAGE;
    static constexpr uint32_t OFF_P = OFF_V + NVS * V_STAGE;
    static constexpr uint32_t OFF_MAX = OFF_P + 2 * P_BUF;            // [2 buffers][64 rows][4] row maxima
    static constexpr uint32_t OFF_SUM = OFF_MAX + 2 * kApRows * 16;   // [2 accumulators][64 rows][4] row sums
    static constexpr uint32_t OFF_ML = OFF_SUM + 2 * kApRows * 16;    // [4 slices][64 rows] (m, l)
    static constexpr uint32_t OFF_BAR = OFF_ML + 4 * kApRows * 8;
    static constexpr uint32_t TOTAL = OFF_BAR + 256 + 1024;
    static_assert(TOTAL <= 227u * 1024u, "shared memory budget");
    static_assert(NKS * K_STAGE >= kApRows * HD * 4, "inbox / partial tile over the K stages");
    static constexpr int C_QFULL = 0, C_KFULL = 1, C_KEMPTY = C_KFULL + NKS, C_VLAND = C_KEMPTY + NKS, C_VEMPTY = C_VLAND + NVS, C_SFULL = C_VEMPTY + NVS,
                         C_PFULL = C_SFULL + 2, C_PVDONE = C_PFULL + 2, C_MFREE = C_PVDONE + 2, C_INBOX = C_MFREE + 1, C_COUNT = C_INBOX + 1;
    static_assert(8 * C_COUNT + 8 <= 256, "barrier area");
};

// EARLY: inside an expert step, the first cached tiles are asked for ahead of the wait.
// DUAL: even and odd tiles have an accumulator each, with a reference maximum and a sum of its own. The key that sets a reference has weight 1, which
// bf16 holds exactly, and twice as many references are twice as many such keys: 898 keys in four slices 2.24e-3 -> 2.13e-3 from 64 bits, what the eight
// slices of chain_attn_kernel give. Split launches take it, they stand where finer slices stood, and unsplit ones where units of 256 rows would be cut
// into slices; it costs a launch 0.1 to 0.5 us.
template <int HD, bool EARLY, bool DUAL>
__global__ void __launch_bounds__(kApThreads, 1)      // clusters of 2 CTAs, or of 2 * nsplit (cluster_merge)
attn_pair_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                 const __grid_constant__ CUtensorMap tm_kd, const __grid_constant__ CUtensorMap tm_vd, const __grid_constant__ CUtensorMap tm_o, const TcParams p)
{
    using L = ApSmem<HD>;
    constexpr int CH = L::CH, VCH = L::VCH, NKS = L::NKS, NVS = L::NVS;
    constexpr uint32_t kColO = 0, kColS = DUAL ? HD : HD / 2, kTmemCols = kColS + 128 <= 256 ? 256 : 512;       // O: HD / 2 columns an accumulator; S: two buffers of 64
    constexpr int OC = HD / 4;                                           // a thread's columns of O
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    auto bar = [&](int i) -> uint32_t { return base + L::OFF_BAR + 8u * (uint32_t)i; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + L::OFF_BAR + 8 * L::C_COUNT);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t crank = cluster_ctarank();
    const uint32_t rank = crank & 1u, lead = crank & ~1u;                // rank inside the pair; cluster rank of its leader
    const uint16_t pair_mask = (uint16_t)(3u << lead);
    const int pair_id = blockIdx.x >> 1;
    const int ns = p.nsplit, split = pair_id % ns, unit = pair_id / ns;
    const int kvh = (unit / p.n_qtiles) % p.Hkv, b = unit / (p.n_qtiles * p.Hkv);
    const int t0 = (2 * (unit % p.n_qtiles) + (int)rank) * p.tile_tokens;
    const int rows = max(0, min(kApRows, (p.T - t0) * p.G));             // rows of this CTA that exist

    if (threadIdx.x == 0) {
        for (int i = 0; i < L::C_COUNT; ++i)
            mbar_init(bar(i), i == L::C_PFULL || i == L::C_PFULL + 1 ? 16u : i == L::C_MFREE ? (uint32_t)ns : 1u);     // (P: the softmax warps of both CTAs)
        *abort_flag = 0u;
        fence_mbar_init();
        if (p.cluster_merge) mbar_expect_tx(bar(L::C_INBOX), (uint32_t)((ns - 1) * rows) * (uint32_t)(HD / ns * 4 + 8));
        prefetch_tmap(&tm_q); prefetch_tmap(&tm_k); prefetch_tmap(&tm_v); prefetch_tmap(&tm_kd); prefetch_tmap(&tm_vd); prefetch_tmap(&tm_o);
    }
    if (warp == 1) tmem_alloc2(smem_u32((const void *)tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    cluster_arrive();
    cluster_wait();   // all barriers of the cluster exist before anything crosses it
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    if (!(EARLY && warp == 0)) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }

    // ---- geometry: 64-key halves of static prefix, ring and dynamic tokens; this pair's slice of the tiles (two halves each) ----
    TileGeom g;
    {
        const StreamState st = p.state[b];
        g.S = st.static_len > 0 ? st.static_len : 0;
        g.N = p.N; g.T = p.T; g.count = st.count;
        g.oldest = (st.head - st.count) % p.N;
        if (g.oldest < 0) g.oldest += p.N;
        g.ns = (g.S + kBN - 1) / kBN;
        g.nr = g.count > 0 ? (p.N + kBN - 1) / kBN : 0;
        g.nd = (p.T + kBN - 1) / kBN;
        g.row_base = (p.layer * p.B + b) * (p.ring_off + p.N);
        g.s_off = st.bank * p.S_max; g.ring_off = p.ring_off; g.b = b;
    }
    const int H = g.ns + g.nr + g.nd, all_tiles = (H + 1) / 2, per = (all_tiles + ns - 1) / ns;
    const int tile0 = split * per, n = max(0, min(all_tiles, tile0 + per) - tile0);      // (may be empty for the last slices)

    auto wait_slow = [&](int i, uint32_t parity, uint32_t code) -> bool {
        const unsigned long long t_start = globaltimer_ns();
        for (uint32_t k = 1;; ++k) {
            if (mbar_try_wait_cluster(bar(i), parity)) return true;
            if ((k & 255u) == 0u) {
                if (*abort_flag) return false;
                if (globaltimer_ns() - t_start > kWaitNs) break;
            }
        }
        *abort_flag = 1u;
        atomicCAS(p.status, 0u, status_word(kSiteAttnPair + code));
        return false;
    };
    auto wait = [&](int i, uint32_t parity, uint32_t code) -> bool { return mbar_try_wait(bar(i), parity) || wait_slow(i, parity, code); };

    if (warp == 0) {
        // ---------------- TMA producer (both CTAs) ----------------
        if (lane == 0) {
            bool ok = true;
            auto issue_k = [&](int j) {
                const int st = j % NKS, h0 = 2 * (tile0 + j), h = h0 + (int)rank;
                if (j >= NKS) ok = ok && wait(L::C_KEMPTY + st, (uint32_t)(j / NKS - 1) & 1u, 1);
                if (!ok) return;
                if (rank == 0) mbar_expect_tx(bar(L::C_KFULL + st), (h0 + 1 < H ? 2u : 1u) * L::K_STAGE);
                if (h < H) {
                    const TileRef tr = g.decode(h);
                    for (int c = 0; c < CH; ++c)
                        tma2_load_3d(base + L::OFF_K + st * L::K_STAGE + c * (64 * 128), tr.dyn ? &tm_kd : &tm_k, bar(L::C_KFULL + st) & kPeerBitMask, c * 64, kvh, tr.row0);
                }
            };
            auto issue_v = [&](int j) {
                const int st = j % NVS, h0 = 2 * (tile0 + j);
                if (j >= NVS) ok = ok && wait(L::C_VEMPTY + st, (uint32_t)(j / NVS - 1) & 1u, 2);
                if (!ok) return;
                mbar_expect_tx(bar(L::C_VLAND + st), (h0 + 1 < H ? 2u : 1u) * L::V_HALF);
                for (int h = h0; h <= h0 + 1 && h < H; ++h) {
                    const TileRef tr = g.decode(h);
                    for (int c = 0; c < VCH; ++c)
                        tma_load_3d(base + L::OFF_V + st * L::V_STAGE + c * (128 * 128) + (h & 1) * (64 * 128), tr.dyn ? &tm_vd : &tm_v, bar(L::C_VLAND + st),
                                    ((int)rank * VCH + c) * 64, kvh, tr.row0);
                }
            };
            int ahead = 0;                 // tiles that lie in the cached regions altogether and fit the stages
            if constexpr (EARLY) {
                ahead = max(0, min(min(NKS, n), (g.ns + g.nr) / 2 - tile0));
                for (int j = 0; j < ahead; ++j) { issue_k(j); issue_v(j); }
                asm volatile("griddepcontrol.wait;" ::: "memory");
            }
            if (n > 0) {
                if (rank == 0) mbar_expect_tx(bar(L::C_QFULL), 2 * L::Q_BYTES);
                for (int c = 0; c < CH; ++c)
                    tma2_load_4d(base + L::OFF_Q + c * (kApRows * 128), &tm_q, bar(L::C_QFULL) & kPeerBitMask, c * 64, kvh * p.G, t0, b);
            }
            // K runs one tile ahead of V, in the order in which the tensor pipe frees their stages: Q K^T 0, 1, P V 0, Q K^T 2, ...
            if (n > 0 && ahead < 1) issue_k(0);
            for (int j = 0; j < n && ok; ++j) {
                if (j + 1 < n && j + 1 >= ahead) issue_k(j + 1);
                if (j >= ahead) issue_v(j);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA; the warp stays converged, one elected lane issues) ----------------
        // Q K^T of tile j + 1 is issued ahead of P V of tile j. One thread's MMAs run in order, so the logits of tile j exist only once P V of tile
        // j - 2 is complete: its P buffer may then be written again.
        if (rank == 0 && n > 0) {
            constexpr uint32_t idesc_qk = umma_idesc_bf16(2 * kApRows, 128, false), idesc_pv = umma_idesc_bf16(2 * kApRows, HD, true);
            auto qk = [&](int j) -> bool {
                const int st = j % NKS, buf = j & 1;
                if (!wait(L::C_KFULL + st, (uint32_t)(j / NKS) & 1u, 3)) return false;
                tc_fence_after();
                uint64_t qd = umma_desc_sw128(base + L::OFF_Q, 16, 1024), kd = umma_desc_sw128(base + L::OFF_K + st * L::K_STAGE, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < HD / 16; ++kk) {
                    umma2_ss_elect(tmem + kColS + buf * 64, qd, kd, idesc_qk, kk > 0 ? 1u : 0u);
                    umma_desc_advance(qd, (kk & 3) == 3 ? kApRows * 128 - 96 : 32);      // 16 columns on: inside a 64-column chunk, or to the next
                    umma_desc_advance(kd, (kk & 3) == 3 ? 64 * 128 - 96 : 32);
                }
                umma2_commit_mc_elect(bar(L::C_KEMPTY + st), pair_mask);
                umma2_commit_mc_elect(bar(L::C_SFULL + buf), pair_mask);
                return true;
            };
            bool ok = wait(L::C_QFULL, 0u, 4) && qk(0);
            for (int j = 0; j < n && ok; ++j) {
                const int st = j % NVS, buf = j & 1;
                if (j + 1 < n) { ok = qk(j + 1); if (!ok) break; }
                ok = wait(L::C_PFULL + buf, (uint32_t)(j >> 1) & 1u, 5);
                if (!ok) break;
                tc_fence_after();
                uint64_t vd = umma_desc_sw128(base + L::OFF_V + st * L::V_STAGE, 128 * 128, 1024);
                uint64_t pd = umma_desc_sw128(base + L::OFF_P + buf * L::P_BUF, 16, 1024);
                // (a second half past the last key: its P was never written, its V never loaded)
                const int ksteps = 2 * (tile0 + j) + 1 < H ? 8 : 4;
#pragma unroll 4
                for (int kk = 0; kk < ksteps; ++kk) {
                    umma2_ss_elect(tmem + kColO + (DUAL ? buf * (HD / 2) : 0), pd, vd, idesc_pv, (j > (DUAL ? 1 : 0) || kk > 0) ? 1u : 0u);
                    umma_desc_advance(pd, (kk & 3) == 3 ? kApRows * 128 - 96 : 32);
                    umma_desc_advance(vd, 16 * 128);
                }
                umma2_commit_mc_elect(bar(L::C_VEMPTY + st), pair_mask);
                umma2_commit_mc_elect(bar(L::C_PVDONE + buf), pair_mask);
            }
        }
    } else {
        // ---------------- softmax and epilogue (both CTAs): four threads per row ----------------
        const int quarter = warp & 3, half = quarter >> 1, part = (warp - 2) >> 2;
        const int row = (quarter & 1) * 32 + lane, t_row = t0 + row / p.G;
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint32_t leader_pfull = mapa(bar(L::C_PFULL), lead);
        float *xmax = reinterpret_cast<float *>(smem + L::OFF_MAX);
        const Ex2PolyConsts pk = ex2_poly_consts();
        bool ok = true;
        float m_ref = -INFINITY, l = 0.f, m_oth = -INFINITY, l_oth = 0.f;      // of this tile's accumulator and of the other one
        for (int j = 0; j < n; ++j) {
            const int buf = j & 1, st = j % NVS, h = 2 * (tile0 + j) + half;
            const bool dead = h >= H;                         // a half past the last key: its threads only take part in the row exchange
            uint64_t tmask = 0ull;                            // liveness of the 64 keys of this half for every row ...
            uint32_t smask = 0u;                              // ... and of this thread's 32 for this row
            if (!dead) {
                const TileRef tr = g.decode(h);
                tmask = g.tile_mask(tr);
                uint64_t rmask = tmask;
                if (tr.kind == 2 && p.dyn_mask) {
                    const int lim = t_row - tr.idx * kBN;
                    rmask &= (lim < 0) ? 0ull : (lim >= 63 ? ~0ull : ((2ull << lim) - 1ull));
                }
                smask = (uint32_t)(rmask >> (part * 32));
            }
            ok = ok && wait(L::C_SFULL + buf, (uint32_t)(j >> 1) & 1u, 6);
            tc_fence_after();
            float s[32], mx = -INFINITY;
            if (!dead) {
                uint32_t r[32];
                tmem_ld32(taddr + kColS + buf * 64 + part * 32, r);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 32; ++c) s[c] = __uint_as_float(r[c]);
                if (tmask != ~0ull) {
                    // dead keys get weight 0, but 0 x (stale NaN/Inf bytes) would still poison O: clear their V rows
                    ok = ok && wait(L::C_VLAND + st, (uint32_t)(j / NVS) & 1u, 7);
                    if (!((tmask >> row) & 1ull)) {
#pragma unroll
                        for (int c = 0; c < VCH; ++c) {
                            uint4 *vr = reinterpret_cast<uint4 *>(smem + L::OFF_V + st * L::V_STAGE + c * (128 * 128) + (half * 64 + row) * 128) + part * 4;
#pragma unroll
                            for (int i = 0; i < 4; ++i) vr[i] = make_uint4(0, 0, 0, 0);
                        }
                    }
                }
                if (smask != 0xFFFFFFFFu) {
#pragma unroll
                    for (int c = 0; c < 32; ++c)
                        if (!((smask >> c) & 1u)) s[c] = -INFINITY;
                }
                float m4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
                for (int c = 4; c < 28; c += 8) {
                    m4[0] = max3_nan_f32(m4[0], s[c], s[c + 1]); m4[1] = max3_nan_f32(m4[1], s[c + 2], s[c + 3]);
                    m4[2] = max3_nan_f32(m4[2], s[c + 4], s[c + 5]); m4[3] = max3_nan_f32(m4[3], s[c + 6], s[c + 7]);
                }
                m4[0] = max3_nan_f32(m4[0], s[28], s[29]); m4[1] = max3_nan_f32(m4[1], s[30], s[31]);
                mx = max_nan_f32(max_nan_f32(m4[0], m4[1]), max_nan_f32(m4[2], m4[3]));
                if (!(mx < INFINITY)) l = __int_as_float(0x7fc00000);      // a logit that is NaN or +inf makes the row NaN (the polynomial below would lose it)
            }
            // the threads of a row agree on its maximum
            xmax[(buf * kApRows + row) * 4 + half * 2 + part] = mx;
            asm volatile("bar.sync 1, 256;" ::: "memory");
            {
                const float4 v = *reinterpret_cast<const float4 *>(xmax + (buf * kApRows + row) * 4);
                mx = fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w));
            }
            if (j < (DUAL ? 2 : 1)) {
                m_ref = mx;
            } else {
                const bool grow = (mx - m_ref) * p.scale_log2 > kRescaleThreshold;
                if (__any_sync(0xffffffffu, grow)) {
                    // O (and l) were accumulated against m_ref: bring them to the new reference before this tile's P V
                    const float alpha = grow ? ex2((m_ref - mx) * p.scale_log2) : 1.f;
                    if (grow) m_ref = mx;
                    l *= alpha;
                    ok = ok && (DUAL ? wait(L::C_PVDONE + buf, (uint32_t)((j - 2) >> 1) & 1u, 8) : wait(L::C_PVDONE + (buf ^ 1), (uint32_t)((j - 1) >> 1) & 1u, 8));
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < OC / 32; ++c) {
                        uint32_t o[32];
                        tmem_ld32(taddr + kColO + (DUAL ? buf * (HD / 2) : 0) + part * OC + c * 32, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st32(taddr + kColO + (DUAL ? buf * (HD / 2) : 0) + part * OC + c * 32, o);
                    }
                    tmem_wait_st();
                }
            }
            if (!dead) {
                const float mr = m_ref == -INFINITY ? 0.f : m_ref * p.scale_log2;
                const uint64_t sc2 = pack_f32x2(p.scale_log2, p.scale_log2), nm2 = pack_f32x2(-mr, -mr);
                uint64_t sum2[2] = {0ull, 0ull};
                uint32_t packed[16];
#pragma unroll
                for (int c = 0; c < 32; c += 2) {
                    float x0, x1, p0, p1;
                    unpack_f32x2(fma_f32x2(pack_f32x2(s[c], s[c + 1]), sc2, nm2), x0, x1);
                    if (((c >> 1) & 7) < kTc2PolyEighths) ex2_poly_f32x2(x0, x1, pk, p0, p1);      // (as many on the FMA pipe as in attn_tc2_kernel)
                    else { p0 = ex2(x0); p1 = ex2(x1); }
                    sum2[(c >> 1) & 1] = add_f32x2(sum2[(c >> 1) & 1], pack_f32x2(p0, p1));
                    __nv_bfloat162 hh = __floats2bfloat162_rn(p0, p1);
                    packed[c >> 1] = *reinterpret_cast<uint32_t *>(&hh);
                }
                float a0, a1;
                unpack_f32x2(add_f32x2(sum2[0], sum2[1]), a0, a1);
                l += a0 + a1;
                if (smask != 0xFFFFFFFFu) {
                    // (the polynomial gives a masked key 2^-125 instead of 0)
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        if (((c >> 1) & 7) < kTc2PolyEighths) {
                            const uint32_t two = (smask >> c) & 3u;
                            packed[c >> 1] &= ((two & 1u) ? 0x0000FFFFu : 0u) | ((two & 2u) ? 0xFFFF0000u : 0u);
                        }
                    }
                }
                uint8_t *pr = smem + L::OFF_P + buf * L::P_BUF + half * (kApRows * 128) + row * 128;
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    *reinterpret_cast<uint4 *>(pr + (((part * 4 + i) ^ (row & 7)) << 4)) = make_uint4(packed[4 * i], packed[4 * i + 1], packed[4 * i + 2], packed[4 * i + 3]);
            }
            ok = ok && wait(L::C_VLAND + st, (uint32_t)(j / NVS) & 1u, 9);      // the arrival below also says that this CTA's V half is in place
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_pfull + 8u * (uint32_t)buf);
            if constexpr (DUAL) {
                const float m_tmp = m_ref, l_tmp = l;
                m_ref = m_oth; l = l_oth; m_oth = m_tmp; l_oth = l_tmp;
            }
        }
        // ---- epilogue ----
        if (n > 0) ok = ok && wait(L::C_PVDONE + ((n - 1) & 1), (uint32_t)((n - 1) >> 1) & 1u, 10);
        if (DUAL && n > 1) ok = ok && wait(L::C_PVDONE + (n & 1), (uint32_t)((n - 2) >> 1) & 1u, 10);
        if (*abort_flag) ok = false;
        tc_fence_after();
        float *xsum = reinterpret_cast<float *>(smem + L::OFF_SUM);    // [accumulator][64 rows][4]
        const bool odd = DUAL && (n & 1) != 0;                         // m_ref and l are the second accumulator's
        xsum[row * 4 + half * 2 + part] = odd ? l_oth : l;
        if constexpr (DUAL) xsum[(kApRows + row) * 4 + half * 2 + part] = odd ? l : l_oth;
        asm volatile("bar.sync 1, 256;" ::: "memory");
        float w0 = 1.f, w1 = 0.f;                                      // the two become one
        {
            const float4 v = *reinterpret_cast<const float4 *>(xsum + row * 4);
            l = (v.x + v.y) + (v.z + v.w);
        }
        if constexpr (DUAL) {
            const float m0 = odd ? m_oth : m_ref, m1 = odd ? m_ref : m_oth;
            m_ref = fmaxf(m0, m1);
            w0 = m0 == -INFINITY ? 0.f : ex2((m0 - m_ref) * p.scale_log2);
            w1 = m1 == -INFINITY ? 0.f : ex2((m1 - m_ref) * p.scale_log2);
            const float4 u = *reinterpret_cast<const float4 *>(xsum + (kApRows + row) * 4);
            l = fmaf(w0, l, w1 * ((u.x + u.y) + (u.z + u.w)));
        }
        // 32 columns of the row's unnormalised O (an accumulator that was never written counts as zero; after a failed wait NaN)
        auto load_o = [&](int c, float (&o)[32]) {
            uint32_t a[32];
            tmem_ld32(taddr + kColO + part * OC + c * 32, a);
            if constexpr (DUAL) {
                uint32_t b2[32];
                tmem_ld32(taddr + kColO + HD / 2 + part * OC + c * 32, b2);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    o[i] = n > 0 ? __uint_as_float(a[i]) * w0 : 0.f;
                    if (n > 1) o[i] = fmaf(__uint_as_float(b2[i]), w1, o[i]);
                }
            } else {
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = n > 0 ? __uint_as_float(a[i]) : 0.f;
            }
            if (!ok) {
#pragma unroll
                for (int i = 0; i < 32; ++i) o[i] = __int_as_float(0x7fc00000);
            }
        };
        const int col0 = half * (HD / 2) + part * OC;                  // this thread's first column of O
        if (ns == 1) {
            // O / l through the idle Q buffer, laid out like it, and TMA stores
            const float inv = ok && m_ref != -INFINITY ? 1.f / l : __int_as_float(0x7fc00000);      // (NaN too where every logit is -inf)
#pragma unroll
            for (int c = 0; c < OC / 32; ++c) {
                float o[32];
                load_o(c, o);
                const int col = col0 + c * 32;
                uint8_t *srow = smem + L::OFF_Q + (col / 64) * (kApRows * 128) + row * 128;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    uint4 v;
                    uint32_t *vv = reinterpret_cast<uint32_t *>(&v);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        __nv_bfloat162 hh = __floats2bfloat162_rn(o[8 * i + 2 * k] * inv, o[8 * i + 2 * k + 1] * inv);
                        vv[k] = *reinterpret_cast<uint32_t *>(&hh);
                    }
                    *reinterpret_cast<uint4 *>(srow + ((((col & 63) / 8 + i) ^ (row & 7)) << 4)) = v;
                }
            }
            fence_proxy_async_smem();
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (threadIdx.x == 64 && rows > 0) {
                for (int c = 0; c < CH; ++c) tma_store_4d(&tm_o, base + L::OFF_Q + c * (kApRows * 128), c * 64, kvh * p.G, t0, b);
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");      // (the writes are complete when the grid is)
            }
        } else if (p.cluster_merge) {
            // ---- the pairs of the cluster hold slices of the keys for the same rows; pair q finishes columns [q, q + 1) * HD / ns ----
            float2 *ml = reinterpret_cast<float2 *>(smem + L::OFF_ML);
            const int cols = HD / ns, owner = col0 / cols;
            const bool exists = row < rows;
            float fm = m_ref == -INFINITY ? -INFINITY : m_ref * p.scale_log2, fl = ok ? l : __int_as_float(0x7fc00000);
            if (fl == 0.f) fm = -INFINITY;                             // a slice that saw nothing live has no say
            if (threadIdx.x - 64 < ns) mbar_arrive_cluster_release(mapa(bar(L::C_MFREE), 2u * (threadIdx.x - 64) + rank));      // this CTA's K stages are idle
            if (half == 0 && part == 0 && exists) {
                const uint32_t at = smem_u32(ml + split * kApRows + row);
                for (int q = 0; q < ns; ++q)
                    if (q != split) st_async_v2(mapa(at, 2u * q + rank), mapa(bar(L::C_INBOX), 2u * q + rank), __float_as_uint(fm), __float_as_uint(fl));
                ml[split * kApRows + row] = make_float2(fm, fl);
            }
            const bool free = mbar_try_wait_cluster(bar(L::C_MFREE), 0u) || wait_slow(L::C_MFREE, 0u, 11);
            const uint32_t slot = L::OFF_K + (uint32_t)((split * cols + col0 - owner * cols) / 4 * kApRows + row) * 16u;
            const uint32_t dst = mapa(base + slot, 2u * owner + rank), ib = mapa(bar(L::C_INBOX), 2u * owner + rank);
#pragma unroll
            for (int c = 0; c < OC / 32; ++c) {
                float o[32];
                load_o(c, o);
                if (exists && free) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint32_t at = (uint32_t)(c * 8 + i) * (kApRows * 16);
                        if (owner == split) *reinterpret_cast<float4 *>(smem + slot + at) = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                        else st_async_v4(dst + at, ib, __float_as_uint(o[4 * i]), __float_as_uint(o[4 * i + 1]), __float_as_uint(o[4 * i + 2]), __float_as_uint(o[4 * i + 3]));
                    }
                }
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");             // this CTA's own share
            const bool got = (mbar_try_wait_cluster(bar(L::C_INBOX), 0u) || wait_slow(L::C_INBOX, 0u, 12)) && free;
            const int t = threadIdx.x - 64, r = t & 63, cg = t >> 6;   // a row and a quarter of this CTA's columns
            if (r < rows) {
                float w[4], mstar = -INFINITY, l_all = 0.f;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (q < ns) mstar = fmaxf(mstar, ml[q * kApRows + r].x);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    w[q] = 0.f;
                    if (q < ns) {
                        const float2 v = ml[q * kApRows + r];
                        w[q] = v.x == -INFINITY ? 0.f : ex2(v.x - mstar);
                        l_all = fmaf(v.y, w[q], l_all);
                        if (v.y != v.y) l_all = v.y;
                    }
                }
                // A row that exists is always written: NaN where a logit was not finite or a wait ran out, as in the unsplit form
                const float inv = got && l_all > 0.f ? 1.f / l_all : __int_as_float(0x7fc00000);
#pragma unroll
                for (int q = 0; q < 4; ++q) w[q] *= inv;
                const int cpt = cols / 4;                              // columns of this thread: 32, 16 or 8
                const float4 *in = reinterpret_cast<const float4 *>(smem + L::OFF_K) + (cg * cpt / 4) * kApRows + r;
                __nv_bfloat16 *out = (__nv_bfloat16 *)p.out + (((size_t)b * p.T + t0 + r / p.G) * p.Hq + kvh * p.G + r % p.G) * HD + split * cols + cg * cpt;
                for (int c = 0; c < cpt; c += 8) {
                    float a[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) a[i] = 0.f;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (q < ns && w[q] != 0.f) {                   // (NaN weights pass)
                            const float4 v0 = in[(q * cols + c) / 4 * kApRows], v1 = in[((q * cols + c) / 4 + 1) * kApRows];
                            a[0] = fmaf(v0.x, w[q], a[0]); a[1] = fmaf(v0.y, w[q], a[1]); a[2] = fmaf(v0.z, w[q], a[2]); a[3] = fmaf(v0.w, w[q], a[3]);
                            a[4] = fmaf(v1.x, w[q], a[4]); a[5] = fmaf(v1.y, w[q], a[5]); a[6] = fmaf(v1.z, w[q], a[6]); a[7] = fmaf(v1.w, w[q], a[7]);
                        }
                    }
                    uint32_t o[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        __nv_bfloat162 hh = __floats2bfloat162_rn(a[2 * k], a[2 * k + 1]);
                        o[k] = *reinterpret_cast<uint32_t *>(&hh);
                    }
                    *reinterpret_cast<uint4 *>(out + c) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
        } else {
            // ---- (m, l, unnormalised O) for the merge kernel; the tile is staged over the idle K stages and leaves as whole rows ----
            const int rows_total = p.T * p.Hq;
            const size_t n_slots = (size_t)p.B * rows_total * ns;
            auto slot_of = [&](int r) { return partial_slot(b, rows_total, (t0 + r / p.G) * p.Hq + kvh * p.G + r % p.G, ns, split); };
            if (half == 0 && part == 0 && row < rows) {
                float *pml = partial_ml(p.partials, n_slots, slot_of(row), HD);
                pml[0] = m_ref == -INFINITY ? -INFINITY : m_ref * p.scale;
                pml[1] = ok ? l : __int_as_float(0x7fc00000);
            }
            if (n > 0) {
                constexpr int PR = HD / 4;                             // 16-byte pieces per row, swizzled: piece i of row r at i ^ (r % 32)
                float4 *stage = reinterpret_cast<float4 *>(smem + L::OFF_K);
#pragma unroll
                for (int c = 0; c < OC / 32; ++c) {
                    float o[32];
                    load_o(c, o);
#pragma unroll
                    for (int i = 0; i < 8; ++i) stage[row * PR + (((col0 + c * 32) / 4 + i) ^ (row & 31))] = make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
                }
                asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll 2
                for (int rr = 0; rr < kApRows / 8; ++rr) {
                    const int r = (warp - 2) * (kApRows / 8) + rr;
                    if (r >= rows) continue;
                    float4 *dst = reinterpret_cast<float4 *>(partial_o(p.partials, slot_of(r), HD));
#pragma unroll
                    for (int i = 0; i < PR / 32; ++i) dst[i * 32 + lane] = stage[r * PR + ((i * 32 + lane) ^ (r & 31))];
                }
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_arrive_relaxed();
    cluster_wait();   // no CTA retires while another can still touch its shared memory or barriers (nothing to release)
    if (warp == 1) tmem_dealloc2(tmem, kTmemCols);
}

}  // namespace reflex
