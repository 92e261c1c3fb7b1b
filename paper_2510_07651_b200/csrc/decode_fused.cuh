// The whole decode step as one kernel, for few units (included by decode.cu, whose chunk helpers it uses).
//
// A small step is a chain of latencies, and as four kernels most of it is their beginnings and ends.  Here a thread-block
// cluster takes a (b, g): one chunk of N slots and N threads per CTA.  K and V of the chunk come to shared memory once,
// logits and positions stay with the thread of their slot, the partial outputs are merged over distributed shared memory,
// and one launch does it all.  With many units the waits for the cluster leave the SMs idle, so those keep the four kernels
// (see fused_chunk for the line between them).
#pragma once

template <int G, int N> constexpr size_t kFusedBytes = 2 * (size_t)N * 256 + (size_t)G * N * 4 + 1024;   // K rows, V rows, probabilities

template <int G, int N>
__global__ void __launch_bounds__(N)
decode_fused_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                    DecodeShape s, TensorView q, TensorView kt, TensorView vt, TensorView kc, TensorView vc,
                    float* s_acc, int32_t* pos, int32_t* state, int step_pos) {
    constexpr int NW = N / 32, RING = 16, MAXC = 16;
    extern __shared__ __align__(16) uint4 sRaw[];
    uint4* sK = reinterpret_cast<uint4*>(((uintptr_t)sRaw + 1023) & ~(uintptr_t)1023);   // the swizzle's 1024-byte frame
    uint4* sV = sK + N * 16;
    float (*sP)[N] = reinterpret_cast<float (*)[N]>(sV + N * 16);                        // [G]: logits, then probabilities
    // over the K rows, once the logits are out: per-warp partial outputs [NW][G][kD], then v . o_r (r < G) and ||v||^2 per slot
    float* sO = reinterpret_cast<float*>(sK);
    float (*sT)[N] = reinterpret_cast<float (*)[N]>(sO + NW * G * kD);
    static_assert(NW * G * kD * 4 + (G + 1) * N * 4 <= N * 256, "both fit the K rows");
    __shared__ uint64_t sBar[2];
    __shared__ float sRedM[NW][G], sRedL[NW][G];
    __shared__ __align__(16) float sPart[G][kD];           // this chunk's outputs, read by the other CTAs,
    __shared__ float2 sMl[G];                              // and its (max, sum) per head
    __shared__ float sLse[G], sNo[G];
    __shared__ __align__(16) uint32_t sOhi[G][kD / 2], sOlo[G][kD / 2];   // merged o as two bf16 parts, in the MMA lanes' order
    __shared__ MinCand sMin[NW], sRankMin[MAXC];
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int unit = blockIdx.x / C, b = unit / s.Hkv, g = unit % s.Hkv, c0 = rank * N;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, slot = c0 + tid;
    const int gq = lane >> 2, tq = lane & 3;               // MMA fragments: row in a group of eight, lane in the quad
    const size_t ubase = (size_t)unit * s.cap;
    if (tid == 0) { chunk_bar_init(&sBar[0]); chunk_bar_init(&sBar[1]); }
    pdl_wait();                                            // the kernel before this one may have written the caches
    if (tid == 0) {
        copy_chunk_tma<N>(sK, &map_k, &sBar[0], b, g, c0);
        copy_chunk_tma<N>(sV, &map_v, &sBar[1], b, g, c0);
    }
    const int live_old = state[unit * 4], next = state[unit * 4 + 1], hi_old = state[unit * 4 + 2];
    const int pos_in = slot < s.cap ? pos[ubase + slot] : -1;
    const float acc_old = slot < s.cap ? s_acc[ubase + slot] : 0.f;
    uint32_t qf[8][2];                                     // B operand of the logits: head gq, channels 16 ks + 2 tq .. and + 8
    {
        const uint32_t* qrow = reinterpret_cast<const uint32_t*>(bf_row(q, b, g * G + (gq < G ? gq : 0), 0));
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            qf[ks][0] = gq < G ? qrow[ks * 8 + tq] : 0u;
            qf[ks][1] = gq < G ? qrow[ks * 8 + 4 + tq] : 0u;
        }
    }
    const bool valid = next >= 0 && next < s.cap;
    const int hi = min(valid ? max(hi_old, next + 1) : hi_old, s.cap);
    const bool owns_new = valid && next >= c0 && next < c0 + N;
    uint4 new_row = make_uint4(0, 0, 0, 0);                // threads 0-15: k of the new token, 16-31: v
    if (owns_new && tid < 32) {
        new_row = reinterpret_cast<const uint4*>(tid < 16 ? bf_row(kt, b, g, 0) : bf_row(vt, b, g, 0))[tid & 15];
        const_cast<uint4*>(reinterpret_cast<const uint4*>(tid < 16 ? bf_row(kc, b, g, next) : bf_row(vc, b, g, next)))[tid & 15] = new_row;
    }
    const bool is_new = valid && slot == next;
    const int my_pos = is_new ? step_pos : slot < hi ? pos_in : -1;
    const bool live = my_pos >= 0;
    // the ring of per-step scores of this slot, on its way while the rest is computed (a new token enters with an empty history)
    float* hcol = s.acc_window > 0 ? s.s_hist + (size_t)unit * s.acc_window * s.cap + slot : nullptr;
    const int ring_now = s.acc_window > 0 ? step_pos % s.acc_window : 0;
    float ring[RING];
#pragma unroll
    for (int u = 0; u < RING; ++u) ring[u] = (live && !is_new && u < s.acc_window && u != ring_now) ? hcol[(size_t)u * s.cap] : 0.f;
    __syncthreads();                                       // the barriers are initialised for every waiter

    // ---- logits: MMA over the warp's 32 slots, then one thread per slot ----------------------------------------
    bool copy_failed = !chunk_wait(&sBar[0], 0);
    if (owns_new) {                                        // the bulk copy may have read the cache before the new row was written
        if (tid < 16) sK[staged_piece<N>(next - c0, tid)] = new_row;
        __syncthreads();
    }
#pragma unroll
    for (int tile = 0; tile < 2; ++tile) {
        const int row0 = warp * 32 + tile * 16, sl = row0 + gq, h0 = 2 * tq;
        float acc[2][4] = {};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            uint32_t a[4];
            ldsm_x4(a, tile_addr<N>(sK, row0, 2 * ks, lane, true));
            mma_bf16(acc[ks & 1], a, qf[ks][0], qf[ks][1]);
        }
        // [0], [1]: slot sl, heads h0, h0 + 1; [2], [3]: slot sl + 8
        if (h0 < G) { sP[h0][sl] = acc[0][0] + acc[1][0]; sP[h0][sl + 8] = acc[0][2] + acc[1][2]; }
        if (h0 + 1 < G) { sP[h0 + 1][sl] = acc[0][1] + acc[1][1]; sP[h0 + 1][sl + 8] = acc[0][3] + acc[1][3]; }
    }
    __syncwarp();
    const float sl2 = s.scale * kLog2e;
    float z2[G];
#pragma unroll
    for (int r = 0; r < G; ++r) {
        z2[r] = live ? sP[r][tid] * sl2 : -INFINITY;
        const float wm = warp_max(z2[r]);
        if (lane == 0) sRedM[warp][r] = wm;
    }
    __syncthreads();                                       // also: the K rows are no longer read
#pragma unroll
    for (int r = 0; r < G; ++r) {
        float m = sRedM[0][r];
#pragma unroll
        for (int w = 1; w < NW; ++w) m = fmaxf(m, sRedM[w][r]);
        const float p = live ? exp2f(z2[r] - m) : 0.f;
        sP[r][tid] = p;
        const float l = warp_sum(p);
        if (lane == 0) { sRedL[warp][r] = l; if (warp == 0) sMl[r].x = m; }
    }
    copy_failed |= !chunk_wait(&sBar[1], 0);
    if (owns_new && tid >= 16 && tid < 32) sV[staged_piece<N>(next - c0, tid & 15)] = new_row;
    // rows without a live token may hold anything, and 0 x NaN would spoil the outputs: freed slots one by one, those past the
    // live extent together
    if (!live && slot < hi)
        for (int i = 0; i < 16; ++i) sV[staged_piece<N>(tid, i)] = make_uint4(0, 0, 0, 0);
    if (c0 + N > hi)
        for (int i = tid; i < N * 16; i += N) if (c0 + (i >> 4) >= hi) sV[staged_piece<N>(i >> 4, i & 15)] = make_uint4(0, 0, 0, 0);
    __syncthreads();

    // ---- the chunk's outputs: (16 channels) x (8 heads) tiles of V^T P^T, P as two bf16 parts -------------------
    {
        uint32_t ph[2][2], pl[2][2];                       // [16-slot step][k half]: p of head gq, slots 2 tq, + 1 (+ 8)
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int sl = warp * 32 + kk * 16 + hf * 8 + 2 * tq;
                const float p0 = gq < G ? sP[gq][sl] : 0.f, p1 = gq < G ? sP[gq][sl + 1] : 0.f;
                split_bf16x2(p0, p1, ph[kk][hf], pl[kk][hf]);
            }
        float* sOw = sO + warp * G * kD;
#pragma unroll
        for (int j = 0; j < 8; ++j) {                      // channels 16 j .. 16 j + 15
            float acc[2][4] = {};
#pragma unroll
            for (int kk = 0; kk < 2; ++kk) {
                uint32_t a[4];
                ldsm_x4_trans(a, tile_addr<N>(sV, warp * 32 + kk * 16, 2 * j, lane, false));
                mma_bf16(acc[kk], a, ph[kk][0], ph[kk][1]);
                mma_bf16(acc[kk], a, pl[kk][0], pl[kk][1]);
            }
            // [0], [1]: channel ch, heads h0, h0 + 1; [2], [3]: channel ch + 8
            const int ch = 16 * j + gq, h0 = 2 * tq;
            if (h0 < G) { sOw[h0 * kD + ch] = acc[0][0] + acc[1][0]; sOw[h0 * kD + ch + 8] = acc[0][2] + acc[1][2]; }
            if (h0 + 1 < G) { sOw[(h0 + 1) * kD + ch] = acc[0][1] + acc[1][1]; sOw[(h0 + 1) * kD + ch + 8] = acc[0][3] + acc[1][3]; }
        }
    }
    __syncthreads();
    for (int i = tid; i < G * kD; i += N) {
        float acc = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) acc += sO[w * G * kD + i];
        (&sPart[0][0])[i] = acc;
    }
    if (tid < G) {
        float l = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) l += sRedL[w][tid];
        sMl[tid].y = l;
    }
    __syncthreads();
    cluster.barrier_arrive();                              // outputs and statistics may be read by the other CTAs after their wait

    // ---- ||v||^2 meanwhile: the diagonal of tile x tile^T, whose B operand is the tile's own A fragment ---------
#pragma unroll
    for (int tile = 0; tile < 2; ++tile) {
        const int row0 = warp * 32 + tile * 16;
        float n_lo[4] = {}, n_hi[4] = {};
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            uint32_t a[4];
            ldsm_x4(a, tile_addr<N>(sV, row0, 2 * ks, lane, true));
            mma_bf16(n_lo, a, a[0], a[2]);                 // columns = slots row0 .. + 7
            mma_bf16(n_hi, a, a[1], a[3]);                 // columns = slots row0 + 8 .. + 15
        }
        if (tq == (gq >> 1)) {                             // the lane whose column pair contains its own row
            sT[G][row0 + gq] = (gq & 1) ? n_lo[1] : n_lo[0];
            sT[G][row0 + gq + 8] = (gq & 1) ? n_hi[3] : n_hi[2];
        }
    }
    __syncwarp();
    cluster.barrier_wait();

    // ---- merge over the chunks: a warp per head, four channels per lane ------------------------------------------
    for (int h = warp; h < G; h += NW) {
        float4 part[MAXC];
#pragma unroll
        for (int r = 0; r < MAXC; ++r)                     // all of them on their way before the first use
            if (r < C) part[r] = reinterpret_cast<const float4*>(cluster.map_shared_rank(&sPart[h][0], r))[lane];
        const float2 ml = lane < C ? *cluster.map_shared_rank(&sMl[h], lane < C ? lane : 0) : make_float2(-INFINITY, 0.f);
        const float M = warp_max(ml.x);
        const float w = ml.x == -INFINITY ? 0.f : exp2f(ml.x - M);
        const float L = warp_sum(w * ml.y);
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int r = 0; r < MAXC; ++r)
            if (r < C) {
                const float wr = __shfl_sync(0xffffffffu, w, r);
                o.x = fmaf(part[r].x, wr, o.x); o.y = fmaf(part[r].y, wr, o.y);
                o.z = fmaf(part[r].z, wr, o.z); o.w = fmaf(part[r].w, wr, o.w);
            }
        if (L > 0.f) { o.x /= L; o.y /= L; o.z /= L; o.w /= L; }
        const float sq = warp_sum((o.x * o.x + o.y * o.y) + (o.z * o.z + o.w * o.w));
        if (lane == 0) { sLse[h] = M + log2f(L); sNo[h] = sq; }
        // word w = 8 ks + 4 k + t (channels 2 w, 2 w + 1) goes to word 16 t + 2 ks + k: a lane's sixteen words are four 16-byte loads
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int wd = 2 * lane + e, at = (wd & 3) * 16 + (wd >> 3) * 2 + ((wd >> 2) & 1);
            uint32_t hi2, lo2;
            split_bf16x2(e ? o.z : o.x, e ? o.w : o.y, hi2, lo2);
            sOhi[h][at] = hi2; sOlo[h][at] = lo2;
        }
    }
    __syncthreads();

    // ---- v . o and the scores --------------------------------------------------------------------------------------
    {
        uint32_t oh[8][2], ol[8][2];
        const uint4* hrow = reinterpret_cast<const uint4*>(&sOhi[gq < G ? gq : 0][tq * 16]);
        const uint4* lrow = reinterpret_cast<const uint4*>(&sOlo[gq < G ? gq : 0][tq * 16]);
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
            const uint4 h4 = gq < G ? hrow[k4] : make_uint4(0, 0, 0, 0), l4 = gq < G ? lrow[k4] : make_uint4(0, 0, 0, 0);
            oh[2 * k4][0] = h4.x; oh[2 * k4][1] = h4.y; oh[2 * k4 + 1][0] = h4.z; oh[2 * k4 + 1][1] = h4.w;
            ol[2 * k4][0] = l4.x; ol[2 * k4][1] = l4.y; ol[2 * k4 + 1][0] = l4.z; ol[2 * k4 + 1][1] = l4.w;
        }
#pragma unroll
        for (int tile = 0; tile < 2; ++tile) {
            const int row0 = warp * 32 + tile * 16, sl = row0 + gq, h0 = 2 * tq;
            float th[4] = {}, tl[4] = {};
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
                uint32_t a[4];
                ldsm_x4(a, tile_addr<N>(sV, row0, 2 * ks, lane, true));
                mma_bf16(th, a, oh[ks][0], oh[ks][1]);
                mma_bf16(tl, a, ol[ks][0], ol[ks][1]);
            }
            if (h0 < G) { sT[h0][sl] = th[0] + tl[0]; sT[h0][sl + 8] = th[2] + tl[2]; }
            if (h0 + 1 < G) { sT[h0 + 1][sl] = th[1] + tl[1]; sT[h0 + 1][sl + 8] = th[3] + tl[3]; }
        }
    }
    __syncwarp();                                          // a slot's values come from its own warp
    MinCand cand{INFINITY, -1, -1, 0};
    if (live) {
        float t[G];
#pragma unroll
        for (int r = 0; r < G; ++r) t[r] = sT[r][tid];
        const float sc = slot_score<G>(s.variant, z2, sLse, sNo, t, sT[G][tid]);
        float acc = (is_new ? 0.f : acc_old) + sc;
        if (s.acc_window > 0) {                            // the last acc_window steps only, summed afresh in ring order
            acc = 0.f;
#pragma unroll
            for (int u = 0; u < RING; ++u) acc += u == ring_now ? sc : ring[u];
            for (int r0 = RING; r0 < s.acc_window; r0 += 8) {
                float hv[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) hv[u] = (!is_new && r0 + u < s.acc_window && r0 + u != ring_now) ? hcol[(size_t)(r0 + u) * s.cap] : 0.f;
#pragma unroll
                for (int u = 0; u < 8; ++u) acc += r0 + u == ring_now ? sc : hv[u];
            }
            if (is_new)                                    // the slot's former tenant left its own history
                for (int r = 0; r < s.acc_window; ++r) hcol[(size_t)r * s.cap] = 0.f;
            hcol[(size_t)ring_now * s.cap] = sc;
        }
        s_acc[ubase + slot] = acc;
        if (is_new) pos[ubase + slot] = step_pos;
        if (my_pos >= s.n_sink && my_pos <= step_pos - s.n_recent) cand = MinCand{acc, my_pos, slot, 0};
    }
    if (copy_failed) atomicMax(&state[unit * 4 + 3], 2);
    min_over_warp(cand);
    if (lane == 0) sMin[warp] = cand;
    __syncthreads();
    if (tid == 0) {
#pragma unroll
        for (int w = 1; w < NW; ++w) if (goes_first(sMin[w], cand)) cand = sMin[w];
        *cluster.map_shared_rank(&sRankMin[rank], 0) = cand;
    }
    __syncwarp();
    cluster.sync();                                        // and no CTA leaves while another may read its outputs
    if (rank != 0 || warp != 0) return;
    if (!valid) { if (lane == 0) state[unit * 4 + 3] = 1; return; }        // no room: the step was not applied
    int live_now = live_old + 1, new_next = hi;
    if (live_now > s.budget) {
        MinCand best = lane < C ? sRankMin[lane] : MinCand{INFINITY, -1, -1, 0};
        min_over_warp(best);
        if (best.slot >= 0) {
            if (lane == 0) pos[ubase + best.slot] = -1;
            live_now -= 1;
            new_next = best.slot;
        }
    }
    if (lane == 0) { state[unit * 4 + 0] = live_now; state[unit * 4 + 1] = new_next; state[unit * 4 + 2] = hi; }
}

// how many clusters of the one-kernel step the device holds at once (asked once per thread, device, shape and cluster size)
template <int G, int N>
int fused_clusters(int C) {
    thread_local int seen_dev = -1, seen[17];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev != seen_dev) { for (int& x : seen) x = -1; seen_dev = dev; }
    if (seen[C] < 0) {
        int n = 0;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)C); cfg.blockDim = dim3(N); cfg.dynamicSmemBytes = kFusedBytes<G, N>;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        const auto kernel = decode_fused_kernel<G, N>;
        if (allow_smem(kernel, kFusedBytes<G, N>) != cudaSuccess ||
            cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { n = 0; (void)cudaGetLastError(); }
        seen[C] = n;
    }
    return seen[C];
}

template <int G, int N>
obc_status launch_fused(const CUtensorMap& mk, const CUtensorMap& mv, const DecodeShape& s, TensorView q, TensorView kt, TensorView vt,
                        TensorView kc, TensorView vc, float* s_acc, int32_t* pos, int32_t* state, int step_pos, cudaStream_t stream) {
    const int C = (s.cap + N - 1) / N;
    ProfScope ps("decode_fused", stream);
    OBC_CUDA_TRY(allow_smem(decode_fused_kernel<G, N>, kFusedBytes<G, N>));
    OBC_CUDA_TRY(launch_pdl(decode_fused_kernel<G, N>, dim3((unsigned)(s.B * s.Hkv * C)), dim3(N), kFusedBytes<G, N>, stream, C, mk, mv, s, q, kt, vt, kc, vc,
                            s_acc, pos, state, step_pos));
    return OBC_OK;
}

// The chunk length of the one-kernel step, or 0 for the four kernels.  The line is where the clusters no longer run all at
// once: a step of one wave takes 10 to 14 us against 15 to 17.5 (8 units of 1025 slots 9.8 against 17.5 us, 32 of 701
// 10.7 against 17.3, 8 of 2049 with a window of 16 steps 13.5 against 15.2), of two waves and more longer (52 units of 1572:
// 31 against 22; 224 of 418: 55 against 40).  Chunks of 128 slots where 16 of them hold the cache, else of 256.
template <int G>
int fused_chunk(const DecodeShape& s) {
    const int units = s.B * s.Hkv, c128 = (s.cap + 127) / 128, c256 = (s.cap + 255) / 256;
    if (c128 <= 16) return units <= fused_clusters<G, 128>(c128) ? 128 : 0;
    return c256 <= 16 && units <= fused_clusters<G, 256>(c256) ? 256 : 0;
}
