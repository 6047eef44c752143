// Memory lookup at one exit layer (Sec. 4.2 Eq. 1-2, Sec. 5 Eq. 3-4): cosine similarity of
// each frame's semantic vector against the members of its fast memory, cumulative
// similarity, top-1 / top-2, accumulated confidence and the exit decision.
//
// One CTA per frame.  The semantic vector is staged in shared memory, each warp takes
// fast-memory slots round-robin and reads the member's centre (L2-resident) with 128-bit
// loads; lanes keep four independent fp32 accumulators and combine with xor-shuffles, so
// every dot product has a fixed evaluation order.  Warp 0 then selects the two best slots.
#include <math.h>

#include <algorithm>

#include "lookup_common.cuh"

namespace smtm {

namespace {

constexpr int kThreads = 256;
constexpr int kFinishThreads = 128;  // decision kernel of the dense route: eight CTAs fit an SM, a frame each

// Any whole number of warps up to kThreads per CTA.  kCtas, the CTAs an SM is to hold, is how many registers a thread gets:
// with four (64 registers) a lane's eight pieces of a centre are really asked for together (a step of 256 frames against 101
// classes 91 us, 100 with five; left to itself the compiler goes to 32 registers and takes them one after another); five,
// where that saves a round of CTAs (737 frames of 1024 channels against 64 classes 54 us, 61 with four).
template <int kCtas>
__global__ void __launch_bounds__(kThreads, kCtas) k_score_exit(const LookupArgs a) {
    extern __shared__ float smem[];
    float* sv = smem;                 // [D]
    float* s_cur = sv + a.D;          // [k_max] similarities of this layer
    float* s_acc = s_cur + a.k_max;   // [k_max] cumulative similarities, then [k_max] the slots' classes
    __shared__ float scratch[32];

    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * (SMTM_PROF_SCORE + a.layer) : nullptr);
    const int b = blockIdx.x;
    const int sid_raw = a.stream_id ? a.stream_id[b] : 0;  // in flight with the exit flag
    if (!a.fresh && a.done[b]) return;  // (a batch that starts here: every frame is in, whatever the flags hold)
    const int tid = threadIdx.x, nthreads = blockDim.x;
    const SlotPrefetch pf = prefetch_slots(a, sid_raw);  // in flight with the semantic vector
    const float* row = a.sv + (size_t)b * a.D;
    float nrm = 0.f;
    for (int d = tid; d < a.D; d += nthreads) {
        const float v = row[d];
        sv[d] = v;
        nrm = fmaf(v, v, nrm);
    }
    nrm = block_sum(nrm, scratch);  // also orders the shared writes above
    score_frame<false>(a, b, pf, sv, nrm, s_cur, s_acc);
}

// The best two keys of the CTA, valid in thread 0.  (b1, b2): this thread's best two; s_keys: [2 * warps].
__device__ __forceinline__ Top2 block_top2_keys(unsigned long long b1, unsigned long long b2, unsigned long long* s_keys) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long k1 = warp_max_u64(b1);
    const unsigned long long k2 = warp_max_u64(b1 == k1 ? b2 : b1);  // keys are unique: the runner-up sits below the winner or elsewhere
    if (lane == 0) {
        s_keys[2 * warp] = k1;
        s_keys[2 * warp + 1] = k2;
    }
    __syncthreads();
    Top2 t{0.f, 0.f, -1, -1};
    if (threadIdx.x == 0) {
        unsigned long long c1 = 0ull, c2 = 0ull;
        for (int i = 0; i < 2 * int(blockDim.x >> 5); ++i) keep_two(s_keys[i], c1, c2);
        rank_key_decode(c1, &t.v1, &t.id1);
        rank_key_decode(c2, &t.v2, &t.id2);
    }
    __syncthreads();
    return t;
}

// ---- large fast memories that all frames share, scored in fp32 ---------------------------------------
//
// A cache with one stream scores every frame against the same slots, so a centre that has been fetched serves several
// frames.  A cluster of P CTAs takes F frames: every CTA keeps the F semantic vectors in shared memory and scores its share
// of the slots, a warp 32 / F slots (at most eight) at a time; where the share is too small for eight warps they divide the
// vector length as well.  The dot products of frame f meet, through distributed shared memory, in CTA f % P of the cluster,
// which decides it.  What bounds it: the centres' way from L2 (k D words per cluster instead of per frame) and, for small
// problems, the trips to memory ([exit flags, slots] -> [vectors, centres] -> decision).
constexpr int kShareMost = 8;                    // frames, and CTAs, of a cluster at most
// Words of centres (at least 64 to a slot) below which a CTA per frame scores: 65 to 71 slots of up to 64 channels, 10.4 us for
// 8 frames of one pixel and 22 for 600, where the clusters, from 72 slots on 6.9 and 17, would be faster too.
constexpr long long kShareWork = 4608;
constexpr size_t kShareSmem = 200 * 1024;
// Frames to a cluster: eight, fewer until every SM has a CTA.  CTAs to a cluster: eight, fewer where they would queue up for a
// place on an SM (two each) and would have at most 64 slots.  Pooling and scoring of 1x1 maps by a CTA per frame and here, us,
// 1024 channels: 256 frames against 101 slots 24 and 18, 1024 frames 56 and 32 (in clusters of eight 48), 256 against 999 167
// and 39, 1024 400 and 126 (in clusters of two 108, but with a fifth of the frames left 105 instead of 36); 8 frames of 32
// channels against 72 slots 10.9 and 6.9, 600 of 64 channels 23 and 17.
constexpr int kShareSlots = 64;
// F vectors [F][D] | [F / P][k_max] dot products of the frames this CTA decides | [k_max] the slots' classes | partial sums
// [8 warps][32].
__host__ __device__ constexpr size_t share_smem(int F, int P, int D, int k_max) {
    return (size_t(F) * D + size_t((F + P - 1) / P + 1) * size_t((k_max + 3) / 4 * 4) + 8 * 32) * sizeof(float);
}

// Which frames: those of F consecutive ones that are still in, decided by the same cluster, so that nobody else's decision
// can change them.  Where that would leave much undone by clusters whose frames have mostly left (more CTAs than the chip
// holds, or much work to a CTA), every CTA lists the frames still in for itself and a cluster takes the next F of the list;
// their exits stay pending until the launch is over.  Half of the frames still in, us, as they lie and listed: 256 frames
// of 2048 channels against 101 classes 24.8 and 20.7, 600 of 1024 against 301 40.2 and 31.4, 64 of 64 (a frame to a cluster:
// nothing to gain) 11.0 and 13.4; the few that are left as they lie and would be faster listed are crowds of short vectors
// (600 of 64 channels against 75 classes 18.3 and 13.9).
constexpr int kShareOwnWork = 1 << 17, kShareOwnWorkCrowd = 1 << 14;  // products to a CTA; the second in clusters of fewer than eight

template <int F>
__global__ void __launch_bounds__(kThreads, 2) k_score_shared(const LookupArgs a, int P) {
    constexpr int T = 32 / F < 8 ? 32 / F : 8;   // slots a warp scores together
    constexpr int kSums = T * F;                 // 32, or fewer with one or two frames
    constexpr int kWarps = kThreads / kWarp;
    extern __shared__ __align__(16) float smem[];
    __shared__ float scratch[33];
    __shared__ unsigned long long s_keys[2 * kWarps];
    __shared__ int s_frames[F];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k_pad = (a.k_max + 3) / 4 * 4;
    float* sv = smem;
    float* dots = sv + size_t(F) * a.D;
    int32_t* s_ids = reinterpret_cast<int32_t*>(dots + (F + P - 1) / P * k_pad);
    float* s_part = reinterpret_cast<float*>(s_ids + k_pad);
    const int group = int(blockIdx.x) / P, rank = int(blockIdx.x) - group * P;
    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * (SMTM_PROF_SCORE + a.layer) : nullptr);
    // This cluster's frames.
    const int k = a.k[0];
    for (int j = tid; j < a.k_max; j += kThreads) s_ids[j] = a.members[j];  // in flight with the exit flags
    if (a.fresh) {
        if (tid < F) s_frames[tid] = group * F + tid < a.B ? group * F + tid : -1;
    } else if (F == 1 || !a.pending) {
        if (warp == 0) {
            const int b = group * F + lane;
            const bool in = lane < F && b < a.B && !a.done[min(b, a.B - 1)];
            const unsigned m = __ballot_sync(kFull, in);
            if (lane < F) s_frames[lane] = -1;
            __syncwarp();
            if (in) s_frames[__popc(m & ((1u << lane) - 1u))] = b;
        }
    } else {
        if (tid < F) s_frames[tid] = -1;
        constexpr int kPer = 4;
        __syncthreads();
        int before = 0;
        for (int t0 = 0; t0 < a.B && before < (group + 1) * F; t0 += kPer * kThreads) {
            int act[kPer], mine = 0;
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                act[i] = a.done[min(t0 + tid * kPer + i, a.B - 1)];
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                act[i] = (t0 + tid * kPer + i < a.B && act[i] == 0) ? 1 : 0;
                mine += act[i];
            }
            int cnt;
            int at = before + block_exclusive_scan(mine, reinterpret_cast<int*>(scratch), &cnt) - group * F;
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                if (act[i]) {
                    if (at >= 0 && at < F) s_frames[at] = t0 + tid * kPer + i;
                    ++at;
                }
            before += cnt;
        }
    }
    __syncthreads();
    if (s_frames[0] < 0) return;  // no frame is left for this cluster (the same for all its CTAs)
    cluster_arrive();             // (waited for before the first store to a peer: it has to have started)
    const int D4 = a.D >> 2;
    for (int f = 0; f < F; ++f) {  // (a frame too few: the first one's vector again, dropped below)
        const float4* row = reinterpret_cast<const float4*>(a.sv + (size_t)max(s_frames[f] < 0 ? s_frames[0] : s_frames[f], 0) * a.D);
        for (int i = tid; i < D4; i += kThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(reinterpret_cast<float4*>(sv) + f * D4 + i)), "l"(row + i)
                         : "memory");
    }
    // what the first of this CTA's decisions needs, in flight with the vectors
    float clen = 0.f, old = 0.f;
    if (tid < k && rank < F && s_frames[rank < F ? rank : 0] >= 0) {
        clen = a.cnorm[s_ids[tid]];
        old = a.fresh ? 0.f : a.sa[(size_t)s_frames[rank < F ? rank : 0] * a.k_max + tid];
    }
    // this CTA's slots, the warps' groups of them and parts of the vector length
    const int share = (k + P - 1) / P;
    const int lo = min(k, rank * share), hi = min(k, lo + share);
    const int groups = (share + T - 1) / T;
    const int parts = groups >= 5 ? 1 : groups >= 3 ? 2 : groups == 2 ? 4 : 8;
    const int part = warp % parts, per = (D4 + parts - 1) / parts;
    const int q_lo = min(D4, part * per), q_hi = min(D4, q_lo + per);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    cluster_wait();
    const float4* v4 = reinterpret_cast<const float4*>(sv);
    const auto deliver = [&](int j, int f, float v) { peer_store(peer_smem(dots + f / P * k_pad + j, f % P), v); };
    for (int g = warp / parts; g < groups; g += kWarps / parts) {
        const int s0 = lo + g * T;
        float d[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) d[e] = 0.f;
        const float4* row[T];
#pragma unroll
        for (int t = 0; t < T; ++t)
            row[t] = reinterpret_cast<const float4*>(a.centers + (size_t)s_ids[min(s0 + t, a.k_max - 1)] * a.D);
        constexpr int kAhead = T <= 4 ? 2 : 1;  // pieces of a centre a lane asks for together
        for (int q0 = q_lo; q0 < q_hi; q0 += kAhead * kWarp) {
            float4 c[kAhead][T];
#pragma unroll
            for (int h = 0; h < kAhead; ++h)
#pragma unroll
                for (int t = 0; t < T; ++t) c[h][t] = row[t][min(q0 + h * kWarp + lane, q_hi - 1)];
#pragma unroll
            for (int h = 0; h < kAhead; ++h) {
                const int q = q0 + h * kWarp + lane;
                if (q < q_hi) {
#pragma unroll
                    for (int f = 0; f < F; ++f) {
                        const float4 x = v4[f * D4 + q];
#pragma unroll
                        for (int t = 0; t < T; ++t)
                            d[t * F + f] += fmaf(c[h][t].w, x.w, fmaf(c[h][t].z, x.z, fmaf(c[h][t].y, x.y, c[h][t].x * x.x)));
                    }
                }
            }
        }
        // kSums sums over 32 lanes, halving what a lane still holds at every step; lane l ends up with sum number l / (32 / kSums)
#pragma unroll
        for (int o = 16, half = kSums / 2; o > 0; o >>= 1, half >>= 1) {
            if (half > 0) {
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int e = 0; e < (half > 0 ? half : 1); ++e) {
                    const float give = up ? d[e] : d[e + half], keep = up ? d[e + half] : d[e];
                    d[e] = keep + __shfl_xor_sync(kFull, give, o);
                }
            } else {
                d[0] += __shfl_xor_sync(kFull, d[0], o);
            }
        }
        const int e = lane / (kWarp / kSums);
        if (parts > 1) {
            if (lane % (kWarp / kSums) == 0) s_part[warp * kWarp + e] = d[0];
        } else {
            const int j = s0 + e / F, f = e % F;
            if (lane % (kWarp / kSums) == 0 && j < hi) deliver(j, f, d[0]);
        }
    }
    if (parts > 1) {
        __syncthreads();
        const int g = tid / kSums, e = tid - g * kSums, j = lo + g * T + e / F;
        if (g < groups && j < hi) {
            float s = 0.f;
            for (int p = 0; p < parts; ++p) s += s_part[(g * parts + p) * kWarp + e];
            deliver(j, e % F, s);
        }
    }
    __syncwarp();
    cluster_sync_all();  // every slot of every frame is in
    const float weight = float(1u << a.layer);  // 2^(l-1) with l = layer + 1
    for (int f = rank; f < F && s_frames[f] >= 0; f += P) {
        const int b = s_frames[f];
        const int k_b = stream_of(a, b) < 0 ? 0 : k;  // a stream id outside the cache: nothing to score against
        float nrm = 0.f;
        for (int i = tid; i < D4; i += kThreads) {
            const float4 x = v4[f * D4 + i];
            nrm = fmaf(x.x, x.x, nrm); nrm = fmaf(x.y, x.y, nrm); nrm = fmaf(x.z, x.z, nrm); nrm = fmaf(x.w, x.w, nrm);
        }
        nrm = block_sum(nrm, scratch);
        unsigned long long a1 = 0ull, a2 = 0ull, c1 = 0ull, c2 = 0ull;
        for (int j = tid; j < a.k_max; j += kThreads) {
            float* sa = a.sa + (size_t)b * a.k_max + j;
            if (j < k_b) {
                if (f != rank || j != tid) {  // (the first is here already)
                    clen = a.cnorm[s_ids[j]];
                    old = a.fresh ? 0.f : *sa;
                }
                const float sim = cosine_from(dots[f / P * k_pad + j], nrm, clen);  // Eq. 1
                const float acc = __fmaf_rn(sim, weight, old);                      // Eq. 3
                *sa = acc;
                keep_two(rank_key(acc, s_ids[j]), a1, a2);
                if (a.sep) keep_two(rank_key(sim, s_ids[j]), c1, c2);  // only Eq. 2 (a diagnostic) needs it
            } else if (a.fresh) {
                *sa = 0.f;  // unused slots start from zero too
            }
        }
        const Top2 ta = block_top2_keys(a1, a2, s_keys);
        Top2 ts{0.f, 0.f, -1, -1};
        if (a.sep) ts = block_top2_keys(c1, c2, s_keys);
        if (tid == 0) decide_from_top2<(F > 1)>(a, b, ta, ts);
    }
}

// Turns the exits that a lookup has left pending (see decide_core) into exit flags, exit layers and labels.  One trip to memory
// after the lookup (512 streams, a step 48.7 -> 49.5 us; in stream order, without the early start, 49.7).
constexpr int kSettleThreads = 128;
__global__ void __launch_bounds__(kSettleThreads) k_settle_exits(const LookupArgs a) {
    chain_wait();
    chain_release();
    const int b = blockIdx.x * kSettleThreads + threadIdx.x;
    if (b >= a.B) return;
    const int gone = a.done[b], left = a.exit_layer[b];
    if (gone || left >= 0) return;
    a.done[b] = 1;
    a.exit_layer[b] = a.layer + 1;
    a.pred[b] = -1 - left;
}

// Finishing kernel of the tensor-core path: one CTA per frame turns the frame's row of dot products into
// similarities of its fast-memory slots and decides.  The row (its parts added) and the
// centres' lengths come in with coalesced 16-byte loads and are parked in shared memory, from where the slots
// pick their class's entry: a gather straight from global memory costs a sector per slot, and a thousand slots
// for each of a thousand frames are then bound by that.  Everything a frame needs after its stream id is fetched
// in one trip: the size and the members of its fast memory, the carries, the row, the lengths and the semantic
// vector (for its length).  Every thread keeps the two best of its own slots as 64-bit ranking keys; warps merge
// by two warp-wide maxima, the CTA through shared memory.  With a.fresh the carry is taken as SA = 0, nobody done.
constexpr int kFinishSlots = 4;  // slots a thread fetches per trip

template <bool kTwoParts>  // the usual number of parts of a problem that fills the chip
__global__ void __launch_bounds__(kFinishThreads, kTwoParts ? 10 : 8) k_finish_dense(const LookupArgs a, const DenseDots dd) {
    constexpr int kPieces = kTwoParts ? 1 : 2;       // pieces of the row a thread fetches per trip
    extern __shared__ __align__(16) float s_row[];  // [ld] dot products, then [ld] lengths of the centres
    __shared__ float scratch[32];
    __shared__ unsigned long long s_keys[2 * (kFinishThreads / kWarp)];
    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * SMTM_PROF_FINISH_DENSE : nullptr);
    const int b = blockIdx.x, tid = threadIdx.x;
    const int gone = a.fresh ? 0 : a.done[b];
    const int sid = stream_of(a, b);  // (in flight with the flag)
    if (gone) return;
    float* s_len = s_row + dd.ld;
    const int32_t* mem = a.members + (size_t)max(sid, 0) * a.k_max;
    float* sa_row = a.sa + (size_t)b * a.k_max;
    const float weight = float(1u << a.layer);
    // this trip: the fast memory's size, the first slots' classes and carries (unconditional: up to k_max) ...
    const int k = sid < 0 ? 0 : a.k[sid];  // a stream id outside the cache: nothing to score against
    int cls[kFinishSlots];
    float old[kFinishSlots];
#pragma unroll
    for (int u = 0; u < kFinishSlots; ++u) {
        const int j = min(u * kFinishThreads + tid, a.k_max - 1);
        cls[u] = mem[j];
        old[u] = a.fresh ? 0.f : sa_row[j];
    }
    // ... the row of dot products (the parts of the vector length added in order) and the lengths, all asked for before
    // anything is stored (ordinary loads: the kernels before may have written it while this one was already resident) ...
    const float4* drow = reinterpret_cast<const float4*>(dd.dots + (size_t)b * dd.ld);
    const float4* clen = reinterpret_cast<const float4*>(a.cnorm);
    const size_t part = dd.stride / 4;
    const int n4 = dd.ld / 4;
    float4 d[kPieces], e[kPieces], len[kPieces];
    const auto fetch = [&](int c0) {
#pragma unroll
        for (int u = 0; u < kPieces; ++u) {
            const int c4 = min(c0 + u * kFinishThreads, n4 - 1);
            d[u] = drow[c4];
            e[u] = kTwoParts || dd.parts > 1 ? drow[part + c4] : make_float4(0.f, 0.f, 0.f, 0.f);
            len[u] = clen[c4];
        }
    };
    const auto park = [&](int c0) {
#pragma unroll
        for (int u = 0; u < kPieces; ++u) {
            const int c4 = c0 + u * kFinishThreads;
            if (c4 < n4) {
                d[u].x += e[u].x; d[u].y += e[u].y; d[u].z += e[u].z; d[u].w += e[u].w;
                if (!kTwoParts)
#pragma unroll 4
                    for (int s0 = 2; s0 < dd.parts; ++s0) {
                        const float4 f = drow[s0 * part + c4];
                        d[u].x += f.x; d[u].y += f.y; d[u].z += f.z; d[u].w += f.w;
                    }
                reinterpret_cast<float4*>(s_row)[c4] = d[u];
                reinterpret_cast<float4*>(s_len)[c4] = len[u];
            }
        }
    };
    fetch(tid);
    // ... and the squared length of the semantic vector (D is a multiple of 8 on this route)
    const float4* row4 = reinterpret_cast<const float4*>(a.sv + (size_t)b * a.D);
    float q[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int i = tid; i < a.D / 4; i += kFinishThreads) {
        const float4 v = row4[i];
        q[0] = fmaf(v.x, v.x, q[0]);
        q[1] = fmaf(v.y, v.y, q[1]);
        q[2] = fmaf(v.z, v.z, q[2]);
        q[3] = fmaf(v.w, v.w, q[3]);
    }
    park(tid);
    for (int c0 = tid + kPieces * kFinishThreads; c0 < n4; c0 += kPieces * kFinishThreads) {
        fetch(c0);
        park(c0);
    }
    const float nrm = block_sum((q[0] + q[1]) + (q[2] + q[3]), scratch);  // (also orders the shared writes above)
    const float sv_len = __fsqrt_rn(nrm);
    unsigned long long a1 = 0ull, a2 = 0ull, c1 = 0ull, c2 = 0ull;  // best two cumulative / single-layer keys
    for (int j0 = 0; j0 < k; j0 += kFinishSlots * kFinishThreads) {
        if (j0 > 0) {  // a fast memory of more than 512 slots: one more trip per 512
#pragma unroll
            for (int u = 0; u < kFinishSlots; ++u) {
                const int j = min(j0 + u * kFinishThreads + tid, a.k_max - 1);
                cls[u] = mem[j];
                old[u] = a.fresh ? 0.f : sa_row[j];
            }
        }
#pragma unroll
        for (int u = 0; u < kFinishSlots; ++u) {
            const int j = j0 + u * kFinishThreads + tid;
            if (j < k) {
                const float dot = s_row[cls[u]], cl = s_len[cls[u]];
                const float sim = (nrm == 0.f || cl == 0.f) ? 0.f : __fdiv_rn(dot, __fmul_rn(sv_len, cl));  // Eq. 1
                const float acc = __fmaf_rn(sim, weight, old[u]);                                              // Eq. 3
                sa_row[j] = acc;
                keep_two(rank_key(acc, cls[u]), a1, a2);
                if (a.sep) keep_two(rank_key(sim, cls[u]), c1, c2);  // only Eq. 2 (a diagnostic) needs it
            }
        }
    }
    if (a.fresh)
        for (int j = k + tid; j < a.k_max; j += kFinishThreads) sa_row[j] = 0.f;  // unused slots start from zero too
    const Top2 ta = block_top2_keys(a1, a2, s_keys);
    Top2 ts{0.f, 0.f, -1, -1};
    if (a.sep) ts = block_top2_keys(c1, c2, s_keys);
    if (tid == 0) decide_from_top2(a, b, ta, ts);
}

__global__ void k_batch_reset(float* __restrict__ sa, uint8_t* __restrict__ done, int32_t* __restrict__ exit_layer,
                              int32_t* __restrict__ pred, int B, long long n_sa) {
    chain_wait();
    chain_release();
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = i0; i < n_sa; i += step) sa[i] = 0.f;
    for (long long i = i0; i < B; i += step) {
        done[i] = 0;
        exit_layer[i] = 0;
        pred[i] = -1;
    }
}

// The wait of the streaming kernels (mbar_wait_bounded), on a barrier that never completes its phase.
__global__ void k_wait_selftest(int* status) {
    __shared__ uint64_t bar;
    chain_wait();
    chain_release();
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init_fence();
        mbar_wait_bounded(&bar, 0, status);  // gives up after its limit and records the time-out
    }
}

}  // namespace

cudaError_t launch_wait_selftest(int* status, cudaStream_t st, int64_t* launches) {
    ++*launches;
    return launch_chained(k_wait_selftest, 1, kWarp, 0, st, status);
}

cudaError_t lookup_setup() {
    cudaError_t e = allow_max_dynamic_smem(k_score_exit<4>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_settle_exits);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_score_exit<5>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_score_shared<1>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_score_shared<2>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_score_shared<4>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_score_shared<8>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_score_exit<4>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_score_exit<5>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_finish_dense<true>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_finish_dense<false>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_finish_dense<false>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_finish_dense<true>);  // (two words per class: 64 KB at 8192 classes)
    return e;
}

cudaError_t launch_batch_reset(float* sa, uint8_t* done, int32_t* exit_layer, int32_t* pred, int B, int k_max,
                               cudaStream_t st, int64_t* launches) {
    if (B <= 0) return cudaSuccess;
    const long long n_sa = (long long)B * k_max;
    const int grid = int(std::min<long long>((n_sa + 255) / 256, 1184));
    ++*launches;
    return launch_chained(k_batch_reset, grid, 256, 0, st, sa, done, exit_layer, pred, B, n_sa);
}

cudaError_t launch_finish_dense(const LookupArgs& a, const DenseDots& dots, bool beside_pooling, cudaStream_t st,
                                int64_t* launches) {
    if (a.B <= 0) return cudaSuccess;
    ++*launches;
    const size_t smem = 2 * size_t(dots.ld) * sizeof(float);
    const auto kernel = dots.parts == 2 ? k_finish_dense<true> : k_finish_dense<false>;
    if (beside_pooling) return launch_ordered(kernel, a.B, kFinishThreads, smem, st, a, dots);
    return launch_chained(kernel, a.B, kFinishThreads, smem, st, a, dots);
}

cudaError_t launch_settle_exits(const LookupArgs& a, cudaStream_t st, int64_t* launches) {
    ++*launches;
    return launch_chained(k_settle_exits, (a.B + kSettleThreads - 1) / kSettleThreads, kSettleThreads, 0, st, a);
}

// Frames to a cluster of k_score_shared, or 0 where a CTA per frame scores them; *ctas: CTAs of a cluster.
static int shared_frames(const LookupArgs& a, int sm_count, int* ctas) {
    if (a.S != 1 || a.k_max <= kFusedMaxK || (a.D & 3) || (long long)a.k_max * std::max(a.D, 64) < kShareWork) return 0;
    const int frames = a.fresh ? a.B : (a.B + 1) / 2;  // (after a first lookup half of them are taken to be still in)
    const auto groups = [&](int F) { return (frames + F - 1) / F; };
    int F = kShareMost, P = kShareMost;
    while (F > 1 && groups(F) * P < sm_count) F /= 2;
    while (P > 1 && groups(F) * P > 2 * sm_count && a.k_max <= kShareSlots * P) P /= 2;
    while (F > 1 && share_smem(F, P, a.D, a.k_max) > kShareSmem) F /= 2;
    *ctas = P;
    return share_smem(F, P, a.D, a.k_max) > kShareSmem ? 0 : F;
}

cudaError_t launch_score_exit(const LookupArgs& a, cudaStream_t st, int sm_count, int64_t* launches, int threads,
                              bool in_order) {
    if (a.B <= 0) return cudaSuccess;
    int P = 0;
    if (const int F = shared_frames(a, sm_count, &P)) {
        const auto kernel = F == 1 ? k_score_shared<1> : F == 2 ? k_score_shared<2> : F == 4 ? k_score_shared<4> : k_score_shared<8>;
        const size_t smem = share_smem(F, P, a.D, a.k_max);
        const int ctas = (a.B + F - 1) / F * P;
        LookupArgs s = a;
        const long long work = (long long)F * ((a.k_max + P - 1) / P) * a.D;
        s.pending = !a.fresh && F > 1 && (4 * ctas > 9 * sm_count || work > (P < kShareMost ? kShareOwnWorkCrowd : kShareOwnWork));
        ++*launches;
        const cudaError_t e = in_order ? launch_ordered_cluster(kernel, ctas, kThreads, smem, P, st, s, P)
                                       : launch_chained_cluster(kernel, ctas, kThreads, smem, P, st, s, P);
        return e == cudaSuccess && s.pending ? launch_settle_exits(s, st, launches) : e;
    }
    const auto rounds = [&](int ctas) { return (a.B + ctas * sm_count - 1) / (ctas * sm_count); };
    const auto kernel = rounds(5) < rounds(4) ? k_score_exit<5> : k_score_exit<4>;
    const size_t smem = (size_t(a.D) + 3 * size_t(a.k_max)) * sizeof(float);
    ++*launches;
    if (in_order) return launch_ordered(kernel, a.B, threads > 0 ? threads : kThreads, smem, st, a);
    return launch_chained(kernel, a.B, threads > 0 ? threads : kThreads, smem, st, a);
}

}  // namespace smtm
