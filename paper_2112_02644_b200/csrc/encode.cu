// Semantic-vector encoding (Sec. 4.1): SV[b][c] = mean over H x W of the feature map.
//
// The feature maps are read exactly once from HBM; this is the only step of the hot path
// whose traffic grows with C*H*W, so everything here is organised around streaming.
//
// NCHW.  A frame is a flat run of C channels of H*W elements.  Channels are grouped into
// "units": the smallest number G of consecutive channels whose bytes are a multiple of 16
// (7x7 bf16: 8 channels = 784 B).  A persistent CTA per SM runs a ring of shared-memory
// stages; one producer thread fills stages with 1-D bulk asynchronous copies of whole
// chunks (a run of units, <= 25 KB) completing on an mbarrier, and eight consumer warps each
// reduce the chunks of their own stages and write the channel means straight to SV.
// Chunks partition channels, so no two warps ever touch the same output: no atomics, and
// the summation order of every channel is fixed.
//   * unit-per-lane reducer (H*W small and odd-sized): lane i owns unit i of the chunk and
//     walks its 16-byte vectors; the stride between lanes is an odd number of vectors, so the
//     128-bit shared loads are conflict-free; the element -> channel map is resolved at compile time.
//   * team reducer: T lanes share a channel, stride over its vectors and combine with xor-shuffles;
//     channels that begin or end inside a vector have their edges added element by element.
//   * lane-per-channel reducer (channels of odd widths below 128 bytes): 32-bit words.
// Small batches, and the few NCHW shapes bulk copies cannot serve, are pooled by the last two straight from global
// memory (k_pool_direct).
// NHWC.  Consecutive 16-byte vectors of a frame are consecutive channel groups of a pixel;
// each thread owns one channel group and a pixel phase, loads coalesced 128-bit vectors
// directly and the phases are combined through shared memory in a fixed order; few frames are
// divided between the CTAs of clusters.
#include <algorithm>
#include <cmath>

#include "lookup_common.cuh"

namespace smtm {

namespace {

constexpr int kStages = 8;             // ring depth
constexpr int kConsumers = 8;          // consumer warps; stage s belongs to warp s % kConsumers
constexpr int kStageCap = 25600;       // bytes per stage

struct NchwParams {
    const uint8_t* x;
    const uint8_t* skip;
    float* sv;
    __nv_bfloat16* sv_hi;    // optional bf16 head and tail of sv (sv = hi + lo), same indexing; may be null
    __nv_bfloat16* sv_lo;
    int* status;
    int B;                   // frames
    int C;
    int chunks_per_frame;
    int chunk_channels;      // channels in a full chunk
    int ch_bytes;            // bytes of one channel
    long long frame_bytes;
    float inv_hw;
    int hw, es;              // elements per channel, bytes per element
    int team;                // the team reducers: lanes per channel (power of two)
    int max_in_flight;       // copies the producer keeps outstanding (<= stages)
    int stages;              // k_encode_nchw: ring depth, 2 .. kStages (the fused kernel always uses kStages)
    int consumers;           // k_encode_nchw: consumer warps, 1 .. kConsumers; the CTA has one more warp, the producer's
    unsigned long long* clock;  // nullptr, or two words for the device-clock stamps of the pooling kernel
};

// Writes the bf16 head and tail of n consecutive values (n a multiple of 2, dst 4-byte aligned).
template <int N>
__device__ __forceinline__ void store_split(const float (&v)[N], __nv_bfloat16* hi, __nv_bfloat16* lo) {
#pragma unroll
    for (int g = 0; g < N; g += 2) {
        const __nv_bfloat16 h0 = __float2bfloat16_rn(v[g]), h1 = __float2bfloat16_rn(v[g + 1]);
        const __nv_bfloat16 l0 = __float2bfloat16_rn(v[g] - __bfloat162float(h0));
        const __nv_bfloat16 l1 = __float2bfloat16_rn(v[g + 1] - __bfloat162float(h1));
        *reinterpret_cast<__nv_bfloat162*>(hi + g) = __nv_bfloat162(h0, h1);
        *reinterpret_cast<__nv_bfloat162*>(lo + g) = __nv_bfloat162(l0, l1);
    }
}

// ---- reducers --------------------------------------------------------------------------

// Lane i reduces unit i: G channels of HW elements stored as UW consecutive 16-byte vectors.
template <class E, int HW>
struct UnitPerLane {
    static constexpr int kUnitBytesRaw = HW * E::kSize;
    static constexpr int gcd16(int a) { return (a % 16 == 0) ? 16 : (a % 8 == 0) ? 8 : (a % 4 == 0) ? 4 : (a % 2 == 0) ? 2 : 1; }
    static constexpr int G = 16 / gcd16(kUnitBytesRaw);
    static constexpr int UW = G * kUnitBytesRaw / 16;

    static __device__ __forceinline__ void run(const uint8_t* stage, int, int nch, int lane, float* out, float* out_s,
                                               float inv_hw, const NchwParams& p) {
        const int units = nch / G;
        if (lane >= units) return;
        const uint4* u = reinterpret_cast<const uint4*>(stage) + lane * UW;
        float acc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = 0.f;
#pragma unroll
        for (int i = 0; i < UW; ++i) {
            const uint4 v = u[i];
#pragma unroll
            for (int j = 0; j < E::kPerVec; ++j) acc[(i * E::kPerVec + j) / HW] += E::at(v, j);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] *= inv_hw;
        float* o = out + lane * G;  // G floats, aligned to G * 4 bytes
        if (G == 2) {
            *reinterpret_cast<float2*>(o) = make_float2(acc[0], acc[1]);
        } else {
#pragma unroll
            for (int g = 0; g + 3 < G; g += 4)
                *reinterpret_cast<float4*>(o + g) = make_float4(acc[g], acc[g + 1], acc[g + 2], acc[g + 3]);
        }
        if (p.sv_hi) {
            const ptrdiff_t at = (o - p.sv);
            store_split<G>(acc, p.sv_hi + at, p.sv_lo + at);
        }
        if (out_s) {
            float* os = out_s + lane * G;
            if (G == 2) {
                *reinterpret_cast<float2*>(os) = make_float2(acc[0], acc[1]);
            } else {
#pragma unroll
                for (int g = 0; g + 3 < G; g += 4)
                    *reinterpret_cast<float4*>(os + g) = make_float4(acc[g], acc[g + 1], acc[g + 2], acc[g + 3]);
            }
        }
    }
};

// Writes a channel's mean wherever it is wanted.
__device__ __forceinline__ void store_mean(const NchwParams& p, float v, int c, float* out, float* out_s) {
    out[c] = v;
    if (out_s) out_s[c] = v;
    if (p.sv_hi) {
        const ptrdiff_t at = (out + c) - p.sv;
        const __nv_bfloat16 hh = __float2bfloat16_rn(v);
        p.sv_hi[at] = hh;
        p.sv_lo[at] = __float2bfloat16_rn(v - __bfloat162float(hh));
    }
}

// T lanes per channel, 16-byte vectors.  Eight lanes read 128 consecutive bytes (one conflict-free phase of a shared
// load, one line of global memory); channels shorter than that have as many lanes as whole vectors.  kEdges: channels
// may begin and end inside a vector (`off`: elements of the stage before the first channel); the whole vectors in
// between are walked as usual and the at most seven elements before and after are a load of their own in one lane
// each, which takes T = 8.  Two channels per team are folded at a time, four vectors of each in flight: what bounds
// a warp here is the latency of a chunk (a stage of the ring is held meanwhile), not the instructions.
template <class E, bool kEdges>
struct TeamVectors {
    static constexpr int kShortChannel = 1024;  // bytes

    template <int NB, int U>
    static __device__ __forceinline__ void group(const uint8_t* stage, int off, int nch, int first, int stride, int r, int T,
                                                 int lane, float* out, float* out_s, float inv_hw, const NchwParams& p) {
        constexpr int V = E::kPerVec;
        float a[NB][V];
        const uint4* u[NB];
        int n[NB], n_min = 1 << 30, n_max = 0;
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            const int c = min(first + h * stride, nch - 1);  // (a channel past the end: the last one, dropped below)
            const int e0 = (kEdges ? off : 0) + c * p.hw, e1 = e0 + p.hw;
            const int v0 = kEdges ? (e0 + V - 1) / V : e0 / V, v1 = e1 / V;
            u[h] = reinterpret_cast<const uint4*>(stage) + v0;
            n[h] = v1 - v0;
            n_min = min(n_min, n[h]);
            n_max = max(n_max, n[h]);
#pragma unroll
            for (int j = 0; j < V; ++j) a[h][j] = 0.f;
            if (kEdges) {
                if (r < v0 * V - e0) a[h][0] = E::scalar(stage, e0 + r);
                if (r < e1 - v1 * V) a[h][1] = E::scalar(stage, v1 * V + r);
            }
        }
        int i = r;
        for (; i + (U - 1) * T < n_min; i += U * T) {
            uint4 v[NB][U];
#pragma unroll
            for (int h = 0; h < NB; ++h)
#pragma unroll
                for (int k = 0; k < U; ++k) v[h][k] = u[h][i + k * T];
#pragma unroll
            for (int k = 0; k < U; ++k)
#pragma unroll
                for (int h = 0; h < NB; ++h)
#pragma unroll
                    for (int j = 0; j < V; ++j) a[h][j] += E::at(v[h][k], j);
        }
        for (; i < n_max; i += T) {
            uint4 v[NB];
#pragma unroll
            for (int h = 0; h < NB; ++h) v[h] = i < n[h] ? u[h][i] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int h = 0; h < NB; ++h)
#pragma unroll
                for (int j = 0; j < V; ++j) a[h][j] += E::at(v[h], j);
        }
        float s[NB];
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            s[h] = (a[h][0] + a[h][1]) + (a[h][2] + a[h][3]);
            if (V == 8) s[h] += (a[h][4 % V] + a[h][5 % V]) + (a[h][6 % V] + a[h][7 % V]);
        }
        for (int o = T >> 1; o > 0; o >>= 1)
#pragma unroll
            for (int h = 0; h < NB; ++h) s[h] += __shfl_xor_sync(kFull, s[h], o);
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            const int c = first + h * stride;
            if (c < nch && r == 0) store_mean(p, s[h] * inv_hw, c, out, out_s);
        }
    }

    // Short channels: a few vectors per lane, so that adding the lanes up would cost more than the vectors.  NB
    // channels per team go through the reduction together, each step halving what a lane still holds (seven
    // exchanges for eight channels over eight lanes), and every lane writes its share.
    template <int T, int NB>
    static __device__ __forceinline__ void short_group(const uint8_t* stage, int off, int nch, int first, int r, float* out,
                                                       float* out_s, float inv_hw, const NchwParams& p) {
        constexpr int V = E::kPerVec;
        constexpr int kStride = kWarp / T;
        float s[NB];
        const uint4* u[NB];
        int n[NB], n_max = 0;
#pragma unroll
        for (int h = 0; h < NB; ++h) {
            const int c = first + h * kStride;
            const int e0 = (kEdges ? off : 0) + c * p.hw, e1 = e0 + p.hw;
            const int v0 = kEdges ? (e0 + V - 1) / V : e0 / V, v1 = e1 / V;
            u[h] = reinterpret_cast<const uint4*>(stage) + v0;
            n[h] = c < nch ? v1 - v0 : 0;
            n_max = max(n_max, n[h]);
            s[h] = 0.f;
            if (kEdges && c < nch) {
                if (r < v0 * V - e0) s[h] = E::scalar(stage, e0 + r);
                if (r < e1 - v1 * V) s[h] += E::scalar(stage, v1 * V + r);
            }
        }
        for (int i = r; i < n_max; i += T) {
            uint4 v[NB];
#pragma unroll
            for (int h = 0; h < NB; ++h) v[h] = i < n[h] ? u[h][i] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int h = 0; h < NB; ++h) {
                float t = (E::at(v[h], 0) + E::at(v[h], 1)) + (E::at(v[h], 2) + E::at(v[h], 3));
                if (V == 8) t += (E::at(v[h], 4 % V) + E::at(v[h], 5 % V)) + (E::at(v[h], 6 % V) + E::at(v[h], 7 % V));
                s[h] += t;
            }
        }
        int held = NB, h0 = 0;  // this lane ends up with the channels h0 .. h0 + held - 1 of its team
#pragma unroll
        for (int o = T / 2; o > 0; o >>= 1) {
            const bool up = (r & o) != 0;
            if (held > 1) {
                held >>= 1;
#pragma unroll
                for (int e = 0; e < NB / 2; ++e)
                    if (e < held) {
                        const float give = up ? s[e] : s[e + held], keep = up ? s[e + held] : s[e];
                        s[e] = keep + __shfl_xor_sync(kFull, give, o);
                    }
                h0 += up ? held : 0;
            } else {
                s[0] += __shfl_xor_sync(kFull, s[0], o);
            }
        }
        constexpr int kHeld = NB > T ? NB / T : 1;
        const bool writes = NB >= T || (r & (T / NB - 1)) == 0;  // (fewer channels than lanes: one lane of each run that holds the same)
#pragma unroll
        for (int e = 0; e < kHeld; ++e) {
            const int c = first + (h0 + e) * kStride;
            if (writes && c < nch) store_mean(p, s[e] * inv_hw, c, out, out_s);
        }
    }

    template <int T>
    static __device__ __forceinline__ void run_short(const uint8_t* stage, int off, int nch, int lane, float* out, float* out_s,
                                                     float inv_hw, const NchwParams& p) {
        constexpr int kStride = kWarp / T;
        const int team = lane / T, r = lane % T;
        int c0 = 0;
        for (; c0 + 2 * kStride < nch; c0 += 8 * kStride) short_group<T, 8>(stage, off, nch, c0 + team, r, out, out_s, inv_hw, p);
        if (c0 < nch) short_group<T, 2>(stage, off, nch, c0 + team, r, out, out_s, inv_hw, p);
    }

    static __device__ __forceinline__ void run(const uint8_t* stage, int off, int nch, int lane, float* out, float* out_s,
                                               float inv_hw, const NchwParams& p) {
        if (p.ch_bytes < kShortChannel) {
            if (kEdges || p.team == 8) run_short<8>(stage, off, nch, lane, out, out_s, inv_hw, p);
            else if (p.team == 4) run_short<4>(stage, off, nch, lane, out, out_s, inv_hw, p);
            else if (p.team == 2) run_short<2>(stage, off, nch, lane, out, out_s, inv_hw, p);
            else run_short<1>(stage, off, nch, lane, out, out_s, inv_hw, p);
            return;
        }
        constexpr int T = 8, kStride = kWarp / T;
        const int team = lane / T, r = lane % T;
        int c0 = 0;
        for (; c0 + kStride < nch; c0 += 2 * kStride)
            group<2, 4>(stage, off, nch, c0 + team, kStride, r, T, lane, out, out_s, inv_hw, p);
        if (c0 < nch) group<1, 8>(stage, off, nch, c0 + team, kStride, r, T, lane, out, out_s, inv_hw, p);
    }
};

// A lane per channel for short channels of any number of bytes (below 128): each is walked in 32-bit words, whichever
// element of the stage it begins at (`off`: elements before the first channel).  With 16-bit elements a channel that
// begins or ends inside a word gets that element by a load of its own.
template <class E>
struct LanePerChannel {
    static __device__ __forceinline__ float low(uint32_t w) { return E::at(make_uint4(w, 0, 0, 0), 0); }
    static __device__ __forceinline__ float high(uint32_t w) { return E::kSize == 2 ? E::at(make_uint4(w, 0, 0, 0), 1) : 0.f; }

    static __device__ __forceinline__ void run(const uint8_t* stage, int off, int nch, int lane, float* out, float* out_s,
                                               float inv_hw, const NchwParams& p) {
        constexpr int kPerWord = 4 / E::kSize;
        constexpr int kBatch = 8;  // words in flight per lane
        const uint32_t* words = reinterpret_cast<const uint32_t*>(stage);
        for (int c = lane; c < nch; c += kWarp) {
            const int e0 = off + c * p.hw, e1 = e0 + p.hw;
            int w = (e0 + kPerWord - 1) / kPerWord;   // the words that are all this channel's
            const int w1 = e1 / kPerWord;
            float lo[4] = {0.f, 0.f, 0.f, 0.f}, hi[4] = {0.f, 0.f, 0.f, 0.f};
            if (kPerWord == 2 && (e0 & 1)) hi[1] = E::scalar(stage, e0);
            if (kPerWord == 2 && (e1 & 1)) lo[1] = E::scalar(stage, e1 - 1);
            for (; w + kBatch <= w1; w += kBatch) {
                uint32_t v[kBatch];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) v[u] = words[w + u];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    lo[u & 3] += low(v[u]);
                    if (kPerWord == 2) hi[u & 3] += high(v[u]);
                }
            }
            if (w < w1) {
                uint32_t v[kBatch];
#pragma unroll
                for (int u = 0; u < kBatch - 1; ++u) v[u] = w + u < w1 ? words[w + u] : 0u;
#pragma unroll
                for (int u = 0; u < kBatch - 1; ++u) {
                    lo[u & 3] += low(v[u]);
                    if (kPerWord == 2) hi[u & 3] += high(v[u]);
                }
            }
            float s = (lo[0] + lo[1]) + (lo[2] + lo[3]);
            if (kPerWord == 2) s += (hi[0] + hi[1]) + (hi[2] + hi[3]);
            store_mean(p, s * inv_hw, c, out, out_s);
        }
    }
};

// ---- persistent bulk-copy pipeline -------------------------------------------------------
//
// What bounds it: HBM, once a CTA's warps do next to nothing per chunk besides their own share.  A warp steps from
// chunk to chunk by additions alone (frame and chunk-of-frame advance by constants), and only over its own chunks:
// with a 64-bit division per chunk and every warp looking at every chunk the loop itself was the bound (1.64 GB of
// 56x56 maps in 312 us, 5.3 TB/s).  Four 25 KB copies in flight per SM saturate the reads (7.2 TB/s in a
// copy-only ring; 200 KB in flight are slower again).
// Without skip flags a batch is one run of B * C channels (chunks may span frames, so that small maps make
// full-sized copies: one thread issues a copy per 0.27 us and would cap 4 KB copies at 2.2 TB/s).  With them the
// frames still in are listed first, a tile of frames at a time.
constexpr int kListFrames = 2048;  // frames listed at a time

// The chunk a warp is at: chunk `ci` of listed frame `f`; step() moves on by `stride` chunks.  (one_frame: nothing to
// divide by, which is a quarter of a microsecond before the first copy.)
struct ChunkWalk {
    int f, ci, df, dci, cpf;
    __device__ __forceinline__ ChunkWalk(int first, int stride, int chunks_per_frame, bool one_frame)
        : f(0), ci(first), df(0), dci(stride), cpf(chunks_per_frame) {
        if (one_frame) return;
        f = first / cpf;
        ci = first - f * cpf;
        df = stride / cpf;
        dci = stride - df * cpf;
    }
    __device__ __forceinline__ void step() {
        f += df;
        ci += dci;
        if (ci >= cpf) {
            ci -= cpf;
            ++f;
        }
    }
};

// (At most 128 registers, as for 512 threads: on the pipelined route they decide how many CTAs of the other kernels fit
// on an SM beside this one.)
template <class R>
__global__ void __launch_bounds__(512, 1) k_encode_nchw(const NchwParams p) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    uint8_t* stages = base;
    const int n_stages = p.stages;
    uint64_t* full = reinterpret_cast<uint64_t*>(base + size_t(n_stages) * kStageCap);
    uint64_t* empty = full + n_stages;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init_fence();
    }
    __syncthreads();
    chain_wait();  // the barriers are set up while the previous kernel finishes
    chain_release();
    const ClockScope stamps(p.clock);

    const int n_consumers = p.consumers;
    const bool producer = warp == n_consumers;  // last warp; lane 0 issues the copies
    const uint64_t stream_once = l2_evict_first_policy();
    int* list = reinterpret_cast<int*>(empty + n_stages);  // [kListFrames + 33], only there with skip flags
    const int grid = int(gridDim.x), cpf = p.chunks_per_frame;
    int it0 = 0;         // chunks of this CTA in the tiles of frames before this one
    int issued = 0;
    bool failed = false;
    const auto span_of = [&](int c0, int nch, long long& begin, int& off) {  // a chunk's bytes, widened to 16-byte boundaries
        const long long lo = (long long)c0 * p.ch_bytes;
        begin = lo & ~15ll;
        off = int(lo - begin);
        return uint32_t((off + nch * p.ch_bytes + 15) & ~15);
    };
    for (int t0 = 0; t0 < p.B; t0 += kListFrames) {
        int frames = p.B;  // no flags: all of them (one "frame" of B * C channels), in a single round
        if (p.skip) {
            frames = 0;
            int* s_scan = list + kListFrames;
            __syncthreads();  // the list of the tile before is read to the end
            for (int u0 = t0; u0 < min(p.B, t0 + kListFrames); u0 += int(blockDim.x)) {
                const int b = u0 + int(threadIdx.x);
                const int act = (b < min(p.B, t0 + kListFrames) && !p.skip[b]) ? 1 : 0;
                int cnt;
                const int pos = block_exclusive_scan(act, s_scan, &cnt);
                if (act) list[frames + pos] = b;
                frames += cnt;
            }
            __syncthreads();
        }
        const int chunks = frames * cpf;
        if (producer) {
            if (lane == 0) {
                ChunkWalk at(int(blockIdx.x), grid, cpf, p.B == 1);
                int stage = 0, old_stage = 0;
                uint32_t phase = 0u, old_phase = 0u;
                int old = it0 - p.max_in_flight;  // the copy that has to have landed before this one is issued
                if (it0 > 0) {  // (a second listing)
                    stage = it0 % n_stages;
                    phase = uint32_t(it0 / n_stages) & 1u;
                    old_stage = old >= 0 ? old % n_stages : 0;
                    old_phase = old >= 0 ? uint32_t(old / n_stages) & 1u : 0u;
                }
                for (int g = int(blockIdx.x), i = 0; g < chunks; g += grid, ++i, ++old) {
                    if (it0 + i >= n_stages && !mbar_wait_bounded(&empty[stage], phase ^ 1u, p.status)) failed = true;
                    if (!failed && old >= 0) {
                        if (!mbar_wait_bounded(&full[old_stage], old_phase, p.status)) failed = true;
                        if (++old_stage == n_stages) {
                            old_stage = 0;
                            old_phase ^= 1u;
                        }
                    }
                    if (failed) break;
                    const int c0 = at.ci * p.chunk_channels, nch = min(p.chunk_channels, p.C - c0);
                    const long long b = p.skip ? list[at.f] : at.f;
                    long long begin;
                    int off;
                    const uint32_t bytes = span_of(c0, nch, begin, off);
                    mbar_expect_tx(&full[stage], bytes);
                    bulk_load_hint(stages + size_t(stage) * kStageCap, p.x + b * p.frame_bytes + begin, bytes, &full[stage],
                                   stream_once);
                    issued = it0 + i + 1;
                    at.step();
                    if (++stage == n_stages) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
        } else {
            // chunk number `it` of this CTA goes to warp it % n_consumers and sits in stage it % n_stages
            int first = warp, stage = warp;  // (no more consumers than stages)
            uint32_t phase = 0u;
            if (it0 > 0) {
                first = (warp - it0 % n_consumers + n_consumers) % n_consumers;
                stage = (it0 + first) % n_stages;
                phase = uint32_t((it0 + first) / n_stages) & 1u;
            }
            const int stride = n_consumers * grid;
            ChunkWalk at(int(blockIdx.x) + first * grid, stride, cpf, p.B == 1);
            for (int g = int(blockIdx.x) + first * grid; g < chunks; g += stride) {
                const int c0 = at.ci * p.chunk_channels, nch = min(p.chunk_channels, p.C - c0);
                const long long b = p.skip ? list[at.f] : at.f;
                long long begin;
                int off;
                span_of(c0, nch, begin, off);
                if (!mbar_wait_bounded(&full[stage], phase, p.status)) {
                    failed = true;
                    break;
                }
                R::run(stages + size_t(stage) * kStageCap, off / p.es, nch, lane, p.sv + b * p.C + c0, nullptr, p.inv_hw, p);
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[stage]);
                at.step();
                stage += n_consumers;
                if (stage >= n_stages) {
                    stage -= n_stages;
                    phase ^= 1u;
                }
            }
        }
        if (!p.skip) break;
        it0 += chunks > int(blockIdx.x) ? (chunks - int(blockIdx.x) + grid - 1) / grid : 0;
    }
    // No thread leaves before every copy that was issued has landed: shared memory must
    // stay allocated until the copy engine is done with it.
    const int any_failed = __syncthreads_or(failed ? 1 : 0);
    if (any_failed && producer && lane == 0) {
        for (int s = 0; s < n_stages && s < issued; ++s) {
            const uint32_t last_use = uint32_t((issued - 1 - s) / n_stages);
            mbar_wait_bounded(&full[s], last_use & 1, p.status);
        }
    }
}

// ---- fused lookup: encode + similarity scoring + decision in one persistent kernel ------------
//
// A frame is cut into P parts (runs of chunks_per_unit chunks, i.e. slices of its channels) and
// a thread-block cluster of P CTAs takes whole frames: CTA `rank` of the cluster streams and
// scores part `rank`.  Every CTA first compacts the frames that are still active; cluster c
// takes the frames c, c + clusters, ... of that list, so exited frames cost nothing and the
// load is even.  Per frame the reducer warps leave the slice of the semantic vector in shared
// memory (four buffers) as well as in the SV stash; eight dot warps then share the slice's dot
// products, slot j on warp j % 8: each lane has every load of its slot's centre slice in
// flight at once, so a frame costs one trip to L2.  The partial dot products and the partial
// squared length go, through distributed shared memory, to a receive buffer in the cluster's
// first CTA, whose finisher warp adds the parts up in rank order and decides: Eq. 1, Eq. 3,
// top-2, Eq. 4 / Eq. 2 and the exit rule.  No atomics on floating point and no global scratch:
// the evaluation order of every sum is fixed.
constexpr int kReducersF = 4;       // reducer warps of the fused kernel; stage s belongs to warp s % kReducersF
constexpr int kDotWarps = 8;        // warps that share the dot products of a slice
constexpr int kSvBufs = 4;          // shared-memory slices; frame u passes through buffer u % kSvBufs
constexpr int kRx = 4;              // receive buffers between the dot warps and the finisher
constexpr int kRxRow = kFusedMaxK + 4;  // words per row of a receive buffer
// A receive buffer holds P + 2 rows: one per part (the partial dots, then the partial squared length at
// [kFusedMaxK]) and, from the first CTA's own dot warps, the slots' classes (then k at [kFusedMaxK]) and the
// lengths of their centres, so that the finisher has nothing to fetch once the parts are in.
constexpr int kMaxCluster = 8;      // CTAs per cluster = parts per frame
constexpr int kThreadsFused = (kReducersF + 1 + kDotWarps + 1) * kWarp;  // reducers, producer, dot warps, finisher
constexpr int kMaxUnits = 1024;     // frames per cluster
constexpr int kMaxSlice = 1024;     // floats of a semantic-vector slice (eight 16-byte vectors per lane)
constexpr size_t kSmemLimit = 227 * 1024;
static_assert(kStages % kReducersF == 0, "stage ownership must be periodic");

struct FusedParams {
    NchwParams e;
    LookupArgs a;
    int parts;            // P: CTAs per cluster, one part of every frame each (divides chunks_per_frame)
    int chunks_per_unit;  // chunks_per_frame / P
    int slice_cap;        // channels of a full slice = chunks_per_unit * chunk_channels (multiple of 4)
};

constexpr size_t fused_smem(int slice_cap, int parts) {
    return size_t(kStages) * kStageCap + size_t(kSvBufs) * size_t(slice_cap) * 4 +
           size_t(kRx) * size_t(parts + 2) * kRxRow * 4 + kMaxUnits * 4 + 40 * 4 +
           (2 * kStages + 2 * kSvBufs + 2 * kRx) * 8 + 192;
}

template <class R>
__global__ void __launch_bounds__(kThreadsFused, 1) k_lookup_nchw(const FusedParams f) {
    extern __shared__ uint8_t smem_raw[];
    const NchwParams& p = f.e;
    const LookupArgs& a = f.a;
    const int P = f.parts, cpu = f.chunks_per_unit;
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    uint8_t* stages = base;
    float* sv_s = reinterpret_cast<float*>(base + size_t(kStages) * kStageCap);  // [kSvBufs][slice_cap]
    float* rx = sv_s + kSvBufs * f.slice_cap;                                    // [kRx][P + 2][kRxRow]
    int* my_units = reinterpret_cast<int*>(rx + kRx * (P + 2) * kRxRow);               // [kMaxUnits] frames of this cluster
    int* s_scan = my_units + kMaxUnits;                                          // [36]
    unsigned int* s_ctr = reinterpret_cast<unsigned int*>(s_scan + 36);          // [4] lookups, near, exits
    uint64_t* full = reinterpret_cast<uint64_t*>(
        (reinterpret_cast<uintptr_t>(s_scan + 40) + 7) & ~uintptr_t(7));         // [kStages]
    uint64_t* empty = full + kStages;                                            // [kStages]
    uint64_t* sv_full = empty + kStages;                                         // [kSvBufs]  slice written
    uint64_t* sv_empty = sv_full + kSvBufs;                                      // [kSvBufs]  slice read by all dot warps
    uint64_t* rx_full = sv_empty + kSvBufs;                                      // [kRx]  every part has arrived here
    uint64_t* rx_empty = rx_full + kRx;                                          // [kRx]  every rank: the finisher is done with it

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = int(blockIdx.x) % P;       // clusters are runs of P consecutive CTAs
    const int cluster = int(blockIdx.x) / P, n_clusters = int(gridDim.x) / P;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kSvBufs; ++s) {
            mbar_init(&sv_full[s], cpu);
            mbar_init(&sv_empty[s], kDotWarps);
        }
        for (int s = 0; s < kRx; ++s) {
            mbar_init(&rx_full[s], P * kDotWarps);
            mbar_init(&rx_empty[s], 1);
        }
        mbar_init_fence();
        s_ctr[0] = s_ctr[1] = s_ctr[2] = 0u;
    }

    // ---- the active frames and this cluster's share of them ---------------------------------
    int n_active = a.fresh ? a.B : 0;  // a batch that starts here has every frame active: no flags to read
    for (int idx = threadIdx.x; a.fresh && idx < kMaxUnits; idx += kThreadsFused) {
        const long long u = (long long)cluster + (long long)idx * n_clusters;
        if (u < a.B) my_units[idx] = int(u);
    }
    // Everything above touched shared memory only and overlaps the previous kernel's tail.
    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * a.layer : nullptr);  // profiling
    if (!a.fresh && !a.pending) {  // clusters for every frame: a cluster's own, if it is still in
        if (cluster < a.B && !a.done[cluster]) {
            if (threadIdx.x == 0) my_units[0] = cluster;
            n_active = cluster + 1;
        }
    }
    for (int t0 = 0; a.pending && t0 < a.B; t0 += kThreadsFused) {
        const int b = t0 + threadIdx.x;
        // (A finisher of this launch may already have decided the frame: its exit is pending, the flag is what it was
        // before, so every CTA gets the same list whenever it looks.)
        const int act = (b < a.B && !a.done[b]) ? 1 : 0;
        int cnt;
        const int pos = block_exclusive_scan(act, s_scan, &cnt);
        if (act) {
            const int u = n_active + pos;
            if (u % n_clusters == cluster && u / n_clusters < kMaxUnits) my_units[u / n_clusters] = b;
        }
        n_active += cnt;
    }
    int nu = n_active > cluster ? (n_active - cluster + n_clusters - 1) / n_clusters : 0;
    nu = min(nu, kMaxUnits);
    __syncthreads();
    if (P > 1) cluster_sync_all();  // every CTA's barriers exist before anyone arrives on them

    const int n_chunks = nu * cpu;
    bool failed = false;
    int issued = 0;
    if (warp < kReducersF) {
        // ---- reducers: warp w owns the stages w, w + kReducersF, ... -----------------------------
        for (int it = warp; it < n_chunks; it += kReducersF) {
            const int i = it / cpu, c = it - i * cpu;
            const int b = my_units[i];
            const int c0 = (rank * cpu + c) * p.chunk_channels;
            const int nch = min(p.chunk_channels, p.C - c0);
            const int stage = it % kStages;
            const int buf = i % kSvBufs, round = i / kSvBufs;
            if (round > 0 && !mbar_wait_bounded(&sv_empty[buf], (round - 1) & 1, p.status)) { failed = true; break; }
            if (!mbar_wait_bounded(&full[stage], (it / kStages) & 1, p.status)) { failed = true; break; }
            R::run(stages + size_t(stage) * kStageCap, 0, nch, lane, p.sv + (long long)b * p.C + c0,
                   sv_s + buf * f.slice_cap + c * p.chunk_channels, p.inv_hw, p);
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&empty[stage]);
                mbar_arrive(&sv_full[buf]);
            }
        }
    } else if (warp == kReducersF) {
        // ---- producer -------------------------------------------------------------------------
        if (lane == 0) {
            const uint64_t stream_once = l2_evict_first_policy();
            for (int it = 0; it < n_chunks; ++it) {
                const int i = it / cpu, c = it - i * cpu;
                const int b = my_units[i];
                const int c0 = (rank * cpu + c) * p.chunk_channels;
                const int nch = min(p.chunk_channels, p.C - c0);
                const int stage = it % kStages;
                const uint32_t use = uint32_t(it / kStages);
                if (use > 0 && !mbar_wait_bounded(&empty[stage], (use - 1) & 1, p.status)) { failed = true; break; }
                if (it >= p.max_in_flight) {  // bound the bytes in flight: wait for an older copy to land
                    const int old = it - p.max_in_flight;
                    if (!mbar_wait_bounded(&full[old % kStages], (old / kStages) & 1, p.status)) { failed = true; break; }
                }
                const uint32_t bytes = uint32_t(nch) * uint32_t(p.ch_bytes);
                mbar_expect_tx(&full[stage], bytes);
                bulk_load_hint(stages + size_t(stage) * kStageCap,
                               p.x + (long long)b * p.frame_bytes + (long long)c0 * p.ch_bytes, bytes, &full[stage], stream_once);
                issued = it + 1;
            }
        }
    } else if (warp <= kReducersF + kDotWarps) {
        // ---- dot warps: all of them work on frame u together, slot j on warp j % kDotWarps -------
        const int dw = warp - kReducersF - 1;
        const int sb = rank * f.slice_cap;          // first channel of this CTA's slice
        const int Dp = max(0, min(f.slice_cap, p.C - sb));  // channels in it (a multiple of 4)
        const int n4 = Dp >> 2;
        // fast memory of the frame in hand, fetched one frame ahead
        int nx_k = 0, nx_ids[2] = {0, 0};
        if (nu > 0) {
            const int b = my_units[0];
            const int sid = stream_of(a, b);
            nx_k = sid < 0 ? 0 : min(a.k[sid], kFusedMaxK);  // a stream id outside the cache: nothing to score against
            const int32_t* mem = a.members + (size_t)max(sid, 0) * a.k_max;
            nx_ids[0] = lane < nx_k ? mem[lane] : 0;
            nx_ids[1] = lane + kWarp < nx_k ? mem[lane + kWarp] : 0;
        }
        for (int u = 0; u < nu; ++u) {
            const int k = nx_k;
            const int ids[2] = {nx_ids[0], nx_ids[1]};  // lane l knows the classes of slots l and l + 32
            const int buf = u % kSvBufs, x = u % kRx;
            int nb_sid = 0;
            if (u + 1 < nu) {
                const int nb = my_units[u + 1];
                nb_sid = a.stream_id ? a.stream_id[nb] : 0;  // in flight while this frame is scored
            }
            // The CTAs of a cluster take turns at finishing: frame u goes to CTA u % P.  This part's
            // row of receive buffer x over there:
            const int fin = u % P;
            const uint32_t out = peer_smem(rx + (x * (P + 2) + rank) * kRxRow, fin);
            // the centre slice of this warp's first slot is fetched while the slice of the
            // semantic vector is still being pooled
            float4 cc[kMaxSlice / 4 / kWarp];  // every load of a slot in flight at once
            float clen = 0.f;
            if (dw < k) {
                const int cls = __shfl_sync(kFull, ids[0], dw);
                const float4* crow = reinterpret_cast<const float4*>(a.centers + (size_t)cls * p.C + sb);
                if (rank == fin && lane == 0) clen = a.cnorm[cls];
#pragma unroll
                for (int r = 0; r < kMaxSlice / 4 / kWarp; ++r) {
                    const int q = lane + r * kWarp;
                    cc[r] = q < n4 ? crow[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
            if (!mbar_wait_bounded(&sv_full[buf], (u / kSvBufs) & 1, p.status)) { failed = true; break; }
            if (u >= kRx && !mbar_wait_cluster_bounded(&rx_empty[x], (u / kRx - 1) & 1, p.status)) { failed = true; break; }
            const float4* v4 = reinterpret_cast<const float4*>(sv_s + buf * f.slice_cap);
            int* meta_ids = reinterpret_cast<int*>(rx + (x * (P + 2) + P) * kRxRow);  // in the finishing CTA only
            float* meta_len = rx + (x * (P + 2) + P + 1) * kRxRow;
            if (rank == fin && dw == 0) {  // the slots' classes and k, in the layout the finisher's lanes want
                meta_ids[lane] = ids[0];
                meta_ids[lane + kWarp] = ids[1];
                if (lane == 0) meta_ids[kFusedMaxK] = k;
            }
            if (dw == kDotWarps - 1) {  // partial squared length of the semantic vector
                float nn = 0.f;
                for (int q = lane; q < n4; q += kWarp) {
                    const float4 xv = v4[q];
                    nn = fmaf(xv.x, xv.x, nn); nn = fmaf(xv.y, xv.y, nn); nn = fmaf(xv.z, xv.z, nn); nn = fmaf(xv.w, xv.w, nn);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(kFull, nn, o);
                if (lane == 0) peer_store(out + kFusedMaxK * 4, nn);
            }
            for (int j = dw; j < k; j += kDotWarps) {  // partial dot product of slot j (Eq. 1's numerator)
                if (j != dw) {  // the first slot's loads are already under way
                    const int cls = __shfl_sync(kFull, (j & 32) ? ids[1] : ids[0], j & 31);
                    const float4* crow = reinterpret_cast<const float4*>(a.centers + (size_t)cls * p.C + sb);
                    if (rank == fin && lane == 0) clen = a.cnorm[cls];  // in flight with the centre
#pragma unroll
                    for (int r = 0; r < kMaxSlice / 4 / kWarp; ++r) {
                        const int q = lane + r * kWarp;
                        cc[r] = q < n4 ? crow[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                float d = 0.f;
#pragma unroll
                for (int r = 0; r < kMaxSlice / 4 / kWarp; ++r) {
                    const int q = lane + r * kWarp;
                    if (q < n4) {
                        const float4 xv = v4[q];
                        d = fmaf(cc[r].x, xv.x, d); d = fmaf(cc[r].y, xv.y, d);
                        d = fmaf(cc[r].z, xv.z, d); d = fmaf(cc[r].w, xv.w, d);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(kFull, d, o);
                if (lane == 0) {
                    peer_store(out + j * 4, d);
                    if (rank == fin) meta_len[j] = clen;
                }
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&sv_empty[buf]);
                peer_arrive(peer_smem(&rx_full[x], fin));  // this warp's share of the part has been delivered
            }
            if (u + 1 < nu) {  // fast memory of the next frame (its stream id has arrived by now)
                nb_sid = stream_checked(a, nb_sid);
                nx_k = nb_sid < 0 ? 0 : min(a.k[nb_sid], kFusedMaxK);
                const int32_t* mem = a.members + (size_t)max(nb_sid, 0) * a.k_max;
                nx_ids[0] = lane < nx_k ? mem[lane] : 0;
                nx_ids[1] = lane + kWarp < nx_k ? mem[lane + kWarp] : 0;
            }
        }
    } else {
        // ---- finisher warp: every P-th frame of the cluster; lane l looks after slots l and l + 32 ----
        const float weight = float(1u << a.layer);  // 2^(l-1) with l = layer + 1
        const int reuse = max(P, kRx);              // frames between two uses of a receive buffer in this CTA
        for (int u = rank; u < nu; u += P) {
            const int b = my_units[u], x = u % kRx;
            float sa_old[2];  // the carry, fetched while the frame is being scored
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + h * kWarp;
                sa_old[h] = (j < a.k_max && !a.fresh) ? a.sa[(size_t)b * a.k_max + j] : 0.f;
            }
            if (!mbar_wait_cluster_bounded(&rx_full[x], (u / reuse) & 1, p.status)) { failed = true; break; }
            const int* meta_ids = reinterpret_cast<const int*>(rx + (x * (P + 2) + P) * kRxRow);
            const float* meta_len = rx + (x * (P + 2) + P + 1) * kRxRow;
            const int k = meta_ids[kFusedMaxK];
            const int ids[2] = {meta_ids[lane], meta_ids[lane + kWarp]};
            const float clen[2] = {lane < k ? meta_len[lane] : 0.f, lane + kWarp < k ? meta_len[lane + kWarp] : 0.f};
            float nn = 0.f, dots[2] = {0.f, 0.f};
            for (int r = 0; r < P; ++r) {  // the parts in rank order
                const float* row = rx + (x * (P + 2) + r) * kRxRow;
                nn += row[kFusedMaxK];
                if (lane < k) dots[0] += row[lane];
                if (lane + kWarp < k) dots[1] += row[lane + kWarp];
            }
            __syncwarp();
            // every rank may fill buffer x again; nobody waits for that after the last kRx frames
            if (lane < P && u + kRx < nu) peer_arrive(peer_smem(&rx_empty[x], lane));
            float s_cur[2] = {0.f, 0.f}, s_acc[2] = {0.f, 0.f};
            const float sv_len = __fsqrt_rn(nn);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + h * kWarp;
                if (j < k) {
                    s_cur[h] = (nn == 0.f || clen[h] == 0.f) ? 0.f : __fdiv_rn(dots[h], __fmul_rn(sv_len, clen[h]));  // Eq. 1
                    s_acc[h] = __fmaf_rn(s_cur[h], weight, sa_old[h]);   // Eq. 3
                    a.sa[(size_t)b * a.k_max + j] = s_acc[h];
                } else if (a.fresh && j < a.k_max) {
                    a.sa[(size_t)b * a.k_max + j] = 0.f;                 // unused slots start from zero too
                }
            }
            const Top2 ta = warp_top2_keys(s_acc, ids, k, lane);
            Top2 ts{0.f, 0.f, -1, -1};
            if (a.sep) ts = warp_top2_keys(s_cur, ids, k, lane);  // only Eq. 2 (a diagnostic) needs it
            if (lane == 0) {
                const int r = decide_core<true>(a, b, ta, ts);
                s_ctr[0] += 1u;  // only this lane touches the tallies until the CTA is done
                if (r & 2) s_ctr[1] += 1u;
                if (r & 1) s_ctr[2] += 1u;
            }
        }
    }
    // No thread leaves before every copy that was issued has landed, and no CTA before its
    // peers are done with its shared memory.
    const int any_failed = __syncthreads_or(failed ? 1 : 0);
    if (threadIdx.x < 3 && s_ctr[threadIdx.x]) {  // this CTA's tallies: lookups, near-threshold, exits
        const int slot = threadIdx.x == 0 ? SMTM_CTR_LOOKUPS : threadIdx.x == 1 ? SMTM_CTR_NEAR : SMTM_CTR_EXITS + a.layer;
        atomicAdd(&a.counters[slot], (unsigned long long)s_ctr[threadIdx.x]);
    }
    if (any_failed && warp == kReducersF && lane == 0) {
        for (int s = 0; s < kStages && s < issued; ++s) {
            const uint32_t last_use = uint32_t((issued - 1 - s) / kStages);
            mbar_wait_bounded(&full[s], last_use & 1, p.status);
        }
    }
    __syncthreads();
    if (P > 1) cluster_sync_all();
}

// ---- pooling of the few frames still in at a later layer, by small CTAs ------------------------
//
// When most frames have left at an earlier layer, the streaming kernel above is the wrong tool: it
// wants a whole SM per CTA, and on a device whose SMs are held by another streaming kernel (the
// pooling of the next step's first layer, see the pipelined route in api.cu) it would wait for one.
// This kernel pools the active frames with CTAs of 128 threads and a single 12.5 KB stage, so that
// several fit beside such a kernel.  The grid is cpf x G CTAs: CTA c looks after chunk c % cpf of the
// active frames number c / cpf, c / cpf + G, ... (every CTA compacts the list of active frames for
// itself, as the fused kernel does).  A chunk is fetched with plain coalesced 16-byte loads, all in
// flight at once, and reduced by the reducers of the streaming kernel, the warps sharing its
// channels.  (Small batches of short channels are pooled by other reducers where no ring is used, so that the last bits of a
// frame's vector depend on the kernel its batch is served by; the same call gives the same bits.)
constexpr int kLightThreads = 128;
constexpr int kLightStageCap = 12800;   // bytes of a chunk here (half a stage of the streaming kernel)
constexpr int kLightFrames = 256;       // frames a CTA can be given

struct LightParams {
    NchwParams e;   // chunking as for the streaming kernel, with chunks of at most kLightStageCap bytes
    int groups;     // G
    int gran;       // channels that must stay in one warp's share (the reducer's unit)
};

template <class R>
__global__ void __launch_bounds__(kLightThreads) k_pool_sparse(const LightParams f) {
    __shared__ __align__(16) uint8_t stage[kLightStageCap];
    __shared__ int my_frames[kLightFrames];
    __shared__ int s_scan[33];
    const NchwParams& p = f.e;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int B = p.B;
    const int ci = int(blockIdx.x) % p.chunks_per_frame, group = int(blockIdx.x) / p.chunks_per_frame;
    chain_wait();  // the exit flags are the previous kernel's
    chain_release();
    const ClockScope stamps(p.clock);
    uint8_t flags[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int n_active = 0;
    for (int t0 = 0; t0 < B; t0 += kLightThreads) {
        const int b = t0 + tid;
        int act = b < B ? 1 : 0;
        if (p.skip) {  // the flags of eight tiles in one trip to memory
            if ((t0 / kLightThreads) % 8 == 0) {
#pragma unroll
                for (int u = 0; u < 8; ++u) flags[u] = p.skip[min(b + u * kLightThreads, B - 1)];
            }
            uint8_t mine = 0;
#pragma unroll
            for (int u = 0; u < 8; ++u) mine = ((t0 / kLightThreads) % 8 == u) ? flags[u] : mine;
            act = (b < B && !mine) ? 1 : 0;
        }
        int cnt;
        const int pos = block_exclusive_scan(act, s_scan, &cnt);
        if (act) {
            const int u = n_active + pos;
            if (u % f.groups == group && u / f.groups < kLightFrames) my_frames[u / f.groups] = b;
        }
        n_active += cnt;
    }
    const int nu = n_active > group ? min((n_active - group + f.groups - 1) / f.groups, kLightFrames) : 0;
    __syncthreads();
    const int c0 = ci * p.chunk_channels;
    const int nch = min(p.chunk_channels, p.C - c0);
    const int vectors = nch * p.ch_bytes / 16;
    // this warp's share of the chunk's channels (whole reducer units)
    const int units = (nch + f.gran - 1) / f.gran;
    const int u_lo = min(units, warp * ((units + 3) / 4)), u_hi = min(units, u_lo + (units + 3) / 4);
    const int w_c0 = u_lo * f.gran, w_nch = min(nch, u_hi * f.gran) - w_c0;
    for (int k = 0; k < nu; ++k) {
        const int b = my_frames[k];
        const uint4* src = reinterpret_cast<const uint4*>(p.x + (long long)b * p.frame_bytes + (long long)c0 * p.ch_bytes);
        uint4* dst = reinterpret_cast<uint4*>(stage);
        for (int v0 = 0; v0 < vectors; v0 += 8 * kLightThreads) {  // eight loads per thread in flight
            uint4 r[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) r[u] = load_once(src + min(v0 + u * kLightThreads + tid, vectors - 1));
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (v0 + u * kLightThreads + tid < vectors) dst[v0 + u * kLightThreads + tid] = r[u];
        }
        __syncthreads();
        if (w_nch > 0)
            R::run(stage + size_t(w_c0) * p.ch_bytes, 0, w_nch, lane, p.sv + (long long)b * p.C + c0 + w_c0, nullptr, p.inv_hw, p);
        __syncthreads();  // the stage is free for the next frame
    }
}

// ---- the same frames looked up whole: pooling, scoring and the decision by a cluster of small CTAs ----
//
// A thread-block cluster of P CTAs takes active frames one at a time; CTA `rank` fetches chunk `rank` of the
// frame (one trip to memory for the whole frame), pools it, and scores its slice of the semantic vector
// against the frame's fast-memory centres; the partial dot products and the partial squared length go
// through distributed shared memory to the cluster's first CTA, whose first warp adds the parts in rank
// order and decides (Eq. 1, Eq. 3, top-2, Eq. 4, the exit rule), as the fused streaming kernel does.  One
// cluster-wide barrier per frame; two receive buffers take turns.  P = chunks per frame <= 8, and a chunk
// here is a chunk of the streaming kernel (<= 25 KB): a whole frame is in flight at once.  What bounds it beside the pooling
// kernel is how many clusters find a place.  With a whole chunk in shared memory three CTAs fit on an SM, and 55 clusters of
// eight not all on the chip: the last ones began when the first were done (51 frames of 2048 7x7 channels out of 512 30 us,
// alone 17).  With kHalves one half of a chunk is on its way to shared memory and the other to registers, from where it
// follows, and four CTAs fit: a step of 512 streams 52.5 -> 47.4 us.  Where the frames are few enough for one round the
// second pass is the longer way (64 frames in four exit layers 62.9 us a step, 65.2 in halves; 200 frames of 512 15x15 and
// 1024 8x8 channels 38.0 and 39.6), so halves are for batches of more than four times the clusters that fit with whole
// chunks (a later layer has a fraction of the batch).
constexpr int kSparseStageCap = kStageCap;
constexpr int kSparseFrames = 64;    // frames a cluster can be given
constexpr int kSparseSlice = 1024;   // channels of a chunk at most (as the fused kernel's slices)
// Up to eight CTAs to an SM a frame has a cluster of its own, which leaves at once if the frame has: nothing is listed, and no
// decision has to wait for the end of the launch.  A step of 40 frames in two layers, a tenth still in, 24.5 -> 23.3 us (clusters
// of eight), of 512 frames in single CTAs 27.1 -> 25.8; beyond, the clusters that leave cost more than the list and
// k_settle_exits: 256 frames in clusters of eight, half of them still in, 43.2 and 44.9.
constexpr int kSparseOwn = 8;

struct SparseParams {
    NchwParams e;
    LookupArgs a;
    int groups;  // clusters
    int gran;    // channels that must stay in one warp's share (the reducer's unit)
    int staged;  // channels of a chunk that the stage holds
};

constexpr size_t sparse_smem(int slice, size_t stage) {
    return (stage + 15) / 16 * 16 + size_t(slice) * 4 + 2 * size_t(kMaxCluster) * kRxRow * 4 + 2 * kSparseFrames * 4 + 64 * 4 + 64;
}

// (Registers for three or four CTAs to an SM beside the 128 threads of the pooling kernel.)
template <class R, bool kHalves>
__global__ void __launch_bounds__(kLightThreads, kHalves ? 5 : 4) k_lookup_sparse(const SparseParams f) {
    extern __shared__ uint8_t smem_raw[];
    const NchwParams& p = f.e;
    const LookupArgs& a = f.a;
    uint8_t* stage = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 15) & ~uintptr_t(15));
    float* sv_s = reinterpret_cast<float*>(stage + ((size_t(f.staged) * p.ch_bytes + 15) & ~size_t(15)));  // [chunk_channels] this CTA's slice
    float* rx = sv_s + p.chunk_channels;                                   // [2][P][kRxRow] (used in the first CTA)
    int* my_frames = reinterpret_cast<int*>(rx + 2 * kMaxCluster * kRxRow);  // [kSparseFrames]
    int* my_sids = my_frames + kSparseFrames;                              // [kSparseFrames] their stream ids
    int* s_scan = my_sids + kSparseFrames;                                 // [33]
    const int P = p.chunks_per_frame;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int B = a.B;
    const int rank = int(blockIdx.x) % P, group = int(blockIdx.x) / P;
    chain_wait();  // the exit flags are the previous kernel's
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * a.layer : nullptr);
    // The active frames of this cluster and their streams: the cluster's own, or from a list, for which every thread looks
    // at four consecutive frames, one trip to memory and one scan for 512.  Where the clusters do not all fit beside the streaming kernel, one of the first may have
    // decided a frame before the last ones begin: its exit is pending, the flag is what it was before the launch, so that
    // every cluster gets the same list whenever it looks.
    constexpr int kPer = 4;
    int n_active = 0;
    if (!a.pending) {  // a cluster per frame
        const int sid = a.stream_id ? a.stream_id[group] : 0;  // in flight with the exit flag
        if (a.done[group]) return;
        if (tid == 0) {
            my_frames[0] = group;
            my_sids[0] = sid;
        }
        n_active = B;
    }
    for (int t0 = 0; a.pending && t0 < B; t0 += kPer * kLightThreads) {
        const int b0 = t0 + tid * kPer;
        int act[kPer], sids[kPer], mine = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            act[i] = a.done[min(b0 + i, B - 1)];
            sids[i] = a.stream_id ? a.stream_id[min(b0 + i, B - 1)] : 0;
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            act[i] = (b0 + i < B && act[i] == 0) ? 1 : 0;
            mine += act[i];
        }
        int cnt;
        int u = n_active + block_exclusive_scan(mine, s_scan, &cnt);
#pragma unroll
        for (int i = 0; i < kPer; ++i)
            if (act[i]) {
                const int at = u / f.groups;
                if (u - at * f.groups == group && at < kSparseFrames) {
                    my_frames[at] = b0 + i;
                    my_sids[at] = sids[i];
                }
                ++u;
            }
        n_active += cnt;
    }
    const int nu = n_active > group ? min((n_active - group + f.groups - 1) / f.groups, kSparseFrames) : 0;
    __syncthreads();
    if (P > 1) cluster_arrive_relaxed();  // (waited for before the first store to a peer: it has to have started)
    const int c0 = rank * p.chunk_channels;
    const int nch = min(p.chunk_channels, p.C - c0);   // channels of this CTA's slice (a multiple of 4)
    const int vectors = nch * p.ch_bytes / 16;
    const int n4 = nch >> 2;
    const int pp = (n4 + kWarp - 1) / kWarp;       // 16-byte pieces of a centre's slice per lane (at most 8)
    const int spr = max(1, 8 / max(pp, 1));        // slots a warp scores per trip to memory
    const float weight = float(1u << a.layer);     // 2^(l-1) with l = layer + 1
    constexpr int kLoads = (kSparseStageCap / 2 / 16 + kLightThreads - 1) / kLightThreads;  // 7: the second half of a chunk
    const int first = kHalves ? min(nch, f.staged) : nch, v_first = first * p.ch_bytes / 16;
    for (int k_it = 0; k_it < nu; ++k_it) {
        const int b = my_frames[k_it];
        const int sid = stream_checked(a, my_sids[k_it]);
        const uint4* src = reinterpret_cast<const uint4*>(p.x + (long long)b * p.frame_bytes + (long long)c0 * p.ch_bytes);
        uint4* dst = reinterpret_cast<uint4*>(stage);
        for (int v = tid; v < v_first; v += kLightThreads)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + v)), "l"(src + v) : "memory");
        uint4 r[kHalves ? kLoads : 1];
        if (kHalves) {
#pragma unroll
            for (int u = 0; u < kLoads; ++u) r[u] = load_once(src + min(v_first + u * kLightThreads + tid, vectors - 1));
        }
        // the frame's fast memory: its size and this warp's classes (slot j = warp + 4 i), in flight with the chunk
        const int32_t* mem = a.members + (size_t)max(sid, 0) * a.k_max;
        const int k = sid < 0 ? 0 : min(a.k[sid], kFusedMaxK);
        int cls_w = 0;  // lane i < 16 holds the class of slot warp + 4 i
        if (lane < kFusedMaxK / 4 && warp + 4 * lane < a.k_max) cls_w = mem[warp + 4 * lane];
        // the finisher's own loads: the slots' classes (lane l: slots l and l + 32)
        int ids[2] = {0, 0};
        if (rank == 0 && warp == 0) {
            ids[0] = lane < a.k_max ? mem[lane] : 0;
            ids[1] = lane + kWarp < a.k_max ? mem[lane + kWarp] : 0;
        }
        const auto pool = [&](int h0, int hn) {  // the channels h0 .. of the chunk, by all warps: whole units each
            const int share = ((hn + f.gran - 1) / f.gran + 3) / 4 * f.gran;
            const int w_c0 = min(hn, warp * share), w_nch = min(hn, w_c0 + share) - w_c0;
            if (w_nch > 0)
                R::run(stage + size_t(w_c0) * p.ch_bytes, 0, w_nch, lane, p.sv + (long long)b * p.C + c0 + h0 + w_c0, sv_s + h0 + w_c0,
                       p.inv_hw, p);
        };
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        pool(0, first);
        __syncthreads();  // the first part of the slice is complete, the stage free
        if (kHalves && first < nch) {
#pragma unroll
            for (int u = 0; u < kLoads; ++u)
                if (v_first + u * kLightThreads + tid < vectors) dst[u * kLightThreads + tid] = r[u];
            __syncthreads();
            pool(first, nch - first);
            __syncthreads();
        }
        if (P > 1 && k_it == 0) cluster_wait();
        const uint32_t out = peer_smem(rx + ((k_it & 1) * kMaxCluster + rank) * kRxRow, 0);
        const float4* v4 = reinterpret_cast<const float4*>(sv_s);
        // the centres' lengths and the carry, for the finisher: in flight with the centre slices below
        float clen[2] = {0.f, 0.f}, sa_old[2] = {0.f, 0.f};
        if (rank == 0 && warp == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + h * kWarp;
                if (j < k) {
                    clen[h] = a.cnorm[ids[h]];
                    sa_old[h] = a.fresh ? 0.f : a.sa[(size_t)b * a.k_max + j];
                }
            }
        }
        if (warp == 3) {  // partial squared length of the semantic vector
            float nn = 0.f;
            for (int q = lane; q < n4; q += kWarp) {
                const float4 xv = v4[q];
                nn = fmaf(xv.x, xv.x, nn); nn = fmaf(xv.y, xv.y, nn); nn = fmaf(xv.z, xv.z, nn); nn = fmaf(xv.w, xv.w, nn);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(kFull, nn, o);
            if (lane == 0) peer_store(out + kFusedMaxK * 4, nn);
        }
        // this warp's slots, `spr` of them per trip to memory: eight pieces of centre slices per lane in flight
        for (int i0 = 0; warp + 4 * i0 < k; i0 += spr) {
            float4 c[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int si = e / pp, piece = e - si * pp;       // slot within the round, piece of its slice
                const int j = warp + 4 * (i0 + si), q = lane + piece * kWarp;
                const int cls = __shfl_sync(kFull, cls_w, min(i0 + si, kFusedMaxK / 4 - 1));
                c[e] = (si < spr && j < k && q < n4)
                           ? reinterpret_cast<const float4*>(a.centers + (size_t)cls * p.C + c0)[q]
                           : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            for (int si = 0; si < spr; ++si) {
                const int j = warp + 4 * (i0 + si);
                if (j >= k) break;
                float d = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int q = lane + (e - si * pp) * kWarp;
                    if (e / pp == si && q < n4) {
                        const float4 xv = v4[q];
                        d = fmaf(c[e].x, xv.x, d); d = fmaf(c[e].y, xv.y, d); d = fmaf(c[e].z, xv.z, d); d = fmaf(c[e].w, xv.w, d);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(kFull, d, o);
                if (lane == 0) peer_store(out + j * 4, d);
            }
        }
        // every part of this frame has been delivered (and the previous frame's decision is made)
        if (P > 1) cluster_sync_all(); else __syncthreads();
        if (rank == 0 && warp == 0) {
            const float* rxb = rx + (k_it & 1) * kMaxCluster * kRxRow;
            float nn = 0.f, dots[2] = {0.f, 0.f};
            for (int rr = 0; rr < P; ++rr) {  // the parts in rank order
                const float* row = rxb + rr * kRxRow;
                nn += row[kFusedMaxK];
                if (lane < k) dots[0] += row[lane];
                if (lane + kWarp < k) dots[1] += row[lane + kWarp];
            }
            float s_cur[2] = {0.f, 0.f}, s_acc[2] = {0.f, 0.f};
            const float sv_len = __fsqrt_rn(nn);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + h * kWarp;
                if (j < k) {
                    s_cur[h] = (nn == 0.f || clen[h] == 0.f) ? 0.f : __fdiv_rn(dots[h], __fmul_rn(sv_len, clen[h]));  // Eq. 1
                    s_acc[h] = __fmaf_rn(s_cur[h], weight, sa_old[h]);   // Eq. 3
                    a.sa[(size_t)b * a.k_max + j] = s_acc[h];
                } else if (a.fresh && j < a.k_max) {
                    a.sa[(size_t)b * a.k_max + j] = 0.f;                 // unused slots start from zero too
                }
            }
            const Top2 ta = warp_top2_keys(s_acc, ids, k, lane);
            Top2 ts{0.f, 0.f, -1, -1};
            if (a.sep) ts = warp_top2_keys(s_cur, ids, k, lane);  // only Eq. 2 (a diagnostic) needs it
            if (lane == 0) decide_from_top2<true>(a, b, ta, ts);
        }
    }
    if (P > 1 && nu == 0) cluster_wait();
    else if (P > 1) cluster_sync_all();  // no CTA leaves while a peer may still write to its shared memory
}

// ---- lookup of small frames: a cluster of small CTAs per frame, nothing persistent -----------------
//
// With little to stream (shallow exits with tiny maps, a single camera's frame) a lookup is bound by the number of
// dependent trips to memory and by what a CTA sets up before the first one, not by bytes.  CTA `rank` of the
// frame's cluster takes a slice of the semantic vector: [exit flag, stream id] -> [its part of the map, the fast
// memory's size and classes] -> [centre slices, lengths, carries, while the map lands] -> decision.  The partial dot
// products meet in the first CTA through distributed shared memory, whose first warp decides; a frame that has
// exited costs CTAs that leave at once.
constexpr int kFrameWarps = 8;
constexpr int kFrameThreads = kFrameWarps * kWarp;
constexpr int kFrameSlice = 8192;           // channels of a slice at most
constexpr int kFrameStageCap = 104 * 1024;    // bytes of a slice of an NCHW map at most
// A frame has as few CTAs as its slices fit, more until every SM has half a CTA, and few bytes stay a CTA's own.  With 32
// slots and more the scoring counts too, and is shared: slices of up to 64 KB instead of 104, down to 4 KB instead of 8.
// A cluster per frame is refused where its CTAs would queue up twice (with many slots four times) over what the chip holds
// of them, two to an SM: 69 frames of 56x56x32 fp32 channels 17.0 us in clusters of eight, 10.7 by the streaming kernel.
// Small frames that are all new, in a crowd, with a few slots each are bound by the CTAs a frame costs and are pooled and
// scored apart: from 3 to an SM (630 frames of 96 20x20 16-bit channels 21.4 us here, 16.4 apart), narrow channels from 2
// to an SM (1727 frames of 128 3x3 ones 22.9 and 13.8).
constexpr int kFrameStageWanted = 104 * 1024, kFrameStageWantedMany = 64 * 1024;  // bytes of a slice that a cluster is enlarged for
constexpr int kFrameStageLeast = 8 * 1024, kFrameStageLeastMany = 4 * 1024;       // ... below which it is not enlarged to fill the chip
constexpr int kFrameManySlots = 32, kFrameResident = 2;                           // CTAs an SM holds
constexpr int kCrowdSlots = 8, kCrowdNarrowSlots = 16, kCrowdFrame = 128 * 1024;
constexpr long long kFrameBatchMost = 64ll << 20;  // bytes of the batch above which the streaming kernel takes over
// When a cluster shares a frame of an NHWC map (its CTAs have half the threads of the CTA that takes a frame alone, and wait
// for one another's column sums).  Lookups: up to half as many frames as SMs, frames of 96 KB and more, six pixels a thread of the CTA it
// replaces and more, as many CTAs as the chip holds at once (768 KB: twice as many).  With 32 slots and more the clusters also share the scoring: a CTA on every SM at least; so do, with 16, the handful of
// frames of a stream or a few.  In
// geometric mean over 525 lookups of 1 .. 2048 frames 20 % faster than a CTA per frame; the line it replaces, which let four
// CTAs to an SM in, gave 15 %, and 139 frames of 48x48x256 16-bit channels took 61 us against 34 by a CTA each.
constexpr int kNhwcShared = 96 * 1024, kNhwcLong = 768 * 1024;  // bytes of a frame
constexpr int kNhwcManySlots = 32, kNhwcManyLeast = 32 * 1024, kNhwcPixels = 6;
constexpr int kNhwcSomeSlots = 16, kNhwcSomeLeast = 24 * 1024;
// Pooling alone: a CTA keeps what its threads ask for in one trip, eight loads each; beyond that the frame is shared, three
// CTAs to an SM at most (19 frames of 40x40x40 16-bit channels 6.0 us by a CTA each, 4.7 in clusters, but one of
// 13x14x64, six pixels a thread, 3.0 and 4.1).  Parts of 64 KB and more fill what four CTAs to an SM leave: a warm-up with
// 512 frames of 28x28x512 16-bit channels 114 us by a CTA each, 108 in clusters of two.
constexpr int kNhwcPoolLoads = 8;
constexpr int kNhwcPartLong = 64 * 1024;

struct FrameParams {
    NchwParams e;
    LookupArgs a;
    int parts;  // P: CTAs per frame
    int slice;  // channels per CTA
    int gran;   // channels that must stay in one warp's share
};

// What the scorers of a frame fetch before its semantic vector is known: the fast memory's size, the classes of this
// warp's slots (slot j = warp + kFrameWarps * i in lane i) and, in the warp that decides, of all slots.
struct FrameSlots {
    int k, cls_w, ids[2];
};
__device__ __forceinline__ FrameSlots fetch_slots(const LookupArgs& a, int sid, bool decides) {
    FrameSlots s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int32_t* mem = a.members + (size_t)max(sid, 0) * a.k_max;
    s.k = sid < 0 ? 0 : min(a.k[sid], kFusedMaxK);  // a stream id outside the cache: nothing to score against
    const int j = warp + kFrameWarps * lane;
    s.cls_w = j < min(a.k_max, kFusedMaxK) ? mem[j] : 0;
    s.ids[0] = decides && lane < a.k_max ? mem[lane] : 0;
    s.ids[1] = decides && lane + kWarp < a.k_max ? mem[lane + kWarp] : 0;
    return s;
}

// The pieces of the centres' slices (channels c0 .., n4 16-byte pieces) for `8 >> lg` slots of this warp, from the
// warp's slot number i0 on; a slot has at most 1 << lg pieces per lane at a time, from piece q0 on.
__device__ __forceinline__ void fetch_centres(const LookupArgs& a, const FrameSlots& s, int i0, int lg, int c0, int q0, int n4,
                                              float4 (&c)[8]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int i = i0 + (e >> lg), q = q0 + lane + (e & ((1 << lg) - 1)) * kWarp;
        const int cls = __shfl_sync(kFull, s.cls_w, min(i, kWarp - 1));
        c[e] = (warp + kFrameWarps * i < s.k && q < n4) ? reinterpret_cast<const float4*>(a.centers + (size_t)cls * a.D + c0)[q]
                                                        : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// An entry of the semantic vector whose pixels did not arrive before the wait for them gave up (which the status word records):
// it makes every similarity of the frame a NaN, and a NaN exceeds no threshold, so that nothing is decided from it.
constexpr float kNeverArrived = __builtin_nanf("");

// A part's value for the CTA that decides: counted on its barrier, or (bar == 0, a cluster of one) a plain store.
__device__ __forceinline__ void deliver(uint32_t addr, float v, uint32_t bar) {
    if (bar) peer_store_counted(addr, v, bar);
    else peer_store(addr, v);
}
// What the deciding CTA's barrier has to count: a dot product per slot and a squared length from every part.
__device__ __forceinline__ uint32_t parts_bytes(int P, int k) { return uint32_t(P) * uint32_t(k + 1) * 4u; }

// Eq. 1's partial dot products of this warp's slots over the slice, into this part's row of the receive buffer in the
// cluster's first CTA (`row`: its address there; bar: 0, or the barrier there that counts what arrives).  c: the pieces of the first slots, fetched already.  Eight sums are
// reduced over the warp together, halving what is left to exchange at every step: nine shuffles for eight.
__device__ __forceinline__ void score_slots(const LookupArgs& a, const FrameSlots& s, int lg, int c0, int n4,
                                            const float4* v4, uint32_t row, uint32_t bar, float4 (&c)[8]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per_trip = 8 >> lg;
    for (int i0 = 0; warp + kFrameWarps * i0 < s.k; i0 += per_trip) {
        float d[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) d[e] = 0.f;
        for (int q0 = 0; q0 < n4; q0 += 8 * kWarp) {  // (once, but for slices of more than 1024 channels)
            if (i0 > 0 || q0 > 0) fetch_centres(a, s, i0, lg, c0, q0, n4, c);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int q = q0 + lane + (e & ((1 << lg) - 1)) * kWarp;
                const float4 x = q < n4 ? v4[q] : make_float4(0.f, 0.f, 0.f, 0.f);
                d[e] = fmaf(c[e].w, x.w, fmaf(c[e].z, x.z, fmaf(c[e].y, x.y, fmaf(c[e].x, x.x, d[e]))));
            }
        }
        if (lg >= 1) { d[0] += d[1]; d[2] += d[3]; d[4] += d[5]; d[6] += d[7]; }
        if (lg >= 2) { d[0] += d[2]; d[4] += d[6]; }
        if (lg >= 3) d[0] += d[4];
#pragma unroll
        for (int o = 16, half = 4; half > 0; o >>= 1, half >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int e = 0; e < half; ++e) {
                const float give = up ? d[e] : d[e + half], keep = up ? d[e + half] : d[e];
                d[e] = keep + __shfl_xor_sync(kFull, give, o);
            }
        }
        d[0] += __shfl_xor_sync(kFull, d[0], 2);
        d[0] += __shfl_xor_sync(kFull, d[0], 1);
        const int e = lane >> 2, j = warp + kFrameWarps * (i0 + (e >> lg));  // this lane's sum is number lane >> 2
        if ((lane & 3) == 0 && (e & ((1 << lg) - 1)) == 0 && j < s.k) deliver(row + j * 4, d[0], bar);
    }
}

// Squared length of the slice, by one warp.
__device__ __forceinline__ void slice_norm(const float4* v4, int n4, uint32_t row, uint32_t bar) {
    const int lane = threadIdx.x & 31;
    float nn = 0.f;
    for (int q = lane; q < n4; q += kWarp) {
        const float4 x = v4[q];
        nn = fmaf(x.x, x.x, nn); nn = fmaf(x.y, x.y, nn); nn = fmaf(x.z, x.z, nn); nn = fmaf(x.w, x.w, nn);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(kFull, nn, o);
    if (lane == 0) deliver(row + kFusedMaxK * 4, nn, bar);
}

// The decision by the first warp of the cluster's first CTA once every part's row is in: the parts added in rank
// order, Eq. 1, Eq. 3, top-2, Eq. 4 / Eq. 2, the exit rule.
__device__ __forceinline__ void decide_parts(const LookupArgs& a, int b, const FrameSlots& s, const float* rx, int P,
                                             const float (&clen)[2], const float (&sa_old)[2]) {
    const int lane = threadIdx.x & 31;
    float nn = 0.f, dots[2] = {0.f, 0.f};
    for (int r = 0; r < P; ++r) {
        const float* row = rx + r * kRxRow;
        nn += row[kFusedMaxK];
        if (lane < s.k) dots[0] += row[lane];
        if (lane + kWarp < s.k) dots[1] += row[lane + kWarp];
    }
    const float weight = float(1u << a.layer);  // 2^(l-1) with l = layer + 1
    const float sv_len = __fsqrt_rn(nn);
    float s_cur[2] = {0.f, 0.f}, s_acc[2] = {0.f, 0.f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = lane + h * kWarp;
        if (j < s.k) {
            s_cur[h] = (nn == 0.f || clen[h] == 0.f) ? 0.f : __fdiv_rn(dots[h], __fmul_rn(sv_len, clen[h]));  // Eq. 1
            s_acc[h] = __fmaf_rn(s_cur[h], weight, sa_old[h]);                                             // Eq. 3
            a.sa[(size_t)b * a.k_max + j] = s_acc[h];
        } else if (a.fresh && j < a.k_max) {
            a.sa[(size_t)b * a.k_max + j] = 0.f;  // unused slots start from zero too
        }
    }
    const Top2 ta = warp_top2_keys(s_acc, s.ids, s.k, lane);
    Top2 ts{0.f, 0.f, -1, -1};
    if (a.sep) ts = warp_top2_keys(s_cur, s.ids, s.k, lane);  // only Eq. 2 (a diagnostic) needs it
    if (lane == 0) decide_from_top2(a, b, ta, ts);
}

// Lengths of the centres and carries, for the deciding warp (in flight with the centres).
__device__ __forceinline__ void fetch_lengths(const LookupArgs& a, int b, const FrameSlots& s, float (&clen)[2], float (&sa_old)[2]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = lane + h * kWarp;
        clen[h] = j < s.k ? a.cnorm[s.ids[h]] : 0.f;
        sa_old[h] = (j < s.k && !a.fresh) ? a.sa[(size_t)b * a.k_max + j] : 0.f;
    }
}

// log2 of the 16-byte pieces of a slice per lane, rounded up.
__device__ __forceinline__ int pieces_log2(int n4) { return n4 <= kWarp ? 0 : n4 <= 2 * kWarp ? 1 : n4 <= 4 * kWarp ? 2 : 3; }

template <class R>
__global__ void __launch_bounds__(kFrameThreads, 2) k_lookup_frame(const FrameParams f) {
    extern __shared__ __align__(128) uint8_t frame_smem[];  // the map's slice | [slice] semantic vector | [P][kRxRow] receive rows
    __shared__ uint64_t landed[kFrameWarps];  // per warp: its share of the map
    __shared__ uint64_t delivered;            // the first CTA's: every part's values
    const NchwParams& p = f.e;
    const LookupArgs& a = f.a;
    const int P = f.parts;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = int(blockIdx.x) / P, rank = int(blockIdx.x) - b * P;
    // this warp's share of the slice's channels
    const int c0 = rank * f.slice, nch = max(0, min(f.slice, p.C - c0));
    const int groups = (nch + f.gran - 1) / f.gran;
    const int share = (groups + kFrameWarps - 1) / kFrameWarps * f.gran;
    const int w_c0 = min(nch, warp * share), w_nch = min(nch, w_c0 + share) - w_c0;
    const uint64_t stream_once = l2_evict_first_policy();
    if (lane == 0) {
        mbar_init(&landed[warp], 1);
        if (warp == 0) mbar_init(&delivered, 1);
        mbar_init_fence();
    }
    __syncwarp();
    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * a.layer : nullptr);
    const int sid_raw = a.stream_id ? a.stream_id[b] : 0;  // in flight with the exit flag
    // (the cluster cannot have decided yet: the decision waits for what every CTA delivers after all its threads are past here)
    if (!a.fresh && a.done[b]) return;
    if (P > 1) cluster_arrive();  // (waited for before the first store to a peer: it has to have started)
    const uint32_t bytes = uint32_t(w_nch) * uint32_t(p.ch_bytes);
    uint8_t* stage = frame_smem + size_t(w_c0) * p.ch_bytes;
    if (lane == 0 && bytes) {
        mbar_expect_tx(&landed[warp], bytes);
        bulk_load_hint(stage, p.x + (long long)b * p.frame_bytes + (long long)(c0 + w_c0) * p.ch_bytes, bytes, &landed[warp],
                       stream_once);
    }
    float* sv_s = reinterpret_cast<float*>(frame_smem + ((size_t(f.slice) * p.ch_bytes + 15) & ~size_t(15)));
    float* rx = sv_s + f.slice;
    const bool decides = rank == 0 && warp == 0;
    const int sid = stream_checked(a, sid_raw);
    const FrameSlots slots = fetch_slots(a, sid, decides);
    if (P > 1 && decides && lane == 0) mbar_expect_tx(&delivered, parts_bytes(P, slots.k));
    const int n4 = nch >> 2, lg = pieces_log2(n4);
    float4 cen[8];
    fetch_centres(a, slots, 0, lg, c0, 0, n4, cen);
    float clen[2] = {0.f, 0.f}, sa_old[2] = {0.f, 0.f};
    if (decides) fetch_lengths(a, b, slots, clen, sa_old);
    if (bytes) {
        if (__builtin_expect(mbar_wait_arrivals<false>(&landed[warp], 0, p.status), 1))
            R::run(stage, 0, w_nch, lane, p.sv + (long long)b * p.C + c0 + w_c0, sv_s + w_c0, p.inv_hw, p);
        else
            for (int c = lane; c < w_nch; c += kWarp) sv_s[w_c0 + c] = kNeverArrived;
    }
    __syncthreads();
    if (P > 1) cluster_wait();
    const uint32_t row = peer_smem(rx + rank * kRxRow, 0), bar = P > 1 ? peer_smem(&delivered, 0) : 0u;
    const float4* v4 = reinterpret_cast<const float4*>(sv_s);
    if (warp == kFrameWarps - 1) slice_norm(v4, n4, row, bar);
    score_slots(a, slots, lg, c0, n4, v4, row, bar, cen);
    if (P == 1) __syncthreads();
    if (decides && (P == 1 || mbar_wait_arrivals<true>(&delivered, 0, p.status)))  // every part has been delivered
        decide_parts(a, b, slots, rx, P, clen, sa_old);
}

// ---- NHWC, small fast memory: pooling, scoring and the decision by a cluster per frame ---------------
//
// A frame of an NHWC map is H*W rows of C channels: pooling is a column sum.  CTA `rank` of the frame's cluster sums a
// run of pixels (thread = 16-byte column group and pixel phase, several loads in flight), the phases are added in
// ascending order through shared memory, and then CTA r adds slice r of the columns over the cluster's CTAs in rank
// order (distributed shared memory) and goes on with that slice as the NCHW kernel above does.
struct FrameNhwcParams {
    const uint8_t* x;
    LookupArgs a;
    float* sv;
    int C, HW;
    float inv_hw;
    int parts;   // P: CTAs per frame
    int pixels;  // per CTA
    int slice;   // channels per CTA (a multiple of 4)
};

// First round of adding the phases' column sums up, so that narrow maps (24 channels of 16 bits: 85 phases in 256 threads)
// do not leave most threads idle: thread (g, c) adds the phases g, g + groups, ... in place.  Returns the rows that are
// left to add.  Up to 64 phases the second barrier costs more than the idle threads (lookups of 256-channel maps, 16 phases:
// 0.4 us of 6; 32-channel ones, 128 phases, gain 0.3).
constexpr int kFoldPhases = 64;
template <int T>
__device__ __forceinline__ int fold_phases(float* part, int phases, int cols) {
    const int groups = T / cols;
    if (groups <= 1 || phases <= kFoldPhases) return phases;
    const int g = threadIdx.x / cols, c = threadIdx.x - g * cols;
    if (g < groups) {
        float s = part[threadIdx.x];
        for (int q = g + groups; q < phases; q += groups) s += part[q * cols + c];
        part[threadIdx.x] = s;
    }
    __syncthreads();
    return groups;
}

// Sums pixels [px0, px1) of a frame over this CTA, U loads of a thread in flight; emit(c, sum) gets each column's, after one
// call of before() by all threads; `part`: T / cgs x cgs * V floats.
template <class E, int T, int U, class Before, class Emit>
__device__ __forceinline__ void column_sums(const uint8_t* frame, int C, int px0, int px1, float* part, Before before, Emit emit) {
    constexpr int V = E::kPerVec;
    const int CG = C / V;  // 16-byte vectors per pixel
    const uint4* f = reinterpret_cast<const uint4*>(frame);
    for (int cg0 = 0; cg0 < CG; cg0 += T) {
        const int cgs = min(CG - cg0, T);  // column groups handled in this sweep
        const int phases = T / cgs;
        const int ph = threadIdx.x / cgs, cg = threadIdx.x - ph * cgs;
        if (ph < phases) {
            float acc[V];
#pragma unroll
            for (int j = 0; j < V; ++j) acc[j] = 0.f;
            const uint4* col = f + cg0 + cg;
            int px = px0 + ph;
            for (; px + (U - 1) * phases < px1; px += U * phases) {
                uint4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = load_once(col + (long long)(px + u * phases) * CG);
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int j = 0; j < V; ++j) acc[j] += E::at(v[u], j);
            }
            if (px < px1) {
                uint4 v[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = load_once(col + (long long)min(px + u * phases, px1 - 1) * CG);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (px + u * phases < px1) {
#pragma unroll
                        for (int j = 0; j < V; ++j) acc[j] += E::at(v[u], j);
                    }
            }
            float4* dst = reinterpret_cast<float4*>(part + (size_t(ph) * cgs + cg) * V);
#pragma unroll
            for (int j = 0; j < V; j += 4) dst[j / 4] = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        }
        __syncthreads();
        const int cols = cgs * V, rows = fold_phases<T>(part, phases, cols);
        if (cg0 == 0) before();
        for (int c = threadIdx.x; c < cols; c += T) {
            float s = 0.f;
            for (int q = 0; q < rows; ++q) s += part[q * cols + c];
            emit(cg0 * V + c, s);
        }
        __syncthreads();
    }
}

// Column c's sum over this CTA's pixels to the CTA whose slice it belongs to: psum there holds a row of `slice` per CTA.
__device__ __forceinline__ void send_column(float* psum, uint64_t* bar, int c, int slice, int rank, float s) {
    const int r = c / slice;
    peer_store_counted(peer_smem(psum + rank * slice + (c - r * slice), r), s, peer_smem(bar, r));
}

// Pooling alone: CTA `rank` of a frame's cluster sums a run of its pixels, then slice `rank` of the columns over the
// cluster, as k_lookup_frame_nhwc does.
// 512 frames of 28x28x512 16-bit maps: 69 us with a CTA of four loads per thread each, 61 us here; 64 of them 54 and 11 us.
// kLoads: loads of a thread in flight.  With two or four pixels a thread the CTAs an SM holds count, and the registers of
// eight loads are in the way: 1895 frames of 10x10x40 fp32 channels 10.4 us with eight, 7.7 with four; 1181 of 4x4x64 ones
// 6.0, and 4.1 with two.
template <class E, int kLoads>
__global__ void __launch_bounds__(kFrameThreads, kLoads == 2 ? 8 : kLoads == 4 ? 6 : 4) k_encode_nhwc(const uint8_t* x, const uint8_t* skip, float* sv, int C, int HW, float inv_hw, int P,
                                                                  int pixels, int slice, __nv_bfloat16* hi, __nv_bfloat16* lo,
                                                                  int* status, unsigned long long* clock) {
    extern __shared__ __align__(16) float nhwc_smem[];  // column sums of this CTA's slice [P][slice] (clusters only) | phases' sums
    __shared__ uint64_t summed;                         // every CTA's sums of this slice are in
    float* psum = nhwc_smem;
    const int b = int(blockIdx.x) / P, rank = int(blockIdx.x) - b * P;
    if (P > 1 && threadIdx.x == 0) {
        mbar_init(&summed, 1);
        mbar_init_fence();
    }
    chain_wait();
    chain_release();
    const ClockScope stamps(clock);
    if (skip && skip[b]) return;  // (the same for the whole cluster)
    const int px0 = rank * pixels, px1 = min(HW, px0 + pixels);
    const auto write = [&](int c, float s) {
        s *= inv_hw;
        const long long at = (long long)b * C + c;
        sv[at] = s;
        if (hi) {
            const __nv_bfloat16 h = __float2bfloat16_rn(s);
            hi[at] = h;
            lo[at] = __float2bfloat16_rn(s - __bfloat162float(h));
        }
    };
    const uint8_t* frame = x + (long long)b * HW * C * E::kSize;
    if (P == 1) {
        column_sums<E, kFrameThreads, kLoads>(frame, C, 0, HW, psum, [] {}, write);
        return;
    }
    cluster_arrive();  // (waited for before the first store to a peer: it has to have started)
    const int c0 = rank * slice, c1 = min(C, c0 + slice);
    if (threadIdx.x == 0 && c1 > c0) mbar_expect_tx(&summed, uint32_t(P) * uint32_t(c1 - c0) * 4u);
    column_sums<E, kFrameThreads, kLoads>(frame, C, px0, px1, psum + P * slice, [] { cluster_wait(); },
                                          [&](int c, float s) { send_column(psum, &summed, c, slice, rank, s); });
    if (c1 <= c0 || !mbar_wait_arrivals<true>(&summed, 0, status)) return;
    for (int c = c0 + threadIdx.x; c < c1; c += kFrameThreads) {
        float s = 0.f;
        for (int r = 0; r < P; ++r) s += psum[r * slice + (c - c0)];
        write(c, s);
    }
}

template <class E>
__global__ void __launch_bounds__(kFrameThreads, 2) k_lookup_frame_nhwc(const FrameNhwcParams f) {
    extern __shared__ __align__(16) float nhwc_smem[];  // column sums of this CTA's slice [P][slice] | slice [slice] | receive rows [P][kRxRow] | phases' sums
    __shared__ uint64_t summed, delivered;              // every CTA's sums of this slice; the first CTA's: every part's values
    const LookupArgs& a = f.a;
    const int P = f.parts;
    float* psum = nhwc_smem;
    float* sv_s = psum + P * f.slice;
    float* rx = sv_s + f.slice;
    float* part = rx + P * kRxRow;
    const int warp = threadIdx.x >> 5;
    const int b = int(blockIdx.x) / P, rank = int(blockIdx.x) - b * P;
    if (threadIdx.x == 0) {
        mbar_init(&summed, 1);
        mbar_init(&delivered, 1);
        mbar_init_fence();
    }
    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * a.layer : nullptr);
    const int sid_raw = a.stream_id ? a.stream_id[b] : 0;  // in flight with the exit flag
    // (the cluster cannot have decided yet: the decision waits for what every CTA delivers after all its threads are past here)
    if (!a.fresh && a.done[b]) return;
    cluster_arrive();  // (waited for before the first store to a peer: it has to have started)
    const bool decides = rank == 0 && warp == 0;
    const int c0 = rank * f.slice, nch = max(0, min(f.slice, f.C - c0));
    const FrameSlots slots = fetch_slots(a, stream_checked(a, sid_raw), decides);  // in flight with the map
    if (threadIdx.x == 0 && nch > 0) mbar_expect_tx(&summed, uint32_t(P) * uint32_t(nch) * 4u);
    const int px0 = rank * f.pixels, px1 = min(f.HW, px0 + f.pixels);
    column_sums<E, kFrameThreads, 8>(f.x + (long long)b * f.HW * f.C * E::kSize, f.C, px0, px1, part, [] { cluster_wait(); },
                                     [&](int c, float s) { send_column(psum, &summed, c, f.slice, rank, s); });
    if (decides && threadIdx.x == 0) mbar_expect_tx(&delivered, parts_bytes(P, slots.k));
    const int n4 = nch >> 2, lg = pieces_log2(n4);
    float4 cen[8];
    fetch_centres(a, slots, 0, lg, c0, 0, n4, cen);  // in flight with the exchange
    float clen[2] = {0.f, 0.f}, sa_old[2] = {0.f, 0.f};
    if (decides) fetch_lengths(a, b, slots, clen, sa_old);
    const bool complete = nch <= 0 || mbar_wait_arrivals<true>(&summed, 0, a.status);
    for (int c = threadIdx.x; c < nch; c += kFrameThreads) {
        float s = 0.f;
        for (int r = 0; r < P; ++r) s += psum[r * f.slice + c];
        s = complete ? s * f.inv_hw : kNeverArrived;
        sv_s[c] = s;
        if (complete) f.sv[(long long)b * f.C + c0 + c] = s;
    }
    __syncthreads();
    const uint32_t row = peer_smem(rx + rank * kRxRow, 0), bar = peer_smem(&delivered, 0);
    const float4* v4 = reinterpret_cast<const float4*>(sv_s);
    if (warp == kFrameWarps - 1) slice_norm(v4, n4, row, bar);
    score_slots(a, slots, lg, c0, n4, v4, row, bar, cen);
    if (decides && mbar_wait_arrivals<true>(&delivered, 0, a.status))  // every part has been delivered
        decide_parts(a, b, slots, rx, P, clen, sa_old);
}

// ---- NHWC, small fast memory: pooling, scoring and the decision by one CTA per frame ---------------
//
// A frame of an NHWC map is H*W rows of C channels: pooling is a column sum, and one CTA holds all of a
// frame's column sums at the end, so the same CTA goes on to Eq. 1, Eq. 3, Eq. 4 and the exit rule (one
// launch per layer).  Thread = (16-byte column group, pixel phase); every thread keeps eight loads in
// flight (a frame is a few dozen KB: the CTA's time is the number of trips to memory it makes); the
// phases are added in ascending order through shared memory.  Frames that have exited cost a CTA that
// leaves at once.
constexpr int kThreadsNhwcLookup = 512;  // more threads, fewer trips to memory per thread: a frame is one CTA's

// (Two CTAs to an SM with eight elements to a piece, three with four.)
template <class E>
__global__ void __launch_bounds__(kThreadsNhwcLookup, E::kSize == 4 ? 3 : 2) k_lookup_nhwc(const uint8_t* x, int C, int HW, float inv_hw, float* sv_out,
                                                                    const LookupArgs a) {
    extern __shared__ float nhwc_smem[];  // sv [C] | s_cur [k_max] | s_acc [k_max] | classes [k_max] | part [phases][cgs * V]
    __shared__ float scratch[32];
    float* sv_s = nhwc_smem;
    float* s_cur = sv_s + C;
    float* s_acc = s_cur + a.k_max;
    float* part = s_acc + 2 * a.k_max;
    chain_wait();
    chain_release();
    const ClockScope stamps(a.clock ? a.clock + 2 * a.layer : nullptr);
    const int b = blockIdx.x;
    const int sid_raw = a.stream_id ? a.stream_id[b] : 0;  // in flight with the exit flag
    if (!a.fresh && a.done[b]) return;
    const SlotPrefetch pf = prefetch_slots(a, sid_raw);    // in flight with the map
    constexpr int V = E::kPerVec;
    constexpr int T = kThreadsNhwcLookup;
    const int CG = C / V;  // 16-byte vectors per pixel
    const uint4* f = reinterpret_cast<const uint4*>(x + (long long)b * HW * C * E::kSize);
    constexpr bool kOwnNorm = E::kSize == 2;
    float nrm = 0.f;
    for (int cg0 = 0; cg0 < CG; cg0 += T) {
        const int cgs = min(CG - cg0, T);  // column groups handled in this sweep
        const int phases = T / cgs;
        const int ph = threadIdx.x / cgs, cg = threadIdx.x - ph * cgs;
        float acc[V];
#pragma unroll
        for (int j = 0; j < V; ++j) acc[j] = 0.f;
        if (ph < phases) {
            const uint4* col = f + cg0 + cg;
            for (int px = ph; px < HW; px += 8 * phases) {
                uint4 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) v[u] = load_once(col + (long long)min(px + u * phases, HW - 1) * CG);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (px + u * phases < HW) {
#pragma unroll
                        for (int j = 0; j < V; ++j) acc[j] += E::at(v[u], j);
                    }
            }
            float* dst = part + (size_t(ph) * cgs + cg) * V;
#pragma unroll
            for (int j = 0; j < V; ++j) dst[j] = acc[j];
        }
        __syncthreads();
        const int rows = fold_phases<T>(part, phases, cgs * V);
        for (int c = threadIdx.x; c < cgs * V; c += T) {
            float s = 0.f;
            for (int q = 0; q < rows; ++q) s += part[size_t(q) * cgs * V + c];
            s *= inv_hw;
            sv_s[cg0 * V + c] = s;
            sv_out[(long long)b * C + cg0 * V + c] = s;
            if (!kOwnNorm) nrm = fmaf(s, s, nrm);
        }
        __syncthreads();
    }
    if (!kOwnNorm) nrm = block_sum(nrm, scratch);
    score_frame<kOwnNorm>(a, b, pf, sv_s, nrm, s_cur, s_acc);
}

// ---- NCHW without a stage: a warp per run of channels, straight from global memory -------------
//
// For small batches, where the streaming kernel's set-up (a ring of most of an SM's shared memory, one copy after
// another) costs more than the bytes, and for the shapes its copies cannot serve (frames that are no multiple of 16
// bytes, channels longer than a stage).  The reducers are the same; nothing is shared between warps.
constexpr int kDirectThreads = 128;

template <class R>
__global__ void __launch_bounds__(kDirectThreads) k_pool_direct(const NchwParams p) {
    const int warp = int(blockIdx.x) * (kDirectThreads / kWarp) + int(threadIdx.x >> 5), lane = threadIdx.x & 31;
    chain_wait();
    chain_release();
    const ClockScope stamps(p.clock);
    const int warps = int(gridDim.x) * (kDirectThreads / kWarp);
    const long long chunks = (long long)p.B * p.chunks_per_frame;
    for (long long g = warp; g < chunks; g += warps) {
        const int b = int(g / p.chunks_per_frame), ci = int(g - (long long)b * p.chunks_per_frame);
        if (p.skip && p.skip[b]) continue;
        const int c0 = ci * p.chunk_channels, nch = min(p.chunk_channels, p.C - c0);
        const long long lo = b * p.frame_bytes + (long long)c0 * p.ch_bytes, begin = lo & ~15ll;
        R::run(p.x + begin, int(lo - begin) / p.es, nch, lane, p.sv + (long long)b * p.C + c0, nullptr, p.inv_hw, p);
    }
}

// ---- NCHW, narrow channels: a thread each ------------------------------------------------------
//
// Channels of a handful of elements that begin anywhere in a 16-byte piece: a batch of them is a launch and a trip to
// memory, and a thread that adds its elements up in order has the least to set up (1206 frames of 160 3x3 16-bit channels
// 2.9 us, by words and lanes 3.7; 1484 frames of 2048 2x2 ones 15 and 24 us).
template <class E>
__global__ void k_pool_narrow(const NchwParams p) {
    chain_wait();
    chain_release();
    const ClockScope stamps(p.clock);
    const long long total = (long long)p.B * p.C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        if (p.skip && p.skip[i / p.C]) continue;
        float s = 0.f;
        for (int px = 0; px < p.hw; ++px) s += E::scalar(p.x, size_t(i) * p.hw + px);
        store_mean(p, s * p.inv_hw, 0, p.sv + i, nullptr);
    }
}

// ---- NHWC, any number of channels: one thread per (frame, channel) ---------------------------

template <class E>
__global__ void k_encode_nhwc_generic(const void* x, const uint8_t* skip, float* sv, int B, int C, int HW, float inv_hw, unsigned long long* clock) {
    chain_wait();
    chain_release();
    const ClockScope stamps(clock);
    const long long total = (long long)B * C;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int b = int(i / C), c = int(i - (long long)b * C);
        if (skip && skip[b]) continue;
        const size_t f0 = size_t(b) * C * HW;
        float s = 0.f;
        for (int px = 0; px < HW; ++px) s += E::scalar(x, f0 + size_t(px) * C + c);
        sv[i] = s * inv_hw;
    }
}

__global__ void k_row_norm2(const float* sv, const uint8_t* skip, int B, int D, float* out) {
    __shared__ float scratch[32];
    chain_wait();
    chain_release();
    const int b = blockIdx.x;
    if (skip && skip[b]) return;
    float s = 0.f;
    for (int d = threadIdx.x; d < D; d += blockDim.x) {
        const float v = sv[(size_t)b * D + d];
        s = fmaf(v, v, s);
    }
    s = block_sum(s, scratch);
    if (threadIdx.x == 0) out[b] = s;
}

constexpr size_t nchw_smem(int stages, bool listed) {
    return size_t(stages) * kStageCap + 2 * size_t(stages) * sizeof(uint64_t) + 128 +
           (listed ? (kListFrames + 33) * sizeof(int) : 0);
}

template <class R>
cudaError_t launch_nchw(const NchwParams& p, int grid, cudaStream_t st) {
    return launch_chained(k_encode_nchw<R>, grid, (p.consumers + 1) * kWarp, nchw_smem(p.stages, p.skip != nullptr), st, p);
}

template <class R>
cudaError_t opt_in() {
    return cudaFuncSetAttribute(k_encode_nchw<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(nchw_smem(kStages, true)));
}

template <class E>
cudaError_t launch_nhwc_generic(const EncodeArgs& a, cudaStream_t st) {
    const long long total = (long long)a.B * a.C;
    const int grid = int(std::min<long long>((total + 255) / 256, 148 * 16));
    return launch_chained(k_encode_nhwc_generic<E>, grid, 256, 0, st, a.x, a.skip, a.sv, a.B, a.C, a.H * a.W,
                          1.0f / float(a.H * a.W), a.clock);
}

int pow2_floor(int v) {
    int p = 1;
    while (p * 2 <= v) p *= 2;
    return p;
}



// Copies the producer keeps outstanding.  Four 25 KB copies per SM (15 MB over the chip) cover
// the bandwidth-delay product of HBM with margin; more only lengthens the queues that the
// centre loads of the dot warps wait in.
constexpr int kMaxInFlight = 4;

// Which reducer a shape is served by, and the chunking that goes with it.
enum Reducer {
    kNone, kUnitBf16x49, kUnitBf16x196, kUnitF16x49, kUnitF16x196, kUnitF32x49, kTeamF32, kTeamF16, kTeamBf16,
    kEdgeF32, kEdgeF16, kEdgeBf16, kLaneF32, kLaneF16, kLaneBf16
};

bool unit_reducer(Reducer r) { return r >= kUnitBf16x49 && r <= kUnitF32x49; }
bool any_width_reducer(Reducer r) { return r >= kEdgeF32; }  // channels that are no whole 16-byte vectors

Reducer of_type(Reducer f32, int dtype) { return Reducer(f32 + (dtype == SMTM_F32 ? 0 : dtype == SMTM_F16 ? 1 : 2)); }

// The reducer of channels that are no whole vectors.
Reducer any_width_of(int ch_bytes, int dtype) { return of_type(ch_bytes < 128 ? kLaneF32 : kEdgeF32, dtype); }

// Channels of H*W elements whose bytes together are a multiple of 16.
int aligned_channels(int ch_bytes) {
    int g = 1;
    while ((g * ch_bytes) % 16) g *= 2;
    return g;
}

// Lanes that share a channel: eight (128 bytes in a row), fewer when it has fewer whole vectors, one below 128 bytes
// where it has edges.
int team_lanes(int ch_bytes) { return ch_bytes % 16 == 0 ? std::min(8, pow2_floor(ch_bytes / 16)) : ch_bytes < 128 ? 1 : 8; }

// The longest channel a stage holds, in bytes: one that is no whole vectors may begin and end inside a 16-byte piece.
int stage_room(int ch_bytes) { return ch_bytes % 16 == 0 ? kStageCap : kStageCap - 32; }

// Channels a chunk of at most `cap` bytes holds, in multiples of `gran` where it holds one.
int channels_in(int cap, int ch_bytes, int gran) {
    const int cc = cap / ch_bytes;
    return cc > gran ? cc - cc % gran : cc;
}

constexpr long long kLongFrame = 2ll << 20;  // bytes of a frame that pooling and scoring apart spread over the chip

// The plan of the kernels that take a frame's chunks one by one: every chunk begins on a 16-byte boundary.
Reducer plan_nchw(const EncodeArgs& a, NchwParams* p) {
    const int HW = a.H * a.W;
    const int es = a.dtype == SMTM_F32 ? 4 : 2;
    *p = NchwParams{};
    p->x = static_cast<const uint8_t*>(a.x);
    p->skip = a.skip;
    p->sv = a.sv;
    p->sv_hi = static_cast<__nv_bfloat16*>(a.sv_hi);
    p->sv_lo = static_cast<__nv_bfloat16*>(a.sv_lo);
    p->status = a.status;
    p->clock = a.clock;
    p->B = a.B;
    p->C = a.C;
    p->hw = HW;
    p->es = es;
    p->ch_bytes = HW * es;
    p->frame_bytes = (long long)a.C * p->ch_bytes;
    p->inv_hw = 1.0f / float(HW);
    p->max_in_flight = a.ring_in_flight > 0 ? std::min(a.ring_in_flight, kMaxInFlight) : kMaxInFlight;
    p->stages = (a.ring_stages >= 2 && a.ring_stages <= kStages) ? a.ring_stages : kStages;
    if (p->max_in_flight > p->stages - 1) p->max_in_flight = p->stages - 1;
    p->consumers = (a.ring_consumers >= 1 && a.ring_consumers <= kConsumers) ? a.ring_consumers : kConsumers;
    p->consumers = std::min(p->consumers, p->stages);
    // A stage passes from warp to warp unless their number divides the ring's depth.  The warp that is next to use a stage
    // must not look at its barrier while the copy before is still under way (the parity it waits for would be that of
    // the copy before that, which is complete): it gets there after a chunk issued stages - consumers later, so that
    // copy has to have been issued after the one before had landed.
    if (p->stages % p->consumers) p->max_in_flight = std::min(p->max_in_flight, p->stages - p->consumers);
    p->team = team_lanes(p->ch_bytes);
    if (p->ch_bytes > stage_room(p->ch_bytes)) return kNone;
    // unit-per-lane shapes (compile-time H*W)
    int G = 0;
    if ((HW == 49 || HW == 196) && es == 2) G = HW == 49 ? 8 : 2;
    if (HW == 49 && es == 4) G = 4;
    if (G && a.C % G == 0) {
        p->chunk_channels = 32 * G;
        p->chunks_per_frame = (a.C + p->chunk_channels - 1) / p->chunk_channels;
        if (es == 4) return kUnitF32x49;
        if (a.dtype == SMTM_BF16) return HW == 49 ? kUnitBf16x49 : kUnitBf16x196;
        return HW == 49 ? kUnitF16x49 : kUnitF16x196;
    }
    // team-per-channel: channel bytes a multiple of 16
    if (p->ch_bytes % 16 == 0) {
        p->chunk_channels = std::min(channels_in(kStageCap, p->ch_bytes, 32 / p->team), a.C);
        p->chunks_per_frame = (a.C + p->chunk_channels - 1) / p->chunk_channels;
        return of_type(kTeamF32, a.dtype);
    }
    // any other width: runs of channels that are whole 16-byte pieces, which a stage has to hold
    const int run = aligned_channels(p->ch_bytes);
    // (channels below one 16-byte piece are left to the plain route: a 2x2 map of 512 channels is 4 KB, and the fused
    // kernel takes 8 us for 128 such frames, pooling and scoring apart 6)
    if (a.C % run || run * p->ch_bytes > kStageCap || p->ch_bytes < 16) return kNone;
    p->chunk_channels = std::min(channels_in(kStageCap, p->ch_bytes, std::max(run, 32 / p->team)), a.C);
    p->chunk_channels -= p->chunk_channels % run;
    p->chunks_per_frame = (a.C + p->chunk_channels - 1) / p->chunk_channels;
    return any_width_of(p->ch_bytes, a.dtype);
}

// Where the ring does not serve.  Batches of short channels are pooled straight from global memory below 16 MB: 376 frames
// of 256 5x5 16-bit channels (5 MB) take 3.2 us so and 5.8 through the ring, 134 frames of 160 9x9 ones (3 MB) 4.1 and 8.3,
// 256 frames of 256 8x8 ones (8 MB) 4.3 and 5.4; from 16 MB on the ring is the faster one.  Channels of half a kilobyte
// and more, and a few hundred of a quarter, keep too few warps busy that way; shapes with a reducer of their own take
// 0.4 us more.  Narrow channels of odd widths have a thread each (k_pool_narrow) up to 32 MB.
constexpr long long kDirectBatch = 16ll << 20, kNarrowBatch = 32ll << 20;  // bytes
constexpr int kNarrowChannel = 64, kShortChannel = 256, kDirectChannel = 512, kDirectLeast = 1024;

bool pooled_by_threads(const NchwParams& p, long long batch_bytes) {
    return p.ch_bytes % 16 != 0 && p.ch_bytes < kNarrowChannel && batch_bytes < kNarrowBatch;
}
bool pooled_directly(const NchwParams& p, long long channels) {
    return channels * p.ch_bytes < kDirectBatch &&
           (p.ch_bytes < kShortChannel || (p.ch_bytes <= kDirectChannel && channels >= kDirectLeast));
}

// The plan of k_encode_nchw, or kNone where the kernels without a ring serve.  Chunks may begin anywhere in a 16-byte piece (the copy is widened to whole pieces, which
// lie inside the frame when its bytes are a multiple of 16), so every channel that fits a stage is served.  Chunks are cut so that every CTA gets the same number of nearly equal ones.
Reducer plan_ring(const EncodeArgs& a, int grid, NchwParams* p) {
    Reducer r = plan_nchw(a, p);
    if (p->ch_bytes > stage_room(p->ch_bytes)) return kNone;
    if (!unit_reducer(r) && (pooled_by_threads(*p, a.B * p->frame_bytes) || pooled_directly(*p, (long long)a.B * a.C))) return kNone;
    if (r == kNone) r = any_width_of(p->ch_bytes, a.dtype);
    if (p->frame_bytes % 16) return kNone;  // (with and without flags alike: a channel's sum does not depend on them)
    const bool flat = !a.skip && (long long)a.B * a.C < (1ll << 30);
    if (flat) {
        p->frame_bytes *= a.B;
        p->C *= a.B;
        p->B = 1;
    }
    int gran = 1;  // channels a warp takes in one go
    if (unit_reducer(r)) gran = p->chunk_channels / 32;
    else gran = 32 / p->team;
    int most = unit_reducer(r) ? p->chunk_channels : channels_in(stage_room(p->ch_bytes), p->ch_bytes, gran);
    most = std::min(most, p->C);
    const int runs = flat ? grid : 1;  // with flags: whole frames, dealt out chunk by chunk
    const int rounds = (p->C + runs * most - 1) / (runs * most);
    const int even = (p->C + runs * rounds - 1) / (runs * rounds);
    p->chunk_channels = std::max(1, std::min(most, (even + gran - 1) / gran * gran));
    p->chunks_per_frame = (p->C + p->chunk_channels - 1) / p->chunk_channels;
    return r;
}

#define SMTM_FOR_TEAM_REDUCER(r, CALL)                              \
    switch (r) {                                                    \
        case kTeamF32: CALL(TeamVectors<F32, false>); break;        \
        case kTeamF16: CALL(TeamVectors<F16, false>); break;        \
        case kTeamBf16: CALL(TeamVectors<BF16, false>); break;      \
        case kEdgeF32: CALL(TeamVectors<F32, true>); break;         \
        case kEdgeF16: CALL(TeamVectors<F16, true>); break;         \
        case kEdgeBf16: CALL(TeamVectors<BF16, true>); break;       \
        case kLaneF32: CALL(LanePerChannel<F32>); break;            \
        case kLaneF16: CALL(LanePerChannel<F16>); break;            \
        case kLaneBf16: CALL(LanePerChannel<BF16>); break;          \
        default: break;                                             \
    }

#define SMTM_FOR_REDUCER(r, CALL)                                   \
    switch (r) {                                                    \
        case kUnitBf16x49: CALL(UnitPerLane<BF16, 49>); break;      \
        case kUnitBf16x196: CALL(UnitPerLane<BF16, 196>); break;    \
        case kUnitF16x49: CALL(UnitPerLane<F16, 49>); break;        \
        case kUnitF16x196: CALL(UnitPerLane<F16, 196>); break;      \
        case kUnitF32x49: CALL(UnitPerLane<F32, 49>); break;        \
        default: SMTM_FOR_TEAM_REDUCER(r, CALL)                     \
    }

#define SMTM_FOR_TYPE(t, CALL)               \
    switch (t) {                             \
        case SMTM_F32: CALL(F32); break;     \
        case SMTM_F16: CALL(F16); break;     \
        default: CALL(BF16); break;          \
    }

// Small new frames in a crowd (see above): pooled, then scored.
bool scored_apart(const EncodeArgs& a, const LookupArgs& l, int sm_count) {
    const long long channel = (long long)a.H * a.W * (a.dtype == SMTM_F32 ? 4 : 2);
    if (!l.fresh || a.C * channel >= kCrowdFrame) return false;
    const bool narrow = channel % 16 != 0 && channel < kNarrowChannel;
    return (narrow && l.k_max <= kCrowdNarrowSlots && a.B >= 2 * sm_count) || (l.k_max <= kCrowdSlots && a.B > 3 * sm_count);
}

// The plan of k_lookup_frame: a slice per CTA that is whole 16-byte pieces of the map and of the vector.
Reducer plan_frame(const EncodeArgs& a, const LookupArgs& l, int sm_count, FrameParams* f) {
    if (a.layout != SMTM_NCHW || l.k_max > kFusedMaxK || (a.C & 3)) return kNone;
    const int es = a.dtype == SMTM_F32 ? 4 : 2;
    if ((long long)a.H * a.W * es > kFrameStageCap) return kNone;
    (void)plan_nchw(a, &f->e);
    NchwParams& p = f->e;
    const int run = aligned_channels(p.ch_bytes);
    if (a.C % run) return kNone;
    const int unit = std::max(4, run);
    const auto slice_of = [&](int parts) { return ((a.C + parts - 1) / parts + unit - 1) / unit * unit; };
    const bool many = l.k_max >= kFrameManySlots;
    const int wanted = many ? kFrameStageWantedMany : kFrameStageWanted, least = many ? kFrameStageLeastMany : kFrameStageLeast;
    const int frames = l.fresh ? a.B : (a.B + 1) / 2;  // (after a first lookup half of them are taken to be still in)
    int best = 0;
    for (int P = 1; P <= kMaxCluster; P *= 2) {
        const int slice = slice_of(P);
        const long long bytes = (long long)slice * p.ch_bytes;
        if (P > 1 && slice * (P - 1) >= a.C) break;  // a CTA without channels
        if (slice > kFrameSlice || bytes > kFrameStageCap) continue;
        best = P;
        if (bytes <= least || (bytes <= wanted && 2LL * frames * P > sm_count)) break;
    }
    if (best == 0 || (long long)a.B * a.C * p.ch_bytes > kFrameBatchMost) return kNone;
    if (best > 1 && (long long)a.B * best > (many ? 4LL : 2LL) * kFrameResident * sm_count) return kNone;
    f->parts = best;
    f->slice = slice_of(best);
    f->gran = run;
    return p.ch_bytes % 16 == 0 ? of_type(kTeamF32, a.dtype) : any_width_of(p.ch_bytes, a.dtype);
}

// How the clusters of the NHWC kernels divide a frame: pixels between the CTAs, then columns.  Wider rows than a CTA of a
// cluster (or of a lookup) has shared memory for are pooled by a CTA per frame, which keeps the sums of a sweep only.
constexpr int kNhwcWide = 8192;
bool plan_frame_nhwc(const EncodeArgs& a, const LookupArgs* l, int sm_count, FrameNhwcParams* f) {
    const int V = a.dtype == SMTM_F32 ? 4 : 8, es = a.dtype == SMTM_F32 ? 4 : 2;
    if (a.layout != SMTM_NHWC || a.C % V) return false;
    const int HW = a.H * a.W;
    const long long frame = (long long)HW * a.C * es;
    int P = 1;
    const int frames = l && !l->fresh ? (a.B + 1) / 2 : a.B;  // (after a first lookup half of them are taken to be still in)
    const auto enlarge = [&](long long ctas, int most, long long pixels) {  // pixels: a CTA's that are not divided again
        while (P < most && 2 * P <= HW && 2LL * frames * P <= ctas && HW > pixels * P) P *= 2;
    };
    if (l) {
        const int phases = kThreadsNhwcLookup / std::min(kThreadsNhwcLookup, a.C / V);
        if (2 * frames <= sm_count && frame >= kNhwcShared)
            enlarge((frame >= kNhwcLong ? 4LL : 2LL) * sm_count, kMaxCluster, kNhwcPixels * phases);
        if (l->k_max >= kNhwcManySlots) enlarge(sm_count, frame >= kNhwcManyLeast ? kMaxCluster : 4, 0);
        else if (l->k_max >= kNhwcSomeSlots && 8 * frames <= sm_count && frame >= kNhwcSomeLeast) enlarge(sm_count, 4, 0);
    } else if (a.C <= kNhwcWide) {
        const int phases = kFrameThreads / std::min(kFrameThreads, a.C / V);
        while (P < kMaxCluster && 2 * P <= HW &&
               ((HW > kNhwcPoolLoads * phases * P && 2LL * a.B * P <= 3LL * sm_count) ||
                ((long long)a.B * P < 4LL * sm_count && frame / (2 * P) >= kNhwcPartLong)))
            P *= 2;
    }
    f->x = static_cast<const uint8_t*>(a.x);
    f->sv = a.sv;
    f->C = a.C;
    f->HW = HW;
    f->inv_hw = 1.0f / float(HW);
    f->parts = P;
    f->pixels = (HW + P - 1) / P;
    f->slice = ((a.C + P - 1) / P + 3) / 4 * 4;
    return true;
}

// Shared memory of the column sums: the slice's sums (a row per CTA of a cluster) and the phases' parts.
size_t nhwc_smem_bytes(const EncodeArgs& a, const FrameNhwcParams& f) {
    const int V = a.dtype == SMTM_F32 ? 4 : 8;
    const int cgs = std::min(a.C / V, kFrameThreads);
    return ((f.parts > 1 ? size_t(f.parts) * f.slice : 0) + size_t(kFrameThreads / cgs) * cgs * V) * sizeof(float);
}

template <class R>
cudaError_t opt_in_fused() {
    return cudaFuncSetAttribute(k_lookup_nchw<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmemLimit));
}

// Clusters of `parts` CTAs of the fused kernel that the device runs at once (each CTA fills an SM).
template <class R>
cudaError_t max_clusters(int parts, size_t smem, int* out) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(parts));
    cfg.blockDim = dim3(kThreadsFused);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(parts);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(out, k_lookup_nchw<R>, &cfg);
}

}  // namespace

template <class R>
cudaError_t carveout_pipelined() {
    cudaError_t e = prefer_max_smem_carveout(k_encode_nchw<R>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_pool_sparse<R>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_lookup_sparse<R, false>);
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_lookup_sparse<R, true>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_lookup_sparse<R, false>);
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_lookup_sparse<R, true>);
    return e;
}

cudaError_t encode_setup() {
    cudaError_t e = cudaSuccess;
#define SMTM_OPT_IN(E)                                                             \
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_lookup_frame_nhwc<E>);      \
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_lookup_frame_nhwc<E>);    \
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_lookup_nhwc<E>);            \
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_encode_nhwc<E, 2>);         \
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_encode_nhwc<E, 4>);         \
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_encode_nhwc<E, 8>);
    SMTM_OPT_IN(F32) SMTM_OPT_IN(F16) SMTM_OPT_IN(BF16)
#undef SMTM_OPT_IN
#define SMTM_OPT_IN(...)                                                             \
    if (e == cudaSuccess) e = allow_max_dynamic_smem(k_lookup_frame<__VA_ARGS__>);   \
    if (e == cudaSuccess) e = prefer_max_smem_carveout(k_lookup_frame<__VA_ARGS__>);
    for (int r = kTeamF32; r <= kLaneBf16; ++r) SMTM_FOR_TEAM_REDUCER(r, SMTM_OPT_IN)
#undef SMTM_OPT_IN
#define SMTM_OPT_IN(...)                                        \
    if (e == cudaSuccess) e = opt_in<__VA_ARGS__>();            \
    if (e == cudaSuccess) e = carveout_pipelined<__VA_ARGS__>();  \
    if (e == cudaSuccess) e = opt_in_fused<__VA_ARGS__>();
    for (int r = kUnitBf16x49; r <= kLaneBf16; ++r) SMTM_FOR_REDUCER(r, SMTM_OPT_IN)
#undef SMTM_OPT_IN
    return e;
}

cudaError_t launch_encode(const EncodeArgs& a, int sm_count, cudaStream_t st, int64_t* launches, bool* wrote_split) {
    if (wrote_split) *wrote_split = false;
    if (a.B <= 0) return cudaSuccess;
    ++*launches;
    if (a.layout == SMTM_NHWC) {
        FrameNhwcParams f{};
        if (plan_frame_nhwc(a, nullptr, sm_count, &f)) {
            cudaError_t e = cudaSuccess;
            if (wrote_split) *wrote_split = a.sv_hi != nullptr;
            const int phases = kFrameThreads / std::min(kFrameThreads, a.C / (a.dtype == SMTM_F32 ? 4 : 8));
            const int loads = f.pixels <= 2 * phases ? 2 : f.pixels <= (a.B > 4 * sm_count ? 8 : 4) * phases ? 4 : 8;
#define SMTM_LAUNCH(E) \
    e = launch_chained_cluster(loads == 2 ? k_encode_nhwc<E, 2> : loads == 4 ? k_encode_nhwc<E, 4> : k_encode_nhwc<E, 8>, a.B * f.parts, kFrameThreads, nhwc_smem_bytes(a, f), f.parts, st, f.x, a.skip, \
                               a.sv, a.C, f.HW, f.inv_hw, f.parts, f.pixels, f.slice, static_cast<__nv_bfloat16*>(a.sv_hi), \
                               static_cast<__nv_bfloat16*>(a.sv_lo), a.status, a.clock)
            SMTM_FOR_TYPE(a.dtype, SMTM_LAUNCH)
#undef SMTM_LAUNCH
            return e;
        }
    } else {
        NchwParams p;
        const Reducer r = plan_ring(a, sm_count, &p);
        if (r != kNone) {
            cudaError_t e = cudaSuccess;
            if (wrote_split) *wrote_split = p.sv_hi != nullptr;
#define SMTM_LAUNCH(...) e = launch_nchw<__VA_ARGS__>(p, sm_count, st)
            SMTM_FOR_REDUCER(r, SMTM_LAUNCH)
#undef SMTM_LAUNCH
            return e;
        }
        if (pooled_by_threads(p, a.B * p.frame_bytes)) {
            const int ctas = int(std::min<long long>(((long long)a.B * a.C + 255) / 256, 16LL * sm_count));
            cudaError_t e = cudaSuccess;
            if (wrote_split) *wrote_split = p.sv_hi != nullptr;
#define SMTM_LAUNCH(E) e = launch_chained(k_pool_narrow<E>, ctas, 256, 0, st, p)
            SMTM_FOR_TYPE(a.dtype, SMTM_LAUNCH)
#undef SMTM_LAUNCH
            return e;
        }
        p.chunk_channels = std::min(a.C, p.ch_bytes < 1024 && p.team > 1 ? 64 / p.team : 32 / p.team);
        p.chunks_per_frame = (a.C + p.chunk_channels - 1) / p.chunk_channels;
        const long long warps = (long long)a.B * p.chunks_per_frame;
        const int ctas = int(std::min<long long>((warps + 3) / 4, 16LL * sm_count));
        if (wrote_split) *wrote_split = p.sv_hi != nullptr;
        const Reducer d = p.ch_bytes % 16 == 0 ? of_type(kTeamF32, a.dtype) : any_width_of(p.ch_bytes, a.dtype);
        cudaError_t e = cudaErrorInvalidValue;
#define SMTM_LAUNCH(...) e = launch_chained(k_pool_direct<__VA_ARGS__>, ctas, kDirectThreads, 0, st, p)
        SMTM_FOR_TEAM_REDUCER(d, SMTM_LAUNCH)
#undef SMTM_LAUNCH
        return e;
    }
    if (a.dtype == SMTM_F32) return launch_nhwc_generic<F32>(a, st);
    if (a.dtype == SMTM_F16) return launch_nhwc_generic<F16>(a, st);
    return launch_nhwc_generic<BF16>(a, st);
}

// Channels of a chunk that must stay in one warp's share when the warps of a CTA divide it.
static int share_granularity(Reducer r, const NchwParams& p) {
    if (unit_reducer(r)) return p.chunk_channels / 32;
    return std::max(any_width_reducer(r) ? aligned_channels(p.ch_bytes) : 1, 32 / std::max(1, p.team));
}

bool launch_encode_nhwc_vector_supported(const EncodeArgs& a) {
    if (a.B <= 0) return false;
    FrameNhwcParams f{};
    return plan_frame_nhwc(a, nullptr, 1, &f);
}

bool launch_encode_fills_sms(const EncodeArgs& a, int sm_count) {
    if (a.layout == SMTM_NHWC) {
        FrameNhwcParams f{};
        return plan_frame_nhwc(a, nullptr, sm_count, &f);
    }
    NchwParams p;
    return plan_ring(a, sm_count, &p) != kNone;
}

bool launch_encode_split_supported(const EncodeArgs& a) { return a.layout == SMTM_NCHW && a.B > 0; }

bool launch_pool_sparse_supported(const EncodeArgs& a) {
    if (a.layout != SMTM_NCHW || a.B <= 0) return false;
    NchwParams p;
    const Reducer r = plan_nchw(a, &p);
    return r != kNone && (any_width_reducer(r) ? aligned_channels(p.ch_bytes) : 1) * p.ch_bytes <= kLightStageCap;
}

cudaError_t launch_pool_sparse(const EncodeArgs& a, int sm_count, cudaStream_t st, int64_t* launches) {
    LightParams f{};
    if (!launch_pool_sparse_supported(a)) return cudaErrorInvalidValue;
    const Reducer r = plan_nchw(a, &f.e);
    // chunks of at most kLightStageCap bytes: half the units of a unit-per-lane chunk, or as many whole channels as fit
    f.gran = share_granularity(r, f.e);
    if (unit_reducer(r)) {
        f.e.chunk_channels /= 2;
    } else {
        f.e.chunk_channels = std::min(channels_in(kLightStageCap, f.e.ch_bytes, f.gran), a.C);
        if (any_width_reducer(r)) f.e.chunk_channels -= f.e.chunk_channels % aligned_channels(f.e.ch_bytes);
    }
    f.e.chunks_per_frame = (a.C + f.e.chunk_channels - 1) / f.e.chunk_channels;
    // about four CTAs to an SM; enough groups that no CTA is given more frames than it can list
    const int cpf = f.e.chunks_per_frame;
    int groups = std::max(1, std::min(a.B, 8 * sm_count / cpf));
    groups = std::max(groups, (a.B + kLightFrames - 1) / kLightFrames);
    f.groups = groups;
    cudaError_t e = cudaSuccess;
    ++*launches;
#define SMTM_LAUNCH(...) e = launch_chained(k_pool_sparse<__VA_ARGS__>, cpf * groups, kLightThreads, 0, st, f)
    SMTM_FOR_REDUCER(r, SMTM_LAUNCH)
#undef SMTM_LAUNCH
    return e;
}

// The layout of a sparse lookup, or kNone when the shape is not served: chunks as the streaming kernel cuts
// them, at most 8 to a frame, slices that are whole 16-byte pieces and fit the scorers' registers.
Reducer plan_sparse(const EncodeArgs& e, const LookupArgs& a, SparseParams* f) {
    if (e.layout != SMTM_NCHW || e.B <= 0 || a.k_max > kFusedMaxK || (e.C & 3)) return kNone;
    const Reducer r = plan_nchw(e, &f->e);
    if (r == kNone) return kNone;
    if (f->e.chunks_per_frame > kMaxCluster || (f->e.chunk_channels & 3) || f->e.chunk_channels > kSparseSlice) return kNone;
    f->staged = f->e.chunk_channels;
    f->gran = share_granularity(r, f->e);
    return r;
}

bool launch_lookup_sparse_supported(const EncodeArgs& e, const LookupArgs& a) {
    SparseParams f{};
    return plan_sparse(e, a, &f) != kNone;
}

cudaError_t launch_lookup_sparse(const EncodeArgs& e, const LookupArgs& a, int sm_count, cudaStream_t st, int64_t* launches,
                                 const cudaEvent_t* timing) {
    SparseParams f{};
    const Reducer r = plan_sparse(e, a, &f);
    if (r == kNone) return cudaErrorInvalidValue;
    f.a = a;
    const int P = f.e.chunks_per_frame;
    // three or four CTAs to an SM (they sit beside a streaming kernel); enough clusters that none is given more
    // frames than it can list
    const bool halves = e.B > 4 * (3 * sm_count / P);
    if (halves) {
        const int unit = unit_reducer(r) ? f.e.chunk_channels / 32 : any_width_reducer(r) ? aligned_channels(f.e.ch_bytes) : 1;
        f.staged = std::min(f.staged, ((f.staged + 1) / 2 + unit - 1) / unit * unit);
        if (f.staged < 4 * f.gran) f.gran = unit;  // (few channels: a warp takes fewer than it could)
    }
    int groups = std::max(1, std::min(e.B, (halves ? 4 : 3) * sm_count / P));
    groups = std::max(groups, (e.B + kSparseFrames - 1) / kSparseFrames);
    f.a.pending = (long long)e.B * P > (long long)kSparseOwn * sm_count;
    f.groups = groups = f.a.pending ? groups : e.B;
    const size_t smem = sparse_smem(f.e.chunk_channels, size_t(f.staged) * f.e.ch_bytes);
    cudaError_t err = cudaSuccess;
    ++*launches;
    if (timing) record_timing(timing[0], st);
    // (in stream order, without the early start: the clusters would wait on the SMs for the scoring kernel before
    // them and keep the next step's pooling CTAs out meanwhile)
#define SMTM_LAUNCH(...) err = launch_ordered_cluster(halves ? k_lookup_sparse<__VA_ARGS__, true> : k_lookup_sparse<__VA_ARGS__, false>, P * groups, kLightThreads, smem, P, st, f)
    SMTM_FOR_REDUCER(r, SMTM_LAUNCH)
#undef SMTM_LAUNCH
    if (timing) record_timing(timing[1], st);
    return err == cudaSuccess && f.a.pending ? launch_settle_exits(f.a, st, launches) : err;
}

cudaError_t launch_lookup_fused(const EncodeArgs& e, const LookupArgs& a, int sm_count, FusedCaps* caps, cudaStream_t st,
                                int64_t* launches, LookupServed* served, const cudaEvent_t* timing) {
    *served = kNotServed;
    if (e.B <= 0 || a.k_max > kFusedMaxK) return cudaSuccess;
    if (e.layout == SMTM_NHWC) {
        FrameNhwcParams f{};
        if (e.C > kNhwcWide || !plan_frame_nhwc(e, &a, sm_count, &f)) return cudaSuccess;
        f.a = a;
        cudaError_t err = cudaSuccess;
        if (timing) record_timing(timing[0], st);
        if (f.parts > 1) {
            const size_t smem = nhwc_smem_bytes(e, f) + (size_t(f.slice) + size_t(f.parts) * kRxRow) * sizeof(float);
#define SMTM_LAUNCH(E) err = launch_chained_cluster(k_lookup_frame_nhwc<E>, e.B * f.parts, kFrameThreads, smem, f.parts, st, f)
            SMTM_FOR_TYPE(e.dtype, SMTM_LAUNCH)
#undef SMTM_LAUNCH
        } else {  // frames enough for the chip: a CTA each
            const int V = e.dtype == SMTM_F32 ? 4 : 8, cgs = std::min(e.C / V, kThreadsNhwcLookup);
            const size_t smem = (size_t(e.C) + 3 * size_t(a.k_max) + size_t(kThreadsNhwcLookup / cgs) * cgs * V) * sizeof(float);
#define SMTM_LAUNCH(E) \
    err = launch_chained(k_lookup_nhwc<E>, e.B, kThreadsNhwcLookup, smem, st, f.x, e.C, f.HW, f.inv_hw, e.sv, a)
            SMTM_FOR_TYPE(e.dtype, SMTM_LAUNCH)
#undef SMTM_LAUNCH
        }
        if (timing) record_timing(timing[1], st);
        ++*launches;
        *served = kServedFused;
        return err;
    }
    if (scored_apart(e, a, sm_count)) return cudaSuccess;
    {
        FrameParams f{};
        const Reducer r = plan_frame(e, a, sm_count, &f);
        if (r != kNone) {
            f.a = a;
            const size_t smem = ((size_t(f.slice) * f.e.ch_bytes + 15) & ~size_t(15)) +
                                (size_t(f.slice) + size_t(f.parts) * kRxRow) * sizeof(float);
            cudaError_t err = cudaErrorInvalidValue;
            if (timing) record_timing(timing[0], st);
#define SMTM_LAUNCH(...) err = launch_chained_cluster(k_lookup_frame<__VA_ARGS__>, e.B * f.parts, kFrameThreads, smem, f.parts, st, f)
            SMTM_FOR_TEAM_REDUCER(r, SMTM_LAUNCH)
#undef SMTM_LAUNCH
            if (timing) record_timing(timing[1], st);
            ++*launches;
            NchwParams streamed;
            *served = plan_nchw(e, &streamed) != kNone ? kServedFused : kServedPlain;
            return err;
        }
    }
    FusedParams f{};
    const Reducer r = plan_nchw(e, &f.e);
    if (r == kNone) return cudaSuccess;
    const int cpf = f.e.chunks_per_frame;
    if (e.C & 3) return cudaSuccess;
    // Parts per frame = CTAs per cluster.  A part must fit the scorers' registers (slice <= kMaxSlice
    // channels, a multiple of 4) and the CTA's shared memory; among 1, 2, 4, 8 take the smallest
    // that keeps the SMs 95 % busy over the rounds of frames (else the busiest).
    static_assert(kLaneBf16 < 16 && kMaxCluster < 9, "FusedCaps holds an entry per (reducer, cluster size)");
    int best_P = 0, best_grid = 0;
    double best_eff = -1.0;
    for (int P = 1; P <= kMaxCluster; P *= 2) {
        if (cpf % P || (cpf / P) * f.e.chunk_channels > kMaxSlice) continue;
        if (((cpf / P) * f.e.chunk_channels) & 3) continue;  // the scorers read a part's slice as 16-byte vectors
        const size_t smem = fused_smem((cpf / P) * f.e.chunk_channels, P);
        if (smem > kSmemLimit) continue;
        int clusters = sm_count;
        if (P > 1) {
            int& cap = caps->clusters[r][P];  // clusters the device runs at once, 0 = not asked yet
            if (cap == 0) {
                cudaError_t err = cudaSuccess;
#define SMTM_ASK(...) err = max_clusters<__VA_ARGS__>(P, smem, &cap)
                SMTM_FOR_REDUCER(r, SMTM_ASK)
#undef SMTM_ASK
                if (err != cudaSuccess) {
                    (void)cudaGetLastError();
                    cap = -1;
                }
            }
            if (cap <= 0) continue;
            clusters = std::min(cap, sm_count / P);
        }
        if (clusters < 1 || ((long long)e.B + clusters - 1) / clusters > kMaxUnits) continue;
        const double rounds = double(e.B) / clusters;
        const double eff = rounds / std::ceil(rounds) * double(clusters * P) / sm_count;
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best_P = P;
            best_grid = clusters * P;
        }
        if (eff >= 0.95) break;
    }
    if (best_P == 0) return cudaSuccess;
    // At most eight CTAs share a frame, so that a few frames of megabytes, or the few of a batch that are still in, leave most
    // of the chip idle; pooled apart, a frame is dealt out to every SM, chunk by chunk: 2 frames of 2048 48x48 16-bit
    // channels 31 us and 14, 6 of 2048 32x32 fp32 ones 30 and 18, 144 of 1024 26x26 ones, few of them still in, 54 and 13.
    // Below 2 MB CTAs on 70 % of the SMs speak for one kernel, on a quarter of them where 32 slots and more are to be scored
    // (13 frames of 256 48x48 channels, 32 slots, 11 us and 31).  Frames that the kernel of small frames refuses for their
    // number alone are many.
    const long long frame = f.e.frame_bytes;
    const int share = a.k_max < kFrameManySlots ? 70 : 25;
    if (frame >= kLongFrame || (frame > (long long)kMaxCluster * kFrameStageCap && 100LL * e.B * best_P < (long long)share * sm_count))
        return cudaSuccess;
    const int P = best_P;
    f.a = a;
    f.a.pending = !a.fresh && a.B > best_grid / P;
    f.parts = P;
    f.chunks_per_unit = cpf / P;
    f.slice_cap = f.chunks_per_unit * f.e.chunk_channels;
    const size_t smem = fused_smem(f.slice_cap, P);
    cudaError_t err = cudaSuccess;
    if (timing) record_timing(timing[0], st);
#define SMTM_LAUNCH(...) err = launch_chained_cluster(k_lookup_nchw<__VA_ARGS__>, best_grid, kThreadsFused, smem, P, st, f)
    SMTM_FOR_REDUCER(r, SMTM_LAUNCH)
#undef SMTM_LAUNCH
    if (timing) record_timing(timing[1], st);
    ++*launches;
    *served = kServedFused;
    return err == cudaSuccess && f.a.pending ? launch_settle_exits(f.a, st, launches) : err;
}

cudaError_t launch_row_norm2(const float* sv, const uint8_t* skip, int B, int D, float* out, cudaStream_t st,
                             int64_t* launches) {
    if (B <= 0) return cudaSuccess;
    ++*launches;
    return launch_chained(k_row_norm2, B, 256, 0, st, sv, skip, B, D, out);
}

}  // namespace smtm
