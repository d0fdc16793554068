// Cache maintenance kernels: state initialisation, static-prefix write (Sec. 3.1) and the in-place
// sliding-ring append with circular pointer arithmetic (Sec. 3.4, App. B.2). Byte movers: rows are
// opaque 16-byte units, so one kernel serves bf16 and fp32 storage.
#include "reflex_internal.cuh"
#include "sm100_ptx.cuh"

namespace reflex {

// The kernels that write cache regions or state take part in programmatic dependent launch like the rest of the library: they
// may be scheduled while the kernel ahead of them still runs, wait for all of it before they touch memory, and only then let
// the next one be scheduled. (The order matters: an expert step's attention reads cached rows ahead of its own wait, which is
// sound because its predecessor could only pass its wait once every earlier kernel was complete.) A prefix of 8 streams staged
// and committed: the second launch costs 1.3 us behind the first instead of 5.3.
__device__ __forceinline__ void wait_then_release()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
static cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    count_launch();
    return e;
}

__global__ void state_init_kernel(StreamState *state, int64_t *total, uint32_t *status, const int32_t *head0, int B, int N)
{
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b == 0) *status = 0u;
    if (b >= B) return;
    StreamState s;
    s.static_len = -1;
    int h = head0 ? head0[b] : 0;
    s.head = ((h % N) + N) % N;
    s.count = 0;
    s.ticket = 0;
    s.bank = 0;
    s.staged_len = -1;
    state[b] = s;
    total[b] = 0;
}

cudaError_t launch_state_init(StreamState *state, int64_t *total, uint32_t *status, const int32_t *head0, int B, int N,
                              cudaStream_t st)
{
    state_init_kernel<<<(B + 127) / 128, 128, 0, st>>>(state, total, status, head0, B, N);
    count_launch();
    return cudaGetLastError();
}

// One (stream, layer) prefix is a single contiguous run of S*row_bytes bytes on both sides.
// grid = (chunks, L, n); 16-byte units. Memory bound: a thread asks for all its units of K and V before it stores the first,
// and no thread comes back for more (the compiler's own loop kept two pairs in flight and blocks of eight rounds left a ragged
// last wave). 8 streams x 18 layers x 816 rows (236 MB moved): 40.5 -> 37.4 us, 6.3 TB/s; 12 x 18 x 1000 70.6 -> 67.1. With 2
// units of each 39.3, with 4 37.1 (but 6.95 against 6.5 where everything stays in L2, 8 x 10 x 300; 6.2 before), with 8 37.2; through shared memory with
// bulk copies 38.7 to 41.0 and 73.3 to 74.6.
constexpr int kCopyUnits = 6;

// Uneven prefixes: blockIdx.x counts the blocks of all streams, first[i] being stream i's first. One grid over the longest prefix launches
// blocks without work for every other stream (32 streams, one of 816 rows and 31 of one: 16.6 us with blocks of eight rounds, 23.7 with one round, 6.3 so).
struct CopyStarts {
    int n;                            // streams; 0: even prefixes, blockIdx.z is the stream
    int first[kStreamsPerLaunch];
};

__global__ void __launch_bounds__(256)
init_static_kernel(uint4 *k_slab, uint4 *v_slab, const uint4 *k_src, const uint4 *v_src, StreamState *state, StreamBatch batch, int src_stream0, int L, int B,
                   int rows_per_block /* ring_off + N */, int S_max, int S_src, int row_units, int to_other_bank, CopyStarts starts)
{
    wait_then_release();
    int i = blockIdx.z, chunk = blockIdx.x;
    if (starts.n > 0) {
        i = 0;
        for (int step = kStreamsPerLaunch / 2; step > 0; step >>= 1)
            if (i + step < starts.n && starts.first[i + step] <= chunk) i += step;
        chunk -= starts.first[i];
    }
    const int l = blockIdx.y;
    const int b = batch.id[i];
    const int S = batch.len[i];
    const size_t units = (size_t)S * row_units;
    const size_t src_off = ((size_t)(src_stream0 + i) * L + l) * S_src * row_units;
    // the bank attention reads, or (staging a new prefix while the current one is in use) the other one
    const int bank = ((const volatile StreamState *)state)[b].bank ^ (to_other_bank ? 1 : 0);
    const size_t dst_off = (((size_t)l * B + b) * rows_per_block + (size_t)bank * S_max) * row_units;
    const size_t u0 = (size_t)chunk * (256 * kCopyUnits) + threadIdx.x;
    uint4 k[kCopyUnits], v[kCopyUnits];
#pragma unroll
    for (int j = 0; j < kCopyUnits; ++j)
        if (u0 + j * 256 < units) k[j] = __ldcg(k_src + src_off + u0 + j * 256);
#pragma unroll
    for (int j = 0; j < kCopyUnits; ++j)
        if (u0 + j * 256 < units) v[j] = __ldcg(v_src + src_off + u0 + j * 256);
#pragma unroll
    for (int j = 0; j < kCopyUnits; ++j)
        if (u0 + j * 256 < units) k_slab[dst_off + u0 + j * 256] = k[j];
#pragma unroll
    for (int j = 0; j < kCopyUnits; ++j)
        if (u0 + j * 256 < units) v_slab[dst_off + u0 + j * 256] = v[j];
    if (chunk == 0 && l == 0 && threadIdx.x == 0) {
        if (to_other_bank) state[b].staged_len = S;
        else state[b].static_len = S;
    }
}

cudaError_t launch_init_static(void *k_slab, void *v_slab, const void *k_src, const void *v_src, StreamState *state,
                               const StreamBatch &batch, int n, int src_stream0, int L, int B, int S_max, int ring_off, int N, int S_src, int to_other_bank,
                               size_t row_bytes, cudaStream_t st)
{
    const int row_units = (int)(row_bytes / 16);
    CopyStarts starts = {};
    long long all = 0, longest = 1;
    for (int i = 0; i < n; ++i) {
        const long long units = (long long)batch.len[i] * row_units, blocks = units > 0 ? (units + 256 * kCopyUnits - 1) / (256 * kCopyUnits) : 1;
        starts.first[i] = (int)all;
        all += blocks;
        longest = blocks > longest ? blocks : longest;
    }
    // a quarter of the even grid's blocks without work: the search that each of the others then makes is cheaper
    const bool uneven = all * 4 <= longest * n * 3 && all <= 0x7FFFFFFF;
    starts.n = uneven ? n : 0;
    return launch_overlapped(init_static_kernel, uneven ? dim3((unsigned)all, L, 1) : dim3((unsigned)longest, L, n), 256, st, (uint4 *)k_slab, (uint4 *)v_slab,
                             (const uint4 *)k_src, (const uint4 *)v_src, state, batch, src_stream0, L, B, ring_off + N, S_max, S_src, row_units, to_other_bank, starts);
}

// grid = (chunks, n). Every block reads (head, count) of its stream, copies its share of the
// L*m rows to slots (head + i) mod N, then takes a ticket; the last block to arrive publishes the new
// state. No block waits for another, so there is no spin and nothing to time out.
__global__ void __launch_bounds__(256)
append_sliding_kernel(uint4 *k_slab, uint4 *v_slab, const uint4 *k_src, const uint4 *v_src, StreamState *state, int64_t *total, StreamBatch batch,
                      int src_stream0, int L, int B, int ring_off, int N, int m, int row_units)
{
    wait_then_release();
    const int i = blockIdx.y;
    const int b = batch.id[i];
    __shared__ int s_head;
    if (threadIdx.x == 0) s_head = ((volatile StreamState *)state)[b].head;
    __syncthreads();
    const int head = s_head;
    const unsigned units = (unsigned)L * m * row_units;              // 16-byte units of one stream (2^32 of them would be 64 GB)
    const size_t src_base = (size_t)(src_stream0 + i) * units;
    const int rows_per_block = ring_off + N;
    // A thread's units of K and V are asked for together, two of each at a time (8 streams x 18 layers x 5 rows: 5.7 us with one pair behind
    // the other, 4.6 so; four of each are no faster there and slower, 8.4 us against 7.2, at 32 streams x 18 x 32).
    for (unsigned u0 = blockIdx.x * 512u + threadIdx.x; u0 < units; u0 += gridDim.x * 512u) {
        uint4 k[2], v[2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (u0 + j * 256u < units) { k[j] = __ldcg(k_src + src_base + u0 + j * 256u); v[j] = __ldcg(v_src + src_base + u0 + j * 256u); }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const unsigned u = u0 + j * 256u;
            if (u >= units) break;
            const unsigned r = u / (unsigned)row_units, off = u - r * row_units, l = r / (unsigned)m;
            int slot = head + (int)(r - l * m);
            if (slot >= N) slot -= N;
            const size_t dst = (((size_t)l * B + b) * rows_per_block + ring_off + slot) * row_units + off;
            k_slab[dst] = k[j];
            v_slab[dst] = v[j];
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const int arrived = atomicAdd(&state[b].ticket, 1);
        if (arrived == (int)gridDim.x - 1) {
            // every block of this launch has read `head` and finished its copies: publish the new state
            const int count_old = ((volatile StreamState *)state)[b].count;
            state[b].head = (head + m) % N;
            state[b].count = min(count_old + m, N);
            total[b] += m;
            __threadfence();
            state[b].ticket = 0;
        }
    }
}

cudaError_t launch_append_sliding(void *k_slab, void *v_slab, const void *k_src, const void *v_src, StreamState *state,
                                  int64_t *total, const StreamBatch &batch, int n, int src_stream0, int L, int B, int ring_off,
                                  int N, int m, size_t row_bytes, cudaStream_t st)
{
    const int row_units = (int)(row_bytes / 16);
    const size_t units = (size_t)L * m * row_units;
    int chunks = (int)((units + 256 * 4 - 1) / (256 * 4));
    if (chunks < 1) chunks = 1;
    if (chunks > 32) chunks = 32;
    dim3 grid(chunks, n);
    return launch_overlapped(append_sliding_kernel, grid, 256, st, (uint4 *)k_slab, (uint4 *)v_slab, (const uint4 *)k_src, (const uint4 *)v_src,
                             state, total, batch, src_stream0, L, B, ring_off, N, m, row_units);
}

// The staged prefix becomes the one attention reads: flip the bank, take over the staged length.
__global__ void commit_static_kernel(StreamState *state, StreamBatch batch, int n)
{
    wait_then_release();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int b = batch.id[i];
    StreamState s = state[b];
    if (s.staged_len >= 0) {
        s.bank ^= 1;
        s.static_len = s.staged_len;
        s.staged_len = -1;
        state[b] = s;
    }
}

cudaError_t launch_commit_static(StreamState *state, const StreamBatch &batch, int n, cudaStream_t st)
{
    return launch_overlapped(commit_static_kernel, dim3((n + 127) / 128), 128, st, state, batch, n);
}

// Self-test of the bounded-wait convention every kernel of the library follows: one thread waits on an mbarrier that
// nothing will ever complete, with a time limit, and on expiry records the wait site in the status word and returns.
// Nothing here can hang: the limit is clamped by the launcher, and the loop leaves on its own.
__global__ void wait_limit_probe_kernel(uint32_t *status, unsigned long long limit_ns)
{
    __shared__ __align__(8) unsigned long long probe_bar;
    using namespace ptx;
    const uint32_t bar = smem_u32(&probe_bar);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        const unsigned long long t_start = globaltimer_ns();
        bool done = false;
        for (uint32_t n = 1; !done; ++n) {
            if (mbar_try_wait(bar, 0)) done = true;                                   // (never: nothing arrives)
            else if ((n & 63u) == 0u && globaltimer_ns() - t_start > limit_ns) break;
        }
        if (!done) atomicCAS(status, 0u, status_word(kSiteProbe));
    }
}

cudaError_t launch_wait_limit_probe(uint32_t *status, unsigned long long limit_ns, cudaStream_t st)
{
    wait_limit_probe_kernel<<<1, 32, 0, st>>>(status, limit_ns);
    count_launch();
    return cudaGetLastError();
}

}  // namespace reflex
