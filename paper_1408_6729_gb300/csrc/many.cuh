// many.cuh -- a kernel's launch for one sort call, or for all the instances of
// a batch at once.
//
// A kernel takes Many<A>: one argument block by value, or (MANY) a table of
// them, one per call, with the first block of each call's share of the grid.  A
// CTA of a MANY launch finds its call by binary search over those starts and
// copies its arguments to shared memory.  `block` and `blocks` stand for
// blockIdx.x and gridDim.x inside the call's share.
//
// A batch of 150 instances of 2^8 to 2^22 keys: 3.4 ms; recorded instance by
// instance into a graph of eight lanes, with 40 launches each, 10.3 ms.
#pragma once

#include <cstring>
#include <functional>
#include <vector>

#include "kernels.cuh"

namespace bsps {

template <typename A> struct Many {
    A one;
    const A *all;
    const uint32_t *first;  // count + 1 entries
    int count;
};

template <bool MANY, typename A> struct Pick;
template <typename A> struct Pick<false, A> {
    const A &a;
    const uint32_t block, blocks;
    __device__ explicit Pick(const Many<A> &m) : a(m.one), block(blockIdx.x), blocks(gridDim.x) {}
};
template <typename A> struct Pick<true, A> {
    const A &a;
    uint32_t block, blocks;
    __device__ static A &slot() {
        __shared__ A s;
        return s;
    }
    __device__ explicit Pick(const Many<A> &m) : a(slot()) {
        int lo = 0, hi = m.count - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (m.first[mid] <= blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        block = blockIdx.x - m.first[lo];
        blocks = m.first[lo + 1] - m.first[lo];
        static_assert(sizeof(A) % 4 == 0, "copied by words");
        const uint32_t *src = reinterpret_cast<const uint32_t *>(m.all + lo);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&slot());
        for (int i = threadIdx.x; i < (int)(sizeof(A) / 4); i += blockDim.x) dst[i] = src[i];
        __syncthreads();
    }
};

// What the launchers run on: one call on its stream, or -- `many` -- the calls
// of a batch, whose argument tables gather in host memory and whose launches
// are kept until the tables are on the device.
struct Exec {
    const Ctx *calls;
    int count;
    cudaStream_t stream;
    bool many = false;
    std::vector<unsigned char> *tables = nullptr;
    const unsigned char *device_tables = nullptr;
    std::vector<std::function<cudaError_t()>> *later = nullptr;

    template <typename T> size_t put(const std::vector<T> &v) {
        const size_t at = (tables->size() + 15) & ~size_t(15);
        tables->resize(at + v.size() * sizeof(T));
        std::memcpy(tables->data() + at, v.data(), v.size() * sizeof(T));
        return at;
    }
};

// A call of a batch that is in the table but adds no blocks to the grid.
constexpr uint32_t kNoBlocks = 0xffffffffu;

// Launches `single` for the one call, or `all` once for every call of a batch.
// make(ctx, args) fills a call's arguments and returns its blocks (0: the call
// does not run this kernel); smem.bytes is enough for any of them.
template <typename A, typename K1, typename KN, typename Make>
cudaError_t launch_calls(Exec &x, K1 single, KN all, unsigned threads, DynSmem smem, Make make) {
    if (!x.many) {
        Many<A> m = {};
        const uint32_t blocks = make(x.calls[0], m.one);
        if (blocks == 0) return cudaSuccess;
        const cudaError_t e = smem.allow(single);
        if (e != cudaSuccess) return e;
        single<<<blocks, threads, smem.bytes, x.stream>>>(m);
        return cudaGetLastError();
    }
    std::vector<A> args;
    std::vector<uint32_t> first(1, 0u);
    for (int i = 0; i < x.count; ++i) {
        A a = {};
        const uint32_t blocks = make(x.calls[i], a);
        if (blocks == 0) continue;
        args.push_back(a);
        first.push_back(first.back() + (blocks == kNoBlocks ? 0u : blocks));
    }
    if (args.empty()) return cudaSuccess;
    const size_t at = x.put(args), ft = x.put(first);
    Many<A> m = {};
    m.all = reinterpret_cast<const A *>(x.device_tables + at);
    m.first = reinterpret_cast<const uint32_t *>(x.device_tables + ft);
    m.count = (int)args.size();
    const unsigned grid = first.back();
    const cudaStream_t stream = x.stream;
    x.later->push_back([=]() -> cudaError_t {
        const cudaError_t e = smem.allow(all);
        if (e != cudaSuccess) return e;
        all<<<grid, threads, smem.bytes, stream>>>(m);
        return cudaGetLastError();
    });
    return cudaSuccess;
}

// launchers of the keys-only random path (sample.cu, mlp.cu, route_keys.cu,
// route.cu, bucket.cu)
cudaError_t launch_sample_random(Exec &x);   // also clears the call's status, cursors and flags
cudaError_t launch_sample_sort(Exec &x);
cudaError_t launch_splitters(Exec &x);
cudaError_t launch_mlp_train(Exec &x);
cudaError_t launch_route_keys(Exec &x);
cudaError_t launch_bucket_finish(Exec &x);
cudaError_t launch_bucket_keys(Exec &x);
cudaError_t launch_route_words(Exec &x);     // single calls of 4-byte keys with payloads, as words
cudaError_t launch_pair_words(Exec &x);      // ... and their final step (pairs.cu)
cudaError_t launch_bucket_pairs(Exec &x);    // single calls
cudaError_t launch_repeats_cluster(Exec &x); // single calls of 4-byte keys with payloads, on both routes

// api.cu: a call's plan, checks and layout, and the path above for calls that
// are ready (random sampling, keys only, at least one key each)
int prepare_keys_call(Ctx &c, const void *keys_in, void *keys_out, int64_t n, int32_t dtype, const bsps_params *prm,
                      int64_t *bucket_sizes, void *ws, size_t ws_bytes, void *stream);
int run_keys_calls(Exec &x);

} // namespace bsps
