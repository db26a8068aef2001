// Replays of whole calls as CUDA graphs.
//
// A call of this library is a fixed sequence of launches for given descriptors, pointers and switches, and a program that
// steps through the same buffers makes the same call again and again: the launches (2-3 us of host time each) are then
// most of what a small call costs.  The cache keys a call by everything its launch sequence depends on.  The first two
// calls with a key are enqueued directly; the third is captured (on a stream of the cache's own, since the caller's may be
// the legacy default stream) and instantiated, and from then on the call is one graph launch.  Nothing of a call's result
// is kept.  The cache is bounded: with kMaxGraphs held, a new one is made only in place of one that has not been used for
// kStaleCalls calls (so a program with more calls than that in its loop keeps the graphs it has), and all go with the
// context.  (An executable graph that is still running when it is destroyed is freed on completion.)
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <memory>
#include <vector>

namespace sc {

class CallKey {
public:
    void reset(uint32_t call) { buf_.clear(); add(&call, sizeof(call)); }
    void add(const void* p, size_t n) {
        const uint32_t len = p ? (uint32_t)n : 0xFFFFFFFFu;        // an absent part differs from any present one
        push(&len, sizeof(len));
        if (p) push(p, n);
    }
    template <typename T> void val(T v) { push(&v, sizeof(v)); }
    uint64_t hash() const {
        uint64_t h = 0x9E3779B97F4A7C15ull ^ buf_.size();
        size_t i = 0;
        for (; i + 8 <= buf_.size(); i += 8) { uint64_t w; memcpy(&w, &buf_[i], 8); h = (h ^ w) * 0xD6E8FEB86659FD93ull; h ^= h >> 32; }
        for (; i < buf_.size(); ++i) h = (h ^ (uint8_t)buf_[i]) * 0x100000001B3ull;
        return h ^ (h >> 29);
    }
    const std::vector<char>& bytes() const { return buf_; }
private:
    void push(const void* p, size_t n) { const char* c = (const char*)p; buf_.insert(buf_.end(), c, c + n); }
    std::vector<char> buf_;
};

class GraphCache {
public:
    static constexpr int kMaxGraphs = 64, kMaxSeen = 256, kDirectCalls = 2, kStaleCalls = 1024;
    ~GraphCache() { clear(); }
    void clear() {
        for (auto& e : graphs_) cudaGraphExecDestroy(e->exec);
        graphs_.clear(); seen_.clear();
        if (stream_) { cudaStreamDestroy(stream_); stream_ = nullptr; }
    }

    // Runs `body(stream)` -- which enqueues the call and returns a status -- or replays it.  *launches is the caller's
    // launch counter; a replay advances it by what the captured call advanced it.
    template <typename F>
    int run(const CallKey& key, cudaStream_t stream, int64_t* launches, int cuda_error, F&& body) {
        const uint64_t h = key.hash();
        ++clock_;
        for (auto& e : graphs_) {
            if (e->hash != h || e->key != key.bytes()) continue;
            if (!capturable(stream)) return body(stream);
            e->used = clock_;
            if (cudaGraphLaunch(e->exec, stream) != cudaSuccess) return cuda_error;
            *launches += e->launches;
            return 0;
        }
        size_t old = graphs_.size();                 // where the new graph goes
        if ((int)graphs_.size() == kMaxGraphs) {
            old = 0;
            for (size_t i = 1; i < graphs_.size(); ++i) if (graphs_[i]->used < graphs_[old]->used) old = i;
            if (clock_ - graphs_[old]->used < kStaleCalls) return body(stream);
        }
        if (!worth(h) || !capturable(stream)) return body(stream);
        if (!stream_ && cudaStreamCreateWithFlags(&stream_, cudaStreamNonBlocking) != cudaSuccess) { cudaGetLastError(); return body(stream); }
        if (cudaStreamBeginCapture(stream_, cudaStreamCaptureModeThreadLocal) != cudaSuccess) { cudaGetLastError(); return body(stream); }
        const int64_t l0 = *launches;
        const int rc = body(stream_);
        cudaGraph_t graph = nullptr;
        const bool ended = cudaStreamEndCapture(stream_, &graph) == cudaSuccess && graph;
        const int64_t n = *launches - l0;
        *launches = l0;
        cudaGraphExec_t exec = nullptr;
        const bool ok = rc == 0 && ended && cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
        if (graph) cudaGraphDestroy(graph);
        if (rc != 0 && rc != cuda_error) return rc;  // the call was refused; nothing was enqueued
        if (!ok) { cudaGetLastError(); return body(stream); }
        if (old < graphs_.size()) {
            cudaGraphExecDestroy(graphs_[old]->exec);
            graphs_.erase(graphs_.begin() + old);
        }
        graphs_.push_back(std::unique_ptr<Entry>(new Entry{h, key.bytes(), exec, n, clock_}));
        if (cudaGraphLaunch(exec, stream) != cudaSuccess) return cuda_error;
        *launches += n;
        return 0;
    }

private:
    struct Entry { uint64_t hash; std::vector<char> key; cudaGraphExec_t exec; int64_t launches; uint64_t used; };
    struct Seen { uint64_t hash; int count; };
    std::vector<std::unique_ptr<Entry>> graphs_;
    std::vector<Seen> seen_;                         // ring of recent keys that have no graph yet
    size_t seen_next_ = 0;
    uint64_t clock_ = 0;
    cudaStream_t stream_ = nullptr;

    // the caller is capturing (its own graph takes the launches), or some capture makes the legacy stream unusable
    static bool capturable(cudaStream_t s) {
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &st) != cudaSuccess) { cudaGetLastError(); return false; }
        return st == cudaStreamCaptureStatusNone;
    }
    bool worth(uint64_t h) {
        for (Seen& s : seen_) if (s.hash == h) return ++s.count > kDirectCalls;
        if (seen_.size() < kMaxSeen) seen_.push_back(Seen{h, 1});
        else { seen_[seen_next_] = Seen{h, 1}; seen_next_ = (seen_next_ + 1) % kMaxSeen; }
        return false;
    }
};

}  // namespace sc
