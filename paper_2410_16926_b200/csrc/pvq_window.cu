// Host side of the windowed search tables (pvq_window.cuh): chooses the windows, computes the tables in
// exact integers and keeps them on the device.
#include <algorithm>
#include <cmath>
#include <list>
#include <memory>
#include <mutex>
#include <new>

#include "pvq_bigint.h"
#include "pvq_window.cuh"

namespace pvq {

namespace {

double log2_of(const BigU& v) {
    const int b = v.bit_length();
    if (b == 0) return -1e30;
    return b <= 32 ? std::log2(static_cast<double>(v.w[0])) : std::log2(static_cast<double>(v.bits_at(b - 32))) + (b - 32);
}

// v >> pos, or v << -pos: the low 32 bits
uint32_t word_at(const BigU& v, int pos) {
    if (pos >= 0) return v.bits_at(pos);
    return pos <= -32 ? 0u : v.w[0] << -pos;
}

// What the kernel computes from the leading `words` words of a number whose block has `bits` bits.
uint32_t aligned_key(const BigU& v, int bits, int words) {
    unsigned __int128 f = 0;
    for (int w = 1; w <= words; ++w) f = f << 32 | word_at(v, bits - 32 * w);
    if (f == 0) return 0u;
    const uint64_t high = static_cast<uint64_t>(f >> 64), low = static_cast<uint64_t>(f);
    const int e = high ? 127 - __builtin_clzll(high) : 63 - __builtin_clzll(low);
    const uint32_t mant = static_cast<uint32_t>(e >= 23 ? f >> (e - 23) : f << (23 - e));
    return (static_cast<uint32_t>(e + 127) << 23) | (mant & 0x7fffffu);
}

struct Builder {
    int N, K;
    std::vector<BigU> cnt;  // N(n,k), n = 0..N
    std::vector<double> lg;
    std::vector<int> lo, hi, bits, words;  // windows of the positions; bits and words of the blocks
    WinTables t;
    std::vector<uint32_t> data, thr;

    const BigU& count(int n, int k) const { return cnt[static_cast<size_t>(n) * (K + 1) + k]; }
    BigU threshold(int n, int m) const {
        BigU v = count(n + 1, m >> 1);
        if (m & 1) v.add(count(n, m >> 1));
        return v;
    }

    bool counts() {
        cnt.resize(static_cast<size_t>(N + 1) * (K + 1));
        CountColumn c(N);
        for (int k = 0; k <= K; ++k) {
            if (k > 0 && !c.advance()) return false;
            for (int n = 0; n <= N; ++n) cnt[static_cast<size_t>(n) * (K + 1) + k] = c.col[static_cast<size_t>(n)];
        }
        lg.resize(cnt.size());
        for (size_t i = 0; i < cnt.size(); ++i) lg[i] = log2_of(cnt[i]);
        return true;
    }

    // of all codes, the share with k pulses left after position i is N(i+1, K-k) N(n,k) / N(N,K)
    int windows(double eps) {
        lo.assign(N, 0);
        hi.assign(N, 0);
        const double total = lg[static_cast<size_t>(N) * (K + 1) + K];
        for (int i = 0; i < N; ++i) {
            const int n = N - 1 - i;
            auto share = [&](int k) {
                return std::exp2(lg[static_cast<size_t>(i + 1) * (K + 1) + K - k] + lg[static_cast<size_t>(n) * (K + 1) + k] - total);
            };
            double s = 0.0;
            int a = 0, b = K;
            while (a < K && s + share(a) < eps) s += share(a++);
            s = 0.0;
            while (b > a && s + share(b) < eps) s += share(b--);
            lo[i] = a;
            hi[i] = b;
        }
        int most = 0;
        for (int i = N - 1; i >= 0; --i) {
            if (i + 1 < N) hi[i] = std::max(hi[i], hi[i + 1]);
        }
        for (int i = N - 1; i >= 0; --i) {
            // the lowest threshold has to show in the words that make up the key, with some bits to tell it from others
            const int b0 = i & ~3;
            const double top = lg[static_cast<size_t>(N - b0) * (K + 1) + before(b0)];
            while (lo[i] < hi[i] && lg[static_cast<size_t>(N - i) * (K + 1) + lo[i]] < top - (32 * win_key_words(N) - 8)) ++lo[i];
            if (i + 1 < N) lo[i] = std::max(lo[i], lo[i + 1]);
            most = std::max(most, 2 * (hi[i] - lo[i]) + 2);
        }
        return most;
    }
    int before(int i) const { return i > 0 ? hi[i - 1] : K; }

    // Fills t, data and thr for the current windows; false: cannot be done.
    bool layout(const int plane) {
        const int blocks = N / 4;
        bits.assign(blocks, 0);
        words.assign(blocks, 0);
        std::memset(&t, 0, sizeof t);
        t.plane = plane;
        data.clear();
        thr.clear();
        std::vector<int> last_m(N);
        std::vector<char> closed(N);  // no q of the row is beyond its last threshold
        for (int i = 0; i < N; ++i) {
            const int n = N - 1 - i;
            last_m[i] = hi[i] == K ? 2 * K : 2 * hi[i] + 1;
            const BigU top = threshold(n, last_m[i]);
            closed[i] = !top.less(count(n + 1, K));
            bits[i / 4] = std::max({bits[i / 4], top.bit_length(), count(n + 1, before(i)).bit_length()});
        }
        for (int b = 1; b < blocks; ++b) bits[b] = std::min(bits[b - 1], std::max(bits[b], bits[b - 1] - 16));
        for (int b = 0; b < blocks; ++b) {
            words[b] = (bits[b] + 31) / 32;
            if (words[b] > 32) return false;
            for (int w = 0; w <= words[b]; ++w) ++t.args.blocks_of[w];
            const int delta = (b > 0 ? bits[b - 1] : 32 * words[0]) - bits[b];
            const int W = words[b], up = 32 * W - bits[b], kw = std::min(W, win_key_words(N));
            t.args.up[b] = static_cast<uint8_t>(up);
            const size_t at = data.size(), planes = static_cast<size_t>(4) * W * plane;
            t.args.block_off[b] = static_cast<uint32_t>(at * 4);
            t.args.thr_off[b] = static_cast<uint32_t>(thr.size() * 4);
            const size_t e_at = at + kWinHead / 4;
            data.resize(e_at + planes, 0u);
            uint32_t dlo4 = 0, klo4 = 0, width4 = 0;
            const size_t tat = thr.size();
            thr.resize(tat + planes, 0u);
            for (int s = 0; s < 4; ++s) {
                const int i = 4 * b + s, n = N - 1 - i;
                const int dlo = (i > 0 ? lo[i - 1] : K) - lo[i];
                // |y| and the sums of the packed arithmetic stay below 256, and an out-of-window index behind one inside shows
                if (dlo < 0 || dlo > 127 || before(i) - lo[i] >= 127 || last_m[i] - 2 * lo[i] + 1 > plane) return false;
                t.args.klo[i] = static_cast<int16_t>(lo[i]);
                klo4 |= static_cast<uint32_t>(lo[i] & 255) << (8 * (3 - s));  // (read where K <= 255)
                width4 |= static_cast<uint32_t>(hi[i] - lo[i]) << (8 * (3 - s));
                dlo4 |= static_cast<uint32_t>(dlo) << (8 * s);
                std::vector<uint32_t> key;
                const bool below = lo[i] > 0;
                if (below) key.push_back(aligned_key(threshold(n, 2 * lo[i] - 1), bits[b], kw));
                for (int m = 2 * lo[i]; m <= last_m[i]; ++m) {
                    const BigU T = threshold(n, m);
                    BigU M = T;
                    M.sub(count(n, m >> 1));
                    uint64_t carry = 1;
                    for (int w = 0; w < W; ++w) {
                        const size_t o = (static_cast<size_t>(s) * W + w) * plane + (m - 2 * lo[i]);
                        carry += static_cast<uint32_t>(~word_at(M, 32 * w - up));
                        data[e_at + o] = static_cast<uint32_t>(carry);
                        carry >>= 32;
                        thr[tat + o] = word_at(T, 32 * w - up);
                    }
                    key.push_back(aligned_key(T, bits[b], kw));
                }
                if (key[0] == 0u) return false;
                int shift = -1;
                for (int f = 0; f <= 12 && shift < 0; ++f) {
                    bool distinct = true;
                    for (size_t j = 1; j < key.size() && distinct; ++j) distinct = (key[j] >> (23 - f)) != (key[j - 1] >> (23 - f));
                    if (distinct) shift = 23 - f;
                }
                if (shift < 0) return false;
                const uint32_t first = (key[0] >> shift) + (below ? 1u : 0u);
                const uint32_t many = (key.back() >> shift) - first + (closed[i] ? 1u : 0u);
                const WinRow r = {first << shift, many << shift, static_cast<uint32_t>(shift), static_cast<uint32_t>((data.size() - at) * 4)};
                std::memcpy(&data[at + 4 * s], &r, sizeof r);
                uint32_t m0 = 0;
                for (uint32_t x = 0; x < many; ++x) {
                    const uint32_t k = key[m0 + (below ? 1 : 0)];
                    uint32_t e = (m0 - ((x << shift) >> 24)) << 24;
                    if ((k >> shift) == first + x) {
                        // an integer below 2^23 is its key: half a step more, and equal keys need no further look
                        const bool exact = bits[b] <= 32 * kw && threshold(n, 2 * lo[i] + static_cast<int>(m0)).bit_length() < 23;
                        e |= ~(k + (exact ? 1u : 0u) - r.base) & 0xffffffu;
                        ++m0;
                    }
                    data.push_back(e);
                }
                data.push_back((255u - (r.last >> 24)) << 24);
            }
            data[at + kWinDlo4 / 4] = dlo4;
            data[at + kWinDelta / 4] = static_cast<uint32_t>(delta);
            data[at + kWinKlo4 / 4] = klo4;
            data[at + kWinWidth4 / 4] = width4;
            t.args.words[b] = static_cast<uint8_t>(W);
            t.max_rows = std::max(t.max_rows, win_rows_bytes(W, plane));
            // (an out-of-window index reads up to 256 entries from the start of a plane)
            while ((data.size() & 3u) || data.size() < e_at + planes + 256 - plane) data.push_back(0u);
            t.max_block = std::max(t.max_block, static_cast<uint32_t>((data.size() - at) * 4));
        }
        t.args.block_off[blocks] = static_cast<uint32_t>(data.size() * 4);
        BigU q(1u);
        for (int i = 0, k = K; i < N; ++i) {
            const int n = N - 1 - i, left = std::min(k, (lo[i] + hi[i]) / 2), m = 2 * left + (left < k ? 1 : 0);
            q.add(threshold(n, m));
            q.sub(count(n, left));
            k = left;
        }
        for (int w = 0; w < kWinWords; ++w) t.args.typical[w] = q.w[w];
        return words[0] <= kWinWords;
    }

    // The widest windows (the smallest share outside) whose tables fit beside the output slots of 32 warps (N = 64); where
    // none does, the tables are streamed, and the widest are taken that 160 (192 at N = 64) entries a row hold.
    bool choose(uint32_t smem_max) {
        const uint32_t room = smem_max - 128u - 32u * 32u * (N + 4);
        for (int plane : {96, N == 64 ? 192 : 160})
            for (double eps : {1e-8, 3e-8, 1e-7, 3e-7, 1e-6, 3e-6, 1e-5, 3e-5, 1e-4, 3e-4, 1e-3}) {
                if (plane == 96 && N > 64) break;
                if (windows(eps) <= plane && layout(plane) && (plane != 96 || t.args.block_off[N / 4] <= room)) return true;
            }
        return false;
    }
};

struct Kept : WinTables {
    int dev, N, K;
    uint8_t* mem = nullptr;
    bool captured = false;  // a stream capture has recorded a launch with these addresses: kept for good
};

std::mutex g_build_mu;  // one thread builds at a time
std::mutex g_mu;        // the lists; held for a look, never while something is computed, allocated, copied or freed
std::list<std::shared_ptr<Kept>>& kept() {  // oldest first; lives as long as the process
    static auto* l = new std::list<std::shared_ptr<Kept>>;
    return *l;
}
std::list<std::shared_ptr<Kept>>& retired() {  // no longer found; freed when no launch holds them any more
    static auto* l = new std::list<std::shared_ptr<Kept>>;
    return *l;
}

std::shared_ptr<Kept> find_kept(int dev, int N, int K) {
    for (auto& k : kept())
        if (k->dev == dev && k->N == N && k->K == K) return k;
    return nullptr;
}

// Room for one more table on the device: the oldest one that no capture holds goes.  False where there is none.
bool make_room(int dev) {
    std::lock_guard<std::mutex> lock(g_mu);
    auto& l = kept();
    const auto mine = [dev](const std::shared_ptr<Kept>& o) { return o->dev == dev; };
    if (std::count_if(l.begin(), l.end(), mine) < kWinKept) return true;
    const auto it = std::find_if(l.begin(), l.end(), [dev](const std::shared_ptr<Kept>& o) { return o->dev == dev && !o->captured; });
    if (it == l.end()) return false;
    retired().splice(retired().end(), l, it);
    return true;
}

// Frees what has been retired and is in no launching thread's hands (nobody can get hold of it any more; cudaFree waits
// for the kernels that may be reading it).
void free_retired(int dev) {
    std::list<std::shared_ptr<Kept>> gone;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        for (auto it = retired().begin(); it != retired().end();) {
            const auto o = it++;
            if ((*o)->dev == dev && o->use_count() == 1) gone.splice(gone.end(), retired(), o);
        }
    }
    for (const auto& o : gone) cudaFree(o->mem);
}

// Copies to the device and waits until the copy is there: launches on any stream may follow.  (A plain cudaMemcpy from
// pageable memory returns when the data is staged, and orders only the legacy stream behind it.)
bool upload(uint8_t* dst, const std::vector<uint32_t>& src) {
    cudaStream_t s = nullptr;
    if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return false;
    const bool ok = cudaMemcpyAsync(dst, src.data(), src.size() * 4, cudaMemcpyHostToDevice, s) == cudaSuccess;
    const bool there = cudaStreamSynchronize(s) == cudaSuccess;
    cudaStreamDestroy(s);
    return ok && there;
}

struct FreeOnDevice {
    void operator()(uint8_t* p) const { cudaFree(p); }
};

// (std::bad_alloc leaves everything as it was)
void compute_and_keep(int dev, int N, int K, uint32_t smem_max) {
    Builder b;
    b.N = N;
    b.K = K;
    if (!b.counts() || !b.choose(smem_max)) return;
    auto k = std::make_shared<Kept>();
    static_cast<WinTables&>(*k) = b.t;
    k->dev = dev, k->N = N, k->K = K;
    std::list<std::shared_ptr<Kept>> entry(1, k);
    const bool room = make_room(dev);
    free_retired(dev);
    const size_t data_bytes = (b.data.size() * 4 + 255) & ~size_t(255), thr_bytes = b.thr.size() * 4;
    void* mem = nullptr;
    if (!room || cudaMalloc(&mem, data_bytes + thr_bytes) != cudaSuccess) return;
    std::unique_ptr<uint8_t, FreeOnDevice> held(static_cast<uint8_t*>(mem));
    if (!upload(held.get(), b.data) || !upload(held.get() + data_bytes, b.thr)) return;
    k->args.data = held.get();
    k->args.thr = held.get() + data_bytes;
    k->mem = held.release();
    std::lock_guard<std::mutex> lock(g_mu);
    kept().splice(kept().end(), entry);
}

}  // namespace

std::shared_ptr<const WinTables> window_tables(int N, int K, cudaStream_t stream) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(g_mu);
    auto k = find_kept(dev, N, K);
    if (k && !k->captured) {
        // a graph replays the launch with these addresses, whatever has been built in between
        cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess) return nullptr;
        k->captured = capturing != cudaStreamCaptureStatusNone;
    }
    return k;
}

void build_window_tables(int N, int K, cudaStream_t stream) {
    if (!has_window_tables(N, code_words_for(N, K), K) || count_fills_its_words(N, K)) return;
    int dev = 0;
    DeviceInfo di;
    if (cudaGetDevice(&dev) != cudaSuccess || device_info(&di) != PVQ_OK) return;
    std::lock_guard<std::mutex> building(g_build_mu);
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (find_kept(dev, N, K)) return;
    }
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &capturing) != cudaSuccess || capturing != cudaStreamCaptureStatusNone) return;
    // (these calls concern nobody's capture: the memory is this function's own)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    try {
        compute_and_keep(dev, N, K, static_cast<uint32_t>(di.smem_max));
    } catch (const std::bad_alloc&) {  // a few MB to 50 MB of host memory are not there: done without, as said above
    }
    cudaGetLastError();
    cudaThreadExchangeStreamCaptureMode(&mode);
}

}  // namespace pvq
