// Exact integers of the host side: counts N(n,k) up to 1536 bits (choosing K, laying out the decoders' tables).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <vector>

namespace pvq {

constexpr int kLimbs = 48;

// Unsigned integer of kLimbs 32-bit limbs.
struct BigU {
    uint32_t w[kLimbs];
    BigU() { std::memset(w, 0, sizeof w); }
    explicit BigU(uint32_t v) {
        std::memset(w, 0, sizeof w);
        w[0] = v;
    }
    // *this += o; false when the sum overflows kLimbs
    bool add(const BigU& o) {
        uint64_t c = 0;
        for (int i = 0; i < kLimbs; ++i) {
            uint64_t s = static_cast<uint64_t>(w[i]) + o.w[i] + c;
            w[i] = static_cast<uint32_t>(s);
            c = s >> 32;
        }
        return c == 0;
    }
    // *this -= o (o <= *this)
    void sub(const BigU& o) {
        int64_t b = 0;
        for (int i = 0; i < kLimbs; ++i) {
            const int64_t d = static_cast<int64_t>(w[i]) - o.w[i] + b;
            w[i] = static_cast<uint32_t>(d);
            b = d >> 32;  // 0 or -1
        }
    }
    bool less(const BigU& o) const {
        for (int i = kLimbs - 1; i >= 0; --i)
            if (w[i] != o.w[i]) return w[i] < o.w[i];
        return false;
    }
    int bit_length() const {
        for (int i = kLimbs - 1; i >= 0; --i)
            if (w[i]) return 32 * i + (32 - __builtin_clz(w[i]));
        return 0;
    }
    bool is_pow2() const {
        int ones = 0;
        for (int i = 0; i < kLimbs; ++i) ones += __builtin_popcount(w[i]);
        return ones == 1;
    }
    // ceil(log2 v) for v >= 1
    int ceil_log2() const { return is_pow2() ? bit_length() - 1 : bit_length(); }
    // bits [pos, pos + 32)
    uint32_t bits_at(int pos) const {
        const int l = pos >> 5, s = pos & 31;
        const uint64_t v = (l + 1 < kLimbs ? static_cast<uint64_t>(w[l + 1]) << 32 : 0) | (l < kLimbs ? w[l] : 0u);
        return static_cast<uint32_t>(v >> s);
    }
};

// col[n] = N(n,k) for n = 0..N, advanced from k to k+1 with
// N(n,k+1) = N(n-1,k+1) + N(n,k) + N(n-1,k)   (Sec. 2.4).
struct CountColumn {
    std::vector<BigU> col;
    int k = 0;
    explicit CountColumn(int N) : col(static_cast<size_t>(N) + 1, BigU(1u)) {}  // N(n,0) = 1
    bool advance() {
        std::vector<BigU> nxt(col.size());
        nxt[0] = BigU(0u);  // N(0,k>=1) = 0
        for (size_t n = 1; n < col.size(); ++n) {
            nxt[n] = nxt[n - 1];
            if (!nxt[n].add(col[n]) || !nxt[n].add(col[n - 1])) return false;
        }
        col.swap(nxt);
        ++k;
        return true;
    }
};

}  // namespace pvq
