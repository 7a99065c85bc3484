// Host packing of read codes (0..3, anything above is N) into the batch layout:
// 2 bits a base and an N bit a base, eight codes at a time.
#pragma once

#include <cstdint>
#include <cstring>

namespace aln {

// Appends bases to the two bit streams from base index `at` on.  Words it fills
// whole are stored; the first word of a start inside a word, and the last one
// left part-filled (finish()), are ORed in, so that a neighbouring packer may own
// the rest of them: those words have to be zero before.
class Packer {
public:
    Packer(uint32_t *bases, uint32_t *nmask, uint64_t at)
        : b_(bases + at / 16), n_(nmask + at / 32), bn_(2 * (at % 16)), nn_(at % 32), b_shared_(bn_ != 0),
          n_shared_(nn_ != 0) {}

    void read(const uint8_t *codes, uint32_t len) {
        uint32_t t = 0;
        for (; t + 8 <= len; t += 8) eight(codes + t, 8);
        if (t < len) eight(codes + t, len - t);
    }

    void finish() {
        if (bn_) __atomic_fetch_or(b_, static_cast<uint32_t>(bacc_), __ATOMIC_RELAXED);
        if (nn_) __atomic_fetch_or(n_, static_cast<uint32_t>(nacc_), __ATOMIC_RELAXED);
    }

private:
    void eight(const uint8_t *c, uint32_t count) {
        uint64_t x = 0;
        std::memcpy(&x, c, count);  // little-endian: code i in byte i
        const uint64_t big = x & 0xFCFCFCFCFCFCFCFCull;
        const uint64_t one = ((((big & 0x7F7F7F7F7F7F7F7Full) + 0x7F7F7F7F7F7F7F7Full) | big) >> 7) & 0x0101010101010101ull;
        uint64_t y = x & 0x0303030303030303ull & ~(one * 255);  // an N is stored as 0
        y = (y | (y >> 6)) & 0x000F000F000F000Full;
        y = (y | (y >> 12)) & 0x000000FF000000FFull;
        y = (y | (y >> 24)) & 0xFFFFull;
        bacc_ |= y << bn_;
        bn_ += 2 * count;
        if (bn_ >= 32) {
            put(b_, static_cast<uint32_t>(bacc_), b_shared_);
            bacc_ >>= 32;
            bn_ -= 32;
        }
        nacc_ |= ((one * 0x0102040810204080ull) >> 56) << nn_;
        nn_ += count;
        if (nn_ >= 32) {
            put(n_, static_cast<uint32_t>(nacc_), n_shared_);
            nacc_ >>= 32;
            nn_ -= 32;
        }
    }

    static void put(uint32_t *&to, uint32_t v, bool &shared) {
        if (shared) __atomic_fetch_or(to, v, __ATOMIC_RELAXED);
        else *to = v;
        shared = false;
        to++;
    }

    uint32_t *b_, *n_;
    uint64_t bacc_ = 0, nacc_ = 0;
    unsigned bn_, nn_;
    bool b_shared_, n_shared_;
};

}  // namespace aln
