// pfc_words.h -- words handed out from one page that many objects share.
#pragma once

#include <stdint.h>

#include <mutex>

namespace pfc {

// Up to N words at a time, from one page of N that is made on first use and
// kept: taking and giving back a word is cheap where making its memory is not.
// Safe with several threads.  Page: static double* make() (null where it fails)
// and static bool alive(double*) (false once something else has freed it: a new
// page is made then, and words of the old one that come back are ignored).
template <class Page, int N = 512>
class WordPool {
public:
    struct Word {
        double* p = nullptr;        // null: none left (or no page)
        unsigned page = 0;
    };
    Word take()
    {
        std::lock_guard<std::mutex> lock(m_);
        if (base_ && !Page::alive(base_)) base_ = nullptr;
        if (!base_) {
            base_ = Page::make();
            if (!base_) return {};
            ++page_;
            for (uint64_t& u : used_) u = 0;
        }
        for (int k = 0; k < N; ++k)
            if (!(used_[k / 64] >> (k % 64) & 1)) {
                used_[k / 64] |= uint64_t(1) << (k % 64);
                return { base_ + k, page_ };
            }
        return {};
    }
    void give(Word w)
    {
        std::lock_guard<std::mutex> lock(m_);
        if (!w.p || !base_ || w.page != page_) return;
        const long k = w.p - base_;
        used_[k / 64] &= ~(uint64_t(1) << (k % 64));
    }

private:
    static_assert(N % 64 == 0, "whole words of the bit set");
    std::mutex m_;
    double* base_ = nullptr;
    unsigned page_ = 0;
    uint64_t used_[N / 64] = {};
};

}  // namespace pfc
