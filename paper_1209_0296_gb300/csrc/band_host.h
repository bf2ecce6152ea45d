// band_host.h -- host-side bookkeeping of band launches that needs no CUDA
// call of its own (plain C++, tested without a GPU).
#pragma once

#include <cstddef>
#include <deque>
#include <mutex>
#include <utility>
#include <vector>

namespace lat {

// Words that kernels write and the host reads (an error word per lattice).  A
// word given back is handed out again only when the work that may still write
// it is complete, so no two live owners ever share one.
class WordPool {
public:
    using Page = int *(*)(size_t words);   // new words, or null
    using Done = bool (*)(void *event);    // the work recorded in event is complete (then the event is freed)

    WordPool(Page page, Done done, size_t words) : page_(page), done_(done), words_(words) {}

    // A zeroed word, or null when there is no memory.
    int *take()
    {
        std::lock_guard<std::mutex> g(mu_);
        try {
            if (free_.empty()) collect(pending_.size());
            if (free_.empty()) {
                free_.reserve(words_);
                int *p = page_(words_);
                if (p == nullptr) return nullptr;
                for (size_t i = words_; i-- > 0;) free_.push_back(p + i);
            }
        } catch (...) {   // a word that cannot be listed is lost, never shared
            return nullptr;
        }
        int *w = free_.back();
        free_.pop_back();
        *w = 0;
        return w;
    }

    // Give w back, free once event is complete (null: at once).  The oldest such
    // words are looked at here, so that taking one asks nothing.
    void give(int *w, void *event)
    {
        std::lock_guard<std::mutex> g(mu_);
        try {
            if (event == nullptr) free_.push_back(w);
            else pending_.emplace_back(w, event);
            collect(2);
        } catch (...) {
        }
    }

private:
    // Free the words of the `most` oldest events that are complete.
    void collect(size_t most)
    {
        while (most-- > 0 && !pending_.empty() && done_(pending_.front().second)) {
            int *w = pending_.front().first;
            pending_.pop_front();
            free_.push_back(w);
        }
    }

    const Page page_;
    const Done done_;
    const size_t words_;
    std::mutex mu_;
    std::vector<int *> free_;
    std::deque<std::pair<int *, void *>> pending_;
};

// A value found once per device (function attributes and SM counts belong to
// one); devices past kMax are asked every time.
template <typename T>
class PerDevice {
public:
    template <typename F>
    T get(int device, F find)
    {
        if (device < 0 || device >= kMax) return find();
        std::call_once(once_[device], [&] { value_[device] = find(); });
        return value_[device];
    }

private:
    static constexpr int kMax = 64;
    std::once_flag once_[kMax];
    T value_[kMax] = {};
};

}  // namespace lat
