// Order of the contact fills of a process (plain C++, no CUDA): the first use of a block
// size on a device runs alone, everything else side by side.
//
// Several host threads at the first use of a block size have stood still (see fill_leads in
// lead.cu); whoever fills contact entries -- any context, any number of entries -- passes
// through here.  A first use waits for the fills that run, holds back those that come, and
// ends with its first entry: the rest of that fill and the held-back ones then run together.
#pragma once
#include <condition_variable>
#include <mutex>
#include <set>
#include <utility>

namespace pwqt {

class FirstUse {
public:
    // One fill's stay.  first(): nobody else is inside and (dev, n) has not been used before;
    // the caller does its first entry and says known(), after which others may enter beside it.
    class Pass {
    public:
        Pass(FirstUse& g, int dev, int n) : g_(g), key_(dev, n) { first_ = g_.enter(key_); }
        Pass(const Pass&) = delete;
        Pass& operator=(const Pass&) = delete;
        ~Pass() { g_.leave(first_); }
        bool first() const { return first_; }
        void known() {
            if (first_) g_.share(key_);
            first_ = false;
        }

    private:
        FirstUse& g_;
        std::pair<int, int> key_;
        bool first_;
    };

private:
    using Key = std::pair<int, int>;      // device, block size
    bool enter(const Key& k) {
        std::unique_lock<std::mutex> l(m_);
        // a first use goes before later comers, or a stream of fills would keep it waiting
        if (!known_.count(k)) {
            ++waiting_;
            cv_.wait(l, [&] { return known_.count(k) ? !alone_ : !alone_ && running_ == 0; });
            --waiting_;
        } else {
            cv_.wait(l, [&] { return !alone_ && waiting_ == 0; });
        }
        ++running_;
        alone_ = !known_.count(k);
        cv_.notify_all();
        return alone_;
    }
    void share(const Key& k) {
        std::lock_guard<std::mutex> l(m_);
        known_.insert(k);
        alone_ = false;
        cv_.notify_all();
    }
    void leave(bool first) {
        std::lock_guard<std::mutex> l(m_);
        --running_;
        if (first) alone_ = false;        // the first entry failed: the next user is the first
        cv_.notify_all();
    }
    std::mutex m_;
    std::condition_variable cv_;
    std::set<Key> known_;
    int running_ = 0, waiting_ = 0;
    bool alone_ = false;
};

}  // namespace pwqt
