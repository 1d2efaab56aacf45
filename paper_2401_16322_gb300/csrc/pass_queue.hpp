// Queue of the passes of one step that go out as one launch (host code).
//
// Between begin(true) and end(), add() keeps passes and hands them on Chain::capacity at a time:
// all(chain) sends them as one launch and says whether it could.  Where it could not, one(pass)
// sends those kept one by one, and so it does with every pass added after that (`broken()`) or
// after begin(false).
#pragma once

namespace ewv {

template <class Chain>
class PassQueue {
public:
    void begin(bool together) {
        together_ = together && !broken_;
        chain_.n = 0;
    }
    template <class Pass, class All, class One>
    void add(const Pass& p, All&& all, One&& one) {
        if (together_ && chain_.n == Chain::capacity) flush(all, one);
        if (together_) chain_.pass[chain_.n++] = p;       // (the flush may have ended that)
        else one(p);
    }
    template <class All, class One>
    void end(All&& all, One&& one) {
        flush(all, one);
        together_ = false;
    }
    bool collecting() const { return together_; }
    bool broken() const { return broken_; }

private:
    template <class All, class One>
    void flush(All& all, One& one) {
        if (together_ && chain_.n > 0 && !all(chain_)) {
            broken_ = true;
            together_ = false;
            for (int k = 0; k < chain_.n; ++k) one(chain_.pass[k]);
        }
        chain_.n = 0;
    }
    Chain chain_;
    bool together_ = false, broken_ = false;
};

}  // namespace ewv
