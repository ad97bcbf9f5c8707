// Marks, for the calling thread, the launches that run beside others on the
// lanes of one batch; they take one split of the SMs' L1 (launch.cuh).
#pragma once

namespace catfhe {

class LaneScope {
   public:
    explicit LaneScope(bool on) : before_(flag()) { flag() = on; }
    ~LaneScope() { flag() = before_; }
    LaneScope(const LaneScope &) = delete;
    LaneScope &operator=(const LaneScope &) = delete;
    static bool active() { return flag(); }

   private:
    static bool &flag() {
        thread_local bool on = false;
        return on;
    }
    bool before_;
};

}  // namespace catfhe
