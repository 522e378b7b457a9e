// How many streams of the process share the device with a launch.
#include <chrono>
#include <mutex>

#include "common.cuh"

namespace rbgs {
namespace {

// Streams whose launches may still run, so that several small solvers at once each take a part of
// the device and not one after the other all of it (a launch that fills the GPU is fastest alone,
// and recomputes the most overlap for it).  A launch adds an estimate of its time to its stream; a stream counts as busy until then, or until its context waits for it.
// Times are taken at three quarters: past the end of the work a stream must not count, or a lone
// solver would be given a part of the device.
//
// The number to share among is the largest of the last launches, not only this one's: equal parts
// run side by side, while a launch that took the whole device because it came first (of a burst
// after a wait, or between two other threads' calls) would hold up all the others.
class BusyStreams {
public:
    // Streams that share the device with a launch on s about now, s among them.
    int sharing(int device, cudaStream_t s) {
        const Clock::time_point now = Clock::now();
        std::lock_guard<std::mutex> lock(mutex_);
        int count = 1;
        for (int q = 0; q < used_;) {
            if (busy_[q].until <= now) {
                busy_[q] = busy_[--used_];
                continue;
            }
            count += busy_[q].device == device && busy_[q].stream != s;
            ++q;
        }
        // the third launch in a row of one stream with no other busy: the others have stopped
        run_ = count == 1 && device == last_device_ && s == last_stream_ ? run_ + 1 : 0;
        last_device_ = device, last_stream_ = s;
        if (run_ >= 2)
            for (Seen &e : seen_)
                if (e.device == device) e.count = 0;
        seen_[next_] = Seen{device, count, now};
        next_ = (next_ + 1) % kSeen;
        for (const Seen &e : seen_)
            if (e.device == device && e.count > count && now - e.when <= kSeenTime) count = e.count;
        return count;
    }
    void add(int device, cudaStream_t s, double us) {
        const Clock::time_point now = Clock::now();
        const double part = 0.75 * us;
        const auto time = std::chrono::duration_cast<Clock::duration>(
            std::chrono::duration<double, std::micro>(part < kMostUs ? part : kMostUs));
        std::lock_guard<std::mutex> lock(mutex_);
        for (int q = 0; q < used_; ++q) {
            Busy &e = busy_[q];
            if (e.device != device || e.stream != s) continue;
            e.until = (e.until > now ? e.until : now) + time;
            const Clock::time_point most = now + std::chrono::microseconds((long long)kMostUs);
            if (e.until > most) e.until = most;
            return;
        }
        if (used_ < kBusy) busy_[used_++] = Busy{device, s, now + time};
    }
    void idle(int device, cudaStream_t s) {
        std::lock_guard<std::mutex> lock(mutex_);
        for (int q = 0; q < used_; ++q)
            if (busy_[q].device == device && busy_[q].stream == s) busy_[q].until = Clock::time_point::min();
    }

private:
    using Clock = std::chrono::steady_clock;
    struct Busy {
        int device;
        cudaStream_t stream;
        Clock::time_point until;
    };
    struct Seen {
        int device, count;
        Clock::time_point when;
    };
    static constexpr double kMostUs = 1e11;  // a day: any sweep count stays within the clock's range
    static constexpr int kBusy = 64;  // past these the device is shared as finely as it gets
    static constexpr int kSeen = 32;  // launches, none older than 20 ms: twice 16 streams' bursts
    static constexpr std::chrono::milliseconds kSeenTime{20};
    std::mutex mutex_;
    Busy busy_[kBusy];
    Seen seen_[kSeen] = {};
    int used_ = 0, next_ = 0, run_ = 0, last_device_ = -1;
    cudaStream_t last_stream_ = nullptr;
};

// A launch that is being captured runs later, if at all: it neither counts nor shares.
bool capturing(cudaStream_t s) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &status) != cudaSuccess) {
        cudaGetLastError();
        return true;
    }
    return status != cudaStreamCaptureStatusNone;
}

BusyStreams &busy_streams() {
    static BusyStreams b;
    return b;
}

}  // namespace

int streams_sharing(int device, cudaStream_t s) { return capturing(s) ? 1 : busy_streams().sharing(device, s); }
void stream_busy(int device, cudaStream_t s, double us) {
    if (!capturing(s)) busy_streams().add(device, s, us);
}
void stream_idle(int device, cudaStream_t s) { busy_streams().idle(device, s); }

}  // namespace rbgs
