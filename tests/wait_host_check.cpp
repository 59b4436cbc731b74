// Host build of the device code's bounded wait: two threads stand in for two warps of a block.
//   case "complete": both parties arrive at a counter that expects two arrivals -> both waits return true.
//   case "withheld": one arrival never comes -> the first waiter runs out of time, returns false and raises the
//                    abort word; the second waiter sees the abort word and returns false without waiting out its
//                    own limit.
// Prints one line per case: <case> <result of waiter 0> <result of waiter 1> <abort word> <elapsed ms of waiter 1>.
//
// Then four threads stand in for the lanes of one warp, which see the same memory at slightly different times:
//   case "lanes_<what>":       a wait with the warp's vote
//   case "lanes_<what>_alone": the same schedule with every lane deciding for itself (what the vote is for)
// where <what> is "phase" (the phase completes for lanes 0 and 1 at the poll at which lanes 2 and 3 find the abort word set) or
// "clock" (lane 3's clock is past the limit while the phase completes for the others at their next poll).
// Prints <case> <results of the lanes 0 1 2 3> <abort word> <lanes that were left behind in a vote>.
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <thread>

#include "../paper_2503_05931_b200/csrc/bounded_wait.h"

static long long now_us()
{
    return std::chrono::duration_cast<std::chrono::microseconds>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

static bool alone(bool p) { return p; }

static void run_case(const char *name, bool second_arrives)
{
    std::atomic<int> arrivals{0};
    volatile int abort_word = 0;
    bool r0 = true, r1 = true;
    long long t1 = 0;
    auto ready = [&] { return arrivals.load(std::memory_order_acquire) >= 2; };
    std::thread a([&] {
        arrivals.fetch_add(1, std::memory_order_release);
        r0 = aed::bounded_poll(ready, now_us, 50 * 1000, &abort_word, alone);          // 50 ms
    });
    std::thread b([&] {
        if (second_arrives) arrivals.fetch_add(1, std::memory_order_release);
        const long long s = now_us();
        r1 = aed::bounded_poll(ready, now_us, 5 * 1000 * 1000, &abort_word, alone);    // 5 s: must end through the abort word
        t1 = now_us() - s;
    });
    a.join();
    b.join();
    std::printf("%s %d %d %d %lld\n", name, (int)r0, (int)r1, (int)abort_word, t1 / 1000);
}

// A vote of kLanes threads: true in all of them if p was true in all.  A lane whose companions do not come within a second is
// counted as left behind (on the device it would hang).
constexpr int kLanes = 4;
struct Vote {
    std::mutex m;
    std::condition_variable cv;
    int arrived = 0, round = 0, left_behind = 0;
    bool conj = true, result[2] = {true, true};
    bool all(bool p)
    {
        std::unique_lock<std::mutex> lock(m);
        const int mine = round;
        conj = conj && p;
        if (++arrived == kLanes) {
            result[mine & 1] = conj;
            conj = true;
            arrived = 0;
            ++round;
            cv.notify_all();
            return result[mine & 1];
        }
        if (!cv.wait_for(lock, std::chrono::seconds(1), [&] { return round != mine; })) { ++left_behind; return p; }
        return result[mine & 1];
    }
};

static void run_lanes(const char *what, bool voted)
{
    const bool by_clock = !std::strcmp(what, "clock");
    Vote vote;
    volatile int abort_word = 0;
    bool result[kLanes];
    std::thread lanes[kLanes];
    for (int l = 0; l < kLanes; ++l)
        lanes[l] = std::thread([&, l] {
            int polls = 0, reads = 0;
            volatile int own_word = 0;              // the abort word as this lane sees it
            auto ready = [&] {
                ++polls;
                if (by_clock) return polls >= 3 && l != 3;
                if (polls == 3 && l >= 2) own_word = 1;
                return polls >= 3 && l < 2;
            };
            auto now = [&] { return by_clock && l == 3 && reads++ > 0 ? 1000ll : 0ll; };
            if (voted) result[l] = aed::bounded_poll(ready, now, 100, &own_word, [&](bool p) { return vote.all(p); });
            else result[l] = aed::bounded_poll(ready, now, 100, &own_word, alone);
            if (own_word) abort_word = 1;
        });
    for (auto &t : lanes) t.join();
    const std::string name = std::string("lanes_") + what + (voted ? "" : "_alone");
    std::printf("%s %d %d %d %d %d %d\n", name.c_str(), (int)result[0], (int)result[1], (int)result[2], (int)result[3], (int)abort_word, vote.left_behind);
}

int main()
{
    run_case("complete", true);
    run_case("withheld", false);
    for (const char *what : {"phase", "clock"}) {
        run_lanes(what, true);
        run_lanes(what, false);
    }
    return 0;
}
