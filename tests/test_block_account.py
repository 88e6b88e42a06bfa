"""The device's blocks divided among concurrent calls, on the CPU (im_host.h):
two servers' queries and plain contexts' calls take from one account, so that
what they hold together never exceeds the device, and every waiting call gets
its share; and the wait limit of a phase on a share."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_14047_gb300", "csrc")

PROGRAM = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
#include "im_host.h"

static std::atomic<int> in_flight[2], bad{0};  // per device

static void hold(int device, int total, int h) {
    if (h < 1 || in_flight[device].fetch_add(h) + h > total) bad = 1;
}

// A caller of `calls` calls: a server's worker or a plain context; seeds
// of a selection (0: a step-level call, one phase).
static void caller(int device, int total, int calls, unsigned seed) {
    for (int i = 0; i < calls; ++i) {
        imi::BlockAccount* a = imi::account_of(device, total);  // as each call asks for it
        a->enter();
        if (rand_r(&seed) % 8 == 0) { a->leave(0); continue; }  // it fails before its first phase
        if (rand_r(&seed) % 4 == 0) std::this_thread::yield();
        int h = a->take();
        hold(device, total, h);
        for (int k = rand_r(&seed) % 6; k > 0; --k) {
            if (rand_r(&seed) % 2) std::this_thread::yield();
            in_flight[device] -= h;  // nothing of it is in flight
            h = a->adjust(h);
            hold(device, total, h);
        }
        in_flight[device] -= h;
        a->leave(h);
    }
}

int main(int argc, char** argv) {
    const int total = atoi(argv[1]), threads = atoi(argv[2]);
    // every server and every context of a device has the same account
    if (imi::account_of(0, total) != imi::account_of(0, total) || imi::account_of(0, total) == imi::account_of(1, total))
        return puts("not one account a device"), 1;
    std::vector<std::thread> t;
    for (int i = 0; i < threads; ++i) t.emplace_back(caller, i % 8 == 7 ? 1 : 0, total, 400, i + 1);
    for (auto& x : t) x.join();
    if (bad) return puts("more blocks in flight than the device holds"), 1;
    // all of them are back: one caller alone holds the device
    imi::BlockAccount* a = imi::account_of(0, total);
    a->enter();
    int h = a->take();
    if (h != total || a->total() != total) return puts("blocks were lost"), 1;
    // a second one waits until the first comes down, then both have half
    std::atomic<int> got{0};
    a->enter();
    std::thread second([&] { got = a->take(); });
    std::this_thread::sleep_for(std::chrono::milliseconds(50));
    if (got != 0) return puts("a share out of nothing"), 1;
    h = a->adjust(h);
    second.join();
    if (total > 1 && (h != total / 2 || got != total / 2)) return puts("uneven shares"), 1;
    a->leave(got);
    h = a->adjust(h);
    if (h != total) return puts("a share not taken up"), 1;
    a->leave(h);
    puts("ok");
    return 0;
}
"""


@pytest.mark.parametrize("total,threads", [(304, 16), (304, 3), (7, 24), (2, 24)])
def test_callers_of_a_device_never_hold_more_than_it_has(tmp_path, total, threads):
    assert _run(tmp_path, PROGRAM, total, threads) == ["ok"]


LIMITS = r"""
#include <cstdio>
#include "im_host.h"
int main() {
    const unsigned long long ns[] = {0, 1, 2000000000ull, ~0ull / 2, ~0ull};
    for (unsigned long long n : ns)
        for (int blocks : {304, 303, 152, 101, 7, 4, 1}) printf("%llu\n", (unsigned long long)imi::wait_limit(n, 304, blocks));
}
"""


def test_wait_limit_grows_with_what_a_share_lacks(tmp_path):
    got = iter(int(x) for x in _run(tmp_path, LIMITS))
    for ns in (0, 1, 2 * 10**9, (2**64 - 1) // 2, 2**64 - 1):
        for blocks in (304, 303, 152, 101, 7, 4, 1):
            assert next(got) == min(2**64 - 1, ns * -(-304 // blocks)), (ns, blocks)


def _run(tmp_path, program, *args):
    src = tmp_path / "account.cpp"
    src.write_text(program)
    exe = tmp_path / "account"
    try:
        r = subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                           capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("no C++ compiler")
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
    return r.stdout.split()
