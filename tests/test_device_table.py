"""The library's per-device set-up as host code alone: every device is set up once, also when a second one is used after the
first; a set-up that failed is tried again; an ordinal outside the table is refused; threads that ask at the same time see one
set-up."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2311_04951_b200", "csrc")
PROGRAM = r"""
#include <thread>
#include <vector>
#include "device_table.h"
#define CHECK(x) do { if (!(x)) return __LINE__; } while (0)
struct Info { int num_sms; };
int main() {
    ssd::DeviceTable<Info> t;
    int calls[3] = {0, 0, 0};
    auto ask = [&](int dev, const Info **out) {
        return t.get(dev, [&](Info &i) { i.num_sms = 100 + dev; return ++calls[dev] == 1 && dev == 2 ? 7 : 0; }, out);
    };
    const Info *a, *b, *c;
    CHECK(ask(0, &a) == 0 && ask(1, &b) == 0 && ask(0, &a) == 0 && ask(1, &b) == 0);
    CHECK(calls[0] == 1 && calls[1] == 1 && a->num_sms == 100 && b->num_sms == 101);
    CHECK(ask(2, &c) == 7 && ask(2, &c) == 0 && ask(2, &c) == 0 && calls[2] == 2 && c->num_sms == 102);
    CHECK(ask(-1, &a) == -1 && ask(ssd::DeviceTable<Info>::kMax, &a) == -1);
    ssd::DeviceTable<Info> u;
    std::atomic<int> set_up{0}, good{0};
    std::vector<std::thread> th;
    for (int i = 0; i < 8; ++i)
        th.emplace_back([&] {
            const Info *x;
            if (u.get(5, [&](Info &v) { ++set_up; v.num_sms = 9; return 0; }, &x) == 0 && x->num_sms == 9) ++good;
        });
    for (auto &x : th) x.join();
    CHECK(set_up == 1 && good == 8);
    return 0;
}
"""


def test_every_device_is_set_up_once(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-o", str(exe), str(src)])
    subprocess.check_call([str(exe)])
