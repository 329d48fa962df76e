"""Host state of a device (csrc/device_once.h): a kernel's dynamic shared memory limit holds for the device on which it
was set, so it is set once on each of them, again after a failure, and the SM count is looked up per device.
The second device is a fake here. No launch may keep such a setting in a process-wide flag, which leaves a second
device's kernels at 48 KB."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_05800_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    chemgb::DeviceOnce once;
    int limit[66] = {0}, calls = 0;
    auto launch = [&](int dev, int rc = 0) { return once.run(dev, [&] { ++calls; if (!rc) limit[dev] = 230000; return rc; }); };
    CHECK(launch(0) == 0 && launch(0) == 0 && calls == 1);
    CHECK(launch(1, 7) == 7 && limit[1] == 0);            // refused: set again by the next launch
    CHECK(launch(1) == 0 && limit[1] == 230000 && calls == 3 && launch(1) == 0 && calls == 3);
    CHECK(launch(63) == 0 && limit[63] == 230000 && launch(63) == 0 && calls == 4);
    CHECK(launch(64) == 0 && launch(64) == 0 && calls == 6);
    chemgb::DeviceInt sms;
    std::vector<std::thread> th;
    int bad = 0;
    for (int t = 0; t < 8; ++t)
        th.emplace_back([&] { for (int d = 0; d < 66; ++d) if (sms.value(d, [d] { return 100 + d; }) != 100 + d) bad = 1; });
    for (auto &t : th) t.join();
    CHECK(!bad && sms.value(1, [] { return 5; }) == 101);
    std::printf("ok\n");
}
"""


def test_state_is_kept_per_device(tmp_path):
    src, exe = tmp_path / "once.cc", tmp_path / "once"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, str(src), "-o", str(exe), "-pthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_no_process_wide_flag_beside_a_device_setting():
    for f in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")):
        text = open(f).read()
        found = re.search(r"static\s+(bool|size_t|int)\s+(configured|sms)\b", text)
        assert not found, (os.path.basename(f), found.group(0))
        # the one place that sets the limit: anywhere else it would be the last launch's size for all threads
        sets = len(re.findall(r"cudaFuncSetAttribute", text))
        assert sets == (1 if f.endswith("internal.cuh") else 0), os.path.basename(f)
