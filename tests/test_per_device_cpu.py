"""The values that the library keeps per device (csrc/per_device.h), on the
host: a launch attribute set on one device is set on the next one too.  The
header is compiled as it is, with a stand-in for the CUDA call."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2412_04787_gb300", "csrc")


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "per_device.h"\n#include <cstdio>\n#include <thread>\n#include <vector>\n'
                   + body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


def test_each_device_is_set_once(tmp_path):
    """One call per device, a failed one is tried again, devices beyond the
    table are set on each call."""
    out = _run(tmp_path, """
      int main() {
        static dqt::PerDevice p;
        int calls = 0, v = 0;
        auto set = [&](int& x) { ++calls; x = 1; return true; };
        auto fail = [&](int&) { ++calls; return false; };
        for (int dev : {0, 0, 1, 1, 0, 63, 63}) if (!p.get(dev, v, set) || v != 1) return 1;
        std::printf("%d ", calls);
        if (p.get(2, v, fail) || !p.get(2, v, set)) return 1;
        std::printf("%d ", calls);
        for (int i = 0; i < 2; ++i) if (!p.get(64, v, set)) return 1;
        std::printf("%d", calls);
      }""")
    assert out == ["3", "5", "7"]


def test_threads_see_whole_values(tmp_path):
    """A query that writes its result in two steps: no thread reads the first."""
    out = _run(tmp_path, """
      int main() {
        int bad = 0;
        for (int round = 0; round < 50; ++round) {
          dqt::PerDevice p;
          std::atomic<int> wrong{0}, ready{0};
          std::vector<std::thread> ts;
          for (int i = 0; i < 4; ++i)
            ts.emplace_back([&] {
              ++ready;
              while (ready.load() < 4) std::this_thread::yield();
              int v = 0;
              for (int k = 0; k < 20; ++k)
                if (!p.get(0, v, [](int& x) { x = -1; std::this_thread::yield(); x = 7; return true; }) || v != 7) ++wrong;
            });
          for (auto& t : ts) t.join();
          bad += wrong;
        }
        std::printf("%d", bad);
      }""")
    assert out == ["0"]


def test_the_norms_occupancy_is_not_queried_into_shared_memory():
    src = open(os.path.join(CSRC, "decoder_ops.cu")).read()
    assert "static int occ" not in src


def test_launch_attributes_of_the_norm_are_per_device():
    """The norm's backward needs a raised shared-memory limit, which belongs to
    a device: no process-wide flag stands before that call."""
    src = open(os.path.join(CSRC, "decoder_ops.cu")).read()
    body = src[src.index("static int rms_bwd_launch"):]
    body = body[:body.index("\n}\n")]
    assert "static bool" not in body and "PerDevice" in body
