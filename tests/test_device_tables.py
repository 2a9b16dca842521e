"""Constant tables reach every device of the process, once each, whatever thread
creates a context there; a failed upload is reported and tried again.  (Host logic
with a fake upload: one GPU cannot show it.)"""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2308_01957_gb300", "csrc")

PROGRAM = r"""
#include "ap_device_once.cuh"
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#define CHECK(x) if (!(x)) { std::printf("failed: %s\n", #x); return 1; }
int main() {
  {
    ap::DeviceOnce once;
    int n[3] = {0, 0, 0};
    auto up = [&](int d) { return once.run(d, [&] { ++n[d]; return 0; }); };
    CHECK(up(0) == 0 && up(0) == 0 && up(2) == 0 && up(0) == 0 && up(1) == 0 && up(2) == 0);
    CHECK(n[0] == 1 && n[1] == 1 && n[2] == 1);
  }
  {
    ap::DeviceOnce once;
    int calls = 0;
    CHECK(once.run(0, [&] { ++calls; return 7; }) == 7);
    CHECK(once.run(0, [&] { ++calls; return 0; }) == 0);
    CHECK(once.run(0, [&] { ++calls; return 7; }) == 0);
    CHECK(calls == 2);
  }
  {
    ap::DeviceOnce once;
    std::atomic<int> calls{0}, finished{0}, early{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
      t.emplace_back([&] {
        once.run(0, [&] {
          ++calls;
          std::this_thread::sleep_for(std::chrono::milliseconds(50));
          ++finished;
          return 0;
        });
        if (finished != 1) ++early;
      });
    for (auto& x : t) x.join();
    CHECK(calls == 1 && early == 0);
  }
  std::puts("ok");
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


def test_tables_are_uploaded_per_device_and_checked():
    """The upload asks for the device, and every copy's result is looked at."""
    text = open(os.path.join(CSRC, "ap_render.cu")).read()
    body = text[text.index("int upload_tables(int device)"):]
    body = body[:body.index("\n}\n")]
    assert "once.run(device" in body
    copies = re.findall(r"^(.*)cudaMemcpyToSymbol\(", text, re.M)
    assert len(copies) == 5 and all(c.strip() for c in copies), copies
    api = open(os.path.join(CSRC, "ap_api.cu")).read()
    assert re.search(r"if \(upload_tables\(opt->device\) != 0\)", api)
