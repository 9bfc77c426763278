"""Who gets the SMs (SmTokens, csrc/resident_plan.cpp), on the CPU with 152 SMs."""
import os
import shutil
import subprocess

import pytest

from tests.conftest import ROOT

SOURCE = r'''
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "resident_plan.hpp"
using namespace lpop;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  {  // plans that fit side by side; a third that does not is stepped, and the crowd begins beyond eight GPUs' worth
    SmTokens t(152);
    t.announce(100, false);
    t.announce(52, false);
    CHECK(t.acquire_resident(100) && t.acquire_resident(52));
    t.announce(152, false);
    t.announce(152, false);
    CHECK(!t.acquire_resident(152) && !t.acquire_resident(20));
    CHECK(!t.crowded());
    t.announce(8 * 152, false);
    CHECK(t.crowded());
    t.withdraw(8 * 152, false);
    t.release(100);
    t.release(52);
    CHECK(!t.acquire_resident(152));  // four of them still
    CHECK(t.acquire_resident(19));    // a small one
    t.release(19);
  }
  {  // two that do not fit take turns
    SmTokens t(152);
    t.announce(152, false);
    t.announce(120, false);
    CHECK(t.acquire_resident(152));
    std::atomic<bool> got{false};
    std::thread other([&] { got = t.acquire_resident(120); });
    std::this_thread::sleep_for(std::chrono::milliseconds(50));
    CHECK(!got);
    t.release(152);
    other.join();
    CHECK(got);
  }
  {  // a round: beside it what is free, and nobody waits for its end
    SmTokens t(152);
    t.announce(3, true);
    CHECK(t.acquire(2, 3) == 3);
    t.announce(120, false);
    CHECK(t.acquire_resident(120));
    t.release(120);
    t.withdraw(120, false);
    t.announce(152, false);
    CHECK(!t.acquire_resident(152));
    t.announce(12, false);
    CHECK(t.acquire_resident(12));
    t.release(12);
    CHECK(t.acquire(2, 149) == 149);  // (another round takes the rest)
    CHECK(!t.acquire_resident(12));
    t.release(149);
    t.release(3);
    t.withdraw(3, true);
    t.withdraw(12, false);
    CHECK(t.acquire_resident(152));
    t.release(152);
  }
  {  // many threads, periods and rounds: everyone ends, and no more than the SMs are ever held
    SmTokens t(152);
    std::atomic<int> held{0}, most{0}, periods{0};
    std::vector<std::thread> pool;
    const int size[] = {152, 120, 43, 12, 5, 152, 76, 19};
    auto hold = [&](int n) {
      const int h = held += n;
      int m = most;
      while (m < h && !most.compare_exchange_weak(m, h)) {}
      std::this_thread::sleep_for(std::chrono::microseconds(20));
      held -= n;
    };
    for (int k = 0; k < 8; ++k)
      pool.emplace_back([&, k] {
        t.announce(size[k], false);
        for (int i = 0; i < 300; ++i) {
          if (!t.acquire_resident(size[k])) continue;
          hold(size[k]);
          t.release(size[k]);
          ++periods;
        }
        t.withdraw(size[k], false);
      });
    pool.emplace_back([&] {
      for (int i = 0; i < 200; ++i) {
        t.announce(100, true);
        const int got = t.acquire(8, 100);
        hold(got);
        t.release(got);
        t.withdraw(100, true);
      }
    });
    for (std::thread& p : pool) p.join();
    CHECK(most <= 152 && held == 0 && periods > 0);
    CHECK(t.acquire(152, 152) == 152);
  }
  std::printf("ok\n");
}
'''


def test_tokens(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    csrc = os.path.join(ROOT, "paper_2506_17650_gb300", "csrc")
    src, exe = tmp_path / "tokens.cpp", str(tmp_path / "tokens")
    src.write_text(SOURCE)
    subprocess.run([gxx, "-O1", "-std=c++17", "-pthread", "-I", csrc, str(src), os.path.join(csrc, "resident_plan.cpp"),
                    "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout
