"""Host-side answers shared by the handles of all threads (csrc/per_device.h), compiled for the CPU."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_0748_gb300", "csrc")


def _run(tmp_path, body, *flags):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include <thread>\n#include <vector>\n#include "per_device.h"\n' + body)
    made = subprocess.run(["g++", "-std=c++17", "-g", "-O1", "-pthread", "-I" + CSRC, *flags, str(src), "-o", str(exe)],
                          capture_output=True, text=True)
    if made.returncode and flags:
        pytest.skip("no sanitizer runtime: " + made.stderr[-200:])
    assert made.returncode == 0, made.stderr
    return subprocess.run([str(exe)], capture_output=True, text=True)


def test_threads_share_it_without_a_data_race(tmp_path):
    body = """
int main() {
  static kb::PerDevice known;
  int bad = 0;
  std::vector<std::thread> t;
  std::vector<int> got(8 * 1000);
  for (int i = 0; i < 8; ++i)
    t.emplace_back([&got, i] {
      for (int r = 0; r < 1000; ++r) got[i * 1000 + r] = known.get(r % 70, [&] { return 1 + r % 70; });
    });
  for (auto& x : t) x.join();
  for (int j = 0; j < 8000; ++j) bad += got[j] != 1 + j % 1000 % 70;
  return bad ? 1 : 0;
}
"""
    plain = _run(tmp_path, body)
    assert plain.returncode == 0, plain.stderr
    checked = _run(tmp_path, body, "-fsanitize=thread")
    if "unexpected memory mapping" in checked.stderr:
        pytest.skip("the sanitizer cannot map its memory here")
    assert checked.returncode == 0 and "data race" not in checked.stderr, checked.stderr[-2000:]


def test_a_failed_query_is_asked_again(tmp_path):
    """A query fails by returning 0; neither that nor a negative answer is kept."""
    body = """
int main() {
  static kb::PerDevice known;
  int asked = 0;
  const int answers[] = {0, -1, 5, 7};
  auto query = [&] { return answers[asked++]; };
  const bool ok = known.get(3, query) == 0 && known.get(3, query) == -1 && known.get(3, query) == 5 &&
                  known.get(3, query) == 5 && asked == 3 && known.get(2, query) == 7;
  return ok ? 0 : 1;
}
"""
    assert _run(tmp_path, body).returncode == 0
