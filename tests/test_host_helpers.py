"""Host helpers of the library (csrc/dw_host.cuh), compiled by themselves; no GPU."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0706_2298_gb300", "csrc")


def run(tmp_path, body):
    src = tmp_path / "t.cpp"
    src.write_text('#include "dw_host.cuh"\n#include <cstdio>\n#include <thread>\n#include <vector>\n'
                   '#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); return 1; } } while (0)\n'
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I" + CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_once_per_device(tmp_path):
    """A limit set on one device is not taken for set on another, and a failure is tried again."""
    run(tmp_path, """
      DeviceOnce once;
      int calls = 0, status = 0;
      auto f = [&] { ++calls; return status; };
      CHECK(once(0, f) == 0 && calls == 1);
      CHECK(once(0, f) == 0 && calls == 1);
      CHECK(once(1, f) == 0 && calls == 2);
      CHECK(once(63, f) == 0 && once(64, f) == 0 && once(128, f) == 0 && once(255, f) == 0 && calls == 6);
      CHECK(once(63, f) == 0 && once(64, f) == 0 && once(128, f) == 0 && once(255, f) == 0 && calls == 6);
      status = 2;
      CHECK(once(2, f) == 2 && calls == 7);
      CHECK(once(2, f) == 2 && calls == 8);
      CHECK(once(0, f) == 0 && calls == 8);
      status = 0;
      CHECK(once(2, f) == 0 && calls == 9);
      CHECK(once(2, f) == 0 && calls == 9);
      CHECK(once(256, f) == 0 && once(256, f) == 0 && once(-1, f) == 0 && calls == 12);
      DeviceOnce shared;
      std::atomic<int> n{0};
      std::vector<std::thread> ts;
      for (int t = 0; t < 8; ++t) ts.emplace_back([&] { for (int d = 0; d < 256; ++d) shared(d, [&] { ++n; return 0; }); });
      for (auto& t : ts) t.join();
      const int before = n;
      CHECK(before >= 256);
      for (int d = 0; d < 256; ++d) shared(d, [&] { ++n; return 0; });
      CHECK(n == before);
    """)


def test_group_fits_the_memory(tmp_path):
    """A group that memory cannot be had for is halved down to one; other failures and success end the search."""
    run(tmp_path, """
      std::vector<int> tried;
      int room = 0, n = 0;
      auto alloc = [&](int k) { tried.push_back(k); return k <= room ? 0 : 2; };
      n = 8; room = 8;
      CHECK(fit_group(n, 2, alloc) == 0 && n == 8 && tried == std::vector<int>({8}));
      tried.clear(); n = 8; room = 3;
      CHECK(fit_group(n, 2, alloc) == 0 && n == 2 && tried == std::vector<int>({8, 4, 2}));
      tried.clear(); n = 7; room = 1;
      CHECK(fit_group(n, 2, alloc) == 0 && n == 1 && tried == std::vector<int>({7, 4, 2, 1}));
      tried.clear(); n = 5; room = 0;
      CHECK(fit_group(n, 2, alloc) == 2 && n == 1 && tried == std::vector<int>({5, 3, 2, 1}));
      tried.clear(); n = 1; room = 0;
      CHECK(fit_group(n, 2, alloc) == 2 && tried == std::vector<int>({1}));
      tried.clear(); n = 6;
      CHECK(fit_group(n, 2, [&](int k) { tried.push_back(k); return 77; }) == 77 && tried == std::vector<int>({6}));
    """)


def test_kernel_limits_go_through_it():
    """No launch keeps the state of its kernel's shared-memory limit for the process as a whole."""
    for name in ("dw_ptnet.cu", "dw_sap.cu"):
        assert "cudaFuncSetAttribute" not in open(os.path.join(CSRC, name)).read(), name
