"""Properties of the kernel sources that no run can show (CPU only)."""
import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_08733_gb300", "csrc")


def _sources(*ext):
    return {os.path.basename(f): open(f).read() for e in ext for f in glob.glob(os.path.join(CSRC, "*" + e))}


def test_no_restrict_name_for_a_buffer_the_kernel_writes():
    """A kernel that reads the residuals (or the auxiliaries' residuals) also writes them, and
    what it reads may be what the launch before it still writes: no name of such a
    buffer may promise the compiler that nothing else touches it."""
    for name, text in _sources(".cuh").items():
        bound = re.findall(r"__restrict__\s+\w+\s*=\s*static_cast<[^>]*>\(prm\.(\w+)\)", text)
        assert not bound, (name, bound)


def test_launchers_opt_in_to_shared_memory_on_each_device(tmp_path):
    """The opt-in to more than 48 KB of shared memory holds per device: a plan on a second device
    needs it too (OncePerDevice), and no launcher remembers it in a plain flag."""
    for name, text in _sources(".cuh", ".cu").items():
        assert not re.search(r"static\s+bool\s+\w+\s*=", text), name
        if "cudaFuncAttributeMaxDynamicSharedMemorySize" in text:
            assert "OncePerDevice" in text, name
    src = tmp_path / "once.cpp"
    src.write_text("""
#include <cstdio>
#include <thread>
#include <vector>
#include "dgm_once.h"
int main() {
    dgm::OncePerDevice o;
    int calls = 0;
    auto ok = [&] { ++calls; return true; };
    auto bad = [&] { ++calls; return false; };
    if (!o.ensure(0, ok) || !o.ensure(0, ok) || calls != 1) return 1;
    if (!o.ensure(1, ok) || calls != 2) return 2;                 // another device
    if (o.ensure(2, bad) || !o.ensure(2, ok) || calls != 4) return 3;   // again after a failure
    if (!o.ensure(64, ok) || !o.ensure(64, ok) || calls != 6) return 4;  // past what it remembers
    if (!o.ensure(63, ok) || !o.ensure(63, ok) || calls != 7) return 5;
    dgm::OncePerDevice m;
    std::atomic<int> n{0};
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i)
        t.emplace_back([&, i] { for (int d = 0; d < 8; ++d) m.ensure((d + i) % 8, [&] { ++n; return true; }); });
    for (auto& x : t) x.join();
    const int first = n;
    for (int d = 0; d < 8; ++d) m.ensure(d, [&] { ++n; return true; });
    return n == first && first >= 8 ? 0 : 6;
}
""")
    exe = str(tmp_path / "once")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_bench_names_the_kernel_it_times(tmp_path):
    """Counters of one kernel are not reported beside another."""
    import sys
    sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    import bench
    name = bench.kernel_name(0, 196608, 20, 1)
    assert name == "tang_kernel<3,float,32,4,LSRK,unsigned int>"
    assert bench.kernel_name(0, 1296, 20, 1).startswith("tang_kernel<3,float,32,8,")
    assert bench.kernel_name(5, 196608, 20, 1).startswith("stage_kernel<")
    f = tmp_path / "p.md"
    f.write_text("traffic_bytes_per_element_stage variant=0 tile_groups=6 loads=bulk: 2034\n"
                 "traffic_bytes_per_element_stage kernel=tang_kernel variant=0 tile_groups=12 loads=bulk: 1800\n")
    assert bench.profiled_traffic(str(f), 0, 6, 10, "bulk", name) is None
    assert bench.profiled_traffic(str(f), 0, 12, 10, "bulk", name) == 18000
    assert bench.profiled_traffic(str(f), 0, 12, 10, "bulk", "stage_kernel<3>") is None
    committed = os.path.join(os.path.dirname(CSRC), "..", "profiles", bench.TRAFFIC_PROFILE)
    assert bench.profiled_traffic(committed, 0, 6, 196608, "bulk", name) is not None


def test_generated_operators_belong_to_the_machine(monkeypatch):
    """A header generated on one architecture is not taken on another, whose compiler rounds the
    literals differently in the last bit."""
    import importlib
    import platform
    from paper_2002_08733_gb300 import build as B
    here = B.GEN_HEADER
    try:
        monkeypatch.setattr(platform, "machine", lambda: "another")
        assert importlib.reload(B).GEN_HEADER != here
    finally:
        monkeypatch.undo()
        importlib.reload(B)
    assert B.GEN_HEADER == here
