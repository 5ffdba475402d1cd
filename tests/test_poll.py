"""The wait for counts that a kernel writes to host memory (cs_poll.cuh):
host code, compiled and run on the CPU with a stand-in for the stream."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "cs_poll.cuh"
int main() {
    uint32_t flag = 6;
    int waits = 0;
    auto done = [&] { ++waits; return true; };
    auto writes = [&] { ++waits; flag = 7; return true; };
    auto fails = [&] { ++waits; flag = 7; return false; };
    auto report = [&](cs::Arrival a) { std::printf("%d %d ", (int)a, waits); };
    // never written, although the stream has finished
    report(cs::wait_for(&flag, 7u, 100, done));
    // written while the stream was waited for
    report(cs::wait_for(&flag, 7u, 100, writes));
    // there at once: the stream is not waited for
    report(cs::wait_for(&flag, 7u, 100, done));
    flag = 6;
    report(cs::wait_for(&flag, 7u, 0, fails));
}
"""


def test_counts_that_never_come_are_an_error(tmp_path):
    src, exe = tmp_path / "poll.cpp", tmp_path / "poll"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2501_17792_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    there, missing, failed = "0", "1", "2"
    assert out == [missing, "1", there, "2", there, "2", failed, "3"]


@pytest.mark.gpu
def test_a_frame_behind_work_that_outlasts_the_polls():
    """The counts come some tens of milliseconds late: the host's polls run
    out and it waits for the stream.  Same image."""
    torch = pytest.importorskip("torch")
    from paper_2501_17792_gb300 import binding
    from paper_2501_17792_gb300 import scene as S
    sc = S.crowd(n_templates=1, n_gauss=300, sh_degree=0, cols=3, rows=2, width=96, height=64)
    st = torch.cuda.Stream()
    r = binding.Renderer(device=0, stream=st)
    r.upload_templates(sc.templates)
    r.set_lod(sc.lod)
    r.set_instances(sc.instances.template_id, sc.instances.root, sc.instances.pose)
    img = []
    for busy in (False, True):
        out = torch.empty((64, 96, 4), device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.stream(st):
            if busy:
                torch.cuda._sleep(200_000_000)  # clocks: a tenth of a second
            r.render(sc.camera, out=out)
        torch.cuda.synchronize()
        img.append(out)
    assert float(img[0][..., 3].max()) > 0.5 and torch.equal(img[0], img[1])
    r.close()
