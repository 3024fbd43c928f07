"""What a captured step leaves behind on the host is kept and set again as
one object: a context's list flags come back with its buffers.  Compiled
against the library's own headers; no GPU."""
import subprocess

from paper_2107_01276_gb300 import build as B

PROGRAM = r"""
#include "api.cuh"
int main() {
    sph_ctx c;
    double a = 0, b = 0;
    int64_t id = 0;
    c.f[F_X] = &a;
    c.falt[F_P0] = &b;
    c.id_alt = &id;
    c.tmask = 7;
    c.skin = 1.1f;
    c.rows = true;
    c.wall_lists_valid = true;
    sph_ctx::StepGraph g;
    g.after = c;                       // as a capture keeps it
    c.f[F_X] = c.falt[F_P0] = nullptr; // a right-hand side on plain lists
    c.id_alt = nullptr;
    c.tmask = 1;
    c.skin = 1.0f;
    c.rows = c.wall_lists_valid = false;
    c.n = 5;
    static_cast<StepHost &>(c) = g.after;   // as a replay sets it
    return !(c.f[F_X] == &a && c.falt[F_P0] == &b && c.id_alt == &id && c.tmask == 7 &&
             c.skin == 1.1f && c.rows && c.wall_lists_valid && c.n == 5);
}
"""


def test_a_replay_sets_everything_a_step_leaves_on_the_host(tmp_path):
    src, exe = tmp_path / "step_host.cu", tmp_path / "step_host"
    src.write_text(PROGRAM)
    r = subprocess.run([B._nvcc()] + B.ARCH + ["-std=c++17", "--extended-lambda", "-I", B.INCLUDE,
                                               "-I", B.CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)]).returncode == 0
