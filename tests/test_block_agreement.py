"""Threads of a block must agree before they meet at a barrier, and see what
another thread wrote only after one.  Device code runs here on the host, thread by thread, in
the order that shows a disagreement."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2301_04642_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

pytestmark = pytest.mark.skipif(
    not (shutil.which("g++") and os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h"))),
    reason="needs g++ and the CUDA headers")


def _host(name):
    """A source file with its inline PTX taken out."""
    s = open(os.path.join(CSRC, name)).read()
    return re.sub(r"\basm volatile\(.*?\);", ";", s, flags=re.S)


def _run(tmp_path, main, files=(), snippet=""):
    for f in ("fe_dev.cuh", "fe_kernels.cuh") + tuple(files):
        (tmp_path / f).write_text(_host(f))
    (tmp_path / "main.cpp").write_text('#include "cuda_emu.h"\n' + snippet + main)
    exe = str(tmp_path / "main")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I", str(tmp_path), "-I", os.path.join(ROOT, "tests", "emu"),
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.join(CUDA, "include"),
                        str(tmp_path / "main.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


LOAD_OP = r"""
int main() {
    fe::MmaProb pr;
    memset(&pr, 0, sizeof pr);
    pr.mats[2].master = reinterpret_cast<float *>(64);
    fe::ProdOp op;
    memset(&op, 0, sizeof op);
    op.nout = 2;
    op.part_out = 1;
    op.E1 = op.E2 = -1;
    op.inv = 0.5f;
    for (int o = 0; o < 3; ++o) op.out[o].a = 1.0f + o, op.out[o].mat = 2, op.out[o].flags = 3;
    fe::OpCache oc;
    memset(&oc, 0xee, sizeof oc);
    std::vector<int> order;
    for (int t = 31; t >= 0; --t) order.push_back(t);  // the lanes that write come last
    int bad = 0;
    const int stuck = emu::run(32, order, [&](int lane) {
        fe::load_op(oc, pr, op, lane);
        bad += !(oc.nout == 2 && oc.pout == 1 && oc.inv == 0.5f && oc.E2 == nullptr && oc.out[0].a == 1.0f &&
                 oc.out[1].a == 2.0f && oc.out[1].master == pr.mats[2].master);
    });
    printf("stuck %d, lanes with stale operands %d\n", stuck, bad);
    return stuck || bad;
}
"""


def test_operand_copy_is_seen_by_every_lane(tmp_path):
    """load_op: four lanes write the warp's copy of the step's operands, all read it."""
    s = _host("k_mma.cu")
    part = s[s.index("struct OutCache {"):s.index("// FP64 partials of a tile")]
    _run(tmp_path, LOAD_OP, snippet='#include "fe_dev.cuh"\n#include "fe_kernels.cuh"\nnamespace fe {\n' + part + "}\n")


SETUP = r"""
#include "k_control.cuh"
#include "k_control.cu"
static std::vector<int> reversed_warps(int n) {  // warp by warp, a warp's last lane first
    std::vector<int> o;
    for (int w = 0; w < n; w += 32)
        for (int t = w + 31; t >= w; --t) o.push_back(t);
    return o;
}
"""

CONTROL_KERNEL = SETUP + r"""
int main() {
    static fe::SolveState st, before;
    static double part[4 * 608];
    fe::MmaProb pr;
    memset(&pr, 0, sizeof pr);
    pr.st = &st;
    pr.part = part;
    pr.ntiles = 2;
    st.kind = fe::kTcSplit;  // a product that is still to run: k_control passes
    before = st;
    fe::StepFlags fl{};
    fl.controlled = 1;
    fe::DevCtl ctl{};
    gridDim.x = 1;
    const int stuck = emu::run(256, reversed_warps(256),
                               [&](int) { fe::k_control(&pr, 1, &ctl, &fl, 0, 0, 1); });
    const int changed = memcmp(&st, &before, sizeof st) != 0;
    printf("stuck %d, state changed %d, steps %u, controls %u\n", stuck, changed, fl.n_steps, fl.n_ctl);
    return stuck || changed || fl.n_steps != 0 || fl.n_ctl != 1 || fl.controlled != 0;
}
"""


def test_control_kernel_takes_one_decision_per_block(tmp_path):
    """k_control clears the flags it acts on; a late warp must not act on the cleared ones."""
    _run(tmp_path, CONTROL_KERNEL, files=("k_control.cuh", "k_control.cu"))


CONTROL_STEP = SETUP + r"""
int main(int argc, char **argv) {
    int bad = 0;
    // a bounded wait of another block runs out after the k-th thread had its turn
    for (int k : {0, 31, 127, 254}) {
        static fe::SolveState st;
        static double part[4 * 608];
        memset(&st, 0, sizeof st);
        fe::MmaProb pr;
        memset(&pr, 0, sizeof pr);
        pr.st = &st;
        pr.part = part;
        st.n = 2;
        st.bad_input = 1;  // ends the problem with FE_EINVAL when the step is taken
        fe::DevCtl ctl{};
        fe::ControlSmem sh;
        int taken = 0;
        std::vector<int> order;
        for (int t = 0; t < 256; ++t) order.push_back(t);
        const int stuck = emu::run(256, order,
                                   [&](int t) { taken += fe::control_one(pr, &ctl, &sh, t, [] { emu::meet(0); }); },
                                   [&](int done) { if (done == k) ctl.err = fe::kErrTimeoutGrid; });
        printf("after thread %d: stuck %d, taken by %d, status %d\n", k, stuck, taken, st.status);
        bad += stuck || taken != 256 || !st.done || (st.status != -1 && st.status != -4);
    }
    return bad;
}
"""


def test_control_step_takes_one_decision_per_block(tmp_path):
    """control_one inside a launch whose other blocks still run: an error recorded
    between two threads' reads must not leave some of them at a barrier."""
    _run(tmp_path, CONTROL_STEP, files=("k_control.cuh", "k_control.cu"))


COEFFICIENTS = SETUP + r"""
int main() {
    const double in = 1.0, tiny = 0x1p-126;
    std::vector<double> xs = {0.0, -0.0, in, -in, 0x1.0000010000000p0, 0x1.0000030000000p0, 0x1.fffffeffffffep0,
                              tiny, 0.75 * tiny, -tiny / 1024, 0x1p-149, 0x1p-150, 0x1.8p-150, 0x1p-151, 0x1p-1074,
                              0x1.fffffefffffffp127, 0x1.ffffffp127, -0x1p128, 0x1p1023, INFINITY, -INFINITY, NAN};
    for (int e = -152; e < 129; ++e) xs.push_back(std::ldexp(1.2345678901234567, e)), xs.push_back(-std::ldexp(1.9999999, e));
    int bad = 0;
    auto same = [&](float got, double x, const char *what) {
        const float want = static_cast<float>(x);
        if (std::isnan(want) ? std::isnan(got) : memcmp(&got, &want, 4) == 0) return;
        printf("%s %a: %a, not %a\n", what, x, got, want);
        ++bad;
    };
    for (double x : xs) {
        fe::OutSpec o;
        fe::set_out(o, 0, 0, x, x, x, 0.0, 1.0);
        same(o.a, x, "a"), same(o.b1, x, "b1"), same(o.b2, x, "b2");
        fe::out_d(o, 0, 0, x, 1.0);
        same(o.a, x, "diagonal a");
        fe::set_e(o, 0, x, x, x, 0, x, x, x);
        same(o.b1, x, "e b1"), same(o.g1r, x, "g1r"), same(o.g1c, x, "g1c");
        same(o.b2, x, "e b2"), same(o.g2r, x, "g2r"), same(o.g2c, x, "g2c");
    }
    return bad != 0;
}
"""


def test_coefficients_are_the_nearest_fp32(tmp_path):
    """The control step's coefficients over all of FP32: subnormals, overflow, NaN."""
    _run(tmp_path, COEFFICIENTS, files=("k_control.cuh", "k_control.cu"))
