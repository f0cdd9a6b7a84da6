"""The host rules that choose a sweep kernel, without a GPU: a small program
linked against the library prints what the rules say for given sizes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OPTIN = 227 << 10

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "spvar_internal.h"
using namespace spvar;
int main(int argc, char **argv)
{
    auto arg = [&](int i) { return i < argc ? std::atoi(argv[i]) : 0; };
    if (!std::strcmp(argv[1], "request")) {
        // block, n, quads, degree: taken as a request, shared memory of the launch, second table
        const QuadLayout l = pm1q_layout(arg(2), arg(3), arg(4), arg(5));
        std::printf("%d %zu %d\n", (int)pm1q_request_ok(arg(2), arg(3), arg(4), arg(5), kSmemOptin), l.bytes + l.stat,
                    (int)l.tabs);
    }
    if (!std::strcmp(argv[1], "candidates") || !std::strcmp(argv[1], "key") || !std::strcmp(argv[1], "sample")) {
        // spins, colour classes (of equal size), degree, dmax, +-1, largest coupler, starts, samples, plain form,
        // solving samples, sweeps, phases, elite in percent: the shapes the autotuner times, the key they are
        // kept by, or the quad-group shape of one sample
        Problem P;
        std::memset(&P.hdr, 0, sizeof(P.hdr));
        P.hdr.n = arg(2);
        P.hdr.ncol = arg(3);
        for (int c = 0; c < arg(3); ++c) P.csize[c] = arg(2) / arg(3) + (c < arg(2) % arg(3));
        P.jabs_max = arg(7);
        if (argv[1][0] == 's') {
            P.hdr.maxdeg = arg(4);
            const SweepShape s = quad_group_shape(&P, (arg(9) + 3) / 4, 152, kSmemOptin, arg(5) + 1, arg(6) != 0);
            std::printf("%d:%d:%d\n", s.kind, s.block, s.Q);
            return 0;
        }
        PlanGeometry g;
        g.probs.push_back(&P);
        g.prm.form = arg(10) ? SPVAR_FORM_PLAIN : SPVAR_FORM_BATCHED;
        g.C.S_fix = arg(9);
        g.C.S_solve = argc > 11 ? arg(11) : arg(9);
        g.C.Smax = std::max(g.C.S_fix, g.C.S_solve);
        g.T = argc > 12 ? arg(12) : 1000;
        g.iters_max = argc > 13 ? arg(13) : 2;
        g.prm.elite_threshold = argc > 14 ? 0.01 * arg(14) : 0.1;
        g.prm.beta1 = 3.0;
        g.prm.fix_num = g.prm.fix_den = 1;
        g.C.nslots = arg(8);
        g.max_n0 = arg(2);
        g.max_deg = arg(4);
        g.dmax = arg(5);
        g.thr_stride = arg(5) + 1;
        g.jabs_max = arg(7);
        g.pm1 = g.ujs = arg(6) != 0;
        g.ncol_max = arg(3);
        g.class_max = P.csize[0];
        g.sms = 152;
        if (argv[1][0] == 'k')
            for (int64_t x : tune_key(&g)) std::printf("%lld ", (long long)x);
        else
            for (const SweepShape &s : candidate_shapes(&g, kSmemOptin)) std::printf("%d:%d:%d ", s.kind, s.block, s.Q);
    }
    if (!std::strcmp(argv[1], "few")) std::printf("%d\n", (int)server_few_quads(std::atoll(argv[2]), arg(3), arg(4)));
    if (!std::strcmp(argv[1], "trial")) std::printf("%d\n", trial_step(arg(2), arg(3)));
    return 0;
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_1706_07826_gb300 import build as B
    lib = B.build()
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, str(d / "rules.cpp"), lib, "-cudart", "shared",
                    "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", str(d / "rules")], check=True)
    return lambda *a: subprocess.run([str(d / "rules")] + [str(x) for x in a], check=True, capture_output=True,
                                     text=True).stdout.split()


@pytest.mark.parametrize("maxd", [6, 8])
def test_requested_quads_are_taken_where_the_launch_fits(rules, maxd):
    """One quad per item: every size up to 28585 spins, as with one quad per
    word, and none whose launch does not fit a block's shared memory."""
    for n in (27000, 28200, 28275, 28276, 28400, 28585, 28787, 28788, 28800, 29055):
        ok, smem, tabs = rules("request", 256, n, 1, maxd)
        assert int(ok) == (int(smem) <= OPTIN)
        if n <= 28585:
            assert int(ok) == 1
        if n < 28200:
            assert int(tabs) == (maxd == 6)
    assert rules("request", 256, 28800, 1, maxd)[0] == "0"


GENERAL, REGISTER, STREAMING, WARP, QUADS, INTEGER_QUADS = 0, 1, 2, 4, 6, 7


def _kinds(rules, n, deg=6, dmax=12, pm1=True, jmax=1, starts=20, samples=250, plain=False, ncol=2):
    out = rules("candidates", n, ncol, deg, dmax, int(pm1), jmax, starts, samples, int(plain))
    return {int(x.split(":")[0]) for x in out}


@pytest.mark.parametrize("dmax", [32, 100, 254])
@pytest.mark.parametrize("n,starts,samples,plain", [(64, 20, 250, False), (729, 20, 250, False), (729, 1, 69, False),
                                                    (2744, 8, 200, False), (1728, 4, 100, True)])
def test_large_biases_time_every_kernel(rules, dmax, n, starts, samples, plain):
    """+-1 couplers past the byte-lane forms' biases: the warp-per-quad and the
    streaming kernel are timed beside the integer quad groups."""
    assert {STREAMING, WARP, INTEGER_QUADS} <= _kinds(rules, n, dmax=dmax, starts=starts, samples=samples, plain=plain)


def test_problems_past_the_quad_groups_time_the_general_kernel(rules):
    assert QUADS in _kinds(rules, 28200) and GENERAL not in _kinds(rules, 28200)
    assert QUADS not in _kinds(rules, 28800) and GENERAL in _kinds(rules, 28800)


@pytest.mark.parametrize("pm1,jmax,dmax", [(True, 1, 12), (True, 1, 60), (False, 3, 30), (False, 90, 900)])
@pytest.mark.parametrize("n", [8, 27, 64, 191])
def test_small_problems_time_the_general_kernel(rules, n, pm1, jmax, dmax):
    """A block of small problems' quads leaves most threads of a quad-group
    block idle: the general kernel's items of 4 and 8 quads are timed too."""
    out = rules("candidates", n, 2, 6, dmax, int(pm1), jmax, 20, 250, 0)
    assert {"0:128:4", "0:128:8", "0:256:4", "0:256:8", "0:512:4", "0:512:8"} <= set(out)
    assert GENERAL not in _kinds(rules, 192, dmax=dmax, pm1=pm1, jmax=jmax)


@pytest.mark.parametrize("T", [0, 1, 100, 127, 128, 129, 200, 255, 256, 1000, 4097])
@pytest.mark.parametrize("t", [128, 512])
def test_trials_reach_the_schedules_end(rules, T, t):
    step = int(rules("trial", T, t)[0])
    sweeps = T // step
    assert min(T, t) <= sweeps < 2 * t and sweeps * step <= T  # no row past the table
    assert T - sweeps * step < step                            # and the cold end is reached


def test_plans_that_share_a_choice_have_the_same_candidates(rules):
    """Two plans of one key are timed over the same shapes: the solving sample,
    which decides whether few quads are launched, is part of it, and so is what
    the trials depend on."""
    seen = {}
    for fixing, solving in ((50, 50), (50, 1000), (50, 0), (1000, 50)):
        for starts in (1, 4, 40):
            for T, phases, elite in ((100, 2, 10), (1000, 2, 10), (1000, 9, 10), (1000, 2, 50)):
                a = (729, 2, 6, 12, 1, 1, starts, fixing, 0, solving, T, phases, elite)
                key, shapes = tuple(rules("key", *a)), rules("candidates", *a)
                assert key not in seen
                seen[key] = shapes
    base = (729, 2, 6, 12, 1, 1, 4, 100, 0, 100)
    assert rules("key", *base, 1000, 2, 10) == rules("key", *base, 600, 2, 12)  # a scan's neighbours share it
    assert rules("key", *base, 1000, 2, 10) != rules("key", *base, 400, 2, 10)


def test_server_steps_of_few_quads(rules):
    """Three quads of the largest problem in flight per SM, smaller problems by their spins."""
    for quads, n, few in ((26, 1728, 1), (456, 216, 1), (457, 216, 0), (800, 729, 0)):
        assert int(rules("few", quads * n, n, 152)[0]) == few
    assert int(rules("few", 400 * 64 + 400 * 1728, 1728, 152)[0]) == 1
    assert int(rules("few", 16384 * 4096 * 32768, 32768, 152)[0]) == 0  # past 32 bits


@pytest.mark.parametrize("n,ncol,deg,dmax,samples,quads", [
    (200, 4, 8, 472, 40, 1),        # ten items of one quad, not two of eight whose units fill idle warps
    (200, 4, 8, 472, 600, 1),
    (27, 3, 6, 900, 16000, 16),     # one round of 250 items, not two of 500
    (27, 3, 6, 900, 9728, 8)])
def test_quads_per_item_of_an_integer_sample(rules, n, ncol, deg, dmax, samples, quads):
    kind, block, q = rules("sample", n, ncol, deg, dmax, 0, 40, 1, samples, 0)[0].split(":")
    assert (int(kind), int(q)) == (INTEGER_QUADS, quads)


def test_small_and_many_classes_time_a_warp_per_quad(rules):
    """Past four classes the register kernel has no slots for a +-1 problem, and
    small classes leave a quad-group block's threads idle."""
    for n, ncol in ((20, 5), (83, 8), (286, 4), (511, 2), (2000, 5)):
        assert WARP in _kinds(rules, n, deg=8, dmax=18, ncol=ncol)
    assert WARP not in _kinds(rules, 512, deg=8, dmax=18, ncol=4)
