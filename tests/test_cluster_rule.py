"""Batches of small lattices in clusters or in the step kernels: every cluster has the blocks
of the largest lattice, and clusters beyond those resident wait for a whole call's steps."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# blocks, lattices, resident clusters, us per step with the step kernels and with clusters
# (unit relaxation times and, from 608 / 148 / 33 / 14 resident on, two-phase with the source)
MEASURED = [(1, 1024, 912, 9.89, 6.40), (1, 4096, 912, 27.2, 16.3), (2, 256, 456, 11.4, 9.7),
            (2, 801, 456, 10.4, 8.4), (4, 128, 222, 9.0, 7.4), (4, 801, 222, 10.5, 15.5), (8, 64, 110, 11.5, 7.5),
            (8, 401, 110, 8.5, 15.2), (8, 801, 110, 10.6, 28.7), (16, 32, 47, 6.4, 5.3), (16, 65, 47, 6.4, 7.7),
            (16, 201, 47, 7.6, 18.1), (16, 801, 47, 10.7, 65.8), (16, 33, 21, 5.8, 7.7), (16, 401, 21, 9.2, 68.3),
            (16, 801, 21, 10.7, 134.0), (1, 512, 608, 27.9, 13.4), (4, 201, 148, 9.7, 8.4), (4, 401, 148, 11.3, 12.5),
            (16, 101, 33, 8.9, 13.5), (16, 16, 14, 8.0, 10.8), (16, 401, 14, 12.4, 109.6)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("clusterrule") / "cluster_rule")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-o", exe,
                    os.path.join(ROOT, "tests", "native", "cluster_rule_host.cpp")], check=True)

    def ask(rows):
        text = "\n".join("%d %d %d" % r[:3] for r in rows)
        return [int(x) for x in subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()]

    return ask


def test_rule_takes_the_faster_side(rule):
    assert rule(MEASURED) == [int(r[4] < r[3]) for r in MEASURED]


def test_no_cluster_fits(rule):
    assert rule([(1, 1, 0), (16, 5, 0), (16, 5, -1)]) == [0, 0, 0]


@pytest.mark.gpu
@pytest.mark.parametrize("relax", [dict(), dict(kind=1, tau_l=0.6, visc_ratio=3.0)])
def test_many_small_lattices_beside_a_large_one(relax):
    """401 lattices, one of 4,096 nodes: bitwise the single lattices, and a step within four
    times that of 17 (in clusters of the largest lattice's shape it took ten times)."""
    torch = pytest.importorskip("torch")
    import lbm_inputs as I
    import paper_2107_06355_gb300 as P

    eos, rel = P.EOSParams(P.EOS_SMOOTH, 0.6, 0.387, 2.0, 0.834), P.Relax(**relax)
    d = P.eos_setup(eos)

    def batch(n):
        shapes = [(64, 64)] + [(10, 6)] * n
        b = P.Batch([(x, y, P.BC_PERIODIC) for x, y in shapes], [eos] * (n + 1), [rel] * (n + 1))
        inits = []
        for i, (x, y) in enumerate(shapes):
            rho = I.perturbed(I.planar(x, y, d["rho_v"], d["rho_l"], W=6.0), 1e-3, i % 7)
            inits.append((rho, *I.random_velocity(rho.shape, 0.01, i % 7)))
            b.init_equilibrium(i, *inits[-1])
        return b, shapes, inits

    def time_of(b):
        best = 1e9
        for _ in range(5):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            e0.record()
            b.step(40)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    many, shapes, inits = batch(400)
    many.step(5)
    for k in (0, 1, 200, 400):
        ref = P.Simulation(*shapes[k], P.BC_PERIODIC, eos, rel)
        ref.init_equilibrium(*inits[k])
        ref.step(5)
        assert torch.equal(many.get_f(k).view(torch.int64), ref.get_f().view(torch.int64)), k
        ref.close()
    few = batch(16)[0]
    assert time_of(many) < 4.0 * time_of(few)
    many.close()
    few.close()
