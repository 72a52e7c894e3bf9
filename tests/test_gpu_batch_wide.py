"""The grouped GEMM kernel of a gene is settled by the suite and by whether the gene carries the chain,
not by the genes measured beside it: a suite of unaligned sizes runs the chains' problems in a
launch of their own, any other suite runs all in one, and every gene's results carry the bits of
the same gene without fusion, alone."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
FUSED, PLAIN = [0b111111, 0b001111], [0b110011, 0b000010]


@pytest.fixture(scope="module")
def gao():
    from paper_1806_01430_gb300 import _build
    _build.build()
    import paper_1806_01430_gb300 as g
    return g


@pytest.mark.parametrize("prec,sizes,wide", [(2, [257, 129, 65, 301], True), (2, [257, 128, 64, 300], False),
                                             (3, [257, 129, 65, 301], False)])
def test_kernel_of_a_gene(gao, prec, sizes, wide):
    progs = [W.six_loop(n, 3500 + i, outputs=("C", "D", "E", "r", "f")) for i, n in enumerate(sizes)]
    names = ("C", "D", "E", "r", "f")
    want = {}
    handles = [gao.prog_from_workload(p, gemm_prec=prec) for p in progs]
    b = gao.batch_create(handles)
    for g in FUSED + PLAIN:
        gao.batch_evaluate(b, [g])
        want[g] = [{nm: gao.prog_output(h, p.index(nm)).copy() for nm in names} for h, p in zip(handles, progs)]
    gao.batch_destroy(b)
    handles = [gao.prog_from_workload(p, gemm_prec=prec, fuse_chains=gao.FUSE_ON) for p in progs]
    b = gao.batch_create(handles, replicas=4)
    for group in (FUSED, PLAIN, [FUSED[0], PLAIN[0], FUSED[1], PLAIN[1]], PLAIN[:1] + FUSED[:1]):
        gao.batch_set_replicas(b, 4)  # clears the cache
        before = gao.batch_stats(b)
        _, sec, _ = gao.batch_evaluate(b, group)
        after = gao.batch_stats(b)
        mixed = len({g in FUSED for g in group}) == 2
        assert after["grouped_launches"] - before["grouped_launches"] == (2 if wide and mixed else 1)
        assert after["grouped_genes"] - before["grouped_genes"] == len(group)
        assert all(s > 0 for s in sec)
        for r, g in enumerate(group):
            for i, p in enumerate(progs):
                h = gao.batch_replica_prog(b, r, i)
                got = {nm: gao.prog_output(h, p.index(nm)) for nm in names}
                for nm in ("C", "D", "E", "r"):
                    assert np.array_equal(got[nm].view(np.uint32), want[g][i][nm].view(np.uint32)), (g, i, nm)
                # binary64 partials of the same squares (fused) against binary32 ones of four each
                assert abs(got["f"][0, 0] - want[g][i]["f"][0, 0]) <= 2e-7 * want[g][i]["f"][0, 0]
    gao.batch_destroy(b)
