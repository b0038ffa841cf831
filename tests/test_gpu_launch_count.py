"""gp_stats.launches of a full evaluation counts every launch of the pass over
cached nodes, which takes 32 case blocks at a time."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,more", [(48, 2, 0), (1024, 1, 0), (1025, 1, 1), (2048, 1, 1), (2049, 1, 2), (2048, 2, 0),
                                      (2049, 2, 1), (4096, 4, 0)])
def test_launches_of_a_full_evaluation(C, K, more):
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    w = synth.workload(3, n_trees=8, target=3_000)
    x, t = synth.cases(6, C)
    pop = gp.Population(x, t, w["consts"], w["ops"], w["off"], max_nodes=6_000, cases_per_lane=K)
    for _ in range(2):
        pop.eval_full()
        assert pop.stats()["launches"] == 15 + more
    pop.close()
