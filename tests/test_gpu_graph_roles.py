"""A captured graph between eager generations and reloads: its kernels hold the
buffers of the capture, so a replay is refused while parents and children are
in each other's buffers, and in fitness-first order until the loaded trees
have a plan of their own.  What is not refused equals the eager run bit for
bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pop(lazy):
    import synth
    import paper_2205_03251_gb300 as gp
    gp.build()
    w = synth.workload(3, n_trees=96, target=8_000)
    pop = gp.Population(w["x"], w["t"], w["consts"], w["ops"], w["off"], max_nodes=20_000, cache_threshold=64, seed=5,
                        lazy=lazy)
    return gp, w, pop


def _state(pop):
    import oracle
    return oracle.canon_nan(pop.fitness()).tobytes(), [pop.tree(i).tobytes() for i in range(pop.P)]


def _generation(pop, g):
    pop.crossover(g)
    pop.eval_incremental()


def _refused(gp, pop):
    with pytest.raises(gp.GpError) as e:
        pop.graph_launch()
    assert e.value.code == gp.GP_ESTATE


def test_replay_after_an_odd_number_of_generations_is_refused():
    gp, w, ref = _pop(False)
    ref.eval_full()
    want = []
    for g in (0, 1, 2, 3, 2, 3):
        _generation(ref, g)
        want.append(_state(ref))
    ref.close()
    gp, w, pop = _pop(False)
    pop.set_graph_mode(True)
    pop.eval_full()
    pop.graph_capture(0, 2)
    pop.graph_launch()
    assert _state(pop) == want[1]
    _generation(pop, 2)
    _refused(gp, pop)
    assert _state(pop) == want[2]
    _generation(pop, 3)
    assert _state(pop) == want[3]
    pop.graph_launch()                                # the second replay: generations 2 and 3
    assert _state(pop) == want[5]
    pop.close()


def test_replay_of_a_reloaded_fitness_first_population():
    gp, w, pop = _pop(True)
    pop.set_graph_mode(True)
    pop.eval_full()
    _generation(pop, 0)
    pop.graph_capture(1, 2)
    pop.graph_launch()
    want = _state(pop)
    pop.load_trees(w["ops"], w["off"])
    pop.eval_full()
    _refused(gp, pop)                                 # no plan of these trees yet
    _generation(pop, 0)
    _refused(gp, pop)                                 # the second generation outside the graph: buffers changed
    pop.graph_capture(1, 2)
    pop.graph_launch()
    assert _state(pop) == want
    pop.close()
