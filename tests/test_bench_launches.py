"""bench.py reports the kernels that the library says it launched."""
import bench


class Counting:
    launched = 7

    def step_launches(self):
        return self.launched


def test_launches_of_the_timed_steps_are_the_librarys():
    sim = Counting()
    before = bench.step_launches(sim)
    sim.launched += 1 + 15 * 20
    assert bench.timed_launches(sim, before, 20) == 301


def test_a_handle_that_does_not_count():
    assert bench.step_launches(object()) is None
    assert bench.timed_launches(object(), None, 3) == 3 * 16 + 2
