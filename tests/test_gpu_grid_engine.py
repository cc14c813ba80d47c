"""The grid engine on lattices that the on-chip engine takes by default: the
parity tests of solves, guesses, forces, trajectories, observables and the
exact-block form with HH_ENGINE_ONCHIP=0."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_exact_block import (test_exact_block_force, test_exact_block_solve,  # noqa: E402,F401
                                  test_exact_block_trajectories_match_oracle)
from test_gpu_parity import (hh, test_action_heatbath_identity, test_chebyshev_pcg_matches_oracle,  # noqa: E402,F401
                             test_chronological_guess_trajectory_matches_oracle, test_force_matches_oracle,
                             test_leapfrog_reversible_on_gpu, test_observables_match_oracle,
                             test_omelyan_trajectories_match_oracle, test_solve_from_initial_guess,
                             test_solve_true_residual_and_solution, test_solve_zero_rhs_and_iteration_cap,
                             test_trajectories_match_oracle)


@pytest.fixture(autouse=True)
def grid_engine(monkeypatch):
    monkeypatch.setenv("HH_ENGINE_ONCHIP", "0")


def test_the_switch_selects_the_grid_engine(hh):  # noqa: F811
    with hh.Context(1, 32, 64) as ctx:
        assert ctx.solver_layout(1)["onchip"] == 0
