"""The register qubits of a stage, chosen with all candidates followed together, in the forms of plan
that have rules of their own: phases that wait for the next gate on their qubit (pipelined plain plans)
and gates behind a block's matrix that close its qubits (the tensor-core plans)."""
import pytest

import host_cpp


@pytest.fixture(scope='module')
def planner(tmp_path_factory):
    return host_cpp.build(tmp_path_factory.mktemp('planner'), 'planner_choices', ['plan.cpp'], ['-DSV_PLAN_CHECK'])


@pytest.mark.parametrize('form', ['pipelined', 'matrix_stages', 'blocks_of_5', 'blocks_of_4'])
def test_register_qubits_are_those_of_a_search_one_by_one(planner, form):
    r = host_cpp.run(planner, form)
    assert r.returncode == 0, r.stdout + r.stderr
