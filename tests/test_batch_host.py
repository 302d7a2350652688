"""Host logic of the batched sampler and of the one-column solve on a stand-in for the CUDA runtime
(batch_host.cpp), linked with the library's own object files."""
import os
import subprocess

import pytest

from paper_2510_20604_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    _build.build()
    exe = str(tmp_path_factory.mktemp("batch") / "batch_host")
    inc = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    objs = [os.path.join(_build.BUILD, o) for o in ("batch.o", "graph.o", "estimate.o", "solver.o", "cg1.o")]
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", _build.INCLUDE, "-I", inc, "-o", exe,
                    os.path.join(HERE, "batch_host.cpp")] + objs, check=True)
    return exe


@pytest.mark.parametrize("use_graph", [0, 1])
def test_every_pull_is_a_tree(driver, use_graph):
    """A launch has as many pulls as trees for every remainder of the tree
    count (a block that skips pulls passes none of a tree's barriers between
    two writes of the shared pull number)."""
    r = subprocess.run([driver, "-1", str(use_graph)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("nth", [0, 1, 2])
def test_a_failed_rebuild_leaves_nothing_stale(driver, nth, use_graph):
    """The nth allocation of a call with another tree count fails (the two
    classes' items, the spill array); the next call with the first count gives
    no freed memory to a launch."""
    r = subprocess.run([driver, str(nth), str(use_graph)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_solve_takes_as_many_blocks_as_the_device_holds(driver):
    """A context that refuses the cooperative launch gets at least half of the
    blocks that it holds at once, not one."""
    r = subprocess.run([driver, "solve"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_dense_graphs_are_not_solved_by_a_few_blocks(driver):
    """A graph of few rows and many arcs gets blocks for its arcs."""
    r = subprocess.run([driver, "dense"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_few_trees_take_wide_blocks(driver):
    """A tree that has an SM to itself is run by 256 threads, one of at most 448
    vertices by a warp."""
    r = subprocess.run([driver, "few"], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
