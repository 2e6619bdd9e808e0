"""The tasks a warp takes together: of one width, every cell of a row once, the padding written by the right ones."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="session")
def tasks(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("tasks") / "tree_tasks")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-o", exe,
                    os.path.join(ROOT, "tests", "tree_tasks.cu")], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


# a part that fills iterations of four end layers and more, rows of one cell, wide windows, mixed layer kinds in front (and past
# the first depths), one device type, an odd layer count
@pytest.mark.parametrize("layers,first_moe,delta,nodes,node_size", [(96, 0, 205, "64,32,16,16", 8), (60, 1, 205, "12,8,8,4", 8), (33, 0, 205, "4,4", 8),
                                                                    (16, 0, -1, "1,1", 4), (255, 0, -1, "8", 8), (12, 5, 300, "3,1", 2), (29, 29, 205, "3,3,1", 8)])
def test_tasks_cover_the_rows(tasks, layers, first_moe, delta, nodes, node_size):
    rows = tasks(layers, first_moe, delta, nodes, node_size)
    assert rows and all(faults == 0 for *_, faults in rows), rows
    # the split is searched for without laying out, or putting in order, the tasks of the numbers of parts that are not taken
    assert all(allocated <= 100 * parts + 60 * PP for PP, *_, parts, allocated, _ in rows), rows
    if layers >= 60 and delta > 0:                       # all three widths occur
        assert all(sum(r[i] for r in rows) > 0 for i in (1, 2, 3)), rows


@pytest.fixture(scope="session")
def walk(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("walk") / "tree_walk")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-o", exe,
                    os.path.join(ROOT, "tests", "tree_walk.cu")], check=True)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


# as above, and: 1,820 mappings at 16 stages, few configurations (other numbers of parts), a narrow window, no homogeneous stages
@pytest.mark.parametrize("layers,first_moe,delta,nodes,node_size,n_conf", [
    (96, 0, 205, "64,32,16,16", 8, 1000), (60, 1, 205, "12,8,8,4", 8, 1000), (33, 0, 205, "4,4", 8, 50), (16, 0, -1, "1,1", 4, 1000), (255, 0, -1, "8", 8, 1000),
    (12, 5, 300, "3,1", 2, 1000), (29, 29, 205, "3,3,1", 8, 1000), (60, 0, 205, "24,8", 8, 728), (17, 0, 205, "1,1", 8, 10), (31, 2, 150, "2,1,1", 8, 200),
    (255, 0, 205, "72,27,16,13", 8, 7)])
def test_tasks_reach_every_split(walk, layers, first_moe, delta, nodes, node_size, n_conf):
    """Walked on the host as the kernel walks them, tasks, last stages and ways back give every mapping's own bottleneck and partition, and
    read nothing that was not written or lies outside of the row before."""
    rows = walk(layers, first_moe, delta, nodes, node_size, n_conf)
    assert rows and all(faults == 0 for *_, faults in rows), rows


def test_calls_that_share_blocks_between_configurations(tmp_path):
    """64 devices, three policies: the classes of two mappings share blocks.  The whole pass and ranges of half a wave of items take the
    grouped form; a rank's share with fewer, or whose items are mostly of other classes, does not.  A search
    asks for half of them, a pass for a quarter."""
    exe = str(tmp_path / "tree_groups")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-o", exe,
                    os.path.join(ROOT, "tests", "tree_groups.cu")], check=True)
    conf = (1024, 900, 676, 400, 144, 36)
    ranges = {(0, 3180): (1, 1), (0, 300): (1, 1), (0, 100): (0, 0), (1024, 400): (1, 1), (2600, 580): (1, 0), (0, 1924): (1, 1), (1924, 676): (0, 0), (2600, 400): (0, 0),
              (3144, 36): (0, 0), (17, 0): (0, 0)}
    out = subprocess.run([exe, "32", "205", "4,4", "8", "3", ",".join(map(str, conf)), *(str(x) for r in ranges for x in r)],
                         check=True, capture_output=True, text=True).stdout.split()
    parts, group = out[0:12:2], out[1:12:2]
    assert all((int(g) > 1) == (int(n) <= 2) for n, g in zip(parts, group)) and "4" in group
    assert [int(v) for v in out[12:]] == [v for r in ranges.values() for v in r]
