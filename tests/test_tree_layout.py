"""What the host lays out for the prefix trees: how full an item keeps the warps of its block."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WARPS, BLOCKS = 4, 5                       # of a block, of an SM


@pytest.fixture(scope="session")
def layout(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("layout") / "tree_layout")
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O1", "-o", exe,
                    os.path.join(ROOT, "tests", "tree_layout.cu")], check=True)

    def run(layers, nodes, first_moe=0, delta=205, levels=2, node_size=8, n_conf=1000):
        out = subprocess.run([exe, *map(str, (layers, first_moe, delta, levels, nodes, node_size, n_conf))], check=True, capture_output=True, text=True).stdout
        return [dict(zip(("PP", "nmap", "parts", "items", "smem", "low"), map(int, line.split()))) for line in out.splitlines()]
    return run


# about a thousand devices of four types: no stage size homogeneous; one of them (840 mappings); three types; two
@pytest.mark.parametrize("layers,nodes", [(96, "72,27,16,13"), (77, "61,33,21,13"), (60, "72,27,16,13"), (96, "64,32,16,16"), (96, "59,27,10"), (60, "11,9,7,5")])
def test_items_of_deep_classes_keep_their_block_busy(layout, layers, nodes):
    """Classes of few mappings, too: at least three of the four warps of a block have a part of their own, and five blocks
    find room on an SM."""
    rows = layout(layers, nodes)
    assert rows
    for c in rows:
        assert c["smem"] + 1280 <= 227 * 1024 // BLOCKS, c
        if c["PP"] >= 8:
            assert c["parts"] / c["items"] >= min(WARPS - 1, c["nmap"]), c


@pytest.mark.parametrize("layers,nodes,first_moe,delta,node_size", [(96, "72,27,16,13", 0, 205, 8), (60, "12,8,8,4", 1, 205, 8), (16, "1,1", 0, -1, 4),
                                                                    (32, "2,1,1", 0, 150, 8), (12, "3,1", 5, 300, 2), (255, "8", 0, -1, 8)])
def test_scans_stay_inside_the_row_before(layout, layers, nodes, first_moe, delta, node_size):
    """The window of a scan moves down by one entry a length and asks for two entries more than it uses: the lowest slot
    any task or last stage reads is one of its row buffer."""
    for c in layout(layers, nodes, first_moe, delta, 2, node_size):
        assert c["low"] >= 0, c
