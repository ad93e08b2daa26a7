"""Which kernels a run launches, with how many blocks, and what the host side makes of their status words: the library over
a CUDA runtime that launches nothing (fake_cuda.cpp), on the CPU."""
import ctypes as C
import json
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))

CHILD = """
import ctypes as C, json, sys
fake = C.CDLL(sys.argv[1], mode=C.RTLD_GLOBAL)               # before the library, which then finds these definitions
sys.path[:0] = sys.argv[2:4]
import workloads as W
from paper_2407_13585_b200 import binding as B, build
B.load_kernel_library(build.TEST_LIB)
fake.fake_launches.restype = C.c_char_p
fake.fake_status.restype = C.POINTER(C.c_uint32)
lib = B.lib()


def bound(prog, pi=None, recompute=0):
    g = B.Graph(prog.nodes, prog.outputs)
    g.set_partition_recompute(pi or [-1 if nd.kind == "input" else 0 for nd in prog.nodes], recompute)
    address = 1 << 40
    for i, nd in enumerate(prog.nodes):
        count = 1
        for e in nd.shape:
            count *= e
        assert lib.acc_bind(g._h, i, C.c_void_p(address), C.c_size_t(4 * count)) == 0
        address += (4 * count + 255) // 256 * 256
    return g


def run(g, workspace=1 << 50):
    code = lib.acc_run(g._h, C.c_void_p(workspace), C.c_size_t(1 << 44), None, B.FUSED)
    assert code == 0, (code, lib.acc_last_error())


def launches(prog, pi=None, recompute=0):
    fake.fake_clear()
    g = bound(prog, pi, recompute)
    run(g)
    out = []
    for line in fake.fake_launches().decode().splitlines():
        name, grid, block, how = line.split("|")
        out.append([name.split("<")[0].split("::")[-1], "<" + name.split("<", 1)[1], int(grid), int(block), how == "C"])
    return out
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    """Runs a script behind CHILD in a process of its own and returns what it leaves in `result`."""
    fake = str(tmp_path_factory.mktemp("fake") / "fake_cuda.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-o", fake, os.path.join(HERE, "fake_cuda.cpp"), "-ldl", "-pthread"], check=True)

    def run(script):
        p = subprocess.run([sys.executable, "-c", CHILD + script + "\nprint('RESULT' + json.dumps(result))", fake, os.path.dirname(HERE), HERE],
                           capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, p.stderr[-3000:]
        return json.loads(p.stdout.rsplit("RESULT", 1)[1])
    return run


def test_the_ring_has_no_more_blocks_than_a_look_back_warp_adds_up(child):
    """The first block's look-back warps cover 160 tiles a round: on a device with more SMs the grid stays at that."""
    got = child("""
result = []
for sms in (100, 148, 160, 170):
    fake.fake_device(sms, 1)
    result.append(launches(W.row_scans(1, 1 << 24), [-1, 0, 1, 1]))
""")
    assert [[k[0] for k in run] for run in got] == [["k_scan_ring", "k_scan_ring"]] * 4
    assert [{k[2] for k in run} for run in got] == [{100}, {148}, {160}, {160}]


def test_which_kernel_scans(child):
    """Rows of one scan: blocks per row, the ring, and between them k_scan where it is quicker (see look_back_is_quicker)."""
    got = child("""
def kinds(prog, pi):
    return [k[0] + ("" if k[0] != "k_scan" else " resident" if k[4] else " ticket") for k in launches(prog, pi)]
result = {}
for rows, cols in json.loads('[[1,16381],[1,20000],[1,20001],[64,17000],[148,33000],[300,17000],[32,30001],[3,500001],[148,33001],[1,900001],'
                             '[1,300000],[1,2097152],[1,3000000]]'):
    result["%d x %d" % (rows, cols)] = kinds(W.row_scans(rows, cols), [-1, 0, 1, 1])
for n in (6144, 6145, 16381, 16382, 131072, 131073):
    result["gather %d" % n] = kinds(W.config3(n), [-1, -1, 0, 0, 0, 0])
    result["two gathers %d" % n] = kinds(W.sum_of_two_gathers(n), None)
""")
    ring, back, rows = ["k_scan_ring"] * 2, ["k_scan resident"] * 2, ["k_scan_rows"] * 2
    want = {"1 x 16381": rows, "1 x 20000": back, "1 x 20001": ring, "64 x 17000": back, "148 x 33000": back, "300 x 17000": ring,
            "32 x 30001": back, "3 x 500001": back, "148 x 33001": ring, "1 x 900001": back, "1 x 300000": back, "1 x 2097152": back, "1 x 3000000": ring}
    assert {k: v for k, v in got.items() if "gather" not in k} == want
    assert [got["gather %d" % n][0] for n in (6144, 6145, 16381)] == ["k_scan_rows", "k_scan resident", "k_scan resident"]
    assert [got["gather %d" % n][0] for n in (16382, 131072, 131073)] == ["k_scan ticket", "k_scan ticket", "k_scan_ring"]
    assert [got["two gathers %d" % n] for n in (16381, 16382, 131072, 131073)] == [["k_scan resident"]] + [["k_scan ticket"]] * 3


def test_a_block_reads_a_row_with_as_many_chunks_as_it_has(child):
    got = child("""
result = [launches(W.row_scans(10, cols), [-1, 0, 1, 1])[0][:2] for cols in (1024, 1025, 4093, 4094, 8189, 8190, 16381)]
""")
    assert {g[0] for g in got} == {"k_scan_rows"}
    assert [g[1].split(", ", 1)[1] for g in got] == ["1, 4>", "16, 2>", "16, 2>", "16, 4>", "16, 4>", "16, 8>", "16, 8>"]


def test_a_block_has_as_many_warps_as_a_row_has_chunks_for(child):
    got = child("""
result = [launches(W.row_scans(10, cols), [-1, 0, 1, 1])[0][3] // 32 for cols in (1025, 1277, 1278, 1280, 4093, 4094, 4605, 4606, 8189, 8190, 9213, 9214, 16381)]
""")
    assert got == [5, 5, 6, 5, 16, 9, 9, 10, 16, 9, 9, 10, 16]


STATUS = """
def finish(g, workspace):
    return lib.acc_finish(g._h, C.c_void_p(workspace), None)


def reports_to():                                            # the status words of the last launch, and its run's number
    run_id = C.c_uint32()
    return fake.fake_status(C.byref(run_id)), run_id.value

prog = W.config1(4096)
"""


def test_no_run_in_flight_loses_its_report(child):
    """Runs of one handle over more workspaces than it keeps lines for: each wait reports its own run, as often as it is asked."""
    got = child(STATUS + """
g = bound(prog)
spaces = [(1 << 50) + (k << 32) for k in range(200)]
lines = []
for ws in spaces:
    run(g, ws)
    lines.append(reports_to())
for words, run_id in (lines[0], lines[100], lines[199]):     # three kernels meet an empty segment
    words[2] = run_id
result = {"lines": len({C.addressof(w.contents) for w, _ in lines}), "codes": [finish(g, ws) for ws in spaces]}
# further workspaces: lines of runs with nothing to report are used again, the others' are not
for k in range(200, 1000):
    run(g, (1 << 50) + (k << 32))
    finish(g, (1 << 50) + (k << 32))
result["again"] = [finish(g, ws) for ws in spaces]
result["pages"] = fake.fake_pages()
""")
    bad = got["codes"][0]
    want = [bad if k in (0, 100, 199) else 0 for k in range(200)]
    assert bad < 0 and got["codes"] == want and got["again"] == want
    assert got["lines"] == 200 and got["pages"] == 1


def test_lines_of_runs_that_nobody_waited_for_are_handed_on_last(child):
    got = child(STATUS + """
def line_of(wait):
    g = bound(prog)
    run(g)
    at = C.addressof(reports_to()[0].contents)
    if wait:
        finish(g, 1 << 50)
    lib.acc_graph_destroy(g._h)
    g._h = None
    return at
first = line_of(False)
after = [line_of(True) for k in range(100)]
result = {"again": first in after, "used": len(set(after)), "pages": fake.fake_pages()}
""")
    assert got == {"again": False, "used": 1, "pages": 1}


def test_lines_of_captured_runs_come_back_when_handle_and_graph_are_gone(child):
    """A captured run's line is the graph's too: it is no other handle's while the graph can be replayed, whether or not its
    handle is left, and then goes to the next one."""
    got = child(STATUS + """
def used_after(k):
    lines = set()
    for _ in range(k):
        g = bound(prog)
        run(g)
        lines.add(C.addressof(reports_to()[0].contents))
        finish(g, 1 << 50)
        lib.acc_graph_destroy(g._h)
        g._h = None
    return lines
result = []
for round in range(20):
    fake.fake_capturing(1)
    captured = set()
    for _ in range(100):
        g = bound(prog)
        run(g)
        captured.add(C.addressof(reports_to()[0].contents))
        lib.acc_graph_destroy(g._h)
        g._h = None
    fake.fake_capturing(0)
    result.append([len(captured), len(captured & used_after(5)), fake.fake_pages()])
    fake.fake_destroy_graph()
""")
    assert [g[:2] for g in got] == [[100, 0]] * 20
    assert max(g[2] for g in got) <= 2


def test_a_histogram_waits_for_its_slowest_cta_as_long_as_a_walk_may_take(child):
    """Eight polls per element of a CTA's share on top of the usual limit, whatever else the plan holds."""
    got = child("""
fake.fake_second_argument.restype = C.POINTER(C.c_int32)
result = []
for n in (1 << 18, 1 << 27, 1 << 30):
    names = [k[0] for k in launches(W.config5(n, 1 << 15), [-1, -1, 0, 0, 0, 0, 1])]
    plan = fake.fake_second_argument()
    result.append([names[0], plan[4] > 0, plan[5]])
""")
    shares = [(1 << 18) // 32, (1 << 27) // 148, (1 << 30) // 148]
    assert [g[:2] for g in got] == [["k_hist", True]] * 3
    assert [g[2] for g in got] == [(1 << 20) + 8 * s for s in shares]


def test_few_elements_are_folded_by_one_cluster_of_blocks(child):
    """... counted over all arrays that are read or stored (the third cluster reads two); a gather below the fold keeps the grid."""
    got = child("""
result = [[k[0], k[2]] for n in (262144, 262145) for k in launches(W.config1(n))]
result += [launches(W.config1(n), [-1, 0, 0, 0, 1])[1][0] for n in (262144, 262145)]
result += [launches(W.config1(n), [-1, 0, 0, 1, 1])[1][0] for n in (131072, 131073)]
""")
    assert got == [["k_stream_few", 8], ["k_stream", 256]] + ["k_stream_few", "k_stream"] * 2


def test_few_tiles_are_folded_by_clusters_of_blocks(child):
    got = child("""
result = [launches(W.config2(rows), [-1, 0, 0, 0])[0][:3:2] for rows in (63, 64, 65, 128, 129, 2559)]
""")
    assert got == [["k_rowfold", 63], ["k_tile_pair_tma", 1], ["k_tile_rows", 16], ["k_tile_rows", 16], ["k_tile_rows", 24], ["k_tile_rows", 320]]


def test_two_arrays_are_folded_by_clusters_of_blocks_while_these_run_all_at_once(child):
    """... which 34 blocks of rows with two arrays' tiles do not (2176 rows: 18.4 us, by pairs of tiles 14.3)."""
    got = child("""
result = [launches(W.diagonal_of_product(rows), [-1, -1, 0, 0, 0])[0][0] for rows in (65, 2111, 2112, 2113, 2176, 2559)]
""")
    assert got == ["k_tile_rows"] * 3 + ["k_tile_pair", "k_tile_pair_tma", "k_tile_pair"]


def test_one_segmented_fold_alone_takes_its_operands_through_registers(child):
    """Two that share the walk have them land in shared memory: eight warps, two steps of 2 KB each."""
    got = child("""
fake.fake_seg_shared.restype = C.c_size_t
result = []
for pi in ([-1, -1, 0, 0, 0], [-1, -1, 0, 0, 1], [-1, -1, 0, 1, 2]):
    launches(W.segmented_sums(10**6, 10**5), pi)
    result.append(fake.fake_seg_shared())                     # of the last cluster's
""")
    assert got == [8 * 2 * 2048, 0, 0]


def test_unaligned_tile_pairs_are_copied_from_2720_rows_on(child):
    got = child("""
result = [launches(W.config2(rows), [-1, 0, 0, 0])[0][0] for rows in (2561, 2719, 2721, 64, 2560)]
""")
    assert got == ["k_tile_pair", "k_tile_pair", "k_tile_pair_tma", "k_tile_pair_tma", "k_tile_pair_tma"]


def test_the_forms_of_a_look_back_that_the_gpu_tests_let_run_out(child):
    """The programs of test_each_look_back_that_runs_out_is_reported take the kernels that it names."""
    got = child("""
result = [[k[0], k[4]] for k in launches(W.sum_of_two_gathers(1 << 20)) + launches(W.row_scans(1, 1 << 20), [-1, 0, 1, 1]) +
          launches(W.row_scans(1, 1 << 23), [-1, 0, 1, 1]) + launches(W.config3(1 << 25))[-1:]]
""")
    assert got == [["k_scan", False]] + [["k_scan", True]] * 2 + [["k_scan_ring", True]] * 2 + [["k_scan_merge_pipelined", True]]


def test_one_thread_waits_while_another_enqueues(child):
    got = child(STATUS + """
g = bound(prog)
result = fake.fake_run_and_wait(C.cast(lib.acc_run, C.c_void_p), C.cast(lib.acc_finish, C.c_void_p), g._h, B.FUSED, 3000)
""")
    assert got == 0
