"""World-size-2 check (gloo, CPU) of the benchmark's multi-rank host logic: record sharding
and the whole-job rate (images of all ranks / slowest rank's time)."""
import os
import socket
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _worker(rank, world, port, q):
    sys.path.insert(0, ROOT)
    os.environ.update(MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port), RANK=str(rank), WORLD_SIZE=str(world))
    import torch.distributed as dist
    import bench
    dist.init_process_group("gloo", rank=rank, world_size=world)
    ms = 100.0 if rank == 0 else 250.0          # rank 1 is the slow one
    rate = bench.whole_job_rate(1024, 10, ms, world)
    mx = bench.reduce_max(ms, world)
    q.put((rank, bench.rank_record_index(rank), rate, mx))
    dist.destroy_process_group()


def test_two_ranks_shard_records_and_take_the_slowest_time():
    import torch.multiprocessing as mp
    s = socket.socket(); s.bind(("127.0.0.1", 0)); port = s.getsockname()[1]; s.close()
    ctx = mp.get_context("spawn")
    q = ctx.Queue()
    ps = [ctx.Process(target=_worker, args=(r, 2, port, q)) for r in range(2)]
    for p in ps:
        p.start()
    res = sorted(q.get(timeout=120) for _ in ps)
    for p in ps:
        p.join(timeout=60)
        assert p.exitcode == 0
    assert [r[1] for r in res] == [0, 1]                      # distinct records, no overlap
    for _, _, rate, mx in res:
        assert mx == 250.0
        assert rate == pytest.approx(2 * 1024 * 10 / 0.250)   # both ranks' images over the slowest time


def test_single_rank_needs_no_process_group():
    sys.path.insert(0, ROOT)
    import bench
    assert bench.reduce_max(3.5, 1) == 3.5
    assert bench.whole_job_rate(100, 2, 50.0, 1) == pytest.approx(100 * 2 / 0.05)


def test_algorithmic_bytes_model():
    sys.path.insert(0, ROOT)
    import bench
    # one 32x32 image: 24 padded blocks, Y unpadded 16 blocks, chroma 4 each
    scans = [(3, 0, 0, 0, 0, 0, 100), (1, 0, 1, 5, 0, 0, 50), (1, 0, 1, 63, 2, 1, 70)]
    m = bench.algorithmic_bytes(scans, [(32, 32)], 3)
    assert m["clear"] == 128 * 24 and m["pixels"] == 128 * 24 + 3 * 1024
    assert m["index"] == 220
    assert m["entropy0"] == 100 + 2 * 1 * 24 + 50 + 2 * 5 * 16
    assert m["entropy1"] == 70 + 2 * 63 * 16 * 2
    m2 = bench.algorithmic_bytes(scans, [(32, 32)], 1)
    assert "entropy1" not in m2 and m2["index"] == 100


def test_layout_bytes_model():
    sys.path.insert(0, ROOT)
    import bench
    # one 17x20 image: 2x2 MCUs, so 16 + 4 + 4 padded blocks; Y unpadded 3 x 3, chroma 2 x 2 each
    scans = [(3, 0, 0, 0, 0, 0, 100), (1, 0, 1, 5, 0, 0, 50), (1, 0, 6, 63, 0, 0, 60), (1, 0, 1, 63, 2, 1, 70), (3, 0, 0, 0, 1, 1, 3),
             (1, 0, 1, 63, 1, 2, 90)]
    infos = [(17, 20)]
    m = bench.layout_bytes(scans, infos, 6)
    assert m["index"] == 2 * 373
    assert m["entropy0"] == 210 + 2 * 24                      # DC values; what AC first passes write depends on the contents
    assert m["entropy1"] == 70 + (32 + 2 * 8) * 9 + 3 + 4 * 24   # masks of two earlier scans, DC bits read and written
    assert m["entropy2"] == 90 + (32 + 8) * 9                 # the earlier refinement's mask covers both
    assert m["pixels"] == 3 * 340 + 18 * 24 + (16 + 32 + 32) * 16
    assert m["total"] == sum(v for n, v in m.items() if n != "total")
    c = bench.layout_bytes(scans, infos, 6, chains=True)
    assert c["total"] == m["total"] and c["chains"] == m["entropy2"] + 70 + (32 + 2 * 8) * 9 and c["entropy1"] == 3 + 4 * 24
    assert bench.layout_bytes(scans, infos, 1)["pixels"] == 3 * 340 + 2 * 24
    assert bench.layout_bytes(scans, infos, 2)["pixels"] == 3 * 340 + 18 * 24
    b = bench.layout_bytes([(3, 0, 0, 63, 0, 0, 400)], infos, 1)        # baseline
    assert b["entropy0"] == 400 + 2 * 24 and b["pixels"] == 3 * 340 + (18 + 16) * 24


def test_counters_outlive_comments_and_nothing_else():
    """The committed ncu counters are quoted while the kernels' code is what they were taken on: comments and line breaks may
    change, code and string literals may not."""
    sys.path.insert(0, ROOT)
    import bench
    a = bench.source_code('int f(int x) {  // twice\n    return 2 * x;\n}\nasm("add.u32 //x;");\n')
    assert a == bench.source_code('/* doubles\n   x */int f(int x) {\n  return 2 * x;  /* not 3 */\n}\n// an addition\nasm("add.u32 //x;");\n').lstrip()
    for other in ("int f(int x) {\n return 3 * x;\n}\nasm(\"add.u32 //x;\");\n", "int f(int x) {\n return 2 * x;\n}\nasm(\"add.u32 //y;\");\n"):
        assert bench.source_code(other) != a
