"""The bench's record of DRAM traffic: found for the walk sources it was taken on,
by bin, and for no others."""
import bench


def test_record_of_the_current_sources(tmp_path):
    sha = bench.walk_sources_sha()
    assert len(bench.BINS) == bench.NBINS
    path = tmp_path / "traffic.txt"
    path.write_text("".join(f"bin={b} src_sha={sha} workload={bench.WORKLOAD} "
                            f"bytes_per_build={k + 1}\n" for k, b in enumerate(bench.BINS)))
    assert [bench.recorded_traffic(k, str(path)) for k in range(bench.NBINS)] == [1, 2, 3, 4, 5]
    path.write_text(path.read_text().replace(sha, "0" * 16))
    assert all(bench.recorded_traffic(k, str(path)) is None for k in range(bench.NBINS))
    assert bench.recorded_traffic(0, str(tmp_path / "none.txt")) is None


def test_committed_record_is_read():
    """Every line of the committed record names a bin and a workload of the bench."""
    import os
    lines = open(os.path.join(bench.ROOT, "profiles", "traffic.txt")).read().split("\n")
    for ln in filter(None, lines):
        kv = dict(x.split("=", 1) for x in ln.split())
        assert kv["bin"] in bench.BINS and kv["workload"] == bench.WORKLOAD
        assert float(kv["bytes_per_build"]) > 0 and len(kv["src_sha"]) == 16
