"""bench.py's DRAM traffic figure: a capture speaks for another size only where both the
captured and the present visited sets are far larger than the L2."""
import pytest

SUMMARY = "# a comment = not a key\npass_kernel_code_sha256_16 = {key}\nvisited_bytes = {visited}\ndram_bytes_per_entry = {per}\n"


@pytest.fixture
def bench(tmp_path, monkeypatch):
    import bench
    (tmp_path / "profiles").mkdir()
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    monkeypatch.setattr(bench, "kernel_code_hash", lambda: "k")
    return bench


def _write(tmp_path, **kw):
    (tmp_path / "profiles" / "pass_kernel_traffic.txt").write_text(SUMMARY.format(**kw))


def test_a_capture_of_the_l2s_size_is_not_scaled_up(bench, tmp_path):
    _write(tmp_path, key="k", visited=126835180, per=12.423)  # a visited set of about the L2's size
    assert bench.pass_traffic(2.0 ** 30) is None
    _write(tmp_path, key="k", visited=2147483648, per=15.75)
    assert bench.pass_traffic(2.0 ** 30) == 15.75 * 2.0 ** 30
    assert bench.pass_traffic(2.0 ** 24) is None  # this size keeps entries in the L2
    _write(tmp_path, key="other", visited=2147483648, per=15.75)
    assert bench.pass_traffic(2.0 ** 30) is None


def test_a_summary_without_its_size_is_not_used(bench, tmp_path):
    (tmp_path / "profiles" / "pass_kernel_traffic.txt").write_text(
        "pass_kernel_code_sha256_16 = k\ndram_bytes_per_entry = 12.4230\n")
    assert bench.pass_traffic(2.0 ** 30) is None

