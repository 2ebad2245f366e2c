"""The bench reports a captured DRAM traffic only for the device source it was taken on, all of it."""
import hashlib

from paper_2205_05681_gb300 import build


def test_traffic_is_tied_to_every_device_source(monkeypatch):
    import bench
    wl = "ch4_111_batched"
    text = [open(p, "rb").read() for p in build.DEVICE]
    assert len(text) == 2
    monkeypatch.setitem(bench.MEASURED_TRAFFIC, "device_src_sha1", hashlib.sha1(b"".join(text)).hexdigest())
    assert bench.measured_traffic(wl, True) == bench.MEASURED_TRAFFIC[wl]
    assert bench.measured_traffic(wl, False) is None
    for t in text:  # one of the two alone
        monkeypatch.setitem(bench.MEASURED_TRAFFIC, "device_src_sha1", hashlib.sha1(t).hexdigest())
        assert bench.measured_traffic(wl, True) is None
