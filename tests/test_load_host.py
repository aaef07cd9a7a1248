"""rs.load() with several threads: the library is given out once its tuned
table is in place, not before."""
import threading
import time

from paper_1511_03404_gb300 import rs


def test_no_thread_gets_the_library_before_its_table(monkeypatch):
    rs.load()
    order = []

    def apply(lib, path=None):
        other = threading.Thread(target=lambda: (rs.load(), order.append("other thread")))
        other.start()
        time.sleep(0.3)
        order.append("table")
        threads.append(other)
        return 0

    threads = []
    monkeypatch.setattr(rs, "_apply_tuned_table", apply)
    monkeypatch.setattr(rs, "_lib", None)
    lib = rs.load()
    for t in threads:
        t.join(30)
    assert order == ["table", "other thread"]
    assert rs.load() is lib
