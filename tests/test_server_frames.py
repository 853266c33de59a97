"""The server's hold on CUDA frames (on the CPU, with the library's calls replaced): a submission drops
every frame that has been processed and holds on to the others; a drained server holds none."""
import types

from paper_2308_00763_gb300 import binding


class _Frame:
    pass


def test_submit_drops_the_frames_that_are_done(monkeypatch):
    done = [0]
    monkeypatch.setattr(binding, "_frame_ptr", lambda f: (4096, 64, 1, f))
    monkeypatch.setattr(binding, "pf_server_submit", lambda *a: 0)
    monkeypatch.setattr(binding, "pf_server_frames_done", lambda h, sid: done[0])
    s = binding.Server.__new__(binding.Server)
    s.h, s._keep, s.cfg = None, {}, types.SimpleNamespace(queue_depth=4)
    frames = [_Frame() for _ in range(4)]

    def held():
        return [t for _, t in s._keep[7][1]]

    assert s.submit(7, frames[0]) and s.submit(7, frames[1])
    assert held() == frames[:2]           # neither is done
    done[0] = 2
    assert s.submit(7, frames[2])
    assert held() == frames[2:3]
    assert s.submit(7, frames[3])
    assert held() == frames[2:]
    monkeypatch.setattr(binding, "pf_server_drain", lambda h: 0)
    s.drain()
    assert held() == []
    assert s.submit(7, frames[0]) and held() == frames[:1]
