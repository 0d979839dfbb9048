"""Many steps per launch beside themselves: shots of several host threads on
streams of their own, shots on several streams of one thread, and a shot
captured into a graph and replayed, each with the results of the shot alone."""
import threading

import numpy as np
import pytest

from helpers import Case, DeviceShot

pytestmark = pytest.mark.gpu


class Shot:
    """One shot with buffers of its own, its results by a first run alone."""

    def __init__(self, seed, r=4, offgrid=False, storage="ckpt"):
        import torch

        import paper_1603_03971_gb300 as rtm

        self.case = Case(nx=44, ny=40, nz=36, nb=10, r=r, nt=24, seed=seed, storage=storage,
                         ckpt_every=7, src=(20, 18, 3))
        self.g = g = DeviceShot(self.case)
        self.dobs = torch.from_numpy(self.case.d_obs(g.nrec).astype(np.float32)).cuda()
        self.img = torch.zeros(rtm.model_shape(g.p), device="cuda")
        self.data = torch.empty((g.p.nt, g.nrec), device="cuda")
        self.taps = (rtm.offgrid_taps(g.p, (20.3, 18.2, 3.4), g.rec_np + 0.3, "cuda")
                     if offgrid else None)
        self.run()
        torch.cuda.synchronize()
        rtm.check(g.ws)
        self.want = self.img.cpu().numpy(), self.data.cpu().numpy()

    def run(self, stream=None):
        import paper_1603_03971_gb300 as rtm

        g = self.g
        if self.taps is None:
            rtm.shot(g.p, g.c, g.rec, self.dobs, g.ws, self.img, data=self.data, stream=stream)
        else:
            rtm.shot_offgrid(g.p, g.c, self.taps, self.dobs, g.ws, self.img, data=self.data,
                             stream=stream)

    def reset(self):
        self.img.zero_()
        self.data.fill_(-1.0)

    def check(self, tol=0.0):
        import paper_1603_03971_gb300 as rtm

        rtm.check(self.g.ws)
        for got, want in zip((self.img.cpu().numpy(), self.data.cpu().numpy()), self.want):
            assert np.abs(got - want).max() <= tol * np.abs(want).max()


def _shots():
    return [Shot(1), Shot(2, r=8), Shot(3, storage="all"), Shot(4), Shot(5, storage="all")]


def test_shots_of_several_threads():
    import torch

    shots = _shots()
    streams = [torch.cuda.Stream() for _ in shots]
    for s in shots:
        s.reset()
    torch.cuda.synchronize()
    errors = []

    def work(k):
        try:
            for _ in range(4):
                with torch.cuda.stream(streams[k]):
                    shots[k].img.zero_()
                shots[k].run(streams[k])
            streams[k].synchronize()
        except Exception as e:  # noqa: BLE001 - reported by the test's thread
            errors.append(e)
    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(shots))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for s in shots:
        s.check()


def test_shots_on_several_streams():
    import torch

    shots = _shots()
    streams = [torch.cuda.Stream() for _ in shots]
    for s in shots:
        s.reset()
    torch.cuda.synchronize()
    for k, s in enumerate(shots):
        s.run(streams[k])
    torch.cuda.synchronize()
    for s in shots:
        s.check()


@pytest.mark.parametrize("offgrid", [False, True])
def test_captured_shot_replays(offgrid):
    import torch

    shot = Shot(6, offgrid=offgrid)
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        shot.run(stream)
    for _ in range(3):
        shot.reset()
        graph.replay()
        torch.cuda.synchronize()
        # off the grid the receivers' taps meet in atomic sums
        shot.check(tol=512 * 24 * 2.0 ** -24 if offgrid else 0.0)
