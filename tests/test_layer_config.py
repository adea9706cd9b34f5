"""The index arrays of a configuration that layers of several widths share (on the CPU: they are plain tensors)."""
import copy

import numpy as np


def test_index_arrays_of_every_width_stay():
    from paper_2510_27527_b200 import binding as b

    cfg = b.LayerConfig(outliers=np.array([1, 5]), concurrent=False)
    mine = cfg.prepare(16, "cpu")
    other = cfg.index(24, "cpu")  # what a module of another width does
    assert cfg.index(16, "cpu") is mine and cfg.index(24, "cpu") is other
    assert cfg._keep is mine[1] and mine[1].numel() == 14 and other[1].numel() == 22
    c = cfg.c()
    assert (c.outlier_cols, c.keep_cols, c.col_map) == tuple(t.data_ptr() for t in mine)
    c = cfg.c(other)
    assert (c.outlier_cols, c.keep_cols, c.col_map) == tuple(t.data_ptr() for t in other)


def test_index_arrays_go_by_value_and_are_bounded():
    from paper_2510_27527_b200 import binding as b

    cfg = b.LayerConfig(outliers=np.array([1, 5]))
    first = cfg.index(16, "cpu")
    cfg.outliers[1] = 7
    outl, keep, cmap = cfg.index(16, "cpu")
    assert outl.tolist() == [1, 7] and 5 in keep.tolist() and cmap.tolist()[5] == 4 and cmap.tolist()[7] == -1
    cfg.outliers = [1, 5]
    assert cfg.index(16, "cpu") is first
    for D in range(20, 60):
        cfg.index(D, "cpu")
    assert len(cfg._arrays._of) == b.IndexCache.MOST
    again = cfg.index(16, "cpu")
    assert again is not first and all(np.array_equal(a, f) for a, f in zip(again, first))
    assert copy.deepcopy(cfg)._arrays._of == {}  # no device memory goes into a copy or a file


def test_index_arrays_are_recorded_on_a_stream_of_their_own_device(monkeypatch):
    """A module whose input lies on another device than the current one launches there (no second device is needed to see which
    stream is asked for)."""
    import torch

    from paper_2510_27527_b200 import binding as b

    class Piece:
        device = torch.device("cuda", 1)
        recorded = []

        def record_stream(self, stream):
            self.recorded.append(stream)

    streams = {0: 10, 1: 21}
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: streams[index], raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: ("stream", 0 if device is None else torch.device(device).index))
    arrays = b.IndexArrays([Piece()] * 3)
    arrays.streams = {21}  # uploaded there
    arrays.here()
    assert Piece.recorded == [] and arrays.streams == {21}
    streams[1] = 22
    arrays.here().here()
    assert Piece.recorded == [("stream", 1)] and arrays.streams == {21, 22}
