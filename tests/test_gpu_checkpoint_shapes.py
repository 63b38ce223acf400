"""Checkpoints hold the loop launch shape and the version of the sums that wrote them: a flow is continued with both or not at
all (it continues bit for bit), and tufrg_loop_tiles reports the shape that is stored."""
import struct

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1710_08830_gb300 import inputs  # noqa: E402

VERSION, RANGES = 8, 60   # byte offsets in the checkpoint's header


def _spec(model):
    if model == "bilayer":
        return inputs.rashba_bilayer(Lq=4, nc=3, n_ff=5)
    return inputs.rashba_hubbard(tp=-0.15, alpha=0.3, U=3.3, mu=-0.8, Lq=6, nc=8, n_ff=5)


@pytest.mark.parametrize("model,prec,version", [("rashba", "SPLIT32", 1), ("rashba", "FP64", 2), ("bilayer", "SPLIT32", 2), ("bilayer", "FP64", 2)])
def test_checkpoint_shape_and_version(model, prec, version, tmp_path):
    from paper_1710_08830_gb300 import api
    spec, p = _spec(model), getattr(api, prec)
    m = api.Model(spec, p)
    ck = tmp_path / "flow.ckpt"
    m.flow(stop=6.0, checkpoint_path=str(ck), checkpoint_every=2, stop_after=2)
    raw = ck.read_bytes()
    at = lambda o: struct.unpack_from("<i", raw, o)[0]
    assert at(VERSION) == version and at(RANGES) == m.loop_ky_chunks >= 1

    def resume(offset, value):
        b = bytearray(raw)
        struct.pack_into("<i", b, offset, value)
        f = tmp_path / "changed.ckpt"
        f.write_bytes(bytes(b))
        return m.flow(stop=6.0, resume_from=str(f), stop_after=1)[1]

    assert resume(RANGES, at(RANGES))["n_steps"] == 3
    # no range, more than the rows allow, and a shape that only a model with timed shapes can take up
    for n in (0, 17, -1):
        with pytest.raises(api.TufrgError, match="EINVAL"):
            resume(RANGES, n)
    other = 2 if at(RANGES) == 1 else 1
    if m.loop_tiles_tuning_ms:
        assert resume(RANGES, other)["n_steps"] == 3
    else:
        with pytest.raises(api.TufrgError, match="EINVAL"):
            resume(RANGES, other)
    for v in {1, 2, 3} - {version}:
        with pytest.raises(api.TufrgError, match="EINVAL"):
            resume(VERSION, v)
