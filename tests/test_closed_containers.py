"""A closed container in an operand list is refused: NULL in such a list means
that the operand is not wanted."""
import pytest

from helpers import skel


def test_operand_lists():
    sk = skel()
    x, y, closed = (sk.Container.empty(4) for _ in range(3))
    closed.close()
    for call in (lambda: sk.skel_map("add", [x, closed], y, stream=0),
                 lambda: sk.skel_map_bwd("mul", [x, y], x, [y, closed], stream=0),
                 lambda: sk.skel_map_bwd("tanh", [closed], x, [y], stream=0),
                 lambda: sk.skel_mapreduce("sq", "add", [closed], stream=0)):
        with pytest.raises(sk.SkelError) as e:
            call()
        assert e.value.code == -1
    assert len(sk._handles([x, None])) == 2 and sk._handles([None])[0] is None
    assert sk._handles([x])[0] == x.handle.value
