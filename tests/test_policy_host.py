"""The policy context manager puts back what it found on entry, whatever the block did.  Needs no
device."""
import pytest

import paper_2203_10213_gb300 as vkt


def now():
    p = vkt.get_policy()
    return p.stream or 0, p.path, p.debug, p.printTimes


@pytest.fixture(autouse=True)
def found():
    before = vkt.get_policy()
    yield now()
    vkt.check(vkt._lib.vktSetThreadExecutionPolicy(before))


# a block whose entry changes nothing, and one whose entry does
@pytest.mark.parametrize("args", [{"stream": 0}, {"stream": 0, "path": "direct"}])
@pytest.mark.parametrize("inner", [{"path": "separable", "debug": True}, {"stream": 4096},
                                   {"print_times": True}])
def test_restores_after_set_policy(found, args, inner):
    with vkt.policy(**args):
        vkt.set_policy(**{"stream": 0, **inner})
        assert now() != found
    assert now() == found
    with pytest.raises(KeyError):
        with vkt.policy(**args):
            vkt.set_policy(**{"stream": 0, **inner})
            raise KeyError
    assert now() == found


def test_one_object_nested_and_as_decorator(found):
    p = vkt.policy(stream=0, path="direct")
    with p:
        with p:
            vkt.set_policy(stream=0, path="separable")
        assert now()[1] == vkt.PATH_DIRECT
    assert now() == found

    @p
    def inside():
        vkt.set_policy(stream=0, path="separable")
        return now()[1]

    assert inside() == vkt.PATHS["separable"]
    assert now() == found
