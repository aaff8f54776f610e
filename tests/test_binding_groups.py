"""The channel groups of a cache as the binding takes them: any mapping, not dicts alone.  Without a GPU the marshalling gets as far
as the first tensor that is not on one."""
import collections
import types

import pytest
import torch

import paper_2504_19874_b200 as tq


class NoPlan:
    handle = 0


def group():
    channels = torch.zeros((1, 64), dtype=torch.int32)
    return {"plan_k": NoPlan(), "plan_v": NoPlan(), "k_idx": None, "k_channels": channels, "v_channels": channels}


@pytest.mark.parametrize("kind", [dict, types.MappingProxyType, collections.UserDict, collections.OrderedDict])
def test_groups_are_mappings(kind):
    x = torch.zeros((1, 128))
    with pytest.raises(ValueError, match="CUDA tensor"):
        tq.tq_kv_append([kind(group())], 1, 4, 0, x, x)
    lacking = group()
    del lacking["plan_v"]
    with pytest.raises(KeyError, match="plan_v"):
        tq.tq_kv_append((kind(lacking),), 1, 4, 0, x, x)


def test_what_is_no_mapping_is_refused():
    x = torch.zeros((1, 128))
    for wrong in (5, "group", None, [1, 2]):
        with pytest.raises((TypeError, ValueError, AttributeError)):
            tq.tq_kv_append([wrong], 1, 4, 0, x, x)
