"""Joining the counts of both directions of an expert-parallel call: without a copy where they are neighbours, right where not."""
import torch

from paper_2605_18643_b200.ep import side_by_side


def test_neighbours_are_joined_in_place_and_others_copied():
    row = torch.arange(12, dtype=torch.int32)
    a, b = row[2:5], row[5:11].view(2, 3)
    joined = side_by_side(a, b)
    assert joined.tolist() == list(range(2, 11)) and joined.data_ptr() == a.data_ptr()
    for x, y in ((row[2:5], row[6:9]), (row[6:9], row[2:6]), (row[2:5], row[5:11:2]), (row[2:5], row[5:8].clone()),
                 (row[0:0], row[3:5]), (row[2:5], row[5:5])):
        assert side_by_side(x, y).tolist() == x.tolist() + y.tolist()
