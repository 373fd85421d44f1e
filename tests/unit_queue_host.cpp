// UnitQueue (csrc/tc_units.cuh) on barriers of this program, which runs one role at a time: a wait that is not fulfilled yet runs
// out at once, as one does in a kernel that is giving up.  Prints nothing and returns 0, or the number of what went wrong.
#include "tc_units.cuh"

struct Unit { int tile, count; };

struct Io {
    int *flag;          // raised by a wait that runs out
    uint64_t *count;    // arrivals that the barriers of `bars` have seen, and how many complete a phase
    const uint64_t *need;
    uint64_t *bars;
    int *left;          // units that the scheduler still hands over
    bool *others;       // whether the waits of the group's other warps have succeeded
    bool wait(uint64_t *bar, uint32_t parity) const
    {
        const long b = bar - bars;
        if (((count[b] / need[b]) & 1) != parity) return true;   // the phase with that parity has completed
        *flag = 1;
        return false;
    }
    bool late() const { return *flag; }
    bool all(bool x) const { return x; }
    bool all_warps(bool x) const { return x && *others; }
    void arrive(uint64_t *bar) const { ++count[bar - bars]; }
    void request(void *, uint64_t *bar) const { arrive(bar); }   // the answer is there at once
    bool answer(void *, int &bx, int &by) const { bx = 7; by = 8; return (*left)-- > 0; }
};

constexpr int kReaders = 3;
struct World {
    Unit slots[2] = {{-5, 0}, {-5, 0}};
    int late = 0, left;
    bool others = true;
    uint64_t bars[5] = {}, count[5] = {};
    const uint64_t need[5] = {1, 1, kReaders, kReaders, 1};
    attn::tc::UnitQueue<Unit, Io> q;
    explicit World(int units) : left(units - 1), q{slots, bars, bars + 2, bars + 4, nullptr, {&late, count, need, bars, &left, &others}} {}
    bool put(int t) const
    {
        volatile Unit *u = q.claim(t);
        if (!u) return false;
        u->tile = 100 + t; u->count = t;
        q.publish(t);
        q.ask();
        return true;
    }
    void read(int t, int times) const { for (int i = 0; i < times; ++i) q.io.arrive(&q.empty[t & 1]); }
};

int main()
{
    int bx = 0, by = 0;
    for (int units = 1; units <= 7; ++units) {   // as it should go
        World w(units);
        for (int t = 0; t < units; ++t) {
            if (!w.put(t) || !w.q.take(t) || !w.q.take_alone(t) || !w.q.take_together(t) || w.slots[t & 1].tile != 100 + t) return 1;
            if (t > 0) w.read(t - 1, kReaders);
            if (w.q.next(t, bx, by) != (t + 1 < units) || w.late) return 2;
        }
        if (w.q.take(units) || w.q.take_together(units) || w.late) return 3;   // published: there is none
    }
    {   // a role that is still at unit 0: its slot is not given away and nothing is published
        World w(9);
        if (!w.put(0) || !w.q.next(0, bx, by) || !w.put(1) || !w.q.next(1, bx, by)) return 4;
        w.read(0, kReaders - 1);
        if (w.put(2) || !w.late || w.slots[0].tile != 100 || w.q.take(2)) return 5;
    }
    {   // the same at the end of the work: the slot is not marked either
        World w(2);
        if (!w.put(0) || !w.q.next(0, bx, by) || !w.put(1)) return 6;
        w.read(0, kReaders - 1);
        if (w.q.next(1, bx, by) || !w.late || w.slots[0].tile != 100 || w.q.take(2)) return 7;
    }
    {   // no answer, and an answer after a wait of another role has run out: there is no next unit, and no end is published
        World w(9);
        volatile Unit *u = w.q.claim(0);
        u->tile = 100;
        w.q.publish(0);
        if (w.q.next(0, bx, by) || !w.late || w.q.take(1)) return 8;
        w.q.ask();
        if (w.q.next(0, bx, by) || w.q.take(1)) return 9;
    }
    {   // a unit that is there, but not for every warp of a group: none of them takes it
        World w(2);
        w.others = false;
        if (!w.put(0) || !w.q.take(0) || w.q.take_together(0)) return 10;
    }
    return 0;
}
