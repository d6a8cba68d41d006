// Device memory that a context keeps for the checkerboard phases, and how it
// grows (no counterpart in the paper).  Host code only, with the allocator as
// a parameter, so that the rules can be checked without a GPU:
//   void* get(size_t)   device memory, or null
//   bool full()         the last get failed because the memory is used up
//   void put(void*)     gives it back once the work enqueued on it is done
//   size_t available()  free bytes of the device
//   bool capturing()    the call is being captured into a graph of the caller
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

struct WsBuffer {
    void* p = nullptr;
    size_t bytes = 0;
    bool captured = false;   // a graph of the caller may read it
};

struct PhaseWorkspace {
    WsBuffer draws;      // the refinement perturbations of an iteration
    WsBuffer windows;    // the stored windows
    size_t limit = (size_t)16 << 30;   // most bytes of stored windows
    size_t refused = SIZE_MAX;         // windows of this many bytes or more did not fit, although they seemed to
    std::vector<void*> retired;        // replaced buffers of captured calls, kept as long as the context
};

// Takes a buffer out of use: only later calls of this context would use it,
// or a graph that the caller captured a call into.
template <class A>
void ws_release(PhaseWorkspace& w, WsBuffer& b, A& a) {
    if (b.captured) w.retired.push_back(b.p);
    else if (b.p) a.put(b.p);
    b = WsBuffer();
}

// Device memory for anything else of the context: the windows give way to it.
template <class A>
void* ws_get(PhaseWorkspace& w, size_t bytes, A& a) {
    void* p = a.get(bytes);
    if (!p && a.full() && w.windows.p && !w.windows.captured) {
        ws_release(w, w.windows, a);
        p = a.get(bytes);
    }
    return p;
}

// n buffers, all or none.
template <class A>
bool ws_get_all(PhaseWorkspace& w, const size_t* bytes, void** p, int n, A& a) {
    for (int i = 0; i < n; ++i) {
        p[i] = ws_get(w, bytes[i], a);
        if (p[i]) continue;
        while (i > 0) a.put(p[--i]);
        return false;
    }
    return true;
}

// Makes `draws` bytes and, when they can be had, `windows` bytes ready for one
// call; false when the first cannot.  *stored: whether the windows are there.
// The caller takes the two pointers once, for all views of the call.  A buffer
// that is large enough stays where it is, so that a call of the same size
// costs nothing and the graph captured for it stays valid; a larger one is
// there before the smaller one goes.  The windows take at most half of what is
// free, so that the rest of the process finds memory too; asking first also
// spares the calls on a full device an allocation that fails.
template <class A>
bool ws_reserve(PhaseWorkspace& w, size_t draws, size_t windows, bool* stored, A& a) {
    *stored = false;
    if (w.draws.bytes < draws) {
        void* p = ws_get(w, draws, a);
        if (!p) return false;
        ws_release(w, w.draws, a);
        w.draws.p = p;
        w.draws.bytes = draws;
    }
    const bool capturing = a.capturing();   // (nothing can be allocated then)
    w.draws.captured |= capturing;
    if (windows == 0 || windows > w.limit) return true;
    if (w.windows.bytes < windows) {
        if (capturing || windows >= w.refused || windows > (a.available() + w.windows.bytes) / 2) return true;
        void* p = a.get(windows);
        if (!p) {
            if (a.full()) w.refused = windows;
            return true;
        }
        ws_release(w, w.windows, a);
        w.windows.p = p;
        w.windows.bytes = windows;
    }
    w.windows.captured |= capturing;
    *stored = true;
    return true;
}
